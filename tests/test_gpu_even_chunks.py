"""Chunks the FP32 step takes by itself on grids of few planes per CTA slot.

Such grids are cut into chunks of two lengths, one plane apart.  A chunking
changes which CTA works on a plane, not the arithmetic, so the state after a
few steps is bitwise that of one chunk per column.
"""
import numpy as np
import pytest

import oracle
from parity_util import STATE_HI, STATE_LO, initial_f, sim_for

pytestmark = pytest.mark.gpu

# one plane; a chunk per plane; even and uneven cuts; more tiles than CTA slots
SHAPES = [(33, 17, 1), (36, 30, 31), (64, 64, 64), (61, 35, 48), (500, 40, 44), (352, 224, 9), (1, 1, 40)]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_even_chunks_equal_whole_columns(shape):
    nx, ny, nz = shape
    cfg = oracle.Cfg(nx=nx, ny=ny, nz=nz, c1=2.0, c2=6.0, eta0=4.0, gamma=1.4, tau=2e-4, dt=2e-4, dx=0.02,
                     bc_lo=(1, 0, 0), bc_hi=(1, 0, 0), fixed_lo=(STATE_LO,) * 3, fixed_hi=(STATE_HI,) * 3)
    f0 = initial_f(cfg, seed=300 + nz)
    out = []
    for zchunk in (0, nz):
        s = sim_for(cfg, "fp32")
        s.set_launch("tiled", zchunk, 0)
        s.set_f(f0.astype(np.float32))
        s.step(4)
        out.append(s.get_f())
        assert s.health() == 0
        s.close()
    assert np.isfinite(out[0]).all()
    assert np.array_equal(out[0], out[1])


# few planes per slot (even chunks), more (long and short chunks over grids of
# different heights), more tiles than slots
BATCHES = [[(64, 64, 20), (33, 17, 9), (36, 30, 31)], [(96, 96, 40), (64, 70, 64), (128, 64, 50)],
           [(320, 248, 4), (33, 9, 1)]]


@pytest.mark.parametrize("shapes", BATCHES, ids=["even", "long_and_short", "many_tiles"])
def test_batch_chunks_equal_whole_columns(shapes):
    from paper_1010_4135_gb300 import sim as S
    out = []
    for whole in (False, True):
        sims = []
        for nx, ny, nz in shapes:
            cfg = oracle.Cfg(nx=nx, ny=ny, nz=nz, c1=2.0, c2=6.0, eta0=4.0, gamma=1.4, tau=2e-4, dt=2e-4, dx=0.02,
                             bc_lo=(1, 0, 0), bc_hi=(1, 0, 0), fixed_lo=(STATE_LO,) * 3, fixed_hi=(STATE_HI,) * 3)
            s = sim_for(cfg, "fp32")
            if whole:
                s.set_launch("tiled", nz, 0)
            s.set_f(initial_f(cfg, seed=300 + nz).astype(np.float32))
            sims.append(s)
        S.step_batch(sims, 4)
        out.append([s.get_f() for s in sims])
        assert all(s.health() == 0 for s in sims)
        for s in sims:
            s.close()
    for a, b in zip(*out):
        assert np.isfinite(a).all() and np.array_equal(a, b)
