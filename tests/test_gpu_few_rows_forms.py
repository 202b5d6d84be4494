"""Periodic images in grids of any height in the kernel forms that serve few rows.

Those forms run for grids of one to three periodic rows, for every grid of a
batch that has such a member, and for dt != tau and the upwind schemes, where
the other grids have four rows or many.  A batched state is bitwise the one
of the grid stepped alone; the states are checked against the oracle (the
FP32 bar, 5e-5 per field after ten steps).  A tall grid's step may not cost a
walk over its rows: the batch of a tall and a three-row grid takes less than
twice the time of the tall grid alone (256^3 beside 200 x 3 x 3: 1.08 times; nine
times with a walk).
"""
import numpy as np
import pytest

import oracle
from parity_util import NTHREADS, STATE_HI, STATE_LO, field_errors, initial_f, sim_for

pytestmark = pytest.mark.gpu
P, F, E, R = 0, 1, 2, 3
STEPS = 10


def _cfg(n, tau=2e-4, scheme=oracle.NND, bc=((F, P, P), (E, P, P))):
    return oracle.Cfg(nx=n[0], ny=n[1], nz=n[2], c1=2.0, c2=6.0, eta0=4.0, gamma=1.4, tau=tau, dt=2e-4, dx=0.02,
                      bc_lo=bc[0], bc_hi=bc[1], fixed_lo=(STATE_LO,) * 3, fixed_hi=(STATE_HI,) * 3, scheme=scheme)


@pytest.mark.parametrize("tau,scheme", [(2e-4, oracle.NND), (5e-4, oracle.NND), (2e-4, oracle.UPWIND2),
                                        (5e-4, oracle.UPWIND1)])
def test_rows_of_every_height_with_a_few_row_member(tau, scheme):
    from paper_1010_4135_gb300 import sim as S
    cfgs = [_cfg((33, ny, nz), tau, scheme) for ny, nz in ((1, 3), (2, 5), (3, 4), (4, 4), (5, 3), (19, 6))]
    f0 = [initial_f(c, seed=40 + c.ny).astype(np.float32) for c in cfgs]
    together = []
    for c, f in zip(cfgs, f0):
        s = sim_for(c, "fp32")
        s.set_f(f)
        together.append(s)
    S.step_batch(together, STEPS)
    for c, f, b in zip(cfgs, f0, together):
        s = sim_for(c, "fp32")
        s.set_f(f)
        s.step(STEPS)
        assert s.health() == 0
        assert np.array_equal(s.get_f(), b.get_f()), c.ny
        ref = oracle.run(c, f.astype(np.float64), STEPS, NTHREADS)
        assert field_errors(s.get_f(), ref).max() <= 5e-5, c.ny


def test_a_few_row_member_leaves_a_tall_grid_its_speed():
    import torch
    from paper_1010_4135_gb300 import sim as S

    def us(n_sims):
        sims = []
        for n in ((64, 512, 64), (64, 3, 3))[:n_sims]:
            s = sim_for(_cfg(n), "fp32")
            s.init(*(np.ones(((3,) if k == 1 else ()) + s.shape) * (0.0 if k == 1 else 1.0) for k in range(3)))
            sims.append(s)
        S.step_batch(sims, 5)
        best = float("inf")
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record(sims[0].stream)
            S.step_batch(sims, 20)
            b.record(sims[0].stream)
            b.synchronize()
            best = min(best, a.elapsed_time(b) * 50.0)
        return best

    assert us(2) < 2.0 * us(1)
