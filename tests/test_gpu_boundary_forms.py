"""Boundary layers the FP32 pair kernel forms or wraps itself.

The planes of a periodic z axis are read where they are, and the layers of
reflecting faces and of extrapolating x faces are formed as they are read;
where a face does not qualify (odd nx at x-hi, odd ny at y-hi, y and z
extrapolation) a fill launch writes them.  Each grid is checked against the
oracle (the FP32 bar of the parity tests, 5e-5 per field after ten steps),
and bitwise over chunkings (a chunk may start or end at, or one plane away
from, a face), the fill variant, the other tile width and a batched step.
"""
import dataclasses

import numpy as np
import pytest

import oracle
from parity_util import NTHREADS, STATE_HI, STATE_LO, field_errors, initial_f, sim_for

pytestmark = pytest.mark.gpu

FP32_TOL = 5e-5
STEPS = 10
P, F, E, R = 0, 1, 2, 3  # periodic, fixed, extrapolate, reflect

# (nx, ny, nz), kinds of the lo faces, kinds of the hi faces
GRIDS = {
    "reflect_even": ((34, 10, 9), (R, R, R), (R, R, R)),
    "reflect_odd": ((33, 9, 6), (R, R, R), (R, R, R)),
    "reflect_one_plane": ((32, 8, 1), (E, R, R), (E, R, R)),
    "reflect_two_planes": ((64, 16, 2), (E, R, R), (F, R, R)),
    "extrapolate_pair": ((2, 8, 3), (E, P, P), (E, P, P)),
    "extrapolate_odd": ((35, 7, 4), (E, P, P), (E, P, P)),
    "extrapolate_all": ((36, 12, 7), (E, E, E), (E, E, E)),
    "periodic_z1": ((32, 16, 1), (F, P, P), (E, P, P)),
    "periodic_z2": ((33, 5, 2), (P, P, P), (P, P, P)),
    "periodic_z3": ((40, 3, 3), (P, P, P), (P, P, P)),
    "one_row": ((33, 1, 4), (F, P, P), (E, P, P)),
    "two_rows": ((64, 2, 5), (F, P, P), (F, P, P)),
    "three_rows_and_walls": ((34, 3, 6), (E, P, R), (F, P, R)),
    "mixed_walls": ((64, 8, 13), (F, R, E), (E, F, R)),
}


def _cfg(name, **kw):
    (nx, ny, nz), lo, hi = GRIDS[name]
    return oracle.Cfg(nx=nx, ny=ny, nz=nz, c1=2.0, c2=6.0, eta0=4.0, gamma=1.4, tau=2e-4, dt=2e-4, dx=0.02,
                      bc_lo=lo, bc_hi=hi, fixed_lo=(STATE_LO,) * 3, fixed_hi=(STATE_HI,) * 3, **kw)


def _run(cfg, f0, launch=("tiled", 0, 0), recovery=0.0):
    s = sim_for(cfg, "fp32")
    s.set_launch(*launch)
    s.set_t_recovery(recovery)
    s.set_f(f0)
    s.step(STEPS)
    assert s.health() == 0
    return s.get_f()


@pytest.mark.parametrize("scheme", [oracle.NND, oracle.UPWIND2, oracle.UPWIND1])
@pytest.mark.parametrize("name", sorted(GRIDS))
def test_boundary_forms(name, scheme):
    from paper_1010_4135_gb300 import sim as S
    cfg = _cfg(name, scheme=scheme)
    f0 = initial_f(cfg, seed=200 + len(name)).astype(np.float32)
    got = _run(cfg, f0)
    ref = oracle.run(cfg, f0.astype(np.float64), STEPS, NTHREADS)
    assert field_errors(got, ref).max() <= FP32_TOL
    for launch in (("tiled", 1, 0), ("tiled", 2, 0), ("tiled", 3, 1), ("tiled", 5, 2), ("tiled_fill", 0, 0),
                   ("tiled64", 0, 0), ("split", 2, 0)):
        assert np.array_equal(got, _run(cfg, f0, launch)), launch
    pair = []
    for _ in range(2):
        s = sim_for(cfg, "fp32")
        s.set_f(f0)
        pair.append(s)
    S.step_batch(pair, STEPS)
    assert all(np.array_equal(got, s.get_f()) for s in pair)


@pytest.mark.parametrize("name", ["reflect_even", "extrapolate_odd"])
def test_boundary_forms_with_recovery_and_other_relaxation(name):
    """The form with all parts: dt != tau, and the FP64 temperature recovery (its layers come from the fill)."""
    cfg = dataclasses.replace(_cfg(name), tau=5e-4)
    f0 = initial_f(cfg, seed=300).astype(np.float32)
    ref = oracle.run(cfg, f0.astype(np.float64), STEPS, NTHREADS)
    for kappa in (0.0, 1.0):
        got = _run(cfg, f0, recovery=kappa)
        assert field_errors(got, ref).max() <= FP32_TOL
        assert np.array_equal(got, _run(cfg, f0, ("tiled", 1, 0), kappa))
