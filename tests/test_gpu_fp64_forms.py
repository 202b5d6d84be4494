"""The FP64 step kernel's forms: its split of small grids over blocks, its
wrapped periodic axes, and its fixed-point sums with their double fallback.

Bounds: 1e-12 per field against the oracle (the FP64 bar).  The step is
homogeneous of degree one in f (rho scales, u and T do not), so scaling f by
a power of two scales every value, difference, sum and product exactly: the
results are bitwise the same, as long as both runs take the fixed-point form.
"""
import numpy as np
import pytest

import oracle
from parity_util import NTHREADS, STATE_HI, STATE_LO, field_errors, initial_f, sim_for

pytestmark = pytest.mark.gpu

FP64_TOL = 1e-12
P, F, E, R = 0, 1, 2, 3


def _cfg(n, lo=(P, P, P), hi=(P, P, P), dt=2e-4, tau=2e-4, **kw):
    return oracle.Cfg(nx=n[0], ny=n[1], nz=n[2], c1=2.0, c2=6.0, eta0=4.0, gamma=1.4, tau=tau, dt=dt, dx=0.02,
                      bc_lo=lo, bc_hi=hi, fixed_lo=(STATE_LO,) * 3, fixed_hi=(STATE_HI,) * 3, **kw)


def _run(cfg, f0, steps):
    s = sim_for(cfg, "fp64")
    s.set_f(f0)
    s.step(steps)
    return s.get_f(), s.health()


# warps of 32 cells: 7 blocks per row up to 304 of them, 3 up to 912, 8 rows per block from 2432 on (152 SMs)
@pytest.mark.parametrize("scheme", [oracle.NND, oracle.UPWIND2, oracle.UPWIND1])
@pytest.mark.parametrize("n", [(1, 1, 1), (3, 2, 1), (33, 8, 19), (32, 16, 20), (70, 17, 18), (40, 31, 33), (64, 48, 60)])
def test_block_splits(n, scheme):
    for lo, hi, tau in (((P, P, P), (P, P, P), 2e-4), ((F, R, P), (F if n[0] < 2 else E, R, P), 5e-4)):
        cfg = _cfg(n, lo, hi, tau=tau, scheme=scheme, dissipation=int(tau < 4e-4))
        f0 = initial_f(cfg, seed=sum(n))
        got, health = _run(cfg, f0, 4)
        assert health == 0
        assert field_errors(got, oracle.run(cfg, f0, 4, NTHREADS)).max() <= FP64_TOL


@pytest.mark.parametrize("power", [-60, 1, 60])
def test_scaling_by_a_power_of_two_is_bitwise(power):
    cfg = _cfg((37, 12, 9), (P, R, P), (P, R, P))
    f0 = initial_f(cfg, seed=5)
    a, _ = _run(cfg, f0, 5)
    b, health = _run(cfg, f0 * 2.0 ** power, 5)
    assert health == 0
    assert np.array_equal(a * 2.0 ** power, b)


@pytest.mark.parametrize("power", [-880, 0])
def test_double_fallback(power):
    """Tiny populations (below the fixed-point range) and exact zeros over whole stencils."""
    cfg = _cfg((37, 12, 9), (P, R, P), (P, R, P), tau=5e-4)
    f0 = initial_f(cfg, seed=6)
    if power == 0:
        f0[5] = 0.0
        f0[9, :5, :7, 3:20] = 0.0
        f0[0, 2, 3, 4] = 0.0
    got, _ = _run(cfg, f0 * 2.0 ** power, 5)
    ref = oracle.run(cfg, f0, 5, NTHREADS)
    assert field_errors(got * 2.0 ** -power, ref).max() <= FP64_TOL


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_values_reach_the_cells_whose_differences_hold_them(bad):
    """The limiter takes its other argument where one is not finite, so a
    value spreads in one step to its own cell (every field, by the moments)
    and to the cells it is the upwind neighbour of: for (+,+,-), x+1, y+1, z-1."""
    from paper_1010_4135_gb300 import _abi as A
    cfg = _cfg((20, 9, 7))
    f0 = initial_f(cfg, seed=7)
    f0[8, 3, 4, 10] = bad
    got, health = _run(cfg, f0, 1)
    assert health & A.LBM_HEALTH_NONFINITE
    want = np.zeros(f0.shape, dtype=bool)
    want[:, 3, 4, 10] = want[8, 3, 4, 11] = want[8, 3, 5, 10] = want[8, 2, 4, 10] = True
    assert np.array_equal(~np.isfinite(got), want)
