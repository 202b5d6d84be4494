"""Initialisation, moments and conservation sums: the integer forms of their
FP64 work (conversion to float, fixed-point sums) against the FP64 sim's
results, the oracle and exact sums, at the ends of their ranges."""
import math

import numpy as np
import pytest

import oracle
import workloads
from parity_util import case_cfg, initial_f, sim_for

pytestmark = pytest.mark.gpu

CFG = "wide_70x9x5"


@pytest.mark.parametrize("scale", [1.0, 1e-30, 3e-38, 1e-44, 2e37, 1e39, 0.0])
def test_fp32_init_rounds_the_fp64_equilibrium(scale):
    """Both precisions evaluate f^eq by the same FP64 operations, so the FP32
    state is the FP64 one rounded to nearest: bitwise, through the subnormal
    range, zero and overflow."""
    cfg = case_cfg(CFG)
    rho, u, T = workloads.smooth_random_fields(cfg.nx, cfg.ny, cfg.nz, 3, amp=0.2)
    out = {}
    for prec in ("fp64", "fp32"):
        s = sim_for(cfg, prec)
        s.init(rho * scale, u, T)
        out[prec] = s.get_f()
    with np.errstate(over="ignore"):
        assert np.array_equal(out["fp32"], out["fp64"].astype(np.float32))


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("power", [0, -100, 100, -120])
def test_moments_of_scaled_states(precision, power):
    """rho scales with f, u and T do not; -100 and -120 leave the float sums' fixed-point range."""
    cfg = case_cfg(CFG)
    f = initial_f(cfg, seed=4)
    if precision == "fp32":
        f = f.astype(np.float32)
    s = sim_for(cfg, precision)
    s.set_f(f * f.dtype.type(2.0) ** power)
    r, u, T = s.moments()
    ro, uo, To = oracle.macros(cfg, f.astype(np.float64))
    tol = 1e-12 if power > -120 or precision == "fp64" else 1e-4  # subnormal floats hold fewer bits
    assert np.abs(r * 2.0 ** -power - ro).max() <= tol * np.abs(ro).max()
    assert np.abs(u - uo).max() <= tol * np.abs(uo).max()
    assert np.abs(T - To).max() <= tol * np.abs(To).max()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("name", ["wide_70x9x5", "periodic_37x19x11", "single_cell_1x1x1", "full_tiles_64x16x10"])
def test_conserved_against_exact_sums(precision, name):
    cfg = case_cfg(name)
    f = initial_f(cfg, seed=8)
    if precision == "fp32":
        f = f.astype(np.float32)
    s = sim_for(cfg, precision)
    s.set_f(f)
    got = s.conserved()
    v, eta = oracle.velocities(cfg)
    total = [math.fsum(f[i].astype(np.float64).ravel()) for i in range(15)]
    size = [math.fsum(np.abs(f[i]).astype(np.float64).ravel()) for i in range(15)]
    w = np.vstack([np.ones(15), v.T, (v * v).sum(1) + eta * eta])
    for q in range(5):
        want = math.fsum(w[q, i] * total[i] for i in range(15))
        scale = math.fsum(abs(w[q, i]) * size[i] for i in range(15))
        assert abs(got[q] - want) <= 1e-14 * scale


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("at", [(0, 0, 0, 0), (14, 4, 8, 69), (7, 2, 3, 68)])
def test_conserved_flags_non_finite_values(precision, bad, at):
    from paper_1010_4135_gb300 import _abi as A
    cfg = case_cfg(CFG)
    f = initial_f(cfg, seed=9)
    f[at] = bad
    s = sim_for(cfg, precision)
    s.set_f(f if precision == "fp64" else f.astype(np.float32))
    with pytest.raises(A.LbmError):
        s.conserved()
    assert s.health() & A.LBM_HEALTH_NONFINITE
