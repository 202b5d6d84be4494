"""Conservation sums of floats whose running sums leave the float range.

The values are finite and the sums are doubles, so the result is the exact
sum (1e-14 of the sum of magnitudes, the bound of the other exact-sum test)
and no health bit is raised, however many of them a lane adds.
"""
import numpy as np
import pytest

import oracle
from parity_util import sim_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("value", [1e30, 1e37, -1e37, 2.9e38 / 2])
@pytest.mark.parametrize("n", [(64, 160, 160), (200, 3, 5), (1, 1, 1)])
def test_finite_floats_of_any_size(n, value):
    cfg = oracle.Cfg(nx=n[0], ny=n[1], nz=n[2], c1=2.0, c2=6.0, eta0=4.0, gamma=1.4, tau=2e-4, dt=2e-4, dx=0.02)
    f = np.full((15, n[2], n[1], n[0]), value, dtype=np.float32)
    s = sim_for(cfg, "fp32")
    s.set_f(f)
    got = s.conserved()
    assert s.health() == 0
    v, eta = oracle.velocities(cfg)
    w = np.vstack([np.ones(15), v.T, (v * v).sum(1) + eta * eta])
    total = float(np.float32(value)) * (n[0] * n[1] * n[2])
    for q in range(5):
        assert abs(got[q] - w[q].sum() * total) <= 1e-14 * np.abs(w[q]).sum() * abs(total)


@pytest.mark.parametrize("at", [(0, 0, 0, 0), (3, 4, 2, 199), (14, 2, 1, 130)])
def test_a_nan_beside_large_finite_values_is_flagged(at):
    from paper_1010_4135_gb300 import _abi as A
    cfg = oracle.Cfg(nx=200, ny=3, nz=5, c1=2.0, c2=6.0, eta0=4.0, gamma=1.4, tau=2e-4, dt=2e-4, dx=0.02)
    f = np.full((15, 5, 3, 200), 1e37, dtype=np.float32)
    f[at] = np.nan
    s = sim_for(cfg, "fp32")
    s.set_f(f)
    with pytest.raises(A.LbmError):
        s.conserved()
    assert s.health() & A.LBM_HEALTH_NONFINITE
