"""Von Neumann service far from stability: the growth of steps of any length.

With dt/dx times a velocity, or dt/tau, of 1e10 to 1e150 G's entries are that
large (its diagonal in the first case, all of it in the second), and so is its
spectral radius, which the oracle (LAPACK) gives to its precision: the
service's bound, 1e-10 relative, holds as at ordinary steps.
"""
import math

import numpy as np
import pytest

from oracle import vonneumann

pytestmark = pytest.mark.gpu

STATES = [(1.0, 0.0, 0.0, 0.0, 1.0), (2.7, 1.5, -0.4, 0.2, 1.7)]
DIRS = [(1.0, 0.0, 0.0), (0.0, 1.0, 2.0)]


@pytest.mark.parametrize("nk", [5, 700])  # eight, four lanes per matrix
@pytest.mark.parametrize("dt", [1e10, 1e40, 1e70, 1e78, 1e90, 1e120, 1e148])
def test_growth_of_long_steps(dt, nk):
    from paper_1010_4135_gb300 import stability
    params = [(2.0, 6.0, 4.0, 1.4, dt, dt, 1.0 / 64), (3.0, 9.0, 6.0, 1.4, dt, 3.0 * dt, 1.0 / 64),
              (2.0, 6.0, 4.0, 1.4, 1e-5, 1e-5 / dt, 1.0 / 64), (3.0, 9.0, 6.0, 1.4, dt, 1.0 / 64, 1.0 / 64)]
    got = stability.max_growth_device(STATES, params, directions=DIRS, nk=nk)
    sample = range(1, nk + 1) if nk < 10 else (1, nk // 2, nk)
    kdx = math.pi * np.array(list(sample)) / nk
    for p, value in zip(params, got):
        want = max(vonneumann.max_growth(s[0], s[1:4], s[4], *p[:4], p[4], p[5], p[6], kdx, d)
                   for s in STATES for d in DIRS)
        if nk < 10:
            assert abs(value - want) <= 1e-10 * want, (p, value, want)
        else:  # the oracle on a few of the wave numbers: a lower bound of the maximum
            assert np.isfinite(value) and value >= want * (1.0 - 1e-10), (p, value, want)
