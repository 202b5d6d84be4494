"""The von Neumann kernel's two splits (eight lanes per matrix below 16
matrices per SM, four from there on): a batch on either side of the line, and
counts that leave the last block partly empty, agree with the oracle to the
service's bound (1e-10 relative)."""
import math

import numpy as np
import pytest

from oracle import vonneumann

pytestmark = pytest.mark.gpu

TOL = 1e-10
STATES = [(1.0, 0.0, 0.0, 0.0, 1.0), (2.7, 1.5, -0.4, 0.2, 1.7), (0.3, 2.0, 0.0, 0.1, 5.0)]
PARAMS = [(c1, 3.0 * c1, 2.0 * c1, 1.4, dt, tau, 1.0 / 64) for c1 in (2.0, 3.0, 5.0) for dt, tau in
          ((1e-5, 1e-5), (1e-5, 3e-5))]


@pytest.mark.parametrize("nstates,nparams,nk", [(1, 1, 1), (1, 2, 5), (3, 6, 67), (3, 6, 68), (3, 5, 83)])
def test_lane_splits(nstates, nparams, nk):
    from paper_1010_4135_gb300 import stability
    dirs = [(1.0, 0.0, 0.0), (0.0, 1.0, 2.0)]
    states, params = STATES[:nstates], PARAMS[:nparams]
    got = stability.max_growth_device(states, params, directions=dirs, nk=nk)
    kdx = math.pi * np.arange(1, nk + 1) / nk
    for p, value in zip(params, got):
        want = max(vonneumann.max_growth(s[0], s[1:4], s[4], *p[:4], p[4], p[5], p[6], kdx, d)
                   for s in states for d in dirs)
        assert abs(value - want) <= TOL * want, (p, value, want)


@pytest.mark.parametrize("nparams", [1, 80])
def test_non_finite_matrices_report_infinity(nparams):
    from paper_1010_4135_gb300 import stability
    bad = (2.0, 6.0, 4.0, 1.4, float("nan"), 1e-5, 1.0 / 64)
    got = stability.max_growth_device(STATES[:1], [bad] + [PARAMS[0]] * nparams, nk=24)
    assert np.isinf(got[0]) and np.isfinite(got[1:]).all()
