"""With temperature recovery on, the step handles the same boundary layers as without it.

The layers take the FP32 moments of the cells at the face in either case, so
no fill is launched between steps where none is without recovery, and a
bound that no cell exceeds leaves the state bitwise what it is without.
"""
import numpy as np
import pytest

import oracle
from parity_util import STATE_HI, STATE_LO, initial_f, sim_for

pytestmark = pytest.mark.gpu
P, F, E, R = 0, 1, 2, 3


@pytest.mark.parametrize("n,lo,hi", [((64, 16, 10), (F, P, P), (E, P, P)), ((34, 10, 9), (E, R, R), (R, R, R)),
                                     ((36, 2, 5), (E, P, R), (R, P, R))])
def test_no_fill_between_steps_with_recovery(n, lo, hi):
    cfg = oracle.Cfg(nx=n[0], ny=n[1], nz=n[2], c1=2.0, c2=6.0, eta0=4.0, gamma=1.4, tau=2e-4, dt=2e-4, dx=0.02,
                     bc_lo=lo, bc_hi=hi, fixed_lo=(STATE_LO,) * 3, fixed_hi=(STATE_HI,) * 3)
    f0 = initial_f(cfg, seed=90).astype(np.float32)
    fills, states = [], []
    for kappa in (0.0, 1.0, 1e30):
        s = sim_for(cfg, "fp32")
        s.set_t_recovery(kappa)
        s.set_f(f0)
        s.step(2)
        s.timing(reset=True)
        s.step(10)
        fills.append(s.timing()["fill"][1])
        states.append(s.get_f())
        assert s.health() == 0
    assert fills == [fills[0]] * 3 and fills[0] == 0
    assert np.array_equal(states[0], states[2])
