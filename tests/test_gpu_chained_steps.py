"""Chained steps equal separate ones.

The step and fill kernels overlap their successor's start (programmatic
dependent launch).  Many steps in one call, in which each kernel is resident
before its predecessor ends, give bitwise the state of the same steps with a
synchronisation after each.  Faces that a fill writes before each step, odd
extents (boundary cells and layers in one line) and every form of the FP64
step (seven, three, one block per row) are among the cases.
"""
import numpy as np
import pytest

import oracle
from parity_util import STATE_HI, STATE_LO, initial_f, sim_for

pytestmark = pytest.mark.gpu
P, F, E, R = 0, 1, 2, 3

CASES = [((201, 3, 3), (E, P, P), (E, P, P)), ((33, 9, 7), (F, R, E), (E, E, R)), ((61, 17, 19), (E, R, R), (F, R, R)),
         ((127, 33, 29), (F, E, R), (E, R, E)), ((65, 64, 62), (R, E, E), (E, E, R))]


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("n,lo,hi", CASES, ids=lambda v: "x".join(map(str, v)))
def test_chained_steps_equal_separate_ones(n, lo, hi, precision):
    cfg = oracle.Cfg(nx=n[0], ny=n[1], nz=n[2], c1=2.0, c2=6.0, eta0=4.0, gamma=1.4, tau=2e-4, dt=2e-4, dx=0.02,
                     bc_lo=lo, bc_hi=hi, fixed_lo=(STATE_LO,) * 3, fixed_hi=(STATE_HI,) * 3)
    f0 = initial_f(cfg, seed=700 + n[0])
    out = []
    for chained in (True, False):
        s = sim_for(cfg, precision)
        s.set_f(f0 if precision == "fp64" else f0.astype(np.float32))
        if chained:
            s.step(60)
        else:
            for _ in range(60):
                s.step(1)
                s.sync()
        out.append(s.get_f())
        assert s.health() == 0
        s.close()
    assert np.isfinite(out[0]).all() and np.array_equal(*out)
