"""The pair kernel's forms give bitwise the same state.

A launch takes the form of the kernel with the parts its grids need; a batch
takes the one that serves all its members.  So a grid stepped alone, in its
own form, must equal the same grid batched with a few-row grid between walls,
which takes the form with all parts.
"""
import numpy as np
import pytest

import oracle
from parity_util import NTHREADS, STATE_HI, STATE_LO, field_errors, initial_f, sim_for

pytestmark = pytest.mark.gpu
P, F, E, R = 0, 1, 2, 3
STEPS = 10
TUBE = ((F, P, P), (E, P, P))
BOX = ((E, R, R), (F, R, R))
# whole tiles and cut ones, without and with x faces, walls, few rows
GRIDS = [((64, 16, 10), ((P, P, P), (P, P, P))), ((64, 16, 10), TUBE), ((37, 11, 9), ((F, P, P), (F, P, P))),
         ((38, 11, 9), TUBE), ((34, 10, 9), BOX), ((70, 3, 5), TUBE)]


def _cfg(n, bc, tau, scheme):
    return oracle.Cfg(nx=n[0], ny=n[1], nz=n[2], c1=2.0, c2=6.0, eta0=4.0, gamma=1.4, tau=tau, dt=2e-4, dx=0.02,
                      bc_lo=bc[0], bc_hi=bc[1], fixed_lo=(STATE_LO,) * 3, fixed_hi=(STATE_HI,) * 3, scheme=scheme)


def _sim(cfg, f0, recovery):
    s = sim_for(cfg, "fp32")
    s.set_t_recovery(recovery)
    s.set_f(f0)
    return s


@pytest.mark.parametrize("scheme", [oracle.NND, oracle.UPWIND2, oracle.UPWIND1])
@pytest.mark.parametrize("tau,recovery", [(2e-4, 0.0), (5e-4, 0.0), (2e-4, 1.0), (5e-4, 4.0)])
@pytest.mark.parametrize("n,bc", GRIDS)
def test_own_form_equals_the_form_with_all_parts(n, bc, tau, recovery, scheme):
    from paper_1010_4135_gb300 import sim as S
    cfg = _cfg(n, bc, tau, scheme)
    f0 = initial_f(cfg, seed=60 + n[0]).astype(np.float32)
    alone = _sim(cfg, f0, recovery)
    alone.step(STEPS)
    assert alone.health() == 0
    ref = oracle.run(cfg, f0.astype(np.float64), STEPS, NTHREADS)
    assert field_errors(alone.get_f(), ref).max() <= 5e-5  # the FP32 bar of the parity tests
    other = _cfg((33, 3, 4), ((F, P, R), (E, P, R)), tau, scheme)
    batch = [_sim(cfg, f0, recovery), _sim(other, initial_f(other, seed=3).astype(np.float32), 4.0)]
    S.step_batch(batch, STEPS)
    assert np.array_equal(alone.get_f(), batch[0].get_f())
