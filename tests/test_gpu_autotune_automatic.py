"""A tuned launch is not slower than the automatic one.

Grids whose automatic chunks no explicit (z chunk, tail) pair gives: two
lengths a plane apart, and tails of four planes.  Both sides are timed here,
the best of five runs of many steps each; 5 % covers what such runs differ by.
"""
import pytest

import oracle
from parity_util import STATE_HI, STATE_LO, initial_f, sim_for

pytestmark = pytest.mark.gpu


def _us(s, steps):
    import torch
    best = float("inf")
    s.step(5)
    for _ in range(5):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(s.stream)
        s.step(steps)
        b.record(s.stream)
        b.synchronize()
        best = min(best, a.elapsed_time(b) / steps * 1e3)
    return best


@pytest.mark.parametrize("n", [(64, 64, 64), (192, 128, 128)], ids=lambda n: "x".join(map(str, n)))
def test_tuned_is_not_slower_than_untuned(n, tmp_path):
    import numpy as np

    from paper_1010_4135_gb300 import autotune
    cfg = oracle.Cfg(nx=n[0], ny=n[1], nz=n[2], c1=2.0, c2=6.0, eta0=4.0, gamma=1.4, tau=2e-4, dt=2e-4, dx=0.02,
                     bc_lo=(1, 0, 0), bc_hi=(2, 0, 0), fixed_lo=(STATE_LO,) * 3, fixed_hi=(STATE_HI,) * 3)
    s = sim_for(cfg, "fp32")
    s.set_f(initial_f(cfg, seed=12, noise=0.0).astype(np.float32))
    untuned = _us(s, 100)
    autotune.tune(s, path=str(tmp_path / "launch.json"))
    assert _us(s, 100) <= 1.05 * untuned
