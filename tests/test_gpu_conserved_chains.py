"""Conservation sums of large grids of like values, FP64 storage.

Where all values are alike (as in most of an initial state) every addition of
a lane's running sum rounds the same way, so the error grows with the length
of that chain.  The kernel's scheme (pairs of a load, 32 of them, then those
sums), followed here on paper for 400 random values at this grid's chain of
432 values per lane, is off by 1.5e-15 of the sum at most, one chain by
1.2e-14: the bound is 2e-15.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TOL = 2e-15
N = 256


@pytest.mark.parametrize("kind", ["uniform", "halves", "rows"])
def test_conserved_of_like_values(kind):
    import torch

    from paper_1010_4135_gb300 import sim as S
    s = S.Sim(N, N, N, 2.0, 6.0, 4.0, 2e-4, 2e-4, 0.02, gamma=1.4, precision="fp64", bc_lo=(0, 0, 0), bc_hi=(0, 0, 0))
    f = torch.empty((15, N, N, N), dtype=torch.float64, device=s.device)
    v = np.array([[0.0] * 3] + [[2.0 * g * (a == b) for b in range(3)] for a in range(3) for g in (1, -1)] +
                 [[x, y, z] for x in (1, -1) for y in (1, -1) for z in (1, -1)], dtype=np.longdouble)
    v[7:] *= np.longdouble(6) / np.sqrt(np.longdouble(3))
    eta2 = np.array([16.0] + [0.0] * 14, dtype=np.longdouble)
    w = np.vstack([np.ones(15, dtype=np.longdouble), v.T, (v * v).sum(1) + eta2])
    for seed in range(8):
        a, b = np.random.default_rng(seed).uniform(0.01, 1.0, (2, 15))
        f[:] = torch.from_numpy(a).to(s.device)[:, None, None, None]
        if kind == "halves":
            f[..., N // 2:] = torch.from_numpy(b).to(s.device)[:, None, None, None]
        elif kind == "rows":
            f[:, :, 1::2] = torch.from_numpy(b).to(s.device)[:, None, None, None]
        total = np.longdouble(N ** 3) * (a if kind == "uniform" else (a.astype(np.longdouble) + b) / 2)
        s.set_f(f)
        got = s.conserved()
        for q in range(5):
            assert abs(got[q] - w[q] @ total) <= TOL * (np.abs(w[q]) @ total), (seed, q)
