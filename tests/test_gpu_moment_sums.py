"""Rounding of the FP64 moments, whose sums the kernels take in fixed point.

A cell's 15 values are aligned to the largest and truncated below 2^-58 of it,
summed exactly and rounded once per sum.  So each momentum component, c1 a +
s d with a and d sums over 2 and 8 values, is within s 10 2^-58 max|f| (s >=
c1) plus five roundings of its two products (the sums', s's own, the
product's, the fused add's), and u within that over rho plus three roundings
(rho, its reciprocal, the product).
"""
import numpy as np
import pytest

import oracle
from parity_util import initial_f, sim_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(37, 19, 11), (1, 1, 1), (64, 8, 3)], ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("noise", [0.02, 0.5])
def test_moments_within_the_sums_roundings(shape, noise):
    nx, ny, nz = shape
    cfg = oracle.Cfg(nx=nx, ny=ny, nz=nz, c1=2.0, c2=6.0, eta0=4.0, gamma=1.4, tau=2e-4, dt=2e-4, dx=0.02,
                     bc_lo=(0, 0, 0), bc_hi=(0, 0, 0))
    f = initial_f(cfg, seed=500 + nx, noise=noise)
    s = sim_for(cfg, "fp64")
    s.set_f(f)
    rho, u, _ = s.moments()
    q = np.asarray(f, dtype=np.longdouble)
    v = q.reshape((15,) + rho.shape)
    c1, sq = np.longdouble(cfg.c1), np.longdouble(cfg.c2) / np.sqrt(np.longdouble(3))
    total = v.sum(0)
    largest = np.abs(v).max(0)
    r = np.longdouble(2) ** -53
    assert (np.abs(rho - total) <= 15 * np.longdouble(2) ** -58 * largest + r * np.abs(total)).all()
    signs = np.array([[1, 1, 1, 1, -1, -1, -1, -1], [1, 1, -1, -1, 1, 1, -1, -1], [1, -1, 1, -1, 1, -1, 1, -1]])
    u = np.asarray(u).reshape((3,) + rho.shape)
    for a in range(3):
        axis = v[1 + 2 * a] - v[2 + 2 * a]
        diag = sum(int(signs[a][j]) * v[7 + j] for j in range(8))
        exact = (c1 * axis + sq * diag) / total
        bound = (sq * 10 * np.longdouble(2) ** -58 * largest + 5 * r * (np.abs(c1 * axis) + np.abs(sq * diag))) / total
        bound += np.abs(exact) * (3 * r + 15 * np.longdouble(2) ** -58 * largest / total)
        assert (np.abs(u[a] - exact) <= bound).all(), a
