"""The FP64 step keeps its bits beside a neighbour of any size.

In a NND gradient the second upwind value and the downwind one only bound the
limited differences; in the upwind schemes the downwind one (and for the first
order the second upwind one too) does not enter at all.  So the update of a
velocity does not depend on how large such a value is once it is past the
bound: with one cell's populations scaled by a factor, every value for which
that cell takes only these places is bitwise the one with the factor 4 of the
same sign (at which no kernel form has to drop bits of the others).
"""
import numpy as np
import pytest

import oracle
from parity_util import initial_f, sim_for

pytestmark = pytest.mark.gpu

SIGNS = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)] + \
        [(a, b, c) for a in (1, -1) for b in (1, -1) for c in (1, -1)]
# the three splits of the kernel: one velocity pair per block, three parts, whole rows
GRIDS = [(40, 12, 9), (40, 20, 20), (64, 48, 60)]


def _free_cells(f, factor, scheme, dissipation, i, p):
    """Cells whose update of velocity i has cell p (scaled by `factor`) only
    where it is not added, and past the bound of the limited difference."""
    shape = np.array(f.shape[:0:-1])

    def at(c):
        return f[(i,) + tuple((c % shape)[::-1])]

    out = []
    big = factor * at(p)
    for a in range(3):
        s = SIGNS[i][a]
        e = np.eye(3, dtype=int)[a]
        if s == 0:
            if i > 0 and not dissipation:
                out += [p + e, p - e]
            continue
        down, up2 = p - s * e, p + 2 * s * e  # p is the downwind, the second upwind value of these
        for t, use, x, way in ((down, i > 6 or not dissipation, big - at(down), big),
                               (up2, scheme != oracle.UPWIND2, at(up2 - s * e) - big, -big)):
            d = at(t) - at(t - s * e)
            limited = scheme != oracle.NND or (x * way > 0 and (abs(x) >= abs(d) or x * d < 0))
            if use and limited:
                out.append(t)
    return out


@pytest.mark.parametrize("scheme", [oracle.NND, oracle.UPWIND2, oracle.UPWIND1])
@pytest.mark.parametrize("dissipation", [1, 0])
@pytest.mark.parametrize("n", GRIDS)
def test_a_large_neighbour_that_is_not_added(n, dissipation, scheme):
    cfg = oracle.Cfg(nx=n[0], ny=n[1], nz=n[2], c1=2.0, c2=6.0, eta0=4.0, gamma=1.4, tau=5e-4, dt=2e-4, dx=0.02,
                     scheme=scheme, dissipation=dissipation)
    f0 = initial_f(cfg, seed=30)
    cells = [np.array(p) for p in ((5, 4, 4), (17, 6, 3), (38, 1, 5), (0, 9, 0))]  # the last two wrap

    def step(factor):
        f = f0.copy().reshape(15, n[2], n[1], n[0])
        for p in cells:
            f[:, p[2], p[1], p[0]] *= factor
        s = sim_for(cfg, "fp64")
        s.set_f(f)
        s.step(1)
        return s.get_f().reshape(15, n[2], n[1], n[0])

    f0v = f0.reshape(15, n[2], n[1], n[0])
    for sign in (1.0, -1.0):
        base = step(4.0 * sign)
        free = [(i,) + tuple((t % np.array(n))[::-1]) for i in range(1, 15) for p in cells
                for t in _free_cells(f0v, 4.0 * sign, scheme, dissipation, i, p)]
        assert len(free) >= 20 * len(cells)
        for factor in (64.0, 1e2, 1.1e3, 1e5, 3e7, 1e15, 1e30, 1e290, np.inf):
            got = step(factor * sign)
            for at in free:
                assert got[at] == base[at], (factor * sign, at)
