"""rho, u and T of cells whose populations differ by orders of magnitude.

Each sum of the moments is taken in fixed point on the scale of its own
values: a value is truncated below 2^-58 of the largest in its sum, and a sum
loses up to one such unit where it is brought to the scale of another.  So a
momentum component is within 2 and 8 of its pair's and the diagonal values'
units (times c1 and s), and not of the largest population's, which would be
more than the bound here from a contrast of about 1e3 on.  Roundings are
counted as 2^-53 of their operands.
"""
import numpy as np
import pytest

import oracle
from parity_util import sim_for

pytestmark = pytest.mark.gpu

Q = np.longdouble
N = (37, 9, 5)
SIGNS = np.array([[0, 0, 0], [1, 0, 0], [-1, 0, 0], [0, 1, 0], [0, -1, 0], [0, 0, 1], [0, 0, -1]] +
                 [[a, b, c] for a in (1, -1) for b in (1, -1) for c in (1, -1)])
GROUPS = {"rest": [0], "axes": list(range(1, 7)), "one_axis": [1, 2], "one_value": [4], "diagonals": list(range(7, 15)),
          "one_diagonal": [12], "none": []}


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("contrast", [1e-6, 1e2, 1e3, 1e5, 1e9, 1e15])
@pytest.mark.parametrize("group", sorted(GROUPS))
def test_moments_of_unequal_populations(group, contrast, precision):
    cfg = oracle.Cfg(nx=N[0], ny=N[1], nz=N[2], c1=2.0, c2=6.0, eta0=4.0, gamma=1.4, tau=2e-4, dt=2e-4, dx=0.02,
                     bc_lo=(0, 0, 0), bc_hi=(0, 0, 0))
    f = np.random.default_rng(17).uniform(0.5, 1.5, (15, N[2], N[1], N[0]))
    f[GROUPS[group]] *= contrast
    if precision == "fp32":
        f = f.astype(np.float32)
    s = sim_for(cfg, precision)
    s.set_f(f)
    rho, u, T = s.moments()

    q = f.astype(Q)
    r, unit = Q(2) ** -53, Q(2) ** -58
    c1, sq = Q(2), Q(6) / np.sqrt(Q(3))
    axes, diag = q[1:7].max(0), q[7:].max(0)
    rho_x = q.sum(0)
    rho_b = 20 * unit * q.max(0) + r * rho_x
    assert (np.abs(rho - rho_x) <= rho_b).all()
    u_x, u_b = [], []
    for a in range(3):
        pair = c1 * (q[1 + 2 * a] - q[2 + 2 * a])
        cross = sq * np.tensordot(SIGNS[7:, a].astype(Q), q[7:], 1)
        p_b = c1 * 2 * unit * np.maximum(q[1 + 2 * a], q[2 + 2 * a]) + sq * 8 * unit * diag \
            + 5 * r * (np.abs(pair) + np.abs(cross))
        u_x.append((pair + cross) / rho_x)
        u_b.append((p_b + np.abs(pair + cross) * (3 * r + rho_b / rho_x)) / rho_x)
        assert (np.abs(u[a] - u_x[a]) <= u_b[a]).all(), a
    parts = [Q(16) * q[0], c1 * c1 * q[1:7].sum(0), Q(36) * q[7:].sum(0)]
    energy = sum(parts)
    e_b = c1 * c1 * 9 * unit * axes + Q(36) * 8 * unit * diag + Q(16) * unit * q.max(0) + 4 * r * energy
    usq = sum(v * v for v in u_x)
    T_x = (energy / rho_x - usq) / 5
    T_b = ((e_b + energy * (3 * r + rho_b / rho_x)) / rho_x + 2 * sum(np.abs(v) * b for v, b in zip(u_x, u_b))
           + 4 * r * usq) / 5 + 4 * r * np.abs(T_x)
    assert (np.abs(T - T_x) <= T_b).all()
