"""Rounding of one interaction of the FP64 isolated walk: with a single massive cell every target's potential
and acceleration are one term each, m / d and m d / |d|^3, compared with 50-digit arithmetic on the
same FP64 separations; once with an opening angle so small that all leaf cells interact one by one, once with
an ordinary one, where few lanes share a leaf-cell group and nodes stand for the cell."""
from decimal import Decimal, getcontext

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("theta,unit_mass,at,seed", [(1e-6, False, 1234, 0), (1e-6, False, 3, 1), (0.5, True, 2777, 2),
                                                     (0.9, True, 40, 3)])
def test_one_interaction(theta, unit_mass, at, seed):
    import torch
    from paper_1708_06142_gb300 import inputs
    from paper_1708_06142_gb300.treesolver import TreeSolver
    getcontext().prec = 50
    rng = np.random.default_rng(seed)
    mesh = inputs.uniform_mesh(16, box=tuple(rng.uniform(0.5, 2.0, 3)))
    lf = mesh.leaves
    e = mesh.size[lf] / 8
    dv = float((e[:, 0] * e[:, 1] * e[:, 2])[at // 512])
    rho = np.zeros(mesh.ncell)
    rho[at] = rng.uniform(0.5, 2.0)
    if unit_mass:   # mass 1: the centre of mass of every node that holds the cell is the cell's centre exactly
        r = 1.0 / dv
        rho[at] = next(x for x in (r, np.nextafter(r, 0), np.nextafter(r, np.inf)) if x * dv == 1.0)
    m = rho[at] * dv
    # cell centres as FP64 forms them: lo + ((i + 1/2) size) / 8
    c = (np.arange(8) + 0.5)
    ax = [mesh.lo[lf, a, None] + (c * mesh.size[lf, a, None]) * 0.125 for a in range(3)]
    pos = np.empty((len(lf), 8, 8, 8, 3))
    pos[..., 0], pos[..., 1], pos[..., 2] = ax[0][:, None, None, :], ax[1][:, None, :, None], ax[2][:, :, None, None]
    pos = pos.reshape(-1, 3)
    ts = TreeSolver(0)
    ts.tree_build(mesh, torch.from_numpy(rho).cuda())
    pot = torch.empty(mesh.ncell, dtype=torch.float64, device="cuda")
    acc = torch.empty(mesh.ncell, 3, dtype=torch.float64, device="cuda")
    ts.gravity_walk(pot, acc, theta=theta, precision="fp64")
    ts.sync()
    p, a = pot.cpu().numpy(), acc.cpu().numpy()
    assert p[at] == 0.0 and not a[at].any()
    u = Decimal(2) ** -53
    mm = Decimal(float(m))
    worst_p = worst_a = Decimal(0)
    for i in rng.choice(np.delete(np.arange(mesh.ncell), at), 1500, replace=False):
        d = [Decimal(float(pos[at, k] - pos[i, k])) for k in range(3)]
        d2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
        inv = 1 / d2.sqrt()
        worst_p = max(worst_p, abs(Decimal(float(p[i])) / (-mm * inv) - 1))
        g3 = mm * inv / d2
        for k in range(3):
            if d[k]:
                worst_a = max(worst_a, abs(Decimal(float(a[i, k])) / (g3 * d[k]) - 1))
            else:
                assert a[i, k] == 0.0
    # m / d and m / d^3: the rounding and 7.5 2^-60 from truncated products (1.06 u); the acceleration is one more rounding (u)
    assert worst_p <= Decimal("1.1") * u, worst_p / u
    assert worst_a <= Decimal("2.1") * u, worst_a / u


def test_sums(oracle):
    import torch
    from paper_1708_06142_gb300 import inputs
    from paper_1708_06142_gb300.treesolver import TreeSolver
    mesh = inputs.build_mesh(lambda lev, lo, sz: lev < 2 or (lev < 4 and bool(np.all(lo < 0.2))))
    rho = np.exp(np.random.default_rng(7).standard_normal(mesh.ncell))
    ts = TreeSolver(0)
    ts.tree_build(mesh, torch.from_numpy(rho).cuda())
    pot = torch.empty(mesh.ncell, dtype=torch.float64, device="cuda")
    acc = torch.empty(mesh.ncell, 3, dtype=torch.float64, device="cuda")
    for kw in (dict(mac="bh", theta=0.6), dict(mac="ape", a_lim=0.03 * rho.mean())):
        ts.gravity_walk(pot, acc, precision="fp64", **kw)
        ts.sync()
        p, a, _ = oracle.gravity_walk(mesh, rho.reshape(-1, 8, 8, 8), **kw)
        # ~1000 terms of one sign (potential), each and each partial sum within 2^-53: sqrt(1000) 2^-53 twice
        assert np.abs(pot.cpu().numpy() - p).max() <= 8e-15 * np.abs(p).max()
        assert np.abs(acc.cpu().numpy() - a).max() <= 8e-15 * np.abs(a).max()
