"""Units in which operands of the FP64 walk's FP32 tests are subnormal or vanish in FP32 (long lengths with
small acceleration limits, masses below the FP32 range, domains of subnormal size): the interaction counts
must still be the FP64 oracle's."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mac,scale,mass,G,eta", [
    ("ape", 1e18, 1e-6, 1.0, 1.2),    # limits around 5e-44: a few bits left in FP32
    ("ape", 1e19, 1e-6, 1.0, 1.2),    # 0 in FP32
    ("ape", 1e20, 1e-9, 1.0, 0.0),
    ("ape", 1.0, 1e-42, 1e30, 1.2),   # node masses down to 1e-48
    ("ape", 1e3, 1e-42, 1e30, 1.2),
    ("ape", 1e10, 1e-20, 1e-20, 1.2),  # G m subnormal
    ("ape", 1.0, 1.0, 1e-42, 1.2),    # G subnormal
    ("ape", 1e-43, 1.0, 1.0, 1.2), ("bh", 1e-43, 1.0, 1.0, 2.6),   # a cell is one step of FP32
    ("ape", 1.0, 0.0, 1.0, 1.2),      # no mass at all
])
def test_counts(oracle, mac, scale, mass, G, eta):
    import torch
    from paper_1708_06142_gb300 import inputs
    from paper_1708_06142_gb300.treesolver import TreeSolver
    refine = lambda lev, lo, sz: lev < 2 or (lev < 4 and bool(np.all(lo < 0.2 * scale)))
    mesh = inputs.build_mesh(refine, box=(scale,) * 3)
    rho = np.exp(np.random.default_rng(7).standard_normal(mesh.ncell)) / scale ** 3 * mass
    a_lim = 3e-2 * G * rho.mean() * scale if mass else 1e-3
    ts = TreeSolver(0)
    ts.tree_build(mesh, torch.from_numpy(rho).cuda())
    pot = torch.empty(mesh.ncell, dtype=torch.float64, device="cuda")
    acc = torch.empty(mesh.ncell, 3, dtype=torch.float64, device="cuda")
    kw = dict(mac=mac, theta=0.6, a_lim=a_lim, G=G, safe_box=eta)
    ts.gravity_walk(pot, acc, precision="fp64", **kw)
    ts.sync()
    p, a, cnt = oracle.gravity_walk(mesh, rho.reshape(-1, 8, 8, 8), **kw)
    assert ts.stats()["interactions"] == cnt["interactions"]
    # ~1000 positive terms of relative rounding 2^-53 each, in another order
    assert np.abs(pot.cpu().numpy() - p).max() <= 1e-13 * np.abs(p).max()
    assert np.abs(acc.cpu().numpy() - a).max() <= 1e-12 * np.abs(a).max()
