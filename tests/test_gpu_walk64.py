"""The FP64 isolated walk decides MAC and safe-box tests in FP32 outside a guard band and in FP64 inside
it: interaction counts must equal the FP64 oracle's exactly and the sums agree to FP64 rounding, also
where FP32 cannot decide anything (boxes far from the origin, far outside the FP32 range), where masses
vanish or have both signs, and for boxes that put targets exactly on a safe box's faces."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mac,scale,origin,eta,mass", [
    ("bh", 1.0, 0.0, 1.2, "pos"), ("bh", 1.0, 3e4, 1.2, "pos"), ("bh", 1.0, -0.5, 0.0, "pos"),
    ("bh", 1e-25, 0.0, 1.2, "pos"), ("bh", 1e25, 0.0, 2.6, "pos"), ("bh", 1e45, 0.0, 1.2, "pos"),
    ("bh", 1.0, 0.0, 1.25, "signed"), ("ape", 1.0, 0.0, 1.25, "pos"), ("ape", 1.0, 3e4, 1.2, "pos"),
    ("ape", 1.0, 0.0, 1.2, "zero"), ("ape", 1e-25, 0.0, 1.2, "pos"), ("ape", 1e25, -1e25, 1.2, "pos"),
    ("ape", 1.0, 0.0, 1.2, "signed"),
])
def test_fp64_decisions(oracle, mac, scale, origin, eta, mass):
    import torch
    from paper_1708_06142_gb300 import inputs
    from paper_1708_06142_gb300.treesolver import TreeSolver
    refine = lambda lev, lo, sz: lev < 2 or (lev < 4 and bool(np.all(lo - origin < 0.2 * scale)))
    mesh = inputs.build_mesh(refine, box=(scale,) * 3, origin=(origin,) * 3)
    rng = np.random.default_rng(7)
    rho = np.exp(rng.standard_normal(mesh.ncell)) / scale ** 3
    if mass == "zero":
        rho[rng.random(mesh.ncell // 512).repeat(512) < 0.5] = 0.0
    if mass == "signed":
        rho = np.where(rng.random(mesh.ncell) < 0.3, -0.5 * rho, rho)
    a_lim = 3e-2 * abs(rho.mean()) * scale
    ts = TreeSolver(0)
    ts.tree_build(mesh, torch.from_numpy(rho).cuda())
    pot = torch.empty(mesh.ncell, dtype=torch.float64, device="cuda")
    acc = torch.empty(mesh.ncell, 3, dtype=torch.float64, device="cuda")
    ts.gravity_walk(pot, acc, mac=mac, theta=0.6, a_lim=a_lim, safe_box=eta, precision="fp64")
    ts.sync()
    st = ts.stats()
    p, a, cnt = oracle.gravity_walk(mesh, rho.reshape(-1, 8, 8, 8), mac=mac, theta=0.6, a_lim=a_lim, safe_box=eta)
    assert st["interactions"] == cnt["interactions"]
    # ~1000 terms of relative rounding 2^-53 each, summed in another order; terms of both signs cancel by
    # two digits at most
    assert np.abs(pot.cpu().numpy() - p).max() <= 1e-11 * np.abs(p).max()
    assert np.abs(acc.cpu().numpy() - a).max() <= 1e-11 * np.abs(a).max()
