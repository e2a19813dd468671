"""The walk of meshes of few cells (8 targets per warp) against the paired walk's decisions: interaction
counts equal the FP64 oracle's up to FP32 ties, results agree with the FP64 walk, and ranges and block
updates give the whole walk's bits; at the smallest mesh, on either side of the rule's line, and with
both MACs and a safe box that matters."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _mesh(kind):
    from paper_1708_06142_gb300 import inputs
    if kind == "one":
        return inputs.uniform_mesh(8)
    if kind == "cuboid":
        return inputs.uniform_mesh(16, box=(1.0, 2.0, 0.5))
    limit = {"below": 0.47, "above": 0.53}[kind]   # leaf-blocks on either side of 1216 / 16 = 76
    return inputs.build_mesh(lambda lev, lo, sz: lev < 3 or (lev < 4 and bool(np.all(lo + sz <= limit)) and lo[2] < 0.2))


@pytest.mark.parametrize("mac,rel,eta", [("bh", False, 1.2), ("bh", False, 3.0), ("ape", False, 1.2), ("ape", True, 0.0)])
@pytest.mark.parametrize("kind", ["one", "cuboid", "below", "above"])
def test_few_cells(kind, mac, rel, eta):
    import torch
    from paper_1708_06142_gb300.treesolver import TreeSolver
    mesh = _mesh(kind)
    rng = np.random.default_rng(3)
    rho = np.exp(rng.standard_normal(mesh.ncell))
    ts = TreeSolver(0)
    ts.tree_build(mesh, torch.from_numpy(rho).cuda())
    new = lambda dt: (torch.empty(mesh.ncell, dtype=dt, device="cuda"), torch.empty(mesh.ncell, 3, dtype=dt, device="cuda"))
    a_old = torch.from_numpy(np.exp(0.3 * rng.standard_normal(mesh.ncell)).astype(np.float32)).cuda() if rel else None
    kw = dict(mac=mac, theta=0.6, safe_box=eta, a_lim=0.0 if rel else 0.05, a_old=a_old, eps_rel=0.05 if rel else 0.0)
    p, a = new(torch.float32)
    ts.gravity_walk(p, a, **kw)
    ts.sync()
    n32 = ts.stats()["interactions"]
    p64, a64 = new(torch.float64)
    ts.gravity_walk(p64, a64, precision="fp64", **kw)
    ts.sync()
    # a decision within FP32 rounding of its limit may differ from the FP64 one: a few in a million
    assert abs(n32 - ts.stats()["interactions"]) <= 1e-5 * n32 + 200
    # FP32 coordinates and interactions (a few 2^-24 each) summed over ~500 terms
    assert np.quantile((a.double() - a64).abs().max(1).values.cpu().numpy(), 0.99) <= 5e-6 * float(a64.abs().max())
    assert np.quantile((p.double() - p64).abs().cpu().numpy(), 0.99) <= 5e-6 * float(p64.abs().max())
    # ranges and the block update run the kernel of the whole walk
    q, b = new(torch.float32)
    n = mesh.nleaf
    for lo, hi in ((0, n // 3), (n // 3, n)):
        ts.gravity_walk_range(q, b, lo, hi, **kw)
    ts.sync()
    assert torch.equal(p, q) and torch.equal(a, b)
    assert ts.walk_block_counts().sum() == n32
    assert ts.gravity_walk_abu(q, b, 1e-30, **kw) == 0 and torch.equal(a, b)
