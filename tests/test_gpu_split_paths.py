"""The walk of meshes of few cells: the block update's warp list gives the whole walk's bits, and the decisions
are the paired walk's (a batch's walk) one for one."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _mesh(kind):
    from paper_1708_06142_gb300 import inputs
    if kind == "one":
        return inputs.uniform_mesh(8)
    if kind == "cuboid":
        return inputs.uniform_mesh(32, box=(1.0, 2.0, 0.5))
    return inputs.build_mesh(lambda lev, lo, sz: lev < 2 or (lev < 4 and bool(np.all(lo + sz <= 0.5))))


@pytest.mark.parametrize("mac,eta", [("bh", 1.2), ("bh", 3.0), ("ape", 1.2), ("ape", 0.0)])
@pytest.mark.parametrize("kind", ["one", "cuboid", "amr"])
def test_block_update_and_decisions(kind, mac, eta):
    import torch
    from paper_1708_06142_gb300.treesolver import Batch, TreeSolver
    mesh = _mesh(kind)
    assert mesh.nleaf * 16 <= 1216
    rho = np.exp(np.random.default_rng(3).standard_normal(mesh.ncell))
    ts = TreeSolver(0)
    ts.tree_build(mesh, torch.from_numpy(rho).cuda())
    new = lambda dt=torch.float32: (torch.empty(mesh.ncell, dtype=dt, device="cuda"), torch.empty(mesh.ncell, 3, dtype=dt, device="cuda"))
    kw = dict(mac=mac, theta=0.6, safe_box=eta, a_lim=0.05)
    p, a = new()
    ts.gravity_walk(p, a, **kw)
    ts.sync()
    n = ts.stats()["interactions"]
    q, b = new()
    q.zero_()
    b.zero_()
    torch.cuda.synchronize()
    assert ts.gravity_walk_abu(q, b, 0.0, **kw) == mesh.nleaf
    assert torch.equal(p, q) and torch.equal(a, b)
    batch = Batch([ts])
    batch.run(ts.gravity_params(**kw), [q], [b], use_graph=False)
    assert batch.sync()["interactions"] == n
    # the same terms in another order: FP32 rounding of ~8 terms a group, compensated across groups
    assert float((p - q).abs().max()) <= 1e-6 * float(q.abs().max())
    assert float((a - b).abs().max()) <= 2e-6 * float(b.abs().max())
