"""The paired periodic walk (one target per lane) against the scalar walk that shares its tables and
against the FP64 walk, at the edges of its lookup: smallest, odd and largest tables, cuboid boxes, every
supported mix of boundaries, adaptive meshes, and masses of both signs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _walk(ts, ncell, fp64=False, **kw):
    import torch
    dt = torch.float64 if fp64 else torch.float32
    pot, acc = torch.empty(ncell, dtype=dt, device="cuda"), torch.empty(ncell, 3, dtype=dt, device="cuda")
    ts.gravity_walk(pot, acc, precision="fp64" if fp64 else "fp32", **kw)
    ts.sync()
    return pot.cpu().numpy().astype(np.float64), acc.cpu().numpy().astype(np.float64)


@pytest.mark.parametrize("ewald", ["table", "taylor"])
@pytest.mark.parametrize("bc,box,ntab,mac,signed", [
    ((1, 1, 1), (1.0, 1.0, 1.0), 8, "bh", False),
    ((1, 1, 1), (0.7, 0.9, 1.3), 33, "ape", False),
    ((1, 1, 1), (3.0, 3.0, 3.0), 256, "bh", False),
    ((1, 1, 0), (1.0, 1.3, 4.0), 31, "bh", False),
    ((1, 1, 0), (1.0, 1.0, 0.5), 64, "mpe", False),
    ((1, 0, 0), (1.0, 0.8, 1.1), 16, "bh", False),
    ((1, 1, 1), (1.0, 1.0, 1.0), 64, "bh", True),
])
def test_paired_lookup(ewald, bc, box, ntab, mac, signed):
    import torch
    from paper_1708_06142_gb300 import inputs
    from paper_1708_06142_gb300.treesolver import TreeSolver
    # three levels with one refined corner: both cells and nodes of several depths
    refine = lambda lev, lo, sz: lev < 2 or (lev < 3 and bool(np.all(lo < 0.25 * np.array(box))))
    mesh = inputs.build_mesh(refine, box=box, bc=bc)
    rng = np.random.default_rng(11)
    rho = np.exp(rng.standard_normal(mesh.ncell))
    if signed:   # mostly positive: some nodes' centres of mass leave their cells
        rho = np.where(rng.random(mesh.ncell) < 0.3, -0.5 * rho, rho)
    ts = TreeSolver(0)
    ts.tree_build(mesh, torch.from_numpy(rho).cuda())
    ts.ewald_field(ntab)
    vol = float(np.prod(box))
    kw = dict(mac=mac, theta=0.55, a_lim=3e-2 * rho.mean() * vol ** (1.0 / 3.0), ewald=ewald)
    p1, a1 = _walk(ts, mesh.ncell, **kw)
    p2, a2 = _walk(ts, mesh.ncell, fp64=True, **kw)
    # FP32 coordinates and table entries carry relative errors of a few 2^-24, and ~500 terms are summed.
    # Against the FP64 walk the bulk is held: a node within rounding of its acceptance limit or of a
    # grid-point tie may be decided otherwise in a few cells.
    sa, sp = np.abs(a2).max(), np.abs(p2 - p2.mean()).max()
    ea, ep = np.abs(a1 - a2).max(1) / sa, np.abs(p1 - p2) / max(sp, 1e-2 * np.abs(p2).max())
    assert np.quantile(ea, 0.98) < 2e-5
    assert np.quantile(ep, 0.98) < 2e-5
    if mac != "mpe":   # the scalar walk of two targets per lane: the same decisions, so every cell agrees
        ts.set_walk_grouping("fp32", 2)
        p3, a3 = _walk(ts, mesh.ncell, **kw)
        assert (np.abs(a1 - a3).max(1) / sa).max() < 2e-5
        assert (np.abs(p1 - p3) / max(sp, 1e-2 * np.abs(p2).max())).max() < 2e-5
