"""Meshes of extremely small cells: their squared separations can be subnormal in FP32, so they take
the paired walk that rescales subnormal inputs of the reciprocal square root.  With every length
scaled by a power of two and the masses kept, each FP32 operation of the walk scales exactly, so both
kernels must give the same bits up to that scale."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


# extra 3: more leaf-blocks than the walk for meshes of few cells takes
@pytest.mark.parametrize("mac,extra", [("bh", 0), ("ape", 0), ("mpe", 0), ("bh", 1), ("bh", 3), ("ape", 3)])
def test_small_cells_scale_exactly(mac, extra):
    import torch
    from paper_1708_06142_gb300 import inputs
    from paper_1708_06142_gb300.treesolver import TreeSolver
    k = 34   # box 2^-34: cell edges 2^-38 = 3.6e-12, below the line of 1e-11
    out = []
    for e in (0, k):
        refine = lambda lev, lo, sz: lev < 2 or (extra and lev < 3 + extra - 1 and float(lo.max()) < 2.0 ** (-1 - e))
        mesh = inputs.build_mesh(refine, box=(2.0 ** -e,) * 3)
        rng = np.random.default_rng(5)
        rho = np.exp(0.5 * rng.standard_normal(mesh.ncell)) * 2.0 ** (3 * e)
        ts = TreeSolver(0)
        ts.tree_build(mesh, torch.from_numpy(rho).cuda())
        pot, acc = torch.empty(mesh.ncell, device="cuda"), torch.empty(mesh.ncell, 3, device="cuda")
        ts.gravity_walk(pot, acc, mac=mac, theta=0.6, a_lim=2e-2 * 2.0 ** (2 * e))
        ts.sync()
        out.append((pot.cpu().numpy() * 2.0 ** -e, acc.cpu().numpy() * np.float64(2.0) ** (-2 * e)))
    np.testing.assert_array_equal(out[0][0], out[1][0])
    np.testing.assert_array_equal(out[0][1], out[1][1])


@pytest.mark.parametrize("n_side,nq", [(1, 0), (2, 2)])
def test_small_cells_columns_scale_exactly(n_side, nq):
    """The column walk's bins depend on directions and ratios only, so the maps scale exactly too."""
    import torch
    from paper_1708_06142_gb300 import inputs
    from paper_1708_06142_gb300.treesolver import TreeSolver
    k = 34
    out = []
    for e in (0, k):
        refine = lambda lev, lo, sz: lev < 2 or (lev < 3 and float(lo.max()) < 2.0 ** (-1 - e))
        mesh = inputs.build_mesh(refine, box=(2.0 ** -e,) * 3)
        rng = np.random.default_rng(6)
        rho = np.exp(0.5 * rng.standard_normal((3, mesh.ncell))) * 2.0 ** (3 * e)
        ts = TreeSolver(0)
        ts.tree_build(mesh, torch.from_numpy(rho[0].copy()).cuda())
        if nq:
            ts.column_quantities(torch.from_numpy(rho[1:1 + nq].copy()).cuda())
        cols = torch.empty(mesh.ncell, 1 + nq, 12 * n_side ** 2, device="cuda")
        ts.column_walk(cols, ts.column_params(n_side=n_side, theta=0.6))
        ts.sync()
        out.append(cols.cpu().numpy() * np.float64(2.0) ** (-2 * e))
    np.testing.assert_array_equal(out[0], out[1])
