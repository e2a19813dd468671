"""The block sums of the tree build are formed by whichever block completes a group of siblings: the same
bits on every build, whatever the order, on a chain of refinements and on a broad mesh, against sums in
octant order."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["chain", "broad"])
def test_block_moments(kind):
    import torch
    from paper_1708_06142_gb300 import inputs
    from paper_1708_06142_gb300.treesolver import TreeSolver
    refine = (lambda lev, lo, sz: lev < 14 and bool(np.all(lo == 0.0))) if kind == "chain" else (lambda lev, lo, sz: lev < 5)
    mesh = inputs.build_mesh(refine)
    rho = np.exp(np.random.default_rng(3).standard_normal(mesh.ncell))
    ts = TreeSolver(0)
    d = torch.from_numpy(rho).cuda()
    ts.tree_build(mesh, d)
    mass, com = ts.block_moments(mesh.nblocks)
    for b in range(mesh.nblocks - 1, -1, -1):   # parents precede their children in the list
        ch = mesh.child[b]
        if ch[0] < 0:
            continue
        m, s = 0.0, np.zeros(3)
        for c in ch:
            m += mass[c]
            s += mass[c] * com[c]
        assert mass[b] == m and np.array_equal(com[b], s / m)
    for _ in range(100):
        ts.tree_build(None, d)
        m2, c2 = ts.block_moments(mesh.nblocks)
        assert np.array_equal(m2, mass) and np.array_equal(c2, com)
