"""Walks captured into a caller's graph: the first walk after a mesh is ingested must not leave a part of its
set-up to the graph alone."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_walk_before_the_first_replay_of_a_captured_one():
    import torch
    from paper_1708_06142_gb300 import inputs
    from paper_1708_06142_gb300.treesolver import TreeSolver
    st = torch.cuda.Stream()
    ts = TreeSolver(0, st)
    out = lambda m: (torch.empty(m.ncell, device="cuda"), torch.empty(m.ncell, 3, device="cuda"))
    m0, m1 = inputs.uniform_mesh(16), inputs.uniform_mesh(16, box=(2.0, 1.0, 4.0))
    rho = torch.from_numpy(np.exp(np.random.default_rng(2).standard_normal(m0.ncell))).cuda()
    torch.cuda.synchronize()
    p, a = out(m0)
    ts.tree_build(m0, rho)
    ts.gravity_walk(p, a)
    ts.sync()
    ts.tree_build(m1, rho)
    g = torch.cuda.CUDAGraph()
    q, b = out(m1)
    with torch.cuda.graph(g, stream=st):
        ts.gravity_walk(q, b)
    ts.gravity_walk(p, a)      # directly, before any replay
    ts.sync()
    ref = TreeSolver(0)
    ref.tree_build(m1, rho)
    r, c = out(m1)
    ref.gravity_walk(r, c)
    ref.sync()
    assert torch.equal(p, r) and torch.equal(a, c)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(q, r) and torch.equal(b, c)
