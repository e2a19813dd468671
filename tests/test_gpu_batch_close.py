"""Batches and their solvers closed or collected in any order."""
import gc

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _pair():
    import torch
    from paper_1708_06142_gb300 import inputs
    from paper_1708_06142_gb300.treesolver import Batch, TreeSolver
    mesh = inputs.uniform_mesh(8)
    rho = torch.ones(mesh.ncell, dtype=torch.float64, device="cuda")
    solvers = [TreeSolver(0), TreeSolver(0)]
    for s in solvers:
        s.tree_build(mesh, rho)
        s.sync()
    b = Batch(solvers)
    outs = [(torch.empty(mesh.ncell, device="cuda"), torch.empty(mesh.ncell, 3, device="cuda")) for _ in solvers]
    run = lambda: b.run(solvers[0].gravity_params(), [o[0] for o in outs], [o[1] for o in outs], densities=[rho, rho])
    run()
    b.sync()
    return solvers, b, run


@pytest.mark.parametrize("first", [0, 1])
def test_solver_closed_before_its_batch(first):
    from paper_1708_06142_gb300.treesolver import TSError
    solvers, b, run = _pair()
    solvers[first].close()
    with pytest.raises(TSError) as e:
        run()
    assert e.value.status == 1
    with pytest.raises(TSError):
        b.sync()
    b.close()
    solvers[1 - first].close()


def test_collected_in_a_cycle():
    for _ in range(3):
        solvers, b, _ = _pair()
        ring = [solvers, b]
        ring.append(ring)
        del solvers, b, ring, _
        gc.collect()


def test_batch_closed_first():
    solvers, b, _ = _pair()
    b.close()
    assert all(not s._batches for s in solvers)
    solvers[0].close()
    solvers[1].close()
