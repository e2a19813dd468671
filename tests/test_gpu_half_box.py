"""Minimum images of separations of exactly half a period: in boxes whose 1 / L is not exact in FP32 the
paired walks must pick the image that the scalar walk and the FP64 oracle pick.  A small opening angle
makes cells half a box apart interact one by one."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

BOXES = [(1.0, 1.0, 1.0), (0.75, 0.75, 0.75), (0.1, 1.0, 1.0), (1.3, 0.7, 0.9)]


def _case(box):
    import torch
    from paper_1708_06142_gb300 import inputs
    from paper_1708_06142_gb300.treesolver import TreeSolver
    mesh = inputs.uniform_mesh(16, box=box, bc=(1, 1, 1))
    rho = np.exp(np.random.default_rng(5).standard_normal(mesh.ncell))
    ts = TreeSolver(0)
    ts.tree_build(mesh, torch.from_numpy(rho).cuda())
    return mesh, rho, ts


@pytest.mark.parametrize("ewald", ["table", "taylor"])
@pytest.mark.parametrize("box", BOXES)
def test_gravity(box, ewald):
    import torch
    mesh, _, ts = _case(box)
    ts.ewald_field(32)
    out = []
    for t in (1, 2):   # paired, scalar
        ts.set_walk_grouping("fp32", t)
        p, a = torch.empty(mesh.ncell, device="cuda"), torch.empty(mesh.ncell, 3, device="cuda")
        ts.gravity_walk(p, a, theta=0.2, ewald=ewald)
        ts.sync()
        out.append(a)
    # the same terms, a few 2^-24 apart each, ~3000 of them
    assert float((out[0] - out[1]).abs().max()) <= 2e-6 * float(out[1].abs().max())


# (not the last box: its half periods are no FP32 numbers, so which side of a tie a pair falls on depends on how
# its coordinates round, in FP32 and in FP64)
@pytest.mark.parametrize("box", BOXES[:3])
def test_columns(oracle, box):
    import torch
    mesh, rho, ts = _case(box)
    cols = torch.empty(mesh.ncell, 48, device="cuda")
    ts.column_walk(cols, n_side=2, theta=0.2)
    ts.sync()
    tg = np.arange(0, mesh.ncell, 29)
    ref, _ = oracle.column_walk(mesh, rho.reshape(-1, 8, 8, 8), tg, nside=2, theta=0.2)
    rel = np.abs(cols.cpu().numpy().astype(np.float64)[tg] - ref) / ref
    # column tolerance 1e-4; a direction within rounding of a bin's edge may fall on the other side
    assert (rel > 1e-4).mean() < 1e-3
