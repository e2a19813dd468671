"""A batch's captured graph and the state of its contexts: a replay must follow changes of the contexts
(FP64 records switched on, another mesh of as many cells) that reach the captured tree builds."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _mesh(octant):
    """A root of 8 blocks, one of which is refined: 15 leaf-blocks whichever it is."""
    from paper_1708_06142_gb300 import inputs
    off = np.array([octant & 1, (octant >> 1) & 1, octant >> 2]) * 0.5
    return inputs.build_mesh(lambda lev, lo, sz: lev < 2 or (lev < 3 and bool(np.all(lo == off))))


def _rho(mesh, seed):
    import torch
    return torch.from_numpy(np.exp(np.random.default_rng(seed).standard_normal(mesh.ncell))).cuda()


def _solver(mesh, rho):
    from paper_1708_06142_gb300.treesolver import TreeSolver
    ts = TreeSolver(0)
    ts.tree_build(mesh, rho)
    return ts


def _out(mesh, dtype=None):
    import torch
    dtype = dtype or torch.float32
    return torch.empty(mesh.ncell, dtype=dtype, device="cuda"), torch.empty(mesh.ncell, 3, dtype=dtype, device="cuda")


@pytest.mark.parametrize("mode", [0, 1])
def test_replay_writes_fp64_records_switched_on_after_the_capture(mode):
    import torch
    from paper_1708_06142_gb300.treesolver import Batch
    mesh = _mesh(0)
    rho, rho2 = _rho(mesh, 1), _rho(mesh, 2)
    ts = _solver(mesh, rho)
    ts.fp64_records(False)
    b = Batch([ts])
    b.set_mode(mode, 2)
    gp = ts.gravity_params(theta=0.5)
    p, a = _out(mesh)
    b.run(gp, [p], [a], densities=[rho])
    b.sync()
    ts.fp64_records(True)
    ts.tree_build(None, rho)
    ts.sync()
    rho.copy_(rho2)
    torch.cuda.synchronize()
    b.run(gp, [p], [a], densities=[rho])
    b.sync()
    p64, a64 = _out(mesh, torch.float64)
    ts.gravity_walk(p64, a64, precision="fp64")
    ts.sync()
    ref = _solver(mesh, rho2)
    q64, b64 = _out(mesh, torch.float64)
    ref.gravity_walk(q64, b64, precision="fp64")
    ref.sync()
    assert torch.equal(p64, q64) and torch.equal(a64, b64)


@pytest.mark.parametrize("mode", [0, 1])
def test_replay_follows_another_mesh_of_as_many_cells(mode):
    import torch
    from paper_1708_06142_gb300.treesolver import Batch
    m0, m1 = _mesh(0), _mesh(5)
    assert m0.ncell == m1.ncell
    rho = _rho(m0, 3)
    solvers = [_solver(m0, rho), _solver(m0, rho)]
    gp = solvers[0].gravity_params(theta=0.5, zero_mean=True)
    outs = [_out(m0), _out(m0)]
    b = Batch(solvers)
    b.set_mode(mode, 2)
    run = lambda bb, oo, g: bb.run(gp, [o[0] for o in oo], [o[1] for o in oo], densities=[rho, rho], use_graph=g)
    run(b, outs, True)
    b.sync()
    solvers[1].tree_build(m1, rho)
    solvers[1].sync()
    for _ in range(2):   # a new capture, its replay
        run(b, outs, True)
        b.sync()
    fresh = [_solver(m0, rho), _solver(m1, rho)]
    c = Batch(fresh)
    c.set_mode(mode, 2)
    want = [_out(m0), _out(m1)]
    run(c, want, False)
    c.sync()
    for o, w in zip(outs, want):
        # (the FP64 mean is summed in no fixed order: one FP32 rounding of the potential before the shift)
        assert float((o[0] - w[0]).abs().max()) <= 2.0 ** -22 * float(w[0].abs().max())
        assert torch.equal(o[1], w[1])


def test_mpe_walk_and_quantities_after_a_run_with_new_densities():
    import torch
    from paper_1708_06142_gb300.treesolver import Batch
    mesh = _mesh(0)
    rho, rho2 = _rho(mesh, 4), _rho(mesh, 5)
    ts = _solver(mesh, rho)
    kw = dict(mac="mpe", a_lim=0.05)
    p, a = _out(mesh)
    ts.gravity_walk(p, a, **kw)              # moments of the first density
    ts.column_quantities(torch.stack([rho, rho]))
    gp = ts.gravity_params(theta=0.5)
    b = Batch([ts])
    for g in (False, True, True):            # direct, captured, replayed
        rho.copy_(_rho(mesh, 6) if g else rho2)
        torch.cuda.synchronize()
        b.run(gp, [p], [a], densities=[rho], use_graph=g)
        b.sync()
        ts.gravity_walk(p, a, **kw)
        cols = torch.empty(mesh.ncell, 48, device="cuda")
        ts.column_walk(cols)
        ts.sync()
        ref = _solver(mesh, rho)
        q, c = _out(mesh)
        ref.gravity_walk(q, c, **kw)
        want = torch.empty(mesh.ncell, 48, device="cuda")
        ref.column_walk(want)
        ref.sync()
        assert torch.equal(p, q) and torch.equal(a, c) and torch.equal(cols, want)


@pytest.mark.parametrize("mac", ["bh", "ape"])
def test_both_forms_give_the_same_bits(mac):
    import torch
    from paper_1708_06142_gb300 import inputs
    from paper_1708_06142_gb300.treesolver import Batch
    meshes = [inputs.uniform_mesh(n, bc=bc) for n, bc in ((8, (0, 0, 0)), (32, (0, 0, 0)), (16, (1, 1, 1)), (16, (0, 0, 0)))]
    rhos = [_rho(m, k) for k, m in enumerate(meshes)]
    solvers = [_solver(m, r) for m, r in zip(meshes, rhos)]
    solvers[2].ewald_field(16)
    gp = solvers[0].gravity_params(mac=mac, theta=0.5, a_lim=0.05)
    cp = solvers[0].column_params(n_side=1)
    out = []
    for mode in (0, 1):
        b = Batch(solvers)
        b.set_mode(mode, 3)
        pots, accs = zip(*[_out(m) for m in meshes])
        cols = [torch.empty(m.ncell, 12, device="cuda") for m in meshes]
        b.run(gp, pots, accs, cp, cols, densities=rhos, use_graph=False)
        b.sync()
        out.append((*pots, *accs, *cols))
    for x, y in zip(*out):
        assert torch.equal(x, y)
