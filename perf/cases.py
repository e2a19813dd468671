"""Performance cases of the tree solver: what a user's program calls, over the sizes it calls it with.

A simulation calls the solver once per time step with a new density on a mesh it ingested earlier, so
a pass is `tree_build(None, density)` followed by the walk of the step: gravity (isolated, fully
periodic or x,y-periodic boxes; BH, APE or MPE acceptance; FP32 or FP64; trilinear, Taylor or learned
correction), column densities (with or without the H2 and CO maps and their shielding averages), or
both for a batch of independent grids.  Meshes are the uniform and the adaptive block octrees of
`paper_1708_06142_gb300.inputs`; densities are seeded and made on the GPU.

`exact` repeats a pass in 64 bits with plain torch: moments, walk, Ewald series and its lookup,
node-ray table and maps are written out here from their definitions.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1708_06142_gb300 import inputs
from paper_1708_06142_gb300.treesolver import Batch, TreeSolver

DEV = "cuda:0"
NTAB = 64          # correction-table points per axis (the library's default)
PLUMMER_A = 0.05   # Plummer radius of the adaptive meshes
NET = 8900         # parameters of the 4-64-64-64-4 network
NET_B = (0.5, 2.0)  # aspect range of the network
CO_TAB = (40, 40)  # CO shielding table points


def _grav(name, mesh, n, density, bc="iso", theta=0.5, mac="bh", limit=0.0, precision="fp32", ewald="table",
          by=1.0, bz=1.0, thresh=0.0):
    return dict(name=name, kind="gravity", mesh=mesh, n=n, thresh=thresh, density=density, bc=bc, by=by, bz=bz, mac=mac,
                theta=theta, limit=limit, precision=precision, ewald=ewald)


def _cols(name, n, density, bc, n_side, theta, species):
    return dict(name=name, kind="columns", mesh="uniform", n=n, thresh=0.0, density=density, bc=bc, by=1.0, bz=1.0,
                n_side=n_side, theta=theta, species=species)


def _batch(name, count, base, mode, ewald, n_side):
    return dict(name=name, kind="batch", count=count, base=base, mode=mode, ewald=ewald, n_side=n_side, theta=0.5)


def listed():
    return [
        # the smallest grid anybody runs, a 32^3 test sphere: launches and latency
        _grav("sphere32", "uniform", 32, "sphere"),
        # collapsing core on an adaptive mesh of 4096 blocks, the benchmark's step
        _grav("plummer2m", "amr", 6, "plummer", thresh=0.0013),
        # the same mesh with the error-bounded MPE criterion
        _grav("plummer2m_mpe", "amr", 6, "plummer", thresh=0.0013, mac="mpe", limit=1e-2),
        # a coarser adaptive mesh with the APE criterion relative to the last step's acceleration
        _grav("plummer_ape_rel", "amr", 5, "plummer", thresh=0.0013, mac="ape_rel", limit=1e-2),
        # the paper's own precision, for a run that wants it throughout
        _grav("plummer_fp64", "amr", 5, "plummer", thresh=0.0013, precision="fp64"),
        # turbulence in a periodic box with the fast lookup
        _grav("turbulent128_taylor", "uniform", 128, "turbulent", bc="3p", ewald="taylor"),
        # the same physics at 64^3 with the default lookup
        _grav("turbulent64_table", "uniform", 64, "turbulent", bc="3p"),
        # stratified disk, periodic in the plane, elongated box and cells
        _grav("disk64_taylor", "uniform", 64, "disk", bc="2p1i", bz=4.0, ewald="taylor"),
        # the same disk with the learned correction, small as that lookup is the dearest
        _grav("disk32_learned", "uniform", 32, "disk", bc="2p1i", bz=4.0, ewald="mlp"),
        # optical depths of a turbulent periodic box, 48 directions
        _cols("columns128", 128, "turbulent", "3p", 2, 0.5, False),
        # the same with H2 and CO maps and the shielding averages the chemistry takes, isolated cloud
        _cols("columns64_species", 64, "plummer", "iso", 2, 0.5, True),
        # a sweep of independent boxes, gravity and columns in one graph
        _batch("batch9", 9, 32, 1, "taylor", 2),
    ]


def draw(rng):
    r = rng.random()
    theta = round(rng.uniform(0.4, 0.8), 3)
    if r < 0.40:   # isolated gravity, FP32 or (smaller) FP64
        fp64 = rng.random() < 0.25
        mac = rng.choice(["bh", "bh", "bh", "ape", "ape_rel", "mpe"])
        limit = 0.0 if mac == "bh" else round(10 ** rng.uniform(-2.5, -1.5), 5)
        prec = "fp64" if fp64 else "fp32"
        if rng.random() < 0.4:
            return _drawn(_grav("", "uniform", rng.choice([16, 32, 64] if fp64 else [16, 32, 64, 128]),
                                rng.choice(["sphere", "plummer"]), theta=theta, mac=mac, limit=limit, precision=prec,
                                by=rng.choice([1.0, 1.0, 2.0])))
        return _drawn(_grav("", "amr", rng.choice([4, 5] if fp64 else [4, 5, 6]), "plummer", theta=theta, mac=mac, limit=limit,
                            precision=prec, thresh=round(10 ** rng.uniform(-2.9, -2.1), 6)))
    if r < 0.58:   # periodic boxes
        return _drawn(_grav("", "uniform", rng.choice([16, 32, 64, 128]), rng.choice(["turbulent", "plummer"]), bc="3p",
                            theta=theta, ewald=rng.choice(["table", "taylor"]), mac=rng.choice(["bh", "bh", "ape"]),
                            limit=1e-2, by=rng.choice([1.0, 1.0, 0.75])))
    if r < 0.70:   # disks
        ew = rng.choice(["table", "taylor", "taylor", "mlp"])
        return _drawn(_grav("", "uniform", rng.choice([16, 32]) if ew == "mlp" else rng.choice([16, 32, 64]), "disk",
                            bc="2p1i", theta=theta, ewald=ew, by=rng.choice([1.0, 1.25]), bz=rng.choice([2.0, 4.0])))
    if r < 0.88:   # column densities
        species = rng.random() < 0.4
        n_side = rng.choice([1, 2, 3] if species else [1, 2, 2, 4])
        n = rng.choice([16, 32, 64] if species or n_side == 4 else [16, 32, 64, 128])
        return _drawn(_cols("", n, rng.choice(["turbulent", "plummer", "sphere"]), rng.choice(["iso", "3p"]), n_side, theta,
                            species))
    b = _batch("", rng.randint(2, 9), rng.choice([16, 32]), rng.choice([0, 1]), rng.choice(["table", "taylor"]),
               rng.choice([1, 2]))
    return _drawn(dict(b, theta=theta))


def _drawn(case):
    del case["name"]
    return case


# ------------------------------------------------------------------------------ inputs
BCS = {"iso": (0, 0, 0), "3p": (1, 1, 1), "2p1i": (1, 1, 0)}


@functools.lru_cache(maxsize=32)
def _mesh(mesh, n, thresh, bc, by, bz):
    if mesh == "uniform":
        return inputs.uniform_mesh(n, box=(1.0, by, bz), bc=BCS[bc])
    return inputs.build_mesh(inputs.plummer_refine(a=PLUMMER_A, thresh=thresh, min_level=3, max_level=n), bc=BCS[bc])


def _case_mesh(c):
    return _mesh(c["mesh"], c["n"], c["thresh"], c["bc"], c["by"], c["bz"])


def _dev(a, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype, device=DEV)


def _centres(mesh):
    """[nleaf, 8, 8, 8, 3] cell centres (z, y, x order) and [nleaf, 3] cell edges."""
    lf = mesh.leaves
    lo, dx = _dev(mesh.lo[lf]), _dev(mesh.size[lf]) / 8
    i = torch.arange(8, device=DEV, dtype=torch.float64) + 0.5
    ax = [lo[:, a, None] + i * dx[:, a, None] for a in range(3)]
    shape = (len(lf), 8, 8, 8)
    return torch.stack([ax[0][:, None, None, :].expand(shape), ax[1][:, None, :, None].expand(shape),
                        ax[2][:, :, None, None].expand(shape)], -1), dx


def _field(mesh, n, slope, gen):
    """Unit-variance Gaussian random field with P(k) ~ k^slope on a uniform mesh, by leaf-block."""
    k = torch.fft.fftfreq(n, device=DEV, dtype=torch.float64) * n
    kk = torch.sqrt(k[:, None, None] ** 2 + k[None, :, None] ** 2 + (torch.fft.rfftfreq(n, device=DEV, dtype=torch.float64) * n) ** 2)
    amp = torch.where(kk > 0, kk.clamp_min(1.0) ** (slope / 2), torch.zeros_like(kk))
    f = torch.fft.irfftn(torch.fft.rfftn(torch.randn((n, n, n), generator=gen, device=DEV, dtype=torch.float64)) * amp, s=(n, n, n))
    f = (f - f.mean()) / f.std()
    lf = mesh.leaves
    b = np.rint((mesh.lo[lf] - mesh.lo[0]) / mesh.size[lf]).astype(np.int64)
    nb = n // 8
    g = f.view(nb, 8, nb, 8, nb, 8).permute(0, 2, 4, 1, 3, 5).reshape(nb ** 3, 8, 8, 8)
    return g[_dev((b[:, 2] * nb + b[:, 1]) * nb + b[:, 0], torch.int64)]


def _density(mesh, n, kind, seed):
    """Density [ncell] in the library's cell order."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(0x5EED + int(seed))
    x, _ = _centres(mesh)
    mid = _dev(mesh.lo[0] + 0.5 * mesh.size[0])
    noise = lambda: torch.randn(x.shape[:-1], generator=gen, device=DEV, dtype=torch.float64)   # noqa: E731
    if kind == "sphere":
        inside = ((x - mid) ** 2).sum(-1).sqrt() < 0.3
        rho = torch.where(inside, 1.0, 1e-3) * (1.0 + 0.1 * noise()).clamp_min(0.05)
    elif kind == "plummer":
        r2 = ((x - mid) ** 2).sum(-1)
        rho = (1.0 + r2 / PLUMMER_A ** 2) ** -2.5 * torch.exp(0.2 * noise() - 0.02)
    elif kind == "turbulent":
        rho = torch.exp(1.5 * _field(mesh, n, -4.0, gen) - 1.125)
    else:
        rho = torch.exp(-(x[..., 2] - mid[2]).abs() / 0.05) * (1.0 + 0.3 * _field(mesh, n, -2.0, gen))
        rho = rho.clamp_min(1e-6)
    return rho.reshape(-1).contiguous()


def _species(rho, seed):
    """H2 and CO densities of a cloud: fractions that rise with density, with scatter."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(0xC0 + int(seed))
    s = torch.exp(0.3 * torch.randn((2, rho.numel()), generator=gen, device=DEV, dtype=torch.float64))
    f = rho / (rho + 0.02)
    return torch.stack([0.5 * f * rho, 1e-4 * f * f * rho]) * s


def _co_table():
    c, h = np.linspace(10, 19, CO_TAB[0]), np.linspace(16, 23, CO_TAB[1])
    return np.exp(-((10.0 ** (c[:, None] - 16.5)) ** 0.4) - 0.2 * 10.0 ** (h[None, :] - 22.0))


SHIELD = dict(k_av=2.0, k_h2=1e21, b5=3.0, k_co=1e21, lg_co=(10.0, 19.0), lg_h2=(16.0, 23.0))


def _accel_scale(mesh, rho):
    """Largest acceleration of a Plummer sphere of the mesh's mass: the scale of the MAC's limits."""
    x, dx = _centres(mesh)
    mass = float((rho.view(x.shape[0], -1) * dx.prod(-1)[:, None]).sum())
    return mass, 0.385 * mass / PLUMMER_A ** 2


def _limits(c, mesh, rho):
    """(a_lim, a_old): the absolute limit, or |a| of the last step as a program has it (a smooth model)."""
    mass, amax = _accel_scale(mesh, rho)
    if c["density"] != "plummer":
        amax = mass / 0.3 ** 2
    if c["mac"] in ("ape", "mpe"):
        return c["limit"] * amax, None
    if c["mac"] == "ape_rel":
        x, _ = _centres(mesh)
        mid = _dev(mesh.lo[0] + 0.5 * mesh.size[0])
        r2 = ((x - mid) ** 2).sum(-1).reshape(-1)
        return 0.0, (mass * r2.sqrt() / (r2 + PLUMMER_A ** 2) ** 1.5 + 1e-3 * amax).float()
    return 0.0, None


def _network(seed):
    """Weights, normalisation and aspect range of a network such as training gives it."""
    g = torch.Generator().manual_seed(77 + int(seed))
    w = [torch.randn(o, i, generator=g) * (1.6 / i ** 0.5) for i, o in ((4, 64), (64, 64), (64, 64), (64, 4))]
    b = [0.3 * torch.randn(o, generator=g) for o in (64, 64, 64, 4)]
    params = torch.cat([t.reshape(-1) for p in zip(w, b) for t in p])
    norm = torch.tensor([1.5, 1.0, 1.0, 2.0, -2.5, 0.6, 0.6, 3.0])
    return params.numpy(), norm.numpy()


@functools.lru_cache(maxsize=1)
def _stream():
    return torch.cuda.Stream(device=DEV)   # one stream for the program, as a simulation has it


def _batch_grids(c):
    """(mesh, side, density kind) of every grid: sides base, 2 base, 4 base, rotating boundaries."""
    out = []
    for g in range(c["count"]):
        n = c["base"] * 2 ** (g % 3)
        bc = ("iso", "3p", "2p1i")[(g // 3) % 3]
        out.append((_mesh("uniform", n, 0.0, bc, 1.0, 1.0), n, "plummer" if g % 2 == 0 else "turbulent"))
    return out


# ------------------------------------------------------------------------------ the passes
def prepare(case, seed):
    c = case
    if c["kind"] == "batch":
        grids, rhos, solvers = _batch_grids(c), [], []
        for g, (mesh, n, kind) in enumerate(grids):
            rho = _density(mesh, n, kind, 100 * seed + g)
            ts = TreeSolver(0, _stream())
            torch.cuda.current_stream().synchronize()
            ts.tree_build(mesh, rho)
            if any(mesh.bc):
                ts.ewald_field(NTAB)
            solvers.append(ts)
            rhos.append(rho)
        b = Batch(solvers)
        b.set_mode(c["mode"], 16 if c["mode"] == 1 else 8)
        npix = 12 * c["n_side"] ** 2
        return dict(kind="batch", batch=b, rhos=rhos, gp=TreeSolver.gravity_params(theta=c["theta"], ewald=c["ewald"], zero_mean=False),
                    cp=TreeSolver.column_params(n_side=c["n_side"], theta=c["theta"]),
                    pots=[torch.empty(m.ncell, device=DEV) for m, _, _ in grids],
                    accs=[torch.empty(m.ncell, 3, device=DEV) for m, _, _ in grids],
                    cols=[torch.empty(m.ncell, npix, device=DEV) for m, _, _ in grids])
    mesh = _case_mesh(c)
    rho = _density(mesh, c["n"], c["density"], seed)
    ts = TreeSolver(0, _stream())
    s = dict(kind=c["kind"], ts=ts, rho=rho)
    if c["kind"] == "columns":
        npix = 12 * c["n_side"] ** 2
        lq = 3 if c["species"] else 1
        s.update(q=_species(rho, seed) if c["species"] else None, cols=torch.empty(mesh.ncell, lq, npix, device=DEV),
                 out=torch.empty(mesh.ncell, 3 if c["species"] else 1, device=DEV), co=_co_table(),
                 params=TreeSolver.column_params(n_side=c["n_side"], theta=c["theta"]))
    else:
        fp64 = c["precision"] == "fp64"
        dt = torch.float64 if fp64 else torch.float32
        a_lim, a_old = _limits(c, mesh, rho)
        mac = "ape" if c["mac"] == "ape_rel" else c["mac"]
        s.update(pot=torch.empty(mesh.ncell, dtype=dt, device=DEV), acc=torch.empty(mesh.ncell, 3, dtype=dt, device=DEV), a_old=a_old,
                 params=TreeSolver.gravity_params(mac=mac, theta=c["theta"], a_lim=a_lim, a_old=a_old,
                                                  eps_rel=c["limit"] if a_old is not None else 0.0, precision=c["precision"],
                                                  zero_mean=c["bc"] != "iso", ewald=c["ewald"]))
        ts.fp64_records(fp64)
    torch.cuda.current_stream().synchronize()
    ts.tree_build(mesh, rho)
    if c["kind"] == "gravity" and c["bc"] != "iso":
        if c["ewald"] == "mlp":
            params, norm = _network(seed)
            ts.surrogate_set(params, norm, NET_B)
        else:
            ts.ewald_field(NTAB)
            if c["ewald"] == "taylor":
                ts.ewald_taylor_table()
    return s


def run(state):
    s = state
    if s["kind"] == "batch":
        s["batch"].run(gravity=s["gp"], pots=s["pots"], accs=s["accs"], column=s["cp"], cols=s["cols"], densities=s["rhos"])
        return {"pot": s["pots"], "acc": s["accs"], "cols": s["cols"]}
    ts = s["ts"]
    ts.tree_build(None, s["rho"])
    if s["kind"] == "gravity":
        ts.gravity_walk(s["pot"], s["acc"], s["params"])
        return {"pot": s["pot"], "acc": s["acc"]}
    if s["q"] is not None:
        ts.column_quantities(s["q"])
    ts.column_walk(s["cols"], s["params"])
    if s["q"] is not None:
        ts.column_shielding(s["cols"], s["out"], co_table=s["co"], **SHIELD)
    else:
        ts.column_av(s["cols"][:, 0], k=SHIELD["k_av"], av=s["out"][:, 0])
    return {"cols": s["cols"], "out": s["out"]}


# ------------------------------------------------------------------------------ work
FLOP_PAIR, FLOP_MAC, FLOP_IMAGE = 20, 15, 9        # one interaction, one acceptance test, minimum image
FLOP_LOOKUP = {"table": 93, "taylor": 36, "mlp": 17408}
FLOP_COLUMN, FLOP_PIXEL = 40, 3 * 2.05             # bins of one node, and its pixels


_SEEN = {}


def _rates(mesh, n, density, c):
    """Interactions and acceptance tests per cell, from the 64-bit walk of a sample of cells."""
    key = (mesh.bc, mesh.ncell, density, tuple(sorted((k, v) for k, v in c.items() if k != "name")))
    if key in _SEEN:
        return _SEEN[key]
    rho = _density(mesh, n, density, 1)
    tree = _Tree(mesh, rho)
    at = _dev(inputs.sample_cells(mesh.ncell, 1024), torch.int64)
    pairs = 0

    def visit(t, node, d, d2, base):
        nonlocal pairs
        pairs += t.numel()

    tests = tree.walk(_criterion(c, mesh, rho, tree), visit, at)
    _SEEN[key] = pairs / at.numel(), tests / at.numel()
    return _SEEN[key]


def work(case):
    c = case
    grids = _batch_grids(c) if c["kind"] == "batch" else [(_case_mesh(c), c["n"], c["density"])]
    nbytes = flops = 0.0
    for mesh, n, density in grids:
        per, tests = _rates(mesh, n, density, c)
        image = FLOP_IMAGE if any(mesh.bc) else 0
        cells = mesh.ncell
        nbytes += 8 * cells
        if c["kind"] != "columns":
            lookup = FLOP_LOOKUP[c["ewald"]] if any(mesh.bc) else 0
            flops += cells * (per * (FLOP_PAIR + image + lookup) + tests * (FLOP_MAC + image))
            nbytes += cells * (32 if c.get("precision") == "fp64" else 16) + (4 * cells if c.get("mac") == "ape_rel" else 0)
        if c["kind"] != "gravity":
            lq = 3 if c.get("species") else 1
            npix = 12 * c["n_side"] ** 2
            flops += cells * (per * (FLOP_COLUMN + image + lq * FLOP_PIXEL) + tests * (FLOP_MAC + image))
            nbytes += cells * 4 * lq * npix
            if c["kind"] == "columns":
                nbytes += cells * (16 + 4 * 3 if c["species"] else 4)
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------------------ 64-bit reference
class _Tree:
    """The octree in 64 bits: internal nodes (blocks, then 8 + 64 nodes per leaf-block), then cells."""

    def __init__(self, mesh, rho):
        lf = mesh.leaves
        nl, nb = len(lf), mesh.nblocks
        x, dx = _centres(mesh)
        self.mesh, self.ni = mesh, nb + 72 * nl
        total = self.ni + 512 * nl
        self.m = torch.zeros(total, dtype=torch.float64, device=DEV)
        self.com = torch.zeros(total, 3, dtype=torch.float64, device=DEV)
        self.cen = torch.zeros(self.ni, 3, dtype=torch.float64, device=DEV)
        self.half = torch.zeros(total, 3, dtype=torch.float64, device=DEV)
        self.kids = torch.zeros(self.ni, 8, dtype=torch.int64, device=DEV)
        leaf = torch.arange(nl, device=DEV)

        def octants(v):   # [nl, 2k, 2k, 2k, ...] -> [nl, k, k, k, 8, ...], octant = x + 2 y + 4 z
            k = v.shape[1] // 2
            v = v.view(nl, k, 2, k, 2, k, 2, *v.shape[4:])
            return v.permute(0, 1, 3, 5, 2, 4, 6, *range(7, v.dim())).reshape(nl, k, k, k, 8, *v.shape[7:])

        ids = (self.ni + torch.arange(512 * nl, device=DEV)).view(nl, 8, 8, 8)
        m, com, cen = rho.view(nl, 8, 8, 8) * dx.prod(-1)[:, None, None, None], x, x
        self.m[self.ni:], self.com[self.ni:] = m.reshape(-1), com.reshape(-1, 3)
        self.half[self.ni:] = (0.5 * dx)[:, None].expand(nl, 512, 3).reshape(-1, 3)
        for k, start in ((4, 8), (2, 0), (1, None)):
            km, kc, kx, ki = octants(m), octants(com), octants(cen), octants(ids)
            m = km.sum(-1)
            cen = kx.mean(-2)
            com = torch.where(m[..., None] > 0, (km[..., None] * kc).sum(-2) / m.clamp_min(1e-300)[..., None], cen)
            if start is None:
                ids = _dev(lf, torch.int64).view(nl, 1, 1, 1)
            else:
                ids = (nb + 72 * leaf[:, None] + start + torch.arange(k ** 3, device=DEV)).view(nl, k, k, k)
            at = ids.reshape(-1)
            self.m[at], self.com[at], self.cen[at] = m.reshape(-1), com.reshape(-1, 3), cen.reshape(-1, 3)
            self.half[at] = (0.5 * (8 // k) * dx)[:, None].expand(nl, k ** 3, 3).reshape(-1, 3)
            self.kids[at] = ki.reshape(-1, 8)
        level = mesh.level
        for lev in range(int(level.max()), 0, -1):   # amr blocks, deepest first
            up = np.nonzero((level == lev) & (mesh.child[:, 0] >= 0))[0]
            if not up.size:
                continue
            at, kid = _dev(up, torch.int64), _dev(mesh.child[up], torch.int64)
            km, kc = self.m[kid], self.com[kid]
            self.m[at] = km.sum(-1)
            self.cen[at] = _dev(mesh.lo[up] + 0.5 * mesh.size[up])
            self.com[at] = (km[..., None] * kc).sum(1) / km.sum(-1)[:, None]
            self.half[at] = _dev(0.5 * mesh.size[up])
            self.kids[at] = kid
        self.h = 2 * self.half.max(-1).values
        self.box = [(a, float(mesh.size[0][a])) for a in range(3) if mesh.bc[a]]

    def image(self, d):
        for a, L in self.box:
            d[:, a] -= L * torch.round(d[:, a] / L)
        return d

    def moments(self):
        """B2, B3 of every internal node about its centre of mass (MPE)."""
        b = torch.zeros(self.ni, 2, dtype=torch.float64, device=DEV)
        parent = torch.zeros(self.m.numel(), dtype=torch.int64, device=DEV)
        parent[self.kids.reshape(-1)] = torch.arange(self.ni, device=DEV).repeat_interleave(8)
        pos, m = self.com[self.ni:], self.m[self.ni:]
        up = parent[self.ni:]
        for _ in range(3 + int(self.mesh.level.max())):
            u = ((pos - self.com[up]) ** 2).sum(-1)
            v = torch.stack([m * u, m * u * u.sqrt()], -1)
            v[up < 0] = 0
            b.index_add_(0, up.clamp_min(0), v)
            root = up <= 0
            up = torch.where(root, torch.full_like(up, -1), parent[up.clamp_min(0)])
        return b

    def walk(self, accepts, visit, targets=None, chunk=16384):
        """Walk of every target cell; visit(t, node, d, d2, base) for accepted (target, node) pairs in target order."""
        n = self.m.numel() - self.ni
        every = torch.arange(n, device=DEV) if targets is None else targets
        tests = 0
        for base in range(0, every.numel(), chunk):
            me = every[base:base + chunk]
            pos = self.com[self.ni + me]
            t = torch.arange(me.numel(), device=DEV)
            node = torch.zeros_like(t)
            while t.numel():
                d = self.image(pos[t] - self.com[node])
                d2 = (d * d).sum(-1)
                leaf = node >= self.ni
                take = leaf & (node != self.ni + me[t])
                inner = torch.nonzero(~leaf).squeeze(1)
                tests += inner.numel()
                if inner.numel():
                    k = node[inner]
                    g = self.image(pos[t[inner]] - self.cen[k]).abs()
                    ok = accepts(me[t[inner]], k, d2[inner]) & (g > 1.2 * self.half[k]).any(-1)
                    take[inner] = ok
                    opened = inner[~ok]
                s = torch.nonzero(take).squeeze(1)
                if s.numel():
                    visit(t[s], node[s], d[s], d2[s], base)
                if not inner.numel():
                    break
                t, node = t[opened].repeat_interleave(8), self.kids[node[opened]].reshape(-1)
        return tests


def _criterion(c, mesh, rho, tree):
    mac = c.get("mac", "bh")
    if mac == "bh":
        th2 = c["theta"] ** 2
        return lambda me, k, d2: tree.h[k] ** 2 < th2 * d2
    a_lim, a_old = _limits(c, mesh, rho)
    lim = (lambda me: c["limit"] * a_old[me].double()) if a_old is not None else (lambda me: a_lim)
    if mac != "mpe":
        return lambda me, k, d2: tree.m[k] * tree.h[k] ** 2 < lim(me) * d2 * d2
    b = tree.moments()
    bmax = (tree.half[:tree.ni] + (tree.com[:tree.ni] - tree.cen).abs()).norm(dim=-1)

    def mpe(me, k, d2):
        inv = d2.rsqrt()
        q = 1 - bmax[k] * inv
        return (q > 0) & (inv * inv * (3 * b[k, 0] * inv * inv - 2 * b[k, 1] * inv ** 3) < lim(me) * q * q)
    return mpe


def _sums(t, v, n):
    """Sums of the rows of v by their (sorted) target index."""
    return torch.segment_reduce(v, "sum", lengths=torch.bincount(t, minlength=n), axis=0, initial=0)


def _images(d, shifts, alpha):
    """Real-space Ewald sums of C and A_c: the unit mass's own image without its 1/r, and the others."""
    C, A = torch.zeros_like(d[..., 0]), torch.zeros_like(d)
    for s in shifts:
        v = d - torch.tensor(s, dtype=torch.float64, device=DEV)
        u = (v * v).sum(-1)
        r = u.sqrt()
        x = alpha * r
        if any(s):
            e = torch.erfc(x)
            C += e / r
            A += v * (alpha * 2 / math.sqrt(math.pi) * torch.exp(-x * x) / u + e / (u * r))[..., None]
        else:
            near, rs = x < 0.05, r.clamp_min(1e-30)
            x2 = x * x
            sp = 1 - x2 / 3 + x2 ** 2 / 10 - x2 ** 3 / 42 + x2 ** 4 / 216
            sa = -2 * (1 / 3 - x2 / 5 + x2 ** 2 / 14 - x2 ** 3 / 54 + x2 ** 4 / 264)
            k = 2 * alpha / math.sqrt(math.pi)
            C -= torch.where(near, k * sp, torch.erf(x) / rs)
            A += v * torch.where(near, k * alpha ** 2 * sa,
                                 k * torch.exp(-x2) / rs ** 2 - torch.erf(x) / rs ** 3)[..., None]
    return C, A


def _series(d, bc, box):
    """Correction (C, A_c) of separations d [..., 3] by the Ewald series, alpha = 2 / Lx."""
    Lx, Ly, Lz = box
    b, alpha = Ly / Lx, 2 / Lx
    R, K = 15.0, 10.0
    span = lambda lim, f: range(-int(math.sqrt(lim) * f), int(math.sqrt(lim) * f) + 1)   # noqa: E731
    if bc == "3p":
        cz = Lz / Lx
        C, A = _images(d, [(i * Lx, j * Ly, k * Lz) for k in span(R, 1 / cz) for j in span(R, 1 / b) for i in span(R, 1)
                           if i * i + (b * j) ** 2 + (cz * k) ** 2 <= R], alpha)
        V = Lx * Ly * Lz
        for n in span(K, cz):
            for m in span(K, b):
                for l in span(K, 1):
                    s2 = l * l + (m / b) ** 2 + (n / cz) ** 2
                    if s2 == 0 or s2 > K:
                        continue
                    k = torch.tensor([2 * math.pi * l / Lx, 2 * math.pi * m / Ly, 2 * math.pi * n / Lz], dtype=torch.float64, device=DEV)
                    kk = float((k * k).sum())
                    amp, ph = 4 * math.pi / (V * kk) * math.exp(-kk / (4 * alpha ** 2)), d @ k
                    C += amp * torch.cos(ph)
                    A += amp * torch.sin(ph)[..., None] * k
        return C - math.pi / (alpha ** 2 * V), A
    C, A = _images(d, [(i * Lx, j * Ly, 0.0) for j in span(R, 1 / b) for i in span(R, 1) if i * i + (b * j) ** 2 <= R], alpha)
    zeta = math.pi ** 2 / 4
    sz = math.sqrt(zeta)
    gam = 2 * math.pi * d[..., 2] / Lx
    ag, sg = gam.abs(), torch.where(gam < 0, -1.0, 1.0)
    for m in span(K, b):
        for l in span(K, 1):
            s = math.sqrt(l * l + (m / b) ** 2)
            if s * s > K:
                continue
            if s == 0:
                I = -math.pi * (ag * torch.erf(ag / (2 * sz)) + 2 * math.sqrt(zeta / math.pi) * torch.exp(-ag ** 2 / (4 * zeta)))
                I = I + 2 * math.sqrt(math.pi * zeta)
                D = -math.pi * torch.erf(ag / (2 * sz))
            else:
                p = torch.exp(-ag ** 2 / (4 * zeta) - zeta * s * s) * torch.special.erfcx((zeta * s + ag / 2) / sz)
                q = torch.exp(-ag * s) * torch.erfc((zeta * s - ag / 2) / sz)
                I, D = math.pi / (2 * s) * (p + q), math.pi / 2 * (p - q)
            ph = 2 * math.pi * (l * d[..., 0] / Lx + m * d[..., 1] / Ly)
            cs, sn = torch.cos(ph), torch.sin(ph)
            C += cs * I / (math.pi * Lx * b)
            A[..., 0] += 2 * l * sn * I / (b * Lx ** 2)
            A[..., 1] += 2 * m * sn * I / (b * b * Lx ** 2)
            A[..., 2] -= 2 * cs * sg * D / (b * Lx ** 2)
    return C, A


@functools.lru_cache(maxsize=6)
def _lookup(bc, box, taylor):
    """Table of the correction on the folded grid (with its Jacobian for the Taylor form), its spacing and far distance."""
    Lx, Ly, Lz = box
    far = math.inf if bc == "3p" else 2 * max(Lx, Ly)
    ext = (Lx / 2, Ly / 2, Lz / 2 if bc == "3p" else min(Lz, far))
    h = torch.tensor([e / (NTAB - 1) for e in ext], dtype=torch.float64, device=DEV)
    i = torch.arange(NTAB, device=DEV, dtype=torch.float64)
    d = torch.stack(torch.meshgrid(i * h[0], i * h[1], i * h[2], indexing="ij"), -1).reshape(-1, 3)
    C, A = _series(d, bc, box)
    tab = torch.cat([C[:, None], A], -1)
    J = None
    if taylor:
        J = torch.empty(d.shape[0], 3, 3, dtype=torch.float64, device=DEV)
        for a in range(3):
            e = torch.zeros(3, dtype=torch.float64, device=DEV)
            e[a] = 1e-5 * Lx
            J[:, :, a] = (_series(d + e, bc, box)[1] - _series(d - e, bc, box)[1]) / (2e-5 * Lx)
        J = 0.5 * (J + J.transpose(1, 2))
    return tab, J, h, far


def _correction(d, bc, box, taylor):
    """(C, A_c) at separations d, looked up as the walk does, and where the far-field form applies."""
    tab, J, h, far = _lookup(bc, box, taylor)
    a = d.abs()
    flat = lambda i: (i[:, 0] * NTAB + i[:, 1]) * NTAB + i[:, 2]   # noqa: E731
    u = a / h
    if taylor:
        g = torch.floor(u + 0.5).long().clamp_max(NTAB - 1)
        k, w = flat(g), a - g * h
        C = tab[k, 0] - (tab[k, 1:] * w).sum(-1)
        A = tab[k, 1:] + (J[k] * w[:, None, :]).sum(-1)
    else:
        u = u.clamp_max(NTAB - 1)
        i = u.long().clamp_max(NTAB - 2)
        f = u - i
        v = 0
        for o in range(8):
            off = torch.tensor([o & 1, (o >> 1) & 1, o >> 2], device=DEV)
            v = v + torch.where(off == 1, f, 1 - f).prod(-1)[:, None] * tab[flat(i + off)]
        C, A = v[:, 0], v[:, 1:]
    return C, torch.where(d < 0, -A, A), a[:, 2] > far


def _far_2p1i(d, box):
    """The far-field potential and acceleration of one unit mass (x, y periodic)."""
    Lx, Ly = box[:2]
    slope = 2 * math.pi / (Ly * Lx)
    A = torch.zeros_like(d)
    A[:, 2] = torch.copysign(torch.full_like(d[:, 2], slope), d[:, 2])
    return 2 * math.sqrt(math.pi * math.pi ** 2 / 4) / (math.pi * Ly) - slope * d[:, 2].abs(), A


def _net_correction(d, box, params, norm):
    """(C, A_c) of the learned correction, and where the far-field form applies."""
    Lx, Ly = box[:2]
    b = Ly / Lx
    scale = _dev([Lx / 2, Ly / 2, 2 * Lx * max(1.0, NET_B[1])])
    x = torch.cat([d.abs() / scale, torch.full_like(d[:, :1], (b - NET_B[0]) / (NET_B[1] - NET_B[0]))], -1) * 2 - 1
    p, at = _dev(params), 0
    for i, o in ((4, 64), (64, 64), (64, 64), (64, 4)):
        w, bias = p[at:at + i * o].view(o, i), p[at + i * o:at + i * o + o]
        at += i * o + o
        x = x @ w.T + bias
        if o == 64:
            x = torch.nn.functional.silu(x)
    nm = _dev(norm)
    x = x * nm[:4] + nm[4:]
    A = x[:, 1:] / Lx ** 2
    return x[:, 0] / Lx, torch.where(d < 0, -A, A), d[:, 2].abs() > 2 * max(Lx, Ly)


def _gravity64(c, mesh, rho, zero_mean, seed):
    tree = _Tree(mesh, rho)
    n = mesh.ncell
    out = torch.zeros(n, 4, dtype=torch.float64, device=DEV)
    box = tuple(float(v) for v in mesh.size[0])
    bc = {v: k for k, v in BCS.items()}[tuple(mesh.bc)]
    net = _network(seed) if c["ewald"] == "mlp" else None
    chunk = 16384 if bc != "2p1i" else 2048

    def pairs(t, node, d, d2, base):
        inv = d2.rsqrt()
        pot, A = inv, d * (inv ** 3)[:, None]
        if bc != "iso":
            C, Ac, far = _net_correction(d, box, *net) if net else _correction(d, bc, box, c["ewald"] == "taylor")
            pot, A = pot + C, A + Ac
            if bc == "2p1i":
                fp, fA = _far_2p1i(d, box)
                pot, A = torch.where(far, fp, pot), torch.where(far[:, None], fA, A)
        m = tree.m[node]
        k = min(chunk, n - base)
        out[base:base + k] -= _sums(t, torch.cat([(m * pot)[:, None], m[:, None] * A], -1), k)

    def visit(t, node, d, d2, base):   # (in pieces at target boundaries where the pairs are many)
        if t.numel() <= 1 << 24:
            return pairs(t, node, d, d2, base)
        cuts = [int(torch.searchsorted(t, v)) for v in range(0, chunk, chunk // 16)] + [t.numel()]
        for a, b in zip(cuts[:-1], cuts[1:]):
            if b > a:
                pairs(t[a:b], node[a:b], d[a:b], d2[a:b], base)

    tree.walk(_criterion(c, mesh, rho, tree), visit, chunk=chunk)
    pot = out[:, 0]
    if zero_mean:
        _, dx = _centres(mesh)
        dv = dx.prod(-1).repeat_interleave(512)
        pot = pot - (dv * pot).sum() / dv.sum()
    return pot, out[:, 1:].clone()


def _pixel(ns, z, phi):
    """HEALPix RING pixel of directions (z = cos theta, azimuth)."""
    t = torch.remainder(phi, 2 * math.pi) * (2 / math.pi)
    za = z.abs()
    u, v = ns * (0.5 + t), 0.75 * ns * z
    up, dn = torch.floor(u - v), torch.floor(u + v)
    ring = ns + 1 + up - dn
    odd = 1 - torch.remainder(ring, 2)
    ip = torch.remainder(torch.floor((up + dn - ns + odd + 1) / 2), 4 * ns)
    belt = 2 * ns * (ns - 1) + (ring - 1) * 4 * ns + ip
    f = t - torch.floor(t)
    s = ns * torch.sqrt(3 * (1 - za))
    r = torch.floor(f * s) + torch.floor((1 - f) * s) + 1
    ip = torch.remainder(torch.floor(t * r), 4 * r)
    cap = torch.where(z > 0, 2 * r * (r - 1) + ip, 12 * ns * ns - 2 * r * (r + 1) + ip)
    return torch.where(za <= 2 / 3, belt, cap).long()


@functools.lru_cache(maxsize=4)
def _noderay(ns, nth=25, nph=50, nps=25, pmin=1e-3, pmax=1.0, nsub=8):
    """Share of a cube's sub-cubes in every pixel, by bins of direction and angular size."""
    i = lambda n: torch.arange(n, device=DEV, dtype=torch.float64) + 0.5   # noqa: E731
    th, ph = (i(nth) * math.pi / nth)[:, None, None], (i(nph) * 2 * math.pi / nph)[None, :, None]
    psi = (pmin * (pmax / pmin) ** (i(nps) / nps))[None, None, :]
    npix = 12 * ns * ns
    w = torch.zeros(nth, nph, nps, npix, dtype=torch.float64, device=DEV)
    off = (i(nsub) / nsub - 0.5).tolist()
    one = torch.full((nth, nph, nps, 1), 1.0 / nsub ** 3, dtype=torch.float64, device=DEV)
    for a in off:
        for b in off:
            for e in off:
                x, y, z = torch.sin(th) * torch.cos(ph) + psi * a, torch.sin(th) * torch.sin(ph) + psi * b, torch.cos(th) + psi * e
                r = torch.sqrt(x * x + y * y + z * z)
                w.scatter_add_(3, _pixel(ns, z / r, torch.atan2(y, x))[..., None], one)
    return w.view(-1, npix)


def _columns64(c, mesh, rho, q):
    tree = _Tree(mesh, rho)
    ns, n = c["n_side"], mesh.ncell
    npix = 12 * ns * ns
    table = _noderay(ns)
    ni = tree.ni
    masses = [tree.m]
    for k in range(0 if q is None else 2):
        masses.append(_Tree(mesh, q[k]).m)
    out = torch.zeros(n, len(masses), npix, dtype=torch.float64, device=DEV)
    chunk = 4096
    lps = math.log2(1e-3)

    def visit(t, node, d, d2, base):
        r = d2.sqrt()
        it = torch.floor(torch.acos((-d[:, 2] / r).clamp(-1, 1)) / math.pi * 25).clamp(0, 24).long()
        ph = torch.atan2(-d[:, 1], -d[:, 0])
        ph = torch.where(ph < 0, ph + 2 * math.pi, ph)
        ip = torch.floor(ph / (2 * math.pi) * 50).clamp(0, 49).long()
        iq = torch.floor((torch.log2(tree.h[node] / r) - lps) * (25 / -lps)).clamp(0, 24).long()
        w = table[(it * 50 + ip) * 25 + iq] * (npix / (4 * math.pi) / d2)[:, None]
        k = min(chunk, n - base)
        for j, m in enumerate(masses):
            out[base:base + k, j] += _sums(t, w * m[node][:, None], k)

    tree.walk(_criterion(dict(c, mac="bh"), mesh, rho, tree), visit, chunk=chunk)
    _, dx = _centres(mesh)
    own = (0.5 / (dx[:, 1] * dx[:, 2])).repeat_interleave(512)
    for j, m in enumerate(masses):
        out[:, j] += (m[ni:] * own)[:, None]
    return out


def _averages64(cols):
    """A_V, and with species the H2 and CO shielding averages, of 64-bit maps."""
    lnp = math.log(cols.shape[-1])
    av = -(torch.logsumexp(-2.5 * SHIELD["k_av"] * cols[:, 0], -1) - lnp) / 2.5
    if cols.shape[1] == 1:
        return av[:, None]
    nh, nc = SHIELD["k_h2"] * cols[:, 1], SHIELD["k_co"] * cols[:, 2]
    x = nh / 5e14
    h2 = (0.965 / (1 + x / SHIELD["b5"]) ** 2 + 0.035 / (1 + x).sqrt() * torch.exp(-8.5e-4 * (1 + x).sqrt())).mean(-1)
    tab = _dev(_co_table())

    def place(v, lim, k):
        u = ((torch.log10(v.clamp_min(1e-30)) - lim[0]) * ((k - 1) / (lim[1] - lim[0]))).clamp(0, k - 1)
        i = u.long().clamp_max(k - 2)
        return i, u - i
    ic, fc = place(nc, SHIELD["lg_co"], CO_TAB[0])
    ih, fh = place(nh, SHIELD["lg_h2"], CO_TAB[1])
    co = (tab[ic, ih] * (1 - fh) + tab[ic, ih + 1] * fh) * (1 - fc) + (tab[ic + 1, ih] * (1 - fh) + tab[ic + 1, ih + 1] * fh) * fc
    return torch.stack([av, h2, co.mean(-1)], -1)


def exact(case, seed):
    c = case
    if c["kind"] == "batch":   # gravity of every grid; of the maps, those of the smaller grids
        out = {"pot": [], "acc": [], "cols": []}
        for g, (mesh, n, kind) in enumerate(_batch_grids(c)):
            rho = _density(mesh, n, kind, 100 * seed + g)
            pot, acc = _gravity64(c, mesh, rho, False, seed)
            out["pot"].append(pot)
            out["acc"].append(acc)
            out["cols"].append(_columns64(c, mesh, rho, None)[:, 0] if n <= 32 else None)
        return out
    mesh = _case_mesh(c)
    rho = _density(mesh, c["n"], c["density"], seed)
    if c["kind"] == "columns":
        if c["n"] > 64:
            return None   # minutes of 64-bit scatters
        cols = _columns64(c, mesh, rho, _species(rho, seed) if c["species"] else None)
        return {"cols": cols, "out": _averages64(cols)}
    pot, acc = _gravity64(c, mesh, rho, c["bc"] != "iso", seed)
    return {"pot": pot, "acc": acc}
