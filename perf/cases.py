"""The work that a user of this library has it do, as measurable cases.

Every case goes through the Python binding (paper_1812_01448_gb300.api), with host arrays in the
caller's numbering, as a simulation script does: a mesh is loaded and set up once (``prepare``),
then a pass writes the initial fields, advances them and reads them back, or sets up, analyses,
optimises or trains.  Meshes are jittered triangle lattices on a rectangle, some with a round
perfectly conducting hole; sizes follow the repository's own workloads (1,024-triangle cavity,
1M-triangle plasma square, 4M-triangle scatterer, batches of 5k to 200k triangles, training
corpora of 1k to 50k triangles per mesh).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1812_01448_gb300 as ue
from paper_1812_01448_gb300 import learned

W0, T0, TAU = 2 * math.pi * 20, 0.1, 0.05      # the line source of the workloads
KINDS = ("march", "batch", "setup", "modes", "relax", "train")


def listed():
    return [
        # the smallest call: a 1k-triangle PEC cavity, a TE mode, every option at its default
        dict(name="cavity-1k", kind="march", nx=32, ny=16, hole=False, tiles="none", depth=0, fp64=False,
             plasma=False, frame=0, source=False, watchdog=0, steps=200),
        # an ordinary mesh with the default options, a source and the energy watchdog on
        dict(name="plain-90k", kind="march", nx=233, ny=193, hole=True, tiles="none", depth=0, fp64=False,
             plasma=False, frame=0, source=True, watchdog=32, steps=256),
        # the double precision check build on a plasma
        dict(name="plain-fp64-240k", kind="march", nx=347, ny=347, hole=False, tiles="none", depth=0, fp64=True,
             plasma=True, frame=0, source=True, watchdog=0, steps=96),
        # the scatterer workload, temporally blocked as the benchmark runs it
        dict(name="scatterer-4m", kind="march", nx=1407, ny=1405, hole=True, tiles="rings", depth=10, fp64=False,
             plasma=False, frame=0, source=True, watchdog=0, steps=200),
        # the plasma workload, temporally blocked
        dict(name="plasma-500k", kind="march", nx=501, ny=499, hole=False, tiles="rings", depth=8, fp64=False,
             plasma=True, frame=0, source=True, watchdog=0, steps=200),
        # open boundaries: a 16-cell PML frame around a scatterer, temporally blocked
        dict(name="frame-500k", kind="march", nx=500, ny=500, hole=True, tiles="rings", depth=8, fp64=False,
             plasma=False, frame=16, source=True, watchdog=0, steps=160),
        # many independent meshes in one batch, each with its own scatterer, time step and source
        dict(name="batch-12", kind="batch", meshes=12, n_min=5000, n_max=120000, depth=8, steps=160),
        # setup of a loaded mesh: geometry and the time step from the power iteration
        dict(name="setup-240k", kind="setup", nx=351, ny=349, hole=True, iters=200),
        # setup of a small mesh, as in a parameter study
        dict(name="setup-10k", kind="setup", nx=71, ny=73, hole=True, iters=200),
        # the highest eigenmodes, which set the stability limit
        dict(name="modes-90k", kind="modes", nx=213, ny=211, hole=True, n_modes=8, iters=100),
        # mesh optimisation of a randomly seeded node cloud
        dict(name="relax-20k", kind="relax", points=20011, iters=100, flip_every=20),
        # one epoch of training the spectral-radius predictor on a corpus of meshes
        dict(name="train-400", kind="train", meshes=400, n_min=1000, n_max=50000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("march", "march", "march", "batch", "setup", "modes", "relax", "train"))
    if kind == "march":
        tiles = rng.choice(("none", "rings"))
        nx = _log_int(rng, 40, 400) if tiles == "none" else _log_int(rng, 120, 700)
        fp64 = tiles == "none" and rng.random() < 0.25
        frame = rng.choice((0, 0, 0, 8, 12, 16))
        ny = max(8, int(nx * rng.uniform(0.6, 1.0)))
        ny += ny % 2 if frame else 0
        return dict(kind="march", nx=nx, ny=ny, hole=rng.random() < 0.5, tiles=tiles,
                    depth=rng.choice((4, 6, 8)) if tiles == "rings" else 0, fp64=fp64,
                    plasma=rng.random() < 0.3, frame=frame, source=rng.random() < 0.8,
                    watchdog=rng.choice((0, 0, 50)), steps=rng.randint(50, 250))
    if kind == "batch":
        return dict(kind="batch", meshes=rng.randint(3, 12), n_min=5000, n_max=rng.randint(20000, 120000),
                    depth=rng.choice((4, 6, 8)), steps=rng.randint(50, 200))
    if kind == "setup":
        nx = _log_int(rng, 30, 500)
        return dict(kind="setup", nx=nx, ny=max(8, int(nx * rng.uniform(0.6, 1.0))), hole=rng.random() < 0.5,
                    iters=rng.choice((100, 200, 300)))
    if kind == "modes":
        nx = _log_int(rng, 40, 300)
        return dict(kind="modes", nx=nx, ny=max(20, int(nx * rng.uniform(0.6, 1.0))), hole=rng.random() < 0.5,
                    n_modes=rng.choice((2, 4, 6, 8, 11, 16)), iters=rng.randint(30, 120))
    if kind == "relax":
        return dict(kind="relax", points=_log_int(rng, 1000, 25000), iters=rng.randint(40, 120),
                    flip_every=rng.choice((10, 20, 25)))
    return dict(kind="train", meshes=rng.randint(20, 400), n_min=1000, n_max=rng.randint(10000, 50000))


# --- meshes ---------------------------------------------------------------------------------

def _lattice(nx, ny, seed, hole, jitter=0.08):
    """Rows of isosceles triangles (base h, height h) on [0, nx h] x [0, ny h], h = 1/nx, the sides
    straight, interior nodes moved by up to jitter h; with a hole, the triangles that lay inside
    a disc are left out.  Boundary spacing is h on all four sides for even ny.  Returns (xy, tris)."""
    rng = np.random.default_rng(seed)
    h = 1.0 / nx
    even = np.arange(nx + 1) * h
    odd = np.concatenate([[0.0], (np.arange(nx) + 0.5) * h, [nx * h]])
    width = np.where(np.arange(ny + 1) % 2 == 0, nx + 1, nx + 2)
    off = np.concatenate([[0], np.cumsum(width)])
    x = np.concatenate([even if j % 2 == 0 else odd for j in range(ny + 1)])
    y = np.repeat(np.arange(ny + 1) * h, width)
    edge = np.zeros(off[-1], bool)
    edge[off[:-1]] = edge[off[1:] - 1] = True
    edge[:width[0]] = edge[off[-2]:] = True
    xy = np.stack([x, y], axis=1)
    flat = xy.copy()
    free = np.nonzero(~edge)[0]
    xy[free] += rng.uniform(-jitter * h, jitter * h, size=(free.size, 2))
    i = np.arange(nx)
    k = np.arange(nx + 1)
    rows = []
    for j in range(ny):
        lo, up = off[j], off[j + 1]
        if j % 2 == 0:      # nx + 1 nodes below, nx + 2 above
            rows.append(np.stack([lo + i, lo + i + 1, up + i + 1], axis=1))
            rows.append(np.stack([lo + k, up + k + 1, up + k], axis=1))
        else:               # nx + 2 nodes below, nx + 1 above
            rows.append(np.stack([up + i, lo + i + 1, up + i + 1], axis=1))
            rows.append(np.stack([lo + k, lo + k + 1, up + k], axis=1))
    tris = np.concatenate(rows)
    if hole:
        c = flat[tris].mean(axis=1) - np.array([0.52, 0.47 * ny * h])
        tris = tris[(c ** 2).sum(axis=1) > (0.12 * ny * h) ** 2]
        used = np.zeros(xy.shape[0], bool)
        used[tris.reshape(-1)] = True
        tris = (np.cumsum(used) - 1)[tris]
        xy = xy[used]
    return np.ascontiguousarray(xy), np.ascontiguousarray(tris.astype(np.int32))


def _edges(tris, n_nodes):
    """Caller edges: unique (low, high) node pairs in lexicographic order; per half-edge its edge
    and its sign (+1 where the counter-clockwise triangle runs it low -> high)."""
    t = torch.as_tensor(tris, device="cuda").long()
    a, b = t.reshape(-1), t[:, [1, 2, 0]].reshape(-1)
    key, inv = torch.unique(torch.minimum(a, b) * n_nodes + torch.maximum(a, b), return_inverse=True)
    return torch.stack([key // n_nodes, key % n_nodes], dim=1), inv, torch.where(a < b, 1.0, -1.0).double()


def _line_source(xy, tris, x_s, h):
    """The soft vertical line source of the workloads, on interior edges near x = x_s."""
    e, inv, _ = _edges(tris, xy.shape[0])
    inside = (torch.bincount(inv, minlength=e.shape[0]) == 2).cpu().numpy()
    e = e.cpu().numpy()
    v = xy[e[:, 1]] - xy[e[:, 0]]
    ey = v[:, 1] / np.hypot(v[:, 0], v[:, 1])
    xm = 0.5 * (xy[e[:, 0], 0] + xy[e[:, 1], 0])
    ids = np.nonzero(inside & (np.abs(xm - x_s) < 4.5 * h) & (np.abs(ey) > 0))[0]
    return ids.astype(np.int32), ey[ids] * np.exp(-((xm[ids] - x_s) / (1.5 * h)) ** 2)


def _start(xy, tris, seed, n_edges, plasma):
    """Initial fields: a few low cavity modes in B, smooth E (and current, in a plasma)."""
    rng = np.random.default_rng(seed + 1)
    c = xy[tris].mean(axis=1)
    ly = xy[:, 1].max()
    B = sum(rng.uniform(-1, 1) * np.cos(p * math.pi * c[:, 0]) * np.cos(q * math.pi * c[:, 1] / ly)
            for p, q in ((1, 1), (2, 1), (3, 2)))
    s = np.arange(n_edges) / n_edges
    E = 0.3 * np.sin(2 * math.pi * (3 * s + rng.random()))
    j = 0.1 * np.cos(2 * math.pi * (2 * s + rng.random())) if plasma else None
    return E, B, j


def _pinned(a, dtype):
    return None if a is None else torch.tensor(np.asarray(a, dtype)).pin_memory().numpy()


def _density(xy, ly):
    r2 = (xy[:, 0] - 0.5) ** 2 + (xy[:, 1] - 0.5 * ly) ** 2
    return (0.8 * W0) ** 2 * np.exp(-r2 / (2 * 0.15 ** 2))


def _march_inputs(case, seed):
    xy, tris = _lattice(case["nx"], case["ny"], seed, case["hole"])
    h = 1.0 / case["nx"]
    src = _line_source(xy, tris, 0.35, h) if case["source"] else None
    dens = _density(xy, case["ny"] * h) if case["plasma"] else None
    return xy, tris, h, 0.15 * h, src, dens


def _batch_specs(case, seed):
    size = np.random.default_rng(case["meshes"])
    rng = np.random.default_rng(seed)
    out = []
    for k in range(case["meshes"]):
        n = math.exp(size.uniform(math.log(case["n_min"]), math.log(case["n_max"])))
        out.append(dict(nx=max(16, int(math.sqrt(n / 2))), seed=int(rng.integers(1 << 30)),
                        w0=2 * math.pi * float(rng.uniform(10, 30))))
    return out


def _corpus_sizes(case):
    rng = np.random.default_rng(case["meshes"])
    n = np.exp(rng.uniform(math.log(case["n_min"]), math.log(case["n_max"]), case["meshes"])).astype(np.int64)
    return np.concatenate([[0], np.cumsum(n)])


# --- what a program has in hand before the call -----------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    if kind == "march":
        xy, tris, h, dt, src, dens = _march_inputs(case, seed)
        blocked = case["tiles"] == "rings"
        tile = 2200 if case["depth"] > 8 else 2400      # the halo of so many rings fits the kernel
        m = ue.Mesh(xy, tris, **(dict(reorder=ue.UE_REORDER_GREEDY_RINGS, tile_tris=tile) if blocked else {}))
        if case["frame"]:
            m.frame_attach(case["frame"])
        opt = dict(dt_mode=ue.UE_DT_GIVEN, dt=dt, watchdog_every=case["watchdog"])
        if blocked:
            opt.update(variant=ue.UE_VARIANT_BLOCKED, block_depth=case["depth"])
        if case["fp64"]:
            opt["precision"] = ue.UE_PREC_FP64
        m.geometry_build(**opt)
        if src is not None:
            m.set_source(*src, W0, T0, TAU)
        if dens is not None:
            m.set_plasma(dens, 0.01 * W0)
        m.step_prepare()
        E, B, j = _start(xy, tris, seed, m.n_edges, case["plasma"])
        # fields travel as the benchmark moves them: pinned, in the product's precision; framed,
        # double precision and batched meshes move doubles
        dtype = np.float64 if case["frame"] or case["fp64"] else np.float32
        state = dict(kind=kind, m=m, f32=dtype is np.float32, steps=case["steps"], j=case["plasma"],
                     fields=[_pinned(a, dtype) for a in (E, B, j)],
                     out={k: _pinned(np.zeros(n), dtype) for k, n in
                          (("E", m.n_edges), ("B", m.n_tris), ("j", m.n_edges))})
        return state
    if kind == "batch":
        singles, E, B = [], [], []
        for sp in _batch_specs(case, seed):
            xy, tris = _lattice(sp["nx"], sp["nx"], sp["seed"], True)
            m = ue.Mesh(xy, tris, reorder=ue.UE_REORDER_GREEDY_RINGS, tile_tris=2200)
            m.geometry_build(dt_mode=ue.UE_DT_GIVEN, dt=0.15 / sp["nx"], variant=ue.UE_VARIANT_BLOCKED,
                             block_depth=case["depth"])
            m.set_source(*_line_source(xy, tris, 0.35, 1.0 / sp["nx"]), sp["w0"], T0, TAU)
            e, b, _ = _start(xy, tris, sp["seed"], m.n_edges, False)
            singles.append(m)
            E.append(e)
            B.append(b)
        bt = ue.batch_create(singles)
        for m in singles:
            m.close()
        bt.step_prepare()
        return dict(kind="march", m=bt, f32=False, steps=case["steps"], j=False,
                    fields=[_pinned(np.concatenate(E), np.float64), _pinned(np.concatenate(B), np.float64), None],
                    out={k: _pinned(np.zeros(n), np.float64) for k, n in (("E", bt.n_edges), ("B", bt.n_tris))})
    if kind in ("setup", "modes"):
        xy, tris = _lattice(case["nx"], case["ny"], seed, case["hole"])
        m = ue.Mesh(xy, tris)
        if kind == "modes":
            m.geometry_build(dt_mode=ue.UE_DT_GIVEN, dt=0.15 / case["nx"])
        return dict(kind=kind, m=m, case=case, seed=seed % 1000)
    if kind == "relax":
        rng = np.random.default_rng(seed)
        n = case["points"]
        side = np.linspace(0, 1, max(4, int(math.sqrt(n))))[:-1]
        z, o = np.zeros_like(side), np.ones_like(side)
        ring = np.concatenate([np.stack(p, axis=1) for p in ((side, z), (o, side), (1 - side, o), (z, 1 - side))])
        xy = np.concatenate([ring, rng.uniform(0.004, 0.996, size=(n, 2))])
        tris, _ = ue.triangulate(xy)
        return dict(kind=kind, xy=xy, tris=tris, case=case)
    # training: features of the corpus' triangles (the ranges rho_features gives), labels, weights
    off = _corpus_sizes(case)
    n, k = int(off[-1]), case["meshes"]
    g = torch.Generator(device="cuda").manual_seed(seed)
    X = torch.empty(n, 12, device="cuda")
    X[:, :3] = 1.05 + 0.25 * torch.randn(n, 3, device="cuda", generator=g)         # angles
    X[:, 3:6] = 0.42 + 0.2 * torch.randn(n, 3, device="cuda", generator=g)         # log edge lengths
    X[:, 6:9] = -0.2 + 0.35 * torch.randn(n, 3, device="cuda", generator=g)        # log dual lengths
    X[:, 9:] = 0.15 * torch.randn(n, 3, device="cuda", generator=g)                # log area ratios
    grade = torch.rand(k, device="cuda", generator=g).repeat_interleave(torch.as_tensor(np.diff(off), device="cuda"))
    base = 6.0 + 2.0 * grade + 0.3 * torch.randn(n, device="cuda", generator=g)
    p = torch.from_numpy(learned.load_weights()).cuda()
    new = lambda *s, dtype=torch.float32: torch.zeros(*s, dtype=dtype, device="cuda")  # noqa: E731
    return dict(kind=kind, X=X, base=base, off=torch.as_tensor(off, device="cuda"), p=p,
                target=7.5 + torch.randn(k, device="cuda", generator=g),
                m1=1e-3 * torch.randn(p.shape[0], device="cuda", generator=g), m2=new(p.shape[0]) + 1e-4,
                z=new(n), best=new(k), arg=new(k, dtype=torch.int64), dz=new(k), loss=new(k), grad=new(p.shape[0]),
                work=new(k, p.shape[0]))


# --- one pass ---------------------------------------------------------------------------------

def run(s):
    kind = s["kind"]
    if kind == "march":
        m = s["m"]
        (m.write_fields_f32 if s["f32"] else m.write_fields)(*s["fields"])
        m.set_step(0)
        m.step_n(s["steps"])
        E, B, j = (m.read_fields_f32 if s["f32"] else m.read_fields)(j=s["j"], out=s["out"])
        return (E, B, j) if s["j"] else (E, B)
    if kind == "setup":
        s["m"].geometry_build(power_iters=s["case"]["iters"], power_seed=s["seed"])
        dt, rho, _ = s["m"].get_dt()
        return np.array([dt, rho])
    if kind == "modes":
        return s["m"].modes(s["case"]["n_modes"], iters=s["case"]["iters"], seed=s["seed"], vectors=True)
    if kind == "relax":
        return ue.mesh_relax(s["xy"], s["tris"], s["case"]["iters"], flip_every=s["case"]["flip_every"])
    ue.mlp_forward(s["p"], s["X"], s["z"], bf16=True)
    ue.seg_argmax(s["z"], s["base"], s["off"], s["best"], s["arg"])
    ue.rho_loss(s["best"], s["target"], s["dz"], s["loss"])
    ue.mlp_backward(s["p"], s["X"], s["arg"], s["dz"], s["grad"], s["work"], bf16=True)
    p, m1, m2 = s["p"].clone(), s["m1"].clone(), s["m2"].clone()    # this epoch's weights are kept
    ue.adam(p, s["grad"], m1, m2, 5, lr=3e-3)
    return s["z"], s["best"], s["arg"], s["loss"], s["grad"], p, m1, m2


# --- what a pass cannot do without ----------------------------------------------------------------

def work(case):
    kind = case["kind"]
    if kind == "march":
        # the fields in and out of the device once, the mesh's tables and coefficients read once
        n_t = 2 * case["nx"] * case["ny"]
        n_e = 1.5 * n_t
        f = 8 if case["fp64"] else 4
        host = 8 if case["frame"] or case["fp64"] else 4
        per = n_e * (8 + f + (f if case["plasma"] else 0)) + n_t * (12 + f)
        flops = case["steps"] * (n_e * (3 + (5 if case["plasma"] else 0)) + 4 * n_t)
        return dict(bytes=per + 2 * host * (n_e * (2 if case["plasma"] else 1) + n_t), flops=flops)
    if kind == "batch":
        a, b = math.log(case["n_min"]), math.log(case["n_max"])
        n_t = case["meshes"] * (case["n_max"] - case["n_min"]) / (b - a)
        return dict(bytes=n_t * (1.5 * 12 + 16 + 2 * 8 * 2.5), flops=case["steps"] * n_t * (1.5 * 3 + 4))
    if kind == "setup":
        n_t = 2 * case["nx"] * case["ny"]
        return dict(bytes=n_t * (8 + 12 + 1.5 * 24 + 8 + 12), flops=case["iters"] * n_t * 10.0)
    if kind == "modes":
        n_t, m = 2 * case["nx"] * case["ny"], min(32, 2 * case["n_modes"])
        return dict(bytes=n_t * (12 + 1.5 * 16 + 8 + 8 * case["n_modes"]),
                    flops=case["iters"] * n_t * m * 8.0)
    if kind == "relax":
        n = case["points"]
        return dict(bytes=n * (32 + 24 + 24), flops=case["iters"] * n * 150.0)
    a, b = math.log(case["n_min"]), math.log(case["n_max"])
    n = case["meshes"] * (case["n_max"] - case["n_min"]) / (b - a)
    return dict(bytes=n * (48 + 4 + 4), flops=n * 2.0 * (12 * 64 + 64 * 64 + 64))


# --- the same results in 64 bits ------------------------------------------------------------------

class _Geometry:
    """Edges, R/L, lengths, dual lengths and areas of a mesh, in double precision on the GPU."""

    def __init__(self, xy, tris):
        self.t = torch.as_tensor(tris, device="cuda").long()
        self.xy = xy = torch.as_tensor(xy, device="cuda")
        self.e, self.inv, self.sgn = _edges(tris, xy.shape[0])
        n_e, n_t = self.e.shape[0], self.t.shape[0]
        p = xy[self.t]
        u, v = p[:, 1] - p[:, 0], p[:, 2] - p[:, 0]
        det = u[:, 0] * v[:, 1] - u[:, 1] * v[:, 0]
        self.S = 0.5 * det
        uu, vv = (u * u).sum(1), (v * v).sum(1)
        self.O = p[:, 0] + torch.stack([v[:, 1] * uu - u[:, 1] * vv, u[:, 0] * vv - v[:, 0] * uu], 1) / (2 * det)[:, None]
        w = xy[self.e[:, 1]] - xy[self.e[:, 0]]
        self.len = w.norm(dim=1)
        q = torch.arange(3, device="cuda")
        a, b, o = p[:, q], p[:, (q + 1) % 3], p[:, (q + 2) % 3]
        ua, ub = a - o, b - o
        cot = (ua * ub).sum(2) / (ua[..., 0] * ub[..., 1] - ua[..., 1] * ub[..., 0]).abs()
        self.d = 0.5 * self.len * torch.zeros(n_e, dtype=torch.float64, device="cuda").index_add_(0, self.inv, cot.reshape(-1))
        tri = torch.arange(n_t, device="cuda").repeat_interleave(3)
        self.R = torch.full((n_e,), n_t, device="cuda")      # n_t: no triangle
        self.L = self.R.clone()
        up = self.sgn > 0
        self.R[self.inv[up]] = tri[up]
        self.L[self.inv[~up]] = tri[~up]
        self.inside = (self.R < n_t) & (self.L < n_t)
        self.c = torch.where(self.inside, self.len / self.d, torch.zeros_like(self.d))

    def K(self, V):
        """K V = (1/S) sum_q s_q |e_q|/d_q (V_R - V_L), V [n_t, m]."""
        Vp = torch.cat([V, torch.zeros_like(V[:1])])
        g = self.c[:, None] * (Vp[self.R] - Vp[self.L])
        return (self.sgn[:, None] * g[self.inv]).reshape(-1, 3, V.shape[1]).sum(1) / self.S[:, None]


class _Frame:
    """Berenger split-field cells around the mesh, the mesh's outer edges among their sides."""

    def __init__(self, G, W, nx, ny, dt):
        h = 1.0 / nx
        self.W, self.NX, self.NY = W, nx + 2 * W, ny + 2 * W
        new = lambda *s: torch.zeros(*s, dtype=torch.float64, device="cuda")  # noqa: E731
        self.H, self.V = new(self.NY + 1, self.NX), new(self.NY, self.NX + 1)
        self.Bx, self.By = new(self.NY, self.NX), new(self.NY, self.NX)
        self.cell = torch.ones(self.NY, self.NX, dtype=torch.bool, device="cuda")
        self.cell[W:W + ny, W:W + nx] = False
        self.hm, self.vm = torch.zeros_like(self.H, dtype=torch.bool), torch.zeros_like(self.V, dtype=torch.bool)
        self.hm[1:-1] = self.cell[1:] & self.cell[:-1]
        self.vm[:, 1:-1] = self.cell[:, 1:] & self.cell[:, :-1]
        smax = 4 * math.log(1e6) / (2 * W * h)

        def ab(n, at, span, scale):
            x = (torch.arange(n, dtype=torch.float64, device="cuda") + at - W) * h
            s = smax * (torch.clamp(torch.maximum(-x, x - span * h), min=0) / (W * h)) ** 3
            return (1 - 0.5 * dt * s) / (1 + 0.5 * dt * s), scale / (1 + 0.5 * dt * s)
        self.aH, self.bH = (v[:, None] for v in ab(self.NY + 1, 0, ny, dt))
        self.aV, self.bV = ab(self.NX + 1, 0, nx, dt)
        self.ax, self.bx = ab(self.NX, 0.5, nx, dt / h ** 2)
        self.ay, self.by = (v[:, None] for v in ab(self.NY, 0.5, ny, dt / h ** 2))
        a, b = G.xy[G.e[:, 0]], G.xy[G.e[:, 1]]
        mid = 0.5 * (a + b)
        tol, ly = 1e-9, ny * h
        self.sides = []
        for ax, wall, nin in ((1, 0.0, 1.0), (1, ly, -1.0), (0, 0.0, 1.0), (0, 1.0, -1.0)):
            on = torch.nonzero(~G.inside & ((a[:, ax] - wall).abs() < tol) & ((b[:, ax] - wall).abs() < tol))[:, 0]
            tri = torch.minimum(G.R[on], G.L[on])
            c = (G.O[tri, ax] - wall) * nin + 0.5 * h
            along = 1 - ax
            k = W + torch.floor(mid[on, along] / h).long()
            out = torch.full_like(k, W - 1 if wall == 0.0 else W + (ny if ax == 1 else nx))      # the frame cell's row or column
            line = torch.full_like(k, W if wall == 0.0 else W + (ny if ax == 1 else nx))         # the side's row or column
            I, J = (k, out) if ax == 1 else (out, k)
            ahead = torch.sign(b[on, along] - a[on, along])
            right = (G.R[on] == tri).double() * 2 - 1                                            # the triangle is R: +1
            self.sides.append((on, tri, J, I, right, dt * G.len[on] / c, ahead, ax, k, line))

    def e_half(self, U, B):
        F = self.Bx + self.By
        for on, tri, J, I, right, c, ahead, ax, k, line in self.sides:
            U[on] += c * right * (B[tri] - F[J, I])
        self.H[1:-1] = torch.where(self.hm[1:-1], self.aH[1:-1] * self.H[1:-1] + self.bH[1:-1] * (F[1:] - F[:-1]), self.H[1:-1])
        self.V[:, 1:-1] = torch.where(self.vm[:, 1:-1], self.aV[1:-1] * self.V[:, 1:-1] + self.bV[1:-1] * (F[:, :-1] - F[:, 1:]), self.V[:, 1:-1])

    def b_half(self, U):
        for on, tri, J, I, right, c, ahead, ax, k, line in self.sides:
            if ax == 1:
                self.H[line, k] = ahead * U[on]
            else:
                self.V[k, line] = ahead * U[on]
        self.Bx = torch.where(self.cell, self.ax * self.Bx - self.bx * (self.V[:, 1:] - self.V[:, :-1]), self.Bx)
        self.By = torch.where(self.cell, self.ay * self.By - self.by * (self.H[:-1] - self.H[1:]), self.By)


def _march64(xy, tris, dt, steps, E, B, j, src, w0, dens, nu, frame):
    G = _Geometry(xy, tris)
    dev = lambda a: torch.as_tensor(np.asarray(a, np.float64), device="cuda")  # noqa: E731
    fr = _Frame(G, *frame, dt) if frame else None
    outer = torch.zeros_like(G.inside)
    if fr:
        for s in fr.sides:
            outer[s[0]] = True
    live = (G.inside | outer).double()
    U = dev(E) * G.len * live
    Bp = torch.cat([dev(B), torch.zeros(1, dtype=torch.float64, device="cuda")])
    n_t = G.t.shape[0]
    cB = dt / G.S
    if dens is not None:
        nb = dev(dens)[G.e].mean(1)
        pa, pb = (1 - 0.5 * nu * dt) / (1 + 0.5 * nu * dt), dt * nb / (1 + 0.5 * nu * dt)
        inside = G.inside.double()
        J = dev(j) * G.len * inside
    if src is not None:
        ids, amp = torch.as_tensor(src[0], device="cuda").long(), dev(src[1])
        amp = dt * G.len[ids] * amp
    for n in range(steps):
        if dens is not None:
            J = (pa * J + pb * U) * inside
        U += dt * G.c * (Bp[G.R] - Bp[G.L])
        if dens is not None:
            U -= dt * J
        if src is not None:
            t = (n + 0.5) * dt
            U[ids] += amp * math.sin(w0 * t) * math.exp(-((t - T0) / TAU) ** 2)
        if fr:
            fr.e_half(U, Bp)
        Bp[:n_t] -= cB * (G.sgn * U[G.inv]).reshape(-1, 3).sum(1)
        if fr:
            fr.b_half(U)
    out = [U / G.len * live, Bp[:n_t]]
    return out + [J / G.len] if dens is not None else out


def _splitmix(x):
    with np.errstate(over="ignore"):
        z = x + np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    return torch.as_tensor((z >> np.uint64(11)).astype(np.float64) * 2.0 ** -53 * 2 - 1, device="cuda")


def exact(case, seed):
    kind = case["kind"]
    if kind == "march":
        xy, tris, h, dt, src, dens = _march_inputs(case, seed)
        n_e = _edges(tris, xy.shape[0])[0].shape[0]
        start = _start(xy, tris, seed, n_e, case["plasma"])
        if not (case["frame"] or case["fp64"]):
            start = [None if a is None else a.astype(np.float32) for a in start]
        frame = (case["frame"], case["nx"], case["ny"]) if case["frame"] else None
        return _march64(xy, tris, dt, case["steps"], *start, src, W0, dens, 0.01 * W0, frame)
    if kind == "batch":
        E, B = [], []
        for sp in _batch_specs(case, seed):
            xy, tris = _lattice(sp["nx"], sp["nx"], sp["seed"], True)
            h = 1.0 / sp["nx"]
            n_e = _edges(tris, xy.shape[0])[0].shape[0]
            e, b, _ = _start(xy, tris, sp["seed"], n_e, False)
            e, b = _march64(xy, tris, 0.15 * h, case["steps"], e, b, None,
                            _line_source(xy, tris, 0.35, h), sp["w0"], None, 0.0, None)
            E.append(e)
            B.append(b)
        return torch.cat(E), torch.cat(B)
    if kind in ("setup", "modes"):
        xy, tris = _lattice(case["nx"], case["ny"], seed, case["hole"])
        G = _Geometry(xy, tris)
        n_t, m = tris.shape[0], 1 if kind == "setup" else min(32, 2 * case["n_modes"])
        key = np.uint64(seed % 1000 << 32) + np.arange(n_t * m, dtype=np.uint64)
        V = _splitmix(key).reshape(n_t, m)
        if kind == "setup":
            v = V / (G.S[:, None] * V * V).sum().sqrt()
            for _ in range(case["iters"]):
                w = G.K(v)
                rho = math.sqrt(float((G.S[:, None] * v * w).sum()))
                v = w / (G.S[:, None] * w * w).sum().sqrt()
            return np.array([1.0 / rho, rho])

        def orth(W):
            for _ in range(2):
                R = torch.linalg.cholesky((W.T @ (G.S[:, None] * W)).cpu(), upper=True).to(W.device)
                W = W @ torch.linalg.inv(R)
            return W
        V = orth(V)
        for _ in range(case["iters"]):
            V = orth(G.K(V))
        lam = torch.linalg.eigvalsh((V.T @ (G.S[:, None] * G.K(V))).cpu())
        return lam.flip(0)[:case["n_modes"]].clamp(min=0).sqrt(), None
    if kind == "train":
        s = prepare(case, seed)
        W1, b1, W2, b2, w3, b3 = torch.split(s["p"].double(), [768, 64, 4096, 64, 64, 1])
        z = torch.cat([torch.relu(torch.relu(x.double() @ W1.reshape(64, 12).T + b1) @ W2.reshape(64, 64).T + b2) @ w3 + b3
                       for x in s["X"].split(1 << 20)])
        return z, None, None, None, None, None, None, None
    return None
