"""The work that a program has this library do, as measurable cases.

Every case calls the public entry points of `paper_2011_14998_gb300` on inputs made from a seed:

  solve   J of one model through `Context.solve_J` into a device tensor
  batch   J of one or several models through `Context.solve_J_batch`
  host    the whole step of a program that gets a new model in host memory: load the mesh, lines and
          rays, solve, read J back, free the model
  rays    a new adaptive ray set, read back, and the traced lists of some origins
  train   training of the reduction network
  reduce  one mesh reduction: features, the learned weighted thinning and the plain criterion

`exact` restates the method in torch, in 64 bits, from its definition.
"""
import math

import numpy as np
import torch

import paper_2011_14998_gb300 as mgx
from paper_2011_14998_gb300.learned import delaunay_neighbours

DEV = "cuda:0"
NU0 = 115.2712018e9  # Hz; only ratios of line centres enter
C_KMS = 299792.458
PRECISION = {"fp64": mgx.MGX_FP64, "fp32": mgx.MGX_FP32, "dt64": mgx.MGX_FP32_DT64}


def listed():
    wind = dict(mesh="wind", lines=1, bins=50, l_min=2, l_max=2, precision="fp32", order=2)
    return [
        # the smallest call: a reduced test mesh, adaptive rays; latency and an idle chip count
        dict(wind, name="tiny_wind_fp32", kind="solve", n=400, bins=20, l_min=0, l_max=2),
        # the closed-form check everybody runs first: homogeneous 16^3 cube, plain double-precision form
        dict(name="grid_fp64", kind="solve", mesh="grid", n=4096, lines=1, bins=31, l_min=0, l_max=0,
             precision="fp64", order=2),
        # the plain double-precision form on a stellar wind, as a reference solution is made
        dict(wind, name="wind_fp64", kind="solve", n=4001, precision="fp64"),
        # single-precision bulk with double-precision increments and pivots
        dict(wind, name="wind_dt64", kind="solve", n=6007, precision="dt64"),
        # the fourth-order scheme in single precision
        dict(wind, name="wind_hermitian", kind="solve", n=12000, order=4),
        # an ordinary repeated call of the per-model form: two lines on an adaptively refined octree
        dict(name="octree_fp32", kind="solve", mesh="octree", n=20000, lines=2, bins=64, l_min=0, l_max=3,
             precision="fp32", order=2),
        # the benchmark's step: the 50 000-point wind, ray sets rebuilt, replayed from a CUDA graph
        dict(wind, name="wind50k_graph", kind="batch", n=50000, models=1, graph=True),
        # several uneven models in one planned launch, four lines each, a new plan per call
        dict(name="mixed_batch", kind="batch", mesh="mixed", n=3500, models=5, lines=4, bins=100, l_min=0, l_max=3,
             precision="fp32", order=2, graph=False),
        # the end-to-end step from pinned host memory to J in host memory
        dict(wind, name="wind_host", kind="host", n=20000),
        # ray sets of the paper's range (levels 1 to 4, 10^4 sampled directions a point), inspected lists
        dict(name="rays_trace", kind="rays", mesh="octree", n=30000, l_min=1, l_max=4, origins=100),
        # training of the reduction network on one model's dropped points, default batch
        dict(name="train", kind="train", n=20011, batch=256, epochs=2),
        # one reduction of a large octree, learned and plain
        dict(name="reduce", kind="reduce", mesh="octree", n=200000, keep=0.2, alpha=2.0),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["solve", "solve", "solve", "batch", "batch", "host", "rays", "train", "reduce"])
    levels = rng.choice([(0, 0), (1, 1), (2, 2), (0, 2), (0, 3), (1, 3)])
    c = dict(kind=kind, l_min=levels[0], l_max=levels[1])
    if kind in ("solve", "batch", "host"):
        c.update(mesh=rng.choice(["wind", "wind", "octree", "grid"]), lines=rng.choice([1, 1, 1, 2, 3, 4]),
                 bins=size(7, 100), precision="fp32", order=2)
    if kind == "solve":
        c["precision"] = rng.choice(["fp32", "fp32", "fp64", "dt64"])
        if c["precision"] != "dt64" and c["mesh"] != "octree":
            c["order"] = rng.choice([2, 2, 4])
        most = 12000 if c["precision"] == "fp32" else 1500
        c.update(n=size(60, most), lines=min(c["lines"], 2))
    elif kind == "batch":
        c.update(n=size(200, 5000), models=rng.choice([1, 3, 6]), graph=rng.random() < 0.5)
        if c["models"] > 1:
            c["mesh"] = "mixed"
    elif kind == "host":
        c.update(n=size(500, 12000))
    elif kind == "rays":
        levels = rng.choice([(0, 2), (0, 3), (1, 3), (1, 4)])
        c.update(mesh=rng.choice(["wind", "octree"]), n=size(2000, 20000), l_min=levels[0], l_max=levels[1],
                 origins=size(10, 300))
    elif kind == "train":
        c = dict(kind=kind, n=size(1000, 30000), batch=rng.choice([64, 256, 1000]), epochs=rng.choice([1, 2]))
    else:
        c = dict(kind=kind, mesh="octree", n=size(5000, 200000), keep=round(rng.uniform(0.05, 0.5), 3),
                 alpha=rng.choice([1.0, 2.0, 3.0]))
    return c


# ------------------------------------------------------------------ inputs
def _csr(n, a, b):
    """Symmetric neighbour lists, rows ascending, of the pairs (a, b) (device tensors)."""
    key = torch.unique(torch.cat([a * n + b, b * n + a]))
    src, dst = torch.div(key, n, rounding_mode="floor"), key % n
    off = torch.zeros(n + 1, dtype=torch.int64, device=key.device)
    off[1:] = torch.cumsum(torch.bincount(src, minlength=n), 0)
    return off.cpu().numpy(), dst.to(torch.int32).cpu().numpy()


_HALF26 = [(i, j, k) for i in (-1, 0, 1) for j in (-1, 0, 1) for k in (-1, 0, 1) if (i, j, k) > (0, 0, 0)]


def _touching(cells, n):
    """Neighbour lists of the ids on a 3-D voxel array whose voxels touch (26-neighbourhood)."""
    g = cells.shape
    keys = []
    for d in _HALF26:
        sa = tuple(slice(max(0, -x), w - max(0, x)) for x, w in zip(d, g))
        sb = tuple(slice(max(0, x), w - max(0, -x)) for x, w in zip(d, g))
        a, b = cells[sa].reshape(-1).long(), cells[sb].reshape(-1).long()
        m = a != b
        keys.append(torch.unique(torch.minimum(a, b)[m] * n + torch.maximum(a, b)[m]))
    key = torch.cat(keys)
    return _csr(n, torch.div(key, n, rounding_mode="floor"), key % n)


def _widths(T):
    return np.sqrt(2.0 * 1.380649e-23 * T / (28.0 * 1.66053906660e-27)) / 1e3  # thermal, km/s


def _lines(m, chi, S, lines, ratio, cont=1e-4):
    n = len(chi)
    chi0 = chi[:, None] * ratio ** np.arange(lines)[None, :]
    chi_c = cont * chi
    m.update(nu0=NU0 * (1.0 + 1e-3 * np.arange(lines)), chi0=np.ascontiguousarray(chi0),
             eta0=np.ascontiguousarray(chi0 * S[:, None]), chi_c=chi_c, eta_c=chi_c * S)
    assert m["dvw"].shape == (n,)
    return m


def _modes(pos, rng, rms, box):
    """Smooth random velocity: 64 Fourier modes of wavelengths box/8 to box."""
    k = rng.normal(size=(64, 3))
    k /= np.linalg.norm(k, axis=1, keepdims=True)
    lam = box * np.exp(rng.uniform(np.log(1 / 8), 0.0, 64))
    amp = rng.normal(size=(64, 3)) * (lam / box)[:, None]
    ph = rng.uniform(0.0, 2 * np.pi, 64)
    p = torch.from_numpy(pos).to(DEV)
    t = torch.from_numpy(k * (2 * np.pi / lam)[:, None]).to(DEV)
    v = (torch.cos(p @ t.T + torch.from_numpy(ph).to(DEV)) @ torch.from_numpy(amp).to(DEV)).cpu().numpy()
    v -= v.mean(0)
    return v * (rms / v.std(0))


def _wind(n, lines, seed):
    """Stellar wind: r log-uniform in [1, 100], n ~ r^-2, 15 km/s beta law, Delaunay neighbours."""
    rng = np.random.default_rng([seed, 1])
    r = np.exp(rng.uniform(0.0, np.log(100.0), n))
    mu, ph = rng.uniform(-1.0, 1.0, n), rng.uniform(0.0, 2.0 * np.pi, n)
    st = np.sqrt(1.0 - mu * mu)
    rhat = np.stack([st * np.cos(ph), st * np.sin(ph), mu], axis=1)
    pos = np.ascontiguousarray(rhat * r[:, None])
    off, nbr = delaunay_neighbours(pos)
    T = 2000.0 * r ** -0.7
    m = dict(pos=pos, vel=np.ascontiguousarray(rhat * (15.0 * np.sqrt(1.0 - 1.0 / r))[:, None]), nbr_off=off,
             nbr_idx=nbr, dvw=_widths(T), rho=r ** -2.0, T=T)
    return _lines(m, 10.0 / 0.99 * m["rho"], T / 2000.0, lines, 0.5)


def _grid(n, lines, seed):
    """Static homogeneous cube, 26 neighbours; the seed sets its opacity and source function."""
    k = max(3, int(round(n ** (1 / 3))))
    rng = np.random.default_rng([seed, 2])
    g = np.arange(k, dtype=np.float64) / (k - 1)
    pos = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)
    off, nbr = _touching(torch.arange(k ** 3, device=DEV).reshape(k, k, k), k ** 3)
    one = np.ones(k ** 3)
    m = dict(pos=pos, vel=np.zeros((k ** 3, 3)), nbr_off=off, nbr_idx=nbr, dvw=one, rho=one, T=2000.0 * one)
    return _lines(m, rng.uniform(3.0, 8.0) * one, rng.uniform(0.5, 1.5) * one, lines, 0.5, 1e-10)


def _octree(n, lines, seed, box=1000.0):
    """Octree leaves refined around three clumps of contrast 10^3 in a turbulent 2 km/s field.  The
    clumps' layout goes with n (so every seed has as many leaves), their orientation and the
    fields with the seed."""
    lay, rng = np.random.default_rng([n, 3]), np.random.default_rng([seed, 3])
    cen, sig = lay.uniform(-0.3 * box, 0.3 * box, (3, 3)), lay.uniform(30.0, 80.0, 3)
    hi = max(5, min(7, int(np.log2(n) / 3) + 3))
    lo = 2 if n < 1500 else 3

    def density(x):
        return 1.0 + 999.0 * np.exp(-((x[:, None] - cen) ** 2).sum(-1) / (2 * sig * sig)).sum(-1)

    def leaves(thr):
        ijk = np.stack(np.meshgrid(*([np.arange(2 ** lo)] * 3), indexing="ij"), -1).reshape(-1, 3)
        out = []
        for l in range(lo, hi + 1):
            h = box / 2 ** l
            c0 = -box / 2 + ijk * h
            near = np.clip(cen[None], c0[:, None], c0[:, None] + h)
            peak = 1.0 + 999.0 * np.exp(-((near - cen) ** 2).sum(-1) / (2 * sig * sig)).sum(-1)
            split = peak > thr * 2.0 ** (l - lo) if l < hi else np.zeros(len(ijk), bool)
            out.append(np.concatenate([np.full((int((~split).sum()), 1), l), ijk[~split]], 1))
            kid = np.array([(a, b, c) for a in (0, 1) for b in (0, 1) for c in (0, 1)])
            ijk = (2 * ijk[split][:, None] + kid).reshape(-1, 3)
            if len(ijk) > 4 * n + 64:
                return None  # far too many already
        return np.concatenate(out)

    t0, t1, best = 1e-3, 1e3, None
    for _ in range(22):  # the leaf count falls with the threshold
        thr = math.sqrt(t0 * t1)
        lv = leaves(thr)
        if lv is None or len(lv) > n:
            t0 = thr
        else:
            t1, best = thr, lv
    lv = best if best is not None else leaves(1e3)
    n = len(lv)
    cells = torch.empty((2 ** hi,) * 3, dtype=torch.int32, device=DEV)
    ids = torch.arange(n, dtype=torch.int32, device=DEV)
    for l in range(lo, hi + 1):
        sel = torch.from_numpy(np.where(lv[:, 0] == l)[0]).to(DEV)
        s = 2 ** (hi - l)
        v = cells.view(2 ** l, s, 2 ** l, s, 2 ** l, s).permute(0, 2, 4, 1, 3, 5)
        i, j, k = torch.from_numpy(lv[:, 1:]).to(DEV)[sel].unbind(1)
        v[i, j, k] = ids[sel][:, None, None, None].expand(-1, s, s, s)
    off, nbr = _touching(cells, n)
    pos = -box / 2 + (lv[:, 1:] + 0.5) * (box / 2.0 ** lv[:, :1])
    rho = density(pos) * rng.uniform(0.8, 1.25)
    pos = pos[:, rng.permutation(3)] * rng.choice([-1.0, 1.0], 3)
    T = 1000.0 * rho ** -0.2
    m = dict(pos=np.ascontiguousarray(pos), vel=_modes(pos, rng, 2.0, box), nbr_off=off, nbr_idx=nbr, dvw=_widths(T),
             rho=rho, T=T)
    return _lines(m, rho / box, T / 1000.0, lines, 0.1)


def _model(case, seed, mesh=None, n=None):
    mesh = mesh or case["mesh"]
    m = {"wind": _wind, "grid": _grid, "octree": _octree}[mesh](n or case["n"], case.get("lines", 1), seed)
    n = len(m["pos"])
    rng = np.random.default_rng([seed, 4])
    smp = np.arange(n) if n <= 10000 else np.sort(rng.choice(n, 10000, replace=False))
    m.update(n_freq=case.get("bins", 50), x_span=4.0, l_min=case.get("l_min", 0), l_max=case.get("l_max", 0),
             sample=smp.astype(np.int32))
    return m


def _models(case, seed):
    if case.get("mesh") != "mixed":
        return [_model(case, seed + 1000 * k) for k in range(case.get("models", 1))]
    rng = np.random.default_rng([case["n"], 5])  # sizes spread over a factor of eight, generators in turn
    sizes = (case["n"] * np.exp(rng.uniform(-math.log(8) / 2, math.log(8) / 2, case["models"]))).astype(int)
    return [_model(case, seed + 1000 * k, ("grid", "wind", "octree")[k % 3], max(60, int(s)))
            for k, s in enumerate(sizes)]


def _theta(seed):
    """He-normal initial parameters of the 8-64-64-1 network."""
    rng = np.random.default_rng([seed, 6])
    return np.concatenate([rng.normal(0, 0.5, 512), np.zeros(64), rng.normal(0, math.sqrt(2 / 64), 4096), np.zeros(64),
                           rng.normal(0, 0.125, 64), [-1.5]]).astype(np.float32)


def _training_set(case, seed):
    """Standardised features and log10 errors with the spread of a real set."""
    rng = np.random.default_rng([seed, 7])
    X = rng.normal(size=(case["n"], 8))
    y = -1.5 + 0.4 * X[:, 0] + 0.3 * np.tanh(X[:, 1]) * X[:, 2] + 0.2 * np.abs(X[:, 4]) + rng.normal(0, 0.3, case["n"])
    return X.astype(np.float32), y.astype(np.float32)


def prepare(case, seed):
    ctx = mgx.Context(0)
    st = dict(case=case, ctx=ctx)
    kind = case["kind"]
    if kind == "train":
        st["X"], st["y"] = _training_set(case, seed)
        st["theta"], st["shuffle"] = _theta(seed), seed
        return st
    models = _models(case, seed)
    if kind == "host":  # a program that streams models in keeps them in pinned host memory
        m = {k: torch.from_numpy(v).pin_memory() if isinstance(v, np.ndarray) else v for k, v in models[0].items()}
        m["nu0"] = models[0]["nu0"]
        st["model"] = m
        st["J"] = torch.empty((len(models[0]["pos"]), case["lines"] * case["bins"]), dtype=torch.float64).pin_memory()
        return st
    if kind == "reduce":
        m = models[0]
        st["mid"], st["rho"], st["T"], st["seed"] = ctx.load(m, rays=False), m["rho"], m["T"], seed
        mgx.mgx_mlp_set_params(ctx.ptr, _theta(seed))
        X = mgx.mgx_mlp_features(ctx.ptr, st["mid"], m["rho"], m["T"])
        st["mean"], st["std"] = X.mean(0), np.maximum(X.std(0), 1e-6)
        return st
    if kind == "rays":
        m = models[0]
        st["mid"], st["sample"] = ctx.load(m, rays=False), m["sample"]
        st["lists"] = _lists(case, len(m["pos"]))
        return st
    st["mids"] = [ctx.load(m) for m in models]
    st["outs"] = [torch.empty((len(m["pos"]), case["lines"] * case["bins"]), dtype=torch.float64, device=DEV)
                  for m in models]
    return st


def _lists(case, n):
    """The inspecting program's own buffers for the traced lists: ids, distances, velocities."""
    cap = int(2 * _pairs(case["l_min"], case["l_max"]) * min(case["origins"], n) * (4 * n ** (1 / 3) + 8))
    return np.zeros(cap, np.int32), np.zeros(cap), np.zeros(cap)


def run(st):
    case, ctx = st["case"], st["ctx"]
    kind = case["kind"]
    if kind == "solve":
        return ctx.solve_J(st["mids"][0], precision=PRECISION[case["precision"]], out=st["outs"][0],
                           order=case["order"])
    if kind == "batch":
        flags = mgx.MGX_BATCH_RAYS | (mgx.MGX_BATCH_GRAPH if case["graph"] else 0)
        return ctx.solve_J_batch(st["mids"], precision=PRECISION[case["precision"]], outs=st["outs"], flags=flags)
    if kind == "host":
        mid = ctx.load(st["model"])
        ctx.solve_J_batch([mid], precision=PRECISION[case["precision"]], outs=[st["J"]], flags=mgx.MGX_BATCH_RAYS)
        ctx.free(mid)
        return st["J"]
    if kind == "rays":
        ctx.set_rays(st["mid"], case["l_min"], case["l_max"], st["sample"])
        rays = ctx.rays(st["mid"])
        off, idx, Z, delta = ctx.trace(st["mid"], 0, min(case["origins"], len(rays)), with_delta=True)
        for buf, got in zip(st["lists"], (idx, Z, delta)):
            buf[:len(got)] = got
        return dict(rays=rays.view(np.int32), off=off, idx=st["lists"][0], Z=st["lists"][1], delta=st["lists"][2])
    if kind == "train":
        mgx.mgx_mlp_set_params(ctx.ptr, st["theta"])
        losses = mgx.mgx_mlp_train(ctx.ptr, st["X"], st["y"], case["epochs"], case["batch"], 2e-3, st["shuffle"])
        return dict(losses=losses, theta=mgx.mgx_mlp_get_params(ctx.ptr))
    X = mgx.mgx_mlp_features(ctx.ptr, st["mid"], st["rho"], st["T"])
    Xs = ((X - st["mean"]) / st["std"]).astype(np.float32)
    keep, kept, scale = mgx.mgx_reduce_mesh_learned_weighted(ctx.ptr, st["mid"], Xs, case["keep"], case["alpha"],
                                                             st["seed"])
    Gf, L, ell, plain, n_plain = ctx.reduce_mesh(st["mid"], st["rho"], 1.0, 2.15, 0.21, st["seed"])
    return dict(X=X, keep=keep, kept=kept, scale=scale, Gf=Gf, L=L, ell=ell, plain=plain, n_plain=n_plain)


# ------------------------------------------------------------------ what a pass cannot do without
def _pairs(l_min, l_max):
    left, out = 6 * 4 ** l_min, 0
    for _ in range(l_min, l_max):  # the top half of the candidate pairs is refined at each level
        out += left - left // 2
        left = 4 * (left // 2)
    return out + left


def work(case):
    kind = case["kind"]
    if kind == "train":  # forward 2 (8 64 + 64 64 + 64) flops a row, backward twice that
        return dict(bytes=case["n"] * 36 + 8 * 4801, flops=case["epochs"] * case["n"] * 6 * (8 * 64 + 64 * 64 + 64))
    n = case["n"] * case.get("models", 1)
    deg = 16 if case["mesh"] == "wind" else 26
    if kind == "reduce":
        return dict(bytes=n * (4 * deg + 48 + 64 + 16 + 2 * 32 + 1 + 25), flops=n * (deg * 30 + 2 * 4672))
    pairs = _pairs(case["l_min"], case["l_max"])
    mesh = n * (48 + 8 + 4 * deg)
    if kind == "rays":  # one direction test of about 30 flops a sampled point, then the lists of the origins
        pts = 2 * pairs * case["origins"] * 0.7 * case["n"] ** (1 / 3)
        return dict(bytes=mesh + 4 * n * pairs + 20 * pts, flops=n * min(case["n"], 10000) * 30 + pts * deg * 20)
    # velocity samples of a pair line: as many as its points or more, growing with the mesh's resolution
    samples = {"grid": 0.8, "wind": 7.5, "octree": 9.0, "mixed": 6.0}[case["mesh"]] * case["n"] ** (1 / 3)
    nb = case["lines"] * case["bins"]
    return dict(bytes=mesh + n * 8 * (3 + 2 * case["lines"] + nb) + 4 * n * pairs,
                flops=n * pairs * nb * samples * (14 + 9 * case["lines"]))


# ------------------------------------------------------------------ the method in 64 bits, in torch
def _pix2vec(l, p):
    """Centres of nested HEALPix pixels p (numpy) of level l."""
    ns = 1 << l
    f, q = p >> (2 * l), p & (ns * ns - 1)
    x, y = np.zeros_like(q), np.zeros_like(q)
    for b in range(l):
        x |= ((q >> (2 * b)) & 1) << b
        y |= ((q >> (2 * b + 1)) & 1) << b
    row, col = np.array([2] * 4 + [3] * 4 + [4] * 4)[f], np.array([1, 3, 5, 7, 0, 2, 4, 6, 1, 3, 5, 7])[f]
    jr = row * ns - x - y - 1
    nr = np.where(jr < ns, jr, np.where(jr > 3 * ns, 4 * ns - jr, ns))
    z = np.where(jr < ns, 1.0 - nr * nr / (3.0 * ns * ns),
                 np.where(jr > 3 * ns, nr * nr / (3.0 * ns * ns) - 1.0, 2.0 * (2 * ns - jr) / (3.0 * ns)))
    shift = np.where((jr < ns) | (jr > 3 * ns), 0, (jr - ns) & 1)
    jp = (col * nr + x - y + 1 + shift) // 2
    jp = np.where(jp > 4 * nr, jp - 4 * nr, np.where(jp < 1, jp + 4 * nr, jp))
    phi = (2 * jp - 1 - shift) * np.pi / (4.0 * nr)
    s = np.sqrt((1.0 - z) * (1.0 + z))
    return np.stack([s * np.cos(phi), s * np.sin(phi), z], -1)


def _vec2pix(l, d):
    """Nested pixels of level l that hold the directions d [..., 3] (torch, 64 bits)."""
    ns = 1 << l
    z = d[..., 2] / torch.sqrt((d[..., 0] * d[..., 0] + d[..., 1] * d[..., 1]) + d[..., 2] * d[..., 2])
    t = torch.atan2(d[..., 1], d[..., 0]) * (2 / math.pi)
    t = torch.where(t < 0, t + 4.0, t)
    t = torch.where(t >= 4.0, t - 4.0, t)
    c1, c2 = ns * (0.5 + t), ns * (0.75 * z)
    asc, dsc = (c1 - c2).long(), (c1 + c2).long()
    fa, fd = asc >> l, dsc >> l
    face = torch.where(fa == fd, fa | 4, torch.where(fa < fd, fa, fd + 8))
    x, y = dsc & (ns - 1), ns - 1 - (asc & (ns - 1))
    q = torch.clamp(t.long(), max=3)
    w = ns * torch.sqrt(3.0 * (1.0 - z.abs()))
    a = torch.clamp(((t - q) * w).long(), max=ns - 1)
    b = torch.clamp(((1.0 - (t - q)) * w).long(), max=ns - 1)
    cap, north = z.abs() > 2.0 / 3.0, z >= 0
    face = torch.where(cap, torch.where(north, q, q + 8), face)
    x = torch.where(cap, torch.where(north, ns - 1 - b, a), x)
    y = torch.where(cap, torch.where(north, ns - 1 - a, b), y)
    p = face << (2 * l)
    for k in range(l):
        p = p + (((x >> k) & 1) << (2 * k)) + (((y >> k) & 1) << (2 * k + 1))
    return p


def _antipodes(l):
    p = np.arange(12 * 4 ** l)
    return _vec2pix(l, torch.from_numpy(-_pix2vec(l, p))).numpy()


def _rayset(m):
    """Pair directions [n, pairs, 3] and weights [n, pairs] of a model's ray set, pairs ascending."""
    n, lo, hi = len(m["pos"]), m["l_min"], m["l_max"]
    pos = torch.from_numpy(m["pos"]).to(DEV)
    p0 = np.arange(12 * 4 ** lo)
    first = p0[p0 < _antipodes(lo)]
    cand = torch.from_numpy(first).to(DEV).expand(n, -1)
    counts = None
    if lo < hi:
        npix, smp = 12 * 4 ** hi, torch.from_numpy(m["sample"]).long().to(DEV)
        counts = torch.zeros(n * npix, dtype=torch.int64, device=DEV)
        step = max(1, 20_000_000 // max(1, len(smp)))
        for o in range(0, n, step):
            d = pos[smp][None] - pos[o:o + step, None]
            own = torch.arange(o, min(n, o + step), device=DEV)
            ok = (smp[None] != own[:, None]) & (d != 0).any(-1)
            counts += torch.bincount((_vec2pix(hi, d) + own[:, None] * npix)[ok], minlength=n * npix)
        counts = counts.view(n, npix)
    done = []
    for l in range(lo, hi):
        anti = torch.from_numpy(_antipodes(l)).to(DEV)
        h = counts.view(n, 12 * 4 ** l, -1).sum(-1)
        score = torch.gather(h, 1, cand) + torch.gather(h, 1, anti[cand])
        order = torch.argsort(-score * (12 * 4 ** l) + cand, dim=1)  # by count, ties to the smaller pixel
        half = cand.shape[1] // 2
        cand_sorted = torch.gather(cand, 1, order)
        done.append((l, cand_sorted[:, half:]))
        kids = (4 * cand_sorted[:, :half, None] + torch.arange(4, device=DEV)).reshape(n, -1)
        anti = torch.from_numpy(_antipodes(l + 1)).to(DEV)
        cand = torch.minimum(kids, anti[kids])
    done.append((hi, cand))
    key = torch.sort(torch.cat([c + (l << 28) for l, c in done], 1), 1)[0]
    lev, pix = key >> 28, key & 0x0FFFFFFF
    table = torch.from_numpy(np.concatenate([_pix2vec(l, np.arange(12 * 4 ** l)) for l in range(hi + 1)])).to(DEV)
    return table[4 * (4 ** lev - 1) + pix], 2.0 / (12.0 * 4.0 ** lev.double())


def _trace(m, o, d):
    """Half-rays from origins o [H] along d [H, 3]: lengths and point ids [H, longest], nearest first."""
    off = torch.from_numpy(m["nbr_off"]).to(DEV)
    idx, pos = torch.from_numpy(m["nbr_idx"]).long().to(DEV), torch.from_numpy(m["pos"]).to(DEV)
    deg = off[1:] - off[:-1]
    H = len(o)
    cur, zc, act = o.clone(), torch.zeros(H, dtype=torch.float64, device=DEV), torch.arange(H, device=DEV)
    cnt, cols = torch.zeros(H, dtype=torch.int64, device=DEV), []
    while len(act):
        nxt, zn_ = torch.full_like(act, -1), torch.zeros(len(act), dtype=torch.float64, device=DEV)
        step = max(1, 12_000_000 // max(1, int(deg.max())))
        for s in range(0, len(act), step):
            a = act[s:s + step]
            k = torch.arange(int(deg[cur[a]].max()), device=DEV)
            has = k[None] < deg[cur[a]][:, None]
            nb = idx[torch.where(has, off[cur[a]][:, None] + k[None], 0)]
            x, da = pos[nb] - pos[o[a]][:, None], d[a][:, None]
            z = (x[..., 0] * da[..., 0] + x[..., 1] * da[..., 1]) + x[..., 2] * da[..., 2]
            e = x - z[..., None] * da
            q = (e[..., 0] * e[..., 0] + e[..., 1] * e[..., 1]) + e[..., 2] * e[..., 2]
            q = torch.where(has & (z > zc[a][:, None]), q, math.inf)
            best = q.min(1, keepdim=True)[0]
            j = torch.where((q == best) & torch.isfinite(q), k[None].expand_as(q), 1 << 30).min(1)[0]  # rows ascend
            ok = j < (1 << 30)
            j = torch.where(ok, j, 0)[:, None]
            nxt[s:s + step] = torch.where(ok, torch.gather(nb, 1, j)[:, 0], -1)
            zn_[s:s + step] = torch.gather(z, 1, j)[:, 0]
        go = nxt >= 0
        act, nxt, zn_ = act[go], nxt[go], zn_[go]
        cur[act], zc[act] = nxt, zn_
        cnt[act] += 1
        cols.append((act, nxt))
    ids = torch.full((H, max(1, len(cols))), -1, dtype=torch.int32, device=DEV)
    for k, (a, nx) in enumerate(cols):
        ids[a, k] = nx.to(torch.int32)
    return cnt, ids


def _project(m, o, d, p):
    """Projected distances and velocity differences of points p (o itself: 0) along d."""
    out = []
    for key in ("pos", "vel"):
        x = torch.from_numpy(m[key]).to(DEV)
        u = x[p] - x[o]
        out.append((u[..., 0] * d[..., 0] + u[..., 1] * d[..., 1]) + u[..., 2] * d[..., 2])
    return out


class _Sweep:
    """Elimination of H half-lines times NB bins from their far ends, in the scaled 1+B form."""

    def __init__(self, H, NB, order):
        self.order = order
        for name, v in dict(DF=1.0, zh=0.0, h=-1.0, chi=0.0, S=0.0, Sp=0.0).items():
            setattr(self, name, torch.full((H, NB), v, dtype=torch.float64, device=DEV))

    NAMES = ("DF", "zh", "h", "chi", "S", "Sp")

    def row(self, sel, dt, chi, S):
        """The row of the current sample, the increment to the next (chi, S) being dt; sel: mask or None."""
        if self.order == 2:
            hb = torch.where(self.h < 0, dt, self.h + dt) / 2
            F = hb + self.DF
            D = 1 / (1 + dt * F)
            zh = D * (hb * self.S + self.zh)
        else:
            hm, first = self.h, self.h < 0
            comp = ~((dt > 64 * hm) | (hm > 64 * dt))
            oml = torch.where(comp, (hm * hm + hm * dt - dt * dt) / 12, 0.0)
            mu = torch.where(comp, (dt * dt + hm * dt - hm * hm) / 12, 0.0)
            hr = (hm + dt) / 2 * self.S + oml / hm * (self.Sp - self.S) + mu / dt * (S - self.S)
            k = torch.where(first, 1 - dt * dt / 6, 1 - mu)
            F = torch.where(first, 1 + dt / 2, (hm + dt) / 2 + (1 - oml) * self.DF) / k
            D = 1 / (1 + dt * F)
            zh = D / k * torch.where(first, dt * (self.S / 3 + S / 6) + self.zh, hr + (1 - oml) * self.zh)
        new = dict(DF=D * F, zh=zh, h=dt, chi=chi, S=S, Sp=self.S)
        for name, v in new.items():
            setattr(self, name, v if sel is None else torch.where(sel, v, getattr(self, name)))


def _half(m, o, d, sgn, cnt, ids, order, dtau_max=0.5, dv_max=1.0 / 3.0):
    """Sweeps all bins of the half-lines (o, d) to the origin row: DF, zh, h, Sp [H, NB]."""
    dev = {k: torch.from_numpy(np.ascontiguousarray(m[k])).to(DEV) for k in ("dvw", "chi_c", "eta_c", "chi0", "eta0")}
    L, F, NB, H = len(m["nu0"]), m["n_freq"], len(m["nu0"]) * m["n_freq"], len(o)
    x = -m["x_span"] + 2 * m["x_span"] * np.arange(F) / (F - 1) if F > 1 else np.zeros(1)
    x = torch.from_numpy(np.tile(x, L)).to(DEV)
    ratio = torch.from_numpy(np.repeat(m["nu0"], F)[:, None] / m["nu0"][None, :]).to(DEV)  # [NB, L]

    def optics(ub, q, dl):
        chi, eta = q["chi_c"][:, None].expand(-1, NB), q["eta_c"][:, None].expand(-1, NB)
        for l in range(L):
            r = ratio[:, l][None]
            a = ((C_KMS * (r - 1) + r * ub) + r * (1 + ub / C_KMS) * dl[:, None]) / q["dvw"][:, None]
            g = torch.exp(-(a * a))
            chi, eta = chi + q["chi0"][:, l:l + 1] * g, eta + q["eta0"][:, l:l + 1] * g
        return chi, eta

    out = _Sweep(H, NB, order)
    act = torch.nonzero(cnt > 0)[:, 0]

    def point(a, q):  # entry q of the half-lines a, far end first; cnt: the origin
        k = cnt[a] - 1 - q
        return torch.where(k >= 0, ids[a, torch.clamp(k, min=0)].long(), o[a])

    w = _Sweep(len(act), NB, order)
    ub = x[None] * dev["dvw"][o[act]][:, None]
    q = torch.zeros(len(act), dtype=torch.int64, device=DEV)
    pa = point(act, q)
    za, da = _project(m, o[act], d[act], pa)
    w.chi, eta = optics(ub, {k: v[pa] for k, v in dev.items()}, da)
    w.S, w.eta = eta / w.chi, eta
    j = torch.zeros_like(q)  # samples already stepped in the interval q -> q + 1
    while len(act):
        pa, pb = point(act, q), point(act, q + 1)
        (za, da), (zb, db) = _project(m, o[act], d[act], pa), _project(m, o[act], d[act], pb)
        zb, db = torch.where(pb == o[act], 0.0, zb), torch.where(pb == o[act], 0.0, db)
        jump, lim = (db - da).abs(), dv_max * torch.minimum(dev["dvw"][pa], dev["dvw"][pb])
        nv = torch.where(jump > lim, torch.ceil(jump / lim), 1.0)
        j = j + 1

        def lerp(va, vb, jj):  # from the earlier point along +r
            v0, v1, i = (va, vb, jj) if sgn < 0 else (vb, va, nv - jj)
            t = i / nv
            if va.dim() > 1:
                t, i, n_ = t[:, None], i[:, None], nv[:, None]
            else:
                n_ = nv
            return torch.where(i == 0, v0, torch.where(i == n_, v1, v0 + (v1 - v0) * t))

        jd = j.double()
        ds = (lerp(sgn * za, sgn * zb, jd) - lerp(sgn * za, sgn * zb, jd - 1)).abs()[:, None]
        chi, eta = optics(ub, {k: lerp(v[pa], v[pb], jd) for k, v in dev.items()}, lerp(da, db, jd))
        ni = torch.clamp(torch.ceil(torch.maximum(w.chi, chi) * ds / dtau_max), min=1.0)
        c0, e0, more = w.chi, w.eta, int(ni.max())
        hs = ds / ni
        for k in range(1, more + 1):  # Eq. 2's sub-intervals, chi and eta linear
            t = k / ni
            ck = torch.where(t >= 1, chi, c0 + (chi - c0) * t)
            ek = torch.where(t >= 1, eta, e0 + (eta - e0) * t)
            dt = hs * (w.chi + ck) * 0.5
            if k == 1:
                w.row(None, dt, ck, ek / ck)
                continue
            on = torch.nonzero((ni >= k).any(1))[:, 0]  # the few lines that are split this far
            sub = _Sweep(0, NB, order)
            for name in _Sweep.NAMES:
                setattr(sub, name, getattr(w, name)[on])
            sub.row((ni >= k)[on], dt[on], ck[on], (ek / ck)[on])
            for name in _Sweep.NAMES:
                getattr(w, name)[on] = getattr(sub, name)
        w.eta = eta
        nxt = j >= nv.long()
        q, j = torch.where(nxt, q + 1, q), torch.where(nxt, 0, j)
        end = q >= cnt[act]
        if bool(end.any()):
            for name in _Sweep.NAMES:
                getattr(out, name)[act[end]] = getattr(w, name)[end]
            go = ~end
            act, q, j, ub, w.eta = act[go], q[go], j[go], ub[go], w.eta[go]
            for name in _Sweep.NAMES:
                setattr(w, name, getattr(w, name)[go])
    po = {k: v[o] for k, v in dev.items()}
    chi, eta = optics(x[None] * dev["dvw"][o][:, None], po, torch.zeros(H, dtype=torch.float64, device=DEV))
    return out, eta / chi


def _solve(m, order):
    """J [n, NB] of a model."""
    n, NB = len(m["pos"]), len(m["nu0"]) * m["n_freq"]
    dirs, wts = _rayset(m)
    P = dirs.shape[1]
    J = torch.zeros((n, NB), dtype=torch.float64, device=DEV)
    step = max(1, 24_000_000 // (P * NB))
    for o0 in range(0, n, step):
        o = torch.arange(o0, min(n, o0 + step), device=DEV)
        oo, r = o.repeat_interleave(P), dirs[o].reshape(-1, 3)
        b, _ = _half(m, oo, -r, -1.0, *_trace(m, oo, -r), order)
        f, So = _half(m, oo, r, 1.0, *_trace(m, oo, r), order)
        hb, hf = torch.clamp(b.h, min=0.0), torch.clamp(f.h, min=0.0)
        if order == 2:
            hh = (hb + hf) / 2
            u = (hh * So + b.zh + f.zh) / (hh + b.DF + f.DF)
        else:
            comp = ~((hf > 64 * hb) | (hb > 64 * hf))
            oml = torch.where(comp, (hb * hb + hb * hf - hf * hf) / 12, 0.0)
            mu = torch.where(comp, (hf * hf + hb * hf - hb * hb) / 12, 0.0)
            u = ((hb + hf) / 2 * So + oml / hb * (b.Sp - So) + mu / hf * (f.Sp - So) + (1 - oml) * b.zh + (1 - mu) * f.zh)
            u = u / ((hb + hf) / 2 + (1 - oml) * b.DF + (1 - mu) * f.DF)
            for w, v in ((b, f), (f, b)):  # one half empty: the origin row is the boundary row (I = 0)
                k1 = 1 - w.h * w.h / 6
                e = (w.h * (So / 3 + w.Sp / 6) + k1 * w.zh) / (1 + w.h / 2 + k1 * w.DF)
                u = torch.where(v.h < 0, e, u)
        u = torch.where((b.h < 0) & (f.h < 0), 0.0, u)
        J[o] = (wts[o][..., None] * u.view(len(o), P, NB)).sum(1)
    return J


def _shuffles(seed, n, epochs):
    """The training order of each epoch: Fisher-Yates from SplitMix64."""
    mask, state, out = (1 << 64) - 1, seed & ((1 << 64) - 1), []
    for _ in range(epochs):
        order = list(range(n))
        for i in range(n - 1, 0, -1):
            state = (state + 0x9E3779B97F4A7C15) & mask
            z = ((state ^ (state >> 30)) * 0xBF58476D1CE4E5B9) & mask
            z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
            j = (z ^ (z >> 31)) % (i + 1)
            order[i], order[j] = order[j], order[i]
        out.append(torch.tensor(order))
    return out


def _net(theta, X):
    W1, b1, W2, b2, W3, b3 = torch.split(theta, [512, 64, 4096, 64, 64, 1])
    h = torch.relu(torch.relu(X @ W1.view(8, 64) + b1) @ W2.view(64, 64) + b2)
    return h @ W3 + b3


def _train(case, seed):
    X, y = (torch.from_numpy(a).double() for a in _training_set(case, seed))
    theta = torch.from_numpy(_theta(seed)).double().requires_grad_()
    m, v, t, losses = torch.zeros_like(theta), torch.zeros_like(theta), 0, []
    for order in _shuffles(seed, case["n"], case["epochs"]):
        total = 0.0
        for rows in order.split(case["batch"]):
            e2 = (_net(theta, X[rows]) - y[rows]) ** 2
            g, = torch.autograd.grad(e2.mean(), theta)
            total += float(e2.detach().sum())
            with torch.no_grad():
                t += 1
                m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
                theta -= 2e-3 * (m / (1 - 0.9 ** t)) / (torch.sqrt(v / (1 - 0.999 ** t)) + 1e-8)
        losses.append(total / case["n"])
    return dict(losses=np.array(losses), theta=theta.detach().numpy())


def _criterion(m):
    """Features and the plain criterion of Eqs. 6-8."""
    n, off = len(m["pos"]), m["nbr_off"]
    row, nb, deg = np.repeat(np.arange(n), np.diff(off)), m["nbr_idx"], np.diff(off)

    def top(v):
        out = np.zeros(n)
        np.maximum.at(out, row, v)
        return out

    dist = np.sqrt(((m["pos"][nb] - m["pos"][row]) ** 2).sum(1))
    L = np.bincount(row, dist, n) / np.maximum(deg, 1)
    lr = np.log(m["rho"])
    X = np.stack([lr, top(np.abs(lr[nb] - lr[row])), top(np.sqrt(((m["vel"][nb] - m["vel"][row]) ** 2).sum(1))) / m["dvw"],
                  np.log(m["T"]), np.log(L + 1e-30), deg, np.log(np.sqrt((m["pos"] ** 2).sum(1)) + 1e-30),
                  np.log(m["chi0"][:, 0] * L + 1e-30)], 1)
    Gf = top(np.abs((m["rho"][row] - m["rho"][nb]) / (m["rho"][row] + m["rho"][nb])))
    return X, Gf, L, L * np.where(Gf >= 0.21, 1.0, 2.15)


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return _train(case, seed)
    if kind in ("solve", "batch", "host") and work(case)["flops"] > 7e11:
        return None  # over about 20 seconds
    models = _models(case, seed)
    if kind == "reduce":
        X, Gf, L, ell = _criterion(models[0])
        return dict(X=X, keep=None, kept=None, scale=None, Gf=Gf, L=L, ell=ell, plain=None, n_plain=None)
    if kind == "rays":
        m = models[0]
        n_o = min(case["origins"], len(m["pos"]))
        dirs = _rayset(m)[0][:n_o]
        d = torch.stack([-dirs, dirs], 2).reshape(-1, 3)
        o = torch.arange(n_o, device=DEV).repeat_interleave(2 * dirs.shape[1])
        cnt, ids = _trace(m, o, d)
        h, k = torch.nonzero(ids >= 0, as_tuple=True)
        Z, delta = _project(m, o[h], d[h], ids[h, k].long())
        _, bufZ, bufd = _lists(case, len(m["pos"]))
        bufZ[:len(Z)], bufd[:len(Z)] = Z.cpu().numpy(), delta.cpu().numpy()
        return dict(rays=None, off=None, idx=None, Z=bufZ, delta=bufd)
    J = [_solve(m, case["order"]) for m in models]
    return J if kind == "batch" else J[0].cpu() if kind == "host" else J[0]
