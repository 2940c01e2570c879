"""The workloads this library's speed is measured on.

Every case is a call, or a few calls, of the public binding
(``paper_2305_11335_gb300``) as a user's program makes them.  ``listed()``
gives the fixed ones and ``draw()`` more of the same ranges: 1 to 8
dimensions, a thousand to ten million points, one point set or a packed batch,
one cutoff or a sweep, int32 or float32 coordinates, both precision modes.
Points are seeded synthetic sets made on the GPU:

``blobs``  isotropic Gaussian blobs with uniform noise, the usual test set of
           density clustering; the cutoff is picked as an analyst picks it, the
           median distance to the k-th neighbour over a sample of the points
``walk``   a seed spreader: 100 points in a ball of radius 100 around every
           step of a random walk in [0, 1e5]^d, with d_cut = 30
``aniso``  anisotropic Gaussian blobs, an embedding-like set in 5 to 8 dimensions
"""
import math

import numpy as np
import torch

import paper_2305_11335_gb300 as dpc

DEV = "cuda"
PAIRS = 5e10  # pair evaluations exact() may spend (a few seconds in binary64)


def listed():
    return [
        # densities of a small set with no allocation inside the call (a latency-critical host): the smallest call
        dict(name="static_2d_1e3", kind="static", family="blobs", n=1000, d=2, dtype="f32", k=16, blobs=4),
        # the paper-sized toy set clustered over and over, the call replayed as a CUDA graph: launches count
        dict(name="graph_2d_int_1e4", kind="graph", family="blobs", n=10000, d=2, dtype="i32", k=24, blobs=5),
        # an analyst's ordinary integer set in the plain binary64 mode, noise points left out of the search
        dict(name="run_2d_fp64_1e5", kind="run", family="blobs", n=100003, d=2, dtype="i32", k=30, blobs=40,
             cuts=1, precision="fp64", skip_noise=True),
        # the ordinary clustering call: a million points in the plane
        dict(name="run_2d_1e6", kind="run", family="blobs", n=1000000, d=2, dtype="f32", k=30, blobs=50, cuts=1,
             precision="fp32", skip_noise=False),
        # the large call: ten million points in space, layouts tuned once at start-up as a server does
        dict(name="run_3d_1e7", kind="run", family="walk", n=10000000, d=3, dtype="f32", k=49, blobs=0, cuts=1,
             precision="fp32", skip_noise=False, autotune=True),
        # embedding-like points with a sweep of four cutoffs: the heaviest call
        dict(name="run_7d_2e6_x4", kind="run", family="aniso", n=2000000, d=7, dtype="f32", k=30, blobs=30, cuts=4,
             precision="fp32", skip_noise=False),
        # a packed batch of ragged instances of three dimensions with eight cutoffs each
        dict(name="batch_128_x8", kind="batch", inst=128, n_lo=1000, n_hi=200000, k=8, cuts=8),
        # picking a cutoff: the densities alone for a sweep in 5 dimensions
        dict(name="density_5d_x4", kind="density", family="blobs", n=100003, d=5, dtype="f32", k=16, blobs=20, cuts=4),
        # densities in hand: dependent points above the noise threshold, then labels for two sets of thresholds
        dict(name="requery_3d_int", kind="requery", family="walk", n=150001, d=3, dtype="i32", k=49, blobs=0),
        # the whole pipeline on pinned host buffers, copies included
        dict(name="host_2d_1e6", kind="host", family="blobs", n=1000000, d=2, dtype="f32", k=30, blobs=50, cuts=1),
        # the decision graph of a large result: the best 1024 centers and the binned (rho, delta) counts
        dict(name="decision_1e7", kind="decision", n=10000000, inst=1, k=1024, rho_bins=24, delta_bins=48),
        # priority range queries against one set, the 64 smallest ids of each
        dict(name="range_3d_1e6", kind="range", family="blobs", n=1000000, d=3, dtype="f32", k=16, blobs=50,
             queries=20000, max_out=64, half=0.01),
    ]


def _log(rng, lo, hi):
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return min(max(n, lo), hi)


def draw(rng):
    kind = rng.choice(["run", "run", "run", "batch", "density", "static", "graph", "requery", "host", "decision",
                       "range"])
    if kind == "batch":
        return dict(kind=kind, inst=rng.randint(8, 128), n_lo=1000, n_hi=rng.choice([20000, 100000, 200000]),
                    k=rng.choice([8, 12, 16]), cuts=rng.randint(1, 8))
    if kind == "decision":
        return dict(kind=kind, n=_log(rng, 10000, 10000000), inst=rng.choice([1, 1, 7, 100]),
                    k=rng.choice([16, 100, 1024]), rho_bins=24, delta_bins=48)
    d = rng.choice([1, 2, 2, 3, 3, 4, 5, 7, 8])
    hi = {1: 2000000, 2: 3000000, 3: 6000000, 4: 1000000, 5: 600000, 7: 400000, 8: 300000}[d]
    family = rng.choice(["blobs", "walk"]) if 2 <= d <= 3 else ("blobs" if d <= 4 else rng.choice(["blobs", "aniso"]))
    if kind == "static":
        n = _log(rng, 1000, dpc.DPC_STATIC_MAX_POINTS)
    elif kind == "graph":
        n = _log(rng, 1000, 100000)
    else:
        n = _log(rng, 1000, hi)
    c = dict(kind=kind, family=family, n=n, d=d, dtype="i32" if family != "aniso" and rng.random() < 0.3 else "f32",
             k=rng.choice([12, 16, 30, 48]), blobs=rng.choice([5, 20, 50]))
    if kind in ("run", "density", "host"):
        c["cuts"] = rng.choice([1, 1, 2, 4])
    if kind == "run":
        c["precision"] = "fp64" if n <= 100000 and rng.random() < 0.25 else "fp32"
        c["skip_noise"] = rng.random() < 0.25
    if kind == "range":
        c.update(queries=_log(rng, 500, 20000), max_out=rng.choice([0, 16, 64]), half=rng.choice([0.003, 0.01, 0.03]))
    return c


# ---------------------------------------------------------------------------
# points


def _mix(seed):
    return np.random.default_rng([seed % (1 << 32), 20231])


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) % (1 << 62))
    return g


def _blobs(n, d, nb, seed, noise=0.05, lo=2e-3, hi=2e-2):
    """[n, d] float32 in about [0, 1]^d, and the blob profile exp(-r^2 / 2) of every point (0 for noise)."""
    r, g = _mix(seed), _gen(seed)
    cen = torch.from_numpy(r.random((nb, d)).astype(np.float32)).to(DEV)
    sig = torch.from_numpy(np.exp(r.uniform(math.log(lo), math.log(hi), nb)).astype(np.float32)).to(DEV)
    edge = torch.from_numpy(np.cumsum(r.dirichlet(np.full(nb, 2.0))).astype(np.float32)).to(DEV)
    which = torch.searchsorted(edge, torch.rand(n, device=DEV, generator=g)).clamp_(max=nb - 1)
    z = torch.randn(n, d, device=DEV, generator=g)
    p = cen[which] + sig[which, None] * z
    q = torch.exp(-0.5 * (z * z).sum(1))
    out = torch.rand(n, device=DEV, generator=g) < noise
    p = torch.where(out[:, None], torch.rand(n, d, device=DEV, generator=g), p)
    return p, torch.where(out, torch.zeros_like(q), q)


def _walk(n, d, seed, box=1e5, step=50.0, radius=100.0, restart=1e-4):
    r, g = _mix(seed), _gen(seed)
    steps = max(1, n // 100)
    u = r.standard_normal((steps, d))
    u *= step / np.linalg.norm(u, axis=1, keepdims=True)
    begin = r.random(steps) < restart
    begin[0] = True
    run = np.cumsum(u, axis=0)
    seg = np.cumsum(begin) - 1
    at = np.flatnonzero(begin)
    pos = r.uniform(0.0, box, (len(at), d))[seg] + run - run[at][seg]
    pos = np.abs((pos + box) % (2 * box) - box)  # reflected at the faces of the box
    pos = torch.from_numpy(pos.astype(np.float32)).to(DEV)
    v = torch.randn(n, d, device=DEV, generator=g)
    v *= (radius * torch.rand(n, device=DEV, generator=g).pow_(1.0 / d) / v.norm(dim=1))[:, None]
    which = torch.arange(n, device=DEV).div_(100, rounding_mode="floor").clamp_(max=steps - 1)
    p = pos[which] + v
    out = torch.rand(n, device=DEV, generator=g) < 1e-3
    p = torch.where(out[:, None], box * torch.rand(n, d, device=DEV, generator=g), p)
    return p[torch.randperm(n, device=DEV, generator=g)]


def _aniso(n, d, nb, seed, noise=0.02):
    r, g = _mix(seed), _gen(seed)
    cen = torch.from_numpy(r.random((nb, d)).astype(np.float32)).to(DEV)
    maps = []
    for _ in range(nb):
        q, _ = np.linalg.qr(r.standard_normal((d, d)))
        maps.append(np.sqrt(np.exp(r.uniform(math.log(1e-4), math.log(1e-2), d)))[:, None] * q.T)
    maps = torch.from_numpy(np.stack(maps).astype(np.float32)).to(DEV)
    z = torch.randn(n, d, device=DEV, generator=g)
    which = torch.randint(nb, (n,), device=DEV, generator=g)
    p = cen[which]
    for a in range(d):
        p = p + z[:, a, None] * maps[which, a]
    out = torch.rand(n, device=DEV, generator=g) < noise
    return torch.where(out[:, None], torch.rand(n, d, device=DEV, generator=g), p)


def _points(c, seed):
    """The points of a case and, for ``blobs``, their profile."""
    prof = None
    if c["family"] == "walk":
        p = _walk(c["n"], c["d"], seed)
    elif c["family"] == "aniso":
        p = _aniso(c["n"], c["d"], c["blobs"], seed)
    else:
        p, prof = _blobs(c["n"], c["d"], c["blobs"], seed)
        if c["dtype"] == "i32":
            p = p * 1e7  # ten million units across, as digitised coordinates come
    p = p.round().to(torch.int32) if c["dtype"] == "i32" else p
    return p.contiguous(), prof


def _kth(p, k, seed, samples=96):
    """Median distance to the k-th nearest point (itself included) over a sample of the points (0-dim tensor)."""
    n = p.shape[0]
    idx = torch.from_numpy(_mix(seed + 1).integers(0, n, samples)).to(DEV)
    x = p.float()
    got = []
    step = max(1, int(2e8) // n)
    for s in range(0, samples, step):
        q = x[idx[s:s + step]]
        dist = torch.zeros(q.shape[0], n, device=DEV)
        for a in range(x.shape[1]):
            dist += (q[:, a, None] - x[None, :, a]).square_()
        got.append(dist.topk(min(k, n), dim=1, largest=False).values[:, -1])
    return torch.cat(got).median().sqrt()


def _cutoffs(c, p, seed):
    d0 = 30.0 if c["family"] == "walk" else float(_kth(p, c["k"], seed))
    return [d0 * 1.25 ** j for j in range(c.get("cuts", 1))]


# ---------------------------------------------------------------------------
# the cases


def prepare(case, seed):
    c = dict(case)
    kind = c["kind"]
    if kind == "batch":
        return _prepare_batch(c, seed)
    if kind == "decision":
        return _prepare_decision(c, seed)
    p, prof = _points(c, seed)
    n, d = c["n"], c["d"]
    s = dict(case=c, pts=p)
    if kind == "range":
        s["rho"] = (1 + (200.0 * prof if prof is not None else 200.0 * torch.rand(n, device=DEV, generator=_gen(
            seed + 5))).to(torch.int32)).to(torch.int32)
        s["batch"] = dpc.Batch.single(n, d, _cutoffs(c, p, seed)[0])
        r = _mix(seed + 2)
        at = p[torch.from_numpy(r.integers(0, n, c["queries"])).to(DEV)].double().cpu()
        width = float((p.double().amax(0) - p.double().amin(0)).max()) * c["half"]
        w = torch.from_numpy(np.exp(r.uniform(math.log(0.2), 0.0, (c["queries"], d)))) * width
        s["boxes"] = dpc.range_boxes(at - w, at + w, device=DEV)
        s["q_inst"] = torch.zeros(c["queries"], dtype=torch.int32, device=DEV)
        s["q_rho"] = torch.from_numpy(r.integers(0, 100, c["queries"]).astype(np.int32)).to(DEV)
        return s
    cuts = _cutoffs(c, p, seed)
    s["cuts"] = cuts
    s["d_cut"] = cuts[0]
    if kind == "static":
        return s
    s["batch"] = dpc.Batch.single(n, d, cuts)
    s["rho_noise"], s["delta_min"] = 2 * c["k"], 5.0 * cuts[0]
    s["params"] = dpc.make_params(s["batch"], s["rho_noise"], s["rho_noise"], s["delta_min"])
    if kind == "requery":
        s["rho"] = dpc.dpc_density(p, s["batch"])[0]
        s["params2"] = dpc.make_params(s["batch"], s["rho_noise"], 2 * s["rho_noise"], 10.0 * cuts[0])
    elif kind == "host":
        s["pts"] = p.cpu().pin_memory()
        shape = (len(cuts), n)
        s["out"] = {"rho": torch.empty(shape, dtype=torch.int32).pin_memory(),
                    "lam": torch.empty(shape, dtype=torch.int32).pin_memory(),
                    "delta": torch.empty(shape, dtype=torch.float64).pin_memory(),
                    "label": torch.empty(shape, dtype=torch.int32).pin_memory()}
    elif kind == "graph":  # a server's loop: its own stream and buffers, the graph captured at start-up
        torch.cuda.current_stream().synchronize()
        s["stream"] = torch.cuda.Stream()
        s["out"] = dpc.dpc_run(p, s["batch"], s["params"], graph=True, stream=s["stream"])
        s["stream"].synchronize()
    elif c.get("autotune"):
        dpc.dpc_run(p, s["batch"], s["params"], precision=c["precision"], autotune=True)
    return s


def _prepare_batch(c, seed):
    r = _mix(c["inst"] * 1000 + c["cuts"])  # the case's shape; the points come from the seed
    sizes = np.rint(np.exp(r.uniform(math.log(c["n_lo"]), math.log(c["n_hi"]), c["inst"]))).astype(int).tolist()
    dims = r.choice([2, 3, 5], c["inst"]).tolist()
    nb = r.integers(2, 41, c["inst"]).tolist()
    parts, cut0 = [], []
    for i, (n, d) in enumerate(zip(sizes, dims)):
        p, _ = _blobs(n, d, nb[i], seed * 1000 + i, noise=0.0, lo=1e-3)
        parts.append(p.reshape(-1))
        cut0.append(_kth(p, c["k"], seed * 1000 + i, samples=32))
    cut0 = torch.stack(cut0).cpu().double().tolist()
    cuts = [[x * 1.25 ** j for j in range(c["cuts"])] for x in cut0]
    batch = dpc.Batch.packed(sizes, dims, cuts)
    noise = [int(2 * c["k"] * 1.25 ** (j * d / 2)) for d in dims for j in range(c["cuts"])]
    params = dpc.make_params(batch, noise, noise, [5.0 * x for row in cuts for x in row])
    return dict(case=c, pts=torch.cat(parts), batch=batch, params=params)


def _prepare_decision(c, seed):
    """(rho, delta) as a run leaves them: log-normal densities, delta mostly below the cutoff with a heavy tail, one
    +inf per instance."""
    n, m = c["n"], c["inst"]
    g, r = _gen(seed), _mix(n + m)
    rho = torch.exp(3.6 + 0.8 * torch.randn(n, device=DEV, generator=g)).to(torch.int32) + 1
    delta = 30.0 * torch.exp(-1.2 + 0.6 * torch.randn(n, device=DEV, generator=g, dtype=torch.float64))
    far = torch.rand(n, device=DEV, generator=g) < 2e-3
    delta = torch.where(far, delta * torch.exp(4.0 * torch.rand(n, device=DEV, generator=g, dtype=torch.float64)), delta)
    cut = np.sort(r.choice(np.arange(1, n), m - 1, replace=False)).tolist() if m > 1 else []
    off = [0] + [int(x) for x in cut] + [n]
    delta[torch.tensor(off[:-1], device=DEV)] = math.inf
    return dict(case=c, rho=rho, delta=delta, batch=dpc.Batch(off, [3] * m, [[30.0]] * m))


def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "static":
        return dpc.dpc_density_static(s["pts"], s["d_cut"])
    if kind == "graph":
        return dpc.dpc_run(s["pts"], s["batch"], s["params"], graph=True, stream=s["stream"], out=s["out"])
    if kind == "run":
        return dpc.dpc_run(s["pts"], s["batch"], s["params"], precision=c["precision"], skip_noise=c["skip_noise"],
                           autotune=c.get("autotune", False))
    if kind == "batch":
        return dpc.dpc_run(s["pts"], s["batch"], s["params"])
    if kind == "density":
        return dpc.dpc_density(s["pts"], s["batch"])
    if kind == "requery":
        lam, delta = dpc.dpc_dependent(s["pts"], s["batch"], 0, s["rho"], rho_skip=s["rho_noise"])
        one = dpc.dpc_cluster(s["batch"], 0, s["params"], s["rho"], lam, delta)
        two = dpc.dpc_cluster(s["batch"], 0, s["params2"], s["rho"], lam, delta)
        return {"lam": lam, "delta": delta, "label": one, "label2": two}
    if kind == "host":
        return dpc.dpc_run_host(s["pts"], s["batch"], s["params"], out=s["out"])
    if kind == "decision":
        return dpc.dpc_decision_graph(s["batch"], s["rho"], s["delta"], k=c["k"], rho_bins=c["rho_bins"],
                                      delta_bins=c["delta_bins"], delta_lo=0.5)
    return dpc.dpc_priority_range(s["pts"], s["batch"], s["rho"], s["q_inst"], s["boxes"], s["q_rho"],
                                  max_out=c["max_out"])


def work(case):
    """Coordinates read once, results written once; three operations per coordinate for every pair within the cutoff
    (about k per point), which any exact method has to look at or count."""
    c = case
    kind = c["kind"]
    if kind == "decision":
        return {"bytes": 12.0 * c["n"] + 12.0 * c["inst"] * c["k"] + 8.0 * c["inst"] * c["rho_bins"] * c["delta_bins"],
                "flops": 2.0 * c["n"]}
    if kind == "batch":
        mean = (c["n_hi"] - c["n_lo"]) / math.log(c["n_hi"] / c["n_lo"])
        n, d, k = c["inst"] * mean, 10.0 / 3.0, c["k"] * 2.0
        return {"bytes": n * (4 * d + 20.0 * c["cuts"]), "flops": n * c["cuts"] * 3 * d * k}
    n, d, k = float(c["n"]), c["d"], c["k"]
    cuts = c.get("cuts", 1)
    flops = 3.0 * d * n * k * cuts
    if kind in ("static", "density"):
        return {"bytes": n * (4 * d + 4 * cuts), "flops": flops}
    if kind == "requery":
        return {"bytes": n * (4 * d + 4 + 12 + 2 * 4), "flops": flops}
    if kind == "range":
        return {"bytes": n * (4 * d + 4) + c["queries"] * (2.0 * 8 * d + 8 + 8 + 4 * c["max_out"]),
                "flops": 2.0 * d * c["queries"] * (64 + c["max_out"])}
    return {"bytes": n * (4 * d + 20 * cuts), "flops": flops}


# ---------------------------------------------------------------------------
# the same results from the definitions, in binary64


def _sq(x, a, b):
    s = None
    for k in range(x.shape[1]):
        t = x[a:b, k, None] - x[None, :, k]
        t = t * t
        s = t if s is None else s + t
    return s


def _rows(n):
    return max(1, int(1.2e8) // n)


def _rho(x, cuts):
    n = x.shape[0]
    out = torch.empty(len(cuts), n, dtype=torch.int32, device=x.device)
    for a in range(0, n, _rows(n)):
        s = _sq(x, a, min(n, a + _rows(n)))
        for j, dc in enumerate(cuts):
            out[j, a:a + s.shape[0]] = (s <= dc * dc).sum(1)
    return out


def _dependent(x, rho, skip):
    n = x.shape[0]
    ids = torch.arange(n, device=x.device)
    lam = torch.empty(n, dtype=torch.int32, device=x.device)
    delta = torch.empty(n, dtype=torch.float64, device=x.device)
    for a in range(0, n, _rows(n)):
        b = min(n, a + _rows(n))
        up = (rho[None, :] > rho[a:b, None]) | ((rho[None, :] == rho[a:b, None]) & (ids[None, :] < ids[a:b, None]))
        s = _sq(x, a, b).masked_fill_(~up, math.inf)
        best = s.amin(1)
        at = torch.where(s == best[:, None], ids[None, :], n).amin(1)
        lam[a:b] = torch.where(torch.isinf(best), -1, at).to(torch.int32)
        delta[a:b] = best.sqrt()
    low = rho < skip
    lam[low] = -1
    delta[low] = math.nan
    return lam, delta


def _labels(rho, lam, delta, noise, rho_min, delta_min):
    ids = torch.arange(rho.shape[0], device=rho.device)
    root = (lam < 0) | ((rho >= rho_min) & (delta >= delta_min))
    par = torch.where(root, ids, lam.long())
    low = rho < noise
    par = torch.where(low, ids, par)
    while True:
        nxt = par[par]
        if torch.equal(nxt, par):
            break
        par = nxt
    return torch.where(low[par], -1, par).to(torch.int32)


def exact(case, seed):
    c = dict(case)
    kind = c["kind"]
    if kind == "batch":
        return None
    if kind == "decision":
        return _exact_decision(prepare(case, seed))
    if kind == "range":
        if float(c["n"]) * c["queries"] > PAIRS:
            return None
        return _exact_range(prepare(case, seed))
    phases = {"static": 1, "density": 1, "requery": 2}.get(kind, 1 + c.get("cuts", 1))
    if float(c["n"]) ** 2 * phases * max(2, c["d"]) / 3.0 > PAIRS:
        return None
    p, _ = _points(c, seed)
    cuts = _cutoffs(c, p, seed)
    x = p.double()
    rho = _rho(x, cuts)
    if kind == "static":
        return rho[0]
    if kind == "density":
        return rho
    noise, dmin = 2 * c["k"], 5.0 * cuts[0]
    if kind == "requery":
        lam, delta = _dependent(x, rho[0], noise)
        return {"lam": lam, "delta": delta, "label": _labels(rho[0], lam, delta, noise, noise, dmin),
                "label2": _labels(rho[0], lam, delta, noise, 2 * noise, 10.0 * cuts[0])}
    out = {"rho": rho, "lam": [], "delta": [], "label": []}
    for j in range(len(cuts)):
        lam, delta = _dependent(x, rho[j], noise if c.get("skip_noise") else 0)
        out["lam"].append(lam)
        out["delta"].append(delta)
        out["label"].append(_labels(rho[j], lam, delta, noise, noise, dmin))
    return {k: v if k == "rho" else torch.stack(v) for k, v in out.items()}


def _exact_decision(s):
    c, off = s["case"], s["batch"].pt_offset
    top = torch.full((c["inst"], c["k"]), -1, dtype=torch.int32, device=DEV)
    gamma = torch.full((c["inst"], c["k"]), math.nan, dtype=torch.float64, device=DEV)
    hist = torch.zeros(c["inst"], c["rho_bins"], c["delta_bins"], dtype=torch.int64, device=DEV)
    for i in range(c["inst"]):
        r, dl = s["rho"][off[i]:off[i + 1]].double(), s["delta"][off[i]:off[i + 1]]
        v, at = torch.sort(r * dl, descending=True, stable=True)
        k = min(c["k"], v.numel())
        gamma[i, :k], top[i, :k] = v[:k], at[:k].to(torch.int32)
        a = (torch.frexp(r).exponent - 1).clamp(max=c["rho_bins"] - 1).long()
        ratio = dl / 0.5
        b = torch.where(torch.isinf(ratio), c["delta_bins"] - 1,
                        (torch.frexp(ratio).exponent - 1).clamp(0, c["delta_bins"] - 1)).long()
        b = torch.where(dl > 0.5, b, 0)
        hist[i] = torch.bincount(a * c["delta_bins"] + b, minlength=hist[i].numel()).reshape(hist[i].shape)
    return {"top": top, "gamma": gamma, "hist": hist}


def _exact_range(s):
    c, x, rho, box = s["case"], s["pts"].double(), s["rho"], s["boxes"]
    n, d, nq, m = c["n"], c["d"], c["queries"], c["max_out"]
    count = torch.empty(nq, dtype=torch.int64, device=DEV)
    ids = torch.full((nq, max(m, 1)), -1, dtype=torch.int32, device=DEV)
    step = max(1, int(2e8) // n)
    for a in range(0, nq, step):
        b = min(nq, a + step)
        ok = rho[None, :] > s["q_rho"][a:b, None]
        for k in range(d):
            ok &= (x[None, :, k] >= box[a:b, 0, k, None]) & (x[None, :, k] <= box[a:b, 1, k, None])
        count[a:b] = ok.sum(1)
        at = ok.nonzero()
        first = torch.cumsum(count[a:b], 0) - count[a:b]
        rank = torch.arange(at.shape[0], device=DEV) - first[at[:, 0]]
        keep = rank < m
        ids[a + at[keep, 0], rank[keep]] = at[keep, 1].to(torch.int32)
    return {"count": count, "ids": ids} if m > 0 else {"count": count}
