"""Timed cases of the engine: the calls that a trial-design program makes.

Each case is one pass through the public entry points of
paper_2005_10494_gb300 on inputs made from a seed:

  line    one cutoff line (101 designs in the published configuration): the
          one-shot estimate, then the smoothed line and its argmax;
  step    one step of the gradient search: estimate and likelihood-ratio
          gradient of a single design through a plan;
  grid    scenarios x (cutoff x allocation) grids through a plan: forward or
          with both gradients, one stream per scenario (common random
          numbers) or one per design, FP32 or all-FP64 sampling, optionally
          replayed from a CUDA graph and followed by smoothing and argmax;
  batch   scenarios of uneven dimension, design count and draw count in one
          launch;
  fwer    alpha splits calibrated to the family-wise error rate;
  spline  thin-plate splines of scattered estimates and their maximisers;
  gcv     cross-validation scores of one spline;
  smooth  smoothing and argmax of many regular grids.
"""
import math

import numpy as np
import torch

import paper_2005_10494_gb300 as pkg

ALPHA0 = 0.025          # family-wise error rate
INFO = 211.0            # information units of the trial
H = 0.01                # bandwidth of the smoothed indicator
EXACT_WORK = 2.5e11     # design-draw-coordinates that exact() takes on


# ------------------------------------------------------------------- cases
def listed():
    return [
        # the smallest everyday call: the cutoff line of the plain method
        {"name": "line-101", "kind": "line", "d": 3, "designs": 101, "draws": 100_000},
        # one step of a gradient-driven search at d=10
        {"name": "search-step-d10", "kind": "step", "d": 10, "draws": 10_000_000},
        # the benchmark step: 16 scenarios on a 64 x 64 grid, common random
        # numbers, both gradients, smoothing and argmax
        {"name": "grid-adjoint-d3", "kind": "grid", "d": 3, "scen": 16, "g1": 64, "g2": 64, "draws": 1_000_000,
         "grad": True, "crn": True, "fp64": False, "graph": True, "smooth": True},
        # estimates alone on such grids (grid search without the adjoint)
        {"name": "grid-forward-d3", "kind": "grid", "d": 3, "scen": 4, "g1": 64, "g2": 64, "draws": 1_000_000,
         "grad": False, "crn": True, "fp64": False, "graph": False, "smooth": True},
        # independent streams per design (unbiased comparisons between designs)
        {"name": "grid-independent-d3", "kind": "grid", "d": 3, "scen": 1, "g1": 64, "g2": 64, "draws": 1_000_000,
         "grad": True, "crn": False, "fp64": False, "graph": False, "smooth": False},
        # ten nested populations, AR(1)
        {"name": "grid-adjoint-d10", "kind": "grid", "d": 10, "scen": 1, "g1": 32, "g2": 32, "draws": 10_000_000,
         "grad": True, "crn": True, "fp64": False, "graph": False, "smooth": False},
        # the largest dimension, block correlation
        {"name": "grid-adjoint-d20", "kind": "grid", "d": 20, "scen": 1, "g1": 64, "g2": 64, "draws": 1_000_000,
         "grad": True, "crn": True, "fp64": False, "graph": False, "smooth": False},
        # uneven scenarios in one persistent launch, replayed from a graph
        {"name": "batch-uneven", "kind": "batch", "scen": 64, "draws_lo": 100_000, "draws_hi": 1_000_000,
         "grad": False, "graph": True},
        # calibration of the alpha splits of one optimisation problem
        {"name": "fwer-2000", "kind": "fwer", "d": 3, "designs": 2000, "draws": 4_000_000, "rounds": 8},
        # the spline of one optimisation problem and its maximiser
        {"name": "spline-2000", "kind": "spline", "surf": 1, "points": 2000, "k": 2, "smoothing": 1e-6},
        # smoothing throughput, FP64 estimates as the sampler writes them
        {"name": "smooth-f64", "kind": "smooth", "scen": 2048, "g1": 256, "g2": 256, "f32": False, "degree": 2,
         "bandwidth": 3.0, "raw": False},
        # FP32 grids of odd extents, with the raw argmax beside the smoothed
        {"name": "smooth-f32-odd", "kind": "smooth", "scen": 513, "g1": 301, "g2": 203, "f32": True, "degree": 2,
         "bandwidth": 3.0, "raw": True},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["line", "step", "grid", "grid", "grid", "grid", "batch", "fwer", "spline", "gcv", "smooth",
                       "smooth"])
    if kind == "line":
        return {"kind": "line", "d": rng.randint(2, 20), "designs": _logint(rng, 25, 400),
                "draws": _logint(rng, 20_000, 500_000)}
    if kind == "step":
        return {"kind": "step", "d": rng.randint(2, 20), "draws": _logint(rng, 100_000, 10_000_000)}
    if kind == "grid":
        d = rng.choice([2, 3, 3, 4, 5, 6, 7, 8, 9, 10, 12, 13, 16, 20])
        mode = rng.choice(["crn", "crn", "crn", "independent", "fp64"])
        g1, g2 = _logint(rng, 6, 72), _logint(rng, 6, 72)
        scen = _logint(rng, 1, 16)
        if mode == "fp64":
            g1, g2, scen, budget = min(g1, 9), min(g2, 9), 1, 1.5e7 / d
        elif mode == "independent":
            budget = 4e9 / d
        else:
            budget = 1.5e10 / d
        draws = min(_logint(rng, 20_000, 10_000_000), int(budget * 3 / (scen * g1 * g2)))
        return {"kind": "grid", "d": d, "scen": scen, "g1": g1, "g2": g2, "draws": max(draws, 1000),
                "grad": rng.random() < 0.6, "crn": mode == "crn", "fp64": mode == "fp64",
                "graph": rng.random() < 0.3, "smooth": rng.random() < 0.5}
    if kind == "batch":
        lo = _logint(rng, 20_000, 100_000)
        return {"kind": "batch", "scen": _logint(rng, 4, 64), "draws_lo": lo, "draws_hi": lo * rng.randint(2, 5),
                "grad": rng.random() < 0.5, "graph": rng.random() < 0.5}
    if kind == "fwer":
        return {"kind": "fwer", "d": rng.randint(2, 10), "designs": _logint(rng, 100, 2000),
                "draws": _logint(rng, 50_000, 1_000_000), "rounds": rng.randint(6, 14)}
    if kind == "spline":
        return {"kind": "spline", "surf": _logint(rng, 1, 12), "points": _logint(rng, 40, 1500), "k": rng.randint(1, 3),
                "smoothing": 10.0 ** rng.uniform(-6, -3)}
    if kind == "gcv":
        return {"kind": "gcv", "points": _logint(rng, 40, 700), "k": rng.randint(1, 3), "values": rng.randint(2, 5)}
    return {"kind": "smooth", "scen": _logint(rng, 1, 1024), "g1": _logint(rng, 1, 256) + 3, "g2": _logint(rng, 8, 320),
            "f32": rng.random() < 0.5, "degree": rng.choice([1, 2, 2]), "bandwidth": rng.choice([2.5, 3.0, 3.0, 4.0]),
            "raw": rng.random() < 0.5}


# ------------------------------------------------------------------ inputs
def _ndtri(p):
    return torch.special.ndtri(torch.as_tensor(np.asarray(p, dtype=np.float64))).numpy()


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float64), device="cuda")


def _correlation(d, rng):
    """Equicorrelated up to d=4, blocks of at most five for d > 12, AR(1) between."""
    if d <= 4:
        rho = rng.uniform(0.2, 0.7)
        return (1.0 - rho) * np.eye(d) + rho
    if d > 12:
        block = np.arange(d) // 5
        rin, rout = rng.uniform(0.5, 0.7), rng.uniform(0.05, 0.15)
        S = np.where(block[:, None] == block[None, :], rin, rout)
        np.fill_diagonal(S, 1.0)
        return S
    i = np.arange(d)
    return rng.uniform(0.2, 0.4) ** np.abs(i[:, None] - i[None, :])


def _random_correlation(d, rng):
    W = rng.standard_normal((d, d + 3))
    C = W @ W.T
    s = 1.0 / np.sqrt(np.diag(C))
    return C * np.outer(s, s)


def _designs(d, q, a, dp, dm):
    """mu, b [n, d] and the Jacobian [n, d, 4] of t = b - mu with respect to
    (cutoff quantile, allocation, effect with and without the biomarker) for
    arrays q, a: nested populations r, hazard reductions linear in r and the
    level split w = (1 - a, a/(d-1), ...)."""
    i = np.arange(d, dtype=np.float64)
    r = 1.0 - q[:, None] * i / (d - 1)
    delta = dp - (dp - dm) * r
    theta = -np.log1p(-delta)
    sq = np.sqrt(r * INFO)
    w = np.repeat(a[:, None] / (d - 1), d, axis=1)
    w[:, 0] = 1.0 - a
    dw = np.full(d, 1.0 / (d - 1))
    dw[0] = -1.0
    b = _ndtri(1.0 - ALPHA0 * w)
    dth = 1.0 / (1.0 - delta)
    dmu_dr = 0.5 * math.sqrt(INFO) / np.sqrt(r) * theta - sq * dth * (dp - dm)
    phi = np.exp(-0.5 * b * b) / math.sqrt(2.0 * math.pi)
    jac = np.stack([dmu_dr * i / (d - 1), -ALPHA0 * dw / phi, -sq * dth * (1.0 - r), -sq * dth * r], axis=2)
    return sq * theta, b, jac


def _batch_shape(case):
    """(dimension, designs) of each scenario of a batch: the same for every seed."""
    rng = np.random.default_rng([case["scen"], case["draws_lo"]])
    return [(int(rng.integers(3, 11)), int(rng.integers(32, 257))) for _ in range(case["scen"])]


def _host_problem(case, seed):
    """The problem of a sampling case on the host: dict of numpy arrays."""
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    if kind == "batch":
        dims, sig, scen, mu, b, n = [], [], [], [], [], []
        for s, (d, m) in enumerate(_batch_shape(case)):
            dims.append(d)
            sig.append(_random_correlation(d, rng).ravel())
            scen.append(np.full(m, s))
            mu.append(rng.normal(0.3, 0.2, m * d))
            b.append(np.full(m * d, float(_ndtri(1.0 - ALPHA0 / d))))
            n.append(np.exp(rng.uniform(math.log(case["draws_lo"]), math.log(case["draws_hi"]), m)).round())
        scen = np.concatenate(scen)
        return {"dims": np.array(dims), "sigma": np.concatenate(sig), "scen": scen, "mu": np.concatenate(mu),
                "b": np.concatenate(b), "n": np.concatenate(n).astype(np.uint64), "key": np.arange(scen.size),
                "jac": None, "k": 0}
    d = case["d"]
    if kind == "fwer":
        w = rng.dirichlet(np.ones(d), case["designs"])
        J = case["designs"]
        return {"dims": np.array([d]), "sigma": _correlation(d, rng).ravel(), "scen": np.zeros(J, int),
                "mu": np.zeros(J * d), "b": np.zeros(J * d), "n": np.full(J, case["draws"]), "key": np.zeros(J, int),
                "w": w, "jac": None, "k": 0}
    if kind == "line":
        q = np.linspace(0.05, 0.95, case["designs"])
        mu, b, _ = _designs(d, q, np.full(q.size, (d - 1.0) / d), rng.uniform(0.4, 0.6), rng.uniform(0.05, 0.15))
        return {"dims": np.array([d]), "sigma": _correlation(d, rng).ravel(), "scen": np.zeros(q.size, int),
                "mu": mu.ravel(), "b": b.ravel(), "n": np.full(q.size, case["draws"]), "key": np.zeros(q.size, int),
                "jac": None, "k": 0}
    if kind == "step":
        mu, b, jac = _designs(d, rng.uniform(0.2, 0.8, 1), rng.uniform(0.3, 0.7, 1), 0.5, 0.1)
        return {"dims": np.array([d]), "sigma": _correlation(d, rng).ravel(), "scen": np.zeros(1, int),
                "mu": mu.ravel(), "b": b.ravel(), "n": np.full(1, case["draws"]), "key": np.zeros(1, int),
                "jac": jac[:, :, :2], "k": 2}
    S, g1, g2 = case["scen"], case["g1"], case["g2"]
    q, a = (v.ravel() for v in np.meshgrid(np.linspace(0.05, 0.95, g1), np.linspace(0.2, 0.8, g2), indexing="ij"))
    sig, mu, b, jac = [], [], [], []
    for s in range(S):
        dp, dm = rng.uniform(0.3, 0.7), rng.uniform(0.0, 0.2)
        sig.append(_correlation(d, rng).ravel())
        m_, b_, j_ = _designs(d, q, a, dp, dm)
        mu.append(m_), b.append(b_), jac.append(j_)
    scen = np.repeat(np.arange(S), g1 * g2)
    k = 4 if d == 3 else 2
    return {"dims": np.full(S, d), "sigma": np.concatenate(sig), "scen": scen, "mu": np.concatenate(mu).ravel(),
            "b": np.concatenate(b).ravel(), "n": np.full(scen.size, case["draws"]),
            "key": scen if case["crn"] else np.arange(scen.size),
            "jac": np.concatenate(jac)[:, :, :k] if case["grad"] else None, "k": k if case["grad"] else 0}


def _scattered(case, seed):
    """Scattered points and noisy estimates of a smooth power surface."""
    S, N, k = case.get("surf", 1), case["points"], case["k"]
    rng = np.random.default_rng(seed)
    x = rng.uniform(0.0, 1.0, (S, N, k))
    peak = rng.uniform(0.3, 0.7, (S, 1, k))
    p = 0.9 - 0.5 * ((x - peak) ** 2).sum(-1)
    return x, p + rng.normal(0.0, 2e-4, (S, N))


def _grids(case, seed):
    """Noisy estimates of smooth surfaces on regular grids (device tensor)."""
    S, g1, g2 = case["scen"], case["g1"], case["g2"]
    ft = torch.float32 if case["f32"] else torch.float64
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    peak = torch.rand(S, 2, 1, 1, device="cuda", generator=gen) * 0.6 + 0.2
    u = torch.linspace(0, 1, g1, device="cuda").reshape(1, g1, 1)
    v = torch.linspace(0, 1, g2, device="cuda").reshape(1, 1, g2)
    z = torch.randn(S, g1, g2, device="cuda", generator=gen)
    p = 0.9 - 0.4 * (u - peak[:, 0]) ** 2 - 0.3 * (v - peak[:, 1]) ** 2
    return (p.double() + 2e-3 * z.double()).to(ft).reshape(-1).contiguous()


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case, "seed": seed, "ctx": pkg.Context(0)}
    if kind in ("spline", "gcv"):
        x, y = _scattered(case, seed)
        st["x"], st["y"] = _dev(x), _dev(y)
        st["lo"], st["hi"] = _dev(np.zeros(case["k"])), _dev(np.ones(case["k"]))
        if kind == "gcv":
            st["s"] = np.logspace(-6, -2, case["values"])
        return st
    if kind == "smooth":
        st["values"] = _grids(case, seed)
        return st
    hp = _host_problem(case, seed)
    st["prob"] = pkg.DeviceProblem(hp["dims"], hp["scen"], hp["n"], hp["key"], _dev(hp["sigma"]), _dev(hp["mu"]),
                                   _dev(hp["b"]))
    if kind == "fwer":
        st["w"] = _dev(hp["w"].ravel())
    st["jac"] = None if hp["jac"] is None else _dev(hp["jac"].ravel())
    if kind in ("step", "grid", "batch"):
        st["grad"] = kind == "step" or case["grad"]
        st["h"] = 0.0 if kind == "step" else H
        st["plan"] = pkg.Plan(st["ctx"], st["prob"], grad=st["grad"], k=hp["k"], graph=case.get("graph", False),
                              fp64=case.get("fp64", False), shared=case.get("crn", False))
        st["stream"] = torch.cuda.Stream() if case.get("graph") else None   # graphs replay off the default stream
    return st


# --------------------------------------------------------------------- run
def run(state):
    case, kind, ctx = state["case"], state["case"]["kind"], state["ctx"]
    if kind == "line":
        out = pkg.mc_design_eval(ctx, state["prob"], state["seed"])
        sm = pkg.mc_smooth_argmax(ctx, out["p"], 1, 1, case["designs"], raw=True)
        return {**out, **sm}
    if kind == "fwer":
        return pkg.mc_fwer_calibrate(ctx, state["prob"], state["w"], ALPHA0, rounds=case["rounds"], seed=state["seed"])
    if kind == "spline":
        fit = pkg.mc_tps_fit(ctx, state["x"], state["y"], smoothing=case["smoothing"])
        best = pkg.mc_tps_argmax(ctx, state["x"], fit, state["lo"], state["hi"], iters=300)
        return {**fit, "x": best["x"], "f": best["f"]}
    if kind == "gcv":
        return {"score": pkg.mc_tps_gcv(ctx, state["x"][0], state["y"][0], state["s"])}
    if kind == "smooth":
        out = pkg.mc_smooth_argmax(ctx, state["values"], case["scen"], case["g1"], case["g2"],
                                   bandwidth=case["bandwidth"], degree=case["degree"], raw=case["raw"])
        return {k: v for k, v in out.items() if v is not None}
    stream = state["stream"]
    caller = torch.cuda.current_stream()
    if stream is not None:
        stream.wait_stream(caller)
    if state["grad"]:
        out = state["plan"].grad(state["seed"], state["jac"], state["h"], stream=stream)
    else:
        out = state["plan"].eval(state["seed"], stream=stream)
    if stream is not None:
        caller.wait_stream(stream)
    if case.get("smooth"):
        sm = pkg.mc_smooth_argmax(ctx, out["p"], case["scen"], case["g1"], case["g2"])
        out = {**out, "smoothed": sm["smoothed"], "argmax_idx": sm["argmax_idx"], "argmax_val": sm["argmax_val"]}
    return out


# -------------------------------------------------------------------- work
def _sampling_work(dims, J, draws, pairs, grad, rounds=1):
    """Bytes and operations of a sampling pass: J designs of dimension `dims`,
    `draws` distinct draws, `pairs` design-draw pairs.  A normal takes about
    14 operations (a quarter of a ten-round generator call, half a Box-Muller
    pair), the transform d(d + 1), the region test d and a count, and the
    adjoint adds the two gradient sums of d terms."""
    d = dims
    flops = draws * (14 * d + d * (d + 1)) + pairs * (d + 1 + (2 * d if grad else 0))
    byts = J * 8 * (2 * d + 3 + ((4 * d + 9) if grad else 0))
    return {"bytes": int(byts), "flops": int(rounds * flops)}


def work(case):
    kind = case["kind"]
    if kind == "line":
        pairs = case["designs"] * case["draws"]
        return _sampling_work(case["d"], case["designs"], case["draws"], pairs, False)
    if kind == "step":
        return _sampling_work(case["d"], 1, case["draws"], case["draws"], True)
    if kind == "grid":
        J = case["scen"] * case["g1"] * case["g2"]
        distinct = case["draws"] * (case["scen"] if case["crn"] else J)
        return _sampling_work(case["d"], J, distinct, J * case["draws"], case["grad"])
    if kind == "batch":
        lo, hi = case["draws_lo"], case["draws_hi"]
        mean = (hi - lo) / math.log(hi / lo)
        parts = [_sampling_work(d, m, m * mean, m * mean, case["grad"]) for d, m in _batch_shape(case)]
        return {key: sum(p[key] for p in parts) for key in ("bytes", "flops")}
    if kind == "fwer":
        return _sampling_work(case["d"], case["designs"], case["draws"], case["designs"] * case["draws"], False,
                              case["rounds"])
    if kind in ("spline", "gcv"):
        N, k = case["points"], case["k"]
        n = case.get("surf", case.get("values"))
        per = 2.0 * N ** 3 / 3.0 * (1 if kind == "spline" else 2) + 10.0 * N * N
        return {"bytes": int(8 * N * (k + 1) + 8 * n * N * (2 if kind == "spline" else 0)), "flops": int(n * per)}
    pts = case["scen"] * case["g1"] * case["g2"]
    reach = int(math.ceil(case["bandwidth"])) - 1
    return {"bytes": pts * (8 if case["f32"] else 16), "flops": pts * 2 * (2 * reach + 1) ** 2}


# ------------------------------------------------------------------- exact
_M = 0xffffffff


def _philox(call, key, seed):
    """Philox4x32-10 words [n, 4] of int64 tensor `call`, 32-bit halves in int64."""
    x0, x1 = call & _M, call >> 32
    x2 = torch.full_like(call, key & _M)
    x3 = torch.full_like(call, key >> 32)
    k0, k1 = seed & _M, seed >> 32
    for _ in range(10):
        p0, p1 = x0 * 0xD2511F53, x2 * 0xCD9E8D57           # wraps modulo 2^64
        x0, x1, x2, x3 = ((p1 >> 32) & _M) ^ x1 ^ k0, p1 & _M, ((p0 >> 32) & _M) ^ x3 ^ k1, p0 & _M
        k0, k1 = (k0 + 0x9E3779B9) & _M, (k1 + 0xBB67AE85) & _M
    return torch.stack([x0, x1, x2, x3], 1)


def _normals(first, count, d, key, seed, dev):
    """Draws first .. first + count - 1 of a stream: FP64 normals [count, d]."""
    m0, m1 = first * d, (first + count) * d
    w = _philox(torch.arange(m0 // 4, (m1 + 3) // 4, device=dev), key, seed).reshape(-1, 2)
    u = (2.0 * (w >> 9).double() + 1.0) * 2.0 ** -24
    r = torch.sqrt(-2.0 * torch.log(u[:, 0]))
    ang = 2.0 * math.pi * u[:, 1]
    z = torch.stack([r * torch.cos(ang), r * torch.sin(ang)], 1).reshape(-1)
    return z[m0 % 4:m0 % 4 + (m1 - m0)].reshape(count, d)


def _sums(L, t, N, key, seed, grad, h):
    """Over one stream and its designs t [J, d]: hits, and for the adjoint
    sum 1_R z [J, d], sum z [d] and the sigmoid sums [J, d], in FP64."""
    dev, (J, d) = t.device, t.shape
    hits = torch.zeros(J, dtype=torch.float64, device=dev)
    A = torch.zeros(J, d, dtype=torch.float64, device=dev)
    B = torch.zeros(d, dtype=torch.float64, device=dev)
    G = torch.zeros(J, d, dtype=torch.float64, device=dev)
    step = max(256, int(6e7 / J))
    for s in range(0, N, step):
        n = min(step, N - s)
        z = _normals(s, n, d, key, seed, dev)
        y = z @ L.T
        dmin = t[:, :1] - y[:, 0]
        for i in range(1, d):
            dmin = torch.minimum(dmin, t[:, i:i + 1] - y[:, i])
        hits += (dmin < 0).sum(1)
        if grad:
            A += (dmin < 0).double() @ z
            B += z.sum(0)
        if grad and h > 0:
            # pairs farther than 40 h from the region's boundary add less than 1e-17
            j, m = torch.nonzero(dmin.abs() < 40.0 * h, as_tuple=True)
            keep = torch.sigmoid((t[j] - y[m]) / h)
            G.index_add_(0, j, keep.prod(1, keepdim=True) * (1.0 - keep))
    return hits, A, B, G


def _streams(hp):
    return np.unique(hp["key"]).size


def _exact_sampling(case, seed, grad, h):
    """p, se, grad_lr, grad_sig of a sampling case in FP64."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    hp = _host_problem(case, seed)
    dims = hp["dims"][hp["scen"]]
    if float((hp["n"].astype(np.float64) * dims).sum()) > EXACT_WORK * (0.08 if _streams(hp) > 512 else 1.0):
        return None
    off = np.concatenate([[0], np.cumsum(dims)])
    soff = np.concatenate([[0], np.cumsum(hp["dims"].astype(int) ** 2)])
    J = dims.size
    p, lr, sg = np.zeros(J), [None] * J, [None] * J
    for key in np.unique(hp["key"]):
        js = np.nonzero(hp["key"] == key)[0]
        s, d, N = hp["scen"][js[0]], int(dims[js[0]]), int(hp["n"][js[0]])
        L = torch.linalg.cholesky(torch.as_tensor(hp["sigma"][soff[s]:soff[s + 1]].reshape(d, d))).to(dev)
        t = np.stack([(hp["b"] - hp["mu"])[off[j]:off[j + 1]] for j in js])
        hits, A, B, G = _sums(L, torch.as_tensor(t, device=dev), N, int(key), seed, grad, h)
        ph = hits / N
        p[js] = ph.cpu().numpy()
        if not grad:
            continue
        g = torch.linalg.solve_triangular(L.T, ((A - ph[:, None] * B) / N).T, upper=True).T.cpu().numpy()
        gs = (G / (h * N)).cpu().numpy() if h > 0 else None
        for q, j in enumerate(js):
            Jm = None if hp["jac"] is None else hp["jac"][j]
            lr[j] = g[q] if Jm is None else -Jm.T @ g[q]
            if h > 0:
                sg[j] = gs[q] if Jm is None else -Jm.T @ gs[q]
    out = {"p": p}
    if grad:
        out["grad_lr"] = np.concatenate(lr)
        if h > 0:
            out["grad_sig"] = np.concatenate(sg)
    else:
        n = hp["n"].astype(np.float64)
        out["se"] = np.sqrt(p * (1.0 - p) / n)
    return out


def _exact_fwer(case, seed):
    hp = _host_problem(case, seed)
    d, N, w = case["d"], case["draws"], hp["w"]
    if float(w.size) * N * case["rounds"] > EXACT_WORK:
        return None
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    L = torch.linalg.cholesky(torch.as_tensor(hp["sigma"].reshape(d, d))).to(dev)
    lo, hi = ALPHA0 / w.sum(1), ALPHA0 / w.max(1)
    lo = np.minimum(lo, hi)
    flo, fhi, side, s = np.zeros(len(w)), np.ones(len(w)), np.zeros(len(w), int), lo.copy()
    for r in range(case["rounds"]):
        b = -_ndtri(s[:, None] * w)
        F = (_sums(L, torch.as_tensor(b, device=dev), N, 0, seed, False, 0.0)[0] / N).cpu().numpy()
        if r == case["rounds"] - 1:
            return {"scale": s, "b": b.ravel(), "fwer": F}
        if r == 0:
            flo, nxt = F, hi
        else:
            low, high = (F <= ALPHA0) & (r > 1), (F > ALPHA0) & (r > 1)
            fhi = F if r == 1 else fhi
            fhi = np.where(low & (side < 0), ALPHA0 + 0.5 * (fhi - ALPHA0), fhi)
            flo = np.where(high & (side > 0), ALPHA0 - 0.5 * (ALPHA0 - flo), flo)
            lo, flo = np.where(low, s, lo), np.where(low, F, flo)
            hi, fhi = np.where(high, s, hi), np.where(high, F, fhi)
            side = np.where(low, -1, np.where(high, 1, side))
            with np.errstate(divide="ignore", invalid="ignore"):
                nxt = np.clip(lo + (ALPHA0 - flo) * (hi - lo) / (fhi - flo), lo, hi)
            nxt = np.where(flo >= ALPHA0, lo, np.where(fhi <= ALPHA0, hi, nxt))
        s = nxt


def _eta(x, k):
    r = np.sqrt(((x[:, None, :] - x[None, :, :]) ** 2).sum(-1))
    if k == 1:
        return r ** 3
    return np.where(r > 0, r * r * np.log(np.where(r > 0, r, 1.0)), 0.0) if k == 2 else -r


def _exact_spline(x, y, s):
    """Coefficients of one smoothing spline: the saddle-point system in FP64
    with three refinement steps whose residuals take longer accumulators."""
    N, k = x.shape
    P = np.concatenate([np.ones((N, 1)), x], 1)
    A = np.zeros((N + k + 1, N + k + 1))
    A[:N, :N] = _eta(x, k) + s * np.eye(N)
    A[:N, N:], A[N:, :N] = P, P.T
    rhs = np.concatenate([y, np.zeros(k + 1)])
    T = torch.as_tensor(A)
    lu, piv = torch.linalg.lu_factor(T)
    solve = lambda v: torch.linalg.lu_solve(lu, piv, torch.as_tensor(v)[:, None])[:, 0].numpy()
    c = solve(rhs)
    Al = A.astype(np.longdouble)
    for _ in range(3):
        c = c + solve((rhs - Al @ c.astype(np.longdouble)).astype(np.float64))
    return c


def _exact_gcv(case, seed):
    x, y = _scattered(case, seed)
    x, y, k = x[0], y[0], case["k"]
    N = y.size
    Q, _ = np.linalg.qr(np.concatenate([np.ones((N, 1)), x], 1), mode="complete")
    Q2 = Q[:, k + 1:]
    lam, U = np.linalg.eigh(Q2.T @ _eta(x, k) @ Q2)
    c = U.T @ (Q2.T @ y)
    return {"score": np.array([N * ((c / (lam + s)) ** 2).sum() / (1.0 / (lam + s)).sum() ** 2
                               for s in np.logspace(-6, -2, case["values"])])}


def _exact_smooth(value, case):
    """Local-polynomial smoothing of value [S, g1, g2] (a grid with one row is
    a line): the least-squares weights of every pair of edge classes."""
    bw, deg = case["bandwidth"], case["degree"]
    R = int(math.ceil(bw)) - 1
    S, g1, g2 = value.shape
    tri = lambda u: (1.0 - np.abs(u) ** 3) ** 3
    lines = g1 == 1

    def spans(G):
        """(first, count) runs of positions whose window is cut alike."""
        edge = [(i, 1) for i in range(min(R, G))]
        mid = [(R, G - 2 * R)] if G > 2 * R else []
        tail = [(i, 1) for i in range(max(R, G - R), G)]
        return edge + mid + tail

    out = torch.empty_like(value)
    for r0, nr in ([(0, 1)] if lines else spans(g1)):
        dxs = [0] if lines else [u for u in range(-R, R + 1) if 0 <= r0 + u < g1]
        for c0, nc in spans(g2):
            dys = [v for v in range(-R, R + 1) if 0 <= c0 + v < g2]
            X = np.array([[float(u), float(v)] for u in dxs for v in dys])
            W = tri(X[:, 0] / bw) * tri(X[:, 1] / bw)
            cols = [np.ones(len(X))]
            if deg >= 1:
                cols += [X[:, 1]] if lines else [X[:, 0], X[:, 1]]
            if deg >= 2:
                cols += [X[:, 1] ** 2] if lines else [X[:, 0] ** 2, X[:, 0] * X[:, 1], X[:, 1] ** 2]
            M = np.stack(cols, 1)
            st = W * (M @ np.linalg.solve(M.T @ (W[:, None] * M), np.eye(M.shape[1])[0]))
            acc = torch.zeros(S, nr, nc, dtype=torch.float64, device=value.device)
            for wt, (u, v) in zip(st, X.astype(int)):
                acc += float(wt) * value[:, r0 + u:r0 + u + nr, c0 + v:c0 + v + nc]
            out[:, r0:r0 + nr, c0:c0 + nc] = acc
    return out


def _layout(case, vals):
    """`vals` under the names of run's outputs, None where there is no value."""
    kind = case["kind"]
    names = {"line": ["hits", "p", "se", "smoothed", "argmax_idx", "argmax_val", "raw_idx", "raw_val"],
             "fwer": ["scale", "b", "fwer"], "spline": ["coef", "fitted", "x", "f"], "gcv": ["score"],
             "smooth": ["smoothed", "argmax_idx", "argmax_val"]}.get(kind)
    if kind == "smooth" and case["raw"]:
        names += ["raw_idx", "raw_val"]
    if names is None:
        grad = kind == "step" or case["grad"]
        names = ["hits", "p"] + (["grad_lr", "grad_se"] + ([] if kind == "step" else ["grad_sig"]) if grad else ["se"])
        if case.get("smooth"):
            names += ["smoothed", "argmax_idx", "argmax_val"]
    return {n: (torch.as_tensor(vals[n]).cpu() if n in vals else None) for n in names}


def exact(case, seed):
    kind = case["kind"]
    if kind == "gcv":
        return _layout(case, _exact_gcv(case, seed))
    if kind == "spline":
        x, y = _scattered(case, seed)
        if x.shape[0] * x.shape[1] ** 2 > 5e6:
            return None
        c = np.stack([_exact_spline(x[q], y[q], case["smoothing"]) for q in range(x.shape[0])])
        return _layout(case, {"coef": c, "fitted": y - case["smoothing"] * c[:, :y.shape[1]]})
    if kind == "smooth":
        v = _grids(case, seed).double().reshape(case["scen"], case["g1"], case["g2"])
        sm = _exact_smooth(v, case)
        flat = sm.reshape(case["scen"], -1)
        vals = {"smoothed": sm.reshape(-1), "argmax_val": flat.max(1).values}
        if case["raw"]:
            vals["raw_val"] = v.reshape(case["scen"], -1).max(1).values
        return _layout(case, vals)
    if kind == "fwer":
        vals = _exact_fwer(case, seed)
        return None if vals is None else _layout(case, vals)
    grad = kind == "step" or bool(case.get("grad"))
    vals = _exact_sampling(case, seed, grad, 0.0 if kind == "step" else H)
    if vals is None:
        return None
    if kind == "line" or case.get("smooth"):
        shape = (1, 1, case["designs"]) if kind == "line" else (case["scen"], case["g1"], case["g2"])
        sm = _exact_smooth(torch.as_tensor(vals["p"]).reshape(shape), {"bandwidth": 3.0, "degree": 2})
        vals["smoothed"] = sm.reshape(-1)
        vals["argmax_val"] = sm.reshape(shape[0], -1).max(1).values
        if kind == "line":
            vals["raw_val"] = vals["p"].max(keepdims=True)
    return _layout(case, vals)
