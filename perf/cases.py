"""Performance cases of the PCF integral-matrix library.

Each case is one call (or one training step) a user's program makes through
the package's public functions, on seeded synthetic collections of the kinds
the library is tested and benchmarked on (the recipes of
``paper_2404_07183_gb300.synth``, drawn on the GPU).  Schedules, precisions
and checks are the defaults of those functions unless a comment says why not.
"""
import math

import torch

import paper_2404_07183_gb300 as P

METRICS3 = ["l1", "l2", "gram"]
CROSS3 = ["l1", "l2", ("lp", 3.0)]


def listed():
    return [
        # the smallest call: the distance matrix of a handful of curves, in a script or
        # a notebook (few pairs: latency, launches and the input check are what counts)
        {"name": "pdist_tiny", "kind": "pdist", "n": 97},
        # the paper's ordinary call: float64 L1 distances of a thousand short curves
        {"name": "pdist_1000", "kind": "pdist", "n": 1000},
        # a service that compares batches of a few hundred curves over and over, with its
        # workspace and matrices kept and the check left to the end of its loop
        {"name": "curves_batch", "kind": "curves_kept", "n": 701},
        # the library's main workload at its full size: three float32 matrices of 20,000
        # stable-rank curves given in float64
        {"name": "curves_20000", "kind": "curves", "n": 20000, "precision": "f32c"},
        # the same curves where float64 results are wanted
        {"name": "curves_float64", "kind": "curves", "n": 2501, "precision": "f64"},
        # a Gram matrix for a kernel method over very uneven float32 curves, upper triangle
        {"name": "uneven_gram", "kind": "uneven_gram", "n": 30000},
        # one step of fitting curves by their L2 distances: forward and backward
        {"name": "l2_training_step", "kind": "training_step", "n": 2048},
        # train-against-test block of Euler-curve-like float32 curves, p = 1, 2, 3 at once
        {"name": "euler_cross", "kind": "euler_cross", "n": 3001, "m": 4000, "points": 1000},
        # the paper's synthetic recipe: long curves on very different time scales, float32
        # L1 distances of float64 curves
        {"name": "scales_l1", "kind": "scales_l1", "n": 9001},
        # norms of a large collection (one pass over its breakpoints)
        {"name": "norms_100000", "kind": "norms", "n": 100000},
        # the mean curve of each group of a large collection (real values: every breakpoint
        # of a group stays in its mean)
        {"name": "group_means", "kind": "group_means", "groups": 160, "m": 128},
        # a few very long curves (high-resolution recordings)
        {"name": "few_long", "kind": "few_long", "n": 25, "points": 60001},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["pdist", "curves_kept", "curves", "uneven_gram", "training_step",
                       "euler_cross", "scales_l1", "norms", "group_means", "few_long"])
    c = {"kind": kind}
    if kind == "pdist":
        c["n"] = _log_int(rng, 20, 1000)
    elif kind == "curves_kept":
        c["n"] = _log_int(rng, 200, 2000)
    elif kind == "curves":
        c["precision"] = rng.choice(["f32c", "f64"])
        c["n"] = _log_int(rng, 1000, 16000 if c["precision"] == "f32c" else 2500)
    elif kind == "uneven_gram":
        c["n"] = _log_int(rng, 3000, 30000)
    elif kind == "training_step":
        c["n"] = _log_int(rng, 150, 2048)
    elif kind == "euler_cross":
        c["n"], c["m"] = _log_int(rng, 300, 3000), _log_int(rng, 300, 4000)
        c["points"] = _log_int(rng, 100, 1000)
    elif kind == "scales_l1":
        c["n"] = _log_int(rng, 1000, 9000)
    elif kind == "norms":
        c["n"] = _log_int(rng, 3000, 100000)
    elif kind == "group_means":
        c["m"] = rng.randint(5, 128)
        c["groups"] = _log_int(rng, 4, 160)
    else:
        c["n"], c["points"] = rng.randint(5, 25), _log_int(rng, 5000, 60000)
    return c


# ---- inputs ----------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _offsets(lens):
    o = torch.zeros(lens.numel() + 1, dtype=torch.int64, device="cuda")
    o[1:] = torch.cumsum(lens, 0)
    return o


def _strict(offsets, t):
    """Times that rounded together moved up by one ulp (strictly increasing curves)."""
    first = torch.zeros(t.numel(), dtype=torch.bool, device=t.device)
    first[offsets[:-1]] = True
    for _ in range(1000):
        bad = ((t[1:] <= t[:-1]) & ~first[1:]).nonzero().flatten() + 1
        if bad.numel() == 0:
            return t
        t[bad] = torch.nextafter(t[bad - 1], torch.full_like(t[bad], math.inf))
    raise RuntimeError("could not make times strictly increasing")


def _padded(lens):
    """Mask of the entries (i, k), k < lens[i], of a rectangular array."""
    k = torch.arange(int(lens.max()), device="cuda")
    return k[None, :] < lens[:, None]


def _walk_times(g, lens, mean=1.0):
    """Running sums of exponential gaps from 0, curve by curve, in float64 (the few
    curves of more than 512 breakpoints in a rectangle of their own)."""
    out = torch.empty(int(lens.sum()), dtype=torch.float64, device="cuda")
    is_long = lens > 512
    for rows in (~is_long, is_long):
        if not bool(rows.any()):
            continue
        m = _padded(lens[rows])
        t = torch.empty(m.shape, dtype=torch.float64, device="cuda")
        t.exponential_(1.0 / mean, generator=g)
        t[:, 0] = 0.0
        out[torch.repeat_interleave(rows, lens)] = torch.cumsum(t, 1)[m]
    return out


def _set(lens, t, v, dtype=torch.float64):
    o = _offsets(lens)
    return P.PcfTensors(o, _strict(o, t.to(dtype)), v.to(dtype))


def _normals_last_zero(g, lens):
    v = torch.randn(int(lens.sum()), dtype=torch.float64, device="cuda", generator=g)
    v[torch.cumsum(lens, 0) - 1] = 0.0
    return v


def _lens(g, n, lo, hi):
    """Breakpoint counts spread evenly over lo .. hi, in a random order (the same total
    for every seed)."""
    lens = lo + torch.arange(n, device="cuda") * (hi - lo + 1) // n
    return lens[torch.randperm(n, device="cuda", generator=g)]


def _short_curves(seed, n, lo=10, hi=100):
    g = _gen(seed)
    lens = _lens(g, n, lo, hi)
    return _set(lens, _walk_times(g, lens), _normals_last_zero(g, lens))


def _stable_rank(seed, n):
    """50 to 500 breakpoints, gaps of mean 0.1, non-increasing integers from 200 to 0."""
    g = _gen(seed)
    lens = _lens(g, n, 50, 500)
    m = _padded(lens)
    k = torch.arange(m.shape[1], device="cuda")[None, :]
    v = torch.randint(0, 201, m.shape, device="cuda", generator=g)
    v[k >= lens[:, None] - 2] = -1
    mid = torch.sort(v, dim=1, descending=True).values[:, :-1]
    v[:, 1:] = mid.clamp_(min=0)
    v[:, 0] = 200
    v[k == lens[:, None] - 1] = 0
    return _set(lens, _walk_times(g, lens, 0.1), v[m].double())


def _uneven(seed, n):
    """Log-normal breakpoint counts (median 100, 2 to 10,000), float32."""
    g = _gen(seed)
    z = torch.special.ndtri((torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) / n)
    lens = torch.exp(z + math.log(100.0)).round().clamp(2, 10000).long()
    lens = lens[torch.randperm(n, device="cuda", generator=g)]
    return _set(lens, _walk_times(g, lens), _normals_last_zero(g, lens), torch.float32)


def _euler(g, n, points):
    """Integer random walks (steps of 1 to 3 either way) at exponential times, float32."""
    lens = torch.full((n,), points, device="cuda")
    j = torch.randint(1, 4, (n, points), device="cuda", generator=g)
    j *= 2 * torch.randint(0, 2, (n, points), device="cuda", generator=g) - 1
    j[:, 0] = 0
    v = torch.cumsum(j, 1).double()
    v[:, -1] = 0.0
    return _set(lens, _walk_times(g, lens), v.flatten(), torch.float32)


def _scales(seed, n):
    """10 to 1,000 breakpoints at |alpha| * sorted |normal| times, normal values."""
    g = _gen(seed)
    lens = _lens(g, n, 10, 1000)
    m = _padded(lens)
    alpha = torch.randn(n, dtype=torch.float64, device="cuda", generator=g).abs()
    t = torch.randn(m.shape, dtype=torch.float64, device="cuda", generator=g).abs()
    t[~m] = math.inf
    t[:, 0] = -1.0
    t = torch.sort(t, dim=1).values * alpha[:, None]
    t[:, 0] = 0.0
    return _set(lens, t[m], _normals_last_zero(g, lens))


def prepare(case, seed):
    kind = case["kind"]
    if kind == "pdist":
        x = _short_curves(seed, case["n"])
    elif kind in ("curves", "curves_kept"):
        x = _stable_rank(seed, case["n"])
    elif kind in ("uneven_gram", "norms"):
        x = _uneven(seed, case["n"])
    elif kind == "training_step":
        x = _short_curves(seed, case["n"], 20, 200)
    elif kind == "euler_cross":
        g = _gen(seed)
        x = _euler(g, case["n"], case["points"])
    elif kind == "scales_l1":
        x = _scales(seed, case["n"])
    elif kind == "group_means":
        x = _short_curves(seed, case["groups"] * case["m"], 50, 500)
    else:
        g = _gen(seed)
        lens = _lens(g, case["n"], case["points"] * 4 // 5, case["points"])
        x = _set(lens, _walk_times(g, lens), _normals_last_zero(g, lens), torch.float32)
    state = {"case": case, "x": x}
    if kind == "curves_kept":
        n = case["n"]
        state["out"] = [torch.empty(n, n, device="cuda") for _ in METRICS3]
        state["workspace"] = torch.empty(P.pcf_workspace_size(x, None, "f32c"), dtype=torch.uint8,
                                         device="cuda")
    elif kind == "euler_cross":
        state["y"] = _euler(g, case["m"], case["points"])
    elif kind == "training_step":
        n = case["n"]
        state["g"] = torch.randn(n, n, dtype=torch.float64, device="cuda",
                                 generator=_gen(seed + 1_000_003))
        x.values.requires_grad_(True)
        x.times.requires_grad_(True)
    return state


# ---- one pass --------------------------------------------------------------

def run(state):
    case, x = state["case"], state["x"]
    kind = case["kind"]
    if kind == "pdist":
        return P.pdist(x)
    if kind == "curves_kept":
        return P.pcf_pairwise(x, METRICS3, out=state["out"], workspace=state["workspace"],
                              check=False)
    if kind == "curves":
        return P.pcf_pairwise(x, METRICS3, precision=case["precision"],
                              out_dtype=torch.float64 if case["precision"] == "f64"
                              else torch.float32)
    if kind == "uneven_gram":
        return P.pcf_pairwise(x, "gram", layout="upper")
    if kind == "training_step":
        d = P.PairwiseFn.apply(x.values, x.times, x.offsets)
        gv, gt = torch.autograd.grad(d, (x.values, x.times), state["g"])
        return {"distances": d.detach(), "grad_values": gv, "grad_times": gt}
    if kind == "euler_cross":
        return P.pcf_cross(x, state["y"], metrics=CROSS3)
    if kind == "scales_l1":
        return P.pcf_pairwise(x)
    if kind == "norms":
        return P.pcf_segment_integrals(x, "lp", 2.0, True, precision="f32c")
    if kind == "group_means":
        r = P.mean(x, case["m"])
        return {"offsets": r.offsets, "times": r.times, "values": r.values}
    return P.pcf_pairwise(x)


# ---- what a pass cannot do without -----------------------------------------

def work(case):
    """Inputs read once and outputs written once; per rectangle of a merge walk its width,
    and per metric the integrand and one fused multiply-add (counted as two)."""
    kind = case["kind"]
    mean_len = {"pdist": 55.0, "curves": 275.0, "curves_kept": 275.0, "uneven_gram": 164.9,
                "training_step": 110.0, "scales_l1": 505.0, "norms": 164.9, "group_means": 275.0}
    if kind == "euler_cross":
        pairs, length = case["n"] * case["m"], float(case["points"])
        return {"bytes": 8.0 * length * (case["n"] + case["m"]) + 12.0 * pairs,
                "flops": pairs * 2.0 * length * (2 + 2 + 3 + 4)}
    if kind == "few_long":
        length, pairs = 0.9 * case["points"], case["n"] * (case["n"] + 1) / 2.0
        return {"bytes": 8.0 * length * case["n"] + 4.0 * case["n"] ** 2,
                "flops": pairs * 2.0 * length * 4}
    length = mean_len[kind]
    if kind == "norms":
        return {"bytes": 8.0 * length * case["n"] + 16.0 * case["n"],
                "flops": 4.0 * length * case["n"]}
    if kind == "group_means":
        nnz = length * case["groups"] * case["m"]
        # every breakpoint is read once and appears once in its group's mean
        return {"bytes": 32.0 * nnz, "flops": nnz * math.ceil(math.log2(case["m"]))}
    n = case["n"]
    pairs = n * (n + 1) / 2.0
    steps = pairs * (2.0 * length - 1.0)
    if kind == "uneven_gram":
        return {"bytes": 8.0 * length * n + 4.0 * pairs, "flops": steps * 4}
    if kind == "scales_l1":
        return {"bytes": 16.0 * length * n + 4.0 * n * n, "flops": steps * 4}
    if kind == "pdist":
        return {"bytes": 16.0 * length * n + 8.0 * n * n, "flops": steps * 4}
    if kind == "training_step":
        # the forward's L2 walk and the walk of the adjoint
        return {"bytes": 48.0 * length * n + 16.0 * n * n, "flops": steps * (5 + 10)}
    size = 8 if case.get("precision") == "f64" else 4
    return {"bytes": 16.0 * length * n + 3.0 * size * n * n, "flops": steps * 10}


# ---- the results in 64 bits ------------------------------------------------

def _rect(x):
    """Times (padded by inf) and values (padded by each curve's last) as rectangular float64."""
    lens = x.offsets[1:] - x.offsets[:-1]
    m = _padded(lens)
    T = torch.full(m.shape, math.inf, dtype=torch.float64, device="cuda")
    V = x.values.detach().double()[x.offsets[1:] - 1][:, None].repeat(1, m.shape[1])
    T[m] = x.times.detach().double()
    V[m] = x.values.detach().double()
    return T, V


def _row(t, v, T, V, metrics):
    """Integrals of one curve (t, v) against every row of (T, V): on the union of each pair's
    breakpoints, both curves read by binary search."""
    U = torch.sort(torch.cat([T, t[None, :].expand(T.shape[0], -1)], 1), dim=1).values
    L = U[:, :-1].contiguous()
    w = U[:, 1:] - L
    w[~torch.isfinite(w)] = 0.0
    a = v[(torch.searchsorted(t, L, right=True) - 1).clamp_(min=0)]
    b = torch.gather(V, 1, (torch.searchsorted(T, L, right=True) - 1).clamp_(min=0))
    out = []
    for m in metrics:
        if m == "gram":
            out.append((a * b * w).sum(1))
        else:
            p = {"l1": 1.0, "l2": 2.0}[m] if isinstance(m, str) else m[1]
            out.append(((a - b).abs().pow(p) * w).sum(1).pow(1.0 / p))
    return out


def _matrices(x, y, metrics):
    Tx, Vx = _rect(x)
    Ty, Vy = _rect(y)
    last = (x.offsets[1:] - x.offsets[:-1]).tolist()
    rows = [_row(Tx[i, :last[i]].contiguous(), Vx[i, :last[i]], Ty, Vy, metrics)
            for i in range(x.n)]
    return [torch.stack([r[k] for r in rows]) for k in range(len(metrics))]


def _exact_step(state):
    """Distances, and the gradients of sum(G * distances): each distance's slope 1 / (2 d)
    times the slopes of int (f - g)^2 in f's values and breakpoints."""
    x, G = state["x"], state["g"]
    D = _matrices(x, x, ("l2",))[0]
    D.fill_diagonal_(0.0)
    W = (G + G.T) / (2.0 * torch.where(D > 0, D, torch.ones_like(D)))
    W.fill_diagonal_(0.0)
    t, v, o = x.times.detach(), x.values.detach(), x.offsets
    lens = o[1:] - o[:-1]
    row = torch.repeat_interleave(torch.arange(x.n, device="cuda"), lens)
    last = torch.zeros(t.numel(), dtype=torch.bool, device="cuda")
    last[o[1:] - 1] = True
    first = torch.zeros_like(last)
    first[o[:-1]] = True
    nxt = torch.where(last, t, torch.roll(t, -1))
    before = torch.where(first, v, torch.roll(v, 1))
    gv, gt = torch.zeros_like(t), torch.zeros_like(t)
    for j in range(x.n):
        tj, vj = t[o[j]:o[j + 1]], v[o[j]:o[j + 1]]
        A = torch.zeros_like(tj)
        A[1:] = torch.cumsum(vj[:-1] * (tj[1:] - tj[:-1]), 0)
        k = torch.searchsorted(tj, t, right=True) - 1
        F = A[k] + vj[k] * (t - tj[k])
        part = torch.where(last, A[-1] - F, torch.roll(F, -1) - F)   # all curves end at 0
        w = W[row, j]
        gv += 2.0 * w * (v * (nxt - t) - part)
        g = vj[(torch.searchsorted(tj, t) - 1).clamp_(min=0)]
        gt += w * ((before - g) ** 2 - (v - g) ** 2)
    gt[first] = 0.0
    return {"distances": D, "grad_values": gv, "grad_times": gt}


def _exact_means(x, m):
    """The changes of a group's curves in time order, summed within the group."""
    o = x.offsets
    lens = o[1:] - o[:-1]
    group = torch.repeat_interleave(torch.arange(x.n, device="cuda") // m, lens)
    jump = x.values.clone()
    inner = torch.ones(jump.numel(), dtype=torch.bool, device="cuda")
    inner[o[:-1]] = False
    jump[inner] -= x.values[:-1][inner[1:]]
    order = torch.argsort(x.times, stable=True)
    order = order[torch.argsort(group[order], stable=True)]
    t, g = x.times[order], group[order]
    total = torch.cumsum(jump[order], 0)          # every group's curves end at 0
    end = torch.ones(t.numel(), dtype=torch.bool, device="cuda")
    end[:-1] = (t[1:] != t[:-1]) | (g[1:] != g[:-1])
    return {"offsets": None, "times": t[end], "values": total[end] / m}


def exact(case, seed):
    kind, n = case["kind"], case.get("n", 0)
    too_long = {"curves": 2600, "uneven_gram": 0, "euler_cross": 0, "scales_l1": 0}
    if n > too_long.get(kind, n):
        return None
    state = prepare(case, seed)
    x = state["x"]
    if kind == "pdist":
        return _matrices(x, x, ("l1",))[0]
    if kind in ("curves", "curves_kept"):
        return _matrices(x, x, METRICS3)
    if kind == "training_step":
        return _exact_step(state)
    if kind == "norms":
        lens = x.offsets[1:] - x.offsets[:-1]
        t, v = x.times.double(), x.values.double()
        w = torch.zeros_like(t)
        w[:-1] = t[1:] - t[:-1]
        w[x.offsets[1:] - 1] = 0.0
        i = torch.repeat_interleave(torch.arange(x.n, device="cuda"), lens)
        return torch.zeros(x.n, dtype=torch.float64, device="cuda").index_add_(0, i, v * v * w).sqrt()
    if kind == "group_means":
        return _exact_means(x, case["m"])
    return _matrices(x, x, ("l1",))
