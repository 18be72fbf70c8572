"""The workloads the sampler is timed on: what each one is, its inputs, one pass, and its answer in 64 bits.

A pass is a user's run on new observations with a sampler built once for the field: the observations go up from
pinned host memory (`Sampler.set_data`, which restarts the chains), `sweeps` chromatic Gibbs sweeps run (the first
`burn_in` of them not accumulated), and the posterior moments pooled over the chains come back into pinned memory;
programs on small fields also take every chain's state, moments and parameter traces.  The library hands every
result out as float64; what a single-precision sampler holds is float32, so a program that keeps the results keeps
them as float32, and so does `run`.

`exact` restates the method (Philox4x32-10 counters as documented in include/gmrf.h, Box-Muller, the full
conditionals class by class, Marsaglia-Tsang Gamma variates, running moments) in torch and numpy in 64 bits.
"""
import math

import numpy as np
import torch

from paper_1702_05518_gb300 import gmrf
from paper_1702_05518_gb300 import workloads as wl

DEFAULTS = {"chains": 1, "fp64": False, "rho": 1.0, "intercept": False, "weighted": False, "per_chain": False,
            "map_seed": 3}


def listed():
    return [
        # The smallest field: a 64 x 64 image in double precision, one chain (launch latency); every result is kept.
        {"name": "image64_fp64", "family": "image", "neighbours": 4, "rows": 64, "cols": 64, "chains": 1, "fp64": True,
         "sweeps": 200, "burn_in": 100, "graph_sweeps": 50, "per_chain": True},
        # The paper's simulation study: a 50 x 50 image, intercept, three chains; every result is kept.
        {"name": "paper50", "family": "image", "neighbours": 8, "rows": 50, "cols": 50, "chains": 3, "intercept": True,
         "sweeps": 500, "burn_in": 250, "graph_sweeps": 100, "per_chain": True},
        # Its scaling study's largest image: 512 x 512, noise 50 times as large, three chains.
        {"name": "paper512", "family": "image", "neighbours": 8, "rows": 512, "cols": 512, "chains": 3,
         "intercept": True, "sweeps": 300, "burn_in": 150, "graph_sweeps": 100},
        # A 1024 x 1024 image, second-order neighbours, one chain.
        {"name": "image1024", "family": "image", "neighbours": 8, "rows": 1024, "cols": 1024, "chains": 1,
         "sweeps": 400, "burn_in": 200, "graph_sweeps": 50},
        # A large image of odd extents, first-order neighbours, one chain (more tiles than the chip holds at once).
        {"name": "image_large", "family": "image", "neighbours": 4, "rows": 2047, "cols": 1931, "chains": 1,
         "sweeps": 100, "burn_in": 50, "graph_sweeps": 25},
        # An irregular areal map: Delaunay graph, proper prior, eight chains.
        {"name": "delaunay16k", "family": "graph", "sites": 16384, "chains": 8, "rho": 0.95, "sweeps": 600,
         "burn_in": 300, "graph_sweeps": 50},
        # A map of many areas with border-length weights, four chains (one launch per colour).
        {"name": "graph_weighted", "family": "graph", "sites": 100003, "chains": 4, "weighted": True, "sweeps": 200,
         "burn_in": 100, "graph_sweeps": 50},
        # Binomial counts with the logistic link on a map of precincts (Polya-Gamma augmentation), proper prior.
        {"name": "election", "family": "election", "sites": 14926, "chains": 1, "rho": 0.995, "sweeps": 200,
         "burn_in": 100, "graph_sweeps": 50, "per_chain": True},
        # Many independent fields of uneven sizes in one sampler: 112 images (sides 32 .. 512), 16 maps (1k .. 50k).
        {"name": "batched", "family": "batch", "images": 112, "graphs": 16, "chains": 1, "sweeps": 200,
         "burn_in": 100, "graph_sweeps": 25},
        # An image volume of odd extents, one chain.
        {"name": "volume_one_chain", "family": "volume", "planes": 91, "rows": 109, "cols": 91, "chains": 1,
         "sweeps": 200, "burn_in": 100, "graph_sweeps": 25},
        # A volume in double precision, two chains: the run that single precision is held against.
        {"name": "volume_fp64", "family": "volume", "planes": 48, "rows": 48, "cols": 48, "chains": 2, "fp64": True,
         "sweeps": 100, "burn_in": 50, "graph_sweeps": 25},
        # The largest: a 256^3 volume, eight chains (state far beyond the caches).
        {"name": "volume256", "family": "volume", "planes": 256, "rows": 256, "cols": 256, "chains": 8,
         "sweeps": 100, "burn_in": 50, "graph_sweeps": 25},
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def run_length(updates, most):
        # a pass of about 2e9 site-updates at most, between 20 and `most` sweeps; the run is cut
        # into graphs of 25 or 50 sweeps or launched directly
        sweeps = max(20, min(most, int(2e9 / updates), log_int(50, most)))
        return {"sweeps": sweeps, "burn_in": sweeps // 2, "graph_sweeps": rng.choice([0, 25, 50])}

    family = rng.choice(["image", "image", "image", "volume", "volume", "graph", "graph", "batch", "election"])
    if family == "image":
        fp64 = rng.random() < 0.2
        side = 512 if fp64 else 2048
        case = {"family": family, "neighbours": rng.choice([4, 8]), "rows": log_int(32, side),
                "cols": log_int(32, side), "chains": rng.choice([1, 1, 2, 3, 4, 8]), "fp64": fp64,
                "intercept": rng.random() < 0.4, "rho": rng.choice([1.0, 1.0, 0.99])}
        n = case["rows"] * case["cols"]
        return {**case, **run_length(n * case["chains"], 150 if fp64 else 400), "per_chain": n * case["chains"] <= 8192}
    if family == "volume":
        fp64 = rng.random() < 0.2
        side = 64 if fp64 else 224
        case = {"family": family, "planes": log_int(16, side), "rows": log_int(16, side), "cols": log_int(16, side),
                "chains": rng.choice([1, 1, 2, 3, 4, 6, 8]), "fp64": fp64, "intercept": rng.random() < 0.25,
                "rho": rng.choice([1.0, 1.0, 0.99])}
        updates = case["planes"] * case["rows"] * case["cols"] * case["chains"]
        return {**case, **run_length(updates, 60 if fp64 else 200)}
    if family == "graph":
        case = {"family": family, "sites": log_int(1000, 100000), "chains": rng.choice([1, 2, 3, 4, 8]),
                "rho": rng.choice([1.0, 0.95]), "weighted": rng.random() < 0.4, "map_seed": rng.randrange(1 << 16)}
        return {**case, **run_length(case["sites"] * case["chains"], 600)}
    if family == "batch":
        case = {"family": family, "images": log_int(8, 112), "graphs": rng.randint(0, 16), "chains": rng.choice([1, 2]),
                "map_seed": rng.randrange(1 << 16)}
        return {**case, **run_length(60000 * case["images"] * case["chains"], 200)}
    sites = log_int(2000, 15000)
    return {"family": family, "sites": sites, "chains": 1, "rho": 0.995, "map_seed": rng.randrange(1 << 16),
            **run_length(sites, 200), "per_chain": True}


# ---------------------------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------------------------
def _full(case):
    return {**DEFAULTS, **case}


def _volume_truth(dims, g):
    """50 solid ellipsoids, amplitudes U(0.5, 2), semi-axes U(4, 32), in a volume (built on the GPU)."""
    amp, cen = g.uniform(0.5, 2.0, 50), g.uniform(0.0, 1.0, (50, 3)) * np.array(dims)
    axes = g.uniform(4.0, 32.0, (50, 3))
    grid = [torch.arange(d, device="cuda", dtype=torch.float64) for d in dims]
    truth = torch.zeros(dims, device="cuda", dtype=torch.float64)
    for e in range(50):
        q = [((grid[k] - cen[e, k]) / axes[e, k]) ** 2 for k in range(3)]
        truth += amp[e] * ((q[0][:, None, None] + q[1][:, None] + q[2]) <= 1.0)
    return truth


def _graph(sites, map_seed, g):
    """A field on a Delaunay map of uniform points: the map belongs to the case, the observations are drawn from g."""
    rp, ci, pts = wl.delaunay_graph(sites, np.random.Generator(np.random.PCG64(map_seed)))
    truth = ((np.floor(4 * pts[:, 0]) + np.floor(4 * pts[:, 1])) % 4).astype(np.float64)
    y = truth + 0.5 * g.standard_normal(sites)
    return {"kind": gmrf.CSR, "dims": (sites, 0, 0), "n": sites, "y": y, "row_ptr": rp, "col_idx": ci,
            "color_seed": map_seed, "points": pts}


def _batch_sizes(case):
    """Image sides and graph sizes of a batch: evenly spread over the logarithms of 32 .. 512 and 1000 .. 50000."""
    def spread(lo, hi, count):
        return [int(round(lo * (hi / lo) ** ((k + 0.5) / count))) for k in range(count)]

    return spread(32, 512, case["images"]), spread(1000, 50000, case["graphs"])


def _fields(case, seed):
    """The fields of a case, as `Sampler` takes them, with observations made from the seed alone."""
    g = np.random.Generator(np.random.PCG64(seed))
    family = case["family"]
    if family == "image":
        H, W = case["rows"], case["cols"]
        kind = gmrf.LATTICE2D_4 if case["neighbours"] == 4 else gmrf.LATTICE2D_8
        if case["intercept"]:  # the paper's image; the noise of its scaling study on the large ones
            v, w = np.linspace(-3.0, 3.0, H), np.linspace(-3.0, 3.0, W)
            truth = 5.0 * np.exp(-(v[:, None] ** 2 + w[None, :] ** 2) / 2.0) / np.pi
            noise = 1.0 if H * W < 10000 else 50.0
        elif kind == gmrf.LATTICE2D_8:
            truth, noise = wl.gaussian_bumps(H, W, 20, g), 1.0
        else:
            truth, noise = wl.block_image(H, W), 0.5
        return [{"kind": kind, "dims": (H, W), "n": H * W, "y": (truth + noise * g.standard_normal((H, W))).ravel()}]
    if family == "volume":
        dims = (case["planes"], case["rows"], case["cols"])
        noise = torch.Generator(device="cuda").manual_seed(int(g.integers(1 << 40)))
        y = _volume_truth(dims, g) + torch.randn(dims, device="cuda", dtype=torch.float64, generator=noise)
        return [{"kind": gmrf.LATTICE3D_6, "dims": dims, "n": y.numel(), "y": y.reshape(-1).cpu().numpy()}]
    if family == "graph":
        f = _graph(case["sites"], case["map_seed"], g)
        if case["weighted"]:  # symmetric positive weights: one over the distance of the two areas, at most 5
            rows = np.repeat(np.arange(f["n"]), np.diff(f["row_ptr"]))
            d = np.linalg.norm(f["points"][rows] - f["points"][f["col_idx"]], axis=1) * math.sqrt(f["n"])
            f["weights"] = 1.0 / np.maximum(d, 0.2)
        return [f]
    if family == "batch":
        fields = []
        sides, sizes = _batch_sizes(case)
        for s in sides:
            y = wl.block_image(s, s) + 0.5 * g.standard_normal((s, s))
            fields.append({"kind": gmrf.LATTICE2D_4, "dims": (s, s), "n": s * s, "y": y.ravel()})
        for k, m in enumerate(sizes):
            fields.append(_graph(m, case["map_seed"] + k, g))
        return fields
    # precinct counts: trials log-uniform in 1 .. 64, one site in 45 without data, successes from the prior's logits
    f = _graph(case["sites"], case["map_seed"], g)
    m = np.floor(np.exp(g.uniform(0.0, math.log(65), f["n"]))).astype(np.int32)
    m[g.uniform(size=f["n"]) < 0.022] = 0
    truth = wl.prior_draw(f["row_ptr"], f["col_idx"], 2.0, case["rho"], g)
    f["trials"], f["y"] = m, g.binomial(m, 1.0 / (1.0 + np.exp(-0.4 - truth))).astype(np.float64)
    return [f]


def _sampler_options(case, seed):
    opts = {"precision": gmrf.FP64 if case["fp64"] else gmrf.FP32, "chains": case["chains"], "seed": seed,
            "prior": gmrf.PRIOR_ICAR if case["rho"] == 1.0 else gmrf.PRIOR_PCAR, "rho": case["rho"],
            "burn_in": case["burn_in"], "graph_sweeps": case["graph_sweeps"], "trace_capacity": case["sweeps"],
            "intercept": case["intercept"]}
    if case["intercept"]:
        opts.update(a_tau=0.001, b_tau=0.001, a_sigma=0.001, b_sigma=0.001)
    if case["family"] == "election":
        opts.update(likelihood=gmrf.LIKELIHOOD_BINOMIAL, a_tau=1.0, b_tau=1.0, beta0_prior=(0.0, 1000.0))
    return opts


class _State:
    """A sampler, its observations in pinned memory, and pinned memory for the pooled moments."""

    def __init__(self, case, seed):
        fields = _fields(case, seed)
        self.case = case
        self.sampler = gmrf.Sampler(fields, **_sampler_options(case, seed))
        self.y = [torch.from_numpy(np.ascontiguousarray(f["y"], np.float64)).pin_memory().numpy() for f in fields]
        self.trials = [f.get("trials") for f in fields]
        ends = np.cumsum([f["n"] for f in fields])
        total = int(ends[-1])
        self.pooled = torch.empty((2, total), dtype=torch.float64).pin_memory()
        self.kept = self.pooled if case["fp64"] else torch.empty((2, total), dtype=torch.float32)
        self.views = [(self.pooled[0, e - f["n"]:e].numpy(), self.pooled[1, e - f["n"]:e].numpy())
                      for f, e in zip(fields, ends)]


def prepare(case, seed):
    return _State(_full(case), int(seed))


# ---------------------------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------------------------
def run(state):
    s, case = state.sampler, state.case
    for k, y in enumerate(state.y):
        s.set_data(k, y, state.trials[k])
    s.sweep(case["sweeps"])
    for k, (mean, var) in enumerate(state.views):
        s.fetch_pooled(k, mean=mean, var=var)
    if state.kept is not state.pooled:
        state.kept.copy_(state.pooled)
    out = {"mean": state.kept[0], "var": state.kept[1]}
    if case["per_chain"]:
        kind = np.float64 if case["fp64"] else np.float32
        binomial = case["family"] == "election"
        for c in range(case["chains"]):
            r = s.fetch(0, c, trace=case["sweeps"])
            for key in ("x", "mean", "var", "tau_trace") + (() if binomial else ("sigma2_trace",)):
                out["%s_%d" % (key, c)] = r[key].astype(kind)
            if binomial or case["intercept"]:
                out["beta0_trace_%d" % c] = s.fetch_intercept(0, c, trace=case["sweeps"])["beta0_trace"].astype(kind)
    return out


# ---------------------------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------------------------
def _sites(case):
    """(sites, directed neighbour pairs, bytes of graph structure) of a case."""
    family = case["family"]
    if family == "image":
        n = case["rows"] * case["cols"]
        return n, n * case["neighbours"], 0
    if family == "volume":
        n = case["planes"] * case["rows"] * case["cols"]
        return n, n * 6, 0
    if family == "batch":
        sides, sizes = _batch_sizes(case)
        lat, gra = sum(s * s for s in sides), sum(sizes)
        return lat + gra, 4 * lat + 6 * gra, gra * 28
    n = case["sites"]
    return n, n * 6, n * (28 + (48 if case["weighted"] else 0))


def work(case):
    """Per sweep every chain's state is read and written once, the observations and the graph are read once; an
    accumulated sweep also reads and writes the running mean and squared deviations; the observations come in and
    the pooled moments go out once.  Per site-update: two operations per neighbour for its sum and two for its edge
    in the prior's quadratic form (each edge once), 15 for the update and the sums, 40 for the random numbers."""
    case = _full(case)
    n, pairs, graph = _sites(case)
    S, C, T = 8 if case["fp64"] else 4, case["chains"], case["sweeps"]
    acc = T - case["burn_in"]
    nbytes = T * (2 * n * C * S + n * S + graph) + acc * 4 * n * C * S + 8 * n + 2 * n * S
    return {"bytes": nbytes, "flops": T * C * (2.0 * pairs + 55.0 * n)}


# ---------------------------------------------------------------------------------------------
# The answer in 64 bits
# ---------------------------------------------------------------------------------------------
M32 = 0xFFFFFFFF


def _philox(c, seed):
    """Philox4x32-10 (Salmon et al., SC'11) of four int64 counter words (tensors or arrays, each below 2^32)."""
    k0, k1 = seed & M32, (seed >> 32) & M32
    c0, c1, c2, c3 = c
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = ((p1 >> 32) & M32) ^ c1 ^ k0, p1 & M32, ((p0 >> 32) & M32) ^ c3 ^ k1, p0 & M32
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return c0, c1, c2, c3


def _uniform(w):
    return ((w.double() if torch.is_tensor(w) else w) + 0.5) * 2.0 ** -32


def _box_muller(wa, wb):
    r, t = torch.sqrt(-2.0 * torch.log(_uniform(wa))), 2.0 * math.pi * _uniform(wb)
    return r * torch.cos(t), r * torch.sin(t)


def _gammas(shape, tag, T, streams, C, seed):
    """Unit-rate Marsaglia-Tsang variates [T, fields, C] of one parameter (shape: per field)."""
    a0 = np.broadcast_to(np.asarray(shape, np.float64)[None, :, None], (T, len(streams), C)).ravel()
    sweep, stream, chain = (v.ravel() for v in
                            np.meshgrid(np.arange(T), np.asarray(streams), np.arange(C), indexing="ij"))
    boost = a0 < 1.0
    a = np.where(boost, a0 + 1.0, a0)
    d = a - 1.0 / 3.0
    c = 1.0 / np.sqrt(9.0 * d)
    out = d.copy()
    todo = np.arange(len(a))
    for attempt in range(64):
        with np.errstate(over="ignore"):
            w = _philox((np.full(len(todo), attempt, np.int64), sweep[todo].astype(np.int64),
                         stream[todo].astype(np.int64), (tag << 24) | chain[todo].astype(np.int64)), seed)
        z = np.sqrt(-2.0 * np.log(_uniform(w[0]))) * np.cos(2.0 * math.pi * _uniform(w[1]))
        v = 1.0 + c[todo] * z
        ok = v > 0.0
        v = np.where(ok, v, 1.0) ** 3
        dd = d[todo]
        ok &= np.log(_uniform(w[2])) < 0.5 * z * z + dd - dd * v + dd * np.log(v)
        g = dd * v * np.where(boost[todo], _uniform(w[3]) ** (1.0 / a0[todo]), 1.0)
        out[todo[ok]] = g[ok]
        todo = todo[~ok]
        if not len(todo):
            break
    return out.reshape(T, len(streams), C)


def _beta_normals(T, streams, C, seed):
    sweep, stream, chain = (v.ravel().astype(np.int64) for v in
                            np.meshgrid(np.arange(T), np.asarray(streams), np.arange(C), indexing="ij"))
    with np.errstate(over="ignore"):
        w = _philox((np.zeros_like(sweep), sweep, stream, (7 << 24) | chain), seed)
    z = np.sqrt(-2.0 * np.log(_uniform(w[0]))) * np.cos(2.0 * math.pi * _uniform(w[1]))
    return z.reshape(T, len(streams), C)


def _lattice_neighbours(field):
    """(neighbours [n, D], -1 where there is none; colours [n]) of a lattice field, on the GPU."""
    dims = [int(d) for d in field["dims"]]
    idx = torch.arange(field["n"], device="cuda").reshape(dims)
    at = torch.meshgrid(*[torch.arange(d, device="cuda") for d in dims], indexing="ij")
    if field["kind"] == gmrf.LATTICE2D_8:
        steps = [(a, b) for a in (-1, 0, 1) for b in (-1, 0, 1) if a or b]
        colour = 2 * (at[0] & 1) + (at[1] & 1)
    else:
        eye = np.eye(len(dims), dtype=int)
        steps = [tuple(int(v) for v in s * e) for e in eye for s in (-1, 1)]
        colour = sum(at) & 1
    cols = []
    for st in steps:
        inside = torch.ones(dims, dtype=torch.bool, device="cuda")
        off = 0
        for k, d in enumerate(dims):
            inside &= (at[k] + st[k] >= 0) & (at[k] + st[k] < d)
            off = off * d + st[k]
        cols.append(torch.where(inside, idx + off, -1).reshape(-1).to(torch.int32))
    return torch.stack(cols, 1), colour.reshape(-1)


def _greedy(field):
    """First-fit greedy colouring, vertices by decreasing (min(degree, 255), random priority, index)."""
    rp, ci, n = field["row_ptr"], field["col_idx"], field["n"]
    v = np.arange(n, dtype=np.int64)
    with np.errstate(over="ignore"):
        w = _philox((v, v * 0, v * 0, v * 0 + (3 << 24)), int(field["color_seed"]))[0]
    prio = (np.minimum(np.diff(rp).astype(np.int64), 255) << 24) | (w >> 8)
    order = np.lexsort((v, prio))[::-1]
    colours, cl, rl = [-1] * n, ci.tolist(), rp.tolist()
    for i in order.tolist():
        taken = {colours[j] for j in cl[rl[i]:rl[i + 1]]}
        c = 0
        while c in taken:
            c += 1
        colours[i] = c
    return torch.tensor(colours, device="cuda")


def _graph_neighbours(field):
    rp, ci = field["row_ptr"].astype(np.int64), field["col_idx"]
    deg = np.diff(rp)
    rows, k = np.repeat(np.arange(field["n"]), deg), np.arange(len(ci)) - np.repeat(rp[:-1], deg)
    nbr = np.full((field["n"], int(deg.max())), -1, np.int32)
    nbr[rows, k] = ci
    w = np.zeros(nbr.shape)
    w[rows, k] = field.get("weights", np.ones(len(ci)))
    return torch.from_numpy(nbr).cuda(), torch.from_numpy(w).cuda()


def _components(field):
    if field["kind"] != gmrf.CSR:
        return 1
    from scipy.sparse import csr_matrix
    from scipy.sparse.csgraph import connected_components

    m = csr_matrix((np.ones(len(field["col_idx"])), field["col_idx"], field["row_ptr"]), shape=(field["n"],) * 2)
    return int(connected_components(m, directed=False)[0])


def _exact_moments(case, seed):
    """All fields as one graph of n sites: per-site tensors [n, C], per-field parameters [fields, C]."""
    fields = _fields(case, seed)
    opts = _sampler_options(case, seed)
    C, T, burn, rho = case["chains"], case["sweeps"], case["burn_in"], case["rho"]
    F, f64 = len(fields), torch.float64
    n_of = np.array([f["n"] for f in fields], np.float64)
    start = np.concatenate([[0], np.cumsum([f["n"] for f in fields])])
    n = int(start[-1])
    fid = torch.repeat_interleave(torch.arange(F, device="cuda"), torch.tensor([f["n"] for f in fields], device="cuda"))
    colour = torch.empty(n, dtype=torch.int64, device="cuda")
    parts = []
    for k, f in enumerate(fields):
        if f["kind"] == gmrf.CSR:
            nbr, w = _graph_neighbours(f)
            colour[start[k]:start[k + 1]] = _greedy(f)
        else:
            nbr, col = _lattice_neighbours(f)
            colour[start[k]:start[k + 1]] = col
            w = None
        parts.append((torch.where(nbr >= 0, nbr + int(start[k]), n), w))
    D = max(p[0].shape[1] for p in parts)
    weighted = any(p[1] is not None for p in parts)
    nbr = torch.full((n, D), n, dtype=torch.int32, device="cuda")
    wts = torch.zeros((n, D), dtype=f64, device="cuda") if weighted else None
    for k, (p, w) in enumerate(parts):
        nbr[start[k]:start[k + 1], :p.shape[1]] = p
        if weighted:
            wts[start[k]:start[k + 1], :p.shape[1]] = (p < n).to(f64) if w is None else w
    del parts
    deg = wts.sum(1) if weighted else (nbr < n).sum(1).to(f64)
    classes = [(i := torch.nonzero(colour == c).reshape(-1), nbr[i], None if wts is None else wts[i])
               for c in range(int(colour.max()) + 1)]
    y = torch.cat([torch.from_numpy(np.ascontiguousarray(f["y"])) for f in fields]).cuda()
    site = torch.cat([torch.arange(f["n"], device="cuda") for f in fields])

    rank = n_of - np.array([_components(f) for f in fields]) if rho == 1.0 else n_of
    prior = {k: opts.get(k, v) for k, v in (("a_tau", 1.0), ("b_tau", 0.01), ("a_sigma", 1.0), ("b_sigma", 0.01))}
    g_tau = torch.from_numpy(_gammas(prior["a_tau"] + 0.5 * rank, 1, T, range(F), C, seed)).cuda()
    g_sig = torch.from_numpy(_gammas(prior["a_sigma"] + 0.5 * n_of, 2, T, range(F), C, seed)).cuda()
    z_beta = torch.from_numpy(_beta_normals(T, range(F), C, seed)).cuda()
    nf = torch.from_numpy(n_of).cuda()[:, None]

    lanes = 1 if C == 1 else 2 if C == 2 else 4
    shift = {4: 0, 2: 1, 1: 2}[lanes]

    def normals(t):
        out = []
        for q in range(-(-C // 4)):
            w = _philox((site >> shift, torch.full_like(site, t), fid, torch.full_like(site, q)), seed)
            z = torch.stack(_box_muller(w[0], w[1]) + _box_muller(w[2], w[3]), 1)
            if lanes < 4:
                first = (site & ((1 << shift) - 1)) * lanes
                z = torch.gather(z, 1, first[:, None] + torch.arange(lanes, device="cuda"))
            out.append(z)
        return torch.cat(out, 1)[:, :C]

    def by_field(v):  # sums over the sites of each field
        return v.sum(0, keepdim=True) if F == 1 else torch.zeros((F, C), dtype=f64, device="cuda").index_add_(0, fid, v)

    def per_site(p, i=None):  # a parameter's value at each site
        return p if F == 1 else p[fid if i is None else fid[i]]

    x = torch.zeros((n + 1, C), dtype=f64, device="cuda")
    x[:n] = y[:, None]
    tau = torch.ones((F, C), dtype=f64, device="cuda")
    s2, beta = tau.clone(), torch.zeros_like(tau)
    mean, m2 = torch.zeros((n, C), dtype=f64, device="cuda"), torch.zeros((n, C), dtype=f64, device="cuda")
    traces = {"tau": [], "sigma2": [], "beta0": []}
    for t in range(T):
        z = normals(t)
        for i, nb, w in classes:
            s = torch.zeros((len(i), C), dtype=f64, device="cuda")
            for k in range(D):
                xn = x[nb[:, k]]
                s += xn if w is None else w[:, k:k + 1] * xn
            tt, ss = per_site(tau, i), 1.0 / per_site(s2, i)
            P = tt * deg[i][:, None] + ss
            x[i] = (tt * rho * s + (y[i][:, None] - per_site(beta, i)) * ss) / P + z[i] / torch.sqrt(P)
        del z
        quad = torch.zeros((n, C), dtype=f64, device="cuda")
        for k in range(D):
            d = x[:n] - x[nbr[:, k]]
            quad += (0.5 * rho) * (d * d) * ((nbr[:, k] < n)[:, None] if wts is None else wts[:, k:k + 1])
        if rho != 1.0:
            quad += (1.0 - rho) * deg[:, None] * x[:n] ** 2
        if case["intercept"]:
            beta = by_field(y[:, None] - x[:n]) / nf + torch.sqrt(s2 / nf) * z_beta[t]
        tau = g_tau[t] / (prior["b_tau"] + 0.5 * by_field(quad))
        s2 = (prior["b_sigma"] + 0.5 * by_field((y[:, None] - per_site(beta) - x[:n]) ** 2)) / g_sig[t]
        traces["tau"].append(tau)
        traces["sigma2"].append(s2)
        traces["beta0"].append(beta)
        if t >= burn:
            d = x[:n] - mean
            mean += d / (t - burn + 1)
            m2 += d * (x[:n] - mean)
    return x[:n], mean, m2, T - burn, {k: torch.stack(v) for k, v in traces.items()}


def exact(case, seed):
    case = _full(case)
    if case["family"] == "election":
        return None  # the augmentation's accept/reject steps depend on the rounding of the state
    x, mean, m2, kept, traces = _exact_moments(case, int(seed))
    C = case["chains"]
    mu = mean.mean(1)
    var = (m2 + kept * (mean - mu[:, None]) ** 2).sum(1) / (C * kept - 1)
    out = {"mean": mu.cpu(), "var": var.cpu()}
    if case["per_chain"]:
        for c in range(C):
            out["x_%d" % c], out["mean_%d" % c] = x[:, c].cpu(), mean[:, c].cpu()
            out["var_%d" % c] = (m2[:, c] / (kept - 1)).cpu()
            out["tau_trace_%d" % c] = traces["tau"][:, 0, c].cpu()
            out["sigma2_trace_%d" % c] = traces["sigma2"][:, 0, c].cpu()
            if case["intercept"]:
                out["beta0_trace_%d" % c] = traces["beta0"][:, 0, c].cpu()
    return out
