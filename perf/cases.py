"""Performance cases of the triad-census library: what its users have it do, with seeded inputs.

Every case goes through the public binding, as a user's program does:

  census    a census of a graph that is resident on the GPU, the counts on the host (`tc_census`)
            or left on the device (`tc_census_async`, the form for back-to-back censuses)
  build     arcs to counts: build the graph from an arc list, take its census, drop it
  batch     one launch over many small graphs, replayed
  serve     a burst of requests on the graphs of a running server
  interval  a monitoring session: arcs pushed as they arrive, a census of the window at intervals
  census64  the 64 labelled triad states of a resident graph
  matrix    the dense (matrix) form of a resident graph's census

The graphs are R-MAT (a, b, c, d = .57, .19, .19, .05, ids permuted) and Chung-Lu (exponent 2.1),
the generators of this repository's tests and benchmark, drawn here on the GPU: raw arc lists
with the loops and repeats that such draws hold, and a share of the arcs also reversed.
"""
import math
import random

import numpy as np
import torch

import paper_1209_6308_gb300 as tc

TRIANGLE = {"algo": tc.TC_ALGO_TRIANGLE}
LIMB = (1 << 62) - 1          # counts above 62 bits are returned as two limbs
CHUNK = 1 << 25               # arcs drawn at a time


def listed():
    return [
        # the smallest call: a census of a few thousand arcs, where launches and the wait count
        {"name": "census_rmat10", "kind": "census", "graph": "rmat", "scale": 10, "degree": 16, "recip": 0.15,
         "form": "triangle", "wait": True},
        # the medium workload, lists that fit the L2
        {"name": "census_rmat20", "kind": "census", "graph": "rmat", "scale": 20, "degree": 16, "recip": 0.2,
         "form": "triangle", "wait": False},
        # the largest single-GPU workload, 1.3 G arcs
        {"name": "census_rmat26", "kind": "census", "graph": "rmat", "scale": 26, "degree": 16, "recip": 0.2,
         "form": "triangle", "wait": False},
        # a call with no options set (the union walk), odd sizes
        {"name": "census_default_chunglu300k", "kind": "census", "graph": "chunglu", "n": 300_007, "degree": 8,
         "recip": 0.1, "form": "default", "wait": True},
        # arcs to counts of a small graph: the build's launches and waits
        {"name": "build_chunglu5k", "kind": "build", "graph": "chunglu", "n": 5_003, "degree": 8, "recip": 0.1,
         "arcs": "device"},
        # arcs to counts from page-locked host arrays, as an ingesting service holds them
        {"name": "build_rmat20_host", "kind": "build", "graph": "rmat", "scale": 20, "degree": 16, "recip": 0.2,
         "arcs": "pinned"},
        # arcs to counts of the largest workload
        {"name": "build_rmat26", "kind": "build", "graph": "rmat", "scale": 26, "degree": 16, "recip": 0.2,
         "arcs": "device"},
        # many small graphs in one launch (ego networks, households), replayed
        {"name": "batch_1024", "kind": "batch", "graphs": 1024, "lo": 32, "hi": 65_536, "degree": 8, "recip": 0.1},
        # a server that answers a burst of requests, small graphs asked for most
        {"name": "serve_256", "kind": "serve", "graphs": 16, "lo": 1_000, "hi": 1_000_000, "degree": 8, "recip": 0.1,
         "requests": 256},
        # a monitoring session of 21 censuses over a sliding window
        {"name": "interval_rmat18", "kind": "interval", "scale": 18, "degree": 16, "recip": 0.2, "window": 200,
         "every": 40},
        # labelled triad states
        {"name": "census64_rmat20", "kind": "census64", "graph": "rmat", "scale": 20, "degree": 16, "recip": 0.2},
        # the dense form, an odd size near its largest
        {"name": "matrix_chunglu16k", "kind": "matrix", "graph": "chunglu", "n": 16_001, "degree": 16, "recip": 0.2},
    ]


def draw(rng: random.Random):
    def log(lo, hi):
        return math.exp(rng.uniform(math.log(lo), math.log(hi)))

    def graph(lo, hi):
        """A graph of about lo..hi vertices."""
        g = {"degree": rng.choice([4, 8, 12, 16]), "recip": rng.choice([0.0, 0.1, 0.15, 0.2, 0.35])}
        if rng.random() < 0.5:
            return dict(g, graph="rmat", scale=min(24, int(math.log2(log(lo, hi)))))
        return dict(g, graph="chunglu", n=int(min(1e7, log(lo, hi))) | 1)

    kind = rng.choice(["census", "census", "census", "build", "build", "batch", "serve", "interval", "census64",
                       "matrix"])
    if kind == "census":
        form = rng.choice(["triangle", "triangle", "triangle", "suffix", "default"])
        hi = 2 ** 24.9 if form == "triangle" else 2 ** 18.9     # the walks per pair cost far more per arc
        return dict(graph(1e3, hi), kind=kind, form=form, wait=rng.random() < 0.5)
    if kind == "build":
        return dict(graph(1e3, 2 ** 24.9), kind=kind, arcs=rng.choice(["device", "pinned"]))
    if kind == "batch":
        return {"kind": kind, "graphs": int(log(16, 1024)), "lo": 32, "hi": int(log(1024, 65_536)),
                "degree": rng.choice([4, 8, 12]), "recip": rng.choice([0.0, 0.1, 0.2])}
    if kind == "serve":
        return {"kind": kind, "graphs": rng.randint(4, 16), "lo": 1_000, "hi": int(log(1e4, 1e6)),
                "degree": rng.choice([4, 8]), "recip": 0.1, "requests": int(log(32, 512))}
    if kind == "interval":
        return {"kind": kind, "scale": rng.randint(12, 19), "degree": rng.choice([8, 16]), "recip": 0.2,
                "window": rng.choice([50, 200, 400]), "every": rng.choice([40, 80])}
    if kind == "census64":
        return dict(graph(1e3, 2 ** 20.9), kind=kind)
    return {"kind": kind, "graph": "chunglu", "n": int(log(500, 16_384)), "degree": rng.choice([8, 16]),
            "recip": rng.choice([0.1, 0.2])}


# ---------------------------------------------------------------- inputs
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _vertices(case):
    return 1 << case["scale"] if case.get("graph", "rmat") == "rmat" else case["n"]


def _reversed_share(src, dst, m, recip, gen):
    """Fill [m, len) of src and dst with the reverses of randomly chosen arcs of [0, m)."""
    for i in range(m, len(src), CHUNK):
        j = min(i + CHUNK, len(src))
        pick = torch.randint(m, (j - i,), generator=gen, device="cuda")
        src[i:j], dst[i:j] = dst[pick], src[pick]


def _rmat(scale, degree, recip, gen):
    m = degree << scale
    total = m + int(recip * m)
    src = torch.empty(total, dtype=torch.int32, device="cuda")
    dst = torch.empty(total, dtype=torch.int32, device="cuda")
    perm = torch.randperm(1 << scale, generator=gen, device="cuda").to(torch.int32)
    # four levels of the descent at a time: one of 4^4 quadrant strings per draw
    quad = torch.tensor([0.57, 0.19, 0.19, 0.05], dtype=torch.float64)
    tables = {}
    for levels in {min(4, scale - k) for k in range(0, scale, 4)}:
        p, s, d = torch.ones(1, dtype=torch.float64), torch.zeros(1, dtype=torch.int32), torch.zeros(1, dtype=torch.int32)
        for _ in range(levels):
            p = (p[:, None] * quad).reshape(-1)
            s = (2 * s[:, None] + torch.tensor([0, 0, 1, 1], dtype=torch.int32)).reshape(-1)
            d = (2 * d[:, None] + torch.tensor([0, 1, 0, 1], dtype=torch.int32)).reshape(-1)
        tables[levels] = (p.cumsum(0)[:-1].to(torch.float32).cuda(), s.cuda(), d.cuda())
    for i in range(0, m, CHUNK):
        c = min(CHUNK, m - i)
        a = torch.zeros(c, dtype=torch.int32, device="cuda")
        b = torch.zeros(c, dtype=torch.int32, device="cuda")
        for k in range(0, scale, 4):
            levels = min(4, scale - k)
            cdf, s, d = tables[levels]
            q = torch.searchsorted(cdf, torch.rand(c, generator=gen, device="cuda"), right=True, out_int32=True)
            a = (a << levels) | s[q]
            b = (b << levels) | d[q]
        src[i:i + c], dst[i:i + c] = perm[a], perm[b]
    _reversed_share(src, dst, m, recip, gen)
    return 1 << scale, src, dst


def _chung_lu(n, degree, recip, gen):
    m = degree * n
    total = m + int(recip * m)
    w = torch.arange(1, n + 1, dtype=torch.float64, device="cuda") ** (-1.0 / 1.1)
    w = (w * (m / w.sum())).clamp_(max=n - 1)
    order_out = torch.randperm(n, generator=gen, device="cuda").to(torch.int32)
    order_in = torch.randperm(n, generator=gen, device="cuda").to(torch.int32)
    cdf = w.cumsum(0)
    cdf = cdf / cdf[-1].clone()
    src = torch.empty(total, dtype=torch.int32, device="cuda")
    dst = torch.empty(total, dtype=torch.int32, device="cuda")
    for i in range(0, m, CHUNK):
        c = min(CHUNK, m - i)
        for out, order in ((src, order_out), (dst, order_in)):
            u = torch.rand(c, generator=gen, dtype=torch.float64, device="cuda")
            out[i:i + c] = order[torch.searchsorted(cdf, u, right=True).clamp_(max=n - 1)]
    _reversed_share(src, dst, m, recip, gen)
    return n, src, dst


def _arcs(case, seed):
    gen = _generator(seed)
    if case.get("graph", "rmat") == "rmat":
        return _rmat(case["scale"], case["degree"], case["recip"], gen)
    return _chung_lu(case["n"], case["degree"], case["recip"], gen)


def _pool(case, seed):
    """Chung-Lu graphs of log-uniform sizes in [lo, hi], resident."""
    rng = random.Random(seed)
    graphs = []
    for _ in range(case["graphs"]):
        n = int(math.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"]))))
        graphs.append(tc.Graph.from_arcs(*_chung_lu(n, case["degree"], case["recip"], _generator(rng.getrandbits(48)))))
    return graphs


class _Batch:
    """A batch handle and the graphs that must outlive it."""

    def __init__(self, graphs):
        self.graphs = graphs
        self.handle = tc.tc_batch_create([g.handle for g in graphs], options=TRIANGLE)

    def __del__(self):
        tc.tc_batch_destroy(self.handle)


class _Server:
    """A running server, the graphs registered with it and the requests of one burst."""

    def __init__(self, graphs, requests, seed):
        self.server = tc.Server(census=TRIANGLE)
        self.graphs = graphs
        ids = [self.server.add(g) for g in graphs]
        # every graph draws the same volume of arcs: small ones are asked for most
        weights = [1.0 / g.stats()["arcs"] for g in graphs]
        self.requests = random.Random(seed).choices(ids, weights, k=requests)

    def __del__(self):
        self.server.close()


def prepare(case, seed):
    kind = case["kind"]
    state = {"kind": kind}
    if kind in ("census", "census64", "matrix"):
        n, src, dst = _arcs(case, seed)
        state["graph"] = tc.Graph.from_arcs(n, src, dst)
        if kind == "census":
            state["options"] = {"triangle": TRIANGLE, "suffix": {"algo": tc.TC_ALGO_SUFFIX}, "default": None}[case["form"]]
            state["out"] = None if case["wait"] else torch.zeros(16, dtype=torch.int64, device="cuda")
    elif kind == "build":
        n, src, dst = _arcs(case, seed)
        if case["arcs"] == "pinned":
            src, dst = src.cpu().pin_memory(), dst.cpu().pin_memory()
            src, dst = src.numpy().view(np.uint32), dst.numpy().view(np.uint32)
        state["n"], state["src"], state["dst"] = n, src, dst
    elif kind == "batch":
        state["batch"] = _Batch(_pool(case, seed))
        state["out"] = torch.zeros(16 * case["graphs"], dtype=torch.int64, device="cuda")
    elif kind == "serve":
        state["server"] = _Server(_pool(case, seed), case["requests"], seed)
    else:
        n, src, dst = _arcs(case, seed)
        gen = _generator(seed + 1)
        order = torch.randperm(len(src), generator=gen, device="cuda")
        times = torch.randint(1000, (len(src),), generator=gen, device="cuda").sort().values
        state["n"], state["window"] = n, case["window"]
        src, dst = src[order].cpu().numpy().view(np.uint32), dst[order].cpu().numpy().view(np.uint32)
        times = times.cpu().numpy().astype(np.uint64)
        stops = list(range(200, 1001, case["every"]))
        cuts = [0] + list(np.searchsorted(times, stops, side="right"))
        state["steps"] = [(t, src[a:b], dst[a:b], times[a:b]) for t, a, b in zip(stops, cuts, cuts[1:])]
    return state


# ---------------------------------------------------------------- passes
def _limbs(counts):
    """Counts of up to 124 bits as an array of (low 62 bits, the rest)."""
    return np.array([[c & LIMB, c >> 62] for c in counts], dtype=np.int64)


def run(state):
    kind = state["kind"]
    if kind == "census":
        if state["out"] is None:
            return _limbs(state["graph"].census(options=state["options"]))
        tc.tc_census_async(state["graph"].handle, state["out"], options=state["options"])
        return state["out"]
    if kind == "build":
        with tc.Graph.from_arcs(state["n"], state["src"], state["dst"]) as g:
            return {"counts": _limbs(g.census(options=TRIANGLE)), "stats": g.stats()}
    if kind == "batch":
        tc.tc_batch_census_async(state["batch"].handle, state["out"])
        return state["out"]
    if kind == "serve":
        server = state["server"].server
        ids = [server.submit(g) for g in state["server"].requests]
        got = {}
        while len(got) < len(ids):
            got.update((r.id, r.census()) for r in server.poll(timeout_ms=1000))
        return np.stack([_limbs(got[i]) for i in ids])
    if kind == "interval":
        with tc.Stream(state["n"], state["window"], options=TRIANGLE) as stream:
            counts = []
            for t, src, dst, times in state["steps"]:
                stream.push(src, dst, times)
                counts.append(_limbs(stream.census(t)[0]))
            return np.stack(counts)
    if kind == "census64":
        return _limbs(state["graph"].census64())
    return _limbs(state["graph"].census_matrix())


def work(case):
    """The arcs or the compact structure read once and the counts written: 8 bytes per arc drawn
    (two ids, or the two list entries of a connected pair) and 8 per vertex offset; the dense form
    is six products of n x n matrices."""
    kind = case["kind"]
    if kind in ("batch", "serve"):
        mean = (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"])     # of the log-uniform sizes
        if kind == "serve":      # requests in inverse proportion to the arcs: the harmonic mean size
            mean = math.log(case["hi"] / case["lo"]) / (1.0 / case["lo"] - 1.0 / case["hi"])
        count = case["graphs"] if kind == "batch" else case["requests"]
        return {"bytes": count * (8 * mean * (1 + case["degree"]) + 256), "flops": 0}
    n = _vertices(case)
    arcs = 8 * case["degree"] * n * (1 + case["recip"])
    if kind == "build":
        return {"bytes": arcs + 256, "flops": 0}
    if kind == "interval":       # every arc pushed once, and each window's arcs read once
        windows = len(range(200, 1001, case["every"]))
        return {"bytes": arcs * (1 + windows * min(case["window"], 1000) / 1000) + 256 * windows, "flops": 0}
    flops = 6 * 2.0 * n ** 3 if kind == "matrix" else 0
    return {"bytes": arcs + 8 * n + (1024 if kind == "census64" else 256), "flops": flops}


def exact(case, seed):
    """The 16 counts of a small graph from dense 64-bit matrix products (every entry a whole number
    below 2^53): the class counts as masked sums of products of the one-way, mutual and null dyads."""
    if case["kind"] not in ("census", "matrix") or _vertices(case) > 4096 or not case.get("wait", True):
        return None
    n, src, dst = _arcs(case, seed)
    a = torch.zeros((n, n), dtype=torch.float64, device="cuda")
    a[src.long(), dst.long()] = 1.0
    a.fill_diagonal_(0.0)
    mut, one = a * a.t(), a * (1.0 - a.t())
    null = 1.0 - torch.maximum(a, a.t())
    null.fill_diagonal_(0.0)
    nn, ss, sts, sst, mm, nm = null @ null, one @ one, one.t() @ one, one @ one.t(), mut @ mut, null @ mut

    def total(mask, prod, by=1):
        return int((mask * prod).sum(dtype=torch.float64).item()) // by

    counts = [total(null, nn, 6), total(one, nn), total(mut, nn, 2), total(null, sts, 2), total(null, sst, 2),
              total(null, ss), total(one, nm), total(one.t(), nm), total(one, ss), total(one.t(), ss, 3),
              total(null, mm, 2), total(mut, sts, 2), total(mut, sst, 2), total(mut, ss), total(one, mm),
              total(mut, mm, 6)]
    return _limbs(counts)
