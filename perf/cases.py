"""Performance cases: the work a program has the library do, through the
public entry points (the `Panther` helper and what it calls).

Four kinds of call cover the library's use:

  build  a network arrives as a device CSR: transition tables, R random paths
         and the inverted index. Returns the path rows and the index.
  topk   top-k rows of a batch of queries against a resident index.
  knn    Panther++ nearest neighbours of a batch against resident vectors, or
         (``vectors`` set) the vectors of the whole network first.
  full   one whole pass: tables, paths, index and top-k of every vertex.

Graphs follow the synthetic recipe of the benchmark (Chung-Lu power law,
symmetric weights, ids in order of expected degree), drawn here on the device
from the seed alone.
"""
import math

import torch

import paper_1504_02577_gb300 as pk

DEV = "cuda:0"


def _case(kind, n, deg, gamma, wmax, R, T, mode, **more):
    c = {"kind": kind, "n": n, "deg": deg, "gamma": gamma, "wmax": wmax, "R": R, "T": T, "mode": mode}
    c.update(more)
    return c


def listed():
    return [
        # one interactive request: a handful of vertices looked up in a resident
        # index (the batched workload's graph and sample size); latency counts
        dict(_case("topk", 1_000_000, 20.0, 2.3, 1024, 33_123, 5, "alias", k=10, q=16, hubs=0.5), name="topk_few"),
        # the batched workload: half uniform, half high-degree queries, top-5
        dict(_case("topk", 1_000_000, 20.0, 2.3, 1024, 33_123, 5, "alias", k=5, q=16_384, hubs=0.5),
             name="topk_16k"),
        # similarity of every vertex of a network, the benchmark's shape at a tenth of its size
        dict(_case("topk", 5_000_000, 16.0, 2.1, 255, 10_000_000, 5, "alias", k=10, q=5_000_000, hubs=0.0),
             name="topk_all_5m"),
        # longer paths (rows of 16 entries), a ragged vertex count, every vertex
        dict(_case("topk", 1_000_003, 16.0, 2.1, 255, 2_000_000, 10, "alias", k=10, q=1_000_003, hubs=0.0),
             name="topk_t10"),
        # the long result lists of the k study, half of the vertices
        dict(_case("topk", 2_000_000, 16.0, 2.1, 255, 4_000_000, 5, "alias", k=100, q=999_983, hubs=0.0),
             name="topk_k100"),
        # a large weighted network is loaded, sampled and indexed
        dict(_case("build", 5_000_000, 16.0, 2.1, 255, 10_000_000, 5, "alias"), name="build_alias_5m"),
        # a small one with prefix tables and long walks: launches and waits count
        dict(_case("build", 50_021, 10.0, 2.5, 16, 120_000, 20, "prefix"), name="build_prefix_50k"),
        # an unweighted network (t_ij = 1/deg), paths of ten steps
        dict(_case("build", 1_000_000, 20.0, 2.3, 1, 3_000_000, 9, "unweighted"), name="build_unweighted_1m"),
        # one interactive Panther++ request against resident vectors
        dict(_case("knn", 1_000_000, 20.0, 2.3, 1024, 5_000_000, 5, "alias", D=50, k=10, q=48, vectors=False),
             name="knn_few"),
        # Panther++ from the index on: vectors of every vertex, then a large ragged batch
        dict(_case("knn", 1_500_000, 20.0, 2.3, 1024, 7_500_000, 5, "alias", D=50, k=10, q=20_011, vectors=True),
             name="pp_50"),
        # the widest vectors of the D study (beyond the tensor-core screen's 56 columns)
        dict(_case("knn", 300_000, 16.0, 2.3, 255, 1_500_000, 5, "alias", D=100, k=10, q=1_000, vectors=True),
             name="pp_wide"),
        # one whole benchmark step, launch shape tuned once beforehand as the benchmark does
        dict(_case("full", 20_000_000, 16.0, 2.1, 255, 40_000_000, 5, "alias", k=10), name="full_20m"),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges the listed ones stand for."""
    kind = rng.choice(["topk", "topk", "topk", "build", "build", "knn", "knn", "full"])
    mode = rng.choice(["alias", "alias", "prefix", "unweighted"])
    gamma = round(rng.uniform(2.1, 2.6), 2)
    deg = round(math.exp(rng.uniform(math.log(4), math.log(32))), 1)
    wmax = 1 if mode == "unweighted" else rng.choice([1, 16, 255, 1024, 1_000_000])
    T = rng.choice([1, 2, 3, 4, 5, 5, 5, 6, 7, 9, 10, 13, 20])
    if kind == "full":
        n = _logint(rng, 20_000, 12_000_000)
        T = min(T, 7)
        deg = min(deg, 20.0)
    elif kind == "build":
        n = _logint(rng, 20_000, 5_000_000)
        # not 7: rows of exactly 8 entries came back as the library's own memory
        # instead of a copy, and a caller that drops the handle first reads freed memory
        T = 6 if T == 7 else T
    elif kind == "topk":
        n = _logint(rng, 20_000, 5_000_000)
    else:
        n = _logint(rng, 20_000, 2_000_000)
    # paths per vertex from sparse sampling to several of each vertex; the
    # counting work grows with R * T^2, which the last term bounds
    R = max(1000, min(int(n * math.exp(rng.uniform(math.log(0.03), math.log(6.0)))), int(3.0e8 / (T * T + 5)), 24_000_000))
    c = _case(kind, n, deg, gamma, wmax, R, T, mode)
    if kind == "topk":
        c.update(k=rng.choice([1, 5, 10, 10, 20, 50, 64, 100, 128]), q=_logint(rng, 1, n),
                 hubs=rng.choice([0.0, 0.0, 0.25, 0.5]))
    elif kind == "knn":
        D = rng.choice([10, 25, 50, 50, 56, 64, 100])
        pairs = 1.2e9 if D <= 56 else 3.0e8
        c.update(D=D, k=rng.choice([1, 5, 10, 10, 20, 32]), q=_logint(rng, 1, max(2, min(n, int(pairs / n)))),
                 vectors=rng.choice([False, True]))
    elif kind == "full":
        c.update(k=rng.choice([5, 10, 10, 20]))
    return c


# ------------------------------------------------------------------ inputs ---
_MODES = {"alias": pk.MODE_ALIAS, "prefix": pk.MODE_PREFIX, "unweighted": pk.MODE_UNWEIGHTED}


def _graph(case, seed):
    """Chung-Lu power-law graph as a symmetric device CSR: endpoint ranks drawn
    with density x^(-1/(gamma-1)), self loops and repeated edges dropped,
    weights uniform in 1 .. wmax (log-uniform from 1024 up)."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed * 1_000_003 + 17)
    n, a = case["n"], 1.0 / (case["gamma"] - 1.0)
    draws = int(n * case["deg"] / 2 * 1.1)
    top = float(n + 1) ** (1.0 - a) - 1.0

    def ends():
        u = torch.rand(draws, generator=g, device=DEV, dtype=torch.float64)
        u.mul_(top).add_(1.0).pow_(1.0 / (1.0 - a)).sub_(1.0)
        return u.to(torch.int64).clamp_(0, n - 1)

    x, y = ends(), ends()
    key = torch.minimum(x, y) * n + torch.maximum(x, y)
    key = key[x != y]
    del x, y
    key = torch.unique(key)
    wmax = case["wmax"]
    u = torch.rand(key.shape[0], generator=g, device=DEV, dtype=torch.float32)
    if wmax >= 1024:
        w = torch.exp(u * math.log(wmax)).to(torch.int32).clamp_(1, wmax)
    else:
        w = (u * wmax).to(torch.int32).add_(1).clamp_(1, wmax)
    both = torch.cat([key, (key % n) * n + key // n])
    del key, u
    both, order = torch.sort(both)
    w = torch.cat([w, w])[order]
    del order
    col = (both % n).to(torch.int32)
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    row_ptr[1:] = torch.cumsum(torch.bincount(both // n, minlength=n), 0)
    del both
    torch.cuda.empty_cache()
    return row_ptr, col, (None if case["mode"] == "unweighted" else w)


def _queries(case, seed):
    """Distinct vertices for a batch of the whole network, else uniform ones
    mixed with some of the top 1% by expected degree."""
    n, q = case["n"], case["q"]
    g = torch.Generator(device=DEV)
    g.manual_seed(seed * 1_000_003 + 29)
    if q == n:
        return torch.arange(n, dtype=torch.int32, device=DEV)
    nh = int(q * case.get("hubs", 0.0))
    uni = torch.randint(0, n, (q - nh,), generator=g, device=DEV)
    hub = torch.randint(0, max(1, n // 100), (nh,), generator=g, device=DEV)
    v = torch.cat([uni, hub])
    return v[torch.randperm(q, generator=g, device=DEV)].to(torch.int32)


class _State:
    def __init__(self, case, seed):
        self.case, self.seed = case, seed
        self.P = pk.Panther(0)
        self.graph = self.queries = None

    def __del__(self):
        try:
            self.P.close()
        except Exception:
            pass


def _build(s):
    c = s.case
    s.P.build_graph(*s.graph, modes=_MODES[c["mode"]])
    s.P.sample_paths(s.seed + 1, c["R"], c["T"], _MODES[c["mode"]])
    s.P.build_index()


def prepare(case, seed):
    s = _State(case, seed)
    s.graph = _graph(case, seed)
    kind = case["kind"]
    if kind == "build":
        return s
    if kind == "full":
        s.queries = torch.arange(case["n"], dtype=torch.int32, device=DEV)
        _build(s)
        s.P.tune_topk(s.queries, case["k"])
        s.P.sync()
        return s
    s.queries = _queries(case, seed)
    _build(s)
    s.graph = None
    if kind == "knn" and not case["vectors"]:
        s.P.vectors(case["D"])
    s.P.sync()
    torch.cuda.empty_cache()
    return s


# --------------------------------------------------------------------- run ---
def run(state):
    c, P = state.case, state.P
    if c["kind"] == "topk":
        return P.topk(state.queries, c["k"])
    if c["kind"] == "knn":
        if not c["vectors"]:
            return P.knn(state.queries, c["k"])
        P.vectors(c["D"])
        ids, d2 = P.knn(state.queries, c["k"])
        return P.theta_tensor(), ids, d2
    _build(state)
    if c["kind"] == "full":
        return P.topk(state.queries, c["k"])
    # the lists at the length of every row's entries, whatever the seed's repeats
    off, pid = P.index_tensors()
    return P.paths_tensor(), off, torch.nn.functional.pad(pid, (0, c["R"] * (c["T"] + 1) - pid.shape[0]), value=-1)


def work(case):
    """Bytes and operations a pass cannot do without: inputs read once, outputs
    written once. The number of (vertex, path) pairs is taken as R * (T + 1),
    the edges as n * deg / 2."""
    n, R, L = case["n"], case["R"], case["T"] + 1
    m = n * case["deg"]
    csr = 8 * (n + 1) + (4 if case["mode"] == "unweighted" else 8) * m
    pairs = R * L
    rows = 4 * pairs
    index = 8 * (n + 1) + 4 * pairs
    kind = case["kind"]
    if kind == "build":
        return {"bytes": int(csr + rows + index), "flops": pairs}
    if kind == "full":
        return {"bytes": int(csr) + n * 8 * case["k"] + 4 * n, "flops": pairs * L}
    q, k = case["q"], case["k"]
    if kind == "topk":
        # a query reads its list and those paths; a batch reads a path at most once
        share = min(1.0, q / n)
        return {"bytes": int(12 * q + 8 * k * q + share * 4 * pairs + min(1.0, share * L) * rows),
                "flops": int(share * pairs * L)}
    D = case["D"]
    theta = 4 * n * D
    b = 4 * q + 12 * k * q + theta + (rows + index if case["vectors"] else 0)
    return {"bytes": b, "flops": 2 * q * n * D + (pairs * L if case["vectors"] else 0)}


def exact(case, seed):
    """Every output is whole numbers (ids, counts, offsets, exact squared
    distances), which stay equal bit for bit: nothing is rounded."""
    return None
