"""The team counting kernels of the batched top-k (one warp or one CTA per
query, tables in shared memory) at the sizes where they can go wrong. Every
row must equal the oracle's (Algorithm 1, Eq. (4)): the results are integers,
so the tolerance is zero.

A batch above 16,384 queries runs the classified tiers (warp, CTA, largest
tables), a smaller one the one-launch form; both are compared.
"""
import os

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
THREADS = os.cpu_count() or 1
BIG_BATCH = 17_000


@pytest.fixture(scope="module")
def pk():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1504_02577_gb300 as pk
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return pk


def _compare(pk, g, R, T, seed, vertices, ks, tiles):
    ref = oracle.sample_paths(g, seed, R, T, oracle.ALIAS, threads=THREADS)
    o = oracle.Oracle(g.n, ref)
    v = np.asarray(vertices, dtype=np.int32)
    with pk.Panther(0) as P:
        P.build_graph(g.row_ptr, g.col, g.w, pk.MODE_ALIAS)
        P.sample_paths(seed, R, T, pk.MODE_ALIAS)
        P.build_index()
        for k in ks:
            rid, rcnt = o.topk_many(v, k, threads=THREADS)
            for reps in tiles:
                q = torch.as_tensor(np.tile(v, reps), device="cuda:0")
                ids, cnt = P.topk(q, k)
                P.sync()
                ids = ids.cpu().numpy().reshape(reps, v.size, k)
                cnt = cnt.cpu().numpy().astype(np.uint32).reshape(reps, v.size, k)
                assert (ids == rid).all() and (cnt == rcnt).all(), (T, R, k, reps)
        P.vectors(min(128, max(ks)))           # counts only, every vertex
        theta = P.theta_tensor().cpu().numpy().view(np.uint32)
        P.sync()
    assert np.array_equal(theta, o.theta_all(min(128, max(ks)), threads=THREADS))


# rows of 8 entries full and not, 16, 32 and 64; R so that the lists run from
# a few paths (single occurrences decide) to more than the 4,096-path warp bound
@pytest.mark.parametrize("T,R", [(1, 4_000), (3, 30_000), (7, 2_500), (7, 60_000), (8, 3_000), (11, 12_000),
                                 (12, 30_001), (15, 2_000), (16, 9_000), (20, 4_000), (31, 2_000), (40, 1_500)])
def test_all_vertices_both_forms(pk, T, R):
    g = synth.workload_graph("small")
    _compare(pk, g, R, T, 6, np.arange(g.n), (1, 10, 33, 64, 65, 128), (1, -(-BIG_BATCH // g.n)))


def test_small_graph_many_paths(pk):
    # 40 vertices: a table of 128 slots, up to 39 candidates, thousands of paths each
    g = synth.chung_lu(40, 8, 2.5, ("uniform", 1, 4), seed=5)
    _compare(pk, g, 50_000, 5, 3, np.arange(g.n), (1, 10, 39, 64), (1, BIG_BATCH // g.n + 1))


def test_many_large_equal_counts(pk):
    # a complete graph of 600 vertices, about 150 shared paths per pair: more
    # candidates in one coded bin of large counts than the ranking buffer holds
    n = 600
    col = np.concatenate([np.delete(np.arange(n, dtype=np.int32), v) for v in range(n)])
    g = synth.Graph(n, np.arange(n + 1, dtype=np.int64) * (n - 1), col, np.ones(col.size, np.uint32), 0, n - 1, 0)
    _compare(pk, g, 1_800_000, 5, 2, np.arange(0, n, 7), (10, 128), (1, ))


@pytest.mark.parametrize("R", [15_000, 100_000])
def test_clustered_ids(pk, R):
    # a star whose leaves are one low id and 20,000 ids far above it: hundreds
    # (warp table) or thousands (CTA table) of single occurrences in one coded
    # bin of id distances, so the search for the smallest ids goes inside the bin
    n, lo, leaves = 1_050_000, 1_000_000, 20_000
    leaf = np.concatenate([[3], np.arange(lo, lo + leaves)]).astype(np.int32)
    hub = n - 1
    deg = np.zeros(n, np.int64)
    deg[leaf] = 1
    deg[hub] = leaf.size
    row_ptr = np.concatenate([[0], np.cumsum(deg)]).astype(np.int64)
    col = np.concatenate([np.full(leaf.size, hub, np.int32), leaf])
    g = synth.Graph(n, row_ptr, col, np.ones(col.size, np.uint32), 0, leaf.size, 0)
    ref = oracle.sample_paths(g, 4, R, 1, oracle.ALIAS, threads=THREADS)
    o = oracle.Oracle(n, ref)
    with pk.Panther(0) as P:
        P.build_graph(g.row_ptr, g.col, g.w, pk.MODE_ALIAS)
        P.sample_paths(4, R, 1, pk.MODE_ALIAS)
        P.build_index()
        for k in (10, 40, 128):
            rid, rcnt = o.topk_many(np.array([hub], np.int32), k)
            for reps in (1, BIG_BATCH):
                ids, cnt = P.topk(torch.full((reps,), hub, dtype=torch.int32, device="cuda:0"), k)
                P.sync()
                assert (ids.cpu().numpy() == rid).all() and (cnt.cpu().numpy() == rcnt).all(), (R, k, reps)
