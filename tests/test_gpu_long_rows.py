"""Top-k over long paths (rows of 64 and 128 entries, T >= 32) at the edges of
the lanes a path takes: (T + 1 + 3) / 4 of 9, 16, 17, 24, 31 and 32 lanes, so
three, two or one path per warp and up to fourteen spare lanes. Rows equal the
oracle's (integers, no tolerance), in the small-batch and the classified form."""
import os
import time

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
THREADS = os.cpu_count() or 1


@pytest.fixture(scope="module")
def pk():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1504_02577_gb300 as pk
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return pk


@pytest.mark.parametrize("T,R", [(32, 1500), (35, 300), (36, 1501), (62, 900), (63, 60), (64, 1000), (95, 400),
                                 (100, 700), (123, 200), (124, 333), (127, 500)])
def test_long_rows_match_the_oracle(pk, T, R):
    g = synth.workload_graph("small")
    ref = oracle.sample_paths(g, 6, R, T, oracle.ALIAS, threads=THREADS)
    o = oracle.Oracle(g.n, ref)
    v = np.arange(g.n, dtype=np.int32)
    with pk.Panther(0) as P:
        P.build_graph(g.row_ptr, g.col, g.w, pk.MODE_ALIAS)
        P.sample_paths(6, R, T, pk.MODE_ALIAS)
        P.build_index()
        for k in (1, 10, 64, 128):
            rid, rcnt = o.topk_many(v, k, threads=THREADS)
            for reps in (1, 9):                       # 2,000 queries, 18,000
                ids, cnt = P.topk(torch.as_tensor(np.tile(v, reps), device="cuda:0"), k)
                P.sync()
                ids = ids.cpu().numpy().reshape(reps, g.n, k)
                cnt = cnt.cpu().numpy().astype(np.uint32).reshape(reps, g.n, k)
                assert (ids == rid).all() and (cnt == rcnt).all(), (T, R, k, reps)


def test_no_cliff_above_32_entries(pk):
    # all vertices of 100,000: twice the entries of twice as many paths a query
    # are four times the work; 15 times the time would be another algorithm
    g = synth.chung_lu(100_000, 16, 2.3, ("uniform", 1, 255), seed=3)
    q = torch.arange(g.n, dtype=torch.int32, device="cuda:0")
    t = {}
    with pk.Panther(0) as P:
        P.build_graph(g.row_ptr, g.col, g.w, pk.MODE_ALIAS)
        for T in (31, 64):
            P.sample_paths(9, 50_000, T, pk.MODE_ALIAS)
            P.build_index()
            best = 1e9
            for _ in range(4):
                torch.cuda.synchronize()
                t0 = time.perf_counter()
                P.topk(q, 10)
                torch.cuda.synchronize()
                best = min(best, time.perf_counter() - t0)
            t[T] = best
    assert t[64] < 15 * t[31], t
