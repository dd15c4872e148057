"""k-NN of networks of few candidate tiles (256 vertices each): 15 and 16 tiles
(the sample that bounds the k-th keys starts at 16), 127 and 128 (its share
changes), one tile; lists that fill (many rows of a warp insert at once, each by
its own lane) and lists that are full. Answers are integers: picked rows equal
the oracle's, all rows equal those of the FP32 form, which inserts row by row."""
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


@pytest.mark.parametrize("n", [200, 3_840, 3_841, 4_096, 10_001, 32_512, 32_513])
def test_knn_small_networks(pk, n):
    D = 50
    g = synth.chung_lu(n, 10, 2.3, ("uniform", 1, 9), seed=4)
    ref = oracle.sample_paths(g, 2, 3 * n, 5, oracle.ALIAS, threads=THREADS)
    theta = oracle.Oracle(g.n, ref).theta_all(D, threads=THREADS)
    pick = np.linspace(0, n - 1, 12).astype(np.int32)
    with pk.Panther(0) as P:
        P.build_graph(g.row_ptr, g.col, g.w, pk.MODE_ALIAS)
        P.sample_paths(2, 3 * n, 5, pk.MODE_ALIAS)
        P.build_index()
        P.vectors(D)
        every = torch.arange(n, dtype=torch.int32, device="cuda:0")
        for k in (1, 2, 10, 20, 32):
            want = [oracle.knn(theta, int(v), k) for v in pick]
            rid, rd = np.stack([a for a, _ in want]), np.stack([b for _, b in want])
            # one query tile of rows that all insert the same candidates, then every vertex
            v = np.resize(pick[::-1], 100)
            ids, d2 = P.knn(torch.as_tensor(v, device="cuda:0"), k)
            P.sync()
            at = pick.size - 1 - np.arange(100) % pick.size
            assert np.array_equal(ids.cpu().numpy(), rid[at]), (n, k)
            assert np.array_equal(d2.cpu().numpy().view(np.uint64), rd[at]), (n, k)
            ids, d2 = P.knn(every, k)
            fid, fd2 = P.knn(every, k, fp32=True)
            P.sync()
            assert torch.equal(ids, fid) and torch.equal(d2, fd2), (n, k)
            assert np.array_equal(ids.cpu().numpy()[pick], rid), (n, k)


def test_no_cliff_below_the_larger_sample(pk):
    # 125 and 129 candidate tiles: nearly the same work on both sides of a rule
    t = {}
    for n in (32_000, 33_000):
        g = synth.chung_lu(n, 10, 2.3, ("uniform", 1, 9), seed=4)
        with pk.Panther(0) as P:
            P.build_graph(g.row_ptr, g.col, g.w, pk.MODE_ALIAS)
            P.sample_paths(2, 3 * n, 5, pk.MODE_ALIAS)
            P.build_index()
            P.vectors(50)
            q = torch.arange(n, dtype=torch.int32, device="cuda:0")
            best = 1e9
            for _ in range(5):
                torch.cuda.synchronize()
                t0 = time.perf_counter()
                P.knn(q, 10)
                torch.cuda.synchronize()
                best = min(best, time.perf_counter() - t0)
            t[n] = best
    assert t[32_000] < 2 * t[33_000], t
