"""Exact k-NN (Sec. 3.3) over the ways the screen's work is cut: one query tile
over all SMs, query tiles that do not divide among them, whole tiles per CTA;
with and without the sample that bounds the k-th keys (from 128 candidate tiles
on), with rows beyond BF16-exact values among the candidates. Answers are
integers: rows equal the oracle's, and a batch's rows equal each other's."""
import os

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


# (n, R): 79 candidate tiles and no sample; 157 and a sample of 9; R = 4e5 puts
# counts above 256 into the heaviest rows
# D = 57, 120, 121 and 128: the edges of operand rows of 64, 128 and 192 columns
@pytest.mark.parametrize("n,R", [(20_001, 60_000), (40_000, 400_000)])
@pytest.mark.parametrize("D", [10, 50, 56, 57, 100, 120, 121, 128])
def test_knn_batches(pk, n, R, D):
    g = synth.chung_lu(n, 10, 2.3, ("uniform", 1, 9), seed=4)
    ref = oracle.sample_paths(g, 2, R, 5, oracle.ALIAS, threads=THREADS)
    o = oracle.Oracle(g.n, ref)
    theta = o.theta_all(D, threads=THREADS)
    rng = np.random.default_rng(1)
    heavy = np.argsort(-theta.max(axis=1).astype(np.int64))[:8].astype(np.int32)
    pick = np.unique(np.concatenate([heavy, rng.integers(0, n, 24).astype(np.int32)]))
    with pk.Panther(0) as P:
        P.build_graph(g.row_ptr, g.col, g.w, pk.MODE_ALIAS)
        P.sample_paths(2, R, 5, pk.MODE_ALIAS)
        P.build_index()
        P.vectors(D)
        for k in (1, 10, 32):
            want = [oracle.knn(theta, int(v), k) for v in pick]
            rid = np.stack([a for a, _ in want])
            rd = np.stack([b for _, b in want])
            # one padded tile, its edges, the single-launch slot bound, more
            # tiles than SMs, and (once) whole tiles per CTA: 16 per SM
            sizes = [pick.size, 127, 129, 4096, 4097, 20_011] + ([320_000] if (k, D) == (10, 50) else [])
            for q in sizes:
                v = np.resize(pick, q).astype(np.int32)
                ids, d2 = P.knn(torch.as_tensor(v, device="cuda:0"), k)
                P.sync()
                ids = ids.cpu().numpy()
                d2 = d2.cpu().numpy().view(np.uint64)
                at = np.arange(q) % pick.size
                assert np.array_equal(ids, rid[at]), (n, D, k, q)
                assert np.array_equal(d2, rd[at]), (n, D, k, q)
