"""Top-k queries with very long path lists: counts so large that one coded bin of
the ranking holds more candidates than its buffer. Results are integers and equal
the oracle's."""
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


def _complete(n):
    col = np.concatenate([np.delete(np.arange(n, dtype=np.int32), v) for v in range(n)])
    return synth.Graph(n, np.arange(n + 1, dtype=np.int64) * (n - 1), col, np.ones(col.size, np.uint32), 0, n - 1, 0)


def _check(pk, P, o, v, k):
    rid, rcnt = o.topk_many(v, k, threads=THREADS)
    ids, cnt = P.topk(torch.as_tensor(v, device="cuda:0"), k)
    P.sync()
    assert np.array_equal(ids.cpu().numpy(), rid), (v.size, k)
    assert np.array_equal(cnt.cpu().numpy().astype(np.uint32), rcnt), (v.size, k)


def test_one_coded_bin_of_counts_above_4096(pk):
    # a complete graph: most of a row's 299 counts lie in one coded bin, 6,656 to
    # 7,167, more than the ranking buffer of 256
    n, R = 300, 20_690_000
    g = _complete(n)
    ref = oracle.sample_paths(g, 2, R, 5, oracle.ALIAS, threads=THREADS)
    o = oracle.Oracle(g.n, ref)
    rows = np.sort(ref[(ref == 43).any(axis=1)], axis=1)
    c = np.bincount(np.concatenate([rows[:, 0], rows[:, 1:][rows[:, 1:] != rows[:, :-1]]]), minlength=n)
    c[43] = 0
    assert ((c >= 6656) & (c < 7168)).sum() > 256 and c.max() < 7168
    with pk.Panther(0) as P:
        P.build_graph(g.row_ptr, g.col, g.w, pk.MODE_ALIAS)
        P.sample_paths(2, R, 5, pk.MODE_ALIAS)
        P.build_index()
        for k in (1, 10, 64, 65, 128):
            _check(pk, P, o, np.arange(0, n, 43, dtype=np.int32), k)
