"""The screen where its claims have the least room. Rows of 57 to 128 entries
between 200 and 256 are BF16-exact, and the screened value of a pair has to be
exact as well: at D = 128 its partial sums reach 2^24. And the sample's bound
when each segment of a query tile gives four minima per column slice (13 to 64
segments, networks of 200,000 to 2 million vertices): one too low would drop
true neighbours. Answers equal the oracle's."""
import os
import struct

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


def _check(pk, P, theta, q, k):
    ids, d2 = P.knn(torch.as_tensor(q, device="cuda:0"), k)
    P.sync()
    ids, d2 = ids.cpu().numpy(), d2.cpu().numpy().view(np.uint64)
    for i, v in enumerate(q):
        rid, rd = oracle.knn(theta, int(v), k)
        assert ids[i].tolist() == rid.tolist() and d2[i].tolist() == rd.tolist(), (k, i)


def test_exact_rows_near_the_limit(pk, tmp_path):
    # paths of one step loaded from a file: three groups of 150 vertices, every
    # pair of a group on 200 to 256 paths, so all distances are small and close
    rng = np.random.default_rng(5)
    size, groups = 150, 3
    u, v = np.triu_indices(size, 1)
    rows = []
    for b in range(groups):
        c = rng.integers(200 + 20 * b, 257, u.size)   # group 2: 240 to 256
        rows.append(np.repeat(np.stack([u, v], 1) + b * size, c, axis=0))
    rows = np.concatenate(rows).astype(np.int32)
    n, R = size * groups, rows.shape[0]
    full = np.full((R, 8), -1, np.int32)
    full[:, :2] = rows
    f = tmp_path / "paths.bin"
    with open(f, "wb") as h:
        h.write(struct.pack("<8s6I3qQ", b"PNTHPATH", 1, 1, 2, 8, pk.MODE_ALIAS, 0, n, R, 0, 1))
        full.tofile(h)
    with pk.Panther(0) as P:
        P.h.paths = pk.panther_load_paths(P.h.ctx, str(f))
        f.unlink()
        P.build_index()
        for D in (57, 100, 120, 121, 127, 128):
            P.vectors(D)
            theta = P.theta_tensor().cpu().numpy().view(np.uint32)
            assert theta.max() == 256 and (theta >= 200).all()
            for k in (1, 10, 32):
                _check(pk, P, theta, np.arange(n, dtype=np.int32)[::3], k)


@pytest.mark.parametrize("n", [220_000, 300_001])
def test_four_minima_per_segment(pk, n):
    g = synth.chung_lu(n, 10, 2.2, ("uniform", 1, 9), seed=4)
    with pk.Panther(0) as P:
        P.build_graph(g.row_ptr, g.col, g.w, pk.MODE_ALIAS)
        P.sample_paths(2, 4 * n, 5, pk.MODE_ALIAS)
        P.build_index()
        for D in (50, 100):
            P.vectors(D)
            theta = P.theta_tensor().cpu().numpy().view(np.uint32)
            top = theta.max(axis=1)
            assert (top > 256).any()                  # rows beyond BF16-exact values too
            heavy = np.argsort(-top.astype(np.int64))[:6]
            q = np.concatenate([heavy, np.random.default_rng(1).integers(0, n, 18)]).astype(np.int32)
            for k in (1, 10, 32):
                _check(pk, P, theta, q, k)
