"""The vertex records of the sampler: up to 2^22 vertices the 8-byte ones share an
allocation with the 16-byte ones. Walks on both sides of that size equal the
oracle's, and an unweighted build (no weights to upload) allocates less often than a
prefix one."""
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


def _allocations(pk, ctx, g, mode):
    for nth in range(64):
        pk.panther_debug_fail_alloc(ctx, nth)
        try:
            h = pk.panther_build_graph(ctx, g.n, g.m, g.row_ptr, g.col, g.w, pk.MEM_HOST, mode)
        except pk.PantherError as e:
            assert e.code == pk.ENOMEM
            continue
        finally:
            pk.panther_debug_fail_alloc(ctx, -1)
        pk.panther_free_graph(h)
        return nth
    raise AssertionError("no build succeeded")


def test_unweighted_build_allocates_less_than_prefix(pk):
    g = synth.workload_graph("small")
    ctx = pk.panther_create(0)
    try:
        n = {m: _allocations(pk, ctx, g, m) for m in (pk.MODE_PREFIX, pk.MODE_UNWEIGHTED)}
        pk.panther_sync(ctx)
    finally:
        pk.panther_destroy(ctx)
    assert n[pk.MODE_UNWEIGHTED] < n[pk.MODE_PREFIX], n


@pytest.mark.parametrize("n", [(1 << 22) - 1, 1 << 22, (1 << 22) + 1])
def test_walks_around_the_shared_block(pk, n):
    g = synth.chung_lu(n, 4, 2.5, ("uniform", 1, 9), seed=1)
    R, T = 20_000, 5
    unit = synth.Graph(g.n, g.row_ptr, g.col, np.ones(g.m, np.uint32), 0, 0, 0)
    for mode, want in ((pk.MODE_ALIAS, oracle.sample_paths(g, 3, R, T, oracle.ALIAS, threads=THREADS)),
                       (pk.MODE_UNWEIGHTED, oracle.sample_paths(unit, 3, R, T, oracle.PREFIX, threads=THREADS))):
        with pk.Panther(0) as P:
            P.build_graph(g.row_ptr, g.col, g.w, mode)
            P.sample_paths(3, R, T, mode)
            got = P.paths_tensor()
            P.sync()
            assert np.array_equal(got.cpu().numpy(), want), (n, mode)
            P.build_graph(g.row_ptr, g.col, g.w, pk.MODE_BOTH)     # and freed, built again
            P.sample_paths(3, R, T, pk.MODE_ALIAS)
            P.sync()
