"""Device memory that one context has freed serves the next context's calls:
contexts share the device's pool, so several of them used in turn do not each
keep the peak of their scratch."""
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def pk():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1504_02577_gb300 as pk
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return pk


def test_second_context_reuses_freed_scratch(pk):
    g = synth.workload_graph("small")
    R, T = 8_000_000, 5
    temporaries = 16 * R * (T + 1)                    # two key and two value arrays: 768 MB

    def used():
        free, total = torch.cuda.mem_get_info(0)
        return total - free

    with pk.Panther(0) as P, pk.Panther(0) as Q:
        P.build_graph(g.row_ptr, g.col, g.w, pk.MODE_ALIAS)
        P.sample_paths(1, R, T, pk.MODE_ALIAS)
        P.build_index()
        pk.panther_free_index(P.h.index)
        P.h.index = None
        P.sync()
        before = used()
        ix = pk.panther_build_index(Q.h.ctx, P.h.paths)
        Q.sync()
        after = used()
        pk.panther_free_index(ix)
    assert after - before < temporaries // 4, (after - before, temporaries)
