"""paths_tensor() is a copy at every path length, also where a row fills its
stored width exactly (T + 1 = 8, 16): a tensor that aliased the library's rows
would be freed memory once the handle is gone."""
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("T", [5, 7, 15])
def test_paths_tensor_owns_its_memory(T):
    import __graft_entry__
    __graft_entry__.build()
    import paper_1504_02577_gb300 as pk
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g = synth.workload_graph("small")
    with pk.Panther(0) as P:
        P.build_graph(g.row_ptr, g.col, g.w, pk.MODE_ALIAS)
        P.sample_paths(1, 1000, T, pk.MODE_ALIAS)
        t = P.paths_tensor()
        rows = pk.panther_paths_view(P.h.paths)[0]
        P.sync()
        assert t.shape == (1000, T + 1) and t.is_contiguous() and t.data_ptr() != rows
