"""Vectors of more than 56 columns when the device has no room for their BF16
operand rows: the vectors are made without them, and k-NN takes the FP32 form.
The allocation fails by injection, one after the other."""
import numpy as np
import pytest

import oracle
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


@pytest.mark.parametrize("D", [57, 128])
def test_wide_vectors_without_operand_rows(pk, D):
    g = synth.workload_graph("small")
    q = np.arange(0, g.n, 13, dtype=np.int32)
    failed, made = [], []
    with pk.Panther(0) as P:
        P.build_graph(g.row_ptr, g.col, g.w, pk.MODE_ALIAS)
        P.sample_paths(1, 200_000, 5, pk.MODE_ALIAS)
        P.build_index()
        for nth in range(64):
            pk.panther_debug_fail_alloc(P.h.ctx, nth)
            try:
                P.vectors(D)
            except pk.PantherError as e:
                assert e.code == pk.ENOMEM, nth
                failed.append(nth)
                continue
            finally:
                pk.panther_debug_fail_alloc(P.h.ctx, -1)
            made.append(nth)
            theta = P.theta_tensor().cpu().numpy().view(np.uint32)
            ids, d2 = P.knn(torch.as_tensor(q, device="cuda:0"), 10)
            P.sync()
            for i, v in enumerate(q):
                rid, rd = oracle.knn(theta, int(v), 10)
                assert ids[i].tolist() == rid.tolist() and d2[i].tolist() == rd.tolist(), (nth, i)
            if nth > 0 and made[-2:] == [nth - 1, nth]:
                break                                 # beyond the last allocation
    # one allocation of several may fail without failing the call
    assert len(failed) >= 4 and made[0] < failed[-1], (failed, made)
