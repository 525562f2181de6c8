"""The CSR copied out into device or host arrays: one pass splits the (col, w) pairs."""
import ctypes

import numpy as np
import pytest

import inputs
import oracle

pytestmark = pytest.mark.gpu


def _graph(cd, kind, arena):
    e = inputs.rmat(9, 8, 1000, 5) if kind == "rmat" else inputs.grid(3, 100, 1)
    og = oracle.build_csr(e.n, e.src, e.dst, e.w, lcc=True)
    if not arena:
        return cd.build_csr(e.src, e.dst, e.w, e.n), og
    a = cd.arena_create()
    f = inputs.grid(5, 100, 2)  # an arena graph starts where the one before it ends: any 8-byte boundary
    a.add(f.src, f.dst, f.w, f.n)
    return a.graph(a.add(e.src, e.dst, e.w, e.n)), og


@pytest.mark.parametrize("kind", ["rmat", "grid"])
@pytest.mark.parametrize("arena", [False, True])
@pytest.mark.parametrize("col_on,w_on", [("cuda", "cuda"), ("cuda", "cpu"), ("cpu", "cuda"), (None, "cuda"),
                                         ("cpu", None), ("cpu", "cpu")])
def test_copy_destinations(kind, arena, col_on, w_on):
    import torch

    import paper_1506_03265_gb300 as cd
    g, og = _graph(cd, kind, arena)
    z = g.nnz
    assert z == og.nnz

    def dest(where):  # guard words on both sides, the array itself on a 4-byte boundary only
        return None if where is None else torch.full((z + 2,), -7, dtype=torch.int32, device=where)

    c, w = dest(col_on), dest(w_on)
    p = lambda t: None if t is None else ctypes.c_void_p(t.data_ptr() + 4)  # noqa: E731
    torch.cuda.synchronize()
    assert cd.load().cldiam_graph_copy(g.handle, None, p(c), p(w), None) == cd.OK
    for t, ref in ((c, og.col), (w, og.wt)):
        if t is not None:
            t = t.cpu().numpy()
            assert t[0] == -7 and t[-1] == -7
            assert np.array_equal(t[1:-1].view(np.uint32), ref)
