"""CLUSTER over several resident launches: the limit on a launch's phases may fall after any of them (a draw, a listing, a
step with its frontier in the warps' hands or in lists, a doubling, a contraction), and the clustering, its counters and
the steps that a cap allows stay those of one launch."""
import ctypes

import numpy as np
import pytest

import inputs
import oracle

pytestmark = pytest.mark.gpu


def _edges(kind):
    rng = np.random.default_rng(5)
    if kind == "path":
        return np.arange(1999), np.arange(1, 2000), rng.integers(1, 50, 1999), 2000
    if kind == "stars":  # hubs: frontiers that the warps cannot hold
        h = np.arange(30)
        src, dst = np.concatenate([h, np.repeat(h, 900)]), np.concatenate([(h + 1) % 30, 30 + np.arange(27_000)])
        return src, dst, rng.integers(1, 50, src.size), 27_030
    e = inputs.grid(60, 1000, 11) if kind == "mesh" else inputs.rmat(12, 8, 1000, 5)
    return e.src, e.dst, e.w, e.n


@pytest.mark.parametrize("kind", ["path", "stars", "mesh", "rmat"])
@pytest.mark.parametrize("phases", [1, 2, 3, 4, 7])
def test_every_kind_of_work_is_cut_off(kind, phases):
    import paper_1506_03265_gb300 as cd
    src, dst, w, n = _edges(kind)
    src, dst, w = (np.asarray(x).astype(np.uint32) for x in (src, dst, w))
    g, og = cd.build_csr(src, dst, w, n), oracle.build_csr(n, src, dst, w)
    fn = cd.load().cldiam_internal_cluster_phases
    fn.argtypes = [ctypes.c_void_p, ctypes.c_double, ctypes.c_uint64, ctypes.c_void_p, ctypes.c_uint32, ctypes.c_void_p]
    for mode, cap, delta0, tau in ((0, 0, 0, 0.2), (1, 0, 1, 0.05), (0, 3, 1, 0.2), (1, 2, 0, 0.2)):
        opts = dict(delta0_mode=cd.DELTA0_EXPLICIT, delta0=delta0) if delta0 else {}
        o, h = cd.make_opts(contract_mode=mode, step_cap=cap, **opts), ctypes.c_void_p()
        assert fn(g.handle, tau, 9, ctypes.byref(o), phases, ctypes.byref(h)) == 0
        c = cd.Clustering(h.value, g)
        oc = oracle.cluster(og, tau, 9, delta0 or oracle.delta0(og), contract_mode=mode, step_cap=cap)
        center, D, _ = c.copy()
        assert np.array_equal(center, oc.center) and np.array_equal(D.astype(np.uint64), oc.D)
        for f in ("stages", "steps", "doublings", "delta_end", "guard_exits", "node_updates", "centers_drawn"):
            assert c.info()[f] == int(oc.stats[f]), (f, mode, cap)
