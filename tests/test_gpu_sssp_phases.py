"""Delta-stepping over several resident launches: the limit on a launch's rounds and splits may fall on either, and what
it leaves undone is done by the next launch."""
import ctypes

import numpy as np
import pytest

import inputs
import oracle

pytestmark = pytest.mark.gpu


def test_path_longer_than_a_launch():
    """A unit-weight path from one end: 16 rounds and a split per bucket, the split at the default limit of 2^20."""
    import paper_1506_03265_gb300 as cd
    n = 1_000_000
    a = np.arange(n, dtype=np.uint32)
    g = cd.build_csr(a[:-1], a[1:], np.ones(n - 1, np.uint32), n)
    dist, ecc, _ = cd.sssp_delta(g, 0)
    assert ecc == n - 1 and np.array_equal(dist, a)


def _edges(kind):
    rng = np.random.default_rng(3)
    if kind == "path":
        n = 900
        return np.arange(n - 1), np.arange(1, n), rng.integers(1, 40, n - 1), n
    e = inputs.grid(40, 1000, 3) if kind == "mesh" else inputs.rmat(11, 8, 1000, 3)
    return e.src, e.dst, e.w, e.n


@pytest.mark.parametrize("kind", ["path", "mesh", "rmat"])
@pytest.mark.parametrize("phases", [1, 2, 3, 5, 17])
def test_every_kind_of_work_is_cut_off(kind, phases):
    import paper_1506_03265_gb300 as cd
    src, dst, w, n = _edges(kind)
    src, dst, w = (np.asarray(x).astype(np.uint32) for x in (src, dst, w))
    g = cd.build_csr(src, dst, w, n)
    ref = oracle.dijkstra(oracle.build_csr(n, src, dst, w), 7)
    ref = np.where(ref == oracle.UNREACHABLE, 0xFFFFFFFF, ref)
    fn = cd.load().cldiam_internal_sssp_phases
    fn.argtypes = [ctypes.c_void_p] + [ctypes.c_uint32] * 3 + [ctypes.c_void_p] * 2
    for delta in (1, 100, 1000):
        dist, ecc = np.zeros(g.n, np.uint32), ctypes.c_uint64()
        assert fn(g.handle, 7, delta, phases, dist.ctypes.data, ctypes.byref(ecc)) == 0
        assert np.array_equal(dist, ref) and ecc.value == ref[ref != 0xFFFFFFFF].max(), delta
