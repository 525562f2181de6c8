"""CLUSTER2's edge-balanced rounds at the edges of a warp's 128-position chunk: hubs of 127 .. 129 and more
entries, rows that start and end inside a chunk, against the literal oracle."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("leaves", [1, 31, 32, 126, 127, 128, 129, 255, 2000])
@pytest.mark.parametrize("tail", [0, 3, 130])
@pytest.mark.parametrize("wmax", [1, 40])
def test_star_with_a_tail(leaves, tail, wmax):
    import paper_1506_03265_gb300 as cd
    rng = np.random.default_rng(1000 * leaves + tail)
    src = np.concatenate([np.zeros(leaves, int), np.arange(leaves, leaves + tail)])  # a star, a path from a leaf
    dst = src * 0 + np.arange(1, leaves + tail + 1)
    n = leaves + tail + 1
    extra = rng.integers(0, n, (2, leaves // 2))
    src, dst = np.concatenate([src, extra[0]]).astype(np.uint32), np.concatenate([dst, extra[1]]).astype(np.uint32)
    w = rng.integers(1, wmax + 1, src.size).astype(np.uint32)
    g = cd.build_csr(src, dst, w, n)
    og = oracle.build_csr(n, src, dst, w, lcc=True)
    for tau, seed in ((0.05, 1), (0.4, 2)):
        c = cd.cluster2(g, tau, seed)
        oc = oracle.cluster2(og, tau, seed, oracle.delta0(og))
        center, D, _ = c.copy()
        assert np.array_equal(center, oc.center) and np.array_equal(D.astype(np.uint64), oc.D)
