"""The largest component where the sampled dominant tree holds less than half of the nodes: counted trees, ties by the
smallest id, nodes without an edge."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _paths(sizes, n, order):
    """Paths of the given sizes over the node ids in `order`; the other nodes have no edge."""
    src, dst, at = [], [], 0
    for k in sizes:
        ids = order[at:at + k]
        src.append(ids[:-1])
        dst.append(ids[1:])
        at += k
    return np.concatenate(src), np.concatenate(dst)


@pytest.mark.parametrize("sizes,n", [([2], 5000), ([2, 2, 2], 3000), ([5, 7, 7, 6], 100), ([40] * 50 + [41], 9000),
                                     ([1200, 1199, 1200], 4000), ([300, 900], 1300), ([3] * 1000, 3000),
                                     ([1], 40)])
@pytest.mark.parametrize("seed", [0, 1])
def test_components(sizes, n, seed):
    import paper_1506_03265_gb300 as cd
    rng = np.random.default_rng(seed)
    src, dst = _paths(sizes, n, rng.permutation(n))
    src, dst = src.astype(np.uint32), dst.astype(np.uint32)
    w = rng.integers(1, 100, src.size).astype(np.uint32)
    g, og = cd.build_csr(src, dst, w, n), oracle.build_csr(n, src, dst, w, lcc=True)
    assert (g.n, g.nnz) == (og.n, og.nnz)
    for mine, ref in zip(g.copy(), (og.off, og.col, og.wt, og.orig)):
        assert np.array_equal(mine, ref)


def test_rmat_with_many_lone_nodes():
    import inputs
    import paper_1506_03265_gb300 as cd
    e = inputs.rmat(16, 1, 1000, 8)
    g, og = cd.build_csr(e.src, e.dst, e.w, e.n), oracle.build_csr(e.n, e.src, e.dst, e.w, lcc=True)
    assert g.n < e.n // 2
    for mine, ref in zip(g.copy(), (og.off, og.col, og.wt, og.orig)):
        assert np.array_equal(mine, ref)


@pytest.mark.parametrize("n", [3000, 100_000])
def test_dominant_tree_hooked_late(n):
    """The dominant tree's root is hooked under a smaller id by an edge that only the last pass takes: node 0's first two
    neighbours (in id order) are in its own small tree, the third one is in the dominant tree; lone nodes keep that tree
    below half of the nodes."""
    import paper_1506_03265_gb300 as cd
    k = n * 2 // 5
    ids = np.arange(10, 10 + k)
    src = np.concatenate([[0, 0, 0], ids[:-1]]).astype(np.uint32)
    dst = np.concatenate([[1, 2, 10 + k - 1], ids[1:]]).astype(np.uint32)
    w = np.ones(src.size, np.uint32)
    g, og = cd.build_csr(src, dst, w, n), oracle.build_csr(n, src, dst, w, lcc=True)
    assert g.n == k + 3
    for mine, ref in zip(g.copy(), (og.off, og.col, og.wt, og.orig)):
        assert np.array_equal(mine, ref)
