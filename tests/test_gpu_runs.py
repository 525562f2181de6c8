"""De-duplication of (key, weight) pairs with long runs of equal keys (many parallel edges): each run's
minimum is reduced inside warps of 256 items, so lengths around 32, 256 and the 2,048-item tile matter."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

N = 70_000  # 2 x 17 id bits + 31 weight bits do not fit one word: the pair form


def _check(src, dst, w, lcc):
    import paper_1506_03265_gb300 as cd
    src, dst, w = (np.asarray(a, np.uint32) for a in (src, dst, w))
    g = cd.build_csr(src, dst, w, N, lcc=lcc)
    og = oracle.build_csr(N, src, dst, w, lcc=lcc)
    off, col, ww, orig = g.copy()
    assert np.array_equal(off, og.off) and np.array_equal(col, og.col)
    assert np.array_equal(ww, og.wt) and np.array_equal(orig, og.orig)


@pytest.mark.parametrize("lcc", [False, True])
@pytest.mark.parametrize("lens", [[1], [31, 1, 32, 33], [255, 256, 257], [2047, 2, 2048, 2049], [40_000],
                                  [3, 5000, 1, 1, 700, 256, 256], [1] * 3000])
def test_run_lengths(lens, lcc):
    rng = np.random.default_rng(len(lens) + sum(lens))
    src, dst = [], []
    for i, k in enumerate(lens):
        src += [i] * k
        dst += [i + 1] * k
    order = rng.permutation(len(src))
    w = rng.integers(1 << 20, (1 << 31) - 1, len(src))
    _check(np.array(src)[order], np.array(dst)[order], w, lcc)


def test_self_loops_behind_a_long_run():
    rng = np.random.default_rng(3)
    src = np.concatenate([np.full(3000, 7), np.arange(900)])
    dst = np.concatenate([np.full(3000, 9), np.arange(900)])  # 900 self-loops: dropped, they sort last
    _check(src, dst, rng.integers(1 << 20, (1 << 31) - 1, src.size), False)


@pytest.mark.parametrize("clusters", [2, 5])
def test_quotient_sort_few_heavy_pairs(clusters):
    """A dense graph in few clusters: the sort form sees runs of thousands of equal cluster pairs."""
    import paper_1506_03265_gb300 as cd
    rng = np.random.default_rng(clusters)
    n, m = 600, 60_000
    src, dst = rng.integers(0, n, m).astype(np.uint32), rng.integers(0, n, m).astype(np.uint32)
    w = rng.integers(1, 1000, m).astype(np.uint32)
    g = cd.build_csr(src, dst, w, n)
    tau = clusters / 20
    q = [cd.quotient_build(cd.cluster(g, tau, 3, quotient_mode=mode)) for mode in (cd.QUOTIENT_SORT, cd.QUOTIENT_DENSE)]
    for a, b in zip(q[0].copy(), q[1].copy()):
        assert np.array_equal(a, b)
    og = oracle.build_csr(n, src, dst, w, lcc=True)
    oq = oracle.quotient(og, oracle.cluster(og, tau, 3, oracle.delta0(og)))
    off, col, ww = q[0].copy()
    assert np.array_equal(off, oq.off) and np.array_equal(col, oq.col) and np.array_equal(ww.astype(np.uint64), oq.w)
