"""The radix sort at the edges of its two tiles (1,024 items; 7,168 keys or 5,632 64-bit pairs) and at the
item count that chooses between them, seen through the CSR it builds."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

BIG = 3 << 17


@pytest.mark.parametrize("m", [1, 2, 1023, 1024, 1025, 3 * 1024, BIG // 2 + 1, BIG - 1, BIG, BIG + 1, 7168 * 60 - 1,
                               7168 * 60, 7168 * 60 + 1, 5632 * 80, 5632 * 80 + 1])
@pytest.mark.parametrize("ids", ["random", "two", "ordered"])  # distinct digits, one digit, runs of one digit
@pytest.mark.parametrize("w_max", [1000, (1 << 31) - 1])  # one word per edge, or (key, weight) pairs
def test_item_counts(m, ids, w_max):
    import paper_1506_03265_gb300 as cd
    rng = np.random.default_rng(m)
    n = 1 << 18
    if ids == "ordered":
        src = np.sort(rng.integers(0, n, m))
        dst = (src + rng.integers(1, 4, m)) % n
    else:
        src, dst = rng.integers(0, n if ids == "random" else 2, (2, m))
    src, dst = src.astype(np.uint32), dst.astype(np.uint32)
    w = rng.integers(1, w_max, m, dtype=np.uint32, endpoint=True)
    # the pair form sorts twice the items (both directions), the word form each edge once
    g, og = cd.build_csr(src, dst, w, n, lcc=False), oracle.build_csr(n, src, dst, w, lcc=False)
    off, col, ww, _ = g.copy()
    assert np.array_equal(off, og.off) and np.array_equal(col, og.col) and np.array_equal(ww, og.wt)


@pytest.mark.parametrize("scale", [12, 16])  # 32-bit pairs: below and above the choice
def test_quotient_pairs(scale):
    import inputs
    import paper_1506_03265_gb300 as cd
    e = inputs.rmat(scale, 16, 1000, 3)
    g, og = cd.build_csr(e.src, e.dst, e.w, e.n), oracle.build_csr(e.n, e.src, e.dst, e.w)
    c = cd.cluster(g, 2.0, 5, quotient_mode=cd.QUOTIENT_SORT)
    q = cd.quotient_build(c)
    oq = oracle.quotient(og, oracle.cluster(og, 2.0, 5, oracle.delta0(og)))
    off, col, w = q.copy()
    assert np.array_equal(off, oq.off) and np.array_equal(col, oq.col) and np.array_equal(w, oq.w)
