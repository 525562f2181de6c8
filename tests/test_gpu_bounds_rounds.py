"""The quotient diameter by bounds where the sum of the heaviest entries passes 2^32: rounds bound the sums instead, and
where these pass it too every source is taken, with OVERFLOW where that reports it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("wmax", [1 << 22, 1 << 24, 1 << 26, 1 << 27, 1 << 28, 1 << 29, 1 << 31])
@pytest.mark.parametrize("n,extra", [(200, 3), (700, 4), (3000, 2), (3000, 20)])
@pytest.mark.parametrize("chain", [0, 12])  # a tail of nodes in a row: more rounds
def test_rounds_guard(wmax, n, extra, chain):
    import paper_1506_03265_gb300 as cd
    rng = np.random.default_rng(n + extra + chain)
    dst = np.arange(1, n)
    src = (rng.random(n - 1) * dst).astype(int)
    src[n - 1 - chain:] = dst[n - 1 - chain:] - 1
    more = rng.integers(0, n - chain, (2, extra * n))
    src, dst = (np.concatenate([a, b]).astype(np.uint32) for a, b in ((src, more[0]), (dst, more[1])))
    w = rng.integers(max(1, wmax // 2), wmax, src.size).astype(np.uint32)
    g = cd.build_csr(src, dst, w, n)
    q = cd.quotient_build(cd.cluster(g, 1e9, 1))  # no center is drawn: every node is a cluster
    off, col, ww = q.copy()
    assert q.info()[0] == n
    try:
        want = cd.apsp_max(n, off, col, ww)
    except cd.CldiamError as e:
        with pytest.raises(cd.CldiamError) as e2:
            cd.estimate(q)
        assert e2.value.status == e.status
    else:
        assert cd.estimate(q)["phi_gc"] == want


def test_unconnected_quotient():
    import paper_1506_03265_gb300 as cd
    rng = np.random.default_rng(4)
    n = 400  # two parts that no edge joins, each 200 nodes
    dst = np.concatenate([np.arange(1, 200), np.arange(201, 400)])
    src = np.concatenate([np.zeros(199, int), np.full(199, 200)])
    w = rng.integers(1 << 25, 1 << 26, src.size).astype(np.uint32)
    g = cd.build_csr(src.astype(np.uint32), dst.astype(np.uint32), w, n, lcc=False)
    q = cd.quotient_build(cd.cluster(g, 1e9, 1))
    off, col, ww = q.copy()
    assert cd.estimate(q)["phi_gc"] == cd.apsp_max(n, off, col, ww)
