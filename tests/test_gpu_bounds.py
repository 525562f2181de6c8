"""The quotient diameter by eccentricity bounds (estimate) against every source (cldiam_apsp_max on the same CSR): tau
so large that no center is drawn makes every node a cluster, so the quotient is the graph itself."""
import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu


def _graph(kind, n, wmax, rng):
    if kind == "path":
        src, dst = np.arange(n - 1), np.arange(1, n)
    elif kind == "cycle":
        src, dst = np.arange(n), (np.arange(n) + 1) % n
    elif kind == "star":
        src, dst = np.zeros(n - 1, int), np.arange(1, n)
    elif kind == "hubs":  # two hubs of n / 2 leaves, a path between them and random chords
        src = np.concatenate([np.zeros(n // 2, int), np.full(n - n // 2 - 1, 1)])
        dst = np.arange(1, n)
        dst[0] = 1
        extra = rng.integers(2, n, (2, n // 10 + 1))
        src, dst = np.concatenate([src, extra[0]]), np.concatenate([dst, extra[1]])
    elif kind == "tree":
        dst = np.arange(1, n)
        src = (rng.random(n - 1) * dst).astype(int)
    else:  # sparse random, connected by a random tree
        dst = np.arange(1, n)
        src = (rng.random(n - 1) * dst).astype(int)
        extra = rng.integers(0, n, (2, 2 * n))
        src, dst = np.concatenate([src, extra[0]]), np.concatenate([dst, extra[1]])
    w = rng.integers(1, wmax + 1, src.size)
    return src.astype(np.uint32), dst.astype(np.uint32), w.astype(np.uint32)


def _check(cd, src, dst, w, n):
    g = cd.build_csr(src, dst, w, n)
    q = cd.quotient_build(cd.cluster(g, 1e9, 1))
    off, col, ww = q.copy()
    assert q.info()[0] == g.n
    want = err = None
    try:
        want = cd.apsp_max(g.n, off, col, ww)
    except cd.CldiamError as e:
        err = e.status
    if err is None:
        assert cd.estimate(q)["phi_gc"] == want
    else:
        with pytest.raises(cd.CldiamError) as e2:
            cd.estimate(q)
        assert e2.value.status == err


@pytest.mark.parametrize("kind", ["path", "cycle", "star", "hubs", "tree", "random"])
@pytest.mark.parametrize("n", [30, 151, 153, 305, 513, 2000])
@pytest.mark.parametrize("wmax", [1, 1000])
def test_shapes(kind, n, wmax):
    import paper_1506_03265_gb300 as cd
    _check(cd, *_graph(kind, n, wmax, np.random.default_rng(n + wmax)), n)


@pytest.mark.parametrize("kind", ["path", "random", "star"])
@pytest.mark.parametrize("wmax", [1 << 24, 1 << 30])  # the bounds' guard fails: every source, OVERFLOW where it was
def test_wide_weights(kind, wmax):
    import paper_1506_03265_gb300 as cd
    _check(cd, *_graph(kind, 600, wmax, np.random.default_rng(wmax % 1009)), 600)


def test_large_k():
    import paper_1506_03265_gb300 as cd
    e = inputs.grid(120, 1000, 3)  # k = 14,400
    _check(cd, e.src, e.dst, e.w, e.n)
