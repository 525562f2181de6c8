"""The default bucket width of Delta-stepping by a graph's size and degrees: what the rounds read and how many there are,
for a graph of its own and for one of an arena."""
import numpy as np
import pytest

import inputs
import oracle

pytestmark = pytest.mark.gpu


def _uniform(n, ef):
    rng = np.random.default_rng(n)
    return rng.integers(0, n, n * ef), rng.integers(0, n, n * ef), rng.integers(1, 1 << 20, n * ef), n


@pytest.mark.parametrize("form", ["graph", "arena"])
@pytest.mark.parametrize("kind", ["uniform", "rmat"])
def test_reads_and_rounds(kind, form):
    import paper_1506_03265_gb300 as cd
    if kind == "uniform":
        src, dst, w, n = _uniform(1 << 15, 12)
    else:
        e = inputs.rmat(14, 16, 1 << 20, 3)
        src, dst, w, n = e.src, e.dst, e.w, e.n
    src, dst, w = (np.asarray(x).astype(np.uint32) for x in (src, dst, w))
    arena = cd.arena_create()
    g = cd.build_csr(src, dst, w, n) if form == "graph" else arena.graph(arena.add(src, dst, w, n))
    dist, _, rounds, scanned = cd.sssp_delta(g, 5, with_scanned=True)
    avg = g.delta0()
    _, _, rounds_avg, scanned_avg = cd.sssp_delta(g, 5, avg, with_scanned=True)
    _, _, rounds_8, scanned_8 = cd.sssp_delta(g, 5, 8 * avg, with_scanned=True)
    ref = oracle.dijkstra(oracle.build_csr(n, src, dst, w), 5)
    assert np.array_equal(dist, np.where(ref == oracle.UNREACHABLE, 0xFFFFFFFF, ref))
    # the width is one average weight without hubs, where eight read several times as much, and eight with them, where
    # one takes more rounds (a bucket's end, and so both counts, may differ by a little between two runs)
    if kind == "uniform":
        assert scanned < 1.25 * scanned_avg < 0.75 * scanned_8
    else:
        assert rounds <= rounds_8 + 1 < rounds_avg
