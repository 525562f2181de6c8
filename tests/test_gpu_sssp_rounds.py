"""Delta-stepping against Dijkstra where its rounds change form: lists and piles at the edges of a warp's 128 positions,
rounds in one launch and on the whole device, bucket widths from one weight unit to all distances, unconnected graphs,
sums at the end of the 32-bit range."""
import numpy as np
import pytest

import inputs
import oracle

pytestmark = pytest.mark.gpu


def _check(src, dst, w, n, source, deltas, lcc=False):
    import paper_1506_03265_gb300 as cd
    src, dst, w = (np.asarray(a).astype(np.uint32) for a in (src, dst, w))
    g, og = cd.build_csr(src, dst, w, n, lcc=lcc), oracle.build_csr(n, src, dst, w, lcc=lcc)
    ref = oracle.dijkstra(og, source)
    ref = np.where(ref == oracle.UNREACHABLE, 0xFFFFFFFF, ref).astype(np.uint64)
    for delta in deltas:
        dist, ecc, rounds = cd.sssp_delta(g, source, delta)
        assert np.array_equal(dist.astype(np.uint64), ref), delta
        assert ecc == ref[ref != 0xFFFFFFFF].max()


@pytest.mark.parametrize("leaves", [1, 31, 33, 127, 128, 129, 1025, 5000])
@pytest.mark.parametrize("from_hub", [True, False])
def test_star_and_paths(leaves, from_hub):
    rng = np.random.default_rng(leaves)
    src = np.concatenate([np.zeros(leaves, int), np.arange(1, leaves), rng.integers(0, leaves, leaves)])
    dst = np.concatenate([np.arange(1, leaves + 1), np.arange(2, leaves + 1), rng.integers(0, leaves, leaves)])
    _check(src, dst, rng.integers(1, 500, src.size), leaves + 3, 0 if from_hub else leaves, (0, 1, 60, 1 << 31))


@pytest.mark.parametrize("scale,ef", [(12, 16), (17, 16)])  # the larger one's middle rounds leave the launch
def test_power_law(scale, ef):
    e = inputs.rmat(scale, ef, 1000, 3)
    _check(e.src, e.dst, e.w, e.n, 5, (0, 17, 150, 4000), lcc=True)


@pytest.mark.parametrize("side", [3, 90, 600])
def test_meshes(side):
    e = inputs.grid(side, 1000, 3)
    _check(e.src, e.dst, e.w, e.n, side, (0, 700, 1 << 20))


def test_unconnected_and_single():
    _check([0, 3], [1, 4], [5, 7], 6, 0, (0, 1, 9))
    _check([], [], [], 1, 0, (0, 3))


def test_end_of_the_range():
    import paper_1506_03265_gb300 as cd
    top = 0xFFFFFFFE  # largest distance that fits
    src, dst = np.array([0, 1, 2], np.uint32), np.array([1, 2, 3], np.uint32)
    for last in (top - (1 << 31) - 5, top - (1 << 31) - 4):
        g = cd.build_csr(src, dst, np.array([1 << 31, 5, last], np.uint32), 4)
        for delta in (0, 3, 1 << 31):
            # every edge is relaxed from both ends: the last one backwards, at the full distance, does not fit
            with pytest.raises(cd.CldiamError) as e:
                cd.sssp_delta(g, 0, delta)
            assert e.value.status == -3, last
    g = cd.build_csr(src, dst, np.array([1 << 30, 5, 1 << 30], np.uint32), 4)
    for delta in (0, 3, 1 << 31):
        assert cd.sssp_delta(g, 0, delta)[1] == (1 << 31) + 5
