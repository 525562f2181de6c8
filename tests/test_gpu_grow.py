"""Growing steps run back to back by one thread-block cluster, against the same clustering on the grid kernels (a set
number of CTAs turns the resident form off) at the edges of its rules: node counts around 2^17, steps below and above
2^18 entries, several launches in a row."""
import numpy as np
import pytest

import inputs
import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cd():
    import paper_1506_03265_gb300 as m
    m.load()
    yield m
    m.tuning_set()


def _same(cd, e, tau, seeds, **opts):
    g = cd.build_csr(e.src, e.dst, e.w, e.n)
    for seed in seeds:
        cd.tuning_set()
        a = cd.cluster(g, tau, seed, **opts)
        cd.tuning_set(relax_ctas_per_sm=8)
        b = cd.cluster(g, tau, seed, **opts)
        cd.tuning_set()
        assert a.info() == b.info()
        for x, y in zip(a.copy(), b.copy()):
            assert np.array_equal(x, y)


@pytest.mark.parametrize("side", [362, 363, 500])  # 131,044 and 131,769 nodes: stages in and out of the launch
@pytest.mark.parametrize("mode", [0, 1])
def test_mesh_sizes(cd, side, mode):
    _same(cd, inputs.grid(side, 1000, 7), 0.6, (1, 2), contract_mode=mode, delta0_mode=mode)


@pytest.mark.parametrize("scale,ef", [(12, 16), (15, 16), (17, 16)])  # the largest steps leave the launch
@pytest.mark.parametrize("cap", [0, 2])
def test_power_law(cd, scale, ef, cap):
    _same(cd, inputs.rmat(scale, ef, 1000, 3), 0.9, (1, 2), step_cap=cap)


def test_road(cd):
    _same(cd, inputs.road_mesh(700, 1000, 3), 1.0, (1, 2, 3))


@pytest.mark.parametrize("n", [2, 3, 33, 1025])
def test_small_against_the_oracle(cd, n):
    rng = np.random.default_rng(n)
    src = np.concatenate([np.arange(n - 1), rng.integers(0, n, n // 2)]).astype(np.uint32)
    dst = np.concatenate([np.arange(1, n), rng.integers(0, n, n // 2)]).astype(np.uint32)
    w = rng.integers(1, 30, src.size).astype(np.uint32)
    g, og = cd.build_csr(src, dst, w, n), oracle.build_csr(n, src, dst, w, lcc=True)
    for tau in (0.01, 0.2):
        c, oc = cd.cluster(g, tau, 5), oracle.cluster(og, tau, 5, oracle.delta0(og))
        center, D, _ = c.copy()
        assert np.array_equal(center, oc.center) and np.array_equal(D.astype(np.uint64), oc.D)


def test_repeated_runs_are_equal(cd):
    e = inputs.grid(200, 1000, 4)
    g = cd.build_csr(e.src, e.dst, e.w, e.n)
    first = cd.cluster(g, 0.5, 1).copy()
    for _ in range(50):
        for x, y in zip(cd.cluster(g, 0.5, 1).copy(), first):
            assert np.array_equal(x, y)
