"""A step's changed nodes among which hubs are: the first positions of their chunks at the edges of a lane's own share
(eight chunks of 128) and of a warp's 32, by the grid kernels and the resident ones, against the oracle."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

DEGREES = (3, 127, 128, 1022, 1023, 1024, 1025, 4095, 4096, 4097, 9000)


@pytest.mark.parametrize("ctas", [0, 8])  # 8: the grid kernels alone
@pytest.mark.parametrize("mode", [0, 1])
def test_hubs_of_every_size(ctas, mode):
    import paper_1506_03265_gb300 as cd
    rng = np.random.default_rng(4)
    deg = np.repeat(DEGREES, 3)
    hubs = deg.size
    h = np.arange(hubs)
    src = np.concatenate([h, np.repeat(h, deg)]).astype(np.uint32)  # a ring of hubs with their leaves
    dst = np.concatenate([(h + 1) % hubs, hubs + np.arange(deg.sum())]).astype(np.uint32)
    w = rng.integers(1, 20, src.size).astype(np.uint32)
    n = int(hubs + deg.sum())
    g, og = cd.build_csr(src, dst, w, n), oracle.build_csr(n, src, dst, w)
    try:
        cd.tuning_set(relax_ctas_per_sm=ctas)
        for tau, seed in ((0.02, 1), (0.3, 2)):
            c, oc = cd.cluster(g, tau, seed, contract_mode=mode), oracle.cluster(og, tau, seed, oracle.delta0(og),
                                                                                 contract_mode=mode)
            center, D, _ = c.copy()
            assert np.array_equal(center, oc.center) and np.array_equal(D.astype(np.uint64), oc.D)
            assert c.info()["steps"] == int(oc.stats["steps"])
    finally:
        cd.tuning_set()
