"""Delta-stepping where few nodes hold most entries: a round of hubs is short by its node count and large by its entries,
so it leaves the resident launch for the whole device."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("deg,leaves_launch", [(1500, False), (2000, True)])  # 300 hubs: 450,000 and 600,000 entries
def test_round_of_hubs(deg, leaves_launch):
    import paper_1506_03265_gb300 as cd
    rng = np.random.default_rng(deg)
    hubs, n = 300, 300 + 20_000
    src = np.repeat(np.arange(hubs), deg).astype(np.uint32)
    dst = (hubs + np.concatenate([rng.permutation(n - hubs)[:deg] for _ in range(hubs)])).astype(np.uint32)
    w = np.ones(src.size, np.uint32)
    g, og = cd.build_csr(src, dst, w, n), oracle.build_csr(n, src, dst, w)
    cd.sssp_delta(g, 0, 1 << 20)
    cd.profile_reset()
    dist, ecc, _ = cd.sssp_delta(g, 0, 1 << 20)
    launches = cd.profile_get()["delta_stepping"]["launches"]
    assert np.array_equal(dist, oracle.dijkstra(og, 0)) and ecc == 3
    # initialisation, hub 0 and its leaves in one launch, then the other hubs: there too, or listed and pushed by two
    # launches of their own; the last leaves (a list above its node limit) by two, the largest distance
    assert launches == (7 if leaves_launch else 5)
