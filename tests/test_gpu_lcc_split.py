"""The largest component around the node count from which the joining pass runs in two parts."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,p,w_max", [((1 << 22) - 1, 0.7, 1000), (1 << 22, 0.7, 1000), ((1 << 22) + 37, 0.7, 1000),
                                       ((1 << 22) + 37, 0.48, 1000),          # no component holds half of the nodes
                                       ((1 << 22) + 37, 0.7, (1 << 32) - 1)])  # the (key, weight) form
def test_split_joining_pass(n, p, w_max):
    import torch

    import paper_1506_03265_gb300 as cd
    rng = np.random.default_rng(n % 97)
    cols = 2048
    v = np.arange(n, dtype=np.uint32)
    right, down = v[(v % cols != cols - 1) & (v + 1 < n)], v[: n - cols]
    src = np.concatenate([right, down])
    dst = np.concatenate([right + np.uint32(1), down + np.uint32(cols)])
    keep = rng.random(src.size) < p
    src, dst = src[keep], dst[keep]
    w = rng.integers(1, w_max, src.size, dtype=np.uint32, endpoint=True)
    t = [torch.from_numpy(x.view(np.int32)).cuda() for x in (src, dst, w)]
    g, og = cd.build_csr(*t, n), oracle.build_csr(n, src, dst, w, lcc=True)
    assert (g.n, g.nnz) == (og.n, og.nnz)
    for mine, ref in zip(g.copy(), (og.off, og.col, og.wt, og.orig)):
        assert np.array_equal(mine, ref)
