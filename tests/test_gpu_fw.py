"""Blocked Floyd-Warshall at the edges of its 64 x 64 tiles, in the fast form (connected), the checked form
(unconnected pairs) and without allocation (always checked), against a plain numpy closure."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _graph(k, density, parts, wmax, seed):
    """Weights of a symmetric graph as a k x k matrix (0 = no edge), in `parts` unconnected blocks of nodes."""
    rng = np.random.default_rng(seed)
    w = np.triu(np.where(rng.random((k, k)) < density, rng.integers(1, wmax, (k, k)), 0), 1)
    part = np.arange(k) * parts // k
    w[part[:, None] != part[None, :]] = 0
    for i in range(k - 1):  # each block connected by a path
        if part[i] == part[i + 1]:
            w[i, i + 1] = wmax
    return w + w.T


@pytest.mark.parametrize("k", [2, 3, 63, 64, 65, 127, 128, 129, 191, 257, 511])
@pytest.mark.parametrize("parts", [1, 2])
@pytest.mark.parametrize("wmax", [1000, 1 << 22])
def test_dense_closure(k, parts, wmax):
    import torch

    import paper_1506_03265_gb300 as cd
    w = _graph(k, 0.7, parts, wmax, k)
    d = np.where(w > 0, w, 1 << 40).astype(np.int64)
    np.fill_diagonal(d, 0)
    for p in range(k):
        np.minimum(d, d[:, p:p + 1] + d[p:p + 1], out=d)
    want = int(d[d < (1 << 40)].max())
    r, c = np.nonzero(w)
    off = np.concatenate([[0], np.cumsum((w > 0).sum(1))]).astype(np.int64)
    dev = [torch.from_numpy(a).cuda() for a in (off, c.astype(np.int32), w[r, c].astype(np.int32))]
    torch.cuda.synchronize()
    assert cd.apsp_max(k, *dev) == want
    if len(c):
        assert cd.apsp_max_noalloc(k, *dev) == want
