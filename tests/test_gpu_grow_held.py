"""Resident growing steps whose frontier the warps hold between steps: a warp's 128 nodes and 512 positions, hubs that
send the step back to the lists, frontiers that outgrow the cluster's and one CTA's share."""
import numpy as np
import pytest

import inputs
import oracle

pytestmark = pytest.mark.gpu


def _caterpillar(n, deg):
    """A path every node of which has deg - 2 leaves."""
    spine = n // (deg - 1)
    src = [np.arange(spine - 1)] + [np.arange(spine)] * (deg - 2)
    dst = [np.arange(1, spine)] + [spine + i * spine + np.arange(spine) for i in range(deg - 2)]
    return np.concatenate(src), np.concatenate(dst), spine * (deg - 1)


def _star_ring(hubs, leaves):
    """A ring of hubs, each with its leaves."""
    h = np.arange(hubs)
    src = np.concatenate([h, np.repeat(h, leaves)])
    dst = np.concatenate([(h + 1) % hubs, hubs + np.arange(hubs * leaves)])
    return src, dst, hubs * (leaves + 1)


def _graph(kind, rng):
    if kind.startswith("caterpillar"):
        src, dst, n = _caterpillar(30_000, int(kind[11:]))
    elif kind.startswith("stars"):
        src, dst, n = _star_ring(40, int(kind[5:]))
    else:
        e = inputs.grid(300, 1000, 11) if kind == "mesh" else inputs.rmat(13, 8, 1000, 5)
        return e.src, e.dst, e.w, e.n
    return src.astype(np.uint32), dst.astype(np.uint32), rng.integers(1, 50, src.size).astype(np.uint32), n


@pytest.mark.parametrize("kind", ["caterpillar3", "caterpillar5", "caterpillar17", "stars31", "stars127", "stars511",
                                  "stars513", "stars2000", "mesh", "rmat"])
@pytest.mark.parametrize("mode", [0, 1])
def test_one_graph_and_batch_against_the_oracle(kind, mode):
    import paper_1506_03265_gb300 as cd
    src, dst, w, n = _graph(kind, np.random.default_rng(7))
    g, og = cd.build_csr(src, dst, w, n), oracle.build_csr(n, src, dst, w, lcc=True)
    arena = cd.arena_create()
    gid = arena.add(src, dst, w, n)
    # (delta0 = 1 reaches steps whose changed nodes all end at Delta: an empty frontier before the next doubling)
    for tau, seed, delta0 in ((0.05, 3, None), (0.5, 4, None), (0.3, 5, 1)):
        opts = {} if delta0 is None else dict(delta0_mode=cd.DELTA0_EXPLICIT, delta0=delta0)
        c = cd.cluster(g, tau, seed, contract_mode=mode, **opts)
        oc = oracle.cluster(og, tau, seed, oracle.delta0(og) if delta0 is None else delta0, contract_mode=mode)
        center, D, _ = c.copy()
        assert np.array_equal(center, oc.center) and np.array_equal(D.astype(np.uint64), oc.D)
        info = c.info()
        for f in ("stages", "steps", "doublings", "delta_end", "guard_exits", "node_updates", "centers_drawn"):
            assert info[f] == int(oc.stats[f]), f
        if delta0 is None:
            r = arena.run([gid], [tau], [seed], contract_mode=mode)[0][0]
            for f in ("stages", "steps", "doublings", "delta_end", "node_updates", "centers_drawn"):
                assert r[f] == int(oc.stats[f]), f


def test_seeds_on_a_small_mesh():
    """Many seeds: stages that end with an empty frontier (all changed nodes at Delta) among them."""
    import paper_1506_03265_gb300 as cd
    e = inputs.grid(80, 1000, 3)
    g, og = cd.build_csr(e.src, e.dst, e.w, e.n), oracle.build_csr(e.n, e.src, e.dst, e.w)
    for seed in range(1, 120):
        c, oc = cd.cluster(g, 0.36, seed), oracle.cluster(og, 0.36, seed, oracle.delta0(og))
        assert c.info()["steps"] == int(oc.stats["steps"]) and np.array_equal(c.copy()[0], oc.center)
