"""The end of a many-graph job: ranks, the dense quotient and its diameter, against the one-graph path, over quotient
shapes on both sides of each rule (dense and sparse around the shared Floyd-Warshall limit, up to the dense capacity,
sums that might overflow)."""
import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu


def _edges(kind, n, wmax, rng):
    if kind == "path":
        src, dst = np.arange(n - 1), np.arange(1, n)
    elif kind == "dense":
        src, dst = np.triu_indices(n, 1)
    else:
        dst = np.arange(1, n)
        src = (rng.random(n - 1) * dst).astype(int)
        extra = rng.integers(0, n, (2, n))
        src, dst = np.concatenate([src, extra[0]]), np.concatenate([dst, extra[1]])
    return src.astype(np.uint32), dst.astype(np.uint32), rng.integers(1, wmax + 1, src.size).astype(np.uint32)


def _one(cd, g, tau, seed):
    try:
        return cd.estimate(cd.quotient_build(cd.cluster(g, tau, seed))), 0
    except cd.CldiamError as e:
        return None, e.status


@pytest.mark.parametrize("wmax", [1000, 1 << 22, 1 << 30])
def test_all_singletons(wmax):
    """tau so large that every node is a cluster: the quotient is the graph."""
    import paper_1506_03265_gb300 as cd
    rng = np.random.default_rng(wmax % 1013)
    a, sizes = cd.arena_create(), []
    for kind in ("path", "sparse", "dense"):
        for n in (2, 31, 33, 199, 200, 201, 500, 1023, 1024, 1025, 4100):
            if kind == "dense" and n > 600:
                continue
            a.add(*_edges(kind, n, wmax, rng), n)
            sizes.append(n)
    ids = np.arange(len(sizes))
    res, sts = a.run(ids, [1e9] * len(ids), [1] * len(ids), raise_on_error=False)
    for i, n in enumerate(sizes):
        want, st = _one(cd, a.graph(i), 1e9, 1)
        if sts[i] == -3 and st == 0:
            # up to 200 nodes the many-graph form's Floyd-Warshall also adds two long paths, and refuses
            assert n <= 200 and wmax == 1 << 30, (i, n)
            continue
        assert sts[i] == st, (i, n)
        if st == 0:
            assert res[i] == want, (i, n)


def test_mixture_equals_one_graph_path():
    import paper_1506_03265_gb300 as cd
    a = cd.arena_create()
    for i in range(40):
        e = inputs.mix_graph(17, i)
        a.add(e.src, e.dst, e.w, e.n, lcc=i % 3 != 0)  # every third graph may be unconnected
    for mode in (0, 1):
        cd.tuning_set(batch_split=1)
        try:
            res, _ = a.run(np.arange(40), [0.4] * 40, np.arange(40), contract_mode=mode)
        finally:
            cd.tuning_set()
        for i in range(40):
            c = cd.cluster(a.graph(i), 0.4, i, contract_mode=mode)
            assert res[i] == cd.estimate(cd.quotient_build(c)), i


@pytest.mark.parametrize("mode,cap", [(0, 0), (1, 2)])
def test_groups_beside_small_jobs(mode, cap):
    """Few large jobs among many small ones: the large ones run on groups of CTAs."""
    import paper_1506_03265_gb300 as cd
    a, taus = cd.arena_create(), []
    big = [(inputs.grid(140, 1000, 1), True, 0.5), (inputs.grid(333, 1000, 2), True, 0.7),
           (inputs.rmat(15, 8, 1000, 3), False, 0.5), (inputs.road_mesh(400, 1000, 4), False, 0.8),
           (inputs.rmat(16, 8, 1000, 5), True, 30.0),  # k above the dense capacity: finished on the one-graph path
           (inputs.grid(250, 1 << 24, 6), True, 0.6)]  # path sums that may overflow
    for e, lcc, tau in big:
        a.add(e.src, e.dst, e.w, e.n, lcc=lcc)
        taus.append(tau)
    for i in range(30):
        e = inputs.grid(8 + i, 100, i)
        a.add(e.src, e.dst, e.w, e.n)
        taus.append(0.1)
    ids = np.arange(len(taus))
    res, sts = a.run(ids, taus, ids, raise_on_error=False, contract_mode=mode, step_cap=cap)
    start, end = a.job_times(len(ids))
    assert np.all(end >= start)
    for i in ids:
        try:
            c = cd.cluster(a.graph(int(i)), taus[i], int(i), contract_mode=mode, step_cap=cap)
            want, st = cd.estimate(cd.quotient_build(c)), 0
        except cd.CldiamError as e:
            want, st = None, e.status
        assert sts[i] == st, i
        if st == 0:
            assert res[i] == want, i
    again, _ = a.run(ids, taus, ids, raise_on_error=False, contract_mode=mode, step_cap=cap)
    assert [r for r, s in zip(again, sts) if s == 0] == [r for r, s in zip(res, sts) if s == 0]
