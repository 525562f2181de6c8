"""sssp_delta_scale: 0 is the rule over the graph, any other value that multiple of the average weight, 1 among them."""
import numpy as np
import pytest

import paper_1506_03265_gb300 as cd


@pytest.fixture(autouse=True)
def clean():
    cd.load()
    cd.tuning_set()
    cd.tuning_cache_clear()
    yield
    cd.tuning_set()
    cd.tuning_cache_clear()


def _search(times, **start):
    seen = []

    def measure(k):
        seen.append(k["sssp_delta_scale"])
        return times[k["sssp_delta_scale"]], 1

    return cd.autotune_search(measure, ["sssp_delta_scale"], start=start)[0], seen


def test_search_measures_the_rule_and_every_multiple():
    best, seen = _search({0: 1.0, 1: 0.5, 2: 0.9, 4: 0.9, 8: 0.9})
    assert seen == [0, 1, 2, 4, 8] and best["sssp_delta_scale"] == 1
    assert _search({0: 0.5, 1: 0.9, 2: 0.9, 4: 0.4, 8: 0.9})[0]["sssp_delta_scale"] == 4
    assert _search({0: 0.5, 1: 0.9, 2: 0.9, 4: 0.9, 8: 0.9})[0]["sssp_delta_scale"] == 1  # the rule, filled in
    assert _search({1: 0.5, 2: 0.9, 4: 0.9, 8: 0.9}, sssp_delta_scale=2)[1] == [2, 1, 4, 8]


@pytest.mark.gpu
def test_widths_in_effect():
    # a tree: every distance is set once, so the number of rounds is that of the width
    n, rng = 50_000, np.random.default_rng(1)
    v = np.arange(1, n, dtype=np.uint32)
    g = cd.build_csr((v - 1) // 2, v, rng.integers(1, 1000, n - 1).astype(np.uint32), n)
    avg = g.delta0()
    want = {m: cd.sssp_delta(g, 0, m * avg)[2] for m in (1, 2, 4, 8, 16)}
    assert len(set(want.values())) == 5
    assert cd.sssp_delta(g, 0)[2] == want[16]  # the rule for sparse graphs
    for m in (1, 2, 4, 8):
        cd.tuning_set(sssp_delta_scale=m)
        assert cd.sssp_delta(g, 0)[2] == want[m], m
        cd.tuning_set()
        cd.tuning_cache_put(0, cd.size_class(g.nnz), sssp_delta_scale=m)
        assert cd.sssp_delta(g, 0)[2] == want[m], m
        cd.tuning_cache_clear()
    best = cd.autotune_sssp(g, 0, reps=2)
    cached = cd.tuning_cache_get(0, cd.size_class(g.nnz))["sssp_delta_scale"]
    assert best["sssp_delta_scale"] == (cached or 1.0) and cd.sssp_delta(g, 0)[2] == want[int(cached) or 16]


@pytest.mark.gpu
def test_tuning_again_replaces_an_earlier_choice():
    # a tree of small weights: the rule's wide buckets beat every candidate of up to eight average weights
    n = 1 << 17
    v = np.arange(1, n, dtype=np.uint32)
    g = cd.build_csr((v - 1) // 2, v, np.random.default_rng(2).integers(1, 1 << 20, n - 1).astype(np.uint32), n)
    cls = cd.size_class(g.nnz)
    cd.tuning_cache_put(0, cls, sssp_delta_scale=2, apsp_fw_density=16)
    rounds = cd.sssp_delta(g, 0)[2]
    assert cd.autotune_sssp(g, 0)["sssp_delta_scale"] == 1.0
    cached = cd.tuning_cache_get(0, cls)
    assert cached["sssp_delta_scale"] == 0 and cached["apsp_fw_density"] == 16
    assert cd.sssp_delta(g, 0)[2] < rounds
