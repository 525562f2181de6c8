"""CLUSTER beside a live server, whose persistent kernel holds most SMs for good: one-graph calls and the server's own
large-graph lane finish long before its idle limit, and give what they give alone."""
import time

import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu


def test_one_graph_calls_beside_a_server():
    import paper_1506_03265_gb300 as cd
    e = inputs.grid(64, 100, 1)
    big = inputs.rmat(12, 8, 1000, 3)
    g = cd.build_csr(e.src, e.dst, e.w, e.n)
    alone = cd.cluster(g, 0.3, 1)
    arena = cd.arena_create()
    small_id = arena.add(e.src, e.dst, e.w, e.n)
    big_id = arena.add(big.src, big.dst, big.w, big.n)
    gb = arena.graph(big_id)
    want = cd.estimate(cd.quotient_build(cd.cluster(gb, 0.5, 2)))
    srv = cd.server_create(arena, big_nodes=100, idle_seconds=60.0)  # default CTAs: all but a few SMs
    try:
        t0 = time.time()
        beside = cd.cluster(g, 0.3, 1)
        assert beside.info() == alone.info()
        for x, y in zip(beside.copy(), alone.copy()):
            assert np.array_equal(x, y)
        ticket = srv.submit(big_id, 0.5, 2)
        while (r := srv.poll(ticket)) is None and time.time() - t0 < 30:
            time.sleep(0.001)
        assert r == want
        assert time.time() - t0 < 30 and small_id == 0
    finally:
        srv.free()
    after = cd.cluster(g, 0.3, 1)
    assert after.info() == alone.info()
