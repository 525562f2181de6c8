"""What a batch leaves an arena holding: workspaces for the CTAs that had jobs, and nothing that a budget has no room for."""
import pytest

import inputs

pytestmark = pytest.mark.gpu

SIDE = 400  # large enough for a group of CTAs of its own


def _arena(cd, count, budget=0):
    arena = cd.arena_create(hbm_budget_bytes=budget)
    for i in range(count):
        e = inputs.grid(SIDE, 1000, i + 1)
        arena.add(e.src, e.dst, e.w, e.n)
    return arena


@pytest.mark.parametrize("count", [1, 4])
def test_workspaces_of_the_jobs_alone(count):
    import paper_1506_03265_gb300 as cd
    arena = _arena(cd, count)
    before = arena.info()[1]
    arena.run(list(range(count)), [0.5] * count, [1] * count)
    # at most a workspace per job: some 92 bytes a node, three dense matrices of 4 MiB (152 of them: 2 GB)
    assert arena.info()[1] - before <= count * (SIDE * SIDE * 100 + (13 << 20))


@pytest.mark.parametrize("count", [1, 4])
def test_budget(count):
    import paper_1506_03265_gb300 as cd
    free = _arena(cd, count)
    used = free.info()[1]
    args = (list(range(count)), [0.5] * count, list(range(1, count + 1)))
    want = free.run(*args)
    # room for another graph's arrays (they double), not for the workspaces of 28 MB each beside them: the batch may hold
    # those meanwhile, an add takes their place
    arena = _arena(cd, count, used + count * (10 << 20))
    for _ in range(2):
        assert arena.run(*args) == want
    e = inputs.grid(100, 1000, 9)
    assert arena.add(e.src, e.dst, e.w, e.n) == count and arena.info()[1] <= used + count * (10 << 20)
    assert arena.run(args[0] + [count], args[1] + [0.5], args[2] + [3])[1] == [0] * (count + 1)
    # a server too: its own workspaces, one a CTA, need the room
    arena = _arena(cd, count)
    assert arena.run(*args) == want
    cd.server_create(arena, ctas=2, hbm_budget_bytes=used + (60 << 20)).free()
