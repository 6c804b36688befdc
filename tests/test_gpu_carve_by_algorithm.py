"""A plan is the one of its own algorithm's run, whatever ran before, and runs
of several algorithms in turn keep the resident partitions: budgets that hold
one, two and more staging slots."""
import numpy as np
import pytest

from gen import graphgen as gg

from test_gpu_parity import engine, hy  # noqa: F401

pytestmark = pytest.mark.gpu

BUDGETS = range(34000, 120000, 1708)


@pytest.fixture(scope="module", params=[True, False], ids=["weighted", "unweighted"])
def eng(hy, request):
    g = gg.random_graph(4001, 65536, seed=9, weights=request.param)
    e = engine(hy, g, 1 << 20, part_bytes=8192)
    e.algos = ["bfs", "pagerank"] + (["sssp"] if request.param else [])
    yield e
    e.close()


def carve(e):
    i = e.info()
    return i["n_cached"], i["budget_used_bytes"], i["compact_edges"]


def test_history(eng):
    act = np.ones(eng.V, np.uint8)

    def plan(algo):
        routes, counts = eng.plan(algo, act)
        return (routes.tolist(), counts.tolist(), *carve(eng))

    for budget in BUDGETS:
        eng.set_budget(budget)
        want = {a: plan(a) for a in eng.algos}
        for before in eng.algos:
            eng.run(before, None if before == "pagerank" else 3)
            assert carve(eng) == want[before][2:], (budget, before)
            for a in eng.algos:
                assert plan(a) == want[a], (budget, before, a)


def test_cache_kept(eng):
    for budget in BUDGETS:
        eng.set_budget(budget)
        for n, algo in enumerate(["bfs", "ppr", "bfs", "ppr"]):
            eng.run(algo, 5)
            assert (eng.stats()["cache_fill_bytes"] > 0) == (n == 0 and carve(eng)[0] > 0), (budget, n)
