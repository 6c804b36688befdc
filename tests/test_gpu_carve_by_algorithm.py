"""A plan is the one of its own algorithm's run, whatever ran before, and runs
of several algorithms in turn keep the resident partitions."""
import numpy as np
import pytest

from gen import graphgen as gg

from test_gpu_parity import engine, hy  # noqa: F401

pytestmark = pytest.mark.gpu


def test_history(hy):
    g = gg.rmat(13, seed=9)
    e = engine(hy, g, g.E * 8, part_bytes=8192)
    act = np.ones(g.V, np.uint8)
    first = int(np.flatnonzero(np.diff(g.off.astype(np.int64)))[0])

    def plan(algo):
        routes, counts = e.plan(algo, act)[:2]
        i = e.info()
        return routes.tolist(), np.asarray(counts).tolist(), i["n_cached"], i["budget_used_bytes"], i["compact_edges"]

    def run(algo):
        e.run(algo, None if algo == "pagerank" else first)
        i = e.info()
        return i["n_cached"], i["budget_used_bytes"], i["compact_edges"]

    sizes = set()
    for budget in range(g.E * 2, g.E * 4, g.E // 16 + 52):
        e.set_budget(budget)
        want = {a: plan(a) for a in ("bfs", "pagerank", "sssp")}
        for before in ("bfs", "pagerank", "sssp"):
            assert run(before) == want[before][2:], (budget, before)
            for a in want:
                assert plan(a) == want[a], (budget, before, a)
        sizes.add(want["bfs"][2])
    assert len(sizes) > 3


def test_cache_kept(hy):
    g = gg.rmat(13, seed=9, weights=False)
    e = engine(hy, g, g.E * 8, part_bytes=8192)
    for budget in range(int(g.E * 1.5), int(g.E * 3.5), g.E // 16 + 52):
        e.set_budget(budget)
        for n, algo in enumerate(["bfs", "ppr", "bfs", "ppr"]):
            e.run(algo, 5)
            st = e.stats()
            assert (st["cache_fill_bytes"] > 0) == (n == 0 and e.info()["n_cached"] > 0), (budget, n)
