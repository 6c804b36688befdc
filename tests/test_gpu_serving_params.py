"""Parameters set while a serving session is open: the next step makes what
they need (the second pass's arrays, a new carve of the edge side beside the
queries' frames), and queries in flight end with the right result."""
import numpy as np
import pytest

from gen import graphgen as gg
from oracle import oracle as orc

from test_gpu_parity import PR_TOL, hy  # noqa: F401

pytestmark = pytest.mark.gpu

CHANGES = [[("two_pass", 1)], [("two_pass", 1), ("two_pass", 0), ("two_pass", 2)], [("part_bytes", 4096)],
           [("part_bytes", 65536), ("two_pass", 1)], [("streams", 1), ("k", 1), ("prefetch_slots", 0)],
           [("staging_frac", 0.5), ("compact_frac", 0.01)], [("part_bytes", 8192), ("f_ahead", 1), ("part_bytes", 16384)]]


@pytest.fixture(scope="module")
def g():
    return gg.rmat(13, seed=8)


@pytest.mark.parametrize("changes", CHANGES, ids=lambda c: "-".join(f"{k}{v}" for k, v in c))
@pytest.mark.parametrize("algo", ["ppr", "sssp"])
def test_set_between_steps(hy, g, algo, changes):
    frames = g.V * (96 if algo == "ppr" else 32) * 2
    e = hy.Engine(g, budget=int(g.E * 8 * 0.6) + frames + (1 << 17), params={"part_bytes": 16384, "two_pass": 0})
    rng = np.random.default_rng(3)
    src = rng.choice(np.flatnonzero(np.diff(g.off.astype(np.int64)) > 0), 12, replace=False).tolist()
    a = hy.ALGOS[algo]
    hy.hytg_serve_begin(e.ctx, a, 10)                 # two frames of eight queries
    todo, slot, out, step = list(range(12)), {}, {}, 0
    changes = list(changes)
    while todo or slot:
        for s in range(10):
            if s not in slot and todo:
                slot[s] = todo.pop()
                hy.hytg_serve_admit(e.ctx, s, src[slot[s]])
        step += 1
        if step % 2 == 0 and changes:
            e.set_param(*changes.pop(0))
        fin, _ = hy.hytg_serve_step(e.ctx)
        for s in [s for s in slot if (fin >> s) & 1]:
            out[slot.pop(s)] = hy.hytg_serve_fetch(e.ctx, s, g.V, a)
    hy.hytg_serve_end(e.ctx)
    assert not changes
    for k, got in out.items():
        if algo == "sssp":
            assert np.array_equal(got, orc.sssp(g, src[k])[0])
        else:
            x, _, _ = orc.pagerank(g, tol=1e-13, seed=src[k])
            assert float(np.abs(got.astype(np.float64) - x).sum()) <= PR_TOL
    e.close()


@pytest.mark.parametrize("replace", ["graph", "budget", "frontier"])
@pytest.mark.parametrize("algo", ["ppr", "bfs"])
def test_replaced_under_a_session(hy, g, algo, replace):
    """A session whose graph, device budget or frontier is replaced can only be
    closed."""
    budget = g.E * 8 + g.V * 96 * 2 + (1 << 17)
    e = hy.Engine(g, budget=budget, params={"part_bytes": 16384})
    a = hy.ALGOS[algo]
    hy.hytg_serve_begin(e.ctx, a, 2)
    hy.hytg_serve_admit(e.ctx, 0, 3)
    hy.hytg_serve_step(e.ctx)
    if replace == "frontier":
        e.plan(algo, np.ones(g.V, np.uint8))
    else:
        e.load(g) if replace == "graph" else e.set_budget(budget)
    for call in (lambda: hy.hytg_serve_step(e.ctx), lambda: hy.hytg_serve_admit(e.ctx, 1, 4),
                 lambda: hy.hytg_serve_fetch(e.ctx, 0, g.V, a)):
        with pytest.raises(hy.HytgError) as ex:
            call()
        assert ex.value.status == hy.HYTG_ERR_STATE
    hy.hytg_serve_end(e.ctx)
    hy.hytg_serve_begin(e.ctx, a, 2)
    hy.hytg_serve_admit(e.ctx, 0, 3)
    while not hy.hytg_serve_step(e.ctx)[0] & 1:
        pass
    got = hy.hytg_serve_fetch(e.ctx, 0, g.V, a)
    hy.hytg_serve_end(e.ctx)
    if algo == "bfs":
        assert np.array_equal(got, orc.bfs(g, 3)[0])
    else:
        assert float(np.abs(got.astype(np.float64) - orc.pagerank(g, tol=1e-13, seed=3)[0]).sum()) <= PR_TOL
    e.close()
