"""Batched PPR's copies of the hub rows: no copies, one id, a few, and all 64
(fewer hubs than that on the small graph), with and without a second pass,
in one run and in serving, where a slot is used again after a finished query."""
import numpy as np
import pytest

from gen import graphgen as gg
from oracle import oracle as orc

from test_gpu_parity import PR_TOL, engine, hy  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", params=[301, 9001], ids=["v301", "v9001"])
def g(request):
    return gg.chung_lu(request.param, 12 * request.param, seed=4)


def check(g, got, src):
    x, _, _ = orc.pagerank(g, tol=1e-13, seed=src)
    assert float(np.abs(got.astype(np.float64) - x).sum()) <= PR_TOL, src


@pytest.mark.parametrize("two_pass", [0, 1])
@pytest.mark.parametrize("replicas", [0, 2, 7, 4096])
def test_hub_rows(hy, g, replicas, two_pass):
    rng = np.random.default_rng(replicas + 1)
    src = rng.choice(np.flatnonzero(np.diff(g.off.astype(np.int64)) > 0), 13, replace=False).tolist()
    e = hy.Engine(g, budget=4 * (g.E * 8 + g.V * 8) + 4 * g.V * 96 + (1 << 20),
                  params={"part_bytes": 4096, "hub_replicas": replicas, "two_pass": two_pass})
    rows = e.run("ppr", src)
    for k in (0, 7, 12):
        check(g, rows[k], src[k])
    one = e.run("ppr", src[0])                       # single-source replicas share the memory
    check(g, one, src[0])
    ppr = hy.ALGOS["ppr"]
    hy.hytg_serve_begin(e.ctx, ppr, 3)
    todo, slot = list(src[:7]), {}
    while todo or slot:
        for s in range(3):
            if s not in slot and todo:
                slot[s] = todo.pop()
                hy.hytg_serve_admit(e.ctx, s, slot[s])
        fin, _ = hy.hytg_serve_step(e.ctx)
        for s in [s for s in slot if (fin >> s) & 1]:
            check(g, hy.hytg_serve_fetch(e.ctx, s, g.V, ppr), slot.pop(s))
    hy.hytg_serve_end(e.ctx)
    e.close()
