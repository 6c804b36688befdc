"""Accuracy of PageRank and PPR against 64 bits: many F tasks with their second
passes, a resident graph, hubs that take most edges, and a number of hub
replicas that no vector of four divides; and without replicas."""
import numpy as np
import pytest

from gen import graphgen as gg
from oracle import oracle as orc

from test_gpu_parity import engine, hy  # noqa: F401

pytestmark = pytest.mark.gpu

# The sums of a run are of some hundred 32-bit additions (a take per iteration);
# were each one's rounding kept in the result, rms 2^-24 / sqrt(3) of the value,
# a hundred would leave 3.4e-7 in the 2-norm where they point at random.  Half of
# it is asked for.
TOL = 1.7e-7


@pytest.mark.parametrize("graph", ["rmat", "chunglu"])
@pytest.mark.parametrize("algo,src", [("pagerank", None), ("ppr", 5)])
@pytest.mark.parametrize("budget", [0.3, 4.0])
@pytest.mark.parametrize("params", [dict(), dict(device_loop=2), dict(hub_replicas=1001)],
                         ids=lambda p: "-".join(f"{k}{v}" for k, v in p.items()) or "default")
def test_error(hy, graph, algo, src, budget, params):
    error(hy, graph, algo, src, budget, params, TOL)


@pytest.mark.parametrize("graph", ["rmat", "chunglu"])
@pytest.mark.parametrize("budget", [0.3, 4.0])
def test_no_replicas(hy, graph, budget):
    """Block sums then meet in one 32-bit residual, up to ten thousand an
    iteration: at random 100 roundings' worth of one, 2^-24 / sqrt(3) each,
    of a residual that is a fraction of the rank: 2^-20."""
    error(hy, graph, "pagerank", None, budget, dict(hub_replicas=0), 2.0 ** -20)


def error(hy, graph, algo, src, budget, params, tol):
    g = gg.rmat(17, seed=3, weights=False) if graph == "rmat" else gg.chung_lu(120001, 2000000, seed=3)
    e = engine(hy, g, g.E * 4 * budget + (1 << 18), part_bytes=1 << 17, **params)
    # the engine's damping is a 32-bit number: the 2.8e-8 by which it is off
    # count once per step of a walk, 6.7 times on average
    x, _, _ = orc.pagerank(g, d=float(np.float32(0.85)), tol=1e-14, **({} if src is None else {"seed": src}))
    for _ in range(2):
        got = e.run(algo, src).astype(np.float64)
        assert float(np.linalg.norm(got - x) / np.linalg.norm(x)) <= tol
    rank, delta = e.pagerank_state()
    s = float(rank.astype(np.float64).sum())
    assert np.linalg.norm(rank / s - got) <= 2.0 ** -23 * np.linalg.norm(got)
    e.close()
