"""PageRank and PPR relaxes that sum hub ids in shared memory: graphs with fewer
vertices than the sums, with V around their numbers, without hub sorting, and
with a few targets that take most edges; every route, with and without the
second pass and the device loop."""
import numpy as np
import pytest

from gen import graphgen as gg

from test_gpu_parity import check, engine, hy  # noqa: F401

pytestmark = pytest.mark.gpu


def star(V, E, seed):
    """Most edges end in a handful of vertices, some in one."""
    rng = np.random.default_rng(seed)
    src = np.sort(rng.integers(0, V, E))
    dst = np.where(rng.random(E) < 0.3, 1 % V, np.where(rng.random(E) < 0.5, rng.integers(0, min(V, 70), E),
                                                      rng.integers(0, V, E)))
    o = np.lexsort((dst, src))
    off = np.zeros(V + 1, np.uint64)
    off[1:] = np.cumsum(np.bincount(src, minlength=V)).astype(np.uint64)
    return gg.CSR(V, E, off, dst[o].astype(np.uint32), None, "star")


@pytest.mark.parametrize("V", [255, 256, 1027, 4095, 4096, 16385])
@pytest.mark.parametrize("params", [dict(force_route=1), dict(force_route=2), dict(force_route=3), dict(force_route=4),
                                    dict(force_route=5, seed=3), dict(two_pass=0), dict(device_loop=0),
                                    dict(device_loop=2), dict(hub_frac=0.0)],
                         ids=lambda p: "-".join(f"{k}{v}" for k, v in p.items()))
def test_small(hy, V, params):
    g = star(V, 40000, V)
    budget = g.E * 8 + (1 << 17) if params.get("force_route") == 1 else g.E * 2 + (1 << 16)
    e = engine(hy, g, budget, part_bytes=16384, **params)
    check(g, "pagerank", e.run("pagerank"))
    check(g, "ppr", e.run("ppr", 3), 3)
    e.close()


def test_wide(hy):
    """Above the size where a block sums 16,384 ids."""
    g = gg.rmat(19, seed=5, weights=False)
    e = engine(hy, g, g.E * 6, part_bytes=4 << 20)
    check(g, "pagerank", e.run("pagerank"))
    e.set_budget(int(g.E * 1.5))
    check(g, "pagerank", e.run("pagerank"))
    e.close()
