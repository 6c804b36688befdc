"""Small-frontier iterations of the device loop: one cluster runs whole
iterations until a frontier outgrows its queue, a warp's lists get long, or a
route needs copies, and the loop's body goes on from there.  Results,
iterations, edges and routes must be those of the host loop."""
import numpy as np
import pytest

from gen import graphgen as gg
from oracle import oracle as orc

from test_gpu_parity import check, engine, hy  # noqa: F401

pytestmark = pytest.mark.gpu


def from_edges(V, src, dst, seed, wmax=50):
    o = np.lexsort((dst, src))
    src, dst = np.asarray(src)[o], np.asarray(dst)[o]
    off = np.zeros(V + 1, np.uint64)
    off[1:] = np.cumsum(np.bincount(src, minlength=V)).astype(np.uint64)
    w = np.random.default_rng(seed).integers(1, wmax + 1, len(src)).astype(np.uint32)
    return gg.CSR(V, len(src), off, dst.astype(np.uint32), w, "small")


def chain_and_fan(fan, seed=1):
    """A path of 300 vertices, a vertex with `fan` children, each with a path of
    40 more: frontiers of one vertex, then of `fan` for 40 iterations."""
    src, dst = list(range(300)), list(range(1, 301))
    base = 301
    for k in range(40):
        a = np.arange(fan) + base + k * fan
        src += [300] * fan if k == 0 else (a - fan).tolist()
        dst += a.tolist()
    return from_edges(base + 40 * fan, src, dst, seed)


GRAPHS = {
    "fan100": lambda: chain_and_fan(100),
    "fan1500": lambda: chain_and_fan(1500),            # a list above a warp's 1,024 edges
    "fan4097": lambda: chain_and_fan(4097),            # a frontier above the queue
    "mesh": lambda: gg.mesh(257, 33, shortcut_frac=0.002, radius=8, wmax=1000),
}


@pytest.mark.parametrize("name", sorted(GRAPHS))
@pytest.mark.parametrize("algo", ["bfs", "sssp", "cc"])
@pytest.mark.parametrize("force", [-1, 1, 4])
def test_same_run(hy, name, algo, force):
    g = GRAPHS[name]()
    if algo == "cc" and name != "mesh":
        g = gg.symmetrize(g)
    budget = g.E * 16 + (1 << 17) if force == 1 else g.E * 3 + (1 << 16)
    runs = {}
    for loop in (0, 1):
        e = engine(hy, g, budget, part_bytes=4096, force_route=force, device_loop=loop)
        got = e.run(algo, None if algo == "cc" else 0)
        check(g, algo, got)
        runs[loop] = (got, e.stats(), e.iterations())
        e.close()
    assert np.array_equal(runs[0][0], runs[1][0])
    assert runs[1][1]["graph_iterations"] > 0
    if algo != "cc":                                   # pointer jumping reads labels while they change
        a, b = runs[0][1], runs[1][1]
        for k in ("iterations", "edges_relaxed", "vertices_processed", "route_partitions", "route_vertices",
                  "route_edges", "link_bytes"):
            assert a[k] == b[k], k
        key = ("active_vertices", "active_edges", "route_partitions", "route_edges", "link_bytes")
        assert [[r[k] for k in key] for r in runs[0][2]] == [[r[k] for k in key] for r in runs[1][2]]


@pytest.mark.parametrize("delta", [0, 7, 300])
def test_buckets(hy, delta):
    g = GRAPHS["mesh"]()
    its = set()
    for loop in (0, 1):
        e = engine(hy, g, g.E * 3, part_bytes=4096, sssp_delta=delta, device_loop=loop)
        check(g, "sssp", e.run("sssp", 5), 5)
        its.add((e.stats()["iterations"], e.stats()["edges_relaxed"]))
        e.close()
    assert len(its) == 1


@pytest.mark.parametrize("cap", [1, 2, 17, 250])
def test_iteration_cap(hy, cap):
    g = GRAPHS["fan100"]()
    e = engine(hy, g, g.E * 16 + (1 << 17), part_bytes=4096, max_iters=cap)
    got = e.run("bfs", 0)
    assert e.stats()["iterations"] == cap
    want, _ = orc.bfs(g, 0)
    assert np.array_equal(got, np.where(want <= cap, want, np.uint32(0xFFFFFFFF)))
    e.close()


def test_many_records(hy):
    """More iterations than the loop's record ring holds."""
    n = 5000
    g = from_edges(n, np.arange(n - 1), np.arange(1, n), 2)
    e = engine(hy, g, g.E * 16 + (1 << 17), part_bytes=1 << 16)
    check(g, "bfs", e.run("bfs", 0))
    its = e.iterations()
    # the last vertex has no edge: its iteration relaxes none
    assert len(its) == e.stats()["iterations"] == n
    assert sum(r["active_edges"] for r in its) == e.stats()["edges_relaxed"] == n - 1
    e.close()
