"""The relax kernels' walk over a route's edges (runs of 32 to 256 edges, windows
of 31 lists, tiles of 2,048 edges) and the second passes' lists, on degree
patterns that put list bounds on, before and after those sizes."""
import numpy as np
import pytest

from gen import graphgen as gg
from oracle import oracle as orc

from test_gpu_parity import PR_TOL, check, engine, hy  # noqa: F401

pytestmark = pytest.mark.gpu

PATTERNS = {
    "ones": [1] * 3000,                                   # windows of 31 lists inside every run
    "steps": [31, 32, 33] * 300,
    "runs": [255, 256, 257, 1, 0, 2] * 40,
    "tiles": [2047, 1, 2048, 2049, 0, 0, 3] * 8,
    "hub": [70001] + [0] * 500 + [1, 5] * 200,            # one list over many tiles
}


def graph(degrees, seed):
    """Row v has degrees[v] random targets, sorted, and weights in [1, 64]."""
    rng = np.random.default_rng(seed)
    V = len(degrees)
    off = np.zeros(V + 1, np.uint64)
    off[1:] = np.cumsum(np.asarray(degrees, np.uint64))
    E = int(off[-1])
    src = np.repeat(np.arange(V), degrees)
    dst = rng.integers(0, V, E)
    dst = dst[np.lexsort((dst, src))].astype(np.uint32)
    return gg.CSR(V, E, off, dst, rng.integers(1, 65, E).astype(np.uint32), "pattern")


@pytest.mark.parametrize("name", sorted(PATTERNS))
@pytest.mark.parametrize("force", [1, 2, 3, 4])
def test_patterns(hy, name, force):
    g = graph(PATTERNS[name], 5)
    budget = g.E * 16 + (1 << 16) if force == 1 else g.E * 8 + (1 << 16)
    e = engine(hy, g, budget, force_route=force, part_bytes=8192, hub_frac=0.0, two_pass=2,
               two_pass_min_degree=0)
    src = int(np.argmax(np.diff(g.off.astype(np.int64))))
    for algo in ("bfs", "sssp", "pagerank"):
        check(g, algo, e.run(algo, None if algo == "pagerank" else src), src)
        if algo == "pagerank" and force <= 2:
            assert e.stats()["extra_edges"] > 0           # the second passes' lists were used
    rows = e.run("sssp", [src, 0, g.V - 1])
    for row, s in zip(rows, (src, 0, g.V - 1)):
        assert np.array_equal(row, orc.sssp(g, s)[0])
    rows = e.run("ppr", [src, 0])
    for row, s in zip(rows, (src, 0)):
        x, _, _ = orc.pagerank(g, tol=1e-13, seed=s)
        assert float(np.abs(row.astype(np.float64) - x).sum()) <= PR_TOL
    e.close()
