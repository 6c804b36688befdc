"""The planning walk visits the frontier in units of four bitmap words (128
vertices): graphs that end inside a unit, partitions that end inside one, and
request sizes that are not powers of two, against the oracle's counts."""
import numpy as np
import pytest

from gen import graphgen as gg
from oracle import oracle as orc

from test_gpu_parity import check, engine, hy, internal_graph  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V", [31, 127, 128, 129, 1025, 40001])
@pytest.mark.parametrize("m", [128, 96])
def test_counts(hy, V, m):
    g = gg.random_graph(V, 6 * V, seed=V, skew=1.1)
    e = engine(hy, g, 1 << 22, part_bytes=4 * 64, m=m)       # partitions of one or two words
    vb = e.partitions()
    g2, perm = internal_graph(e, g)
    rng = np.random.default_rng(V)
    for algo, n_arrays in (("bfs", 1), ("sssp", 2), ("pagerank", 1)):
        for dens in (0.01, 0.5, 1.0):
            act = (rng.random(V) < dens).astype(np.uint8)
            _, counts = e.plan(algo, act)
            want = orc.partition_counts(g2, act[perm], vb, 4, n_arrays, m)
            assert np.array_equal(counts.T, np.array(want)), (algo, dens)
    e.close()


@pytest.mark.parametrize("V", [33, 129, 4097])
def test_results(hy, V):
    """Lists of units that span partitions of different routes."""
    g = gg.random_graph(V, 8 * V, seed=V + 1, skew=1.2)
    e = engine(hy, g, 1 << 20, part_bytes=4 * 96, force_route=5, seed=3)
    for algo, src in (("bfs", 0), ("sssp", V - 1), ("pagerank", None)):
        check(g, algo, e.run(algo, src), 0 if src is None else src)
    got = e.run("sssp", [0, V // 2, V - 1])
    for row, s in zip(got, (0, V // 2, V - 1)):
        assert np.array_equal(row, orc.sssp(g, s)[0])
    e.close()
