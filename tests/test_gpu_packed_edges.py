"""Bit-packed edge arrays: widths from one bit to all 32, entries that cross
words, and every way a packed run of edges reaches a kernel (cache, explicit
copy by the copy engine, by a kernel or inside the device loop, gather, host
compaction, zero-copy)."""
import numpy as np
import pytest

from gen import graphgen as gg
from oracle import oracle as orc

from test_gpu_parity import check, engine, hy  # noqa: F401

pytestmark = pytest.mark.gpu

# (vertices, largest weight): target widths 1, 2, 5, 6, 11, 17 bits
SHAPES = [(2, 1), (3, 2), (32, 3), (33, 1 << 16), (1025, (1 << 20) - 1), (70001, 1 << 24)]
ROUTES = [dict(force_route=1), dict(force_route=2), dict(force_route=2, f_copy=1, f_ahead=1),
          dict(force_route=2, device_loop=2), dict(force_route=3), dict(force_route=3, compact_host=3),
          dict(force_route=4), dict(force_route=4, hub_frac=0.0), dict(force_route=5, seed=2)]


def graph(V, wmax, seed):
    g = gg.random_graph(V, 9 * V + 5, seed=seed, skew=1.2)
    rng = np.random.default_rng(seed)
    w = rng.integers(1, wmax + 1, g.E).astype(np.uint32)
    w[rng.integers(0, g.E)] = wmax
    return gg.CSR(g.V, g.E, g.off, g.dst, w, "packed")


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: f"V{s[0]}w{s[1]}")
@pytest.mark.parametrize("params", ROUTES, ids=lambda p: "-".join(f"{k}{v}" for k, v in p.items()))
def test_widths(hy, shape, params):
    V, wmax = shape
    g = graph(V, wmax, V)
    budget = g.E * 32 + (1 << 17) if params["force_route"] == 1 else g.E * 8 + (1 << 17)
    e = engine(hy, g, budget, part_bytes=2048, **params)
    for src in sorted({0, V // 2, V - 1}):
        check(g, "bfs", e.run("bfs", src), src)
        check(g, "sssp", e.run("sssp", src), src)
    srcs = [0, V - 1, V // 2]
    for row, s in zip(e.run("sssp", srcs), srcs):
        assert np.array_equal(row, orc.sssp(g, s)[0])
    assert e.info()["pinned_host_bytes"] <= g.E * 8 + 64
    e.close()


@pytest.mark.parametrize("force", [1, 2, 3, 4])
def test_full_width_weights(hy, force):
    """Weights of all 32 bits beside small ones (32-bit entries need no shift)."""
    V = 600
    g = graph(V, 50, 7)
    w = g.w.copy()
    w[:: g.E // 7] = 0x80000001
    g = gg.CSR(V, g.E, g.off, g.dst, w, "wide")
    want, _, ovf = orc.sssp(g, 1)
    assert not ovf
    e = engine(hy, g, g.E * 16 + (1 << 17), part_bytes=2048, force_route=force)
    assert np.array_equal(e.run("sssp", 1), want)
    e.close()


def test_symmetry_check_reads_packed_rows(hy):
    g = gg.random_graph(777, 5000, seed=3)
    s = gg.symmetrize(g)
    e = engine(hy, s, 1 << 20, part_bytes=4096)
    check(s, "cc", e.run("cc"))
    e.load(g)
    with pytest.raises(hy.HytgError) as ex:
        e.run("cc")
    assert ex.value.status == hy.HYTG_ERR_ARG
    e.close()
