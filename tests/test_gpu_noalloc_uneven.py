"""The allocation-free planning call on partitions of very different widths:
the isolated vertices of a degree-ordered graph in one partition, partitions
without a vertex, a table that starts or ends inside the graph, and every
number of words around the limits of its two forms; and its time there."""
from fractions import Fraction

import numpy as np
import pytest

from gen import graphgen as gg
from oracle import oracle as orc
from oracle import planner as pl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def call():
    torch = pytest.importorskip("torch")
    from paper_2208_14935_gb300 import build, hytg
    build.build()
    hytg.load()

    def make(off, vb, act):
        V, n = len(off) - 1, len(vb) - 1
        pad = np.zeros(-(-V // 32) * 32, np.uint8)
        pad[:V] = act
        d = [torch.from_numpy(x).cuda() for x in (np.packbits(pad, bitorder="little").view(np.int32).copy(),
                                                  off.astype(np.int64), vb.astype(np.int64))]
        routes = torch.full((n,), 255, dtype=torch.uint8, device="cuda")
        counts = torch.full((3 * n,), -1, dtype=torch.int64, device="cuda")

        def run():
            st = hytg.hytg_plan_noalloc(hytg.ALGOS["bfs"], d[0].data_ptr(), d[1].data_ptr(), V, d[2].data_ptr(), n,
                                        n // 3, routes.data_ptr(), counts.data_ptr(), params={"m": 128, "MR": 8},
                                        stream=torch.cuda.current_stream().cuda_stream)
            assert st == hytg.HYTG_OK
            return routes, counts
        return run
    return make


def tail_graph(V, seed):
    """Rows of the first half only, targets anywhere."""
    rng = np.random.default_rng(seed)
    deg = np.zeros(V, np.int64)
    deg[:V // 2 + 1] = rng.integers(1, 12, V // 2 + 1)
    off = np.zeros(V + 1, np.uint64)
    off[1:] = deg.cumsum()
    E = int(off[-1])
    return gg.CSR(V, E, off, rng.integers(0, V, E).astype(np.uint32), None)


def bounds(V, n, kind):
    cuts = np.unique(np.linspace(0, V // 2, n).astype(np.int64) // 32 * 32)
    vb = np.append(cuts[cuts < V], V)
    if kind == "repeats":                             # partitions without a vertex, also at both ends
        vb = np.sort(np.concatenate([vb, vb[::3], [0, 0, V, V]]))
    return vb


@pytest.mark.parametrize("kind", ["tail", "repeats"])
@pytest.mark.parametrize("n", [2, 40, 400, 3000])
@pytest.mark.parametrize("V", [33, 16384, 16385, 65536, 65537, 131073, 1100001])
def test_counts(call, V, n, kind):
    g = tail_graph(V, V + n)
    vb = bounds(V, n, kind)
    n = len(vb) - 1
    act = (np.random.default_rng(n).random(V) < 0.4).astype(np.uint8)
    routes, counts = call(g.off, vb, act)()
    na, ae, ln = orc.partition_counts(g, act, vb.astype(np.uint64), 4, 1, 128)
    assert np.array_equal(counts.cpu().numpy().reshape(n, 3), np.stack([na, ae, ln], 1).astype(np.int64))
    E_part = np.diff(g.off[vb].astype(np.int64))
    want = pl.plan(E_part, na, ae, ln, 4, resident=range(n // 3), m=128, MR=8, alpha=Fraction("0.8"),
                   beta=Fraction("0.4"), gamma=Fraction("0.625"))
    assert routes.cpu().tolist() == want


@pytest.mark.parametrize("V", [16384, 131073])
def test_captured(call, V):
    torch = pytest.importorskip("torch")
    g = tail_graph(V, V)
    vb = bounds(V, 40, "tail")
    run = call(g.off, vb, (np.random.default_rng(V).random(V) < 0.4).astype(np.uint8))
    want = [x.clone() for x in run()]
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        got = run()
    for _ in range(3):
        for x in got:
            x.fill_(7)
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(got, want))


def test_time(call):
    """Half the vertices in the last of 2,048 partitions against equal
    partitions: the same words and rows are read, so at most twice the time
    (launches, and a last wave that is not full)."""
    torch = pytest.importorskip("torch")
    V, n = 1 << 22, 2048
    off = np.minimum(np.arange(V + 1, dtype=np.int64), V // 2) * 8
    act = np.ones(V, np.uint8)

    def us(vb):
        run = call(off, vb, act)
        best = 1e9
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            run()
            a.record()
            for _ in range(20):
                run()
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b) / 20 * 1e3)
        return best
    even = us(np.linspace(0, V, n + 1).astype(np.int64) // 32 * 32)
    assert us(bounds(V, n, "tail")) <= 2 * even
