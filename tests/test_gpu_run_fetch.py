"""hytg_run_fetch: the run's result in one call, with the buffer's pages faulted
in by host threads meanwhile.  Buffers at and around the size where that
starts, at odd addresses, longer than the result, and too small; and several
contexts at once."""
import threading

import numpy as np
import pytest

from gen import graphgen as gg
from oracle import oracle as orc

from test_gpu_parity import engine, hy  # noqa: F401

pytestmark = pytest.mark.gpu


def run_into(hy, e, algo, src, out, nbytes):
    import ctypes
    s = np.ascontiguousarray(src, np.uint32)
    return hy.load().hytg_run_fetch(e.ctx, hy.ALGOS[algo], s.ctypes.data_as(ctypes.c_void_p), len(s),
                                    out.ctypes.data_as(ctypes.c_void_p), nbytes)


@pytest.mark.parametrize("V", [1000, 1048575, 1048576, 1048577, 1400003])
def test_buffers(hy, V):
    g = gg.random_graph(V, 3 * V, seed=V)
    e = engine(hy, g, g.E * 8 + (1 << 20))
    want, _ = orc.bfs(g, 7)
    for off in (0, 1, 16383, 16384):                   # words: page and off-page starts
        buf = np.full(off + V + 20000, 0xABABABAB, np.uint32)
        assert run_into(hy, e, "bfs", [7], buf[off:], (V + 20000) * 4) == hy.HYTG_OK
        assert np.array_equal(buf[off:off + V], want)
        assert (buf[:off] == 0xABABABAB).all() and (buf[off + V:] == 0xABABABAB).all()
    out = np.full(3 * V, 5, np.uint32)
    assert run_into(hy, e, "bfs", [7, 0, V - 1], out, out.nbytes) == hy.HYTG_OK
    for row, s in zip(out.reshape(3, V), (7, 0, V - 1)):
        assert np.array_equal(row, orc.bfs(g, s)[0])
    assert run_into(hy, e, "bfs", [7], out, 4 * V - 4) == hy.HYTG_ERR_ARG      # too small for the result
    assert run_into(hy, e, "bfs", [V], out, out.nbytes) == hy.HYTG_ERR_ARG     # the run's own error
    assert np.array_equal(e.run("bfs", 7), want)                               # the context stays usable
    e.close()


def test_contexts_in_threads(hy):
    g = gg.random_graph(1200000, 2400000, seed=4)
    engines = [engine(hy, g, g.E * 8 + (1 << 20)) for _ in range(3)]
    want = [orc.bfs(g, s)[0] for s in range(6)]
    bad = []

    def work(k):
        for rep in range(4):
            s = (k + rep) % 6
            if not np.array_equal(engines[k].run("bfs", s), want[s]):
                bad.append((k, s))

    th = [threading.Thread(target=work, args=(k,)) for k in range(3)]
    for t in th:
        t.start()
    for t in th:
        t.join()
    for e in engines:
        e.close()
    assert not bad
