"""Arrays made on first use: a call that runs out of device memory at any of
them (made on the host by HYTG_INJECT_DEVMEM_FAIL) says so, and the next call
makes what is missing and gives the right result."""
import pytest

from gen import graphgen as gg
from oracle import oracle as orc

from test_gpu_parity import PR_TOL, check, hy  # noqa: F401

pytestmark = pytest.mark.gpu

SECOND_PASS = ["d_sp_ebase", "d_sp_soff", "d_sp_tiles", "d_sp_cursor"]


@pytest.fixture
def e(hy):
    g = gg.rmat(12, seed=6)
    eng = hy.Engine(g, budget=g.E * 8 + 4 * g.V * 96 + (1 << 17), params={"part_bytes": 8192})
    eng.graph = g
    yield eng
    eng.close()


def refused(hy, call):
    with pytest.raises(hy.HytgError) as ex:
        call()
    assert ex.value.status == hy.HYTG_ERR_CUDA and "device allocation" in str(ex.value)


@pytest.mark.parametrize("name", SECOND_PASS + ["d_rank_lo"])
@pytest.mark.parametrize("algo", ["pagerank", "ppr"])
def test_second_pass(hy, e, monkeypatch, name, algo):
    before = e.info()["vertex_state_bytes"]
    src = None if algo == "pagerank" else 3
    monkeypatch.setenv("HYTG_INJECT_DEVMEM_FAIL", name)
    refused(hy, lambda: e.run(algo, src))
    refused(hy, lambda: e.run(algo, src))
    monkeypatch.delenv("HYTG_INJECT_DEVMEM_FAIL")
    check(e.graph, algo, e.run(algo, src), src)
    info = e.info()
    n = info["n_parts"]
    assert info["vertex_state_bytes"] - before == e.V * 20 + (e.graph.E // 2048 + n + 2) * 4 + n * 8


@pytest.mark.parametrize("name", SECOND_PASS + ["d_sp_pay64", "d_sp_vid", "d_pay64", "d_vid", "d_bout", "bs.fr32", "frame"])
def test_batched_ppr(hy, e, monkeypatch, name):
    src = [3, 5, 9]
    monkeypatch.setenv("HYTG_INJECT_DEVMEM_FAIL", name)
    refused(hy, lambda: e.run("ppr", src))
    monkeypatch.delenv("HYTG_INJECT_DEVMEM_FAIL")
    for row, s in zip(e.run("ppr", src), src):
        x, _, _ = orc.pagerank(e.graph, tol=1e-13, seed=s)
        assert float(abs(row.astype("f8") - x).sum()) <= PR_TOL


@pytest.mark.parametrize("name", ["d_pay64", "d_vid", "bs.fr", "bs.vis", "bs.nxt", "frame"])
def test_batched_sssp(hy, e, monkeypatch, name):
    src = [3, 5, 9]
    monkeypatch.setenv("HYTG_INJECT_DEVMEM_FAIL", name)
    refused(hy, lambda: e.run("sssp", src))
    monkeypatch.delenv("HYTG_INJECT_DEVMEM_FAIL")
    for row, s in zip(e.run("sssp", src), src):
        check(e.graph, "sssp", row, s)


@pytest.mark.parametrize("name", ["d_sp_soff", "d_sp_vid", "d_vid"])
def test_serving(hy, e, monkeypatch, name):
    """A session that cannot be opened leaves none behind: a run, then a
    session, work."""
    monkeypatch.setenv("HYTG_INJECT_DEVMEM_FAIL", name)
    refused(hy, lambda: hy.hytg_serve_begin(e.ctx, hy.ALGOS["ppr"], 2))
    monkeypatch.delenv("HYTG_INJECT_DEVMEM_FAIL")
    check(e.graph, "bfs", e.run("bfs", 3), 3)
    hy.hytg_serve_begin(e.ctx, hy.ALGOS["ppr"], 2)
    hy.hytg_serve_admit(e.ctx, 0, 3)
    while not hy.hytg_serve_step(e.ctx)[0] & 1:
        pass
    check(e.graph, "ppr", hy.hytg_serve_fetch(e.ctx, 0, e.V, hy.ALGOS["ppr"]), 3)
    hy.hytg_serve_end(e.ctx)
