"""Small-frontier iterations with the compaction route: the same run as the
host loop's, and the same link reads where an iteration has one edge; and a
run that passes its deadline inside them, after which the context runs on."""
import numpy as np
import pytest

from test_gpu_parity import check, engine, hy  # noqa: F401
from test_gpu_small_frontiers import GRAPHS, from_edges

pytestmark = pytest.mark.gpu


def chain(n):
    return from_edges(n, np.arange(n - 1), np.arange(1, n), 2)


@pytest.mark.parametrize("resident", [False, True])
@pytest.mark.parametrize("name", ["fan100", "mesh", "chain"])
@pytest.mark.parametrize("algo", ["bfs", "sssp"])
@pytest.mark.parametrize("force", [1, 3, 4])
def test_forced_route(hy, name, algo, force, resident):
    g = chain(700) if name == "chain" else GRAPHS[name]()
    runs = []
    for loop in (0, 1):
        e = engine(hy, g, g.E * 16 + (1 << 17) if resident else g.E * 3 + (1 << 16), part_bytes=4096,
                   force_route=force, device_loop=loop)
        check(g, algo, e.run(algo, 0))
        runs.append((e.stats(), e.iterations()))
        assert not resident or e.info()["n_cached"] == e.info()["n_parts"]
        e.close()
    (a, ia), (b, ib) = runs
    assert b["graph_iterations"] > 0
    for k in ("iterations", "edges_relaxed", "route_partitions", "route_edges", "link_bytes"):
        assert a[k] == b[k], k
    assert [r["link_bytes"] for r in ia] == [r["link_bytes"] for r in ib]
    if name == "chain":
        assert a["link_sector_bytes"] == b["link_sector_bytes"]
        assert a["link_line_bytes"] == b["link_line_bytes"]
        assert force == 1 or sum(b["link_sector_bytes"]) >= 32 * (g.V - 1)
    elif force != 1:
        assert b["link_sector_bytes"][force] > 0


@pytest.mark.parametrize("algo", ["bfs", "sssp"])
def test_deadline(hy, algo):
    g = chain(60000)
    e = engine(hy, g, g.E * 16 + (1 << 17), part_bytes=1 << 16, run_timeout_ms=5)
    with pytest.raises(hy.HytgError) as ex:
        e.run(algo, 0)
    assert ex.value.status == hy.HYTG_ERR_TIMEOUT
    e.set_param("run_timeout_ms", 0)
    check(g, algo, e.run(algo, 0))
    assert e.stats()["iterations"] >= g.V
    e.close()
