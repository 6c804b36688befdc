"""F copies inside the device loop are counted as copied, bit-packed: the same
bytes, in the totals and in every iteration's record, as the host loop counts
for one copy per partition ("k" 1).  Not batched SSSP: it pushes values as they
stand, so its iterations differ from run to run."""
import numpy as np
import pytest

from gen import graphgen as gg

from test_gpu_parity import engine, hy  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("force", [-1, 2])
@pytest.mark.parametrize("algo,src,loop", [("bfs", 1, 2), ("sssp", 1, 2), ("bfs", [1, 2, 7], 1)],
                         ids=lambda x: str(x).replace(" ", ""))
def test_same_as_host_loop(hy, algo, src, loop, force):
    g = gg.random_graph(9001, 150000, seed=3)
    runs = []
    for device_loop in (loop, 0):
        e = engine(hy, g, g.E * (8 if algo == "sssp" else 4) // 3, part_bytes=8192, k=1, force_route=force,
                   device_loop=device_loop)
        r = e.run(algo, src)
        st, its = e.stats(), e.iterations()
        e.close()
        runs.append((r, st, [int(i["link_bytes"]) for i in its]))
    (a, sa, la), (b, sb, lb) = runs
    assert np.array_equal(a, b)
    assert sa["graph_iterations"] > 0 and sb["graph_iterations"] == 0
    assert sa["link_bytes"][2] == sb["link_bytes"][2]
    assert sa["link_bytes"][2] > 0 or force == -1         # the cost model may find every edge a better route
    assert sa["link_sector_bytes"][2] == sb["link_sector_bytes"][2] == sa["link_bytes"][2]
    assert la == lb
