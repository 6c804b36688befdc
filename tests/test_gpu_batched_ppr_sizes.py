"""Batched PPR on both sides of the size where its F and C iterations leave the
device loop, with seed counts that fill frames of 8 and halves of 4 in part
(eight lanes share an edge of the push, four seeds each)."""
import numpy as np
import pytest

from gen import graphgen as gg
from oracle import oracle as orc

from test_gpu_parity import PR_TOL, engine, hy  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", params=[15, 17], ids=["rmat15", "rmat17"])
def g(request):
    return gg.rmat(request.param, seed=2)


@pytest.mark.parametrize("K", [2, 4, 9, 20])
def test_sizes(hy, g, K):
    rng = np.random.default_rng(K)
    src = rng.choice(np.flatnonzero(np.diff(g.off.astype(np.int64)) > 0), K, replace=False).tolist()
    e = engine(hy, g, g.E)
    got = e.run("ppr", src)
    for k in (0, K // 2, K - 1):
        x, _, _ = orc.pagerank(g, tol=1e-13, seed=src[k])
        assert float(np.abs(got[k].astype(np.float64) - x).sum()) <= PR_TOL, k
    st = e.stats()
    if g.E <= 1 << 20:
        assert st["graph_iterations"] >= st["iterations"] // 2
    e.close()
