"""The allocation-free planning call over the shapes of its grid: one block per
partition, and partitions cut into slices, with a frontier that ends inside a
word and bits set beyond V, against the oracle's counts and routes."""
from fractions import Fraction

import numpy as np
import pytest

from gen import graphgen as gg
from oracle import oracle as orc
from oracle import planner as pl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V,step", [
    (1, 32), (33, 32), (4097, 32), (4097, 8192),     # a word per partition; one partition
    (300001, 9216), (300001, 65536),                 # 288 and 2,048 words: slices
    (2000003, 2000032),                              # one partition of 62,501 words
])
@pytest.mark.parametrize("m", [128, 96])
def test_shapes(V, step, m):
    torch = pytest.importorskip("torch")
    from paper_2208_14935_gb300 import build, hytg
    build.build()
    hytg.load()
    g = gg.random_graph(V, 4 * V, seed=V, skew=1.2)
    vb = np.array(list(range(0, V, step)) + [V], np.uint64)
    n = len(vb) - 1
    rng = np.random.default_rng(V + m)
    off = torch.from_numpy(g.off.view(np.int64)).cuda()
    vbd = torch.from_numpy(vb.view(np.int64)).cuda()
    E_part = np.diff(g.off[vb.astype(np.int64)].astype(np.int64))
    for algo, d1, arrays in (("bfs", 4, 1), ("sssp", 8, 2)):
        act = (rng.random(V) < 0.3).astype(np.uint8)
        pad = np.ones(-(-V // 32) * 32, np.uint8)    # bits beyond V are ignored
        pad[:V] = act
        fr = torch.from_numpy(np.packbits(pad, bitorder="little").view(np.int32).copy()).cuda()
        routes = torch.full((n,), 255, dtype=torch.uint8, device="cuda")
        counts = torch.full((3 * n,), -1, dtype=torch.int64, device="cuda")
        st = hytg.hytg_plan_noalloc(hytg.ALGOS[algo], fr.data_ptr(), off.data_ptr(), V, vbd.data_ptr(), n, n // 3,
                                    routes.data_ptr(), counts.data_ptr(), params={"m": m, "MR": 8},
                                    stream=torch.cuda.current_stream().cuda_stream)
        assert st == hytg.HYTG_OK
        torch.cuda.synchronize()
        na, ae, ln = orc.partition_counts(g, act, vb, 4, arrays, m)
        got = counts.cpu().numpy().reshape(n, 3)
        assert np.array_equal(got, np.stack([na, ae, ln], 1).astype(np.int64))
        want = pl.plan(E_part, na, ae, ln, d1, resident=range(n // 3), m=m, MR=8, alpha=Fraction("0.8"),
                       beta=Fraction("0.4"), gamma=Fraction("0.625"))
        assert routes.cpu().tolist() == want
