"""The shared-table sums of the phase calls.  Aggregation at the total degrees where a community changes kernel (64, 512,
2048 entries, tasks of 2048) and in each form of the table values: 32-bit units
beside their key, 64-bit units, float64."""
import numpy as np
import pytest
import torch

import oracle
from paper_2402_11454_gb300 import graphgen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gsp():
    from paper_2402_11454_gb300 import build
    build.build()
    from paper_2402_11454_gb300 import gsp as g
    return g


TOTALS = (1, 63, 64, 65, 127, 128, 129, 511, 512, 513, 2047, 2048, 2049, 4096, 4097, 9000)


def stars():
    """Vertex t has TOTALS[t] neighbours of degree one (its community's total
    degree when it is alone); the leaves form communities of five."""
    base = len(TOTALS)
    u = np.concatenate([np.full(d, t) for t, d in enumerate(TOTALS)])
    v = base + np.arange(len(u))
    n = base + len(u)
    off, tgt, _ = graphgen.edges_to_csr(n, u.astype(np.uint64), v.astype(np.uint64))
    C = np.concatenate([np.arange(base), base + np.arange(len(u)) // 5]).astype(np.uint32)
    return off, tgt, C


@pytest.mark.parametrize("values", ["unit", "whole", "real", "wide"])
@pytest.mark.parametrize("self_edges", [False, True])
def test_aggregate_at_class_boundaries(gsp, values, self_edges):
    off, tgt, C = stars()
    if self_edges:  # every other star's leaves join its community
        leaf_of = np.repeat(np.arange(len(TOTALS)), TOTALS)
        inside = leaf_of % 2 == 0
        C = C.copy()
        C[len(TOTALS):][inside] = leaf_of[inside]
    C, _ = oracle.renumber(C)
    k = int(C.max()) + 1
    rng = np.random.default_rng(2)
    w = {"unit": np.ones(len(tgt)), "whole": rng.integers(1, 100, len(tgt)),
         "real": rng.integers(1 << 20, 1 << 24, len(tgt)) / 2.0 ** 20,     # total above 2^32 units
         "wide": 2.0 ** rng.integers(-30, 30, len(tgt)).astype(np.float64)}[values].astype(np.float32)
    want = oracle.aggregate(oracle.Graph(off, tgt, w.astype(np.float64)), C, k)
    oo, ot, ow = want.offsets, want.targets, want.weights
    go, gt, gw = gsp.aggregate(torch.from_numpy(off.astype(np.int64)).cuda(),
                               torch.from_numpy(tgt.astype(np.int32)).cuda(), torch.from_numpy(w).cuda(),
                               torch.from_numpy(C.astype(np.int32)).cuda(), k)
    assert np.array_equal(go.cpu().numpy().astype(np.uint64), oo)
    assert np.array_equal(gt.cpu().numpy().astype(np.uint32), ot)
    # "wide" spans 60 binary orders: float64 sums in any order, n terms
    assert np.allclose(gw.cpu().numpy(), ow, rtol=0 if values != "wide" else 9000 * 2.0 ** -53, atol=0)


@pytest.mark.parametrize("shift", [0, 1, 2, 3])
@pytest.mark.parametrize("parts", ["giant", "few", "own"])
def test_sums_on_views_and_crowded_communities(gsp, shift, parts):
    """Targets and weights that start off a 16-byte boundary, and communities
    that hold most rows, a handful or one row each: K, Q and the super-graph
    are exact (whole weights)."""
    off, tgt, _ = graphgen.rmat(12, 10, seed=3)
    n = len(off) - 1
    rng = np.random.default_rng(shift)
    w = rng.integers(1, 50, len(tgt)).astype(np.float32)
    C = {"giant": np.where(rng.random(n) < 0.9, 7, np.arange(n)), "few": rng.integers(0, 5, n),
         "own": np.arange(n)}[parts].astype(np.uint32)
    g = oracle.Graph(off, tgt, w.astype(np.float64))

    def view(x):
        t = torch.from_numpy(np.concatenate([np.zeros(shift, x.dtype), x])).cuda()
        return t[shift:]

    dev = (torch.from_numpy(off.astype(np.int64)).cuda(), view(tgt.astype(np.int32)), view(w))
    K, m = gsp.vertex_weights(*dev)
    Ko, mo = oracle.vertex_weights(g)
    assert np.array_equal(K.cpu().numpy(), Ko) and m == mo
    dC = torch.from_numpy(C.astype(np.int32)).cuda()
    assert gsp.modularity(*dev, dC) == pytest.approx(oracle.modularity(g, C), rel=1e-12, abs=1e-14)
    D, k = gsp.renumber(dC)
    want = oracle.aggregate(g, oracle.renumber(C)[0], k)
    go, gt, gw = gsp.aggregate(*dev, D, k)
    assert np.array_equal(go.cpu().numpy().astype(np.uint64), want.offsets)
    assert np.array_equal(gt.cpu().numpy().astype(np.uint32), want.targets)
    assert np.array_equal(gw.cpu().numpy(), want.weights)
