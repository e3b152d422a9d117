"""Member degrees that a tile sums in two halves, around the 16 bits of the low
one: aggregation of stars whose centres lie in one tile."""
import numpy as np
import pytest
import torch

import oracle
from paper_2402_11454_gb300 import graphgen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("parts", ["one", "own", "centres"])
@pytest.mark.parametrize("degrees", [(65535,), (65536, 1), (65537, 65535), (65535, 65535, 65535), (131072, 65536, 3)],
                         ids=str)
def test_degrees_around_16_bits(degrees, parts):
    from paper_2402_11454_gb300 import gsp
    V = len(degrees)
    n = V + max(degrees)
    u = np.repeat(np.arange(V), degrees).astype(np.uint64)
    v = np.concatenate([V + np.arange(d) for d in degrees]).astype(np.uint64)
    off, tgt, w = graphgen.edges_to_csr(n, u, v)
    i = np.arange(n)
    C = {"one": i * 0, "own": i, "centres": np.where(i < V, 0, 1 + i % 5)}[parts]
    C, _ = oracle.renumber(C.astype(np.uint32))
    k = int(C.max()) + 1
    want = oracle.aggregate(oracle.Graph(off, tgt, w.astype(np.float64)), C, k)
    go, gt, gw = gsp.aggregate(torch.from_numpy(off.astype(np.int64)).cuda(),
                               torch.from_numpy(tgt.astype(np.int32)).cuda(), torch.from_numpy(w).cuda(),
                               torch.from_numpy(C.astype(np.int32)).cuda(), k)
    assert np.array_equal(go.cpu().numpy().astype(np.uint64), want.offsets)
    assert np.array_equal(gt.cpu().numpy().astype(np.uint32), want.targets)
    assert np.array_equal(gw.cpu().numpy(), want.weights)  # whole sums
