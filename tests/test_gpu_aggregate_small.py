"""Aggregation of small graphs: sizes around a tile of 256 vertices, around the
size where the tiles grow to 1024, and numbers of small communities around the
one up to which one launch serves both warp classes."""
import numpy as np
import pytest
import torch

import oracle
from paper_2402_11454_gb300 import graphgen

pytestmark = pytest.mark.gpu


def check(n, C):
    from paper_2402_11454_gb300 import gsp
    i = np.arange(n - 1, dtype=np.uint64)
    skip = np.arange(n - 3, dtype=np.uint64)
    off, tgt, w = graphgen.edges_to_csr(n, np.concatenate([i, skip]), np.concatenate([i + 1, skip + 3]))
    C, _ = oracle.renumber(C.astype(np.uint32))
    k = int(C.max()) + 1
    want = oracle.aggregate(oracle.Graph(off, tgt, w.astype(np.float64)), C, k)
    go, gt, gw = gsp.aggregate(torch.from_numpy(off.astype(np.int64)).cuda(), torch.from_numpy(tgt.astype(np.int32)).cuda(),
                               torch.from_numpy(w).cuda(), torch.from_numpy(C.astype(np.int32)).cuda(), k)
    assert np.array_equal(go.cpu().numpy().astype(np.uint64), want.offsets)
    assert np.array_equal(gt.cpu().numpy().astype(np.uint32), want.targets)
    assert np.array_equal(gw.cpu().numpy(), want.weights)  # whole sums


@pytest.mark.parametrize("blocks", [0, 1, 2, 304])  # whole tiles of 256 before the odd vertices
@pytest.mark.parametrize("odd", [-1, 0, 1, 5])
@pytest.mark.parametrize("parts", ["own", "mod", "giant"])
def test_sizes_around_a_tile(blocks, odd, parts):
    n = 256 * blocks + odd
    if n < 4:
        pytest.skip("too few vertices")
    i = np.arange(n)
    check(n, {"own": i, "mod": i % 7, "giant": np.where(i % 10, 0, i)}[parts])


@pytest.mark.parametrize("small", [0, 1, 3])  # communities of the 128-slot class among them
@pytest.mark.parametrize("count", [1215, 1216, 1217])
def test_communities_around_one_launch(small, count):
    big = count - small  # 40 vertices, total degree about 160
    C = np.concatenate([np.repeat(np.arange(big), 40), big + np.repeat(np.arange(small), 4)])
    check(len(C), C)
