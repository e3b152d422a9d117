"""Float64 decisions of rows at the limits of the block and hub classes, with
numbers of communities around a warp's lanes: candidates are packed over the
lanes before they are scored, and weights of one community are summed over the
lanes before they are stored.  Decisions equal the oracle's bit for bit."""
import numpy as np
import pytest
import torch

import oracle
from paper_2402_11454_gb300 import graphgen

pytestmark = pytest.mark.gpu

DEGREES = (513, 2047, 2048, 2049, 4096, 4097, 8191, 8192, 8193, 12000)


def rows(communities, shuffled):
    """One centre per degree; its leaves lie in `communities` communities (0:
    each in its own), one after the other or shuffled, the first in the centre's."""
    rng = np.random.default_rng(communities + 7)
    V = len(DEGREES)
    first = V + np.concatenate([[0], np.cumsum(DEGREES)])
    n = int(first[-1])
    u, v = np.repeat(np.arange(V), DEGREES).astype(np.uint64), np.arange(V, n).astype(np.uint64)
    w = rng.integers(1, 9, n - V).astype(np.float32)  # whole weights: sums are exact in any order
    off, tgt, w = graphgen.edges_to_csr(n, u, v, w)
    C = np.arange(n)
    for h in range(V):
        leaves = np.arange(first[h], first[h + 1])
        if communities:
            part = leaves[0] + np.arange(len(leaves)) * communities // len(leaves)
            C[leaves] = rng.permutation(part) if shuffled else part
        C[leaves[:1]] = h
    K = np.concatenate([np.add.reduceat(w, off[:-1].astype(np.int64))]).astype(np.float64)
    Sigma = np.bincount(C, weights=K, minlength=n)
    active = np.zeros(n, dtype=np.uint8)
    active[:V] = 1
    return off, tgt, w, C.astype(np.uint32), K, Sigma, K.sum() / 2, active


@pytest.mark.parametrize("communities", [1, 2, 31, 32, 33, 64, 97, 1000, 0])
@pytest.mark.parametrize("shuffled", [False, True])
def test_long_rows_decide_as_the_oracle(communities, shuffled):
    from paper_2402_11454_gb300 import gsp
    off, tgt, w, C, K, Sigma, m, active = rows(communities, shuffled)
    g = oracle.Graph(off, tgt, w.astype(np.float64))
    want = oracle.move_sweep_sync(g, C, K, Sigma, m, active)[0]
    dev = [torch.from_numpy(x).cuda() for x in (off.astype(np.int64), tgt.astype(np.int32), w, C.astype(np.int32), K,
                                                Sigma)]
    V = len(DEGREES)
    assert (want[:V] != C[:V]).any()
    for weights in (dev[2], dev[2].double()):
        choice = gsp.move_sweep(dev[0], dev[1], weights, *dev[3:], float(m),
                                active=torch.from_numpy(active).cuda(), precision="fp64")[0]
        assert np.array_equal(choice.cpu().numpy()[:V].astype(np.uint32), want[:V])
