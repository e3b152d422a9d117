"""The degree-class lists at the sizes where their tiles change (256 vertices,
2048, the largest graph with small tiles), with one wave (ranks taken by the
lanes of a key together) and with several: each vertex is listed once."""
import numpy as np
import pytest
import torch

import oracle
from paper_2402_11454_gb300 import graphgen

pytestmark = pytest.mark.gpu

SMS = 152
SIZES = [3, 255, 256, 257, 2047, 2049, 256 * 4 * SMS - 1, 256 * 4 * SMS, 256 * 4 * SMS + 1]


def combs(n):
    """Paths of up to 40 vertices, every third also tied to the vertex two on;
    some vertices without edges."""
    i = np.arange(n - 1)
    i = i[i % 41 != 0]
    j = np.arange(n - 2)
    j = j[(j % 3 == 0) & (j % 41 < 38) & (j % 41 > 0)]
    return graphgen.edges_to_csr(n, np.concatenate([i, j]).astype(np.uint64),
                                 np.concatenate([i + 1, j + 2]).astype(np.uint64))


@pytest.mark.parametrize("n", SIZES)
def test_lists_hold_every_vertex(n):
    from paper_2402_11454_gb300 import gsp
    off, tgt, w = combs(n)
    g = oracle.Graph(off, tgt, w.astype(np.float64))
    dev = (torch.from_numpy(off.astype(np.int64)).cuda(), torch.from_numpy(tgt.astype(np.int32)).cuda())
    C = (np.arange(n) // 41).astype(np.uint32)
    lab, _ = gsp.split(*dev, torch.from_numpy(C.astype(np.int32)).cuda(), mode="lp")  # one wave
    assert np.array_equal(lab.cpu().numpy().astype(np.uint32), oracle.split_lp(g, C)[0])
    wd = torch.from_numpy(w).cuda()
    for waves in (1, 17):
        K, m = gsp.vertex_weights(*dev, wd)
        ident, S = torch.arange(n, dtype=torch.int32, device="cuda"), K.clone()
        gsp.local_move(*dev, wd, ident, K, S, m, tolerance=0.0, max_iterations=2, waves=waves, wave_repeats=1,
                       no_return_from=0)
        want = oracle.move(g, np.arange(n), K.cpu().numpy(), K.cpu().numpy(), m, 0.0, max_iterations=2, waves=waves)
        assert np.array_equal(ident.cpu().numpy().astype(np.uint32), want[0])
