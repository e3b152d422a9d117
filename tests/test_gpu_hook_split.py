"""The hooking split at the lengths where a row changes hands (sampled entries,
a warp, a block, a column of blocks), on partitions that leave long rows
outside their community's tree, and in a workspace without room for its lists."""
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


LENGTHS = (1, 7, 8, 9, 40, 263, 264, 265, 16391, 16392, 16393, 40000)


@pytest.fixture(scope="module")
def fans():
    """Vertex t of the first few is joined to LENGTHS[t] high ids; a sparse
    chain runs through every seventh id."""
    n = 60000
    rng = np.random.default_rng(11)
    u = [np.arange(100, n - 7, 7)]
    v = [np.arange(107, n, 7)]
    for t, d in enumerate(LENGTHS):
        u.append(np.full(d, t))
        v.append(rng.choice(np.arange(len(LENGTHS), n), size=d, replace=False))
    off, tgt, w = graphgen.edges_to_csr(n, np.concatenate(u).astype(np.uint64), np.concatenate(v).astype(np.uint64))
    return oracle.Graph(off, tgt, w.astype(np.float64)), (torch.from_numpy(off.astype(np.int64)).cuda(),
                                                          torch.from_numpy(tgt.astype(np.int32)).cuda())


@pytest.mark.parametrize("parts", ["one", "halves", "random", "late", "own"])
@pytest.mark.parametrize("mode", ["lpp", "sv"])
def test_hook_split_matches_oracle(gsp, fans, parts, mode):
    g, dev = fans
    n = dev[0].numel() - 1
    rng = np.random.default_rng(3)
    C = {"one": np.zeros(n), "halves": np.arange(n) % 2, "random": rng.integers(0, 50, n),
         # the long rows share a community with targets that come late in their rows only
         "late": np.where(np.arange(n) < len(LENGTHS), n - 1, np.where(np.arange(n) > n // 2, n - 1, 5)),
         "own": np.arange(n)}[parts].astype(np.uint32)
    want = oracle.split_bfs(g, C)
    for _ in range(3):
        lab, k = gsp.split(*dev, torch.from_numpy(C.astype(np.int32)).cuda(), mode=mode)
        assert np.array_equal(lab.cpu().numpy().astype(np.uint32), want)
        assert k == len(np.unique(want))


def test_smallest_workspace_gives_the_same(gsp):
    off, tgt, w = graphgen.rmat(13, 8, seed=5)
    dev = (torch.from_numpy(off.astype(np.int64)).cuda(), torch.from_numpy(tgt.astype(np.int32)).cuda(),
           torch.from_numpy(w).cuda())
    for kw in ({"max_passes": 1}, {}):
        C, q, st = gsp.louvain(*dev, **kw)
        lo, hi = 0, st["workspace_bytes"]
        buf = torch.empty(hi + 256, dtype=torch.uint8, device="cuda")
        base = (-buf.data_ptr()) % 256
        while hi - lo > 256:  # the smallest accepted size, and the same result at every accepted one
            size = (lo + hi) // 2 // 256 * 256
            try:
                Cs, qs, _ = gsp.louvain(*dev, workspace=buf[base:base + size], **kw) if size else (None, None, None)
            except RuntimeError:
                Cs = None
            if Cs is None:
                lo = size
                continue
            hi = size
            assert torch.equal(Cs, C) and qs == q
        assert hi <= st["workspace_bytes"]
