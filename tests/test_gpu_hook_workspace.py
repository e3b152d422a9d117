"""The hooking split without room for its trees and lists of long rows: the
count of disconnected communities at the end of a call that does not aggregate
sets the workspace's peak, so a slightly smaller workspace runs it without them."""
import numpy as np
import pytest
import torch

import oracle
from paper_2402_11454_gb300 import graphgen

pytestmark = pytest.mark.gpu


def fans():
    """Rows from one entry to a column of blocks, and a sparse chain."""
    n, lengths = 60000, (1, 8, 9, 264, 265, 16392, 16393, 40000)
    rng = np.random.default_rng(12)
    u = [np.arange(100, n - 7, 7)] + [np.full(d, t) for t, d in enumerate(lengths)]
    v = [np.arange(107, n, 7)] + [rng.choice(np.arange(len(lengths), n), size=d, replace=False) for d in lengths]
    return graphgen.edges_to_csr(n, np.concatenate(u).astype(np.uint64), np.concatenate(v).astype(np.uint64))


@pytest.mark.parametrize("graph", ["rmat", "fans"])
def test_count_without_room_for_the_lists(graph):
    from paper_2402_11454_gb300 import _lib, gsp
    off, tgt, w = graphgen.rmat(12, 24, seed=5) if graph == "rmat" else fans()
    dev = (torch.from_numpy(off.astype(np.int64)).cuda(), torch.from_numpy(tgt.astype(np.int32)).cuda(),
           torch.from_numpy(w).cuda())
    kw = dict(split="none", count_disconnected=True, aggregation_tolerance=1e-9, precision="fp64")
    gsp.louvain(*dev, **kw)
    before = gsp.kernel_launches()
    C, q, st = gsp.louvain(*dev, **kw)
    with_room = gsp.kernel_launches() - before
    g = oracle.Graph(off, tgt, w.astype(np.float64))
    assert st["disconnected"] == oracle.disconnected(g, C.cpu().numpy().astype(np.uint32))[0]
    peak = st["workspace_bytes"]
    buf = torch.empty(peak + 256, dtype=torch.uint8, device="cuda")
    base = (-buf.data_ptr()) % 256
    with pytest.raises(_lib.GspError):
        gsp.set_tuning(groups_blocks_per_sm=0)
    failed = _lib.load().gsp_last_error()
    without = 0
    for size in range(peak // 256 * 256, 0, -256):
        before = gsp.kernel_launches()
        try:
            Cs, qs, sts = gsp.louvain(*dev, workspace=buf[base:base + size], **kw)
        except _lib.GspError as e:
            assert "(-5)" in str(e) or "(-2)" in str(e)  # too small for the rest of the call
            break
        launched = gsp.kernel_launches() - before
        assert torch.equal(Cs, C) and qs == q and sts["disconnected"] == st["disconnected"]
        assert launched in (with_room, with_room - 2)  # one pass to the roots and the long rows' launch less
        without += launched == with_room - 2
        assert _lib.load().gsp_last_error() == failed  # no call has failed since
        if without == 4:
            break
    assert without
