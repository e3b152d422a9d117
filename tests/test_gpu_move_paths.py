"""Which of its paths (one cluster, one cooperative launch per sweep, launches
per wave) local moving takes, told by the kernels launched, and the same result
from each: graphs on both sides of the cluster's limits."""
import numpy as np
import pytest
import torch

from paper_2402_11454_gb300 import graphgen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gsp():
    from paper_2402_11454_gb300 import build
    build.build()
    from paper_2402_11454_gb300 import gsp as g
    return g


@pytest.fixture()
def restore(gsp):
    saved = gsp.get_tuning()
    yield
    gsp.set_tuning(**saved)


def dev(off, tgt, w):
    return (torch.from_numpy(off.astype(np.int64)).cuda(), torch.from_numpy(tgt.astype(np.int32)).cuda(),
            torch.from_numpy(w).cuda())


def launches(gsp, fn):
    before = gsp.kernel_launches()
    out = fn()
    return out, gsp.kernel_launches() - before


# unit weights: the mixed mode's float32 sums are exact in any order.  2 K
# vertices: every pass on the cluster; 40 K (640 K entries): the first is above its limits
@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("n,k", [(2000, 12), (40000, 100)])
def test_persistent_sweep_comes_first_where_asked_for(gsp, restore, n, k, precision):
    d = dev(*graphgen.planted(n=n, k=k, mean_degree=16, p_intra=0.8, seed=6))
    gsp.set_tuning(persist_max_vertices=0)
    (C0, q0, st0), without = launches(gsp, lambda: gsp.louvain(*d, precision=precision))
    gsp.set_tuning(persist_max_vertices=1 << 20)
    (C1, q1, st1), asked = launches(gsp, lambda: gsp.louvain(*d, precision=precision))
    assert st1["iterations"] == st0["iterations"] and torch.equal(C0, C1) and q0 == q1
    # a pass asked for takes two launches a sweep (the sweep, its iteration number), on the cluster one in all
    more = sum(2 * s - 1 for s in st0["iterations"])
    if n == 2000:
        assert asked - without == more
    else:  # the first pass: 17 waves run three times in the first sweep, a decision and an application each
        assert without - asked + more >= 17 * 3 * 2 - 1
    # graphs above the setting keep the library's choice
    gsp.set_tuning(persist_max_vertices=1)
    assert launches(gsp, lambda: gsp.louvain(*d, precision=precision))[1] == without


def test_autotune_leaves_caps_that_nothing_reads(gsp, restore):
    d = dev(*graphgen.planted(n=3000, k=12, mean_degree=16, p_intra=0.8, seed=6))  # every pass on the cluster
    odd = dict(groups_blocks_per_sm=5, w512_blocks_per_sm=5, block_blocks_per_sm=7, hub_blocks_per_sm=3)
    gsp.set_tuning(**odd)
    _, one = launches(gsp, lambda: gsp.louvain(*d))
    (caps, _, _), all_runs = launches(gsp, lambda: gsp.autotune(*d))
    assert {k: caps[k] for k in odd} == odd
    # the four boundaries' trials and the final pair, not the 18 candidates of the caps twice each
    assert all_runs < 36 * one
