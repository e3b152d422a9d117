"""Which of its paths (one cluster, one cooperative launch per sweep, launches
per wave) local moving takes, told by the kernels launched, and the same result
from each: graphs on both sides of the cluster's limits."""
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


@pytest.fixture(scope="module")
def above_the_cluster():
    """R-MAT of 16 K vertices, above the cluster's float64 limits, and the oracle's partition."""
    off, tgt, w = graphgen.rmat(14, 16, seed=2)
    assert len(tgt) > 1 << 18
    return dev(off, tgt, w), oracle.louvain(oracle.Graph(off, tgt, w.astype(np.float64)), oracle.LouvainOptions(sync=True))


@pytest.mark.parametrize("caps", [{}, dict(groups_blocks_per_sm=1, w512_blocks_per_sm=1, block_blocks_per_sm=1, hub_blocks_per_sm=1),
                                  dict(groups_blocks_per_sm=3, w512_blocks_per_sm=32, block_blocks_per_sm=2, hub_blocks_per_sm=7),
                                  dict(group_max_degree=64, warp_max_degree=256, block_max_degree=1024, big_max_degree=1025)], ids=str)
def test_class_kernels_equal_the_oracle_under_any_caps(gsp, restore, above_the_cluster, caps):
    d, (Co, ost) = above_the_cluster
    gsp.set_tuning(**caps)
    (C, q, st), count = launches(gsp, lambda: gsp.louvain(*d, precision="fp64"))
    assert count > 17 * 3 * 3  # the first sweep's wave runs: groups, warps, an application at least
    assert st["iterations"] == ost["iterations"]
    assert np.array_equal(C.cpu().numpy().astype(np.uint32), Co)


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("n,k", [(700, 8), (9000, 60)])
def test_small_graphs_move_in_one_launch(gsp, restore, n, k, precision):
    """On the cluster a phase takes the same launches whatever its sweeps."""
    d = dev(*graphgen.planted(n=n, k=k, mean_degree=14, p_intra=0.8, seed=3))
    gsp.set_tuning(persist_max_vertices=0)
    K, m = gsp.vertex_weights(*d)

    def phase(sweeps):
        C, S = torch.arange(n, dtype=torch.int32, device="cuda"), K.clone()
        return gsp.local_move(*d, C, K, S, m, max_iterations=sweeps, precision=precision)

    (one, first), (more, second) = launches(gsp, lambda: phase(1)), launches(gsp, lambda: phase(20))
    assert one == 1 and more > 2 and first == second


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("n", [150000, 200000, 700000, 1300000])
def test_more_moves_than_threads_apply_them(gsp, n, precision):
    """One wave in which most vertices of a path move: each thread of the
    application takes up to four moves a round, for several rounds."""
    i = np.arange(n - 1, dtype=np.uint64)
    off, tgt, w = graphgen.edges_to_csr(n, i, i + 1, (1 + i * i % 7).astype(np.float32))  # whole weights
    d = dev(off, tgt, w)
    K, m = gsp.vertex_weights(*d)
    C, S = torch.arange(n, dtype=torch.int32, device="cuda"), K.clone()
    sweeps = gsp.local_move(*d, C, K, S, m, tolerance=0.0, max_iterations=3, waves=1, wave_repeats=1, no_return_from=0,
                            precision=precision)
    if precision == "fp64":
        want = oracle.move(oracle.Graph(off, tgt, w.astype(np.float64)), np.arange(n), K.cpu().numpy(), K.cpu().numpy(), m,
                           0.0, max_iterations=3, waves=1)
        assert sweeps == want[2]
        assert np.array_equal(C.cpu().numpy().astype(np.uint32), want[0])
    total = torch.zeros(n, dtype=torch.float64, device="cuda").scatter_add_(0, C.long(), K)
    assert torch.equal(S, total)  # whole sums
    assert int((C != torch.arange(n, dtype=torch.int32, device="cuda")).sum()) > n // 3
