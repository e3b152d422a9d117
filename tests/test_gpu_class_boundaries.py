"""A vertex's decision must not depend on which degree class serves it: the
boundaries between the classes are tunable."""
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


# degrees at the limits of the block classes, several vertices of each
DEGREES = np.repeat([520, 2048, 2050, 4096, 4098, 6000, 8192, 8194, 12000], 6)


@pytest.fixture(scope="module")
def ties():
    """Stars whose centre has half its leaves in its own community and half in
    one other, with totals Sigma that make staying and leaving an exact tie: the
    float32 rounding of the two scores alone decides, as numpy computes here."""
    rng = np.random.default_rng(5)
    V = len(DEGREES)
    first = V + np.concatenate([[0], np.cumsum(DEGREES)])
    n = int(first[-1])
    u = np.repeat(np.arange(V), DEGREES)
    off, tgt, w = graphgen.edges_to_csr(n, u.astype(np.uint64), np.arange(V, n).astype(np.uint64))
    C = np.arange(n, dtype=np.int32)
    K, Sigma = np.ones(n), np.ones(n)
    moves = np.zeros(V, dtype=bool)
    for h, deg in enumerate(DEGREES):
        here, there = np.arange(first[h], first[h] + deg // 2), np.arange(first[h] + deg // 2, first[h] + deg)
        C[here], C[there] = h, there[0]
        K[h] = np.float32(rng.uniform(1.0, 2.0))  # 2m = 1: also the factor of Sigma
        Sc = rng.uniform(0.3, 0.45) * deg / K[h]
        Sigma[there[0]], Sigma[h] = Sc, Sc + K[h]
        k, f, x, y = np.float32(deg // 2), np.float32(K[h]), np.float32(Sc), np.float32(Sigma[h] - K[h])
        leave = np.float32(float(k) - float(f) * float(x))  # one rounding: the product is exact in float64
        stay = np.float32(float(k) - float(f) * float(y)) if deg > 8192 else k - np.float32(f * y)
        moves[h] = leave - stay > 0
    active = np.zeros(n, dtype=np.uint8)
    active[:V] = 1
    dev = [torch.from_numpy(np.asarray(x)).cuda() for x in (off.astype(np.int64), tgt.astype(np.int32), w, C, K, Sigma)]
    want = np.where(moves, C[first[:-1] + DEGREES // 2], np.arange(V))
    assert 0 < moves.sum() < V and not moves[DEGREES > 8192].any()
    return dev, torch.from_numpy(active).cuda(), want


@pytest.mark.parametrize("bounds", [{}, {"big_max_degree": 4096}, {"big_max_degree": 2049},
                                    {"group_max_degree": 64, "warp_max_degree": 256, "block_max_degree": 1024}],
                         ids=str)
def test_exact_ties_do_not_depend_on_the_boundaries(gsp, restore, ties, bounds):
    dev, active, want = ties
    gsp.set_tuning(**bounds)
    choice = gsp.move_sweep(*dev, 0.5, active=active, precision="mixed")[0]
    assert np.array_equal(choice.cpu().numpy()[:len(want)], want)
