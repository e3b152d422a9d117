"""Small graphs move inside one thread-block cluster, large ones by a launch
per class and wave; a graph's result must not depend on which of the two
served it.  A batch member gets its solo result, and a batch as a whole takes
the path of its total size: members beside a large filler run on the launches,
alone on the cluster."""
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


def degree_edges(n, degrees, seed):
    """A sparse random graph of n vertices in which vertex d has degrees[d]
    neighbours or a few more (the edges of the degree classes and tables)."""
    rng = np.random.default_rng(seed)
    u = [rng.integers(0, n, n), ]
    v = [rng.integers(0, n, n), ]
    for i, d in enumerate(degrees):
        u.append(np.full(d, i))
        v.append(rng.choice(np.arange(len(degrees), n), size=d, replace=False))
    return np.concatenate(u).astype(np.uint64), np.concatenate(v).astype(np.uint64)


def whole_weights(off, tgt, k, seed):
    """Symmetric whole-number weights 1..k."""
    i = np.repeat(np.arange(len(off) - 1, dtype=np.uint64), np.diff(off).astype(np.int64))
    a, b = np.minimum(i, tgt.astype(np.uint64)), np.maximum(i, tgt.astype(np.uint64))
    h = (a * np.uint64(0x9E3779B97F4A7C15) + b * np.uint64(0xBF58476D1CE4E5B9) + np.uint64(seed)) >> np.uint64(40)
    return (1 + h % np.uint64(k)).astype(np.float32)


def small_graphs():
    out = []
    for n, degrees, seed in ((700, (8, 9, 16, 17, 32, 33, 128, 129, 512, 513), 1),
                             (6144, (2048, 2049, 511, 129, 6000), 2), (6145, (2047, 2050, 4100), 3),
                             (12288, (8192, 8193, 12000, 600), 4), (12289, (8192, 9000), 5), (2, (), 6)):
        off, tgt, w = graphgen.edges_to_csr(n, *degree_edges(n, degrees, seed))
        out.append((off, tgt, w))
        out.append((off, tgt, whole_weights(off, tgt, 7, seed)))
    out.append(graphgen.planted(n=3000, k=12, mean_degree=40, p_intra=0.6, seed=4))
    out.append(graphgen.rmat(11, 24, seed=4))
    return out


SMALL = small_graphs()


def dev(off, tgt, w):
    return (torch.from_numpy(np.asarray(off).astype(np.int64)).cuda(),
            torch.from_numpy(np.asarray(tgt).astype(np.int32)).cuda(),
            torch.from_numpy(np.asarray(w).astype(np.float32)).cuda())


@pytest.mark.parametrize("kw", [{}, {"precision": "fp64"}, {"waves": 1, "wave_repeats": 2}, {"waves": 64},
                                {"max_iterations": 1}, {"singleton_rule": False, "waves": 3, "no_return_from": 1}],
                         ids=lambda kw: ",".join(f"{k}={v}" for k, v in kw.items()) or "default")
def test_cluster_path_equals_launches(gsp, kw):
    kw = dict(kw, max_passes=3)
    filler = graphgen.planted(n=40000, k=100, mean_degree=32, p_intra=0.7, seed=9)
    gs = SMALL + [filler]
    n = [len(g[0]) - 1 for g in gs]
    gvo = np.concatenate([[0], np.cumsum(n)]).astype(np.uint64)
    ends = np.concatenate([[0], np.cumsum([len(g[1]) for g in gs])]).astype(np.uint64)
    off = np.concatenate([[0]] + [g[0][1:].astype(np.uint64) + e for g, e in zip(gs, ends)])
    tgt = np.concatenate([g[1].astype(np.uint64) + v for g, v in zip(gs, gvo)])
    w = np.concatenate([g[2] for g in gs])
    C, q, _ = gsp.louvain_batched(gvo, *dev(off, tgt, w), **kw)
    C, q = C.cpu().numpy(), q.cpu().numpy()
    for i, g in enumerate(SMALL):
        Cs, qs, _ = gsp.louvain(*dev(*g), **kw)
        assert np.array_equal(C[int(gvo[i]):int(gvo[i + 1])], Cs.cpu().numpy()), f"graph {i}"
        assert q[i] == pytest.approx(qs, rel=1e-12, abs=1e-15), f"graph {i}"


@pytest.mark.parametrize("exp", [-100, -21, 20, 90])
@pytest.mark.parametrize("graph", ["rmat", "wide"])
def test_mixed_scores_do_not_depend_on_the_weights_scale(gsp, graph, exp):
    """Scaling every weight by a power of two scales the float32 scores
    exactly, so every decision stays the same whatever the exponents of Sigma
    (its conversion to float32 works on the bits)."""
    off, tgt, w = SMALL[-1] if graph == "rmat" else SMALL[1]
    C, q, st = gsp.louvain(*dev(off, tgt, w))
    Cs, qs, sts = gsp.louvain(*dev(off, tgt, np.ldexp(w, exp)))
    assert torch.equal(C, Cs)
    assert sts["iterations"] == st["iterations"]
    assert qs == pytest.approx(q, rel=1e-12)
