"""Setup stages bit for bit against the oracle where their kernels' tiles end: the
pivoted QR in clusters of 1 to 8 CTAs (few to many nodes a level), more columns than
one pass of its warps, equal columns (ties), blocks that lose rank or nearly all
their size; random-projection neighbor lists with leaves past one chunk of 512
candidates, duplicates, and coordinates that are no multiple of 4; subnormal, zero
and negative-zero coordinates (the exact widening to FP64)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _same(X, **kw):
    import oracle
    from paper_1410_0260_gb300 import askit
    o = oracle.Tree(X, oracle.Config(**kw))
    g = askit.Tree(torch.from_numpy(X).cuda(), askit.Config(**kw))
    ids, dist = o.knn()
    assert np.array_equal(g.structure(askit.STRUCT_KNN), ids)
    assert np.array_equal(g.structure(askit.STRUCT_KNN_DIST), dist)
    assert np.array_equal(g.structure(askit.STRUCT_PERM), o.perm())
    nodes = [o.node(a) for a in range(2, o.nnodes)]
    assert np.array_equal(g.structure(askit.STRUCT_SKEL_IDS), np.concatenate([n["skel"] for n in nodes]))
    assert np.array_equal(g.structure(askit.STRUCT_P), np.concatenate([n["P"].ravel() for n in nodes]))
    g.close()


@pytest.mark.parametrize("N,leaf,s_max,tol,h,kind", [
    (260, 130, 33, 0.0, 1.0, "plain"),           # two nodes: clusters of 8
    (1500, 700, 100, 0.0, 1.0, "plain"),         # 375 columns a leaf
    (2600, 1300, 40, 1e-3, 0.7, "plain"),        # 1300 columns: several groups a warp
    (3000, 20, 12, 0.0, 1.0, "plain"),           # 128 leaves and more: one CTA a node
    (640, 80, 64, 1e-12, 1.0, "duplicates"),     # equal columns
    (640, 80, 64, 0.0, 1e4, "plain"),            # nearly rank one
    (640, 80, 64, 0.0, 0.02, "plain"),           # nearly empty blocks: tiny norms
    (512, 64, 16, 0.0, 1.0, "same"),             # rank one exactly
])
def test_skeletons(N, leaf, s_max, tol, h, kind):
    rng = np.random.default_rng(N + leaf)
    X = rng.standard_normal((N, 4)).astype(np.float32)
    if kind == "duplicates":
        X[1::2] = X[::2]
    elif kind == "same":
        X[:] = X[0]
    _same(X, leaf_size=leaf, kappa=6, knn_mode=0, s_max=s_max, id_tol=tol, h=h, seed=3)


@pytest.mark.parametrize("N,d,leaf,kappa,kind", [
    (100, 3, 40, 1, "plain"),
    (1400, 5, 700, 32, "plain"),                 # leaves of 700: two chunks
    (5000, 8, 64, 16, "duplicates"),
    (9000, 7, 2048, 8, "plain"),                 # whole-level sorts, then segments
    (3000, 6, 100, 8, "odd_values"),
])
def test_random_projection_lists(N, d, leaf, kappa, kind):
    rng = np.random.default_rng(N + d)
    X = rng.standard_normal((N, d)).astype(np.float32)
    if kind == "duplicates":
        X[1::3] = X[::3][: len(X[1::3])]
    elif kind == "odd_values":
        X[:, 0] = np.where(rng.random(N) < 0.5, np.float32(-0.0), np.float32(0.0))
        X[:, 1] *= np.float32(1e-41)             # subnormal
        X[:, 2] *= np.float32(1e15)
    _same(X, leaf_size=leaf, kappa=kappa, knn_mode=1, rp_iters=3, s_max=8, id_tol=0.0, h=1.0, seed=4)
