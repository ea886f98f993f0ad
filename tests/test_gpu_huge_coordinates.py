"""Neighbor lists, bit for bit against the oracle, where squared distances leave FP32's
range (coordinates of 1e19 and more: outliers, missing-value markers) and only their
FP64 values are finite."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _points(N, d, kind, rng):
    X = rng.standard_normal((N, d)).astype(np.float32)
    if kind == "outliers":
        X[5::97] *= np.float32(1e20)
    elif kind == "marker":
        X[::11, d // 2] = np.float32(-1e30)
    elif kind == "all":
        X *= np.float32(2e19)                        # most distances past the range
    return X


def _lists(X, **kw):
    import oracle
    from paper_1410_0260_gb300 import askit
    o = oracle.Tree(X, oracle.Config(**kw))
    g = askit.Tree(torch.from_numpy(X).cuda(), askit.Config(**kw))
    ids, dist = o.knn()
    assert ids.max() < len(X) and ids.min() >= 0
    assert np.array_equal(g.structure(askit.STRUCT_KNN), ids)
    assert np.array_equal(g.structure(askit.STRUCT_KNN_DIST), dist)
    assert np.array_equal(g.structure(askit.STRUCT_PERM), o.perm())
    return g


@pytest.mark.parametrize("N,d,leaf,kappa,kind", [
    (600, 5, 64, 8, "outliers"),
    (600, 8, 64, 32, "marker"),
    (1300, 4, 600, 16, "all"),                       # leaves past one chunk of 512 candidates
])
def test_random_projection_lists_past_the_fp32_range(N, d, leaf, kappa, kind):
    X = _points(N, d, kind, np.random.default_rng(N + d))
    _lists(X, leaf_size=leaf, kappa=kappa, knn_mode=1, rp_iters=3, s_max=8, id_tol=0.0, h=1.0, seed=4).close()


@pytest.mark.parametrize("N,d,kappa,kind", [(300, 5, 8, "outliers"), (700, 8, 32, "marker"), (1300, 70, 16, "all")])
def test_exhaustive_lists_past_the_fp32_range(N, d, kappa, kind):
    import oracle
    rng = np.random.default_rng(N + d)
    X = _points(N, d, kind, rng)
    g = _lists(X, leaf_size=64, kappa=kappa, knn_mode=0, s_max=8, id_tol=0.0, h=1.0, seed=4)
    # the tree's own points as queries, and (d > 64) new points
    rows = np.arange(0, N, 7, dtype=np.int32)
    ids, dist = g.knn_points(torch.from_numpy(rows).cuda())
    oi, od = oracle.knn_exact(X, kappa, rows=rows.astype(np.int64))
    assert np.array_equal(ids.cpu().numpy(), oi) and np.array_equal(dist.cpu().numpy(), od)
    if d > 64:
        Y = _points(40, d, kind, rng)
        ids, dist = g.knn_targets(torch.from_numpy(Y).cuda())
        oi, od = oracle.knn_exact(X, kappa, Y=Y)
        assert np.array_equal(ids.cpu().numpy(), oi) and np.array_equal(dist.cpu().numpy(), od)
    g.close()


@pytest.mark.parametrize("scale", [4e18, 1e-19])
def test_new_points_at_the_ends_of_the_fp32_range(scale):
    """Norms around the mean overflow for some points (4e18), or the tensor-core
    scale's square does (1e-19), while the neighbors themselves are ordinary."""
    import oracle
    rng = np.random.default_rng(3)
    X = (rng.standard_normal((5000, 8)) * scale).astype(np.float32)
    Y = (rng.standard_normal((500, 8)) * 1.2 * scale).astype(np.float32)
    g = _lists(X, leaf_size=128, kappa=8, knn_mode=0, s_max=8, id_tol=0.0, h=scale, seed=4)
    ids, dist = g.knn_targets(torch.from_numpy(Y).cuda())
    oi, od = oracle.knn_exact(X, 8, Y=Y)
    assert np.array_equal(ids.cpu().numpy(), oi) and np.array_equal(dist.cpu().numpy(), od)
    g.close()
