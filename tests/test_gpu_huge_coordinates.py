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
