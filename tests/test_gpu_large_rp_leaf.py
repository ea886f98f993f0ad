"""Random-projection lists with a leaf of more than 65,535 blocks of 64 queries (the
second grid dimension's limit): on a line of integers the nearest neighbor of every
point is known."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_one_leaf_of_more_than_4194240_points():
    from paper_1410_0260_gb300 import askit
    N = 65535 * 64 + 100
    val = np.random.default_rng(1).permutation(N)            # point i lies at val[i]
    t = askit.Tree(torch.from_numpy(val.astype(np.float32)[:, None]).cuda(),
                   askit.Config(leaf_size=2048, kappa=1, knn_mode=1, rp_iters=1, rp_leaf=N, s_max=2, h=1000.0))
    ids, dist = t.structure(askit.STRUCT_KNN).ravel(), t.structure(askit.STRUCT_KNN_DIST).ravel()
    t.close()
    at = np.empty(N, np.int64)
    at[val] = np.arange(N)                                   # the point at each integer
    left = np.where(val > 0, at[np.maximum(val - 1, 0)], N)
    right = np.where(val < N - 1, at[np.minimum(val + 1, N - 1)], N)
    assert np.array_equal(ids, np.minimum(left, right))      # both at distance 1: the smaller id
    assert np.all(dist == 1.0)
