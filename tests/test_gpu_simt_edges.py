"""Plain FP32 Evaluate with pruning off (the direct sum) against FP64 where its
tiles end: coordinates around a slice of 64, leaves around 128 rows, and every
vector class."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,d,leaf,r", [(1, 1, 2, 1), (130, 1, 129, 1), (257, 31, 128, 4), (300, 64, 100, 5),
                                        (513, 65, 257, 2), (400, 130, 64, 17), (200, 40, 33, 64)])
def test_direct_sum_matches_fp64(N, d, leaf, r):
    from paper_1410_0260_gb300 import askit
    rng = np.random.default_rng(N + d)
    N = max(N, 2)
    X = rng.standard_normal((N, d)).astype(np.float32)
    W = rng.standard_normal((N, r)).astype(np.float32)
    h = np.float32(1.1 * np.sqrt(d))
    t = askit.Tree(torch.from_numpy(X).cuda(), askit.Config(leaf_size=leaf, kappa=1, prune=0, s_max=8, h=float(h),
                                                            precision="simt_fp32"))
    t.set_weights(torch.from_numpy(W).cuda())
    U = t.evaluate().cpu().numpy()
    X64 = X.astype(np.float64)
    D = ((X64[:, None] - X64[None]) ** 2).sum(2)
    K = np.exp(-D / (2 * float(h) ** 2))
    # d + 2 roundings of the distance move the exponent (at most 2 here) by (d + 3) ulp
    # of itself, exp2f and the scale a few more; N additions of the terms' sum
    eps = (3 * (d + 3) + 8 + N) * 2.0 ** -24
    assert np.all(np.abs(U - K @ W) <= eps * (K @ np.abs(W)) + 1e-30)
    # a weight vector's sum does not depend on how many others share the evaluation
    t.set_weights(torch.from_numpy(np.ascontiguousarray(W[:, r - 1:])).cuda())
    assert np.array_equal(t.evaluate().cpu().numpy()[:, 0], U[:, r - 1])
    t.close()

