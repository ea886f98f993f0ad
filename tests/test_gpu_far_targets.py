"""Out-of-sample targets far outside the data in FP16x3: their sums are zero (or the
oracle's), not infinite splits' NaN, and the other targets of the batch keep theirs --
global and per-sub-block centering, and d past the narrow kernels."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,centering,r", [(30, "auto", 1), (30, "auto", 6), (30, "block", 3), (100, "auto", 2)])
@pytest.mark.parametrize("far", [100.0, 1e7, 1e17])
def test_far_targets_are_finite(d, centering, r, far):
    import oracle
    from paper_1410_0260_gb300 import askit, workloads as wl
    N, T = 4000, 300
    X = wl.manifold(N, d, 4, 0.01, 1)
    Y = wl.manifold_queries(T, d, 4, 0.01, 1, 5)
    Y[11] = far
    Y[200, d - 1] = -far
    W = np.random.default_rng(3).standard_normal((N, r)).astype(np.float32)
    kw = dict(leaf_size=100, kappa=8, knn_mode=0, s_max=64, id_tol=1e-4, h=0.5)
    o = oracle.Tree(X, oracle.Config(**kw))
    o.set_weights(W.astype(np.float64))
    ref = o.evaluate_oos(Y)
    t = askit.Tree(torch.from_numpy(X).cuda(), askit.Config(precision="fp16x3", **kw))
    t.set_fp16_centering(centering)
    t.set_weights(torch.from_numpy(W).cuda())
    U = t.evaluate_targets(torch.from_numpy(Y).cuda()).cpu().numpy().reshape(T, r)
    t.sync()
    t.close()
    assert np.isfinite(U).all()
    assert np.all(U[[11, 200]] == 0) and np.all(np.abs(ref[[11, 200]]) < 1e-300)
    assert np.linalg.norm(U - ref) <= 1e-4 * np.linalg.norm(ref)      # the split-product tolerance
