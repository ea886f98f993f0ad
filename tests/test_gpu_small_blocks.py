"""Small out-of-sample batches: most source sub-blocks have a single work item,
so a kernel's loader groups have blocks without an item of theirs."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# the split-product tolerance of every tensor-core precision, the plain FP32 one
TOL = {"simt_fp32": 1e-5, "tf32x3": 1e-4, "bf16x3": 1e-4, "fp16x3": 1e-4}


@pytest.mark.parametrize("r", [1, 3])
@pytest.mark.parametrize("T", [40, 300])
def test_small_target_batches_match_the_oracle(T, r):
    import oracle
    from paper_1410_0260_gb300 import askit, workloads as wl
    X = wl.manifold(6000, 60, 4, 0.01, seed=3)
    Y = wl.manifold_queries(T, 60, 4, 0.01, 3, 17)
    W = np.random.default_rng(5).standard_normal((6000, r)).astype(np.float32)
    kw = dict(leaf_size=200, kappa=8, knn_mode=0, s_max=64, id_tol=1e-4, h=0.5, seed=1)
    o = oracle.Tree(X, oracle.Config(**kw))
    o.set_weights(W.astype(np.float64))
    ref = o.evaluate_oos(Y)
    g = askit.Tree(torch.from_numpy(X).cuda(), askit.Config(**kw))
    g.set_weights(torch.from_numpy(W).cuda())
    Yd = torch.from_numpy(Y).cuda()
    for prec, tol in TOL.items():
        g.set_precision(prec)
        for _ in range(3):
            U = g.evaluate_targets(Yd).cpu().numpy()
            g.sync()
            assert np.linalg.norm(U - ref) <= tol * np.linalg.norm(ref), prec
    g.close()
