"""Evaluate where nodes straddle separated clusters (a number of them that is no power
of two, so that median splits leave leaves and skeletons with parts of two): the
squared distances of near points must not cancel around a center far from both."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# the split-product tolerance, and the plain FP32 one
TOL = {"tf32x3": 1e-4, "simt_fp32": 1e-5}


@pytest.mark.parametrize("N,d,box,seed,leaf,varh,h,r", [
    (4096, 4, 100, 1, 128, False, 1.0, 1),      # one bandwidth, one vector: the compact column data
    (4096, 4, 100, 1, 128, False, 1.0, 3),
    (4096, 4, 100, 1, 128, False, 1.0, 16),
    (4096, 4, 60, 1, 128, True, 1.0, 1),        # a bandwidth a point
    (3000, 10, 100, 5, 300, False, 2.0, 3),     # leaves of more than one sub-block
])
def test_separated_clusters_match_the_oracle(N, d, box, seed, leaf, varh, h, r):
    import oracle
    from paper_1410_0260_gb300 import askit
    rng = np.random.default_rng(seed)
    mu = rng.uniform(-box / 2, box / 2, (3, d))
    X = (mu[rng.integers(0, 3, N)] + rng.standard_normal((N, d))).astype(np.float32)
    Y = (mu[rng.integers(0, 3, 777)] + rng.standard_normal((777, d))).astype(np.float32)
    W = np.random.default_rng(7).standard_normal((N, r)).astype(np.float32)
    kw = dict(leaf_size=leaf, kappa=16, knn_mode=0, s_max=leaf // 2, id_tol=1e-5, h=h,
              bw_mode=askit.BW_KNN if varh else askit.BW_CONSTANT, bw_k=16)
    o = oracle.Tree(X, oracle.Config(**kw))
    o.set_weights(W.astype(np.float64))
    g = askit.Tree(torch.from_numpy(X).cuda(), askit.Config(**kw))
    g.set_weights(torch.from_numpy(W).cuda())
    Yd = torch.from_numpy(Y).cuda()
    ref, ref_y = o.evaluate(), o.evaluate_oos(Y)
    for prec, tol in TOL.items():
        g.set_precision(prec)
        for got, want in ((g.evaluate(), ref), (g.evaluate_targets(Yd), ref_y)):
            U = got.cpu().numpy().reshape(want.shape)
            g.sync()
            assert np.linalg.norm(U - want) <= tol * np.linalg.norm(want), prec
    g.close()
