"""Exact neighbors of new points, bit for bit against the oracle, where the search's
tiles and lists end: N and T around the 256-row and 128-query tiles, kappa 1 and
32, both row widths (d_pad 32 and 64), one leaf, queries outside the FP16-safe
range, duplicates (ties by id) and points far from the origin."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,d,T,kappa,leaf,kind", [
    (255, 3, 1, 1, 300, "plain"),
    (257, 32, 127, 32, 64, "plain"),
    (1024, 33, 129, 7, 100, "duplicates"),
    (3000, 64, 300, 32, 128, "far_query"),
    (2500, 20, 200, 16, 90, "far_origin"),
    (5000, 8, 1000, 32, 40, "plain"),
    (300, 5, 2600, 9, 50, "far_query"),          # enough queries for eight a block
    (1200, 64, 2501, 32, 128, "duplicates"),
])
def test_knn_targets_match_the_oracle(N, d, T, kappa, leaf, kind):
    import oracle
    from paper_1410_0260_gb300 import askit
    rng = np.random.default_rng(N + d)
    X = rng.standard_normal((N, d)).astype(np.float32)
    Y = rng.standard_normal((T, d)).astype(np.float32)
    if kind == "duplicates":
        X[1::2] = X[::2]
        Y[:50] = X[:50]
    elif kind == "far_query":
        Y[::7] *= np.float32(1e6)
        Y[1::7] *= np.float32(40)
    elif kind == "far_origin":
        X += np.float32(300)
        Y += np.float32(300)
    t = askit.Tree(torch.from_numpy(X).cuda(), askit.Config(leaf_size=leaf, kappa=kappa, s_max=16, h=1.0))
    ids, dist = t.knn_targets(torch.from_numpy(Y).cuda())
    t.sync()
    oi, od = oracle.knn_exact(X, kappa, Y=Y)
    assert np.array_equal(ids.cpu().numpy(), oi)
    assert np.array_equal(dist.cpu().numpy(), od)
    t.close()


@pytest.mark.parametrize("d,kappa", [(5, 7), (40, 32)])
def test_many_queries_match_the_same_in_pieces(d, kappa):
    """From 2^31 (query, point) pairs on the queries are taken in the order of their
    home leaves; pieces below that are not.  The neighbors are exact either way."""
    from paper_1410_0260_gb300 import askit
    N, T, piece = 50001, 43001, 9001
    g = torch.Generator().manual_seed(d)
    X = torch.randn(N, d, generator=g)
    X[1:200:2] = X[0:200:2]
    Y = torch.randn(T, d, generator=g)
    Y[:100] = X[:100]
    Y[5::401] *= 1e6                 # the exhaustive search's rows go back to their own places
    Y = Y.cuda()
    t = askit.Tree(X.cuda(), askit.Config(leaf_size=200, kappa=kappa, s_max=16, h=1.0))
    ids, dist = t.knn_targets(Y)
    for a in range(0, T, piece):
        i, x = t.knn_targets(Y[a:a + piece].contiguous())
        assert torch.equal(ids[a:a + piece], i) and torch.equal(dist[a:a + piece], x)
    t.sync()
    t.close()
