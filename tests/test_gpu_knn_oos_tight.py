"""Exact neighbors of new points where the tensor-core shortlist's margin takes in more
candidates than a query keeps: tight clusters far from the data mean, equal points, one
leaf, a curve -- bit for bit, and not at the cost of the exhaustive search."""
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _tight(N, d, n, width, rng):
    mu = rng.uniform(-50, 50, (n, d))
    return lambda m: (mu[rng.integers(0, n, m)] + width * rng.standard_normal((m, d))).astype(np.float32)


@pytest.mark.parametrize("N,d,T,kappa,leaf,n,width", [
    (6000, 5, 300, 1, 100, 3, 1e-3),
    (6000, 33, 129, 32, 333, 2, 1e-2),
    (6001, 64, 200, 16, 128, 3, 1e-4),
    (4000, 7, 150, 9, 90, 2, 0.0),                   # equal points: ties by id past any list
    (2000, 20, 100, 8, 2000, 1, 1e-4),               # one leaf
    (9000, 3, 2700, 5, 64, 4, 1e-3),                 # enough queries for eight a block
])
def test_overflowing_queries_match_the_oracle(N, d, T, kappa, leaf, n, width):
    import oracle
    from paper_1410_0260_gb300 import askit
    rng = np.random.default_rng(N + d)
    draw = _tight(N, d, n, width, rng)
    X, Y = draw(N), draw(T)
    Y[::9] += np.float32(3)                          # some between the clusters
    Y[4::50] *= np.float32(1e6)                      # and some far outside the data
    t = askit.Tree(torch.from_numpy(X).cuda(), askit.Config(leaf_size=leaf, kappa=kappa, s_max=16, h=1.0))
    ids, dist = t.knn_targets(torch.from_numpy(Y).cuda())
    t.sync()
    oi, od = oracle.knn_exact(X, kappa, Y=Y)
    assert np.array_equal(ids.cpu().numpy(), oi)
    assert np.array_equal(dist.cpu().numpy(), od)
    t.close()


def test_sorted_overflowing_queries_match_the_same_in_pieces():
    """From 2^31 (query, point) pairs on the queries are taken in the order of their
    home leaves; pieces below that are not."""
    from paper_1410_0260_gb300 import askit
    rng = np.random.default_rng(2)
    draw = _tight(50001, 6, 20, 1e-3, rng)
    X, Y = draw(50001), draw(43001)
    Y[5::401] *= np.float32(1e6)
    Y = torch.from_numpy(Y).cuda()
    t = askit.Tree(torch.from_numpy(X).cuda(), askit.Config(leaf_size=200, kappa=7, s_max=16, h=1.0))
    ids, dist = t.knn_targets(Y)
    for a in range(0, 43001, 9001):
        i, x = t.knn_targets(Y[a:a + 9001].contiguous())
        assert torch.equal(ids[a:a + 9001], i) and torch.equal(dist[a:a + 9001], x)
    t.sync()
    t.close()


def test_overflowing_queries_do_not_cost_the_exhaustive_search():
    """Against the exhaustive search of as many of the tree's own points, on a curve and on
    tight clusters: a small part of its time (a half would already be the fallback)."""
    from paper_1410_0260_gb300 import askit, workloads as wl
    for X in (wl.curve(1 << 20, 3, 1), _tight(0, 16, 64, 0.1, np.random.default_rng(1))(131072)):
        t = askit.Tree(torch.from_numpy(X).cuda(), askit.Config(leaf_size=512, kappa=16, knn_mode=1, rp_iters=2, s_max=16,
                                                                id_tol=1e-3, h=0.3))
        rows = torch.arange(0, 3001, dtype=torch.int32, device="cuda") * (len(X) // 3001)
        Y = torch.from_numpy(X).cuda()[rows.long()] + 1e-4

        def best(f):
            took = []
            for _ in range(4):
                torch.cuda.synchronize()
                t0 = time.perf_counter()
                f()
                torch.cuda.synchronize()
                took.append(time.perf_counter() - t0)
            return min(took[1:])

        a, b = best(lambda: t.knn_targets(Y)), best(lambda: t.knn_points(rows))
        t.close()
        assert a < 0.5 * b, (a, b)


@pytest.mark.parametrize("T", [300, 15001])
def test_queries_without_a_bound_match_the_oracle(T):
    """Home leaves of fewer than kappa points bound nothing: few such queries scan the
    leaves, many take the exhaustive search."""
    import oracle
    from paper_1410_0260_gb300 import askit
    rng = np.random.default_rng(T)
    X = rng.standard_normal((3000, 5)).astype(np.float32)
    X[1:50:2] = X[0:49:2]
    Y = rng.standard_normal((T, 5)).astype(np.float32)
    t = askit.Tree(torch.from_numpy(X).cuda(), askit.Config(leaf_size=8, kappa=32, s_max=8, h=1.0))
    ids, dist = t.knn_targets(torch.from_numpy(Y).cuda())
    t.sync()
    t.close()
    oi, od = oracle.knn_exact(X, 32, Y=Y)
    assert np.array_equal(ids.cpu().numpy(), oi)
    assert np.array_equal(dist.cpu().numpy(), od)
