"""The default launch (paired items where most have a partner, runs sized to the
work) gives what the plain unpaired launch gives, in and out of sample, at sizes
with all, some and no pairs and with fewer items than SMs."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,d,leaf,s_max,r", [
    (300, 6, 100, 20, 1),       # no pairs, a handful of items
    (5000, 24, 256, 256, 1),    # every block paired
    (5000, 24, 256, 100, 4),    # leaves paired, skeletons single
    (9001, 12, 640, 384, 3),    # odd numbers of sub-blocks a node
    (3000, 72, 256, 200, 1),    # wide rows
])
def test_default_launch_matches_the_unpaired_one(N, d, leaf, s_max, r):
    from paper_1410_0260_gb300 import askit, workloads as wl
    X = torch.from_numpy(wl.manifold(N, d, 4, 0.01, seed=N)).cuda()
    Y = torch.from_numpy(wl.manifold_queries(150, d, 4, 0.01, N, 9)).cuda()
    t = askit.Tree(X, askit.Config(leaf_size=leaf, kappa=8, s_max=s_max, id_tol=0.0, h=0.6, precision="fp16x3"))
    t.set_weights(torch.from_numpy(np.random.default_rng(3).standard_normal((N, r)).astype(np.float32)).cuda())
    U, V = t.evaluate().clone(), t.evaluate_targets(Y).clone()
    t.set_launch("lpt", 3, True, False)
    for a, b in ((U, t.evaluate()), (V, t.evaluate_targets(Y))):
        # each entry's partial sum is formed the same way in both layouts
        assert torch.equal(a, b), float((a - b).norm() / b.norm())
    t.sync()
    t.close()
