"""Coordinates that are no number or infinite have no neighbors at a finite distance:
setup and out-of-sample Evaluate return an error instead of indexing by unfilled
lists, and the tree serves later calls."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("d,knn_mode", [(6, 0), (6, 1), (70, 0)])
def test_not_finite_is_refused(bad, d, knn_mode):
    from paper_1410_0260_gb300 import askit
    rng = np.random.default_rng(1)
    X = rng.standard_normal((500, d)).astype(np.float32)
    cfg = askit.Config(leaf_size=64, kappa=8, knn_mode=knn_mode, s_max=16, h=1.0)
    Xb = X.copy()
    Xb[77, d - 1] = bad
    with pytest.raises(askit.AskitError, match="not finite"):
        askit.Tree(torch.from_numpy(Xb).cuda(), cfg)
    t = askit.Tree(torch.from_numpy(X).cuda(), cfg)
    t.set_weights(torch.from_numpy(rng.standard_normal((500, 1)).astype(np.float32)).cuda())
    Y = torch.from_numpy(rng.standard_normal((90, d)).astype(np.float32)).cuda()
    Yb = Y.clone()
    Yb[41, 0] = bad
    for prec in ("fp16x3", "simt_fp32"):
        t.set_precision(prec)
        good = t.evaluate_targets(Y).clone()
        with pytest.raises(askit.AskitError, match="not finite"):
            t.evaluate_targets(Yb)
        assert torch.equal(t.evaluate_targets(Y), good)
    t.sync()
    t.close()
