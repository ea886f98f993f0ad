"""Memory of the out-of-sample calls: what a tree keeps for the next call is counted in
its device bytes, and the admission estimate covers what a call takes."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _tree(N, d, kappa, r):
    from paper_1410_0260_gb300 import askit, workloads as wl
    t = askit.Tree(torch.from_numpy(wl.manifold(N, d, 4, 0.01, 1)).cuda(),
                   askit.Config(leaf_size=256, kappa=kappa, s_max=64, id_tol=1e-3, h=0.5, precision="fp16x3"))
    t.set_weights(torch.randn(N, r, device="cuda"))
    return t


@pytest.mark.parametrize("N,d,kappa,r,T", [(20000, 8, 8, 1, 30000), (20000, 64, 32, 1, 3001), (9000, 33, 16, 16, 20000),
                                           (5000, 100, 16, 2, 9000)])
def test_kept_memory_is_counted_and_estimated(N, d, kappa, r, T):
    from paper_1410_0260_gb300 import workloads as wl
    _tree(2000, d, kappa, r).evaluate_targets(torch.randn(300, d, device="cuda"))      # modules loaded
    t = _tree(N, d, kappa, r)
    t.evaluate()
    Y = torch.from_numpy(wl.manifold_queries(T, d, 4, 0.01, 1, 5)).cuda()
    U = torch.empty(T, r, device="cuda")
    torch.cuda.synchronize()
    before, free = t.info()["device_bytes"], torch.cuda.mem_get_info()[0]
    U.copy_(t.evaluate_targets(Y))
    torch.cuda.synchronize()
    kept, gone = t.info()["device_bytes"] - before, free - torch.cuda.mem_get_info()[0]
    slack = 64 << 20                     # the pool's and the caching allocator's granularity
    assert kept > 0
    assert gone <= kept + slack
    assert kept <= t.footprint(1, T, r) + slack
    t.close()
