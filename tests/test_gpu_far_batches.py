"""Batches of one weight context on two streams at once, one of them with a target outside
the FP16-safe range (another kernel, other column data): each equals its serial result."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r", [1, 3, 9])
def test_far_and_near_batches_at_once(r):
    from paper_1410_0260_gb300 import askit, workloads as wl
    N, d = 20000, 30
    t = askit.Tree(torch.from_numpy(wl.manifold(N, d, 4, 0.01, 1)).cuda(),
                   askit.Config(leaf_size=100, kappa=8, s_max=64, id_tol=1e-3, h=0.5, precision="fp16x3"))
    t.set_weights(torch.from_numpy(np.random.default_rng(2).standard_normal((N, r)).astype(np.float32)).cuda())
    near = torch.from_numpy(wl.manifold_queries(3000, d, 4, 0.01, 1, 5)).cuda()
    far = near.clone()
    far[11] = 1e7
    want = [t.evaluate_targets(y).clone() for y in (near, far)]
    errors = []

    def serve(k):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(150):
                    u = t.evaluate_targets((near, far)[k])
                    torch.cuda.current_stream().synchronize()
                    assert torch.equal(u, want[k]), k
        except Exception as e:
            errors.append(repr(e))

    threads = [threading.Thread(target=serve, args=(k,)) for k in range(2)]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    assert not errors, errors[0]
    t.sync()
    t.close()
