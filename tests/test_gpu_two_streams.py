"""Weight contexts of one tree on two streams at once: launches that may start before the
kernel ahead of them has ended must still see that kernel's results, and neither stream
the other's."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,d,r", [("fp16x3", 24, 1), ("fp16x3", 24, 7), ("tf32x3", 24, 3), ("bf16x3", 24, 1),
                                           ("simt_fp32", 24, 2), ("fp16x3", 90, 4)])
def test_steps_on_two_streams_equal_the_serial_ones(precision, d, r):
    from paper_1410_0260_gb300 import askit, workloads as wl
    N = 6000
    t = askit.Tree(torch.from_numpy(wl.manifold(N, d, 4, 0.01, 1)).cuda(),
                   askit.Config(leaf_size=100, kappa=8, s_max=64, id_tol=1e-4, h=0.5, precision=precision))
    Y = torch.from_numpy(wl.manifold_queries(200, d, 4, 0.01, 1, 5)).cuda()
    W = [torch.from_numpy(np.random.default_rng(k).standard_normal((N, r)).astype(np.float32)).cuda() for k in range(6)]
    ctx = [t.weights_context(), t.weights_context()]
    want = []
    for w in W:
        ctx[0].set(w)
        want.append((ctx[0].evaluate().clone(), ctx[0].evaluate_targets(Y).clone()))
    ctx[1].set(W[0])
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    got = []
    for step in range(24):
        for k in range(2):                            # no waiting between the steps of either stream
            w = (step + 3 * k) % 6
            with torch.cuda.stream(streams[k]):
                ctx[k].set(W[w], stream=streams[k])
                got.append((w, 0, ctx[k].evaluate(stream=streams[k])))
                if step % 8 == 7:
                    got.append((w, 1, ctx[k].evaluate_targets(Y, stream=streams[k])))
    torch.cuda.synchronize()
    t.sync()
    for w, which, u in got:
        assert torch.equal(u, want[w][which]), (w, which)
    for c in ctx:
        c.close()
    t.close()
