"""Autotuning one precision leaves what it does not vary -- stages, pairs -- at the
automatic choices of the tree's other precisions: FP16x3 launches the same kernel
variant before and after."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _kernels(f):
    from torch.profiler import ProfilerActivity, profile
    for _ in range(5):                               # a process's first session may record nothing
        with profile(activities=[ProfilerActivity.CUDA]) as p:
            f()
            torch.cuda.synchronize()
        names = sorted({e.key for e in p.key_averages() if "eval_g16_kernel" in e.key or "eval_tcw_kernel" in e.key})
        if names:
            break
    return names


@pytest.mark.parametrize("d,precision,r", [(16, "simt_fp32", 1), (16, "tf32x3", 1), (16, "bf16x3", 1), (16, "fp16x3", 6),
                                           (72, "simt_fp32", 1)])
def test_other_precisions_keep_their_variant(d, precision, r):
    from paper_1410_0260_gb300 import askit, workloads as wl
    N = 8000
    t = askit.Tree(torch.from_numpy(wl.manifold(N, d, 4, 0.01, 1)).cuda(),
                   askit.Config(leaf_size=256, kappa=8, s_max=256, id_tol=0.0, h=0.6, precision="fp16x3"))
    W = torch.from_numpy(np.random.default_rng(1).standard_normal((N, r)).astype(np.float32)).cuda()
    w1 = W[:, :1].contiguous()
    t.set_weights(w1)
    before = _kernels(t.evaluate)
    assert len(before) == 1, before
    t.set_precision(precision)
    t.set_weights(W)
    t.autotune(reps=1)
    t.set_precision("fp16x3")
    t.set_weights(w1)
    if precision != "fp16x3":
        assert _kernels(t.evaluate) == before
    else:                                            # r > 4 tunes the stages, not the pairs
        assert [k.split(",")[2] for k in _kernels(t.evaluate)] == [k.split(",")[2] for k in before]
    t.close()
