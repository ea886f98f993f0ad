"""Plain FP32 Evaluate in many dimensions: rounding of the squared distance does not
grow with d.  Two groups of equal points differ by 1.22 in every coordinate, so every
addition of a single chain of 3,000 would round the same way (700 units of 2^-24)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r", [1, 3, 5])
def test_distance_rounding_is_that_of_slices(r):
    from paper_1410_0260_gb300 import askit
    N, d, a = 64, 3000, np.float32(1.22)
    X = np.zeros((N, d), np.float32)
    X[1::2] = a
    W = np.zeros((N, r), np.float32)
    W[1::2] = 1.0                                        # the other group alone, seen from the even points
    D = d * float(a) ** 2
    h = np.float32(np.sqrt(D / 2))
    t = askit.Tree(torch.from_numpy(X).cuda(), askit.Config(leaf_size=32, kappa=1, prune=0, s_max=8, h=float(h),
                                                            precision="simt_fp32"))
    t.set_weights(torch.from_numpy(W).cuda())
    U = t.evaluate().cpu().numpy().reshape(N, r)[::2]
    t.close()
    want = N / 2 * np.exp(-D / (2 * float(h) ** 2))
    # 64 roundings a slice, one a slice, 3 of a difference and its scale, in an exponent
    # of 1; 8 for the scale and exp2f; N additions of the terms
    eps = (64 + (d + 63) // 64 + 3 + 8 + N) * 2.0 ** -24
    assert np.all(np.abs(U - want) <= eps * want)
