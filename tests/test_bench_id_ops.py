"""The FP64 operation count of the interpolative decomposition that bench.py reports,
against a step-by-step count of what the factorization issues."""
import types

import numpy as np

import bench
from paper_1410_0260_gb300 import askit


def test_id_operation_count():
    N, d, s_max, L = 400, 5, 12, 2
    s = np.array([0, 0, 12, 12, 12, 9, 12, 12])
    c = np.array([0, 0, 24, 21, 100, 100, 100, 100])
    tree = types.SimpleNamespace(structure=lambda k: s if k == askit.STRUCT_SKEL_S else c, info=lambda: {"L": L})
    got = bench._id_fp64_cost(tree, types.SimpleNamespace(N=N, d=d, s_max=s_max), 2.0)
    want = 0
    for a in range(2, 8):
        ell = min(s_max + 20, N - N // (1 << (a.bit_length() - 1)))
        for k in range(min(s[a] + 1, ell, c[a])):
            norms = c[a] if k == 0 else 1                          # columns whose exact norm is formed
            want += 2 * (ell - k) * norms                          # product and sum an element
            want += 4 * (ell - k) * max(c[a] - k - 1, 0)           # dot product and update
        want += s[a] * s[a] * (c[a] - s[a]) + ell * c[a] * (3 * d + 30)
    assert got["id_fp64_ops"] == want
    assert got["id_fp64_instr_per_s"] == want / 2.0
