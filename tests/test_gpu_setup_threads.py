"""Trees built by two threads at once, whose factorizations need little shared memory
and more than the 48 KB that a kernel has to ask for."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_two_threads_build_trees_of_different_sizes():
    from paper_1410_0260_gb300 import askit
    X = torch.from_numpy(np.random.default_rng(1).standard_normal((60000, 3)).astype(np.float32)).cuda()
    small = (X[:3000].contiguous(), askit.Config(leaf_size=20, kappa=4, s_max=4, ell_extra=4, id_tol=1e-1, h=1.0))
    large = (X, askit.Config(leaf_size=1900, kappa=4, s_max=4, ell_extra=6200, id_tol=1e-1, h=1.0))

    def skeletons(args):
        t = askit.Tree(*args)
        ids = t.structure(askit.STRUCT_SKEL_IDS)
        t.close()
        return ids

    want = [skeletons(small), skeletons(large)]
    errors, done = [], threading.Event()

    def build(k):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                n = 0
                while n < 3 if k else not done.is_set():
                    assert np.array_equal(skeletons((small, large)[k]), want[k])
                    n += 1
        except Exception as e:
            errors.append(repr(e))
        if k:
            done.set()

    threads = [threading.Thread(target=build, args=(k,)) for k in range(2)]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    assert not errors, errors[0]
