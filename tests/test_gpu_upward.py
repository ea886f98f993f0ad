"""Skeleton weights of the upward pass against an FP64 pass over the oracle's
interpolation matrices, at the sizes where its kernel's tiling ends: ranks and
column counts that are no multiple of 4, more than one staged chunk of 1024
columns, one row, and every vector-count class."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,leaf,s_max,tol,r", [
    (1000, 40, 33, 0.0, 1),         # odd leaves, nr = 7 .. 33
    (1500, 64, 64, 1e-2, 3),        # adaptive ranks: ragged columns
    (2400, 1200, 20, 0.0, 5),       # 1180 remaining columns: two staged chunks
    (2400, 1200, 300, 0.0, 16),     # rows past one block's, 900 columns
    (900, 100, 1, 0.0, 17),         # one row a node, vectors past one group of 16
    (700, 50, 50, 0.0, 4),          # full rank at the leaves: nothing remains
])
def test_upward_pass_matches_fp64(N, leaf, s_max, tol, r):
    import oracle
    from paper_1410_0260_gb300 import askit
    rng = np.random.default_rng(N + r)
    X = rng.standard_normal((N, 5)).astype(np.float32)
    W = rng.standard_normal((N, r)).astype(np.float32)
    kw = dict(leaf_size=leaf, kappa=8, knn_mode=0, s_max=s_max, id_tol=tol, h=1.0, seed=1)
    g = askit.Tree(torch.from_numpy(X).cuda(), askit.Config(precision="simt_fp32", **kw))
    o = oracle.Tree(X, oracle.Config(**kw))
    g.set_weights(torch.from_numpy(W).cuda())
    got = g.structure(askit.STRUCT_WSKEL).astype(np.float64)
    nn, first = o.nnodes, o.nnodes // 2
    wsk, bound = {}, {}             # FP64 skeleton weights, and the sums of |terms| that bound the rounding
    for a in range(nn - 1, 1, -1):
        nd = o.node(a)
        if a >= first:
            v = W[nd["cols"]].astype(np.float64)
            b = np.abs(v)
        else:
            v = np.concatenate([wsk[2 * a], wsk[2 * a + 1]])
            b = np.concatenate([bound[2 * a], bound[2 * a + 1]])
        s = len(nd["skel"])
        P = nd["P"].reshape(s, -1)
        piv = nd["piv"]
        wsk[a] = v[piv[:s]] + P @ v[piv[s:]]
        bound[a] = b[piv[:s]] + np.abs(P) @ b[piv[s:]]
    off = 0
    for a in range(2, nn):
        s = len(wsk[a])
        # a level rounds P, and adds at most 2 (columns / 32 + 8) rounded terms;
        # errors of the levels below pass through |P| like the bound itself
        eps = o.L * (leaf / 16 + 2 * s_max / 16 + 20) * 2.0 ** -24
        err = np.abs(got[off: off + s] - wsk[a])
        assert np.all(err <= eps * bound[a] + 1e-30), (a, float((err / bound[a]).max()))
        off += s
    assert off == len(got)
    g.close()
