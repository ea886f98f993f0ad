"""The work a user of this framework has it do, as cases that can be timed.

Every case goes through the public binding (`askit.Tree`, its weight, target, host and
graph calls).  Points follow the repository's recipes: a mixture of Gaussians, or a
low-dimensional manifold embedded in d dimensions with a little noise, drawn on the GPU
from the seed alone.

`op` says what one pass is:

* ``weights``  new weight vectors on a resident tree: upward pass and Evaluate;
* ``graph``    the same step captured once as a CUDA graph and replayed (autotuned);
* ``host``     the same step from and to pinned host buffers;
* ``targets``  a batch of out-of-sample targets against resident weights;
* ``build``    a tree from its points (kNN, tree, skeletons, work lists), and one step.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1410_0260_gb300 import askit

DEV = "cuda:0"


def _case(name, op, N, d, k, h, m, kappa, s_max, tol, r=1, T=0, prec="fp16x3", points="manifold", noise=0.01,
          law="normal", varh=False, s_min=1, rp=6):
    c = dict(op=op, N=N, d=d, k=k, h=h, m=m, kappa=kappa, s_max=s_max, tol=tol, r=r, T=T, prec=prec, points=points,
             noise=noise, law=law, varh=varh, s_min=s_min, rp=rp)
    return dict(c, name=name) if name else c


def listed():
    serve = dict(d=64, k=8, h=0.4, m=512, kappa=32, s_max=256, tol=1e-4)
    m6 = dict(d=64, k=6, h=0.35, m=512, kappa=32, s_max=256, tol=1e-4)
    return [
        # one small problem solved again and again for new weights: launches and latency count
        _case("weights_4k_d8", "weights", 4096, 8, 0, 1.0, 128, 16, 64, 1e-6, points="mixture", rp=0),
        # the benchmark's step at full size: an iterative solver that replays one captured step
        _case("graph_1m_d64", "graph", 1 << 20, **m6),
        # many right-hand sides at once (multi-vector regression), large leaves and skeletons
        _case("weights_65k_r16", "weights", 65536, 64, 10, 0.5, 1024, 32, 512, 1e-4, r=16, law="uniform"),
        # a serving request of a few weight vectors on a tree of odd size
        _case("weights_50003_r3", "weights", 50003, r=3, **serve),
        # high-dimensional points with a bandwidth per point, skeleton ranks chosen by tolerance
        _case("weights_10007_d1000", "weights", 10007, 1000, 12, 1.0, 256, 16, 1024, 1e-3, noise=0.001, varh=True,
              s_min=32, rp=4),
        # the default precision of a Config
        _case("weights_65k_tf32x3", "weights", 65536, prec="tf32x3", **m6),
        # plain FP32, what the split precisions are judged against
        _case("weights_65k_fp32", "weights", 65536, prec="simt_fp32", **m6),
        # out-of-sample requests against a resident tree: small, ordinary (odd size), large
        _case("targets_100", "targets", 65536, T=100, **serve),
        _case("targets_3001", "targets", 131072, T=3001, **serve),
        _case("targets_100000", "targets", 131072, T=100000, **serve),
        # a new data set: everything from its points to the first result
        _case("build_65k_d64", "build", 65536, **m6),
        # the step with its inputs and results on the host
        _case("host_65k_d64", "host", 65536, **m6),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["weights", "weights", "weights", "targets", "targets", "build", "graph", "host"])
    wide = op in ("weights", "targets") and rng.random() < 0.15
    N = _log(rng, 2000, 12000 if wide else 40000)
    d = _log(rng, 65, 1000) if wide else _log(rng, 3, 64)
    m = rng.choice([128, 256, 512])
    points = "mixture" if d <= 16 and rng.random() < 0.5 else "manifold"
    prec = "fp16x3" if op == "graph" or rng.random() < 0.6 else rng.choice(
        ["bf16x3", "simt_fp32"] if wide else ["tf32x3", "simt_fp32"])
    return _case("", op, N, d, min(d, rng.randint(2, 12)), 1.0 if points == "mixture" else round(rng.uniform(0.3, 0.8), 3),
                 m, rng.choice([16, 32]), rng.choice([64, m // 2, m]), rng.choice([1e-3, 1e-4]),
                 r=1 if rng.random() < 0.5 else rng.randint(2, 16), T=_log(rng, 10, 100000) if op == "targets" else 0,
                 prec=prec, points=points, law=rng.choice(["normal", "uniform"]), varh=rng.random() < 0.15,
                 rp=rng.choice([0, 4, 6]) if N <= 32768 else 6)


# ---------------------------------------------------------------------------------- inputs
def _inputs(c, seed):
    """Points X, weights W and out-of-sample targets Y of the same distribution (FP32)."""
    g = torch.Generator(device=DEV).manual_seed(seed)

    def normal(*shape):
        return torch.randn(*shape, generator=g, device=DEV, dtype=torch.float64)

    def uniform(*shape):
        return torch.rand(*shape, generator=g, device=DEV, dtype=torch.float64)

    if c["points"] == "mixture":
        means = uniform(4, c["d"]) * 10 - 5
    else:
        means = torch.linalg.qr(normal(c["d"], c["k"]).cpu())[0].to(DEV)

    def points(n):
        if c["points"] == "mixture":
            return (means[(uniform(n) * 4).long().clamp_(max=3)] + normal(n, c["d"])).float()
        return (normal(n, c["k"]) @ means.T + c["noise"] * normal(n, c["d"])).float()

    X = points(c["N"])
    W = (normal(c["N"], c["r"]) if c["law"] == "normal" else uniform(c["N"], c["r"]) * 2 - 1).float()
    return X, W, points(c["T"]) if c["T"] else None


def _config(c):
    return askit.Config(leaf_size=c["m"], kappa=c["kappa"], knn_mode=1 if c["rp"] else 0, rp_iters=c["rp"] or 4,
                        s_max=c["s_max"], s_min=c["s_min"], bw_mode=askit.BW_KNN if c["varh"] else askit.BW_CONSTANT,
                        bw_k=min(16, c["kappa"]), precision=c["prec"], id_tol=c["tol"], h=c["h"], seed=1)


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.c, s.cfg = case, _config(case)
    s.X, s.W, s.Y = _inputs(case, seed)
    if case["op"] == "build":
        return s
    s.tree = askit.Tree(s.X, s.cfg)
    if case["op"] == "graph":
        s.tree.set_weights(s.W)
        s.tree.autotune()
        s.U = torch.empty_like(s.W)
        s.graph = s.tree.capture(s.W, s.U)
    elif case["op"] == "targets":
        s.tree.set_weights(s.W)
    elif case["op"] == "host":
        s.W_host = s.W.cpu().pin_memory().numpy()
        s.U_host = torch.empty(s.W.shape, dtype=torch.float32, pin_memory=True).numpy()
    return s


def run(s):
    op = s.c["op"]
    if op == "weights":
        s.tree.set_weights(s.W)
        return s.tree.evaluate()
    if op == "graph":
        s.graph.launch()
        return s.U
    if op == "host":
        return s.tree.evaluate_host(s.W_host, out=s.U_host)
    if op == "targets":
        return s.tree.evaluate_targets(s.Y)
    tree = askit.Tree(s.X, s.cfg)
    tree.set_weights(s.W)
    out = {"u": tree.evaluate(), "perm": tree.structure(askit.STRUCT_PERM)}
    tree.close()
    return out


# ------------------------------------------------------------------------------------ work
def _depth(N, m):
    L = 0
    while -(-N >> L) > m:
        L += 1
    return L


def work(case):
    """The kernel evaluations follow the tree, which only the points fix: near leaves and far
    nodes per target are those the recipes measure (6 intrinsic dimensions: 5.5 near and 7.7
    far at 5 levels, half a leaf and 3.7 nodes more for every level), in proportion to the
    intrinsic dimension."""
    N, d, r, m, T = case["N"], case["d"], case["r"], case["m"], case["T"]
    L = _depth(N, m)
    f = (case["k"] or 4) / 6
    near = min(2.0 ** L, max(1.0, f * (5.5 + 0.5 * (L - 5))))
    far = min(2.0 ** L - near, max(0.0, f * (7.7 + 3.65 * (L - 5)))) if L else 0.0
    leaf = N / 2 ** L
    s = min(case["s_max"], leaf)
    nodes = (2 << L) - 2
    pairs = near * leaf + far * s
    t = T if case["op"] == "targets" else N
    flops = t * pairs * (2 * d + 2 * r)                     # one distance product and the weight sums
    skeletons = nodes * s * (d + r) * 4.0
    if case["op"] == "targets":
        return {"bytes": 4.0 * (N * (d + r) + T * (d + r)) + skeletons, "flops": flops}
    upward = nodes * s * s * 4.0                            # interpolation matrices, read once
    flops += nodes * s * s * 2 * r
    if case["op"] == "build":
        ell = s + 20
        flops += nodes * (ell * 2 * s * s * 4 + ell * 2 * s * 2 * d)   # pivoted QR and its kernel block
        flops += max(1, case["rp"]) * N * (max(2 * case["kappa"] + 2, m) if case["rp"] else N) * 2.0 * d
    return {"bytes": 4.0 * N * (d + 2 * r) + skeletons + upward, "flops": flops}


# ----------------------------------------------------------------- the same in 64 bits (torch)
# The method restated (March, Xiao & Biros, arXiv:1410.0260) with the same readings as the
# framework documents: level-wise median splits, random-projection kNN, node neighbor lists,
# sampled rows, column-pivoted QR with recomputed norms, then Evaluate over Near and Far.
def _philox(k1, c0, n, seed):
    """The first n words of the counter-based stream keyed (seed, k1), blocks (c0, 0), (c0, 1), ..."""
    out = []
    for b in range(-(-n // 4)):
        gen = np.random.Philox(key=seed | (k1 << 64), counter=(c0 + (b << 64) - 1) % (1 << 256))
        out.append(gen.random_raw(4))
    return np.concatenate(out)[:n]


def _tree(X, L, key):
    """Leaves of a tree of depth L in order, as ascending id arrays; key(points' ids, node)."""
    level = [torch.arange(X.shape[0], device=DEV)]
    for t in range(L):
        nxt = []
        for g, ids in enumerate(level):
            o = ids[torch.sort(key(ids, (1 << t) + g), stable=True)[1]]
            half = (len(ids) + 1) // 2
            nxt += [o[:half].sort()[0], o[half:].sort()[0]]
        level = nxt
    return level


def _d2(A, B):
    out = torch.empty(A.shape[0], B.shape[0], dtype=torch.float64, device=DEV)
    step = max(1, (1 << 27) // max(1, B.shape[0] * B.shape[1]))
    for a in range(0, A.shape[0], step):
        out[a:a + step] = (A[a:a + step, None, :] - B[None]).square_().sum(2)
    return out


def _nearest(D, ids, kappa):
    """The kappa smallest by (distance, id) of candidates whose ids ascend along the rows."""
    v, o = torch.sort(D, dim=1, stable=True)
    return v[:, :kappa], ids[o[:, :kappa]]


def _knn(X, c):
    N, kappa = X.shape[0], c["kappa"]
    if not c["rp"]:
        step = max(1, (1 << 25) // N)
        all_ids = torch.arange(N, device=DEV)
        got = []
        for a in range(0, N, step):
            D = _d2(X[a:a + step], X)
            D[torch.arange(D.shape[0]), torch.arange(a, a + D.shape[0])] = math.inf
            got.append(_nearest(D, all_ids, kappa))
        return torch.cat([g[0] for g in got]), torch.cat([g[1] for g in got])
    L, dists, ids = _depth(N, max(2 * kappa + 2, c["m"])), [], []
    for it in range(c["rp"]):
        def key(p, node):
            bits = _philox(it + 1, node, -(-c["d"] // 64), 1).view(np.uint8)
            sign = np.unpackbits(bits, bitorder="little")[:c["d"]].astype(np.float64) * -2 + 1
            return X[p] @ torch.from_numpy(sign).to(DEV)
        dd = torch.empty(N, kappa, dtype=torch.float64, device=DEV)
        ii = torch.empty(N, kappa, dtype=torch.int64, device=DEV)
        for leaf in _tree(X, L, key):
            D = _d2(X[leaf], X[leaf])
            D.fill_diagonal_(math.inf)
            dd[leaf], ii[leaf] = _nearest(D, leaf, kappa)
        dists.append(dd)
        ids.append(ii)
    ii, o = torch.sort(torch.cat(ids, 1), dim=1, stable=True)
    dd = torch.cat(dists, 1).gather(1, o)
    dd[:, 1:][ii[:, 1:] == ii[:, :-1]] = math.inf
    dd, o = torch.sort(dd, dim=1, stable=True)
    return dd[:, :kappa], ii.gather(1, o)[:, :kappa]


def _id(A, ncol, tol, s_lo, s_hi):
    """Pivoted Householder QR of a batch [B, ell, c] (zero columns past ncol): R, pivots, ranks."""
    B, rows, cols = A.shape
    at = torch.arange(B, device=DEV)
    piv = torch.arange(cols, device=DEV).repeat(B, 1)
    rank = torch.minimum(ncol, torch.tensor(min(s_hi, rows), device=DEV))
    cap, low = rank.clone(), torch.minimum(ncol, torch.tensor(s_lo, device=DEV))
    done = torch.zeros(B, dtype=torch.bool, device=DEV)
    r00 = None
    for k in range(min(s_hi, rows, cols)):
        norms = A[:, k:, k:].square().sum(1)
        best, p = norms.max(1)
        p = p + k
        nrm = best.sqrt()
        r00 = nrm if r00 is None else r00
        stop = ~done & ((nrm == 0) | ((k >= low) & (nrm <= tol * r00)))
        rank = torch.where(stop, torch.minimum(cap, torch.tensor(k, device=DEV)), rank)
        done |= stop | (cap <= k + 1)
        for M in (A.transpose(1, 2), piv):
            x, y = M[:, k].clone(), M[at, p].clone()
            M[:, k] = y
            M[at, p] = x
        alpha = A[:, k, k].clone()
        beta = torch.where(alpha >= 0, -nrm, nrm)
        safe = torch.where(beta == 0, torch.ones_like(beta), beta)
        v = A[:, k:, k] / torch.where(alpha - beta == 0, torch.ones_like(beta), alpha - beta)[:, None]
        v[:, 0] = 1
        A[:, k:, k + 1:] -= ((beta - alpha) / safe)[:, None, None] * v[:, :, None] * (v[:, None, :] @ A[:, k:, k + 1:])
        A[:, k:, k] = 0
        A[:, k, k] = beta
        if bool(done.all()):
            break
    return A, piv, rank


def exact(case, seed):
    c = case
    # a restatement in torch operations: only while it takes seconds
    if c["N"] > 140000 or (c["d"] > 64 and not c["rp"] and c["N"] > 8192) or (not c["rp"] and c["N"] > 33000):
        return None
    X32, W, Y = _inputs(c, seed)
    X, W, N, kappa = X32.double(), W.double(), c["N"], c["kappa"]
    dist, knn = _knn(X, c)
    if c["varh"]:
        h = dist[:, min(16, kappa) - 1].sqrt().float().double()
    else:
        h = torch.full((N,), float(np.float32(c["h"])), dtype=torch.float64, device=DEV)

    def kernel(A, ids):
        B = X[ids]
        D = (A.square().sum(1)[:, None] + B.square().sum(1)[None] - 2 * (A @ B.T)).clamp_(min=0)
        return torch.exp(D.mul_(-0.5 / h[ids].square()))

    def split_key(ids, node):
        P = X[ids]
        a = P[(P - P.mean(0)).square().sum(1).argmax()]
        b = P[(P - a).square().sum(1).argmax()]
        return (P - a) @ (b - a)

    L = _depth(N, c["m"])
    mean = X.mean(0)
    leaves = _tree(X, L, split_key)
    X = X - mean                                            # only differences of points enter from here on
    leaf_of = torch.empty(N, dtype=torch.int64, device=DEV)
    for g, ids in enumerate(leaves):
        leaf_of[ids] = g
    n_leaf, ell_max = 1 << L, c["s_max"] + 20
    lists, skel, wsk = {}, {}, {}
    for t in range(L, 0, -1):
        level = range(1 << t, 2 << t)
        size = 0
        cols, rows = [], []
        for a in level:
            g = a - (1 << t)
            if t == L:
                mine = leaves[g]
                j, key = knn[mine].reshape(-1), dist[mine].reshape(-1)
                n_mine = len(mine)
                cols.append(mine)
            else:
                j, key = (torch.cat([lists[2 * a][q], lists[2 * a + 1][q]]) for q in (0, 1))
                n_mine = sum(len(x) for x in leaves[g << (L - t):(g + 1) << (L - t)])
                cols.append(torch.cat([skel[2 * a], skel[2 * a + 1]]))
            out = (leaf_of[j] >> (L - t)) != g
            j, key = j[out], key[out]
            key, o = torch.sort(key, stable=True)
            j, o = torch.sort(j[o], stable=True)
            key = key[o]
            first = torch.ones_like(j, dtype=torch.bool)
            first[1:] = j[1:] != j[:-1]
            key, o = torch.sort(key[first], stable=True)
            lists[a] = (j[first][o][:ell_max], key[:ell_max])
            ell = min(ell_max, N - n_mine)
            took = lists[a][0][:ell].tolist()
            seen, n_draw, leaf_h = set(took), 0, None
            while len(took) < ell:
                n_draw = max(2 * ell, 2 * n_draw)
                words = (_philox(0, a, n_draw, 1) >> np.uint64(32)) * np.uint64(N) >> np.uint64(32)
                took, seen = lists[a][0][:ell].tolist(), set(lists[a][0][:ell].tolist())
                leaf_h = leaf_of[torch.from_numpy(words.astype(np.int64)).to(DEV)].cpu().numpy() >> (L - t)
                for w, inside in zip(words.tolist(), (leaf_h == g).tolist()):
                    if len(took) < ell and not inside and w not in seen:
                        took.append(w)
                        seen.add(w)
            rows.append(torch.tensor(took, dtype=torch.int64, device=DEV))
            size = max(size, len(cols[-1]))
        n_row = max(len(x) for x in rows)
        step = max(1, int(4e8 // (n_row * max(1, size))))
        for b in range(0, len(rows), step):
            part = range(b, min(b + step, len(rows)))
            A = torch.zeros(len(part), n_row, size, dtype=torch.float64, device=DEV)
            for q, i in enumerate(part):
                A[q, :len(rows[i]), :len(cols[i])] = kernel(X[rows[i]], cols[i])
            ncol = torch.tensor([min(len(cols[i]), len(rows[i])) for i in part], device=DEV)
            A, piv, rank = _id(A, ncol, c["tol"], c["s_min"], c["s_max"])
            for q, (i, s) in enumerate(zip(part, rank.tolist())):
                a, nc = (1 << t) + i, len(cols[i])
                v = W[cols[i]] if t == L else torch.cat([wsk[2 * a], wsk[2 * a + 1]])
                order = piv[q][piv[q] < nc]
                keep = torch.nonzero(piv[q] < nc)[:, 0]
                R = A[q][:s][:, keep]
                skel[a] = cols[i][order[:s]]
                wsk[a] = v[order[:s]]
                if 0 < s < nc:
                    wsk[a] = wsk[a] + torch.linalg.solve_triangular(R[:, :s], R[:, s:] @ v[order[s:]], upper=True)

    if c["op"] == "targets":
        Z = Y.double()
        near_of = torch.empty(len(Z), kappa, dtype=torch.int64, device=DEV)
        step = max(1, (1 << 27) // N)
        Z = Z - mean
        for a in range(0, len(Z), step):
            D = Z[a:a + step].square().sum(1)[:, None] + X.square().sum(1)[None] - 2 * (Z[a:a + step] @ X.T)
            near_of[a:a + step] = leaf_of[D.topk(kappa, dim=1, largest=False)[1]]
    else:
        Z = X
        near_of = torch.cat([leaf_of[:, None], leaf_of[knn]], 1)
    u = torch.zeros(len(Z), c["r"], dtype=torch.float64, device=DEV)
    inside = torch.zeros(len(Z), n_leaf, dtype=torch.bool, device=DEV)
    inside.scatter_(1, near_of, True)

    def add(which, ids, w):
        for q in torch.nonzero(which)[:, 0].split(max(1, (1 << 27) // max(1, len(ids)))):
            u.index_add_(0, q, kernel(Z[q], ids) @ w)

    for g, ids in enumerate(leaves):
        add(inside[:, g], ids, W[ids])
    for t in range(L, 0, -1):
        up = inside.view(len(Z), -1, 2).any(2)
        for g in range(1 << t):
            a = (1 << t) + g
            if len(skel[a]):
                add(up[:, g // 2] & ~inside[:, g], skel[a], wsk[a])
        inside = up
    if c["op"] == "host":
        return u.cpu().numpy()
    return {"u": u, "perm": None} if c["op"] == "build" else u
