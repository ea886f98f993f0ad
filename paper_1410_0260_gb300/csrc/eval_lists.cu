// Evaluation operands and work lists.
//
// Algorithm 4 visits, for target i, exactly the nodes of
//   U_i = union over j in {i} U N_i of the ancestors of leaf(j)
// (eq. (2.5): those nodes cannot be pruned).  The leaves of U_i are summed
// directly (Near(i)); every child of a node of U_i that is not itself in U_i
// is pruned and contributes through its skeleton (Far(i)).  The GPU forms
// every (target, source sub-block) pair of these sets -- an entry -- sorts
// the entries by (sub-block, target) and cuts each sub-block's run into work
// items of at most 128 targets (EvalItem: the sub-block's rows, the item's
// first entry and count), so every item is a dense tile of targets that all
// need the whole sub-block; one persistent kernel then runs all items and
// writes one partial sum per entry, reduced per target in a fixed order.
// Source sub-blocks are at most 128 contiguous rows: of a leaf's points in
// the tree-ordered coordinate array, or of a node's skeleton in the
// skeleton pool.
#include <limits.h>
#include <math.h>

#include <algorithm>
#include <functional>
#include <queue>
#include <vector>

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "askit_impl.cuh"

namespace {

inline unsigned nblk(int64_t n, int b) { return (unsigned)((n + b - 1) / b); }

// Tree-ordered, zero-padded coordinates, squared norms (FP64 sum, rounded)
// and the per-source exponent scale c log2(e) / h_j^2.
__global__ void gather_rows_kernel(const float *X, int d, int d_pad, const int32_t *ids, int64_t n,
                                   int64_t n_rows, const float *hsrc, double kscale, float *out,
                                   float *nrm, float *sc) {
    int64_t row = blockIdx.x;
    if (row >= n_rows) return;
    int32_t id = row < n ? ids[row] : -1;
    for (int k = threadIdx.x; k < d_pad; k += blockDim.x)
        out[row * d_pad + k] = (id >= 0 && k < d) ? X[(int64_t)id * d + k] : 0.0f;
    if (threadIdx.x == 0) {
        double acc = 0.0;
        if (id >= 0)
            for (int k = 0; k < d; ++k) acc += (double)X[(int64_t)id * d + k] * X[(int64_t)id * d + k];
        nrm[row] = (float)acc;
        if (sc) {
            double h = id >= 0 ? (double)hsrc[id] : 1.0;
            sc[row] = id >= 0 ? (float)(kscale * 1.4426950408889634 / (h * h)) : 0.0f;
        }
    }
}

// Skeleton pool row ids: rows [spool[a], spool[a] + s_a) hold S_a, the
// padding up to a multiple of ASK_ROW_PAD is empty (-1).
__global__ void spool_ids_kernel(int64_t n_nodes, const int64_t *spool, const int64_t *skoff,
                                 const int32_t *s, const int32_t *skel_ids, int32_t *rows) {
    int64_t a = 2 + blockIdx.x;
    if (a >= n_nodes) return;
    int64_t r0 = spool[a], r1 = spool[a + 1];
    for (int64_t r = r0 + threadIdx.x; r < r1; r += blockDim.x) {
        int64_t q = r - r0;
        rows[r] = q < s[a] ? skel_ids[skoff[a] + q] : -1;
    }
}

// Adaptive kappa_i (the per-point selection Section 3 proposes from the
// distance to the neighbors): with a kernel cut a > 0, the neighbors kept in
// the prune set run up to the last rank whose kernel value exceeds e^-a,
// kappa_i = 1 + max{ z : c D_z / h_z^2 < a } (0 if none), h_z the
// neighbor's bandwidth, decided in canonical FP64 like the oracle; a <= 0
// keeps all kappa.
__device__ __forceinline__ int kappa_of(const double *dist, const int32_t *ids, int kappa, const float *hsrc,
                                        double kscale, double cut) {
    if (!(cut > 0.0)) return kappa;
    int ki = 0;
    for (int z = 0; z < kappa; ++z) {
        const double h = (double)hsrc[ids[z]];
        if (c_div(c_mul(kscale, dist[z]), c_mul(h, h)) < cut) ki = z + 1;
    }
    return ki;
}

// Prune set of each in-sample target (tree position q): the sorted distinct
// leaves of {i} U N_i (the first kappa_i neighbors), padded with INT_MAX to
// kappa + 1 entries.
__global__ void insample_sets_kernel(const int32_t *perm, const int32_t *leafof, const int32_t *knn,
                                     const double *knnd, const float *hsrc, double kscale, double cut,
                                     int64_t N, int kappa, int32_t *sets) {
    int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (q >= N) return;
    int32_t i = perm[q];
    int32_t *o = sets + q * (kappa + 1);
    int n = 0;
    const int ki = kappa_of(knnd + (int64_t)i * kappa, knn + (int64_t)i * kappa, kappa, hsrc, kscale, cut);
    for (int z = -1; z < ki; ++z) {
        int32_t lf = leafof[z < 0 ? i : knn[(int64_t)i * kappa + z]];
        int p = n;
        bool dup = false;
        for (int u = 0; u < n; ++u) dup |= (o[u] == lf);
        if (dup) continue;
        while (p > 0 && o[p - 1] > lf) { o[p] = o[p - 1]; --p; }
        o[p] = lf;
        ++n;
    }
    for (int u = n; u < kappa + 1; ++u) o[u] = INT_MAX;
}

// Pruning switched off: every leaf is near for every target.
__global__ void all_leaves_sets_kernel(int64_t N, int L, int32_t *sets) {
    int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    int64_t M = (int64_t)1 << L;
    if (e >= N * M) return;
    sets[e] = (int32_t)(M + e % M);
}

// Leaf-grouped prune sets, step 1: for the point at tree position q, its
// own leaf and its neighbors' leaves, at q (kappa + 1) .. (q + 1)(kappa + 1);
// a leaf's points are consecutive positions, so each leaf owns one segment.
__global__ void leaf_keys_kernel(const int32_t *perm, const int32_t *leafof, const int32_t *knn, const double *knnd,
                                 const float *hsrc, double kscale, double cut, int64_t N, int kappa, int32_t *keys) {
    int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (q >= N) return;
    const int32_t i = perm[q];
    int32_t *o = keys + q * (kappa + 1);
    o[0] = leafof[i];
    // neighbors past kappa_i repeat the own leaf (removed with the duplicates)
    const int ki = kappa_of(knnd + (int64_t)i * kappa, knn + (int64_t)i * kappa, kappa, hsrc, kscale, cut);
    for (int z = 0; z < kappa; ++z) o[z + 1] = z < ki ? leafof[knn[(int64_t)i * kappa + z]] : o[0];
}

// Step 2 (a warp per leaf, its segment sorted): count the distinct leaves
// (stride == 0), or write them to the leaf's row of `stride` entries padded
// with INT_MAX.
__global__ void leaf_unique_kernel(const int32_t *keys, const int32_t *beg, const int32_t *end, int stride,
                                   int32_t *rows, int32_t *cnt) {
    const int a = blockIdx.x, lane = threadIdx.x;
    const int32_t b0 = beg[a], b1 = end[a];
    int n = 0;
    for (int32_t base = b0; base < b1; base += 32) {
        const int32_t e = base + lane;
        const bool in = e < b1;
        const int32_t v = in ? keys[e] : 0;
        const bool first = in && (e == b0 || keys[e - 1] != v);
        const unsigned m = __ballot_sync(0xffffffffu, first);
        if (stride > 0 && first) rows[(int64_t)a * stride + n + __popc(m & ((1u << lane) - 1u))] = v;
        n += __popc(m);
    }
    if (stride > 0)
        for (int u = n + lane; u < stride; u += 32) rows[(int64_t)a * stride + u] = INT_MAX;
    else if (lane == 0)
        cnt[a] = n;
}

// Step 3: each target's row is its leaf's.
__global__ void leaf_row_kernel(const int32_t *perm, const int32_t *leafof, int64_t N, int32_t M, int32_t *row) {
    int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (q >= N) return;
    row[q] = leafof[perm[q]] - M;
}

// Out-of-sample prune sets: the sorted distinct leaves of N_y (its first kappa_y
// neighbors; no self term), a warp per target, a neighbor per lane (kappa <= 32).  A
// list that was not filled (ids past N) sets *bad.
__global__ void oos_sets_kernel(const int32_t *leafof, const int32_t *knn, const double *dist, const int32_t *order,
                                const float *hsrc, double kscale, double cut, int64_t N, int64_t T, int kappa, int stride,
                                int32_t *sets, int *bad) {
    const int lane = threadIdx.x & 31;
    const int64_t q = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5);
    if (q >= T) return;                                    // warp-uniform
    const int64_t src = (int64_t)order[q] * kappa + lane;  // target q's neighbors: the caller's row order[q]
    const int32_t j = lane < kappa ? knn[src] : 0;
    const bool in = lane < kappa && j >= 0 && j < N;
    const int32_t id = in ? j : 0;
    if (lane < kappa && !in) *bad = 1;
    int ky = kappa;                                        // kappa_of over the lanes
    if (cut > 0.0) {
        const double h = (double)hsrc[id];
        const bool keep = in && c_div(c_mul(kscale, dist[src]), c_mul(h, h)) < cut;
        const unsigned m = __ballot_sync(0xffffffffu, keep);
        ky = m ? 32 - __clz(m) : 0;
    }
    int32_t v = in && lane < ky ? leafof[id] : INT_MAX;
#pragma unroll
    for (int k = 2; k <= 32; k <<= 1)
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            const int32_t o = __shfl_xor_sync(0xffffffffu, v, j);
            v = (((lane & j) == 0) == ((lane & k) == 0)) ? min(v, o) : max(v, o);
        }
    const int32_t prev = __shfl_up_sync(0xffffffffu, v, 1);
    const bool first = v != INT_MAX && (lane == 0 || v != prev);
    const unsigned m = __ballot_sync(0xffffffffu, first);
    int32_t *o = sets + q * stride;
    if (first) o[__popc(m & ((1u << lane) - 1u))] = v;
    for (int u = __popc(m) + lane; u < stride; u += 32) o[u] = INT_MAX;
}

// Prune-set row of target q: its own row, or a shared one (leaf-grouped).
__device__ __forceinline__ const int32_t *set_of(const int32_t *sets, int stride, const int32_t *set_row, int64_t q) {
    return sets + (set_row ? (int64_t)set_row[q] : q) * stride;
}

// Near and Far sets of one target from its sorted prune leaves, a warp per
// target.  Near = the leaves; Far = for each depth, the sibling of every distinct
// ancestor at that depth when the sibling is not itself an ancestor of a near
// leaf.  With a height limit fh >= 0 (skeletons only for nodes at most fh levels
// above the leaves, Section 3's level restriction), a higher Far node is replaced
// by its descendants fh levels above the leaves (none holds a near leaf).
// Every sub-block (<= ASK_BLK_N rows) of a Near or Far node is an entry; entries
// are in the order near leaves ascending, then far nodes from the deepest level
// up, which fixes the order their partial sums are added in.  EMIT false: counts
// the target's entries into cnt and adds the near nodes, far nodes and pairs to
// tot[0 .. 2]; EMIT true: writes the entries from off[q] on: key = sub-block
// index, val = the entry's own position, tq = the target.
// The lanes take 32 leaves at a time: a thread a target spent 70 us on 100
// targets (each walk a chain of dependent loads), a warp 10.
template <bool EMIT>
__global__ void __launch_bounds__(256) lists_kernel(const int32_t *sets, int stride, const int32_t *set_row, int64_t T,
                                                    int L, int fh, const int32_t *nsize, const int32_t *s,
                                                    const int32_t *leaf_cbase, const int32_t *node_cbase,
                                                    const int64_t *off, int64_t *cnt, unsigned long long *tot,
                                                    uint32_t *keys, int32_t *vals, int32_t *tq) {
    __shared__ unsigned long long sum[3];
    const int lane = threadIdx.x & 31;
    const int64_t q = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5);
    if (!EMIT) {
        if (threadIdx.x < 3) sum[threadIdx.x] = 0;
        __syncthreads();
    }
    if (q < T) {                                           // warp-uniform
        const int32_t *set = set_of(sets, stride, set_row, q);
        const int32_t leaf0 = (int32_t)1 << L;
        int n = 0;
        for (int b = 0; b < stride; b += 32) {
            const unsigned m = __ballot_sync(0xffffffffu, b + lane < stride && set[b + lane] != INT_MAX);
            n += __popc(m);
            if (m != 0xffffffffu) break;
        }
        int64_t run = EMIT ? off[q] : 0;
        unsigned long long c_near = 0, c_far = 0, c_pairs = 0;
        // this lane's nodes first .. first + k - 1 (none for k = 0)
        auto take = [&](int32_t first, int32_t k, bool far) {
            int c = 0;
            for (int32_t i = 0; i < k; ++i) {
                const int rows = far ? s[first + i] : nsize[first + i];
                c += (rows + ASK_BLK_N - 1) / ASK_BLK_N;
                c_pairs += rows;
            }
            (far ? c_far : c_near) += k;
            int incl = c;
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += v;
            }
            if (EMIT) {
                int64_t o = run + incl - c;
                for (int32_t i = 0; i < k; ++i) {
                    const int32_t node = first + i;
                    const int rows = far ? s[node] : nsize[node];
                    const int32_t c0 = far ? node_cbase[node] : leaf_cbase[node - leaf0];
                    for (int ch = 0; ch * ASK_BLK_N < rows; ++ch, ++o) {
                        keys[o] = (uint32_t)(c0 + ch);
                        vals[o] = (int32_t)o;
                        tq[o] = (int32_t)q;
                    }
                }
            }
            run += __shfl_sync(0xffffffffu, incl, 31);
        };
        for (int b = 0; b < n; b += 32) {
            const int u = b + lane;
            take(u < n ? set[u] : 0, u < n ? 1 : 0, false);
        }
        for (int depth = L; depth >= 1; --depth) {
            const int sh = L - depth;
            for (int b = 0; b < n; b += 32) {
                const int u = b + lane;
                int32_t first = 0, k = 0;
                if (u < n) {
                    const int32_t anc = set[u] >> sh;
                    if (u == 0 || (set[u - 1] >> sh) != anc) {       // the first leaf below its ancestor
                        const int32_t sib = anc ^ 1, lo = sib << sh;
                        // the leaves under sib form one run of the sorted set
                        int x = 0, z = n;
                        while (x < z) {
                            const int mid = (x + z) >> 1;
                            if (set[mid] < lo) x = mid + 1; else z = mid;
                        }
                        if (!(x < n && (set[x] >> sh) == sib)) {
                            const int down = fh >= 0 && sh > fh ? sh - fh : 0;
                            first = sib << down;
                            k = (int32_t)1 << down;
                        }
                    }
                }
                take(first, k, true);
            }
        }
        if (!EMIT) {
            for (int o = 16; o > 0; o >>= 1) {
                c_near += __shfl_xor_sync(0xffffffffu, c_near, o);
                c_far += __shfl_xor_sync(0xffffffffu, c_far, o);
                c_pairs += __shfl_xor_sync(0xffffffffu, c_pairs, o);
            }
            if (lane == 0) {
                cnt[q] = run;
                if (tot) {
                    atomicAdd(&sum[0], c_near);
                    atomicAdd(&sum[1], c_far);
                    atomicAdd(&sum[2], c_pairs);
                }
            }
        }
    }
    if (!EMIT && tot) {
        __syncthreads();
        if (threadIdx.x < 3) atomicAdd(tot + threadIdx.x, sum[threadIdx.x]);
    }
}

// After the stable sort by sub-block: slot of every emitted entry and the target
// of every sorted entry.
__global__ void scatter_kernel(const int32_t *emit_of, const int32_t *tq, int64_t n, int32_t *slot_of_emit,
                               int32_t *tgt) {
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= n) return;
    const int32_t o = emit_of[e];
    slot_of_emit[o] = (int32_t)e;
    tgt[e] = tq[o];
}

// First entry of every sub-block c (the number of smaller keys), c = 0 .. n_sub.
__global__ void sub_start_kernel(const uint32_t *keys, int64_t n, int64_t n_sub, int32_t *start) {
    const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (c > n_sub) return;
    int64_t lo = 0, hi = n;
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (keys[mid] < (uint32_t)c) lo = mid + 1; else hi = mid;
    }
    start[c] = (int32_t)lo;
}

// Items of block b = sub-block blk_sub[b]: its entries in runs of ASK_TILE_M.
__global__ void build_items_kernel(const int32_t *blk_sub, const int32_t *block_off, const int32_t *start,
                                   const int64_t *sb_row0, const int32_t *sb_nr, const int32_t *sb_wide, int64_t n_leaf_sub,
                                   EvalItem *items) {
    const int b = blockIdx.x;
    const int32_t c = blk_sub[b], i0 = block_off[b], n = block_off[b + 1] - i0;
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
        EvalItem x;
        x.row0 = (int32_t)sb_row0[c];
        x.nrows = sb_nr[c] | (c >= n_leaf_sub ? (int32_t)0x80000000 : 0);
        x.e0 = start[c] + k * ASK_TILE_M;
        x.cnt = min(ASK_TILE_M, start[c + 1] - x.e0);
        x.cidx = c;
        x.wide = sb_wide ? sb_wide[c] : 0;
        x.pad_[0] = x.pad_[1] = 0;
        items[i0 + k] = x;
    }
}

// U of target q = the sum of its entries' partials in emission order; a thread
// takes one target and one vector.  Bound by HBM/L2 sectors of the partials and
// the 4-byte slots.  A target's slots are a contiguous run: read one at a time,
// the 32 runs of a warp cost 32 sectors an entry, so they are read 16 bytes at a
// time from the aligned groups that cover the run, the next group and two groups'
// eight partials in flight together.  1M x 64, r = 1 (97 M entries): 405 -> 300 us;
// 64K, r = 16 (9 M entries, 64 bytes each): 140 us either way (16-byte loads of
// four vectors a thread measured slower, 165 us: fewer loads in flight).
__global__ void __launch_bounds__(256) reduce_partials_kernel(const float *partial, const int64_t *off,
                                                              const int32_t *slot_of_emit, int64_t T, int r,
                                                              const int32_t *out_rows, float *U, int64_t ldu) {
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t q = r == 1 ? t : t / r;
    const int z = r == 1 ? 0 : (int)(t % r);
    if (q >= T) {
        pdl_wait();
        return;
    }
    const int64_t o0 = off[q], o1 = off[q + 1];
    // groups of 4 slots at 16-byte boundaries: the first and the last may hold
    // slots of other targets (the array is allocated with 4 spare ones)
    const int4 *sl = reinterpret_cast<const int4 *>(slot_of_emit);
    const int64_t g1 = (o1 + 3) >> 2, gf = o1 >> 2;        // groups up to gf - 1 end inside the run
    int64_t g = o0 >> 2;
    int4 cur = g < g1 ? sl[g] : make_int4(0, 0, 0, 0);
    const int64_t row = out_rows[q];
    pdl_wait();
    float acc = 0.f;
    auto load = [&](int32_t slot) { return partial[(int64_t)slot * r + z]; };
    auto part = [&](int64_t gg, const int4 &c4) {          // a group with slots of other targets
        const int32_t c[4] = {c4.x, c4.y, c4.z, c4.w};
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (4 * gg + k >= o0 && 4 * gg + k < o1) acc += load(c[k]);
    };
    if (g < g1 && (4 * g < o0 || 4 * g + 4 > o1)) {
        part(g, cur);
        ++g;
        if (g < g1) cur = sl[g];
    }
    for (; g + 2 <= gf; g += 2) {
        const int4 c1 = sl[g + 1];
        const float v0 = load(cur.x), v1 = load(cur.y), v2 = load(cur.z), v3 = load(cur.w);
        const float v4 = load(c1.x), v5 = load(c1.y), v6 = load(c1.z), v7 = load(c1.w);
        if (g + 2 < g1) cur = sl[g + 2];
        acc += v0; acc += v1; acc += v2; acc += v3;
        acc += v4; acc += v5; acc += v6; acc += v7;
    }
    for (; g < g1; ++g) {
        part(g, cur);
        if (g + 1 < g1) cur = sl[g + 1];
    }
    U[row * ldu + z] = acc;
}

}  // namespace

askit_status build_eval_operands(askit_tree t, cudaStream_t s) {
    const int64_t N = t->N;
    t->N_pad = (N + ASK_TILE_M - 1) / ASK_TILE_M * ASK_TILE_M + 256;
    ASK_TRY(t->arena.alloc(&t->Xt, (size_t)t->N_pad * t->d_pad));
    ASK_TRY(t->arena.alloc(&t->nrm_t, t->N_pad));
    ASK_TRY(t->arena.alloc(&t->sc_t, t->N_pad));
    gather_rows_kernel<<<(unsigned)t->N_pad, 128, 0, s>>>(t->X, t->d, t->d_pad, t->perm, N, t->N_pad, t->hsrc,
                                                         t->prm.kernel_scale, t->Xt, t->nrm_t, t->sc_t);
    ASK_LAUNCH();
    int64_t rows = std::max<int64_t>(t->spool_rows, 1) + 256;
    int32_t *ids = nullptr;
    ASK_TRY(t->arena.alloc(&ids, rows));
    ASK_CUDA(cudaMemsetAsync(ids, 0xff, sizeof(int32_t) * rows, s));
    if (t->n_nodes > 2)
        spool_ids_kernel<<<(unsigned)(t->n_nodes - 2), 128, 0, s>>>(t->n_nodes, t->d_spool, t->d_skoff, t->d_s,
                                                                   t->skel_ids, ids);
    ASK_LAUNCH();
    ASK_TRY(t->arena.alloc(&t->Xs, (size_t)rows * t->d_pad));
    ASK_TRY(t->arena.alloc(&t->nrm_s, rows));
    ASK_TRY(t->arena.alloc(&t->sc_s, rows));
    gather_rows_kernel<<<(unsigned)rows, 128, 0, s>>>(t->X, t->d, t->d_pad, ids, rows, rows, t->hsrc,
                                                     t->prm.kernel_scale, t->Xs, t->nrm_s, t->sc_s);
    ASK_LAUNCH();
    ASK_CUDA(cudaStreamSynchronize(s));
    t->arena.release(ids);
    return ASKIT_OK;
}

// One CTA per source sub-block: its center (FP64 mean of the rows of the
// sub-block's node, rounded), the centered rows split for the tensor cores -- TF32 (narrow
// rows only): hi = the FP32 value with the 13 low mantissa bits cleared,
// lo = x - hi; BF16: hi = bf16(x), lo = bf16(x - hi); FP16 likewise on the
// prescaled value -- and the squared norms of the centered rows.  Rows are
// kw wide (zeros past d); one warp per row, lanes across the columns.  Wide
// rows (kgplanes) store the 16-bit splits as planes of K groups,
// [kw / 8][rows_total][8], so that a K chunk of consecutive rows is a few
// contiguous runs (the wide kernel's TMA boxes).
__global__ void tc_prep_kernel(const float *X, int d_pad, int kw, bool kgplanes, const int64_t *sb_row0,
                               const int32_t *sb_nrows,
                               const int64_t *nd_row0, const int32_t *nd_nrows, int64_t rows_total, float f16_scale,
                               float *cent, float *Xhi, float *Xlo, uint16_t *Bhi, uint16_t *Blo, uint16_t *Hhi,
                               uint16_t *Hlo, float *nrmc) {
    extern __shared__ float c[];   // [kw]
    const int g = blockIdx.x;
    const int64_t r0 = sb_row0[g];
    const int nr = sb_nrows[g];
    // the center is the mean of the whole node (leaf or skeleton) the
    // sub-block belongs to, so that all sub-blocks of a node share it
    const int64_t n0 = nd_row0[g];
    const int nn = nd_nrows[g];
    for (int k = threadIdx.x; k < kw; k += blockDim.x) {
        double acc = 0.0;
        if (k < d_pad)
            for (int q = 0; q < nn; ++q) acc += (double)X[(n0 + q) * d_pad + k];
        c[k] = nn > 0 ? (float)(acc / nn) : 0.f;
        cent[(int64_t)g * kw + k] = c[k];
    }
    __syncthreads();
    // only the sub-block's own rows: the 128-row window of a short sub-block
    // overlaps the next one, whose rows its own CTA writes
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int q = warp; q < nr; q += nw) {
        const int64_t row = r0 + q;
        if (row >= rows_total) break;
        double nn = 0.0;
        for (int k = lane; k < kw; k += 32) {
            const float x = (k < d_pad) ? X[row * d_pad + k] - c[k] : 0.f;
            nn += (double)x * x;
            const int64_t o = kgplanes ? (((int64_t)(k >> 3) * rows_total + row) << 3) + (k & 7) : row * kw + k;
            if (Xhi) {
                const float hi = __uint_as_float(__float_as_uint(x) & 0xffffe000u);
                Xhi[o] = hi;
                Xlo[o] = x - hi;
            }
            const __nv_bfloat16 bh = __float2bfloat16_rn(x);
            const __nv_bfloat16 bl = __float2bfloat16_rn(x - __bfloat162float(bh));
            Bhi[o] = __bfloat16_as_ushort(bh);
            Blo[o] = __bfloat16_as_ushort(bl);
            const float xs = x * f16_scale;
            const __half hh = __float2half_rn(xs);
            const __half hl = __float2half_rn(xs - __half2float(hh));
            Hhi[o] = __half_as_ushort(hh);
            Hlo[o] = __half_as_ushort(hl);
        }
        for (int o = 16; o > 0; o >>= 1) nn += __shfl_xor_sync(0xffffffffu, nn, o);
        if (lane == 0) nrmc[row] = (float)nn;
    }
}

// Sub-blocks too wide for 3xTF32 on their common center (ASK_WIDE_RHO); a norm
// that is no number or infinite counts as wide.
__global__ void wide_kernel(const int64_t *sb_row0, const int32_t *sb_nr, int64_t n_leaf_sub, const float *sc_t,
                            const float *sc_s, const float *nrm_t, const float *nrm_s, int32_t *wide) {
    const int64_t b = blockIdx.x;
    const int lane = threadIdx.x;
    const bool far = b >= n_leaf_sub;
    float sc = 0.f, n = 0.f;
    bool bad = false;
    for (int q = lane; q < sb_nr[b]; q += 32) {
        const int64_t row = sb_row0[b] + q;
        const float v = (far ? nrm_s : nrm_t)[row];
        bad |= !(v <= 3.4e38f);
        n = fmaxf(n, v);
        sc = fmaxf(sc, (far ? sc_s : sc_t)[row]);
    }
    for (int o = 16; o > 0; o >>= 1) {
        sc = fmaxf(sc, __shfl_xor_sync(0xffffffffu, sc, o));
        n = fmaxf(n, __shfl_xor_sync(0xffffffffu, n, o));
    }
    bad = __any_sync(0xffffffffu, bad);
    if (lane == 0) wide[b] = bad || !(sc * n <= ASK_WIDE_RHO);
}

// Largest |x_k| over the data (bounds every centered coordinate by twice it).
__global__ void extent_kernel(const float *X, int64_t N, int d, float *ext) {
    int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    float v = e < N * d ? fabsf(X[e]) : 0.f;
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    if ((threadIdx.x & 31) == 0) atomicMax(reinterpret_cast<int *>(ext), __float_as_int(v));
}

askit_status build_tc_operands(askit_tree t, cudaStream_t s) {
    const int64_t nn = t->n_nodes, M = (int64_t)1 << t->L;
    std::vector<int32_t> lcb(M), ncb(nn, 0);
    std::vector<int64_t> r0;
    std::vector<int32_t> nr;
    std::vector<int64_t> node_r0;    // per sub-block: first row and rows of its node
    std::vector<int32_t> node_nr;    //   (every sub-block of a node shares the node's center)
    std::vector<int64_t> sub_node;   // per sub-block: heap index of its node
    for (int64_t l = 0; l < M; ++l) {
        lcb[l] = (int32_t)r0.size();
        int64_t a = M + l, sz = t->h_size[a];
        for (int64_t ch = 0; ch * ASK_BLK_N < sz; ++ch) {
            r0.push_back(t->h_start[a] + ch * ASK_BLK_N);
            nr.push_back((int32_t)std::min<int64_t>(ASK_BLK_N, sz - ch * ASK_BLK_N));
            node_r0.push_back(t->h_start[a]);
            node_nr.push_back((int32_t)sz);
            sub_node.push_back(a);
        }
    }
    int64_t n_leaf_sub = (int64_t)r0.size();
    for (int64_t a = 2; a < nn; ++a) {
        ncb[a] = (int32_t)(r0.size() - n_leaf_sub);
        int64_t sz = t->h_s[a];
        for (int64_t ch = 0; ch * ASK_BLK_N < sz; ++ch) {
            r0.push_back(t->h_spool[a] + ch * ASK_BLK_N);
            nr.push_back((int32_t)std::min<int64_t>(ASK_BLK_N, sz - ch * ASK_BLK_N));
            node_r0.push_back(t->h_spool[a]);
            node_nr.push_back((int32_t)sz);
            sub_node.push_back(a);
        }
    }
    for (int64_t a = 2; a < nn; ++a) ncb[a] += (int32_t)n_leaf_sub;
    t->n_sub = (int64_t)r0.size();
    // schedule order of the sub-blocks: the tree position of their node's
    // first point (leaf sub-blocks: their own first row), then their index
    t->h_sub_node = sub_node;
    t->h_sub_pos.assign(t->n_sub, 0);
    for (int64_t q = 0; q < n_leaf_sub; ++q) t->h_sub_pos[q] = r0[q];
    for (int64_t a = 2; a < nn; ++a)
        for (int64_t ch = 0; ch * ASK_BLK_N < t->h_s[a]; ++ch) t->h_sub_pos[ncb[a] + ch] = t->h_start[a];
    ASK_TRY(t->arena.alloc(&t->leaf_cbase, M));
    ASK_TRY(t->arena.alloc(&t->node_cbase, nn));
    ASK_CUDA(cudaMemcpyAsync(t->leaf_cbase, lcb.data(), sizeof(int32_t) * M, cudaMemcpyHostToDevice, s));
    ASK_CUDA(cudaMemcpyAsync(t->node_cbase, ncb.data(), sizeof(int32_t) * nn, cudaMemcpyHostToDevice, s));
    // narrow rows (d <= TC_K) get TC_K columns and all three splits; wide
    // rows keep their d_pad columns (a multiple of 32, the K chunk of the
    // wide kernel) and get the 16-bit splits only
    const bool wide = t->d > TC_K;
    const int kw = wide ? t->d_pad : TC_K;
    ASK_TRY(t->arena.alloc(&t->sb_row0, std::max<int64_t>(1, t->n_sub)));
    ASK_TRY(t->arena.alloc(&t->sb_nr, std::max<int64_t>(1, t->n_sub)));
    ASK_CUDA(cudaMemcpyAsync(t->sb_row0, r0.data(), sizeof(int64_t) * t->n_sub, cudaMemcpyHostToDevice, s));
    ASK_CUDA(cudaMemcpyAsync(t->sb_nr, nr.data(), sizeof(int32_t) * t->n_sub, cudaMemcpyHostToDevice, s));
    t->n_leaf_sub = n_leaf_sub;
    if (kw > 8192) {                    // no tensor-core operands (plain FP32 path only)
        ASK_CUDA(cudaStreamSynchronize(s));
        return ASKIT_OK;
    }
    t->kw = kw;
    int64_t *d_r0 = t->sb_row0;
    int32_t *d_nr = t->sb_nr;
    int64_t *d_nd0 = nullptr;
    int32_t *d_ndn = nullptr;
    ASK_CUDA(cudaMallocAsync(&d_nd0, sizeof(int64_t) * std::max<int64_t>(1, t->n_sub), s));
    ASK_CUDA(cudaMallocAsync(&d_ndn, sizeof(int32_t) * std::max<int64_t>(1, t->n_sub), s));
    ASK_CUDA(cudaMemcpyAsync(d_nd0, node_r0.data(), sizeof(int64_t) * t->n_sub, cudaMemcpyHostToDevice, s));
    ASK_CUDA(cudaMemcpyAsync(d_ndn, node_nr.data(), sizeof(int32_t) * t->n_sub, cudaMemcpyHostToDevice, s));
    t->srows = std::max<int64_t>(t->spool_rows, 1) + 256;
    const size_t et = (size_t)t->N_pad * kw, es = (size_t)t->srows * kw;
    ASK_TRY(t->arena.alloc(&t->cent, (size_t)std::max<int64_t>(1, t->n_sub) * kw));
    if (!wide) {
        ASK_TRY(t->arena.alloc(&t->Xt_hi, et));
        ASK_TRY(t->arena.alloc(&t->Xt_lo, et));
        ASK_TRY(t->arena.alloc(&t->Xs_hi, es));
        ASK_TRY(t->arena.alloc(&t->Xs_lo, es));
        ASK_CUDA(cudaMemsetAsync(t->Xt_hi, 0, sizeof(float) * et, s));
        ASK_CUDA(cudaMemsetAsync(t->Xt_lo, 0, sizeof(float) * et, s));
        ASK_CUDA(cudaMemsetAsync(t->Xs_hi, 0, sizeof(float) * es, s));
        ASK_CUDA(cudaMemsetAsync(t->Xs_lo, 0, sizeof(float) * es, s));
    }
    uint16_t **h16[8] = {&t->Xt_bhi, &t->Xt_blo, &t->Xt_hhi, &t->Xt_hlo, &t->Xs_bhi, &t->Xs_blo, &t->Xs_hhi, &t->Xs_hlo};
    for (int i = 0; i < 8; ++i) {
        const size_t n = i < 4 ? et : es;
        ASK_TRY(t->arena.alloc(h16[i], n));
        ASK_CUDA(cudaMemsetAsync(*h16[i], 0, sizeof(uint16_t) * n, s));
    }
    ASK_TRY(t->arena.alloc(&t->nrmc_t, t->N_pad));
    ASK_TRY(t->arena.alloc(&t->nrmc_s, t->srows));
    ASK_CUDA(cudaMemsetAsync(t->nrmc_t, 0, sizeof(float) * t->N_pad, s));
    ASK_CUDA(cudaMemsetAsync(t->nrmc_s, 0, sizeof(float) * t->srows, s));
    // FP16 prescale: a power of 2 that maps the data's widest coordinate
    // range to at most 2^14, so centered values and their differences stay
    // far below the FP16 maximum (65504)
    {
        float *ext = nullptr;
        ASK_CUDA(cudaMalloc(&ext, sizeof(float)));
        ASK_CUDA(cudaMemsetAsync(ext, 0, sizeof(float), s));
        extent_kernel<<<(unsigned)((t->N * t->d + 255) / 256), 256, 0, s>>>(t->X, t->N, t->d, ext);
        float hext = 0.f;
        ASK_CUDA(cudaMemcpyAsync(&hext, ext, sizeof(float), cudaMemcpyDeviceToHost, s));
        ASK_CUDA(cudaStreamSynchronize(s));
        cudaFree(ext);
        int e = 0;
        if (hext > 0.f) frexpf(16384.f / (2.f * hext), &e);
        t->f16_scale = ldexpf(1.f, e - 1);
    }
    const size_t csm = sizeof(float) * kw;
    if (n_leaf_sub > 0)
        tc_prep_kernel<<<(unsigned)n_leaf_sub, 256, csm, s>>>(t->Xt, t->d_pad, kw, wide, d_r0, d_nr, d_nd0, d_ndn, t->N_pad,
                                                            t->f16_scale, t->cent, t->Xt_hi, t->Xt_lo, t->Xt_bhi,
                                                            t->Xt_blo, t->Xt_hhi, t->Xt_hlo, t->nrmc_t);
    if (t->n_sub > n_leaf_sub)
        tc_prep_kernel<<<(unsigned)(t->n_sub - n_leaf_sub), 256, csm, s>>>(
            t->Xs, t->d_pad, kw, wide, d_r0 + n_leaf_sub, d_nr + n_leaf_sub, d_nd0 + n_leaf_sub, d_ndn + n_leaf_sub,
            t->srows, t->f16_scale, t->cent + n_leaf_sub * kw, t->Xs_hi, t->Xs_lo, t->Xs_bhi, t->Xs_blo, t->Xs_hhi,
            t->Xs_hlo, t->nrmc_s);
    if (!wide && t->n_sub > 0) {
        ASK_TRY(t->arena.alloc(&t->sb_wide, t->n_sub));
        wide_kernel<<<(unsigned)t->n_sub, 32, 0, s>>>(t->sb_row0, t->sb_nr, n_leaf_sub, t->sc_t, t->sc_s, t->nrmc_t,
                                                      t->nrmc_s, t->sb_wide);
    }
    ASK_LAUNCH();
    cudaFreeAsync(d_nd0, s);
    cudaFreeAsync(d_ndn, s);
    std::vector<int32_t> h_wide(t->sb_wide ? t->n_sub : 0);
    if (t->sb_wide)
        ASK_CUDA(cudaMemcpyAsync(h_wide.data(), t->sb_wide, sizeof(int32_t) * t->n_sub, cudaMemcpyDeviceToHost, s));
    ASK_CUDA(cudaStreamSynchronize(s));
    t->any_wide = std::find(h_wide.begin(), h_wide.end(), 1) != h_wide.end();
    if (!wide) ASK_TRY(build_g16_operands(t, s));
    return ASKIT_OK;
}

void free_prune_sets(PruneSets &ps) {
    if (ps.sets) cudaFree(ps.sets);
    if (ps.set_row) cudaFree(ps.set_row);
    ps = PruneSets();
}

// Leaf-grouped prune sets: the sorted distinct leaves of {p} U N_p over the
// points p of each leaf (one row per leaf), and every target's row index.
askit_status leaf_prune_sets(askit_tree t, PruneSets &ps, cudaStream_t s) {
    const int64_t N = t->N, M = (int64_t)1 << t->L, k1 = t->kappa + 1;
    if (N * k1 >= ((int64_t)1 << 31)) {
        askit_set_error("leaf-grouped lists need N (kappa + 1) < 2^31");
        return ASKIT_ERR_UNSUPPORTED;
    }
    int32_t *keys = nullptr, *keys_s = nullptr, *beg = nullptr, *cnt = nullptr;
    void *tmp = nullptr;
    size_t tb = 0;
    askit_status rc = ASKIT_OK;
    std::vector<int32_t> hb(2 * M), hc(M);
    for (int64_t a = 0; a < M; ++a) {
        hb[a] = (int32_t)(t->h_start[M + a] * k1);
        hb[M + a] = (int32_t)((t->h_start[M + a] + t->h_size[M + a]) * k1);
    }
    int mx = 0;
#define PCHK(x) do { cudaError_t e_ = (x); if (e_ != cudaSuccess) { askit_set_error("leaf prune sets: %s", cudaGetErrorString(e_)); rc = e_ == cudaErrorMemoryAllocation ? ASKIT_ERR_OOM : ASKIT_ERR_CUDA; goto out; } } while (0)
#define PTRY(x) do { rc = (x); if (rc != ASKIT_OK) goto out; } while (0)
    PCHK(cudaMalloc(&keys, sizeof(int32_t) * N * k1));
    PCHK(cudaMalloc(&keys_s, sizeof(int32_t) * N * k1));
    PCHK(cudaMalloc(&beg, sizeof(int32_t) * 2 * M));
    PCHK(cudaMalloc(&cnt, sizeof(int32_t) * M));
    PCHK(cudaMemcpyAsync(beg, hb.data(), sizeof(int32_t) * 2 * M, cudaMemcpyHostToDevice, s));
    leaf_keys_kernel<<<nblk(N, 128), 128, 0, s>>>(t->perm, t->leafof, t->knn, t->knnd, t->hsrc, t->prm.kernel_scale,
                                                  t->kappa_cut, N, t->kappa, keys);
    PCHK(cudaGetLastError());
    PTRY(seg_sort_i32(nullptr, nullptr, N * k1, (int)M, beg, beg + M, nullptr, &tb, s));
    PCHK(cudaMalloc(&tmp, tb));
    PTRY(seg_sort_i32(keys, keys_s, N * k1, (int)M, beg, beg + M, tmp, &tb, s));
    leaf_unique_kernel<<<(unsigned)M, 32, 0, s>>>(keys_s, beg, beg + M, 0, nullptr, cnt);
    PCHK(cudaGetLastError());
    PCHK(cudaMemcpyAsync(hc.data(), cnt, sizeof(int32_t) * M, cudaMemcpyDeviceToHost, s));
    PCHK(cudaStreamSynchronize(s));
    for (int64_t a = 0; a < M; ++a) mx = std::max(mx, hc[a]);
    ps.stride = std::max(mx, 1);
    PCHK(cudaMalloc(&ps.sets, sizeof(int32_t) * M * ps.stride));
    PCHK(cudaMalloc(&ps.set_row, sizeof(int32_t) * N));
    leaf_unique_kernel<<<(unsigned)M, 32, 0, s>>>(keys_s, beg, beg + M, ps.stride, ps.sets, cnt);
    leaf_row_kernel<<<nblk(N, 256), 256, 0, s>>>(t->perm, t->leafof, N, (int32_t)M, ps.set_row);
    PCHK(cudaGetLastError());
    PCHK(cudaStreamSynchronize(s));
out:
#undef PCHK
#undef PTRY
    for (void *q : {(void *)keys, (void *)keys_s, (void *)beg, (void *)cnt, tmp})
        if (q) cudaFree(q);
    if (rc != ASKIT_OK) free_prune_sets(ps);
    return rc;
}

askit_status insample_prune_sets(askit_tree t, PruneSets &ps, cudaStream_t s) {
    if (t->prm.prune == 2) return leaf_prune_sets(t, ps, s);
    // {i} U N_i as leaves; with pruning off, every leaf
    ps.stride = t->prm.prune ? t->kappa + 1 : (int)((int64_t)1 << t->L);
    ps.set_row = nullptr;
    ASK_CUDA(cudaMalloc(&ps.sets, sizeof(int32_t) * t->N * ps.stride));
    if (!t->prm.prune) {
        int64_t n = t->N << t->L;
        all_leaves_sets_kernel<<<nblk(n, 256), 256, 0, s>>>(t->N, t->L, ps.sets);
        ASK_LAUNCH();
        return ASKIT_OK;
    }
    insample_sets_kernel<<<nblk(t->N, 128), 128, 0, s>>>(t->perm, t->leafof, t->knn, t->knnd, t->hsrc,
                                                         t->prm.kernel_scale, t->kappa_cut, t->N, t->kappa, ps.sets);
    ASK_LAUNCH();
    return ASKIT_OK;
}

askit_status oos_prune_sets(askit_tree t, const int32_t *knn, const double *dist, const int32_t *order, int64_t T,
                            int stride, int32_t *sets, int *bad, cudaStream_t s) {
    oos_sets_kernel<<<nblk(T, 8), 256, 0, s>>>(t->leafof, knn, dist, order, t->hsrc, t->prm.kernel_scale, t->kappa_cut, t->N, T,
                                                 t->kappa, stride, sets, bad);
    ASK_LAUNCH();
    return ASKIT_OK;
}

namespace {

// Deals runs with the given costs, in order, each to the CTA with the least work
// so far (ties to the lowest): cta_off [nc + 1] and the runs of each CTA.
void deal(const std::vector<std::pair<int32_t, int64_t>> &runs, int nc, std::vector<int32_t> &cta_off,
          std::vector<int32_t> &cta_runs) {
    std::vector<int32_t> cta(runs.size());
    bool equal = true;
    for (size_t k = 1; k < runs.size(); ++k) equal = equal && runs[k].second == runs[0].second;
    if (equal) {
        for (size_t k = 0; k < runs.size(); ++k) cta[k] = (int32_t)(k % nc);
    } else {
        typedef std::pair<int64_t, int> Load;   // (work, CTA)
        std::priority_queue<Load, std::vector<Load>, std::greater<Load>> heap;
        for (int c = 0; c < nc; ++c) heap.push({0, c});
        for (size_t k = 0; k < runs.size(); ++k) {
            Load top = heap.top();
            heap.pop();
            cta[k] = top.second;
            top.first += runs[k].second;
            heap.push(top);
        }
    }
    cta_off.assign(nc + 1, 0);
    for (int32_t c : cta) ++cta_off[c + 1];
    for (int c = 0; c < nc; ++c) cta_off[c + 1] += cta_off[c];
    cta_runs.resize(runs.size());
    std::vector<int32_t> at(cta_off.begin(), cta_off.end() - 1);
    for (size_t k = 0; k < runs.size(); ++k) cta_runs[at[cta[k]]++] = runs[k].first;
}

}  // namespace

// Work lists for T targets (slot order) with the given prune sets: every
// (target, source sub-block) pair becomes an entry; entries are sorted by
// (sub-block, target); each sub-block's entries are cut into items of up to
// ASK_TILE_M targets.  partial[e] receives the sub-block's contribution to
// the entry's target; reduce() then sums each target's entries in emission
// order (Near leaves ascending, then Far nodes from the deepest level up),
// which is fixed, so the result does not depend on scheduling.
// Emission is in target order, so a stable sort by the sub-block index alone (two
// passes of 32-bit keys and values up to 65,536 sub-blocks; a 64-bit sort of
// (sub-block, target) took eight) gives the order, and the sub-blocks' first
// entries follow from binary searches.  The host reads those starts back, makes
// the schedules from them and uploads one array.
askit_status build_work_lists(askit_tree t, const int32_t *sets, int stride, const int32_t *set_row, int64_t T,
                              WorkLists &wlst, DevArena &arena, bool all_schedules, cudaStream_t s) {
    int64_t *cnt = nullptr;
    unsigned long long *tot = nullptr;
    uint32_t *keys = nullptr, *keys_s = nullptr;
    int32_t *vals = nullptr, *emit_of = nullptr, *tq = nullptr, *start = nullptr;
    void *tmp = nullptr;
    size_t tb = 0, tb2 = 0;
    askit_status rc = ASKIT_OK;
    cudaError_t e = cudaSuccess;
    int64_t total = 0;
    const int64_t n_sub = t->n_sub;
    unsigned long long h_tot[3] = {0, 0, 0};
    int bits = 1;
    while (((int64_t)1 << bits) < n_sub) ++bits;
    WorkLists &w = wlst;
    w.T = T;
    auto temp = [&](void **p, size_t bytes) {
        return arena.async ? cudaMallocFromPoolAsync(p, bytes, arena.pool, s) : cudaMallocAsync(p, bytes, s);
    };
#define WCHK(x) do { e = (x); if (e != cudaSuccess) goto fail; } while (0)
#define WTRY(x) do { rc = (x); if (rc != ASKIT_OK) goto out; } while (0)
    WCHK(temp((void **)&cnt, sizeof(int64_t) * (T + 1)));
    WCHK(temp((void **)&tot, sizeof(unsigned long long) * 3));
    WTRY(arena.alloc(&w.off, T + 1));
    WCHK(cudaMemsetAsync(cnt + T, 0, sizeof(int64_t), s));
    WCHK(cudaMemsetAsync(tot, 0, sizeof(unsigned long long) * 3, s));
    lists_kernel<false><<<nblk(T, 8), 256, 0, s>>>(sets, stride, set_row, T, t->L, t->far_height, t->nsize, t->d_s,
                                                   t->leaf_cbase, t->node_cbase, nullptr, cnt, tot, nullptr, nullptr,
                                                   nullptr);
    WCHK(cudaGetLastError());
    WTRY(scan_i64(nullptr, nullptr, T + 1, nullptr, &tb, s));
    WCHK(temp((void **)&tmp, tb));
    WTRY(scan_i64(cnt, w.off, T + 1, tmp, &tb, s));
    WCHK(cudaMemcpyAsync(&total, w.off + T, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    WCHK(cudaMemcpyAsync(h_tot, tot, sizeof h_tot, cudaMemcpyDeviceToHost, s));
    WCHK(cudaStreamSynchronize(s));
    cudaFreeAsync(tmp, s);
    tmp = nullptr;
    w.n_entries = total;
    if (total >= ((int64_t)1 << 31)) {
        // entry offsets (work items, slots) are 32-bit
        askit_set_error("%lld (target, sub-block) entries in one work list; at most 2^31 - 1 (lower batch_entries)",
                        (long long)total);
        rc = ASKIT_ERR_UNSUPPORTED;
        goto out;
    }
    WCHK(temp((void **)&keys, sizeof(uint32_t) * std::max<int64_t>(1, total)));
    WCHK(temp((void **)&keys_s, sizeof(uint32_t) * std::max<int64_t>(1, total)));
    WCHK(temp((void **)&vals, sizeof(int32_t) * std::max<int64_t>(1, total)));
    WCHK(temp((void **)&emit_of, sizeof(int32_t) * std::max<int64_t>(1, total)));
    WCHK(temp((void **)&tq, sizeof(int32_t) * std::max<int64_t>(1, total)));
    WCHK(temp((void **)&start, sizeof(int32_t) * (n_sub + 1)));
    lists_kernel<true><<<nblk(T, 8), 256, 0, s>>>(sets, stride, set_row, T, t->L, t->far_height, t->nsize, t->d_s,
                                                  t->leaf_cbase, t->node_cbase, w.off, nullptr, nullptr, keys, vals, tq);
    WCHK(cudaGetLastError());
    WTRY(sort_u32_i32(nullptr, nullptr, nullptr, nullptr, total, bits, nullptr, &tb2, s));
    WCHK(temp((void **)&tmp, tb2));
    WTRY(sort_u32_i32(keys, keys_s, vals, emit_of, total, bits, tmp, &tb2, s));
    sub_start_kernel<<<nblk(n_sub + 1, 128), 128, 0, s>>>(keys_s, total, n_sub, start);
    WCHK(cudaGetLastError());
    {
        std::vector<int32_t> h_start(n_sub + 1);
        WCHK(cudaMemcpyAsync(h_start.data(), start, sizeof(int32_t) * (n_sub + 1), cudaMemcpyDeviceToHost, s));
        // the copy above comes first on the stream, so the host works while the
        // entries are scattered
        cudaEvent_t ev = nullptr;
        WCHK(cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
        e = cudaEventRecord(ev, s);
        if (e == cudaSuccess) {
            rc = arena.alloc(&w.slot_of_emit, total + 4);   // read in groups of 4
            if (rc == ASKIT_OK) rc = arena.alloc(&w.tgt, total);
            if (rc == ASKIT_OK) {
                if (total > 0)
                    scatter_kernel<<<nblk(total, 256), 256, 0, s>>>(emit_of, tq, total, w.slot_of_emit, w.tgt);
                e = cudaGetLastError();
            }
            const cudaError_t es = cudaEventSynchronize(ev);
            if (e == cudaSuccess) e = es;
        }
        cudaEventDestroy(ev);
        if (rc != ASKIT_OK) goto out;
        if (e != cudaSuccess) goto fail;
        // blocks: the sub-blocks with entries, in index order
        std::vector<int32_t> blk_sub, boff(1, 0);
        for (int64_t c = 0; c < n_sub; ++c) {
            const int32_t n = h_start[c + 1] - h_start[c];
            if (n == 0) continue;
            blk_sub.push_back((int32_t)c);
            boff.push_back(boff.back() + (n + ASK_TILE_M - 1) / ASK_TILE_M);
        }
        const int64_t nb = (int64_t)blk_sub.size(), nit = boff.back();
        auto n_items = [&](int32_t b) { return boff[b + 1] - boff[b]; };
        std::vector<int32_t> order(nb);
        for (int64_t b = 0; b < nb; ++b) order[b] = (int32_t)b;
        std::stable_sort(order.begin(), order.end(), [&](int32_t x, int32_t y) { return n_items(x) > n_items(y); });
        // Pairs: sub-blocks 2k and 2k + 1 of one node need the same targets (a
        // target needing a node needs all its sub-blocks), so their items match
        // one to one and a kernel can take both in one 256-column item.  A leader
        // is never the last sub-block of its node, so it is full and its
        // follower's rows start ASK_BLK_N rows later.  The leader keeps its
        // items, the follower's are skipped.
        std::vector<int32_t> partner(nb, -1);
        std::vector<char> follower(nb, 0);
        w.n_pairs = w.pair_items = 0;
        int64_t lead_items = 0;
        for (int64_t b = 0, first = 0; b < nb; ++b) {
            const int32_t c = blk_sub[b];
            if (b > 0 && t->h_sub_node[c] != t->h_sub_node[blk_sub[b - 1]]) first = b;
            if (follower[b]) continue;
            lead_items += n_items(b);
            if (!((b - first) & 1) && b + 1 < nb && blk_sub[b + 1] == c + 1 &&
                t->h_sub_node[c + 1] == t->h_sub_node[c] && h_start[c + 2] - h_start[c + 1] == h_start[c + 1] - h_start[c]) {
                partner[b] = (int32_t)(b + 1);
                follower[b + 1] = 1;
                ++w.n_pairs;
                w.pair_items += n_items(b);
            }
        }
        w.n_items = nit;
        w.n_blocks = nb;
        int dev = 0, sms = 0;
        WCHK(cudaGetDevice(&dev));
        WCHK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        // Items a run, narrow rows: about 24 runs a CTA, of 8 to 64 items -- short
        // enough to deal the work evenly (64K x 64, paired: 165 us an Evaluate
        // against 186 with whole blocks), long enough that the source tiles (74 KB
        // a pair) are not reloaded all the time (1M x 64: 3.94 ms with whole
        // blocks, 4.12 in runs of 8); fewer where that leaves CTAs without work.
        // Wide rows, whose sub-blocks stream through shared memory for every item:
        // ASK_SEG_ITEMS.
        // Unpaired items take half as long, so a reload weighs more: 6 runs a CTA.
        auto run_items = [&](int64_t items, bool pair) -> int32_t {
            const int64_t least = std::max<int64_t>(1, std::min<int64_t>(8, (items + 2 * sms - 1) / (2 * sms)));
            if (t->d > TC_K) return (int32_t)std::min<int64_t>(ASK_SEG_ITEMS, least);
            return (int32_t)std::max<int64_t>(least, std::min<int64_t>(64, items / ((pair ? 24 : 6) * (int64_t)sms)));
        };
        // the upload: blk_sub, block_off, block_order, then each schedule's arrays
        std::vector<int32_t> up(blk_sub);
        const size_t o_boff = up.size();
        up.insert(up.end(), boff.begin(), boff.end());
        const size_t o_order = up.size();
        up.insert(up.end(), order.begin(), order.end());
        size_t o_run[3], o_part = 0, o_cta[3], o_list[3];
        const bool paired = take_pairs(t, w);
        for (int k = 0; k < 3; ++k) {
            w.sched[k] = WorkLists::Sched();
            if (!all_schedules && k != (t->tune_sched & 1) && !(k == 2 && paired)) continue;
            std::vector<int32_t> ord = order;
            if (k == 1)
                std::stable_sort(ord.begin(), ord.end(), [&](int32_t x, int32_t y) {
                    const int64_t px = t->h_sub_pos[blk_sub[x]], py = t->h_sub_pos[blk_sub[y]];
                    return px != py ? px < py : x < y;
                });
            const int32_t len = run_items(k == 2 ? lead_items : nit, k == 2);
            std::vector<int32_t> roff, rfirst(nb), rpart;
            for (int64_t b = 0; b < nb; ++b) {
                rfirst[b] = (int32_t)roff.size();
                for (int32_t i = boff[b]; i < boff[b + 1]; i += len) roff.push_back(i);
            }
            roff.push_back((int32_t)nit);
            if (k == 2) {
                rpart.assign(roff.size(), -1);
                for (int64_t b = 0; b < nb; ++b)
                    if (partner[b] >= 0)
                        for (int32_t r = 0; r < (n_items(b) + len - 1) / len; ++r)
                            rpart[rfirst[b] + r] = rfirst[partner[b]] + r;
            }
            // a run costs its items plus a fixed reload of its source tile
            std::vector<std::pair<int32_t, int64_t>> runs;
            for (int32_t b : ord) {
                if (k == 2 && follower[b]) continue;
                const int64_t f = k == 2 && partner[b] >= 0 ? 2 : 1;
                for (int32_t r = rfirst[b]; roff[r] < boff[b + 1]; ++r)
                    runs.push_back({r, ((int64_t)std::min(roff[r + 1], boff[b + 1]) - roff[r]) * 4 * f + 3 * f});
            }
            const int nc = (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)runs.size(), sms));
            std::vector<int32_t> cta_off, cta_runs;
            deal(runs, nc, cta_off, cta_runs);
            w.sched[k].n_ctas = nc;
            o_run[k] = up.size();
            up.insert(up.end(), roff.begin(), roff.end());
            if (k == 2) {
                o_part = up.size();
                up.insert(up.end(), rpart.begin(), rpart.end());
            }
            o_cta[k] = up.size();
            up.insert(up.end(), cta_off.begin(), cta_off.end());
            o_list[k] = up.size();
            up.insert(up.end(), cta_runs.begin(), cta_runs.end());
        }
        WTRY(arena.alloc(&w.plan, up.size()));
        WTRY(arena.alloc(&w.items, nit));
        WCHK(cudaMemcpyAsync(w.plan, up.data(), sizeof(int32_t) * up.size(), cudaMemcpyHostToDevice, s));
        w.block_off = w.plan + o_boff;
        w.block_order = w.plan + o_order;
        for (int k = 0; k < 3; ++k) {
            if (!w.sched[k].n_ctas) continue;
            w.sched[k].run_off = w.plan + o_run[k];
            w.sched[k].partner = k == 2 ? w.plan + o_part : nullptr;
            w.sched[k].cta_off = w.plan + o_cta[k];
            w.sched[k].cta_runs = w.plan + o_list[k];
        }
        w.use = t->tune_sched & 1;
        if (nb > 0)
            build_items_kernel<<<(unsigned)nb, 128, 0, s>>>(w.plan, w.block_off, start, t->sb_row0, t->sb_nr,
                                                            t->sb_wide, t->n_leaf_sub, w.items);
        WCHK(cudaGetLastError());
        w.pairs_alg = (int64_t)h_tot[2];
        w.pairs_cmp = nit * (int64_t)ASK_TILE_M * ASK_BLK_N;
        w.near_tot = (int64_t)h_tot[0];
        w.far_tot = (int64_t)h_tot[1];
        WCHK(cudaStreamSynchronize(s));                     // the upload's source goes out of scope
    }
    goto out;
fail:
    askit_set_error("work lists: %s", cudaGetErrorString(e));
    rc = e == cudaErrorMemoryAllocation ? ASKIT_ERR_OOM : ASKIT_ERR_CUDA;
out:
#undef WCHK
#undef WTRY
    if (rc != ASKIT_OK) cudaStreamSynchronize(s);
    for (void *q : {(void *)cnt, (void *)tot, (void *)vals, (void *)emit_of, (void *)tq, (void *)start, (void *)keys,
                    (void *)keys_s, tmp})
        if (q) cudaFreeAsync(q, s);
    return rc;
}

// The in-sample work lists in batches of consecutive target slots: a count
// pass over all N targets, then cuts wherever the next target would take the
// running batch past the entry budget.  A sub-block's items and a pair's
// matching lists never straddle a cut (both are lists of targets), and every
// entry's partial sum is computed the same way in whichever batch holds it.
askit_status build_insample_lists(askit_tree t, const PruneSets &ps, cudaStream_t s) {
    const int64_t N = t->N;
    const int32_t *sets = ps.sets, *set_row = ps.set_row;
    const int stride = ps.stride;
    const int64_t budget = t->prm.batch_entries > 0 ? t->prm.batch_entries : ASK_BATCH_ENTRIES;
    std::vector<int64_t> h_cnt(N);
    {
        int64_t *buf = nullptr;
        ASK_CUDA(cudaMallocAsync(&buf, sizeof(int64_t) * N, s));
        lists_kernel<false><<<nblk(N, 8), 256, 0, s>>>(sets, stride, set_row, N, t->L, t->far_height, t->nsize, t->d_s,
                                                       t->leaf_cbase, t->node_cbase, nullptr, buf, nullptr, nullptr,
                                                       nullptr, nullptr);
        cudaError_t e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaMemcpyAsync(h_cnt.data(), buf, sizeof(int64_t) * N, cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        cudaFreeAsync(buf, s);
        ASK_CUDA(e);
    }
    t->wl.clear();
    t->wl_t0.assign(1, 0);
    int64_t acc = 0;
    for (int64_t q = 0; q < N; ++q) {
        if (acc > 0 && acc + h_cnt[q] > budget) {
            t->wl_t0.push_back(q);
            acc = 0;
        }
        acc += h_cnt[q];
    }
    t->wl_t0.push_back(N);
    const size_t nb = t->wl_t0.size() - 1;
    t->wl.resize(nb);
    t->wl_entries = t->wl_entries_max = 0;
    for (size_t b = 0; b < nb; ++b) {
        const int64_t t0 = t->wl_t0[b], T = t->wl_t0[b + 1] - t0;
        // a batch's targets start at t0: shift the shared-row index, or the rows
        if (set_row)
            ASK_TRY(build_work_lists(t, sets, stride, set_row + t0, T, t->wl[b], t->arena, true, s));
        else
            ASK_TRY(build_work_lists(t, sets + t0 * stride, stride, nullptr, T, t->wl[b], t->arena, true, s));
        if (t->wl[b].n_entries >= ((int64_t)1 << 31)) {
            askit_set_error("a single target has more than 2^31 work entries");
            return ASKIT_ERR_UNSUPPORTED;
        }
        t->wl_entries += t->wl[b].n_entries;
        t->wl_entries_max = std::max(t->wl_entries_max, t->wl[b].n_entries);
    }
    return ASKIT_OK;
}

void free_work_lists(WorkLists &w, DevArena &arena) {
    void *ptrs[] = {w.off, w.slot_of_emit, w.tgt, w.items, w.plan};
    for (void *p : ptrs)
        if (p) arena.release(p);
    w = WorkLists();
}

// The CTA schedule the kernels use without pairs: heaviest first or tree order
// (askit_set_launch).
void use_schedule(askit_tree t) {
    for (WorkLists &w : t->wl) w.use = t->tune_sched & 1;
}

askit_status reduce_partials(const WorkLists &w, const float *partial, int r, const int32_t *out_rows, float *U,
                             int64_t ldu, cudaStream_t s) {
    if (w.T == 0) return ASKIT_OK;
    return launch_pdl(reduce_partials_kernel, dim3(nblk(w.T * r, 256)), dim3(256), 0, s, partial, w.off,
                      w.slot_of_emit, w.T, r, out_rows, U, ldu);
}
