// Tree build and nearest-neighbor search on the GPU (Section 2.2).
//
// Both the ASKIT tree and the random-projection (RP) trees of the kNN search
// are built level by level: every node of a level computes its projection
// key per point, the level's nodes are sorted segment-wise by (key, id), the
// lower ceil(n/2) points form the left child, and each child is re-sorted by
// id.  All leaves sit at one depth L, the least depth at which no node holds
// more than the leaf size.  Distances and projections are FP64 sums in
// ascending coordinate order with no fused multiply-add, so the trees and
// neighbor lists are bit-exact functions of the input.
#include <float.h>
#include <limits.h>

#include <mutex>

#include "askit_impl.cuh"
#include "knn_warp.cuh"

namespace {

// Squared distance with an FP64 first operand (the node center).
__device__ __forceinline__ double c_dist2_df(const double *x, const float *y, int d) {
    double acc = 0.0;
    for (int k = 0; k < d; ++k) {
        double t = c_sub(x[k], c_f2d(y[k]));
        acc = c_add(acc, c_mul(t, t));
    }
    return acc;
}

// Segment (node) of each position at one tree level, by binary search over
// the level's node starts.
__global__ void seg_of_pos_kernel(const int32_t *lvl_start, int nseg, int64_t N, int32_t *seg) {
    int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (q >= N) return;
    int lo = 0, hi = nseg - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (lvl_start[mid] <= q) lo = mid; else hi = mid - 1;
    }
    seg[q] = lo;
}

// Node centers: FP64 mean, points summed in the node's (ascending id) order.
__global__ void center_kernel(const float *X, int d, const int32_t *order, const int32_t *lvl_start,
                              const int32_t *lvl_size, double *xc) {
    int node = blockIdx.x;
    int k = blockIdx.y * blockDim.x + threadIdx.x;
    if (k >= d) return;
    int64_t b = lvl_start[node], n = lvl_size[node];
    double acc = 0.0;
    // one chain of additions a coordinate, 64 cycles each: the next 16 rows' loads,
    // and the ids of the 16 after them, are in flight during this group's
    int64_t q = 0;
    constexpr int G = 16;
    float x[G];
    int32_t id[G];
    auto ids = [&](int64_t q0) {
#pragma unroll
        for (int u = 0; u < G; ++u) id[u] = q0 + G <= n ? order[b + q0 + u] : 0;
    };
    if (n >= G) {
        ids(0);
#pragma unroll
        for (int u = 0; u < G; ++u) x[u] = X[(int64_t)id[u] * d + k];
        ids(G);
    }
    for (; q + G <= n; q += G) {
        float y[G];
#pragma unroll
        for (int u = 0; u < G; ++u) y[u] = X[(int64_t)id[u] * d + k];     // (row 0 past the last group)
        ids(q + 2 * G);
#pragma unroll
        for (int u = 0; u < G; ++u) acc = c_add(acc, c_f2d(x[u]));
#pragma unroll
        for (int u = 0; u < G; ++u) x[u] = y[u];
    }
    for (; q < n; ++q) acc = c_add(acc, c_f2d(X[(int64_t)order[b + q] * d + k]));
    xc[(int64_t)node * d + k] = c_div(acc, (double)n);
}

// Farthest point from a per-node reference: max D, ties to the smallest id.
// Pass 1 raises best_bits to the largest D (non-negative doubles order like
// their bit patterns); pass 2 lowers best_id among the points attaining it.
template <bool FROM_CENTER>
__global__ void far_pass1(const float *X, int d, const int32_t *order, const int32_t *seg, int64_t N,
                          const double *xc, const int32_t *ref_id, double *Dq,
                          unsigned long long *best_bits) {
    int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (q >= N) return;
    int node = seg[q];
    const float *xj = X + (int64_t)order[q] * d;
    double D = FROM_CENTER ? c_dist2_df(xc + (int64_t)node * d, xj, d)
                           : c_dist2(X + (int64_t)ref_id[node] * d, xj, d);
    Dq[q] = D;
    atomicMax(best_bits + node, (unsigned long long)__double_as_longlong(D));
}

__global__ void far_pass2(const int32_t *order, const int32_t *seg, int64_t N, const double *Dq,
                          const unsigned long long *best_bits, int32_t *best_id) {
    int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (q >= N) return;
    int node = seg[q];
    if ((unsigned long long)__double_as_longlong(Dq[q]) == best_bits[node]) atomicMin(best_id + node, order[q]);
}

// Projection on the line (x_l, x_r) with origin x_l.
__global__ void proj_line_kernel(const float *X, int d, const int32_t *order, const int32_t *seg,
                                 int64_t N, const int32_t *xl, const int32_t *xr, double *p) {
    int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (q >= N) return;
    int node = seg[q];
    const float *xj = X + (int64_t)order[q] * d;
    const float *a = X + (int64_t)xl[node] * d;
    const float *b = X + (int64_t)xr[node] * d;
    double acc = 0.0;
    for (int k = 0; k < d; ++k) {
        double u = c_sub(c_f2d(xj[k]), c_f2d(a[k]));
        double v = c_sub(c_f2d(b[k]), c_f2d(a[k]));
        acc = c_add(acc, c_mul(u, v));
    }
    p[q] = acc;
}

// Projection on a Rademacher direction: bit k%64 of Philox word k/64 keyed
// (seed, iter + 1) with counter (node, word/4) set means -1.
__global__ void proj_rp_kernel(const float *X, int d, const int32_t *order, const int32_t *seg,
                               int64_t N, int64_t node0, uint64_t seed, int iter, double *p) {
    int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (q >= N) return;
    int64_t node = node0 + seg[q];
    const float *xj = X + (int64_t)order[q] * d;
    double acc = 0.0;
    uint64_t w = 0;
    for (int k = 0; k < d; ++k) {
        if ((k & 63) == 0) w = philox_word(seed, (uint64_t)iter + 1, (uint64_t)node, (uint64_t)(k >> 6));
        // +-1 times the coordinate: its sign
        acc = c_add(acc, c_f2d(((w >> (k & 63)) & 1) ? -xj[k] : xj[k]));
    }
    p[q] = acc;
}

__global__ void iota_kernel(int32_t *a, int64_t n) {
    int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (q < n) a[q] = (int32_t)q;
}

template <class T>
__global__ void fill_kernel(T *a, int64_t n, T v) {
    int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (q < n) a[q] = v;
}

inline unsigned nblk(int64_t n, int b) { return (unsigned)((n + b - 1) / b); }

// Every point of an RP-tree leaf against its leaf-mates: block y nleaf + leaf takes the
// leaf's points 64 y .. + 63 as queries, the leaf as candidates, 512 at a time (one grid
// dimension: a leaf may have more query blocks than the second one allows).
// FP32 squared distances (difference form) in 64 x 128 tiles from shared memory, 4 x 8
// pairs a thread; a warp then takes a query's 512 distances: the kappa-th smallest
// (a best-32 list of floats) and the list so far bound what can be among the
// kappa nearest -- an FP32 distance is within (1 +- gam) of the exact one -- and
// only those get their canonical FP64 distance, 32 to a batch.  An FP64
// warp instruction takes 64 cycles of its quarter of the SM for one lane as for
// 32: with the candidates tested 32 at a time against the FP64 list nearly every
// group had a survivor and paid a batch (22.7 ms a tree of 64K x 64, leaves of
// 512; now 1.8).  The list of each point lives in (bd, bi)[point * 32 + lane].
constexpr int KL_Q = 64, KL_C = 512, KL_TILE = 128, KL_K = 32;
constexpr int KL_DT = KL_C + 4, KL_QS = KL_Q + 4, KL_CS = KL_TILE + 4;
constexpr size_t KL_SMEM = sizeof(float) * (KL_Q * KL_DT + KL_K * (KL_QS + KL_CS));

__global__ void __launch_bounds__(256) knn_leaf_kernel(const float *X, int d, const int32_t *order, const int32_t *beg,
                                                       const int32_t *end, unsigned nleaf, int kappa, double *bd,
                                                       int *bi) {
    extern __shared__ __align__(16) float kl[];
    float *dt = kl, *qs = kl + KL_Q * KL_DT, *cs = qs + KL_K * KL_QS;   // [query][candidate], [k][query], [k][candidate]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tx = tid & 15, ty = tid >> 4;                // pairs: queries 4 ty .., candidates 4 tx .. and 64 + 4 tx ..
    const unsigned leaf = blockIdx.x % nleaf;
    const int b0 = beg[leaf], n = end[leaf] - b0, q0 = (int)(blockIdx.x / nleaf) * KL_Q;
    if (q0 >= n) return;                                   // block-uniform
    const int nq = min(KL_Q, n - q0);
    const int32_t *ids = order + b0;
    const float gam = (float)(d + 2) * 5.9604645e-8f * 1.25f + 1e-6f;
    const bool vec = (d & 3) == 0;
    for (int c0 = 0; c0 < n; c0 += KL_C) {
        const int nc = min(KL_C, n - c0);
        for (int t0 = 0; t0 < nc; t0 += KL_TILE) {
            float acc[4][8];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
            for (int k0 = 0; k0 < d; k0 += KL_K) {
                __syncthreads();                           // the last slice, or the last chunk's distances, are read
                for (int e = tid; e < KL_Q * KL_K; e += 256) {
                    const int q = e / KL_K, k = e % KL_K;
                    qs[k * KL_QS + q] = (q < nq && k0 + k < d) ? X[(int64_t)ids[q0 + q] * d + k0 + k] : 0.f;
                }
                for (int e = tid; e < KL_TILE * KL_K; e += 256) {
                    const int c = e / KL_K, k = e % KL_K;
                    cs[k * KL_CS + c] = (t0 + c < nc && k0 + k < d) ? X[(int64_t)ids[c0 + t0 + c] * d + k0 + k] : 0.f;
                }
                __syncthreads();
                const int kn = min(KL_K, d - k0);
                for (int k = 0; k < kn; ++k) {
                    const float4 q4 = *reinterpret_cast<const float4 *>(qs + k * KL_QS + 4 * ty);
                    const float4 ca = *reinterpret_cast<const float4 *>(cs + k * KL_CS + 4 * tx);
                    const float4 cb = *reinterpret_cast<const float4 *>(cs + k * KL_CS + 64 + 4 * tx);
                    const float qv[4] = {q4.x, q4.y, q4.z, q4.w};
                    const float cv[8] = {ca.x, ca.y, ca.z, ca.w, cb.x, cb.y, cb.z, cb.w};
#pragma unroll
                    for (int i = 0; i < 4; ++i)
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            const float t = qv[i] - cv[j];
                            acc[i][j] = fmaf(t, t, acc[i][j]);
                        }
                }
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                float *o = dt + (4 * ty + i) * KL_DT + t0 + 4 * tx;
                *reinterpret_cast<float4 *>(o) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
                *reinterpret_cast<float4 *>(o + 64) = make_float4(acc[i][4], acc[i][5], acc[i][6], acc[i][7]);
            }
        }
        __syncthreads();
        for (int u = warp; u < nq; u += 8) {
            const int self = ids[q0 + u];
            const int64_t slot = (int64_t)self * 32 + lane;
            double ld = bd[slot];
            int li = bi[slot];
            const float *row = dt + u * KL_DT;
            const double kth = __shfl_sync(FULL, ld, kappa - 1);
            // above this an exact distance exceeds the list's kappa-th
            float lim = kth < 1e38 ? __double2float_ru(kth) * (1.f + 2.f * gam) + 1e-37f : INFINITY;
            float l = 3.4e38f;
            const int me = q0 + u - c0;                    // the query's own place among the candidates
            for (int b = 0; b < nc; b += 32) {
                const float v = b + lane < nc && b + lane != me ? row[b + lane] : 3.4e38f;
                warp_offer_f32(l, v <= lim ? v : 3.4e38f, kappa, lane);
            }
            // only a real distance bounds: fewer than kappa below FP32's range leave the
            // limit as it is, and distances past that range (+inf here) stay in
            const float lk = __shfl_sync(FULL, l, kappa - 1);
            if (lk < 3.0e38f) lim = fminf(lim, lk * (1.f + 3.f * gam) + 1e-37f);
            int have = 0;
            int32_t held = 0;
            auto offer = [&]() {
                // not listed yet (every lane takes part in the exchange)
                bool fresh = lane < have;
#pragma unroll 8
                for (int z = 0; z < 32; ++z) {
                    const int listed = __shfl_sync(FULL, li, z);
                    if (listed == held) fresh = false;
                }
                double cd = DBL_MAX;
                int ci = INT_MAX;
                if (fresh) {
                    const float *xq = X + (int64_t)self * d, *xj = X + (int64_t)held * d;
                    double acc = 0.0;
                    if (vec) {
                        for (int k = 0; k < d; k += 4) {
                            const float4 xa = *reinterpret_cast<const float4 *>(xq + k);
                            const float4 xb = *reinterpret_cast<const float4 *>(xj + k);
                            double t = c_sub(c_f2d(xa.x), c_f2d(xb.x));
                            acc = c_add(acc, c_mul(t, t));
                            t = c_sub(c_f2d(xa.y), c_f2d(xb.y));
                            acc = c_add(acc, c_mul(t, t));
                            t = c_sub(c_f2d(xa.z), c_f2d(xb.z));
                            acc = c_add(acc, c_mul(t, t));
                            t = c_sub(c_f2d(xa.w), c_f2d(xb.w));
                            acc = c_add(acc, c_mul(t, t));
                        }
                    } else {
                        acc = c_dist2(xq, xj, d);
                    }
                    cd = acc;
                    ci = held;
                }
                warp_offer(ld, li, cd, ci, kappa, false, lane);
                have = 0;
            };
            for (int b = 0; b < nc; b += 32) {
                // not "above the limit", so a distance that is no number, or infinite, stays in
                const bool pass = b + lane < nc && b + lane != me && !(row[b + lane] > lim);
                const unsigned m = __ballot_sync(FULL, pass);
                if (!m) continue;
                const int32_t p = pass ? ids[c0 + b + lane] : 0;
                warp_collect(m, p, have, held, lane, offer);
            }
            if (have > 0) offer();
            bd[slot] = ld;
            bi[slot] = li;
        }
    }
}

// Tiled exhaustive search: block (qb, sp) takes queries [64 qb, 64 qb + 64)
// against the candidate split [c0, c1).  FP32 squared distances of 64 x 128
// tiles (difference form, k ascending, one FMA per coordinate: the same
// rounding bound as the per-warp search) go to shared memory; warp w then
// filters the rows of its 8 queries against their current kappa-th FP64
// distance and recomputes the survivors in canonical FP64.  Each split
// writes its own best-32 lists; knn_merge_kernel merges the splits.
constexpr int KT_Q = 64, KT_C = 128, KT_K = 32;
// Points a segment above which a tree level is sorted as a whole.  64K x 64, leaves of
// 128, six RP trees (kNN stage) and the tree itself, line at 256, 512, 1024, 2048, 4096,
// 8192 and 16384: 20.6, 19.2, 18.2, 17.1, 16.3, 15.8 and 16.4 ms; 11.1, 10.9, 10.7, 10.6,
// 10.4, 10.4 and 10.5 ms.  1M: 155 to 151 ms and 147 to 146 ms.  Segments of 2048 and
// less are better off sorted one a block; 8192 would gain another 1.2 ms of that build.
constexpr int64_t TREE_RADIX = 2048;

__global__ void __launch_bounds__(256) knn_tiled_kernel(const float *X, int64_t N, int d, const float *Y,
                                                         int64_t Q, int64_t split_len, int kappa, double *bd,
                                                         int *bi, const int32_t *self) {
    // the distance tile reuses the chunk buffers (the selection ends before
    // the next tile's first chunk is loaded)
    __shared__ float sbuf[KT_Q * (KT_C + 1)];
    float (*qs)[KT_Q + 1] = reinterpret_cast<float (*)[KT_Q + 1]>(sbuf);
    float (*cs)[KT_C + 1] = reinterpret_cast<float (*)[KT_C + 1]>(sbuf + KT_K * (KT_Q + 1));
    float (*dt)[KT_C + 1] = reinterpret_cast<float (*)[KT_C + 1]>(sbuf);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tx = tid & 15, ty = tid >> 4;
    const int64_t q0 = (int64_t)blockIdx.x * KT_Q;
    const int64_t c0 = (int64_t)blockIdx.y * split_len;
    const int64_t c1 = c0 + split_len < N ? c0 + split_len : N;
    const float gam = (float)(d + 2) * 5.9604645e-8f * 1.25f + 1e-6f;
    double ld[8];
    int li[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) { ld[u] = DBL_MAX; li[u] = INT_MAX; }
    for (int64_t cb = c0; cb < c1; cb += KT_C) {
        float acc[4][8];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
        for (int k0 = 0; k0 < d; k0 += KT_K) {
            __syncthreads();
            // query chunk [64 x 32] and candidate chunk [128 x 32], transposed, zeros outside
            for (int e = tid; e < KT_Q * KT_K; e += 256) {
                const int qq = e / KT_K, kk = e % KT_K;
                const int64_t q = q0 + qq;
                float v = 0.f;
                if (q < Q && k0 + kk < d) v = Y ? Y[q * d + k0 + kk] : X[q * d + k0 + kk];
                qs[kk][qq] = v;
            }
            for (int e = tid; e < KT_C * KT_K; e += 256) {
                const int cc = e / KT_K, kk = e % KT_K;
                const int64_t j = cb + cc;
                cs[kk][cc] = (j < c1 && k0 + kk < d) ? X[j * d + k0 + kk] : 0.f;
            }
            __syncthreads();
            const int kn = d - k0 < KT_K ? d - k0 : KT_K;
            for (int kk = 0; kk < kn; ++kk) {
                float qv[4], cv[8];
#pragma unroll
                for (int i = 0; i < 4; ++i) qv[i] = qs[kk][ty + 16 * i];
#pragma unroll
                for (int j = 0; j < 8; ++j) cv[j] = cs[kk][tx + 16 * j];
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const float t = qv[i] - cv[j];
                        acc[i][j] = fmaf(t, t, acc[i][j]);
                    }
            }
        }
        __syncthreads();     // every thread is done with the chunk buffers
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) dt[ty + 16 * i][tx + 16 * j] = acc[i][j];
        __syncthreads();
        // selection: warp w owns queries 8w .. 8w+7 of the tile
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int qq = 8 * warp + u;
            const int64_t q = q0 + qq;
            if (q >= Q) continue;                         // warp-uniform
            const float *xq = Y ? Y + q * d : X + q * d;
            for (int rr = 0; rr < KT_C / 32; ++rr) {
                const int64_t j = cb + rr * 32 + lane;
                // queries Y exclude no point unless `self` names the point each
                // query is (the tree's own points as queries)
                const bool valid = j < c1 && (self ? j != self[q] : (Y || j != q));
                const float d32 = dt[qq][rr * 32 + lane];
                const double kth = __shfl_sync(FULL, ld[u], kappa - 1);
                // (a distance past FP32's range, or no number, is left to FP64)
                const bool need = valid && (!(d32 < 3.0e38f) || (double)d32 * (1.0 - (double)gam) <= kth);
                if (!__ballot_sync(FULL, need)) continue;
                double cd = DBL_MAX;
                int ci = INT_MAX;
                if (need) {
                    const float *xj = X + j * d;
                    double a = 0.0;
                    for (int k = 0; k < d; ++k) {
                        const double t = c_sub(c_f2d(xq[k]), c_f2d(xj[k]));
                        a = c_add(a, c_mul(t, t));
                    }
                    cd = a;
                    ci = (int)j;
                }
                warp_offer(ld[u], li[u], cd, ci, kappa, false, lane);
            }
        }
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const int64_t q = q0 + 8 * warp + u;
        if (q < Q) {
            const int64_t o = ((int64_t)blockIdx.y * Q + q) * 32 + lane;
            bd[o] = ld[u];
            bi[o] = li[u];
        }
    }
}

// Merge the splits' best-32 lists of each query (one warp per query) and
// write the kappa nearest.
__global__ void knn_merge_kernel(const double *bd, const int *bi, int64_t Q, int nsplit, int kappa,
                                 int32_t *ids, double *dist) {
    const int lane = threadIdx.x & 31;
    const int64_t q = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (q >= Q) return;                                   // warp-uniform
    double ld = DBL_MAX;
    int li = INT_MAX;
    for (int sp = 0; sp < nsplit; ++sp) {
        const int64_t o = ((int64_t)sp * Q + q) * 32 + lane;
        warp_offer(ld, li, bd[o], bi[o], kappa, false, lane);
    }
    if (lane < kappa) {
        ids[q * kappa + lane] = li;
        dist[q * kappa + lane] = ld;
    }
}

__global__ void knn_extract_kernel(const double *bd, const int *bi, int64_t Q, int kappa,
                                   int32_t *ids, double *dist) {
    int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= Q * kappa) return;
    int64_t q = t / kappa;
    int z = (int)(t % kappa);
    ids[t] = bi[q * 32 + z];
    dist[t] = bd[q * 32 + z];
}

__global__ void knn_dist_kernel(const float *X, int64_t N, int d, int kappa, const int32_t *ids,
                                double *dist) {
    int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= N * kappa) return;
    int64_t i = t / kappa;
    dist[t] = c_dist2(X + i * d, X + (int64_t)ids[t] * d, d);
}

// The sorted positions' segments and ids.
__global__ void seg_gather_kernel(const int32_t *pos, const int32_t *seg, const int32_t *order, int64_t n,
                                  uint32_t *skey, int32_t *ids) {
    const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (q >= n) return;
    skey[q] = (uint32_t)seg[pos[q]];
    ids[q] = order[pos[q]];
}

// Scratch shared by one tree build.
struct TreeScratch {
    int32_t *pos0 = nullptr, *pos1 = nullptr;
    uint32_t *skey0 = nullptr, *skey1 = nullptr;
    int32_t *seg = nullptr, *tmp_ids = nullptr, *bid = nullptr, *xl = nullptr;
    double *keys = nullptr, *keys_out = nullptr, *xc = nullptr, *Dq = nullptr;
    unsigned long long *bbits = nullptr;
    int32_t *lvl_start = nullptr, *lvl_end = nullptr, *lvl_size = nullptr;
    void *cub = nullptr;
    size_t cub_bytes = 0;
};

void free_scratch(TreeScratch &s) {
    cudaFree(s.pos0); cudaFree(s.pos1); cudaFree(s.skey0); cudaFree(s.skey1);
    cudaFree(s.seg); cudaFree(s.tmp_ids); cudaFree(s.bid); cudaFree(s.xl); cudaFree(s.keys);
    cudaFree(s.keys_out); cudaFree(s.xc); cudaFree(s.Dq); cudaFree(s.bbits); cudaFree(s.lvl_start);
    cudaFree(s.lvl_end); cudaFree(s.lvl_size); cudaFree(s.cub);
}

}  // namespace

int tree_depth(int64_t N, int64_t leaf) {
    int L = 0;
    while (((N + ((int64_t)1 << L) - 1) >> L) > leaf) ++L;
    return L;
}

void tree_ranges(int64_t N, int L, std::vector<int64_t> &start, std::vector<int64_t> &size) {
    int64_t nn = (int64_t)2 << L;
    start.assign(nn, 0);
    size.assign(nn, 0);
    size[1] = N;
    for (int64_t a = 1; a < ((int64_t)1 << L); ++a) {
        start[2 * a] = start[a];
        size[2 * a] = (size[a] + 1) / 2;
        start[2 * a + 1] = start[a] + (size[a] + 1) / 2;
        size[2 * a + 1] = size[a] / 2;
    }
}

// kind 0: ASKIT split (center, two farthest-point scans, line projection);
// kind 1: RP split (Rademacher direction of (seed, iter, node)).
askit_status build_tree_gpu(const float *X, int64_t N, int d, int L, int kind, uint64_t seed,
                            int iter, int32_t *order, cudaStream_t s) {
    std::vector<int64_t> st, sz;
    tree_ranges(N, L, st, sz);
    int64_t nn = (int64_t)2 << L;
    std::vector<int32_t> hs(nn), he(nn), hz(nn);
    for (int64_t a = 0; a < nn; ++a) {
        hs[a] = (int32_t)st[a];
        he[a] = (int32_t)(st[a] + sz[a]);
        hz[a] = (int32_t)sz[a];
    }
    TreeScratch sc;
    askit_status rc = ASKIT_OK;
    auto fail = [&](cudaError_t e, const char *what) {
        askit_set_error("tree build: %s: %s", what, cudaGetErrorString(e));
        rc = e == cudaErrorMemoryAllocation ? ASKIT_ERR_OOM : ASKIT_ERR_CUDA;
    };
#define TCHK(x, what) do { cudaError_t e_ = (x); if (e_ != cudaSuccess) { fail(e_, what); goto done; } } while (0)
    {
        int64_t half = (int64_t)1 << (L > 0 ? L - 1 : 0);
        TCHK(cudaMalloc(&sc.seg, sizeof(int32_t) * N), "alloc");
        TCHK(cudaMalloc(&sc.tmp_ids, sizeof(int32_t) * N), "alloc");
        TCHK(cudaMalloc(&sc.keys, sizeof(double) * N), "alloc");
        TCHK(cudaMalloc(&sc.keys_out, sizeof(double) * N), "alloc");
        TCHK(cudaMalloc(&sc.Dq, sizeof(double) * N), "alloc");
        TCHK(cudaMalloc(&sc.bid, sizeof(int32_t) * half), "alloc");
        TCHK(cudaMalloc(&sc.xl, sizeof(int32_t) * half), "alloc");
        TCHK(cudaMalloc(&sc.bbits, sizeof(unsigned long long) * half), "alloc");
        TCHK(cudaMalloc(&sc.xc, sizeof(double) * half * d), "alloc");
        TCHK(cudaMalloc(&sc.lvl_start, sizeof(int32_t) * nn), "alloc");
        TCHK(cudaMalloc(&sc.lvl_end, sizeof(int32_t) * nn), "alloc");
        TCHK(cudaMalloc(&sc.lvl_size, sizeof(int32_t) * nn), "alloc");
        TCHK(cudaMemcpyAsync(sc.lvl_start, hs.data(), sizeof(int32_t) * nn, cudaMemcpyHostToDevice, s), "copy");
        TCHK(cudaMemcpyAsync(sc.lvl_end, he.data(), sizeof(int32_t) * nn, cudaMemcpyHostToDevice, s), "copy");
        TCHK(cudaMemcpyAsync(sc.lvl_size, hz.data(), sizeof(int32_t) * nn, cudaMemcpyHostToDevice, s), "copy");
        // scratch for the largest segmented sort (all N keys, up to 2^L segments)
        size_t b1 = 0, b2 = 0;
        if ((rc = seg_sort_f64_i32(nullptr, nullptr, nullptr, nullptr, N, (int)half, nullptr, nullptr, nullptr, &b1, s)) != ASKIT_OK) goto done;
        if ((rc = seg_sort_i32(nullptr, nullptr, N, (int)(2 * half), nullptr, nullptr, nullptr, &b2, s)) != ASKIT_OK) goto done;
        sc.cub_bytes = b1 > b2 ? b1 : b2;
        if ((rc = sort_f64_i32(nullptr, nullptr, nullptr, nullptr, N, nullptr, &b1, s)) != ASKIT_OK) goto done;
        if ((rc = sort_u32_i32(nullptr, nullptr, nullptr, nullptr, N, 32, nullptr, &b2, s)) != ASKIT_OK) goto done;
        sc.cub_bytes = std::max(sc.cub_bytes, b1 > b2 ? b1 : b2);
        TCHK(cudaMalloc(&sc.pos0, sizeof(int32_t) * N), "alloc");
        TCHK(cudaMalloc(&sc.pos1, sizeof(int32_t) * N), "alloc");
        TCHK(cudaMalloc(&sc.skey0, sizeof(uint32_t) * N), "alloc");
        TCHK(cudaMalloc(&sc.skey1, sizeof(uint32_t) * N), "alloc");
        TCHK(cudaMalloc(&sc.cub, sc.cub_bytes), "alloc");

        iota_kernel<<<nblk(N, 256), 256, 0, s>>>(order, N);
        int id_bits = 1;
        while (((int64_t)1 << id_bits) < N) ++id_bits;
        for (int t = 0; t < L; ++t) {
            int64_t a0 = (int64_t)1 << t;
            int nseg = (int)a0;
            const int32_t *ls = sc.lvl_start + a0, *le = sc.lvl_end + a0, *lz = sc.lvl_size + a0;
            seg_of_pos_kernel<<<nblk(N, 256), 256, 0, s>>>(ls, nseg, N, sc.seg);
            if (kind == 0) {
                center_kernel<<<dim3(nseg, (d + 63) / 64), 64, 0, s>>>(X, d, order, ls, lz, sc.xc);
                // x_l: farthest from the center
                fill_kernel<unsigned long long><<<nblk(nseg, 256), 256, 0, s>>>(sc.bbits, nseg, 0ull);
                fill_kernel<int32_t><<<nblk(nseg, 256), 256, 0, s>>>(sc.bid, nseg, INT_MAX);
                far_pass1<true><<<nblk(N, 256), 256, 0, s>>>(X, d, order, sc.seg, N, sc.xc, nullptr, sc.Dq, sc.bbits);
                far_pass2<<<nblk(N, 256), 256, 0, s>>>(order, sc.seg, N, sc.Dq, sc.bbits, sc.bid);
                TCHK(cudaMemcpyAsync(sc.xl, sc.bid, sizeof(int32_t) * nseg, cudaMemcpyDeviceToDevice, s), "copy");
                // x_r: farthest from x_l
                fill_kernel<unsigned long long><<<nblk(nseg, 256), 256, 0, s>>>(sc.bbits, nseg, 0ull);
                fill_kernel<int32_t><<<nblk(nseg, 256), 256, 0, s>>>(sc.bid, nseg, INT_MAX);
                far_pass1<false><<<nblk(N, 256), 256, 0, s>>>(X, d, order, sc.seg, N, nullptr, sc.xl, sc.Dq, sc.bbits);
                far_pass2<<<nblk(N, 256), 256, 0, s>>>(order, sc.seg, N, sc.Dq, sc.bbits, sc.bid);
                proj_line_kernel<<<nblk(N, 256), 256, 0, s>>>(X, d, order, sc.seg, N, sc.xl, sc.bid, sc.keys);
            } else {
                proj_rp_kernel<<<nblk(N, 256), 256, 0, s>>>(X, d, order, sc.seg, N, a0, seed, iter, sc.keys);
            }
            TCHK(cudaGetLastError(), "projection kernels");
            if (N / nseg > TREE_RADIX) {
                // Few large segments: the segmented sort takes one block for each (a
                // 64K segment about 1 ms, a 1M one 16 ms), so the whole level is radix-
                // sorted by key, then stably by segment (the line: TREE_RADIX).
                iota_kernel<<<nblk(N, 256), 256, 0, s>>>(sc.pos0, N);
                if ((rc = sort_f64_i32(sc.keys, sc.keys_out, sc.pos0, sc.pos1, N, sc.cub, &sc.cub_bytes, s)) != ASKIT_OK) goto done;
                seg_gather_kernel<<<nblk(N, 256), 256, 0, s>>>(sc.pos1, sc.seg, order, N, sc.skey0, sc.pos0);
                if ((rc = sort_u32_i32(sc.skey0, sc.skey1, sc.pos0, sc.tmp_ids, N, t + 1, sc.cub, &sc.cub_bytes, s)) != ASKIT_OK) goto done;
                // children back to ascending id: by id, then stably by child
                seg_of_pos_kernel<<<nblk(N, 256), 256, 0, s>>>(sc.lvl_start + 2 * a0, 2 * nseg, N, sc.pos0);
                if ((rc = sort_u32_i32(reinterpret_cast<uint32_t *>(sc.tmp_ids), sc.skey0, sc.pos0, sc.pos1, N, id_bits, sc.cub, &sc.cub_bytes, s)) != ASKIT_OK) goto done;
                if ((rc = sort_u32_i32(reinterpret_cast<uint32_t *>(sc.pos1), sc.skey1, reinterpret_cast<int32_t *>(sc.skey0), order, N, t + 2, sc.cub, &sc.cub_bytes, s)) != ASKIT_OK) goto done;
                TCHK(cudaGetLastError(), "level sort");
                continue;
            }
            // (key, id) order inside every node: stable sort of an id-ascending segment
            if ((rc = seg_sort_f64_i32(sc.keys, sc.keys_out, order, sc.tmp_ids, N, nseg, ls, le, sc.cub, &sc.cub_bytes, s)) != ASKIT_OK) goto done;
            // children back to ascending id
            if ((rc = seg_sort_i32(sc.tmp_ids, order, N, 2 * nseg, sc.lvl_start + 2 * a0, sc.lvl_end + 2 * a0, sc.cub, &sc.cub_bytes, s)) != ASKIT_OK) goto done;
        }
        TCHK(cudaStreamSynchronize(s), "sync");
    }
done:
#undef TCHK
    cudaStreamSynchronize(s);
    free_scratch(sc);
    return rc;
}

namespace {
askit_status knn_lists_init(int64_t Q, double **bd, int **bi, cudaStream_t s) {
    ASK_CUDA(cudaMallocAsync(bd, sizeof(double) * Q * 32, s));
    ASK_CUDA(cudaMallocAsync(bi, sizeof(int) * Q * 32, s));
    fill_kernel<double><<<nblk(Q * 32, 256), 256, 0, s>>>(*bd, Q * 32, DBL_MAX);
    fill_kernel<int><<<nblk(Q * 32, 256), 256, 0, s>>>(*bi, Q * 32, INT_MAX);
    ASK_LAUNCH();
    return ASKIT_OK;
}
}  // namespace

// Exact kNN: every point (Y == nullptr, self excluded) or every row of Y
// against all N points.  Query tiles of 64 x candidate splits, chosen so that
// about four blocks per SM have work; the splits' lists are merged.
askit_status knn_exact_gpu(const float *X, int64_t N, int d, int kappa, const float *Y, int64_t Q,
                           int32_t *ids, double *dist, cudaStream_t s, const int32_t *self) {
    const int64_t nqb = (Q + KT_Q - 1) / KT_Q;
    int64_t nsplit = (4 * 152 + nqb - 1) / nqb;
    nsplit = std::max<int64_t>(1, std::min<int64_t>(nsplit, N / (4 * KT_C)));
    nsplit = std::min<int64_t>(nsplit, 65535);
    int64_t split_len = (N + nsplit - 1) / nsplit;
    split_len = (split_len + KT_C - 1) / KT_C * KT_C;
    nsplit = (N + split_len - 1) / split_len;
    double *bd = nullptr;
    int *bi = nullptr;
    cudaError_t e = cudaMallocAsync(&bd, sizeof(double) * nsplit * Q * 32, s);
    if (e == cudaSuccess) e = cudaMallocAsync(&bi, sizeof(int) * nsplit * Q * 32, s);
    if (e == cudaSuccess) {
        knn_tiled_kernel<<<dim3((unsigned)nqb, (unsigned)nsplit), 256, 0, s>>>(X, N, d, Y, Q, split_len, kappa, bd, bi,
                                                                               self);
        knn_merge_kernel<<<nblk(Q * 32, 256), 256, 0, s>>>(bd, bi, Q, (int)nsplit, kappa, ids, dist);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    askit_status rc = ASKIT_OK;
    if (e != cudaSuccess) {
        askit_set_error("exact kNN: %s", cudaGetErrorString(e));
        rc = ASKIT_ERR_CUDA;
    }
    if (bd) cudaFreeAsync(bd, s);
    if (bi) cudaFreeAsync(bi, s);
    return rc;
}

// RP-tree kNN (Section 2.2): iters trees; in each, every point searches its
// leaf exhaustively and the best kappa candidates are kept across trees.
askit_status knn_rp_gpu(const float *X, int64_t N, int d, int kappa, int iters, int64_t rp_leaf,
                        uint64_t seed, int32_t *ids, double *dist, cudaStream_t s) {
    int L = tree_depth(N, rp_leaf);
    std::vector<int64_t> st, sz;
    tree_ranges(N, L, st, sz);
    int64_t nleaf = (int64_t)1 << L;
    std::vector<int32_t> h(2 * nleaf);
    for (int64_t a = 0; a < nleaf; ++a) {
        h[a] = (int32_t)st[nleaf + a];
        h[nleaf + a] = (int32_t)(st[nleaf + a] + sz[nleaf + a]);
    }
    const int64_t max_leaf = sz[nleaf];                    // the first leaf is the largest
    static std::atomic<uint64_t> opted{0};
    ASK_TRY(opt_in_smem(knn_leaf_kernel, KL_SMEM, opted));
    double *bd = nullptr;
    int *bi = nullptr;
    int32_t *order = nullptr, *segs = nullptr;
    askit_status rc = knn_lists_init(N, &bd, &bi, s);
    cudaError_t e = cudaSuccess;
    if (rc == ASKIT_OK) {
        e = cudaMalloc(&order, sizeof(int32_t) * N);
        if (e == cudaSuccess) e = cudaMalloc(&segs, sizeof(int32_t) * 2 * nleaf);
        if (e == cudaSuccess) e = cudaMemcpyAsync(segs, h.data(), sizeof(int32_t) * 2 * nleaf, cudaMemcpyHostToDevice, s);
    }
    for (int it = 0; rc == ASKIT_OK && e == cudaSuccess && it < iters; ++it) {
        rc = build_tree_gpu(X, N, d, L, 1, seed, it, order, s);
        if (rc != ASKIT_OK) break;
        knn_leaf_kernel<<<(unsigned)(nleaf * nblk(max_leaf, KL_Q)), 256, KL_SMEM, s>>>(
            X, d, order, segs, segs + nleaf, (unsigned)nleaf, kappa, bd, bi);
        e = cudaGetLastError();
    }
    if (rc == ASKIT_OK && e == cudaSuccess) {
        knn_extract_kernel<<<nblk(N * kappa, 256), 256, 0, s>>>(bd, bi, N, kappa, ids, dist);
        e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    }
    if (rc == ASKIT_OK && e != cudaSuccess) {
        askit_set_error("RP kNN: %s", cudaGetErrorString(e));
        rc = ASKIT_ERR_CUDA;
    }
    cudaFreeAsync(bd, s); cudaFreeAsync(bi, s); cudaFree(order); cudaFree(segs);
    return rc;
}

askit_status knn_dist_gpu(const float *X, int64_t N, int d, int kappa, const int32_t *ids,
                          double *dist, cudaStream_t s) {
    knn_dist_kernel<<<nblk(N * kappa, 256), 256, 0, s>>>(X, N, d, kappa, ids, dist);
    ASK_LAUNCH();
    return ASKIT_OK;
}

// ---------------------------------------------------------------------------
// Allocation-free exact kNN (askit_knn_noalloc).
//
// The per-query best-32 lists live in this file-scope device array instead
// of memory from cudaMalloc: KNN_NOALLOC_MAX_Q queries x 32 slots x (8-byte
// distance + 4-byte id) = 3 MiB, held by every GPU that loads the library
// until the process exits.  Every call reuses it, so each call first resets
// the lists it uses, and calls that overlap on the GPU (on different
// streams, or from different threads) race on it.
// ---------------------------------------------------------------------------
namespace {

constexpr int64_t KNN_NOALLOC_MAX_Q = 8192;
constexpr int KNN_NOALLOC_QPB = 64;   // queries per block
static __device__ __align__(256) unsigned char g_knn_scratch[KNN_NOALLOC_MAX_Q * 32 * (sizeof(double) + sizeof(int))];

// Host-side address of g_knn_scratch on each device (the array's name is
// only a host stand-in; kernels must be given the device address).
std::mutex g_knn_scratch_mu;
void *g_knn_scratch_dev[64] = {nullptr};

askit_status knn_scratch_address(void **out) {
    int dev = 0;
    ASK_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) {
        askit_set_error("device ordinal %d out of range for the allocation-free kNN", dev);
        return ASKIT_ERR_UNSUPPORTED;
    }
    std::lock_guard<std::mutex> lock(g_knn_scratch_mu);
    if (!g_knn_scratch_dev[dev]) {
        void *p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_knn_scratch);
        if (e != cudaSuccess || !p) {
            askit_set_error("cudaGetSymbolAddress(knn scratch): %s", cudaGetErrorString(e));
            return ASKIT_ERR_CUDA;
        }
        g_knn_scratch_dev[dev] = p;
    }
    *out = g_knn_scratch_dev[dev];
    return ASKIT_OK;
}

// Exhaustive search of all N points for queries [64 b, 64 b + 64): one warp
// per query; Y == nullptr means the queries are the points themselves (self
// excluded).  Same FP64 distance and (D, id) order as the setup's kNN.
__global__ void knn_noalloc_kernel(const float *X, int64_t N, int d, const float *Y, int64_t Q, double *bd,
                                   int *bi, int kappa) {
    extern __shared__ float sq[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int64_t q0 = (int64_t)blockIdx.x * KNN_NOALLOC_QPB;
    const int64_t q1 = q0 + KNN_NOALLOC_QPB < Q ? q0 + KNN_NOALLOC_QPB : Q;
    float *myq = sq + (int64_t)warp * d;
    for (int64_t q = q0 + warp; q < q1; q += nw) {
        const int64_t self = Y ? -1 : q;
        const float *xq = Y ? Y + q * d : X + q * d;
        for (int k = lane; k < d; k += 32) myq[k] = xq[k];
        __syncwarp();
        double ld = bd[q * 32 + lane];
        int li = bi[q * 32 + lane];
        for (int64_t cb = 0; cb < N; cb += 32) {
            double cd = DBL_MAX;
            int ci = INT_MAX;
            if (cb + lane < N && cb + lane != self) {
                const float *xj = X + (cb + lane) * d;
                double acc = 0.0;
                for (int k = 0; k < d; ++k) {
                    double t = c_sub(c_f2d(myq[k]), c_f2d(xj[k]));
                    acc = c_add(acc, c_mul(t, t));
                }
                cd = acc;
                ci = (int)(cb + lane);
            }
            warp_offer(ld, li, cd, ci, kappa, false, lane);
        }
        bd[q * 32 + lane] = ld;
        bi[q * 32 + lane] = li;
        __syncwarp();
    }
}

}  // namespace

extern "C" askit_status askit_knn_noalloc(const float *X_dev, int64_t N, int32_t d, const float *Y_dev, int64_t Q,
                                          int32_t kappa, int32_t *ids_dev, double *dist_dev, void *stream) {
    if (!X_dev || !ids_dev || !dist_dev) {
        askit_set_error("X_dev, ids_dev and dist_dev must be non-NULL");
        return ASKIT_ERR_INVALID_ARG;
    }
    if (N < 1 || d < 1 || Q < 1 || kappa < 1 || kappa > 32) {
        askit_set_error("need N >= 1, d >= 1, Q >= 1 and 1 <= kappa <= 32");
        return ASKIT_ERR_INVALID_ARG;
    }
    if (N >= ((int64_t)1 << 31) - 1024) {   // ids are int32 (the setup's bound)
        askit_set_error("askit_knn_noalloc handles N below 2^31 - 1024");
        return ASKIT_ERR_UNSUPPORTED;
    }
    if (Q > KNN_NOALLOC_MAX_Q) {
        askit_set_error("askit_knn_noalloc handles at most %lld queries per call (got %lld)",
                        (long long)KNN_NOALLOC_MAX_Q, (long long)Q);
        return ASKIT_ERR_INVALID_ARG;
    }
    if (!Y_dev && Q != N) {
        askit_set_error("with Y_dev == NULL the queries are the N points: Q must equal N");
        return ASKIT_ERR_INVALID_ARG;
    }
    if (kappa > (Y_dev ? N : N - 1)) {
        askit_set_error("kappa exceeds the number of candidate neighbors");
        return ASKIT_ERR_INVALID_ARG;
    }
    if ((size_t)8 * d * sizeof(float) > 48 * 1024) {
        askit_set_error("askit_knn_noalloc handles d <= %d", (int)(48 * 1024 / (8 * sizeof(float))));
        return ASKIT_ERR_UNSUPPORTED;
    }
    void *scratch = nullptr;
    ASK_TRY(knn_scratch_address(&scratch));
    double *bd = static_cast<double *>(scratch);
    int *bi = reinterpret_cast<int *>(bd + KNN_NOALLOC_MAX_Q * 32);
    cudaStream_t s = (cudaStream_t)stream;
    // the array keeps the previous call's lists: reset the ones used here
    fill_kernel<double><<<nblk(Q * 32, 256), 256, 0, s>>>(bd, Q * 32, DBL_MAX);
    fill_kernel<int><<<nblk(Q * 32, 256), 256, 0, s>>>(bi, Q * 32, INT_MAX);
    knn_noalloc_kernel<<<(unsigned)((Q + KNN_NOALLOC_QPB - 1) / KNN_NOALLOC_QPB), 256, 8 * d * sizeof(float), s>>>(
        X_dev, N, d, Y_dev, Q, bd, bi, kappa);
    knn_extract_kernel<<<nblk(Q * kappa, 256), 256, 0, s>>>(bd, bi, Q, kappa, ids_dev, dist_dev);
    ASK_LAUNCH();
    return ASKIT_OK;
}
