// Skeletonization on the GPU (Sections 2.1-2.2, Algorithms 2 and 3).
//
//  * Node neighbor lists (Algorithm 2): a leaf collects its points' kNN
//    entries outside the leaf, an internal node its children's lists minus
//    its own points; each id keeps its smallest recorded distance, the list
//    is ordered by (distance, id) and truncated to ell = s_max + ell_extra.
//  * Sampled targets (eq. (2.4)): the list, then uniform draws without
//    replacement outside the node and the list (Philox stream of the node).
//  * ID (Section 2.1): FP64 kernel block K(T_a, C_a), Householder QR with
//    column pivoting on recomputed trailing norms, rank by |R_kk| <= tol
//    |R_00| within [s_min, s_max], P = R11^{-1} R12 by back substitution.
// Every FP64 operation is explicitly rounded and sequenced so the lists,
// pivots and skeletons reproduce bit for bit on any IEEE machine.
#include <float.h>
#include <limits.h>

#include <algorithm>

#include "askit_impl.cuh"

namespace {

inline unsigned nblk(int64_t n, int b) { return (unsigned)((n + b - 1) / b); }

__device__ __forceinline__ bool in_subtree(int32_t leaf, int64_t a, int L, int depth_a) {
    return ((int64_t)leaf >> (L - depth_a)) == a;
}

// Leaf-level candidates: entry (q, z) of tree position q is the z-th
// neighbor of point perm[q]; neighbors inside the point's own leaf are
// removed (id INT_MAX, key DBL_MAX).
__global__ void leaf_cand_kernel(const int32_t *perm, const int32_t *leafof, const int32_t *knn,
                                 const double *knnd, int64_t N, int kappa, int32_t *cj, double *ck) {
    int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= N * kappa) return;
    int64_t q = e / kappa;
    int z = (int)(e % kappa);
    int32_t i = perm[q];
    int32_t j = knn[(int64_t)i * kappa + z];
    if (leafof[j] == leafof[i]) {
        cj[e] = INT_MAX;
        ck[e] = DBL_MAX;
    } else {
        cj[e] = j;
        ck[e] = knnd[(int64_t)i * kappa + z];
    }
}

// Internal-level candidates: node a = a0 + g takes both children's lists,
// removing ids inside a.  Slots [g * 2 ell, (g + 1) * 2 ell).
__global__ void inner_cand_kernel(int64_t a0, int ngroups, int ell, int L, int depth,
                                  const int32_t *leafof, const int32_t *nl_cnt, const int32_t *nl_ids,
                                  const double *nl_key, int32_t *cj, double *ck) {
    int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= (int64_t)ngroups * 2 * ell) return;
    int64_t g = e / (2 * ell);
    int slot = (int)(e % (2 * ell));
    int64_t a = a0 + g;
    int64_t ch = 2 * a + (slot >= ell);
    int q = slot % ell;
    int32_t j = INT_MAX;
    double k = DBL_MAX;
    if (q < nl_cnt[ch]) {
        int32_t jj = nl_ids[ch * ell + q];
        if (!in_subtree(leafof[jj], a, L, depth)) {
            j = jj;
            k = nl_key[ch * ell + q];
        }
    }
    cj[e] = j;
    ck[e] = k;
}

// After a stable sort by id: the first entry of each id group carries the
// group's smallest key; the rest are removed.  Counts survivors per segment.
__global__ void dedupe_kernel(const int32_t *sj, const double *sk, int32_t *oj, double *ok,
                              const int32_t *seg_of, const int32_t *seg_beg, int64_t n,
                              int32_t *seg_cnt) {
    int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= n) return;
    int32_t j = sj[e];
    int g = seg_of[e];
    bool first = (j != INT_MAX) && (e == seg_beg[g] || sj[e - 1] != j);
    if (!first) {
        oj[e] = INT_MAX;
        ok[e] = DBL_MAX;
        return;
    }
    double m = sk[e];
    int64_t end = n;
    for (int64_t f = e + 1; f < end && sj[f] == j && seg_of[f] == g; ++f) m = fmin(m, sk[f]);
    oj[e] = j;
    ok[e] = m;
    atomicAdd(seg_cnt + g, 1);
}

__global__ void seg_of_kernel(const int32_t *beg, const int32_t *end, int nseg, int32_t *seg_of) {
    int g = blockIdx.x;
    if (g >= nseg) return;
    for (int64_t e = beg[g] + threadIdx.x; e < end[g]; e += blockDim.x) seg_of[e] = g;
}

__global__ void nl_write_kernel(int64_t a0, int nseg, const int32_t *beg, const int32_t *sj,
                                const double *sk, const int32_t *cnt, int ell, int32_t *nl_cnt,
                                int32_t *nl_ids, double *nl_key) {
    int g = blockIdx.x;
    if (g >= nseg) return;
    int64_t a = a0 + g;
    int c = min(cnt[g], ell);
    if (threadIdx.x == 0) nl_cnt[a] = c;
    for (int q = threadIdx.x; q < ell; q += blockDim.x) {
        nl_ids[a * ell + q] = q < c ? sj[beg[g] + q] : -1;
        nl_key[a * ell + q] = q < c ? sk[beg[g] + q] : 0.0;
    }
}

// Sampled targets of node a (one thread per node): T_a = the first
// min(|N_a|, ell_a) list entries, then draw n gives j = floor(u N / 2^32)
// with u the top 32 bits of Philox word n keyed (seed, 0), counter (a, n/4);
// rejected inside a, in the list or already drawn.
__global__ void sample_kernel(int64_t n_nodes, int64_t N, int L, int ell, const int32_t *nsize,
                              const int32_t *leafof, const int32_t *nl_cnt, const int32_t *nl_ids,
                              uint64_t seed, int32_t *trows) {
    int64_t a = 2 + blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (a >= n_nodes) return;
    int depth = heap_depth(a);
    int64_t ell_a = (N - nsize[a] < ell) ? N - nsize[a] : ell;
    int32_t *rows = trows + a * ell;
    int nr = min(nl_cnt[a], (int)ell_a);
    for (int q = 0; q < nr; ++q) rows[q] = nl_ids[a * ell + q];
    for (uint64_t draw = 0; nr < ell_a; ++draw) {
        uint64_t w = philox_word(seed, 0, (uint64_t)a, draw);
        int32_t j = (int32_t)(((w >> 32) * (uint64_t)N) >> 32);
        if (in_subtree(leafof[j], a, L, depth)) continue;
        bool seen = false;
        for (int q = 0; q < nr && !seen; ++q) seen = (rows[q] == j);
        if (seen) continue;
        rows[nr++] = j;
    }
    for (int q = nr; q < ell; ++q) rows[q] = -1;
}

// Columns of each node of a level: leaf points in tree order (ascending id)
// or the children's skeletons (left then right, pivot order).
__global__ void cols_kernel(int64_t a0, int nseg, bool leaf_level, const int32_t *perm,
                            const int32_t *nstart, const int32_t *nsize, const int32_t *skel_fixed,
                            const int32_t *s, int s_max, int cmax, int32_t *cols) {
    int g = blockIdx.x;
    if (g >= nseg) return;
    int64_t a = a0 + g;
    int32_t *out = cols + (int64_t)g * cmax;
    if (leaf_level) {
        for (int q = threadIdx.x; q < nsize[a]; q += blockDim.x) out[q] = perm[nstart[a] + q];
    } else {
        int sl = s[2 * a], sr = s[2 * a + 1];
        for (int q = threadIdx.x; q < sl + sr; q += blockDim.x)
            out[q] = q < sl ? skel_fixed[(2 * a) * s_max + q] : skel_fixed[(2 * a + 1) * s_max + (q - sl)];
    }
}

// K(T_a, C_a) with the canonical exp: entry (i, q) = exp(-(c D) / h_q^2).
__global__ void fill_kernel(const float *X, int d, const float *hsrc, double kscale, int64_t a0,
                            const int32_t *batch_nodes, const int64_t *woff, const int32_t *ncol,
                            const int32_t *ellv, const int32_t *trows, int ell, const int32_t *cols,
                            int cmax, double *work) {
    int g = blockIdx.y;
    int64_t a = batch_nodes[g];
    int c = ncol[a], rows = ellv[a];
    int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= (int64_t)rows * c) return;
    int i = (int)(e / c), q = (int)(e % c);
    int32_t ri = trows[a * ell + i];
    int32_t cq = cols[(a - a0) * cmax + q];
    double D = c_dist2(X + (int64_t)ri * d, X + (int64_t)cq * d, d);
    double h = (double)hsrc[cq];
    double arg = c_div(c_mul(kscale, D), c_mul(h, h));
    work[woff[g] + e] = c_exp(-arg);
}

// Column-pivoted Householder QR of one node's block and the interpolation
// matrix P = R11^{-1} R12, a cluster of C CTAs per node.  At step k the pivot is the
// column with the largest trailing squared norm (recomputed; ties to the smallest
// position), |R_kk| is its norm, the reflector is H = I - tau v v^T with v_k = 1 and
// beta = -sign(alpha) ||x||.
//
// Bound by FP64: a warp instruction takes 64 cycles of its quarter of the SM (76 with
// all four quarters busy) whatever its active lanes, and as long to be used.  Three
// things follow.
// (1) A step needs the products with v and the update (4 operations an element);
// the trailing norms (2 more) are needed exactly only for the columns that can be
// the pivot.  The update therefore also sums each column's norm in FP32 (elements
// taken from the double's bits, scaled by the last pivot's exponent, no FP64
// instruction), and only columns within the sum's error bound of the largest get
// their canonical FP64 norm.  (2) A level with fewer nodes than SMs spreads each
// node over a cluster: 32-column groups are dealt to the CTAs' warps in turn, so
// that the columns left are shared evenly at every step.  The block stays in
// L2; rows written by another CTA are read past L1.  (3) A lone candidate's norm
// takes the warp's lanes for its products, and a step's square root and divisions
// one warp.
// All levels: 64K x 64, s = 256 (7 levels) 318 -> 125 ms; 10K x 1000, s = 1024 (6
// levels) 5.7 -> 1.1 s; 1M x 64 (11 levels) 1.7 -> 1.1 s of skeletons.
constexpr int QR_THREADS = 512;
constexpr int QR_WARPS = QR_THREADS / 32;

__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// Stores v at `p` (an address of this CTA's shared memory) in CTA `rank`.
__device__ __forceinline__ void cluster_store(uint64_t *p, uint32_t rank, uint64_t v) {
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
    uint32_t ra;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a), "r"(rank));
    asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(ra), "l"(v) : "memory");
}

// |a| 2^-e as a float, truncated (e: the exponent of a bound of |a|); lim =
// max(897 + e, 1) << 20 cuts what would be below the smallest normal float.
__device__ __forceinline__ float scaled_abs(double a, int base, int lim) {
    const int hi = __double2hiint(a) & 0x7fffffff;
    return hi < lim ? 0.f : __uint_as_float(((uint32_t)(hi - base) << 3) | ((uint32_t)__double2loint(a) >> 29));
}

// f(i, x, p) for rows i .. rows - 1 of a column (p: its element of row i, rows
// `cols` apart), eight loads at a time; AHEAD: the next eight in flight during these.
template <bool AHEAD, class L, class F>
__device__ __forceinline__ void walk_column(double *p, int64_t cols, int i, int rows, L ld, F f) {
    double x[8];
    if (AHEAD && i + 8 <= rows) {
#pragma unroll
        for (int u = 0; u < 8; ++u) x[u] = ld(p + u * cols);
    }
    for (; i + 8 <= rows; i += 8, p += 8 * cols) {
        double y[8];
        if (AHEAD) {
            const bool more = i + 16 <= rows;
#pragma unroll
            for (int u = 0; u < 8; ++u) y[u] = more ? ld(p + (8 + u) * cols) : 0.0;
        } else {
#pragma unroll
            for (int u = 0; u < 8; ++u) x[u] = ld(p + u * cols);
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) f(i + u, x[u], p + u * cols);
        if (AHEAD) {
#pragma unroll
            for (int u = 0; u < 8; ++u) x[u] = y[u];
        }
    }
    for (; i < rows; ++i, p += cols) f(i, ld(p), p);
}

// With two or four CTAs a node a column's chain is short of warps to hide the loads
// behind, so they run ahead, at one CTA an SM; clusters of eight CTAs that each need
// an SM do not all fit the GPCs at once (16 nodes: two waves), so those stay at two.
template <int C>
constexpr bool QR_AHEAD = C == 2 || C == 4;

template <int C>
__global__ void __launch_bounds__(QR_THREADS, QR_AHEAD<C> ? 1 : 2) cpqr_kernel(
    const int32_t *batch_nodes, const int64_t *woff, const int64_t *poff_ws, const int32_t *ncol,
    const int32_t *ellv, double tol, int s_min, int s_max, double *work, int32_t *piv_fixed,
    int cmax, int32_t *s_out) {
    extern __shared__ double sh[];           // v[rows], then float nf[this CTA's columns]
    __shared__ double red_v[QR_WARPS];
    __shared__ int red_j[QR_WARPS];
    __shared__ float red_f[QR_WARPS];
    __shared__ double st_nrm, st_beta, st_tau, st_scal;      // the step's scalars
    __shared__ int st_p;
    // the CTAs' results of a reduction (slot = rank): largest FP32 norm; norm and position
    __shared__ uint64_t x_f[C], x_v[C], x_j[C];
    const int g = blockIdx.x / C, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const uint32_t rank = C > 1 ? cluster_rank() : 0;
    const int64_t a = batch_nodes[g];
    const int cols = ncol[a], rows = ellv[a];
    double *A = work + woff[g];
    double *P = work + poff_ws[g];
    int32_t *piv = piv_fixed + a * cmax;
    double *v = sh;
    float *nf = reinterpret_cast<float *>(sh + rows);
    const int s_hi = min(min(s_max, cols), rows);
    const int s_lo = min(min(s_min, cols), s_hi);
    auto sync_all = [&]() {
        __syncwarp();
        if (C > 1) cluster_sync();
        else __syncthreads();
    };
    // column groups of this warp: blk = wid C + rank, every QR_WARPS C; local slot
    // of a group's FP32 norms: 32 (blk / C)
    const int blk0 = wid * C + (int)rank;
    auto ld = [&](const double *p) { return C > 1 ? __ldcg(p) : *p; };
    auto norm_of = [&](int j, int k) {
        double acc = 0.0;
        walk_column<QR_AHEAD<C>>(A + (int64_t)k * cols + j, cols, k, rows, ld,
                             [&](int, double x, double *) { acc = c_add(acc, c_mul(x, x)); });
        return acc;
    };
    // the same sum with the whole warp on one column: 32 products an instruction,
    // then one chain of additions
    auto norm_of_one = [&](int j, int k) {
        double acc = 0.0;
        auto row = [&](int i) { return i + lane < rows ? ld(A + (int64_t)(i + lane) * cols + j) : 0.0; };
        double x = row(k);
        for (int i = k; i < rows; i += 32) {
            const double next = row(i + 32), xx = c_mul(x, x);
            const int n = min(32, rows - i);
            for (int u = 0; u < n; ++u) acc = c_add(acc, __shfl_sync(0xffffffffu, xx, u));
            x = next;
        }
        return acc;
    };
    if (rank == 0)
        for (int j = tid; j < cols; j += QR_THREADS) piv[j] = j;
    // the bound of an FP32 norm's relative error: `rows` truncated elements, squared
    // and added in order
    const float rel = (float)(rows + 8) * 2.4e-7f;
    double r00 = 0.0;                                     // (the first warp's)
    int s = s_hi;
    bool have_nf = false;
    for (int k = 0; k < s_hi; ++k) {
        // the columns that can be the pivot: all at the first step
        float thr = -1.f;
        if (have_nf) {
            float m = -1.f;
            for (int blk = blk0; blk * 32 < cols; blk += QR_WARPS * C) {
                const int j = blk * 32 + lane;
                if (j >= k && j < cols) m = fmaxf(m, nf[32 * (blk / C) + lane]);
            }
            for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
            if (lane == 0) red_f[wid] = m;
            __syncthreads();
            if (wid == 0) {
                m = lane < QR_WARPS ? red_f[lane] : -1.f;
                for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
                if (C > 1) {
                    if (lane < C) cluster_store(&x_f[rank], lane, (uint64_t)__float_as_uint(m));
                } else if (lane == 0) {
                    x_f[0] = (uint64_t)__float_as_uint(m);
                }
            }
            sync_all();
            m = -1.f;
#pragma unroll
            for (int c = 0; c < C; ++c) m = fmaxf(m, __uint_as_float((uint32_t)x_f[c]));
            // (sums this small may have lost terms to the float range: all columns)
            thr = m < 1e-25f ? -1.f : m * (1.f - rel);
        }
        double best = -1.0;
        int bj = INT_MAX;
        for (int blk = blk0; blk * 32 < cols; blk += QR_WARPS * C) {
            const int j = blk * 32 + lane;
            const bool can = j >= k && j < cols && (!have_nf || nf[32 * (blk / C) + lane] >= thr);
            const unsigned m = __ballot_sync(0xffffffffu, can);
            double acc = -1.0;
            if (__popc(m) == 1) {
                const double one = norm_of_one(blk * 32 + __ffs(m) - 1, k);
                if (can) acc = one;
            } else if (can) {
                acc = norm_of(j, k);
            }
            __syncwarp();
            if (acc > best) { best = acc; bj = j; }       // j increases: ties keep the smaller
        }
        for (int o = 16; o > 0; o >>= 1) {
            double ob = __shfl_xor_sync(0xffffffffu, best, o);
            int oj = __shfl_xor_sync(0xffffffffu, bj, o);
            if (ob > best || (ob == best && oj < bj)) { best = ob; bj = oj; }
        }
        if (lane == 0) { red_v[wid] = best; red_j[wid] = bj; }
        __syncthreads();
        if (wid == 0) {
            best = lane < QR_WARPS ? red_v[lane] : -1.0;
            bj = lane < QR_WARPS ? red_j[lane] : INT_MAX;
            for (int o = 16; o > 0; o >>= 1) {
                double ob = __shfl_xor_sync(0xffffffffu, best, o);
                int oj = __shfl_xor_sync(0xffffffffu, bj, o);
                if (ob > best || (ob == best && oj < bj)) { best = ob; bj = oj; }
            }
            if (C > 1) {
                // (every warp instruction in FP64 costs 64 cycles, so nothing below
                // is computed by more than one warp a CTA)
                if (lane < C) {
                    cluster_store(&x_v[rank], lane, (uint64_t)__double_as_longlong(best));
                    cluster_store(&x_j[rank], lane, (uint64_t)(uint32_t)bj);
                }
            } else if (lane == 0) {
                x_v[0] = (uint64_t)__double_as_longlong(best);
                x_j[0] = (uint64_t)(uint32_t)bj;
            }
        }
        sync_all();
        if (wid == 0) {
            best = __longlong_as_double((long long)x_v[0]);
            int p = (int)(uint32_t)x_j[0];
#pragma unroll
            for (int c = 1; c < C; ++c) {
                const double ob = __longlong_as_double((long long)x_v[c]);
                const int oj = (int)(uint32_t)x_j[c];
                if (ob > best || (ob == best && oj < p)) { best = ob; p = oj; }
            }
            const double nrm = __dsqrt_rn(best);
            if (k == 0) r00 = nrm;
            const bool stop = p == INT_MAX || nrm == 0.0 || (k >= s_lo && nrm <= c_mul(tol, r00));
            if (!stop) {
                const double alpha = ld(A + (int64_t)k * cols + p);
                const double beta = (alpha >= 0.0) ? -nrm : nrm;
                const double tau = c_div(c_sub(beta, alpha), beta);
                if (lane == 0) {
                    st_nrm = nrm;
                    st_beta = beta;
                    st_tau = tau;
                    st_scal = c_sub(alpha, beta);
                }
            }
            if (lane == 0) st_p = stop ? -1 : p;
        }
        __syncthreads();
        const int p = st_p;
        if (p < 0) { s = k; break; }
        const double nrm = st_nrm, beta = st_beta, tau = st_tau, scal = st_scal;
        // v from the pivot column where it is; then columns k and p change places
        // (the first CTA), the new column k's part below the diagonal becomes zero
        for (int i = k + 1 + tid; i < rows; i += QR_THREADS) v[i] = c_div(ld(A + (int64_t)i * cols + p), scal);
        if (tid == 0) v[k] = 1.0;
        sync_all();                                       // every CTA has read column p
        if (rank == 0) {
            for (int i = tid; i < rows; i += QR_THREADS) {
                double *row = A + (int64_t)i * cols;
                const double xk = ld(row + k), xp = ld(row + p);
                row[k] = i < k ? xp : i == k ? beta : 0.0;
                if (p != k) row[p] = xk;
            }
            if (tid == 0 && p != k) { int t = piv[k]; piv[k] = piv[p]; piv[p] = t; }
        }
        sync_all();
        // exponent of the norms' bound: every trailing element is at most nrm
        const int e = (int)((__double2hiint(nrm) >> 20) & 0x7ff) - 1023;
        const int base = (896 + e) * (1 << 20), lim = max(897 + e, 1) << 20;
        for (int blk = blk0; blk * 32 < cols; blk += QR_WARPS * C) {
            const int j = blk * 32 + lane;
            if (j <= k || j >= cols) continue;
            double dot = 0.0;
            double *p0 = A + (int64_t)k * cols + j;
            walk_column<QR_AHEAD<C>>(p0, cols, k, rows, ld,
                                 [&](int i, double x, double *) { dot = c_add(dot, c_mul(v[i], x)); });
            const double tdot = c_mul(tau, dot);
            float f = 0.f;
            bool bad = false;
            walk_column<QR_AHEAD<C>>(p0, cols, k, rows, ld, [&](int i, double x, double *dst) {
                const double y = c_sub(x, c_mul(tdot, v[i]));
                *dst = y;
                const float t = scaled_abs(y, base, lim);
                bad |= (__double2hiint(y) & 0x7ff00000) == 0x7ff00000;
                if (i > k) f = fmaf(t, t, f);
            });
            nf[32 * (blk / C) + lane] = bad ? -1.f : f;   // a column that is not finite is never a pivot
        }
        have_nf = true;
        sync_all();
    }
    sync_all();
    const int nr = cols - s;
    for (int blk = blk0; blk * 32 < nr; blk += QR_WARPS * C) {
        const int j = blk * 32 + lane;
        if (j >= nr) continue;
        for (int i = s - 1; i >= 0; --i) {
            double acc = ld(A + (int64_t)i * cols + (s + j));
            const double *ai = A + (int64_t)i * cols;
            int t = i + 1;
            double x[8], y[8];
            auto rows8 = [&](int t0, double (&xx)[8], double (&yy)[8]) {
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    xx[u] = ld(ai + t0 + u);
                    yy[u] = P[(int64_t)(t0 + u) * nr + j];
                }
            };
            if (QR_AHEAD<C> && t + 8 <= s) rows8(t, x, y);
            for (; t + 8 <= s; t += 8) {
                double xn[8], yn[8];
                if (QR_AHEAD<C>) {
                    if (t + 16 <= s) rows8(t + 8, xn, yn);
                } else {
                    rows8(t, x, y);
                }
#pragma unroll
                for (int u = 0; u < 8; ++u) acc = c_sub(acc, c_mul(x[u], y[u]));
                if (QR_AHEAD<C>) {
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        x[u] = xn[u];
                        y[u] = yn[u];
                    }
                }
            }
            for (; t < s; ++t) acc = c_sub(acc, c_mul(ld(ai + t), P[(int64_t)t * nr + j]));
            P[(int64_t)i * nr + j] = c_div(acc, ld(ai + i));
        }
    }
    if (rank == 0 && tid == 0) s_out[a] = s;
    __syncwarp();
    if (C > 1) cluster_sync();                            // no CTA leaves while another may store to it
}

template <int C>
askit_status launch_cpqr(int nb, size_t smem, cudaStream_t s, const int32_t *nodes, const int64_t *woff,
                         const int64_t *pws, askit_tree t, const int32_t *ell, int s_max, double *work, int32_t *piv,
                         int cmax) {
    // the most a block can have, whatever this launch takes: setups of several threads
    // share the attribute
    static std::atomic<uint64_t> opted{0};
    cudaFuncAttributes fa;
    int dev = 0, most = 0;
    ASK_CUDA(cudaFuncGetAttributes(&fa, cpqr_kernel<C>));
    ASK_CUDA(cudaGetDevice(&dev));
    ASK_CUDA(cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    ASK_TRY(opt_in_smem(cpqr_kernel<C>, (size_t)most - fa.sharedSizeBytes, opted));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(nb * C));
    cfg.blockDim = dim3(QR_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = C;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    ASK_CUDA(cudaLaunchKernelEx(&cfg, cpqr_kernel<C>, nodes, woff, pws, (const int32_t *)t->d_ncol, ell, t->prm.id_tol,
                                (int)t->prm.s_min, s_max, work, piv, cmax, t->d_s));
    return ASKIT_OK;
}

// Skeleton ids of the batch's nodes (first s pivots) and P into the level pool.
__global__ void skel_out_kernel(const int32_t *batch_nodes, int64_t a0, const int64_t *poff_ws,
                                const int64_t *poff_lvl, const int32_t *s, const int32_t *ncol,
                                const int32_t *cols, int cmax, const int32_t *piv_fixed, int s_max,
                                const double *work, int32_t *skel_fixed, double *P64) {
    int g = blockIdx.x;
    int64_t a = batch_nodes[g];
    int sa = s[a], c = ncol[a];
    for (int q = threadIdx.x; q < sa; q += blockDim.x)
        skel_fixed[a * s_max + q] = cols[(a - a0) * cmax + piv_fixed[a * cmax + q]];
    int64_t np = (int64_t)sa * (c - sa);
    for (int64_t e = threadIdx.x; e < np; e += blockDim.x) P64[poff_lvl[g] + e] = work[poff_ws[g] + e];
}

// The FP32 copy of P the upward pass reads: node a = 2 + block, rows padded
// with zeros to a multiple of 4 columns.
__global__ void p32_kernel(const double *P64, const int64_t *poff, const int64_t *p32off, const int32_t *s,
                           const int32_t *ncol, float *P32) {
    const int64_t a = 2 + blockIdx.x;
    const int sa = s[a], nr = ncol[a] - sa, ldp = (nr + 3) & ~3;
    const double *src = P64 + poff[a];
    float *dst = P32 + p32off[a];
    for (int64_t e = threadIdx.x; e < (int64_t)sa * ldp; e += blockDim.x) {
        const int64_t q = e / ldp;
        const int u = (int)(e % ldp);
        dst[e] = u < nr ? (float)src[q * nr + u] : 0.f;
    }
}

// Segmented dedupe + (key, id) sort + truncation shared by all levels.
askit_status dedupe_sort_truncate(int64_t a0, int nseg, const std::vector<int32_t> &hbeg,
                                  const std::vector<int32_t> &hend, int32_t *cj, double *ck,
                                  int64_t n, int ell, askit_tree t, cudaStream_t s) {
    int32_t *beg = nullptr, *end = nullptr, *seg_of = nullptr, *cnt = nullptr, *tj = nullptr;
    double *tk = nullptr;
    void *tmp = nullptr;
    askit_status rc = ASKIT_OK;
    size_t b1 = 0, b2 = 0;
    cudaError_t e = cudaSuccess;
#define DCHK(x) do { e = (x); if (e != cudaSuccess) goto fail; } while (0)
    DCHK(cudaMalloc(&beg, sizeof(int32_t) * nseg));
    DCHK(cudaMalloc(&end, sizeof(int32_t) * nseg));
    DCHK(cudaMalloc(&cnt, sizeof(int32_t) * nseg));
    DCHK(cudaMalloc(&seg_of, sizeof(int32_t) * (n ? n : 1)));
    DCHK(cudaMalloc(&tj, sizeof(int32_t) * (n ? n : 1)));
    DCHK(cudaMalloc(&tk, sizeof(double) * (n ? n : 1)));
    DCHK(cudaMemcpyAsync(beg, hbeg.data(), sizeof(int32_t) * nseg, cudaMemcpyHostToDevice, s));
    DCHK(cudaMemcpyAsync(end, hend.data(), sizeof(int32_t) * nseg, cudaMemcpyHostToDevice, s));
    DCHK(cudaMemsetAsync(cnt, 0, sizeof(int32_t) * nseg, s));
    if ((rc = seg_sort_i32_f64(nullptr, nullptr, nullptr, nullptr, n, nseg, nullptr, nullptr, nullptr, &b1, s)) != ASKIT_OK) goto out;
    if ((rc = seg_sort_f64_i32(nullptr, nullptr, nullptr, nullptr, n, nseg, nullptr, nullptr, nullptr, &b2, s)) != ASKIT_OK) goto out;
    b1 = std::max(b1, b2);
    DCHK(cudaMalloc(&tmp, b1));
    seg_of_kernel<<<nseg, 256, 0, s>>>(beg, end, nseg, seg_of);
    // by id (stable): each id's entries become contiguous
    if ((rc = seg_sort_i32_f64(cj, tj, ck, tk, n, nseg, beg, end, tmp, &b1, s)) != ASKIT_OK) goto out;
    dedupe_kernel<<<nblk(n, 256), 256, 0, s>>>(tj, tk, cj, ck, seg_of, beg, n, cnt);
    DCHK(cudaGetLastError());
    // by key (stable over ascending ids): (key, id) order, removed entries last
    if ((rc = seg_sort_f64_i32(ck, tk, cj, tj, n, nseg, beg, end, tmp, &b1, s)) != ASKIT_OK) goto out;
    nl_write_kernel<<<nseg, 256, 0, s>>>(a0, nseg, beg, tj, tk, cnt, ell, t->nl_cnt, t->nl_ids, t->nl_key);
    DCHK(cudaGetLastError());
    DCHK(cudaStreamSynchronize(s));
    goto out;
fail:
    askit_set_error("node lists: %s", cudaGetErrorString(e));
    rc = e == cudaErrorMemoryAllocation ? ASKIT_ERR_OOM : ASKIT_ERR_CUDA;
out:
#undef DCHK
    cudaStreamSynchronize(s);
    cudaFree(beg); cudaFree(end); cudaFree(cnt); cudaFree(seg_of); cudaFree(tj); cudaFree(tk); cudaFree(tmp);
    return rc;
}

}  // namespace

askit_status build_node_lists(askit_tree t, cudaStream_t s) {
    const int L = t->L, ell = t->ell_max, kappa = t->kappa;
    const int64_t N = t->N;
    if (L == 0) return ASKIT_OK;
    // leaves
    {
        int64_t n = N * kappa;
        int32_t *cj = nullptr;
        double *ck = nullptr;
        ASK_CUDA(cudaMalloc(&cj, sizeof(int32_t) * n));
        ASK_CUDA(cudaMalloc(&ck, sizeof(double) * n));
        leaf_cand_kernel<<<nblk(n, 256), 256, 0, s>>>(t->perm, t->leafof, t->knn, t->knnd, N, kappa, cj, ck);
        int64_t a0 = (int64_t)1 << L;
        int nseg = (int)a0;
        std::vector<int32_t> hb(nseg), he(nseg);
        for (int g = 0; g < nseg; ++g) {
            hb[g] = (int32_t)(t->h_start[a0 + g] * kappa);
            he[g] = (int32_t)((t->h_start[a0 + g] + t->h_size[a0 + g]) * kappa);
        }
        askit_status rc = dedupe_sort_truncate(a0, nseg, hb, he, cj, ck, n, ell, t, s);
        cudaFree(cj);
        cudaFree(ck);
        ASK_TRY(rc);
    }
    // internal levels, bottom-up
    for (int depth = L - 1; depth >= 1; --depth) {
        int64_t a0 = (int64_t)1 << depth;
        int nseg = (int)a0;
        int64_t n = (int64_t)nseg * 2 * ell;
        int32_t *cj = nullptr;
        double *ck = nullptr;
        ASK_CUDA(cudaMalloc(&cj, sizeof(int32_t) * n));
        ASK_CUDA(cudaMalloc(&ck, sizeof(double) * n));
        inner_cand_kernel<<<nblk(n, 256), 256, 0, s>>>(a0, nseg, ell, L, depth, t->leafof, t->nl_cnt,
                                                      t->nl_ids, t->nl_key, cj, ck);
        std::vector<int32_t> hb(nseg), he(nseg);
        for (int g = 0; g < nseg; ++g) {
            hb[g] = (int32_t)((int64_t)g * 2 * ell);
            he[g] = (int32_t)((int64_t)(g + 1) * 2 * ell);
        }
        askit_status rc = dedupe_sort_truncate(a0, nseg, hb, he, cj, ck, n, ell, t, s);
        cudaFree(cj);
        cudaFree(ck);
        ASK_TRY(rc);
    }
    return ASKIT_OK;
}

askit_status build_samples(askit_tree t, cudaStream_t s) {
    if (t->L == 0) return ASKIT_OK;
    int64_t n = t->n_nodes - 2;
    sample_kernel<<<nblk(n, 64), 64, 0, s>>>(t->n_nodes, t->N, t->L, t->ell_max, t->nsize, t->leafof,
                                            t->nl_cnt, t->nl_ids, t->prm.seed, t->trows);
    ASK_LAUNCH();
    ASK_CUDA(cudaStreamSynchronize(s));
    return ASKIT_OK;
}

// Bottom-up skeletonization, one tree level at a time, in batches of nodes
// whose FP64 blocks fit a workspace budget.
askit_status skeletonize(askit_tree t, cudaStream_t s) {
    const int L = t->L, ell = t->ell_max, d = t->d;
    const int s_max = t->prm.s_max;
    const int64_t N = t->N, nn = t->n_nodes;
    t->h_s.assign(nn, 0);
    t->h_ncol.assign(nn, 0);
    if (L == 0) return ASKIT_OK;
    const int cmax = (int)std::max<int64_t>(t->h_size[(int64_t)1 << L], 2 * (int64_t)s_max);
    std::vector<int32_t> h_ell(nn, 0);
    for (int64_t a = 2; a < nn; ++a) h_ell[a] = (int32_t)std::min<int64_t>(ell, N - t->h_size[a]);
    int32_t *d_ell = nullptr, *skel_fixed = nullptr, *piv_fixed = nullptr;
    ASK_TRY(t->arena.alloc(&d_ell, nn));
    ASK_TRY(t->arena.alloc(&skel_fixed, (size_t)nn * s_max));
    ASK_TRY(t->arena.alloc(&piv_fixed, (size_t)nn * cmax));
    ASK_CUDA(cudaMemcpyAsync(d_ell, h_ell.data(), sizeof(int32_t) * nn, cudaMemcpyHostToDevice, s));
    ASK_CUDA(cudaMemsetAsync(t->d_s, 0, sizeof(int32_t) * nn, s));

    std::vector<double *> lvl_P64(L + 1, nullptr);
    std::vector<int64_t> lvl_ptot(L + 1, 0);
    std::vector<int64_t> node_poff(nn, 0);   // offset within its level pool
    const size_t budget = (size_t)6 << 30;   // FP64 workspace per batch
    int dev = 0, sms = 0;
    ASK_CUDA(cudaGetDevice(&dev));
    ASK_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));

    for (int depth = L; depth >= 1; --depth) {
        int64_t a0 = (int64_t)1 << depth, a1 = (int64_t)2 << depth;
        for (int64_t a = a0; a < a1; ++a)
            t->h_ncol[a] = depth == L ? (int32_t)t->h_size[a] : t->h_s[2 * a] + t->h_s[2 * a + 1];
        ASK_CUDA(cudaMemcpyAsync(t->d_ncol + a0, t->h_ncol.data() + a0, sizeof(int32_t) * (a1 - a0),
                                 cudaMemcpyHostToDevice, s));
        int32_t *cols = nullptr;
        ASK_CUDA(cudaMalloc(&cols, sizeof(int32_t) * (a1 - a0) * cmax));
        cols_kernel<<<(unsigned)(a1 - a0), 128, 0, s>>>(a0, (int)(a1 - a0), depth == L, t->perm, t->nstart,
                                                       t->nsize, skel_fixed, t->d_s, s_max, cmax, cols);
        ASK_LAUNCH();
        // level pool for P (sizes known only after the QR of each batch)
        std::vector<double *> batch_P64;
        std::vector<int64_t> batch_tot;
        int64_t a = a0;
        int64_t lvl_run = 0;   // offset of the current batch inside the level pool
        while (a < a1) {
            // pick a batch
            std::vector<int32_t> nodes;
            std::vector<int64_t> woff, pws;
            size_t used = 0;
            while (a < a1) {
                int64_t c = t->h_ncol[a], r = h_ell[a];
                int64_t sh = std::min<int64_t>(std::min<int64_t>(s_max, c), r);
                size_t need = (size_t)(r * c + sh * c + 2) * sizeof(double);
                if (!nodes.empty() && used + need > budget) break;
                nodes.push_back((int32_t)a);
                woff.push_back((int64_t)(used / sizeof(double)));
                pws.push_back((int64_t)(used / sizeof(double)) + r * c);
                used += need;
                ++a;
            }
            int nb = (int)nodes.size();
            double *work = nullptr;
            int32_t *d_nodes = nullptr;
            int64_t *d_woff = nullptr, *d_pws = nullptr, *d_plvl = nullptr;
            ASK_CUDA(cudaMalloc(&work, used ? used : 8));
            ASK_CUDA(cudaMalloc(&d_nodes, sizeof(int32_t) * nb));
            ASK_CUDA(cudaMalloc(&d_woff, sizeof(int64_t) * nb));
            ASK_CUDA(cudaMalloc(&d_pws, sizeof(int64_t) * nb));
            ASK_CUDA(cudaMalloc(&d_plvl, sizeof(int64_t) * nb));
            ASK_CUDA(cudaMemcpyAsync(d_nodes, nodes.data(), sizeof(int32_t) * nb, cudaMemcpyHostToDevice, s));
            ASK_CUDA(cudaMemcpyAsync(d_woff, woff.data(), sizeof(int64_t) * nb, cudaMemcpyHostToDevice, s));
            ASK_CUDA(cudaMemcpyAsync(d_pws, pws.data(), sizeof(int64_t) * nb, cudaMemcpyHostToDevice, s));
            int64_t maxent = 0;
            for (int g = 0; g < nb; ++g) maxent = std::max<int64_t>(maxent, (int64_t)h_ell[nodes[g]] * t->h_ncol[nodes[g]]);
            if (maxent > 0) {
                fill_kernel<<<dim3(nblk(maxent, 256), nb), 256, 0, s>>>(
                    t->X, d, t->hsrc, t->prm.kernel_scale, a0, d_nodes, d_woff, t->d_ncol, d_ell, t->trows,
                    ell, cols, cmax, work);
                ASK_LAUNCH();
            }
            int maxrows = 0;
            for (int g = 0; g < nb; ++g) maxrows = std::max(maxrows, h_ell[nodes[g]]);
            // a cluster per node while the CTAs stay within the SMs and each has four
            // column groups, one for every quarter of its SM (64K x 64, 512 columns:
            // a level takes 14.7 ms with four CTAs a node, 15.5 with eight)
            int maxcols = 0;
            for (int g = 0; g < nb; ++g) maxcols = std::max(maxcols, t->h_ncol[nodes[g]]);
            int c = 1;
            while (c < 8 && 2 * c * nb <= sms && 2 * c * 128 <= maxcols) c *= 2;
            const size_t smem = sizeof(double) * (size_t)(maxrows + 1) +
                                sizeof(float) * 32 * (((size_t)cmax + 31) / 32 / c + 1);
            ASK_TRY((c == 1 ? launch_cpqr<1> : c == 2 ? launch_cpqr<2> : c == 4 ? launch_cpqr<4> : launch_cpqr<8>)(
                nb, smem, s, d_nodes, d_woff, d_pws, t, d_ell, s_max, work, piv_fixed, cmax));
            ASK_CUDA(cudaMemcpyAsync(t->h_s.data() + nodes[0], t->d_s + nodes[0], sizeof(int32_t) * nb,
                                     cudaMemcpyDeviceToHost, s));
            ASK_CUDA(cudaStreamSynchronize(s));
            std::vector<int64_t> plvl(nb);
            int64_t tot = 0;
            for (int g = 0; g < nb; ++g) {
                int64_t nd = nodes[g];
                plvl[g] = tot;
                node_poff[nd] = lvl_run + tot;
                tot += (int64_t)t->h_s[nd] * (t->h_ncol[nd] - t->h_s[nd]);
            }
            double *P64 = nullptr;
            ASK_CUDA(cudaMalloc(&P64, sizeof(double) * (tot ? tot : 1)));
            ASK_CUDA(cudaMemcpyAsync(d_plvl, plvl.data(), sizeof(int64_t) * nb, cudaMemcpyHostToDevice, s));
            skel_out_kernel<<<nb, 256, 0, s>>>(d_nodes, a0, d_pws, d_plvl, t->d_s, t->d_ncol, cols, cmax,
                                              piv_fixed, s_max, work, skel_fixed, P64);
            ASK_LAUNCH();
            ASK_CUDA(cudaStreamSynchronize(s));
            cudaFree(work); cudaFree(d_nodes); cudaFree(d_woff); cudaFree(d_pws); cudaFree(d_plvl);
            batch_P64.push_back(P64);
            batch_tot.push_back(tot);
            lvl_run += tot;
        }
        cudaFree(cols);
        // concatenate the level's batches
        int64_t ltot = 0;
        for (auto x : batch_tot) ltot += x;
        ASK_CUDA(cudaMalloc(&lvl_P64[depth], sizeof(double) * (ltot ? ltot : 1)));
        int64_t off = 0;
        for (size_t b = 0; b < batch_tot.size(); ++b) {
            ASK_CUDA(cudaMemcpyAsync(lvl_P64[depth] + off, batch_P64[b], sizeof(double) * batch_tot[b], cudaMemcpyDeviceToDevice, s));
            off += batch_tot[b];
        }
        ASK_CUDA(cudaStreamSynchronize(s));
        for (size_t b = 0; b < batch_P64.size(); ++b) cudaFree(batch_P64[b]);
        lvl_ptot[depth] = ltot;
    }

    // heap-order pools: level 1 first
    t->h_poff.assign(nn + 1, 0);
    t->h_skoff.assign(nn + 1, 0);
    t->h_pivoff.assign(nn + 1, 0);
    t->h_spool.assign(nn + 1, 0);
    int64_t ptot = 0;
    std::vector<int64_t> lvl_base(L + 1, 0);
    for (int depth = 1; depth <= L; ++depth) { lvl_base[depth] = ptot; ptot += lvl_ptot[depth]; }
    for (int64_t a = 2; a < nn; ++a) t->h_poff[a] = lvl_base[heap_depth(a)] + node_poff[a];
    t->h_poff[nn] = ptot;
    t->p_total = ptot;
    ASK_TRY(t->arena.alloc(&t->P64, ptot));
    for (int depth = 1; depth <= L; ++depth) {
        if (lvl_ptot[depth])
            ASK_CUDA(cudaMemcpyAsync(t->P64 + lvl_base[depth], lvl_P64[depth], sizeof(double) * lvl_ptot[depth], cudaMemcpyDeviceToDevice, s));
    }
    // the FP32 copy: padded rows, in heap order
    std::vector<int64_t> p32off(nn + 1, 0);
    t->lvl_nr.assign(L + 1, 0);
    int64_t p32tot = 0;
    for (int64_t a = 2; a < nn; ++a) {
        const int nr = t->h_ncol[a] - t->h_s[a];
        p32off[a] = p32tot;
        p32tot += (int64_t)t->h_s[a] * ((nr + 3) & ~3);
        int &mx = t->lvl_nr[heap_depth(a)];
        mx = std::max(mx, nr);
    }
    p32off[nn] = p32tot;
    ASK_TRY(t->arena.alloc(&t->P32, p32tot));
    int64_t sk = 0, pv = 0, sp = 0;
    for (int64_t a = 0; a < nn; ++a) {
        t->h_skoff[a] = sk;
        t->h_pivoff[a] = pv;
        t->h_spool[a] = sp;
        if (a >= 2) {
            sk += t->h_s[a];
            pv += t->h_ncol[a];
            sp += (t->h_s[a] + ASK_ROW_PAD - 1) / ASK_ROW_PAD * ASK_ROW_PAD;
        }
    }
    t->h_skoff[nn] = sk; t->h_pivoff[nn] = pv; t->h_spool[nn] = sp;
    t->skel_total = sk; t->piv_total = pv; t->spool_rows = sp;
    ASK_TRY(t->arena.alloc(&t->skel_ids, sk));
    ASK_TRY(t->arena.alloc(&t->piv, pv));
    for (int64_t a = 2; a < nn; ++a) {
        if (t->h_s[a])
            ASK_CUDA(cudaMemcpyAsync(t->skel_ids + t->h_skoff[a], skel_fixed + a * s_max, sizeof(int32_t) * t->h_s[a], cudaMemcpyDeviceToDevice, s));
        if (t->h_ncol[a])
            ASK_CUDA(cudaMemcpyAsync(t->piv + t->h_pivoff[a], piv_fixed + a * cmax, sizeof(int32_t) * t->h_ncol[a], cudaMemcpyDeviceToDevice, s));
    }
    ASK_TRY(t->arena.alloc(&t->d_p32off, nn + 1));
    int64_t *d_poff = nullptr;      // offsets in P64
    ASK_CUDA(cudaMallocAsync(&d_poff, sizeof(int64_t) * (nn + 1), s));
    ASK_TRY(t->arena.alloc(&t->d_skoff, nn + 1));
    ASK_TRY(t->arena.alloc(&t->d_pivoff, nn + 1));
    ASK_TRY(t->arena.alloc(&t->d_spool, nn + 1));
    ASK_CUDA(cudaMemcpyAsync(d_poff, t->h_poff.data(), sizeof(int64_t) * (nn + 1), cudaMemcpyHostToDevice, s));
    ASK_CUDA(cudaMemcpyAsync(t->d_p32off, p32off.data(), sizeof(int64_t) * (nn + 1), cudaMemcpyHostToDevice, s));
    p32_kernel<<<(unsigned)(nn - 2), 256, 0, s>>>(t->P64, d_poff, t->d_p32off, t->d_s, t->d_ncol, t->P32);
    ASK_LAUNCH();
    cudaFreeAsync(d_poff, s);
    ASK_CUDA(cudaMemcpyAsync(t->d_skoff, t->h_skoff.data(), sizeof(int64_t) * (nn + 1), cudaMemcpyHostToDevice, s));
    ASK_CUDA(cudaMemcpyAsync(t->d_pivoff, t->h_pivoff.data(), sizeof(int64_t) * (nn + 1), cudaMemcpyHostToDevice, s));
    ASK_CUDA(cudaMemcpyAsync(t->d_spool, t->h_spool.data(), sizeof(int64_t) * (nn + 1), cudaMemcpyHostToDevice, s));
    ASK_CUDA(cudaStreamSynchronize(s));
    for (int depth = 1; depth <= L; ++depth) cudaFree(lvl_P64[depth]);
    t->arena.release(skel_fixed);
    t->arena.release(piv_fixed);
    t->arena.release(d_ell);
    return ASKIT_OK;
}
