// Exact kappa nearest tree points of out-of-sample queries (d <= 64).
//
// 1. Home: the two leaves whose centers are nearest to each query (FP32 tiles).
// 2. Seed: the kappa-th smallest FP32 distance over the points of those leaves,
//    rounded up by the FP32 sum's error bound, is an upper bound U of the query's
//    true kappa-th distance.
// 3. Shortlist: every tree point against every query on the tensor cores, FP16x3;
//    a point within U and the products' error margin becomes a candidate.
// 4. Re-rank: FP32 distances of the candidates leave those that can be among the
//    kappa nearest; only these get their canonical FP64 distance, ordered by
//    (distance, id).
// A query with more than KO_CAP candidates -- the margin, in proportion to the squared
// distance from the data mean, takes in whole clusters or stretches of a curve where
// points lie that close -- scans the leaves whose ball around their center can hold a
// point within U.  A query whose coordinates leave the FP16-safe range takes the
// exhaustive search, and every query does where norms or
// scales would leave FP32's range (fp32_safe): no FP32 distance below overflows.
//
// An FP64 warp instruction takes 64 cycles of its quarter of the SM here, so the FP64
// distances are what the steps avoid: seeding in FP64 over the two leaves took 74 of the 110 ms that
// 100,000 queries spent against 131,072 points (d = 64), the FP64 re-rank of every
// candidate 8.8 ms, the shortlist with operands split on the chip 18.6 ms.
// Now, the same 100,000 queries: home 0.19, seed 0.96, shortlist 3.8, re-rank 1.2 ms.
#include <cuda.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <mutex>

#include "askit_impl.cuh"
#include "knn_warp.cuh"
#include "tc_ptx.cuh"

namespace {

using namespace tcx;

inline unsigned nblk(int64_t n, int b) { return (unsigned)((n + b - 1) / b); }

constexpr int KO_CAP = 1024;                   // candidates a query keeps
constexpr int KO_BAD = 1 << 30;                // count of a query outside the FP16-safe range
// The margin of the FP16x3 distance n_q + n_j - 2 a.b (both sides centered on the
// data mean, a.b in three split products): the splits keep 22 significant bits and
// the FP32 accumulation adds a few 2^-23 |a||b| a step, below 2^-18 (n_q + n_j)
// together; eta = 2^-16.  Coordinates below 2^-13 of the scaled range lose bits of
// their low half to the FP16 subnormal step 2^-24, an absolute error of at most
// 2^-25 / sigma a coordinate; by the inequality of the means its share of the
// distance is below eta/2 (n_q + n_j) + KO_ABS / sigma^2.
constexpr float KO_ETA = 1.52587890625e-05f;
constexpr float KO_ABS = 5.9604645e-08f;       // 2^-24

// Relative bound of an FP32 sum of d squared differences, in any order.
__host__ __device__ __forceinline__ float sum_gam(int d) { return (float)(d + 2) * 5.9604645e-8f * 1.25f + 1e-6f; }

// Queries as FP16x3 operands of the shortlist: (y - xbar) sigma split hi + lo
// [T_pad, 64], n = |y - xbar|^2; a query outside the FP16-safe range gets zero
// rows and the count KO_BAD (hits on the zero rows add to it: N < 2^30 here).  A warp per row; rows past T are zero.  Row i is
// query order[i] (order null: query i), here and in the steps that follow.
__global__ void ko_split_kernel(const float *Y, int d, const int32_t *order, int64_t T, int64_t T_pad, const float *xbar, float sigma,
                                uint16_t *hi, uint16_t *lo, float *nq, int *cnt) {
    const int lane = threadIdx.x & 31;
    const int64_t row = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5);
    if (row >= T_pad) return;                              // warp-uniform
    const int64_t src = order && row < T ? order[row] : row;
    float v[2], acc = 0.f;
    bool bad = false;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int k = lane + 32 * h;
        const float x = (row < T && k < d) ? Y[src * d + k] - xbar[k] : 0.f;
        v[h] = x * sigma;
        acc = fmaf(x, x, acc);
        bad |= !(fabsf(v[h]) <= 30000.f);
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(FULL, acc, o);
    bad = __any_sync(FULL, bad);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int64_t o = row * TC_K + lane + 32 * h;
        const __half vh = __float2half_rn(bad ? 0.f : v[h]);
        hi[o] = __half_as_ushort(vh);
        lo[o] = __half_as_ushort(__float2half_rn(bad ? 0.f : v[h] - __half2float(vh)));
    }
    if (lane == 0) {
        nq[row] = acc;
        if (row < T) cnt[row] = bad ? KO_BAD : 0;
    }
}

// Step 1.  Block (x, y): queries 64 x .. + 63 against the leaf centers of split y,
// 64 at a time, FP32 differences from shared memory (4 queries x 8 centers a
// thread: three 16-byte reads for 64 operations; a warp a query with scalar reads
// of the centers took 5.5 ms at 100,000 queries and 256 leaves).  Writes the two
// nearest centers of the split.
constexpr int HO_T = 64, HO_LD = HO_T + 4;
__global__ void __launch_bounds__(128) ko_home_kernel(const float *Y, int d, int64_t T, const float *cent,
                                                      const int32_t *leaf_cbase, int64_t M, int64_t split_len,
                                                      float *hd, int32_t *hi_) {
    __shared__ __align__(16) float qs[TC_K][HO_LD], cs[TC_K][HO_LD];
    const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3;
    const int64_t q0 = (int64_t)blockIdx.x * HO_T;
    const int64_t l0 = (int64_t)blockIdx.y * split_len, l1 = min(M, l0 + split_len);
    for (int e = tid; e < HO_T * TC_K; e += 128) {
        const int q = e / TC_K, k = e % TC_K;
        qs[k][q] = (q0 + q < T && k < d) ? Y[(q0 + q) * d + k] : 0.f;
    }
    float b0[4], b1[4];
    int i0[4], i1[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) { b0[i] = b1[i] = 3.4e38f; i0[i] = i1[i] = (int)l0; }
    for (int64_t lb = l0; lb < l1; lb += HO_T) {
        __syncthreads();
        for (int e = tid; e < HO_T * TC_K; e += 128) {
            const int c = e / TC_K, k = e % TC_K;
            cs[k][c] = (lb + c < l1 && k < d) ? cent[(int64_t)leaf_cbase[lb + c] * TC_K + k] : 0.f;
        }
        __syncthreads();
        float acc[4][8];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
        for (int k = 0; k < d; ++k) {
            const float4 q4 = *reinterpret_cast<const float4 *>(&qs[k][4 * ty]);
            const float4 ca = *reinterpret_cast<const float4 *>(&cs[k][8 * tx]);
            const float4 cb = *reinterpret_cast<const float4 *>(&cs[k][8 * tx + 4]);
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
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int64_t l = lb + 8 * tx + j;
            if (l >= l1) continue;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (acc[i][j] < b0[i]) { b1[i] = b0[i]; i1[i] = i0[i]; b0[i] = acc[i][j]; i0[i] = (int)l; }
                else if (acc[i][j] < b1[i]) { b1[i] = acc[i][j]; i1[i] = (int)l; }
            }
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        for (int o = 4; o > 0; o >>= 1) {                  // merge the 8 threads of a query
            const float ob0 = __shfl_xor_sync(FULL, b0[i], o), ob1 = __shfl_xor_sync(FULL, b1[i], o);
            const int oi0 = __shfl_xor_sync(FULL, i0[i], o), oi1 = __shfl_xor_sync(FULL, i1[i], o);
            if (ob0 < b0[i]) {
                const bool second = b0[i] < ob1;
                b1[i] = second ? b0[i] : ob1;
                i1[i] = second ? i0[i] : oi1;
                b0[i] = ob0;
                i0[i] = oi0;
            } else if (ob0 < b1[i]) {
                b1[i] = ob0;
                i1[i] = oi0;
            }
        }
        const int64_t q = q0 + 4 * ty + i;
        if (tx == 0 && q < T) {
            const int64_t o = ((int64_t)blockIdx.y * T + q) * 2;
            hd[o] = b0[i];
            hd[o + 1] = b1[i];
            hi_[o] = i0[i];
            hi_[o + 1] = i1[i];
        }
    }
}

// The nearest home leaf of each query, the key of the queries' order, and 0 .. T - 1.
__global__ void ko_key_kernel(const float *hd, const int32_t *hi_, int nsplit, int64_t T, uint32_t *key, int32_t *iota) {
    const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (q >= T) return;
    float m = 3.4e38f;
    int32_t leaf = 0;
    for (int p = 0; p < nsplit; ++p) {
        const int64_t o = ((int64_t)p * T + q) * 2;
        if (hd[o] < m) {
            m = hd[o];
            leaf = hi_[o];
        }
    }
    key[q] = (uint32_t)leaf;
    iota[q] = (int32_t)q;
}

// A warp's FP32 squared distances of 32 tree rows to its query: eight lanes a row,
// each with every eighth 16-byte piece (NJ pieces a lane, d_pad = 32 NJ), four rows
// a load, so that a load takes whole 128-byte lines (with four lanes a row it took
// halves of eight lines, twice the cycles in the load unit, which bound the seed at
// 91 %: 1.74 ms for 100,000 queries, 1.17 with this and the gathered offers below); the lanes' sums meet in a transposing butterfly.  Lane l ends with the
// distance of pos(4 (l & 7) + (l >> 3)).
// PACK: two coordinates an instruction, which the leaf scan gains from (50,000 queries
// in a cluster of 65,536 points, 16 dimensions 32.5 -> 29.9 ms, 64 dimensions 86 -> 69)
// and the seed and the re-rank lose by (100,000 queries 8.1 -> 8.6 ms).
template <int NJ, bool PACK, class F>
__device__ __forceinline__ float rows32(const float *Xt, const float4 (&y)[NJ], int lane, F pos) {
    const int sub = lane & 7, r4 = lane >> 3;
    float4 x[8][NJ];
#pragma unroll
    for (int g = 0; g < 8; ++g) {
        const float4 *row = reinterpret_cast<const float4 *>(Xt + (int64_t)pos(4 * g + r4) * (32 * NJ)) + sub;
#pragma unroll
        for (int j = 0; j < NJ; ++j) x[g][j] = row[8 * j];
    }
    float a[8];
#pragma unroll
    for (int g = 0; g < 8; ++g) {
        a[g] = 0.f;
        float2 s = make_float2(0.f, 0.f);
        const float2 m1 = make_float2(-1.f, -1.f);
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
            if (!PACK) {
                const float t0 = y[j].x - x[g][j].x, t1 = y[j].y - x[g][j].y, t2 = y[j].z - x[g][j].z, t3 = y[j].w - x[g][j].w;
                a[g] = fmaf(t0, t0, a[g]);
                a[g] = fmaf(t1, t1, a[g]);
                a[g] = fmaf(t2, t2, a[g]);
                a[g] = fmaf(t3, t3, a[g]);
                continue;
            }
            const float2 t0 = __ffma2_rn(make_float2(x[g][j].x, x[g][j].y), m1, make_float2(y[j].x, y[j].y));
            const float2 t1 = __ffma2_rn(make_float2(x[g][j].z, x[g][j].w), m1, make_float2(y[j].z, y[j].w));
            s = __ffma2_rn(t0, t0, s);
            s = __ffma2_rn(t1, t1, s);
        }
        if (PACK) a[g] = s.x + s.y;
    }
    // lanes with bit m of sub set keep the upper half of the values left
#pragma unroll
    for (int m = 4; m >= 1; m >>= 1) {
        const bool up = sub & m;
#pragma unroll
        for (int k = 0; k < m; ++k) {
            const float keep = up ? a[k + m] : a[k], give = up ? a[k] : a[k + m];
            a[k] = keep + __shfl_xor_sync(FULL, give, m);
        }
    }
    return a[0];
}

template <int NJ>
__device__ __forceinline__ void load_query(const float *y, int d, int lane, float4 (&q)[NJ]) {
    const int sub = lane & 7;
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
        const int k = 4 * (sub + 8 * j);
        q[j] = make_float4(k < d ? y[k] : 0.f, k + 1 < d ? y[k + 1] : 0.f, k + 2 < d ? y[k + 2] : 0.f,
                           k + 3 < d ? y[k + 3] : 0.f);
    }
}

// Offers one value per lane to the list l by way of buf (64 floats of the warp,
// `have` < 32 of them waiting): only values below the list's kappa-th are taken,
// and 32 of them are sorted and merged at a time (22 shuffles, otherwise spent on
// nearly every batch of 32 for the few values that still enter).
__device__ __forceinline__ void gather_f32(float &l, float v, float *buf, int &have, int kappa, int lane) {
    const bool useful = v < __shfl_sync(FULL, l, kappa - 1);
    const unsigned m = __ballot_sync(FULL, useful);
    if (!m) return;
    if (useful) buf[have + __popc(m & ((1u << lane) - 1u))] = v;
    have += __popc(m);
    __syncwarp();
    if (have < 32) return;
    have -= 32;
    const float first = buf[lane], rest = buf[32 + (lane < have ? lane : 0)];
    __syncwarp();
    if (lane < have) buf[lane] = rest;
    __syncwarp();
    warp_offer_f32(l, first, kappa, lane);
}

// Step 2, W warps per query: U.  The splits' candidates give the two home leaves;
// their points' FP32 distances pass through the warps' best-32 lists, merged at
// the end.  One warp a query where the queries fill the GPU, four below that (one
// query is a chain of about 32 rounds of loads and merges: 51 us at 100 queries with one warp, 24 with four).
template <int NJ, int W>
__global__ void __launch_bounds__(256) ko_seed_kernel(const float *Xt, const float *Y, int d, const int32_t *order,
                                                      int64_t T, const float *hd,
                                                      const int32_t *hi_, int nsplit, int64_t M, const int32_t *nstart,
                                                      const int32_t *nsize, int kappa, float *U) {
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int64_t qw = blockIdx.x * (int64_t)(8 / W) + warp / W;
    const int64_t q = qw < T ? qw : T - 1;                 // warps past T repeat the last query
    const int64_t src = order ? order[q] : q;
    __shared__ float lists[8][64];
    int have = 0;
    float bd = 3.4e38f;
    int bi = 0;
    if (lane < 2 * nsplit) {
        const int64_t o = ((int64_t)(lane >> 1) * T + src) * 2 + (lane & 1);
        bd = hd[o];
        bi = hi_[o];
    }
    int leaf[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        float m = bd;
        int w = lane;
        for (int o = 16; o > 0; o >>= 1) {
            const float om = __shfl_xor_sync(FULL, m, o);
            const int ow = __shfl_xor_sync(FULL, w, o);
            if (om < m || (om == m && ow < w)) { m = om; w = ow; }
        }
        leaf[h] = __shfl_sync(FULL, bi, w);
        if (lane == w) bd = 3.4e38f;
    }
    float4 y[NJ];
    load_query<NJ>(Y + src * d, d, lane, y);
    float l = 3.4e38f;
    for (int h = 0; h < 2; ++h) {
        if (h == 1 && leaf[1] == leaf[0]) break;
        const int p0 = nstart[M + leaf[h]], np = nsize[M + leaf[h]];
        for (int b = 32 * (warp % W); b < np; b += 32 * W) {
            // rows past the leaf are other points or the zero rows past N
            const float v = rows32<NJ, false>(Xt, y, lane, [&](int i) { return p0 + b + i; });
            const int i = b + 4 * (lane & 7) + (lane >> 3);
            gather_f32(l, i < np ? v : 3.4e38f, lists[warp], have, kappa, lane);
        }
    }
    warp_offer_f32(l, lane < have ? lists[warp][lane] : 3.4e38f, kappa, lane);
    if (W > 1) {
        __syncwarp();
        lists[warp][lane] = l;
        __syncthreads();
        if (warp % W) return;
        for (int w = 1; w < W; ++w) warp_offer_f32(l, lists[warp + w][lane], kappa, lane);
    }
    const float kth = __shfl_sync(FULL, l, kappa - 1);
    if (lane == 0 && qw < T) U[q] = kth < 3.0e38f ? __fadd_ru(__fmul_ru(kth, 1.f + 2.f * sum_gam(d)), 1e-37f) : 3.4e38f;
}

// Step 4, a warp per query, W warps a block: eight where the queries fill the GPU,
// one below that (a query is a chain of about 20 loads and 200 FP64 instructions, so
// few queries are spread over as many SMs as they can reach: 54 -> 39 us at 100
// queries).  100,000 queries 1.73 -> 1.22 ms with the lists ordered by integer
// comparisons; the FP64 distances of 32 candidates a query alone take 0.98.
template <int NJ, int W>
__global__ void __launch_bounds__(32 * W) ko_rerank_kernel(const float *Xt, const float *Y, int d,
                                                           const int32_t *order, int64_t T, const int32_t *perm,
                                                           const int *cnt, const int32_t *cand, int kappa,
                                                           int32_t *ids, double *dist, int *n_ovf, int32_t *ovf,
                                                           int32_t *wide, const float *U, bool many) {
    __shared__ float sd[W][KO_CAP];
    __shared__ float sy[W][TC_K];
    __shared__ float sl[W][64];
    int have_l = 0;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t q = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (q >= T) return;                                    // warp-uniform
    const int64_t src = order ? order[q] : q;
    const int n = cnt[q];
    // (fewer than kappa cannot be: U bounds kappa points.)  Where the home leaves hold
    // fewer than kappa points U bounds nothing, no leaf can be left out, and many such
    // queries are better off in the exhaustive search's tiles
    if (n >= KO_BAD || n < kappa || (n > KO_CAP && many && !(U[q] < 3.0e38f))) {
        if (lane == 0) ovf[atomicAdd(n_ovf, 1)] = (int32_t)src;
        return;
    }
    if (n > KO_CAP) {
        if (lane == 0) wide[atomicAdd(n_ovf + 1, 1)] = (int32_t)q;
        return;
    }
    const int32_t *c = cand + q * KO_CAP;
    float4 y[NJ];
    load_query<NJ>(Y + src * d, d, lane, y);
    for (int k = lane; k < d; k += 32) sy[warp][k] = Y[src * d + k];
    float l = 3.4e38f;
    for (int b = 0; b < n; b += 32) {
        const int32_t mine = c[min(b + lane, n - 1)];
        const float v = rows32<NJ, false>(Xt, y, lane, [&](int i) { return __shfl_sync(FULL, mine, i); });
        const int i = b + 4 * (lane & 7) + (lane >> 3);
        if (i < n) sd[warp][i] = v;
        gather_f32(l, i < n ? v : 3.4e38f, sl[warp], have_l, kappa, lane);
    }
    warp_offer_f32(l, lane < have_l ? sl[warp][lane] : 3.4e38f, kappa, lane);
    __syncwarp();
    // a point among the kappa nearest has an FP32 distance within (1 + gam) /
    // (1 - gam) of the kappa-th smallest one
    const float lim = __shfl_sync(FULL, l, kappa - 1) * (1.f + 3.f * sum_gam(d)) + 1e-37f;
    double ld = DBL_MAX;
    int li = INT_MAX;
    int have = 0;
    int32_t held = 0;                                      // lane < have: a candidate's tree position
    auto offer = [&]() {
        double cd = DBL_MAX;
        int ci = INT_MAX;
        if (lane < have) {
            ci = perm[held];
            const float *x = Xt + (int64_t)held * (32 * NJ);
            double acc = 0.0;
            float4 nx = *reinterpret_cast<const float4 *>(x);
            for (int k = 0; k < d; k += 4) {
                const float4 xv = nx;
                nx = *reinterpret_cast<const float4 *>(x + min(k + 4, 32 * NJ - 4));
                const float xs[4] = {xv.x, xv.y, xv.z, xv.w};
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (k + e < d) {
                        const double t = c_sub(c_f2d(sy[warp][k + e]), c_f2d(xs[e]));
                        acc = c_add(acc, c_mul(t, t));
                    }
            }
            cd = acc;
        }
        warp_offer(ld, li, cd, ci, kappa, false, lane);
        have = 0;
    };
    for (int b = 0; b < n; b += 32) {
        // not "above the limit", so a NaN distance stays in
        const bool pass = b + lane < n && !(sd[warp][b + lane] > lim);
        const unsigned m = __ballot_sync(FULL, pass);
        const int32_t p = pass ? c[b + lane] : 0;
        // the passing lanes' positions, in order, behind those held
        warp_collect(m, p, have, held, lane, offer);
    }
    if (have > 0) offer();
    if (lane < kappa) {
        ids[src * kappa + lane] = li;
        dist[src * kappa + lane] = ld;
    }
}

// Radius of every leaf's ball around its center, rounded up, from the squared norms of
// its centered rows (FP64 sums of FP32 differences, rounded).
__global__ void ko_radius_kernel(const float *nrmc, const int32_t *nstart, const int32_t *nsize, int64_t M, float *rad) {
    const int lane = threadIdx.x & 31;
    const int64_t l = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (l >= M) return;                                    // warp-uniform
    float m = 0.f;
    for (int i = lane; i < nsize[M + l]; i += 32) m = fmaxf(m, nrmc[nstart[M + l] + i]);
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(FULL, m, o));
    if (lane == 0) rad[l] = sqrtf(m) * (1.f + 2e-6f) + 1e-18f;
}

// A query with too many candidates, a block per query: its warps take the leaves in
// turn, 32 centers at a time (a lane each), and scan those that |y - c| - radius leaves
// within sqrt(U), or the root of the warp's kappa-th FP64 distance so far.  FP32
// distances within the same limit get their FP64 distance, 32 to a batch; the warps'
// lists are merged at the end.
// Overflow comes with tight clusters or few intrinsic dimensions, where the balls rule
// out nearly all leaves: 3,001 queries against 1M points of a curve in 3 dimensions
// took 38.4 ms with the exhaustive search here, 1.6 so; 50,000 against 64 clusters of
// 2,048 points 88.3 ms and 7.6.  Where they rule out little -- two clusters of 65,536
// points in 16 and in 64 dimensions -- 50,000 queries take 29.9 and 69 ms (92 and 231).
constexpr int BA_WARPS = 8;
template <int NJ>
__global__ void __launch_bounds__(32 * BA_WARPS) ko_ball_kernel(const float *Xt, const float *Y, int d,
                                                                const int32_t *order, const int32_t *rows,
                                                                const int32_t *perm, const float *U, const float *cent,
                                                                const int32_t *leaf_cbase, const float *rad, int64_t M,
                                                                const int32_t *nstart, const int32_t *nsize, int kappa,
                                                                int32_t *ids, double *dist) {
    __shared__ float sy[TC_K];
    __shared__ double sd[BA_WARPS][32];
    __shared__ int si[BA_WARPS][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t q = rows[blockIdx.x], src = order ? order[q] : q;
    for (int k = threadIdx.x; k < TC_K; k += 32 * BA_WARPS) sy[k] = k < d ? Y[src * d + k] : 0.f;
    float4 y[NJ];
    load_query<NJ>(Y + src * d, d, lane, y);
    __syncthreads();
    const float gam = sum_gam(d);
    float lim = U[q] * (1.f + gam) + 1e-37f;               // FP32 distances of the kappa nearest are within this
    double ld = DBL_MAX;
    int li = INT_MAX, have = 0;
    int32_t held = 0;                                      // lane < have: a candidate's tree position
    auto offer = [&]() {
        double cd = DBL_MAX;
        int ci = INT_MAX;
        if (lane < have) {
            ci = perm[held];
            cd = c_dist2(sy, Xt + (int64_t)held * (32 * NJ), d);
        }
        warp_offer(ld, li, cd, ci, kappa, false, lane);
        have = 0;
        // the limit follows the list here alone: its two FP64 instructions would hold the
        // warp's quarter of the SM in every step of the scan
        const double kth = __shfl_sync(FULL, ld, kappa - 1);
        if (kth < 1e38) lim = fminf(lim, __double2float_ru(kth) * (1.f + 2.f * gam) + 1e-37f);
    };
    for (int64_t l0 = 32 * (int64_t)warp; l0 < M; l0 += 32 * BA_WARPS) {
        const int64_t l = l0 + lane;
        bool in = l < M;
        if (in) {
            const float4 *c = reinterpret_cast<const float4 *>(cent + (int64_t)leaf_cbase[l] * TC_K);
            float acc = 0.f;
#pragma unroll 4
            for (int k = 0; k < 8 * NJ; ++k) {
                const float4 v = c[k];
                const float t0 = sy[4 * k] - v.x, t1 = sy[4 * k + 1] - v.y, t2 = sy[4 * k + 2] - v.z, t3 = sy[4 * k + 3] - v.w;
                acc = fmaf(t0, t0, acc);
                acc = fmaf(t1, t1, acc);
                acc = fmaf(t2, t2, acc);
                acc = fmaf(t3, t3, acc);
            }
            in = !(sqrtf(acc) * (1.f - gam - 4e-6f) - rad[l] > sqrtf(lim) * (1.f + 2e-6f));
        }
        unsigned m = __ballot_sync(FULL, in);
        while (m) {
            const int64_t leaf = l0 + __ffs(m) - 1;
            m &= m - 1;
            const int p0 = nstart[M + leaf], np = nsize[M + leaf];
            for (int b = 0; b < np; b += 32) {
                // rows past the leaf are other points or the zero rows past N
                const float v = rows32<NJ, true>(Xt, y, lane, [&](int i) { return p0 + b + i; });
                const int i = b + 4 * (lane & 7) + (lane >> 3);
                const unsigned hit = __ballot_sync(FULL, i < np && v <= lim);
                // the lanes' rows are not in lane order: positions travel with the hits
                if (hit) warp_collect(hit, p0 + i, have, held, lane, offer);
            }
        }
    }
    if (have > 0) offer();
    sd[warp][lane] = ld;
    si[warp][lane] = li;
    __syncthreads();
    if (warp) return;
    for (int w = 1; w < BA_WARPS; ++w) warp_offer(ld, li, sd[w][lane], si[w][lane], kappa, false, lane);
    if (lane < kappa) {
        ids[src * kappa + lane] = li;
        dist[src * kappa + lane] = ld;
    }
}

// ---------------------------------------------------------------------------
// Step 3.  A tile of 256 tree positions stays in shared memory while tiles of 128
// queries stream through four stages (TMA, 128-byte swizzled K-major FP16 hi and
// lo); 12 tcgen05.mma (128 x 256 x 16) a tile pair leave sigma^2 a.b in one of two
// 256-column TMEM accumulators; each of the four epilogue groups takes 64 columns:
// n_j - 2 a.b / sigma^2 against the query's threshold, 32 columns' minimum first.
// 12 MMAs of 128 cycles a tile pair against about 1300 issue slots of the epilogue:
// with two groups the epilogue's latency bound it (tensor pipe 43 %, issue 36 %).
// (source tile, query tile) pairs are dealt in contiguous ranges of equal length,
// one CTA an SM.
//   warps 0-15 epilogue, group g = columns 64 g ..
//   warp 16    TMA
//   warp 17    TMEM allocation, MMA issue
// Every wait is bounded (ASK_DEV_TIMEOUT).
// ---------------------------------------------------------------------------
constexpr int KS_REGION = 128 * 128;           // 128 rows x 64 FP16
constexpr int KS_NA = 4;
struct KS {
    static constexpr int B_HI = 0, B_LO = 2 * KS_REGION;
    static constexpr int A0 = 4 * KS_REGION;                   // stage: hi, lo
    static constexpr int COL = A0 + KS_NA * 2 * KS_REGION;     // float [2][256] n_j
    static constexpr int BAR = COL + 2 * 256 * 4;              // 20 mbarriers
    static constexpr int MISC = BAR + 20 * 8;
    static constexpr int BYTES = MISC + 16;
    static constexpr int THREADS = 576;
};
struct KSArgs {
    int64_t N, T, units;                       // units = source tiles x query tiles
    int n_qt;
    const float *nt;                           // [N_pad] |x - xbar|^2 of the tree rows
    const float *nq, *U;                       // per query
    float m2u, eta, abs;                       // -2 / sigma^2, KO_ETA, KO_ABS / sigma^2
    int *cnt;
    int32_t *cand;
    int *status;
};

__global__ void __launch_bounds__(KS::THREADS, 1)
ko_shortlist_kernel(const __grid_constant__ CUtensorMap map_qh, const __grid_constant__ CUtensorMap map_ql,
                    const __grid_constant__ CUtensorMap map_th, const __grid_constant__ CUtensorMap map_tl,
                    const KSArgs args) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t *sm = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const uint32_t sbase = smem_u32(sm), bar0 = sbase + KS::BAR;
    auto BAR_A_FULL = [&](int s) { return bar0 + 8 * s; };
    auto BAR_A_EMPTY = [&](int s) { return bar0 + 8 * (4 + s); };
    const uint32_t BAR_B_FULL = bar0 + 8 * 8, BAR_B_EMPTY = bar0 + 8 * 9;
    auto BAR_T_FULL = [&](int a) { return bar0 + 8 * (10 + a); };
    auto BAR_T_EMPTY = [&](int a) { return bar0 + 8 * (12 + a); };
    auto BAR_C_FULL = [&](int s) { return bar0 + 8 * (14 + s); };   // n_j of source tile (slot lb & 1)
    auto BAR_C_EMPTY = [&](int s) { return bar0 + 8 * (16 + s); };
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(sm + KS::MISC);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(sm + KS::MISC + 4);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        for (int s = 0; s < KS_NA; ++s) {
            mbar_init(BAR_A_FULL(s), 1);
            mbar_init(BAR_A_EMPTY(s), 1);
        }
        mbar_init(BAR_B_FULL, 1);
        mbar_init(BAR_B_EMPTY, 1);
        for (int a = 0; a < 2; ++a) {
            mbar_init(BAR_T_FULL(a), 1);
            mbar_init(BAR_T_EMPTY(a), 512);
            mbar_init(BAR_C_FULL(a), 1);
            mbar_init(BAR_C_EMPTY(a), 512);
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 17) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(tmem_slot)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    // this CTA's units u0 .. u1 - 1; unit u: source tile u / n_qt, query tile u % n_qt
    const int64_t u0 = args.units * blockIdx.x / gridDim.x, u1 = args.units * (blockIdx.x + 1) / gridDim.x;
    const int n_qt = args.n_qt;

    if (warp < 16) {
        const int q4 = warp & 3, eg = warp >> 2, row = q4 * 32 + lane;
        int li = 0, lb = -1;
        int64_t bt = -1;
        const float *col = nullptr;
        const float m2 = args.m2u / (1.f - args.eta);
        const float2 m22 = make_float2(m2, m2);
        // this row's query of a unit: n_j (1 - eta) - 2 a.b <= U (1 + eta) - n_q (1 - eta) + abs
        auto load = [&](int64_t u, float &un, float &nn) {
            const int64_t q = u < u1 ? (u % n_qt) * 128 + row : args.T;
            un = q < args.T ? args.U[q] : -INFINITY;
            nn = q < args.T ? args.nq[q] : 0.f;
        };
        float un, nn;
        load(u0, un, nn);
        // A unit's hits stay in two masks; their places in the query's list come
        // from one counter update a unit, whose answer is waited for only after the
        // next unit (waiting for one a chunk made the epilogue three times as long
        // as the MMAs)
        uint32_t ph[2] = {0, 0};
        int pk = 0;
        int64_t pq = 0, pp = 0;
        auto flush = [&]() {
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                uint32_t m = pk < KO_CAP ? ph[c] : 0u;     // a full list takes no more
                while (m) {
                    const int j = __ffs(m) - 1;
                    m &= m - 1;
                    if (pk < KO_CAP) args.cand[pq * KO_CAP + pk] = (int32_t)(pp + 32 * c + j);
                    ++pk;
                }
            }
            __syncwarp();
        };
        for (int64_t u = u0; u < u1; ++u, ++li) {
            const int64_t b = u / n_qt;
            const int qt = (int)(u - b * n_qt);
            if (b != bt) {
                if (lb >= 0) mbar_arrive(BAR_C_EMPTY(lb & 1));
                ++lb;
                bt = b;
                if (!mbar_wait(BAR_C_FULL(lb & 1), (lb >> 1) & 1, abort_flag, args.status)) break;
                col = reinterpret_cast<const float *>(sm + KS::COL) + (lb & 1) * 256 + 64 * eg;
            }
            const int64_t q = (int64_t)qt * 128 + row;
            const float thr = (un * (1.f + args.eta) + args.abs) / (1.f - args.eta) - nn;
            load(u + 1, un, nn);
            const int a = li & 1;
            if (!mbar_wait(BAR_T_FULL(a), (li >> 1) & 1, abort_flag, args.status)) break;
            tc_fence_after();
            const uint32_t tbase = tmem + ((uint32_t)(q4 * 32) << 16) + (uint32_t)(a * 256 + 64 * eg);
            const int64_t pos0 = b * 256 + 64 * eg;
            auto chunk = [&](int c, const uint32_t (&g)[32]) -> uint32_t {
                float dd[32], m4[4] = {INFINITY, INFINITY, INFINITY, INFINITY};
#pragma unroll
                for (int j = 0; j < 32; j += 4) {
                    const float4 n4 = *reinterpret_cast<const float4 *>(col + c * 32 + j);
                    const float2 x = __ffma2_rn(make_float2(__uint_as_float(g[j]), __uint_as_float(g[j + 1])), m22,
                                                make_float2(n4.x, n4.y));
                    const float2 z = __ffma2_rn(make_float2(__uint_as_float(g[j + 2]), __uint_as_float(g[j + 3])), m22,
                                                make_float2(n4.z, n4.w));
                    dd[j] = x.x;
                    dd[j + 1] = x.y;
                    dd[j + 2] = z.x;
                    dd[j + 3] = z.y;
                    m4[(j >> 2) & 3] = fminf(m4[(j >> 2) & 3], fminf(fminf(x.x, x.y), fminf(z.x, z.y)));
                }
                const float m = fminf(fminf(m4[0], m4[1]), fminf(m4[2], m4[3]));
                uint32_t hit = 0;
                if (__any_sync(FULL, m <= thr)) {
                    uint32_t h4[4] = {0, 0, 0, 0};         // four chains instead of one of 32
#pragma unroll
                    for (int j = 0; j < 32; ++j) h4[j & 3] |= dd[j] <= thr ? 1u << j : 0u;
                    hit = (h4[0] | h4[1]) | (h4[2] | h4[3]);
                    const int64_t p0 = pos0 + c * 32;
                    if (p0 + 32 > args.N) hit &= p0 < args.N ? (1u << (args.N - p0)) - 1u : 0u;   // rows past N
                }
                return hit;
            };
            uint32_t ga[32], gb[32], hit[2];
            tmem_ld32_async(tbase, ga);
            tmem_wait_pin(ga);
            tmem_ld32_async(tbase + 32, gb);
            hit[0] = chunk(0, ga);
            tmem_wait_pin(gb);
            tc_fence_before();
            mbar_arrive(BAR_T_EMPTY(a));       // all columns are in registers
            hit[1] = chunk(1, gb);
            flush();
            const int n = __popc(hit[0]) + __popc(hit[1]);
            if (n) pk = atomicAdd(args.cnt + q, n);
            __syncwarp();
            pq = q;
            pp = pos0;
#pragma unroll
            for (int c = 0; c < 2; ++c) ph[c] = hit[c];
        }
        flush();
    } else if (warp == 16 && lane == 0) {
        int li = 0, lb = -1;
        int64_t bt = -1;
        for (int64_t u = u0; u < u1; ++u, ++li) {
            const int64_t b = u / n_qt;
            const int qt = (int)(u - b * n_qt);
            if (b != bt) {
                ++lb;
                bt = b;
                const int cs = lb & 1;
                if (!mbar_wait(BAR_C_EMPTY(cs), ((lb >> 1) & 1) ^ 1, abort_flag, args.status)) { --lb; goto tma_done; }
                mbar_expect_tx(BAR_C_FULL(cs), 1024);
                bulk_copy(sbase + KS::COL + cs * 1024, args.nt + b * 256, 1024, BAR_C_FULL(cs));
                if (!mbar_wait(BAR_B_EMPTY, (lb & 1) ^ 1, abort_flag, args.status)) {
                    mbar_drain(BAR_C_FULL(cs), (lb >> 1) & 1);
                    --lb;
                    goto tma_done;
                }
                mbar_expect_tx(BAR_B_FULL, 4 * KS_REGION);
                for (int h = 0; h < 2; ++h) {
                    tma_load_2d(sbase + KS::B_HI + h * KS_REGION, &map_th, 0, (int)(b * 256 + 128 * h), BAR_B_FULL);
                    tma_load_2d(sbase + KS::B_LO + h * KS_REGION, &map_tl, 0, (int)(b * 256 + 128 * h), BAR_B_FULL);
                }
            }
            const int s = li % KS_NA;
            if (!mbar_wait(BAR_A_EMPTY(s), ((li / KS_NA) & 1) ^ 1, abort_flag, args.status)) goto tma_done;
            const uint32_t st = sbase + KS::A0 + s * 2 * KS_REGION;
            mbar_expect_tx(BAR_A_FULL(s), 2 * KS_REGION);
            tma_load_2d(st, &map_qh, 0, qt * 128, BAR_A_FULL(s));
            tma_load_2d(st + KS_REGION, &map_ql, 0, qt * 128, BAR_A_FULL(s));
        }
    tma_done:
        // nothing may land in shared memory after the CTA has left (no-ops unless
        // a wait gave up)
        for (int k = li > KS_NA ? li - KS_NA : 0; k < li; ++k) mbar_drain(BAR_A_FULL(k % KS_NA), (k / KS_NA) & 1);
        if (lb >= 0) {
            mbar_drain(BAR_B_FULL, lb & 1);
            mbar_drain(BAR_C_FULL(lb & 1), (lb >> 1) & 1);
        }
    } else if (warp == 17 && lane == 0) {
        constexpr uint32_t IDESC = make_idesc(0u, 128, 256);
        int li = 0, lb = -1, done = -1;
        int64_t bt = -1;
        for (int64_t u = u0; u < u1; ++u, ++li) {
            const int64_t b = u / n_qt;
            if (b != bt) {
                if (lb >= 0) tc_commit(BAR_B_EMPTY);       // the last tile's MMAs have read it
                ++lb;
                bt = b;
                if (!mbar_wait(BAR_B_FULL, lb & 1, abort_flag, args.status)) break;
            }
            const int s = li % KS_NA, a = li & 1;
            if (!mbar_wait(BAR_A_FULL(s), (li / KS_NA) & 1, abort_flag, args.status)) break;
            if (!mbar_wait(BAR_T_EMPTY(a), ((li >> 1) & 1) ^ 1, abort_flag, args.status)) break;
            tc_fence_after();
            const uint32_t dt = tmem + (uint32_t)(a * 256);
            const uint32_t ah = sbase + KS::A0 + s * 2 * KS_REGION, al = ah + KS_REGION;
            const uint32_t bh = sbase + KS::B_HI, bl = sbase + KS::B_LO;
#pragma unroll
            for (int k = 0; k < 4; ++k) {                  // the small cross terms first
                const uint32_t off = (uint32_t)(k * 32);
                tc_mma<ASKIT_PREC_FP16X3>(dt, sw128_desc(ah + off), sw128_desc(bl + off), IDESC, k > 0);
                tc_mma<ASKIT_PREC_FP16X3>(dt, sw128_desc(al + off), sw128_desc(bh + off), IDESC, 1);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t off = (uint32_t)(k * 32);
                tc_mma<ASKIT_PREC_FP16X3>(dt, sw128_desc(ah + off), sw128_desc(bh + off), IDESC, 1);
            }
            tc_commit(BAR_A_EMPTY(s));
            tc_commit(BAR_T_FULL(a));
            done = li;
        }
        // MMAs in flight after an abort end before TMEM is freed
        if (done >= 0) mbar_drain(BAR_T_FULL(done & 1), (done >> 1) & 1);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 17) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
    }
}

__global__ void ko_gather_kernel(const float *Y, int d, const int32_t *rows, int64_t n, float *out) {
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= n * d) return;
    out[e] = Y[(int64_t)rows[e / d] * d + e % d];
}

__global__ void ko_scatter_kernel(const int32_t *ids_s, const double *dist_s, const int32_t *rows, int64_t n,
                                  int kappa, int32_t *ids, double *dist) {
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= n * kappa) return;
    const int64_t q = rows[e / kappa];
    ids[q * kappa + e % kappa] = ids_s[e];
    dist[q * kappa + e % kappa] = dist_s[e];
}

// Tensor maps of the tree's split target rows, here the shortlist's sources.
askit_status tree_maps(askit_tree t, EncodeTiledFn fn, CUtensorMap *th, CUtensorMap *tl) {
    ASK_TRY(encode_2d(fn, th, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, t->Xg_hi, t->N_pad, TC_K, 64, 128,
                      CU_TENSOR_MAP_SWIZZLE_128B));
    return encode_2d(fn, tl, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, t->Xg_lo, t->N_pad, TC_K, 64, 128,
                     CU_TENSOR_MAP_SWIZZLE_128B);
}

// Whether the shortlist's FP32 figures stay finite and normal: the tree's norms below
// 1e37, those of queries in the FP16-safe range (|y_k - xbar_k| sigma <= 30000) at most
// 5.8e10 / sigma^2 < 6e36, so every squared distance below 3.2e37; and 2 / sigma^2,
// KO_ABS / sigma^2 normal.
bool fp32_safe(const askit_tree_s *t) {
    const double s2 = (double)t->g_sigma * t->g_sigma;
    return t->g_r2max < 1e37 && s2 > 1e-26 && s2 < 1e30;
}

}  // namespace

askit_status knn_oos(askit_tree t, const float *Y, int64_t T, int kappa, int32_t *ids, double *dist, cudaStream_t s) {
    if (!t->Xg_hi || t->d > TC_K || kappa > 32 || !fp32_safe(t))
        return knn_exact_gpu(t->X, t->N, t->d, kappa, Y, T, ids, dist, s);
    const int d = t->d;
    const int64_t M = (int64_t)1 << t->L, N = t->N;
    const int64_t T_pad = (T + 127) / 128 * 128;
    // splits of the leaf centers, so that few queries still fill the GPU
    int sms = 0, dev = 0;
    ASK_CUDA(cudaGetDevice(&dev));
    ASK_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const int64_t qb = (T + HO_T - 1) / HO_T;
    int64_t nsplit = std::max<int64_t>(1, std::min<int64_t>(16, std::min<int64_t>((M + HO_T - 1) / HO_T, sms / qb)));
    const int64_t split_len = ((M + nsplit - 1) / nsplit + HO_T - 1) / HO_T * HO_T;
    nsplit = (M + split_len - 1) / split_len;
    DevArena tmp;
    tmp.async = true;
    tmp.stream = s;
    tmp.pool = t->pool;
    // one allocation: every part at a multiple of 256 bytes
    size_t used = 0;
    auto part = [&](size_t bytes) {
        const size_t o = used;
        used += (bytes + 255) / 256 * 256;
        return o;
    };
    const size_t o_hi = part((size_t)T_pad * TC_K * 2), o_lo = part((size_t)T_pad * TC_K * 2), o_nq = part((size_t)T_pad * 4),
                 o_hd = part((size_t)nsplit * T * 8), o_hx = part((size_t)nsplit * T * 8), o_u = part((size_t)T * 4),
                 o_cnt = part((size_t)T * 4), o_ord = part((size_t)T * 4), o_ovf = part((size_t)(2 * T + 2) * 4),
                 o_rad = part((size_t)M * 4), o_cand = part((size_t)T * KO_CAP * 4);
    uint8_t *buf = nullptr;
    ASK_TRY(tmp.alloc(&buf, used));
    uint16_t *qh = reinterpret_cast<uint16_t *>(buf + o_hi), *ql = reinterpret_cast<uint16_t *>(buf + o_lo);
    float *nq = reinterpret_cast<float *>(buf + o_nq), *hd = reinterpret_cast<float *>(buf + o_hd),
          *U = reinterpret_cast<float *>(buf + o_u);
    int32_t *hx = reinterpret_cast<int32_t *>(buf + o_hx), *cand = reinterpret_cast<int32_t *>(buf + o_cand);
    int *cnt = reinterpret_cast<int *>(buf + o_cnt), *n_ovf = reinterpret_cast<int *>(buf + o_ovf);
    int32_t *ovf = n_ovf + 2, *wide = ovf + T;
    float *rad = reinterpret_cast<float *>(buf + o_rad);
    const int32_t *order = nullptr;
    int h_n[2] = {0, 0}, h_ovf = 0;
    askit_status rc = ASKIT_OK;
#define QTRY(x) do { rc = (x); if (rc != ASKIT_OK) goto out; } while (0)
#define QCHK(x) do { const cudaError_t e_ = (x); if (e_ != cudaSuccess) { askit_set_error("out-of-sample kNN: %s", cudaGetErrorString(e_)); rc = e_ == cudaErrorMemoryAllocation ? ASKIT_ERR_OOM : ASKIT_ERR_CUDA; goto out; } } while (0)
    QCHK(cudaMemsetAsync(n_ovf, 0, 2 * sizeof(int), s));
    ko_home_kernel<<<dim3((unsigned)qb, (unsigned)nsplit), 128, 0, s>>>(Y, d, T, t->cent, t->leaf_cbase, M, split_len, hd,
                                                                        hx);
    // Queries in the order of their home leaves: the 128 of a tile then have their
    // candidates in the same few source tiles, and nearly all other tile pairs skip
    // the hit path; the seed's leaves are shared by neighboring warps.  The saving is
    // in proportion to the (query, point) pairs, the sort's few launches (about 20 us)
    // are not.  knn_targets against 131,072 points of 64 dimensions, in the given order
    // and sorted: 3,001 queries 557 and 567 us, 5,000 735 and 730, 10,000 (1.3e9 pairs)
    // 1073 and 1026, 16,400 (2.1e9) 1510 and 1405, 100,000 7.15 and 6.43 ms; against
    // 1M, 2,500 (2.6e9) 1343 and 1334 us, 20,000 15.05 and 14.86 ms.  It pays from
    // about 10^9 pairs on; the line lies at 2^31, where it does at every size measured.
    if (t->L > 0 && T >= 16 * sms && T * N >= (int64_t)1 << 31) {
        // the sort's buffers lie in the candidate lists, which are written later
        const size_t T4 = ((size_t)T * 4 + 255) / 256 * 256;
        uint8_t *sb = buf + o_cand;
        uint32_t *key = reinterpret_cast<uint32_t *>(sb), *key2 = reinterpret_cast<uint32_t *>(sb + T4);
        int32_t *iota = reinterpret_cast<int32_t *>(sb + 2 * T4);
        size_t tb = 0;
        QTRY(sort_u32_i32(key, key2, iota, iota, T, t->L, nullptr, &tb, s));
        if (3 * T4 + tb <= (size_t)T * KO_CAP * 4) {
            int32_t *ord = reinterpret_cast<int32_t *>(buf + o_ord);
            ko_key_kernel<<<nblk(T, 256), 256, 0, s>>>(hd, hx, (int)nsplit, T, key, iota);
            QTRY(sort_u32_i32(key, key2, iota, ord, T, t->L, sb + 3 * T4, &tb, s));
            order = ord;
        }
    }
    ko_split_kernel<<<nblk(T_pad, 8), 256, 0, s>>>(Y, d, order, T, T_pad, t->g_xbar, t->g_sigma, qh, ql, nq, cnt);
    {
        // Below 16 queries an SM one warp a query leaves the GPU short of warps.  Against
        // 131,072 points, four warps and one: 500 queries 373 and 393 us, 1,000 408 and
        // 433, 1,500 444 and 454, 2,432 (the line) 505 and 502, 5,000 725 and 726,
        // 16,400 1452 and 1402
        const bool few = T < 16 * sms;
        auto seed = d <= 32 ? (few ? ko_seed_kernel<1, 4> : ko_seed_kernel<1, 1>)
                            : (few ? ko_seed_kernel<2, 4> : ko_seed_kernel<2, 1>);
        seed<<<nblk(T, few ? 2 : 8), 256, 0, s>>>(t->Xt, Y, d, order, T, hd, hx, (int)nsplit, M, t->nstart, t->nsize, kappa, U);
    }
    QCHK(cudaGetLastError());
    {
        EncodeTiledFn fn = nullptr;
        CUtensorMap mth, mtl, mqh, mql;
        QTRY(encode_fn(&fn));
        QTRY(tree_maps(t, fn, &mth, &mtl));
        QTRY(encode_2d(fn, &mqh, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, qh, T_pad, TC_K, 64, 128, CU_TENSOR_MAP_SWIZZLE_128B));
        QTRY(encode_2d(fn, &mql, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, ql, T_pad, TC_K, 64, 128, CU_TENSOR_MAP_SWIZZLE_128B));
        KSArgs a;
        a.N = N;
        a.T = T;
        a.n_qt = (int)(T_pad / 128);
        a.units = (N + 255) / 256 * a.n_qt;
        a.nt = t->ng_t;
        a.nq = nq;
        a.U = U;
        a.m2u = -2.f / (t->g_sigma * t->g_sigma);
        a.eta = KO_ETA;
        a.abs = KO_ABS / (t->g_sigma * t->g_sigma);
        a.cnt = cnt;
        a.cand = cand;
        a.status = t->d_status;
        constexpr size_t smem = KS::BYTES + 1024;
        static_assert(smem <= 232448, "shared-memory plan exceeds 227 KB");
        static std::atomic<uint64_t> opted{0};
        QTRY(opt_in_smem(ko_shortlist_kernel, smem, opted));
        ko_shortlist_kernel<<<(unsigned)std::min<int64_t>(sms, a.units), KS::THREADS, smem, s>>>(mqh, mql, mth, mtl, a);
        QCHK(cudaGetLastError());
    }
    {
        // (Queries without a bound, 131,072 x 64, leaves of 12: 100 / 3,001 / 50,000 take 2.6 /
        // 23 / 370 ms leaf by leaf, 8.0 / 64 / 239 in the exhaustive search's tiles, whose
        // lines cross at about 14,400: 96 an SM.)
        // One warp a block or eight: against 131,072 points within 1 % either way from 500
        // queries on (500 380 and 372 us, 2,432 510 and 505, 16,400 1391 and 1403); against
        // 1M, 500 queries 605 and 628
        const bool few = T < 16 * sms;
        auto rerank = t->d_pad == 32 ? (few ? ko_rerank_kernel<1, 1> : ko_rerank_kernel<1, 8>)
                                     : (few ? ko_rerank_kernel<2, 1> : ko_rerank_kernel<2, 8>);
        rerank<<<nblk(T, few ? 1 : 8), few ? 32 : 256, 0, s>>>(t->Xt, Y, d, order, T, t->perm, cnt, cand, kappa, ids, dist,
                                                              n_ovf, ovf, wide, U, T >= 96 * sms);
    }
    QCHK(cudaGetLastError());
    QCHK(cudaMemcpyAsync(h_n, n_ovf, sizeof h_n, cudaMemcpyDeviceToHost, s));
    QCHK(cudaStreamSynchronize(s));
    h_ovf = h_n[0];
    if (h_n[1] > 0) {
        ko_radius_kernel<<<nblk(M, 8), 256, 0, s>>>(t->nrmc_t, t->nstart, t->nsize, M, rad);
        auto ball = t->d_pad == 32 ? ko_ball_kernel<1> : ko_ball_kernel<2>;
        ball<<<(unsigned)h_n[1], 32 * BA_WARPS, 0, s>>>(t->Xt, Y, d, order, wide, t->perm, U, t->cent, t->leaf_cbase, rad, M,
                                                       t->nstart, t->nsize, kappa, ids, dist);
        QCHK(cudaGetLastError());
        if (h_ovf == 0) QCHK(cudaStreamSynchronize(s));
    }
    if (h_ovf > 0) {
        // the exhaustive search
        float *Ys = nullptr;
        int32_t *ids_s = nullptr;
        double *dist_s = nullptr;
        QTRY(tmp.alloc(&Ys, (size_t)h_ovf * d));
        QTRY(tmp.alloc(&ids_s, (size_t)h_ovf * kappa));
        QTRY(tmp.alloc(&dist_s, (size_t)h_ovf * kappa));
        ko_gather_kernel<<<nblk((int64_t)h_ovf * d, 256), 256, 0, s>>>(Y, d, ovf, h_ovf, Ys);
        QTRY(knn_exact_gpu(t->X, N, d, kappa, Ys, h_ovf, ids_s, dist_s, s));
        ko_scatter_kernel<<<nblk((int64_t)h_ovf * kappa, 256), 256, 0, s>>>(ids_s, dist_s, ovf, h_ovf, kappa, ids, dist);
        QCHK(cudaGetLastError());
        QCHK(cudaStreamSynchronize(s));
    }
out:
#undef QTRY
#undef QCHK
    tmp.free_all();
    return rc;
}
