// Evaluate (Algorithm 4) on CUDA cores in plain FP32: the reference
// precision the split tensor-core paths are measured against.
//
// A block takes items of one source sub-block (a leaf's points, evaluated
// directly, or a node's skeleton, Algorithm 4 lines 1-2): up to 128 targets
// against up to 128 sources, 256 threads, 8 x 8 pairs a thread, with the distance
// in difference form (no cancellation), coordinates ascending, one FMA each, slices of
// SI_K summed apart and then added up, and the exponent on exp2f:
//     sum_j exp(-c ||x - y_j||^2 / h_j^2) w_j
// Bound by the FP32 lanes (2 d operations a pair).  A thread a target with its
// sources read one word at a time was bound by shared memory at a quarter of them
// (one 4-byte read for two operations); here 6 16-byte reads a thread and
// coordinate serve 128 operations, as 64 packed instructions: target coordinates
// are staged twice over, (x, x), and sources negated, so that a packed add gives
// two differences and a packed FMA two squares.  Two blocks share an SM, one
// computing while the other stages.
// The kernel values pass through shared memory (over the staged targets) to the
// weight sums: thread (t, h) sums target t over the sources of half h, in order,
// and the halves are added, whatever the number of vectors, so that a vector's
// result does not depend on how many others share its evaluation.
// Measured, 64K x 64, r = 1 (468 M pairs): 10.1 -> 2.2 ms, 0.67 of the lanes' rate.
#include <algorithm>

#include "askit_impl.cuh"

namespace {

constexpr int SI_THREADS = 256;
constexpr int SI_K = 64;                          // coordinates per staged slice
constexpr int SI_X = SI_K * ASK_TILE_M * 2;       // floats: (x, x) pairs [k][128], later the kernel values [source][128]
constexpr int SI_Y = SI_K * ASK_BLK_N;            // floats: -y [k][128]
constexpr int SI_SC = SI_X + SI_Y;                // c log2(e) / h^2 [128]
constexpr int SI_W = SI_SC + ASK_BLK_N;           // weights [128][rz], then the second half's sums [128][ZC]
static_assert(SI_X == ASK_TILE_M * ASK_BLK_N, "the kernel values take the staged targets' place");

// Kernel value of target t and source j: 16-byte pieces of a source's row are
// permuted by the source, so that both the stores (a warp: 16 source groups) and
// the reads (a warp: 32 targets of one source) are free of bank conflicts.
__device__ __forceinline__ int si_kv(int j, int t) {
    return j * ASK_TILE_M + ((((t >> 2) ^ (j >> 2)) & 31) << 2) + (t & 3);
}

// DEEP (d_pad > SI_K): the slices' sums are added up in a second set of registers, at
// one block an SM.  A single chain of d additions rounds d times at the full distance:
// relative error against FP64 for 2,000 points 2.7e-7 (d = 300), 4.3e-7 (1000) and
// 5.3e-7 (4000), with the slices apart 1.8e-7, 1.8e-7 and 1.4e-7; 10K x 1000 5.2 ms an
// Evaluate (4.6 in a chain at two blocks an SM).
template <int ZC, bool DEEP>
__global__ void __launch_bounds__(SI_THREADS, DEEP ? 1 : 2) eval_simt_kernel(
    const float *__restrict__ Xq, int64_t ldq, const EvalItem *__restrict__ items,
    const int32_t *__restrict__ block_off, const int32_t *__restrict__ block_order,
    const int32_t *__restrict__ tgt, float *__restrict__ partial, const float *__restrict__ Xt,
    const float *__restrict__ Xs, const float *__restrict__ sc_t, const float *__restrict__ sc_s,
    const float *__restrict__ Wt, const float *__restrict__ Ws, int d_pad, int r) {
    extern __shared__ __align__(16) float sm[];
    const int b = block_order[blockIdx.x];
    const int i0 = block_off[b] + blockIdx.y, i1 = block_off[b + 1];
    if (i0 >= i1) return;                                       // block-uniform
    const int tid = threadIdx.x;
    const int t = tid & 127, h = tid >> 7;                      // staging and weight sums
    const int ty = tid >> 4, tx = tid & 15;                     // pairs: targets 8 ty .., sources 4 tx .. and 64 + 4 tx ..
    const int rz = (r + ZC - 1) / ZC * ZC;
    float *sx = sm, *sy = sm + SI_X, *ssc = sm + SI_SC, *sw = sm + SI_W, *comb = sw + ASK_BLK_N * rz;
    const EvalItem first = items[i0];
    const bool far = first.nrows < 0;
    const int nrows = first.nrows & 0x7fffffff;
    const float *Y = (far ? Xs : Xt) + (int64_t)first.row0 * d_pad;
    const float *WW = (far ? Ws : Wt) + (int64_t)first.row0 * r;
    if (tid < ASK_BLK_N) ssc[tid] = tid < nrows ? (far ? sc_s : sc_t)[first.row0 + tid] : 0.f;
    for (int e = tid; e < ASK_BLK_N * rz; e += SI_THREADS) {
        const int j = e / rz, z = e % rz;
        sw[e] = (j < nrows && z < r) ? WW[(int64_t)j * r + z] : 0.f;
    }
    auto stage_y = [&](int k0) {
        for (int k4 = h; k4 < SI_K / 4; k4 += 2) {
            const bool in = t < nrows && k0 + 4 * k4 < d_pad;
            const float4 v = in ? *reinterpret_cast<const float4 *>(Y + (int64_t)t * d_pad + k0 + 4 * k4)
                                : make_float4(0.f, 0.f, 0.f, 0.f);
            sy[(4 * k4 + 0) * ASK_BLK_N + t] = -v.x;
            sy[(4 * k4 + 1) * ASK_BLK_N + t] = -v.y;
            sy[(4 * k4 + 2) * ASK_BLK_N + t] = -v.z;
            sy[(4 * k4 + 3) * ASK_BLK_N + t] = -v.w;
        }
    };
    const bool one_slice = d_pad <= SI_K;
    if (one_slice) stage_y(0);                                  // the run's sources stay
    for (int it = i0; it < i1; it += gridDim.y) {
        const EvalItem item = items[it];
        const float *xrow = Xq + (int64_t)tgt[item.e0 + (t < item.cnt ? t : 0)] * ldq;
        float2 acc[8][4];
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int p = 0; p < 4; ++p) acc[i][p] = make_float2(0.f, 0.f);
        float2 total[DEEP ? 8 : 1][4];
        if constexpr (DEEP) {
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int p = 0; p < 4; ++p) total[i][p] = make_float2(0.f, 0.f);
        }
        for (int k0 = 0; k0 < d_pad; k0 += SI_K) {
            __syncthreads();                                    // the last slice, or the last item's kernel values, are read
            float2 *x2 = reinterpret_cast<float2 *>(sx);
#pragma unroll 4
            for (int k4 = h; k4 < SI_K / 4; k4 += 2) {
                const float4 v = k0 + 4 * k4 < d_pad ? *reinterpret_cast<const float4 *>(xrow + k0 + 4 * k4)
                                                     : make_float4(0.f, 0.f, 0.f, 0.f);
                x2[(4 * k4 + 0) * ASK_TILE_M + t] = make_float2(v.x, v.x);
                x2[(4 * k4 + 1) * ASK_TILE_M + t] = make_float2(v.y, v.y);
                x2[(4 * k4 + 2) * ASK_TILE_M + t] = make_float2(v.z, v.z);
                x2[(4 * k4 + 3) * ASK_TILE_M + t] = make_float2(v.w, v.w);
            }
            if (!one_slice) stage_y(k0);
            __syncthreads();
            const int kn = min(SI_K, d_pad - k0);
#pragma unroll 2
            for (int k = 0; k < kn; ++k) {
                const float4 *px = reinterpret_cast<const float4 *>(x2 + k * ASK_TILE_M + 8 * ty);
                const float4 ya = *reinterpret_cast<const float4 *>(sy + k * ASK_BLK_N + 4 * tx);
                const float4 yb = *reinterpret_cast<const float4 *>(sy + k * ASK_BLK_N + 64 + 4 * tx);
                const float2 y[4] = {make_float2(ya.x, ya.y), make_float2(ya.z, ya.w), make_float2(yb.x, yb.y),
                                     make_float2(yb.z, yb.w)};
#pragma unroll
                for (int i2 = 0; i2 < 4; ++i2) {
                    const float4 xx = px[i2];
                    const float2 x[2] = {make_float2(xx.x, xx.y), make_float2(xx.z, xx.w)};
#pragma unroll
                    for (int i = 0; i < 2; ++i)
#pragma unroll
                        for (int p = 0; p < 4; ++p) {
                            const float2 df = __fadd2_rn(x[i], y[p]);
                            acc[2 * i2 + i][p] = __ffma2_rn(df, df, acc[2 * i2 + i][p]);
                        }
                }
            }
            if constexpr (DEEP) {
#pragma unroll
                for (int i = 0; i < 8; ++i)
#pragma unroll
                    for (int p = 0; p < 4; ++p) {
                        total[i][p] = __fadd2_rn(total[i][p], acc[i][p]);
                        acc[i][p] = make_float2(0.f, 0.f);
                    }
            }
        }
        if constexpr (DEEP) {
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int p = 0; p < 4; ++p) acc[i][p] = total[i][p];
        }
        __syncthreads();                                        // the staged targets are read
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int j = (p >> 1) * 64 + 4 * tx + 2 * (p & 1) + e;
                const float msc = -ssc[j];
                float kv[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) kv[i] = j < nrows ? exp2f(msc * (e ? acc[i][p].y : acc[i][p].x)) : 0.f;
                *reinterpret_cast<float4 *>(sx + si_kv(j, 8 * ty)) = make_float4(kv[0], kv[1], kv[2], kv[3]);
                *reinterpret_cast<float4 *>(sx + si_kv(j, 8 * ty + 4)) = make_float4(kv[4], kv[5], kv[6], kv[7]);
            }
        __syncthreads();
        for (int z0 = 0; z0 < r; z0 += ZC) {
            float s[ZC];
#pragma unroll
            for (int z = 0; z < ZC; ++z) s[z] = 0.f;
#pragma unroll 4
            for (int jj = 0; jj < 64; ++jj) {
                const int j = 64 * h + jj;
                const float k = sx[si_kv(j, t)];
                const float *wj = sw + j * rz + z0;
                if constexpr (ZC == 1) {
                    s[0] = fmaf(k, wj[0], s[0]);
                } else {
#pragma unroll
                    for (int z = 0; z < ZC; z += 4) {
                        const float4 w4 = *reinterpret_cast<const float4 *>(wj + z);
                        s[z] = fmaf(k, w4.x, s[z]);
                        s[z + 1] = fmaf(k, w4.y, s[z + 1]);
                        s[z + 2] = fmaf(k, w4.z, s[z + 2]);
                        s[z + 3] = fmaf(k, w4.w, s[z + 3]);
                    }
                }
            }
            if (z0 > 0) __syncthreads();                        // the last vectors' sums are read
            if (h == 1) {
#pragma unroll
                for (int z = 0; z < ZC; ++z) comb[z * ASK_TILE_M + t] = s[z];
            }
            __syncthreads();
            if (h == 0 && t < item.cnt) {
                float *p = partial + (int64_t)(item.e0 + t) * r + z0;
#pragma unroll
                for (int z = 0; z < ZC; ++z)
                    if (z0 + z < r) p[z] = s[z] + comb[z * ASK_TILE_M + t];
            }
        }
    }
}

template <int ZC, bool DEEP>
askit_status launch_simt(askit_tree t, const WeightCtx &c, const float *Xq, int64_t ldq, const WorkLists &w,
                         float *partial, cudaStream_t s) {
    const int rz = (c.r + ZC - 1) / ZC * ZC;
    const size_t smem = sizeof(float) * (size_t)(SI_W + ASK_BLK_N * rz + ASK_TILE_M * ZC);
    constexpr int SMEM_MAX = (int)sizeof(float) * (SI_W + ASK_BLK_N * 64 + ASK_TILE_M * 16);
    static_assert(SMEM_MAX <= 232448, "shared-memory plan exceeds 227 KB");
    static std::atomic<uint64_t> opted{0};
    ASK_TRY(opt_in_smem(eval_simt_kernel<ZC, DEEP>, SMEM_MAX, opted));
    // a sub-block's items over several blocks where there are few sub-blocks:
    // about eight waves of two blocks an SM
    const int64_t split = std::max<int64_t>(1, std::min<int64_t>(64, 8 * 2 * 152 / w.n_blocks));
    eval_simt_kernel<ZC, DEEP><<<dim3((unsigned)w.n_blocks, (unsigned)split), SI_THREADS, smem, s>>>(
        Xq, ldq, w.items, w.block_off, w.block_order, w.tgt, partial, t->Xt, t->Xs, t->sc_t, t->sc_s, c.Wt, c.Ws,
        t->d_pad, c.r);
    ASK_LAUNCH();
    return ASKIT_OK;
}

template <int ZC>
askit_status launch_simt(askit_tree t, const WeightCtx &c, const float *Xq, int64_t ldq, const WorkLists &w,
                         float *partial, cudaStream_t s) {
    return t->d_pad > SI_K ? launch_simt<ZC, true>(t, c, Xq, ldq, w, partial, s)
                           : launch_simt<ZC, false>(t, c, Xq, ldq, w, partial, s);
}

}  // namespace

askit_status eval_simt(askit_tree t, const WeightCtx &c, const float *Xq, int64_t ldq, const WorkLists &w,
                       float *partial, cudaStream_t s) {
    if (w.n_blocks == 0) return ASKIT_OK;
    ASK_TRY(ktimer_mark(t, s, false));
    if (c.r == 1) ASK_TRY(launch_simt<1>(t, c, Xq, ldq, w, partial, s));
    else if (c.r <= 4) ASK_TRY(launch_simt<4>(t, c, Xq, ldq, w, partial, s));
    else ASK_TRY(launch_simt<16>(t, c, Xq, ldq, w, partial, s));
    return ktimer_mark(t, s, true);
}

// ---------------------------------------------------------------------------
// Direct sum of eq. (1.1) at selected points: every source point, no
// approximation (the yardstick of ASKIT's error, Section 4).  One block per
// target; threads stride over the sources in tree order and reduce in a
// fixed order.
// ---------------------------------------------------------------------------
namespace {
constexpr int DIRECT_THREADS = 256;
template <int RMAX>
__global__ void __launch_bounds__(DIRECT_THREADS) direct_kernel(const float *__restrict__ X, int d,
                                                               const int32_t *__restrict__ tgt,
                                                               const float *__restrict__ Xt, int d_pad, int64_t N,
                                                               const float *__restrict__ sc_t,
                                                               const float *__restrict__ Wt, int r, float *U,
                                                               int64_t ldu) {
    __shared__ float xs[1024];
    __shared__ float red[DIRECT_THREADS / 32][RMAX];
    const int q = blockIdx.x;
    const int64_t i = tgt[q];
    for (int k = threadIdx.x; k < d_pad; k += blockDim.x) xs[k] = k < d ? X[i * d + k] : 0.f;
    __syncthreads();
    float acc[RMAX];
#pragma unroll
    for (int z = 0; z < RMAX; ++z) acc[z] = 0.f;
    for (int64_t j = threadIdx.x; j < N; j += blockDim.x) {
        const float *y = Xt + j * d_pad;
        float D = 0.f;
        for (int k = 0; k < d_pad; k += 4) {
            const float4 v = *reinterpret_cast<const float4 *>(y + k);
            const float a = xs[k] - v.x, b = xs[k + 1] - v.y, c = xs[k + 2] - v.z, e = xs[k + 3] - v.w;
            D = fmaf(a, a, D); D = fmaf(b, b, D); D = fmaf(c, c, D); D = fmaf(e, e, D);
        }
        const float kv = exp2f(-sc_t[j] * D);
#pragma unroll
        for (int z = 0; z < RMAX; ++z)
            if (z < r) acc[z] = fmaf(kv, Wt[j * r + z], acc[z]);
    }
#pragma unroll
    for (int z = 0; z < RMAX; ++z) {
        float v = acc[z];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5][z] = v;
    }
    __syncthreads();
    if (threadIdx.x < RMAX && threadIdx.x < r) {
        float v = 0.f;
        for (int w = 0; w < DIRECT_THREADS / 32; ++w) v += red[w][threadIdx.x];
        U[q * ldu + threadIdx.x] = v;
    }
}
}  // namespace

extern "C" askit_status askit_direct(askit_tree t, const int32_t *tgt_dev, int64_t T, float *U_dev, int64_t ldu,
                                     void *stream) {
    if (!t || !tgt_dev || !U_dev) { askit_set_error("tree, tgt_dev and U_dev must be non-NULL"); return ASKIT_ERR_INVALID_ARG; }
    if (!t->dw.ready) { askit_set_error("askit_set_weights has not been called"); return ASKIT_ERR_NOT_READY; }
    if (T < 1 || T > (1 << 30) || ldu < t->dw.r) { askit_set_error("need 1 <= T and ldu >= r"); return ASKIT_ERR_INVALID_ARG; }
    if (t->d_pad > 1024) { askit_set_error("askit_direct handles d <= 1024"); return ASKIT_ERR_UNSUPPORTED; }
    cudaStream_t s = (cudaStream_t)stream;
    const WeightCtx &c = t->dw;
    if (c.r <= 1)
        direct_kernel<1><<<(unsigned)T, DIRECT_THREADS, 0, s>>>(t->X, t->d, tgt_dev, t->Xt, t->d_pad, t->N, t->sc_t, c.Wt, c.r, U_dev, ldu);
    else if (c.r <= 16)
        direct_kernel<16><<<(unsigned)T, DIRECT_THREADS, 0, s>>>(t->X, t->d, tgt_dev, t->Xt, t->d_pad, t->N, t->sc_t, c.Wt, c.r, U_dev, ldu);
    else
        direct_kernel<64><<<(unsigned)T, DIRECT_THREADS, 0, s>>>(t->X, t->d, tgt_dev, t->Xt, t->d_pad, t->N, t->sc_t, c.Wt, c.r, U_dev, ldu);
    ASK_LAUNCH();
    return ASKIT_OK;
}
