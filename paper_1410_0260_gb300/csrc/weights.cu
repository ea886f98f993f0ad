// Weights into tree order and the upward pass of skeleton weights
// (Section 2.1 and Algorithm 3): w~_a = v(S_a) + P_a v(R), where v is w on
// the leaf's points, or the concatenated skeleton weights [w~_l; w~_r] of
// the children; S and R are the first s and the remaining columns of the
// node's pivot order.  FP32, one kernel per tree level, leaves first.
#include <algorithm>

#include "askit_impl.cuh"

namespace {

__global__ void permute_in_kernel(const float *W, int64_t ldw, int r, const int32_t *perm, int64_t N,
                                  float *Wt) {
    pdl_trigger();
    int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= N * r) return;
    int64_t q = e / r;
    int z = (int)(e % r);
    Wt[e] = W[(int64_t)perm[q] * ldw + z];
}

// The upward pass reads every node's P once (4 s (c - s) bytes: HBM-bound on the
// wide levels near the leaves) and is a chain of L launches on the narrow ones
// near the root (latency-bound).  Block (a, y) takes 8 R rows of node a's w~_a,
// a warp R of them: lane l reads P's columns 128 i + 4 l .. + 3 as one 16-byte
// load a row (R loads in flight, the next step's R issued before this step's
// products), and every load of a v(R) value from shared memory serves R rows.
// The row sums are reduced over the lanes by a transposing butterfly (R RC sums
// in about R RC shuffles).  R = 8 (r <= 4) or 4 (r > 4: R RC accumulators in
// registers) at every level: R = 2 near the root, for more blocks there, was no
// faster at 4K, 64K or 1M points and cost 1-4 us a call at 50K, r = 3, where every
// block stages its own v(R).  Levels are launched with programmatic serialization: a
// level's blocks resolve their pivots and read their first P rows while the
// level below still runs.
// Measured (a set_weights call with its permutation, GB300; before: one row a
// warp, 4-byte loads, r > 4 bound by its shared-memory loads):
//   1M x 64, s = 256, r = 1     398 -> 275 us (1.07 GB of P: 158 us at the copy rate)
//   64K x 64, s = 512, r = 16  2587 -> 107 us (147 with 4-byte loads of v)
//   50K x 64, s = 256, r = 3    163 ->  39 us
constexpr int UP_KU = 1024;      // columns of P staged at a time
constexpr int UP_WARPS = 8;

// floats between consecutive columns' v values: conflict-free 16-byte reads
template <int RC>
__host__ __device__ constexpr int up_stride() { return RC == 16 ? 20 : RC; }

template <int RC, int R>
__global__ void __launch_bounds__(32 * UP_WARPS) upward_kernel(
    int64_t a0, bool leaf_level, int r, int ku_max, const int32_t *nstart, const int32_t *s, const int32_t *ncol,
    const int64_t *pivoff, const int32_t *piv, const int64_t *p32off, const float *P32, const int64_t *spool,
    const float *Wt, float *Ws) {
    extern __shared__ float vs[];          // [ku_max][STR] values, then [ku_max] rows of v
    constexpr int STR = up_stride<RC>(), V = R * RC;
    pdl_trigger();
    int32_t *vrows = reinterpret_cast<int32_t *>(vs + (size_t)ku_max * STR);
    const int64_t a = a0 + blockIdx.x;
    const int sa = s[a], nr = ncol[a] - sa, ldp = (nr + 3) & ~3;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int q0 = (blockIdx.y * UP_WARPS + warp) * R;
    if ((int)blockIdx.y * UP_WARPS * R >= sa) {            // block-uniform
        pdl_wait();
        return;
    }
    // v of column col: row vrow(col) of `src` (weights in tree order at a leaf,
    // the children's skeleton weights above)
    const int32_t *pv = piv + pivoff[a];
    const int sl = leaf_level ? 0 : s[2 * a];
    const int64_t rl = leaf_level ? nstart[a] : spool[2 * a], rr_ = leaf_level ? 0 : spool[2 * a + 1] - sl;
    const float *src = leaf_level ? Wt : Ws;
    auto vrow = [&](int col) -> int32_t { return (int32_t)((leaf_level || col < sl ? rl : rr_) + col); };
    float *out = Ws + spool[a] * r;
    const float *Prow[R];
#pragma unroll
    for (int k = 0; k < R; ++k) Prow[k] = P32 + p32off[a] + (int64_t)min(q0 + k, sa - 1) * ldp + 4 * lane;
    // the sums this lane holds after the butterfly (value j of NV: row jb / RC,
    // vector jb % RC of the warp's R x RC)
    constexpr int NV = V > 32 ? V / 32 : 1;
    int jb = 0;
    bool writer = true;
    {
        int n = V;
#pragma unroll
        for (int m = 16; m >= 1; m >>= 1) {
            if (n > 1) {
                n >>= 1;
                jb += (lane & m) ? n : 0;
            } else {
                writer = writer && !(lane & m);
            }
        }
    }
    bool waited = false;
    for (int z0 = 0; z0 < r; z0 += RC) {
        float acc[V];
#pragma unroll
        for (int e = 0; e < V; ++e) acc[e] = 0.f;
        for (int u0 = 0; u0 < nr; u0 += UP_KU) {
            const int ku = min(nr - u0, UP_KU), ni = (ku + 127) >> 7, lim = ldp - u0 - 4 * lane;
            float4 p[R];
#pragma unroll
            for (int k = 0; k < R; ++k)
                p[k] = lim > 0 ? *reinterpret_cast<const float4 *>(Prow[k] + u0) : make_float4(0.f, 0.f, 0.f, 0.f);
            __syncthreads();                               // the last chunk's values are no longer read
            for (int e = threadIdx.x; e < 128 * ni; e += 32 * UP_WARPS) vrows[e] = e < ku ? vrow(pv[sa + u0 + e]) : -1;
            if (!waited) {
                pdl_wait();
                waited = true;
            }
            __syncthreads();
            // column 128 i + 4 l + c at slot (4 i + c) 32 + l; eight gathered loads
            // in flight a thread, 16 bytes each where the rows allow it
            auto slot_of = [](int u) { return ((u >> 7) * 4 + (u & 3)) * 32 + ((u >> 2) & 31); };
            constexpr int UB = 8;
            if (RC > 1 && (r & 3) == 0) {
                constexpr int Q = RC > 1 ? RC / 4 : 1;             // 16-byte pieces of a column
                for (int e0 = threadIdx.x; e0 < 128 * ni * Q; e0 += UB * 32 * UP_WARPS) {
                    float4 x[UB];
#pragma unroll
                    for (int b = 0; b < UB; ++b) {
                        const int e = e0 + b * 32 * UP_WARPS, z = z0 + 4 * (e % Q);
                        const int32_t row = e < 128 * ni * Q ? vrows[e / Q] : -1;
                        x[b] = (row >= 0 && z < r) ? *reinterpret_cast<const float4 *>(src + (int64_t)row * r + z)
                                                   : make_float4(0.f, 0.f, 0.f, 0.f);
                    }
#pragma unroll
                    for (int b = 0; b < UB; ++b) {
                        const int e = e0 + b * 32 * UP_WARPS;
                        if (e < 128 * ni * Q) *reinterpret_cast<float4 *>(vs + slot_of(e / Q) * STR + 4 * (e % Q)) = x[b];
                    }
                }
            } else {
                for (int e0 = threadIdx.x; e0 < 128 * ni * RC; e0 += UB * 32 * UP_WARPS) {
                    float x[UB];
#pragma unroll
                    for (int b = 0; b < UB; ++b) {
                        const int e = e0 + b * 32 * UP_WARPS, z = z0 + e % RC;
                        const int32_t row = e < 128 * ni * RC ? vrows[e / RC] : -1;
                        x[b] = (row >= 0 && z < r) ? src[(int64_t)row * r + z] : 0.f;
                    }
#pragma unroll
                    for (int b = 0; b < UB; ++b) {
                        const int e = e0 + b * 32 * UP_WARPS;
                        if (e < 128 * ni * RC) vs[slot_of(e / RC) * STR + e % RC] = x[b];
                    }
                }
            }
            __syncthreads();
#pragma unroll 1
            for (int i = 0; i < ni; ++i) {
                float4 pn[R];
                const bool more = i + 1 < ni && 128 * (i + 1) < lim;
#pragma unroll
                for (int k = 0; k < R; ++k)
                    pn[k] = more ? *reinterpret_cast<const float4 *>(Prow[k] + u0 + 128 * (i + 1))
                                 : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const float *v = vs + ((4 * i + c) * 32 + lane) * STR;
                    float pc[R];
#pragma unroll
                    for (int k = 0; k < R; ++k) pc[k] = c == 0 ? p[k].x : c == 1 ? p[k].y : c == 2 ? p[k].z : p[k].w;
                    if constexpr (RC == 1) {
                        const float x = v[0];
#pragma unroll
                        for (int k = 0; k < R; ++k) acc[k] = fmaf(pc[k], x, acc[k]);
                    } else {
#pragma unroll
                        for (int z4 = 0; z4 < RC / 4; ++z4) {
                            const float4 x = *reinterpret_cast<const float4 *>(v + 4 * z4);
#pragma unroll
                            for (int k = 0; k < R; ++k) {
                                float *ak = acc + k * RC + 4 * z4;
                                ak[0] = fmaf(pc[k], x.x, ak[0]);
                                ak[1] = fmaf(pc[k], x.y, ak[1]);
                                ak[2] = fmaf(pc[k], x.z, ak[2]);
                                ak[3] = fmaf(pc[k], x.w, ak[3]);
                            }
                        }
                    }
                }
#pragma unroll
                for (int k = 0; k < R; ++k) p[k] = pn[k];
            }
        }
        if (!waited) {
            pdl_wait();
            waited = true;
        }
        // sums over the lanes: at mask m a lane keeps the half of its values that
        // bit m of its number selects, until one is left
        int n = V;
#pragma unroll
        for (int m = 16; m >= 1; m >>= 1) {
            if (n > 1) {
                n >>= 1;
                const bool up = lane & m;
#pragma unroll
                for (int j = 0; j < V / 2; ++j)
                    if (j < n) {
                        const float send = up ? acc[j] : acc[j + n], keep = up ? acc[j + n] : acc[j];
                        acc[j] = keep + __shfl_xor_sync(0xffffffffu, send, m);
                    }
            } else {
                acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], m);
            }
        }
        if (writer) {
#pragma unroll
            for (int j = 0; j < NV; ++j) {
                const int q = q0 + (jb + j) / RC, z = z0 + (jb + j) % RC;
                if (q < sa && z < r) out[(int64_t)q * r + z] = src[(int64_t)vrow(pv[q]) * r + z] + acc[j];
            }
        }
    }
}

template <int RC>
askit_status launch_upward(askit_tree t, WeightCtx &c, int depth, int r, cudaStream_t s) {
    constexpr int STR = up_stride<RC>(), R = RC <= 4 ? 8 : 4;
    // set once per kernel instance (thread-safe static initialisation)
    static std::atomic<uint64_t> opted{0};
    ASK_TRY(opt_in_smem(upward_kernel<RC, R>, UP_KU * (STR * sizeof(float) + sizeof(int32_t)), opted));
    const int64_t a0 = (int64_t)1 << depth;
    const int ku_max = std::max(128, std::min(UP_KU, (t->lvl_nr[depth] + 127) / 128 * 128));
    const size_t smem = (size_t)ku_max * (STR * sizeof(float) + sizeof(int32_t));
    const unsigned ny = (unsigned)((std::max(1, t->prm.s_max) + UP_WARPS * R - 1) / (UP_WARPS * R));
    return launch_pdl(upward_kernel<RC, R>, dim3((unsigned)a0, ny), dim3(32 * UP_WARPS), smem, s, a0, depth == t->L, r,
                      ku_max, t->nstart, t->d_s, t->d_ncol, t->d_pivoff, t->piv, t->d_p32off, t->P32, t->d_spool, c.Wt,
                      c.Ws);
}

}  // namespace

// Buffers of a weight context for r vectors (grow-only in r and in the work
// lists' entries; the padding rows of Wt and Ws stay zero).
askit_status weights_reserve(askit_tree t, WeightCtx &c, int r, cudaStream_t s) {
    if (r <= c.r_cap && t->wl_entries_max <= c.ent_cap) {
        c.r = r;
        return ASKIT_OK;
    }
    const int r_req = r;
    r = std::max(r, c.r_cap);      // the capacity never shrinks
    c.arena.free_all();
    c.Wt = c.Ws = c.partial = nullptr;
    c.colv = nullptr;
    c.colw = nullptr;
    const int64_t srows = std::max<int64_t>(t->spool_rows, 1) + 256;
    ASK_TRY(c.arena.alloc(&c.Wt, (size_t)t->N_pad * r));
    ASK_TRY(c.arena.alloc(&c.Ws, (size_t)srows * r));
    ASK_TRY(c.arena.alloc(&c.partial, (size_t)std::max<int64_t>(1, t->wl_entries_max) * r));
    c.ent_cap = t->wl_entries_max;
    // per-sub-block column data of the 16-bit tensor-core kernel
    if (t->n_sub > 0 && t->d <= TC_K) {
        ASK_TRY(c.arena.alloc(&c.colv, (size_t)t->n_sub * 128));
        // [n_sub, 128, 16] floats, or (r > 4, the global-centered kernel's
        // weight MMA) split FP16 weights and 16 factors per sub-block
        if (r > 1) ASK_TRY(c.arena.alloc(&c.colw, (size_t)t->n_sub * (128 * 16 + 16)));
    }
    ASK_CUDA(cudaMemsetAsync(c.Wt, 0, sizeof(float) * t->N_pad * r, s));
    ASK_CUDA(cudaMemsetAsync(c.Ws, 0, sizeof(float) * srows * r, s));
    c.r_cap = r;
    c.r = r_req;
    c.ready = true;
    return ASKIT_OK;
}

askit_status upward_weights(askit_tree t, WeightCtx &c, const float *W, int r, int64_t ldw, cudaStream_t s) {
    ASK_TRY(weights_reserve(t, c, r, s));
    int64_t N = t->N;
    // rows of Wt/Ws are r apart: with a smaller r than the capacity, rows past
    // the first r columns are not used, so a fresh layout per call is fine
    permute_in_kernel<<<(unsigned)((N * r + 255) / 256), 256, 0, s>>>(W, ldw, r, t->perm, N, c.Wt);
    ASK_LAUNCH();
    for (int depth = t->L; depth >= 1; --depth) {
        if (r == 1)
            ASK_TRY(launch_upward<1>(t, c, depth, r, s));
        else if (r <= 4)
            ASK_TRY(launch_upward<4>(t, c, depth, r, s));
        else
            ASK_TRY(launch_upward<16>(t, c, depth, r, s));
    }
    c.ready = true;
    return ASKIT_OK;
}
