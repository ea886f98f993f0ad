// Evaluate (Algorithm 4) on the tcgen05 tensor cores in 3xTF32, d <= 64.
//
// Work item = one source sub-block (<= 128 rows of a leaf or a skeleton) against up
// to 128 targets that need it.  Both sides are centered on the sub-block's mean c_B
// (sources pre-split in HBM), as in the FP16x3 kernel of eval_tc16.cu:
//     a = x - c_B,  b = y - c_B,  r^2 = |a|^2 + |b|^2 - 2 a.b
//     partial_t = sum_j exp2(-c log2(e) r^2 / h_j^2) w_j
// with a.b from three TF32 split products, the small cross terms first, FP32
// accumulation.
//
// A sub-block whose rows reach far from c_B (EvalItem::wide) centers each target row on
// the nearest of four of the item's targets instead (the first, the last and two
// between), with the exact rewriting
//     a = x - c,  r^2 = |a|^2 + 2 a.(c - c_B) + |y - c|^2 - 2 a.b
// Around c_B the norms of near points in a far cluster cancel; these terms stay at the
// scale of |a|, which is small also where an item's targets (in tree order) lie in
// several clusters.  Three clusters in 4 dimensions, centers in a box of 100 h,
// relative error: 1.6e-4 on c_B, 8.9e-5 on the first target alone, 2.0e-6 on the nearest
// of four.  The column terms -sc |y - c|^2 belong to the item then: the loader thread of
// target row t forms those of source row t, one a center, from the FP32 rows.
//
// The targets' split rows are the MMA's A operand in TMEM: a loader thread owns a
// row, so it centers, splits and stores it (tcgen05.st) without a layout in shared
// memory, and the tensor core reads only B there (an item's 24 MMAs of 128 x 128 x 8
// take 64 cycles each and would read 128 bytes a cycle with A in shared memory as
// well).  Rows arrive by cp.async, a row's 16-byte pieces coalesced, into rows of
// 16 spare bytes, which a warp reads a row a lane without bank conflicts; a column's
// data (bandwidth, |b|^2, weights) is built once per Evaluate.  The kernel this
// replaces centered every item on its first target, with target and source rows
// read again from global memory by every thread: 10,400 cycles an item (64K x 64,
// r = 1: 960 us; now 374, shared-memory wavefronts 46 %, tensor pipe 40 % busy).
//
// One CTA per SM, 640 threads; item li of the CTA's order belongs to side li & 1:
//   warps 0-7    two loader groups (a side each);
//   warps 8-15   two epilogue groups (a side each);
//   warps 16,17  lane 0: the MMAs of a side (an MMA costs its issuing thread about a
//                hundred cycles); warp 16 also loads the sub-blocks and owns TMEM;
//   warps 18,19  copy target rows, three stages.
// TMEM: two 128-column accumulators, two A operands of 64 + 64 columns.  Every wait
// is bounded (ASK_DEV_TIMEOUT on expiry, all roles leave, copies and MMAs in flight
// are waited for, TMEM is freed).
#include <cuda.h>

#include <mutex>
#include <type_traits>

#include "askit_impl.cuh"
#include "tc_ptx.cuh"

namespace {

using namespace tcx;

constexpr int F_REGION = 128 * 128;            // 128 rows x 32 TF32, 128-byte swizzle
constexpr int F_NRAW = 3;
constexpr int F_THREADS = 640;
constexpr int F_NCEN = 4;                      // centers of a wide item's targets

template <int RC>
struct SF {
    static constexpr int B_HI = 0, B_LO = 2 * F_REGION;
    static constexpr int RAW = 4 * F_REGION;
    static constexpr int RAWSTAGE = 128 * (TC_K * 4 + 16);
    static constexpr int BLK = RAW + F_NRAW * RAWSTAGE;        // [2]: c_B, column data, weights
    static constexpr int BLK_COLV = 256, BLK_COLW = BLK_COLV + 128 * 16;
    static constexpr int BLKSLOT = BLK_COLW + (RC > 1 ? 128 * RC * 4 : 0);
    static constexpr int ANORM = BLK + 2 * BLKSLOT;            // float [2][128]
    static constexpr int BITEM = ANORM + 2 * 128 * 4;          // float [2][F_NCEN][128]: B of a wide item's columns by center
    static constexpr int PICK = BITEM + 2 * F_NCEN * 128 * 4;  // int [2][128]: center of a wide item's row
    static constexpr int BAR = PICK + 2 * 128 * 4;             // 24 mbarriers
    static constexpr int MISC = BAR + 24 * 8;
    static constexpr int BYTES = MISC + 16;
};

struct FArgs {
    const EvalItem *items;
    const int32_t *block_off, *cta_off, *cta_blocks;
    const int32_t *tgt;
    const float *q;                // target rows [*, d_pad]
    const float *Xt, *Xs;          // source rows [*, d_pad] and their c log2(e) / h^2 (wide items)
    const float *sc_t, *sc_s;
    int d_pad;
    const float *cent;             // [n_sub, TC_K]
    const float4 *colv;            // [n_sub, 128] {A_j, A_j+1, B_j, B_j+1}, {C_j, C_j+1, w_j, w_j+1}
    const float *colw;             // [n_sub, 128, RC]
    int r;
    float uni_a, uni_c;            // UNI: A = 2 sc and C = -sc
    float *partial;
    int *status;
    int spin;
};

// D += A B with A in TMEM, one TF32 element a 32-bit column.
__device__ __forceinline__ void mma_tf32_ts(uint32_t d, uint32_t a, uint64_t b, uint32_t idesc, uint32_t accum) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::tf32 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d), "r"(a), "l"(b), "r"(idesc), "r"(accum)
        : "memory");
}

// UNI (r = 1): one bandwidth for all sources; the column data is {B_j, B_j+1, w_j,
// w_j+1} a pair, and A and C are scalars, which halves the epilogue's shared-memory
// reads (two reads a pair: 484 us at 64K x 64).  WIDE: the tree has wide sub-blocks
// (64K x 64 without any: 429 us, 444 with the test in every item).
template <int RC, bool UNI, bool WIDE>
__global__ void __launch_bounds__(F_THREADS, 1)
eval_tf32_kernel(const __grid_constant__ CUtensorMap map_t_hi, const __grid_constant__ CUtensorMap map_t_lo,
                 const __grid_constant__ CUtensorMap map_s_hi, const __grid_constant__ CUtensorMap map_s_lo,
                 const FArgs args) {
    using S = SF<RC>;
    static_assert(!UNI || RC == 1, "the uniform-bandwidth layout serves r = 1");
    constexpr int CV = UNI ? 64 : 128;         // float4 of column data per sub-block
    extern __shared__ uint8_t smem_raw[];
    uint8_t *sm = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const uint32_t sbase = smem_u32(sm), bar0 = sbase + S::BAR;
    float *a_norm = reinterpret_cast<float *>(sm + S::ANORM), *b_item = reinterpret_cast<float *>(sm + S::BITEM);
    int *pick = reinterpret_cast<int *>(sm + S::PICK);
    auto BAR_R_FULL = [&](int s) { return bar0 + 8 * s; };            // raw rows of stage s landed (64)
    auto BAR_R_EMPTY = [&](int s) { return bar0 + 8 * (3 + s); };     // loaders done with stage s (128)
    auto BAR_A_FULL = [&](int g) { return bar0 + 8 * (6 + g); };      // split rows of side g in TMEM (128)
    auto BAR_A_EMPTY = [&](int g) { return bar0 + 8 * (8 + g); };     // MMAs read them (commit)
    auto BAR_T_FULL = [&](int g) { return bar0 + 8 * (10 + g); };     // accumulator g complete (commit)
    auto BAR_T_EMPTY = [&](int g) { return bar0 + 8 * (12 + g); };    // drained (128)
    auto BAR_N_EMPTY = [&](int g) { return bar0 + 8 * (14 + g); };    // row terms of side g, a wide item's B, read (128)
    auto BAR_BLK_FULL = [&](int s) { return bar0 + 8 * (16 + s); };   // c_B, column data of slot s landed
    auto BAR_BLK_EMPTY = [&](int s) { return bar0 + 8 * (18 + s); };  // epilogue done with slot s (256)
    const uint32_t BAR_B_FULL = bar0 + 8 * 20, BAR_B_EMPTY = bar0 + 8 * 21;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(sm + S::MISC);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(sm + S::MISC + 4);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        for (int s = 0; s < F_NRAW; ++s) {
            mbar_init(BAR_R_FULL(s), 64);
            mbar_init(BAR_R_EMPTY(s), 128);
        }
        for (int g = 0; g < 2; ++g) {
            mbar_init(BAR_A_FULL(g), 128);
            mbar_init(BAR_A_EMPTY(g), 1);
            mbar_init(BAR_T_FULL(g), 1);
            mbar_init(BAR_T_EMPTY(g), 128);
            mbar_init(BAR_N_EMPTY(g), 128);
            mbar_init(BAR_BLK_FULL(g), 1);
            mbar_init(BAR_BLK_EMPTY(g), 256);
        }
        mbar_init(BAR_B_FULL, 1);
        mbar_init(BAR_B_EMPTY, 2);             // one commit per issuer and block
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 16) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(tmem_slot)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    pdl_wait();          // the set-up above overlaps the kernels before; everything below reads their results
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    const int c_begin = args.cta_off[blockIdx.x], c_end = args.cta_off[blockIdx.x + 1];
    const int rst = args.d_pad * 4 + 16;       // bytes of a raw row
    auto A_TMEM = [&](int g) { return tmem + 256u + 128u * (uint32_t)g; };   // 64 columns hi, 64 lo

    if (warp < 8) {
        // ------------------------------------------------------------ loaders
        const int g = warp >> 2, row = (warp & 3) * 32 + lane;
        const uint32_t ta = A_TMEM(g) + ((uint32_t)((warp & 3) * 32) << 16);
        int li = 0, lb = 0;
        for (int ci = c_begin; ci < c_end && !*abort_flag; ++ci, ++lb) {
            const int b = args.cta_blocks[ci];
            const int i0 = args.block_off[b], i1 = args.block_off[b + 1];
            bool need_blk = true;
            for (int it = i0; it < i1; ++it, ++li) {
                if ((li & 1) != g) continue;
                const EvalItem item = args.items[it];
                const int cnt = item.cnt;
                const int sr = li % F_NRAW, par = ((li >> 1) & 1) ^ 1;
                if (need_blk) {
                    if (!mbar_wait(BAR_BLK_FULL(lb & 1), (lb >> 1) & 1, abort_flag, args.status, args.spin)) goto loader_done;
                    need_blk = false;
                }
                if (!mbar_wait(BAR_R_FULL(sr), (li / F_NRAW) & 1, abort_flag, args.status, args.spin)) goto loader_done;
                if (!mbar_wait(BAR_A_EMPTY(g), par, abort_flag, args.status, args.spin)) goto loader_done;
                if (!mbar_wait(BAR_N_EMPTY(g), par, abort_flag, args.status, args.spin)) goto loader_done;
                tc_fence_after();
                const uint8_t *x = sm + S::RAW + sr * S::RAWSTAGE + row * rst;
                const float4 *cb = reinterpret_cast<const float4 *>(sm + S::BLK + (lb & 1) * S::BLKSLOT);
                const bool mine = row < cnt, wide = WIDE && item.wide != 0;   // (wide: warp-uniform)
                float2 nn = make_float2(0.f, 0.f);
                const float2 m1 = make_float2(-1.f, -1.f);
                const float4 *ctr = cb;
                if (wide) {
                    const float4 *ct[F_NCEN];
#pragma unroll
                    for (int k = 0; k < F_NCEN; ++k)
                        ct[k] = reinterpret_cast<const float4 *>(sm + S::RAW + sr * S::RAWSTAGE +
                                                                 k * (cnt - 1) / (F_NCEN - 1) * rst);
                    const bool far = item.nrows < 0;
                    const bool src = row < (item.nrows & 0x7fffffff);
                    const int64_t srow = (int64_t)item.row0 + (src ? row : 0);
                    const float4 *yr = reinterpret_cast<const float4 *>((far ? args.Xs : args.Xt) + srow * args.d_pad);
                    const float msc = -(far ? args.sc_s : args.sc_t)[srow];
                    float2 dx[F_NCEN], dy[F_NCEN];
#pragma unroll
                    for (int k = 0; k < F_NCEN; ++k) dx[k] = dy[k] = make_float2(0.f, 0.f);
                    for (int j = 0; j < args.d_pad / 4; ++j) {
                        const float4 xv = *reinterpret_cast<const float4 *>(x + 16 * j), yv = yr[j];
#pragma unroll
                        for (int k = 0; k < F_NCEN; ++k) {
                            const float4 tv = ct[k][j];
                            const float2 t0 = make_float2(tv.x, tv.y), t1 = make_float2(tv.z, tv.w);
                            float2 u = __ffma2_rn(t0, m1, make_float2(xv.x, xv.y));
                            dx[k] = __ffma2_rn(u, u, dx[k]);
                            u = __ffma2_rn(t1, m1, make_float2(xv.z, xv.w));
                            dx[k] = __ffma2_rn(u, u, dx[k]);
                            u = __ffma2_rn(t0, m1, make_float2(yv.x, yv.y));
                            dy[k] = __ffma2_rn(u, u, dy[k]);
                            u = __ffma2_rn(t1, m1, make_float2(yv.z, yv.w));
                            dy[k] = __ffma2_rn(u, u, dy[k]);
                        }
                    }
                    int pk = 0;
                    float near = dx[0].x + dx[0].y;
                    ctr = ct[0];
#pragma unroll
                    for (int k = 0; k < F_NCEN; ++k) {
                        const float dk = dx[k].x + dx[k].y;
                        if (dk < near) {
                            near = dk;
                            pk = k;
                            ctr = ct[k];
                        }
                        b_item[(F_NCEN * g + k) * 128 + row] = src ? msc * (dy[k].x + dy[k].y) : UNI ? -INFINITY : 0.f;
                    }
                    pick[g * 128 + row] = pk;
                }
                for (int c = 0; c < args.d_pad / 16; ++c) {        // 16 columns at a time
                    uint32_t hi[16], lo[16];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float4 xv = *reinterpret_cast<const float4 *>(x + 64 * c + 16 * j);
                        const float4 mv = ctr[4 * c + j];
                        float2 a[2] = {__ffma2_rn(make_float2(mv.x, mv.y), m1, make_float2(xv.x, xv.y)),
                                       __ffma2_rn(make_float2(mv.z, mv.w), m1, make_float2(xv.z, xv.w))};
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            if (!mine) a[e] = make_float2(0.f, 0.f);
                            nn = __ffma2_rn(a[e], a[e], nn);
                            const float h0 = __uint_as_float(__float_as_uint(a[e].x) & 0xffffe000u);
                            const float h1 = __uint_as_float(__float_as_uint(a[e].y) & 0xffffe000u);
                            hi[4 * j + 2 * e] = __float_as_uint(h0);
                            hi[4 * j + 2 * e + 1] = __float_as_uint(h1);
                            lo[4 * j + 2 * e] = __float_as_uint(a[e].x - h0);
                            lo[4 * j + 2 * e + 1] = __float_as_uint(a[e].y - h1);
                        }
                    }
                    tmem_st16(ta + 16 * c, hi);
                    tmem_st16(ta + 64 + 16 * c, lo);
                }
                float rowterm = nn.x + nn.y;
                if (wide) {
                    float2 dd = make_float2(0.f, 0.f);             // a.(c - c_B)
                    for (int j = 0; j < args.d_pad / 4; ++j) {
                        const float4 xv = *reinterpret_cast<const float4 *>(x + 16 * j), tv = ctr[j], bv = cb[j];
                        const float2 t0 = make_float2(tv.x, tv.y), t1 = make_float2(tv.z, tv.w);
                        dd = __ffma2_rn(__ffma2_rn(t0, m1, make_float2(xv.x, xv.y)),
                                        __ffma2_rn(make_float2(bv.x, bv.y), m1, t0), dd);
                        dd = __ffma2_rn(__ffma2_rn(t1, m1, make_float2(xv.z, xv.w)),
                                        __ffma2_rn(make_float2(bv.z, bv.w), m1, t1), dd);
                    }
                    rowterm = mine ? fmaf(2.f, dd.x + dd.y, rowterm) : 0.f;
                }
                a_norm[g * 128 + row] = rowterm;
                mbar_arrive(BAR_R_EMPTY(sr));
                tmem_st_wait();
                tc_fence_before();
                mbar_arrive(BAR_A_FULL(g));
            }
        }
    loader_done:;
    } else if (warp < 16) {
        // ----------------------------------------------------------- epilogue
        const int g = (warp - 8) >> 2, q = warp & 3, row = q * 32 + lane;
        const uint32_t tbase = tmem + ((uint32_t)(q * 32) << 16) + 128u * (uint32_t)g;
        int li = 0, lb = 0;
        for (int ci = c_begin; ci < c_end && !*abort_flag; ++ci, ++lb) {
            const int b = args.cta_blocks[ci], bs = lb & 1;
            if (!mbar_wait(BAR_BLK_FULL(bs), (lb >> 1) & 1, abort_flag, args.status, args.spin)) goto epi_done;
            const float4 *cv4 = reinterpret_cast<const float4 *>(sm + S::BLK + bs * S::BLKSLOT + S::BLK_COLV);
            const float *cwp = reinterpret_cast<const float *>(sm + S::BLK + bs * S::BLKSLOT + S::BLK_COLW);
            const int i0 = args.block_off[b], i1 = args.block_off[b + 1];
            for (int it = i0; it < i1; ++it, ++li) {
                if ((li & 1) != g) continue;
                const EvalItem item = args.items[it];
                const int nch = ((item.nrows & 0x7fffffff) + 31) >> 5;
                if (!mbar_wait(BAR_T_FULL(g), (li >> 1) & 1, abort_flag, args.status, args.spin)) goto epi_done;
                tc_fence_after();
                const float pt = a_norm[g * 128 + row];
                const bool wide = WIDE && item.wide != 0;
                const float2 *bi = reinterpret_cast<const float2 *>(b_item + (F_NCEN * g + (wide ? pick[g * 128 + row] : 0)) * 128);
                if (!wide) mbar_arrive(BAR_N_EMPTY(g));
                float acc[RC];
#pragma unroll
                for (int z = 0; z < RC; ++z) acc[z] = 0.f;
                float2 acc2[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
                float2 accw[RC > 1 ? RC / 2 : 1];
#pragma unroll
                for (int z = 0; z < (RC > 1 ? RC / 2 : 1); ++z) accw[z] = make_float2(0.f, 0.f);
                if (q * 32 < item.cnt) {                           // warp-uniform
                    const float2 pt2 = make_float2(pt, pt);
                    // arg = g A + (C p + B) = -sc (p + q - 2 g); columns past the rows
                    // carry A = B = C = w = 0
                    auto cols = [&](int c, const uint32_t (&gr)[32], auto is_wide) {
#pragma unroll
                        for (int jj = 0; jj < 32; jj += 2) {
                            if constexpr (UNI) {
                                float4 bw = cv4[(c * 32 + jj) >> 1];
                                if constexpr (decltype(is_wide)::value) {
                                    const float2 b2 = bi[(c * 32 + jj) >> 1];
                                    bw.x = b2.x;
                                    bw.y = b2.y;
                                }
                                const float2 in = __ffma2_rn(make_float2(args.uni_c, args.uni_c), pt2, make_float2(bw.x, bw.y));
                                const float2 ag = __ffma2_rn(make_float2(__uint_as_float(gr[jj]), __uint_as_float(gr[jj + 1])),
                                                             make_float2(args.uni_a, args.uni_a), in);
                                const float2 kk = make_float2(ex2_approx(ag.x), ex2_approx(ag.y));
                                acc2[(jj >> 1) & 1] = __ffma2_rn(kk, make_float2(bw.z, bw.w), acc2[(jj >> 1) & 1]);
                                continue;
                            }
                            float4 ab = cv4[c * 32 + jj];
                            const float4 cw = cv4[c * 32 + jj + 1];
                            if constexpr (decltype(is_wide)::value) {
                                const float2 b2 = bi[(c * 32 + jj) >> 1];
                                ab.z = b2.x;
                                ab.w = b2.y;
                            }
                            const float2 inner = __ffma2_rn(make_float2(cw.x, cw.y), pt2, make_float2(ab.z, ab.w));
                            const float2 arg = __ffma2_rn(make_float2(__uint_as_float(gr[jj]), __uint_as_float(gr[jj + 1])),
                                                          make_float2(ab.x, ab.y), inner);
                            const float2 k = make_float2(ex2_approx(arg.x), ex2_approx(arg.y));
                            if constexpr (RC == 1) {
                                acc2[(jj >> 1) & 1] = __ffma2_rn(k, make_float2(cw.z, cw.w), acc2[(jj >> 1) & 1]);
                            } else {
                                const float2 ka = make_float2(k.x, k.x), kb = make_float2(k.y, k.y);
                                const float4 *wa = reinterpret_cast<const float4 *>(cwp + (c * 32 + jj) * RC);
                                const float4 *wb = wa + RC / 4;
#pragma unroll
                                for (int z = 0; z < RC / 4; ++z) {
                                    const float4 va = wa[z], vb = wb[z];
                                    accw[2 * z] = __ffma2_rn(ka, make_float2(va.x, va.y), accw[2 * z]);
                                    accw[2 * z + 1] = __ffma2_rn(ka, make_float2(va.z, va.w), accw[2 * z + 1]);
                                    accw[2 * z] = __ffma2_rn(kb, make_float2(vb.x, vb.y), accw[2 * z]);
                                    accw[2 * z + 1] = __ffma2_rn(kb, make_float2(vb.z, vb.w), accw[2 * z + 1]);
                                }
                            }
                        }
                    };
                    // the other group's warp on the sub-partition covers a load
#pragma unroll 1
                    for (int c = 0; c < nch; ++c) {
                        uint32_t ga[32];
                        tmem_ld32_async(tbase + (uint32_t)(c * 32), ga);
                        tmem_wait_pin(ga);
                        if constexpr (WIDE) {
                            if (wide) {
                                cols(c, ga, std::true_type());
                                continue;
                            }
                        }
                        cols(c, ga, std::false_type());
                    }
                    if constexpr (RC == 1) {
                        acc[0] = (acc2[0].x + acc2[0].y) + (acc2[1].x + acc2[1].y);
                    } else {
#pragma unroll
                        for (int z = 0; z < RC / 2; ++z) {
                            acc[2 * z] = accw[z].x;
                            acc[2 * z + 1] = accw[z].y;
                        }
                    }
                }
                tc_fence_before();
                if (wide) mbar_arrive(BAR_N_EMPTY(g));
                mbar_arrive(BAR_T_EMPTY(g));
                if (row < item.cnt) {
                    float *p = args.partial + (int64_t)(item.e0 + row) * args.r;
#pragma unroll
                    for (int z = 0; z < RC; ++z)
                        if (z < args.r) p[z] = acc[z];
                }
            }
            mbar_arrive(BAR_BLK_EMPTY(bs));
        }
    epi_done:;
    } else if (warp < 18) {
        // --------------------------- MMA issuers; warp 16 also loads the sub-blocks
        if (lane == 0) {
            const int g = warp - 16;
            const int ks = args.d_pad / 8;                         // K = 8 an MMA
            int li = 0, lb = 0, li_done = -1, b_issued = 0;
            for (int ci = c_begin; ci < c_end && !*abort_flag; ++ci, ++lb) {
                const int b = args.cta_blocks[ci], bs = lb & 1;
                const int i0 = args.block_off[b], i1 = args.block_off[b + 1];
                const EvalItem first = args.items[i0];
                if (g == 0) {
                    const bool far = first.nrows < 0;
                    if (!mbar_wait(BAR_B_EMPTY, (lb & 1) ^ 1, abort_flag, args.status, args.spin)) goto mma_done;
                    if (!mbar_wait(BAR_BLK_EMPTY(bs), ((lb >> 1) & 1) ^ 1, abort_flag, args.status, args.spin)) goto mma_done;
                    b_issued = lb + 1;
                    mbar_expect_tx(BAR_B_FULL, 4 * F_REGION);
                    for (int h = 0; h < 2; ++h) {
                        tma_load_2d(sbase + S::B_HI + h * F_REGION, far ? &map_s_hi : &map_t_hi, 32 * h, first.row0, BAR_B_FULL);
                        tma_load_2d(sbase + S::B_LO + h * F_REGION, far ? &map_s_lo : &map_t_lo, 32 * h, first.row0, BAR_B_FULL);
                    }
                    const uint32_t slot = sbase + S::BLK + bs * S::BLKSLOT;
                    const uint32_t wbytes = RC > 1 ? 128 * RC * 4 : 0;
                    mbar_expect_tx(BAR_BLK_FULL(bs), 256 + CV * 16 + wbytes);
                    bulk_copy(slot, args.cent + (int64_t)first.cidx * TC_K, 256, BAR_BLK_FULL(bs));
                    bulk_copy(slot + S::BLK_COLV, args.colv + (int64_t)first.cidx * CV, CV * 16, BAR_BLK_FULL(bs));
                    if constexpr (RC > 1)
                        bulk_copy(slot + S::BLK_COLW, args.colw + (int64_t)first.cidx * 128 * RC, wbytes, BAR_BLK_FULL(bs));
                }
                // every block's tiles are waited for, items of this side or not: a
                // parity wait may fall at most one phase behind the loads
                if (!mbar_wait(BAR_B_FULL, lb & 1, abort_flag, args.status, args.spin)) goto mma_done;
                // N covers every 32-column chunk the epilogue reads
                const uint32_t idesc = make_idesc(2u, 128, ((first.nrows & 0x7fffffff) + 31) & ~31);
                for (int it = i0; it < i1; ++it, ++li) {
                    if ((li & 1) != g) continue;
                    if (!mbar_wait(BAR_A_FULL(g), (li >> 1) & 1, abort_flag, args.status, args.spin)) goto mma_done;
                    if (!mbar_wait(BAR_T_EMPTY(g), ((li >> 1) & 1) ^ 1, abort_flag, args.status, args.spin)) goto mma_done;
                    tc_fence_after();
                    const uint32_t dt = tmem + 128u * (uint32_t)g, ah = A_TMEM(g), al = ah + 64;
                    for (int k = 0; k < ks; ++k) {                 // the small cross terms first
                        const uint32_t off = (uint32_t)((k >> 2) * F_REGION + (k & 3) * 32);
                        mma_tf32_ts(dt, ah + 8 * k, sw128_desc(sbase + S::B_LO + off), idesc, k > 0);
                        mma_tf32_ts(dt, al + 8 * k, sw128_desc(sbase + S::B_HI + off), idesc, 1);
                    }
                    for (int k = 0; k < ks; ++k) {
                        const uint32_t off = (uint32_t)((k >> 2) * F_REGION + (k & 3) * 32);
                        mma_tf32_ts(dt, ah + 8 * k, sw128_desc(sbase + S::B_HI + off), idesc, 1);
                    }
                    tc_commit(BAR_A_EMPTY(g));
                    tc_commit(BAR_T_FULL(g));
                    li_done = li;
                }
                tc_commit(BAR_B_EMPTY);        // this thread's MMAs of the block have read the tiles
            }
        mma_done:
            // after an abort: tiles and column data may still be landing, MMAs still
            // be writing TMEM (no-ops on the normal path)
            if (b_issued > 0) {
                mbar_drain(BAR_B_FULL, (b_issued - 1) & 1);
                for (int k = b_issued > 1 ? b_issued - 2 : 0; k < b_issued; ++k) mbar_drain(BAR_BLK_FULL(k & 1), (k >> 1) & 1);
            }
            if (li_done >= 0) mbar_drain(BAR_T_FULL(g), (li_done >> 1) & 1);
        }
    } else {
        // ----------------------------------------------------- target-row copiers
        // Copier warp w takes rows 64 w .. + 63 of every item; lane l holds the
        // target slots of rows 64 w + 2 l and + 1; nch lanes along a row.  An item's
        // copies form one commit group, reported full one item later.
        const int cw = warp - 18;
        const int nch = args.d_pad / 4, rp = 32 / nch;             // lanes a row, rows an instruction
        const int u = lane / nch, j = lane % nch;
        const char *qx = reinterpret_cast<const char *>(args.q);
        const int64_t qrow = (int64_t)args.d_pad * 4;
        int cc = c_begin, cit = 0, cend = 0;
        if (cc < c_end) {
            const int b = args.cta_blocks[cc];
            cit = args.block_off[b];
            cend = args.block_off[b + 1];
        }
        struct Desc { int e0, cnt; bool ok; };
        auto load_desc = [&]() -> Desc {
            Desc dd = {0, 0, cc < c_end};
            if (!dd.ok) return dd;
            const EvalItem item = args.items[cit];
            dd.e0 = item.e0;
            dd.cnt = item.cnt;
            if (++cit == cend && ++cc < c_end) {                   // every run has an item
                const int b = args.cta_blocks[cc];
                cit = args.block_off[b];
                cend = args.block_off[b + 1];
            }
            return dd;
        };
        auto load_rows = [&](const Desc &dd, int (&r)[2]) {
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const int rw = 64 * cw + 2 * lane + k;
                r[k] = dd.ok ? args.tgt[dd.e0 + (rw < dd.cnt ? rw : 0)] : 0;
            }
        };
        Desc d0 = load_desc(), d1 = load_desc();
        int r0[2], r1[2];
        load_rows(d0, r0);
        int li = 0;
        for (; d0.ok && !*abort_flag; ++li) {
            const Desc d2 = load_desc();
            load_rows(d1, r1);
            const int sr = li % F_NRAW;
            if (!mbar_wait(BAR_R_EMPTY(sr), ((li / F_NRAW) & 1) ^ 1, abort_flag, args.status, args.spin)) goto copy_done;
            __syncwarp();
            const uint32_t dst = sbase + S::RAW + sr * S::RAWSTAGE;
            for (int m = 0; m < 64; m += rp) {
                const int rl = m + u;                              // row of this warp's 64
                const int s0 = __shfl_sync(0xffffffffu, r0[0], rl >> 1);
                const int s1 = __shfl_sync(0xffffffffu, r0[1], rl >> 1);
                const int slot = (rl & 1) ? s1 : s0;
                cp_async16(dst + (uint32_t)((64 * cw + rl) * rst + 16 * j), qx + slot * qrow + 16 * j);
            }
            cp_async_commit();
            if (li >= 1) {
                cp_async_wait<1>();                                // item li - 1 has landed
                mbar_arrive(BAR_R_FULL((li - 1) % F_NRAW));
            }
            d0 = d1;
            d1 = d2;
            r0[0] = r1[0];
            r0[1] = r1[1];
        }
        cp_async_wait<0>();
        if (!*abort_flag && li > 0) mbar_arrive(BAR_R_FULL((li - 1) % F_NRAW));
    copy_done:
        cp_async_wait<0>();                                        // nothing lands after the CTA has left
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 16) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
    }
}

// Tensor maps over the tree's TF32 split source rows (boxes of 32 x 128, 128-byte
// swizzle): [leaf rows hi, lo, skeleton rows hi, lo].
struct FState {
    CUtensorMap map[4];
};

std::mutex g_f_mu;

askit_status f_state(askit_tree t, FState **out) {
    std::lock_guard<std::mutex> lock(g_f_mu);
    if (!t->tf32) {
        EncodeTiledFn fn = nullptr;
        ASK_TRY(encode_fn(&fn));
        FState st;
        const void *arr[4] = {t->Xt_hi, t->Xt_lo, t->Xs_hi, t->Xs_lo};
        for (int i = 0; i < 4; ++i)
            ASK_TRY(encode_2d(fn, &st.map[i], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, arr[i], i < 2 ? t->N_pad : t->srows,
                              TC_K, 32, 128, CU_TENSOR_MAP_SWIZZLE_128B));
        t->tf32 = new FState(st);
    }
    *out = (FState *)t->tf32;
    return ASKIT_OK;
}

template <int RC, bool UNI, bool WIDE>
askit_status run_tf32(askit_tree t, const WeightCtx &c, FState *st, FArgs a, int grid, cudaStream_t s) {
    using S = SF<RC>;
    constexpr size_t smem = S::BYTES + 1024;
    static_assert(smem <= 232448, "shared-memory plan exceeds 227 KB");
    static std::atomic<uint64_t> opted{0};
    ASK_TRY(opt_in_smem(eval_tf32_kernel<RC, UNI, WIDE>, smem, opted));
    ASK_TRY(block_columns(t, c, RC, UNI, 1.f, s));
    a.colv = c.colv;
    a.colw = c.colw;
    ASK_TRY(ktimer_mark(t, s, false));
    ASK_TRY(launch_pdl(eval_tf32_kernel<RC, UNI, WIDE>, dim3((unsigned)grid), dim3(F_THREADS), smem, s, st->map[0], st->map[1],
                       st->map[2], st->map[3], a));
    return ktimer_mark(t, s, true);
}

template <int RC, bool UNI>
askit_status run_tf32(askit_tree t, const WeightCtx &c, FState *st, const FArgs &a, int grid, cudaStream_t s) {
    return t->any_wide ? run_tf32<RC, UNI, true>(t, c, st, a, grid, s) : run_tf32<RC, UNI, false>(t, c, st, a, grid, s);
}

}  // namespace

askit_status eval_tf32(askit_tree t, const WeightCtx &c, const float *Xq, int64_t ldq, const WorkLists &w,
                       float *partial, cudaStream_t s) {
    if (w.n_blocks == 0) return ASKIT_OK;
    if (ldq != t->d_pad || (reinterpret_cast<uintptr_t>(Xq) & 15) || !t->Xt_hi || !c.colv || (c.r > 1 && !c.colw)) {
        askit_set_error("target rows must be 16-byte aligned with d_pad columns and the TF32 operands must exist");
        return ASKIT_ERR_INVALID_ARG;
    }
    FState *st = nullptr;
    ASK_TRY(f_state(t, &st));
    const WorkLists::Sched &sc = w.sched[w.use];
    FArgs a;
    a.items = w.items;
    a.block_off = sc.run_off;
    a.cta_off = sc.cta_off;
    a.cta_blocks = sc.cta_runs;
    a.tgt = w.tgt;
    a.q = Xq;
    a.d_pad = t->d_pad;
    a.Xt = t->Xt;
    a.Xs = t->Xs;
    a.sc_t = t->sc_t;
    a.sc_s = t->sc_s;
    a.cent = t->cent;
    a.colv = nullptr;
    a.colw = nullptr;
    a.r = c.r;
    a.partial = partial;
    a.status = t->d_status;
    a.spin = t->spin_limit > 0 ? t->spin_limit : SPIN_LIMIT;
    a.uni_a = a.uni_c = 0.f;
    if (c.r == 1 && t->prm.bw_mode == ASKIT_BW_CONSTANT) {
        // the same rounding as the per-row values (h held in FP32)
        const double hf = (double)(float)t->prm.h;
        const float sc1 = (float)(t->prm.kernel_scale * 1.4426950408889634 / (hf * hf));
        a.uni_a = 2.f * sc1;
        a.uni_c = -sc1;
        return run_tf32<1, true>(t, c, st, a, sc.n_ctas, s);
    }
    if (c.r == 1) return run_tf32<1, false>(t, c, st, a, sc.n_ctas, s);
    if (c.r <= 4) return run_tf32<4, false>(t, c, st, a, sc.n_ctas, s);
    return run_tf32<16, false>(t, c, st, a, sc.n_ctas, s);
}

void eval_tf32_free(askit_tree t) {
    delete (FState *)t->tf32;
    t->tf32 = nullptr;
}
