// Evaluate (Algorithm 4) on the tcgen05 tensor cores in BF16x3, d <= 64.
//
// Work item = one source sub-block (<= 128 rows of a leaf's points for the
// direct near field, or of a node's skeleton for the far field) against up
// to 128 targets that all need it (see eval_lists.cu).  For each item
//
//     G = A B^T             (tcgen05.mma, 128 x 128 x 64, FP32 accumulators in TMEM)
//     r^2 = (|a|^2 + 2 a.delta) + |y - c_T|^2 - 2 G
//     partial_t = sum_j exp2(-c log2(e) r^2 / h_j^2) w_j
//
// with a = x - c_T (targets centered on the item's first target c_T),
// b = y - c_B (sources centered on their sub-block's mean c_B, pre-split in
// HBM) and delta = c_T - c_B, an exact rewriting of |x - y|^2.  Every term
// is bounded by the spread of the item's targets or by |x - y| itself, so
// the FP32 rounding of the norm expansion stays at that scale even for the
// wide skeletons of high tree nodes.  The contraction is split in three
// products (hi*hi + hi*lo + lo*hi) of BF16 parts with FP32
// accumulation.
//
// One CTA per SM, warp-specialized, 448 threads:
//   warps 0-7  loaders, two groups taking alternate items: thread t centers
//              and splits the item's gathered target row t and stores it in
//              the 128-byte-swizzled K-major layout the tensor core reads
//              (stage = group); it also forms the row term of target t and
//              the column data of source row t;
//   warps 8-11 epilogue: tcgen05.ld of their 32 TMEM lanes (one row each),
//              exponent on MUFU.EX2, reduction against the weights;
//   warp 12    one thread issues the TMA loads of the sub-block (centered,
//              pre-split rows) and the tcgen05.mma instructions, and commits
//              them to mbarriers;
//   warp 13    gathers the items' target rows (TMA tile::gather4).
// Two TMEM accumulators (2 x 128 columns) let the MMAs of item i+1 run
// while the epilogue drains item i.  Every mbarrier wait is bounded: on
// timeout the kernel records ASK_DEV_TIMEOUT, all roles leave their loops,
// and TMEM is freed before the kernel returns.
#include <cuda.h>
#include <cuda_bf16.h>

#include <mutex>

#include "askit_impl.cuh"
#include "tc_ptx.cuh"

namespace {

using namespace tcx;

constexpr int TC_THREADS = 448;
constexpr int TILE_ROWS = 128;                  // M = N = 128
constexpr int REGION = TILE_ROWS * 128;         // one 128-row x 128-byte swizzled region (16 KB)
constexpr uint32_t TMEM_COLS = 256;             // two 128-column FP32 accumulators

// Precision traits: element bytes, swizzle regions per operand (TC_K
// elements x element bytes / 128), MMA K steps, tcgen05 operand format.
template <int P> struct Prec;
template <> struct Prec<ASKIT_PREC_BF16X3> {
    static constexpr int EB = 2, NREG = 1, KSTEPS = 4;   // K = 16 per MMA
    static constexpr uint32_t FMT = 1;                   // BF16 in .kind::f16
};

// Shared-memory plan (offsets from a 1024-byte aligned base).
template <int P>
struct Smem {
    // targets are gathered by TMA (tile::gather4) and the loaders work from shared
    // memory only
    static constexpr int OPB = Prec<P>::NREG * REGION;    // one operand (hi or lo) of one tile
    static constexpr int B_HI = 0, B_LO = OPB;
    static constexpr int A0 = 2 * OPB;                     // stage s: hi at A0 + s*2*OPB, lo at + OPB
    static constexpr int TILES = 6 * OPB;
    static constexpr int RAWSTAGE = TILE_ROWS * TC_K * 4;  // one stage of gathered FP32 target rows
    static constexpr int RAW = TILES;                      // [2] stages
    static constexpr int RAWB = RAW + 2 * RAWSTAGE;        // raw FP32 source rows
    static constexpr int CENT = RAWB + RAWSTAGE;           // float [TC_K] c_B of the sub-block
    static constexpr int ANORM = CENT + TC_K * 4;                         // float [2][128] |a|^2 + 2 a.delta
    static constexpr int COLV = ANORM + 2 * 128 * 4;       // float4 [2][128]: per source pair {A, B}, {C, w} (see loader)
    static constexpr int RC_MAX = 16;
    static constexpr int COLW = COLV + 2 * 128 * 16;       // float [2][128][RC_MAX] weights (r > 1)
    static constexpr int BAR = COLW + 2 * 128 * RC_MAX * 4;   // 15 mbarriers
    static constexpr int MISC = BAR + 16 * 8;              // tmem address, abort flag
    static constexpr int BYTES = MISC + 16;
};

struct TcArgs {
    const EvalItem *items;
    const int32_t *block_off;
    const int32_t *cta_off, *cta_blocks;   // this CTA's sub-blocks: cta_blocks[cta_off[c] .. cta_off[c+1])
    const int32_t *tgt;       // entry -> target slot
    int d_pad;
    const float *cent;        // [n_sub, TC_K]
    const float *sc_t, *sc_s; // c log2(e) / h^2 per source row
    const float *Wt, *Ws;
    int r;
    float f16_scale;          // prescale of the 16-bit operands (1: BF16 is not prescaled)
    float g_unscale;          // 1 / f16_scale^2
    float *partial;
    int *status;
};

template <int P, int RC>
__global__ void __launch_bounds__(TC_THREADS, 1)
eval_tc_kernel(const __grid_constant__ CUtensorMap map_t_hi, const __grid_constant__ CUtensorMap map_t_lo,
               const __grid_constant__ CUtensorMap map_s_hi, const __grid_constant__ CUtensorMap map_s_lo,
               const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_rt,
               const __grid_constant__ CUtensorMap map_rs, const TcArgs args) {
    using S = Smem<P>;
    constexpr int EB = Prec<P>::EB, NREG = Prec<P>::NREG, KSTEPS = Prec<P>::KSTEPS;
    constexpr uint32_t IDESC = make_idesc(Prec<P>::FMT, TILE_ROWS, TILE_ROWS);
    extern __shared__ uint8_t smem_raw[];
    uint8_t *sm = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const uint32_t sbase = smem_u32(sm);
    float *a_norm = reinterpret_cast<float *>(sm + S::ANORM);
    float4 *colv = reinterpret_cast<float4 *>(sm + S::COLV);
    float *colw = reinterpret_cast<float *>(sm + S::COLW);
    const uint32_t bar0 = sbase + S::BAR;
    auto BAR_A_FULL = [&](int s) { return bar0 + 8 * s; };
    auto BAR_A_EMPTY = [&](int s) { return bar0 + 8 * (2 + s); };
    // the sub-block's tiles: block lb completes phase lb >> 1 of barrier lb & 1.
    // A loader group may have no item in a block, but has one in any two
    // consecutive blocks, so it never waits for a phase more than one ahead of
    // the last one it knows complete (with one barrier for all blocks it did,
    // and could pass on the parity of a phase two back).
    auto BAR_B_FULL = [&](int s) { return bar0 + 8 * (s ? 14 : 4); };
    const uint32_t BAR_B_EMPTY = bar0 + 8 * 5;
    auto BAR_T_FULL = [&](int a) { return bar0 + 8 * (6 + a); };
    auto BAR_T_EMPTY = [&](int a) { return bar0 + 8 * (8 + a); };
    auto BAR_R_FULL = [&](int a) { return bar0 + 8 * (10 + a); };    // gathered target rows landed
    auto BAR_R_EMPTY = [&](int a) { return bar0 + 8 * (12 + a); };   // loader done with the raw stage
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(sm + S::MISC);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(sm + S::MISC + 4);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        mbar_init(BAR_A_FULL(0), 128);
        mbar_init(BAR_A_FULL(1), 128);
        mbar_init(BAR_A_EMPTY(0), 1);
        mbar_init(BAR_A_EMPTY(1), 1);
        mbar_init(BAR_B_FULL(0), 1);
        mbar_init(BAR_B_FULL(1), 1);
        mbar_init(BAR_B_EMPTY, 1);
        mbar_init(BAR_T_FULL(0), 1);
        mbar_init(BAR_T_FULL(1), 1);
        mbar_init(BAR_T_EMPTY(0), 128);
        mbar_init(BAR_T_EMPTY(1), 128);
        mbar_init(BAR_R_FULL(0), 1);
        mbar_init(BAR_R_FULL(1), 1);
        mbar_init(BAR_R_EMPTY(0), 128);
        mbar_init(BAR_R_EMPTY(1), 128);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 12) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(tmem_slot)), "r"(TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    pdl_wait();          // the set-up above overlaps the kernels before; everything below reads their results
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp < 8) {
        // ------------------------------------------------------------ loaders
        // two groups of four warps take alternate items (group g fills stage g);
        // thread t of a group owns target row t and source row t of its items
        const int grp = warp >> 2;
        const int t = tid & 127;
        const int nk4 = args.d_pad / 4;            // 16-byte chunks of a coordinate row
        int li = 0, lb = 0;
        for (int ci = args.cta_off[blockIdx.x]; ci < args.cta_off[blockIdx.x + 1] && !*abort_flag; ++ci) {
            const int b = args.cta_blocks[ci];
            const int i0 = args.block_off[b], i1 = args.block_off[b + 1];
            const int li_block_end = li + (i1 - i0);
            EvalItem item = args.items[i0];
            const bool far = item.nrows < 0;
            const int nrows = item.nrows & 0x7fffffff;
            const bool has_src = t < nrows;
            const int64_t srow = (int64_t)item.row0 + t;
            // block-constant column data of source row t: c log2(e) / h^2 and w
            const float sc = has_src ? __ldg((far ? args.sc_s : args.sc_t) + srow) : 0.f;
            const float *wrow = (far ? args.Ws : args.Wt) + srow * args.r;
            const float w0 = has_src ? __ldg(wrow) : 0.f;
            bool waited_b = false;   // B_FULL of this block waited (gather path)
            // this group's first item of the block
            int it = i0 + (((li & 1) ^ grp) & 1);
            if (it < i1) item = args.items[it];
            bool next_tgt = it < i1 && t < item.cnt;
            li += ((li & 1) ^ grp) & 1;
            for (; it < i1; it += 2, li += 2) {
                const int s = li & 1;
                const uint32_t par = ((li >> 1) & 1) ^ 1;
                const bool has_tgt = next_tgt;
                // this group's next item of the block, ahead (only its size: the
                // gather warp fetches the rows)
                if (it + 2 < i1) {
                    item = args.items[it + 2];
                    next_tgt = t < item.cnt;
                }
                if (!mbar_wait(BAR_A_EMPTY(s), par, abort_flag, args.status)) goto loader_done;
                if (!mbar_wait(BAR_T_EMPTY(s), par, abort_flag, args.status)) goto loader_done;
                uint8_t *ahi = sm + S::A0 + s * 2 * S::OPB;
                uint8_t *alo = ahi + S::OPB;
                float nn = 0.f, dd = 0.f, qq = 0.f;
                {
                    // gathered target rows (stage s) and the sub-block's raw rows
                    if (!mbar_wait(BAR_R_FULL(s), (li >> 1) & 1, abort_flag, args.status)) goto loader_done;
                    if (!waited_b) {
                        if (!mbar_wait(BAR_B_FULL(lb & 1), (lb >> 1) & 1, abort_flag, args.status)) goto loader_done;
                        waited_b = true;
                    }
                    const float *raw = reinterpret_cast<const float *>(sm + S::RAW + s * S::RAWSTAGE);
                    const float *rawb = reinterpret_cast<const float *>(sm + S::RAWB);
                    const float *cBs = reinterpret_cast<const float *>(sm + S::CENT);
                    const int dp = args.d_pad;
                    // packed FP32x2 arithmetic: two coordinates per instruction
                    const float2 m1 = make_float2(-1.f, -1.f), z2 = make_float2(0.f, 0.f);
                    const float2 sc2 = make_float2(args.f16_scale, args.f16_scale);
                    float2 nn2 = z2, dd2 = z2, qq2 = z2;
#pragma unroll 4
                    for (int j = 0; j < TC_K / 4; ++j) {
                        // chunks in an order rotated by the row: conflict-free shared loads
                        const int k4 = (j + t) & (nk4 - 1);
                        float2 xa[2] = {z2, z2};
                        int kst = j;   // chunk to store (zeros past d_pad)
                        if (j < nk4) {
                            kst = k4;
                            const float4 tt = *reinterpret_cast<const float4 *>(raw + 4 * k4);   // c_T = row 0
                            const float4 bb = *reinterpret_cast<const float4 *>(cBs + 4 * k4);
                            const float4 xx = has_tgt ? *reinterpret_cast<const float4 *>(raw + t * dp + 4 * k4) : tt;
                            const float4 yy = has_src ? *reinterpret_cast<const float4 *>(rawb + t * dp + 4 * k4) : tt;
                            const float2 tv[2] = {make_float2(tt.x, tt.y), make_float2(tt.z, tt.w)};
                            const float2 bv[2] = {make_float2(bb.x, bb.y), make_float2(bb.z, bb.w)};
                            const float2 xv[2] = {make_float2(xx.x, xx.y), make_float2(xx.z, xx.w)};
                            const float2 yv[2] = {make_float2(yy.x, yy.y), make_float2(yy.z, yy.w)};
#pragma unroll
                            for (int e = 0; e < 2; ++e) {
                                xa[e] = __ffma2_rn(tv[e], m1, xv[e]);                        // a = x - c_T
                                nn2 = __ffma2_rn(xa[e], xa[e], nn2);
                                dd2 = __ffma2_rn(xa[e], __ffma2_rn(bv[e], m1, tv[e]), dd2);   // a . delta
                                const float2 ya = __ffma2_rn(tv[e], m1, yv[e]);              // y - c_T
                                qq2 = __ffma2_rn(ya, ya, qq2);
                            }
                        }
                        // 4 elements = 8 bytes of the 128-byte row; packed 2-wide conversions
                        uint32_t hv[2], lv[2];
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            const float2 v = xa[e];
                            const __nv_bfloat162 h = __float22bfloat162_rn(v);
                            const __nv_bfloat162 l = __float22bfloat162_rn(__ffma2_rn(__bfloat1622float2(h), m1, v));
                            hv[e] = *reinterpret_cast<const uint32_t *>(&h);
                            lv[e] = *reinterpret_cast<const uint32_t *>(&l);
                        }
                        const int off = t * 128 + (((kst >> 1) ^ (t & 7)) << 4) + (kst & 1) * 8;
                        *reinterpret_cast<uint2 *>(ahi + off) = make_uint2(hv[0], hv[1]);
                        *reinterpret_cast<uint2 *>(alo + off) = make_uint2(lv[0], lv[1]);
                    }
                    nn = nn2.x + nn2.y;
                    dd = dd2.x + dd2.y;
                    qq = qq2.x + qq2.y;
                    if (!has_tgt) nn = dd = 0.f;
                }
                // row term |a|^2 + 2 a.delta; column data of source row t:
                // arg = g (2 u sc) + (-sc) p_t + (-sc q) = -sc (p_t + q - 2 u g)
                a_norm[s * 128 + t] = nn + 2.f * dd;
                {
                    // column pairs: [pair][0] = {A_j, A_j+1, B_j, B_j+1}, [pair][1] = {C_j, C_j+1, w_j, w_j+1}
                    float *cp = reinterpret_cast<float *>(colv + s * 128 + 2 * (t >> 1));
                    const int h = t & 1;
                    cp[0 + h] = 2.f * args.g_unscale * sc;
                    cp[2 + h] = -sc * qq;
                    cp[4 + h] = -sc;
                    cp[6 + h] = w0;
                }
                if (RC > 1) {
#pragma unroll
                    for (int z = 0; z < RC; ++z)
                        colw[(s * 128 + t) * RC + z] = (has_src && z < args.r) ? __ldg(wrow + z) : 0.f;
                }
                // generic-proxy stores -> visible to the tensor core's async proxy
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                mbar_arrive(BAR_A_FULL(s));
                mbar_arrive(BAR_R_EMPTY(s));
            }
            // li now points past this block for this group; realign to the block end
            li = li_block_end;
            ++lb;
        }
    loader_done:;
    } else if (warp < 12) {
        // ----------------------------------------------------------- epilogue
        const int row = tid - 256;                 // TMEM lane = target row of the item
        const int q = warp & 3;                    // this warp's TMEM lane quadrant
        int li = 0;
        for (int ci = args.cta_off[blockIdx.x]; ci < args.cta_off[blockIdx.x + 1] && !*abort_flag; ++ci) {
            const int b = args.cta_blocks[ci];
            for (int it = args.block_off[b]; it < args.block_off[b + 1]; ++it, ++li) {
                const int a = li & 1;
                const uint32_t par = (li >> 1) & 1;
                const EvalItem item = args.items[it];
                const int nrows = item.nrows & 0x7fffffff;
                if (!mbar_wait(BAR_A_FULL(a), par, abort_flag, args.status)) goto epi_done;
                if (!mbar_wait(BAR_T_FULL(a), par, abort_flag, args.status)) goto epi_done;
                tc_fence_after();
                float acc[RC];
#pragma unroll
                for (int z = 0; z < RC; ++z) acc[z] = 0.f;
                float2 acc2[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};   // RC == 1
                if (q * 32 < item.cnt) {   // warp-uniform: skip quadrants with no target
                    const float pt = a_norm[a * 128 + row];
                    const float2 pt2 = make_float2(pt, pt);
                    const float4 *cv4 = colv + a * 128;
                    const float *cwp = colw + a * 128 * RC;
                    // columns of 32 in pairs: both TMEM loads issued before one wait
                    auto cols = [&](int c, const uint32_t (&gr)[32]) {
                        float g[32];
#pragma unroll
                        for (int jj = 0; jj < 32; ++jj) g[jj] = __uint_as_float(gr[jj]);
                        if constexpr (RC == 1) {
                            // two columns per step with packed FP32x2 FMAs:
                            // arg = g A + (C p + B) = -sc (p + q - 2 u g); columns past
                            // nrows carry w = 0
#pragma unroll
                            for (int jj = 0; jj < 32; jj += 2) {
                                const float4 ab = cv4[c * 32 + jj];
                                const float4 cw = cv4[c * 32 + jj + 1];
                                const float2 inner = __ffma2_rn(make_float2(cw.x, cw.y), pt2, make_float2(ab.z, ab.w));
                                const float2 arg = __ffma2_rn(make_float2(g[jj], g[jj + 1]), make_float2(ab.x, ab.y), inner);
                                const float2 k = make_float2(ex2_approx(arg.x), ex2_approx(arg.y));
                                acc2[(jj >> 1) & 1] = __ffma2_rn(k, make_float2(cw.z, cw.w), acc2[(jj >> 1) & 1]);
                            }
                        } else {
#pragma unroll
                            for (int jj = 0; jj < 32; ++jj) {
                                const int j = c * 32 + jj;
                                const float4 ab = cv4[j & ~1];
                                const float4 cw = cv4[(j & ~1) + 1];
                                const bool h = j & 1;
                                const float A = h ? ab.y : ab.x, B = h ? ab.w : ab.z, Cc = h ? cw.y : cw.x;
                                const float k = ex2_approx(fmaf(g[jj], A, fmaf(Cc, pt, B)));
#pragma unroll
                                for (int z = 0; z < RC; ++z) acc[z] = fmaf(k, cwp[j * RC + z], acc[z]);
                            }
                        }
                    };
                    const uint32_t tbase = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(a * 128);
#pragma unroll 1
                    for (int c = 0; c < 4 && c * 32 < nrows; c += 2) {
                        uint32_t g0[32], g1[32];
                        const bool two = (c + 1) * 32 < nrows;      // warp-uniform
                        tmem_ld32_async(tbase + (uint32_t)(c * 32), g0);
                        if (two) tmem_ld32_async(tbase + (uint32_t)((c + 1) * 32), g1);
                        tmem_wait_pin(g0);
                        cols(c, g0);
                        if (two) {
                            reg_pin(g1);
                            cols(c + 1, g1);
                        }
                    }
                    if constexpr (RC == 1) acc[0] = (acc2[0].x + acc2[0].y) + (acc2[1].x + acc2[1].y);
                }
                tc_fence_before();
                mbar_arrive(BAR_T_EMPTY(a));
                if (row < item.cnt) {
                    float *p = args.partial + (int64_t)(item.e0 + row) * args.r;
#pragma unroll
                    for (int z = 0; z < RC; ++z)
                        if (z < args.r) p[z] = acc[z];
                }
            }
        }
    epi_done:;
    } else if (warp == 13) {
        // ---------------------------------------------- target-row gatherer (warp 13)
        {
            const uint32_t bytes = (uint32_t)(TILE_ROWS * args.d_pad * 4);
            int li = 0, issued = 0;
            for (int ci = args.cta_off[blockIdx.x]; ci < args.cta_off[blockIdx.x + 1] && !*abort_flag; ++ci) {
                const int b = args.cta_blocks[ci];
                for (int it = args.block_off[b]; it < args.block_off[b + 1]; ++it, ++li) {
                    const int s = li & 1;
                    if (!mbar_wait(BAR_R_EMPTY(s), ((li >> 1) & 1) ^ 1, abort_flag, args.status)) goto gather_done;
                    const EvalItem item = args.items[it];
                    const int first = args.tgt[item.e0];
                    int r[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int row = 4 * lane + i;   // rows past cnt repeat the first target
                        r[i] = row < item.cnt ? args.tgt[item.e0 + row] : first;
                    }
                    ++issued;
                    if (lane == 0) mbar_expect_tx(BAR_R_FULL(s), bytes);
                    __syncwarp();
                    tma_gather4(sbase + S::RAW + s * S::RAWSTAGE + 4 * lane * args.d_pad * 4, &map_q, 0, r[0], r[1],
                                r[2], r[3], BAR_R_FULL(s));
                }
            }
        gather_done:
            // rows of the last two items may still be landing after an abort
            for (int gg = issued > 2 ? issued - 2 : 0; gg < issued; ++gg) mbar_drain(BAR_R_FULL(gg & 1), (gg >> 1) & 1);
        }
    } else if (warp == 12 && lane == 0) {
        // ------------------------------------------------- TMA + MMA issuer
        // hi + lo of one 128-row sub-block, and its raw FP32 rows
        const uint32_t TX = 2 * NREG * REGION + (uint32_t)(TILE_ROWS * args.d_pad * 4 + TC_K * 4);
        int li = 0, lb = 0, b_issued = 0;
        for (int ci = args.cta_off[blockIdx.x]; ci < args.cta_off[blockIdx.x + 1] && !*abort_flag; ++ci, ++lb) {
            const int b = args.cta_blocks[ci];
            const EvalItem first = args.items[args.block_off[b]];
            const bool far = first.nrows < 0;
            if (!mbar_wait(BAR_B_EMPTY, (lb & 1) ^ 1, abort_flag, args.status)) goto mma_done;
            b_issued = lb + 1;
            mbar_expect_tx(BAR_B_FULL(lb & 1), TX);
            const CUtensorMap *mh = far ? &map_s_hi : &map_t_hi;
            const CUtensorMap *ml = far ? &map_s_lo : &map_t_lo;
#pragma unroll
            for (int g = 0; g < NREG; ++g) {
                const int x = g * (128 / EB);      // first element of swizzle region g
                tma_load_2d(sbase + S::B_HI + g * REGION, mh, x, first.row0, BAR_B_FULL(lb & 1));
                tma_load_2d(sbase + S::B_LO + g * REGION, ml, x, first.row0, BAR_B_FULL(lb & 1));
            }
            tma_load_2d(sbase + S::RAWB, far ? &map_rs : &map_rt, 0, first.row0, BAR_B_FULL(lb & 1));
            bulk_copy(sbase + S::CENT, args.cent + (int64_t)first.cidx * TC_K, TC_K * 4, BAR_B_FULL(lb & 1));
            const int i0 = args.block_off[b], i1 = args.block_off[b + 1];
            for (int it = i0; it < i1; ++it, ++li) {
                const int s = li & 1;
                const uint32_t par = (li >> 1) & 1;
                if (!mbar_wait(BAR_A_FULL(s), par, abort_flag, args.status)) goto mma_done;
                if (it == i0 && !mbar_wait(BAR_B_FULL(lb & 1), (lb >> 1) & 1, abort_flag, args.status)) goto mma_done;
                if (!mbar_wait(BAR_T_EMPTY(s), par ^ 1, abort_flag, args.status)) goto mma_done;
                tc_fence_after();
                const uint32_t d_tmem = tmem + (uint32_t)(s * 128);
                const uint32_t a_hi = sbase + S::A0 + s * 2 * S::OPB, a_lo = a_hi + S::OPB;
                const uint32_t b_hi = sbase + S::B_HI, b_lo = sbase + S::B_LO;
                // The tensor core rounds each accumulation step to the running
                // sum's precision, so the small cross terms go in first (while the
                // accumulator is small) and the hi*hi products last.
#pragma unroll
                for (int k = 0; k < KSTEPS; ++k) {
                    // K step k: 32 bytes into swizzle region k / 4
                    const uint32_t off = (uint32_t)((k >> 2) * REGION + (k & 3) * 32);
                    tc_mma<P>(d_tmem, sw128_desc(a_hi + off), sw128_desc(b_lo + off), IDESC, k > 0);
                    tc_mma<P>(d_tmem, sw128_desc(a_lo + off), sw128_desc(b_hi + off), IDESC, 1);
                }
#pragma unroll
                for (int k = 0; k < KSTEPS; ++k) {
                    const uint32_t off = (uint32_t)((k >> 2) * REGION + (k & 3) * 32);
                    tc_mma<P>(d_tmem, sw128_desc(a_hi + off), sw128_desc(b_hi + off), IDESC, 1);
                }
                tc_commit(BAR_A_EMPTY(s));
                tc_commit(BAR_T_FULL(s));
                if (it == i1 - 1) tc_commit(BAR_B_EMPTY);
            }
        }
    mma_done:
        // the last sub-block's copies may still be landing after an abort
        if (b_issued > 0) mbar_drain(BAR_B_FULL((b_issued - 1) & 1), ((b_issued - 1) >> 1) & 1);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 12) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
    }
}

// Tensor maps: the split source rows (boxes of 64 x 128, 128-byte swizzle) [t_hi,
// t_lo, s_hi, s_lo], and the raw FP32 source rows in 128-row boxes.
struct TcState {
    CUtensorMap map[4], raw_t, raw_s;
    bool ready = false;
    EncodeTiledFn encode = nullptr;
};

std::mutex g_tc_mu;   // the tensor maps are built once, under a lock

askit_status tc_state(askit_tree t, TcState **out) {
    std::lock_guard<std::mutex> lock(g_tc_mu);
    if (!t->tc) t->tc = new TcState();
    TcState *st = (TcState *)t->tc;
    if (!st->ready) {
        ASK_TRY(encode_fn(&st->encode));
        const void *arr[4] = {t->Xt_bhi, t->Xt_blo, t->Xs_bhi, t->Xs_blo};
        for (int i = 0; i < 4; ++i)
            ASK_TRY(encode_2d(st->encode, &st->map[i], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, arr[i],
                              i < 2 ? t->N_pad : t->srows, TC_K, 64, TILE_ROWS, CU_TENSOR_MAP_SWIZZLE_128B));
        ASK_TRY(encode_2d(st->encode, &st->raw_t, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, t->Xt, t->N_pad, t->d_pad, t->d_pad,
                          TILE_ROWS, CU_TENSOR_MAP_SWIZZLE_NONE));
        ASK_TRY(encode_2d(st->encode, &st->raw_s, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, t->Xs, t->srows, t->d_pad, t->d_pad,
                          TILE_ROWS, CU_TENSOR_MAP_SWIZZLE_NONE));
        st->ready = true;
    }
    *out = st;
    return ASKIT_OK;
}

template <int P, int RC>
askit_status launch(askit_tree t, TcState *st, const CUtensorMap &map_q, const TcArgs &a, int grid, cudaStream_t s) {
    const size_t smem = Smem<P>::BYTES + 1024;
    static std::atomic<uint64_t> opted{0};
    ASK_TRY(opt_in_smem(eval_tc_kernel<P, RC>, smem, opted));
    ASK_TRY(ktimer_mark(t, s, false));
    ASK_TRY(launch_pdl(eval_tc_kernel<P, RC>, dim3((unsigned)grid), dim3(TC_THREADS), smem, s, st->map[0], st->map[1],
                       st->map[2], st->map[3], map_q, st->raw_t, st->raw_s, a));
    return ktimer_mark(t, s, true);
}

}  // namespace

askit_status eval_tc(askit_tree t, const WeightCtx &c, int precision, const float *Xq, int64_t ldq,
                     int64_t q_rows, const QuerySplit *qs, const WorkLists &w, float *partial, cudaStream_t s) {
    if (t->d > TC_K) return eval_tc_wide(t, c, precision, Xq, ldq, q_rows, w, partial, s);
    // FP16x3 with pre-split, globally centered targets where that keeps FP32
    // grade (eval_g16.cu)
    if (precision == ASKIT_PREC_FP16X3 && qs && use_g16(t)) return eval_g16(t, c, *qs, w, partial, s);
    // FP16x3 and 3xTF32 center both sides on the sub-block mean (eval_tc16.cu,
    // eval_tf32.cu, there except in sub-blocks that are too wide for it); BF16x3 keeps the per-item target centering below: its 8-bit
    // significands leave a residual of about 2^-17 of |a| |b| per product, so the
    // smaller |a| of the per-item center is what keeps it within the split-path
    // tolerance
    if (precision == ASKIT_PREC_FP16X3) return eval_tc16(t, c, precision, Xq, ldq, q_rows, w, partial, s);
    if (precision != ASKIT_PREC_TF32X3 && precision != ASKIT_PREC_BF16X3) {
        askit_set_error("unknown tensor-core precision %d", precision);
        return ASKIT_ERR_INVALID_ARG;
    }
    if (c.r > Smem<ASKIT_PREC_BF16X3>::RC_MAX) {
        askit_set_error("tensor-core evaluation covers r <= %d; use ASKIT_PREC_SIMT_FP32", Smem<ASKIT_PREC_BF16X3>::RC_MAX);
        return ASKIT_ERR_UNSUPPORTED;
    }
    if (w.n_blocks == 0) return ASKIT_OK;
    if (ldq != t->d_pad) {
        askit_set_error("target rows must have d_pad columns");
        return ASKIT_ERR_INVALID_ARG;
    }
    if (precision == ASKIT_PREC_TF32X3) return eval_tf32(t, c, Xq, ldq, w, partial, s);
    TcState *st = nullptr;
    ASK_TRY(tc_state(t, &st));
    // gather map over this call's target rows (one box row per gathered row)
    CUtensorMap map_q;
    ASK_TRY(encode_2d(st->encode, &map_q, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, Xq, q_rows, t->d_pad, t->d_pad, 1,
                      CU_TENSOR_MAP_SWIZZLE_NONE));
    const WorkLists::Sched &sc = w.sched[w.use];
    TcArgs a;
    a.items = w.items;
    a.block_off = sc.run_off;
    a.cta_off = sc.cta_off;
    a.cta_blocks = sc.cta_runs;
    a.tgt = w.tgt;
    a.d_pad = t->d_pad;
    a.cent = t->cent;
    a.sc_t = t->sc_t;
    a.sc_s = t->sc_s;
    a.Wt = c.Wt;
    a.Ws = c.Ws;
    a.r = c.r;
    a.partial = partial;
    a.status = t->d_status;
    a.f16_scale = 1.f;
    a.g_unscale = 1.f / (a.f16_scale * a.f16_scale);
    if (c.r == 1) return launch<ASKIT_PREC_BF16X3, 1>(t, st, map_q, a, sc.n_ctas, s);
    if (c.r <= 4) return launch<ASKIT_PREC_BF16X3, 4>(t, st, map_q, a, sc.n_ctas, s);
    return launch<ASKIT_PREC_BF16X3, 16>(t, st, map_q, a, sc.n_ctas, s);
}

void eval_tc_free(askit_tree t) {
    delete (TcState *)t->tc;
    t->tc = nullptr;
    eval_tc_wide_free(t);
    eval_tc16_free(t);
    eval_tf32_free(t);
    eval_g16_free(t);
}
