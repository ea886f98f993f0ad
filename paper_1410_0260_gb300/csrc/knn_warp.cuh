// Warp-level best-32 lists of the nearest-neighbor searches.
#pragma once
#include <float.h>
#include <limits.h>

#include "askit_impl.cuh"

namespace {

constexpr unsigned FULL = 0xffffffffu;

// Order by (D, id).  Distances are sums of squares, never negative nor -0, so their
// bits order them as integers (a NaN behind every number): two FP64 comparisons would
// hold the warp's quarter of the SM for 128 cycles.
__device__ __forceinline__ bool kv_less(double da, int ia, double db, int ib) {
    const unsigned long long a = (unsigned long long)__double_as_longlong(da);
    const unsigned long long b = (unsigned long long)__double_as_longlong(db);
    return a < b || (a == b && ia < ib);
}

// ---------------------------------------------------------------------------
// Warp-level best-32 list: lane l holds the l-th smallest (D, id) so far.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void warp_sort32(double &d, int &i, int lane) {
#pragma unroll
    for (int k = 2; k <= 32; k <<= 1) {
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            double od = __shfl_xor_sync(FULL, d, j);
            int oi = __shfl_xor_sync(FULL, i, j);
            bool keep_min = (((lane & j) == 0) == ((lane & k) == 0));
            bool sw = keep_min ? kv_less(od, oi, d, i) : kv_less(d, i, od, oi);
            if (sw) { d = od; i = oi; }
        }
    }
}

// Merge sorted candidates (cd, ci) into the sorted list (ld, li), keeping the
// 32 smallest: half-cleaner against the reversed candidates, then a bitonic merge.
__device__ __forceinline__ void warp_merge32(double &ld, int &li, double cd, int ci, int lane) {
    double rd = __shfl_sync(FULL, cd, 31 - lane);
    int ri = __shfl_sync(FULL, ci, 31 - lane);
    if (kv_less(rd, ri, ld, li)) { ld = rd; li = ri; }
#pragma unroll
    for (int j = 16; j > 0; j >>= 1) {
        double od = __shfl_xor_sync(FULL, ld, j);
        int oi = __shfl_xor_sync(FULL, li, j);
        bool lower = (lane & j) == 0;
        bool sw = lower ? kv_less(od, oi, ld, li) : kv_less(ld, li, od, oi);
        if (sw) { ld = od; li = oi; }
    }
}

// Offer one batch of candidates (one per lane) to the list.  `dedup` drops
// candidates whose id is already listed (RP iterations revisit pairs).
__device__ __forceinline__ void warp_offer(double &ld, int &li, double cd, int ci, int kappa,
                                           bool dedup, int lane) {
    double wd = __shfl_sync(FULL, ld, kappa - 1);
    int wi = __shfl_sync(FULL, li, kappa - 1);
    bool useful = kv_less(cd, ci, wd, wi);
    if (!__ballot_sync(FULL, useful)) return;
    if (dedup) {
        bool dup = false;
#pragma unroll 8
        for (int l = 0; l < 32; ++l) dup |= (__shfl_sync(FULL, li, l) == ci);
        if (dup) useful = false;
    }
    if (!useful) { cd = DBL_MAX; ci = INT_MAX; }
    warp_sort32(cd, ci, lane);
    warp_merge32(ld, li, cd, ci, lane);
}

// The same list of FP32 keys without ids: lane l holds the l-th smallest value;
// offers one value per lane (values past 3.4e38, or NaN, never enter).
__device__ __forceinline__ void warp_offer_f32(float &l, float v, int kappa, int lane) {
    v = v < 3.4e38f ? v : 3.4e38f;
    if (!__ballot_sync(FULL, v < __shfl_sync(FULL, l, kappa - 1))) return;
#pragma unroll
    for (int k = 2; k <= 32; k <<= 1)
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            const float o = __shfl_xor_sync(FULL, v, j);
            const bool keep_min = (((lane & j) == 0) == ((lane & k) == 0));
            v = keep_min ? fminf(v, o) : fmaxf(v, o);
        }
    l = fminf(l, __shfl_sync(FULL, v, 31 - lane));
#pragma unroll
    for (int j = 16; j > 0; j >>= 1) {
        const float o = __shfl_xor_sync(FULL, l, j);
        l = (lane & j) == 0 ? fminf(l, o) : fmaxf(l, o);
    }
}

// Gathers the values p of the lanes in m, in lane order, behind the `have` values
// already held one a lane; at 32 calls full() (which takes them and sets have = 0)
// and the rest start the next group.
template <class F>
__device__ __forceinline__ void warp_collect(unsigned m, int32_t p, int &have, int32_t &held, int lane, F full) {
    const int k = __popc(m);
    const int src = lane >= have && lane < have + k ? (int)__fns(m, 0, lane - have + 1) : 0;
    const int32_t moved = __shfl_sync(FULL, p, src);
    if (lane >= have && lane < have + k) held = moved;
    if (have + k < 32) {
        have += k;
        return;
    }
    const int rest = have + k - 32;
    have = 32;
    full();
    const int src2 = lane < rest ? (int)__fns(m, 0, k - rest + lane + 1) : 0;
    held = __shfl_sync(FULL, p, src2);
    have = rest;
}

}  // namespace
