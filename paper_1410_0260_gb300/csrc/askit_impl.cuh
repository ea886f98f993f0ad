// Internal declarations of the GB300 ASKIT library: the tree object, error
// plumbing, and the canonical FP64 arithmetic that makes the setup stages
// (kNN, tree, skeletons) reproducible bit for bit on any IEEE machine.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <chrono>
#include <string>
#include <vector>

#include "askit.h"

// ---------------------------------------------------------------------------
// Errors
// ---------------------------------------------------------------------------
void askit_set_error(const char *fmt, ...);

#define ASK_CUDA(call)                                                                 \
    do {                                                                               \
        cudaError_t e_ = (call);                                                       \
        if (e_ != cudaSuccess) {                                                       \
            askit_set_error("%s:%d %s: %s", __FILE__, __LINE__, #call,                 \
                            cudaGetErrorString(e_));                                   \
            return e_ == cudaErrorMemoryAllocation ? ASKIT_ERR_OOM : ASKIT_ERR_CUDA;   \
        }                                                                              \
    } while (0)

#define ASK_TRY(call)                                \
    do {                                             \
        askit_status s_ = (call);                    \
        if (s_ != ASKIT_OK) return s_;               \
    } while (0)

#define ASK_LAUNCH()                                 \
    do {                                             \
        ASK_CUDA(cudaGetLastError());                \
    } while (0)

// Lets kernel k take `bytes` of dynamic shared memory.  The attribute belongs to a
// device, so it is set at the first launch on each; `opted` (static at the caller, one a
// kernel) has the bits of those where it is.
template <class... KArgs>
inline askit_status opt_in_smem(void (*k)(KArgs...), size_t bytes, std::atomic<uint64_t> &opted) {
    int dev = 0;
    ASK_CUDA(cudaGetDevice(&dev));
    const uint64_t bit = dev < 64 ? (uint64_t)1 << dev : 0;
    if (opted.load() & bit) return ASKIT_OK;
    ASK_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
    opted.fetch_or(bit);
    return ASKIT_OK;
}

// Launches kernel k so that it may start while the kernel before it on the
// stream still runs (programmatic stream serialization).  Every kernel launched
// this way calls pdl_wait() in every thread before it reads or writes anything
// that an earlier kernel of the stream touches; what it does before that
// (barriers, TMEM, operands fixed at setup) overlaps the earlier kernel's tail.
// set_weights starts with a normal launch; Evaluate with its column data, launched this
// way: before its wait that kernel reads constants of the tree alone.
template <class... KArgs, class... Args>
inline askit_status launch_pdl(void (*k)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                               const Args &...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    ASK_CUDA(cudaLaunchKernelEx(&cfg, k, static_cast<KArgs>(args)...));
    return ASKIT_OK;
}
// Lets the next kernel of the stream be launched once every block has got here.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// Waits until the earlier kernels of the stream have completed (no-op after a
// normal launch).
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Sticky device status codes (written by kernels with bounded waits).
enum { ASK_DEV_OK = 0, ASK_DEV_TIMEOUT = 1, ASK_DEV_BAD_ITEM = 2 };

// Rows of each skeleton block and of the target/source arrays are padded to a
// multiple of this, so that tensor-core tiles never straddle two blocks.
constexpr int ASK_ROW_PAD = 32;
// Targets per evaluation item (one tensor-core M tile).
constexpr int ASK_TILE_M = 128;
// Source rows per sub-block (one tensor-core N tile); leaves and skeletons
// longer than this are split into consecutive sub-blocks.
constexpr int ASK_BLK_N = 128;
// Items of one run of a sub-block's items with wide rows (d > TC_K).
constexpr int ASK_SEG_ITEMS = 8;
// Sub-blocks past this value of rho = sc_max max |y - c_B|^2 (sc = c log2(e) / h^2)
// are too wide for the 3xTF32 kernel's common center c_B: the exponent's rounding
// error is about 1.6e-7 rho where a target meets near points far from c_B (a node
// that median splits left with parts of two clusters, or with an outlier), 2e-5 at
// this line, a fifth of the split products' tolerance.  Points without gaps stay
// below it: at most 106 over the leaves and skeletons of 64K x 64 manifold points.
constexpr float ASK_WIDE_RHO = 128.f;
// Columns of the tensor-core operand arrays (d <= TC_K).
constexpr int TC_K = 64;
// Default and largest entries of one in-sample work-list batch (entry
// offsets inside a batch are int32).
constexpr int64_t ASK_BATCH_ENTRIES = (int64_t)1 << 28;
constexpr int64_t ASK_BATCH_ENTRIES_MAX = (int64_t)1 << 30;

// ---------------------------------------------------------------------------
// Device memory owned by a tree: every allocation is recorded and freed by
// askit_destroy.
// ---------------------------------------------------------------------------
struct DevArena {
    std::vector<void *> ptrs;
    size_t bytes = 0;
    // stream-ordered mode (per-call temporaries): allocated from the pool and freed
    // on `stream`, so freeing does not synchronize the device
    bool async = false;
    cudaStream_t stream = nullptr;
    cudaMemPool_t pool = nullptr;
    // otherwise: a pool whose unused memory is given back before an allocation fails
    cudaMemPool_t trim = nullptr;
    template <class T>
    askit_status alloc(T **p, size_t count) {
        *p = nullptr;
        if (count == 0) count = 1;
        void *q = nullptr;
        cudaError_t e = async ? cudaMallocFromPoolAsync(&q, count * sizeof(T), pool, stream) : cudaMalloc(&q, count * sizeof(T));
        if (e == cudaErrorMemoryAllocation && !async && trim) {
            cudaGetLastError();
            cudaDeviceSynchronize();                       // frees still in their streams' order
            cudaMemPoolTrimTo(trim, 0);
            e = cudaMalloc(&q, count * sizeof(T));
        }
        if (e != cudaSuccess) {
            askit_set_error("cudaMalloc(%zu bytes): %s", count * sizeof(T), cudaGetErrorString(e));
            return e == cudaErrorMemoryAllocation ? ASKIT_ERR_OOM : ASKIT_ERR_CUDA;
        }
        ptrs.push_back(q);
        bytes += count * sizeof(T);
        *p = static_cast<T *>(q);
        return ASKIT_OK;
    }
    void release(void *p) {
        for (auto &q : ptrs)
            if (q == p) { cudaFree(q); q = nullptr; }
    }
    void free_all() {
        for (void *q : ptrs)
            if (q) {
                if (async) cudaFreeAsync(q, stream);
                else cudaFree(q);
            }
        ptrs.clear();
        bytes = 0;
    }
};

// One evaluation work item: one source sub-block (up to ASK_BLK_N rows of a
// leaf's points, evaluated directly, or of a node's skeleton) against up to
// ASK_TILE_M targets that all need it.  Its targets are entries
// e0 .. e0 + cnt - 1 of the work lists' sorted entry array.
struct __align__(16) EvalItem {
    int32_t row0;    // first source row (in Xt for leaves, in the skeleton pool else)
    int32_t nrows;   // valid source rows; bit 31 set = skeleton (far-field) block
    int32_t e0;      // first entry
    int32_t cnt;     // targets (entries) of this item
    int32_t cidx;    // sub-block index (its center in the centered operand arrays)
    int32_t wide;    // 1: the 3xTF32 kernel centers this item on its targets (sb_wide)
    int32_t pad_[2];
};

// Target rows of one evaluation in the global-centered FP16x3 form: hi / lo
// [rows, TC_K] FP16 of (x - xbar) g_sigma and the norm blocks x [rows, 16].
struct QuerySplit {
    const uint16_t *hi = nullptr, *lo = nullptr, *x = nullptr;
    int64_t rows = 0;
};

// Work lists of one set of targets (in-sample, or one out-of-sample batch).
struct WorkLists {
    int64_t T = 0, n_entries = 0, n_items = 0, n_blocks = 0;
    int64_t *off = nullptr;          // [T + 1] entries of target q: emission slots off[q] .. off[q+1)
    int32_t *slot_of_emit = nullptr; // [n_entries] sorted position of each emitted entry
    int32_t *tgt = nullptr;          // [n_entries] target slot of each sorted entry
    EvalItem *items = nullptr;       // [n_items], grouped by sub-block
    const int32_t *block_off = nullptr;    // [n_blocks + 1] items of each sub-block
    const int32_t *block_order = nullptr;  // [n_blocks] heaviest first
    // Schedules of the persistent kernels.  Every sub-block's items are cut into
    // runs (a paired follower's at its leader's cuts), and the runs are dealt to
    // n_ctas CTAs.  [0]: heaviest sub-block first, its runs one after another,
    // each to the CTA with the least work so far; [1]: the same in tree order;
    // [2]: paired -- the leaders' and the single sub-blocks' runs, partner the
    // follower's run of each run (else -1).  A schedule that was not built
    // (out-of-sample lists have those that a kernel may take) has n_ctas = 0.
    struct Sched {
        int n_ctas = 0;
        const int32_t *run_off = nullptr;    // [runs + 1] items of each run
        const int32_t *partner = nullptr;    // [runs] ([2] only)
        const int32_t *cta_off = nullptr;    // [n_ctas + 1]
        const int32_t *cta_runs = nullptr;   // runs of each CTA, in order
    } sched[3];
    int32_t *plan = nullptr;         // the device array that holds the above, block_off and block_order
    int use = 0;                     // schedule in use without pairs: 0 or 1
    int64_t n_pairs = 0;             // leader sub-blocks with a paired follower
    int64_t pair_items = 0;          // their items (a follower has as many)
    int64_t pairs_alg = 0, pairs_cmp = 0, near_tot = 0, far_tot = 0;
};

// Weights of one evaluation context: W in tree order, the skeleton weights
// of the upward pass, and the per-entry partial sums of Evaluate.  A tree
// has a default context; askit_weights_create adds independent ones, so
// several weight sets can be evaluated concurrently on different streams.
struct WeightCtx {
    int r = 0, r_cap = 0;
    float *Wt = nullptr;       // [N_pad, r] weights in tree order
    float *Ws = nullptr;       // [rows of the skeleton pool, r] skeleton weights
    float *partial = nullptr;  // [in-sample entries, r_cap]
    float4 *colv = nullptr;    // [n_sub, 128] per-sub-block column data (16-bit tensor-core path)
    float *colw = nullptr;     // [n_sub, 128 * 16 + 16] per-sub-block weights (r > 1)
    int64_t ent_cap = 0;       // entries the partial sums hold
    bool ready = false;
    DevArena arena;
};

struct askit_tree_s;
struct askit_weights_s {
    askit_tree_s *t = nullptr;
    WeightCtx ctx;
};

// A captured set_weights + evaluate step with its own weight context.
struct askit_graph_s {
    askit_tree_s *t = nullptr;
    WeightCtx ctx;
    cudaGraphExec_t exec = nullptr;
    int64_t n_nodes = 0;
};

// Bytes of freed temporaries a tree's pool keeps for the next call.
constexpr uint64_t ASK_POOL_KEEP = (uint64_t)1 << 30;

struct askit_tree_s {
    askit_params prm;
    // Temporaries of the out-of-sample calls.  The device's default pool returns
    // freed memory to the system at every synchronization, and mapping it again
    // cost most of a small call (100 targets: 0.75 ms, 0.33 of it kernels) and
    // 3 ms of a large one; this pool keeps up to ASK_POOL_KEEP of it, never makes
    // one stream wait for another's free, and goes with the tree.
    cudaMemPool_t pool = nullptr;
    int64_t N = 0;
    int d = 0, d_pad = 0, L = 0, kappa = 0, rp_leaf = 0, ell_max = 0;
    int64_t n_nodes = 0;
    DevArena arena;

    // caller-order data
    float *X = nullptr;        // [N, d]
    float *hsrc = nullptr;     // [N]
    int32_t *knn = nullptr;    // [N, kappa]
    double *knnd = nullptr;    // [N, kappa]

    // tree
    int32_t *perm = nullptr;   // [N] tree position -> point id
    int32_t *pos = nullptr;    // [N] point id -> tree position
    int32_t *leafof = nullptr; // [N] point id -> leaf heap index
    std::vector<int64_t> h_start, h_size;
    int32_t *nstart = nullptr, *nsize = nullptr;  // [n_nodes]

    // node neighbor lists and sampled targets ([n_nodes, ell_max])
    int32_t *nl_cnt = nullptr, *nl_ids = nullptr;
    double *nl_key = nullptr;
    int32_t *trows = nullptr;

    // skeletons, heap order pools
    std::vector<int32_t> h_s, h_ncol;
    std::vector<int64_t> h_skoff, h_pivoff, h_poff, h_spool;
    int64_t skel_total = 0, piv_total = 0, p_total = 0, spool_rows = 0;
    int32_t *skel_ids = nullptr;  // [skel_total]
    int32_t *piv = nullptr;       // [piv_total]
    double *P64 = nullptr;        // [p_total]
    // FP32 copy for the upward pass: node a's rows start at d_p32off[a] and are
    // (c_a - s_a) floats padded with zeros to a multiple of 4 apart (16-byte loads)
    float *P32 = nullptr;
    std::vector<int> lvl_nr;      // [L + 1] largest c_a - s_a of each level
    int64_t *d_skoff = nullptr, *d_pivoff = nullptr, *d_p32off = nullptr, *d_spool = nullptr;
    int32_t *d_s = nullptr, *d_ncol = nullptr;

    // evaluation operands
    int64_t N_pad = 0;
    float *Xt = nullptr;       // [N_pad, d_pad] tree order, zero padded
    float *Xs = nullptr;       // [spool_rows, d_pad] skeleton coordinate pool
    float *nrm_t = nullptr, *nrm_s = nullptr;   // squared norms
    float *sc_t = nullptr, *sc_s = nullptr;     // c * log2(e) / h_j^2 per source row
    WeightCtx dw;              // default weight context (askit_set_weights)
    int precision = ASKIT_PREC_TF32X3;

    // in-sample work lists, one per batch of consecutive target slots
    // [wl_t0[b], wl_t0[b + 1]); the partial sums are sized for the largest
    std::vector<WorkLists> wl;
    std::vector<int64_t> wl_t0;
    int64_t wl_entries = 0, wl_entries_max = 0;

    // tensor-core operands: every source sub-block centered on its own mean,
    // split into hi + lo parts (TF32 and BF16), kw columns (TC_K, or d_pad
    // for wide rows, whose 16-bit splits are stored as planes of 8-column K
    // groups, [kw / 8][rows][8]), and the squared norms of the centered rows
    int64_t n_sub = 0;
    int32_t *leaf_cbase = nullptr; // [2^L] first sub-block of each leaf
    int32_t *node_cbase = nullptr; // [n_nodes] first sub-block of each skeleton
    float *cent = nullptr;         // [n_sub, kw]
    float *Xt_hi = nullptr, *Xt_lo = nullptr, *Xs_hi = nullptr, *Xs_lo = nullptr;   // TF32 split
    uint16_t *Xt_bhi = nullptr, *Xt_blo = nullptr, *Xs_bhi = nullptr, *Xs_blo = nullptr; // BF16 split
    uint16_t *Xt_hhi = nullptr, *Xt_hlo = nullptr, *Xs_hhi = nullptr, *Xs_hlo = nullptr; // FP16 split (prescaled)
    float f16_scale = 1.f;         // power of 2 keeping centered coordinates within FP16 range
    float *nrmc_t = nullptr, *nrmc_s = nullptr;
    int64_t srows = 0;             // rows of the skeleton-pool arrays

    // global-centered FP16x3 operands (d <= TC_K, eval_g16.cu): every point
    // centered on the data mean g_xbar; targets (x - xbar) g_sigma and
    // sources (y - xbar) 2 sc_j / g_sigma split into FP16 hi + lo; the norm
    // blocks of targets [rows, 16] and of every source sub-block (scales
    // g_tau, g_kappa); n = |x - xbar|^2, g_r2max the largest.  g_rho = max_j sc_j * max_i n_i
    // decides the automatic choice (g_ok)
    uint16_t *Xg_hi = nullptr, *Xg_lo = nullptr, *Xg_x = nullptr;   // tree points as targets
    uint16_t *Xb_hi = nullptr, *Xb_lo = nullptr;                    // tree points as sources
    uint16_t *Sb_hi = nullptr, *Sb_lo = nullptr;                    // skeleton pool as sources
    uint16_t *g_bx = nullptr;                                       // [n_sub, 128 x 16]
    float *ng_t = nullptr, *ng_s = nullptr;
    float *g_xbar = nullptr;       // [TC_K] device
    float g_sigma = 1.f, g_tau = 1.f, g_kappa = 1.f;
    double g_rho = 0.0, g_r2max = 0.0;
    bool g_ok = false;
    int fp16_centering = 0;        // 0 automatic (global when g_ok), 1 per sub-block, 2 global
    void *g16 = nullptr;           // tensor maps of the global-centered kernel

    int *d_status = nullptr;       // sticky kernel status
    int *d_ticket = nullptr;       // persistent-kernel work counter
    void *tc = nullptr;            // tensor-core kernel state (tensor maps)
    void *tcw = nullptr;           // the same for the wide (d > TC_K) kernel
    void *tc16 = nullptr;          // the same for the 16-bit narrow kernel
    void *tf32 = nullptr;          // the same for the 3xTF32 kernel
    int64_t *sb_row0 = nullptr;    // [n_sub] first row of each sub-block (Xt rows, then Xs rows)
    int32_t *sb_nr = nullptr;      // [n_sub] rows of each sub-block
    // [n_sub] (d <= TC_K) 1 where sc_max max |y - c_B|^2 over the sub-block's rows
    // exceeds ASK_WIDE_RHO: too wide for 3xTF32 with both sides centered on c_B
    int32_t *sb_wide = nullptr;
    bool any_wide = false;         // one at least
    int64_t n_leaf_sub = 0;        // sub-blocks of leaves (the rest are skeleton sub-blocks)
    std::vector<int64_t> h_sub_pos; // [n_sub] tree position of each sub-block's node (schedule order)
    std::vector<int64_t> h_sub_node; // [n_sub] heap index of each sub-block's node
    // launch configuration of the evaluation kernels (askit_autotune)
    int tune_sched = 0;            // block-to-CTA schedule: 0 LPT, 1 tree-order ranges
    int tune_stages = 0;           // target-row stages of the FP16x3 kernels (2 to 4; 0: each kernel's default)
    int tune_runs = 1;             // 8-row tiled loads for runs of consecutive targets
    int tune_pairs = -1;           // items over two sub-blocks of a node (256 columns): 0, 1, or -1 (take_pairs)
    int spin_limit = 0;            // polls of the FP16x3 kernel's bounded waits (0: default)
    // refinements of the pruning (askit_set_pruning): skeletons only for nodes
    // at most far_height levels above the leaves (-1: all), and the kernel cut
    // of the adaptive kappa_i (0: all kappa neighbors)
    int far_height = -1;
    double kappa_cut = 0.0;
    int kw = TC_K;                 // row width of the pre-split operands and centers
    // wall time of the setup stages (askit_info.setup_ms)
    double setup_ms[7] = {0, 0, 0, 0, 0, 0, 0};
    std::chrono::steady_clock::time_point stage_t0;
    // CUDA events around each launch of the evaluation kernel while timing
    // is on (askit_kernel_timing): begin/end pairs, reused across sessions
    struct KTimer {
        bool on = false;
        std::vector<cudaEvent_t> ev;
        size_t used = 0;
    } kt;
};

// Whether the global-centered and the K-chunked kernel take paired items.  An item
// costs them about the same with one sub-block or two, so by default pairs are
// taken where most items have a partner: 1M x 64 3.94 ms an Evaluate against 4.37
// unpaired, 64K x 64 165 us against 182, 10K x 1000 888 us against 1090; but 6K x
// 700 with single-block skeletons, more singles than pairs, 230 us against 201.
inline bool take_pairs(const askit_tree_s *t, const WorkLists &w) {
    if (t->tune_pairs == 0) return false;
    return t->tune_pairs == 1 || w.pair_items > w.n_items - 2 * w.pair_items;
}

// Records the begin (end = false) or end event of one evaluation-kernel
// launch on stream s while the tree's kernel timer is on; a no-op otherwise
// and while s is being captured into a graph.
askit_status ktimer_mark(askit_tree t, cudaStream_t s, bool end);

// ---------------------------------------------------------------------------
// Canonical FP64 arithmetic (device).  Every operation is an explicitly
// rounded IEEE operation, so no multiply-add is ever fused and results are
// identical to any sequential IEEE-754 binary64 evaluation in the same order.
// ---------------------------------------------------------------------------
__device__ __forceinline__ double c_add(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double c_sub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double c_mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double c_div(double a, double b) { return __ddiv_rn(a, b); }

// x as a double (exact).  The conversion instruction runs on the FP64 pipe, 64
// cycles a warp like an addition, so normal numbers are widened with integer
// operations (a conversion and an addition: 141 cycles, this and an addition: 71).
__device__ __forceinline__ double c_f2d(float x) {
    const unsigned b = __float_as_uint(x), a = b & 0x7fffffffu;
    if (a - 0x00800000u < 0x7f000000u)                     // normal: neither zero, subnormal, infinite nor NaN
        return __hiloint2double((int)((b & 0x80000000u) | ((a >> 3) + 0x38000000u)), (int)(b << 29));
    if (a == 0) return __hiloint2double((int)b, 0);
    return (double)x;
}

// Squared distance, coordinates ascending: sum (x_k - y_k)^2.
__device__ __forceinline__ double c_dist2(const float *x, const float *y, int d) {
    double acc = 0.0;
    for (int k = 0; k < d; ++k) {
        double t = c_sub(c_f2d(x[k]), c_f2d(y[k]));
        acc = c_add(acc, c_mul(t, t));
    }
    return acc;
}

// exp(a) for the ID's kernel matrices: Cody-Waite reduction a = n ln2 + r
// with ln2 split into a 32-significant-bit head and its tail, the degree-13
// Taylor polynomial of e^r in Horner form, and an exact scaling by 2^n
// (n >= -1010 keeps the result normal).  Arguments below -700 give 0.
__device__ __forceinline__ double c_exp(double a) {
    if (a < -700.0) return 0.0;
    if (a > 700.0) return __longlong_as_double(0x7ff0000000000000LL);
    const double inv_ln2 = 0x1.71547652b82fep+0;
    const double ln2_head = 0x1.62e42ff000000p-1;
    const double ln2_tail = -0x1.718432a1b0e26p-35;
    double n = rint(c_mul(a, inv_ln2));
    double r = c_sub(c_sub(a, c_mul(n, ln2_head)), c_mul(n, ln2_tail));
    // 1/k! for k = 13 down to 0
    const double coef[14] = {0x1.6124613a86d09p-33, 0x1.1eed8eff8d898p-29, 0x1.ae64567f544e4p-26,
                             0x1.27e4fb7789f5cp-22, 0x1.71de3a556c734p-19, 0x1.a01a01a01a01ap-16,
                             0x1.a01a01a01a01ap-13, 0x1.6c16c16c16c17p-10, 0x1.1111111111111p-7,
                             0x1.5555555555555p-5,  0x1.5555555555555p-3,  0x1.0000000000000p-1,
                             0x1.0000000000000p+0,  0x1.0000000000000p+0};
    double p = coef[0];
#pragma unroll
    for (int k = 1; k < 14; ++k) p = c_add(c_mul(p, r), coef[k]);
    long long e = (long long)n + 1023;
    return c_mul(p, __longlong_as_double(e << 52));
}

// Philox4x64-10 (Salmon et al., SC'11): 10 rounds of the two 64x64->128
// multiplications with key bumps between rounds.
__device__ __forceinline__ void philox4x64_10(uint64_t c[4], uint64_t k0, uint64_t k1) {
    const uint64_t M0 = 0xD2E7470EE14C6C93ULL, M1 = 0xCA5A826395121157ULL;
    const uint64_t W0 = 0x9E3779B97F4A7C15ULL, W1 = 0xBB67AE8584CAA73BULL;
#pragma unroll
    for (int round = 0; round < 10; ++round) {
        if (round) { k0 += W0; k1 += W1; }
        uint64_t hi0 = __umul64hi(M0, c[0]), lo0 = M0 * c[0];
        uint64_t hi1 = __umul64hi(M1, c[2]), lo1 = M1 * c[2];
        uint64_t n0 = hi1 ^ c[1] ^ k0, n2 = hi0 ^ c[3] ^ k1;
        c[0] = n0; c[1] = lo1; c[2] = n2; c[3] = lo0;
    }
}

// Word n of the stream keyed (k0, k1) under counter prefix c0: block n/4, lane n%4.
__device__ __forceinline__ uint64_t philox_word(uint64_t k0, uint64_t k1, uint64_t c0, uint64_t n) {
    uint64_t c[4] = {c0, n >> 2, 0, 0};
    philox4x64_10(c, k0, k1);
    return c[n & 3];
}

// Depth of heap node a (root 1 has depth 0).
__host__ __device__ __forceinline__ int heap_depth(int64_t a) {
    int t = 0;
    while (((int64_t)2 << t) <= a) ++t;
    return t;
}

// ---------------------------------------------------------------------------
// Stage entry points (one translation unit each)
// ---------------------------------------------------------------------------
// setup_sort.cu: segmented sorts (CUB) used by the tree and node-list stages.
askit_status seg_sort_f64_i32(const double *kin, double *kout, const int32_t *vin, int32_t *vout,
                              int64_t n, int nseg, const int32_t *beg, const int32_t *end,
                              void *tmp, size_t *tmp_bytes, cudaStream_t s);
askit_status seg_sort_i32_f64(const int32_t *kin, int32_t *kout, const double *vin, double *vout,
                              int64_t n, int nseg, const int32_t *beg, const int32_t *end,
                              void *tmp, size_t *tmp_bytes, cudaStream_t s);
askit_status seg_sort_i32(const int32_t *kin, int32_t *kout, int64_t n, int nseg,
                          const int32_t *beg, const int32_t *end, void *tmp, size_t *tmp_bytes,
                          cudaStream_t s);
askit_status sort_f64_i32(const double *kin, double *kout, const int32_t *vin, int32_t *vout, int64_t n, void *tmp,
                          size_t *tmp_bytes, cudaStream_t s);
// stable, keys below 2^bits
askit_status sort_u32_i32(const uint32_t *kin, uint32_t *kout, const int32_t *vin, int32_t *vout,
                          int64_t n, int bits, void *tmp, size_t *tmp_bytes, cudaStream_t s);
askit_status scan_i64(const int64_t *in, int64_t *out, int64_t n, void *tmp, size_t *tmp_bytes,
                      cudaStream_t s);

// setup_tree.cu
int tree_depth(int64_t N, int64_t leaf);
void tree_ranges(int64_t N, int L, std::vector<int64_t> &start, std::vector<int64_t> &size);
askit_status build_tree_gpu(const float *X, int64_t N, int d, int L, int kind, uint64_t seed,
                            int iter, int32_t *order, cudaStream_t s);
// self (optional, [Q]): the point id each query Y row is, excluded from its list
askit_status knn_exact_gpu(const float *X, int64_t N, int d, int kappa, const float *Y, int64_t Q,
                           int32_t *ids, double *dist, cudaStream_t s, const int32_t *self = nullptr);
askit_status knn_rp_gpu(const float *X, int64_t N, int d, int kappa, int iters, int64_t rp_leaf,
                        uint64_t seed, int32_t *ids, double *dist, cudaStream_t s);
askit_status knn_dist_gpu(const float *X, int64_t N, int d, int kappa, const int32_t *ids,
                          double *dist, cudaStream_t s);

// setup_skel.cu
askit_status build_node_lists(askit_tree t, cudaStream_t s);
askit_status build_samples(askit_tree t, cudaStream_t s);
askit_status skeletonize(askit_tree t, cudaStream_t s);

// eval_lists.cu
askit_status build_eval_operands(askit_tree t, cudaStream_t s);
askit_status build_tc_operands(askit_tree t, cudaStream_t s);
// Prune sets of a set of targets: rows of `stride` sorted leaf indices
// padded with INT_MAX; target q uses row set_row[q] (leaf-grouped lists, one
// row per leaf) or, with set_row == nullptr, row q.  cudaMalloc'd.
struct PruneSets {
    int32_t *sets = nullptr;
    int stride = 0;
    int32_t *set_row = nullptr;
};
void free_prune_sets(PruneSets &ps);
askit_status build_insample_lists(askit_tree t, const PruneSets &ps, cudaStream_t s);
void use_schedule(askit_tree t);
askit_status build_work_lists(askit_tree t, const int32_t *sets, int stride, const int32_t *set_row, int64_t T,
                              WorkLists &w, DevArena &arena, bool all_schedules, cudaStream_t s);
askit_status reduce_partials(const WorkLists &w, const float *partial, int r, const int32_t *out_rows,
                             float *U, int64_t ldu, cudaStream_t s);
askit_status insample_prune_sets(askit_tree t, PruneSets &ps, cudaStream_t s);
askit_status oos_prune_sets(askit_tree t, const int32_t *knn, const double *dist, const int32_t *order, int64_t T,
                            int stride, int32_t *sets, int *bad, cudaStream_t s);
// every array of w back to the arena
void free_work_lists(WorkLists &w, DevArena &arena);

// weights.cu
askit_status weights_reserve(askit_tree t, WeightCtx &c, int r, cudaStream_t s);
askit_status upward_weights(askit_tree t, WeightCtx &c, const float *W, int r, int64_t ldw, cudaStream_t s);

// eval_simt.cu / eval_tc.cu: partial[e * r + z] for every entry e of w
askit_status eval_simt(askit_tree t, const WeightCtx &c, const float *Xq, int64_t ldq, const WorkLists &w,
                       float *partial, cudaStream_t s);
askit_status eval_tc(askit_tree t, const WeightCtx &c, int precision, const float *Xq, int64_t ldq,
                     int64_t q_rows, const QuerySplit *qs, const WorkLists &w, float *partial, cudaStream_t s);
void eval_tc_free(askit_tree t);
askit_status eval_tc_wide(askit_tree t, const WeightCtx &c, int precision, const float *Xq, int64_t ldq,
                          int64_t q_rows, const WorkLists &w, float *partial, cudaStream_t s);
void eval_tc_wide_free(askit_tree t);
askit_status eval_tc16(askit_tree t, const WeightCtx &c, int precision, const float *Xq, int64_t ldq, int64_t q_rows,
                       const WorkLists &w, float *partial, cudaStream_t s);
void eval_tc16_free(askit_tree t);
// Column data {A, B, C, w} of every sub-block into c.colv (and, rc = 4 or 16, the
// weights into c.colw): A = 2 sc g_unscale, B = -sc |b|^2, C = -sc; uni (rc = 1):
// {B, w} alone
askit_status block_columns(askit_tree t, const WeightCtx &c, int rc, bool uni, float g_unscale, cudaStream_t s);
// eval_tf32.cu: 3xTF32
askit_status eval_tf32(askit_tree t, const WeightCtx &c, const float *Xq, int64_t ldq, const WorkLists &w,
                       float *partial, cudaStream_t s);
void eval_tf32_free(askit_tree t);
// eval_g16.cu: the global-centered FP16x3 kernel (targets pre-split in q)
askit_status eval_g16(askit_tree t, const WeightCtx &c, const QuerySplit &q, const WorkLists &w, float *partial,
                      cudaStream_t s);
void eval_g16_free(askit_tree t);
askit_status build_g16_operands(askit_tree t, cudaStream_t s);
// target rows X [rows, ldx] (d columns) in the global-centered form of tree t;
// *overflow (if given) is set when a value leaves the FP16-safe range; with an
// order, row i is X[order[i]] (zero from n_order on)
askit_status g16_split_rows(const float *X, int64_t ldx, int d, int64_t rows, const askit_tree_s *t, uint16_t *hi,
                            uint16_t *lo, uint16_t *nx, int *overflow, cudaStream_t s,
                            const int32_t *order = nullptr, int64_t n_order = 0);
// whether FP16x3 evaluations of this tree take the global-centered kernel
inline bool use_g16(const askit_tree_s *t) {
    return t->Xg_hi && (t->fp16_centering == 2 || (t->fp16_centering == 0 && t->g_ok));
}
// knn_oos.cu:
// exact kNN of out-of-sample points Y [T, d] against the tree's points:
// tensor-core shortlist + canonical FP64 re-rank where the operands exist,
// else the tiled exhaustive search; ids / dist [T, kappa] as knn_exact_gpu
askit_status knn_oos(askit_tree t, const float *Y, int64_t T, int kappa, int32_t *ids, double *dist, cudaStream_t s);
