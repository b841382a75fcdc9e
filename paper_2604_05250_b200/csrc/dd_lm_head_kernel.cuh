// Language-model heads fused with the verification algorithm (Algorithm 1, verification phase:
// the verifier's distribution p_V(. | x^D) at every position goes straight into A(p_D, p_V, x^D)).
//
// logits[t, x] = sum_k hidden[t, k] * weight[x, k] is a [rows, K] x [K, V] product whose result,
// 253 KB per position at the LLaDA vocabulary, is only ever reduced: per row its maximum, the
// lowest index of the maximum and the softmax normaliser (Eq. 7), and in the KL mode the sums of
// Eq. 4-5 over the drafter's logits, which are a second product of the same shape.  The kernel
// therefore keeps the products in tensor memory and never stores a logit: a persistent CTA takes
// work items of 256 rows x N vocabulary entries, accumulates them with tcgen05 MMAs (accumulators
// of 128 rows, fp32) from operand tiles that a TMA producer streams through a ring of up to nine stages,
// and its epilogue warps turn every accumulator row into one partial (maximum, first index,
// sum 2^(l*log2e - M); KL: also the drafter's maximum, sum and the weighted logit differences) of
// the same form as the streaming kernel's chunk partials, stored in the same global table ("chunk"
// = vocabulary tile).  A second, small kernel behind it on the stream (lm_head_fold_kernel) folds
// every flagged row's partials in fp64 with the streaming kernel's fold and runs dd_verify's
// decision stage per sequence.
//
// Only flagged positions need logits.  Where that can pay, a first small kernel (lm_head_rows_kernel) lists the flagged
// rows and, where that leaves fewer 128-row tiles, copies their hidden states one after the other
// into scratch; the products then run over those.  How many there are is known on the device only:
// it picks the width N of the vocabulary tiles too (a tensor map per width travels with the launch).
// 16 sequences of 256 positions, 62 % of them flagged, K = 4096, V = 126464: 3024 us
// with every row multiplied, 1961 us so.
//
// More than 128 rows are multiplied by pairs of CTAs where that is faster (dd_lm_head_pair.cuh; the rule is dd_lm_head_verify's).
//
// Tensor memory (512 columns): TRUST/CONF, N <= 256: the verifier's two accumulators at columns 0
// and 256.  KL, N <= 128: the drafter's at 0 and 128, the verifier's at 256 and 384; a work item
// runs the k loop over the drafter's operands first, then over the verifier's.  An item with no more
// than 128 rows (the last row block, or the only one) uses one accumulator and leaves the other to
// the next such item: its products run while this one is reduced.
//
//   warps 0-3   epilogue of rows 0-127 of the item (thread = row = tensor-memory lane)
//   warps 4-7   epilogue of rows 128-255
//   warp  8     one thread feeds the ring: per 64-wide k-step the two 128-row tiles of the hidden
//               states and the N-row tile of the weights (2-D tensor maps, 128-byte swizzle, rows
//               past the end read as zero; no multicast)
//   warp  9     one thread issues the MMAs and commits them to the ring's and the accumulators'
//               barriers
// Included by dd_verify.cu.
#pragma once

#include <cuda.h>

#include <type_traits>

#include "dd_ptx.cuh"
#include "dd_verify_decide_block.cuh"

namespace ddlm {

using namespace ddptx;

constexpr int kThreads = 320;
constexpr int kEpilogueWarps = 8;
constexpr int kLoadWarp = 8, kMmaWarp = 9;
constexpr int kTileRows = 128;
constexpr int kRowsPerItem = 2 * kTileRows; // two accumulators
constexpr int kBlockK = 64;                // one 128-byte swizzled box per k-step
constexpr int kMaxStages = 9;
constexpr int kCheckedRows = 4 * kThreads;
constexpr int kMaxN = 256;
constexpr uint32_t kTmemCols = 512;        // see the layout above
constexpr int kATileBytes = kTileRows * kBlockK * 2;                  // 16 KB: 128 rows x 64 bf16
constexpr int kRingBytes = 3 * (2 * kATileBytes + kMaxN * kBlockK * 2);   // 192 KB: three stages of the largest kind
constexpr int kSmemBytes = kRingBytes + 1024 + 256;
constexpr unsigned kErrLmFull = 0xC00, kErrLmEmpty = 0xD00, kErrLmAcc = 0xE00;

// Widths of the vocabulary tiles: multiples of 32 downwards from the largest.  Below half of it only where that leaves SMs idle
// (dd_lm_head_verify).
template <bool KL>
struct Widths {
    static constexpr int max_n = KL ? kMaxN / 2 : kMaxN;
    static constexpr int count = max_n / 32;
};

// What the first kernel finds out, for those behind it.
struct LmPlan {
    int n_rows;                // rows to multiply: the flagged ones, or all of them where that costs no more
    int gathered;              // 1: their hidden states stand one after the other in the scratch
    int N;                     // vocabulary entries per work item
    int n_tiles;               // ceil(V / N): the "chunks" of a row
    int pairs;                 // 1: lm_head_pair_kernel multiplies, 0: lm_head_kernel
};

struct LmParams {
    int rows, K, V;            // rows = B * P
    int ctas;                  // CTAs the tile width is chosen for
    int pairs;                 // 0: the products are lm_head_kernel's, 2: lm_head_pair_kernel's, 1: of more than 128 rows
    int min_n;                 // the narrowest width the scratch has partials for
    int rows_per_block;        // rows that a block of the first kernel copies: a multiple of kRowsWarps
    LmPlan *plan;              // null: nothing is gathered, the plan is all_rows and the first kernel is not launched
    LmPlan all_rows;
    int *row_map;              // [rows]: the row that gathered row i is (not written where nothing is gathered)
};

// Tensor maps of one launch: hidden states (as passed, and as gathered) and weights (a map per width).
template <bool KL>
struct LmMaps {
    CUtensorMap h, h_gathered, w[Widths<KL>::count];
    CUtensorMap hd, hd_gathered, wd[KL ? Widths<KL>::count : 1];      // the drafter's, KL only
};

// Vocabulary entries per work item: the width for which the slowest of `ctas` CTAs finishes first.
// A work item of n entries takes about (fixed + n) units of time: the hidden-state tiles it loads and
// the MMAs' shared-memory reads of them do not shrink with n.  `pairs`: pairs of CTAs work on two tiles at a time
// (dd_lm_head_pair.cuh; any constant from 60 to 250 picks as well there).  Measured at K = 4096 (time per item
// against n, tile widths forced): fixed = 140 for one product per item, 157 for the KL mode's two.
// Counting n alone picked tiles of 128 entries at 4096 rows, 25 % slower than 256.
template <bool KL>
__host__ __device__ inline int pick_tile_n(int V, long n_rows, int ctas, int min_n, bool pairs)
{
    constexpr int fixed = KL ? 157 : 140;
    const long row_blocks = (n_rows + kRowsPerItem - 1) / kRowsPerItem;
    int best = Widths<KL>::max_n;
    long best_cost = -1;
    for (int i = 0; i < Widths<KL>::count; ++i) {
        const int n = Widths<KL>::max_n - 32 * i;
        if (n < min_n) break;
        const long tiles = (V + n - 1) / n;
        const long items = !pairs ? tiles * row_blocks
                         : KL ? (tiles + 1) / 2 * row_blocks
                              : tiles * (row_blocks / 2) + (row_blocks % 2 ? (tiles + 1) / 2 : 0);
        const long workers = pairs ? (ctas + 1) / 2 : ctas;
        const long cost = ((items + workers - 1) / workers) * (fixed + n);
        if (best_cost < 0 || cost < best_cost) { best_cost = cost; best = n; }
    }
    return best;
}

template <bool KL>
__host__ __device__ inline LmPlan plan_for(const LmParams &q, int n_rows, bool gathered)
{
    LmPlan plan;
    plan.n_rows = n_rows;
    plan.gathered = gathered;
    plan.pairs = q.pairs == 2 || (q.pairs == 1 && n_rows > kTileRows);
    plan.N = pick_tile_n<KL>(q.V, n_rows, q.ctas, q.min_n, plan.pairs != 0);
    plan.n_tiles = (q.V + plan.N - 1) / plan.N;
    return plan;
}

// First launch of dd_lm_head_verify, where gathering can pay.  Every block counts all flags and the flags before its
// own rows; the first one writes the plan.  Gathering pays where it leaves fewer 128-row tiles (at
// K = 4096, V = 126464 a tile of rows costs 85 us, copying 128 rows less than one), and with one or two tiles of the
// vocabulary, whose products are no more than reading the rows, where few are flagged: a gathered row is read twice
// and written once (105150 rows, 60 %, K = 320, V = 102: 131 us without, 169 with; 38520, 5 %, 3072, 242: 118 and 79).
// Elsewhere nothing is copied.  One warp per row; at most kRowsBlocks blocks, so that the counting stays linear in the rows.
constexpr int kRowsThreads = 256;
constexpr int kRowsWarps = kRowsThreads / 32;
constexpr int kRowsBlocks = 1024;
template <bool KL>
__global__ void __launch_bounds__(kRowsThreads)
lm_head_rows_kernel(const LmParams q, const ddv::VerifyParams p, const uint4 *hidden, uint4 *gathered,
                    const uint4 *hidden_d, uint4 *gathered_d)
{
    grid_trigger();
    grid_wait();
    const uint8_t *flags = p.flags;
    __shared__ int s_before, s_all;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int first = blockIdx.x * q.rows_per_block;
    if (tid == 0) s_before = s_all = 0;
    __syncthreads();
    int before = 0, all = 0;
    auto count = [&](int i, int n) { all += n; before += i < first ? n : 0; };
    int done = 0;
    if ((reinterpret_cast<uintptr_t>(flags) & 7) == 0) {           // eight flags at a time (first is a multiple of eight)
        done = q.rows & ~7;
#pragma unroll 4
        for (int i = 8 * tid; i < done; i += 8 * kRowsThreads) {
            const uint2 w = *reinterpret_cast<const uint2 *>(flags + i);
            count(i, __popc(__vsetne4(w.x, 0u)) + __popc(__vsetne4(w.y, 0u)));
        }
    }
    for (int i = done + tid; i < q.rows; i += kRowsThreads) count(i, flags[i] != 0);
    before = __reduce_add_sync(0xFFFFFFFFu, before);
    all = __reduce_add_sync(0xFFFFFFFFu, all);
    if (lane == 0) { atomicAdd(&s_before, before); atomicAdd(&s_all, all); }
    __syncthreads();
    all = s_all;
    const int unit = q.pairs == 2 || (q.pairs == 1 && all > kTileRows) ? kRowsPerItem : kTileRows;           // rows that cost as much as one
    const bool gather = (all + unit - 1) / unit < (q.rows + unit - 1) / unit &&
                        (q.all_rows.n_tiles > 2 || 3L * all < (long)q.rows * q.all_rows.n_tiles);
    if (blockIdx.x == 0 && tid == 0) *q.plan = plan_for<KL>(q, gather ? all : q.rows, gather);
    if (!gather) return;
    const int vecs = q.K / 8;                                      // 16-byte vectors per row
    int seen = s_before;                                           // flags before the warps' next rows
    for (int row0 = first; row0 < min(first + q.rows_per_block, q.rows); row0 += kRowsWarps) {
        const bool flagged = lane < kRowsWarps && row0 + lane < q.rows && flags[row0 + lane] != 0;
        const unsigned mask = __ballot_sync(0xFFFFFFFFu, flagged);
        const int at = seen + __popc(mask & ((1u << warp) - 1u));
        seen += __popc(mask);
        if (!(mask >> warp & 1u)) continue;
        const int row = row0 + warp;
        if (lane == 0) q.row_map[ddv::checked(p, at, q.rows, ddv::kSiteRow)] = row;
        auto copy = [&](uint4 *dst, const uint4 *src) {
            dst += ddv::checked_run(p, (long)at * vecs, vecs, (long)q.rows * vecs, ddv::kSiteHidden);
            src += ddv::checked_run(p, (long)row * vecs, vecs, (long)q.rows * vecs, ddv::kSiteHidden);
#pragma unroll 8
            for (int i = lane; i < vecs; i += 32) dst[i] = src[i];
        };
        copy(gathered, hidden);
        if (KL) copy(gathered_d, hidden_d);
    }
}

// One row's partial of one vocabulary tile into the global table.  Nothing else happens in this
// kernel: rows are folded and sequences decided by lm_head_fold_kernel, launched behind it on the
// same stream.  (Folding in here, by whichever warp stores a row's last tile, put every fold of the
// launch on the one CTA that finishes last: all rows of a row block complete together, with the
// last tile.  170 of 217 us on a 256-row, 143-tile problem were that CTA folding alone.)
__device__ __forceinline__ void store_partial(const ddv::VerifyParams &p, const ddv::Partial &c, int row, int tile, int n_tiles)
{
    ddv::Partial *dst = p.partials + ddv::checked(p, (long)row * n_tiles + tile, (long)p.B * p.P * n_tiles, ddv::kSitePartial);
    __stcg(reinterpret_cast<float4 *>(dst), make_float4(c.m_v, c.s_v, __int_as_float(c.idx), c.m_d));
    __stcg(reinterpret_cast<float4 *>(dst) + 1, make_float4(c.s_d, c.t, 0.f, 0.f));
}

// Last launch of dd_lm_head_verify: one warp per row folds the row's tile partials (fp64, tile order: the
// streaming kernel's fold) and stores score and argmax; the CTA counts its rows in their sequences and decides
// those it completes with all its threads (a warp per deciding sequence took 12-16 us from a cold
// instruction cache: 16 rows of 126464 entries 204 -> 194 us, 8 x 512 of 8000 41.5 -> 39.8).  The partials were written by the previous kernel on the stream.
constexpr int kFoldThreads = 256;
template <bool KL>
__global__ void __launch_bounds__(kFoldThreads) lm_head_fold_kernel(const __grid_constant__ ddv::VerifyParams p, const LmParams q)
{
    grid_trigger();
    grid_wait();
    const int rows = q.rows;
    __shared__ ddv::BlockReport s_report;
    const int row0 = blockIdx.x * (kFoldThreads / 32);
    const int w = row0 + (threadIdx.x >> 5);
    if (w < rows && p.flags[w]) {
        float score;
        int argmax;
        const int n_tiles = q.plan ? q.plan->n_tiles : q.all_rows.n_tiles;
        ddv::fold_partials<KL, true>(p.partials + ddv::checked_run(p, (long)w * n_tiles, n_tiles, (long)rows * n_tiles, ddv::kSitePartial),
                               n_tiles, score, argmax);
        if ((threadIdx.x & 31) == 0) {
            const size_t row_at = ddv::checked(p, w, (long)p.B * p.P, ddv::kSiteRow);
            __stcg(p.row_score + row_at, score);
            __stcg(p.row_argmax + row_at, argmax);
        }
    }
    ddv::report_rows(p, row0, kFoldThreads / 32, s_report);
}

// The work items of a CTA, in order: every role walks the same way.  Items that follow each other share a
// vocabulary tile (weights from L2).
struct Walk {
    int item, n_items, row_blocks, n_rows;
    int tile, row0;
    bool two;              // the item has more than 128 rows: both accumulators
    int one;               // else: the accumulator it uses (such items take turns)
    __device__ __forceinline__ Walk(const LmPlan &plan)
    {
        n_rows = plan.n_rows;
        row_blocks = (n_rows + kRowsPerItem - 1) / kRowsPerItem;
        n_items = plan.n_tiles * row_blocks;
        item = blockIdx.x;
        one = 1;
        set();
    }
    __device__ __forceinline__ void set()
    {
        if (item >= n_items) return;
        tile = item / row_blocks;
        row0 = (item - tile * row_blocks) * kRowsPerItem;
        two = n_rows - row0 > kTileRows;
        if (!two) one ^= 1;
    }
    __device__ __forceinline__ bool valid() const { return item < n_items; }
    __device__ __forceinline__ void next() { item += gridDim.x; set(); }
    __device__ __forceinline__ bool uses(int acc) const { return two || one == acc; }
};

// One row of a tile of N entries: its columns of the accumulators (dacc: the drafter's, KL only) become a partial: the
// verifier's maximum m_v, its lowest index and s_v = sum 2^(l*log2e - M); KL (Eq. 4-5): also the drafter's maximum m_d, s_d = sum
// 2^(d*log2e - M_d) and t = sum 2^(d*log2e - M_d) * (d - v).
// The columns are read twice, for the maxima and for the sums.  Nothing else of the CTA hides this, so what counts is the length of the chains (as one
// pass with a running maximum and its index it was 32 dependent steps per 32 columns) and the size of the code, which is
// cold every time: two short loops, four chains for every sum.  256 columns, eight warps 7400 -> 6200 cycles (8960 -> 6420 the
// first time; one pass with four chains 5900 and 7300), KL 128 columns 7200 -> 5800; 8192 rows, K = 512, V = 2000 38.7 -> 36.5 us,
// KL 62.0 -> 58.8; 1024, 2048, 50000 172 -> 164.
template <bool KL>
__device__ __forceinline__ ddv::Partial reduce_columns(uint32_t tacc, uint32_t dacc, int N, int col0, int V)
{
    const int columns = min(N, V - col0);                        // that exist
    float m = -INFINITY, m_d = -INFINITY;
    uint32_t r[32], rd[32];                                      // rd: the drafter's logits, KL only
    auto load = [&](int cb) {
        tmem_ld32(tacc + cb, r);
        if constexpr (KL) tmem_ld32(dacc + cb, rd);
        tmem_wait_ld(r);
        if constexpr (KL) tmem_wait_ld(rd);
    };
    auto top = [&](const uint32_t (&x)[32], float m) {
        float c[4] = {m, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
        for (int i = 0; i < 32; i += 2) c[i / 2 % 4] = max3(c[i / 2 % 4], __uint_as_float(x[i]), __uint_as_float(x[i + 1]));
        return max3(c[0], c[1], fmaxf(c[2], c[3]));
    };
    // 32 columns of which `valid` exist: the others are out of every maximum and sum
    auto clip = [&](uint32_t (&x)[32], int valid, uint32_t with) {
#pragma unroll
        for (int i = 0; i < 32; ++i) x[i] = i < valid ? x[i] : with;
    };
    constexpr uint32_t kMinusInf = 0xFF800000u;
#pragma unroll 1
    for (int cb = 0; cb < columns; cb += 32) {
        load(cb);
        if (columns - cb < 32) { clip(r, columns - cb, kMinusInf); if constexpr (KL) clip(rd, columns - cb, kMinusInf); }
        m = top(r, m);
        if constexpr (KL) m_d = top(rd, m_d);
    }
    const float M = m * ddv::kLog2e, M_d = m_d * ddv::kLog2e;
    float s[4] = {0.f, 0.f, 0.f, 0.f}, s_d[4] = {0.f, 0.f, 0.f, 0.f}, t[4] = {0.f, 0.f, 0.f, 0.f};
    int idx = 0x7FFFFFFF;
#pragma unroll 1
    for (int cb = 0; cb < columns; cb += 32) {
        load(cb);
        int at[4] = {32, 32, 32, 32};
        auto sums = [&](auto is_masked) {
            const int valid = columns - cb;
#pragma unroll
            for (int i = 31; i >= 0; --i) {
                if (decltype(is_masked)::value && i >= valid) continue;
                const float v = __uint_as_float(r[i]);
                if (v == m) at[i / 8] = i;
                s[i % 4] += ex2(fmaf(v, ddv::kLog2e, -M));
                if constexpr (KL) {
                    const float d = __uint_as_float(rd[i]), e = ex2(fmaf(d, ddv::kLog2e, -M_d));
                    s_d[i % 4] += e;
                    t[i % 4] = fmaf(e, d - v, t[i % 4]);
                }
            }
        };
        if (columns - cb >= 32) sums(std::false_type());
        else sums(std::true_type());
        const int first = min(min(at[0], at[1]), min(at[2], at[3]));
        if (first < 32) idx = min(idx, col0 + cb + first);
    }
    ddv::Partial c;
    c.m_v = m;
    c.s_v = (s[0] + s[1]) + (s[2] + s[3]);
    c.idx = m == -INFINITY ? 0x7FFFFFFF : idx;               // nothing above -inf: no token
    c.m_d = KL ? m_d : 0.f;
    c.s_d = (s_d[0] + s_d[1]) + (s_d[2] + s_d[3]);
    c.t = (t[0] + t[1]) + (t[2] + t[3]);
    c.pad0 = c.pad1 = 0.f;
    return c;
}

// Epilogue warps: every accumulator row becomes one partial; KL: the drafter's accumulator is read beside the verifier's.
template <bool KL>
__device__ __forceinline__ void epilogue(const LmParams &q, const LmPlan &plan, const ddv::VerifyParams &p, uint32_t tmem,
                                         uint32_t bars_acc_full, uint32_t bars_acc_empty, volatile uint32_t *abort_flag)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int acc = warp >> 2;
    const uint32_t lane_off = (uint32_t)((warp & 3) * 32) << 16;          // this warp's 32 tensor-memory lanes
    const uint32_t tacc = tmem + lane_off + (KL ? 256u + (uint32_t)acc * 128u : (uint32_t)acc * 256u);   // verifier
    const uint32_t dacc = tmem + lane_off + (uint32_t)acc * 128u;                                          // drafter (KL)
    Walk walk(plan);
    for (uint32_t n_done = 0; walk.valid(); walk.next()) {
        if (!walk.uses(acc)) continue;
        const int tile = walk.tile, col0 = tile * plan.N;
        int row = walk.row0 + (walk.two ? acc * kTileRows : 0) + (warp & 3) * 32 + lane;
        // the row of the caller's tensors, or -1: nothing to store
        if (row >= plan.n_rows) row = -1;
        else if (plan.gathered) row = q.row_map[ddv::checked(p, row, q.rows, ddv::kSiteRow)];
        else if (!p.flags[row]) row = -1;
        bool arrived = false;
#pragma unroll 1
        for (uint32_t it = 0; it < (1u << 22); ++it) {
            if (mbar_try_wait(bars_acc_full + 8u * acc, n_done & 1)) { arrived = true; break; }
            if (it > 64) {
                __nanosleep(64);
                if (*abort_flag) break;
            }
        }
        ++n_done;
        if (!arrived) {
            if (lane == 0) {
                *abort_flag = 1u;
                ddv::report_expired(p, kErrLmAcc);
            }
            return;
        }
        tc_fence_after();
        const ddv::Partial c = reduce_columns<KL>(tacc, dacc, plan.N, col0, q.V);
        // the accumulator may be overwritten once its four epilogue warps have read their lanes
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bars_acc_empty + 8u * acc);
        if (row >= 0) store_partial(p, c, row, tile, plan.n_tiles);
    }
}

// KL: every work item runs the k loop twice, first over the drafter's hidden states and weights
// into accumulators [0,N) and [128,128+N), then over the verifier's into [256,..) and [384,..)
// (N <= 128); the epilogue reads both.  Otherwise only the verifier's maps are used and the
// accumulators are [0,N) and [256,256+N) (N <= 256).
template <bool KL>
__global__ void __launch_bounds__(kThreads, 1)
lm_head_kernel(const __grid_constant__ LmMaps<KL> maps, const LmParams q, const ddv::VerifyParams p)
{
    // the rows' kernel may have left the products to lm_head_pair_kernel
    if (q.pairs == 1) {
        grid_wait();
        if (q.plan->pairs) return;
    }
    extern __shared__ __align__(1024) unsigned char smem_dyn[];
    const uint32_t smem_base = (smem_u32(smem_dyn) + 1023u) & ~1023u;     // swizzled tiles: 1024-byte aligned
    unsigned char *smem_gen = smem_dyn + (smem_base - smem_u32(smem_dyn));
    const uint32_t bars = smem_base + kRingBytes;
    auto bar_full = [&](int s) { return bars + 8u * s; };
    auto bar_empty = [&](int s) { return bars + 8u * (kMaxStages + s); };
    const uint32_t bars_acc_full = bars + 8u * (2 * kMaxStages), bars_acc_empty = bars_acc_full + 16u;
    const uint32_t tmem_slot = bars_acc_empty + 16u;
    volatile uint32_t *tmem_slot_gen = reinterpret_cast<volatile uint32_t *>(smem_gen + (tmem_slot - smem_base));
    volatile uint32_t *abort_flag = tmem_slot_gen + 1;

    const int tid = threadIdx.x, warp = warp_uniform(tid >> 5);
    if (tid == 0) {
        for (int s = 0; s < kMaxStages; ++s) { mbar_init(bar_full(s), 1); mbar_init(bar_empty(s), 1); }
        for (int a = 0; a < 2; ++a) {
            mbar_init(bars_acc_full + 8u * a, 1);
            mbar_init(bars_acc_empty + 8u * a, kEpilogueWarps / 2);
        }
        fence_mbar_init();
        *abort_flag = 0u;
    }
    if (warp == 0) { tmem_alloc(tmem_slot, kTmemCols); tmem_relinquish(); }
    grid_wait();                                              // what follows reads what the kernels before left
    LmPlan plan = q.plan ? *q.plan : q.all_rows;
    // few rows, none listed: perhaps none of them is flagged, and there is nothing to multiply
    int any = 1;
    if (!q.plan && q.rows <= kCheckedRows) {
        any = 0;
        for (int i = tid; i < q.rows; i += kThreads) any |= p.flags[i];
    }
    const int k_steps = q.K / kBlockK;
    // a stage: one or two tiles of hidden states (two unless no item has more than 128 rows), one of weights
    const uint32_t a_bytes = plan.n_rows > kTileRows ? 2 * kATileBytes : kATileBytes;
    const uint32_t b_bytes = (uint32_t)plan.N * kBlockK * 2;
    const uint32_t stage_bytes = a_bytes + b_bytes;
    const uint32_t stages = min((uint32_t)kMaxStages, kRingBytes / stage_bytes);

    tc_fence_before();
    if (!__syncthreads_or(any)) plan.n_rows = 0;
    tc_fence_after();
    const uint32_t tmem = warp_uniform(*tmem_slot_gen);

    // a wait that gives up: the code goes to the health word, every role winds down
    auto give_up = [&](unsigned code) {
        *abort_flag = 1u;
        ddv::report_expired(p, code);
    };
    auto wait = [&](uint32_t bar, uint32_t parity) {
#pragma unroll 1
        for (uint32_t it = 0; it < (1u << 22); ++it) {
            if (mbar_try_wait(bar, parity)) return true;
            if (it > 64) {
                __nanosleep(32);
                if (*abort_flag) return false;
            }
        }
        return false;
    };

    if (warp == kLoadWarp && elect_one()) {
        // ===================================================================== TMA producer
        const int width = (Widths<KL>::max_n - plan.N) / 32;
        const CUtensorMap *h = plan.gathered ? &maps.h_gathered : &maps.h, *w = &maps.w[width];
        const CUtensorMap *hd = plan.gathered ? &maps.hd_gathered : &maps.hd, *wd = &maps.wd[KL ? width : 0];
        prefetch_tmap(h); prefetch_tmap(w);
        if (KL) { prefetch_tmap(hd); prefetch_tmap(wd); }
        uint32_t s = 0, round = 0;                            // stage, and how often the ring has been gone round
        bool ok = true;
        for (Walk walk(plan); walk.valid() && ok; walk.next()) {
            const int col0 = walk.tile * plan.N;
            const uint32_t bytes = (walk.two ? 2 * kATileBytes : kATileBytes) + b_bytes;
            for (int ks2 = 0; ks2 < (KL ? 2 : 1) * k_steps; ++ks2) {
                if (round > 0 && !wait(bar_empty(s), (round - 1) & 1)) { give_up(kErrLmEmpty); ok = false; break; }
                const uint32_t dst = smem_base + s * stage_bytes;
                const bool drafter = KL && ks2 < k_steps;                 // the drafter's pass comes first
                const int ks = ks2 < k_steps ? ks2 : ks2 - k_steps;
                const CUtensorMap *mh = drafter ? hd : h, *mw = drafter ? wd : w;
                mbar_expect_tx(bar_full(s), bytes);
                tma_load_2d(dst, mh, bar_full(s), ks * kBlockK, walk.row0);
                if (walk.two) tma_load_2d(dst + kATileBytes, mh, bar_full(s), ks * kBlockK, walk.row0 + kTileRows);
                tma_load_2d(dst + a_bytes, mw, bar_full(s), ks * kBlockK, col0);
                if (++s == stages) { s = 0; ++round; }
            }
        }
        grid_trigger();
    } else if (warp == kMmaWarp && elect_one()) {
        // ===================================================================== MMA issuer
        const uint32_t idesc = idesc_bf16(128, plan.N, false);
        uint32_t s = 0, round = 0;
        uint32_t uses[2] = {0, 0};                            // items each accumulator has taken part in
        bool ok = true;
        for (Walk walk(plan); walk.valid() && ok; walk.next()) {
            // the epilogue of the accumulators' previous item has read them
            for (int a = 0; a < 2 && ok; ++a) {
                if (!walk.uses(a)) continue;
                if (uses[a] > 0 && !wait(bars_acc_empty + 8u * a, (uses[a] - 1) & 1)) { give_up(kErrLmAcc); ok = false; }
                ++uses[a];
            }
            if (!ok) break;
            tc_fence_after();
            for (int ks2 = 0; ks2 < (KL ? 2 : 1) * k_steps; ++ks2) {
                if (!wait(bar_full(s), round & 1)) { give_up(kErrLmFull); ok = false; break; }
                tc_fence_after();
                const int ks = ks2 < k_steps ? ks2 : ks2 - k_steps;
                // accumulator columns of this pass: see the layout above
                const uint32_t half = (KL && ks2 >= k_steps) ? 256u : 0u, other = KL ? 128u : 256u;
                const uint32_t acc0 = tmem + half + (!walk.two && walk.one ? other : 0u), acc1 = tmem + half + other;
                const uint32_t base = smem_base + s * stage_bytes;
                const uint64_t a0 = smem_desc_sw128(base, 16, 1024), a1 = smem_desc_sw128(base + kATileBytes, 16, 1024);
                const uint64_t b = smem_desc_sw128(base + a_bytes, 16, 1024);
#pragma unroll
                for (int kk = 0; kk < kBlockK / 16; ++kk) {
                    const uint32_t off = (uint32_t)(kk * 32) >> 4;            // 16 bf16 = 32 bytes per MMA
                    mma_ss(acc0, a0 + off, b + off, idesc, (ks > 0 || kk > 0));
                    if (walk.two) mma_ss(acc1, a1 + off, b + off, idesc, (ks > 0 || kk > 0));
                }
                mma_commit(bar_empty(s));                                      // the stage is free once these have run
                if (++s == stages) { s = 0; ++round; }
            }
            if (!ok) break;
            for (int a = 0; a < 2; ++a)
                if (walk.uses(a)) mma_commit(bars_acc_full + 8u * a);
        }
    } else if (warp < kEpilogueWarps) {
        epilogue<KL>(q, plan, p, tmem, bars_acc_full, bars_acc_empty, abort_flag);
    }

    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (*abort_flag) {
        // a wait expired: give copies that may still be in flight time to land before the shared
        // memory is released
#pragma unroll 1
        for (int i = 0; i < 2000; ++i) __nanosleep(1000);
    }
    if (warp == 0) { __syncwarp(); tmem_dealloc(tmem, kTmemCols); }
}

}  // namespace ddlm
