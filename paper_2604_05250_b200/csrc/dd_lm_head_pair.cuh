// The products of dd_lm_head_verify by pairs of CTAs (tcgen05 cta_group::2), for more than 128 rows, in the KL mode (Eq. 4-5 from
// both models' hidden states: two products per vocabulary tile) and in the others where dd_lm_head_verify says so, or the kernel that lists the
// flagged rows (LmParams::pairs).
//
// What bounds lm_head_kernel is neither the tensor core nor memory but the operands' way from L2 into the SMs, some 45 bytes
// per clock and SM (10-11 TB/s over the chip): 64 KB a k-step for 256 x 256 x 64 products, 48 KB for 256 x 128 x 64 in the KL
// mode, where each model's product needs accumulators of its own.  The tensor cores of a pair read both CTAs' halves of the
// weights, so that each CTA holds twice the accumulators per byte: KL, 256 rows x 2 N entries, 128 rows and N (up to 128) entries in each CTA, 32 KB a
// k-step for twice the products; else 512 rows x N (up to 256) entries or, of a last or only block of up to 256 rows, 256 rows x 2 N, 48 KB for twice the products.
// Then the tensor core is at work in 84-90 % of the cycles (KL, 256 x 4096 x 126464: 459 of 509 thousand) and the clock is
// what power allows, 1.0-1.2 GHz.
//
// KL: a work item runs the k loop over the drafter's operands into accumulator columns [0, 2N), then over the verifier's
// into [256, 256 + 2N); the same ring of stages feeds both.  The epilogue reads both: in each CTA warps 0-3 take the
// first N columns of its 128 rows, warps 4-7 the other N.  To the fold, that is two vocabulary tiles of N entries.
// Else: two products per k-step, with the other rows or the other tile, into columns [0, N) and [256, 256 + N); warps 0-3
// reduce the one, 4-7 the other.
//
//   warps 0-7   epilogue
//   warp  8     one thread in each CTA loads this CTA's operands; all copies complete on the leading CTA's barrier
//   warp  9     one thread in the leading CTA issues the MMAs and commits them to the barriers of both
//
// us, lm_head_kernel : this one (rows, K, V), KL: 256, 4096, 126464 514 : 461 (under the power cap 585 : 504); 512, 3072, 10000
// 95.6 : 74.3; 150, 4096, 50000 239 : 202; 400, 2048, 30000 151 : 135; 200, 1024, 20000 45.9 : 41.2; 635 of 1024, 4096,
// 126464 1270 : 1167; 8192, 512, 2000 61.6 : 61.0.  Up to 128 rows the second CTA's rows are all padding, and
// lm_head_kernel's items of 128 rows are quicker: 128, 4096, 126464 390 : 422; 40 380 : 434.  The other modes: at dd_lm_head_verify's rule.
// Tried: the next 1 to 4 KB of each row of weights prefetched into L2 by the loading thread, 566 to 900 us at 256 rows, KL (the thread does not
// keep up, and copies of 128 bytes a row already read memory at 5.6 TB/s in lm_head_kernel).
// Every wait is bounded and reports to the verify health word.  Included by dd_verify.cu, after dd_lm_head_kernel.cuh.
#pragma once

namespace ddlm {

constexpr int kPairBars = 2 * kMaxStages + 2;

// The work items of a pair, in order: every role walks the same way.  The items of two vocabulary tiles follow each other,
// so that all row blocks take the weights from L2.
template <bool KL>
struct PairWalk {
    int item, n_items, step, n_tiles;
    int blocks, per_group;     // row blocks of the full kind, items per two tiles
    int tile, row0;            // the item's first tile and row
    bool wide;                 // KL: all; else: two tiles of one block of up to 256 rows (not: one tile of a block of up to 512)
    __device__ __forceinline__ explicit PairWalk(const LmPlan &plan)
    {
        n_tiles = plan.n_tiles;
        blocks = KL ? (plan.n_rows + kRowsPerItem - 1) / kRowsPerItem : (plan.n_rows + kRowsPerItem - 1) / (2 * kRowsPerItem);
        const int rest = !KL && plan.n_rows > blocks * 2 * kRowsPerItem;
        per_group = KL ? blocks : 2 * blocks + rest;
        // (KL: an item with the last of an odd number of tiles has one to reduce; else the last tile alone has an item per block)
        n_items = KL ? (n_tiles + 1) / 2 * blocks : n_tiles / 2 * per_group + (n_tiles & 1) * (blocks + rest);
        item = (int)blockIdx.x >> 1;
        step = (int)gridDim.x >> 1;
        set();
    }
    __device__ __forceinline__ void set()
    {
        const int group = item / max(per_group, 1), k = item - group * per_group;
        const int tiles = KL ? 2 : min(2, n_tiles - 2 * group);        // in this group
        wide = KL || k == tiles * blocks;
        tile = 2 * group + (!wide && k >= blocks);
        row0 = (wide && !KL ? blocks : k >= blocks ? k - blocks : k) * (KL ? 1 : 2) * kRowsPerItem;
    }
    __device__ __forceinline__ bool valid() const { return item < n_items; }
    __device__ __forceinline__ void next() { item += step; set(); }
};

template <bool KL>
__global__ void __launch_bounds__(kThreads, 1)
lm_head_pair_kernel(const __grid_constant__ LmMaps<KL> maps, const LmParams q, const ddv::VerifyParams p)
{
    // ... or to lm_head_kernel (the same answer in both CTAs)
    if (q.pairs == 1) {
        grid_wait();
        if (!q.plan->pairs) return;
    }
    extern __shared__ __align__(1024) unsigned char smem_dyn[];
    const uint32_t smem_base = (smem_u32(smem_dyn) + 1023u) & ~1023u;     // the same in both CTAs
    unsigned char *smem_gen = smem_dyn + (smem_base - smem_u32(smem_dyn));
    const uint32_t bars = smem_base + kRingBytes;
    auto bar_full = [&](int s) { return bars + 8u * s; };                 // the leading CTA's counts both CTAs' copies
    auto bar_empty = [&](int s) { return bars + 8u * (kMaxStages + s); };
    const uint32_t bar_acc_full = bars + 8u * (2 * kMaxStages), bar_acc_empty = bar_acc_full + 8u;
    const uint32_t tmem_slot = bars + 8u * kPairBars;
    volatile uint32_t *tmem_slot_gen = reinterpret_cast<volatile uint32_t *>(smem_gen + (tmem_slot - smem_base));
    volatile uint32_t *abort_flag = tmem_slot_gen + 1;

    const int tid = threadIdx.x, warp = warp_uniform(tid >> 5), lane = tid & 31;
    const int rank = blockIdx.x & 1;
    if (tid == 0) {
        for (int s = 0; s < kMaxStages; ++s) { mbar_init(bar_full(s), 1); mbar_init(bar_empty(s), 1); }
        mbar_init(bar_acc_full, 1);
        mbar_init(bar_acc_empty, 2 * kEpilogueWarps);
        fence_mbar_init();
        *abort_flag = 0u;
    }
    if (warp == 0) { __syncwarp(); tmem_alloc_pair(tmem_slot, kTmemCols); tmem_relinquish_pair(); }
    grid_wait();                                              // what follows reads what the kernels before left
    LmPlan plan = q.plan ? *q.plan : q.all_rows;
    // few rows, none listed: perhaps none of them is flagged, and there is nothing to multiply
    int any = 1;
    if (!q.plan && q.rows <= kCheckedRows) {
        any = 0;
        for (int i = tid; i < q.rows; i += kThreads) any |= p.flags[i];
    }
    const int k_steps = q.K / kBlockK;
    // a stage of one CTA: KL: 128 rows and N entries; else 256 rows and N / 2 entries, or 128 rows and twice N / 2
    const uint32_t b_bytes = (uint32_t)(KL ? plan.N : plan.N / 2) * kBlockK * 2;
    const uint32_t stage_bytes = KL ? kATileBytes + b_bytes : max(2 * kATileBytes + b_bytes, kATileBytes + 2 * b_bytes);
    const uint32_t stages = min((uint32_t)kMaxStages, kRingBytes / stage_bytes);

    tc_fence_before();
    if (!__syncthreads_or(any)) plan.n_rows = 0;
    __syncwarp();
    cluster_arrive();              // the other CTA's barriers are set up before anything completes on them
    cluster_wait();
    tc_fence_after();
    const uint32_t tmem = warp_uniform(*tmem_slot_gen);

    // a wait that gives up: the code goes to the health word, every role of both CTAs winds down
    auto give_up = [&](unsigned code) {
        *abort_flag = 1u;
        st_cluster(cluster_addr(tmem_slot + 4u, rank ^ 1), 1u);
        ddv::report_expired(p, code);
    };
    auto wait = [&](uint32_t bar, uint32_t parity) {
#pragma unroll 1
        for (uint32_t it = 0; it < (1u << 22); ++it) {
            if (mbar_try_wait_cluster(bar, parity)) return true;
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
        for (PairWalk<KL> walk(plan); walk.valid() && ok; walk.next()) {
            const int row0 = walk.row0 + rank * kTileRows;
            const int col0 = KL ? (walk.tile + rank) * plan.N : walk.tile * plan.N + rank * (plan.N / 2);
            const uint32_t bytes = KL ? kATileBytes + b_bytes : walk.wide ? kATileBytes + 2 * b_bytes : 2 * kATileBytes + b_bytes;
            for (int ks2 = 0; ks2 < (KL ? 2 : 1) * k_steps; ++ks2) {
                if (round > 0 && !wait(bar_empty(s), (round - 1) & 1)) { give_up(kErrLmEmpty); ok = false; break; }
                const uint32_t dst = smem_base + s * stage_bytes, bar = cluster_addr(bar_full(s), 0);
                const bool drafter = KL && ks2 < k_steps;                 // the drafter's pass comes first
                const int x = (!KL || drafter ? ks2 : ks2 - k_steps) * kBlockK;
                if (rank == 0) mbar_expect_tx(bar_full(s), 2 * bytes);
                tma_load_2d_pair(dst, drafter ? hd : h, bar, x, row0);
                if (!KL && !walk.wide) tma_load_2d_pair(dst + kATileBytes, h, bar, x, row0 + kRowsPerItem);
                const uint32_t b = dst + (KL || walk.wide ? kATileBytes : 2 * kATileBytes);
                tma_load_2d_pair(b, drafter ? wd : w, bar, x, col0);
                if (!KL && walk.wide) tma_load_2d_pair(b + b_bytes, w, bar, x, col0 + plan.N);
                if (++s == stages) { s = 0; ++round; }
            }
        }
        grid_trigger();
    } else if (warp == kMmaWarp && rank == 0 && elect_one()) {
        // ===================================================================== MMA issuer
        const uint32_t idesc = idesc_bf16(256, KL ? 2 * plan.N : plan.N, false);
        uint32_t s = 0, round = 0, n = 0;
        bool ok = true;
        for (PairWalk<KL> walk(plan); walk.valid() && ok; walk.next(), ++n) {
            // both CTAs' epilogues have read the previous item's accumulators
            if (n > 0 && !wait(bar_acc_empty, (n - 1) & 1)) { give_up(kErrLmAcc); break; }
            tc_fence_after();
            for (int ks2 = 0; ks2 < (KL ? 2 : 1) * k_steps; ++ks2) {
                if (!wait(bar_full(s), round & 1)) { give_up(kErrLmFull); ok = false; break; }
                tc_fence_after();
                const uint32_t base = smem_base + s * stage_bytes;
                const uint64_t a = smem_desc_sw128(base, 16, 1024);
                const uint64_t b = smem_desc_sw128(base + (KL || walk.wide ? kATileBytes : 2 * kATileBytes), 16, 1024);
                // the second product's operands: the other rows, or the other tile
                const uint64_t a1 = a + (!KL && !walk.wide ? kATileBytes >> 4 : 0), b1 = b + (!KL && walk.wide ? b_bytes >> 4 : 0);
                const uint32_t acc = tmem + (KL && ks2 >= k_steps ? 256u : 0u);
#pragma unroll
                for (int kk = 0; kk < kBlockK / 16; ++kk) {
                    const uint32_t off = (uint32_t)(kk * 32) >> 4;            // 16 bf16 = 32 bytes per MMA
                    const bool more = kk > 0 || (ks2 != 0 && (!KL || ks2 != k_steps));
                    mma_ss_pair(acc, a + off, b + off, idesc, more);
                    if (!KL) mma_ss_pair(acc + 256u, a1 + off, b1 + off, idesc, more);
                }
                mma_commit_pair(bar_empty(s));                                 // the stage is free in both CTAs once these have run
                if (++s == stages) { s = 0; ++round; }
            }
            if (ok) mma_commit_pair(bar_acc_full);
        }
    } else if (warp < kEpilogueWarps) {
        // ===================================================================== epilogue
        const int half = warp >> 2;
        const uint32_t lane_off = (uint32_t)((warp & 3) * 32) << 16;          // this warp's 32 tensor-memory lanes
        const uint32_t dacc = tmem + lane_off + (uint32_t)(half * plan.N), tacc = KL ? dacc + 256u : tmem + lane_off + half * 256u;
        const uint32_t acc_empty = cluster_addr(bar_acc_empty, 0);
        uint32_t n = 0;
        for (PairWalk<KL> walk(plan); walk.valid(); walk.next(), ++n) {
            const int tile = walk.tile + (walk.wide ? half : 0);
            int row = walk.row0 + (walk.wide ? 0 : half * kRowsPerItem) + rank * kTileRows + (warp & 3) * 32 + lane;
            // the row of the caller's tensors, or -1: nothing to store
            if (row >= plan.n_rows || tile >= plan.n_tiles) row = -1;
            else if (plan.gathered) row = q.row_map[ddv::checked(p, row, q.rows, ddv::kSiteRow)];
            else if (!p.flags[row]) row = -1;
            if (!wait(bar_acc_full, n & 1)) {
                if (lane == 0) give_up(kErrLmAcc);
                break;
            }
            tc_fence_after();
            const ddv::Partial c = reduce_columns<KL>(tacc, dacc, plan.N, tile * plan.N, q.V);
            // the accumulators may be overwritten once all epilogue warps of the pair have read them
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(acc_empty);
            if (row >= 0) store_partial(p, c, row, tile, plan.n_tiles);
        }
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
    // no CTA leaves, or gives its tensor memory back, while the other may still use it
    __syncwarp();
    cluster_arrive();
    cluster_wait();
    if (warp == 0) { __syncwarp(); tmem_dealloc_pair(tmem, kTmemCols); }
}

}  // namespace ddlm
