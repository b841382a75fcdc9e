// The KL mode of dd_lm_head_verify (Eq. 4-5 from both models' hidden states) for more than 128 rows: two products per
// vocabulary tile, by pairs of CTAs (tcgen05 cta_group::2).
//
// What bounded lm_head_kernel here was neither the tensor core nor memory but the operands' way from L2 into the SMs: 48 KB a
// k-step for 256 x 128 x 64 products, at some 45 bytes per clock and SM (10-11 TB/s over the chip).  It has no larger items,
// since each model's product needs its own accumulators.  A pair computes 256 rows x 2 N entries: each CTA
// holds 128 of the rows and N (up to 128) of the entries, the tensor cores read both CTAs' halves of the weights, and a
// k-step of the same size per CTA takes 32 KB.  Now the tensor core is at work in 90 % of the cycles (459 of 509 thousand at 256 x
// 4096 x 126464), and the clock is what power allows, 1.0-1.2 GHz; the epilogue, which nothing overlaps, is 4 %.
//
// A work item runs the k loop over the drafter's operands into accumulator columns [0, 2N), then over the verifier's
// into [256, 256 + 2N); the same ring of stages feeds both.  The epilogue reads both: in each CTA warps 0-3 take the
// first N columns of its 128 rows, warps 4-7 the other N.  To the fold, that is two vocabulary tiles of N entries.
//
// us, lm_head_kernel : this one (rows, K, V): 256, 4096, 126464 514 : 461 (under the power cap 585 : 504); 512, 3072, 10000
// 95.6 : 74.3; 150, 4096, 50000 239 : 202; 400, 2048, 30000 151 : 135; 200, 1024, 20000 45.9 : 41.2; 635 of 1024, 4096,
// 126464 1270 : 1167; 8192, 512, 2000 61.6 : 61.0.  Up to 128 rows the second CTA's rows are all padding, and
// lm_head_kernel's items of 128 rows are quicker: 128, 4096, 126464 390 : 422; 40 380 : 434.
// Tried: the weights' next 1 to 4 KB of each row prefetched into L2 by the loading thread, 566 to 900 us at 256 rows (the thread does not
// keep up, and copies of 128 bytes a row already read memory at 5.6 TB/s in lm_head_kernel).
//
//   warps 0-7   epilogue
//   warp  8     one thread in each CTA loads this CTA's operands; all copies complete on the leading CTA's barrier
//   warp  9     one thread in the leading CTA issues the MMAs and commits them to the barriers of both
// Every wait is bounded and reports to the verify health word.  Included by dd_verify.cu, after dd_lm_head_kernel.cuh.
#pragma once

namespace ddlm {

constexpr int kPairBars = 2 * kMaxStages + 2;

__global__ void __launch_bounds__(kThreads, 1)
lm_head_pair_kernel(const __grid_constant__ LmMaps<true> maps, const LmParams q, const ddv::VerifyParams p)
{
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
    const int rank = blockIdx.x & 1, pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
    LmPlan plan = q.plan ? *q.plan : q.all_rows;
    // few rows, none listed: perhaps none of them is flagged, and there is nothing to multiply
    int any = 1;
    if (!q.plan && q.rows <= kCheckedRows) {
        any = 0;
        for (int i = tid; i < q.rows; i += kThreads) any |= p.flags[i];
    }
    const int k_steps = q.K / kBlockK;
    const uint32_t stage_bytes = kATileBytes + (uint32_t)plan.N * kBlockK * 2;      // of one CTA
    const uint32_t stages = min((uint32_t)kMaxStages, kRingBytes / stage_bytes);

    if (tid == 0) {
        for (int s = 0; s < kMaxStages; ++s) { mbar_init(bar_full(s), 1); mbar_init(bar_empty(s), 1); }
        mbar_init(bar_acc_full, 1);
        mbar_init(bar_acc_empty, 2 * kEpilogueWarps);
        fence_mbar_init();
        *abort_flag = 0u;
    }
    if (warp == 0) { __syncwarp(); tmem_alloc_pair(tmem_slot, kTmemCols); tmem_relinquish_pair(); }
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
    // pairs of vocabulary tiles x blocks of 256 rows; items that follow each other share the weights
    const int row_blocks = (plan.n_rows + kRowsPerItem - 1) / kRowsPerItem;
    const int n_items = (plan.n_tiles + 1) / 2 * row_blocks;

    if (warp == kLoadWarp && elect_one()) {
        // ===================================================================== TMA producer
        const int width = (Widths<true>::max_n - plan.N) / 32;
        const CUtensorMap *h = plan.gathered ? &maps.h_gathered : &maps.h, *w = &maps.w[width];
        const CUtensorMap *hd = plan.gathered ? &maps.hd_gathered : &maps.hd, *wd = &maps.wd[width];
        prefetch_tmap(h); prefetch_tmap(w); prefetch_tmap(hd); prefetch_tmap(wd);
        uint32_t s = 0, round = 0;                            // stage, and how often the ring has been gone round
        bool ok = true;
        for (int item = pair; item < n_items && ok; item += n_pairs) {
            const int tile = item / row_blocks;
            const int row0 = (item - tile * row_blocks) * kRowsPerItem + rank * kTileRows, col0 = (2 * tile + rank) * plan.N;
            for (int ks2 = 0; ks2 < 2 * k_steps; ++ks2) {
                if (round > 0 && !wait(bar_empty(s), (round - 1) & 1)) { give_up(kErrLmEmpty); ok = false; break; }
                const uint32_t dst = smem_base + s * stage_bytes, bar = cluster_addr(bar_full(s), 0);
                const bool drafter = ks2 < k_steps;                       // the drafter's pass comes first
                const int x = (drafter ? ks2 : ks2 - k_steps) * kBlockK;
                if (rank == 0) mbar_expect_tx(bar_full(s), 2 * stage_bytes);
                tma_load_2d_pair(dst, drafter ? hd : h, bar, x, row0);
                tma_load_2d_pair(dst + kATileBytes, drafter ? wd : w, bar, x, col0);
                if (++s == stages) { s = 0; ++round; }
            }
        }
    } else if (warp == kMmaWarp && rank == 0 && elect_one()) {
        // ===================================================================== MMA issuer
        const uint32_t idesc = idesc_bf16(256, 2 * plan.N, false);
        uint32_t s = 0, round = 0, n = 0;
        bool ok = true;
        for (int item = pair; item < n_items && ok; item += n_pairs, ++n) {
            // both CTAs' epilogues have read the previous item's accumulators
            if (n > 0 && !wait(bar_acc_empty, (n - 1) & 1)) { give_up(kErrLmAcc); break; }
            tc_fence_after();
            for (int ks2 = 0; ks2 < 2 * k_steps; ++ks2) {
                if (!wait(bar_full(s), round & 1)) { give_up(kErrLmFull); ok = false; break; }
                tc_fence_after();
                const uint32_t acc = tmem + (ks2 < k_steps ? 0u : 256u);
                const uint32_t base = smem_base + s * stage_bytes;
                const uint64_t a = smem_desc_sw128(base, 16, 1024), b = smem_desc_sw128(base + kATileBytes, 16, 1024);
#pragma unroll
                for (int kk = 0; kk < kBlockK / 16; ++kk) {
                    const uint32_t off = (uint32_t)(kk * 32) >> 4;            // 16 bf16 = 32 bytes per MMA
                    mma_ss_pair(acc, a + off, b + off, idesc, (kk > 0 || (ks2 != 0 && ks2 != k_steps)));
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
        const uint32_t dacc = tmem + lane_off + (uint32_t)(half * plan.N), tacc = dacc + 256u;
        const uint32_t acc_empty = cluster_addr(bar_acc_empty, 0);
        uint32_t n = 0;
        for (int item = pair; item < n_items; item += n_pairs, ++n) {
            const int block = item / row_blocks, tile = 2 * block + half;
            int row = (item - block * row_blocks) * kRowsPerItem + rank * kTileRows + (warp & 3) * 32 + lane;
            // the row of the caller's tensors, or -1: nothing to store
            if (row >= plan.n_rows || tile >= plan.n_tiles) row = -1;
            else if (plan.gathered) row = q.row_map[ddv::checked(p, row, q.rows, ddv::kSiteRow)];
            else if (!p.flags[row]) row = -1;
            if (!wait(bar_acc_full, n & 1)) {
                if (lane == 0) give_up(kErrLmAcc);
                break;
            }
            tc_fence_after();
            const ddv::Partial c = reduce_columns<true>(tacc, dacc, plan.N, tile * plan.N, q.V);
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
