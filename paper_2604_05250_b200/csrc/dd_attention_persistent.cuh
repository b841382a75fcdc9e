// The square, head-major case of dd_bidir_attention (Section 2.2; Eq. 3) where there are more work items than SMs and at least two key
// tiles: persistent CTAs, one per SM, each walking over work items blockIdx.x,
// blockIdx.x + gridDim.x, ...  An item is two tiles of 128 query rows of one head (the second one may be empty).  Roles and
// arithmetic are those of attention_kernel; the pipeline never drains between items.
//
// One stream of rounds.  Round r of a CTA is one key tile of one item, for both query tiles g:
// O_g += P_g V, and the S_g that follows.  The K tile a round needs beside its V tile is the one of the
// next round, whichever item that belongs to, so V of round r and K of round r + 1 form a pair: one
// barrier announces both, and one commit at the end of the round releases both.  Items therefore
// follow each other like rounds do: the next item's first scores are computed while the softmax
// groups still work on the current item's last tile or write its result.
//   * A barrier wait costs the issuing thread some cycles (10-40 under elect.sync) even when its phase is complete,
//     which the tensor core spends on products already queued, but only so many; so there are few of them: one
//     per round for the pair and two per group for its weights.
//   * The weights of a tile are handed over in two parts: the product starts with the first three
//     quarters of the keys while the softmax group still computes the last.
//   * A group that has received S of round r + 1 knows that P V of round r has completed (same thread,
//     issued earlier), so O has a barrier of its own only at an item's end.
//   * Q buffers: Q_g of the next item goes into a buffer whose last S product has been committed
//     (q_free), a round before the item ends, not into one whose result has been written: results go from
//     registers straight to global memory, so that five key/value tiles fit beside two query tiles.  (Staged in shared
//     memory, with four: 16 x 32 heads of 512 tokens 83 -> 88 us, of 1024 269 -> 289.)
//   * Every lane storing its own row, 32 bytes at a time, took 2500 to 2900 cycles per item and group; four lanes
//     now exchange pieces first and store 128 bytes of a row together: 2000 (16 x 32 of 512 71.3 -> 68.5 us in short bursts).
//   * A group writes an item's result behind the weights of the next item's first tile, whose products the stores then overlap: 68.5
//     -> 67.2 in bursts; both, under the power cap, 84.7 -> 78.0.
//   * o_free: the group has read the finished accumulator out of tensor memory; the next item's
//     first P V may overwrite it.
// Every wait is bounded and reports to the attention health word.  Included by dd_attention.cu
// (inside its unnamed namespace, after the softmax helpers).
#pragma once

constexpr int kReleases = 8;         // release barriers: round r completes phase r / 8 of barrier r % 8

template <int D>
struct SmemL {
    static constexpr int kTileBytes = kBlockN * D * 2;
    static constexpr int kQ = 2;                                    // query tiles
    static constexpr int kSlots = D == 128 ? 5 : 9;                 // key and value tiles
    static constexpr int kPairs = kSlots / 2 + 1;                   // pair barriers
    static constexpr int kRing = kQ * kTileBytes;
    static constexpr int kBars = kRing + kSlots * kTileBytes;
    // q_full[kQ], q_free[kQ], pair[kPairs], release[kReleases], k0_full,
    // s_full[2], p_early[2], p_full[2], o_full[2], o_free[2]
    static constexpr int kNumBars = 2 * kQ + kPairs + kReleases + 1 + 10;
    static constexpr int kTmemSlot = kBars + 8 * kNumBars;
    static constexpr int kTotal = kTmemSlot + 16;
    static_assert(kTileBytes % 1024 == 0 && kBars % 8 == 0, "tiles on swizzle boundaries, barriers on 8 bytes");
    static_assert(kTotal + 1024 <= 227 * 1024, "shared memory of one CTA");
    // A barrier may not get two phases ahead of a waiter: the producer is at most (kSlots - 1) / 2 + 1 rounds
    // past the release it waits for, and at most kPairs pairs past the one the issuing thread waits for.
    static_assert((kSlots - 1) / 2 + 1 <= kReleases, "release barriers");
};

template <int D>
__global__ void __launch_bounds__(kThreads, 1)
attention_persistent_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                            const __grid_constant__ CUtensorMap tm_v, const AttnParams p)
{
    using L = SmemL<D>;
    constexpr uint32_t kQ = L::kQ, kSlots = L::kSlots;
    extern __shared__ __align__(1024) unsigned char smem_dyn[];
    const uint32_t smem_base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
    unsigned char *smem_gen = smem_dyn + (smem_base - smem_u32(smem_dyn));
    constexpr uint32_t kTileBytes = L::kTileBytes;
    const uint32_t sQ = smem_base, sRing = smem_base + L::kRing;
    const uint32_t bars = smem_base + L::kBars;
    auto bar_q_full = [&](uint32_t b) { return bars + 8u * b; };
    auto bar_q_free = [&](uint32_t b) { return bars + 8u * (kQ + b); };
    auto bar_pair = [&](uint32_t i) { return bars + 8u * (2 * kQ + i); };
    auto bar_release = [&](uint32_t i) { return bars + 8u * (2 * kQ + L::kPairs + i); };
    constexpr uint32_t kFixed = 2 * kQ + L::kPairs + kReleases;
    const uint32_t bar_k0 = bars + 8u * kFixed;
    auto bar_s_full = [&](int g) { return bars + 8u * (kFixed + 1 + g); };
    auto bar_p_early = [&](int g) { return bars + 8u * (kFixed + 3 + g); };
    auto bar_p_full = [&](int g) { return bars + 8u * (kFixed + 5 + g); };
    auto bar_o_full = [&](int g) { return bars + 8u * (kFixed + 7 + g); };
    auto bar_o_free = [&](int g) { return bars + 8u * (kFixed + 9 + g); };
    const uint32_t tmem_slot = smem_base + L::kTmemSlot;
    volatile uint32_t *tmem_slot_gen = reinterpret_cast<volatile uint32_t *>(smem_gen + L::kTmemSlot);

    const int tid = threadIdx.x, warp = warp_uniform(tid >> 5), lane = tid & 31;
    const int n_items = p.BH * p.m_blocks;
    const int nkv = (p.Nkv + kBlockN - 1) / kBlockN;            // rounds per item (>= 2)
    const int my_items = (n_items - 1 - (int)blockIdx.x) / (int)gridDim.x + 1;
    constexpr int kBoxes = D / 64;
    constexpr uint32_t kBoxBytes = 128 * 128;
    constexpr uint32_t kColS = 0, kColO = 256;       // S_0, S_1 (128 columns each, P over them), O_0, O_1 (D each)
    struct Item { int bh, row0; };
    auto item_at = [&](int n) {
        const int item = (int)blockIdx.x + n * (int)gridDim.x;
        Item t;
        t.bh = item / p.m_blocks;
        t.row0 = (item - t.bh * p.m_blocks) * (kQTiles * kBlockM);
        return t;
    };
    auto load_tile = [&](uint32_t dst, const CUtensorMap *tm, uint32_t bar, int row, int bh) {
#pragma unroll
        for (int cx = 0; cx < kBoxes; ++cx) tma_load_3d(dst + cx * kBoxBytes, tm, bar, cx * 64, row, bh);
    };

    // The producer thread sets up the barriers its copies complete on and sends Q tile 0 and K tile 0
    // on their way before the CTA's first barrier: they travel while tensor memory is allocated and
    // the other barriers are set up.  (Also when an earlier wait has expired and the CTA will do
    // nothing: such a CTA lingers at its end until copies in flight have landed.)
    if (warp == kLoadWarp && elect_one()) {
        prefetch_tmap(&tm_q); prefetch_tmap(&tm_k); prefetch_tmap(&tm_v);
        for (uint32_t i = 0; i < kQ; ++i) mbar_init(bar_q_full(i), 1);
        for (int i = 0; i < L::kPairs; ++i) mbar_init(bar_pair(i), 1);
        mbar_init(bar_k0, 1);
        fence_mbar_init();
        grid_wait();
        const Item t = item_at(0);
        mbar_expect_tx(bar_q_full(0), kTileBytes);
        load_tile(sQ, &tm_q, bar_q_full(0), t.row0, t.bh);
        mbar_expect_tx(bar_k0, kTileBytes);
        load_tile(sRing, &tm_k, bar_k0, 0, t.bh);
    }
    if (tid == 0) {
        for (uint32_t i = 0; i < kQ; ++i) mbar_init(bar_q_free(i), 1);
        for (int i = 0; i < kReleases; ++i) mbar_init(bar_release(i), 1);
        for (int g = 0; g < kQTiles; ++g) {
            mbar_init(bar_s_full(g), 1);
            mbar_init(bar_p_early(g), kBlockM);
            mbar_init(bar_p_full(g), kBlockM);
            mbar_init(bar_o_full(g), 1);
            mbar_init(bar_o_free(g), kBlockM);
        }
        fence_mbar_init();
        grid_wait();
        // a wait that expired in an earlier CTA or launch stops the rest from queueing up behind it
        tmem_slot_gen[1] = *reinterpret_cast<volatile unsigned int *>(p.status);
    }
    if (warp == 0) { tmem_alloc(tmem_slot, kTmemCols); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = warp_uniform(*tmem_slot_gen);
    const bool healthy = tmem_slot_gen[1] == 0;

    if (!healthy) {
        // nothing to do
    } else if (warp < kSoftmaxWarps) {
        // =================================================================== softmax warpgroups
        reg_inc<216>();
        const int g = warp >> 2;
        const uint32_t lane_off = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t tS = tmem + lane_off + kColS + g * kBlockN;
        const uint32_t tO = tmem + lane_off + kColO + g * D;
        const float c = p.scale_log2;
        const bool sectors = (reinterpret_cast<uintptr_t>(p.out) & 31) == 0;     // rows start on 32-byte boundaries
        uint32_t t_run = 0;              // key tiles so far: phase
        unsigned err = 0;
        // An item's result is written after the weights of the next item's first tile have been handed over: the stores then
        // overlap that tile's products, and the group does not stand still for its last P V.
        float l_prev = 0.f;
        for (int n = 0; n <= my_items && err == 0; ++n) {
            float m_ref = -INFINITY, l_run = 0.f;
            for (int j = 0; j < nkv; ++j) {
                if (n < my_items) {
                    if (!mbar_wait(bar_s_full(g), t_run & 1)) { err = kErrWaitS; break; }
                    tc_fence_after();
                    softmax_tile<D, false>(tS, tO, j == 0, p.Nkv - j * kBlockN, c, m_ref, l_run,
                        [&] {                        // three quarters of the weights are stored
                            tmem_wait_st();
                            tc_fence_before();
                            mbar_arrive(bar_p_early(g));
                        });
                    tmem_wait_st();
                    tc_fence_before();
                    mbar_arrive(bar_p_full(g));
                    ++t_run;
                }
                if (j == 0 && n > 0) {
                    // ---- epilogue of the item before: O / l -> bf16 -> global
                    if (!mbar_wait(bar_o_full(g), (n - 1) & 1)) { err = kErrWaitO; break; }
                    tc_fence_after();
                    uint32_t acc[D];
#pragma unroll
                    for (int cb = 0; cb < D / 32; ++cb)
                        tmem_ld32(tO + cb * 32, *reinterpret_cast<uint32_t(*)[32]>(&acc[cb * 32]));
                    tmem_wait_ld();
                    tc_fence_before();
                    mbar_arrive(bar_o_free(g));      // this item's first P V may overwrite the accumulator
                    const Item t = item_at(n - 1);
                    const int row = t.row0 + g * kBlockM + (warp & 3) * 32 + (lane & ~3);       // of the quad's first lane
                    unsigned char *dst = reinterpret_cast<unsigned char *>(p.out) + ((size_t)t.bh * p.Nq + row) * (D * 2) + (lane & 3) * 32;
                    const float inv = 1.f / l_prev;
#pragma unroll
                    for (int h = 0; h < D / 64; ++h) {
                        // 64 columns of four rows: each lane turns its row's four 32-byte pieces into one piece of every row
                        uint32_t w[4][8];
#pragma unroll
                        for (int q = 0; q < 4; ++q)
#pragma unroll
                            for (int i = 0; i < 8; ++i) {
                                const int e = 64 * h + 16 * q + 2 * i;
                                __nv_bfloat162 v = __floats2bfloat162_rn(__uint_as_float(acc[e]) * inv, __uint_as_float(acc[e + 1]) * inv);
                                w[q][i] = *reinterpret_cast<uint32_t *>(&v);
                            }
                        quad_transpose(w, lane);
#pragma unroll
                        for (int r = 0; r < 4; ++r) {
                            if (row + r >= p.Nq) break;
                            unsigned char *to = dst + r * (D * 2) + h * 128;
                            if (sectors) st_global_v8(to, w[r]);
                            else {
                                reinterpret_cast<uint4 *>(to)[0] = make_uint4(w[r][0], w[r][1], w[r][2], w[r][3]);
                                reinterpret_cast<uint4 *>(to)[1] = make_uint4(w[r][4], w[r][5], w[r][6], w[r][7]);
                            }
                        }
                    }
                }
                if (n == my_items) break;
            }
            l_prev = l_run;
        }
        if (err != 0) report(p, err);
    } else {
        reg_dec<72>();
        if (warp == kLoadWarp && elect_one()) {
            // =============================================================== TMA producer
            uint32_t qi = 1;             // query tiles sent so far
            auto load_q = [&](const Item &t, int g) -> bool {
                const uint32_t b = qi % kQ, use = qi / kQ;
                if (use > 0 && !mbar_wait(bar_q_free(b), (use - 1) & 1)) return false;
                mbar_expect_tx(bar_q_full(b), kTileBytes);
                load_tile(sQ + b * kTileBytes, &tm_q, bar_q_full(b), t.row0 + g * kBlockM, t.bh);
                ++qi;
                return true;
            };
            // ring position i: 0 is the first K tile, 2r + 1 the V tile of round r, 2r + 2 the K tile of
            // round r + 1; the slot is free once the round that read position i - kSlots has completed
            uint32_t released = 0;       // rounds known to have completed
            auto slot_free = [&](uint32_t i) -> bool {
                if (i < kSlots) return true;
                const uint32_t r = i == kSlots ? 0u : (i - kSlots - 1) >> 1;
                for (; released <= r; ++released)
                    if (!mbar_wait(bar_release(released % kReleases), (released / kReleases) & 1)) return false;
                return true;
            };
            Item t = item_at(0);
            bool ok = load_q(t, 1);
            uint32_t r = 0;
            for (int n = 0; n < my_items && ok; ++n) {
                const bool more_items = n + 1 < my_items;
                const Item next = more_items ? item_at(n + 1) : t;
                for (int j = 0; j < nkv && ok; ++j, ++r) {
                    const bool last = j + 1 == nkv, with_k = !last || more_items;
                    const uint32_t bar = bar_pair(r % L::kPairs);
                    if (!slot_free(2 * r + 1)) { ok = false; break; }
                    mbar_expect_tx(bar, with_k ? 2 * kTileBytes : kTileBytes);
                    load_tile(sRing + ((2 * r + 1) % kSlots) * kTileBytes, &tm_v, bar, j * kBlockN, t.bh);
                    if (with_k) {
                        if (!slot_free(2 * r + 2)) { ok = false; break; }
                        load_tile(sRing + ((2 * r + 2) % kSlots) * kTileBytes, &tm_k, bar, last ? 0 : (j + 1) * kBlockN,
                                  last ? next.bh : t.bh);
                    }
                    if (last && more_items) ok = load_q(next, 0) && load_q(next, 1);
                }
                t = next;
            }
            grid_trigger();
            if (!ok) report(p, kErrWaitSlot);
        } else if (warp == kMmaWarp && elect_one()) {
            // =============================================================== MMA issuer
            constexpr uint32_t kIdescS = idesc_bf16(kBlockM, kBlockN, false);
            constexpr uint32_t kIdescO = idesc_bf16(kBlockM, D, true);
            const uint64_t desc_q0 = smem_desc_sw128(sQ, 16, 1024);
            const uint64_t desc_k0 = smem_desc_sw128(sRing, 16, 1024);            // K-major operand (K tile)
            const uint64_t desc_v0 = smem_desc_sw128(sRing, kBoxBytes, 1024);     // MN-major operand (V tile)
            unsigned err = 0;
            auto issue_s = [&](int g, uint32_t q_buf, uint32_t slot) {
                const uint64_t a = desc_q0 + (uint64_t)(q_buf * (kTileBytes >> 4));
                const uint64_t b = desc_k0 + (uint64_t)(slot * (kTileBytes >> 4));
                const uint32_t tS = tmem + kColS + g * kBlockN;
#pragma unroll
                for (int ks = 0; ks < D / 16; ++ks) {
                    const uint32_t off = ((ks / 4) * kBoxBytes + (ks % 4) * 32) >> 4;   // 16 bf16 = 32 bytes per k-step
                    mma_ss(tS, a + off, b + off, kIdescS, ks > 0);
                }
                mma_commit(bar_s_full(g));
            };
            // O_g (+)= P_g V, the weights of the last quarter of the keys as soon as they are there
            auto issue_o = [&](int g, uint32_t slot, bool first, uint32_t parity) -> bool {
                const uint64_t b = desc_v0 + (uint64_t)(slot * (kTileBytes >> 4));
                const uint32_t tP = tmem + kColS + g * kBlockN, tO = tmem + kColO + g * D;
#pragma unroll
                for (int ks = 0; ks < kBlockN / 16; ++ks) {
                    // 16 keys = two 8-row groups of 1024 bytes; column blocks of 64 are one box apart
                    if (ks == 6) {
                        if (!mbar_wait(bar_p_full(g), parity)) return false;
                        tc_fence_after();
                    }
                    mma_ts(tO, tP + ks * 8, b + (uint32_t)(ks * (2048 >> 4)), kIdescO, (!first || ks > 0));
                }
                return true;
            };
            uint32_t qi = 0;                       // query tiles taken over so far
            uint32_t q_cur[2] = {0, 0};            // their buffers, of the item whose scores are being issued
            auto take_q = [&](int g) -> bool {
                const uint32_t b = qi % kQ;
                if (!mbar_wait(bar_q_full(b), (qi / kQ) & 1)) return false;
                q_cur[g] = b;
                ++qi;
                return true;
            };
            // first scores of the first item
            for (int g = 0; g < kQTiles && !err; ++g) {
                if (!take_q(g)) { err = kErrWaitQ; break; }
                if (g == 0 && !mbar_wait(bar_k0, 0)) { err = kErrWaitKV; break; }
                tc_fence_after();
                issue_s(g, q_cur[g], 0);
            }
            uint32_t r = 0;                        // rounds so far: the phase of the weights' barriers
            for (int n = 0; n < my_items && !err; ++n) {
                for (int j = 0; j < nkv && !err; ++j, ++r) {
                    const bool last = j + 1 == nkv;
                    const bool more = !last || n + 1 < my_items;         // there is a next S
                    const uint32_t slot_v = (2 * r + 1) % kSlots, slot_k = (2 * r + 2) % kSlots;
                    // V of this round, K of the next
                    if (!mbar_wait(bar_pair(r % L::kPairs), (r / L::kPairs) & 1)) { err = kErrWaitKV; break; }
                    auto next_s = [&](int g) {
                        if (!more) return;
                        if (last && !take_q(g)) { err = kErrWaitQ; return; }
                        if (last) tc_fence_after();
                        issue_s(g, q_cur[g], slot_k);
                        if (j + 2 == nkv) mma_commit(bar_q_free(q_cur[g]));      // its query tile's last
                    };
#pragma unroll
                    for (int g = 0; g < kQTiles; ++g) {
                        if (err) break;
                        if (!mbar_wait(bar_p_early(g), r & 1)) { err = kErrWaitP; break; }
                        // the first product of an item overwrites the accumulator: the group must
                        // have read the previous item's result out of it
                        if (j == 0 && n > 0 && !mbar_wait(bar_o_free(g), (uint32_t)(n - 1) & 1)) { err = kErrWaitO; break; }
                        tc_fence_after();
                        if (!issue_o(g, slot_v, j == 0, r & 1)) { err = kErrWaitP; break; }
                        if (last) mma_commit(bar_o_full(g));
                        next_s(g);
                    }
                    mma_commit(bar_release(r % kReleases));
                }
            }
            if (err) report(p, err);
        }
    }

    __syncwarp();
    if (*reinterpret_cast<volatile unsigned int *>(p.status) != 0) {
        // a wait expired somewhere: give copies that may still be in flight time to land before the
        // shared memory is released
#pragma unroll 1
        for (int i = 0; i < 2000; ++i) __nanosleep(1000);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) { __syncwarp(); tmem_dealloc(tmem, kTmemCols); }
}
