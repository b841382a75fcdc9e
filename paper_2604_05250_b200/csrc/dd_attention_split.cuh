// dd_block_attention for short query blocks (Section 2.2; Eq. 3 over stored keys and values): a CTA owns one
// tile of up to 128 query rows of one head and a contiguous part of its key tiles, two CTAs share an SM, and
// the CTAs of a cluster share one item's keys.  Roles are those of attention_kernel with one softmax group:
//   warps 0-3   softmax (thread = query row = TMEM lane); warps without a query row sit out
//   warp  4     one thread feeds a ring of K/V tiles by TMA
//   warp  5     one thread issues every tcgen05 MMA
//   warps 6-7   only fill the register-allocation group
// The parts of a split item meet at the end: every CTA leaves its accumulator in fp32 (the ring's memory,
// which no copy or product uses any more) and its rows' reference points and sums in its own shared memory,
// and after a cluster barrier each CTA combines its share of the columns over distributed shared memory, in
// key order.  No scratch in global memory, no counters: calls on any streams may overlap, and the result
// does not depend on timing.
//
// What bounds it.  One tile's chain (copy -> S -> softmax -> P V, some 2600 cycles a key tile, and 4-5 us of start and
// end) keeps neither the memory nor the tensor core busy; the SM's other CTA fills in.  attention_kernel has an SM to
// itself with two query tiles' worth of shared memory and, for a single tile, both softmax groups on it: faster for one
// item, but the next one's start is exposed.  16 sequences x 32 heads, 32 queries over 256-1024 keys: 49.7 -> 43.5 us;
// 64 x 32 heads 174.8 -> 134.7; 40 x 16 heads of 200 keys at D = 64 30.0 -> 21.7.  Where there are few items the
// splitting is what counts: 2 x 8 heads, 16 queries over 4096 keys 32.3 -> 17.0 us.  Built and not faster: persistent
// CTAs that take the next item over from the launch queue (clusterlaunchcontrol) and load it behind the current
// one's tiles, 51 against 43.5 and 160 against 135 us.
//
// Every wait is bounded and reports to the attention health word.  Included by dd_attention.cu (inside its
// unnamed namespace, after the softmax helpers).
#pragma once

constexpr int kSplitThreads = 256;
constexpr int kSplitMax = 8;                                     // CTAs per item (a portable cluster)
constexpr int kSplitLoadWarp = 4, kSplitMmaWarp = 5;
constexpr int kSplitSmem = 112 * 1024 + 1024;                    // two CTAs per SM: Q and ring, alignment slack and barriers

// Q takes q_rows (64 or 128) rows, the ring what is left of 112 KB: two to six tiles.
template <int D>
struct SplitLayout {
    static constexpr int kTileBytes = kBlockN * D * 2;
    static __host__ __device__ constexpr int q_bytes(int q_rows) { return q_rows * D * 2; }
    static __host__ __device__ constexpr int slots(int q_rows) { return (112 * 1024 - q_bytes(q_rows)) / kTileBytes; }
    static constexpr int kMaxSlots = (112 * 1024 - 64 * D * 2) / kTileBytes;
    // q_full, s_full, p_early, p_full, o_full, kv_full[], kv_empty[]
    static constexpr int kNumBars = 5 + 2 * kMaxSlots;
    static constexpr int kBarBytes = 8 * kNumBars + 16;
    static_assert(kBarBytes <= 256, "barriers fit whichever side of the tiles the alignment leaves free");
    static_assert(slots(128) * kTileBytes >= 128 * D * 4, "the ring holds a whole accumulator in fp32");
    static_assert(q_bytes(64) >= 128 * 8, "the query buffer holds the rows' reference points and sums");
};

template <int D>
__global__ void __launch_bounds__(kSplitThreads, 2)
attention_split_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                       const __grid_constant__ CUtensorMap tm_v, const AttnParams p, const int q_rows, const int parts)
{
    using L = SplitLayout<D>;
    constexpr uint32_t kTileBytes = L::kTileBytes;
    constexpr int kBoxes = D / 64;
    constexpr uint32_t kBoxBytes = 128 * 128;
    extern __shared__ __align__(1024) unsigned char smem_dyn[];
    const uint32_t pad = (1024u - (smem_u32(smem_dyn) & 1023u)) & 1023u;
    unsigned char *tiles_gen = smem_dyn + pad;
    const uint32_t sQ = smem_u32(tiles_gen), sRing = sQ + (uint32_t)L::q_bytes(q_rows);
    // the barriers: before the tiles if the alignment left room there, behind them otherwise
    unsigned char *bars_gen = pad >= 256 ? smem_dyn : tiles_gen + 112 * 1024;
    const uint32_t bars = smem_u32(bars_gen);
    const int slots = L::slots(q_rows);
    const uint32_t bar_q = bars, bar_s_full = bars + 8, bar_p_early = bars + 16, bar_p_full = bars + 24, bar_o_full = bars + 32;
    auto bar_kv_full = [&](int s) { return bars + 8u * (5 + s); };
    auto bar_kv_empty = [&](int s) { return bars + 8u * (5 + L::kMaxSlots + s); };
    const uint32_t tmem_slot = bars + 8u * L::kNumBars;
    volatile uint32_t *tmem_slot_gen = reinterpret_cast<volatile uint32_t *>(bars_gen + 8 * L::kNumBars);

    const int tid = threadIdx.x, warp = warp_uniform(tid >> 5), lane = tid & 31;
    const int item = (int)blockIdx.x / parts, part = (int)blockIdx.x - item * parts;
    const int head = item / p.m_blocks, row0 = (item - head * p.m_blocks) * kBlockM;
    int keys;
    const int b_idx = sequence_at(p, head / p.H, keys), h_idx = head % p.H, bh = b_idx * p.H + h_idx;
    const bool hm = p.head_major != 0;
    const int rows = min(p.Nq - row0, kBlockM);                   // query rows of this tile (>= 1)
    const int row_warps = (rows + 31) / 32;
    const int nkv = (keys + kBlockN - 1) / kBlockN;
    const int j_begin = part * nkv / parts, n_tiles = (part + 1) * nkv / parts - j_begin;      // key tiles of this CTA
    auto load_box = [&](uint32_t dst, const CUtensorMap *tm, uint32_t bar, int c0, int n0) {
        if (hm) tma_load_3d(dst, tm, bar, c0, n0, bh);
        else tma_load_4d(dst, tm, bar, c0, n0, h_idx, b_idx);
    };
    auto load_tile = [&](int slot, const CUtensorMap *tm, int j) {
        mbar_expect_tx(bar_kv_full(slot), kTileBytes);
#pragma unroll
        for (int cx = 0; cx < kBoxes; ++cx)
            load_box(sRing + slot * kTileBytes + cx * kBoxBytes, tm, bar_kv_full(slot), cx * 64, j * kBlockN);
    };

    // The producer thread sets up the barriers its copies complete on and sends the query tile, the first key
    // and the first value tile on their way before the CTA's first barrier.
    if (warp == kSplitLoadWarp && elect_one()) {
        prefetch_tmap(&tm_q); prefetch_tmap(&tm_k); prefetch_tmap(&tm_v);
        mbar_init(bar_q, 1);
        for (int s = 0; s < slots; ++s) mbar_init(bar_kv_full(s), 1);
        fence_mbar_init();
        if (n_tiles > 0) {
            mbar_expect_tx(bar_q, (uint32_t)L::q_bytes(q_rows));
#pragma unroll
            for (int cx = 0; cx < kBoxes; ++cx) load_box(sQ + cx * (q_rows * 128), &tm_q, bar_q, cx * 64, row0);
            load_tile(0, &tm_k, j_begin);
            load_tile(1, &tm_v, j_begin);
        }
    }
    if (tid == 0) {
        for (int s = 0; s < slots; ++s) mbar_init(bar_kv_empty(s), 1);
        mbar_init(bar_s_full, 1);
        mbar_init(bar_p_early, row_warps * 32);
        mbar_init(bar_p_full, row_warps * 32);
        mbar_init(bar_o_full, 1);
        fence_mbar_init();
        // a wait that expired in an earlier CTA or launch stops the rest from queueing up behind it
        tmem_slot_gen[1] = *reinterpret_cast<volatile unsigned int *>(p.status);
    }
    if (warp == 0) { tmem_alloc(tmem_slot, 256); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = warp_uniform(*tmem_slot_gen);
    const bool healthy = tmem_slot_gen[1] == 0;
    constexpr uint32_t kColS = 0, kColO = 128;

    // one row of the result: columns c0 .. c0 + 15
    const bool sectors = (reinterpret_cast<uintptr_t>(p.out) & 31) == 0;
    auto store16 = [&](int row, int c0, const float *v, float f) {
        const size_t at = hm ? (size_t)bh * p.Nq + row0 + row : ((size_t)b_idx * p.Nq + row0 + row) * p.H + h_idx;
        unsigned char *dst = reinterpret_cast<unsigned char *>(p.out) + (at * D + c0) * 2;
        uint32_t w[8];
#pragma unroll
        for (int h = 0; h < 8; ++h) {
            __nv_bfloat162 x = __floats2bfloat162_rn(v[2 * h] * f, v[2 * h + 1] * f);
            w[h] = *reinterpret_cast<uint32_t *>(&x);
        }
        if (sectors) st_global_v8(dst, w);
        else {
            reinterpret_cast<uint4 *>(dst)[0] = make_uint4(w[0], w[1], w[2], w[3]);
            reinterpret_cast<uint4 *>(dst)[1] = make_uint4(w[4], w[5], w[6], w[7]);
        }
    };

    if (warp < 4) {
        reg_inc<200>();
        if (healthy && warp < row_warps) {
            // =============================================================== softmax warps
            const uint32_t lane_off = (uint32_t)(warp * 32) << 16;
            const uint32_t tS = tmem + lane_off + kColS, tO = tmem + lane_off + kColO;
            const float c = p.scale_log2;
            const int row = warp * 32 + lane;
            float m_ref = -INFINITY, l_run = 0.f;
            unsigned err = 0;
            for (int i = 0; i < n_tiles; ++i) {
                if (!mbar_wait(bar_s_full, i & 1)) { err = kErrWaitS; break; }
                tc_fence_after();
                const int valid = keys - (j_begin + i) * kBlockN;
                // Keys past the sequence's end have weight zero, but 0 x NaN is NaN in the product P V, and
                // padding may hold any bit pattern: its value rows are cleared in the ring slot (whole
                // 128-byte rows, which the swizzle maps onto themselves) before the weights are handed over.
                // Rows past the end of the tensor were zero-filled by the copy.
                const bool clear = valid < kBlockN && keys < p.Nkv;
                softmax_tile<D>(tS, tO, i == 0, valid, c, m_ref, l_run, [&] {
                    if (clear) return;
                    tmem_wait_st();
                    tc_fence_before();
                    mbar_arrive(bar_p_early);
                });
                if (clear) {
                    const int tile_v = 2 * i + 1, slot_v = tile_v % slots;
                    if (!mbar_wait(bar_kv_full(slot_v), (tile_v / slots) & 1)) { err = kErrWaitKV; break; }
                    for (int r = valid + warp * 4 + (lane >> 3); r < kBlockN; r += row_warps * 4)
#pragma unroll
                        for (int cx = 0; cx < kBoxes; ++cx)
                            st_shared_v4(sRing + slot_v * kTileBytes + cx * kBoxBytes + r * 128 + (lane & 7) * 16, 0u, 0u, 0u, 0u);
                    fence_proxy_async_smem();
                }
                tmem_wait_st();
                tc_fence_before();
                if (clear) mbar_arrive(bar_p_early);
                mbar_arrive(bar_p_full);
            }
            if (err == 0 && n_tiles > 0 && !mbar_wait(bar_o_full, 0)) err = kErrWaitO;
            if (err != 0) report(p, err);
            // ---- epilogue: the whole accumulator row in one go
            tc_fence_after();
            uint32_t acc[D];
            if (n_tiles > 0) {
#pragma unroll
                for (int cb = 0; cb < D / 32; ++cb)
                    tmem_ld32(tO + cb * 32, *reinterpret_cast<uint32_t(*)[32]>(&acc[cb * 32]));
                tmem_wait_ld();
            } else {
#pragma unroll
                for (int i = 0; i < D; ++i) acc[i] = 0u;
            }
            if (parts == 1) {
                const float inv = nkv > 0 ? 1.f / l_run : 0.f;
                if (err == 0 && row < rows)
#pragma unroll
                    for (int c0 = 0; c0 < D; c0 += 16) store16(row, c0, reinterpret_cast<float *>(&acc[c0]), inv);
            } else {
                // columns 4 c .. 4 c + 3 of the tile's rows lie together: conflict-free here and in the reader
                reinterpret_cast<float2 *>(tiles_gen)[row] = make_float2(m_ref, l_run);
#pragma unroll
                for (int i = 0; i < D; i += 4)
                    st_shared_v4(sRing + ((i / 4) * kBlockM + row) * 16, acc[i], acc[i + 1], acc[i + 2], acc[i + 3]);
            }
        }
    } else {
        reg_dec<56>();
        if (healthy && warp == kSplitLoadWarp && elect_one()) {
            // =============================================================== TMA producer
            // ring tiles: 2i = K tile i, 2i + 1 = V tile i; the first two are on their way
            for (int t = 2, slot = 2 % slots, use = 2 / slots; t < 2 * n_tiles; ++t) {
                if (use > 0 && !mbar_wait(bar_kv_empty(slot), (use - 1) & 1)) { report(p, kErrWaitSlot); break; }
                load_tile(slot, (t & 1) ? &tm_v : &tm_k, j_begin + (t >> 1));
                if (++slot == slots) { slot = 0; ++use; }
            }
        } else if (healthy && warp == kSplitMmaWarp && elect_one()) {
            // =============================================================== MMA issuer
            constexpr uint32_t kIdescS = idesc_bf16(kBlockM, kBlockN, false);
            constexpr uint32_t kIdescO = idesc_bf16(kBlockM, D, true);
            const uint64_t desc_q = smem_desc_sw128(sQ, 16, 1024);
            const uint64_t desc_k0 = smem_desc_sw128(sRing, 16, 1024);            // K-major operand (K tile)
            const uint64_t desc_v0 = smem_desc_sw128(sRing, kBoxBytes, 1024);     // MN-major operand (V tile)
            unsigned err = 0;
            int slot = 0;
            uint32_t phase = 0;                        // ring position of the next tile to be read
            auto next_slot = [&] { if (++slot == slots) { slot = 0; phase ^= 1; } };
            // S = Q K^T.  All 128 rows of the instruction are computed; those past the query buffer's read
            // whatever follows it in shared memory, and nothing reads their scores.
            auto issue_s = [&] {
                const uint64_t b = desc_k0 + (uint64_t)(slot * (kTileBytes >> 4));
#pragma unroll
                for (int ks = 0; ks < D / 16; ++ks) {
                    const uint32_t off_a = ((ks / 4) * (uint32_t)(q_rows * 128) + (ks % 4) * 32) >> 4;
                    const uint32_t off_b = ((ks / 4) * kBoxBytes + (ks % 4) * 32) >> 4;
                    mma_ss(tmem + kColS, desc_q + off_a, b + off_b, kIdescS, ks > 0);
                }
                mma_commit(bar_s_full);
                mma_commit(bar_kv_empty(slot));
            };
            do {
                if (n_tiles == 0) break;
                if (!mbar_wait(bar_q, 0)) { err = kErrWaitQ; break; }
                if (!mbar_wait(bar_kv_full(slot), phase)) { err = kErrWaitKV; break; }
                tc_fence_after();
                issue_s();
                next_slot();
                for (int i = 0; i < n_tiles; ++i) {
                    if (!mbar_wait(bar_kv_full(slot), phase)) { err = kErrWaitKV; break; }
                    if (!mbar_wait(bar_p_early, i & 1)) { err = kErrWaitP; break; }
                    tc_fence_after();
                    const uint64_t b = desc_v0 + (uint64_t)(slot * (kTileBytes >> 4));
                    bool ok = true;
#pragma unroll
                    for (int ks = 0; ks < kBlockN / 16; ++ks) {
                        // 16 keys = two 8-row groups of 1024 bytes; column blocks of 64 are one box apart
                        if (ks == 6) {
                            if (!mbar_wait(bar_p_full, i & 1)) { ok = false; break; }
                            tc_fence_after();
                        }
                        mma_ts(tmem + kColO, tmem + kColS + ks * 8, b + (uint32_t)(ks * (2048 >> 4)), kIdescO, (i > 0 || ks > 0));
                    }
                    if (!ok) { err = kErrWaitP; break; }
                    if (i + 1 == n_tiles) { mma_commit(bar_o_full); break; }
                    mma_commit(bar_kv_empty(slot));
                    next_slot();
                    if (!mbar_wait(bar_kv_full(slot), phase)) { err = kErrWaitKV; break; }
                    tc_fence_after();
                    issue_s();
                    next_slot();
                }
            } while (false);
            if (err) report(p, err);
        }
    }

    __syncwarp();
    if (*reinterpret_cast<volatile unsigned int *>(p.status) != 0) {
        // a wait expired somewhere: give copies that may still be in flight time to land before the
        // shared memory is released
        for (int i = 0; i < 2000; ++i) __nanosleep(1000);
    }
    tc_fence_before();
    if (parts > 1) {
        // ---- the parts meet: every thread of every CTA of the cluster takes part in both barriers
        __syncwarp();
        cluster_arrive();
        cluster_wait();
        if (healthy && warp < 4) {
            constexpr int kGroups = D / 16;                      // of 16 columns
            const int units = row_warps * kGroups;
            for (int u = warp * parts + part; u < units; u += 4 * parts) {
                const int row = (u / kGroups) * 32 + lane, c0 = (u % kGroups) * 16;
                float2 ml[kSplitMax];
                float m_all = -INFINITY;
                for (int i = 0; i < parts; ++i) {
                    ml[i] = make_float2(-INFINITY, 0.f);
                    if ((i + 1) * nkv / parts == i * nkv / parts) continue;       // no key tile, nothing written
                    ml[i] = ld_cluster_v2(cluster_addr(sQ + row * 8, i));
                    m_all = fmaxf(m_all, ml[i].x);
                }
                float sum = 0.f, acc[16];
#pragma unroll
                for (int k = 0; k < 16; ++k) acc[k] = 0.f;
                for (int i = 0; i < parts; ++i) {
                    if ((i + 1) * nkv / parts == i * nkv / parts) continue;
                    const float w = ex2(ml[i].x - m_all);
                    sum += ml[i].y * w;
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const float4 v = ld_cluster_v4(cluster_addr(sRing + ((c0 / 4 + k) * kBlockM + row) * 16, i));
                        acc[4 * k] += v.x * w; acc[4 * k + 1] += v.y * w; acc[4 * k + 2] += v.z * w; acc[4 * k + 3] += v.w * w;
                    }
                }
                if (row < rows) store16(row, c0, acc, nkv > 0 ? 1.f / sum : 0.f);
            }
        }
        __syncwarp();
        cluster_arrive();            // no CTA leaves while another reads its shared memory
        cluster_wait();
    }
    __syncthreads();
    if (warp == 0) { __syncwarp(); tmem_dealloc(tmem, 256); }
}
