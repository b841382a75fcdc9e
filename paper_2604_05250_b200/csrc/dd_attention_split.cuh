// dd_block_attention for short query blocks (Section 2.2; Eq. 3 over stored keys and values): a CTA owns one
// tile of up to 128 query rows of one head and a contiguous part of its key tiles, two CTAs share an SM, and
// the CTAs of a cluster share one item's keys.  Roles are those of attention_kernel with one softmax group:
//   warps 0-3   softmax (thread = query row = TMEM lane); warps without a query row sit out
//   warp  4     one thread feeds a ring of K/V tiles by TMA
//   warp  5     one thread issues every tcgen05 MMA
//   warps 6-7   clear the value rows behind a sequence's end
// The parts of a split item meet at the end: every CTA leaves its accumulator in fp32 (the ring's memory,
// which no copy or product uses any more) and its rows' reference points and sums in its own shared memory,
// and after a cluster barrier each CTA combines its share of the columns over distributed shared memory, in
// key order.  No scratch in global memory, no counters: calls on any streams may overlap, and the result
// does not depend on timing.
//
// What bounds it.  One tile's chain (copy -> S -> softmax -> P V, some 2600 cycles a key tile, and 4-5 us of start and
// end) keeps neither the memory nor the tensor core busy; the SM's other CTA fills in.  attention_kernel has an SM to
// itself with two query tiles' worth of shared memory and, for a single tile, both softmax groups on it: faster for one
// item, but the next one's start is exposed.  16 sequences x 32 heads, 32 queries over 256-1024 keys: 49.7 -> 43.5 us
// (before copies and order, below and in sequence_at: 37.7 now); 64 x 32 heads 174.8 -> 134.7; 40 x 16 heads of up to 200
// keys at D = 64 30.0 -> 21.7.  Where there are few items the
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
    // q_full, s_full, p_early, p_full, o_full, v_last, v_clear, kv_full[], kv_empty[]
    static constexpr int kFixedBars = 7;
    static constexpr int kNumBars = kFixedBars + 2 * kMaxSlots;
    static constexpr int kBarBytes = 8 * kNumBars + 16;
    static_assert(kBarBytes <= 256, "barriers fit whichever side of the tiles the alignment leaves free");
    static_assert(slots(128) * kTileBytes >= 128 * D * 4, "the ring holds a whole accumulator in fp32");
    static_assert(q_bytes(64) >= 2 * 128 * 8, "the query buffer holds the rows' reference points and sums");
};

// softmax_tile for a row that takes only the tile's keys key0 .. key0 + K - 1; the others' weights are not written, and
// the products with those keys leave the row alone.
template <int D, int K>
__device__ __forceinline__ void softmax_part(uint32_t tS, uint32_t tO, int key0, bool first, int valid, float c, float &m_ref,
                                             float &l_run)
{
    float s[K];
#pragma unroll
    for (int cb = 0; cb < K / 32; ++cb)
        tmem_ld32(tS + key0 + cb * 32, *reinterpret_cast<uint32_t(*)[32]>(&s[cb * 32]));
    tmem_wait_ld();
    const int own = valid - key0;
    const bool masked = own < K;
    const float mx = own <= 0 ? -INFINITY : (masked ? row_max<true>(s, own) : row_max<false>(s, own)) * c;
    move_reference<D, true>(tO, first, mx, m_ref, l_run);
    float2 sum_a = make_float2(0.f, 0.f), sum_b = sum_a;
    auto weights = [&](auto is_masked, auto poly) {
#pragma unroll
        for (int q = 0; q < K / 32; ++q)
            weights_to_tmem<decltype(is_masked)::value, decltype(poly)::value>(s, q, own, c, m_ref, tS + key0 / 2, sum_a, sum_b);
    };
    if (masked) weights(std::true_type(), std::integral_constant<int, 0>());
    else weights(std::false_type(), std::integral_constant<int, kPolyOneIn<D>>());
    sum_a = __fadd2_rn(sum_a, sum_b);
    l_run += sum_a.x + sum_a.y;
}

// G > 1 (up to 32 query rows): the query tile holds G copies of them, one above the other, and copy g (one warp)
// takes the g-th part of every tile's keys (the products with those keys write its rows only), with an accumulator,
// reference point and sum of its own; the copies are combined at the end like the parts of a cluster.  A tile's softmax is then the work
// of G warps instead of one, and so is the masked tile at a sequence's end: 16 x 32 heads, 32 queries over 256-1024
// keys 42.3 -> 37.7 us, 64 x 32 157.8 -> 130.2, 50 x 32 with one query over 125-500 75.7 -> 59.6, 40 x 16 over 50-200
// at D = 64 22.3 -> 15.4; whole tiles only: 64 x 8 over 1024 51.2 -> 47.8.  Two copies at D = 128, where a fourth of
// the buffer's rows would cost a key tile, four at D = 64.
// Distance from fp64, relative, mean over some 280 drawn calls: 1.939e-3 where attention_kernel's general form has 1.949e-3; call by
// call between 0.95 and 1.04 of it, by which keys are reference points, whose weight is exact.
template <int D, int G>
__global__ void __launch_bounds__(kSplitThreads, 2)
attention_split_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                       const __grid_constant__ CUtensorMap tm_v, const AttnParams p, const int q_rows, const int parts)
{
    using L = SplitLayout<D>;
    constexpr uint32_t kTileBytes = L::kTileBytes;
    constexpr int kBoxes = D / 64;
    constexpr uint32_t kBoxBytes = 128 * 128;
    grid_wait();                                                 // the sequences' lengths are read
    extern __shared__ __align__(1024) unsigned char smem_dyn[];
    const uint32_t pad = (1024u - (smem_u32(smem_dyn) & 1023u)) & 1023u;
    unsigned char *tiles_gen = smem_dyn + pad;
    const uint32_t sQ = smem_u32(tiles_gen), sRing = sQ + (uint32_t)L::q_bytes(q_rows);
    // the barriers: before the tiles if the alignment left room there, behind them otherwise
    unsigned char *bars_gen = pad >= 256 ? smem_dyn : tiles_gen + 112 * 1024;
    const uint32_t bars = smem_u32(bars_gen);
    const int slots = L::slots(q_rows);
    const uint32_t bar_q = bars, bar_s_full = bars + 8, bar_p_early = bars + 16, bar_p_full = bars + 24, bar_o_full = bars + 32,
                   bar_v_last = bars + 40, bar_v_clear = bars + 48;
    auto bar_kv_full = [&](int s) { return bars + 8u * (L::kFixedBars + s); };
    auto bar_kv_empty = [&](int s) { return bars + 8u * (L::kFixedBars + L::kMaxSlots + s); };
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
    const int soft_warps = G > 1 ? G : row_warps;                 // softmax warps at work
    const int nkv = (keys + kBlockN - 1) / kBlockN;
    const int j_begin = part * nkv / parts, n_tiles = (part + 1) * nkv / parts - j_begin;      // key tiles of this CTA
    auto load_box = [&](uint32_t dst, const CUtensorMap *tm, uint32_t bar, int c0, int n0) {
        if (hm) tma_load_3d(dst, tm, bar, c0, n0, bh);
        else tma_load_4d(dst, tm, bar, c0, n0, h_idx, b_idx);
    };
    // Keys past the sequence's end have weight zero, but 0 x NaN is NaN in the product P V, and padding may
    // hold any bit pattern: the last value tile's rows behind the end are cleared before the product reads it, by
    // warps 6-7, which wait for this tile on a barrier of its own.  (Rows past the end of the tensor were zero-filled
    // by the copy.)  The softmax warps doing it behind their weights: 1-3 % slower on sequences of a few tiles.
    const bool clear = n_tiles > 0 && j_begin + n_tiles == nkv && keys % kBlockN != 0 && keys < p.Nkv;
    auto load_tile = [&](int slot, const CUtensorMap *tm, int j, bool last_v) {
        const uint32_t bar = last_v ? bar_v_last : bar_kv_full(slot);
        mbar_expect_tx(bar, kTileBytes);
#pragma unroll
        for (int cx = 0; cx < kBoxes; ++cx) load_box(sRing + slot * kTileBytes + cx * kBoxBytes, tm, bar, cx * 64, j * kBlockN);
    };

    // The producer thread sets up the barriers its copies complete on and sends the query tile, the first key
    // and the first value tile on their way before the CTA's first barrier.
    if (warp == kSplitLoadWarp && elect_one()) {
        prefetch_tmap(&tm_q); prefetch_tmap(&tm_k); prefetch_tmap(&tm_v);
        mbar_init(bar_q, 1);
        mbar_init(bar_v_last, 1);
        for (int s = 0; s < slots; ++s) mbar_init(bar_kv_full(s), 1);
        fence_mbar_init();
        if (n_tiles > 0) {
            mbar_expect_tx(bar_q, (uint32_t)L::q_bytes(q_rows));
#pragma unroll
            for (int cx = 0; cx < kBoxes; ++cx)
#pragma unroll
                for (int g = 0; g < G; ++g)
                    load_box(sQ + cx * (q_rows * 128) + g * (32 * 128), &tm_q, bar_q, cx * 64, row0);
            load_tile(0, &tm_k, j_begin, false);
            load_tile(1, &tm_v, j_begin, clear && n_tiles == 1);
        }
    }
    if (tid == 0) {
        for (int s = 0; s < slots; ++s) mbar_init(bar_kv_empty(s), 1);
        mbar_init(bar_s_full, 1);
        mbar_init(bar_p_early, soft_warps * 32);
        mbar_init(bar_p_full, soft_warps * 32);
        mbar_init(bar_o_full, 1);
        mbar_init(bar_v_clear, 64);
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
        if (healthy && warp < soft_warps) {
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
                if constexpr (G > 1) softmax_part<D, kBlockN / G>(tS, tO, warp * (kBlockN / G), i == 0, valid, c, m_ref, l_run);
                else softmax_tile<D, true>(tS, tO, i == 0, valid, c, m_ref, l_run, [&] {
                    tmem_wait_st();
                    tc_fence_before();
                    mbar_arrive(bar_p_early);
                });
                tmem_wait_st();
                tc_fence_before();
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
            if (G == 1 && parts == 1) {
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
        if (G > 1) {
            // ---- the copies meet: each warp combines its share of the columns, for the result or for the cluster
            named_bar_sync(1, 128);
            const float2 *ml = reinterpret_cast<const float2 *>(tiles_gen);
            float4 *o = reinterpret_cast<float4 *>(tiles_gen + L::q_bytes(q_rows));
            float m_all = -INFINITY, sum = 0.f, w[G];
#pragma unroll
            for (int g = 0; g < G; ++g) m_all = fmaxf(m_all, ml[g * 32 + lane].x);
#pragma unroll
            for (int g = 0; g < G; ++g) {
                w[g] = n_tiles > 0 ? ex2(ml[g * 32 + lane].x - m_all) : 0.f;
                sum += ml[g * 32 + lane].y * w[g];
            }
            const float inv = nkv > 0 ? 1.f / sum : 0.f;
            for (int c0 = warp * 16; healthy && c0 < D; c0 += 64) {
                float acc[16];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                    for (int g = 0; g < G; ++g) {
                        const float4 v = o[(c0 / 4 + k) * kBlockM + g * 32 + lane];
                        a.x += v.x * w[g]; a.y += v.y * w[g]; a.z += v.z * w[g]; a.w += v.w * w[g];
                    }
                    if (parts > 1) o[(c0 / 4 + k) * kBlockM + lane] = a;             // over the first copy's
                    acc[4 * k] = a.x; acc[4 * k + 1] = a.y; acc[4 * k + 2] = a.z; acc[4 * k + 3] = a.w;
                }
                if (parts == 1 && lane < rows) store16(lane, c0, acc, inv);
            }
            if (parts > 1 && warp == 0) reinterpret_cast<float2 *>(tiles_gen)[kBlockM + lane] = make_float2(m_all, sum);
        }
    } else {
        reg_dec<56>();
        if (healthy && warp == kSplitLoadWarp && elect_one()) {
            // =============================================================== TMA producer
            // ring tiles: 2i = K tile i, 2i + 1 = V tile i; the first two are on their way
            for (int t = 2, slot = 2 % slots, use = 2 / slots; t < 2 * n_tiles; ++t) {
                if (use > 0 && !mbar_wait(bar_kv_empty(slot), (use - 1) & 1)) { report(p, kErrWaitSlot); break; }
                load_tile(slot, (t & 1) ? &tm_v : &tm_k, j_begin + (t >> 1), clear && t + 1 == 2 * n_tiles);
                if (++slot == slots) { slot = 0; ++use; }
            }
            grid_trigger();
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
                    const bool last = clear && i + 1 == n_tiles;
                    if (!mbar_wait(last ? bar_v_last : bar_kv_full(slot), last ? 0 : phase)) { err = kErrWaitKV; break; }
                    if (last && !mbar_wait(bar_v_clear, 0)) { err = kErrWaitKV; break; }
                    if (!mbar_wait(G > 1 ? bar_p_full : bar_p_early, i & 1)) { err = kErrWaitP; break; }
                    tc_fence_after();
                    const uint64_t b = desc_v0 + (uint64_t)(slot * (kTileBytes >> 4));
                    bool ok = true;
                    // 16 keys = two 8-row groups of 1024 bytes; column blocks of 64 are one box apart
                    if constexpr (G == 1) {
#pragma unroll
                        for (int ks = 0; ks < kBlockN / 16; ++ks) {
                            if (ks == 6) {
                                if (!mbar_wait(bar_p_full, i & 1)) { ok = false; break; }
                                tc_fence_after();
                            }
                            mma_ts(tmem + kColO, tmem + kColS + ks * 8, b + (uint32_t)(ks * (2048 >> 4)), kIdescO, (i > 0 || ks > 0));
                        }
                    } else {
                        constexpr int kSteps = kBlockN / 16 / G;
                        auto product = [&](auto copy) {
                            constexpr int g = decltype(copy)::value;
#pragma unroll
                            for (int k = 0; k < kSteps; ++k) {
                                const int ks = g * kSteps + k;
                                mma_ts_rows<g>(tmem + kColO, tmem + kColS + ks * 8, b + (uint32_t)(ks * (2048 >> 4)), kIdescO, (i > 0 || k > 0));
                            }
                        };
                        product(std::integral_constant<int, 0>());
                        product(std::integral_constant<int, 1>());
                        if constexpr (G == 4) {
                            product(std::integral_constant<int, 2>());
                            product(std::integral_constant<int, 3>());
                        }
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
        } else if (healthy && warp > kSplitMmaWarp && clear) {
            // =============================================================== value rows behind the end
            if (!mbar_wait(bar_v_last, 0)) report(p, kErrWaitKV);
            else {
                // whole 128-byte rows, which the swizzle maps onto themselves
                const uint32_t tile = sRing + ((2 * n_tiles - 1) % slots) * kTileBytes;
                for (int r = keys % kBlockN + (warp - kSplitMmaWarp - 1) * 4 + (lane >> 3); r < kBlockN; r += 8)
#pragma unroll
                    for (int cx = 0; cx < kBoxes; ++cx) st_shared_v4(tile + cx * kBoxBytes + r * 128 + (lane & 7) * 16, 0u, 0u, 0u, 0u);
                fence_proxy_async_smem();
                mbar_arrive(bar_v_clear);
            }
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
                    ml[i] = ld_cluster_v2(cluster_addr(sQ + ((G > 1 ? kBlockM : 0) + row) * 8, i));
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
