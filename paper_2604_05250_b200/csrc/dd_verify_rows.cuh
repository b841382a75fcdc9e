// Row kernel of dd_verify: a row per warp, CTA or cluster (16-byte aligned logits, any V).
//
// The streaming kernel is built for the bandwidth of large problems and pays for it at the start (flag
// scan, ranges, rings) and at the end (partials of cut rows, publishing warp, a decision by one warp): 10 us
// on the smallest problem, 20 where the logits take 5-10 us to read.  Here the pieces of a row are read
// straight into registers by `wpr` warps in turn (1, 2, 4 or 8, so that a CTA has 8 / wpr rows) or by the
// eight warps of each CTA of a cluster; the arithmetic per piece and per lane is the streaming kernel's.
// One warp folds the row's partials from shared memory (the cluster's first CTA reads its peers'), the CTA
// reports its rows to their sequences (one fence and one counter update per CTA and sequence), and the CTA
// that completes a sequence decides it with all its threads.  Results do not depend on which CTA runs when.
#pragma once

#include "dd_ptx.cuh"
#include "dd_verify_decide_block.cuh"
#include "dd_verify_stream.cuh"

namespace ddv {

constexpr int kRWarps = 8;
constexpr int kRMaxCluster = 8;

__device__ __forceinline__ uint4 ld_streamed(const uint16_t *ptr, uint64_t policy)
{
    uint4 r;
    asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.v4.u32 {%0,%1,%2,%3}, [%4], %5;"
                 : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "l"(ptr), "l"(policy));
    return r;
}

// The same where `wanted`, under a predicate: a branch would make the warp wait for its loads where the paths meet.
__device__ __forceinline__ void ld_streamed_if(uint4 &r, const uint16_t *ptr, uint64_t policy, bool wanted)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %6, 0;\n\t"
                 "@p ld.global.nc.L1::no_allocate.L2::cache_hint.v4.u32 {%0,%1,%2,%3}, [%4], %5;\n\t}"
                 : "+r"(r.x), "+r"(r.y), "+r"(r.z), "+r"(r.w) : "l"(ptr), "l"(policy), "r"((int)wanted));
}

struct RowsShape {
    int wpr;          // warps per row
    int cluster;      // CTAs per row (then wpr is 8)
    int mapped;       // 1: flagged rows first (mapped_row; wpr is 8, no cluster)
};

// Lowest finite bf16 in both halves: what stands where a piece has no logit.  Its weight is 0, its term in T is an exact 0, and
// it is no maximum unless every logit is lower, which the scalar routine sorts out.
constexpr uint32_t kAbsent2 = 0xFF7FFF7Fu;
constexpr float kLowestLogit = -3.38e38f;        // (bf16's lowest finite is -3.3895e38)

// A piece: lane_pass1 and lane_pass2 in one, for registers that are all filled.  Logits are not raised to finite ones beforehand, which
// only excluded tokens (-inf) need: their terms of T come out as NaN or infinity, and then the lane computes the piece's
// terms again that way.
// A warp's share of a row is up to kLongShare pieces, twice a chunk of the streaming kernel and more, and its sums must not be less
// exact for that.  KL: a piece is summed by itself and added to the lane's sums.  Else the chains are sum_v, which the pieces use in turn: half of
// them go through the caller's second one (adding each piece's sum cost 3 to 14 % there).  256 rows of 126464, mean error of KL relative
// to 64 bits 5.6e-8 as one chain, 4.3e-8 so and in the streaming kernel; no difference in time.
template <bool KL>
__device__ __forceinline__ void lane_piece(LaneState &L, float2 &sum_v, const uint4 (&rv)[kVecPerThread], const uint4 (&rd)[kVecPerThread], int ordinal, bool first)
{
    lane_pass1<KL>(L, rv, rd, ordinal, first);
    if (first) {
        // a lane without a logit has a finite reference point all the same
        L.M_v = fmaxf(L.M_v, -1e30f);
        if (KL) L.M_d = fmaxf(L.M_d, -1e30f);
    }
    const float2 log2e2 = make_float2(kLog2e, kLog2e), neg1 = make_float2(-1.f, -1.f);
    const float2 nMv2 = make_float2(-L.M_v, -L.M_v), nMd2 = make_float2(-L.M_d, -L.M_d);
    const float2 zero = make_float2(0.f, 0.f);
    float2 s_v = KL ? zero : sum_v, s_d = zero, t = zero;
#pragma unroll
    for (int j = 0; j < (KL ? 1 : 2) * kVecPerThread; ++j) {
        const uint4 &x = j < kVecPerThread ? rv[j] : rd[j - kVecPerThread];
        const uint32_t wv[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            const float2 v2 = make_float2(bf16lo(wv[h]), bf16hi(wv[h]));
            const float2 a = __ffma2_rn(v2, log2e2, nMv2);
            s_v = __fadd2_rn(s_v, make_float2(ex2_approx(a.x), ex2_approx(a.y)));
            if (KL) {
                const uint32_t wd[4] = {rd[j].x, rd[j].y, rd[j].z, rd[j].w};
                const float2 d2 = make_float2(bf16lo(wd[h]), bf16hi(wd[h]));
                const float2 b = __ffma2_rn(d2, log2e2, nMd2);
                const float2 e2 = make_float2(ex2_approx(b.x), ex2_approx(b.y));
                s_d = __fadd2_rn(s_d, e2);
                t = __ffma2_rn(e2, __ffma2_rn(v2, neg1, d2), t);          // e * (d - v)
            }
        }
    }
    if (KL && !isfinite(t.x + t.y)) {
        // Both logits raised to the lowest finite one: a token that the drafter excludes adds an exact 0, one that only the verifier
        // excludes e * 3.4e38 (kExcludedExcess).
        t = zero;
#pragma unroll 1
        for (int j = 0; j < kVecPerThread; ++j) {
            uint4 v = rv[0], d = rd[0];
#pragma unroll
            for (int i = 1; i < kVecPerThread; ++i)
                if (i == j) { v = rv[i]; d = rd[i]; }
            const uint32_t wv[4] = {v.x, v.y, v.z, v.w}, wd[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                const uint32_t w = bf16x2_max(wv[h], kAbsent2), e = bf16x2_max(wd[h], kAbsent2);
                const float2 v2 = make_float2(bf16lo(w), bf16hi(w)), d2 = make_float2(bf16lo(e), bf16hi(e));
                const float2 b = __ffma2_rn(d2, log2e2, nMd2);
                t = __ffma2_rn(make_float2(ex2_approx(b.x), ex2_approx(b.y)), __ffma2_rn(v2, neg1, d2), t);
            }
        }
    }
    if (KL) {
        L.s_v = __fadd2_rn(L.s_v, s_v);
        L.s_d = __fadd2_rn(L.s_d, s_d);
        L.t = __fadd2_rn(L.t, t);
    } else {
        sum_v = s_v;
    }
}

// The part of a row that one warp takes: the pieces at x0, x0 + stride, ... (logits, counted from the row's first vector), from
// global memory straight into registers.  Few pieces to a warp: little code, which is cold.
template <bool KL>
__device__ __forceinline__ Partial row_part(const VerifyParams &p, int row, int x0, int stride)
{
    constexpr int kStep = PieceOf<KL>::value;
    const int lane = threadIdx.x & 31;
    const long n_rows = (long)p.B * p.P;
    LaneState L;
    lane_reset(L);
    const int head = row_head(row, p.V), extent = head + p.V;      // from the row's first vector on
    const size_t off = (size_t)row * p.V - head;
    // what the tensor holds from there on, as far as the row's vectors reach: a vector that goes beyond is not loaded
    // whole (the last row's last one; of fewer than eight logits also that of the rows before it)
    const int present = (int)min(n_rows * p.V - (long)off, (long)extent + 7);
    const uint16_t *ver = p.verifier + off, *dra = KL ? p.drafter + off : p.verifier + off;
    const uint64_t policy = l2_evict_first_policy();
    int ordinal = 0;
#pragma unroll 1
    for (int x = x0; x < extent; x += stride, ++ordinal) {
        const int n = min(kStep, extent - x), whole = min((n + 7) & ~7, present - x);      // logits in vectors loaded whole
        uint4 rv[kVecPerThread], rd[kVecPerThread];
        const uint4 ninf = make_uint4(0xFF80FF80u, 0xFF80FF80u, 0xFF80FF80u, 0xFF80FF80u);
        auto load = [&](const uint16_t *src, int vec) {
            const int e = vec * 8;
            if (e + 8 > whole) return ninf;
            return ld_streamed(src + checked_run(p, x + e, 8, n_rows * p.V - (long)off, kSiteLogit), policy);
        };
#pragma unroll
        for (int j = 0; j < kVecPerThread; ++j) {
            rv[j] = load(ver, lane + 32 * j);
            rd[j] = load(dra, lane + 32 * (KL ? j : kVecPerThread + j));
        }
        if (n < kStep || (head != 0 && x == 0)) {
            // the vectors that the row shares with its neighbours, and one that the tensor does not fill
            const int from = x == 0 ? head : 0;
            auto edge = [&](uint4 &r, int vec, const uint16_t *src) {
                const int e0 = vec * 8;
                if (e0 >= n || (e0 + 8 <= n && e0 >= from)) return;
                uint32_t w[4] = {r.x, r.y, r.z, r.w};
                const bool apart = e0 + 8 > whole;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int e = e0 + i;
                    uint32_t v = i & 1 ? w[i / 2] >> 16 : w[i / 2] & 0xFFFFu;
                    if (apart && e < n) v = __ldg(src + checked(p, x + e, n_rows * p.V - (long)off, kSiteLogit));
                    if (e >= n || e < from) v = 0xFF80u;
                    w[i / 2] = i & 1 ? (w[i / 2] & 0xFFFFu) | v << 16 : (w[i / 2] & 0xFFFF0000u) | v;
                }
                r = make_uint4(w[0], w[1], w[2], w[3]);
            };
#pragma unroll
            for (int j = 0; j < kVecPerThread; ++j) {
                edge(rv[j], lane + 32 * j, ver);
                edge(rd[j], lane + 32 * (KL ? j : kVecPerThread + j), dra);
            }
        }
        lane_pass1<KL>(L, rv, rd, ordinal, ordinal == 0);
        if (n == kStep) lane_pass2<KL, true>(L, rv, rd, n, lane);
        else lane_pass2<KL, false>(L, rv, rd, n, lane);
    }
    Partial part = lanes_to_partial<KL>(L, x0 - head, lane, stride);
    if (x0 < extent &&
        (!(isfinite(part.s_v) && isfinite(part.s_d) && isfinite(part.t) && part.m_v > -INFINITY) ||
         (KL && fabsf(part.t) > kExcludedExcess * part.s_d))) {
        // the scalar routine, piece by piece
        const size_t row_off = (size_t)row * p.V;
        for (int x = x0, i = 0; x < extent; x += stride, ++i) {
            const Partial c = careful_chunk_partial<KL>(p.verifier + row_off, KL ? p.drafter + row_off : nullptr,
                                                        max(0, x - head), min(p.V, x - head + kStep));
            if (i == 0) part = c;
            else merge_partial<KL>(part, c);
        }
    }
    return part;
}

// The same with more than a few pieces to a warp: the next one is on its way while one is worked on, pieces that are all there are loaded
// without a comparison per vector, and -inf is dealt with where it occurs (lane_piece).  The pieces' loop holds no branch around a
// load.  1 x 256 positions, V = 126464, KL (363 instructions a piece; in the short form 470, one piece at a time): 36.8 -> 29.9 us; 1 x 128
// 23.9 -> 20.4; 1 x 400, half flagged, CONF 25.4 -> 19.9.
template <bool KL>
__device__ __forceinline__ Partial row_part_deep(const VerifyParams &p, int row, int x0, int stride)
{
    constexpr int kStep = PieceOf<KL>::value;
    const int lane = threadIdx.x & 31;
    const long n_rows = (long)p.B * p.P;
    LaneState L;
    lane_reset(L);
    const int head = row_head(row, p.V), extent = head + p.V;      // from the row's first vector on
    const size_t off = (size_t)row * p.V - head;
    // what the tensor holds from there on, as far as the row's vectors reach: a vector that goes beyond is not loaded
    // whole (the last row's last one; of fewer than eight logits also that of the rows before it)
    const long left = n_rows * p.V - (long)off;
    const int present = (int)min(left, (long)extent + 7);
    const uint16_t *ver = p.verifier + off, *dra = KL ? p.drafter + off : p.verifier + off;
    const uint64_t policy = l2_evict_first_policy();
    auto load_full = [&](uint4 (&rv)[kVecPerThread], uint4 (&rd)[kVecPerThread], int x, bool wanted) {
        const size_t at = (wanted ? checked_run(p, x, kStep, left, kSiteLogit) : 0) + lane * 8;
#pragma unroll
        for (int j = 0; j < kVecPerThread; ++j) {
            ld_streamed_if(rv[j], ver + at + 256 * j, policy, wanted);
            ld_streamed_if(rd[j], dra + at + 256 * (KL ? j : kVecPerThread + j), policy, wanted);
        }
    };
    auto load_edge = [&](uint4 (&rv)[kVecPerThread], uint4 (&rd)[kVecPerThread], int x) {
        const int n = extent - x;
        // the row's ends: vectors that it shares with its neighbours, that the tensor does not fill, or beyond both
        const int whole = min((min(n, kStep) + 7) & ~7, present - x), from = x == 0 ? head : 0;
        auto load = [&](uint4 &r, const uint16_t *src, int vec) {
            const int e0 = vec * 8;
            const bool there = e0 + 8 <= whole;
            r = make_uint4(kAbsent2, kAbsent2, kAbsent2, kAbsent2);
            ld_streamed_if(r, src + (there ? checked_run(p, x + e0, 8, left, kSiteLogit) : 0), policy, there);
        };
#pragma unroll
        for (int j = 0; j < kVecPerThread; ++j) {
            load(rv[j], ver, lane + 32 * j);
            load(rd[j], dra, lane + 32 * (KL ? j : kVecPerThread + j));
        }
        auto trim = [&](uint4 &r, const uint16_t *src, int vec) {
            const int e0 = vec * 8;
            if (e0 >= n || (e0 + 8 <= n && e0 >= from)) return;
            const bool apart = e0 + 8 > whole;
            uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int e = e0 + i;
                uint32_t v = i & 1 ? w[i / 2] >> 16 : w[i / 2] & 0xFFFFu;
                if (apart && e < n) v = __ldg(src + checked(p, x + e, left, kSiteLogit));
                if (e >= n || e < from) v = kAbsent2 & 0xFFFFu;
                w[i / 2] = i & 1 ? (w[i / 2] & 0xFFFFu) | v << 16 : (w[i / 2] & 0xFFFF0000u) | v;
            }
            r = make_uint4(w[0], w[1], w[2], w[3]);
        };
#pragma unroll
        for (int j = 0; j < kVecPerThread; ++j) {
            trim(rv[j], ver, lane + 32 * j);
            trim(rd[j], dra, lane + 32 * (KL ? j : kVecPerThread + j));
        }
    };
    float2 second = make_float2(0.f, 0.f);               // the other chain (lane_piece)
    uint4 av[kVecPerThread], ad[kVecPerThread];
#pragma unroll
    for (int j = 0; j < kVecPerThread; ++j) av[j] = ad[j] = make_uint4(0u, 0u, 0u, 0u);
    int x = x0, ordinal = 0;
    auto edge = [&] {
        load_edge(av, ad, x);
        lane_piece<KL>(L, L.s_v, av, ad, ordinal, ordinal == 0);
        x += stride;
        ++ordinal;
    };
    if (head != 0 && x0 == 0) edge();
    auto full = [&](int x) { return x + kStep <= extent; };
    if (full(x)) {
        load_full(av, ad, x, true);
        uint4 bv[kVecPerThread], bd[kVecPerThread];
#pragma unroll
        for (int j = 0; j < kVecPerThread; ++j) bv[j] = bd[j] = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll 1
        for (;;) {
            x += stride;
            load_full(bv, bd, x, full(x));
            lane_piece<KL>(L, L.s_v, av, ad, ordinal, ordinal == 0);
            ++ordinal;
            if (!full(x)) break;
            x += stride;
            load_full(av, ad, x, full(x));
            lane_piece<KL>(L, second, bv, bd, ordinal, false);
            ++ordinal;
            if (!full(x)) break;
        }
    }
    if (x < extent) edge();
    if (!KL) L.s_v = __fadd2_rn(L.s_v, second);
    Partial part = lanes_to_partial<KL>(L, x0 - head, lane, stride);
    if (x0 < extent &&
        (!(isfinite(part.s_v) && isfinite(part.s_d) && isfinite(part.t) && part.m_v > kLowestLogit) ||
         (KL && (fabsf(part.t) > kExcludedExcess * part.s_d || !(part.m_d > kLowestLogit))))) {
        // the scalar routine, piece by piece
        const size_t row_off = (size_t)row * p.V;
        for (int x = x0, i = 0; x < extent; x += stride, ++i) {
            const Partial c = careful_chunk_partial<KL>(p.verifier + row_off, KL ? p.drafter + row_off : nullptr,
                                                        max(0, x - head), min(p.V, x - head + kStep));
            if (i == 0) part = c;
            else merge_partial<KL>(part, c);
        }
    }
    return part;
}

// The row that stands for CTA v: the flagged rows come first, in order, then the others, so that the former are spread evenly over
// the SMs: two long rows on one SM take 23 us where one takes 14 (126464 logits, KL), and by their places that happens long before
// there are more of them than SMs.  1 x 256 positions, V = 126464, KL, 25 % flagged 29.0 -> 22.3 us, 50 % 29.5 -> 23.3; 2 x 300, 32001, 25 % 19.0 ->
// 16.3; where all are flagged it costs some 0.3 us.  Up to kMappedRows rows; every thread of the CTA calls it.
constexpr int kMappedRows = 1024;
__device__ __forceinline__ int mapped_row(const VerifyParams &p, int v, uint32_t (&words)[kMappedRows / 32], bool &flagged)
{
    const unsigned full = 0xFFFFFFFFu;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n = p.B * p.P;
    bool f[kMappedRows / 32 / kRWarps];
#pragma unroll
    for (int i = 0; i < kMappedRows / 32 / kRWarps; ++i) {
        const int r = (warp + i * kRWarps) * 32 + lane;
        f[i] = r < n && p.flags[checked(p, min(r, n - 1), n, kSiteFlag)] != 0;
    }
#pragma unroll
    for (int i = 0; i < kMappedRows / 32 / kRWarps; ++i) {
        const uint32_t b = __ballot_sync(full, f[i]);
        if (lane == 0) words[warp + i * kRWarps] = b;
    }
    __syncthreads();
    // a word to a lane: its flagged rows, or the others
    uint32_t m = words[lane];
    int incl = __popc(m);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(full, incl, o);
        if (lane >= o) incl += u;
    }
    const int all = __shfl_sync(full, incl, 31);
    flagged = v < all;
    int rank = v;
    if (!flagged) {
        rank -= all;
        m = ~m;                                          // (beyond the last row too: those come last)
        incl = 32 * (lane + 1) - incl;
    }
    const int src = __ffs(__ballot_sync(full, rank < incl)) - 1;
    const uint32_t word = __shfl_sync(full, m, src);
    rank -= __shfl_sync(full, incl - __popc(m), src);
    const bool here = (word >> lane & 1u) && __popc(word & ((1u << lane) - 1u)) == rank;
    return src * 32 + __ffs(__ballot_sync(full, here)) - 1;
}

// kDeep: row_part_deep, whose registers leave room for two CTAs on an SM instead of three.
template <bool KL, bool kDeep>
__global__ void __launch_bounds__(32 * kRWarps, kDeep ? 2 : 3) verify_rows_kernel(const __grid_constant__ VerifyParams p, const RowsShape shape)
{
    __shared__ __align__(16) Partial s_part[kRWarps];
    __shared__ __align__(16) Partial s_all[kRMaxCluster * kRWarps];
    __shared__ BlockReport s_report;
    __shared__ uint32_t s_words[kMappedRows / 32];
    ddptx::grid_wait();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const long n_rows = (long)p.B * p.P;
    const int wpr = shape.wpr, cluster = shape.cluster;
    const int rank = cluster > 1 ? (int)(blockIdx.x % (unsigned)cluster) : 0;
    const int rows_here = kRWarps / wpr;                            // 1 in a cluster
    int row0 = (int)(blockIdx.x / (unsigned)cluster) * rows_here;
    bool mine = false;
    if (shape.mapped) row0 = mapped_row(p, row0, s_words, mine);
    const int row = row0 + warp / wpr;                              // this warp's row
    const int first = rank * kRWarps + warp % wpr;                  // its first piece, and how far apart the next ones are
    constexpr int kStep = PieceOf<KL>::value;
    const int stride = cluster * wpr * kStep;
    if (!shape.mapped) mine = row < n_rows && p.flags[checked(p, row, n_rows, kSiteFlag)] != 0;

    if (mine) {
        const Partial part = kDeep ? row_part_deep<KL>(p, row, first * kStep, stride) : row_part<KL>(p, row, first * kStep, stride);
        if (lane == 0) s_part[warp] = part;
        __syncwarp();
        if (wpr > 1 && cluster == 1) cta_bar_sync(1 + warp / wpr, 32 * wpr);
    }
    ddptx::grid_trigger();
    const int pieces = (row_head(row, p.V) + p.V + kStep - 1) / kStep;
    const Partial *parts = s_part + warp - warp % wpr;
    if (cluster > 1) {
        // (the flag is the same in the whole cluster)
        if (mine) {
            ddptx::cluster_arrive();
            ddptx::cluster_wait();
            if (rank == 0 && warp == 0) {
                // 32 bytes of every warp of the cluster, in the order of their pieces
                for (int i = lane; i < cluster * kRWarps; i += 32) {
                    const uint32_t src = ddptx::cluster_addr(s_addr(s_part + i % kRWarps), i / kRWarps);
                    reinterpret_cast<float4 *>(s_all + i)[0] = ddptx::ld_cluster_v4(src);
                    reinterpret_cast<float4 *>(s_all + i)[1] = ddptx::ld_cluster_v4(src + 16);
                }
                __syncwarp();
            }
            ddptx::cluster_arrive();                                 // a peer's shared memory outlives its reads
            ddptx::cluster_wait();
        }
        if (rank != 0) return;
        parts = s_all;
    }
    if (mine && warp % wpr == 0) {
        float score;
        int argmax;
        fold_partials<KL, true>(parts, min(cluster * wpr, pieces), score, argmax);
        if (lane == 0) {
            __stcg(p.row_score + row, score);
            __stcg(p.row_argmax + row, argmax);
        }
    }
    report_rows(p, row0, rows_here, s_report);
}

}  // namespace ddv
