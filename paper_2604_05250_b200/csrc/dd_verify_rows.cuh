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

struct RowsShape {
    int wpr;          // warps per row
    int cluster;      // CTAs per row (then wpr is 8)
};

template <bool KL>
__global__ void __launch_bounds__(32 * kRWarps, 3) verify_rows_kernel(const __grid_constant__ VerifyParams p, const RowsShape shape)
{
    __shared__ __align__(16) Partial s_part[kRWarps];
    __shared__ __align__(16) Partial s_all[kRMaxCluster * kRWarps];
    __shared__ BlockReport s_report;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const long n_rows = (long)p.B * p.P;
    const int wpr = shape.wpr, cluster = shape.cluster;
    const int rank = cluster > 1 ? (int)(blockIdx.x % (unsigned)cluster) : 0;
    const int rows_here = kRWarps / wpr;                            // 1 in a cluster
    const int row0 = (int)(blockIdx.x / (unsigned)cluster) * rows_here;
    const int row = row0 + warp / wpr;                              // this warp's row
    const int first = rank * kRWarps + warp % wpr;                  // its first piece, and how far apart the next ones are
    constexpr int kStep = PieceOf<KL>::value;
    const int stride = cluster * wpr * kStep;
    const bool mine = row < n_rows && p.flags[checked(p, row, n_rows, kSiteFlag)] != 0;

    if (mine) {
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
        for (int x = first * kStep; x < extent; x += stride, ++ordinal) {
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
        Partial part = lanes_to_partial<KL>(L, first * kStep - head, lane, stride);
        if (first * kStep < extent &&
            (!(isfinite(part.s_v) && isfinite(part.s_d) && isfinite(part.t) && part.m_v > -INFINITY) ||
             (KL && fabsf(part.t) > kExcludedExcess * part.s_d))) {
            // the scalar routine, piece by piece
            const size_t row_off = (size_t)row * p.V;
            for (int x = first * kStep, i = 0; x < extent; x += stride, ++i) {
                const Partial c = careful_chunk_partial<KL>(p.verifier + row_off, KL ? p.drafter + row_off : nullptr,
                                                            max(0, x - head), min(p.V, x - head + kStep));
                if (i == 0) part = c;
                else merge_partial<KL>(part, c);
            }
        }
        if (lane == 0) s_part[warp] = part;
        __syncwarp();
        if (wpr > 1 && cluster == 1) cta_bar_sync(1 + warp / wpr, 32 * wpr);
    }
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
        fold_partials<KL>(parts, min(cluster * wpr, pieces), score, argmax);
        if (lane == 0) {
            __stcg(p.row_score + row, score);
            __stcg(p.row_argmax + row, argmax);
        }
    }
    report_rows(p, row0, rows_here, s_report);
}

}  // namespace ddv
