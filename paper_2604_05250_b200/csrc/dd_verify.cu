// dd_verify: the verification algorithm A(p_D, p_V, x^D) of Algorithm 1
// (Section 3.2) as one memory-bound kernel launch.
//
// Work decomposition.  A flagged row (one position of the drafter-decoded set)
// is V logits from the verifier and, in KL mode, V from the drafter.  The row is
// cut into chunks; every (row, chunk) yields one partial
//     m_V, S_V = sum 2^(l_V*log2e - M_V), lowest index of the maximum,
//     m_D, S_D = sum 2^(l_D*log2e - M_D), T = sum 2^(l_D*log2e - M_D) (l_D - l_V)
// (M = m*log2e rounded once; any reference works as long as it is reused), and
// each logit is read from HBM exactly once.
//
// Row kernel (16-byte aligned logits, any V, small and middle-sized problems; dd_verify_rows.cuh): a row per
// warp, CTA or cluster, read straight into registers.
// Streaming kernel (the same, large problems; dd_verify_stream.cuh):
// persistent CTAs; a producer warp feeds per-warp rings in shared memory with bulk
// asynchronous copies, consumer warps accumulate chunks of up to 8192 logits from
// them, a publishing warp counts, folds and decides.
// Element-wise kernel (logits off 16-byte boundaries; this file): one CTA of 256 threads
// per chunk of at most 8192 logits, 2-byte loads with bounds checks.
//
// The warp that sees a row's last chunk folds the row's chunk partials in chunk
// order in fp64 into  c_i = 2^(..)/S_V  (Eq. 7)  and
//     KL_i = T/S_D - lse_D + lse_V                                   (Eq. 5)
// and the warp that sees a sequence's last row runs the decision stage for it:
// Eq. 6 normaliser, Philox uniforms, threshold / probabilistic rule, the
// minimum-keep top-k, and the emitted tokens.  "Last" is decided with
// __threadfence + atomic counters that the last arriver resets to zero, so the
// scratch is ready for the next launch; every fold runs in a fixed order, so the
// result does not depend on the order in which warps finish.
#include <stdio.h>

#include <algorithm>
#include <atomic>
#include <mutex>

#include "dd_verify_stream.cuh"
#include "dd_verify_rows.cuh"
#include "dd_lm_head_kernel.cuh"
#include "dd_lm_head_pair.cuh"

namespace {

using namespace ddv;

// ---------------------------------------------------------------------------
// Element-wise kernel.
constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kMaxChunk = kThreads * kVecPerThread * 8;       // 8192 logits

// The thread's share of a chunk of n logits: vectors t, t+256, t+512, t+768 (8 logits each),
// -inf beyond the chunk's end.
__device__ __forceinline__ void load_chunk_elementwise(const uint16_t *row, int n, int tid,
                                                       uint4 (&r)[kVecPerThread])
{
#pragma unroll
    for (int j = 0; j < kVecPerThread; ++j) {
        const int e0 = (tid + j * kThreads) * 8;
        uint32_t w[4];
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            const int a = e0 + 2 * h, b = a + 1;
            const uint32_t lo = a < n ? (uint32_t)__ldg(row + a) : 0xFF80u;
            const uint32_t hi = b < n ? (uint32_t)__ldg(row + b) : 0xFF80u;
            w[h] = lo | (hi << 16);
        }
        r[j] = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

__device__ __forceinline__ float vectors_max(const uint4 (&r)[kVecPerThread])
{
    __nv_bfloat162 m = __halves2bfloat162(__ushort_as_bfloat16(0xFF80), __ushort_as_bfloat16(0xFF80));
#pragma unroll
    for (int j = 0; j < kVecPerThread; ++j) {
        const uint32_t w[4] = {r[j].x, r[j].y, r[j].z, r[j].w};
#pragma unroll
        for (int h = 0; h < 4; ++h) m = __hmax2(m, *reinterpret_cast<const __nv_bfloat162 *>(&w[h]));
    }
    const uint32_t mw = *reinterpret_cast<uint32_t *>(&m);
    return fmaxf(bf16lo(mw), bf16hi(mw));
}

// Warp-level partial of the vectors the 32 lanes hold (thread t of kThreads; the chunk has n
// logits and starts at logit e_begin of the row).
template <bool KL>
__device__ __forceinline__ void warp_partial(const uint4 (&rv)[kVecPerThread], const uint4 (&rd)[kVecPerThread],
                                             int n, int e_begin, int t, Partial &out)
{
    const float m_v = warp_max(vectors_max(rv));
    float m_d = 0.f;
    if (KL) m_d = warp_max(vectors_max(rd));
    int idx = 0x7FFFFFFF;
#pragma unroll
    for (int j = kVecPerThread - 1; j >= 0; --j) {
        const uint32_t w[4] = {rv[j].x, rv[j].y, rv[j].z, rv[j].w};
#pragma unroll
        for (int h = 3; h >= 0; --h) {
            const int e = e_begin + (t + j * kThreads) * 8 + 2 * h;
            if (bf16hi(w[h]) == m_v) idx = e + 1;
            if (bf16lo(w[h]) == m_v) idx = e;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) idx = min(idx, __shfl_xor_sync(0xFFFFFFFFu, idx, o));

    // one ex2 per logit against the warp's reference
    const float M_v = m_v * kLog2e, M_d = m_d * kLog2e;
    float s_v0 = 0.f, s_v1 = 0.f, s_d0 = 0.f, s_d1 = 0.f, t0 = 0.f, t1 = 0.f;
#pragma unroll
    for (int j = 0; j < kVecPerThread; ++j) {
        const int e0 = (t + j * kThreads) * 8;
        if (e0 < n) {
            const uint32_t wv[4] = {rv[j].x, rv[j].y, rv[j].z, rv[j].w};
            uint32_t wd[4] = {0u, 0u, 0u, 0u};
            if (KL) { wd[0] = rd[j].x; wd[1] = rd[j].y; wd[2] = rd[j].z; wd[3] = rd[j].w; }
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                const bool ok0 = e0 + 2 * h < n, ok1 = e0 + 2 * h + 1 < n;
                const float v0 = bf16lo(wv[h]), v1 = bf16hi(wv[h]);
                // a logit of -inf is probability zero: no term (also when every logit of the warp is -inf)
                if (ok0 && v0 != -INFINITY) s_v0 += ex2_approx(fmaf(v0, kLog2e, -M_v));
                if (ok1 && v1 != -INFINITY) s_v1 += ex2_approx(fmaf(v1, kLog2e, -M_v));
                if (KL) {
                    const float d0 = bf16lo(wd[h]), d1 = bf16hi(wd[h]);
                    if (ok0 && d0 != -INFINITY) {
                        const float e = ex2_approx(fmaf(d0, kLog2e, -M_d));
                        s_d0 += e;
                        if (e > 0.f) t0 = fmaf(e, d0 - v0, t0);      // p_D = 0 contributes no term
                    }
                    if (ok1 && d1 != -INFINITY) {
                        const float e = ex2_approx(fmaf(d1, kLog2e, -M_d));
                        s_d1 += e;
                        if (e > 0.f) t1 = fmaf(e, d1 - v1, t1);
                    }
                }
            }
        }
    }
    out.m_v = m_v;
    out.s_v = warp_sum(s_v0 + s_v1);
    out.idx = idx;
    out.m_d = m_d;
    out.s_d = 0.f;
    out.t = 0.f;
    if (KL) {
        out.s_d = warp_sum(s_d0 + s_d1);
        out.t = warp_sum(t0 + t1);
    }
    out.pad0 = out.pad1 = 0.f;
}

constexpr int kEDecideKeys = 2048;      // keys of one sequence the element-wise kernel's deciding warp keeps in shared memory

template <bool KL>
__global__ void __launch_bounds__(kThreads, 3) verify_elementwise_kernel(const VerifyParams p)
{
    __shared__ Partial warp_part[kWarps];
    __shared__ uint32_t s_decide_keys[kEDecideKeys];   // decision stage (warp 0 only)
    DecideStage s_decide;
    s_decide.key = s_decide_keys;
    s_decide.capacity = kEDecideKeys;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int row = (int)checked(p, blockIdx.x / p.nchunks, (long)p.B * p.P, kSiteFlag);
    const int chunk = blockIdx.x - row * p.nchunks;

    if (!p.flags[row]) {
        // Unflagged rows cost nothing; warp 0 of their chunk-0 CTA reports the row as complete.
        if (chunk == 0 && warp == 0) row_done(p, row / p.P, &s_decide);
        return;
    }
    const int e_begin = chunk * p.chunk;
    const int n = min(p.chunk, p.V - e_begin);
    const size_t off = checked_run(p, (long)row * p.V + e_begin, n, (long)p.B * p.P * p.V, kSiteLogit);

    uint4 rv[kVecPerThread], rd[kVecPerThread];
    load_chunk_elementwise(p.verifier + off, n, tid, rv);
    if (KL) load_chunk_elementwise(p.drafter + off, n, tid, rd);
    Partial part;
    warp_partial<KL>(rv, rd, n, e_begin, tid, part);
    if (lane == 0) warp_part[warp] = part;
    __syncthreads();
    if (warp != 0) return;

    // warp 0 folds the eight warp partials in warp order (every lane the same arithmetic)
    Partial c = warp_part[0];
#pragma unroll
    for (int w = 1; w < kWarps; ++w) merge_partial<KL>(c, warp_part[w]);
    chunk_done<KL>(p, row, chunk, c, &s_decide);
}

// ---------------------------------------------------------------------------
// Host side.

// Counters live in their own allocation: it holds nothing else, so it is all zero whenever no
// launch is in flight, whatever (B, P) the previous call used.  Its last 256 bytes are not
// counters: they hold the health word and the plan of the fused heads.
constexpr size_t kControlBytes = 256;
constexpr size_t kStatusOffset = 0;
constexpr size_t kPlanOffset = 128;              // dd_lm_head_verify: what its kernels tell each other

size_t counter_bytes(int B, int P)
{
    const size_t bp = (size_t)B * P;
    return ((bp * 4 + 255) & ~size_t(255)) + (((size_t)B * 4 + 255) & ~size_t(255));
}

size_t workspace_bytes(int B, int P, int nchunks)
{
    const size_t bp = (size_t)B * P;
    size_t bytes = 0;
    bytes += (bp * 4 + 255) & ~size_t(255);           // row_score
    bytes += (bp * 4 + 255) & ~size_t(255);           // row_argmax
    bytes += bp * nchunks * sizeof(Partial);
    return bytes;
}

// Rows may start anywhere (V need not be a multiple of eight), the tensors themselves on 16 bytes.  V = 32001,
// 2 x 300 positions, half of them flagged, KL: element-wise kernel 41.5 us, streaming 37.6, row kernel 23.1;
// V = 50001, 8 x 256, CONF: element-wise 108, streaming 40.1.
bool streaming_path(const void *drafter, const void *verifier, bool kl)
{
    return ((uintptr_t)verifier & 15) == 0 && (!kl || ((uintptr_t)drafter & 15) == 0);
}

// Streaming path: stages per chunk (a chunk is the work of one warp and yields one partial).
// Four stages (16 KB of logits) keep the cost of ending a chunk small; fewer when the rows are
// too few to give every streaming warp of `sms` CTAs a couple of units; eight where every warp
// has many units anyway, or where the partials would not fit `max_partials` (0: no limit).
// The choice depends on the device, never on the grid actually launched.
int pick_pieces(int V, long rows, int sms, long max_partials, bool kl)
{
    const long step = kl ? kPiece : 2 * kPiece;
    auto chunks_of = [&](int k) { return (V + k * step - 1) / (k * step); };
    const int k_max = kl ? kMaxPiecesPerChunk : kMaxPiecesPerChunk / 2;      // 8192 logits either way
    int k = 4;
    const long want = 2L * kSConsumers * sms;
    while (k > 1 && rows * chunks_of(k) < want) k >>= 1;
    // The coarsest cut costs least (half the chunk ends, half the partials to fold and to publish)
    // as long as every CTA still gets about two units per streaming warp: cfg2 shape 5.95 against
    // 5.76 TB/s, cfg1 35.0 against 36.8 us; below that the ranges no longer balance (512 rows of a
    // 32000-entry vocabulary: 30.0 against 27.5 us).
    if (k == 4 && k_max == 8 && rows * chunks_of(8) >= 24L * sms) k = 8;
    while (max_partials > 0 && k < k_max && rows * chunks_of(k) > max_partials) k <<= 1;
    return k;
}

void chunking(int V, bool streaming, bool kl, int pieces, int *nchunks, int *chunk)
{
    if (streaming) {
        *chunk = pieces * (kl ? kPiece : 2 * kPiece);
        *nchunks = (V + *chunk - 1) / *chunk;
        return;
    }
    const int n = (V + kMaxChunk - 1) / kMaxChunk;
    int c = (V + n - 1) / n;
    c = (c + 7) & ~7;
    *nchunks = (V + c - 1) / c;
    *chunk = c;
}

std::mutex g_mu;                 // guards the per-device caches below
int g_sm_count[64] = {};
std::atomic<int> g_max_ctas{0};  // 0: one CTA per SM; otherwise a cap on the streaming kernel's grid

// Number of SMs of the current device (cached), or a negative status.
int sm_count_of_current_device()
{
    int dev = 0;
    DD_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return dd::cuda_fail(cudaErrorInvalidDevice, "dd_verify: device index");
    std::lock_guard<std::mutex> lock(g_mu);
    if (!g_sm_count[dev]) DD_CUDA_TRY(cudaDeviceGetAttribute(&g_sm_count[dev], cudaDevAttrMultiProcessorCount, dev));
    return g_sm_count[dev];
}

template <bool KL, bool kRagged>
int launch_stream(const VerifyParams &p, cudaStream_t stream)
{
    const int sms = sm_count_of_current_device();
    if (sms < 0) return sms;
    int dev = 0;
    DD_CUDA_TRY(cudaGetDevice(&dev));
    {
        static bool attr_done[64] = {};
        std::lock_guard<std::mutex> lock(g_mu);
        if (!attr_done[dev]) {
            DD_CUDA_TRY(cudaFuncSetAttribute(verify_stream_kernel<KL, kRagged>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             kSRingBytes));
            // the same split of the SM's memory as the attention kernel that runs before and after
            DD_CUDA_TRY(cudaFuncSetAttribute(verify_stream_kernel<KL, kRagged>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                             cudaSharedmemCarveoutMaxShared));
            attr_done[dev] = true;
        }
    }
    const long units = (long)p.B * p.P * p.nchunks;
    long grid = units < sms ? units : sms;
    const int cap = g_max_ctas.load(std::memory_order_relaxed);
    if (cap > 0 && grid > cap) grid = cap;
    // An ordinary launch: its CTAs fill the shared memory of their SMs, so none could arrive before the previous kernel's have left, and
    // the programmatic form cost 1-2 % (8 x 512 rows of 126464 189.3 -> 193.0 us, 3 x 400 of 99999 45.1 -> 46.1).
    verify_stream_kernel<KL, kRagged><<<(unsigned)grid, kSThreads, kSRingBytes, stream>>>(p);
    DD_CUDA_TRY(cudaGetLastError());
    dd::count_launch();
    return DD_OK;
}

// The row kernel or the streaming kernel.  In pieces of 4 KB (1024 logits of both tensors, 2048 of one), whatever
// share of the rows is flagged (the host does not know): up to 160 pieces per SM the row kernel.
// Measured (us, row against streaming kernel; B x P, V, share flagged): 1 x 128, 1024, KL 25 %: 10.0 / 13.9;
// 4 x 128, 4096, KL: 11.6 / 21.9; 1 x 256, 16000, KL: 12.9 / 21.9; 1 x 512, 32000, KL 100 %: 30.0 / 34.1, 25 %: 21.7 /
// 29.9; 1 x 32, 126464, KL: 14.2 / 24.2; 1 x 128: 25.9 / 31.9; 16 x 512, 1000, CONF: 23.0 / 38.3.  Beyond the line: 8 x
// 256, 32000, CONF: 36.6 / 31.7; 1 x 256, 126464, KL: 38.7 / 37.5; 16 x 512, 8000, KL 50 %: 58.4 / 51.1.
long row_pieces(int V, bool kl) { return ((long)V + 7) / (kl ? kPiece : 2 * kPiece) + 1; }

// Warps per row: enough to fill the GPU (24 per SM), but at least two pieces for each.  Few rows: clusters
// of CTAs, as long as two CTAs per SM hold them all (32 rows of 126464: 27 us with eight warps a row,
// 14 with clusters of eight; 128 rows: clusters of two 25.9, of four 30.1).
RowsShape rows_shape(long rows, long pieces, int sms)
{
    RowsShape shape = {1, 1, 0};
    while (shape.wpr < kRWarps && 4 * shape.wpr <= pieces + 1 && rows * shape.wpr < 24L * sms) shape.wpr *= 2;
    while (shape.wpr == kRWarps && shape.cluster < kRMaxCluster && 4 * kRWarps * shape.cluster <= pieces + 1 &&
           2 * shape.cluster * rows <= 2L * sms)
        shape.cluster *= 2;
    return shape;
}

// Beyond 160 pieces per SM, up to four rows per SM of no more than kLongShare pieces a warp: the deep form (below), in whose two rounds
// or so the streaming kernel's fixed cost is not earned back.  us, row : streaming: 1 x 256, 126464, KL 31.6 : 37.0; 1 x 400, KL 100 % 45.1 :
// 50.7, 50 % 32.6 : 39.5, CONF 28.4 : 38.2, 20.7 : 34.6; 2 x 256, KL 100 % 56.1 : 57.6, 50 % 34.0 : 37.6, 25 % 32.0 : 31.1, but 80 %, where
// some SMs have a third row, 57.0 : 50.0.  A row is one CTA's, so that an SM with one row more costs the more, the
// longer the rows: KL, 2 x 75 rows of 180000 (22 pieces a warp) the same, 2 x 100 of 262144 (32) 54 : 52, 2 x 75 of 524288 92 : 70;
// CONF, 2 x 128 of 262144 (16) 1.26 times as fast, 2 x 150 of 330000 (20) 0.91 to 1.0, of 524288 0.86.  The bound also
// keeps a warp's sums short, and the places of its maxima far from the 2048 pieces (KL: 4096) that LaneState counts: below the line of 160
// a warp has at most 160 / 64 per SM (one row in a cluster of eight).
constexpr long kLongShare = 20;
bool rows_path(int V, long rows, int sms, bool kl)
{
    const long pieces = row_pieces(V, kl);
    if (rows * pieces <= 160L * sms && rows <= 32L * 1024) return true;
    const RowsShape shape = rows_shape(rows, pieces, sms);
    return rows <= 4L * sms && pieces <= kLongShare * shape.wpr * shape.cluster;
}

template <bool KL>
int launch_rows(const VerifyParams &p, cudaStream_t stream)
{
    const int sms = sm_count_of_current_device();
    if (sms < 0) return sms;
    const long rows = (long)p.B * p.P;
    const long pieces = row_pieces(p.V, KL);
    RowsShape shape = rows_shape(rows, pieces, sms);
    const long groups = (rows + kRWarps / shape.wpr - 1) / (kRWarps / shape.wpr);
    // Two CTAs per SM and deep loads (row_part_deep), where all CTAs fit at once and a warp has a few pieces, or rows are few and long;
    // with more rows a third CTA per SM is worth more than deep loads.  us, three CTAs : deep (B x P, V): 1 x 256, 126464, KL 36.8 : 29.9; 1 x 128
    // 23.9 : 20.4; 1 x 32 14.1 : 12.8; 1 x 200, 50000, KL 19.9 : 18.2; but 1 x 256, 16000, KL 11.8 : 12.0, 1 x 256, 16001, CONF 8.8 : 9.6; 2 x 300,
    // 32001, KL 50 % 19.9 : 22.0; 4 x 256, 8000, KL 50 % 13.4 : 16.8; 16 x 512, 1000, CONF 17.8 : 22.4.
    // Not with too few pieces a warp for its start to be earned back (pieces a warp, us three CTAs : deep): where every CTA has an SM, CONF: 3.1,
    // 1 x 36, 49203 11.8 : 12.7, 4 x 37 13.4 : 14.7 (KL 4 x 25, 24576 the same); clusters of four, two CTAs on an SM: 2.0, 4 x 18, 64000, KL
    // 15.3 : 17.0, 2.5, 80000 16.8 : 18.4, 3.1, 100001 18.8 : 20.9, 3.9, 126464 20.8 : 20.9 (of two: 2.8, 4 x 37, 45000 16.0 : 15.0).
    const long ctas = groups * shape.cluster;
    const int least2 = shape.cluster == 1 ? (KL || ctas > sms ? 6 : 7) : shape.cluster >= 4 && ctas > sms ? 7 : 0;
    const bool deep = (ctas <= 2L * sms && 2 * pieces >= least2 * shape.wpr * shape.cluster) || rows * pieces > 160L * sms;
    // flagged rows first (mapped_row): a row per CTA, and long ones (all flagged: 1 x 512, 32000, CONF 16.9 : 18.5, 3 x 200, 60000, CONF 23.8 :
    // 24.9, 2 x 300, 32001, KL 28.5 : 28.1)
    // Not where the mask is written over the flags: every CTA derives its row from all of them, and would see those of sequences already
    // decided changed; by its place it reads its own row's only.
    const uintptr_t flags = (uintptr_t)p.flags, mask = (uintptr_t)p.out_mask;
    const bool in_place = flags < mask + (size_t)rows && mask < flags + (size_t)rows;
    shape.mapped = shape.wpr == kRWarps && shape.cluster == 1 && rows <= kMappedRows && (deep || (KL && pieces >= 24)) && !in_place;
    // Early only in the short form and where every CTA has an SM to itself (the deep one reads for longer than the gap between two kernels): CTAs that arrive early pile up on the SMs that are free first, and waiting ones of a second
    // round take up the room of the first one's last.  us, early : ordinary, after attention of 32 heads of 1024: 256 rows of 126464, KL
    // 55.5 : 53.0, 2 x 300 of 32001 42.7 : 39.3, 1 x 100 of 50000, CONF 35.1 : 33.1, 1 x 512 of 32000, CONF 39.2 : 38.3; but 128 of
    // 1024, KL 27.1 : 28.4, 64 of 1000 27.9 : 28.5.  One after the other, 1024 of 4000, KL 19.4 : 18.7.
    const bool early = !deep && ctas <= sms;
    DD_CUDA_TRY(dd::launch_as(early, deep ? verify_rows_kernel<KL, true> : verify_rows_kernel<KL, false>, (unsigned)ctas,
                              32 * kRWarps, 0, stream, shape.cluster, p, shape));
    dd::count_launch();
    return DD_OK;
}

template <bool KL>
int launch_elementwise(const VerifyParams &p, cudaStream_t stream)
{
    const long grid = (long)p.B * p.P * p.nchunks;
    verify_elementwise_kernel<KL><<<(unsigned)grid, kThreads, 0, stream>>>(p);
    DD_CUDA_TRY(cudaGetLastError());
    dd::count_launch();
    return DD_OK;
}

int launch(const VerifyParams &p, bool streaming, cudaStream_t s)
{
    const bool kl = p.algo == DD_MODE_KL;
    if (!streaming) return kl ? launch_elementwise<true>(p, s) : launch_elementwise<false>(p, s);
    const int sms = sm_count_of_current_device();
    if (sms < 0) return sms;
    if (rows_path(p.V, (long)p.B * p.P, sms, kl)) return kl ? launch_rows<true>(p, s) : launch_rows<false>(p, s);
    if (p.V % 8 != 0) return kl ? launch_stream<true, true>(p, s) : launch_stream<false, true>(p, s);
    return kl ? launch_stream<true, false>(p, s) : launch_stream<false, false>(p, s);
}

int check_args(const void *drafter_logits, const void *verifier_logits, const int32_t *tokens,
               const uint8_t *mask_flags, int mode, float tau, int k, const int32_t *out_tokens,
               const uint8_t *out_mask, int B, int P, int V)
{
    const int algo = mode & 0xFF;
    if (!verifier_logits || !tokens || !mask_flags || !out_tokens || !out_mask) return DD_ERR_INVALID_ARG;
    if (B <= 0 || P <= 0 || V <= 0 || k < 0) return DD_ERR_INVALID_ARG;
    if (algo != DD_MODE_TRUST && algo != DD_MODE_KL && algo != DD_MODE_CONF) return DD_ERR_INVALID_ARG;
    if (mode & ~(0xFF | DD_FLAG_PROBABILISTIC | DD_FLAG_EMIT_DRAFTER)) return DD_ERR_INVALID_ARG;
    if (algo == DD_MODE_KL && !drafter_logits) return DD_ERR_INVALID_ARG;
    if (tau != tau) return DD_ERR_INVALID_ARG;
    if (P > kMaxP) return DD_ERR_UNSUPPORTED;
    if ((long)V >= (1L << 30)) return DD_ERR_UNSUPPORTED;
    return DD_OK;
}

void fill_params(VerifyParams &p, const void *drafter_logits, const void *verifier_logits,
                 const int32_t *tokens, const uint8_t *mask_flags, int mode, float tau, int k, uint64_t seed,
                 int32_t *out_tokens, uint8_t *out_mask, float *out_score, int B, int P, int V)
{
    p.drafter = (const uint16_t *)drafter_logits;
    p.verifier = (const uint16_t *)verifier_logits;
    p.tokens = tokens;
    p.flags = mask_flags;
    p.out_tokens = out_tokens;
    p.out_mask = out_mask;
    p.out_score = out_score;
    p.B = B; p.P = P; p.V = V;
    p.algo = mode & 0xFF;
    p.probabilistic = (mode & DD_FLAG_PROBABILISTIC) != 0;
    p.emit_drafter = (mode & DD_FLAG_EMIT_DRAFTER) != 0;
    p.tau = tau;
    p.k = k;
    p.seed_lo = (uint32_t)(seed & 0xFFFFFFFFu);
    p.seed_hi = (uint32_t)(seed >> 32);
}

}  // namespace

extern "C" size_t dd_verify_workspace_bytes(int B, int P, int V)
{
    if (B <= 0 || P <= 0 || V <= 0) return 0;
    int nchunks, chunk;
    chunking(V, true, true, 1, &nchunks, &chunk);             // the finest cut a launch may choose
    return workspace_bytes(B, P, nchunks) + counter_bytes(B, P) + kControlBytes;
}

extern "C" int dd_verify(const void *drafter_logits, const void *verifier_logits,
                         const int32_t *tokens, const uint8_t *mask_flags,
                         int mode, float tau, int k, uint64_t seed,
                         int32_t *out_tokens, uint8_t *out_mask, float *out_score,
                         int B, int P, int V, void *stream)
{
    int rc = check_args(drafter_logits, verifier_logits, tokens, mask_flags, mode, tau, k, out_tokens, out_mask,
                        B, P, V);
    if (rc != DD_OK) return rc;
    const bool kl = (mode & 0xFF) == DD_MODE_KL;
    const bool streaming = streaming_path(drafter_logits, verifier_logits, kl);

    VerifyParams p;
    int pieces = 4;
    if (streaming) {
        const int sms = sm_count_of_current_device();
        if (sms < 0) return sms;
        pieces = pick_pieces(V, (long)B * P, sms, 0, kl);
    }
    chunking(V, streaming, kl, pieces, &p.nchunks, &p.chunk);
    if ((long)B * P * p.nchunks >= (1L << 31) - (1L << 24)) return DD_ERR_UNSUPPORTED;

    dd::DeviceCtx *ctx = dd::current_ctx();
    if (!ctx) return DD_ERR_CUDA;
    if ((rc = dd::ensure_mirror(ctx)) != DD_OK) return rc;
    if ((rc = dd::check_mirror(ctx, 1)) != DD_OK) return rc;      // an earlier launch gave up a wait: nothing is launched
    rc = dd::ensure_bytes(&ctx->verify_ws, &ctx->verify_ws_bytes, workspace_bytes(B, P, p.nchunks));
    if (rc != DD_OK) return rc;
    rc = dd::ensure_bytes(&ctx->verify_cnt, &ctx->verify_cnt_bytes, counter_bytes(B, P) + kControlBytes);
    if (rc != DD_OK) return rc;

    const size_t bp = (size_t)B * P;
    p.row_counter = (unsigned int *)ctx->verify_cnt;
    p.seq_counter = (unsigned int *)((char *)ctx->verify_cnt + ((bp * 4 + 255) & ~size_t(255)));
    char *control = (char *)ctx->verify_cnt + ctx->verify_cnt_bytes - kControlBytes;
    p.status = (unsigned int *)(control + kStatusOffset);
    p.mirror = ctx->mirror_dev + 1;
    char *w = (char *)ctx->verify_ws;
    p.row_score = (float *)w;          w += (bp * 4 + 255) & ~size_t(255);
    p.row_argmax = (int *)w;           w += (bp * 4 + 255) & ~size_t(255);
    p.partials = (Partial *)w;

    fill_params(p, drafter_logits, verifier_logits, tokens, mask_flags, mode, tau, k, seed,
                out_tokens, out_mask, out_score, B, P, V);
    return launch(p, streaming, (cudaStream_t)stream);
}

// Unmask(p, x) of Algorithm 1's drafting phase: the confidence rule of dd_verify on one logits
// tensor.  "Stays masked" is "fails the threshold and is not among the k most confident": the
// CONF-mode decision with the roles of the outputs renamed, so it runs the same launch.
extern "C" int dd_unmask(const void *logits, const int32_t *tokens, const uint8_t *mask_flags,
                         float tau, int k, int32_t *out_tokens, uint8_t *out_mask, float *out_conf,
                         int B, int P, int V, void *stream)
{
    return dd_verify(nullptr, logits, tokens, mask_flags, DD_MODE_CONF, tau, k, 0, out_tokens, out_mask, out_conf,
                     B, P, V, stream);
}

extern "C" int dd_debug_set_max_ctas(int max_ctas)
{
    if (max_ctas < 0) return DD_ERR_INVALID_ARG;
    g_max_ctas.store(max_ctas, std::memory_order_relaxed);
    return DD_OK;
}

// ---------------------------------------------------------------------------
// dd_lm_head_verify: the verifier's language-model head fused with the verification algorithm.
namespace {

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *,
                                  CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                  CUtensorMapFloatOOBfill);

// bf16 matrix [n_rows, K], K innermost, as a 2-D tensor map with boxes of 64 columns x box_rows rows,
// 128-byte swizzle; rows past the end read as zero.
int make_matrix_tmap(CUtensorMap *m, const void *base, long n_rows, int K, int box_rows)
{
    static EncodeTiledFn fn = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_mu);
        if (!fn) {
            void *sym = nullptr;
            cudaDriverEntryPointQueryResult qr;
            if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &sym, cudaEnableDefault, &qr) == cudaSuccess &&
                qr == cudaDriverEntryPointSuccess)
                fn = reinterpret_cast<EncodeTiledFn>(sym);
        }
    }
    if (!fn) return dd::cuda_fail(cudaErrorSymbolNotFound, "cuTensorMapEncodeTiled entry point");
    const cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)n_rows};
    const cuuint64_t strides[1] = {(cuuint64_t)K * 2};
    const cuuint32_t box[2] = {64, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return dd::cuda_fail(cudaErrorInvalidValue, "cuTensorMapEncodeTiled");
    return DD_OK;
}

// Whether multiplying fewer rows can earn back the launch that finds out which (2 to 4 us; the host does not know how
// many are flagged).  It cannot where there is one tile of rows, and hardly where all items run at the same time: with
// fewer rows there are then fewer at work.  Measured over 400 calls, shares flagged 5 % to 100 % (us, every row against flagged
// rows only; rows, K, V): one round 52, 64, 863 12.2 : 15.7; 6980, 64, 150 28.9 : 34.4; nearly full rounds of long items
// 456, 2624, 17002 43.9 : 32.5, 2923, 1280, 2689 32.0 : 24.8; more rounds 4320, 320, 2259 24.7 : 21.7, 868, 192, 83158 KL
// 149 : 57; with nothing to leave out some 3 us are lost, 903, 1920, 19487 71.0 : 74.7.
bool gathering_can_pay(const ddlm::LmParams &q, bool kl)
{
    if (q.rows <= ddlm::kTileRows) return false;
    // Outside the KL mode counted in tiles of half the widest or more: narrower ones fill SMs that had no item, and fewer rows leave those idle
    // again (counted too, 2952 of 3240, 2880, 1024 27.1 : 38.1, 828 of 942, 3968, 2240 31.2 : 41.7; KL, 226 of 404, 4032, 2334 55.6 : 45.3).
    const int n = kl ? q.all_rows.N : std::max(q.all_rows.N, ddlm::Widths<false>::max_n / 2), tiles = (q.V + n - 1) / n;
    const long items = (long)tiles * ((q.rows + ddlm::kRowsPerItem - 1) / ddlm::kRowsPerItem);
    if (items > q.ctas) return true;
    const long item_cost = (kl ? 2L : 1L) * q.K * (150 + n);                 // 30 to 35 us a million
    return tiles > 2 && 5 * items >= 4 * q.ctas && item_cost >= 400000;
}

template <bool KL>
int launch_lm_head(ddlm::LmParams q, VerifyParams p, const void *dh, const void *dw, const void *vh, const void *vw,
                   char *gathered, size_t gathered_bytes, int ctas, cudaStream_t stream)
{
    using namespace ddlm;
    int rc, dev = 0;
    DD_CUDA_TRY(cudaGetDevice(&dev));
    {
        static bool attr_done[64] = {};
        std::lock_guard<std::mutex> lock(g_mu);
        if (!attr_done[dev]) {
            DD_CUDA_TRY(cudaFuncSetAttribute(lm_head_kernel<KL>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes));
            DD_CUDA_TRY(cudaFuncSetAttribute(lm_head_pair_kernel<KL>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes));
            attr_done[dev] = true;
        }
    }
    LmMaps<KL> m;
    if ((rc = make_matrix_tmap(&m.h, vh, q.rows, q.K, kTileRows)) != DD_OK) return rc;
    if (!q.plan) { gathered = (char *)const_cast<void *>(vh); gathered_bytes = 0; }      // (the maps are not read)
    if ((rc = make_matrix_tmap(&m.h_gathered, gathered, q.rows, q.K, kTileRows)) != DD_OK) return rc;
    m.hd = m.h; m.hd_gathered = m.h_gathered;          // not read outside the KL mode
    if (KL) {
        if ((rc = make_matrix_tmap(&m.hd, dh, q.rows, q.K, kTileRows)) != DD_OK) return rc;
        if ((rc = make_matrix_tmap(&m.hd_gathered, gathered + gathered_bytes, q.rows, q.K, kTileRows)) != DD_OK) return rc;
    }
    // a map per width that the device may choose; one where the host has chosen.  `part`: what one CTA loads at a time is N / part
    auto weight_maps = [&](LmMaps<KL> &to, int part) {
        for (int i = 0; i < Widths<KL>::count; ++i) {
            const int width = Widths<KL>::max_n - 32 * i;
            if (q.plan ? width < q.min_n : width != q.all_rows.N) continue;
            if ((rc = make_matrix_tmap(&to.w[i], vw, q.V, q.K, width / part)) != DD_OK) return rc;
            if (KL && (rc = make_matrix_tmap(&to.wd[i], dw, q.V, q.K, width / part)) != DD_OK) return rc;
        }
        return (int)DD_OK;
    };
    const bool single = q.pairs < 2, pairs = q.pairs > 0;          // both: the number of rows to be multiplied decides which of them works
    LmMaps<KL> m2 = m;                                 // lm_head_pair_kernel's
    if (single && (rc = weight_maps(m, 1)) != DD_OK) return rc;
    if (pairs && KL && single) m2 = m;
    else if (pairs && (rc = weight_maps(m2, KL ? 1 : 2)) != DD_OK) return rc;
    // One CTA per SM, fewer if even the narrowest tiles of all rows do not make that many items.
    const long items = (long)((q.V + q.min_n - 1) / q.min_n) * ((q.rows + kRowsPerItem - 1) / kRowsPerItem);
    const unsigned grid = (unsigned)(items < ctas ? items : ctas);
    if (q.plan) {
        q.rows_per_block = kRowsWarps * ((q.rows + kRowsWarps * kRowsBlocks - 1) / (kRowsWarps * kRowsBlocks));
        DD_CUDA_TRY(dd::launch(lm_head_rows_kernel<KL>, (unsigned)((q.rows + q.rows_per_block - 1) / q.rows_per_block), kRowsThreads, 0, stream, 1,
                               q, p, static_cast<const uint4 *>(vh), reinterpret_cast<uint4 *>(gathered),
                               static_cast<const uint4 *>(dh), reinterpret_cast<uint4 *>(gathered + gathered_bytes)));
    }
    if (pairs) DD_CUDA_TRY(dd::launch(lm_head_pair_kernel<KL>, grid + (grid & 1), ddlm::kThreads, kSmemBytes, stream, 2, m2, q, p));
    if (single) DD_CUDA_TRY(dd::launch(lm_head_kernel<KL>, grid, ddlm::kThreads, kSmemBytes, stream, 1, m, q, p));
    // one warp per row
    const unsigned fold_grid = (unsigned)(((long)q.rows + kFoldThreads / 32 - 1) / (kFoldThreads / 32));
    DD_CUDA_TRY(dd::launch(lm_head_fold_kernel<KL>, fold_grid, kFoldThreads, 0, stream, 1, p, q));
    dd::count_launch(1 + (q.plan ? 1 : 0) + (pairs ? 1 : 0) + (single ? 1 : 0));
    return DD_OK;
}

}  // namespace

extern "C" int dd_lm_head_verify(const void *drafter_hidden, const void *drafter_weight,
                                 const void *verifier_hidden, const void *verifier_weight,
                                 const int32_t *tokens, const uint8_t *mask_flags,
                                 int mode, float tau, int k, uint64_t seed,
                                 int32_t *out_tokens, uint8_t *out_mask, float *out_score,
                                 int B, int P, int K, int V, void *stream)
{
    if (!verifier_hidden || !verifier_weight) return DD_ERR_INVALID_ARG;
    if (K <= 0) return DD_ERR_INVALID_ARG;
    const bool kl = (mode & 0xFF) == DD_MODE_KL;
    if (kl && !drafter_weight) return DD_ERR_INVALID_ARG;
    int rc = check_args(kl ? drafter_hidden : nullptr, verifier_hidden, tokens, mask_flags, mode, tau, k, out_tokens,
                        out_mask, B, P, V);
    if (rc != DD_OK) return rc;
    if (K % ddlm::kBlockK != 0) return DD_ERR_UNSUPPORTED;
    if ((((uintptr_t)verifier_hidden | (uintptr_t)verifier_weight) & 15) != 0) return DD_ERR_UNSUPPORTED;
    if (kl && (((uintptr_t)drafter_hidden | (uintptr_t)drafter_weight) & 15) != 0) return DD_ERR_UNSUPPORTED;
    const long rows = (long)B * P;
    const int sms = sm_count_of_current_device();
    if (sms < 0) return sms;
    int cap = g_max_ctas.load(std::memory_order_relaxed);
    const int ctas = cap > 0 && cap < sms ? cap : sms;

    // the narrowest tiles that the device may choose bound the partials
    constexpr long kMaxPartials = (1L << 31) - (1L << 24);
    // Pairs of CTAs (dd_lm_head_pair.cuh): beyond one tile of rows; outside the KL mode, whose single CTAs have the smaller items, where the k
    // loop is long enough to pay for the meeting of the two and there are items for half of the SMs.  us, lm_head_kernel : pairs (rows, K, V):
    // 256, 4096, 126464 262 : 239 (short bursts 240 : 219); 150, 4096, 126464 243 : 224; 300, 2048, 128256 245 : 216; 1000 of 4000,
    // 4096, 32000 221 : 207; 256, 2048, 126464 149 : 136; 512, 3072, 10000 42.5 : 39.9; 2540 of 4096, 4096, 126464 the same; 400, 4096, 3000
    // 32.3 : 34.1; 960 of 2400, 1024, 12000 38.7 : 40.9; 8192, 512, 2000 38.7 : 40.9.
    const bool pairs = rows > ddlm::kTileRows &&
                       (kl || (K >= 2048 && 2 * ((V + ddlm::kMaxN - 1) / ddlm::kMaxN) * ((rows + ddlm::kRowsPerItem - 1) / ddlm::kRowsPerItem) >= sms));
    const int max_n = kl ? ddlm::Widths<true>::max_n : ddlm::Widths<false>::max_n;
    auto tiles_of = [&](int n) { return (V + n - 1) / n; };
    // Half of the widest, or, where that leaves SMs without an item, narrower ones: an SM takes 45 to 55 bytes per clock, whoever
    // is idle beside it.  Every tile costs the fold a partial per row, though, so with short rows of weights only while a lane has one
    // (us, half : narrower; rows, K, V: 100, 4096, 3072 28.6 : 25.1; 400, 4096, 3000 34.3 : 31.5; 512, 1024, 6000 19.4 : 18.7; 64, 512, 1000
    // 13.1 : 11.7, KL 13.5 : 12.7; 16, 512, 4000 13.2 : 14.9).
    int min_n = max_n / 2;
    const long row_blocks = (rows + ddlm::kRowsPerItem - 1) / ddlm::kRowsPerItem;
    while (min_n > 32 && tiles_of(min_n) * row_blocks < sms && (K >= 1024 || tiles_of(min_n - 32) <= 32)) min_n -= 32;
    while (rows * tiles_of(min_n) >= kMaxPartials) {
        if (min_n == max_n) return DD_ERR_UNSUPPORTED;
        min_n += 32;
    }

    VerifyParams p;
    dd::DeviceCtx *ctx = dd::current_ctx();
    if (!ctx) return DD_ERR_CUDA;
    if ((rc = dd::ensure_mirror(ctx)) != DD_OK) return rc;
    if ((rc = dd::check_mirror(ctx, 1)) != DD_OK) return rc;
    if (dd::try_bytes(&ctx->verify_ws, &ctx->verify_ws_bytes, workspace_bytes(B, P, tiles_of(min_n)), (cudaStream_t)stream) != DD_OK) {
        // no room for the narrowest, or none may be made: of half the widest at least, and no narrower than what is picked where every row is
        // multiplied
        min_n = std::max(min_n, max_n / 2);
        min_n = kl ? ddlm::pick_tile_n<true>(V, rows, sms, min_n, pairs) : ddlm::pick_tile_n<false>(V, rows, sms, min_n, pairs);
        rc = dd::ensure_bytes(&ctx->verify_ws, &ctx->verify_ws_bytes, workspace_bytes(B, P, tiles_of(min_n)));
        if (rc != DD_OK) return rc;
    }
    rc = dd::ensure_bytes(&ctx->verify_cnt, &ctx->verify_cnt_bytes, counter_bytes(B, P) + kControlBytes);
    if (rc != DD_OK) return rc;
    const size_t bp = (size_t)rows;
    char *control = (char *)ctx->verify_cnt + ctx->verify_cnt_bytes - kControlBytes;
    p.nchunks = tiles_of(min_n);
    p.chunk = min_n;
    p.row_counter = (unsigned int *)ctx->verify_cnt;
    p.seq_counter = (unsigned int *)((char *)ctx->verify_cnt + ((bp * 4 + 255) & ~size_t(255)));
    p.status = (unsigned int *)(control + kStatusOffset);
    p.mirror = ctx->mirror_dev + 1;
    char *w = (char *)ctx->verify_ws;
    p.row_score = (float *)w;          w += (bp * 4 + 255) & ~size_t(255);
    p.row_argmax = (int *)w;           w += (bp * 4 + 255) & ~size_t(255);
    p.partials = (Partial *)w;
    fill_params(p, nullptr, nullptr, tokens, mask_flags, mode, tau, k, seed, out_tokens, out_mask, out_score, B, P, V);

    ddlm::LmParams q;
    q.rows = (int)rows; q.K = K; q.V = V;
    q.min_n = min_n;
    q.pairs = pairs ? 2 : 0;
    q.ctas = sms;
    q.plan = nullptr;
    q.all_rows = kl ? ddlm::plan_for<true>(q, q.rows, false) : ddlm::plan_for<false>(q, q.rows, false);
    // A copy of the flagged rows' hidden states, where multiplying fewer rows can pay for it; without room for it every
    // row is multiplied.  The list of those rows stands where the last kernel will put the rows' maxima, when nothing
    // reads the list any more.
    const size_t gathered_bytes = ((size_t)rows * K * 2 + 255) & ~size_t(255);
    if (gathering_can_pay(q, kl) &&
        dd::try_bytes(&ctx->head_ws, &ctx->head_ws_bytes, (kl ? 2 : 1) * gathered_bytes, (cudaStream_t)stream) == DD_OK)
        q.plan = (ddlm::LmPlan *)(control + kPlanOffset);
    // Of more rows than one tile the flagged ones may fit one, and half of a pair's products are then with padding: with more than two rounds of tiles (KL)
    // the device chooses the kernel, and the other one finds nothing to do (1.6 us).  us, pairs : single CTAs (flagged of rows, K, V): KL,
    // 107 of 180, 576, 79839 74.0 : 58.0, 76 of 324, 512, 46208 51.1 : 38.9, 100 of 1060, 2560, 91072 218 : 180; others 42 of 266, 3648, 107112
    // 165 : 143, 45 of 513, 3520, 54830 95.4 : 85.2.  With less to read pairs are the faster ones all the same (KL, 54 of 216, 2880, 16960 53.7 : 62.9, 118 of
    // 189, 2624, 13376 43.9 : 53.9; others 115 of 184, 3008, 31232 50.7 : 53.5), or the second launch costs as much as it gains.
    if (q.pairs && q.plan && (long)V > 256L * sms) q.pairs = 1;
    q.row_map = p.row_argmax;
    char *gathered = (char *)ctx->head_ws;
    return kl ? launch_lm_head<true>(q, p, drafter_hidden, drafter_weight, verifier_hidden, verifier_weight, gathered,
                                     gathered_bytes, ctas, (cudaStream_t)stream)
              : launch_lm_head<false>(q, p, nullptr, nullptr, verifier_hidden, verifier_weight, gathered, 0, ctas,
                                      (cudaStream_t)stream);
}

// ---------------------------------------------------------------------------
// dd_verify_static: the same kernel with its scratch in a fixed device array.
//
// Some callers must not allocate device memory at all: code running inside a
// pre-sized memory budget (an inference server that has handed every free byte
// to its KV cache), code that may not trigger the implicit device
// synchronisation of cudaMalloc/cudaFree, or a process whose allocator is owned
// by another runtime.  For them the partials, row results and completion
// counters live in the file-scope array below, which every GPU that loads this
// library holds until the process exits.
namespace {

constexpr int kStaticMaxRows = 4096;          // B * P
constexpr int kStaticMaxPartials = 65536;     // B * P * ceil(V / 8192)
constexpr size_t kStaticRowsSlot = ((size_t)kStaticMaxRows * 4 + 255) & ~size_t(255);
constexpr size_t kStaticCounterBytes = 2 * kStaticRowsSlot + kControlBytes;   // rows, sequences, control words
constexpr size_t kStaticRowBytes = 2 * kStaticRowsSlot;                       // score + argmax
constexpr size_t kStaticScratchBytes = kStaticCounterBytes + kStaticRowBytes +
                                       (size_t)kStaticMaxPartials * sizeof(Partial);

// In host code this name is only a handle for cudaGetSymbolAddress, never an address to pass on.
static __device__ __align__(256) unsigned char g_static_scratch[kStaticScratchBytes];

// Device address of g_static_scratch per device, resolved on the first call made on that device
// (guarded by g_mu).
unsigned char *g_static_ptr[64] = {};

// The array's address on the current device (null if no call has resolved it yet).
unsigned char *static_scratch_if_resolved()
{
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
    std::lock_guard<std::mutex> lock(g_mu);
    return g_static_ptr[dev];
}

}  // namespace

extern "C" int dd_verify_static(const void *drafter_logits, const void *verifier_logits,
                                const int32_t *tokens, const uint8_t *mask_flags,
                                int mode, float tau, int k, uint64_t seed,
                                int32_t *out_tokens, uint8_t *out_mask, float *out_score,
                                int B, int P, int V, void *stream)
{
    int rc = check_args(drafter_logits, verifier_logits, tokens, mask_flags, mode, tau, k, out_tokens, out_mask,
                        B, P, V);
    if (rc != DD_OK) return rc;
    const bool kl = (mode & 0xFF) == DD_MODE_KL;
    const bool streaming = streaming_path(drafter_logits, verifier_logits, kl);

    VerifyParams p;
    // the fixed scratch bounds the problem size (stated for chunks of 8192 logits; a finer cut is
    // only chosen where its partials still fit)
    const long coarse_chunks = (V + kSChunk - 1) / kSChunk;
    if ((long)B * P > kStaticMaxRows || (long)B * P * coarse_chunks > kStaticMaxPartials) return DD_ERR_UNSUPPORTED;
    int pieces = 4;
    if (streaming) {
        const int sms = sm_count_of_current_device();
        if (sms < 0) return sms;
        pieces = pick_pieces(V, (long)B * P, sms, kStaticMaxPartials, kl);
    }
    chunking(V, streaming, kl, pieces, &p.nchunks, &p.chunk);
    if ((long)B * P * p.nchunks > kStaticMaxPartials) return DD_ERR_UNSUPPORTED;

    int dev = -1;
    DD_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return dd::cuda_fail(cudaErrorInvalidDevice, "dd_verify_static: device index");
    unsigned char *base = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_mu);
        if (!g_static_ptr[dev]) {
            // set-up, once per device, with that device current
            void *ptr = nullptr;
            DD_CUDA_TRY(cudaGetSymbolAddress(&ptr, g_static_scratch));
            g_static_ptr[dev] = static_cast<unsigned char *>(ptr);
        }
        base = g_static_ptr[dev];
    }
    const size_t bp = (size_t)B * P;
    unsigned char *control = base + 2 * kStaticRowsSlot;
    p.row_counter = (unsigned int *)base;
    p.seq_counter = (unsigned int *)(base + kStaticRowsSlot);
    p.status = (unsigned int *)(control + kStatusOffset);
    {
        // the host copy of the health word is used if an earlier call of another entry point made
        // it; this entry point allocates nothing, not even pinned host memory
        dd::DeviceCtx *ctx = dd::current_ctx();
        if (!ctx) return DD_ERR_CUDA;
        if ((rc = dd::check_mirror(ctx, 1)) != DD_OK) return rc;
        p.mirror = ctx->mirror_dev ? ctx->mirror_dev + 1 : nullptr;
    }
    p.row_score = (float *)(base + kStaticCounterBytes);
    p.row_argmax = (int *)(base + kStaticCounterBytes + kStaticRowsSlot);
    p.partials = (Partial *)(base + kStaticCounterBytes + kStaticRowBytes);

    fill_params(p, drafter_logits, verifier_logits, tokens, mask_flags, mode, tau, k, seed,
                out_tokens, out_mask, out_score, B, P, V);

    cudaStream_t s = (cudaStream_t)stream;
    // The array keeps whatever the previous call left: the counters must start at zero (the
    // health word is left alone: it is sticky, like dd_verify's).
    DD_CUDA_TRY(cudaMemsetAsync(p.row_counter, 0, bp * 4, s));
    DD_CUDA_TRY(cudaMemsetAsync(p.seq_counter, 0, (size_t)B * 4, s));
    return launch(p, streaming, s);
}

extern "C" int dd_verify_status(void)
{
    dd::DeviceCtx *ctx = dd::current_ctx();
    if (!ctx) return DD_ERR_CUDA;
    unsigned char *fixed = static_scratch_if_resolved();
    if (!ctx->verify_cnt && !fixed) return DD_OK;
    unsigned int word = 0, word_fixed = 0;
    DD_CUDA_TRY(cudaDeviceSynchronize());
    if (ctx->verify_cnt)
        DD_CUDA_TRY(cudaMemcpy(&word, (char *)ctx->verify_cnt + ctx->verify_cnt_bytes - kControlBytes + kStatusOffset,
                               sizeof word, cudaMemcpyDeviceToHost));
    if (fixed)
        DD_CUDA_TRY(cudaMemcpy(&word_fixed, fixed + 2 * kStaticRowsSlot + kStatusOffset, sizeof word_fixed,
                               cudaMemcpyDeviceToHost));
    if (word == 0) word = word_fixed;
    if (word != 0) {
        char text[96];
        snprintf(text, sizeof text, "verify kernel: bounded wait expired, code 0x%08x", word);
        dd::set_error_text(text);
        return DD_ERR_TIMEOUT;
    }
    return DD_OK;
}

// ---------------------------------------------------------------------------
// Recovery and its test hook.

namespace {

// One thread waits on an mbarrier that nothing will ever complete, gives up after a few hundred
// polls and records the expiry exactly as the real kernels do.  The launch ends by itself within
// microseconds: this is how the error path is exercised without stalling a GPU.
__global__ void expire_wait_kernel(unsigned int *status, unsigned int *mirror, unsigned code)
{
    __shared__ __align__(8) unsigned long long bar;
    const uint32_t b = ddv::s_addr(&bar);
    ddv::sbar_init(b, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    bool arrived = false;
    for (int spin = 0; spin < 512 && !arrived; ++spin) arrived = ddv::sbar_try_wait(b, 0);
    if (!arrived && atomicCAS(status, 0u, code) == 0u && mirror) {
        *reinterpret_cast<volatile unsigned int *>(mirror) = code;
        __threadfence_system();
    }
}

}  // namespace

extern "C" int dd_debug_expire_wait(int which, void *stream)
{
    if (which != 0 && which != 1) return DD_ERR_INVALID_ARG;
    dd::DeviceCtx *ctx = dd::current_ctx();
    if (!ctx) return DD_ERR_CUDA;
    int rc = dd::ensure_mirror(ctx);
    if (rc != DD_OK) return rc;
    unsigned int *word = nullptr;
    if (which == 0) {
        if (!ctx->attn_status) {
            DD_CUDA_TRY(cudaMalloc(&ctx->attn_status, 256));
            DD_CUDA_TRY(cudaMemset(ctx->attn_status, 0, 256));
        }
        word = ctx->attn_status;
    } else {
        rc = dd::ensure_bytes(&ctx->verify_cnt, &ctx->verify_cnt_bytes, counter_bytes(1, 1) + kControlBytes);
        if (rc != DD_OK) return rc;
        word = (unsigned int *)((char *)ctx->verify_cnt + ctx->verify_cnt_bytes - kControlBytes + kStatusOffset);
    }
    expire_wait_kernel<<<1, 1, 0, (cudaStream_t)stream>>>(word, ctx->mirror_dev + which, 0xE000u + (unsigned)which);
    DD_CUDA_TRY(cudaGetLastError());
    return DD_OK;
}

extern "C" int dd_clear_status(void)
{
    dd::DeviceCtx *ctx = dd::current_ctx();
    if (!ctx) return DD_ERR_CUDA;
    DD_CUDA_TRY(cudaDeviceSynchronize());
    if (ctx->attn_status) DD_CUDA_TRY(cudaMemset(ctx->attn_status, 0, sizeof(unsigned int)));
    if (ctx->verify_cnt)
        DD_CUDA_TRY(cudaMemset((char *)ctx->verify_cnt + ctx->verify_cnt_bytes - kControlBytes + kStatusOffset, 0,
                               sizeof(unsigned int)));
    if (unsigned char *fixed = static_scratch_if_resolved())
        DD_CUDA_TRY(cudaMemset(fixed + 2 * kStaticRowsSlot + kStatusOffset, 0, sizeof(unsigned int)));
    if (ctx->mirror) ctx->mirror[0] = ctx->mirror[1] = 0u;
    return DD_OK;
}
