// dd_bidir_attention: full-sequence bidirectional attention (Section 2.2; Eq. 3
// evaluated over the whole key range) for sm_100a, and dd_block_attention: the same
// equation for a block of Nq queries against Nkv (cached) keys, with a per-sequence
// number of valid keys and either memory layout.  One kernel serves both; a persistent form of
// it takes more items than there are SMs, and a form with one query tile and two CTAs per SM takes short query blocks and
// problems too small to fill the chip, whose keys it splits over clusters (see attention_impl, split_parts).
//
// One CTA owns two tiles of 128 query rows of one (batch, head) and walks over
// the keys in tiles of 128.  The CTA is warp-specialised:
//   warps 0-3   softmax of query tile 0 (thread = query row = TMEM lane)
//   warps 4-7   softmax of query tile 1
//   warp  8     one thread feeds a ring of K/V tiles by TMA (tensor maps over
//               (D, N, B*H) or, heads interleaved, (D, N, H, B); 128-byte swizzle;
//               rows past N read as zero)
//   warp  9     one thread issues every tcgen05 MMA
// S_g = Q_g K^T goes to tensor memory; the softmax thread reads its row, keeps the
// running maximum and sum in fp32 (online softmax in base 2, scale*log2e folded
// into one FMA), writes P = 2^(S - m) as bf16 over the first half of the S columns,
// and O_g += P V is a second MMA whose A operand is read from tensor memory.  While
// one tile's softmax runs, the tensor core works on the other tile.  The reference
// point m of a row only moves when the row maximum has outgrown it by more than 2^24
// (a power-of-two factor common to P and to the row sum changes neither bf16's nor
// fp32's relative precision; the step only has to leave fp32 its range); only then
// is O rescaled in tensor memory.  O is normalised by the row sum at the end and
// rounded to bf16 once.
//
// What bounds it.  The chain of one query tile: softmax (some 2000 cycles a key tile) -> P V (512) -> next S
// (512) -> softmax, plus the hand-overs; the other query tile's chain fills the tensor core meanwhile.  So
// the weights are handed over in two parts, P V starting on the first three quarters of the keys while the
// last quarter is computed, and the issuing thread runs under elect_one: N = 8192 1076 -> 920 us, 32 heads
// of 1024 tokens 23.4 -> 20.4.  Under this load the SM clock sits at 1.6-1.75 GHz (power), which is the
// other bound.  Built and not faster: scores in two halves of 64 keys with barriers of their own (S products
// of 128 x 64 are bound by shared memory), two threads per row (sixteen softmax warps), the scores read
// twice in rolled loops instead of kept in 128 registers.
#include <cuda.h>
#include <cuda_bf16.h>
#include <float.h>
#include <math.h>

#include <mutex>
#include <type_traits>

#include "dd_common.cuh"
#include "dd_ptx.cuh"

namespace {

using namespace ddptx;

constexpr int kBlockM = 128;        // query rows per tile
constexpr int kQTiles = 2;          // query tiles per CTA
constexpr int kBlockN = 128;        // keys per step
constexpr int kStages = 5;          // K/V ring slots (one tile each)
constexpr int kThreads = 384;
constexpr int kSoftmaxWarps = 8;
constexpr int kLoadWarp = 8, kMmaWarp = 9;
constexpr uint32_t kTmemCols = 512; // S_0 [0,128)  S_1 [128,256)  O_0 [256,256+D)  O_1 [256+D,256+2D)
// log2 of the largest P tolerated before the reference point moves.  A move costs the row's warp a
// pass over the accumulator in tensor memory in front of the tile's weights: with a step of 8, rows whose scores are peaked (a planted low-rank
// component; trained heads) moved often enough to cost 25-40 % of the throughput (when a move meant a
// second weighting as well).  With 24 the sum
// of a row's weights stays below N * 2^24 and fp32 holds O for |v| * N < 2^100.
constexpr float kRescaleStep = 24.f;

enum : unsigned { kErrWaitQ = 0x100, kErrWaitKV = 0x200, kErrWaitS = 0x300, kErrWaitO = 0x400,
                  kErrWaitP = 0x500, kErrWaitSlot = 0x600 };

struct AttnParams {
    int BH, H, Nq, Nkv, D;
    int m_blocks;              // CTAs per (batch, head) = ceil(Nq / 256)
    const int *kv_len;         // [B] keys of each sequence that exist (clamped to 0..Nkv), or null: Nkv
    int head_major;            // 1: [B,H,N,D], tensor maps are 3-D over (D, N, B*H); 0: [B,N,H,D], 4-D maps (D, N, H, B)
    float scale_log2;          // scale * log2(e)
    unsigned int *status;      // health word of the attention kernel on this device
    unsigned int *mirror;      // its copy in mapped host memory (written only when a wait expires)
    int longest_first;         // 1: sequences by falling number of keys (kv_len given; see attention_impl)
    void *out;                 // where attention_persistent_kernel stores its result (the others through a tensor map)
};

template <int D>
struct Smem {
    static constexpr int kTileBytes = kBlockN * D * 2;             // one 128 x D bf16 tile
    static constexpr int kQ = 0;                                   // two query tiles
    static constexpr int kRing = kQTiles * kTileBytes;             // kStages K/V tiles
    static constexpr int kBars = kRing + kStages * kTileBytes;
    // barriers (8 bytes each): q_full[2], kv_full[kStages], kv_empty[kStages], s_full[2], p_full[2], o_full[2], p_early[2]
    static constexpr int kNumBars = 2 + 2 * kStages + 8;
    static constexpr int kTmemSlot = kBars + 8 * kNumBars;
    static constexpr int kTotal = kTmemSlot + 16;
    // every tile starts on the 1024-byte boundary the 128-byte swizzle needs, the barriers on 8 bytes,
    // and the whole layout plus the alignment slack fits what one CTA may ask for
    static_assert(kTileBytes % 1024 == 0 && kBars % 8 == 0, "tiles on swizzle boundaries, barriers on 8 bytes");
    static_assert(kTotal + 1024 <= 227 * 1024, "shared memory of one CTA");
};

__device__ __forceinline__ void report(const AttnParams &p, unsigned code)
{
    const unsigned word = code | (unsigned)(blockIdx.x & 0xFF);
    if (atomicCAS(p.status, 0u, word) == 0u && p.mirror) {
        *reinterpret_cast<volatile unsigned int *>(p.mirror) = word;      // the host sees it without a synchronisation
        __threadfence_system();
    }
}

// One pair of exponentials in this many is computed on the FMA pipe (0: none).  At D = 64 a key tile costs
// half the tensor time and the same number of exponentials, and the special-function unit (16 per clock)
// is what both query tiles of a CTA compete for: one in eight gained 8 %, one in four 12 % (3 x 24 heads of
// 1357 tokens 72.9 -> 66.2 us, 32 heads of 4096 239 -> 208).  At D = 128 the tensor core, and the
// chip's power, are the bound, and the extra instructions cost 5-10 %.
template <int D> constexpr int kPolyOneIn = D == 64 ? 4 : 0;

// 2^x of two values on the FMA pipe: x = n + f with n the nearest integer (read off the low bits of
// x + 1.5 * 2^23), 2^f on [-1/2, 1/2] as a polynomial of degree five (relative error 1.5e-7, fitted
// by weighted least squares; ex2.approx has 2^-22 = 2.4e-7), n added to the exponent.  From x = -127 downwards (-inf
// included) the result is 2^-149, which is 0 as bf16; between that and -125.5 it is a number below 2^-125.  A NaN gives the
// largest float: infinite as bf16, so that the row's sum is infinite and its result NaN.
__device__ __forceinline__ float2 ex2_poly(float2 x)
{
    auto c = [](float v) { return make_float2(v, v); };
    x.x = max_nan(x.x, -127.f);
    x.y = max_nan(x.y, -127.f);
    const float2 t = __fadd2_rn(x, c(12582912.f));
    const float2 f = __ffma2_rn(__fadd2_rn(t, c(-12582912.f)), c(-1.f), x);
    float2 y = __ffma2_rn(f, c(0.001327647129073739f), c(0.009675541892647743f));
    y = __ffma2_rn(y, f, c(0.05550713092088699f));
    y = __ffma2_rn(y, f, c(0.24022120237350464f));
    y = __ffma2_rn(y, f, c(0.6931469440460205f));
    y = __ffma2_rn(y, f, c(1.0000001192092896f));
    return make_float2(__int_as_float(__float_as_int(y.x) + (__float_as_int(t.x) << 23)),
                       __int_as_float(__float_as_int(y.y) + (__float_as_int(t.y) << 23)));
}

// Row maximum of the raw scores of one key tile (keys past the sequence end excluded).
template <bool kMasked, int N>
__device__ __forceinline__ float row_max(const float (&s)[N], int valid)
{
    float m[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
    for (int i = 0; i < N; i += 8)
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int e = i + 2 * u;
            if (!kMasked) {
                m[u] = max3(m[u], s[e], s[e + 1]);
            } else {
                if (e < valid) m[u] = fmaxf(m[u], s[e]);
                if (e + 1 < valid) m[u] = fmaxf(m[u], s[e + 1]);
            }
        }
    return fmaxf(fmaxf(m[0], m[1]), fmaxf(m[2], m[3]));
}

// Weights P = 2^(s*c - m_ref) of 32 keys (from key q * 32 of the tile) as packed bf16 into tensor memory (16
// columns); adds the weights as rounded to sum_a + sum_b, so that O / l is an exact convex combination (two mixed
// additions per pair: unpacked first, by a shift and a mask, they kept the integer pipe busy beside conversion and maximum;
// D = 64, 3 x 24 heads of 1357 tokens 66.4 -> 62.7 us, 32 heads of 4096 207.6 -> 199.9; D = 128 within 1 %).  Two
// values per instruction where the hardware has a packed form; one pair in kPoly (0: none) goes to the
// FMA pipe.
template <bool kMasked, int kPoly, int N>
__device__ __forceinline__ void weights_to_tmem(const float (&s)[N], int q, int valid, float c, float m_ref,
                                                uint32_t tmem_p, float2 &sum_a, float2 &sum_b)
{
    const float2 c2 = make_float2(c, c), nm2 = make_float2(-m_ref, -m_ref);
    uint32_t pk[16];
#pragma unroll
    for (int i = 0; i < 32; i += 2) {
        const int e = q * 32 + i;
        const float2 a = __ffma2_rn(make_float2(s[e], s[e + 1]), c2, nm2);
        float2 p;
        if (!kMasked && kPoly > 0 && (i / 2) % (kPoly > 0 ? kPoly : 1) == kPoly - 1) p = ex2_poly(a);
        else p = make_float2(ex2(a.x), ex2(a.y));
        if (kMasked) {
            // keys past the end of the sequence get weight zero (a select, not -inf arithmetic: scale may be 0)
            p.x = e < valid ? p.x : 0.f;
            p.y = e + 1 < valid ? p.y : 0.f;
        }
        __nv_bfloat162 b = __floats2bfloat162_rn(p.x, p.y);
        const uint32_t w = *reinterpret_cast<uint32_t *>(&b);
        pk[i / 2] = w;
        add_bf16x2((i & 2) ? sum_a : sum_b, w);
    }
    tmem_st16(tmem_p + q * 16, pk);
}

// A key tile with maximum mx (times scale) meets a row: the first tile sets the row's reference point, a later one
// moves it if it outgrows it by more than the allowed step; then O is rescaled in tensor memory.
// kPart: the row's keys are shared out, and these may all have a score of -inf where others do not; the reference point is
// then the lowest number, so that their weights are 0 and not NaN.
template <int D, bool kPart>
__device__ __forceinline__ void move_reference(uint32_t tO, bool first, float mx, float &m_ref, float &l_run)
{
    if (first) {
        m_ref = kPart ? fmaxf(mx, -FLT_MAX) : mx;
    } else if (__any_sync(0xffffffffu, mx > m_ref + kRescaleStep)) {
        const float m_new = mx > m_ref + kRescaleStep ? mx : m_ref;
        const float alpha = ex2(m_ref - m_new);       // 1 where the row does not move
        m_ref = m_new;
        l_run *= alpha;
#pragma unroll
        for (int cb = 0; cb < D / 32; ++cb) {
            uint32_t r[32];
            tmem_ld32(tO + cb * 32, r);
            tmem_wait_ld(r);
#pragma unroll
            for (int i = 0; i < 32; ++i) r[i] = __float_as_uint(__uint_as_float(r[i]) * alpha);
            tmem_st32(tO + cb * 32, r);
        }
    }
}

// One key tile of one query row, shared by both attention kernels: reads the row's 128 scores from tensor
// memory (the S product has completed), moves the row's reference point if the tile's maximum outgrows
// it by more than the allowed step (the first tile sets it), and writes the weights over S.  They are handed
// to the issuing thread in two parts: `early` after three quarters of the keys, the rest by the caller
// (each time: wait for the stores, fence, arrive), so that P V runs while the last quarter is computed.  A
// row that moves rescales O in tensor memory.  O then holds the sum over the earlier tiles: their P V
// products were issued before this S product by the same thread, so they had completed when S arrived.
template <int D, bool kPart, typename Early>
__device__ __forceinline__ void softmax_tile(uint32_t tS, uint32_t tO, bool first, int valid, float c, float &m_ref,
                                             float &l_run, Early early)
{
    float s[kBlockN];
#pragma unroll
    for (int cb = 0; cb < kBlockN / 32; ++cb)
        tmem_ld32(tS + cb * 32, *reinterpret_cast<uint32_t(*)[32]>(&s[cb * 32]));
    tmem_wait_ld();
    const bool masked = valid < kBlockN;
    const float mx = (masked ? row_max<true>(s, valid) : row_max<false>(s, valid)) * c;
    move_reference<D, kPart>(tO, first, mx, m_ref, l_run);
    float2 sum_a = make_float2(0.f, 0.f), sum_b = sum_a;
    auto weights = [&](auto is_masked, auto poly) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (q == 3) early();
            weights_to_tmem<decltype(is_masked)::value, decltype(poly)::value>(s, q, valid, c, m_ref, tS, sum_a, sum_b);
        }
    };
    // One branch for the whole tile and not one per 32 keys: every basic block ends with its exponentials
    // drained (N = 8192: 962 -> 920 us).
    if (masked) weights(std::true_type(), std::integral_constant<int, 0>());
    else weights(std::false_type(), std::integral_constant<int, kPolyOneIn<D>>());
    sum_a = __fadd2_rn(sum_a, sum_b);
    l_run += sum_a.x + sum_a.y;
}

// 32 columns of one output row, scaled, rounded to bf16 and written to the staging tile in the
// 128-byte-swizzled layout of the output tensor map (`stage` = the row's first byte in the tile,
// r = the row, cb = which 32 columns).
__device__ __forceinline__ void columns_to_staging(const uint32_t *acc, float f, uint32_t stage, int r, int cb)
{
    constexpr uint32_t kBoxBytes = 128 * 128;
    const uint32_t box = stage + (cb / 2) * kBoxBytes;   // 64 columns per box
#pragma unroll
    for (int i = 0; i < 32; i += 8) {
        uint32_t w[4];
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            __nv_bfloat162 v = __floats2bfloat162_rn(__uint_as_float(acc[i + 2 * h]) * f, __uint_as_float(acc[i + 2 * h + 1]) * f);
            w[h] = *reinterpret_cast<uint32_t *>(&v);
        }
        const int chunk = (cb % 2) * 4 + i / 8;          // 16-byte chunk of the 128-byte row
        st_shared_v4(box + ((chunk ^ (r & 7)) << 4), w[0], w[1], w[2], w[3]);
    }
}

// Four neighbouring lanes exchange pieces of 32 bytes: lane t gives its piece c to lane c, as piece t.
__device__ __forceinline__ void quad_transpose(uint32_t (&w)[4][8], int lane)
{
#pragma unroll
    for (int b = 1; b < 4; b *= 2) {
        const bool upper = lane & b;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            if (c & b) continue;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const uint32_t got = __shfl_xor_sync(0xFFFFFFFFu, upper ? w[c][i] : w[c | b][i], b);
                if (upper) w[c][i] = got;
                else w[c | b][i] = got;
            }
        }
    }
}

// The sequence that the `pos`-th group of CTAs works on, and how many keys it has.  With p.longest_first the
// sequences of unequal length are taken longest first (within runs of 32, by key tiles; ties in order), so that the
// launch does not end with a long one that began late.  Every warp finds this out for itself: 32 lengths are one
// load, and a lane's place is the number of lanes with a longer one.
__device__ __forceinline__ int sequence_at(const AttnParams &p, int pos, int &keys)
{
    auto clamped = [&](int b) { return min(max(p.kv_len[b], 0), p.Nkv); };
    if (!p.kv_len) { keys = p.Nkv; return pos; }
    if (!p.longest_first) { keys = clamped(pos); return pos; }
    const int lane = threadIdx.x & 31, run = pos & ~31, B = p.BH / p.H;
    const int n = min(32, B - run);
    const int own = lane < n ? clamped(run + lane) : -1;
    const int tiles = (own + kBlockN - 1) / kBlockN;             // 0 for a lane without a sequence, as for an empty one
    int place = 0;
    for (int i = 0; i < n; ++i) {
        const int other = __shfl_sync(0xFFFFFFFFu, tiles, i);
        place += other > tiles || (other == tiles && i < lane);
    }
    const int src = __ffs(__ballot_sync(0xFFFFFFFFu, lane < n && place == (pos & 31))) - 1;
    keys = __shfl_sync(0xFFFFFFFFu, own, src);
    return run + src;
}

// kBlock = false: the square, head-major, unpadded case of dd_bidir_attention with nothing of the
// general case compiled in.
template <int D, bool kBlock>
__global__ void __launch_bounds__(kThreads, 1)
attention_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                 const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_o,
                 const AttnParams p)
{
    if (kBlock) grid_wait();                              // the sequences' lengths are read
    extern __shared__ __align__(1024) unsigned char smem_dyn[];
    // 128-byte-swizzled tiles must start on a 1024-byte boundary
    const uint32_t smem_base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
    unsigned char *smem_gen = smem_dyn + (smem_base - smem_u32(smem_dyn));
    constexpr uint32_t kTileBytes = Smem<D>::kTileBytes;
    const uint32_t sQ = smem_base + Smem<D>::kQ, sRing = smem_base + Smem<D>::kRing;
    const uint32_t bars = smem_base + Smem<D>::kBars;
    auto bar_q = [&](int g) { return bars + 8u * g; };
    auto bar_kv_full = [&](int s) { return bars + 8u * (2 + s); };
    auto bar_kv_empty = [&](int s) { return bars + 8u * (2 + kStages + s); };
    auto bar_s_full = [&](int g) { return bars + 8u * (2 + 2 * kStages + g); };
    auto bar_p_full = [&](int g) { return bars + 8u * (4 + 2 * kStages + g); };
    auto bar_o_full = [&](int g) { return bars + 8u * (6 + 2 * kStages + g); };
    auto bar_p_early = [&](int g) { return bars + 8u * (8 + 2 * kStages + g); };
    const uint32_t tmem_slot = smem_base + Smem<D>::kTmemSlot;
    volatile uint32_t *tmem_slot_gen = reinterpret_cast<volatile uint32_t *>(smem_gen + Smem<D>::kTmemSlot);

    const int tid = threadIdx.x, warp = warp_uniform(tid >> 5), lane = tid & 31;
    const int head = blockIdx.x / p.m_blocks;
    const int mb = blockIdx.x - head * p.m_blocks;
    const int row0 = mb * (kQTiles * kBlockM);
    int keys = p.Nkv;                                     // keys that exist
    const int b_idx = kBlock ? sequence_at(p, head / p.H, keys) : 0, h_idx = kBlock ? head % p.H : 0;
    const int bh = kBlock ? b_idx * p.H + h_idx : head;
    const bool hm = !kBlock || p.head_major != 0;
    // one tile of 128 rows x 64 columns of head (b_idx, h_idx), rows from n0
    auto load_box = [&](uint32_t dst, const CUtensorMap *tm, uint32_t bar, int c0, int n0) {
        if (hm) tma_load_3d(dst, tm, bar, c0, n0, bh);
        else tma_load_4d(dst, tm, bar, c0, n0, h_idx, b_idx);
    };
    const int nkv = (keys + kBlockN - 1) / kBlockN;       // 0: the sequence has no key, the output is zero
    const int ntiles = (p.Nq - row0 > kBlockM) ? 2 : 1;   // query tiles of this CTA that hold rows
    // A CTA with a single query tile (a short query block) gives its key tiles to the two softmax
    // groups in turn: both keep a copy of the query tile and an accumulator of their own, and the
    // two partial results are combined at the end.  The tensor core then works for one group
    // while the other computes its weights, as with two query tiles.
    const bool split = kBlock && ntiles == 1 && nkv >= 2;
    const int groups = split ? 2 : ntiles;                // softmax groups at work
    constexpr int kBoxes = D / 64;                 // 64-column (128-byte) boxes per tile row
    constexpr uint32_t kBoxBytes = 128 * 128;      // 128 rows x 128 bytes
    constexpr uint32_t kColS = 0, kColO = 256;

    // The producer thread sets up the barriers its copies complete on and sends the first copies
    // on their way (Q tile 0, K tile 0; not for a sequence without keys, whose Q buffers only stage
    // zeros) before the CTA's first barrier: they travel while tensor memory is allocated and the
    // other barriers are set up (cfg1: 22.9 -> 22.0 us).  Nothing else in the CTA touches those
    // buffers or barriers before the __syncthreads below.
    const bool early = !kBlock || nkv > 0;
    if (warp == kLoadWarp && elect_one()) {
        prefetch_tmap(&tm_q); prefetch_tmap(&tm_k); prefetch_tmap(&tm_v);
        mbar_init(bar_q(0), 1); mbar_init(bar_q(1), 1);
        for (int s = 0; s < kStages; ++s) mbar_init(bar_kv_full(s), 1);
        fence_mbar_init();
        if (!kBlock) grid_wait();
        // (also when an earlier wait has expired and the CTA will do nothing: such a CTA lingers at
        // its end until copies in flight have landed)
        if (early) {
            mbar_expect_tx(bar_q(0), kTileBytes);
#pragma unroll
            for (int cx = 0; cx < kBoxes; ++cx) load_box(sQ + cx * kBoxBytes, &tm_q, bar_q(0), cx * 64, row0);
            mbar_expect_tx(bar_kv_full(0), kTileBytes);
#pragma unroll
            for (int cx = 0; cx < kBoxes; ++cx) load_box(sRing + cx * kBoxBytes, &tm_k, bar_kv_full(0), cx * 64, 0);
        }
    }
    if (tid == 0) {
        prefetch_tmap(&tm_o);
        for (int s = 0; s < kStages; ++s) mbar_init(bar_kv_empty(s), 1);
        for (int g = 0; g < kQTiles; ++g) {
            mbar_init(bar_s_full(g), 1);
            mbar_init(bar_p_full(g), kBlockM);
            mbar_init(bar_p_early(g), kBlockM);
            mbar_init(bar_o_full(g), 1);
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
        const uint32_t lane_off = (uint32_t)((warp & 3) * 32) << 16;   // this warp's 32 TMEM lanes
        const uint32_t tS = tmem + lane_off + kColS + g * kBlockN;
        const uint32_t tO = tmem + lane_off + kColO + g * D;
        const float c = p.scale_log2;
        float m_ref = -INFINITY, l_run = 0.f;
        unsigned err = 0;

        // key tiles of this group: j_first, j_first + j_step, ...
        const int j_first = split ? g : 0, j_step = split ? 2 : 1;
        const int my_tiles = nkv > j_first ? (nkv - j_first + j_step - 1) / j_step : 0;
        if (g < groups) {
            for (int i = 0; i < my_tiles; ++i) {
                const int j = j_first + i * j_step;
                if (!mbar_wait(bar_s_full(g), i & 1)) { err = kErrWaitS; break; }
                tc_fence_after();
                const int valid = keys - j * kBlockN;      // keys of this tile that exist
                const bool masked = valid < kBlockN;
                softmax_tile<D, false>(tS, tO, i == 0, valid, c, m_ref, l_run, [&] {
                    if (kBlock && masked) return;          // not before the value rows below are clear
                    tmem_wait_st();
                    tc_fence_before();
                    mbar_arrive(bar_p_early(g));
                });
                if (kBlock && masked) {
                    // Keys past the end of the sequence have weight zero, but 0 x NaN is NaN in the
                    // product P V, and padding may hold any bit pattern: clear their value rows in
                    // the ring slot (whole 128-byte rows, which the swizzle maps onto themselves)
                    // before the weights are handed over.  The slot cannot be refilled before this
                    // group's product has read it.
                    const int item_v = 2 * j + 1, slot_v = item_v % kStages;
                    if (!mbar_wait(bar_kv_full(slot_v), (item_v / kStages) & 1)) { err = kErrWaitKV; break; }
                    const int r = (warp & 3) * 32 + lane;
                    if (r >= valid) {
                        const uint32_t row = sRing + slot_v * kTileBytes + r * 128;
#pragma unroll
                        for (int cx = 0; cx < kBoxes; ++cx)
#pragma unroll
                            for (int c16 = 0; c16 < 8; ++c16)
                                st_shared_v4(row + cx * kBoxBytes + c16 * 16, 0u, 0u, 0u, 0u);
                    }
                    fence_proxy_async_smem();
                }
                tmem_wait_st();
                tc_fence_before();
                if (kBlock && masked) mbar_arrive(bar_p_early(g));
                mbar_arrive(bar_p_full(g));
            }
            if (err == 0 && (!kBlock || nkv > 0) && !mbar_wait(bar_o_full(g), 0)) err = kErrWaitO;
            // ---- split keys: group 1 hands its reference point and row sum to group 0 (through its
            // own Q buffer, which no MMA reads any more) and is done; group 0 adds group 1's
            // accumulator, read from tensor memory, to its own.  Every thread of both groups takes
            // part in the hand-over, also after an expired wait.
            float scale_own = 1.f, scale_other = 0.f;
            float2 *hand_over = reinterpret_cast<float2 *>(smem_gen + Smem<D>::kQ + kTileBytes);
            if (kBlock && split) {
                const int r = (warp & 3) * 32 + lane;
                if (g == 1) {
                    hand_over[r] = make_float2(m_ref, l_run);
                    __threadfence_block();
                    named_bar_arrive(3, 2 * kBlockM);
                } else {
                    named_bar_sync(3, 2 * kBlockM);
                    const float2 other = hand_over[r];
                    if (err == 0 && !mbar_wait(bar_o_full(1), 0)) err = kErrWaitO;
                    const float m_all = fmaxf(m_ref, other.x);
                    scale_own = ex2(m_ref - m_all);
                    scale_other = ex2(other.x - m_all);
                    l_run = l_run * scale_own + other.y * scale_other;
                }
            }
            if (err != 0) report(p, err);
            const bool stores = !(kBlock && split && g == 1);
            if (stores && err == 0) {
                // ---- epilogue: O / l -> bf16 -> this tile's Q buffer (every MMA that read it has
                // completed), in the swizzled layout of the tensor map, -> global by TMA (rows past N
                // are clipped by the map)
                tc_fence_after();
                const int r = (warp & 3) * 32 + lane;                 // row within the tile
                const float inv = (!kBlock || nkv > 0) ? 1.f / l_run : 0.f;
                const float w_own = scale_own * inv, w_other = scale_other * inv;
                const uint32_t stage = sQ + g * kTileBytes + r * 128;
                if constexpr (!kBlock) {
                    // the whole accumulator row in one go: every load is in flight before the first is waited for
                    uint32_t acc[D];
#pragma unroll
                    for (int cb = 0; cb < D / 32; ++cb)
                        tmem_ld32(tO + cb * 32, *reinterpret_cast<uint32_t(*)[32]>(&acc[cb * 32]));
                    tmem_wait_ld();
#pragma unroll
                    for (int cb = 0; cb < D / 32; ++cb) columns_to_staging(&acc[cb * 32], inv, stage, r, cb);
                } else
#pragma unroll
                for (int cb = 0; cb < D / 32; ++cb) {
                    uint32_t acc[32];
                    if (!kBlock || nkv > 0) {
                        tmem_ld32(tO + cb * 32, acc);
                        tmem_wait_ld();
                        if (kBlock && split) {
                            uint32_t acc1[32];
                            tmem_ld32(tO + D + cb * 32, acc1);          // group 1's accumulator, same rows
                            tmem_wait_ld();
#pragma unroll
                            for (int i = 0; i < 32; ++i)
                                acc[i] = __float_as_uint(__uint_as_float(acc[i]) * w_own + __uint_as_float(acc1[i]) * w_other);
                        }
                    } else {
#pragma unroll
                        for (int i = 0; i < 32; ++i) acc[i] = 0u;       // no key: nothing was accumulated
                    }
                    columns_to_staging(acc, (kBlock && split) ? 1.f : inv, stage, r, cb);      // split: already weighted
                }
                fence_proxy_async_smem();
            }
            // every thread of the warpgroup comes here, also after an expired wait
            named_bar_sync(1 + g, kBlockM);
            if (stores && err == 0 && (warp & 3) == 0 && lane == 0) {
#pragma unroll
                for (int cx = 0; cx < kBoxes; ++cx)
                    if (hm) tma_store_3d(&tm_o, sQ + g * kTileBytes + cx * kBoxBytes, cx * 64, row0 + g * kBlockM, bh);
                    else tma_store_4d(&tm_o, sQ + g * kTileBytes + cx * kBoxBytes, cx * 64, row0 + g * kBlockM, h_idx, b_idx);
                tma_store_commit();
                tma_store_wait_read();
            }
        }
    } else {
        reg_dec<72>();
        if (warp == kLoadWarp && elect_one()) {
            // =============================================================== TMA producer
            // what the first MMA needs comes first: Q tile 0, K tile 0, then Q tile 1
            // buffer g takes query tile g, or, with split keys, a second copy of tile 0
            auto load_q = [&](int g) {
                mbar_expect_tx(bar_q(g), kTileBytes);
#pragma unroll
                for (int cx = 0; cx < kBoxes; ++cx)
                    load_box(sQ + g * kTileBytes + cx * kBoxBytes, &tm_q, bar_q(g), cx * 64,
                             row0 + (split ? 0 : g * kBlockM));
            };
            // ring items: 2j = K tile j, 2j+1 = V tile j
            for (int item = 1; item < 2 * nkv; ++item) {
                if (item == 1 && groups > 1) load_q(1);
                const int slot = item % kStages, use = item / kStages;
                if (use > 0 && !mbar_wait(bar_kv_empty(slot), (use - 1) & 1)) { report(p, kErrWaitSlot); break; }
                const uint32_t dst = sRing + slot * kTileBytes;
                const CUtensorMap *tm = (item & 1) ? &tm_v : &tm_k;
                mbar_expect_tx(bar_kv_full(slot), kTileBytes);
#pragma unroll
                for (int cx = 0; cx < kBoxes; ++cx)
                    load_box(dst + cx * kBoxBytes, tm, bar_kv_full(slot), cx * 64, (item >> 1) * kBlockN);
            }
            grid_trigger();
        } else if (warp == kMmaWarp && elect_one()) {
            // =============================================================== MMA issuer
            constexpr uint32_t kIdescS = idesc_bf16(kBlockM, kBlockN, false);
            constexpr uint32_t kIdescO = idesc_bf16(kBlockM, D, true);
            // descriptors of a tile are the tile's base descriptor plus the byte offset / 16
            const uint64_t desc_q0 = smem_desc_sw128(sQ, 16, 1024);
            const uint64_t desc_k0 = smem_desc_sw128(sRing, 16, 1024);            // K-major operand (K tile)
            const uint64_t desc_v0 = smem_desc_sw128(sRing, kBoxBytes, 1024);     // MN-major operand (V tile)
            unsigned err = 0;
            // S_g = Q_g K^T for the K tile in `slot`
            auto issue_s = [&](int g, int slot) {
                const uint64_t a = desc_q0 + (uint64_t)(g * (kTileBytes >> 4));
                const uint64_t b = desc_k0 + (uint64_t)(slot * (kTileBytes >> 4));
                const uint32_t tS = tmem + kColS + g * kBlockN;
#pragma unroll
                for (int ks = 0; ks < D / 16; ++ks) {
                    const uint32_t off = ((ks / 4) * kBoxBytes + (ks % 4) * 32) >> 4;   // 16 bf16 = 32 bytes per k-step
                    mma_ss(tS, a + off, b + off, kIdescS, ks > 0);
                }
                mma_commit(bar_s_full(g));
            };
            // O_g (+)= P_g V for the V tile in `slot`
            // (three quarters of the keys' weights are there, the rest when parity `par` of p_full completes)
            auto issue_o = [&](int g, int slot, bool first, bool last, uint32_t par) -> bool {
                const uint64_t b = desc_v0 + (uint64_t)(slot * (kTileBytes >> 4));
                const uint32_t tS = tmem + kColS + g * kBlockN, tO = tmem + kColO + g * D;
#pragma unroll
                for (int ks = 0; ks < kBlockN / 16; ++ks) {
                    // 16 keys = two 8-row groups of 1024 bytes; column blocks of 64 are one box apart
                    if (ks == 6) {
                        if (!mbar_wait(bar_p_full(g), par)) return false;
                        tc_fence_after();
                    }
                    mma_ts(tO, tS + ks * 8, b + (uint32_t)(ks * (2048 >> 4)), kIdescO, (!first || ks > 0));
                }
                if (last) mma_commit(bar_o_full(g));
                return true;
            };
            auto wait_item = [&](int item) {
                return mbar_wait(bar_kv_full(item % kStages), (item / kStages) & 1);
            };
            // Split keys: key tile t belongs to group t & 1.  S_0(0), S_1(1), then per tile t:
            // O_g (+)= P_g V_t, S_g(t + 2).  Every ring item is read by one group only.
            if (kBlock && split) {
                do {
                    for (int g = 0; g < 2; ++g) {
                        if (!mbar_wait(bar_q(g), 0)) { err = kErrWaitQ; break; }
                        if (!wait_item(2 * g)) { err = kErrWaitKV; break; }
                        tc_fence_after();
                        issue_s(g, (2 * g) % kStages);
                        mma_commit(bar_kv_empty((2 * g) % kStages));
                    }
                    for (int t = 0; t < nkv && err == 0; ++t) {
                        const int g = t & 1, i = t >> 1;
                        const int item_v = 2 * t + 1, item_k = 2 * (t + 2);
                        if (!wait_item(item_v)) { err = kErrWaitKV; break; }
                        if (!mbar_wait(bar_p_early(g), i & 1)) { err = kErrWaitP; break; }
                        tc_fence_after();
                        if (!issue_o(g, item_v % kStages, i == 0, t + 2 >= nkv, i & 1)) { err = kErrWaitP; break; }
                        mma_commit(bar_kv_empty(item_v % kStages));
                        if (t + 2 < nkv) {
                            if (!wait_item(item_k)) { err = kErrWaitKV; break; }
                            tc_fence_after();
                            issue_s(g, item_k % kStages);
                            mma_commit(bar_kv_empty(item_k % kStages));
                        }
                    }
                } while (false);
            } else
            do {
                if (kBlock && nkv == 0) break;
                if (!mbar_wait(bar_q(0), 0)) { err = kErrWaitQ; break; }
                if (!wait_item(0)) { err = kErrWaitKV; break; }
                tc_fence_after();
                issue_s(0, 0);
                if (ntiles > 1) {
                    if (!mbar_wait(bar_q(1), 0)) { err = kErrWaitQ; break; }
                    tc_fence_after();
                    issue_s(1, 0);
                }
                mma_commit(bar_kv_empty(0));
                for (int j = 0; j < nkv && err == 0; ++j) {
                    const int item_v = 2 * j + 1, item_k = 2 * j + 2;
                    const bool more = j + 1 < nkv;
                    // both tiles this round reads are waited for here, not between two groups of MMAs:
                    // a wait in between lets the tensor core run dry
                    if (!wait_item(item_v)) { err = kErrWaitKV; break; }
                    if (more && !wait_item(item_k)) { err = kErrWaitKV; break; }
                    for (int g = 0; g < ntiles; ++g) {
                        if (!mbar_wait(bar_p_early(g), j & 1)) { err = kErrWaitP; break; }
                        tc_fence_after();
                        if (!issue_o(g, item_v % kStages, j == 0, !more, j & 1)) { err = kErrWaitP; break; }
                        if (more) issue_s(g, item_k % kStages);
                    }
                    if (err) break;
                    mma_commit(bar_kv_empty(item_v % kStages));
                    if (more) mma_commit(bar_kv_empty(item_k % kStages));
                }
            } while (false);
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

#include "dd_attention_persistent.cuh"
#include "dd_attention_split.cuh"

// ---------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *,
                                  CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                  CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn()
{
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void *sym = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &sym, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(sym);
    }
    return fn;
}

// bf16 view of a [B,H,N,D] tensor as (D, N, B*H) (head_major: batch and head merge into one
// dimension) or of a [B,N,H,D] tensor as (D, N, H, B); box = 64 columns x 128 rows x 1 (x 1),
// 128-byte swizzle, zero fill: a tile never reaches into the next head or sequence, and rows
// past N read as zero / are not written.
int make_tmap(CUtensorMap *m, const void *base, int B, int H, int N, int D, bool head_major, int box_rows = 128)
{
    EncodeTiledFn fn = encode_fn();
    if (!fn) return dd::cuda_fail(cudaErrorSymbolNotFound, "cuTensorMapEncodeTiled entry point");
    const cuuint64_t row = (cuuint64_t)D * 2;
    const cuuint32_t box[4] = {64, (cuuint32_t)box_rows, 1, 1};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    CUresult r;
    if (head_major) {
        const cuuint64_t dims[3] = {(cuuint64_t)D, (cuuint64_t)N, (cuuint64_t)B * H};
        const cuuint64_t strides[2] = {row, row * N};
        r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(base), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    } else {
        const cuuint64_t dims[4] = {(cuuint64_t)D, (cuuint64_t)N, (cuuint64_t)H, (cuuint64_t)B};
        const cuuint64_t strides[3] = {row * H, row, row * N * H};      // between rows, heads, sequences
        r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void *>(base), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    }
    if (r != CUDA_SUCCESS) return dd::cuda_fail(cudaErrorInvalidValue, "cuTensorMapEncodeTiled");
    return DD_OK;
}

template <int D, bool kBlock>
int launch(const CUtensorMap &tq, const CUtensorMap &tk, const CUtensorMap &tv, const CUtensorMap &to,
           const AttnParams &p, cudaStream_t s)
{
    static bool attr_done[64] = {};
    static std::mutex attr_mu;
    int dev = 0;
    DD_CUDA_TRY(cudaGetDevice(&dev));
    const int smem = Smem<D>::kTotal + 1024;
    {
        std::lock_guard<std::mutex> lock(attr_mu);
        if (dev >= 0 && dev < 64 && !attr_done[dev]) {
            DD_CUDA_TRY(cudaFuncSetAttribute(attention_kernel<D, kBlock>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
            attr_done[dev] = true;
        }
    }
    const long grid = (long)p.BH * p.m_blocks;
    DD_CUDA_TRY(dd::launch(attention_kernel<D, kBlock>, (unsigned)grid, kThreads, smem, s, 1, tq, tk, tv, to, p));
    dd::count_launch();
    return DD_OK;
}

// The persistent kernels: one CTA per SM (or per item, if there are fewer).
template <typename Kernel, typename... Args>
int launch_persistent(Kernel kernel, int smem, bool (&attr_done)[64], const AttnParams &p, int sms, cudaStream_t s, const Args &...maps)
{
    static std::mutex attr_mu;
    int dev = 0;
    DD_CUDA_TRY(cudaGetDevice(&dev));
    {
        std::lock_guard<std::mutex> lock(attr_mu);
        if (dev >= 0 && dev < 64 && !attr_done[dev]) {
            DD_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
            attr_done[dev] = true;
        }
    }
    const long items = (long)p.BH * p.m_blocks;
    const unsigned grid = (unsigned)(items < sms ? items : sms);
    DD_CUDA_TRY(dd::launch(kernel, grid, kThreads, smem, s, 1, maps..., p));
    dd::count_launch();
    return DD_OK;
}

// Short query blocks: `parts` CTAs (a cluster) per head and tile of 128 query rows.
template <int D, int G>
int launch_split(const CUtensorMap &tq, const CUtensorMap &tk, const CUtensorMap &tv, const AttnParams &p, int q_rows, int parts,
                 cudaStream_t s)
{
    static bool attr_done[64] = {};
    static std::mutex attr_mu;
    int dev = 0;
    DD_CUDA_TRY(cudaGetDevice(&dev));
    {
        std::lock_guard<std::mutex> lock(attr_mu);
        if (dev >= 0 && dev < 64 && !attr_done[dev]) {
            DD_CUDA_TRY(cudaFuncSetAttribute(attention_split_kernel<D, G>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSplitSmem));
            attr_done[dev] = true;
        }
    }
    DD_CUDA_TRY(dd::launch(attention_split_kernel<D, G>, (unsigned)((long)p.BH * p.m_blocks * parts), kSplitThreads, kSplitSmem, s, parts,
                           tq, tk, tv, p, q_rows, parts));
    dd::count_launch();
    return DD_OK;
}

int sm_count(int *out)
{
    static int cached[64] = {};
    static std::mutex mu;
    int dev = 0;
    DD_CUDA_TRY(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lock(mu);
    if (dev < 0 || dev >= 64) return DD_ERR_UNSUPPORTED;
    if (cached[dev] == 0) DD_CUDA_TRY(cudaDeviceGetAttribute(&cached[dev], cudaDevAttrMultiProcessorCount, dev));
    *out = cached[dev];
    return DD_OK;
}

// How many CTAs of attention_split_kernel share one query tile's keys; 0: one of the other kernels is faster.
// `tiles`: query tiles of 128 rows over all heads; n: key tiles.  Figures in us on 148 SMs, D = 128 unless noted, this
// kernel : attention_kernel.
//   * One key tile: where attention_kernel's general form is the other side, or it takes more than one round (the
//     start and end of a CTA are all there is; the square form is quicker in one, 4 x 128 4.5 : 5.3).  8 heads, 8 queries 5.5 : 6.0, 1024 heads 22.7 :
//     39.8, of unequal length 26.6 : 51.3; 128 queries, 160 heads 7.9 : 10.0, 1024 29.8 : 39.7.
//   * More tiles than SMs, one per head: a CTA per tile, two on an SM.  Up to 32 queries (keys shared by a CTA's
//     warps): 320 heads, n = 12 52.9 : 56.2, of unequal length 35.4 : 44.2; 1024, n = 16 175 : 193 and 118 : 141; 256,
//     n = 32 84 : 95; 1024 at D = 64, n = 16 93 : 139 and 63 : 108.  Not where long sequences of unequal length take one
//     round, which attention_kernel's faster single item wins at D = 128 (160 heads, n = 32 50 : 44; 256 65 : 61).
//     33 to 128 queries: two CTAs on an SM take 1.2 (short keys) to 1.9 times (long ones) as long as one of
//     attention_kernel, so from n = 9 on waves are compared, and beyond 16 there is nothing to win.  128 queries, n = 8:
//     256 heads 29 : 32, 400 51 : 48 (two waves to three), 512 55 : 61; n = 16: 256 heads 51 : 53, 400 93 : 81, 512
//     97 : 107; n = 32: 512 heads 194 : 195.
//   * Too few tiles to fill the chip: eight CTAs a tile while that leaves an SM to each, four up to 1.75 an SM (288 CTAs
//     in clusters of four are not resident at a time: 72 heads, n = 16 27.7 : 20.7, 64 19.0 : 20.3), two beyond that
//     (only heads of several tiles, of which attention_kernel gives a CTA two).  With two key tiles a part
//     or fewer the meeting of the parts (some 3 us) is hardly earned back.  Up to 32 queries: 8 heads, n = 32 14.7 :
//     31.3, n = 16 11.3 : 18.3, n = 4 8.3 : 9.0; 32 heads, n = 32 19.4 : 32.7, n = 8 10.4 : 12.0, n = 4 8.8 : 9.1; 64
//     heads, n = 12 16.2 : 16.7, n = 8 13.4 : 12.8; D = 64, 64 heads, n = 8 10.2 : 11.5, and without splitting n = 4 7.5 :
//     8.1, 128 heads n = 16 18.6 : 19.4.  128 queries (a ring of two tiles): 32 heads, n = 16 17.4 : 19.6, n = 8 13.5 :
//     12.4; 64 heads, n = 32 33.3 : 35.2, n = 16 23.3 : 21.1.  256 queries: 8 heads, n = 8 12.5 : 18.5; 32 heads, n = 8
//     17.2 : 19.1; 64 heads, n = 16 29.4 : 34.0, n = 8 21.5 : 20.4.
int split_parts(long tiles, int nkv, int Nq, int D, bool general, bool unequal, int sms)
{
    const bool copies = Nq <= 32, one_tile = Nq <= kBlockM;
    if (one_tile && nkv == 1) return general || tiles > sms ? 1 : 0;
    if (one_tile && tiles > sms) {
        if (copies) return unequal && D == 128 && nkv > 16 && 4 * tiles <= 7L * sms ? 0 : 1;
        const long waves = (tiles + sms - 1) / sms, waves2 = (tiles + 2 * sms - 1) / (2 * sms);
        return nkv <= 16 && (nkv <= 8 || 9 * waves2 < 5 * waves) ? 1 : 0;
    }
    int parts = tiles * 8 <= sms ? 8 : tiles * 16 <= 7L * sms ? 4 : tiles * 8 <= 7L * sms && !one_tile ? 2 : 0;
    if (parts == 8 && nkv < (tiles * 16 <= sms ? 16 : 24)) parts = 4;
    const bool roomy = tiles * parts <= sms;              // an SM for each CTA
    if (copies) {
        const int least = D == 64 ? 6 : roomy ? 4 : 12;
        if (parts && nkv >= least) return parts;
        return D == 64 || nkv == 2 ? 1 : 0;
    }
    const int least = !one_tile ? (parts == 2 ? 16 : 8) : Nq > 64 ? (roomy ? 16 : 32) : roomy ? 8 : 16;
    return nkv >= least ? parts : 0;
}

int attention_impl(const void *q, const void *k, const void *v, void *out, int B, int H, int Nq, int Nkv, int D,
                   const int32_t *kv_len, int layout, float scale, void *stream)
{
    if (!q || !k || !v || !out) return DD_ERR_INVALID_ARG;
    if (B <= 0 || H <= 0 || Nq <= 0 || Nkv <= 0 || D <= 0) return DD_ERR_INVALID_ARG;
    if (layout != DD_LAYOUT_BHND && layout != DD_LAYOUT_BNHD) return DD_ERR_INVALID_ARG;
    if (!isfinite(scale)) return DD_ERR_INVALID_ARG;
    if (scale < 0.f) return DD_ERR_UNSUPPORTED;
    if (D != 64 && D != 128) return DD_ERR_UNSUPPORTED;
    if ((((uintptr_t)q | (uintptr_t)k | (uintptr_t)v | (uintptr_t)out) & 15) != 0) return DD_ERR_UNSUPPORTED;
    const long BH = (long)B * H;
    const int m_blocks = (Nq + kQTiles * kBlockM - 1) / (kQTiles * kBlockM);
    if (BH * m_blocks >= (1L << 31) || BH >= (1L << 31)) return DD_ERR_UNSUPPORTED;

    dd::DeviceCtx *ctx = dd::current_ctx();
    if (!ctx) return DD_ERR_CUDA;
    int rc = dd::ensure_mirror(ctx);
    if (rc != DD_OK) return rc;
    if ((rc = dd::check_mirror(ctx, 0)) != DD_OK) return rc;      // an earlier launch gave up a wait: nothing is launched
    if (!ctx->attn_status) {
        DD_CUDA_TRY(cudaMalloc(&ctx->attn_status, 256));
        DD_CUDA_TRY(cudaMemset(ctx->attn_status, 0, 256));
    }
    const bool head_major = layout == DD_LAYOUT_BHND;
    CUtensorMap tq, tk, tv, to;
    if ((rc = make_tmap(&tk, k, B, H, Nkv, D, head_major)) != DD_OK) return rc;
    if ((rc = make_tmap(&tv, v, B, H, Nkv, D, head_major)) != DD_OK) return rc;

    AttnParams p;
    p.BH = (int)BH; p.H = H; p.Nq = Nq; p.Nkv = Nkv; p.D = D;
    p.m_blocks = m_blocks;
    p.kv_len = kv_len;
    p.head_major = head_major ? 1 : 0;
    p.scale_log2 = scale * 1.4426950408889634f;
    p.status = ctx->attn_status;
    p.mirror = ctx->mirror_dev;
    p.out = out;
    p.longest_first = 0;
    cudaStream_t s = (cudaStream_t)stream;
    const bool general = kv_len != nullptr || !head_major || Nq != Nkv;
    int sms = 0;
    if ((rc = sm_count(&sms)) != DD_OK) return rc;
    const int nkv = (Nkv + kBlockN - 1) / kBlockN;
    // Sequences of unequal length, longest first: where the launch takes more than one round of CTAs and no more than
    // two, what starts in the second is then short (16 x 32 heads, 32 queries over 256-1024 keys: 45.0 -> 41.6 us; 8 x
    // 32 heads, 256 queries over 512-2048: 66.7 -> 62.0).  With more rounds, CTAs of equal length start and end
    // together, which costs more (20 x 32 heads of the former 51.1 -> 55.0, 64 x 32 151 -> 156).
    auto longest_first = [&](long ctas, long at_a_time) { return kv_len && B > 1 && ctas > at_a_time && ctas <= 2 * at_a_time; };
    const long tiles = BH * ((Nq + kBlockM - 1) / kBlockM);
    if (const int parts = split_parts(tiles, nkv, Nq, D, general, kv_len && B > 1, sms)) {
        // copies of the query rows in a tile (see attention_split_kernel)
        const int copies = Nq > 32 ? 1 : D == 64 ? 4 : 2;
        const int q_rows = copies > 1 ? 32 * copies : Nq <= 64 ? 64 : 128;
        if ((rc = make_tmap(&tq, q, B, H, Nq, D, head_major, copies > 1 ? 32 : q_rows)) != DD_OK) return rc;
        p.m_blocks = (Nq + kBlockM - 1) / kBlockM;
        p.longest_first = longest_first(tiles * parts, 2 * sms);
        if (copies > 1)
            return D == 64 ? launch_split<64, 4>(tq, tk, tv, p, q_rows, parts, s) : launch_split<128, 2>(tq, tk, tv, p, q_rows, parts, s);
        return D == 64 ? launch_split<64, 1>(tq, tk, tv, p, q_rows, parts, s) : launch_split<128, 1>(tq, tk, tv, p, q_rows, parts, s);
    }
    if ((rc = make_tmap(&tq, q, B, H, Nq, D, head_major)) != DD_OK) return rc;
    p.longest_first = longest_first(BH * m_blocks, sms);
    // More items than SMs: persistent CTAs, whose rounds run across items.  us, a CTA per item : persistent: D = 128, 16 x 32 heads of
    // 512 tokens 101 : 78, 40 x 32 of 330 (a short kernel with rounds of its own, until then) 164 : 134, 64 x 32 of 256 148 : 91, 4 x
    // 32 of 4096 936 : 875, 32 of 8192 954 : 937, 3 x 24 of 1357 73.3 : 66.6; D = 64, 3 x 24 of 1357 61.5 : 56.8, 16 x 32 of 512 60.0 :
    // 54.8, 32 x 32 of 384 105 : 78.  With one round of items the one-item kernel's shorter start counts: 32 x 300 11.1 : 11.2, 16
    // x 512 at D = 128 11.65 : 11.8, 2 x 16 of 640 at D = 64 12.2 : 12.4.
    if (!general && nkv >= 2 && BH * m_blocks > sms) {
        static bool attr_done[2][64] = {};
        if (D == 64) return launch_persistent(attention_persistent_kernel<64>, SmemL<64>::kTotal + 1024, attr_done[0], p, sms, s, tq, tk, tv);
        return launch_persistent(attention_persistent_kernel<128>, SmemL<128>::kTotal + 1024, attr_done[1], p, sms, s, tq, tk, tv);
    }
    // (only this kernel stores through a map)
    if ((rc = make_tmap(&to, out, B, H, Nq, D, head_major)) != DD_OK) return rc;
    if (general) return D == 64 ? launch<64, true>(tq, tk, tv, to, p, s) : launch<128, true>(tq, tk, tv, to, p, s);
    return D == 64 ? launch<64, false>(tq, tk, tv, to, p, s) : launch<128, false>(tq, tk, tv, to, p, s);
}

}  // namespace

extern "C" int dd_bidir_attention(const void *q, const void *k, const void *v, void *out,
                                  int B, int H, int N, int D, float scale, void *stream)
{
    return attention_impl(q, k, v, out, B, H, N, N, D, nullptr, DD_LAYOUT_BHND, scale, stream);
}

extern "C" int dd_block_attention(const void *q, const void *k, const void *v, void *out,
                                  int B, int H, int Nq, int Nkv, int D,
                                  const int32_t *kv_len, int layout, float scale, void *stream)
{
    return attention_impl(q, k, v, out, B, H, Nq, Nkv, D, kv_len, layout, scale, stream);
}
