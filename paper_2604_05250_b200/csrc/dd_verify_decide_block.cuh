// Decision stage of one sequence run by all threads of a CTA: the rules and results of
// decide_sequence_impl.  One pass over the positions takes the flags and scores into keys in shared
// memory; the k-th largest key is found by radix selection, eight bits at a time (four short passes with
// a histogram in shared memory, where a warp's bitwise search takes 33); the last pass stores.  It runs
// once per sequence, from a cold instruction cache: a few hundred instructions in rolled loops, about 2 us,
// where the warp's unrolled forms take 12-16 cold and 3 after a rehearsal.
#pragma once

#include "dd_verify_common.cuh"

namespace ddv {

constexpr int kBlockDecideMaxThreads = 256;

struct BlockDecide {                 // in shared memory
    uint32_t key[kMaxP];
    unsigned hist[256];
    double part[kBlockDecideMaxThreads / 32];
    unsigned digit, above, count;
};

// Every thread of the CTA calls it; the number of threads is a multiple of 32, at most
// kBlockDecideMaxThreads.
__device__ __noinline__ void decide_block(const VerifyParams &p, int b, BlockDecide &s)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, threads = blockDim.x;
    const unsigned full = 0xFFFFFFFFu;
    const long base = (long)checked(p, b, p.B, kSiteSeq) * p.P;      // every access below is at base + i with i < P
    const bool kl_mode = p.algo == DD_MODE_KL;
    auto score_of = [&](uint32_t key) -> float {     // inverse of the key map (key != 0)
        const float rel = __uint_as_float((key & 0x80000000u) ? (key ^ 0x80000000u) : ~key);
        return kl_mode ? 0.0f - rel : rel;
    };
    // keys: order-preserving image of the reliability, 0 outside the set; and Eq. 6's normaliser
    if (tid == 0) s.count = 0u;
    double part = 0.0;
    unsigned flagged = 0;
    for (int i = tid; i < p.P; i += threads) {
        const uint8_t f = p.flags[base + i];
        const float sc = __ldcg(p.row_score + base + i);
        const uint32_t key = f ? orderable(kl_mode ? 0.0f - sc : sc) : 0u;
        s.key[i] = key;
        if (key) { ++flagged; part += (double)score_of(key); }
    }
    __syncthreads();
    flagged = __reduce_add_sync(full, flagged);
    if (lane == 0) atomicAdd(&s.count, flagged);
    double kl_sum = 0.0;
    if (kl_mode && p.probabilistic) {
        part = warp_sum(part);
        if (lane == 0) s.part[warp] = part;
        __syncthreads();
        for (int w = 0; w < threads / 32; ++w) kl_sum += s.part[w];          // a fixed order
    }
    auto fails = [&](int i, float sc) -> bool {
        if (p.algo == DD_MODE_TRUST) return false;
        if (!p.probabilistic) return kl_mode ? (sc > p.tau) : (sc < p.tau);
        const uint32_t w = philox_first_word((uint32_t)i, (uint32_t)b, p.seed_lo, p.seed_hi);
        const double u = (double)(w >> 8) * (1.0 / 16777216.0);
        const double prob = kl_mode ? (kl_sum > 0.0 ? (double)sc / kl_sum : 0.0) : 1.0 - (double)sc;
        return u < prob;
    };
    bool any = false;
    if (p.k > 0 && p.algo != DD_MODE_TRUST)
        for (int i = tid; i < p.P; i += threads) {
            const uint32_t key = s.key[i];
            any |= key != 0u && fails(i, score_of(key));
        }
    any = __syncthreads_or(any);                     // (also: the count is complete)
    const bool keep_all = any && (int)s.count <= p.k;
    const bool topk = any && !keep_all;
    // thr = the k-th largest key; of the positions equal to it, `quota` are kept, lowest index first
    uint32_t thr = 0u, mask = 0u;
    unsigned quota = (unsigned)p.k;
    if (topk) {
#pragma unroll 1
        for (int shift = 24; shift >= 0; shift -= 8) {
            for (int i = tid; i < 256; i += threads) s.hist[i] = 0u;
            __syncthreads();
            for (int i = tid; i < p.P; i += threads) {
                const uint32_t key = s.key[i];
                if (key != 0u && (key & mask) == thr) atomicAdd(&s.hist[(key >> shift) & 255u], 1u);
            }
            __syncthreads();
            if (warp == 0) {
                // lane l holds digits 255 - 8 l .. 248 - 8 l; how many keys have a larger digit than a lane's
                unsigned h[8], sum = 0;
#pragma unroll
                for (int u = 0; u < 8; ++u) { h[u] = s.hist[255 - 8 * lane - u]; sum += h[u]; }
                unsigned incl = sum;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const unsigned v = __shfl_up_sync(full, incl, o);
                    if (lane >= o) incl += v;
                }
                unsigned above = incl - sum;
                if (above < quota && quota <= incl) {                 // one lane: the quota-th key is among its digits
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        if (above < quota && quota <= above + h[u]) { s.digit = 255 - 8 * lane - u; s.above = above; }
                        above += h[u];
                    }
                }
            }
            __syncthreads();
            thr |= s.digit << shift;
            mask |= 255u << shift;
            quota -= s.above;
        }
        // ties: the positions equal to thr that come first.  Warp 0 finds the index of the quota-th of them.
        if (warp == 0) {
            unsigned seen = 0, last = 0;
            for (int i0 = 0; i0 < p.P; i0 += 32) {
                const bool eq = i0 + lane < p.P && s.key[i0 + lane] == thr;
                const unsigned m = __ballot_sync(full, eq);
                const unsigned rank = seen + __popc(m & ((1u << lane) - 1u));
                const unsigned hit = __ballot_sync(full, eq && rank + 1u == quota);
                if (hit) { last = (unsigned)(i0 + __ffs(hit) - 1); break; }
                seen += __popc(m);
            }
            if (lane == 0) s.count = last;
        }
        __syncthreads();
    }
    const unsigned last_equal = s.count;
    for (int i = tid; i < p.P; i += threads) {
        const long t = base + i;
        const uint32_t key = s.key[i];
        const int32_t tok = p.tokens[t];
        if (key == 0u) {
            p.out_tokens[t] = tok;
            p.out_mask[t] = 0;
            if (p.out_score) p.out_score[t] = 0.0f;
            continue;
        }
        const float sc = score_of(key);              // exactly the stored score
        const bool protect = keep_all || (topk && (key > thr || (key == thr && (unsigned)i <= last_equal)));
        const bool remask = fails(i, sc) && !protect;
        p.out_mask[t] = remask ? 1 : 0;
        p.out_tokens[t] = (remask || p.emit_drafter) ? tok : __ldcg(p.row_argmax + t);
        if (p.out_score) p.out_score[t] = sc;
    }
}

// The same for sequences of at most 512 positions and two per thread: everything about a position is loaded
// in one batch and stays in registers, and the k-th largest key is found from keys in registers, three bits at a time:
// seven warps count the keys from one candidate each, a barrier, and every warp picks the next three bits.  It begins below the
// bits that all keys share and ends as soon as exactly k keys are left (4-6 rounds; more only for ties).  Bit by bit in one warp, without
// barriers, from the highest bit on, it took 1.5 to 2.7 us of a call; together with a report that is prepared while the first
// warp folds and a fold that exchanges among as many lanes as there are partials: 1 x 128 positions, V = 1024, KL 7.7 -> 7.2 us; 16 x 512,
// 1000, CONF 19.7 -> 17.9; 1 x 300, 5000 10.4 -> 9.0; 1 x 512, 32000 18.6 -> 17.0; 2 x 300, 32001, KL 20.3 -> 19.8.
// At least eight warps.
__device__ __noinline__ void decide_block_short(const VerifyParams &p, int b, BlockDecide &s)
{
    constexpr int R = 2;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, threads = blockDim.x;
    const unsigned full = 0xFFFFFFFFu;
    const long base = (long)checked(p, b, p.B, kSiteSeq) * p.P;
    const bool kl_mode = p.algo == DD_MODE_KL;
    uint32_t key[R];
    int32_t tok[R], top[R];
    float score[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int i = min(tid + r * threads, p.P - 1);
        const uint8_t f = p.flags[base + i];
        score[r] = __ldcg(p.row_score + base + i);
        tok[r] = p.tokens[base + i];
        top[r] = __ldcg(p.row_argmax + base + i);
        key[r] = f && tid + r * threads < p.P ? orderable(kl_mode ? 0.0f - score[r] : score[r]) : 0u;
    }
#pragma unroll
    for (int r = 0; r < R; ++r)
        if (tid + r * threads < 512) s.key[tid + r * threads] = key[r];      // zeros past the sequence
    double kl_sum = 0.0;
    if (kl_mode && p.probabilistic) {
        double part = 0.0;
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (key[r]) part += (double)score[r];
        part = warp_sum(part);
        if (lane == 0) s.part[warp] = part;
        __syncthreads();
        for (int w = 0; w < threads / 32; ++w) kl_sum += s.part[w];          // a fixed order
    }
    bool fail[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        fail[r] = false;
        if (key[r] == 0u || p.algo == DD_MODE_TRUST) continue;
        if (!p.probabilistic) {
            fail[r] = kl_mode ? score[r] > p.tau : score[r] < p.tau;
        } else {
            const uint32_t w = philox_first_word((uint32_t)(tid + r * threads), (uint32_t)b, p.seed_lo, p.seed_hi);
            const double u = (double)(w >> 8) * (1.0 / 16777216.0);
            const double prob = kl_mode ? (kl_sum > 0.0 ? (double)score[r] / kl_sum : 0.0) : 1.0 - (double)score[r];
            fail[r] = u < prob;
        }
    }
    const bool any = __syncthreads_or(p.k > 0 && (fail[0] || fail[1]));
    uint32_t thr = 0u;               // kept: keys above thr, and of those equal to it the positions up to last_equal
    unsigned last_equal = 0;
    bool keep_all = false;
    if (any) {
        uint32_t kr[16];                                 // all keys, in every warp
#pragma unroll
        for (int r = 0; r < 16; ++r) kr[r] = r * 32 < p.P ? s.key[lane + 32 * r] : 0u;
        auto count_from = [&](uint32_t bound) -> int {   // keys not below it
            int c0 = 0, c1 = 0;
#pragma unroll
            for (int r = 0; r < 4; r += 2) { c0 += kr[r] >= bound; c1 += kr[r + 1] >= bound; }
            if (p.P > 128) {
#pragma unroll
                for (int r = 4; r < 16; r += 2) { c0 += kr[r] >= bound; c1 += kr[r + 1] >= bound; }
            }
            return __reduce_add_sync(full, c0 + c1);
        };
        if (count_from(1u) > p.k) {
            // every key has the bits above `pos` of the largest
            uint32_t high = 0u, low = 0xFFFFFFFFu;
#pragma unroll
            for (int r = 0; r < 16; ++r) {
                high = max(high, kr[r]);
                low = min(low, kr[r] - 1u);              // (0, no key, becomes the largest)
            }
            high = __reduce_max_sync(full, high);
            low = __reduce_min_sync(full, low) + 1u;
            int pos = 32 - __clz(high ^ low);
            thr = pos < 32 ? high >> pos << pos : 0u;
            bool exact = false;
#pragma unroll 1
            for (unsigned *n = s.hist; pos > 0 && !exact; n = s.hist + ((n - s.hist) ^ 8)) {
                const int bits = min(pos, 3);
                pos -= bits;
                const int mine = count_from(thr | (uint32_t)warp << pos);
                if (lane == 0 && warp < 8) n[warp] = (unsigned)mine;
                __syncthreads();
                unsigned best = 0, left = 0;
#pragma unroll
                for (unsigned w = 1; w < 8; ++w)
                    if (w < (1u << bits) && n[w] >= (unsigned)p.k) { best = w; left = n[w]; }
                thr |= best << pos;
                exact = best > 0 && left == (unsigned)p.k;
            }
            last_equal = 0xFFFFFFFFu;                    // every position equal to thr
            if (!exact) {
                // ties at the threshold: kept lowest index first
                if (warp == 0) {
                    unsigned last = 0xFFFFFFFFu;
                    int quota = p.k - (thr == 0xFFFFFFFFu ? 0 : count_from(thr + 1u)), seen = 0;
#pragma unroll 1
                    for (int i0 = 0; i0 < p.P; i0 += 32) {
                        const bool eq = s.key[i0 + lane] == thr;
                        const unsigned m = __ballot_sync(full, eq);
                        const int rank = seen + __popc(m & ((1u << lane) - 1u));
                        const unsigned hit = __ballot_sync(full, eq && rank + 1 == quota);
                        if (hit) { last = (unsigned)(i0 + __ffs(hit) - 1); break; }
                        seen += __popc(m);
                    }
                    if (lane == 0) s.count = last;
                }
                __syncthreads();
                last_equal = s.count;
            }
        }                                                // else: no more than k, all are kept (thr stays 0)
        keep_all = thr == 0u;
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int i = tid + r * threads;
        if (i >= p.P) break;
        const long t = base + i;
        const bool protect = any && (keep_all || key[r] > thr || (key[r] == thr && (unsigned)i <= last_equal));
        const bool remask = fail[r] && !protect;
        p.out_mask[t] = remask ? 1 : 0;
        p.out_tokens[t] = (key[r] == 0u || remask || p.emit_drafter) ? tok[r] : top[r];
        if (p.out_score) p.out_score[t] = key[r] != 0u ? score[r] : 0.0f;
    }
}

__device__ __forceinline__ unsigned add_acq_rel(unsigned *ptr, unsigned n)
{
    unsigned old;
    asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], %2;" : "=r"(old) : "l"(ptr), "r"(n) : "memory");
    return old;
}

struct BlockReport {                 // in shared memory
    BlockDecide decide;
    int seq[32];                     // the sequence that a row belongs to
    unsigned rows[32];               // how many of the CTA's rows belong to it (with the first of them), else 0
    unsigned complete;               // bit i: the CTA's row i stands for a complete sequence
};

// The CTA has finished (folded and stored, or found not flagged) the rows row0 .. row0 + n - 1 (n <= 32, rows past
// the last one do not count): they are counted in their sequences, one fence and one counter update per
// sequence, and the sequences that this completes are decided.  Every thread of the CTA calls it.
__device__ __forceinline__ void report_rows(const VerifyParams &p, int row0, int n, BlockReport &s)
{
    const unsigned full = 0xFFFFFFFFu;
    const int lane = threadIdx.x & 31;
    if (threadIdx.x >= blockDim.x - 32) {                            // (the first warp may still be folding)
        const int r = row0 + lane;
        const int b = lane < n && (long)r < (long)p.B * p.P ? r / p.P : -1;
        const unsigned same = __match_any_sync(full, b);
        s.seq[lane] = b;
        s.rows[lane] = b >= 0 && lane == __ffs(same) - 1 ? __popc(same) : 0;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        const unsigned count = s.rows[lane];
        bool complete = false;
        if (count > 0) {
            const int b = s.seq[lane];
            // (orders what this CTA stored before the count, and what the others stored before theirs after it)
            complete = add_acq_rel(p.seq_counter + checked(p, b, p.B, kSiteSeq), count) + count == (unsigned)p.P;
            if (complete) p.seq_counter[b] = 0u;                     // ready for the next launch
        }
        const unsigned all = __ballot_sync(full, complete);
        if (lane == 0) s.complete = all;
    }
    __syncthreads();
    for (unsigned m = s.complete; m; m &= m - 1) {
        const int b = s.seq[__ffs(m) - 1];
        if (p.P <= 512 && p.P <= 2 * (int)blockDim.x) decide_block_short(p, b, s.decide);
        else decide_block(p, b, s.decide);
        __syncthreads();
    }
}

}  // namespace ddv
