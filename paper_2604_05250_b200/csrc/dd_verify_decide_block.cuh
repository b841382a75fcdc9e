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
// in one batch and stays in registers, and the k-th largest key is found by warp 0 from keys in registers, bit
// by bit without a barrier, ending as soon as exactly k keys are left above the candidate (12-16 steps; all 32
// only for ties).  1 x 128 positions: 9700 cycles for the general form, of which 4700 for the selection, 6200 for
// this one (cold; with the cheaper report below 2 us of a call).
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
        if (warp == 0) {
            uint32_t kr[16];
#pragma unroll
            for (int r = 0; r < 16; ++r) kr[r] = r * 32 < p.P ? s.key[lane + 32 * r] : 0u;
            auto count_above = [&](uint32_t bound) -> int {
                int c0 = 0, c1 = 0;
#pragma unroll
                for (int r = 0; r < 4; r += 2) { c0 += kr[r] > bound; c1 += kr[r + 1] > bound; }
                if (p.P > 128) {
#pragma unroll
                    for (int r = 4; r < 16; r += 2) { c0 += kr[r] > bound; c1 += kr[r + 1] > bound; }
                }
                return __reduce_add_sync(full, c0 + c1);
            };
            unsigned last = 0xFFFFFFFFu;                 // every position equal to thr
            if (count_above(0u) > p.k) {
                bool exact = false;
#pragma unroll 1
                for (int bit = 31; bit >= 0; --bit) {
                    const uint32_t cand = thr | (1u << bit);
                    const int n = count_above(cand - 1u);
                    if (n >= p.k) thr = cand;
                    if (n == p.k) { exact = true; break; }
                }
                if (!exact) {
                    // ties at the threshold: kept lowest index first
                    int quota = p.k - count_above(thr), seen = 0;
#pragma unroll 1
                    for (int i0 = 0; i0 < p.P; i0 += 32) {
                        const bool eq = s.key[i0 + lane] == thr;
                        const unsigned m = __ballot_sync(full, eq);
                        const int rank = seen + __popc(m & ((1u << lane) - 1u));
                        const unsigned hit = __ballot_sync(full, eq && rank + 1 == quota);
                        if (hit) { last = (unsigned)(i0 + __ffs(hit) - 1); break; }
                        seen += __popc(m);
                    }
                }
            }                                            // else: no more than k, all are kept (thr stays 0)
            if (lane == 0) { s.digit = thr; s.count = last; }
        }
        __syncthreads();
        thr = s.digit;
        last_equal = s.count;
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
    unsigned complete;
};

// The CTA has finished (folded and stored, or found not flagged) the rows row0 .. row0 + n - 1 (n <= 32, rows past
// the last one do not count): they are counted in their sequences, one fence and one counter update per
// sequence, and the sequences that this completes are decided.  Every thread of the CTA calls it.
__device__ __forceinline__ void report_rows(const VerifyParams &p, int row0, int n, BlockReport &s)
{
    const unsigned full = 0xFFFFFFFFu;
    const int lane = threadIdx.x & 31;
    __syncthreads();
    if (threadIdx.x < 32) {
        const int r = row0 + lane;
        const bool valid = lane < n && (long)r < (long)p.B * p.P;
        const int b = valid ? r / p.P : -1;
        const unsigned same = __match_any_sync(full, b);
        bool complete = false;
        if (valid && lane == __ffs(same) - 1) {
            const unsigned count = __popc(same);
            // (orders what this CTA stored before the count, and what the others stored before theirs after it)
            complete = add_acq_rel(p.seq_counter + checked(p, b, p.B, kSiteSeq), count) + count == (unsigned)p.P;
            if (complete) p.seq_counter[b] = 0u;                     // ready for the next launch
        }
        const unsigned all = __ballot_sync(full, complete);          // bit i: row0 + i stands for a complete sequence
        if (lane == 0) s.complete = all;
    }
    __syncthreads();
    for (unsigned m = s.complete; m; m &= m - 1) {
        const int b = (row0 + __ffs(m) - 1) / p.P;
        if (p.P <= 512 && p.P <= 2 * (int)blockDim.x) decide_block_short(p, b, s.decide);
        else decide_block(p, b, s.decide);
        __syncthreads();
    }
}

}  // namespace ddv
