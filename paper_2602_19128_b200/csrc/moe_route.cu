// Router (softmax -> top-k -> renormalise) and the stable sort-scatter by expert.
//
// Paper, Sec. 4.5 "Routing": each token gets scores for E experts and the top k are picked with
// warp-level cooperation; "Expert FFN computation", step (2): tokens are reordered by expert into
// contiguous memory.  Here one warp owns one token (E <= 256 logits fit in 8 registers per lane).  It selects under
// the strict order
//     e before e'  <=>  logit[e] > logit[e']  or  (logit[e] == logit[e'] and e < e')
// by cutting the experts down to a few candidates and ranking those against each other (select_candidates), and the
// sort-scatter is a counting sort made stable without ordered atomics:
//   1. every router block histograms the assignments of its own 32 tokens (one "chunk");
//   2. the [chunk, expert] histogram becomes start positions (scan over chunks, by one block or by a block per 32
//      experts); the one, or the last to finish, scans over the experts and derives the GEMM token-tile schedule;
//   3. one warp per chunk walks its assignments in flat order, 32 at a time, ranking equal
//      experts inside a group with match_any and carrying per-expert counters between groups.
// Batches of up to 1024 tokens do all of it in one launch (route_fused_kernel).
// Integer results are therefore unique and reproducible.
#include "moe_internal.cuh"

#include <limits.h>
#include <math.h>

#include <mutex>

namespace moe {
namespace {

constexpr unsigned kFullMask = 0xffffffffu;
// A chunk's block has a warp per token while every block has an SM of its own, and 16 warps of two tokens each beyond: at
// 64 registers two such blocks fit on an SM, and the 256 blocks of an 8192-token batch run in one wave, not in two.
// Router and sort of 64 experts, top 2, a warp per token / two tokens: 4096 tokens 16.4 / 16.4 us, 1025 14.4 / 15.4; 8192
// 19.5 / 18.4.
constexpr int kRouteThreads = 1024, kRouteThreadsManyChunks = 512, kRouteSms = 148;

// Order-preserving map from float to unsigned: a > b  <=>  ordered_key(a) > ordered_key(b) (for non-NaN values;
// -0 is first folded into +0 so that the two compare equal, as the floats do).
__device__ __forceinline__ unsigned ordered_key(float f) {
    const unsigned u = __float_as_uint(f + 0.0f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// k rounds of a warp arg-max under the strict order (larger key first, ties to the lower expert index).  Expert
// e = 32 i + lane has key[i] in its lane (kRegs = ceil(E / 32), rounded up to 1, 4 or 8); entries with e >= E must hold key 0 and are
// never selected while a real candidate is left.  Each round: every lane finds its best remaining entry, one warp reduction gives the largest
// key, a second one the lowest expert index among the lanes that hold it.  Lane j < k returns rank j's expert.
template <int kRegs>
__device__ __forceinline__ int select_top_k(const unsigned (&key)[kRegs], int E, int k, int lane) {
    unsigned taken = 0;
    int my_id = 0;
    for (int j = 0; j < k; ++j) {
        unsigned best = 0;
        int best_e = INT_MAX;  // no candidate
#pragma unroll
        for (int i = 0; i < kRegs; ++i) {
            const int e = i * 32 + lane;
            const bool free_slot = e < E && !((taken >> i) & 1u);
            if (free_slot && (best_e == INT_MAX || key[i] > best)) { best = key[i]; best_e = e; }
        }
        const unsigned top = __reduce_max_sync(kFullMask, best_e == INT_MAX ? 0u : best);
        int winner = (int)__reduce_min_sync(kFullMask, (best_e != INT_MAX && best == top) ? (unsigned)best_e : 0xffffffffu);
        if (winner < 0 || winner >= E) winner = 0;  // unreachable for k <= E; keeps the index in range regardless
        if ((winner & 31) == lane) taken |= 1u << (winner >> 5);
        if (lane == j) my_id = winner;
    }
    return my_id;
}

// Per-warp scratch of select_candidates.
struct Candidates {
    unsigned key[32];
    int e[32];
    float score[32];
};

// The k first experts under the strict order, cut down to candidates first.  Among the 32 lane maxima the k-th largest is
// a bound that at least k experts reach (equal maxima are struck out together, which only lowers it); the experts that
// reach it -- k and a few on ordinary logits -- are collected in ascending index order, one per lane, and every candidate
// counts the candidates before it.  More than 32 candidates (many equal logits, k near 32) fall back to select_top_k.
// About half the warp instructions, at E = 256 and k = 8, of k rounds of a full arg-max over eight registers, and a chain
// of k short reductions instead of k long ones (8192 tokens: router and sort 43 -> 25 us, grouped 56 -> 33 us).
// k = 1 is a single arg-max (route_topk_kernel, 1500 tokens of 32 experts: 5.8 -> 5.1 us).
// Lane j < k returns rank j's expert with its key and score.
template <int kRegs>
__device__ __forceinline__ void select_candidates(const unsigned (&key)[kRegs], const float (&score)[kRegs], int E,
                                                  int k, int lane, Candidates *c, int &my_id, unsigned &my_key, float &my_score) {
    if (k == 1) {  // one arg-max
        unsigned best = key[0];
        int e = lane;
        float v = score[0];
#pragma unroll
        for (int i = 1; i < kRegs; ++i)
            if (key[i] > best) { best = key[i]; e = i * 32 + lane; v = score[i]; }
        my_key = __reduce_max_sync(kFullMask, lane < E ? best : 0u);
        my_id = (int)__reduce_min_sync(kFullMask, lane < E && best == my_key ? (unsigned)e : (unsigned)INT_MAX);
        my_score = __shfl_sync(kFullMask, v, my_id & 31);
        return;
    }
    int n;
    unsigned cand_key = key[0];
    int cand_e = lane;
    float cand_score = score[0];
    if (E <= 32) {  // every expert is a candidate, in its own lane already
        n = E;
    } else {
        unsigned m = key[0];
#pragma unroll
        for (int i = 1; i < kRegs; ++i) m = max(m, key[i]);
        unsigned bound = 0;
        for (int j = 0; j < k; ++j) {
            bound = __reduce_max_sync(kFullMask, m);
            if (m == bound) m = 0;
        }
        n = 0;
#pragma unroll
        for (int i = 0; i < kRegs; ++i) {
            const bool in = key[i] >= bound;  // (a bound of 0 takes all slots, 128 or 256: the fallback)
            const unsigned mask = __ballot_sync(kFullMask, in);
            const int at = n + __popc(mask & ((1u << lane) - 1u));
            if (in && at < 32) { c->key[at] = key[i]; c->e[at] = i * 32 + lane; c->score[at] = score[i]; }
            n += __popc(mask);
        }
        __syncwarp();
        if (n > 32) {
            my_id = select_top_k(key, E, k, lane);
            my_key = 0;
            my_score = 0.f;
#pragma unroll
            for (int i = 0; i < kRegs; ++i) {  // expert my_id lives in lane my_id % 32, register my_id / 32
                const unsigned got_key = __shfl_sync(kFullMask, key[i], my_id & 31);
                const float got_score = __shfl_sync(kFullMask, score[i], my_id & 31);
                if ((my_id >> 5) == i) { my_key = got_key; my_score = got_score; }
            }
            return;
        }
        if (lane < n) { cand_key = c->key[lane]; cand_e = c->e[lane]; cand_score = c->score[lane]; }
    }
    int rank = 0;
#pragma unroll 4
    for (int j = 0; j < n; ++j) {
        const unsigned other = __shfl_sync(kFullMask, cand_key, j);
        rank += (other > cand_key || (other == cand_key && j < lane)) ? 1 : 0;
    }
    __syncwarp();
    if (lane < n && rank < k) { c->key[rank] = cand_key; c->e[rank] = cand_e; c->score[rank] = cand_score; }
    __syncwarp();
    my_id = lane < k ? c->e[lane] : 0;
    my_key = lane < k ? c->key[lane] : 0u;
    my_score = lane < k ? c->score[lane] : 0.f;
    __syncwarp();  // (the next token of this warp writes here)
}

// Router for one token by one warp: top-k of the E logits (kRegs per lane) under the strict order, then the
// renormalised softmax weights.  Softmax's normaliser cancels in the renormalisation, so only the k selected
// logits are exponentiated: w_j = exp(l_j - l_0) / sum_j' exp(l_j' - l_0), the sum in rank order.
// Lane j < k returns rank j's expert and weight.
template <int kRegs>
__device__ __forceinline__ void route_one_token(const float *__restrict__ row, int E, int k, int lane, Candidates *cand, int &my_id,
                                                float &my_w) {
    float v[kRegs];
    unsigned key[kRegs];
#pragma unroll
    for (int i = 0; i < kRegs; ++i) {
        const int e = i * 32 + lane;
        v[i] = e < E ? row[e] : 0.f;
        key[i] = e < E ? ordered_key(v[i]) : 0u;
    }
    unsigned my_key;
    float my_l;
    select_candidates(key, v, E, k, lane, cand, my_id, my_key, my_l);
    const float top_l = __shfl_sync(kFullMask, my_l, 0);  // rank 0 holds the largest logit
    const float my_p = lane < k ? expf(my_l - top_l) : 0.f;
    float denom = 0.f;  // ascending rank, the order the definition states
    for (int j = 0; j < k; ++j) denom += __shfl_sync(kFullMask, my_p, j);
    my_w = my_p / denom;
}

// ---- grouped sigmoid router ("DeepSeek-V3 style" routing, Sec. 4.5) ---------------------------------------
// Selection is an integer decision taken from floating-point values, so every operation that feeds it is one
// correctly rounded binary32 operation in a fixed order (the _rn intrinsics keep the compiler from fusing or
// reassociating them); e^x follows a fixed recipe: clamp to [-87, 88], n = nearest integer of x * log2(e),
// r = x - n * ln 2 (ln 2 in two parts, fused multiply-adds), degree-7 Taylor polynomial in Horner form, times 2^n.
__device__ __forceinline__ float exp_fixed(float x) {
    x = fminf(fmaxf(x, -87.0f), 88.0f);
    const float n = rintf(__fmul_rn(x, 1.44269502f));
    float r = __fmaf_rn(n, -0.693145752f, x);
    r = __fmaf_rn(n, -1.42860677e-06f, r);
    float p = 1.98412701e-04f;
    p = __fmaf_rn(p, r, 1.38888892e-03f);
    p = __fmaf_rn(p, r, 8.33333377e-03f);
    p = __fmaf_rn(p, r, 4.16666679e-02f);
    p = __fmaf_rn(p, r, 1.66666672e-01f);
    p = __fmaf_rn(p, r, 0.5f);
    p = __fmaf_rn(p, r, 1.0f);
    p = __fmaf_rn(p, r, 1.0f);
    return __fmul_rn(p, __int_as_float(((int)n + 127) << 23));
}
// (the reciprocal is correctly rounded, as the quotient 1 / x is: the same result for fewer instructions)
__device__ __forceinline__ float sigmoid_fixed(float l) { return __frcp_rn(__fadd_rn(1.0f, exp_fixed(-l))); }

// Merge two (largest, second largest) pairs.
__device__ __forceinline__ void top2_merge(float &t1, float &t2, float o1, float o2) {
    const float lo = fminf(t1, o1);
    t1 = fmaxf(t1, o1);
    t2 = fmaxf(lo, fmaxf(t2, o2));
}

// One token by one warp.  Expert e = 32 i + lane lives in register i of its lane; a group is G = E / n_group
// consecutive experts, G a power of two: either a segment of G lanes within one register index (G <= 32) or all
// lanes of G / 32 consecutive register indices.
template <int kRegs>
__device__ __forceinline__ void route_one_token_grouped(const float *__restrict__ row, int E, int k, int lane,
                                                        const RouterParams &rp, Candidates *cand, int &my_id, float &my_w) {
    const int G = E / rp.n_group;
    // All loads, then all sigmoids, then what does not exist is put right.  (With a condition around each expert's load and sigmoid
    // the eight of a lane ran one after the other, each behind its own load: router and sort of 8192 tokens of 256 experts, top 8, 31.1 ->
    // 28.7 us, 1056 tokens 22.6 -> 20.5.)
    float s[kRegs], c[kRegs];
#pragma unroll
    for (int i = 0; i < kRegs; ++i) {
        const int e = i * 32 + lane;
        s[i] = e < E ? row[e] : 0.f;
        c[i] = e < E && rp.bias ? rp.bias[e] : 0.f;
    }
#pragma unroll
    for (int i = 0; i < kRegs; ++i) {
        s[i] = sigmoid_fixed(s[i]);
        if (rp.bias) c[i] = __fadd_rn(s[i], c[i]); else c[i] = s[i];
    }
#pragma unroll
    for (int i = 0; i < kRegs; ++i)
        if (i * 32 + lane >= E) { s[i] = 0.f; c[i] = -INFINITY; }
    if (G == 32) {
        // Groups of 32 (256 experts in 8 groups): register i of all lanes is group i.  The eight reductions over 32 lanes
        // are folded into one by halving: each exchange leaves a lane half of the groups, so 9 exchanges of a pair do the
        // work of 40, and lane l ends with the group whose number is the bits 16, 8, 4 of l.
        float a1[4], a2[4];
        const bool b16 = (lane & 16) != 0, b8 = (lane & 8) != 0, b4 = (lane & 4) != 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {  // (a single score has no second: -inf)
            const float lo = i < kRegs ? c[i % kRegs] : -INFINITY, hi = 4 + i < kRegs ? c[(4 + i) % kRegs] : -INFINITY;
            const float o1 = __shfl_xor_sync(kFullMask, b16 ? lo : hi, 16);
            a1[i] = b16 ? hi : lo;
            a2[i] = -INFINITY;
            top2_merge(a1[i], a2[i], o1, -INFINITY);
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const float o1 = __shfl_xor_sync(kFullMask, b8 ? a1[i] : a1[2 + i], 8);
            const float o2 = __shfl_xor_sync(kFullMask, b8 ? a2[i] : a2[2 + i], 8);
            a1[i] = b8 ? a1[2 + i] : a1[i];
            a2[i] = b8 ? a2[2 + i] : a2[i];
            top2_merge(a1[i], a2[i], o1, o2);
        }
        {
            const float o1 = __shfl_xor_sync(kFullMask, b4 ? a1[0] : a1[1], 4), o2 = __shfl_xor_sync(kFullMask, b4 ? a2[0] : a2[1], 4);
            a1[0] = b4 ? a1[1] : a1[0];
            a2[0] = b4 ? a2[1] : a2[0];
            top2_merge(a1[0], a2[0], o1, o2);
        }
#pragma unroll
        for (int off = 2; off > 0; off >>= 1) {
            const float o1 = __shfl_xor_sync(kFullMask, a1[0], off), o2 = __shfl_xor_sync(kFullMask, a2[0], off);
            top2_merge(a1[0], a2[0], o1, o2);
        }
        const float mine = __fadd_rn(a1[0], a2[0]);
        const int gid = (b16 ? 4 : 0) + (b8 ? 2 : 0) + (b4 ? 1 : 0);
        // a group is eligible if fewer than topk_group groups rank before it (ties to the lower group index)
        int rank = 0;
        for (int g = 0; g < rp.n_group; ++g) {
            const float val = __shfl_sync(kFullMask, mine, g * 4);
            rank += (val > mine || (val == mine && g < gid)) ? 1 : 0;
        }
        const unsigned eligible = __ballot_sync(kFullMask, gid < rp.n_group && rank < rp.topk_group);  // group g: bit 4 g
#pragma unroll
        for (int i = 0; i < kRegs; ++i)
            if (!((eligible >> (4 * i)) & 1u)) c[i] = -INFINITY;
    } else {
        // the two largest biased scores of every group
        float t1[kRegs], t2[kRegs];
#pragma unroll
        for (int i = 0; i < kRegs; ++i) {
            t1[i] = c[i];
            t2[i] = -INFINITY;
        }
        if (G > 32) {  // registers of the same group first
            const int m = G >> 5;
#pragma unroll
            for (int i = 0; i < kRegs; ++i) {
                const int first = i & ~(m - 1);
                float a1 = -INFINITY, a2 = -INFINITY;
#pragma unroll
                for (int j = 0; j < kRegs; ++j)
                    if (j >= first && j < first + m) top2_merge(a1, a2, c[j], -INFINITY);
                t1[i] = a1;
                t2[i] = a2;
            }
        }
        for (int off = (G < 32 ? G : 32) >> 1; off > 0; off >>= 1) {
#pragma unroll
            for (int i = 0; i < kRegs; ++i) {
                const float o1 = __shfl_xor_sync(kFullMask, t1[i], off), o2 = __shfl_xor_sync(kFullMask, t2[i], off);
                top2_merge(t1[i], t2[i], o1, o2);
            }
        }
        float gs[kRegs];  // score of the group that holds this register's expert
#pragma unroll
        for (int i = 0; i < kRegs; ++i) gs[i] = G >= 2 ? __fadd_rn(t1[i], t2[i]) : t1[i];
        // a group is eligible if fewer than topk_group groups rank before it (ties to the lower group index)
        if (rp.n_group <= 32) {
            // lane g fetches group g's score from the lane and register that hold the group's first expert ...
            const int first = lane < rp.n_group ? lane * G : 0;
            float mine = 0.f;
#pragma unroll
            for (int i = 0; i < kRegs; ++i) {
                const float got = __shfl_sync(kFullMask, gs[i], first & 31);
                if ((first >> 5) == i) mine = got;
            }
            // ... ranks it against the others, and the eligible groups become a bit mask
            int rank = 0;
            for (int g = 0; g < rp.n_group; ++g) {
                const float val = __shfl_sync(kFullMask, mine, g);
                rank += (val > mine || (val == mine && g < lane)) ? 1 : 0;
            }
            const unsigned eligible = __ballot_sync(kFullMask, lane < rp.n_group && rank < rp.topk_group);
#pragma unroll
            for (int i = 0; i < kRegs; ++i)
                if (!((eligible >> ((i * 32 + lane) / G)) & 1u)) c[i] = -INFINITY;
        } else {  // more groups than lanes (groups of at most 4 experts): every register ranks its own group
            int rank[kRegs];
#pragma unroll
            for (int i = 0; i < kRegs; ++i) rank[i] = 0;
            for (int g = 0; g < rp.n_group; ++g) {
                const int e0 = g * G, ip = e0 >> 5;
                float pick = gs[0];
#pragma unroll
                for (int i = 1; i < kRegs; ++i) pick = ip == i ? gs[i] : pick;
                const float val = __shfl_sync(kFullMask, pick, e0 & 31);
#pragma unroll
                for (int i = 0; i < kRegs; ++i) {
                    const int gid = (i * 32 + lane) / G;
                    rank[i] += (val > gs[i] || (val == gs[i] && g < gid)) ? 1 : 0;
                }
            }
#pragma unroll
            for (int i = 0; i < kRegs; ++i)
                if (rank[i] >= rp.topk_group) c[i] = -INFINITY;
        }
    }

    // top-k of the eligible biased scores; the weight uses the unbiased score of the selected expert
    unsigned key[kRegs];
#pragma unroll
    for (int i = 0; i < kRegs; ++i) key[i] = i * 32 + lane < E ? ordered_key(c[i]) : 0u;
    unsigned my_key;
    float my_s;
    select_candidates(key, s, E, k, lane, cand, my_id, my_key, my_s);
    if (lane >= k) my_s = 0.f;
    float denom = 0.f;  // ascending rank
    for (int j = 0; j < k; ++j) denom = __fadd_rn(denom, __shfl_sync(kFullMask, my_s, j));
    my_w = __fmul_rn(__fdiv_rn(my_s, denom), rp.scale);
}

constexpr uint32_t kNoIds = 0xFFFFFFFFu;
// Routes tokens [t0, t1) of the block (warp w takes tokens t0 + w, t0 + w + n_warps, ...) and writes ids and weights;
// hist, if given, collects the histogram over the resident experts (zeroed by the caller); all tokens' ids are left, a byte each,
// in the array at address ids_smem of the cluster's shared memory too, if there is one (0 would be an address; kNoIds is none).
template <int kRegs>
__device__ __forceinline__ void route_tokens(const float *__restrict__ logits, int t0, int t1, int E, int k, int local_offset,
                                             int n_local, const RouterParams &rp, int *topk_ids, float *topk_w, Candidates *cand,
                                             int *hist, uint32_t ids_smem = kNoIds) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
#pragma unroll 1
    for (int t = t0 + warp; t < t1; t += n_warps) {
        int my_id;
        float my_w;
        if (rp.grouped)
            route_one_token_grouped<kRegs>(logits + (size_t)t * E, E, k, lane, rp, &cand[warp], my_id, my_w);
        else
            route_one_token<kRegs>(logits + (size_t)t * E, E, k, lane, &cand[warp], my_id, my_w);
        if (lane < k) {
            topk_ids[(size_t)t * k + lane] = my_id;
            topk_w[(size_t)t * k + lane] = my_w;
            if (ids_smem != kNoIds)
                asm volatile("st.shared::cluster.u8 [%0], %1;" ::"r"(ids_smem + (uint32_t)(t * k + lane)), "r"(my_id) : "memory");
            const int local = my_id - local_offset;  // only experts resident here are scheduled
            if (hist && local >= 0 && local < n_local) atomicAdd(&hist[local], 1);
        }
    }
}

// The tile schedule is in memory: a forward call's GEMMs, which may be resident already, start on it (gemm_chain_start).  By
// one thread, behind a block barrier that follows the last write of the schedule.
// A kernel in front of the call may have written the weights through the generic proxy, and no wait for a grid stands between it
// and the GEMMs' first TMA copies of them, only this flag: the thread that will raise it links the two by a proxy fence
// (fence_weights), behind its own wait for what is in front and far ahead of the flag, where it costs nothing (in front of the
// copies it cost 0.15 us of the tiny layer's 19.6).  The token side has a fence of its own (handover_wait_expert).
__device__ __forceinline__ void fence_weights() { asm volatile("fence.proxy.async.global;" ::: "memory"); }
__device__ __forceinline__ void raise_schedule_flag(int *status) {
    asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(status + kHandoverFlagInt), "r"(1) : "memory");
}

template <int kThreads, int kRegs>
__global__ void __launch_bounds__(kThreads, 1024 / kThreads)
route_topk_kernel(const float *__restrict__ logits, int T, int E, int k, int local_offset, int n_local,
                  const RouterParams rp, int *__restrict__ topk_ids, float *__restrict__ topk_w,
                  int *__restrict__ chunk_counts) {
    __shared__ int hist[kMaxExperts];  // indexed by local expert (expert id - local_offset)
    __shared__ Candidates cand[kThreads / 32];
    chain_release();
    for (int e = threadIdx.x; e < n_local; e += kThreads) hist[e] = 0;
    __syncthreads();
    chain_wait();
    const int t0 = blockIdx.x * kRouteTokensPerBlock;
    route_tokens<kRegs>(logits, t0, min(T, t0 + kRouteTokensPerBlock), E, k, local_offset, n_local, rp, topk_ids, topk_w, cand, hist);
    __syncthreads();
    for (int e = threadIdx.x; e < n_local; e += kThreads) chunk_counts[(size_t)blockIdx.x * n_local + e] = hist[e];
}

constexpr int kScanThreads = 1024;

// Inclusive prefix sum over the lanes of a warp.
__device__ __forceinline__ int warp_inclusive_scan(int v, int lane) {
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int n = __shfl_up_sync(kFullMask, v, off);
        if (lane >= off) v += n;
    }
    return v;
}

// The schedule's row quantum with ceil(2^32 / q): the rows of a tile are rounded up without a division.  n / q is the upper half of
// n * inverse for every n with n q < 2^32, tiles and quanta being 384 at most; a quantum of 1 has no 32-bit inverse (launch_route
// refuses it).
constexpr int kMaxTileRows = 384;
struct RowQuantum {
    int q;
    unsigned inverse;
    constexpr explicit RowQuantum(int quantum) : q(quantum), inverse((unsigned)(((1ull << 32) + quantum - 1) / quantum)) {}
    static constexpr bool valid(int quantum) { return quantum >= 2 && quantum <= kMaxTileRows; }
};
constexpr bool divides_exactly(int quantum) {
    for (unsigned n = 0; n < 2 * kMaxTileRows; ++n)
        if ((unsigned)(((unsigned long long)n * RowQuantum(quantum).inverse) >> 32) != n / quantum) return false;
    return true;
}
static_assert(divides_exactly(2) && divides_exactly(16) && divides_exactly(32) && divides_exactly(64) && divides_exactly(128) &&
              divides_exactly(160) && divides_exactly(240) && divides_exactly(kMaxTileRows), "rounding a tile's rows");

// Schedule phase, run by one block of 1024 threads: exclusive scan over the experts' row counts and the token-tile
// schedule.  `count` is expert threadIdx.x's rows in threads 0..E-1 and 0 in the others; `started(row)` is called by
// thread e < E with expert e's first row, and what it writes is visible to the block on return.  The schedule's flag is
// raised (by the first thread of the last warp) as soon as the schedule is in memory.
// This is a chain of short steps, between the router's last id and everything else of the call: two block barriers, the
// first scan and the ranking side by side, the second scan by one warp, beside whatever the caller does next.  (With a
// barrier per step -- twelve -- and a thousand threads counting spans of a few ids, the tiny layer's 32 ids took 3.9 us
// from the last id to the flag; now 2.5.)  Every instruction runs once or a few times per call, so what is not a loop costs its
// fetch more than its issue: loops are unrolled only where loads have to overlap.
struct ScheduleShared {
    int warp_sums[kMaxExperts / 32];
    __align__(16) unsigned keys[kMaxExperts];
    __align__(16) int tiles_at[kMaxExperts];
    int tiles[kMaxExperts];
};
template <typename Started>
__device__ __forceinline__ void schedule_phase(int count, int E, int nt_max, RowQuantum row_quantum, int *expert_offsets, int *tile_prefix,
                                               int *tile_order, int *tile_rows, int *status, ScheduleShared &sh, Started started) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int incl = 0;
    if (tid < kMaxExperts) {
        // More rows first, ties to the lower index: one unsigned number per expert (past 2^24 rows the order is the index's).
        sh.keys[tid] = ((unsigned)min(count, 0xFFFFFF) << 8) | (unsigned)(kMaxExperts - 1 - tid);
        incl = warp_inclusive_scan(count, lane);
        if (lane == 31) sh.warp_sums[warp] = incl;
        // token tiles of this expert: one tile if it fits under nt_max; otherwise as few as fit under min(nt_max, 256) --
        // a wide bound (320 / 384) exists to keep an expert in ONE pass over its weights, and consecutive tiles wider than
        // half of tensor memory cannot overlap their epilogues, so experts that need several tiles get 256-row ones --
        // evenly sized, rounded up to the row quantum
        // (16 rows, the MMA's N granularity; the MX path with a bound of up to 256 passes its tile size, so that every tile
        // is exactly that many rows)
        int n_tiles = 0, rows = 0;
        if (count > 0) {
            const int multi = nt_max > 256 ? 256 : nt_max;
            n_tiles = count <= nt_max ? 1 : (count + multi - 1) / multi;
            const int per_tile = n_tiles == 1 ? count : (count + n_tiles - 1) / n_tiles;
            rows = (int)__umulhi((unsigned)(per_tile + row_quantum.q - 1), row_quantum.inverse) * row_quantum.q;
        }
        sh.tiles[tid] = n_tiles;
        if (tid < E) tile_rows[tid] = rows; else sh.tiles_at[tid] = 0;
    }
    __syncthreads();
    // Schedule order: experts with more rows first (ties to the lower index), so that tiles of similar cost are adjacent and
    // the GEMMs' static tile assignment stays balanced; the small tiles come last.  All-pairs ranking, E^2 comparisons: four
    // neighbouring threads share an expert's opponents, four per load.
    {
        const int e = tid >> 2, part = tid & 3;
        int before = 0;
        if (e < E) {
            const unsigned mine = sh.keys[e];
#pragma unroll 2
            for (int o = part * 4; o < E; o += 16) {  // (keys past E rank behind every real one)
                const uint4 c = *reinterpret_cast<const uint4 *>(&sh.keys[o]);
                before += (c.x > mine) + (c.y > mine) + (c.z > mine) + (c.w > mine);
            }
        }
        before += __shfl_xor_sync(kFullMask, before, 1);
        before += __shfl_xor_sync(kFullMask, before, 2);
        if (e < E && part == 0) {
            sh.tiles_at[before] = sh.tiles[e];
            tile_order[before] = e;
        }
    }
    if (tid < kMaxExperts) {
        int base = 0, total = 0;
#pragma unroll
        for (int w = 0; w < kMaxExperts / 32; ++w) {
            const int v = sh.warp_sums[w];
            if (w < warp) base += v;
            total += v;
        }
        if (tid < E) {
            const int row = base + incl - count;
            expert_offsets[tid] = row;
            started(row);
        }
        if (tid == 0) expert_offsets[E] = total;
    }
    __syncthreads();
    if (warp == kScanThreads / 32 - 1) {  // tile counts in schedule order -> first tile of each position
        int v[8], sum = 0;
#pragma unroll
        for (int i = 0; i < 2; ++i)
            *reinterpret_cast<int4 *>(&v[4 * i]) = *reinterpret_cast<const int4 *>(&sh.tiles_at[lane * 8 + 4 * i]);
#pragma unroll
        for (int i = 0; i < 8; ++i) sum += v[i];
        int at = warp_inclusive_scan(sum, lane) - sum;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            if (lane * 8 + i <= E) tile_prefix[lane * 8 + i] = at;
            at += v[i];
        }
        if (E == kMaxExperts && lane == 31) tile_prefix[E] = at;
        __syncwarp();
        if (lane == 0) raise_schedule_flag(status);
    }
}

// Scan over the chunks, in groups of 32 experts: a warp takes a contiguous share of the chunks for one group, lane l its
// l-th expert, so that a load is one 128-byte line and up to kScanBatch of them are in flight per thread.  The counts are
// replaced by the rows of all earlier chunks.  Either one block takes all groups, a share of its warps each, and goes
// straight on to the schedule phase; or every block takes a group, and the one that finishes last (a counter zeroed by the
// call's memset) has every expert's total and runs the schedule phase.  Several blocks share the traffic of many chunks
// (256 chunks, up to 256 KB in and out of one SM: 17-24 us by one block, 9-10 us by eight), but their hand-over costs 2 us:
// one block while its threads hold all their counts in registers (kScanBatch).  Router and sort, one block / several:
// 1500 tokens, 64 experts, top 2 14.4 / 16.5 us; 4096, 128, 8 18.5 / 20.5; 2400, 256, 8 22.6 / 20.5; 8192, 256, 8 32.8 /
// 24.6.  A share has at least four chunks: the block's threads add up the shares one after the other (1500 tokens of 8
// experts 14.3 -> 12.3 us).
constexpr int kScanWarps = kScanThreads / 32, kScanBatch = 16, kScanLeast = 4;
__host__ __device__ inline int scan_warps_per_group(int n_chunks, int groups) {
    const int most = kScanWarps / groups, useful = (n_chunks + kScanLeast - 1) / kScanLeast;
    return useful < most ? useful : most;
}
__global__ void __launch_bounds__(kScanThreads)
route_scan_kernel(int *chunk_counts, int n_chunks, int E, int nt_max, RowQuantum row_quantum, int *expert_offsets,
                  int *tile_prefix, int *tile_order, int *tile_rows, int *totals, int *status) {
    __shared__ int partial[kScanWarps][32], all_totals[kMaxExperts];
    __shared__ ScheduleShared sh;
    __shared__ int is_last;
    const bool one_block = gridDim.x == 1;
    const int groups = one_block ? (E + 31) / 32 : 1, warps_per_group = scan_warps_per_group(n_chunks, groups);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, group = warp / warps_per_group, share = warp - group * warps_per_group;
    const int e = group < groups ? ((one_block ? group : (int)blockIdx.x) * 32 + lane) : E;  // (warps left over: no expert)
    chain_release();
    chain_wait();
    if (threadIdx.x == kScanThreads - 32) fence_weights();  // (the thread that raises the schedule's flag)
    const int per = (n_chunks + warps_per_group - 1) / warps_per_group;
    const int b_begin = min(n_chunks, share * per), b_end = min(n_chunks, b_begin + per);
    const bool one_batch = per <= kScanBatch;  // then the counts stay in registers between the passes
    int first[kScanBatch];
    int sum = 0;
    for (int b0 = b_begin; b0 < b_end; b0 += kScanBatch) {
        int c[kScanBatch];
#pragma unroll
        for (int i = 0; i < kScanBatch; ++i) c[i] = e < E && b0 + i < b_end ? __ldcg(&chunk_counts[(size_t)(b0 + i) * E + e]) : 0;
#pragma unroll
        for (int i = 0; i < kScanBatch; ++i) {
            sum += c[i];
            if (one_batch) first[i] = c[i];
        }
    }
    partial[warp][lane] = sum;
    __syncthreads();
    int run = 0, total = 0;
    if (e < E) {
#pragma unroll 4
        for (int w = 0; w < warps_per_group; ++w) {
            const int v = partial[group * warps_per_group + w][lane];
            if (w < share) run += v;
            total += v;
        }
    }
    if (e < E) {
        for (int b0 = b_begin; b0 < b_end; b0 += kScanBatch) {
            int c[kScanBatch];
#pragma unroll
            for (int i = 0; i < kScanBatch; ++i)
                c[i] = one_batch ? first[i] : (b0 + i < b_end ? __ldcg(&chunk_counts[(size_t)(b0 + i) * E + e]) : 0);
#pragma unroll
            for (int i = 0; i < kScanBatch; ++i) {
                if (b0 + i < b_end) chunk_counts[(size_t)(b0 + i) * E + e] = run;
                run += c[i];
            }
        }
        if (share == 0) {
            if (one_block) all_totals[e] = total; else totals[e] = total;
        }
    }
    int count = 0;
    if (one_block) {
        __syncthreads();
        if ((int)threadIdx.x < E) count = all_totals[threadIdx.x];
    } else {
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) is_last = atomicAdd(status + kDoneCounterInt, 1) == (int)gridDim.x - 1;
        __syncthreads();
        if (!is_last) return;
        __threadfence();
        if ((int)threadIdx.x < E) count = __ldcg(&totals[threadIdx.x]);
        __syncthreads();  // (the totals may sit where the schedule is written)
    }
    schedule_phase(count, E, nt_max, row_quantum, expert_offsets, tile_prefix, tile_order, tile_rows, status, sh, [](int) {});
}

// Stable scatter of 32 consecutive assignments by one warp: lane l holds assignment a (flat order) of local expert e;
// next[] is the warp's per-expert cursor.
__device__ __forceinline__ void scatter_group(int e, int a, bool valid, int n_local, int *next, int *sorted_to_flat,
                                              int *flat_to_sorted, int lane) {
    const bool kept = valid && e >= 0 && e < n_local;  // assignments to experts that are not resident are dropped
    const int key = kept ? e : -1 - lane;             // ... and never match anything
    const unsigned same = __match_any_sync(kFullMask, key);
    const int rank = __popc(same & ((1u << lane) - 1u));
    const int pos = kept ? next[e] + rank : -1;
    __syncwarp();
    if (kept && rank == 0) next[e] += __popc(same);
    __syncwarp();
    if (valid) flat_to_sorted[a] = pos;
    if (kept) sorted_to_flat[pos] = a;
}

// Stable scatter of one chunk (32 tokens) by one warp; next[] is that warp's per-expert cursor.
__device__ __forceinline__ void scatter_chunk(int chunk, const int *topk_ids, const int *chunk_starts,
                                              const int *expert_offsets, int A, int n_local, int local_offset, int k,
                                              int *sorted_to_flat, int *flat_to_sorted, int *next, int lane) {
    // first position of this chunk's assignments to expert e = segment start + rows of earlier chunks
    // (all loads issued before the first use: the loop is a chain of L2 round trips otherwise)
    {
        int start[kMaxExperts / 32];
#pragma unroll
        for (int i = 0; i < kMaxExperts / 32; ++i) {
            const int e = i * 32 + lane;
            start[i] = e < n_local ? __ldcg(&expert_offsets[e]) + __ldcg(&chunk_starts[(size_t)chunk * n_local + e]) : 0;
        }
#pragma unroll
        for (int i = 0; i < kMaxExperts / 32; ++i)
            if (i * 32 + lane < n_local) next[i * 32 + lane] = start[i];
    }
    __syncwarp();
    const int a0 = chunk * kRouteTokensPerBlock * k;
    const int a1 = min(A, a0 + kRouteTokensPerBlock * k);
    constexpr int kAhead = 4;  // groups of 32 assignments whose ids are fetched together
    for (int base0 = a0; base0 < a1; base0 += 32 * kAhead) {
        int ids[kAhead];
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
            const int a = base0 + u * 32 + lane;
            ids[u] = a < a1 ? __ldcg(&topk_ids[a]) - local_offset : -1;
        }
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
            const int a = base0 + u * 32 + lane;
            if (base0 + u * 32 >= a1) break;  // uniform over the warp
            scatter_group(ids[u], a, a < a1, n_local, next, sorted_to_flat, flat_to_sorted, lane);
        }
    }
}

__global__ void __launch_bounds__(32)
route_scatter_kernel(const int *topk_ids, const int *chunk_starts, const int *expert_offsets, int A, int n_local,
                     int local_offset, int k, int *sorted_to_flat, int *flat_to_sorted) {
    __shared__ int next[kMaxExperts];
    chain_release();
    chain_wait();
    scatter_chunk(blockIdx.x, topk_ids, chunk_starts, expert_offsets, A, n_local, local_offset, k, sorted_to_flat,
                  flat_to_sorted, next, threadIdx.x);
}

// Small batches (at most 1024 tokens): everything in ONE launch.  The tokens are dealt out to up to 64 blocks (a token is a
// chain of warp reductions: spread over the SMs, not queued on a few); one block -- the first of a cluster, or the one that
// finishes last (a counter in the status word's padding) -- sorts all assignments from their ids alone: warp w takes the
// w-th span of the flat order, counts it, turns the counts into start positions and walks it as scatter_chunk does.
// Which block is last does not affect any result.
// Counts, starts and cursors stay in shared memory: through global memory each hand-over cost an L2 round trip, and with
// one warp per 32 tokens the walk of 1024 assignments ran on four warps.  Measured as a call of its own (replayed): 22.6 ->
// 14.2 us at 128 tokens of 256 experts, 28.7 -> 16.4 us with the grouped router, 11.8 -> 8.2 us at 16 tokens of 8.
constexpr int kFusedThreads = 1024;
constexpr int kFusedMaxChunks = 32;  // of kRouteTokensPerBlock tokens
constexpr int kFusedWarps = kFusedThreads / 32;
// Two ways from the blocks to the one that sorts.  Up to 16 tokens: one block.  Up to 256 (and kFusedClusterIds ids): the blocks are
// a cluster of eight, which leave their ids in the first one's shared memory and meet at the cluster's barrier; that
// block also zeroes the call's status region, so the call needs neither a memset in front nor an atomic count and a trip of
// the ids through L2.  Beyond, eight SMs would have more than a token per warp, and up to 64 blocks count themselves.
// Layers, 64 blocks / a cluster: 100 tokens of 8 experts of 256 x 512, top 2, 23.6 / 21.5 us; 64 tokens of 32 of 1024 x 1024,
// top 4, 57.6 / 54.8; 64 tokens on 32 of 256 bf16 experts of 7168 x 2048, top 8, grouped router, 361.9 / 355.7.
constexpr int kFusedOneBlockTokens = 16, kFusedClusterTokens = 256, kFusedCluster = 8, kFusedClusterIds = 2048;
constexpr int kFusedIds = 8192;  // ids the sorting block holds in shared memory, a byte each; further ones are read where they lie
constexpr int kFusedAhead = 4;   // ... in groups of 32, so many together
// Spans of the flat order, one per sorting warp: at least four groups of 32 each, since every further span is one more count
// per expert to add up.
constexpr int kFusedSpanGroups = 4;
inline int fused_spans(int A) {
    const int useful = (A + 32 * kFusedSpanGroups - 1) / (32 * kFusedSpanGroups);
    return useful < kFusedWarps ? useful : kFusedWarps;
}

template <int kRegs>
__global__ void __launch_bounds__(kFusedThreads)
route_fused_kernel(const float *__restrict__ logits, int T, int E, int k, int local_offset, int n_local, int nt_max,
                   RowQuantum row_quantum, int tokens_per_block, int spans, int span, const RouterParams rp, int *topk_ids, float *topk_w,
                   int *expert_offsets, int *tile_prefix, int *tile_order, int *tile_rows, int *sorted_to_flat, int *flat_to_sorted,
                   int *status, int status_ints) {
    __shared__ ScheduleShared sh;
    __shared__ union Scratch {
        Candidates cand[kFusedWarps];        // while routing
        int next[kFusedWarps][kMaxExperts];  // then: counts, start positions, cursors of each warp's span
    } u;
    __shared__ int is_last;
    __shared__ __align__(16) unsigned char ids_here[kFusedIds];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool ids_local = status_ints > 0;  // one block or a cluster: the first block sorts from its shared memory
    const bool cluster = ids_local && gridDim.x > 1;
    if (cluster) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");  // (the blocks have started)
    if (ids_local) {
        // The first block's last warp zeroes the call's status region, before any kernel that looks at it may start; the
        // others go on (a block that waited for the zeroes routed its tokens half a microsecond later).
        chain_wait();
        if (warp == kFusedWarps - 1) {
            if (blockIdx.x == 0) {
                for (int i = lane; i < status_ints / 4; i += 32) reinterpret_cast<int4 *>(status)[i] = make_int4(0, 0, 0, 0);
                __threadfence();
                __syncwarp();
            }
            if (lane == 0) chain_release();
        }
    } else {
        chain_release();
        chain_wait();
    }
    if (tid == kFusedThreads - 32) fence_weights();  // (the thread that raises the schedule's flag)
    uint32_t ids_smem = kNoIds;
    if (ids_local) {
        ids_smem = (uint32_t)__cvta_generic_to_shared(ids_here);
        if (cluster) {
            asm volatile("mapa.shared::cluster.u32 %0, %0, 0;" : "+r"(ids_smem));
            asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        }
    }
    const int t0 = blockIdx.x * tokens_per_block;
    route_tokens<kRegs>(logits, t0, min(T, t0 + tokens_per_block), E, k, local_offset, n_local, rp, topk_ids, topk_w, u.cand, nullptr, ids_smem);
    if (cluster) {
        __syncwarp();
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        if (blockIdx.x != 0) return;
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    } else if (!ids_local) {
        __threadfence();  // this block's ids and weights are visible before it is counted as done
        __syncthreads();
        if (tid == 0) is_last = atomicAdd(status + kDoneCounterInt, 1) == (int)gridDim.x - 1;
        __syncthreads();
        if (!is_last) return;
        __threadfence();
    } else {
        __syncthreads();
    }
    const int A = T * k;
    if (!ids_local) {  // this block's copy of all ids, in one round trip
        const int n = min(A, kFusedIds);
#pragma unroll 4
        for (int a = tid; a < n; a += kFusedThreads) ids_here[a] = (unsigned char)__ldcg(&topk_ids[a]);
        __syncthreads();
    }
    // this warp's span of the assignments: whole groups of 32 (the first `spans` warps have one), those up to a_here from shared
    // memory.  Further ids come from L2, kFusedAhead groups' loads side by side.  (One group's at a time, router and sort of 1024
    // tokens of 32 experts, top 32: 63.5 us, now 55.3; of 128, top 16 36.8 / 30.8; 700 of 128, top 16 28.6 / 24.7.)
    const int a0 = min(A, warp * span), a1 = min(A, a0 + span), a_here = min(a1, kFusedIds);
    auto fetch_ids = [&](int base, int (&ids)[kFusedAhead]) {
#pragma unroll
        for (int i = 0; i < kFusedAhead; ++i) {
            const int a = base + i * 32 + lane;
            ids[i] = a < a1 ? __ldcg(&topk_ids[a]) - local_offset : -1;
        }
    };
    int *next = u.next[warp];
    if (warp < spans) {
#pragma unroll 1
        for (int e = lane; e < n_local; e += 32) next[e] = 0;
        __syncwarp();
#pragma unroll 1
        for (int a = a0 + lane; a < a_here; a += 32) {
            const int e = (int)ids_here[a] - local_offset;
            if (e >= 0 && e < n_local) atomicAdd(&next[e], 1);
        }
#pragma unroll 1
        for (int base = max(a0, kFusedIds); base < a1; base += 32 * kFusedAhead) {
            int ids[kFusedAhead];
            fetch_ids(base, ids);
#pragma unroll
            for (int i = 0; i < kFusedAhead; ++i)
                if (ids[i] >= 0 && ids[i] < n_local) atomicAdd(&next[ids[i]], 1);
        }
    }
    __syncthreads();
    int count = 0;  // rows of expert tid
    if (tid < n_local) {
#pragma unroll 4
        for (int w = 0; w < spans; ++w) count += u.next[w][tid];
    }
    schedule_phase(count, n_local, nt_max, row_quantum, expert_offsets, tile_prefix, tile_order, tile_rows, status, sh, [&](int row) {
        // counts -> first positions of expert tid in the spans
#pragma unroll 4
        for (int w = 0; w < spans; ++w) {
            const int c = u.next[w][tid];
            u.next[w][tid] = row;
            row += c;
        }
    });
    if (warp >= spans) return;
#pragma unroll 1
    for (int base = a0; base < a_here; base += 32) {
        const int a = base + lane;
        scatter_group(a < a_here ? (int)ids_here[a] - local_offset : -1, a, a < a_here, n_local, next, sorted_to_flat, flat_to_sorted, lane);
    }
#pragma unroll 1
    for (int base = max(a0, kFusedIds); base < a1; base += 32 * kFusedAhead) {
        int ids[kFusedAhead];
        fetch_ids(base, ids);
#pragma unroll
        for (int i = 0; i < kFusedAhead; ++i) {
            const int a = base + i * 32 + lane;
            if (base + i * 32 >= a1) break;  // uniform over the warp
            scatter_group(ids[i], a, a < a1, n_local, next, sorted_to_flat, flat_to_sorted, lane);
        }
    }
}

// Token rows into expert-contiguous order, token-major: a warp reads (a share of) token t's row once and stores
// it to the up to top_k rows flat_to_sorted[t*k + j] >= 0.  Reading each row once instead of once per assignment
// halves the traffic of a top-8 layer; the copies are streamed past L2 (the GEMM reads them from memory anyway).
__global__ void __launch_bounds__(256)
scatter_rows_kernel(const uint4 *__restrict__ x, const int *__restrict__ flat_to_sorted, int T, int k, int vec_per_row,
                    int warps_per_token, uint4 *__restrict__ x_perm) {
    chain_release();
    chain_wait();
    const int lane = threadIdx.x & 31;
    const long long w = (long long)blockIdx.x * 8 + (threadIdx.x >> 5);
    const int t = (int)(w / warps_per_token), part = (int)(w % warps_per_token);
    if (t >= T) return;
    const int my_row = lane < k ? flat_to_sorted[(size_t)t * k + lane] : -1;  // lane j holds rank j's destination
    if (!__any_sync(kFullMask, my_row >= 0)) return;  // none of the token's experts is resident here: nothing to copy
    const uint4 *src = x + (size_t)t * vec_per_row;
    constexpr int kInFlight = 4;  // independent 16-byte loads per lane before the first is used
    const int stride = 32 * warps_per_token;
    for (int i0 = part * 32 + lane; i0 < vec_per_row + lane; i0 += kInFlight * stride) {  // (i0 - lane) uniform
        uint4 v[kInFlight];
#pragma unroll
        for (int u = 0; u < kInFlight; ++u)
            if (i0 + u * stride < vec_per_row) v[u] = src[i0 + u * stride];
        for (int j = 0; j < k; ++j) {
            const int row = __shfl_sync(kFullMask, my_row, j);
            if (row < 0) continue;  // assignment to an expert that is not resident here
            uint4 *dst = x_perm + (size_t)row * vec_per_row;
#pragma unroll
            for (int u = 0; u < kInFlight; ++u)
                if (i0 + u * stride < vec_per_row) __stcs(dst + i0 + u * stride, v[u]);
        }
    }
}

// One thread per 16-byte column of one token: the up to eight rows of a batch are fetched together (eight independent
// 16-byte loads in flight per thread), then added one rank after the other, so the summation order is fixed.
constexpr int kCombineThreads = 128, kCombineBatch = 8;
__global__ void __launch_bounds__(kCombineThreads)
combine_kernel(const uint4 *__restrict__ y, const float *__restrict__ topk_w, const int *__restrict__ flat_to_sorted,
               int k, int vec_per_row, int blocks_per_token, uint4 *__restrict__ out) {
    __shared__ int rows[kMaxTopK];
    __shared__ float weights[kMaxTopK];
    chain_release();
    chain_wait();
    const int t = blockIdx.x / blocks_per_token;
    const int i = (blockIdx.x - t * blocks_per_token) * kCombineThreads + threadIdx.x;
    if (threadIdx.x < k) {
        rows[threadIdx.x] = flat_to_sorted[(size_t)t * k + threadIdx.x];
        weights[threadIdx.x] = topk_w[(size_t)t * k + threadIdx.x];
    }
    __syncthreads();
    if (i >= vec_per_row) return;
    float acc[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) acc[c] = 0.f;
    for (int j0 = 0; j0 < k; j0 += kCombineBatch) {
        uint4 v[kCombineBatch];
#pragma unroll
        for (int u = 0; u < kCombineBatch; ++u) {
            const bool live = j0 + u < k && rows[j0 + u] >= 0;  // rank exists and its expert is resident here
            v[u] = live ? __ldcs(&y[(size_t)rows[j0 + u] * vec_per_row + i]) : make_uint4(0, 0, 0, 0);
        }
#pragma unroll
        for (int u = 0; u < kCombineBatch; ++u) {  // ascending rank
            if (j0 + u >= k || rows[j0 + u] < 0) continue;  // contributes nothing (not even a signed zero)
            const float wj = weights[j0 + u];
            const __nv_bfloat162 *h2 = reinterpret_cast<const __nv_bfloat162 *>(&v[u]);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float2 f = __bfloat1622float2(h2[c]);
                acc[2 * c] = fmaf(wj, f.x, acc[2 * c]);
                acc[2 * c + 1] = fmaf(wj, f.y, acc[2 * c + 1]);
            }
        }
    }
    uint4 o;
    __nv_bfloat162 *o2 = reinterpret_cast<__nv_bfloat162 *>(&o);
#pragma unroll
    for (int c = 0; c < 4; ++c) o2[c] = __floats2bfloat162_rn(acc[2 * c], acc[2 * c + 1]);
    out[(size_t)t * vec_per_row + i] = o;
}

// The same sum for a layer with a resident subset of the experts, where most ranks of most tokens have no row here
// (the paper's 32 of 256: one live rank per token on average).  There the kernel above has one 16-byte load in flight
// per thread and is bound by the latency of that load (3.1 TB/s alone on the machine, 0.09 ms for 8192 tokens).
// Here a block takes kTokens consecutive tokens, lists their live (token, rank) pairs in order, and every
// thread fetches up to kSparseBatch rows at once before it sums them, token after token, rank after rank: the
// same order of summation, the same result, kSparseBatch loads in flight.  All threads build the list, one pair each,
// in one round trip (one warp took four, and its block waited): 60 -> 40 us for 8192 tokens of 7168 features, 0.23 GB, 5.9
// TB/s.  Where sixteen tokens per block make less than two blocks per SM a block takes four: with sixteen, 128 tokens make
// 56 blocks and a chain of two batches each (11 -> 5 us).  Layers of 4096 features with small experts, four / sixteen: 8 of
// 64 experts resident, top 4, 600 tokens 39.0 / 41.0 us, 1500 tokens 57.5 / 55.6; 7168 features, 1500 tokens 83.1 / 78.3.
constexpr int kSparseBatch = 16;
template <int kTokens>
__global__ void __launch_bounds__(kCombineThreads)
combine_sparse_kernel(const uint4 *__restrict__ y, const float *__restrict__ topk_w, const int *__restrict__ flat_to_sorted,
                      int T, int k, int vec_per_row, int blocks_per_group, uint4 *__restrict__ out) {
    __shared__ int live_row[kTokens * kMaxTopK], live_tok[kTokens * kMaxTopK];
    __shared__ float live_w[kTokens * kMaxTopK];
    __shared__ int warp_live[kCombineThreads / 32];
    chain_release();
    chain_wait();
    const int group = blockIdx.x / blocks_per_group;
    const int t0 = group * kTokens, i = (blockIdx.x - group * blocks_per_group) * kCombineThreads + threadIdx.x;
    const int n_tok = min(kTokens, T - t0);
    int n_live = 0;
    for (int e0 = 0; e0 < n_tok * k; e0 += kCombineThreads) {  // the live pairs, in (token, rank) order
        const int e = e0 + threadIdx.x, warp = threadIdx.x >> 5;
        const int row = e < n_tok * k ? flat_to_sorted[(size_t)t0 * k + e] : -1;
        const float w = e < n_tok * k ? topk_w[(size_t)t0 * k + e] : 0.f;
        const unsigned mask = __ballot_sync(kFullMask, row >= 0);
        if ((threadIdx.x & 31) == 0) warp_live[warp] = __popc(mask);
        __syncthreads();
        int at = n_live + __popc(mask & ((1u << (threadIdx.x & 31)) - 1u));
#pragma unroll
        for (int q = 0; q < kCombineThreads / 32; ++q) {
            if (q < warp) at += warp_live[q];
            n_live += warp_live[q];
        }
        if (row >= 0) {
            live_row[at] = row;
            live_tok[at] = e / k;
            live_w[at] = w;
        }
        __syncthreads();  // (warp_live is written again)
    }
    if (i >= vec_per_row) return;
    const int L = n_live;
    float acc[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) acc[c] = 0.f;
    int cur = 0;  // the token whose sum is in acc
    auto flush = [&]() {
        uint4 o;
        __nv_bfloat162 *o2 = reinterpret_cast<__nv_bfloat162 *>(&o);
#pragma unroll
        for (int c = 0; c < 4; ++c) o2[c] = __floats2bfloat162_rn(acc[2 * c], acc[2 * c + 1]);
        out[(size_t)(t0 + cur) * vec_per_row + i] = o;
#pragma unroll
        for (int c = 0; c < 8; ++c) acc[c] = 0.f;
        ++cur;
    };
    for (int base = 0; base < L; base += kSparseBatch) {
        uint4 v[kSparseBatch];
#pragma unroll
        for (int u = 0; u < kSparseBatch; ++u)
            v[u] = base + u < L ? __ldcs(&y[(size_t)live_row[base + u] * vec_per_row + i]) : make_uint4(0, 0, 0, 0);
#pragma unroll
        for (int u = 0; u < kSparseBatch; ++u) {
            if (base + u >= L) break;  // (uniform over the block)
            const int tok = live_tok[base + u];
            while (cur < tok) flush();
            const float wj = live_w[base + u];
            const __nv_bfloat162 *h2 = reinterpret_cast<const __nv_bfloat162 *>(&v[u]);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float2 f = __bfloat1622float2(h2[c]);
                acc[2 * c] = fmaf(wj, f.x, acc[2 * c]);
                acc[2 * c + 1] = fmaf(wj, f.y, acc[2 * c + 1]);
            }
        }
    }
    while (cur < n_tok) flush();
}

}  // namespace

int choose_nt_max(int T, int E, int k, bool wide_ok) {
    const double avg = (double)T * k / E;
    const int options[3] = {32, 64, 128};
    for (int nt : options)
        if (1.5 * avg <= nt) return nt;
    // Between about 160 and 350 rows per expert on average, experts with 257..384 rows are common: a wide bound
    // keeps each of them in one tile (320 while the mean plus 2.5 standard deviations of a uniform routing fits, else
    // 384).  With more rows than that nearly every expert needs several tiles anyway, and those are 256-row tiles.
    if (!wide_ok || avg <= 160.0 || avg > 352.0) return 256;
    return avg + 2.5 * sqrt(avg) <= 320.0 ? 320 : 384;
}

cudaError_t launch_route(const float *logits, int T, int E, int k, LocalExperts local, int nt_max, int *topk_ids,
                         float *topk_w, int *expert_offsets, int *sorted_to_flat, int *flat_to_sorted,
                         RouteScratch scratch, int *status, cudaStream_t stream, int row_quantum, RouterParams router,
                         size_t status_bytes) {
    if (!RowQuantum::valid(row_quantum)) return cudaErrorInvalidValue;
    const int A = T * k;
    if (scratch.n_chunks <= kFusedMaxChunks) {
        // One block, a cluster of eight, or up to 64 blocks of at least four tokens (the comment at kFusedOneBlockTokens).
        const bool ids_local = T <= kFusedOneBlockTokens || (T <= kFusedClusterTokens && A <= kFusedClusterIds);
        int blocks = 1, per_block = T;
        if (T > kFusedOneBlockTokens) {
            per_block = ids_local ? (T + kFusedCluster - 1) / kFusedCluster : (T + 63) / 64 < 4 ? 4 : (T + 63) / 64;
            blocks = ids_local ? kFusedCluster : (T + per_block - 1) / per_block;
        }
        if (!ids_local) {
            const cudaError_t err = cudaMemsetAsync(status, 0, status_bytes, stream);
            if (err != cudaSuccess) return err;
        }
        // (The cluster starts when everything before it is done.  Launched early, its blocks of 48 KB and 1024 threads held SMs
        // while the last kernels of the call before were still at work: 64 tokens on 32 MX experts of 7168 x 2048 202.8 -> 214 us.)
        const bool cluster = ids_local && blocks > 1;
        const int spans = fused_spans(A), span = ((A + 32 * spans - 1) / (32 * spans)) * 32;
        auto kernel = E <= 32 ? route_fused_kernel<1> : E <= 128 ? route_fused_kernel<4> : route_fused_kernel<8>;
        return launch_clusters(kernel, !cluster, cluster ? blocks : 1, blocks, kFusedThreads, 0, stream, logits, T, E, k,
                               local.offset, local.count, nt_max, RowQuantum(row_quantum), per_block, spans, span, router, topk_ids, topk_w,
                               expert_offsets, scratch.tile_prefix, scratch.tile_order, scratch.tile_rows, sorted_to_flat,
                               flat_to_sorted, status, ids_local ? (int)(status_bytes / sizeof(int)) : 0);
    }
    cudaError_t err = cudaMemsetAsync(status, 0, status_bytes, stream);  // the status word and what shares its region
    if (err != cudaSuccess) return err;
    const bool many = scratch.n_chunks > kRouteSms;
    auto topk_kernel = many ? (E <= 32 ? route_topk_kernel<kRouteThreadsManyChunks, 1>
                               : E <= 128 ? route_topk_kernel<kRouteThreadsManyChunks, 4> : route_topk_kernel<kRouteThreadsManyChunks, 8>)
                            : (E <= 32 ? route_topk_kernel<kRouteThreads, 1>
                               : E <= 128 ? route_topk_kernel<kRouteThreads, 4> : route_topk_kernel<kRouteThreads, 8>);
    err = launch_chained(topk_kernel, scratch.n_chunks,
                         many ? kRouteThreadsManyChunks : kRouteThreads, 0, stream, logits, T, E, k, local.offset, local.count,
                         router, topk_ids, topk_w, scratch.chunk_counts);
    if (err != cudaSuccess) return err;
    // (the blocks' totals per expert sit where the last block then writes the tile rows)
    const int groups = (local.count + 31) / 32, warps_per_group = scan_warps_per_group(scratch.n_chunks, groups);
    const int scan_blocks = (scratch.n_chunks + warps_per_group - 1) / warps_per_group <= kScanBatch ? 1 : groups;
    err = launch_chained(route_scan_kernel, scan_blocks, kScanThreads, 0, stream, scratch.chunk_counts, scratch.n_chunks,
                         local.count, nt_max, RowQuantum(row_quantum), expert_offsets, scratch.tile_prefix, scratch.tile_order,
                         scratch.tile_rows, scratch.tile_rows, status);
    if (err != cudaSuccess) return err;
    return launch_chained(route_scatter_kernel, scratch.n_chunks, 32, 0, stream, topk_ids, scratch.chunk_counts,
                          expert_offsets, A, local.count, local.offset, k, sorted_to_flat, flat_to_sorted);
}

// Warps per token: enough warps to fill the device when there are few tokens, at most one per 32 vectors.
static int scatter_warps_per_token(long long tokens, int vec_per_row) {
    const long long target = 32768;
    long long per = tokens > 0 ? (target + tokens - 1) / tokens : 1;
    const int most = (vec_per_row + 31) / 32;
    if (per > most) per = most;
    return per < 1 ? 1 : (int)per;
}

cudaError_t launch_scatter_rows(const __nv_bfloat16 *x, const int *flat_to_sorted, int T, int k, int H, __nv_bfloat16 *x_perm,
                                cudaStream_t stream) {
    const int wpt = scatter_warps_per_token(T, H / 8);
    const long long warps = (long long)T * wpt;
    return launch_chained(scatter_rows_kernel, (unsigned)((warps + 7) / 8), 256, 0, stream,
                          reinterpret_cast<const uint4 *>(x), flat_to_sorted, T, k, H / 8, wpt, reinterpret_cast<uint4 *>(x_perm));
}

cudaError_t launch_combine(const __nv_bfloat16 *y, const float *topk_w, const int *flat_to_sorted, int T, int k,
                           int H, __nv_bfloat16 *out, cudaStream_t stream, bool resident_subset) {
    const int vec_per_row = H / 8, blocks_per_token = (vec_per_row + kCombineThreads - 1) / kCombineThreads;
    if (resident_subset) {
        const int tokens = ((long long)T + 15) / 16 * blocks_per_token >= 2 * kRouteSms ? 16 : 4;
        const long long groups = ((long long)T + tokens - 1) / tokens;
        return launch_chained(tokens == 16 ? combine_sparse_kernel<16> : combine_sparse_kernel<4>,
                              (unsigned)(groups * blocks_per_token), kCombineThreads, 0, stream,
                              reinterpret_cast<const uint4 *>(y), topk_w, flat_to_sorted, T, k, vec_per_row, blocks_per_token,
                              reinterpret_cast<uint4 *>(out));
    }
    return launch_chained(combine_kernel, (unsigned)((long long)T * blocks_per_token), kCombineThreads, 0, stream,
                          reinterpret_cast<const uint4 *>(y), topk_w, flat_to_sorted, k, vec_per_row, blocks_per_token,
                          reinterpret_cast<uint4 *>(out));
}

}  // namespace moe

// ---- moe_route_static: the router + sort-scatter for callers that cannot allocate --------------------
//
// The scratch (status word, per-chunk histograms, tile schedule) lives in a file-scope device array,
// so the caller passes only inputs and outputs.  In host code the array's name is only a handle for
// the runtime, not a device address: its address is looked up once per device with
// cudaGetSymbolAddress (with that device current) and that pointer is what the kernels receive.
namespace moe {
namespace {

constexpr size_t kStaticScratchBytes = 512 * 1024;
static __device__ __align__(256) unsigned char g_route_static_scratch[kStaticScratchBytes];

constexpr int kMaxDevices = 64;
std::mutex g_static_mutex;
void *g_static_scratch_ptr[kMaxDevices] = {nullptr};

// Device address of the static scratch on the current device (looked up on the first call per device).
cudaError_t static_scratch_address(void **out) {
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_static_mutex);
    if (!g_static_scratch_ptr[dev]) {
        void *ptr = nullptr;
        err = cudaGetSymbolAddress(&ptr, g_route_static_scratch);
        if (err != cudaSuccess) return err;
        g_static_scratch_ptr[dev] = ptr;
    }
    *out = g_static_scratch_ptr[dev];
    return cudaSuccess;
}

}  // namespace
}  // namespace moe

extern "C" int moe_route_static(const float *router_logits, int T, int E, int top_k, int32_t *topk_ids,
                                float *topk_weights, int32_t *expert_offsets, int32_t *sorted_to_flat,
                                int32_t *flat_to_sorted, void *stream) {
    using namespace moe;
    const int args = check_route_args(router_logits, T, E, top_k, topk_ids, topk_weights, expert_offsets, sorted_to_flat,
                                      flat_to_sorted);
    if (args == MOE_ERR_SHAPE || args == MOE_ERR_UNSUPPORTED) return args;
    if (256 + route_scratch_bytes(T, E) > kStaticScratchBytes) return MOE_ERR_STATIC_LIMIT;
    if (args != MOE_OK) return args;
    const int arch = check_device();
    if (arch != MOE_OK) return arch;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (T == 0)
        return cudaMemsetAsync(expert_offsets, 0, (size_t)(E + 1) * sizeof(int), s) == cudaSuccess ? MOE_OK : MOE_ERR_CUDA;
    void *scratch = nullptr;
    if (static_scratch_address(&scratch) != cudaSuccess || !scratch) return MOE_ERR_CUDA;
    char *base = static_cast<char *>(scratch);
    // The array keeps the previous call's contents.  The status word is cleared by launch_route; the
    // histogram and schedule regions are fully overwritten for this T and E before they are read.
    RouteScratch rs = carve_route_scratch(base + 256, T, E);
    const cudaError_t err = launch_route(router_logits, T, E, top_k, LocalExperts{0, E}, 256, topk_ids, topk_weights,
                                         expert_offsets, sorted_to_flat, flat_to_sorted, rs,
                                         reinterpret_cast<int *>(base), s);
    return err == cudaSuccess ? MOE_OK : MOE_ERR_CUDA;
}

