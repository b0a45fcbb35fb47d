// One decode step of grouped-query attention over a paged key-value cache (paper, Sec. 4.6 "Kernel Analysis: GQA
// Paged Decode"): every batch item has one query token, which attends over the keys and values stored in its pages.
//
// The work is HBM-bound (every cached key and value is read once; 8 flops per byte at a group of 8 query heads), so
// the design is about the stream, not the tensor pipe:
//   * a block works on one (sequence part, key-value head, batch item) at a time; its 4 warps keep the 16 x 128 query tile of the
//     group (Hq / Hkv heads, padded to the MMA's 16 rows) in registers, so a key or value byte is fetched from
//     memory once for all heads of the group (Sec. 4.6 / Table 2: "fusing multiple query heads per KV head");
//   * tokens arrive in chunks of 64 through a pipeline of TMA copies that follow the page table and complete on the
//     stage's mbarrier ("vectorized/async paged-KV gather with pipelined global to shared memory prefetch").  Page
//     sizes that are powers of two of at least 8 take the TILED gather: the cache is a 5-D tensor (64 dims, slot,
//     half of the dims, head, page) and one `cp.async.bulk.tensor` box brings a page's slots (up to 64) of one head
//     as two 128-byte-swizzled blocks, so a chunk of 16-token pages is eight boxes.  A fifth warp issues them and
//     does nothing else, three stages deep, two blocks per SM; full / empty mbarriers hand the stages back and
//     forth, and the compute warps' loop has no block-wide barrier.  Other page sizes take the ROW gather, one
//     256-byte `cp.async.bulk` per token row and compute thread into rows padded to 272 bytes, two stages in three
//     blocks per SM.  What was measured on the way, B = 64 x 16k tokens: sixteen 16-byte cp.async per thread and
//     chunk, 4.0 TB/s (800 instructions per warp and chunk, instruction-latency bound at 8 warps per SM); the row
//     gather 4.0 TB/s with and 5.2 TB/s without the arithmetic, one 256-byte request per 14 cycles and SM being all
//     the copy engine took; the tiled gather with one compute warp issuing 6.1 TB/s, with the boxes dealt out to
//     the four compute warps 6.3 TB/s (a thread is held 5 to 9 cycles per 128-byte row of a box it issues), with
//     the copy warp 6.6-6.9 TB/s, the measured copy bandwidth;
//   * each warp owns 16 tokens of a chunk: S = Q K^T (mma.sync m16n8k16, bf16 in, fp32 out: the tile is 16 rows, far
//     too small for a tcgen05 tile, and the kernel is bound by the copy stream), an online softmax in the base-2
//     domain, O += P V with the probabilities re-used from the accumulator registers;
//   * the four warps' (max, sum, O) are merged in shared memory; a part of a sequence writes its unnormalised result to
//     the workspace, bumps the (item, head) counter, and the block that finds itself last merges the parts and writes
//     out / lse (Sec. 4.6 "Parallelism over the sequence").  A sequence in one part skips the round trip.  The merge
//     fetches the parts' outputs together with their (max, sum) pairs: one sequence of 65 536 tokens in 49 parts 42 -> 37 us.
// The merge is a fixed-order sum over parts, so results do not depend on which block arrives last.
// Every wait on a stage's barrier is bounded: a block that gives up records MOE_ERR_DEVICE_TIMEOUT in the
// workspace's status word (read it with moe_last_status) and leaves without writing a result for the segment it was in.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include "gqa_decode.h"
#include "moe_internal.cuh"

namespace moe {
namespace tc {
// (moe_tc_host.cu) 5-D bf16 tensor map of a paged cache [num_pages, page_size, Hkv, 128], dimensions ordered (64
// dims, slot, half of the dims, head, page): box = 64 dims x box_rows slots x both halves of one head of one page,
// 128-byte swizzle; encoded through the driver entry point and cached.
bool encode_kv_cache_map(CUtensorMap *map, const void *cache, uint64_t num_pages, uint32_t page_size, uint32_t Hkv,
                         uint32_t box_rows);
// (moe_tc_host.cu) cudaFuncAttributeMaxDynamicSharedMemorySize, set once per kernel and device, under a mutex.
bool set_max_dynamic_smem_once(const void *kernel, int bytes);
}  // namespace tc
}  // namespace moe

namespace gqa {
namespace {

constexpr int kD = 128;            // head dimension
constexpr int kRows = 16;          // query heads per block: the MMA's M; groups of up to 16 heads
constexpr int kChunk = 64;         // tokens per pipeline stage
constexpr int kWarps = 4;          // each owns 16 tokens of a chunk
constexpr int kThreads = kWarps * 32;
constexpr int kStages = 2;         // one chunk in flight while the previous one is used ...
constexpr int kBlocksPerSm = 3;    // ... in each of three blocks per SM (168 registers per thread, 69 KiB each)
constexpr int kRowBytes = kD * 2;  // 256 bytes per token and head in the cache
// Two layouts of a 64-token tile in shared memory, one per kernel:
//   tiled: one block per TMA box, [64 / box_rows boxes][2 halves of the dims][box_rows rows][128 bytes], each half
//          block in TMA's 128-byte swizzle: 16 KiB;
//   rows:  [64 rows][272 bytes], the 16 bytes of padding keeping ldmatrix free of bank conflicts: 17 KiB.
constexpr int kRowPitch = kRowBytes + 16;
constexpr int kTileBytes = kChunk * kRowPitch;
constexpr int kStageBytes = 2 * kTileBytes;           // keys, then values: 34 KiB
constexpr int kModelBlocksPerSm = 2;  // blocks per SM the split model counts with (the tiled kernel's)
constexpr int kSmemBytes = kStages * kStageBytes + 1024;  // (the base is rounded up to 1024 bytes)
// The tiled gather: three stages in each of two blocks per SM, and the segment merge's buffer behind them.
constexpr int kTiledStages = 3, kTiledTileBytes = kChunk * kRowBytes, kTiledStageBytes = 2 * kTiledTileBytes;
static_assert(kTiledTileBytes % 1024 == 0, "tiles must keep the swizzle's alignment");
constexpr int kWaitLimit = 1 << 22;                   // polls of a stage's barrier before the block gives up
constexpr int kMaxSplits = 128;
constexpr float kLog2e = 1.4426950408889634f;

struct Params {
    const __nv_bfloat16 *q, *k_cache, *v_cache;
    const int *kv_indptr, *kv_indices, *kv_last_page_len;
    __nv_bfloat16 *out;
    float *lse;
    int *status;       // the workspace's status word, zeroed before the launch (or by its first block: own_status)
    int *counters;     // [B * Hkv], zeroed before the launch (not with own_status: nothing is counted)
    float *part_ml;    // [slots, group, 2]  (max in the base-2 domain, sum); at least B * Hkv * n_splits slots
    float *part_o;     // [slots, group, D]  unnormalised
    int B, Hq, Hkv, group, page_size, split_tokens, n_splits;
    int box_rows;      // tiled gather: token rows one TMA box brings (min(page_size, 64))
    int own_status;    // no memset in front: the first block zeroes the status word
    float scale_log2;  // sm_scale * log2(e)
};

// ---- the launches of a call --------------------------------------------------------------------------------------
// Where parts of sequences may have to be counted, a memset in front of the kernel zeroes the status word and the counters.
// Where no sequence is split there is nothing to count, and the kernel's first block zeroes the status word: one launch
// (Params::own_status), and where that is faster with programmatic serialisation (kChained), so that a kernel's start overlaps the end of the
// one in front (behind a memset it cannot).
// Loops without / with: 40 sequences of 31..251 tokens 8.2 / 7.5 us, 162 of 410..821 44.3 / 42.8, 256 of 256..2048 105.9 / 103.5.
// Memset / one launch, in a loop / on the first pass over new inputs: 1 sequence of 100 tokens 8.5 -> 7.6 us / 25.7 ->
// 21.7, 256 of 256..2048 105.5 -> 102.8 / 138 -> 133.  A wait gives up after 4 million polls, long after that block has started.
// (A small kernel that zeroed the words beside a decode kernel launched with programmatic serialisation made loops 0.7 to 2
// us shorter, but first passes 2.3 longer, memset / small kernel: 1 sequence of 65 536 tokens 36.9 / 36.2 and 58.3 / 61.3, 1 of
// 4000 14.3 / 13.2 and 32.4 / 34.8, 16 of 8000 51.1 / 50.2 and 73.7 / 75.6.)
// Chained or not: the blocks of a chained call are placed while those of the call in front still sit on their SMs.  Few find SMs of their
// own, and a grid that fills the machine is placed evenly all the same; in between several land on one SM, and long ones wait for
// it.  Equal lengths over 4 heads, plain / chained, loops: tiled, 108 blocks of 300 tokens 8.2 / 7.6 us, 800 14.4 / 14.8, 915 16.4 / 17.0;
// 32 of 600 12.3 / 10.5; 68 of 700 12.6 / 12.7; 152 of 700 15.8 / 14.4, of 1100 22.2 / 21.0; row gather, 120 blocks of 128 8.2 /
// 7.2, of 256 12.3 / 12.5; 108 of 512 19.0 / 20.9; 32 of 384 15.6 / 13.9; 68 of 384 15.9 / 16.5; 240 of 256 12.6 / 12.7; 480 of 128
// 14.4 / 12.9, of 384 34.5 / 33.1.  (The row gather's loop is at the limit of its registers: the wait in front of it cost 216 blocks
// of 1059..2118 tokens 3 %, 75.2 / 77.5.)
constexpr unsigned kSms = 148;
static bool chaining_is_faster(bool tiled, unsigned blocks, int max_kv_len) {
    if (max_kv_len <= (tiled ? 384 : 128)) return true;
    return 4 * blocks <= kSms || (tiled ? blocks >= kSms : blocks >= 3 * kSms && max_kv_len <= 384);
}

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done) : "r"(bar), "r"(parity) : "memory");
    return done != 0;
}
// One bulk copy of `bytes` (a multiple of 16, both addresses 16-byte aligned) that completes on an mbarrier.
__device__ __forceinline__ void bulk_copy(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}

// One box of the cache's 5-D tensor map -- coordinates (dim 0, slot, half 0, head, page): the innermost is always 0 --
// that completes on an mbarrier.
__device__ __forceinline__ void tma_load_box(uint32_t dst, const CUtensorMap *map, int slot, int head, int page, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, %6}], [%7];"
        ::"r"(dst), "l"(map), "r"(0), "r"(slot), "r"(0), "r"(head), "r"(page), "r"(bar) : "memory");
}

__device__ __forceinline__ void ldmatrix_x4(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
// D (16x8, f32) += A (16x16, bf16, row) * B (16x8, bf16, col)
__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t *>(&v);
}

// Bounded wait on an mbarrier: false once `limit` polls have passed (the status word then says so: the call's first
// expired wait records MOE_ERR_DEVICE_TIMEOUT, site 12 and the block) or once another thread of the block has given up.
__device__ __forceinline__ bool bounded_wait(uint32_t bar, uint32_t parity, int limit, volatile int *gave_up, int *status) {
    for (int i = 0; i < limit; ++i) {
        if (mbar_try_wait(bar, parity)) return true;
        if (*gave_up) return false;
    }
    *gave_up = 1;
    if (atomicCAS(status, 0, (int)MOE_ERR_DEVICE_TIMEOUT) == 0) { status[1] = 12; status[2] = blockIdx.x; }
    return false;
}

// Byte offset, inside a 64-token tile, of 16-byte piece `piece` (0..15) of token row `row`.
// `sh` = log2(box_rows) (tiled only).
template <bool kTiled>
__device__ __forceinline__ uint32_t tile_offset(int row, int piece, int sh) {
    if (kTiled)
        return ((row >> sh) << (sh + 8)) + ((piece >> 3) << (sh + 7)) + ((row & ((1 << sh) - 1)) << 7) +
               (((piece & 7) ^ (row & 7)) << 4);
    return row * kRowPitch + (piece << 4);
}

// One warp's share of a chunk: 16 tokens, rows row_base .. +15 of the key and value tiles, the first of them token
// tok_base (< end) of the sequence.  Updates the running maxima, sums and the unnormalised output.
template <bool kTiled>
__device__ __forceinline__ void attend_16_tokens(const uint32_t (&qa)[kD / 16][4], float (&o_acc)[kD / 8][4], float (&m_run)[2],
                                                 float (&l_run)[2], uint32_t k_tile, uint32_t v_tile, int row_base, int tok_base,
                                                 int end, int sh, float scale_log2, int lane) {
    if (kTiled && tok_base + 16 > end) {
        // A box brings whole pages: value rows past the end of the sequence hold whatever the cache holds there
        // (and rows of pages that were not fetched, whatever the stage held).  Zero them, so that a masked
        // probability of 0 meets a finite value.  The rows are this warp's own.
        const int valid = end - tok_base;  // 1..15
        for (int i = lane; i < 16 * 16; i += 32) {
            const int r = i >> 4;
            if (r >= valid)
                asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};"
                             ::"r"(v_tile + tile_offset<true>(row_base + r, i & 15, sh)), "r"(0) : "memory");
        }
        // A block that goes on to another sequence hands this stage back, and the next copy into it is an async-proxy
        // write: without a proxy fence by the lanes that stored, the barrier alone does not order the two.
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
    }
    // S = Q K^T for 16 tokens: two n-tiles of 8 tokens, 8 K-steps.  A warp is one of one to three on its
    // scheduler, so the latency of its own chain is what counts: fragments are fetched two steps ahead of the
    // MMAs that use them, and even and odd K-steps accumulate separately (chains of four instead of eight).
    float s[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
    float s_odd[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
    const int m4 = lane >> 3, rr = lane & 7;
    const int k_row = row_base + ((m4 >> 1) << 3) + rr, v_row = row_base + ((m4 & 1) << 3) + rr;
    // Piece 2 i + b of a row from piece b: an XOR of the swizzle's bits (the row's part of the address has none below 128)
    // and, for the upper half of the dims, a step -- two instructions per fragment and no register per offset.
    const uint32_t k_first = k_tile + tile_offset<kTiled>(k_row, m4 & 1, sh), v_first = v_tile + tile_offset<kTiled>(v_row, m4 >> 1, sh);
    const uint32_t upper = kTiled ? 1u << (sh + 7) : 0u;
    auto piece_addr = [&](uint32_t first, int i) {
        return kTiled ? (first ^ (uint32_t)(((2 * i) & 7) << 4)) + (i >= 4 ? upper : 0u) : first + (uint32_t)(i * 32);
    };
    constexpr int kAhead = 2;
    uint32_t kb[kAhead + 1][4];
#pragma unroll
    for (int ks = 0; ks < kAhead; ++ks) ldmatrix_x4(kb[ks], piece_addr(k_first, ks));
#pragma unroll
    for (int ks = 0; ks < kD / 16; ++ks) {
        if (ks + kAhead < kD / 16)
            ldmatrix_x4(kb[(ks + kAhead) % (kAhead + 1)], piece_addr(k_first, ks + kAhead));
        const uint32_t(&f)[4] = kb[ks % (kAhead + 1)];
        if (ks & 1) {
            mma_bf16(s_odd[0], qa[ks], f[0], f[1]);
            mma_bf16(s_odd[1], qa[ks], f[2], f[3]);
        } else {
            mma_bf16(s[0], qa[ks], f[0], f[1]);
            mma_bf16(s[1], qa[ks], f[2], f[3]);
        }
    }
    // the first value fragments are on their way while the softmax runs
    uint32_t vb[kAhead + 1][4];
#pragma unroll
    for (int j = 0; j < kAhead; ++j) ldmatrix_x4_trans(vb[j], piece_addr(v_first, j));
#pragma unroll
    for (int n = 0; n < 2; ++n)
#pragma unroll
        for (int i = 0; i < 4; ++i) s[n][i] += s_odd[n][i];
    // online softmax in the base-2 domain; columns past the end of the sequence are masked
    float row_max[2] = {-INFINITY, -INFINITY};
#pragma unroll
    for (int n = 0; n < 2; ++n)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int tok = tok_base + n * 8 + (lane & 3) * 2 + (i & 1);
            s[n][i] = tok < end ? s[n][i] * scale_log2 : -INFINITY;
            row_max[i >> 1] = fmaxf(row_max[i >> 1], s[n][i]);
        }
    float alpha[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        row_max[r] = fmaxf(row_max[r], __shfl_xor_sync(0xffffffffu, row_max[r], 1));
        row_max[r] = fmaxf(row_max[r], __shfl_xor_sync(0xffffffffu, row_max[r], 2));
        const float m_new = fmaxf(m_run[r], row_max[r]);  // finite: the warp's first token is valid
        alpha[r] = exp2f(m_run[r] - m_new);               // 0 on the first chunk (m_run = -inf)
        m_run[r] = m_new;
    }
    float row_sum[2] = {0.f, 0.f};
    uint32_t pa[4];
    {
        float pv[2][4];
#pragma unroll
        for (int n = 0; n < 2; ++n)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                pv[n][i] = exp2f(s[n][i] - m_run[i >> 1]);
                row_sum[i >> 1] += pv[n][i];
            }
        // the probabilities as the A operand of P V: (row, k) and (row, k+8) are n-tiles 0 and 1
        pa[0] = pack_bf16(pv[0][0], pv[0][1]);
        pa[1] = pack_bf16(pv[0][2], pv[0][3]);
        pa[2] = pack_bf16(pv[1][0], pv[1][1]);
        pa[3] = pack_bf16(pv[1][2], pv[1][3]);
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        row_sum[r] += __shfl_xor_sync(0xffffffffu, row_sum[r], 1);
        row_sum[r] += __shfl_xor_sync(0xffffffffu, row_sum[r], 2);
        l_run[r] = l_run[r] * alpha[r] + row_sum[r];
    }
    // O = O * alpha + P V: 16 n-tiles of 8 dims, two per transposed ldmatrix.  Once the running maxima have
    // settled alpha is exactly 1 for every row, and the 64 multiplications are skipped (same result).
    if (__any_sync(0xffffffffu, alpha[0] != 1.f || alpha[1] != 1.f)) {
#pragma unroll
        for (int n = 0; n < kD / 8; ++n)
#pragma unroll
            for (int i = 0; i < 4; ++i) o_acc[n][i] *= alpha[i >> 1];
    }
#pragma unroll
    for (int j = 0; j < kD / 16; ++j) {  // n-tiles 2j and 2j + 1
        if (j + kAhead < kD / 16)
            ldmatrix_x4_trans(vb[(j + kAhead) % (kAhead + 1)], piece_addr(v_first, j + kAhead));
        const uint32_t(&f)[4] = vb[j % (kAhead + 1)];
        mma_bf16(o_acc[2 * j], pa, f[0], f[1]);
        mma_bf16(o_acc[2 * j + 1], pa, f[2], f[3]);
    }
}

// ---- shared by the two kernels ----------------------------------------------------------------------------------
__device__ __forceinline__ void sync_compute() { asm volatile("bar.sync 1, %0;" ::"n"(kThreads) : "memory"); }
// The same barrier, and whether any of the 128 threads passed true: what they do next, they do together.
__device__ __forceinline__ bool any_compute(bool flag) {
    uint32_t any;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 q, %1, 0;\n\t"
        "bar.red.or.pred p, 1, %2, q;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(any) : "r"((uint32_t)flag), "n"(kThreads) : "memory");
    return any != 0;
}

// Self-test of the error path: one of the four compute warps waits, with a small bound, on a barrier at which nothing
// arrives.  All four must come to the same answer, that the block has no result, and count themselves in the fourth word.
__global__ void __launch_bounds__(kThreads) gqa_wait_timeout_selftest_kernel(int *status) {
    __shared__ __align__(8) unsigned long long bar;
    __shared__ int gave_up;
    if (threadIdx.x == 0) {
        mbar_init(smem_u32(&bar), 1);
        gave_up = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    const bool ok = threadIdx.x >= 32 || bounded_wait(smem_u32(&bar), 0, 1 << 14, &gave_up, status);
    __syncwarp();
    if (any_compute(!ok) && (threadIdx.x & 31) == 0) atomicAdd(status + 3, 1);
}

// By the first block of a kernel that is alone.  (In the row gather within the barrier's set-up, as one store by one thread:
// first thing in the kernel, by four threads, it cost the row gather 2 %, 70 sequences of 1087..2175 131.3 -> 134.6 us.)
__device__ __forceinline__ void zero_own_status(const Params &p, bool first_block, int tid) {
    if (p.own_status && first_block && tid == 0) *reinterpret_cast<uint4 *>(p.status) = make_uint4(0, 0, 0, 0);
}

// A word of the page table.  __ldg is for memory that nothing writes while the kernel lives, and a chained kernel lives before what
// is in front of it, which may write the table, is done: its loads are ordinary ones, behind the wait.  (They cost what __ldg
// costs; as plain C++ loads, whose order to each other and to the copies the compiler chose anew, they cost a call 0.1 to 0.5 us:
// 40 sequences of 700 tokens 15.4 / 15.8, 256 of 256..2048 103.5 / 104.2.)
template <bool kChained>
__device__ __forceinline__ int load_index(const int *at) {
    if (!kChained) return __ldg(at);
    int v;
    asm volatile("ld.global.b32 %0, [%1];" : "=r"(v) : "l"(at) : "memory");
    return v;
}
// The wait of a chained kernel for what is in front.  That may have written the caches through the generic proxy: the threads
// that copy them into shared memory link the two by a fence, here, where nothing of theirs is under way yet.
__device__ __forceinline__ void wait_for_inputs(bool copies) {
    moe::chain_wait();
    if (copies) asm volatile("fence.proxy.async.global;" ::: "memory");
}

// Cached tokens of an item; its first entry in the page table, which a chained kernel would otherwise load twice.
template <bool kChained>
__device__ __forceinline__ int cached_tokens(const Params &p, int b, int &first) {
    first = load_index<kChained>(&p.kv_indptr[b]);
    const int behind = load_index<kChained>(&p.kv_indptr[b + 1]);
    const int last = load_index<kChained>(&p.kv_last_page_len[b]);  // (all three in flight: one round trip)
    return behind > first ? (behind - first - 1) * p.page_size + last : 0;
}
template <bool kChained>
__device__ __forceinline__ int cached_tokens(const Params &p, int b) {
    int first;
    return cached_tokens<kChained>(p, b, first);
}
// out = 0, lse = -inf for the heads of one key-value head (all 128 compute threads call).
__device__ __forceinline__ void write_empty(const Params &p, int b, int head0, int tid) {
    for (int i = tid; i < p.group * kD; i += kThreads)
        p.out[((size_t)b * p.Hq + head0 + i / kD) * kD + (i % kD)] = __float2bfloat16_rn(0.f);
    if (p.lse && tid < p.group) p.lse[(size_t)b * p.Hq + head0 + tid] = -INFINITY;
}
// The group's queries as MMA A fragments: 8 K-steps of 16 dims, rows = heads (zero beyond the group).
__device__ __forceinline__ void load_queries(const Params &p, int b, int head0, int lane, uint32_t (&qa)[kD / 16][4]) {
    const int r0 = lane >> 2, c0 = (lane & 3) * 2;
    const __nv_bfloat16 *q0 = p.q + ((size_t)b * p.Hq + head0 + r0) * kD;
    const __nv_bfloat16 *q1 = q0 + 8 * kD;
#pragma unroll
    for (int ks = 0; ks < kD / 16; ++ks) {
        const int c = ks * 16 + c0;
        qa[ks][0] = r0 < p.group ? *reinterpret_cast<const uint32_t *>(q0 + c) : 0u;
        qa[ks][1] = r0 + 8 < p.group ? *reinterpret_cast<const uint32_t *>(q1 + c) : 0u;
        qa[ks][2] = r0 < p.group ? *reinterpret_cast<const uint32_t *>(q0 + c + 8) : 0u;
        qa[ks][3] = r0 + 8 < p.group ? *reinterpret_cast<const uint32_t *>(q1 + c + 8) : 0u;
    }
}

// What a block computed: a part of the sequence of (item b, key-value head kvh), or all of it.  Part i of n_parts keeps
// its unnormalised result in slot first_slot (i = 0) or second_slot + (i - 1) * slot_step.
struct Segment {
    int b, kvh, n_parts, slot_step;
    long long slot, first_slot, second_slot;  // `slot` is this block's own
};
// a / b for non-negative a and positive b, in 32 bits where they fit (a 64-bit division is a hundred instructions).
__device__ __forceinline__ long long divide(long long a, long long b) {
    return ((a | b) >> 32) == 0 ? (long long)((uint32_t)a / (uint32_t)b) : a / b;
}
// Shared memory store_segment and merge_parts need: three foreign quarters of eight output rows per warp, (max, sum) per
// warp and row, and the heads' sums.
constexpr int kMergeFloats = kWarps * (kWarps - 1) * 4 * 32 * 2, kMergeBytes = (kMergeFloats + kWarps * kRows * 2 + kRows) * 4;

// End of a segment, by the 128 compute threads: the four warps' (max, sum, O) are merged -- warp w ends up with dims 32 w ..
// 32 w + 31 of every head, eight heads per pass, summed in warp order -- and written to out / lse, or, for a part of a
// sequence, to the part's slot.  The caller has passed a barrier of these threads since the buffer was last read.
__device__ __forceinline__ void store_segment(const Params &p, const Segment &seg, const float (&o_acc)[kD / 8][4],
                                              const float (&m_run)[2], const float (&l_run)[2], float *merge, int warp, int lane) {
    float2 *foreign = reinterpret_cast<float2 *>(merge);                        // [to warp][from][4 n-tiles][32 lanes]
    float2 *ml_w = reinterpret_cast<float2 *>(merge + kMergeFloats);            // [4 warps][16 rows] (max, sum)
    const int head0 = seg.kvh * p.group, r0 = lane >> 2, c0 = (lane & 3) * 2;
    float *part_o = p.part_o + seg.slot * p.group * kD;
    float2 *part_ml = reinterpret_cast<float2 *>(p.part_ml) + seg.slot * p.group;
#pragma unroll
    for (int pass = 0; pass < 2; ++pass) {  // heads 8 pass .. 8 pass + 7
        if (pass * 8 >= p.group) break;
        if (pass > 0) sync_compute();       // (the buffer's previous readers are done)
        if ((lane & 3) == 0) ml_w[warp * kRows + pass * 8 + r0] = make_float2(m_run[pass], l_run[pass]);
#pragma unroll
        for (int to = 0; to < kWarps; ++to)
            if (to != warp) {
#pragma unroll
                for (int n = 0; n < 4; ++n)
                    foreign[((to * (kWarps - 1) + (warp > to ? warp - 1 : warp)) * 4 + n) * 32 + lane] =
                        make_float2(o_acc[to * 4 + n][2 * pass], o_acc[to * 4 + n][2 * pass + 1]);
            }
        sync_compute();
        const int g = pass * 8 + r0;
        float m = -INFINITY;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) m = fmaxf(m, ml_w[w * kRows + g].x);
        float l = 0.f;
        float2 o[4];
#pragma unroll
        for (int n = 0; n < 4; ++n) o[n] = make_float2(0.f, 0.f);
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            const float2 mlw = ml_w[w * kRows + g];
            const float f = mlw.x == -INFINITY ? 0.f : exp2f(mlw.x - m);  // a warp without valid tokens contributes nothing
            l += mlw.y * f;
#pragma unroll
            for (int n = 0; n < 4; ++n) {
                const float2 v = w == warp ? make_float2(o_acc[w * 4 + n][2 * pass], o_acc[w * 4 + n][2 * pass + 1])
                                           : foreign[((warp * (kWarps - 1) + (w > warp ? w - 1 : w)) * 4 + n) * 32 + lane];
                o[n].x += v.x * f;
                o[n].y += v.y * f;
            }
        }
        if (g < p.group) {
            if (seg.n_parts == 1) {  // no other part: finish here
                __nv_bfloat16 *dst = p.out + ((size_t)seg.b * p.Hq + head0 + g) * kD + warp * 32 + c0;
#pragma unroll
                for (int n = 0; n < 4; ++n)
                    *reinterpret_cast<__nv_bfloat162 *>(dst + n * 8) = __floats2bfloat162_rn(o[n].x / l, o[n].y / l);
                if (p.lse && warp == 0 && (lane & 3) == 0)
                    p.lse[(size_t)seg.b * p.Hq + head0 + g] = (m + log2f(l)) * 0.6931471805599453f;
            } else {
                float *dst = part_o + (size_t)g * kD + warp * 32 + c0;
#pragma unroll
                for (int n = 0; n < 4; ++n) *reinterpret_cast<float2 *>(dst + n * 8) = o[n];
                if (warp == 0 && (lane & 3) == 0) part_ml[g] = make_float2(m, l);
            }
        }
    }
}

// The parts of one sequence, merged in ascending order by the block that counted the last of them.  A chain of round trips
// to L2 for one block, so loads are kept in flight: the outputs of the first eight parts are fetched together with all
// parts' (max, sum) pairs, eight threads per head, which leave the parts' factors in shared memory; the outputs then go
// eight parts deep.
constexpr int kMergeDeep = 8, kMergeBatch = 8 * kMergeDeep;  // parts whose factors are in shared memory at a time
static_assert(kMergeBatch * kRows <= kMergeFloats, "factors of a batch of parts");
__device__ __forceinline__ void merge_parts(const Params &p, const Segment &seg, float *merge, int tid) {
    const int lane = tid & 31, head0 = seg.kvh * p.group, n_parts = seg.n_parts, group = p.group;
    const long long first_slot = seg.first_slot, second_slot = seg.second_slot;
    const int step = seg.slot_step;
    auto slot_of = [&](int i) { return i == 0 ? first_slot : second_slot + (long long)(i - 1) * step; };
    const float2 *all_ml = reinterpret_cast<const float2 *>(p.part_ml);
    float *factor = merge;                                            // [part of the batch][head]
    float *head_l = merge + kMergeFloats + kWarps * kRows * 2;        // [16]
    // thread t owns four dims of heads t / 32, t / 32 + 4, ...: two heads at a time
    constexpr int kHeadsPerThread = kRows / kWarps;
    float4 o[kHeadsPerThread], v0[kMergeDeep], v1[kMergeDeep];
    auto fetch = [&](int first, int j0) {  // parts first .. first + 7 (clamped), heads t / 32 + 4 j0 and the next
        const int g0 = (tid >> 5) + kWarps * j0, g1 = g0 + kWarps;
#pragma unroll
        for (int u = 0; u < kMergeDeep; ++u) {
            const float *src = p.part_o + (size_t)(slot_of(min(first + u, n_parts - 1)) * group) * kD + lane * 4;
            v0[u] = g0 < group ? __ldcg(reinterpret_cast<const float4 *>(src + g0 * kD)) : make_float4(0.f, 0.f, 0.f, 0.f);
            v1[u] = g1 < group ? __ldcg(reinterpret_cast<const float4 *>(src + g1 * kD)) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    };
    const int mg = tid >> 3, sub = tid & 7;
    float2 ml[kMergeDeep];
    auto fetch_ml = [&](int first) {  // parts first + sub, first + sub + 8, ...
#pragma unroll
        for (int u = 0; u < kMergeDeep; ++u)
            ml[u] = mg < group && first + sub + 8 * u < n_parts ? __ldcg(&all_ml[slot_of(first + sub + 8 * u) * group + mg])
                                                                : make_float2(-INFINITY, 0.f);
    };
    fetch_ml(0);
    fetch(0, 0);
    // Weight of a sum taken relative to the maximum `from` in one relative to `to`.  No difference is taken of equal maxima:
    // parts whose scores are all NaN have a maximum of -inf and a NaN sum, which must reach lse as a NaN.
    auto factor_of = [](float from, float to) { return from == to ? 1.f : exp2f(from - to); };
    float m = -INFINITY, l = 0.f;
    for (int base = 0;;) {
        float m_new = m;
#pragma unroll
        for (int u = 0; u < kMergeDeep; ++u) m_new = fmaxf(m_new, ml[u].x);
        l *= factor_of(m, m_new);
#pragma unroll
        for (int u = 0; u < kMergeDeep; ++u) l += ml[u].y * factor_of(ml[u].x, m_new);
        m = m_new;
        base += kMergeBatch;
        if (base >= n_parts) break;
        fetch_ml(base);
    }
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) {  // (a fixed tree)
        const float om = __shfl_xor_sync(0xffffffffu, m, off), ol = __shfl_xor_sync(0xffffffffu, l, off);
        const float mm = fmaxf(m, om);
        l = l * factor_of(m, mm) + ol * factor_of(om, mm);
        m = mm;
    }
    sync_compute();  // (the buffers' previous readers are done)
    if (mg < group && sub == 0) {
        head_l[mg] = l;
        if (p.lse) p.lse[(size_t)seg.b * p.Hq + head0 + mg] = (m + log2f(l)) * 0.6931471805599453f;
    }
#pragma unroll
    for (int j = 0; j < kHeadsPerThread; ++j) o[j] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int base = 0; base < n_parts; base += kMergeBatch) {
        const int n = min(kMergeBatch, n_parts - base);
        if (n_parts > kMergeBatch) {
            if (base > 0) sync_compute();  // the previous batch's factors have been used
            fetch_ml(base);
        }
#pragma unroll
        for (int u = 0; u < kMergeDeep; ++u)
            if (mg < group && sub + 8 * u < n) factor[(sub + 8 * u) * group + mg] = exp2f(ml[u].x - m);
        sync_compute();
#pragma unroll
        for (int j0 = 0; j0 < kHeadsPerThread; j0 += 2) {
            const int g0 = (tid >> 5) + kWarps * j0, g1 = g0 + kWarps;
            if (g0 >= group) break;
            for (int i0 = 0; i0 < n; i0 += kMergeDeep) {
                if (base + i0 > 0 || j0 > 0) fetch(base + i0, j0);
#pragma unroll
                for (int u = 0; u < kMergeDeep; ++u) {
                    if (i0 + u >= n) break;
                    const float f0 = factor[(i0 + u) * group + g0], f1 = g1 < group ? factor[(i0 + u) * group + g1] : 0.f;
                    o[j0].x += v0[u].x * f0; o[j0].y += v0[u].y * f0; o[j0].z += v0[u].z * f0; o[j0].w += v0[u].w * f0;
                    o[j0 + 1].x += v1[u].x * f1; o[j0 + 1].y += v1[u].y * f1; o[j0 + 1].z += v1[u].z * f1; o[j0 + 1].w += v1[u].w * f1;
                }
            }
        }
    }
#pragma unroll
    for (int j = 0; j < kHeadsPerThread; ++j) {
        const int g = (tid >> 5) + kWarps * j;
        if (g >= group) break;
        const float l_all = head_l[g];
        __nv_bfloat162 lo = __floats2bfloat162_rn(o[j].x / l_all, o[j].y / l_all), hi = __floats2bfloat162_rn(o[j].z / l_all, o[j].w / l_all);
        uint2 packed;
        packed.x = *reinterpret_cast<uint32_t *>(&lo);
        packed.y = *reinterpret_cast<uint32_t *>(&hi);
        *reinterpret_cast<uint2 *>(&p.out[((size_t)seg.b * p.Hq + head0 + g) * kD + lane * 4]) = packed;
    }
    sync_compute();  // (a second merge of this block writes the same buffers)
}

// Up to two parts a block has stored are counted at their sequences (thread i of the block: part i); the block that arrives
// last merges the sequence, so the result does not depend on which block that is.  Once, at the block's end: a fence and an
// atomic's round trip in the middle would stop the stream for a microsecond or two each.
struct BlockParts {
    Segment part[2];
    int is_last[2];
};
__device__ __forceinline__ void count_and_merge(const Params &p, BlockParts &s, float *merge, volatile int *gave_up, int tid) {
    sync_compute();  // the parts are stored ...
    if (s.part[0].n_parts <= 1 && s.part[1].n_parts <= 1) return;
    if (tid < 2) {
        const Segment &seg = s.part[tid];
        __threadfence();  // ... and visible before they are counted
        s.is_last[tid] = seg.n_parts > 1 && *gave_up == 0 &&
                         atomicAdd(&p.counters[(size_t)seg.b * p.Hkv + seg.kvh], 1) == seg.n_parts - 1;
        __threadfence();
    }
    sync_compute();
    for (int i = 0; i < 2; ++i)
        if (s.is_last[i]) merge_parts(p, s.part[i], merge, tid);
}

// The row gather, for page sizes TMA boxes cannot follow: one 256-byte bulk copy per token row, issued by the 128 compute
// threads themselves, two stages in three blocks per SM, a block barrier per chunk; one block per (sequence split,
// key-value head, item).
template <bool kChained>
__global__ void __launch_bounds__(kThreads, kBlocksPerSm)
gqa_row_decode_kernel(const Params p) {
    extern __shared__ __align__(128) uint8_t smem_raw[];
    uint8_t *smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    __shared__ int gave_up;
    __shared__ BlockParts parts;
    __shared__ __align__(8) unsigned long long full_bar[kStages];
    const int split = blockIdx.x, kvh = blockIdx.y, b = blockIdx.z;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool first_block = (blockIdx.x | blockIdx.y | blockIdx.z) == 0;
    if (kChained) {
        moe::chain_release();
        wait_for_inputs(true);
    }
    int first_page;
    const int L = cached_tokens<kChained>(p, b, first_page);
    const int head0 = kvh * p.group;

    if (L <= 0) {  // nothing cached: out = 0, lse = -inf (written by the first split's block)
        if (split == 0) write_empty(p, b, head0, tid);
        zero_own_status(p, first_block, tid);
        return;
    }
    const int n_active = min(p.n_splits, (L + p.split_tokens - 1) / p.split_tokens);
    if (split >= n_active) return;
    const int begin = split * p.split_tokens;
    const int end = split == n_active - 1 ? L : begin + p.split_tokens;  // the last active split runs to the end
    const int n_chunks = (end - begin + kChunk - 1) / kChunk;
    uint32_t qa[kD / 16][4];
    load_queries(p, b, head0, lane, qa);

    // Thread i brings ONE token row per chunk -- row i % 64 of the keys (i < 64) or of the values -- and arrives on the
    // stage's barrier once per chunk, with its bytes when its row exists.
    const int *page_list = p.kv_indices + (kChained ? first_page : p.kv_indptr[b]);
    const size_t token_stride = (size_t)p.Hkv * kD;  // elements between consecutive slots of a page
    const uint32_t smem_base = smem_u32(smem), bar_base = smem_u32(full_bar);
    const int my_row = tid & (kChunk - 1);
    const bool my_values = tid >= kChunk;
    const __nv_bfloat16 *my_cache = (my_values ? p.v_cache : p.k_cache) + (size_t)kvh * kD;
    const uint32_t my_dst = (my_values ? (uint32_t)kTileBytes : 0u) + (uint32_t)(my_row * kRowPitch);
    if (tid == 0) {
        for (int s = 0; s < kStages; ++s) mbar_init(bar_base + s * 8, kThreads);
        gave_up = 0;
        zero_own_status(p, first_block, tid);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncthreads();
    // Where this thread's row of a chunk lives (its slot in the cache), -1 past the end of the split.  The page table is
    // read ONE CHUNK AHEAD of the copy that needs it, so its latency never sits between copies.
    auto locate = [&](int chunk) -> int {
        const int tok = begin + chunk * kChunk + my_row;
        if (chunk >= n_chunks || tok >= end) return -1;
        return load_index<kChained>(&page_list[tok / p.page_size]) * p.page_size + tok % p.page_size;
    };
    int next_loc = locate(0);
    auto issue_chunk = [&](int chunk) {  // called for chunk 0, 1, 2, ... in order
        if (chunk < n_chunks) {
            const int stage = chunk % kStages;
            const uint32_t dst = smem_base + stage * kStageBytes + my_dst, bar = bar_base + stage * 8;
            if (next_loc >= 0) {
                mbar_arrive_expect_tx(bar, kRowBytes);
                bulk_copy(dst, my_cache + (size_t)next_loc * token_stride, kRowBytes, bar);
            } else {  // a row past the end: zeros, so that a masked probability of 0 meets a finite value
#pragma unroll
                for (int i = 0; i < kRowBytes / 16; ++i)
                    asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(dst + i * 16), "r"(0) : "memory");
                mbar_arrive(bar);
            }
        }
        next_loc = locate(chunk + 1);
    };

    float o_acc[kD / 8][4];  // this warp's 16 x 128 output tile: 16 n-tiles of 8 dims
#pragma unroll
    for (int n = 0; n < kD / 8; ++n)
#pragma unroll
        for (int i = 0; i < 4; ++i) o_acc[n][i] = 0.f;
    float m_run[2] = {-INFINITY, -INFINITY}, l_run[2] = {0.f, 0.f};  // rows lane/4 and lane/4 + 8

    for (int c = 0; c < kStages - 1; ++c) issue_chunk(c);
    bool ok = true;
    for (int chunk = 0; chunk < n_chunks; ++chunk) {
        ok = bounded_wait(bar_base + (chunk % kStages) * 8, (uint32_t)(chunk / kStages) & 1u, kWaitLimit, &gave_up, p.status);
        ok = __syncthreads_and(ok);           // chunk `chunk` has landed and every thread is done with chunk - 1's stage
        if (!ok) break;
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // (that stage is about to be overwritten by copies)
        issue_chunk(chunk + kStages - 1);
        const uint32_t k_tile = smem_base + (chunk % kStages) * kStageBytes;
        const int tok_base = begin + chunk * kChunk + warp * 16;
        if (tok_base < end)                   // (uniform over the warp)
            attend_16_tokens<false>(qa, o_acc, m_run, l_run, k_tile, k_tile + kTileBytes, warp * 16, tok_base, end, 0,
                                    p.scale_log2, lane);
    }
    // A block that gave up waits (bounded) for its copies in flight, then leaves without a result: the status word says so.
    if (!ok) {
        for (int i = 0; i < 1000; ++i) __nanosleep(1000);
        return;
    }
    __syncthreads();  // all copies were waited for: the pipeline's shared memory becomes the merge buffer
    const long long bh = (long long)b * p.Hkv + kvh;
    Segment seg;
    seg.b = b; seg.kvh = kvh;
    seg.n_parts = n_active;
    seg.first_slot = bh * p.n_splits;
    seg.second_slot = seg.first_slot + 1;
    seg.slot = seg.first_slot + split;
    seg.slot_step = 1;
    if (tid == 0) {
        parts.part[0] = seg;
        parts.part[1].n_parts = 1;
    }
    store_segment(p, seg, o_acc, m_run, l_run, reinterpret_cast<float *>(smem), warp, lane);
    count_and_merge(p, parts, reinterpret_cast<float *>(smem), &gave_up, tid);
}

// The tiled gather: the page size is a power of two of at least 8, and a chunk is one TMA box per (page, keys or values),
// issued by a fifth warp that does nothing else, three stages deep, in two blocks per SM: the four compute warps never
// touch the copy engine, and stages are handed back and forth on full / empty mbarriers, so the loop has no block-wide
// barrier.  (A thread is held for as long as the engine takes to turn its box into requests, 5 to 9 cycles per
// 128-byte row: 600 cycles per chunk and warp when the four compute warps shared the issuing, against 1000 for the
// arithmetic.)
//
// Which tokens a block takes.  The lengths are known on the device only.  With a fixed share per block (one sequence, or
// one of its fixed splits) the kernel's time on a ragged batch is that of the longest share while most of the machine
// waits.  The balanced form lays all chunks of the batch on one line, sequence after sequence, and gives each of the
// resident blocks an equal piece of it: a few whole sequences and a part of one at either end, through ONE copy pipeline
// that never drains between sequences; a block leaves at most two partial results.  It costs the counting and merging of
// those parts at the end, when every block finishes at once, so the blocks of a batch that fits the machine once or twice
// (kAdaptive) read all lengths first and take the form that balanced_is_faster says.  In the fixed form they then take the
// i-th of the shares that have tokens, not the i-th of the grid: blocks that found their share empty only after reading all
// lengths had already made the others share an SM (one sequence of 20 000 tokens, an empty one and a hint of 40 000:
// 28.6 -> 26.7 us).  Batches of more blocks than that balance themselves.
constexpr int kBalancedBlocks = (int)kSms * 2;  // as many as are resident
constexpr int kMinPiece = 4;              // chunks a balanced block takes at least
constexpr int kSmemBytesTiled = kTiledStages * kTiledStageBytes + kMergeBytes + 1024;
static_assert(kSmemBytesTiled + 1024 <= 113 * 1024, "two blocks per SM");
static_assert(kMergeBytes <= kStages * kStageBytes, "the row kernel merges in its pipeline's memory");

// Which form is faster, fitted to 500 measured batches (1 to 150 sequences of 128 to 65 536 tokens, equal and ragged, with
// empty ones among them, length hints of 1 to 16 times the longest).  Balanced: 5 ns per chunk of the batch, the memory's
// rate, and about 15 us.  Fixed shares in one wave: that stream, or the longest share alone (0.9 us per chunk), whichever is
// longer; 0.15 us per chunk that the longest share is longer than the average one; about 4 us; and, where sequences are cut,
// their merge, which costs the balanced form more the more parts they are cut into anyway.  Fixed shares in two waves lost 5
// to 35 us to the balanced form wherever the lengths differed and the longest sequence had 64 chunks or more, and were even
// with it or ahead elsewhere.  The form taken was 0.7 % slower than the better one on average over the 500 batches, and 2 %
// over 400 others.
// Fixed / balanced, us: 64 sequences of 1024..8192 tokens 120 / 105, equal 8192 164 / 179; 4 of 4096 over 8 heads with a
// hint of 16 384 33 / 24; 7 of 20 000 beside an empty one, hint 40 000, 70 / 60; 30 equal ones of 4000 over 8 heads 77 / 87.
__device__ __forceinline__ bool balanced_is_faster(long long total, int longest_share, int n_shares, int longest_sequence,
                                                   int n_sequences, int most_parts) {
    if (n_shares > kBalancedBlocks)
        return longest_sequence >= 64 && (float)longest_sequence * (float)n_sequences > 1.15f * (float)total;
    const float stream = 0.005f * (float)total, average = (float)total / (float)n_shares, longest = (float)longest_share;
    const float merge = most_parts > 1 ? 8.5f - 0.7f * (float)most_parts : 0.f;
    return fmaxf(stream, 0.9f * longest) + 0.15f * (longest - average) + merge > stream + 11.f;
}

template <bool kAdaptive, bool kChained>
__global__ void __launch_bounds__(kThreads + 32, 2)
gqa_tiled_decode_kernel(const Params p, const __grid_constant__ CUtensorMap k_map, const __grid_constant__ CUtensorMap v_map) {
    extern __shared__ __align__(128) uint8_t smem_raw[];
    uint8_t *smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    __shared__ BlockParts parts;
    __shared__ struct { long long total, begin, end; int n_blocks; bool balanced; } line;  // (fixed: n_blocks = the sequence's parts)
    __shared__ int gave_up, range_start[kThreads], warp_sum[kWarps], warp_longest[kWarps], warp_sequence[kWarps],
        warp_shares[kWarps];
    __shared__ __align__(8) unsigned long long full_bar[kTiledStages], empty_bar[kTiledStages];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t smem_base = smem_u32(smem), full_base = smem_u32(full_bar), empty_base = smem_u32(empty_bar);
    const int sh = 31 - __clz(p.box_rows);  // log2 of the rows of a box
    static_assert(!kAdaptive || !kChained, "parts may be counted");
    if (kChained) moe::chain_release();
    else if (!kAdaptive) zero_own_status(p, blockIdx.x == 0, tid);
    if (tid == 0) {
        for (int s = 0; s < kTiledStages; ++s) {
            mbar_init(full_base + s * 8, 32);       // the copy warp's lanes
            mbar_init(empty_base + s * 8, kWarps);  // one arrival per compute warp
        }
        gave_up = 0;
        parts.part[0].n_parts = parts.part[1].n_parts = 1;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }

    if (kChained) {
        wait_for_inputs(warp == kWarps);  // (the set-up above overlaps the end of what is in front)
        zero_own_status(p, blockIdx.x == 0, tid);
    }

    // ---- this block's piece: w_end - w chunks, the first of them chunk c of sequence (b, kvh) ----
    int b, kvh, c, L, n_chunks;  // the sequence the cursor is in, its tokens and chunks
    int first_page = 0;          // (chained: of the block's only sequence)
    long long w = 0, w_end = 0;
    const int split_chunks = p.split_tokens / kChunk;
    bool balanced = false;
    if (kAdaptive) {
        // chunks per item, 128 ranges of items, and what the fixed shares would be: every block computes the same
        const int per = (p.B + kThreads - 1) / kThreads;
        int sum = 0, longest = 0, sequence = 0, shares = 0;
        if (tid < kThreads)
            for (int i = tid * per; i < min(p.B, (tid + 1) * per); ++i) {
                const int n = (cached_tokens<kChained>(p, i) + kChunk - 1) / kChunk;
                if (n <= 0) continue;  // an item without tokens has no share
                const int parts_of = min(p.n_splits, (n + split_chunks - 1) / split_chunks);
                sum += n;
                sequence = max(sequence, n);
                shares += parts_of;
                if (parts_of > 1) longest = max(longest, split_chunks);
                longest = max(longest, n - (parts_of - 1) * split_chunks);
            }
        int incl = sum, shares_incl = shares;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, off), u = __shfl_up_sync(0xffffffffu, shares_incl, off);
            if (lane >= off) { incl += v; shares_incl += u; }
        }
        longest = __reduce_max_sync(0xffffffffu, longest);
        sequence = __reduce_max_sync(0xffffffffu, sequence);
        if (warp < kWarps && lane == 31) {
            warp_sum[warp] = incl;
            warp_longest[warp] = longest;
            warp_sequence[warp] = sequence;
            warp_shares[warp] = shares_incl;
        }
        __syncthreads();
        int before = incl - sum, chunks = 0, shares_before = shares_incl - shares;
        longest = sequence = shares = 0;
#pragma unroll
        for (int i = 0; i < kWarps; ++i) {
            if (i < warp) { before += warp_sum[i]; shares_before += warp_shares[i]; }
            chunks += warp_sum[i];
            longest = max(longest, warp_longest[i]);
            sequence = max(sequence, warp_sequence[i]);
            shares += warp_shares[i];
        }
        const long long total = (long long)chunks * p.Hkv;
        balanced = total > 0 && balanced_is_faster(total, longest, shares * p.Hkv, sequence, p.B * p.Hkv,
                                                   min(p.n_splits, (sequence + split_chunks - 1) / split_chunks));
        if (tid < kThreads) range_start[tid] = balanced ? before : shares_before;
        __syncthreads();
        // items without tokens are dealt out to the blocks
        if (tid < kThreads)
            for (int i = blockIdx.x; i < p.B; i += gridDim.x)
                if (cached_tokens<kChained>(p, i) <= 0)
                    for (int h = 0; h < p.Hkv; ++h) write_empty(p, i, h * p.group, tid);
        // The blocks' work starts at a chunk of the line (balanced) or at a share; both lie item after item, head after head.
        int n_blocks = shares * p.Hkv;
        long long start = blockIdx.x;
        if (balanced) {
            // no block takes less than kMinPiece chunks: short lines use fewer blocks
            const long long most = (total + kMinPiece - 1) / kMinPiece;
            n_blocks = (int)(most < kBalancedBlocks ? most : kBalancedBlocks);
        }
        if ((int)blockIdx.x >= n_blocks) return;
        if (balanced) {
            w = divide(total * blockIdx.x, n_blocks);
            w_end = divide(total * (blockIdx.x + 1), n_blocks);
            start = w;
            if (tid == 0) { line.total = total; line.begin = w; line.end = w_end; line.n_blocks = n_blocks; line.balanced = true; }
            if (blockIdx.x == 0 && tid == 0) p.status[3] = 1;  // (reporting: the batch was cut into equal pieces)
        }
        const int x = (int)divide(start, p.Hkv);
        int r = 0;  // the last range that starts at or before chunk or share x of the items
#pragma unroll
        for (int step = kThreads / 2; step > 0; step >>= 1)
            if (range_start[r + step] <= x) r += step;
        int at = range_start[r], units;  // `units`: the item's chunks or shares per head
        b = r * per - 1;
        do {
            L = cached_tokens<kChained>(p, ++b);
            n_chunks = (L + kChunk - 1) / kChunk;
            units = balanced ? n_chunks : min(p.n_splits, (n_chunks + split_chunks - 1) / split_chunks);
            at += max(units, 0);
        } while (at <= x);
        at -= units;
        const int rest = (int)(start - (long long)at * p.Hkv);
        kvh = rest / units;
        c = rest - kvh * units;
        if (!balanced) {
            c *= split_chunks;
            w_end = (c + split_chunks >= units * split_chunks ? n_chunks : c + split_chunks) - c;  // the last split runs to the end
            if (tid == 0) { line.n_blocks = units; line.balanced = false; }
        }
    } else {
        const int split = blockIdx.x % p.n_splits;
        kvh = (blockIdx.x / p.n_splits) % p.Hkv;
        b = blockIdx.x / p.n_splits / p.Hkv;
        L = cached_tokens<kChained>(p, b, first_page);
        n_chunks = (L + kChunk - 1) / kChunk;
        if (L <= 0) {
            if (split == 0 && tid < kThreads) write_empty(p, b, kvh * p.group, tid);
            return;
        }
        const int n_parts = min(p.n_splits, (n_chunks + split_chunks - 1) / split_chunks);
        if (split >= n_parts) return;
        c = split * split_chunks;
        w_end = (split == n_parts - 1 ? n_chunks : c + split_chunks) - c;  // the last split runs to the end
        if (tid == 0) { line.n_blocks = n_parts; line.balanced = false; }
    }
    __syncthreads();
    auto next_sequence = [&]() {
        c = 0;
        if (++kvh == p.Hkv) {
            kvh = 0;
            do {
                L = cached_tokens<kChained>(p, ++b);  // (there is one: the line goes on)
            } while (L <= 0);
            n_chunks = (L + kChunk - 1) / kChunk;
        }
    };

    if (warp == kWarps) {
        // ---- the copy warp: chunk after chunk into the ring, each stage as soon as the four compute warps are done with
        // its previous use.  A chunk is 128 / box_rows boxes -- (page of the chunk, keys or values), both halves of the dims
        // in one box -- one per lane; every lane arrives on the stage's barrier.  The page table is read one chunk ahead
        // of the copy that needs it.
        const bool has_box = lane < (2 * kChunk >> sh), my_values = lane & 1;
        const int my_row = (lane >> 1) << sh;
        const CUtensorMap *map = my_values ? &v_map : &k_map;
        const uint32_t my_dst = (my_values ? (uint32_t)kTiledTileBytes : 0u) + (uint32_t)(my_row * kRowBytes);
        const int *page_list = p.kv_indices + (kChained ? first_page : __ldg(&p.kv_indptr[b]));
        int page, slot, head;
        auto locate = [&]() {
            const int tok = c * kChunk + my_row;
            page = has_box && tok < L ? load_index<kChained>(&page_list[tok / p.page_size]) : -1;
            slot = tok & (p.page_size - 1);
            head = kvh;
        };
        locate();
        int stage = 0;
        uint32_t parity = 1;  // (a fresh barrier counts as handed back)
        for (long long left = w_end - w; left > 0; --left) {
            const bool free_ = bounded_wait(empty_base + stage * 8, parity, kWaitLimit, &gave_up, p.status);
            if (!__all_sync(0xffffffffu, free_)) break;
            const uint32_t bar = full_base + stage * 8;
            if (page >= 0) {
                mbar_arrive_expect_tx(bar, p.box_rows * kRowBytes);
                tma_load_box(smem_base + stage * kTiledStageBytes + my_dst, map, slot, head, page, bar);
            } else {
                mbar_arrive(bar);
            }
            if (left > 1) {
                if (++c == n_chunks) {
                    const int old_b = b;
                    next_sequence();
                    if (b != old_b) page_list = p.kv_indices + load_index<kChained>(&p.kv_indptr[b]);
                }
                locate();
            }
            if (++stage == kTiledStages) { stage = 0; parity ^= 1u; }
        }
        return;
    }

    // ---- the compute warps: segment after segment, each a run of chunks of one sequence.  (What is only needed between
    // segments stays in shared memory: the loop over chunks has no registers to spare.)
    float *merge = reinterpret_cast<float *>(smem + kTiledStages * kTiledStageBytes);
    int stage = 0;
    uint32_t parity = 0;
    bool ok = true;
    for (long long left = w_end - w; left > 0;) {
        const int run = (int)(left < n_chunks - c ? left : n_chunks - c);
        uint32_t qa[kD / 16][4];
        load_queries(p, b, kvh * p.group, lane, qa);
        float o_acc[kD / 8][4];  // this warp's 16 x 128 output tile: 16 n-tiles of 8 dims
#pragma unroll
        for (int n = 0; n < kD / 8; ++n)
#pragma unroll
            for (int i = 0; i < 4; ++i) o_acc[n][i] = 0.f;
        float m_run[2] = {-INFINITY, -INFINITY}, l_run[2] = {0.f, 0.f};  // rows lane/4 and lane/4 + 8
        int tok_base = c * kChunk + warp * 16;
        for (int i = run; i > 0; --i, tok_base += kChunk) {
            if (ok) ok = __all_sync(0xffffffffu, bounded_wait(full_base + stage * 8, parity, kWaitLimit, &gave_up, p.status));
            if (!ok) break;
            const uint32_t k_tile = smem_base + stage * kTiledStageBytes;
            if (tok_base < L)  // (uniform over the warp)
                attend_16_tokens<true>(qa, o_acc, m_run, l_run, k_tile, k_tile + kTiledTileBytes, warp * 16, tok_base, L, sh,
                                       p.scale_log2, lane);
            __syncwarp();  // this warp is done with the stage (also when none of its tokens exist)
            if (lane == 0) mbar_arrive(empty_base + stage * 8);
            if (++stage == kTiledStages) { stage = 0; parity ^= 1u; }
        }
        // A block one of whose warps gave up stores and counts nothing more: what it would store is not the whole segment.
        if (any_compute(!ok)) { ok = false; break; }
        Segment seg;
        seg.b = b; seg.kvh = kvh;
        bool first = true;
        if (kAdaptive && line.balanced) {
            // the blocks that share this sequence: those whose pieces hold its first and its last chunk
            const long long total = line.total, w0 = line.end - left - c, w1 = w0 + n_chunks - 1;
            const int n_blocks = line.n_blocks;
            const int g0 = (int)divide((w0 + 1) * n_blocks + total - 1, total) - 1, g1 = (int)divide((w1 + 1) * n_blocks + total - 1, total) - 1;
            first = line.end - left == line.begin;
            // a block's slots: 2 g for a sequence its piece begins with, 2 g + 1 for one it enters later
            seg.n_parts = g1 - g0 + 1;
            seg.slot = 2ll * blockIdx.x + (first ? 0 : 1);
            seg.first_slot = 2ll * g0 + (divide(total * g0, n_blocks) == w0 ? 0 : 1);
            seg.second_slot = 2ll * (g0 + 1);
            seg.slot_step = 2;
        } else {
            const long long bh = (long long)b * p.Hkv + kvh;
            seg.n_parts = line.n_blocks;
            seg.first_slot = bh * p.n_splits;
            seg.second_slot = seg.first_slot + 1;
            seg.slot = seg.first_slot + c / split_chunks;
            seg.slot_step = 1;
        }
        store_segment(p, seg, o_acc, m_run, l_run, merge, warp, lane);
        if (seg.n_parts > 1 && tid == 0) parts.part[first ? 0 : 1] = seg;  // at most two: the piece's first sequence, and its last
        left -= run;
        if (left > 0) next_sequence();
    }
    count_and_merge(p, parts, merge, &gave_up, tid);
    // A block that gave up waits (bounded) for its copies in flight before it leaves.
    if (!ok)
        for (int i = 0; i < 1000; ++i) __nanosleep(1000);
}

bool envelope_ok(long long B, int Hq, int Hkv, int D, long long max_kv_len) {
    if (B < 0 || Hq < 1 || Hkv < 1 || D != kD || max_kv_len < 0) return false;
    if (Hq % Hkv != 0 || Hq / Hkv > kRows) return false;
    return B <= 65535 && Hkv <= 65535;  // grid dimensions y and z
}

// Sequence splits, from a model of the kernel's time in units of one chunk streamed by a block on a full machine
// (1.4 us).  148 SMs x 2 blocks are resident at a time (the copy-warp variant), so blocks run in waves; a block costs
// its chunks plus 3 (pipeline fill, the warps' merge); a wave that fills a fraction f of the machine runs in
// max(0.47, f) of a full wave's time (a block alone streams a chunk in 0.47 of the time, and 0.86 of a wave already
// saturates the memory); a split sequence pays the partial results' round trip and the last block's merge once,
// 5 + n / 10; and while the machine is not full, 0.3 x (the idle share) of a block's length is added for the tail that
// sequences shorter than max_kv_len leave (their lengths are known to the device only; on a full machine the blocks
// that remain speed up as others finish, on a part-empty one they already run at their own limit).  The constants
// were fitted to measured split sweeps (batches of 1 to 256, 2k to 64k tokens, equal and ragged lengths); the chosen
// count was within 10 % of the best measured one in each.  Ties go to fewer splits; no split is shorter than four
// chunks.
void choose_fixed_split(int B, int Hkv, int max_kv_len, int *split_tokens, int *n_splits) {
    const long long base = (long long)B * Hkv, slots = 148 * kModelBlocksPerSm;
    const long long chunks = max_kv_len > 0 ? ((long long)max_kv_len + kChunk - 1) / kChunk : 1;
    long long most = (chunks + 3) / 4;
    if (most > kMaxSplits) most = kMaxSplits;
    if (most < 1) most = 1;
    long long best_n = 1;
    double best_cost = -1.0;
    for (long long n = 1; n <= most; ++n) {
        const long long per_block = (chunks + n - 1) / n, n_eff = (chunks + per_block - 1) / per_block;
        if (n_eff != n) continue;  // (the same split as a smaller n)
        const long long blocks = (base > 0 ? base : 1) * n, full_waves = blocks / slots;
        const double f = (double)(blocks - full_waves * slots) / (double)slots;
        const double last_wave = f > 0.0 ? (f > 0.47 ? f : 0.47) : 0.0;
        const double idle = blocks < slots ? 1.0 - (double)blocks / (double)slots : 0.0;
        const double cost = ((double)per_block + 3.0) * ((double)full_waves + last_wave) +
                            0.3 * idle * (double)per_block + (n > 1 ? 5.0 + 0.1 * (double)n : 0.0);
        if (best_cost < 0 || cost < best_cost * (1.0 - 1e-9)) { best_cost = cost; best_n = n; }
    }
    const long long per_block = (chunks + best_n - 1) / best_n;
    *split_tokens = (int)(per_block * kChunk);
    *n_splits = (int)((chunks + per_block - 1) / per_block);
}

// Slots per (item, key-value head) the workspace is sized for: the fixed splits, or more where a long sequence's batch would
// otherwise have fewer slots than the balanced blocks need, two each.  Sequences of up to 32 chunks keep the fixed
// split's: there the batch either has slots enough or its blocks are short anyway.
int choose_slots(int B, int Hkv, int max_kv_len, int fixed_splits) {
    const long long base = (long long)B * Hkv, chunks = ((long long)max_kv_len + kChunk - 1) / kChunk;
    if (base < 1 || chunks <= 32 || base * fixed_splits >= 2 * kBalancedBlocks) return fixed_splits;
    long long n = (2 * kBalancedBlocks + base - 1) / base;
    if (n > chunks / 4) n = chunks / 4;
    if (n > kMaxSplits) n = kMaxSplits;
    if (n <= fixed_splits) return fixed_splits;
    const long long per_slot = chunks / n;  // (rounded down: at least n slots, in whole runs of chunks)
    const long long slots = (chunks + per_slot - 1) / per_slot;
    return slots > kMaxSplits ? fixed_splits : (int)slots;
}

size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

size_t workspace_bytes_for(int B, int Hq, int Hkv, int slots) {
    const size_t bh = (size_t)B * Hkv, group = Hq / Hkv;
    return 256 + align_up(bh * sizeof(int), 256) + align_up(bh * slots * group * 2 * sizeof(float), 256) +
           align_up(bh * slots * group * kD * sizeof(float), 256) + 256;
}

}  // namespace
}  // namespace gqa

extern "C" {

size_t gqa_decode_workspace_bytes(int B, int Hq, int Hkv, int D, int max_kv_len) {
    using namespace gqa;
    if (!envelope_ok(B, Hq, Hkv, D, max_kv_len)) return 0;
    int st, ns;
    choose_fixed_split(B, Hkv, max_kv_len, &st, &ns);
    return workspace_bytes_for(B, Hq, Hkv, choose_slots(B, Hkv, max_kv_len, ns));
}

int gqa_selftest_wait_timeout(void *workspace, size_t workspace_bytes, void *stream) {
    using namespace gqa;
    if (!workspace) return MOE_ERR_NULL;
    if (reinterpret_cast<uintptr_t>(workspace) % 256 != 0) return MOE_ERR_ALIGN;
    if (workspace_bytes < 256) return MOE_ERR_WORKSPACE;
    const int arch = moe::check_device();
    if (arch != MOE_OK) return arch;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (cudaMemsetAsync(workspace, 0, 256, st) != cudaSuccess) return MOE_ERR_CUDA;
    gqa_wait_timeout_selftest_kernel<<<1, kThreads, 0, st>>>(static_cast<int *>(workspace));
    return cudaGetLastError() == cudaSuccess ? MOE_OK : MOE_ERR_CUDA;
}

int gqa_decode_split_tokens(int B, int Hq, int Hkv, int D, int max_kv_len) {
    using namespace gqa;
    if (!envelope_ok(B, Hq, Hkv, D, max_kv_len)) return 0;
    int st, ns;
    choose_fixed_split(B, Hkv, max_kv_len, &st, &ns);
    return st;
}

int gqa_paged_decode(const void *q, const void *k_cache, const void *v_cache, const int32_t *kv_indptr,
                     const int32_t *kv_indices, const int32_t *kv_last_page_len, int B, int Hq, int Hkv, int D,
                     int page_size, int num_pages, int max_kv_len, float sm_scale, void *out, float *lse, void *workspace,
                     size_t workspace_bytes, void *stream) {
    using namespace gqa;
    if (B < 0 || Hq < 1 || Hkv < 1 || D < 1 || page_size < 1 || num_pages < 0 || max_kv_len < 0) return MOE_ERR_SHAPE;
    if (!envelope_ok(B, Hq, Hkv, D, max_kv_len)) return MOE_ERR_UNSUPPORTED;
    if ((long long)num_pages * page_size >= (1ll << 31)) return MOE_ERR_UNSUPPORTED;  // slot numbers are 32-bit
    if (B == 0) return MOE_OK;
    if (!q || !k_cache || !v_cache || !kv_indptr || !kv_indices || !kv_last_page_len || !out || !workspace) return MOE_ERR_NULL;
    auto misaligned = [](const void *ptr, size_t a) { return (reinterpret_cast<uintptr_t>(ptr) % a) != 0; };
    if (misaligned(q, 16) || misaligned(k_cache, 16) || misaligned(v_cache, 16) || misaligned(out, 16) ||
        misaligned(kv_indptr, 4) || misaligned(kv_indices, 4) || misaligned(kv_last_page_len, 4) || misaligned(lse, 4) ||
        misaligned(workspace, 256))
        return MOE_ERR_ALIGN;
    // A workspace that holds the fixed splits' results only is enough too: the fixed form then.
    int fixed_tokens, fixed_splits;
    choose_fixed_split(B, Hkv, max_kv_len, &fixed_tokens, &fixed_splits);
    int slots = choose_slots(B, Hkv, max_kv_len, fixed_splits);
    if (workspace_bytes < workspace_bytes_for(B, Hq, Hkv, slots)) slots = fixed_splits;
    if (workspace_bytes < workspace_bytes_for(B, Hq, Hkv, slots)) return MOE_ERR_WORKSPACE;
    const int arch = moe::check_device();
    if (arch != MOE_OK) return arch;

    Params p;
    p.q = static_cast<const __nv_bfloat16 *>(q);
    p.k_cache = static_cast<const __nv_bfloat16 *>(k_cache);
    p.v_cache = static_cast<const __nv_bfloat16 *>(v_cache);
    p.kv_indptr = kv_indptr;
    p.kv_indices = kv_indices;
    p.kv_last_page_len = kv_last_page_len;
    p.out = static_cast<__nv_bfloat16 *>(out);
    p.lse = lse;
    p.B = B; p.Hq = Hq; p.Hkv = Hkv; p.group = Hq / Hkv; p.page_size = page_size;
    p.split_tokens = fixed_tokens;
    p.n_splits = fixed_splits;
    p.scale_log2 = sm_scale * kLog2e;
    const size_t bh = (size_t)B * Hkv;
    char *ws = static_cast<char *>(workspace);
    p.status = reinterpret_cast<int *>(ws);  // status word first, as in the layer's workspace: moe_last_status reads it
    p.counters = reinterpret_cast<int *>(ws + 256);
    ws += 256 + align_up(bh * sizeof(int), 256);
    p.part_ml = reinterpret_cast<float *>(ws);
    ws += align_up(bh * slots * p.group * 2 * sizeof(float), 256);
    p.part_o = reinterpret_cast<float *>(ws);

    cudaStream_t st = static_cast<cudaStream_t>(stream);
    // Page sizes that are powers of two of at least 8 take the tiled gather: one 5-D tensor map per cache,
    // (64 dims, slot, half, head, page), a box of min(page_size, 64) slots x both halves in the 128-byte swizzle.
    const bool tiled = page_size >= 8 && (page_size & (page_size - 1)) == 0 && num_pages > 0;
    CUtensorMap k_map, v_map;
    memset(&k_map, 0, sizeof(k_map));
    memset(&v_map, 0, sizeof(v_map));
    p.box_rows = page_size < kChunk ? page_size : kChunk;
    if (tiled && (!moe::tc::encode_kv_cache_map(&k_map, k_cache, (uint64_t)num_pages, (uint32_t)page_size, (uint32_t)Hkv, (uint32_t)p.box_rows) ||
                  !moe::tc::encode_kv_cache_map(&v_map, v_cache, (uint64_t)num_pages, (uint32_t)page_size, (uint32_t)Hkv, (uint32_t)p.box_rows)))
        return MOE_ERR_CUDA;
    const unsigned shares = (unsigned)(bh * p.n_splits);
    // Two slots per balanced block: where the workspace has them, and the fixed shares fill the machine at most twice.
    const bool adaptive = tiled && bh * slots >= 2 * kBalancedBlocks && bh * p.n_splits <= 2 * kBalancedBlocks;
    p.own_status = p.n_splits == 1 && !adaptive;  // (no part is ever counted)
    const bool chained = p.own_status && chaining_is_faster(tiled, shares, max_kv_len);
    auto launch = [&](auto kernel, dim3 grid, int threads, int smem_bytes, const auto &...args) {
        if (!moe::tc::set_max_dynamic_smem_once(reinterpret_cast<const void *>(kernel), smem_bytes)) return MOE_ERR_CUDA;
        if (!p.own_status && cudaMemsetAsync(p.status, 0, 256 + bh * sizeof(int), st) != cudaSuccess) return MOE_ERR_CUDA;
        return moe::launch_clusters(kernel, chained, 1, grid, threads, smem_bytes, st, args...) == cudaSuccess ? MOE_OK : MOE_ERR_CUDA;
    };
    if (!tiled)
        return launch(chained ? gqa_row_decode_kernel<true> : gqa_row_decode_kernel<false>, dim3(p.n_splits, Hkv, B), kThreads, kSmemBytes, p);
    if (adaptive)
        return launch(gqa_tiled_decode_kernel<true, false>, shares > kBalancedBlocks ? shares : kBalancedBlocks, kThreads + 32, kSmemBytesTiled, p, k_map, v_map);
    return launch(chained ? gqa_tiled_decode_kernel<false, true> : gqa_tiled_decode_kernel<false, false>, shares, kThreads + 32, kSmemBytesTiled, p, k_map, v_map);
}

}  // extern "C"
