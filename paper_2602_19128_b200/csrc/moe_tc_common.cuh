// Device-side PTX wrappers, descriptors and the tile schedule decoder shared by the tcgen05 grouped-GEMM
// kernels (bf16, FP8-dequantising and MX FP8; one CTA per tile and CTA pairs), plus the host-side tensor-map
// encoders.
#pragma once

#include "moe_internal.cuh"

namespace moe {
namespace tc {

constexpr int kBlockK = 64;                        // K elements per ring slot = one 128-byte swizzle row
constexpr int kTileM = 128;                        // weight rows per CTA (MMA M per CTA)
constexpr int kSlotABytes = kTileM * kBlockK * 2;  // 16 KiB
constexpr int kRowBytes = kBlockK * 2;             // 128
constexpr int kThreads = 192;                      // warp 0 TMA, warp 1 MMA, warps 2..5 epilogue
constexpr int kEpilogueWarps = 4;
constexpr long long kWaitLimitCycles = 4000000000LL;  // about two seconds at full clock
constexpr uint32_t kWaitSuspendNs = 20000;            // upper bound of one hardware-suspended wait
constexpr int kNumActMaps = 16;                    // activation boxes of q, 2q, ..., 16q rows (q = 16, or 8 for pairs)

// Tensor maps of one grouped GEMM.  `w` is either a 2-D map over [E*w_rows, K] with a 128-row box
// (down projection) or a 5-D map over w13 viewed as [E][I/16][gate|up][16][H] whose
// {64,16,2,4,1} box delivers 64 features as 4 x (16 gate rows, 16 up rows) in one copy.
// act[i]: box of q * (i + 1) rows, so any token tile is ONE copy.  A kernel's parameters carry the boxes its tiles can have and
// no more (kMaps): a map is 128 bytes that the host looks up and copies and the launch carries, and sixteen where two are used
// made the tiny layer's call 18.6 us of host time, now 16.3 (in a loop 18.6 us per call, now 17.0).
template <int kMaps>
struct TensorMapsOf {
    CUtensorMap w;
    CUtensorMap act[kMaps];
    TensorMapsOf() {}
    template <int kMore>
    explicit TensorMapsOf(const TensorMapsOf<kMore> &m) : w(m.w) {
        static_assert(kMore >= kMaps, "the first of more");
        for (int i = 0; i < kMaps; ++i) act[i] = m.act[i];
    }
};
using TensorMaps = TensorMapsOf<kNumActMaps>;  // on the host, while it is filled

struct KernelParams {
    __nv_bfloat16 *out;
    const int *expert_offsets, *tile_prefix, *tile_order, *tile_rows;
    int *status;
    int E, n_k_blocks, n_out, w_rows, n_feature_tiles;
    const float *w_scale;  // FP8-weight kernels only: [E, w_rows/128, K/128] block scales
    int handover_role;     // hand-over between the two GEMMs of a call (moe_internal.cuh)
    int *handover;
    int handover_per_token_tile;
    // gather-in-load (wide-tile gate/up GEMM only): token rows are fetched from the layer's input by row index
    int gather_tokens = 0;
    const int *sorted_to_flat = nullptr;
    int top_k = 1;
};

// ---- PTX wrappers -----------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    return done != 0;
}
// The same test, but the thread may be suspended by the hardware for up to `hint_ns` (it is woken
// when the phase completes), so a long wait costs neither issue slots nor power.
__device__ __forceinline__ bool mbar_try_wait_suspend(uint32_t bar, uint32_t parity, uint32_t hint_ns) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(bar), "r"(parity), "r"(hint_ns)
        : "memory");
    return done != 0;
}
// Bounded wait.  Returns false if the CTA is aborting (this wait expired, or another role's did).
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag, int *status,
                                          int site) {
    if (mbar_try_wait(bar, parity)) return true;
    const long long start = clock64();
    while (true) {
        if (mbar_try_wait_suspend(bar, parity, kWaitSuspendNs)) {
            return true;
        }
        if (*abort_flag) return false;
        if (clock64() - start > kWaitLimitCycles) {
            *abort_flag = 1;
            if (atomicCAS(status, 0, (int)MOE_ERR_DEVICE_TIMEOUT) == 0) {
                status[1] = site;
                status[2] = blockIdx.x;
            }
            return false;
        }
    }
}

// True in exactly one lane of a converged warp, always the same lane.  Waits and bookkeeping between tiles are run by
// whole warps.  An MMA warp enters this predicate once per TILE and its thread waits for and issues all of the tile's
// slots: the election, the vote on the wait's result and the warp barrier of every slot had cost more issue time than a
// narrow slot's MMAs take (one-token Mixtral-shaped layer 160 -> 137 us, FP8-weight layer of 32 tokens 291 -> 267 us,
// MX prefill on 32 resident experts 585 -> 572 us).  The one-CTA kernels' producers do the same (137 -> 135 us, one-token
// MX layer 87.6 -> 85.7); the pair kernels' producers (MX prefill 572 -> 576 us) and the power-bound bf16 wide-tile
// kernel (no change) keep the election per slot.  With a single lane running the whole loop under `lane == 0` instead,
// every TMA or MMA instruction cost about 150 cycles.
__device__ __forceinline__ bool elect_one() {
    uint32_t pred;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "elect.sync _|p, 0xffffffff;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(pred));
    return pred != 0;
}
// Ring position after n more slots.
template <int kStages>
__device__ __forceinline__ void ring_advance(int &stage, uint32_t &phase, int n) {
    const int uses = stage + n;
    phase ^= (uint32_t)(uses / kStages) & 1u;
    stage = uses % kStages;
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, int c0, int c1, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap *map, int c0, int c1, int c2, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void tma_load_5d(uint32_t dst, const CUtensorMap *map, int c0, int c1, int c2, int c3,
                                            int c4, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, %6}], [%7];"
        ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(bar)
        : "memory");
}

// A tensor map into the descriptor cache, ahead of the first copy that uses it.
__device__ __forceinline__ void prefetch_map(const CUtensorMap *map) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory");
}

__device__ __forceinline__ void tcgen05_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tcgen05_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// 16 consecutive fp32 columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_load_16(uint32_t taddr, float (&v)[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// 32 of them, as two groups of 16.
__device__ __forceinline__ void tmem_load_2x16(uint32_t taddr, float (&v)[2][16]) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
        "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i >> 4][i & 15] = __uint_as_float(r[i]);
}

// Shared-memory matrix descriptor for a K-major bf16 tile whose rows are 128 bytes with the 128-byte
// swizzle TMA applies: start address, leading offset 1 (unused for swizzled K-major), stride between
// 8-row groups 1024 bytes, descriptor version 1, layout type 2 (128-byte swizzle).
__device__ __forceinline__ uint64_t smem_desc_k_major_sw128(uint32_t smem_addr) {
    uint64_t d = 0;
    d |= (uint64_t)((smem_addr & 0x3FFFFu) >> 4);
    d |= (uint64_t)1 << 16;
    d |= (uint64_t)(1024 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}
// Instruction descriptor: fp32 accumulator, bf16 A and B, both K-major, M = m (128, or 256 for a CTA
// pair), N = n.
__device__ __forceinline__ uint32_t instr_desc_bf16(int m, int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

// The map whose box holds exactly n_rows activation rows (n_rows a multiple of the quantum the maps
// were encoded with: 16 rows up to 256 for the one-CTA kernel, 8 rows up to 128 for each CTA of a pair).
// One copy per ring slot and operand: every TMA copy has a fixed cost in the copy engine that is
// comparable to moving several KiB, so a token tile is never assembled from smaller boxes.
// OR of `flag` over the 128 epilogue threads (named barrier 1), so that they leave their loop together.
__device__ __forceinline__ bool epilogue_any(bool flag) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 q, %1, 0;\n\t"
        "bar.red.or.pred p, 1, 128, q;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(r)
        : "r"((uint32_t)flag)
        : "memory");
    return r != 0;
}
template <int kQuantum, int kMaps>
__device__ __forceinline__ const CUtensorMap *act_map(const TensorMapsOf<kMaps> &maps, int n_rows) {
    return &maps.act[n_rows / kQuantum - 1];
}

struct Tile {
    int e, f, row0, n_valid;
    int n_tok_tiles;  // token tiles of this tile's expert
};
// Tile order: experts in schedule order (most rows first), then weight slab, then the expert's token
// tiles (fastest), so tiles that share a weight slab run at the same time on neighbouring CTAs.
__device__ __forceinline__ Tile decode_tile(int tile, const KernelParams &p) {
    int lo = 0, hi = p.E;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (p.tile_prefix[mid] * p.n_feature_tiles <= tile) lo = mid; else hi = mid;
    }
    Tile t;
    t.e = p.tile_order[lo];
    const int first = p.tile_prefix[lo], n_tok_tiles = p.tile_prefix[lo + 1] - first;
    const int local = tile - first * p.n_feature_tiles;
    t.f = local / n_tok_tiles;
    const int j = local - t.f * n_tok_tiles;
    const int rows = p.tile_rows[t.e];
    const int begin = p.expert_offsets[t.e], count = p.expert_offsets[t.e + 1] - begin;
    t.row0 = begin + j * rows;
    t.n_valid = min(rows, count - j * rows);
    t.n_tok_tiles = n_tok_tiles;
    return t;
}

// Static tile assignment: worker w of n_workers takes, in round i, tile i*n_workers + w on even rounds
// and i*n_workers + (n_workers-1-w) on odd rounds.  With tiles ordered by decreasing cost this
// back-and-forth deal keeps every worker's total within about 1 % of the mean, without atomics.
__device__ __forceinline__ int tile_of_round(int round, int worker, int n_workers) {
    return round * n_workers + ((round & 1) ? n_workers - 1 - worker : worker);
}

// ---- tiles decoded ahead ---------------------------------------------------------------------------------------------
// The walk from a tile number to its expert, slab and rows is a chain of dependent loads (a binary search over the experts'
// tile counts, then the expert's entries): beside the operand streams 5000-6000 cycles, in front of every tile of every role,
// more than a ring of six or seven slots hides where a tile has few slots.  So one warp decodes the CTA's tiles in order, a
// few ahead, and the others take them from a small queue.  4096 tokens of 32 experts of 1024 x
// 1024, top 4: bf16 139.1 -> 134, MX 167.2 -> 155; 256 of them 60.3 -> 58.8 and 51.9 -> 48.9.
//   kDepth entries of eight words, then full[kDepth] (the decoder's arrival) and empty[kDepth] (one per taking warp)
// Tiles are handed out on demand where a tile is at least two rings of slots: with a static assignment the CTAs of the down GEMM
// of 128 DeepSeek-V3-shaped tokens ended between 2993 and 3177 us of the call, whatever ran slower waited for by everything
// behind it.  Where tiles are shorter the next one is wanted before it could be drawn (200 tokens of 32 experts of 1024 x 1024, top 4,
// sixteen slots: 53.8 decoded ahead, 54.8 us on demand).
enum { kNoQueue = 0, kStaticQueue = 1, kBatchedQueue = 2, kOnDemand = 3 };
inline bool tiles_on_demand(int slots_per_tile, int ring) { return slots_per_tile >= 2 * ring && slots_per_tile >= 20; }
inline int static_queue(int slots_per_tile, bool many) { return slots_per_tile <= 4 && many ? kBatchedQueue : kStaticQueue; }
struct TileQueue {
    static constexpr int kDepth = 4, kBytes = kDepth * 32 + 2 * kDepth * 8;
    int *entries;
    uint32_t full, empty;
    __device__ __forceinline__ TileQueue(uint8_t *base_ptr, uint32_t base, int offset)
        : entries(reinterpret_cast<int *>(base_ptr + offset)), full(base + offset + kDepth * 32), empty(full + kDepth * 8) {}
    __device__ __forceinline__ void init(int takers) const {  // by one thread
        for (int i = 0; i < kDepth; ++i) {
            mbar_init(full + i * 8, 1);
            mbar_init(empty + i * 8, takers);
        }
    }
    // The CTA's n-th tile, by a whole warp; false if the CTA is aborting.  wait(bar, parity): a bounded wait.
    template <typename T, typename Wait>
    __device__ __forceinline__ bool take(T &t, int n, int lane, Wait wait) const {
        const int i = n & (kDepth - 1);
        const bool ok = __all_sync(0xffffffffu, wait(full + i * 8, (n / kDepth) & 1));
        int *w = reinterpret_cast<int *>(&t);
        const volatile int *e = entries + i * 8;
#pragma unroll
        for (int k = 0; k < (int)(sizeof(T) / 4); ++k) w[k] = e[k];
        __syncwarp();
        if (lane == 0) mbar_arrive(empty + i * 8);
        return ok;
    }
    template <typename T>
    __device__ __forceinline__ void publish(const T &t, int n, int lane) const {
        static_assert(sizeof(T) <= 32, "an entry");
        const int i = n & (kDepth - 1);
        if (lane == 0) {
            const int *w = reinterpret_cast<const int *>(&t);
            volatile int *e = entries + i * 8;
#pragma unroll
            for (int k = 0; k < (int)(sizeof(T) / 4); ++k) e[k] = w[k];
            mbar_arrive(full + i * 8);
        }
        __syncwarp();
    }
    // The decoder warp, static assignment: the tiles of this worker from its n-th on, up to kDepth ahead.  Returns their end.
    template <typename Decode, typename Wait>
    __device__ __forceinline__ int fill(int worker, int n_workers, int total_tiles, int lane, Decode decode, Wait wait, int n = 0) const {
        for (;; ++n) {
            const int tile = tile_of_round(n, worker, n_workers);
            if (tile >= total_tiles) break;
            const auto t = decode(tile);
            if (!__all_sync(0xffffffffu, wait(empty + (n & (kDepth - 1)) * 8, ((n / kDepth) & 1) ^ 1))) break;
            publish(t, n, lane);
        }
        return n;
    }
    // The same for tiles of very few slots, which one walk after the other holds up: after the first, 32 tiles at a time are
    // decoded, one per lane.
    template <typename T, typename Decode, typename Wait>
    __device__ __forceinline__ void fill_batched(int worker, int n_workers, int total_tiles, int lane, Decode decode, Wait wait) const {
        T batch;
        for (int n = 0;; ++n) {
            if (tile_of_round(n, worker, n_workers) >= total_tiles) break;
            T t;
            if (n == 0) {
                t = decode(worker);
            } else {
                if ((n & 31) == 1) {
                    const int tile = tile_of_round(n + lane, worker, n_workers);
                    if (tile < total_tiles) batch = decode(tile);
                    __syncwarp();
                }
                int *w = reinterpret_cast<int *>(&t);
                const int *mine = reinterpret_cast<const int *>(&batch);
#pragma unroll
                for (int k = 0; k < (int)(sizeof(T) / 4); ++k) w[k] = __shfl_sync(0xffffffffu, mine[k], (n - 1) & 31);
            }
            if (!__all_sync(0xffffffffu, wait(empty + (n & (kDepth - 1)) * 8, ((n / kDepth) & 1) ^ 1))) break;
            publish(t, n, lane);
        }
    }
    // The decoder warp, tiles on demand: the worker's own number first, then whatever the call's counter says; the next one is drawn
    // when the last role (the epilogue) has begun with the one before it.  An entry whose expert is -1 ends the work.
    template <typename T, typename Decode, typename Wait>
    __device__ __forceinline__ void fill_on_demand(int worker, int n_workers, int total_tiles, int *counter, int lane, Decode decode,
                                                   Wait wait) const {
        for (int n = 0;; ++n) {
            int tile = worker;
            if (n > 0) {
                const int m = n - 1;
                if (!__all_sync(0xffffffffu, wait(empty + (m & (kDepth - 1)) * 8, (m / kDepth) & 1))) break;
                if (lane == 0) tile = n_workers + atomicAdd(counter, 1);
                tile = __shfl_sync(0xffffffffu, tile, 0);
            }
            T t;
            t.e = -1;
            if (tile < total_tiles) t = decode(tile);
            publish(t, n, lane);
            if (t.e < 0) break;
        }
    }
};

// ---- hand-over between the gate/up and the down GEMM of one call -------------------------------------------
// Bounded poll of an int in global memory until it reaches `target` (acquire); on expiry the CTA aborts as for an
// expired barrier wait.
__device__ __forceinline__ bool poll_at_least(const int *addr, int target, volatile int *abort_flag, int *status, int site,
                                              long long limit_cycles = kWaitLimitCycles) {
    const long long start = clock64();
    while (true) {
        int v;
        asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(addr) : "memory");
        if (v >= target) return true;
        if (*abort_flag) return false;
        if (clock64() - start > limit_cycles) {
            *abort_flag = 1;
            if (atomicCAS(status, 0, (int)MOE_ERR_DEVICE_TIMEOUT) == 0) {
                status[1] = site;
                status[2] = blockIdx.x;
            }
            return false;
        }
        __nanosleep(200);
    }
}
// Start of a GEMM kernel's work, after its prologue.  The two GEMMs of a hand-over pair (roles 1 and 2) do not wait for the
// grids before them: they wait for the flag the router raises once the tile schedule is complete, and fetch weights from
// then on; only their token side waits for more (handover_wait_expert).  Every other kernel waits for its predecessors.
__device__ __forceinline__ bool gemm_chain_start(int role, int *handover, volatile int *abort_flag, int *status) {
    if (role != 0) {
        bool ok = true;
        if (threadIdx.x == 0) ok = poll_at_least(handover + kHandoverFlagInt, 1, abort_flag, status, kSiteHandoverFlag);
        __syncthreads();
        return !*abort_flag && ok;
    }
    chain_wait();
    return true;
}
// End of a GEMM kernel's work, before its teardown.  A grid of a hand-over pair never waited for the grid before it, only
// for flags and counts; it waits here (that grid is finished or finishing by now, so this costs nothing), so that "this grid
// is complete" again implies "everything before it in the stream is complete" for whatever follows.
__device__ __forceinline__ void gemm_chain_finish(int role) {
    if (role != 0) chain_wait();
}
// Role 1, called by every epilogue warp after it has stored its part of a tile: the stores of all its lanes are
// made visible, then the expert's count goes up by one.
__device__ __forceinline__ void handover_count_tile(int role, int *handover, int expert, int lane) {
    if (role != 1) return;
    __threadfence();
    __syncwarp();
    if (lane == 0) {
        atomicAdd(handover + kReadyCounterInt + expert, 1);
        atomicAdd(handover + kReadyTotalInt, 1);
    }
}
// Called by the token-side producer warp before the first load of a tile.  Role 1: its token rows are complete with the grid
// before this one.  Role 2: all gate/up tiles of the expert must have been counted; then generic-proxy writes become visible
// to the TMA loads that follow.
// Once everything has been seen complete (`all_done`, kept by the caller across tiles) nothing is
// read any more: a load from global memory in front of every tile would starve the ring of a memory-bound GEMM.
// (whole warp: lane 0 reads, every lane fences, the result is uniform)
__device__ __forceinline__ bool handover_wait_expert(int role, int *handover, int expert, int n_tok_tiles, int per_token_tile,
                                                     int total_token_tiles, bool &all_done, volatile int *abort_flag,
                                                     int *status, int lane) {
    if (role == 0 || all_done) return true;
    if (role == 1) {
        chain_wait();
        all_done = true;
        asm volatile("fence.proxy.async;" ::: "memory");
        return true;
    }
    bool ok = true, done = false;
    if (lane == 0) {
        int total;
        asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(total) : "l"(handover + kReadyTotalInt) : "memory");
        done = total >= total_token_tiles * per_token_tile;
        if (!done)
            ok = poll_at_least(handover + kReadyCounterInt + expert, n_tok_tiles * per_token_tile, abort_flag, status,
                               kSiteHandoverCount);
    }
    ok = __all_sync(0xffffffffu, ok);
    all_done = __any_sync(0xffffffffu, done);
    asm volatile("fence.proxy.async;" ::: "memory");
    return ok;
}

// Clock probe: block 0 of a GEMM grid leaves its SM cycle counter and the global nanosecond timer, at the start of its
// work and at its end, in the call's status region (kClockProbeInt, 4 x int64 per GEMM: cycles begin / end, ns begin /
// end).  Their quotient is the clock the SM really ran at during THAT kernel, which a benchmark needs to tell a slow
// kernel from a power-capped GPU; two stores per block-0 thread-0, nothing else.
__device__ __forceinline__ void clock_probe_begin(int *status, int which) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        long long *slot = reinterpret_cast<long long *>(status + kClockProbeInt) + 4 * which;
        unsigned long long ns;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(ns));
        slot[0] = clock64();
        slot[2] = (long long)ns;
    }
}
__device__ __forceinline__ void clock_probe_end(int *status, int which) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        long long *slot = reinterpret_cast<long long *>(status + kClockProbeInt) + 4 * which;
        unsigned long long ns;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(ns));
        slot[1] = clock64();
        slot[3] = (long long)ns;
    }
}

// SiLU(g) * u with the fast exponential; exp overflow gives g / inf = -0 for very negative g.
__device__ __forceinline__ float swiglu(float g, float u) { return __fdividef(g, 1.f + __expf(-g)) * u; }

// ---- epilogue: 16 accumulator columns of a warp's 32 rows to global memory ---------------------------------------
// Every value is computed before the first store, and the stores of whole groups carry no condition.  With "compute and store
// if the column exists" per value, each of the eight or sixteen became a branch of its own with the whole chain (exponential,
// reciprocal, products, conversion) inside it, one after the other: 2000 cycles per group of a gate/up tile, 30 000 per
// 256-row tile, more than its MMAs take for K of up to 4096.  Layers of 32 experts of
// 1024 x 1024, top 4, 4096 tokens: bf16 180 -> 140 us, MX 227 -> 177, FP8 weights 210 -> 143; 8 experts of 256 x 512, 1024
// tokens 43.0 -> 36.8; Mixtral-shaped in MX, 1024 tokens 436 -> 370; 4096 tokens of 128 experts of 4096 x 1536 in MX 812 -> 732.
//
// Gate/up: lanes 0..15 hold gate, lanes 16..31 up of the same 16 features; each half-warp finishes eight columns.
__device__ __forceinline__ void swiglu_16(const float (&v)[16], int lane, float (&h)[8]) {
    const bool hi = (lane & 16) != 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const float other = __shfl_xor_sync(0xffffffffu, hi ? v[i] : v[8 + i], 16);
        h[i] = swiglu(hi ? other : v[i], hi ? v[8 + i] : other);
    }
}
// n values, one per row of `stride` elements from `dst` on; of rows that exist (`left` of them, which may be 0 or less).
template <int N>
__device__ __forceinline__ void store_column(const float (&v)[N], int left, __nv_bfloat16 *dst, size_t stride) {
    __nv_bfloat16 b[N];
#pragma unroll
    for (int i = 0; i < N; ++i) b[i] = __float2bfloat16_rn(v[i]);
    if (left >= N) {
#pragma unroll
        for (int i = 0; i < N; ++i) dst[(size_t)i * stride] = b[i];
    } else {
#pragma unroll
        for (int i = 0; i < N; ++i)
            if (i < left) dst[(size_t)i * stride] = b[i];
    }
}
// A warp's rows of one tile: n_mma columns from taddr on, n_valid of which are rows of the result (dst: this lane's feature
// in the first).
template <bool SWIGLU>
__device__ __forceinline__ void drain_accumulator(uint32_t taddr, int n_mma, int n_valid, __nv_bfloat16 *dst, size_t stride, int lane) {
    for (int c0 = 0; c0 < n_mma; c0 += 16) {
        float v[16];
        tmem_load_16(taddr + c0, v);
        if (SWIGLU) {
            float h[8];
            swiglu_16(v, lane, h);
            const int first = c0 + ((lane & 16) >> 1);
            store_column(h, n_valid - first, dst + (size_t)first * stride, stride);
        } else {
            store_column(v, n_valid - c0, dst + (size_t)c0 * stride, stride);
        }
    }
}

// ---- the same through shared memory -------------------------------------------------------------------------------
// Stored from its registers, a warp's 32 rows of the accumulator are 64 bytes (gate/up: 32) of each token's row, two bytes
// per lane, and every such piece costs the load/store unit about 18 cycles beside the operand copies: 1200 cycles per group
// of 16 columns, whatever was computed.  Here the four warps of a CTA transpose a step of columns through shared memory and
// store whole rows, 16 bytes per lane: 128 features of the down projection are 256 bytes, 64 of h are 128.  Two buffers and
// one barrier of the 128 threads per step: a step's writes cannot pass the barrier of the step before it.  4096 tokens of 32 experts
// of 1024 x 1024, top 4: bf16 141.9 -> 139.1 us, MX 176.7 -> 167.2; 1024 tokens 75.8 -> 72.8 and 71.2 -> 68.9.
// Where the buffers cost a ring slot, kernels with K of 4096 and more store directly: their slots hide the epilogue, and
// want the depth (direct / staged: 512 Mixtral-shaped tokens 498 / 516 us, MX prefill on 32 of 256 experts of 7168 x 2048
// 477 / 496; staged wins at K = 2048, 2000 tokens of 64 MX experts, top 4, 234 / 231, and below).
constexpr int kDirectFromK = 4096;
__device__ __forceinline__ void epilogue_sync() { asm volatile("bar.sync 4, 128;" ::: "memory"); }
template <bool SWIGLU>
struct Stage {
    static constexpr int kGroups = SWIGLU ? 2 : 1;                 // of 16 tokens, per step
    static constexpr int kRowBytes = SWIGLU ? kTileM : 2 * kTileM;  // a token's features of this CTA, bf16
    // Byte `byte` of a token's row.  Gate/up: 16-byte pieces are swizzled, since the half-warps write eight rows apart.
    __device__ static int at(int token, int byte) {
        return token * kRowBytes + (SWIGLU ? byte ^ (((token & 7) ^ ((token >> 1) & 4)) << 4) : byte);
    }
    static constexpr int kBufferBytes = kGroups * 16 * kRowBytes;
    static constexpr int kBytes = 2 * kBufferBytes;
};
constexpr int kStageBytes = Stage<true>::kBytes;
static_assert(Stage<true>::kBytes == Stage<false>::kBytes, "either GEMM's buffers");
// One step: kGroups x 16 columns of this warp's 32 rows.  row_of(token): where this CTA's features of the step's token go in
// the result, or null if there is no such row.
template <bool SWIGLU, typename RowOf>
__device__ __forceinline__ void store_staged(const float (&v)[Stage<SWIGLU>::kGroups][16], uint8_t *stage, int &flip, RowOf row_of,
                                             int q, int lane) {
    using S = Stage<SWIGLU>;
    flip ^= 1;
    uint8_t *buf = stage + flip * S::kBufferBytes;
    if constexpr (SWIGLU) {
        float h[S::kGroups][8];
#pragma unroll
        for (int g = 0; g < S::kGroups; ++g) swiglu_16(v[g], lane, h[g]);
#pragma unroll
        for (int g = 0; g < S::kGroups; ++g)
#pragma unroll
            for (int i = 0; i < 8; ++i)
                *reinterpret_cast<__nv_bfloat16 *>(buf + S::at(g * 16 + ((lane & 16) >> 1) + i, (q * 16 + (lane & 15)) * 2)) = __float2bfloat16_rn(h[g][i]);
    } else {
#pragma unroll
        for (int i = 0; i < 16; ++i)
            *reinterpret_cast<__nv_bfloat16 *>(buf + S::at(i, (q * 32 + lane) * 2)) = __float2bfloat16_rn(v[0][i]);
    }
    epilogue_sync();
    constexpr int kLanes = S::kRowBytes / 16, kRows = 32 / kLanes;  // lanes per row, rows per warp instruction
#pragma unroll
    for (int it = 0; it < S::kGroups * 16 / 4 / kRows; ++it) {
        const int token = q * (S::kGroups * 4) + it * kRows + lane / kLanes;
        const uint4 val = *reinterpret_cast<const uint4 *>(buf + S::at(token, (lane % kLanes) * 16));
        __nv_bfloat16 *row = row_of(token);
        if (row) *reinterpret_cast<uint4 *>(row + (lane % kLanes) * 8) = val;
    }
}
// A tile: n_mma columns from taddr on, n_valid of which are rows of the result (dst: this CTA's first feature in the first).
template <bool SWIGLU>
__device__ __forceinline__ void drain_staged(uint32_t taddr, int n_mma, int n_valid, __nv_bfloat16 *dst, size_t stride, uint8_t *stage,
                                             int &flip, int q, int lane) {
    constexpr int kStep = Stage<SWIGLU>::kGroups * 16;
    for (int c0 = 0; c0 < n_mma; c0 += kStep) {
        float v[Stage<SWIGLU>::kGroups][16];
        if constexpr (SWIGLU) {
            if (c0 + 32 <= n_mma) {
                tmem_load_2x16(taddr + c0, v);
            } else {
                tmem_load_16(taddr + c0, v[0]);
#pragma unroll
                for (int i = 0; i < 16; ++i) v[1][i] = 0.f;
            }
        } else {
            tmem_load_16(taddr + c0, v[0]);
        }
        store_staged<SWIGLU>(v, stage, flip, [&](int token) -> __nv_bfloat16 * {
            return c0 + token < n_valid ? dst + (size_t)(c0 + token) * stride : nullptr;
        }, q, lane);
    }
}

// ---- host side ----------------------------------------------------------------------------------
bool encode_weight_map_2d(CUtensorMap *map, const void *w, uint64_t rows, uint64_t K);
bool encode_map_chunks(CUtensorMap *map, const void *base, uint64_t rows, uint64_t K, int box_rows, int chunks);
bool encode_weight_map_gate_up(CUtensorMap *map, const void *w13, int E, int I, int H);
bool encode_act_maps_chunks(CUtensorMap *maps, const void *act, uint64_t rows, uint64_t K, int row_quantum, int chunks, int count);
bool encode_act_maps(CUtensorMap *maps, const void *act, uint64_t rows, uint64_t K, int row_quantum, int count);
bool encode_row_map(CUtensorMap *map, const void *act, uint64_t rows, uint64_t K);
bool encode_mx_weight_map_2d(CUtensorMap *map, const void *w, uint64_t rows, uint64_t K);
bool encode_mx_weight_map_gate_up(CUtensorMap *map, const void *w13, int E, int I, int H);
bool encode_mx_act_maps(CUtensorMap *maps, const void *act, uint64_t rows, uint64_t K, int row_quantum, int count);
int sm_count();
bool set_max_dynamic_smem_once(const void *kernel, int bytes);

}  // namespace tc
}  // namespace moe
