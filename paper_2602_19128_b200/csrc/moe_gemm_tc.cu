// Grouped expert GEMMs on the Blackwell tensor cores: tcgen05.mma with TMEM accumulators, operands
// staged in shared memory by TMA, warp-specialised and persistent.
//
// Paper, Sec. 4.5 "Expert FFN computation": after the sort-scatter every expert's tokens are
// contiguous; the gate and up projections are computed together and combined through SiLU, the
// down projection follows; experts without tokens are skipped.  The paper's kernel used 16x16
// WMMA tiles with double buffering.  Here:
//
//  * The weights sit on the MMA's M side (128 weight rows per tile, the hardware's full-rate
//    shape) and the tokens on its N side, so a token tile can have any multiple of 16 rows up
//    to NT_MAX.  An expert with 4 tokens costs one N=16 instruction per 128x16 weight slab
//    instead of a mostly empty 128-row token tile, and every weight byte is fetched once per
//    token tile.  D[128, N] = W_tile[128, K] * X_tile[N, K]^T, both operands K-major.
//  * gemm1 interleaves gate and up rows inside one 128-row A tile in groups of 16
//    (rows 32q..32q+15 = gate features, 32q+16..32q+31 = the matching up features), so each
//    epilogue warp finds gate and up of the same 16 features in its own 32 TMEM lanes and
//    pairs them with one shuffle; SiLU(gate)*up is applied before anything is stored.
//  * One CTA per SM walks tiles  tile = blockIdx.x + i*gridDim.x  of a device-built schedule
//    (no host round trip; long tiles are drawn from a counter, TileQueue).  Tiles of the same expert and weight slab are adjacent in
//    that order, so they run at the same time on neighbouring SMs and share the slab in L2.
//  * Warp 0 issues TMA loads into a STAGES-deep ring; warp 1 issues the MMAs and commits ring
//    slots back; warps 2..5 drain the accumulator (double-buffered in TMEM, so the epilogue of
//    one tile overlaps the MMAs of the next).
//  * A down GEMM with fewer tiles than half of the SMs (a token or two on a few experts) has two CTAs on each tile, 64 of its
//    128 weight rows each (HALVES): an SM takes in about 100 GB/s, so 32 or 64 of them do not reach the memory's rate.  Every
//    sum runs over K as it does with one CTA per tile, so the results are the same bit for bit.  The MMA has 64 rows (with
//    128, half of them unused, its reads of shared memory took as long as the stream), token rows come in eights, and
//    a slot holds four 64-wide K chunks, each operand one copy: with one chunk per slot the handling of a slot took as long
//    as its 8 KiB.  One Mixtral-shaped token 134.1 -> 126.5 us (128 rows and one chunk 137.0, two chunks 131.6; 64 rows and
//    two chunks 129.3, three 126.3), the same on one expert 90.8 -> 80.7, 16 tokens of 8 experts of 512 x 4096, top 2, 45.7 ->
//    38.0, one token of 1024 x 2048 25.6 -> 23.1.
//  * Every wait is bounded: if one expires the CTA records MOE_ERR_DEVICE_TIMEOUT and the site in
//    the status word, every role stops, TMEM is released and the kernel returns.
#include "moe_tc_common.cuh"

namespace moe {
namespace {

using namespace tc;

// D[tmem] (+)= A[smem] * B[smem]^T, bf16 inputs, fp32 accumulate, issued by one thread.
__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                          uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// Arrive on an mbarrier once all MMAs issued so far by this thread have completed.
__device__ __forceinline__ void umma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

constexpr int kHalfChunks = 4, kHalfStages = 4;  // HALVES: 64-wide K chunks per slot, slots

// Tiles of more than 32 rows are stored through shared memory (Stage); a smaller tile is one or two groups of columns, whose
// stores do not show.
template <int NT_MAX, int STAGES, bool HALVES>
struct SmemLayout {
    static constexpr bool kStaged = NT_MAX > 32;
    static constexpr int kRows = HALVES ? kTileM / 2 : kTileM;    // weight rows of this CTA's part of a tile
    static constexpr int kChunks = HALVES ? kHalfChunks : 1;  // 64-wide K chunks per slot: weights [chunk][rows], tokens [chunk][n_mma rows]
    static constexpr int kSlotABytes = kChunks * kRows * kRowBytes;
    static constexpr int kSlotBBytes = kChunks * NT_MAX * kRowBytes;
    static constexpr int kA = 0;
    static constexpr int kB = STAGES * kSlotABytes;
    static constexpr int kStage = kB + STAGES * kSlotBBytes;
    // full[STAGES], empty[STAGES], acc_full[2], acc_empty[2]
    static constexpr int kBars = kStage + (kStaged ? kStageBytes : 0);
    static constexpr int kTmemSlot = kBars + (2 * STAGES + 4) * 8;
    static constexpr int kAbort = kTmemSlot + 4;
    static constexpr int kTiles = (kAbort + 4 + 15) / 16 * 16;  // TileQueue
    static constexpr int kBytes = kTiles + TileQueue::kBytes;
    static constexpr int kDynamicBytes = kBytes + 1024;  // slack to align the base to 1024 bytes
    static constexpr int kQuantum = HALVES ? 8 : 16;     // token rows come in multiples of it: the MMA's step in N for so many rows
    using Maps = TensorMapsOf<NT_MAX / kQuantum>;
};

template <int NT_MAX, int STAGES, bool SWIGLU, bool HALVES, int QUEUE>
__global__ void __launch_bounds__(QUEUE != kNoQueue ? kThreads + 32 : kThreads, 1)
grouped_gemm_tc_kernel(const __grid_constant__ typename SmemLayout<NT_MAX, STAGES, HALVES>::Maps maps, const KernelParams p) {
    using L = SmemLayout<NT_MAX, STAGES, HALVES>;
    static_assert(!HALVES || (!SWIGLU && !L::kStaged), "the halves of a tile are stored row by row");
    constexpr int kRows = L::kRows;
    constexpr int kQuantum = L::kQuantum;
    constexpr int kTmemCols = 2 * NT_MAX;
    static_assert(kTmemCols >= 32 && kTmemCols <= 512 && (kTmemCols & (kTmemCols - 1)) == 0,
                  "a tensor-memory allocation must be a power of two between 32 and 512 columns");
    constexpr int kSiteOffset = SWIGLU ? 0 : 4;  // the down GEMM reports sites 5..8
    chain_release();  // the next kernel of the forward call may be scheduled; it waits for what it needs of this grid
    extern __shared__ uint8_t smem_raw[];
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *base_ptr = smem_raw + (base - smem_u32(smem_raw));
    const uint32_t bar_full = base + L::kBars, bar_empty = bar_full + STAGES * 8;
    const uint32_t bar_acc_full = bar_empty + STAGES * 8, bar_acc_empty = bar_acc_full + 16;
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(base_ptr + L::kTmemSlot);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(base_ptr + L::kAbort);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    auto wait = [&](uint32_t bar, uint32_t parity, int site) {
        return mbar_wait(bar, parity, abort_flag, p.status, site + kSiteOffset);
    };
    const TileQueue tiles(base_ptr, base, L::kTiles);
    auto decode = [&](int tile) { return decode_tile(tile, p); };
    auto queue_wait = [&](uint32_t bar, uint32_t parity) { return wait(bar, parity, kSiteProducerEmpty); };
    // the n-th tile, from the decoder warp or decoded here; false at the end of the work
    auto next_tile = [&](Tile &t, int n, int tile) {
        if constexpr (QUEUE != kNoQueue) return tiles.take(t, n, lane, queue_wait) && (QUEUE != kOnDemand || t.e >= 0);
        t = decode(tile);
        return true;
    };
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(bar_full + s * 8, 1);
            mbar_init(bar_empty + s * 8, 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(bar_acc_full + a * 8, 1);
            mbar_init(bar_acc_empty + a * 8, kEpilogueWarps);
        }
        tiles.init(2 + kEpilogueWarps);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 0 && lane == 0) {
        prefetch_map(&maps.w);
        prefetch_map(&maps.act[0]);
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(base + L::kTmemSlot),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tcgen05_fence_before();
    __syncthreads();
    tcgen05_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    // everything above overlapped the kernels in front; from here on there is a schedule (the token side waits for more)
    const bool started = gemm_chain_start(p.handover_role, p.handover, abort_flag, p.status);
    const int total_tiles = started ? p.tile_prefix[p.E] * p.n_feature_tiles : 0;
    const int worker = HALVES ? blockIdx.x >> 1 : blockIdx.x, n_workers = HALVES ? gridDim.x >> 1 : gridDim.x;
    const int row_half = HALVES ? blockIdx.x & 1 : 0;  // which 64 of a tile's rows are this CTA's
    const int n_slots = HALVES ? (p.n_k_blocks + L::kChunks - 1) / L::kChunks : p.n_k_blocks;

    if (warp == 0) {
        // ---------------- TMA producer: one elected thread issues a whole tile's copies ----------------
        int stage = 0;
        uint32_t phase = 0;
        bool ok = true, gate_up_done = false;
        auto load_weights = [&](const Tile &t, int w_row, int kb, int slot) {  // by one thread
            const uint32_t sa = base + L::kA + slot * L::kSlotABytes, full = bar_full + slot * 8;
            if (SWIGLU)  // 64 features = groups 4f..4f+3 of 16, gate and up rows interleaved per group
                tma_load_5d(sa, &maps.w, kb * kBlockK, 0, 0, t.f * 4, t.e, full);
            else
                HALVES ? tma_load_3d(sa, &maps.w, 0, w_row, L::kChunks * kb, full) : tma_load_2d(sa, &maps.w, kb * kBlockK, w_row, full);
        };
        for (int round = 0; ok; ++round) {
            const int tile = tile_of_round(round, worker, n_workers);
            if (QUEUE != kOnDemand && tile >= total_tiles) break;
            Tile t;
            ok = next_tile(t, round, tile);
            if (!ok) break;
            const int n_mma = (t.n_valid + kQuantum - 1) & -kQuantum;
            const int w_row = t.e * p.w_rows + t.f * kTileM + row_half * kRows;  // down projection: 128 rows of w2[e], or 64
            const uint32_t tx_bytes = L::kSlotABytes + L::kChunks * n_mma * kRowBytes;
            // The first tile's weights do not wait for its token rows: the ring's slots are filled with them beforehand (a
            // one-token Mixtral-shaped layer streams weights while the rows are scattered, and while the last gate/up tiles run).
            int filled = 0;
            if (round == 0 && p.handover_role != 0) {
                filled = n_slots < STAGES ? n_slots : STAGES;
                if (elect_one())
                    for (int kb = 0; kb < filled; ++kb) {
                        mbar_expect_tx(bar_full + kb * 8, tx_bytes);
                        load_weights(t, w_row, kb, kb);
                    }
                __syncwarp();
            }
            ok = handover_wait_expert(p.handover_role, p.handover, t.e, t.n_tok_tiles, p.handover_per_token_tile,
                                      p.tile_prefix[p.E], gate_up_done, abort_flag, p.status, lane);
            if (!ok) break;
            if (elect_one()) {
                int slot = stage;
                uint32_t ph = phase;
                for (int kb = 0; kb < n_slots; ++kb) {
                    if (kb >= filled) {
                        ok = wait(bar_empty + slot * 8, ph ^ 1u, kSiteProducerEmpty);
                        if (!ok) break;
                        mbar_expect_tx(bar_full + slot * 8, tx_bytes);
                        load_weights(t, w_row, kb, slot);
                    }
                    if (HALVES)
                        tma_load_3d(base + L::kB + slot * L::kSlotBBytes, act_map<kQuantum>(maps, n_mma), 0, t.row0, L::kChunks * kb, bar_full + slot * 8);
                    else
                        tma_load_2d(base + L::kB + slot * L::kSlotBBytes, act_map<kQuantum>(maps, n_mma), kb * kBlockK, t.row0, bar_full + slot * 8);
                    if (++slot == STAGES) { slot = 0; ph ^= 1u; }
                }
            }
            __syncwarp();
            ok = __all_sync(0xffffffffu, ok);
            ring_advance<STAGES>(stage, phase, n_slots);
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer: one elected thread walks a whole tile's slots ----------------
        // (With the election, the vote and the warp barrier in the K loop a slot took longer to issue than a weight slot
        // takes to arrive: 160 -> 137 us on a one-token Mixtral-shaped layer.)
        int stage = 0, acc = 0;
        uint32_t phase = 0, acc_phase = 0;
        bool ok = true;
        for (int round = 0; ok; ++round) {
            const int tile = tile_of_round(round, worker, n_workers);
            if (QUEUE != kOnDemand && tile >= total_tiles) break;
            Tile t;
            ok = next_tile(t, round, tile);
            if (!ok) break;
            const int n_mma = (t.n_valid + kQuantum - 1) & -kQuantum;
            const uint32_t idesc = instr_desc_bf16(kRows, n_mma);
            ok = __all_sync(0xffffffffu, wait(bar_acc_empty + acc * 8, acc_phase ^ 1u, kSiteMmaTmemEmpty));
            if (!ok) break;
            tcgen05_fence_after();
            const uint32_t d_tmem = tmem_base + acc * NT_MAX;
            if (elect_one()) {
                int s = stage;
                uint32_t ph = phase;
                for (int kb = 0; kb < n_slots; ++kb) {
                    ok = wait(bar_full + s * 8, ph, kSiteMmaFull);
                    if (!ok) break;
                    tcgen05_fence_after();
                    const uint64_t a_desc = smem_desc_k_major_sw128(base + L::kA + s * L::kSlotABytes);
                    const uint64_t b_desc = smem_desc_k_major_sw128(base + L::kB + s * L::kSlotBBytes);
#pragma unroll
                    for (int j = 0; j < L::kChunks; ++j) {
                        if (j && L::kChunks * kb + j == p.n_k_blocks) break;  // (the last slot may have fewer)
#pragma unroll
                        for (int kk = 0; kk < kBlockK / 16; ++kk)  // 16 K-elements = 32 bytes = 2 descriptor units
                            umma_bf16(d_tmem, a_desc + (uint32_t)(j * (kRows * kRowBytes >> 4)) + 2 * kk,
                                      b_desc + (uint32_t)(j * (n_mma * kRowBytes >> 4)) + 2 * kk, idesc, (kb | j | kk) != 0);
                    }
                    umma_commit(bar_empty + s * 8);
                    if (++s == STAGES) { s = 0; ph ^= 1u; }
                }
                if (ok) umma_commit(bar_acc_full + acc * 8);
            }
            __syncwarp();
            ok = __all_sync(0xffffffffu, ok);
            ring_advance<STAGES>(stage, phase, n_slots);
            if (!ok) break;
            if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
        }
    } else if (warp < 6) {
        // ---------------- epilogue: TMEM -> registers -> global ----------------
        const int q = warp & 3;  // a warp may only read TMEM lanes 32*(warp%4) .. +31
        int acc = 0, flip = 0;
        uint32_t acc_phase = 0;
        bool ok = true;
        for (int round = 0; ok; ++round) {
            const int tile = tile_of_round(round, worker, n_workers);
            if (QUEUE != kOnDemand && tile >= total_tiles) break;
            Tile t;
            const bool taken = next_tile(t, round, tile);  // (at the end of the work the four warps leave as if they gave up: together)
            const int n_mma = (t.n_valid + kQuantum - 1) & -kQuantum;
            ok = taken && wait(bar_acc_full + acc * 8, acc_phase, kSiteEpilogueTmemFull);
            if (L::kStaged ? epilogue_any(!ok) : !__all_sync(0xffffffffu, ok)) break;  // (the four warps meet inside a staged tile)
            tcgen05_fence_after();
            const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + acc * NT_MAX;
            __nv_bfloat16 *rows = p.out + (size_t)t.row0 * p.n_out + t.f * (SWIGLU ? kTileM / 2 : kTileM) + row_half * kRows;  // this CTA's features
            if constexpr (L::kStaged) {
                drain_staged<SWIGLU>(taddr, n_mma, t.n_valid, rows, (size_t)p.n_out, base_ptr + L::kStage, flip, q, lane);
            } else {
                // (the accumulator of an MMA of 64 rows: row 16 q + j in lane 32 q + j, the other lanes unused)
                constexpr int kWarpRows = kRows / 4;
                drain_accumulator<SWIGLU>(taddr, n_mma, lane < kWarpRows ? t.n_valid : 0,
                                          rows + (SWIGLU ? q * 16 + (lane & 15) : q * kWarpRows + lane % kWarpRows), (size_t)p.n_out, lane);
            }
            tcgen05_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_acc_empty + acc * 8);
            handover_count_tile(p.handover_role, p.handover, t.e, lane);  // (after the accumulator is handed back)
            if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
        }
    } else if (QUEUE != kNoQueue && warp == 6) {
        // ---------------- decoder ----------------
        const auto tile_at = decode;
        if constexpr (QUEUE == kOnDemand)
            tiles.fill_on_demand<Tile>(worker, n_workers, total_tiles, p.status + kTileCounterInt + (SWIGLU ? 0 : 1), lane, tile_at, queue_wait);
        else if constexpr (QUEUE == kBatchedQueue)
            tiles.fill_batched<Tile>(worker, n_workers, total_tiles, lane, tile_at, queue_wait);
        else
            tiles.fill(worker, n_workers, total_tiles, lane, tile_at, queue_wait);
    }

    // ---------------- teardown ----------------
    gemm_chain_finish(p.handover_role);
    tcgen05_fence_before();
    __syncthreads();
    if (*abort_flag) {
        // give copies that may still be in flight time to land before the CTA's memory is released
        for (int i = 0; i < 1000; ++i) __nanosleep(1000);
    }
    if (warp == 1) {
        tcgen05_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
    }
}

template <int NT_MAX, int STAGES, bool SWIGLU, bool HALVES = false, int QUEUE = kNoQueue>
int launch_instance(const TensorMaps &maps, const KernelParams &p, int grid, cudaStream_t stream) {
    using L = SmemLayout<NT_MAX, STAGES, HALVES>;
    static_assert(L::kDynamicBytes <= 232448, "ring does not fit in shared memory");
    auto kernel = grouped_gemm_tc_kernel<NT_MAX, STAGES, SWIGLU, HALVES, QUEUE>;
    if (!set_max_dynamic_smem_once(reinterpret_cast<const void *>(kernel), L::kDynamicBytes))
        return MOE_ERR_CUDA;
    return launch_chained(kernel, grid, QUEUE != kNoQueue ? kThreads + 32 : kThreads, L::kDynamicBytes, stream, typename L::Maps(maps), p) == cudaSuccess
               ? MOE_OK : MOE_ERR_CUDA;
}

// How a CTA comes by its tiles.  Where it has more than one: on demand if they are long enough (tiles_on_demand), else decoded ahead
// (kStaticQueue) if a tile's slots do not hide the walk.
// Without a queue / on demand: one token of 128 experts of 4096 x 1536, top 8, 71.9 / 64.3 us; 100 tokens 707 / 697; 64 of 64 of
// 1536 x 1536, top 4, 153.9 / 146.6; 128 of 256 of 7168 x 2048, top 8, 3147 / 3047; Mixtral-shaped, one token, 122.0 / 120.1.
// Without / decoded ahead: 16 tokens of 32 experts of 1024 x 1024, top 4, 51.5 / 50.4; on demand there 45.8 against 45.6 decoded ahead,
// 64 tokens 53.2 / 52.6.  One tile per CTA, the tiny layer: 19.2 without, 19.7 with.
template <int NT_MAX, int STAGES, bool SWIGLU>
int launch_queue(const TensorMaps &maps, const KernelParams &p, int grid, int tiles_per_cta, cudaStream_t s) {
    if (tiles_per_cta <= 1) return launch_instance<NT_MAX, STAGES, SWIGLU>(maps, p, grid, s);
    if (tiles_on_demand(p.n_k_blocks, STAGES)) return launch_instance<NT_MAX, STAGES, SWIGLU, false, kOnDemand>(maps, p, grid, s);
    if (p.n_k_blocks * kBlockK > 1024) return launch_instance<NT_MAX, STAGES, SWIGLU>(maps, p, grid, s);
    return static_queue(p.n_k_blocks, tiles_per_cta >= 8) == kBatchedQueue
               ? launch_instance<NT_MAX, STAGES, SWIGLU, false, kBatchedQueue>(maps, p, grid, s)
               : launch_instance<NT_MAX, STAGES, SWIGLU, false, kStaticQueue>(maps, p, grid, s);
}
template <bool SWIGLU>
int dispatch(int nt_max, const TensorMaps &maps, const KernelParams &p, int grid, int tiles_per_cta, cudaStream_t s) {
    switch (nt_max) {
        case 32: return launch_queue<32, 10, SWIGLU>(maps, p, grid, tiles_per_cta, s);
        case 64: return launch_queue<64, 8, SWIGLU>(maps, p, grid, tiles_per_cta, s);
        case 128: return launch_queue<128, 6, SWIGLU>(maps, p, grid, tiles_per_cta, s);
        case 256: return launch_queue<256, 4, SWIGLU>(maps, p, grid, tiles_per_cta, s);
        default: return MOE_ERR_UNSUPPORTED;
    }
}

__global__ void __launch_bounds__(32)
wait_timeout_selftest_kernel(int *status) {
    __shared__ int abort_flag;
    if (threadIdx.x == 0) abort_flag = 0;
    __syncwarp();
    // the flag was zeroed by the caller's memset and nobody sets it: the poll must give up after its limit
    if (threadIdx.x == 0) poll_at_least(status + kHandoverFlagInt, 1, &abort_flag, status, kSiteSelfTest, 200000000LL);
}

}  // namespace

cudaError_t launch_wait_timeout_selftest(int *status, cudaStream_t stream) {
    cudaError_t err = cudaMemsetAsync(status, 0, kStatusBytesForward, stream);
    if (err != cudaSuccess) return err;
    wait_timeout_selftest_kernel<<<1, 32, 0, stream>>>(status);
    return cudaGetLastError();
}

int launch_grouped_gemm_tc(const GroupedGemmArgs &a, cudaStream_t stream) {
    if (a.K % kBlockK != 0 || a.A <= 0 || a.nt_max > 256) return MOE_ERR_UNSUPPORTED;
    const int features_per_tile = a.swiglu ? kTileM / 2 : kTileM;
    if (a.n_out % features_per_tile != 0) return MOE_ERR_UNSUPPORTED;

    // The tile count is only known on the device; this is its upper bound.
    const long long max_token_tiles = (long long)(a.A < a.E ? a.A : a.E) + a.A / a.nt_max;
    const long long max_tiles = max_token_tiles * (a.n_out / features_per_tile);
    const int sms = sm_count();
    // Two CTAs per tile (HALVES): a down GEMM of small token tiles that leaves half of the SMs or more without a tile, with K long
    // enough that a tile's stream of weights is what takes the time.  One CTA per tile / two: 1 token of 16 experts of 2048 x 2112,
    // top 2, 29.8 / 26.9 us; of 8 of 7168 x 2048, top 1, 42.0 / 42.1; of 8 of 4096 x 1536, top 2, 33.9 / 35.1; 16 tokens of 8 of
    // 1024 x 512, top 2, 22.4 / 23.6.
    const bool halves = !a.swiglu && a.nt_max == 32 && 2 * max_tiles <= sms && a.K >= 2048;

    TensorMaps maps;
    const bool ok_w = halves ? encode_map_chunks(&maps.w, a.w, (uint64_t)a.E * a.w_rows, a.K, kTileM / 2, kHalfChunks)
                    : a.swiglu ? encode_weight_map_gate_up(&maps.w, a.w, a.E, a.n_out, a.K)
                               : encode_weight_map_2d(&maps.w, a.w, (uint64_t)a.E * a.w_rows, a.K);
    if (!ok_w || !(halves ? encode_act_maps_chunks(maps.act, a.act, a.A, a.K, 8, kHalfChunks, a.nt_max / 8)
                        : encode_act_maps(maps.act, a.act, a.A, a.K, 16, a.nt_max / 16))) return MOE_ERR_CUDA;

    KernelParams p;
    p.out = a.out;
    p.expert_offsets = a.expert_offsets;
    p.tile_prefix = a.tile_prefix;
    p.tile_order = a.tile_order;
    p.tile_rows = a.tile_rows;
    p.status = a.status;
    p.E = a.E;
    p.n_k_blocks = a.K / kBlockK;
    p.n_out = a.n_out;
    p.w_rows = a.w_rows;
    p.w_scale = nullptr;
    p.handover_role = a.handover_role;
    p.handover = a.handover;
    p.handover_per_token_tile = a.handover_per_token_tile;
    p.n_feature_tiles = a.n_out / features_per_tile;

    if (halves)
        return launch_instance<32, kHalfStages, false, true>(maps, p, 2 * (int)max_tiles, stream);
    const int grid = (int)(max_tiles < sms ? max_tiles : sms);
    const int tiles_per_cta = (int)((max_tiles + sms - 1) / sms);
    return a.swiglu ? dispatch<true>(a.nt_max, maps, p, grid, tiles_per_cta, stream) : dispatch<false>(a.nt_max, maps, p, grid, tiles_per_cta, stream);
}

}  // namespace moe
