// Grouped expert GEMMs with FP8 (E4M3) block-scaled weights, one CTA per 128 x N tile.
//
// Paper: the workload is an "FP8 MoE" (Table 2; Sec. 4.5) and the paper's kernel feeds 16-bit
// tensor-core tiles, so stored FP8 weights are converted and rescaled on their way to the MMA.  Here
// the weights stay FP8 in HBM (half the bytes of the bf16 layer, which is what bounds the decode- and
// Mixtral-sized workloads) and the conversion happens between shared memory and tensor memory:
//
//   warp 0       weight TMA: per ring slot (128 K-elements = one scale block) the 128 x 128 tile of codes (16 KiB)
//                in the 128-byte swizzle, which a warp reads by rows without bank conflicts
//   warp 6       token TMA: the bf16 token tile of a slot as two 128-byte-swizzled 64-wide chunks, one copy, a ring of
//                its own (weights come from HBM and want a deep ring, tokens from L2)
//   warps 8..    converters: a thread owns one weight row (= its lane of tensor memory), turns 64 of the slot's 128
//                codes into bf16 * block scale and stores them to tensor memory, the MMA's A operand
//   warp 1       MMA: A from tensor memory, B straight from the token slot
//   warps 2..5   epilogue (SwiGLU or plain, two accumulators)
//   warp 7       decodes tiles ahead (QUEUE)
//
// What bounds it and why A sits in tensor memory: with A rebuilt in shared memory a slot of 96 token rows moved 144 KiB
// through shared memory (codes in, codes out, 32 KiB of bf16 in and out again, tokens in and out), 1150 cycles at 128
// bytes per cycle, above the 700 cycles a slot takes at the HBM rate, and the conversion issued 2.5 ALU instructions
// per weight.  Now a slot moves 80 KiB and the conversion is two ALU instructions and one multiply per TWO weights
// (one more for the byte permute).
//
// A weight is decode(code) * scale[row/128][k/128].  A CTA's 128 weight rows lie in one scale block
// (down projection) or in one gate block and one up block (gate/up), and a slot is one 128-wide K
// block, so a slot needs one or two scalar scales.  Conversion: the code's exponent and
// mantissa bits are moved into a bf16 bit pattern worth value * 2^-120, then one bf16x2 multiply by
// scale * 2^120 per pair.  The scale is
// rounded to bf16 once per slot and the product once per weight: at most 2^-8 relative on a weight, an
// order of magnitude inside the layer's tolerance.  Scales must stay below 2^7 for scale * 2^120 to be finite.
#include "moe_fp8w_tc.cuh"

namespace moe {
namespace {

using namespace tc;
using namespace fp8w;

// D[tmem] (+)= A[tmem] * B[smem]^T, bf16 inputs, fp32 accumulate, issued by one thread.
__device__ __forceinline__ void umma_bf16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                             uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

template <int NT_MAX, int STAGES_Q>
struct Fp8Smem {
    static constexpr bool kStaged = NT_MAX > 32 && NT_MAX < 192;     // through shared memory (Stage), where there is room
    // converted slots in tensor memory (beside two accumulators), token tiles in shared memory, and converter groups
    static constexpr int kConv = NT_MAX > 128 ? 2 : NT_MAX > 64 ? 3 : 4;
    static constexpr int kThreads = (kFirstConvWarp + kConv * kGroupWarps) * 32;
    static constexpr int kSlotBBytes = 2 * NT_MAX * kRowBytes;       // two swizzled token tiles (K 0..63 | 64..127)
    static constexpr int kB = 0;                                     // kConv token-tile pairs
    static constexpr int kQ = kB + kConv * kSlotBBytes;           // STAGES_Q code tiles
    static constexpr int kStage = kQ + STAGES_Q * kSlotQBytes;
    // q_full[SQ], q_empty[SQ], op_full[C], op_empty[C], acc_full[2], acc_empty[2]
    static constexpr int kBars = kStage + (kStaged ? kStageBytes : 0);
    static constexpr int kTmemSlot = kBars + (2 * STAGES_Q + 2 * kConv + 4) * 8;
    static constexpr int kAbort = kTmemSlot + 4;
    static constexpr int kTiles = (kAbort + 4 + 15) / 16 * 16;  // TileQueue
    static constexpr int kBytes = kTiles + TileQueue::kBytes;
    static constexpr int kDynamicBytes = kBytes + 1024;
};

template <int NT_MAX, int STAGES_Q, bool SWIGLU, int QUEUE>
__global__ void __launch_bounds__((Fp8Smem<NT_MAX, STAGES_Q>::kThreads), 1)
grouped_gemm_tc_fp8w_kernel(const __grid_constant__ TensorMapsOf<NT_MAX / 16> maps, const KernelParams p) {
    using L = Fp8Smem<NT_MAX, STAGES_Q>;
    constexpr int kConv = L::kConv;
    constexpr int kColsUsed = 2 * NT_MAX + kConv * kConvCols;
    constexpr int kTmemCols = kColsUsed <= 256 ? 256 : 512;  // (a power of two)
    static_assert(kColsUsed <= 512 && kConv * kConvCols <= 256, "accumulators and converted slots exceed tensor memory");
    constexpr int kSiteOffset = SWIGLU ? 0 : 4;
    chain_release();  // the next kernel of the forward call may be scheduled; it waits for what it needs of this grid
    extern __shared__ uint8_t smem_raw[];
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *base_ptr = smem_raw + (base - smem_u32(smem_raw));
    const uint32_t bar_q_full = base + L::kBars, bar_q_empty = bar_q_full + STAGES_Q * 8;
    const uint32_t bar_op_full = bar_q_empty + STAGES_Q * 8, bar_op_empty = bar_op_full + kConv * 8;
    const uint32_t bar_acc_full = bar_op_empty + kConv * 8, bar_acc_empty = bar_acc_full + 16;
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(base_ptr + L::kTmemSlot);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(base_ptr + L::kAbort);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    auto wait = [&](uint32_t bar, uint32_t parity, int site) {
        return mbar_wait(bar, parity, abort_flag, p.status, site + kSiteOffset);
    };
    const TileQueue tiles(base_ptr, base, L::kTiles);
    auto queue_wait = [&](uint32_t bar, uint32_t parity) { return wait(bar, parity, kSiteProducerEmpty); };
    // the n-th tile, from the decoder warp or decoded here; false at the end of the work
    auto next_tile = [&](Tile &t, int n, int tile) {
        if constexpr (QUEUE != kNoQueue) return tiles.take(t, n, lane, queue_wait) && (QUEUE != kOnDemand || t.e >= 0);
        t = decode_tile(tile, p);
        return true;
    };
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES_Q; ++s) {
            mbar_init(bar_q_full + s * 8, 1);
            mbar_init(bar_q_empty + s * 8, kGroupWarps);
        }
        for (int c = 0; c < kConv; ++c) {
            mbar_init(bar_op_full + c * 8, kGroupWarps + 1);  // the converter warps, and the token tile's bytes
            mbar_init(bar_op_empty + c * 8, 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(bar_acc_full + a * 8, 1);
            mbar_init(bar_acc_empty + a * 8, kEpilogueWarps);
        }
        tiles.init(3 + kEpilogueWarps + kConv * kGroupWarps);
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
    const int worker = blockIdx.x, n_workers = gridDim.x;

    if (warp == 0) {
        // ---------------- weight TMA ----------------
        int stage = 0;
        uint32_t phase = 0;
        bool ok = true;
        for (int round = 0; ok; ++round) {
            const int tile = tile_of_round(round, worker, n_workers);
            if (QUEUE != kOnDemand && tile >= total_tiles) break;
            Tile t;
            ok = next_tile(t, round, tile);
            if (!ok) break;
            const int w_row = t.e * p.w_rows + t.f * kTileM;
            for (int kb = 0; kb < p.n_k_blocks; ++kb) {
                ok = __all_sync(0xffffffffu, wait(bar_q_empty + stage * 8, phase ^ 1u, kSiteProducerEmpty));
                if (!ok) break;
                if (elect_one()) {
                    const uint32_t full = bar_q_full + stage * 8;
                    mbar_expect_tx(full, kSlotQBytes);
                    const uint32_t sq = base + L::kQ + stage * kSlotQBytes;
                    const int k0 = kb * kSlotK;
                    if (SWIGLU)
                        tma_load_5d(sq, &maps.w, k0, 0, 0, t.f * 4, t.e, full);
                    else
                        tma_load_2d(sq, &maps.w, k0, w_row, full);
                }
                __syncwarp();
                if (++stage == STAGES_Q) { stage = 0; phase ^= 1u; }
            }
        }
    } else if (warp == kTokenWarp) {
        // ---------------- token TMA ----------------
        int stage = 0;
        uint32_t phase = 0;
        bool ok = true, gate_up_done = false;
        for (int round = 0; ok; ++round) {
            const int tile = tile_of_round(round, worker, n_workers);
            if (QUEUE != kOnDemand && tile >= total_tiles) break;
            Tile t;
            ok = next_tile(t, round, tile);
            if (!ok) break;
            const int n_mma = (t.n_valid + 15) & ~15;
            ok = handover_wait_expert(p.handover_role, p.handover, t.e, t.n_tok_tiles, p.handover_per_token_tile,
                                      p.tile_prefix[p.E], gate_up_done, abort_flag, p.status, lane);
            if (!ok) break;
            for (int kb = 0; kb < p.n_k_blocks; ++kb) {
                ok = __all_sync(0xffffffffu, wait(bar_op_empty + stage * 8, phase ^ 1u, kSiteProducerEmpty));
                if (!ok) break;
                if (elect_one()) {
                    const uint32_t full = bar_op_full + stage * 8;
                    mbar_expect_tx(full, 2 * n_mma * kRowBytes);
                    // one copy: rows x (two 64-wide K chunks), each chunk landing as its own swizzled tile of n_mma rows
                    tma_load_3d(base + L::kB + stage * L::kSlotBBytes, act_map<16>(maps, n_mma), 0, t.row0, 2 * kb, full);
                }
                __syncwarp();
                if (++stage == kConv) { stage = 0; phase ^= 1u; }
            }
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer ----------------
        // One elected thread walks a whole tile's slots.  With the election, the vote and the warp barrier inside the
        // K loop a slot took 560 cycles to issue beside busy converter warps, more than its MMAs take (N/2 + 10 each with
        // A in tensor memory, measured): 0.400 against 0.379 ms on the 333-token layer, 0.291 against 0.267 on 32 tokens.
        int op = 0, acc = 0;
        uint32_t op_phase = 0, acc_phase = 0;
        bool ok = true;
        const uint64_t b_desc0 = smem_desc_k_major_sw128(base + L::kB);
        for (int round = 0; ok; ++round) {
            const int tile = tile_of_round(round, worker, n_workers);
            if (QUEUE != kOnDemand && tile >= total_tiles) break;
            Tile t;
            ok = next_tile(t, round, tile);
            if (!ok) break;
            const int n_mma = (t.n_valid + 15) & ~15;
            const uint32_t idesc = instr_desc_bf16(kTileM, n_mma);
            ok = __all_sync(0xffffffffu, wait(bar_acc_empty + acc * 8, acc_phase ^ 1u, kSiteMmaTmemEmpty));
            if (!ok) break;
            const uint32_t d_tmem = tmem_base + acc * NT_MAX;
            if (elect_one()) {
                int o = op;
                uint32_t ph = op_phase;
                for (int kb = 0; kb < p.n_k_blocks; ++kb) {
                    ok = wait(bar_op_full + o * 8, ph, kSiteMmaFull);
                    if (!ok) break;
                    tcgen05_fence_after();
                    const uint32_t a_tmem = tmem_base + 2 * NT_MAX + o * kConvCols;
                    const uint64_t b_desc = b_desc0 + (uint32_t)(o * (L::kSlotBBytes >> 4));
#pragma unroll
                    for (int j = 0; j < 2; ++j)  // the slot's two 64-wide K chunks
#pragma unroll
                        for (int kk = 0; kk < kBlockK / 16; ++kk)  // 16 K-elements = 8 columns of A, 2 descriptor units of B
                            umma_bf16_ts(d_tmem, a_tmem + (j * (kBlockK / 16) + kk) * 8,
                                         b_desc + (uint32_t)(j * (n_mma * kRowBytes >> 4)) + 2 * kk, idesc, (kb | j | kk) != 0);
                    umma_commit(bar_op_empty + o * 8);
                    if (++o == kConv) { o = 0; ph ^= 1u; }
                }
                if (ok) umma_commit(bar_acc_full + acc * 8);
            }
            __syncwarp();
            ok = __all_sync(0xffffffffu, ok);
            ring_advance<kConv>(op, op_phase, p.n_k_blocks);
            if (!ok) break;
            if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
        }
    } else if (warp >= kFirstConvWarp) {
        // ---------------- converters: FP8 codes -> scaled bf16 in tensor memory ----------------
        // Group g (four warps) takes the ring slots g, g + kConv, ... of the CTA's whole sequence and always converts
        // into operand buffer g.  A warp may only touch lanes 32 * (warp % 4) .. +31 of tensor memory: its threads own
        // rows 32 * (warp % 4) + lane and convert the row's 128 codes, eight 16-byte pieces of the swizzled row.
        // A stage of the weight ring belongs to one group: a wait on its parity is only valid for a warp that has seen the
        // stage's previous use complete.
        static_assert(STAGES_Q % kConv == 0, "a stage of the weight ring must always go to the same converter group");
        static_assert(kFirstConvWarp % 4 == 0 && kGroupWarps == 4, "converter lane mapping");
        const int q = warp & 3, group = (warp - kFirstConvWarp) / kGroupWarps, row = q * 32 + lane;
        const uint32_t a_tmem = tmem_base + ((uint32_t)(q * 32) << 16) + 2 * NT_MAX + group * kConvCols;
        const uint32_t full = bar_op_full + group * 8, empty = bar_op_empty + group * 8;
        const uint8_t *my_row = base_ptr + L::kQ + row * kSlotK;
        const int swz = row & 7;
        int stage = group, turn = 0;
        uint32_t phase = 0, op_phase = 0;
        bool ok = true;
        for (int round = 0; ok; ++round) {
            const int tile = tile_of_round(round, worker, n_workers);
            if (QUEUE != kOnDemand && tile >= total_tiles) break;
            Tile t;
            ok = next_tile(t, round, tile);
            if (!ok) break;
            // this row's scales: its tile's gate block or up block (gate/up: 16 gate rows, 16 up rows in turn), or the
            // tile's single block (down)
            const int row_blocks = p.w_rows >> 7;
            const int block = !SWIGLU ? t.f : ((row & 16) ? (p.n_out + t.f * 64) >> 7 : (t.f * 64) >> 7);
            const float *scale = p.w_scale + ((size_t)t.e * row_blocks + block) * p.n_k_blocks;
            int kb = (group - turn + kConv) % kConv;  // first slot of this tile that is this group's
            turn = (turn + p.n_k_blocks) % kConv;
            float next = kb < p.n_k_blocks ? __ldg(scale + kb) : 0.f;
            for (; kb < p.n_k_blocks; kb += kConv) {
                const __nv_bfloat162 s2 = __float2bfloat162_rn(next * 1329227995784915872903807060280344576.0f);  // 2^120
                if (kb + kConv < p.n_k_blocks) next = __ldg(scale + kb + kConv);  // off the critical path
                ok = __all_sync(0xffffffffu, wait(bar_q_full + stage * 8, phase, kSiteMmaFull));
                if (!ok) break;
                const uint8_t *src = my_row + stage * kSlotQBytes;
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    uint4 codes[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        codes[i] = *reinterpret_cast<const uint4 *>(src + (((half * 4 + i) ^ swz) << 4));
                    uint32_t v[32];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const uint32_t w[4] = {codes[i].x, codes[i].y, codes[i].z, codes[i].w};
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            v[i * 8 + c * 2] = convert_two<0x9180>(w[c], s2);
                            v[i * 8 + c * 2 + 1] = convert_two<0xB3A2>(w[c], s2);
                        }
                    }
                    if (half == 0) {  // the MMAs that read the buffer's previous contents are complete
                        ok = __all_sync(0xffffffffu, wait(empty, op_phase ^ 1u, kSiteProducerEmpty));
                        if (!ok) break;
                        tcgen05_fence_after();
                    }
                    __syncwarp();  // (the store is an aligned warp instruction)
                    tmem_store_32(a_tmem + half * (kConvCols / 2), v);
                }
                if (!ok) break;
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                tcgen05_fence_before();
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(full);
                    mbar_arrive(bar_q_empty + stage * 8);
                }
                __syncwarp();
                op_phase ^= 1u;
                stage += kConv;
                if (stage >= STAGES_Q) { stage = group; phase ^= 1u; }
            }
        }
    } else if (warp < kTokenWarp) {
        // ---------------- epilogue: TMEM -> registers -> global ----------------
        const int q = warp & 3;
        int acc = 0, flip = 0;
        uint32_t acc_phase = 0;
        bool ok = true;
        for (int round = 0; ok; ++round) {
            const int tile = tile_of_round(round, worker, n_workers);
            if (QUEUE != kOnDemand && tile >= total_tiles) break;
            Tile t;
            const bool taken = next_tile(t, round, tile);  // (at the end of the work the four warps leave as if they gave up: together)
            const int n_mma = (t.n_valid + 15) & ~15;
            ok = taken && wait(bar_acc_full + acc * 8, acc_phase, kSiteEpilogueTmemFull);
            if (L::kStaged ? epilogue_any(!ok) : !__all_sync(0xffffffffu, ok)) break;  // (the four warps meet inside a staged tile)
            tcgen05_fence_after();
            const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + acc * NT_MAX;
            __nv_bfloat16 *rows = p.out + (size_t)t.row0 * p.n_out + t.f * (SWIGLU ? kTileM / 2 : kTileM);  // this tile's features
            __nv_bfloat16 *dst = rows + (SWIGLU ? q * 16 + (lane & 15) : q * 32 + lane);
            if constexpr (L::kStaged) {
                drain_staged<SWIGLU>(taddr, n_mma, t.n_valid, rows, (size_t)p.n_out, base_ptr + L::kStage, flip, q, lane);
            } else {
                drain_accumulator<SWIGLU>(taddr, n_mma, t.n_valid, dst, (size_t)p.n_out, lane);
            }
            tcgen05_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_acc_empty + acc * 8);
            handover_count_tile(p.handover_role, p.handover, t.e, lane);  // (after the accumulator is handed back)
            if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
        }
    } else if (QUEUE != kNoQueue && warp == 7) {
        // ---------------- decoder ----------------
        const auto tile_at = [&](int tile) { return decode_tile(tile, p); };
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
        for (int i = 0; i < 1000; ++i) __nanosleep(1000);
    }
    if (warp == 1) {
        tcgen05_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
    }
}

template <int NT_MAX, int STAGES_Q, bool SWIGLU, int QUEUE>
int launch_fp8_instance(const TensorMaps &maps, const KernelParams &p, int grid, cudaStream_t stream) {
    using L = Fp8Smem<NT_MAX, STAGES_Q>;
    static_assert(L::kDynamicBytes <= 232448, "rings do not fit in shared memory");
    auto kernel = grouped_gemm_tc_fp8w_kernel<NT_MAX, STAGES_Q, SWIGLU, QUEUE>;
    if (!set_max_dynamic_smem_once(reinterpret_cast<const void *>(kernel), L::kDynamicBytes))
        return MOE_ERR_CUDA;
    return launch_chained(kernel, grid, L::kThreads, L::kDynamicBytes, stream, TensorMapsOf<NT_MAX / 16>(maps), p) == cudaSuccess
               ? MOE_OK : MOE_ERR_CUDA;
}

// How a CTA comes by its tiles, where it has more than one: decoded ahead (TileQueue), since the converters and the MMA run two to four
// slots ahead of one another and stood still for every walk, and on demand if they are long enough.  Without / decoded ahead:
// 389 tokens of 256 experts of 256 x 2048, top 6, 162.3 / 137.9 us (walks batched 133.0); 77 of 128 of 1536 x 2432, top 1, 153.6 / 141.1; 16
// of 256 of 7168 x 2048, top 8, 757 / 722; 1968 of 60 of 4608 x 4736, top 1, 768 / 746; one tile per CTA, 100 tokens of 8 of 256 x 512,
// top 2, 19.1 / 19.3.  Decoded ahead / on demand: one token of 128 experts of 4096 x 1536, top 8, 57.1 / 52.5; Mixtral-shaped, 32 tokens,
// 243.5 / 239.4, one 93.3 / 91.0.
template <int NT_MAX, int STAGES_Q, bool SWIGLU>
int launch_fp8_queue(const TensorMaps &maps, const KernelParams &p, int grid, int tiles_per_cta, cudaStream_t s) {
    if (tiles_per_cta <= 1) return launch_fp8_instance<NT_MAX, STAGES_Q, SWIGLU, kNoQueue>(maps, p, grid, s);
    if (tiles_on_demand(p.n_k_blocks, STAGES_Q)) return launch_fp8_instance<NT_MAX, STAGES_Q, SWIGLU, kOnDemand>(maps, p, grid, s);
    return static_queue(p.n_k_blocks, tiles_per_cta >= 8) == kBatchedQueue
               ? launch_fp8_instance<NT_MAX, STAGES_Q, SWIGLU, kBatchedQueue>(maps, p, grid, s)
               : launch_fp8_instance<NT_MAX, STAGES_Q, SWIGLU, kStaticQueue>(maps, p, grid, s);
}
template <bool SWIGLU>
int dispatch_fp8(int nt_max, const TensorMaps &maps, const KernelParams &p, int grid, int tiles_per_cta, cudaStream_t s) {
    switch (nt_max) {
        case 32: return launch_fp8_queue<32, 12, SWIGLU>(maps, p, grid, tiles_per_cta, s);
        case 64: return launch_fp8_queue<64, 8, SWIGLU>(maps, p, grid, tiles_per_cta, s);
        case 128: return launch_fp8_queue<128, 6, SWIGLU>(maps, p, grid, tiles_per_cta, s);
        case 192: return launch_fp8_queue<192, 8, SWIGLU>(maps, p, grid, tiles_per_cta, s);
        default: return MOE_ERR_UNSUPPORTED;
    }
}

}  // namespace

int launch_grouped_gemm_tc_fp8w(const GroupedGemmArgs &a, cudaStream_t stream) {
    if (a.K % 128 != 0 || a.A <= 0 || !a.w_scale || a.w_rows % 128 != 0) return MOE_ERR_UNSUPPORTED;
    if (a.nt_max > 192) return MOE_ERR_UNSUPPORTED;
    const int features_per_tile = a.swiglu ? kTileM / 2 : kTileM;
    if (a.n_out % 128 != 0) return MOE_ERR_UNSUPPORTED;  // gate and up halves must both start on a scale block

    // The tile count is only known on the device; this is its upper bound.
    const long long max_token_tiles = (long long)(a.A < a.E ? a.A : a.E) + a.A / a.nt_max;
    const long long max_tiles = max_token_tiles * (a.n_out / features_per_tile);
    const int sms = sm_count();

    TensorMaps maps;
    const bool ok_w = a.swiglu ? encode_mx_weight_map_gate_up(&maps.w, a.w, a.E, a.n_out, a.K)
                               : encode_mx_weight_map_2d(&maps.w, a.w, (uint64_t)a.E * a.w_rows, a.K);
    if (!ok_w || !encode_act_maps_chunks(maps.act, a.act, a.A, a.K, 16, 2, a.nt_max / 16)) return MOE_ERR_CUDA;

    KernelParams p;
    p.out = a.out;
    p.expert_offsets = a.expert_offsets;
    p.tile_prefix = a.tile_prefix;
    p.tile_order = a.tile_order;
    p.tile_rows = a.tile_rows;
    p.status = a.status;
    p.E = a.E;
    p.n_k_blocks = a.K / kSlotK;  // slots of 128 K-elements
    p.n_out = a.n_out;
    p.w_rows = a.w_rows;
    p.n_feature_tiles = a.n_out / features_per_tile;
    p.w_scale = a.w_scale;
    p.handover_role = a.handover_role;
    p.handover = a.handover;
    p.handover_per_token_tile = a.handover_per_token_tile;

    const int grid = (int)(max_tiles < sms ? max_tiles : sms);
    const int tiles_per_cta = (int)((max_tiles + sms - 1) / sms);
    return a.swiglu ? dispatch_fp8<true>(a.nt_max, maps, p, grid, tiles_per_cta, stream) : dispatch_fp8<false>(a.nt_max, maps, p, grid, tiles_per_cta, stream);
}

}  // namespace moe
