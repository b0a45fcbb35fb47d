// Grouped expert GEMMs with FP8 (E4M3) block-scaled weights on CTA pairs: a 256 x N tile per pair.
//
// What is computed and how codes become bf16 is told in moe_gemm_tc_fp8w.cu, the kernel for one CTA per tile.  Per CTA here:
//
//   warp 0       weight TMA: per slot (128 K-elements = one scale block) this CTA's 128 x 128 tile of codes (16 KiB)
//   warp 6       token TMA: HALF of the bf16 token tile's rows, two 128-byte-swizzled 64-wide chunks, one copy
//   warps 8..    converters: a thread owns one weight row (= its lane of tensor memory)
//   warp 1       MMA (leader CTA): A from the tensor memory of both CTAs, B halves from both CTAs' token slots
//   warps 2..5   epilogue (SwiGLU or plain, two accumulators)
//   warp 7       draws tiles (on demand)
//
// What bounded the one-CTA kernel at 64 rows per tile and more: a slot of 96 rows takes in 16 KiB of codes and 24 KiB of
// tokens, 640 cycles at 64 bytes per cycle, and three token slots, tied to the three converted ones, do not cover the
// microsecond a token slot takes to arrive from L2: 1030 cycles per slot.  A pair's CTA takes in half of the tokens and keeps
// six token slots, two per converted one.  333 Mixtral-shaped tokens 338 -> 311 us, 2000 tokens 1380 -> 1186 us, 4096 tokens
// of 128 experts of 4096 x 1536 1559 -> 1330 us.  What bounds it now: a slot takes 620 to 750 cycles, and the MMA thread
// never waits for an operand there, so it is the eight MMAs (about 77 cycles each at N = 96, where the shape asks for 48: why
// is not established); the converters' ALU and FMA pipes are half busy beside them.
//
// Pair protocol (rank 0 = leader), as in the bf16 pair kernel (moe_gemm_tc_pair.cu):
//   q_full, q_empty      each CTA's own weight ring, between its weight producer and its converters
//   op_full[s]           in the leader: the token slot's bytes of BOTH CTAs and one arrival per converter warp of BOTH
//   op_empty[s], acc_full   one per CTA, arrived on by the leader's commits (both CTAs at once)
//   acc_empty[a]         in the leader, one arrival per epilogue warp of both CTAs
// Before leaving, token producers, converters and the MMA warp wait for everything they have handed over to come back, so
// no arrival can reach a CTA that has exited.
#include "moe_fp8w_tc.cuh"
#include "moe_tc_pair.cuh"

namespace moe {
namespace {

using namespace tc;
using namespace fp8w;

// D[tmem of both CTAs] (+)= A[tmem of both CTAs] * B^T over the pair: M = 256, B halves from both CTAs.
__device__ __forceinline__ void umma_bf16_ts_pair(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                                  uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void tma_load_3d_pair(uint32_t dst, const CUtensorMap *map, int c0, int c1, int c2, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(bar)
        : "memory");
}

// ---- the tile schedule in shared memory ---------------------------------------------------------------------
// A walk from a tile number to its expert, slab and rows is a chain of dependent loads (a binary search over the experts'
// tile counts, then the expert's entries).  Through global memory, beside the operand streams, it took 5000-6000 cycles in
// front of every tile of every role, and the converters and the MMA warp run only two or three slots ahead of one another:
// they stood still for it.  So the CTA copies the schedule once, in one round trip, and walks its copy (200-300 cycles):
// 333-token Mixtral-shaped layer 342 -> 324 us, 4096 tokens of 128 experts 1531 -> 1493 us.  (The other GEMMs, whose
// producers run a ring of six slots or more ahead, lost up to 1 % by the same copy; their short tiles are decoded ahead by a warp
// of its own, TileQueue.)
constexpr int kLookAheadSlots = 16;  // of a tile drawn on demand: so many slots before the end its successor is asked for
constexpr int kScheduleInts = 3 * kMaxExperts + 2;
struct Schedule {
    const int *prefix, *offsets;  // [E+1] token tiles before a schedule position; first row of an expert
    const int *packed;            // [E] expert at a schedule position | rows per token tile of the expert of that number << 8
    int total_token_tiles;
};
// Run by all threads of the CTA.  ok = false: an empty schedule.
__device__ __forceinline__ Schedule stage_schedule(const KernelParams &p, int *buf, bool ok) {
    Schedule s;
    s.prefix = buf;
    s.offsets = buf + p.E + 1;
    s.packed = buf + 2 * p.E + 2;
    if (ok) {
        for (int i = threadIdx.x; i <= p.E; i += blockDim.x) {
            const int prefix = p.tile_prefix[i], offset = p.expert_offsets[i];
            const int order = i < p.E ? p.tile_order[i] : 0, rows = i < p.E ? p.tile_rows[i] : 0;
            buf[i] = prefix;
            buf[p.E + 1 + i] = offset;
            if (i < p.E) buf[2 * p.E + 2 + i] = order | (rows << 8);
        }
    }
    __syncthreads();
    s.total_token_tiles = ok ? s.prefix[p.E] : 0;
    return s;
}
// decode_tile (moe_tc_common.cuh) on the copy.
__device__ __forceinline__ Tile decode_tile(int tile, const KernelParams &p, const Schedule &s) {
    int lo = 0, hi = p.E;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (s.prefix[mid] * p.n_feature_tiles <= tile) lo = mid; else hi = mid;
    }
    Tile t;
    t.e = s.packed[lo] & 255;
    const int first = s.prefix[lo], n_tok_tiles = s.prefix[lo + 1] - first;
    const int local = tile - first * p.n_feature_tiles;
    t.f = local / n_tok_tiles;
    const int rows = s.packed[t.e] >> 8;
    t.row0 = s.offsets[t.e] + (local - t.f * n_tok_tiles) * rows;
    t.n_valid = min(rows, s.offsets[t.e + 1] - t.row0);
    t.n_tok_tiles = n_tok_tiles;
    return t;
}

// Tiles on demand: the queue's entries are numbers, which every role looks up in its CTA's copy of the schedule.
struct TileNumber {
    int e, tile;  // e = -1: the end of the work
};

// Rings of one instance: converted slots beside two accumulators in tensor memory, a converter group for each; shared memory
// is split between codes (from HBM: at least 96 KiB in flight) and token slots (from L2).  With 128 rows per tile, converted
// slots / weight stages / token stages of 3 / 6 / 6 took 328 us on the 333-token Mixtral-shaped layer, 4 / 8 / 4 339 us and
// 2 / 8 / 6 368 us.
template <int NT_MAX>
struct Fp8PairSmem {
    static constexpr int kConv = NT_MAX > 128 ? 2 : 3;
    static constexpr int kStagesQ = 6;
    static constexpr int kStagesT = NT_MAX > 128 ? 4 : 6;
    static constexpr int kThreads = (kFirstConvWarp + kConv * kGroupWarps) * 32;
    static_assert(kStagesT % kConv == 0 && kStagesQ % kConv == 0, "a slot's token stage, weight stage and buffer go together");
    static constexpr int kSlotBBytes = NT_MAX * kRowBytes;  // this CTA's rows, two swizzled chunks (K 0..63 | 64..127)
    static constexpr int kB = 0;                                     // kStagesT token slots
    static constexpr int kQ = kB + kStagesT * kSlotBBytes;           // kStagesQ code tiles
    static constexpr int kStage = kQ + kStagesQ * kSlotQBytes;       // the epilogue's buffers
    static constexpr int kBars = kStage + kStageBytes;
    static constexpr int kNumBars = 2 * kStagesQ + 2 * kStagesT + 4;
    static constexpr int kTmemSlot = kBars + kNumBars * 8;
    static constexpr int kAbort = kTmemSlot + 4;
    static constexpr int kSchedule = kAbort + 4;
    static constexpr int kTiles = (kSchedule + kScheduleInts * 4 + 15) / 16 * 16;  // PairTileQueue
    static constexpr int kBytes = kTiles + PairTileQueue::kBytes;
    static constexpr int kDynamicBytes = kPairDynamicSmemBytes;  // (kBytes + 1024 of it are used)
};

template <int NT_MAX, bool SWIGLU, int QUEUE>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__((Fp8PairSmem<NT_MAX>::kThreads), 1)
grouped_gemm_tc_fp8w_pair_kernel(const __grid_constant__ TensorMapsOf<NT_MAX / 16> maps, const KernelParams p) {
    using L = Fp8PairSmem<NT_MAX>;
    constexpr int kConv = L::kConv, kStagesQ = L::kStagesQ, kStagesT = L::kStagesT;
    constexpr int kColsUsed = 2 * NT_MAX + kConv * kConvCols;
    constexpr int kTmemCols = kColsUsed <= 256 ? 256 : 512;  // (a power of two)
    static_assert(kColsUsed <= 512 && kConv * kConvCols <= 256, "accumulators and converted slots exceed tensor memory");
    constexpr int kSiteOffset = SWIGLU ? 0 : 4;
    constexpr int kFeatPerCta = SWIGLU ? kTileM / 2 : kTileM;
    chain_release();  // the next kernel of the forward call may be scheduled; it waits for what it needs of this grid
    extern __shared__ uint8_t smem_raw[];
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *base_ptr = smem_raw + (base - smem_u32(smem_raw));
    const uint32_t bar_q_full = base + L::kBars, bar_q_empty = bar_q_full + kStagesQ * 8;
    const uint32_t bar_op_full = bar_q_empty + kStagesQ * 8, bar_op_empty = bar_op_full + kStagesT * 8;
    const uint32_t bar_acc_full = bar_op_empty + kStagesT * 8, bar_acc_empty = bar_acc_full + 16;
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(base_ptr + L::kTmemSlot);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(base_ptr + L::kAbort);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();
    const uint32_t peer_abort = map_to_cta(base + L::kAbort, rank ^ 1u);
    auto wait = [&](uint32_t bar, uint32_t parity, int site) {
        return pair_wait(bar, parity, abort_flag, peer_abort, p.status, site + kSiteOffset);
    };
    const PairTileQueue tiles(base_ptr, base, L::kTiles);
    auto queue_wait = [&](uint32_t bar, uint32_t parity) { return wait(bar, parity, kSiteProducerEmpty); };
    if (threadIdx.x == 0) {
        if constexpr (QUEUE == kOnDemand) tiles.init((rank == 0 ? 3 : 2) + kEpilogueWarps + L::kConv * kGroupWarps);
        for (int s = 0; s < kStagesQ; ++s) {
            mbar_init(bar_q_full + s * 8, 1);
            mbar_init(bar_q_empty + s * 8, kGroupWarps);
        }
        for (int s = 0; s < kStagesT; ++s) {
            mbar_init(bar_op_full + s * 8, 2 * kGroupWarps + 1);  // the converter warps of both CTAs, and the tokens' bytes
            mbar_init(bar_op_empty + s * 8, 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(bar_acc_full + a * 8, 1);
            mbar_init(bar_acc_empty + a * 8, 2 * kEpilogueWarps);
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 0 && lane == 0) {
        prefetch_map(&maps.w);
        prefetch_map(&maps.act[0]);
    }
    if (warp == 1) {  // collective over the same warp of both CTAs
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(base + L::kTmemSlot),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tcgen05_fence_before();
    __syncthreads();
    cluster_sync_all();  // the peer's barriers exist before anything can signal them
    tcgen05_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    // everything above overlapped the kernels in front; from here on there is a schedule (the token side waits for more)
    const bool started = gemm_chain_start(p.handover_role, p.handover, abort_flag, p.status);
    const Schedule sched = stage_schedule(p, reinterpret_cast<int *>(base_ptr + L::kSchedule), started);
    const int total_tiles = sched.total_token_tiles * p.n_feature_tiles;
    const int n_pairs = gridDim.x >> 1, pair = blockIdx.x >> 1;
    // The tile of a round (by a whole warp), or total_tiles at the end of the work (also of a CTA that is aborting).
    auto tile_at = [&](int round) {
        if constexpr (QUEUE == kOnDemand) {
            TileNumber t;
            return tiles.take(t, round, lane, queue_wait) && t.e >= 0 ? t.tile : total_tiles;
        }
        return tile_of_round(round, pair, n_pairs);
    };

    if (warp == 0) {
        // ---------------- weight TMA (both CTAs, each its own rows) ----------------
        int stage = 0;
        uint32_t phase = 0;
        bool ok = true;
        for (int round = 0; ok; ++round) {
            const int tile = tile_at(round);
            if (tile >= total_tiles) break;
            const Tile t = decode_tile(tile, p, sched);
            const int feat0 = (2 * t.f + (int)rank) * kFeatPerCta;
            for (int kb = 0; kb < p.n_k_blocks; ++kb) {
                ok = __all_sync(0xffffffffu, wait(bar_q_empty + stage * 8, phase ^ 1u, kSiteProducerEmpty));
                if (!ok) break;
                if (elect_one()) {
                    const uint32_t full = bar_q_full + stage * 8;
                    mbar_expect_tx(full, kSlotQBytes);
                    const uint32_t sq = base + L::kQ + stage * kSlotQBytes;
                    const int k0 = kb * kSlotK;
                    if (SWIGLU)
                        tma_load_5d(sq, &maps.w, k0, 0, 0, feat0 >> 4, t.e, full);
                    else
                        tma_load_2d(sq, &maps.w, k0, t.e * p.w_rows + feat0, full);
                }
                __syncwarp();
                if (++stage == kStagesQ) { stage = 0; phase ^= 1u; }
            }
        }
    } else if (warp == kTokenWarp) {
        // ---------------- token TMA (both CTAs, each half of the rows) ----------------
        int stage = 0;
        uint32_t phase = 0;
        bool ok = true, gate_up_done = false;
        for (int round = 0; ok; ++round) {
            const int tile = tile_at(round);
            if (tile >= total_tiles) break;
            const Tile t = decode_tile(tile, p, sched);
            const int n_mma = (t.n_valid + 15) & ~15, my_rows = n_mma >> 1;
            ok = handover_wait_expert(p.handover_role, p.handover, t.e, t.n_tok_tiles, p.handover_per_token_tile,
                                      sched.total_token_tiles, gate_up_done, abort_flag, p.status, lane);
            if (!ok) {
                store_cluster_u32(peer_abort, 1u);
                break;
            }
            for (int kb = 0; kb < p.n_k_blocks; ++kb) {
                ok = __all_sync(0xffffffffu, wait(bar_op_empty + stage * 8, phase ^ 1u, kSiteProducerEmpty));
                if (!ok) break;
                if (elect_one()) {
                    if (rank == 0) mbar_expect_tx(bar_op_full + stage * 8, 2 * n_mma * kRowBytes);
                    // one copy: rows x (two 64-wide K chunks), each chunk landing as its own swizzled tile of my_rows rows
                    tma_load_3d_pair(base + L::kB + stage * L::kSlotBBytes, act_map<8>(maps, my_rows), 0,
                                     t.row0 + (int)rank * my_rows, 2 * kb, map_to_cta(bar_op_full + stage * 8, 0));
                }
                __syncwarp();
                if (++stage == kStagesT) { stage = 0; phase ^= 1u; }
            }
        }
        for (int s = 0; ok && s < kStagesT; ++s) {  // every slot handed back: no commit may arrive here after exit
            ok = __all_sync(0xffffffffu, wait(bar_op_empty + stage * 8, phase ^ 1u, kSiteProducerEmpty));
            if (++stage == kStagesT) { stage = 0; phase ^= 1u; }
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer (leader CTA only): one elected thread walks a whole tile's slots ----------------
        if (rank == 0) {
            int stage = 0, acc = 0;
            uint32_t phase = 0, acc_phase = 0;
            bool ok = true;
            const uint64_t b_desc0 = smem_desc_k_major_sw128(base + L::kB);
            for (int round = 0; ok; ++round) {
                const int tile = tile_at(round);
                if (tile >= total_tiles) break;
                const Tile t = decode_tile(tile, p, sched);
                const int n_mma = (t.n_valid + 15) & ~15, my_rows = n_mma >> 1;
                const uint32_t idesc = instr_desc_bf16(2 * kTileM, n_mma);
                ok = __all_sync(0xffffffffu, wait(bar_acc_empty + acc * 8, acc_phase ^ 1u, kSiteMmaTmemEmpty));
                if (!ok) break;
                const uint32_t d_tmem = tmem_base + acc * NT_MAX;
                if (elect_one()) {
                    int st = stage;
                    uint32_t ph = phase;
                    for (int kb = 0; kb < p.n_k_blocks; ++kb) {
                        ok = wait(bar_op_full + st * 8, ph, kSiteMmaFull);
                        if (!ok) break;
                        tcgen05_fence_after();
                        const uint32_t a_tmem = tmem_base + 2 * NT_MAX + (st % kConv) * kConvCols;
                        const uint64_t b_desc = b_desc0 + (uint32_t)(st * (L::kSlotBBytes >> 4));
#pragma unroll
                        for (int j = 0; j < 2; ++j)  // the slot's two 64-wide K chunks
#pragma unroll
                            for (int kk = 0; kk < kBlockK / 16; ++kk)  // 16 K-elements = 8 columns of A, 2 descriptor units of B
                                umma_bf16_ts_pair(d_tmem, a_tmem + (j * (kBlockK / 16) + kk) * 8,
                                                  b_desc + (uint32_t)(j * (my_rows * kRowBytes >> 4)) + 2 * kk, idesc,
                                                  (kb | j | kk) != 0);
                        umma_commit_pair(bar_op_empty + st * 8);
                        if (++st == kStagesT) { st = 0; ph ^= 1u; }
                    }
                    if (ok) umma_commit_pair(bar_acc_full + acc * 8);
                }
                __syncwarp();
                ok = __all_sync(0xffffffffu, ok);
                ring_advance<kStagesT>(stage, phase, p.n_k_blocks);
                if (!ok) break;
                if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
            }
            for (int a = 0; ok && a < 2; ++a) {  // both accumulators released by both CTAs' epilogues
                ok = __all_sync(0xffffffffu, wait(bar_acc_empty + acc * 8, acc_phase ^ 1u, kSiteMmaTmemEmpty));
                if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
            }
        }
    } else if (warp >= kFirstConvWarp) {
        // ---------------- converters (both CTAs): FP8 codes -> scaled bf16 in tensor memory ----------------
        // Group g (four warps) takes the slots g, g + kConv, ... of the CTA's whole sequence and always converts
        // into operand buffer g.  A warp may only touch lanes 32 * (warp % 4) .. +31 of tensor memory: its threads own
        // rows 32 * (warp % 4) + lane and convert the row's 128 codes, eight 16-byte pieces of the swizzled row.
        // A stage of a ring belongs to one group: a wait on its parity is only valid for a warp that has seen the
        // stage's previous use complete.
        static_assert(kFirstConvWarp % 4 == 0 && kGroupWarps == 4, "converter lane mapping");
        const int q = warp & 3, group = (warp - kFirstConvWarp) / kGroupWarps, row = q * 32 + lane;
        const uint32_t a_tmem = tmem_base + ((uint32_t)(q * 32) << 16) + 2 * NT_MAX + group * kConvCols;
        const uint32_t leader_full = map_to_cta(bar_op_full, 0);
        const uint8_t *my_row = base_ptr + L::kQ + row * kSlotK;
        const int swz = (row & 7) << 4;
        int stage = group, turn = 0;
        uint32_t phase = 0;
        // the slot's token stage, and the stage and phase of the slot that last used this group's buffer
        int op = group, last = (group + kStagesT - kConv) % kStagesT;
        uint32_t last_phase = 1, op_phase = 0;  // (a fresh barrier counts as handed back)
        bool ok = true;
        // A tile's row of scales, and the first of them that is this group's, are fetched while the tile before it is
        // converted: the schedule walk and a load from memory in front of every tile would stall all groups at once.
        const int row_blocks = p.w_rows >> 7;
        auto scale_row = [&](int tile) {
            const Tile t = decode_tile(tile, p, sched);
            // this row's scales: its tile's gate block or up block (gate/up: 16 gate rows, 16 up rows in turn), or the
            // CTA's single block (down)
            const int gate_row = (2 * t.f + (int)rank) * kFeatPerCta;
            const int block = !SWIGLU ? 2 * t.f + (int)rank : ((row & 16) ? p.n_out + gate_row : gate_row) >> 7;
            return p.w_scale + ((size_t)t.e * row_blocks + block) * p.n_k_blocks;
        };
        int tile = tile_at(0), kb = group;
        const float *scale = tile < total_tiles ? scale_row(tile) : nullptr;
        float next = scale && kb < p.n_k_blocks ? __ldg(scale + kb) : 0.f;
        for (int round = 0; ok && tile < total_tiles; ++round) {
            int tile_ahead = QUEUE == kOnDemand ? -1 : tile_of_round(round + 1, pair, n_pairs);
            turn = (turn + p.n_k_blocks) % kConv;
            const int kb_ahead = (group - turn + kConv) % kConv;  // first slot of the next tile that is this group's
            const float *scale_ahead = nullptr;
            float next_ahead = 0.f;
            auto look_ahead = [&]() {
                if (scale_ahead || tile_ahead >= total_tiles) return;
                if (QUEUE == kOnDemand) {
                    tile_ahead = tile_at(round + 1);
                    if (tile_ahead >= total_tiles) return;
                }
                scale_ahead = scale_row(tile_ahead);
                if (kb_ahead < p.n_k_blocks) next_ahead = __ldg(scale_ahead + kb_ahead);
            };
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
                    for (int i = 0; i < 4; ++i) codes[i] = *reinterpret_cast<const uint4 *>(src + (((half * 4 + i) << 4) ^ swz));
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
                        ok = __all_sync(0xffffffffu, wait(bar_op_empty + last * 8, last_phase, kSiteProducerEmpty));
                        if (!ok) break;
                        tcgen05_fence_after();
                    }
                    tmem_store_32(a_tmem + half * (kConvCols / 2), v);
                }
                if (!ok) break;
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                tcgen05_fence_before();
                __syncwarp();
                if (lane == 0) {
                    // (the arrival orders tensor-memory stores only, complete by now: with release semantics at cluster scope
                    // it waits for the scale on its way from memory, 3000 cycles per slot)
                    mbar_arrive_cluster_relaxed(leader_full + op * 8);
                    mbar_arrive(bar_q_empty + stage * 8);
                }
                last = op;
                last_phase = op_phase;
                op += kConv;
                if (op >= kStagesT) { op = group; op_phase ^= 1u; }
                stage += kConv;
                if (stage >= kStagesQ) { stage = group; phase ^= 1u; }
                // (behind the tile's first slot of this group; a tile still to be drawn is not waited for until the last slots)
                if (QUEUE != kOnDemand || kb + kLookAheadSlots >= p.n_k_blocks) look_ahead();
            }
            look_ahead();
            tile = tile_ahead;
            kb = kb_ahead;
            scale = scale_ahead;
            next = next_ahead;
        }
        // the buffer's last contents have been read (the token producer waits for the last commits themselves)
    } else if (warp < kTokenWarp) {
        // ---------------- epilogue (both CTAs): own 128 weight rows x all N tokens, TMEM -> registers -> global ----------------
        const int q = warp & 3;
        int acc = 0, flip = 0;
        uint32_t acc_phase = 0;
        bool ok = true;
        for (int round = 0; ok; ++round) {
            const int tile = tile_at(round);
            if (QUEUE != kOnDemand && tile >= total_tiles) break;
            ok = tile < total_tiles;  // (on demand the four warps leave at the end as if they gave up: together)
            Tile t = {};
            if (ok) t = decode_tile(tile, p, sched);
            const int n_mma = (t.n_valid + 15) & ~15;
            const int feat0 = (2 * t.f + (int)rank) * kFeatPerCta;
            ok = ok && wait(bar_acc_full + acc * 8, acc_phase, kSiteEpilogueTmemFull);
            if (epilogue_any(!ok)) break;  // the four warps meet inside the tile: they leave together
            tcgen05_fence_after();
            drain_staged<SWIGLU>(tmem_base + ((uint32_t)(q * 32) << 16) + acc * NT_MAX, n_mma, t.n_valid,
                                 p.out + (size_t)t.row0 * p.n_out + feat0, (size_t)p.n_out, base_ptr + L::kStage, flip, q, lane);
            tcgen05_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster_relaxed(map_to_cta(bar_acc_empty + acc * 8, 0));
            handover_count_tile(p.handover_role, p.handover, t.e, lane);  // (after the accumulator is handed back)
            if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
        }
    } else if (QUEUE == kOnDemand && warp == 7) {
        // ---------------- decoder ----------------
        tiles.fill_pair_on_demand<TileNumber>(rank, pair, n_pairs, total_tiles, p.status + kTileCounterInt + (SWIGLU ? 0 : 1), lane, 1,
                                              InOrder{}, [](int tile) { return TileNumber{0, tile}; }, queue_wait, [&](uint32_t bar, uint32_t parity) {
            return pair_wait_acquire(bar, parity, abort_flag, peer_abort, p.status, kSiteProducerEmpty + kSiteOffset);
        });
    }

    // ---------------- teardown ----------------
    gemm_chain_finish(p.handover_role);
    tcgen05_fence_before();
    __syncthreads();
    cluster_sync_all();
    if (*abort_flag) {
        for (int i = 0; i < 1000; ++i) __nanosleep(1000);
    }
    tmem_release_pair(tmem_base, kTmemCols, warp);
}

template <int NT_MAX, bool SWIGLU>
int launch_fp8w_pair_instance(const TensorMaps &maps, const KernelParams &p, int grid, cudaStream_t stream) {
    using L = Fp8PairSmem<NT_MAX>;
    static_assert(L::kBytes + 1024 <= L::kDynamicBytes, "rings do not fit in shared memory");
    auto kernel = pair_tiles_on_demand(p.n_k_blocks) ? grouped_gemm_tc_fp8w_pair_kernel<NT_MAX, SWIGLU, kOnDemand>
                                                     : grouped_gemm_tc_fp8w_pair_kernel<NT_MAX, SWIGLU, kStaticQueue>;
    if (!set_max_dynamic_smem_once(reinterpret_cast<const void *>(kernel), L::kDynamicBytes))
        return MOE_ERR_CUDA;
    return launch_chained(kernel, grid, L::kThreads, L::kDynamicBytes, stream, TensorMapsOf<NT_MAX / 16>(maps), p) == cudaSuccess ? MOE_OK : MOE_ERR_CUDA;
}

}  // namespace

// Tiles of more than 64 rows, in K loops of eight slots or more (shorter ones do not hide what a pair's barriers cost), whose
// features fill whole pair tiles.  One CTA per tile / pairs: 2000 tokens of 8 experts of 4096 x 14336, top 2, 1380 / 1186 us;
// 1024 of 64 of 7168 x 2048, top 8, 971 / 817; 1500 of 128 of 4096 x 1536, top 8, 742 / 641; 1200 of 20 of 2048 x 1024, top 2,
// 83.1 / 78.8; 2000 of 16 of 1280 x 1280, top 2, 85.0 / 84.7; at eight slots 4096 of 32 of 1024 x 1024, top 4, 157 / 144, but calls of
// few tiles lose, 2000 of 16, top 2, 70.1 / 72.2; below, 2000 of 16 of 768 x 768, top 2, 55.5 / 57.4 and 8192 of 8 of 256 x 512, top 2,
// 68.8 / 71.4.  (Tiles of up to 64 rows, with an earlier epilogue: 150 of 8 of 4096 x 14336, top 2, 278 / 292.)
bool grouped_gemm_tc_fp8w_pair_applies(const GroupedGemmArgs &a) {
    return (a.nt_max == 128 || a.nt_max == 192) && a.K >= 8 * kSlotK && a.n_out % (a.swiglu ? kTileM : 2 * kTileM) == 0;
}

int launch_grouped_gemm_tc_fp8w_pair(const GroupedGemmArgs &a, cudaStream_t stream) {
    if (a.K % 128 != 0 || a.A <= 0 || !a.w_scale || a.w_rows % 128 != 0) return MOE_ERR_UNSUPPORTED;
    if (!grouped_gemm_tc_fp8w_pair_applies(a)) return MOE_ERR_UNSUPPORTED;
    const int features_per_tile = a.swiglu ? kTileM : 2 * kTileM;  // of a pair
    if (a.n_out % 128 != 0) return MOE_ERR_UNSUPPORTED;  // gate and up halves must both start on a scale block

    TensorMaps maps;
    const bool ok_w = a.swiglu ? encode_mx_weight_map_gate_up(&maps.w, a.w, a.E, a.n_out, a.K)
                               : encode_mx_weight_map_2d(&maps.w, a.w, (uint64_t)a.E * a.w_rows, a.K);
    if (!ok_w || !encode_act_maps_chunks(maps.act, a.act, a.A, a.K, 8, 2, a.nt_max / 16)) return MOE_ERR_CUDA;

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

    const long long max_token_tiles = (long long)(a.A < a.E ? a.A : a.E) + a.A / a.nt_max;
    const long long max_tiles = max_token_tiles * p.n_feature_tiles;
    const int pairs_on_device = sm_count() / 2;
    const int n_pairs = (int)(max_tiles < pairs_on_device ? max_tiles : pairs_on_device);
    const int grid = 2 * (n_pairs > 0 ? n_pairs : 1);
    if (a.nt_max == 128)
        return a.swiglu ? launch_fp8w_pair_instance<128, true>(maps, p, grid, stream)
                        : launch_fp8w_pair_instance<128, false>(maps, p, grid, stream);
    return a.swiglu ? launch_fp8w_pair_instance<192, true>(maps, p, grid, stream)
                    : launch_fp8w_pair_instance<192, false>(maps, p, grid, stream);
}

}  // namespace moe
