// PTX wrappers shared by the CTA-pair (cta_group::2) grouped-GEMM kernels, bf16 and MX FP8.
#pragma once

#include "moe_tc_common.cuh"

namespace moe {
namespace tc {

// Every CTA-pair kernel asks for ALL of an SM's shared memory, whatever its ring needs, so that it never shares an SM
// with another block.  Found the hard way: with a few KiB left over (a 216 KiB ring), small blocks of ANOTHER stream's
// call (the sort-scatter's one-warp blocks, 1 KiB of shared memory each) were scheduled next to pair CTAs, and on two
// streams a later pair on that TPC then waited in tcgen05.alloc for ever -- about once per thousand calls, with every
// pair kernel that left room, the 128-row instance included; with the SM to themselves the same kernels ran tens of
// thousands of overlapping calls.  The cause inside the hardware was not established; exclusivity is what the
// library's pair kernels now guarantee by construction.
constexpr int kPairDynamicSmemBytes = 232448;  // the opt-in maximum: no other block fits (each needs 1 KiB reserved)

__device__ __forceinline__ uint32_t cluster_ctarank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// Address of the same shared-memory location in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t map_to_cta(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
// The same arrival without release semantics: for hand-backs that order nothing but tensor-memory reads, which
// tcgen05.wait::ld has already completed.  (A release at cluster scope makes the arriving thread wait until its
// earlier global stores are visible to the peer SM; the epilogue would then drain its stores at every hand-back.)
__device__ __forceinline__ void mbar_arrive_cluster_relaxed(uint32_t cluster_addr) {
    asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
__device__ __forceinline__ void store_cluster_u32(uint32_t cluster_addr, uint32_t v) {
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(cluster_addr), "r"(v) : "memory");
}
// TMA copies whose completion is signalled on a barrier that may live in the peer CTA.
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap *map, int c0, int c1, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void tma_load_5d_pair(uint32_t dst, const CUtensorMap *map, int c0, int c1, int c2, int c3,
                                                 int c4, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.5d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, %6}], [%7];"
        ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(bar)
        : "memory");
}
// Arrive, on the barrier at this offset in BOTH CTAs, once the MMAs issued so far have completed.
__device__ __forceinline__ void umma_commit_pair(uint32_t bar) {
    const uint16_t both = 3;
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 ::"r"(bar), "h"(both)
                 : "memory");
}
// Release of a CTA pair's tensor memory, as the last act of both CTAs.  The deallocation is a collective of the two
// CTAs; each must still be there when the other makes its half of it, so a cluster barrier FOLLOWS it as well as
// precedes it.  (Found with two streams running wide-tile GEMMs: a CTA delayed between the barrier and its
// deallocation -- other streams' small blocks may share its SM -- while its peer had already left, exited with its
// columns still allocated; the next pair on that TPC then waited in tcgen05.alloc for ever.)
__device__ __forceinline__ void tmem_release_pair(uint32_t tmem_base, uint32_t n_cols, int warp) {
    if (warp == 1) {
        tcgen05_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(n_cols) : "memory");
    }
    __syncthreads();
    cluster_sync_all();
}
// Bounded wait that also raises the peer's abort flag when it expires.
__device__ __forceinline__ bool pair_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag, uint32_t peer_abort,
                                          int *status, int site) {
    const bool ok = mbar_wait(bar, parity, abort_flag, status, site);
    if (!ok) store_cluster_u32(peer_abort, 1u);
    return ok;
}

// The same, acquiring at cluster scope: for a barrier behind which the peer has written this CTA's shared memory.
__device__ __forceinline__ bool pair_wait_acquire(uint32_t bar, uint32_t parity, volatile int *abort_flag, uint32_t peer_abort,
                                                  int *status, int site) {
    const long long start = clock64();
    while (true) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, %3;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(bar), "r"(parity), "r"(kWaitSuspendNs)
            : "memory");
        if (done) return true;
        bool expired = *abort_flag != 0;
        if (!expired && clock64() - start > kWaitLimitCycles) {
            *abort_flag = 1;
            expired = true;
            if (atomicCAS(status, 0, (int)MOE_ERR_DEVICE_TIMEOUT) == 0) {
                status[1] = site;
                status[2] = blockIdx.x;
            }
        }
        if (expired) {
            store_cluster_u32(peer_abort, 1u);
            return false;
        }
    }
}

// Which pair GEMMs draw their tiles: those with K loops of 80 slots and more, whose tiles are so long that the static assignment's
// rounds show (512 Mixtral-shaped tokens: 128 tiles of the down GEMM on 74 pairs, which began up to 30 us apart).  Static / on demand,
// medians of alternating bursts of 40 ms, all else alike: that call 519 / 507 us, 1024 tokens 722 / 700, 333 FP8-weight tokens 354 / 343
// (1024 MX tokens 421 / 411, no more than two runs of the static form differ; the power cap evens it out in longer runs).  With shorter
// loops the next tile is wanted before the epilogue, which is then most of a tile behind, lets it be drawn: at 32 slots 4096 MX
// tokens of 128 experts of 4096 x 1536, top 8, 860 / 884 us, skewed 731 / 775; 2000 tokens of 64 of 2048 x 2048, top 4, 346 / 353.  Drawn
// two ahead those are level, but 512 Mixtral-shaped tokens took 8 % longer.
__host__ __device__ constexpr bool pair_tiles_on_demand(int slots_per_tile) { return slots_per_tile >= 80; }

// The bf16 kernels with token tiles of 256 rows and more are built to draw from 20 slots on, where they do so, two ahead, if LightTiles
// finds the routing skewed; otherwise their decoders keep to the static assignment (drawn all the same, 700 tokens of 12 experts of
// 4096 x 4096, top 2, take 239.5 us instead of 237.2, 512 Mixtral-shaped ones 507 instead of 502).  Below 20 slots not measured; a
// tile is then too short for its draw.  With 128 rows they draw from 80 slots on, and deal light tiles there too.
__host__ __device__ constexpr bool wide_pair_tiles_on_demand(int slots_per_tile, int nt_max) { return slots_per_tile >= (nt_max >= 256 ? 20 : 80); }
__host__ __device__ __forceinline__ int pair_tiles_ahead(int slots_per_tile) { return slots_per_tile >= 80 ? 1 : 2; }

// Tiles drawn in the schedule's order.
struct InOrder {
    static constexpr bool drawn = true;
    __device__ __forceinline__ void prepare() {}
    __device__ __forceinline__ int operator()(int n) const { return n; }
};

// Tiles drawn so that the light ones run beside the heavy ones.  With experts of most rows first a GEMM over skewed routing is two
// phases: full tiles, bound by matrix work while the memory idles, then tiles of few rows, bound by the stream of their weights while
// the tensor cores idle (4096 tokens of 128 experts of 4096 x 1536, top 8, Zipf: 14 experts have 96 % of the rows, 29 others bring two
// thirds of the weights; the larger of both times, summed over the experts, is 1.03 ms, the larger of both sums 0.89).  A pair takes in
// its slab faster than its share of the memory's rate when the others compute.  So tiles of at most kLightRows, half of the 230 or so
// rows at which both take as long, are dealt evenly among the heavy ones, if the first expert has more than twice as many rows.  The
// first draws of all pairs stay in order (the search for the first light tile runs beside the first tile), and the last n_pairs light
// tiles stay last, where short tiles even out the end.  Both GEMMs deal alike, so the down GEMM asks for experts in the order in which
// the gate/up GEMM finishes them.  "Light" is an expert of at most kLightRows rows: with a bound of 128 rows an expert of more may
// have tiles of fewer (410 rows: four of 112), which stay in order.  In order / dealt, alternating under the power cap: that case
// 1225 / 1209 us (another part 1290 / 1244), 2048 tokens of 64 experts of 4096 x 4096, top 4, 886 / 855 (935 / 872), 1500 of 64 of
// 7168 x 2048, top 6, 942 / 919, 4096 of 64 of 2048 x 1024, top 8, 458 / 453; with 128-row tiles 600 of 16 of 5120 x 5120, top 2,
// 332 / 317, 1024 of 64 of 7168 x 2048, top 4, 538 / 518, 800 of 16 of 7168 x 7168, top 1, 424 / 393.  A line at 64 or 144 rows and
// none or three times n_pairs kept for the end are within the spread.
struct LightTiles {
    static constexpr int kLightRows = 112;
    const KernelParams &p;
    int total_tiles, n_pairs, begin, lane;  // numbers below `begin` are in order
    bool drawn = true;
    int first = 0, spread = 0, end = 0;     // numbers begin .. end - 1 hold the `spread` tiles from tile `first` on among the others
    __device__ __forceinline__ LightTiles(const KernelParams &p, int total_tiles, int n_pairs, int lane)
        : p(p), total_tiles(total_tiles), n_pairs(n_pairs), begin(pair_tiles_ahead(p.n_k_blocks) * n_pairs), lane(lane) {}
    __device__ __forceinline__ void prepare() {  // by a whole warp
        int heavy = 0;  // the schedule ranks experts by rows: those of more than kLightRows come first
#pragma unroll 4
        for (int i = 0; i < p.E; i += 32) {
            const bool mine = i + lane < p.E;
            const int e = p.tile_order[mine ? i + lane : 0];
            heavy += __popc(__ballot_sync(0xffffffffu, mine && p.expert_offsets[e + 1] - p.expert_offsets[e] > kLightRows));
        }
        first = p.tile_prefix[heavy] * p.n_feature_tiles;
        spread = total_tiles - n_pairs - first;
        const int top = p.tile_order[0];
        const bool skewed = p.expert_offsets[top + 1] - p.expert_offsets[top] > 2 * kLightRows;
        end = skewed && first > begin && spread > 0 ? first + spread : 0;
        drawn = end > 0 || pair_tiles_on_demand(p.n_k_blocks);
    }
    __device__ __forceinline__ int operator()(int n) const {
        if (n < begin || n >= end) return n;
        const unsigned long long numbers = end - begin;
        const int before = (int)((unsigned long long)(n - begin) * spread / numbers);
        const int after = (int)((unsigned long long)(n - begin + 1) * spread / numbers);
        return after > before ? first + before : n - before;
    }
};

// Tiles on demand for a CTA pair: the leader's decoder draws them and passes each on to the peer's decoder through one entry in the
// peer's shared memory; both publish them in their own CTA's queue.
//   behind the queue: the inbox entry of eight words, inbox_full (in the peer: the leader's arrival), inbox_empty (in the leader: the
//   peer's)
struct PairTileQueue : TileQueue {
    static constexpr int kBytes = TileQueue::kBytes + 32 + 16;
    int *inbox;
    uint32_t inbox_addr, inbox_full, inbox_empty;
    __device__ __forceinline__ PairTileQueue(uint8_t *base_ptr, uint32_t base, int offset)
        : TileQueue(base_ptr, base, offset), inbox(reinterpret_cast<int *>(base_ptr + offset + TileQueue::kBytes)),
          inbox_addr(base + offset + TileQueue::kBytes), inbox_full(inbox_addr + 32), inbox_empty(inbox_addr + 40) {}
    __device__ __forceinline__ void init(int takers) const {  // by one thread
        TileQueue::init(takers);
        mbar_init(inbox_full, 1);
        mbar_init(inbox_empty, 1);
    }
    // ahead: a pair's first `ahead` tiles are assigned, and tile n is drawn once tile n - ahead has been taken by every role.
    // order: prepare() by a whole warp after the first tile, then the tile of a drawn number.
    // wait / wait_acquire(bar, parity): bounded waits, the second acquiring at cluster scope.
    template <typename T, typename Order, typename Decode, typename Wait, typename WaitAcquire>
    __device__ __forceinline__ void fill_pair_on_demand(uint32_t rank, int pair, int n_pairs, int total_tiles, int *counter, int lane, int ahead,
                                                        Order order, Decode decode, Wait wait, WaitAcquire wait_acquire) const {
        constexpr int kWords = (int)(sizeof(T) / 4);
        T t;
        t.e = -1;
        if (pair < total_tiles) t = decode(pair);
        publish(t, 0, lane);
        if (t.e < 0) return;
        order.prepare();
        if (!order.drawn) {
            const int n = fill(pair, n_pairs, total_tiles, lane, decode, wait, 1);
            t.e = -1;
            if (__all_sync(0xffffffffu, wait(empty + (n & (kDepth - 1)) * 8, ((n / kDepth) & 1) ^ 1))) publish(t, n, lane);
            return;
        }
        for (int n = 1; t.e >= 0; ++n) {
            int *w = reinterpret_cast<int *>(&t);
            if (rank == 0) {
                int tile = n * n_pairs + pair;
                if (n >= ahead) {
                    const int m = n - ahead;
                    if (!__all_sync(0xffffffffu, wait(empty + (m & (kDepth - 1)) * 8, (m / kDepth) & 1))) break;
                    if (lane == 0) tile = ahead * n_pairs + atomicAdd(counter, 1);
                    tile = __shfl_sync(0xffffffffu, tile, 0);
                    if (tile < total_tiles) tile = order(tile);
                }
                t.e = -1;
                if (tile < total_tiles) t = decode(tile);
                publish(t, n, lane);
                if (n > 1 && !__all_sync(0xffffffffu, wait(inbox_empty, n & 1))) break;
                if (lane == 0) {
                    const uint32_t dst = map_to_cta(inbox_addr, 1);
#pragma unroll
                    for (int k = 0; k < kWords; ++k) store_cluster_u32(dst + 4 * k, (uint32_t)w[k]);
                    mbar_arrive_cluster(map_to_cta(inbox_full, 1));
                }
                __syncwarp();
            } else {
                if (!__all_sync(0xffffffffu, wait_acquire(inbox_full, (n - 1) & 1))) break;
                const volatile int *in = inbox;
#pragma unroll
                for (int k = 0; k < kWords; ++k) w[k] = in[k];
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(map_to_cta(inbox_empty, 0));
                if (!__all_sync(0xffffffffu, wait(empty + (n & (kDepth - 1)) * 8, ((n / kDepth) & 1) ^ 1))) break;
                publish(t, n, lane);
            }
        }
    }
};

}  // namespace tc
}  // namespace moe
