// Device helpers shared by the two MX FP8 grouped-GEMM kernels (one CTA per tile, and CTA pairs):
// the tile decoder with the scale-atom index, descriptors of the block-scaled MMA and of the scale
// copies, and the gate/up epilogue that quantises h.
#pragma once

#include <cuda_fp8.h>

#include "moe_tc_common.cuh"

namespace moe {
namespace mxtc {

using namespace tc;

constexpr int kMxSlotK = 128;                     // K elements = bytes per operand row per ring slot
constexpr int kMxSlotABytes = kTileM * kMxSlotK;  // 16 KiB
constexpr int kTmemColsMx = 512;

struct MxParams {
    void *out;
    uint8_t *out_sf;
    const uint8_t *w_sf, *act_sf;
    const int *expert_offsets, *tile_prefix, *tile_order, *tile_rows;
    int *status;
    int E, n_k_blocks, n_out, w_rows, n_feature_tiles, n_atoms;
    int tile_stride;     // stride of the tile numbering: min(token-tile bound, 256) (moe_internal.cuh)
    int atoms_per_tile;  // ceil(token-tile bound / 128)
    int handover_role;   // hand-over between the two GEMMs of a call (moe_internal.cuh)
    int *handover;
    int handover_per_token_tile;
};

struct MxTile {
    int e, f, row0, n_valid;
    int atom;         // first activation scale atom of the tile
    int n_tok_tiles;  // token tiles of this tile's expert
};

__device__ __forceinline__ MxTile decode_mx_tile(int tile, const MxParams &p) {
    int lo = 0, hi = p.E;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (p.tile_prefix[mid] * p.n_feature_tiles <= tile) lo = mid; else hi = mid;
    }
    MxTile t;
    t.e = p.tile_order[lo];
    const int first = p.tile_prefix[lo], n_tok_tiles = p.tile_prefix[lo + 1] - first;
    const int local = tile - first * p.n_feature_tiles;
    t.f = local / n_tok_tiles;
    const int j = local - t.f * n_tok_tiles;
    const int rows = p.tile_rows[t.e];  // rows of every tile of this expert (the bound itself for bounds up to 256)
    const int begin = p.expert_offsets[t.e], count = p.expert_offsets[t.e + 1] - begin;
    t.row0 = begin + j * rows;
    t.n_valid = min(rows, count - j * rows);
    t.atom = (begin / p.tile_stride + t.e + j) * p.atoms_per_tile;
    t.n_tok_tiles = n_tok_tiles;
    return t;
}

// Shared-memory descriptor of one scale atom: 32 rows of 16 bytes, no swizzle, 8-row groups 128 bytes apart.
__device__ __forceinline__ uint64_t smem_desc_sf_atom(uint32_t smem_addr) {
    uint64_t d = 0;
    d |= (uint64_t)((smem_addr & 0x3FFFFu) >> 4);
    d |= (uint64_t)1 << 16;
    d |= (uint64_t)(128 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    return d;
}
// Block-scaled instruction descriptor: E4M3 A and B (format 0), both K-major, E8M0 scales, M = m (128, or
// 256 for a CTA pair), N = n, scale byte `sf` of each row (the K-block within the slot) for both operands.
__device__ __forceinline__ uint32_t instr_desc_mx(int m, int n, int sf) {
    return ((uint32_t)sf << 4) | ((uint32_t)(n >> 3) << 17) | (1u << 23) | ((uint32_t)(m >> 4) << 24) |
           ((uint32_t)sf << 29);
}

// Barrier of the two epilogue warps (64 threads) that share a block of 32 features.
__device__ __forceinline__ void pair_sync(int pair) {
    asm volatile("bar.sync %0, 64;" ::"r"(2 + pair) : "memory");
}

__device__ __forceinline__ uint32_t mx_scale_byte(uint32_t amax_bits) {
    const uint32_t e = amax_bits >> 23;
    if (e == 255u) return 255u;
    return e > 8u ? e - 8u : 0u;
}

// Maxima of eight values over the 16 lanes of a half-warp by recursive halving: 8 shuffles instead of the 32 of a
// butterfly per value.  Afterwards lanes j and j ^ 1 (j = lane % 16) both hold the maximum of value j / 2.
__device__ __forceinline__ uint32_t half_warp_max8(const uint32_t (&mag)[8], int j) {
    uint32_t m4[4], m2[2];
    const bool b8 = (j & 8) != 0, b4 = (j & 4) != 0, b2 = (j & 2) != 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t recv = __shfl_xor_sync(0xffffffffu, b8 ? mag[i] : mag[4 + i], 8);
        m4[i] = max(b8 ? mag[4 + i] : mag[i], recv);
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const uint32_t recv = __shfl_xor_sync(0xffffffffu, b4 ? m4[i] : m4[2 + i], 4);
        m2[i] = max(b4 ? m4[2 + i] : m4[i], recv);
    }
    uint32_t m1 = max(b2 ? m2[1] : m2[0], __shfl_xor_sync(0xffffffffu, b2 ? m2[0] : m2[1], 2));
    return max(m1, __shfl_xor_sync(0xffffffffu, m1, 1));
}

// Gate/up epilogue of one warp for G groups of 16 accumulator columns: its 32 TMEM lanes hold, for 16 features, the gate rows
// (lanes 0..15) and the up rows (lanes 16..31).  Computes h = SiLU(gate) * up, quantises it in blocks of 32 features (this
// warp's 16 and its partner warp's 16, warps q and q^1; their maxima are exchanged through shared memory), and stores the
// codes and the scale bytes.  As in the bf16 epilogue (moe_tc_common.cuh) everything is computed before the first store, and
// whole groups are stored without conditions; two groups share one exchange.
//   left     rows of the tile from the first group's first column on
//   dst      -> code of this lane's feature in that first row; row stride n_out bytes
//   sf_dst   -> byte of the block's scale in row 0 of the tile's first atom (K-slot and block already applied); c0: that
//               first row within the tile
//   amax_s   [2][4][32] exchange buffer in shared memory; buf is flipped every call (across tiles too): a
//            warp may run one call ahead of its partner
//   stage    STAGED: two buffers of kMxStageBytes through which the CTA's 64 features of a token are stored as one row
//            (as in moe_tc_common.cuh, Stage; flipped with buf)
constexpr int kAmaxBytes = 2 * 4 * 32 * 4;
constexpr int kMxStagePitch = 80, kMxStageBytes = 32 * kMxStagePitch + 16;
__device__ __forceinline__ int mx_stage_at(int token) { return token * kMxStagePitch + ((token >> 3) & 1) * 16; }
template <int G, bool STAGED>
__device__ __forceinline__ void store_swiglu_mx(const float (&v)[G][16], int left, uint8_t *dst, size_t n_out, uint8_t *sf_dst, int c0,
                                                uint32_t *amax_s, int &buf, uint8_t *stage, int q, int lane) {
    const int hi = lane >> 4, j = lane & 15;
    float hv[G][8];
#pragma unroll
    for (int g = 0; g < G; ++g) swiglu_16(v[g], lane, hv[g]);
    buf ^= 1;
    uint32_t *mine = &amax_s[(buf * 4 + q) * 32 + hi * 8];
    const uint32_t *partner = &amax_s[(buf * 4 + (q ^ 1)) * 32 + hi * 8];
    uint32_t col_max[G];
#pragma unroll
    for (int g = 0; g < G; ++g) {
        uint32_t mag[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) mag[i] = __float_as_uint(hv[g][i]) & 0x7FFFFFFFu;  // magnitudes compare as integers; NaN and inf on top
        col_max[g] = half_warp_max8(mag, j);  // of column hi * 8 + j / 2 over this warp's 16 features
        if ((j & 1) == 0) mine[g * 16 + (j >> 1)] = col_max[g];
    }
    pair_sync(q >> 1);
#pragma unroll
    for (int g = 0; g < G; ++g) {
        // The two lanes that hold a column's maximum make its scale, and the sixteen fetch all eight by shuffles.  (Every lane had made
        // all eight, 68 instructions against 17, and where K is short the epilogue is what a tile takes: 4096 tokens of 32 experts of 1024 x
        // 1024, top 4, 150.2 -> 136.1 us, 2244 skewed ones of 160 of 768 x 3584, top 8, 361 -> 317, 4096 of 8 of 256 x 512 59.3 -> 54.7.)  A block with an infinity or
        // a NaN is all NaN codes: its factor is a NaN.
        const uint32_t sb = mx_scale_byte(max(col_max[g], partner[g * 16 + (j >> 1)]));
        const uint32_t inverse = sb == 255u ? 0x7FFFFFFFu : (254u - sb) << 23;
        uint8_t code[8];
#pragma unroll
        for (int i = 0; i < 8; i += 2) {
            const float lo = __uint_as_float(__shfl_sync(0xffffffffu, inverse, hi * 16 + 2 * i));
            const float up = __uint_as_float(__shfl_sync(0xffffffffu, inverse, hi * 16 + 2 * i + 2));
            const uint32_t two = __nv_cvt_float2_to_fp8x2(make_float2(hv[g][i] * lo, hv[g][i + 1] * up), __NV_SATFINITE, __NV_E4M3);
            code[i] = (uint8_t)two;
            code[i + 1] = (uint8_t)(two >> 8);
        }
        const int here = left - g * 16 - hi * 8;
        if constexpr (STAGED) {
#pragma unroll
            for (int i = 0; i < 8; ++i) stage[buf * kMxStageBytes + mx_stage_at(g * 16 + hi * 8 + i) + q * 16 + j] = code[i];
        } else {
            uint8_t *row = dst + (size_t)(g * 16 + hi * 8) * n_out;
            if (left >= (g + 1) * 16) {
#pragma unroll
                for (int i = 0; i < 8; ++i) row[(size_t)i * n_out] = code[i];
            } else {
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if (i < here) row[(size_t)i * n_out] = code[i];
            }
        }
        if ((q & 1) == 0 && (j & 1) == 0 && (j >> 1) < here) {  // row r of the tile: atom r / 128, atom row r % 128
            const int r = c0 + g * 16 + hi * 8 + (j >> 1);
            sf_dst[(size_t)(r >> 7) * kMxSfAtomBytes + mx_atom_byte(r & 127, 0)] = (uint8_t)sb;
        }
    }
    if constexpr (STAGED) {  // four lanes per token: warp q stores tokens 4 G q .. 4 G q + 4 G - 1
        epilogue_sync();
        const int token = q * (4 * G) + (lane >> 2);
        if (lane < 16 * G && token < left) {
            const uint4 val = *reinterpret_cast<const uint4 *>(stage + buf * kMxStageBytes + mx_stage_at(token) + (lane & 3) * 16);
            // (dst is this lane's feature: back to the CTA's first)
            *reinterpret_cast<uint4 *>(dst - (q * 16 + j) + (size_t)token * n_out + (lane & 3) * 16) = val;
        }
    }
}
// ... and for a tile's n_mma columns, of which n_valid are rows of h (dst: this lane's feature in the first).
template <bool STAGED>
__device__ __forceinline__ void drain_swiglu_mx(uint32_t taddr, int n_mma, int n_valid, uint8_t *dst, size_t n_out,
                                                uint8_t *sf_dst, uint32_t *amax_s, int &buf, uint8_t *stage, int q, int lane) {
    int c0 = 0;
    for (; c0 + 32 <= n_mma; c0 += 32) {
        float v[2][16];
        tmem_load_2x16(taddr + c0, v);
        store_swiglu_mx<2, STAGED>(v, n_valid - c0, dst + (size_t)c0 * n_out, n_out, sf_dst, c0, amax_s, buf, stage, q, lane);
    }
    if (c0 < n_mma) {
        float v[1][16];
        tmem_load_16(taddr + c0, v[0]);
        store_swiglu_mx<1, STAGED>(v, n_valid - c0, dst + (size_t)c0 * n_out, n_out, sf_dst, c0, amax_s, buf, stage, q, lane);
    }
}

// Scale tensor maps (host side): the atom arrays seen as [rows of 512 bytes] of 32-bit words.
bool encode_mx_scale_map(CUtensorMap *map, const void *atoms, uint64_t n_atoms, uint32_t atoms_per_box);

}  // namespace mxtc
}  // namespace moe
