// Device helpers shared by the FP8-weight grouped GEMMs (one CTA per tile, and CTA pairs): the converters' geometry, the
// stores to tensor memory, and the conversion of E4M3 codes to scaled bf16.
#pragma once

#include "moe_tc_common.cuh"

namespace moe {
namespace fp8w {

using namespace tc;

constexpr int kGroupWarps = 4;                     // converter warps per slot: one per quarter of tensor memory's lanes
constexpr int kFirstConvWarp = 8;
constexpr int kTokenWarp = 6;
constexpr int kSlotK = 128;                        // K elements per ring slot: one scale block, two MMA K-chunks of 64
constexpr int kSlotQBytes = kTileM * kSlotK;       // 16 KiB of codes
constexpr int kConvCols = kSlotK / 2;              // tensor-memory columns of a converted slot (two bf16 per column)

// 32 consecutive 32-bit columns of this thread's tensor-memory lane (tcgen05.wait::st completes it).
__device__ __forceinline__ void tmem_store_32(uint32_t taddr, const uint32_t (&v)[32]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
        "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
        ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]),
          "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]), "r"(v[16]), "r"(v[17]),
          "r"(v[18]), "r"(v[19]), "r"(v[20]), "r"(v[21]), "r"(v[22]), "r"(v[23]), "r"(v[24]), "r"(v[25]), "r"(v[26]),
          "r"(v[27]), "r"(v[28]), "r"(v[29]), "r"(v[30]), "r"(v[31])
        : "memory");
}

// Two E4M3 codes (bytes `kSel` of a word) -> two bf16 values times the block scale.  The permute puts each code in the
// low byte of a 16-bit lane under its replicated sign bit; shifted left by four, exponent and mantissa sit at the top of
// bf16's exponent-low / mantissa-high positions, and the mask keeps them and the sign.  That bit pattern is a bf16
// number equal to the code's value times 2^-120, for normal AND subnormal codes alike (E4M3's bias is 7, bf16's 127, and
// a zero exponent field means "no hidden one" in both); one bf16x2 multiply by scale * 2^120 finishes it.
template <uint32_t kSel>
__device__ __forceinline__ uint32_t convert_two(uint32_t codes, __nv_bfloat162 scale2) {
    uint32_t x;
    asm("prmt.b32 %0, %1, 0, %2;" : "=r"(x) : "r"(codes), "n"(kSel));
    const uint32_t bits = (x << 4) & 0x87F087F0u;
    __nv_bfloat162 v;
    *reinterpret_cast<uint32_t *>(&v) = bits;
    v = __hmul2(v, scale2);
    return *reinterpret_cast<uint32_t *>(&v);
}

}  // namespace fp8w
}  // namespace moe
