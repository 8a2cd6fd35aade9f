// Device helpers shared by the W4A8 kernels: BF16 / E4M3 conversions and the INT4 -> E4M3
// look-up-table dequantizer that implements Eq. 10.  sm_100a only.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/w4a8.h"

namespace w4a8 {


constexpr int kGroup = 128;           // group size along K (Sec. 4.1: "group size of 128")
constexpr float kE4M3Max = 448.0f;    // Z_max of Eq. 3 / Eq. 13

// Device status word bits.
constexpr unsigned int kStatusTimeout = 1u;   // a bounded device-side wait gave up
constexpr unsigned int kStatusBadCode = 2u;   // prepack met a code the target format cannot hold

__device__ __forceinline__ float bf16_bits_to_float(uint32_t bits16) {
    return __uint_as_float(bits16 << 16);
}

// Two fp32 values -> two E4M3 bytes (round-to-nearest-even, saturate to +-448).
// Result bits [7:0] = encode(lo), bits [15:8] = encode(hi).
__device__ __forceinline__ uint32_t cvt_e4m3x2(float hi, float lo) {
    uint16_t r;
    asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(r) : "f"(hi), "f"(lo));
    return (uint32_t)r;
}

// Four fp32 values -> four E4M3 bytes, v0 in the lowest byte.  (Both halves in one asm block: the second conversion then
// merges the first one's result, 5 cycles of a sub-partition; a shift and an OR behind them made it 8.)
__device__ __forceinline__ uint32_t cvt_e4m3x4(float v0, float v1, float v2, float v3) {
    uint32_t r;
    asm("{\n\t"
        ".reg .b16 lo, hi;\n\t"
        "cvt.rn.satfinite.e4m3x2.f32 lo, %2, %1;\n\t"
        "cvt.rn.satfinite.e4m3x2.f32 hi, %4, %3;\n\t"
        "mov.b32 %0, {lo, hi};\n\t"
        "}\n"
        : "=r"(r)
        : "f"(v0), "f"(v1), "f"(v2), "f"(v3));
    return r;
}

__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
    uint32_t d;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
    return d;
}

// The expansion is bound by the integer pipe (a warp's instruction every other cycle: logic, shifts, byte permutes), so what
// can is done beside it on the multipliers: shifts as multiplications, sums as multiply-adds.  The factors must not be known to
// ptxas, which turns constants back into shifts and plain sums: they come from the block's z extent, 1 in every launch here, which
// is read where a launch's parameters are.  (From __constant__ variables each launch waited half a microsecond for the first one.)
__device__ __forceinline__ uint32_t expand_one() { return blockDim.z; }

// Selector of the upper four nibbles (a byte permute reads the low half only): 0 * low half + 1 * high half.
__device__ __forceinline__ uint32_t high_half(uint32_t w) {
    uint32_t d;
    asm("dp2a.lo.u32.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(w), "r"(blockDim.z << 8), "r"(0u));
    return d;
}

// Two fp32 lanes per instruction.
__device__ __forceinline__ unsigned long long fma_f32x2(unsigned long long a, unsigned long long b, unsigned long long c) {
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ unsigned long long mul_f32x2(unsigned long long a, unsigned long long b) {
    unsigned long long d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ unsigned long long add_f32x2(unsigned long long a, unsigned long long b) {
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ unsigned long long pack_f32x2(float lo, float hi) {
    unsigned long long d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
    return d;
}
__device__ __forceinline__ void unpack_f32x2(unsigned long long v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}

// Two BF16 lanes: (x - off) * sc, the subtraction exact for the small integers it is used on, the
// product rounded once to nearest even.
__device__ __forceinline__ uint32_t bf16x2_sub_mul(uint32_t x, uint32_t off, uint32_t sc) {
    uint32_t d;
    asm("{\n\t"
        ".reg .b32 t;\n\t"
        "sub.rn.bf16x2 t, %1, %2;\n\t"
        "mul.rn.bf16x2 %0, t, %3;\n\t"
        "}\n"
        : "=r"(d)
        : "r"(x), "r"(off), "r"(sc));
    return d;
}

// Eq. 10 as a 16-entry table for one (row, group): entry u holds nearest_E4M3((u - z) * s).
// (u - z) is a small integer and s a BF16 value, so the fp32 product is exact and the table
// entry is the exact product rounded once -- the same bits as converting element by element.
struct DequantLut {
    uint32_t t[4];  // t[j] byte i = entry 4*j + i
    __device__ __forceinline__ void build(float s, int z) {
        float fz = (float)z;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            float d0 = (float)(4 * j + 0) - fz;
            float d1 = (float)(4 * j + 1) - fz;
            float d2 = (float)(4 * j + 2) - fz;
            float d3 = (float)(4 * j + 3) - fz;
            t[j] = cvt_e4m3x4(__fmul_rn(d0, s), __fmul_rn(d1, s), __fmul_rn(d2, s),
                              __fmul_rn(d3, s));
        }
    }
    // w holds eight codes, element i in bits [4i+3 : 4i].  out0 = E4M3 bytes of elements 0..3,
    // out1 = elements 4..7 (element order = byte order).
    template <bool = false>
    __device__ __forceinline__ void dequant8(uint32_t w, uint32_t& out0, uint32_t& out1) const {
        uint32_t lo3 = w & 0x77777777u;                               // low three bits: entry within a half table
        uint32_t pick = ((w >> 1) & 0x44444444u) | 0x32103210u;      // bit 3 chooses the half table
        uint32_t a0 = prmt(t[0], t[1], lo3);
        uint32_t b0 = prmt(t[2], t[3], lo3);
        out0 = prmt(a0, b0, pick);
        uint32_t lo3h = high_half(lo3), pickh = high_half(pick);
        uint32_t a1 = prmt(t[0], t[1], lo3h);
        uint32_t b1 = prmt(t[2], t[3], lo3h);
        out1 = prmt(a1, b1, pickh);
    }
};

}  // namespace w4a8
