// bf16 -> MXFP4 of one 32-element block in registers, and the places of a row's codes and scale byte in the operand tiles
// that the block-scaled MMAs read.  Shared by the operand preparation and the few-query forward.
#pragma once

#include "efq_common.cuh"

namespace efq {

// Larger magnitudes of the two halves of two words (the signs of the result mean nothing); a NaN wins.
__device__ __forceinline__ uint32_t bf16x2_absmax(uint32_t a, uint32_t b)
{
    uint32_t d;
    asm("max.NaN.xorsign.abs.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}

// Product of packed bf16 pairs; exact where one factor is a power of two.
__device__ __forceinline__ uint32_t bf16x2_mul(uint32_t a, uint32_t b)
{
    uint32_t d;
    asm("mul.rn.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}

__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }

// Eight scaled elements -> eight codes, e0 in bits 0-3.  The conversions and the gathering of their bytes are one asm block
// so that the bytes land in the word without shifts.
__device__ __forceinline__ uint32_t e2m1_word(float e0, float e1, float e2, float e3, float e4, float e5, float e6, float e7)
{
    uint32_t out;
    asm("{\n\t.reg .b8 b0, b1, b2, b3;\n\t"
        "cvt.rn.satfinite.e2m1x2.f32 b0, %2, %1;\n\t"
        "cvt.rn.satfinite.e2m1x2.f32 b1, %4, %3;\n\t"
        "cvt.rn.satfinite.e2m1x2.f32 b2, %6, %5;\n\t"
        "cvt.rn.satfinite.e2m1x2.f32 b3, %8, %7;\n\t"
        "mov.b32 %0, {b0, b1, b2, b3};\n\t}\n"
        : "=r"(out) : "f"(e0), "f"(e1), "f"(e2), "f"(e3), "f"(e4), "f"(e5), "f"(e6), "f"(e7));
    return out;
}

// Shared exponents of two blocks at once, from the packed magnitudes of their largest elements: field is the exponent field
// (in place, at least 2), the scale byte of a block is its field - 2 (e = field - 129 >= -127), and the elements are taken
// times 2^-e, returned as packed bf16.
__device__ __forceinline__ uint32_t mxfp4_fields(uint32_t amax2)
{
    uint32_t d;
    asm("max.u16x2 %0, %1, %2;" : "=r"(d) : "r"(amax2 & 0x7f807f80u), "r"(0x01000100u));
    return d;
}
__device__ __forceinline__ uint32_t mxfp4_scales(uint32_t fields) { return 0x80008000u - fields; }
__device__ __forceinline__ uint32_t mxfp4_byte_lo(uint32_t fields) { return ((fields & 0xffffu) >> 7) - 2u; }
__device__ __forceinline__ uint32_t mxfp4_byte_hi(uint32_t fields) { return (fields >> 23) - 2u; }

// 32 bf16 values (as 16 packed 32-bit words, element 2u in the low half) -> 16 bytes of codes + scale byte.
// About 90 instructions, 40 fewer than with a float multiplication per element and shifted bytes.
__device__ __forceinline__ void mxfp4_block(const uint32_t (&w)[16], uint4& codes, uint32_t& byte)
{
    uint32_t two = bf16x2_absmax(w[0], w[1]);
#pragma unroll
    for (int i = 2; i < 16; ++i) two = bf16x2_absmax(two, w[i]);
    two = bf16x2_absmax(two, __byte_perm(two, two, 0x1032));
    const uint32_t fields = mxfp4_fields(two), s2 = mxfp4_scales(fields);
    uint32_t out[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const uint32_t a = bf16x2_mul(w[4 * q], s2), b = bf16x2_mul(w[4 * q + 1], s2), c = bf16x2_mul(w[4 * q + 2], s2), d = bf16x2_mul(w[4 * q + 3], s2);
        out[q] = e2m1_word(bf16_lo(a), bf16_hi(a), bf16_lo(b), bf16_hi(b), bf16_lo(c), bf16_hi(c), bf16_lo(d), bf16_hi(d));
    }
    codes = make_uint4(out[0], out[1], out[2], out[3]);
    if ((two & 0x7fffu) == 0u) codes = make_uint4(0, 0, 0, 0);       // negative zeros too
    byte = mxfp4_byte_lo(fields);
}

// byte of (row r, 32-element block b) in a 512-byte scale tile of 128 rows
__device__ __forceinline__ uint32_t sf_tile_offset(uint32_t r, uint32_t b) { return (r & 31u) * 16u + (r >> 5) * 4u + b; }

// 16-byte chunk (one block) of a 64-byte code row in a shared-memory operand tile (64-byte swizzle)
__device__ __forceinline__ uint32_t code_tile_offset(uint32_t row, uint32_t chunk)
{
    return (row >> 3) * 512u + (row & 7u) * 64u + ((chunk ^ ((row >> 1) & 3u)) << 4);
}

}  // namespace efq
