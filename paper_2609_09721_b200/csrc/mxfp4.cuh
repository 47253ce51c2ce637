// bf16 -> MXFP4 of one 32-element block in registers, and the places of a row's codes and scale byte in the operand tiles
// that the block-scaled MMAs read.  Shared by the operand preparation and the few-query forward.
#pragma once

#include "efq_common.cuh"

namespace efq {

// 32 bf16 values (as 16 packed 32-bit words, element 2u in the low half) -> 16 bytes of codes + scale byte
__device__ __forceinline__ void mxfp4_block(const uint32_t (&w)[16], uint4& codes, uint32_t& byte)
{
    uint32_t two = 0;    // bf16 magnitudes compare like unsigned integers: both halves of a word at once
#pragma unroll
    for (int i = 0; i < 16; ++i) two = __vmaxu2(two, w[i] & 0x7fff7fffu);
    const uint32_t amax = max(two & 0xffffu, two >> 16);
    if (amax == 0) {
        codes = make_uint4(0, 0, 0, 0);
        byte = 0;
        return;
    }
    int e = static_cast<int>(amax >> 7) - 127 - 2;   // exponent field of the largest magnitude, minus 2
    e = max(e, -127);
    const float s = __uint_as_float(static_cast<uint32_t>(127 - e) << 23);   // 2^-e, field in [2, 254]
    uint32_t out[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        uint32_t word = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            uint32_t v = w[q * 4 + i];
            const float lo = __uint_as_float(v << 16) * s;
            const float hi = __uint_as_float(v & 0xffff0000u) * s;
            word |= (cvt_e2m1x2(lo, hi) & 0xffu) << (8 * i);
        }
        out[q] = word;
    }
    codes = make_uint4(out[0], out[1], out[2], out[3]);
    byte = static_cast<uint32_t>(e + 127);
}

// byte of (row r, 32-element block b) in a 512-byte scale tile of 128 rows
__device__ __forceinline__ uint32_t sf_tile_offset(uint32_t r, uint32_t b) { return (r & 31u) * 16u + (r >> 5) * 4u + b; }

// 16-byte chunk (one block) of a 64-byte code row in a shared-memory operand tile (64-byte swizzle)
__device__ __forceinline__ uint32_t code_tile_offset(uint32_t row, uint32_t chunk)
{
    return (row >> 3) * 512u + (row & 7u) * 64u + ((chunk ^ ((row >> 1) & 3u)) << 4);
}

}  // namespace efq
