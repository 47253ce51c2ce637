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

// Codes of a 128 x 128 tile in shared memory without swizzle (K or V^T as the A operand): 8 rows x 16 bytes (a 32-element block) form a core matrix of
// 128 bytes.  Strides that are no multiple of 128 keep the stores free of bank conflicts: lanes that write one row of
// eight row groups (V^T) or eight rows of one block (K) meet 32 different banks.
constexpr uint32_t kARowGroup = 144, kABlock = 16 * kARowGroup + 32;
__device__ __forceinline__ uint32_t a_offset(uint32_t row, uint32_t blk) { return blk * kABlock + (row >> 3) * kARowGroup + (row & 7u) * 16u; }

// A V tile in flight: a lane takes eight channels of eight neighbouring keys, a warp 64 channels of a 32-key block (full
// 128-byte lines per load), eight warps the tile.  Codes go to `a` (layout above, row = channel), scale bytes to `sf` (one
// 512-byte scale tile).
struct VTileLane {
    int ch, key;             // first channel and first key of the lane inside the tile
    int kg, blk;             // group of eight keys inside the block, block inside the tile
    __device__ __forceinline__ VTileLane(int warp, int lane)
    {
        kg = lane >> 3;
        blk = warp >> 1;
        ch = (warp & 1) * 64 + (lane & 7) * 8;
        key = blk * 32 + kg * 8;
    }
};
__device__ __forceinline__ void mxfp4_v_tile(const uint4 (&vv)[8], const VTileLane& L, uint8_t* a, uint8_t* sf)
{
    uint32_t w[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i) { w[i][0] = vv[i].x; w[i][1] = vv[i].y; w[i][2] = vv[i].z; w[i][3] = vv[i].w; }
    // a channel pair per word: block maxima over the four lanes that share the channels
    uint32_t fields[4];
#pragma unroll
    for (int p = 0; p < 4; ++p)
        fields[p] = bf16x2_absmax(bf16x2_absmax(bf16x2_absmax(w[0][p], w[1][p]), bf16x2_absmax(w[2][p], w[3][p])),
                                  bf16x2_absmax(bf16x2_absmax(w[4][p], w[5][p]), bf16x2_absmax(w[6][p], w[7][p])));
#pragma unroll
    for (int p = 0; p < 4; ++p) fields[p] = bf16x2_absmax(fields[p], __shfl_xor_sync(0xffffffffu, fields[p], 8));
#pragma unroll
    for (int p = 0; p < 4; ++p) fields[p] = mxfp4_fields(bf16x2_absmax(fields[p], __shfl_xor_sync(0xffffffffu, fields[p], 16)));
    uint8_t* const dst = a + a_offset(L.ch, L.blk) + L.kg * 4;
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        const uint32_t s2 = mxfp4_scales(fields[p]);
        uint32_t e[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) e[i] = bf16x2_mul(w[i][p], s2);
        *reinterpret_cast<uint32_t*>(dst + 32 * p) = e2m1_word(bf16_lo(e[0]), bf16_lo(e[1]), bf16_lo(e[2]), bf16_lo(e[3]),
                                                               bf16_lo(e[4]), bf16_lo(e[5]), bf16_lo(e[6]), bf16_lo(e[7]));
        *reinterpret_cast<uint32_t*>(dst + 32 * p + 16) = e2m1_word(bf16_hi(e[0]), bf16_hi(e[1]), bf16_hi(e[2]), bf16_hi(e[3]),
                                                                    bf16_hi(e[4]), bf16_hi(e[5]), bf16_hi(e[6]), bf16_hi(e[7]));
    }
    // scale bytes: lane group kg writes channel pair kg
    const uint32_t f = L.kg < 2 ? (L.kg == 0 ? fields[0] : fields[1]) : (L.kg == 2 ? fields[2] : fields[3]);
    uint8_t* const d = sf + sf_tile_offset(L.ch + 2 * L.kg, L.blk);
    d[0] = static_cast<uint8_t>(mxfp4_byte_lo(f));
    d[16] = static_cast<uint8_t>(mxfp4_byte_hi(f));
}

// 16-byte chunk (one block) of a 64-byte code row in a shared-memory operand tile (64-byte swizzle)
__device__ __forceinline__ uint32_t code_tile_offset(uint32_t row, uint32_t chunk)
{
    return (row >> 3) * 512u + (row & 7u) * 64u + ((chunk ^ ((row >> 1) & 3u)) << 4);
}

}  // namespace efq
