// Probability producers for one 32-key microscaling block held in registers: the EFQ rule (Algorithm 1)
// and the exp-then-quantize comparison producer.  Shared by the fused forward and the in-SM microbenchmark.
#pragma once

#include "efq_common.cuh"

namespace efq {

__device__ __forceinline__ float max3(float a, float b, float c)
{
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
__device__ __forceinline__ float fma_sat(float a, float b, float c)
{
    float d;
    asm("fma.rn.sat.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
__device__ __forceinline__ uint64_t pack2(float lo, float hi)
{
    uint64_t d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
    return d;
}

// Largest of 32 scores with 3-input maxima.
__device__ __forceinline__ float block_max32(const float* r)
{
    float m[11];
#pragma unroll
    for (int i = 0; i < 10; ++i) m[i] = max3(r[3 * i], r[3 * i + 1], r[3 * i + 2]);
    m[10] = fmaxf(r[30], r[31]);
    const float a = max3(m[0], m[1], m[2]), b = max3(m[3], m[4], m[5]), c = max3(m[6], m[7], m[8]);
    return max3(max3(a, b, c), m[9], m[10]);
}

// 32 scores of one microscaling block -> 16 bytes of codes + scale byte.
// PRODUCER: 0 = EFQ (affine rule), 1 / 2 = exp-then-quantize with the block maximum in [4, 8) / (3, 6],
// 3 = EFQ-LUT, 4 = exp-then-quantize [4, 8) with the scale folded into the exponential, 5 = the same with 2 of 8
// exponentials computed by a polynomial on the FMA pipe, 6 = producer 1 that also adds its 32 FP32 exponentials to
// *psum (for the baseline whose denominator is the sum of the exponentials instead of the quantised operand).
//
// EFQ (Algorithm 1), two FMA-pipe instructions and half a pack per element, bit-identical to
// c = floor(min(max(fma(r, A, Bb), 0), 7)):
//   w = fma.rn.sat(r, A/8, Bb/8) = clamp(fma(r, A, Bb), 0, 8) / 8     (scaling by 2^-3 commutes with rounding)
//   mul.rm(w, 2^-146)            = floor(8 w) 2^-149                  (a subnormal, whose bits are the integer itself)
//   cvt.pack.sat.s4              two integers to two nibbles behind the ones packed before; 8 (only when the affine form
//                                reaches 8) saturates to 7
// Measured against four codes accumulated Horner-style in a mantissa by packed FMAs (0.75 more FMA-pipe instructions per
// element, and a masked subtraction per word for the 8): 604 against 727 cycles per 128 x 128 tile with two warps per
// scheduler, block maxima and operand stores included.
template <int PRODUCER>
__device__ __forceinline__ void produce32(const float* r, float rmax, float m_s, const ProducerConsts& K, uint4& codes,
                                          uint32_t& byte, float* psum = nullptr)
{
    uint32_t w[4];
    if (PRODUCER == 0) {
        BlockScale s = efq_block_scale(rmax, m_s, K);
        byte = s.byte;
        const float A8 = K.A * 0.125f, B8 = s.Bb * 0.125f;
        const float to_bits = __uint_as_float(8u);       // 2^-146
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            uint32_t c[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                float t;
                asm("mul.rm.f32 %0, %1, %2;" : "=f"(t) : "f"(fma_sat(r[q * 8 + i], A8, B8)), "f"(to_bits));
                c[i] = __float_as_uint(t);
            }
            uint32_t word = 0u;
#pragma unroll
            for (int i = 3; i >= 0; --i) asm("cvt.pack.sat.s4.s32.b32 %0, %1, %2, %0;" : "+r"(word) : "r"(c[2 * i + 1]), "r"(c[2 * i]));
            w[q] = word;   // a block without a finite score has w = 0 everywhere (sat(-inf) and sat(NaN) are 0)
        }
    } else if (PRODUCER == 3) {
        // LUT variant: the same block scale, 16-level index, folding table (one element at a time: the
        // accuracy-oriented comparison point of the paper, not the fast path)
        BlockScale s = efq_block_scale(rmax, m_s, K);
        byte = s.byte;
        const float A16 = K.A * 0.0625f, B16 = s.Bb * 0.0625f;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            uint32_t word = 0;
#pragma unroll
            for (int i = 0; i < 8; ++i) word |= lut_code(r[q * 8 + i], A16, B16) << (4 * i);
            w[q] = word;
        }
    } else if (PRODUCER == 4 || PRODUCER == 5) {
        // exp-then-quantize (block maximum in [4, 8)) with the scale folded into the exponential: one FMA, one ex2
        // and half a conversion per element; bound by the exponential unit.  PRODUCER 5 moves 2 of every 8
        // exponentials onto the FMA pipe (cubic polynomial).
        const FoldedScale f = etq_folded_scale(rmax, m_s, K);
        byte = f.byte;
        auto ex2 = [&](const int i) {
            const float t = __fmaf_rn(r[i], f.c1, f.c0e);
            return (PRODUCER == 5 && ex2_by_poly(i)) ? ex2_poly3(t) : ex2_approx(t);
        };
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint32_t word = e2m1_word(ex2(q * 8), ex2(q * 8 + 1), ex2(q * 8 + 2), ex2(q * 8 + 3), ex2(q * 8 + 4), ex2(q * 8 + 5),
                                            ex2(q * 8 + 6), ex2(q * 8 + 7));
            w[q] = f.live ? word : 0u;
        }
    } else {
        float p[32];
        float sum = 0.0f;
#pragma unroll
        for (int i = 0; i < 32; ++i) {
            float x = __fsub_rn(__fmul_rn(K.sigma, r[i]), m_s);
            p[i] = ex2_approx(__fmul_rn(x, K.LOG2E));
            if (PRODUCER == 6) sum += p[i];       // masked scores (-inf) give exactly 0
        }
        if (PRODUCER == 6) *psum += sum;
        const float amax = fmaxf(block_max32(p), 0.0f);      // a row without a finite score has NaN everywhere: 0
        if (amax == 0.0f) {
            byte = 0;
            w[0] = w[1] = w[2] = w[3] = 0;
        } else {
            const uint32_t bits = __float_as_uint(amax);
            const int E = static_cast<int>((bits >> 23) & 0xffu) - 127;
            int e = (PRODUCER == 1 || PRODUCER == 6) ? E - 2 : ((bits & 0x7fffffu) > 0x400000u ? E - 1 : E - 2);
            e = max(e, -127);
            const float s = __uint_as_float(static_cast<uint32_t>(127 - e) << 23);
            byte = static_cast<uint32_t>(e + 127);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float* x = p + q * 8;
                const uint32_t word = e2m1_word(x[0] * s, x[1] * s, x[2] * s, x[3] * s, x[4] * s, x[5] * s, x[6] * s, x[7] * s);
                w[q] = word;
            }
        }
    }
    codes = make_uint4(w[0], w[1], w[2], w[3]);
}

}  // namespace efq
