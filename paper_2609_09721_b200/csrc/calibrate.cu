// Offline selection of the affine rule's parameters (Algorithm 3, Sec. "Parameter Calibration") and its helpers:
//   efq_exact_attention_fwd   softmax attention in FP32 on the unquantised bf16 inputs: the reference output O_ref
//                             of the calibration objective, and the "exact" side of every error figure reported;
//   efq_relative_error        rho = ||A - R||_F / ||R||_F, the objective itself (sums kept in double);
//   efq_calibrate             the grid search: operands quantised once, one fused forward per candidate (tau, h),
//                             rho of each, the first minimum in scan order.
// None of this is on the inference path: the selected pair stays fixed afterwards.
//
// The reference attention keeps FP32 throughout on the bf16 tensor cores: products of bf16 numbers are exact in the FP32
// accumulator, so Q K^T needs one MMA pass, and the FP32 probabilities are split into three bf16 terms (8 + 8 + 8
// significant bits) whose products with V are exact too, so P V needs three.  The product of a tile is taken from a fresh
// accumulator and added to the row's sum in registers, in FP32 with rounding.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <atomic>
#include <vector>

#include "efq_common.cuh"
#include "efq_internal.cuh"
#include "sm100_ptx.cuh"

namespace efq {
namespace {

constexpr int kD = 128;
constexpr int kTile = 128;                   // query rows per CTA, keys per step
constexpr int kHalfBytes = kTile * 128;      // 128 rows of 64 bf16 channels
constexpr uint32_t kColS = 0, kColP = 128, kColO = 320;      // scores | three terms of P, two keys per column | P V of the tile

struct __align__(1024) ExactSmem {
    uint8_t q[2][kHalfBytes], k[2][kHalfBytes], v[2][kHalfBytes];       // [channels 0-63, 64-127], 128-byte swizzle
    float tile_max[2][2][kTile];             // [step mod 2][half of the keys][row]
    float l_half[2][kTile];
    uint64_t q_full, k_full, v_full, s_done, o_done;
    uint32_t tmem_base;
    volatile uint32_t failed;
};

// Bounded (20000 polls, 0.07 s when nothing comes); on expiry the block is marked as failed, which ends its other waits too.  What depends on the wait -
// a load into the buffer, an MMA - is left out after a false: a barrier whose phase has not ended must not get another arrival.
__device__ __forceinline__ bool wait_for(uint64_t* bar, uint32_t parity, ExactSmem* sm)
{
    if (ptx::mbar_try_wait(bar, parity)) return true;
    for (int i = 0; i < 20000; ++i) {
        if (ptx::mbar_try_wait_suspend(bar, parity, 50000u)) return true;
        if (sm->failed != 0u) return false;
    }
    sm->failed = 1u;
    return false;
}

__device__ __forceinline__ uint32_t bf16_pair(float lo, float hi)
{
    uint32_t d;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
    return d;
}

// 256 threads: thread = (query row, half of the keys for the scores and half of the channels for the output).  The step is a
// serial chain (scores, maxima, exponentials, P V, add), but S of the next step runs beside P V, and K and V of the next step
// load while the tensor core and the exponentials do not need their buffer.
__global__ void __launch_bounds__(256, 1)
exact_attention_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                       float* __restrict__ o, int heads, int Hq, int Hkv, int Sq, int Sk, int causal, float sigma, int inject_skip_loads)
{
    extern __shared__ uint8_t smem_raw[];
    ExactSmem* const sm = reinterpret_cast<ExactSmem*>(smem_raw + ptx::smem_round_up(smem_raw, 1024u));
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int bh = static_cast<int>(blockIdx.x % static_cast<unsigned>(heads)), hkv_row = (bh / Hq) * Hkv + (bh % Hq) / (Hq / Hkv);
    const int q0 = static_cast<int>((gridDim.x - 1u - blockIdx.x) / static_cast<unsigned>(heads)) * kTile;      // long rows first
    int n_steps = (Sk + kTile - 1) / kTile;
    if (causal) {
        const int last_key = min(q0 + kTile, Sq) - 1 + Sk - Sq;
        n_steps = min(n_steps, last_key < 0 ? 0 : last_key / kTile + 1);
    }
    const int half = warp >> 2, row = (warp & 3) * 32 + lane;
    float* const dst = o + (static_cast<int64_t>(bh) * Sq + q0 + row) * kD + 64 * half;
    const bool row_valid = q0 + row < Sq;
    if (n_steps == 0) {                      // nothing visible: zero rows
        if (row_valid)
            for (int i = 0; i < 16; ++i) reinterpret_cast<float4*>(dst)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        return;
    }
    auto load_pair = [&](uint8_t (*buf)[kHalfBytes], const CUtensorMap* map, int y, uint64_t* bar) {
        ptx::mbar_arrive_expect_tx(bar, 2 * kHalfBytes);
        ptx::tma_load_2d(buf[0], map, 0, y, bar);
        ptx::tma_load_2d(buf[1], map, 64, y, bar);
    };
    if (warp == 0) ptx::tmem_alloc(&sm->tmem_base, 512);
    if (tid == 32) {
        sm->failed = 0u;
        ptx::mbar_init(&sm->q_full, 1);
        ptx::mbar_init(&sm->k_full, 1);
        ptx::mbar_init(&sm->v_full, 1);
        ptx::mbar_init(&sm->s_done, 1);
        ptx::mbar_init(&sm->o_done, 1);
        ptx::mbar_init_fence();
        load_pair(sm->q, &map_q, bh * Sq + q0, &sm->q_full);
        if (!inject_skip_loads) {
            load_pair(sm->k, &map_k, hkv_row * Sk, &sm->k_full);
            load_pair(sm->v, &map_v, hkv_row * Sk, &sm->v_full);
        }
    }
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::tc_fence_after_sync();
    const uint32_t tmem = sm->tmem_base;
    const uint32_t lane_base = static_cast<uint32_t>((warp & 3) * 32) << 16;
    // S = Q K^T: both operands K-major (channels), eight steps of 16 channels
    auto issue_s = [&]() {
        const uint64_t da = ptx::smem_desc(ptx::smem_u32(sm->q[0]), 16, 1024, ptx::kLayoutSw128), db = ptx::smem_desc(ptx::smem_u32(sm->k[0]), 16, 1024, ptx::kLayoutSw128);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const uint64_t off = static_cast<uint64_t>(((i >> 2) * kHalfBytes + (i & 3) * 32) >> 4);
            ptx::mma_bf16(tmem + kColS, da + off, db + off, ptx::bf16_idesc(128, false), i > 0 ? 1u : 0u);
        }
        ptx::mma_commit(&sm->s_done);
    };
    // P V: P from tensor memory, V with the channels contiguous (transposed operand), three terms of eight steps of 16 keys
    auto issue_pv = [&]() {
        const uint64_t dv = ptx::smem_desc(ptx::smem_u32(sm->v[0]), kHalfBytes, 1024, ptx::kLayoutSw128);
#pragma unroll
        for (int t = 0; t < 3; ++t)
#pragma unroll
            for (int i = 0; i < 8; ++i)
                ptx::mma_bf16_ts(tmem + kColO, tmem + kColP + 64 * t + 8 * i, dv + static_cast<uint64_t>(i * 2048 >> 4), ptx::bf16_idesc(128, true), t + i > 0 ? 1u : 0u);
        ptx::mma_commit(&sm->o_done);
    };
    const int limit = min(causal ? q0 + row + Sk - Sq : Sk - 1, Sk - 1);      // last visible key of the row
    float m = -INFINITY, l = 0.0f;
    float acc[64];
#pragma unroll
    for (int i = 0; i < 64; ++i) acc[i] = 0.0f;
    if (warp == 0) {
        const bool ok = __all_sync(0xffffffffu, wait_for(&sm->q_full, 0, sm) && wait_for(&sm->k_full, 0, sm));
        ptx::tc_fence_after_sync();
        if (ok && ptx::elect_one()) issue_s();
        __syncwarp();
    }
    int k_loads = inject_skip_loads ? 0 : 1, v_loads = k_loads;       // what thread 32 has asked for
    for (int j = 0; j < n_steps; ++j) {
        const uint32_t ph = j & 1;
        const bool s_ready = wait_for(&sm->s_done, ph, sm);
        ptx::tc_fence_after_sync();
        if (tid == 32 && s_ready && j + 1 < n_steps) {
            load_pair(sm->k, &map_k, hkv_row * Sk + (j + 1) * kTile, &sm->k_full);
            ++k_loads;
        }
        const int key0 = j * kTile + 64 * half;
        float s[64];
        ptx::tmem_ld32f<0>(tmem + lane_base + kColS + 64 * half, s);
        ptx::tmem_ld32f<32>(tmem + lane_base + kColS + 64 * half + 32, s);
        ptx::tmem_wait_ld();
        float mx = -INFINITY;
#pragma unroll
        for (int i = 0; i < 64; ++i) {
            s[i] = key0 + i <= limit ? s[i] * sigma : -INFINITY;
            mx = fmaxf(mx, s[i]);
        }
        sm->tile_max[ph][half][row] = mx;
        if (Sk - j * kTile < kTile) {        // rows of V past the sequence belong to somebody else: 0 x anything has to be 0
            wait_for(&sm->v_full, ph, sm);
            for (int i = tid; i < 2 * kTile * 8; i += 256) {
                const int r = (i >> 3) & (kTile - 1);
                if (r >= Sk - j * kTile) reinterpret_cast<uint4*>(sm->v[i >> 10])[(r << 3) + (i & 7)] = make_uint4(0, 0, 0, 0);
            }
            ptx::fence_proxy_async_smem();
        }
        __syncthreads();
        if (sm->failed != 0u) break;         // the same for all: nobody waits, and so nobody fails, between the two barriers
        const float m_new = fmaxf(m, fmaxf(sm->tile_max[ph][0][row], sm->tile_max[ph][1][row]));
        const float alpha = m == -INFINITY ? 0.0f : expf(m - m_new);
        const float base = m_new == -INFINITY ? 0.0f : m_new;        // nothing visible yet: every exponential is exp(-inf) = 0
        m = m_new;
        float sum = 0.0f;
        uint32_t t1[32], t2[32], t3[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) {
            const float p0 = expf(s[2 * i] - base), p1 = expf(s[2 * i + 1] - base);
            sum += p0;
            sum += p1;
            t1[i] = bf16_pair(p0, p1);
            const float r0 = p0 - __uint_as_float(t1[i] << 16), r1 = p1 - __uint_as_float(t1[i] & 0xffff0000u);
            t2[i] = bf16_pair(r0, r1);
            t3[i] = bf16_pair(r0 - __uint_as_float(t2[i] << 16), r1 - __uint_as_float(t2[i] & 0xffff0000u));
        }
        l = l * alpha + sum;
        ptx::tmem_st32<0>(tmem + lane_base + kColP + 32 * half, t1);
        ptx::tmem_st32<0>(tmem + lane_base + kColP + 64 + 32 * half, t2);
        ptx::tmem_st32<0>(tmem + lane_base + kColP + 128 + 32 * half, t3);
        ptx::tmem_wait_st();
        ptx::tc_fence_before_sync();
        __syncthreads();
        if (warp == 0) {
            const bool ok = __all_sync(0xffffffffu, wait_for(&sm->v_full, ph, sm) && (j + 1 == n_steps || wait_for(&sm->k_full, ph ^ 1u, sm)));
            ptx::tc_fence_after_sync();
            if (ok && ptx::elect_one()) {
                issue_pv();
                if (j + 1 < n_steps) issue_s();
            }
            __syncwarp();
        }
        const bool o_ready = wait_for(&sm->o_done, ph, sm);
        ptx::tc_fence_after_sync();
        if (tid == 32 && o_ready && j + 1 < n_steps) {
            load_pair(sm->v, &map_v, hkv_row * Sk + (j + 1) * kTile, &sm->v_full);
            ++v_loads;
        }
        float d[64];
        ptx::tmem_ld32f<0>(tmem + lane_base + kColO + 64 * half, d);
        ptx::tmem_ld32f<32>(tmem + lane_base + kColO + 64 * half + 32, d);
        ptx::tmem_wait_ld();
        ptx::tc_fence_before_sync();
#pragma unroll
        for (int i = 0; i < 64; ++i) acc[i] = fmaf(acc[i], alpha, d[i]);
    }
    if (tid == 32 && sm->failed != 0u) {     // its own copies in flight end before the block does
        auto landed = [](uint64_t* bar, int loads) {
            for (int i = 0; loads > 0 && i < 1000 && !ptx::mbar_try_wait_suspend(bar, (loads - 1) & 1, 50000u); ++i) {}
        };
        landed(&sm->q_full, 1);
        landed(&sm->k_full, k_loads);
        landed(&sm->v_full, v_loads);
    }
    sm->l_half[half][row] = l;
    __syncthreads();
    const float total = sm->l_half[0][row] + sm->l_half[1][row];
    const float inv = sm->failed != 0u ? __uint_as_float(0x7fc00000u) : total > 0.0f ? 1.0f / total : 0.0f;     // a failed wait: NaN, not a wrong number
    if (row_valid) {
#pragma unroll
        for (int i = 0; i < 16; ++i)
            reinterpret_cast<float4*>(dst)[i] = make_float4(acc[4 * i] * inv, acc[4 * i + 1] * inv, acc[4 * i + 2] * inv, acc[4 * i + 3] * inv);
    }
    ptx::tc_fence_before_sync();
    __syncthreads();
    if (warp == 0) ptx::tmem_dealloc(tmem, 512);
}

// sums[0] += sum (a - r)^2, sums[1] += sum r^2, in double.  Bound by the reads (from L2 where both arrays fit): 16 bytes per
// load, four loads in flight per thread.  Its blocks may be there before the kernel that makes the rows is done: no read-only loads.
__global__ void __launch_bounds__(256) error_sums_kernel(const float* __restrict__ a, const float* __restrict__ r,
                                                         int64_t n, double* sums)
{
    ptx::grid_wait();
    ptx::grid_launch_next();
    double d2 = 0.0, r2 = 0.0;
    auto add = [&](float af, float rf) {
        const double x = static_cast<double>(af), y = static_cast<double>(rf);
        d2 += (x - y) * (x - y);
        r2 += y * y;
    };
    const int64_t thread = static_cast<int64_t>(blockIdx.x) * 256 + threadIdx.x, threads = static_cast<int64_t>(gridDim.x) * 256;
    const bool vec = ((reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(r)) & 15u) == 0;
    const int64_t n4 = vec ? n / 4 : 0;
    int64_t i = thread;
    for (; i + threads < n4; i += 2 * threads) {
        const float4 x0 = __ldcg(reinterpret_cast<const float4*>(a) + i), x1 = __ldcg(reinterpret_cast<const float4*>(a) + i + threads);
        const float4 y0 = __ldcg(reinterpret_cast<const float4*>(r) + i), y1 = __ldcg(reinterpret_cast<const float4*>(r) + i + threads);
        add(x0.x, y0.x); add(x0.y, y0.y); add(x0.z, y0.z); add(x0.w, y0.w);
        add(x1.x, y1.x); add(x1.y, y1.y); add(x1.z, y1.z); add(x1.w, y1.w);
    }
    if (i < n4) {
        const float4 x = __ldcg(reinterpret_cast<const float4*>(a) + i), y = __ldcg(reinterpret_cast<const float4*>(r) + i);
        add(x.x, y.x); add(x.y, y.y); add(x.z, y.z); add(x.w, y.w);
    }
    for (int64_t k = 4 * n4 + thread; k < n; k += threads) add(__ldcg(a + k), __ldcg(r + k));
    for (int off = 16; off > 0; off >>= 1) {
        d2 += __shfl_xor_sync(0xffffffffu, d2, off);
        r2 += __shfl_xor_sync(0xffffffffu, r2, off);
    }
    __shared__ double sd[8], sr[8];
    if ((threadIdx.x & 31) == 0) { sd[threadIdx.x >> 5] = d2; sr[threadIdx.x >> 5] = r2; }
    __syncthreads();
    if (threadIdx.x == 0) {
        double td = 0.0, tr = 0.0;
        for (int w = 0; w < 8; ++w) { td += sd[w]; tr += sr[w]; }
        atomicAdd(&sums[0], td);
        atomicAdd(&sums[1], tr);
    }
}

bool is_sm100()
{
    int dev = 0, major = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return false;
    if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess) return false;
    return major == 10;
}

}  // namespace
}  // namespace efq

static efq_status_t exact_attention(const void* q, const void* k, const void* v, float* o, int B, int Hq, int Hkv, int64_t Sq, int64_t Sk, int d,
                                    int causal, float softmax_scale, void* stream, bool inject_skip_loads)
{
    if (!q || !k || !v || !o) return EFQ_ERR_INVALID_ARG;
    if (B <= 0 || Hq <= 0 || Hkv <= 0 || Sq <= 0 || Sk <= 0 || Hq % Hkv != 0) return EFQ_ERR_INVALID_ARG;
    if (d != 128) return EFQ_ERR_UNSUPPORTED;
    if ((reinterpret_cast<uintptr_t>(q) | reinterpret_cast<uintptr_t>(k) | reinterpret_cast<uintptr_t>(v) |
         reinterpret_cast<uintptr_t>(o)) & 15u)
        return EFQ_ERR_ALIGNMENT;
    if (static_cast<int64_t>(B) * Hq > 65535) return EFQ_ERR_UNSUPPORTED;
    if (!efq::is_sm100()) return EFQ_ERR_ARCH;
    const float sigma = softmax_scale > 0.0f ? softmax_scale : 0.08838834764831845f;
    const int64_t rows_q = static_cast<int64_t>(B) * Hq * Sq, rows_k = static_cast<int64_t>(B) * Hkv * Sk, q_tiles = (Sq + efq::kTile - 1) / efq::kTile;
    if (rows_q >= (1ll << 31) - 128 || rows_k >= (1ll << 31) - 128 || q_tiles * B * Hq >= (1ll << 31)) return EFQ_ERR_UNSUPPORTED;      // 32-bit tile coordinates
    constexpr int smem = static_cast<int>(sizeof(efq::ExactSmem)) + 1024;
    static std::atomic<uint64_t> done{0};        // the shared-memory attribute belongs to the device: set once for each
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return EFQ_ERR_CUDA;
    if ((done.load(std::memory_order_relaxed) >> dev & 1u) == 0u) {
        if (cudaFuncSetAttribute(efq::exact_attention_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess) return EFQ_ERR_CUDA;
        done.fetch_or(1ull << dev, std::memory_order_relaxed);
    }
    CUtensorMap mq, mk, mv;
    if (!efq::encode_bf16_map(&mq, q, 128, static_cast<uint64_t>(rows_q)) || !efq::encode_bf16_map(&mk, k, 128, static_cast<uint64_t>(rows_k)) ||
        !efq::encode_bf16_map(&mv, v, 128, static_cast<uint64_t>(rows_k)))
        return EFQ_ERR_CUDA;
    const dim3 grid(static_cast<unsigned>(q_tiles * B * Hq));
    efq::exact_attention_kernel<<<grid, 256, smem, static_cast<cudaStream_t>(stream)>>>(mq, mk, mv, o, B * Hq, Hq, Hkv, static_cast<int>(Sq),
                                                                                        static_cast<int>(Sk), causal ? 1 : 0, sigma,
                                                                                        inject_skip_loads ? 1 : 0);
    return cudaGetLastError() == cudaSuccess ? EFQ_OK : EFQ_ERR_CUDA;
}

extern "C" efq_status_t efq_exact_attention_fwd(const void* q, const void* k, const void* v, float* o, int B, int Hq,
                                                int Hkv, int64_t Sq, int64_t Sk, int d, int causal,
                                                float softmax_scale, void* stream)
{
    return exact_attention(q, k, v, o, B, Hq, Hkv, Sq, Sk, d, causal, softmax_scale, stream, false);
}

extern "C" efq_status_t efq_exact_attention_fwd_inject_timeout(const void* q, const void* k, const void* v, float* o, int B, int Hq, int Hkv,
                                                               int64_t Sq, int64_t Sk, int d, void* stream)
{
    return exact_attention(q, k, v, o, B, Hq, Hkv, Sq, Sk, d, 0, 0.0f, stream, true);
}

static cudaError_t launch_error_sums(const float* a, const float* ref, int64_t n, double* sums, cudaStream_t s)
{
    int64_t blocks = (n + 2047) / 2048;
    if (blocks > 148 * 8) blocks = 148 * 8;
    return efq::launch_overlapped(efq::error_sums_kernel, dim3(static_cast<unsigned>(blocks)), 256, 0, s, a, ref, n, sums);
}

extern "C" efq_status_t efq_relative_error(const float* a, const float* ref, int64_t n, double* sums, void* stream)
{
    if (!a || !ref || !sums || n < 0) return EFQ_ERR_INVALID_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (cudaMemsetAsync(sums, 0, 2 * sizeof(double), s) != cudaSuccess) return EFQ_ERR_CUDA;
    if (n == 0) return EFQ_OK;
    return launch_error_sums(a, ref, n, sums, s) == cudaSuccess ? EFQ_OK : EFQ_ERR_CUDA;
}

extern "C" efq_status_t efq_calibrate(const void* q, const void* k, const void* v, const float* o_ref, float* o_tmp,
                                      int B, int Hq, int Hkv, int64_t Sq, int64_t Sk, int d, int causal,
                                      float softmax_scale, const float* taus, int n_tau, const float* hs, int n_h,
                                      double* sums, double* rho, float* best_tau, float* best_h, void* workspace,
                                      size_t workspace_bytes, void* stream)
{
    if (!o_ref || !o_tmp || !taus || !hs || !sums || !rho || n_tau <= 0 || n_h <= 0) return EFQ_ERR_INVALID_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    efq_status_t st = efq_quantize_qkv(q, k, v, B, Hq, Hkv, Sq, Sk, d, workspace, workspace_bytes, stream);
    if (st != EFQ_OK) return st;
    const int64_t n = static_cast<int64_t>(B) * Hq * Sq * d;
    const int n_cand = n_tau * n_h;
    if (cudaMemsetAsync(sums, 0, 2 * static_cast<size_t>(n_cand) * sizeof(double), s) != cudaSuccess) return EFQ_ERR_CUDA;
    for (int it = 0; it < n_tau; ++it) {
        for (int ih = 0; ih < n_h; ++ih) {
            efq_params_t p;
            p.tau = taus[it];
            p.h = hs[ih];
            p.variant = 0;
            p.kv_tile = 0;
            p.rescale_threshold = 0.0f;
            st = efq_attention_fwd_quantized(o_tmp, B, Hq, Hkv, Sq, Sk, d, causal, softmax_scale, 0, &p, workspace,
                                             workspace_bytes, nullptr, stream);
            if (st != EFQ_OK) return st;
            if (launch_error_sums(o_tmp, o_ref, n, sums + 2 * (it * n_h + ih), s) != cudaSuccess) return EFQ_ERR_CUDA;
        }
    }
    std::vector<double> host(2 * static_cast<size_t>(n_cand));
    if (cudaMemcpyAsync(host.data(), sums, host.size() * sizeof(double), cudaMemcpyDeviceToHost, s) != cudaSuccess)
        return EFQ_ERR_CUDA;
    st = efq_poll_status(workspace, stream);          // synchronises the stream; reports an expired device-side wait
    if (st != EFQ_OK) return st;
    double best = INFINITY;
    if (best_tau) *best_tau = taus[0];
    if (best_h) *best_h = hs[0];
    for (int i = 0; i < n_cand; ++i) {
        rho[i] = host[2 * i + 1] > 0.0 ? sqrt(host[2 * i] / host[2 * i + 1]) : (host[2 * i] > 0.0 ? INFINITY : 0.0);
        if (rho[i] < best) {                          // strict: the first minimum in scan order (tau outer, h inner)
            best = rho[i];
            if (best_tau) *best_tau = taus[i / n_h];
            if (best_h) *best_h = hs[i % n_h];
        }
    }
    return EFQ_OK;
}
