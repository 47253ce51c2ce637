// Operand preparation for the fused forward: bf16 Q, K, V -> MXFP4 (packed E2M1 codes + one E8M0
// byte per 32 elements) in the layouts the TMA loads and tcgen05 block-scaled MMAs consume.
// This is the surrounding kernel's "existing low-bit path" (Sec. 3.1); EFQ itself does not touch it.
//
// OCP microscaling rule per 32-element block: shared exponent e = floor(log2 amax) - 2 (clamped to
// the E8M0 range), elements rounded to nearest-even E2M1 of x * 2^-e, saturating at +-6; an all-zero
// block gets byte 0 and zero codes.
//
// Layouts written (S_pad = S rounded up to 128; padding rows/keys are zero codes, byte 0):
//   Q, K codes   [B*H, S_pad, 64 B]          row-major, 2 codes per byte, element 2u in the low nibble
//                (few query tokens: the query heads of a KV group packed into one 128-row tile, [B*Hkv, 128, 64 B])
//   V^T codes    [B*Hkv, 128 (channel), S_pad/2 B]   keys contiguous: the P~V contraction runs over keys
//                (packed variable-length batch: [Hkv, 128, sum of S_pad / 2 B], the sequences side by side along the keys)
//   scale tiles  one 512-byte tile per 128 rows (Q, K: rows = tokens, 4 blocks along d;
//                V: rows = channels, 4 key blocks of the 128-key tile); byte of (row r, block b) at
//                (r % 32) * 16 + (r / 32) * 4 + b, the order the scale-factor copy into TMEM expects.
#include <cuda_bf16.h>

//
// Memory-bound.  A block of 256 threads takes one 128-row (Q, K) or 128-key (V) tile, 32 KB of bf16: loads of 16 or 32
// bytes that fill their sectors, all of a thread's 128 bytes in flight at once; V codes pass through shared memory, so that a
// channel's 64 bytes of a tile are written together.
#include "efq_common.cuh"
#include "efq_internal.cuh"
#include "mxfp4.cuh"
#include "sm100_ptx.cuh"

namespace efq {

struct QuantSmem {
    uint8_t codes[4 * kABlock];
    __align__(16) uint8_t sf[512];
};

// 32 bytes of one row, bypassing L1 (32-byte aligned)
__device__ __forceinline__ void load32(const void* p, uint32_t* w)
{
    asm volatile("ld.global.L1::no_allocate.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]), "=r"(w[6]), "=r"(w[7]) : "l"(p));
}
__device__ __forceinline__ void load16x2(const void* p, uint32_t* w)
{
    const uint4 a = __ldcs(static_cast<const uint4*>(p)), b = __ldcs(static_cast<const uint4*>(p) + 1);
    w[0] = a.x; w[1] = a.y; w[2] = a.z; w[3] = a.w; w[4] = b.x; w[5] = b.y; w[6] = b.z; w[7] = b.w;
}

// Tile `tile` of a Q or K segment: two (row, block) pairs per thread, four neighbouring lanes per row.
__device__ __forceinline__ void quantize_rows(const QuantSeg& g, int tile)
{
    const int tiles_per_head = static_cast<int>(g.S_pad >> 7);
    const int head = tile / tiles_per_head, row0 = (tile - head * tiles_per_head) * 128;
    const int blk = threadIdx.x & 3;
    const bool wide = (reinterpret_cast<uintptr_t>(g.src) & 31u) == 0;      // strides are multiples of 256 bytes
    uint32_t w[2][16];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int row = row0 + (threadIdx.x >> 2) + 64 * h;
        if (row < g.S) {
            int64_t src_head = head, src_row = row;
            if (g.pack_G > 1) {                // packed query tile: rows run over (query head of the group, token)
                const int gq = row / g.pack_lq;
                src_head = static_cast<int64_t>(head) * g.pack_G + gq;
                src_row = row - gq * g.pack_lq;
            }
            const __nv_bfloat16* src = g.src + src_head * g.head_stride + src_row * g.row_stride + blk * 32;
            if (wide) { load32(src, w[h]); load32(src + 16, w[h] + 8); }
            else { load16x2(src, w[h]); load16x2(src + 16, w[h] + 8); }
        } else {
#pragma unroll
            for (int i = 0; i < 16; ++i) w[h][i] = 0u;
        }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int row = (threadIdx.x >> 2) + 64 * h;
        uint4 c;
        uint32_t byte;
        mxfp4_block(w[h], c, byte);
        *reinterpret_cast<uint4*>(g.codes + (static_cast<int64_t>(tile) * 128 + row) * 64 + blk * 16) = c;
        uint32_t word = byte;
        word |= __shfl_down_sync(0xffffffffu, byte, 1) << 8;
        word |= __shfl_down_sync(0xffffffffu, byte, 2) << 16;
        word |= __shfl_down_sync(0xffffffffu, byte, 3) << 24;
        if (blk == 0) *reinterpret_cast<uint32_t*>(g.sf + static_cast<int64_t>(tile) * 512 + sf_tile_offset(row, 0)) = word;
    }
}

// Key tile `tile` of a V segment.
__device__ __forceinline__ void quantize_keys(const QuantSeg& g, int tile, QuantSmem* sm)
{
    const int tiles_per_head = static_cast<int>(g.S_pad >> 7);
    const int head = tile / tiles_per_head, kt = tile - head * tiles_per_head;
    const VTileLane L(threadIdx.x >> 5, threadIdx.x & 31);
    const int64_t left = g.S - (static_cast<int64_t>(kt) * 128 + L.key);      // valid keys from the lane's first on
    const uint4* src = reinterpret_cast<const uint4*>(g.src + static_cast<int64_t>(head) * g.head_stride + (static_cast<int64_t>(kt) * 128 + L.key) * g.row_stride + L.ch);
    const int64_t step = g.row_stride / 8;
    uint4 vv[8];
    if (left >= 8) {
#pragma unroll
        for (int i = 0; i < 8; ++i) vv[i] = __ldcs(src + i * step);
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) vv[i] = i < left ? __ldcs(src + i * step) : make_uint4(0, 0, 0, 0);
    }
    mxfp4_v_tile(vv, L, sm->codes, sm->sf);
    __syncthreads();
    uint8_t* const dst = g.codes + static_cast<int64_t>(head) * 128 * g.v_row_bytes + g.v_x0 + kt * 64;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int ch = (threadIdx.x >> 2) + 64 * h, blk = threadIdx.x & 3;
        *reinterpret_cast<uint4*>(dst + ch * g.v_row_bytes + blk * 16) = *reinterpret_cast<const uint4*>(sm->codes + a_offset(ch, blk));
    }
    if (threadIdx.x < 32)
        reinterpret_cast<uint4*>(g.sf + (head * g.v_sf_tiles_per_head + g.v_sf_tile0 + kt) * 512)[threadIdx.x] = reinterpret_cast<const uint4*>(sm->sf)[threadIdx.x];
}

struct QuantArgs {
    QuantSeg q, k, v;
    uint32_t* status;           // 256 words, cleared here: the forward that follows starts from a clean status
    int q_ctas, k_ctas;         // the grid: Q tiles, then K tiles, then V tiles
};

// The three operands in one launch.
__global__ void __launch_bounds__(256) quantize_qkv_kernel(const __grid_constant__ QuantArgs a)
{
    __shared__ QuantSmem sm;
    ptx::grid_wait();
    ptx::grid_launch_next();
    const int cta = static_cast<int>(blockIdx.x);
    if (cta == 0) a.status[threadIdx.x] = 0u;
    if (cta < a.q_ctas) quantize_rows(a.q, cta);
    else if (cta < a.q_ctas + a.k_ctas) quantize_rows(a.k, cta - a.q_ctas);
    else quantize_keys(a.v, cta - a.q_ctas - a.k_ctas, &sm);
}

// The jobs of a packed batch in one launch: a CTA finds its job by bisection of the prefix sums.  The CTAs after the last
// job write the item table of the forward that follows (a thread per place).
__global__ void __launch_bounds__(256) quantize_jobs_kernel(const QuantJob* __restrict__ jobs, const int32_t* __restrict__ first_cta,
                                                            int n_jobs, int n_quant, const ItemGroup* __restrict__ groups, int n_groups,
                                                            const int32_t* __restrict__ places, int n_places,
                                                            ItemDesc* __restrict__ items, uint32_t* status)
{
    __shared__ QuantSmem sm;
    ptx::grid_wait();
    ptx::grid_launch_next();
    const int cta = blockIdx.x;
    if (cta == 0 && status != nullptr) status[threadIdx.x] = 0u;
    if (cta >= n_quant) {
        const int place = (cta - n_quant) * 256 + static_cast<int>(threadIdx.x);
        if (place >= n_places) return;
        const int item = places != nullptr ? __ldg(places + place) : place;
        if (item < 0) {
            items[place] = ItemDesc{0, 0, 0, -1, 0, 0, 0, 0};
            return;
        }
        int lo = 0, hi = n_groups;            // groups[lo].first_item <= item < groups[hi].first_item
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (__ldg(&groups[mid].first_item) <= item) lo = mid; else hi = mid;
        }
        const ItemGroup g = groups[lo];
        items[place] = ItemDesc{g.seq, g.qt, item - g.first_item, g.n_tiles, g.Sq, g.Sk, g.packed, 0};
        return;
    }
    int lo = 0, hi = n_jobs;                  // first_cta[lo] <= cta < first_cta[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(first_cta + mid) <= cta) lo = mid; else hi = mid;
    }
    const QuantJob& job = jobs[lo];
    const int tile = cta - __ldg(first_cta + lo);
    if (job.kind == kQuantRows) quantize_rows(job.seg, tile);
    else quantize_keys(job.seg, tile, &sm);
}

int64_t quantize_job_ctas(const QuantJob& job) { return job.seg.heads * (job.seg.S_pad / 128); }

cudaError_t launch_quantize_qkv(const QuantSeg& q, const QuantSeg& k, const QuantSeg& v, uint32_t* status, cudaStream_t stream)
{
    const int64_t nq = q.heads * (q.S_pad / 128), nk = k.heads * (k.S_pad / 128), nv = v.heads * (v.S_pad / 128), grid = nq + nk + nv;
    if (grid <= 0 || grid > 0x7fffffffll) return cudaErrorInvalidValue;
    QuantArgs a;
    a.q = q; a.k = k; a.v = v;
    a.status = status;
    a.q_ctas = static_cast<int>(nq);
    a.k_ctas = static_cast<int>(nk);
    return launch_overlapped(quantize_qkv_kernel, dim3(static_cast<unsigned>(grid)), 256, 0, stream, a);
}

cudaError_t launch_quantize_jobs(const QuantJob* jobs, const int32_t* first_cta, int n_jobs, int64_t total_ctas, const ItemGroup* groups,
                                 int n_groups, const int32_t* places, int64_t n_places, ItemDesc* items, uint32_t* status, cudaStream_t stream)
{
    const int64_t grid = total_ctas + (n_places + 255) / 256;
    if (n_jobs <= 0 || total_ctas <= 0 || grid > 0x7fffffffll) return cudaErrorInvalidValue;
    return launch_overlapped(quantize_jobs_kernel, dim3(static_cast<unsigned>(grid)), 256, 0, stream, jobs, first_cta, n_jobs,
                             static_cast<int>(total_ctas), groups, n_groups, places, static_cast<int>(n_places), items, status);
}

}  // namespace efq
