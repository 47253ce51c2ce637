// Attention forward for few query rows (decode steps, short chunks): the rows of the query heads of a KV group - at
// most 24 of them - meet a long K/V of which every byte is used once.  What bounds it is the read of the bf16 K and V,
// so nothing of theirs goes back to memory: two streaming kernels quantise the tiles on their way into shared memory
// and feed them to the tensor core there.
//
//   few_scores_kernel   K tile -> MXFP4 operand; S^T[key, row] = K^ Q^^T (128 keys x 8..24 rows); raw scores and the
//                       maxima of the 32-key blocks go to the workspace (4 bytes per row and key against 256 of K)
//   few_values_kernel   the running maximum of every row before the chunk from the block maxima; Algorithm 1 with
//                       thread = key (a microscaling block is a warp); V tile -> MXFP4 operand, transposed;
//                       O^T[channel, row] += V^^T P~; the partial sums of a chunk take the place of its first tile's scores
//   few_merge_kernel    the chunks of a row added up
//
// The KV range is cut into chunks by a rule on the sequence's own shape, so the result of a sequence does not depend on
// its neighbours.  The shifted scores use the running maximum over all keys up to the tile (Algorithm 2), which the first
// kernel makes available to every chunk: the codes are those of the one-pass forward, bit for bit.
//
// A block takes one chunk, or where few chunks do not fill the chip a half to an eighth of one, whose tiles the merge then adds up
// in the chunk's order (few_merge_tiles_kernel).  Several blocks per SM hide the latencies of one another's tiles (load, quantise, MMA,
// accumulator).  Loads by TMA with a role per warp (two blocks of 16 warps) were built too and are no faster: the short
// dependent sequences of the code warps then wait behind the quantisers of their scheduler.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "efq_common.cuh"
#include "efq_internal.cuh"
#include "efq_producers.cuh"
#include "mxfp4.cuh"
#include "sm100_ptx.cuh"

namespace efq {
namespace {

constexpr int kTile = 128;
constexpr int kFewThreads = 256;
constexpr int kStateRing = 4;
constexpr uint32_t kFewTmemCols = 128;      // four CTAs per SM share the 512 columns
constexpr uint32_t kColD = 0;               // 2 x 32
constexpr uint32_t kColSfA = 64;            // 2 x 4
constexpr uint32_t kColSfB = 72;            // 2 x 4

// One (sequence, KV head, chunk) of the grid.  Heads run fastest: the CTAs in flight read neighbouring heads of the same
// tokens, which lie side by side in a token-major cache.
struct Unit {
    int seq, head, chunk, n_chunks;
    int Sq, Sk, Sk_pad, j0, j1;
    const __nv_bfloat16 *q, *k, *v;
    float* o;
    int64_t s_off;             // first score of the (sequence, head) in the workspace, rows Sk_pad apart
};

__device__ __forceinline__ Unit find_unit(const FewParams& P, int id)
{
    Unit u;
    int64_t kp;
    if (P.n_seqs == 0) {                    // [B, H, S, d]
        u.head = id % P.Hkv;
        id /= P.Hkv;
        u.chunk = id % P.dense_chunks;
        u.seq = id / P.dense_chunks;
        u.Sq = P.Sq; u.Sk = P.Sk;
        kp = static_cast<int64_t>(u.seq) * P.Sk_pad;
        u.q = P.q + u.seq * P.q_seq; u.k = P.k + u.seq * P.k_seq; u.v = P.v + u.seq * P.k_seq; u.o = P.o + u.seq * P.q_seq;
    } else {
        const FewSeq* t = P.seqs != nullptr ? P.seqs : P.inline_seqs;
        int lo = 0, hi = P.n_seqs;          // t[lo].first_unit <= id < t[hi].first_unit
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (t[mid].first_unit <= id) lo = mid; else hi = mid;
        }
        const FewSeq s = t[lo];
        id -= s.first_unit;
        u.seq = lo;
        u.head = id % P.Hkv;
        u.chunk = id / P.Hkv;
        u.Sq = s.Sq; u.Sk = s.Sk;
        kp = s.k_pad0;
        u.q = P.q + s.q0 * P.q_row; u.k = P.k + s.k0 * P.k_row; u.v = P.v + s.k0 * P.k_row; u.o = P.o + s.q0 * P.q_row;
    }
    const int n_tiles = (u.Sk + kTile - 1) / kTile, per = few_chunk_tiles(n_tiles, P.G * u.Sq);
    u.n_chunks = (n_tiles + per - 1) / per;
    u.j0 = u.chunk * per;
    u.j1 = min(u.j0 + per, n_tiles);
    u.Sk_pad = n_tiles * kTile;
    u.q += static_cast<int64_t>(u.head) * P.G * P.q_head;
    u.o += static_cast<int64_t>(u.head) * P.G * P.q_head;
    u.k += u.head * P.k_head;
    u.v += u.head * P.k_head;
    u.s_off = (kp * P.Hkv + static_cast<int64_t>(u.head) * u.Sk_pad) * P.row_cap;
    return u;
}

// 2^-split of a chunk for this block, whose index says which; false if the chunk, as the last of a sequence may be, is too short for it
__device__ __forceinline__ bool take_part(Unit& u, int rows, int split)
{
    const int per = max(1, few_chunk_tiles(u.Sk_pad / kTile, rows) >> split), part = static_cast<int>(blockIdx.x) & ((1 << split) - 1);
    u.j0 = min(u.j0 + part * per, u.j1);
    u.j1 = min(u.j0 + per, u.j1);
    return u.j0 < u.j1;
}

// The factors of one tile and row, where the values were taken tile by tile
__device__ __forceinline__ float* tile_stat(const FewParams& P, const Unit& u, int tile, int row)
{
    return P.stats + (u.s_off / kTile + static_cast<int64_t>(tile) * P.row_cap + row) * kFewStatFloats;
}

__device__ __forceinline__ float warp_max(float x)
{
    float m;
    asm("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(m) : "f"(x));
    return m;
}

// N consecutive columns (a multiple of 8) of this thread's TMEM lane
template <int N>
__device__ __forceinline__ void tmem_ld_cols(uint32_t addr, float (&r)[N])
{
#pragma unroll
    for (int o = 0; o < N; o += 8)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                     : "=f"(r[o]), "=f"(r[o + 1]), "=f"(r[o + 2]), "=f"(r[o + 3]), "=f"(r[o + 4]), "=f"(r[o + 5]), "=f"(r[o + 6]), "=f"(r[o + 7])
                     : "r"(addr + o) : "memory");
}

struct __align__(1024) FewSmem {
    uint8_t b[2][32 * 64];          // Q codes ([0] only), or the probability operand of a tile
    uint8_t a[2][4 * kABlock];      // K or V^T codes of a tile
    uint8_t sf_a[2][512];
    uint8_t sf_b[2][512];
    // row state of a tile [tile mod 4][row]: raw running maximum, the same in scaled units, the rescale factor, and per key
    // block the additive term of the code rule and the scale byte
    float m_raw[kStateRing][32], m_s[kStateRing][32], alpha[kStateRing][32];
    float par[kStateRing][4][32];
    uint32_t byte[kStateRing][4][32];
    float4 bmax[kFewMaxChunk][32];  // [tile of the chunk][row]: its block maxima
    uint64_t mma_done[2];
    uint32_t tmem_base;
    volatile uint32_t gave_up;      // a bounded wait of this CTA ran out
};

// Bounded wait for a completion of this CTA's own MMAs (20000 polls, 0.07 s when nothing comes).  On expiry the status word takes
// the error; the CTA carries on with whatever the accumulator holds, so that every thread still meets the block's barriers, and
// no further wait of it lasts.  Every 128 polls, some 0.4 ms, it also looks whether another CTA has given up already: by then
// block 0, the first to start, has cleared the word long ago.
__device__ __forceinline__ void wait_done(FewSmem* sm, int buf, uint32_t parity, uint32_t* status)
{
    for (int i = 1; i <= 20000; ++i) {
        if (ptx::mbar_try_wait_suspend(&sm->mma_done[buf], parity, 50000u)) return;
        if (sm->gave_up != 0u) return;
        if ((i & 127) == 0 && *reinterpret_cast<volatile uint32_t*>(status) != 0u) break;
    }
    sm->gave_up = 1u;
    atomicExch(status, static_cast<uint32_t>(EFQ_ERR_DEVICE_TIMEOUT));
}

// Operand rows past the last query row are never written: they only reach accumulator columns that nobody reads.
__device__ __forceinline__ void few_setup(FewSmem* sm, int warp)
{
    if (warp == 0) ptx::tmem_alloc(&sm->tmem_base, kFewTmemCols);
    if (threadIdx.x == 32) {
        ptx::mbar_init(&sm->mma_done[0], 1);
        ptx::mbar_init(&sm->mma_done[1], 1);
        sm->gave_up = 0u;
        ptx::mbar_init_fence();
    }
}

// D[128, N] = A B^T of one tile: two K = 64 steps, a fresh accumulator
__device__ __forceinline__ void few_mma(const FewParams& P, FewSmem* sm, uint32_t tmem, int buf, int b_buf, uint32_t n)
{
    if (P.inject_skip_mma) return;
    const uint64_t d_sw64 = ptx::smem_desc(0, 16, 512, ptx::kLayoutSw64);
    const uint64_t d_sf = ptx::smem_desc(0, 16, 128, ptx::kLayoutNone);
    const uint32_t sfa = tmem + kColSfA + 4 * buf, sfb = tmem + kColSfB + 4 * b_buf, d = tmem + kColD + 32 * buf;
    ptx::tmem_cp_sf(sfa, d_sf + (ptx::smem_u32(sm->sf_a[buf]) >> 4));
    ptx::tmem_cp_sf(sfb, d_sf + (ptx::smem_u32(sm->sf_b[b_buf]) >> 4));
    const uint64_t da = ptx::smem_desc(ptx::smem_u32(sm->a[buf]), kABlock, kARowGroup, ptx::kLayoutNone), db = d_sw64 + (ptx::smem_u32(sm->b[b_buf]) >> 4);
    ptx::mma_mxf4(d, da, db, ptx::mxf4_idesc(n, 0), sfa, sfb, 0u);
    ptx::mma_mxf4(d, da + (2 * kABlock >> 4), db + 2, ptx::mxf4_idesc(n, 2), sfa | (2u << 30), sfb | (2u << 30), 1u);
    ptx::mma_commit(&sm->mma_done[buf]);
}

// N: query rows rounded up to a multiple of 8 (the N of the MMA)
template <int N>
__global__ void __launch_bounds__(kFewThreads, N <= 8 ? 4 : 3) few_scores_kernel(const __grid_constant__ FewParams P)
{
    __shared__ FewSmem smem;
    FewSmem* const sm = &smem;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    few_setup(sm, warp);             // before the search for the unit, which takes longer
    ptx::grid_wait();                // the kernels before: inputs, and the workspace of an earlier call
    ptx::grid_launch_next();
    // A block takes 2^-split of a chunk: the scores of a tile need nothing of another, and a few chunks do not fill the chip.
    Unit u = find_unit(P, static_cast<int>(blockIdx.x) >> P.split);
    const int R = P.G * u.Sq;
    const bool work = take_part(u, R, P.split);
    if (blockIdx.x == 0) P.status[tid] = 0u;
    if (!work) {
        __syncthreads();
        if (warp == 0) ptx::tmem_dealloc(sm->tmem_base, kFewTmemCols);
        return;
    }
    // K: a quad of lanes takes a key, a lane every fourth 16-byte piece of it - a load instruction reads 64 contiguous
    // bytes of every key - and so a quarter of each of the four blocks
    const int quad = tid & 3, key_in_tile = tid >> 2;
    uint4 kk[2][4];
    const uint4* k_src = reinterpret_cast<const uint4*>(u.k + (u.j0 * kTile + key_in_tile) * P.k_row) + quad;
    const int64_t k_half = 8 * P.k_row;                  // 64 keys on, in 16-byte pieces
    auto load_k = [&](int j) {
        if ((j + 1) * kTile <= u.Sk) {
#pragma unroll
            for (int i = 0; i < 4; ++i) kk[0][i] = __ldcs(k_src + 4 * i);
#pragma unroll
            for (int i = 0; i < 4; ++i) kk[1][i] = __ldcs(k_src + k_half + 4 * i);
        } else {
            const bool in0 = j * kTile + key_in_tile < u.Sk, in1 = j * kTile + key_in_tile + 64 < u.Sk;
#pragma unroll
            for (int i = 0; i < 4; ++i) kk[0][i] = in0 ? __ldcs(k_src + 4 * i) : make_uint4(0, 0, 0, 0);
#pragma unroll
            for (int i = 0; i < 4; ++i) kk[1][i] = in1 ? __ldcs(k_src + k_half + 4 * i) : make_uint4(0, 0, 0, 0);
        }
        k_src += 2 * k_half;
    };
    load_k(u.j0);
    // Q: one thread per (row, block)
    for (int t = tid; t < 4 * R; t += kFewThreads) {
        const int row = t >> 2, blk = t & 3, g = row / u.Sq;
        const uint4* src = reinterpret_cast<const uint4*>(u.q + g * P.q_head + (row - g * u.Sq) * P.q_row + blk * 32);
        uint32_t w[16];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint4 x = src[i];
            w[4 * i] = x.x; w[4 * i + 1] = x.y; w[4 * i + 2] = x.z; w[4 * i + 3] = x.w;
        }
        uint4 c;
        uint32_t byte;
        mxfp4_block(w, c, byte);
        *reinterpret_cast<uint4*>(sm->b[0] + code_tile_offset(row, blk)) = c;
        sm->sf_b[0][sf_tile_offset(row, blk)] = static_cast<uint8_t>(byte);
    }
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::tc_fence_after_sync();
    const uint32_t tmem = sm->tmem_base;
    const int n_tiles = u.Sk_pad / kTile, nblk = 4 * n_tiles;
    const int quarter = warp & 3, half = warp >> 2;      // 32 keys of the tile; rows 2 i + half
    // last visible key of row `lane`
    const int limit = min(P.causal ? lane % u.Sq + u.Sk - u.Sq : u.Sk, u.Sk - 1);

    float* dst = P.scores + u.s_off + few_row_offset(half, n_tiles) + u.j0 * kTile + quarter * 32 + lane;
    float* dst_max = P.block_max + u.s_off / 32 + half * nblk + u.j0 * 4 + quarter;
    // raw scores of a finished tile: thread = key, two rows of the half side by side
    auto put_scores = [&](int j) {
        const int buf = (j - u.j0) & 1;
        wait_done(sm, buf, static_cast<uint32_t>(j - u.j0) >> 1 & 1u, P.status);
        ptx::tc_fence_after_sync();
        float s[N];
        tmem_ld_cols<N>(tmem + (static_cast<uint32_t>(quarter * 32) << 16) + kColD + 32 * buf, s);
        ptx::tmem_wait_ld();
        ptx::tc_fence_before_sync();
        const int key = j * kTile + quarter * 32 + lane;
#pragma unroll
        for (int i = 0; i < N; i += 4) {
            const int row = i + half;
            if (row < R) {
                const float x0 = key <= __shfl_sync(0xffffffffu, limit, row) ? (half ? s[i + 1] : s[i]) : -INFINITY;
                const float x1 = key <= __shfl_sync(0xffffffffu, limit, row + 2) ? (half ? s[i + 3] : s[i + 2]) : -INFINITY;
                const float m0 = warp_max(x0), m1 = warp_max(x1);
                dst[few_row_offset(i, n_tiles)] = x0;
                if (row + 2 < R) dst[few_row_offset(i + 2, n_tiles)] = x1;
                if (lane == 0) {
                    dst_max[i * nblk] = m0;
                    if (row + 2 < R) dst_max[(i + 2) * nblk] = m1;
                }
            }
        }
        dst += kTile;
        dst_max += 4;
    };

    for (int j = u.j0; j < u.j1; ++j) {
        const int buf = (j - u.j0) & 1;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int row = key_in_tile + 64 * h;
            uint32_t m[4];
#pragma unroll
            for (int b = 0; b < 4; ++b)
                m[b] = bf16x2_absmax(bf16x2_absmax(kk[h][b].x, kk[h][b].y), bf16x2_absmax(kk[h][b].z, kk[h][b].w));
            // two blocks in one register (low half, high half), then over the quad
            uint32_t t0 = bf16x2_absmax(__byte_perm(m[0], m[1], 0x5410), __byte_perm(m[0], m[1], 0x7632));
            uint32_t t1 = bf16x2_absmax(__byte_perm(m[2], m[3], 0x5410), __byte_perm(m[2], m[3], 0x7632));
            t0 = bf16x2_absmax(t0, __shfl_xor_sync(0xffffffffu, t0, 1));
            t1 = bf16x2_absmax(t1, __shfl_xor_sync(0xffffffffu, t1, 1));
            t0 = mxfp4_fields(bf16x2_absmax(t0, __shfl_xor_sync(0xffffffffu, t0, 2)));
            t1 = mxfp4_fields(bf16x2_absmax(t1, __shfl_xor_sync(0xffffffffu, t1, 2)));
            const uint32_t s01 = mxfp4_scales(t0), s23 = mxfp4_scales(t1);
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const uint32_t s2 = __byte_perm(b < 2 ? s01 : s23, 0u, (b & 1) ? 0x3232 : 0x1010);
                const uint32_t w0 = bf16x2_mul(kk[h][b].x, s2), w1 = bf16x2_mul(kk[h][b].y, s2), w2 = bf16x2_mul(kk[h][b].z, s2), w3 = bf16x2_mul(kk[h][b].w, s2);
                *reinterpret_cast<uint32_t*>(sm->a[buf] + a_offset(row, b) + quad * 4) =
                    e2m1_word(bf16_lo(w0), bf16_hi(w0), bf16_lo(w1), bf16_hi(w1), bf16_lo(w2), bf16_hi(w2), bf16_lo(w3), bf16_hi(w3));
            }
            if (quad == 0)
                *reinterpret_cast<uint32_t*>(sm->sf_a[buf] + sf_tile_offset(row, 0)) =
                    mxfp4_byte_lo(t0) | mxfp4_byte_hi(t0) << 8 | mxfp4_byte_lo(t1) << 16 | mxfp4_byte_hi(t1) << 24;
        }
        if (j + 1 < u.j1) load_k(j + 1);
        ptx::fence_proxy_async_smem();
        ptx::tc_fence_before_sync();
        __syncthreads();
        if (warp == 0) {
            ptx::tc_fence_after_sync();
            if (ptx::elect_one()) few_mma(P, sm, tmem, buf, 0, N);
            __syncwarp();
        }
        if (j > u.j0) put_scores(j - 1);
    }
    put_scores(u.j1 - 1);
    ptx::tc_fence_before_sync();
    __syncthreads();
    if (warp == 0) ptx::tmem_dealloc(tmem, kFewTmemCols);
}

// One code (nibble) of this lane's key and row.  par is the row's additive term of the producer (lane-parallel state of the
// caller, broadcast); the exponential producers of the plain form also return the block's scale byte, equal in all lanes.
template <int PRODUCER>
__device__ __forceinline__ uint32_t key_code(float r, float par, const ProducerConsts& K, int lane, uint32_t& byte, float& p)
{
    if (PRODUCER == 0) {
        float t;
        asm("fma.rm.f32 %0, %1, %2, %3;" : "=f"(t) : "f"(fma_sat(r, K.A * 0.125f, par * 0.125f)), "f"(8.0f), "f"(8388608.0f));
        return min(__float_as_uint(t) & 15u, 7u);
    } else if (PRODUCER == 3) {
        return lut_code(r, K.A * 0.0625f, par * 0.0625f);
    } else if (PRODUCER == 4 || PRODUCER == 5) {
        const float t = __fmaf_rn(r, __fmul_rn(K.sigma, K.LOG2E), par);
        const float e = PRODUCER == 5 && ex2_by_poly(lane) ? ex2_poly3(t) : ex2_approx(t);
        return cvt_e2m1x2(e, 0.0f) & 15u;
    } else {
        p = ex2_approx(__fmul_rn(__fsub_rn(__fmul_rn(K.sigma, r), par), K.LOG2E));
        const float amax = fmaxf(warp_max(p), 0.0f);      // a row without a finite score has NaN everywhere: 0
        if (amax == 0.0f) { byte = 0u; return 0u; }
        const uint32_t bits = __float_as_uint(amax);
        const int E = static_cast<int>((bits >> 23) & 0xffu) - 127;
        int e = PRODUCER != 2 ? E - 2 : ((bits & 0x7fffffu) > 0x400000u ? E - 1 : E - 2);
        e = max(e, -127);
        byte = static_cast<uint32_t>(e + 127);
        return cvt_e2m1x2(p * __uint_as_float(static_cast<uint32_t>(127 - e) << 23), 0.0f) & 15u;
    }
}

// Optional dump of one query head (all lanes): the row's score and code of this lane's key, the block's byte, the tile's maximum.
__device__ __forceinline__ void few_dump(const FewParams& P, const Unit& u, int j, int quarter, int lane, int row, float score, uint32_t word,
                                         float m_s, uint32_t byte)
{
    const int g = row / u.Sq, tok = row - g * u.Sq, blk = j * 4 + quarter, key = blk * 32 + lane;
    if (u.head * P.G + g != P.dbg.head || tok < P.dbg.q_begin || tok >= P.dbg.q_end) return;
    const int64_t drow = tok - P.dbg.q_begin, blocks = (u.Sk + 31) / 32;
    if (P.dbg.raw_scores != nullptr && key < u.Sk) P.dbg.raw_scores[drow * u.Sk + key] = score;
    if (P.dbg.row_max != nullptr && quarter == 0 && lane == 0) P.dbg.row_max[drow * (u.Sk_pad / kTile) + j] = m_s;
    if (blk >= blocks) return;
    if (P.dbg.codes != nullptr && (lane & 7) == 0) reinterpret_cast<uint32_t*>(P.dbg.codes + (drow * blocks + blk) * 16)[lane >> 3] = word;
    if (P.dbg.scales != nullptr && lane == 0) P.dbg.scales[drow * blocks + blk] = static_cast<uint8_t>(byte);
}

// Row state of one tile, lane = row (one warp): the running maximum (Eq. rowmax-update), the factor its growth asks for
// (Eq. alpha) and the scale rule of the four key blocks.
template <int PRODUCER>
__device__ __forceinline__ void few_row_state(FewSmem* sm, const FewParams& P, int t, int slot, float m_run, int lane)
{
    const float4 b4 = sm->bmax[t][lane];
    const float bmax[4] = {b4.x, b4.y, b4.z, b4.w};
    float m_new = fmaxf(m_run, fmaxf(fmaxf(bmax[0], bmax[1]), fmaxf(bmax[2], bmax[3])));
    if (P.rescale_threshold > 0.0f && m_run != -INFINITY &&
        !(__fsub_rn(__fmul_rn(P.K.sigma, m_new), __fmul_rn(P.K.sigma, m_run)) > P.rescale_threshold))
        m_new = m_run;
    const float m_s = __fmul_rn(P.K.sigma, m_new);
    const bool grew = m_new > m_run && m_run != -INFINITY;
    sm->m_raw[slot][lane] = m_new;
    sm->m_s[slot][lane] = m_s;
    sm->alpha[slot][lane] = grew ? ex2_approx(__fmul_rn(__fsub_rn(__fmul_rn(P.K.sigma, m_run), m_s), P.K.LOG2E)) : 1.0f;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        float par = m_s;
        uint32_t byte = 0u;
        if (PRODUCER == 0 || PRODUCER == 3) {
            const BlockScale s = efq_block_scale(bmax[b], m_s, P.K);
            par = s.Bb; byte = s.byte;
        } else if (PRODUCER == 4 || PRODUCER == 5) {
            const FoldedScale f = etq_folded_scale(bmax[b], m_s, P.K);
            par = f.live ? f.c0e : -INFINITY;    // a block without a finite score: 2^-inf = 0 everywhere
            byte = f.byte;
        }
        sm->par[slot][b][lane] = par;
        sm->byte[slot][b][lane] = byte;
    }
}

// TILES: a block takes 2^-split of a chunk and leaves the product of every tile by itself, beside its factors, for the merge to
// add up as the chunk's block would have (same operations, same order, same bits).
template <int N, int PRODUCER, bool TILES>
__global__ void __launch_bounds__(kFewThreads, 3) few_values_kernel(const __grid_constant__ FewParams P)
{
    __shared__ FewSmem smem;
    FewSmem* const sm = &smem;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    ptx::grid_launch_next();
    Unit u = find_unit(P, static_cast<int>(blockIdx.x) >> (TILES ? P.split : 0));
    const int R = P.G * u.Sq;
    if (TILES && !take_part(u, R, P.split)) return;
    few_setup(sm, warp);
    const VTileLane L(warp, lane);
    uint4 vv[8];
    const int64_t v_step = P.k_row / 8;                  // a key on, in 16-byte pieces
    const uint4* v_src = reinterpret_cast<const uint4*>(u.v + (u.j0 * kTile + L.key) * P.k_row + L.ch);
    auto load_v = [&](int j) {
        if ((j + 1) * kTile <= u.Sk) {
            const uint4* src = v_src;
#pragma unroll
            for (int i = 0; i < 8; ++i, src += v_step) vv[i] = __ldcs(src);
        } else {
            const int left = u.Sk - (j * kTile + L.key);
#pragma unroll
            for (int i = 0; i < 8; ++i) vv[i] = i < left ? __ldcs(v_src + i * v_step) : make_uint4(0, 0, 0, 0);
        }
        v_src += kTile * v_step;
    };
    load_v(u.j0);       // an input: whatever produced it had finished before the scores kernel allowed this one to start
    ptx::grid_wait();

    // the chunk's block maxima and the running maximum of every row before the chunk
    const float* const bm = P.block_max + u.s_off / 32;
    const int n_tiles = u.Sk_pad / kTile, nblk = 4 * n_tiles;
    for (int i = tid; i < R * (u.j1 - u.j0); i += kFewThreads) {
        const int t = i / R, row = i - t * R;
        sm->bmax[t][row] = __ldcg(reinterpret_cast<const float4*>(bm + row * nblk) + u.j0 + t);
    }
    if (!(P.rescale_threshold > 0.0f)) {
        for (int row = warp; row < R; row += 8) {
            float m = -INFINITY;
            for (int b = lane; b < u.j0; b += 32) {
                const float4 x = __ldcg(reinterpret_cast<const float4*>(bm + row * nblk) + b);
                m = fmaxf(fmaxf(m, fmaxf(x.x, x.y)), fmaxf(x.z, x.w));
            }
            m = warp_max(m);
            if (lane == 0) sm->m_raw[kStateRing - 1][row] = m;
        }
    } else if (tid < R) {                    // optional policy: the kept maximum depends on the order of the tiles
        float m = -INFINITY;
        for (int j = 0; j < u.j0; ++j) {
            const float4 b = __ldcg(reinterpret_cast<const float4*>(bm + tid * nblk) + j);
            const float c = fmaxf(m, fmaxf(fmaxf(b.x, b.y), fmaxf(b.z, b.w)));
            if (m == -INFINITY || __fsub_rn(__fmul_rn(P.K.sigma, c), __fmul_rn(P.K.sigma, m)) > P.rescale_threshold) m = c;
        }
        sm->m_raw[kStateRing - 1][tid] = m;
    }
    // Codes: thread = key of block `quarter`; the warps of a half take the rows 2 i + half.  O^T: thread = channel.
    constexpr int NH = N / 2;
    const int quarter = warp & 3, half = warp >> 2;
    float* s_src = P.scores + u.s_off + few_row_offset(half, n_tiles) + u.j0 * kTile + quarter * 32 + lane;
    float* const tile_part = s_src;
    float x[NH];
    auto load_scores = [&]() {
#pragma unroll
        for (int i = 0; i < NH; ++i) x[i] = 2 * i + half < R ? __ldcg(s_src + few_row_offset(2 * i, n_tiles)) : -INFINITY;
        s_src += kTile;
    };
    load_scores();
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::tc_fence_after_sync();
    const uint32_t tmem = sm->tmem_base;
    if (warp == 0 && lane < R) few_row_state<PRODUCER>(sm, P, 0, 0, sm->m_raw[kStateRing - 1][lane], lane);
    __syncthreads();

    const int my_row = 2 * lane + half;      // lane i keeps the denominator (of this block position) of row 2 i + half
    const bool has_row = my_row < R;
    float l_run = 0.0f;
    float acc[NH];
#pragma unroll
    for (int i = 0; i < NH; ++i) acc[i] = 0.0f;
    auto add_tile = [&](int t) {
        const int buf = t & 1;
        wait_done(sm, buf, static_cast<uint32_t>(t >> 1) & 1u, P.status);
        ptx::tc_fence_after_sync();
        float d[N];
        tmem_ld_cols<N>(tmem + (static_cast<uint32_t>(quarter * 32) << 16) + kColD + 32 * buf, d);
        ptx::tmem_wait_ld();
        ptx::tc_fence_before_sync();
#pragma unroll
        for (int i = 0; i < NH; ++i) {
            const float x = half ? d[2 * i + 1] : d[2 * i];
            if (!TILES) acc[i] = fmaf(acc[i], sm->alpha[t % kStateRing][2 * i + half], x);
            // the tile's scores may go, as below
            else if (2 * i + half < R) tile_part[few_row_offset(2 * i, n_tiles) + t * kTile] = x;
        }
    };
    const bool dump = P.has_dbg && u.seq == P.dbg.batch && u.head == P.dbg.head / P.G;
    for (int j = u.j0; j < u.j1; ++j) {
        const int t = j - u.j0, buf = t & 1, slot = t % kStateRing;
        // ---- Algorithm 1, two rows side by side so that their chains of shuffles overlap
        uint32_t byte = has_row ? sm->byte[slot][quarter][my_row] : 0u;
        int count = 0;                       // of lane i: twice the sum of its row's E2M1 values in this block
        float psum = 0.0f;
#pragma unroll
        for (int i0 = 0; i0 < NH; i0 += 2) {
            if (2 * i0 + half < R) {
                uint32_t c[2], b[2] = {0u, 0u};
                float p[2] = {0.0f, 0.0f};
                int n[2];
#pragma unroll
                for (int i = 0; i < 2; ++i) c[i] = key_code<PRODUCER>(x[i0 + i], sm->par[slot][quarter][2 * (i0 + i) + half], P.K, lane, b[i], p[i]);
#pragma unroll
                for (int i = 0; i < 2; ++i) n[i] = __reduce_add_sync(0xffffffffu, static_cast<int>((0xC8643210u >> (4u * c[i])) & 15u));
                if (PRODUCER == 6)
                    for (int o = 16; o > 0; o >>= 1) {
                        p[0] += __shfl_xor_sync(0xffffffffu, p[0], o);
                        p[1] += __shfl_xor_sync(0xffffffffu, p[1], o);
                    }
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    if (lane == i0 + i) {
                        count = n[i];
                        psum = p[i];
                        if (PRODUCER == 1 || PRODUCER == 2 || PRODUCER == 6) byte = b[i];
                    }
                    c[i] |= __shfl_down_sync(0xffffffffu, c[i], 1) << 4;
                }
                c[0] |= __shfl_down_sync(0xffffffffu, c[0], 2) << 8;
                c[1] |= __shfl_down_sync(0xffffffffu, c[1], 2) << 8;
                c[0] |= __shfl_down_sync(0xffffffffu, c[0], 4) << 16;
                c[1] |= __shfl_down_sync(0xffffffffu, c[1], 4) << 16;
                const int row = 2 * i0 + half;
                if ((lane & 7) == 0) {
                    *reinterpret_cast<uint32_t*>(sm->b[buf] + code_tile_offset(row, quarter) + (lane >> 1)) = c[0];
                    *reinterpret_cast<uint32_t*>(sm->b[buf] + code_tile_offset(row + 2, quarter) + (lane >> 1)) = c[1];
                }
                if (dump) {
                    few_dump(P, u, j, quarter, lane, row, x[i0], c[0], sm->m_s[slot][row], __shfl_sync(0xffffffffu, byte, i0));
                    if (row + 2 < R) few_dump(P, u, j, quarter, lane, row + 2, x[i0 + 1], c[1], sm->m_s[slot][row + 2], __shfl_sync(0xffffffffu, byte, i0 + 1));
                }
            }
        }
        if (has_row) {
            sm->sf_b[buf][sf_tile_offset(my_row, quarter)] = static_cast<uint8_t>(byte);
            const float unit = byte != 0u ? __uint_as_float(byte << 23) : __uint_as_float(0x00400000u);
            const float add = PRODUCER == 6 ? psum : __fmul_rn(static_cast<float>(count) * 0.5f, unit), alpha = sm->alpha[slot][my_row];
            if (!TILES) {
                l_run = __fmaf_rn(l_run, alpha, add);
            } else {
                float* const stat = tile_stat(P, u, j, my_row);
                stat[quarter] = add;
                if (quarter == 0) { stat[4] = sm->m_s[slot][my_row]; stat[5] = alpha; }
            }
        }
        if (j + 1 < u.j1) load_scores();
        // ---- V^T operand of the tile
        mxfp4_v_tile(vv, L, sm->a[buf], sm->sf_a[buf]);
        if (j + 1 < u.j1) load_v(j + 1);
        if (warp == ((t + 1) & 7) && j + 1 < u.j1 && lane < R)
            few_row_state<PRODUCER>(sm, P, t + 1, (t + 1) % kStateRing, sm->m_raw[slot][lane], lane);
        ptx::fence_proxy_async_smem();
        ptx::tc_fence_before_sync();
        __syncthreads();
        if (warp == 0) {
            ptx::tc_fence_after_sync();
            if (ptx::elect_one()) few_mma(P, sm, tmem, buf, buf, N);
            __syncwarp();
        }
        if (t > 0) add_tile(t - 1);
    }
    add_tile(u.j1 - u.j0 - 1);

    // ---- partial result of the chunk.  Its scores may go: the block's threads used the last of them before the barrier of the last
    // tile, and no other block reads them.
#pragma unroll
    for (int i = 0; i < NH; ++i)
        if (!TILES && 2 * i + half < R) tile_part[few_row_offset(2 * i, n_tiles)] = acc[i];
    if (!TILES && has_row) {
        float* const stat = P.stats + (static_cast<size_t>(blockIdx.x) * P.row_cap + my_row) * kFewStatFloats;
        stat[quarter] = l_run;
        if (quarter == 0) stat[4] = sm->m_s[(u.j1 - u.j0 - 1) % kStateRing][my_row];
    }
    ptx::tc_fence_before_sync();
    __syncthreads();
    if (warp == 0) ptx::tmem_dealloc(tmem, kFewTmemCols);
}

// What the merges share: a chunk's weight against the row's last maximum, and the row's sum over its partial sums.
__device__ __forceinline__ float chunk_weight(float m, float m_last, const ProducerConsts& K)
{
    // equal maxima by comparison: both are infinite where the inputs or a score overflowed
    return m == -INFINITY ? 0.0f : m == m_last ? 1.0f : ex2_approx(__fmul_rn(__fsub_rn(m, m_last), K.LOG2E));
}
__device__ __forceinline__ void add_chunk(float4& a, float& l, const float4& x, const float4& lp, float w)
{
    l = fmaf((lp.x + lp.y) + (lp.z + lp.w), w, l);
    a.x = fmaf(x.x, w, a.x); a.y = fmaf(x.y, w, a.y); a.z = fmaf(x.z, w, a.z); a.w = fmaf(x.w, w, a.w);
}
struct MergeRow {
    Unit u;              // the first chunk, whose length is that of all but the last
    int first_id, row;
    __device__ __forceinline__ MergeRow(const FewParams& P) : row(static_cast<int>(blockIdx.y))
    {
        const int head = static_cast<int>(blockIdx.x) % P.Hkv, seq = static_cast<int>(blockIdx.x) / P.Hkv;
        first_id = head + (P.n_seqs == 0 ? seq * P.dense_chunks * P.Hkv : (P.seqs != nullptr ? P.seqs : P.inline_seqs)[seq].first_unit);
        u = find_unit(P, first_id);
    }
    __device__ __forceinline__ void store(const FewParams& P, const float4 (&sum)[4][32], const float (&den)[4]) const
    {
        if (threadIdx.x >= 128u) return;
        const float* s = reinterpret_cast<const float*>(sum) + threadIdx.x;
        const float t = (s[0] + s[128]) + (s[256] + s[384]), d = (den[0] + den[1]) + (den[2] + den[3]);
        const int g = row / u.Sq;
        u.o[g * P.q_head + (row - g * u.Sq) * P.q_row + threadIdx.x] = t * (d > 0.0f ? 1.0f / d : 0.0f);
    }
};

// Adds up the chunks of one row (a block per sequence, KV head and row): a warp takes every fourth chunk, a lane four
// channels, so that all loads of a short list of chunks are in flight together.
__global__ void __launch_bounds__(128) few_merge_kernel(const __grid_constant__ FewParams P)
{
    __shared__ float4 sum[4][32];
    __shared__ float den[4];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const MergeRow r(P);
    const Unit& u = r.u;
    ptx::grid_wait();
    if (r.row >= P.G * u.Sq) return;
    const float4* const part = reinterpret_cast<const float4*>(P.scores + u.s_off + few_row_offset(r.row, u.Sk_pad / kTile)) + lane;
    const int part_step = u.j1 * (kTile / 4);
    const float* const stat = P.stats + (static_cast<size_t>(r.first_id) * P.row_cap + r.row) * kFewStatFloats;
    const size_t stat_step = static_cast<size_t>(P.Hkv) * P.row_cap * kFewStatFloats;
    const float m_last = __ldcg(stat + (u.n_chunks - 1) * stat_step + 4);
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
    float l = 0.0f;
#pragma unroll 4
    for (int c = warp; c < u.n_chunks; c += 4) {
        const float m = __ldcg(stat + c * stat_step + 4);
        const float4 x = __ldcg(part + static_cast<int64_t>(c) * part_step);
        const float4 lp = __ldcg(reinterpret_cast<const float4*>(stat + c * stat_step));
        add_chunk(a, l, x, lp, chunk_weight(m, m_last, P.K));
    }
    sum[warp][lane] = a;
    if (lane == 0) den[warp] = l;
    __syncthreads();
    r.store(P, sum, den);
}

// The same where the values were taken tile by tile: sixteen warps first make a chunk each of its tiles, with the operations of the
// block that would have had it, then four of them add the chunks as above.
constexpr int kMergeWarps = 16;
__global__ void __launch_bounds__(32 * kMergeWarps) few_merge_tiles_kernel(const __grid_constant__ FewParams P)
{
    __shared__ float4 chunk_sum[kMergeWarps][32], chunk_den[kMergeWarps], sum[4][32];
    __shared__ float chunk_max[kMergeWarps], den[4];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const MergeRow r(P);
    const Unit& u = r.u;
    ptx::grid_wait();
    if (r.row >= P.G * u.Sq) return;
    const int n_tiles = u.Sk_pad / kTile, per = u.j1;
    const float4* const part = reinterpret_cast<const float4*>(P.scores + u.s_off + few_row_offset(r.row, n_tiles)) + lane;
    const float m_last = __ldcg(tile_stat(P, u, n_tiles - 1, r.row) + 4);
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
    float l = 0.0f;
    for (int c0 = 0; c0 < u.n_chunks; c0 += kMergeWarps) {
        const int j0 = (c0 + warp) * per, tiles = min(per, n_tiles - j0);
        if (tiles > 0) {
            float4 d[kFewMaxChunk], add[kFewMaxChunk];
            float2 f[kFewMaxChunk];                  // maximum, factor
#pragma unroll
            for (int t = 0; t < kFewMaxChunk; ++t)
                if (t < tiles) {
                    const float* const ts = tile_stat(P, u, j0 + t, r.row);
                    d[t] = __ldcg(part + static_cast<int64_t>(j0 + t) * (kTile / 4));
                    add[t] = __ldcg(reinterpret_cast<const float4*>(ts));
                    f[t] = __ldcg(reinterpret_cast<const float2*>(ts + 4));
                }
            float4 x = make_float4(0.f, 0.f, 0.f, 0.f), lp = x;
            float m = -INFINITY;
#pragma unroll
            for (int t = 0; t < kFewMaxChunk; ++t)
                if (t < tiles) {
                    m = f[t].x;
                    x.x = fmaf(x.x, f[t].y, d[t].x); x.y = fmaf(x.y, f[t].y, d[t].y); x.z = fmaf(x.z, f[t].y, d[t].z); x.w = fmaf(x.w, f[t].y, d[t].w);
                    lp.x = __fmaf_rn(lp.x, f[t].y, add[t].x); lp.y = __fmaf_rn(lp.y, f[t].y, add[t].y);
                    lp.z = __fmaf_rn(lp.z, f[t].y, add[t].z); lp.w = __fmaf_rn(lp.w, f[t].y, add[t].w);
                }
            chunk_sum[warp][lane] = x;
            if (lane == 0) { chunk_den[warp] = lp; chunk_max[warp] = m; }
        }
        __syncthreads();
        if (warp < 4)
            for (int c = warp; c < min(kMergeWarps, u.n_chunks - c0); c += 4)       // c0 is a multiple of four
                add_chunk(a, l, chunk_sum[c][lane], chunk_den[c], chunk_weight(chunk_max[c], m_last, P.K));
        __syncthreads();
    }
    if (warp < 4) {
        sum[warp][lane] = a;
        if (lane == 0) den[warp] = l;
    }
    __syncthreads();
    r.store(P, sum, den);
}

template <int N, bool TILES>
cudaError_t launch_values(int producer, const FewParams& P, cudaStream_t stream)
{
    const dim3 grid(static_cast<unsigned>(P.n_units) << P.split);
    switch (producer) {
        case 0: return launch_overlapped(few_values_kernel<N, 0, TILES>, grid, kFewThreads, 0, stream, P);
        case 1: return launch_overlapped(few_values_kernel<N, 1, TILES>, grid, kFewThreads, 0, stream, P);
        case 2: return launch_overlapped(few_values_kernel<N, 2, TILES>, grid, kFewThreads, 0, stream, P);
        case 3: return launch_overlapped(few_values_kernel<N, 3, TILES>, grid, kFewThreads, 0, stream, P);
        case 4: return launch_overlapped(few_values_kernel<N, 4, TILES>, grid, kFewThreads, 0, stream, P);
        case 5: return launch_overlapped(few_values_kernel<N, 5, TILES>, grid, kFewThreads, 0, stream, P);
        case 6: return launch_overlapped(few_values_kernel<N, 6, TILES>, grid, kFewThreads, 0, stream, P);
        default: return cudaErrorInvalidValue;
    }
}

template <int N>
cudaError_t launch_n(int producer, const FewParams& P, cudaStream_t stream)
{
    cudaError_t e = launch_overlapped(few_scores_kernel<N>, dim3(static_cast<unsigned>(P.n_units) << P.split), kFewThreads, 0, stream, P);
    if (e != cudaSuccess) return e;
    e = P.split > 0 ? launch_values<N, true>(producer, P, stream) : launch_values<N, false>(producer, P, stream);
    if (e != cudaSuccess) return e;
    const dim3 rows(static_cast<unsigned>(P.n_heads), static_cast<unsigned>(P.row_cap));
    return P.split > 0 ? launch_overlapped(few_merge_tiles_kernel, rows, 32 * kMergeWarps, 0, stream, P) : launch_overlapped(few_merge_kernel, rows, 128, 0, stream, P);
}

}  // namespace

cudaError_t launch_few(int producer, FewParams& P, cudaStream_t stream)
{
    if (P.n_units <= 0) return cudaErrorInvalidValue;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return cudaErrorInvalidDevice;
    // Chunks in halves, quarters, eighths as long as every part has a tile and the blocks are all on the chip together (three on each
    // SM; with four or six 32 heads of 3000 keys 19.1 -> 19.2 and 22.8 us, 28 / 4 heads of 20000 22.0 -> 22.2 and 24.1).  Whole
    // chunks -> parts: one head of 2000 keys 12.0 -> 9.5 us, 32 / 8 heads of 3000 keys 14.3 -> 11.8, of 6000 19.9 -> 14.4, 16 rows of 4000
    // 35.7 -> 11.2.  Blocks without a tile cost more than they spread: chunks of one tile in eight, 32 / 8 heads of 700 keys
    // 10.1 -> 11.1 us, of 1500 10.8 -> 12.1, 10.1 and 10.8 with none; chunks of two in eight, four heads of 3000 keys 12.2, 10.1 with none.
    // The merge of parts has a block of 512 threads for every row, two on an SM at a time.  With more of them than that, parts of short
    // chunks cost more than they spread: whole -> parts 16 rows of 96 heads, 300 keys 17.0 -> 31.2 us, of 64 heads, 600 keys 16.4 -> 25.8, of
    // 32 heads, 984 keys 16.0 -> 18.9, 12 rows of 32 heads, 300 keys 13.9 -> 14.3, but of 24 heads 13.7 -> 12.7.  Of eight tiles they gain
    // with every number of rows that this leaves (16 rows of 32 heads, 4200 keys 39.5 -> 39.3, 6000 keys 48.9 -> 43.2, of 55 heads, 4096 keys
    // 50.7 -> 47.4).
    P.split = 0;
    const int sms = sm_count(dev);
    if (P.longest_chunk == kFewMaxChunk || static_cast<int64_t>(P.n_heads) * P.row_cap <= 2 * sms)
        while ((2 << P.split) <= P.longest_chunk && (static_cast<int64_t>(P.n_units) << (P.split + 1)) <= 3 * sms) ++P.split;
    if (P.row_cap <= 8) return launch_n<8>(producer, P, stream);
    if (P.row_cap <= 16) return launch_n<16>(producer, P, stream);
    return launch_n<24>(producer, P, stream);
}

FewPlan plan_few(int64_t keys_padded_all_heads, int rows)
{
    FewPlan w;
    size_t off = 0;
    auto take = [&](size_t bytes) { const size_t at = off; off = (off + bytes + 1023) / 1024 * 1024; return at; };
    w.scores = take(static_cast<size_t>(keys_padded_all_heads) * rows * sizeof(float));
    w.block_max = take(static_cast<size_t>(keys_padded_all_heads / 32) * rows * sizeof(float));
    w.stats = take(static_cast<size_t>(keys_padded_all_heads / kTile) * rows * kFewStatFloats * sizeof(float));
    w.total = off;
    return w;
}

}  // namespace efq
