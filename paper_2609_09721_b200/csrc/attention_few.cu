// Attention forward for few query rows (decode steps, short chunks): the rows of the query heads of a KV group - at
// most 24 of them - meet a long K/V of which every byte is used once.  What bounds it is the read of the bf16 K and V,
// so nothing of theirs goes back to memory: two streaming kernels quantise the tiles on their way into shared memory
// and feed them to the tensor core there.
//
//   few_scores_kernel   K tile -> MXFP4 operand; S^T[key, row] = K^ Q^^T (128 keys x 8..24 rows); raw scores and the
//                       maxima of the 32-key blocks go to the workspace (4 bytes per row and key against 256 of K)
//   few_values_kernel   the running maximum of every row before the chunk from the block maxima; Algorithm 1 with
//                       thread = key (a microscaling block is a warp); V tile -> MXFP4 operand, transposed;
//                       O^T[channel, row] += V^^T P~; the last chunk of a head to finish adds the chunks up
//
// The KV range is cut into chunks of kChunkTiles tiles whatever the batch, so the result of a sequence does not depend on
// its neighbours.  The shifted scores use the running maximum over all keys up to the tile (Algorithm 2), which the first
// kernel makes available to every chunk: the codes are those of the one-pass forward, bit for bit.
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
constexpr int kChunkTiles = kFewChunkTiles;
constexpr uint32_t kFewTmemCols = 128;      // four CTAs per SM share the 512 columns
constexpr uint32_t kColD = 0;               // 2 x 32
constexpr uint32_t kColSfA = 64;            // 2 x 4
constexpr uint32_t kColSfB = 72;            // 2 x 4

// One (sequence, KV head, chunk) of the grid.  Heads run fastest: the CTAs in flight read neighbouring heads of the same
// tokens, which lie side by side in a token-major cache.
struct Unit {
    int seq, head, chunk, n_chunks;
    int Sq, Sk, n_tiles;       // n_tiles: tiles that any row sees
    const __nv_bfloat16 *q, *k, *v;
    float* o;
    int64_t s_off;             // first score of the (sequence, head) in the workspace, rows Sk_pad apart
    int Sk_pad;
};

__device__ __forceinline__ Unit find_unit(const FewParams& P)
{
    Unit u;
    int id = static_cast<int>(blockIdx.x);
    int64_t kp;
    if (P.n_seqs == 0) {                    // [B, H, S, d]
        const int n_chunks = P.dense_chunks;
        u.head = id % P.Hkv;
        id /= P.Hkv;
        u.chunk = id % n_chunks;
        u.seq = id / n_chunks;
        u.n_chunks = n_chunks;
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
        u.n_chunks = ((s.Sk + kTile - 1) / kTile + kChunkTiles - 1) / kChunkTiles;
        kp = static_cast<int64_t>(s.k_pad0) ;
        u.q = P.q + s.q0 * P.q_row; u.k = P.k + s.k0 * P.k_row; u.v = P.v + s.k0 * P.k_row; u.o = P.o + s.q0 * P.q_row;
    }
    u.Sk_pad = (u.Sk + kTile - 1) / kTile * kTile;
    u.n_tiles = u.Sk_pad / kTile;
    u.q += static_cast<int64_t>(u.head) * P.G * P.q_head;
    u.o += static_cast<int64_t>(u.head) * P.G * P.q_head;
    u.k += u.head * P.k_head;
    u.v += u.head * P.k_head;
    u.s_off = (kp * P.Hkv + static_cast<int64_t>(u.head) * u.Sk_pad) * P.row_cap;
    return u;
}

// Bounded wait for a completion of this CTA's own MMAs.  On expiry the status word takes the error; the CTA carries on
// with whatever the accumulator holds, so that every thread still meets the block's barriers.
__device__ __forceinline__ void wait_mma(uint64_t* bar, uint32_t parity, uint32_t* status)
{
    for (int i = 0; i < 20000; ++i)
        if (ptx::mbar_try_wait_suspend(bar, parity, 50000u)) return;
    atomicExch(status, static_cast<uint32_t>(EFQ_ERR_DEVICE_TIMEOUT));
}

__device__ __forceinline__ float warp_max(float x)
{
    float m;
    asm("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(m) : "f"(x));
    return m;
}

// N consecutive columns (a multiple of 4) of this thread's TMEM lane
template <int N>
__device__ __forceinline__ void tmem_ld_cols(uint32_t addr, float (&d)[N])
{
#pragma unroll
    for (int i = 0; i < N; i += 4)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                     : "=f"(d[i]), "=f"(d[i + 1]), "=f"(d[i + 2]), "=f"(d[i + 3]) : "r"(addr + i) : "memory");
}

struct __align__(1024) FewSmem {
    uint8_t a[2][kTile * 64];       // K or V^T codes of a tile
    uint8_t b[2][32 * 64];          // Q codes ([0] only), or the probability operand of a tile
    uint8_t sf_a[2][512];
    uint8_t sf_b[2][512];
    float alpha[4][32];             // [tile mod 4][row]: a warp may be a tile ahead of one that still reads the tile before
    float m_start[32];
    float lsum[4][32];              // [key block of the tile][row]
    float bmax[kChunkTiles * 4][32];
    uint64_t mma_done[2];
    uint32_t tmem_base;
    uint32_t is_last;
};

__device__ __forceinline__ void few_setup(FewSmem* sm, int warp)
{
    if (warp == 0) ptx::tmem_alloc(&sm->tmem_base, kFewTmemCols);
    if (threadIdx.x == 32) {
        ptx::mbar_init(&sm->mma_done[0], 1);
        ptx::mbar_init(&sm->mma_done[1], 1);
        ptx::mbar_init_fence();
    }
    // rows and blocks that nobody writes: zero codes, byte 0
    for (int i = threadIdx.x; i < static_cast<int>(sizeof(sm->b) / 16); i += kFewThreads) reinterpret_cast<uint4*>(sm->b)[i] = make_uint4(0, 0, 0, 0);
    if (threadIdx.x < 64) reinterpret_cast<uint4*>(sm->sf_b)[threadIdx.x] = make_uint4(0, 0, 0, 0);
}

// D[128, N] = A B^T of one tile: two K = 64 steps, a fresh accumulator
__device__ __forceinline__ void few_mma(FewSmem* sm, uint32_t tmem, int buf, int b_buf, uint32_t n)
{
    const uint64_t d_sw64 = ptx::smem_desc(0, 16, 512, ptx::kLayoutSw64);
    const uint64_t d_sf = ptx::smem_desc(0, 16, 128, ptx::kLayoutNone);
    const uint32_t sfa = tmem + kColSfA + 4 * buf, sfb = tmem + kColSfB + 4 * b_buf, d = tmem + kColD + 32 * buf;
    ptx::tmem_cp_sf(sfa, d_sf + (ptx::smem_u32(sm->sf_a[buf]) >> 4));
    ptx::tmem_cp_sf(sfb, d_sf + (ptx::smem_u32(sm->sf_b[b_buf]) >> 4));
    const uint64_t da = d_sw64 + (ptx::smem_u32(sm->a[buf]) >> 4), db = d_sw64 + (ptx::smem_u32(sm->b[b_buf]) >> 4);
    ptx::mma_mxf4(d, da, db, ptx::mxf4_idesc(n, 0), sfa, sfb, 0u);
    ptx::mma_mxf4(d, da + 2, db + 2, ptx::mxf4_idesc(n, 2), sfa | (2u << 30), sfb | (2u << 30), 1u);
    ptx::mma_commit(&sm->mma_done[buf]);
}

// N: query rows rounded up to a multiple of 8 (the N of the MMA)
template <int N>
__global__ void __launch_bounds__(kFewThreads, 4) few_scores_kernel(const __grid_constant__ FewParams P)
{
    __shared__ FewSmem smem;
    FewSmem* const sm = &smem;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const Unit u = find_unit(P);
    const int R = P.G * u.Sq;
    if (blockIdx.x == 0) {                   // the status words, and the counters of the chunks that have finished
        P.status[tid] = 0u;
        for (int i = tid; i < P.n_counters; i += kFewThreads) P.counters[i] = 0u;
    }
    few_setup(sm, warp);
    __syncthreads();
    // Q: one thread per (row, block)
    if (tid < 4 * N) {
        const int row = tid >> 2, blk = tid & 3;
        uint32_t byte = 0;
        if (row < R) {
            const int g = row / u.Sq, tok = row - g * u.Sq;
            const uint4* src = reinterpret_cast<const uint4*>(u.q + g * P.q_head + tok * P.q_row + blk * 32);
            uint32_t w[16];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint4 x = __ldg(src + i);
                w[4 * i] = x.x; w[4 * i + 1] = x.y; w[4 * i + 2] = x.z; w[4 * i + 3] = x.w;
            }
            uint4 c;
            mxfp4_block(w, c, byte);
            *reinterpret_cast<uint4*>(sm->b[0] + code_tile_offset(row, blk)) = c;
            sm->sf_b[0][sf_tile_offset(row, blk)] = static_cast<uint8_t>(byte);
        }
    }
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::tc_fence_after_sync();
    const uint32_t tmem = sm->tmem_base;
    const int j0 = u.chunk * kChunkTiles, j1 = min(j0 + kChunkTiles, u.n_tiles);
    float* const S = P.scores + u.s_off;
    float* const bm = P.block_max + u.s_off / 32;
    const int nblk = u.Sk_pad / 32;
    constexpr int NH = N / 2;                // rows per half of the CTA; each half has one warp per 32 keys
    const int quarter = warp & 3, r_first = (warp >> 2) * NH;

    // raw scores of a finished tile: thread = key
    auto put_scores = [&](int j) {
        const int buf = j & 1;
        wait_mma(&sm->mma_done[buf], static_cast<uint32_t>((j - j0) >> 1) & 1u, P.status);
        ptx::tc_fence_after_sync();
        float s[NH];
        tmem_ld_cols<NH>(tmem + (static_cast<uint32_t>(quarter * 32) << 16) + kColD + 32 * buf + r_first, s);
        ptx::tmem_wait_ld();
        ptx::tc_fence_before_sync();
        const int key = j * kTile + quarter * 32 + lane;
#pragma unroll
        for (int i = 0; i < NH; ++i) {
            const int row = r_first + i;
            if (row < R) {
                const int tok = row % u.Sq;
                const int limit = P.causal ? min(tok + u.Sk - u.Sq, u.Sk - 1) : u.Sk - 1;
                const float x = key <= limit ? s[i] : -INFINITY;
                S[static_cast<int64_t>(row) * u.Sk_pad + key] = x;
                const float m = warp_max(x);
                if (lane == 0) bm[static_cast<int64_t>(row) * nblk + (key >> 5)] = m;
            }
        }
    };

    for (int j = j0; j < j1; ++j) {
        const int buf = j & 1;
        // two (key, block) pairs per thread; both loads set out before the tile before is finished with
        uint32_t w[2][16];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int key = j * kTile + (tid >> 2) + 64 * h;
            const uint4* src = reinterpret_cast<const uint4*>(u.k + key * P.k_row + (tid & 3) * 32);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint4 x = key < u.Sk ? __ldcs(src + i) : make_uint4(0, 0, 0, 0);
                w[h][4 * i] = x.x; w[h][4 * i + 1] = x.y; w[h][4 * i + 2] = x.z; w[h][4 * i + 3] = x.w;
            }
        }
        if (j > j0) put_scores(j - 1);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint32_t row = static_cast<uint32_t>(tid >> 2) + 64u * h;
            uint4 c;
            uint32_t byte;
            mxfp4_block(w[h], c, byte);
            *reinterpret_cast<uint4*>(sm->a[buf] + code_tile_offset(row, tid & 3)) = c;
            uint32_t word = byte;
            word |= __shfl_down_sync(0xffffffffu, byte, 1) << 8;
            word |= __shfl_down_sync(0xffffffffu, byte, 2) << 16;
            word |= __shfl_down_sync(0xffffffffu, byte, 3) << 24;
            if ((tid & 3) == 0) *reinterpret_cast<uint32_t*>(sm->sf_a[buf] + sf_tile_offset(row, 0)) = word;
        }
        ptx::fence_proxy_async_smem();
        ptx::tc_fence_before_sync();
        __syncthreads();
        if (warp == 0) {
            ptx::tc_fence_after_sync();
            if (ptx::elect_one()) few_mma(sm, tmem, buf, 0, N);
            __syncwarp();
        }
    }
    put_scores(j1 - 1);
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
        const float amax = warp_max(p);
        if (amax == 0.0f) { byte = 0u; return 0u; }
        const uint32_t bits = __float_as_uint(amax);
        const int E = static_cast<int>((bits >> 23) & 0xffu) - 127;
        int e = PRODUCER != 2 ? E - 2 : ((bits & 0x7fffffu) > 0x400000u ? E - 1 : E - 2);
        e = max(e, -127);
        byte = static_cast<uint32_t>(e + 127);
        return cvt_e2m1x2(p * __uint_as_float(static_cast<uint32_t>(127 - e) << 23), 0.0f) & 15u;
    }
}

template <int N, int PRODUCER>
__global__ void __launch_bounds__(kFewThreads, 3) few_values_kernel(const __grid_constant__ FewParams P)
{
    __shared__ FewSmem smem;
    FewSmem* const sm = &smem;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const Unit u = find_unit(P);
    const int R = P.G * u.Sq;
    few_setup(sm, warp);
    const int j0 = u.chunk * kChunkTiles, j1 = min(j0 + kChunkTiles, u.n_tiles);
    constexpr int NH = N / 2;
    const int half = warp >> 2, quarter = warp & 3;
    // V: a thread takes two channels of a 32-key block, a warp 128 contiguous bytes of every key
    const int ch = (tid & 63) * 2, kb = tid >> 6;
    uint32_t vv[32];
    auto load_v = [&](int j) {
        const int key0 = j * kTile + kb * 32;
        const uint32_t* src = reinterpret_cast<const uint32_t*>(u.v + key0 * P.k_row + ch);
        const int64_t step = P.k_row / 2;
#pragma unroll
        for (int i = 0; i < 32; ++i) vv[i] = key0 + i < u.Sk ? __ldcs(src + i * step) : 0u;
    };
    load_v(j0);                              // an input: needs nothing of the scores kernel
    asm volatile("griddepcontrol.wait;" ::: "memory");

    // running maximum of every row before the chunk, and the chunk's own block maxima
    const float* bm = P.block_max + u.s_off / 32;
    const int nblk = u.Sk_pad / 32;
    if (!(P.rescale_threshold > 0.0f)) {
        for (int row = warp; row < R; row += 8) {
            float m = -INFINITY;
            for (int b = lane; b < j0 * 4; b += 32) m = fmaxf(m, __ldcg(bm + static_cast<int64_t>(row) * nblk + b));
            m = warp_max(m);
            if (lane == 0) sm->m_start[row] = m;
        }
    } else if (tid < R) {                    // optional policy: the kept maximum depends on the order of the tiles
        float m = -INFINITY;
        for (int j = 0; j < j0; ++j) {
            const float4 b = __ldcg(reinterpret_cast<const float4*>(bm + static_cast<int64_t>(tid) * nblk + 4 * j));
            const float c = fmaxf(m, fmaxf(fmaxf(b.x, b.y), fmaxf(b.z, b.w)));
            if (m == -INFINITY || __fsub_rn(__fmul_rn(P.K.sigma, c), __fmul_rn(P.K.sigma, m)) > P.rescale_threshold) m = c;
        }
        sm->m_start[tid] = m;
    }
    for (int i = tid; i < R * kChunkTiles * 4; i += kFewThreads) {
        const int row = i / (kChunkTiles * 4), b = i % (kChunkTiles * 4);
        if (j0 * 4 + b < nblk) sm->bmax[b][row] = __ldcg(bm + static_cast<int64_t>(row) * nblk + j0 * 4 + b);
    }
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::tc_fence_after_sync();
    const uint32_t tmem = sm->tmem_base;
    const float* const S = P.scores + u.s_off;

    // lane-parallel row state: lane i keeps the maximum and the denominator (this warp's key blocks) of row 2 i + half
    const int my_row = 2 * lane + half;
    const bool has_row = lane < NH && my_row < R;
    float m_run = has_row ? sm->m_start[my_row] : -INFINITY;
    float l_run = 0.0f;
    float acc[NH];                           // O^T: channel = TMEM lane of this thread, rows half * NH + i
#pragma unroll
    for (int i = 0; i < NH; ++i) acc[i] = 0.0f;

    auto add_tile = [&](int j) {
        const int buf = j & 1;
        wait_mma(&sm->mma_done[buf], static_cast<uint32_t>((j - j0) >> 1) & 1u, P.status);
        ptx::tc_fence_after_sync();
        float d[NH];
        tmem_ld_cols<NH>(tmem + (static_cast<uint32_t>(quarter * 32) << 16) + kColD + 32 * buf + half * NH, d);
        ptx::tmem_wait_ld();
        ptx::tc_fence_before_sync();
#pragma unroll
        for (int i = 0; i < NH; ++i) acc[i] = fmaf(acc[i], sm->alpha[j & 3][half * NH + i], d[i]);
    };

    // optional dump of one query head (all lanes; byte and m_s are the block's and the tile's)
    const bool dump = P.has_dbg && u.seq == P.dbg.batch && u.head == P.dbg.head / P.G;
    auto dump_row = [&](int j, int row, float score, uint32_t word, float m_s, uint32_t byte) {
        const int g = row / u.Sq, tok = row - g * u.Sq, blk = j * 4 + quarter, key = blk * 32 + lane;
        if (u.head * P.G + g != P.dbg.head || tok < P.dbg.q_begin || tok >= P.dbg.q_end) return;
        const int64_t drow = tok - P.dbg.q_begin, blocks = (u.Sk + 31) / 32;
        if (P.dbg.raw_scores != nullptr && key < u.Sk) P.dbg.raw_scores[drow * u.Sk + key] = score;
        if (P.dbg.row_max != nullptr && quarter == 0 && lane == 0) P.dbg.row_max[drow * u.n_tiles + j] = m_s;
        if (blk >= blocks) return;
        if (P.dbg.codes != nullptr && (lane & 7) == 0) reinterpret_cast<uint32_t*>(P.dbg.codes + (drow * blocks + blk) * 16)[lane >> 3] = word;
        if (P.dbg.scales != nullptr && lane == 0) P.dbg.scales[drow * blocks + blk] = static_cast<uint8_t>(byte);
    };

    for (int j = j0; j < j1; ++j) {
        const int buf = j & 1;
        // ---- row state of the tile (Eq. rowmax-update, Eq. alpha) and the row's part of the scale rule, one row per lane
        float par = 0.0f, bmax = -INFINITY, m_s = -INFINITY;
        uint32_t byte = 0u;
        bool live = false;
        if (has_row) {
            const float* b4 = &sm->bmax[(j - j0) * 4][my_row];
            bmax = b4[32 * quarter];
            float m_new = fmaxf(m_run, fmaxf(fmaxf(b4[0], b4[32]), fmaxf(b4[64], b4[96])));
            if (P.rescale_threshold > 0.0f && m_run != -INFINITY &&
                !(__fsub_rn(__fmul_rn(P.K.sigma, m_new), __fmul_rn(P.K.sigma, m_run)) > P.rescale_threshold))
                m_new = m_run;
            m_s = __fmul_rn(P.K.sigma, m_new);
            const bool grew = m_new > m_run && m_run != -INFINITY;
            const float alpha = grew ? ex2_approx(__fmul_rn(__fsub_rn(__fmul_rn(P.K.sigma, m_run), m_s), P.K.LOG2E)) : 1.0f;
            m_run = m_new;
            l_run *= alpha;
            if (quarter == 0) sm->alpha[j & 3][my_row] = alpha;
            live = bmax != -INFINITY;
            if (PRODUCER == 0 || PRODUCER == 3) {
                const BlockScale s = efq_block_scale(bmax, m_s, P.K);
                par = s.Bb; byte = s.byte;
            } else if (PRODUCER == 4 || PRODUCER == 5) {
                const FoldedScale f = etq_folded_scale(bmax, m_s, P.K);
                par = f.c0e; byte = f.byte;
            } else {
                par = m_s;
            }
        } else if (quarter == 0 && lane < NH) {
            sm->alpha[j & 3][my_row] = 1.0f;
        }
        // ---- Algorithm 1, thread = key: codes of the rows of this half
        const float* s_tile = S + j * kTile + quarter * 32 + lane;
        float x[NH];
#pragma unroll
        for (int i = 0; i < NH; ++i) x[i] = 2 * i + half < R ? __ldcg(s_tile + static_cast<int64_t>(2 * i + half) * u.Sk_pad) : -INFINITY;
        int count = 0;                       // of lane i: twice the sum of its row's E2M1 values in this block
        float psum = 0.0f;
#pragma unroll
        for (int i = 0; i < NH; ++i) {
            const int row = 2 * i + half;
            if (row < R) {
                uint32_t b = 0u;
                float p = 0.0f;
                uint32_t c = key_code<PRODUCER>(x[i], __shfl_sync(0xffffffffu, par, i), P.K, lane, b, p);
                if (PRODUCER == 4 || PRODUCER == 5) c = __shfl_sync(0xffffffffu, live, i) ? c : 0u;
                const int n = __reduce_add_sync(0xffffffffu, static_cast<int>((0xC8643210u >> (4u * c)) & 15u));
                if (PRODUCER == 6)
                    for (int o = 16; o > 0; o >>= 1) p += __shfl_xor_sync(0xffffffffu, p, o);
                if (lane == i) {
                    count = n;
                    psum = p;
                    if (PRODUCER == 1 || PRODUCER == 2 || PRODUCER == 6) byte = b;
                }
                c |= __shfl_down_sync(0xffffffffu, c, 1) << 4;
                c |= __shfl_down_sync(0xffffffffu, c, 2) << 8;
                c |= __shfl_down_sync(0xffffffffu, c, 4) << 16;
                if (dump) dump_row(j, row, x[i], c, __shfl_sync(0xffffffffu, m_s, i), __shfl_sync(0xffffffffu, byte, i));
                if ((lane & 7) == 0) *reinterpret_cast<uint32_t*>(sm->b[buf] + code_tile_offset(row, quarter) + (lane >> 1)) = c;
            }
        }
        if (has_row) {
            sm->sf_b[buf][sf_tile_offset(my_row, quarter)] = static_cast<uint8_t>(byte);
            l_run += PRODUCER == 6 ? psum : static_cast<float>(count) * 0.5f * (byte != 0u ? __uint_as_float(byte << 23) : __uint_as_float(0x00400000u));
        }
        // ---- V^T operand of the tile
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            uint32_t w[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) w[i] = __byte_perm(vv[2 * i], vv[2 * i + 1], h == 0 ? 0x5410 : 0x7632);
            uint4 c;
            uint32_t vb;
            mxfp4_block(w, c, vb);
            *reinterpret_cast<uint4*>(sm->a[buf] + code_tile_offset(ch + h, kb)) = c;
            sm->sf_a[buf][sf_tile_offset(ch + h, kb)] = static_cast<uint8_t>(vb);
        }
        if (j + 1 < j1) load_v(j + 1);
        ptx::fence_proxy_async_smem();
        ptx::tc_fence_before_sync();
        __syncthreads();
        if (warp == 0) {
            ptx::tc_fence_after_sync();
            if (ptx::elect_one()) few_mma(sm, tmem, buf, buf, N);
            __syncwarp();
        }
        if (j > j0) add_tile(j - 1);
    }
    add_tile(j1 - 1);
    if (has_row) sm->lsum[quarter][my_row] = l_run;
    if (quarter == 0 && has_row) sm->m_start[my_row] = __fmul_rn(P.K.sigma, m_run);   // scaled maximum the chunk refers to
    ptx::tc_fence_before_sync();
    __syncthreads();
    if (warp == 0) ptx::tmem_dealloc(tmem, kFewTmemCols);

    const int channel = quarter * 32 + lane;
    auto l_of = [&](int row) { return (sm->lsum[0][row] + sm->lsum[1][row]) + (sm->lsum[2][row] + sm->lsum[3][row]); };
    auto out_row = [&](int row) { const int g = row / u.Sq; return u.o + g * P.q_head + (row - g * u.Sq) * P.q_row; };
    if (u.n_chunks == 1) {
#pragma unroll
        for (int i = 0; i < NH; ++i) {
            const int row = half * NH + i;
            if (row < R) {
                const float l = l_of(row);
                out_row(row)[channel] = acc[i] * (l > 0.0f ? 1.0f / l : 0.0f);
            }
        }
        return;
    }
    // ---- partial result of the chunk; the last chunk of the head to arrive adds them up
    const size_t part_floats = static_cast<size_t>(P.row_cap) * 130;     // [row][128] | maximum [row] | denominator [row]
    float* const part = P.partials + blockIdx.x * part_floats;
#pragma unroll
    for (int i = 0; i < NH; ++i) {
        const int row = half * NH + i;
        if (row < R) part[row * 128 + channel] = acc[i];
    }
    if (tid < R) {
        part[P.row_cap * 128 + tid] = sm->m_start[tid];
        part[P.row_cap * 129 + tid] = l_of(tid);
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) sm->is_last = atomicAdd(P.counters + (u.seq * P.Hkv + u.head), 1u) == static_cast<uint32_t>(u.n_chunks - 1);
    __syncthreads();
    if (sm->is_last == 0u) return;
    __threadfence();
    const float* const first = P.partials + (blockIdx.x - static_cast<size_t>(u.chunk) * P.Hkv) * part_floats;
    const size_t step = part_floats * P.Hkv;
    for (int row = tid >> 7; row < R; row += 2) {
        const int c_ch = tid & 127;
        const float m_last = __ldcg(first + (u.n_chunks - 1) * step + P.row_cap * 128 + row);
        float a = 0.0f, l = 0.0f;
#pragma unroll 4
        for (int c = 0; c < u.n_chunks; ++c) {
            const float* p = first + c * step;
            const float m = __ldcg(p + P.row_cap * 128 + row);
            const float w = m == -INFINITY ? 0.0f : ex2_approx(__fmul_rn(__fsub_rn(m, m_last), P.K.LOG2E));
            l = fmaf(__ldcg(p + P.row_cap * 129 + row), w, l);
            a = fmaf(__ldcg(p + row * 128 + c_ch), w, a);
        }
        out_row(row)[c_ch] = a * (l > 0.0f ? 1.0f / l : 0.0f);
    }
}

template <int N, int PRODUCER>
cudaError_t launch_values(unsigned units, const FewParams& P, cudaStream_t stream)
{
    // may start while the last scores CTAs still run: its first V tile does not depend on them
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(units);
    cfg.blockDim = dim3(kFewThreads);
    cfg.stream = stream;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, few_values_kernel<N, PRODUCER>, P);
}

template <int N>
cudaError_t launch_n(int producer, unsigned units, const FewParams& P, cudaStream_t stream)
{
    few_scores_kernel<N><<<units, kFewThreads, 0, stream>>>(P);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    switch (producer) {
        case 0: return launch_values<N, 0>(units, P, stream);
        case 1: return launch_values<N, 1>(units, P, stream);
        case 2: return launch_values<N, 2>(units, P, stream);
        case 3: return launch_values<N, 3>(units, P, stream);
        case 4: return launch_values<N, 4>(units, P, stream);
        case 5: return launch_values<N, 5>(units, P, stream);
        case 6: return launch_values<N, 6>(units, P, stream);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

cudaError_t launch_few(int producer, int64_t units, const FewParams& P, cudaStream_t stream)
{
    if (units <= 0 || units > 0x7fffffffll) return cudaErrorInvalidValue;
    const unsigned n = static_cast<unsigned>(units);
    if (P.row_cap <= 8) return launch_n<8>(producer, n, P, stream);
    if (P.row_cap <= 16) return launch_n<16>(producer, n, P, stream);
    return launch_n<24>(producer, n, P, stream);
}

FewPlan plan_few(int64_t units, int64_t heads, int64_t keys_padded_all_heads, int rows)
{
    FewPlan w;
    size_t off = 0;
    auto take = [&](size_t bytes) { const size_t at = off; off = (off + bytes + 1023) / 1024 * 1024; return at; };
    w.scores = take(static_cast<size_t>(keys_padded_all_heads) * rows * sizeof(float));
    w.block_max = take(static_cast<size_t>(keys_padded_all_heads / 32) * rows * sizeof(float));
    w.partials = take(static_cast<size_t>(units) * rows * 130 * sizeof(float));
    w.counters = take(static_cast<size_t>(heads) * sizeof(uint32_t));
    w.total = off;
    return w;
}

}  // namespace efq
