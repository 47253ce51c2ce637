// Fused block-scaled FP4 attention forward with in-register probability generation
// (Algorithm 2 looped over KV tiles, Algorithm 1 per 32-key microscaling block), sm_100a.
//
// One CTA owns one 128-row query tile of one (batch, head) and walks the KV tiles of width 128:
//   warp 0      TMA producer: Q tile once, then K_j / V^T_j code tiles (SW64 layout) and their
//               512-byte scale tiles through 4-stage mbarrier rings
//   warps 1, 2  MMA issuers (one elected lane each): scale tiles smem -> TMEM (tcgen05.cp), then warp 1
//               S_j = Q^ K^_j^T  and warp 2  [dA | dl] = P~_j [V^_j | 1]  as kind::mxf4 block-scaled MMAs,
//               FP32 accumulators in TMEM; S runs up to two tiles ahead of P~V.  The 16 "ones" rows appended to V^T give the denominator
//               P~1 from the very operand that feeds the numerator.
//   warps 12-15 historical rescaling: when a row's maximum grew in tile j, its accumulator row and denominator in
//               TMEM are multiplied by alpha_j after P~V_{j-1} and before P~V_j, beside the code generation.
//   warps 4-11  probability generation, two groups of four warps: group 0 takes the even KV tiles,
//               group 1 the odd ones, so one group's latency-bound steps (TMEM load, hand-over of the
//               running maximum, accumulator rescaling) overlap the other group's code generation.
//               Thread = query row: the 128 scores of the row come from TMEM straight into registers;
//               block maxima, scale and codes are thread-local; codes go as 16-byte packed stores into
//               the swizzled shared-memory A operand, the four scale bytes as one word into the scale
//               tile.  No FP16/FP32 probability tile exists anywhere.  Per tile a warp publishes once (running
//               maximum, alpha, hand-back of the S buffer), asks each barrier one step before it needs the
//               answer, and sends for the scores of its next tile as soon as its registers are free.
// The online recurrence is unchanged: when a row's maximum grows, the accumulator rows in TMEM
// are rescaled by alpha = exp(m_old - m_new) before the next P~V MMA is released (warps 12-15).
//
// TMEM columns: S double buffer 2 x 128 | O 144 (128 channels + 16 denominator) | scale factors.
// Every wait is bounded: one thread of warp 3 watches whether P~V goes on, and if it does not the CTA records EFQ_ERR_DEVICE_TIMEOUT
// in the workspace status word, all roles drain, TMEM is released and the kernel returns.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <mutex>
#include <vector>

#include "efq_common.cuh"
#include "efq_internal.cuh"
#include "efq_producers.cuh"
#include "item_order.h"
#include "mxfp4.cuh"
#include "sm100_ptx.cuh"

namespace efq {

namespace {

constexpr int kTile = 128;            // query rows per CTA and keys per KV tile (Bc)
constexpr int kStages = 4;            // K and V ring depth
constexpr int kThreads = 512;         // 16 warps = 4 warpgroups: {TMA, QK, PV, idle}, 2 x probability generation, rescaling
constexpr int kGroupWarps = 4;        // warps per probability group (one thread per query row)
constexpr int kTileBytes = kTile * 64;          // 128 rows x 64 B of packed E2M1
constexpr int kSfBytes = 512;
constexpr int kVStageBytes = kTileBytes + 1024; // + 16 ones rows
constexpr int kOutRowBytes = 528;       // staging row of the output: 512 bytes that start 4 banks apart, so that 128-bit stores
                                        // of a warp (a row per lane) do not collide
constexpr uint32_t kTimeoutCycles = 1500000000u;

// TMEM column map
constexpr uint32_t kColS = 0;         // 2 x 128
constexpr uint32_t kColO = 256;       // 144
constexpr uint32_t kColSfQ = 400;     // 4
constexpr uint32_t kColSfK = 404;     // 2 x 4
constexpr uint32_t kColSfP = 412;     // 2 x 4
constexpr uint32_t kColSfV = 420;     // 2 x 8 (4 for V, 4 for the ones rows)
constexpr uint32_t kTmemCols = 512;

struct __align__(1024) Smem {
    uint8_t q[kTileBytes];
    uint8_t k[kStages][kTileBytes];     // k and v together: staging of the finished rows, once every load has been consumed
    uint8_t v[kStages][kVStageBytes];
    uint8_t p[2][kTileBytes];
    uint8_t sf_q[kSfBytes];
    uint8_t sf_k[kStages][kSfBytes];
    uint8_t sf_v[kStages][kSfBytes];
    uint8_t sf_p[2][kSfBytes];
    uint8_t sf_ones[kSfBytes];
    float lsum_x[2][kTile];   // FP32-denominator baseline only: each group's sum of exponentials ...
    float mref_x[2][kTile];   // ... and the scaled maximum it refers to
    float runmax[2][kTile];   // running row maximum after the group's latest tile, raw score units
    float alpha[4][kTile];    // [tile mod 4]: rescale factor of the tile, per row (1 where the maximum did not grow)
    uint64_t q_full;
    uint64_t k_full[kStages], k_empty[kStages];
    uint64_t v_full[kStages], v_empty[kStages];
    uint64_t s_full[2], s_empty[2];
    uint64_t p_full[2], p_empty[2];
    uint64_t a_bar[4][4];     // [tile mod 4][lane quarter]: running maximum and alpha of that tile are published
    uint64_t o_ready[4];      // [tile mod 4]: accumulator rows rescaled (or found unchanged) for that tile
    uint64_t o_done;          // the last P~V of the work item has completed
    uint64_t l_bar;           // FP32-denominator baseline only: all eight probability warps have written lsum_x / mref_x
    uint32_t tmem_base;
    volatile uint32_t abort_flag;
    volatile uint32_t progress; // tiles whose P~V has been issued
};

static_assert(sizeof(Smem::k) + sizeof(Smem::v) >= kTile * kOutRowBytes, "finished rows fit where K and V were");

struct FwdParams {
    int B, Hq, Hkv;
    int64_t Sq, Sk, Sq_pad, Sk_pad;
    int causal;
    ProducerConsts K;
    const uint8_t* sf_q;      // [B*Hq*Sq_pad/128][512]
    const uint8_t* sf_k;      // [B*Hkv*Sk_pad/128][512]
    const uint8_t* sf_v;
    float* o;
    int64_t o_tokens;         // packed batch: query tokens in all
    int64_t o_head, o_row;    // strides of o in elements: row i of (batch b, head h) starts at o[(b * Hq + h) * o_head + i * o_row]
    uint32_t* status;
    efq_debug_t dbg;
    int has_dbg;
    int packed;               // dense batch with few query tokens: the query heads of a KV group share one query tile
    const SeqDesc* seqs;      // packed variable-length batch: sequence table and one item per CTA (device memory);
    const ItemDesc* items;    //   NULL for a [B, H, S, d] batch, whose items follow from the block index
    uint32_t heads_magic;     // [B, H, S, d]: ceil(2^32 / (B * Hq)), 0 for one head (persistent kernel)
    int64_t v_tiles_per_head; // packed batch: 128-key tiles per KV head in the V^T code matrix (all sequences)
    int inject_skip_loads;    // test hook: the TMA thread loads Q only, so the first wait on K/V runs out
    float rescale_threshold;  // 0: Algorithm 2; > 0: the shifting maximum is kept while the true one is at most this far above
};

// Waits end with the completion or, false, when the CTA gave up.  That is one warp's business (wait_watching): the kernels inline
// some twenty-five waits, and a clock in each of them made a sixth of the code, which outgrows the instruction cache as it is.
__device__ __forceinline__ bool wait1(uint64_t* bar, uint32_t parity, Smem* sm)
{
#pragma unroll 1
    while (!ptx::mbar_try_wait(bar, parity))
        if (sm->abort_flag) return false;
    return true;
}
// The same wait executed by all lanes of a warp.  All lanes poll the same barrier; only the rare timeout path
// can split a warp, so the verdict is made warp-uniform there and nowhere else.
__device__ __forceinline__ bool wait_all(uint64_t* bar, uint32_t parity, Smem* sm)
{
    if (ptx::mbar_try_wait(bar, parity)) return true;
    return __all_sync(__activemask(), wait1(bar, parity, sm));
}
// The watch over all waits of the CTA, by the one thread that waits for its result: between two of its own polls it looks whether
// P~V goes on.  Without another tile within the limit the CTA gives up, and the status word says so.
__device__ __forceinline__ bool wait_watching(uint64_t* bar, uint32_t parity, Smem* sm, uint32_t* status)
{
    uint32_t t0 = ptx::clock32(), seen = sm->progress;
#pragma unroll 1
    while (!ptx::mbar_try_wait(bar, parity)) {
        if (sm->abort_flag) return false;
        const uint32_t now = sm->progress;
        if (now != seen) { seen = now; t0 = ptx::clock32(); }
        if (ptx::clock32() - t0 > kTimeoutCycles) {
            sm->abort_flag = 1u;
            atomicExch(status, static_cast<uint32_t>(EFQ_ERR_DEVICE_TIMEOUT));
            return false;
        }
    }
    return true;
}

// o[0 .. 31] *= a, two at a time
__device__ __forceinline__ void scale32(uint32_t* o, uint64_t a)
{
#pragma unroll
    for (int i = 0; i < 32; i += 2) {
        uint64_t v;
        asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "r"(o[i]), "r"(o[i + 1]));
        asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(v) : "l"(v), "l"(a));
        asm("mov.b64 {%0, %1}, %2;" : "=r"(o[i]), "=r"(o[i + 1]) : "l"(v));
    }
}

template <int PRODUCER, bool DEBUG>
__global__ void __launch_bounds__(kThreads, 1)
attention_fwd_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                     const __grid_constant__ CUtensorMap map_v, const FwdParams P)
{
    extern __shared__ uint8_t smem_raw[];
    Smem* sm = reinterpret_cast<Smem*>(smem_raw + ptx::smem_round_up(smem_raw, 1024u));
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;

    // ---- work item.  [B, H, S, d] batch: heaviest query tiles first, the heads of a GQA group adjacent.  Packed
    // variable-length batch: the item and its sequence come from the tables.  Either way the item is one 128-row
    // query tile: rows q0 .. q0 + 127 of query head head0, or - "packed", when the sequence has so few query tokens
    // that the G query heads of a KV group fit into one tile - row r = token r % Sq of query head head0 + r / Sq.
    const int G = P.Hq / P.Hkv;
    int64_t Sq, Sk, o_base, q0;
    int b, head0, hkv, q_row, k_row0, v_x0, v_y0;
    int64_t sfv_tile0;
    bool packed;
    if (P.items != nullptr) {
        ptx::grid_wait();                                     // the item table is written by the kernel before
        const ItemDesc it = P.items[blockIdx.x];
        const SeqDesc sd = P.seqs[it.seq];
        Sq = sd.Sq; Sk = sd.Sk; o_base = sd.o_off; b = it.seq;
        packed = sd.packed != 0;
        if (packed) { hkv = it.head; head0 = hkv * G; q0 = 0; q_row = sd.q_row0 + hkv * kTile; }
        else { head0 = it.head; hkv = head0 / G; q0 = static_cast<int64_t>(it.qt) * kTile; q_row = sd.q_row0 + head0 * sd.Sq_pad + it.qt * kTile; }
        k_row0 = sd.k_row0 + hkv * sd.Sk_pad;
        v_x0 = sd.k_col0 / 2;
        v_y0 = hkv * kTile;
        sfv_tile0 = static_cast<int64_t>(hkv) * P.v_tiles_per_head + sd.k_col0 / kTile;
    } else {
        Sq = P.Sq; Sk = P.Sk;
        packed = P.packed != 0;
        // 32-bit arithmetic: a 64-bit division costs hundreds of cycles that nothing hides here
        const uint32_t n_qtiles = packed ? 1u : static_cast<uint32_t>(P.Sq_pad / kTile);
        const uint32_t heads = packed ? P.Hkv : P.Hq;         // heads that own query tiles
        const uint32_t bh_count = P.B * heads;
        const uint32_t qt = n_qtiles - 1u - blockIdx.x / bh_count;
        const uint32_t bh = blockIdx.x % bh_count;
        b = static_cast<int>(bh / heads);
        const int hh = static_cast<int>(bh % heads);
        if (packed) { hkv = hh; head0 = hkv * G; q0 = 0; q_row = static_cast<int>(bh * kTile); }
        else { head0 = hh; hkv = hh / G; q0 = static_cast<int64_t>(qt) * kTile; q_row = static_cast<int>(bh * static_cast<uint32_t>(P.Sq_pad) + q0); }
        const int64_t kvh = static_cast<int64_t>(b) * P.Hkv + hkv;
        k_row0 = static_cast<int>(kvh * P.Sk_pad);
        v_x0 = 0;
        v_y0 = static_cast<int>(kvh * kTile);
        sfv_tile0 = kvh * (P.Sk_pad / kTile);
        o_base = static_cast<int64_t>(b) * P.Hq * P.o_head;
    }
    const int64_t shift = Sk - Sq;                         // causal: query i sees keys <= i + shift
    int n_tiles = static_cast<int>((Sk + kTile - 1) / kTile);          // shapes stay below 2^31 rows: 32-bit tile counters
    if (P.causal) {
        int64_t last_row = packed ? Sq - 1 : (q0 + kTile - 1 < Sq ? q0 + kTile - 1 : Sq - 1);
        int64_t last_key = last_row + shift;               // may be negative: nothing visible
        const int need = last_key < 0 ? 0 : static_cast<int>(last_key / kTile) + 1;
        if (need < n_tiles) n_tiles = need;
    }

    // ---- setup.  Warp 0 makes the barriers and goes on to load at once; the others wait for it in a named barrier that it
    // only arrives at.
    if (warp == 0) {
        if (lane == 0) {
            ptx::prefetch_tensormap(&map_q);
            ptx::prefetch_tensormap(&map_k);
            ptx::prefetch_tensormap(&map_v);
            sm->abort_flag = 0u;
            sm->progress = 0u;
            ptx::mbar_init(&sm->q_full, 1);
            ptx::mbar_init(&sm->o_done, 1);
            ptx::mbar_init(&sm->l_bar, 2 * kGroupWarps);
            for (int s = 0; s < kStages; ++s) {
                ptx::mbar_init(&sm->k_full[s], 1);
                ptx::mbar_init(&sm->k_empty[s], 1);
                ptx::mbar_init(&sm->v_full[s], 1);
                ptx::mbar_init(&sm->v_empty[s], 1);
            }
            for (int i = 0; i < 2; ++i) {
                ptx::mbar_init(&sm->s_full[i], 1);
                ptx::mbar_init(&sm->s_empty[i], kGroupWarps);
                ptx::mbar_init(&sm->p_full[i], kGroupWarps);
                ptx::mbar_init(&sm->p_empty[i], 1);
            }
            for (int i = 0; i < 4; ++i) ptx::mbar_init(&sm->o_ready[i], 4);
            for (int i = 0; i < 4; ++i)
                for (int qd = 0; qd < 4; ++qd) ptx::mbar_init(&sm->a_bar[i][qd], 1);
            ptx::mbar_init_fence();
        }
        __syncwarp();
        asm volatile("bar.arrive 1, 512;" ::: "memory");
    } else {
        if (warp == 1) ptx::tmem_alloc(&sm->tmem_base, kTmemCols);
        // constant parts of the B operand of P~V: 16 rows of E2M1 1.0 (0x22) after each V^T stage, unit scales
        for (int i = threadIdx.x - 32; i < kStages * 64; i += kThreads - 32)
            reinterpret_cast<uint4*>(sm->v[i / 64] + kTileBytes)[i % 64] = make_uint4(0x22222222u, 0x22222222u, 0x22222222u, 0x22222222u);
        for (int i = threadIdx.x - 32; i < kSfBytes / 4; i += kThreads - 32)
            reinterpret_cast<uint32_t*>(sm->sf_ones)[i] = (i < 64 && (i & 3) == 0) ? 0x7f7f7f7fu : 0u;
        ptx::fence_proxy_async_smem();
        ptx::tc_fence_before_sync();
        asm volatile("bar.sync 1, 512;" ::: "memory");
        ptx::tc_fence_after_sync();
    }
    const uint32_t tmem = warp == 0 ? 0u : sm->tmem_base;
    const bool run = n_tiles > 0;

    // Register budget: the probability warpgroups take what the other two give up.  setmaxnreg moves registers
    // inside the CTA's own allocation only (512 threads x 128 at launch = 16 x 128 per lane), so the budgets must
    // add up to no more than that: 4 x 32 + 8 x 184 + 4 x 112 = 2048.  A role that asks for more waits for good.
    if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 32;");
    if (run && warp == 0 && lane == 0) {
        // =============================== TMA producer (one thread) ===============================
        // The operands come from the kernel before.  Whatever else this kernel writes or reads follows from the loads.
        ptx::grid_wait();
        ptx::mbar_arrive_expect_tx(&sm->q_full, kTileBytes + kSfBytes);
        ptx::tma_load_2d(sm->q, &map_q, 0, q_row, &sm->q_full);
        ptx::bulk_load_1d(sm->sf_q, P.sf_q + static_cast<int64_t>(q_row / kTile) * kSfBytes, kSfBytes, &sm->q_full);
        const int64_t sfk_tile0 = k_row0 / kTile;
        int s = 0;
        uint32_t ph = 0;
        for (int j = 0; j < (P.inject_skip_loads ? 0 : n_tiles); ++j) {
            // Stage barriers of their own: a waiter on a barrier that other roles may complete twice before it
            // looks (S runs ahead) could not tell which completion it sees by parity.
            if (!wait1(&sm->k_empty[s], ph ^ 1u, sm)) break;
            ptx::mbar_arrive_expect_tx(&sm->k_full[s], kTileBytes + kSfBytes);
            ptx::tma_load_2d(sm->k[s], &map_k, 0, k_row0 + static_cast<int>(j * kTile), &sm->k_full[s]);
            ptx::bulk_load_1d(sm->sf_k[s], P.sf_k + (sfk_tile0 + j) * kSfBytes, kSfBytes, &sm->k_full[s]);
            if (!wait1(&sm->v_empty[s], ph ^ 1u, sm)) break;
            ptx::mbar_arrive_expect_tx(&sm->v_full[s], kTileBytes + kSfBytes);
            ptx::tma_load_2d(sm->v[s], &map_v, v_x0 + static_cast<int>(j * 64), v_y0, &sm->v_full[s]);
            ptx::bulk_load_1d(sm->sf_v[s], P.sf_v + (sfv_tile0 + j) * kSfBytes, kSfBytes, &sm->v_full[s]);
            if (++s == kStages) { s = 0; ph ^= 1u; }
        }
    } else if (warp == 3 && lane == 0) {
        ptx::grid_wait();
        // an earlier CTA of this launch gave up: the waits of this one end soon instead of after their limit
        if (*reinterpret_cast<volatile uint32_t*>(P.status) != 0u) sm->abort_flag = 1u;
        // No early launch of what follows: the next call's blocks get in the way of this one's (36 heads, causal, 512 tokens 10.2 us, with it
        // 11.2; one head, 8192 tokens 51.2 and 51.6).
        if (run) wait_watching(&sm->o_done, 0, sm, P.status);
    } else if (run && warp == 1) {
        // =============================== S = Q K^T issuer ===============================
        // The whole warp runs the loop with warp-uniform state; one elected lane issues the tcgen05
        // instructions.  Descriptors differ from tile to tile only in the start-address field (address >> 4).
        const uint64_t d_sw64 = ptx::smem_desc(0, 16, 512, ptx::kLayoutSw64);
        const uint64_t d_sf = ptx::smem_desc(0, 16, 128, ptx::kLayoutNone);
        const uint64_t dq0 = d_sw64 + (ptx::smem_u32(sm->q) >> 4);
        const uint32_t sfq = tmem + kColSfQ;
        bool ok = wait_all(&sm->q_full, 0, sm);
        ptx::tc_fence_after_sync();
        if (ok && ptx::elect_one()) ptx::tmem_cp_sf(sfq, d_sf + (ptx::smem_u32(sm->sf_q) >> 4));
        int ks = 0;
        uint32_t kph = 0;
        for (int t = 0; ok && t < n_tiles; ++t) {
            const int sb = static_cast<int>(t & 1);
            if (!wait_all(&sm->k_full[ks], kph, sm)) break;
            if (!wait_all(&sm->s_empty[sb], static_cast<uint32_t>((t >> 1) & 1) ^ 1u, sm)) break;
            ptx::tc_fence_after_sync();
            if (ptx::elect_one()) {
                const uint32_t sfk = tmem + kColSfK + 4 * sb;
                ptx::tmem_cp_sf(sfk, d_sf + (ptx::smem_u32(sm->sf_k[ks]) >> 4));
                const uint64_t dk0 = d_sw64 + (ptx::smem_u32(sm->k[ks]) >> 4);
                const uint32_t d_s = tmem + kColS + 128 * sb;
                ptx::mma_mxf4(d_s, dq0, dk0, ptx::mxf4_idesc(128, 0), sfq, sfk, 0u);
                ptx::mma_mxf4(d_s, dq0 + 2, dk0 + 2, ptx::mxf4_idesc(128, 2), sfq | (2u << 30), sfk | (2u << 30), 1u);
                ptx::mma_commit(&sm->s_full[sb]);
                ptx::mma_commit(&sm->k_empty[ks]);
            }
            __syncwarp();
            if (++ks == kStages) { ks = 0; kph ^= 1u; }
        }
    } else if (run && warp == 2) {
        // =============================== [dA | dl] = P~ [V | 1] issuer ===============================
        const uint64_t d_sw64 = ptx::smem_desc(0, 16, 512, ptx::kLayoutSw64);
        const uint64_t d_sf = ptx::smem_desc(0, 16, 128, ptx::kLayoutNone);
        if (ptx::elect_one()) {
            const uint64_t d1 = d_sf + (ptx::smem_u32(sm->sf_ones) >> 4);
            ptx::tmem_cp_sf(tmem + kColSfV + 4, d1);
            ptx::tmem_cp_sf(tmem + kColSfV + 12, d1);
        }
        __syncwarp();
        int vs = 0;
        uint32_t vph = 0;
        for (int j = 0; j < n_tiles; ++j) {
            const int pb = static_cast<int>(j & 1);
            if (!wait_all(&sm->v_full[vs], vph, sm)) break;
            if (!wait_all(&sm->p_full[pb], static_cast<uint32_t>((j >> 1) & 1), sm)) break;
            if (!wait_all(&sm->o_ready[j & 3], static_cast<uint32_t>((j >> 2) & 1), sm)) break;
            ptx::tc_fence_after_sync();
            if (ptx::elect_one()) {
                const uint32_t sfp = tmem + kColSfP + 4 * pb;
                const uint32_t sfv = tmem + kColSfV + 8 * pb;
                ptx::tmem_cp_sf(sfp, d_sf + (ptx::smem_u32(sm->sf_p[pb]) >> 4));
                ptx::tmem_cp_sf(sfv, d_sf + (ptx::smem_u32(sm->sf_v[vs]) >> 4));
                const uint64_t dp0 = d_sw64 + (ptx::smem_u32(sm->p[pb]) >> 4);
                const uint64_t dv0 = d_sw64 + (ptx::smem_u32(sm->v[vs]) >> 4);
                ptx::mma_mxf4(tmem + kColO, dp0, dv0, ptx::mxf4_idesc(144, 0), sfp, sfv, j > 0 ? 1u : 0u);
                ptx::mma_mxf4(tmem + kColO, dp0 + 2, dv0 + 2, ptx::mxf4_idesc(144, 2), sfp | (2u << 30), sfv | (2u << 30), 1u);
                ptx::mma_commit(&sm->p_empty[pb]);
                ptx::mma_commit(&sm->v_empty[vs]);
                if (j + 1 == n_tiles) ptx::mma_commit(&sm->o_done);
                sm->progress = static_cast<uint32_t>(j) + 1u;
            }
            __syncwarp();
            if (++vs == kStages) { vs = 0; vph ^= 1u; }
        }
    }
    } else if (warp >= 12) {
    // =============================== historical rescaling (Eq. alpha) ===============================
    // One warp per TMEM lane quarter.  When a row's maximum grew in tile j, its accumulator row and its
    // denominator are multiplied by alpha_j after P~V_{j-1} has landed and before P~V_j is released; this runs
    // beside the code generation of tile j instead of inside it.  A quarter without growth releases P~V_j at once, so it
    // may run behind P~V_{j-1} without a gap.  Bound: P~V waits for this step, and what takes its time is the latency of
    // the TMEM accesses and the issue slots that the probability warps leave.  So the load of the next 32 columns is on
    // its way while 32 are multiplied and stored (S = 16384, causal, 32 heads, when this form was taken: 1509 -> 1497 us; 64 columns
    // at a time 1885).  Registers of the three kinds of warp, measured on the persistent form, S = 16384 / S = 32760 not causal / 512 keys:
    // 56, 184, 88 (which spills) 1339 us / 7491 / 218; 48, 184, 96 1315 / 7340 / 214; 40, 184, 104 1306 / 7327 / 207; 32, 184, 112 1298 /
    // 7301 / 207; 24, 184, 120 1318 / 7401 / 209; 40, 176, 120 1327 / 7399 / 200; 40, 192, 88 1356 / 7506 / 223.
    asm volatile("setmaxnreg.dec.sync.aligned.u32 112;");
    const int quarter = warp & 3;
    const uint32_t row = quarter * 32 + lane;
    const uint32_t o_addr = tmem + (static_cast<uint32_t>(quarter * 32) << 16) + kColO;
    if (run) {
        for (int j = 0; j < n_tiles; ++j) {
            if (!wait_all(&sm->a_bar[j & 3][quarter], static_cast<uint32_t>((j >> 2) & 1), sm)) break;
            const float alpha = sm->alpha[j & 3][row];
            if (j > 0 && __any_sync(0xffffffffu, alpha != 1.0f)) {
                // The end of P~V_{j-1} frees its V stage.  The parity says so only if P~V_{j-5}, the stage's use before, has ended,
                // and it has: the probability warps waited for it before they stored the codes of tile j-3.
                if (!wait_all(&sm->v_empty[(j - 1) & 3], static_cast<uint32_t>((j - 1) >> 2) & 1u, sm)) break;
                ptx::tc_fence_after_sync();
                const uint64_t alpha2 = pack2(alpha, alpha);
                uint32_t oa[32], ob[32];
                // a store reads its registers asynchronously: not before wait::st may a load overwrite them
                ptx::tmem_ld32<0>(o_addr, oa);
                const uint32_t lcol = ptx::tmem_ld1(o_addr + 128);            // the denominator travels with the first columns
                ptx::tmem_wait_ld();
                ptx::tmem_ld32<0>(o_addr + 32, ob);
                scale32(oa, alpha2);
                ptx::tmem_st32<0>(o_addr, oa);
                ptx::tmem_st1(o_addr + 128, __float_as_uint(__uint_as_float(lcol) * alpha));
                ptx::tmem_wait_ld();
                scale32(ob, alpha2);
                ptx::tmem_wait_st();
                ptx::tmem_ld32<0>(o_addr + 64, oa);
                ptx::tmem_st32<0>(o_addr + 32, ob);
                ptx::tmem_wait_ld();
                scale32(oa, alpha2);
                ptx::tmem_wait_st();
                ptx::tmem_ld32<0>(o_addr + 96, ob);
                ptx::tmem_st32<0>(o_addr + 64, oa);
                ptx::tmem_wait_ld();
                scale32(ob, alpha2);
                ptx::tmem_st32<0>(o_addr + 96, ob);
                ptx::tmem_wait_st();
                ptx::tc_fence_before_sync();
            }
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&sm->o_ready[j & 3]);
        }
    }
    } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 184;");
    const int quarter = warp & 3;                       // TMEM lane quarter this warp may touch
    const int group = (warp - 4) >> 2;                  // group 0 takes the even KV tiles, group 1 the odd ones
    const uint32_t row = quarter * 32 + lane;           // row inside the query tile: one thread owns one row
    // this thread's query: token index inside the sequence, query head, and whether the row exists
    int64_t grow;
    int hq;
    bool row_valid;
    if (packed) {
        const int lq = static_cast<int>(Sq);
        const int gq = static_cast<int>(row) / lq;
        grow = static_cast<int>(row) - gq * lq;
        hq = head0 + gq;
        row_valid = gq < G;
    } else {
        grow = q0 + row;
        hq = head0;
        row_valid = grow < Sq;
    }
    const uint32_t lane_base = static_cast<uint32_t>(quarter * 32) << 16;
    if (run) {
        // =============================== probability generation ===============================
        const ProducerConsts K = P.K;
        int64_t limit = P.causal ? grow + shift : Sk - 1; // last visible key of this row
        if (limit > Sk - 1) limit = Sk - 1;
        const bool dbg_row = DEBUG && P.has_dbg && b == P.dbg.batch && hq == P.dbg.head && grow >= P.dbg.q_begin &&
                             grow < P.dbg.q_end && row_valid;
        const int64_t drow = grow - P.dbg.q_begin;
        const int64_t nblk_all = (Sk + 31) / 32;
        const int64_t ntile_all = (Sk + kTile - 1) / kTile;
        bool ok = true;
        bool in_flight = false;           // the scores of this tile were asked for at the end of the group's previous tile
        // FP32-denominator baseline (PRODUCER 6): this thread's sum of the row's FP32 exponentials over the group's
        // own tiles, relative to the scaled maximum m_ref of the latest of them
        float lsum = 0.0f, m_ref = -INFINITY;
        float r[128];
        const uint32_t s_addr = tmem + lane_base + kColS + 128 * group;

        for (int64_t j = group; j < n_tiles; j += 2) {
            const int sb = group;                                         // S, P and exchange buffers belong to the group
            const uint32_t ph2 = static_cast<uint32_t>((j >> 1) & 1);

            // ---- scores of tile j: TMEM -> registers (Algorithm 2, step 1 happened on the tensor core)
            if (!in_flight) {
                if (!wait_all(&sm->s_full[sb], ph2, sm)) { ok = false; break; }
                ptx::tc_fence_after_sync();
                ptx::tmem_ld32f<0>(s_addr, r);
                ptx::tmem_ld32f<32>(s_addr + 32, r);
                ptx::tmem_ld32f<64>(s_addr + 64, r);
                ptx::tmem_ld32f<96>(s_addr + 96, r);
            }
            float bmax[4];
            bool have_prev;
            float m_prev = -INFINITY;
            {
                // the other group's publication and the maximum it carries are asked for while the scores travel
                // (S = 131072: 78.2 ms, 79.3 with the maximum read after the scores)
                have_prev = j == 0 || ptx::mbar_try_wait(&sm->a_bar[(j - 1) & 3][quarter], static_cast<uint32_t>((j - 1) >> 2) & 1u);
                if (j > 0 && have_prev) m_prev = sm->runmax[sb ^ 1][row];
                ptx::tmem_wait_ld();
                ptx::tc_fence_before_sync();          // the S buffer is handed back with the joint publication below
                const int64_t last64 = limit - j * kTile;              // last visible key of the row inside the tile
                if (__any_sync(0xffffffffu, last64 < 127)) {           // diagonal or ragged tile: keys past the row's limit are masked in place
                    const int last = static_cast<int>(last64 < -1 ? -1 : last64 > 127 ? 127 : last64);
#pragma unroll
                    for (int g = 0; g < 4; ++g) {          // a bit per key: predicates come out of a word seven at a time
                        const int n = last - 32 * g + 1;   // keys of the block that the row sees
                        const uint32_t bits = n >= 32 ? 0xffffffffu : n <= 0 ? 0u : (1u << n) - 1u;
#pragma unroll
                        for (int i = 0; i < 32; ++i)
                            if ((bits & (1u << i)) == 0u) r[32 * g + i] = -INFINITY;
                    }
                }
            }
#pragma unroll
            for (int g = 0; g < 4; ++g) bmax[g] = block_max32(&r[32 * g]);

            // ---- running row maximum (Eq. rowmax-update): handed over from the group that owns tile j-1
            if (!have_prev) {
                if (!wait_all(&sm->a_bar[(j - 1) & 3][quarter], static_cast<uint32_t>((j - 1) >> 2) & 1u, sm)) { ok = false; break; }
                m_prev = sm->runmax[sb ^ 1][row];
            }
            float m_new = fmaxf(fmaxf(m_prev, bmax[0]), max3(bmax[1], bmax[2], bmax[3]));
            if (P.rescale_threshold > 0.0f && m_prev != -INFINITY) {      // optional policy: keep the old maximum
                const float ahead = __fsub_rn(__fmul_rn(K.sigma, m_new), __fmul_rn(K.sigma, m_prev));
                if (!(ahead > P.rescale_threshold)) m_new = m_prev;
            }
            const float m_s_prev = __fmul_rn(K.sigma, m_prev);
            const float m_s = __fmul_rn(K.sigma, m_new);
            const bool grew = m_new > m_prev && m_prev != -INFINITY;      // history exists and must be rescaled
            const float alpha = grew ? ex2_approx(__fmul_rn(__fsub_rn(m_s_prev, m_s), K.LOG2E)) : 1.0f;
            // One publication for both readers: the running maximum for the other group, alpha for the rescaling
            // warps.  alpha sits in a ring of four tiles: slot j mod 4 was last read for tile j-4, before P~V_{j-4}
            // was released, and this group waited for the end of P~V_{j-4} before it stored the codes of tile j-2.
            sm->runmax[sb][row] = m_new;
            sm->alpha[j & 3][row] = alpha;
            __syncwarp();
            if (lane == 0) {
                ptx::mbar_arrive(&sm->a_bar[j & 3][quarter]);
                ptx::mbar_arrive(&sm->s_empty[sb]);           // every lane's scores are in registers (wait::ld above)
            }
            // P~V of tile j-2 reads the group's P buffer: asked here, answered while block 0 is computed
            const bool have_p = ptx::mbar_try_wait(&sm->p_empty[sb], ph2 ^ 1u);

            if (PRODUCER == 6) {          // bring the sum to the new reference maximum (two tiles of alpha in one step)
                if (lsum != 0.0f) lsum *= ex2_approx(__fmul_rn(__fsub_rn(m_ref, m_s), K.LOG2E));
                m_ref = m_s;
            }
            // ---- probability operand (Algorithm 1 per block): codes and scales straight into the MMA operand
            uint32_t sfword = 0;
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                uint4 codes;
                uint32_t byte;
                produce32<PRODUCER>(&r[g * 32], bmax[g], m_s, K, codes, byte, &lsum);
                if (g == 0 && !have_p) {      // P~V of tile j-2 must have finished: it reads the group's P buffer
                    if (!wait_all(&sm->p_empty[sb], ph2 ^ 1u, sm)) { ok = false; break; }
                }
                *reinterpret_cast<uint4*>(sm->p[sb] + code_tile_offset(row, g)) = codes;
                sfword |= byte << (8 * g);
                if (DEBUG && dbg_row) {
                    const int64_t blk = j * 4 + g;
                    if (blk < nblk_all) {
                        if (P.dbg.codes) *reinterpret_cast<uint4*>(P.dbg.codes + (drow * nblk_all + blk) * 16) = codes;
                        if (P.dbg.scales) P.dbg.scales[drow * nblk_all + blk] = static_cast<uint8_t>(byte);
                    }
                }
            }
            if (!ok) break;               // the bounded wait inside the block loop gave up
            *reinterpret_cast<uint32_t*>(sm->sf_p[sb] + (row & 31u) * 16u + (row >> 5) * 4u) = sfword;
            if (DEBUG && dbg_row) {
                if (P.dbg.raw_scores) {
                    for (int i = 0; i < 128; ++i)
                        if (j * kTile + i < Sk) P.dbg.raw_scores[drow * Sk + j * kTile + i] = r[i];
                }
                if (P.dbg.row_max) P.dbg.row_max[drow * ntile_all + j] = m_s;
            }

            // The registers are free: if S of the group's next tile is there already (it is as a rule, S runs ahead),
            // its scores set out now and travel while the operand is handed over and the loop turns.
            in_flight = j + 2 < n_tiles && ptx::mbar_try_wait(&sm->s_full[sb], ph2 ^ 1u);
            if (in_flight) {
                ptx::tc_fence_after_sync();
                ptx::tmem_ld32f<0>(s_addr, r);
                ptx::tmem_ld32f<32>(s_addr + 32, r);
                ptx::tmem_ld32f<64>(s_addr + 64, r);
                ptx::tmem_ld32f<96>(s_addr + 96, r);
            }
            ptx::fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&sm->p_full[sb]);
        }
        ptx::tmem_wait_ld();              // nothing may be in flight when a bounded wait gave up inside the loop

        if (PRODUCER == 6) {              // both groups' partial denominators meet in shared memory
            sm->lsum_x[group][row] = lsum;
            sm->mref_x[group][row] = m_ref;
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&sm->l_bar);
        }
        // ---- final normalisation O = A / l: each group writes 64 of the 128 channels
        // (a barrier of its own: a group that skipped a phase of the other group's p_empty could not tell
        // an old completion from the last one by parity)
        if (ok) ok = wait_all(&sm->o_done, 0, sm);
        if (ok && PRODUCER == 6) ok = wait_all(&sm->l_bar, 0, sm);
        if (ok) {
            ptx::tc_fence_after_sync();
            uint32_t o[64];
            const uint32_t o_addr = tmem + lane_base + kColO + 64 * group;
            ptx::tmem_ld32<0>(o_addr, o);
            ptx::tmem_ld32<32>(o_addr + 32, o);
            const uint32_t lcol = ptx::tmem_ld1(tmem + lane_base + kColO + 128);
            ptx::tmem_wait_ld();
            float l = __uint_as_float(lcol);
            if (PRODUCER == 6) {
                // the accumulator refers to the maximum of the last tile, the larger of the two groups' references
                const float l0 = sm->lsum_x[0][row], l1 = sm->lsum_x[1][row];
                const float m0 = sm->mref_x[0][row], m1 = sm->mref_x[1][row];
                const float mf = fmaxf(m0, m1);
                l = (l0 != 0.0f ? l0 * ex2_approx(__fmul_rn(__fsub_rn(m0, mf), K.LOG2E)) : 0.0f) +
                    (l1 != 0.0f ? l1 * ex2_approx(__fmul_rn(__fsub_rn(m1, mf), K.LOG2E)) : 0.0f);
            }
            const float inv = l > 0.0f ? 1.0f / l : 0.0f;
            // Through shared memory, inside the warp: a lane holds 256 bytes of a row, and storing them from registers would
            // touch 32 rows per instruction (5000 cycles for the tile).  Read back, 16 lanes store 256 bytes of one row.
            uint8_t* const stage = sm->k[0] + 256 * group + (row - lane) * kOutRowBytes;
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                float4 v;
                v.x = __uint_as_float(o[4 * i + 0]) * inv;
                v.y = __uint_as_float(o[4 * i + 1]) * inv;
                v.z = __uint_as_float(o[4 * i + 2]) * inv;
                v.w = __uint_as_float(o[4 * i + 3]) * inv;
                *reinterpret_cast<float4*>(stage + lane * kOutRowBytes + 16 * i) = v;
            }
            __syncwarp();
            const uint64_t my_dst = row_valid ? reinterpret_cast<uint64_t>(P.o + (o_base + hq * P.o_head + grow * P.o_row + 64 * group)) : 0ull;
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const int r = 2 * i + (lane >> 4);
                const uint64_t dst = __shfl_sync(0xffffffffu, my_dst, r);
                const float4 v = *reinterpret_cast<const float4*>(stage + r * kOutRowBytes + 16 * (lane & 15));
                if (dst != 0ull) __stcs(reinterpret_cast<float4*>(dst) + (lane & 15), v);
            }
        }
    } else {
        // no visible key for the whole tile: rows are zero
        ptx::grid_wait();
        if (row_valid) {
            float4* dst = reinterpret_cast<float4*>(P.o + (o_base + hq * P.o_head + grow * P.o_row + 64 * group));
            for (int i = 0; i < 16; ++i) dst[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
    }
    }

    ptx::tc_fence_before_sync();
    __syncthreads();
    if (warp == 1) {
        if (sm->abort_flag) __nanosleep(1000000u);  // loads may be in flight: a millisecond, before shared memory is another CTA's
        ptx::tmem_dealloc(tmem, kTmemCols);
    }
}

#include "attention_short.cuh"

// ------------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------------

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

constexpr int kMaxDevices = 64;   // device ordinals the per-device tables of this file cover

EncodeTiledFn get_encode()
{
    static std::once_flag once;
    static EncodeTiledFn fn = nullptr;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    });
    return fn;
}

// A descriptor depends on nothing but the base, the shape and the kind of map, so the last few are kept: a serving loop
// that calls with the same buffers and shape (decode steps above all) does not pay for driver calls per forward.
// kMapRowsOut: FP32 rows of 128 channels, [heads, tokens] or, kMapRowsOutPacked, [tokens, heads]; coordinates (channel, token, head).
enum MapKind : uint32_t { kMapCodes, kMapBf16, kMapRowsOut, kMapRowsOutPacked };
struct MapCacheEntry {
    const void* base;
    uint64_t row_bytes, rows;      // of the outputs: heads, tokens
    MapKind kind;
    CUtensorMap map;
};
constexpr int kMapCacheSize = 32;
std::mutex g_map_mutex;
MapCacheEntry g_map_cache[kMapCacheSize] = {};
int g_map_next = 0;

bool encode_any(CUtensorMap* map, const void* base, uint64_t row_bytes, uint64_t rows, MapKind kind)
{
    {
        std::lock_guard<std::mutex> lock(g_map_mutex);
        for (int i = 0; i < kMapCacheSize; ++i) {
            const MapCacheEntry& e = g_map_cache[i];
            if (e.base == base && e.row_bytes == row_bytes && e.rows == rows && e.kind == kind) {
                *map = e.map;
                return true;
            }
        }
    }
    EncodeTiledFn enc = get_encode();
    if (!enc) return false;
    const cuuint32_t estr[3] = {1, 1, 1};
    CUresult r;
    if (kind == kMapCodes || kind == kMapBf16) {
        const bool codes = kind == kMapCodes;
        const cuuint64_t dims[2] = {codes ? row_bytes : row_bytes / 2, rows}, strides[1] = {row_bytes};
        const cuuint32_t box[2] = {64, 128};
        r = enc(map, codes ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box,
                estr, CU_TENSOR_MAP_INTERLEAVE_NONE, codes ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B,
                CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    } else {
        const uint64_t heads = row_bytes;
        const cuuint64_t dims[3] = {128, rows, heads};
        const cuuint64_t strides[2] = {kind == kMapRowsOut ? 512 : 512 * heads, kind == kMapRowsOut ? 512 * rows : 512};
        const cuuint32_t box[3] = {32, 32, 1};
        r = enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    }
    if (r != CUDA_SUCCESS) return false;
    std::lock_guard<std::mutex> lock(g_map_mutex);
    g_map_cache[g_map_next] = MapCacheEntry{base, row_bytes, rows, kind, *map};
    g_map_next = (g_map_next + 1) % kMapCacheSize;
    return true;
}
// [rows, row_bytes] matrix of packed codes, box 64 B x 128 rows, 64-byte swizzle
bool encode_map(CUtensorMap* map, const void* base, uint64_t row_bytes, uint64_t rows) { return encode_any(map, base, row_bytes, rows, kMapCodes); }

struct Workspace {
    size_t status, qc, qsf, kc, ksf, vt, vsf, total;
    int64_t Sq_pad, Sk_pad;
};

size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

bool use_few(int Hq, int Hkv, int64_t Sq, int64_t Sk);

Workspace plan_workspace(int B, int Hq, int Hkv, int64_t Sq, int64_t Sk)
{
    Workspace w;
    w.Sq_pad = (Sq + kTile - 1) / kTile * kTile;
    w.Sk_pad = (Sk + kTile - 1) / kTile * kTile;
    size_t off = 0;
    w.status = off; off += 1024;
    w.qc = off;  off = align_up(off + static_cast<size_t>(B) * Hq * w.Sq_pad * 64, 1024);
    w.qsf = off; off = align_up(off + static_cast<size_t>(B) * Hq * (w.Sq_pad / kTile) * kSfBytes, 1024);
    w.kc = off;  off = align_up(off + static_cast<size_t>(B) * Hkv * w.Sk_pad * 64, 1024);
    w.ksf = off; off = align_up(off + static_cast<size_t>(B) * Hkv * (w.Sk_pad / kTile) * kSfBytes, 1024);
    w.vt = off;  off = align_up(off + static_cast<size_t>(B) * Hkv * 128 * (w.Sk_pad / 2), 1024);
    w.vsf = off; off = align_up(off + static_cast<size_t>(B) * Hkv * (w.Sk_pad / kTile) * kSfBytes, 1024);
    w.total = off;
    return w;
}

// what a call needs: the few-row path has a layout of its own in the same workspace
size_t workspace_bytes_for(int B, int Hq, int Hkv, int64_t Sq, int64_t Sk)
{
    size_t total = plan_workspace(B, Hq, Hkv, Sq, Sk).total;
    if (use_few(Hq, Hkv, Sq, Sk)) {
        const int64_t heads = static_cast<int64_t>(B) * Hkv;
        const size_t few = 1024 + plan_few(heads * ((Sk + kTile - 1) / kTile * kTile), static_cast<int>(Hq / Hkv * Sq)).total;
        if (few > total) total = few;
    }
    return total;
}

bool shape_ok(int B, int Hq, int Hkv, int64_t Sq, int64_t Sk, int d)
{
    return B > 0 && Hq > 0 && Hkv > 0 && Sq > 0 && Sk > 0 && d == 128 && Hq % Hkv == 0 &&
           static_cast<int64_t>(B) * Hq * ((Sq + kTile - 1) / kTile * kTile) < (1ll << 31) &&
           static_cast<int64_t>(B) * Hkv * ((Sk + kTile - 1) / kTile * kTile) < (1ll << 31);
}

template <int PRODUCER, bool DEBUG>
cudaError_t launch_one(dim3 grid, size_t smem, cudaStream_t stream, const CUtensorMap& mq, const CUtensorMap& mk,
                       const CUtensorMap& mv, const FwdParams& P)
{
    // the shared-memory attribute belongs to (function, device): set once for each
    static std::mutex mu;
    static bool done[kMaxDevices] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    {
        std::lock_guard<std::mutex> lock(mu);
        if (!done[dev]) {
            cudaError_t e = cudaFuncSetAttribute(attention_fwd_kernel<PRODUCER, DEBUG>,
                                                 cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
            if (e != cudaSuccess) return e;
            done[dev] = true;
        }
    }
    return launch_overlapped(attention_fwd_kernel<PRODUCER, DEBUG>, grid, kThreads, smem, stream, mq, mk, mv, P);
}

// More query tiles than SMs: persistent CTAs, at every length of the KV walk (the measurements are in attention_short.cuh); with
// fewer, a CTA has one item and nothing to overlap it with, and the form made for one starts sooner (causal: one head, 1024 tokens
// 12.1 us against 12.4, 4096 28.7 / 29.0, 16384 94.3 / 93.6; 36 heads, 512 tokens 10.2 / 10.5).  The table form of the rule loses in long
// walks: 24 heads, 8000 queries, not causal, 4096 keys 495 us with one CTA per tile, 471 persistent, 8192 keys 914 / 911, 12288 keys
// 1329 / 1349; its line is at a mean walk of 48 tiles.  A packed batch is judged by its longest sequence.
// Little more tiles than SMs and the heaviest of them outlasting the rest: both forms end with that tile, and the line is not drawn for
// it.  One CTA per tile / persistent, causal, affine rule 8 heads of 2600 tokens 22.3 / 21.8 us, 8 of 2432 20.9 / 20.8, 16 of 1400 17.0 /
// 15.4, 40 of 512 14.8 / 11.0; plain exponentials 16 of 1400 20.8 / 21.1, 8 of 2600 32.5 / 32.1, 40 of 512 16.3 / 12.5; table 16 of 1280
// 19.5 / 20.0, 8 of 2600 33.1 / 33.5, 40 of 512 16.4 / 12.6.  A packed batch whose heaviest tile takes 1.2 times the mean of a CTA is slower
// by 1 to 5 % persistent (one head, causal, one sequence of 3000 tokens and 30 of up to 1500: 34.9 / 36.5).
// P.Sk: the keys of the problem or, with P.Sq = 0, of the longest sequence.
bool use_short(int producer, bool debug, int64_t items, int sms, const FwdParams& P)
{
    if (debug || producer == 6 || P.packed || items <= sms) return false;
    const int64_t mean = P.causal ? P.Sk - std::min(P.Sq, P.Sk) / 2 : P.Sk;
    return producer != 3 || mean <= 48 * kTile;
}

template <int PRODUCER, bool TABLE>
cudaError_t launch_short_one(unsigned items, unsigned sms, int dev, cudaStream_t stream, const CUtensorMap& mq, const CUtensorMap& mk, const CUtensorMap& mv,
                         const CUtensorMap& mo, const FwdParams& P)
{
    constexpr int smem = static_cast<int>(sizeof(ShortSmem)) + 1024;
    static std::atomic<uint64_t> done{0};        // the shared-memory attribute belongs to (function, device): set once for each
    if ((done.load(std::memory_order_relaxed) >> dev & 1u) == 0u) {
        const cudaError_t e = cudaFuncSetAttribute(attention_short_kernel<PRODUCER, TABLE>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        done.fetch_or(1ull << dev, std::memory_order_relaxed);
    }
    return launch_overlapped(attention_short_kernel<PRODUCER, TABLE>, dim3(sms), kThreads, smem, stream, mq, mk, mv, mo, P, items);
}

template <int PRODUCER>
cudaError_t launch_short(unsigned items, unsigned sms, int dev, cudaStream_t stream, const CUtensorMap& mq, const CUtensorMap& mk,
                         const CUtensorMap& mv, const CUtensorMap& mo, const FwdParams& P)
{
    return P.items ? launch_short_one<PRODUCER, true>(items, sms, dev, stream, mq, mk, mv, mo, P) : launch_short_one<PRODUCER, false>(items, sms, dev, stream, mq, mk, mv, mo, P);
}

template <int PRODUCER>
cudaError_t launch_main(bool debug, dim3 grid, size_t smem, cudaStream_t stream, const CUtensorMap& mq, const CUtensorMap& mk,
                        const CUtensorMap& mv, const FwdParams& P)
{
    return debug ? launch_one<PRODUCER, true>(grid, smem, stream, mq, mk, mv, P) : launch_one<PRODUCER, false>(grid, smem, stream, mq, mk, mv, P);
}

// The query heads of a KV group share one 128-row query tile when they fit: a decode step (one query token) of a
// model with 4 query heads per KV head then fills 4 rows of one tile instead of 1 row of each of 4 tiles, and each
// K/V tile is loaded once per KV head.  Rows are independent of one another on the whole path, so the result is
// the unpacked one bit for bit.
bool use_packed_tile(int Hq, int Hkv, int64_t Sq) { return Hq / Hkv > 1 && static_cast<int64_t>(Hq / Hkv) * Sq <= kTile; }

// Few query rows per KV group: K and V are read once whatever the kernel does, so the path that quantises them on the way to
// the tensor core takes over (attention_few.cu; the line and its measurements: few_takes).  Depends on the sequence's own shape
// alone, so that a sequence takes the same path by itself and in a packed batch.
bool use_few(int Hq, int Hkv, int64_t Sq, int64_t Sk) { return few_takes(static_cast<int64_t>(Hq / Hkv) * Sq, (Sk + kTile - 1) / kTile); }

int64_t few_chunks(int64_t Sk, int64_t rows)
{
    const int n_tiles = static_cast<int>((Sk + kTile - 1) / kTile), per = few_chunk_tiles(n_tiles, static_cast<int>(rows));
    return (n_tiles + per - 1) / per;
}

cudaError_t launch_forward(int producer, bool debug, int64_t items, cudaStream_t stream, const CUtensorMap& mq,
                           const CUtensorMap& mk, const CUtensorMap& mv, const FwdParams& P)
{
    if (items <= 0 || items > 0x7fffffffll) return cudaErrorInvalidValue;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    const int sms = sm_count(dev);
    if (sms > 0 && use_short(producer, debug, items, sms, P)) {
        CUtensorMap mo;
        const bool packed_batch = P.items != nullptr;
        if (!encode_any(&mo, P.o, packed_batch ? P.Hq : static_cast<uint64_t>(P.B) * P.Hq, packed_batch ? P.o_tokens : P.Sq,
                        packed_batch ? kMapRowsOutPacked : kMapRowsOut))
            return cudaErrorInvalidValue;
        switch (producer) {
            case 0: return launch_short<0>(static_cast<unsigned>(items), static_cast<unsigned>(sms), dev, stream, mq, mk, mv, mo, P);
            case 1: return launch_short<1>(static_cast<unsigned>(items), static_cast<unsigned>(sms), dev, stream, mq, mk, mv, mo, P);
            case 2: return launch_short<2>(static_cast<unsigned>(items), static_cast<unsigned>(sms), dev, stream, mq, mk, mv, mo, P);
            case 3: return launch_short<3>(static_cast<unsigned>(items), static_cast<unsigned>(sms), dev, stream, mq, mk, mv, mo, P);
            case 4: return launch_short<4>(static_cast<unsigned>(items), static_cast<unsigned>(sms), dev, stream, mq, mk, mv, mo, P);
            case 5: return launch_short<5>(static_cast<unsigned>(items), static_cast<unsigned>(sms), dev, stream, mq, mk, mv, mo, P);
            default: return cudaErrorInvalidValue;
        }
    }
    dim3 grid(static_cast<unsigned>(items));
    // more than half of the SM's shared memory: one CTA per SM, since each CTA takes all 512 TMEM columns
    const size_t smem = sizeof(Smem) + 1024 > 120 * 1024 ? sizeof(Smem) + 1024 : 120 * 1024;
    switch (producer) {
        case 0: return launch_main<0>(debug, grid, smem, stream, mq, mk, mv, P);
        case 1: return launch_main<1>(debug, grid, smem, stream, mq, mk, mv, P);
        case 2: return launch_main<2>(debug, grid, smem, stream, mq, mk, mv, P);
        case 3: return launch_main<3>(debug, grid, smem, stream, mq, mk, mv, P);
        case 4: return launch_main<4>(debug, grid, smem, stream, mq, mk, mv, P);
        case 5: return launch_main<5>(debug, grid, smem, stream, mq, mk, mv, P);
        case 6: return launch_main<6>(debug, grid, smem, stream, mq, mk, mv, P);
        default: return cudaErrorInvalidValue;
    }
}

efq_status_t check_device()
{
    int dev = 0, major = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return EFQ_ERR_CUDA;
    if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess) return EFQ_ERR_CUDA;
    return major == 10 ? EFQ_OK : EFQ_ERR_ARCH;
}

efq_status_t attention_impl(const void* q, const void* k, const void* v, float* o, int B, int Hq, int Hkv, int64_t Sq,
                            int64_t Sk, int d, int causal, float softmax_scale, int producer, float tau, float h,
                            void* workspace, size_t workspace_bytes, const efq_debug_t* debug, cudaStream_t stream,
                            bool do_quantize, bool do_forward, bool inject = false, float rescale_threshold = 0.0f)
{
    // q [B, Hq, Sq, d], k, v [B, Hkv, Sk, d], o [B, Hq, Sq, d]
    if (!q || !k || !v || !o) return EFQ_ERR_INVALID_ARG;
    if (B <= 0 || Hq <= 0 || Hkv <= 0 || Sq <= 0 || Sk <= 0 || Hq % Hkv != 0) return EFQ_ERR_INVALID_ARG;
    if (d != 128) return EFQ_ERR_UNSUPPORTED;
    if (!shape_ok(B, Hq, Hkv, Sq, Sk, d)) return EFQ_ERR_UNSUPPORTED;
    if (producer < 0 || producer > 6) return EFQ_ERR_INVALID_ARG;
    if (!(softmax_scale > 0.0f)) softmax_scale = static_cast<float>(1.0 / sqrt(static_cast<double>(d)));
    if (!isfinite(softmax_scale) || !isfinite(tau) || !isfinite(h) || !(h > 0.0f)) return EFQ_ERR_INVALID_ARG;
    auto mis = [](const void* p, uintptr_t a) { return (reinterpret_cast<uintptr_t>(p) & (a - 1)) != 0; };
    if (mis(q, 16) || mis(k, 16) || mis(v, 16) || mis(o, 16)) return EFQ_ERR_ALIGNMENT;
    const Workspace w = plan_workspace(B, Hq, Hkv, Sq, Sk);
    if (!workspace || workspace_bytes < workspace_bytes_for(B, Hq, Hkv, Sq, Sk)) return EFQ_ERR_WORKSPACE;
    if (mis(workspace, 256)) return EFQ_ERR_ALIGNMENT;
    const efq_status_t dev_st = check_device();
    if (dev_st != EFQ_OK) return dev_st;

    uint8_t* ws = static_cast<uint8_t*>(workspace);
    const int G = Hq / Hkv;
    if (do_quantize && do_forward && use_few(Hq, Hkv, Sq, Sk)) {
        FewParams F{};
        F.q = static_cast<const __nv_bfloat16*>(q); F.k = static_cast<const __nv_bfloat16*>(k); F.v = static_cast<const __nv_bfloat16*>(v);
        F.o = o;
        F.Hkv = Hkv; F.G = G; F.causal = causal ? 1 : 0;
        F.Sq = static_cast<int32_t>(Sq); F.Sk = static_cast<int32_t>(Sk); F.Sk_pad = static_cast<int32_t>(w.Sk_pad);
        F.dense_chunks = static_cast<int32_t>(few_chunks(Sk, G * Sq));
        F.q_row = 128; F.q_head = Sq * 128; F.q_seq = Hq * F.q_head;
        F.k_row = 128; F.k_head = Sk * 128; F.k_seq = Hkv * F.k_head;
        F.row_cap = static_cast<int32_t>(G * Sq);
        F.n_heads = B * Hkv;
        F.rescale_threshold = rescale_threshold;
        F.K = producer == 3 ? make_producer_consts_lut(softmax_scale) : make_producer_consts(softmax_scale, tau, h);
        const int64_t units = static_cast<int64_t>(B) * Hkv * F.dense_chunks;
        if (units > 0x7fffffffll) return EFQ_ERR_UNSUPPORTED;
        F.n_units = static_cast<int32_t>(units);
        F.longest_chunk = few_longest_chunk(static_cast<int>(w.Sk_pad / kTile), G * static_cast<int>(Sq));
        const FewPlan fp = plan_few(static_cast<int64_t>(B) * Hkv * w.Sk_pad, F.row_cap);
        F.scores = reinterpret_cast<float*>(ws + 1024 + fp.scores); F.block_max = reinterpret_cast<float*>(ws + 1024 + fp.block_max);
        F.stats = reinterpret_cast<float*>(ws + 1024 + fp.stats);
        F.status = reinterpret_cast<uint32_t*>(ws);
        F.inject_skip_mma = inject ? 1 : 0;
        F.has_dbg = debug != nullptr ? 1 : 0;
        if (debug != nullptr) F.dbg = *debug;
        return launch_few(producer, F, stream) == cudaSuccess ? EFQ_OK : EFQ_ERR_CUDA;
    }
    const bool packed = use_packed_tile(Hq, Hkv, Sq);
    const int64_t q_rows = packed ? static_cast<int64_t>(B) * Hkv * kTile : static_cast<int64_t>(B) * Hq * w.Sq_pad;
    if (do_quantize) {
        QuantSeg sq{}, sk{}, sv{};
        sq.src = static_cast<const __nv_bfloat16*>(q);
        sq.heads = packed ? static_cast<int64_t>(B) * Hkv : static_cast<int64_t>(B) * Hq;
        sq.S = packed ? G * Sq : Sq;
        sq.S_pad = packed ? kTile : w.Sq_pad;
        sq.head_stride = Sq * 128; sq.row_stride = 128;
        sq.pack_lq = packed ? static_cast<int32_t>(Sq) : 0; sq.pack_G = packed ? G : 1;
        sq.codes = ws + w.qc; sq.sf = ws + w.qsf;
        sk.src = static_cast<const __nv_bfloat16*>(k);
        sk.heads = static_cast<int64_t>(B) * Hkv; sk.S = Sk; sk.S_pad = w.Sk_pad;
        sk.head_stride = Sk * 128; sk.row_stride = 128; sk.pack_G = 1;
        sk.codes = ws + w.kc; sk.sf = ws + w.ksf;
        sv = sk;
        sv.src = static_cast<const __nv_bfloat16*>(v);
        sv.codes = ws + w.vt; sv.sf = ws + w.vsf;
        sv.v_row_bytes = w.Sk_pad / 2; sv.v_x0 = 0; sv.v_sf_tiles_per_head = w.Sk_pad / kTile; sv.v_sf_tile0 = 0;
        // one launch for the three operands; it also clears the status words the forward starts from
        if (launch_quantize_qkv(sq, sk, sv, reinterpret_cast<uint32_t*>(ws + w.status), stream) != cudaSuccess) return EFQ_ERR_CUDA;
    }
    if (!do_forward) return EFQ_OK;

    CUtensorMap mq, mk, mv;
    if (!encode_map(&mq, ws + w.qc, 64, static_cast<uint64_t>(q_rows))) return EFQ_ERR_CUDA;
    if (!encode_map(&mk, ws + w.kc, 64, static_cast<uint64_t>(B) * Hkv * w.Sk_pad)) return EFQ_ERR_CUDA;
    if (!encode_map(&mv, ws + w.vt, static_cast<uint64_t>(w.Sk_pad / 2), static_cast<uint64_t>(B) * Hkv * 128)) return EFQ_ERR_CUDA;

    FwdParams P{};
    P.B = B; P.Hq = Hq; P.Hkv = Hkv; P.Sq = Sq; P.Sk = Sk; P.Sq_pad = w.Sq_pad; P.Sk_pad = w.Sk_pad;
    P.causal = causal ? 1 : 0;
    P.K = producer == 3 ? make_producer_consts_lut(softmax_scale) : make_producer_consts(softmax_scale, tau, h);
    P.sf_q = ws + w.qsf; P.sf_k = ws + w.ksf; P.sf_v = ws + w.vsf;
    P.o = o;
    P.o_head = Sq * 128;
    P.o_row = 128;
    P.status = reinterpret_cast<uint32_t*>(ws + w.status);
    P.packed = packed ? 1 : 0;
    P.seqs = nullptr; P.items = nullptr; P.v_tiles_per_head = 0;
    P.inject_skip_loads = inject ? 1 : 0;
    P.rescale_threshold = rescale_threshold;
    P.has_dbg = debug ? 1 : 0;
    if (debug) P.dbg = *debug; else P.dbg = efq_debug_t{};

    const uint64_t heads = static_cast<uint64_t>(B) * Hq;
    P.heads_magic = heads > 1 ? static_cast<uint32_t>(((1ull << 32) + heads - 1) / heads) : 0u;
    const int64_t items = packed ? static_cast<int64_t>(B) * Hkv : (w.Sq_pad / kTile) * B * Hq;
    return launch_forward(producer, debug != nullptr, items, stream, mq, mk, mv, P) == cudaSuccess ? EFQ_OK : EFQ_ERR_CUDA;
}

// ------------------------------------------------------------------------------------------------
// Packed variable-length batch: every sequence quantised by itself.  Two launches for all sequences of the general path,
// three for all that have few query rows (attention_few.cu).
// ------------------------------------------------------------------------------------------------
// Workspace: status words | tables from the host (sequences, quantiser jobs, their CTA prefix sums, query tiles in the order
// of their weight, the places of their items if they are not one after the other) | item table (written on the device: it has an
// entry per head) |
// Q codes [rows of all sequences, 64 B] | Q scale tiles | K codes | K scale tiles |
// V^T codes [Hkv * 128, sum of Sk_pad / 2 B] (the sequences side by side along the keys) | V scale tiles.
struct VarlenPlan {
    int n_active;                    // sequences with query and key tokens that take the general path
    int n_few, few_rows;             // ... and the few-row path (attention_few.cu); the most query rows of one of them
    int64_t few_units, few_keys;     // their chunks times KV heads; their keys, padded to 128
    int64_t q_rows, k_rows, k_cols;  // rows of the Q and K code matrices, keys along V^T (all padded to 128)
    int64_t items, groups, quant_ctas;
    int64_t longest;                 // keys of the longest sequence of the general path
    size_t tables, seqs_off, jobs_off, prefix_off, groups_off, places_off, items_off, qc, qsf, kc, ksf, vt, vsf, few_table, few, total;
};

// checks the two prefix arrays and lays the workspace out; false with st set on bad input
bool plan_varlen(const int64_t* cu_q, const int64_t* cu_k, int n_seqs, int Hq, int Hkv, int d, VarlenPlan& p, efq_status_t& st)
{
    st = EFQ_OK;
    if (!cu_q || !cu_k || n_seqs < 0 || Hq <= 0 || Hkv <= 0 || Hq % Hkv != 0) { st = EFQ_ERR_INVALID_ARG; return false; }
    if (d != 128) { st = EFQ_ERR_UNSUPPORTED; return false; }
    if (n_seqs > 0 && (cu_q[0] != 0 || cu_k[0] != 0)) { st = EFQ_ERR_INVALID_ARG; return false; }
    p = VarlenPlan{};
    size_t copies = 0;      // MXFP4 copies of the few-row sequences: not made, but the size a caller plans with still covers them
    for (int s = 0; s < n_seqs; ++s) {
        const int64_t lq = cu_q[s + 1] - cu_q[s], lk = cu_k[s + 1] - cu_k[s];
        if (lq < 0 || lk < 0) { st = EFQ_ERR_INVALID_ARG; return false; }
        if (lq == 0 || lk == 0) continue;
        if (use_few(Hq, Hkv, lq, lk)) {
            ++p.n_few;
            p.few_rows = std::max(p.few_rows, static_cast<int>(Hq / Hkv * lq));
            p.few_units += few_chunks(lk, Hq / Hkv * lq) * Hkv;
            p.few_keys += (lk + kTile - 1) / kTile * kTile;
            copies += static_cast<size_t>(Hkv) * (kTile + 2 * ((lk + kTile - 1) / kTile * kTile)) * (64 + 4);
            continue;
        }
        const bool packed = use_packed_tile(Hq, Hkv, lq);
        const int64_t lq_pad = packed ? kTile : (lq + kTile - 1) / kTile * kTile, lk_pad = (lk + kTile - 1) / kTile * kTile;
        ++p.n_active;
        p.q_rows += (packed ? Hkv : Hq) * lq_pad;
        p.k_rows += Hkv * lk_pad;
        p.k_cols += lk_pad;
        p.longest = std::max(p.longest, lk);
        p.items += packed ? Hkv : (lq_pad / kTile) * Hq;
        p.groups += lq_pad / kTile;
        p.quant_ctas += (packed ? Hkv : Hq) * (lq_pad / kTile) + 2 * Hkv * (lk_pad / kTile);
    }
    // 32-bit tile coordinates and grid sizes
    if (p.q_rows >= (1ll << 31) || p.k_rows >= (1ll << 31) || p.k_cols >= (1ll << 31) || p.items >= (1ll << 31) ||
        p.quant_ctas >= (1ll << 31) || p.few_units >= (1ll << 31) || p.few_keys >= (1ll << 31)) { st = EFQ_ERR_UNSUPPORTED; return false; }
    size_t off = 1024;
    p.seqs_off = off;   off = align_up(off + sizeof(SeqDesc) * p.n_active, 256);
    p.jobs_off = off;   off = align_up(off + sizeof(QuantJob) * 3 * p.n_active, 256);
    p.prefix_off = off; off = align_up(off + sizeof(int32_t) * (3 * p.n_active + 1), 256);
    p.groups_off = off; off = align_up(off + sizeof(ItemGroup) * static_cast<size_t>(p.groups), 256);
    p.places_off = off; off = align_up(off + sizeof(int32_t) * static_cast<size_t>(order_places(std::min(p.items, kOrderMaxItems))), 1024);
    p.tables = off - 1024;
    p.items_off = off;  off = align_up(off + sizeof(ItemDesc) * static_cast<size_t>(order_places(p.items)), 1024);
    p.qc = off;  off = align_up(off + static_cast<size_t>(p.q_rows) * 64, 1024);
    p.qsf = off; off = align_up(off + static_cast<size_t>(p.q_rows / kTile) * kSfBytes, 1024);
    p.kc = off;  off = align_up(off + static_cast<size_t>(p.k_rows) * 64, 1024);
    p.ksf = off; off = align_up(off + static_cast<size_t>(p.k_rows / kTile) * kSfBytes, 1024);
    p.vt = off;  off = align_up(off + static_cast<size_t>(Hkv) * 128 * (p.k_cols / 2), 1024);
    p.vsf = off; off = align_up(off + static_cast<size_t>(Hkv) * (p.k_cols / kTile) * kSfBytes, 1024);
    p.few_table = off;
    if (p.n_few > kFewInlineSeqs) off = align_up(off + sizeof(FewSeq) * p.n_few, 1024);
    p.few = off;
    if (p.n_few > 0) off += std::max(plan_few(p.few_keys * Hkv, p.few_rows).total, align_up(copies, 1024));
    p.total = off;
    return true;
}

// Host table to the workspace.  Pageable memory: the call returns once the bytes sit in the driver's staging area, so the vector
// may go - but a copy recorded into a graph reads them at every replay, so there the graph takes the vector over and frees it when it
// and all that was instantiated from it are destroyed.
template <typename T>
cudaError_t copy_table(void* dst, std::vector<T>& host, cudaStream_t stream)
{
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    cudaGraph_t graph = nullptr;
    cudaError_t e = cudaStreamGetCaptureInfo(stream, &capture, nullptr, &graph, nullptr, nullptr);
    if (e != cudaSuccess) return e;
    e = cudaMemcpyAsync(dst, host.data(), sizeof(T) * host.size(), cudaMemcpyHostToDevice, stream);
    if (e != cudaSuccess || capture != cudaStreamCaptureStatusActive) return e;
    auto* const kept = new std::vector<T>(std::move(host));          // the bytes stay where they are
    cudaUserObject_t owner;
    e = cudaUserObjectCreate(&owner, kept, [](void* p) { delete static_cast<std::vector<T>*>(p); }, 1, cudaUserObjectNoDestructorSync);
    if (e != cudaSuccess) { host = std::move(*kept); delete kept; return e; }
    return cudaGraphRetainUserObject(graph, owner, 1, cudaGraphUserObjectMove);
}

}  // namespace

int sm_count(int dev)
{
    static std::atomic<int> known[kMaxDevices] = {};
    int n = dev >= 0 && dev < kMaxDevices ? known[dev].load(std::memory_order_relaxed) : 0;
    if (n == 0 && cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && dev < kMaxDevices) known[dev].store(n, std::memory_order_relaxed);
    return n;
}

bool encode_bf16_map(CUtensorMap* map, const void* base, uint64_t cols, uint64_t rows) { return encode_any(map, base, 2 * cols, rows, kMapBf16); }

}  // namespace efq

extern "C" size_t efq_attention_workspace_bytes(int B, int Hq, int Hkv, int64_t Sq, int64_t Sk, int d)
{
    if (!efq::shape_ok(B, Hq, Hkv, Sq, Sk, d)) return 0;
    return efq::workspace_bytes_for(B, Hq, Hkv, Sq, Sk);
}

// Producer ids inside the library: 0 = EFQ (affine rule), 1 / 2 = exp-then-quantize scale4 / scale6, 3 = EFQ-LUT,
// 4 = exp-then-quantize scale4 with the scale folded into the exponential, 5 = the same with 2 of 8 exponentials by polynomial,
// 6 = exp-then-quantize scale4 whose denominator is the sum of the FP32 exponentials (the ones columns are ignored).
static bool read_params(const efq_params_t* params, float& tau, float& h, bool& lut, float& threshold, efq_status_t& st)
{
    tau = -3.06f;
    h = 2.30f;
    lut = false;
    threshold = 0.0f;
    st = EFQ_OK;
    if (params) {
        if (params->variant != 0 && params->variant != 1) { st = EFQ_ERR_UNSUPPORTED; return false; }
        if (params->kv_tile != 0 && params->kv_tile != 128) { st = EFQ_ERR_UNSUPPORTED; return false; }
        if (!(params->rescale_threshold >= 0.0f)) { st = EFQ_ERR_INVALID_ARG; return false; }   // negative or NaN
        threshold = params->rescale_threshold;
        lut = params->variant == 1;
        if (!lut) {                 // the LUT variant has its own fixed (tau16, h16): tau and h are not read
            tau = params->tau;
            h = params->h;
        }
    }
    return true;
}

extern "C" efq_status_t efq_attention_fwd(const void* q, const void* k, const void* v, float* o, int B, int Hq, int Hkv,
                                          int64_t Sq, int64_t Sk, int d, int causal, float softmax_scale,
                                          const efq_params_t* params, void* workspace, size_t workspace_bytes,
                                          const efq_debug_t* debug, void* stream)
{
    float tau, h, threshold;
    bool lut;
    efq_status_t st;
    if (!read_params(params, tau, h, lut, threshold, st)) return st;
    return efq::attention_impl(q, k, v, o, B, Hq, Hkv, Sq, Sk, d, causal, softmax_scale, lut ? 3 : 0, tau, h, workspace,
                               workspace_bytes, debug, static_cast<cudaStream_t>(stream), true, true, false, threshold);
}

extern "C" efq_status_t exp_then_quantize_attention_fwd(const void* q, const void* k, const void* v, float* o, int B,
                                                        int Hq, int Hkv, int64_t Sq, int64_t Sk, int d, int causal,
                                                        float softmax_scale, int scale_mode, void* workspace,
                                                        size_t workspace_bytes, const efq_debug_t* debug, void* stream)
{
    if (scale_mode < 0 || scale_mode > 4) return EFQ_ERR_INVALID_ARG;
    return efq::attention_impl(q, k, v, o, B, Hq, Hkv, Sq, Sk, d, causal, softmax_scale, scale_mode >= 2 ? scale_mode + 2 : 1 + scale_mode, 0.0f, 1.0f,
                               workspace, workspace_bytes, debug, static_cast<cudaStream_t>(stream), true, true);
}

extern "C" efq_status_t efq_attention_fwd_inject_timeout(const void* q, const void* k, const void* v, float* o, int B,
                                                         int Hq, int Hkv, int64_t Sq, int64_t Sk, int d, void* workspace,
                                                         size_t workspace_bytes, void* stream)
{
    return efq::attention_impl(q, k, v, o, B, Hq, Hkv, Sq, Sk, d, 0, 0.0f, 0, -3.06f, 2.30f, workspace, workspace_bytes,
                               nullptr, static_cast<cudaStream_t>(stream), true, true, true);
}

extern "C" efq_status_t efq_quantize_qkv(const void* q, const void* k, const void* v, int B, int Hq, int Hkv, int64_t Sq,
                                         int64_t Sk, int d, void* workspace, size_t workspace_bytes, void* stream)
{
    const void* nz_o = reinterpret_cast<const void*>(16);   // no output is written by the preparation step
    return efq::attention_impl(q, k, v, static_cast<float*>(const_cast<void*>(nz_o)), B, Hq, Hkv, Sq, Sk, d, 0, 0.0f, 0,
                               -3.06f, 2.30f, workspace, workspace_bytes, nullptr, static_cast<cudaStream_t>(stream), true,
                               false);
}

extern "C" efq_status_t efq_attention_fwd_quantized(float* o, int B, int Hq, int Hkv, int64_t Sq, int64_t Sk, int d,
                                                    int causal, float softmax_scale, int producer,
                                                    const efq_params_t* params, void* workspace, size_t workspace_bytes,
                                                    const efq_debug_t* debug, void* stream)
{
    float tau, h, threshold;
    bool lut;
    efq_status_t st;
    if (!read_params(params, tau, h, lut, threshold, st)) return st;
    if (producer == 0 && lut) producer = 3;
    const void* nz = reinterpret_cast<const void*>(16);   // operands already live in the workspace
    return efq::attention_impl(nz, nz, nz, o, B, Hq, Hkv, Sq, Sk, d, causal, softmax_scale, producer, tau, h, workspace,
                               workspace_bytes, debug, static_cast<cudaStream_t>(stream), false, true, false, threshold);
}

extern "C" efq_status_t efq_attention_fwd_host(const void* q_host, const void* k_host, const void* v_host, float* o_host,
                                               void* q_dev, void* k_dev, void* v_dev, float* o_dev, int B, int Hq, int Hkv,
                                               int64_t Sq, int64_t Sk, int d, int causal, float softmax_scale, int producer,
                                               const efq_params_t* params, void* workspace, size_t workspace_bytes,
                                               void* stream)
{
    if (!q_host || !k_host || !v_host || !o_host || !q_dev || !k_dev || !v_dev || !o_dev) return EFQ_ERR_INVALID_ARG;
    if (B <= 0 || Hq <= 0 || Hkv <= 0 || Sq <= 0 || Sk <= 0) return EFQ_ERR_INVALID_ARG;
    float tau, h, threshold;
    bool lut;
    efq_status_t st;
    if (!read_params(params, tau, h, lut, threshold, st)) return st;
    if (producer == 0 && lut) producer = 3;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const size_t qb = static_cast<size_t>(B) * Hq * Sq * d * 2, kb = static_cast<size_t>(B) * Hkv * Sk * d * 2;
    if (cudaMemcpyAsync(q_dev, q_host, qb, cudaMemcpyHostToDevice, s) != cudaSuccess) return EFQ_ERR_CUDA;
    if (cudaMemcpyAsync(k_dev, k_host, kb, cudaMemcpyHostToDevice, s) != cudaSuccess) return EFQ_ERR_CUDA;
    if (cudaMemcpyAsync(v_dev, v_host, kb, cudaMemcpyHostToDevice, s) != cudaSuccess) return EFQ_ERR_CUDA;
    st = efq::attention_impl(q_dev, k_dev, v_dev, o_dev, B, Hq, Hkv, Sq, Sk, d, causal, softmax_scale, producer, tau, h,
                             workspace, workspace_bytes, nullptr, s, true, true, false, threshold);
    if (st != EFQ_OK) return st;
    if (cudaMemcpyAsync(o_host, o_dev, static_cast<size_t>(B) * Hq * Sq * d * 4, cudaMemcpyDeviceToHost, s) != cudaSuccess)
        return EFQ_ERR_CUDA;
    return EFQ_OK;
}

namespace efq {
namespace {
// dst takes src's status if src reports one (keeps the first problem seen across the chunks of a pipelined call)
__global__ void merge_status_kernel(uint32_t* dst, const uint32_t* src, int overwrite)
{
    const uint32_t v = *src;
    if (overwrite || v != 0u) *dst = v;
}
}  // namespace
}  // namespace efq

extern "C" efq_status_t efq_attention_fwd_host_pipelined(const void* q_host, const void* k_host, const void* v_host,
                                                         float* o_host, void* q_dev, void* k_dev, void* v_dev,
                                                         float* o_dev, int B, int Hq, int Hkv, int64_t Sq, int64_t Sk,
                                                         int d, int causal, float softmax_scale, int producer,
                                                         const efq_params_t* params, void* workspace,
                                                         size_t workspace_bytes, int n_chunks, void* stream_in,
                                                         void* stream_compute, void* stream_out)
{
    if (!q_host || !k_host || !v_host || !o_host || !q_dev || !k_dev || !v_dev || !o_dev) return EFQ_ERR_INVALID_ARG;
    if (B <= 0 || Hq <= 0 || Hkv <= 0 || Sq <= 0 || Sk <= 0 || Hq % Hkv != 0 || n_chunks <= 0) return EFQ_ERR_INVALID_ARG;
    if (!workspace) return EFQ_ERR_WORKSPACE;
    float tau, h, threshold;
    bool lut;
    efq_status_t st;
    if (!read_params(params, tau, h, lut, threshold, st)) return st;
    if (producer == 0 && lut) producer = 3;
    cudaStream_t s_in = static_cast<cudaStream_t>(stream_in), s_c = static_cast<cudaStream_t>(stream_compute),
                 s_out = static_cast<cudaStream_t>(stream_out);
    // chunks are runs of KV heads inside one batch entry: contiguous slices of q, k, v and o
    int per_batch = n_chunks / B;
    if (per_batch < 1) per_batch = 1;
    if (per_batch > Hkv) per_batch = Hkv;
    const int heads_per_chunk = (Hkv + per_batch - 1) / per_batch;
    const int group = Hq / Hkv;
    if (B == 1 && heads_per_chunk >= Hkv)        // nothing to overlap: the plain form on the compute stream
        return efq_attention_fwd_host(q_host, k_host, v_host, o_host, q_dev, k_dev, v_dev, o_dev, B, Hq, Hkv, Sq, Sk, d,
                                      causal, softmax_scale, producer == 3 ? 0 : producer, params, workspace,
                                      workspace_bytes, stream_compute);
    if (!efq::shape_ok(1, heads_per_chunk * group, heads_per_chunk, Sq, Sk, d)) return EFQ_ERR_UNSUPPORTED;
    const size_t slot = efq::workspace_bytes_for(1, heads_per_chunk * group, heads_per_chunk, Sq, Sk);
    if (workspace_bytes < slot + 256) return EFQ_ERR_WORKSPACE;
    uint8_t* ws = static_cast<uint8_t*>(workspace);
    uint32_t* agg = reinterpret_cast<uint32_t*>(ws + slot);          // first problem seen by any chunk
    if (cudaMemsetAsync(agg, 0, 4, s_c) != cudaSuccess) return EFQ_ERR_CUDA;

    const size_t q_head = static_cast<size_t>(Sq) * d * 2, kv_head = static_cast<size_t>(Sk) * d * 2;
    const size_t o_head = static_cast<size_t>(Sq) * d * 4;
    cudaEvent_t ev = nullptr;
    auto fail = [&](efq_status_t code) { if (ev) cudaEventDestroy(ev); return code; };
    // The staging buffers are reused from call to call: this call's input copies must not overtake the forwards
    // of an earlier call that still read them, so stream_in first waits for what stream_compute holds now.
    if (cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) != cudaSuccess) return EFQ_ERR_CUDA;
    if (cudaEventRecord(ev, s_c) != cudaSuccess || cudaStreamWaitEvent(s_in, ev, 0) != cudaSuccess) return fail(EFQ_ERR_CUDA);
    cudaEventDestroy(ev);
    ev = nullptr;
    for (int b = 0; b < B; ++b) {
        for (int h0 = 0; h0 < Hkv; h0 += heads_per_chunk) {
            const int nh = h0 + heads_per_chunk <= Hkv ? heads_per_chunk : Hkv - h0;
            const size_t q_off = (static_cast<size_t>(b) * Hq + static_cast<size_t>(h0) * group) * q_head;
            const size_t kv_off = (static_cast<size_t>(b) * Hkv + h0) * kv_head;
            const size_t o_off = (static_cast<size_t>(b) * Hq + static_cast<size_t>(h0) * group) * o_head;
            const uint8_t* qh = static_cast<const uint8_t*>(q_host) + q_off;
            const uint8_t* kh = static_cast<const uint8_t*>(k_host) + kv_off;
            const uint8_t* vh = static_cast<const uint8_t*>(v_host) + kv_off;
            uint8_t* qd = static_cast<uint8_t*>(q_dev) + q_off;
            uint8_t* kd = static_cast<uint8_t*>(k_dev) + kv_off;
            uint8_t* vd = static_cast<uint8_t*>(v_dev) + kv_off;
            uint8_t* od = reinterpret_cast<uint8_t*>(o_dev) + o_off;
            // inputs of this chunk: stream_in
            if (cudaMemcpyAsync(qd, qh, q_head * nh * group, cudaMemcpyHostToDevice, s_in) != cudaSuccess) return fail(EFQ_ERR_CUDA);
            if (cudaMemcpyAsync(kd, kh, kv_head * nh, cudaMemcpyHostToDevice, s_in) != cudaSuccess) return fail(EFQ_ERR_CUDA);
            if (cudaMemcpyAsync(vd, vh, kv_head * nh, cudaMemcpyHostToDevice, s_in) != cudaSuccess) return fail(EFQ_ERR_CUDA);
            if (cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) != cudaSuccess) return EFQ_ERR_CUDA;
            if (cudaEventRecord(ev, s_in) != cudaSuccess || cudaStreamWaitEvent(s_c, ev, 0) != cudaSuccess) return fail(EFQ_ERR_CUDA);
            cudaEventDestroy(ev);     // released once the recorded work has completed
            ev = nullptr;
            // forward of this chunk: stream_compute (in order, so the one workspace slot is reused safely)
            st = efq::attention_impl(qd, kd, vd, reinterpret_cast<float*>(od), 1, nh * group, nh, Sq, Sk, d, causal,
                                     softmax_scale, producer, tau, h, ws, slot, nullptr, s_c, true, true, false, threshold);
            if (st != EFQ_OK) return st;
            efq::merge_status_kernel<<<1, 1, 0, s_c>>>(agg, reinterpret_cast<const uint32_t*>(ws), 0);
            if (cudaGetLastError() != cudaSuccess) return EFQ_ERR_CUDA;
            if (cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) != cudaSuccess) return EFQ_ERR_CUDA;
            if (cudaEventRecord(ev, s_c) != cudaSuccess || cudaStreamWaitEvent(s_out, ev, 0) != cudaSuccess) return fail(EFQ_ERR_CUDA);
            cudaEventDestroy(ev);
            ev = nullptr;
            // output of this chunk: stream_out
            if (cudaMemcpyAsync(static_cast<uint8_t*>(static_cast<void*>(o_host)) + o_off, od, o_head * nh * group,
                                cudaMemcpyDeviceToHost, s_out) != cudaSuccess)
                return EFQ_ERR_CUDA;
        }
    }
    // the status word efq_poll_status() reads takes the aggregate; stream_compute then waits for the last copies,
    // so that synchronising stream_compute alone completes the call
    efq::merge_status_kernel<<<1, 1, 0, s_c>>>(reinterpret_cast<uint32_t*>(ws), agg, 1);
    if (cudaGetLastError() != cudaSuccess) return EFQ_ERR_CUDA;
    if (cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) != cudaSuccess) return EFQ_ERR_CUDA;
    if (cudaEventRecord(ev, s_out) != cudaSuccess || cudaStreamWaitEvent(s_c, ev, 0) != cudaSuccess) return fail(EFQ_ERR_CUDA);
    cudaEventDestroy(ev);
    return EFQ_OK;
}

// ------------------------------------------------------------------------------------------------
// Packed variable-length batch: the sequences of the batch lie one after the other along the token axis
// ------------------------------------------------------------------------------------------------
extern "C" size_t efq_attention_varlen_workspace_bytes(const int64_t* cu_seqlens_q, const int64_t* cu_seqlens_k, int n_seqs,
                                                       int Hq, int Hkv, int d)
{
    efq_status_t st;
    efq::VarlenPlan p;
    if (!efq::plan_varlen(cu_seqlens_q, cu_seqlens_k, n_seqs, Hq, Hkv, d, p, st)) return 0;
    return p.total;
}

extern "C" efq_status_t efq_attention_fwd_varlen(const void* q, const void* k, const void* v, float* o,
                                                 const int64_t* cu_seqlens_q, const int64_t* cu_seqlens_k, int n_seqs,
                                                 int Hq, int Hkv, int d, int causal, float softmax_scale, int producer,
                                                 const efq_params_t* params, void* workspace, size_t workspace_bytes,
                                                 void* stream)
{
    using namespace efq;
    float tau, h, threshold;
    bool lut;
    efq_status_t st;
    if (!read_params(params, tau, h, lut, threshold, st)) return st;
    if (producer == 0 && lut) producer = 3;
    if (producer < 0 || producer > 6) return EFQ_ERR_INVALID_ARG;
    VarlenPlan p;
    if (!plan_varlen(cu_seqlens_q, cu_seqlens_k, n_seqs, Hq, Hkv, d, p, st)) return st;
    if (n_seqs == 0 || cu_seqlens_q[n_seqs] == 0) return EFQ_OK;     // no query token: nothing to write
    if (!q || !k || !v || !o) return EFQ_ERR_INVALID_ARG;
    if (!(softmax_scale > 0.0f)) softmax_scale = static_cast<float>(1.0 / sqrt(static_cast<double>(d)));
    if (!isfinite(softmax_scale) || !isfinite(tau) || !isfinite(h) || !(h > 0.0f)) return EFQ_ERR_INVALID_ARG;
    auto mis = [](const void* ptr, uintptr_t a) { return (reinterpret_cast<uintptr_t>(ptr) & (a - 1)) != 0; };
    if (mis(q, 16) || mis(k, 16) || mis(v, 16) || mis(o, 16)) return EFQ_ERR_ALIGNMENT;
    if (!workspace || workspace_bytes < p.total) return EFQ_ERR_WORKSPACE;
    if (mis(workspace, 256)) return EFQ_ERR_ALIGNMENT;
    const efq_status_t dev_st = check_device();
    if (dev_st != EFQ_OK) return dev_st;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    uint8_t* ws = static_cast<uint8_t*>(workspace);
    const int G = Hq / Hkv;

    // host copies of the tables, in the layout of the workspace's table region
    std::vector<uint8_t> tables(p.tables, 0);
    SeqDesc* seqs = reinterpret_cast<SeqDesc*>(tables.data() + (p.seqs_off - 1024));
    ItemGroup* groups = reinterpret_cast<ItemGroup*>(tables.data() + (p.groups_off - 1024));
    QuantJob* jobs = reinterpret_cast<QuantJob*>(tables.data() + (p.jobs_off - 1024));
    int32_t* prefix = reinterpret_cast<int32_t*>(tables.data() + (p.prefix_off - 1024));
    const __nv_bfloat16* qb = static_cast<const __nv_bfloat16*>(q);
    const __nv_bfloat16* kb = static_cast<const __nv_bfloat16*>(k);
    const __nv_bfloat16* vb = static_cast<const __nv_bfloat16*>(v);
    struct QueryTile { int32_t weight, seq, qt; };   // weight: KV tiles that it walks
    std::vector<QueryTile> order;
    order.reserve(static_cast<size_t>(p.groups));
    int64_t q_row = 0, k_row = 0, k_col = 0, ctas = 0, few_unit = 0, few_key = 0;
    int a = 0, f = 0;
    FewParams F{};
    std::vector<FewSeq> few_long;            // more sequences than the kernel parameters hold
    if (p.n_few > kFewInlineSeqs) few_long.resize(p.n_few);
    FewSeq* const few_seqs = few_long.empty() ? F.inline_seqs : few_long.data();
    for (int i = 0; i < n_seqs; ++i) {
        const int64_t q0 = cu_seqlens_q[i], k0 = cu_seqlens_k[i];
        const int64_t lq = cu_seqlens_q[i + 1] - q0, lk = cu_seqlens_k[i + 1] - k0;
        if (lq == 0) continue;
        if (lk == 0) {               // no key at all: the rows are zero, as for a causal row that sees nothing
            if (cudaMemsetAsync(o + q0 * Hq * 128, 0, static_cast<size_t>(lq) * Hq * 128 * sizeof(float), s) != cudaSuccess) return EFQ_ERR_CUDA;
            continue;
        }
        if (use_few(Hq, Hkv, lq, lk)) {
            few_seqs[f++] = FewSeq{static_cast<int32_t>(lq), static_cast<int32_t>(lk), static_cast<int32_t>(q0), static_cast<int32_t>(k0),
                                   static_cast<int32_t>(few_key), static_cast<int32_t>(few_unit)};
            few_key += (lk + kTile - 1) / kTile * kTile;
            F.longest_chunk = std::max(F.longest_chunk, few_longest_chunk(static_cast<int>((lk + kTile - 1) / kTile), G * static_cast<int>(lq)));
            few_unit += few_chunks(lk, Hq / Hkv * lq) * Hkv;
            continue;
        }
        const bool packed = use_packed_tile(Hq, Hkv, lq);
        const int64_t lq_pad = packed ? kTile : (lq + kTile - 1) / kTile * kTile, lk_pad = (lk + kTile - 1) / kTile * kTile;
        SeqDesc& sd = seqs[a];
        sd.Sq = lq; sd.Sk = lk; sd.o_off = q0 * Hq * 128; sd.token0 = static_cast<int32_t>(q0);
        sd.q_row0 = static_cast<int32_t>(q_row); sd.Sq_pad = static_cast<int32_t>(lq_pad);
        sd.k_row0 = static_cast<int32_t>(k_row); sd.Sk_pad = static_cast<int32_t>(lk_pad);
        sd.k_col0 = static_cast<int32_t>(k_col); sd.packed = packed ? 1 : 0;
        for (int64_t qt = 0; qt < lq_pad / kTile; ++qt) {
            int64_t keys = lk;
            if (causal) keys = std::min(lk, std::min((qt + 1) * kTile, lq) + lk - lq);
            order.push_back(QueryTile{static_cast<int32_t>((std::max<int64_t>(keys, 0) + kTile - 1) / kTile), a, static_cast<int32_t>(qt)});
        }
        // quantiser jobs: the sequence's own Q, K, V (token-major source: a head is 128 elements, a token H * 128)
        QuantJob& jq = jobs[3 * a];
        QuantJob& jk = jobs[3 * a + 1];
        QuantJob& jv = jobs[3 * a + 2];
        jq.kind = kQuantRows; jk.kind = kQuantRows; jv.kind = kQuantV;
        jq.seg.src = qb + q0 * Hq * 128;
        jq.seg.heads = packed ? Hkv : Hq; jq.seg.S = packed ? G * lq : lq; jq.seg.S_pad = lq_pad;
        jq.seg.head_stride = 128; jq.seg.row_stride = static_cast<int64_t>(Hq) * 128;
        jq.seg.pack_lq = packed ? static_cast<int32_t>(lq) : 0; jq.seg.pack_G = packed ? G : 1;
        jq.seg.codes = ws + p.qc + q_row * 64; jq.seg.sf = ws + p.qsf + (q_row / kTile) * kSfBytes;
        jk.seg.src = kb + k0 * Hkv * 128;
        jk.seg.heads = Hkv; jk.seg.S = lk; jk.seg.S_pad = lk_pad;
        jk.seg.head_stride = 128; jk.seg.row_stride = static_cast<int64_t>(Hkv) * 128; jk.seg.pack_G = 1;
        jk.seg.codes = ws + p.kc + k_row * 64; jk.seg.sf = ws + p.ksf + (k_row / kTile) * kSfBytes;
        jv.seg = jk.seg;
        jv.seg.src = vb + k0 * Hkv * 128;
        jv.seg.codes = ws + p.vt; jv.seg.sf = ws + p.vsf;
        jv.seg.v_row_bytes = p.k_cols / 2; jv.seg.v_x0 = k_col / 2;
        jv.seg.v_sf_tiles_per_head = p.k_cols / kTile; jv.seg.v_sf_tile0 = k_col / kTile;
        for (int t = 0; t < 3; ++t) {
            prefix[3 * a + t] = static_cast<int32_t>(ctas);
            ctas += quantize_job_ctas(jobs[3 * a + t]);
        }
        q_row += (packed ? Hkv : Hq) * lq_pad;
        k_row += Hkv * lk_pad;
        k_col += lk_pad;
        ++a;
    }
    if (p.n_few > 0) {
        F.q = qb; F.k = kb; F.v = vb; F.o = o;
        F.Hkv = Hkv; F.G = G; F.causal = causal ? 1 : 0;
        F.n_seqs = p.n_few;
        F.q_head = 128; F.q_row = static_cast<int64_t>(Hq) * 128;
        F.k_head = 128; F.k_row = static_cast<int64_t>(Hkv) * 128;
        F.row_cap = p.few_rows;
        F.n_heads = p.n_few * Hkv;
        F.n_units = static_cast<int32_t>(p.few_units);
        F.rescale_threshold = threshold;
        F.K = producer == 3 ? make_producer_consts_lut(softmax_scale) : make_producer_consts(softmax_scale, tau, h);
        const FewPlan fp = plan_few(p.few_keys * Hkv, p.few_rows);
        uint8_t* const fw = ws + p.few;
        F.scores = reinterpret_cast<float*>(fw + fp.scores); F.block_max = reinterpret_cast<float*>(fw + fp.block_max);
        F.stats = reinterpret_cast<float*>(fw + fp.stats);
        F.status = reinterpret_cast<uint32_t*>(ws);
        if (!few_long.empty()) {
            if (copy_table(ws + p.few_table, few_long, s) != cudaSuccess) return EFQ_ERR_CUDA;
            F.seqs = reinterpret_cast<const FewSeq*>(ws + p.few_table);
        }
        if (launch_few(producer, F, s) != cudaSuccess) return EFQ_ERR_CUDA;
        if (p.n_active == 0) return EFQ_OK;
    }
    if (p.n_active == 0)             // nothing to launch: the status word still has to read "no problem"
        return cudaMemsetAsync(ws, 0, 4, s) == cudaSuccess ? EFQ_OK : EFQ_ERR_CUDA;
    prefix[3 * p.n_active] = static_cast<int32_t>(ctas);
    // The heaviest query tiles of the whole batch first, so that the last CTAs to start are short ones.
    std::stable_sort(order.begin(), order.end(), [](const QueryTile& x, const QueryTile& y) { return x.weight > y.weight; });
    int64_t n_items = 0;
    std::vector<ItemRun> runs;
    for (size_t i = 0; i < order.size(); ++i) {
        const SeqDesc& sd = seqs[order[i].seq];
        groups[i] = ItemGroup{static_cast<int32_t>(n_items), order[i].seq, order[i].qt, order[i].weight, static_cast<int32_t>(sd.Sq),
                              static_cast<int32_t>(sd.Sk), sd.packed};
        const int heads = sd.packed ? Hkv : Hq;
        if (i > 0 && order[i].weight == order[i - 1].weight) runs.back().count += heads;
        else runs.push_back(ItemRun{order[i].weight, heads});
        n_items += heads;
    }

    FwdParams P{};
    P.B = p.n_active; P.Hq = Hq; P.Hkv = Hkv; P.Sq = 0; P.Sk = p.longest; P.Sq_pad = 0; P.Sk_pad = 0;
    P.causal = causal ? 1 : 0;
    P.K = producer == 3 ? make_producer_consts_lut(softmax_scale) : make_producer_consts(softmax_scale, tau, h);
    P.sf_q = ws + p.qsf; P.sf_k = ws + p.ksf; P.sf_v = ws + p.vsf;
    P.o = o;
    P.o_head = 128;                                   // token-major: a head is 128 elements, a token Hq * 128
    P.o_row = static_cast<int64_t>(Hq) * 128;
    P.o_tokens = cu_seqlens_q[n_seqs];
    P.status = reinterpret_cast<uint32_t*>(ws);
    P.packed = 0;
    P.seqs = reinterpret_cast<const SeqDesc*>(ws + p.seqs_off);
    P.items = reinterpret_cast<const ItemDesc*>(ws + p.items_off);
    P.v_tiles_per_head = p.k_cols / kTile;
    P.inject_skip_loads = 0;
    P.rescale_threshold = threshold;
    P.has_dbg = 0;
    P.dbg = efq_debug_t{};

    // persistent CTAs: places of the items, if one after the other is not good enough
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return EFQ_ERR_CUDA;
    const int sms = sm_count(dev);
    int64_t n_places = 0;
    if (use_short(producer, false, n_items, sms, P)) n_places = order_items(runs, n_items, sms, reinterpret_cast<int32_t*>(tables.data() + (p.places_off - 1024)));
    const int32_t* const places = n_places > 0 ? reinterpret_cast<const int32_t*>(ws + p.places_off) : nullptr;
    tables.resize(p.places_off - 1024 + sizeof(int32_t) * static_cast<size_t>(n_places));
    if (n_places == 0) n_places = n_items;

    if (copy_table(ws + 1024, tables, s) != cudaSuccess) return EFQ_ERR_CUDA;
    if (launch_quantize_jobs(reinterpret_cast<const QuantJob*>(ws + p.jobs_off), reinterpret_cast<const int32_t*>(ws + p.prefix_off),
                             3 * p.n_active, ctas, reinterpret_cast<const ItemGroup*>(ws + p.groups_off), static_cast<int>(order.size()), places, n_places,
                             reinterpret_cast<ItemDesc*>(ws + p.items_off), p.n_few > 0 ? nullptr : reinterpret_cast<uint32_t*>(ws), s) != cudaSuccess)
        return EFQ_ERR_CUDA;

    CUtensorMap mq, mk, mv;
    if (!encode_map(&mq, ws + p.qc, 64, static_cast<uint64_t>(p.q_rows))) return EFQ_ERR_CUDA;
    if (!encode_map(&mk, ws + p.kc, 64, static_cast<uint64_t>(p.k_rows))) return EFQ_ERR_CUDA;
    if (!encode_map(&mv, ws + p.vt, static_cast<uint64_t>(p.k_cols / 2), static_cast<uint64_t>(Hkv) * 128)) return EFQ_ERR_CUDA;

    return launch_forward(producer, false, n_places, s, mq, mk, mv, P) == cudaSuccess ? EFQ_OK : EFQ_ERR_CUDA;
}

extern "C" efq_status_t efq_poll_status(void* workspace, void* stream)
{
    if (!workspace) return EFQ_ERR_INVALID_ARG;
    uint32_t word = 0;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (cudaMemcpyAsync(&word, workspace, 4, cudaMemcpyDeviceToHost, s) != cudaSuccess) return EFQ_ERR_CUDA;
    if (cudaStreamSynchronize(s) != cudaSuccess) return EFQ_ERR_CUDA;
    return word == 0 ? EFQ_OK : (word == EFQ_ERR_DEVICE_TIMEOUT ? EFQ_ERR_DEVICE_TIMEOUT : EFQ_ERR_CUDA);
}

// ------------------------------------------------------------------------------------------------
// Forward without a caller-supplied workspace
// ------------------------------------------------------------------------------------------------
// Scratch for efq_attention_fwd_static: lives in the library image, one copy per device that loads it.
static __device__ __align__(256) uint8_t g_static_scratch[EFQ_STATIC_SCRATCH_BYTES];

namespace {

constexpr int kMaxDevices = 64;   // device ordinals this table covers
std::mutex g_static_mutex;
void* g_static_ptr[kMaxDevices] = {};   // device address of g_static_scratch, per device ordinal

// The array's name is only a host-side handle; kernels need its device address, which differs per device.
// Looked up once per device with that device current.
efq_status_t static_scratch_for_current_device(void** out)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return EFQ_ERR_CUDA;
    if (dev < 0 || dev >= kMaxDevices) return EFQ_ERR_UNSUPPORTED;
    std::lock_guard<std::mutex> lock(g_static_mutex);
    if (!g_static_ptr[dev]) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_static_scratch) != cudaSuccess || !p) return EFQ_ERR_CUDA;
        g_static_ptr[dev] = p;
    }
    *out = g_static_ptr[dev];
    return EFQ_OK;
}

}  // namespace

extern "C" efq_status_t efq_attention_fwd_static(const void* q, const void* k, const void* v, float* o, int B, int Hq,
                                                 int Hkv, int64_t Sq, int64_t Sk, int d, int causal,
                                                 float softmax_scale, const efq_params_t* params, void* stream)
{
    float tau, h, threshold;
    bool lut;
    efq_status_t st;
    if (!read_params(params, tau, h, lut, threshold, st)) return st;
    // the argument rules of efq_attention_fwd, in its order, before the size of the problem is looked at
    if (!q || !k || !v || !o) return EFQ_ERR_INVALID_ARG;
    if (B <= 0 || Hq <= 0 || Hkv <= 0 || Sq <= 0 || Sk <= 0 || Hq % Hkv != 0) return EFQ_ERR_INVALID_ARG;
    if (d != 128) return EFQ_ERR_UNSUPPORTED;
    const size_t need = efq_attention_workspace_bytes(B, Hq, Hkv, Sq, Sk, d);
    if (need == 0) return EFQ_ERR_UNSUPPORTED;
    if (need > EFQ_STATIC_SCRATCH_BYTES) return EFQ_ERR_STATIC_LIMIT;
    void* scratch = nullptr;
    st = static_scratch_for_current_device(&scratch);
    if (st != EFQ_OK) return st;
    return efq::attention_impl(q, k, v, o, B, Hq, Hkv, Sq, Sk, d, causal, softmax_scale, lut ? 3 : 0, tau, h, scratch,
                               EFQ_STATIC_SCRATCH_BYTES, nullptr, static_cast<cudaStream_t>(stream), true, true, false, threshold);
}
