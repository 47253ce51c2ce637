// Fused forward with persistent CTAs: the kernel of attention_fwd.cu (which includes this file) for more query tiles than SMs, at
// every length of the KV walk (its name is from the short walks that it was made for).
//
// A CTA of attention_fwd_kernel spends about 10000 cycles outside its tiles: start, barriers, TMEM, the latency of the first
// loads and scores, the last P~V, the rows on their way out.  Against 512 keys, 4 tiles of about 1500 cycles, that is more than
// the work.  Here one CTA per SM walks a list of query tiles and nothing of that stands between two of them: Q is
// double-buffered and loads run ahead into the next item, S of its first tiles is computed while the last codes of this one
// are generated, and the rescaling warps take the finished rows out while the probability warps are in the next item.  The
// tile counter t runs over all items of the CTA: it picks buffers and phases, the tile j inside the item picks the keys.
// Everything else, the arithmetic above all, is that of attention_fwd_kernel, and so is the result, bit for bit.
//
// What bounds it: the probability warps in long walks; in short ones what stands between the last P~V of an item and the first
// rescaling of the next, and the size of the code.  The five kinds of warp run different code at the same time and evict one
// another from the instruction cache: with 65 KB of code 13 % of its lookups missed against 256 keys and 10 % against 512, with the 51 KB of
// now 6 % and 5 %; a form of 75 KB, not kept, missed 40 %, and warps without an instruction were its largest stall.  Hence waits of
// a few instructions, masks from a bit word, loops that are not unrolled, no divisions from item to item.
//
// Measured against one CTA per tile, whole call, us.  Affine rule, 24 heads, 16000 queries, not causal: 128 keys 146 -> 65, 256 keys
// 159 -> 83, 512 191 -> 109, 1024 254 -> 167, 2048 378 -> 288, 4096 619 -> 527, 16384 1998 -> 1897; causal, 32 heads: 32 x 128 tokens
// 55 -> 32, 2048 tokens 49 -> 37, 4096 129 -> 107, 16384 1436 -> 1300, 32768 5228 -> 4952.  Packed, 32 / 8 heads, causal: 64 of 64 to
// 128 tokens 128 -> 93, 16 of 100 to 3000 548 -> 383 (not causal 743 -> 580), 4 x 8192 1702 -> 1460, 4 x 16384 5772 -> 5355.
// Plain exponentials: 4096 keys 500 -> 450, 16384 keys 1738 -> 1696, causal 4096 tokens 187 -> 162, 16384 2300 -> 2158; folded ones
// 401 -> 355, 1358 -> 1315, 152 -> 129, 1806 -> 1660.
#pragma once

struct __align__(1024) ShortSmem : Smem {
    uint8_t q1[kTileBytes];                // query tile of every other item (the first one's is Smem::q)
    uint8_t stage[4][kTile * 128];         // finished rows on their way out: 32 channels of each, 128-byte swizzle
    uint8_t sf_q1[kSfBytes];
    uint64_t q_ready[2], q_empty[2];
    uint64_t finished;                     // the rescaling warps have left their loop
};
constexpr uint32_t kColSfQ1 = 440;         // scales of q1: 4 columns behind those of V

// The items of this CTA, one after the other: the CTAs take items in turn, every other round in reverse, so that the heavier items
// of a round go to those that had the lighter ones before.  Every role walks them for itself, so a step has to be short: it
// stands between the last tile of an item and the first of the next.  [B, H, S, d] batch (heaviest query tiles first, the heads of a
// GQA group adjacent): query tile and head by additions.  Packed batch (TABLE; items in the places of a table, item_order.h): the
// entry of the next item is on its way while this one is worked on; an empty place is the end.
template <bool TABLE>
struct ShortWalk {
    uint32_t k;                    // items before this one
    uint32_t quo, rem;             // dense: index of the item divided by the heads
    uint32_t step[2];              // dense: the way to the next item after an even, an odd k: quotient << 16 | remainder
    ItemDesc it, next;             // packed batch; n_tiles < 0 past the last item

    __device__ __forceinline__ ItemDesc fetch(const FwdParams& P, uint32_t n_items, uint32_t i) const
    {
        const uint32_t index = i * gridDim.x + ((i & 1u) ? gridDim.x - 1u - blockIdx.x : blockIdx.x);
        ItemDesc d;
        d.n_tiles = -1;
        if (index < n_items) d = P.items[index];
        return d;
    }
    __device__ __forceinline__ ShortWalk(const FwdParams& P, uint32_t n_items) : k(0)
    {
        if (TABLE) {
            it = fetch(P, n_items, 0);
            next = fetch(P, n_items, 1);
        } else {
            const uint32_t heads = static_cast<uint32_t>(P.B) * P.Hq, even = 2u * (gridDim.x - blockIdx.x) - 1u, odd = 2u * blockIdx.x + 1u;
            // numbers up to twice the SMs: exact for every count of heads, and a remainder fits 16 bits
            auto div = [&](uint32_t x) { return P.heads_magic != 0u ? __umulhi(x, P.heads_magic) : x; };
            quo = div(blockIdx.x); rem = blockIdx.x - quo * heads;
            step[0] = div(even); step[0] = step[0] << 16 | (even - step[0] * heads);
            step[1] = div(odd); step[1] = step[1] << 16 | (odd - step[1] * heads);
        }
    }
    __device__ __forceinline__ void advance(const FwdParams& P, uint32_t n_items)
    {
        ++k;
        if (TABLE) {
            it = next;
            next = fetch(P, n_items, k + 1);
        } else {
            const uint32_t heads = static_cast<uint32_t>(P.B) * P.Hq, s = (k & 1u) ? step[0] : step[1];
            quo += s >> 16;
            rem += s & 0xffffu;
            if (rem >= heads) { rem -= heads; ++quo; }
        }
    }
    __device__ __forceinline__ bool valid(const FwdParams& P) const { return TABLE ? it.n_tiles >= 0 : quo < static_cast<uint32_t>(P.Sq_pad) / kTile; }
    __device__ __forceinline__ bool packed() const { return TABLE && it.packed != 0; }
    __device__ __forceinline__ int Sq(const FwdParams& P) const { return TABLE ? it.Sq : static_cast<int>(P.Sq); }
    __device__ __forceinline__ int Sk(const FwdParams& P) const { return TABLE ? it.Sk : static_cast<int>(P.Sk); }
    __device__ __forceinline__ int q0(const FwdParams& P) const     // first row (packed: 0)
    {
        return TABLE ? it.qt * kTile : static_cast<int>(static_cast<uint32_t>(P.Sq_pad) / kTile - 1u - quo) * kTile;
    }
    __device__ __forceinline__ int n_tiles(const FwdParams& P) const
    {
        if (TABLE) return it.n_tiles;
        const int all = (Sk(P) + kTile - 1) / kTile;
        if (!P.causal) return all;
        const int last_key = min(q0(P) + kTile, Sq(P)) - 1 + Sk(P) - Sq(P);       // may be negative: nothing visible
        return last_key < 0 ? 0 : min(all, last_key / kTile + 1);
    }
};

// Where an item's operands and rows lie: rows q0 .. q0 + 127 of a query head or - "packed", in a variable-length batch - row r =
// token r % Sq of query head r / Sq of a KV group.  Each role uses the fields that it needs; the others are never computed.
struct ShortItem {
    int q_row, k_row0, v_x0, v_row0;      // in the code matrices
    int64_t sfv_tile0, o;                 // o: element offset of row 0 of its (first) query head in the output
    int o_y, o_z;                         // the item's first row in the tensor map of the output: token, head
};
template <bool TABLE>
__device__ __forceinline__ ShortItem short_decode(const FwdParams& P, const ShortWalk<TABLE>& walk)
{
    ShortItem w;
    const int q0 = walk.q0(P);
    if (TABLE) {
        const SeqDesc sd = P.seqs[walk.it.seq];
        const int G = P.Hq / P.Hkv, head = walk.it.head;
        const int hkv = walk.packed() ? head : head / G, head0 = walk.packed() ? head * G : head;
        w.q_row = sd.q_row0 + (walk.packed() ? hkv * kTile : head0 * sd.Sq_pad + q0);
        w.k_row0 = sd.k_row0 + hkv * sd.Sk_pad;
        w.v_x0 = sd.k_col0 / 2;
        w.v_row0 = hkv * kTile;
        w.sfv_tile0 = static_cast<int64_t>(hkv) * P.v_tiles_per_head + sd.k_col0 / kTile;
        w.o = sd.o_off + head0 * P.o_head;
        w.o_y = sd.token0 + q0; w.o_z = head0;
    } else {
        const uint32_t bh = walk.rem, kvh = bh / static_cast<uint32_t>(P.Hq / P.Hkv);      // B * Hkv heads, G of Q for each
        w.q_row = static_cast<int>(bh * static_cast<uint32_t>(P.Sq_pad)) + q0;
        w.k_row0 = static_cast<int>(kvh * static_cast<uint32_t>(P.Sk_pad));
        w.v_x0 = 0;
        w.v_row0 = static_cast<int>(kvh) * kTile;
        w.sfv_tile0 = w.k_row0 / kTile;
        w.o = static_cast<int64_t>(bh) * P.o_head;
        w.o_y = q0; w.o_z = static_cast<int>(bh);
    }
    return w;
}

template <int PRODUCER, bool TABLE>
__global__ void __launch_bounds__(kThreads, 1)
attention_short_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                       const __grid_constant__ CUtensorMap map_v, const __grid_constant__ CUtensorMap map_o, const FwdParams P, const uint32_t n_items)
{
    static_assert(PRODUCER != 6, "the denominator of FP32 exponentials is summed by attention_fwd_kernel only");
    extern __shared__ uint8_t smem_raw[];
    ShortSmem* sm = reinterpret_cast<ShortSmem*>(smem_raw + ptx::smem_round_up(smem_raw, 1024u));
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;

    if (warp == 0) {
        if (lane == 0) {
            ptx::prefetch_tensormap(&map_q);
            ptx::prefetch_tensormap(&map_k);
            ptx::prefetch_tensormap(&map_v);
            ptx::prefetch_tensormap(&map_o);
            sm->abort_flag = 0u;
            sm->progress = 0u;
            for (int s = 0; s < kStages; ++s) {
                ptx::mbar_init(&sm->k_full[s], 1);
                ptx::mbar_init(&sm->k_empty[s], 1);
                ptx::mbar_init(&sm->v_full[s], 1);
                ptx::mbar_init(&sm->v_empty[s], 1);
            }
            for (int i = 0; i < 2; ++i) {
                ptx::mbar_init(&sm->q_ready[i], 1);
                ptx::mbar_init(&sm->q_empty[i], 1);
                ptx::mbar_init(&sm->s_full[i], 1);
                ptx::mbar_init(&sm->s_empty[i], kGroupWarps);
                ptx::mbar_init(&sm->p_full[i], kGroupWarps);
                ptx::mbar_init(&sm->p_empty[i], 1);
            }
            ptx::mbar_init(&sm->finished, 4);
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

    // 4 x 32 + 8 x 184 + 4 x 112 = 2048 registers per lane, what the launch holds
    if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 32;");
    if (warp == 0 && lane == 0) {
        // =============================== TMA producer (one thread) ===============================
        // The operands come from the kernel before.  Whatever else this kernel writes or reads follows from the loads.
        ptx::grid_wait();
        int s = 0, n = 0;
        uint32_t ph = 0;
        bool ok = true;
        for (ShortWalk<TABLE> walk(P, n_items); ok && walk.valid(P); walk.advance(P, n_items)) {
            const int n_tiles = walk.n_tiles(P);
            if (n_tiles <= 0) continue;
            const ShortItem w = short_decode<TABLE>(P, walk);
            const int qb = n & 1;
            if (!wait1(&sm->q_empty[qb], (static_cast<uint32_t>(n >> 1) & 1u) ^ 1u, sm)) break;
            ptx::mbar_arrive_expect_tx(&sm->q_ready[qb], kTileBytes + kSfBytes);
            ptx::tma_load_2d(qb ? sm->q1 : sm->q, &map_q, 0, w.q_row, &sm->q_ready[qb]);
            ptx::bulk_load_1d(qb ? sm->sf_q1 : sm->sf_q, P.sf_q + static_cast<int64_t>(w.q_row / kTile) * kSfBytes, kSfBytes, &sm->q_ready[qb]);
            ++n;
            const int64_t sfk_tile0 = w.k_row0 / kTile;
            for (int j = 0; j < (P.inject_skip_loads ? 0 : n_tiles); ++j) {
                // Stage barriers of their own: a waiter on a barrier that other roles may complete twice before it
                // looks (S runs ahead) could not tell which completion it sees by parity.
                if (!wait1(&sm->k_empty[s], ph ^ 1u, sm)) { ok = false; break; }
                ptx::mbar_arrive_expect_tx(&sm->k_full[s], kTileBytes + kSfBytes);
                ptx::tma_load_2d(sm->k[s], &map_k, 0, w.k_row0 + j * kTile, &sm->k_full[s]);
                ptx::bulk_load_1d(sm->sf_k[s], P.sf_k + (sfk_tile0 + j) * kSfBytes, kSfBytes, &sm->k_full[s]);
                if (!wait1(&sm->v_empty[s], ph ^ 1u, sm)) { ok = false; break; }
                ptx::mbar_arrive_expect_tx(&sm->v_full[s], kTileBytes + kSfBytes);
                ptx::tma_load_2d(sm->v[s], &map_v, w.v_x0 + j * 64, w.v_row0, &sm->v_full[s]);
                ptx::bulk_load_1d(sm->sf_v[s], P.sf_v + (w.sfv_tile0 + j) * kSfBytes, kSfBytes, &sm->v_full[s]);
                if (++s == kStages) { s = 0; ph ^= 1u; }
            }
        }
    } else if (warp == 3 && lane == 0) {
        ptx::grid_wait();
        // an earlier CTA of this launch gave up: the waits of this one end soon instead of after their limit
        if (*reinterpret_cast<volatile uint32_t*>(P.status) != 0u) sm->abort_flag = 1u;
        // No early launch of what follows, as there (2 x 16 heads, causal, 1087 queries of 470 keys 13.2 us, with it 14.4; 2048 tokens 35.3 and
        // 35.4; the 16 forwards of a calibration 794 and 796).
        wait_watching(&sm->finished, 0, sm, P.status);
    } else if (warp == 1) {
        // =============================== S = Q K^T issuer ===============================
        // The whole warp runs the loop with warp-uniform state; one elected lane issues the tcgen05
        // instructions.  Descriptors differ from tile to tile only in the start-address field (address >> 4).
        const uint64_t d_sw64 = ptx::smem_desc(0, 16, 512, ptx::kLayoutSw64);
        const uint64_t d_sf = ptx::smem_desc(0, 16, 128, ptx::kLayoutNone);
        if (TABLE) ptx::grid_wait();                           // the item table is written by the kernel before
        int ks = 0, n = 0;
        uint32_t t = 0;                                       // t: tiles of this CTA so far, over all of its items
        uint32_t kph = 0;
        bool ok = true;
        for (ShortWalk<TABLE> walk(P, n_items); ok && walk.valid(P); walk.advance(P, n_items)) {
            const int n_tiles = walk.n_tiles(P);
            if (n_tiles <= 0) continue;
            const int qb = n & 1;
            const uint64_t dq0 = d_sw64 + (ptx::smem_u32(qb ? sm->q1 : sm->q) >> 4);
            const uint32_t sfq = tmem + (qb ? kColSfQ1 : kColSfQ);
            if (!wait_all(&sm->q_ready[qb], static_cast<uint32_t>(n >> 1) & 1u, sm)) break;
            ++n;
            ptx::tc_fence_after_sync();
            if (ptx::elect_one()) ptx::tmem_cp_sf(sfq, d_sf + (ptx::smem_u32(qb ? sm->sf_q1 : sm->sf_q) >> 4));
            __syncwarp();
            for (int j = 0; j < n_tiles; ++j, ++t) {
                const int sb = static_cast<int>(t & 1u);
                if (!wait_all(&sm->k_full[ks], kph, sm)) { ok = false; break; }
                if (!wait_all(&sm->s_empty[sb], ((t >> 1) & 1u) ^ 1u, sm)) { ok = false; break; }
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
                    if (j + 1 == n_tiles) ptx::mma_commit(&sm->q_empty[qb]);
                }
                __syncwarp();
                if (++ks == kStages) { ks = 0; kph ^= 1u; }
            }
        }
    } else if (warp == 2) {
        // =============================== [dA | dl] = P~ [V | 1] issuer ===============================
        const uint64_t d_sw64 = ptx::smem_desc(0, 16, 512, ptx::kLayoutSw64);
        const uint64_t d_sf = ptx::smem_desc(0, 16, 128, ptx::kLayoutNone);
        if (ptx::elect_one()) {
            const uint64_t d1 = d_sf + (ptx::smem_u32(sm->sf_ones) >> 4);
            ptx::tmem_cp_sf(tmem + kColSfV + 4, d1);
            ptx::tmem_cp_sf(tmem + kColSfV + 12, d1);
        }
        __syncwarp();
        if (TABLE) ptx::grid_wait();
        uint32_t t = 0;
        bool ok = true;
        for (ShortWalk<TABLE> walk(P, n_items); ok && walk.valid(P); walk.advance(P, n_items)) {
            const int n_tiles = walk.n_tiles(P);
            for (int j = 0; j < n_tiles; ++j, ++t) {
                const int pb = static_cast<int>(t & 1u), vs = static_cast<int>(t % kStages);
                if (!wait_all(&sm->v_full[vs], (t / kStages) & 1u, sm)) { ok = false; break; }
                if (!wait_all(&sm->p_full[pb], (t >> 1) & 1u, sm)) { ok = false; break; }
                if (!wait_all(&sm->o_ready[t & 3u], (t >> 2) & 1u, sm)) { ok = false; break; }
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
                    sm->progress = t + 1u;
                }
                __syncwarp();
            }
        }
    }
    } else if (warp >= 12) {
    // =============================== historical rescaling (Eq. alpha), rows out ===============================
    // One warp per TMEM lane quarter: the accumulator rows that grew, as in attention_fwd_kernel, and the finished rows of an
    // item, whose way out takes no time from the probability warps here.
    asm volatile("setmaxnreg.dec.sync.aligned.u32 112;");
    const int quarter = warp & 3;
    const uint32_t row = quarter * 32 + lane;
    const uint32_t o_addr = tmem + (static_cast<uint32_t>(quarter * 32) << 16) + kColO;
    // this lane's row of the staging: 16-byte pieces, their order turned by the row
    uint8_t* const my_stage = sm->stage[0] + row * 128;
    const uint32_t turn = (row & 7u) * 16u;
    // The warp's 32 rows of a finished item wait in the staging as four boxes of 32 channels, which one lane hands to the copy
    // engine.  That takes it some 1500 cycles, in which the first P~V of the next item would wait for its rescaling: so it is done
    // after that rescaling, while P~V runs (32 heads, causal, 16384 tokens 1393 -> 1328 us; 24 heads, 32760 queries, 512 keys 221 -> 210).
    int box_y = -1, box_z = 0;
    auto send_rows = [&]() {
        if (box_y >= 0 && lane == 0) {
#pragma unroll
            for (int c = 0; c < 4; ++c) ptx::tma_store_3d(&map_o, sm->stage[c] + 4096 * quarter, 32 * c, box_y, box_z);
            ptx::bulk_commit();
        }
        box_y = -1;
    };
    ptx::grid_wait();
    uint32_t t = 0;
    bool ok = true;
    if (lane == 0) ptx::mbar_arrive(&sm->o_ready[0]);         // the first tile overwrites the accumulator
    __syncwarp();
    ShortWalk<TABLE> walk(P, n_items);
    for (; ok && walk.valid(P); walk.advance(P, n_items)) {
        const int n_tiles = walk.n_tiles(P);
        if (n_tiles <= 0) {                                   // zeros, below
            if (TABLE) break;
            continue;
        }
        for (int j = 0; j < n_tiles; ++j, ++t) {
            if (j == 0) continue;                         // released when the accumulator was free, below
            if (!wait_all(&sm->a_bar[t & 3u][quarter], (t >> 2) & 1u, sm)) { ok = false; break; }
            const float alpha = sm->alpha[t & 3u][row];
            if (__any_sync(0xffffffffu, alpha != 1.0f)) {
                // The end of P~V of the tile before frees its V stage.  The parity says so only if the stage's use before has
                // ended, and it has: the probability warps waited for it before they stored the codes of the tile two before.
                if (!wait_all(&sm->v_empty[(t - 1u) & 3u], ((t - 1u) >> 2) & 1u, sm)) { ok = false; break; }
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
            if (lane == 0) ptx::mbar_arrive(&sm->o_ready[t & 3u]);
            send_rows();
            __syncwarp();
        }
        // ---- final normalisation O = A / l: out of TMEM, so that P~V of the next item may start, into the staging
        if (!ok || !wait_all(&sm->v_empty[(t - 1u) & 3u], ((t - 1u) >> 2) & 1u, sm)) break;
        ptx::tc_fence_after_sync();
        const uint32_t lcol = ptx::tmem_ld1(o_addr + 128);
        ptx::tmem_wait_ld();
        const float l = __uint_as_float(lcol);
        const float inv = l > 0.0f ? 1.0f / l : 0.0f;
        send_rows();
        if (lane == 0) ptx::bulk_wait_read();             // the rows of the item before have left the staging
        __syncwarp();
#pragma unroll 1
        for (int c = 0; c < 4; ++c) {
            uint32_t o[32];
            ptx::tmem_ld32<0>(o_addr + 32 * c, o);
            ptx::tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 8; ++i)
                *reinterpret_cast<float4*>(my_stage + c * (kTile * 128) + ((16 * i) ^ turn)) =
                    make_float4(__uint_as_float(o[4 * i]) * inv, __uint_as_float(o[4 * i + 1]) * inv, __uint_as_float(o[4 * i + 2]) * inv, __uint_as_float(o[4 * i + 3]) * inv);
        }
        ptx::tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(&sm->o_ready[t & 3u]);        // first tile of the next item, if there is one
        // Rows out: as boxes (send_rows), later.  Rows of several heads, and in a packed batch the last rows of a sequence, whose
        // box would reach into the next one, go the long way.
        ptx::fence_proxy_async_smem();
        __syncwarp();
        const ShortItem w = short_decode<TABLE>(P, walk);
        const int left = walk.Sq(P) - walk.q0(P) - 32 * quarter;              // rows from the warp's first on
        if (!walk.packed() && (!TABLE || left >= 32)) {
            if (left > 0) { box_y = w.o_y + 32 * quarter; box_z = w.o_z; }
            if (n_tiles == 1) send_rows();                    // the next item may have no rescaling either
        } else if (TABLE) {
            const int lq = walk.Sq(P), heads = walk.packed() ? P.Hq / P.Hkv : 1;
#pragma unroll 4
            for (int i = 0; i < 32; ++i) {
                const int r = 32 * quarter + i, gq = walk.packed() ? r / lq : 0, token = walk.packed() ? r - gq * lq : walk.q0(P) + r;
                const float4 v = *reinterpret_cast<const float4*>(sm->stage[lane >> 3] + r * 128 + (((lane ^ r) & 7) * 16));
                if (gq < heads && token < lq) __stcs(reinterpret_cast<float4*>(P.o + (w.o + gq * P.o_head + token * P.o_row)) + lane, v);
            }
        }
        __syncwarp();
    }
    send_rows();
    // Rows without a visible key: zeros, which need no staging, in a loop of their own.  The lightest items come last, so they are what
    // is left of a packed batch; the other form walks again (the faster way in each).  With the boxes that the other rows take, and the
    // code for it in the loop above, two batches of 16 heads, causal, 1087 queries of 470 keys took 16.7 us (scale4: 19.3), 32 heads, 16384
    // queries of 2000 keys 146; without 14.4 (16.3) and 104.
    auto zero_rows = [&](const ShortWalk<TABLE>& at) {
        const ShortItem w = short_decode<TABLE>(P, at);
        const int lq = at.Sq(P), heads = at.packed() ? P.Hq / P.Hkv : 1;
#pragma unroll 1
        for (int r = 32 * quarter; r < 32 * quarter + 32; ++r) {
            const int gq = at.packed() ? r / lq : 0, token = at.packed() ? r - gq * lq : at.q0(P) + r;
            if (gq < heads && token < lq) __stcs(reinterpret_cast<float4*>(P.o + (w.o + gq * P.o_head + token * P.o_row)) + lane, make_float4(0.f, 0.f, 0.f, 0.f));
        }
    };
    if (TABLE) {
        for (; ok && walk.valid(P); walk.advance(P, n_items)) zero_rows(walk);
    } else if (P.causal && P.Sq > P.Sk) {
        for (ShortWalk<TABLE> again(P, n_items); ok && again.valid(P); again.advance(P, n_items))
            if (again.n_tiles(P) <= 0) zero_rows(again);
    }
    if (lane == 0) {
        ptx::bulk_wait_read();                                // shared memory ends with the CTA
        ptx::mbar_arrive(&sm->finished);
    }
    __syncwarp();
    } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 184;");
    const int quarter = warp & 3;                       // TMEM lane quarter this warp may touch
    const int group = (warp - 4) >> 2;                  // group 0 takes the even KV tiles, group 1 the odd ones
    const uint32_t row = quarter * 32 + lane;           // row inside the query tile: one thread owns one row
    const uint32_t lane_base = static_cast<uint32_t>(quarter * 32) << 16;
    const ProducerConsts K = P.K;
    if (TABLE) ptx::grid_wait();
    uint32_t base = 0;                                  // tiles of this CTA before the item: buffers and phases count over all items
    bool ok = true;
    bool in_flight = false;           // the scores of this tile were asked for at the end of the group's previous tile
    float r[128];
    const uint32_t s_addr = tmem + lane_base + kColS + 128 * group;
    for (ShortWalk<TABLE> walk(P, n_items); ok && walk.valid(P); walk.advance(P, n_items)) {
        const int n_tiles = walk.n_tiles(P);
        if (n_tiles <= 0) continue;
        const int token = walk.packed() ? static_cast<int>(row) % walk.Sq(P) : walk.q0(P) + static_cast<int>(row);
        const int sees = P.causal ? token + walk.Sk(P) - walk.Sq(P) : walk.Sk(P) - 1;
        const int limit = min(max(sees, -1), walk.Sk(P) - 1);   // last visible key of this row
        __syncwarp();

        for (int j = static_cast<int>((base & 1u) ^ static_cast<uint32_t>(group)); j < n_tiles; j += 2) {
            const uint32_t t = base + static_cast<uint32_t>(j);
            const int sb = group;                                         // S, P and exchange buffers belong to the group
            const uint32_t ph2 = (t >> 1) & 1u;

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
                // the other group's publication and the maximum it carries are asked for while the scores travel, as in
                // attention_fwd_kernel
                have_prev = t == 0 || ptx::mbar_try_wait(&sm->a_bar[(t - 1u) & 3u][quarter], ((t - 1u) >> 2) & 1u);
                if (j > 0 && have_prev) m_prev = sm->runmax[sb ^ 1][row];
                ptx::tmem_wait_ld();
                ptx::tc_fence_before_sync();          // the S buffer is handed back with the joint publication below
                const int last = limit - j * kTile;       // last visible key of the row inside the tile
                if (__any_sync(0xffffffffu, last < 127)) {     // diagonal or ragged tile: keys past the row's limit are masked in place
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
                if (!wait_all(&sm->a_bar[(t - 1u) & 3u][quarter], ((t - 1u) >> 2) & 1u, sm)) { ok = false; break; }
                if (j > 0) m_prev = sm->runmax[sb ^ 1][row];
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
            sm->alpha[t & 3u][row] = alpha;
            __syncwarp();
            if (lane == 0) {
                ptx::mbar_arrive(&sm->a_bar[t & 3u][quarter]);
                ptx::mbar_arrive(&sm->s_empty[sb]);           // every lane's scores are in registers (wait::ld above)
            }
            // P~V of tile j-2 reads the group's P buffer: asked here, answered while block 0 is computed
            const bool have_p = ptx::mbar_try_wait(&sm->p_empty[sb], ph2 ^ 1u);

            // ---- probability operand (Algorithm 1 per block): codes and scales straight into the MMA operand
            uint32_t sfword = 0;
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                uint4 codes;
                uint32_t byte;
                produce32<PRODUCER>(&r[g * 32], bmax[g], m_s, K, codes, byte);
                if (g == 0 && !have_p) {      // P~V of tile j-2 must have finished: it reads the group's P buffer
                    if (!wait_all(&sm->p_empty[sb], ph2 ^ 1u, sm)) { ok = false; break; }
                }
                *reinterpret_cast<uint4*>(sm->p[sb] + code_tile_offset(row, g)) = codes;
                sfword |= byte << (8 * g);
            }
            if (!ok) break;               // the bounded wait inside the block loop gave up
            *reinterpret_cast<uint32_t*>(sm->sf_p[sb] + (row & 31u) * 16u + (row >> 5) * 4u) = sfword;
            // The registers are free: if S of the group's next tile, of this item or of one after it, is there already (it is as a
            // rule, S runs ahead), its scores set out now and travel while the operand is handed over and the loop turns.
            in_flight = ptx::mbar_test_wait(&sm->s_full[sb], ph2 ^ 1u);
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
        base += static_cast<uint32_t>(n_tiles);
    }
    ptx::tmem_wait_ld();                  // nothing may be in flight when a bounded wait gave up inside the loop
    }

    ptx::tc_fence_before_sync();
    __syncthreads();
    if (warp == 1) {
        if (sm->abort_flag) __nanosleep(1000000u);  // loads may be in flight: a millisecond, before shared memory is another CTA's
        ptx::tmem_dealloc(tmem, kTmemCols);
    }
}
