// Declarations shared by the operand preparation (quantize_qkv.cu) and the fused forward (attention_fwd.cu):
// the job descriptions of the quantiser and the tables a packed variable-length batch hands to the kernels.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "efq_common.cuh"

namespace efq {

// Launches a kernel that may start while the one before it in the stream still runs (its blocks set up meanwhile); what it
// needs of the work before it waits for itself with griddepcontrol.wait.  Takes about 2 microseconds off a call of two
// kernels back to back.
template <typename... Params, typename... Args>
inline cudaError_t launch_overlapped(void (*kernel)(Params...), dim3 grid, int threads, size_t smem, cudaStream_t stream, const Args&... args)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(static_cast<unsigned>(threads));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// One operand of one sequence for the quantiser.  Rows of Q and K are quantised along d (blocks of 32), V along
// the keys (blocks of 32 aligned to the sequence's own key index, per channel) and written transposed.
struct QuantSeg {
    const __nv_bfloat16* src;  // element (head, row, c) at src[head * head_stride + row * row_stride + c]
    int64_t heads;             // heads of the code matrix: query (or KV) heads; KV heads for a packed Q
    int64_t S;                 // valid rows per head (tokens; pack_G * pack_lq rows for a packed Q)
    int64_t S_pad;             // rows per head in the code matrix, a multiple of 128
    int64_t head_stride, row_stride;   // of the source, in elements
    int32_t pack_lq, pack_G;   // Q only; pack_G > 1: row r of KV head h is token r % pack_lq of query head h * pack_G + r / pack_lq
    uint8_t* codes;            // Q, K: [heads * S_pad, 64 B] from here on; V: see v_row_bytes
    uint8_t* sf;               // scale tiles: Q, K one 512-byte tile per 128 rows from here on; V: see v_sf_tile0
    int64_t v_row_bytes;       // V only: bytes of one row (channel) of the transposed code matrix [heads * 128, v_row_bytes]
    int64_t v_x0;              // V only: byte offset of this sequence's first key inside a row
    int64_t v_sf_tiles_per_head, v_sf_tile0;   // V only: tile of (head, 128-key tile t) = head * per_head + tile0 + t
};

enum QuantKind : int32_t { kQuantRows = 0, kQuantV = 1 };

struct QuantJob {
    QuantSeg seg;
    int32_t kind;
    int32_t pad;
};

// The work items of one query tile of one sequence, one per head that owns it, in the order the fused forward takes them.
// The host lists the tiles (heaviest first); the quantiser's launch spreads them into the item table.
struct ItemGroup {
    int32_t first_item, seq, qt, n_tiles, Sq, Sk, packed;
};
struct ItemDesc;

// SMs of a device, asked for once (0: no such device)
int sm_count(int dev);

// Q, K and V of one [B, H, S, d] problem (or one sequence) in one launch; also clears the 256 status words.
cudaError_t launch_quantize_qkv(const QuantSeg& q, const QuantSeg& k, const QuantSeg& v, uint32_t* status, cudaStream_t stream);
// The jobs of a packed batch in one launch: jobs and first_cta (n_jobs + 1 prefix sums of CTAs) live in device memory.
// places: the item in every place of the table, -1 for an empty place; null: the items one after the other (item_order.h).
// status: the words to clear, null if an earlier launch of the call has cleared them.
cudaError_t launch_quantize_jobs(const QuantJob* jobs, const int32_t* first_cta, int n_jobs, int64_t total_ctas, const ItemGroup* groups,
                                 int n_groups, const int32_t* places, int64_t n_places, ItemDesc* items, uint32_t* status, cudaStream_t stream);
// CTAs a job needs (256 threads each)
int64_t quantize_job_ctas(const QuantJob& job);

// Tensor map of a row-major bf16 matrix, box 64 columns (128 B) x 128 rows, 128-byte swizzle; the last few are kept.
bool encode_bf16_map(CUtensorMap* map, const void* base, uint64_t cols, uint64_t rows);

// One sequence of a packed batch as the fused forward sees it.
struct SeqDesc {
    int64_t Sq, Sk;          // query and key tokens of the sequence
    int64_t o_off;           // element offset of the sequence's first output row in o
    int32_t q_row0;          // first row of the sequence in the Q code matrix (head 0, tile 0)
    int32_t Sq_pad;          // rows per head there
    int32_t k_row0, Sk_pad;  // the same for K
    int32_t k_col0;          // first key of the sequence along the key axis of the V^T code matrix (a multiple of 128)
    int32_t packed;          // 1: the query heads of a KV group share one 128-row query tile (few query tokens)
    int32_t token0, pad;     // its first query token in the batch
};
// One work item of the fused forward over a packed batch.  What every role needs at once stands here, the rest in the sequence
// table: a CTA that goes from item to item has the next one's entry loaded in time.
struct __align__(16) ItemDesc {
    int32_t seq;             // index into the sequence table
    int32_t qt;              // query tile inside the sequence (0 when packed)
    int32_t head;            // query head, or KV head when packed
    int32_t n_tiles;         // KV tiles that it walks; -1: an empty place, the CTA is through
    int32_t Sq, Sk, packed;  // of its sequence
    int32_t pad;
};

// ------------------------------------------------------------------------------------------------
// Few query rows (attention_few.cu): the query rows of a KV group are Hq / Hkv * Sq
// ------------------------------------------------------------------------------------------------
constexpr int kFewMaxRows = 24;
// The contexts that take it, by the sequence's own shape: up to 16 rows all, 17 to 24 rows from 64 KV tiles on.  Its time grows with
// the rows (each has its codes made and its scores written for itself), that of the general path does not up to 128; but the
// general path walks a whole context in one CTA a KV head.  Measured, this path against the general one, us a call among others
// with inputs of its own, 1 / 8 / 64 / 256 KV heads:
//    8 rows:  1000 keys 10.4 / 10.8 / 20.2 / 55 against 12.4 / 12.3 / 17.9 / 43, 2000 keys 10.5 / 11.5 / 28.2 / 79 against 18.0 / 18.7 / 28.2
//             / 79, 4000 keys 10.7 / 14.0 / 43 / 127 against 28.8 / 31.0 / 52 / 147, 8100 keys 11.4 / 19.7 / 70 / 246 against 49 / 56 / 98 / 285
//   16 rows:  1000 keys 11.0 / 11.5 / 23.0 / 58 against 12.5 / 12.6 / 18.1 / 43, 2000 keys 11.8 / 12.4 / 34.9 / 100 against 18.5 / 19.0 / 28.6
//             / 80, 4000 keys 11.7 / 15.1 / 60 / 155 against 29.4 / 31.5 / 52 / 148, 8100 keys 12.3 / 22.8 / 93 / 289 against 51 / 57 / 99 / 287,
//             16000 keys 13.9 / 36.7 / 151 / 549 against 92 / 102 / 185 / 556
//   24 rows:  1000 keys 12.8 / 14.6 / 29.0 / 75 against 12.7 / 12.5 / 18.2 / 44, 2000 keys 13.4 / 15.8 / 45 / 129 against 18.5 / 19.2 / 28.8 / 80,
//             4100 keys 13.6 / 20.0 / 78 / 217 against 30.7 / 32.7 / 54 / 153, 6000 keys 14.1 / 21.3 / 86 / 299 against 40 / 44 / 75 / 216,
//             8100 keys 14.3 / 29.0 / 125 / 387 against 51 / 57 / 100 / 288
// The number of heads and sequences must not matter to the line (a sequence gives the same bits alone and in a batch), so it weighs a few
// contexts against wide batches.  Up to 16 rows the gains of the few outweigh a loss of a fifth to a quarter in wide batches of short
// ones.  At 17 to 24 rows the few gain from 2000 keys on by now, but 64 and more heads lose up to 1.7 times below 32 tiles and 1.4 (128
// heads: 1.6) from there to 63; at 64 tiles, where the few gain 2 to 3.6 times, the wide still lose 1.25 to 1.45.
__host__ __device__ inline bool few_takes(int64_t rows, int64_t n_tiles) { return rows <= 16 || (rows <= kFewMaxRows && n_tiles >= 64); }
// Tiles of a chunk of the KV range, by the sequence's own shape: short contexts are cut finely, so that one of them spreads
// over the chip; with many rows a chunk's partial result (544 bytes a row) has to be small against its 64 KB of K and V a tile.
constexpr int kFewMaxChunk = 8;
__host__ __device__ constexpr int few_chunk_tiles(int n_tiles, int rows)
{
    return rows <= 8 ? (n_tiles < 16 ? 1 : n_tiles < 32 ? 2 : n_tiles < 128 ? 4 : kFewMaxChunk) : n_tiles < 32 ? 2 : kFewMaxChunk;
}
constexpr bool few_chunks_halve()
{
    for (int rows = 1; rows <= kFewMaxRows; ++rows)
        for (int tiles = 1; tiles <= 256; ++tiles)
            if (const int n = few_chunk_tiles(tiles, rows); n > kFewMaxChunk || (n & (n - 1)) != 0) return false;
    return true;
}
static_assert(few_chunks_halve(), "a chunk is taken in halves, quarters and eighths of it: another length would lose tiles");
// Tiles that the longest chunk of a context holds
inline int few_longest_chunk(int n_tiles, int rows) { const int n = few_chunk_tiles(n_tiles, rows); return n < n_tiles ? n : n_tiles; }
// Start of row `row` of the scores of a KV head, n_tiles of 128 keys: 64-bit, since 24 rows pass 2^31 scores from 97.6 million keys
// on.  The product of row and tiles fits 32 bits; kept in those, the offsets of a thread's rows take a register each in the loop
// and not two (9 to 16 rows, 16000 keys: 3 to 5 %).  Block maxima (four a tile) are addressed in 32 bits.
__host__ __device__ constexpr int64_t few_row_offset(int row, int n_tiles) { return static_cast<int64_t>(row * n_tiles) * 128; }
static_assert(few_row_offset(kFewMaxRows - 2, 100000000 / 128) == 2200000000ll, "rows of a long context are addressed in 64 bits");
static_assert(int64_t{kFewMaxRows} * (int64_t{1} << 31) / 32 < int64_t{1} << 31, "block maxima of the longest context");
// A chunk's partial result: the 128 values of a row's O^T take the place of the row's scores of the chunk's first tile, which
// nobody reads any more by then; beside them, per row, four parts of the denominator, the maximum they refer to, three unused.
// Where few chunks are taken tile by tile, every tile leaves that, and the factor of its maximum.  So a KV head needs at most
// rows * (528 + 32) bytes a tile, at 24 rows 13440: less than the 17408 of the MXFP4 copies of K and V, and what fits a workspace
// on the general path fits it here.
constexpr int kFewStatFloats = 8;
constexpr int kFewInlineSeqs = 128;      // sequence tables up to this size travel as kernel parameters

struct FewSeq {
    int32_t Sq, Sk;          // tokens of the sequence
    int32_t q0, k0;          // its first query and key token
    int32_t k_pad0;          // keys of the sequences before it, each padded to 128
    int32_t first_unit;      // chunks times KV heads of the sequences before it
};

struct FewParams {
    const __nv_bfloat16 *q, *k, *v;
    float* o;                                  // strides as q
    int32_t Hkv, G, causal;
    int32_t n_seqs;                            // packed batch: sequences in the table; 0: dense [B, H, S, d]
    int32_t Sq, Sk, Sk_pad, dense_chunks;      // dense only
    int64_t q_seq, q_head, q_row, k_seq, k_head, k_row;    // strides in elements
    int32_t row_cap;                           // query rows the workspace holds per KV head (the most of any sequence)
    int32_t n_units, n_heads;                  // chunks times KV heads, and KV heads, of all sequences
    int32_t longest_chunk;                     // tiles
    int32_t split;                             // a chunk is the work of 2^split blocks (set by launch_few)
    float rescale_threshold;
    ProducerConsts K;
    float *scores, *block_max, *stats;         // workspace
    uint32_t* status;
    int32_t inject_skip_mma;                   // test hook: no MMA is issued, so the first wait for one runs out
    int32_t has_dbg;
    efq_debug_t dbg;
    const FewSeq* seqs;                        // device table; null: inline_seqs
    FewSeq inline_seqs[kFewInlineSeqs];
};

struct FewPlan { size_t scores, block_max, stats, total; };   // offsets from a 1024-byte aligned base
FewPlan plan_few(int64_t keys_padded_all_heads, int rows);
// Clears the status words.
cudaError_t launch_few(int producer, FewParams& P, cudaStream_t stream);

}  // namespace efq
