// Tensor-core (tcgen05 / TMA) kernels of the library: interface used by the C ABI.
#pragma once

#include <cuda.h>

#include "common.cuh"

// Whether the tensor-core kernels cover this layer / cache combination.
bool lorc_tc_decode_supported(const lorc_ctx* ctx, const LorcLayer& L, const CacheView& cv);
bool lorc_tc_append_supported(const lorc_ctx* ctx, const LorcLayer& L, const CacheView& cv, int T);

// Scratch bytes the tensor-core decode path wants for (batch, max_seq_len), any layer; with less than that, down to the least it
// works with, the context shares are limited to those of one cluster.
size_t lorc_tc_workspace_bytes(const lorc_ctx* ctx, int batch, int max_seq_len);
size_t lorc_tc_workspace_least(const lorc_ctx* ctx, int batch, int max_seq_len);

// latent_out: `out` receives the normalised latent output [b, H_q, r_v] instead of the up-projected one.
// pos0, q_pos / ml_out: context shards (see lorc_decode_attn_shard): per sequence the position of the first cached row
// and of the query, and where to leave (reference, denominator) [b, H_q, 2] of the softmax over this shard.
cudaError_t lorc_tc_decode(lorc_ctx* ctx, int layer, const LorcLayer& L, const CacheView& cv,
                           const bf16* q, bf16* out, int n_splits, void* ws, size_t ws_bytes,
                           cudaStream_t st, int* launches, bool latent_out = false, const int32_t* pos0 = nullptr,
                           const int32_t* q_pos = nullptr, float* ml_out = nullptr);
cudaError_t lorc_tc_append(lorc_ctx* ctx, int layer, const LorcLayer& L, const CacheView& cv,
                           const bf16* x, int T, cudaStream_t st, int* launches);
// Cache write of compressed layers as a tcgen05 GEMM (tc_append.cu), for prompt-sized launches.
bool lorc_tc_append_gemm_supported(const lorc_ctx* ctx, const LorcLayer& L, const CacheView& cv, int T);
cudaError_t lorc_tc_append_gemm(lorc_ctx* ctx, const LorcLayer& L, const CacheView& cv, const bf16* x, int T,
                                cudaStream_t st, int* launches);

// Contexts with interleaved rotary pairs keep fp32-level precision on the tensor-core decode path: softmax numerators and
// the normalised latent output are carried as two bf16 parts (value rounded, remainder rounded: together 16 significant
// bits).  The plain kernels, which serve what does not fit this path, keep both in fp32; against fp64 the results are off
// by 1.6e-3 either way (the bf16 output), with one bf16 part by 2.9e-3.
inline bool lorc_tc_split(const lorc_ctx* ctx) { return ctx->desc.rope_style == LORC_ROPE_INTERLEAVED; }
// Rows of a sequence that exist: such contexts leave tokens past the capacity, and those whose page lies outside the pool, out
// of the attention (and report them), as the plain kernels do.
inline int lorc_tc_max_rows(const CacheView& cv) { return cv.capacity < INT32_MAX ? (int)cv.capacity : INT32_MAX; }
// Whether a call may take that path now: its tables exist, or may be allocated (the stream is not being captured).
bool lorc_tc_tables_ready(const lorc_ctx* ctx, const CacheView& cv, cudaStream_t st);

// Bytes of one probability tile image (128 tokens of one sequence, all query heads): the bf16 numerators as the PV
// kernel's swizzled MMA operand (split: the rows of the remainders behind those of the rounded values, in every chunk),
// then float m[4][H_q] and float l[4][H_q] (reference and sum per 32-token quarter).
__host__ __device__ inline int lorc_tc_image_bytes(int n_q_heads, bool split) {
    return 2 * n_q_heads * (split ? 2 : 1) * 64 * 2 + 8 * n_q_heads * 4;
}

// Score kernel (tc_score.cu): key reconstruction, rotation, q.k and the softmax numerators; writes one tile image per
// 128 tokens into pimg [b, tiles, image] and raises the row maxima (integers, as order-preserving keys).  rope_tile:
// the in-tile rotation table (33 x 32 float4, lorc_tc_rope_tile_fill).
#define LORC_SCORE_MAX_BATCH 64      // sequences per launch (larger batches take several launches)
cudaError_t lorc_tc_score_set_attrs();
cudaError_t lorc_tc_rope_tile_fill(float2* table, double theta, cudaStream_t st);
cudaError_t lorc_tc_score_launch(lorc_ctx* ctx, const LorcLayer& L, const CacheView& cv, const CUtensorMap& mapCK,
                                 const CUtensorMap& mapBKT, const bf16* q, uint8_t* pimg, unsigned* rowmax,
                                 const float4* rope_tile, int tiles, const int32_t* pos0, const int32_t* q_pos, cudaStream_t st,
                                 int* launches);

// Score kernel of layers without rotation (tc_absorbed.cu): the key up-projection is absorbed into the query
// (q~ = B_K q, written to `qabs`, lorc_tc_absorbed_scratch_bytes of scratch), the scores are a skinny GEMM over the
// latent keys.  Same outputs as lorc_tc_score_launch.
size_t lorc_tc_absorbed_scratch_bytes(const lorc_ctx* ctx, int batch);
cudaError_t lorc_tc_absorbed_set_attrs();
cudaError_t lorc_tc_score_absorbed_launch(lorc_ctx* ctx, const LorcLayer& L, const CacheView& cv, const CUtensorMap& mapCK,
                                          const bf16* q, bf16* qabs, uint8_t* pimg, unsigned* rowmax, int tiles,
                                          cudaStream_t st, int* launches);

// P.C_V and value up-projection (tc_pv.cu).  mapCV: C_V cache in 64-column x 128-row (or page-sized) swizzled boxes;
// mapBVT: B_V^T [n, r_v] in swizzled boxes of 64 latent columns x 32 rows.  The plan says how a launch splits the
// work: column blocks and context shares of each.  The up-projection kernel writes `out` and leaves the row maxima empty again.
// `arrived` (LORC_PV_MAX_CLUSTER words per sequence and column block) is zero before a launch and after it.
#define LORC_PV_MAX_CLUSTER 16       // the largest cluster that a GPU may take
struct LorcPvPlan {
    int n_blk, n_csplit, cluster, n_clusters;        // n_csplit shares of a block in n_clusters clusters of `cluster` blocks
    size_t off_part;
    bool fits;
};
size_t lorc_tc_pv_scratch_least(const lorc_ctx* ctx, int batch);      // without room for shares in several clusters
size_t lorc_tc_pv_scratch_bytes(const lorc_ctx* ctx, int batch, int max_seq_len);
cudaError_t lorc_tc_pv_set_attrs(const lorc_ctx* ctx);
void lorc_tc_pv_plan(lorc_ctx* ctx, const LorcLayer& L, const CacheView& cv, int n_splits_hint, size_t scratch_bytes,
                     LorcPvPlan* plan);
cudaError_t lorc_tc_pv_launch(lorc_ctx* ctx, const LorcLayer& L, const CacheView& cv, const CUtensorMap& mapCV,
                              const CUtensorMap& mapBVT, const uint8_t* pimg, unsigned* rowmax, unsigned* arrived, int tiles,
                              const LorcPvPlan& plan, void* scratch, bf16* out, bool latent_out, const int32_t* pos0,
                              const int32_t* q_pos, float* ml_out, cudaStream_t st, int* launches);

// Prompt processing (tc_prefill.cu): attention of the T newest tokens of every sequence (q, out [b, T, H_q, 128]) over
// the latent cache, causal inside the chunk.  Keys and values are reconstructed once into `scratch`
// (lorc_tc_prefill_scratch_bytes), then a flash-attention kernel runs over them.  mapBKT, mapBVT: B_K^T, B_V^T [n, r] in
// swizzled boxes of 64 latent columns x 128 rows [0] and 64 rows [1].
bool lorc_tc_prefill_shape_ok(const lorc_ctx* ctx);
bool lorc_tc_prefill_supported(const lorc_ctx* ctx, const LorcLayer& L, const CacheView& cv);
size_t lorc_tc_prefill_scratch_bytes(const lorc_ctx* ctx, int batch, int max_seq_len, int T);
cudaError_t lorc_tc_prefill_set_attrs();
cudaError_t lorc_tc_prefill_launch(lorc_ctx* ctx, const LorcLayer& L, const CacheView& cv, const CUtensorMap& mapCK,
                                   const CUtensorMap& mapCV, const CUtensorMap* mapBKT, const CUtensorMap* mapBVT,
                                   const bf16* q, bf16* out, int T, void* scratch, cudaStream_t st, int* launches);
cudaError_t lorc_tc_prefill(lorc_ctx* ctx, int layer, const LorcLayer& L, const CacheView& cv, const bf16* q, bf16* out,
                            int T, void* ws, size_t ws_bytes, cudaStream_t st, int* launches);

// A_cat [D, R] (row-major) -> fragment order [R/8][D/32][32 lanes][8] used by the fast append kernel.  The first
// pair_cols columns (uncompressed mode with half-split rotary pairs: the key columns; otherwise 0) are laid out with the
// two members of each rotary pair side by side.
cudaError_t lorc_fast_retile_factor(const bf16* A_cat, bf16* A_tiled, int D, int R, int pair_cols, int d_head,
                                    cudaStream_t st);

// Tensor maps of an uncompressed layer's cache: boxes of 64 columns x box_rows tokens, 128-byte swizzle.  They are kept with
// the layer and encoded again when the cache's pointers or geometry change.
bool lorc_tc_full_maps(lorc_ctx* ctx, const LorcLayer& L, const CacheView& cv, int box_rows, CUtensorMap** mapK, CUtensorMap** mapV);

// Drop cached per-layer state (tensor maps) when factors are reloaded / the context dies.
void lorc_tc_invalidate_layer(lorc_ctx* ctx, int layer);
void lorc_tc_release(lorc_ctx* ctx);

// The pages of one 128-token tile of a sequence, one per lane (lanes at or past 128 / page_size: 0): a warp fetches them
// with one round trip per tile and shuffles them to the lane that issues the boxes.  (Looked up box by box inside the loop
// over the slices of the rank, a table access stood before every copy: a step of 64 ragged sequences of up to 16384
// tokens, r 384, 64-token pages took 659 us and takes 596 us.)  Pages past the end of the sequence, or with a bad table entry, are read from
// page `none`: 0 (their rows are masked, but every box must deliver its bytes), or n_pages, which lies behind the pool and
// reads as zero.
__device__ __forceinline__ int lorc_tile_page(const int32_t* table, long long seq, int tile, int lane, int len, int page_size,
                                              int max_pages, int n_pages, int* status, int none = 0) {
    const int ppt = 128 / page_size, lp = tile * ppt + lane;
    int page = none;
    if (lane < ppt && (long long)lp * page_size < len && lp < max_pages) {
        page = table[seq * max_pages + lp];
        if (page < 0 || page >= n_pages) {
            lorc_set_status(status, LORC_ERR_CAPACITY);
            page = none;
        }
    }
    return page;
}

// Whether the query of a non-empty sequence (a shard, where pos0 and q_pos are given) neither precedes a cached key nor leaves
// the tables; otherwise the sequence is treated as empty.
__device__ __forceinline__ bool lorc_query_ok(const int32_t* pos0, const int32_t* q_pos, int s, int len, int max_pos) {
    return !q_pos || (pos0[s] >= 0 && q_pos[s] < max_pos && q_pos[s] - pos0[s] >= len - 1);
}

// Order-preserving map from finite floats (and infinities) to unsigned integers: a < b  <=>  key(a) < key(b).  No float
// maps to 0, so 0 can stand for "nothing yet" under an atomic maximum.
__device__ __forceinline__ unsigned lorc_float_key(float f) {
    const unsigned b = __float_as_uint(f);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float lorc_key_float(unsigned k) {
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}
