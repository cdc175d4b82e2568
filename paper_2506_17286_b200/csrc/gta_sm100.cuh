// tcgen05 / TMA (sm_100a) prefill path: interface towards the API layer.
#pragma once

#include "gta_common.cuh"

namespace gta {

// True when the tensor-core kernels cover this shape (bf16, d_h = 64 or 128, d_l % 128 == 0, ...).
bool sm100_prefill_supported(const Dims& d, int dtype);

// Enqueues the tensor-core prefill (attention kernel + decoder kernel) on `stream`.
gta_status_t launch_sm100_prefill(const Dims& d, const void* q, const void* k, const void* c, const void* x,
                                  const void* w_p, const void* w_g, void* out, void* workspace, size_t workspace_bytes,
                                  int32_t* status_word, cudaStream_t stream, int stages, int* launches,
                                  const PageMap& pm = PageMap());

// Attention kernel alone: L[B, n_q, N, d_l] (bf16) = Softmax(scale Q K^T) C per attention map; bf16, d_h = 64 or
// 128, d_l a multiple of 128 or exactly 64.  With a page map, k and c are paged pools (page_size a multiple of 16)
// and token t of sequence b is looked up through the block table.  part: scratch with which the key tiles of a call of few
// items are split over the chip (and merged by a second kernel), into as many units as it holds; nullptr: no split.
// Over pages that are not whole blocks of 64 tokens, L is two bf16 planes [2][B, n_q, N, d_l] (their sum).
size_t sm100_split_workspace_bytes(const Dims& d);     // L (behind which the scratch begins) and the scratch of any split
gta_status_t launch_sm100_attention(const Dims& d, const void* q, const void* k, const void* c, void* l_out,
                                    int32_t* status_word, cudaStream_t stream, int* launches, PageMap pm = PageMap(),
                                    float* part = nullptr, size_t part_bytes = 0);

// Test hooks of the attention kernels' bounded waits (see gta_debug_attention_wait in gta.h).
gta_status_t sm100_attention_debug_wait(unsigned long long limit_ns, int withhold_first_arrive);
gta_status_t short_prefill_debug_wait(unsigned long long limit_ns, int withhold_first_arrive);
gta_status_t sm100_attention_f32_debug_wait(unsigned long long limit_ns, int withhold_first_arrive);
gta_status_t sm100_decoder_f32_debug_wait(unsigned long long limit_ns, int withhold_first_arrive);

// Decoder + gate kernel alone: out = (L W_P) (.) sigmoid(X W_G) with L[B, n_q, N, d_l] in bf16.
// step_lens (optional; the fused append + decode step): lengths that the kernel advances by one, where there is room
// below step_cap, once the kernel before it in the stream is complete.  release: the kernel behind this one may be scheduled
// from then on; behind: this one may overlap the kernel ahead, whose own inputs are then older than its X and W_G.
gta_status_t launch_sm100_decoder(const Dims& d, const void* l_bf16, const void* x, const void* w_p, const void* w_g,
                                  void* out, int32_t* status_word, cudaStream_t stream, int32_t* step_lens = nullptr,
                                  int step_batch = 0, int step_cap = 0, bool release = true, bool behind = true);
// The same for an L in two bf16 planes [2][B, n_q, N, d_l] whose sum it is; the gates are kept in fp32.
gta_status_t launch_sm100_decoder_fine(const Dims& d, const void* l_planes, const void* x, const void* w_p, const void* w_g,
                                       void* out, int32_t* status_word, cudaStream_t stream, bool release = true,
                                       bool behind = true);

// The fp32 kernels below take an operand as three bf16 pieces.  bf16 ends at 2^-133, so an element below 2^-110 loses what it has
// below that: at most 2^-133.  Where the largest element of its row (or column of the weights) is no smaller than this, that is
// 2^-43 of it and less than the sums over the row round; rows and columns of smaller ones are done again with FMAs.
constexpr float kPiecesFloor = 0x1p-90f;

// Attention of an fp32 call on the tensor cores (gta_sm100_f32_attention.cu): d_h = 64, d_l a multiple of 128, contiguous K and
// C; L fp32 [n_q, B, N, d_l]; scratch of the given size (256-byte aligned) for the pieces of K and C; split: CTAs (1, 2 or
// 4) that share the keys of a row tile.
bool sm100_attention_f32_shape(const Dims& d);           // whatever the batch and the lengths
bool sm100_attention_f32_supported(const Dims& d);
size_t sm100_attention_f32_scratch(const Dims& d);
cudaError_t launch_sm100_attention_f32(const Dims& d, const float* q, const float* k, const float* c, float* o_lat, void* scratch,
                                       int32_t* status_word, cudaStream_t stream, int split, int* launches);

// Decoder + gate of an fp32 call on the tensor cores (gta_sm100_f32_decoder.cu): L fp32 [n_q, B, N, d_l]; d_h a multiple of 64;
// nt: columns of an item (256 or 128), whose number is the other function's result.
long long sm100_decoder_f32_units(const Dims& d, int nt);
cudaError_t launch_sm100_decoder_f32(const Dims& d, const float* o_lat, const float* x, const float* w_p, const float* w_g,
                                     float* out, int32_t* status_word, cudaStream_t stream, bool behind, int nt);

// Linear maps of the attention layer around the operator (App. B.1.1), bf16 with fp32 accumulation.
// True when the tcgen05 kernel covers the layer's projections for this shape.
bool sm100_linear_supported(const Dims& d, int dtype);

// [Q | K | C] = X W_qkc for the B x N tokens of a chunk that starts at position pos0: RoPE on q and k,
// q to q_out [B, n_q, N, d_h], k and c to rows pos0 + t of the caches [B, groups, S_cap, width] (with a page map:
// of the paged pools, S_cap then being page_size * max_pages).
// rope_table: sm100_rope_table_bytes(d) bytes of scratch (cos / sin of the chunk's positions).
size_t sm100_rope_table_bytes(const Dims& d);
gta_status_t launch_sm100_project(const Dims& d, int pos0, int S_cap, double rope_base, const void* x,
                                  const void* w_qkc, void* q_out, void* k_cache, void* c_cache, void* rope_table,
                                  int32_t* status_word, cudaStream_t stream, const PageMap& pm = PageMap());

// One decode step of the same projection: one new token per sequence at position seq_lens[b] (RoPE there,
// k and c to that cache row, q to q_out [B, n_q, d_h]), then seq_lens[b] += 1; a sequence whose cache is full
// is skipped and raises GTA_ERR_CACHE_FULL.  With a page map, k_cache / c_cache are the paged pools.  prep: sm100_decode_prep_bytes(d) bytes of scratch.
size_t sm100_decode_prep_bytes(const Dims& d);
gta_status_t launch_sm100_project_step(const Dims& d, int S_cap, double rope_base, const void* x_t, const void* w_qkc,
                                       void* q_out, void* k_cache, void* c_cache, int32_t* seq_lens, void* prep,
                                       int32_t* status_word, cudaStream_t stream, const PageMap& pm = PageMap());

// C[M, n_cols] = A[M, K] W[K, n_cols], row-major.
gta_status_t launch_sm100_matmul(long long M, int K, int n_cols, const void* a, const void* w, void* c_out,
                                 int32_t* status_word, cudaStream_t stream);

// The stream kernel of a decode step over 8-bit caches on the tcgen05 tensor pipe (gta_decode_fp8_tc.cu): same
// schedule (G CTAs, sub-tiles of T tokens) and partial results as decode_stream_fp8_kernel.
bool decode_fp8_tc_supported(const Dims& d, int T);
cudaError_t launch_decode_fp8_tc_stream(const Dims& d, int G, int T, int S_cap, const void* q, const void* k_codes,
                                        const void* c_codes, const float* k_scale, const float* c_scale,
                                        const int32_t* seq_lens, float* part_o, float* part_ml, int32_t* status_word,
                                        cudaStream_t stream);

// The stream kernel of a decode step over bf16 caches on the tcgen05 tensor pipe (gta_decode_tc.cu): same schedule
// (G CTAs, sub-tiles of T tokens), step lengths and partial results as decode_stream_kernel; k_new / c_new != nullptr:
// the fused append + decode step.
bool decode_tc_supported(const Dims& d, int T, int occ, int page_size);
cudaError_t launch_decode_tc_stream(const Dims& d, int G, int T, int S_cap, const void* q, const void* k_cache,
                                    const void* c_cache, const int32_t* seq_lens, float* part_o, float* part_ml,
                                    int32_t* status_word, cudaStream_t stream, const void* k_new, const void* c_new,
                                    const PageMap& pm);

// Test hooks of the bounded waits of the two tensor-memory decode stream kernels (see gta_debug_decode_wait in gta.h).
gta_status_t decode_tc_debug_wait(unsigned long long limit_ns, int withhold_first_arrive);
gta_status_t decode_fp8_tc_debug_wait(unsigned long long limit_ns, int withhold_first_arrive);

}  // namespace gta
