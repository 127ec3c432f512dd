// Kernel declarations shared by the translation units of libquads.
#pragma once
#include <cuda.h>

#include <algorithm>

#include "common.cuh"

namespace quads {

constexpr int kMaxTopk = 16;
constexpr int kMaxExperts = 256;

// header words written by the scan (device side sizes of the dispatch)
enum { kHdrMTiles = 0, kHdrAssignments = 2, kHdrStatus = 3, kHdrArrivals = 4, kHdrRouteArrivals = 5, kHdrWords = 8 };

constexpr int kAmaxPartsMax = 2048;   // partial maxima left by the first pass of the single-tensor quantizer

// ---- quantize.cu
__global__ void amax_kernel(const uint16_t* x, int64_t rows, int64_t K, int64_t ld, int64_t tensor_stride,
                            uint32_t* amax_bits);
__global__ void fused_quantize_kernel(const uint16_t* x, int64_t rows, int64_t K, int64_t ld, int64_t tensor_stride,
                                      int n_tensors, const float* gs_in, uint32_t* amax_bits, uint32_t* counters,
                                      uint8_t* q, uint8_t* sf, uint16_t* fq, float* gs_out, int sf_tiled,
                                      int64_t sf_tensor_stride, int n_groups, long long wait_cycles,
                                      int extra_arrivals, const uint32_t* amax_parts, int n_amax_parts);
template <bool kClear>
__global__ void amax_partial_kernel(const uint16_t* x, int64_t rows, int64_t K, int64_t ld, uint32_t* partials, uint32_t* zero0, int n0,
                                    uint32_t* zero1, int n1);
// Fake-quant of a batch of tensors through shared-memory rings of bulk copies (one CTA per SM,
// four groups of 7 consumer warps + 1 producer warp, one ring of 14 KB stages per group).
constexpr int kRingThreads = 1024;
constexpr int kRingDepth = 3;
constexpr int kRingHeaderBytes = 1024;
constexpr int kRingChunkBytes = 7 * 32 * 2 * 32;
constexpr int kRingSmemBytes = kRingHeaderBytes + 4 * kRingDepth * kRingChunkBytes;
__global__ void fake_quant_ring_kernel(const uint16_t* x, int64_t nblk, int64_t tensor_stride, int n_tensors,
                                       uint32_t* pair, int per, int lead, int split, uint8_t* q, uint8_t* sf, uint16_t* fq,
                                       float* gs_out, int sf_tiled, int64_t sf_tensor_stride, uint32_t k16,
                                       int kt_count);
__global__ void dequantize_kernel(const uint8_t* q, const uint8_t* sf, const float* gs, int64_t nblk, uint32_t k16,
                                  int kt_count, int sf_tiled, int64_t sf_tensor_stride, uint16_t* out, int32_t* zero);
__global__ void channel_stats_kernel(const uint16_t* x, int T, int H, const float* gs_in, const uint32_t* amax_bits,
                                     int rows_per_cta, float* partials);
constexpr int kScoreSlices = 16;
__global__ void score_reduce_kernel(const float* partials, int n_part, int C, double* slice_sums, unsigned int* counters,
                                    unsigned long long* score_keys);
__global__ void clear_kernel(uint4* p, int n);
__global__ void sel_list_kernel(const uint8_t* mask, int C, int32_t* sel_export);
__global__ void export_residual_kernel(int T, int H, const uint8_t* mask, uint32_t flip, const uint8_t* rq, uint8_t* rq_exp);
constexpr int kSwappedSelectMax = 2048;   // channels the operand-swapped second projection can select among
constexpr int kSelectThreads = 1024;   // one CTA per SM: the CTAs of an SM would only repeat each other's search
template <bool kDoubleKeys>            // site 13: float64 scores; site 2: integer totals
__global__ void select_mask_kernel(uint8_t* codes, int n_rows_fixed, uint32_t flip, const int32_t* header, const int32_t* tile_rows,
                                   const unsigned long long* score_keys, int C, int n_sel, uint8_t* mask_out /* or NULL */);
__global__ void combine_kernel(const uint16_t* y_pad, const int32_t* pos_pad, const float* wts, int T, int H,
                               int topk, uint16_t* out, float* out_f32);
__global__ void export_site2_kernel(int A, const int32_t* n_rows_ptr, int I, const int32_t* perm, const int32_t* pos_pad,
                                    const uint8_t* hq_pad, const uint8_t* hsf_tiled, const uint8_t* r2q_pad,
                                    const uint8_t* r2sf_tiled, const uint8_t* mask2, uint8_t* hq, uint8_t* hsf,
                                    uint8_t* r2q, uint8_t* r2sf);

__global__ void mismatch_norms_kernel(const uint16_t* a, const uint16_t* b, int64_t n, double* partials,
                                      unsigned int* counter, double* out);

// ---- front.cu
constexpr int kQuantRowsPerSm = 4;    // resident CTAs of the front kernels
struct QuantRowsArgs {
  const uint16_t* x;
  int T, H, with_residual, sf_tiled;
  const float* gs_in;                 // per-tensor scale, or NULL: amax-derived, ...
  const uint32_t* amax_parts;         // ... from n_amax_parts partial maxima of the preceding kernel, or (NULL) by the CTAs themselves
  int n_amax_parts;
  uint32_t* amax_bits;                // out; zero on entry where the CTAs derive it
  unsigned int* arrivals;             // zero on entry
  int32_t* status;
  float* gs_store;                    // exports, each may be NULL
  uint8_t *xq, *xsf, *rq, *rsf;
  uint8_t *xq_exp, *xsf_exp, *rsf_exp;
  float* partials;                    // [quant_partial_floats(T, H)] scratch of the channel scores
  unsigned int* col_arrivals;         // [kQuantColsMax] zero on entry
  unsigned long long* keys;           // [H] out: channel scores, bit patterns of non-negative float64 values
  int bw, n_col, rows_per_cta;        // filled in at launch
};
constexpr int kQuantCtasMax = 1024;   // CTAs of the quantization role, each with at most 512 channels of a row range ...
constexpr int kQuantColsMax = 128;    // ... in so many column groups (H <= 16384), of at least eight rows but the last
inline size_t quant_partial_floats(int T, int H) { return std::min<size_t>((size_t)kQuantCtasMax * 512, ((size_t)T + 7) / 8 * H); }
// Top-k routing and dispatch order (routing.cuh).
constexpr int kRouteCtasMax = 256;
struct RouteArgs {
  const float* logits;
  int T, E, topk, renormalize, e_lo, e_hi;
  int slot_rows, tile_group;          // valid rows of a 128-row tile at most; tiles per expert are a multiple of tile_group
  int32_t* ids;
  float* wts;
  int32_t* counts;                    // [kRouteCtasMax][E], zero on entry
  unsigned int* arrivals;             // zero on entry
  int32_t* status;
  int32_t *offsets, *tile_prefix, *tile_expert, *tile_rows, *header, *perm, *pos_pad, *row_token;
  int32_t* ids_out;                   // exports, each may be NULL
  float* wts_out;
  int32_t *offsets_out, *perm_out;
};
quads_status launch_front(const QuantRowsArgs& q, const RouteArgs& r, int sm_count, cudaStream_t st);
quads_status launch_quant_rows(const QuantRowsArgs& q, int sm_count, cudaStream_t st);
constexpr int kDispatchThreads = 512, kDispatchPerSm = 3;
struct DispatchArgs {
  int H, n_sel;                       // n_sel == 0: no residual
  const unsigned long long* keys;     // [H] channel scores (QuantRowsArgs::keys)
  uint8_t* mask;                      // [H] out: 1 for the selected channels
  const int32_t *header, *tile_rows, *row_token;
  const uint8_t *xq, *xsf, *rq, *rsf; // token order, linear scales
  uint8_t *xq_pad, *xsf_tiled, *rq_pad, *rsf_tiled;
};
quads_status launch_dispatch(const DispatchArgs& p, int m_tiles_max, int sm_count, cudaStream_t st);

// ---- small_batch.cu: the front of a call with few tokens, two kernels of one cluster each
constexpr int kSmallThreads = 1024;
constexpr int kSmallRouteMaxTokens = 512;
constexpr int kSmallMaxUnits = 16;    // units of 128 channels a CTA of the front kernel takes (H <= 16384 on 8 CTAs)
struct SmallRouteArgs {
  const float* logits;
  int T, E, topk, renormalize, e_lo, e_hi;
  int slot_rows;                      // valid rows of a 128-row tile at most
  float* wts;
  int32_t *offsets, *tile_prefix, *tile_expert, *tile_rows, *header, *perm, *pos_pad, *row_token;
  unsigned long long* zero_u64;       // n_zero words cleared for the kernels that follow
  int n_zero;
  int32_t* ids_out;                   // exports, each may be NULL
  float* wts_out;
  int32_t *offsets_out, *perm_out;
};
struct SmallFrontArgs {
  const uint16_t* x;
  int T, H, topk, n_sel;
  const float* gs_in;                 // per-tensor scale, or NULL: amax-derived (the bits go to amax_bits)
  int after_routing;                  // launched behind route_small_kernel (else it is the call's first kernel)
  int token_order;                    // outputs in token order, scales [T, H/16]; else dispatched copies, tiled scales
  const int32_t* pos_pad;             // [T * topk] dispatched rows, or NULL: row t is token t (topk = 1)
  uint8_t *xq_pad, *xsf, *rq_pad, *rsf;
  uint32_t* amax_bits;
  int32_t* header;                    // its status word is cleared when there is no routing kernel to do it
  float* gs_store;                    // exports, each may be NULL
  uint8_t *mask_out, *xq_exp, *xsf_exp, *rq_exp, *rsf_exp;
};
bool route_small_fits(int T);
bool front_small_fits(int T, int H, bool token_order);
quads_status launch_route_small(const SmallRouteArgs& a, cudaStream_t st);
quads_status launch_front_small(const SmallFrontArgs& a, cudaStream_t st);

// ---- gemm.cu
constexpr int kGemmKSteps = 4;                        // K = 64 MMAs per pipeline stage
constexpr int kGemmStageKBytes = 32 * kGemmKSteps;    // packed FP4 bytes per operand row per stage
enum { kEpiStore = 0, kEpiSwiGLU = 1, kEpiCombine = 2 };

struct GemmParams {
  int K;                 // contraction length in elements (multiple of 64)
  int n_tiles_n;         // tiles along the output-feature dimension
  int n_out;             // output features (I for SwiGLU, else N)
  int b_rows_per_expert; // weight rows per expert
  int half1_row_offset;  // weight-row distance from the tile's first half to its second half
  int has_resid;         // 1: also accumulate the (negated, masked) residual operand
  int dense_rows;        // > 0: one weight and this many activation rows in token order, no routing tables
  int tables_late;       // the preceding kernel wrote the routing tables (operand-swapped first projection)
  int n_experts;         // entries of b_gs (the experts whose weights this call holds)
  int expert_lo;         // global id of the first of them: weights / scales are indexed by (expert - expert_lo)
  const int32_t* header;
  const int32_t* tile_expert;
  const int32_t* tile_rows;
  const uint8_t* a_sf;   // tiled scales of the main activation operand (padded dispatch rows)
  const uint8_t* r_sf;   // tiled scales of the residual operand
  const uint8_t* b_sf;   // tiled weight scales, one block per expert
  size_t b_sf_expert_stride;
  const float* b_gs;     // [E] per-tensor weight scales
  const float* a_gs;     // per-tensor activation scale (pointer), or NULL ...
  const uint32_t* a_amax_bits;  // ... then derived from this amax word
  // epilogue: store / combine
  const int32_t* row_token;    // operand-swapped first projection: token of a padded dispatch row, and the scales of
  const uint8_t* xsf_tok;      // its activation / residual operands in token order, [tokens, K/16]
  const uint8_t* rsf_tok;
  uint16_t* out_bf16;    // kEpiStore: [dense_rows, n_out]
  uint16_t* y_pad;       // kEpiCombine: bf16 [padded dispatch rows, n_out], one row per assignment
  // kEpiCombine with a residual, operand-swapped: the kernel selects the n_sel of K channels with the largest totals
  // and masks the residual rows it loads (sel_keys == NULL: they are masked already)
  const unsigned long long* sel_keys;
  int n_sel;
  uint8_t* mask_out;     // export, may be NULL
  // epilogue: SwiGLU + requantize (site 2)
  const float* h_gs;     // per-tensor scale of h
  int resid2;            // 1: also emit the residual of h and its column statistics
  uint8_t* hq_pad; uint8_t* hsf_tiled; uint8_t* r2q_pad; uint8_t* r2sf_tiled;
  // column scores of the residual of h (Eq. channel-score), accumulated as integers so that the sum does
  // not depend on the order of arrival: every partial sum of squares (one per tile, lane quadrant and
  // column) is divided by the square of h's per-tensor scale, multiplied by 2^score_bits, rounded down
  // and added with a 64-bit integer reduction; the totals are the selection's order-preserving keys
  unsigned long long* keys2;   // [n_out], zero on entry
  int score_bits;
  uint16_t* h_export;    // optional bf16 [A, n_out] in dispatch order
  const int32_t* tile_prefix;
  const int32_t* offsets;
  int32_t* status;       // device status word (QUADS_ERR_TIMEOUT on a failed wait)
};

// Tensor maps of one GEMM launch: packed codes of the activation / residual / weight operands and
// (CTA-pair variant only) their scale atoms viewed as [atoms, 128 x u32].
struct GemmMaps {
  CUtensorMap a, r, b, sfa, sfr, sfb;
};

// Operand-swapped variant for few rows per expert (weights on the M side, tokens in chunks of 32
// on the N side; epi = kEpiSwiGLU or kEpiCombine).  Maps: a / r = activation / residual codes -- of
// the tokens, with boxes of one row, for the first projection, which gathers its rows; of the padded
// dispatch rows, with boxes of 16 rows, for the second -- b = weight codes with boxes of 128 rows;
// p.n_tiles_n counts tiles of 128 output features.  Usable when assignments <= 32 * experts and the slot tables fit.
bool gemm_swapped_ok(int64_t assignments, int n_experts, int m_tiles_max);
quads_status launch_gemm_swapped(int epi, const GemmParams& p, const GemmMaps& m, int n_sms, cudaStream_t stream);

// ---- gemm_dense.cu: dense projection with few output tiles, K split over clusters
bool gemm_dense_ok(int rows, int K, int N, int n_sms);
bool gemm_dense_ahead_of_pairs(int rows, int K, int N, bool resid, int n_sms);
quads_status launch_gemm_dense(const GemmParams& p, const GemmMaps& m, int n_sms, cudaStream_t stream);

// ---- gemm_bf16.cu: out[T, N] = A[T, K] B[N, K]^T, bf16 operands (tensor maps with boxes of 64 elements x kBf16BoxRows
// rows, 128-byte swizzle), float32 accumulation, bf16 output; K % 64 == 0, N % 128 == 0
constexpr int kBf16BoxRows = 64;
// a_early / b_early: the operand is older than the preceding kernel of the stream, which has itself waited for its predecessor
// and has cleared the status word.  Neither: the product is the call's first kernel and clears the word.
quads_status launch_gemm_bf16(const CUtensorMap& tm_a, const CUtensorMap& tm_b, int T, int N, int K, bool a_early, bool b_early, uint16_t* out,
                              int32_t* status, int n_sms, cudaStream_t stream);

// ---- fp8.cu: the FP8 W8A8 comparison path
constexpr int kFp8FewRows = 64;   // rows of a 128-row tile at most in the few-rows form
struct Fp8GemmParams {
  int K;                 // contraction length in elements (multiple of 128)
  int n_tiles_n;         // tiles along the output features
  int n_out;             // output features (I for SwiGLU, else H)
  int b_rows_per_expert;
  int half1_row_offset;
  const int32_t* header;
  const int32_t* tile_expert;
  const int32_t* tile_rows;
  const uint8_t* a_sf;   // activation scale atoms, [m_tiles, K/128, 512]
  const uint8_t* b_sf;   // weight scale atoms, [E, rows/128, K/128, 512]
  size_t b_sf_expert_stride;
  const int32_t* row_token;    // few-rows first projection: token of a padded row, scale bytes in token order [T, K/128]
  const uint8_t* xe_tok;
  int tables_late;             // few rows: the preceding kernel wrote the routing tables
  uint16_t* y_pad;       // kEpiCombine: bf16 [padded rows, n_out]
  uint8_t* hq_pad;       // kEpiSwiGLU: E4M3 codes of h, [padded rows, n_out]
  uint8_t* hsf_atoms;    // kEpiSwiGLU: scale atoms of h, [m_tiles, n_out/128, 512]
  uint16_t* h_export;    // optional bf16 [A, n_out], dispatch order (then hq_export / hexp_export too)
  uint8_t* hq_export;
  uint8_t* hexp_export;
  const int32_t* tile_prefix;
  const int32_t* offsets;
  int32_t* status;
};
quads_status launch_fp8_quantize_act(const uint16_t* x, int64_t rows, int K, uint8_t* codes, uint8_t* exps, int sm_count, cudaStream_t st);
quads_status launch_fp8_front(const uint16_t* x, int64_t rows, int K, uint8_t* codes, uint8_t* exps, const RouteArgs& r, int sm_count,
                              cudaStream_t st);
__global__ void fp8_quantize_weight_kernel(const uint16_t* w, int N, int K, uint8_t* codes, uint8_t* exps, uint8_t* atoms);
__global__ void fp8_dispatch_kernel(int H, const int32_t* header, const int32_t* tile_rows, const int32_t* row_token,
                                    const uint8_t* xq, const uint8_t* xe, uint8_t* xq_pad, uint8_t* xsf_atoms);
quads_status launch_gemm_fp8(int epi, bool few_rows, const Fp8GemmParams& p, const CUtensorMap& tm_a, const CUtensorMap& tm_b, int n_sms,
                             cudaStream_t stream);

quads_status launch_gemm(int epi, int cta_group, const GemmParams& p, const GemmMaps& m, int n_sms,
                         cudaStream_t stream);

}  // namespace quads
