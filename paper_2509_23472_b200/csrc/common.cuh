// Internal declarations shared by the translation units of libloract (not part of the C ABI).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/loract.h"

namespace loract {

// ---------------------------------------------------------------- launch accounting
// Called after every kernel launch: counts it and, while a trace is open (test hook), records an event
// behind it on `stream` under the label set with trace_label().
void count_launch(const char* kernel = "", cudaStream_t stream = nullptr);
void trace_label(const char* label);

// The argument rules every entry point shares (include/loract.h, "Conventions"): LORACT_OK or the error.
loract_status_t check_desc(const loract_desc_t* d);

#define LORACT_CUDA_TRY(expr)                          \
  do {                                                 \
    cudaError_t _e = (expr);                           \
    if (_e != cudaSuccess) return _e;                  \
  } while (0)

// ---------------------------------------------------------------- programmatic dependent launch
// The kernels of one call run back to back on one stream.  Launched with programmatic stream
// serialisation, a kernel may start (be scheduled, set up shared memory, barriers, tensor memory) while
// its predecessor is still running; it must then execute pdl_wait() before its first access to global
// memory, which returns once the predecessor has completed and its writes are visible.
#ifdef __CUDACC__
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename Kern, typename... Args>
cudaError_t launch_pdl(Kern kernel, dim3 grid, dim3 block, size_t smem, cudaStream_t stream, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}
#endif

// ---------------------------------------------------------------- generic contraction
// C (M x N) = sum over terms of  A_t (M x K) * B_t (K x N), fp32 (or fp64) accumulation.
// Operands are row-major arrays; a_mn / b_mn say which index is contiguous in memory:
//   a_mn == false : A stored as [M][K]  (K-major)      a_mn == true : A stored as [K][M]  (M-major)
//   b_mn == false : B stored as [N][K]  (K-major)      b_mn == true : B stored as [K][N]  (N-major)
// Several terms share shapes and leading dimensions; they exist for split-precision products
// (x = hi + lo in bf16: hi*hi + hi*lo + lo*hi).
enum OutMode : int {
  OUT_F32 = 0,    // C0: float
  OUT_BF16 = 1,   // C0: bf16
  OUT_SPLIT = 2,  // C0: bf16 hi, C1: bf16 lo  (hi = bf16(x), lo = bf16(x - hi))
  OUT_F64 = 3,    // C0: double (SIMT path only)
  // C0: bf16, C0[m][n] = row_a[m] * col[n] * E[m][n] - row_b[m] / col[n] * acc[m][n]  (tensor-core path only):
  // the input gradient of the RMS pre-norm unit from a reconstructed tile that is never stored
  OUT_RMS_BWD = 4,
  // C0: bf16, C0[m][n] = E[m][n] * f'(acc[m][n]), f = SiLU (ep_kind 0) or GELU (ep_kind 1)  (tensor-core path
  // only): the input gradient of an element-wise activation from a reconstructed tile that is never stored
  OUT_ACT_BWD = 5
};

enum ElemType : int { ELEM_F32 = 0, ELEM_BF16 = 1, ELEM_F64 = 2 };

struct GemmTerm {
  const void* A;
  const void* B;
};

struct GemmDesc {
  int M = 0, N = 0, K = 0;
  bool a_mn = false, b_mn = false;
  int64_t lda = 0, ldb = 0;  // leading dimension (elements) of the stored arrays
  int a_type = ELEM_BF16, b_type = ELEM_BF16;
  int n_terms = 1;
  GemmTerm terms[4];
  int out = OUT_F32;
  void* C0 = nullptr;
  void* C1 = nullptr;
  int64_t ldc = 0;
  // split over K: split s handles a contiguous K range and writes C0 + s * split_stride (fp32/f64 out)
  int splits = 1;
  int64_t split_stride = 0;
  bool acc64 = false;      // SIMT path: accumulate in double
  bool lower_only = false; // SIMT path, fp32 operands: the caller reads the lower triangle only (32 x 32 tiles above it may be left out)
  bool one_sum = false;    // SIMT path, fp32 operands and result: every output is one running sum over K, in order
  bool accumulate = false; // SIMT path, OUT_F32, splits == 1: C += result
  float alpha = 1.0f;      // SIMT path: C = alpha * sum
  // OUT_RMS_BWD: E (bf16, M x N, leading dimension ep_ld), per-row and per-column coefficients
  const void* ep_E = nullptr;
  int64_t ep_ld = 0;
  const float* ep_row_a = nullptr;
  const float* ep_row_b = nullptr;
  const void* ep_col = nullptr;
  int ep_kind = 0;         // OUT_ACT_BWD: which activation
  // Two-CTA kernel, K-major A: loads of A from this K element on ask L2 to evict them last (a later kernel
  // reads the same bytes again); negative: no hint.
  int64_t a_keep_from_k = -1;
  // The sum of the terms before this one is multiplied by 1/2 before this term's products are added
  // (result = (t_0 + ... + t_{h-1}) / 2 + t_h + ...); 0 or negative: plain sum.  With the pair {A^T A, A^T B} and
  // h = 1 the result D gives D + D^T = A^T A + A^T B + B^T A: a symmetric three-term sum for two terms' work.
  int halve_at_term = 0;
  // What a kernel may read ahead of its own griddepcontrol.wait (here: the gate word and early operands).  A launch without a gate, or
  // with one that is not zero, releases its dependents behind its wait; a gated launch that leaves releases them first and waits
  // then.  So a grid starts once the last kernel of the stream that was not such a launch, K, has passed its wait, and that is once
  // everything ahead of K is complete and visible.  Whatever was written AHEAD OF K may be read early; what K itself wrote may not, even
  // where gated launches stand between K and the reader.  Two launches back is enough only if the launch in between has no gate.
  // (sample_indices_kernel releases first, too; a call whose products load early has a kernel of its own in between.)  Every kernel
  // waits before it ends, so the completion of one implies that of all earlier ones.
  //
  // Tensor-core path: a device word, written ahead of the last kernel without a gate in front of the row of gated launches that read
  // it; when it is zero the launch does nothing (no loads, no products, C untouched).  nullptr: unconditional.
  const uint32_t* gate = nullptr;
  // Tensor-core path: the launch stores zero into the status word before any of its waits can set a bit in it (the
  // first kernel of a call clears the word itself instead of a memset in front of it).
  bool clear_status = false;
  uint32_t* clear_word = nullptr;   // SIMT path: the same, the word to clear
  // Tensor-core path: every A (every B) of the terms was written ahead of the previous kernel of the stream (behind a row of gated
  // launches: ahead of the last kernel in front of the row), so it may be loaded before this grid's own wait, under the
  // predecessor's work (see the rule at `gate`).  Not for a launch with a gate.  OUT_RMS_BWD: both flags together speak for A, B and ep_E.
  bool a_early = false, b_early = false;
  // Tensor-core path: the K-major factor (B where both are K-major, A otherwise) is lower triangular, element (i, k) zero for
  // k > i, and its zeros may be left out: the forms with two accumulators skip the first one's K blocks beyond its rows.
  // (512 columns, a quarter of the work; traced, with an event behind every kernel: application of L^-T to 32768 / 16384 rows 55.3 ->
  // 49.2 / 30.8 -> 26.7 us, test matrix of 512 x 11008 22.4 -> 20.4.)
  bool lower = false;
  // Tensor-core path, both operands K-major, N <= 512: one CTA pair must own whole rows of the product (it has read its rows
  // of A before it stores them, so C may be A); see gemm_tc_can_own_rows.
  bool whole_rows = false;
  // Tensor-core path, OUT_SPLIT: a device word written by an earlier kernel; when it is zero only C0 (the leading bf16
  // part) is written and C1 keeps its old contents.
  const uint32_t* lo_gate = nullptr;
};

// tcgen05 engine: bf16 operands, fp32 accumulation in tensor memory.  Returns cudaErrorNotSupported
// for shapes it does not take (the caller then uses the SIMT kernel).
bool gemm_tc_supported(const GemmDesc& g);
cudaError_t gemm_tc_launch(const GemmDesc& g, uint32_t* dev_status, cudaStream_t stream);
// free_sums: so many partial sums cost nothing to add up (the kernel behind adds them as it reads).
int gemm_tc_pick_splits(int M, int N, int K, bool a_mn, bool b_mn, int max_splits = 32, int free_sums = 1);
// Splits over K of a product with many rows (M x N, both operands K-major) whose tiles do not fill the chip.
int gemm_tc_pick_tall_splits(int M, int N, int K);
// Test hook: the form with two accumulators that a launch takes (0: none, 1: two column tiles, 2: two row tiles).
int gemm_tc_wide_form(const GemmDesc& g);
// Whether a launch with whole_rows set can give one CTA (pair) whole rows of an M x N product.
bool gemm_tc_can_own_rows(int M, int N);
void gemm_tc_set_pair_mode(int on);   // test hook: 0 keeps every contraction on the one-CTA kernel
int gemm_tc_tile_width(const GemmDesc& g);      // test hook: columns of a tile (not of the persistent kernel's)
// Test hooks for the give-up path of the bounded waits: a kernel that waits (with the engine's / the cluster
// kernel's own wait) on a barrier nothing completes, for at most limit_ns, then sets LORACT_DEV_WAIT_EXPIRED.
cudaError_t gemm_tc_wait_probe_launch(uint32_t* dev_status, uint64_t limit_ns, cudaStream_t stream);
cudaError_t small_block_cluster_wait_probe_launch(uint32_t* dev_status, uint64_t limit_ns, cudaStream_t stream);

// W (l x l fp32, both triangles) = (Yh + Yl)^T (Yh + Yl) of a tall bf16 pair (n x l, row-major without padding), 256 < l <= 512
// (units == 0: not taken), with every product and short accumulation chains.  `partials` holds gemm_tc_gram_bytes.
struct GramPlan {
  int tiles = 0, s_diag = 0, s_off = 0, units = 0;
};
GramPlan gemm_tc_gram_plan(int n, int l);
size_t gemm_tc_gram_bytes(const GramPlan& p);
cudaError_t gemm_tc_gram_launch(const void* Yh, const void* Yl, int n, int l, const GramPlan& plan, float* partials, float* W,
                                uint32_t* dev_status, const uint32_t* gate, cudaStream_t stream);

// Plain CUDA-core kernel for any shape and type (fp32 path, small or odd shapes).
cudaError_t gemm_simt_launch(const GemmDesc& g, cudaStream_t stream);

// ---------------------------------------------------------------- sampler and gather
cudaError_t sample_indices_launch(uint64_t seed, uint64_t call_id, uint32_t n_rows, int rank, int32_t* idx_dev,
                                  uint32_t* dev_status, cudaStream_t stream);
// The first kernel of a call: draws the indices (to idx_out if not null), sets the status word, and gathers
// dst (rank x d, stride d) = rows idx of the whole matrix, of which src (stride ld) holds [row0, row0 + n_local); rows that
// live elsewhere are written as zeros.  16-byte loads, elem_bytes 2 or 4.
cudaError_t sample_gather_launch(uint64_t seed, uint64_t call_id, uint32_t n_rows, int rank, int32_t* idx_out,
                                 uint32_t* dev_status, const void* src, int64_t ld, int64_t d, int elem_bytes, int64_t row0,
                                 int64_t n_local, void* dst, cudaStream_t stream);
// Gaussian test matrix for the RSVD comparator: dst (l x d bf16, row-major) with
// dst[c][j] = z(j * l + c), z the Philox + Box-Muller stream (counter word 1 = 1).
cudaError_t gaussian_rows_launch(uint64_t seed, uint64_t call_id, int l, int64_t d,
                                 __nv_bfloat16* dst, cudaStream_t stream);

// ---------------------------------------------------------------- small-block factorisation
// From the symmetric positive semi-definite r x r matrix  W = sum_s P_s  (P_s fp32 or fp64, row-major,
// stride r, consecutive partials `partial_stride` elements apart) computes the inverse of the
// Cholesky factor of  W + shift_rel * mean(diag W) * I :  Linv = L^{-1} (lower triangular), so that
// (Y Linv^T) has orthonormal columns when W = Y^T Y.  Outputs (any may be null): Linv as an fp32 or
// fp64 matrix, and as a bf16 hi/lo pair.  `scratch` holds r*r + 1024*ceil(r/32) doubles, apart from the partials.
struct SmallBlockArgs {
  int r = 0;
  const void* partials = nullptr;
  int partial_type = ELEM_F32;
  int n_partials = 1;
  int64_t partial_stride = 0;
  bool use_f64 = false;  // fp64 arithmetic asked for (it is also used where the shared-memory kernel does not apply)
  void* scratch = nullptr;
  float shift_rel = 0.f;
  // each diagonal entry is also multiplied by (1 + shift_diag_rel), a shift relative to the entry itself (the scale-invariant form, which leaves a
  // matrix whose diagonal spans several orders of magnitude as well conditioned as its scaled form)
  float shift_diag_rel = 0.f;
  // device word (written as GemmDesc::gate says); zero: the launch does nothing.  nullptr: unconditional.
  const uint32_t* gate = nullptr;
  // optional, three words: the decision after the first orthonormalisation round whether a second one is needed, W being the
  // Gram matrix that is factored.  With D = diag(W)^(-1/2) the kernel forms
  //   est = sum_ij (L^-1)_ij^2 W_jj = trace((D W D)^-1)   (W_jj as factored),
  // which lies between 1 / lambda_min and r / lambda_min of the diagonally scaled Gram matrix, the quantity that
  // multiplies the rounding error of W in the orthogonality defect of Y L^-T.  gate_out[0] = 1 if est > gate_threshold, est
  // is not finite, or the status word is non-zero (a clamped pivot, a non-finite input), else 0; gate_out[1] = est (float
  // bits); gate_out[2] = rounds that will run (1 or 2).  Fixed summation order.
  uint32_t* gate_out = nullptr;
  float gate_threshold = 0.f;
  // test hook, up to 256 columns: so many bytes of the shares of the estimate are waited for and never sent
  uint32_t absent_share_bytes = 0;
  void* linv_full = nullptr;  // fp64, r x r
  float* linv_f32 = nullptr;  // fp32 copy, r x r
  __nv_bfloat16* linv_hi = nullptr;
  __nv_bfloat16* linv_lo = nullptr;
  uint32_t* dev_status = nullptr;
  // row strides (elements) of the partial matrices and of the outputs; 0 means r
  int64_t in_ld = 0, out_ld = 0;
};
cudaError_t small_block_launch(const SmallBlockArgs& a, cudaStream_t stream);
// The same computation for r <= 512 in fp32 from fp32 partials, or r <= 192 in fp64 from fp64 partials, entirely in the
// shared memory of a cluster of up to sixteen CTAs (no scratch).  small_block_launch uses it whenever it applies and the
// device can hold such a cluster; the general kernel otherwise.
bool small_block_cluster_supported(const SmallBlockArgs& a);
bool small_block_cluster_resident(const SmallBlockArgs& a);
void small_block_set_big_clusters(int on);   // test hook: 0 treats clusters of sixteen CTAs as not resident
cudaError_t small_block_cluster_launch(const SmallBlockArgs& a, cudaStream_t stream);

// ---------------------------------------------------------------- elementwise helpers
// out = sum_s partials[s] (fixed order), written as fp32 and/or bf16.
cudaError_t reduce_partials_launch(const float* partials, int n_partials, int64_t stride,
                                   int64_t count, float* out_f32, __nv_bfloat16* out_bf16,
                                   cudaStream_t stream, const uint32_t* gate = nullptr);
// hi + lo = sum_s partials[s] (fixed order) as a bf16 pair; count a multiple of 4, everything 16-byte aligned.
cudaError_t reduce_pair_launch(const float* partials, int n_partials, int64_t stride, int64_t count, __nv_bfloat16* hi,
                               __nv_bfloat16* lo, cudaStream_t stream);
// out (r x r) = S + S^T, S the fixed-order sum of the partials (each r x r, leading dimension r).
// gate (optional): device word; zero means the launch does nothing.
cudaError_t reduce_sym_launch(const float* partials, int n_partials, int64_t stride, int r, float* out,
                              cudaStream_t stream, const uint32_t* gate = nullptr);
// dst = src (count bf16 elements, both 16-byte aligned, count a multiple of 8) when *gate != 0; nothing otherwise.
cudaError_t copy_bf16_gated_launch(const __nv_bfloat16* src, __nv_bfloat16* dst, int64_t count, const uint32_t* gate,
                                   cudaStream_t stream);
// out = sum_s partials[s] as a bf16 triple hi + mid + lo (rows x cols, leading dimensions ld_in / ld_out).
cudaError_t reduce_split3_launch(const float* partials, int n_partials, int64_t stride, int rows, int cols,
                                 int64_t ld_in, int64_t ld_out, __nv_bfloat16* hi, __nv_bfloat16* mid,
                                 __nv_bfloat16* lo, cudaStream_t stream);
// dW (d x g, fp32) = V^T T (+ dW), V r x d, T (r x g) the sum of n_partials matrices stored one behind the other: where
// small_dw_supported says so.
bool small_dw_supported(int r, int g, int n_partials);
cudaError_t small_dw_launch(const void* V, int elem_type, int64_t d, int r, int g, const float* partials, int n_partials,
                            float* dW, int accumulate, cudaStream_t stream);
// Section 3.3 backward, row coefficients: inner_i = (1 / d) sum_k U[i][k] P[i][k] (P = grad_A V^T, fp32, n x r, the sum of n_partials
// matrices p_stride elements apart, leading dimension ldp, both multiples of four),
// row_a[i] = rstd[i], row_b[i] = rstd[i] * inner_i.  One warp per row.
cudaError_t rms_backward_rows_launch(const __nv_bfloat16* U, const float* P, int64_t ldp, int n_partials, int64_t p_stride,
                                     const float* rstd, int64_t n, int r, int64_t d, float* row_a, float* row_b, cudaStream_t stream);
// Section 3.3 forward: A = Norm(X); per-row rstd (and mean for LayerNorm).  One warp per row.
cudaError_t norm_forward_launch(const void* X, int64_t n, int64_t d, int64_t ldx, int elem_type,
                                const void* gamma, const void* beta, float eps, int kind, void* A,
                                int64_t lda, float* rstd, float* mean, cudaStream_t stream);

}  // namespace loract
