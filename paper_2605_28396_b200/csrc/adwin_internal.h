// Host-side declarations shared by the translation units of the library (not installed).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/adwin.h"

namespace adwin {

// Launches a kernel of this library: clusters of `cluster` CTAs, and programmatic stream serialization,
// that is, its CTAs may be set up while the kernel before it in the stream drains.  Every kernel
// launched here begins with chain() or chain_wait() (adwin_common.cuh), which wait until that kernel
// has finished and its writes are visible.  A small LM-head update of eleven kernels 207 -> 185 us, an
// update and audit on 12 000 rows of 10 309 entries 143 -> 134, a 195 us update 190.
template <typename... P, typename... A>
cudaError_t launch_chained(void (*kernel)(P...), unsigned grid, int threads, size_t smem, int cluster,
                           cudaStream_t s, const A&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = cluster;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

struct KlParams;

// Time limit of the kernels' handshake waits (consumer / producer / exchange / accumulator
// barriers), 2 s unless the diagnostic entry point shortened it.  The loops that wait for a
// kernel's own copies or MMAs in flight on its way out always keep the 2 s limit.
uint64_t handshake_wait_limit_ns();

// Workspace layout: [0,256) reserved counters; offsets (B+1) int64; range B int32; ewin B int32:
// `total` bytes, the part every call needs.  Optional extension up to `total_ext`: a second
// prefix-sum array over the effective windows, offsets_win (B+1) int64, which lets a call that
// wants scalars over the rollout and the gradient inside the window run as two kernels.
struct WorkspaceLayout {
  size_t off_offsets, off_range, off_ewin, total;
  size_t off_offsets_win, total_ext;
};
WorkspaceLayout workspace_layout(int64_t B);

// Shared body of the forward+backward entry points.  row_coef: null for the plain ones.  plan_rows: the rows of
// the caller's call, of which this may be a part: the row kernel's shape goes by it, so that the
// parts leave the bits that the whole would.
int opd_kl_fwd_bwd_impl(const void* student_logits, const void* teacher_logits, int dtype,
                        int64_t B, int64_t T, int64_t V, int64_t ld, const int32_t* tokens,
                        const int32_t* window, const int32_t* rollout_len, float grad_scale,
                        int grad_mode, int flags, void* grad_student, int grad_dtype,
                        int64_t ld_grad, float* kl, float* logratio, float* gsq,
                        float* lse_student, float* lse_teacher, void* workspace,
                        size_t workspace_bytes, int32_t* dev_status, void* cuda_stream,
                        const float* row_coef, int64_t plan_rows);

cudaError_t launch_rowmap(const int32_t* window, const int32_t* rollout_len, int64_t B, int64_t T,
                          int flags, void* workspace, bool with_window_offsets, float* kl,
                          float* logratio, float* gsq, float* lse_s, float* lse_t, int32_t* status,
                          cudaStream_t s);

cudaError_t launch_zero_tail(const KlParams& p, int grad_dtype, cudaStream_t s);

cudaError_t launch_kl_generic(const KlParams& p, int dtype, int grad_dtype, bool vec, int sm_count,
                              cudaStream_t s);

// Staged cluster kernel.  Returns cudaErrorNotSupported when the shape does not fit its plan
// (the caller then falls back to the generic kernel).  ragged: rows that do not all start and end on
// 16-byte boundaries.
cudaError_t launch_kl_staged(const KlParams& p, int dtype, int grad_dtype, bool ragged, int sm_count,
                             cudaStream_t s);

// Row kernel for calls whose processed rows all get a gradient.  Returns cudaErrorNotSupported when
// the row does not fit its plans.
cudaError_t launch_kl_rows(const KlParams& p, int dtype, int grad_dtype, bool ragged, int sm_count,
                           cudaStream_t s);

cudaError_t launch_window_reduce(const float* kl, const float* logratio, const float* gsq,
                                 const int32_t* window, const int32_t* rollout_len, int64_t B,
                                 int64_t T, double* seq_out, double* batch_out, cudaStream_t s);

cudaError_t launch_probe_align(const float* kl, const float* logratio, const float* gsq,
                               const int32_t* window, const int32_t* rollout_len, int64_t B,
                               int64_t T, const int32_t* candidates, int32_t K, double rho_star,
                               double* seq_stats, double* seq_full, double* batch_stats,
                               int32_t* L_next, int32_t* flags_out, cudaStream_t s);

cudaError_t launch_return_to_go(const float* logratio, const int32_t* window,
                                const int32_t* rollout_len, int64_t B, int64_t T, double gamma,
                                int flags, float* rtg, cudaStream_t s);

cudaError_t launch_teacher_drift(const void* teacher, int dtype, int64_t B, int64_t T, int64_t V,
                                 int64_t ld, const int32_t* tokens, const int32_t* rollout_len,
                                 float* entropy, int32_t* rank, int32_t* status, bool vec,
                                 int sm_count, cudaStream_t s);

cudaError_t launch_drift_curves(const float* entropy, const int32_t* rank,
                                const int32_t* rollout_len, int64_t B, int64_t T,
                                const int32_t* ks, int32_t K, int32_t* worst, double* survival,
                                double* bf_mean, int32_t* n_active, cudaStream_t s);

// Fused LM-head form (lmhead.cu).
size_t lmhead_workspace_bytes(int64_t B, int64_t T, int64_t V, int64_t ds, int64_t dt,
                              int64_t max_rows, bool want_grad);
cudaError_t launch_lmhead(const void* hs, const void* ws, const void* ht, const void* wt, int64_t B,
                          int64_t T, int64_t V, int64_t ds, int64_t dt, const int32_t* tokens,
                          const int32_t* window, const int32_t* rollout_len, float alpha, int mode,
                          int flags, void* dH, int dh_dtype, float* dW, float* kl, float* logratio,
                          float* gsq, float* lse_s, float* lse_t, void* workspace,
                          int64_t max_rows, int32_t* status, int sm_count, cudaStream_t s);
size_t lmhead_align_workspace_bytes(int64_t B, int64_t T, int64_t V, int64_t ds, int64_t dt,
                                    int64_t max_rows, int K);
cudaError_t launch_lmhead_weight_align(const void* hs, const void* ws, const void* ht,
                                       const void* wt, int64_t B, int64_t T, int64_t V, int64_t ds,
                                       int64_t dt, const int32_t* tokens,
                                       const int32_t* rollout_len, const int32_t* cand_host, int K,
                                       double rho_star, int mode, float* kl, float* logratio,
                                       float* gsq, double* batch_stats, int32_t* L_next,
                                       int32_t* flags_out, void* workspace, int64_t max_rows,
                                       int32_t* status, int sm_count, cudaStream_t s);
// Tensor-core GEMM (tc_gemm.cu): C[M,N] = A B, bf16 in.  A is [M,K] (K contiguous, a_mn = false) or
// [K,M] (M contiguous, a_mn = true), B is [K,N].  scratch: tc_gemm_scratch_bytes() for split tiles,
// or null; pace: a zeroed counter of this launch's own, or null.
size_t tc_gemm_scratch_bytes();
cudaError_t launch_tc_gemm(const void* A, int64_t lda, bool a_mn, const void* B, int64_t ldb,
                           int64_t M, int64_t N, int64_t K, void* C, int64_t ldc, bool c_bf16,
                           const int32_t* m_tiles_dev, const int32_t* k_tiles_dev,
                           const int32_t* row_map, float* scratch, unsigned int* pace,
                           int32_t* status, int sm_count, cudaStream_t s);
// n_bins products C_i = A^T B over consecutive ranges of the contraction (A [K,M], B [K,N]):
// bin i takes the 64-row blocks [kblock_dev[i], kblock_dev[i+1]) and writes C + i * bin_stride.
cudaError_t launch_tc_gemm_bins(const void* A, int64_t lda, const void* B, int64_t ldb, int64_t M,
                                int64_t N, int64_t K, float* C, int64_t ldc, int64_t bin_stride,
                                int n_bins, const int32_t* kblock_dev, int32_t* status,
                                int sm_count, cudaStream_t s);

}  // namespace adwin
