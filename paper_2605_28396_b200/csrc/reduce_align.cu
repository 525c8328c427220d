// Per-sequence / per-batch reductions over the [B,T] per-token scalars.
//
// adwin_window_reduce: the loss on the prefix window that the synchronous update uses.
// adwin_probe_align:   the prefix-versus-full alignment audit on a returned probe batch: in logit
//   space the prefix gradient is the full gradient with rows t >= L zeroed, so
//   rho(L) = sqrt(Q(L)/Q_full) with Q = sums of per-token squared gradient norms;
//   SNR = rho^2/(1-rho^2); admissible when rho >= rho_star; L_next = shortest admissible length.
// All sums are float64 in a fixed order (strided per thread, then a fixed tree), so results are
// bitwise reproducible.
//
// These kernels touch O(B*T) floats: latency and launches are all they cost.  Up to kFusedSeqs
// sequences one cluster of CTAs does the whole reduction in one launch (its CTAs take the sequences
// in turn, meet at the cluster barrier, and CTA 0 sums over the batch); larger batches take one
// launch over the sequences and one over the batch, which uses more than one cluster's SMs.  A
// sequence is read once for all its prefix lengths (up to kSlots at a time).
#include "adwin_common.cuh"
#include "adwin_internal.h"

namespace adwin {
namespace {

constexpr int kRedThreads = 512;
constexpr int kRedWarps = kRedThreads / 32;
constexpr int kSlots = 8;          // prefix lengths summed in one pass over a sequence
constexpr int kFusedSeqs = 64;
constexpr int kFusedCtas = 8;

__device__ __forceinline__ int effective_len(const int32_t* rollout_len, int64_t b, int64_t T) {
  int64_t r = rollout_len ? rollout_len[b] : T;
  r = r < 0 ? 0 : (r > T ? T : r);
  return (int)r;
}

// Sums of (gsq, kl, logratio) over t < n[j] of sequence b for NS prefix lengths; out[j][0..2] is valid
// in thread 3j..3j+2 as its return value (other threads: unspecified).
template <int NS>
__device__ __forceinline__ double prefix_sums(const float* kl, const float* c, const float* gsq,
                                              int64_t b, int64_t T, const int (&n)[NS],
                                              double (*sm)[3 * NS]) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int most = 0;
#pragma unroll
  for (int j = 0; j < NS; ++j) most = n[j] > most ? n[j] : most;
  double v[NS][3];
#pragma unroll
  for (int j = 0; j < NS; ++j) v[j][0] = v[j][1] = v[j][2] = 0.0;
#pragma unroll 4
  for (int t = tid; t < most; t += kRedThreads) {
    const int64_t i = b * T + t;
    const double q = gsq ? (double)gsq[i] : 0.0, k = (double)kl[i], r = (double)c[i];
#pragma unroll
    for (int j = 0; j < NS; ++j) {
      if (t < n[j]) {
        v[j][0] += q;
        v[j][1] += k;
        v[j][2] += r;
      }
    }
  }
  __syncthreads();   // the scratch may still be read from the pass before
#pragma unroll
  for (int j = 0; j < NS; ++j)
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      double x = v[j][i];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
      if (lane == 0) sm[warp][j * 3 + i] = x;
    }
  __syncthreads();
  double s = 0.0;
  if (tid < 3 * NS)
    for (int w = 0; w < kRedWarps; ++w) s += sm[w][tid];
  return s;
}

__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::
                   : "memory");
}

// ---------------------------------------------------------------------------- window reduce
struct WindowArgs {
  const float *kl, *c, *gsq;
  const int32_t *window, *rollout_len;
  int64_t B, T;
  double* seq_out;
  double* batch_out;
};

__device__ __forceinline__ void window_seq(const WindowArgs& a, int64_t b, double (*sm)[3]) {
  const int R = effective_len(a.rollout_len, b, a.T);
  const int W = a.window[b] < 0 ? 0 : a.window[b];
  const int E[1] = {W < R ? W : R};
  const double s = prefix_sums<1>(a.kl, a.c, a.gsq, b, a.T, E, sm);
  const int i = threadIdx.x;
  if (i < 3) a.seq_out[b * 4 + (i == 0 ? 2 : i - 1)] = s;   // {kl, logratio, gsq, tokens}
  if (i == 3) a.seq_out[b * 4 + 3] = (double)E[0];
}

// batch_out[i] = sum_b seq_out[b][i], i < 4, sequential in b (one thread per column).
__device__ __forceinline__ void window_batch(const WindowArgs& a) {
  const int i = threadIdx.x;
  if (i < 4) {
    double s = 0.0;
#pragma unroll 8
    for (int64_t b = 0; b < a.B; ++b) s += a.seq_out[b * 4 + i];
    a.batch_out[i] = s;
  }
}

__global__ void __launch_bounds__(kRedThreads) window_reduce_kernel(const WindowArgs a) {
  chain();
  __shared__ double sm[kRedWarps][3];
  for (int64_t b = blockIdx.x; b < a.B; b += gridDim.x) window_seq(a, b, sm);
  __syncthreads();
  cluster_barrier();
  if (blockIdx.x == 0) window_batch(a);
}
__global__ void __launch_bounds__(kRedThreads) window_reduce_seq_kernel(const WindowArgs a) {
  chain();
  __shared__ double sm[kRedWarps][3];
  for (int64_t b = blockIdx.x; b < a.B; b += gridDim.x) window_seq(a, b, sm);
}
__global__ void window_reduce_batch_kernel(const WindowArgs a) { chain(); window_batch(a); }

// ---------------------------------------------------------------------------- alignment audit
__constant__ int32_t kDefaultCandidates[6] = {64, 128, 256, 512, 1024, 2048};

struct AlignArgs {
  const float *kl, *c, *gsq;
  const int32_t *window, *rollout_len;
  int64_t B, T;
  const int32_t* candidates;
  int K;
  double rho_star;
  double *seq_stats, *seq_full, *batch_stats;
  int32_t *L_next, *flags_out;
};

// Length of slot j: a candidate, or (j == K) the training window of sequence b.
__device__ __forceinline__ int slot_len(const AlignArgs& a, int j, int64_t b) {
  const int L = j < a.K ? (a.candidates ? a.candidates[j] : kDefaultCandidates[j]) : a.window[b];
  return L < 0 ? 0 : L;
}

__device__ __forceinline__ void align_seq(const AlignArgs& a, int64_t b, double (*sm)[3 * kSlots],
                                          double* full) {
  const int R = effective_len(a.rollout_len, b, a.T);
  // the rollout first, then the slots, kSlots lengths per pass over the sequence
  for (int j0 = -1; j0 <= a.K; j0 += kSlots) {
    int n[kSlots];
#pragma unroll
    for (int i = 0; i < kSlots; ++i) {
      const int j = j0 + i;
      const int L = j < 0 ? R : (j <= a.K ? slot_len(a, j, b) : 0);
      n[i] = L < R ? L : R;
    }
    const double s = prefix_sums<kSlots>(a.kl, a.c, a.gsq, b, a.T, n, sm);
    const int j = j0 + (int)threadIdx.x / 3, f = threadIdx.x % 3;
    if (j0 < 0 && threadIdx.x == 0) *full = s;
    __syncthreads();
    if (threadIdx.x < 3 * kSlots && j <= a.K) {
      if (j < 0) {
        a.seq_full[b * 3 + f] = s;
      } else {
        double* o = a.seq_stats + ((size_t)b * (a.K + 1) + j) * 4;
        o[f] = s;
        if (f == 0) o[3] = (*full > 0.0) ? sqrt(s / *full) : 1.0;
      }
    }
  }
  __syncthreads();
}

// One thread per slot j: sequential sums over b, then rho / SNR / admissibility; thread 0 picks
// L_next after a barrier.
__device__ __forceinline__ void align_batch(const AlignArgs& a, int* admissible, int* degenerate) {
  const int j = threadIdx.x;
  if (j == 0) *degenerate = 0;
  __syncthreads();
  if (j <= a.K) {
    double qp = 0.0, qf = 0.0, macro = 0.0, ntok = 0.0;
    bool bad = false;
#pragma unroll 4
    for (int64_t b = 0; b < a.B; ++b) {
      const double* o = a.seq_stats + ((size_t)b * (a.K + 1) + j) * 4;
      const double f = a.seq_full[b * 3 + 0];
      qp += o[0];
      qf += f;
      macro += o[3];
      bad |= !(f > 0.0);
      const int R = effective_len(a.rollout_len, b, a.T), L = slot_len(a, j, b);
      ntok += (double)(L < R ? L : R);
    }
    double micro = 1.0;
    if (qf > 0.0) micro = sqrt(qp / qf);
    else bad = true;
    const double r2 = micro * micro;
    double* o = a.batch_stats + j * 5;
    o[0] = micro;
    o[1] = (a.B > 0) ? macro / (double)a.B : 1.0;
    o[2] = (r2 < 1.0) ? r2 / (1.0 - r2) : (double)INFINITY;
    o[3] = (micro >= a.rho_star) ? 1.0 : 0.0;
    o[4] = ntok;
    admissible[j] = (micro >= a.rho_star) ? 1 : 0;
    if (bad) *degenerate = 1;
  }
  __syncthreads();
  if (j == 0) {
    int best = -1, largest = -1;
    for (int i = 0; i < a.K; ++i) {
      const int L = a.candidates ? a.candidates[i] : kDefaultCandidates[i];
      if (L > largest) largest = L;
      if (admissible[i] && (best < 0 || L < best)) best = L;
    }
    int flags = *degenerate ? ADWIN_ALIGN_DEGENERATE : 0;
    if (best < 0) {
      best = largest;
      flags |= ADWIN_ALIGN_NONE_ADMISSIBLE;
    }
    *a.L_next = best;
    *a.flags_out = flags;
  }
}

__global__ void __launch_bounds__(kRedThreads) probe_align_kernel(const AlignArgs a) {
  chain();
  __shared__ double sm[kRedWarps][3 * kSlots];
  __shared__ double full;
  __shared__ int admissible[65], degenerate;
  for (int64_t b = blockIdx.x; b < a.B; b += gridDim.x) align_seq(a, b, sm, &full);
  __syncthreads();
  cluster_barrier();
  if (blockIdx.x == 0) align_batch(a, admissible, &degenerate);
}
__global__ void __launch_bounds__(kRedThreads) probe_align_seq_kernel(const AlignArgs a) {
  chain();
  __shared__ double sm[kRedWarps][3 * kSlots];
  __shared__ double full;
  for (int64_t b = blockIdx.x; b < a.B; b += gridDim.x) align_seq(a, b, sm, &full);
}
__global__ void probe_align_batch_kernel(const AlignArgs a) {
  chain();
  __shared__ int admissible[65], degenerate;
  align_batch(a, admissible, &degenerate);
}

// One launch for up to kFusedSeqs sequences, else one over the sequences and one over the batch.
template <typename Args>
cudaError_t launch_reduction(void (*fused)(Args), void (*seq)(Args), void (*batch)(Args),
                             int batch_threads, const Args& a, cudaStream_t s) {
  if (a.B <= kFusedSeqs) {
    const int ctas = a.B < 1 ? 1 : (int)(a.B < kFusedCtas ? a.B : kFusedCtas);
    return launch_chained(fused, ctas, kRedThreads, 0, ctas, s, a);
  }
  launch_chained(seq, (unsigned)(a.B < 4096 ? a.B : 4096), kRedThreads, 0, 1, s, a);
  launch_chained(batch, 1, batch_threads, 0, 1, s, a);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_window_reduce(const float* kl, const float* logratio, const float* gsq,
                                 const int32_t* window, const int32_t* rollout_len, int64_t B,
                                 int64_t T, double* seq_out, double* batch_out, cudaStream_t s) {
  const WindowArgs a = {kl, logratio, gsq, window, rollout_len, B, T, seq_out, batch_out};
  return launch_reduction(window_reduce_kernel, window_reduce_seq_kernel,
                          window_reduce_batch_kernel, 32, a, s);
}

cudaError_t launch_probe_align(const float* kl, const float* logratio, const float* gsq,
                               const int32_t* window, const int32_t* rollout_len, int64_t B,
                               int64_t T, const int32_t* candidates, int32_t K, double rho_star,
                               double* seq_stats, double* seq_full, double* batch_stats,
                               int32_t* L_next, int32_t* flags_out, cudaStream_t s) {
  const AlignArgs a = {kl, logratio, gsq, window, rollout_len, B, T, candidates, K, rho_star,
                       seq_stats, seq_full, batch_stats, L_next, flags_out};
  return launch_reduction(probe_align_kernel, probe_align_seq_kernel, probe_align_batch_kernel, 96,
                          a, s);
}

}  // namespace adwin
