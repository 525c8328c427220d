// Row kernel for calls with gradient: a row (or a cluster's slice of it) is read from HBM once, kept on
// chip between the two sweeps, several CTAs per SM.
//
// Two to eight small CTAs share an SM, each on a row of its own, so that one CTA's exchange and
// row scalars overlap the other CTAs' streaming.  There are no roles and no hand-shakes: every
// thread loads its own 16-byte pieces with plain coalesced loads, folds them into its sums and
// puts them where only it will look for them again -- shared memory, or the otherwise idle tensor
// memory (tcgen05.st / tcgen05.ld) -- so between the sweeps the threads only exchange sums.  One more
// warp does what is done once per row: it adds up the threads' sums, derives the row's scalars and
// hands them back (the others would otherwise each spend ~300 issue slots on it, as much as a
// tenth of a row of 32 000 entries) and fetches the coming rows' metadata.  The next row is brought
// into L2 meanwhile (cp.async.bulk.prefetch.L2), so that HBM stays busy during both sweeps and the
// loads of the first sweep come from L2.
//
// Exponentials are taken against a reference that the whole row shares (the logit of the sampled
// token), so partial sums add without rescaling.  If the sums overflow it (a sampled token more than
// ~69 nats below the row maximum) the row is summed once more, from its on-chip copy, against
// running maxima.  Rows too long for one CTA are split over a cluster; the CTAs' sums then go to every
// CTA of the cluster.
#include <mutex>
#include <type_traits>

#include "adwin_common.cuh"
#include "adwin_internal.h"
#include "kl_pairs.cuh"
#include "tc_pipeline.cuh"

namespace adwin {
namespace {

constexpr int kRowsThreads = 352;     // threads of a CTA that hold pieces, at most
constexpr int kRowsRegs = 80;         // registers per thread: 819 threads on an SM
constexpr int kU = 2;                 // piece pairs in flight per thread
constexpr int kRowsMaxCl = 4;
constexpr float kSumLimit = 1.2676506e30f;   // 2^100: beyond it the shared reference is unsafe
constexpr int kMetaDepth = 4;

struct RowsPlan {
  int cl;             // CTAs per row
  int nt;             // threads per CTA that hold pieces (one more warp looks ahead)
  int ctas;           // CTAs per SM
  int per_rank;       // 16-byte pieces of a slice (per array)
  int steps;          // piece pairs per thread, rounded up to a multiple of kU
  int tm_steps;       // of these, in tensor memory (a multiple of kU; the first ones)
  int tm_cols;        // tensor-memory columns per CTA (0: none)
  int num_clusters;
};

struct __align__(16) RowsMeta {
  int64_t r;
  int y;
  float w;            // caller-supplied row coefficient (0 when there is none)
  float zy, uy;
};

// What sweep 2 needs of a row.
struct __align__(16) RowsScalars {
  float m2s, coef, c0, gy;
  int again;          // the sums overflowed: sum the row once more against running maxima
};

struct __align__(16) RowsCtrl {
  float safe[kRowsThreads / 32][8];    // the warps' records of the running-maximum pass
  float xrec[2][kRowsMaxCl][4];    // per row parity, one record per CTA of the cluster
  float xsafe[kRowsMaxCl][8];
  RowsScalars out;
  RowsMeta meta[kMetaDepth];
  uint32_t tmem_base;
};
// Shared memory: RowsCtrl, a float4 record per thread (its S, A, St of the row and q of the row
// before), then the threads' pieces.
constexpr int kRowsRec = (int)((sizeof(RowsCtrl) + 127) / 128 * 128);
__host__ __device__ constexpr int rows_ctrl_bytes(int nt) { return kRowsRec + nt * 16; }

// Named barriers of a CTA: the threads with pieces report on kPosted and wait on kReady.
constexpr int kPosted = 1, kReady = 2;
__device__ __forceinline__ void named_sync(int id, int threads) {
  asm volatile("barrier.cta.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void named_arrive(int id, int threads) {
  asm volatile("barrier.cta.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

__device__ __forceinline__ void prefetch_l2(const void* p, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// NT: threads that hold pieces, a template constant so that the strides between a thread's pieces are
// offsets in the instructions.  A group of kU steps in which every thread has a piece takes the path
// without tests (FULL below).
template <typename TIn, typename TOut, int NT, bool TM, bool RAG>
__global__ void __launch_bounds__(NT + 32, 65536 / kRowsRegs / (NT + 32))
kl_rows_kernel(const KlParams p, const RowsPlan plan) {
  chain();
  constexpr int N = Elem<TIn>::N;
  constexpr int NP = Pairs<TIn>::NP;
  constexpr int nt = NT, nw = NT / 32, all = NT + 32;
  constexpr uint32_t array = NT * 16u;
  extern __shared__ __align__(128) char smem[];
  RowsCtrl& ctrl = *reinterpret_cast<RowsCtrl*>(smem);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int cl = plan.cl;
  float4* rec = reinterpret_cast<float4*>(smem + kRowsRec);
  char* stash = smem + rows_ctrl_bytes(NT) + tid * 16;   // [step][array][thread] 16 bytes
#ifdef ADWIN_CHECKED
  uint32_t smem_bytes;
  asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(smem_bytes));
  // a group's pieces from `at` on, and its columns of tensor memory (the same for a whole warp)
  auto stash_ok = [&](const char* at) { return at + (2 * kU - 1) * array + 16 <= smem + smem_bytes; };
  auto columns_ok = [&](int k0) {
    return k0 + kU <= plan.tm_steps && ((tid >> 7) + 1) * plan.tm_steps * 8 <= plan.tm_cols;
  };
#endif
  const uint32_t rank = cl > 1 ? cluster_rank() : 0u;
  const int64_t cluster_id = blockIdx.x / cl;
  const int piece0 = (int)rank * plan.per_rank;
  const int64_t total_rows = p.offsets[p.B];
  const int64_t my_rows =
      cluster_id < total_rows ? (total_rows - cluster_id + plan.num_clusters - 1) / plan.num_clusters : 0;

  if (TM && warp == nw) tm_alloc(smem_u32(&ctrl.tmem_base), (uint32_t)plan.tm_cols);

  // where row r lies in this CTA's slice (base pointers are 16-byte aligned)
  auto span_of = [&](int64_t r) -> RowSpan {
    RowSpan a = {0, 0, -1, -1, N};
    if (RAG) a.shift = (int)((r * p.ld) & (N - 1));
    const int64_t end = a.shift + p.V, total = (end + N - 1) / N, left = total - piece0;
    a.pieces = (int)(left < 0 ? 0 : (left > plan.per_rank ? plan.per_rank : left));
    if (RAG) {
      a.first = (a.shift > 0 && piece0 == 0) ? 0 : -1;
      a.last_n = (int)(end - (total - 1) * N);
      a.last = (a.last_n < N && left > 0 && left <= plan.per_rank) ? (int)left - 1 : -1;
    }
    return a;
  };

  // The next row is brought into L2 ahead of its first sweep: bf16 rows by the row's warp, all at once
  // when the second sweep of this row begins; fp32 rows, which memory bounds and not arithmetic, by
  // thread 0 of the others, one array's part of a group at each group of either sweep, so that HBM has an
  // even load (fp32 V = 32 000: 200 us before, 193 so; bf16, where thread 0's extra work holds its CTA
  // up: 194 us against 202).
  constexpr bool kSpread = sizeof(TIn) == 4;
  auto prefetch = [&](int64_t r, const void* base, int from, int count) {
    const RowSpan sn = span_of(r);
    const int n = min(sn.pieces - from, count);
    if (n > 0 && ADWIN_CHK(((int64_t)piece0 + from + n - (RAG ? 1 : 0)) * N <= p.V + sn.shift, p.status))
      prefetch_l2(static_cast<const char*>(base) +
                      ((size_t)r * p.ld - sn.shift + (size_t)(piece0 + from) * N) * sizeof(TIn),
                  (uint32_t)n * 16u);
  };

  if (TM) asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  if (cl > 1) cluster_sync_all();   // peers run before anything is stored into them
  __syncthreads();
  if (TM) asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const int64_t iters = my_rows > 0 ? my_rows + 1 : 0;   // + one exchange for the last norm
  if (warp == nw) {
    // ------------------------------------------------------------------ the row's own warp
    RowCursor cur;
    cur.init(p);
    bool wg_unused;
    auto fetch = [&](int64_t i) {   // metadata of row i into its slot
      const int64_t r = cur.locate(p, cluster_id + i * plan.num_clusters, wg_unused);
      if (lane == 0 && ADWIN_CHK(r >= 0 && r < p.B * p.T, p.status)) {
        RowsMeta& m = ctrl.meta[i % kMetaDepth];
        const int y = p.tokens[r];
        m.r = r;
        m.y = y;
        fetch_logits_at<TIn>(p, r, y, m.zy, m.uy);
        m.w = p.row_coef ? p.row_coef[r] : 0.f;
      }
    };
    constexpr int kAheadRows = kSpread ? 2 : 1;
    for (int64_t i = 0; i < kAheadRows && i < my_rows; ++i) fetch(i);
    __syncthreads();
    int64_t r_prev = 0;
    for (int64_t i = 0; i < iters; ++i) {
      const bool real = i < my_rows, more = i + 1 < my_rows;
      const int par = (int)(i & 1);
      if (i + kAheadRows < my_rows) fetch(i + kAheadRows);
      named_sync(kPosted, all);
      // fixed-order sums over the threads, then over the CTAs
      float v[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int w = 0; w < nw; ++w) {
        const float4 x = rec[w * 32 + lane];
        v[0] += x.x; v[1] += x.y; v[2] += x.z; v[3] += x.w;
      }
#pragma unroll
      for (int f = 0; f < 4; ++f) v[f] = lane_sum(v[f]);
      if (cl > 1) {
        if (lane < cl && ADWIN_CHK(rank < (uint32_t)kRowsMaxCl, p.status))
          remote_store4(map_to_rank(smem_u32(ctrl.xrec[par][rank]), (uint32_t)lane), v[0], v[1], v[2], v[3]);
        cluster_sync_all();
        v[0] = v[1] = v[2] = v[3] = 0.f;
        for (int j = 0; j < cl; ++j) {
          const float4 x = *reinterpret_cast<const float4*>(ctrl.xrec[par][j]);
          v[0] += x.x; v[1] += x.y; v[2] += x.z; v[3] += x.w;
        }
      }
      if (rank == 0 && lane == 0 && i > 0 && p.gsq) p.gsq[r_prev] = v[3];
      if (!real) break;
      const RowsMeta& m = ctrl.meta[i % kMetaDepth];
      const int64_t ri = m.r;
      RowTotals t;
      t.M2s = m.zy * kLog2e;
      t.M2t = m.uy * kLog2e;
      t.S = v[0];
      t.A = v[1];
      t.St = v[2];
      t.B0 = t.B1 = t.B2 = 0.f;
      // (the totals are identical in every CTA of the cluster, so this branch is too)
      if (!(t.S < kSumLimit) || !(t.St < kSumLimit)) {
        if (lane == 0) ctrl.out.again = 1;
        named_sync(kReady, all);
        named_sync(kPosted, all);
        float x[5] = {-INFINITY, -INFINITY, 0.f, 0.f, 0.f};   // m2s, m2t, S, A, St of the CTA
        if (lane < nw) {
#pragma unroll
          for (int f = 0; f < 5; ++f) x[f] = ctrl.safe[lane][f];
        }
        auto combine = [&]() {
          t.M2s = warp_max(x[0]);
          t.M2t = warp_max(x[1]);
          const float gs = (x[0] == -INFINITY) ? 0.f : ex2f(x[0] - t.M2s);
          const float gt = (x[1] == -INFINITY) ? 0.f : ex2f(x[1] - t.M2t);
          t.S = lane_sum(x[2] * gs);
          t.A = lane_sum(x[3] * gs);
          t.St = lane_sum(x[4] * gt);
        };
        combine();
        if (cl > 1) {
          if (lane < cl && ADWIN_CHK(rank < (uint32_t)kRowsMaxCl, p.status)) {
            const uint32_t dst = map_to_rank(smem_u32(ctrl.xsafe[rank]), (uint32_t)lane);
            remote_store4(dst, t.M2s, t.M2t, t.S, t.A);
            remote_store4(dst + 16, t.St, 0.f, 0.f, 0.f);
          }
          cluster_sync_all();
          x[0] = x[1] = -INFINITY;
          x[2] = x[3] = x[4] = 0.f;
          if (lane < cl) {
#pragma unroll
            for (int f = 0; f < 5; ++f) x[f] = ctrl.xsafe[lane][f];
          }
          combine();
        }
      }
      const bool y_valid = m.y >= 0 && (int64_t)m.y < p.V;
      const RowScalars rs = finish_row(t, m.zy, m.uy, y_valid, 0.f, p.alpha, p.mode,
                                       p.row_coef ? &m.w : nullptr);
      if (lane == 0) {
        ctrl.out.m2s = t.M2s;
        ctrl.out.coef = rs.coef;
        ctrl.out.c0 = rs.c0;
        ctrl.out.gy = rs.gy;
        ctrl.out.again = 0;
      }
      named_sync(kReady, all);
      if (lane == 0) {
        if (!kSpread && more) {
          prefetch(ctrl.meta[(i + 1) % kMetaDepth].r, p.student, 0, plan.per_rank);
          prefetch(ctrl.meta[(i + 1) % kMetaDepth].r, p.teacher, 0, plan.per_rank);
        }
        if (rank == 0 && ADWIN_CHK(ri >= 0 && ri < p.B * p.T, p.status)) {
          p.kl[ri] = rs.kl;
          p.logratio[ri] = rs.c;
          if (p.lse_s) p.lse_s[ri] = rs.lse_s;
          if (p.lse_t) p.lse_t[ri] = rs.lse_t;
          int bits = 0;
          if (!y_valid) bits |= ADWIN_DEV_TOKEN_RANGE;
          if (rs.nonfinite) bits |= ADWIN_DEV_NONFINITE;
          if (bits) atomicOr(p.status, bits);
        }
      }
      __syncwarp();
      r_prev = ri;
    }
  } else {
    __syncthreads();   // the first row's metadata
    // this thread's tensor-memory columns: its lane, the columns split between the warps of a lane group
    const uint32_t tm_lane = TM ? ctrl.tmem_base + ((uint32_t)((warp & 3) * 32) << 16) +
                                      (uint32_t)((warp >> 2) * plan.tm_steps * 8)
                                : 0u;
    const bool full_mode = (p.mode == ADWIN_GRAD_FULL_KL);
    float q_prev = 0.f;       // this thread's share of the previous row's squared norm
    for (int64_t i = 0; i < iters; ++i) {
      const bool real = i < my_rows;
      const RowsMeta& m = ctrl.meta[real ? i % kMetaDepth : 0];
      const bool ahead = kSpread && tid == 0 && i + 1 < my_rows;
      int part = 0;
      auto prefetch_part = [&]() {
        prefetch(ctrl.meta[(i + 1) % kMetaDepth].r, (part & 1) ? p.teacher : p.student,
                 (part >> 1) * kU * nt, kU * nt);
        ++part;
      };
      RowSpan span = {0, 0, -1, -1, N};
      Acc2 a;
      a.reset();
      if (real) {
        // ------------------------------------------------------------ sweep 1
        span = span_of(m.r);
        const size_t off = ((size_t)m.r * p.ld - span.shift + (size_t)piece0 * N) * sizeof(TIn);
        const uint4* zp = reinterpret_cast<const uint4*>(static_cast<const char*>(p.student) + off) + tid;
        const uint4* up = reinterpret_cast<const uint4*>(static_cast<const char*>(p.teacher) + off) + tid;
        const f2_t nrefs = splat2(-m.zy * kLog2e), nreft = splat2(-m.uy * kLog2e);
        char* st = stash;
        int lp0 = tid;     // this thread's piece in the group's first step
        auto group = [&](auto full, int k0) {
          constexpr bool FULL = decltype(full)::value;
          uint4 z[kU], u[kU];
          if (ahead) prefetch_part();
#pragma unroll
          for (int h = 0; h < kU; ++h) {
            if ((FULL || lp0 + h * nt < span.pieces) &&
                ADWIN_CHK(((int64_t)piece0 + lp0 + h * nt + (RAG ? 0 : 1)) * N <= p.V + span.shift, p.status)) {
              z[h] = __ldcs(zp + h * nt);
              u[h] = __ldcs(up + h * nt);
            }
          }
          if (RAG) {
#pragma unroll
            for (int h = 0; h < kU; ++h) {
              const int lp = lp0 + h * nt;
              if (lp == span.first || lp == span.last)
                mask_piece<TIn>(z[h], u[h], span.e0(lp), lp == span.last ? span.last_n : N);
            }
          }
          if (TM && k0 < plan.tm_steps) {   // (every lane takes part)
            if (ADWIN_CHK(columns_ok(k0), p.status)) {
#pragma unroll
              for (int h = 0; h < kU; ++h) tm_store8(tm_lane + (uint32_t)((k0 + h) * 8), z[h], u[h]);
            }
          } else {
#pragma unroll
            for (int h = 0; h < kU; ++h) {
              if ((FULL || lp0 + h * nt < span.pieces) && ADWIN_CHK(stash_ok(st), p.status)) {
                *reinterpret_cast<uint4*>(st + 2 * h * array) = z[h];
                *reinterpret_cast<uint4*>(st + (2 * h + 1) * array) = u[h];
              }
            }
            st += 2 * kU * array;
          }
#pragma unroll
          for (int h = 0; h < kU; ++h) {
            if (FULL || lp0 + h * nt < span.pieces) {
              f2_t Z[NP], U[NP];
              Pairs<TIn>::make(z[h], Z);
              Pairs<TIn>::make(u[h], U);
              acc_grad<NP, 0>(Z, U, nrefs, nreft, a);
            }
          }
          zp += kU * nt;
          up += kU * nt;
          lp0 += kU * nt;
        };
        int k0 = 0;
        for (; (k0 + kU) * nt <= span.pieces; k0 += kU) group(std::true_type{}, k0);
        for (; k0 < plan.steps; k0 += kU) group(std::false_type{}, k0);
        if (TM) tm_wait_st();
      }

      // -------------------------------------------------------------- exchange
      rec[tid] = make_float4(hsum2(a.S), hsum2(a.A), hsum2(a.St), q_prev);
      named_arrive(kPosted, all);
      if (cl > 1) cluster_sync_all();
      if (!real) break;
      named_sync(kReady, all);

      // -------------------------------------------------------------- overflow: running maxima
      if (ctrl.out.again) {
        RowAcc ra;
        ra.reset();
        const char* st = stash;
        for (int k = 0; k < plan.steps; ++k) {
          uint4 zv, uv;
          if (TM && k < plan.tm_steps) {
            if (!ADWIN_CHK(columns_ok(k / kU * kU), p.status)) break;
            tm_load8(tm_lane + (uint32_t)(k * 8), zv, uv);
            tm_wait_ld();
          } else {
            if (!ADWIN_CHK(stash_ok(st - (k % kU) * 2 * array), p.status)) break;
            zv = *reinterpret_cast<const uint4*>(st);
            uv = *reinterpret_cast<const uint4*>(st + array);
            st += 2 * array;
          }
          if (tid + k * nt < span.pieces) {
            float z[N], u[N];
            Elem<TIn>::unpack(zv, z);
            Elem<TIn>::unpack(uv, u);
            acc_piece<N, false>(z, u, 0.f, ra);
          }
        }
        const float wms = warp_max(ra.m2s), wmt = warp_max(ra.m2t);
        const float fs = (ra.m2s == -INFINITY) ? 0.f : ex2f(ra.m2s - wms);
        const float ft = (ra.m2t == -INFINITY) ? 0.f : ex2f(ra.m2t - wmt);
        const float w1 = lane_sum(ra.S * fs), w2 = lane_sum(ra.A * fs), w3 = lane_sum(ra.St * ft);
        if (lane == 0) {
          float* x = ctrl.safe[warp];
          x[0] = wms; x[1] = wmt; x[2] = w1; x[3] = w2; x[4] = w3;
        }
        named_arrive(kPosted, all);
        if (cl > 1) cluster_sync_all();
        named_sync(kReady, all);
      }

      // -------------------------------------------------------------- sweep 2
      const f2_t L2 = splat2(kLog2e), NEG1 = splat2(-1.f);
      const float coef = ctrl.out.coef, c0 = ctrl.out.c0, gy = ctrl.out.gy;
      const f2_t nM2s = splat2(-ctrl.out.m2s), coef2 = splat2(coef);
      // bf16 logits: g = e * (coef*delta - coef*c0) saves one operation per pair; its rounding
      // (relative to coef*delta, not to the difference) is far inside that dtype's tolerance.
      const f2_t nc0 = splat2(sizeof(TIn) == 2 ? -coef * c0 : -c0);
      const int64_t yat = (int64_t)m.y + span.shift;                     // counted from piece 0
      const bool y_valid = m.y >= 0 && (int64_t)m.y < p.V;
      const int ypiece = y_valid ? (int)(yat / N - piece0) : -1;         // slice-relative
      char* gp = static_cast<char*>(p.grad) +
                 ((size_t)m.r * p.ld_grad - span.shift + (size_t)(piece0 + tid) * N) * sizeof(TOut);
      f2_t Q = 0ull;
      const char* st = stash;
      int lp0 = tid;
      auto group = [&](auto full, int k0) {
        constexpr bool FULL = decltype(full)::value;
        uint4 z[kU], u[kU];
        if (ahead) prefetch_part();
        if (TM && k0 < plan.tm_steps) {
          if (ADWIN_CHK(columns_ok(k0), p.status)) {
#pragma unroll
            for (int h = 0; h < kU; ++h) tm_load8(tm_lane + (uint32_t)((k0 + h) * 8), z[h], u[h]);
            tm_wait_ld();
          }
        } else {
#pragma unroll
          for (int h = 0; h < kU; ++h) {
            if ((FULL || lp0 + h * nt < span.pieces) && ADWIN_CHK(stash_ok(st), p.status)) {
              z[h] = *reinterpret_cast<const uint4*>(st + 2 * h * array);
              u[h] = *reinterpret_cast<const uint4*>(st + (2 * h + 1) * array);
            }
          }
          st += 2 * kU * array;
        }
#pragma unroll
        for (int h = 0; h < kU; ++h) {
          const int lp = lp0 + h * nt;
          if (FULL || lp < span.pieces) {
            f2_t Z[NP], U[NP], G[NP];
            Pairs<TIn>::make(z[h], Z);
            Pairs<TIn>::make(u[h], U);
#pragma unroll
            for (int e = 0; e < NP; ++e) {
              const f2_t E = ex2_2(fma2(Z[e], L2, nM2s));
              if (full_mode) {
                if (sizeof(TIn) == 2) G[e] = mul2(E, fma2(fma2(U[e], NEG1, Z[e]), coef2, nc0));
                else G[e] = mul2(E, mul2(add2(fma2(U[e], NEG1, Z[e]), nc0), coef2));
              } else {
                G[e] = mul2(E, coef2);
              }
            }
            if (!full_mode && lp == ypiece) {
              const int ye = (int)(yat % N);
#pragma unroll
              for (int e = 0; e < NP; ++e) {
                float lo, hi;
                upk2(G[e], lo, hi);
                if (ye == 2 * e) lo = gy;
                if (ye == 2 * e + 1) hi = gy;
                G[e] = pk2(lo, hi);
              }
            }
#pragma unroll
            for (int e = 0; e < NP; ++e) Q = fma2(G[e], G[e], Q);
            if (ADWIN_CHK(((int64_t)piece0 + lp + (RAG ? 0 : 1)) * N <= p.V + span.shift && m.r < p.B * p.T, p.status)) {
              char* dst = gp + (size_t)h * nt * N * sizeof(TOut);
              if (RAG && (lp == span.first || lp == span.last)) {   // the row's own entries only
                const int e0 = span.e0(lp), e1 = lp == span.last ? span.last_n : N;
#pragma unroll
                for (int e = 0; e < NP; ++e) {
                  float lo, hi;
                  upk2(G[e], lo, hi);
                  if (2 * e >= e0 && 2 * e < e1) Elem<TOut>::store1(dst, 2 * e, lo);
                  if (2 * e + 1 >= e0 && 2 * e + 1 < e1) Elem<TOut>::store1(dst, 2 * e + 1, hi);
                }
              } else {
                store_pairs<TOut, NP>(dst, G);
              }
            }
          }
        }
        gp += (size_t)kU * nt * N * sizeof(TOut);
        lp0 += kU * nt;
      };
      int k0 = 0;
      for (; (k0 + kU) * nt <= span.pieces; k0 += kU) group(std::true_type{}, k0);
      for (; k0 < plan.steps; k0 += kU) group(std::false_type{}, k0);
      q_prev = hsum2(Q);
    }
  }
  if (TM) asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  if (cl > 1) cluster_sync_all();   // no CTA leaves while a peer may still store into it
  __syncthreads();
  if (TM && warp == nw) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    tm_dealloc(ctrl.tmem_base, (uint32_t)plan.tm_cols);
  }
}

// ---------------------------------------------------------------------------- host side
constexpr int kSmemPerSm = 233472, kSmemReserved = 1024;   // bytes per SM, and taken by every CTA

struct RowsShape {
  int ctas, nt, tm_cols, cl;
  int most_kb;        // bytes of a row (both arrays) up to which the shape is taken, in KB
};
// From many small CTAs to two large ones, then clusters; the first that takes the row and holds it
// is used: the most CTAs per SM, because their number is what hides one row's exchange behind the
// others' streaming.  Tensor memory is shared out in powers of two.  Measured over 2.4 GB of logits
// and gradient (367 us at the copy rate; staged kernel / two sweeps over memory / this kernel):
//   bf16  V =   4 096  2471 / 726 / 475 us  {8, 64}       fp32  V =   4 096  1245 / 454 / 398 us  {5, 128}
//              8 192  1345 / 594 / 439     {5, 128}               12 000   784 / 606 / 401      {3, 224}
//             16 384   987 / 556 / 480     {3, 224}               16 384   599 / 647 / 394      {2, 352}
//             32 000   722 / 814 / 470     {2, 352}               32 000   500 / 686 / 429      {2, 352} x 2
//             50 264   636 / 856 / 499     {2, 352}               50 264   597 / 719 / 474      {2, 352} x 2
//            100 000   653 / 908 / 512     {2, 352} x 2           65 536   503 / 711 / 431      {2, 352} x 4
//            151 936   568 / 852 / 550     {2, 352} x 4
// bf16 rows are bound by arithmetic and latency (19 issue slots per entry, the ex2 unit 57 % busy),
// fp32 rows by memory.  Three or four steps in flight spill at 80 registers and lose, one step at 64
// registers and a third more threads is slower except around 16 384 entries.  (Rows off 16-byte
// boundaries cost the 64-thread bf16 kernels 68 bytes of spills.)
// {3, 224} could hold 126 KB but ends at 100 (25 600 entries of bf16).  {3, 224} / {2, 352}: bf16 12 000
// entries 527 / 566 us, 16 384 487 / 483, 22 000 508 / 487, 25 600 489 / 480, 27 000 523 / 487, 32 000
// 487 / 470; fp32 6 000 484 / 532, 8 192 392 / 400, 12 800 407 / 392, 14 336 413 / 394, 16 000 424 / 397.
// So the line keeps the rows that lose 6 % out; the last of those below it still lose 2 to 4 %.
constexpr RowsShape kShapes[] = {{8, 64, 0, 1, 1 << 20},   {5, 128, 0, 1, 1 << 20},
                                 {3, 224, 128, 1, 100},    {2, 352, 256, 1, 1 << 20},
                                 {2, 352, 256, 2, 1 << 20}, {2, 352, 256, 4, 1 << 20}};

constexpr int shape_smem(int ctas) { return kSmemPerSm / ctas - kSmemReserved; }

constexpr bool shape_plan(const RowsShape& sh, int64_t pieces, RowsPlan& plan) {
  plan.cl = sh.cl;
  plan.nt = sh.nt;
  plan.ctas = sh.ctas;
  plan.per_rank = (int)((pieces + sh.cl - 1) / sh.cl);
  const int need = (plan.per_rank + sh.nt - 1) / sh.nt;
  plan.steps = (need + kU - 1) / kU * kU;
  const int smem = shape_smem(sh.ctas) - rows_ctrl_bytes(sh.nt);
  const int sm_steps = smem / (32 * sh.nt) / kU * kU;
  // a lane group's columns are shared by its warps (every fourth); a piece pair takes 8 columns
  const int tm_most = sh.tm_cols ? sh.tm_cols / ((sh.nt + 127) / 128) / 8 / kU * kU : 0;
  plan.tm_steps = plan.steps < tm_most ? plan.steps : tm_most;
  plan.tm_cols = plan.tm_steps ? sh.tm_cols : 0;
  return plan.steps - plan.tm_steps <= sm_steps;
}

constexpr int rows_smem(const RowsPlan& plan) {
  return rows_ctrl_bytes(plan.nt) + (plan.steps - plan.tm_steps) * 32 * plan.nt;
}

// Bytes a launch asks for.  The CTAs of a cluster hold tensor memory while they wait for one another,
// and tcgen05.alloc waits without a limit: beside a tensor-core kernel of another stream (CTA pairs
// with all 512 columns), a cluster and a pair could each hold an SM's columns and wait for the other's.
// So the CTAs of a cluster take at least kClusterSmem: no CTA of tc_pipeline.cuh (199 KB), nor any
// above 163 KB, fits on an SM beside one, and row CTAs among themselves never need more than 512
// columns.  (A CTA without a cluster waits for nobody once it has its columns.)  Not the whole share of
// an SM, which would leave 28 KB of L1 to the streaming kernel that follows in a call with scalars
// over the rollout (update and audit on 3.8 GB of logits 1215 us so, 1164 with this).
constexpr int kClusterSmem = 65536 - kSmemReserved;
constexpr int launch_smem(const RowsPlan& plan) {
  const int need = rows_smem(plan);
  return plan.cl > 1 && plan.tm_cols > 0 && need < kClusterSmem ? kClusterSmem : need;
}
constexpr bool clusters_exclude_tensor_core_ctas() {
  for (const RowsShape& sh : kShapes) {
    RowsPlan plan = {};
    for (int64_t pieces = sh.cl; sh.cl > 1 && shape_plan(sh, pieces, plan); pieces += sh.cl * sh.nt * kU)
      if (plan.tm_cols > 0 && launch_smem(plan) + tc::kSmemBytes + 2 * kSmemReserved <= kSmemPerSm)
        return false;
  }
  return true;
}
static_assert(clusters_exclude_tensor_core_ctas(), "a cluster could wait for a pair's tensor memory");

bool rows_plan(int64_t pieces, RowsPlan& plan) {
  if (pieces < 1 || pieces > (int64_t)1 << 24) return false;
  for (const RowsShape& sh : kShapes)
    if (pieces * 32 <= (int64_t)sh.most_kb * 1024 && shape_plan(sh, pieces, plan)) return true;
  return false;
}

typedef void (*RowsKernel)(KlParams, RowsPlan);
// Whether the shapes of NT threads use tensor memory (all of them or none; `steps` is never less than
// kU, so a plan of such a shape always does).
constexpr bool uses_tensor_memory(int nt) {
  for (const RowsShape& sh : kShapes)
    if (sh.nt == nt) return sh.tm_cols > 0;
  return false;
}
template <typename TIn, typename TOut, int NT>
RowsKernel rows_kernel_nt(bool ragged) {
  constexpr bool TM = uses_tensor_memory(NT);
  return ragged ? kl_rows_kernel<TIn, TOut, NT, TM, true> : kl_rows_kernel<TIn, TOut, NT, TM, false>;
}
template <typename TIn, typename TOut>
RowsKernel rows_kernel(int nt, bool ragged) {
  switch (nt) {
    case 64: return rows_kernel_nt<TIn, TOut, 64>(ragged);
    case 128: return rows_kernel_nt<TIn, TOut, 128>(ragged);
    case 224: return rows_kernel_nt<TIn, TOut, 224>(ragged);
    case 352: return rows_kernel_nt<TIn, TOut, 352>(ragged);
    default: return nullptr;
  }
}

// Clusters of `cl` CTAs that the GPU holds at a time (some SMs of a GPC are left over when `cl` does
// not divide their number), kept per device.  The occupancy query counts one CTA per SM for kernels
// that allocate tensor memory, so it is asked about a kernel of the same shape without; which one does
// not matter, their launch bounds leave all of them the shape's CTAs per SM.
cudaError_t resident_clusters(const RowsPlan& plan, int sm_count, int& n) {
  constexpr int kDevices = 64;
  static std::mutex mu;
  static int seen[kDevices][kRowsMaxCl + 1];   // (shapes with a cluster differ in `cl` alone)
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kDevices) return cudaErrorNotSupported;
  std::lock_guard<std::mutex> lock(mu);
  n = seen[dev][plan.cl];
  if (n > 0) return cudaSuccess;
  const RowsKernel like = kl_rows_kernel<float, float, kRowsThreads, false, false>;
  const int smem = shape_smem(plan.ctas);
  e = cudaFuncSetAttribute(like, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(plan.cl * sm_count * plan.ctas);
  cfg.blockDim = dim3(plan.nt + 32);
  cfg.dynamicSmemBytes = (size_t)smem;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = plan.cl;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  e = cudaOccupancyMaxActiveClusters(&n, like, &cfg);
  if (e != cudaSuccess) return e;
  if (n < 1) return cudaErrorNotSupported;
  seen[dev][plan.cl] = n;
  return cudaSuccess;
}
constexpr bool cluster_shapes_differ_in_cl_alone() {
  for (const RowsShape& a : kShapes)
    for (const RowsShape& b : kShapes)
      if (a.cl > 1 && b.cl > 1 && (a.nt != kRowsThreads || a.ctas != b.ctas)) return false;
  return true;
}
static_assert(cluster_shapes_differ_in_cl_alone(), "resident_clusters keeps one number per cluster size");

template <typename TIn, typename TOut>
cudaError_t launch_rows_t(const KlParams& p, bool ragged, int sm_count, cudaStream_t s) {
  constexpr int N = Elem<TIn>::N;
  RowsPlan plan = {};
  if (!rows_plan(ragged ? (p.V + 2 * N - 2) / N : p.V / N, plan)) return cudaErrorNotSupported;
  const RowsKernel kernel = rows_kernel<TIn, TOut>(plan.nt, ragged);
  if (!kernel) return cudaErrorNotSupported;
  const int smem = launch_smem(plan);
  plan.num_clusters = plan.ctas * sm_count;
  cudaError_t e;
  if (plan.cl > 1) {
    e = resident_clusters(plan, sm_count, plan.num_clusters);
    if (e != cudaSuccess) return e;
  }
  // the shape's whole share whatever this call needs: the limit belongs to the kernel, which launches of
  // other threads with other row lengths use at the same time
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, shape_smem(plan.ctas));
  if (e != cudaSuccess) return e;
  const int64_t rows = p.B * p.T;
  if (plan.num_clusters > rows) plan.num_clusters = (int)rows;
  return launch_chained(kernel, (unsigned)(plan.cl * plan.num_clusters), plan.nt + 32, (size_t)smem, plan.cl, s,
                        p, plan);
}

}  // namespace

cudaError_t launch_kl_rows(const KlParams& p, int dtype, int grad_dtype, bool ragged, int sm_count,
                           cudaStream_t s) {
  if (dtype == ADWIN_F32)
    return grad_dtype == ADWIN_F32 ? launch_rows_t<float, float>(p, ragged, sm_count, s)
                                   : launch_rows_t<float, __nv_bfloat16>(p, ragged, sm_count, s);
  return grad_dtype == ADWIN_F32 ? launch_rows_t<__nv_bfloat16, float>(p, ragged, sm_count, s)
                                 : launch_rows_t<__nv_bfloat16, __nv_bfloat16>(p, ragged, sm_count, s);
}

}  // namespace adwin
