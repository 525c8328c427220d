// Shape-agnostic row kernel: one CTA per processed row, two sweeps over global memory.
//
// Sweep 1 streams z and u once and accumulates the online log-sum-exp statistics, sum e*delta
// (reverse KL) and the moments of the single-sweep gradient norm.  Sweep 2 (only for rows whose
// gradient is written) re-reads the row and writes g.  Any V, any row stride, any element
// alignment.  VEC: the rows of all arrays share one offset from a 16-byte boundary (always so when
// the arrays start on one and have one stride), and everything but the at most N - 1 entries before
// the first boundary and after the last is moved 16 bytes at a time; otherwise entry by entry.
// Calls without gradient come here, and layouts that the staged cluster kernel does not take.
#include "adwin_common.cuh"
#include "adwin_internal.h"

namespace adwin {

// 128-thread CTAs, one row each, four pairs of 16-byte loads in flight per thread: small CTAs put
// many independent rows on an SM, so one row's reduction overlaps the others' streaming.  The
// read-only pass is at the copy rate on a cool GPU (2.23 ms for 14.9 GB at V = 151 936); in a
// back-to-back series the power cap lowers the clocks and every instruction costs, hence references
// fixed by a thread's first group instead of a maximum per piece, and moments only where the norm
// takes them (series: 2.96 ms before, 2.55 now).  Measured in a series, threads x loads x CTAs per SM:
// 128x3x7 2.56, 128x4x6 2.55, 128x5x5 2.59, 128x6x4 2.67, 64x5x10 2.58, 256x4x3 2.64, 256x5x2 2.99 ms.
constexpr int kGenericThreads = 128;
constexpr int kGenericWarps = kGenericThreads / 32;
constexpr int kGenericUnroll = 4;
constexpr int kGenericMinBlocks = 6;   // CTAs per SM the register allocation leaves room for

// A thread's sums are good up to 2^48: e^2 delta^2, the largest term, stays below 2^128 then for
// logits up to 2^16 apart.
constexpr float kSafeSum = 281474976710656.f;

struct BlockScratch {
  float wm[2][kGenericWarps];
  float ws[6][kGenericWarps];
  float wq[kGenericWarps];
  RowScalars rs;
  RowTotals tot;
};

// Sweep 1 on packed fp32 pairs: sm_100 issues add / mul / fma on two fp32 lanes of a 64-bit
// register pair in one slot, which halves the issue slots of the element-wise part.  Even and odd entries of a piece
// accumulate separately; fold() adds the two lanes.
typedef unsigned long long pair_t;
__device__ __forceinline__ pair_t pair(float lo, float hi) {
  pair_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpair(pair_t v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ pair_t pfma(pair_t a, pair_t b, pair_t c) {
  pair_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ pair_t padd(pair_t a, pair_t b) {
  pair_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ pair_t pmul(pair_t a, pair_t b) {
  pair_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ pair_t pex2(pair_t x) {
  float a, b;
  unpair(x, a, b);
  return pair(ex2f(a), ex2f(b));
}
__device__ __forceinline__ float psum(pair_t v) {
  float a, b;
  unpair(v, a, b);
  return a + b;
}

struct PairAcc {
  float m2s, m2t;                  // running references, as in RowAcc
  pair_t S, A, B0, B1, B2, St;     // the sums of RowAcc, even / odd entries apart
  __device__ __forceinline__ void reset() {
    m2s = -INFINITY;
    m2t = -INFINITY;
    S = A = B0 = B1 = B2 = St = 0ull;   // the bit pattern of {0.f, 0.f}
  }
  __device__ __forceinline__ RowAcc fold() const {
    RowAcc a;
    a.m2s = m2s;
    a.m2t = m2t;
    a.S = psum(S);
    a.A = psum(A);
    a.B0 = psum(B0);
    a.B1 = psum(B1);
    a.B2 = psum(B2);
    a.St = psum(St);
    return a;
  }
};

// The sums of acc_piece<N, true> against the references that `a` holds, on pairs (N even).  MOM: all
// three moments of the gradient norm, or only B0, which is all that the norm of a sampled-token
// gradient takes.
template <int N, bool MOM>
__device__ __forceinline__ void acc_sums(const float (&z)[N], const float (&u)[N], float dref, PairAcc& a) {
  const pair_t L2 = pair(kLog2e, kLog2e), NEG1 = pair(-1.f, -1.f);
  const pair_t nms = pair(-a.m2s, -a.m2s), nmt = pair(-a.m2t, -a.m2t), ndref = pair(-dref, -dref);
#pragma unroll
  for (int i = 0; i < N; i += 2) {
    const pair_t Z = pair(z[i], z[i + 1]), U = pair(u[i], u[i + 1]);
    const pair_t E = pex2(pfma(Z, L2, nms));
    const pair_t D = padd(pfma(U, NEG1, Z), ndref);
    a.S = padd(a.S, E);
    a.B0 = pfma(E, E, a.B0);
    if (MOM) {
      const pair_t ED = pmul(E, D);
      a.A = padd(a.A, ED);
      a.B1 = pfma(E, ED, a.B1);
      a.B2 = pfma(ED, ED, a.B2);
    } else {
      a.A = pfma(E, D, a.A);
    }
    a.St = padd(a.St, pex2(pfma(U, L2, nmt)));
  }
}

// The same after raising the references to the piece's maxima.
template <int N, bool MOM>
__device__ __forceinline__ void acc_piece_pairs(const float (&z)[N], const float (&u)[N], float dref,
                                                PairAcc& a) {
  float zm = z[0], um = u[0];
#pragma unroll
  for (int i = 1; i < N; ++i) {
    zm = fmaxf(zm, z[i]);
    um = fmaxf(um, u[i]);
  }
  const float zl = zm * kLog2e, ul = um * kLog2e;
  if (zl > a.m2s) {
    const float f = ex2f(a.m2s - zl);
    const pair_t F = pair(f, f), F2 = pmul(F, F);
    a.S = pmul(a.S, F);
    a.A = pmul(a.A, F);
    a.B0 = pmul(a.B0, F2);
    if (MOM) {
      a.B1 = pmul(a.B1, F2);
      a.B2 = pmul(a.B2, F2);
    }
    a.m2s = zl;
  }
  if (ul > a.m2t) {
    const float f = ex2f(a.m2t - ul);
    a.St = pmul(a.St, pair(f, f));
    a.m2t = ul;
  }
  acc_sums<N, MOM>(z, u, dref, a);
}

// Combine the per-thread accumulators of a CTA; every thread returns the same totals.
__device__ __forceinline__ RowTotals block_combine(const RowAcc& a, BlockScratch& sm) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const float wms = warp_max(a.m2s), wmt = warp_max(a.m2t);
  const float fs = (a.m2s == -INFINITY) ? 0.f : ex2f(a.m2s - wms);
  const float ft = (a.m2t == -INFINITY) ? 0.f : ex2f(a.m2t - wmt);
  const float fs2 = fs * fs;
  float v[6] = {a.S * fs, a.A * fs, a.B0 * fs2, a.B1 * fs2, a.B2 * fs2, a.St * ft};
#pragma unroll
  for (int i = 0; i < 6; ++i) v[i] = warp_sum(v[i]);
  if (lane == 0) {
    sm.wm[0][warp] = wms;
    sm.wm[1][warp] = wmt;
#pragma unroll
    for (int i = 0; i < 6; ++i) sm.ws[i][warp] = v[i];
  }
  __syncthreads();
  RowTotals t;
  t.M2s = -INFINITY;
  t.M2t = -INFINITY;
#pragma unroll
  for (int w = 0; w < kGenericWarps; ++w) {
    t.M2s = fmaxf(t.M2s, sm.wm[0][w]);
    t.M2t = fmaxf(t.M2t, sm.wm[1][w]);
  }
  float acc[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int w = 0; w < kGenericWarps; ++w) {
    const float gs = (sm.wm[0][w] == -INFINITY) ? 0.f : ex2f(sm.wm[0][w] - t.M2s);
    const float gt = (sm.wm[1][w] == -INFINITY) ? 0.f : ex2f(sm.wm[1][w] - t.M2t);
    const float gs2 = gs * gs;
    acc[0] += sm.ws[0][w] * gs;
    acc[1] += sm.ws[1][w] * gs;
    acc[2] += sm.ws[2][w] * gs2;
    acc[3] += sm.ws[3][w] * gs2;
    acc[4] += sm.ws[4][w] * gs2;
    acc[5] += sm.ws[5][w] * gt;
  }
  t.S = acc[0];
  t.A = acc[1];
  t.B0 = acc[2];
  t.B1 = acc[3];
  t.B2 = acc[4];
  t.St = acc[5];
  return t;
}

template <typename TIn, typename TOut, bool VEC, bool MOM>
__global__ void __launch_bounds__(kGenericThreads, kGenericMinBlocks) kl_generic_kernel(KlParams p) {
  __shared__ BlockScratch sm;
  constexpr int N = VEC ? Elem<TIn>::N : 1;
  const int64_t rows = p.B * p.T;
  const int tid = threadIdx.x;

  for (int64_t r = blockIdx.x; r < rows; r += gridDim.x) {
    const int64_t b = r / p.T;
    const int t = (int)(r - b * p.T);
    if (t >= p.range[b]) continue;  // past the window: the row is never touched
    if (p.skip_below && t < p.skip_below[b]) continue;
    const bool write_grad = (p.grad != nullptr) && (t < p.ewin[b]);

    const char* zrow = static_cast<const char*>(p.student) + (size_t)r * p.ld * sizeof(TIn);
    const char* urow = static_cast<const char*>(p.teacher) + (size_t)r * p.ld * sizeof(TIn);
    const int y = p.tokens[r];
    const bool y_valid = (y >= 0) && ((int64_t)y < p.V);
    const int64_t yi = y_valid ? y : 0;
    const float zy = Elem<TIn>::load1(zrow, yi), uy = Elem<TIn>::load1(urow, yi);
    const float dref = zy - uy;

    RowAcc a;
    a.reset();
    // VEC: `head` entries up to the first boundary, whole pieces, `tail` entries
    int head = 0, tail = 0;
    if (VEC) {
      const int shift = (int)((reinterpret_cast<uintptr_t>(zrow) & 15) / sizeof(TIn));
      head = shift ? N - shift : 0;
      if (head > p.V) head = (int)p.V;
      tail = (int)((p.V - head) % N);
    }
    const int64_t pieces = VEC ? (p.V - head) / N : p.V;
    // the entry before or after the pieces that this thread looks after, or -1
    const int64_t edge = !VEC ? -1
                         : tid < head ? tid
                         : (tid >= 32 && tid - 32 < tail) ? p.V - tail + (tid - 32) : -1;
    if (VEC) {
      PairAcc pa;
      pa.reset();
      // kGenericUnroll pairs of 16-byte loads in flight per thread; a row that is read only once
      // (no gradient) is streamed past the caches, otherwise sweep 2 should find it in L2
      const uint4* zs = reinterpret_cast<const uint4*>(zrow + head * sizeof(TIn));
      const uint4* us = reinterpret_cast<const uint4*>(urow + head * sizeof(TIn));
      auto load = [&](int64_t i, uint4& zv, uint4& uv) {
        zv = write_grad ? __ldg(zs + i) : __ldcs(zs + i);
        uv = write_grad ? __ldg(us + i) : __ldcs(us + i);
      };
      // one piece at a time, the references raised before each
      auto singly = [&](int64_t i, int64_t end) {
        for (; i < end; i += kGenericThreads) {
          float z[N], u[N];
          uint4 zv, uv;
          if (!ADWIN_CHK(head + (i + 1) * N <= p.V, p.status)) break;
          load(i, zv, uv);
          Elem<TIn>::unpack(zv, reinterpret_cast<float(&)[Elem<TIn>::N]>(z));
          Elem<TIn>::unpack(uv, reinterpret_cast<float(&)[Elem<TIn>::N]>(u));
          acc_piece_pairs<N, MOM>(z, u, dref, pa);
        }
      };
      int64_t i = tid;
      bool first = true;
      for (; i + (kGenericUnroll - 1) * kGenericThreads < pieces;
           i += kGenericUnroll * kGenericThreads) {
        uint4 zv[kGenericUnroll], uv[kGenericUnroll];
        if (!ADWIN_CHK(head + (i + (kGenericUnroll - 1) * kGenericThreads + 1) * N <= p.V, p.status)) break;
#pragma unroll
        for (int h = 0; h < kGenericUnroll; ++h) load(i + h * kGenericThreads, zv[h], uv[h]);
        if (first) {   // the references of all whole groups: the maxima of the thread's first one
          first = false;
#pragma unroll
          for (int h = 0; h < kGenericUnroll; ++h) {
            float z[N], u[N];
            Elem<TIn>::unpack(zv[h], reinterpret_cast<float(&)[Elem<TIn>::N]>(z));
            Elem<TIn>::unpack(uv[h], reinterpret_cast<float(&)[Elem<TIn>::N]>(u));
#pragma unroll
            for (int j = 0; j < N; ++j) {
              pa.m2s = fmaxf(pa.m2s, z[j]);
              pa.m2t = fmaxf(pa.m2t, u[j]);
            }
          }
          pa.m2s *= kLog2e;
          pa.m2t *= kLog2e;
        }
#pragma unroll
        for (int h = 0; h < kGenericUnroll; ++h) {
          float z[N], u[N];
          Elem<TIn>::unpack(zv[h], reinterpret_cast<float(&)[Elem<TIn>::N]>(z));
          Elem<TIn>::unpack(uv[h], reinterpret_cast<float(&)[Elem<TIn>::N]>(u));
          acc_sums<N, MOM>(z, u, dref, pa);
        }
      }
      // a sum that has outgrown its reference (or is no number): the groups again, against running maxima
      if (!first && !(psum(pa.S) < kSafeSum && psum(pa.St) < kSafeSum)) {
        pa.reset();
        singly(tid, i);
      }
      singly(i, pieces);
      a = pa.fold();
      if (edge >= 0) {
        const float z[1] = {Elem<TIn>::load1(zrow, edge)}, u[1] = {Elem<TIn>::load1(urow, edge)};
        acc_piece<1, true>(z, u, dref, a);
      }
    } else {
      for (int64_t i = tid; i < pieces; i += kGenericThreads) {
        float z[N], u[N];
        if (!ADWIN_CHK(i < p.ld, p.status)) break;
        z[0] = Elem<TIn>::load1(zrow, i);
        u[0] = Elem<TIn>::load1(urow, i);
        acc_piece<N, true>(z, u, dref, a);
      }
    }
    const RowTotals tot = block_combine(a, sm);
    if (tid == 0)
      sm.rs = finish_row(tot, zy, uy, y_valid, dref, p.alpha, p.mode,
                         p.row_coef ? p.row_coef + r : nullptr);
    __syncthreads();
    const RowScalars rs = sm.rs;

    float q = 0.f;
    if (write_grad) {
      char* grow = static_cast<char*>(p.grad) + (size_t)r * p.ld_grad * sizeof(TOut);
      const bool full = (p.mode == ADWIN_GRAD_FULL_KL);
      auto gradient = [&](float z, float u, int64_t k) {
        const float e = ex2f(fmaf(z, kLog2e, -tot.M2s));
        if (full) return e * (rs.coef * (((z - u) - dref) - rs.c0));
        return (y_valid && k == yi) ? rs.gy : e * rs.coef;
      };
      if (edge >= 0) {
        const float g = gradient(Elem<TIn>::load1(zrow, edge), Elem<TIn>::load1(urow, edge), edge);
        q = fmaf(g, g, q);
        Elem<TOut>::store1(grow, edge, g);
      }
      char* gbody = grow + head * sizeof(TOut);
      for (int64_t i = tid; i < pieces; i += kGenericThreads) {
        float z[N], u[N], g[N];
        if (!ADWIN_CHK(head + (i + 1) * N <= p.V && head + (i + 1) * N <= p.ld_grad, p.status)) break;
        if (VEC) {
          const uint4 zv = __ldg(reinterpret_cast<const uint4*>(zrow + head * sizeof(TIn)) + i);
          const uint4 uv = __ldg(reinterpret_cast<const uint4*>(urow + head * sizeof(TIn)) + i);
          Elem<TIn>::unpack(zv, reinterpret_cast<float(&)[Elem<TIn>::N]>(z));
          Elem<TIn>::unpack(uv, reinterpret_cast<float(&)[Elem<TIn>::N]>(u));
        } else {
          z[0] = Elem<TIn>::load1(zrow, i);
          u[0] = Elem<TIn>::load1(urow, i);
        }
#pragma unroll
        for (int j = 0; j < N; ++j) {
          g[j] = gradient(z[j], u[j], head + i * N + j);
          q = fmaf(g[j], g[j], q);
        }
        if (VEC) {
          if (sizeof(TOut) == 4) {
            float4* o = reinterpret_cast<float4*>(gbody) + i * (N / 4);
#pragma unroll
            for (int j = 0; j < N / 4; ++j)
              o[j] = make_float4(g[4 * j], g[4 * j + 1], g[4 * j + 2], g[4 * j + 3]);
          } else {
            if (N == 8) {
              uint4 o;
              o.x = pack_bf16x2(g[0], g[1]);
              o.y = pack_bf16x2(g[2], g[3]);
              o.z = pack_bf16x2(g[4], g[5]);
              o.w = pack_bf16x2(g[6], g[7]);
              reinterpret_cast<uint4*>(gbody)[i] = o;
            } else {  // fp32 logits, bf16 gradient: 4 entries = 8 bytes
              uint2 o;
              o.x = pack_bf16x2(g[0], g[1]);
              o.y = pack_bf16x2(g[2], g[3]);
              reinterpret_cast<uint2*>(gbody)[i] = o;
            }
          }
        } else {
          Elem<TOut>::store1(grow, i, g[0]);
        }
      }
      // fixed-order CTA sum of the squared entries
      q = warp_sum(q);
      if ((tid & 31) == 0) sm.wq[tid >> 5] = q;
      __syncthreads();
      q = 0.f;
#pragma unroll
      for (int w = 0; w < kGenericWarps; ++w) q += sm.wq[w];
    }
    if (tid == 0 && ADWIN_CHK(r >= 0 && r < rows, p.status)) {
      p.kl[r] = rs.kl;
      p.logratio[r] = rs.c;
      if (p.gsq) p.gsq[r] = write_grad ? q : rs.gsq_expanded;
      if (p.lse_s) p.lse_s[r] = rs.lse_s;
      if (p.lse_t) p.lse_t[r] = rs.lse_t;
      int bits = 0;
      if (!y_valid) bits |= ADWIN_DEV_TOKEN_RANGE;
      if (rs.nonfinite) bits |= ADWIN_DEV_NONFINITE;
      if (bits) atomicOr(p.status, bits);
    }
    __syncthreads();  // scratch is reused by the next row
  }
}

template <typename TIn, typename TOut>
static cudaError_t launch_t(const KlParams& p, bool vec, int grid, cudaStream_t s) {
  if (vec && p.mode == ADWIN_GRAD_FULL_KL)
    kl_generic_kernel<TIn, TOut, true, true><<<grid, kGenericThreads, 0, s>>>(p);
  else if (vec)
    kl_generic_kernel<TIn, TOut, true, false><<<grid, kGenericThreads, 0, s>>>(p);
  else
    kl_generic_kernel<TIn, TOut, false, true><<<grid, kGenericThreads, 0, s>>>(p);
  return cudaGetLastError();
}

cudaError_t launch_kl_generic(const KlParams& p, int dtype, int grad_dtype, bool vec, int sm_count,
                              cudaStream_t s) {
  const int64_t rows = p.B * p.T;
  if (rows == 0) return cudaSuccess;
  const int64_t cap = (int64_t)sm_count * 64;
  const int grid = (int)(rows < cap ? rows : cap);
  if (dtype == ADWIN_F32) {
    return grad_dtype == ADWIN_F32 ? launch_t<float, float>(p, vec, grid, s)
                                   : launch_t<float, __nv_bfloat16>(p, vec, grid, s);
  }
  return grad_dtype == ADWIN_F32 ? launch_t<__nv_bfloat16, float>(p, vec, grid, s)
                                 : launch_t<__nv_bfloat16, __nv_bfloat16>(p, vec, grid, s);
}

}  // namespace adwin
