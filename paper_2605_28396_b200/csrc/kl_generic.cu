// Shape-agnostic row kernel: one CTA per processed row (a cluster, where a call has few rows and
// writes no gradient), two sweeps over global memory.
//
// Sweep 1 streams z and u once and accumulates the online log-sum-exp statistics, sum e*delta
// (reverse KL) and the moments of the single-sweep gradient norm.  Sweep 2 (only for rows whose
// gradient is written) re-reads the row and writes g.  Any V, any row stride, any element
// alignment.  VEC: the rows of all arrays share one offset from a 16-byte boundary (always so when
// the arrays start on one and have one stride), and everything but the at most N - 1 entries before
// the first boundary and after the last is moved 16 bytes at a time; otherwise entry by entry.
// Calls without gradient come here, and layouts that the row kernel does not take.
#include "adwin_common.cuh"
#include "adwin_internal.h"
#include "kl_pairs.cuh"

namespace adwin {

// 128-thread CTAs, one row each, four pairs of 16-byte loads in flight per thread: small CTAs put
// many independent rows on an SM, so one row's reduction overlaps the others' streaming.  The
// read-only pass is at the copy rate on a cool GPU (2.23 ms for 14.9 GB at V = 151 936); in a
// back-to-back series the power cap lowers the clocks and every instruction costs, hence references
// fixed by a thread's first group instead of a maximum per piece, and moments only where the norm
// takes them (series: 2.96 ms before, 2.55 now).  Measured in a series, threads x loads x CTAs per SM:
// 128x3x7 2.56, 128x4x6 2.55, 128x5x5 2.59, 128x6x4 2.67, 64x5x10 2.58, 256x4x3 2.64, 256x5x2 2.99 ms.
// An exponent x = z log2e - reference is good to 2^-24 |x|, so a reference is to be near the entries that
// carry the mass: the sampled token's logit is taken beside the first group, and a step of 1/32 from
// lane to lane keeps equal logits (bf16 has few distinct ones) from sharing one error of the
// exponential.  Root mean square error of the log-ratio at V = 151 936: running maxima 2.4e-7, first
// group alone 3.3e-7, so 2.3e-7; of the squared norm relative to it, N(0,2) logits in bf16: 4.5, 7.1, 5.4e-7.
constexpr int kGenericThreads = 128;
constexpr int kGenericMaxCl = 4;
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
  float xtot[2][kGenericMaxCl][8];   // per row parity, the totals of the row's CTAs (in the first one)
  RowScalars rs;
};

// Sweep 1 on packed fp32 pairs: sm_100 issues add / mul / fma on two fp32 lanes of a 64-bit
// register pair in one slot, which halves the issue slots of the element-wise part.  Even and odd entries of a piece
// accumulate separately; fold() adds the two lanes.
struct PairAcc {
  float m2s, m2t;                  // running references, as in RowAcc
  f2_t S, A, B0, B1, B2, St;     // the sums of RowAcc, even / odd entries apart
  __device__ __forceinline__ void reset() {
    m2s = -INFINITY;
    m2t = -INFINITY;
    S = A = B0 = B1 = B2 = St = 0ull;   // the bit pattern of {0.f, 0.f}
  }
  __device__ __forceinline__ RowAcc fold() const {
    RowAcc a;
    a.m2s = m2s;
    a.m2t = m2t;
    a.S = hsum2(S);
    a.A = hsum2(A);
    a.B0 = hsum2(B0);
    a.B1 = hsum2(B1);
    a.B2 = hsum2(B2);
    a.St = hsum2(St);
    return a;
  }
};

// The sums of acc_piece<N, true> against the references that `a` holds, on pairs (N even).  MOM: all
// three moments of the gradient norm, or only B0, which is all that the norm of a sampled-token
// gradient takes.  That norm subtracts p_y^2 from B0 / S^2, which only agree to the last bits for a
// token with most of the mass when its exponent is taken near zero: it keeps to running maxima.
template <int N, bool MOM>
__device__ __forceinline__ void acc_sums(const float (&z)[N], const float (&u)[N], float dref, PairAcc& a) {
  const f2_t L2 = splat2(kLog2e), NEG1 = splat2(-1.f);
  const f2_t nms = splat2(-a.m2s), nmt = splat2(-a.m2t), ndref = splat2(-dref);
#pragma unroll
  for (int i = 0; i < N; i += 2) {
    const f2_t Z = pk2(z[i], z[i + 1]), U = pk2(u[i], u[i + 1]);
    const f2_t E = ex2_2(fma2(Z, L2, nms));
    const f2_t D = add2(fma2(U, NEG1, Z), ndref);
    a.S = add2(a.S, E);
    a.B0 = fma2(E, E, a.B0);
    if (MOM) {
      const f2_t ED = mul2(E, D);
      a.A = add2(a.A, ED);
      a.B1 = fma2(E, ED, a.B1);
      a.B2 = fma2(ED, ED, a.B2);
    } else {
      a.A = fma2(E, D, a.A);
    }
    a.St = add2(a.St, ex2_2(fma2(U, L2, nmt)));
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
  const float zl = reference_of(zm), ul = reference_of(um);
  if (zl > a.m2s) {
    const float f = ex2f(a.m2s - zl);
    const f2_t F = splat2(f), F2 = mul2(F, F);
    a.S = mul2(a.S, F);
    a.A = mul2(a.A, F);
    a.B0 = mul2(a.B0, F2);
    if (MOM) {
      a.B1 = mul2(a.B1, F2);
      a.B2 = mul2(a.B2, F2);
    }
    a.m2s = zl;
  }
  if (ul > a.m2t) {
    const float f = ex2f(a.m2t - ul);
    a.St = mul2(a.St, splat2(f));
    a.m2t = ul;
  }
  acc_sums<N, MOM>(z, u, dref, a);
}

// Partial sums against references of their own, in the order given.
template <int MAX>
__device__ __forceinline__ RowTotals combine_parts(const RowAcc (&part)[MAX], int n) {
  RowTotals t;
  t.M2s = t.M2t = -INFINITY;
  t.S = t.A = t.B0 = t.B1 = t.B2 = t.St = 0.f;
#pragma unroll
  for (int w = 0; w < MAX; ++w) {
    if (w >= n) break;
    t.M2s = fmaxf(t.M2s, part[w].m2s);
    t.M2t = fmaxf(t.M2t, part[w].m2t);
  }
#pragma unroll
  for (int w = 0; w < MAX; ++w) {
    if (w >= n) break;
    const float gs = (part[w].m2s == -INFINITY) ? 0.f : ex2f(part[w].m2s - t.M2s);
    const float gt = (part[w].m2t == -INFINITY) ? 0.f : ex2f(part[w].m2t - t.M2t);
    const float gs2 = gs * gs;
    t.S += part[w].S * gs;
    t.A += part[w].A * gs;
    t.B0 += part[w].B0 * gs2;
    t.B1 += part[w].B1 * gs2;
    t.B2 += part[w].B2 * gs2;
    t.St += part[w].St * gt;
  }
  return t;
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
  RowAcc part[kGenericWarps];
#pragma unroll
  for (int w = 0; w < kGenericWarps; ++w) {
    part[w].m2s = sm.wm[0][w];
    part[w].m2t = sm.wm[1][w];
    part[w].S = sm.ws[0][w];
    part[w].A = sm.ws[1][w];
    part[w].B0 = sm.ws[2][w];
    part[w].B1 = sm.ws[3][w];
    part[w].B2 = sm.ws[4][w];
    part[w].St = sm.ws[5][w];
  }
  return combine_parts<kGenericWarps>(part, kGenericWarps);
}

// SPLIT: read-only rows, each over a cluster of CTAs that take a run of its pieces.
template <typename TIn, typename TOut, bool VEC, bool MOM, bool SPLIT>
__global__ void __launch_bounds__(kGenericThreads, kGenericMinBlocks) kl_generic_kernel(KlParams p, int clusters_of) {
  chain();
  __shared__ BlockScratch sm;
  constexpr int N = VEC ? Elem<TIn>::N : 1;
  const int64_t rows = p.B * p.T;
  const int tid = threadIdx.x;

  const int cl = SPLIT ? clusters_of : 1, rank = SPLIT ? (int)cluster_rank() : 0;
  int par = 0;
  if (SPLIT) cluster_sync_all();   // every CTA runs before another one stores into it

  for (int64_t r = blockIdx.x / cl; r < rows; r += gridDim.x / cl) {
    const int64_t b = r / p.T;
    const int t = (int)(r - b * p.T);
    if (t >= p.range[b]) continue;  // past the window: the row is never touched
    if (p.skip_below && t < p.skip_below[b]) continue;
    const bool write_grad = !SPLIT && (p.grad != nullptr) && (t < p.ewin[b]);

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
    int64_t pieces = VEC ? (p.V - head) / N : p.V, from = 0;
    if (SPLIT) {
      const int64_t part = ((pieces + cl - 1) / cl + 7) / 8 * 8;   // (whole 128-byte lines)
      from = min(rank * part, pieces);
      pieces = min(from + part, pieces);
    }
    // the entry before or after the pieces that this thread looks after, or -1
    const int64_t edge = !VEC || rank != 0 ? -1
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
      int64_t i = from + tid;
      bool first = true;
      for (; i + (kGenericUnroll - 1) * kGenericThreads < pieces;
           i += kGenericUnroll * kGenericThreads) {
        uint4 zv[kGenericUnroll], uv[kGenericUnroll];
        if (!ADWIN_CHK(head + (i + (kGenericUnroll - 1) * kGenericThreads + 1) * N <= p.V, p.status)) break;
#pragma unroll
        for (int h = 0; h < kGenericUnroll; ++h) load(i + h * kGenericThreads, zv[h], uv[h]);
        if (MOM && first) {   // the references of all whole groups (see the top)
          first = false;
          pa.m2s = zy;
          pa.m2t = uy;
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
          const float apart = (float)(tid & 31) * 0.03125f;
          pa.m2s = reference_of(pa.m2s) + apart;
          pa.m2t = reference_of(pa.m2t) + apart;
        }
#pragma unroll
        for (int h = 0; h < kGenericUnroll; ++h) {
          float z[N], u[N];
          Elem<TIn>::unpack(zv[h], reinterpret_cast<float(&)[Elem<TIn>::N]>(z));
          Elem<TIn>::unpack(uv[h], reinterpret_cast<float(&)[Elem<TIn>::N]>(u));
          if (MOM) acc_sums<N, true>(z, u, dref, pa);
          else acc_piece_pairs<N, false>(z, u, dref, pa);
        }
      }
      // a sum that has outgrown its reference (or is no number): the groups again, against running maxima
      if (MOM && !first && !(hsum2(pa.S) < kSafeSum && hsum2(pa.St) < kSafeSum)) {
        pa.reset();
        singly(from + tid, i);
      }
      singly(i, pieces);
      a = pa.fold();
      if (edge >= 0) {
        const float z[1] = {Elem<TIn>::load1(zrow, edge)}, u[1] = {Elem<TIn>::load1(urow, edge)};
        acc_piece<1, true>(z, u, dref, a);
      }
    } else {
      for (int64_t i = from + tid; i < pieces; i += kGenericThreads) {
        float z[N], u[N];
        if (!ADWIN_CHK(i < p.ld, p.status)) break;
        z[0] = Elem<TIn>::load1(zrow, i);
        u[0] = Elem<TIn>::load1(urow, i);
        acc_piece<N, true>(z, u, dref, a);
      }
    }
    RowTotals tot = block_combine(a, sm);
    if (SPLIT) {
      if (tid == 0) {
        const uint32_t dst = map_to_rank(smem_u32(sm.xtot[par][rank]), 0);
        remote_store4(dst, tot.M2s, tot.M2t, tot.S, tot.A);
        remote_store4(dst + 16, tot.B0, tot.B1, tot.B2, tot.St);
      }
      cluster_sync_all();
      if (rank != 0) {
        par ^= 1;
        continue;
      }
      RowAcc part[kGenericMaxCl];
#pragma unroll
      for (int j = 0; j < kGenericMaxCl; ++j) {
        const float* x = sm.xtot[par][j];
        if (j < cl) part[j] = {x[0], x[2], x[3], x[4], x[5], x[6], x[1], x[7]};
      }
      tot = combine_parts<kGenericMaxCl>(part, cl);
      par ^= 1;
    }
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
static cudaError_t launch_t(const KlParams& p, bool vec, int cl, int clusters, cudaStream_t s) {
  const bool mom = p.mode == ADWIN_GRAD_FULL_KL;
  void (*kernel)(KlParams, int);
  if (cl > 1)
    kernel = !vec ? kl_generic_kernel<TIn, TIn, false, true, true>
             : mom ? kl_generic_kernel<TIn, TIn, true, true, true> : kl_generic_kernel<TIn, TIn, true, false, true>;
  else
    kernel = !vec ? kl_generic_kernel<TIn, TOut, false, true, false>
             : mom ? kl_generic_kernel<TIn, TOut, true, true, false> : kl_generic_kernel<TIn, TOut, true, false, false>;
  return launch_chained(kernel, (unsigned)(clusters * cl), kGenericThreads, 0, cl, s, p, cl);
}

// CTAs per row of a read-only call.  A call of few rows leaves SMs idle or fills its last wave badly; a
// cluster per row makes shorter waves, at a price (one cluster barrier and one more start per row)
// that weighs the more the shorter the row.  Both are put in waves of whole rows; the price was
// fitted to these times (us, one / two / four CTAs per row; `rows` is all the call may hold, the
// lengths are on the device):
//   bf16 V = 151 936:  64 rows 46 / 29 / 20   300 56 / 45 / 46   900 117 / 108 / 107   1500 154 / 158 / 167
//   fp32 V =  93 534: 100 rows 69 / 41 / 26   300 73 / 50 / 54   600  88 /  96 /  87    945 164 / 145 / 136
//   bf16 V =  32 000:  64 rows 17 / 15 / 13   300 19 / 18 / 23   900  34 /  39 /  50   4000  95 / 126 / 185
static int split_rows(int64_t rows, int64_t row_bytes, int sm_count) {
  const int64_t slots = (int64_t)sm_count * kGenericMinBlocks;
  const double price = 0.15 * (512 << 10) / (double)row_bytes;
  int best = 1;
  double cost = 0.0;
  for (int cl = 1, lg = 0; cl <= kGenericMaxCl; cl *= 2, ++lg) {
    const double c = (double)((rows * cl + slots - 1) / slots) / cl * (1.0 + price * lg);
    if (cl == 1 || c < cost) {
      best = cl;
      cost = c;
    }
  }
  return best;
}

cudaError_t launch_kl_generic(const KlParams& p, int dtype, int grad_dtype, bool vec, int sm_count,
                              cudaStream_t s) {
  const int64_t rows = p.B * p.T;
  if (rows == 0) return cudaSuccess;
  const int cl = p.grad ? 1 : split_rows(rows, 2 * p.V * (dtype == ADWIN_F32 ? 4 : 2), sm_count);
  const int64_t cap = (int64_t)sm_count * 64;
  const int grid = (int)(rows < cap ? rows : cap);
  if (dtype == ADWIN_F32) {
    return grad_dtype == ADWIN_F32 ? launch_t<float, float>(p, vec, cl, grid, s)
                                   : launch_t<float, __nv_bfloat16>(p, vec, cl, grid, s);
  }
  return grad_dtype == ADWIN_F32 ? launch_t<__nv_bfloat16, float>(p, vec, cl, grid, s)
                                 : launch_t<__nv_bfloat16, __nv_bfloat16>(p, vec, cl, grid, s);
}

}  // namespace adwin
