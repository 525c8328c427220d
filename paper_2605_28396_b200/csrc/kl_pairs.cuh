// Building blocks shared by the kernels that keep a row on chip between their two sweeps (sm_100a):
// packed fp32 arithmetic on 16-byte pieces, the walk over the compact row list, rows off 16-byte
// boundaries, tensor memory as a scratchpad, and stores into a cluster peer's shared memory.
#pragma once

#include "adwin_common.cuh"

namespace adwin {

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ uint32_t map_to_rank(uint32_t local_addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local_addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void remote_store4(uint32_t addr, float a, float b, float c, float d) {
  asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(a), "f"(b),
               "f"(c), "f"(d)
               : "memory");
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::
                   : "memory");
}
// The two halves of it, for a thread that publishes nothing itself: what it does between them overlaps its
// peers' way to the barrier.
__device__ __forceinline__ void cluster_arrive_relaxed() {
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// Tensor memory as a scratchpad: 512 columns x 128 lanes x 32 bit = 256 KB per SM that a
// kernel without MMAs leaves idle.  A consumer thread parks the 16-byte pieces it has read in
// sweep 1 in its own lane (lane = 32*(warp%4) + laneid, the only lanes a warp may touch) and gets
// them back in sweep 2, so the streamed chunks are neither kept in shared memory nor fetched again.
__device__ __forceinline__ void tm_alloc(uint32_t dst_smem, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(cols) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tm_dealloc(uint32_t taddr, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
}
__device__ __forceinline__ void tm_store8(uint32_t taddr, const uint4& a, const uint4& b) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(taddr),
               "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w) : "memory");
}
__device__ __forceinline__ void tm_store4(uint32_t taddr, const uint4& a) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(taddr), "r"(a.x), "r"(a.y),
               "r"(a.z), "r"(a.w) : "memory");
}
__device__ __forceinline__ void tm_load8(uint32_t taddr, uint4& a, uint4& b) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w), "=r"(b.x), "=r"(b.y), "=r"(b.z), "=r"(b.w)
               : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tm_load4(uint32_t taddr, uint4& a) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w) : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tm_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tm_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Walks the compact list of processed rows.  The prefix sums of the current sequence are cached
// in registers, so locating a row touches global memory only when it crosses into a new sequence.
struct RowCursor {
  int64_t b, lo, hi;   // sequence, offsets[b], offsets[b+1]
  int32_t ew;          // effective window of sequence b
  __device__ __forceinline__ void init(const KlParams& p) {
    b = 0;
    lo = 0;
    hi = p.B > 0 ? p.offsets[1] : 0;
    ew = p.B > 0 ? p.ewin[0] : 0;
  }
  // Global row of processed-row ordinal n (ordinals must not decrease) and whether its gradient
  // is written.
  __device__ __forceinline__ int64_t locate(const KlParams& p, int64_t n, bool& wg) {
    while (n >= hi && b + 1 < p.B) {
      ++b;
      lo = hi;
      hi = p.offsets[b + 1];
      ew = p.ewin[b];
    }
    const int64_t t = n - lo;
    wg = (p.grad != nullptr) && (t < ew);
    return b * p.T + t;
  }
  __device__ __forceinline__ void fetch_row(const KlParams& p, int64_t ordinal, bool in_range,
                                            int64_t& r, int& y, bool& wg) {
    if (in_range) {
      r = locate(p, ordinal, wg);
      y = p.tokens[r];
    }
  }
};

// ---------------------------------------------------------------------------- packed fp32 pairs
// sm_100 issues add/mul/fma on two fp32 lanes held in a 64-bit register pair in one slot
// (add.f32x2 / mul.f32x2 / fma.f32x2).  The sweeps are issue- and MUFU-bound, so all element-wise
// arithmetic is done on pairs; only ex2 (MUFU) is per lane.
typedef unsigned long long f2_t;

__device__ __forceinline__ f2_t pk2(float lo, float hi) {
  f2_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void upk2(f2_t v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f2_t fma2(f2_t a, f2_t b, f2_t c) {
  f2_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ f2_t add2(f2_t a, f2_t b) {
  f2_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f2_t mul2(f2_t a, f2_t b) {
  f2_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f2_t ex2_2(f2_t x) {
  float a, b;
  upk2(x, a, b);
  return pk2(ex2f(a), ex2f(b));
}
__device__ __forceinline__ f2_t splat2(float v) { return pk2(v, v); }
__device__ __forceinline__ f2_t sub2(f2_t a, f2_t b) {
  f2_t d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
// 2^x of a pair on the FMA pipe, to relieve the MUFU unit that bounds sweep 1.  x is clamped to
// [-120, 105] (below that the term is nil against a sum >= 1; at the upper end the result exceeds
// the limit that sends the row to the safe path), rounded to the nearest integer n by adding
// 1.5*2^23, 2^(x-n) comes from a degree-4 polynomial on [-1/2, 1/2] (relative error < 2.7e-6,
// mean 4e-8) and n is added to the exponent field.  A NaN comes out as a finite number: callers
// keep a second, unclamped use of the input so that it still poisons the row.
__device__ __forceinline__ f2_t ex2_poly2(f2_t x) {
  float a, b;
  upk2(x, a, b);
  a = fminf(fmaxf(a, -120.f), 105.f);
  b = fminf(fmaxf(b, -120.f), 105.f);
  const f2_t xc = pk2(a, b);
  const f2_t MG = splat2(12582912.f);
  const f2_t t = add2(xc, MG);
  const f2_t f = sub2(xc, sub2(t, MG));
  f2_t q = fma2(splat2(9.570101276e-03f), f, splat2(5.591785908e-02f));
  q = fma2(q, f, splat2(2.402474433e-01f));
  q = fma2(q, f, splat2(6.931217909e-01f));
  q = fma2(q, f, splat2(9.999992847e-01f));
  float tl, th, ql, qh;
  upk2(t, tl, th);
  upk2(q, ql, qh);
  const uint32_t rl = __float_as_uint(ql) + (__float_as_uint(tl) << 23);
  const uint32_t rh = __float_as_uint(qh) + (__float_as_uint(th) << 23);
  return pk2(__uint_as_float(rl), __uint_as_float(rh));
}
__device__ __forceinline__ float hsum2(f2_t v) {
  float a, b;
  upk2(v, a, b);
  return a + b;
}

// Sums of pairs with what their additions round off (Knuth's two-sum); plain ones without EXACT.
template <bool EXACT>
struct ExactSum {
  f2_t hi, lo;
  __device__ __forceinline__ void set(f2_t x) {
    hi = x;
    lo = 0ull;
  }
  __device__ __forceinline__ void set(f2_t x, f2_t y) {
    hi = add2(x, y);
    lo = 0ull;
    if (EXACT) {
      const f2_t c = sub2(hi, x);
      lo = add2(sub2(x, sub2(hi, c)), sub2(y, c));
    }
  }
  __device__ __forceinline__ void add(f2_t x) {
    const f2_t s = add2(hi, x);
    if (EXACT) {
      const f2_t c = sub2(s, hi);
      lo = add2(lo, add2(sub2(hi, sub2(s, c)), sub2(x, c)));
    }
    hi = s;
  }
  __device__ __forceinline__ void add(const ExactSum& x) {
    if (EXACT) lo = add2(lo, x.lo);
    add(x.hi);
  }
  __device__ __forceinline__ ExactSum of_lane_xor(int o) const {
    ExactSum x;
    x.hi = __shfl_xor_sync(0xffffffffu, hi, o);
    x.lo = EXACT ? __shfl_xor_sync(0xffffffffu, lo, o) : 0ull;
    return x;
  }
};

// A 16-byte piece as NP pairs of consecutive vocabulary entries.
template <typename T>
struct Pairs;
template <>
struct Pairs<__nv_bfloat16> {
  static constexpr int NP = 4;
  __device__ static __forceinline__ void make(const uint4& v, f2_t (&o)[4]) {
    o[0] = pk2(bf16lo(v.x), bf16hi(v.x));
    o[1] = pk2(bf16lo(v.y), bf16hi(v.y));
    o[2] = pk2(bf16lo(v.z), bf16hi(v.z));
    o[3] = pk2(bf16lo(v.w), bf16hi(v.w));
  }
};
template <>
struct Pairs<float> {
  static constexpr int NP = 2;
  __device__ static __forceinline__ void make(const uint4& v, f2_t (&o)[2]) {
    o[0] = pk2(__uint_as_float(v.x), __uint_as_float(v.y));
    o[1] = pk2(__uint_as_float(v.z), __uint_as_float(v.w));
  }
};

// Per-thread accumulators of one row slice, as pairs (even / odd entries).
struct Acc2 {
  f2_t S, A, St, B0, B1, B2;
  __device__ __forceinline__ void reset() {
    S = A = St = B0 = B1 = B2 = 0ull;   // the bit pattern of {0.f, 0.f}
  }
};

// Teacher pairs per 16-byte piece whose exponential is evaluated on the FMA pipe: one of the four
// pairs of a bf16 piece (more than that and the FMA/ALU pipes become the limit, measured); none
// for fp32 logits, whose sweep has half the exponentials per byte and a 1e-5 tolerance.
template <typename T>
__host__ __device__ constexpr int kPolyPairs() { return sizeof(T) == 2 ? 1 : 0; }

// Sweep 1, rows whose gradient is written: e = 2^(z log2e - ref_s), delta = z - u uncentred.
// The first PT teacher pairs of a piece take their exponential from the polynomial (the teacher
// sum only enters through its logarithm, and delta still sees the unclamped logits).
template <int NP, int PT>
__device__ __forceinline__ void acc_grad(const f2_t (&Z)[NP], const f2_t (&U)[NP], f2_t nrefs,
                                         f2_t nreft, Acc2& a) {
  const f2_t L2 = splat2(kLog2e), NEG1 = splat2(-1.f);
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    const f2_t E = ex2_2(fma2(Z[i], L2, nrefs));
    const f2_t D = fma2(U[i], NEG1, Z[i]);
    a.S = add2(a.S, E);
    a.A = fma2(E, D, a.A);
    const f2_t xt = fma2(U[i], L2, nreft);
    a.St = add2(a.St, (i < PT) ? ex2_poly2(xt) : ex2_2(xt));
  }
}

// The same with delta centred on -ndref.
template <int NP>
__device__ __forceinline__ void acc_grad_centred(const f2_t (&Z)[NP], const f2_t (&U)[NP], f2_t nrefs, f2_t nreft,
                                                 f2_t ndref, Acc2& a) {
  const f2_t L2 = splat2(kLog2e), NEG1 = splat2(-1.f);
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    const f2_t E = ex2_2(fma2(Z[i], L2, nrefs));
    const f2_t D = add2(fma2(U[i], NEG1, Z[i]), ndref);
    a.S = add2(a.S, E);
    a.A = fma2(E, D, a.A);
    a.St = add2(a.St, ex2_2(fma2(U[i], L2, nreft)));
  }
}

template <typename TOut, int NP>
__device__ __forceinline__ void store_pairs(char* dst, const f2_t (&G)[NP]) {
  float g[2 * NP];
#pragma unroll
  for (int i = 0; i < NP; ++i) upk2(G[i], g[2 * i], g[2 * i + 1]);
  if (sizeof(TOut) == 4) {
    float4* o = reinterpret_cast<float4*>(dst);
#pragma unroll
    for (int j = 0; j < NP / 2; ++j)
      __stcs(o + j, make_float4(g[4 * j], g[4 * j + 1], g[4 * j + 2], g[4 * j + 3]));
  } else if (NP == 4) {
    uint4 o;
    o.x = pack_bf16x2(g[0], g[1]);
    o.y = pack_bf16x2(g[2], g[3]);
    o.z = pack_bf16x2(g[4], g[5]);
    o.w = pack_bf16x2(g[6], g[7]);
    __stcs(reinterpret_cast<uint4*>(dst), o);
  } else {
    uint2 o;
    o.x = pack_bf16x2(g[0], g[1]);
    o.y = pack_bf16x2(g[2], g[3]);
    __stcs(reinterpret_cast<uint2*>(dst), o);
  }
}

// The two logits at the sampled token (at element 0 when the token is out of range).
template <typename TIn>
__device__ __forceinline__ void fetch_logits_at(const KlParams& p, int64_t r, int y, float& zy,
                                                float& uy) {
  const bool ok = (y >= 0) && ((int64_t)y < p.V);
  const int64_t yi = ok ? y : 0;
  zy = Elem<TIn>::load1(static_cast<const char*>(p.student) + (size_t)r * p.ld * sizeof(TIn), yi);
  uy = Elem<TIn>::load1(static_cast<const char*>(p.teacher) + (size_t)r * p.ld * sizeof(TIn), yi);
}

// Fixed-order sum over the lanes of a warp; every lane returns the same bits.
__device__ __forceinline__ float lane_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Rows that do not start or end on a 16-byte boundary (RAG): the pieces are those of the aligned
// span that covers the row, `shift` entries of the first piece belong to the row before (or to
// padding) and so may the end of the last one.  Reading them is harmless -- a 16-byte granule that
// holds an entry of the row is always readable -- and their values are replaced by one whose
// exponential is zero on both sides.
template <typename TIn>
__device__ __forceinline__ void mask_piece(uint4& z, uint4& u, int e0, int e1) {
  constexpr int N = Elem<TIn>::N;
  uint32_t zw[4] = {z.x, z.y, z.z, z.w}, uw[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
  for (int e = 0; e < N; ++e) {
    if (e >= e0 && e < e1) continue;
    if (sizeof(TIn) == 4) {
      zw[e % 4] = uw[e % 4] = 0xf149f2cau;             // -1e30f
    } else {
      const uint32_t keep = (e & 1) ? 0x0000ffffu : 0xffff0000u, put = (e & 1) ? 0xf1490000u : 0xf149u;
      zw[(e / 2) % 4] = (zw[(e / 2) % 4] & keep) | put;  // bf16 -1e30
      uw[(e / 2) % 4] = (uw[(e / 2) % 4] & keep) | put;
    }
  }
  z = make_uint4(zw[0], zw[1], zw[2], zw[3]);
  u = make_uint4(uw[0], uw[1], uw[2], uw[3]);
}

// Where a row lies in this CTA's slice.
struct RowSpan {
  int pieces;        // pieces of the slice
  int shift;         // entries of piece 0 that precede the row
  int first, last;   // slice-relative index of the row's first / last piece if it is partial, else -1
  int last_n;        // entries of the row in its last piece (counted from the piece's start)
  __device__ __forceinline__ int e0(int piece) const { return piece == first ? shift : 0; }
};

}  // namespace adwin
