// Fused LM-head form of the windowed OPD divergence: the two policies of Eq. 2 are given as hidden
// states times an output embedding, z = H_s W_s^T and u = H_t W_t^T.
//
//   plan      compact order of the processed positions: rows with gradient first, then the rest
//             (or, for the weight-space audit, one segment per candidate bin), 128 rows per tile
//   gather    compact zero-padded copies of the hidden states, the two logits at the sampled token
//   sweep     per (pair of tiles, vocabulary group): 256 x 256 logit tiles of both policies from
//             tcgen05.mma on CTA pairs into tensor memory, read back with tcgen05.ld and folded
//             into online log-sum-exp / KL / squared-norm moments; one partial record per (row,
//             group, column half).  For rows with gradient the fp32 logits of a block of tiles are
//             also left in a scratch buffer
//   merge     partial records -> per-token kl, logratio, gsq, lse (float64 combination) and the
//             per-row coefficients of the gradient
//   gradient  the block's logits -> G = alpha p (d - KL)  or  alpha c (e_y - p)  (Eq. 2 / Eq. 4), bf16
//   dH, dW    dH_s = G W_s and dW_s = G^T H_s as two tensor-core GEMMs over G (tc_gemm.cu)
//
// Without a gradient, all that is ever in memory is one 128 x 256 tile of student logits per CTA (19 MB).
// With one, the fp32 logits of a block of tiles are in the scratch buffer at a time (kKeepBytes: 5120
// positions at V = 151 936; the logits of a call of no more are all there at once).  Keeping them for those few
// milliseconds replaces a second pass of both products: 8 bytes written and read again per logit
// pair against 2 (d_s + d_t) operations.  A long run is bound by the board's 1 kW, so what counts is
// energy: at 34 816 rows, V = 151 936, d = 2048 + 2560 a call takes 87 ms (sweep 38, gradient 10,
// dH 15, dW 17) where computing the products twice on single-CTA tiles took 123 ms (40 + 43 + 17 +
// 19).  At 225 rows, V = 32 000, d = 1024 + 1536: 212 us against 893 us (groups chosen by size, rows
// packed across sequences, dH's contraction split).
#include <cuda_bf16.h>

#include "adwin_common.cuh"
#include "adwin_internal.h"
#include "tc_pipeline.cuh"

namespace adwin {
namespace {

using namespace tc;

constexpr int kRecFields = 8;    // m2s, S, A, B0, B1, B2, m2t, St
constexpr int kTokFields = 4;    // z_y, u_y, has_y, unused
constexpr int kInfoFields = 8;   // L2s, a1, a0, gy, y (bits), unused x3
// Logit value given to the columns past the vocabulary in the last tile: far enough below any
// real logit that its exponential is exactly zero against a real row maximum, and small enough
// that the rounding residual of z*log2e against the running reference stays a fraction of one
// (a partial that sees only such columns keeps finite sums and merges with weight 2^-huge = 0).
constexpr float kMasked = -1.0e6f;
// Scratch for the logits of one block of tiles, or of one pair of tiles where that is more (V above
// 3 million).  Large enough that a block fills the GPU several
// times over (40 tiles at V = 151 936: 7 blocks for 34 816 rows), small beside G.
constexpr size_t kKeepBytes = size_t(6) << 30;
constexpr int kKeepArray = kBM * kBN / 4;            // float4 of one policy's 128 x 256 tile
constexpr size_t kKeepTileChunk = (size_t)2 * kKeepArray * 16;
constexpr int kMaxCand = 16;
constexpr int kMaxSeg = kMaxCand + 1;

// ---------------------------------------------------------------------------- workspace
struct LmLayout {
  size_t off_rowmap, off_hdr, off_seg, off_rowsrc, off_rowdst, off_info, off_tok, off_part, off_park,
      off_hs, off_ht, off_keep, off_q, off_G, off_pieces, total;
  int64_t max_tiles, block_tiles, part_slots;
  int n_chunks, grad_groups;
  int64_t ldG;
};

// n_seg segments of compact rows, each padded to a multiple of seg_pad rows.
LmLayout lm_layout(int64_t B, int64_t T, int64_t V, int64_t ds, int64_t dt, int64_t max_rows,
                   bool want_grad, int n_seg, int seg_pad, int sm_count) {
  auto up = [](size_t x) { return (x + 1023) & ~size_t(1023); };
  LmLayout L;
  int64_t bound = B * T;
  if (max_rows > 0 && max_rows < bound) bound = max_rows;
  bound += (int64_t)n_seg * (seg_pad - 1);
  L.max_tiles = (bound + kBM - 1) / kBM;
  if (L.max_tiles < 1) L.max_tiles = 1;
  L.n_chunks = (int)((V + kBN - 1) / kBN);
  L.ldG = (V + 7) / 8 * 8;
  // equal blocks of an even number of tiles
  int64_t most = (int64_t)(kKeepBytes / ((size_t)L.n_chunks * kKeepTileChunk)) & ~int64_t(1);
  if (most < 2) most = 2;
  const int64_t blocks = (L.max_tiles + most - 1) / most;
  L.block_tiles = ((L.max_tiles + blocks - 1) / blocks + 1) & ~int64_t(1);
  // column groups of the gradient kernel: four blocks per SM and more, 32 groups at least
  int64_t gg = (4 * (int64_t)sm_count + L.block_tiles - 1) / L.block_tiles;
  if (gg < 32) gg = 32;
  L.grad_groups = (int)(gg < L.n_chunks ? gg : L.n_chunks);
  // see lm_sweep_kernel: at most 8 groups per tile, or 8 items per pair of CTAs
  L.part_slots = 8 * (L.max_tiles + 2) + 8 * (int64_t)sm_count;
  const size_t rows = (size_t)L.max_tiles * kBM;
  size_t o = 0;
  L.off_rowmap = o;  o = up(o + workspace_layout(B).total_ext);
  L.off_hdr = o;     o = up(o + 1024);
  L.off_seg = o;     o = up(o + (size_t)n_seg * (B + 1) * 8);
  L.off_rowsrc = o;  o = up(o + rows * 4);
  L.off_rowdst = o;  o = up(o + rows * 4);
  L.off_info = o;    o = up(o + rows * kInfoFields * 4);
  L.off_tok = o;     o = up(o + rows * kTokFields * 4);
  L.off_part = o;    o = up(o + (size_t)L.part_slots * 2 * kRecFields * kBM * 4);
  L.off_park = o;    o = up(o + (size_t)sm_count * kKeepArray * 16);
  L.off_hs = o;      o = up(o + rows * (size_t)ds * 2);
  L.off_ht = o;      o = up(o + rows * (size_t)dt * 2);
  L.off_keep = o;    if (want_grad) o = up(o + (size_t)L.block_tiles * L.n_chunks * kKeepTileChunk);
  L.off_q = o;       if (want_grad) o = up(o + rows * (size_t)L.grad_groups * 2 * 4);
  L.off_G = o;       if (want_grad) o = up(o + rows * (size_t)L.ldG * 2);
  L.off_pieces = o;  if (want_grad) o = up(o + tc_gemm_scratch_bytes());
  L.total = o;
  return L;
}

// ---------------------------------------------------------------------------- plan and gather
// Device header, filled by the gather kernel's first block (n_groups: by the sweep).
struct LmHeader {
  int32_t tiles;                    // tiles of processed rows
  int32_t grad_tiles;               // the leading tiles that hold gradient rows
  int32_t n_groups;                 // vocabulary groups of the latest sweep
  int32_t unused;
  uint32_t pace[60];                // one counter per tensor-core launch
  int32_t seg_kblock[kMaxSeg + 1];  // first 64-row block of every segment
};
static_assert(sizeof(LmHeader) <= 1024, "header too large");

// The compact order: segment 0, segment 1, ..., each in sequence order.  Without cuts (n_seg = 2)
// segment 0 holds the positions with gradient (t < E_b, none unless want_grad) and segment 1 the
// rest of the processed range; with cuts segment i holds the positions in [cut[i-1], cut[i]).
struct SegPlan {
  int n_seg, pad, want_grad, by_cut;
  int32_t cut[kMaxCand];
  __device__ __forceinline__ void range(int i, int E, int P, int& lo, int& hi) const {
    if (by_cut) {
      lo = i == 0 ? 0 : cut[i - 1];
      hi = i == n_seg - 1 ? P : cut[i];
    } else {
      const int g = want_grad ? E : 0;
      lo = i == 0 ? 0 : g;
      hi = i == 0 ? g : P;
    }
    lo = lo < P ? lo : P;
    hi = hi < P ? hi : P;
  }
};

// Exclusive prefix sums over the sequences of every segment's row counts; block i = segment i.
__global__ void __launch_bounds__(1024) lm_plan_kernel(const int32_t* __restrict__ range,
                                                       const int32_t* __restrict__ ewin, int64_t B,
                                                       const SegPlan plan, int64_t* seg) {
  chain();
  __shared__ int64_t part[32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int64_t* out = seg + (int64_t)blockIdx.x * (B + 1);
  int64_t base = 0;
  for (int64_t b0 = 0; b0 < B; b0 += 1024) {
    const int64_t b = b0 + tid;
    int64_t n = 0;
    if (b < B) {
      int lo, hi;
      plan.range(blockIdx.x, ewin[b], range[b], lo, hi);
      n = hi - lo;
    }
    int64_t x = n;   // inclusive scan of the warp
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int64_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) part[warp] = x;
    __syncthreads();
    int64_t before = 0, all = 0;
    for (int w = 0; w < 32; ++w) {
      if (w < warp) before += part[w];
      all += part[w];
    }
    if (b < B) out[b] = base + before + x - n;
    base += all;
    __syncthreads();
  }
  if (tid == 0) out[B] = base;
}

struct GatherParams {
  const __nv_bfloat16* hs;
  const __nv_bfloat16* ht;
  const __nv_bfloat16* ws;
  const __nv_bfloat16* wt;
  const int32_t* tokens;
  const int32_t* range;
  const int32_t* ewin;
  const int64_t* seg;
  int64_t B, T, V, ds, dt, max_tiles;
  LmHeader* hdr;
  int32_t* rowsrc;
  int32_t* rowdst;
  float* tok;
  __nv_bfloat16* hs_c;
  __nv_bfloat16* ht_c;
  int32_t* status;
};

constexpr int kGatherThreads = 128;

// Copies one hidden-state row (d % 8 == 0) and forms this thread's share of its fp32 dot product
// with an embedding row.
__device__ __forceinline__ float copy_dot(const __nv_bfloat16* src, const __nv_bfloat16* w,
                                          __nv_bfloat16* dst, int64_t d) {
  float acc = 0.f;
#pragma unroll 2
  for (int64_t v = threadIdx.x; v < d / 8; v += kGatherThreads) {
    uint4 x = make_uint4(0u, 0u, 0u, 0u);
    if (src) x = __ldg(reinterpret_cast<const uint4*>(src) + v);
    if (w) {
      const uint4 y = __ldg(reinterpret_cast<const uint4*>(w) + v);
      float xf[8], yf[8];
      Elem<__nv_bfloat16>::unpack(x, xf);
      Elem<__nv_bfloat16>::unpack(y, yf);
#pragma unroll
      for (int i = 0; i < 8; ++i) acc = fmaf(xf[i], yf[i], acc);
    }
    reinterpret_cast<uint4*>(dst)[v] = x;
  }
  return acc;
}

// One block per compact row: which position it is, copies of its two hidden-state rows (zeros past
// the rows), and the two logits at its sampled token, z_y = h_s . W_s[y] and u_y = h_t . W_t[y].
// They give the sampled-token log-ratio of Section 2.3 without a search through the logit tiles, and
// their difference is the value the sweep centres z - u on: on a peaked row the sampled token is
// almost surely the peak, where the centred difference is then exactly zero, which keeps the
// single-sweep squared-norm moments well conditioned.
// OWN: every block forms the prefix sums itself, in shared memory, which for a short call costs less than a
// launch of lm_plan_kernel and round trips to memory for the search below, but each block pays for every segment
// of every sequence, and beyond about ten blocks per SM they take turns.  Whole calls at V = 8 192, d = 512, by the two
// kernels / so: two segments of 2 sequences, 512 rows 82.0 / 80.4 us, 1 400 121.6 / 119.3, 1 536 125.6 / 126.4; of 128
// sequences, 512 rows 83.5 / 82.0, 1 280 120.5 / 119.3; seven segments of 16 sequences, 640 rows 127.0 / 123.7, 1 440
// 154.4 / 155.5; of 64, 1 280 rows 149.9 / 153.2; of 128, 512 rows 119.7 / 123.1, 1 280 157.7 / 170.2.
constexpr int kGatherSeqs = 128;
constexpr int64_t kGatherOwnRows = 1408;      // (without the segments' padding)
constexpr int64_t kGatherOwnSums = 256;       // segments times sequences
template <bool OWN>
__global__ void __launch_bounds__(kGatherThreads) lm_gather_kernel(const GatherParams p, const SegPlan plan) {
  chain();
  __shared__ int64_t base[kMaxSeg + 1];
  __shared__ float red[2][kGatherThreads / 32];
  __shared__ int64_t own[OWN ? kMaxSeg : 1][OWN ? kGatherSeqs + 1 : 1];
  if (OWN) {
    const int lane = threadIdx.x & 31;
    for (int i = threadIdx.x >> 5; i < plan.n_seg; i += kGatherThreads / 32) {   // a warp per segment
      int64_t before = 0;
      for (int b0 = 0; b0 < p.B; b0 += 32) {
        int64_t n = 0;
        if (b0 + lane < p.B) {
          int lo, hi;
          plan.range(i, p.ewin[b0 + lane], p.range[b0 + lane], lo, hi);
          n = hi - lo;
        }
        int64_t x = n;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int64_t y = __shfl_up_sync(0xffffffffu, x, o);
          if (lane >= o) x += y;
        }
        if (b0 + lane < p.B) own[i][b0 + lane] = before + x - n;
        before += __shfl_sync(0xffffffffu, x, 31);
      }
      if (lane == 0) own[i][p.B] = before;
    }
    __syncthreads();
  }
  auto offsets = [&](int i) { return OWN ? own[i] : p.seg + (int64_t)i * (p.B + 1); };
  if (threadIdx.x == 0) {
    int64_t o = 0;
    for (int i = 0; i < plan.n_seg; ++i) {
      base[i] = o;
      o += (offsets(i)[p.B] + plan.pad - 1) / plan.pad * plan.pad;
    }
    base[plan.n_seg] = o;
  }
  __syncthreads();
  const int64_t rows = base[plan.n_seg];
  const int64_t grad_rows = plan.by_cut ? rows : base[1];
  int64_t tiles = (rows + kBM - 1) / kBM;
  const bool fits = tiles <= p.max_tiles;
  if (!fits) tiles = 0;
  if (blockIdx.x == 0) {
    if (threadIdx.x == 0) {
      if (!fits) atomicOr(p.status, ADWIN_DEV_WORKSPACE);   // more rows than the workspace is for
      p.hdr->tiles = (int32_t)tiles;
      p.hdr->grad_tiles = fits ? (int32_t)((grad_rows + kBM - 1) / kBM) : 0;
    }
    if (threadIdx.x < 60) p.hdr->pace[threadIdx.x] = 0u;
    if (threadIdx.x <= plan.n_seg)
      p.hdr->seg_kblock[threadIdx.x] = fits ? (int32_t)(base[threadIdx.x] / 64) : 0;
  }
  for (int64_t r = blockIdx.x; r < tiles * kBM; r += gridDim.x) {
    int64_t src = -1;
    if (r < rows) {
      int i = 0;
      while (r >= base[i + 1]) ++i;
      const int64_t* off = offsets(i);
      const int64_t k = r - base[i];
      if (k < off[p.B]) {
        int64_t b = 0, e = p.B;   // the last sequence with off[b] <= k
        while (e - b > 1) {
          const int64_t m = (b + e) / 2;
          if (off[m] <= k) b = m; else e = m;
        }
        int lo, hi;
        plan.range(i, p.ewin[b], p.range[b], lo, hi);
        src = b * p.T + lo + (k - off[b]);
      }
    }
    if (!ADWIN_CHK(src < p.B * p.T && r < p.max_tiles * kBM, p.status)) continue;   // (uniform)
    const int y = src >= 0 ? p.tokens[src] : -1;
    const bool has = y >= 0 && y < p.V;
    const float zp = warp_sum(copy_dot(src >= 0 ? p.hs + src * p.ds : nullptr,
                                       has ? p.ws + (int64_t)y * p.ds : nullptr, p.hs_c + r * p.ds, p.ds));
    const float up = warp_sum(copy_dot(src >= 0 ? p.ht + src * p.dt : nullptr,
                                       has ? p.wt + (int64_t)y * p.dt : nullptr, p.ht_c + r * p.dt, p.dt));
    if ((threadIdx.x & 31) == 0) {
      red[0][threadIdx.x >> 5] = zp;
      red[1][threadIdx.x >> 5] = up;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      float zy = 0.f, uy = 0.f;
      for (int w = 0; w < kGatherThreads / 32; ++w) {
        zy += red[0][w];
        uy += red[1][w];
      }
      p.rowsrc[r] = (int32_t)src;
      p.rowdst[r] = r < grad_rows ? (int32_t)src : -1;
      *reinterpret_cast<float4*>(p.tok + r * kTokFields) = make_float4(zy, uy, has ? 1.f : 0.f, 0.f);
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------- sweep kernel
struct SweepParams {
  LmHeader* hdr;
  const float* tok;             // z_y, u_y per compact row
  int64_t V;
  int ks_blocks, kt_blocks;     // k-blocks of the student / teacher contraction
  int n_chunks;
  int64_t tile0;                // first tile of this launch (unused with rest = 1)
  int64_t tile_cap;             // tiles of this launch, at most
  int rest;                     // 0: gradient tiles, 1: the tiles behind them, 2: all tiles
  float4* keep;                 // logits of the launch's tiles (null: not kept)
  int keep_u;                   // the teacher's as well
  float4* park;                 // one student tile per CTA (when nothing is kept)
  float* part;                  // partial records
  int64_t part_slots;
  unsigned int* pace;
  uint64_t limit_ns;            // limit of the handshake waits
  int32_t* status;
};

// The tiles [lo, hi) of a launch.
__device__ __forceinline__ void launch_tiles(const LmHeader* hdr, int64_t tile0, int64_t cap, int rest,
                                             int64_t& lo, int64_t& hi) {
  const int64_t all = rest ? hdr->tiles : hdr->grad_tiles;
  lo = rest == 1 ? hdr->grad_tiles : tile0;
  hi = lo + cap < all ? lo + cap : all;
  if (hi < lo) hi = lo;
}

// Cost of cutting the vocabulary into g groups, in quarter chunks: rounds of items over the pairs
// of CTAs times the chunks of an item (plus a quarter for its records).
__device__ __forceinline__ unsigned int group_cost(int64_t units, int n_chunks, int pairs, int g) {
  return (unsigned int)((units * g + pairs - 1) / pairs * (4 * ((n_chunks + g - 1) / g) + 1));
}

// chunk range of vocabulary group g
__device__ __forceinline__ void group_chunks(int n_chunks, int n_groups, int g, int& c0, int& c1) {
  c0 = (int)((int64_t)n_chunks * g / n_groups);
  c1 = (int)((int64_t)n_chunks * (g + 1) / n_groups);
}

// Statistics of 256 x 256 logit tiles on CTA pairs (this CTA: 128 of the rows).  The student
// product of a chunk goes to accumulator slot 0, the teacher product to slot 1.  The epilogue takes
// the student tile out of tensor memory as soon as it is complete, while the teacher product runs,
// and parks it in global memory (L2; the same thread reads it back), so the MMAs never wait for
// the arithmetic, which runs on the teacher tile during the next chunk's student product.
// MOMENTS = false drops the squared-norm moments (when every processed row gets its gsq from the
// gradient entries, or no gsq is asked for).
template <bool MOMENTS>
__global__ void __launch_bounds__(kThreads, 1)
lm_sweep_kernel(const __grid_constant__ CUtensorMap map_hs, const __grid_constant__ CUtensorMap map_ws,
                const __grid_constant__ CUtensorMap map_ht, const __grid_constant__ CUtensorMap map_wt,
                const SweepParams p) {
  chain_wait();
  extern __shared__ uint8_t smem_raw[];
  __shared__ unsigned long long s_best;
  Ctrl* ctrl = reinterpret_cast<Ctrl*>(smem_raw);
  const uint32_t stage0 = (smem_addr(smem_raw) + kCtrlBytes + 1023u) & ~1023u;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  volatile int* abort = &ctrl->abort;
  const uint32_t rank = cluster_ctarank();   // 0: the CTA that issues the MMAs
  const int pair = blockIdx.x / 2, pairs = gridDim.x / 2;

  int64_t lo, hi;
  launch_tiles(p.hdr, p.tile0, p.tile_cap, p.rest, lo, hi);
  const int64_t units = (hi - lo + 1) / 2;   // pairs of tiles
  if (threadIdx.x == 0) {
    s_best = ~0ull;
    pair_bars_init(ctrl);
  }
  if (warp == 2) {
    tmem_alloc_pair(smem_addr(&ctrl->tmem_base), kTmemCols);
    tmem_relinquish_pair();
    tc_fence_before_sync();
  }
  __syncthreads();
  // The number of vocabulary groups: the cheapest cut within the record buffer.  (With 8 groups
  // throughout, a call of 225 rows at V = 32 000 had 24 items for 148 SMs.)
  if (units > 0) {
    int64_t most = 4 * pairs / units;
    if (most < 8) most = 8;
    if (most > p.n_chunks) most = p.n_chunks;
    for (int g = 1 + (int)threadIdx.x; g <= most; g += kThreads)
      atomicMin(&s_best, ((unsigned long long)group_cost(units, p.n_chunks, pairs, g) << 32) | (unsigned)g);
  }
  __syncthreads();
  cluster_sync();   // the partner's barriers exist before anything signals them
  tc_fence_after_sync();
  const uint32_t tmem_base = ctrl->tmem_base;
  const int n_groups = units > 0 ? (int)(s_best & 0xffffffffu) : 1;
  if (blockIdx.x == 0 && threadIdx.x == 0) p.hdr->n_groups = n_groups;
  const int64_t n_items = units * n_groups;

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    if (lane == 0) {
      uint32_t it = 0;
      bool ok = true;
      Pace pace(rank == 0 ? p.pace : nullptr, pairs);
      for (int64_t item = pair; ok && item < n_items; item += pairs) {
        const int row0 = (int)(lo + 2 * (item / n_groups) + rank) * kBM;
        int c0, c1;
        group_chunks(p.n_chunks, n_groups, (int)(item % n_groups), c0, c1);
        for (int c = c0; ok && c < c1; ++c) {
          for (int pass = 0; ok && pass < 2; ++pass) {
            const CUtensorMap* ma = pass ? &map_ht : &map_hs;
            const CUtensorMap* mb = pass ? &map_wt : &map_ws;
            const int nk = pass ? p.kt_blocks : p.ks_blocks;
            for (int kb = 0; kb < nk; ++kb, ++it) {
              const uint32_t s = it % kPairStages, ph = (it / kPairStages) & 1;
              pace.kblock(it);
              if (!bar_wait(smem_addr(&ctrl->empty[s]), ph ^ 1, abort, p.limit_ns)) { ok = false; break; }
              const uint32_t bar = smem_addr(&ctrl->full[s]);
              const uint32_t a = stage0 + s * kPairStageBytes, b = a + kABytes;
              if (rank == 0) bar_expect_tx(bar, 2 * kPairStageBytes);   // both CTAs' bytes
              const uint32_t bar0 = map_to_cta(bar, 0);
              load_operand_pair<false>(a, ma, row0, kb * kBK, bar0);
              load_operand_pair<false>(b, mb, c * kBN + (int)rank * (kBN / 2), kb * kBK, bar0);
            }
          }
        }
      }
      pace.done();
      if (!ok && rank == 0) pair_drain_loads(ctrl, it);
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    if (lane == 0 && rank == 0) {
      uint32_t it = 0, acc_it = 0;
      bool ok = true;
      for (int64_t item = pair; ok && item < n_items; item += pairs) {
        int c0, c1;
        group_chunks(p.n_chunks, n_groups, (int)(item % n_groups), c0, c1);
        for (int c = c0; ok && c < c1; ++c, ++acc_it) {
          for (int pass = 0; ok && pass < 2; ++pass) {
            if (!bar_wait(smem_addr(&ctrl->acc_empty[pass]), (acc_it & 1) ^ 1, abort, p.limit_ns)) { ok = false; break; }
            tc_fence_after_sync();
            const int nk = pass ? p.kt_blocks : p.ks_blocks;
            for (int kb = 0; kb < nk; ++kb, ++it) {
              const uint32_t s = it % kPairStages, ph = (it / kPairStages) & 1;
              if (!bar_wait(smem_addr(&ctrl->full[s]), ph, abort, p.limit_ns)) { ok = false; break; }
              tc_fence_after_sync();
              const uint32_t a = stage0 + s * kPairStageBytes, b = a + kABytes;
              issue_kblock_pair<false, false>(tmem_base + pass * kBN, a, b, kb == 0);
              umma_commit_pair(smem_addr(&ctrl->empty[s]));
            }
            if (ok) umma_commit_pair(smem_addr(&ctrl->acc_full[pass]));
          }
        }
      }
      if (!ok) {   // give up: wait until the MMAs already issued have retired
        umma_commit_pair(smem_addr(&ctrl->drain));
        bar_wait_drain(smem_addr(&ctrl->drain), 0);
      }
    }
  } else if (warp >= kEpiWarp0) {
    // ------------------------------------------------------------------ epilogue
    const int ew = warp - kEpiWarp0;
    const int quad = warp & 3;               // TMEM lanes 32*quad .. 32*quad+31
    const int half = ew >> 2;                // columns half*128 .. half*128+127 of the tile
    const int row = quad * 32 + lane;
    const uint32_t t_lane = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(half * 128);
    uint32_t acc_it = 0;
    bool ok = true;
    for (int64_t item = pair; ok && item < n_items; item += pairs) {
      const int64_t tile = lo + 2 * (item / n_groups) + rank;
      const int g = (int)(item % n_groups);
      const bool live = tile < hi;     // the last pair's second tile may not exist
      int c0, c1;
      group_chunks(p.n_chunks, n_groups, g, c0, c1);
      RowAcc acc;
      acc.reset();
      float dref = 0.f;
      if (live) {
        const float* tk = p.tok + (tile * kBM + row) * kTokFields;
        dref = tk[0] - tk[1];      // centre of z - u for this row: the sampled token's difference
      }
      for (int c = c0; ok && c < c1; ++c, ++acc_it) {
        // this thread's place in the 128 x 256 tile: [64 groups of 4 columns][128 rows]
        float4* zp = (p.keep ? p.keep + ((tile - lo) * p.n_chunks + c) * (2 * kKeepArray)
                             : p.park + (int64_t)blockIdx.x * kKeepArray) +
                     (half * 32) * kBM + row;
        if (!__all_sync(0xffffffffu, bar_wait(smem_addr(&ctrl->acc_full[0]), acc_it & 1, abort, p.limit_ns))) {
          ok = false;   // the same decision in every lane: tcgen05.ld below is warp-collective
          break;
        }
        tc_fence_after_sync();
#pragma unroll 1
        for (int j = 0; j < 4; ++j) {
          uint32_t r[32];
          tmem_ld32(t_lane + j * 32, r);
          tmem_ld_wait();
          if (live) {
#pragma unroll
            for (int i = 0; i < 8; ++i)
              zp[(j * 8 + i) * kBM] =
                  make_float4(__uint_as_float(r[4 * i]), __uint_as_float(r[4 * i + 1]),
                              __uint_as_float(r[4 * i + 2]), __uint_as_float(r[4 * i + 3]));
          }
        }
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) pair_release(&ctrl->acc_empty[0], rank);

        if (!__all_sync(0xffffffffu, bar_wait(smem_addr(&ctrl->acc_full[1]), acc_it & 1, abort, p.limit_ns))) {
          ok = false;
          break;
        }
        tc_fence_after_sync();
        const int64_t col_base = (int64_t)c * kBN + half * 128;
        const bool ragged = col_base + 128 > p.V;
#pragma unroll 1
        for (int j = 0; j < 4; ++j) {
          uint32_t ur[32];
          float z[32], u[32];
          if (live) {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              const float4 x = zp[(j * 8 + i) * kBM];
              z[4 * i] = x.x;
              z[4 * i + 1] = x.y;
              z[4 * i + 2] = x.z;
              z[4 * i + 3] = x.w;
            }
          }
          tmem_ld32(t_lane + kBN + j * 32, ur);
          tmem_ld_wait();
          if (!live) continue;
#pragma unroll
          for (int i = 0; i < 32; ++i) u[i] = __uint_as_float(ur[i]);
          if (p.keep && p.keep_u) {
#pragma unroll
            for (int i = 0; i < 8; ++i)
              zp[kKeepArray + (j * 8 + i) * kBM] =
                  make_float4(u[4 * i], u[4 * i + 1], u[4 * i + 2], u[4 * i + 3]);
          }
          if (ragged) {   // columns past the vocabulary: exp -> 0, z - u -> 0
            const int64_t col = col_base + j * 32;
#pragma unroll
            for (int i = 0; i < 32; ++i)
              if (col + i >= p.V) {
                z[i] = kMasked;
                u[i] = kMasked;
              }
          }
          acc_piece<32, MOMENTS, false>(z, u, dref, acc);   // (kMasked: see there)
        }
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) pair_release(&ctrl->acc_empty[1], rank);
      }
      const int64_t slot = (tile - lo) * n_groups + g;
      if (ok && live && ADWIN_CHK(slot < p.part_slots, p.status)) {
        float* o = p.part + ((slot * 2 + half) * kRecFields) * kBM + row;
        o[0 * kBM] = acc.m2s;
        o[1 * kBM] = acc.S;
        o[2 * kBM] = acc.A;
        o[3 * kBM] = acc.B0;
        o[4 * kBM] = acc.B1;
        o[5 * kBM] = acc.B2;
        o[6 * kBM] = acc.m2t;
        o[7 * kBM] = acc.St;
      }
    }
  }
  if (*abort && threadIdx.x == 0) {
    atomicOr(p.status, ADWIN_DEV_TIMEOUT);
    store_cluster_u32(map_to_cta(smem_addr(&ctrl->abort), rank ^ 1u), 1u);   // partner too
  }
  tc_fence_before_sync();
  __syncthreads();
  cluster_sync();   // neither CTA leaves while the other may still use its memory
  if (warp == 2) {
    tc_fence_after_sync();
    tmem_dealloc_pair(tmem_base, kTmemCols);
  }
}

// ---------------------------------------------------------------------------- merge kernel
struct MergeParams {
  const LmHeader* hdr;
  const int32_t* rowsrc;
  const int32_t* rowdst;
  const int32_t* tokens;
  const float* part;
  const float* tok;
  float* info;
  int64_t tile0, tile_cap;
  int rest;
  float alpha;
  int mode;
  float* kl;
  float* logratio;
  float* gsq;
  float* lse_s;
  float* lse_t;
  int32_t* status;
};

// Block = ROWS compact rows, 1024 / ROWS threads per row: combine the partial records of the row in float64
// against common references (fixed order) and derive the per-token outputs and the gradient
// coefficients:
//   g_k = p_k (a1 (z_k - u_k) + a0) (+ gy at k = y),   p_k = 2^(z_k log2e - L2s);
// a row without gradient has L2s = infinity: p_k, and g_k with a1 = a0 = gy = 0, are exactly zero
// whatever its logits (with L2s = 0, p_k overflows beyond z = 88 and 0 * inf spreads over dW).
// Records are read with the row as the fast index (whole 32-byte sectors at least), reduced with the record
// as the lane.  A short call has many records (126 for each of 225 rows at V = 32 000), which is
// why the records are spread over threads, and more so with few tiles: ROWS = 8 up to two, and of many chunks
// of the vocabulary up to four.  Whole calls with 32 rows a block / with 8: V = 32 000, 128 rows
// 165.7 / 164.1 us, 256 176.9 / 175.2, 384 214.8 / 213.9, 512 226.6 / 227.2, 600 270.1 / 272.2; V = 16 000, 128 rows 91.7 /
// 90.1, 512 113.6 / 112.7; V = 8 192, 128 rows 69.1 / 67.8, 256 72.9 / 72.2, 512 77.8 / 80.4.
constexpr int kMergeRows = 32;
bool merge_by_8(int64_t tiles, int n_chunks) { return tiles <= 2 || (tiles <= 4 && n_chunks >= 48); }
template <int ROWS>
__global__ void __launch_bounds__(1024) lm_merge_kernel(const MergeParams p) {
  chain();
  constexpr int kRecs = 1024 / ROWS;   // threads per row
  __shared__ double red[6][32][ROWS];  // a value per warp and row
  int64_t lo, hi;
  launch_tiles(p.hdr, p.tile0, p.tile_cap, p.rest, lo, hi);
  const int64_t tile = lo + blockIdx.x / (kBM / ROWS);
  if (tile >= hi) return;
  const int first = blockIdx.x % (kBM / ROWS) * ROWS;
  const int row = threadIdx.x % ROWS, mine = threadIdx.x / ROWS;
  const int n = p.hdr->n_groups * 2;
  const float* rec = p.part + ((tile - lo) * n * kRecFields) * kBM + first + row;
  auto f = [&](int i, int k) { return (double)rec[((int64_t)i * kRecFields + k) * kBM]; };
  double M2s = -INFINITY, M2t = -INFINITY;
  for (int i = mine; i < n; i += kRecs) {
    M2s = fmax(M2s, f(i, 0));
    M2t = fmax(M2t, f(i, 6));
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o >= ROWS; o >>= 1) {
    M2s = fmax(M2s, __shfl_xor_sync(0xffffffffu, M2s, o));
    M2t = fmax(M2t, __shfl_xor_sync(0xffffffffu, M2t, o));
  }
  if (lane < ROWS) {
    red[0][warp][lane] = M2s;
    red[1][warp][lane] = M2t;
  }
  __syncthreads();
  M2s = red[0][0][row];
  M2t = red[1][0][row];
  for (int w = 1; w < 32; ++w) {
    M2s = fmax(M2s, red[0][w][row]);
    M2t = fmax(M2t, red[1][w][row]);
  }
  __syncthreads();
  double v[6] = {0, 0, 0, 0, 0, 0};   // S, Ac, B0, B1, B2, St
  for (int i = mine; i < n; i += kRecs) {
    const double w = exp2(f(i, 0) - M2s), w2 = w * w;
    v[0] += w * f(i, 1);
    v[1] += w * f(i, 2);
    v[2] += w2 * f(i, 3);
    v[3] += w2 * f(i, 4);
    v[4] += w2 * f(i, 5);
    v[5] += exp2(f(i, 6) - M2t) * f(i, 7);
  }
#pragma unroll
  for (int k = 0; k < 6; ++k) {
#pragma unroll
    for (int o = 16; o >= ROWS; o >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
    if (lane < ROWS) red[k][warp][lane] = v[k];
  }
  __syncthreads();
  if (warp < 6) {   // one field per warp, 32 / ROWS lanes per row
    double t = 0.0;
    for (int w = lane / ROWS; w < 32; w += 32 / ROWS) t += red[warp][w][lane % ROWS];
#pragma unroll
    for (int o = 16; o >= ROWS; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    __syncwarp();
    if (lane < ROWS) red[warp][0][lane] = t;
  }
  __syncthreads();
  if (warp != 0 || lane >= ROWS) return;
  const int64_t crow = tile * kBM + first + lane;
  const double S = red[0][0][lane], Ac = red[1][0][lane], B0 = red[2][0][lane];
  const double B1 = red[3][0][lane], B2 = red[4][0][lane], St = red[5][0][lane];

  float* inf = p.info + crow * kInfoFields;
  const int64_t r = p.rowsrc[crow];
  if (r < 0) {
    inf[0] = INFINITY; inf[1] = 0.f; inf[2] = 0.f; inf[3] = 0.f; inf[4] = __int_as_float(-1);
    return;
  }
  const float* tk = p.tok + crow * kTokFields;
  const bool has_y = tk[2] != 0.f;
  const double zy = tk[0], uy = tk[1];
  const double dref = (double)(tk[0] - tk[1]);   // the centre the sweep used (an fp32 difference)
  const double sh = -Ac / S;                   // centre minus E_p[z - u]
  const double c0 = dref - sh;                 // E_p[z - u]
  const double B2c = B2 + 2.0 * sh * B1 + sh * sh * B0;
  constexpr double kLn2 = 0.69314718055994530942;
  const double lse_s = (M2s + log2(S)) * kLn2, lse_t = (M2t + log2(St)) * kLn2;
  const double delta = lse_s - lse_t;
  const double kl = c0 - delta;
  const double c = has_y ? (zy - uy) - delta : (double)NAN;
  const double alpha = p.alpha;
  double gsq, a1, a0, gy;
  if (p.mode == ADWIN_GRAD_FULL_KL) {
    gsq = alpha * alpha * fmax(B2c, 0.0) / (S * S);
    a1 = alpha;
    a0 = -alpha * c0;
    gy = 0.0;
  } else {
    const double py = has_y ? exp2(zy * 1.4426950408889634074 - M2s) / S : (double)NAN;
    const double rest = fmax(B0 / (S * S) - py * py, 0.0);
    gsq = alpha * alpha * c * c * ((1.0 - py) * (1.0 - py) + rest);
    a1 = 0.0;
    a0 = -alpha * c;
    gy = alpha * c;
  }
  p.kl[r] = (float)kl;
  p.logratio[r] = (float)c;
  if (p.gsq) p.gsq[r] = (float)gsq;
  if (p.lse_s) p.lse_s[r] = (float)lse_s;
  if (p.lse_t) p.lse_t[r] = (float)lse_t;
  const bool in_grad = p.rowdst[crow] >= 0;
  inf[0] = in_grad ? (float)(lse_s * 1.4426950408889634074) : INFINITY;
  inf[1] = in_grad ? (float)a1 : 0.f;
  inf[2] = in_grad ? (float)a0 : 0.f;
  inf[3] = in_grad ? (float)gy : 0.f;
  inf[4] = __int_as_float(in_grad && has_y ? p.tokens[r] : -1);
  if (!has_y) atomicOr(p.status, ADWIN_DEV_TOKEN_RANGE);
  if (!(isfinite(lse_s) && isfinite(lse_t))) atomicOr(p.status, ADWIN_DEV_NONFINITE);
}

// ---------------------------------------------------------------------------- gradient kernel
struct GradParams {
  const LmHeader* hdr;
  const float4* keep;
  const float* info;
  int64_t tile0, tile_cap, V;
  int n_chunks, n_groups;       // column groups of this kernel
  __nv_bfloat16* G;
  int64_t ldG;
  float* q;                     // per-row partial sums of g^2: [tile][group][half][128]
  int64_t max_tiles;
  int32_t* status;
};

// Streams a block's kept logits once and writes G.  One item = (tile, column group); a thread owns
// one row of one 128-column half, so loads are coalesced over rows and every 32 columns of G leave
// as two full 32-byte sectors.  Bound by memory: 8 bytes read and 2 written per entry.
template <bool NEED_U>
__global__ void __launch_bounds__(256, 2) lm_grad_kernel(const GradParams p) {
  chain();
  int64_t lo, hi;
  launch_tiles(p.hdr, p.tile0, p.tile_cap, 0, lo, hi);
  const int64_t tile = lo + blockIdx.x / p.n_groups;
  const int g = blockIdx.x % p.n_groups;
  if (tile >= hi) return;
  const int row = threadIdx.x % kBM, half = threadIdx.x / kBM;
  const int64_t crow = tile * kBM + row;
  const float* inf = p.info + crow * kInfoFields;
  const float L2s = inf[0], a1 = inf[1], a0 = inf[2], gy = inf[3];
  const int y = __float_as_int(inf[4]);
  int c0, c1;
  group_chunks(p.n_chunks, p.n_groups, g, c0, c1);
  const bool sectors = p.ldG % 16 == 0;   // 32 columns of a row are two whole 32-byte sectors
  float q = 0.f;
  for (int c = c0; c < c1; ++c) {
    const float4* zp = p.keep + ((tile - lo) * p.n_chunks + c) * (2 * kKeepArray) +
                       (half * 32) * kBM + row;
    const int64_t col_base = (int64_t)c * kBN + half * 128;
#pragma unroll 1
    for (int j = 0; j < 4; ++j) {
      const int64_t col = col_base + j * 32;
      if (col >= p.V) break;
      float4 z4[8], u4[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        z4[i] = __ldcs(zp + (j * 8 + i) * kBM);
        if (NEED_U) u4[i] = __ldcs(zp + kKeepArray + (j * 8 + i) * kBM);
      }
      float v[32];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float z[4] = {z4[i].x, z4[i].y, z4[i].z, z4[i].w};
        const float u[4] = {u4[i].x, u4[i].y, u4[i].z, u4[i].w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float pz = ex2f(fmaf(z[e], kLog2e, -L2s));
          v[4 * i + e] = pz * (NEED_U ? fmaf(a1, z[e] - u[e], a0) : a0);
        }
      }
      if ((unsigned)(y - (int)col) < 32u) {   // the sampled token's own entry (Eq. 4)
        const int yi = y - (int)col;
#pragma unroll
        for (int i = 0; i < 32; ++i)
          if (i == yi) v[i] += gy;
      }
      uint32_t pk[16];
#pragma unroll
      for (int i = 0; i < 32; ++i)
        if (col + i < p.V) q = fmaf(v[i], v[i], q);
#pragma unroll
      for (int i = 0; i < 32; i += 2) pk[i >> 1] = pack_bf16x2(v[i], v[i + 1]);
      __nv_bfloat16* gp = p.G + crow * p.ldG + col;
      if (sectors && col + 32 <= p.V && ADWIN_CHK(tile < p.max_tiles && col + 32 <= p.ldG, p.status)) {
#pragma unroll
        for (int i = 0; i < 16; i += 8)
          asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(gp + 2 * i),
                       "r"(pk[i]), "r"(pk[i + 1]), "r"(pk[i + 2]), "r"(pk[i + 3]), "r"(pk[i + 4]),
                       "r"(pk[i + 5]), "r"(pk[i + 6]), "r"(pk[i + 7])
                       : "memory");
        continue;
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (col + i * 8 < p.V && ADWIN_CHK(tile < p.max_tiles && col + i * 8 + 8 <= p.ldG, p.status))
          *reinterpret_cast<uint4*>(gp + i * 8) =
              make_uint4(pk[i * 4], pk[i * 4 + 1], pk[i * 4 + 2], pk[i * 4 + 3]);
    }
  }
  p.q[((tile * p.n_groups + g) * 2 + half) * kBM + row] = q;
}

// Squared gradient norm of the rows whose gradient was formed: the sum of g_k^2 over the entries
// themselves (fixed order, float64), which replaces the single-sweep moment value there.  Block = 32
// compact rows, 32 threads per row, as in lm_merge_kernel<32>.
__global__ void __launch_bounds__(1024) lm_gsq_kernel(const LmHeader* hdr, const float* __restrict__ q,
                                                      const int32_t* __restrict__ rowdst,
                                                      int n_groups, float* gsq) {
  chain();
  __shared__ double red[32][kMergeRows];
  const int64_t tile = blockIdx.x / (kBM / kMergeRows);
  if (tile >= hdr->grad_tiles) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int row = blockIdx.x % (kBM / kMergeRows) * kMergeRows + lane;
  double acc = 0.0;
  for (int i = warp; i < n_groups * 2; i += 32)
    acc += (double)q[(tile * n_groups * 2 + i) * kBM + row];
  red[warp][lane] = acc;
  __syncthreads();
  if (warp != 0) return;
  const int32_t dst = rowdst[tile * kBM + row];
  if (dst < 0) return;
  acc = 0.0;
  for (int w = 0; w < 32; ++w) acc += red[w][lane];
  gsq[dst] = (float)acc;
}

// The pass as the plain call and the weight-space audit use it.
struct LmCall {
  const void *hs, *ws, *ht, *wt;
  int64_t B, T, V, ds, dt;
  const int32_t *tokens, *window, *rollout_len;
  float alpha;
  int mode, flags;
  void* dH;
  int dh_dtype;
  float* dW;
  bool want_grad;               // G is formed (for dH, dW or the audit)
  float *kl, *logratio, *gsq, *lse_s, *lse_t;
  char* ws_base;
  int32_t* status;
  int sm_count;
};

cudaError_t run_lmhead(const LmCall& a, const LmLayout& L, const SegPlan& plan, cudaStream_t s) {
  char* wb = a.ws_base;
  const bool range_full = (a.flags & ADWIN_RANGE_FULL) != 0;
  LmHeader* hdr = reinterpret_cast<LmHeader*>(wb + L.off_hdr);
  int64_t* seg = reinterpret_cast<int64_t*>(wb + L.off_seg);
  int32_t* rowsrc = reinterpret_cast<int32_t*>(wb + L.off_rowsrc);
  int32_t* rowdst = reinterpret_cast<int32_t*>(wb + L.off_rowdst);
  float* info = reinterpret_cast<float*>(wb + L.off_info);
  float* tok = reinterpret_cast<float*>(wb + L.off_tok);
  float* part = reinterpret_cast<float*>(wb + L.off_part);
  float* q = reinterpret_cast<float*>(wb + L.off_q);
  float4* keep = reinterpret_cast<float4*>(wb + L.off_keep);
  __nv_bfloat16* hs_c = reinterpret_cast<__nv_bfloat16*>(wb + L.off_hs);
  __nv_bfloat16* ht_c = reinterpret_cast<__nv_bfloat16*>(wb + L.off_ht);
  __nv_bfloat16* G = reinterpret_cast<__nv_bfloat16*>(wb + L.off_G);
  float* pieces = reinterpret_cast<float*>(wb + L.off_pieces);
  const int64_t rows_cap = L.max_tiles * kBM;
  const int64_t ds = a.ds, dt = a.dt, V = a.V;

  cudaError_t e = launch_rowmap(a.window, a.rollout_len, a.B, a.T,
                                a.flags & (ADWIN_RANGE_FULL | ADWIN_STATUS_INIT), wb + L.off_rowmap,
                                false, a.kl, a.logratio, a.gsq, a.lse_s, a.lse_t, a.status, s);
  if (e != cudaSuccess) return e;
  const WorkspaceLayout wl = workspace_layout(a.B);
  GatherParams gp;
  gp.hs = static_cast<const __nv_bfloat16*>(a.hs);
  gp.ht = static_cast<const __nv_bfloat16*>(a.ht);
  gp.ws = static_cast<const __nv_bfloat16*>(a.ws);
  gp.wt = static_cast<const __nv_bfloat16*>(a.wt);
  gp.tokens = a.tokens;
  gp.range = reinterpret_cast<const int32_t*>(wb + L.off_rowmap + wl.off_range);
  gp.ewin = reinterpret_cast<const int32_t*>(wb + L.off_rowmap + wl.off_ewin);
  gp.seg = seg;
  gp.B = a.B; gp.T = a.T; gp.V = V; gp.ds = ds; gp.dt = dt;
  gp.max_tiles = L.max_tiles;
  gp.hdr = hdr;
  gp.rowsrc = rowsrc;
  gp.rowdst = rowdst;
  gp.tok = tok;
  gp.hs_c = hs_c;
  gp.ht_c = ht_c;
  gp.status = a.status;
  const unsigned gather_grid = (unsigned)(rows_cap < 16384 ? rows_cap : 16384);
  if (a.B <= kGatherSeqs && plan.n_seg * a.B <= kGatherOwnSums &&
      rows_cap - (int64_t)plan.n_seg * (plan.pad - 1) <= kGatherOwnRows) {
    launch_chained(lm_gather_kernel<true>, gather_grid, kGatherThreads, 0, 1, s, gp, plan);
  } else {
    launch_chained(lm_plan_kernel, plan.n_seg, 1024, 0, 1, s, gp.range, gp.ewin, a.B, plan, seg);
    launch_chained(lm_gather_kernel<false>, gather_grid, kGatherThreads, 0, 1, s, gp, plan);
  }
  if ((e = cudaGetLastError()) != cudaSuccess) return e;

  CUtensorMap m_hs, m_ws, m_ht, m_wt;
  if (!make_map(&m_hs, hs_c, ds, rows_cap, ds, kBM) || !make_map(&m_ws, a.ws, ds, V, ds, kBN / 2) ||
      !make_map(&m_ht, ht_c, dt, rows_cap, dt, kBM) || !make_map(&m_wt, a.wt, dt, V, dt, kBN / 2))
    return cudaErrorInvalidValue;

  SweepParams sp;
  sp.hdr = hdr;
  sp.tok = tok;
  sp.V = V;
  sp.ks_blocks = (int)((ds + kBK - 1) / kBK);
  sp.kt_blocks = (int)((dt + kBK - 1) / kBK);
  sp.n_chunks = L.n_chunks;
  sp.keep_u = a.mode == ADWIN_GRAD_FULL_KL ? 1 : 0;
  sp.park = reinterpret_cast<float4*>(wb + L.off_park);
  sp.part = part;
  sp.part_slots = L.part_slots;
  sp.limit_ns = handshake_wait_limit_ns();
  sp.status = a.status;

  MergeParams mp;
  mp.hdr = hdr;
  mp.rowsrc = rowsrc;
  mp.rowdst = rowdst;
  mp.tokens = a.tokens;
  mp.part = part;
  mp.tok = tok;
  mp.info = info;
  mp.alpha = a.alpha;
  mp.mode = a.mode;
  mp.kl = a.kl;
  mp.logratio = a.logratio;
  mp.gsq = a.gsq;
  mp.lse_s = a.lse_s;
  mp.lse_t = a.lse_t;
  mp.status = a.status;

  int launch = 0;
  // statistics of the tiles [tile0, tile0 + cap) (rest: see SweepParams)
  auto statistics = [&](int64_t tile0, int64_t cap, int rest, bool kept, bool moments) {
    sp.tile0 = mp.tile0 = tile0;
    sp.tile_cap = mp.tile_cap = cap;
    sp.rest = mp.rest = rest;
    sp.keep = kept ? keep : nullptr;
    sp.pace = launch < 58 ? &hdr->pace[2 + launch] : nullptr;
    ++launch;
    const cudaError_t r =
        moments ? launch_pairs(lm_sweep_kernel<true>, a.sm_count, s, m_hs, m_ws, m_ht, m_wt, sp)
                : launch_pairs(lm_sweep_kernel<false>, a.sm_count, s, m_hs, m_ws, m_ht, m_wt, sp);
    if (r != cudaSuccess) return r;
    if (merge_by_8(cap, L.n_chunks)) launch_chained(lm_merge_kernel<8>, (unsigned)cap * (kBM / 8), 1024, 0, 1, s, mp);
    else launch_chained(lm_merge_kernel<32>, (unsigned)cap * (kBM / 32), 1024, 0, 1, s, mp);
    return cudaGetLastError();
  };
  if (!a.want_grad) return statistics(0, L.max_tiles, 2, false, a.gsq != nullptr);

  GradParams gr;
  gr.hdr = hdr;
  gr.keep = keep;
  gr.info = info;
  gr.V = V;
  gr.n_chunks = L.n_chunks;
  gr.n_groups = L.grad_groups;
  gr.G = G;
  gr.ldG = L.ldG;
  gr.q = q;
  gr.max_tiles = L.max_tiles;
  gr.status = a.status;
  // the moments are only needed for rows whose gsq does not come from the gradient entries
  const bool moments = a.gsq != nullptr && range_full;
  for (int64_t t0 = 0; t0 < L.max_tiles; t0 += L.block_tiles) {
    const int64_t cap = L.block_tiles < L.max_tiles - t0 ? L.block_tiles : L.max_tiles - t0;
    if ((e = statistics(t0, cap, 0, true, moments)) != cudaSuccess) return e;
    gr.tile0 = t0;
    gr.tile_cap = cap;
    const unsigned grid = (unsigned)(cap * L.grad_groups);
    if (a.mode == ADWIN_GRAD_FULL_KL) launch_chained(lm_grad_kernel<true>, grid, 256, 0, 1, s, gr);
    else launch_chained(lm_grad_kernel<false>, grid, 256, 0, 1, s, gr);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  if (range_full && (e = statistics(0, L.max_tiles, 1, false, moments)) != cudaSuccess) return e;
  if (a.gsq)
    launch_chained(lm_gsq_kernel, (unsigned)L.max_tiles * (kBM / kMergeRows), 1024, 0, 1, s, hdr, q,
                   rowdst, L.grad_groups, a.gsq);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;

  if (a.dH) {
    if (a.flags & ADWIN_ZERO_TAIL) {
      e = cudaMemsetAsync(a.dH, 0, (size_t)a.B * a.T * ds * (a.dh_dtype == ADWIN_F32 ? 4 : 2), s);
      if (e != cudaSuccess) return e;
    }
    // dH_s[rows, d_s] = G[rows, V] W_s[V, d_s]: A K-major; rows scattered to [B,T]
    e = launch_tc_gemm(G, L.ldG, false, a.ws, ds, rows_cap, ds, V, a.dH, ds,
                       a.dh_dtype == ADWIN_BF16, &hdr->grad_tiles, nullptr, rowdst, pieces,
                       &hdr->pace[0], a.status, a.sm_count, s);
    if (e != cudaSuccess) return e;
  }
  if (a.dW) {
    // dW_s[V, d_s] = G^T[V, rows] H_s[rows, d_s]: A MN-major, the contraction runs over rows
    e = launch_tc_gemm(G, L.ldG, true, hs_c, ds, V, ds, rows_cap, a.dW, ds, false, nullptr,
                       &hdr->grad_tiles, nullptr, pieces, &hdr->pace[1], a.status, a.sm_count, s);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

int current_sm_count() {
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return 148;
  return n;
}

}  // namespace

size_t lmhead_workspace_bytes(int64_t B, int64_t T, int64_t V, int64_t ds, int64_t dt,
                              int64_t max_rows, bool want_grad) {
  return lm_layout(B, T, V, ds, dt, max_rows, want_grad, 2, 1, current_sm_count()).total;
}

// The whole fused pass; arguments validated by the caller.
cudaError_t launch_lmhead(const void* hs, const void* ws, const void* ht, const void* wt, int64_t B,
                          int64_t T, int64_t V, int64_t ds, int64_t dt, const int32_t* tokens,
                          const int32_t* window, const int32_t* rollout_len, float alpha, int mode,
                          int flags, void* dH, int dh_dtype, float* dW, float* kl, float* logratio,
                          float* gsq, float* lse_s, float* lse_t, void* workspace,
                          int64_t max_rows, int32_t* status, int sm_count, cudaStream_t s) {
  const bool want_grad = dH != nullptr || dW != nullptr;
  const LmCall a = {hs, ws, ht, wt, B, T, V, ds, dt, tokens, window, rollout_len, alpha, mode, flags,
                    dH, dh_dtype, dW, want_grad, kl, logratio, gsq, lse_s, lse_t,
                    static_cast<char*>(workspace), status, sm_count};
  SegPlan plan = {};
  plan.n_seg = 2;
  plan.pad = 1;
  plan.want_grad = want_grad ? 1 : 0;
  return run_lmhead(a, lm_layout(B, T, V, ds, dt, max_rows, want_grad, 2, 1, sm_count), plan, s);
}

// ---------------------------------------------------------------------------- weight-space audit
// Prefix-versus-full cosine of Section 4.2 in the space of the student's LM-head weight.  The
// candidate lengths L_0 < ... < L_{K-1} (multiples of 64) cut every rollout into K+1 bins of
// positions; dW_bin[i] = G[bin i]^T H_s[bin i] is one GEMM per bin over that bin's 64-row k-blocks,
// the prefix gradient of candidate j is the sum of bins 0..j and the full-horizon reference the sum
// of all bins, so the K cosines come from one pass over the K+1 bin matrices.
struct CandList {
  int32_t K;
  int32_t L[kMaxCand];
};

namespace {

// Per block: sums over its share of the elements of  pre_j * full,  pre_j^2  (j < K)  and full^2,
// where pre_j = sum of bins 0..j and full = sum of all bins (NB = K + 1 of them).  Fixed order inside
// the block.  Bound by reading the bin matrices once: four consecutive elements of every bin per
// thread and step, all loads in flight together, the number of bins a compile-time constant so that
// prefixes and sums stay in registers (7 bins of 151 936 x 2048, 8.7 GB: 4.69 -> 1.35 ms, 6.45 TB/s;
// element loads and run-time bounds before).
constexpr int kGramThreads = 256;
constexpr int kGramFields = 2 * kMaxCand + 1;
template <int NB>
__global__ void __launch_bounds__(kGramThreads, 2) lm_gram_kernel(const float4* __restrict__ bins,
                                                                  int64_t n_vec, double* partial) {
  chain();
  double acc[2 * NB - 1];
#pragma unroll
  for (int i = 0; i < 2 * NB - 1; ++i) acc[i] = 0.0;
  for (int64_t e = (int64_t)blockIdx.x * kGramThreads + threadIdx.x; e < n_vec;
       e += (int64_t)gridDim.x * kGramThreads) {
    float4 x[NB];
#pragma unroll
    for (int i = 0; i < NB; ++i) x[i] = __ldcs(bins + (int64_t)i * n_vec + e);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      double pre[NB];
      float run = 0.f;
#pragma unroll
      for (int i = 0; i < NB; ++i) {
        run += c == 0 ? x[i].x : c == 1 ? x[i].y : c == 2 ? x[i].z : x[i].w;
        pre[i] = (double)run;
      }
      const double full = pre[NB - 1];
#pragma unroll
      for (int j = 0; j < NB - 1; ++j) {
        acc[2 * j] = fma(pre[j], full, acc[2 * j]);
        acc[2 * j + 1] = fma(pre[j], pre[j], acc[2 * j + 1]);
      }
      acc[2 * NB - 2] = fma(full, full, acc[2 * NB - 2]);
    }
  }
  __shared__ double red[kGramThreads / 32][2 * NB - 1];
#pragma unroll
  for (int i = 0; i < 2 * NB - 1; ++i) {
    double v = acc[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5][i] = v;
  }
  __syncthreads();
  if (threadIdx.x < 2 * NB - 1) {
    double v = 0.0;
    for (int w = 0; w < kGramThreads / 32; ++w) v += red[w][threadIdx.x];
    // field 2 kMaxCand is the full norm, whatever the number of bins
    partial[(int64_t)blockIdx.x * kGramFields +
            (threadIdx.x == 2 * NB - 2 ? 2 * kMaxCand : (int)threadIdx.x)] = v;
  }
}

template <int NB>
void launch_gram(int nb, const float* bins, int64_t n_elem, double* partial, int blocks, cudaStream_t s) {
  if (nb == NB)
    launch_chained(lm_gram_kernel<NB>, blocks, kGramThreads, 0, 1, s, reinterpret_cast<const float4*>(bins),
                   n_elem / 4, partial);
  else if constexpr (NB < kMaxSeg)
    launch_gram<NB + 1>(nb, bins, n_elem, partial, blocks, s);
}

// batch_stats[j] = { rho_w(L_j), snr, admissible (0/1), n_tokens }; L_next; flags.  One warp per
// field (and per candidate for the token counts), then one thread.
__global__ void __launch_bounds__(1024) lm_align_finish_kernel(
    const double* __restrict__ partial, int n_blocks, CandList cand, double rho_star,
    const int32_t* __restrict__ rollout_len, int64_t B, int64_t T, double* batch_stats,
    int32_t* L_next, int32_t* flags_out) {
  chain();
  __shared__ double tot[kGramFields];
  __shared__ double ntok[kMaxCand];
  const int K = cand.K, lane = threadIdx.x & 31;
  for (int w = threadIdx.x >> 5; w < kGramFields + K; w += 32) {
    double v = 0.0;
    if (w < kGramFields) {
      if (w < 2 * K || w == 2 * kMaxCand)
        for (int b = lane; b < n_blocks; b += 32) v += partial[(int64_t)b * kGramFields + w];
    } else {
      const int64_t L = cand.L[w - kGramFields];
      for (int64_t b = lane; b < B; b += 32) {
        int64_t R = rollout_len ? rollout_len[b] : T;
        R = R < 0 ? 0 : (R > T ? T : R);
        v += (double)(L < R ? L : R);
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) {
      if (w < kGramFields) tot[w] = v;
      else ntok[w - kGramFields] = v;
    }
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  int flags = 0, best = -1;
  const double nf = tot[2 * kMaxCand];
  for (int j = 0; j < K; ++j) {
    double rho;
    if (!(nf > 0.0)) {
      rho = 1.0;
      flags |= ADWIN_ALIGN_DEGENERATE;
    } else {
      rho = tot[2 * j + 1] > 0.0 ? tot[2 * j] / (sqrt(tot[2 * j + 1]) * sqrt(nf)) : 0.0;
    }
    const double r2 = rho * rho;
    batch_stats[j * 4 + 0] = rho;
    batch_stats[j * 4 + 1] = r2 < 1.0 ? r2 / (1.0 - r2) : INFINITY;
    batch_stats[j * 4 + 2] = rho >= rho_star ? 1.0 : 0.0;
    batch_stats[j * 4 + 3] = ntok[j];
    if (rho >= rho_star && best < 0) best = cand.L[j];   // candidates ascend: the first is the shortest
  }
  if (best < 0) {
    best = cand.L[K - 1];
    flags |= ADWIN_ALIGN_NONE_ADMISSIBLE;
  }
  *L_next = best;
  *flags_out = flags;
}

struct AlignLayout {
  size_t off_bins, off_partial, total;
  int gram_blocks;
};

AlignLayout align_layout(const LmLayout& L, int64_t V, int64_t ds, int K) {
  auto up = [](size_t x) { return (x + 1023) & ~size_t(1023); };
  AlignLayout A;
  A.gram_blocks = 592;
  size_t o = L.total;
  A.off_bins = o;     o = up(o + (size_t)(K + 1) * (size_t)V * ds * 4);
  A.off_partial = o;  o = up(o + (size_t)A.gram_blocks * kGramFields * 8);
  A.total = o;
  return A;
}

}  // namespace

size_t lmhead_align_workspace_bytes(int64_t B, int64_t T, int64_t V, int64_t ds, int64_t dt,
                                    int64_t max_rows, int K) {
  return align_layout(lm_layout(B, T, V, ds, dt, max_rows, true, K + 1, 64, current_sm_count()), V,
                      ds, K).total;
}

cudaError_t launch_lmhead_weight_align(const void* hs, const void* ws, const void* ht,
                                       const void* wt, int64_t B, int64_t T, int64_t V, int64_t ds,
                                       int64_t dt, const int32_t* tokens,
                                       const int32_t* rollout_len, const int32_t* cand_host, int K,
                                       double rho_star, int mode, float* kl, float* logratio,
                                       float* gsq, double* batch_stats, int32_t* L_next,
                                       int32_t* flags_out, void* workspace, int64_t max_rows,
                                       int32_t* status, int sm_count, cudaStream_t s) {
  const LmLayout L = lm_layout(B, T, V, ds, dt, max_rows, true, K + 1, 64, sm_count);
  const AlignLayout A = align_layout(L, V, ds, K);
  char* wb = static_cast<char*>(workspace);
  // every position of every rollout carries gradient here: the window is the rollout itself
  // (window == NULL stands for W_b = T in the row map, so E_b = R_b)
  const LmCall a = {hs, ws, ht, wt, B, T, V, ds, dt, tokens, nullptr, rollout_len, 1.0f, mode, 0,
                    nullptr, ADWIN_F32, nullptr, true, kl, logratio, gsq, nullptr, nullptr, wb, status,
                    sm_count};
  CandList cand;
  cand.K = K;
  SegPlan plan = {};
  plan.n_seg = K + 1;
  plan.pad = 64;          // a 64-row k-block never straddles two bins
  plan.want_grad = 1;
  plan.by_cut = 1;
  for (int i = 0; i < kMaxCand; ++i) plan.cut[i] = cand.L[i] = i < K ? cand_host[i] : 0;
  cudaError_t e = run_lmhead(a, L, plan, s);
  if (e != cudaSuccess) return e;
  const LmHeader* hdr = reinterpret_cast<const LmHeader*>(wb + L.off_hdr);
  const __nv_bfloat16* hs_c = reinterpret_cast<const __nv_bfloat16*>(wb + L.off_hs);
  const __nv_bfloat16* G = reinterpret_cast<const __nv_bfloat16*>(wb + L.off_G);
  float* bins = reinterpret_cast<float*>(wb + A.off_bins);
  double* partial = reinterpret_cast<double*>(wb + A.off_partial);
  e = launch_tc_gemm_bins(G, L.ldG, hs_c, ds, V, ds, L.max_tiles * kBM, bins, ds, V * ds, K + 1,
                          hdr->seg_kblock, status, sm_count, s);
  if (e != cudaSuccess) return e;
  launch_gram<2>(K + 1, bins, V * ds, partial, A.gram_blocks, s);   // (V and d_s are multiples of 8)
  launch_chained(lm_align_finish_kernel, 1, 1024, 0, 1, s, partial, A.gram_blocks, cand, rho_star,
                 rollout_len, B, T, batch_stats, L_next, flags_out);
  return cudaGetLastError();
}

}  // namespace adwin
