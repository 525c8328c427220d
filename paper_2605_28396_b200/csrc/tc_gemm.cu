// Tensor-core GEMM over CTA pairs: C[M,N] = A B with bf16 operands read through TMA in either
// major and fp32 accumulation in tensor memory.  It forms dH_s = G W_s and dW_s = G^T H_s of the
// fused LM-head pass.
//
// Two CTAs of a cluster work as one MMA unit (cta_group::2): a tile is 256 rows x 256 columns, each
// CTA stages its own 128 rows of A and half of the columns of B (32 KB per 64-deep k-block, six
// stages) and holds its own 128 rows of the accumulator.  Two accumulator slots: the epilogue of a
// tile overlaps the MMAs of the next one.  Bound by the tensor pipe and, in a long run, by the
// board's power limit; the pair form moves 64 bytes per clock and SM through L2 where single CTAs
// with 128 x 256 tiles move 96.
//
// Tiles are dealt out in whole rounds over the pairs; the tiles of the last, partial round are cut
// along the contraction (split-K) so that they keep every pair busy.  The pieces go to a fixed-order
// sum (gemm_reduce_kernel), so results stay bitwise reproducible.
#include <cuda_bf16.h>

#include <mutex>

#include "adwin_common.cuh"
#include "adwin_internal.h"
#include "tc_pipeline.cuh"

namespace adwin {

using namespace tc;

namespace {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_tiled() {
  static std::mutex mu;
  static EncodeTiledFn fn = nullptr;
  std::lock_guard<std::mutex> lock(mu);
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

}  // namespace

bool make_map(CUtensorMap* m, const void* base, int64_t cols, int64_t rows, int64_t pitch,
              int box_rows) {
  EncodeTiledFn fn = encode_tiled();
  if (!fn || rows < 1 || cols < 1) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)pitch * 2};
  const cuuint32_t box[2] = {(cuuint32_t)kBK, (cuuint32_t)box_rows};
  const cuuint32_t estr[2] = {1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box,
            estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

namespace {

// Pieces of split tiles that the scratch buffer holds (256 KB each).
constexpr int kMaxPieces = 4 * 74;
constexpr int kMinPiece = 8;     // k-blocks of a piece, at least
constexpr size_t kPieceBytes = (size_t)2 * kBM * kBN * 4;

struct GemmParams {
  int64_t M, N;                 // extents of C (rows beyond M / columns beyond N are not stored)
  int m_tiles, n_tiles;         // 128-row tiles of C, 256-column tiles of C
  int k_blocks;
  const int32_t* m_tiles_dev;   // optional device-side override of m_tiles
  const int32_t* k_tiles_dev;   // optional: k_blocks = 2 * (*k_tiles_dev) (128 rows per tile)
  int n_bins;                   // products over consecutive k-ranges (1 without kblock_dev)
  const int32_t* kblock_dev;    // optional: first k-block of every bin, and the end
  int64_t bin_stride;           // elements between the bins' results
  const int32_t* row_map;       // optional: destination row of every C row, or -1 (skip)
  void* C;
  int64_t ldc;
  int c_is_bf16;
  unsigned int* pace;           // zeroed counter that keeps the pairs in step, or null
  float* pieces;                // split-K scratch, or null (no tile is split)
  int32_t* status;
  uint64_t limit_ns;            // limit of the handshake waits
};

// How the tiles are dealt out; the same on every thread of both kernels.
struct GemmWork {
  int m_pairs, nk;
  int64_t M;        // rows of C that exist (row_map is only filled that far)
  int whole;        // tiles taken whole
  int split;        // pieces per remaining tile
  int64_t items;    // whole tiles first, then the pieces
  __device__ __forceinline__ GemmWork(const GemmParams& p, int pairs) {
    const int m_tiles = p.m_tiles_dev ? *p.m_tiles_dev : p.m_tiles;
    m_pairs = (m_tiles + 1) / 2;
    M = p.M < (int64_t)m_tiles * kBM ? p.M : (int64_t)m_tiles * kBM;
    nk = p.k_tiles_dev ? 2 * (*p.k_tiles_dev) : p.k_blocks;
    const int tiles = m_pairs * p.n_tiles;
    whole = tiles;
    split = 1;
    const int rest = tiles % pairs;
    if (p.pieces && rest > 0) {
      // The last round's cost in k-blocks; a piece pays ~8 for filling the pipeline, storing and
      // being summed, so short contractions stay whole.
      int best = nk;
      for (int s = 2; s <= 64 && s * rest <= kMaxPieces && s * kMinPiece <= nk; ++s) {
        const int cost = (s * rest + pairs - 1) / pairs * ((nk + s - 1) / s + 8) + 8;
        if (cost < best) {
          best = cost;
          split = s;
        }
      }
      if (split > 1) whole = tiles - rest;
    }
    items = (whole + (int64_t)(tiles - whole) * split) * p.n_bins;
  }
  __device__ __forceinline__ void item(const GemmParams& p, int64_t i, int& pm, int& n, int& k0,
                                       int& k1, int& piece, int& bin) const {
    int tile;
    bin = 0;
    if (p.kblock_dev) {   // bins: every tile whole, bin after bin
      bin = (int)(i / whole);
      tile = (int)(i % whole);
      k0 = p.kblock_dev[bin];
      k1 = p.kblock_dev[bin + 1];
      piece = -1;
    } else if (i < whole) {
      tile = (int)i;
      k0 = 0;
      k1 = nk;
      piece = -1;
    } else {
      piece = (int)(i - whole);
      tile = whole + piece / split;
      const int s = piece % split;
      k0 = (int)((int64_t)nk * s / split);
      k1 = (int)((int64_t)nk * (s + 1) / split);
    }
    pm = tile / p.n_tiles;
    n = tile % p.n_tiles;
  }
};

// NC consecutive columns (a multiple of 8) of one row of C.
template <int NC>
__device__ __forceinline__ void store_c(const GemmParams& p, int bin, int64_t dst, int64_t n,
                                        const float (&v)[NC]) {
  if (p.c_is_bf16) {
    __nv_bfloat16* cp = static_cast<__nv_bfloat16*>(p.C) + dst * p.ldc + n;
#pragma unroll
    for (int i = 0; i < NC; i += 8)
      if (n + i < p.N)
        *reinterpret_cast<uint4*>(cp + i) =
            make_uint4(pack_bf16x2(v[i], v[i + 1]), pack_bf16x2(v[i + 2], v[i + 3]),
                       pack_bf16x2(v[i + 4], v[i + 5]), pack_bf16x2(v[i + 6], v[i + 7]));
  } else {
    float* cp = static_cast<float*>(p.C) + (int64_t)bin * p.bin_stride + dst * p.ldc + n;
    if ((reinterpret_cast<uintptr_t>(cp) & 31) == 0) {   // whole 32-byte sectors
#pragma unroll
      for (int i = 0; i < NC; i += 8)
        if (n + i < p.N)   // (N % 8 == 0)
          asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(cp + i),
                       "f"(v[i]), "f"(v[i + 1]), "f"(v[i + 2]), "f"(v[i + 3]), "f"(v[i + 4]),
                       "f"(v[i + 5]), "f"(v[i + 6]), "f"(v[i + 7])
                       : "memory");
    } else {
#pragma unroll
      for (int i = 0; i < NC; i += 4)
        if (n + i < p.N)
          *reinterpret_cast<float4*>(cp + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
    }
  }
}

template <bool A_MN, bool B_MN>
__global__ void __launch_bounds__(kThreads, 1)
tc_gemm_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
               const GemmParams p) {
  chain_wait();
  extern __shared__ uint8_t smem_raw[];
  Ctrl* ctrl = reinterpret_cast<Ctrl*>(smem_raw);
  const uint32_t stage0 = (smem_addr(smem_raw) + kCtrlBytes + 1023u) & ~1023u;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  volatile int* abort = &ctrl->abort;
  const uint32_t rank = cluster_ctarank();   // 0: the CTA that issues the MMAs

  if (threadIdx.x == 0) pair_bars_init(ctrl);
  if (warp == 2) {
    tmem_alloc_pair(smem_addr(&ctrl->tmem_base), kTmemCols);
    tmem_relinquish_pair();
    tc_fence_before_sync();
  }
  __syncthreads();
  cluster_sync();   // the partner's barriers exist before anything signals them
  tc_fence_after_sync();
  const uint32_t tmem_base = ctrl->tmem_base;

  const int pair = blockIdx.x / 2, pairs = gridDim.x / 2;
  const GemmWork w(p, pairs);

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    if (lane == 0) {
      uint32_t it = 0;
      bool ok = true;
      Pace pace(rank == 0 ? p.pace : nullptr, pairs);
      for (int64_t item = pair; ok && item < w.items; item += pairs) {
        int pm, n, k0, k1, piece, bin;
        w.item(p, item, pm, n, k0, k1, piece, bin);
        const int m0 = (2 * pm + (int)rank) * kBM, n0 = n * kBN + (int)rank * (kBN / 2);
        for (int kb = k0; kb < k1; ++kb, ++it) {
          const uint32_t s = it % kPairStages, ph = (it / kPairStages) & 1;
          pace.kblock(it);
          if (!bar_wait(smem_addr(&ctrl->empty[s]), ph ^ 1, abort, p.limit_ns)) { ok = false; break; }
          const uint32_t bar = smem_addr(&ctrl->full[s]);
          const uint32_t a = stage0 + s * kPairStageBytes, b = a + kABytes;
          if (rank == 0) bar_expect_tx(bar, 2 * kPairStageBytes);   // both CTAs' bytes
          const uint32_t bar0 = map_to_cta(bar, 0);
          load_operand_pair<A_MN>(a, &map_a, m0, kb * kBK, bar0);
          load_operand_pair<B_MN>(b, &map_b, n0, kb * kBK, bar0);
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
      for (int64_t item = pair; ok && item < w.items; item += pairs, ++acc_it) {
        int pm, n, k0, k1, piece, bin;
        w.item(p, item, pm, n, k0, k1, piece, bin);
        const uint32_t slot = acc_it & 1, aph = (acc_it >> 1) & 1;
        if (!bar_wait(smem_addr(&ctrl->acc_empty[slot]), aph ^ 1, abort, p.limit_ns)) { ok = false; break; }
        tc_fence_after_sync();
        const uint32_t tmem_d = tmem_base + slot * kBN;
        for (int kb = k0; kb < k1; ++kb, ++it) {
          const uint32_t s = it % kPairStages, ph = (it / kPairStages) & 1;
          if (!bar_wait(smem_addr(&ctrl->full[s]), ph, abort, p.limit_ns)) { ok = false; break; }
          tc_fence_after_sync();
          const uint32_t a = stage0 + s * kPairStageBytes, b = a + kABytes;
          issue_kblock_pair<A_MN, B_MN>(tmem_d, a, b, kb == k0);
          umma_commit_pair(smem_addr(&ctrl->empty[s]));
        }
        if (ok) {
          if (k1 > k0) {
            umma_commit_pair(smem_addr(&ctrl->acc_full[slot]));
          } else {
            bar_arrive(smem_addr(&ctrl->acc_full[slot]));
            bar_arrive_cluster(map_to_cta(smem_addr(&ctrl->acc_full[slot]), 1));
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
    const int quad = warp & 3, half = ew >> 2;
    const int row = quad * 32 + lane;
    uint32_t acc_it = 0;
    bool ok = true;
    for (int64_t item = pair; ok && item < w.items; item += pairs, ++acc_it) {
      int pm, nt, k0, k1, piece, bin;
      w.item(p, item, pm, nt, k0, k1, piece, bin);
      const uint32_t slot = acc_it & 1, aph = (acc_it >> 1) & 1;
      const int64_t m = (int64_t)(2 * pm + (int)rank) * kBM + row;
      const int64_t n0 = (int64_t)nt * kBN + half * 128;
      int64_t dst = m;
      if (p.row_map) dst = (m < w.M) ? p.row_map[m] : -1;
      const bool store = m < w.M && dst >= 0 && ADWIN_CHK(n0 < (int64_t)p.n_tiles * kBN, p.status);
      if (!__all_sync(0xffffffffu, bar_wait(smem_addr(&ctrl->acc_full[slot]), aph, abort, p.limit_ns))) {
        ok = false;   // the same decision in every lane: tcgen05.ld below is warp-collective
        break;
      }
      tc_fence_after_sync();
      const uint32_t t_lane =
          tmem_base + ((uint32_t)(quad * 32) << 16) + slot * kBN + (uint32_t)(half * 128);
      // a piece is kept as [64 column groups of 4][128 rows] float4 per CTA: coalesced over rows
      float4* pc = piece < 0 ? nullptr
                             : reinterpret_cast<float4*>(p.pieces) +
                                   ((size_t)piece * 2 + rank) * (kBM * kBN / 4) +
                                   (size_t)(half * 32) * kBM + row;
#pragma unroll 1
      for (int j = 0; j < 4; ++j) {
        uint32_t r[32];
        if (k1 > k0) {
          tmem_ld32(t_lane + j * 32, r);
          tmem_ld_wait();
        } else {
#pragma unroll
          for (int i = 0; i < 32; ++i) r[i] = 0u;
        }
        float v[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
        if (pc) {
          if (ADWIN_CHK(piece < kMaxPieces, p.status)) {
#pragma unroll
            for (int i = 0; i < 8; ++i)
              pc[(size_t)(j * 8 + i) * kBM] =
                  make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
          }
        } else if (store) {
          store_c<32>(p, bin, dst, n0 + j * 32, v);
        }
      }
      tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) pair_release(&ctrl->acc_empty[slot], rank);
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

// Sums the pieces of the split tiles in order and stores C; a thread owns 8 columns of a row.
__global__ void __launch_bounds__(128) gemm_reduce_kernel(const GemmParams p, int pairs) {
  chain();
  const GemmWork w(p, pairs);
  if (w.split == 1) return;
  const int rest = w.m_pairs * p.n_tiles - w.whole;
  const int row = threadIdx.x;
  for (int u = blockIdx.x; u < rest * 64; u += gridDim.x) {   // 2 CTAs x 32 column groups of 8
    const int t = u / 64, rank = (u / 32) & 1, j = u % 32;
    const int tile = w.whole + t;
    const int64_t m = (int64_t)(2 * (tile / p.n_tiles) + rank) * kBM + row;
    const int64_t n = (int64_t)(tile % p.n_tiles) * kBN + j * 8;
    int64_t dst = m;
    if (p.row_map) dst = (m < w.M) ? p.row_map[m] : -1;
    if (m >= w.M || dst < 0 || n >= p.N) continue;
    float v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = 0.f;
    const float4* pc = reinterpret_cast<const float4*>(p.pieces) +
                       ((size_t)t * w.split * 2 + rank) * (kBM * kBN / 4) + (size_t)(j * 2) * kBM + row;
#pragma unroll 6
    for (int s = 0; s < w.split; ++s, pc += kBM * kBN / 2) {
      const float4 x = __ldcs(pc), y = __ldcs(pc + kBM);
      v[0] += x.x; v[1] += x.y; v[2] += x.z; v[3] += x.w;
      v[4] += y.x; v[5] += y.y; v[6] += y.z; v[7] += y.w;
    }
    store_c<8>(p, 0, dst, n, v);
  }
}

cudaError_t launch_gemm(const void* A, int64_t lda, bool a_mn, const void* B, int64_t ldb, int64_t K,
                        GemmParams p, int sm_count, cudaStream_t s) {
  CUtensorMap ma, mb;
  const bool oka = a_mn ? make_map(&ma, A, p.M, K, lda, 64) : make_map(&ma, A, K, p.M, lda, kBM);
  if (!oka || !make_map(&mb, B, p.N, K, ldb, 64)) return cudaErrorInvalidValue;
  p.m_tiles = (int)((p.M + kBM - 1) / kBM);
  p.n_tiles = (int)((p.N + kBN - 1) / kBN);
  p.k_blocks = (int)((K + kBK - 1) / kBK);
  p.limit_ns = handshake_wait_limit_ns();
  const cudaError_t e = a_mn ? launch_pairs(tc_gemm_kernel<true, true>, sm_count, s, ma, mb, p)
                             : launch_pairs(tc_gemm_kernel<false, true>, sm_count, s, ma, mb, p);
  if (e != cudaSuccess || !p.pieces || p.k_blocks < 2 * kMinPiece) return e;   // (nothing is split)
  launch_chained(gemm_reduce_kernel, sm_count * 4, 128, 0, 1, s, p, sm_count / 2);
  return cudaGetLastError();
}

}  // namespace

size_t tc_gemm_scratch_bytes() { return kMaxPieces * kPieceBytes; }

cudaError_t launch_tc_gemm(const void* A, int64_t lda, bool a_mn, const void* B, int64_t ldb,
                           int64_t M, int64_t N, int64_t K, void* C, int64_t ldc, bool c_bf16,
                           const int32_t* m_tiles_dev, const int32_t* k_tiles_dev,
                           const int32_t* row_map, float* scratch, unsigned int* pace,
                           int32_t* status, int sm_count, cudaStream_t s) {
  GemmParams p = {};
  p.M = M;
  p.N = N;
  p.m_tiles_dev = m_tiles_dev;
  p.k_tiles_dev = k_tiles_dev;
  p.n_bins = 1;
  p.row_map = row_map;
  p.C = C;
  p.ldc = ldc;
  p.c_is_bf16 = c_bf16 ? 1 : 0;
  p.pace = pace;
  p.pieces = scratch;
  p.status = status;
  return launch_gemm(A, lda, a_mn, B, ldb, K, p, sm_count, s);
}

cudaError_t launch_tc_gemm_bins(const void* A, int64_t lda, const void* B, int64_t ldb, int64_t M,
                                int64_t N, int64_t K, float* C, int64_t ldc, int64_t bin_stride,
                                int n_bins, const int32_t* kblock_dev, int32_t* status,
                                int sm_count, cudaStream_t s) {
  GemmParams p = {};
  p.M = M;
  p.N = N;
  p.n_bins = n_bins;
  p.kblock_dev = kblock_dev;
  p.bin_stride = bin_stride;
  p.C = C;
  p.ldc = ldc;
  p.status = status;
  return launch_gemm(A, lda, true, B, ldb, K, p, sm_count, s);
}

}  // namespace adwin
