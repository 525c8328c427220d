// Row kernel for calls with gradient: a row (or a cluster's slice of it) is read from HBM once and kept on
// chip between its two sweeps; a row's second sweep and the next row's first run together.
//
// A row needs its sums before its gradient can be formed, so a CTA that finished one row before it began the
// next would leave HBM idle during the exchange and the arithmetic of the second sweep.  Here every thread goes
// through one stream of 16-byte pieces: for each group of pieces it forms the gradient of the row that has its
// sums, puts the next row's pieces into the places that fall free, folds them into that row's sums and asks for the
// group after (so loads are always one group ahead in registers).  The places are a ring of groups in
// tensor memory (tcgen05.st / tcgen05.ld; no MMA runs here) and shared memory, each thread's its own: no
// hand-shakes over data.  The ring has room for up to three groups more than a row, which are taken while
// the row's sums travel, so the exchange costs no idle time either (the longest rows of a shape leave none).  Rows are brought into L2 three groups
// ahead (cp.async.bulk.prefetch.L2).  (All at once a row ahead is too early: rows of 100 000 bf16 entries were
// pushed out of L2 again, 609 us against 489 for 2.4 GB.)
//
// One more warp does what is done once per row: it adds up the threads' sums, derives the row's scalars and
// hands them back, fetches the coming rows' metadata, and looks after the few entries before a row's first
// and after its last whole piece.  Pieces are counted from the 128-byte line in which a row starts: a warp's
// loads and stores are whole lines whatever the row's offset (fp32, rows of 50 264 entries: 435 us before, 380 so).
//
// Exponentials are taken against a reference that the whole row shares (the logit of the sampled
// token), so partial sums add without rescaling.  If the sums overflow it (a sampled token more than
// ~69 nats below the row maximum) the row is summed once more, from its on-chip copy (the teacher's
// pieces from memory where only the student's are kept), against running maxima.  Rows too long for one CTA, and
// the rows of calls with few, are split over a cluster; the CTAs' sums then go to every CTA of the cluster.
#include <iterator>
#include <mutex>
#include <type_traits>

#include "adwin_common.cuh"
#include "adwin_internal.h"
#include "kl_pairs.cuh"
#include "tc_pipeline.cuh"

namespace adwin {
namespace {

constexpr int kRowsThreads = 512;     // threads of a CTA that hold pieces, at most
// Steps of a group: the piece pairs that a thread has in flight.  One: 540 us where two take 430 (32 000
// entries of bf16; the ring's bookkeeping is per group); four spill.
constexpr int kU = 2;
constexpr int kRowsMaxCl = 4;
constexpr float kSumLimit = 1.2676506e30f;   // 2^100: beyond it the shared reference is unsafe
// Rows' metadata: the row's own warp has written that of row i + kMetaAhead when it gives out row i's scalars
// (kReady), and the other threads may look at no row beyond before they are through the next kReady.  A load is one group
// ahead of its sweep, which itself runs `ahead` groups into row i + 1 before row i's kReady: rows of one group
// are asked for two rows after i + 1.  metadata_precedes_its_readers() holds every plan against this.
constexpr int kMetaAhead = 4;
constexpr int kMetaDepth = 8;
constexpr int kMostEarly = 3;         // groups from a piece's way into L2 to its load, at most
constexpr int kLine = 128;
constexpr int64_t kShortRow = 14336;  // entries
constexpr int kEdges = 16;            // entries beside a row's whole pieces: less than 8 on each side
constexpr float kMaskedEdge = -1e30f;

struct RowsPlan {
  int cl;             // CTAs per row
  int nt;             // threads per CTA that hold pieces (one more warp does the row's own work)
  int ctas;           // CTAs per SM
  int per_rank;       // 16-byte pieces of a slice (per array)
  int groups;         // groups of kU steps (a piece of every thread each) that a slice takes
  int early;          // groups between a piece's way into L2 and its first sweep (at most `groups`)
  int ahead;          // groups of the next row that are taken before this row's second sweep
  int tm_groups;      // groups kept in tensor memory (the ring's first ones); the rest in shared memory
  int tm_cols;        // tensor-memory columns per CTA (0: none)
  int num_clusters;
};

struct RowsShape {
  int ctas, nt, tm_cols, cl;
  int most;           // pieces of a row up to which the shape is taken
  int few;            // and, where a call has no more rows than the GPU holds at a time so, from which (0: never)
};
// The first that takes the row is used: the more and smaller CTAs, the less of a group lies idle at a row's
// end; beyond 57 000 entries of bf16 one CTA per SM and not two in clusters (151 936 entries: two CTAs in clusters of
// four, of which 71 fit on 148 SMs, 496 us where this took 421).  Registers allow 20 warps of 96 (or 24 of 80, which is what
// the 64-thread kernels take): 22 warps of 80 in {2, 352} 443 us where {2, 256} took 422 (32 000 entries).
// Tensor memory is shared out in powers of two.  Measured over 2.4 GB of logits and gradient (367 us at the
// copy rate; a kernel that ended one row before it began the next, on {8, 64} to {2, 352} x 4 / this one):
//   bf16  V =   4 096  477 / 440 us  {8, 64}       fp32  V =   4 096  416 / 376 us  {4, 128}
//              5 000  506 / 491     {8, 64}                5 001  479 / 379     {4, 128}
//              8 192  443 / 430     {4, 128}              50 264  480 / 372     {1, 512}
//             16 384  486 / 411     {4, 128}             100 000  495 / 380     {1, 512} x 2
//             32 000  470 / 407     {2, 256}        bf16, sampled-token estimator
//             50 257  508 / 415     {2, 256}              32 000  466 / 411     {2, 256}
//             57 344  512 / 395     {2, 256}              64 000  498 / 387     {1, 512}
//             80 000  515 / 394     {1, 512}             151 936  547 / 382     {1, 512}
//            114 688  560 / 394     {1, 512}
//            151 936  555 / 411     {1, 512} x 2
//            229 376  631 / 414     {1, 512} x 2
//            262 144  614 / 441     {1, 512} x 4
// (57 344, 114 688 and 229 376 fill their shapes, whose ring then has no group to spare for the exchange.)
// fp32 rows are at the copy rate.  bf16 rows (163 issue slots and 24 of ex2 for eight entries, where the copy
// rate leaves 273 clocks) are bound by arithmetic, short ones also by what is done once per row.
// (The small shapes hold twice as much of a row whose second sweep takes the student alone, but are slower there:
// 10 309 entries on {8, 64} 140 us where {4, 128} takes 131.)
// A call of so few rows that each gets a CTA or cluster of its own anyway takes the last (widest) shape for
// which that holds, from `few` pieces on.  B * T counts as its rows, which is what the host knows of them, so a
// shape is never too wide for the rows there are.  Device time of a call (the shape by length alone / this one /
// a kernel with up to four CTAs of 352 threads a row that did not join the sweeps):
//   bf16  13 rows of 151 936   21.1 / 15.7 / 17.4 us  x 4    64 rows  25.0 / 23.2 / 22.8 us  x 2
//                     80 000   19.0 / 12.7 / 17.8     x 4             21.7 / 17.6 / 19.0     x 2
//                     50 257   19.2 / 12.2 / 18.3     x 4             21.2 / 15.9 / 19.4     x 2
//                      4 096    8.2 /  7.5 /  7.9     {2, 256}         8.3 /  7.5 /  8.0     {2, 256}
// With a piece or two per thread a row's exchange costs more than its sweeps: 16 384 entries, 8 rows, four
// CTAs 9.3, two 9.6, one 9.05; 24 576 entries 9.5, 10.5, 10.2; 4 096 entries {1, 512} 7.65, {2, 256} 7.2.
constexpr RowsShape kShapes[] = {{8, 64, 0, 1, 768, 0}, {4, 128, 128, 1, 3584, 0}, {2, 256, 256, 1, 7168, 512},
                                 {1, kRowsThreads, 512, 1, 1 << 24, 1024}, {1, kRowsThreads, 512, 2, 1 << 24, 3584},
                                 {1, kRowsThreads, 512, 4, 1 << 24, 3584}};
// CTAs per SM of the shapes with nt threads, and whether they use tensor memory (the same for all of them).
constexpr int ctas_of(int nt) {
  for (const RowsShape& sh : kShapes)
    if (sh.nt == nt) return sh.ctas;
  return 1;
}
constexpr bool uses_tensor_memory(int nt) {
  for (const RowsShape& sh : kShapes)
    if (sh.nt == nt) return sh.tm_cols > 0;
  return false;
}

struct __align__(16) RowsMeta {
  int64_t r;
  int y;
  float w;            // caller-supplied row coefficient (0 when there is none)
  float zy, uy;
  float dref;         // z - u at the sampled token
  float pad;
  // as pairs and negated: the references of the student's and the teacher's sums, the centre of delta, which
  // is exactly zero then at the peak of most peaked rows (it is the sampled token): beside a term of that size
  // the rest of the row would lose the bits that the difference from the mean is made of
  float nref[8];
  float edge[kEdges][2];   // logits of the entries beside the row's whole pieces (kMaskedEdge where there is none)
};
// A row's constants stay in shared memory and are read with every group: both sweeps' would take ten
// registers that the loads in flight need.
__device__ __forceinline__ void row_pairs(const float* at, f2_t& a, f2_t& b) {
  asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "r"(smem_u32(at)));
}

// What the second sweep needs of a row, as pairs: -m2s, the coefficient, the (scaled) centre.
struct __align__(16) RowsScalars {
  float nm2s[2], coef[2];
  float nc0[2], gy;
  int again;          // the sums overflowed: sum the row once more against running maxima
};

struct __align__(16) RowsCtrl {
  float safe[kRowsThreads / 32][8];    // the warps' records of the running-maximum pass
  float xrec[2][kRowsMaxCl][8];    // per row parity, one record per CTA of the cluster
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

// A row in a CTA's slice.  With RAG pieces are counted from the 128-byte line that the student's row starts in, so
// that a warp's 512 bytes are whole lines; without, from the row's start (a line's, but for short rows).
struct RowSlice {
  int begin, pieces;   // the slice's pieces [begin, pieces) are the row's
  int shift;           // entries from the line's start to the row's
};

// NT: threads that hold pieces, a template constant so that the strides between a thread's pieces are
// offsets in the instructions.  A group of kU steps in which every thread has whole pieces takes the path
// without tests (FULL below), with ALONE also where one sweep runs alone (see lone_sweeps).  FULLKL: the gradient of Eq. 2; without it, of Eq. 4, whose second sweep
// takes the student's logits alone, so only they are kept.
template <typename TIn, typename TOut, int NT, bool TM, bool RAG, bool FULLKL, bool ALONE>
__global__ void __launch_bounds__(NT + 32, ctas_of(NT))
kl_rows_kernel(const KlParams p, const RowsPlan plan) {
  chain();
  constexpr int N = Elem<TIn>::N;
  constexpr int NP = Pairs<TIn>::NP;
  constexpr int nt = NT, nw = NT / 32, all = NT + 32;
  constexpr uint32_t array = NT * 16u;
  constexpr int kKept = FULLKL ? 2 : 1;             // arrays kept
  // delta is summed about a centre (RowsMeta::dref) and the reference chosen for the coefficient's product with the
  // mean (see there) where a thread's chain of additions is longest; fp32 rows keep to delta itself, whose
  // tolerance a centre far from the mean would cost.  (2.4 GB of rows of 32 000 entries 420 -> 424 us with both, where
  // shorter ones would pay more: 8 192 436 -> 453, 5 000 519 -> 539.)
  constexpr bool kCentred = sizeof(TIn) == 2 && NT >= 256;
  // Where a thread's chains of additions are longer, and rows are added up over more threads, than in the kernel that
  // did not join the sweeps: what the additions over the threads round off is kept (S and A over all of them, the teacher's
  // sum and the norm over lanes and CTAs), and a thread's norm is two sums.  Median errors against a 64-bit
  // evaluation, of that kernel / of plain sums / of these:
  //   tokens drawn uniformly, 50 248 entries   KL 1.06e-7 / 1.16e-7 / 0.94e-7   log-ratio 0.54e-7 / 0.53e-7 / 0.48e-7
  //                                            squared norm 1.48e-7 / 1.60e-7 / 1.29e-7
  //   spikes, 151 936 entries                  KL 0.73e-7 / 0.84e-7 / 0.66e-7   log-ratio 0.87e-7 / 0.87e-7 / 0.82e-7
  //                                            squared norm 1.24e-7 / 1.59e-7 / 1.24e-7
  // (2.4 GB: rows of 32 000 entries 405 us with plain sums and so, 151 936 402 and 412, 50 257 429 and 434.  All four
  // sums over all threads: 151 936 440.)
  constexpr bool kExact = NT >= 256;
  constexpr int kNorms = kExact && FULLKL ? kU : 1;
  constexpr uint32_t group_bytes = kU * kKept * array;
  constexpr int group_cols = kU * kKept * 4;
  extern __shared__ __align__(128) char smem[];
  RowsCtrl& ctrl = *reinterpret_cast<RowsCtrl*>(smem);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int cl = plan.cl;
  float4* rec = reinterpret_cast<float4*>(smem + kRowsRec);
  char* stash = smem + rows_ctrl_bytes(NT) + tid * 16;   // [group][step][array][thread] 16 bytes
#ifdef ADWIN_CHECKED
  uint32_t smem_bytes;
  asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(smem_bytes));
  // a group's pieces from `at` on, and its columns of tensor memory (the same for a whole warp)
  auto stash_ok = [&](const char* at) {
    return at >= stash && at + (kU * kKept - 1) * array + 16 <= smem + smem_bytes;
  };
  auto columns_ok = [&](int pos) {
    return pos >= 0 && pos < plan.tm_groups && ((tid >> 7) + 1) * plan.tm_groups * group_cols <= plan.tm_cols;
  };
#endif
  const uint32_t rank = cl > 1 ? cluster_rank() : 0u;
  const int64_t cluster_id = blockIdx.x / cl;
  const int piece0 = (int)rank * plan.per_rank;
  const int64_t total_rows = p.offsets[p.B];
  const int my_rows =
      cluster_id < total_rows ? (int)((total_rows - cluster_id + plan.num_clusters - 1) / plan.num_clusters) : 0;

  if (TM && warp == nw) tm_alloc(smem_u32(&ctrl.tmem_base), (uint32_t)plan.tm_cols);

  // where row r lies in this CTA's slice (base pointers are 16-byte aligned; without RAG rows are whole pieces).
  // The at most N - 1 entries before its first and after its last whole piece are its own warp's.
  auto slice_of = [&](int64_t r) -> RowSlice {
    RowSlice a = {0, 0, 0};
    if (RAG) {
      a.shift = (int)((reinterpret_cast<uintptr_t>(p.student) / sizeof(TIn) + r * p.ld) & (kLine / sizeof(TIn) - 1));
      if (piece0 == 0) a.begin = (a.shift + N - 1) / N;
    }
    const int64_t left = (a.shift + p.V) / N - piece0;
    a.pieces = (int)(left < 0 ? 0 : (left > plan.per_rank ? plan.per_rank : left));
    return a;
  };
  // its groups [full_from, full_to) have a piece for every thread in every step
  auto full_from = [&](const RowSlice& a) { return RAG && a.begin > 0 ? 1 : 0; };
  auto full_to = [&](const RowSlice& a) { return a.pieces / (kU * nt); };
  auto holds = [&](const RowSlice& a, int lp) { return lp < a.pieces && (!RAG || lp >= a.begin); };
  [[maybe_unused]] auto inside = [&](const RowSlice& a, int lp) {
    return lp >= a.begin && ((int64_t)piece0 + lp + 1) * N <= a.shift + p.V;
  };

  // Rows are brought into L2 a few groups (plan.early) ahead of their first sweep, each group's pieces by
  // one thread of the warp whose turn it is.
  auto prefetch = [&](int64_t r, const void* base, int from, int count) {
    const RowSlice sn = slice_of(r);
    const int lo = max(from, sn.begin), n = min(sn.pieces, from + count) - lo;
    if (n > 0 && ADWIN_CHK(inside(sn, lo) && inside(sn, lo + n - 1), p.status))
      prefetch_l2(static_cast<const char*>(base) +
                      ((size_t)r * p.ld - sn.shift + (size_t)(piece0 + lo) * N) * sizeof(TIn),
                  (uint32_t)n * 16u);
  };

  if (TM) asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  if (cl > 1) cluster_sync_all();   // peers run before anything is stored into them
  __syncthreads();
  if (TM) asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == nw) {
    // ------------------------------------------------------------------ the row's own warp
    RowCursor cur;
    cur.init(p);
    bool wg_unused;
    // the entry beside row r's whole pieces that this lane looks after (lanes 0-7 before, 8-15 behind), or -1
    const bool edges = RAG && rank == 0 && (p.ld % N != 0 || p.V % N != 0);   // (rows of whole pieces have none)
    auto edge_of = [&](int64_t r) -> int64_t {
      if (!edges) return -1;
      const int shift = slice_of(r).shift, head = (N - shift % N) % N;
      if (lane < 8) return lane < head && lane < p.V ? lane : -1;
      const int64_t k = ((shift + p.V) / N) * N - shift + (lane - 8);   // (rows have several pieces)
      return lane < 16 && k < p.V ? k : -1;
    };
    auto fill = [&](int i, int64_t r) {    // row i's metadata into its slot
      if (!ADWIN_CHK(r >= 0 && r < p.B * p.T, p.status)) return;
      RowsMeta& m = ctrl.meta[i % kMetaDepth];
      const int y = p.tokens[r];
      m.r = r;
      m.y = y;
      float zy, uy;
      fetch_logits_at<TIn>(p, r, y, zy, uy);
      m.zy = zy;
      m.uy = uy;
      m.nref[0] = m.nref[1] = -zy * kLog2e;
      m.nref[2] = m.nref[3] = -uy * kLog2e;
      // (a token far from the others' differences, or masked in one policy, is no centre)
      const float dref = kCentred && fabsf(zy - uy) <= 16.f ? zy - uy : 0.f;
      m.dref = dref;
      m.nref[4] = m.nref[5] = -dref;
      m.nref[6] = m.nref[7] = 0.f;
      m.w = p.row_coef ? p.row_coef[r] : 0.f;
    };
    auto edge_logits = [&](int64_t r, float& z, float& u) {
      const int64_t k = edge_of(r);
      const bool has = k >= 0 && ADWIN_CHK(k < p.V && r < p.B * p.T, p.status);
      z = has ? Elem<TIn>::load1(p.student, r * p.ld + k) : kMaskedEdge;
      u = has ? Elem<TIn>::load1(p.teacher, r * p.ld + k) : kMaskedEdge;
    };
    auto put_edges = [&](int i, float z, float u) {
      if (!edges || lane >= kEdges) return;
      float* at = ctrl.meta[i % kMetaDepth].edge[lane];
      at[0] = z;
      at[1] = u;
    };
    auto row_of = [&](int i) { return cur.locate(p, cluster_id + (int64_t)i * plan.num_clusters, wg_unused); };
    auto fetch = [&](int i) {
      const int64_t r = row_of(i);
      if (lane == 0) fill(i, r);
      float z, u;
      edge_logits(r, z, u);
      put_edges(i, z, u);
    };
    // The first rows at once, a lane each (one after another they are three round trips to memory each).  Before
    // them the first row's first groups set out for L2; the rest follows as in every row.  (All of the row at once, and
    // its groups once more as their turn came: one row a CTA, 280 rows of 32 000 entries of bf16, 20.9 us, 19.6 so;
    // of 50 257 entries 27.6 and 25.5.)
    {
      const int n = min(kMetaAhead, my_rows);
      const int64_t r = row_of(min(lane, max(n - 1, 0)));
      if (lane == 0 && n > 0) {
        prefetch(r, p.student, 0, plan.early * kU * nt);
        prefetch(r, p.teacher, 0, plan.early * kU * nt);
      }
      float z[kMetaAhead], u[kMetaAhead];   // (all asked for before the first is stored)
#pragma unroll
      for (int i = 0; i < kMetaAhead; ++i) {
        const int64_t ri = __shfl_sync(0xffffffffu, r, i);
        if (i < n) edge_logits(ri, z[i], u[i]);
      }
      if (lane < n) fill(lane, r);
#pragma unroll
      for (int i = 0; i < kMetaAhead; ++i)
        if (i < n) put_edges(i, z[i], u[i]);
    }
    __syncthreads();
    int64_t r_prev = 0;
    float q_edge = 0.f;   // this lane's share of the previous row's squared norm
    // one more exchange than rows, for the last norm
    for (int i = 0; i <= my_rows && my_rows > 0; ++i) {
      const bool real = i < my_rows;
      const int par = i & 1;
      // (the others have begun no row before i - 1 ended, and read no further than kMetaAhead says)
      if (i + kMetaAhead < my_rows) fetch(i + kMetaAhead);
      named_sync(kPosted, all);
      // fixed-order sums over the threads, then over the CTAs: S and A, St and the norm (what kReady waits for
      // beside the others' issue slots: every operation counts here)
      ExactSum<kExact> sa[nw / 2], TQ;
      f2_t tq[nw / 2];
#pragma unroll
      for (int w = 0; w < nw / 2; ++w) {
        f2_t x, y, x2, y2;
        row_pairs(&rec[w * 32 + lane].x, x, y);
        row_pairs(&rec[(w + nw / 2) * 32 + lane].x, x2, y2);
        sa[w].set(x, x2);
        tq[w] = add2(y, y2);
      }
#pragma unroll
      for (int n = nw / 4; n > 0; n /= 2) {
#pragma unroll
        for (int w = 0; w < n; ++w) {
          sa[w].add(sa[w + n]);
          tq[w] = add2(tq[w], tq[w + n]);
        }
      }
      ExactSum<kExact> SA = sa[0];
      TQ.set(tq[0]);
      float ze = kMaskedEdge, ue = kMaskedEdge;
      if (edges) {
        float e_t = 0.f;
        if (real) {
          const RowsMeta& m = ctrl.meta[i % kMetaDepth];
          if (lane < kEdges) {
            ze = m.edge[lane][0];
            ue = m.edge[lane][1];
          }
          const float e = ex2f(fmaf(ze, kLog2e, m.nref[0]));
          SA.add(pk2(e, e * ((ze - ue) + m.nref[4])));
          e_t = ex2f(fmaf(ue, kLog2e, m.nref[2]));
        }
        TQ.add(pk2(e_t, q_edge));
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        SA.add(SA.of_lane_xor(o));
        TQ.add(TQ.of_lane_xor(o));
      }
      if (cl > 1) {
        if (lane < cl && ADWIN_CHK(rank < (uint32_t)kRowsMaxCl, p.status)) {
          const uint32_t dst = map_to_rank(smem_u32(ctrl.xrec[par][rank]), (uint32_t)lane);
          float v[8];
          upk2(SA.hi, v[0], v[1]);
          upk2(TQ.hi, v[2], v[3]);
          upk2(SA.lo, v[4], v[5]);
          upk2(TQ.lo, v[6], v[7]);
          remote_store4(dst, v[0], v[1], v[2], v[3]);
          remote_store4(dst + 16, v[4], v[5], v[6], v[7]);
        }
        cluster_sync_all();
        SA.set(0ull);
        TQ.set(0ull);
        for (int j = 0; j < cl; ++j) {
          ExactSum<kExact> x, y;
          row_pairs(ctrl.xrec[par][j], x.hi, y.hi);
          row_pairs(ctrl.xrec[par][j] + 4, x.lo, y.lo);
          SA.add(x);
          TQ.add(y);
        }
      }
      RowTotals t;
      float S_off, A_off, St_off, q, q_off;
      upk2(SA.hi, t.S, t.A);
      upk2(SA.lo, S_off, A_off);
      upk2(TQ.hi, t.St, q);
      upk2(TQ.lo, St_off, q_off);
      t.St += St_off;
      if (rank == 0 && lane == 0 && i > 0 && p.gsq) p.gsq[r_prev] = isfinite(q) ? q + q_off : q;
      if (!real) break;
      const RowsMeta& m = ctrl.meta[i % kMetaDepth];
      const int64_t ri = m.r;
      t.M2s = m.zy * kLog2e;
      t.M2t = m.uy * kLog2e;
      t.B0 = t.B1 = t.B2 = 0.f;
      // (the totals are identical in every CTA of the cluster, so this branch is too; an infinite sum's St_off is
      // not a number)
      if (!(t.S < kSumLimit) || !(t.St < kSumLimit)) {
        if (lane == 0) ctrl.out.again = 1;
        named_sync(kReady, all);
        named_sync(kPosted, all);
        float x[5] = {-INFINITY, -INFINITY, 0.f, 0.f, 0.f};   // m2s, m2t, S, A, St of the CTA
        if (lane < nw) {
#pragma unroll
          for (int f = 0; f < 5; ++f) x[f] = ctrl.safe[lane][f];
        }
        if (edges && edge_of(ri) >= 0) {   // this lane's entry beside the pieces
          RowAcc ra;
          ra.m2s = x[0]; ra.m2t = x[1]; ra.S = x[2]; ra.A = x[3]; ra.St = x[4];
          const float z1[1] = {ze}, u1[1] = {ue};
          acc_piece<1, false>(z1, u1, m.dref, ra);
          x[0] = ra.m2s; x[1] = ra.m2t; x[2] = ra.S; x[3] = ra.A; x[4] = ra.St;
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
        S_off = A_off = 0.f;
      }
      const bool y_valid = m.y >= 0 && (int64_t)m.y < p.V;
      const float inv0 = 1.f / t.S, inv = kExact ? fmaf(-S_off * inv0, inv0, inv0) : inv0;
      // the mean of delta over the row, as a sum of two floats
      const float about = t.A * inv;
      const float about_off = (fmaf(-about, t.S, t.A) + fmaf(-about, S_off, A_off)) * inv;
      const float near_mean = about + m.dref, back = near_mean - about;
      const float near_off = ((about - (near_mean - back)) + (m.dref - back)) + about_off;
      float mean = near_mean + near_off, rest = near_off - (mean - near_mean);
      if (!isfinite(mean)) {   // (a difference of logits that is: no rounding to look after)
        mean = near_mean;
        rest = 0.f;
      }
      float coef = p.alpha * inv, nc0 = -mean, nm2s = -t.M2s;
      if constexpr (FULLKL && sizeof(TIn) == 2) {
        // bf16 logits: g = e * (coef*delta - coef*mean) saves one operation per pair; its rounding
        // (relative to coef*delta, not to the difference) is far inside that dtype's tolerance.  But that of
        // coef*mean is common to the row, and a peaked row's norm, all of it from a delta beside the mean, is off
        // by twice the rounding times mean / (delta - mean).  Another reference for e makes another coefficient: of 32
        // references 2^-16 apart the one whose coefficient needs the least rounding in its product with
        // the mean is taken.  (2^-s = 1 - x + x^2 / 2 with x = s ln 2 < 2e-4; the next term is 2^-39.)
        // An infinite mean, of a teacher's entry masked by -infinity, has no rounding to look after.
        if (kCentred && fabsf(coef) > 1e-30f && fabsf(coef) < 1e30f && fabsf(mean) < 1e30f) {
          const float ref = nm2s + (float)(lane - 16) * 0x1p-16f;     // (rounded: the step is the difference below)
          const float x = (ref - nm2s) * 0.69314718f, c = fmaf(coef, x * fmaf(x, 0.5f, -1.f), coef);
          const float prod = c * mean, low = fmaf(c, rest, fmaf(c, mean, -prod)), near = prod + low;
          const float off = fabsf(low - (near - prod));
          const unsigned best = __reduce_min_sync(0xffffffffu, (__float_as_uint(off) & ~31u) | (unsigned)lane) & 31u;
          nm2s = __shfl_sync(0xffffffffu, ref, (int)best);
          nc0 = -__shfl_sync(0xffffffffu, near, (int)best);
          coef = __shfl_sync(0xffffffffu, c, (int)best);
        } else {
          nc0 = -coef * mean;
        }
      }
      auto publish = [&](float gy) {
        if (lane == 0) {
          ctrl.out.nm2s[0] = ctrl.out.nm2s[1] = nm2s;
          ctrl.out.coef[0] = ctrl.out.coef[1] = coef;
          ctrl.out.nc0[0] = ctrl.out.nc0[1] = nc0;
          ctrl.out.gy = gy;
          ctrl.out.again = 0;
        }
        named_sync(kReady, all);
      };
      // what the second sweep of Eq. 2's gradient takes needs no logarithm (as finish_row has it)
      if constexpr (FULLKL) publish(0.f);
      const RowScalars rs = finish_row(t, m.zy, m.uy, y_valid, m.dref, p.alpha, FULLKL ? ADWIN_GRAD_FULL_KL : ADWIN_GRAD_SAMPLED,
                                       p.row_coef ? &m.w : nullptr, p.lse_s || p.lse_t);
      if constexpr (!FULLKL) {
        coef = rs.coef;
        publish(rs.gy);
      }
      if (edges) {   // the gradient of the edge entries, as in the second sweep
        const int64_t k = edge_of(ri);
        const float e = ex2f(fmaf(ze, kLog2e, nm2s));
        float g;
        if (!FULLKL) g = k == m.y ? rs.gy : e * coef;
        else if (sizeof(TIn) == 2) g = e * fmaf(ze - ue, coef, nc0);
        else g = e * ((ze - ue + nc0) * coef);
        q_edge = k >= 0 ? g * g : 0.f;
        if (k >= 0 && ADWIN_CHK(k < p.V && ri < p.B * p.T, p.status))
          Elem<TOut>::store1(p.grad, ri * p.ld_grad + k, g);
      }
      if (lane == 0) {
        if (rank == 0 && ADWIN_CHK(ri >= 0 && ri < p.B * p.T, p.status)) {
          p.kl[ri] = (mean - rs.lse_diff) + rest;
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
    __syncthreads();   // the first rows' metadata
    // this thread's tensor-memory columns: its lane, the columns split between the warps of a lane group
    const uint32_t tm_lane = TM ? ctrl.tmem_base + ((uint32_t)((warp & 3) * 32) << 16) +
                                      (uint32_t)((warp >> 2) * plan.tm_groups * group_cols)
                                : 0u;
    const int ring = plan.groups + plan.ahead;
    int pos = 0;              // the ring's group that comes next

    // ---- loads: the pieces of the first sweep's next group, always one group ahead of it
    uint4 zn[kU], un[kU];
    const char* zp = nullptr;   // the next piece of the student's row to be loaded
    int left = 0;               // pieces of the slice from it on
    bool before = false;        // (the piece belongs to the row before: only the first one may)
    int load_row = -1, load_group = 0;
    const ptrdiff_t to_teacher = static_cast<const char*>(p.teacher) - static_cast<const char*>(p.student);
    auto load = [&](int h, uint4 (&zn)[kU], uint4 (&un)[kU]) {
      if (left > h * nt && !(RAG && h == 0 && before) &&
          ADWIN_CHK((zp - static_cast<const char*>(p.student)) + (h * nt + 1) * 16 <=
                        ((p.B * p.T - 1) * p.ld + p.V) * (int64_t)sizeof(TIn), p.status)) {
        zn[h] = __ldcs(reinterpret_cast<const uint4*>(zp) + h * nt);
        un[h] = __ldcs(reinterpret_cast<const uint4*>(zp + to_teacher) + h * nt);
      }
    };
    auto next_load_row = [&]() {
      ++load_row;
      load_group = 0;
      left = 0;
      if (load_row < my_rows) {
        const int64_t r = ctrl.meta[load_row % kMetaDepth].r;
        const RowSlice sn = slice_of(r);
        zp = static_cast<const char*>(p.student) +
             ((size_t)r * p.ld - sn.shift + (size_t)(piece0 + tid) * N) * sizeof(TIn);
        left = sn.pieces - tid;
        if (RAG) before = tid < sn.begin;
      }
    };
    auto loaded = [&]() {       // a whole group has been asked for
      zp += kU * array;
      left -= kU * nt;
      before = false;
      if (++load_group == plan.groups) next_load_row();
    };

    // ---- first sweep: the row's sums and copies
    RowSlice sp1 = slice_of(0);   // (without RAG the same for all rows)
    const float* refs = nullptr;
    Acc2 a;
    auto begin_sums = [&](int i) {
      const RowsMeta& m = ctrl.meta[i % kMetaDepth];
      if (RAG) sp1 = slice_of(m.r);
      refs = m.nref;
      a.reset();
    };
    // ---- second sweep: what it takes of its row
    RowSlice sp2 = sp1;
    f2_t Q[kNorms] = {};
    float gy = 0.f;
    int yleft = -1;           // pieces from this thread's next one to the sampled token's (< 0: passed, or elsewhere)
    int ye = 0;
    char* gp = nullptr;

    // One group: the second sweep's group g2 (TWO) and the first sweep's group g1 of the row after (ONE),
    // which takes its place in the ring.  g1's pieces are in zn and un; with LOAD the next in line replace them.
    auto group_of = [&](auto one_, auto two_, auto full_, auto load_, int g1, int g2, uint4 (&zn)[kU],
                        uint4 (&un)[kU]) __attribute__((always_inline)) {
      constexpr bool ONE = decltype(one_)::value, TWO = decltype(two_)::value, FULL = decltype(full_)::value;
      constexpr bool LOAD = decltype(load_)::value;
      const bool in_tm = TM && pos < plan.tm_groups;
      const uint32_t tm_at = TM ? tm_lane + (uint32_t)(pos * group_cols) : 0u;
      char* st = stash + (size_t)((uint32_t)(pos - plan.tm_groups) * group_bytes);
      const int l1 = tid + g1 * (kU * nt), l2 = tid + g2 * (kU * nt);   // this thread's pieces of the first step
      const f2_t L2 = splat2(kLog2e), NEG1 = splat2(-1.f);
      f2_t nM2s, coef2, nc0, nrefs, nreft, ndref, unused;
      if constexpr (TWO) {
        row_pairs(ctrl.out.nm2s, nM2s, coef2);
        if constexpr (FULLKL) row_pairs(ctrl.out.nc0, nc0, unused);
      }
      if constexpr (ONE) {
        row_pairs(refs, nrefs, nreft);
        if constexpr (kCentred) row_pairs(refs + 4, ndref, unused);
      }
#pragma unroll
      for (int h = 0; h < kU; ++h) {
        if constexpr (TWO) {
          const int lp = l2 + h * nt;
          uint4 z, u;
          if (in_tm) {   // (every lane takes part)
            if (ADWIN_CHK(columns_ok(pos), p.status)) {
              if constexpr (FULLKL) tm_load8(tm_at + (uint32_t)(h * 8), z, u);
              else tm_load4(tm_at + (uint32_t)(h * 4), z);
              tm_wait_ld();
            }
          } else if ((FULL || holds(sp2, lp)) && ADWIN_CHK(stash_ok(st), p.status)) {
            z = *reinterpret_cast<const uint4*>(st + kKept * h * array);
            if constexpr (FULLKL) u = *reinterpret_cast<const uint4*>(st + (kKept * h + 1) * array);
          }
          if (FULL || holds(sp2, lp)) {
            f2_t Z[NP], U[NP], G[NP];
            Pairs<TIn>::make(z, Z);
            if constexpr (FULLKL) Pairs<TIn>::make(u, U);
#pragma unroll
            for (int e = 0; e < NP; ++e) {
              const f2_t E = ex2_2(fma2(Z[e], L2, nM2s));
              if constexpr (FULLKL) {
                if (sizeof(TIn) == 2) G[e] = mul2(E, fma2(fma2(U[e], NEG1, Z[e]), coef2, nc0));
                else G[e] = mul2(E, mul2(add2(fma2(U[e], NEG1, Z[e]), nc0), coef2));
              } else {
                G[e] = mul2(E, coef2);
              }
            }
            if constexpr (!FULLKL) {
              if (yleft == h * nt) {
#pragma unroll
                for (int e = 0; e < NP; ++e) {
                  float lo, hi;
                  upk2(G[e], lo, hi);
                  if (ye == 2 * e) lo = gy;
                  if (ye == 2 * e + 1) hi = gy;
                  G[e] = pk2(lo, hi);
                }
              }
            }
#pragma unroll
            for (int e = 0; e < NP; ++e) Q[h % kNorms] = fma2(G[e], G[e], Q[h % kNorms]);
            char* dst = gp + (size_t)h * nt * N * sizeof(TOut);
            if (ADWIN_CHK(inside(sp2, lp), p.status)) {
              store_pairs<TOut, NP>(dst, G);
            }
          }
        }
        if constexpr (ONE) {
          const int lp = l1 + h * nt;
          if (in_tm) {   // (every lane takes part)
            if (ADWIN_CHK(columns_ok(pos), p.status)) {
              if constexpr (FULLKL) tm_store8(tm_at + (uint32_t)(h * 8), zn[h], un[h]);
              else tm_store4(tm_at + (uint32_t)(h * 4), zn[h]);
            }
          } else if ((FULL || holds(sp1, lp)) && ADWIN_CHK(stash_ok(st), p.status)) {
            *reinterpret_cast<uint4*>(st + kKept * h * array) = zn[h];
            if constexpr (FULLKL) *reinterpret_cast<uint4*>(st + (kKept * h + 1) * array) = un[h];
          }
          if (FULL || holds(sp1, lp)) {
            f2_t Z[NP], U[NP];
            Pairs<TIn>::make(zn[h], Z);
            Pairs<TIn>::make(un[h], U);
            if constexpr (kCentred) acc_grad_centred<NP>(Z, U, nrefs, nreft, ndref, a);
            else acc_grad<NP, 0>(Z, U, nrefs, nreft, a);
          }
          if constexpr (LOAD) load(h, zn, un);
        }
      }
      if constexpr (TWO) {
        gp += (size_t)kU * nt * N * sizeof(TOut);
        if constexpr (!FULLKL) yleft -= kU * nt;
      }
      if constexpr (ONE && LOAD) loaded();
      pos = pos + 1 == ring ? 0 : pos + 1;
    };
    constexpr std::true_type yes{};
    constexpr std::false_type no{};
    auto group = [&](auto one, auto two, auto full, int g1, int g2) __attribute__((always_inline)) {
      group_of(one, two, full, yes, g1, g2, zn, un);
    };
    // the group `plan.early` groups behind group g of row i in the order of the first sweeps
    auto early = [&](int i, int g) {
      if (warp == g % nw && lane == 0) {
        g += plan.early;
        if (g >= plan.groups) {
          g -= plan.groups;
          ++i;
        }
        if (i < my_rows) {
          const int64_t r = ctrl.meta[i % kMetaDepth].r;
          prefetch(r, p.student, g * kU * nt, kU * nt);
          prefetch(r, p.teacher, g * kU * nt, kU * nt);
        }
      }
    };
    auto post = [&](float q) {
      rec[tid] = make_float4(hsum2(a.S), hsum2(a.A), hsum2(a.St), q);
      named_arrive(kPosted, all);
      if (cl > 1) cluster_arrive_relaxed();
    };

    next_load_row();
#pragma unroll
    for (int h = 0; h < kU; ++h) load(h, zn, un);
    loaded();
#pragma unroll 1
    for (int i = -1; i < my_rows; ++i) {
      const bool next = i + 1 < my_rows;
      if (RAG) sp2 = sp1;
      // the next row's first groups (all of them for the first row), into the part of the ring that this
      // row does not take: this row's sums travel meanwhile
      if (next) {
        begin_sums(i + 1);
        const int to = i < 0 ? plan.groups : plan.ahead;
        if (i >= 0) pos = pos + plan.groups >= ring ? pos - plan.ahead : pos + plan.groups;
        int g = 0;
        // The first row has no second sweep beside it to fill the time of a load: two groups are in flight.  Clusters of
        // two, 60 rows of 151 936 entries of bf16: 23.6 us with one, 22.7 with two; 1400 rows 226 and 220.  (Not in the other
        // kernels: {2, 256} and rows off the lines pay for the registers in the loop below, 700 rows of 50 257 entries
        // 49.0 -> 53.5 us; fp32 rows, which have less to do per byte, gain nothing.)
        if constexpr (sizeof(TIn) == 2 && NT == kRowsThreads && !RAG) {
          const int whole = i < 0 ? min(to, full_to(sp1)) : 0;
#pragma unroll 1
          for (; g + 2 <= whole; g += 2) {
            early(i + 1, g);
            early(i + 1, g + 1);
            uint4 z2[kU], u2[kU];
#pragma unroll
            for (int h = 0; h < kU; ++h) load(h, z2, u2);
            loaded();
            group_of(yes, no, yes, yes, g, 0, zn, un);
            group_of(yes, no, yes, no, g + 1, 0, z2, u2);
          }
        }
#pragma unroll 1
        for (; g < to; ++g) {
          early(i + 1, g);
          if (ALONE && g >= full_from(sp1) && g < full_to(sp1)) {
            if constexpr (ALONE) group(yes, no, yes, g, 0);
          } else {
            group(yes, no, no, g, 0);
          }
        }
      }
      if (i < 0) {
        pos = 0;
        if (next) post(0.f);
        continue;
      }
      const RowsMeta& m = ctrl.meta[i % kMetaDepth];
      if (cl > 1) cluster_wait();
      named_sync(kReady, all);
      if (TM) tm_wait_st();

      // -------------------------------------------------------------- overflow: running maxima
      if (ctrl.out.again) {
        RowAcc ra;
        ra.reset();
        const uint4* uq = nullptr;
        if (!FULLKL)
          uq = reinterpret_cast<const uint4*>(
                   static_cast<const char*>(p.teacher) +
                   ((size_t)m.r * p.ld - sp2.shift + (size_t)piece0 * N) * sizeof(TIn)) + tid;
#pragma unroll 1
        for (int k = 0; k < plan.groups * kU; ++k) {
          const int at = pos + k / kU >= ring ? pos + k / kU - ring : pos + k / kU;
          const int lp = tid + k * nt;
          uint4 zv = make_uint4(0u, 0u, 0u, 0u), uv = zv;
          if (TM && at < plan.tm_groups) {
            if (!ADWIN_CHK(columns_ok(at), p.status)) break;
            const uint32_t col = tm_lane + (uint32_t)(at * group_cols + k % kU * kKept * 4);
            if (FULLKL) tm_load8(col, zv, uv);
            else tm_load4(col, zv);
            tm_wait_ld();
          } else if (holds(sp2, lp)) {
            const char* st = stash + (size_t)((uint32_t)(at - plan.tm_groups) * group_bytes);
            if (!ADWIN_CHK(stash_ok(st), p.status)) break;
            zv = *reinterpret_cast<const uint4*>(st + k % kU * kKept * array);
            if (FULLKL) uv = *reinterpret_cast<const uint4*>(st + (k % kU * kKept + 1) * array);
          }
          if (holds(sp2, lp)) {
            if (!FULLKL && ADWIN_CHK(inside(sp2, lp), p.status)) uv = __ldg(uq + k * nt);
            float z[N], u[N];
            Elem<TIn>::unpack(zv, z);
            Elem<TIn>::unpack(uv, u);
            acc_piece<N, false>(z, u, m.dref, ra);
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

      // -------------------------------------------------------------- second sweep, next row's first
      {
        gy = ctrl.out.gy;
        const int64_t yat = (int64_t)m.y + sp2.shift;                     // counted from piece 0
        const bool y_valid = m.y >= 0 && (int64_t)m.y < p.V;
        yleft = y_valid ? (int)(yat / N - piece0) - tid : -1;             // (slice-relative)
        ye = (int)(yat % N);
        gp = static_cast<char*>(p.grad) +
             ((size_t)m.r * p.ld_grad - sp2.shift + (size_t)(piece0 + tid) * N) * sizeof(TOut);
        Q[0] = Q[kNorms - 1] = 0ull;
      }
      const int groups = plan.groups, both = next ? groups - plan.ahead : 0;
      // whole groups of both rows
      const int lo = max(full_from(sp2), full_from(sp1) - plan.ahead), hi = min(full_to(sp2), full_to(sp1) - plan.ahead);
#pragma unroll 1
      for (int g = 0; g < groups; ++g) {
        const int g1 = g + plan.ahead;
        if (g >= both) {
          if (ALONE && g >= full_from(sp2) && g < full_to(sp2)) {
            if constexpr (ALONE) group(no, yes, yes, 0, g);
          } else {
            group(no, yes, no, 0, g);
          }
        } else {
          early(i + 1, g1);
          if (g >= lo && g < hi) group(yes, yes, yes, g1, g);
          else group(yes, yes, no, g1, g);
        }
      }
      if (!next) a.reset();
      post(hsum2(kNorms > 1 ? add2(Q[0], Q[kNorms - 1]) : Q[0]));
    }
    if (cl > 1 && my_rows > 0) cluster_wait();
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

constexpr int shape_smem(int ctas) { return kSmemPerSm / ctas - kSmemReserved; }

// kept: arrays of which the second sweep needs a copy (2, or the student's alone).
constexpr bool shape_plan(const RowsShape& sh, int64_t pieces, int kept, RowsPlan& plan) {
  plan.cl = sh.cl;
  plan.nt = sh.nt;
  plan.ctas = sh.ctas;
  plan.per_rank = (int)((pieces + sh.cl - 1) / sh.cl + kLine / 16 - 1) / (kLine / 16) * (kLine / 16);   // whole lines
  plan.groups = (plan.per_rank + sh.nt * kU - 1) / (sh.nt * kU);
  plan.early = plan.groups < kMostEarly ? plan.groups : kMostEarly;
  const int sm_groups = (shape_smem(sh.ctas) - rows_ctrl_bytes(sh.nt)) / (kU * kept * 16 * sh.nt);
  // a lane group's columns are shared by its warps (every fourth); a piece takes 4 columns
  const int tm_groups = sh.tm_cols ? sh.tm_cols / ((sh.nt + 127) / 128) / (kU * kept * 4) : 0;
  const int spare = sm_groups + tm_groups - plan.groups;
  if (spare < 0) return false;
  // one group covers the exchange of two CTAs on an SM, of one CTA two, a cluster's takes three (151 936 entries
  // 418 us with two, 410 with three; 80 000 entries 395 with one, 391 with two); more only run the sweeps apart
  // (32 000 entries 404 with one, 409 with two)
  const int most = sh.cl > 1 ? 3 : sh.ctas == 1 ? 2 : 1;
  plan.ahead = spare < most ? spare : most;
  if (plan.ahead > plan.groups) plan.ahead = plan.groups;
  const int ring = plan.groups + plan.ahead;
  plan.tm_groups = ring < tm_groups ? ring : tm_groups;
  plan.tm_cols = plan.tm_groups ? sh.tm_cols : 0;
  return true;
}

constexpr int rows_smem(const RowsPlan& plan, int kept) {
  return rows_ctrl_bytes(plan.nt) +
         (plan.groups + plan.ahead - plan.tm_groups) * kU * kept * 16 * plan.nt;
}

// Bytes a launch asks for.  The CTAs of a cluster hold tensor memory while they wait for one another,
// and tcgen05.alloc waits without a limit: beside a tensor-core kernel of another stream (CTA pairs
// with all 512 columns), a cluster and a pair could each hold an SM's columns and wait for the other's.
// So the CTAs of a cluster take at least kClusterSmem: no CTA of tc_pipeline.cuh (199 KB), nor any
// above 112 KB, and no other cluster's fits on an SM beside one.  (A CTA without a cluster waits for
// nobody once it has its columns.)  Not the whole share of an SM, which would leave 28 KB of L1 to the
// streaming kernel that follows in a call with scalars over the rollout (update and audit on 3.8 GB of
// logits 1215 us so, 1164 with less).
constexpr int kClusterSmem = kSmemPerSm / 2;
constexpr int launch_smem(const RowsPlan& plan, int kept) {
  const int need = rows_smem(plan, kept);
  return plan.cl > 1 && plan.tm_cols > 0 && need < kClusterSmem ? kClusterSmem : need;
}
constexpr bool clusters_exclude_one_another_and_tensor_core_ctas() {
  for (const RowsShape& sh : kShapes) {
    RowsPlan plan = {};
    for (int kept = 1; kept <= 2; ++kept)
      for (int64_t pieces = sh.cl; sh.cl > 1 && shape_plan(sh, pieces, kept, plan); pieces += sh.cl * sh.nt * kU)
        if (plan.tm_cols > 0 &&
            (launch_smem(plan, kept) + tc::kSmemBytes + 2 * kSmemReserved <= kSmemPerSm ||
             2 * (launch_smem(plan, kept) + kSmemReserved) <= kSmemPerSm))
          return false;
  }
  return true;
}
static_assert(clusters_exclude_one_another_and_tensor_core_ctas(), "a cluster could wait for another's tensor memory");

constexpr bool metadata_precedes_its_readers() {
  for (const RowsShape& sh : kShapes) {
    RowsPlan plan = {};
    for (int kept = 1; kept <= 2; ++kept)
      for (int64_t pieces = 1; shape_plan(sh, pieces, kept, plan); pieces += sh.cl * sh.nt * kU) {
        // the last rows, counted from i, that are loaded from and brought into L2 before row i's kReady
        const int loaded = 1 + (plan.ahead + 1) / plan.groups;
        const int prefetched = plan.ahead ? 1 + (plan.ahead - 1 + plan.early) / plan.groups : 1;
        if (loaded >= kMetaAhead || prefetched >= kMetaAhead) return false;
      }
  }
  return kMetaAhead + 1 < kMetaDepth;   // row i - 1 is in use while that of row i + kMetaAhead is written
}
static_assert(metadata_precedes_its_readers(), "a row's metadata could be read before it is written");

typedef void (*RowsKernel)(KlParams, RowsPlan);
// (72 kernels: two types in and out, four thread counts, on and off the lines, both estimators -- the sampled-token
// one keeps half as much, 151 936 entries on one CTA and not two -- and some with ALONE both ways.)
// ALONE: a call of one row a CTA has lone sweeps only (280 rows of 32 000 entries of bf16 23.4 us with the tests
// there, 20.9 without), one of many rows a group or two a row, beside whose code the loop of both sweeps comes out faster
// or slower.  2.4 GB without / with it: bf16 rows on the lines 4 096 entries 451 / 446 us, 20 032 452 / 437, 80 000 449 /
// 420; fp32 4 096 376 / 382; off the lines 5 000 513 / 570, 9 001 506 / 564, 33 001 447 / 456, 50 257 415 / 424, 80 001 408 /
// 414, sampled 421 / 414; sampled 32 000 413 / 435.  Calls of few rows do not take the small shapes; most of those of 256
// threads are built both ways.
constexpr bool lone_sweeps(int nt, bool ragged, bool full_kl, bool few, size_t entry) {
  if (nt == 256) return few || (full_kl && !ragged);
  return nt > 256 || (!ragged && entry == 2);
}
template <typename TIn, typename TOut, int NT, bool RAG, bool FULLKL>
RowsKernel rows_kernel_of(bool few) {
  constexpr bool TM = uses_tensor_memory(NT);
  constexpr bool kFew = lone_sweeps(NT, RAG, FULLKL, true, sizeof(TIn));
  constexpr bool kMany = lone_sweeps(NT, RAG, FULLKL, false, sizeof(TIn));
  return few ? kl_rows_kernel<TIn, TOut, NT, TM, RAG, FULLKL, kFew>
             : kl_rows_kernel<TIn, TOut, NT, TM, RAG, FULLKL, kMany>;
}
template <typename TIn, typename TOut, int NT>
RowsKernel rows_kernel_nt(bool ragged, bool full_kl, bool few) {
  if (full_kl) return ragged ? rows_kernel_of<TIn, TOut, NT, true, true>(few) : rows_kernel_of<TIn, TOut, NT, false, true>(few);
  return ragged ? rows_kernel_of<TIn, TOut, NT, true, false>(few) : rows_kernel_of<TIn, TOut, NT, false, false>(few);
}
template <typename TIn, typename TOut>
RowsKernel rows_kernel(int nt, bool ragged, bool full_kl, bool few) {
  switch (nt) {
    case 64: return rows_kernel_nt<TIn, TOut, 64>(ragged, full_kl, few);
    case 128: return rows_kernel_nt<TIn, TOut, 128>(ragged, full_kl, few);
    case 256: return rows_kernel_nt<TIn, TOut, 256>(ragged, full_kl, few);
    case kRowsThreads: return rows_kernel_nt<TIn, TOut, kRowsThreads>(ragged, full_kl, few);
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
  const RowsKernel like = kl_rows_kernel<float, float, kRowsThreads, false, false, true, false>;
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

// The plan of a call of at most `rows` rows, and how many rows the GPU holds at a time so.
cudaError_t rows_plan(int64_t pieces, int kept, int64_t rows, int sm_count, RowsPlan& plan) {
  if (pieces < 1 || pieces > (int64_t)1 << 24) return cudaErrorNotSupported;
  const RowsShape* by_length = std::begin(kShapes);
  while (!(pieces <= by_length->most && shape_plan(*by_length, pieces, kept, plan)))
    if (++by_length == std::end(kShapes)) return cudaErrorNotSupported;
  for (const RowsShape* sh = std::end(kShapes) - 1;; --sh) {
    plan.num_clusters = sh->ctas * sm_count / sh->cl;
    const bool wider = sh != by_length;
    if (wider && (!sh->few || pieces < sh->few || rows > plan.num_clusters)) continue;
    if (!shape_plan(*sh, pieces, kept, plan)) continue;
    if (plan.cl > 1) {
      const cudaError_t e = resident_clusters(plan, sm_count, plan.num_clusters);
      if (wider && e == cudaErrorNotSupported) continue;
      if (e != cudaSuccess) return e;
    }
    if (wider && rows > plan.num_clusters) continue;
    return cudaSuccess;
  }
}

template <typename TIn, typename TOut>
cudaError_t launch_rows_t(const KlParams& p, bool ragged, int sm_count, cudaStream_t s) {
  constexpr int N = Elem<TIn>::N;
  RowsPlan plan = {};
  const bool full_kl = p.mode == ADWIN_GRAD_FULL_KL;
  const int kept = full_kl ? 2 : 1;
  // Rows of whole pieces off the lines: pieces are counted from the line (see RowSlice) except in short bf16 rows, which
  // lose more by the groups that are then partial at both ends.  2.4 GB, from the line / from the row: 4 104 entries 572 /
  // 537 us, 5 000 513 / 495, 7 000 518 / 484, 9 000 493 / 466, 20 008 436 / 440, 50 264 427 / 443; fp32 2 500 395 / 431.
  const bool off_lines = (p.ld * sizeof(TIn)) % kLine != 0 || reinterpret_cast<uintptr_t>(p.student) % kLine != 0;
  ragged = ragged || (off_lines && (sizeof(TIn) == 4 || p.V > kShortRow));
  const int64_t lead = ragged ? kLine / (int64_t)sizeof(TIn) - 1 : 0;   // entries of a line before the row, at most
  cudaError_t e = rows_plan((lead + p.V + N - 1) / N, kept, p.plan_rows, sm_count, plan);
  if (e != cudaSuccess) return e;
  const RowsKernel kernel = rows_kernel<TIn, TOut>(plan.nt, ragged, full_kl, p.B * p.T <= plan.num_clusters);
  if (!kernel) return cudaErrorNotSupported;
  if (plan.num_clusters > p.B * p.T) plan.num_clusters = (int)(p.B * p.T);
  const int smem = launch_smem(plan, kept);
  // the shape's whole share whatever this call needs: the limit belongs to the kernel, which launches of
  // other threads with other row lengths use at the same time
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, shape_smem(plan.ctas));
  if (e != cudaSuccess) return e;
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
