// K1b: similarity S = Xhat Xhat^T (Eq. 7) on the 5th-generation tensor cores
// (BF16 or FP8-E4M3 operands, FP32 accumulation in TMEM) with the selection of
// each row's K best columns (Eq. 8).  S never leaves the SM.
//
// The main path is three kernels.  A sampling pass scores every row against a
// few hundred columns and keeps a rank of them as the row's floor; the append
// pass (CTA pairs, 16 epilogue warps) computes the whole square and appends the
// columns that reach a row's floor to its segments; k_select sorts out the K best.
// The list kernels, whose epilogue keeps a sorted list per row, serve the
// rechecks, a request's gallery rows, single CTAs and tight budgets:
//
// One persistent CTA per SM walks work items (row block of 128 rows, chunk of
// 256-column tiles); items are ordered so that CTAs running together share
// the chunk, so the column tiles they stream are L2 hits, and so that a row's
// later chunks run after its earlier ones (see the floors below).  Roles:
//   warp 0 (one thread)  TMA producer: per k-block, the 128-row A slab and
//                        the 256-row B slab (128-byte swizzle) into a
//                        4-stage shared-memory ring;
//   warp 1 (one thread)  MMA issuer: 4 tcgen05.mma (K = 16 BF16 / 32 FP8) per
//                        k-block into one of two 128 x 256 FP32 accumulators
//                        in TMEM (512 columns), commit frees the ring slot;
//                        the tile's last commit hands the accumulator over;
//   warps 2-5 (or 2-9)    epilogue: each thread owns one TMEM lane = one row,
//                        reads its 256 scores with tcgen05.ld (32 at a time),
//                        applies the FP8 row/column scales, sets S_ii = 1 and
//                        admits the columns that beat the row's threshold into
//                        its sorted top-K list; then releases the accumulator
//                        (pairs: the lists are in shared memory, merged by the
//                        whole warp).
// The two accumulators let the MMA of tile t+1 run under the epilogue of
// tile t.  At the end of a work item the list is written as one
// partial candidate list per (row, chunk), merged and certified by K2.
//
// Split mode (the recheck of rows whose list could not be certified): the
// operands are the hi/lo BF16 halves of the unit rows, x = hi + lo + r, and
// the k-loop runs three times over the feature dimension so that the one
// accumulator collects hi_i.hi_j + lo_i.hi_j + hi_i.lo_j.  The A rows are the
// gathered rows being rechecked; their count is read on the device.
#include <cuda.h>
#include <cfloat>
#include <atomic>
#include <climits>
#include <cmath>

#include <cstdlib>
#include <type_traits>

#include "common.cuh"
#include "f32x2.cuh"
#include "internal.hpp"
#include "tc_ptx.cuh"
#include "topk_heap.cuh"  // score_key / key_score

namespace rr {
namespace {

constexpr int TBM = 128;
constexpr int TBN = 256;
constexpr int STAGES = 4;  // ring stages of a single CTA
constexpr int A_BYTES = TBM * 128;    // one 128-byte swizzle row per operand row
constexpr int B_BYTES = TBN * 128;
constexpr int KLIST = 64;  // largest candidate list the kernel supports
// Epilogue warp groups: group g owns columns [g, g+1) * TBN / EG of every tile
// and keeps its own list per row (EG lists per row and chunk).  Two groups
// when the MMA work per tile is short (K depth <= 1024), so that the
// epilogue keeps pace; one otherwise (fewer, longer lists).
constexpr int EG_MAX = 2;
constexpr int AEG = 4;  // epilogue groups of the append pass: 64 columns of every tile each
constexpr int threads_of(int eg) { return 64 + 128 * eg; }  // TMA warp, MMA warp, 4 epilogue warps per group
constexpr uint32_t WAIT_LIMIT = 1u << 22;

// BF16 / FP8: one matrix against itself (or a rectangular block);
// SPLIT: gathered rows, hi/lo products; GATHER: gathered rows, one BF16 product.
enum { MODE_BF16 = 0, MODE_FP8 = 1, MODE_SPLIT = 2, MODE_GATHER = 3 };
__host__ __device__ constexpr bool gathered(int mode) { return mode == MODE_SPLIT || mode == MODE_GATHER; }

// The operand ring comes first: its slots are 1024-byte aligned (128-byte swizzle).
template <int STG, int BBYTES>
struct TcRing {
  static constexpr int kStages = STG;
  uint8_t a[STG][A_BYTES];
  uint8_t b[STG][BBYTES];
};

// Barriers and the dynamic item order's ring (see next_item).
constexpr int IQ = 4;  // item ring depth
template <int STG>
struct TcSync {
  uint64_t full[STG];
  uint64_t empty[STG];
  uint64_t tfull[2];
  uint64_t tempty[2];
  uint64_t done;
  int item_q[IQ];
  uint64_t ifull[IQ];
  uint64_t iempty[IQ];
  uint32_t tmem_base;
  int abort;
};

// Shared memory of a single CTA (its lists live in registers).
struct alignas(1024) TcSmem : TcRing<STAGES, B_BYTES>, TcSync<STAGES> {
  float batch[EG_MAX][32][TBM];  // per group: scores of the 32 columns being folded in
};

// Shared memory of a CTA of a pair: it holds only its half of the B rows (128
// of the tile's 256), and per row and epilogue group the sorted list of the
// KL best columns so far and a queue of QN admitted ones not yet in it.
// Columns are 16-bit offsets from the item's first column (an item covers at
// most kMaxItemTiles tiles).  The odd row strides (in 4-byte words) keep both
// access patterns free of bank conflicts: a lane per row at the same place,
// and a warp over consecutive places of one row.
constexpr int pair_stages(int kl, int egn) { return egn == 2 ? 3 : (kl > 48 ? 4 : 5); }
template <int KL, int EGN>
struct alignas(1024) TcSmemPair : TcRing<pair_stages(KL, EGN), B_BYTES / 2>, TcSync<pair_stages(KL, EGN)> {
  static constexpr int QN = EGN == 2 && KL > 48 ? 16 : 32;
  float ls[EGN * TBM][KL + 1];
  float qs[EGN * TBM][QN + 1];
  uint16_t lc[EGN * TBM][KL + 2];
  uint16_t qc[EGN * TBM][QN + 2];
};
constexpr int kMaxItemTiles = 256;
// Pairs whose epilogue keeps nothing in shared memory (sampling and append
// passes): operand stages only.
struct alignas(1024) TcSmemRing : TcRing<6, B_BYTES / 2>, TcSync<6> {};

// What the epilogue does with the scores.
enum { KIND_LISTS = 0, KIND_SAMPLE = 1, KIND_APPEND = 2 };
template <bool PAIR, int KL, int EG, int KIND>
using SmemOf = typename std::conditional<
    KIND != KIND_LISTS, TcSmemRing, typename std::conditional<PAIR, TcSmemPair<KL, EG>, TcSmem>::type>::type;

// Batched launches: up to kMaxBatchInst instances, each a matrix against
// itself; their tensor maps travel as one kernel parameter.
constexpr int kMaxBatchInst = 64;
struct TcMaps {
  CUtensorMap m[kMaxBatchInst];
};
struct TcMaps2 {  // the instances' maps, then those of their samples
  CUtensorMap m[2 * kMaxBatchInst];
};
struct TcInst {
  int64_t n;                // rows = columns of the instance
  int row_blocks, col_tiles, chunks, kblocks, K;
  int item_begin;           // first item of the instance in the launch's item space
  const float* inv_scale;
  int* row_floor;
  float* part_s;
  int32_t* part_i;
  uint2* cand;              // append pass: rows x segs x cap admitted (score bits, vertex)
  int32_t* seg_cnt;         // rows x segs
  int cap;
  int floor_rank;           // sampling pass
  const float* sample_scale;
  long long* status;
};

struct TcArgs {
  int64_t n;                // columns of B (valid column indices 0 .. n-1)
  int64_t a_rows;           // outside split mode: valid rows of A
  int64_t row0;             // outside split mode: vertex index of A row 0
  int64_t col0;             // vertex index of B column 0
  int row_blocks;           // outside split mode
  int col_tiles, chunks, kblocks, K;
  const float* inv_scale;   // FP8 only: 1 / s_i per row
  const int32_t* rows;      // split mode: global row of each A row
  const int32_t* count;     // split mode: number of A rows
  int* row_floor;           // per A row: score_key of the best K-th score any finished chunk found
  int stall;                // test hook: the TMA warp issues nothing, so every wait runs out
  float* part_s;
  int32_t* part_i;
  long long* status;
  const TcInst* insts;      // batched launch: the instances (device memory), else null
  int ninst, items_total;
  const float* sample_scale;  // sampling pass, FP8: 1 / s_i of the sampled columns
  int floor_rank;           // sampling pass: which largest maximum becomes the floor
  uint2* cand;              // append pass: rows x (chunks * AEG) x cap admitted (score bits, vertex)
  int32_t* seg_cnt;         // append pass: entries per segment; cap + 1 when it ran over
  int cap;
  int rb0;                  // append pass: first row block of the launch (cand holds its rows on)
  int mb_off;               // batched sampling pass: index of instance 0's sample map
  int* work;                // non-null: items are taken in order from this counter (zero at launch)
};

// One work item (a row block against a chunk of column tiles) with the
// parameters of its instance.
struct TcItem {
  const CUtensorMap* ma0;
  const CUtensorMap* ma1;
  const CUtensorMap* mb0;
  const CUtensorMap* mb1;
  int rb, chunk, t0, t1, kblocks, K, chunks;
  int64_t n, nrows, row0, col0;
  const float* inv_scale;
  int* row_floor;
  float* part_s;
  int32_t* part_i;
  uint2* cand;
  int32_t* seg_cnt;
  int cap, floor_rank;
  const float* sample_scale;
};

// Gathered launches (recheck): the row count is known on the device only, so
// the number of column chunks is chosen there, by the host's rule (whole waves
// of items over the grid, each chunk charged three tiles for its cold start),
// up to the A.chunks lists per row the caller reads (and, where that many
// chunks allow it, no item of more than kMaxItemTiles tiles).
__device__ __forceinline__ int pick_chunks(int row_blocks, int maxc, int col_tiles, int grid) {
  int best = maxc;
  long long best_cost = LLONG_MAX;
  for (int c = tmin(maxc, (col_tiles + kMaxItemTiles - 1) / kMaxItemTiles); c <= maxc; ++c) {
    const long long waves = (static_cast<long long>(row_blocks) * c + grid - 1) / grid;
    const long long cost = waves * ((col_tiles + c - 1) / c + 3);
    if (cost < best_cost) {
      best_cost = cost;
      best = c;
    }
  }
  return best;
}

// chunks: column chunks of this launch (<= A.chunks, the lists per row in the output).
template <bool BATCH>
__device__ __forceinline__ void get_item(const TcArgs& A, const CUtensorMap* ma0, const CUtensorMap* ma1,
                                         const CUtensorMap* mb0, const CUtensorMap* mb1, const CUtensorMap* bmaps,
                                         int row_blocks, int64_t nrows, int item, TcItem& it, int chunks) {
  if (!BATCH) {
    it.ma0 = ma0;
    it.ma1 = ma1;
    it.mb0 = mb0;
    it.mb1 = mb1;
    it.rb = A.rb0 + item % row_blocks;
    it.chunk = item / row_blocks;
    it.t0 = int(int64_t(it.chunk) * A.col_tiles / chunks);
    it.t1 = int(int64_t(it.chunk + 1) * A.col_tiles / chunks);
    it.kblocks = A.kblocks;
    it.K = A.K;
    it.chunks = A.chunks;
    it.n = A.n;
    it.nrows = nrows;
    it.row0 = A.row0;
    it.col0 = A.col0;
    it.inv_scale = A.inv_scale;
    it.row_floor = A.row_floor;
    it.part_s = A.part_s;
    it.part_i = A.part_i;
    it.cand = A.cand;
    it.seg_cnt = A.seg_cnt;
    it.cap = A.cap;
    it.floor_rank = A.floor_rank;
    it.sample_scale = A.sample_scale;
  } else {
    int lo = 0, hi = A.ninst - 1;  // last instance whose items begin at or before `item`
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (A.insts[mid].item_begin <= item) lo = mid;
      else hi = mid - 1;
    }
    const TcInst& I = A.insts[lo];
    const int local = item - I.item_begin;
    it.ma0 = it.ma1 = bmaps + lo;
    it.mb0 = it.mb1 = bmaps + A.mb_off + lo;
    it.rb = local % I.row_blocks;
    it.chunk = local / I.row_blocks;
    it.t0 = int(int64_t(it.chunk) * I.col_tiles / I.chunks);
    it.t1 = int(int64_t(it.chunk + 1) * I.col_tiles / I.chunks);
    it.kblocks = I.kblocks;
    it.K = I.K;
    it.chunks = I.chunks;
    it.n = I.n;
    it.nrows = I.n;
    it.row0 = 0;
    it.col0 = 0;
    it.inv_scale = I.inv_scale;
    it.row_floor = I.row_floor;
    it.part_s = I.part_s;
    it.part_i = I.part_i;
    it.cand = I.cand;
    it.seg_cnt = I.seg_cnt;
    it.cap = I.cap;
    it.floor_rank = I.floor_rank;
    it.sample_scale = I.sample_scale;
  }
}

// Timeout: every instance of the launch reports it.
template <bool BATCH>
__device__ void report_timeout(const TcArgs& A) {
  if (!BATCH) {
    set_error(A.status, kErrTimeout);
  } else {
    for (int k = 0; k < A.ninst; ++k) set_error(A.insts[k].status, kErrTimeout);
  }
}



// Give loads this CTA issued time to land before it leaves (pair mode, after a
// timeout: their bytes complete on the even CTA's barrier, which this CTA
// cannot poll).  A tile load takes microseconds; wait about 200 us.
__device__ __forceinline__ void drain_delay() {
  for (int k = 0; k < 200; ++k) __nanosleep(1000);
}

// Insert (cs, ci) into a row's sorted list: slot j takes cs where cs first
// beats ls[j], and slot j-1's old entry for every later slot.  For the sorted
// scores that is max(min(ls[j-1], cs), ls[j]); the columns follow the same
// choice.  All tests use the old list: no serial dependency.  Columns arrive
// in increasing order, so an equal score keeps the earlier, lower column in
// front (score desc, column asc); cs = -inf changes nothing.
template <int KL>
__device__ __forceinline__ void list_insert(float (&ls)[KL], int (&li)[KL], float cs, int ci) {
#pragma unroll
  for (int j = KL - 1; j > 0; --j) {
    const bool bj = cs > ls[j], bp = cs > ls[j - 1];
    li[j] = bp ? li[j - 1] : (bj ? ci : li[j]);
    ls[j] = fmaxf(fminf(ls[j - 1], cs), ls[j]);
  }
  li[0] = cs > ls[0] ? ci : li[0];
  ls[0] = fmaxf(cs, ls[0]);
}

// Item order.  Static: unit, unit + units, ...  Dynamic (A.work set): the
// publisher (the TMA thread of a CTA, or of the even CTA of a pair) takes the
// next item number from the global counter and hands it to every consumer of
// the work through a ring in shared memory (both CTAs' rings for a pair):
// the MMA thread, the epilogue warps and, in the odd CTA of a pair, its TMA
// thread.  A slot is reused once all consumers released it on the even CTA's
// `iempty`.  Items still come in increasing order overall, but a unit that
// finishes early takes more of them, which evens out the per-item cost of the
// top-K epilogue.  Every consumer reads the same sequence; the first number
// >= items ends it.
struct ItemRing {
  uint32_t qs = 0, qph = 0;
};

template <bool PAIR, class Smem>
__device__ __forceinline__ int next_item(Smem& sm, const TcArgs& A, bool publisher, bool leader, int prev, int unit,
                                         int units, ItemRing& rg, volatile int* abort, bool& ok) {
  if (!A.work) return prev < 0 ? unit : prev + units;
  int it = INT_MAX;
  if (publisher) {
    it = atomicAdd(A.work, 1);
    if (!tc::mbar_wait(&sm.iempty[rg.qs], rg.qph ^ 1u, abort, WAIT_LIMIT)) {
      ok = false;
      return INT_MAX;
    }
    reinterpret_cast<volatile int*>(sm.item_q)[rg.qs] = it;
    if (PAIR) {
      tc::st_cluster(tc::map_to_rank(&sm.item_q[rg.qs], 1), it);
      tc::mbar_arrive_cluster(tc::map_to_rank(&sm.ifull[rg.qs], 1));
    }
    tc::mbar_arrive(&sm.ifull[rg.qs]);
  } else {
    const bool got = PAIR ? tc::mbar_wait_cluster(&sm.ifull[rg.qs], rg.qph, abort, WAIT_LIMIT)
                          : tc::mbar_wait(&sm.ifull[rg.qs], rg.qph, abort, WAIT_LIMIT);
    if (!got) {
      ok = false;
      return INT_MAX;
    }
    it = reinterpret_cast<volatile int*>(sm.item_q)[rg.qs];
    if (PAIR && !leader) tc::mbar_arrive_cluster(tc::map_to_rank(&sm.iempty[rg.qs], 0));
    else tc::mbar_arrive(&sm.iempty[rg.qs]);
  }
  if (++rg.qs == IQ) {
    rg.qs = 0;
    rg.qph ^= 1u;
  }
  return it;
}

// A whole warp waits for an accumulator.  The lanes' waits run out one by one,
// so they agree on the outcome: a lane that gave up alone would be missing from
// the warp's TMEM loads and votes.
template <class Smem>
__device__ __forceinline__ bool wait_tile(Smem& sm, uint32_t ab, uint32_t phase) {
  return __all_sync(kFull, tc::mbar_wait(&sm.tfull[ab], phase, &sm.abort, WAIT_LIMIT));
}

// One warp takes the next item from the ring (lane 0) and shares it.
template <bool PAIR, class Smem>
__device__ __forceinline__ int take_item(Smem& sm, const TcArgs& A, bool leader, int prev, int unit, int units,
                                         ItemRing& rg, int lane, bool& ok) {
  int v = 0;
  bool good = true;
  if (lane == 0) v = next_item<PAIR>(sm, A, false, leader, prev, unit, units, rg, &sm.abort, good);
  v = __shfl_sync(kFull, v, 0);
  good = __shfl_sync(kFull, good ? 1 : 0, 0) != 0;
  if (!good) ok = false;
  return v;
}

// Merges a row's queue of cnt <= 32 admitted columns into its sorted list of
// the K best (K <= KL <= 64), by the whole warp: an entry's new place is its
// own place plus the number of entries of the other sequence that go before
// it.  The queue's columns come after the list's, so an equal score keeps the
// list's entry (and, inside the queue, the earlier entry) in front: score
// descending, column ascending.  List entries are counted against the queue's
// scores (one shuffle each), queue entries by a binary search in the list;
// nothing here is a serial chain, so a merge of 28 entries costs about 300
// issue slots, about 11 per entry.
template <int KL>
__device__ __forceinline__ void merge_row(float* ls, uint16_t* lc, const float* qs, const uint16_t* qc, int cnt,
                                          int K, int lane) {
  const float q = lane < cnt ? qs[lane] : -INFINITY;
  const uint16_t qcol = lane < cnt ? qc[lane] : uint16_t(0);
  const int j1 = lane + kWarp;
  const float a = lane < K ? ls[lane] : -INFINITY;
  const float b = j1 < K ? ls[j1] : -INFINITY;
  const uint16_t ac = lane < K ? lc[lane] : uint16_t(0);
  const uint16_t bc = j1 < K ? lc[j1] : uint16_t(0);
  // list entries that go before this queue entry
  int before = 0;
#pragma unroll
  for (int step = KL > 48 ? 64 : 32; step > 0; step >>= 1) {
    const int e = before + step;
    if (e <= K && ls[e - 1] >= q) before = e;
  }
  int ra = lane, rb = j1, rq = before;
  for (int u0 = 0; u0 < cnt; u0 += 8) {
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const float su = __shfl_sync(kFull, q, u0 + u);
      ra += su > a ? 1 : 0;
      rb += su > b ? 1 : 0;
      rq += (su > q || (su == q && u0 + u < lane)) ? 1 : 0;
    }
  }
  __syncwarp();
  if (lane < cnt && rq < K) {
    ls[rq] = q;
    lc[rq] = qcol;
  }
  if (lane < K && ra != lane && ra < K) {
    ls[ra] = a;
    lc[ra] = ac;
  }
  if (j1 < K && rb != j1 && rb < K) {
    ls[rb] = b;
    lc[rb] = bc;
  }
  __syncwarp();
}

// The CTA's shared memory block.
template <class Smem>
__device__ __forceinline__ Smem& smem_block() {
  extern __shared__ uint8_t smem_raw[];
  return *reinterpret_cast<Smem*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
}

// Merges the queues of `rows` (one bit per lane of the warp), one after
// another.  w0: the warp's first row in the list arrays; qn: each lane's queue length.
template <class Smem, int KL>
__device__ __noinline__ void merge_rows(unsigned rows, int w0, int qn, int K, int lane) {
  Smem& sm = smem_block<Smem>();
  __syncwarp();  // the queue entries written by their lanes
  while (rows) {
    const int r = __ffs(rows) - 1;
    rows &= rows - 1u;
    merge_row<KL>(sm.ls[w0 + r], sm.lc[w0 + r], sm.qs[w0 + r], sm.qc[w0 + r], __shfl_sync(kFull, qn, r), K, lane);
  }
}

// Appends (s, col) to a queue when s > thr: five predicated instructions, no branch.
__device__ __forceinline__ void queue_push(uint32_t& aqs, uint32_t& aqc, float s, float thr, int col) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.gt.f32 p, %2, %3;\n\t"
      "@p st.shared.f32 [%0], %2;\n\t@p st.shared.u16 [%1], %4;\n\t"
      "@p add.u32 %0, %0, 4;\n\t@p add.u32 %1, %1, 2;\n\t}\n"
      : "+r"(aqs), "+r"(aqc)
      : "f"(s), "f"(thr), "h"(uint16_t(col))
      : "memory");
}

// Epilogue of the paired kernels: warps 2 .. 2 + 4 EGROUPS.  Warp w reads TMEM
// lanes 32 (w % 4) .. + 31 (its rows); the groups split the tile's columns, and
// each keeps its own list per row (EGROUPS lists per chunk).
//
// What bounds it: at d <= 1024 the MMAs of a tile are shorter than the scan of
// its 128 x 256 scores and the list updates.  A lane per row scans the
// scores four at a time (the maximum of the four against the row's threshold,
// one vote per group) and appends what is admitted to the row's queue in
// shared memory; a queue about to overflow is merged into the row's list by
// the whole warp (merge_row).
template <int MODE, int KL, int EGROUPS, bool BATCH, class Smem>
__device__ __forceinline__ bool epilogue_pair(Smem& sm, const CUtensorMap* pA0, const CUtensorMap* pA1,
                                              const CUtensorMap* pB0, const CUtensorMap* pB1,
                                              const CUtensorMap* bmaps, const TcArgs& A, uint32_t tmem, uint32_t rank,
                                              int row_blocks, int64_t nrows, int items, int chunks) {
  constexpr int QN = Smem::QN;
  constexpr int NBATCH = TBN / 32 / EGROUPS;  // batches of 32 columns per tile and group
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool leader = rank == 0;
  const int unit = int(blockIdx.x >> 1), units = int(gridDim.x >> 1);
  const int q = warp & 3;
  const int eg = (warp - 2) >> 2;
  const uint32_t tlane = tmem + (uint32_t(q * 32) << 16);
  const uint32_t tempty_leader0 = tc::map_to_rank(&sm.tempty[0], 0);
  const uint32_t tempty_leader1 = tc::map_to_rank(&sm.tempty[1], 0);
  const int w0 = eg * TBM + q * 32;  // the warp's first row in the list arrays
  float* const my_ls = sm.ls[w0 + lane];
  const uint32_t aqs0 = tc::smem_u32(sm.qs[w0 + lane]), aqc0 = tc::smem_u32(sm.qc[w0 + lane]);
  uint32_t tcount = 0;
  bool ok = true;
  ItemRing rg;
  for (int item = take_item<true>(sm, A, leader, -1, unit, units, rg, lane, ok); item < items && ok;
       item = take_item<true>(sm, A, leader, item, unit, units, rg, lane, ok)) {
    TcItem it;
    get_item<BATCH>(A, pA0, pA1, pB0, pB1, bmaps, row_blocks, nrows, item, it, chunks);
    const int K = it.K;
    const int64_t arow0 = int64_t(it.rb) * (2 * TBM) + int(rank) * TBM + q * 32;  // the warp's first A row
    const int64_t arow = arow0 + lane;
    const bool live = arow < it.nrows;
    const int64_t grow = gathered(MODE) ? (live ? int64_t(A.rows[arow]) : -1) : it.row0 + arow;  // vertex
    for (int j = 0; j < K; ++j) my_ls[j] = -FLT_MAX;  // an empty place
    uint32_t aqs = aqs0, aqc = aqc0;  // next free places of the row's queue (shared-memory addresses)
    // Admission: beat the list's K-th best so far and reach the row's floor (s >= floor,
    // i.e. s > the float below it).  The floor is the best K-th score any
    // chunk of this row has published: chunks publish their running K-th
    // after every tile, and an item re-reads the floor before every tile,
    // so chunks of a row that run at the same time raise each other's bar.
    // A partial list's K-th best is at most the row's final K-th best, so a
    // column below the floor can never be among the row's K best.
    int seen = live ? __ldcg(it.row_floor + arow) : INT_MAX;  // floor key in use (also: last published)
    float kth = -FLT_MAX;                                      // the list's K-th best
    float thr = live ? nextafterf(key_score(seen), -INFINITY) : INFINITY;
    const float rinv = (MODE == MODE_FP8 && live) ? it.inv_scale[grow] : 1.0f;
    // Merge the queues of `rows` and raise their lanes' thresholds.
    auto merge = [&](unsigned rows) {
      merge_rows<Smem, KL>(rows, w0, int(aqs - aqs0) >> 2, K, lane);
      if ((rows >> lane) & 1u) {
        aqs = aqs0;
        aqc = aqc0;
        kth = my_ls[K - 1];
        thr = fmaxf(thr, kth);
      }
    };
    for (int ct = it.t0; ct < it.t1; ++ct) {
      const int fk = (live && ct > it.t0) ? __ldcg(it.row_floor + arow) : seen;
      const uint32_t ab = tcount & 1u, tph = (tcount >> 1) & 1u;
      if (!wait_tile(sm, ab, tph)) {
        ok = false;
        break;
      }
      tc::tc_fence_after();
      if (fk > seen) {
        seen = fk;
        thr = fmaxf(thr, nextafterf(key_score(fk), -INFINITY));
      }
      const int64_t tbase = int64_t(ct) * TBN;  // the tile's first B column
      const int64_t dtile = grow - (it.col0 + tbase);
      const bool patch = __any_sync(kFull, live && dtile >= 0 && dtile < TBN) || tbase + TBN > it.n;
      const uint32_t ta = tlane + ab * TBN + eg * (TBN / EGROUPS);
      const int ctile = (ct - it.t0) * TBN + eg * (TBN / EGROUPS);  // its columns' offset in the item
      auto fold = [&](uint32_t (&v)[32], int cb) {
        const int lb = eg * (TBN / EGROUPS) + cb * 32;  // column in the tile
        if (MODE == MODE_FP8) {
          const float* si = it.inv_scale + it.col0 + tbase + lb;
          const int nv = int(tmin<int64_t>(it.n - tbase - lb, 32));
#pragma unroll
          for (int j = 0; j < 32; ++j)
            v[j] = __float_as_uint(__uint_as_float(v[j]) * rinv * __ldg(j < nv ? si + j : it.inv_scale));
        }
        if (patch) {
          // the diagonal (S_ii = 1) and the columns past the last one
          const int jself = int(tmax<int64_t>(tmin<int64_t>(dtile - lb, 32), -1));
          const int nv = int(tmax<int64_t>(tmin<int64_t>(it.n - tbase - lb, 32), 0));
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            if (j == jself) v[j] = __float_as_uint(1.0f);
            if (j >= nv) v[j] = __float_as_uint(-INFINITY);
          }
        }
        const int cbase = ctile + cb * 32;
#pragma unroll
        for (int g = 0; g < 32; g += 4) {
          const float s0 = __uint_as_float(v[g]), s1 = __uint_as_float(v[g + 1]), s2 = __uint_as_float(v[g + 2]),
                      s3 = __uint_as_float(v[g + 3]);
          if (__any_sync(kFull, fmaxf(fmaxf(s0, s1), fmaxf(s2, s3)) > thr)) {
            queue_push(aqs, aqc, s0, thr, cbase + g);
            queue_push(aqs, aqc, s1, thr, cbase + g + 1);
            queue_push(aqs, aqc, s2, thr, cbase + g + 2);
            queue_push(aqs, aqc, s3, thr, cbase + g + 3);
            const unsigned full = __ballot_sync(kFull, aqs > aqs0 + (QN - 4) * 4);
            if (full) merge(full);
          }
        }
      };
      // Two batches per TMEM wait (no load stays in flight across the merge's call).
      uint32_t va[32], vb[32];
#pragma unroll 1
      for (int cb = 0; cb < NBATCH; cb += 2) {
        tc::tmem_ld32(ta + cb * 32, va);
        tc::tmem_ld32(ta + (cb + 1) * 32, vb);
        tc::tmem_wait_ld(va);
        tc::tmem_wait_ld(vb);
        fold(va, cb);
        fold(vb, cb + 1);
      }
      tc::tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (leader) tc::mbar_arrive(&sm.tempty[ab]);
        else tc::mbar_arrive_cluster(ab ? tempty_leader1 : tempty_leader0);
      }
      ++tcount;
      // Publish this chunk's running K-th best when it raises the row's floor.
      if (live && ct + 1 < it.t1 && kth != -FLT_MAX) {
        const int key = score_key(kth);
        if (key > seen) {
          atomicMax(it.row_floor + arow, key);
          seen = key;
        }
      }
    }
    if (!ok) break;
    const unsigned left = __ballot_sync(kFull, aqs > aqs0);
    if (left) merge(left);
    __syncwarp();
    // The lists, row by row (a row's places are contiguous here and in the output).
    const int vbase = int(it.col0 + int64_t(it.t0) * TBN);  // vertex of offset 0
    const int nlive = int(tmax<int64_t>(tmin<int64_t>(it.nrows - arow0, 32), 0));
    const size_t row_step = size_t(it.chunks) * EGROUPS * K;
    size_t o = ((size_t(arow0) * it.chunks + it.chunk) * EGROUPS + eg) * K;
    for (int rr = 0; rr < nlive; ++rr, o += row_step) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int j = lane + h * kWarp;
        if (j < K) {
          const float sc = sm.ls[w0 + rr][j];
          it.part_s[o + j] = sc;
          it.part_i[o + j] = sc == -FLT_MAX ? kInvalidIdx : vbase + int(sm.lc[w0 + rr][j]);
        }
      }
    }
    if (live) {
      // This chunk's K-th best becomes a floor for the row's later chunks.
      if (kth != -FLT_MAX) atomicMax(it.row_floor + arow, score_key(kth));
      // Lists of chunks this launch does not use are empty (first entry invalid).
      if (gathered(MODE) && it.chunk == 0)
        for (int c = chunks; c < it.chunks; ++c) {
          const size_t oe = ((size_t(arow) * it.chunks + c) * EGROUPS + eg) * K;
          it.part_s[oe] = -FLT_MAX;
          it.part_i[oe] = kInvalidIdx;
        }
    }
    __syncwarp();  // the lists are reused by the next item
  }
  return ok;
}

// Epilogue of the sampling pass (one epilogue group): every row's scores
// against the sampled columns only; the floor_rank-th largest of the maxima of
// 64 interleaved column groups becomes the row's floor (KR: the largest rank,
// a compile-time bound).  One maximum per score, 128 KR instructions per row
// at the end.
template <int MODE, int KR, bool BATCH, class Smem>
__device__ __forceinline__ bool epilogue_sample(Smem& sm, const CUtensorMap* pA0, const CUtensorMap* pB0,
                                                const CUtensorMap* bmaps, const TcArgs& A, uint32_t tmem,
                                                uint32_t rank, int row_blocks, int64_t nrows, int items, int chunks) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool leader = rank == 0;
  const int unit = int(blockIdx.x >> 1), units = int(gridDim.x >> 1);
  const int q = warp & 3;
  const uint32_t tlane = tmem + (uint32_t(q * 32) << 16);
  const uint32_t tempty_leader0 = tc::map_to_rank(&sm.tempty[0], 0);
  const uint32_t tempty_leader1 = tc::map_to_rank(&sm.tempty[1], 0);
  uint32_t tcount = 0;
  for (int item = unit; item < items; item += units) {
    TcItem it;
    get_item<BATCH>(A, pA0, pA0, pB0, pB0, bmaps, row_blocks, nrows, item, it, chunks);
    const int64_t arow = int64_t(it.rb) * (2 * TBM) + int(rank) * TBM + q * 32 + lane;
    float m[64];
#pragma unroll
    for (int j = 0; j < 64; ++j) m[j] = -FLT_MAX;
    for (int ct = it.t0; ct < it.t1; ++ct) {
      const uint32_t ab = tcount & 1u, tph = (tcount >> 1) & 1u;
      if (!wait_tile(sm, ab, tph)) return false;
      tc::tc_fence_after();
#pragma unroll 1
      for (int cb = 0; cb < TBN / 32; cb += 2) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t v[32];
          tc::tmem_ld32(tlane + ab * TBN + (cb + h) * 32, v);
          tc::tmem_wait_ld(v);
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            float sc = __uint_as_float(v[j]);
            if (MODE == MODE_FP8) sc *= __ldg(it.sample_scale + int64_t(ct) * TBN + (cb + h) * 32 + j);
            m[h * 32 + j] = fmaxf(m[h * 32 + j], sc);
          }
        }
      }
      tc::tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (leader) tc::mbar_arrive(&sm.tempty[ab]);
        else tc::mbar_arrive_cluster(ab ? tempty_leader1 : tempty_leader0);
      }
      ++tcount;
    }
    float top[KR];
#pragma unroll
    for (int k = 0; k < KR; ++k) top[k] = -FLT_MAX;
#pragma unroll
    for (int j = 0; j < 64; ++j) {
      float t = m[j];
#pragma unroll
      for (int k = 0; k < KR; ++k) {
        const float hi = fmaxf(top[k], t);
        t = fminf(top[k], t);
        top[k] = hi;
      }
    }
    if (arow < it.nrows) {
      float f = -FLT_MAX;
#pragma unroll
      for (int k = 0; k < KR; ++k)
        if (k == it.floor_rank - 1) f = top[k];
      if (MODE == MODE_FP8) f *= it.inv_scale[arow];
      it.row_floor[arow] = score_key(f);
    }
  }
  return true;
}

// Appends (score, col) at p when score > thr: predicated, no branch.
__device__ __forceinline__ void cand_push(uint64_t& p, uint32_t score, float thr, int col) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.gt.f32 p, %2, %3;\n\t"
      "@p st.global.v2.b32 [%0], {%1, %4};\n\t@p add.u64 %0, %0, 8;\n\t}\n"
      : "+l"(p)
      : "r"(score), "f"(__uint_as_float(score)), "f"(thr), "r"(col)
      : "memory");
}

// Epilogue of the append pass: AEG groups of four warps, each scanning 64
// columns of every tile for its 32 rows.  Every column that reaches the row's
// floor is appended to the row's segment for this (chunk, group) in global
// memory; the selection (k_select) sorts out the K best afterwards.  Nothing is
// kept in order here and no state is shared, so 16 warps fit beside a
// six-stage ring and hide the TMEM, vote and branch latencies that bounded the
// list epilogues at d <= 1024.  A segment with no room for 32 more columns
// takes no more and is marked; its row goes to the recheck.
//
// Measured on a GB300, the similarity stage with per-row lists kept in
// registers (before) and with floors, append and selection (now), lists of 42:
//   n = 23,100, d = 128: 0.983 -> 0.378 ms (append alone 0.30, MMA and hand-over alone 0.14)
//   n = 50,000, d = 512: 3.45 -> 1.74 ms (append alone 1.57, MMA and hand-over alone 1.47)
//   n = 9,973, d = 511: 0.404 -> 0.149 ms
//   n = 23,100, d = 2048: 1.337 -> 1.321 ms (append alone 1.19 = 0.97 of the MMA rate)
template <int MODE, bool BATCH, class Smem>
__device__ __forceinline__ bool epilogue_append(Smem& sm, const CUtensorMap* pA0, const CUtensorMap* pB0,
                                                const CUtensorMap* bmaps, const TcArgs& A, uint32_t tmem,
                                                uint32_t rank, int row_blocks, int64_t nrows, int items, int chunks) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool leader = rank == 0;
  const int unit = int(blockIdx.x >> 1), units = int(gridDim.x >> 1);
  const int q = warp & 3;
  const int eg = (warp - 2) >> 2;
  constexpr int GC = TBN / AEG;  // columns per tile and group
  const uint32_t tlane = tmem + (uint32_t(q * 32) << 16) + uint32_t(eg * GC);
  const uint32_t tempty_leader0 = tc::map_to_rank(&sm.tempty[0], 0);
  const uint32_t tempty_leader1 = tc::map_to_rank(&sm.tempty[1], 0);
  uint32_t tcount = 0;
  bool ok = true;
  ItemRing rg;
  for (int item = take_item<true>(sm, A, leader, -1, unit, units, rg, lane, ok); item < items && ok;
       item = take_item<true>(sm, A, leader, item, unit, units, rg, lane, ok)) {
    TcItem it;
    get_item<BATCH>(A, pA0, pA0, pB0, pB0, bmaps, row_blocks, nrows, item, it, chunks);
    const int64_t arow = int64_t(it.rb) * (2 * TBM) + int(rank) * TBM + q * 32 + lane;
    const bool live = arow < it.nrows;
    // s >= floor, i.e. s > the float below it
    float thr = live ? nextafterf(key_score(__ldg(it.row_floor + arow)), -INFINITY) : INFINITY;
    const float rinv = (MODE == MODE_FP8 && live) ? it.inv_scale[arow] : 1.0f;
    const f32x2 rinv2 = twice(rinv);
    const bool wide = MODE == MODE_FP8 && (reinterpret_cast<uintptr_t>(it.inv_scale) & 15) == 0;
    const size_t brow = live ? size_t(arow - int64_t(A.rb0) * (2 * TBM)) : 0;  // the row's place in the band
    const size_t seg = brow * (it.chunks * AEG) + it.chunk * AEG + eg;
    const uint64_t p0 = reinterpret_cast<uint64_t>(it.cand + seg * it.cap);
    const uint64_t plast = p0 + 8u * (it.cap - 32);  // beyond it a batch might not fit
    uint64_t p = p0;
    bool over = false;
    for (int ct = it.t0; ct < it.t1; ++ct) {
      const uint32_t ab = tcount & 1u, tph = (tcount >> 1) & 1u;
      if (!wait_tile(sm, ab, tph)) {
        ok = false;
        break;
      }
      tc::tc_fence_after();
      const int64_t c0 = int64_t(ct) * TBN + eg * GC;  // the group's first column of the tile
      const int64_t dself = arow - c0;
      const bool patch = __any_sync(kFull, live && dself >= 0 && dself < GC) || c0 + GC > it.n;
      uint32_t va[32], vb[32];
      tc::tmem_ld32(tlane + ab * TBN, va);
      tc::tmem_ld32(tlane + ab * TBN + 32, vb);
      tc::tmem_wait_ld(va);
      tc::tmem_wait_ld(vb);
      tc::tc_fence_before();
      __syncwarp();
      if (lane == 0) {  // the scores are in registers: the accumulator is free
        if (leader) tc::mbar_arrive(&sm.tempty[ab]);
        else tc::mbar_arrive_cluster(ab ? tempty_leader1 : tempty_leader0);
      }
      ++tcount;
      auto fold = [&](uint32_t (&v)[32], int h) {
        const int lb = h * 32;
        if (MODE == MODE_FP8) {
          // Both rows' scales, in packed products of two columns with the scales
          // loaded by fours where they are aligned (a request's may not be):
          // similarity stage at Market 0.88 -> 0.82 ms (bounding a tile's scores
          // by its largest scale first gained nothing: most groups of four hold
          // a candidate of some row).
          const float* si = it.inv_scale + c0 + lb;
          if (!patch && wide) {
#pragma unroll
            for (int j = 0; j < 32; j += 4) {
              const ulonglong2 f = __ldg(reinterpret_cast<const ulonglong2*>(si + j));
              const f32x2 a = mul2(mul2(f32x2(v[j]) | (f32x2(v[j + 1]) << 32), rinv2), f.x);
              const f32x2 b = mul2(mul2(f32x2(v[j + 2]) | (f32x2(v[j + 3]) << 32), rinv2), f.y);
              v[j] = uint32_t(a);
              v[j + 1] = uint32_t(a >> 32);
              v[j + 2] = uint32_t(b);
              v[j + 3] = uint32_t(b >> 32);
            }
          } else {
            const int nv = int(tmin<int64_t>(it.n - c0 - lb, 32));
#pragma unroll
            for (int j = 0; j < 32; ++j)
              v[j] = __float_as_uint(__uint_as_float(v[j]) * rinv * __ldg(j < nv ? si + j : it.inv_scale));
          }
        }
        if (patch) {
          // the diagonal (S_ii = 1) and the columns past the last one
          const int jself = int(tmax<int64_t>(tmin<int64_t>(dself - lb, 32), -1));
          const int nv = int(tmax<int64_t>(tmin<int64_t>(it.n - c0 - lb, 32), 0));
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            if (j == jself) v[j] = __float_as_uint(1.0f);
            if (j >= nv) v[j] = __float_as_uint(-INFINITY);
          }
        }
        if (p > plast) {
          thr = INFINITY;
          over = true;
        }
        // Groups of four columns: a lane flags those whose maximum beats its
        // threshold, one reduction tells the warp which groups any lane flagged,
        // and only their columns are pushed.
        unsigned flags = 0;
#pragma unroll
        for (int g = 0; g < 8; ++g) {
          const float m = fmaxf(fmaxf(__uint_as_float(v[4 * g]), __uint_as_float(v[4 * g + 1])),
                                fmaxf(__uint_as_float(v[4 * g + 2]), __uint_as_float(v[4 * g + 3])));
          flags |= m > thr ? (1u << g) : 0u;
        }
        const unsigned act = __reduce_or_sync(kFull, flags);
        const int cbase = int(c0) + lb;
#pragma unroll
        for (int g = 0; g < 8; ++g) {
          if (act & (1u << g)) {
#pragma unroll
            for (int j = 4 * g; j < 4 * g + 4; ++j) cand_push(p, v[j], thr, cbase + j);
          }
        }
      };
      fold(va, 0);
      fold(vb, 1);
    }
    if (!ok) break;
    if (live) it.seg_cnt[seg] = over ? it.cap + 1 : int32_t((p - p0) >> 3);
  }
  return ok;
}

// Epilogue of the single-CTA kernels: as epilogue_pair, with each row's list
// in its lane's registers and no limit on an item's columns.
template <int MODE, int KL, int EGROUPS, bool BATCH>
__device__ __forceinline__ bool epilogue_single(TcSmem& sm, const CUtensorMap* pA0, const CUtensorMap* pA1,
                                                const CUtensorMap* pB0, const CUtensorMap* pB1,
                                                const CUtensorMap* bmaps, const TcArgs& A, uint32_t tmem,
                                                int row_blocks, int64_t nrows, int items, int chunks) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int unit = int(blockIdx.x), units = int(gridDim.x);
  // Warp w may read TMEM lanes 32 (w % 4) .. + 31 (its rows); the groups split
  // the tile's columns, and each keeps its own list per row (EGROUPS lists per chunk).
  const int q = warp & 3;
  const int eg = (warp - 2) >> 2;
  const int r = q * 32 + lane;
  const uint32_t tlane = tmem + (uint32_t(q * 32) << 16);
  uint32_t tcount = 0;
  bool ok = true;
  // This row's best KL columns of the current chunk: scores ls (descending)
  // and columns li, in registers.  Columns arrive in increasing order, so a
  // new column beats a slot only with a strictly larger score: an equal
  // score keeps the earlier, lower column in front (score desc, column asc).
  float ls[KL];
  int li[KL];
  ItemRing rg;
  for (int item = take_item<false>(sm, A, true, -1, unit, units, rg, lane, ok); item < items && ok;
       item = take_item<false>(sm, A, true, item, unit, units, rg, lane, ok)) {
    TcItem it;
    get_item<BATCH>(A, pA0, pA1, pB0, pB1, bmaps, row_blocks, nrows, item, it, chunks);
    const int chunk = it.chunk;
    const int64_t arow = int64_t(it.rb) * TBM + r;   // row of the A operand
    const bool live = arow < it.nrows;
    const int64_t grow = gathered(MODE) ? (live ? int64_t(A.rows[arow]) : -1) : it.row0 + arow;  // vertex
#pragma unroll
    for (int j = 0; j < KL; ++j) {
      ls[j] = -FLT_MAX;
      li[j] = kInvalidIdx;
    }
    // Admission: beat the last slot and reach the row's floor (s >= floor,
    // i.e. s > the float below it).  The floor is the best K-th score any
    // chunk of this row has published: chunks publish their running K-th
    // after every tile, and an item re-reads the floor before every tile,
    // so chunks of a row that run at the same time raise each other's bar.
    // A partial list's K-th best is at most the row's final K-th best, so a
    // column below the floor can never be among the row's K best.
    int seen = live ? __ldcg(it.row_floor + arow) : INT_MAX;  // floor key in use (also: last published)
    float floor_below = live ? nextafterf(key_score(seen), -INFINITY) : INFINITY;
    const float rinv = (MODE == MODE_FP8 && live) ? it.inv_scale[grow] : 1.0f;
    for (int ct = it.t0; ct < it.t1; ++ct) {
      const int fk = (live && ct > it.t0) ? __ldcg(it.row_floor + arow) : seen;
      const uint32_t ab = tcount & 1u, tph = (tcount >> 1) & 1u;
      if (!wait_tile(sm, ab, tph)) {
        ok = false;
        break;
      }
      tc::tc_fence_after();
      if (fk > seen) {
        seen = fk;
        floor_below = nextafterf(key_score(fk), -INFINITY);
      }
#pragma unroll 1
      for (int cb = eg * (TBN / 32 / EGROUPS); cb < (eg + 1) * (TBN / 32 / EGROUPS); ++cb) {
        uint32_t v[32];
        tc::tmem_ld32(tlane + ab * TBN + cb * 32, v);
        tc::tmem_wait_ld(v);
        // Admission test of the 32 columns, then a warp-convergent drain:
        // every round each lane inserts at most one admitted column with a
        // branch-free pass over its list, so the warp pays per round.
        const int64_t lbase = int64_t(ct) * TBN + cb * 32;  // B column
        const int64_t cbase = it.col0 + lbase;               // its vertex
        const int nvalid = int(tmin<int64_t>(it.n - lbase, 32));
        const int64_t dself = grow - cbase;
        const int jself = (dself >= 0 && dself < 32) ? int(dself) : -1;
        const float thr = fmaxf(ls[KL - 1], floor_below);
        uint32_t mask = 0;
#pragma unroll
        for (int j = 0; j < 32; ++j) {
          float sc = __uint_as_float(v[j]);
          if (MODE == MODE_FP8) sc = sc * rinv * __ldg(it.inv_scale + (j < nvalid ? cbase + j : 0));
          if (j == jself) sc = 1.0f;
          if (j >= nvalid) sc = -INFINITY;
          sm.batch[eg][j][r] = sc;
          mask |= (sc > thr) ? (1u << j) : 0u;
        }
        int rounds = __popc(mask);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) rounds = max(rounds, __shfl_xor_sync(kFull, rounds, o));
#pragma unroll 1
        for (int rd = 0; rd < rounds; ++rd) {
          float cs = -INFINITY;
          int ci = kInvalidIdx;
          if (mask) {
            const int j = __ffs(mask) - 1;
            mask &= mask - 1u;
            cs = sm.batch[eg][j][r];
            ci = int(cbase + j);
          }
          list_insert<KL>(ls, li, cs, ci);
        }
      }
      tc::tc_fence_before();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&sm.tempty[ab]);
      ++tcount;
      // Publish this chunk's running K-th best when it raises the row's floor.
      if (live && ct + 1 < it.t1) {
        float kth = FLT_MAX;
#pragma unroll
        for (int j = 0; j < KL; ++j)
          if (j < it.K) kth = fminf(kth, ls[j]);
        if (kth != -FLT_MAX) {
          const int key = score_key(kth);
          if (key > seen) {
            atomicMax(it.row_floor + arow, key);
            seen = key;
            floor_below = nextafterf(kth, -INFINITY);
          }
        }
      }
    }
    if (!ok) break;
    if (live) {
      const size_t o = ((size_t(arow) * it.chunks + chunk) * EGROUPS + eg) * it.K;
      // The K-th best as a running minimum over the first K slots (the list
      // is never indexed dynamically, so it stays in registers).
      float kth = FLT_MAX;
#pragma unroll
      for (int j = 0; j < KL; ++j) {
        if (j < it.K) {
          it.part_s[o + j] = ls[j];
          it.part_i[o + j] = li[j];
          kth = fminf(kth, ls[j]);
        }
      }
      // This chunk's K-th best becomes a floor for the row's later chunks.
      if (kth != -FLT_MAX) atomicMax(it.row_floor + arow, score_key(kth));
      // Lists of chunks this launch does not use are empty (first entry invalid).
      if (gathered(MODE) && chunk == 0)
        for (int c = chunks; c < it.chunks; ++c) {
          const size_t oe = ((size_t(arow) * it.chunks + c) * EGROUPS + eg) * it.K;
          it.part_s[oe] = -FLT_MAX;
          it.part_i[oe] = kInvalidIdx;
        }
    }
  }
  return ok;
}

// PAIR: the CTAs of a cluster of two compute 256-row tiles together with
// tcgen05 cta_group::2.  The even CTA ("leader") issues the MMAs; each CTA
// loads its own 128 rows of A and its 128 of the tile's 256 B rows, counted
// on the leader's `full` barrier; the MMA's commits reach both CTAs'
// `empty` / `tfull` barriers; both CTAs' epilogue warps release an
// accumulator on the leader's `tempty`.
template <int MODE, int KL, int EGROUPS, bool BATCH, bool PAIR, int KIND = KIND_LISTS>
__device__ __forceinline__ void tc_body(const CUtensorMap* pA0, const CUtensorMap* pA1, const CUtensorMap* pB0,
                                        const CUtensorMap* pB1, const CUtensorMap* bmaps, const TcArgs& A) {
  using Smem = SmemOf<PAIR, KL, EGROUPS, KIND>;
  constexpr int STG = Smem::kStages;
  constexpr int ROWS = PAIR ? 2 * TBM : TBM;  // A rows of one work item
  Smem& sm = smem_block<Smem>();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  volatile int* abort = &sm.abort;
  constexpr int SEGS = MODE == MODE_SPLIT ? 3 : 1;
  const uint32_t rank = PAIR ? tc::cluster_rank() : 0u;
  const bool leader = rank == 0;
  const int unit = PAIR ? int(blockIdx.x >> 1) : int(blockIdx.x);   // cluster (pair) or CTA
  const int units = PAIR ? int(gridDim.x >> 1) : int(gridDim.x);
  const int64_t nrows = gathered(MODE) ? int64_t(*A.count) : A.a_rows;
  const int row_blocks = gathered(MODE) ? int((nrows + ROWS - 1) / ROWS) : A.row_blocks;
  const int chunks = gathered(MODE) ? pick_chunks(row_blocks, A.chunks, A.col_tiles, units) : A.chunks;
  const int items = BATCH ? A.items_total : row_blocks * chunks;

  if (threadIdx.x == 0) {
    for (int st = 0; st < STG; ++st) {
      tc::mbar_init(&sm.full[st], 1);
      tc::mbar_init(&sm.empty[st], 1);
    }
    for (int b = 0; b < 2; ++b) {
      tc::mbar_init(&sm.tfull[b], 1);
      tc::mbar_init(&sm.tempty[b], 4 * EGROUPS * (PAIR ? 2 : 1));
    }
    tc::mbar_init(&sm.done, 1);
    for (int q = 0; q < IQ; ++q) {
      tc::mbar_init(&sm.ifull[q], 1);
      // consumers: the MMA thread and the epilogue warps; for a pair also the
      // odd CTA's TMA thread and epilogue warps (they release on the even CTA's)
      tc::mbar_init(&sm.iempty[q], PAIR ? 2 + 8 * EGROUPS : 1 + 4 * EGROUPS);
    }
    sm.abort = 0;
    tc::fence_barrier_init();
    if (!BATCH) {
      tc::tma_prefetch_desc(pA0);
      tc::tma_prefetch_desc(pB0);
      if (MODE == MODE_SPLIT) {
        tc::tma_prefetch_desc(pA1);
        tc::tma_prefetch_desc(pB1);
      }
    }
  }
  // The pair's allocation is collective over both SMs' tensor memory: neither
  // CTA asks for it before the other one runs.  (When other streams' kernels keep
  // the SMs busy the two CTAs can start far apart, and an allocation issued before
  // the peer had started left the peer's own waiting for ever.)
  if (PAIR) {
    __syncwarp();
    tc::cluster_sync();
  }
  if (warp == 1) {
    if (PAIR) {
      tc::tmem_alloc_pair(&sm.tmem_base, 512);
      tc::tmem_relinquish_pair();
    } else {
      tc::tmem_alloc(&sm.tmem_base, 512);
      tc::tmem_relinquish();
    }
  }
  tc::tc_fence_before();
  __syncthreads();
  if (PAIR) tc::cluster_sync();  // the peer's barriers are initialised before any cross-CTA signal
  tc::tc_fence_after();
  const uint32_t tmem = sm.tmem_base;

  if (warp == 0) {
    if (lane == 0) {
      // ---------------- TMA producer ----------------
      uint32_t stage = 0, phase = 0;
      uint32_t armed = 0;  // bit s: slot s holds a load that may still be in flight
      uint32_t armed_phase = 0;
      bool ok = true;
      ItemRing rg;
      const bool publisher = !PAIR || leader;
      for (int item = A.stall ? INT_MAX : next_item<PAIR>(sm, A, publisher, leader, -1, unit, units, rg, abort, ok);
           item < items && ok;
           item = next_item<PAIR>(sm, A, publisher, leader, item, unit, units, rg, abort, ok)) {
        TcItem it;
        get_item<BATCH>(A, pA0, pA1, pB0, pB1, bmaps, row_blocks, nrows, item, it, chunks);
        const int rb = it.rb;
        const int kb_total = it.kblocks * SEGS;
        for (int ct = it.t0; ct < it.t1 && ok; ++ct) {
          for (int kt = 0; kt < kb_total; ++kt) {
            if (!tc::mbar_wait(&sm.empty[stage], phase ^ 1u, abort, WAIT_LIMIT)) {
              ok = false;
              break;
            }
            const int seg = kt / it.kblocks, kb = kt - seg * it.kblocks;
            const CUtensorMap* ma = seg == 1 ? it.ma1 : it.ma0;
            const CUtensorMap* mb = seg == 2 ? it.mb1 : it.mb0;
            const int kx = kb * (MODE == MODE_FP8 ? 128 : 64);
            if (PAIR) {
              // this CTA's A rows and its half of the tile's B rows; bytes counted on the leader
              const uint32_t bar = tc::map_to_rank(&sm.full[stage], 0);
              if (leader) tc::mbar_arrive_expect_tx(&sm.full[stage], 2 * (A_BYTES + B_BYTES / 2));
              tc::tma_load_2d_pair(sm.a[stage], ma, bar, kx, rb * ROWS + int(rank) * TBM);
              tc::tma_load_2d_pair(sm.b[stage], mb, bar, kx, ct * TBN + int(rank) * (TBN / 2));
            } else {
              tc::mbar_arrive_expect_tx(&sm.full[stage], A_BYTES + B_BYTES);
              tc::tma_load_2d(sm.a[stage], ma, &sm.full[stage], kx, rb * TBM);
              tc::tma_load_2d(sm.b[stage], mb, &sm.full[stage], kx, ct * TBN);
              tc::tma_load_2d(sm.b[stage] + B_BYTES / 2, mb, &sm.full[stage], kx, ct * TBN + TBN / 2);
            }
            armed |= 1u << stage;
            armed_phase = (armed_phase & ~(1u << stage)) | (phase << stage);
            if (++stage == STG) {
              stage = 0;
              phase ^= 1u;
            }
          }
        }
      }
      // Wait until the MMAs have released every slot: the commits that do so
      // arrive on this CTA's `empty` barriers from the even CTA's tensor core,
      // which nothing else orders before the CTA's end.  Without it a late
      // arrival could land in the shared memory of the CTA that another
      // stream's kernel starts on this SM.
      for (int st = 0; st < STG && ok; ++st)
        if (armed & (1u << st)) ok = tc::mbar_wait(&sm.empty[st], (armed_phase >> st) & 1u, abort, WAIT_LIMIT);
      if (!ok) {
        *abort = 1;
        report_timeout<BATCH>(A);
        // Let loads already issued land before the CTA exits.
        if (PAIR && !leader) {
          if (armed) drain_delay();
        } else {
          for (int st = 0; st < STG; ++st)
            if (armed & (1u << st)) tc::mbar_wait(&sm.full[st], (armed_phase >> st) & 1u, abort, WAIT_LIMIT);
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0 && leader) {
      // ---------------- MMA issuer (the leader of a pair) ----------------
      constexpr uint32_t idesc = tc::instr_desc(MODE == MODE_FP8 ? 0u : 1u, ROWS, TBN);
      constexpr uint16_t both = 3;
      uint32_t stage = 0, phase = 0, tcount = 0;
      bool ok = true;
      ItemRing rg;
      for (int item = next_item<PAIR>(sm, A, false, leader, -1, unit, units, rg, abort, ok); item < items && ok;
           item = next_item<PAIR>(sm, A, false, leader, item, unit, units, rg, abort, ok)) {
        TcItem it;
        get_item<BATCH>(A, pA0, pA1, pB0, pB1, bmaps, row_blocks, nrows, item, it, chunks);
        const int kb_total = it.kblocks * SEGS;
        for (int ct = it.t0; ct < it.t1 && ok; ++ct) {
          const uint32_t ab = tcount & 1u, tph = (tcount >> 1) & 1u;
          if (!tc::mbar_wait(&sm.tempty[ab], tph ^ 1u, abort, WAIT_LIMIT)) {
            ok = false;
            break;
          }
          tc::tc_fence_after();
          const uint32_t d = tmem + ab * TBN;
          for (int kt = 0; kt < kb_total; ++kt) {
            if (!tc::mbar_wait(&sm.full[stage], phase, abort, WAIT_LIMIT)) {
              ok = false;
              break;
            }
            tc::tc_fence_after();
            const uint64_t da = tc::desc_sw128(sm.a[stage]);
            const uint64_t db = tc::desc_sw128(sm.b[stage]);
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
              // 32 bytes of K per instruction: advance the start address by 2 (16-byte units).
              const uint32_t acc = (kt | kk) != 0;
              if (PAIR) {
                if (MODE == MODE_FP8) tc::mma_fp8_pair(d, da + 2u * kk, db + 2u * kk, idesc, acc);
                else tc::mma_bf16_pair(d, da + 2u * kk, db + 2u * kk, idesc, acc);
              } else {
                if (MODE == MODE_FP8) tc::mma_fp8(d, da + 2u * kk, db + 2u * kk, idesc, acc);
                else tc::mma_bf16(d, da + 2u * kk, db + 2u * kk, idesc, acc);
              }
            }
            if (PAIR) tc::mma_commit_pair(&sm.empty[stage], both);
            else tc::mma_commit(&sm.empty[stage]);
            if (++stage == STG) {
              stage = 0;
              phase ^= 1u;
            }
          }
          if (!ok) break;
          if (PAIR) tc::mma_commit_pair(&sm.tfull[ab], both);
          else tc::mma_commit(&sm.tfull[ab]);
          ++tcount;
        }
      }
      if (!ok) {
        *abort = 1;
        report_timeout<BATCH>(A);
      }
      // Every MMA issued by this thread has completed once `done` fires.
      if (PAIR) tc::mma_commit_pair(&sm.done, 1);
      else tc::mma_commit(&sm.done);
      tc::mbar_wait(&sm.done, 0, abort, WAIT_LIMIT);
    }
  } else {
    // ---------------- epilogue: warps 2 .. 2 + 4 EGROUPS ----------------
    bool ok;
    if constexpr (KIND == KIND_SAMPLE)  // KL: the largest floor rank
      ok = epilogue_sample<MODE, KL, BATCH>(sm, pA0, pB0, bmaps, A, tmem, rank, row_blocks, nrows, items, chunks);
    else if constexpr (KIND == KIND_APPEND)
      ok = epilogue_append<MODE, BATCH>(sm, pA0, pB0, bmaps, A, tmem, rank, row_blocks, nrows, items, chunks);
    else if constexpr (PAIR)
      ok = epilogue_pair<MODE, KL, EGROUPS, BATCH>(sm, pA0, pA1, pB0, pB1, bmaps, A, tmem, rank, row_blocks, nrows,
                                                   items, chunks);
    else
      ok = epilogue_single<MODE, KL, EGROUPS, BATCH>(sm, pA0, pA1, pB0, pB1, bmaps, A, tmem, row_blocks, nrows, items,
                                                     chunks);
    if (!ok) {
      *abort = 1;
      report_timeout<BATCH>(A);
    }
  }

  __syncwarp();  // the role branches above ran single lanes
  tc::tc_fence_before();
  __syncthreads();
  if (PAIR) tc::cluster_sync();  // neither CTA frees while the pair's MMAs or signals may touch it
  tc::tc_fence_after();
  if (warp == 1) {
    if (PAIR) tc::tmem_dealloc_pair(tmem, 512);
    else tc::tmem_dealloc(tmem, 512);
  }
  if (PAIR) {
    __syncwarp();
    tc::cluster_sync();  // neither CTA leaves before both have freed
  }
}

template <int MODE, int KL, int EGROUPS>
__global__ void __launch_bounds__(threads_of(EGROUPS), 1)
k1_tc_topk(const __grid_constant__ CUtensorMap mA0, const __grid_constant__ CUtensorMap mA1,
           const __grid_constant__ CUtensorMap mB0, const __grid_constant__ CUtensorMap mB1, TcArgs A) {
  tc_body<MODE, KL, EGROUPS, false, false>(&mA0, &mA1, &mB0, &mB1, nullptr, A);
}

// CTA pairs (launched in clusters of two): 256-row items, one cta_group::2
// MMA per k-step for both SMs.
template <int MODE, int KL, int EGROUPS>
__global__ void __launch_bounds__(threads_of(EGROUPS), 1)
k1_tc2_topk(const __grid_constant__ CUtensorMap mA0, const __grid_constant__ CUtensorMap mA1,
            const __grid_constant__ CUtensorMap mB0, const __grid_constant__ CUtensorMap mB1, TcArgs A) {
  tc_body<MODE, KL, EGROUPS, false, true>(&mA0, &mA1, &mB0, &mB1, nullptr, A);
}

// The sampling pass (all rows against the sampled columns; KR: the largest
// floor rank) and the append pass, on one instance or on many.
template <int MODE, int KR>
__global__ void __launch_bounds__(threads_of(1), 1)
k1_tc2_sample(const __grid_constant__ CUtensorMap mA0, const __grid_constant__ CUtensorMap mB0, TcArgs A) {
  tc_body<MODE, KR, 1, false, true, KIND_SAMPLE>(&mA0, &mA0, &mB0, &mB0, nullptr, A);
}
template <int MODE, int KR>
__global__ void __launch_bounds__(threads_of(1), 1)
k1_tc2_sample_batch(const __grid_constant__ TcMaps2 maps, TcArgs A) {
  tc_body<MODE, KR, 1, true, true, KIND_SAMPLE>(nullptr, nullptr, nullptr, nullptr, maps.m, A);
}
template <int MODE>
__global__ void __launch_bounds__(threads_of(AEG), 1)
k1_tc2_append(const __grid_constant__ CUtensorMap mA0, TcArgs A) {
  tc_body<MODE, 0, AEG, false, true, KIND_APPEND>(&mA0, &mA0, &mA0, &mA0, nullptr, A);
}
template <int MODE>
__global__ void __launch_bounds__(threads_of(AEG), 1)
k1_tc2_append_batch(const __grid_constant__ TcMaps maps, TcArgs A) {
  tc_body<MODE, 0, AEG, true, true, KIND_APPEND>(nullptr, nullptr, nullptr, nullptr, maps.m, A);
}

// Copies the sampled rows of the low-precision array (and their FP8 scales):
// one row from each of m equal strata of the n rows, at a hashed place in its
// stratum, so that no ordering of the rows (by identity, by camera) lines up
// with the sample.
__global__ void k_sample_rows(const uint4* __restrict__ x, const float* __restrict__ scale, int64_t n, int m,
                              int vecs, uint4* __restrict__ dst, float* __restrict__ dscale) {
  const int f = int((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (f >= m) return;
  const int64_t a = n * f / m, b = n * (f + 1) / m;
  const uint32_t h = (uint32_t(f) * 2654435761u) >> 8;
  const int64_t src = a + int64_t(h) % (b - a);
  for (int k = lane; k < vecs; k += kWarp) dst[int64_t(f) * vecs + k] = x[src * vecs + k];
  if (scale && lane == 0) dscale[f] = scale[src];
}

// Many instances in one persistent launch: the items of all instances form one
// list that the CTAs walk; each item carries its instance's parameters.
template <int MODE, int KL, int EGROUPS>
__global__ void __launch_bounds__(threads_of(EGROUPS), 1)
k1_tc_topk_batch(const __grid_constant__ TcMaps maps, TcArgs A) {
  tc_body<MODE, KL, EGROUPS, true, false>(nullptr, nullptr, nullptr, nullptr, maps.m, A);
}

// Test hook: RERANK_TEST_TC_STALL set in the environment makes the kernels'
// TMA warp issue nothing, so the MMA and epilogue waits run out and the call
// returns ETIMEOUT (no copy or MMA is ever in flight on that path).
int stall_hook() { return std::getenv("RERANK_TEST_TC_STALL") ? 1 : 0; }

using EncodeFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                              const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                              CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeFn get_encode() {
  static EncodeFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeFn>(p);
  }
  return fn;
}

// Row-major rows x dp matrix, boxes of 128 rows x 128 bytes, 128-byte swizzle.
bool make_map(CUtensorMap* map, const void* base, int64_t rows, int dp, bool fp8) {
  EncodeFn enc = get_encode();
  if (!enc) return false;
  const cuuint64_t dims[2] = {cuuint64_t(dp), cuuint64_t(rows)};
  const cuuint64_t strides[1] = {cuuint64_t(dp) * (fp8 ? 1 : 2)};
  const cuuint32_t box[2] = {fp8 ? 128u : 64u, 128u};
  const cuuint32_t estr[2] = {1, 1};
  return enc(map, fp8 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base),
             dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
             CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int MODE, int KL, int EG>
void launch_kl(const CUtensorMap& a0, const CUtensorMap& a1, const CUtensorMap& b0, const CUtensorMap& b1,
               const TcArgs& A, int grid, cudaStream_t s) {
  const size_t smem = sizeof(TcSmem) + 1024;
  cudaFuncSetAttribute(k1_tc_topk<MODE, KL, EG>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
  k1_tc_topk<MODE, KL, EG><<<grid, threads_of(EG), smem, s>>>(a0, a1, b0, b1, A);
}

// Pairs of one kernel that can be resident at once, per device (-1: not asked yet).
struct PairUnits {
  static constexpr int kDevices = 64;
  std::atomic<int> n[kDevices];
  PairUnits() {
    for (auto& v : n) v.store(-1, std::memory_order_relaxed);
  }
};

// Launches `kernel` on pairs (clusters of two CTAs, one CTA per SM): as many as
// there are items, at most those that can be resident at once.  Their number and
// the kernel's shared-memory limit belong to a device: asked and set by the first
// launch on each (callers and serving workers may be first at the same time; both
// then store the same).  False when no pair can be resident or the launch fails.
template <class Kernel, class... Args>
bool launch_pairs(Kernel kernel, PairUnits& units, size_t smem, int threads, int items, int sm_count, cudaStream_t s,
                  const Args&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(unsigned(sm_count & ~1));
  cfg.blockDim = dim3(unsigned(threads));
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 2;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  int n = dev < PairUnits::kDevices ? units.n[dev].load() : -1;
  if (n < 0) {
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
    if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
      cudaGetLastError();
      n = 0;
    }
    if (dev < PairUnits::kDevices) units.n[dev].store(n);
  }
  if (n < 1) return false;
  cfg.gridDim = dim3(unsigned(2 * (items < n ? items : n)));
  cfg.stream = s;
  return cudaLaunchKernelEx(&cfg, kernel, args...) == cudaSuccess;
}

template <int MODE, int KL, int EG>
bool launch_kl_pair(const CUtensorMap& a0, const CUtensorMap& a1, const CUtensorMap& b0, const CUtensorMap& b1,
                    const TcArgs& A, int items, int sm_count, cudaStream_t s) {
  static PairUnits units;
  return launch_pairs(k1_tc2_topk<MODE, KL, EG>, units, sizeof(TcSmemPair<KL, EG>) + 1024, threads_of(EG), items,
                      sm_count, s, a0, a1, b0, b1, A);
}

template <int MODE, int KR>
bool launch_sample(const CUtensorMap& a, const CUtensorMap& b, const TcArgs& A, int items, int sm_count,
                   cudaStream_t s) {
  static PairUnits units;
  return launch_pairs(k1_tc2_sample<MODE, KR>, units, sizeof(TcSmemRing) + 1024, threads_of(1), items, sm_count, s, a,
                      b, A);
}
template <int MODE, int KR>
bool launch_sample_batch(const TcMaps2& maps, const TcArgs& A, int items, int sm_count, cudaStream_t s) {
  static PairUnits units;
  return launch_pairs(k1_tc2_sample_batch<MODE, KR>, units, sizeof(TcSmemRing) + 1024, threads_of(1), items, sm_count,
                      s, maps, A);
}
template <int MODE>
bool launch_append(const CUtensorMap& a, const TcArgs& A, int items, int sm_count, cudaStream_t s) {
  static PairUnits units;
  return launch_pairs(k1_tc2_append<MODE>, units, sizeof(TcSmemRing) + 1024, threads_of(AEG), items, sm_count, s, a,
                      A);
}
template <int MODE>
bool launch_append_batch(const TcMaps& maps, const TcArgs& A, int items, int sm_count, cudaStream_t s) {
  static PairUnits units;
  return launch_pairs(k1_tc2_append_batch<MODE>, units, sizeof(TcSmemRing) + 1024, threads_of(AEG), items, sm_count,
                      s, maps, A);
}

// items: work items of the launch, or INT_MAX when only the device knows
// them (gathered rows): then every resident pair is launched.
template <int MODE>
bool launch_mode_pair(const CUtensorMap& a0, const CUtensorMap& a1, const CUtensorMap& b0, const CUtensorMap& b1,
                      const TcArgs& A, int eg, int items, int sm_count, cudaStream_t s) {
  if (A.K <= 48)
    return eg == 2 ? launch_kl_pair<MODE, 48, 2>(a0, a1, b0, b1, A, items, sm_count, s)
                   : launch_kl_pair<MODE, 48, 1>(a0, a1, b0, b1, A, items, sm_count, s);
  return eg == 2 ? launch_kl_pair<MODE, KLIST, 2>(a0, a1, b0, b1, A, items, sm_count, s)
                 : launch_kl_pair<MODE, KLIST, 1>(a0, a1, b0, b1, A, items, sm_count, s);
}

// The per-row list lives in registers, so its length is a compile-time choice.
template <int MODE>
void launch_mode(const CUtensorMap& a0, const CUtensorMap& a1, const CUtensorMap& b0, const CUtensorMap& b1,
                 const TcArgs& A, int eg, int grid, cudaStream_t s) {
  if (A.K <= 48) {
    if (eg == 2)
      launch_kl<MODE, 48, 2>(a0, a1, b0, b1, A, grid, s);
    else
      launch_kl<MODE, 48, 1>(a0, a1, b0, b1, A, grid, s);
  } else {
    if (eg == 2)
      launch_kl<MODE, KLIST, 2>(a0, a1, b0, b1, A, grid, s);
    else
      launch_kl<MODE, KLIST, 1>(a0, a1, b0, b1, A, grid, s);
  }
}

__global__ void k_gather_rows(const int32_t* __restrict__ rows, const int32_t* __restrict__ count,
                              const uint4* __restrict__ hi, const uint4* __restrict__ lo, uint4* __restrict__ dhi,
                              uint4* __restrict__ dlo, int64_t n, int vecs) {
  const int64_t f = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (f >= n || f >= *count) return;
  const int64_t src = rows[f];
  for (int k = lane; k < vecs; k += kWarp) {
    dhi[f * vecs + k] = hi[src * vecs + k];
    dlo[f * vecs + k] = lo[src * vecs + k];
  }
}

// The K best of a row's admitted columns (the segments of the append pass),
// sorted by (score desc, vertex asc) into one list of K places; unused places
// are (-FLT_MAX, invalid).  A warp per row, two passes over the segments (the
// second hits L1): the first counts the entries in 384 log-spaced buckets (64
// per octave from 2^-6 up; lower scores share bucket 0), the second scatters
// the entries of the buckets that hold the K best to their bucket's range, and
// an entry's place is its bucket's start plus the better entries inside it.
// About 1,900 issue slots for 350 entries, 59 us at n = 23,100 (a bisection
// on the keys and a quadratic ranking took 3,400 and 162 us).  A row whose last bucket is too crowded for the
// sorted range picks its K best one by one.  A row with a segment that ran
// over gets an empty list (the recheck takes it).
constexpr int SEL_WARPS = 8;
constexpr int SEL_BINS = 384;
constexpr int kMaxSegs = 128;  // segments of a row
constexpr int SEL_OUT = 128;  // entries of the buckets that hold the K best
struct SelWarp {
  int bin[SEL_BINS];  // counts, then places
  int key[SEL_OUT];
  int col[SEL_OUT];
};

__global__ void __launch_bounds__(SEL_WARPS * kWarp)
k_select(const uint2* __restrict__ cand, const int32_t* __restrict__ seg_cnt, int64_t n, int segs, int cap, int K,
         float* __restrict__ part_s, int32_t* __restrict__ part_i, const long long* __restrict__ status) {
  __shared__ SelWarp sel[SEL_WARPS];
  const int lane = threadIdx.x & 31;
  SelWarp& w = sel[threadIdx.x >> 5];
  const int64_t r = int64_t(blockIdx.x) * SEL_WARPS + (threadIdx.x >> 5);
  if (r >= n) return;
  const uint2* row = cand + r * segs * size_t(cap);
  // Segment counts: lane l holds segments l, l + 32, ...
  const int32_t* sc = seg_cnt + r * segs;
  int sn[kMaxSegs / kWarp], sum0 = 0;
  bool over = false;
#pragma unroll
  for (int k = 0; k < kMaxSegs / kWarp; ++k) {
    sn[k] = lane + k * kWarp < segs ? sc[lane + k * kWarp] : 0;
    over = over || sn[k] > cap;
  }
  // (after a similarity stage that timed out the counts may be unwritten)
  if (__any_sync(kFull, over) || (status[kStErr] & kErrTimeout)) segs = 0;
#pragma unroll
  for (int k = 0; k < kMaxSegs / kWarp; ++k) sum0 += k * kWarp < segs ? sn[k] : 0;
  const int total = __reduce_add_sync(kFull, sum0);
  auto each = [&](auto f) {  // f(key, column) over all entries, a lane each
    for (int s0 = 0; s0 < segs; s0 += 4) {  // segs is a multiple of AEG = 4
      uint2 x[4];
      int cnt[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int sg = s0 + u;
        int v = sn[0];
#pragma unroll
        for (int k = 1; k < kMaxSegs / kWarp; ++k) v = sg >= k * kWarp ? sn[k] : v;
        cnt[u] = __shfl_sync(kFull, v, sg & 31);
        if (lane < cnt[u]) x[u] = __ldg(row + sg * cap + lane);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (lane < cnt[u]) f(score_key(__uint_as_float(x[u].x)), int(x[u].y));
        for (int j = lane + kWarp; j < cnt[u]; j += kWarp) {
          const uint2 y = __ldg(row + (s0 + u) * cap + j);
          f(score_key(__uint_as_float(y.x)), int(y.y));
        }
      }
    }
  };
  constexpr int kLow = 121 << 23;  // the key of 2^-6
  auto bucket = [](int key) { return min(max(key - kLow, 0) >> 17, SEL_BINS - 1); };
  float* ps = part_s + r * K;
  int32_t* pi = part_i + r * K;
  constexpr int PL = SEL_BINS / kWarp;  // buckets per lane; lane 0 holds the highest
  int* const mine = w.bin + SEL_BINS - PL * (lane + 1);
#pragma unroll
  for (int k = 0; k < PL; ++k) w.bin[lane + k * kWarp] = 0;
  __syncwarp();
  each([&](int k, int) { atomicAdd(&w.bin[bucket(k)], 1); });
  __syncwarp();
  // First places, from the highest bucket down, and the bucket that holds place K - 1.
  int c[PL], sum = 0;
#pragma unroll
  for (int k = 0; k < PL; ++k) {
    c[k] = mine[PL - 1 - k];
    sum += c[k];
  }
  int incl = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl += y;
  }
  int at = incl - sum;
  const int want = min(K, total);
  int last = -1, nsel = 0;  // the bucket and the entries up to its end, on the lane that holds it
#pragma unroll
  for (int k = 0; k < PL; ++k) {
    mine[PL - 1 - k] = at;
    if (at < want && want <= at + c[k]) {
      last = SEL_BINS - PL * lane - 1 - k;
      nsel = at + c[k];
    }
    at += c[k];
  }
  last = __reduce_max_sync(kFull, last);
  nsel = __reduce_max_sync(kFull, nsel);
  __syncwarp();
  if (nsel <= SEL_OUT) {
    each([&](int k, int v) {
      const int bk = bucket(k);
      if (bk >= last) {
        const int p = atomicAdd(&w.bin[bk], 1);
        w.key[p] = k;
        w.col[p] = v;
      }
    });
    __syncwarp();  // bin[b] is now the end of bucket b, and the start of bucket b - 1
    for (int p = lane; p < nsel; p += kWarp) {
      const int k = w.key[p], v = w.col[p], bk = bucket(k);
      const int b1 = w.bin[bk];
      int rank = bk == SEL_BINS - 1 ? 0 : w.bin[bk + 1];
      for (int j = rank; j < b1; ++j) rank += (w.key[j] > k || (w.key[j] == k && w.col[j] < v)) ? 1 : 0;
      if (rank < K) {
        ps[rank] = key_score(k);
        pi[rank] = v;
      }
    }
  } else {
    // one by one: the best entry after the last one taken
    int lk = INT_MAX, lv = -1;
    for (int m = 0; m < want; ++m) {
      int bk = INT_MIN, bv = INT_MAX;
      each([&](int k, int v) {
        if ((k < lk || (k == lk && v > lv)) && (k > bk || (k == bk && v < bv))) {
          bk = k;
          bv = v;
        }
      });
      lk = __reduce_max_sync(kFull, bk);
      lv = __reduce_min_sync(kFull, bk == lk ? bv : INT_MAX);
      if (lane == 0) {
        ps[m] = key_score(lk);
        pi[m] = lv;
      }
    }
  }
  for (int e = want + lane; e < K; e += kWarp) {
    ps[e] = -FLT_MAX;
    pi[e] = kInvalidIdx;
  }
}

}  // namespace

size_t tc_smem_bytes() { return sizeof(TcSmem) + 1024; }
template <int KL, int EG>
constexpr bool pair_fits() {
  return sizeof(TcSmemPair<KL, EG>) + 1024 <= 227 * 1024;
}
static_assert(kMaxSegs % kWarp == 0 && kMaxSegs % AEG == 0, "k_select walks the segments four at a time");
static_assert(pair_fits<48, 1>() && pair_fits<48, 2>() && pair_fits<KLIST, 1>() && pair_fits<KLIST, 2>(),
              "shared memory of the paired tensor-core kernels");
// Whether the main similarity pass runs on CTA pairs (cta_group::2).  Both
// kernels give identical lists; RERANK_TC_PAIRS=0 selects the single-CTA one.
bool tc_pairs() {
  static const int on = [] {
    const char* e = std::getenv("RERANK_TC_PAIRS");
    return (e && e[0] == '0') ? 0 : 1;
  }();
  return on != 0;
}
int tc_item_rows() { return tc_pairs() ? 2 * TBM : TBM; }
int tc_max_item_tiles() { return kMaxItemTiles; }
// Pairs hold an item's columns as 16-bit offsets (at most kMaxItemTiles tiles);
// longer items, and a device with one SM, take the single-CTA kernels.
static bool use_pairs(int col_tiles, int chunks, int sm_count) {
  return tc_pairs() && sm_count >= 2 && (col_tiles + chunks - 1) / chunks <= kMaxItemTiles;
}
// Whether the main pass takes its items dynamically (see next_item);
// RERANK_TC_DYNAMIC=0 selects the static order (identical lists).
bool tc_dynamic() {
  static const int on = [] {
    const char* e = std::getenv("RERANK_TC_DYNAMIC");
    return (e && e[0] == '0') ? 0 : 1;
  }();
  return on != 0;
}
int tc_lists_per_chunk(int dp, int segs) { return dp * segs <= 1024 ? 2 : 1; }
static_assert(sizeof(TcSmem) + 1024 <= 227 * 1024, "shared memory of the tensor-core kernel");
int tc_kmax() { return KLIST; }
int tc_tile_rows() { return TBM; }
int tc_tile_cols() { return TBN; }

// Plan of the append pass for n rows of np padded ones, lists of K: column
// chunks (from `chunks`), segments and their capacity, and the columns sampled
// for the floors.
//
// A row's floor is the rank-th largest of its sampled scores, with the rank
// such that fewer than K columns reach the floor once in some thousand rows
// (the columns above the r-th largest of a random sample of m number fewer than
// K with the probability that a Poisson variable of mean K m / n is r or more);
// about rank * n / m columns do reach it, whatever the scores are.  The floor
// is an estimate: a row with fewer than K columns above it is certified against
// the floor itself by the refinement, or goes to the recheck.  Up to 1,024
// rows every column is kept and nothing is sampled.
static int sample_rank(int K, int sample, int64_t n) {
  const double lam = double(K) * sample / double(n);
  double term = std::exp(-lam), tail = 1.0 - term;
  int r = 1;
  while (r < 32 && tail > 1e-4) {
    term *= lam / r;
    tail -= term;
    ++r;
  }
  return r;
}
// Room for 3.5 times the expected columns of a segment (the number above a
// floor of rank 5 or more exceeds that for one row in some thousand), and
// for a whole cluster of neighbours stored side by side; at most `most`.
static int segment_cap(int64_t n, int K, int sample, int segs, int most) {
  const double mean = double(sample_rank(K, sample, n) + 1) * double(n) / sample / segs;
  int c = int(3.5 * mean + 5.0 * std::sqrt(mean)) + 64;
  c = (c + 31) / 32 * 32;
  c = c < 128 ? 128 : c;
  return most < c ? most : c;
}
// The same for a few rows against n columns (a serving request's queries): at
// most kRowsAppendChunks chunks, floors from one tile of sampled columns.
constexpr int kRowsAppendChunks = kMaxSegs / AEG;
int tc_rows_append_sample() { return TBN; }
int tc_rows_append_segs() { return kMaxSegs; }
int tc_rows_append_cap(int64_t n, int K, int chunks) {
  const int tiles = int((n + TBN - 1) / TBN);
  return segment_cap(n, K, TBN, chunks * AEG, (tiles + chunks - 1) / chunks * (TBN / AEG));
}
bool tc_append_ok(int64_t np, int sm_count) { return tc_pairs() && sm_count >= 2 && np % (2 * TBM) == 0; }
void tc_append_plan(int64_t n, int64_t np, int dp, int K, int chunks, int* segs, int* cap, int* sample) {
  const int tiles = int(np / TBN);
  chunks = chunks < 1 ? 1 : (chunks > 16 ? 16 : chunks);
  if (chunks > tiles) chunks = tiles;
  const int most = (tiles + chunks - 1) / chunks * (TBN / AEG);  // columns of a segment
  *segs = chunks * AEG;
  if (n <= 1024) {
    *sample = 0;
    *cap = most;
    return;
  }
  // Sampled columns: more of them admit fewer columns but cost their share of
  // the MMAs, which are hidden behind the scan only at small d.  The steps are
  // within 3 % of the best of 256 .. 4,096, within 5 % at d = 128 far from a step
  // (12,000 rows: 165 us with 512, 157 with 2,048); similarity stage, us, BF16:
  //   d     n        256   512   1,024  2,048  4,096
  //   128   6,000    82    82    78
  //   128   16,384   279   256   238    234    238
  //   128   32,768   885   744   685    641    638
  //   512   8,192    119   115   121    127
  //   512   24,000   552   511   501    505    538
  //   512   50,000   2100  1922  1826   1783   1805
  //   1,024 16,384   449   434   431    445    480
  //   2,048 8,192    230   232   254    287
  //   2,048 24,000   1378  1359  1375   1435   1572
  int m = TBN;
  if (n >= 16384) m = dp > 1024 ? 2 * TBN : (n >= 32768 ? 8 * TBN : 4 * TBN);
  else if (n >= 8192 && dp <= 1024) m = 2 * TBN;
  if (n >= 131072) m = int(n / 64 / TBN * TBN);  // beyond it: a fixed share, so that the segments stay short
  *sample = m;
  *cap = segment_cap(n, K, m, *segs, most);
}

// The segments of a large instance would outgrow its lists by far (64 KB a row at
// 16 chunks against some 2 to 3 KB of entries: 65 GB at a million rows), so they are
// kept for bands of rows: 4 GB hold the segments of at least 65,536 rows, and a
// launch over so many has thousands of work items for its 76 pairs.
static size_t tc_segment_bytes() {
  // Test hook: smaller bands on small instances.
  const char* e = std::getenv("RERANK_TEST_SEGMENT_BYTES");
  return e ? size_t(std::atoll(e)) : size_t(4) << 30;
}
int64_t tc_append_band(int64_t n, int segs, int cap) {
  const int64_t block = 2 * TBM;  // a band is whole row blocks
  const int64_t rows = int64_t(tc_segment_bytes() / (size_t(segs) * cap * sizeof(uint2))) / block * block;
  return n < rows ? n : (rows < block ? (n < block ? n : block) : rows);
}

static bool launch_sample_pass(const CUtensorMap& map, const CUtensorMap& smap, const TcArgs& S, bool fp8,
                               int sm_count, cudaStream_t s) {
  const int rk = S.floor_rank, items = S.row_blocks;
  if (fp8)
    return rk <= 8 ? launch_sample<MODE_FP8, 8>(map, smap, S, items, sm_count, s)
                   : rk <= 16 ? launch_sample<MODE_FP8, 16>(map, smap, S, items, sm_count, s)
                              : launch_sample<MODE_FP8, 32>(map, smap, S, items, sm_count, s);
  return rk <= 8 ? launch_sample<MODE_BF16, 8>(map, smap, S, items, sm_count, s)
                 : rk <= 16 ? launch_sample<MODE_BF16, 16>(map, smap, S, items, sm_count, s)
                            : launch_sample<MODE_BF16, 32>(map, smap, S, items, sm_count, s);
}

// Returns the number of kernels launched, or a negative value when the tensor
// map cannot be encoded.  xsample / sample_scale: room for sh.sample rows.
int launch_sim_tc_topk(const Shape& sh, const void* xlow, bool fp8, const float* inv_scale, int* row_floor,
                       float* part_s, int32_t* part_i, long long* status, int sm_count, cudaStream_t s,
                       int32_t* work, const TcAppend& ap) {
  CUtensorMap map;
  if (!make_map(&map, xlow, sh.np, sh.dp, fp8)) return -1;
  TcArgs A{};
  A.n = sh.n;
  A.a_rows = sh.n;
  A.col_tiles = int(sh.np / TBN);
  A.kblocks = fp8 ? sh.dp / 128 : sh.dp / 64;
  A.K = sh.K;
  A.inv_scale = inv_scale;
  A.row_floor = row_floor;
  A.part_s = part_s;
  A.part_i = part_i;
  A.status = status;
  A.stall = stall_hook();
  if (sh.segs > 0) {
    A.row_blocks = int(sh.np / (2 * TBM));
    int nl = 0;
    if (sh.sample > 0) {
      CUtensorMap smap;
      if (!make_map(&smap, ap.xsample, sh.sample, sh.dp, fp8)) return -1;
      nl += launch_sample_rows(sh, xlow, fp8, inv_scale, ap, s);
      TcArgs S = A;
      S.n = sh.sample;
      S.col_tiles = sh.sample / TBN;
      S.chunks = 1;
      S.sample_scale = ap.sample_scale;
      S.floor_rank = sample_rank(sh.K, sh.sample, sh.n);
      if (!launch_sample_pass(map, smap, S, fp8, sm_count, s)) return -1;
      ++nl;
    } else {
      cudaMemsetAsync(row_floor, kFloorResetByte, sizeof(int) * size_t(sh.n), s);
    }
    A.chunks = sh.segs / AEG;
    A.cand = static_cast<uint2*>(ap.cand);
    A.cap = sh.seg_cap;
    if (work && tc_dynamic()) A.work = work;
    // A band's rows are selected before the next band takes their segments.
    for (int64_t r0 = 0; r0 < sh.n; r0 += sh.seg_rows) {
      const int64_t rows = sh.n - r0 < sh.seg_rows ? sh.n - r0 : sh.seg_rows;
      A.rb0 = int(r0 / (2 * TBM));
      A.row_blocks = int((rows + 2 * TBM - 1) / (2 * TBM));
      A.seg_cnt = ap.seg_cnt + r0 * sh.segs;
      if (A.work) cudaMemsetAsync(work, 0, sizeof(int32_t), s);
      const int items = A.row_blocks * A.chunks;
      if (!(fp8 ? launch_append<MODE_FP8>(map, A, items, sm_count, s)
                : launch_append<MODE_BF16>(map, A, items, sm_count, s)))
        return -1;
      nl += 1 + launch_select(sh, ap, r0, rows, part_s, part_i, status, s);
    }
    return nl;
  }
  cudaMemsetAsync(row_floor, kFloorResetByte, sizeof(int) * size_t(sh.n), s);
  const int eg = tc_lists_per_chunk(sh.dp, 1);
  A.chunks = sh.P / eg;  // sh.P counts lists per row
  if (A.chunks < 1 || A.chunks * eg != sh.P || A.chunks > A.col_tiles) return -1;
  if (work && tc_dynamic()) {
    cudaMemsetAsync(work, 0, sizeof(int32_t), s);
    A.work = work;
  }
  const bool pairs = use_pairs(A.col_tiles, A.chunks, sm_count) && sh.np % (2 * TBM) == 0;
  A.row_blocks = int(sh.np / (pairs ? 2 * TBM : TBM));
  const int items = A.row_blocks * A.chunks;
  if (pairs) {
    const bool ok = fp8 ? launch_mode_pair<MODE_FP8>(map, map, map, map, A, eg, items, sm_count, s)
                        : launch_mode_pair<MODE_BF16>(map, map, map, map, A, eg, items, sm_count, s);
    return ok ? 1 : -1;
  }
  const int grid = items < sm_count ? items : sm_count;
  if (fp8)
    launch_mode<MODE_FP8>(map, map, map, map, A, eg, grid, s);
  else
    launch_mode<MODE_BF16>(map, map, map, map, A, eg, grid, s);
  return 1;
}

int launch_sample_rows(const Shape& sh, const void* xlow, bool fp8, const float* inv_scale, const TcAppend& ap,
                       cudaStream_t s) {
  const int vecs = sh.dp * (fp8 ? 1 : 2) / 16;
  k_sample_rows<<<unsigned((sh.sample * kWarp + 255) / 256), 256, 0, s>>>(
      static_cast<const uint4*>(xlow), fp8 ? inv_scale : nullptr, sh.n, sh.sample, vecs,
      static_cast<uint4*>(ap.xsample), ap.sample_scale);
  return 1;
}

int launch_select(const Shape& sh, const TcAppend& ap, int64_t r0, int64_t rows, float* part_s, int32_t* part_i,
                  const long long* status, cudaStream_t s) {
  k_select<<<unsigned((rows + SEL_WARPS - 1) / SEL_WARPS), SEL_WARPS * kWarp, 0, s>>>(
      static_cast<const uint2*>(ap.cand), ap.seg_cnt + r0 * sh.segs, rows, sh.segs, sh.seg_cap, sh.K,
      part_s + r0 * sh.K, part_i + r0 * sh.K, status);
  return 1;
}

int launch_sim_tc_rows_append(const Shape& sh, const void* x, int64_t a_rows, int chunks, bool fp8,
                              const float* inv_scale, int* row_floor, const TcAppend& ap, int cap, float* part_s,
                              int32_t* part_i, long long* status, int sm_count, cudaStream_t s) {
  CUtensorMap map, smap;
  if (!make_map(&map, x, sh.n > TBN ? sh.n : TBN, sh.dp, fp8) || !make_map(&smap, ap.xsample, TBN, sh.dp, fp8))
    return -1;
  TcArgs A{};
  A.n = sh.n;
  A.a_rows = a_rows;
  A.row_blocks = int((a_rows + 2 * TBM - 1) / (2 * TBM));
  A.col_tiles = int((sh.n + TBN - 1) / TBN);
  if (chunks < 1 || chunks > A.col_tiles || chunks > kRowsAppendChunks) return -1;
  A.chunks = chunks;
  A.kblocks = fp8 ? sh.dp / 128 : sh.dp / 64;
  A.K = sh.K;
  A.inv_scale = inv_scale;
  A.row_floor = row_floor;
  A.status = status;
  A.stall = stall_hook();
  A.cand = static_cast<uint2*>(ap.cand);
  A.seg_cnt = ap.seg_cnt;
  A.cap = cap;
  TcArgs S = A;
  S.n = TBN;
  S.col_tiles = 1;
  S.chunks = 1;
  S.sample_scale = ap.sample_scale;
  S.floor_rank = sample_rank(sh.K, TBN, sh.n);
  if (!launch_sample_pass(map, smap, S, fp8, sm_count, s)) return -1;
  const int items = A.row_blocks * A.chunks;
  if (!(fp8 ? launch_append<MODE_FP8>(map, A, items, sm_count, s) : launch_append<MODE_BF16>(map, A, items, sm_count, s)))
    return -1;
  Shape rows = sh;
  rows.segs = chunks * AEG;
  rows.seg_cap = cap;
  return 2 + launch_select(rows, ap, 0, a_rows, part_s, part_i, status, s);
}

int launch_sim_tc_rect_topk(const Shape& sh, const void* a, int64_t a_rows, int64_t row0, const void* b,
                            int64_t b_cols, int64_t col0, int chunks, bool fp8, const float* inv_scale,
                            int* row_floor, float* part_s, int32_t* part_i, long long* status, int sm_count,
                            cudaStream_t s, bool seeded) {
  // The maps span at least one full tile (the caller's buffers hold that many rows).
  CUtensorMap ma, mb;
  if (!make_map(&ma, a, a_rows > TBN ? a_rows : TBN, sh.dp, fp8) ||
      !make_map(&mb, b, b_cols > TBN ? b_cols : TBN, sh.dp, fp8))
    return -1;
  if (!seeded) cudaMemsetAsync(row_floor, kFloorResetByte, sizeof(int) * size_t(a_rows), s);
  TcArgs A{};
  A.n = b_cols;
  A.a_rows = a_rows;
  A.row0 = row0;
  A.col0 = col0;
  A.col_tiles = int((b_cols + TBN - 1) / TBN);
  if (chunks < 1 || chunks > A.col_tiles) return -1;  // the caller reads chunks * tc_lists_per_chunk lists per row
  A.chunks = chunks;
  const bool pairs = use_pairs(A.col_tiles, chunks, sm_count);
  const int irows = pairs ? 2 * TBM : TBM;
  A.row_blocks = int((a_rows + irows - 1) / irows);
  const int eg = tc_lists_per_chunk(sh.dp, 1);
  A.kblocks = fp8 ? sh.dp / 128 : sh.dp / 64;
  A.K = sh.K;
  A.inv_scale = inv_scale;
  A.row_floor = row_floor;
  A.part_s = part_s;
  A.part_i = part_i;
  A.status = status;
  A.stall = stall_hook();
  const int items = A.row_blocks * A.chunks;
  if (pairs) {
    const bool ok = fp8 ? launch_mode_pair<MODE_FP8>(ma, ma, mb, mb, A, eg, items, sm_count, s)
                        : launch_mode_pair<MODE_BF16>(ma, ma, mb, mb, A, eg, items, sm_count, s);
    return ok ? 1 : -1;
  }
  const int grid = items < sm_count ? items : sm_count;
  if (fp8)
    launch_mode<MODE_FP8>(ma, ma, mb, mb, A, eg, grid, s);
  else
    launch_mode<MODE_BF16>(ma, ma, mb, mb, A, eg, grid, s);
  return 1;
}

int launch_sim_tc_split_topk(const Shape& sh, int P3, const __nv_bfloat16* ahi, const __nv_bfloat16* alo,
                             const __nv_bfloat16* bhi, const __nv_bfloat16* blo, const int32_t* rows,
                             const int32_t* count, int* row_floor, float* part_s, int32_t* part_i,
                             long long* status, int sm_count, cudaStream_t s, bool seeded) {
  CUtensorMap a0, a1, b0, b1;
  if (!make_map(&a0, ahi, sh.np, sh.dp, false) || !make_map(&a1, alo, sh.np, sh.dp, false) ||
      !make_map(&b0, bhi, sh.np, sh.dp, false) || !make_map(&b1, blo, sh.np, sh.dp, false))
    return -1;
  if (!seeded) cudaMemsetAsync(row_floor, kFloorResetByte, sizeof(int) * size_t(sh.n), s);
  TcArgs A{};
  A.n = sh.n;
  A.row_blocks = 0;
  A.col_tiles = int(sh.np / TBN);
  const int eg = tc_lists_per_chunk(sh.dp, 3);
  A.chunks = P3 / eg;  // P3 counts lists per row
  if (A.chunks < 1 || A.chunks * eg != P3 || A.chunks > A.col_tiles) return -1;
  A.kblocks = sh.dp / 64;
  A.K = sh.K;
  A.rows = rows;
  A.count = count;
  A.row_floor = row_floor;
  A.part_s = part_s;
  A.part_i = part_i;
  A.status = status;
  A.stall = stall_hook();
  // CTA pairs when the rows come in whole 256-row blocks of the padded buffers.
  if (use_pairs(A.col_tiles, A.chunks, sm_count) && sh.np % (2 * TBM) == 0)
    return launch_mode_pair<MODE_SPLIT>(a0, a1, b0, b1, A, eg, INT_MAX, sm_count, s) ? 1 : -1;
  launch_mode<MODE_SPLIT>(a0, a1, b0, b1, A, eg, sm_count, s);
  return 1;
}

size_t tc_batch_inst_bytes() { return 2 * sizeof(TcInst); }  // with its entry of the sampling pass
int tc_batch_max_inst() { return kMaxBatchInst; }
int tc_stall_hook() { return stall_hook(); }

int launch_sim_tc_batch(const TcBatchInst* in, int ninst, bool fp8, void* insts_dev, void* staging, int sm_count,
                        cudaStream_t s) {
  if (ninst < 1 || ninst > kMaxBatchInst) return -1;
  const bool append = in[0].segs > 0;  // all instances of a launch take the same path
  const int eg = append ? AEG : tc_lists_per_chunk(in[0].dp, 1);
  const int irows = append ? 2 * TBM : TBM;
  TcMaps maps;
  TcInst* hi = static_cast<TcInst*>(staging);
  int items = 0, kmax = 0;
  for (int k = 0; k < ninst; ++k) {
    const TcBatchInst& b = in[k];
    if ((b.segs > 0) != append || (!append && tc_lists_per_chunk(b.dp, 1) != eg)) return -1;
    if (!make_map(&maps.m[k], b.xlow, b.np, b.dp, fp8)) return -1;
    TcInst& t = hi[k];
    t.n = b.n;
    t.row_blocks = int(b.np / irows);
    t.col_tiles = int(b.np / TBN);
    t.chunks = append ? b.segs / AEG : b.P / eg;
    if (t.chunks < 1 || (!append && t.chunks * eg != b.P) || t.chunks > t.col_tiles) return -1;
    t.kblocks = fp8 ? b.dp / 128 : b.dp / 64;
    t.K = b.K;
    t.item_begin = items;
    t.inv_scale = b.inv_scale;
    t.row_floor = b.row_floor;
    t.part_s = b.part_s;
    t.part_i = b.part_i;
    t.cand = static_cast<uint2*>(b.ap.cand);
    t.seg_cnt = b.ap.seg_cnt;
    t.cap = b.seg_cap;
    t.floor_rank = 0;
    t.sample_scale = nullptr;
    t.status = b.status;
    items += t.row_blocks * t.chunks;
    kmax = b.K > kmax ? b.K : kmax;
    if (b.sample == 0) cudaMemsetAsync(b.row_floor, kFloorResetByte, sizeof(int) * size_t(b.n), s);
  }
  TcArgs A{};
  A.status = in[0].status;
  A.stall = stall_hook();
  int nl = 1;
  // The sampled instances' floors: a table of their own behind the main one.
  int ns = 0, sitems = 0, rk = 0;
  TcMaps2 smaps;
  if (append) {
    for (int k = 0; k < ninst; ++k) {
      const TcBatchInst& b = in[k];
      if (b.sample == 0) continue;
      smaps.m[ns] = maps.m[k];
      if (!make_map(&smaps.m[kMaxBatchInst + ns], b.ap.xsample, b.sample, b.dp, fp8)) return -1;
      TcInst& t = hi[ninst + ns];
      t = hi[k];
      t.n = b.n;  // rows; the columns are the sample's
      t.col_tiles = b.sample / TBN;
      t.chunks = 1;
      t.item_begin = sitems;
      t.floor_rank = sample_rank(b.K, b.sample, b.n);
      t.sample_scale = b.ap.sample_scale;
      rk = t.floor_rank > rk ? t.floor_rank : rk;
      sitems += t.row_blocks;
      ++ns;
    }
  }
  cudaMemcpyAsync(insts_dev, staging, sizeof(TcInst) * size_t(ninst + ns), cudaMemcpyHostToDevice, s);
  if (ns > 0) {
    TcArgs S = A;
    S.insts = static_cast<const TcInst*>(insts_dev) + ninst;
    S.ninst = ns;
    S.items_total = sitems;
    S.mb_off = kMaxBatchInst;
    bool ok;
    if (fp8)
      ok = rk <= 8 ? launch_sample_batch<MODE_FP8, 8>(smaps, S, sitems, sm_count, s)
                   : rk <= 16 ? launch_sample_batch<MODE_FP8, 16>(smaps, S, sitems, sm_count, s)
                              : launch_sample_batch<MODE_FP8, 32>(smaps, S, sitems, sm_count, s);
    else
      ok = rk <= 8 ? launch_sample_batch<MODE_BF16, 8>(smaps, S, sitems, sm_count, s)
                   : rk <= 16 ? launch_sample_batch<MODE_BF16, 16>(smaps, S, sitems, sm_count, s)
                              : launch_sample_batch<MODE_BF16, 32>(smaps, S, sitems, sm_count, s);
    if (!ok) return -1;
    ++nl;
  }
  A.insts = static_cast<const TcInst*>(insts_dev);
  A.ninst = ninst;
  A.items_total = items;
  if (append) {
    const bool ok = fp8 ? launch_append_batch<MODE_FP8>(maps, A, items, sm_count, s)
                        : launch_append_batch<MODE_BF16>(maps, A, items, sm_count, s);
    return ok ? nl : -1;
  }
  const bool k48 = kmax <= 48;
  const int grid = items < sm_count ? items : sm_count;
  const size_t smem = sizeof(TcSmem) + 1024;
  auto go = [&](auto kernel) {
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
    kernel<<<grid, threads_of(eg), smem, s>>>(maps, A);
  };
  if (fp8) {
    if (eg == 2) k48 ? go(k1_tc_topk_batch<MODE_FP8, 48, 2>) : go(k1_tc_topk_batch<MODE_FP8, KLIST, 2>);
    else k48 ? go(k1_tc_topk_batch<MODE_FP8, 48, 1>) : go(k1_tc_topk_batch<MODE_FP8, KLIST, 1>);
  } else {
    if (eg == 2) k48 ? go(k1_tc_topk_batch<MODE_BF16, 48, 2>) : go(k1_tc_topk_batch<MODE_BF16, KLIST, 2>);
    else k48 ? go(k1_tc_topk_batch<MODE_BF16, 48, 1>) : go(k1_tc_topk_batch<MODE_BF16, KLIST, 1>);
  }
  return nl;
}

int launch_sim_tc_gather_topk(const Shape& sh, int P, const __nv_bfloat16* ahi, const __nv_bfloat16* bhi,
                              const int32_t* rows, const int32_t* count, int* row_floor, float* part_s,
                              int32_t* part_i, long long* status, int sm_count, cudaStream_t s, bool seeded) {
  CUtensorMap a0, b0;
  if (!make_map(&a0, ahi, sh.np, sh.dp, false) || !make_map(&b0, bhi, sh.np, sh.dp, false)) return -1;
  if (!seeded) cudaMemsetAsync(row_floor, kFloorResetByte, sizeof(int) * size_t(sh.n), s);
  TcArgs A{};
  A.n = sh.n;
  A.row_blocks = 0;
  A.col_tiles = int(sh.np / TBN);
  const int eg = tc_lists_per_chunk(sh.dp, 1);
  A.chunks = P / eg;  // P counts lists per row
  if (A.chunks < 1 || A.chunks * eg != P || A.chunks > A.col_tiles) return -1;
  A.kblocks = sh.dp / 64;
  A.K = sh.K;
  A.rows = rows;
  A.count = count;
  A.row_floor = row_floor;
  A.part_s = part_s;
  A.part_i = part_i;
  A.status = status;
  A.stall = stall_hook();
  if (use_pairs(A.col_tiles, A.chunks, sm_count) && sh.np % (2 * TBM) == 0)
    return launch_mode_pair<MODE_GATHER>(a0, a0, b0, b0, A, eg, INT_MAX, sm_count, s) ? 1 : -1;
  launch_mode<MODE_GATHER>(a0, a0, b0, b0, A, eg, sm_count, s);
  return 1;
}

int launch_gather_rows(const int32_t* rows, const int32_t* count, const __nv_bfloat16* hi, const __nv_bfloat16* lo,
                       __nv_bfloat16* dst_hi, __nv_bfloat16* dst_lo, int64_t n, int dp, cudaStream_t s) {
  const int T = 256;
  k_gather_rows<<<unsigned((n * kWarp + T - 1) / T), T, 0, s>>>(
      rows, count, reinterpret_cast<const uint4*>(hi), reinterpret_cast<const uint4*>(lo),
      reinterpret_cast<uint4*>(dst_hi), reinterpret_cast<uint4*>(dst_lo), n, dp / 8);
  return 1;
}

}  // namespace rr
