// K1a for instances whose similarity matrix fits in memory: S = Xhat Xhat^T in
// FP32 (Eq. 7), half of its tiles computed, then the K best columns of every
// row (Eq. 8).
//
// The streaming kernel (k1_sim_fp32.cu) computes the whole square because a row
// owner folds every tile of its row into its list.  S is symmetric bit for bit:
// an element is one FMA chain over the feature dimension in k order, and its
// products commute.  Here a tile (bi, bj), bi <= bj, is computed once and stored
// with its transpose, and a selection kernel streams the rows.  The stores and
// the reads of S (2 x 4 n^2 bytes, 0.6 ms at n = 23,100) cost a small part of
// the FMAs saved.
//
// The GEMM is bound by the FP32 FMA pipe.  Its inner loop uses the packed
// fma.rn.f32x2 (two IEEE FMAs per lane and instruction: the same values), which
// halves the issue slots of the FMAs.  128 x 128 tiles, 8 x 16 outputs per
// thread as 8 x 8 column pairs; a warp's lanes form a 4 x 8 grid, so that the
// 16-byte loads of A cost four shared-memory cycles and those of B one (a 2 x 16
// grid with 8 x 8 outputs and A stored twice kept shared memory 70 % busy and
// the FMA pipe 59 %: 22.5 ms; 128 x 256 tiles with one CTA of 256 threads per
// SM instead of two of 128: 19.3 ms, they wait together at every barrier).
// Measured at n = 23,100, d = 2048: the stage 44.9 ms with the streaming kernel,
// 17.8 ms now (GEMM 17.3 ms = 63 TFLOP/s, 0.79 of the FMA peak).
#include <cfloat>
#include <climits>

#include "common.cuh"
#include "f32x2.cuh"
#include "internal.hpp"
#include "topk_heap.cuh"  // score_key / key_score

namespace rr {
namespace {

constexpr int BM = 128;      // tile rows
constexpr int BN = 128;      // tile columns
constexpr int BK = 16;       // k-step
constexpr int NT = BN;       // threads
constexpr int BAND = 8;      // row blocks whose tiles run together (they share column tiles in L2)

// Operands k-major.  Row r of step k sits at r ^ 8 ((k / 4) mod 4), which keeps
// 16-byte groups together and makes the transposing stores free of conflicts.
struct SymSmem {
  float a[2][BK][BM];
  float b[2][BK][BN];
};

// Grid: x = column block * BAND + row block of the band, y = band.  Tiles that
// lie below the diagonal are left out; one that crosses it writes some pairs
// twice, the same bits.
__global__ void __launch_bounds__(NT, 256 / NT)
k1_sgemm_sym(const float* __restrict__ x, int64_t np, int dp, float* __restrict__ S) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  SymSmem& sm = *reinterpret_cast<SymSmem*>(smem_raw);
  const int64_t row0 = (int64_t(blockIdx.y) * BAND + blockIdx.x % BAND) * BM, col0 = int64_t(blockIdx.x / BAND) * BN;
  if (row0 >= np || col0 + BN <= row0) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int WC = BN / 128;                          // warps side by side
  const int tr = (warp / WC) * 32 + (lane >> 3) * 4;    // rows tr + i and tr + 16 + i, i < 4
  const int tc = (warp % WC) * 128 + (lane & 7) * 4;    // columns tc + 32 h + j, h < 4, j < 4
  constexpr int LR = NT / 4, LA = BM / LR, LB = BN / LR;  // loader: rows lr + LR s, columns lk .. lk + 3
  const int lr = tid >> 2, lk = (tid & 3) * 4;
  const int lp = lr ^ (8 * (lk >> 2));                  // its place (adding LR keeps the swizzled bits)
  const float* ag[LA];
  const float* bg[LB];
#pragma unroll
  for (int s = 0; s < LA; ++s) ag[s] = x + (row0 + lr + LR * s) * dp + lk;
#pragma unroll
  for (int s = 0; s < LB; ++s) bg[s] = x + tmin<int64_t>(col0 + lr + LR * s, np - 1) * dp + lk;
  f32x2 acc[8][8];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[i][j] = 0ull;
  float4 ra[LA], rb[LB];
  auto fetch = [&](int off) {
#pragma unroll
    for (int s = 0; s < LA; ++s) ra[s] = __ldg(reinterpret_cast<const float4*>(ag[s] + off));
#pragma unroll
    for (int s = 0; s < LB; ++s) rb[s] = __ldg(reinterpret_cast<const float4*>(bg[s] + off));
  };
  auto stash = [&](int st) {
#pragma unroll
    for (int s = 0; s < LA; ++s) {
      sm.a[st][lk + 0][lp + LR * s] = ra[s].x;
      sm.a[st][lk + 1][lp + LR * s] = ra[s].y;
      sm.a[st][lk + 2][lp + LR * s] = ra[s].z;
      sm.a[st][lk + 3][lp + LR * s] = ra[s].w;
    }
#pragma unroll
    for (int s = 0; s < LB; ++s) {
      sm.b[st][lk + 0][lp + LR * s] = rb[s].x;
      sm.b[st][lk + 1][lp + LR * s] = rb[s].y;
      sm.b[st][lk + 2][lp + LR * s] = rb[s].z;
      sm.b[st][lk + 3][lp + LR * s] = rb[s].w;
    }
  };
  fetch(0);
  stash(0);
  __syncthreads();
  const int nk = dp / BK;
  for (int kt = 0; kt < nk; ++kt) {
    const int cur = kt & 1;
    if (kt + 1 < nk) fetch((kt + 1) * BK);
#pragma unroll
    for (int k = 0; k < BK; ++k) {
      const int sw = 8 * ((k >> 2) & 3);
      const float4 a0 = *reinterpret_cast<const float4*>(&sm.a[cur][k][tr ^ sw]);
      const float4 a1 = *reinterpret_cast<const float4*>(&sm.a[cur][k][(tr + 16) ^ sw]);
      ulonglong2 q[4];
#pragma unroll
      for (int h = 0; h < 4; ++h) q[h] = *reinterpret_cast<const ulonglong2*>(&sm.b[cur][k][(tc + 32 * h) ^ sw]);
      const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const f32x2 a2 = twice(av[i]);
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          acc[i][2 * h] = fma2(a2, q[h].x, acc[i][2 * h]);
          acc[i][2 * h + 1] = fma2(a2, q[h].y, acc[i][2 * h + 1]);
        }
      }
    }
    if (kt + 1 < nk) stash(cur ^ 1);
    __syncthreads();
  }
  // The tile, 16 bytes per store (a warp row's eight lanes write 128 bytes), and
  // its transpose (the four lanes of a column write 64 bytes).
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    float* o = S + (row0 + tr + (i < 4 ? i : 12 + i)) * np + col0 + tc;
#pragma unroll
    for (int h = 0; h < 4; ++h)
      if (col0 + tc + 32 * h < np)
        *reinterpret_cast<float4*>(o + 32 * h) =
            make_float4(lo_of(acc[i][2 * h]), hi_of(acc[i][2 * h]), lo_of(acc[i][2 * h + 1]), hi_of(acc[i][2 * h + 1]));
  }
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const int64_t c = col0 + tc + 32 * (j / 4) + j % 4;
    if (c >= np) continue;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float v[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) v[i] = (j & 1) ? hi_of(acc[4 * h + i][j / 2]) : lo_of(acc[4 * h + i][j / 2]);
      *reinterpret_cast<float4*>(S + c * np + row0 + tr + 16 * h) = make_float4(v[0], v[1], v[2], v[3]);
    }
  }
}

// The K best columns of a row of S by (S desc, index asc), S_ii taken as 1, one
// warp per row.  The row is streamed once; columns above the running floor are
// appended to a buffer in shared memory, and a full buffer is cut down to its K
// best, whose last score becomes the floor (columns arrive in increasing order,
// so a later equal score loses to all K).  Two or three cuts per row: the second
// one happens after ~6,000 columns, the third after ~70,000.  A cut counts the
// entries in 384 log-spaced buckets, scatters those of the buckets that hold the K
// best, and ranks them inside their bucket (as k_select does for the
// tensor-core path).  Bound by reading S: n^2 x 4 bytes.
constexpr int RWARPS = 8;
constexpr int RCAP = 512;
constexpr int RBINS = 384;
constexpr int ROUT = 128;
struct RowSel {
  int key[RCAP];
  int col[RCAP];
  int bin[RBINS];
  int okey[ROUT];
  int ocol[ROUT];
};

// Cuts the first `cnt` entries to the K best, in order; returns their number.
__device__ __noinline__ int cut(RowSel& w, int cnt, int K, int lane) {
  constexpr int kLow = 121 << 23;  // the key of 2^-6
  constexpr int PL = RBINS / kWarp;
  auto bucket = [](int key) { return min(max(key - kLow, 0) >> 17, RBINS - 1); };
  const int want = min(K, cnt);
  __syncwarp();
#pragma unroll
  for (int k = 0; k < PL; ++k) w.bin[lane + k * kWarp] = 0;
  __syncwarp();
  for (int e = lane; e < cnt; e += kWarp) atomicAdd(&w.bin[bucket(w.key[e])], 1);
  __syncwarp();
  int* const mine = w.bin + RBINS - PL * (lane + 1);  // lane 0 holds the highest buckets
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
  int at = incl - sum, last = -1, nsel = 0;
#pragma unroll
  for (int k = 0; k < PL; ++k) {
    mine[PL - 1 - k] = at;
    if (at < want && want <= at + c[k]) {
      last = RBINS - PL * lane - 1 - k;
      nsel = at + c[k];
    }
    at += c[k];
  }
  last = __reduce_max_sync(kFull, last);
  nsel = __reduce_max_sync(kFull, nsel);
  __syncwarp();
  if (nsel <= ROUT) {
    for (int e = lane; e < cnt; e += kWarp) {
      const int k = w.key[e], bk = bucket(k);
      if (bk >= last) {
        const int p = atomicAdd(&w.bin[bk], 1);
        w.okey[p] = k;
        w.ocol[p] = w.col[e];
      }
    }
    __syncwarp();  // bin[b] is now the end of bucket b, and the start of bucket b - 1
    for (int p = lane; p < nsel; p += kWarp) {
      const int k = w.okey[p], v = w.ocol[p], bk = bucket(k);
      const int b1 = w.bin[bk];
      const int b0 = bk == RBINS - 1 ? 0 : w.bin[bk + 1];
      int rank = b0;
      for (int j = b0; j < b1; ++j) rank += (w.okey[j] > k || (w.okey[j] == k && w.ocol[j] < v)) ? 1 : 0;
      if (rank < K) {
        w.key[rank] = k;
        w.col[rank] = v;
      }
    }
  } else {
    // A bucket too crowded for the scatter: the best entry after the last one
    // taken, K times.
    int lkey = INT_MAX, lcol = -1;
    for (int m = 0; m < want; ++m) {
      int bk = INT_MIN, bv = INT_MAX;
      for (int e = lane; e < cnt; e += kWarp) {
        const int k = w.key[e], v = w.col[e];
        if ((k < lkey || (k == lkey && v > lcol)) && (k > bk || (k == bk && v < bv))) {
          bk = k;
          bv = v;
        }
      }
      lkey = __reduce_max_sync(kFull, bk);
      lcol = __reduce_min_sync(kFull, bk == lkey ? bv : INT_MAX);
      if (lane == 0) {
        w.okey[m] = lkey;
        w.ocol[m] = lcol;
      }
    }
    __syncwarp();
    for (int e = lane; e < want; e += kWarp) {
      w.key[e] = w.okey[e];
      w.col[e] = w.ocol[e];
    }
  }
  __syncwarp();
  return want;
}

__global__ void __launch_bounds__(RWARPS * kWarp)
k1_select_rows(const float* __restrict__ S, int64_t ld, int64_t n, int K, float* __restrict__ part_s,
               int32_t* __restrict__ part_i) {
  extern __shared__ RowSel rsel[];
  const int lane = threadIdx.x & 31;
  RowSel& w = rsel[threadIdx.x >> 5];
  const int64_t r = int64_t(blockIdx.x) * RWARPS + (threadIdx.x >> 5);
  if (r >= n) return;
  const unsigned lt = (1u << lane) - 1u;
  const float4* row = reinterpret_cast<const float4*>(S + r * ld);
  float thr = -FLT_MAX;
  int cnt = 0;
  constexpr int U = 4;  // loads in flight
  const int64_t step = int64_t(kWarp) * 4;
  for (int64_t c0 = 0; c0 < n; c0 += U * step) {
    float4 v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t c = c0 + u * step + 4 * lane;  // ld covers whole tiles: in range up to the padding
      v[u] = c < ld ? __ldcs(row + c / 4) : make_float4(-FLT_MAX, -FLT_MAX, -FLT_MAX, -FLT_MAX);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t c = c0 + u * step + 4 * lane;
      float s[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
      if (c + 3 >= n) {  // the padding
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (c + j >= n) s[j] = -FLT_MAX;
      }
      if (c <= r && r < c + 4) {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (c + j == r) s[j] = 1.0f;
      }
      if (!__any_sync(kFull, fmaxf(fmaxf(s[0], s[1]), fmaxf(s[2], s[3])) > thr)) continue;
      if (cnt > RCAP - 4 * kWarp) {
        cnt = cut(w, cnt, K, lane);
        if (cnt == K) thr = key_score(w.key[K - 1]);
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const bool take = s[j] > thr;
        const unsigned bal = __ballot_sync(kFull, take);
        if (take) {
          const int p = cnt + __popc(bal & lt);
          w.key[p] = score_key(s[j]);
          w.col[p] = int(c + j);
        }
        cnt += __popc(bal);
      }
    }
  }
  cnt = cut(w, cnt, K, lane);
  for (int e = lane; e < K; e += kWarp) {
    part_s[r * K + e] = e < cnt ? key_score(w.key[e]) : -FLT_MAX;
    part_i[r * K + e] = e < cnt ? w.col[e] : kInvalidIdx;
  }
}

}  // namespace

int launch_sim_sym_topk(const Shape& sh, const float* xhat, float* S, float* part_s, int32_t* part_i, cudaStream_t s) {
  // Above 48 KB; the attribute belongs to the current device, so every launch sets it.
  cudaFuncSetAttribute(k1_select_rows, cudaFuncAttributeMaxDynamicSharedMemorySize, int(RWARPS * sizeof(RowSel)));
  const int64_t rb = sh.np / BM, cb = (sh.np + BN - 1) / BN;
  const dim3 grid(unsigned(cb * BAND), unsigned((rb + BAND - 1) / BAND));
  k1_sgemm_sym<<<grid, NT, sizeof(SymSmem), s>>>(xhat, sh.np, sh.dp, S);
  k1_select_rows<<<unsigned((sh.n + RWARPS - 1) / RWARPS), RWARPS * kWarp, RWARPS * sizeof(RowSel), s>>>(
      S, sh.np, sh.n, sh.K, part_s, part_i);
  return 2;
}

}  // namespace rr
