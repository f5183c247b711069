// Dense initial features h_i^(0) = x_i (Table 1, first column; Eq. 11 with
// the feature vector in place of the adjacency row): the propagation layers
// of Eq. 13-14 on dense N x d_p rows, and the final query-gallery cosines
// (Alg. 1 step 7).  With alpha = 0, the mean aggregator and one layer this is
// local query expansion (Sec. 3.4, Eq. 4) plus the residual of Eq. 13.
//
// Layer: one warp per row i walks the message list of i built by the graph
// stage (entries (j, c_j) in order, the residual folded into the self
// coefficient; max aggregator: the k2 weighted rows combined element-wise by
// max, then the residual entry marked by c = -1 added), lane l owning the
// float4 columns l, l + 32, ...; the row is divided by its L2 norm (a per-lane
// sum of squares, the 32 partials added in FP64).
//
// Scores: s(q, g) = <h_q, h_g> / (||h_q|| ||h_g||) for every query row q and
// gallery row g, 64 x 128 output tiles per CTA, 8 x 8 per thread.  Each
// 32-deep k-chunk is an FP32 FMA chain; the chunks are added in float-float
// (a TwoSum per chunk), so a score is as accurate as a chain of 32 products
// (about 1e-7 for unit rows) whatever d is; the norms are applied in FP64.
#include "common.cuh"
#include "f32x2.cuh"
#include "internal.hpp"

namespace rr {
namespace {

constexpr int DK = 32;   // k-chunk of the scores

// out_i = normalise(sum_m c_m h_{j_m})  (sum / mean), or
// normalise(max_m (c_m h_{j_m}) + h_i)   (max; the residual entry has c < 0).
__global__ void k7_dense_layer(const float* __restrict__ hin, float* __restrict__ hout, int64_t n, int dp,
                               const int32_t* __restrict__ nbr, const float* __restrict__ nbr_w,
                               const int32_t* __restrict__ nbr_n, int k2, int agg_max) {
  const int64_t i = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (i >= n) return;
  const int m = nbr_n[i];
  const int32_t* nb = nbr + i * (k2 + 1);
  const float* nw = nbr_w + i * (k2 + 1);
  const int nv = dp / 4;
  const float4* in4 = reinterpret_cast<const float4*>(hin);
  float4* out4 = reinterpret_cast<float4*>(hout) + i * nv;
  float ss = 0.f;
  // Two passes over the columns: the first builds the row and its sum of
  // squares, the second scales it (the row is re-read from this row's output).
  for (int q = lane; q < nv; q += kWarp) {
    float4 acc;
    if (agg_max) {
      acc = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
      float4 res = make_float4(0.f, 0.f, 0.f, 0.f);
      for (int e = 0; e < m; ++e) {
        const float c = nw[e];
        const float4 v = __ldg(in4 + int64_t(nb[e]) * nv + q);
        if (c < 0.f) {
          res = v;
        } else {
          acc.x = fmaxf(acc.x, c * v.x);
          acc.y = fmaxf(acc.y, c * v.y);
          acc.z = fmaxf(acc.z, c * v.z);
          acc.w = fmaxf(acc.w, c * v.w);
        }
      }
      acc.x += res.x;
      acc.y += res.y;
      acc.z += res.z;
      acc.w += res.w;
    } else {
      acc = make_float4(0.f, 0.f, 0.f, 0.f);
      for (int e = 0; e < m; ++e) {
        const float c = nw[e];
        const float4 v = __ldg(in4 + int64_t(nb[e]) * nv + q);
        acc.x = fmaf(c, v.x, acc.x);
        acc.y = fmaf(c, v.y, acc.y);
        acc.z = fmaf(c, v.z, acc.z);
        acc.w = fmaf(c, v.w, acc.w);
      }
    }
    ss = fmaf(acc.x, acc.x, ss);
    ss = fmaf(acc.y, acc.y, ss);
    ss = fmaf(acc.z, acc.z, ss);
    ss = fmaf(acc.w, acc.w, ss);
    out4[q] = acc;
  }
  const double tot = warp_sum(double(ss));
  const float inv = tot > 0.0 ? float(1.0 / sqrt(tot)) : 0.f;
  __syncwarp();
  for (int q = lane; q < nv; q += kWarp) {
    float4 v = out4[q];
    v.x *= inv;
    v.y *= inv;
    v.z *= inv;
    v.w *= inv;
    out4[q] = v;
  }
}

// 1 / ||h_i|| in FP64 (per-lane FP32 partials over float4 columns, FP64 warp sum).
__global__ void k7_dense_inv_norms(const float* __restrict__ h, int64_t n, int dp, double* __restrict__ inv) {
  const int64_t i = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (i >= n) return;
  const int nv = dp / 4;
  const float4* r = reinterpret_cast<const float4*>(h) + i * nv;
  float ss = 0.f;
  for (int q = lane; q < nv; q += kWarp) {
    const float4 v = __ldg(r + q);
    ss = fmaf(v.x, v.x, ss);
    ss = fmaf(v.y, v.y, ss);
    ss = fmaf(v.z, v.z, ss);
    ss = fmaf(v.w, v.w, ss);
  }
  const double tot = warp_sum(double(ss));
  if (lane == 0) inv[i] = tot > 0.0 ? 1.0 / sqrt(tot) : 0.0;
}

// Float-float accumulation of two outputs at once: (hi, lo) += p, with Knuth's
// TwoSum for the rounding error.
__device__ __forceinline__ void ff_add(f32x2& hi, f32x2& lo, f32x2 p) {
  const f32x2 s = add2(hi, p);
  const f32x2 bb = sub2(s, hi);
  const f32x2 err = add2(sub2(hi, sub2(s, bb)), sub2(p, bb));
  hi = s;
  lo = add2(lo, err);
}

// Scores by 64 x 128 output tiles, 128 threads of 8 x 8 outputs each (the
// lanes of a warp form a 4 x 8 grid: 32 rows by 64 columns, so that the operand
// loads cost five shared-memory cycles per step), two CTAs per SM so that one
// computes while the other waits at its barriers.  Each 32-deep k-chunk is an
// FP32 FMA chain per output in k order and is added to the output's (hi, lo)
// pair by TwoSum, so a score does not depend on the tile shape or on which
// thread computes it.  All of it runs on column pairs (packed FP32: the same
// values, half the instructions).  The chunk sums p and hi live in registers, lo
// in shared memory (read and written once per chunk).  The operand chunks are
// stored k-major; the next chunk's global loads are issued before the current
// chunk is used.  Bound by the FMA pipe (32 FMAs and 7 additions per output and
// chunk): 6.0 ms for 3,368 x 19,732 x 2,048, the pipe 0.70 busy (8.6 ms with scalar
// FMAs, one CTA of 256 threads per SM and 16-byte loads of separate rows).
constexpr int STM = 64, STN = 128;      // output tile: queries x gallery rows
constexpr int STHREADS = 128;
constexpr size_t SSMEM = size_t(DK) * (STM + STN) * 4 + size_t(32) * STHREADS * 8;  // As, Bs, lo

__global__ void __launch_bounds__(STHREADS, 2)
k7_dense_scores(const float* __restrict__ h, int64_t nq, int64_t ng, int dp, const double* __restrict__ inv,
                float* __restrict__ S) {
  extern __shared__ float4 dyn4[];
  float* As = reinterpret_cast<float*>(dyn4);  // [DK][STM]
  float* Bs = As + DK * STM;                   // [DK][STN]
  f32x2* lo = reinterpret_cast<f32x2*>(Bs + DK * STN);  // [32][STHREADS]
  const int t = threadIdx.x, lane = t & 31, wq = t >> 5;
  const int tr = (wq >> 1) * 32 + (lane >> 3) * 4;  // rows tr + i and tr + 16 + i, i < 4
  const int tc = (wq & 1) * 64 + (lane & 7) * 4;    // columns tc + j and tc + 32 + j, j < 4
  // One grid dimension (the second one ends at 65,535 tiles of queries), gallery tiles first.
  const unsigned gtiles = unsigned((ng + STN - 1) / STN);
  const int64_t q0 = int64_t(blockIdx.x / gtiles) * STM, g0 = int64_t(blockIdx.x % gtiles) * STN;
  f32x2 hi[32], p[32];
#pragma unroll
  for (int j = 0; j < 32; ++j) {
    hi[j] = 0ull;
    lo[j * STHREADS + t] = 0ull;
  }
  // Loader: four lanes read 64 bytes of a row, so that every 32-byte sector is
  // used once; rows lr + 32 s, columns lk + 16 g of the chunk.  Row r of step k
  // is stored at r ^ 8 ((k / 4) mod 4), which keeps 16-byte groups together and
  // the transposing stores free of conflicts.
  const int lr = t >> 2, lk = (t & 3) * 4, lp = lr ^ (8 * (t & 3));
  const float4* arow[STM / 32];
  const float4* brow[STN / 32];
  bool aok[STM / 32], bok[STN / 32];
#pragma unroll
  for (int sl = 0; sl < STM / 32; ++sl) {
    const int64_t qa = q0 + lr + 32 * sl;
    aok[sl] = qa < nq;
    arow[sl] = reinterpret_cast<const float4*>(h + size_t(aok[sl] ? qa : 0) * dp + lk);
  }
#pragma unroll
  for (int sl = 0; sl < STN / 32; ++sl) {
    const int64_t ga = g0 + lr + 32 * sl;
    bok[sl] = ga < ng;
    brow[sl] = reinterpret_cast<const float4*>(h + size_t(bok[sl] ? nq + ga : 0) * dp + lk);
  }
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  float4 va[STM / 32][2], vb[STN / 32][2];
  auto fetch = [&](int step) {
#pragma unroll
    for (int g = 0; g < 2; ++g) {
#pragma unroll
      for (int sl = 0; sl < STM / 32; ++sl) va[sl][g] = aok[sl] ? __ldg(arow[sl] + step + 4 * g) : zero;
#pragma unroll
      for (int sl = 0; sl < STN / 32; ++sl) vb[sl][g] = bok[sl] ? __ldg(brow[sl] + step + 4 * g) : zero;
    }
  };
  fetch(0);
  for (int k0 = 0; k0 < dp; k0 += DK) {
    __syncthreads();  // the previous chunk is consumed
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      const int kk = lk + 16 * g;
#pragma unroll
      for (int sl = 0; sl < STM / 32; ++sl) {
        float* o = As + kk * STM + lp + 32 * sl;
        o[0] = va[sl][g].x;
        o[STM] = va[sl][g].y;
        o[2 * STM] = va[sl][g].z;
        o[3 * STM] = va[sl][g].w;
      }
#pragma unroll
      for (int sl = 0; sl < STN / 32; ++sl) {
        float* o = Bs + kk * STN + lp + 32 * sl;
        o[0] = vb[sl][g].x;
        o[STN] = vb[sl][g].y;
        o[2 * STN] = vb[sl][g].z;
        o[3 * STN] = vb[sl][g].w;
      }
    }
    __syncthreads();
    if (k0 + DK < dp) fetch((k0 + DK) / 4);
#pragma unroll
    for (int j = 0; j < 32; ++j) p[j] = 0ull;
#pragma unroll 16
    for (int k = 0; k < DK; ++k) {
      const int sw = 8 * ((k >> 2) & 3);
      const float4 x0 = *reinterpret_cast<const float4*>(As + k * STM + (tr ^ sw));
      const float4 x1 = *reinterpret_cast<const float4*>(As + k * STM + ((tr + 16) ^ sw));
      const ulonglong2 y0 = *reinterpret_cast<const ulonglong2*>(Bs + k * STN + (tc ^ sw));
      const ulonglong2 y1 = *reinterpret_cast<const ulonglong2*>(Bs + k * STN + ((tc + 32) ^ sw));
      const float xa[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
      const f32x2 yb[4] = {y0.x, y0.y, y1.x, y1.y};
#pragma unroll
      for (int a = 0; a < 8; ++a) {
        const f32x2 a2 = twice(xa[a]);
#pragma unroll
        for (int b = 0; b < 4; ++b) p[a * 4 + b] = fma2(a2, yb[b], p[a * 4 + b]);
      }
    }
#pragma unroll
    for (int j = 0; j < 32; ++j) {
      f32x2 l = lo[j * STHREADS + t];
      ff_add(hi[j], l, p[j]);
      lo[j * STHREADS + t] = l;
    }
  }
#pragma unroll
  for (int a = 0; a < 8; ++a) {
    const int64_t q = q0 + tr + (a < 4 ? a : 12 + a);
    if (q >= nq) continue;
#pragma unroll
    for (int b = 0; b < 8; ++b) {
      const int64_t g = g0 + tc + (b < 4 ? b : 28 + b);
      if (g >= ng) continue;
      const f32x2 hv = hi[a * 4 + b / 2], lv = lo[(a * 4 + b / 2) * STHREADS + t];
      const double dot = (b & 1) ? double(hi_of(hv)) + double(hi_of(lv)) : double(lo_of(hv)) + double(lo_of(lv));
      S[q * ng + g] = float(dot * inv[q] * inv[nq + g]);
    }
  }
}

}  // namespace

int launch_dense_layer(const Shape& sh, const float* hin, float* hout, const int32_t* nbr, const float* nbr_w,
                       const int32_t* nbr_n, int aggregator, cudaStream_t s) {
  const int T = 256;
  k7_dense_layer<<<unsigned((sh.n * kWarp + T - 1) / T), T, 0, s>>>(hin, hout, sh.n, sh.dp, nbr, nbr_w, nbr_n,
                                                                   sh.k2, aggregator == RERANK_AGG_MAX ? 1 : 0);
  return 1;
}

int launch_dense_scores(const Shape& sh, const float* h, double* inv, float* S, cudaStream_t s) {
  const int T = 256;
  k7_dense_inv_norms<<<unsigned((sh.n * kWarp + T - 1) / T), T, 0, s>>>(h, sh.n, sh.dp, inv);
  const unsigned grid = unsigned(((sh.ng + STN - 1) / STN) * ((sh.nq + STM - 1) / STM));
  cudaFuncSetAttribute(k7_dense_scores, cudaFuncAttributeMaxDynamicSharedMemorySize, int(SSMEM));
  k7_dense_scores<<<grid, STHREADS, SSMEM, s>>>(h, sh.nq, sh.ng, sh.dp, inv, S);
  return 2;
}

}  // namespace rr
