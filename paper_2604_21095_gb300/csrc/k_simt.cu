// SIMT kernels: marker projection on Q, marker norms, and the plain FP32 scan.
//
// Projection (a reading of Section 2.2, where the paper only standardises each marker):
// every marker is projected on the covariate basis too, so that the correlation with the
// residualised panel is the exact OLS test. Because every column of the residualised
// panel is orthogonal to Q (intercept included), g_res . y_res = g_imputed . y_res, so the
// contraction can use the imputed codes directly and only the norm needs the projection:
// |g_res|^2 = |g_c|^2 - sum_{k>=1} (q_k . g)^2 (q_0 = the intercept direction drops out).
//
// The FP32 scan is the plain-precision form of Eq. 2: FP32 operands, FP32 FFMA, 128 x 128
// tiles of 8 x 8 per thread, followed by the same fused epilogue as the tensor-core path.
#include <cuda_bf16.h>

#include "device.cuh"
#include "internal.h"

namespace tg {
namespace {

// ---------------------------------------------------------------- projection
// qg[k][m] = sum_i A[m][i] QB[k][i]; tile 2,048 / KC markers x KC columns (KC = 16 for up to 16
// columns, else 32), 32 samples per step. K is cut
// into ranges of whole 256-sample chunks over blockIdx.z, each writing its partial sum (a block
// per tile alone left most SMs idle: 47 blocks took 182 us on 3,001 markers x 4,099 samples).
template <int KC>
__global__ void __launch_bounds__(256) k_project(const float* __restrict__ A, long long lda,
                                                 long long M, int K, int range,
                                                 const float* __restrict__ QB, int nq,
                                                 float* __restrict__ qg, long long ldq,
                                                 long long split) {
  constexpr int TM = 2048 / KC;
  __shared__ __align__(16) float As[32][TM + 4];
  __shared__ __align__(16) float Qs[32][KC + 4];
  const int tid = threadIdx.x;
  const long long m0 = (long long)blockIdx.x * TM;
  const int k0 = blockIdx.y * KC;
  const int tx = tid % (KC / 2), ty = tid / (KC / 2);  // 2 columns (k) x 4 markers per thread
  // FP32 partial sums over 256 samples, flushed into FP64 totals
  float acc[4][2] = {{0, 0}, {0, 0}, {0, 0}, {0, 0}};
  double tot[4][2] = {{0, 0}, {0, 0}, {0, 0}, {0, 0}};
  chain_wait(A, QB);
  const int k_lo = (int)blockIdx.z * range, k_hi = min(K, k_lo + range);
  qg += blockIdx.z * split;
  for (int i0 = k_lo; i0 < k_hi; i0 += 32) {
#pragma unroll
    for (int u = 0; u < TM / 32; ++u) {  // A tile: TM rows x 32 samples as 8 TM float4
      const int e = tid + u * 256;
      const int r = e >> 3, c4 = (e & 7) * 4;
      const long long gm = m0 + r;
      float4 v = make_float4(0, 0, 0, 0);
      if (gm < M) v = __ldg(reinterpret_cast<const float4*>(A + gm * lda + i0 + c4));
      As[c4 + 0][r] = v.x;
      As[c4 + 1][r] = v.y;
      As[c4 + 2][r] = v.z;
      As[c4 + 3][r] = v.w;
    }
    if (tid < KC * 8) {  // Q tile: KC columns x 32 samples
      const int r = tid >> 3, c4 = (tid & 7) * 4;
      const float4 v = __ldg(reinterpret_cast<const float4*>(QB + (long long)(k0 + r) * K + i0 + c4));
      Qs[c4 + 0][r] = v.x;
      Qs[c4 + 1][r] = v.y;
      Qs[c4 + 2][r] = v.z;
      Qs[c4 + 3][r] = v.w;
    }
    __syncthreads();
#pragma unroll 8
    for (int i = 0; i < 32; ++i) {
      const float4 a = *reinterpret_cast<const float4*>(&As[i][ty * 4]);
      const float2 q = *reinterpret_cast<const float2*>(&Qs[i][tx * 2]);
      acc[0][0] += a.x * q.x; acc[0][1] += a.x * q.y;
      acc[1][0] += a.y * q.x; acc[1][1] += a.y * q.y;
      acc[2][0] += a.z * q.x; acc[2][1] += a.z * q.y;
      acc[3][0] += a.w * q.x; acc[3][1] += a.w * q.y;
    }
    __syncthreads();
    if (((i0 >> 5) & 7) == 7 || i0 + 32 >= k_hi) {
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b) {
          tot[a][b] += (double)acc[a][b];
          acc[a][b] = 0.0f;
        }
    }
  }
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    const long long gm = m0 + ty * 4 + a;
    if (gm >= M) continue;
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const int k = k0 + tx * 2 + b;
      if (k < nq) qg[k * ldq + gm] = (float)tot[a][b];
    }
  }
}

// ---------------------------------------------------------------- marker norms
// A marker is re-projected in FP64 (refine_projection) when the covariates explain more than
// this share of its variance: |g_res|^2 = |g_c|^2 - sum_k (q_k . g_c)^2 then amplifies the
// rounding of the projections by |g_c|^2 / |g_res|^2 (>= 2 here).
constexpr double kRefineShare = 0.5;

// A marker is tested when it has an observed call, is not constant and its variance inflation
// factor on the covariates, |g_c|^2 / |g_res|^2 = 1 / (1 - R^2 of g on [1, C]), is at most
// kMaxVif: beyond it the covariates explain more than 98% of its variance (the collinearity
// limit PLINK's linear model applies to its predictors by default). Every marker near the
// limit has a ratio far above 1 / (1 - kRefineShare), so its norm is decided in FP64.
constexpr double kMaxVif = 50.0;

__device__ __forceinline__ bool marker_testable(int n_obs, double c2, double r2) {
  return n_obs > 0 && c2 > 0.0 && kMaxVif * r2 >= c2;
}
// complete_n > 0: a marker must also have all complete_n calls observed (the FP4 form, whose
// operand cannot hold a missing call's imputed mean).
__device__ __forceinline__ bool marker_testable(int n_obs, double c2, double r2, int complete_n) {
  return marker_testable(n_obs, c2, r2) && (complete_n <= 0 || n_obs == complete_n);
}

// One block of 8 warps per 32 markers (lane = marker): the warps share the projection columns
// (coalesced reads, the columns being contiguous in the markers), then warp 0 forms the norms
// and warp 1 copies the caller's n_obs and mean. Bound by latency: 12.8 us as three operations on
// 65,536 markers and 19 columns, with row-major products (a sector per value).
constexpr int kNormWarps = 8;

// Markers close to the covariate span (bits of `close`, left by k_marker_norm) are re-projected in
// FP64 by a kernel of their own, marker m by block m % gridDim.x: such markers are neighbours in
// practice (those in linkage with one that is among the covariates), and one costs (q - 1) N
// multiply-adds on units that run two lanes per cycle and SM, so neighbours go to different SMs.
// 65,536 x 16 dosage tests on 23,000 samples with 19 covariates take 424 us, with 32 such markers
// side by side 752 (8,100 when the block of 32 that found them took them one after another). A scan
// without any pays 1.1 to 1.8 us for this launch.
constexpr int kRefineBlocks = 304, kRefineThreads = 256, kRefineCols = 8;

// sum_k (q_k . g_c)^2 over the non-intercept columns of Q in FP64, from the packed genotypes
// (missing calls at the marker's mean, which is also its centre, so they add nothing) and the
// FP64 mean. q_0 . g_c = 0 exactly (q_0 is constant and g_c has zero sum), as in the tensor-core
// projection, which leaves column 0 out. Eight columns at a time share each sample's value. Whole
// block; thread 0 returns the sum.
__device__ double refine_projection(const MarkerRefine& rf, long long j,
                                    double (*red)[kRefineCols]) {
  const double mu = rf.mean[j];
  const uint8_t* row = rf.G + j * rf.ldg;
  const uint32_t* mrow = rf.missing ? rf.missing + j * rf.ldm : nullptr;
  const double c00 = 2.0 - mu, c10 = 1.0 - mu, c11 = -mu;  // 2-bit fields 00, 10, 11; 01 is missing
  double s = 0.0;
  for (int k0 = 1; k0 < rf.q; k0 += kRefineCols) {
    double acc[kRefineCols] = {};
#pragma unroll 2
    for (long long i = threadIdx.x; i < rf.N; i += kRefineThreads) {
      double v;
      if (rf.encoding == TG_ENC_2BIT) {
        const unsigned f = (row[i >> 2] >> (2 * (i & 3))) & 3u;
        v = f == 0u ? c00 : f == 2u ? c10 : f == 3u ? c11 : 0.0;
      } else {
        const bool miss = mrow && ((mrow[i >> 5] >> (i & 31)) & 1u);
        v = miss ? 0.0 : (double)row[i] - mu;
      }
#pragma unroll
      for (int u = 0; u < kRefineCols; ++u)
        if (k0 + u < rf.q) acc[u] = fma(rf.Q[(long long)(k0 + u) * rf.N + i], v, acc[u]);
    }
#pragma unroll
    for (int u = 0; u < kRefineCols; ++u) {
      for (int o = 16; o > 0; o >>= 1) acc[u] += __shfl_xor_sync(0xffffffffu, acc[u], o);
      if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5][u] = acc[u];
    }
    __syncthreads();
    if (threadIdx.x == 0)
      for (int u = 0; u < kRefineCols && k0 + u < rf.q; ++u) {
        double t = 0.0;
        for (int w = 0; w < kRefineThreads / 32; ++w) t += red[w][u];
        s += t * t;
      }
    __syncthreads();
  }
  return s;
}

// The norms of a marker from |g_c|^2 and |g_res|^2 (decode units).
__device__ __forceinline__ void put_norms(const NormOut& out, long long m, int n_obs, double c2,
                                          double r2, int complete_n, double kappa) {
  const bool ok = marker_testable(n_obs, c2, r2, complete_n);
  const double nan = __longlong_as_double(0x7ff8000000000000ll);
  const double inv = ok ? 1.0 / sqrt(r2) : nan;
  if (out.norm2_allele) out.norm2_allele[m] = ok ? r2 * kappa * kappa : nan;
  out.rinv[m] = (float)inv;
  out.rinv64[m] = inv;
}

__global__ void __launch_bounds__(kRefineThreads) k_marker_refine(
    long long M, const int32_t* nobs, const double* gc2, double kappa,
    const __grid_constant__ MarkerRefine rf, const __grid_constant__ NormOut out, int complete_n) {
  __shared__ double red[kRefineThreads / 32][kRefineCols];
  __shared__ unsigned todo[kRefineThreads / 32];
  const int tid = (int)threadIdx.x;
  const long long step = gridDim.x;
  chain_wait();
  for (long long m0 = blockIdx.x; m0 < M; m0 += kRefineThreads * step) {
    const long long j = m0 + tid * step;
    const bool close = j < M && ((out.close[j >> 5] >> (j & 31)) & 1u);
    const unsigned f = __ballot_sync(0xffffffffu, close);
    if ((tid & 31) == 0) todo[tid >> 5] = f;
    if (!__syncthreads_or(close)) continue;
    for (int w = 0; w < kRefineThreads / 32; ++w)  // the same for the whole block
      for (unsigned t = todo[w]; t; t &= t - 1) {
        const long long m = m0 + (32 * w + __ffs(t) - 1) * step;
        const double p = refine_projection(rf, m, red);
        if (tid == 0) put_norms(out, m, nobs[m], gc2[m], gc2[m] - p, complete_n, kappa);
      }
    __syncthreads();
  }
}

// A row's statistics from its exact integer sums: mean = S / n, |g_c|^2 = (n S2 - S^2) / n (the
// numerator exact in 64-bit integers), NaN without an observed call. Byte sums come in two parts
// per piece: n = N (no mask), and S2 <= 255^2 N fits 32 bits for N <= kOnePassMaxN.
__device__ __forceinline__ void row_statistics(const RowSums& sums, long long j, int pieces) {
  long long n, S, S2;
  if (sums.x) {
    uint32_t a = 0, b = 0;
    for (int r = 0; r < 2 * pieces; ++r) {
      a += sums.x[2 * r * sums.ld + j];
      b += sums.x[(2 * r + 1) * sums.ld + j];
    }
    n = sums.N;
    S = a;
    S2 = b;
    sums.nobs[j] = sums.N;
  } else {
    n = sums.nobs[j];
    S = sums.S[j];
    S2 = sums.S2[j];
  }
  const double dn = (double)n, nan = __longlong_as_double(0x7ff8000000000000ll);
  sums.mean[j] = n ? (double)S / dn : nan;
  sums.gc2[j] = n ? (double)(S2 * n - S * S) / dn : nan;
}
__global__ void __launch_bounds__(256) k_row_statistics(long long M, RowSums sums, RawView raw) {
  const long long j = blockIdx.x * 256ll + threadIdx.x;
  chain_wait();
  if (j < M) row_statistics(sums, j, raw_ranges(raw, j, 0));
}

__global__ void __launch_bounds__(kNormWarps * 32) k_marker_norm(
    long long M, const int32_t* nobs, const double* gc2, RawView proj,
    int nq, double kappa, const __grid_constant__ MarkerRefine rf, NormOut out, int complete_n,
    RowSums sums) {
  __shared__ double part[kNormWarps][32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long m0 = blockIdx.x * 32ll, j = m0 + lane;
  const bool in = j < M;
  chain_wait();
  const int ranges = raw_ranges(proj, m0, 0);  // the block's markers and the columns are in one tile
  if ((sums.x || sums.S) && warp == 0 && in) row_statistics(sums, j, ranges);
  // sum of squares in pairs of floats (48 bits): v^2 = p + e exactly, and two-sums. FP64 instructions
  // take 16 cycles of an SM each; with the sum in FP64 a scan takes 0.3 us more on 300 markers, 3.5
  // on 65,536 x 19 columns. The norm's error against 64 bits is the projection's either way (N =
  // 23,000, 19 columns: rms 2.27e-5 of norms near 1e4).
  double s64 = 0.0;
  float hi = 0.0f, lo = 0.0f;
  if (in)
    for (int k = warp; k < nq; k += kNormWarps) {
      const float* x = proj.x + (long long)k * proj.ld + j;
      float v = *x;
      if (proj.sum64) {  // the FP32 form: ranges added in FP64, rounded once
        double w = (double)v;
        for (int r = 1; r < ranges; ++r) w += (double)x[r * proj.split];
        s64 += w * w;
        continue;
      }
      for (int r = 1; r < ranges; ++r) v += x[r * proj.split];
      if (proj.partial) v = fmaf(proj.shift[j], proj.cs[k] * proj.cs_scale, v);
      const float p = v * v;
      const float t = hi + p, z = t - hi;
      lo += fmaf(v, v, -p) + ((hi - (t - z)) + (p - z));
      hi = t;
    }
  part[warp][lane] = proj.sum64 ? s64 : __hiloint2double(__float_as_int(hi), __float_as_int(lo));
  __syncthreads();  // (and the block's writes of the row statistics are visible to the block)
  if (warp == 0) {
    bool close = false;
    if (in) {
      double t = 0.0;
      if (proj.sum64) {
#pragma unroll
        for (int w = 0; w < kNormWarps; ++w) t += part[w][lane];
      } else {
        float h = 0.0f, l = 0.0f;
#pragma unroll
        for (int w = 0; w < kNormWarps; ++w) {
          const float p = __int_as_float(__double2hiint(part[w][lane]));
          const float u = h + p, z = u - h;
          l += __int_as_float(__double2loint(part[w][lane])) + ((h - (u - z)) + (p - z));
          h = u;
        }
        t = (double)h + (double)l;
      }
      const double c2 = gc2[j], r2 = c2 - t;
      put_norms(out, j, nobs[j], c2, r2, complete_n, kappa);
      close = nq > 0 && nobs[j] > 0 && c2 > 0.0 && r2 < (1.0 - kRefineShare) * c2;
    }
    const unsigned f = __ballot_sync(0xffffffffu, close);
    if (lane == 0) {
      if (out.close) out.close[blockIdx.x] = f;
      if (out.hit_start && blockIdx.x == 0) {
        out.hit_start[0] = *out.n_hits;
        out.hit_start[1] = 0ull;
      }
    }
  } else if (warp == 1 && in) {
    if (out.nobs) out.nobs[j] = nobs[j];
    if (out.mean) out.mean[j] = rf.mean[j];
  }
}

// ---------------------------------------------------------------- FP32 scan
// Bound by the FP32 units. A thread's 8 x 8 sums are kept as pairs of columns, so that one packed
// instruction (fma.rn.f32x2, two FMAs with the rounding of two) does the work of two.
// Raw mode (ep.raw_out): K may be split into ranges over blockIdx.z, which write their products
// column-major for k_raw_stats. With 192 tiles on 152 SMs the SMs that got two tiles set the pace
// of 740 us (3,001 markers x 1,000 phenotypes x 4,099 samples).
constexpr int BM = 128, BN = 128, BK = 16;

__device__ __forceinline__ unsigned long long pack2(float a, float b) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void fma2(unsigned long long& c, unsigned long long a,
                                     unsigned long long b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b));
}

__global__ void __launch_bounds__(256, 2) k_sgemm_scan(const float* __restrict__ A, long long lda,
                                                    const float* __restrict__ B, long long ldb,
                                                    int K, int range, EpiParams ep) {
  __shared__ __align__(16) float As[2][BK][BM + 4];
  __shared__ __align__(16) float Bs[2][BK][BN + 4];
  __shared__ unsigned long long colbest[BN];
  const int tid = threadIdx.x;
  const int tx = tid & 15, ty = tid >> 4;
  const long long m0 = (long long)blockIdx.y * BM;
  const int n0 = blockIdx.x * BN;
  // global -> smem mapping: each thread moves 2 float4 of A and 2 of B per K step
  const int lr = tid >> 2, lk = (tid & 3) * 4;
  chain_wait(A, B);
  const int k_lo = (int)blockIdx.z * range, k_hi = min(K, k_lo + range);
  A += k_lo;
  B += k_lo;
  K = k_hi - k_lo;  // a multiple of BK
  const float* Ag0 = A + (m0 + lr) * lda + lk;
  const float* Ag1 = A + (m0 + lr + 64) * lda + lk;
  const float* Bg0 = B + (long long)(n0 + lr) * ldb + lk;
  const float* Bg1 = B + (long long)(n0 + lr + 64) * ldb + lk;
  if (tid < BN) colbest[tid] = 0ull;

  unsigned long long acc2[8][4];  // row a, columns 2b and 2b + 1
#pragma unroll
  for (int a = 0; a < 8; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc2[a][b] = 0ull;

  float4 ra0 = __ldg(reinterpret_cast<const float4*>(Ag0));
  float4 ra1 = __ldg(reinterpret_cast<const float4*>(Ag1));
  float4 rb0 = __ldg(reinterpret_cast<const float4*>(Bg0));
  float4 rb1 = __ldg(reinterpret_cast<const float4*>(Bg1));
  int buf = 0;
  auto stash = [&](int bf) {
    As[bf][lk + 0][lr] = ra0.x; As[bf][lk + 1][lr] = ra0.y; As[bf][lk + 2][lr] = ra0.z; As[bf][lk + 3][lr] = ra0.w;
    As[bf][lk + 0][lr + 64] = ra1.x; As[bf][lk + 1][lr + 64] = ra1.y; As[bf][lk + 2][lr + 64] = ra1.z; As[bf][lk + 3][lr + 64] = ra1.w;
    Bs[bf][lk + 0][lr] = rb0.x; Bs[bf][lk + 1][lr] = rb0.y; Bs[bf][lk + 2][lr] = rb0.z; Bs[bf][lk + 3][lr] = rb0.w;
    Bs[bf][lk + 0][lr + 64] = rb1.x; Bs[bf][lk + 1][lr + 64] = rb1.y; Bs[bf][lk + 2][lr + 64] = rb1.z; Bs[bf][lk + 3][lr + 64] = rb1.w;
  };
  stash(0);
  __syncthreads();
  for (int k0 = 0; k0 < K; k0 += BK) {
    const bool more = k0 + BK < K;
    if (more) {
      ra0 = __ldg(reinterpret_cast<const float4*>(Ag0 + k0 + BK));
      ra1 = __ldg(reinterpret_cast<const float4*>(Ag1 + k0 + BK));
      rb0 = __ldg(reinterpret_cast<const float4*>(Bg0 + k0 + BK));
      rb1 = __ldg(reinterpret_cast<const float4*>(Bg1 + k0 + BK));
    }
#pragma unroll
    for (int k = 0; k < BK; ++k) {
      const float4 a0 = *reinterpret_cast<const float4*>(&As[buf][k][ty * 4]);
      const float4 a1 = *reinterpret_cast<const float4*>(&As[buf][k][64 + ty * 4]);
      const ulonglong2 b0 = *reinterpret_cast<const ulonglong2*>(&Bs[buf][k][tx * 4]);
      const ulonglong2 b1 = *reinterpret_cast<const ulonglong2*>(&Bs[buf][k][64 + tx * 4]);
      const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
#pragma unroll
      for (int a = 0; a < 8; ++a) {
        const unsigned long long aa = pack2(av[a], av[a]);
        fma2(acc2[a][0], aa, b0.x);
        fma2(acc2[a][1], aa, b0.y);
        fma2(acc2[a][2], aa, b1.x);
        fma2(acc2[a][3], aa, b1.y);
      }
    }
    if (more) {
      stash(buf ^ 1);
      __syncthreads();
      buf ^= 1;
    }
  }

  float acc[8][8];
#pragma unroll
  for (int a = 0; a < 8; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b)
      asm("mov.b64 {%0, %1}, %2;" : "=f"(acc[a][2 * b]), "=f"(acc[a][2 * b + 1]) : "l"(acc2[a][b]));
  if (ep.raw_out) {  // four rows of a column at a time (columns start 128-byte aligned)
    float* out = ep.raw_out + (long long)blockIdx.z * ep.raw_split;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const long long row = m0 + 64 * h + ty * 4;
      if (row >= ep.M) continue;  // raw_ld >= M rounded up to 32 holds the whole quad
#pragma unroll
      for (int b = 0; b < 8; ++b) {
        const int col = n0 + (b < 4 ? tx * 4 + b : 64 + tx * 4 + (b - 4));
        if (col < ep.raw_cols)
          *reinterpret_cast<float4*>(out + (long long)col * ep.raw_ld + row) =
              make_float4(acc[4 * h][b], acc[4 * h + 1][b], acc[4 * h + 2][b], acc[4 * h + 3][b]);
      }
    }
    return;
  }

  // epilogue: rows m0 + {ty*4 + a, 64 + ty*4 + a}, columns n0 + {tx*4 + b, 64 + tx*4 + b}
  unsigned long long cb[8];
#pragma unroll
  for (int b = 0; b < 8; ++b) cb[b] = 0ull;
#pragma unroll
  for (int a = 0; a < 8; ++a) {
    const long long row = m0 + (a < 4 ? ty * 4 + a : 64 + ty * 4 + (a - 4));
    if (row >= ep.M) continue;
    const float rinv = ep.row_inv[row];
#pragma unroll
    for (int b = 0; b < 8; ++b) {
      const int col = n0 + (b < 4 ? tx * 4 + b : 64 + tx * 4 + (b - 4));
      if (col >= ep.P) continue;
      const float D = acc[a][b];
      const float r = corr_nan(D, rinv, ep.col_rmul[col]);
      if (ep.do_best) {
        const unsigned long long key = best_key(r, ep.marker_offset + row);
        cb[b] = key > cb[b] ? key : cb[b];
      }
      if (ep.do_hits && r * r >= ep.r2_thr) emit_hit_raw(ep, D, row, col);
      if (ep.do_full) ep.rstore[row * ep.ldo + col] = r;
    }
  }
  if (ep.do_best) {
    // the two ty of a warp share columns: combine, then one shared atomic per column and warp
#pragma unroll
    for (int b = 0; b < 8; ++b) {
      const unsigned long long o = __shfl_xor_sync(0xffffffffu, cb[b], 16);
      cb[b] = o > cb[b] ? o : cb[b];
    }
    if ((tid & 16) == 0) {
#pragma unroll
      for (int b = 0; b < 8; ++b) {
        const int c = b < 4 ? tx * 4 + b : 64 + tx * 4 + (b - 4);
        if (cb[b]) atomicMax(&colbest[c], cb[b]);
      }
    }
    __syncthreads();
    if (tid < BN && n0 + tid < ep.P && colbest[tid]) best_offer(ep.best + n0 + tid, colbest[tid]);
  }
}

}  // namespace

cudaError_t launch_project(const float* A, int64_t lda, int64_t M, int64_t K, const float* QB,
                           int64_t nq, float* out, int64_t ldq, cudaStream_t st, int ranges,
                           int64_t split) {
  if (M == 0 || nq == 0) return cudaSuccess;
  const int64_t range = round_up((K + ranges - 1) / ranges, 256);
  const int kc = nq <= 16 ? 16 : 32, tm = 2048 / kc;
  const dim3 grid((unsigned)((M + tm - 1) / tm), (unsigned)((nq + kc - 1) / kc), (unsigned)ranges);
  // ordinary launches, here and of k_sgemm_scan: several blocks fit an SM, and blocks placed while
  // the kernel before still holds other SMs pile up on the free ones (1,802 x 11 tests, 120 blocks
  // of k_sgemm_scan: on 4,900 samples the scan takes 113 us, 159 with that kernel chained; on
  // 23,000 the kernel takes 273 us, chained 493)
  if (kc == 16)
    k_project<16><<<grid, 256, 0, st>>>(A, lda, M, (int)K, (int)range, QB, (int)nq, out,
                                        (long long)ldq, (long long)split);
  else
    k_project<32><<<grid, 256, 0, st>>>(A, lda, M, (int)K, (int)range, QB, (int)nq, out,
                                        (long long)ldq, (long long)split);
  return cudaGetLastError();
}

cudaError_t launch_row_statistics(int64_t M, const RowSums& sums, const RawView& raw,
                                  cudaStream_t st) {
  if (M == 0) return cudaSuccess;
  return launch_chained(k_row_statistics, dim3((unsigned)((M + 255) / 256)), 256, 0, st, M, sums, raw);
}

cudaError_t launch_marker_norm(int64_t M, const int32_t* nobs, const double* gc2,
                               const RawView& proj, int64_t nq, double kappa,
                               const MarkerRefine& refine, const NormOut& out, cudaStream_t st,
                               int64_t complete_n, const RowSums& sums) {
  if (M == 0) return cudaSuccess;
  NormOut no = out;
  if (nq == 0) no.close = nullptr;  // nothing to re-project
  cudaError_t e = launch_chained(k_marker_norm, dim3((unsigned)((M + 31) / 32)), kNormWarps * 32, 0,
                                 st, M, nobs, gc2, proj, (int)nq, kappa, refine, no,
                                 (int)complete_n, sums);
  if (e != cudaSuccess || nq == 0) return e;
  if (!out.close) return cudaErrorInvalidValue;
  return launch_chained(k_marker_refine, dim3((unsigned)(M < kRefineBlocks ? M : kRefineBlocks)),
                        kRefineThreads, 0, st, M, nobs, gc2, kappa, refine, no, (int)complete_n);
}

cudaError_t launch_sgemm_scan(const float* A, int64_t lda, const float* B, int64_t ldb, int64_t K,
                              const EpiParams& ep, cudaStream_t st) {
  if (ep.M == 0 || ep.P == 0) return cudaSuccess;
  const int ks = ep.raw_out && ep.ksplit > 1 ? ep.ksplit : 1;
  if (ep.raw_out && (ep.raw_cols != ep.P || ep.raw_ld % 32 || ep.raw_ld < ep.M || ep.raw_split % 4))
    return cudaErrorInvalidValue;
  const int64_t range = round_up((K + ks - 1) / ks, BK);
  if ((ks - 1) * range >= K) return cudaErrorInvalidValue;
  dim3 grid((unsigned)((ep.P + BN - 1) / BN), (unsigned)((ep.M + BM - 1) / BM), (unsigned)ks);
  k_sgemm_scan<<<grid, 256, 0, st>>>(A, lda, B, ldb, (int)K, (int)range, ep);
  return cudaGetLastError();
}

}  // namespace tg
