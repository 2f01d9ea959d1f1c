// Panel preparation, run once per phenotype panel (Section 2.1; Section 2.2, Eq. 1).
//
//   1. X = [1, C] (FP64, column-major), with a non-finite check of C.
//   2. Householder QR of X: a column whose remaining norm is at most
//      1e-9 of its own norm is dropped (rank detection); Q = H_0 ... H_{q-1} [I_q; 0].
//   3. Per phenotype: Y_res = (I - Q Q^T)(Y - Ybar), s_p = |y_res|, and the unit-norm column
//      y_res / s_p written as FP32 and as a BF16 pair hi = bf16(y), lo = bf16(y - hi).
//   4. Q columns 1..q-1 (the non-intercept directions) in FP32 and as a BF16 pair for the
//      marker projection.
//   5. Per column of the BF16 pairs, sum_i (hi + lo) in FP64: the scan adds c * sum back for a
//      marker row shifted by c (the split operand is centred; see k_decode.cu).
// A panel of phenotypes observed on a subset of the samples is prepared on the gathered rows
// (steps 1-5 with N_S samples) and its sample-indexed arrays are then scattered back to the
// full sample axis with zeros elsewhere (k_gather, k_scatter); k_pheno_masks gives each
// phenotype's finite-value mask, from which such subsets are formed.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <mutex>

#include "device.cuh"
#include "internal.h"

namespace tg {
namespace {

constexpr double kRankTol = 1e-9;
constexpr double kPhenoTol = 1e-12;

__global__ void k_build_design(double* __restrict__ X, const double* __restrict__ C, long long ldc,
                               long long N, int n_cov, uint32_t* flags) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= N) return;
  X[i] = 1.0;
  bool bad = false;
  for (int k = 0; k < n_cov; ++k) {
    const double v = C[k * ldc + i];
    bad |= !isfinite(v);
    X[(long long)(k + 1) * N + i] = v;
  }
  if (bad) atomicOr(flags, 1u);
}

// Householder QR of X [k][N] (reduced in place) over the whole GPU, one launch per column.
//
// What bounds it is not the arithmetic (N k^2 FP64 operations, 9 M at N = 23,000, k = 20) but
// the chain of k dependent reductions over N. Reducing one column at a time against every later
// column in a single block (two block-wide reductions per pair of columns, 1 SM) took 6.79 ms at
// N = 23,000, k = 20; here each column costs one launch over all SMs, 0.42 ms in all. A step
// needs only the Gram row g_c = sum_{i >= row} x_j[i] x_c[i], c >= j, of the current column: the
// reflector is v = x_j + s |x_j| e_row, so v . x_c = g_c + s |x_j| x_c[row] for every later
// column at once, and the pass that applies the reflector also sums the next column's Gram row.
// Launches, not a grid-wide barrier, order the steps: every block adds the previous step's
// per-block partial sums in the same order, so all take the same decisions, and nothing spins.
// Row `row` of the reflector of kept column number q is row q, so the basis is
// Q = E - V T (V^T E) (the compact form of H_0 ... H_{q-1} applied to the first q unit vectors),
// one Gram of the reflectors and one pass over the rows.
constexpr int kQrThreads = 256;
constexpr int kQrBlocks = 152;
constexpr int kQrCols = 8;  // columns whose sums a thread carries at once

// Device state of the factorisation, in doubles: the partial sums of two successive steps
// [2][kQrBlocks][2 k], the pivot rows [2][k], the columns' own norms [k], the reflectors' betas
// [k], the number of columns kept before step j [k + 1] and the reflectors' Gram [k][k].
struct QrWork {
  double *part, *piv, *own, *beta, *kept, *gram;
};
__host__ __device__ inline QrWork qr_work(double* w, int k) {
  QrWork r;
  r.part = w;
  r.piv = r.part + (size_t)2 * kQrBlocks * 2 * k;
  r.own = r.piv + 2 * k;
  r.beta = r.own + k;
  r.kept = r.beta + k;
  r.gram = r.kept + k + 1;
  return r;
}

// The warp's sums of 8 per-lane values: lane l returns the sum of column
// 4 [l & 16] + 2 [l & 8] + [l & 4]. Halving the columns as the lanes pair up takes 9 FP64 adds
// per lane instead of 40 (FP64 runs at 2 lanes per cycle and SM).
__device__ __forceinline__ double warp_sum8(const double (&a)[kQrCols], int lane) {
  double b[4], c[2];
  const bool h16 = lane & 16, h8 = lane & 8, h4 = lane & 4;
#pragma unroll
  for (int u = 0; u < 4; ++u)
    b[u] = (h16 ? a[u + 4] : a[u]) + __shfl_xor_sync(0xffffffffu, h16 ? a[u] : a[u + 4], 16);
#pragma unroll
  for (int u = 0; u < 2; ++u)
    c[u] = (h8 ? b[u + 2] : b[u]) + __shfl_xor_sync(0xffffffffu, h8 ? b[u] : b[u + 2], 8);
  double d = (h4 ? c[1] : c[0]) + __shfl_xor_sync(0xffffffffu, h4 ? c[0] : c[1], 4);
  d += __shfl_xor_sync(0xffffffffu, d, 2);
  return d + __shfl_xor_sync(0xffffffffu, d, 1);
}

// Block sums of 8 columns into out[0 .. n), n <= 8.
__device__ __forceinline__ void block_sum8(const double (&a)[kQrCols], int n,
                                           double (*red)[kQrCols], double* out) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const double s = warp_sum8(a, lane);
  if ((lane & 3) == 0) red[warp][((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1)] = s;
  __syncthreads();
  if ((int)threadIdx.x < n) {
    double t = 0.0;
#pragma unroll
    for (int w = 0; w < kQrThreads / 32; ++w) t += red[w][threadIdx.x];
    out[threadIdx.x] = t;
  }
  __syncthreads();
}

// The columns' own sums of squares (partials [k, 2k)) and the first column's Gram row ([0, k)).
__global__ void __launch_bounds__(kQrThreads) k_qr_first(const double* __restrict__ X, long long N,
                                                         int k, double* work) {
  __shared__ double red[kQrThreads / 32][kQrCols];
  const QrWork w = qr_work(work, k);
  const long long step = (long long)gridDim.x * kQrThreads;
  const long long t0 = blockIdx.x * (long long)kQrThreads + threadIdx.x;
  double* out = w.part + (size_t)blockIdx.x * 2 * k;
  for (int c0 = 0; c0 < k; c0 += kQrCols) {
    double g[kQrCols] = {}, o[kQrCols] = {};
    for (long long i = t0; i < N; i += step) {
      const double x0 = X[i];
#pragma unroll
      for (int u = 0; u < kQrCols; ++u)
        if (c0 + u < k) {
          const double v = X[(long long)(c0 + u) * N + i];
          g[u] = fma(x0, v, g[u]);
          o[u] = fma(v, v, o[u]);
        }
    }
    const int n = k - c0 < kQrCols ? k - c0 : kQrCols;
    block_sum8(g, n, red, out + c0);
    block_sum8(o, n, red, out + k + c0);
  }
  if (t0 == 0) {
    for (int c = 0; c < k; ++c) w.piv[c] = X[(long long)c * N];
    w.kept[0] = 0.0;
  }
}

// Step j: the reflector of column j (none if the column is dropped: what is left of it is at most
// kRankTol of its own norm), its application to the later columns, and the Gram row of column
// j + 1 below the next row.
__global__ void __launch_bounds__(kQrThreads) k_qr_step(double* __restrict__ X,
                                                        double* __restrict__ V, long long N, int k,
                                                        int j, double* work, int* rank_out) {
  __shared__ double red[kQrThreads / 32][kQrCols];
  __shared__ double sums[2 * QMAX];
  __shared__ double coef[QMAX];
  const QrWork w = qr_work(work, k);
  const int tid = threadIdx.x, nb = gridDim.x;
  const double* in = w.part + (size_t)(j & 1) * kQrBlocks * 2 * k;
  double* out = w.part + (size_t)((j + 1) & 1) * kQrBlocks * 2 * k + (size_t)blockIdx.x * 2 * k;
  const double* piv = w.piv + (j & 1) * k;
  // the previous launch's partial sums, four threads to a column, in the same order in every block
  const int ncol = j == 0 ? 2 * k : k;
  for (int c0 = j; c0 < ncol; c0 += kQrThreads / 4) {
    const int c = c0 + tid / 4;
    double s = 0.0;
    if (c < ncol)
      for (int b = tid & 3; b < nb; b += 4) s += in[(size_t)b * 2 * k + c];
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    s += __shfl_xor_sync(0xffffffffu, s, 2);
    if (c < ncol && (tid & 3) == 0) sums[c] = s;
  }
  __syncthreads();
  const int q = (int)w.kept[j];  // columns kept so far = this reflector's row
  const double s = sums[j], nrm = sqrt(s);
  const double own = j == 0 ? sqrt(sums[k]) : w.own[j];
  const bool keep = q < N && !(own == 0.0 || nrm <= kRankTol * own);
  const double x0 = piv[j], shift = (x0 >= 0.0 ? 1.0 : -1.0) * nrm;
  // v = x + sign(x0) |x| e_row, |v|^2 = 2 |x|^2 + 2 |x0| |x|
  const double beta = keep ? 2.0 / (2.0 * s + 2.0 * fabs(x0) * nrm) : 0.0;
  if (tid > j && tid < k) coef[tid] = beta * (sums[tid] + shift * piv[tid]);
  const int row = keep ? q + 1 : q;  // the next step's row
  if (blockIdx.x == 0) {
    if (j == 0 && tid < k) w.own[tid] = sqrt(sums[k + tid]);
    if (tid == 0) {
      if (keep) w.beta[q] = beta;
      w.kept[j + 1] = (double)row;
      if (j == k - 1) *rank_out = row;
    }
  }
  __syncthreads();
  double* pnext = w.piv + ((j + 1) & 1) * k;
  const double* xj = X + (long long)j * N;
  double* v = V + (long long)q * N;
  const long long step = (long long)nb * kQrThreads;
  const long long t0 = blockIdx.x * (long long)kQrThreads + tid;
  if (j == k - 1) {
    if (keep)
      for (long long i = t0; i < N; i += step)
        v[i] = i < q ? 0.0 : i == q ? x0 + shift : xj[i];
    return;
  }
  for (int c0 = j + 1; c0 < k; c0 += kQrCols) {
    const int n = k - c0 < kQrCols ? k - c0 : kQrCols;
    double g[kQrCols] = {};
    for (long long i = t0; i < N; i += step) {
      const double vi = i < q ? 0.0 : i == q ? x0 + shift : xj[i];
      if (keep && c0 == j + 1) v[i] = vi;
      if (i < q) continue;
      double xn = 0.0;  // column j + 1 after this reflector (updated in the first group)
      if (c0 > j + 1) xn = X[(long long)(j + 1) * N + i];
#pragma unroll
      for (int u = 0; u < kQrCols; ++u)
        if (u < n) {
          double* xc = X + (long long)(c0 + u) * N + i;
          double x = *xc;
          if (keep) {
            x = fma(-coef[c0 + u], vi, x);
            *xc = x;
          }
          if (u == 0 && c0 == j + 1) xn = x;
          if (i == row) pnext[c0 + u] = x;
          if (i >= row) g[u] = fma(xn, x, g[u]);
        }
    }
    block_sum8(g, n, red, out + c0);
  }
}

// gram[a][b] = v_a . v_b of the reflectors, a < b, one block per pair.
__global__ void __launch_bounds__(256) k_qr_gram(const double* __restrict__ V, long long N, int k,
                                                 double* work) {
  __shared__ double red[33];
  const QrWork w = qr_work(work, k);
  const int a = blockIdx.x, b = blockIdx.y, q = (int)w.kept[k];
  if (a >= b || b >= q) return;
  double s = 0.0;
  for (long long i = b + threadIdx.x; i < N; i += blockDim.x)  // v_b is zero above row b
    s = fma(V[(long long)a * N + i], V[(long long)b * N + i], s);
  s = block_sum(s, red);
  if (threadIdx.x == 0) w.gram[a * k + b] = s;
}

// Q = E - V W with W = T V_top^T: T the upper triangular factor of the compact form
// (T_jj = beta_j, T_ij = -beta_j sum_{i <= m < j} T_im gram_mj), V_top the first q rows of V.
// Every block forms T and W for itself (q^3 / 3 operations), then its rows.
__global__ void __launch_bounds__(256) k_qr_basis(const double* __restrict__ V, long long N, int k,
                                                  double* work, double* __restrict__ Q) {
  extern __shared__ double tw[];  // T [k][k], W [k][k]
  const QrWork w = qr_work(work, k);
  const int q = (int)w.kept[k], tid = threadIdx.x;
  double *T = tw, *W = tw + k * k;
  for (int j = 0; j < q; ++j) {
    if (tid == j) T[j * k + j] = w.beta[j];
    if (tid < j) {
      double s = 0.0;
      for (int m = tid; m < j; ++m) s = fma(T[tid * k + m], w.gram[m * k + j], s);
      T[tid * k + j] = -w.beta[j] * s;
    }
    __syncthreads();
  }
  for (int e = tid; e < q * q; e += blockDim.x) {
    const int a = e / q, c = e - a * q;
    double s = 0.0;
    for (int b = a; b <= c; ++b) s = fma(T[a * k + b], V[(long long)b * N + c], s);
    W[a * k + c] = s;
  }
  __syncthreads();
  for (long long i = blockIdx.x * (long long)blockDim.x + tid; i < N;
       i += (long long)gridDim.x * blockDim.x)
    for (int c0 = 0; c0 < q; c0 += kQrCols) {
      double s[kQrCols] = {};
      for (int a = 0; a < q; ++a) {
        const double va = V[(long long)a * N + i];
#pragma unroll
        for (int u = 0; u < kQrCols; ++u)
          if (c0 + u < q) s[u] = fma(va, W[a * k + c0 + u], s[u]);
      }
#pragma unroll
      for (int u = 0; u < kQrCols; ++u)
        if (c0 + u < q) Q[(long long)(c0 + u) * N + i] = (i == c0 + u ? 1.0 : 0.0) - s[u];
    }
}

// bf16(x + e) in round to nearest even, as the high half of a float, for |e| at most half a unit
// in the last place of x: e only decides where x lies halfway between two bf16 values.
__device__ __forceinline__ uint32_t bf16_bits_of_sum(float x, float e) {
  const uint32_t b = __float_as_uint(x), low = b & 0xFFFFu;
  bool up = low > 0x8000u || (low == 0x8000u && ((b >> 16) & 1u));
  if (low == 0x8000u && e != 0.0f) up = (e > 0.0f) == (x > 0.0f);
  return (b >> 16) + (up ? 1u : 0u);
}
// x += y with the rounding error of the addition returned (Knuth's two-sum).
__device__ __forceinline__ float add_err(float& x, float y) {
  const float t = x + y, z = t - x;
  const float e = (x - (t - z)) + (y - z);
  x = t;
  return e;
}

// Two phenotype columns per block (kResT), which share each load of Q, or one.
//
// FP64 arithmetic bounds it: GB300 runs 2 FP64 lanes per cycle and SM, so each FP64 instruction
// per sample and phenotype costs about 0.08 ms at N = 23,000, P = 2,048, q = 20, where the 40
// multiply-adds of the two projection passes alone take 3.1 ms. So the passes keep what is not
// those products off the FP64 units: the centred value is converted once per ten columns (was
// eight), the centred norm comes from |y_res|^2 + |Q^T y_c|^2, and the bf16 pair and its column
// sum are formed in FP32 from u = f + g, two floats that hold 48 bits of u (the pair is that of
// the FP64 value, see bf16_bits_of_sum; the column sum is a compensated one): 5.86 -> 5.50 ms.
//
// Up to kResOne phenotypes a block takes one: with two, the FP64 chain of a block is twice as long
// while SMs are idle. Preparing 1, 100, 304, 400 and 608 phenotypes at N = 23,000, q = 20 took 1,450,
// 1,490, 1,700, 2,050 and 2,560 us with one per block against 1,800, 1,885, 1,930, 2,370 and 2,450
// with two. A phenotype's arithmetic is the same either way.
constexpr int kResCols = 10, kResOne = 3 * 152;
template <int kResT>
__global__ void __launch_bounds__(256) k_residualise(
    const float* __restrict__ Y, long long ldy, const double* __restrict__ Q, long long N, int P,
    int q, long long Npad, double* __restrict__ Yres, double* __restrict__ s_out,
    float* __restrict__ col_s, float* __restrict__ col_rmul, __nv_bfloat16* __restrict__ Bhi,
    __nv_bfloat16* __restrict__ Blo, float* __restrict__ B32, float* __restrict__ col_cs,
    uint32_t* flags) {
  __shared__ double red[33];
  __shared__ double coef[kResT][QMAX];
  const int p0 = blockIdx.x * kResT;
  const int np = P - p0 < kResT ? P - p0 : kResT;
  const int tid = threadIdx.x, nt = blockDim.x;
  const float* y[kResT];
  double ybar[kResT];
#pragma unroll
  for (int t = 0; t < kResT; ++t) y[t] = Y + (long long)(p0 + (t < np ? t : 0)) * ldy;
  // mean and finiteness
  bool bad = false;
#pragma unroll
  for (int t = 0; t < kResT; ++t) {
    double sum = 0.0;
    for (long long i = tid; i < N; i += nt) {
      const float v = y[t][i];
      bad |= !isfinite(v);
      sum += (double)v;
    }
    ybar[t] = block_sum(sum, red) / (double)N;
  }
  if (bad) atomicOr(flags, 2u);
  // coefficients Q^T (y - ybar), kResCols at a time
  for (int k0 = 0; k0 < q; k0 += kResCols) {
    double acc[kResT][kResCols];
#pragma unroll
    for (int t = 0; t < kResT; ++t)
#pragma unroll
      for (int u = 0; u < kResCols; ++u) acc[t][u] = 0.0;
    for (long long i = tid; i < N; i += nt) {
      double yc[kResT];
#pragma unroll
      for (int t = 0; t < kResT; ++t) yc[t] = (double)y[t][i] - ybar[t];
#pragma unroll
      for (int u = 0; u < kResCols; ++u)
        if (k0 + u < q) {
          const double qv = Q[(long long)(k0 + u) * N + i];
#pragma unroll
          for (int t = 0; t < kResT; ++t) acc[t][u] = fma(qv, yc[t], acc[t][u]);
        }
    }
#pragma unroll
    for (int u = 0; u < kResCols; ++u)
      if (k0 + u < q)
#pragma unroll
        for (int t = 0; t < kResT; ++t) {
          const double c = block_sum(acc[t][u], red);
          if (tid == 0) coef[t][k0 + u] = c;
        }
  }
  __syncthreads();
  // residuals and their norms
  double rs[kResT] = {};
  for (long long i = tid; i < N; i += nt) {
    double r[kResT];
#pragma unroll
    for (int t = 0; t < kResT; ++t) r[t] = (double)y[t][i] - ybar[t];
#pragma unroll 4
    for (int k = 0; k < q; ++k) {
      const double qv = Q[(long long)k * N + i];
#pragma unroll
      for (int t = 0; t < kResT; ++t) r[t] = fma(-qv, coef[t][k], r[t]);
    }
#pragma unroll
    for (int t = 0; t < kResT; ++t) {
      if (t < np) Yres[(p0 + t) * N + i] = r[t];
      rs[t] = fma(r[t], r[t], rs[t]);
    }
  }
#pragma unroll
  for (int t = 0; t < kResT; ++t) {
    const double r2 = block_sum(rs[t], red);
    if (t >= np) continue;  // uniform over the block
    const long long p = p0 + t;
    const double s = sqrt(r2);
    double c2 = r2;  // |y - ybar|^2
    for (int k = 0; k < q; ++k) c2 = fma(coef[t][k], coef[t][k], c2);
    const bool ok = s > kPhenoTol * sqrt(c2);
    if (tid == 0) {
      s_out[p] = s;
      col_s[p] = ok ? (float)s : __int_as_float(0x7fc00000);
      col_rmul[p] = ok ? 1.0f : __int_as_float(0x7fc00000);
    }
    const double inv = ok ? 1.0 / s : 0.0;
    const double* yr = Yres + p * N;
    uint16_t* bh = reinterpret_cast<uint16_t*>(Bhi + p * Npad);
    uint16_t* bl = reinterpret_cast<uint16_t*>(Blo + p * Npad);
    float* bf = B32 + p * Npad;
    float sum = 0.0f, low = 0.0f;  // sum_i (hi + lo), compensated
    for (long long i = tid; i < Npad; i += nt) {
      const double u = (i < N) ? yr[i] * inv : 0.0;
      const float f = (float)u;
      const float g = (float)(u - (double)f);
      const uint32_t hb = bf16_bits_of_sum(f, g);
      const float h = __uint_as_float(hb << 16);
      float r = f - h;  // exact
      const float e = add_err(r, g);
      const uint32_t lb = bf16_bits_of_sum(r, e);
      bh[i] = (uint16_t)hb;
      bl[i] = (uint16_t)lb;
      bf[i] = f;
      low += add_err(sum, h);
      low += add_err(sum, __uint_as_float(lb << 16));
    }
    const double bsum = block_sum((double)sum + (double)low, red);
    if (tid == 0) col_cs[p] = (float)bsum;
  }
}

// Row sums of the bf16 pair of the projection columns.
__global__ void __launch_bounds__(256) k_qcolsum(const __nv_bfloat16* __restrict__ QBhi,
                                                 const __nv_bfloat16* __restrict__ QBlo,
                                                 long long Npad, float* __restrict__ qcs) {
  __shared__ double red[33];
  const long long r = blockIdx.x;
  double cs = 0.0;
  for (long long i = threadIdx.x; i < Npad; i += blockDim.x)
    cs += (double)__bfloat162float(QBhi[r * Npad + i]) + (double)__bfloat162float(QBlo[r * Npad + i]);
  cs = block_sum(cs, red);
  if (threadIdx.x == 0) qcs[r] = (float)cs;
}

__global__ void k_qcols(const double* __restrict__ Q, long long N, int q, long long Npad,
                        float* __restrict__ QB, __nv_bfloat16* __restrict__ QBhi,
                        __nv_bfloat16* __restrict__ QBlo) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const int r = blockIdx.y;  // QB row r = Q column r + 1
  if (i >= Npad) return;
  const double v = (r + 1 < q && i < N) ? Q[(long long)(r + 1) * N + i] : 0.0;
  const long long o = (long long)r * Npad + i;
  QB[o] = (float)v;
  const __nv_bfloat16 h = __double2bfloat16(v);
  QBhi[o] = h;
  QBlo[o] = __double2bfloat16(v - (double)__bfloat162float(h));
}

// The joint operand of a small panel in f16, for the joint pass that decodes dosage rows in
// shared memory (k_fused.cu): rows [0, nq) = Q columns 1..nq, rows [nq, nq + P) = the unit-norm
// residualised phenotypes (0 for an untestable one), the rest 0; each value v (|v| <= 1) scaled
// by 2^14 and split into hi = f16(2^14 v), lo = f16(2^14 v - hi), about 22 significant bits
// (|2^14 v| <= 16,384, inside f16's range, and lo stays a normal number down to |v| ~ 2^-25).
// cs[r] = sum_i (hi + lo) in FP64, rounded to FP32, the scaled column sum of the shift add-back.
__global__ void __launch_bounds__(256) k_joint_f16(const double* __restrict__ Q, long long N, int nq,
                                                   const double* __restrict__ Yres,
                                                   const double* __restrict__ s,
                                                   const float* __restrict__ rmul, int P,
                                                   long long Npad, __half* __restrict__ hi,
                                                   __half* __restrict__ lo, float* __restrict__ cs) {
  __shared__ double red[33];
  const int r = blockIdx.x;
  const double* src = nullptr;
  double mul = 0.0;
  if (r < nq) {
    src = Q + (long long)(r + 1) * N;
    mul = kJointF16Scale;
  } else if (r < nq + P) {
    const int p = r - nq;
    if (rmul[p] == rmul[p]) {  // a testable phenotype: y_res / s, as the bf16 panel
      src = Yres + (long long)p * N;
      mul = (1.0 / s[p]) * kJointF16Scale;
    }
  }
  double sum = 0.0;
  for (long long i = threadIdx.x; i < Npad; i += blockDim.x) {
    const double u = (src && i < N) ? src[i] * mul : 0.0;
    const __half h = __double2half(u);
    const __half l = __double2half(u - (double)__half2float(h));
    hi[(long long)r * Npad + i] = h;
    lo[(long long)r * Npad + i] = l;
    sum += (double)__half2float(h) + (double)__half2float(l);
  }
  sum = block_sum(sum, red);
  if (threadIdx.x == 0) cs[r] = (float)sum;
}

// dst[r][i] = src[r * lds + idx[i]] for r < R, i < ns (rows of a compact copy).
template <class T>
__global__ void k_gather(const T* __restrict__ src, long long lds, T* __restrict__ dst, long long ldd,
                         const int* __restrict__ idx, int ns, int R) {
  const long long total = (long long)R * ns;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const long long r = e / ns;
    const int i = (int)(e - r * ns);
    dst[r * ldd + i] = src[r * lds + idx[i]];
  }
}

// dst[r * ldd + idx[i]] = src[r][i] (dst zeroed beforehand).
template <class T>
__global__ void k_scatter(const T* __restrict__ src, long long lds, T* __restrict__ dst, long long ldd,
                          const int* __restrict__ idx, int ns, int R) {
  const long long total = (long long)R * ns;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const long long r = e / ns;
    const int i = (int)(e - r * ns);
    dst[r * ldd + idx[i]] = src[r * lds + i];
  }
}

// masks[p][w] bit b = Y[p][32 w + b] is finite (bits past N are 0).
__global__ void k_pheno_masks(const float* __restrict__ Y, long long ldy, long long N, long long P,
                              uint32_t* __restrict__ masks, long long ldm) {
  const long long nw = (N + 31) / 32;
  const long long total = P * nw;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const long long p = e / nw, w = e - p * nw;
    uint32_t m = 0;
    for (int b = 0; b < 32; ++b) {
      const long long i = 32 * w + b;
      if (i < N && isfinite(Y[p * ldy + i])) m |= 1u << b;
    }
    masks[p * ldm + w] = m;
  }
}

template <class T>
unsigned grid_for(long long n) {
  long long g = (n + 255) / 256;
  return (unsigned)(g < 152 * 16 ? (g > 0 ? g : 1) : 152 * 16);
}

}  // namespace

cudaError_t launch_gather_f32(const float* src, int64_t lds, float* dst, int64_t ldd, const int* idx,
                              int64_t ns, int64_t R, cudaStream_t st) {
  if (ns == 0 || R == 0) return cudaSuccess;
  k_gather<float><<<grid_for<float>(R * ns), 256, 0, st>>>(src, lds, dst, ldd, idx, (int)ns, (int)R);
  return cudaGetLastError();
}
cudaError_t launch_gather_f64(const double* src, int64_t lds, double* dst, int64_t ldd,
                              const int* idx, int64_t ns, int64_t R, cudaStream_t st) {
  if (ns == 0 || R == 0) return cudaSuccess;
  k_gather<double><<<grid_for<double>(R * ns), 256, 0, st>>>(src, lds, dst, ldd, idx, (int)ns, (int)R);
  return cudaGetLastError();
}
cudaError_t launch_scatter(const void* src, int64_t lds, void* dst, int64_t ldd, const int* idx,
                           int64_t ns, int64_t R, int elem_bytes, cudaStream_t st) {
  if (ns == 0 || R == 0) return cudaSuccess;
  const unsigned g = grid_for<char>(R * ns);
  if (elem_bytes == 8)
    k_scatter<double><<<g, 256, 0, st>>>(static_cast<const double*>(src), lds, static_cast<double*>(dst), ldd, idx, (int)ns, (int)R);
  else if (elem_bytes == 4)
    k_scatter<float><<<g, 256, 0, st>>>(static_cast<const float*>(src), lds, static_cast<float*>(dst), ldd, idx, (int)ns, (int)R);
  else if (elem_bytes == 2)
    k_scatter<unsigned short><<<g, 256, 0, st>>>(static_cast<const unsigned short*>(src), lds, static_cast<unsigned short*>(dst), ldd, idx, (int)ns, (int)R);
  else
    return cudaErrorInvalidValue;
  return cudaGetLastError();
}
cudaError_t launch_pheno_masks(const float* Y, int64_t ldy, int64_t N, int64_t P, uint32_t* masks,
                               int64_t ldm, cudaStream_t st) {
  if (P == 0) return cudaSuccess;
  k_pheno_masks<<<grid_for<char>(P * ((N + 31) / 32)), 256, 0, st>>>(Y, ldy, N, P, masks, ldm);
  return cudaGetLastError();
}

cudaError_t launch_build_design(double* X, const double* C, int64_t ldc, int64_t N, int64_t n_cov,
                                uint32_t* flags, cudaStream_t st) {
  const int tb = 256;
  k_build_design<<<(unsigned)((N + tb - 1) / tb), tb, 0, st>>>(X, C, ldc, N, (int)n_cov, flags);
  return cudaGetLastError();
}

size_t householder_doubles(int64_t N, int64_t k) {
  // X, the reflectors V, the state of the factorisation
  return (size_t)(2 * k * N) + (size_t)2 * kQrBlocks * 2 * k + 2 * k + k + k + (k + 1) + k * k;
}

cudaError_t launch_householder(double* X, int64_t N, int64_t k, double* Q, int* rank_out,
                               cudaStream_t st) {
  double* V = X + k * N;
  double* work = V + k * N;
  const size_t smem = sizeof(double) * 2 * (size_t)(k * k);  // 64 KB at the largest k
  static std::once_flag once;
  static cudaError_t attr = cudaSuccess;
  std::call_once(once, [] {
    attr = cudaFuncSetAttribute(k_qr_basis, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)(sizeof(double) * 2 * QMAX * QMAX));
  });
  if (attr != cudaSuccess) return attr;
  // blocks of a row or so per thread, at most one per SM
  const unsigned nb = (unsigned)std::min<int64_t>(kQrBlocks, (N + kQrThreads - 1) / kQrThreads);
  k_qr_first<<<nb, kQrThreads, 0, st>>>(X, N, (int)k, work);
  for (int64_t j = 0; j < k; ++j)
    k_qr_step<<<nb, kQrThreads, 0, st>>>(X, V, N, (int)k, (int)j, work, rank_out);
  k_qr_gram<<<dim3((unsigned)k, (unsigned)k), 256, 0, st>>>(V, N, (int)k, work);
  k_qr_basis<<<nb, 256, smem, st>>>(V, N, (int)k, work, Q);
  return cudaGetLastError();
}

cudaError_t launch_residualise(const float* Y, int64_t ldy, const double* Q, int64_t N, int64_t P,
                               int64_t q, int64_t Npad, double* Yres, double* s, float* col_s,
                               float* col_rmul, __nv_bfloat16* Bhi, __nv_bfloat16* Blo, float* B32,
                               float* col_cs, uint32_t* flags, cudaStream_t st) {
  if (P == 0) return cudaSuccess;
  const bool one = P <= kResOne;
  const auto k = one ? k_residualise<1> : k_residualise<2>;
  k<<<(unsigned)(one ? P : (P + 1) / 2), 256, 0, st>>>(
      Y, ldy, Q, N, (int)P, (int)q, Npad, Yres, s, col_s, col_rmul, Bhi, Blo, B32, col_cs, flags);
  return cudaGetLastError();
}

cudaError_t launch_joint_f16(const double* Q, int64_t N, int64_t nq, const double* Yres,
                             const double* s, const float* rmul, int64_t P, int64_t rows,
                             int64_t Npad, __half* hi, __half* lo, float* cs, cudaStream_t st) {
  if (rows <= 0) return cudaSuccess;
  k_joint_f16<<<(unsigned)rows, 256, 0, st>>>(Q, N, (int)nq, Yres, s, rmul, (int)P, Npad, hi, lo, cs);
  return cudaGetLastError();
}

cudaError_t launch_qcols(const double* Q, int64_t N, int64_t q, int64_t Npad, float* QB,
                         __nv_bfloat16* QBhi, __nv_bfloat16* QBlo, float* qcs, cudaStream_t st) {
  dim3 grid((unsigned)((Npad + 255) / 256), QCOLS);
  k_qcols<<<grid, 256, 0, st>>>(Q, N, (int)q, Npad, QB, QBhi, QBlo);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_qcolsum<<<QCOLS, 256, 0, st>>>(QBhi, QBlo, Npad, qcs);
  return cudaGetLastError();
}

}  // namespace tg
