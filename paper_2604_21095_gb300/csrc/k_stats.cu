// Statistics of Eq. 3 and the P value, after the contraction (Section 2.2).
//
// The contraction epilogues only keep what needs the accumulator: r for every element in FULL
// mode (stored in one of the caller's output arrays) and raw hit records (marker, phenotype,
// product D). These kernels turn them into
//   t = r sqrt(df / ((1 - r)(1 + r))),  beta = r s_p / (kappa |a_res|),
//   se = s_p / (kappa |a_res|) sqrt((1 - r)(1 + r) / df),  -log10 p with p = I_{1-r^2}(df/2, 1/2).
// Every hit, and every FULL element whose 1 - r^2 is below kExactOmr2, is recomputed in FP64:
// the product g_j . y_res,p from the packed genotype row (missing calls at the FP64 mean) and
// the panel's FP64 residualised phenotype, r from it and the FP64 marker norm, and -log10 p
// in FP64 (the continued fraction, or Hill's deviate where that is within 0.05 of the
// tolerance and the fraction converges slowly; pvalue.cuh). Near |r| = 1 the p-value's slope in r, df / (1 - r^2),
// turns the FP32 product's rounding into errors above the tolerance (see kExactOmr2). The
// other FULL elements take their p-values in FP32 log space (see pvalue.cuh).
#include "device.cuh"
#include "internal.h"

namespace tg {
namespace {

// sum over this thread's groups of 8 samples (8t, 8(t + nt), ...) of (g_i - mean) y_res,p,i in
// FP64, for the marker in block row `row` (the centring adds nothing, since y_res,p sums to zero,
// but keeps the terms small). The eight loads of a group are issued before any is used, so that
// a few hundred threads keep enough loads in flight to stream the 8 N bytes of y_res,p.
__device__ __forceinline__ double exact_partial(const ExactArgs& x, long long row, int col, int t,
                                                int nt) {
  const uint8_t* g = x.G + row * x.ldg;
  const uint32_t* mrow = x.missing ? x.missing + row * x.ldm : nullptr;
  const double mu = x.mean[row];
  const double* y = x.Yres + (long long)col * x.ldy;
  // 2-bit fields 00 (2 copies), 10 (1), 11 (0) minus the mean; 01 (missing) is the mean itself
  const double c00 = 2.0 - mu, c10 = 1.0 - mu, c11 = -mu;
  // dosage bytes minus the rounded mean, exactly, as (2^52 + byte) - (2^52 + round(mean)): one FP64
  // addition instead of a conversion and a subtraction on units that do two a cycle. What is left
  // of the centring multiplies sum_i y_res,p,i = 0; a missing call holds mean - round(mean).
  const double cr = rint(mu), magic = 4503599627370496.0 + cr, cm = mu - cr;
  double acc0 = 0.0, acc1 = 0.0;
  for (int i0 = 8 * t; i0 < x.N; i0 += 8 * nt) {
    const bool whole = i0 + 8 <= x.N;
    double yv[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) yv[u] = (whole || i0 + u < x.N) ? y[i0 + u] : 0.0;
    double v[8];
    if (x.encoding == TG_ENC_2BIT) {  // samples i0..i0+7 in bytes i0/4 and i0/4 + 1
      const unsigned w = (unsigned)g[i0 >> 2] | ((i0 + 4 < x.N ? (unsigned)g[(i0 >> 2) + 1] : 0u) << 8);
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const unsigned f = (w >> (2 * u)) & 3u;
        v[u] = f == 0u ? c00 : f == 2u ? c10 : f == 3u ? c11 : 0.0;
      }
    } else {
      uint2 b = make_uint2(0u, 0u);
      if (whole) {
        b = *reinterpret_cast<const uint2*>(g + i0);  // row starts 16-byte aligned, i0 % 8 == 0
      } else {
        for (int u = 0; i0 + u < x.N; ++u) (u < 4 ? b.x : b.y) |= (unsigned)g[i0 + u] << (8 * (u & 3));
      }
      const unsigned mb = mrow ? (mrow[i0 >> 5] >> (i0 & 31)) & 0xFFu : 0u;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const unsigned byte = ((u < 4 ? b.x : b.y) >> (8 * (u & 3))) & 0xFFu;
        v[u] = ((mb >> u) & 1u) ? cm : __hiloint2double(0x43300000, (int)byte) - magic;
      }
    }
#pragma unroll
    for (int u = 0; u < 8; u += 2) {
      acc0 = fma(v[u], yv[u], acc0);
      acc1 = fma(v[u + 1], yv[u + 1], acc1);
    }
  }
  return acc0 + acc1;
}

// The FP64 statistics of one element from its FP64 product D = g . y_res,p (decode units).
struct Stats64 {
  float beta, se, t, mlp;
};
__device__ __forceinline__ Stats64 stats_exact(const EpiParams& ep, long long row, int col, double D) {
  const double s = ep.col_s64[col];
  const double rinv = ep.row_inv64[row];
  double r = D / s * rinv;
  r = fmin(1.0, fmax(-1.0, r));
  const double omr2 = (1.0 - r) * (1.0 + r);
  const double scale = s * rinv / ep.kappa64;
  Stats64 o;
  o.beta = (float)(r * scale);
  o.se = (float)(scale * sqrt(omr2 / ep.df));
  o.t = (float)(r * sqrt(ep.df / omr2));
  o.mlp = (float)mlog10p_r_dev(r, ep.df, ep.lnB);
  return o;
}

// One FULL element recomputed in FP64 by a whole warp, written by lane `src`. Out of line: it is
// rare, and inlined its registers halve the warps that the ordinary elements run on.
__device__ __noinline__ void full_exact(const EpiParams& ep, long long row, int col, int src) {
  const int lane = threadIdx.x & 31;
  double D = exact_partial(ep.exact, row, col, lane, 32);
  for (int k = 16; k > 0; k >>= 1) D += __shfl_xor_sync(0xffffffffu, D, k);
  if (lane != src) return;
  const long long o = row * ep.ldo + col;
  const Stats64 v = stats_exact(ep, row, col, D);
  if (ep.beta) ep.beta[o] = v.beta;
  if (ep.se) ep.se[o] = v.se;
  if (ep.t) ep.t[o] = v.t;
  if (ep.mlp) ep.mlp[o] = v.mlp;
}

// The FULL statistics of one element per lane (none where !in) from its r; elements near |r| = 1
// are recomputed by the warp. Every lane of the warp calls it.
__device__ __forceinline__ void full_elements(const EpiParams& ep, long long row, int col, float r,
                                              bool in) {
  const float omr2 = (1.0f - r) * (1.0f + r);
  const bool exact = in && ep.exact.G != nullptr && omr2 < kExactOmr2;  // false for NaN
  if (in && !exact) {
    const long long o = row * ep.ldo + col;
    const float rinv = ep.row_inv[row];
    const float scale = ep.col_s[col] * rinv / ep.kappa;
    if (ep.beta) ep.beta[o] = r * scale;
    const float sq = sqrtf(omr2 / ep.df_f);  // t = r sqrt(df / (1 - r^2)) = r / sq
    if (ep.se) ep.se[o] = scale * sq;
    if (ep.t) ep.t[o] = r / sq;
    if (ep.mlp) ep.mlp[o] = mlog10p_r_f(r, ep.df_f, (float)ep.lnB);
  }
  unsigned todo = __ballot_sync(0xffffffffu, exact);
  while (todo) {
    const int src = __ffs(todo) - 1;
    todo &= todo - 1;
    full_exact(ep, __shfl_sync(0xffffffffu, row, src), __shfl_sync(0xffffffffu, col, src), src);
  }
}

// FULL statistics of a block whose contraction left r in one of the outputs. Each warp walks 32
// consecutive elements at a time (all lanes stay in the loop); a lane's row and column advance
// by a fixed stride (drow rows and dcol columns), so that no element costs a 64-bit division.
constexpr int kFullThreads = 256;
__global__ void __launch_bounds__(kFullThreads, 4)
    k_full_stats(const __grid_constant__ EpiParams ep, long long drow, int dcol) {
  chain_wait();
  const long long total = (long long)ep.M * ep.P;
  const long long stride = (long long)gridDim.x * kFullThreads;
  long long e = blockIdx.x * (long long)kFullThreads + threadIdx.x;
  long long row = e / ep.P;
  int col = (int)(e - row * ep.P);
  for (long long base = e - (threadIdx.x & 31); base < total; base += stride, e += stride) {
    const bool in = e < total;
    full_elements(ep, row, col, in ? ep.rstore[row * ep.ldo + col] : 0.0f, in);
    row += drow;
    col += dcol;
    if (col >= ep.P) {
      col -= ep.P;
      row += 1;
    }
  }
}

// Statistics from raw products (EpiParams::raw_out), after the marker norms: per element the
// arithmetic of the contraction epilogue, r = D / |a_res| clamped, the hit test on r^2, the
// column's best marker. A block of 8 warps takes 8 CPW phenotypes, CPW columns per warp, lane =
// marker: the products are column-major, so the reads are whole sectors. Without FULL output
// it takes 128 markers, four per lane, so that a column offers a best marker once per 128.
// In FULL mode it takes 32 markers; the tile of r then goes through shared memory and
// consecutive threads take consecutive phenotypes of a marker, so that the four outputs are
// written in whole sectors too, and r makes no trip through memory.
// CPW = 1 gives a thread one element of a FULL block: on a small one the p-value's chain is the
// whole time (300 x 40 at df = 774: a warp per 32 x 32 elements took 215 us). CPW = 4 (2 with four
// markers per lane) keeps more loads in flight once the block fills the SMs anyway.
constexpr int kRawWarps = 8;
template <bool FULL, int CPW>
__global__ void __launch_bounds__(kRawWarps * 32)
    k_raw_stats(const RawView raw, const __grid_constant__ EpiParams ep, int cgroups) {
  constexpr int R = FULL ? 1 : 4, CW = kRawWarps * CPW;
  __shared__ float tile[FULL ? 32 : 1][CW + 1];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // one grid dimension (the second holds 65,535 blocks), the column groups of a row block in a row
  const int c0 = (int)(blockIdx.x % (unsigned)cgroups) * CW;
  const int cols = min(CW, ep.P - c0);
  const long long row0 = (long long)(blockIdx.x / (unsigned)cgroups) * (32 * R);
  chain_wait();
  float d[R][CPW];
#pragma unroll
  for (int i = 0; i < R; ++i)
#pragma unroll
    for (int u = 0; u < CPW; ++u) d[i][u] = 0.0f;
  // the block's rows are in one tile; a warp's columns may be in two
  int ranges[CPW], most = 0;
#pragma unroll
  for (int u = 0; u < CPW; ++u) {
    const int c = warp * CPW + u;
    ranges[u] = c < cols ? raw_ranges(raw, row0, c0 + c) : 0;
    most = max(most, ranges[u]);
  }
  float rinv[R], shift[R];  // NaN past the block's rows: no test, no hit, no key
#pragma unroll
  for (int i = 0; i < R; ++i) {
    const long long row = row0 + 32 * i + lane;
    const bool in = row < ep.M;
    rinv[i] = in ? ep.row_inv[row] : __int_as_float(0x7fc00000);
    shift[i] = in && raw.partial && raw.cs ? raw.shift[row] : 0.0f;
  }
  // two ranges' loads in flight together (added in range order)
  for (int s = 0; s < most; s += 2) {
    float v[2][R][CPW];
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
      for (int u = 0; u < CPW; ++u)
#pragma unroll
        for (int i = 0; i < R; ++i) {
          const long long row = row0 + 32 * i + lane;
          v[k][i][u] = row < ep.M && s + k < ranges[u]
                           ? raw.x[(s + k) * raw.split + (c0 + warp * CPW + u) * raw.ld + row]
                           : 0.0f;
        }
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
      for (int u = 0; u < CPW; ++u)
#pragma unroll
        for (int i = 0; i < R; ++i)
          if (s + k < ranges[u]) d[i][u] += v[k][i][u];
  }
#pragma unroll
  for (int u = 0; u < CPW; ++u) {
    const int c = warp * CPW + u, col = c0 + c;
    if (c >= cols) break;  // the same for the whole warp
    const float rmul = ep.col_rmul[col];
    const float cs = raw.partial && raw.cs ? raw.cs[col] * raw.cs_scale : 0.0f;
    uint32_t key = 0u, key_row = 0u;  // bits(|r|) + 1 of this lane's best marker (0: none)
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const float D = raw.partial ? fmaf(shift[i], cs, d[i][u]) : d[i][u];
      const float r = corr_nan(D, rinv[i], rmul);
      if (ep.do_hits && r * r >= ep.r2_thr) emit_hit_raw(ep, D, row0 + 32 * i + lane, col);
      if (FULL) tile[lane][c] = r;
      const uint32_t k = r == r ? __float_as_uint(fabsf(r)) + 1u : 0u;
      if (k > key) {  // rows ascend: the smallest marker of equal keys stays
        key = k;
        key_row = 32u * i + lane;
      }
    }
    if (ep.do_best) {
      const uint32_t top = __reduce_max_sync(0xffffffffu, key);
      const uint32_t first = __reduce_min_sync(0xffffffffu, key == top ? key_row : 0xFFFFFFFFu);
      if (top && lane == 0)
        best_offer(ep.best + col,
                   ((unsigned long long)(top - 1u) << 32) |
                       (unsigned long long)(0xFFFFFFFFu -
                                            (uint32_t)(ep.marker_offset + row0 + first)));
    }
  }
  if (!FULL) return;
  __syncthreads();
#pragma unroll 1
  for (int e = threadIdx.x; e < 32 * CW; e += kRawWarps * 32) {  // whole warps stay in the loop
    const int rr = e / CW, cc = e % CW;
    const bool in = cc < cols && row0 + rr < ep.M;
    full_elements(ep, row0 + rr, c0 + cc, in ? tile[rr][cc] : 0.0f, in);
  }
}

// Hit records: the product of each is recomputed in FP64 and one thread writes its FP64 statistics.
// Bound by the FP64 units (two lanes per cycle and SM), with few hits by one hit's chain: its
// sum, then the 17 us of the statistics' own FP64 chain. Few hits leave most SMs idle, so on long
// sample axes the kernel runs in clusters, and while there are at most as many hits as clusters a
// whole cluster shares a hit, each block a part of the samples, added up by the first one (80
// hits on 23,000 samples: 33 us with one block per hit, 23 with 8). With more hits every block
// takes its own: a cluster's blocks would wait for each hit's chain in turn (65,536 x 100 tests on
// 23,000 samples with 6,501 hits: the scan took 3,480 us, now 1,305; with 65,319 hits 30.0 ms, now
// 7.7). On short sample axes the chain is the time (17 us at 5,001 samples, 20 with 8 blocks): one
// block per hit up to kHitSplitN samples.
constexpr int kHitThreads = 256, kHitCluster = 8, kHitSplitN = 8192;
__global__ void __launch_bounds__(kHitThreads)
    k_hit_stats(const __grid_constant__ EpiParams ep, unsigned long long* start) {
  __shared__ double red[33];
  __shared__ double parts[kHitCluster];  // of the first block of a cluster that shares a hit
  __shared__ unsigned long long next[2];
  cluster_arrive();  // the cluster's blocks have all started before any writes to the first one's
  chain_wait();      // shared memory; the wait for the kernel before hides it
  cluster_wait();
  const int tid = (int)threadIdx.x;
  const unsigned long long s0 = start[0];
  unsigned long long s1 = *ep.n_hits;
  if (s1 > (unsigned long long)ep.hit_cap) s1 = (unsigned long long)ep.hit_cap;
  const auto write = [&](unsigned long long i, const tg_hit& h, double D) {
    const Stats64 v = stats_exact(ep, (long long)h.marker - ep.marker_offset, (int)h.pheno, D);
    tg_hit o = h;
    o.beta = v.beta;
    o.se = v.se;
    o.t = v.t;
    o.mlog10p = v.mlp;
    ep.hits[i] = o;
  };
  unsigned nrank;  // blocks per cluster
  asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(nrank));
  if (nrank > 1 && s1 <= s0 + gridDim.x / nrank) {  // the same for the whole grid
    const unsigned rank = blockIdx.x % nrank;
    const unsigned long long i = s0 + blockIdx.x / nrank;
    if (i >= s1) return;
    const tg_hit h = ep.hits[i];
    double D = block_sum(exact_partial(ep.exact, (long long)h.marker - ep.marker_offset,
                                       (int)h.pheno, (int)(rank * kHitThreads) + tid,
                                       (int)(kHitThreads * nrank)), red);
    if (tid == 0) {
      uint32_t dst;
      asm volatile("mapa.shared::cluster.u32 %0, %1, 0;"
                   : "=r"(dst)
                   : "r"((uint32_t)__cvta_generic_to_shared(&parts[rank])));
      asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(dst), "d"(D) : "memory");
    }
    // every block has read the record and delivered its part; the first one stays to read them
    __syncwarp();
    cluster_arrive();
    cluster_wait();
    if (rank == 0 && tid == 0) {
      D = 0.0;
      for (unsigned k = 0; k < nrank; ++k) D += parts[k];
      write(i, h, D);
    }
    return;
  }
  // Each block starts with a hit of its own; further ones come from a counter (cleared before), one
  // ahead: a block that starts late, the grid being more than fits at once, finds less left instead
  // of a fixed share (65,319 hits: 7.7 ms against 10.7).
  const bool more = s1 > s0 + gridDim.x;  // the same for the whole grid
  unsigned long long i = s0 + blockIdx.x;
  for (int turn = 0; i < s1; turn ^= 1) {
    const tg_hit h = ep.hits[i];
    if (more && tid == 0) next[turn] = s0 + gridDim.x + atomicAdd(start + 1, 1ull);
    const double D = block_sum(exact_partial(ep.exact, (long long)h.marker - ep.marker_offset,
                                             (int)h.pheno, tid, kHitThreads), red);
    // (the slot is written again only past another block_sum)
    const unsigned long long after = more ? next[turn] : s1;
    if (tid == 0) write(i, h, D);
    i = after;
  }
}

// Deterministic pseudo-random bytes (SplitMix64 of the index); used for timing trial blocks.
__global__ void k_fill_random(uint8_t* __restrict__ p, size_t n, unsigned long long seed) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x) {
    unsigned long long z = seed + 0x9E3779B97F4A7C15ull * (i + 1);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    p[i] = (uint8_t)((z ^ (z >> 31)) >> 24);
  }
}

}  // namespace

cudaError_t launch_fill_random(uint8_t* p, size_t n, unsigned long long seed, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  k_fill_random<<<152 * 8, 256, 0, st>>>(p, n, seed);
  return cudaGetLastError();
}

cudaError_t launch_full_stats(const EpiParams& ep, cudaStream_t st) {
  if (ep.M == 0 || ep.P == 0) return cudaSuccess;
  const long long total = (long long)ep.M * ep.P;
  long long grid = (total + kFullThreads - 1) / kFullThreads;
  if (grid > 152 * 32) grid = 152 * 32;  // a grid-stride loop: 32 blocks per SM at most
  const long long stride = grid * kFullThreads;
  return launch_chained(k_full_stats, dim3((unsigned)grid), kFullThreads, 0, st, ep, stride / ep.P, (int)(stride % ep.P));
}

cudaError_t launch_raw_stats(const RawView& raw, const EpiParams& ep, cudaStream_t st) {
  if (ep.M == 0 || ep.P == 0) return cudaSuccess;
  const bool small = (long long)ep.M * ep.P < 152ll * 8192;
  const int cw = kRawWarps * (small ? 1 : ep.do_full ? 4 : 2);
  const long long rows = ep.do_full ? 32 : 128;
  const int cgroups = (ep.P + cw - 1) / cw;
  const long long blocks = ((long long)ep.M + rows - 1) / rows * cgroups;
  if (blocks > INT32_MAX) return cudaErrorInvalidConfiguration;
  const dim3 grid((unsigned)blocks);
  constexpr int T = kRawWarps * 32;
  if (ep.do_full)
    return small ? launch_chained(k_raw_stats<true, 1>, grid, T, 0, st, raw, ep, cgroups)
                 : launch_chained(k_raw_stats<true, 4>, grid, T, 0, st, raw, ep, cgroups);
  return small ? launch_chained(k_raw_stats<false, 1>, grid, T, 0, st, raw, ep, cgroups)
               : launch_chained(k_raw_stats<false, 2>, grid, T, 0, st, raw, ep, cgroups);
}

cudaError_t launch_hit_stats(const EpiParams& ep, unsigned long long* start, cudaStream_t st) {
  if (ep.exact.G == nullptr) return cudaErrorInvalidValue;  // hits are always recomputed in FP64
  const unsigned nrank = ep.exact.N > kHitSplitN ? kHitCluster : 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(nrank * (nrank > 1 ? 76 : 304));
  cfg.blockDim = dim3(kHitThreads);
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = nrank;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // as launch_chained
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, k_hit_stats, ep, start);
}

}  // namespace tg
