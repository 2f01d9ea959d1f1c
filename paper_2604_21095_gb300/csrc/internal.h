// Internal declarations shared by the library's translation units (not part of the ABI).
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <string>
#include <vector>

#include "../../include/tg.h"

namespace tg {

// Latched device status bits (ctx->status).
enum : uint32_t { ST_CAPACITY = 1u, ST_TIMEOUT = 2u };

constexpr int KPAD = 64;     // sample dimension (GEMM K) padding of every operand row
constexpr int kAccumChunkKB = 32;  // tensor-core accumulation chunk: 32 K blocks of 32 samples
constexpr int PPAD = 256;    // phenotype rows padding of the panel operands (tensor-core N tile)
constexpr int QMAX = 64;     // intercept + at most 63 covariates
constexpr int kMaxHostBufs = 4;  // block buffers of the host-streamed scan, at most
// blocks of the host-streamed scan in flight at once (their scan-done events), at most
constexpr int kRingEvents = 8 * kMaxHostBufs + 8;
// blocks of a host-streamed scan (the second to the ninth) whose copies and scans are timed for
// the next call's block growth
constexpr int kRateBlocks = 8;
constexpr int QCOLS = 64;    // projection columns (Q columns 1..q-1), zero padded
constexpr int JCOLS = 512;   // widest joint operand: projection columns + panel in one pass
constexpr int MT = 128;      // marker rows per tensor-core tile
constexpr int kFp4Pieces = 6;  // E2M1 pieces of the panel in the FP4 form (k_fp4.cu)
// Scale of the f16 joint operand (k_joint_f16): values of at most 1 in magnitude become at most
// 2^14, inside f16's range, with the low piece a normal number for |v| >= ~2^-25.
constexpr double kJointF16Scale = 16384.0;

enum Stage { STAGE_DECODE = 0, STAGE_PROJECT = 1, STAGE_NORM = 2, STAGE_GEMM = 3, STAGE_H2D = 4,
             STAGE_STATS = 5 };

inline int64_t round_up(int64_t x, int64_t m) { return (x + m - 1) / m * m; }

// Columns of a CTA-pair tile for an operand of `cols` columns: the fewest tiles of at most 256
// columns, all of one width, a multiple of 32 (the MMA's step). Against 256-column tiles that
// saves the products of the padding, 300 columns being 2 x 160 instead of 2 x 256.
inline int64_t tile_cols(int64_t cols) {
  const int64_t c = cols > 0 ? cols : 1, n = (c + 255) / 256;
  return round_up((c + n - 1) / n, 32);
}

// What the FP64 recomputation of a product g_j . y_res,p needs (hits, and FULL elements near
// |r| = 1): the packed genotype block, its FP64 observed means (decode units; a missing call is
// imputed with it) and the panel's FP64 residualised phenotypes [P][ldy]. G = NULL: off.
struct ExactArgs {
  const uint8_t* G;
  long long ldg;
  int encoding;
  int N;
  const uint32_t* missing;  // dosage mask [M][ldm] or NULL
  long long ldm;
  const double* mean;       // [M]
  const double* Yres;       // [P][ldy], zero outside a subset panel's samples
  long long ldy;
};

// FULL elements whose FP32 1 - r^2 is below this are recomputed in FP64 (hits always are):
// r from the FP32 product carries an absolute error of up to ~5e-7, and d(-log10 p)/dr =
// df |r| / ((1 - r^2) ln 10) makes that exceed the 1e-5 relative tolerance on -log10 p once
// (1 - r^2) ln(1 / (1 - r^2)) < ~0.1, i.e. 1 - r^2 < ~0.03, at every df.
constexpr float kExactOmr2 = 0.05f;

// Per-element statistics inputs shared by both contraction kernels' epilogues.
struct EpiParams {
  int M, P;                    // block rows (markers) and panel phenotypes
  long long marker_offset;
  double df;                   // N - q - 1
  float df_f;
  double lnB;                  // ln Beta(df/2, 1/2)
  float kappa;                 // allele units per decode unit (1 or 2/255), FP32 kernels
  double kappa64;              // the same in FP64 (hit statistics)
  float r2_thr;                // hit threshold on r^2 (> 1 disables)
  int do_full, do_hits, do_best;
  const float* row_inv;        // [M] 1/|a_res| (decode units), NaN = untestable
  const double* row_inv64;     // [M]
  const float* col_s;          // [P] s_p, NaN = untestable phenotype
  const double* col_s64;       // [P]
  const float* col_rmul;       // [P] 1 or NaN
  const float* row_shift;      // [M] c the operand row was shifted by (NULL = none)
  const float* col_cs;         // [P] sum_i of the B operand column (the shift's add-back)
  float *beta, *se, *t, *mlp;  // FULL outputs, [M][ldo]
  float* rstore;               // FULL mode: where the contraction leaves r (one of the above)
  long long ldo;
  tg_hit* hits;
  long long hit_cap;
  unsigned long long* n_hits;
  unsigned long long* best;
  uint32_t* status;
  unsigned long long* wave_ctr;  // CTA-pair lockstep counter (zeroed per launch), NULL = off
  // raw mode: the product of row m and column k < raw_cols goes to raw_out[k * raw_ld + m]
  // (column-major, so that the 32 rows of a warp store whole sectors). Unsplit, that is D with
  // the shift's add-back. With split-K (raw mode only, ksplit > 1: K in `ksplit` chunk-aligned
  // ranges) range s writes its partial sums, without the add-back, raw_split floats further
  // on; the kernels that read them (k_marker_norm, k_raw_stats) add the ranges in order.
  float* raw_out;
  int raw_cols;
  long long raw_ld, raw_split;
  int ksplit;
  ExactArgs exact;             // FP64 recomputation of hits and of FULL elements near |r| = 1
};

// Packed genotypes for a contraction kernel that decodes its A operand in the producer
// (2-bit calls, or dosage bytes without a missing mask; split form only). The kernel loads the
// packed rows through `tmG` (uint8, {ldg, M}, boxes of 32 or 16 bytes x 128 rows).
constexpr int kOnePassMaxN = 66051;  // 255^2 * N < 2^32
struct DecodeArgs {
  CUtensorMap tmG;
  int N;                  // samples; K columns >= N are zero
  int M;                  // rows of the block; rows >= M are zero
  const float* shift;     // [M] row shift c
  const uint32_t* mh;     // [M] bf16 bits of (mean - c), the missing-call value
  // Dosage rows without a mask in the joint pass: when sums is set, the pass takes each row's
  // shift from the row's first 64 samples (read through G) instead of reading `shift`, writes it
  // to shift_out, and leaves the sums of the row's bytes and of their squares, in parts that
  // k_marker_norm adds up (RowSums), so no counting pass runs.
  const uint8_t* G;
  long long ldg;
  float* shift_out;
  uint32_t* sums;
  long long sums_ld;
  // The projection pass of a larger panel (the 64 projection columns alone): when a_out is set,
  // the pass also stores each expanded row as the block's bf16 operand (row-major, lda_out
  // elements per row, every column of rows < M), which the panel's contraction then reads as it
  // would the decoded operand.
  __nv_bfloat16* a_out;
  long long lda_out;
};

struct Events {
  cudaEvent_t a, b;
  int stage;
};

// Arguments of one block scan (the tg_scan_block call).
struct ScanArgs {
  const uint8_t* G;
  int64_t ldg;
  int encoding;
  int64_t N, M, marker_offset;
  const uint32_t* missing;
  int64_t ldm;
  tg_scan_opts opts;
  tg_outputs out;
};

// Kernel choice per block-size bucket (floor(log2 M)), set by tg_autotune.
enum { TUNE_DEFAULT = 0, TUNE_PAIR = 1, TUNE_SINGLE = 2 };
constexpr int kTuneBuckets = 40;
inline int tune_bucket(int64_t M) {
  int b = 0;
  while ((M >> (b + 1)) > 0 && b + 1 < kTuneBuckets) ++b;
  return b;
}

}  // namespace tg

struct tg_panel {
  int device = 0;
  int64_t N = 0, P = 0, n_cov = 0, q = 0, df = 0, Npad = 0, Ppad = 0;
  std::vector<void*> memory;    // the allocations that hold every buffer below but the FP4 form's
  int64_t NS = 0;               // samples the panel's phenotypes use (N unless a subset)
  uint32_t* samples = nullptr;  // [ceil(N/32)] bit mask of those samples (subset panels only)
  double* X = nullptr;        // [(1+n_cov)][N] design, reduced in place by the QR; its workspace
  double* Q = nullptr;        // [q][N] (column-major N x q)
  double* Yres = nullptr;     // [P][N]
  double* s = nullptr;        // [P]
  float* col_s = nullptr;     // [P]
  float* col_rmul = nullptr;  // [Ppad]
  float* col_cs = nullptr;    // [Ppad] sum_i (Bhi + Blo)[p][i], in FP32
  __nv_bfloat16* Bhi = nullptr;  // [Ppad][Npad] unit-norm panel, high part
  __nv_bfloat16* Blo = nullptr;  // [Ppad][Npad] low part
  float* B32 = nullptr;          // [Ppad][Npad] unit-norm panel in FP32
  float* QB = nullptr;           // [QCOLS][Npad] Q columns 1..q-1 in FP32 (rest zero)
  __nv_bfloat16* QBhi = nullptr; // [QCOLS][Npad] the same split into bf16 hi + lo
  __nv_bfloat16* QBlo = nullptr;
  float* qcs = nullptr;          // [QCOLS] sum_i (QBhi + QBlo)[k][i]
  double lnB = 0;                // ln B(df/2, 1/2), df = N - q - 1
  double lnB_paper = 0;          // ln B((N-2)/2, 1/2) for the paper's printed form
  CUtensorMap tmBhi, tmBlo;      // phenotype panel, 256-row boxes
  // rows of the projection operand that a pass reads: q - 1 rounded up to 16
  int proj_bn() const { return (int)tg::round_up(q > 1 ? q - 1 : 1, 16); }
  int bn = 0;                    // columns of a CTA-pair tile (tile_cols(P))
  CUtensorMap tmBhi2, tmBlo2;    // phenotype panel, boxes of bn / 2 rows (one CTA's half of a pair tile)
  CUtensorMap tmQhi, tmQlo;      // covariate projection columns, boxes of proj_bn() rows
  CUtensorMap tmBhi64, tmBlo64;  // phenotype panel, 64-row boxes (64-column tiles, P <= 64)
  // Panels with P + q - 1 <= JCOLS: the projection columns and the phenotypes in one operand,
  // rows [0, q-1) = QB rows, rows [q-1, q-1+P) = the panel, rest zero, so that one pass over a
  // block's operand gives both Q^T a and the panel's products (joint_cols = 0 and NULL buffers
  // when the panel is larger). Up to 128 rows the operand has joint_cols = 64 or 128 rows, one
  // tile of the one-CTA kernels, which read joint_bn of them (P + q - 1 rounded up to 16, the
  // maps' boxes); above, it has joint_cols = n x joint_bn rows, n = 1 or 2 tiles of joint_bn
  // columns of the CTA-pair kernel (the maps' boxes hold half a tile).
  int joint_cols = 0, joint_bn = 0;
  __nv_bfloat16* QYhi = nullptr;  // [joint_cols][Npad]
  __nv_bfloat16* QYlo = nullptr;
  float* qycs = nullptr;          // [joint_cols] qcs then col_cs
  CUtensorMap tmQYhi, tmQYlo;     // boxes of joint_bn rows (joint_bn / 2 above 128)
  // The same joint operand as f16 hi + lo of 2^14 v (joint_cols <= 128 only), for the joint pass
  // that decodes dosage rows in shared memory into f16 (k_fused.cu); scaled column sums.
  __half* QYhi16 = nullptr;       // [joint_cols][Npad]
  __half* QYlo16 = nullptr;
  float* qycs16 = nullptr;        // [joint_cols]
  CUtensorMap tmQYhi16, tmQYlo16;
  // The projection columns alone in the same f16 form (64 rows; panels with P + q - 1 > JCOLS),
  // for the projection pass over dosage rows that also writes the block's operand (k_fused.cu).
  __half* QBhi16 = nullptr;       // [QCOLS][Npad]
  __half* QBlo16 = nullptr;
  float* qcs16 = nullptr;         // [QCOLS]
  CUtensorMap tmQhi16, tmQlo16;
  // The FP4 form's E2M1 pieces (built on the panel's first FP4 scan): the panel's columns
  // [kFp4Pieces][Ppad][Npad/2] and the projection columns [kFp4Pieces][QCOLS][Npad/2], each with
  // its column scale 2^-e (NaN: no test) and scaled column sum.
  uint8_t* fp4B = nullptr;
  float* fp4B_scale = nullptr;
  float* fp4B_cs = nullptr;
  uint8_t* fp4Q = nullptr;
  float* fp4Q_scale = nullptr;
  float* fp4Q_cs = nullptr;
  CUtensorMap tmFB, tmFQ;
};

struct tg_ctx {
  int device = 0;
  int sm_count = 0;
  cudaStream_t side = nullptr;
  uint32_t* status = nullptr;   // device word (ST_* bits)
  uint32_t* scratch = nullptr;  // small device scratch (rank, flags)
  // decode / projection workspace
  int64_t cap_rows = 0, cap_npad = 0;          // A buffers: rows x npad
  __nv_bfloat16* Ahi = nullptr;                 // centred split operand
  uint8_t* Afp4 = nullptr;                      // E2M1 operand of the FP4 form
  int64_t cap_fp4 = 0;                          // its bytes
  float* A32 = nullptr;
  int64_t cap_m = 0;                            // per-marker arrays
  int32_t* nobs = nullptr;
  double* mean = nullptr;
  float* shift = nullptr;                       // [cap_m] per-row shift of the split operand
  double* gc2s = nullptr;                       // [cap_m] |g_c|^2 over a subset panel's samples
  uint32_t* mh = nullptr;                       // [cap_m] bf16 bits of the missing-call value
  double* gc2 = nullptr;
  int64_t* S = nullptr;                         // sum of a row's observed calls and of their
  int64_t* S2 = nullptr;                        // squares (decode units), from the counting pass
  float* raw = nullptr;                         // raw products, [ranges][columns][rows]
  size_t cap_raw = 0;                           // its floats
  float* rinv = nullptr;
  double* rinv64 = nullptr;
  uint32_t* close = nullptr;                    // bit per marker: close to the covariate span
  // host-streamed scan: a device ring of host_bufs block buffers' bytes (stage_cap allocated)
  uint8_t* stage = nullptr;
  size_t stage_cap = 0;
  int host_bufs = 3;
  tg_hit* dhits = nullptr;
  int64_t dhits_cap = 0;
  unsigned long long* dnhits = nullptr;
  unsigned long long* dbest = nullptr;
  int64_t dbest_cap = 0;
  cudaEvent_t ev_copied = nullptr;
  cudaEvent_t ev_free[tg::kRingEvents] = {};
  // timing of one block's copy (0, 1) and scan (2, 3) in a host-streamed scan, and their ratio
  // (scan time / copy time, 0 = not measured yet), which sets the next call's block ramp
  cudaEvent_t ev_rate[4 * tg::kRateBlocks] = {};
  double ramp_ratio = 0.0;
  double ramp_fixed = 0.0;  // > 0: a fixed growth factor set by the caller
  // profiling
  bool prof = false;
  std::vector<tg::Events> pending;
  std::vector<cudaEvent_t> event_pool;
  double stage_ms[TG_N_STAGES] = {0, 0, 0, 0, 0, 0};
  int64_t launches[TG_N_STAGES] = {0, 0, 0, 0, 0, 0};
  // captured scan graphs that hold pointers into this workspace
  int graphs_alive = 0;
  // split-form scans decode 2-bit / unmasked dosage blocks in the contraction producer
  // (off by default: slower than the decoded operand on GB300, see tg_set_fused_decode)
  bool fuse_decode = false;
  // small panels' joint projection pass reads the packed rows and decodes them in shared memory
  // (on by default: it removes the decoded operand's round trip through HBM)
  bool fuse_joint = true;
  // autotuned kernel per block-size bucket
  int tune_kernel[tg::kTuneBuckets] = {};
  int tune_group[tg::kTuneBuckets] = {};
  int tune_split[tg::kTuneBuckets] = {};        // split-K of the one-CTA kernel (0 = none)
};

namespace tg {

// error reporting and orchestration (api.cu)
tg_status fail(tg_status s, const std::string& msg);
tg_status cuda_fail(cudaError_t e, const char* what);
tg_status check_scan_args(const tg_ctx* c, const tg_panel* p, const ScanArgs& a);
tg_status scan_impl(tg_ctx* c, const tg_panel* p, const ScanArgs& a, cudaStream_t st);
// Degrees of freedom and ln B(df/2, 1/2) of the statistic a scan mode computes.
void mode_df(const tg_panel* p, int mode, double* df, double* lnB);
bool make_tmap(CUtensorMap* m, const void* ptr, int64_t rows, int64_t K, int64_t ld,
               uint32_t box_rows);
// uint8 map over packed genotype rows [rows][ld], boxes of box_bytes x box_rows, zero fill;
// swizzle: boxes of 64 or 128 bytes get the swizzle of that size.
bool make_tmap_packed(CUtensorMap* m, const void* ptr, int64_t rows, int64_t ld, uint32_t box_bytes,
                      uint32_t box_rows = 128, bool swizzle = false);

// Launch a kernel that starts with chain_wait() (device.cuh) so that it may be scheduled while the
// kernel before it on the stream still runs: each boundary between the four or five kernels of a
// small scan cost 1.5 to 2.5 us. Behind anything else it is an ordinary launch.
template <class... P, class... A>
cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, unsigned block, size_t smem,
                           cudaStream_t st, const A&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

// panel kernels (k_panel.cu)
cudaError_t launch_build_design(double* X, const double* C, int64_t ldc, int64_t N, int64_t n_cov,
                                uint32_t* flags, cudaStream_t st);
// X [k][N] is followed by the reflectors and the factorisation's state: householder_doubles(N, k)
// doubles in all.
size_t householder_doubles(int64_t N, int64_t k);
cudaError_t launch_householder(double* X, int64_t N, int64_t k, double* Q, int* rank_out,
                               cudaStream_t st);
cudaError_t launch_residualise(const float* Y, int64_t ldy, const double* Q, int64_t N, int64_t P,
                               int64_t q, int64_t Npad, double* Yres, double* s, float* col_s,
                               float* col_rmul, __nv_bfloat16* Bhi, __nv_bfloat16* Blo, float* B32,
                               float* col_cs, uint32_t* flags, cudaStream_t st);
// The joint operand of a small panel as scaled f16 hi + lo (rows of the q - 1 projection columns,
// then the P phenotypes, zero to `rows`), with its scaled column sums.
cudaError_t launch_joint_f16(const double* Q, int64_t N, int64_t nq, const double* Yres,
                             const double* s, const float* rmul, int64_t P, int64_t rows,
                             int64_t Npad, __half* hi, __half* lo, float* cs, cudaStream_t st);
cudaError_t launch_qcols(const double* Q, int64_t N, int64_t q, int64_t Npad, float* QB,
                         __nv_bfloat16* QBhi, __nv_bfloat16* QBlo, float* qcs, cudaStream_t st);
// subset panels: rows gathered to a compact copy and scattered back (elements of 2, 4 or 8
// bytes), and per-phenotype finite-value masks
cudaError_t launch_gather_f32(const float* src, int64_t lds, float* dst, int64_t ldd, const int* idx,
                              int64_t ns, int64_t R, cudaStream_t st);
cudaError_t launch_gather_f64(const double* src, int64_t lds, double* dst, int64_t ldd,
                              const int* idx, int64_t ns, int64_t R, cudaStream_t st);
cudaError_t launch_scatter(const void* src, int64_t lds, void* dst, int64_t ldd, const int* idx,
                           int64_t ns, int64_t R, int elem_bytes, cudaStream_t st);
cudaError_t launch_pheno_masks(const float* Y, int64_t ldy, int64_t N, int64_t P, uint32_t* masks,
                               int64_t ldm, cudaStream_t st);

// decode (k_decode.cu)
cudaError_t launch_decode(const uint8_t* G, int64_t ldg, int encoding, int64_t N, int64_t M,
                          const uint32_t* missing, int64_t ldm, int precision, void* Ahi,
                          float* shift, uint32_t* mh, int64_t lda, int32_t* nobs, int64_t* S,
                          int64_t* S2, double* mean, double* gc2, cudaStream_t st);
// |g_c|^2 over the samples of a subset panel (decode units; the imputed value is the marker's
// all-sample mean, S / nobs where S is given, else `mean`)
cudaError_t launch_subset_stats(const uint8_t* G, int64_t ldg, int encoding, int64_t N, int64_t M,
                                const uint32_t* missing, int64_t ldm, const uint32_t* samples,
                                const double* mean, const int32_t* nobs, const int64_t* S,
                                double* gc2s, cudaStream_t st);

// The CTA-pair kernel's units (one 256 x bn tile x one accumulation chunk) and their even split over
// the pairs: pair w takes the units [w per, (w + 1) per), tile (m-tile pair t / n_nt, column tile
// t % n_nt) holding the units t chunks .., so at most `pieces` pairs share a tile. chunks may be more
// than the tile has (a multiple of per, so that no pair crosses into another tile).
struct PairUnits {
  int n_nt, chunks, per, pairs, pieces;
};

// Raw products as the contraction kernels leave them (EpiParams::raw_out): element (m, k) of
// range s at x[s * split + k * ld + m]. With `partial` the ranges are partial sums, which are
// added in range order, and then shift[m] * cs[k] * cs_scale. per > 0: the ranges are the pieces of
// a tile of 256 rows and bn columns, as many as the CTAs or pairs that share it (FusedUnits,
// PairUnits), tiles counted over n_nt column tiles; column k here is column col0 + k of the pass.
struct RawView {
  const float* x;
  long long ld, split;
  int ranges;
  bool partial;
  const float* shift;
  const float* cs;
  float cs_scale;
  int per, chunks, n_nt, bn, col0;
  bool sum64;  // k_marker_norm adds the ranges in FP64 (the FP32 form; no add-back)
};
// A block's integer sums, from which k_marker_norm makes the row statistics (nobs, mean, gc2):
// byte sums of dosage rows left by the joint pass in two parts per piece (x, DecodeArgs::sums;
// n_obs = N), or the counting pass's S and S2 with its nobs. Neither: the statistics are there.
struct RowSums {
  const uint32_t* x;
  long long ld;
  int N;
  const int64_t* S;
  const int64_t* S2;
  int32_t* nobs;
  double* mean;
  double* gc2;
};
// The statistics of `sums` on their own, where something reads the means before the norms.
cudaError_t launch_row_statistics(int64_t M, const RowSums& sums, const RawView& raw,
                                  cudaStream_t st);
// SIMT kernels (k_simt.cu)
// Projections of the FP32 operand, column-major: out[k * ldq + m], range r of K `split` floats on.
cudaError_t launch_project(const float* A, int64_t lda, int64_t M, int64_t K, const float* QB,
                           int64_t nq, float* out, int64_t ldq, cudaStream_t st, int ranges = 1,
                           int64_t split = 0);
// What the FP64 re-projection of markers close to the covariate span needs: the packed block,
// the FP64 means (units) and the panel's FP64 basis Q ([q][N], column 0 the intercept).
struct MarkerRefine {
  const uint8_t* G;
  int64_t ldg;
  int encoding;
  int64_t N;
  const uint32_t* missing;
  int64_t ldm;
  const double* mean;
  const double* Q;
  int q;
};
// Outputs of the norm kernel: 1/|g_res| of each marker (NaN = untestable) and, where not NULL,
// |g_res|^2 in allele units, copies of n_obs and of the mean for the caller, and
// the hit counter's value before this block (hit_start[0] = *n_hits, hit_start[1] = 0).
struct NormOut {
  double* norm2_allele;
  float* rinv;
  double* rinv64;
  int32_t* nobs;
  double* mean;
  unsigned long long* hit_start;
  const unsigned long long* n_hits;
  uint32_t* close;  // [ceil(M/32)] bit per marker: re-projected in FP64 (nq > 0)
};
// complete_n > 0: markers with fewer than complete_n observed calls are untestable too.
cudaError_t launch_marker_norm(int64_t M, const int32_t* nobs, const double* gc2,
                               const RawView& proj, int64_t nq, double kappa,
                               const MarkerRefine& refine, const NormOut& out, cudaStream_t st,
                               int64_t complete_n = 0, const RowSums& sums = RowSums{});
cudaError_t launch_sgemm_scan(const float* A, int64_t lda, const float* B, int64_t ldb, int64_t K,
                              const EpiParams& ep, cudaStream_t st);

// statistics after the contraction (k_stats.cu)
cudaError_t launch_full_stats(const EpiParams& ep, cudaStream_t st);
// start: [0] the hit count before the block, [1] a counter, as k_marker_norm leaves them (NormOut).
cudaError_t launch_hit_stats(const EpiParams& ep, unsigned long long* start, cudaStream_t st);
cudaError_t launch_fill_random(uint8_t* p, size_t n, unsigned long long seed, cudaStream_t st);

// tensor-core kernel (k_tc.cu)
// With `dec` non-NULL the A operand is decoded from packed genotypes in the kernel (tmA unused).
// `bn`: columns of a tile, the B maps' box rows: a multiple of 16 up to 128 (the covariate
// projection, a small panel's joint operand, or a panel of at most 64 phenotypes), or 256.
// Raw mode (ep.raw_out) takes split-K.
cudaError_t launch_tc_scan(const CUtensorMap* tmA, const CUtensorMap* tmBhi,
                           const CUtensorMap* tmBlo, int64_t K, const EpiParams& ep, int sm_count,
                           long long spin_ns, cudaStream_t st, int group_m = 16,
                           const DecodeArgs* dec = nullptr, int encoding = 0, int bn = 256);

// The joint projection pass of a small panel (joint operand of at most 128 rows) with the decode
// fused in (k_fused.cu): reads the packed rows through da.tmG, whose boxes must be kFusedRows
// rows of 128 bytes with the 128-byte swizzle (dosage) or 32 bytes (2-bit calls); raw mode only, K
// a multiple of 64, bn (a multiple of 16) the operand's box rows. Writes the raw products as
// fu.pieces partial sums per tile, without the shift's add-back.
constexpr int kFusedRows = 256;
// Its units (one tile x one accumulation chunk) and their even split over the CTAs: CTA w takes the
// units [w per, (w + 1) per), so tile t is shared by the CTAs t chunks / per to
// ((t + 1) chunks - 1) / per, at most `pieces` of them.
struct FusedUnits {
  int chunks, units, per, grid, pieces;
};
// whole: whole tiles only, one piece each.
inline FusedUnits fused_units(int64_t M, int64_t K, int sm_count, bool whole = false) {
  FusedUnits f;
  f.chunks = (int)((K / 32 + kAccumChunkKB - 1) / kAccumChunkKB);
  f.units = (int)((M + kFusedRows - 1) / kFusedRows) * f.chunks;
  const int ctas = f.units < sm_count ? f.units : sm_count;
  f.per = (f.units + ctas - 1) / ctas;
  if (whole) f.per = (f.per + f.chunks - 1) / f.chunks * f.chunks;
  f.grid = (f.units + f.per - 1) / f.per;
  f.pieces = f.per % f.chunks == 0 ? 1 : (f.chunks + f.per - 2) / f.per + 1;
  return f;
}
// f16 (dosage rows): they are expanded into f16 (b - c exact) against the f16 operand (tmBhi / tmBlo
// then map QYhi16 / QYlo16 and the products are scaled back by 2^-14); else, and for 2-bit calls,
// into bf16 against the bf16 operand.
cudaError_t launch_joint_fused(const CUtensorMap* tmBhi, const CUtensorMap* tmBlo, int64_t K,
                               const EpiParams& ep, const FusedUnits& fu, int bn, long long spin_ns,
                               cudaStream_t st, const DecodeArgs& da, int encoding, bool f16);

// The statistics of a block from its raw products (k_stats.cu): the same per-element epilogue as
// the contraction kernels and, in FULL mode, every statistic (no launch_full_stats after it).
cudaError_t launch_raw_stats(const RawView& raw, const EpiParams& ep, cudaStream_t st);

// The FP4 form (k_fp4.cu). Pieces: rows r < nrows of src (stride lds; divided by div[r] when
// div is not NULL; skipped where valid[r] is NaN) as kFp4Pieces E2M1 pieces, out[k][rows_pad][Npad/2]
// bytes, with scale[r] = 2^-e (NaN for a skipped row) and cs[r] = the scaled column sum.
cudaError_t launch_fp4_pieces(const double* src, int64_t lds, const double* div, const float* valid,
                              int64_t nrows, int64_t rows_pad, int64_t N, int64_t Npad, uint8_t* out,
                              float* scale, float* cs, cudaStream_t st);
// The FP4 form's decode of 2-bit rows in one pass: the E2M1 operand [M][lda] bytes (lda =
// Npad / 2, a multiple of 32) and each row's n_obs, FP64 mean, |g_c|^2 and shift = -mean.
cudaError_t launch_fp4_decode(const uint8_t* G, int64_t ldg, int64_t N, int64_t M, uint8_t* A,
                              int64_t lda, int32_t* nobs, double* mean, double* gc2, float* shift,
                              cudaStream_t st);
// The contraction: tmA over the E2M1 operand (boxes of 64 bytes x 128 rows, 64-byte swizzle),
// tmB over kFp4Pieces x b_rows_pad piece rows (boxes of 64 bytes x 128 rows, or 64 rows in raw
// mode: the covariate projection, at most 64 columns).
cudaError_t launch_fp4_scan(const CUtensorMap* tmA, const CUtensorMap* tmB, int b_rows_pad,
                            int64_t Npad, const EpiParams& ep, int sm_count, long long spin_ns,
                            cudaStream_t st);

// tensor-core kernel on CTA pairs, 256 x bn tiles (k_tc2.cu); bn a multiple of 32, at most 256,
// the B maps with boxes of bn / 2 rows. Raw mode (ep.raw_out) takes an even split of its units.
cudaError_t launch_tc2_scan(const CUtensorMap* tmA, const CUtensorMap* tmBhi,
                            const CUtensorMap* tmBlo, int64_t K, const EpiParams& ep, int sm_count,
                            long long spin_ns, cudaStream_t st, int group_m = 16,
                            const DecodeArgs* dec = nullptr, int encoding = 0, int bn = 256,
                            const PairUnits* pu = nullptr);

// bounded wait test (k_tc.cu)
cudaError_t launch_wait_test(const uint32_t* flag, long long limit_ns, uint32_t* result,
                             cudaStream_t st);

// p-value helpers on the host (pvalue.cuh)
double host_lnbeta_half(double df);
double host_r2_threshold(double mlog10p, double df, double lnB);

}  // namespace tg
