// Projection (and small-panel) pass with the genotype decode fused into it (Section 2.2: the
// covariate projection of each marker and Eq. 2 for a panel of P <= 128 - (q - 1) phenotypes,
// read from the packed genotype block in one pass; Section 2.4: the scan is bound by the bytes it
// reads).
//
// For a small panel the whole scan is one pass over the block: the joint B operand holds the
// q - 1 covariate projection columns and the P phenotype columns (64 or 128 rows), so a single
// contraction gives both Q^T a and the panel's products. With the decoded operand in HBM that
// pass reads 2 bytes per sample and marker after the decode wrote them; here it reads the packed
// rows instead (1 byte per sample for dosages, 1/4 for 2-bit calls) and expands them on the way
// into tensor memory, which removes the operand's round trip through HBM.
//
// Tiles of 256 markers (two 128-row sub-tiles sharing every B stage). The work is cut into units
// of one tile x one accumulation chunk (1,024 samples), and each CTA takes the same number of
// consecutive units, so a tile may be shared by two CTAs (more when there are fewer tiles than
// SMs): no SM waits for the last wave (65,536 markers are 256 tiles on 152 SMs, 1.68 waves that
// cost 2), and small blocks fill the chip too. Each CTA writes its part of a tile as one piece
// of partial sums; the kernels that read them add a tile's pieces in order.
//
// Persistent kernel, one CTA per SM, 640 threads:
//   warp 0 lane 0  TMA producer: the packed rows of each stage (four K blocks, 128 samples: a box
//                  of 128 bytes per row with the 128-byte swizzle for dosages, 32 bytes for 2-bit
//                  calls; 256 rows) into a ring of its own, kept PS - 1 stages ahead of the
//                  decoders, and the joint B operand's hi and lo rows for each stage into the B
//                  ring (bn rows: the columns rounded up to 16, not the 64 or 128 of the tile)
//   warps 1, 2     MMA issuers (one elected lane), one per sub-tile: per stage 4 K blocks x 2 k-steps
//                  x 2 products (hi, lo) of tcgen05.mma 128 x bn x 16 with A read from tensor
//                  memory, a fresh accumulator per 1,024 samples as in k_tc_scan
//   warps 4..19    decoders, then epilogue. A warp has 32 rows of a sub-tile and two of the stage's
//                  K blocks: each stage it expands its rows' 64 samples from the packed slot
//                  (genotype.cuh: code - c exactly, bf16(mean - c) for a missing call, 0 past N)
//                  and writes them with tcgen05.st straight into the stage's A columns of tensor
//                  memory. It drains each chunk (tcgen05.ld) into FP32 totals of its half of the
//                  columns a few stages into the next one.
// What bounds it is the decoders' chain of waits, loads, expansion and tcgen05.st per stage, so
// they are as many as the registers allow. With 8 warps (a row's whole 64 samples per thread)
// the schedulers issued in 44% of the cycles (2.5 eligible warps short of one) and a stage took
// 1,417 cycles with 64 columns (dosages) and 1,937 with 128 columns (2-bit calls, A then in shared
// memory), against 700 for the dosage bytes from HBM and 1,024 for the products.
// The projection of a larger panel (P + q - 1 > 512) runs as the same pass with the 64
// projection columns alone; there the decoders also write the block's bf16 operand for the
// panel's contraction as they expand each stage (staged per warp in shared memory so that each
// store instruction writes whole 64-byte row segments). The operand is then written once and
// read once, by the contraction, and the projection reads the packed rows instead of it.
// Dosage rows without a counting pass (one pass, DecodeArgs::sums): a row's shift is the rounded
// mean of its first 64 bytes, and each thread sums the bytes it expands and their squares;
// k_marker_norm makes the row's statistics from the parts.
// TMEM: accumulators of 2 x 64 or 2 x 128 columns from column 0 (two alternating, or one, which
// the products then wait ~2% of the time for), two A stages of 128 columns (two sub-tiles, two
// 16-bit values per column) from column 256.
// Every wait is bounded: past the limit the kernel latches ST_TIMEOUT, raises a shared abort
// flag, lets in-flight copies and products finish (again bounded), frees its TMEM and returns.
#include <cuda.h>
#include <cuda_bf16.h>

#include <type_traits>

#include "device.cuh"
#include "internal.h"
#include "tc_common.cuh"

namespace tg {
namespace {

using namespace tcx;

// 16 decoder warps and 4 others: 640 threads, 96 registers each at launch. Warpgroup 0 (producer,
// MMA issuers, an idle warp) gives back down to 40 and the decoders take 104:
// 128 x 40 + 512 x 104 = 58,368, within the launch total of 61,440.
constexpr int kDecWarps = 16;
constexpr int kFThreads = 128 + 32 * kDecWarps;
constexpr int kLaunchRegs = 96, kFLow = 40, kFHigh = 104;
static_assert(128 * kFLow + 32 * kDecWarps * kFHigh <= kFThreads * kLaunchRegs, "register split");
static_assert(kFThreads * kLaunchRegs <= 65536, "registers at launch");

// Packed rows and the form they are expanded to: 2-bit calls to bf16, dosage bytes to bf16 or f16.
// The f16 form takes 2 instructions per pair of samples (bf16: 5), but its products have more
// bits below the accumulator's last one, which the tensor core drops toward zero: |t| comes out
// low by 1.85e-6 against 1.35e-6 (8,192 markers x 23,000 samples). The caller chooses it for large
// blocks (internal.h).
enum { F_2BIT = 0, F_U8_BF16 = 1, F_U8_F16 = 2 };

// K blocks per stage: 128 samples. The decoders' waits, votes, fences and arrivals cost about as
// much per stage as expanding 32 samples does, so a stage gives each decoder 64.
constexpr int kStageKB = 4;

template <int OPA, int BR>
struct FCfg {
  static constexpr int kRows = kFusedRows;                         // tile rows
  static constexpr int kBoxP = OPA != F_2BIT ? 128 : 32;           // packed bytes per row per stage
  static constexpr int kPackBytes = kRows * kBoxP;                 // one packed slot
  static constexpr int kBk = BR * TBK * 2;                         // one K block of B rows
  static constexpr int kStageBytes = 2 * kStageKB * kBk;           // Bhi, Blo of the K blocks
  static constexpr int kPS = OPA == F_2BIT ? 6 : BR == 128 ? 3 : 4;  // packed ring slots
  static constexpr int kStages = 2;                                // B ring slots = A stages in TMEM
  static constexpr int kAccCols = 2 * BR;                          // both sub-tiles
  static constexpr int kNAcc = 256 / kAccCols;                     // chunk accumulators
  // stages of the next chunk that the decoders expand before they drain a chunk: with one
  // accumulator fewer than the ring holds (the products wait for the drain), with two enough
  // for the chunk to be complete by then
  static constexpr int kLag = kNAcc == 1 ? 1 : 3;
  static constexpr int kAccKB = kChunkKB;  // K blocks per accumulator: 1,024 samples, as in k_tc_scan
  static constexpr int kACol = 256;
  static constexpr int kAStageCols = 32 * kStageKB;
  static_assert(kNAcc * kAccCols <= kACol && kACol + kStages * kAStageCols <= kTmemCols, "TMEM");
  static_assert(kNAcc > 1 || kLag < kStages, "a drain the products wait for comes within the ring");
  static constexpr int kBarBytes = 256;
  // the operand write (64-column pass): each decoder warp stages its 32 rows x 64 bytes
  static constexpr int kStgWarp = 32 * 64;
  static constexpr int kStgBytes = BR == 64 ? kDecWarps * kStgWarp : 0;
  static constexpr int kSmem =
      kStages * kStageBytes + kPS * kPackBytes + kBarBytes + kStgBytes + 1024;
  static_assert(kSmem <= 227 * 1024, "shared memory");
};

// The units [u, u1) of a CTA, stage by stage: a unit is chunk u % ch of tile u / ch; consecutive
// units of one tile form an item (the K blocks [kb_lo, kb_hi) of the tile).
struct Items {
  int u, u1, ch, num_kb;
  int tile, kb_lo, kb_hi;
  __device__ __forceinline__ Items(int per, int units, int ch_, int num_kb_)
      : u((int)blockIdx.x * per), u1(min(units, ((int)blockIdx.x + 1) * per)), ch(ch_),
        num_kb(num_kb_), tile(0), kb_lo(0), kb_hi(0) {}
  __device__ __forceinline__ bool next() {
    if (u >= u1) return false;
    tile = u / ch;
    const int c = u - tile * ch, n = min(ch - c, u1 - u);
    kb_lo = c * kChunkKB;
    kb_hi = min(num_kb, (c + n) * kChunkKB);
    u += n;
    return true;
  }
};

// 16 dosage bytes v minus the row's shift c as f16 pairs, exactly: byte b placed under the f16
// exponent of 1024 is the f16 value 1024 + b (bits 0x6400 | b, one byte permute per pair), and
// one f16x2 subtraction of 1024 + c (c an integer in [0, 255]) leaves b - c, exact in f16.
__device__ __forceinline__ void split16_u8_f16(uint4 v, uint32_t c2, uint32_t* o) {
  const uint32_t w4[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int p = 0; p < 8; ++p) {
    const uint32_t h = __byte_perm(w4[p >> 1], 0x64646464u, (p & 1) ? 0x4342u : 0x4140u);
    asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(o[p]) : "r"(h), "r"(c2));
  }
}

// Zero the 16-bit values of samples >= N among the 16 starting at i0 (8 words).
__device__ __forceinline__ void zero_tail16p(uint32_t* o, int i0, int N) {
#pragma unroll
  for (int p = 0; p < 8; ++p) {
    const int i = i0 + 2 * p;
    if (i >= N) o[p] = 0u;
    else if (i + 1 >= N) o[p] &= 0xFFFFu;
  }
}

__device__ __forceinline__ void tc_st16(uint32_t taddr, const uint32_t* v) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, "
      "%12, %13, %14, %15, %16};" ::"r"(taddr),
      "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
      "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
      : "memory");
}

// 16 consecutive FP32 columns of this thread's TMEM lane.
__device__ __forceinline__ void tc_ld16(uint32_t taddr, float v[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, "
      "%12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// A from tensor memory: D (+)= A[a_tmem] B[b_desc]^T.
__device__ __forceinline__ void tc_mma_ta(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc,
                                          uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
      "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// Sum and sum of squares of 16 dosage bytes whose first sample is i0, the samples >= N left out
// (past N the packed row holds the caller's padding).
__device__ __forceinline__ void sums16_u8(uint4 v, int i0, int N, uint32_t& s, uint32_t& s2) {
  const uint32_t w4[4] = {v.x, v.y, v.z, v.w};
  if (i0 + 16 <= N) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      s = __dp4a(w4[q], 0x01010101u, s);
      s2 = __dp4a(w4[q], w4[q], s2);
    }
  } else {
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const uint32_t u = (w4[q] >> (8 * b)) & 0xFFu;
        if (i0 + 4 * q + b < N) {
          s += u;
          s2 += u * u;
        }
      }
  }
}

// A dosage row's shift without its mean: the rounded mean of its first min(N, 64) bytes. Any
// integer shift leaves b - c exact in f16; one near the row's mean keeps the partial sums of the
// products small, as the full mean does.
__device__ __forceinline__ uint32_t first_bytes_shift_u8(const uint8_t* row, int N) {
  uint32_t s = 0, s2 = 0;
#pragma unroll 1
  for (int g = 0; g < 4 && 16 * g < N; ++g)
    sums16_u8(reinterpret_cast<const uint4*>(row)[g], 16 * g, N, s, s2);
  const int n = N < 64 ? N : 64;
  const int c = (int)rintf((float)s / (float)n);
  return (uint32_t)(c < 0 ? 0 : c > 255 ? 255 : c);
}

// Expand 32 samples (K block q of a stage, the first one sample i0) of tile row r from the packed
// slot into o (two 16-bit values per word): 2-bit calls as bf16 (k = the row's lookup pair), dosage
// bytes as f16 (k.x = the f16 pair of 1024 + c) or bf16 (k.x = the float 2^23 + c). Dosage slots
// carry the TMA's 128-byte swizzle (16-byte chunk j of row r at r * 128 + 16 * (j ^ (r & 7))), so
// the 8 threads of a quarter warp, 8 consecutive rows, read 8 distinct bank groups. With `sum`
// (f16), dosage bytes are also added into s and s2 (their sum and sum of squares, samples < N only).
template <int OPA>
__device__ __forceinline__ void expand32(uint32_t slot, int r, int q, uint2 k, bool row_ok,
                                         int i0, int N, bool sum, uint32_t (&o)[16], uint32_t& s,
                                         uint32_t& s2) {
  if (OPA == F_2BIT) {
    uint32_t w[2];
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];"
                 : "=r"(w[0]), "=r"(w[1])
                 : "r"(slot + (uint32_t)(r * 32 + q * 8)));
#pragma unroll
    for (int g = 0; g < 2; ++g)
      split16_2bit(w[g], k.x, k.y, *reinterpret_cast<uint32_t(*)[8]>(o + 8 * g));
  } else {
    const uint32_t sw = (uint32_t)(r & 7);
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      uint4 v;
      asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                   : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                   : "r"(slot + (uint32_t)(r * 128) + ((((uint32_t)(2 * q + g)) ^ sw) << 4)));
      if (OPA == F_U8_F16) {
        split16_u8_f16(v, k.x, o + 8 * g);
        if (sum) sums16_u8(v, i0 + 16 * g, N, s, s2);
      } else {
        split16_u8(v, __uint_as_float(k.x), 0u, 0u, *reinterpret_cast<uint32_t(*)[8]>(o + 8 * g));
      }
    }
  }
  if (!row_ok) {
#pragma unroll
    for (int p = 0; p < 16; ++p) o[p] = 0u;
  } else if (i0 + 32 > N) {
    zero_tail16p(o, i0, N);
    zero_tail16p(o + 8, i0 + 16, N);
  }
}

// Write one K block of a stage to the block's bf16 operand from the expanded rows of one decoder
// warp: lane l holds 32 samples of row l of the warp's 32 (16 words, two 16-bit values each). The
// rows go through the warp's staging area in shared memory (`stg`, 32 rows of 64 bytes; 16-byte
// chunk c of row l at chunk c ^ ((l >> 1) & 3), which keeps each quarter warp on distinct banks
// both ways), then each store instruction writes 8 rows of 64 bytes, whole segments, instead of
// 32 scattered 16-byte pieces. Row l goes to dst0 + l * ld (16-byte aligned); rows at or past
// `rows` are skipped. The bf16 forms' values go out as they are; the f16 form's are b - c,
// integers of magnitude at most 255 (or 0 past N), which bf16 holds exactly, so the conversion
// through f32 is exact and gives the decoded operand's values.
template <int OPA>
__device__ __forceinline__ void store_operand_warp(uint32_t stg, const uint32_t (&o)[16], int lane,
                                                   __nv_bfloat16* dst0, long long ld, int rows) {
  __syncwarp();  // the previous stage's staged rows have been read
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      uint32_t x = o[4 * c + i];
      if (OPA == F_U8_F16) {
        __half2 h;
        memcpy(&h, &x, 4);
        const __nv_bfloat162 b = __float22bfloat162_rn(__half22float2(h));
        memcpy(&x, &b, 4);
      }
      w[i] = x;
    }
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(
                     stg + (uint32_t)(lane * 64 + ((c ^ ((lane >> 1) & 3)) << 4))),
                 "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3])
                 : "memory");
  }
  __syncwarp();
  const int cc = lane & 3;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = i * 8 + (lane >> 2);
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "r"(stg + (uint32_t)(r * 64 + ((cc ^ ((r >> 1) & 3)) << 4))));
    if (r < rows) *reinterpret_cast<uint4*>(dst0 + r * ld + cc * 8) = v;
  }
}

template <int OPA, int BR>
__global__ void __launch_bounds__(kFThreads, 1)
    k_joint_fused(const __grid_constant__ CUtensorMap tmBhi, const __grid_constant__ CUtensorMap tmBlo,
                  int num_kb, int chunks, int per, int units, int bn, long long spin_ns,
                  const __grid_constant__ EpiParams ep, const __grid_constant__ DecodeArgs da) {
  using C = FCfg<OPA, BR>;
  constexpr int S = C::kStages, PS = C::kPS;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* gbase = smem_raw + (base - raw);
  const uint32_t pk_base = base + S * C::kStageBytes;
  const uint32_t bars = pk_base + PS * C::kPackBytes;
  auto full_bar = [&](int s) { return bars + 8u * s; };
  auto empty_bar = [&](int s) { return bars + 8u * (S + s); };
  auto pfull_bar = [&](int p) { return bars + 8u * (2 * S + p); };
  auto pempty_bar = [&](int p) { return bars + 8u * (2 * S + PS + p); };
  auto cfull_bar = [&](int a) { return bars + 8u * (2 * S + 2 * PS + a); };
  auto cempty_bar = [&](int a) { return bars + 8u * (2 * S + 2 * PS + 2 + a); };
  const uint32_t drain_bar = bars + 8u * (2 * S + 2 * PS + 4);
  uint32_t* tmem_slot =
      reinterpret_cast<uint32_t*>(gbase + (bars - base) + 8 * (2 * S + 2 * PS + 5));
  static_assert(8 * (2 * S + 2 * PS + 5) + 8 <= C::kBarBytes, "barrier area");
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const uint32_t stg_base = bars + C::kBarBytes;  // the operand write's staging rows

  auto sBhi = [&](int s, int h) { return base + (uint32_t)(s * C::kStageBytes + h * C::kBk); };
  auto sBlo = [&](int s, int h) {
    return base + (uint32_t)(s * C::kStageBytes + (kStageKB + h) * C::kBk);
  };
  auto sPk = [&](int p) { return pk_base + (uint32_t)(p * C::kPackBytes); };
  // accumulator of the CTA's g-th chunk, and the parity of its use
  auto acc_of = [](uint32_t g) { return (int)(g % C::kNAcc); };
  auto use_of = [](uint32_t g) { return (g / C::kNAcc) & 1u; };

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(full_bar(s), 1 + kDecWarps);  // the producer's B bytes + one arrival per decoder warp
      mbar_init(empty_bar(s), 2);  // both issuers' products have read the stage
    }
    for (int p = 0; p < PS; ++p) {
      mbar_init(pfull_bar(p), 1);
      mbar_init(pempty_bar(p), kDecWarps);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(cfull_bar(a), 2);
      mbar_init(cempty_bar(a), kDecWarps);
    }
    mbar_init(drain_bar, 2);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *reinterpret_cast<volatile uint32_t*>(tmem_slot);
  chain_wait();
  Items it(per, units, chunks, num_kb);

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kFLow));
    if (warp == 0 && lane == 0) {
      // ---------------------------------------------------------- TMA producer
      // the packed rows run PS - 1 stages ahead of the B rows, over the same sequence
      Items pk = it;
      int jp = 0, j = 0;       // stages whose packed rows, B rows were requested
      int pkb = 0;             // next K block of pk's item
      bool more = pk.next();
      pkb = pk.kb_lo;
      auto load_packed = [&]() -> bool {
        if (!more) return true;
        const int p = jp % PS;
        if (!mbar_wait(pempty_bar(p), (uint32_t)((jp / PS) & 1) ^ 1u, abort_flag, spin_ns, ep.status))
          return false;
        mbar_expect_tx(pfull_bar(p), (uint32_t)C::kPackBytes);
        tma_load_2d(&da.tmG, sPk(p), pfull_bar(p), (pkb / kStageKB) * C::kBoxP, pk.tile * C::kRows);
        ++jp;
        pkb += kStageKB;
        if (pkb >= pk.kb_hi) {
          more = pk.next();
          pkb = pk.kb_lo;
        }
        return true;
      };
      bool ok = true;
      for (int i = 0; i < PS - 1 && ok; ++i) ok = load_packed();
      while (ok && it.next()) {
        for (int kb = it.kb_lo; kb < it.kb_hi; kb += kStageKB) {
          const int s = j % S;
          if (!load_packed() ||
              !mbar_wait(empty_bar(s), (uint32_t)((j / S) & 1) ^ 1u, abort_flag, spin_ns, ep.status)) {
            ok = false;
            break;
          }
          mbar_expect_tx(full_bar(s), (uint32_t)(2 * kStageKB * bn * TBK * 2));
#pragma unroll
          for (int h = 0; h < kStageKB; ++h) {  // (a K block past the operand's end reads zeros)
            tma_load_2d(&tmBhi, sBhi(s, h), full_bar(s), (kb + h) * TBK, 0);
            tma_load_2d(&tmBlo, sBlo(s, h), full_bar(s), (kb + h) * TBK, 0);
          }
          ++j;
        }
      }
      // copies still in flight land before the CTA leaves (bounded)
      for (int i = j - S > 0 ? j - S : 0; i < j; ++i)
        mbar_wait(full_bar(i % S), (uint32_t)((i / S) & 1), abort_flag, spin_ns, ep.status);
      for (int i = jp - PS > 0 ? jp - PS : 0; i < jp; ++i)
        mbar_wait(pfull_bar(i % PS), (uint32_t)((i / PS) & 1), abort_flag, spin_ns, ep.status);
    } else if (warp == 1 || warp == 2) {
      // ---------------------------------------------------------- MMA issuers (A from TMEM)
      // one warp per sub-tile; A and B both bf16, or both f16 (the scaled f16 operand)
      const int sub = warp - 1;
      const bool lead = elect_one();
      const uint32_t idesc = OPA == F_U8_F16 ? idesc_f16(bn) : idesc_bf16(bn);
      // of stage 0: B_hi's first K block and k-step (the others a fixed number of 16-byte units
      // further on) and the sub-tile's A columns
      const uint64_t desc0 = sdesc_sw64(sBhi(0, 0));
      const uint32_t a0 = tmem_base + (uint32_t)(C::kACol + sub * 16 * kStageKB);
      uint32_t g = 0;
      int s = 0;
      uint32_t phase = 0;
      bool ok = true;
      while (ok && it.next()) {
        for (int kb0 = it.kb_lo; kb0 < it.kb_hi && ok; kb0 += C::kAccKB, ++g) {
          const int acc = acc_of(g);
          if (!mbar_wait_warp(cempty_bar(acc), use_of(g) ^ 1u, abort_flag, spin_ns, ep.status)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t d = tmem_base + (uint32_t)(acc * C::kAccCols + sub * BR);
          const int kb1 = min(kb0 + C::kAccKB, it.kb_hi);
          for (int kb = kb0; kb < kb1; kb += kStageKB) {
            if (!mbar_wait_warp(full_bar(s), phase, abort_flag, spin_ns, ep.status)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint64_t bs = desc0 + (uint64_t)(s * (C::kStageBytes >> 4));
            const uint32_t as = a0 + (uint32_t)(s * C::kAStageCols);
#pragma unroll
            for (int h = 0; h < kStageKB; ++h)
#pragma unroll
              for (int k = 0; k < TBK / 16; ++k) {
                // 16 samples = 8 columns of the sub-tile's 64 (K block h, k-step k)
                const uint32_t a = as + (uint32_t)(h * 16 + k * 8);
                const uint64_t bh = bs + (uint64_t)((h * C::kBk + 32 * k) >> 4);
                if (lead) {
                  tc_mma_ta(d, a, bh, idesc, (kb > kb0 || h > 0 || k > 0) ? 1u : 0u);
                  tc_mma_ta(d, a, bh + (uint64_t)((kStageKB * C::kBk) >> 4), idesc, 1u);
                }
              }
            if (lead) tc_commit(empty_bar(s));
            if (++s == S) {
              s = 0;
              phase ^= 1u;
            }
          }
          if (ok && lead) tc_commit(cfull_bar(acc));
        }
      }
      if (lead) tc_commit(drain_bar);
      __syncwarp();
      mbar_wait_warp(drain_bar, 0u, abort_flag, spin_ns, ep.status);
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kFHigh));
    // ------------------------------------------------------------ decoders, then epilogue
    // 32 rows (TMEM lanes quarter * 32 ..) of sub-tile `sub`, half `part` of each stage's K blocks,
    // columns part * BR / 2 .. of the accumulators
    const int quarter = warp & 3, sub = (warp - 4) >> 3, part = ((warp - 4) >> 2) & 1;
    const int trow = sub * 128 + quarter * 32 + lane;
    const uint32_t lane_addr = tmem_base + ((uint32_t)(quarter * 32) << 16);
    constexpr int NC = BR / 2;
    // dosage rows with the statistics taken here (no counting pass)
    const bool one_pass = OPA == F_U8_F16 && da.sums != nullptr;
    uint32_t g = 0;
    int s = 0, p = 0;  // ring slots of the stage and of its packed rows, and their phases
    uint32_t sph = 1, pph = 0;
    bool ok = true;
    while (ok && it.next()) {
      const long long row = (long long)it.tile * C::kRows + trow;
      const bool row_ok = row < ep.M;
      uint32_t c_row = 0;
      uint2 kc = make_uint2(0u, 0u);
      if (OPA != F_U8_F16) {
        kc = dec_row_consts<OPA == F_2BIT ? OPA_2BIT : OPA_U8>(da, row);
      } else {  // the f16 pair of 1024 + c (c = the row's integer shift)
        if (row_ok)
          c_row = one_pass ? first_bytes_shift_u8(da.G + row * da.ldg, da.N) : (uint32_t)da.shift[row];
        const uint32_t c16 = 0x6400u + c_row;
        kc = make_uint2(c16 | (c16 << 16), 0u);
      }
      uint32_t sum1 = 0, sum2 = 0;  // bytes and their squares (dosage; N <= 66,051)
      float tot[NC];
#pragma unroll
      for (int e = 0; e < NC; ++e) tot[e] = 0.0f;
      auto drain = [&](uint32_t c) -> bool {
        const int acc = acc_of(c);
        if (!mbar_wait_warp(cfull_bar(acc), use_of(c), abort_flag, spin_ns, ep.status)) return false;
        tc_fence_after();
        const uint32_t taddr = lane_addr + (uint32_t)(acc * C::kAccCols + sub * BR + part * NC);
#pragma unroll
        for (int i = 0; i < NC / 16; ++i) {
          if (part * NC + i * 16 >= bn) break;  // columns past the operand's
          float v[16];
          __syncwarp();
          tc_ld16(taddr + (uint32_t)(i * 16), v);
#pragma unroll
          for (int e = 0; e < 16; ++e) tot[i * 16 + e] += v[e];
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(cempty_bar(acc));
        return true;
      };
      bool behind = false;  // the chunk before this one is not drained yet
      for (int kb0 = it.kb_lo; kb0 < it.kb_hi && ok; kb0 += C::kAccKB, ++g) {
        const int kb1 = min(kb0 + C::kAccKB, it.kb_hi);
        for (int kb = kb0; kb < kb1; kb += kStageKB) {
          if (behind && kb == kb0 + kStageKB * C::kLag) {
            if (!drain(g - 1)) {
              ok = false;
              break;
            }
            behind = false;
          }
          // one answer for all lanes: nobody leaves the others at a warp-wide instruction
          ok = mbar_wait(pfull_bar(p), pph, abort_flag, spin_ns, ep.status) &&
               mbar_wait(empty_bar(s), sph, abort_flag, spin_ns, ep.status);
          ok = __all_sync(0xffffffffu, ok) != 0;
          if (!ok) break;
          tc_fence_after();  // the products that read this A stage have completed
          const uint32_t a_st = lane_addr + (uint32_t)(C::kACol + s * C::kAStageCols +
                                                       (sub * kStageKB + part * 2) * 16);
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int q = part * 2 + h;  // K block of the stage
            uint32_t o[16];
            expand32<OPA>(sPk(p), trow, q, kc, row_ok, (kb + q) * TBK, da.N, one_pass, o, sum1, sum2);
            if (h == 1) {
              __syncwarp();
              if (lane == 0) mbar_arrive(pempty_bar(p));  // the packed slot is read
            }
            tc_st16(a_st + 16u * h, o);
            // the projection pass of a larger panel: the expanded rows are also the block's operand
            if (BR == 64 && da.a_out != nullptr && kb + q < num_kb) {
              const long long row0 = row - lane;  // the warp's first row
              const int rows = ep.M - row0 < 32 ? (int)(ep.M - row0) : 32;
              store_operand_warp<OPA>(stg_base + (uint32_t)((warp - 4) * C::kStgWarp), o, lane,
                                      da.a_out + row0 * da.lda_out + (long long)(kb + q) * TBK,
                                      da.lda_out, rows);
            }
          }
          asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(full_bar(s));
          if (++s == S) {
            s = 0;
            sph ^= 1u;
          }
          if (++p == PS) {
            p = 0;
            pph ^= 1u;
          }
        }
        if (ok && behind) ok = drain(g - 1);
        behind = true;
      }
      if (!ok || !drain(g - 1)) {  // the item's last chunk
        ok = false;
        break;
      }
      if (row_ok) {
        // the CTA's piece of the tile: which of the CTAs that share it this one is
        const int piece = (int)blockIdx.x - it.tile * chunks / per;
        if (one_pass) {
          uint32_t* sm = da.sums + (long long)(piece * 2 + part) * 2 * da.sums_ld + row;
          sm[0] = sum1;
          sm[da.sums_ld] = sum2;
          if (part == 0 && it.kb_lo == 0) da.shift_out[row] = (float)c_row;
        }
        // raw products: the first raw_cols columns, without the shift's add-back; the f16 joint
        // operand holds 2^14 v (an exact power of two to take back)
        constexpr float kUnscale = OPA == F_U8_F16 ? (float)(1.0 / kJointF16Scale) : 1.0f;
        float* out = ep.raw_out + (long long)piece * ep.raw_split + row;
  #pragma unroll
        for (int e = 0; e < NC; ++e) {
          const int col = part * NC + e;
          if (col < ep.raw_cols) out[col * ep.raw_ld] = tot[e] * kUnscale;
        }
      }
      __syncwarp();
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) {
    __syncwarp();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base),
                 "r"(kTmemCols)
                 : "memory");
  }
}

template <int OPA, int BR>
cudaError_t go_fused(const CUtensorMap* bh, const CUtensorMap* bl, int64_t K, const EpiParams& ep,
                     const FusedUnits& fu, int bn, long long spin_ns, cudaStream_t st,
                     const DecodeArgs& da) {
  using C = FCfg<OPA, BR>;
  static bool attr_set = false;  // per process and instantiation
  if (!attr_set) {
    cudaError_t e = cudaFuncSetAttribute(k_joint_fused<OPA, BR>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmem);
    if (e != cudaSuccess) return e;
    attr_set = true;
  }
  return launch_chained(k_joint_fused<OPA, BR>, dim3(fu.grid), kFThreads, C::kSmem, st,
      *bh, *bl, (int)(K / TBK), fu.chunks, fu.per, fu.units, bn, spin_ns, ep, da);
}

}  // namespace

cudaError_t launch_joint_fused(const CUtensorMap* tmBhi, const CUtensorMap* tmBlo, int64_t K,
                               const EpiParams& ep, const FusedUnits& fu, int bn, long long spin_ns,
                               cudaStream_t st, const DecodeArgs& da, int encoding, bool f16) {
  if (ep.M == 0 || ep.P == 0) return cudaSuccess;
  // raw mode only (the projection, alone or joint with a small panel), an even number of K
  // blocks, packed rows of the block's M
  if (!ep.raw_out || bn % 16 || bn < 16 || bn > 128 || ep.raw_cols > bn || ep.P != ep.raw_cols ||
      K % (2 * TBK) || da.M != ep.M || ep.ksplit > 1)
    return cudaErrorInvalidValue;
  if (da.sums && (!f16 || da.N > kOnePassMaxN || !da.G || !da.shift_out)) return cudaErrorInvalidValue;
  // the operand write: the 64-column pass, every column of a row in 16-byte stores
  if (da.a_out && (bn > 64 || da.lda_out < K || da.lda_out % 8 ||
                   reinterpret_cast<uintptr_t>(da.a_out) % 16))
    return cudaErrorInvalidValue;
  const auto go = [&](auto form) {
    constexpr int F = decltype(form)::value;
    return bn <= 64 ? go_fused<F, 64>(tmBhi, tmBlo, K, ep, fu, bn, spin_ns, st, da)
                    : go_fused<F, 128>(tmBhi, tmBlo, K, ep, fu, bn, spin_ns, st, da);
  };
  if (encoding == TG_ENC_2BIT) return f16 ? cudaErrorInvalidValue : go(std::integral_constant<int, F_2BIT>());
  return f16 ? go(std::integral_constant<int, F_U8_F16>()) : go(std::integral_constant<int, F_U8_BF16>());
}

}  // namespace tg
