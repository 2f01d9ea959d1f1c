// Conversion of packed genotype codes to the centred split (bf16) operand, shared by the
// decode kernels and the contraction kernels that decode in their producer.
//
// The split operand holds code - c for an observed call (c: the row's shift, a multiple of
// 1/128 for 2-bit calls or an integer for dosage bytes, so the difference is exact in bf16)
// and bf16(mean - c) for a missing call; samples past N are 0.
#pragma once

#include <cuda_bf16.h>
#include <stdint.h>

namespace tg {

// 16 split-form values of 2-bit fields w (sample 16t + k in bits 2k..2k+1): eight bf16x2
// words. lut0 = {field 00, field 01} and lut1 = {field 10, field 11} as bf16 pairs; the byte
// permute's selector byte of field f is 0x10 + 0x22 f (bytes 2f and 2f + 1 of the table).
// The word is taken as a 4 x 4 matrix of fields (row = byte) and transposed with two masked swaps,
// so that samples 4j .. 4j + 3 sit in field j of the four bytes; one multiply-add then makes
// the selectors of four samples: 31 instructions for 16 samples, against 48 with a selector
// built per pair of fields.
__device__ __forceinline__ void split16_2bit(uint32_t w, uint32_t lut0, uint32_t lut1,
                                             uint32_t (&o)[8]) {
  uint32_t t = (w ^ (w >> 6)) & 0x00CC00CCu;
  w ^= t ^ (t << 6);
  t = (w ^ (w >> 12)) & 0x0000F0F0u;
  w ^= t ^ (t << 12);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const uint32_t sel = ((w >> (2 * j)) & 0x03030303u) * 0x22u + 0x10101010u;
    o[2 * j] = __byte_perm(lut0, lut1, sel);
    o[2 * j + 1] = __byte_perm(lut0, lut1, sel >> 16);
  }
}

// 16 split-form values of dosage bytes v: b - c exactly, bf16x2 words; bits of `miss` take
// the missing value mh (a bf16 in the low half of mh2 and in the high half).
__device__ __forceinline__ void split16_u8(uint4 v, float c_plus, uint32_t miss, uint32_t mh2,
                                           uint32_t (&o)[8]) {
  const uint32_t w4[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int p = 0; p < 8; ++p) {
    const uint32_t w = w4[p >> 1];
    const uint32_t k = (uint32_t)(p & 1) * 2u;
    const float a = __uint_as_float(__byte_perm(w, 0x4B000000u, 0x7440u + k)) - c_plus;
    const float b = __uint_as_float(__byte_perm(w, 0x4B000000u, 0x7441u + k)) - c_plus;
    __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    uint32_t r = *reinterpret_cast<uint32_t*>(&h);
    const uint32_t m = (miss >> (2 * p)) & 3u;
    if (m) r = __byte_perm(r, mh2, (m & 1u ? 0x0054u : 0x0010u) | (m & 2u ? 0x7600u : 0x3200u));
    o[p] = r;
  }
}

// Zero the values of samples >= N in the 16-sample group starting at i0 (all of them if i0 >= N).
__device__ __forceinline__ void zero_tail16(uint32_t (&o)[8], int i0, int N) {
#pragma unroll
  for (int p = 0; p < 8; ++p) {
    const int i = i0 + 2 * p;
    if (i >= N) o[p] = 0u;
    else if (i + 1 >= N) o[p] &= 0xFFFFu;
  }
}

// bf16 bits of x (round to nearest even).
__device__ __forceinline__ uint32_t bf16_bits(float x) {
  return (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(x));
}

// The shift c of a row in the split form and the bf16 bits of its missing-call value,
// bf16(mean - c), from its exact sums: c is the mean rounded (half to even) to a multiple of
// 1 / G, G = 128 (2-bit calls) or 1 (dosage bytes). In integers and FP32, with the same bits as
// FP64 gives: the FP64 units take 16 cycles per warp instruction, even for one lane, and three
// divisions per row on them were what bounded the decode (148 us of 65,536 rows x 23,000 samples
// against 56 us for reading them).
// c = k / G with k = rint(G S / n): the FP32 quotient is off by at most one, which the exact
// remainder r = G S - k n sets right. mean - c = r / (G n), rounded to FP32 and then to bf16; where
// the FP32 quotient falls on the middle of two bf16 values, the exact remainder of the division
// (an FMA) decides instead of the tie rule. Exact for G n < 2^24; longer rows take FP64.
template <int G>
__device__ __forceinline__ void row_shift_sums(uint32_t n, unsigned long long S, float& c,
                                               uint32_t& mh) {
  c = 0.0f;
  mh = 0u;
  if (n == 0) return;
  if (n >= (1u << 24) / 256u) {
    const double mean = (double)S / (double)n;
    const double cd = rint(mean * (double)G) * (1.0 / (double)G);
    c = (float)cd;
    mh = (uint32_t)__bfloat16_as_ushort(__double2bfloat16(mean - cd));
    return;
  }
  const int num = (int)((uint32_t)S * (uint32_t)G);  // < 2^24: 2 x 128 n, or 255 n
  int k = (int)rintf((float)num / (float)n);
  int r = num - k * (int)n;
  if (2 * r > (int)n || (2 * r == (int)n && (k & 1))) {
    k += 1;
    r -= (int)n;
  } else if (-2 * r > (int)n || (-2 * r == (int)n && (k & 1))) {
    k -= 1;
    r += (int)n;
  }
  c = (float)k * (1.0f / (float)G);
  const float den = (float)(G * (int)n), q = (float)r / den;
  uint32_t b = __float_as_uint(q);
  const uint32_t low = b & 0xFFFFu;
  const float rem = fmaf(-q, den, (float)r);  // > 0: the quotient lies above q
  bool up = low > 0x8000u || (low == 0x8000u && ((b >> 16) & 1u));
  if (low == 0x8000u && rem != 0.0f) up = (rem > 0.0f) == (q > 0.0f);
  mh = (b >> 16) + (up ? 1u : 0u);
}

// Four dosage bytes w, of which bit k of `use` (4 bits) says that byte k counts: the others set to 0.
__device__ __forceinline__ uint32_t keep_bytes(uint32_t w, uint32_t use) {
  return w & (((use * 0x00204081u) & 0x01010101u) * 0xFFu);
}

// Sums over the 4 x 16 fields of four words of one-bit planes held in the even bits: bytes of the
// result add up to the number of set bits, at most 16 each. Three planes add inside their
// two-bit fields, then pairs of fields into nibbles, pairs of nibbles into bytes: 14 plain
// instructions instead of four population counts, which run at an eighth of their rate.
__device__ __forceinline__ uint32_t plane_bytes(uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  const uint32_t t = a + b + c;
  const uint32_t y = (t & 0x33333333u) + ((t >> 2) & 0x33333333u) + (d & 0x33333333u) +
                     ((d >> 2) & 0x33333333u);
  return (y & 0x0F0F0F0Fu) + ((y >> 4) & 0x0F0F0F0Fu);
}

// Counts of 2-bit fields 64 at a time: high bits, low bits and fields with both (11), in byte sums
// that hold 15 chunks before flush() adds them up.
struct FieldCounts {
  uint32_t high = 0, low = 0, both = 0;
  uint32_t bh = 0, bl = 0, bb = 0;
  int held = 0;
  __device__ __forceinline__ void add(uint4 v) {
    constexpr uint32_t m = 0x55555555u;
    const uint32_t h0 = (v.x >> 1) & m, h1 = (v.y >> 1) & m, h2 = (v.z >> 1) & m, h3 = (v.w >> 1) & m;
    bh += plane_bytes(h0, h1, h2, h3);
    bl += plane_bytes(v.x & m, v.y & m, v.z & m, v.w & m);
    bb += plane_bytes(h0 & v.x, h1 & v.y, h2 & v.z, h3 & v.w);
    if (++held == 15) flush();
  }
  __device__ __forceinline__ void flush() {
    high = __dp4a(bh, 0x01010101u, high);
    low = __dp4a(bl, 0x01010101u, low);
    both = __dp4a(bb, 0x01010101u, both);
    bh = bl = bb = 0;
    held = 0;
  }
};

// Exact counts of one 32-bit word of 2-bit fields (16 samples, the first of which is `left`
// samples before N; fields at or past N are ignored): n observed calls, S the sum of their
// allele-1 counts and S2 the sum of squares (field 00 -> 2, 10 -> 1, 11 -> 0, 01 missing).
__device__ __forceinline__ void count16_2bit(uint32_t w, int left, unsigned long long& n,
                                             unsigned long long& S, unsigned long long& S2) {
  if (left <= 0) return;
  const uint32_t valid = (left >= 16) ? 0x55555555u : (0x55555555u & ((1u << (2 * left)) - 1u));
  const uint32_t lo = w & 0x55555555u;
  const uint32_t hi = (w >> 1) & 0x55555555u;
  const uint32_t two = ~lo & ~hi & valid;
  const uint32_t one = hi & ~lo & valid;
  const uint32_t zero = lo & hi & valid;
  const int c2 = __popc(two), c1 = __popc(one);
  n += (unsigned)(c2 + c1 + __popc(zero));
  S += (unsigned)(2 * c2 + c1);
  S2 += (unsigned)(4 * c2 + c1);
}

}  // namespace tg
