// Digit arithmetic of the FP64-accurate split products (block updates, Gram products, the fused
// 2D mode product): the scaled integer of an FP64 value cut into base-256 digits, and the exact
// rounding of the recombined levels back to FP64.  Two cuts of the same 55-bit integer:
//
//  * digits_pair (BF16; block updates and Gram products, mma.sync):
//    Digits: a = |x| 2^(55 - E) truncated to an integer, E the row exponent (|x| < 2^E), so
//    a < 2^55, written as a = t 2^48 + c1 2^24 + c2 (t <= 127, c < 2^24), each 24-bit chunk
//    c = d0 2^16 + d1 2^8 + d2 with d0 in [0, 256] and |d1|, |d2| <= 128 (two FP32 roundings,
//    exact), the sign of x applied to every digit.  Integers up to 256 are exact in BF16; digit
//    i weighs 2^(E - 7 - 8 i).  The truncation error is below 2^-55 of the row maximum.
//
//    Exactness of the level sums: with these digit bounds the products d_i(A) d_j(Y) of one
//    level l = i + j add up to at most 196352 (l = 5; 163840 to 179968 for l = 6, 7) per
//    contraction index, so over p <= 64 indices every partial sum is an integer below 2^23.6,
//    exact in an FP32 accumulator.
//
//  * digit_pairs (FP16; the fused mode product): q = x 2^(55 - E) rounded to an integer, |q| <=
//    2^55, in seven balanced digits, |d| <= 128.  Integers up to 2048 are exact in FP16: q + 128
//    (1 + 256 + .. ) has the digits plus 128 as its bytes, so a digit of two values is one byte
//    permute, one OR with the FP16 number 1024 (whose unit is 1) and one packed subtraction of
//    1152: fewer instructions (57 against about 70 for a pair of values) but nearly all on the
//    ALU.  In the kernels whose other work is also there the first cut, which spreads over the
//    FP32 and conversion units, is faster (Gram product of 16 and 8 columns of 5.3 M rows 428 us
//    against 451; update of 36 by 8 over 131,584 rows 28.1 against 28.7).
//    The products of one level are at most 7 2^14 per index, below 2^23 over 64.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <cstdint>

namespace tps {
namespace b256 {

constexpr int kUS = 7;                // base-256 digits per operand
constexpr int kUL = 8;                // digit-pair levels kept: i + j <= 7
constexpr float kMagic = 12582912.f;  // 1.5 2^23: x + kMagic - kMagic = rint(x), |x| <= 2^22

__device__ __forceinline__ unsigned raw_exp(double x) {
  return (unsigned)((__double_as_longlong(x) >> 52) & 0x7FF);
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);  // .x in the low half
  return *reinterpret_cast<const uint32_t *>(&v);
}

// packed pairs of FP32 values (f32x2 arithmetic: two lanes' worth per instruction)
__device__ __forceinline__ uint64_t f2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void f2split(uint64_t v, float &lo, float &hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// |x| 2^(55 - E) truncated to an integer a < 2^55, E = raw_max - 1022 (|x| < 2^E), in
// three unsigned parts, t = a >> 48 (< 128), c1 = bits 24..47, c2 = bits 0..23, and the
// sign of x as +-1.0f.  Integer arithmetic on the FP64 fields (the mantissa shifted right
// by raw_max - ex); subnormals and values 2^-55 below the row maximum flush to zero.
__device__ __forceinline__ void chunks(double x, unsigned raw_max, unsigned &t, unsigned &c1,
                                       unsigned &c2, float &sg) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned ex = (hi >> 20) & 0x7FFu;
  const unsigned sh = ex ? min(raw_max - ex, 63u) : 63u;
  const unsigned long long m =
      ((unsigned long long)((((hi & 0xFFFFFu) | 0x100000u) << 2) | (lo >> 30)) << 32) |
      (unsigned long long)(lo << 2);  // mantissa x 4, 55 bits
  const unsigned long long a = m >> sh;
  t = (unsigned)(a >> 48);
  c1 = (unsigned)(a >> 24) & 0xFFFFFFu;
  c2 = (unsigned)a & 0xFFFFFFu;
  sg = __int_as_float(0x3F800000 | (int)(hi & 0x80000000u));
}

// The digits of two values of one row (same exponent), as BF16 pairs: out[i] holds digit i
// of x0 in its low half and of x1 in its high half.  Digit 0 is sg t; the base-256 digits
// of a signed 24-bit chunk c: d0 = rint(c 2^-16), d1 = rint((c - 2^16 d0) 2^-8),
// d2 = c - 2^16 d0 - 2^8 d1, all exact FP32 operations (f32x2, both values at once).
__device__ __forceinline__ void digits_pair(double x0, double x1, unsigned raw_max,
                                            uint32_t (&out)[kUS]) {
  unsigned t0, a0, b0, t1, a1, b1;
  float s0, s1;
  chunks(x0, raw_max, t0, a0, b0, s0);
  chunks(x1, raw_max, t1, a1, b1, s1);
  out[0] = pack_bf16(s0 * (float)t0, s1 * (float)t1);
  const uint64_t sg = f2(s0, s1);
  const uint64_t M = f2(kMagic, kMagic), nM = f2(-kMagic, -kMagic);
  const uint64_t s16 = f2(1.f / 65536.f, 1.f / 65536.f), s8 = f2(1.f / 256.f, 1.f / 256.f);
  const uint64_t m16 = f2(-65536.f, -65536.f), m8 = f2(-256.f, -256.f);
  const unsigned ca[2] = {a0, b0}, cb[2] = {a1, b1};
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    uint64_t f = mul2(f2((float)ca[h], (float)cb[h]), sg);  // |c| < 2^24: exact
    const uint64_t d0 = add2(add2(mul2(f, s16), M), nM);    // |d0| <= 256
    f = fma2(d0, m16, f);                                   // |f| <= 2^15
    const uint64_t d1 = add2(add2(mul2(f, s8), M), nM);     // |d1| <= 128
    const uint64_t d2 = fma2(d1, m8, f);                    // |d2| <= 128
    float l, u;
    f2split(d0, l, u);
    out[1 + 3 * h] = pack_bf16(l, u);
    f2split(d1, l, u);
    out[2 + 3 * h] = pack_bf16(l, u);
    f2split(d2, l, u);
    out[3 + 3 * h] = pack_bf16(l, u);
  }
}

// The seven digits of one value (for alpha Y, once per CTA).
__device__ __forceinline__ void digits7(double x, unsigned raw_max, float (&d)[kUS]) {
  unsigned t, a, b;
  float sg;
  chunks(x, raw_max, t, a, b, sg);
  d[0] = sg * (float)t;
  const unsigned ch[2] = {a, b};
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    float f = sg * (float)ch[h];
    const float d0 = rintf(f * (1.f / 65536.f));
    f = fmaf(-d0, 65536.f, f);
    const float d1 = rintf(f * (1.f / 256.f));
    d[1 + 3 * h] = d0;
    d[2 + 3 * h] = d1;
    d[3 + 3 * h] = fmaf(-d1, 256.f, f);
  }
}

// round(x 2^(55 - E)) + 128 (1 + 2^8 + .. + 2^48), E = raw_max - 1022 (|x| < 2^E), mxe =
// raw_max << 20: bytes 0 .. 5 are the lower six digits plus 128, the bits from 48 on the top
// digit plus 128 (0 .. 256).  Subnormals count as zero.
__device__ __forceinline__ uint64_t biased55(double x, unsigned mxe) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned exe = hi & 0x7FF00000u;
  const unsigned sh = exe ? min((mxe - exe) >> 20, 63u) : 63u;
  // the mantissa times 8 (56 bits), shifted right; with s = 0 or -1 the sign,
  // (a ^ s) + 2 bias + 1 halved is bias +- round(a / 2), halves away from zero
  const uint64_t m =
      ((uint64_t)((((hi & 0xFFFFFu) | 0x100000u) << 3) | (lo >> 29)) << 32) | (lo << 3);
  const uint64_t a = m >> sh;
  const uint64_t s = (uint64_t)(long long)((int)hi >> 31);
  return ((a ^ s) + 0x0101010101010101ULL) >> 1;
}

// The seven digits of two neighbouring elements as FP16 pairs, most significant first.
__device__ __forceinline__ void digit_pairs(uint64_t u0, uint64_t u1, uint32_t (&d)[kUS]) {
  const uint32_t l0 = (uint32_t)u0, h0 = (uint32_t)(u0 >> 32);
  const uint32_t l1 = (uint32_t)u1, h1 = (uint32_t)(u1 >> 32);
  const __half2 off = __half2half2(__ushort_as_half(0x6480));  // 1152
  uint32_t w[kUS];
  w[0] = __byte_perm(h0, h1, 0x7632) | 0x64006400u;
  w[1] = (__byte_perm(h0, h1, 0x5511) & 0x00FF00FFu) | 0x64006400u;
  w[2] = (__byte_perm(h0, h1, 0x5410) & 0x00FF00FFu) | 0x64006400u;
  w[3] = (__byte_perm(l0, l1, 0x7733) & 0x00FF00FFu) | 0x64006400u;
  w[4] = (__byte_perm(l0, l1, 0x7632) & 0x00FF00FFu) | 0x64006400u;
  w[5] = (__byte_perm(l0, l1, 0x5511) & 0x00FF00FFu) | 0x64006400u;
  w[6] = (__byte_perm(l0, l1, 0x5410) & 0x00FF00FFu) | 0x64006400u;
#pragma unroll
  for (int i = 0; i < kUS; ++i) {
    const __half2 h = __hsub2(*reinterpret_cast<const __half2 *>(&w[i]), off);
    d[i] = *reinterpret_cast<const uint32_t *>(&h);
  }
}

// round(x 2^(62 - E)) + 128 (1 + 2^8 + .. + 2^56), E = raw_max - 1022: its bytes are the eight
// digits of the 62-bit integer plus 128.
__device__ __forceinline__ unsigned long long biased62(double x, unsigned raw_max) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int raw = (int)((b >> 52) & 0x7FF);
  long long q = 0;
  if (raw) {
    const long long mant = (long long)((b & ((1ULL << 52) - 1)) | (1ULL << 52));
    const int sh = raw - (int)raw_max + 9;
    if (sh >= 0)
      q = mant << sh;
    else if (sh > -63)
      q = (mant + (1LL << (-sh - 1))) >> (-sh);
    if (b >> 63) q = -q;
  }
  return (unsigned long long)q + 0x8080808080808080ULL;
}
__device__ __forceinline__ int digit(unsigned long long u, int j) {
  return (int)((u >> (8 * (7 - j))) & 0xFF) - 128;
}
__device__ __forceinline__ int digit62(double x, unsigned raw_max, int j) {
  return digit(biased62(x, raw_max), j);
}

// sum_l d_l 2^(104 - 8 l) 2^(E - 117) rounded to FP64: the levels of seven digits of A (scale
// 2^E_A) times eight digits of B, the scale 2^E_B of a column of B being its absolute sum, E =
// E_A + E_B.  As the sum is then below 2^E, the levels add up modulo 2^64 to its integer in
// units of 2^(E - 62); of level 7 (unit 2^(E - 69)) the part below is rounded away, a quarter of
// what the digit pairs that are not kept weigh (2^(E - 60.5), root mean square at 48 indices).
// One conversion on the FP64 pipe rounds the integer (a warp instruction takes that pipe ~64
// cycles; rounding by integer instructions costs ~20 more of them).  w1, w9, w17, w25 = 2, 2^9,
// 2^17, 2^25 come from the kernel's arguments or constant memory: as immediates they would become
// shifts and adds on the ALU, the busiest pipe, where the multiply-adds run on the FMA pipe.
struct LevelWeights {
  int w1, w9, w17, w25;
};
inline LevelWeights level_weights() { return {1 << 1, 1 << 9, 1 << 17, 1 << 25}; }
__device__ __forceinline__ double pow2d(int e);
__device__ __forceinline__ double level_sum(const int (&d)[kUL], int E, const LevelWeights &g) {
  const int t7 = (d[7] + 64) >> 7;
  long long t;
  asm("{\n\t.reg .b64 t;\n\t"
      "cvt.s64.s32 t, %5;\n\t"
      "mad.wide.s32 t, %4, %6, t;\n\t"
      "mad.wide.s32 t, %3, %7, t;\n\t"
      "mad.wide.s32 t, %2, %8, t;\n\t"
      "mad.wide.s32 %0, %1, %9, t;\n\t}"
      : "=l"(t)
      : "r"(d[3]), "r"(d[4]), "r"(d[5]), "r"(d[6]), "r"(t7), "r"(g.w1), "r"(g.w9), "r"(g.w17),
        "r"(g.w25));
  const unsigned top = (unsigned)(d[0] * g.w17) + (unsigned)(d[1] * g.w9) +
                       (unsigned)(d[2] * g.w1);
  t = (long long)((unsigned long long)t + ((unsigned long long)top << 32));
  const int e = E - 62;
  if (e < -1000 || e > 900) {  // near the ends of the range: two factors
    const int h = e / 2;
    return (double)t * pow2d(h) * pow2d(e - h);
  }
  // times 2^e in the exponent field (1023 .. 1086 for a nonzero integer)
  const double v = (double)t;
  const int hi = __double2hiint(v);
  return __hiloint2double(hi ? hi + (e << 20) : 0, __double2loint(v));
}

__device__ __forceinline__ double pow2d(int e) {
  e = e < -1022 ? -1022 : (e > 1023 ? 1023 : e);
  return __longlong_as_double((long long)(e + 1023) << 52);
}

// (hi 2^32 + lo) 2^(E - 70) rounded to the nearest FP64 value (ties to even), |hi|, |lo| <
// 2^49, by integer arithmetic (GB300's FP64 pipe issues one warp instruction per ~64 cycles
// of a sub-partition, the integer pipes one per cycle); results outside the normal range
// take the FP64 formula, which rounds the same way.
__device__ __forceinline__ double combine(long long hi, long long lo, int E) {
  const long long top = hi + (lo >> 32);  // S = top 2^32 + bot exactly, 0 <= bot < 2^32
  const unsigned bot = (unsigned)lo;
  const bool neg = top < 0;
  unsigned long long T;
  unsigned B;
  if (!neg) {
    T = (unsigned long long)top;
    B = bot;
  } else if (bot == 0) {
    T = (unsigned long long)(-top);
    B = 0;
  } else {
    T = (unsigned long long)(-top - 1);
    B = 0u - bot;
  }
  if (T == 0 && B == 0) return 0.0;
  const int lb = T ? 95 - __clzll((long long)T) : 31 - __clz((int)B);  // leading bit of |S|
  int sh = lb - 52;
  unsigned long long mant;
  if (sh <= 0) {
    mant = ((T << 32) | B) << (-sh);  // |S| < 2^53: exact
  } else {                            // sh <= 29: the dropped bits are all in B
    mant = (T << (32 - sh)) | (B >> sh);
    const unsigned rem = B & ((1u << sh) - 1u), half = 1u << (sh - 1);
    if (rem > half || (rem == half && (mant & 1ULL))) {
      ++mant;
      if (mant >> 53) {
        mant >>= 1;
        ++sh;
      }
    }
  }
  const int be = sh + E - 70 + 52 + 1023;
  if (be <= 0 || be >= 2047)
    return fma((double)lo, pow2d(E - 70), (double)hi * pow2d(E - 38));
  return __longlong_as_double((long long)(((unsigned long long)neg << 63) |
                                          ((unsigned long long)be << 52) |
                                          (mant & ((1ULL << 52) - 1))));
}

}  // namespace b256
}  // namespace tps
