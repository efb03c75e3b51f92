// FP64 products on FP16 tensor cores by exact integer slicing (the
// error-free splitting of Ozaki, Ogita, Oishi, Rump, "Error-free
// transformations of matrix multiplication by using fast routines of matrix
// multiplication and its applications", Numer. Algorithms 59, 2012), with
// balanced (signed) base-256 digits.
//
// A value x of a row (or column) whose largest magnitude has biased FP64
// exponent Eref is rounded to the 63-bit fixed-point integer
//   I = round(|x| 2^(1085 - Eref)),   0 <= I < 2^63
// (exact for every x within 2^10 of the maximum), and I is written in eight
// signed base-256 digits
//   I = sum_{a=0..7} d_a 2^(56 - 8a),  d_0 in [0, 128], d_{a>0} in [-128, 127],
// each exact in FP16 (the sign of x is applied to every digit).  A product
// sum_k x_ik y_kj keeps the digit pairs with a + b <= 7; the pairs of one
// level L = a + b are accumulated together in FP32 by tcgen05.mma.  Per term
// a level sums at most 2^15 + 6 * 2^14 = 2^17 in magnitude, so a level
// accumulated over K <= 128 terms is an integer of magnitude <= 2^24, exact in
// FP32.  The levels are combined with 64-bit integer arithmetic into the
// 128-bit
//   T = sum_L acc_L 2^(8(7-L)) = (sum_{L<4} acc_L 2^(8(3-L))) 2^32 + sum_{L>=4} acc_L 2^(8(7-L))
// and T 2^(Erow + Ecol - 2114) is rounded once to FP64.  With R_i, C_j the
// row and column maxima (R_i >= 2^61 units of I), the rounding of I costs at
// most 2^-62 R_i per operand and the dropped pairs (a + b >= 8, at most
// 7 * 2^14 of their level units) at most 7.03 * 2^-60 R_i C_j per term, so
// one term is off by less than 2^-57 R_i C_j, 16 times below the unit
// roundoff; the sum is rounded once.  Everything outside the tensor cores is
// 32/64-bit integer work (FP64 instructions issue to a 1/64-rate pipe on this
// GPU).
#pragma once
#include <cstdint>
#include "common.cuh"

namespace mrcqr {
namespace oz {

constexpr int kSlices = 8;
constexpr int kLevels = 8;
constexpr int kScaleBias = 2114;   // T 2^(Erow + Ecol - kScaleBias) is the product

// Biased FP64 exponent field of |x| from its high word (0 for zero and
// subnormals, which slice to zero against any normal reference).
__device__ __forceinline__ uint32_t exp_field(uint32_t hi) { return (hi >> 20) & 0x7FFu; }

// The fixed-point integer I = round(|x| 2^eoff 2^(1085 - Eref)) of x (FP64
// bits hi:lo) against the reference exponent Eref (biased; >= the exponent of
// x 2^eoff), plus 128 at each of the seven low byte positions: the plain
// bytes of the result are the balanced digits (the top byte d_0, the others
// d_a + 128; the carries do the rest).  Zero and subnormal x give I = 0.  The
// power-of-two scale eoff (a diagonal scaling D of a product (X D)(D^-1 Y))
// never rounds.
//
// The slicing kernels spend most of their instructions here and in
// digits8_pack, on the 64-lane integer pipe, so the common case is kept short:
// with the significand M left-aligned in 64 bits, I = M >> t plus bit t - 1 of
// M (round half up in magnitude), t = Eref - eoff - E + 1 >= 1.  For t <= 32
// these are three funnel shifts.  Values below 2^-31 of the reference, zeros
// and subnormals (t > min(32, Eref - eoff): E = 0 gives t = Eref - eoff + 1)
// take the general form in a branch that a warp normally skips.
__device__ __forceinline__ uint64_t biased_fixed63(uint32_t hi, uint32_t lo, int Eref, int eoff) {
  const int top = Eref - eoff;
  const int E = (int)exp_field(hi);
  const int t = top + 1 - E;
  const uint32_t mh = __funnelshift_l(lo, hi, 11) | 0x80000000u, ml = lo << 11;
  uint32_t rl = __funnelshift_rc(ml, mh, (uint32_t)t), rh = __funnelshift_rc(mh, 0u, (uint32_t)t);
  uint32_t rb = __funnelshift_rc(ml, mh, (uint32_t)(t - 1)) & 1u;
  if (t > min(32, top)) {
    uint64_t v = 0;
    if (E != 0 && t <= 64) {
      const uint64_t M = (uint64_t)mh << 32 | ml;
      v = ((M >> (t - 1)) + 1ull) >> 1;
    }
    rl = (uint32_t)v;
    rh = (uint32_t)(v >> 32);
    rb = 0u;
  }
  return ((uint64_t)rh << 32 | rl) + rb + 0x0080808080808080ull;
}

// Signed digits d[0..7] of x 2^eoff (see biased_fixed63), sign of x included.
__device__ __forceinline__ void digits8(uint32_t hi, uint32_t lo, int Eref, int* d, int eoff = 0) {
  const uint64_t v = biased_fixed63(hi, lo, Eref, eoff);
  const uint32_t l = (uint32_t)v, h = (uint32_t)(v >> 32);
  d[0] = (int)(h >> 24);
  d[1] = (int)((h >> 16) & 255u) - 128;
  d[2] = (int)((h >> 8) & 255u) - 128;
  d[3] = (int)(h & 255u) - 128;
  d[4] = (int)(l >> 24) - 128;
  d[5] = (int)((l >> 16) & 255u) - 128;
  d[6] = (int)((l >> 8) & 255u) - 128;
  d[7] = (int)(l & 255u) - 128;
  if (hi >> 31) {
#pragma unroll
    for (int a = 0; a < kSlices; ++a) d[a] = -d[a];
  }
}

// The eight digits of two values as packed FP16 pairs (digit a of x0 in the
// low half of out[a], of x1 in the high half), straight from the bytes of
// their biased fixed-point words (hi J0h, lo J0l; J1h, J1l) and the sign bits
// of h0, h1: the FP16 bits 0x6400 + byte are the value 1024 + byte (one
// binade, spacing 1), and one fused multiply-add (1024 + byte) s - c s, c =
// 1024 for digit 0 and 1152 (1024 + the bias 128) for the others, is s d
// exactly.  Bytes move in two permutes per 16 bits of both words (pair the
// halves, then put the 0x64 between the bytes): twelve per pair of values and
// no masks.
__device__ __forceinline__ void digits8_pack(uint32_t J0h, uint32_t J0l, uint32_t J1h, uint32_t J1l, uint32_t h0,
                                             uint32_t h1, uint32_t* out) {
  const uint32_t x = __byte_perm(h0, h1, 0x7030u);            // sign bytes of both values
  const uint32_t sb = (x & 0x80008000u) | 0x3C003C00u;        // (+-1, +-1)
  const uint32_t cb = (x & 0x80008000u) ^ 0xE480E480u;        // (-+1152, -+1152)
  const uint32_t c0 = (x & 0x80008000u) ^ 0xE400E400u;        // (-+1024, -+1024)
  const __half2 s2 = *reinterpret_cast<const __half2*>(&sb);
#pragma unroll
  for (int w = 0; w < 4; ++w) {            // 16 bits of each word, from the top: digits 2 w and 2 w + 1
    const uint32_t p = __byte_perm(w < 2 ? J0h : J0l, w < 2 ? J1h : J1l, (w & 1) ? 0x5410u : 0x7632u);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int a = 2 * w + k;
      const uint32_t t = __byte_perm(p, 0x64646464u, k == 0 ? 0x4341u : 0x4240u);
      const uint32_t c = a == 0 ? c0 : cb;
      const __half2 r = __hfma2(*reinterpret_cast<const __half2*>(&t), s2, *reinterpret_cast<const __half2*>(&c));
      out[a] = *reinterpret_cast<const uint32_t*>(&r);
    }
  }
}
__device__ __forceinline__ void digits8_pack(uint64_t J0, uint64_t J1, uint32_t neg0, uint32_t neg1, uint32_t* out) {
  digits8_pack((uint32_t)(J0 >> 32), (uint32_t)J0, (uint32_t)(J1 >> 32), (uint32_t)J1, neg0 << 31, neg1 << 31, out);
}

// The biased fixed-point word of biased_fixed63 without a branch, for
// 0 <= k = E + eoff - Eref + 31 <= 31 (every value from the reference's binade
// down to 2^-31 of it): I = (M 2^k + 2^20) >> 21 with M the 53-bit
// significand.  The variable shift is a multiplication by 2^k, which runs on
// the FMA pipe beside the integer pipe that bounds the slicing, with the
// rounding and the byte biases (shifted up by 21) as its addends; k for
// the caller's range check is OR-ed into kor, c = 31 + eoff - Eref.
__device__ __forceinline__ void fixed63_fast(uint32_t h, uint32_t l, int c, uint32_t& Jh, uint32_t& Jl, uint32_t& kor) {
  // (bias << 21) + 2^20 split at bit 64: the low part is below 2^61, so adding it to l p < 2^63 does not carry out
  constexpr uint64_t kBias = 0x0080808080808080ull;
  constexpr uint64_t kLow = (kBias << 21) + (1ull << 20);
  constexpr uint64_t kHigh = (kBias >> 43) << 32;
  static_assert(kLow < (1ull << 61), "fixed63_fast: carry");
  const uint32_t k = exp_field(h) + (uint32_t)c;
  kor |= k;
  const uint32_t p = __funnelshift_l(0u, 1u, k);   // 2^(k mod 32)
  const uint64_t a = (uint64_t)l * p + kLow;
  const uint64_t b = (uint64_t)((h & 0xFFFFFu) | 0x100000u) * p + (kHigh | (a >> 32));
  Jl = __funnelshift_r((uint32_t)a, (uint32_t)b, 21);
  Jh = __funnelshift_r((uint32_t)b, (uint32_t)(b >> 32), 21);
}

// Exact float of a small signed integer (|v| < 2^22) without a conversion
// instruction: 1.5 * 2^23 + v has v in its low mantissa bits.
__device__ __forceinline__ float small_int_to_float(int v) {
  return __int_as_float(0x4B400000 + v) - 12582912.0f;
}

// Adds one level's exact FP32 accumulator (an integer, |v| <= 2^24) into a
// 64-bit half of T.  The shift is a multiply by 2^(8 (3 - L % 4)) fused with the 64-bit add
// (one mad.wide.s32: a sign-extended 32 x 32 -> 64-bit product plus the
// accumulator), exact for every |v| < 2^31.
__device__ __forceinline__ long long mad_wide_s32(int a, int b, long long c) {
  long long r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
}

// An integer |v| <= 2^22 in FP32 without a conversion instruction (those issue
// at a sixteenth of the FMA rate, and a readout has 128 per thread): the bits
// of v + 1.5 2^23 are kSmallBias + v.  kLevelBias is the bias's share of the
// four levels of a half.
constexpr int kSmallBias = 0x4B400000;
constexpr long long kLevelBias = (long long)kSmallBias * ((1ll << 24) + (1ll << 16) + (1ll << 8) + 1);
__device__ __forceinline__ int small_float_bits(float v) { return __float_as_int(v + 12582912.0f); }

// Signed 128-bit integer as (high word th, low word tl): two's complement.
struct I128 {
  int64_t h;
  uint64_t l;
};

__device__ __forceinline__ I128 i128_from_parts(long long hi, long long lo) {   // hi 2^32 + lo
  I128 r;
  const uint64_t tl = (uint64_t)hi << 32;
  r.h = hi >> 32;
  r.l = tl + (uint64_t)lo;
  r.h += (lo >> 63) + (r.l < tl ? 1 : 0);
  return r;
}

__device__ __forceinline__ void i128_add(I128& a, const I128& b) {
  const uint64_t l = a.l + b.l;
  a.h += b.h + (l < a.l ? 1 : 0);
  a.l = l;
}

// T 2^scale rounded once to FP64 (round to nearest even).
__device__ __forceinline__ double i128_to_double(I128 t, int scale) {
  uint64_t tl = t.l;
  int64_t th = t.h;
  const bool neg = th < 0;
  if (neg) {
    tl = ~tl + 1ull;
    th = (int64_t)(~(uint64_t)th + (tl == 0 ? 1ull : 0ull));
  }
  const uint64_t uh = (uint64_t)th;
  if (uh == 0 && tl == 0) return neg ? -0.0 : 0.0;
  const int p = uh ? 127 - __clzll((long long)uh) : 63 - __clzll((long long)tl);   // msb position
  uint64_t m;
  int e2 = p;   // value = m 2^(p - 52) before scaling
  if (p <= 52) {
    m = tl << (52 - p);
  } else {
    const int sh = p - 52;   // 1 .. 75
    uint64_t q, rem_hi_bit, sticky;
    if (sh < 64) {
      q = (tl >> sh) | (uh << (64 - sh));
      rem_hi_bit = (tl >> (sh - 1)) & 1ull;
      sticky = tl & ((1ull << (sh - 1)) - 1ull);
    } else {
      const int s2 = sh - 64;   // 0 .. 11
      q = uh >> s2;
      if (s2 == 0) {
        rem_hi_bit = tl >> 63;
        sticky = tl & 0x7FFFFFFFFFFFFFFFull;
      } else {
        rem_hi_bit = (uh >> (s2 - 1)) & 1ull;
        sticky = (uh & ((1ull << (s2 - 1)) - 1ull)) | tl;
      }
    }
    m = q;
    if (rem_hi_bit && (sticky || (m & 1ull))) ++m;
    if (m >> 53) {
      m >>= 1;
      ++e2;
    }
  }
  const int E = e2 + scale + 1023;
  if (E <= 0 || E >= 2047) {   // outside the normal range (subnormal results are rounded twice)
    const double v = ldexp((double)(m & ((1ull << 53) - 1ull)), e2 - 52 + scale);
    return neg ? -v : v;
  }
  const uint64_t bits = ((uint64_t)(neg ? 1 : 0) << 63) | ((uint64_t)E << 52) | (m & ((1ull << 52) - 1ull));
  return __longlong_as_double((long long)bits);
}

// (hi 2^32 + lo) 2^scale rounded once to FP64.
__device__ __forceinline__ double i128_to_double(long long hi, long long lo, int scale) {
  return i128_to_double(i128_from_parts(hi, lo), scale);
}

// Out of line: the rare results of the two conversions below (a copy at each of their
// unrolled uses would fill the instruction cache).
static __device__ __noinline__ double t96_general(long long hi, long long lo, int scale) {
  return i128_to_double(hi, lo, scale);
}

// The same for the level sums of one tile entry, |hi|, |lo| < 2^50: 96-bit
// arithmetic on three words, the leading bit found in the upper two of them
// (a smaller or out-of-range result takes the general form).  About 37
// integer-pipe instructions.
__device__ __forceinline__ double t96_to_double(long long hi, long long lo, int scale) {
  const long long s = hi + (lo >> 32);            // T = s 2^32 + l
  uint32_t b = (uint32_t)((uint64_t)s >> 32), a = (uint32_t)s, l = (uint32_t)lo;
  const uint32_t sg = (uint32_t)((int)b >> 31);   // |T|
  const uint64_t al = (((uint64_t)a << 32 | l) ^ ((uint64_t)sg << 32 | sg)) + (sg & 1u);
  b = (b ^ sg) + ((sg != 0u && al == 0) ? 1u : 0u);
  a = (uint32_t)(al >> 32);
  l = (uint32_t)al;
  const bool small = b == 0u;
  const uint32_t x2 = small ? a : b, x1 = small ? l : a, x0 = small ? 0u : l;
  const int z = __clz((int)x2);
  const uint32_t y2 = __funnelshift_l(x1, x2, z), y1 = __funnelshift_l(x0, x1, z), y0 = x0 << (z & 31);
  // bits 63 .. 11 of (y2, y1) are the significand; round to nearest even on the rest
  const uint32_t rest = (y1 & 0x7FFu) | (y0 != 0u ? 1u : 0u);
  const uint32_t up = (rest + 0x3FFu + ((y1 >> 11) & 1u)) >> 11;
  const int E = (small ? 63 : 95) - z + scale + 1023;
  if (x2 == 0u || (uint32_t)(E - 1) >= 2045u) return t96_general(hi, lo, scale);
  const uint64_t bits = ((uint64_t)y2 << 21 | (y1 >> 11)) + up + ((uint64_t)(uint32_t)(E - 1) << 52);
  return __longlong_as_double((long long)(bits | (uint64_t)(sg & 0x80000000u) << 32));
}

// The same with two FP64 additions (the FP64 pipe is otherwise idle in the
// kernels that use this; a warp's addition holds it for 64 cycles, about what
// the integer form takes in all, so they convert half of their entries each
// way): s 2^32 - 2^52 and 2^52 + l are exact, and their sum T is rounded once.
__device__ __forceinline__ double t96_to_double_fp64(long long hi, long long lo, int scale) {
  const long long s = hi + (lo >> 32);
  const uint32_t l = (uint32_t)lo;
  constexpr double kC = 1.5 * 19342813113834066795298816.0 + 4503599627370496.0;   // 1.5 2^84 + 2^52
  const double a = __hiloint2double((int)((uint64_t)s >> 32) + 0x45380000, (int)(uint32_t)s);   // 1.5 2^84 + s 2^32
  const double r = (a - kC) + __hiloint2double(0x43300000, (int)l);
  const uint32_t h = (uint32_t)__double2hiint(r);
  const uint32_t e = exp_field(h), E = e + (uint32_t)scale;
  if (e == 0u || E - 1u >= 2045u) return t96_general(hi, lo, scale);
  return __hiloint2double((int)(h + ((uint32_t)scale << 20)), __double2loint(r));
}

}  // namespace oz
}  // namespace mrcqr
