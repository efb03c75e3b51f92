// Rounding of FP64 tiles to the sketch's tensor-core operands, shared by the
// dense-row and the four-step kernels.  Integer operations throughout: FP64
// instructions run at 1/64 of the FP32 rate.
#pragma once

#include "common.cuh"
#include "tc.cuh"

namespace mrcqr {

// fl_p of two consecutive entries of an operand row, given as FP64 bits scaled
// by 2^e: round to odd into FP32 (integer ops), then one
// packed round-to-nearest-even; exact slow path outside the FP32 range.
template <uint32_t FMT>
__device__ __forceinline__ uint32_t pack2(uint32_t h0, uint32_t l0, uint32_t h1, uint32_t l1, int e) {
  uint32_t f0, f1;
  const bool ok0 = scaled_f32_rto(h0, l0, e, f0);
  const bool ok1 = scaled_f32_rto(h1, l1, e, f1);
  if (ok0 && ok1) {
    if constexpr (FMT == tc::F16) {
      const __half2 v = __floats2half2_rn(__uint_as_float(f0), __uint_as_float(f1));
      return *reinterpret_cast<const uint32_t*>(&v);
    } else {
      const __nv_bfloat162 v = __floats2bfloat162_rn(__uint_as_float(f0), __uint_as_float(f1));
      return *reinterpret_cast<const uint32_t*>(&v);
    }
  }
  scale_bits(h0, l0, e);
  scale_bits(h1, l1, e);
  if constexpr (FMT == tc::F16) return f64bits_to_f16(h0, l0) | (f64bits_to_f16(h1, l1) << 16);
  else return f64bits_to_bf16(h0, l0) | (f64bits_to_bf16(h1, l1) << 16);
}

// Conversion of a column whose largest entry has exponent field Emax (scaled by
// 2^(1036 - Emax)): entries with field >= Emax - 139 are FP32 normal afterwards
// and need a subtraction and a funnel shift each.  kFastE: the line above which
// everything smaller, FP64 subnormals included, is below 2^-126.
constexpr uint32_t kFastE = 141;
__device__ __forceinline__ bool col_fast(uint32_t emax) { return emax - kFastE < 0x7FFu - kFastE; }

struct ColScale {
  uint32_t base, thr;   // subtracted from the high word; the smallest |high word| that stays normal
  __device__ __forceinline__ explicit ColScale(uint32_t emax) : base((emax - 140u) << 20), thr((emax - 139u) << 20) {}
};

// |x| 2^e truncated to FP32 bits (no sign), 29 bits of lo left over
__device__ __forceinline__ uint32_t f32_trunc(uint32_t habs, uint32_t lo, const ColScale& c) {
  return __funnelshift_l(lo, habs - c.base, 3);
}

// pack2 for such a column: the same values, rounded to odd without branches.
template <uint32_t FMT>
__device__ __forceinline__ uint32_t pack2_col(uint32_t h0, uint32_t l0, uint32_t h1, uint32_t l1, const ColScale& c,
                                              int e) {
  const uint32_t a0 = h0 & 0x7FFFFFFFu, a1 = h1 & 0x7FFFFFFFu;
  const bool n0 = a0 >= c.thr, n1 = a1 >= c.thr;
  if constexpr (FMT == tc::BF16) {   // BF16 has FP32's exponents: small nonzero entries may be BF16 subnormals
    if ((!n0 && (a0 | l0) != 0u) || (!n1 && (a1 | l1) != 0u)) return pack2<FMT>(h0, l0, h1, l1, e);
  }
  const uint32_t f0 = (h0 & 0x80000000u) | (n0 ? f32_trunc(a0, l0, c) | min(l0 << 3, 1u) : 0u);
  const uint32_t f1 = (h1 & 0x80000000u) | (n1 ? f32_trunc(a1, l1, c) | min(l1 << 3, 1u) : 0u);
  if constexpr (FMT == tc::F16) {
    const __half2 v = __floats2half2_rn(__uint_as_float(f0), __uint_as_float(f1));
    return *reinterpret_cast<const uint32_t*>(&v);
  } else {
    const __nv_bfloat162 v = __floats2bfloat162_rn(__uint_as_float(f0), __uint_as_float(f1));
    return *reinterpret_cast<const uint32_t*>(&v);
  }
}

// 2^(emax - 1036) in FP32 (0, subnormal or infinite outside its range)
__device__ __forceinline__ float col_unscale(uint32_t emax) {
  const int x = (int)emax - 1036;
  return x >= -126 && x <= 127 ? __uint_as_float((uint32_t)(x + 127) << 23) : ldexpf(1.0f, x);
}

// fl_32 bits of an entry of such a column
__device__ __forceinline__ uint32_t f32_col(uint32_t hi, uint32_t lo, const ColScale& c, int e) {
  const uint32_t ha = hi & 0x7FFFFFFFu;
  if (ha >= c.thr || (ha | lo) == 0u) {
    const uint32_t t = f32_trunc(ha, lo, c);
    return (hi & 0x80000000u) | (ha == 0u ? 0u : t + ((lo << 3) + (t & 1u) > 0x80000000u ? 1u : 0u));
  }
  scale_bits(hi, lo, e);
  return f64bits_to_f32(hi, lo);
}

}  // namespace mrcqr
