// The two-stage emulated-FP64 product pipeline shared by the kernels of
// ozaki.cu and ozaki_planes.cu: one CTA per SM, 512 threads, all 512 TMEM
// columns = 8 level accumulators of 128 x 64; digit panels of a K chunk (32
// deep, K-major SWIZZLE_64B) in shared memory, the 8 digits of the A operand
// against the N-stacked digits of the B operand in 12 MMAs per K step, and
// the exact level sums read out of TMEM into 64-bit integers every 4 chunks.
#pragma once
#include "kernels.h"
#include "ozaki.cuh"
#include "tc.cuh"

namespace mrcqr {
namespace {

constexpr int kOzThreads = 512;
constexpr int kM = 128;                     // MMA M: rows of the A operand
constexpr int kN = 64;                      // MMA N: rows of the B operand, TMEM columns per level
constexpr int kK = 32;                      // K depth of a chunk (one 64-byte FP16 row)
constexpr int kGroupChunks = 4;             // chunks per exact FP32 accumulation (K <= 128)
constexpr uint32_t kAPanel = kM * 64;       // one digit of a 128 x 32 FP16 block (8 KiB)
constexpr uint32_t kBPanel = kN * 64;       // one digit of a 64 x 32 FP16 block (4 KiB)
constexpr uint32_t kStage = oz::kSlices * (kAPanel + kBPanel);   // 96 KiB
constexpr size_t kSmem = 2 * (size_t)kStage + 1024;
constexpr size_t kPartElems = 2 * kM * kN;  // hi and lo of one 128 x 64 item

// The digit-pair products of one chunk (two K steps of 16).  Level L
// accumulates in TMEM columns [64 L, 64 L + 64).  The eight digit panels of B
// are contiguous, so digits 0 .. 7 - a stacked along N form one operand, and
// a single MMA of A digit a against it (N = 64 (8 - a), split at N = 256)
// written at TMEM column 64 a adds A_a B_b to level a + b for every b at once:
// 12 MMAs per K step instead of one per pair (36), with no discarded pairs.
// Issued by one thread; the first MMA (a = 0) of a group overwrites all eight
// levels.  ab / bb: shared addresses of digit 0 of the A and B panels.
__device__ __forceinline__ void oz_issue_chunk(uint32_t tmem, uint32_t ab, uint32_t bb, bool group_start) {
  const uint64_t da = tc::sw64_desc(ab), db = tc::sw64_desc(bb);
#pragma unroll
  for (int kk = 0; kk < kK; kk += 16) {
#pragma unroll
    for (int a = 0; a < oz::kLevels; ++a) {
      const uint64_t adesc = da + (uint64_t)((a * kAPanel + kk * 2) >> 4);
      const int ntot = kN * (oz::kLevels - a);
#pragma unroll
      for (int p0 = 0; p0 < ntot; p0 += 256) {
        const int nn = ntot - p0 < 256 ? ntot - p0 : 256;
        tc::mma_f16(tmem + (uint32_t)(kN * a + p0), adesc, db + (uint64_t)((p0 * 64 + kk * 2) >> 4),
                    tc::idesc(tc::F16, kM, nn), (kk == 0 && a == 0 && group_start) ? 0u : 1u);
      }
    }
  }
}

// Adds the exact level sums of 16 TMEM columns from `base` (level L at column
// offset L * stride) into the 64-bit halves hi / lo.  The sums of |v| over eight
// columns bound every |v|: below 2^22 (for digits of ordinary data about 2^20)
// no conversion instruction is needed; a warp that meets a larger sum corrects
// the readout with conversions.  kLoop: small loop bodies (in the digit-plane
// sketch the unrolled form spills: 63 against 55 ms at m = 2^20, n = 512); else
// unrolled, two levels of eight columns per wait (2 to 4% faster in the others).
template <int kStride, bool kLoop>
__device__ __forceinline__ void oz_readout_cols(uint32_t base, long long* hi, long long* lo) {
  float big = 0.0f;
  if (kLoop) {
#pragma unroll
    for (int half = 0; half < 2; ++half) {   // levels 0 .. 3 into hi, levels 4 .. 7 into lo
      long long* x = half ? lo : hi;
      int mul = 1 << 24;
#pragma unroll 1
      for (int L = 4 * half; L < 4 * half + 4; ++L) {
        float v[16];
        tc::tmem_ld16(base + (uint32_t)(L * kStride), v);
        tc::tmem_wait_ld();
#pragma unroll
        for (int h = 0; h < 16; h += 8) {
          float sum = 0.0f;
#pragma unroll
          for (int c = h; c < h + 8; ++c) {
            sum += fabsf(v[c]);
            x[c] = oz::mad_wide_s32(oz::small_float_bits(v[c]), mul, x[c]);
          }
          big = fmaxf(big, sum);
        }
        mul >>= 8;
      }
    }
  } else {
#pragma unroll
    for (int h = 0; h < 16; h += 8) {
#pragma unroll
      for (int L = 0; L < oz::kLevels; L += 2) {
        float v[2][8];
        tc::tmem_ld8(base + (uint32_t)(L * kStride + h), v[0]);
        tc::tmem_ld8(base + (uint32_t)((L + 1) * kStride + h), v[1]);
        tc::tmem_wait_ld();
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          long long* x = L < 4 ? hi : lo;
          float sum = 0.0f;
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            sum += fabsf(v[u][c]);
            x[h + c] = oz::mad_wide_s32(oz::small_float_bits(v[u][c]), 1 << (24 - 8 * ((L + u) & 3)), x[h + c]);
          }
          big = fmaxf(big, sum);
        }
      }
    }
  }
#pragma unroll
  for (int c = 0; c < 16; ++c) hi[c] -= oz::kLevelBias, lo[c] -= oz::kLevelBias;
  if (__any_sync(0xffffffffu, !(big < 4194304.0f))) {   // replace the sums' contributions by exact conversions
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      long long* x = half ? lo : hi;
#pragma unroll 1
      for (int L = 0; L < 4; ++L) {
        float v[16];
        tc::tmem_ld16(base + (uint32_t)((4 * half + L) * kStride), v);
        tc::tmem_wait_ld();
#pragma unroll
        for (int c = 0; c < 16; ++c) {
          const long long d = (long long)__float2int_rn(v[c]) - ((long long)oz::small_float_bits(v[c]) - oz::kSmallBias);
          x[c] += d << (24 - 8 * L);
        }
      }
    }
  }
}

// The level sums of TMEM lane 32 q + lane, columns 16 g .. 16 g + 15 of a
// 128 x 64 tile (warp w: q = w % 4, g = w / 4).
template <bool kLoop>
__device__ __forceinline__ void oz_readout(uint32_t tmem, int q, int g, long long* hi, long long* lo) {
  oz_readout_cols<kN, kLoop>(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(g * 16), hi, lo);
}

// Digits of two values (FP64 bits, sign flips f0 / f1 applied, scaled by
// 2^eo0 / 2^eo1) against the reference exponent E, packed in pairs into the
// eight digit panels at the shared address dst (and dst2, if nonzero).
__device__ __forceinline__ void oz_store_pair(double v0, double v1, uint32_t f0, uint32_t f1, int E,
                                              uint32_t dst, uint32_t pstride, int eo0 = 0, int eo1 = 0,
                                              uint32_t dst2 = 0, uint32_t pstride2 = 0) {
  const uint32_t h0 = (uint32_t)__double2hiint(v0), h1 = (uint32_t)__double2hiint(v1);
  const uint64_t J0 = oz::biased_fixed63(h0, (uint32_t)__double2loint(v0), E, eo0);
  const uint64_t J1 = oz::biased_fixed63(h1, (uint32_t)__double2loint(v1), E, eo1);
  uint32_t w[oz::kSlices];
  oz::digits8_pack(J0, J1, (h0 >> 31) ^ f0, (h1 >> 31) ^ f1, w);
#pragma unroll
  for (int a = 0; a < oz::kSlices; ++a) tc::st_shared(dst + a * pstride, w[a]);
  if (dst2) {
#pragma unroll
    for (int a = 0; a < oz::kSlices; ++a) tc::st_shared(dst2 + a * pstride2, w[a]);
  }
}

// Digits of four values adjacent along K (reference exponent E, cr = 31 - E or
// a large negative number that forces the general form; sign flips in bits 0 .. 3 of
// flips) stored as 8 bytes per digit panel at the shared address dst (and
// dst2, if nonzero).  Straight-line code with one range check at the end:
// values below 2^-31 of the reference, zeros and subnormals make the thread
// write its digits again from biased_fixed63.
template <bool kFlips = false>
__device__ __forceinline__ void oz_store_quad(const double (&v)[4], uint32_t flips, int E, int cr, uint32_t dst,
                                              uint32_t pstride, uint32_t dst2 = 0, uint32_t pstride2 = 0) {
  uint32_t kor = 0u;
  uint32_t o[2][oz::kSlices];
#pragma unroll
  for (int p = 0; p < 2; ++p) {
    uint32_t h[2], Jh[2], Jl[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      h[k] = (uint32_t)__double2hiint(v[2 * p + k]);
      oz::fixed63_fast(h[k], (uint32_t)__double2loint(v[2 * p + k]), cr, Jh[k], Jl[k], kor);
      if (kFlips) h[k] ^= (flips << (31 - 2 * p - k)) & 0x80000000u;
    }
    oz::digits8_pack(Jh[0], Jl[0], Jh[1], Jl[1], h[0], h[1], o[p]);
  }
#pragma unroll
  for (int a = 0; a < oz::kSlices; ++a) tc::st_shared2(dst + a * pstride, o[0][a], o[1][a]);
  if (dst2) {
#pragma unroll
    for (int a = 0; a < oz::kSlices; ++a) tc::st_shared2(dst2 + a * pstride2, o[0][a], o[1][a]);
  }
  if (kor > 31u) {
#pragma unroll
    for (int p = 0; p < 2; ++p)
      oz_store_pair(v[2 * p], v[2 * p + 1], kFlips ? (flips >> (2 * p)) & 1u : 0u,
                    kFlips ? (flips >> (2 * p + 1)) & 1u : 0u, E, dst + 4 * p, pstride, 0, 0, dst2 ? dst2 + 4 * p : 0u,
                    pstride2);
  }
}

// Constant of oz_store_quad for the reference exponent E (tiny references
// take the general form: a zero's exponent field must not pass for a value's).
__device__ __forceinline__ int oz_quad_cr(int E) { return E > 31 ? 31 - E : -(1 << 30); }

// Four rows from r of one column (col: the column's base), zero from r_end on; vec: the column is
// 16-byte aligned at even rows.
__device__ __forceinline__ void oz_load_quad(const double* __restrict__ col, int64_t r, int64_t r_end, bool vec,
                                             double (&v)[4]) {
  if (r + 4 <= r_end) {
    if (vec) {
      const double2 x = __ldg(reinterpret_cast<const double2*>(col + r));
      const double2 y = __ldg(reinterpret_cast<const double2*>(col + r + 2));
      v[0] = x.x, v[1] = x.y, v[2] = y.x, v[3] = y.y;
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i) v[i] = __ldg(col + r + i);
    }
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = r + i < r_end ? __ldg(col + r + i) : 0.0;
  }
}

// A 32-row chunk of NC columns of a column-major matrix (column col0 + c,
// zero beyond n or r_end) in registers: lane l holds rows 2(l % 16) and
// 2(l % 16) + 1 of columns 32 it + 2 warp + l / 16.  Issued one chunk ahead
// of its use, so the loads are in flight during the MMAs.
template <int NC>
__device__ __forceinline__ void oz_load_cols(const double* __restrict__ X, int64_t ldx, int n, int col0, int64_t r0,
                                             int64_t r_end, int warp, int lane, double (&v)[NC / 32][2]) {
  const int p = lane & 15, h = lane >> 4;
  const int64_t ra = r0 + 2 * p;
#pragma unroll
  for (int it = 0; it < NC / 32; ++it) {
    const int col = col0 + 32 * it + 2 * warp + h;
    v[it][0] = v[it][1] = 0.0;
    if (col < n) {
      const double* src = X + (int64_t)col * ldx;
      if (ra < r_end) v[it][0] = __ldg(src + ra);
      if (ra + 1 < r_end) v[it][1] = __ldg(src + ra + 1);
    }
  }
}

// Digits of the values loaded by oz_load_cols (reference exponent E[c], sign
// flips f0 / f1 of the lane's two rows) into panel rows c.
template <int NC>
__device__ __forceinline__ void oz_store_cols(const double (&v)[NC / 32][2], const uint32_t* E, uint32_t f0,
                                              uint32_t f1, unsigned char* panel, uint32_t pstride, int warp,
                                              int lane) {
  const int p = lane & 15, h = lane >> 4;
#pragma unroll
  for (int it = 0; it < NC / 32; ++it) {
    const int c = 32 * it + 2 * warp + h;
    oz_store_pair(v[it][0], v[it][1], f0, f1, E[c], tc::smem_u32(panel) + tc::sw64_offset(c, 2 * p, 2), pstride);
  }
}

// --- the 128 x 32 tile of the kernels with two CTAs per SM (rowprod.cu, sketch_fd.cu): half of the TMEM each
constexpr int kRN = 32;                           // output tile width = MMA N per level, and K chunk depth
constexpr int kRThreads = 256;
constexpr uint32_t kRBPanel = kRN * 64;           // one digit of a 32 x 32 multiplier block (2 KiB)
constexpr uint32_t kRABytes = oz::kSlices * kAPanel;    // 64 KiB: digits of a 128 x 32 chunk
constexpr uint32_t kRBBytes = oz::kSlices * kRBPanel;   // 16 KiB: digits of a multiplier block
constexpr uint32_t kRTmem = oz::kLevels * kRN;    // 256 columns

// The digit-pair products of one chunk (two K steps of 16): A digit a against
// the stacked B digits 0 .. 7 - a (N = 32 (8 - a)), written from the column of
// level a on.  Issued by one thread.
__device__ __forceinline__ void rp_issue(uint32_t tmem, uint32_t ab, uint32_t bb, bool first) {
  const uint64_t da = tc::sw64_desc(ab), db = tc::sw64_desc(bb);
#pragma unroll
  for (int kk = 0; kk < kRN; kk += 16)
#pragma unroll
    for (int a = 0; a < oz::kLevels; ++a)
      tc::mma_f16(tmem + (uint32_t)(kRN * a), da + (uint64_t)((a * kAPanel + kk * 2) >> 4),
                  db + (uint64_t)((kk * 2) >> 4), tc::idesc(tc::F16, kM, kRN * (oz::kLevels - a)),
                  (kk == 0 && a == 0 && first) ? 0u : 1u);
}

struct OzPipe {
  uint64_t* bar;      // [2]: oz_run commits every batch to bar[0]; two batches in flight alternate bar[0] / bar[1]
  uint32_t tmem;
  uint32_t mph;       // bit b: parity of the next completion of bar[b] (the same in every thread)
  uint32_t mopen;     // issuing thread: bit b = a batch committed to bar[b] and not yet waited for
  int tid, q, g;
};

// Waits (bounded) for the MMA batch of chunk ch (committed to bar[ch & 1]).
__device__ __forceinline__ bool oz_wait_mma(OzPipe& P, int ch) {
  const uint32_t b = (uint32_t)ch & 1u;
  const bool ok = tc::mbar_wait(&P.bar[b], (P.mph >> b) & 1u);
  if (ok) {
    P.mph ^= 1u << b;
    P.mopen &= ~(1u << b);
  }
  return ok;
}

// Runs nchunks chunks through the two stages: produce(ch, a, b) writes the
// digit panels of chunk ch (A at a, B at b, each digit's panel contiguous
// after the previous one) while the MMAs of chunk ch - 1 run; the batch of
// chunk ch is issued once that of ch - 1 is done (all batches commit to
// bar[0]).  Level sums are added into hi / lo after every kGroupChunks chunks
// (the exactness limit of the FP32 level sums) and after the last.  Issuing
// the next batch before the previous one completes (two barriers) was measured
// about 1% slower in these kernels, whose production overlaps the MMAs anyway.
// False when a wait timed out (every thread returns false together).
template <class Produce>
__device__ __forceinline__ bool oz_run(OzPipe& P, unsigned char* smem, int nchunks, Produce&& produce, long long* hi,
                                       long long* lo) {
  for (int ch = 0; ch < nchunks; ++ch) {
    unsigned char* a = smem + (ch & 1) * kStage;
    unsigned char* b = a + oz::kSlices * kAPanel;
    produce(ch, a, b);   // this stage was last read by the MMAs of chunk ch - 2, already complete
    tc::fence_proxy_async();
    bool ok = true;
    if (ch > 0) ok = oz_wait_mma(P, 0);
    if (__syncthreads_or(!ok)) return false;
    if (ch > 0 && (ch - 1) % kGroupChunks == kGroupChunks - 1) {   // group closed at ch - 1
      tc::fence_after();
      oz_readout<false>(P.tmem, P.q, P.g, hi, lo);
      tc::fence_before();
      __syncthreads();
    }
    if (P.tid == 0) {
      tc::fence_after();
      oz_issue_chunk(P.tmem, tc::smem_u32(a), tc::smem_u32(b), ch % kGroupChunks == 0);
      tc::mma_commit(&P.bar[0]);
      P.mopen |= 1u;
    }
  }
  if (nchunks > 0) {
    const bool ok = oz_wait_mma(P, 0);
    if (__syncthreads_or(!ok)) return false;
    tc::fence_after();
    oz_readout<false>(P.tmem, P.q, P.g, hi, lo);
    tc::fence_before();
    __syncthreads();
  }
  return true;
}

// CTA prologue / epilogue shared by the kernels: TMEM (512 columns) and the
// two MMA barriers (bar: a __shared__ uint64_t[2]).
__device__ __forceinline__ OzPipe oz_begin(uint32_t* tmem_slot, uint64_t* bar) {
  const int tid = threadIdx.x, warp = tid >> 5;
  if (warp == 0) tc::tmem_alloc(tmem_slot, 512);
  if (tid == 0) {
    tc::mbar_init(&bar[0], 1);
    tc::mbar_init(&bar[1], 1);
    tc::mbar_fence_init();
  }
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  OzPipe P;
  P.bar = bar;
  P.tmem = *tmem_slot;
  P.mph = 0;
  P.mopen = 0;
  P.tid = tid;
  P.q = warp & 3;
  P.g = warp >> 2;
  return P;
}

__device__ __forceinline__ void oz_end(const OzPipe& P, bool abort, Ctl* ctl) {
  if (abort && P.tid == 0) {
    raise_level_status(ctl, ST_TIMEOUT);
    // MMA batches may still run: wait for them (bounded) before the TMEM is freed
    for (uint32_t b = 0; b < 2; ++b)
      if ((P.mopen >> b) & 1u) tc::mbar_wait(&P.bar[b], (P.mph >> b) & 1u, 1u << 20);
  }
  tc::fence_before();
  __syncthreads();
  if ((P.tid >> 5) == 0) tc::tmem_dealloc(P.tmem, 512);
}

__device__ __forceinline__ unsigned char* oz_smem(unsigned char* raw) {
  return reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(raw) + 1023) & ~uintptr_t(1023));
}

// One item's 128 x 64 partial (hi then lo, [column][row] so that a warp's
// stores are contiguous).
__device__ __forceinline__ void oz_store_partial(long long* out, int q, int g, int lane, const long long* hi,
                                                 const long long* lo) {
  const int il = q * 32 + lane;
#pragma unroll
  for (int c = 0; c < 16; ++c) {
    const int jl = g * 16 + c;
    out[jl * kM + il] = hi[c];
    out[kM * kN + jl * kM + il] = lo[c];
  }
}

__device__ __forceinline__ oz::I128 oz_sum_partials(const long long* part, int nslabs, size_t slab_stride, int il,
                                                    int jl) {
  oz::I128 acc{0, 0};
  for (int sl = 0; sl < nslabs; ++sl) {
    const long long* pp = part + (size_t)sl * slab_stride;
    oz::i128_add(acc, oz::i128_from_parts(pp[jl * kM + il], pp[kM * kN + jl * kM + il]));
  }
  return acc;
}

__device__ __forceinline__ double nan64() { return __longlong_as_double(0x7FF8000000000000ll); }

}  // namespace
}  // namespace mrcqr
