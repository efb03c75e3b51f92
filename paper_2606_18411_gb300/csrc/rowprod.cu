// The two row-block products of stage 2 in emulated FP64 on the FP16 tensor
// cores (ozaki.cuh): W = A R^{-1} (Algorithm 2 step 7, R = R_s upper
// triangular) and Q = W X (Algorithm 1 step 3, X = R_c^{-1} upper triangular).
//
// Both are one pass over 128-row blocks in output tiles of 32 columns:
//   out[:, tile t] = sum over K chunks of 32 columns of (chunk) * (32 x 32 multiplier block),
// FP64 result entries rounded once from the exact level sums.
//  * Q = W X, tiles right to left in place: chunk kc <= t of W against X[kc, t].
//  * W = A R^{-1}, tiles left to right: with X_t the inverse of the 32 x 32
//    diagonal block R_tt,
//      W_t = (A_t - W_{<t} R_{<t,t}) X_t = A_t X_t + W_{<t} Z_t,   Z_t = -R_{<t,t} X_t,
//    so the chunks are A_t (against X_t) and the W_kc already solved (against Z_t).
//    No FP64 arithmetic is left: this GPU issues FP64 at 1/64 rate, and the
//    16 x 16 substitutions that were here before kept its pipe busy for 55% of
//    the kernel at n = 64, while W was sliced again for every 16 columns.
//    Columns enter equilibrated: with F = diag(2^f_c), f_c the exponent of the
//    largest entry of column c of R, the kernel solves W (R F^{-1}) = A F^{-1},
//    the same W (powers of two are exact), so the digits of a row of A cover every
//    column whatever the columns' sizes.  The rows k of W enter scaled by 2^e_k, the
//    binade of the largest entry of row k of R F^{-1}, and Z_t by 2^-e_k, so a
//    graded R pairs balanced operands.
//    X_t = (R F^{-1})_tt^{-1} and Z_t are formed by k_rp_prep_r to 2^-61 of their
//    column maxima (an FP64 substitution corrected once with the residual
//    I - R_tt X_t in 128-bit integers), so the product's error is that of the
//    digits, about 2^-60 max|row| max|column| per entry.  Seen as a backward error
//    of A F^{-1} it is amplified by at most
//      amp = max_j sum_c max|column c of (Z_t; X_t)| |(R F^{-1})_tt[c][j]|,
//    and a panel whose amp exceeds 1024 keeps the substitution: the product is
//    W_{<t} (-R_{<t,t}) alone (A's digits are zeros in it), A_t is added and R_tt solved
//    with in FP64.  (Largest column error of 288 solves, n = 8 .. 64, two spectra, kappa
//    to 1e16, in units of u |W| |R|: amp below 256 0.7, 512 .. 1024 1.9, 1024 .. 2048 3.1,
//    2048 .. 4096 7.1; FP64 substitution 1.0.  Among R of sketched matrices with kappa of
//    1e12 and 1e16 17% pass 1024 at n = 32, 7% at 64, 1% at 100, in their first panels;
//    a kept panel costs about three of the others.)
//    F fits A where W's columns are of one size, as for a factor R of A.  Where R is
//    the caller's (mrcqr_trsm, mrcqr_cholqr_precond) a row block checks it: a panel with a
//    column of A F^{-1} that is zero or below 2^-10 of the largest entry of the block's A F^{-1}
//    or W D could lose that column's digits, and is solved by substitution as well.
//
// Measured at m = 2^20 (before: substitution blocks of 16 columns; Q = W X in
// 128 x 64 tiles by one CTA per SM): W = A R^{-1} 1.78 -> 0.75 ms at n = 64,
// 4.53 -> 1.80 at 128, 12.7 -> 5.9 at 256, 41.3 -> 20.5 at 512 (m = 300001,
// n = 320: 2.94 ms with one reference for all columns, 2.93 with the column
// scales, 2.99 with the check of an R of the caller's); Q = W X 0.99 -> 0.63 at
// n = 64, 2.19 -> 1.61 at 128 (wide W takes 64-column tiles: ozaki.cu, rp_wide).
// What bounds them is integer-pipe work around the products (slicing about 1100
// cycles per SM and chunk, conversion of the results about 2400 per tile, against
// 1340 of MMAs per chunk) and, with two CTAs per SM, the latency of a block's phases.
#include <climits>

#include "kernels.h"
#include "ozaki.cuh"
#include "ozaki_pipe.cuh"
#include "tc.cuh"

namespace mrcqr {

namespace {

// Two CTAs of 256 threads per SM, each with half the TMEM (8 level
// accumulators of 128 x 32): while one CTA's threads slice, read out or
// convert, the other's MMAs run.  A 128 x 64 tile per CTA would take 10% fewer
// MMA cycles and slice the chunk half as often, but holds all of TMEM and
// leaves the tensor cores idle in every other phase of a row block.
constexpr size_t kRSmem = (size_t)kRABytes + 2 * (size_t)kRBBytes + 1024;
constexpr int kNoEntry = -100000, kNonfinite = 100000;
constexpr float kAmpLimit = 1024.0f;
// Binades a column of A F^{-1} may lie below the block's largest entry: 2^-62 2^10 amp sqrt(n) stays at the n u of a
// triangular solve, and a matched R reaches 2^7 (largest of 128 n Gaussians times sqrt(n) against a column's largest).
constexpr int kBalance = 10;

// Multiplier block (t, kc), kc <= t.
__host__ __device__ __forceinline__ size_t rp_block_offset(int t, int kc) {
  return ((size_t)t * (t + 1) / 2 + kc) * kRBBytes;
}

__host__ __device__ __forceinline__ int rp_n32(int n) { return (n + kRN - 1) / kRN * kRN; }
__host__ __device__ __forceinline__ size_t rp_digit_size(int n) { return rp_block_offset(rp_n32(n) / kRN, 0); }

// The TRSM's integers: column exponents of the two multipliers, e_k, -f_c (n32 each) and the panel flags (16).
struct RpInts {
  int *colE, *colE2, *eR, *fN, *flags;
  __host__ __device__ __forceinline__ RpInts(int* p, int n)
      : colE(p), colE2(p + rp_n32(n)), eR(p + 2 * rp_n32(n)), fN(p + 3 * rp_n32(n)), flags(p + 4 * rp_n32(n)) {}
};

struct RpArgs {
  int64_t m;
  int n;
  const double* A;              // TRSM only
  int64_t lda;
  double* W;                    // TRSM: output; finalize: W in, Q out
  int64_t ldw;
  const int* colE;              // reference exponent of each multiplier column
  const unsigned char* Md;      // digit panels of the multiplier blocks
  const int* colE2;             // TRSM: the same for the panels that keep their substitution
  const unsigned char* Md2;
  const int* eR;                // TRSM: row scaling e_k
  const int* fN;                // TRSM: column scaling -f_c
  const int* flags;             // TRSM: 1 = the panel keeps its substitution
  const double* RT;             // TRSM: R transposed, row stride npad
  const double* rinv;
  uint32_t* colHiOut;           // column maxima of the result (high words), or null
};

struct RpCta {
  unsigned char* as;            // digits of the chunk
  unsigned char* bs;            // two stages of multiplier digits
  uint64_t* bar;                // [0]: MMA batches; [1], [2]: multiplier stages
  uint32_t tmem;
  uint32_t commits;             // MMA batches committed (the same in every thread)
  uint32_t bseq;                // multiplier blocks consumed (the same in every thread)
  int* dead;                    // a bounded wait gave up
  int* rowX;                    // TRSM: running maximum exponent of W D per row
  int* rowRef;                  // reference exponent of each row for the current tile
  int (*red)[kM];               // [2][128]
  int* eRs;                     // e_k, padded to 512
  int* fNs;                     // -f_c, padded to 512
  uint32_t* fKs;                // (1024 - f_c) << 20: added to a high word it orders |A F^-1|, without overflow
  uint32_t* cmax;               // column maxima of the result over this CTA's rows
  int* colE;                    // reference exponents of the multiplier columns
  int* emax;                    // largest of the scalings e_k, -f_c and 0
  uint32_t* keep;               // bit t: panel t keeps its substitution
  int* rho;                     // checked solve: largest rowRef of each 32 rows
  uint32_t* mask;               // [2] columns 16 h .. of the panel with an entry near it
};

__device__ __forceinline__ void rp_wait(RpCta& S, uint64_t* bar, uint32_t parity) {
  if (*(volatile int*)S.dead) return;
  if (!tc::mbar_wait(bar, parity, 1u << 20)) *(volatile int*)S.dead = 1;
}

// Starts the copy of multiplier block (t, kc) from Md into stage seq & 1.
__device__ __forceinline__ void rp_fetch_b(const unsigned char* Md, RpCta& S, uint32_t seq, int t, int kc) {
  uint64_t* bar = &S.bar[1 + (seq & 1u)];
  tc::mbar_expect_tx(bar, kRBBytes);
  tc::bulk_load(S.bs + (seq & 1u) * kRBBytes, Md + rp_block_offset(t, kc), kRBBytes, bar);
}

// Slicing of sixteen values of one row into digits: four groups of four
// adjacent columns, group j at the shared address as + off[j] (8 bytes in each digit panel).
// es: the groups' column scalings in shared memory (null: none), at 4-integer
// granules eg[j]; cr = 31 - Eref, or a large negative number that forces the general
// form.  Straight-line code with one range check at the end: values below
// 2^-31 of the reference, zeros and subnormals make the thread write all its
// digits again from biased_fixed63.
__device__ __forceinline__ void rp_slice(const double (&v)[4][4], const int* es, const uint32_t (&eg)[4], int Eref,
                                         int cr, uint32_t as, const uint32_t (&off)[4]) {
  uint32_t kor = 0u;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int4 e = es ? *reinterpret_cast<const int4*>(es + eg[j]) : make_int4(0, 0, 0, 0);
    const int eo[4] = {e.x, e.y, e.z, e.w};
    uint32_t o[2][oz::kSlices];
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      uint32_t h[2], Jh[2], Jl[2];
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        h[k] = (uint32_t)__double2hiint(v[j][2 * p + k]);
        oz::fixed63_fast(h[k], (uint32_t)__double2loint(v[j][2 * p + k]), cr + eo[2 * p + k], Jh[k], Jl[k], kor);
      }
      oz::digits8_pack(Jh[0], Jl[0], Jh[1], Jl[1], h[0], h[1], o[p]);
    }
#pragma unroll
    for (int a = 0; a < oz::kSlices; ++a)
      tc::st_shared2(as + off[j] + a * kAPanel, o[0][a], o[1][a]);
  }
  if (kor > 31u) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int4 e = es ? *reinterpret_cast<const int4*>(es + eg[j]) : make_int4(0, 0, 0, 0);
      oz_store_pair(v[j][0], v[j][1], 0u, 0u, Eref, as + off[j], kAPanel, e.x, e.y);
      oz_store_pair(v[j][2], v[j][3], 0u, 0u, Eref, as + off[j] + 4, kAPanel, e.z, e.w);
    }
  }
}

// Per-problem state of a CTA: the scalings, the kept panels, the column maxima.
template <bool kTrsm>
__device__ __forceinline__ void rp_begin(const RpArgs& a, RpCta& S) {
  __syncthreads();
  if (threadIdx.x == 0) {
    *S.emax = 0;
    *S.keep = 0u;
  }
  __syncthreads();
  for (int k = threadIdx.x; k < 512; k += kRThreads) {
    S.cmax[k] = 0u;
    if (!kTrsm) S.colE[k] = k < a.n ? a.colE[k] : 0;
    if (kTrsm) {
      const int e = k < a.n ? a.eR[k] : 0, f = k < a.n ? a.fN[k] : 0;
      const int E1 = k < a.n ? a.colE[k] : 0, E2 = k < a.n ? a.colE2[k] : 0;   // loads side by side
      const bool keep = k < a.n && a.flags[k / kRN] != 0;
      S.colE[k] = keep ? E2 : E1;
      S.eRs[k] = e;
      S.fNs[k] = f;
      S.fKs[k] = (uint32_t)(f + 1024) << 20;
      if (max(e, f) > 0) atomicMax(S.emax, max(e, f));
      if (keep && k % kRN == 0) atomicOr(S.keep, 1u << (k / kRN));
    }
  }
  __syncthreads();
}

__device__ __forceinline__ void rp_end(const RpArgs& a, RpCta& S) {
  __syncthreads();
  if (a.colHiOut)
    for (int k = threadIdx.x; k < a.n; k += kRThreads)
      if (S.cmax[k]) atomicMax(a.colHiOut + k, S.cmax[k]);
  __syncthreads();
}

// Solves the w x w diagonal block (w = 32, less in the last panel: R has n rows)
// of a panel that keeps its substitution: sb[c][row] holds B = A_t - W_{<t} R_{<t,t}
// and receives B R_tt^{-1} in its first w columns.
__device__ __noinline__ void rp_substitute(const RpArgs& a, double* sb, int c0, int row) {
  const int npad = (a.n + 31) / 32 * 32, w = min(kRN, a.n - c0);
  for (int h = 0; h < kRN; h += 16) {   // half a row in registers: a whole one takes them from the kernel's hot path
    double b[16];
#pragma unroll
    for (int c = 0; c < 16; ++c) b[c] = sb[(h + c) * kM + row];
    const double* r0 = a.RT + (int64_t)c0 * npad + c0 + h;
#pragma unroll 1
    for (int c = 0; c < h && c < w; ++c) {
      const double x = sb[c * kM + row];
#pragma unroll
      for (int c2 = 0; c2 < 16; ++c2) b[c2] = fma(-x, __ldg(r0 + (int64_t)c * npad + c2), b[c2]);
    }
#pragma unroll
    for (int c = 0; c < 16; ++c)
      if (h + c < w) {
        const double x = b[c] * a.rinv[c0 + h + c];
        b[c] = x;
        const double* r = r0 + (int64_t)(h + c) * npad;
#pragma unroll
        for (int c2 = c + 1; c2 < 16; ++c2) b[c2] = fma(-x, __ldg(r + c2), b[c2]);
      }
#pragma unroll
    for (int c = 0; c < 16; ++c) sb[(h + c) * kM + row] = b[c];
  }
}

// A row with a non-finite entry of A in the panel at c0: columns cb .. cb + 15 of the panel by FP64 substitution along
// the row, into sb[c kM], so that the columns before the entry are those of the finite row.
__device__ __noinline__ void rp_solve_row(const RpArgs& a, double* sb, int64_t row, int c0, int cb) {
  const int npad = rp_n32(a.n);
  double x[kRN];
  for (int c = 0; c < cb + 16; ++c) {
    x[c] = 0.0;
    if (c0 + c < a.n) {
      const double* r = a.RT + c0 + c;
      double v = a.A[row + (int64_t)(c0 + c) * a.lda];
      for (int k = 0; k < c0; ++k) v = fma(-a.W[row + (int64_t)k * a.ldw], r[(int64_t)k * npad], v);
      for (int k = 0; k < c; ++k) v = fma(-x[k], r[(int64_t)(c0 + k) * npad], v);
      x[c] = v * a.rinv[c0 + c];
    }
    if (c >= cb) sb[c * kM] = x[c];
  }
}

// Checked solve: the exponent that every column of A F^{-1} in the panel should reach in the row block (kAllZero:
// neither A nor W D has an entry).
constexpr int kAllZero = -4000;
__device__ __forceinline__ int rp_threshold(const RpCta& S) {
  return max(max(max(S.rho[0], S.rho[1]), max(S.rho[2], S.rho[3])) - kBalance, kAllZero);
}

// Whether every column of the panel at c0 has an entry near the block's largest
// (every thread); a column of zeros has none: W there is as large as the
// others make it, which nothing here bounds.  The full look, for panels where
// the first 32 rows do not show it.
__device__ __noinline__ bool rp_balanced_full(const RpArgs& a, const int* fNs, uint32_t* mask, int thr, int64_t r0,
                                              int c0) {
  const int tid = threadIdx.x, pr = tid & (kM - 1), ph = tid >> 7;
  __syncthreads();
  if (tid < 2) mask[tid] = 0u;
  __syncthreads();
  const double* p = a.A + min(r0 + pr, a.m - 1) + (int64_t)(c0 + 16 * ph) * a.lda;
  uint32_t near = 0u;
  for (int c = 0; c < 16; ++c, p += a.lda) {
    if (c0 + 16 * ph + c >= a.n) {   // beyond the last panel's columns
      near |= 0xFFFFu << c & 0xFFFFu;
      break;
    }
    const uint32_t h = (uint32_t)__double2hiint(*p) & 0x7FFFFFFFu;
    if (h != 0u && h < 0x7FF00000u && (int)(h >> 2) + fNs[c0 + 16 * ph + c] * (1 << 18) >= thr) near |= 1u << c;
  }
  near = __reduce_or_sync(0xffffffffu, near);
  if ((tid & 31) == 0) atomicOr(&mask[ph], near);
  __syncthreads();
  return (mask[0] & mask[1]) == 0xFFFFu;
}

__device__ __forceinline__ bool rp_balanced(const RpArgs& a, const RpCta& S, int64_t r0, int c0) {
  const uint32_t all = min(kRN, a.n - c0) == kRN ? 0xFFFFFFFFu : (1u << (a.n - c0)) - 1u;
  const int thr = rp_threshold(S);
  return thr == kAllZero || ((S.mask[0] | S.mask[1] << 16) & all) == all ||
         rp_balanced_full(a, S.fNs, S.mask, thr * (1 << 18), r0, c0);
}

// One block of 128 rows from r0; the CTA's next block is `next` blocks further (0: unknown).  False when a wait
// gave up (every thread).
// kMulti: K may exceed 128 (n > 128), so the level sums are read out and added up several times per tile; else the
// sums of a tile are live only after its last chunk, which leaves the slicing their 64 registers.
// kCheck: the row block decides by its own A whether a panel keeps its substitution (top of the file).
template <bool kTrsm, bool kMulti, bool kCheck>
__device__ __forceinline__ bool rp_block(const RpArgs& a, RpCta& S, int64_t r0, int next) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n = a.n, nt = (n + kRN - 1) / kRN;
  const int pr = tid & (kM - 1), ph = tid >> 7;      // producer: row pr, columns 16 ph .. 16 ph + 15 of the chunk
  const int rot = (lane >> 3) & 1;                   // rows r and r + 8 store the two halves of a 16-byte chunk in
                                                     // opposite order: a half warp's 8-byte stores cover all banks
  const int q = warp & 3, g = warp >> 2;             // readout: rows 32 q + lane, columns 16 g .. 16 g + 15
  const int rr = q * 32 + lane;
  const bool rlive = r0 + rr < a.m;
  double v[4][4];
  uint32_t gcol[4], off[4];   // the thread's four groups of four columns and their panel offsets
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    gcol[j] = (uint32_t)(16 * ph + 8 * (j >> 1) + 4 * ((j & 1) ^ rot));
    off[j] = tc::sw64_offset(pr, (int)gcol[j], 2);
  }
  // rows beyond m read row m - 1 again (their results are not stored)
  const int64_t prow = min(r0 + pr, a.m - 1);
  auto load = [&](const double* X, int64_t ldx, int k0) {   // columns k0 .. k0 + 31, zero beyond n
    const double* base = X + prow + (int64_t)k0 * ldx;
    if (k0 + kRN <= n) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const double* p = base + (int64_t)gcol[j] * ldx;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          v[j][c] = *p;
          p += ldx;
        }
      }
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const double* p = base + (int64_t)gcol[j] * ldx;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          v[j][c] = k0 + (int)gcol[j] + c < n ? *p : 0.0;
          p += ldx;
        }
      }
    }
  };
  {   // the CTA's next row block of the input into L2: this kernel has no registers left to load it ahead
    const int64_t rn = r0 + (int64_t)kM * next;
    if (next && rn < a.m) {
      const double* X = kTrsm ? a.A : a.W;
      const int64_t ldx = kTrsm ? a.lda : a.ldw;
      for (int e = tid; e < 8 * n; e += kRThreads)
        tc::prefetch_l2(X + min(rn + 16 * (e & 7), a.m - 1) + (int64_t)(e >> 3) * ldx);
    }
  }
  if (!kTrsm) {   // row reference exponents over all n columns of W
    uint32_t mx = 0u;
    const double* p = a.W + prow + (int64_t)ph * a.ldw;
#pragma unroll 16
    for (int c = ph; c < n; c += 2) {
      mx = max(mx, (uint32_t)__double2hiint(*p) & 0x7FFFFFFFu);
      p += 2 * a.ldw;
    }
    S.red[ph][pr] = (int)mx;
    __syncthreads();
    if (tid < kM) {
      const int E = (int)oz::exp_field((uint32_t)max(S.red[0][tid], S.red[1][tid]));
      S.rowRef[tid] = E == 2047 ? kNonfinite : E == 0 ? kNoEntry : E;
    }
  } else if (tid < kM) {
    S.rowX[tid] = kNoEntry;
  }
  __syncthreads();
  const uint32_t tbase = S.tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(g * 16);
  bool pending = false;
  if (tid == 0) rp_fetch_b(a.Md, S, S.bseq, kTrsm ? 0 : nt - 1, 0);
  for (int ti = 0; ti < nt; ++ti) {
    const int t = kTrsm ? ti : nt - 1 - ti;
    const int c0 = t * kRN;
    bool keep = kTrsm && ((*S.keep >> t) & 1u) != 0u;
    if (kTrsm) {   // the rows' reference exponents: W D so far and A_t F^{-1} (W D alone in a kept panel)
      load(a.A, a.lda, c0);
      uint32_t mx = 0u, mk = 0u;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint4 f4 = *reinterpret_cast<const uint4*>(S.fKs + c0 + gcol[j]);
        const uint32_t f[4] = {f4.x, f4.y, f4.z, f4.w};
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const uint32_t h = (uint32_t)__double2hiint(v[j][c]) & 0x7FFFFFFFu;
          mx = max(mx, h);
          mk = max(mk, h + f[c]);
          if (keep) v[j][c] = 0.0;
        }
      }
      if ((int)(mk >> 20) - 1024 <= *S.emax && mx != 0u) {   // no entry's exponent, or a zero's 0 - f_c: without zeros
        mk = 0u;
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const uint32_t h = (uint32_t)__double2hiint(v[j][c]) & 0x7FFFFFFFu;
            if (h != 0u) mk = max(mk, h + S.fKs[c0 + gcol[j] + c]);
          }
      }
      S.red[ph][pr] = keep || mx == 0u ? kNoEntry : mx >= 0x7FF00000u ? kNonfinite : (int)(mk >> 20) - 1024;
      __syncthreads();
      if (tid < kM) {
        const int E = max(S.rowX[tid], max(S.red[0][tid], S.red[1][tid]));
        S.rowRef[tid] = E;
        if (kCheck) {
          const int rho = __reduce_max_sync(0xffffffffu, E != kNonfinite ? E : kNoEntry);
          if (lane == 0) S.rho[warp] = rho;
        }
      }
      __syncthreads();
      if (kCheck && (warp & 3) == 0) {   // do 32 rows show every column near the block's largest entry?
        const int thr = rp_threshold(S) * (1 << 18);
        uint32_t mask = 0u;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int4 f4 = *reinterpret_cast<const int4*>(S.fNs + c0 + gcol[j]);
          const int f[4] = {f4.x, f4.y, f4.z, f4.w};
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const uint32_t h = (uint32_t)__double2hiint(v[j][c]) & 0x7FFFFFFFu;
            if (h < 0x7FF00000u && (int)(h >> 2) + f[c] * (1 << 18) >= thr) mask |= 1u << (4 * j + c);
          }
        }
        if (rot) mask = (mask & 0x0F0Fu) << 4 | ((mask >> 4) & 0x0F0Fu);   // from the lane's order to the columns'
        mask = __reduce_or_sync(0xffffffffu, mask);
        if (lane == 0) S.mask[ph] = mask;
      }
    } else {
      load(a.W, a.ldw, 0);
    }
    int Eref = S.rowRef[pr];
    // constant of the fast slicing; a reference so small that a zero's exponent field could pass for a
    // value's takes the general form throughout
    int cr = Eref - *S.emax > 31 ? 31 - Eref : -(1 << 30);
    long long hi[16], lo[16];
    if (kMulti) {
#pragma unroll
      for (int c = 0; c < 16; ++c) hi[c] = lo[c] = 0;
    }
    for (int i = 0; i <= t; ++i) {
      if (pending) rp_wait(S, &S.bar[0], (S.commits - 1) & 1u);   // the chunk's panels are free
      pending = false;
      const uint32_t stage = S.bseq & 1u, bpar = (S.bseq >> 1) & 1u;
      if (tid == 0) {   // the next multiplier block, into the stage that the finished batch read
        if (i < t) {
          if (!(kCheck && i == 0)) rp_fetch_b(keep ? a.Md2 : a.Md, S, S.bseq + 1, t, kTrsm ? i : i + 1);
        } else if (ti + 1 < nt) {
          rp_fetch_b(a.Md, S, S.bseq + 1, kTrsm ? t + 1 : t - 1, kTrsm ? t + 1 : 0);
        }
      }
      const int kW = kTrsm ? i - 1 : i;   // W chunk (TRSM: -1 is A_t)
      rp_slice(v, !kTrsm ? nullptr : i > 0 ? S.eRs + kRN * kW : S.fNs + c0, gcol, Eref, cr, tc::smem_u32(S.as), off);
      tc::fence_proxy_async();
      tc::fence_before();
      __syncthreads();
      if (kCheck && i == 0 && !keep && !rp_balanced(a, S, r0, c0)) {   // uniform: A's digits are zeros after all
        keep = true;
        if (tid < kM) S.rowRef[tid] = S.rowX[tid];
        if (tid < kRN && c0 + tid < n) S.colE[c0 + tid] = a.colE2[c0 + tid];
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int c = 0; c < 4; ++c) v[j][c] = 0.0;
        __syncthreads();
        Eref = S.rowRef[pr];
        cr = Eref - *S.emax > 31 ? 31 - Eref : -(1 << 30);
        rp_slice(v, nullptr, gcol, Eref, cr, tc::smem_u32(S.as), off);
        tc::fence_proxy_async();
        __syncthreads();
      }
      if (tid == 0) {
        if (kCheck && i == 0 && t > 0) rp_fetch_b(keep ? a.Md2 : a.Md, S, S.bseq + 1, t, 0);   // the panel's way is known
        rp_wait(S, &S.bar[1 + stage], bpar);
        tc::fence_after();
        rp_issue(S.tmem, tc::smem_u32(S.as), tc::smem_u32(S.bs + stage * kRBBytes), kMulti ? i % kGroupChunks == 0 : i == 0);
        tc::mma_commit(&S.bar[0]);
      }
      ++S.commits;
      ++S.bseq;
      pending = true;
      const bool group_end = kMulti && i < t && i % kGroupChunks == kGroupChunks - 1;
      if (i < t && !group_end) load(a.W, a.ldw, kRN * (kW + 1));
      if (group_end) {   // at most 128 terms per level sum: exact in FP32
        rp_wait(S, &S.bar[0], (S.commits - 1) & 1u);
        pending = false;
        tc::fence_after();
        oz_readout_cols<kRN, false>(tbase, hi, lo);
        tc::fence_before();
        load(a.W, a.ldw, kRN * (kW + 1));
      }
    }
    rp_wait(S, &S.bar[0], (S.commits - 1) & 1u);
    pending = false;
    tc::fence_after();
    if (!kMulti) {
#pragma unroll
      for (int c = 0; c < 16; ++c) hi[c] = lo[c] = 0;
    }
    oz_readout_cols<kRN, false>(tbase, hi, lo);
    tc::fence_before();
    // the tile: one rounding per entry
    const int Erow = S.rowRef[rr];
    double out[16];
#pragma unroll
    for (int c = 0; c < 16; ++c) {
      const int ce = S.colE[c0 + 16 * g + c];
      out[c] = (c & 1) ? oz::t96_to_double_fp64(hi[c], lo[c], Erow + ce - oz::kScaleBias)
                       : oz::t96_to_double(hi[c], lo[c], Erow + ce - oz::kScaleBias);
      if (ce == kNonfinite) out[c] = nan64();
    }
    if (Erow == kNonfinite) {
#pragma unroll
      for (int c = 0; c < 16; ++c) out[c] = nan64();
    }
    double* sb = reinterpret_cast<double*>(S.as);     // the chunk's panels are free
    if (kTrsm && !keep && rlive && max(S.red[0][rr], S.red[1][rr]) == kNonfinite) {   // in both threads of the row
      rp_solve_row(a, sb + rr, r0 + rr, c0, 16 * g);
#pragma unroll
      for (int c = 0; c < 16; ++c) out[c] = sb[(16 * g + c) * kM + rr];
    }
    if (keep) {
#pragma unroll
      for (int c = 0; c < 16; ++c)
        if (c0 + 16 * g + c < n)
          sb[(16 * g + c) * kM + rr] = a.A[min(r0 + rr, a.m - 1) + (int64_t)(c0 + 16 * g + c) * a.lda] + out[c];
      __syncthreads();
      if (tid < kM) rp_substitute(a, sb, c0, tid);
      __syncthreads();
#pragma unroll
      for (int c = 0; c < 16; ++c) out[c] = sb[(16 * g + c) * kM + rr];
    }
    // stores, column maxima (a shared atomic only where a new maximum appears: after a CTA's first
    // blocks hardly ever) and the rows' running maxima of W D
    if (rlive) {
      double* wp = a.W + r0 + rr + (int64_t)(c0 + 16 * g) * a.ldw;
      uint32_t* cm = S.cmax + c0 + 16 * g;
      const int* er = S.eRs + c0 + 16 * g;
      uint32_t mxh = 0u, mk = 0u;
#pragma unroll
      for (int c = 0; c < 16; ++c) {
        if (c0 + 16 * g + c < n) {
          *wp = out[c];
          const uint32_t h = (uint32_t)__double2hiint(out[c]) & 0x7FFFFFFFu;
          if (h > cm[c]) atomicMax(cm + c, h);
          if (kTrsm) {
            mxh = max(mxh, h);
            mk = max(mk, (h | 0x80000000u) + ((uint32_t)er[c] << 20));   // exponent + e_k + 2048 (e_k <= 0: no overflow)
          }
        }
        wp += a.ldw;
      }
      if (kTrsm && mxh != 0u) {
        // zeros do not count: with e_k over more than 2^1000 a zero's 0 + e_k could pass every entry's exponent
        if (mk >> 20 <= 2048u) {
          mk = 0u;
#pragma unroll
          for (int c = 0; c < 16; ++c) {
            const uint32_t h = (uint32_t)__double2hiint(out[c]) & 0x7FFFFFFFu;
            if (c0 + 16 * g + c < n && h != 0u) mk = max(mk, (h | 0x80000000u) + ((uint32_t)er[c] << 20));
          }
        }
        atomicMax(&S.rowX[rr], mxh >= 0x7FF00000u ? kNonfinite : (int)(mk >> 20) - 2048);
      }
    }
    if (__syncthreads_or(*(volatile int*)S.dead)) return false;   // the tile's W is visible to the next tile's loads
    if (kCheck && keep && ((*S.keep >> t) & 1u) == 0u && tid < kRN && c0 + tid < n) S.colE[c0 + tid] = a.colE[c0 + tid];
  }
  return true;
}

#define MRCQR_RP_CTA(S)                                                        \
  extern __shared__ unsigned char smem_raw[];                                  \
  __shared__ __align__(8) uint64_t bars_s[3];                                  \
  __shared__ uint32_t tmem_slot;                                               \
  __shared__ int dead_s, emax_s;                                               \
  __shared__ uint32_t keep_s;                                                  \
  __shared__ int rho_s[kM / 32];                                               \
  __shared__ uint32_t mask_s[2];                                               \
  __shared__ int rowX_s[kM];                                                   \
  __shared__ int rowRef_s[kM];                                                 \
  __shared__ int red_s[2][kM];                                                 \
  __shared__ __align__(16) int eRs_s[512];                                     \
  __shared__ __align__(16) int fNs_s[512];                                     \
  __shared__ __align__(16) uint32_t fKs_s[512];                                \
  __shared__ __align__(16) uint32_t cmax_s[512];                               \
  __shared__ __align__(16) int colE_s[512];                                             \
  if ((threadIdx.x >> 5) == 0) tc::tmem_alloc(&tmem_slot, kRTmem);             \
  if (threadIdx.x == 0) {                                                      \
    for (int b = 0; b < 3; ++b) tc::mbar_init(&bars_s[b], 1);                  \
    tc::mbar_fence_init();                                                     \
    dead_s = 0;                                                                \
  }                                                                            \
  tc::fence_before();                                                          \
  __syncthreads();                                                             \
  tc::fence_after();                                                           \
  RpCta S;                                                                     \
  S.as = oz_smem(smem_raw);                                                    \
  S.bs = S.as + kRABytes;                                                      \
  S.bar = bars_s;                                                              \
  S.tmem = tmem_slot;                                                          \
  S.commits = 0;                                                               \
  S.bseq = 0;                                                                  \
  S.dead = &dead_s;                                                            \
  S.rowX = rowX_s;                                                             \
  S.rowRef = rowRef_s;                                                         \
  S.red = red_s;                                                               \
  S.eRs = eRs_s;                                                               \
  S.fNs = fNs_s;                                                               \
  S.fKs = fKs_s;                                                               \
  S.cmax = cmax_s;                                                             \
  S.colE = colE_s;                                                             \
  S.emax = &emax_s;                                                            \
  S.keep = &keep_s;                                                            \
  S.rho = rho_s;                                                               \
  S.mask = mask_s;

// Every batch and every copy has been waited for unless a wait gave up; then
// the outstanding ones get one more bounded wait before the TMEM is freed.
__device__ __forceinline__ void rp_cta_end(RpCta& S, bool abort, Ctl* ctl) {
  if (abort && threadIdx.x == 0) {
    if (ctl) raise_level_status(ctl, ST_TIMEOUT);
    if (S.commits) tc::mbar_wait(&S.bar[0], (S.commits - 1) & 1u, 1u << 20);
    tc::mbar_wait(&S.bar[1 + (S.bseq & 1u)], (S.bseq >> 1) & 1u, 1u << 14);
  }
  tc::fence_before();
  __syncthreads();
  if ((threadIdx.x >> 5) == 0) tc::tmem_dealloc(S.tmem, kRTmem);
}

template <bool kTrsm, bool kMulti, bool kCheck>
__global__ void __launch_bounds__(kRThreads, 2) k_rowprod(RpArgs a, Ctl* ctl, int level) {
  if (level_inactive(ctl, level) || ctl->lvl_status != 0) return;
  MRCQR_RP_CTA(S)
  rp_begin<kTrsm>(a, S);
  bool abort = false;
  const int64_t nblocks = (a.m + kM - 1) / kM;
  for (int64_t rb = blockIdx.x; rb < nblocks; rb += gridDim.x)
    if (!rp_block<kTrsm, kMulti, kCheck>(a, S, rb * kM, (int)gridDim.x)) {
      abort = true;
      break;
    }
  if (!abort) rp_end(a, S);
  rp_cta_end(S, abort, ctl);
}

// ---------------------------------------------------------------------------
// Multiplier digits of Q = W X: column j of X against the exponent of its
// maximum.  XT[k][j] = X[k][j], row stride npad; one block per column.
__device__ __forceinline__ void rp_prep_x_col(int n, int npad, const double* __restrict__ XT, int* __restrict__ colE,
                                              unsigned char* __restrict__ Md, uint32_t* __restrict__ colHiOut, int nhi,
                                              int j, uint32_t* red) {
  if (colHiOut && j == 0)     // the product folds the column maxima of Q into these
    for (int i = threadIdx.x; i < nhi; i += blockDim.x) colHiOut[i] = 0u;
  __syncthreads();
  uint32_t mx = 0u;
  for (int k = threadIdx.x; k < n; k += blockDim.x)
    if (j < n) mx = max(mx, (uint32_t)__double2hiint(XT[(int64_t)k * npad + j]) & 0x7FFFFFFFu);
  mx = __reduce_max_sync(0xffffffffu, mx);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
  __syncthreads();
  uint32_t all = 0u;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) all = max(all, red[w]);
  const int E = (int)oz::exp_field(all);
  if (threadIdx.x == 0 && j < n) colE[j] = E == 2047 ? kNonfinite : E;
  const int t = j / kRN, jr = j % kRN;
  for (int k = threadIdx.x; k < kRN * (t + 1); k += blockDim.x) {
    int d[oz::kSlices];
    const double v = (k < n && j < n) ? XT[(int64_t)k * npad + j] : 0.0;
    oz::digits8((uint32_t)__double2hiint(v), (uint32_t)__double2loint(v), E, d);
    unsigned char* panel = Md + rp_block_offset(t, k / kRN) + tc::sw64_offset(jr, k % kRN, 2);
#pragma unroll
    for (int b = 0; b < oz::kSlices; ++b)
      *reinterpret_cast<__half*>(panel + b * kRBPanel) = __float2half_rn(oz::small_int_to_float(d[b]));
  }
}

__global__ void __launch_bounds__(128) k_rp_prep_x(int n, int npad, const double* __restrict__ XT, int* __restrict__ colE,
                                                   unsigned char* __restrict__ Md, uint32_t* __restrict__ colHiOut,
                                                   int nhi, const Ctl* ctl, int level) {
  if (level_inactive(ctl, level) || ctl->lvl_status != 0) return;
  __shared__ uint32_t red[4];
  rp_prep_x_col(n, npad, XT, colE, Md, colHiOut, nhi, blockIdx.x, red);
}

// ---------------------------------------------------------------------------
// -f_c = minus the unbiased exponent of the largest finite |R[k][c]| (0 for a zero
// column), so that no entry of R F^{-1} reaches 2 and e_k <= 0; 32 columns by the
// block's 256 threads; red: [8][32].
__device__ __forceinline__ uint32_t rp_finite_hi(double x) {   // |x|'s high word, 0 for a non-finite x
  const uint32_t h = (uint32_t)__double2hiint(x) & 0x7FFFFFFFu;
  return h < 0x7FF00000u ? h : 0u;
}

__device__ __forceinline__ void rp_col_scale_block(int n, int npad, const double* __restrict__ RT, int* fN, int blk,
                                                   int (*red)[kRN]) {
  const int lane = threadIdx.x & 31, g = threadIdx.x >> 5, c = kRN * blk + lane;
  uint32_t mx = 0u;
  if (c < n)
#pragma unroll 8
    for (int k = g; k <= c; k += 8) mx = max(mx, rp_finite_hi(RT[(int64_t)k * npad + c]));
  __syncthreads();
  red[g][lane] = (int)mx;
  __syncthreads();
  if (g == 0 && c < n) {
    int all = 0;
    for (int w = 0; w < 8; ++w) all = max(all, red[w][lane]);
    const int E = (int)oz::exp_field((uint32_t)all);
    fN[c] = E == 0 ? 0 : 1023 - E;
  }
}

__global__ void __launch_bounds__(256) k_rp_col_scale(int n, int npad, const double* __restrict__ RT, int* fN,
                                                      const Ctl* ctl, int level) {
  if (level_inactive(ctl, level) || ctl->lvl_status != 0) return;
  __shared__ int red[8][kRN];
  rp_col_scale_block(n, npad, RT, fN, blockIdx.x, red);
}

// e_k = unbiased exponent of max_c |R[k][c]| 2^-f_c (0 for a zero or non-finite
// row).  One warp per row.
__device__ __forceinline__ void rp_row_scale_block(int n, int npad, const double* __restrict__ RT, const int* fN, int* eR,
                                                   int blk) {
  const int k = blk * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (k >= n) return;
  uint32_t mx = 0u;
  int me = INT_MIN;
  for (int c = lane; c < n; c += 32) {
    const uint32_t h = (uint32_t)__double2hiint(RT[(int64_t)k * npad + c]) & 0x7FFFFFFFu;
    mx = max(mx, h);
    if (h >= 0x00100000u) me = max(me, (int)(h >> 20) + fN[c]);
  }
  mx = __reduce_max_sync(0xffffffffu, mx);
  me = __reduce_max_sync(0xffffffffu, me);
  if (lane == 0) eR[k] = (mx >= 0x7FF00000u || me == INT_MIN) ? 0 : me - 1023;
}

__global__ void __launch_bounds__(256) k_rp_row_scale(int n, int npad, const double* __restrict__ RT, const int* fN,
                                                      int* eR, const Ctl* ctl, int level) {
  if (level_inactive(ctl, level) || ctl->lvl_status != 0) return;
  rp_row_scale_block(n, npad, RT, fN, eR, blockIdx.x);
}

// Multiplier digits of a 32-column panel t of W = A R^{-1} (top of the file);
// one CTA of 256 threads per panel.  All sums of products of R and X run in
// 128-bit integers (their 64 x 64-bit products are integer-pipe work; the
// same in double-double would be eight times the instructions of the 1/64-rate
// FP64 pipe).
struct RpPrep {
  double R[kRN][kRN + 1];       // (R F^{-1})_tt (identity beyond column n)
  double X[kRN][kRN + 1];       // its inverse in FP64
  float F[kRN][kRN + 1];        // I - R_tt X (scaled)
  long long Ri[kRN][kRN + 1];   // a block of R in fixed point, row k against er[k]
  long long Xi[kRN][kRN + 1];   // X in fixed point, column c against Ex[c]
  int er[kRN], Ex[kRN], cE[kRN];
  int fN[kRpOwnScale];
  double rinv[kRN];             // 1 / diagonal of the scaled panel
  int red[8][kRN];
};

// Signed 63-bit fixed point of x 2^eoff against the exponent E: x 2^(eoff + 1085 - E).
__device__ __forceinline__ long long rp_fix(double x, int E, int eoff = 0) {
  const uint32_t h = (uint32_t)__double2hiint(x);
  const long long v =
      (long long)(oz::biased_fixed63(h, (uint32_t)__double2loint(x), E, eoff) - 0x0080808080808080ull);
  return (h >> 31) ? -v : v;
}

// 2^e for -1023 <= e <= 1022.
__device__ __forceinline__ double rp_pow2(int e) {
  return e > -1023 ? __hiloint2double((e + 1023) << 20, 0) : __hiloint2double(0x00080000, 0);
}

// Index of the leading bit of |v|, -1 for zero.
__device__ __forceinline__ int rp_msb(__int128 v) {
  const unsigned __int128 u = v < 0 ? -(unsigned __int128)v : (unsigned __int128)v;
  const uint64_t h = (uint64_t)(u >> 64), l = (uint64_t)u;
  return h ? 127 - __clzll((long long)h) : l ? 63 - __clzll((long long)l) : -1;
}

// The block of R F^{-1} at (rows 32 kc .., columns of panel t; f: -f_c of this
// thread's column) in fixed point, its row references in er (over finite
// entries).  True if an entry is not finite.
__device__ __forceinline__ bool rp_load_fixed(RpPrep& P, int n, int npad, const double* __restrict__ RT, int kc, int c0,
                                              int f) {
  const int c = threadIdx.x & 31, g = threadIdx.x >> 5;
  bool bad = false;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int k = 4 * g + r;
    double x = c0 + c < n ? RT[(int64_t)(kRN * kc + k) * npad + c0 + c] : 0.0;
    int E = (int)oz::exp_field((uint32_t)__double2hiint(x));
    if (E == 2047) {
      bad = true;
      x = 0.0;
      E = 0;
    }
    int Er = __reduce_max_sync(0xffffffffu, E ? E + f : kNoEntry);
    if (Er == kNoEntry) Er = 0;
    P.Ri[k][c] = rp_fix(x, Er, f);
    if (c == 0) P.er[k] = Er;
  }
  return bad;
}

// sum_j Ri[k][j] Xi[j][c] over j0 <= j <= c, in units of 2^6 of the product.
__device__ __forceinline__ __int128 rp_dot(const RpPrep& P, int k, int c, int j0) {
  __int128 acc = 0;
  for (int j = j0; j <= c; ++j) acc += ((__int128)P.Ri[k][j] * P.Xi[j][c]) >> 6;
  return acc;
}

// f_c of every column and e_k of the rows below `rows` without launches of their own: every block of the preparation
// finds them (they agree).
__device__ __forceinline__ void rp_own_scales(RpPrep& P, int n, int npad, const double* __restrict__ RT, const RpInts& I,
                                              int rows) {
  if (n <= kRN) {   // one panel: rows 4 g .. of column c in this thread, loaded once
    const int c = threadIdx.x & 31, g = threadIdx.x >> 5;
    double x[4];
    uint32_t mx = 0u;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int k = 4 * g + r;
      x[r] = c < n && k <= c ? RT[(int64_t)k * npad + c] : 0.0;
      mx = max(mx, rp_finite_hi(x[r]));
    }
    P.red[g][c] = (int)mx;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < 8; ++w) mx = max(mx, (uint32_t)P.red[w][c]);
    const int E = (int)oz::exp_field(mx), f = E == 0 ? 0 : 1023 - E;
    if (g == 0 && c < n) P.fN[c] = I.fN[c] = f;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const uint32_t h = (uint32_t)__double2hiint(x[r]) & 0x7FFFFFFFu;
      const uint32_t all = __reduce_max_sync(0xffffffffu, h);
      const int me = __reduce_max_sync(0xffffffffu, h >= 0x00100000u ? (int)(h >> 20) + f : INT_MIN);
      if (c == 0 && 4 * g + r < n) I.eR[4 * g + r] = (all >= 0x7FF00000u || me == INT_MIN) ? 0 : me - 1023;
    }
    return;
  }
  for (int blk = 0; blk < (n + kRN - 1) / kRN; ++blk) rp_col_scale_block(n, npad, RT, P.fN, blk, P.red);
  __syncthreads();
  for (int c = threadIdx.x; c < n; c += 256) I.fN[c] = P.fN[c];
  for (int blk = 0; blk < (rows + 7) / 8; ++blk) rp_row_scale_block(n, npad, RT, P.fN, I.eR, blk);
}

// Multiplier of a panel that keeps its substitution: the digits of -D^{-1} R_{<t,t}
// against the columns' largest entries (no X_t, no F: each column has its own reference).
__device__ __forceinline__ void rp_prep_kept(RpPrep& P, int n, int npad, const double* __restrict__ RT, const RpInts& I,
                                             unsigned char* __restrict__ Md2, int t) {
  const int c = threadIdx.x & 31, g = threadIdx.x >> 5, c0 = kRN * t;
  const bool live = c0 + c < n;
  int mE = kNoEntry;
  for (int k = g; k < c0; k += 8) {
    const int E = live ? (int)oz::exp_field((uint32_t)__double2hiint(RT[(int64_t)k * npad + c0 + c])) : 0;
    if (E != 0) mE = max(mE, E == 2047 ? kNonfinite : E - I.eR[k]);
  }
  __syncthreads();
  P.red[g][c] = mE;
  __syncthreads();
  for (int k = 0; k < 8; ++k) mE = max(mE, P.red[k][c]);
  if (g == 0) I.colE2[c0 + c] = mE;
  for (int kc = 0; kc < t; ++kc) {
    uint64_t J[4];
    uint32_t neg[4], d[oz::kSlices][2], o[oz::kSlices];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int k = kRN * kc + 4 * g + r;
      const double x = live && mE != kNonfinite ? RT[(int64_t)k * npad + c0 + c] : 0.0;
      const uint32_t h = (uint32_t)__double2hiint(x);
      J[r] = oz::biased_fixed63(h, (uint32_t)__double2loint(x), mE, -I.eR[k]);
      neg[r] = (h >> 31) ^ 1u;
    }
    oz::digits8_pack(J[0], J[1], neg[0], neg[1], o);
#pragma unroll
    for (int b = 0; b < oz::kSlices; ++b) d[b][0] = o[b];
    oz::digits8_pack(J[2], J[3], neg[2], neg[3], o);
#pragma unroll
    for (int b = 0; b < oz::kSlices; ++b) d[b][1] = o[b];
    unsigned char* panel = Md2 + rp_block_offset(t, kc) + tc::sw64_offset(c, 4 * g, 2);
#pragma unroll
    for (int b = 0; b < oz::kSlices; ++b) *reinterpret_cast<uint2*>(panel + b * kRBPanel) = make_uint2(d[b][0], d[b][1]);
  }
}

__device__ __forceinline__ void rp_prep_r_panel(RpPrep& P, int n, int npad, const double* __restrict__ RT,
                                                const double* __restrict__ rinv, const RpInts& I,
                                                unsigned char* __restrict__ Md, uint32_t* __restrict__ colHiOut,
                                                int nhi, int t, int check) {
  int* eR = I.eR;
  const int tid = threadIdx.x, c = tid & 31, g = tid >> 5;   // this thread: column c, rows 4 g .. 4 g + 3
  const int c0 = kRN * t, w = min(kRN, n - c0);
  if (colHiOut && t == 0)     // the product folds the column maxima of W into these
    for (int i = tid; i < nhi; i += blockDim.x) colHiOut[i] = 0u;
  if (n <= kRpOwnScale) rp_own_scales(P, n, npad, RT, I, min(n, c0 + kRN));
  __syncthreads();
  const int* fN = n <= kRpOwnScale ? P.fN : I.fN;
  const int f = c < w ? fN[c0 + c] : 0;
  // X = (R F^{-1})_tt^{-1} by FP64 back substitution, column c in the lanes, rows over the warps
  const double scale = rp_pow2(f);
  if (g == 0) P.rinv[c] = c < w ? rinv[c0 + c] * rp_pow2(-f) : 1.0;
  double b[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int i = 4 * g + r;
    P.R[i][c] = (i < w && c < w) ? (i <= c ? RT[(int64_t)(c0 + i) * npad + c0 + c] * scale : 0.0) : (i == c ? 1.0 : 0.0);
    b[r] = i == c ? 1.0 : 0.0;
  }
  __syncthreads();
#pragma unroll
  for (int k = kRN - 1; k >= 0; --k) {
    if ((k >> 2) == g) P.X[k][c] = k >= w ? b[k & 3] : c < k ? 0.0 : b[k & 3] * P.rinv[k];
    if (k >= w) continue;   // identity beyond column n
    __syncthreads();
    const double x = P.X[k][c];
#pragma unroll
    for (int r = 0; r < 4; ++r)
      if (4 * g + r < k) b[r] = fma(-P.R[4 * g + r][k], x, b[r]);
  }
  bool bad = false;
  {   // fixed point: X against the exponents of its columns (one bit of headroom), R_tt against its rows'
    int mE = 0;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int E = (int)oz::exp_field((uint32_t)__double2hiint(P.X[4 * g + r][c]));
      mE = max(mE, E);
      const int E2 = (int)oz::exp_field((uint32_t)__double2hiint(P.R[4 * g + r][c]));
      const int Er = (int)__reduce_max_sync(0xffffffffu, (uint32_t)E2);
      bad |= E == 2047 || E2 == 2047;
      P.Ri[4 * g + r][c] = rp_fix(E2 == 2047 ? 0.0 : P.R[4 * g + r][c], Er);
      if (c == 0) P.er[4 * g + r] = Er;
    }
    P.red[g][c] = mE;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 8; ++k) mE = max(mE, P.red[k][c]);
    if (g == 0) P.Ex[c] = mE + 1;
#pragma unroll
    for (int r = 0; r < 4; ++r) P.Xi[4 * g + r][c] = mE == 2047 ? 0 : rp_fix(P.X[4 * g + r][c], mE + 1);
  }
  __syncthreads();
  {   // E = I - R_tt X exactly (up to the fixed point), X += X E.  With acc = E in units of 2^(er_i + Ex_c - 2164),
      // the correction of Xi[i][c] is sum_j Xi[i][j] acc_jc 2^(er_j + Ex_j - 2164): a small fraction of Xi, for which
      // FP32 (24 bits of a 2^-40 correction) is exact enough.
    const int Ex = P.Ex[c];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int i = 4 * g + r;
      __int128 acc = i <= c ? -rp_dot(P, i, c, i) : (__int128)0;
      const int p = 2164 - P.er[i] - Ex;
      if (i == c) {
        if (p < 0 || p > 124) bad = true;
        else acc += (__int128)1 << p;
      }
      const int top = rp_msb(acc), sh = max(top - 30, 0);
      P.F[i][c] = ldexpf((float)(int)(acc >> sh), sh + P.er[i] + P.Ex[i] - 2102);   // times 2^62
    }
    __syncthreads();
    long long add[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int i = 4 * g + r;
      float l = 0.0f;
      for (int j = i; j <= c; ++j) l = fmaf((float)(P.Xi[i][j] >> 31) * 4.656612873077393e-10f, P.F[j][c], l);   // Xi 2^-62
      if (!(fabsf(l) < 0x1p60f)) {
        bad = true;
        l = 0.0f;
      }
      add[r] = __float2ll_rn(l);
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 4; ++r) P.Xi[4 * g + r][c] += add[r];
  }
  // column references over (D^-1 Z; X)
  bool nf = false;
  {
    __syncthreads();
    const int Ex = P.Ex[c];
    int mE = kNoEntry;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int p = rp_msb(P.Xi[4 * g + r][c]);
      if (p >= 0) mE = max(mE, p + Ex - 62);
    }
    for (int kc = 0; kc < t; ++kc) {
      __syncthreads();
      nf |= rp_load_fixed(P, n, npad, RT, kc, c0, f);
      __syncthreads();
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int k = 4 * g + r;
        const int p = rp_msb(rp_dot(P, k, c, 0));
        if (p >= 0) mE = max(mE, p + P.er[k] + Ex - 1141 - eR[kRN * kc + k]);
      }
    }
    __syncthreads();
    P.red[g][c] = nf ? kNonfinite : mE;
    __syncthreads();
    if (g == 0) {
      for (int k = 0; k < 8; ++k) mE = max(mE, P.red[k][c]);
      P.cE[c] = mE;
    }
    __syncthreads();
    float amp = 0.0f;   // sum_i 2^(cE_i - 1022) |R[i][c]|: four rows a thread, then over the warps
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const uint32_t h = (uint32_t)__double2hiint(P.R[4 * g + r][c]) & 0x7FFFFFFFu;
      const float s = __uint_as_float(0x3F800000u | ((h & 0xFFFFFu) << 3) | 7u);   // significand, rounded up
      if (h) amp += ldexpf(s, (int)oz::exp_field(h) - 1023 + P.cE[4 * g + r] - 1022);
    }
    P.red[g][c] = __float_as_int(amp);
    __syncthreads();
    if (g == 0) {
      for (int k = 1; k < 8; ++k) amp += __int_as_float(P.red[k][c]);
      if (!(amp <= kAmpLimit)) bad = true;
    }
  }
  const bool keep = __syncthreads_or(bad || nf) != 0;
  if (tid == 0) I.flags[t] = keep ? 1 : 0;
  if (keep && !check) rp_prep_kept(P, n, npad, RT, I, Md + rp_digit_size(n), t);
  // digits (of a kept panel only the block of X is copied, and multiplied by zeros)
  if (g == 0 && c < w) I.colE[c0 + c] = P.cE[c];
  const int Ex = P.Ex[c], cE = P.cE[c];
  for (int kc = 0; kc <= t; ++kc) {
    if (kc < t) {
      __syncthreads();
      rp_load_fixed(P, n, npad, RT, kc, c0, f);
      __syncthreads();
    }
    uint32_t d[oz::kSlices][2];
    uint64_t J[4];
    uint32_t neg[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int k = 4 * g + r;
      __int128 acc;
      int sh;   // I = |acc| 2^-sh
      if (kc < t) {
        acc = -rp_dot(P, k, c, 0);
        sh = cE - P.er[k] - Ex + eR[kRN * kc + k] + 1079;
      } else {
        acc = P.Xi[k][c];
        sh = cE - Ex;
      }
      neg[r] = acc < 0;
      const unsigned __int128 u = acc < 0 ? -(unsigned __int128)acc : (unsigned __int128)acc;
      uint64_t I = 0;
      if (c < w && cE != kNonfinite && u != 0) {
        if (sh <= 0) I = (uint64_t)(u << -sh);
        else if (sh < 128) I = (uint64_t)(((u >> (sh - 1)) + 1) >> 1);
      }
      J[r] = I + 0x0080808080808080ull;
    }
    uint32_t o[oz::kSlices];
    oz::digits8_pack(J[0], J[1], neg[0], neg[1], o);
#pragma unroll
    for (int k = 0; k < oz::kSlices; ++k) d[k][0] = o[k];
    oz::digits8_pack(J[2], J[3], neg[2], neg[3], o);
#pragma unroll
    for (int k = 0; k < oz::kSlices; ++k) d[k][1] = o[k];
    unsigned char* panel = Md + rp_block_offset(t, kc) + tc::sw64_offset(c, 4 * g, 2);
#pragma unroll
    for (int k = 0; k < oz::kSlices; ++k)
      *reinterpret_cast<uint2*>(panel + k * kRBPanel) = make_uint2(d[k][0], d[k][1]);
  }
}

__global__ void __launch_bounds__(256) k_rp_prep_r(int n, int npad, const double* __restrict__ RT,
                                                   const double* __restrict__ rinv, RpInts I,
                                                   unsigned char* __restrict__ Md, uint32_t* __restrict__ colHiOut,
                                                   int nhi, int check, const Ctl* ctl, int level) {
  if (level_inactive(ctl, level) || ctl->lvl_status != 0) return;
  extern __shared__ unsigned char prep_raw[];
  RpPrep& P = *reinterpret_cast<RpPrep*>(prep_raw);
  const int t = (int)blockIdx.x % (npad / kRN);
  if ((int)blockIdx.x == t) {
    rp_prep_r_panel(P, n, npad, RT, rinv, I, Md, colHiOut, nhi, t, check);
  } else {   // checked solve: a second block per panel prepares its substitution
    if (n <= kRpOwnScale) rp_own_scales(P, n, npad, RT, I, kRN * t);
    __syncthreads();
    rp_prep_kept(P, n, npad, RT, I, Md + rp_digit_size(n), t);
  }
}

// ---------------------------------------------------------------------------
// Grouped forms for batched plans: persistent launches over {problem, block}
// items; an item whose problem is not active at this level, or has raised a
// status, is skipped.  A CTA that moves on to another problem folds its column
// maxima into the previous one's first.
__device__ __forceinline__ bool rp_live(const Prob& P, int level) {
  return P.ctl->active == level && P.ctl->lvl_status == 0;
}

__device__ __forceinline__ int rp_nhi(int n) { return (n + kM - 1) / kM * kM; }

__host__ __device__ __forceinline__ RpArgs rp_trsm_args(int64_t m, int n, const double* A, int64_t lda, double* W,
                                                        int64_t ldw, int* ints, const unsigned char* Rd,
                                                        const double* RT, const double* rinv, uint32_t* colHiOut) {
  const RpInts I(ints, n);
  return RpArgs{m, n, A, lda, W, ldw, I.colE, Rd, I.colE2, Rd + rp_digit_size(n), I.eR, I.fN, I.flags, RT, rinv, colHiOut};
}

__host__ __device__ __forceinline__ RpArgs rp_fin_args(int64_t m, int n, double* Q, int64_t ldq, const int* colE,
                                                       const unsigned char* Xs, uint32_t* colHiOut) {
  return RpArgs{m, n, nullptr, 0, Q, ldq, colE, Xs, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, colHiOut};
}

__device__ __forceinline__ RpArgs rp_args_of(const Prob& P, bool trsm) {
  if (trsm) return rp_trsm_args(P.m, P.n, P.A, P.lda, P.Q, P.ldq, P.oz_cole, P.oz_rd, P.rst, P.rinv, P.oz_colhi);
  return rp_fin_args(P.m, P.n, P.Q, P.ldq, P.oz_xe, P.oz_xs, P.check ? P.oz_colhi : nullptr);
}

template <bool kTrsm>
__global__ void __launch_bounds__(kRThreads, 2) kg_rowprod(Group g, int level) {
  MRCQR_RP_CTA(S)
  __shared__ RpArgs a;   // the current problem's arguments (shared: not held in registers)
  bool abort = false;
  int cur = -1;
  Ctl* actl = nullptr;
  for (int it = blockIdx.x; it < g.nitems; it += gridDim.x) {
    const int4 w = g.items[it];
    const Prob& P = g.probs[w.x];
    if (!rp_live(P, level)) continue;
    if (w.x != cur) {
      if (cur >= 0) rp_end(a, S);
      __syncthreads();
      if (threadIdx.x == 0) a = rp_args_of(P, kTrsm);
      __syncthreads();
      rp_begin<kTrsm>(a, S);
      cur = w.x;
    }
    if (!rp_block<kTrsm, true, false>(a, S, (int64_t)w.y * kM, 0)) {
      abort = true;
      actl = P.ctl;
      break;
    }
  }
  if (!abort && cur >= 0) rp_end(a, S);
  rp_cta_end(S, abort, actl);
}

__global__ void __launch_bounds__(128) kg_rp_prep_x(Group g, int level) {
  __shared__ uint32_t red[4];
  for (int it = blockIdx.x; it < g.nitems; it += gridDim.x) {
    const int4 w = g.items[it];
    const Prob& P = g.probs[w.x];
    if (!rp_live(P, level)) continue;
    rp_prep_x_col(P.n, P.npad, P.xt, P.oz_xe, P.oz_xs, P.check ? P.oz_colhi : nullptr, rp_nhi(P.n), w.y, red);
    __syncthreads();
  }
}

__global__ void __launch_bounds__(256) kg_rp_col_scale(Group g, int level) {
  __shared__ int red[8][kRN];
  for (int it = blockIdx.x; it < g.nitems; it += gridDim.x) {
    const int4 w = g.items[it];
    const Prob& P = g.probs[w.x];
    if (!rp_live(P, level)) continue;
    rp_col_scale_block(P.n, P.npad, P.rst, RpInts(P.oz_cole, P.n).fN, w.y, red);
  }
}

__global__ void __launch_bounds__(256) kg_rp_row_scale(Group g, int level) {
  for (int it = blockIdx.x; it < g.nitems; it += gridDim.x) {
    const int4 w = g.items[it];
    const Prob& P = g.probs[w.x];
    if (!rp_live(P, level)) continue;
    const RpInts I(P.oz_cole, P.n);
    rp_row_scale_block(P.n, P.npad, P.rst, I.fN, I.eR, w.y);
  }
}

__global__ void __launch_bounds__(256) kg_rp_prep_r(Group g, int level) {
  extern __shared__ unsigned char prep_raw[];
  for (int it = blockIdx.x; it < g.nitems; it += gridDim.x) {
    const int4 w = g.items[it];
    const Prob& P = g.probs[w.x];
    if (!rp_live(P, level)) continue;
    __syncthreads();
    rp_prep_r_panel(*reinterpret_cast<RpPrep*>(prep_raw), P.n, P.npad, P.rst, P.rinv, RpInts(P.oz_cole, P.n), P.oz_rd,
                    P.oz_colhi, rp_nhi(P.n), w.y, 0);
  }
}

template <bool kTrsm, bool kCheck>
void rp_launch(const RpArgs& a, Ctl* ctl, int level, cudaStream_t st) {
  const int64_t nblocks = (a.m + kM - 1) / kM, slots = 2 * (int64_t)device_sms();
  const unsigned grid = (unsigned)(nblocks < slots ? nblocks : slots);
  auto kernel = a.n > kRN * kGroupChunks ? k_rowprod<kTrsm, true, kCheck> : k_rowprod<kTrsm, false, kCheck>;
  cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRSmem);
  launch_dep(kernel, grid, kRThreads, kRSmem, st, a, ctl, level);
}

unsigned rp_grid(int nitems, int per_sm) {
  const int cap = device_sms() * per_sm;
  return (unsigned)(nitems < cap ? nitems : cap);
}

}  // namespace

// Workspace sizes: digit panels of the multiplier blocks (the TRSM has two sets), and the exponents.
size_t rp_trsm_digit_bytes(int n) { return 2 * rp_digit_size(n); }
size_t rp_trsm_ints_bytes(int n) { return sizeof(int) * (size_t)(4 * rp_n32(n) + 16); }
size_t rp_fin_digit_bytes(int n) { return rp_wide(n) ? fw_digit_bytes(n) : rp_digit_size(n); }
size_t rp_fin_ints_bytes(int n) { return sizeof(int) * (size_t)rp_n32(n); }
int rp_cols(int n) { return rp_n32(n); }
int rp_panels(int n) { return rp_n32(n) / kRN; }

void launch_trsm_oz(int64_t m, int n, const double* A, int64_t lda, const double* RT, const double* rinv, int* ints,
                    unsigned char* Rd, double* W, int64_t ldw, Ctl* ctl, int level, cudaStream_t st,
                    uint32_t* colHiOut, bool check) {
  const int n32 = rp_n32(n);
  const int nhi = (int)(syrk_oz_colhi_bytes(n) / sizeof(uint32_t));
  const RpInts I(ints, n);
  if (n > kRpOwnScale) {
    launch_dep(k_rp_col_scale, n32 / kRN, 256, 0, st, n, n32, RT, I.fN, ctl, level);
    launch_dep(k_rp_row_scale, (n + 7) / 8, 256, 0, st, n, n32, RT, I.fN, I.eR, ctl, level);
  }
  cudaFuncSetAttribute(k_rp_prep_r, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(RpPrep));
  launch_dep(k_rp_prep_r, (check ? 2 : 1) * n32 / kRN, 256, sizeof(RpPrep), st, n, n32, RT, rinv, I, Rd, colHiOut, nhi, check ? 1 : 0, ctl, level);
  const RpArgs a = rp_trsm_args(m, n, A, lda, W, ldw, ints, Rd, RT, rinv, colHiOut);
  if (check) rp_launch<true, true>(a, ctl, level, st);
  else rp_launch<true, false>(a, ctl, level, st);
}

void launch_finalize_oz(int64_t m, int n, double* Q, int64_t ldq, const double* XT, int* colE, unsigned char* Xs,
                        Ctl* ctl, int level, cudaStream_t st, uint32_t* colHiOut) {
  if (rp_wide(n)) {
    launch_finalize_wide(m, n, Q, ldq, XT, colE, Xs, ctl, level, st, colHiOut);
    return;
  }
  const int n32 = rp_n32(n);
  const int nhi = (int)(syrk_oz_colhi_bytes(n) / sizeof(uint32_t));
  launch_dep(k_rp_prep_x, n32, 128, 0, st, n, n32, XT, colE, Xs, colHiOut, nhi, ctl, level);
  rp_launch<false, false>(rp_fin_args(m, n, Q, ldq, colE, Xs, colHiOut), ctl, level, st);
}

void prepare_g_rowprod() {
  cudaFuncSetAttribute(kg_rowprod<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRSmem);
  cudaFuncSetAttribute(kg_rowprod<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRSmem);
  cudaFuncSetAttribute(kg_rp_prep_r, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(RpPrep));
}

void launch_g_oz_col_scale(const Group& g, int level, cudaStream_t st) {
  if (g.nitems) { ::mrcqr::note_launch(); kg_rp_col_scale<<<rp_grid(g.nitems, 8), 256, 0, st>>>(g, level); }
}
void launch_g_oz_row_scale(const Group& g, int level, cudaStream_t st) {
  if (g.nitems) { ::mrcqr::note_launch(); kg_rp_row_scale<<<rp_grid(g.nitems, 16), 256, 0, st>>>(g, level); }
}
void launch_g_oz_prep_r(const Group& g, int level, cudaStream_t st) {
  if (g.nitems) { ::mrcqr::note_launch(); kg_rp_prep_r<<<rp_grid(g.nitems, 4), 256, sizeof(RpPrep), st>>>(g, level); }
}
void launch_g_oz_trsm(const Group& g, int level, cudaStream_t st) {
  if (g.nitems) { ::mrcqr::note_launch(); kg_rowprod<true><<<rp_grid(g.nitems, 2), kRThreads, kRSmem, st>>>(g, level); }
}
void launch_g_oz_prep_x(const Group& g, int level, cudaStream_t st) {
  if (g.nitems) { ::mrcqr::note_launch(); kg_rp_prep_x<<<rp_grid(g.nitems, 16), 128, 0, st>>>(g, level); }
}
void launch_g_oz_finalize(const Group& g, int level, cudaStream_t st) {
  if (g.nitems) { ::mrcqr::note_launch(); kg_rowprod<false><<<rp_grid(g.nitems, 2), kRThreads, kRSmem, st>>>(g, level); }
}

}  // namespace mrcqr
