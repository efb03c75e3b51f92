// The FP64 sketch (Algorithm 2 steps 2-4 at p = FP64, DCT) as a four-step
// transform in emulated FP64: the dense form (ozaki_planes.cu) multiplies
// every entry of A with s transform entries, 72 s m n tensor operations; here
//   j = j1 + J j2,  J = m / 32,  0 <= j2 < 32,
//   cos(pi k (2 j + 1) / (2m)) = Re e^{i theta_k(j1)} e^{2 pi i k j2 / 64},
//   theta_k(j1) = pi k (2 j1 + 1) / (2m),
// so the sums over j2 depend on k only through k mod 64:
//  1. C_q[j1] + i S_q[j1] = sum_j2 e^{2 pi i q j2 / 64} d_j A_j for q = 0 .. 32
//     (64 real rows: S_0 = S_32 = 0, q > 32 is the conjugate of 64 - q), one
//     emulated product with K = 32 per 128 rows j1 and column (k_fd_pass1);
//  2. Y_k = sum_j1 cos theta C_q - sin theta S_q (+ for the conjugates): the
//     samples of one class q are at most 32-column tiles of an emulated product
//     over the class's 2 J rows (k_fd_pass2).
// That is 72 (64 + s / 16) m n tensor operations (s = 1024: 1/8 of the dense
// form, s = 256: 1/3) for 16 more bytes written and read per entry of A.
//
// No step rounds to FP64 in between: the level sums of pass 1 are shifted to
// 62-bit fixed point against a bound of |C|, |S| over the column (the largest
// sum over j2 of |A|, found with the column maxima) and stored as the 64-bit word whose bytes are the balanced digits plus 128,
// and both cosine tables are evaluated to about 2^-61 by their Taylor series in
// 64-bit integers (the dense form takes FP64 cosines), so the sketch is as
// accurate as the dense form's.  The words take twice the space of A; a
// factorization lends the Q buffer, each column's words in that column, and
// works in two ranges of j1.
//
// Measured (Y; dense form before): m = 2^20, n = 512, s = 1024 55.0 -> 12.7 ms; n = 128, s = 256 4.03 -> 2.63;
// m = 2^18, n = 160, s = 320 2.35 -> 0.98. Pass 1 (0.85 of 2.63 ms at n = 128) is bound by the integer pipe
// (slicing, readout, words), pass 2 (1.3 ms) by the latency of its words and table gathers. At s = 128 the two
// forms do the same tensor work, and the dense one moves 16 bytes less per entry: the rule takes this one from
// s = 160 (kFdMinRows). Streaming loads and stores of the words, which keep the 16 MB digit table in the L2:
// 14.3 -> 12.7 ms at n = 512.
#include <algorithm>

#include "ozaki_pipe.cuh"

namespace mrcqr {

namespace {

constexpr int kR = 32;                 // radix: terms of a first-step sum
constexpr int kRows = 2 * kR;          // real rows of the first step
constexpr int kClasses = kR + 1;       // k mod 64 up to conjugation
constexpr int kFdTile = kRN;           // samples per tile of the second step
constexpr uint64_t kBias8 = 0x8080808080808080ull;
constexpr size_t kPartFd = 2 * (size_t)kM * kFdTile;   // hi and lo of one 128 x 32 item

// cos(pi q / (2 m)) 2^62 for 0 <= q <= m, to about two units: the angle (or
// its complement, at most pi / 4) in 62-bit fixed point and the Taylor series
// of cosine or sine by Horner's rule in 64 x 64-bit integer products.
__device__ __forceinline__ uint64_t fd_mul62(uint64_t a, uint64_t b) {   // a b 2^-62
  return (__umul64hi(a, b) << 2) | ((a * b) >> 62);
}
__device__ uint64_t fd_cos62(uint64_t q, uint64_t m) {
  const bool sine = 2 * q > m;
  const uint64_t p = sine ? m - q : q;             // <= m / 2
  const uint64_t f1 = (p << 32) / m, f0 = (((p << 32) - f1 * m) << 32) / m;   // p / m in 64 fraction bits
  const uint64_t y = __umul64hi(0x6487ED5110B4611Aull, f1 << 32 | f0);        // (pi / 2) (p / m) 2^62
  const uint64_t z = fd_mul62(y, y);
  const uint64_t one = 1ull << 62;
  uint64_t t = one;
#pragma unroll
  for (int k = 10; k >= 1; --k) {                  // z^11 / 22! < 2^-75
    const uint64_t zt = fd_mul62(z, t);
    t = one - (sine ? zt / (uint64_t)((2 * k) * (2 * k + 1)) : zt / (uint64_t)((2 * k - 1) * (2 * k)));
  }
  return sine ? fd_mul62(y, t) : t;
}

// cos(pi r / (2m)), r mod 4m, as the sign and the magnitude's index in the quarter wave.
__device__ __forceinline__ uint64_t fd_quarter(uint64_t r, uint64_t m, uint32_t& neg) {
  if (r >= 2 * m) r = 4 * m - r;
  neg = r > m ? 1u : 0u;
  return neg ? 2 * m - r : r;
}

// Digits (FP16, digit a in 16-bit lane a) of the quarter-wave table.
__global__ void __launch_bounds__(256) k_fd_table(int64_t m, uint4* __restrict__ tabd, const Ctl* ctl, int level) {
  if (level_inactive(ctl, level) || ctl->lvl_status != 0) return;
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q > m) return;
  const uint64_t J = fd_cos62((uint64_t)q, (uint64_t)m) + 0x0080808080808080ull;
  uint32_t w[oz::kSlices];
  oz::digits8_pack(J, J, 0u, 0u, w);
  tabd[q] = make_uint4(__byte_perm(w[0], w[1], 0x5410), __byte_perm(w[2], w[3], 0x5410),
                       __byte_perm(w[4], w[5], 0x5410), __byte_perm(w[6], w[7], 0x5410));
}

// Rademacher signs: bit j2 of sgn[j1] is set when d of row j1 + J j2 is -1.
__global__ void __launch_bounds__(256) k_fd_signs(int64_t J, uint2 key, uint32_t* __restrict__ sgn, const Ctl* ctl,
                                                  int level) {
  if (level_inactive(ctl, level) || ctl->lvl_status != 0) return;
  const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;   // one warp per four words
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int64_t j1 = 4 * w + u;
    if (j1 >= J) return;
    const bool neg = row_sign((uint64_t)(j1 + J * lane), key) < 0.0;
    const uint32_t b = __ballot_sync(0xffffffffu, neg);
    if (lane == 0) sgn[j1] = b;
  }
}

// Sorts the samples by class: tile t holds up to 32 samples of class cls[t]
// in slots 32 t .. (sample number | 2^31 for the conjugate half, -1 for
// an empty slot).  One block; one warp per class, so the order is fixed.
__global__ void __launch_bounds__(1024) k_fd_classes(int s, const uint32_t* __restrict__ idx, int* __restrict__ ntiles,
                                                     int* __restrict__ cls, int* __restrict__ slots, const Ctl* ctl,
                                                     int level) {
  if (level_inactive(ctl, level) || ctl->lvl_status != 0) return;
  __shared__ int cnt[kClasses], first[kClasses];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  auto class_of = [&](int i) {
    const int q = (int)(idx[i] & 63u);
    return q <= kR ? q : 2 * kR - q;
  };
  for (int q = warp; q < kClasses; q += 32) {
    int n = 0;
    for (int i0 = 0; i0 < s; i0 += 32) {
      const bool in = i0 + lane < s && class_of(i0 + lane) == q;
      n += __popc(__ballot_sync(0xffffffffu, in));
    }
    if (lane == 0) cnt[q] = n;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int t = 0;
    for (int q = 0; q < kClasses; ++q) {
      first[q] = t;
      for (int k = 0; k < cnt[q]; k += kFdTile) cls[t++] = q;
    }
    *ntiles = t;
  }
  __syncthreads();
  for (int q = warp; q < kClasses; q += 32) {
    int at = kFdTile * first[q];
    for (int i0 = 0; i0 < s; i0 += 32) {
      const bool in = i0 + lane < s && class_of(i0 + lane) == q;
      const uint32_t b = __ballot_sync(0xffffffffu, in);
      if (in) slots[at + __popc(b & ((1u << lane) - 1u))] = (int)((uint32_t)(i0 + lane) | ((idx[i0 + lane] & 63u) > kR ? 0x80000000u : 0u));
      at += __popc(b);
    }
    const int end = kFdTile * (first[q] + (cnt[q] + kFdTile - 1) / kFdTile);
    for (int k = at + lane; k < end; k += 32) slots[k] = -1;
  }
}

// Per column: the largest |A| (high word, as k_col_hi) and the biased exponent of the largest
// sum over j2 of |A[j1 + J j2]| (rounded up; FP32 relative to the row's own
// maximum, from the high words, so no FP64 instruction runs).  Both arrays zero on entry.
__global__ void __launch_bounds__(256) k_fd_bounds(int64_t J, const double* __restrict__ A, int64_t lda,
                                                   uint32_t* __restrict__ colHi, int* __restrict__ colU, const Ctl* ctl,
                                                   int level) {
  if (level_inactive(ctl, level) || ctl->lvl_status != 0) return;
  const int c = blockIdx.y;
  const int64_t j1 = (int64_t)blockIdx.x * 256 + threadIdx.x;
  uint32_t mx = 0u;
  int e = 0;
  if (j1 < J) {
    const uint2* p = reinterpret_cast<const uint2*>(A + (int64_t)c * lda + j1);
    uint32_t h[kR];
#pragma unroll
    for (int j2 = 0; j2 < kR; ++j2) h[j2] = __ldg(p + J * j2).y & 0x7FFFFFFFu;
#pragma unroll
    for (int j2 = 0; j2 < kR; ++j2) mx = max(mx, h[j2]);
    const int base = (int)(mx & 0x7FF00000u) - (127 << 20);
    float sum = 0.0f;
#pragma unroll
    for (int j2 = 0; j2 < kR; ++j2) sum += __int_as_float((max((int)h[j2] - base, 0) << 3) | 7);
    e = (int)oz::exp_field(mx) + ((__float_as_int(sum) >> 23) - 127);
  }
  __shared__ uint32_t rm[8];
  __shared__ int re[8];
  mx = __reduce_max_sync(0xffffffffu, mx);
  e = __reduce_max_sync(0xffffffffu, e);
  if ((threadIdx.x & 31) == 0) rm[threadIdx.x >> 5] = mx, re[threadIdx.x >> 5] = e;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) mx = max(mx, rm[w]), e = max(e, re[w]);
    atomicMax(colHi + c, mx);
    atomicMax(colU + c, e);
  }
}

// CTA state shared by the two passes: TMEM (256 columns) and one MMA barrier.
struct FdCta {
  unsigned char* smem;
  uint64_t* bar;
  int* dead;
  uint32_t tmem, commits;
};

__device__ __forceinline__ void fd_wait(FdCta& S) {   // for the last batch committed (bounded)
  if (*(volatile int*)S.dead) return;
  if (!tc::mbar_wait(S.bar, (S.commits - 1) & 1u, 1u << 20)) *(volatile int*)S.dead = 1;
}

#define MRCQR_FD_CTA(S)                                               \
  extern __shared__ unsigned char smem_raw[];                         \
  __shared__ __align__(8) uint64_t bar_s;                             \
  __shared__ uint32_t tmem_slot;                                      \
  __shared__ int dead_s;                                              \
  if ((threadIdx.x >> 5) == 0) tc::tmem_alloc(&tmem_slot, kRTmem);    \
  if (threadIdx.x == 0) {                                             \
    tc::mbar_init(&bar_s, 1);                                         \
    tc::mbar_fence_init();                                            \
    dead_s = 0;                                                       \
  }                                                                   \
  tc::fence_before();                                                 \
  __syncthreads();                                                    \
  tc::fence_after();                                                  \
  FdCta S{oz_smem(smem_raw), &bar_s, &dead_s, tmem_slot, 0u};

__device__ __forceinline__ void fd_end(FdCta& S, bool abort, Ctl* ctl) {
  if (abort && threadIdx.x == 0) {
    raise_level_status(ctl, ST_TIMEOUT);
    if (S.commits) tc::mbar_wait(S.bar, (S.commits - 1) & 1u, 1u << 20);
  }
  tc::fence_before();
  __syncthreads();
  if ((threadIdx.x >> 5) == 0) tc::tmem_dealloc(S.tmem, kRTmem);
}

// ---------------------------------------------------------------------------
// Pass 1.  Item = (128 rows j1 from jb, column c): A operand = rows j1, K =
// j2 (loads contiguous in j1); B operand = the 64 x 32 transform digits, kept
// in shared memory by the CTA.  Output words U[c cs + row Jc + j1 - j0].
__global__ void __launch_bounds__(kRThreads, 2)
    k_fd_pass1(int64_t J, int64_t j0, int64_t Jc, int nblocks, int n, const double* __restrict__ A, int64_t lda,
               const uint32_t* __restrict__ colHi, const int* __restrict__ colU, const uint32_t* __restrict__ sgn,
               uint64_t* __restrict__ U, int64_t cs, Ctl* ctl, int level) {
  if (level_inactive(ctl, level) || ctl->lvl_status != 0) return;
  MRCQR_FD_CTA(S)
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  unsigned char* bs = S.smem + kRABytes;   // two 16 KiB tiles: rows 0 .. 31, 32 .. 63
  for (int e = tid; e < kRows * kR; e += kRThreads) {
    const int row = e / kR, j2 = e % kR;
    // cos(2 pi q j2 / 64) = cos(pi r / 32) with r = q j2 mod 64: quarter wave of 16; the sine is a quarter period on
    const int q = row <= kR ? row : row - kR;
    uint32_t neg;
    const uint64_t qi = fd_quarter((uint64_t)((q * j2 + (row <= kR ? 0 : 48)) & 63), 16, neg);
    const uint64_t Jw = fd_cos62(qi, 16) + 0x0080808080808080ull;
    uint32_t w[oz::kSlices];
    oz::digits8_pack(Jw, Jw, neg, neg, w);
    unsigned char* dst = bs + (row / kRN) * kRBBytes + tc::sw64_offset(row % kRN, j2, 2);
#pragma unroll
    for (int a = 0; a < oz::kSlices; ++a) *reinterpret_cast<uint16_t*>(dst + a * kRBPanel) = (uint16_t)w[a];
  }
  __syncthreads();
  const int pr = tid & (kM - 1), ph = tid >> 7, rot = (lane >> 3) & 1;
  const int q = warp & 3, g = warp >> 2;
  const uint32_t tbase = S.tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(g * 16);
  const uint32_t sa = tc::smem_u32(S.smem);
  double v[4][4];
  uint32_t flips = 0u, fl_next = 0u;
  int gk[4];
  uint32_t off[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    gk[j] = 16 * ph + 8 * (j >> 1) + 4 * ((j & 1) ^ rot);
    off[j] = sa + tc::sw64_offset(pr, gk[j], 2);
  }
  const int nitems = nblocks * n;   // < 2^29
  auto load = [&](int item) {
    const int cn = item / nblocks;
    const int64_t j1 = j0 + kM * (item - cn * nblocks) + pr;
    const bool live = j1 < J;
    const double* base = A + cn * lda + (live ? j1 : 0);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const double* p = base + (int64_t)gk[j] * J;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        v[j][k] = live ? __ldg(p) : 0.0;
        p += J;
      }
    }
    fl_next = live ? __ldg(sgn + j1) : 0u;
  };
  bool abort = false;
  if ((int)blockIdx.x < nitems) load((int)blockIdx.x);
  for (int item = (int)blockIdx.x; item < nitems; item += (int)gridDim.x) {
    const int c = item / nblocks;
    const int E = (int)oz::exp_field(__ldg(colHi + c)), cr = oz_quad_cr(E);
    const int sh = 7 + __ldg(colU + c) - E;   // word exponent colU + 1: |word| <= 2^62
    flips = fl_next;
#pragma unroll
    for (int j = 0; j < 4; ++j) oz_store_quad<true>(v[j], flips >> gk[j], E, cr, off[j], kAPanel);
    tc::fence_proxy_async();
    tc::fence_before();
    __syncthreads();
    uint64_t* out = U + c * cs + g * 16 * Jc + kM * (item - c * nblocks) + q * 32 + lane;
#pragma unroll 1
    for (int t = 0; t < 2; ++t) {
      if (tid == 0) {
        tc::fence_after();
        rp_issue(S.tmem, sa, tc::smem_u32(bs) + t * kRBBytes, true);
        tc::mma_commit(S.bar);
      }
      ++S.commits;
      if (t == 0 && item + (int)gridDim.x < nitems) load(item + (int)gridDim.x);
      fd_wait(S);
      tc::fence_after();
      long long hi[16], lo[16];
#pragma unroll
      for (int k = 0; k < 16; ++k) hi[k] = lo[k] = 0;
      oz_readout_cols<kRN, false>(tbase, hi, lo);
      tc::fence_before();
      __syncthreads();   // the accumulators and (t = 1) the panels are free
      // T = hi 2^32 + lo; word = round(T 2^-sh) + bias, 7 <= sh <= 13
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        const long long x = hi[k] + (lo[k] >> 32);
        const uint32_t l = (uint32_t)lo[k], x0 = (uint32_t)x, x1 = (uint32_t)((uint64_t)x >> 32);
        const uint64_t w = ((uint64_t)__funnelshift_r(x0, x1, sh) << 32 | __funnelshift_r(l, x0, sh)) +
                           ((l >> (sh - 1)) & 1u) + kBias8;
        __stcs(reinterpret_cast<unsigned long long*>(out), (unsigned long long)w);
        out += Jc;
      }
      out += 16 * Jc;   // rows 32 .. 63 of the second tile
    }
    if (__syncthreads_or(*(volatile int*)S.dead)) {
      abort = true;
      break;
    }
  }
  fd_end(S, abort, ctl);
}

// ---------------------------------------------------------------------------
// Pass 2.  Item = (sample tile, 128 columns, slab of j1): A operand = columns
// of the class's words, expanded to FP16 digits (four instructions per digit
// pair of two values); B operand = the samples' twiddles, gathered from the
// digit table with the quadrant's sign.  K runs over the slab of C, then of S.
struct Fd2Args {
  int64_t m, J, j0, Jc, rows;   // Jc: words of a row of U; rows: j1 per slab (multiple of 128)
  int64_t jn;                   // j1 of this range, rounded up to 128
  int n, cblocks, slabs;
  const uint64_t* U;
  int64_t cs;                   // words between columns
  const uint32_t* idx;
  const uint4* tabd;
  const int* ntiles;
  const int* cls;
  const int* slots;
  long long* part;              // item ((tile cblocks + cb) slabs_all + slab)
  int slab0, slabs_all;
};

__global__ void __launch_bounds__(kRThreads, 2) k_fd_pass2(Fd2Args a, Ctl* ctl, int level) {
  if (level_inactive(ctl, level) || ctl->lvl_status != 0) return;
  MRCQR_FD_CTA(S)
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int q = warp & 3, g = warp >> 2;
  const uint32_t tbase = S.tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(g * 16);
  const uint32_t sa = tc::smem_u32(S.smem), sb = sa + kRABytes;
  // A: words 4 (lane % 8) .. + 3 of columns 16 warp + 4 it + lane / 8, it < 4: a warp's 16-byte loads cover whole
  // lines, a half warp's 8-byte panel stores two whole rows
  const int cw = 16 * warp + (lane >> 3), kw = 4 * (lane & 7);
  uint32_t aoff[4];
#pragma unroll
  for (int it = 0; it < 4; ++it) aoff[it] = sa + tc::sw64_offset(cw + 4 * it, kw, 2);
  const int fi = tid & 31, fg = (tid >> 5) ^ ((fi >> 3) & 1);   // B: sample fi, rows 4 fg .. 4 fg + 3
  const uint32_t boff = sb + tc::sw64_offset(fi, 4 * fg, 2);
  const uint64_t m = (uint64_t)a.m, fm = 4 * m;
  const int nitems = *a.ntiles * a.cblocks * a.slabs;
  bool abort = false;
  for (int item = blockIdx.x; item < nitems; item += gridDim.x) {
    const int slab = item % a.slabs, cb = (item / a.slabs) % a.cblocks, tile = item / (a.slabs * a.cblocks);
    const int cls = a.cls[tile];
    const int cbase = kM * cb + cw;
    const int slot = a.slots[kFdTile * tile + fi];
    const bool slive = slot != -1;
    const uint64_t k = slive ? (uint64_t)a.idx[slot & 0x7FFFFFFF] : 0ull;
    const int64_t r_begin = (int64_t)slab * a.rows, r_end = min(a.jn, r_begin + a.rows);
    const int nch = (int)((r_end - r_begin + kRN - 1) / kRN);   // jn and rows are multiples of 128
    const int parts = cls == 0 || cls == kR ? 1 : 2;
    const uint64_t dk = (2 * k) % fm, step_chunk = (dk * kRN) % fm;
    long long hi[16], lo[16];
#pragma unroll
    for (int e = 0; e < 16; ++e) hi[e] = lo[e] = 0;
    uint64_t ph = 0;
    const uint64_t* src = nullptr;
    ulonglong2 w[8];
    uint4 u[4];
    auto begin_part = [&](int p) {
      // cos theta; then -sin theta = cos(theta + pi / 2), + sin theta for the conjugate classes
      const uint64_t beta = p == 0 ? k : k + (slot < 0 ? 3 * m : m);
      ph = (dk * (uint64_t)(a.j0 + r_begin + 4 * fg) + beta) % fm;
      src = a.U + (int64_t)(p == 0 ? cls : kR + cls) * a.Jc + r_begin + kw;
    };
    int64_t coff[4];   // the four columns' words (column 0 beyond n: its digits are dropped)
#pragma unroll
    for (int it = 0; it < 4; ++it) coff[it] = (cbase + 4 * it < a.n ? cbase + 4 * it : 0) * a.cs;
    auto gather = [&] {
      uint64_t r = ph;
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        uint32_t neg;
        const uint64_t qi = fd_quarter(r, m, neg);
        u[t] = slive ? __ldg(a.tabd + qi) : make_uint4(0u, 0u, 0u, 0u);
        const uint32_t x = neg ? 0x80008000u : 0u;
        u[t].x ^= x, u[t].y ^= x, u[t].z ^= x, u[t].w ^= x;
        r += dk;
        if (r >= fm) r -= fm;
      }
      ph += step_chunk;
      if (ph >= fm) ph -= fm;
    };
    auto load_words = [&](int h) {
#pragma unroll
      for (int e = 0; e < 4; ++e)
        w[4 * h + e] = __ldcs(reinterpret_cast<const ulonglong2*>(src + coff[2 * h + (e >> 1)]) + (e & 1));
    };
    begin_part(0);
    gather();
    load_words(0);
    bool pending = false;
    const int total = parts * nch;
    for (int ch = 0; ch < total; ++ch) {
      load_words(1);
      if ((ch < nch ? ch : ch - nch) + 2 < nch && (lane & 3) == 0) {   // the lines two chunks on (two per column)
#pragma unroll
        for (int it = 0; it < 4; ++it) tc::prefetch_l2(src + coff[it] + 2 * kRN);
      }
      if (pending) fd_wait(S);
      pending = false;
      // words -> digits: byte b of a word is a digit + 128
#pragma unroll
      for (int it = 0; it < 4; ++it) {
        uint32_t d[oz::kSlices][2];
#pragma unroll
        for (int p = 0; p < 2; ++p) {
          const uint64_t x = w[2 * it + p].x, y = w[2 * it + p].y;
#pragma unroll
          for (int z = 0; z < 4; ++z) {
            const uint32_t pp = __byte_perm((uint32_t)(z < 2 ? x >> 32 : x), (uint32_t)(z < 2 ? y >> 32 : y),
                                            (z & 1) ? 0x5410u : 0x7632u);
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              const uint32_t t = __byte_perm(pp, 0x64646464u, e == 0 ? 0x4341u : 0x4240u);
              const __half2 r = __hsub2(*reinterpret_cast<const __half2*>(&t), __half2half2(__ushort_as_half(0x6480)));
              d[2 * z + e][p] = *reinterpret_cast<const uint32_t*>(&r);
            }
          }
        }
        const bool live = cbase + 4 * it < a.n;
#pragma unroll
        for (int e = 0; e < oz::kSlices; ++e)
          tc::st_shared2(aoff[it] + e * kAPanel, live ? d[e][0] : 0u, live ? d[e][1] : 0u);
      }
      {   // twiddle digits: four rows of sample fi
        const uint32_t x[4][4] = {{u[0].x, u[0].y, u[0].z, u[0].w}, {u[1].x, u[1].y, u[1].z, u[1].w},
                                  {u[2].x, u[2].y, u[2].z, u[2].w}, {u[3].x, u[3].y, u[3].z, u[3].w}};
#pragma unroll
        for (int e = 0; e < oz::kSlices; ++e) {
          const uint32_t sel = (e & 1) ? 0x7632u : 0x5410u;
          tc::st_shared2(boff + e * kRBPanel, __byte_perm(x[0][e >> 1], x[1][e >> 1], sel),
                         __byte_perm(x[2][e >> 1], x[3][e >> 1], sel));
        }
      }
      tc::fence_proxy_async();
      tc::fence_before();
      __syncthreads();
      if (tid == 0) {
        tc::fence_after();
        rp_issue(S.tmem, sa, sb, ch % kGroupChunks == 0);
        tc::mma_commit(S.bar);
      }
      ++S.commits;
      pending = true;
      if (ch + 1 < total) {
        if (ch + 1 == nch) begin_part(1);
        else src += kRN;
        gather();
        load_words(0);
      }
      if (ch % kGroupChunks == kGroupChunks - 1 || ch + 1 == total) {   // at most 128 terms per level sum
        fd_wait(S);
        pending = false;
        tc::fence_after();
        oz_readout_cols<kRN, false>(tbase, hi, lo);
        tc::fence_before();
        __syncthreads();
      }
    }
    long long* out = a.part + ((size_t)(tile * a.cblocks + cb) * a.slabs_all + a.slab0 + slab) * kPartFd;
#pragma unroll
    for (int e = 0; e < 16; ++e) {
      out[(g * 16 + e) * kM + q * 32 + lane] = hi[e];
      out[kM * kFdTile + (g * 16 + e) * kM + q * 32 + lane] = lo[e];
    }
    if (__syncthreads_or(*(volatile int*)S.dead)) {
      abort = true;
      break;
    }
  }
  fd_end(S, abort, ctl);
}

// Y (s x n) from the items' partials: exact sums over the slabs, one rounding,
// times sqrt(2 / s) c_k.  One thread per (slot, column).
__global__ void __launch_bounds__(256) k_fd_reduce(int n, int s, int cblocks, int slabs, const int* __restrict__ ntiles,
                                                   const int* __restrict__ slots, const uint32_t* __restrict__ colHi,
                                                   const int* __restrict__ colU, const uint32_t* __restrict__ idx,
                                                   const long long* __restrict__ part, double* __restrict__ Y, Ctl* ctl,
                                                   int level) {
  if (level_inactive(ctl, level) || ctl->lvl_status != 0) return;
  const int c = (int)blockIdx.y * kM + (threadIdx.x & (kM - 1));
  const int slot = 2 * (int)blockIdx.x + (int)(threadIdx.x >> 7);
  if (c >= n || slot >= kFdTile * *ntiles || slots[slot] == -1) return;
  const int i = slots[slot] & 0x7FFFFFFF;
  const long long* p = part + ((size_t)(slot / kFdTile) * cblocks + blockIdx.y) * slabs * kPartFd +
                       (size_t)(slot % kFdTile) * kM + (c & (kM - 1));
  oz::I128 acc{0, 0};
  for (int sl = 0; sl < slabs; ++sl, p += kPartFd)
    oz::i128_add(acc, oz::i128_from_parts(p[0], p[kM * kFdTile]));
  const uint32_t Ec = oz::exp_field(colHi[c]);
  const double coef = sqrt(2.0 / (double)s) * (idx[i] == 0 ? 0.70710678118654752440 : 1.0);
  const double y = Ec == 2047u ? nan64() : oz::i128_to_double(acc, colU[c] + 1 + 1023 - oz::kScaleBias) * coef;
  Y[(int64_t)c * s + i] = y;
  if (!isfinite(y)) {
    ctl->input_nonfinite = 1;
    raise_level_status(ctl, ST_NONFINITE);
  }
}

// The split of a problem: equal ranges of at most Jc rows j1 (a multiple of
// 128) that fit the scratch, each in slabs; about four items per CTA over all
// tiles.  Only the rows left run in the last range (a range of Jc rows each time
// did twice the work at J just above a multiple of Jc: m = 10^6, n = 128, s = 256, the
// whole mrcqr_sketch call 6.85 ms, 4.30 now; a factorization 11.1 and 9.8).
struct FdPlan {
  int64_t J, Jc, rows;
  int chunks, cblocks, slabs, max_tiles;
  // rows of range k, rounded up to 128, and its slabs
  int64_t range(int k) const { return std::min(Jc, (J + kM - 1) / kM * kM - k * Jc); }
  int range_slabs(int k) const { return (int)((range(k) + rows - 1) / rows); }
};

FdPlan fd_plan(int64_t m, int n, int s, size_t scratch_bytes) {
  FdPlan p{};
  p.J = m / kR;
  const int64_t J128 = (p.J + kM - 1) / kM * kM;
  p.Jc = std::min(J128, (int64_t)(scratch_bytes / (8ull * kRows * (uint64_t)n)) / kM * kM);
  if (p.Jc <= 0) return p;
  p.chunks = (int)((J128 + p.Jc - 1) / p.Jc);
  p.Jc = ((J128 + p.chunks - 1) / p.chunks + kM - 1) / kM * kM;
  p.cblocks = (n + kM - 1) / kM;
  p.max_tiles = kClasses + s / kFdTile;
  const int64_t want = (8 * (int64_t)device_sms() + p.max_tiles * p.cblocks * p.chunks - 1) / (p.max_tiles * p.cblocks * p.chunks);
  const int64_t slabs = std::max<int64_t>(1, std::min(want, p.Jc / kM));
  p.rows = (p.Jc + slabs - 1) / slabs;
  p.rows = (p.rows + kM - 1) / kM * kM;
  p.slabs = (int)((p.Jc + p.rows - 1) / p.rows);
  return p;
}

constexpr size_t kFdSmem = (size_t)kRABytes + 2 * (size_t)kRBBytes + 1024;

}  // namespace

// m a multiple of 32 (the radix) and at least 2^15, DCT, s >= kFdMinRows.
bool sketch_fd_eligible(int64_t m, int n, int s, int tf, const void* scratch, size_t scratch_bytes,
                        size_t scratch_stride) {
  if (tf != T_DCT || m % kR != 0 || m < (1 << 15) || s < kFdMinRows) return false;
  if (!scratch || (reinterpret_cast<uintptr_t>(scratch) & 15) != 0 || scratch_stride % 16 != 0) return false;
  const FdPlan p = fd_plan(m, n, s, scratch_bytes);
  return p.Jc > 0 && p.chunks <= 4;
}

size_t sketch_fd_part_bytes(int64_t m, int n, int s, size_t scratch_bytes) {
  if (m % kR != 0 || m < (1 << 15) || s < kFdMinRows) return 0;
  const FdPlan p = fd_plan(m, n, s, scratch_bytes);
  if (p.Jc <= 0) return 0;
  return sizeof(long long) * kPartFd * (size_t)p.max_tiles * p.cblocks * p.slabs * p.chunks;
}

size_t sketch_fd_ints_bytes(int64_t m, int s) {
  if (m % kR != 0 || m < (1 << 15) || s < kFdMinRows) return 0;
  const int tiles = kClasses + s / kFdTile;
  return sizeof(int) * (size_t)(64 + 512 + tiles + (size_t)kFdTile * tiles) + sizeof(uint32_t) * (size_t)(m / kR) + 1024;
}

void launch_sketch_fd(int64_t m, int n, int s, const double* A, int64_t lda, const uint32_t* idx, uint4* tabd,
                      uint64_t seed, uint32_t* colHi, long long* part, void* ints, double* Y, void* scratch,
                      size_t scratch_bytes, size_t scratch_stride, Ctl* ctl, int level, cudaStream_t st) {
  const FdPlan p = fd_plan(m, n, s, scratch_bytes);
  int* ntiles = static_cast<int*>(ints);
  int* colU = ntiles + 64;
  int* cls = colU + 512;
  int* slots = cls + (p.max_tiles + 63) / 64 * 64;
  uint32_t* sgn = reinterpret_cast<uint32_t*>(slots + kFdTile * p.max_tiles);
  cudaMemsetAsync(colHi, 0, syrk_oz_colhi_bytes(n), st);
  cudaMemsetAsync(colU, 0, sizeof(int) * 512, st);
  launch_dep(k_fd_bounds, dim3((unsigned)((p.J + 255) / 256), (unsigned)n), 256, 0, st, p.J, A, lda, colHi, colU, ctl, level);
  launch_dep(k_fd_table, (unsigned)((m + 256) / 256), 256, 0, st, m, tabd, ctl, level);
  launch_dep(k_fd_signs, (unsigned)((p.J + 31) / 32), 256, 0, st, p.J, seed_key(seed), sgn, ctl, level);
  launch_dep(k_fd_classes, 1, 1024, 0, st, s, idx, ntiles, cls, slots, ctl, level);
  cudaFuncSetAttribute(k_fd_pass1, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFdSmem);
  cudaFuncSetAttribute(k_fd_pass2, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFdSmem);
  uint64_t* U = static_cast<uint64_t*>(scratch);
  const int64_t cs = scratch_stride ? (int64_t)(scratch_stride / 8) : kRows * p.Jc;
  int slab0 = 0, slabs_all = 0;
  for (int k = 0; k < p.chunks; ++k) slabs_all += p.range_slabs(k);
  for (int k = 0; k < p.chunks; ++k) {
    const int64_t j0 = (int64_t)k * p.Jc;
    const int nblocks = (int)(p.range(k) / kM), slabs = p.range_slabs(k);   // rows j1 >= J give zero words
    const int64_t items = (int64_t)nblocks * n;
    launch_dep(k_fd_pass1, (unsigned)std::min<int64_t>(items, 2 * device_sms()), kRThreads, kFdSmem, st, p.J, j0, p.Jc, nblocks, n, A, lda, colHi, colU, sgn, U, cs, ctl, level);
    const Fd2Args a{m, p.J, j0, p.Jc, p.rows, p.range(k), n, p.cblocks, slabs, U, cs, idx, tabd, ntiles, cls, slots, part,
                    slab0, slabs_all};
    slab0 += slabs;
    const int64_t most = (int64_t)p.max_tiles * p.cblocks * slabs;
    launch_dep(k_fd_pass2, (unsigned)std::min<int64_t>(most, 2 * device_sms()), kRThreads, kFdSmem, st, a, ctl, level);
  }
  const dim3 rg((unsigned)(kFdTile * p.max_tiles / 2), (unsigned)p.cblocks);
  launch_dep(k_fd_reduce, rg, 256, 0, st, n, s, p.cblocks, slabs_all, ntiles, slots, colHi, colU, idx, part, Y, ctl, level);
}

}  // namespace mrcqr
