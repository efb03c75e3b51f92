// FP64 products of the method on FP16 tensor cores with exact integer
// slicing (ozaki.cuh): the Gram matrix and the check Q^T Q (Algorithm 1
// step 1, Sec. II-C), the FP64 sketch (Algorithm 2 steps 2-4 at p = FP64) and, for
// wide W, Q = W R_c^{-1}.
// Each result entry is the once-rounded value of a 63-bit fixed-point
// evaluation of its sum.  (The row-block products W = A R_s^{-1} and Q = W R_c^{-1}
// of narrow W are in rowprod.cu.)
//
// All of them run the same two-stage pipeline per CTA (one CTA per SM, 512
// threads, all 512 TMEM columns = 8 level accumulators of 128 x 64): the
// threads write the digit panels of K chunk c + 1 (32 deep, K-major
// SWIZZLE_64B) into one shared-memory stage while the tensor cores run the
// 36 digit-pair MMAs of chunk c from the other; every 4 chunks (K = 128, the
// exactness limit) the level sums are read out of TMEM into 64-bit integers.
#include <algorithm>

#include "kernels.h"
#include "ozaki.cuh"
#include "tc.cuh"
#include "ozaki_pipe.cuh"

namespace mrcqr {

int device_sms() {
  static int cached = 0;
  if (!cached) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cached = sms > 0 ? sms : 152;
  }
  return cached;
}

namespace {

// ---------------------------------------------------------------------------
// Q = W X in place (X = R_c^{-1} upper, Algorithm 1 step 3) in 128 x 64 tiles by
// one CTA per SM, for wide W (rp_wide; rowprod.cu has 128 x 32 tiles by two
// CTAs).  A tile of twice the width slices every chunk of W half as often and issues
// 10% fewer MMA cycles, but one CTA holds all of TMEM, so nothing covers its row
// blocks' other phases: it pays once a block is many chunks long.  Measured at m = 2^20
// (us, 32 / 64 columns): n = 128 1975 / 2135, 192 3786 / 3645, 256 5810 / 5290, 288
// 7392 / 7557, 320 8786 / 7738, 384 11656 / 9945, 512 19111 / 15801; m = 2^18: n = 96 552 / 712,
// 160 1033 / 1167, 352 3064 / 2988.  Integer work around the products bounds both.
// Multiplier digits: block (t, kc), kc <= 2 t + 1, of columns [64 t, 64 t + 64) and
// rows [32 kc, 32 kc + 32) of X as eight K-major SWIZZLE_64B panels.
__host__ __device__ __forceinline__ size_t fw_block_offset(int t, int kc) {
  return ((size_t)t * (t + 1) + kc) * (oz::kSlices * kBPanel);
}

__device__ __forceinline__ void fw_prep_col(int n, int npad, const double* __restrict__ XT, int* __restrict__ colE,
                                            unsigned char* __restrict__ Xs, uint32_t* __restrict__ colHiOut, int nhi,
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
  const int E = (int)oz::exp_field(all), t = j / kN;
  if (threadIdx.x == 0 && j < n) colE[j] = E;
  for (int k = threadIdx.x; k < 2 * kK * (t + 1); k += blockDim.x) {
    int dg[oz::kSlices];
    const double v = (k < n && j < n) ? XT[(int64_t)k * npad + j] : 0.0;
    oz::digits8((uint32_t)__double2hiint(v), (uint32_t)__double2loint(v), E, dg);
    unsigned char* panel = Xs + fw_block_offset(t, k / kK) + tc::sw64_offset(j % kN, k % kK, 2);
#pragma unroll
    for (int b = 0; b < oz::kSlices; ++b)
      *reinterpret_cast<__half*>(panel + b * kBPanel) = __float2half_rn(oz::small_int_to_float(dg[b]));
  }
}

__global__ void __launch_bounds__(128) k_fw_prep(int n, int npad, const double* __restrict__ XT, int* __restrict__ colE,
                                                 unsigned char* __restrict__ Xs, uint32_t* __restrict__ colHiOut, int nhi,
                                                 const Ctl* ctl, int level) {
  if (level_inactive(ctl, level) || ctl->lvl_status != 0) return;
  __shared__ uint32_t red[4];
  fw_prep_col(n, npad, XT, colE, Xs, colHiOut, nhi, blockIdx.x, red);
}

// Row blocks of 128 from block rb0 on, every `step`; output tiles from right to left.  False when a wait gave up.
__device__ __forceinline__ bool fw_blocks(int64_t m, int n, double* __restrict__ Q, int64_t ldq,
                                          const int* __restrict__ colE, const unsigned char* __restrict__ Xs,
                                          uint32_t* __restrict__ colHiOut, int64_t rb0, int64_t step, OzPipe& P,
                                          unsigned char* smem, int* rowE, uint32_t (*red)[kM], uint32_t* cmax) {
  const int tid = threadIdx.x, lane = tid & 31, ntiles = (n + kN - 1) / kN;
  const int pr = tid & (kM - 1), pp = tid >> 7, rot = (lane >> 3) & 1;   // producer: row pr, columns 8 pp .. + 7
  const int rr = P.q * 32 + lane;
  __syncthreads();
  for (int j = tid; j < n; j += kOzThreads) cmax[j] = 0u;   // read after the first row maxima's barrier
  uint32_t off[2];
  int gcol[2];
#pragma unroll
  for (int j = 0; j < 2; ++j) {   // rows r and r + 8 in opposite order: a half warp's 8-byte stores cover all banks
    gcol[j] = 8 * pp + 4 * (j ^ rot);
    off[j] = tc::sw64_offset(pr, gcol[j], 2);
  }
  for (int64_t rb = rb0; rb * kM < m; rb += step) {
    const int64_t r0 = rb * kM, prow = min(r0 + pr, m - 1);   // rows beyond m: row m - 1 again, not stored
    const int64_t rn = r0 + step * kM;
    if (rn < m)   // the next block into L2
      for (int e = tid; e < 8 * n; e += kOzThreads)
        tc::prefetch_l2(Q + min(rn + 16 * (e & 7), m - 1) + (int64_t)(e >> 3) * ldq);
    uint32_t mx = 0u;
    const double* p = Q + prow + (int64_t)pp * ldq;
#pragma unroll 8
    for (int c = pp; c < n; c += 4) {
      mx = max(mx, (uint32_t)__double2hiint(*p) & 0x7FFFFFFFu);
      p += 4 * ldq;
    }
    red[pp][pr] = mx;
    __syncthreads();
    if (tid < kM) rowE[tid] = (int)oz::exp_field(max(max(red[0][tid], red[1][tid]), max(red[2][tid], red[3][tid])));
    __syncthreads();
    const int Er = rowE[pr], cr = oz_quad_cr(Er), Erow = rowE[rr];
    const bool rlive = r0 + rr < m;
    for (int t = ntiles - 1; t >= 0; --t) {
      long long hi[16], lo[16];
#pragma unroll
      for (int c = 0; c < 16; ++c) hi[c] = lo[c] = 0;
      double v[2][4];
      auto load_w = [&](int kc) {
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const int k0 = kc * kK + gcol[j];
          const double* w = Q + prow + (int64_t)k0 * ldq;
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            v[j][c] = k0 + c < n ? *w : 0.0;
            w += ldq;
          }
        }
      };
      load_w(0);
      const int nch = 2 * (t + 1);
      auto produce = [&](int kc, unsigned char* a, unsigned char* b) {
        const unsigned char* src = Xs + fw_block_offset(t, kc);
#pragma unroll
        for (int i = 0; i < (int)(oz::kSlices * kBPanel / 16 / kOzThreads); ++i)
          tc::cp_async16(b + 16 * (tid + kOzThreads * i), src + 16 * (tid + kOzThreads * i));
        const uint32_t sa = tc::smem_u32(a);
#pragma unroll
        for (int j = 0; j < 2; ++j) oz_store_quad(v[j], 0u, Er, cr, sa + off[j], kAPanel);
        if (kc + 1 < nch) load_w(kc + 1);
        tc::cp_async_wait_all();
      };
      if (!oz_run(P, smem, nch, produce, hi, lo)) return false;
      const int c0 = t * kN + P.g * 16;
      double* q = Q + r0 + rr + (int64_t)c0 * ldq;
#pragma unroll
      for (int c = 0; c < 16; ++c) {
        if (rlive && c0 + c < n) {
          const int ce = colE[c0 + c], scale = Erow + ce - oz::kScaleBias;
          double x = (c & 1) ? oz::t96_to_double_fp64(hi[c], lo[c], scale) : oz::t96_to_double(hi[c], lo[c], scale);
          if (Erow == 2047 || ce == 2047) x = nan64();   // non-finite operands
          *q = x;
          const uint32_t h = (uint32_t)__double2hiint(x) & 0x7FFFFFFFu;
          if (h > cmax[c0 + c]) atomicMax(cmax + c0 + c, h);
        }
        q += ldq;
      }
      __syncthreads();   // the tile's Q before the next tile's loads, the panels free
    }
  }
  __syncthreads();
  if (colHiOut)
    for (int j = tid; j < n; j += kOzThreads)
      if (cmax[j]) atomicMax(colHiOut + j, cmax[j]);
  return true;
}

__global__ void __launch_bounds__(kOzThreads, 1)
    k_fw_product(int64_t m, int n, double* __restrict__ Q, int64_t ldq, const int* __restrict__ colE,
                 const unsigned char* __restrict__ Xs, uint32_t* __restrict__ colHiOut, Ctl* ctl, int level) {
  if (level_inactive(ctl, level) || ctl->lvl_status != 0) return;
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t mma_bar[2];
  __shared__ uint32_t tmem_slot;
  __shared__ int rowE[kM];
  __shared__ uint32_t red[4][kM], cmax[512];
  OzPipe P = oz_begin(&tmem_slot, mma_bar);
  const bool ok = fw_blocks(m, n, Q, ldq, colE, Xs, colHiOut, blockIdx.x, gridDim.x, P, oz_smem(smem_raw), rowE, red, cmax);
  oz_end(P, !ok, ctl);
}

// Grouped forms for batched plans: items {i, column < n64} and {i, 128-row block}.
__global__ void __launch_bounds__(128) kg_fw_prep(Group g, int level) {
  __shared__ uint32_t red[4];
  for (int it = blockIdx.x; it < g.nitems; it += gridDim.x) {
    const int4 w = g.items[it];
    const Prob& P = g.probs[w.x];
    if (P.ctl->active != level || P.ctl->lvl_status != 0) continue;
    fw_prep_col(P.n, P.npad, P.xt, P.oz_xe, P.oz_xs, P.check ? P.oz_colhi : nullptr, (P.n + kM - 1) / kM * kM, w.y, red);
    __syncthreads();
  }
}

__global__ void __launch_bounds__(kOzThreads, 1) kg_fw_product(Group g, int level) {
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t mma_bar[2];
  __shared__ uint32_t tmem_slot;
  __shared__ int rowE[kM];
  __shared__ uint32_t red[4][kM], cmax[512];
  OzPipe P = oz_begin(&tmem_slot, mma_bar);
  bool abort = false;
  Ctl* actl = nullptr;
  for (int it = blockIdx.x; it < g.nitems; it += gridDim.x) {
    const int4 w = g.items[it];
    const Prob& B = g.probs[w.x];
    if (B.ctl->active != level || B.ctl->lvl_status != 0) continue;
    if (!fw_blocks(B.m, B.n, B.Q, B.ldq, B.oz_xe, B.oz_xs, B.check ? B.oz_colhi : nullptr, w.y, (B.m + kM - 1) / kM, P,
                   oz_smem(smem_raw), rowE, red, cmax)) {
      abort = true;
      actl = B.ctl;
      break;
    }
  }
  oz_end(P, abort, actl);
}

// ---------------------------------------------------------------------------
// Gram G = W^T W (Algorithm 1 step 1) and the check matrix Q^T Q.  Every
// column of W is sliced against the exponent of its maximum over all m rows,
// so the level sums of all rows share one scale: a work item (output tile of
// 128 x 64 entries, slab of rows) reads its exact level sums out of TMEM
// every 128 rows into 64-bit integer pairs, and a reduction adds the items'
// 128-bit values (exact, so the order does not matter) and rounds each entry
// once.

// Column maxima (as the high word of |x|, whose exponent field is the
// reference exponent) over all rows; colHi must be zero on entry.
__global__ void __launch_bounds__(256) k_col_hi(int64_t m, int n, const double* __restrict__ W, int64_t ldw,
                                                int64_t rows_per_cta, uint32_t* __restrict__ colHi, const Ctl* ctl,
                                                int level) {
  if (level_inactive(ctl, level) || ctl->lvl_status != 0) return;
  const int j = blockIdx.x;
  const int64_t r0 = (int64_t)blockIdx.y * rows_per_cta;
  const int64_t r1 = min(m, r0 + rows_per_cta);
  const double* col = W + (int64_t)j * ldw;
  uint32_t mx = 0u;
  for (int64_t r = r0 + threadIdx.x; r < r1; r += 256)
    mx = max(mx, (uint32_t)__double2hiint(__ldg(col + r)) & 0x7FFFFFFFu);
  __shared__ uint32_t red[8];
  mx = __reduce_max_sync(0xffffffffu, mx);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t v = red[0];
    for (int w = 1; w < 8; ++w) v = max(v, red[w]);
    if (v) atomicMax(colHi + j, v);
  }
}

// One work item (output tile, row slab) of the Gram W^T W; false when a wait
// timed out (every thread together).
// ti, tj: the tile's I block (128 columns) and J block (64 columns); rows
// [r_begin, min(m, r_begin + rows_per_slab)); the partial goes to part_item.
__device__ __forceinline__ bool syrk_oz_item(int64_t m, int n, const double* __restrict__ W, int64_t ldw,
                                             const uint32_t* __restrict__ colHi, int ti, int tj, int64_t r_begin,
                                             int64_t rows_per_slab, long long* __restrict__ part_item, OzPipe& P,
                                             unsigned char* smem, uint32_t* colE) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int i0 = kM * ti, j0 = kN * tj;
  const bool inner = (tj >> 1) == ti;   // J block inside the I block
  const int64_t r_end = min(m, r_begin + rows_per_slab);
  const int nchunks = r_end > r_begin ? (int)((r_end - r_begin + kK - 1) / kK) : 0;
  __syncthreads();
  if (tid < kM) colE[tid] = i0 + tid < n ? oz::exp_field(colHi[i0 + tid]) : 0u;
  else if (tid < kM + kN) colE[tid] = j0 + tid - kM < n ? oz::exp_field(colHi[j0 + tid - kM]) : 0u;
  __syncthreads();
  long long hi[16], lo[16];
#pragma unroll
  for (int c = 0; c < 16; ++c) hi[c] = lo[c] = 0;
  // A operand: column tid / 4 of the I block, 16-byte chunk tid % 4 (two groups of four rows; the second
  // half of each eight columns stores them in opposite order, so a half warp's 8-byte stores hit all banks).
  // B operand of an off-diagonal tile: column tid / 8 of the J block, four rows.
  const int ac = tid >> 2, rot = (lane >> 3) & 1, bc = tid >> 3;
  const bool vec = (reinterpret_cast<uintptr_t>(W) & 15) == 0 && (ldw & 1) == 0;   // slabs start at multiples of 32
  const bool alive = i0 + ac < n, blive = !inner && j0 + bc < n;
  const double* acol = W + (int64_t)(i0 + ac) * ldw;
  const double* bcol = W + (int64_t)(j0 + bc) * ldw;
  const int Ea = (int)colE[ac], Eb = (int)colE[kM + bc];
  const int cra = oz_quad_cr(Ea), crb = oz_quad_cr(Eb);
  uint32_t aoff[2], doff[2];
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const int k = 8 * (tid & 3) + 4 * (j ^ rot);
    aoff[j] = tc::sw64_offset(ac, k, 2);
    const int d = ac - (j0 - i0);   // the J block is part of the I block of an inner tile: store these columns twice
    doff[j] = inner && d >= 0 && d < kN ? oz::kSlices * kAPanel + tc::sw64_offset(d, k, 2) : 0u;
  }
  const uint32_t boff = oz::kSlices * kAPanel + tc::sw64_offset(bc, 4 * (tid & 7), 2);
  double va[2][4], vb[4];
  auto load = [&](int64_t r0) {
    if (alive) {
#pragma unroll
      for (int j = 0; j < 2; ++j) oz_load_quad(acol, r0 + 8 * (tid & 3) + 4 * (j ^ rot), r_end, vec, va[j]);
    }
    if (blive) oz_load_quad(bcol, r0 + 4 * (tid & 7), r_end, vec, vb);
  };
  load(r_begin);
  {   // columns beyond n: zero digits in both stages, written once
    const uint32_t s0 = tc::smem_u32(smem);
#pragma unroll
    for (int st = 0; st < 2; ++st)
#pragma unroll
      for (int a = 0; a < oz::kSlices; ++a) {
        if (!alive) {
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            tc::st_shared2(s0 + st * kStage + aoff[j] + a * kAPanel, 0u, 0u);
            if (doff[j]) tc::st_shared2(s0 + st * kStage + doff[j] + a * kBPanel, 0u, 0u);
          }
        }
        if (!inner && !blive) tc::st_shared2(s0 + st * kStage + boff + a * kBPanel, 0u, 0u);
      }
  }
  auto produce = [&](int ch, unsigned char* a, unsigned char*) {
    const uint32_t sa = tc::smem_u32(a);
    if (alive) {
#pragma unroll
      for (int j = 0; j < 2; ++j)
        oz_store_quad(va[j], 0u, Ea, cra, sa + aoff[j], kAPanel, doff[j] ? sa + doff[j] : 0u, kBPanel);
    }
    if (blive) oz_store_quad(vb, 0u, Eb, crb, sa + boff, kBPanel);
    if (ch + 1 < nchunks) load(r_begin + (int64_t)(ch + 1) * kK);
  };
  if (!oz_run(P, smem, nchunks, produce, hi, lo)) return false;
  oz_store_partial(part_item, P.q, P.g, lane, hi, lo);
  return true;
}

__global__ void __launch_bounds__(kOzThreads, 1)
    k_syrk_oz(int64_t m, int n, const double* __restrict__ W, int64_t ldw, const uint32_t* __restrict__ colHi,
              SyrkOzPlan SP, long long* __restrict__ part, Ctl* ctl, int level) {
  if (level_inactive(ctl, level) || ctl->lvl_status != 0) return;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = oz_smem(smem_raw);
  __shared__ __align__(8) uint64_t mma_bar[2];
  __shared__ uint32_t tmem_slot;
  __shared__ uint32_t colE[kM + kN];
  OzPipe P = oz_begin(&tmem_slot, mma_bar);
  bool abort = false;
  const int nitems = SP.ntiles * SP.slabs;
  for (int item = blockIdx.x; item < nitems; item += gridDim.x) {
    const int tile = item % SP.ntiles, slab = item / SP.ntiles;
    if (!syrk_oz_item(m, n, W, ldw, colHi, SP.ti[tile], SP.tj[tile], (int64_t)slab * SP.rows_per_slab,
                      SP.rows_per_slab, part + (size_t)item * kPartElems, P, smem, colE)) {
      abort = true;
      break;
    }
  }
  oz_end(P, abort, ctl);
}

// Upper triangle of G from the items' partials (exact 128-bit sums over the
// slabs, one rounding); lower triangle zero.
template <class Plan>
__device__ __forceinline__ void syrk_oz_reduce_entry(int n, const uint32_t* __restrict__ colHi, const Plan& SP,
                                                     const long long* __restrict__ part, double* __restrict__ out,
                                                     int64_t e) {
  if (e >= (int64_t)n * n) return;
  const int i = (int)(e % n), j = (int)(e / n);
  if (i > j) {
    out[e] = 0.0;
    return;
  }
  const int I = i / kM, J = j / kN;
  const int tile = SP.tile_of[I][J];
  const oz::I128 acc =
      oz_sum_partials(part + (size_t)tile * kPartElems, SP.slabs, (size_t)SP.ntiles * kPartElems, i - I * kM, j - J * kN);
  const uint32_t Ei = oz::exp_field(colHi[i]), Ej = oz::exp_field(colHi[j]);
  out[e] = (Ei == 2047u || Ej == 2047u) ? nan64() : oz::i128_to_double(acc, (int)Ei + (int)Ej - oz::kScaleBias);
}

__global__ void k_syrk_oz_reduce(int n, const uint32_t* __restrict__ colHi, SyrkOzPlan SP,
                                 const long long* __restrict__ part, double* __restrict__ out, const Ctl* ctl,
                                 int level) {
  if (level_inactive(ctl, level) || ctl->lvl_status != 0) return;
  syrk_oz_reduce_entry(n, colHi, SP, part, out, (int64_t)blockIdx.x * blockDim.x + threadIdx.x);
}

// ---------------------------------------------------------------------------
// FP64 sketch (Algorithm 2 steps 2-4 with p = FP64) as an emulated GEMM:
//   P[c][i] = sum_j (d_j A[j][c]) F[i][j],  F[i][j] = cos(pi r_ij / (2m)),
//   r_ij = k_i (2j + 1) mod 4m,
// with F[i][j] the FP64 quarter-wave table value (the value the FMA kernel
// multiplies with) and d_j the Rademacher sign; then Y[i][c] =
// sqrt(2/s) c_k(i) P[c][i].  A's columns are sliced against their maxima over
// all m rows, the table values against 2^0 (|F| <= 1).  Work item = (block of
// 128 columns of A, 64 sampled rows, slab of rows of A).
// One work item (128 columns of A, 64 sampled rows, row slab) of the FP64
// sketch; false when a wait timed out (every thread together).
__device__ __forceinline__ bool sketch_oz_item(int64_t m, int n, int s, const double* __restrict__ A, int64_t lda,
                                               const uint32_t* __restrict__ colHi, const uint32_t* __restrict__ idx,
                                               const double* __restrict__ tab, uint2 key, const SketchOzPlan& SP,
                                               long long* __restrict__ part, int tf, OzPipe& P,
                                               unsigned char* smem, uint32_t* colE, uint32_t* sgn, int item) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint64_t four_m = 4ull * (uint64_t)m;
  // signs of the rows r0 .. r0 + 31 as a bit mask, one Philox draw per lane of warp 1
  auto sign_mask = [&](int64_t r0, int64_t r_end) {
    const int64_t j = r0 + lane;
    const bool neg = j < r_end && row_sign((uint64_t)j, key) < 0.0;
    return __ballot_sync(0xffffffffu, neg);
  };
  const int ntiles_all = SP.mblocks * SP.ntiles;
  const int nitems = ntiles_all * SP.slabs;
  // transform-panel role: sample fi, rows 4 fg .. 4 fg + 3 of each chunk
  const int fi = tid & (kN - 1), fg = tid >> 6;
  // sign role: rows 2 (lane % 16), 2 (lane % 16) + 1 of each chunk
  const int sp = lane & 15;

  const int tile = item % ntiles_all, slab = item / ntiles_all;
  const int c0 = kM * (tile / SP.ntiles), i0 = kN * (tile % SP.ntiles);
  const int64_t r_begin = (int64_t)slab * SP.rows_per_slab;
  const int64_t r_end = min(m, r_begin + SP.rows_per_slab);
  const int nchunks = r_end > r_begin ? (int)((r_end - r_begin + kK - 1) / kK) : 0;
  __syncthreads();
  if (tid < kM) colE[tid] = c0 + tid < n ? oz::exp_field(colHi[c0 + tid]) : 0u;
  if (warp == 1) {
    const uint32_t mk = sign_mask(r_begin, r_end);
    if (lane == 0) sgn[0] = mk;
  }
  __syncthreads();
  // phase of (sample fi, row r_begin + 4 fg), its advance per chunk and per row
  const bool fval = i0 + fi < s;
  const RowPhase rp = row_phase(tf, fval ? idx[i0 + fi] : 0u, (uint64_t)m);
  uint64_t r = fval ? phase_at(rp, (uint64_t)(r_begin + 4 * fg), four_m) : 0ull;
  const uint64_t step_chunk = (rp.dk * (uint64_t)kK) % four_m;
  const uint64_t step_row = rp.dk;   // < 4m
  long long hi[16], lo[16];
#pragma unroll
  for (int c = 0; c < 16; ++c) hi[c] = lo[c] = 0;
  // chunk 0 ahead: A values, table values of this thread's four rows
  double va[kM / 32][2];
  uint32_t whi[4], wlo[4];
  auto load_chunk = [&](int64_t r0) {
    oz_load_cols<kM>(A, lda, n, c0, r0, r_end, warp, lane, va);
    uint64_t rr = r;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      whi[t] = wlo[t] = 0u;
      if (fval && r0 + 4 * fg + t < r_end) cos_phase_bits(tab, (int64_t)rr, m, whi[t], wlo[t]);
      rr += step_row;
      if (rr >= four_m) rr -= four_m;
    }
    r += step_chunk;
    if (r >= four_m) r -= four_m;
  };
  load_chunk(r_begin);
  auto produce = [&](int ch, unsigned char* a, unsigned char* b) {
    const int64_t r0 = r_begin + (int64_t)ch * kK;
    // Rademacher signs of this lane's two rows (mask of this chunk made one chunk ahead by warp 1;
    // the pipeline's barrier between chunks publishes it)
    const uint32_t mk = sgn[ch & 1];
    const uint32_t f0 = (mk >> (2 * sp)) & 1u, f1 = (mk >> (2 * sp + 1)) & 1u;
    if (warp == 1 && ch + 1 < nchunks) {
      const uint32_t mk1 = sign_mask(r0 + kK, r_end);
      if (lane == 0) sgn[(ch + 1) & 1] = mk1;
    }
    oz_store_cols<kM>(va, colE, f0, f1, a, kAPanel, warp, lane);
#pragma unroll
    for (int t2 = 0; t2 < 2; ++t2)
      oz_store_pair(__hiloint2double((int)whi[2 * t2], (int)wlo[2 * t2]),
                    __hiloint2double((int)whi[2 * t2 + 1], (int)wlo[2 * t2 + 1]), 0u, 0u, 1023u,
                    tc::smem_u32(b) + tc::sw64_offset(fi, 4 * fg + 2 * t2, 2), kBPanel);
    if (ch + 1 < nchunks) load_chunk(r0 + kK);
  };
  if (!oz_run(P, smem, nchunks, produce, hi, lo)) return false;
  oz_store_partial(part + (size_t)item * kPartElems, P.q, P.g, lane, hi, lo);
  return true;
}

__global__ void __launch_bounds__(kOzThreads, 1)
    k_sketch_oz(int64_t m, int n, int s, const double* __restrict__ A, int64_t lda, const uint32_t* __restrict__ colHi,
                const uint32_t* __restrict__ idx, const double* __restrict__ tab, uint2 key, SketchOzPlan SP,
                long long* __restrict__ part, Ctl* ctl, int level, int tf) {
  if (level_inactive(ctl, level) || ctl->lvl_status != 0) return;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = oz_smem(smem_raw);
  __shared__ __align__(8) uint64_t mma_bar[2];
  __shared__ uint32_t tmem_slot;
  __shared__ uint32_t colE[kM];
  __shared__ uint32_t sgn[2];   // Rademacher signs of a chunk's 32 rows (bit i: row r0 + i), by chunk parity
  OzPipe P = oz_begin(&tmem_slot, mma_bar);
  bool abort = false;
  const int nitems = SP.mblocks * SP.ntiles * SP.slabs;
  for (int item = blockIdx.x; item < nitems; item += gridDim.x)
    if (!sketch_oz_item(m, n, s, A, lda, colHi, idx, tab, key, SP, part, tf, P, smem, colE, sgn, item)) {
      abort = true;
      break;
    }
  oz_end(P, abort, ctl);
}

// Y (s x n, column-major) from the items' partials: exact sums over the
// slabs, one rounding, times the row's scale (DCT: sqrt(2/s) c_k; real FFT:
// sqrt(c/m) for c bins).  A non-finite column of A gives a NaN column and
// raises NONFINITE.
__device__ __forceinline__ void sketch_oz_reduce_entry(int n, int s, const uint32_t* __restrict__ colHi,
                                                       const uint32_t* __restrict__ idx, const SketchOzPlan& SP,
                                                       const long long* __restrict__ part, double* __restrict__ Y,
                                                       Ctl* ctl, int tf, int64_t m, int64_t e) {
  if (e >= (int64_t)s * n) return;
  const int i = (int)(e % s), c = (int)(e / s);
  const int tile = (c / kM) * SP.ntiles + i / kN;
  const oz::I128 acc = oz_sum_partials(part + (size_t)tile * kPartElems, SP.slabs,
                                       (size_t)SP.mblocks * SP.ntiles * kPartElems, c % kM, i % kN);
  const uint32_t Ec = oz::exp_field(colHi[c]);
  const double coef = tf == T_DCT ? sqrt(2.0 / (double)s) * (idx[i] == 0 ? 0.70710678118654752440 : 1.0)
                                  : sqrt((double)(tf == T_RFFT_REIM ? s / 2 : s) / (double)m);
  const double y = Ec == 2047u ? nan64() : oz::i128_to_double(acc, (int)Ec + 1023 - oz::kScaleBias) * coef;
  Y[e] = y;
  if (!isfinite(y)) {
    ctl->input_nonfinite = 1;
    raise_level_status(ctl, ST_NONFINITE);
  }
}

__global__ void k_sketch_oz_reduce(int n, int s, const uint32_t* __restrict__ colHi, const uint32_t* __restrict__ idx,
                                   SketchOzPlan SP, const long long* __restrict__ part, double* __restrict__ Y,
                                   Ctl* ctl, int level, int tf, int64_t m) {
  if (level_inactive(ctl, level) || ctl->lvl_status != 0) return;
  sketch_oz_reduce_entry(n, s, colHi, idx, SP, part, Y, ctl, tf, m, (int64_t)blockIdx.x * blockDim.x + threadIdx.x);
}

// ---------------------------------------------------------------------------
// Grouped forms for batched plans (many problems of uneven m and n): one
// persistent launch per kernel walks a work list of {problem, block} items
// with a grid-stride loop; an item whose problem is not active at this
// escalation level, or has raised a status, is skipped.  The per-item work is
// the single-problem kernels' body; a CTA that moves on to another problem
// folds its column maxima into the previous one's first.

__device__ __forceinline__ bool oz_live(const Prob& P, int level) {
  return P.ctl->active == level && P.ctl->lvl_status == 0;
}

__device__ __forceinline__ int oz_nhi(int n) { return (n + kM - 1) / kM * kM; }

// Column maxima of A (high words of |a|), one column per item, entries
// n .. nhi - 1 zero.
__global__ void __launch_bounds__(256) kg_oz_colhi(Group g, int level) {
  __shared__ uint32_t red[8];
  for (int it = blockIdx.x; it < g.nitems; it += gridDim.x) {
    const int4 w = g.items[it];
    const Prob& P = g.probs[w.x];
    if (!oz_live(P, level)) continue;
    const int j = w.y;
    uint32_t mx = 0u;
    if (j < P.n) {
      const double* col = P.A + (int64_t)j * P.lda;
      for (int64_t r = threadIdx.x; r < P.m; r += 256)
        mx = max(mx, (uint32_t)__double2hiint(__ldg(col + r)) & 0x7FFFFFFFu);
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
    __syncthreads();
    if (threadIdx.x == 0) {
      uint32_t v = red[0];
      for (int k = 1; k < 8; ++k) v = max(v, red[k]);
      P.oz_colhi[j] = v;
    }
  }
}

__global__ void __launch_bounds__(kOzThreads, 1) kg_oz_sketch(Group g, int level) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = oz_smem(smem_raw);
  __shared__ __align__(8) uint64_t mma_bar[2];
  __shared__ uint32_t tmem_slot;
  __shared__ uint32_t colE[kM];
  __shared__ uint32_t sgn[2];
  OzPipe pipe = oz_begin(&tmem_slot, mma_bar);
  bool abort = false;
  Ctl* actl = nullptr;
  for (int it = blockIdx.x; it < g.nitems; it += gridDim.x) {
    const int4 w = g.items[it];
    const Prob& P = g.probs[w.x];
    if (!oz_live(P, level)) continue;
    if (!sketch_oz_item(P.m, P.n, P.s, P.A, P.lda, P.oz_colhi, P.idx, P.tab, P.key, P.oz_kp, P.oz_part, P.tf, pipe,
                        smem, colE, sgn, w.y)) {
      abort = true;
      actl = P.ctl;
      break;
    }
  }
  oz_end(pipe, abort, actl);
}

__global__ void __launch_bounds__(256) kg_oz_sketch_reduce(Group g, int level) {
  for (int it = blockIdx.x; it < g.nitems; it += gridDim.x) {
    const int4 w = g.items[it];
    const Prob& P = g.probs[w.x];
    if (!oz_live(P, level)) continue;
    sketch_oz_reduce_entry(P.n, P.s, P.oz_colhi, P.idx, P.oz_kp, P.oz_part, P.y, P.ctl, P.tf, P.m,
                           (int64_t)w.y * 256 + threadIdx.x);
  }
}

__global__ void __launch_bounds__(kOzThreads, 1) kg_oz_syrk(Group g, int level) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = oz_smem(smem_raw);
  __shared__ __align__(8) uint64_t mma_bar[2];
  __shared__ uint32_t tmem_slot;
  __shared__ uint32_t colE[kM + kN];
  OzPipe pipe = oz_begin(&tmem_slot, mma_bar);
  bool abort = false;
  Ctl* actl = nullptr;
  for (int it = blockIdx.x; it < g.nitems; it += gridDim.x) {
    const int4 w = g.items[it];
    const Prob& P = g.probs[w.x];
    if (!oz_live(P, level)) continue;
    const int tile = w.y % P.oz_sp.ntiles, slab = w.y / P.oz_sp.ntiles;
    if (!syrk_oz_item(P.m, P.n, P.Q, P.ldq, P.oz_colhi, P.oz_sp.ti[tile], P.oz_sp.tj[tile],
                      (int64_t)slab * P.oz_sp.rows_per_slab, P.oz_sp.rows_per_slab,
                      P.oz_part + (size_t)w.y * kPartElems, pipe, smem, colE)) {
      abort = true;
      actl = P.ctl;
      break;
    }
  }
  oz_end(pipe, abort, actl);
}

__global__ void __launch_bounds__(256) kg_oz_syrk_reduce(Group g, int check, int level) {
  for (int it = blockIdx.x; it < g.nitems; it += gridDim.x) {
    const int4 w = g.items[it];
    const Prob& P = g.probs[w.x];
    if (!oz_live(P, level)) continue;
    syrk_oz_reduce_entry(P.n, P.oz_colhi, P.oz_sp, P.oz_part, check ? P.e : P.rc, (int64_t)w.y * 256 + threadIdx.x);
  }
}

int gcd_int(int a, int b) { return b ? gcd_int(b, a % b) : a; }

// Row slabs so that tiles x slabs is a multiple of the SM count where the
// rows allow it; at least 256 rows per slab, at most 2^20 (the 64-bit halves
// of an item stay below 2^61).
int choose_slabs(int64_t m, int tiles, int64_t* rows_per_slab) {
  const int sms = device_sms();
  int slabs = tiles >= sms ? 1 : sms / gcd_int(tiles, sms);
  const int64_t max_slabs = (m + 255) / 256;
  if (slabs > max_slabs) slabs = (int)max_slabs;
  const int64_t min_slabs = (m + (1 << 20) - 1) >> 20;
  if (slabs < min_slabs) slabs = (int)min_slabs;
  if (slabs < 1) slabs = 1;
  int64_t rps = (m + slabs - 1) / slabs;
  rps = (rps + kK - 1) / kK * kK;
  *rows_per_slab = rps;
  return (int)((m + rps - 1) / rps);
}

void launch_col_hi(int64_t m, int n, const double* X, int64_t ldx, uint32_t* colHi, const Ctl* ctl, int level,
                   cudaStream_t st);

template <class K>
void set_smem(K kernel) {
  cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
}

}  // namespace

size_t syrk_oz_colhi_bytes(int n) { return sizeof(uint32_t) * (size_t)((n + kM - 1) / kM * kM); }

namespace {
void launch_col_hi(int64_t m, int n, const double* X, int64_t ldx, uint32_t* colHi, const Ctl* ctl, int level,
                   cudaStream_t st) {
  cudaMemsetAsync(colHi, 0, syrk_oz_colhi_bytes(n), st);
  int ysplit = (4 * device_sms() + n - 1) / n;
  const int64_t max_y = (m + 4095) / 4096;
  if (ysplit > max_y) ysplit = (int)max_y;
  if (ysplit < 1) ysplit = 1;
  launch_dep(k_col_hi, dim3(n, ysplit), 256, 0, st, m, n, X, ldx, (m + ysplit - 1) / ysplit, colHi, ctl, level);
}
}  // namespace

void launch_oz_col_hi(int64_t m, int n, const double* X, int64_t ldx, uint32_t* colHi, const Ctl* ctl, int level,
                      cudaStream_t st) {
  launch_col_hi(m, n, X, ldx, colHi, ctl, level, st);
}

void launch_sketch_oz_reduce(int n, int s, const uint32_t* colHi, const uint32_t* idx, const SketchOzPlan& P,
                             const long long* part, double* Y, Ctl* ctl, int level, cudaStream_t st, int tf,
                             int64_t m) {
  const int64_t total = (int64_t)s * n;
  launch_dep(k_sketch_oz_reduce, (unsigned)((total + 255) / 256), 256, 0, st, n, s, colHi, idx, P, part, Y, ctl, level, tf, m);
}

SyrkOzPlan syrk_oz_plan(int64_t m, int n, int64_t rows_per_slab) {
  SyrkOzPlan P{};
  const int nI = (n + kM - 1) / kM, nJ = (n + kN - 1) / kN;
  for (int I = 0; I < 4; ++I)
    for (int J = 0; J < 8; ++J) P.tile_of[I][J] = -1;
  for (int I = 0; I < nI; ++I)
    for (int J = 0; J < nJ; ++J)
      if (kN * J + kN - 1 >= kM * I) {
        P.ti[P.ntiles] = (int8_t)I;
        P.tj[P.ntiles] = (int8_t)J;
        P.tile_of[I][J] = (int8_t)P.ntiles;
        ++P.ntiles;
      }
  if (rows_per_slab > 0) {   // a given slab height (32-row multiple, at most 2^20 rows: the 64-bit halves stay exact)
    int64_t rps = (rows_per_slab + kK - 1) / kK * kK;
    if (rps > (int64_t(1) << 20)) rps = int64_t(1) << 20;
    P.rows_per_slab = rps;
    P.slabs = (int)((m + rps - 1) / rps);
    if (P.slabs < 1) P.slabs = 1;
  } else {
    P.slabs = choose_slabs(m, P.ntiles, &P.rows_per_slab);
  }
  return P;
}

size_t syrk_oz_part_bytes(const SyrkOzPlan& P) { return sizeof(long long) * kPartElems * (size_t)P.ntiles * P.slabs; }

void launch_syrk_oz(int64_t m, int n, const double* W, int64_t ldw, const SyrkOzPlan& P, uint32_t* colHi,
                    long long* part, double* out, Ctl* ctl, int level, cudaStream_t st, bool colhi_ready) {
  if (!colhi_ready) launch_col_hi(m, n, W, ldw, colHi, ctl, level, st);
  set_smem(k_syrk_oz);
  const int nitems = P.ntiles * P.slabs;
  launch_dep(k_syrk_oz, nitems < device_sms() ? nitems : device_sms(), kOzThreads, kSmem, st, m, n, W, ldw, colHi, P, part, ctl,
                                                                               level);
  const int64_t nn = (int64_t)n * n;
  launch_dep(k_syrk_oz_reduce, (unsigned)((nn + 255) / 256), 256, 0, st, n, colHi, P, part, out, ctl, level);
}


size_t fw_digit_bytes(int n) { return fw_block_offset((n + kN - 1) / kN, 0); }

void launch_finalize_wide(int64_t m, int n, double* Q, int64_t ldq, const double* XT, int* colE, unsigned char* Xs,
                          Ctl* ctl, int level, cudaStream_t st, uint32_t* colHiOut) {
  const int nhi = (int)(syrk_oz_colhi_bytes(n) / sizeof(uint32_t)), npad = (n + 31) / 32 * 32;
  launch_dep(k_fw_prep, (n + kN - 1) / kN * kN, 128, 0, st, n, npad, XT, colE, Xs, colHiOut, nhi, ctl, level);
  set_smem(k_fw_product);
  const int64_t nblocks = (m + kM - 1) / kM;
  launch_dep(k_fw_product, (unsigned)std::min<int64_t>(nblocks, device_sms()), kOzThreads, kSmem, st, m, n, Q, ldq, colE, Xs,
             colHiOut, ctl, level);
}

SketchOzPlan sketch_oz_plan(int64_t m, int n, int s) {
  SketchOzPlan P{};
  P.mblocks = (n + kM - 1) / kM;
  P.ntiles = (s + kN - 1) / kN;
  P.slabs = choose_slabs(m, P.mblocks * P.ntiles, &P.rows_per_slab);
  return P;
}

size_t sketch_oz_part_bytes(const SketchOzPlan& P) {
  return sizeof(long long) * kPartElems * (size_t)P.mblocks * P.ntiles * P.slabs;
}

void launch_sketch_oz(int64_t m, int n, int s, const double* A, int64_t lda, const uint32_t* idx, const double* tab,
                      uint64_t seed, const SketchOzPlan& P, uint32_t* colHi, long long* part, double* Y, Ctl* ctl,
                      int level, cudaStream_t st, int tf) {
  launch_col_hi(m, n, A, lda, colHi, ctl, level, st);
  set_smem(k_sketch_oz);
  const int nitems = P.mblocks * P.ntiles * P.slabs;
  launch_dep(k_sketch_oz, nitems < device_sms() ? nitems : device_sms(), kOzThreads, kSmem, st, m, n, s, A, lda, colHi, idx, tab,
                                                                                 seed_key(seed), P, part, ctl, level, tf);
  launch_sketch_oz_reduce(n, s, colHi, idx, P, part, Y, ctl, level, st, tf, m);
}

// ---- grouped launches -------------------------------------------------------
namespace {
unsigned grid_oz(int nitems, int per_sm) {
  const int cap = device_sms() * per_sm;
  return (unsigned)(nitems < cap ? nitems : cap);
}
}  // namespace

void prepare_g_oz_kernels() {
  cudaFuncSetAttribute(kg_oz_sketch, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
  cudaFuncSetAttribute(kg_oz_syrk, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
  cudaFuncSetAttribute(kg_fw_product, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
}

void launch_g_fw_prep(const Group& g, int level, cudaStream_t st) {
  if (g.nitems) { ::mrcqr::note_launch(); kg_fw_prep<<<grid_oz(g.nitems, 16), 128, 0, st>>>(g, level); }
}
void launch_g_fw_product(const Group& g, int level, cudaStream_t st) {
  if (g.nitems) { ::mrcqr::note_launch(); kg_fw_product<<<grid_oz(g.nitems, 1), kOzThreads, kSmem, st>>>(g, level); }
}
void launch_g_oz_colhi(const Group& g, int level, cudaStream_t st) {
  if (g.nitems) { ::mrcqr::note_launch(); kg_oz_colhi<<<grid_oz(g.nitems, 16), 256, 0, st>>>(g, level); }
}
void launch_g_oz_sketch(const Group& g, int level, cudaStream_t st) {
  if (g.nitems) { ::mrcqr::note_launch(); kg_oz_sketch<<<grid_oz(g.nitems, 1), kOzThreads, kSmem, st>>>(g, level); }
}
void launch_g_oz_sketch_reduce(const Group& g, int level, cudaStream_t st) {
  if (g.nitems) { ::mrcqr::note_launch(); kg_oz_sketch_reduce<<<grid_oz(g.nitems, 16), 256, 0, st>>>(g, level); }
}
void launch_g_oz_syrk(const Group& g, bool check, int level, cudaStream_t st) {
  (void)check;   // the item's problem record names W or Q (the Q buffer holds W before the finalize)
  if (g.nitems) { ::mrcqr::note_launch(); kg_oz_syrk<<<grid_oz(g.nitems, 1), kOzThreads, kSmem, st>>>(g, level); }
}
void launch_g_oz_syrk_reduce(const Group& g, bool check, int level, cudaStream_t st) {
  if (g.nitems) { ::mrcqr::note_launch(); kg_oz_syrk_reduce<<<grid_oz(g.nitems, 16), 256, 0, st>>>(g, check ? 1 : 0, level); }
}

}  // namespace mrcqr
