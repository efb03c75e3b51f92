// SketchQR (Algorithm 2 step 5, Sec. II-A): thin Householder QR of the s x n
// sketch Y, in FP32 for the FP16/BF16/FP32 sketches (the paper promotes the
// half-precision sketch to single for the QR) and in FP64 for the FP64
// sketch; R_s is normalised to a positive diagonal (rows flipped) and
// promoted to FP64 (Algorithm 2 step 6).
//
// Sketches of up to 1024 rows take the blocked form (panel kernel + trailing
// updates, below); larger ones, and the batched path, one CTA of 1024 threads
// that walks the columns with the working copy of Y in global memory
// (L2-resident).  Output: R_s
// column-major (n x n), its transpose padded to a row stride npad (for the
// TRSM's uniform row loads, zeros in the padding) and 1/diag(R_s).
#include <type_traits>
#include "kernels.h"

namespace mrcqr {

constexpr int kSqrThreads = 1024;
constexpr int kPadCols = 32;

__host__ __device__ inline int padded(int n) { return (n + kPadCols - 1) / kPadCols * kPadCols; }

template <typename T>
__device__ __forceinline__ void sketch_qr_block(int n, int s, const double* __restrict__ Y, T* __restrict__ W,
                                                double* __restrict__ Rs, double* __restrict__ RsT,
                                                double* __restrict__ rinv) {
  __shared__ T red[33];
  __shared__ T diag[512];
  __shared__ T sh_inv, sh_tau;   // per-column scalars, formed once (FP64 division and sqrt are long sequences)
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
  const int64_t total = (int64_t)s * n;
  for (int64_t e = tid; e < total; e += blockDim.x) W[e] = (T)Y[e];
  __syncthreads();
  for (int j = 0; j < n; ++j) {
    T* col = W + (int64_t)j * s;
    // 2-norm of col[j..s) with scaling by the max (no over/underflow)
    T amax = T(0);
    for (int i = j + tid; i < s; i += blockDim.x) amax = max(amax, (T)fabs(col[i]));
    amax = warp_max(amax);
    __syncthreads();
    if (lane == 0) red[warp] = amax;
    __syncthreads();
    if (warp == 0) {
      T t = lane < nwarps ? red[lane] : T(0);
      t = warp_max(t);
      if (lane == 0) {
        red[32] = t;
        sh_inv = t > T(0) ? T(1) / t : T(0);
      }
    }
    __syncthreads();
    amax = red[32];
    T part = T(0);
    if (amax > T(0)) {
      const T inv = sh_inv;
      for (int i = j + tid; i < s; i += blockDim.x) {
        const T v = col[i] * inv;
        part = fma(v, v, part);
      }
    }
    const T ss = block_sum(part, red);
    if (tid == 0) {
      const T nrm = amax * sqrt(ss);
      const T x0 = col[j];
      const T alpha = (x0 >= T(0)) ? -nrm : nrm;
      // ||v||^2 = 2 nrm (nrm + |x0|), so tau = 2/||v||^2 = 1/(nrm (nrm + |x0|))
      sh_tau = (nrm > T(0)) ? T(1) / (nrm * (nrm + (T)fabs(x0))) : T(0);
      col[j] = x0 - alpha;
      diag[j] = alpha;
    }
    __syncthreads();
    const T tau = sh_tau;
    for (int c = j + 1 + warp; c < n; c += nwarps) {
      T* cc = W + (int64_t)c * s;
      T d = T(0);
      for (int i = j + lane; i < s; i += 32) d = fma(col[i], cc[i], d);
      d = warp_sum(d);
      const T f = tau * d;
      for (int i = j + lane; i < s; i += 32) cc[i] = fma(-f, col[i], cc[i]);
    }
    __syncthreads();
  }
  const int npad = padded(n);
  for (int e = tid; e < npad * n; e += blockDim.x) {
    // e indexes RsT row-major: row r (< n), column c (< npad)
    const int r = e / npad, c = e % npad;
    const double sg = diag[r] < T(0) ? -1.0 : 1.0;
    double v = 0.0;
    if (c < n) {
      if (r < c) v = (double)W[(int64_t)c * s + r] * sg;
      else if (r == c) v = fabs((double)diag[r]);
    }
    RsT[(int64_t)r * npad + c] = v;
    if (c < n) Rs[(int64_t)c * n + r] = v;
  }
  for (int r = tid; r < npad; r += blockDim.x) rinv[r] = r < n ? 1.0 / fabs((double)diag[r]) : 0.0;
  __syncthreads();
}

template <typename T>
__global__ void __launch_bounds__(kSqrThreads) k_sketch_qr(int n, int s, const double* __restrict__ Y,
                                                           T* __restrict__ W, double* __restrict__ Rs,
                                                           double* __restrict__ RsT, double* __restrict__ rinv,
                                                           Ctl* ctl, int level) {
  if (level_inactive(ctl, level)) return;
  if (ctl->lvl_status != 0) return;
  sketch_qr_block<T>(n, s, Y, W, Rs, RsT, rinv);
}


// ---------------------------------------------------------------------------
// Blocked form for s <= 1024 (the single-CTA kernel above keeps the larger
// sketches): panels of kQB columns are factored by one CTA of four warps with
// the panel in registers, and the columns right of a panel are updated by one
// CTA each, so the O(s n^2) reflector applications are spread over the GPU
// (FP64 issues at 1/64 of the FP32 rate here; one warp's FP64 instruction
// holds a quarter of an SM for 64 cycles, so four warps with many independent
// chains each are what one SM can use).  Narrow panels keep the O(s kQB^2)
// work per panel that only one SM does small.
// Measured (before: 16-column panels by one warp per column, updates by one
// warp per column): the figures stand at launch_sketch_qr.
// The working copy holds LAPACK's geqrf layout: beta_j = +-||x|| on the
// diagonal, the reflector v (v_j = 1 implicit) below it; tau = 2 / ||v||^2
// waits in the output array rinv, which k_sqr_out writes last.
constexpr int kQB = 8;           // panel width
constexpr int kQMaxS = 1024;     // rows handled by the blocked form
constexpr int kQThreads = 128;

__global__ void k_sqr_copy(int64_t total, const double* __restrict__ Y, void* __restrict__ Wk, int fp64,
                           const Ctl* ctl, int level) {
  if (level_inactive(ctl, level) || ctl->lvl_status != 0) return;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    if (fp64) static_cast<double*>(Wk)[e] = Y[e];
    else static_cast<float*>(Wk)[e] = (float)Y[e];
  }
}

// Warp-wide sum and max.
template <typename T>
__device__ __forceinline__ T wsum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
template <typename T>
__device__ __forceinline__ T wmax(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// Sum of v over the block (every thread; four warps, red: 4 entries, free again after
// the next barrier).
template <typename T>
__device__ __forceinline__ T qsum(T v, T* red) {
  v = wsum(v);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  return (red[0] + red[1]) + (red[2] + red[3]);
}

// Reflector of a column with head x0 and tail sum of squares `tail`, both
// times inv^2 resp. inv where the column was scaled by inv = 1 / amax:
// beta = -sign(x0) ||x||, scale = 1 / (x0 - beta), tau = 2 / ||v||^2 for
// v = (1, scale * tail entries).
template <typename T>
__device__ __forceinline__ void house_scalars(T x0, T tail, T amax, T inv, T& beta, T& scale, T& tau) {
  const T y0 = x0 * inv;
  const T nrm = amax * sqrt(fma(y0, y0, tail));
  beta = x0 >= T(0) ? -nrm : nrm;
  scale = T(1) / (x0 - beta);   // |x0 - beta| = |x0| + nrm: no cancellation
  const T r = amax * scale;
  tau = T(2) / fma(tail * r, r, T(1));
}

// Panel [c0, c1) of the s x n working copy (column-major, ld s), rows c0 .. s-1:
// thread t holds rows t + 128 r of every panel column in registers.  FP32
// scales each norm by the column maximum so it neither overflows nor
// underflows; FP64 does so only when the plain sum of squares leaves
// [1e-250, 1e250].  The reflector's scalars are formed by one lane per warp
// (the four warps sit on four FP64 pipes).
template <typename T, int kR>
__global__ void __launch_bounds__(kQThreads) k_sqr_panel(int s, int c0, int c1, T* __restrict__ Wk,
                                                         double* __restrict__ taus, const Ctl* ctl, int level) {
  if (level_inactive(ctl, level) || ctl->lvl_status != 0) return;
  __shared__ T red[3][4], head[kQB], dots[2][4][kQB];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rows = s - c0, b = c1 - c0;
  T x[kQB][kR];
#pragma unroll
  for (int c = 0; c < kQB; ++c)
#pragma unroll
    for (int r = 0; r < kR; ++r) {
      const int i = tid + kQThreads * r;
      x[c][r] = c < b && i < rows ? Wk[(int64_t)(c0 + c) * s + c0 + i] : T(0);
    }
#pragma unroll
  for (int jj = 0; jj < kQB; ++jj) {
    if (jj >= b) break;
    if (tid == jj) head[jj] = x[jj][0];
    // tail sum of squares, unscaled (FP64) or scaled by the column maximum
    T amax = T(1), inv = T(1), tail = T(0);
    bool zero = false, scaled = sizeof(T) == 4;
    if (sizeof(T) == 8) {
      T part = T(0);
#pragma unroll
      for (int r = 0; r < kR; ++r)
        if (r > 0 || tid > jj) part = fma(x[jj][r], x[jj][r], part);
      tail = qsum(part, red[0]);
      const T ss = fma(head[jj], head[jj], tail);
      scaled = !(ss > T(1e-250) && ss < T(1e250));
      zero = scaled && !(ss > T(0));   // zero column (or NaN: left as it is)
    }
    if (scaled && !zero) {
      T mx = T(0);
#pragma unroll
      for (int r = 0; r < kR; ++r)
        if (r > 0 || tid >= jj) mx = max(mx, (T)fabs(x[jj][r]));
      mx = wmax(mx);
      if (lane == 0) red[1][warp] = mx;
      __syncthreads();
      amax = max(max(red[1][0], red[1][1]), max(red[1][2], red[1][3]));
      zero = !(amax > T(0));
      inv = zero ? T(0) : T(1) / amax;
      T part = T(0);
#pragma unroll
      for (int r = 0; r < kR; ++r)
        if (r > 0 || tid > jj) {
          const T a = x[jj][r] * inv;
          part = fma(a, a, part);
        }
      tail = qsum(part, red[2]);
    }
    T beta = T(0), scale = T(1), tau = T(0);
    if (!zero) {
      if (lane == 0) house_scalars(head[jj], tail, amax, inv, beta, scale, tau);
      beta = __shfl_sync(0xffffffffu, beta, 0);
      scale = __shfl_sync(0xffffffffu, scale, 0);
      tau = __shfl_sync(0xffffffffu, tau, 0);
    } else {
      beta = head[jj];
    }
    if (tid == 0) taus[c0 + jj] = (double)tau;
    // v, its products with the columns to the right, their update
    T d[kQB];
#pragma unroll
    for (int c = 0; c < kQB; ++c) d[c] = T(0);
#pragma unroll
    for (int r = 0; r < kR; ++r) {
      T v;
      if (r > 0 || tid > jj) {
        x[jj][r] *= scale;
        v = x[jj][r];
      } else {
        v = tid == jj ? T(1) : T(0);
      }
#pragma unroll
      for (int c = jj + 1; c < kQB; ++c) d[c] = fma(v, x[c][r], d[c]);
    }
#pragma unroll
    for (int c = jj + 1; c < kQB; ++c) {
      const T w = wsum(d[c]);
      if (lane == 0) dots[jj & 1][warp][c] = w;
    }
    __syncthreads();
#pragma unroll
    for (int c = jj + 1; c < kQB; ++c) {
      const T* q = &dots[jj & 1][0][c];
      const T f = tau * ((q[0] + q[kQB]) + (q[2 * kQB] + q[3 * kQB]));
#pragma unroll
      for (int r = 0; r < kR; ++r) {
        const T v = r > 0 || tid > jj ? x[jj][r] : tid == jj ? T(1) : T(0);
        x[c][r] = fma(-f, v, x[c][r]);
      }
    }
    if (tid == jj) x[jj][0] = beta;
  }
#pragma unroll
  for (int c = 0; c < kQB; ++c)
#pragma unroll
    for (int r = 0; r < kR; ++r) {
      const int i = tid + kQThreads * r;
      if (c < b && i < rows) Wk[(int64_t)(c0 + c) * s + c0 + i] = x[c][r];
    }
}

// Column c1 + blockIdx.x: the panel's reflectors in order, rows c0 + t + 128 r
// in thread t.
template <typename T, int kR>
__global__ void __launch_bounds__(kQThreads) k_sqr_update(int s, int c0, int c1, T* __restrict__ Wk,
                                                          const double* __restrict__ taus, const Ctl* ctl, int level) {
  if (level_inactive(ctl, level) || ctl->lvl_status != 0) return;
  __shared__ T red[2][4];
  const int tid = threadIdx.x, rows = s - c0;
  T* y = Wk + (int64_t)(c1 + blockIdx.x) * s + c0;
  T x[kR];
#pragma unroll
  for (int r = 0; r < kR; ++r) x[r] = tid + kQThreads * r < rows ? y[tid + kQThreads * r] : T(0);
#pragma unroll 1
  for (int j = c0; j < c1; ++j) {
    const T* v = Wk + (int64_t)j * s + c0;
    const int jj = j - c0;
    T vr[kR], d = T(0);
#pragma unroll
    for (int r = 0; r < kR; ++r) {
      const int i = tid + kQThreads * r;
      vr[r] = i > jj && i < rows ? v[i] : i == jj ? T(1) : T(0);
    }
#pragma unroll
    for (int r = 0; r < kR; ++r) d = fma(vr[r], x[r], d);
    const T f = (T)taus[j] * qsum(d, red[jj & 1]);
#pragma unroll
    for (int r = 0; r < kR; ++r) x[r] = fma(-f, vr[r], x[r]);
  }
#pragma unroll
  for (int r = 0; r < kR; ++r)
    if (tid + kQThreads * r < rows) y[tid + kQThreads * r] = x[r];
}

// ---------------------------------------------------------------------------
// One CTA for the small sketches, the matrix in shared memory (Y in, R_s out: one
// launch, where the blocked form has 2 n / 8 + 1, each of which costs a few
// microseconds even at a level that is not taken).  Warp w owns columns w, w +
// nwarps, ..: at step j every warp applies reflector j to its columns right of
// j, the owner of column j + 1 to that one first and then forms reflector
// j + 1 while the others go on; one barrier per step.
// Householder reflector of x[jj..rows) by one warp (the column's owner):
// beta = -sign(x0) ||x||, v = (1, x[jj+1..] / (x0 - beta)), tau = 2 / ||v||^2.
// x[jj] <- beta, x[jj+1..] <- v[1..]; returns tau (0 for a zero column).
// FP32 scales the norm by the column maximum so it neither overflows nor
// underflows; FP64 does so only when the plain sum of squares leaves
// [1e-250, 1e250] (each FP64 operation is a long-latency step on this GPU).
template <typename T>
__device__ __forceinline__ T house_warp(T* x, int jj, int rows, int lane) {
  if constexpr (sizeof(T) == 8) {   // FP64: unscaled sums of squares unless they leave the normal range
    T t0 = T(0), t1 = T(0);
    int i = jj + 1 + lane;
    for (; i + 32 < rows; i += 64) {
      t0 = fma(x[i], x[i], t0);
      t1 = fma(x[i + 32], x[i + 32], t1);
    }
    if (i < rows) t0 = fma(x[i], x[i], t0);
    const T tail = wsum(t0 + t1);
    const T x0 = x[jj];
    const T ss = fma(x0, x0, tail);
    if (ss > T(1e-250) && ss < T(1e250)) {
      const T nrm = sqrt(ss);
      const T beta = x0 >= T(0) ? -nrm : nrm;
      const T d = x0 - beta;
      const T scale = T(1) / d;
      const T tau = T(2) / fma(tail * scale, scale, T(1));
      __syncwarp();
      for (int k = jj + 1 + lane; k < rows; k += 32) x[k] *= scale;
      if (lane == 0) x[jj] = beta;
      __syncwarp();
      return tau;
    }
    if (!(ss > T(0))) return T(0);   // zero column (or NaN: left as it is)
  }
  T amax = T(0);
  for (int i = jj + lane; i < rows; i += 32) amax = max(amax, (T)fabs(x[i]));
  amax = wmax(amax);
  if (!(amax > T(0))) return T(0);
  const T inv = T(1) / amax;
  T t0 = T(0), t1 = T(0);
  int i = jj + 1 + lane;
  for (; i + 32 < rows; i += 64) {
    const T a = x[i] * inv, b = x[i + 32] * inv;
    t0 = fma(a, a, t0);
    t1 = fma(b, b, t1);
  }
  if (i < rows) {
    const T a = x[i] * inv;
    t0 = fma(a, a, t0);
  }
  const T tail = wsum(t0 + t1);   // sum of (x_i / amax)^2 over i > jj
  const T x0 = x[jj], y0 = x0 * inv;
  const T nrm = amax * sqrt(fma(y0, y0, tail));
  const T beta = x0 >= T(0) ? -nrm : nrm;
  const T d = x0 - beta;   // |d| = |x0| + nrm: no cancellation
  const T scale = T(1) / d;
  const T r = amax * scale;
  const T tau = T(2) / fma(tail * r, r, T(1));
  __syncwarp();
  for (int k = jj + 1 + lane; k < rows; k += 32) x[k] *= scale;
  if (lane == 0) x[jj] = beta;
  __syncwarp();
  return tau;
}

// y <- (I - tau v v^T) y over rows jj..rows-1, v = (1, x[jj+1..]), one warp.
template <typename T>
__device__ __forceinline__ void house_apply_warp(const T* x, T* y, T tau, int jj, int rows, int lane) {
  T d0 = lane == 0 ? y[jj] : T(0), d1 = T(0);
  int i = jj + 1 + lane;
  for (; i + 32 < rows; i += 64) {
    d0 = fma(x[i], y[i], d0);
    d1 = fma(x[i + 32], y[i + 32], d1);
  }
  if (i < rows) d0 = fma(x[i], y[i], d0);
  const T f = tau * wsum(d0 + d1);
  if (lane == 0) y[jj] -= f;
  for (int k = jj + 1 + lane; k < rows; k += 32) y[k] = fma(-f, x[k], y[k]);
  __syncwarp();
}

template <typename T>
__global__ void __launch_bounds__(1024) k_sqr_cta(int n, int s, const double* __restrict__ Y, double* __restrict__ Rs,
                                                  double* __restrict__ RsT, double* __restrict__ rinv, const Ctl* ctl,
                                                  int level) {
  if (level_inactive(ctl, level) || ctl->lvl_status != 0) return;
  extern __shared__ unsigned char sqr_smem[];
  T* P = reinterpret_cast<T*>(sqr_smem);   // column c at P + c s
  __shared__ T taus[2];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  for (int e = tid; e < s * n; e += blockDim.x) P[e] = (T)Y[e];
  __syncthreads();
  if (warp == 0) {
    const T t = house_warp(P, 0, s, lane);
    if (lane == 0) taus[0] = t;
  }
  __syncthreads();
  for (int j = 0; j < n - 1; ++j) {
    const T* x = P + j * s;
    const T tau = taus[j & 1];
    const int next = (j + 1) % nw;
    int c = j + 1 + (warp - next + nw) % nw;   // this warp's first column right of j
    if (warp == next) {
      T* y = P + c * s;
      house_apply_warp(x, y, tau, j, s, lane);
      const T t = house_warp(y, j + 1, s, lane);
      if (lane == 0) taus[(j + 1) & 1] = t;
      c += nw;
    }
    for (; c < n; c += nw) house_apply_warp(x, P + c * s, tau, j, s, lane);
    __syncthreads();
  }
  const int npad = padded(n);
  for (int e = tid; e < npad * n; e += blockDim.x) {
    const int r = e / npad, c = e % npad;
    const double beta = (double)P[r * s + r];
    double v = 0.0;
    if (c < n) {
      if (r < c) v = beta < 0.0 ? -(double)P[c * s + r] : (double)P[c * s + r];
      else if (r == c) v = fabs(beta);
    }
    RsT[(int64_t)r * npad + c] = v;
    if (c < n) Rs[(int64_t)c * n + r] = v;
  }
  for (int r = tid; r < npad; r += blockDim.x) rinv[r] = r < n ? 1.0 / fabs((double)P[r * s + r]) : 0.0;
}

// FP32 up to n = 64 and FP64 up to n = 32, where the sketch fits the shared memory: beyond, one SM takes longer
// than the blocked form and its launches (FP32: n = 64 141 us against 120, but 6 against 49 where the level is
// skipped; n = 100 274 against 191).
template <typename T>
bool sqr_one_cta(int n, int s) {
  return n <= (sizeof(T) == 8 ? 32 : 64) && sizeof(T) * (size_t)n * s <= 200 * 1024;
}

template <typename T>
void launch_sqr_cta(int n, int s, const double* Y, double* Rs, double* RsT, double* rinv, Ctl* ctl, int level,
                    cudaStream_t st) {
  cudaFuncSetAttribute(k_sqr_cta<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  launch_dep(k_sqr_cta<T>, 1, n <= 32 ? 512 : 1024, sizeof(T) * (size_t)n * s, st, n, s, Y, Rs, RsT, rinv, ctl, level);
}

// R_s (column-major), its padded transpose and 1/diag from the factored
// working copy, rows flipped to a positive diagonal.
template <typename T>
__global__ void k_sqr_out(int n, int s, const T* __restrict__ Wk, double* __restrict__ Rs, double* __restrict__ RsT,
                          double* __restrict__ rinv, const Ctl* ctl, int level) {
  if (level_inactive(ctl, level) || ctl->lvl_status != 0) return;
  const int npad = padded(n);
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e < (int64_t)npad * n) {
    const int r = (int)(e / npad), c = (int)(e % npad);
    const double beta = (double)Wk[(int64_t)r * s + r];
    const double sg = beta < 0.0 ? -1.0 : 1.0;
    double v = 0.0;
    if (c < n) {
      if (r < c) v = (double)Wk[(int64_t)c * s + r] * sg;
      else if (r == c) v = fabs(beta);
    }
    RsT[(int64_t)r * npad + c] = v;
    if (c < n) Rs[(int64_t)c * n + r] = v;
  }
  if (e < npad) rinv[e] = e < n ? 1.0 / fabs((double)Wk[e * s + e]) : 0.0;
}

template <typename T>
void launch_sqr_blocked(int n, int s, const double* Y, T* Wk, double* Rs, double* RsT, double* rinv, Ctl* ctl,
                        int level, cudaStream_t st) {
  const int64_t total = (int64_t)s * n;
  launch_dep(k_sqr_copy, (unsigned)((total + 255) / 256 < 1024 ? (total + 255) / 256 : 1024), 256, 0, st, total, Y, Wk, std::is_same<T, double>::value ? 1 : 0, ctl, level);
  for (int c0 = 0; c0 < n; c0 += kQB) {
    const int c1 = c0 + kQB < n ? c0 + kQB : n, rows = s - c0;
    auto panel = rows <= 128 ? k_sqr_panel<T, 1> : rows <= 256 ? k_sqr_panel<T, 2>
               : rows <= 512 ? k_sqr_panel<T, 4> : k_sqr_panel<T, 8>;
    launch_dep(panel, 1, kQThreads, 0, st, s, c0, c1, Wk, rinv, ctl, level);
    if (c1 < n) {
      auto update = rows <= 128 ? k_sqr_update<T, 1> : rows <= 256 ? k_sqr_update<T, 2>
                  : rows <= 512 ? k_sqr_update<T, 4> : k_sqr_update<T, 8>;
      launch_dep(update, (unsigned)(n - c1), kQThreads, 0, st, s, c0, c1, Wk, rinv, ctl, level);
    }
  }
  const int64_t tot = (int64_t)padded(n) * n;
  launch_dep(k_sqr_out<T>, (unsigned)((tot + 255) / 256), 256, 0, st, n, s, Wk, Rs, RsT, rinv, ctl, level);
}

size_t sqr_workspace_bytes(int n, int s) { return (size_t)n * (size_t)s * sizeof(double); }

// One launch with Y in shared memory where it fits and one CTA is faster (FP32
// up to n = 64, FP64 up to n = 32), panels of kQB columns in registers with the
// trailing columns over the chip up to s = kQMaxS, and the kernel over global
// memory beyond.  Measured (s = 2n, us, before / now): FP64 n = 512 8250 /
// 4540, 128 863 / 760; FP32 n = 256 853 / 483, 100 250 / 191, 64 147 / 141,
// 32 63 / 55; a level that is skipped costs one launch instead of up to 25
// (49 / 6 us at n = 64).
void launch_sketch_qr(int prec, int n, int s, const double* Y, void* work, double* Rs, double* RsT, double* rinv,
                      Ctl* ctl, int level, cudaStream_t st) {
  if (prec == P_FP64 ? sqr_one_cta<double>(n, s) : sqr_one_cta<float>(n, s)) {
    if (prec == P_FP64) launch_sqr_cta<double>(n, s, Y, Rs, RsT, rinv, ctl, level, st);
    else launch_sqr_cta<float>(n, s, Y, Rs, RsT, rinv, ctl, level, st);
    return;
  }
  if (s <= kQMaxS) {
    if (prec == P_FP64) launch_sqr_blocked<double>(n, s, Y, (double*)work, Rs, RsT, rinv, ctl, level, st);
    else launch_sqr_blocked<float>(n, s, Y, (float*)work, Rs, RsT, rinv, ctl, level, st);
    return;
  }
  if (prec == P_FP64)
    launch_dep(k_sketch_qr<double>, 1, kSqrThreads, 0, st, n, s, Y, (double*)work, Rs, RsT, rinv, ctl, level);
  else
    launch_dep(k_sketch_qr<float>, 1, kSqrThreads, 0, st, n, s, Y, (float*)work, Rs, RsT, rinv, ctl, level);
}

}  // namespace mrcqr

namespace mrcqr {

// R_s given by the caller (column-major n x n): its padded transpose and
// 1/diag for the substitution kernel.
__global__ void k_rs_prepare(int n, const double* __restrict__ Rs, double* __restrict__ RsT,
                             double* __restrict__ rinv) {
  const int npad = padded(n);
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e < (int64_t)n * npad) {
    const int r = (int)(e / npad), c = (int)(e % npad);
    RsT[e] = (c < n && r <= c) ? Rs[(int64_t)c * n + r] : 0.0;
  }
  if (e < npad) rinv[e] = e < n ? 1.0 / Rs[e * n + e] : 0.0;
}

void launch_rs_prepare(int n, const double* Rs, double* RsT, double* rinv, cudaStream_t st) {
  const int64_t tot = (int64_t)n * padded(n);
  { ::mrcqr::note_launch(); k_rs_prepare<<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(n, Rs, RsT, rinv); }
}

// Grouped sketch QR: one CTA per problem.
namespace {

template <typename T>
__global__ void __launch_bounds__(kSqrThreads) kg_sketch_qr(Group g, int level) {
  for (int it = blockIdx.x; it < g.nitems; it += gridDim.x) {
    const Prob& P = g.probs[g.items[it].x];
    if (P.ctl->active != level || P.ctl->lvl_status != 0) continue;
    sketch_qr_block<T>(P.n, P.s, P.y, static_cast<T*>(P.sqrw), P.rs, P.rst, P.rinv);
  }
}

}  // namespace

void launch_g_sketch_qr(const Group& g, bool fp64, int level, cudaStream_t st) {
  if (!g.nitems) return;
  const unsigned grid = (unsigned)(g.nitems < 152 * 2 ? g.nitems : 152 * 2);
  if (fp64) { ::mrcqr::note_launch(); kg_sketch_qr<double><<<grid, kSqrThreads, 0, st>>>(g, level); }
  else { ::mrcqr::note_launch(); kg_sketch_qr<float><<<grid, kSqrThreads, 0, st>>>(g, level); }
}

}  // namespace mrcqr
