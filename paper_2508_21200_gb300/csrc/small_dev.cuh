// Device parts shared by the one-CTA kernels that factor an r x r matrix.
#pragma once
#include "common.cuh"

namespace lrei {

// 1 / x and 1 / sqrt(x) for normal x > 0 by Newton's method from an FP32 value of the mantissa (the exponent is taken
// off and put back), to about an ulp: chains of 4 and 6 FP64 instructions, where the division takes 7 and a square
// root and a division 18 (445 and 1135 cycles measured).
__device__ __forceinline__ double mantissa_of(double x, int *e) {   // x = m 2^e, 1 <= m < 2
  const int hi = __double2hiint(x);
  *e = ((hi >> 20) & 0x7ff) - 1023;
  return __hiloint2double((hi & 0x800fffff) | 0x3ff00000, __double2loint(x));
}
__device__ __forceinline__ double times_pow2(double x, int e) { return __hiloint2double(__double2hiint(x) + (e << 20), __double2loint(x)); }
__device__ __forceinline__ double newton_recip(double x) {
  int e;
  const double m = mantissa_of(x, &e);
  double y = (double)(1.f / (float)m);
  y = fma(y, fma(-m, y, 1.0), y);
  y = fma(y, fma(-m, y, 1.0), y);
  return times_pow2(y, -e);
}
__device__ __forceinline__ double newton_rsqrt(double x) {
  int e;
  double m = mantissa_of(x, &e);
  if (e & 1) m = times_pow2(m, 1);   // x = m 4^(e >> 1), 1 <= m < 4
  double y = (double)rsqrtf((float)m);
  y = fma(0.5 * y, fma(-m, y * y, 1.0), y);
  y = fma(0.5 * y, fma(-m, y * y, 1.0), y);
  return times_pow2(y, -(e >> 1));
}

// Gaussian elimination of [A | I] by the whole CTA (A Hermitian, its lower triangle in Ls, the identity in X, k x k
// column-major, k <= 64): step j takes the multiple A_ij / A_jj of row j off every row i > j: entry (i, c), c <= i, of A
// where c > j and of X where c <= j.  Leaves in column j of Ls the pivot's column and in X the rows of L^{-1} before their
// scaling by A_ii^{-1/2}.  A pivot at most tolref[j], or not finite, makes column j dead: its step is left out.
// A step is a chain of FP64 instructions of 64 cycles each: one thread per real component of an entry (products, then
// one multiply-add by the pivot's reciprocal), and the thread that finishes the next pivot takes its reciprocal
// before the barrier.  (One thread per entry with a division each: 2200 cycles a step.)  inv, dead: k each.
constexpr int ELIM_OWN = 3;
__device__ __forceinline__ int tri_entry(int e) {   // row i has the entries i (i + 1) / 2 + c
  int i = (int)((sqrtf(8.f * (float)e + 1.f) - 1.f) * 0.5f);
  while ((i + 1) * (i + 2) / 2 <= e) ++i;
  while (i * (i + 1) / 2 > e) --i;
  return i << 16 | (e - i * (i + 1) / 2);
}
__device__ __forceinline__ void eliminate(zd *Ls, zd *X, int k, const double *tolref, double *inv, int *dead) {
  const int nt = blockDim.x, slots = k * (k + 1);
  int ic[ELIM_OWN];
#pragma unroll
  for (int x = 0; x < ELIM_OWN; ++x) ic[x] = tri_entry((int)(threadIdx.x + x * nt) >> 1);   // rows >= k: none
  auto pivot = [&](int j, double piv) {
    const bool ok = piv > tolref[j] && ((__double2hiint(piv) >> 20) & 0x7ff) - 1u < 0x7feu;
    dead[j] = !ok;
    inv[j] = ok ? newton_recip(piv) : 0.0;
  };
  if (threadIdx.x == 0) pivot(0, Ls[0].re);
  __syncthreads();
  for (int j = 0; j < k; ++j) {
    const double iv = inv[j];
    const bool live = !dead[j];
    auto entry = [&](int v, int cm) {
      const int i = v >> 16, c = v & 0xffff;
      if (i <= j || i >= k) return;
      const bool isA = c > j;
      double *dst = reinterpret_cast<double *>((isA ? Ls : X) + c * k + i) + cm;
      double x = *dst;
      if (live) {
        const zd f = isA ? conj(Ls[j * k + c]) : X[c * k + j], l = Ls[j * k + i];
        x = fma(-iv, cm ? fma(l.re, f.im, l.im * f.re) : fma(l.re, f.re, -l.im * f.im), x);
        *dst = x;
      }
      if (i == j + 1 && c == j + 1 && cm == 0) pivot(j + 1, x);
    };
#pragma unroll
    for (int x = 0; x < ELIM_OWN; ++x) entry(ic[x], (threadIdx.x + x * nt) & 1);
    for (int e = threadIdx.x + ELIM_OWN * nt; e < slots; e += nt) entry(tri_entry(e >> 1), e & 1);
    __syncthreads();
  }
}
// Threads for it: one per slot, up to 512.
inline int eliminate_threads(int k) { return k * (k + 1) >= 512 ? 512 : (k * (k + 1) + 31) / 32 * 32; }

// X = L^{-1} for A = L L^H (k x k, leading dimension lda, positive definite: a pivot counts as at least 1e-300, k <= MAX_R), by
// the whole CTA.  Ls: work, k x k.  The columns are scaled by powers of two to a diagonal in [1, 4): the products of two
// entries that the elimination forms stay in range for every A that does (exactly the same X).
__device__ __forceinline__ void chol_inv_cta(const zd *A, int lda, int k, zd *Ls, zd *X) {
  __shared__ double inv[MAX_R], tolref[MAX_R], scale[MAX_R];
  __shared__ int dead[MAX_R];
  __syncthreads();
  for (int i = threadIdx.x; i < k; i += blockDim.x) {
    const int e = ((__double2hiint(A[(size_t)i * lda + i].re) >> 20) & 0x7ff) - 1023;      // a negative, zero or non-finite entry as it is
    const bool ok = A[(size_t)i * lda + i].re > 0.0 && e < 1024;
    scale[i] = __hiloint2double((1023 - (ok ? e >> 1 : 0)) << 20, 0);
    tolref[i] = 1e-300 * scale[i] * scale[i];
  }
  __syncthreads();
  for (int e = threadIdx.x; e < k * k; e += blockDim.x) {
    const zd a = A[(size_t)(e / k) * lda + e % k];
    const double si = scale[e % k], sj = scale[e / k];
    Ls[e] = mk<double>(a.re * si * sj, a.im * si * sj);
    X[e] = mk<double>(e % k == e / k ? 1.0 : 0.0, 0);
  }
  __syncthreads();
  eliminate(Ls, X, k, tolref, inv, dead);
  for (int i = threadIdx.x; i < k; i += blockDim.x) inv[i] = dead[i] ? 1e150 / scale[i] : newton_rsqrt(Ls[i * k + i].re);
  __syncthreads();
  for (int e = threadIdx.x; e < k * k; e += blockDim.x) X[e] = inv[e % k] * (scale[e / k] * X[e]);
  __syncthreads();
}

// X = L^{-1} of a lower triangular k x k matrix, by the whole CTA.
__device__ __forceinline__ void tri_inv_cta(const zd *L, int k, zd *X) {
  for (int e = threadIdx.x; e < k * k; e += blockDim.x) X[e] = mk<double>(e % k == e / k ? 1.0 : 0.0, 0);
  __syncthreads();
  for (int j = 0; j < k; ++j) {   // rows below j, then row j itself by its pivot
    const int nrem = k - j - 1;
    const double inv = 1.0 / L[j * k + j].re;
    for (int e = threadIdx.x; e < nrem * (j + 1); e += blockDim.x) {
      const int i = j + 1 + e % nrem, c = e / nrem;
      const zd l = L[j * k + i];
      X[c * k + i] = X[c * k + i] - mk<double>(l.re * inv, l.im * inv) * X[c * k + j];
    }
    __syncthreads();
    for (int c = threadIdx.x; c <= j; c += blockDim.x) X[c * k + j] = inv * X[c * k + j];
  }
  __syncthreads();
}

// The sum of v over the CTA (at most 32 warps), in every thread of the first warp.  red: 32 doubles.
__device__ __forceinline__ double cta_sum(double v, double *red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  v = (threadIdx.x < blockDim.x / 32) ? red[threadIdx.x] : 0.0;
  if (threadIdx.x < 32)
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

}  // namespace lrei
