// Device parts shared by the one-CTA kernels that factor an r x r matrix.
#pragma once
#include "common.cuh"

namespace lrei {

// Step j of the Gaussian elimination of [A | I] (A Hermitian, its lower triangle in Ls, the identity in X, k x k
// column-major): the multiple A_ij / A_jj (inv = 1 / A_jj) of row j off every row i > j: entry (i, c), c <= i, of A
// where c > j and of X where c <= j.  Thread t owns the entries t, t + blockDim, ... of the lower triangle by rows in
// every step, ic[] holds the first ELIM_OWN of them (i << 16 | c).  No barrier.
constexpr int ELIM_OWN = 3;
__device__ __forceinline__ int tri_entry(int e) {   // row i has the entries i (i + 1) / 2 + c
  int i = (int)((sqrtf(8.f * (float)e + 1.f) - 1.f) * 0.5f);
  while ((i + 1) * (i + 2) / 2 <= e) ++i;
  while (i * (i + 1) / 2 > e) --i;
  return i << 16 | (e - i * (i + 1) / 2);
}
__device__ __forceinline__ void elim_own(int k, int *ic) {
#pragma unroll
  for (int x = 0; x < ELIM_OWN; ++x) ic[x] = tri_entry(threadIdx.x + x * blockDim.x);   // rows >= k: none
}
__device__ __forceinline__ void elim_step(zd *Ls, zd *X, int k, int j, double inv, const int *ic) {
  auto entry = [&](int v) {
    const int i = v >> 16, c = v & 0xffff;
    if (i <= j || i >= k) return;
    zd *dst = (c > j ? Ls : X) + c * k + i;
    const zd f = c > j ? conj(Ls[j * k + c]) : X[c * k + j], l = Ls[j * k + i];
    *dst = *dst - mk<double>(l.re * inv, l.im * inv) * f;
  };
#pragma unroll
  for (int x = 0; x < ELIM_OWN; ++x) entry(ic[x]);
  for (int e = threadIdx.x + ELIM_OWN * blockDim.x; e < k * (k + 1) / 2; e += blockDim.x) entry(tri_entry(e));
}

// X = L^{-1} for A = L L^H (k x k, leading dimension lda, positive definite: a pivot counts as at least 1e-300), by the
// whole CTA.  Ls: work, k x k.
__device__ __forceinline__ void chol_inv_cta(const zd *A, int lda, int k, zd *Ls, zd *X) {
  for (int e = threadIdx.x; e < k * k; e += blockDim.x) {
    Ls[e] = A[(size_t)(e / k) * lda + e % k];
    X[e] = mk<double>(e % k == e / k ? 1.0 : 0.0, 0);
  }
  int ic[ELIM_OWN];
  elim_own(k, ic);
  __syncthreads();
  for (int j = 0; j < k; ++j) {
    elim_step(Ls, X, k, j, 1.0 / fmax(Ls[j * k + j].re, 1e-300), ic);
    __syncthreads();
  }
  // row i of X by A_ii^{-1/2}: all rows' roots in parallel, in the imaginary parts of the pivots
  for (int i = threadIdx.x; i < k; i += blockDim.x) Ls[i * k + i].im = 1.0 / sqrt(fmax(Ls[i * k + i].re, 1e-300));
  __syncthreads();
  for (int e = threadIdx.x; e < k * k; e += blockDim.x) X[e] = Ls[(e % k) * k + e % k].im * X[e];
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
