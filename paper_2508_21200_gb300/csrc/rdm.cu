// Two-spin reduced density matrices R_kl and their entanglement measures (paper Sec. 3.6: the
// partial trace of rho over every spin but k and l, measured from the low-rank factor; the
// concurrence of Wootters (1998) and the negativity of Vidal and Werner (2002) from the 4 x 4).
//
// With rho = Vb Lambda Vb^* (Vb the orthonormalised factor), the rows of the N x r factor fall
// into N/4 groups of four that differ only in the bits of sites k and l; group g with the two
// bits set to s = (s_k, s_l) is row b_s(g), and
//     R[s, s'] = sum_g sum_c lambda_c Vb[b_s(g), c] conj(Vb[b_s'(g), c]),
// the index of R being 2 s_k + s_l (site k the first factor, 0 = spin up).  One pass per pair
// over the factor computes the ten entries s <= s'; each thread owns one column c of a group
// (threads of consecutive columns read consecutive words of a row) and keeps running sums,
// compensated (TwoSum) in the complex64 path, combined per CTA and written as FP64 partials.
// One CTA per pair then sums the partials in a fixed order, applies the Werner weight p (R -> p I/4 + (1 - p) R) and
// evaluates the two measures by 4 x 4 Jacobi, a warp each.
#include "common.cuh"

namespace lrei {

namespace {

__device__ __forceinline__ void two_sum(float &hi, float &lo, float b) {
  const float s = hi + b, bp = s - hi;
  lo += (hi - (s - bp)) + (b - bp);
  hi = s;
}

template <typename T> struct RAcc;
template <> struct RAcc<double> {
  double v[16];
  __device__ void zero() {
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = 0.0;
  }
  __device__ void add(int i, double a, double b, double c, double d) { v[i] = fma(a, b, fma(c, d, v[i])); }   // += a b + c d
  __device__ double get(int i) const { return v[i]; }
};
template <> struct RAcc<float> {
  float v[16], e[16];
  __device__ void zero() {
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = e[i] = 0.f;
  }
  __device__ void add(int i, float a, float b, float c, float d) { two_sum(v[i], e[i], fmaf(a, b, c * d)); }
  __device__ double get(int i) const { return (double)v[i] + (double)e[i]; }
};

__device__ __forceinline__ uint32_t insert_zero(uint32_t x, int pos) {
  const uint32_t low = x & ((1u << pos) - 1u);
  return low | ((x >> pos) << (pos + 1));
}

}  // namespace

// pairs: 2 ints per pair, the bit positions of sites k and l in the basis index.
// partial: [npairs][gridDim.x][16] doubles: the diagonal entries, then (s, s') with s < s' in row order, re/im.
// FP64 multiply-adds bound it (n = 16, r = 7, 120 pairs: 40 per group and column, 1.85 ms with 80).
template <typename T>
__global__ void __launch_bounds__(256) rdm_kernel(const cx<T> *__restrict__ V, long long N, int r,
                                                  const double *__restrict__ lam, const int *__restrict__ pairs,
                                                  double *__restrict__ partial) {
  __shared__ double red[8][16];
  const int p = blockIdx.y;
  const int bk = pairs[2 * p], bl = pairs[2 * p + 1];
  const int lo = bk < bl ? bk : bl, hi = bk < bl ? bl : bk;
  const int tid = threadIdx.x;
  const int gpb = 256 / r;                              // groups per CTA pass (one thread per column)
  const int c = tid % r, gl = tid / r;
  const long long ngroups = N >> 2;
  const T lc = (T)lam[c < r ? c : 0];
  RAcc<T> acc;
  acc.zero();
  if (gl < gpb) {
    for (long long g = (long long)blockIdx.x * gpb + gl; g < ngroups; g += (long long)gridDim.x * gpb) {
      const uint32_t b0 = insert_zero(insert_zero((uint32_t)g, lo), hi);
      cx<T> v[4];
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        const uint32_t b = b0 | ((uint32_t)(s >> 1) << bk) | ((uint32_t)(s & 1) << bl);
        v[s] = V[(size_t)b * r + c];
      }
      int e = 4;
#pragma unroll
      for (int s = 0; s < 4; ++s) {   // lambda_c v_s conj(v_t)
        const cx<T> w = lc * v[s];
        acc.add(s, w.re, v[s].re, w.im, v[s].im);
#pragma unroll
        for (int t = s + 1; t < 4; ++t) {
          acc.add(e++, w.re, v[t].re, w.im, v[t].im);
          acc.add(e++, w.im, v[t].re, -w.re, v[t].im);
        }
      }
    }
  }
  // combine the CTA's threads: warp shuffles, then the warps in a fixed order
  const int lane = tid & 31, wp = tid >> 5;
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    double x = acc.get(i);
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if (lane == 0) red[wp][i] = x;
  }
  __syncthreads();
  if (tid < 16) {
    double s = 0.0;
    for (int w = 0; w < 8; ++w) s += red[w][tid];
    partial[((size_t)p * gridDim.x + blockIdx.x) * 16 + tid] = s;
  }
}

namespace {
// Eigenvalues (w, in the order of the diagonal) and eigenvectors (columns of U, 4 x 4 column-major) of the Hermitian 4 x 4
// matrix A (column-major) by cyclic complex Jacobi, by one warp: lane 8 i + 2 j + m holds component m of entry
// (i, j), and a round applies the two rotations of the pairs x, x ^ mask.  An FP64 instruction takes 64 cycles in a
// chain, a division or square root 7 to 11 of these, so the angle is taken in FP32 (which annihilates to 1e-7 a
// round) and made unitary in FP64 by two Newton steps for c = sqrt(1 - |s|^2).  A is scaled by a power of two to entries
// below 2, so that FP32 has the range.  (One thread per matrix with FP64 angles: 5.0 ms for the 120 pairs of n = 16.)
__device__ __forceinline__ double flip(double x, bool c) { return c ? -x : x; }
__device__ void herm4_eig(const zd *A, zd *U, double *w) {
  const unsigned all = 0xffffffffu;
  const int lane = threadIdx.x & 31, m = lane & 1, j = (lane >> 1) & 3, i = lane >> 3;
  double a = reinterpret_cast<const double *>(A)[2 * (4 * j + i) + m];
  double u = (i == j && m == 0) ? 1.0 : 0.0;
  const unsigned emax = __reduce_max_sync(all, ((unsigned)__double2hiint(a) >> 20) & 0x7ffu);
  const bool finite = emax < 0x7ff;
  const int es = emax == 0 || !finite ? 1023 : max(1, 2046 - (int)emax);
  a *= __hiloint2double(es << 20, 0);
  for (int sweep = 0; finite && sweep < 30; ++sweep) {
    // off-diagonal Frobenius norm against 1e-16 of the whole (a bound on the largest entry that implies it is below the
    // entries' rounding: 4096 multiples of the identity took 2.7 ms a call, and 1.2 when they were exact)
    const float v = (float)a * (float)a;
    float off = i != j ? v : 0.f, tot = v;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      off += __shfl_xor_sync(all, off, o);
      tot += __shfl_xor_sync(all, tot, o);
    }
    if (off <= 1e-32f * tot) break;
#pragma unroll
    for (int mask = 1; mask < 4; ++mask) {
      const int p = min(j, j ^ mask), q = max(j, j ^ mask);
      const double app = __shfl_sync(all, a, 8 * p + 2 * p), aqq = __shfl_sync(all, a, 8 * q + 2 * q);
      const float br = (float)(__shfl_sync(all, a, 8 * p + 2 * q)), bi = (float)(__shfl_sync(all, a, 8 * p + 2 * q + 1));
      const float n2 = fmaf(br, br, bi * bi);
      double c = 1.0, sr = 0.0, si = 0.0;   // [[c, s], [-conj(s), c]] on (p, q)
      if (n2 > 1e-37f) {
        const float h = 0.5f * (float)(aqq - app), g = fmaf(h, h, n2);
        const float f = copysignf(__fdividef(1.f, fabsf(h) + g * rsqrtf(g)), h), vv = fmaf(n2 * f, f, 1.f), cf = rsqrtf(vv);
        sr = (double)(cf * f * br);
        si = (double)(cf * f * bi);
        const double x = fma(-sr, sr, fma(-si, si, 1.0)), hc = (double)(0.5f * vv * cf);
        c = (double)cf;
        c = fma(fma(-c, c, x), hc, c);
        c = fma(fma(-c, c, x), hc, c);
      }
      const bool jq = j & (mask & 2 ? 2 : 1) ? true : false, iq = i & (mask & 2 ? 2 : 1) ? true : false;   // the larger of its pair
      // the rotation of this lane's row pair is the one of column i
      const double ci = __shfl_sync(all, c, 2 * i), sri = __shfl_sync(all, sr, 2 * i), sii = __shfl_sync(all, si, 2 * i);
      const double srj = flip(sr, !jq), sij = flip(si, !m);
      // A J and U J: the other column's components
      const double av = __shfl_xor_sync(all, a, 2 * mask), aw = __shfl_xor_sync(all, a, 2 * mask + 1);
      const double uv = __shfl_xor_sync(all, u, 2 * mask), uw = __shfl_xor_sync(all, u, 2 * mask + 1);
      const double y = fma(c, a, fma(srj, av, sij * aw));
      u = fma(c, u, fma(srj, uv, sij * uw));
      // J^H (A J): the other row's
      const double yv = __shfl_xor_sync(all, y, 8 * mask), yw = __shfl_xor_sync(all, y, 8 * mask + 1);
      a = fma(ci, y, fma(flip(sri, !iq), yv, flip(sii, m) * yw));
      if (i == j && m) a = 0.0;
    }
  }
  reinterpret_cast<double *>(U)[2 * (4 * j + i) + m] = u;
  if (i == j && m == 0) w[i] = a * __hiloint2double((2046 - es) << 20, 0);
  __syncwarp();
}
// C = A B (4 x 4) by one warp; B conjugate-transposed with bh.
__device__ void mul4(const zd *A, const zd *B, bool bh, zd *C) {
  const int lane = threadIdx.x & 31, m = lane & 1, j = (lane >> 1) & 3, i = lane >> 3;
  double v = 0.0;
#pragma unroll
  for (int x = 0; x < 4; ++x) {
    const zd a = A[4 * x + i], b = bh ? conj(B[4 * x + j]) : B[4 * j + x];
    v = fma(a.re, m ? b.im : b.re, fma(m ? a.im : -a.im, m ? b.re : b.im, v));
  }
  reinterpret_cast<double *>(C)[2 * (4 * j + i) + m] = v;
  __syncwarp();
}
}  // namespace

// One CTA per pair: R from the partials, the Werner map, then the concurrence by warp 0 and the negativity by warp 1.
// out: [npairs][32 + 2] doubles: R (4 x 4 complex, column-major), concurrence, negativity.
__global__ void __launch_bounds__(256) rdm_final_kernel(const double *__restrict__ partial, int nparts, int npairs,
                                                        double p_werner, double *__restrict__ out) {
  __shared__ double sl[16][16], s[16];
  __shared__ zd R[16], A[16], U[16], S[16], Rt[16], Tm[16], A1[16], U1[16];
  __shared__ double w[4], w1[4];
  const int q = blockIdx.x, t = threadIdx.x, lane = t & 31;
  {   // slices of the parts, then the slices
    double v = 0.0;
    for (int b = t >> 4; b < nparts; b += 16) v += partial[((size_t)q * nparts + b) * 16 + (t & 15)];
    sl[t >> 4][t & 15] = v;
  }
  __syncthreads();
  if (t < 16) {
    double v = 0.0;
    for (int b = 0; b < 16; ++b) v += sl[b][t];
    s[t] = (1.0 - p_werner) * v;
  }
  __syncthreads();
  double *o = out + (size_t)q * 34;
  if (t < 16) {
    const int i = t % 4, j = t / 4, lo = min(i, j), hi = max(i, j);
    zd v;
    if (i == j) {
      v = mk<double>(s[i] + 0.25 * p_werner, 0.0);
    } else {
      const int e = 4 + 2 * (lo == 0 ? hi - 1 : (lo == 1 ? hi + 1 : 5));   // (0,1) (0,2) (0,3) (1,2) (1,3) (2,3)
      v = mk<double>(s[e], i < j ? s[e + 1] : -s[e + 1]);
    }
    R[t] = v;
    o[2 * t] = v.re;
    o[2 * t + 1] = v.im;
  }
  __syncthreads();
  if (t < 32) {
    // concurrence: C = max(0, s1 - s2 - s3 - s4), s_i the decreasing square roots of the eigenvalues
    // of R Rt, Rt = (Y x Y) conj(R) (Y x Y), which are those of the Hermitian sqrt(R) Rt sqrt(R)
    herm4_eig(R, U, w);
    if (lane < 16) {
      const int i = lane % 4, j = lane / 4;
      // (Y x Y)_{ab} = -1 for (a, b) in {(0,3), (3,0)}, +1 for {(1,2), (2,1)}, 0 otherwise:
      // Rt_ij = sum yy_i,a conj(R_ab) yy_b,j with a = 3 - i, b = 3 - j
      const bool neg = (i == 0 || i == 3) != (j == 0 || j == 3);
      Rt[lane] = (neg ? -1.0 : 1.0) * conj(R[(3 - j) * 4 + 3 - i]);
      Tm[lane] = sqrt(fmax(w[j], 0.0)) * U[lane];
    }
    __syncwarp();
    mul4(Tm, U, true, S);
    mul4(Rt, S, false, Tm);
    mul4(S, Tm, false, A);
    if (lane < 16) {
      const int i = lane % 4, j = lane / 4;
      const zd x = A[lane], y = A[i * 4 + j];
      Tm[lane] = mk<double>(0.5 * (x.re + y.re), i == j ? 0.0 : 0.5 * (x.im - y.im));
    }
    __syncwarp();
    herm4_eig(Tm, U, w);
    const double v = sqrt(fmax(w[lane & 3], 0.0));
    double big = v, sum = v;
#pragma unroll
    for (int x = 1; x <= 2; x <<= 1) {
      big = fmax(big, __shfl_xor_sync(0xffffffffu, big, x));
      sum += __shfl_xor_sync(0xffffffffu, sum, x);
    }
    if (lane == 0) o[32] = fmax(0.0, 2.0 * big - sum);
  } else if (t < 64) {
    // negativity: minus the sum of the negative eigenvalues of the partial transpose on spin l:
    // T[(a0 a1), (b0 b1)] = R[(a0 b1), (b0 a1)]
    if (lane < 16) {
      const int a0 = lane & 1, a1 = (lane >> 1) & 1, b0 = (lane >> 2) & 1, b1 = lane >> 3;
      A1[(2 * b0 + b1) * 4 + (2 * a0 + a1)] = R[(2 * b0 + a1) * 4 + (2 * a0 + b1)];
    }
    __syncwarp();
    herm4_eig(A1, U1, w1);
    if (lane == 0) {
      double neg = 0.0;
      for (int i = 0; i < 4; ++i)
        if (w1[i] < 0.0) neg -= w1[i];
      o[33] = neg;
    }
  }
}

int launch_rdm(bool fp64, const void *V, long long N, int r, const double *lam, const int *pairs, int npairs,
               double *partial, int ncta, cudaStream_t st) {
  if (npairs <= 0 || r < 1 || r > 256 || N < 4) return -1;
  dim3 grid(ncta, npairs);
  ::lrei::count_launch();
  if (fp64) rdm_kernel<double><<<grid, 256, 0, st>>>((const cx<double> *)V, N, r, lam, pairs, partial);
  else rdm_kernel<float><<<grid, 256, 0, st>>>((const cx<float> *)V, N, r, lam, pairs, partial);
  return 0;
}

void launch_rdm_final(const double *partial, int nparts, int npairs, double p_werner, double *out, cudaStream_t st) {
  ::lrei::count_launch();
  rdm_final_kernel<<<npairs, 256, 0, st>>>(partial, nparts, npairs, p_werner, out);
}

}  // namespace lrei
