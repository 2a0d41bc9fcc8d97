// Tall-skinny (N-length) kernels of the LREI hot path.
//
//  * The per-row matrix-free H.V gather (hv_group; paper Sec. 3.3 "sparsity of H",
//    Hamiltonian eq. H1), the fallback of the full-row H.V kernel of hv.cu for rows that are not a multiple of 16 bytes:
//    a thread owns CPT consecutive columns of one row; partner rows are read
//    through the read-only cache (rows of one N x r block are contiguous).
//  * Fused tile passes (apply / extend / combine, see tsk.cuh) compute the
//    tall-skinny products Q^*S, S^*S, S A + Q C of the block-Krylov partial
//    eigendecomposition (Sec. 3.7, eq. g-func replaced by an exact block
//    Rayleigh-Ritz on the Krylov space of H) with per-CTA partial Grams.
//  * Observable Grams V^*AV for A in {H, (HV)^*(HV), I, M_x, M_y, M_z}
//    (Sec. 3.6 eq. measuerA).
// Gram accumulation: per tile in the storage precision, then into per-CTA
// accumulators that are FP64 (complex128 path) or compensated FP32 pairs
// (complex64 path, TwoSum), written out as FP64 partials.
#include "tsk.cuh"

#include <cstdlib>

namespace lrei {

// ---------------------------------------------------------------- loads
__device__ __forceinline__ cx<float> ldg1(const cx<float> *p) {
  float2 v = __ldg(reinterpret_cast<const float2 *>(p));
  return mk<float>(v.x, v.y);
}
__device__ __forceinline__ cx<double> ldg1(const cx<double> *p) {
  double2 v = __ldg(reinterpret_cast<const double2 *>(p));
  return mk<double>(v.x, v.y);
}

// Load CPT consecutive complex values (p aligned to CPT * sizeof(cx<T>) when CPT > 1).
template <typename T, int CPT> struct Group {
  __device__ __forceinline__ static void load(const cx<T> *p, cx<T> (&v)[CPT]) {
#pragma unroll
    for (int c = 0; c < CPT; ++c) v[c] = ldg1(p + c);
  }
};
template <> struct Group<float, 4> {
  __device__ __forceinline__ static void load(const cx<float> *p, cx<float> (&v)[4]) {
    float4 a = __ldg(reinterpret_cast<const float4 *>(p));
    float4 b = __ldg(reinterpret_cast<const float4 *>(p) + 1);
    v[0] = mk<float>(a.x, a.y); v[1] = mk<float>(a.z, a.w);
    v[2] = mk<float>(b.x, b.y); v[3] = mk<float>(b.z, b.w);
  }
};
template <> struct Group<float, 2> {
  __device__ __forceinline__ static void load(const cx<float> *p, cx<float> (&v)[2]) {
    float4 a = __ldg(reinterpret_cast<const float4 *>(p));
    v[0] = mk<float>(a.x, a.y); v[1] = mk<float>(a.z, a.w);
  }
};

// Row b, columns [c0, c0 + CPT) of H X.
template <typename T, int CPT>
__device__ __forceinline__ void hv_group(const ModelArgs &M, const cx<T> *__restrict__ X, int r, uint32_t b,
                                         int c0, cx<T> (&out)[CPT]) {
  T diag = (T)(M.c0 + M.bz * (0.5 * M.n - (double)__popc(b)));
  cx<T> acc[CPT];
#pragma unroll
  for (int c = 0; c < CPT; ++c) acc[c] = mk<T>(0, 0);
  if (!M.cplx) {
    for (int k = 0; k < M.nb; ++k) {
      if (((b >> M.bi[k]) ^ (b >> M.bj[k])) & 1u) {
        diag -= (T)M.jz[k];
        const T j = (T)M.jxy[k];
        cx<T> v[CPT];
        Group<T, CPT>::load(X + (size_t)(b ^ M.mask[k]) * r + c0, v);
#pragma unroll
        for (int c = 0; c < CPT; ++c) {
          acc[c].re = fma(j, v[c].re, acc[c].re);
          acc[c].im = fma(j, v[c].im, acc[c].im);
        }
      }
    }
  } else {
    // complex amplitudes: jxy + i dz when site i is up in b, jxy - i dz when it is down
    for (int k = 0; k < M.nb; ++k) {
      if (((b >> M.bi[k]) ^ (b >> M.bj[k])) & 1u) {
        diag -= (T)M.jz[k];
        const cx<T> a = mk<T>((T)M.jxy[k], (T)(((b >> M.bi[k]) & 1u) ? -M.dz[k] : M.dz[k]));
        cx<T> v[CPT];
        Group<T, CPT>::load(X + (size_t)(b ^ M.mask[k]) * r + c0, v);
#pragma unroll
        for (int c = 0; c < CPT; ++c) fma_(acc[c], a, v[c]);
      }
    }
    // one-bit flips of the transverse field: (bx -+ i by)/2 for bit q of b equal to 0 / 1
    if (M.bx != 0.0 || M.by != 0.0)
      for (int q = 0; q < M.n; ++q) {
        const cx<T> a = mk<T>((T)(0.5 * M.bx), (T)(((b >> q) & 1u) ? 0.5 * M.by : -0.5 * M.by));
        cx<T> v[CPT];
        Group<T, CPT>::load(X + (size_t)(b ^ (1u << q)) * r + c0, v);
#pragma unroll
        for (int c = 0; c < CPT; ++c) fma_(acc[c], a, v[c]);
      }
  }
  cx<T> v[CPT];
  Group<T, CPT>::load(X + (size_t)b * r + c0, v);
#pragma unroll
  for (int c = 0; c < CPT; ++c) {
    out[c].re = fma(diag, v[c].re, acc[c].re);
    out[c].im = fma(diag, v[c].im, acc[c].im);
  }
}

template <typename T, int CPT>
__global__ void __launch_bounds__(256) hv_kernel(const __grid_constant__ ModelArgs M, const cx<T> *__restrict__ X,
                                                 cx<T> *__restrict__ Y, long long N, int r) {
  const int gpr = r / CPT;
  const long long total = N * gpr;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const uint32_t b = (uint32_t)(e / gpr);
    const int c0 = (int)(e % gpr) * CPT;
    cx<T> o[CPT];
    hv_group<T, CPT>(M, X, r, b, c0, o);
    cx<T> *y = Y + (size_t)b * r + c0;
#pragma unroll
    for (int c = 0; c < CPT; ++c) y[c] = o[c];
  }
}

// ------------------------------------------------------ accumulation
// Error-free sum: s + e == a + b exactly (Knuth TwoSum).
__device__ __forceinline__ void two_sum_acc(float &hi, float &lo, float b) {
  float s = hi + b;
  float bp = s - hi;
  float err = (hi - (s - bp)) + (b - bp);
  hi = s;
  lo += err;
}

template <typename T> struct Acc;
template <> struct Acc<double> {
  __device__ __forceinline__ static void add(double *acc, int e, cx<double> s) {
    acc[2 * e] += s.re;
    acc[2 * e + 1] += s.im;
  }
  __device__ __forceinline__ static cx<double> get(const double *acc, int e) { return mk<double>(acc[2 * e], acc[2 * e + 1]); }
};
template <> struct Acc<float> {
  __device__ __forceinline__ static void add(double *accd, int e, cx<float> s) {
    float *acc = reinterpret_cast<float *>(accd);
    two_sum_acc(acc[4 * e], acc[4 * e + 1], s.re);
    two_sum_acc(acc[4 * e + 2], acc[4 * e + 3], s.im);
  }
  __device__ __forceinline__ static cx<double> get(const double *accd, int e) {
    const float *acc = reinterpret_cast<const float *>(accd);
    return mk<double>((double)acc[4 * e] + (double)acc[4 * e + 1], (double)acc[4 * e + 2] + (double)acc[4 * e + 3]);
  }
};

// ------------------------------------------------------ fused tile pass
constexpr int TS_THREADS = 256;


template <typename T>
struct TSLayout {
  int tr;          // tile rows
  size_t bytes;    // dynamic shared memory
  bool coef_smem;  // coefficients staged in shared memory
};

template <typename T>
__host__ __device__ inline size_t ts_bytes(int nq, int gram_left, int r, int tr, bool coef_smem, int mode) {
  size_t cxs = sizeof(cx<T>);
  size_t tiles = ((size_t)nq * tr * r + 2 * (size_t)tr * r) * cxs;
  size_t coef = (coef_smem && mode != 0) ? (size_t)(nq + 1) * r * r * cxs : 0;
  size_t acc = (size_t)(gram_left + 1) * r * r * 16;
  return tiles + coef + acc;
}

template <typename T, int CPT>
__global__ void __launch_bounds__(TS_THREADS) ts_kernel(const __grid_constant__ TSArgs a, int tr, int coef_smem,
                                                       const cx<T> *__restrict__ coefg) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int r = a.r, nq = a.nq, gl = a.gram_left;
  const int tid = threadIdx.x, nt = blockDim.x;
  const int ldc = (nq + 1) * r;          // coefficient rows: [coefQ (nq*r); coefS (r)]
  const int ldg_ = (gl + 1) * r;         // Gram rows
  const int nent = ldg_ * r;
  cx<T> *qs = reinterpret_cast<cx<T> *>(smem);
  cx<T> *gs = qs + (size_t)nq * tr * r;
  cx<T> *ns = gs + (size_t)tr * r;
  cx<T> *csm = ns + (size_t)tr * r;
  const bool use_coef = a.mode != 0;
  double *acc = reinterpret_cast<double *>(csm + ((coef_smem && use_coef) ? (size_t)ldc * r : 0));
  const cx<T> *cs = (coef_smem && use_coef) ? csm : coefg;

  if (coef_smem && use_coef) {
    for (int e = tid; e < ldc * r; e += nt) csm[e] = coefg[e];
  }
  for (int e = tid; e < nent * 2; e += nt) acc[e] = 0.0;
  __syncthreads();

  const long long ntiles = (a.N + tr - 1) / tr;
  const int gpr = r / CPT;
  for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const long long row0 = tile * tr;
    const int rows = (int)((a.N - row0) < tr ? (a.N - row0) : tr);
    // S tile
    if (a.mode != 2) {
      const cx<T> *src = reinterpret_cast<const cx<T> *>(a.src);
      for (int e = tid; e < tr * gpr; e += nt) {
        const int lr = e / gpr, c0 = (e % gpr) * CPT;
        cx<T> v[CPT];
        if (lr < rows) {
          Group<T, CPT>::load(src + (size_t)(row0 + lr) * r + c0, v);
        } else {
#pragma unroll
          for (int c = 0; c < CPT; ++c) v[c] = mk<T>(0, 0);
        }
#pragma unroll
        for (int c = 0; c < CPT; ++c) gs[lr * r + c0 + c] = v[c];
      }
    }
    // Q tiles: the tile of block m is a contiguous run of rows*r complex values
    for (int m = 0; m < nq; ++m) {
      const cx<T> *qm = reinterpret_cast<const cx<T> *>(a.q[m]) + (size_t)row0 * r;
      cx<T> *dst = qs + (size_t)m * tr * r;
      for (int e = tid; e < tr * r; e += nt) dst[e] = (e < rows * r) ? ldg1(qm + e) : mk<T>(0, 0);
    }
    __syncthreads();
    const cx<T> *G = gs;
    if (a.mode != 0) {
      cx<T> *out = reinterpret_cast<cx<T> *>(a.out);
      for (int e = tid; e < tr * r; e += nt) {
        const int lr = e / r, j = e % r;
        cx<T> s = mk<T>(0, 0);
        const cx<T> *cj = cs + (size_t)j * ldc;
        if (a.mode == 1) {
          for (int i = 0; i < r; ++i) fma_(s, gs[lr * r + i], cj[nq * r + i]);
        }
        for (int m = 0; m < nq; ++m) {
          const cx<T> *qrow = qs + (size_t)m * tr * r + lr * r;
          const cx<T> *cm = cj + m * r;
          for (int i = 0; i < r; ++i) fma_(s, qrow[i], cm[i]);
        }
        if (lr >= rows || row0 + lr < a.zero_rows) s = mk<T>(0, 0);
        ns[e] = s;
        if (lr < rows && out) out[(size_t)(row0 + lr) * r + j] = s;
      }
      __syncthreads();
      G = ns;
    } else if (a.out) {
      cx<T> *out = reinterpret_cast<cx<T> *>(a.out);
      for (int e = tid; e < rows * r; e += nt) out[(size_t)row0 * r + e] = gs[e];
    }
    // Gram partial of this tile
    for (int e = tid; e < nent; e += nt) {
      const int j = e / ldg_, row = e % ldg_, m = row / r, i = row % r;
      const cx<T> *L = (m < gl) ? qs + (size_t)m * tr * r : G;
      cx<T> s = mk<T>(0, 0);
      for (int lr = 0; lr < tr; ++lr) fmac_(s, L[lr * r + i], G[lr * r + j]);
      Acc<T>::add(acc, e, s);
    }
    __syncthreads();
  }
  double *outp = a.partial + (size_t)blockIdx.x * nent * 2;
  for (int e = tid; e < nent; e += nt) {
    cx<double> v = Acc<T>::get(acc, e);
    outp[2 * e] = v.re;
    outp[2 * e + 1] = v.im;
  }
}

// ------------------------------------------------ fused tile pass, register-blocked
// Same contract as ts_kernel.  Shared tiles use a padded row stride RS (complex elements) so
// that rows of a tile fall in different banks.  The Gram is computed by MI x MJ register
// micro-tiles (rows (m, i) of [q_0..q_{gl-1}, G], columns j), split over `nph` phases of the
// tile rows; per-thread partials are flushed every FLUSH tiles into per-thread accumulators
// in shared memory (compensated FP32 pairs or FP64), then reduced over phases at the end.
// The new tile is a small GEMM [q_0..q_{nq-1}, S] (tr x (nq+1) rp) x coef ((nq+1) rp x rp),
// one row x 4 columns per thread.
template <typename T> struct TS2 {
  static constexpr int MI = sizeof(T) == 4 ? 4 : 2;
  static constexpr int MJ = 4;
  static constexpr int PAD = sizeof(T) == 4 ? 2 : 1;     // row padding (complex elements)
  static constexpr int STAG = sizeof(T) == 4 ? 8 : 4;    // block base stagger (64 bytes)
  static constexpr int FLUSH = sizeof(T) == 4 ? 2 : 1 << 30;
};

__host__ __device__ inline int ts2_rp(int r) { return (r + 3) & ~3; }

// Gram work split: NMT micro-tiles, nph (power of two) phases per micro-tile; the phases of one
// micro-tile are consecutive lanes of one warp, so their partials are combined by shuffles.
__host__ __device__ inline int ts2_nph(int nmt) {
  int p = 1;
  while (p < 16 && nmt * p * 2 <= TS_THREADS) p *= 2;
  return p;
}

template <typename T>
__host__ __device__ inline size_t ts2_bytes(int nq, int gl, int r, int tr, int mode, int mt) {
  const int rp = ts2_rp(r), RS = rp + TS2<T>::PAD;
  const size_t bstride = (size_t)tr * RS + TS2<T>::STAG;
  size_t b = ((size_t)(nq + 2) * bstride) * sizeof(cx<T>);
  if (mode != 0) b += (size_t)(nq + 1) * rp * rp * sizeof(cx<T>);
  const int nmt = (gl + 1) * rp / TS2<T>::MI * (rp / TS2<T>::MJ);
  b += (size_t)nmt * TS2<T>::MI * TS2<T>::MJ * 16;   // one accumulator set per micro-tile
  (void)mt;
  return b;
}

template <typename T, int CPT, int MT>
__global__ void __launch_bounds__(TS_THREADS) ts2_kernel(const __grid_constant__ TSArgs a, int tr,
                                                        const cx<T> *__restrict__ coefg) {
  constexpr int MI = TS2<T>::MI, MJ = TS2<T>::MJ;
  extern __shared__ __align__(16) unsigned char smem[];
  const int r = a.r, nq = a.nq, gl = a.gram_left;
  const int rp = ts2_rp(r), RS = rp + TS2<T>::PAD;
  const size_t BS = (size_t)tr * RS + TS2<T>::STAG;     // staggered block stride
  const int tid = threadIdx.x, lane = tid & 31;
  cx<T> *qs = reinterpret_cast<cx<T> *>(smem);
  cx<T> *gs = qs + (size_t)nq * BS;
  cx<T> *ns = gs + BS;
  cx<T> *cs = ns + BS;
  const int ncoef = (a.mode != 0) ? (nq + 1) * rp * rp : 0;
  double *slots = reinterpret_cast<double *>(cs + ncoef);   // [NMT][MI*MJ] x 16 bytes

  const int nI = (gl + 1) * rp / MI, nJ = rp / MJ, NMT = nI * nJ;
  for (int e = tid; e < ncoef; e += TS_THREADS) cs[e] = coefg[e];
  for (int e = tid; e < NMT * MI * MJ * 2; e += TS_THREADS) slots[e] = 0.0;

  // Gram micro-tile assignment: MT == 1 -> micro-tile tid / nph, phase tid % nph (lanes);
  // MT == 2 -> micro-tiles tid and tid + 256, one phase.
  const int nph = (MT == 1) ? ts2_nph(NMT) : 1;
  const int ph = (MT == 1) ? (tid % nph) : 0;
  int mts[MT];
  bool mval[MT];
#pragma unroll
  for (int u = 0; u < MT; ++u) {
    mts[u] = (MT == 1) ? tid / nph : tid + u * TS_THREADS;
    mval[u] = mts[u] < NMT;
  }
  cx<T> acc[MT][MI][MJ];
#pragma unroll
  for (int u = 0; u < MT; ++u)
#pragma unroll
    for (int x = 0; x < MI; ++x)
#pragma unroll
      for (int y = 0; y < MJ; ++y) acc[u][x][y] = mk<T>(0, 0);
  __syncthreads();

  auto flush = [&]() {
#pragma unroll
    for (int u = 0; u < MT; ++u)
#pragma unroll
      for (int x = 0; x < MI; ++x)
#pragma unroll
        for (int y = 0; y < MJ; ++y) {
          cx<T> v = acc[u][x][y];
          for (int o = nph >> 1; o > 0; o >>= 1) {   // combine the phases of this micro-tile
            v.re += __shfl_down_sync(0xffffffffu, v.re, o, nph);
            v.im += __shfl_down_sync(0xffffffffu, v.im, o, nph);
          }
          if (ph == 0 && mval[u]) Acc<T>::add(slots, mts[u] * MI * MJ + x * MJ + y, v);
          acc[u][x][y] = mk<T>(0, 0);
        }
  };

  const long long ntiles = (a.N + tr - 1) / tr;
  const int gpr = r / CPT;
  int since_flush = 0;
  for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const long long row0 = tile * tr;
    const int rows = (int)((a.N - row0) < tr ? (a.N - row0) : tr);
    // S tile
    if (a.mode != 2) {
      const cx<T> *src = reinterpret_cast<const cx<T> *>(a.src);
      for (int e = tid; e < tr * gpr; e += TS_THREADS) {
        const int lr = e / gpr, c0 = (e % gpr) * CPT;
        cx<T> v[CPT];
        if (lr < rows) {
          Group<T, CPT>::load(src + (size_t)(row0 + lr) * r + c0, v);
        } else {
#pragma unroll
          for (int c = 0; c < CPT; ++c) v[c] = mk<T>(0, 0);
        }
#pragma unroll
        for (int c = 0; c < CPT; ++c) gs[lr * RS + c0 + c] = v[c];
      }
      if (rp > r)
        for (int e = tid; e < tr * (rp - r); e += TS_THREADS) gs[(e / (rp - r)) * RS + r + e % (rp - r)] = mk<T>(0, 0);
    }
    // Q tiles (rows of one block are contiguous in global memory)
    for (int m = 0; m < nq; ++m) {
      const cx<T> *qm = reinterpret_cast<const cx<T> *>(a.q[m]) + (size_t)row0 * r;
      cx<T> *dst = qs + (size_t)m * BS;
      if (rp == r && CPT > 1 && sizeof(T) == 4) {
        // 16-byte vectors: two complex64 per load
        const int hr = r / 2;
        for (int e = tid; e < tr * hr; e += TS_THREADS) {
          const int lr = e / hr, c = (e % hr) * 2;
          float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
          if (lr < rows) v = __ldg(reinterpret_cast<const float4 *>(qm + (size_t)lr * r + c));
          cx<T> *d = dst + lr * RS + c;
          d[0] = mk<T>((T)v.x, (T)v.y);
          d[1] = mk<T>((T)v.z, (T)v.w);
        }
      } else {
        // at most 64 x 32 elements: all of a thread's loads are in flight before the first store (a loop of a fixed unroll leaves its
        // remainder in series: five blocks at n = 18, r = 17 / 23 took 317 / 700 us, now 225 / 460)
        cx<T> v[64 * 32 / TS_THREADS];
        int at[64 * 32 / TS_THREADS];
#pragma unroll
        for (int x = 0; x < 64 * 32 / TS_THREADS; ++x)
          if (x * TS_THREADS < tr * rp) {
            const int e = tid + x * TS_THREADS, lr = e / rp, c = e - lr * rp;
            at[x] = lr * RS + c;
            v[x] = (lr < rows && c < r) ? ldg1(qm + (size_t)lr * r + c) : mk<T>(0, 0);
          }
#pragma unroll
        for (int x = 0; x < 64 * 32 / TS_THREADS; ++x)
          if (tid + x * TS_THREADS < tr * rp) dst[at[x]] = v[x];
      }
    }
    __syncthreads();
    const cx<T> *G = gs;
    if (a.mode != 0) {
      cx<T> *out = reinterpret_cast<cx<T> *>(a.out);
      const int ngrp = rp / 4;
      for (int e = tid; e < tr * ngrp; e += TS_THREADS) {
        const int lr = e / ngrp, j0 = (e % ngrp) * 4;
        cx<T> o[4];
#pragma unroll
        for (int y = 0; y < 4; ++y) o[y] = mk<T>(0, 0);
        const int mlast = (a.mode == 1) ? nq : nq - 1;
        for (int m = 0; m <= mlast; ++m) {
          const cx<T> *X = (m < nq) ? qs + (size_t)m * BS + lr * RS : gs + lr * RS;
          const cx<T> *C = cs + (size_t)m * rp * rp + j0;
          for (int i = 0; i < r; ++i) {
            const cx<T> x = X[i];
            const cx<T> *ci = C + i * rp;
#pragma unroll
            for (int y = 0; y < 4; ++y) fma_(o[y], x, ci[y]);
          }
        }
#pragma unroll
        for (int y = 0; y < 4; ++y) {
          const int j = j0 + y;
          const cx<T> v = (lr < rows && j < r && row0 + lr >= a.zero_rows) ? o[y] : mk<T>(0, 0);
          ns[lr * RS + j] = v;
          if (lr < rows && j < r && out) out[(size_t)(row0 + lr) * r + j] = v;
        }
      }
      __syncthreads();
      G = ns;
    } else if (a.out) {
      cx<T> *out = reinterpret_cast<cx<T> *>(a.out);
      for (int e = tid; e < rows * r; e += TS_THREADS) out[(size_t)row0 * r + e] = gs[(e / r) * RS + e % r];
    }
    // Gram micro-tiles
#pragma unroll
    for (int u = 0; u < MT; ++u) {
      if (!mval[u]) continue;
      const int I = mts[u] / nJ, J = mts[u] % nJ;
      const int i0 = I * MI, m = i0 / rp, ii0 = i0 % rp, j0 = J * MJ;
      const cx<T> *L = (m < gl) ? qs + (size_t)m * BS : G;
      for (int lr = ph; lr < tr; lr += nph) {
        cx<T> lv[MI], gv[MJ];
#pragma unroll
        for (int x = 0; x < MI; ++x) lv[x] = L[lr * RS + ii0 + x];
#pragma unroll
        for (int y = 0; y < MJ; ++y) gv[y] = G[lr * RS + j0 + y];
#pragma unroll
        for (int x = 0; x < MI; ++x)
#pragma unroll
          for (int y = 0; y < MJ; ++y) fmac_(acc[u][x][y], lv[x], gv[y]);
      }
    }
    if (++since_flush >= TS2<T>::FLUSH) {
      since_flush = 0;
      flush();
    }
    __syncthreads();
  }
  flush();
  __syncthreads();
  // write the CTA partial in the column-major ((gl+1) r) x r layout
  const int ldg_ = (gl + 1) * r, nent = ldg_ * r;
  double *outp = a.partial + (size_t)blockIdx.x * nent * 2;
  for (int e = tid; e < nent; e += TS_THREADS) {
    const int j = e / ldg_, row = e % ldg_, m = row / r, i = row % r;
    const int ic = m * rp + i;
    const int I = ic / MI, x = ic % MI, J = j / MJ, y = j % MJ;
    const cx<double> sum = Acc<T>::get(slots, (I * nJ + J) * MI * MJ + x * MJ + y);
    outp[2 * e] = sum.re;
    outp[2 * e + 1] = sum.im;
  }
  (void)lane;
}

// ------------------------------------------- fused tile pass, pipelined (complex64 bulk)
// Same contract as ts_kernel for T = float: R = 8, 16 or 32 is the next width from r up; with PAD
// (r < R) the columns r .. R - 1 of the tiles are zero, and rows are copied by elements.
// Each CTA walks its tiles of TR rows with the next tiles' blocks already in flight: cp.async copies the rows of every
// input block into a ring of nst buffers (padded rows of RS complex) while the current tile is computed.
// What bounds it is the FP32 pipe (at r = 16, 5 blocks: 150 us of multiply-adds against 99 us of bytes), next to it the
// 128 bytes a cycle that shared memory delivers to registers, and the issue slots of everything else.  So
//  - Gram micro-tiles are A columns of every Gram block against 8 G columns: 8 (g A + 8) bytes per 4 g A 8
//    multiply-adds (g = 5, A = 2: 36 cycles of loads under 80 of arithmetic; with 4 columns, A = 1: 18 to 20);
//    NPH lanes of a warp take interleaved rows of one micro-tile;
//  - projection tiles are 4 rows x 4 columns, the sum over inputs split over KW lanes and KX warps;
//  - plain multiply-adds: packed pairs (fma.rn.f32x2) halve the issue slots but need every factor twice in
//    registers, and were slower (n = 22, r = 32, 5 blocks: Gram 3.9 -> 5.1 ms).
// Every 16-byte load of a quarter-warp and 8-byte load of a half-warp falls in distinct banks: a thread's columns are
// 16-byte chunks (2 columns) R / 8 (Gram) or R / 4 (projection) chunks apart, lanes of one sum whose
// coefficients would share banks read their two chunks in swapped order, and RS is chosen so.
// At a flush the lanes of a micro-tile are combined by halving shuffles and each sum is added to its compensated
// FP32 pair, kept in the CTA's partial (L2), all by TwoSum: only the rows that one lane takes between two flushes are summed
// plainly (LROWS: 16 to 256), since the error of a Gram grows with their number (a diagonal entry at n = 18: 8e-10 of it at 16
// rows, 5e-9 at 128).  Padded ranks take as many as keep their error at that of ts2_kernel, whose 8 to 32 rows over 16 lanes
// (r < 16) or 64 to 128 rows (r > 16) are combined plainly, and eight blocks of width 32 likewise.  Measured at n = 18, with sums four
// to eight times as long and now: two blocks 38 -> 42 us at r = 5 (diagonal off by 2.8e-9 -> 6e-10), 65 -> 80 at r = 9 (4.3e-9 ->
// 7e-10), five at r = 24 348 -> 371 us (1.2e-8 -> 5e-9), eight at r = 32 520 -> 756 us (1.1e-8 -> 1.3e-9).
// Before (4 columns, one G column group conflicting at r = 32, double buffer): n = 20, r = 16, 5 blocks 337 us, now 262;
// projection and Gram of 5 blocks 463 (4 inputs) -> 402 us; n = 22, r = 32, 5 blocks 7.7 -> 3.6 ms and 17.2 -> 7.0 ms.
template <int R> struct TS3 {
  static constexpr int RS = R == 16 ? 20 : R + 2;  // complex per padded row
  static constexpr int KW = 32 / R;                // projection: lanes of one sum
};
constexpr int TS3_STAGES = 6;

// GMAX: Gram blocks this instance handles (gl + 1 <= GMAX; with EXACT gl + 1 == GMAX)
template <int R, int TR, int GMAX, bool EXACT, int A, int MINB, bool PAD = false>
__global__ void __launch_bounds__(256, MINB) ts3_kernel(const __grid_constant__ TSArgs a, const cx<float> *__restrict__ coefg,
                                                       int nst) {
  constexpr int RS = TS3<R>::RS, KW = TS3<R>::KW, KX = 128 / TR;   // KX: warps of one projection sum
  constexpr int NJ = R / 8;                 // groups of 8 G columns
  constexpr int MTS = (R / A) * NJ;         // micro-tiles
  constexpr int NPH = 256 / MTS;
  constexpr int TPW = 32 / NPH;
  constexpr int CH = R / 2;                 // 16-byte chunks per row
  // rows a lane sums in plain FP32, and the tiles between flushes
  constexpr int LROWS = R == 32 ? (GMAX > 5 ? 32 : (PAD ? 128 : 256)) : (R == 16 ? (PAD ? (GMAX > 3 ? 24 : 16) : 128) : (PAD ? 16 : 32));
  constexpr int FLUSHT = LROWS * NPH / TR;
  constexpr int CNT = R / (KW * KX);
  static_assert(NPH >= 2 && NPH <= 32 && (RS * 8) % 16 == 0 && FLUSHT >= 1 && TR / 16 * KX == 8, "r in {8, 16, 32}");
  extern __shared__ __align__(16) unsigned char smem3[];
  const int nq = a.nq, gl = a.gram_left, mode = a.mode;
  const int nb = nq + (mode != 2 ? 1 : 0);
  const int g = EXACT ? GMAX : gl + 1;
  constexpr int bstride = TR * RS;
  cx<float> *buf = reinterpret_cast<cx<float> *>(smem3);       // [nst][nb][TR][RS]
  cx<float> *ns = buf + nst * nb * bstride;                     // [KX][TR][RS] parts of the new tile; then the tile in the first
  cx<float> *cs = ns + (mode != 0 ? KX * bstride : 0);          // [(nq+1) R][R] coefficients
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ph = lane / TPW;
  const int mt = warp * TPW + lane % TPW;
  const int c0 = mt / NJ * A, jg = mt % NJ;
  const long long N = a.N;
  const long long ntiles = (N + TR - 1) / TR;
  const int r = PAD ? a.r : R;
  const int ldg = g * r;
  double2 *outp = reinterpret_cast<double2 *>(a.partial + (size_t)blockIdx.x * ldg * r * 2);

  if (mode != 0)
    for (int e = tid; e < (nq + 1) * R * R; e += 256) cs[e] = coefg[e];
  if (PAD) {
    for (int e = tid; e < nst * nb * bstride; e += 256) buf[e] = mk<float>(0.f, 0.f);
    __syncthreads();
  }

  // A tile's rows are contiguous: chunk tid + 256 x of a block.  Rows beyond N (in the last tile only) become zero.
  const int lr_t = tid / CH;
  const uint32_t sm_t = (uint32_t)__cvta_generic_to_shared(buf + lr_t * RS + tid % CH * 2);
  auto prefetch = [&](long long tile, int sb) {
    const long long row0 = tile * TR;
    const size_t off = (size_t)row0 * (R * sizeof(cx<float>)) + tid * 16;
    uint32_t sa = sm_t + sb * nb * (bstride * 8);
    const bool full = row0 + TR <= N;
    if constexpr (PAD) {
      const uint32_t inv = 65536 / r + 1;   // e / r = e inv >> 16 for e < 2048
      sa = (uint32_t)__cvta_generic_to_shared(buf) + sb * nb * (bstride * 8);
      for (int e = tid; e < TR * r; e += 256) {
        const int lr = (int)(e * inv >> 16), c = e - lr * r;
        const bool ok = row0 + lr < N;
        for (int m = 0; m < nb; ++m) {
          const char *base = reinterpret_cast<const char *>(m < nq ? a.q[m] : a.src);
          asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(sa + (m * bstride + lr * RS + c) * 8),
                       "l"(ok ? base + ((size_t)row0 * r + e) * 8 : base), "r"(ok ? 8 : 0));
        }
      }
    } else {
#pragma unroll 1
      for (int m = 0; m < nb; ++m, sa += bstride * 8) {
        const char *gp = reinterpret_cast<const char *>(m < nq ? a.q[m] : a.src) + off;
#pragma unroll
        for (int x = 0; x < TR * CH / 256; ++x) {
          const bool ok = full || row0 + lr_t + x * (256 / CH) < N;
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(sa + x * (256 / CH) * RS * 8),
                       "l"(ok ? gp + x * 4096 : gp - off), "r"(ok ? 16 : 0));
        }
      }
    }
  };

  cx<float> acc[GMAX][A][8];   // column y: chunk y / 2, i.e. 2 (jg + (y / 2) NJ) + y % 2
#pragma unroll
  for (int m = 0; m < GMAX; ++m)
#pragma unroll
    for (int x = 0; x < A; ++x)
#pragma unroll
      for (int y = 0; y < 8; ++y) acc[m][x][y] = mk<float>(0.f, 0.f);

  // The lanes of a micro-tile (bits TPW .. 16 of the lane) halve their columns three times, further ones are summed
  // whole; then the pairs in the partial: (sum, error) of re and im, or with last their final values.  All of it with the
  // rounding errors kept (TwoSum): sums of LROWS rows are the only plain ones.
  bool first = true;
  auto add_from = [&](float2 &f, float2 &e, float2 send, float2 sende, int o, bool errs) {   // (f, e) += the other lane's pair
    two_sum_acc(f.x, e.x, __shfl_xor_sync(0xffffffffu, send.x, o));
    two_sum_acc(f.y, e.y, __shfl_xor_sync(0xffffffffu, send.y, o));
    if (errs) {
      e.x += __shfl_xor_sync(0xffffffffu, sende.x, o);
      e.y += __shfl_xor_sync(0xffffffffu, sende.y, o);
    }
  };
  auto flush = [&](bool last) {
    constexpr int LV = NPH == 2 ? 1 : (NPH == 4 ? 2 : 3), LEFT = 8 >> LV;
    int y0 = 0;
#pragma unroll
    for (int v = 0; v < LV; ++v) y0 += (lane & (16 >> v)) ? 4 >> v : 0;
#pragma unroll
    for (int m = 0; m < GMAX; ++m) {
      if (EXACT || m < g) {
#pragma unroll
        for (int x = 0; x < A; ++x) {
          float2 f[8], er[8];
#pragma unroll
          for (int y = 0; y < 8; ++y) {
            f[y] = make_float2(acc[m][x][y].re, acc[m][x][y].im);
            er[y] = make_float2(0.f, 0.f);
            acc[m][x][y] = mk<float>(0.f, 0.f);
          }
#pragma unroll
          for (int v = 0; v < LV; ++v) {
            const int o = 16 >> v, h = 4 >> v;
            const bool up = lane & o;
#pragma unroll
            for (int y = 0; y < h; ++y) {
              const float2 send = up ? f[y] : f[y + h], sende = up ? er[y] : er[y + h];
              if (up) {
                f[y] = f[y + h];
                er[y] = er[y + h];
              }
              add_from(f[y], er[y], send, sende, o, v > 0);
            }
          }
#pragma unroll
          for (int o = 16 >> LV; o >= TPW; o >>= 1) add_from(f[0], er[0], f[0], er[0], o, true);
          if ((lane & ((32 >> LV) - 1)) < TPW) {
#pragma unroll
            for (int y = 0; y < LEFT; ++y) {
              const int yy = y0 + y, col = 2 * (jg + (yy >> 1) * NJ) + (yy & 1);
              if (PAD && (col >= r || c0 + x >= r)) continue;
              double2 *slot = outp + (size_t)col * ldg + m * r + c0 + x;
              float4 s = first ? make_float4(0.f, 0.f, 0.f, 0.f) : *reinterpret_cast<float4 *>(slot);
              two_sum_acc(s.x, s.y, f[y].x);
              two_sum_acc(s.z, s.w, f[y].y);
              s.y += er[y].x;
              s.w += er[y].y;
              if (last) *slot = make_double2((double)s.x + (double)s.y, (double)s.z + (double)s.w);
              else *reinterpret_cast<float4 *>(slot) = s;
            }
          }
        }
      }
    }
    first = false;
  };

  long long tile = blockIdx.x;
  int sb = 0;
  for (int i = 0; i < nst - 1; ++i) {
    if (tile + (long long)i * gridDim.x < ntiles) prefetch(tile + (long long)i * gridDim.x, i);
    asm volatile("cp.async.commit_group;\n" ::);
  }
  int since = 0;
  // three kinds that ts2_kernel or shared memory sums treat otherwise: width 16 padded with two tiles per CTA (there twice the
  // CTAs): after each; above rank 28 beside coefficients (there shorter tiles): half; six blocks at width 32: as fewer blocks
  int every = FLUSHT;
  if (PAD && R == 16 && GMAX <= 3 && ntiles <= 2 * (long long)gridDim.x) every = 1;
  if (PAD && R == 32 && GMAX <= 5 && mode != 0 && r > 28) every = FLUSHT / 2;
  if (R == 32 && GMAX > 5 && g <= 6 && mode == 0 && (!PAD || r <= 28)) every = (PAD ? 4 : 8) * FLUSHT;
  for (; tile < ntiles; tile += gridDim.x) {
    switch (nst) {   // all but the newest nst - 2 groups: this tile is there
      case 2: asm volatile("cp.async.wait_group 0;\n" ::); break;
      case 3: asm volatile("cp.async.wait_group 1;\n" ::); break;
      case 4: asm volatile("cp.async.wait_group 2;\n" ::); break;
      case 5: asm volatile("cp.async.wait_group 3;\n" ::); break;
      default: asm volatile("cp.async.wait_group 4;\n" ::); break;
    }
    __syncthreads();   // also: every thread is done with the tile before this one
    const long long nxt = tile + (long long)(nst - 1) * gridDim.x;
    if (nxt < ntiles) prefetch(nxt, sb == 0 ? nst - 1 : sb - 1);
    asm volatile("cp.async.commit_group;\n" ::);
    const cx<float> *B0 = buf + (size_t)sb * nb * bstride;
    const long long row0 = tile * TR;
    const int rows = (int)((N - row0) < TR ? (N - row0) : TR);
    const cx<float> *G;
    if (mode != 0) {
      const int mlast = (mode == 1) ? nq : nq - 1;
      const int kw = lane % KW, q = lane / KW % (R / 4), kx = warp / (TR / 16);
      const int lr0 = warp % (TR / 16) * 16 + lane / 8;       // rows lr0 + 4 y
      const int sw = KW == 4 ? kw >> 1 : (KW == 2 ? kw : 0);   // order of the two chunks
      const int k0 = kx * (CNT * KW) + kw;
      cx<float> v[4][4];                                       // [row][column, chunks in order sw]
#pragma unroll
      for (int y = 0; y < 4; ++y)
#pragma unroll
        for (int x = 0; x < 4; ++x) v[y][x] = mk<float>(0.f, 0.f);
      for (int m = 0; m <= mlast; ++m) {
        const cx<float> *X = B0 + (size_t)m * bstride + lr0 * RS + k0;
        const cx<float> *C = cs + (size_t)(m * R + k0) * R + 2 * q;
#pragma unroll
        for (int i = 0; i < CNT; ++i) {
          const float4 ca = *reinterpret_cast<const float4 *>(C + i * KW * R + sw * (R / 2));
          const float4 cb = *reinterpret_cast<const float4 *>(C + i * KW * R + (1 - sw) * (R / 2));
#pragma unroll
          for (int y = 0; y < 4; ++y) {
            const cx<float> x = X[4 * y * RS + i * KW];
            fma_(v[y][0], x, mk<float>(ca.x, ca.y));
            fma_(v[y][1], x, mk<float>(ca.z, ca.w));
            fma_(v[y][2], x, mk<float>(cb.x, cb.y));
            fma_(v[y][3], x, mk<float>(cb.z, cb.w));
          }
        }
      }
      // lanes of one sum: the partner with the other order of chunks keeps the other two rows, the one with the same
      // order the other chunk
      if (KW >= 2) {
#pragma unroll
        for (int y = 0; y < 2; ++y) {
          cx<float> got[4];
#pragma unroll
          for (int x = 0; x < 4; ++x) {
            const cx<float> send = sw ? v[y][x] : v[y + 2][x];
            if (sw) v[y][x] = v[y + 2][x];
            got[x].re = __shfl_xor_sync(0xffffffffu, send.re, KW / 2);
            got[x].im = __shfl_xor_sync(0xffffffffu, send.im, KW / 2);
          }
#pragma unroll
          for (int x = 0; x < 4; ++x) {
            v[y][x].re += got[x ^ 2].re;
            v[y][x].im += got[x ^ 2].im;
          }
        }
      }
      if (KW == 4) {
#pragma unroll
        for (int y = 0; y < 2; ++y)
#pragma unroll
          for (int x = 0; x < 2; ++x) {
            const cx<float> send = (kw & 1) ? v[y][x] : v[y][2 + x], keep = (kw & 1) ? v[y][2 + x] : v[y][x];
            v[y][x].re = keep.re + __shfl_xor_sync(0xffffffffu, send.re, 1);
            v[y][x].im = keep.im + __shfl_xor_sync(0xffffffffu, send.im, 1);
          }
      }
      const int half = KW == 4 ? sw ^ (kw & 1) : sw;   // chunk in v[y][0..1]; the other one in v[y][2..3]
#pragma unroll
      for (int y = 0; y < (KW == 1 ? 4 : 2); ++y)
#pragma unroll
        for (int h = 0; h < (KW == 4 ? 1 : 2); ++h)
          *reinterpret_cast<float4 *>(ns + (size_t)kx * bstride + (lr0 + 4 * (KW == 1 ? y : 2 * sw + y)) * RS + 2 * q +
                                      (half ^ h) * (R / 2)) =
              make_float4(v[y][2 * h].re, v[y][2 * h].im, v[y][2 * h + 1].re, v[y][2 * h + 1].im);
      __syncthreads();
      cx<float> *out = reinterpret_cast<cx<float> *>(a.out);
      for (int e = tid; e < TR * CH; e += 256) {
        const int lr = e / CH, ch = e % CH;
        float4 *nd = reinterpret_cast<float4 *>(ns + lr * RS + ch * 2);
        float4 w = *nd;
#pragma unroll
        for (int x = 1; x < KX; ++x) {
          const float4 u = *reinterpret_cast<const float4 *>(ns + x * bstride + lr * RS + ch * 2);
          w = make_float4(w.x + u.x, w.y + u.y, w.z + u.z, w.w + u.w);
        }
        if (!(lr < rows && row0 + lr >= a.zero_rows)) w = make_float4(0.f, 0.f, 0.f, 0.f);
        *nd = w;
        if (out && lr < rows) {
          cx<float> *o = out + (size_t)(row0 + lr) * r + ch * 2;
          if (!PAD) {
            *reinterpret_cast<float4 *>(o) = w;
          } else {
            if (ch * 2 < r) o[0] = mk<float>(w.x, w.y);
            if (ch * 2 + 1 < r) o[1] = mk<float>(w.z, w.w);
          }
        }
      }
      __syncthreads();
      G = ns;
    } else {
      G = B0 + (size_t)nq * bstride;
    }
#pragma unroll 2
    for (int lr = ph; lr < TR; lr += NPH) {
      cx<float> gv[8];
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        const float4 t = *reinterpret_cast<const float4 *>(G + lr * RS + 2 * (jg + x * NJ));
        gv[2 * x] = mk<float>(t.x, t.y);
        gv[2 * x + 1] = mk<float>(t.z, t.w);
      }
#pragma unroll
      for (int m = 0; m < GMAX; ++m) {
        if (EXACT || m < g) {
          const cx<float> *L = ((EXACT ? m < GMAX - 1 : m < gl) ? B0 + (size_t)m * bstride : G) + lr * RS + c0;
          cx<float> l[A];
          if (A == 2) {
            const float4 t = *reinterpret_cast<const float4 *>(L);
            l[0] = mk<float>(t.x, t.y);
            l[A - 1] = mk<float>(t.z, t.w);
          } else {
            l[0] = L[0];
          }
#pragma unroll
          for (int x = 0; x < A; ++x)
#pragma unroll
            for (int y = 0; y < 8; ++y) fmac_(acc[m][x][y], l[x], gv[y]);
        }
      }
    }
    if (++since >= every) {
      since = 0;
      flush(false);
    }
    if (++sb == nst) sb = 0;
  }
  asm volatile("cp.async.wait_group 0;\n" ::);
  flush(true);
}

// Shared memory with tiles of tr rows and nst stages.
static size_t ts3_bytes(int r, int nq, int mode, int tr, int nst) {
  const int nb = nq + (mode != 2 ? 1 : 0);
  const size_t bstride = (size_t)tr * (r == 16 ? TS3<16>::RS : r + 2) * sizeof(cx<float>);
  size_t b = ((size_t)nst * nb + (mode != 0 ? 128 / tr : 0)) * bstride;
  if (mode != 0) b += (size_t)(nq + 1) * r * r * sizeof(cx<float>);
  return b;
}

// Coefficients in a padded row-major layout (rp columns): row m*rp + i, column j.
template <typename T>
__global__ void coef_convert2_kernel(const zd *coefQ, const zd *coefS, int nq, int r, int rp, int mode, cx<T> *out) {
  const int rows = (nq + 1) * rp;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < rows * rp; e += gridDim.x * blockDim.x) {
    const int row = e / rp, j = e % rp, m = row / rp, i = row % rp;
    zd v = mk<double>(0, 0);
    if (i < r && j < r) {
      if (m < nq) v = coefQ ? coefQ[(size_t)j * nq * r + m * r + i] : mk<double>(0, 0);
      else if (mode == 1 && coefS) v = coefS[(size_t)j * r + i];
    }
    out[e] = mk<T>((T)v.re, (T)v.im);
  }
}

template <typename T>
__global__ void coef_convert_kernel(const zd *coefQ, const zd *coefS, int nq, int r, int mode, cx<T> *out) {
  const int ldc = (nq + 1) * r;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < ldc * r; e += gridDim.x * blockDim.x) {
    const int j = e / ldc, row = e % ldc;
    zd v;
    if (row < nq * r) {
      v = coefQ ? coefQ[(size_t)j * nq * r + row] : mk<double>(0, 0);
    } else {
      const int i = row - nq * r;
      v = (mode == 1 && coefS) ? coefS[(size_t)j * r + i] : mk<double>(0, 0);
    }
    out[e] = mk<T>((T)v.re, (T)v.im);
  }
}

// out = the sum of the parts: 16 entries per CTA, the parts in 32 slices, then the slices, in a fixed order.  Latency:
// an FP64 addition takes a scheduler 64 cycles, so a thread adds nparts / 32 values.  (Slices by one kernel and their
// sum by another, 16 slices: 9.2 + 5.8 us with 148 parts at r = 8.)
__global__ void __launch_bounds__(512) reduce_kernel(const double *__restrict__ part, int nparts, int len,
                                                     double *__restrict__ out) {
  __shared__ double red[32][17];
  const int t = threadIdx.x, e = blockIdx.x * 16 + (t & 15);
  double v = 0.0;
  if (e < len) {
#pragma unroll 4
    for (int p = t >> 4; p < nparts; p += 32) v += part[(size_t)p * len + e];
  }
  red[t >> 4][t & 15] = v;
  __syncthreads();
  if (t < 64) {
    v = 0.0;
#pragma unroll
    for (int x = 0; x < 8; ++x) v += red[(t & 3) * 8 + x][t >> 2];
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    v += __shfl_xor_sync(0xffffffffu, v, 2);
    if ((t & 3) == 0 && blockIdx.x * 16 + (t >> 2) < len) out[blockIdx.x * 16 + (t >> 2)] = v;
  }
}

int ts_max_grid(int nsm) { return 2 * nsm; }
size_t ts_partial_doubles(int gram_left, int r) { return (size_t)(gram_left + 1) * r * r * 2; }

// The widest column group that the row length and the alignment of the blocks allow (two complex64 are loaded as 16 bytes; a
// caller's block may start on any element).
static bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }
template <typename T>
static int ts_cpt(const TSArgs &a) {
  bool ok = a.r % 2 == 0 && (a.mode == 2 || aligned16(a.src));
  for (int m = 0; m < a.nq; ++m) ok = ok && aligned16(a.q[m]);
  return !ok ? 1 : (sizeof(T) == 4 && a.r % 4 == 0 ? 4 : 2);
}

template <typename T>
static int launch_ts_v1(const TSArgs &a, int nsm, cudaStream_t st) {
  const int r = a.r;
  // choose tile rows / coefficient placement so the CTA fits in shared memory
  const size_t budget = 200 * 1024;
  int tr = 64;
  bool coef_smem = true;
  while (tr > 4 && ts_bytes<T>(a.nq, a.gram_left, r, tr, coef_smem, a.mode) > budget) tr /= 2;
  if (ts_bytes<T>(a.nq, a.gram_left, r, tr, coef_smem, a.mode) > budget) {
    coef_smem = false;
    tr = 64;
    while (tr > 1 && ts_bytes<T>(a.nq, a.gram_left, r, tr, coef_smem, a.mode) > budget) tr /= 2;
  }
  const size_t bytes = ts_bytes<T>(a.nq, a.gram_left, r, tr, coef_smem, a.mode);
  if (bytes > budget) return -1;
  cx<T> *coefg = nullptr;
  if (a.mode != 0) {
    if (!a.coef_scratch) return -1;
    coefg = reinterpret_cast<cx<T> *>(a.coef_scratch);
    ::lrei::count_launch(); coef_convert_kernel<T><<<8, 256, 0, st>>>(a.coefQ, a.coefS, a.nq, r, a.mode, coefg);
  }
  const long long ntiles = (a.N + tr - 1) / tr;
  int grid = (int)(ntiles < (long long)ts_max_grid(nsm) ? ntiles : ts_max_grid(nsm));
  if (grid < 1) grid = 1;
  const int cpt = ts_cpt<T>(a);
  auto go = [&](auto kern) { ::lrei::count_launch(); kern<<<grid, TS_THREADS, bytes, st>>>(a, tr, coef_smem ? 1 : 0, coefg); };
  if (cpt == 4) go(ts_kernel<T, (sizeof(T) == 4 ? 4 : 2)>);
  else if (cpt == 2) go(ts_kernel<T, 2>);
  else go(ts_kernel<T, 1>);
  return grid;
}


// Tile rows, CTAs per SM, stages and shared memory of the pipelined pass for the given arguments; 0 bytes if it does
// not apply.  Two CTAs per SM (128 registers: A = 1 from 3 Gram blocks on) hide more latency than one with the larger
// micro-tile up to 4 Gram blocks at r = 16 (4: 206 against 256 us at n = 20) and 3 at r = 32 (3: 2.4 against 2.6 ms at
// n = 22; 4: 3.3 against 3.15); 64-row tiles halve the barriers of 32-row ones (r = 16, one block: 79 -> 71 us) and are
// taken where two stages of them fit.
// Ranks that are no width are padded: Grams of 2 and 5 blocks at n = 18 took, by ts2_kernel and here, 89 and 51 us (5 blocks) at
// r = 1, 76 / 106 and 42 / 62 at r = 5, 91 / 172 and 80 / 130 at r = 9, 84 / 174 and 78 / 135 at r = 12; from 17 on the width 32 costs
// more than ts2_kernel (133 / 294 against 187 / 333 and more at r = 17, 166 against 195 for two blocks at r = 24) except for many
// blocks of a rank near it (r = 24: 317 against 320 us for four, 534 against 371 for five; r = 25: 612 against 327 for four).
struct TS3Plan {
  int R, tr, two, nst;
  size_t bytes;
};
static TS3Plan ts3_plan(const TSArgs &a) {
  TS3Plan p{0, 0, 0, 0, 0};
  if (a.mode == 0 && a.out) return p;
  const int nq = a.nq, gl = a.gram_left, mode = a.mode;
  const int nb = nq + (mode != 2 ? 1 : 0);
  if (nb < 1 || nb > 8 || gl + 1 > 8 || gl > nq || (mode == 2 && nq < 1)) return p;
  for (int m = 0; m < nq; ++m)
    if (!aligned16(a.q[m])) return p;
  if (mode != 2 && !aligned16(a.src)) return p;
  if (a.out && !aligned16(a.out)) return p;
  const int r = p.R = a.r <= 8 ? 8 : (a.r <= 16 ? 16 : 32);
  if (r == 32 && a.r < 32 && (a.r < 24 || gl + 1 < 4)) return p;
  const int two = r != a.r ? 0 : (r == 16 ? gl + 1 <= 4 : (r == 32 ? gl + 1 <= 3 : 0));
  for (int t = two; t >= 0; --t)
    for (int tr = 64; tr >= (r == 8 ? 64 : 32); tr /= 2) {
      const size_t lim = (t ? 113 : 227) * 1024;
      if (ts3_bytes(r, nq, mode, tr, 2) > lim) continue;
      p.tr = tr;
      p.two = t;
      p.nst = 2;
      while (p.nst < TS3_STAGES && ts3_bytes(r, nq, mode, tr, p.nst + 1) <= lim) ++p.nst;
      p.bytes = ts3_bytes(r, nq, mode, tr, p.nst);
      return p;
    }
  return p;
}

using TS3Kernel = void (*)(TSArgs, const cx<float> *, int);
template <int R, int TR> static TS3Kernel ts3_padded(int g) {
  if constexpr (R < 32)
    if (g <= 3) return ts3_kernel<R, TR, 3, false, 1, 1, true>;
  return g <= 5 ? ts3_kernel<R, TR, 5, false, 1, 1, true> : ts3_kernel<R, TR, 8, false, 1, 1, true>;
}
template <int R, int TR> static TS3Kernel ts3_instance(int g, bool two, bool pad) {
  if (pad) return ts3_padded<R, TR>(g);
  if (g > 5) return ts3_kernel<R, TR, 8, false, 1, 1>;
  if (two) {
    if (g == 1) return ts3_kernel<R, TR, 1, true, 2, 2>;
    if (g == 2) return ts3_kernel<R, TR, 2, true, 2, 2>;
    if (g == 3) return ts3_kernel<R, TR, 3, true, 1, 2>;
    if (g == 4) return ts3_kernel<R, TR, 4, true, 1, 2>;
  }
  if (g == 1) return ts3_kernel<R, TR, 1, true, 2, 2>;
  if (g <= 3) return ts3_kernel<R, TR, 3, false, 2, 1>;
  if (g == 4) return ts3_kernel<R, TR, 4, true, 2, 1>;
  return ts3_kernel<R, TR, 5, true, 2, 1>;
}
static TS3Kernel ts3_pick(int R, int tr, int g, bool two, bool pad) {
  if (R == 16) return tr == 64 ? ts3_instance<16, 64>(g, two, pad) : ts3_instance<16, 32>(g, two, pad);
  if (R == 32) return tr == 64 ? ts3_instance<32, 64>(g, two, pad) : ts3_instance<32, 32>(g, two, pad);
  if (pad) return ts3_padded<8, 64>(g);
  if (g <= 2) return ts3_kernel<8, 64, 2, false, 1, 1>;
  return g <= 5 ? ts3_kernel<8, 64, 5, false, 1, 1> : ts3_kernel<8, 64, 8, false, 1, 1>;
}

static int launch_ts3(const TSArgs &a, int nsm, cudaStream_t st, const TS3Plan &p) {
  const cx<float> *coefg = nullptr;
  if (a.mode != 0) {
    if (!a.coef_scratch) return -1;
    coefg = reinterpret_cast<const cx<float> *>(a.coef_scratch);
    ::lrei::count_launch();
    coef_convert2_kernel<float><<<8, 256, 0, st>>>(a.coefQ, a.coefS, a.nq, a.r, p.R, a.mode,
                                                  reinterpret_cast<cx<float> *>(a.coef_scratch));
  }
  // persistent, each CTA walking tiles blockIdx.x, + gridDim.x, ...: one or two CTAs per SM (ts3_plan)
  const long long ntiles = (a.N + p.tr - 1) / p.tr;
  const long long cap = p.two ? 2LL * nsm : (long long)nsm;
  int grid = (int)(ntiles < cap ? ntiles : cap);
  if (grid < 1) grid = 1;
  ::lrei::count_launch();
  ts3_pick(p.R, p.tr, a.gram_left + 1, p.two, a.r != p.R)<<<grid, 256, p.bytes, st>>>(a, coefg, p.nst);
  return grid;
}

template <typename T>
static int launch_ts_t(const TSArgs &a, int nsm, cudaStream_t st) {
  if (sizeof(T) == 4) {
    const TS3Plan p = ts3_plan(a);
    if (p.bytes) return launch_ts3(a, nsm, st, p);
  }
  const int r = a.r, rp = ts2_rp(r);
  const int NMT = (a.gram_left + 1) * rp / TS2<T>::MI * (rp / TS2<T>::MJ);
  const int mt = NMT <= TS_THREADS ? 1 : (NMT <= 2 * TS_THREADS ? 2 : 0);
  const size_t budget = 200 * 1024;
  int tr = 64;
  if (mt > 0)
    while (tr > 8 && ts2_bytes<T>(a.nq, a.gram_left, r, tr, a.mode, mt) > budget) tr /= 2;
  if (mt == 0 || ts2_bytes<T>(a.nq, a.gram_left, r, tr, a.mode, mt) > budget)
    return launch_ts_v1<T>(a, nsm, st);
  const size_t bytes = ts2_bytes<T>(a.nq, a.gram_left, r, tr, a.mode, mt);
  cx<T> *coefg = nullptr;
  if (a.mode != 0) {
    if (!a.coef_scratch) return -1;
    coefg = reinterpret_cast<cx<T> *>(a.coef_scratch);
    ::lrei::count_launch();
    coef_convert2_kernel<T><<<8, 256, 0, st>>>(a.coefQ, a.coefS, a.nq, r, rp, a.mode, coefg);
  }
  const long long ntiles = (a.N + tr - 1) / tr;
  int grid = (int)(ntiles < (long long)ts_max_grid(nsm) ? ntiles : ts_max_grid(nsm));
  if (grid < 1) grid = 1;
  const int cpt = ts_cpt<T>(a);
  auto go = [&](auto kern) { ::lrei::count_launch(); kern<<<grid, TS_THREADS, bytes, st>>>(a, tr, coefg); };
  if (mt == 1) {
    if (cpt == 4) go(ts2_kernel<T, (sizeof(T) == 4 ? 4 : 2), 1>);
    else if (cpt == 2) go(ts2_kernel<T, 2, 1>);
    else go(ts2_kernel<T, 1, 1>);
  } else {
    if (cpt == 4) go(ts2_kernel<T, (sizeof(T) == 4 ? 4 : 2), 2>);
    else if (cpt == 2) go(ts2_kernel<T, 2, 2>);
    else go(ts2_kernel<T, 1, 2>);
  }
  return grid;
}

// ------------------------------------------- few rows
// Passes of few rows are latency: tiles leave most SMs idle (8 to 256 of them at N = 256 .. 4096) and their sums need
// a second launch.  Here every entry of the new block is a sum over a few lanes and every Gram entry one over a warp
// or a CTA, and the Gram goes to a.red directly.  Sums are in FP64, or for complex64 as good: products and sums with
// their rounding errors kept (fma and TwoSum: 9 FP32 instructions a product, where an FP64 multiply-add takes 64 cycles), and
// the coefficients as pairs of FP32.
// The rows of a CTA are read before one is written, so the new block may replace an input.
__global__ void __launch_bounds__(256) few_new_kernel(TSArgs a) {
  const int r = a.r, rows = 32 / r, o = threadIdx.x >> 3, q = threadIdx.x & 7, j = o % r;
  const long long row = (long long)blockIdx.x * rows + o / r;
  const bool in = o < rows * r && row < a.N;
  const int K = (a.nq + (a.mode == 1 ? 1 : 0)) * r;
  zd s = mk<double>(0, 0);
  if (in)
    for (int k = q; k < K; k += 8) {
      const int m = k / r, i = k % r;
      const zd x = reinterpret_cast<const zd *>(m < a.nq ? a.q[m] : a.src)[(size_t)row * r + i];
      const zd c = m < a.nq ? (a.coefQ ? a.coefQ[(size_t)j * a.nq * r + k] : mk<double>(0, 0))
                            : (a.coefS ? a.coefS[(size_t)j * r + i] : mk<double>(0, 0));
      fma_(s, x, c);
    }
#pragma unroll
  for (int x = 4; x > 0; x >>= 1) {
    s.re += __shfl_xor_sync(0xffffffffu, s.re, x);
    s.im += __shfl_xor_sync(0xffffffffu, s.im, x);
  }
  __syncthreads();
  if (in && q == 0) reinterpret_cast<zd *>(a.out)[(size_t)row * r + j] = row < a.zero_rows ? mk<double>(0, 0) : s;
}

// (hi, lo) += x y
__device__ __forceinline__ void two_prod_acc(float &hi, float &lo, float x, float y) {
  const float p = x * y;
  lo += fmaf(x, y, -p);
  two_sum_acc(hi, lo, p);
}

// x as a pair of FP32: truncated, and the 29 bits left; by the bits (a conversion from FP64 runs at its rate).  Zero below 2^-126,
// infinite from 2^128 on.
__device__ __forceinline__ float2 fp32_pair(double x) {
  const int h = __double2hiint(x), l = __double2loint(x), sg = h & 0x80000000, e = ((h >> 20) & 0x7ff) - 896;
  if (e <= 0) return make_float2(0.f, 0.f);
  if (e >= 255) return make_float2((float)x, 0.f);
  const float rest = (float)(l & 0x1fffffff) * __int_as_float(max(e - 52, 0) << 23);   // below 2^-74: zero
  return make_float2(__int_as_float(sg | e << 23 | (h & 0xfffff) << 3 | (int)((unsigned)l >> 29)), sg ? -rest : rest);
}

// rb rows per CTA, ln lanes per entry of the new block (rb r ln <= 256); the coefficients by blocks of r rows through shared
// memory, so that a CTA splits each of them once.
constexpr int FEW_COEFS = 2048;
__global__ void __launch_bounds__(256) few_new32_kernel(TSArgs a, int rb, int ln) {
  __shared__ float4 cs[FEW_COEFS];   // (re, im), then what their FP32 values leave
  const int r = a.r, nb = a.nq + (a.mode == 1 ? 1 : 0), per = FEW_COEFS / (r * r);
  const int o = threadIdx.x / ln, q = threadIdx.x % ln, j = o % r, lr = o / r;
  const long long row = (long long)blockIdx.x * rb + lr;
  const bool in = lr < rb && row < a.N;
  float2 hi = make_float2(0.f, 0.f), lo = hi;
  for (int m0 = 0; m0 < nb; m0 += per) {
    const int n = min(per, nb - m0) * r;
    __syncthreads();
    for (int e = threadIdx.x; e < n * r; e += 256) {
      const int jj = e / n, kk = e - jj * n, k = m0 * r + kk;
      const zd c = k < a.nq * r ? (a.coefQ ? a.coefQ[(size_t)jj * a.nq * r + k] : mk<double>(0, 0))
                                : (a.coefS ? a.coefS[(size_t)jj * r + k - a.nq * r] : mk<double>(0, 0));
      const float2 re = fp32_pair(c.re), im = fp32_pair(c.im);
      cs[kk * r + jj] = make_float4(re.x, im.x, re.y, im.y);
    }
    __syncthreads();
    if (in)
      for (int m = m0; m < min(nb, m0 + per); ++m) {
        const cx<float> *x = reinterpret_cast<const cx<float> *>(m < a.nq ? a.q[m] : a.src) + (size_t)row * r;
        const float4 *c = cs + (m - m0) * r * r + j;
#pragma unroll 8
        for (int i = q; i < r; i += ln) {
          const cx<float> v = x[i];
          const float4 w = c[i * r];
          two_prod_acc(hi.x, lo.x, v.re, w.x);
          two_prod_acc(hi.x, lo.x, -v.im, w.y);
          two_prod_acc(hi.y, lo.y, v.re, w.y);
          two_prod_acc(hi.y, lo.y, v.im, w.x);
          lo.x = fmaf(v.re, w.z, fmaf(-v.im, w.w, lo.x));
          lo.y = fmaf(v.re, w.w, fmaf(v.im, w.z, lo.y));
        }
      }
  }
  for (int x = ln >> 1; x > 0; x >>= 1) {
    const float2 h = make_float2(__shfl_xor_sync(0xffffffffu, hi.x, x), __shfl_xor_sync(0xffffffffu, hi.y, x));
    lo.x += __shfl_xor_sync(0xffffffffu, lo.x, x);
    lo.y += __shfl_xor_sync(0xffffffffu, lo.y, x);
    two_sum_acc(hi.x, lo.x, h.x);
    two_sum_acc(hi.y, lo.y, h.y);
  }
  __syncthreads();
  if (in && q == 0)
    reinterpret_cast<cx<float> *>(a.out)[(size_t)row * r + j] = row < a.zero_rows ? mk<float>(0.f, 0.f) : mk<float>(hi.x + lo.x, hi.y + lo.y);
}

// TPE threads per entry, 128 per CTA.
template <typename T, int TPE>
__global__ void __launch_bounds__(128) few_gram_kernel(TSArgs a, const cx<T> *__restrict__ G) {
  __shared__ zd part[4];
  const int r = a.r, ldg = (a.gram_left + 1) * r, t = threadIdx.x % TPE;
  const int e = blockIdx.x * (128 / TPE) + threadIdx.x / TPE, j = e / ldg, row = e % ldg, m = row / r, i = row % r;
  zd s = mk<double>(0, 0);
  if (e < ldg * r) {
    const cx<T> *L = m < a.gram_left ? reinterpret_cast<const cx<T> *>(a.q[m]) : G;
    if constexpr (sizeof(T) == 8) {
#pragma unroll 4
      for (int b = t; b < (int)a.N; b += TPE) fmac_(s, L[(size_t)b * r + i], G[(size_t)b * r + j]);
    } else {
      float2 hi = make_float2(0.f, 0.f), lo = hi;
#pragma unroll 8
      for (int b = t; b < (int)a.N; b += TPE) {
        const cx<float> x = L[(size_t)b * r + i], y = G[(size_t)b * r + j];
        two_prod_acc(hi.x, lo.x, x.re, y.re);
        two_prod_acc(hi.x, lo.x, x.im, y.im);
        two_prod_acc(hi.y, lo.y, x.re, y.im);
        two_prod_acc(hi.y, lo.y, -x.im, y.re);
      }
      s = mk<double>((double)hi.x + (double)lo.x, (double)hi.y + (double)lo.y);
    }
  }
#pragma unroll
  for (int x = 16; x > 0; x >>= 1) {
    s.re += __shfl_xor_sync(0xffffffffu, s.re, x);
    s.im += __shfl_xor_sync(0xffffffffu, s.im, x);
  }
  if (TPE > 32) {
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
    __syncthreads();
    s = (part[0] + part[1]) + (part[2] + part[3]);
  }
  if (t == 0 && e < ldg * r) reinterpret_cast<zd *>(a.red)[e] = s;
}

// Up to 4096 rows and 2^20 multiply-adds per Gram, where these launches take less than the tiles' shortest:
// FP64 at n = 8, r = 4, 5 blocks: Gram 24 us as tiles and their sum, 4 here; projection and Gram 20, 8 here.  Complex64 has the same
// lines for its accuracy: tiles take 9 us for the combine of five blocks at n = 12, r = 16 (here 31, with FP64 arithmetic 89) and 6 for
// one block's Gram (13 and 21), but sum in FP32; below 2^10 rows or rank 8 these launches are the faster ones.
template <typename T> static bool launch_few(const TSArgs &a, cudaStream_t st) {
  const int g = a.gram_left + 1;
  if (!a.red || a.N > 4096 || a.N * g * a.r * a.r > (1 << 20) || a.nq + 1 > MAXB + 1) return false;
  if (a.mode == 0 ? a.out != nullptr : a.out == nullptr) return false;
  if (a.mode != 2 && !a.src) return false;
  if (a.mode != 0)
    for (int m = 0; m < a.gram_left; ++m)
      if (a.q[m] == a.out) return false;
  const cx<T> *G = reinterpret_cast<const cx<T> *>(a.mode == 0 ? a.src : a.out);
  if (a.mode != 0) {
    ::lrei::count_launch();
    if (sizeof(T) == 8) {
      const int rows = 32 / a.r;
      few_new_kernel<<<(int)((a.N + rows - 1) / rows), 256, 0, st>>>(a);
    } else {
      int rb = 1, ln = 1;   // about 256 CTAs
      while (rb * 256 < a.N && 2 * rb * a.r <= 256) rb *= 2;
      while (ln < 8 && 2 * ln * rb * a.r <= 256) ln *= 2;
      few_new32_kernel<<<(int)((a.N + rb - 1) / rb), 256, 0, st>>>(a, rb, ln);
    }
  }
  const int entries = g * a.r * a.r;
  ::lrei::count_launch();
  if (a.N <= 512) few_gram_kernel<T, 32><<<(entries + 3) / 4, 128, 0, st>>>(a, G);
  else few_gram_kernel<T, 128><<<entries, 128, 0, st>>>(a, G);
  return true;
}

int launch_ts(bool fp64, const ModelArgs &M, const TSArgs &a, int nsm, cudaStream_t st) {
  if (a.nq > MAXB || a.gram_left > a.nq || a.r < 1 || a.r > MAX_R) return -1;
  if (a.apply_h) {   // H.V by its own kernel, then a pass that only reads
    if (a.mode != 0 || !a.out || a.out == a.src) return -1;
    launch_hv(fp64, M, a.src, a.out, a.N, a.r, nsm, st, a.status);
    TSArgs b = a;
    b.src = a.out;
    b.out = nullptr;
    b.apply_h = 0;
    return launch_ts(fp64, M, b, nsm, st);
  }
  if (fp64 ? launch_few<double>(a, st) : launch_few<float>(a, st)) return 0;
  if (fp64) {
    const int n = launch_tsx(a, nsm, st);
    if (n > 0) return n;
  }
  return fp64 ? launch_ts_t<double>(a, nsm, st) : launch_ts_t<float>(a, nsm, st);
}

void launch_reduce(const double *partial, int nparts, int len_doubles, double *out, cudaStream_t st) {
  ::lrei::count_launch();
  reduce_kernel<<<(len_doubles + 15) / 16, 512, 0, st>>>(partial, nparts, len_doubles, out);
}

void launch_hv(bool fp64, const ModelArgs &M, const void *X, void *Y, long long N, int r, int nsm, cudaStream_t st,
               int *status) {
  if (launch_hv_tiled(fp64, M, X, Y, N, r, nsm, st, status)) return;
  // rows that are not a multiple of 16 bytes, blocks that do not start on one, or fewer than 16 rows: the per-row gather
  auto grid_for = [&](int cpt) {
    long long total = N * (r / cpt);
    long long g = (total + 255) / 256;
    long long cap = (long long)nsm * 16;
    return (int)(g < cap ? g : cap);
  };
  if (fp64) {
    using T = double;
    if (r % 2 == 0) { ::lrei::count_launch(); hv_kernel<T, 2><<<grid_for(2), 256, 0, st>>>(M, (const cx<T> *)X, (cx<T> *)Y, N, r); }
    else { ::lrei::count_launch(); hv_kernel<T, 1><<<grid_for(1), 256, 0, st>>>(M, (const cx<T> *)X, (cx<T> *)Y, N, r); }
  } else {
    using T = float;
    if (r % 4 == 0 && aligned16(X)) { ::lrei::count_launch(); hv_kernel<T, 4><<<grid_for(4), 256, 0, st>>>(M, (const cx<T> *)X, (cx<T> *)Y, N, r); }
    else if (r % 2 == 0 && aligned16(X)) { ::lrei::count_launch(); hv_kernel<T, 2><<<grid_for(2), 256, 0, st>>>(M, (const cx<T> *)X, (cx<T> *)Y, N, r); }
    else { ::lrei::count_launch(); hv_kernel<T, 1><<<grid_for(1), 256, 0, st>>>(M, (const cx<T> *)X, (cx<T> *)Y, N, r); }
  }
}

// ------------------------------------------------------ observables
// Row b of M_x V and M_y V: (1/n) sum over spins q of (1/2) V[b ^ 2^q] and
// (1/2)(bit_q(b) ? +i : -i) V[b ^ 2^q] (sigma_y with bit 0 = spin up).
constexpr int OBS_BLOCKS = 6;

template <typename T>
__global__ void __launch_bounds__(256) obs_kernel(const __grid_constant__ ModelArgs M, const cx<T> *__restrict__ V, long long N, int r,
                                                  int tr, double *partial) {
  extern __shared__ __align__(16) unsigned char smem[];
  cx<T> *vs = reinterpret_cast<cx<T> *>(smem);   // tr x r
  cx<T> *ss = vs + (size_t)tr * r;                // H V
  cx<T> *xs = ss + (size_t)tr * r;                // Mx V
  cx<T> *ys = xs + (size_t)tr * r;                // My V
  cx<T> *zs = ys + (size_t)tr * r;                // Mz V
  double *acc = reinterpret_cast<double *>(zs + (size_t)tr * r);
  const int tid = threadIdx.x, nt = blockDim.x;
  const int nent = OBS_BLOCKS * r * r;
  for (int e = tid; e < nent * 2; e += nt) acc[e] = 0.0;
  __syncthreads();
  const T inv_n = (T)(1.0 / M.n);
  const long long ntiles = (N + tr - 1) / tr;
  for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const long long row0 = tile * tr;
    const int rows = (int)((N - row0) < tr ? (N - row0) : tr);
    for (int e = tid; e < tr * r; e += nt) {
      const int lr = e / r, c = e % r;
      cx<T> v = mk<T>(0, 0), s = v, x = v, y = v, z = v;
      if (lr < rows) {
        const uint32_t b = (uint32_t)(row0 + lr);
        cx<T> o[1];
        hv_group<T, 1>(M, V, r, b, c, o);
        s = o[0];
        v = ldg1(V + (size_t)b * r + c);
        for (int q = 0; q < M.n; ++q) {
          const cx<T> p = ldg1(V + (size_t)(b ^ (1u << q)) * r + c);
          x = x + p;
          // (sigma_y)_{0,1} = -i, (sigma_y)_{1,0} = +i
          if ((b >> q) & 1u) y = y + mk<T>(-p.im, p.re);
          else y = y + mk<T>(p.im, -p.re);
        }
        x = ((T)0.5 * inv_n) * x;
        y = ((T)0.5 * inv_n) * y;
        z = ((T)((0.5 * M.n - (double)__popc(b)) / M.n)) * v;
      }
      vs[e] = v; ss[e] = s; xs[e] = x; ys[e] = y; zs[e] = z;
    }
    __syncthreads();
    for (int e = tid; e < nent; e += nt) {
      const int blk = e / (r * r), j = (e / r) % r, i = e % r;
      const cx<T> *L = (blk == 1) ? ss : vs;
      const cx<T> *R = blk == 0 ? ss : blk == 1 ? ss : blk == 2 ? vs : blk == 3 ? xs : blk == 4 ? ys : zs;
      cx<T> s = mk<T>(0, 0);
      for (int lr = 0; lr < tr; ++lr) fmac_(s, L[lr * r + i], R[lr * r + j]);
      Acc<T>::add(acc, e, s);
    }
    __syncthreads();
  }
  double *outp = partial + (size_t)blockIdx.x * nent * 2;
  for (int e = tid; e < nent; e += nt) {
    cx<double> v = Acc<T>::get(acc, e);
    outp[2 * e] = v.re;
    outp[2 * e + 1] = v.im;
  }
}

int launch_obs(bool fp64, const ModelArgs &M, const void *V, long long N, int r, double *partial, int nsm,
               cudaStream_t st) {
  const int tr = 16;
  const long long ntiles = (N + tr - 1) / tr;
  int grid = (int)(ntiles < (long long)ts_max_grid(nsm) ? ntiles : ts_max_grid(nsm));
  if (grid < 1) grid = 1;
  const size_t nent = (size_t)OBS_BLOCKS * r * r;
  if (fp64) {
    size_t bytes = 5 * (size_t)tr * r * sizeof(cx<double>) + nent * 16;
    ::lrei::count_launch(); obs_kernel<double><<<grid, 256, bytes, st>>>(M, (const cx<double> *)V, N, r, tr, partial);
  } else {
    size_t bytes = 5 * (size_t)tr * r * sizeof(cx<float>) + nent * 16;
    ::lrei::count_launch(); obs_kernel<float><<<grid, 256, bytes, st>>>(M, (const cx<float> *)V, N, r, tr, partial);
  }
  return grid;
}


// Same pass with the number of partial sums capped (used by the allocation-free observables).
int launch_obs_capped(bool fp64, const ModelArgs &M, const void *V, long long N, int r, double *partial,
                      int max_grid, cudaStream_t st) {
  const int tr = 16;
  const long long ntiles = (N + tr - 1) / tr;
  int grid = (int)(ntiles < (long long)max_grid ? ntiles : max_grid);
  if (grid < 1) grid = 1;
  const size_t nent = (size_t)OBS_BLOCKS * r * r;
  if (fp64) {
    size_t bytes = 5 * (size_t)tr * r * sizeof(cx<double>) + nent * 16;
    ::lrei::count_launch(); obs_kernel<double><<<grid, 256, bytes, st>>>(M, (const cx<double> *)V, N, r, tr, partial);
  } else {
    size_t bytes = 5 * (size_t)tr * r * sizeof(cx<float>) + nent * 16;
    ::lrei::count_launch(); obs_kernel<float><<<grid, 256, bytes, st>>>(M, (const cx<float> *)V, N, r, tr, partial);
  }
  return grid;
}


// ------------------------------------------------------ conversion / checks
template <typename S, typename D>
__global__ void convert_kernel(const cx<S> *src, int ld, cx<D> *dst, long long N, int r) {
  const long long total = N * r;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const long long b = e / r;
    const int c = (int)(e % r);
    const cx<S> v = src[b * ld + c];
    dst[e] = mk<D>((D)v.re, (D)v.im);
  }
}

void launch_convert(const void *src, int src_c64, int ld, void *dst, int dst_fp64, long long N, int r,
                    cudaStream_t st) {
  long long total = N * r;
  int grid = (int)((total + 255) / 256 < 4096 ? (total + 255) / 256 : 4096);
  if (grid < 1) grid = 1;
  if (src_c64) {
    if (dst_fp64) { ::lrei::count_launch(); convert_kernel<float, double><<<grid, 256, 0, st>>>((const cx<float> *)src, ld, (cx<double> *)dst, N, r); }
    else { ::lrei::count_launch(); convert_kernel<float, float><<<grid, 256, 0, st>>>((const cx<float> *)src, ld, (cx<float> *)dst, N, r); }
  } else {
    if (dst_fp64) { ::lrei::count_launch(); convert_kernel<double, double><<<grid, 256, 0, st>>>((const cx<double> *)src, ld, (cx<double> *)dst, N, r); }
    else { ::lrei::count_launch(); convert_kernel<double, float><<<grid, 256, 0, st>>>((const cx<double> *)src, ld, (cx<float> *)dst, N, r); }
  }
}

template <typename T>
__global__ void finite_kernel(const T *x, long long n, int *status) {
  bool bad = false;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x)
    if (!isfinite(x[e])) bad = true;
  if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(status, ST_NONFINITE);
}

void launch_check_finite(bool fp64, const void *X, long long N, int r, int *status, cudaStream_t st) {
  long long n = N * r * 2;
  int grid = (int)((n + 255) / 256 < 1024 ? (n + 255) / 256 : 1024);
  if (grid < 1) grid = 1;
  if (fp64) { ::lrei::count_launch(); finite_kernel<double><<<grid, 256, 0, st>>>((const double *)X, n, status); }
  else { ::lrei::count_launch(); finite_kernel<float><<<grid, 256, 0, st>>>((const float *)X, n, status); }
}

}  // namespace lrei

namespace lrei {
// Raise the dynamic shared-memory limit of every tile kernel once (outside any stream capture).
int ts_init() {
  if (hv_tiled_init() || tsx_init()) return -1;
  const int lim = 210 * 1024;
  cudaError_t e = cudaSuccess;
  auto set = [&](const void *f) {
    cudaError_t x = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    if (x != cudaSuccess) e = x;
  };
  auto set3 = [&](const void *f) {
    cudaError_t x = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    if (x != cudaSuccess) e = x;
  };
  for (int g = 1; g <= 8; ++g)
    for (int v = 0; v < 4; ++v)
      for (int R = 8; R <= 32; R *= 2)
        for (int tr = R == 8 ? 64 : 32; tr <= 64; tr *= 2) set3((const void *)ts3_pick(R, tr, g, v & 1, v & 2));
  set((const void *)ts_kernel<double, 2>);
  set((const void *)ts_kernel<double, 1>);
  set((const void *)ts_kernel<float, 4>);
  set((const void *)ts_kernel<float, 2>);
  set((const void *)ts_kernel<float, 1>);
  set((const void *)ts2_kernel<double, 2, 1>);
  set((const void *)ts2_kernel<double, 1, 1>);
  set((const void *)ts2_kernel<double, 2, 2>);
  set((const void *)ts2_kernel<double, 1, 2>);
  set((const void *)ts2_kernel<float, 4, 1>);
  set((const void *)ts2_kernel<float, 2, 1>);
  set((const void *)ts2_kernel<float, 1, 1>);
  set((const void *)ts2_kernel<float, 4, 2>);
  set((const void *)ts2_kernel<float, 2, 2>);
  set((const void *)ts2_kernel<float, 1, 2>);
  set((const void *)obs_kernel<double>);
  set((const void *)obs_kernel<float>);
  return e == cudaSuccess ? 0 : -1;
}
}  // namespace lrei
