// Small dense complex linear algebra for the r x r / k x k part of the LREI step.
//
// These solves are FP64 in every precision mode.  GB300 executes FP64 at a
// small fraction of its FP32 rate per SM, so every kernel here spreads its
// FP64 work over many small CTAs (a warp per output entry or per column)
// instead of running on one SM.  The one exception is the cyclic Jacobi
// eigensolver, which runs in one CTA: the k x k eigenproblem of each stage
// is solved in FP32 and then corrected to FP64 accuracy on its top-r
// invariant subspace (sm_eig_topr), so only r x r Jacobi runs in FP64.
#include "small.cuh"
#include "small_dev.cuh"

#include <algorithm>

namespace lrei {

// [0] FP32 Jacobi calls, [1] FP32 sweeps, [2] FP64 Jacobi calls, [3] FP64 sweeps (diagnostics)
__device__ unsigned long long g_jacobi_counters[4];

__device__ __forceinline__ zd warp_sum(zd v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    v.re += __shfl_xor_sync(0xffffffffu, v.re, o);
    v.im += __shfl_xor_sync(0xffffffffu, v.im, o);
  }
  return v;
}

// State of an eigensolve on the device: [META_ROUNDS] rounds of its FP32 Jacobi, [META_D + p - 1] largest component of the p-th
// Newton correction (float bits).
enum { META_ROUNDS = 0, META_D = 1, META_INTS = 8 };
constexpr int NEWTON_PASSES = 4;
// Whether the corrections up to pass p (1-based) leave nothing to correct: they shrink by a constant factor per pass
// (the FP32 error of Ur), so after pass q about D_q^2 / D_{q-1} is left.
__device__ __forceinline__ bool newton_done(const int *meta, int p) {
  for (int q = 2; q <= p; ++q) {
    const float d = __int_as_float(meta[META_D + q - 1]);
    if (d * d <= 1e-17f * __int_as_float(meta[META_D + q - 2])) return true;
  }
  return false;
}

// ------------------------------------------------------------------ GEMM
__device__ __forceinline__ zd opget(char op, const zd *A, int ld, int i, int p) {
  return op == 'N' ? A[(size_t)p * ld + i] : conj(A[(size_t)i * ld + p]);
}

// One output per LN lanes of a warp: each lane sums every LN-th term, the lanes are combined by shuffles.  An FP64
// instruction takes a scheduler 64 cycles here whatever the number of active lanes (measured, also in a dependent
// chain), so a sum of K terms by one thread is a chain of 4 K x 64 cycles and by LN lanes of 4 K / LN + 2 log2 LN.
template <int LN>
__global__ void __launch_bounds__(128) gemm_kernel(char opA, char opB, int M, int N, int K, zd alpha, const zd *__restrict__ A,
                                                   int lda, const zd *__restrict__ B, int ldb, zd beta, const zd *Cin,
                                                   int ldin, zd *C, int ldc, int herm, const int *meta, int pass) {
  if (meta && newton_done(meta, pass)) return;
  const int w = (blockIdx.x * blockDim.x + threadIdx.x) / LN, lane = threadIdx.x % LN;
  int i, j;
  bool in;
  if (herm) {   // the upper triangle (i <= j) and its mirror; column j holds the outputs j (j + 1) / 2 + i
    in = w < M * (M + 1) / 2;
    j = in ? (int)((sqrtf(8.f * (float)w + 1.f) - 1.f) * 0.5f) : 0;
    while ((j + 1) * (j + 2) / 2 <= w && in) ++j;
    while (j * (j + 1) / 2 > w) --j;
    i = in ? w - j * (j + 1) / 2 : 0;
  } else {
    in = w < M * N;
    i = in ? w % M : 0;
    j = in ? w / M : 0;
  }
  zd s = mk<double>(0, 0);
  for (int p = lane; p < K; p += LN) fma_(s, opget(opA, A, lda, i, p), opget(opB, B, ldb, p, j));
#pragma unroll
  for (int o = LN / 2; o > 0; o >>= 1) {
    s.re += __shfl_xor_sync(0xffffffffu, s.re, o);
    s.im += __shfl_xor_sync(0xffffffffu, s.im, o);
  }
  if (in && lane == 0) {
    zd c = alpha * s;
    if (beta.re != 0.0 || beta.im != 0.0) c = c + beta * Cin[(size_t)j * ldin + i];
    if (herm && i == j) c.im = 0.0;
    C[(size_t)j * ldc + i] = c;
    if (herm && i != j) C[(size_t)i * ldc + j] = conj(c);
  }
}

// Lanes per output: the least of the longest chain (its FP64 instructions at 64 cycles) and the SMs' throughput (one
// FP64 warp instruction in 19 cycles and SM, over 152 SMs).  Measured over an RK4 step at n = 16, r = 8 (K = 8..72):
// 8.7 us a launch with one thread per output, 4.3 with the lanes chosen here; the step 1.58 ms before, 1.40 after.
static int gemm_lanes(double outputs, int K) {
  int best = 4;
  double cost = 1e300;
  for (int ln = 4, lg = 2; ln <= 32; ln *= 2, ++lg) {
    const double instr = 4.0 * ((K + ln - 1) / ln) + 2.0 * lg + 4.0;
    const double warps = outputs * ln / 32.0;
    const double c = std::max(64.0 * instr, warps * instr * 19.0 / 152.0);
    if (c < cost) {
      cost = c;
      best = ln;
    }
  }
  return best;
}

static void gemm_launch(char opA, char opB, int M, int N, int K, zd alpha, const zd *A, int lda, const zd *B, int ldb,
                        zd beta, const zd *Cin, int ldin, zd *C, int ldc, int herm, cudaStream_t st,
                        const int *meta = nullptr, int pass = 0) {
  if (M <= 0 || N <= 0) return;
  const int outputs = herm ? M * (M + 1) / 2 : M * N;
  const int ln = gemm_lanes(outputs, K);
  const int grid = (int)(((long long)outputs * ln + 127) / 128);
  ::lrei::count_launch();
  auto go = [&](auto kern) {
    kern<<<grid, 128, 0, st>>>(opA, opB, M, N, K, alpha, A, lda, B, ldb, beta, Cin, ldin, C, ldc, herm, meta, pass);
  };
  if (ln == 4) go(gemm_kernel<4>);
  else if (ln == 8) go(gemm_kernel<8>);
  else if (ln == 16) go(gemm_kernel<16>);
  else go(gemm_kernel<32>);
}

void sm_gemm(char opA, char opB, int M, int N, int K, zd alpha, const zd *A, int lda, const zd *B, int ldb, zd beta,
             zd *C, int ldc, cudaStream_t st) {
  gemm_launch(opA, opB, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, C, ldc, 0, st);
}

void sm_gemm_herm(char opA, char opB, int M, int K, zd alpha, const zd *A, int lda, const zd *B, int ldb, zd beta,
                  const zd *Cin, int ldin, zd *C, int ldc, cudaStream_t st) {
  gemm_launch(opA, opB, M, M, K, alpha, A, lda, B, ldb, beta, Cin, ldin, C, ldc, 1, st);
}

// ------------------------------------------------------- triangular solves
// Triangular solves (k <= MAX_R), one warp per right-hand side, four warps per CTA sharing one copy of the
// triangle in shared memory.  Right-looking: x_j = b_j / d_j is broadcast from shared memory and
// every lane updates the rows it owns, so the loop has no reductions and no divisions (the
// reciprocal diagonal is precomputed).
__global__ void __launch_bounds__(128) trsv_kernel(char op, const zd *__restrict__ L, int ldl, int k,
                                                   zd *__restrict__ B, int ldb, int ncols) {
  extern __shared__ zd trsv_sm[];
  zd *Ts = trsv_sm;                                  // k x k: Ts[j*k + i] = multiplier of x_j in row i
  zd *xs = trsv_sm + (size_t)k * k;                  // 4 warps x k
  double *rd = reinterpret_cast<double *>(xs + 4 * k);   // k reciprocal diagonal entries
  const int t = threadIdx.x, lane = t & 31, wp = t >> 5;
  for (int i = t; i < k; i += blockDim.x) {
    const double d = L[(size_t)i * ldl + i].re;
    rd[i] = d != 0.0 ? 1.0 / d : 0.0;
  }
  for (int e = t; e < k * k; e += blockDim.x) {
    const int i = e % k, j = e / k;
    zd v = mk<double>(0, 0);
    if (op == 'N') { if (i > j) v = L[(size_t)j * ldl + i]; }          // L(i, j)
    else { if (i < j) v = conj(L[(size_t)i * ldl + j]); }               // (L^H)(i, j) = conj(L(j, i))
    Ts[e] = v;
  }
  const int col = blockIdx.x * 4 + wp;
  zd *x = xs + wp * k;
  zd *bcol = B + (size_t)col * ldb;
  if (col < ncols)
    for (int i = lane; i < k; i += 32) x[i] = bcol[i];
  __syncthreads();
  if (col < ncols) {
    if (op == 'N') {
      for (int j = 0; j < k; ++j) {
        __syncwarp();
        const zd xj = mk<double>(x[j].re * rd[j], x[j].im * rd[j]);
        __syncwarp();
        if (lane == 0) x[j] = xj;
        for (int i = j + 1 + lane; i < k; i += 32) x[i] = x[i] - Ts[j * k + i] * xj;
      }
    } else {
      for (int j = k - 1; j >= 0; --j) {
        __syncwarp();
        const zd xj = mk<double>(x[j].re * rd[j], x[j].im * rd[j]);
        __syncwarp();
        if (lane == 0) x[j] = xj;
        for (int i = lane; i < j; i += 32) x[i] = x[i] - Ts[j * k + i] * xj;
      }
    }
    __syncwarp();
    for (int i = lane; i < k; i += 32) bcol[i] = x[i];
  }
}

void sm_trsv(char op, const zd *L, int ldl, int k, zd *B, int ldb, int ncols, cudaStream_t st) {
  if (ncols <= 0 || k <= 0) return;
  const size_t bytes = ((size_t)k * k + 4 * (size_t)k) * sizeof(zd) + (size_t)k * 8;
  ::lrei::count_launch();
  trsv_kernel<<<(ncols + 3) / 4, 128, bytes, st>>>(op, L, ldl, k, B, ldb, ncols);
}

// ------------------------------------------------------------- Cholesky
// Cholesky A = L L^H of a Hermitian k x k matrix (k <= 64) and the inverse of L, in one CTA: Gaussian elimination on
// [A | I] (eliminate), and the columns are scaled by A_jj^{-1/2} at the end.  The inverse rides along in the chain of the
// steps (a triangular solve of its own took 24 us at k = 16).
// The elimination multiplies two entries before it divides by the pivot, so when a diagonal entry is beyond 2^+-400 the columns are
// scaled by powers of two to a diagonal in [1, 4) first (an unusual unit of energy: the Gram of H V has its square).
// Column j is dead when its pivot is not above tol times a reference: the j-th diagonal entry of `ref` when given (the
// squared norm of the raw column), else the largest diagonal entry of A.  A dead column gets L[j][j] = 1 and a zero
// sub-column (and, with zero_row, a zero row).
__global__ void __launch_bounds__(512) chol_kernel(const zd *__restrict__ A, int lda, int k, zd *__restrict__ Lout, int ldl,
                                                   zd *__restrict__ Iout, int ldi, int inv_h, zd *__restrict__ Rc, int ldrc, double tol,
                                                   int zero_row, int *dead, int *status, int flag_rank,
                                                   const zd *__restrict__ ref, int ldref) {
  extern __shared__ zd Ls[];   // k x k: A's lower triangle, then L before scaling; and k x k: the inverse before scaling
  zd *X = Ls + (size_t)k * k;
  __shared__ double rs[64], tolref[64], inv[64], scale[64];
  __shared__ int deads[64];
  const int t = threadIdx.x, nt = blockDim.x;
  // the diagonal's high words (k <= 64), the same in every warp
  const int i0 = t & 31, i1 = i0 + 32;
  const int h0 = i0 < k ? __double2hiint(A[(size_t)i0 * lda + i0].re) : 0, h1 = i1 < k ? __double2hiint(A[(size_t)i1 * lda + i1].re) : 0;
  for (int e = t; e < k * k; e += nt) {
    const int i = e % k, j = e / k;
    Ls[e] = (i >= j) ? A[(size_t)j * lda + i] : mk<double>(0, 0);
    X[e] = mk<double>(i == j ? 1.0 : 0.0, 0);
  }
  auto exponent = [](int hi) { return (hi >> 20) - 1023; };
  auto usable = [&](int hi) { return hi > 0 && exponent(hi) < 1024; };   // positive and finite
  const bool far = __any_sync(0xffffffffu, (usable(h0) && abs(exponent(h0)) > 400) || (usable(h1) && abs(exponent(h1)) > 400));
  if (far) {
    auto factor = [&](int hi) { return __hiloint2double((1023 - (usable(hi) ? exponent(hi) >> 1 : 0)) << 20, 0); };
    if (t < 32 && i0 < k) scale[i0] = factor(h0);
    if (t < 32 && i1 < k) scale[i1] = factor(h1);
    __syncthreads();
    for (int e = t; e < k * k; e += nt) {
      const double si = scale[e % k], sj = scale[e / k];
      Ls[e] = mk<double>(Ls[e].re * si * sj, Ls[e].im * si * sj);
    }
  }
  if (t < 32) {
    double m = 0.0;
    if (!ref) {
      for (int i = t; i < k; i += 32) m = fmax(m, A[(size_t)i * lda + i].re);
      // not negative: ordered as integers, which run at full rate
      unsigned long long b = __double_as_longlong(m);
      for (int o = 16; o > 0; o >>= 1) b = max(b, __shfl_xor_sync(0xffffffffu, b, o));
      m = __longlong_as_double(b);
    }
    for (int i = t; i < k; i += 32) {
      const double r = ref ? ref[(size_t)i * ldref + i].re : m;
      tolref[i] = r > 0.0 ? tol * r : __longlong_as_double(0x7ff0000000000000ll);   // no positive reference: dead
      if (far) tolref[i] = tolref[i] * scale[i] * scale[i];
    }
  }
  __syncthreads();
  eliminate(Ls, X, k, tolref, inv, deads);
  for (int j = t; j < k; j += nt) rs[j] = deads[j] ? 1.0 : newton_rsqrt(Ls[j * k + j].re);
  __syncthreads();
  for (int e = t; e < k * k; e += nt) {
    const int i = e % k, j = e / k;
    const bool row0 = zero_row && deads[i];   // a dead row without its part left of the diagonal
    zd l = mk<double>(0, 0);
    if (i > j) {
      if (!deads[j] && !row0) l = mk<double>(Ls[e].re * rs[j], Ls[e].im * rs[j]);
    } else if (i == j) {
      l.re = deads[j] ? 1.0 : Ls[e].re * rs[j];
    }
    if (far && !(i == j && deads[j])) l = (1.0 / scale[i]) * l;
    if (Lout) Lout[(size_t)j * ldl + i] = l;
    if (Iout) {
      zd x = mk<double>(0, 0);
      if (i > j && !row0) x = mk<double>(X[e].re * rs[i], X[e].im * rs[i]);
      else if (i == j) x.re = rs[i];
      if (far) x = deads[i] ? (scale[j] / scale[i]) * x : scale[j] * x;
      if (inv_h) Iout[(size_t)i * ldi + j] = conj(x);
      else Iout[(size_t)j * ldi + i] = x;
    }
    // Rc = L^H with the rows of dead columns zeroed: entry (j, i)
    if (Rc) Rc[(size_t)i * ldrc + j] = deads[j] ? mk<double>(0, 0) : conj(l);
  }
  if (dead)
    for (int j = t; j < k; j += nt) dead[j] = deads[j];
  if (flag_rank && status)
    for (int j = t; j < k; j += nt)
      if (deads[j]) atomicOr(status, ST_RANK);
}

void sm_chol(const zd *A, int lda, int k, zd *L, int ldl, double tol, int zero_row, int *dead, int *status,
             int flag_rank, cudaStream_t st, const zd *ref, int ldref, zd *Linv, int ldi, int inv_h, zd *Rc, int ldrc) {
  ::lrei::count_launch();
  chol_kernel<<<1, eliminate_threads(k), 2 * (size_t)k * k * sizeof(zd), st>>>(A, lda, k, L, ldl, Linv, ldi, inv_h, Rc, ldrc, tol, zero_row, dead,
                                                              status, flag_rank, ref, ldref);
}

// --------------------------------------------------------------- Jacobi
// Cyclic Jacobi of a Hermitian matrix in one CTA, round-robin pairs (circle method: position 0 stays, positions
// 1 .. kp-1 rotate by one per round).  A rotation J = [[c, s], [-conj(s), c]] on (p, q) annihilates A_pq; a round applies the kp / 2
// disjoint rotations of its pairs as A <- J^H A J on 2 x 2 blocks of pairs.  Only the upper triangle is kept
// (an element below the diagonal is its mirror's conjugate), so a round touches each pair of pairs once.
__device__ __forceinline__ void round_pair(int pos, int round, int kp, int *p, int *q) {
  auto player = [&](int x) {
    if (x == 0) return 0;
    int y = x - 1 + round;
    if (y >= kp - 1) y -= kp - 1;
    return y + 1;
  };
  const int a = player(pos), b = player(kp - 1 - pos);
  *p = min(a, b);
  *q = max(a, b);
}
// item e of the pairs of positions a < b, e = b (b - 1) / 2 + a; with diag = 1 of a <= b, e = b (b + 1) / 2 + a
__device__ __forceinline__ void tri_item(int e, int *a, int *b, int diag = 0) {
  int y = (int)((sqrtf(8.f * (float)e + 1.f) + 1.f) * 0.5f);
  while (y * (y + 1) / 2 <= e) ++y;
  while (y * (y - 1) / 2 > e) --y;
  *b = y - diag;
  *a = e - y * (y - 1) / 2;
}

constexpr int J32_SWEEPS = 12;
constexpr int J32_KMAX = 162;

// The storage is by position in the tournament, not by row: pair a of every round is the positions (a, kp - 1 - a), and a
// round writes its results where the next one reads them: position x moves to x - 1 (1 to kp - 1, 0 stays), so
// all addresses are the same in every round, and after a sweep (kp - 1 rounds) every row is back in its place.
__device__ __forceinline__ int next_pos(int x, int kp) { return x == 0 ? 0 : (x == 1 ? kp - 1 : x - 1); }
__device__ __forceinline__ int tri_at(int x, int y) { return (y * (y + 1) >> 1) + x; }   // x <= y

// FP32.  A round is a chain of instructions in few warps: the pairs' angles, a barrier, the 2 x 2 blocks of pairs a <= b
// (one thread each, the addresses of its first J32_OWN blocks in registers), a barrier.  The matrix is read from one
// buffer and written to the other.  The eigenvectors are not accumulated here: the rotations (c, s) of every round go
// to rots, and replay_kernel applies them to the rows of U on many SMs.  order[i]: rank of diagonal entry i in decreasing order.
// A round takes 0.35 us at k = 16, 0.53 at k = 40, 0.92 at k = 80, 4.0 at k = 160; by row indices and in place 0.65 at k = 40.
// (Four threads per block, an entry each: 0.38, 0.53 at k = 40, 0.97 at k = 64 against 0.77; the angles by every block's
// thread, without the first barrier: 0.9 at k = 16.)
constexpr int J32_OWN = 2;
__global__ void __launch_bounds__(512) jacobi32_kernel(const zd *__restrict__ Ain, int lda, int k, double *__restrict__ wout,
                                                       int *__restrict__ order, float4 *__restrict__ rots,
                                                       int *__restrict__ meta, float tol) {
  extern __shared__ __align__(16) unsigned char sm[];
  const int kp = k + (k & 1), np = kp / 2, nitem = np * (np + 1) / 2, ntri = kp * (kp + 1) / 2;
  cx<float> *A = reinterpret_cast<cx<float> *>(sm), *B = A + ntri;    // upper triangles: read, written
  __shared__ float red[2][32];
  __shared__ float4 rot[J32_KMAX / 2];
  const int t = threadIdx.x, nt = blockDim.x, lane = t & 31, wp = t >> 5;
  for (int j = wp; j < kp; j += nt / 32)
    for (int i = lane; i <= j; i += 32) A[tri_at(i, j)] = j < k ? cvt<float>(Ain[(size_t)j * lda + i]) : mk<float>(0.f, 0.f);
  // where entry (x, y), x <= y, goes; the sign bit: conjugated
  auto dst = [&](int x, int y) {
    const int u = next_pos(x, kp), v = next_pos(y, kp);
    return u <= v ? tri_at(u, v) : (int)(tri_at(v, u) | 0x80000000);
  };
  struct Block {
    int a, b, w[4];   // where the entries (pa, pb), (pa, qb), (pb, qa), (qb, qa) go
  };
  auto make_block = [&](int e) {
    Block I;
    tri_item(e < nitem ? e : 0, &I.a, &I.b, 1);
    const int qa = kp - 1 - I.a, qb = kp - 1 - I.b;
    I.w[0] = dst(I.a, I.b);
    I.w[1] = dst(I.a, qb);
    I.w[2] = dst(I.b, qa);
    I.w[3] = dst(qb, qa);
    return I;
  };
  Block own[J32_OWN];
#pragma unroll
  for (int x = 0; x < J32_OWN; ++x) own[x] = make_block(t + x * nt);
  int p1 = 0, p2 = 0, p3 = 0;      // pair t: A_pp, A_qq, A_pq
  if (t < np) {
    p1 = tri_at(t, t);
    p2 = tri_at(kp - 1 - t, kp - 1 - t);
    p3 = tri_at(t, kp - 1 - t);
  }
  if (t < META_INTS) meta[t] = 0;
  __syncthreads();
  auto put = [&](int i, cx<float> v) {
    if (i < 0) v.im = -v.im;
    B[i & 0x7fffffff] = v;
  };
  int rounds = 0, sweeps = 0;
  for (; sweeps < J32_SWEEPS; ++sweeps) {
    // convergence test: off-diagonal vs total Frobenius norm
    float off = 0.f, tot = 0.f;
    for (int j = wp; j < kp; j += nt / 32)
      for (int i = lane; i <= j; i += 32) {
        const float v = norm2(A[tri_at(i, j)]);
        if (i == j) tot += v;
        else off += 2.f * v;
      }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      off += __shfl_xor_sync(0xffffffffu, off, o);
      tot += __shfl_xor_sync(0xffffffffu, tot, o);
    }
    if (lane == 0) { red[0][wp] = off; red[1][wp] = tot; }
    __syncthreads();
    off = lane < nt / 32 ? red[0][lane] : 0.f;
    tot = lane < nt / 32 ? red[1][lane] : 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      off += __shfl_xor_sync(0xffffffffu, off, o);
      tot += __shfl_xor_sync(0xffffffffu, tot, o);
    }
    tot += off;
    if (off <= tol * tol * tot || !(tot == tot)) break;
    for (int round = 0; round < kp - 1; ++round, ++rounds) {
      if (t < np) {   // tan = f |b|, f = sign(d - a) / (|h| + sqrt(h^2 + |b|^2)), h = (d - a) / 2
        const cx<float> b = A[p3];
        const float n2 = norm2(b), h = 0.5f * (A[p2].re - A[p1].re), g = fmaxf(fmaf(h, h, n2), 1e-37f);
        const float f = n2 > 1e-37f ? copysignf(__fdividef(1.f, fabsf(h) + g * rsqrtf(g)), h) : 0.f;
        const float c = rsqrtf(fmaf(n2 * f, f, 1.f)), cf = c * f;
        const float4 R = make_float4(c, cf * b.re, cf * b.im, f * n2);
        rot[t] = R;
        rots[(size_t)rounds * np + t] = R;
      }
      __syncthreads();
      auto block = [&](const Block &I) {
        const int pa = I.a, qa = kp - 1 - I.a, pb = I.b, qb = kp - 1 - I.b;
        const float4 Ra = rot[pa], Rb = rot[pb];
        if (pa == pb) {
          put(I.w[0], mk<float>(A[tri_at(pa, pa)].re - Ra.w, 0.f));
          put(I.w[1], mk<float>(0.f, 0.f));
          put(I.w[3], mk<float>(A[tri_at(qa, qa)].re + Ra.w, 0.f));
          return;
        }
        const cx<float> x00 = A[tri_at(pa, pb)], x01 = A[tri_at(pa, qb)], x10 = conj(A[tri_at(pb, qa)]), x11 = conj(A[tri_at(qb, qa)]);
        const cx<float> sa = mk<float>(Ra.y, Ra.z), sb = mk<float>(Rb.y, Rb.z);
        const cx<float> y00 = Rb.x * x00 - conj(sb) * x01, y01 = sb * x00 + Rb.x * x01;    // Y = X J_b
        const cx<float> y10 = Rb.x * x10 - conj(sb) * x11, y11 = sb * x10 + Rb.x * x11;
        put(I.w[0], Ra.x * y00 - sa * y10);                                                // X' = J_a^H Y
        put(I.w[1], Ra.x * y01 - sa * y11);
        put(I.w[2], conj(conj(sa) * y00 + Ra.x * y10));
        put(I.w[3], conj(conj(sa) * y01 + Ra.x * y11));
      };
#pragma unroll
      for (int x = 0; x < J32_OWN; ++x)
        if (t + x * nt < nitem) block(own[x]);
      for (int e = t + J32_OWN * nt; e < nitem; e += nt) block(make_block(e));
      __syncthreads();
      cx<float> *x = A;
      A = B;
      B = x;
    }
  }
  // eigenvalues and their order (decreasing, ties by index)
  for (int i = t; i < k; i += nt) {
    const float wi = A[tri_at(i, i)].re;
    int rank = 0;
    for (int j = 0; j < k; ++j) {
      const float wj = A[tri_at(j, j)].re;
      rank += (wj > wi) || (wj == wi && j < i);
    }
    wout[rank] = (double)wi;
    order[i] = rank;
  }
  if (t == 0) {
    meta[META_ROUNDS] = rounds;
    atomicAdd(&g_jacobi_counters[0], 1ull);
    atomicAdd(&g_jacobi_counters[1], (unsigned long long)sweeps);
  }
}

// U = J_1 J_2 ... applied to the rows of the identity (a row sees every rotation, and no other row): one warp per row, eight
// rows per CTA, the rotations of REPLAY rounds at a time through shared memory.  The row is in registers by position
// as above: lane holds the pairs a = PPL lane + 0 .. PPL - 1, i.e. positions a and kp - 1 - a, and a round ends with the
// move of every position by one.  Writes U with its columns in decreasing order of eigenvalue: all of them in FP32, the
// first nout also in FP64.  (Row in shared memory: 0.28 us a round at k = 80.)
constexpr int REPLAY = 16;
template <int PPL>
__global__ void __launch_bounds__(256) replay_kernel(int k, const float4 *__restrict__ rots, const int *__restrict__ meta,
                                                     const int *__restrict__ order, cx<float> *__restrict__ Uf,
                                                     zd *__restrict__ Uout, int ldu, int nout) {
  extern __shared__ __align__(16) unsigned char sm[];
  const int kp = k + (k & 1), np = kp / 2;
  float4 *R = reinterpret_cast<float4 *>(sm);                       // [REPLAY][np]
  const int t = threadIdx.x, lane = t & 31, wp = t >> 5, row = blockIdx.x * 8 + wp, a0 = lane * PPL;
  cx<float> x[PPL], y[PPL];
#pragma unroll
  for (int p = 0; p < PPL; ++p) {
    x[p] = mk<float>(a0 + p == row ? 1.f : 0.f, 0.f);
    y[p] = mk<float>(kp - 1 - a0 - p == row ? 1.f : 0.f, 0.f);
  }
  const int rounds = meta[META_ROUNDS];
  for (int r0 = 0; r0 < rounds; r0 += REPLAY) {
    const int nr = min(REPLAY, rounds - r0);
    __syncthreads();
    for (int e = t; e < nr * np; e += 256) R[e] = rots[(size_t)r0 * np + e];
    __syncthreads();
#pragma unroll 2
    for (int rd = 0; rd < nr; ++rd) {
      cx<float> x1[PPL], y1[PPL];
#pragma unroll
      for (int p = 0; p < PPL; ++p) {
        const float4 r = R[rd * np + min(a0 + p, np - 1)];
        const cx<float> s = mk<float>(r.y, r.z);
        x1[p] = r.x * x[p] - conj(s) * y[p];
        y1[p] = s * x[p] + r.x * y[p];
      }
      const cx<float> dn = mk<float>(__shfl_down_sync(0xffffffffu, x1[0].re, 1), __shfl_down_sync(0xffffffffu, x1[0].im, 1));
      const cx<float> up = mk<float>(__shfl_up_sync(0xffffffffu, y1[PPL - 1].re, 1), __shfl_up_sync(0xffffffffu, y1[PPL - 1].im, 1));
#pragma unroll
      for (int p = 0; p < PPL; ++p) {
        const cx<float> next = p + 1 < PPL ? x1[p + 1 < PPL ? p + 1 : 0] : dn, prev = p > 0 ? y1[p > 0 ? p - 1 : 0] : up;
        x[p] = a0 + p == 0 ? x1[p] : (a0 + p == np - 1 ? y1[p] : next);
        y[p] = a0 + p == 0 ? (np == 1 ? y1[p] : next) : prev;
      }
    }
  }
  if (row < k)
#pragma unroll
    for (int p = 0; p < PPL; ++p)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int i = h ? kp - 1 - a0 - p : a0 + p;
        if (a0 + p >= np || i >= k) continue;
        const cx<float> u = h ? y[p] : x[p];
        const int rk = order[i];
        Uf[(size_t)rk * k + row] = u;
        if (rk < nout) Uout[(size_t)rk * ldu + row] = cvt<double>(u);
      }
}

static size_t j32_smem(int k) {
  const int kp = k + (k & 1);
  return (size_t)kp * (kp + 1) * sizeof(cx<float>);
}
static size_t replay_smem(int k) { return (size_t)REPLAY * ((k + 1) / 2) * sizeof(float4); }

// Conversions by their bits (a conversion instruction runs at the FP64 rate): x truncated to FP32 (zero below
// 2^-126; x is finite and below 2^128), and back (normal numbers and zero).
__device__ __forceinline__ float f32_bits(double x) {
  const int hi = __double2hiint(x), e = ((hi >> 20) & 0x7ff) - 896;
  return e <= 0 ? 0.f : __int_as_float((hi & 0x80000000) | e << 23 | (hi & 0xfffff) << 3 | (int)((unsigned)__double2loint(x) >> 29));
}
__device__ __forceinline__ double f64_bits(float x) {
  const int b = __float_as_int(x), e = (b >> 23) & 0xff;
  return e == 0 ? 0.0 : __hiloint2double((b & 0x80000000) | (e + 896) << 20 | ((b >> 3) & 0xfffff), b << 29);
}
__device__ __forceinline__ double flip_if(double x, bool c) {
  return __hiloint2double(__double2hiint(x) ^ (c ? 0x80000000 : 0), __double2loint(x));
}

// FP64, k <= 32, one CTA.  An FP64 instruction occupies a scheduler for 64 cycles, a division or square root for 7 to 11 of
// these, so (a) the angle of a rotation is taken in FP32: it annihilates its entry to 1e-7 instead of 1e-16, which leaves the
// number of sweeps as it is, and the rotation is made unitary in FP64, c = sqrt(1 - |s|^2) by two Newton steps from its
// FP32 value; (b) one thread computes one real component (three multiply-adds for A J, three for J^H (A J), the
// neighbours' components by shuffles), eight threads a 2 x 2 block.  A is scaled by a power of two to entries below
// 2, so that FP32 has the range.  (One thread per block and FP64 angles: 55 us a call at k = 8 in a step; 12 us so.)
__global__ void __launch_bounds__(512) jacobi64_kernel(const zd *__restrict__ Ain, int lda, int k, zd *__restrict__ Uout,
                                                       int ldu, double *__restrict__ wout, int max_sweeps, double tol,
                                                       int *status) {
  __shared__ double A[2 * 32 * 33], U[2 * 32 * 33];   // (re, im) pairs, leading dimension ld
  __shared__ double rc[16], rsr[16], rsi[16];
  __shared__ int rpq[16];
  __shared__ unsigned red[2][16];
  const int kp = k + (k & 1), ld = kp + 1, np = kp / 2;
  const int t = threadIdx.x, nt = blockDim.x, lane = t & 31, wp = t >> 5, nw = nt >> 5;
  unsigned emax = 0;
  for (int e = t; e < kp * kp; e += nt) {
    const int i = e % kp, j = e / kp;
    const zd a = (i < k && j < k && i <= j) ? Ain[(size_t)j * lda + i] : mk<double>(0, 0);
    A[2 * (j * ld + i)] = a.re;
    A[2 * (j * ld + i) + 1] = a.im;
    U[2 * (j * ld + i)] = i == j ? 1.0 : 0.0;
    U[2 * (j * ld + i) + 1] = 0.0;
    emax = max(emax, max((unsigned)__double2hiint(a.re) >> 20 & 0x7ffu, (unsigned)__double2hiint(a.im) >> 20 & 0x7ffu));
  }
  emax = __reduce_max_sync(0xffffffffu, emax);
  if (lane == 0) red[0][wp] = emax;
  __syncthreads();
  for (int w = 0; w < nw; ++w) emax = max(emax, red[0][w]);
  const bool finite = emax < 0x7ff;
  const int es = emax == 0 || !finite ? 1023 : max(1, 2046 - (int)emax);
  const double scale = __hiloint2double(es << 20, 0), unscale = __hiloint2double((2046 - es) << 20, 0);
  for (int e = t; e < kp * kp; e += nt) {   // each thread its own elements of the loop above
    A[2 * ((e / kp) * ld + e % kp)] *= scale;
    A[2 * ((e / kp) * ld + e % kp) + 1] *= scale;
  }
  __syncthreads();
  // Stop when the off-diagonal Frobenius norm is below tol times the whole one, both in FP32: entries are below 2 and the largest is
  // at least 1, so squares that FP32 flushes (below 1e-38) are far below tol^2 = 1e-30.  A bound on the largest entry that
  // implies this lies below the entries' own rounding at k = 32 (7 sweeps a call at r = 16 for equal weights, 20 at 32; none so).
  const float tol2 = (float)(tol * tol);
  const int nA = (np * (np + 1) / 2 * 8 + 31) & ~31, nU = (np * kp * 4 + 31) & ~31;
  int sweep = 0;
  for (; finite && sweep < max_sweeps; ++sweep) {
    float off = 0.f, dia = 0.f;
    for (int e = t; e < kp * kp; e += nt) {
      const int i = e % kp, j = e / kp;
      if (i > j) continue;
      const float re = f32_bits(A[2 * (j * ld + i)]), im = f32_bits(A[2 * (j * ld + i) + 1]), v = fmaf(re, re, im * im);
      if (i == j) dia += v;
      else off += 2.f * v;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      off += __shfl_xor_sync(0xffffffffu, off, o);
      dia += __shfl_xor_sync(0xffffffffu, dia, o);
    }
    if (lane == 0) { red[0][wp] = __float_as_uint(off); red[1][wp] = __float_as_uint(dia); }
    __syncthreads();
    off = dia = 0.f;
    for (int w = 0; w < nw; ++w) { off += __uint_as_float(red[0][w]); dia += __uint_as_float(red[1][w]); }
    if (off <= tol2 * (off + dia)) break;
    for (int round = 0; round < kp - 1; ++round) {
      if (t < np) {
        int p, q;
        round_pair(t, round, kp, &p, &q);
        const float br = f32_bits(A[2 * (q * ld + p)]), bi = f32_bits(A[2 * (q * ld + p) + 1]), n2 = fmaf(br, br, bi * bi);
        double c = 1.0, sr = 0.0, si = 0.0;
        if (n2 > 1e-37f) {
          const float h = 0.5f * f32_bits(A[2 * (q * ld + q)] - A[2 * (p * ld + p)]), g = fmaf(h, h, n2);
          const float f = copysignf(__fdividef(1.f, fabsf(h) + g * rsqrtf(g)), h), v = fmaf(n2 * f, f, 1.f);
          const float cf = rsqrtf(v);
          sr = f64_bits(cf * f * br);
          si = f64_bits(cf * f * bi);
          const double x = fma(-sr, sr, fma(-si, si, 1.0)), hc = f64_bits(0.5f * v * cf);   // c^2, 1 / (2 c)
          c = f64_bits(cf);
          c = fma(fma(-c, c, x), hc, c);
          c = fma(fma(-c, c, x), hc, c);
        }
        rc[t] = c;
        rsr[t] = sr;
        rsi[t] = si;
        rpq[t] = p | q << 16;
      }
      __syncthreads();
      for (int base = wp * 32; base < nA + nU; base += nt) {
        const bool isA = base < nA;
        const int f = isA ? base + lane : base - nA + lane;
        const int cm = f & 1, j = (f >> 1) & 1;
        if (isA) {   // component cm of entry (i, j) of the block of pairs a <= b
          const int i = (f >> 2) & 1;
          int a, b;
          const bool in = (f >> 3) < np * (np + 1) / 2;
          tri_item(in ? f >> 3 : 0, &a, &b, 1);
          const int ra = i ? rpq[a] >> 16 : rpq[a] & 0xffff;
          const int cj = j ? rpq[b] >> 16 : rpq[b] & 0xffff, co = j ? rpq[b] & 0xffff : rpq[b] >> 16;
          const double *own = ra <= cj ? A + 2 * (cj * ld + ra) : A + 2 * (ra * ld + cj);
          const double *oth = ra <= co ? A + 2 * (co * ld + ra) : A + 2 * (ra * ld + co);
          // an element below the diagonal is its mirror's conjugate
          const double u = flip_if(own[cm], cm && ra > cj), v = flip_if(oth[cm], cm && ra > co),
                       w = flip_if(oth[1 - cm], !cm && ra > co);
          // Y_0 = c X_0 - conj(s) X_1, Y_1 = c X_1 + s X_0
          const double y = fma(rc[b], u, fma(flip_if(rsr[b], !j), v, flip_if(rsi[b], !cm) * w));
          const double v2 = __shfl_xor_sync(0xffffffffu, y, 4), w2 = __shfl_xor_sync(0xffffffffu, y, 5);
          // X'_0 = c Y_0 - s Y_1, X'_1 = c Y_1 + conj(s) Y_0
          double z = fma(rc[a], y, fma(flip_if(rsr[a], !i), v2, flip_if(rsi[a], cm) * w2));
          double *dst = ra <= cj ? A + 2 * (cj * ld + ra) : A + 2 * (ra * ld + cj);
          if (a == b && i == j && cm) z = 0.0;
          if (in && (a != b || i == j || ra < cj)) dst[cm] = flip_if(z, cm && ra > cj);
        } else {   // U <- U J
          const bool in = (f >> 2) < np * kp;
          const int row = in ? (f >> 2) % kp : 0, b = in ? (f >> 2) / kp : 0;
          const int cj = j ? rpq[b] >> 16 : rpq[b] & 0xffff, co = j ? rpq[b] & 0xffff : rpq[b] >> 16;
          const double u = U[2 * (cj * ld + row) + cm], v = U[2 * (co * ld + row) + cm], w = U[2 * (co * ld + row) + 1 - cm];
          const double y = fma(rc[b], u, fma(flip_if(rsr[b], !j), v, flip_if(rsi[b], !cm) * w));
          __syncwarp();
          if (in) U[2 * (cj * ld + row) + cm] = y;
        }
      }
      __syncthreads();
    }
    if (sweep == max_sweeps - 1 && t == 0 && status) atomicOr(status, ST_EIG_NOCONV);
  }
  if (t == 0) {
    atomicAdd(&g_jacobi_counters[2], 1ull);
    atomicAdd(&g_jacobi_counters[3], (unsigned long long)sweep);
  }
  // sort eigenvalues decreasing (ties by index) and write out
  for (int e = t; e < k * k; e += nt) {
    const int i = e / k, row = e % k;
    const double wi = A[2 * (i * ld + i)];
    int rank = 0;
    for (int j = 0; j < k; ++j) {
      const double wj = A[2 * (j * ld + j)];
      rank += (wj > wi) || (wj == wi && j < i);
    }
    if (row == 0) wout[rank] = wi * unscale;
    Uout[(size_t)rank * ldu + row] = mk<double>(U[2 * (i * ld + row)], U[2 * (i * ld + row) + 1]);
  }
}

void sm_jacobi64(const zd *A, int lda, int k, zd *U, int ldu, double *w, int max_sweeps, double tol, int *status,
                 cudaStream_t st) {
  const int np = (k + 1) / 2, slots = np * (np + 1) * 4 + 8 * np * np + 64;
  const int nt = slots >= 512 ? 512 : slots / 32 * 32;
  ::lrei::count_launch();
  jacobi64_kernel<<<1, nt, 0, st>>>(A, lda, k, U, ldu, w, max_sweeps, tol, status);
}

// ------------------------------------------------------------ top-r eig
// Whether pass p ends with an orthonormalisation: E + D has Gram I + D^H D (D is orthogonal to E), so only after
// the first pass (E is orthonormal to FP32 before it), a large correction, and the last one.
__device__ __forceinline__ bool newton_orth(const int *meta, int p) {
  return p == 1 || p == NEWTON_PASSES || !(__int_as_float(meta[META_D + p - 1]) <= 1e-9f) || newton_done(meta, p);
}

// Block-Newton correction of the top-r invariant subspace, one CTA per column j of E; everything below is local to that
// column once W1 = M E is known:
//   a = E^H W1[:, j],  R = W1[:, j] - E a                  (FP64: the residual is a small difference)
//   X_i = (Ur^H R)_i / (a_j - w_{r+i}),  D = Ur X           (FP32: only the correction's leading digits
//   Enew[:, j] = E[:, j] + D - E (E^H D)                      matter; Ur is FP32-accurate anyway)
// Ur, w_{r+i}: the FP32 eigenpairs of the other k - r eigenvalues (columns r + i of Uf).  Because the correction is driven
// by the residual (which vanishes exactly on the invariant subspace), repeated passes converge to FP64 accuracy although
// Ur is only FP32-accurate.  Ef: E in FP32.  The FP64 sums are chains of 64 cycles per
// instruction, so each is split over lanes: 32 per entry of a, 8 (4 parts x re, im) per entry of R.
constexpr int NEWTON_THREADS = 512;
__global__ void __launch_bounds__(NEWTON_THREADS) newton_chain_kernel(
    const zd *__restrict__ W1, const zd *__restrict__ E, const cx<float> *__restrict__ Ef, const cx<float> *__restrict__ Uf,
    const double *__restrict__ w, int k, int r, zd *__restrict__ Enew, int *meta, int pass) {
  if (newton_done(meta, pass - 1)) return;
  extern __shared__ __align__(16) unsigned char nsm[];
  zd *av = reinterpret_cast<zd *>(nsm);                     // r
  cx<float> *rf = reinterpret_cast<cx<float> *>(av + r);    // k: residual (FP32)
  cx<float> *x = rf + k;                                    // k - r
  cx<float> *d2 = x + k;                                    // k
  cx<float> *g1 = d2 + k;                                   // r
  cx<float> *pd = g1 + r;                                   // 4 x k: parts of D
  float *den = reinterpret_cast<float *>(pd + 4 * k);       // k - r
  const int j = blockIdx.x, t = threadIdx.x, lane = t & 31, wp = t >> 5;
  constexpr int NW = NEWTON_THREADS / 32;
  const zd *w1 = W1 + (size_t)j * k;
  for (int i = wp; i < r; i += NW) {          // a = E^H w1
    zd s = mk<double>(0, 0);
    for (int p = lane; p < k; p += 32) fmac_(s, E[(size_t)i * k + p], w1[p]);
    s = warp_sum(s);
    if (lane == 0) av[i] = s;
  }
  __syncthreads();
  for (int i = t; i < k - r; i += NEWTON_THREADS) den[i] = (float)(av[j].re - w[r + i]);
  for (int base = 0; base < k; base += NEWTON_THREADS / 8) {   // R = w1 - E a
    const int p = base + (t >> 3), cm = t & 1, q = (t >> 1) & 3;
    double s = 0.0;
    if (p < k)
      for (int i = q; i < r; i += 4) {
        const zd e = E[(size_t)i * k + p], a = av[i];
        s = fma(e.re, cm ? a.im : a.re, fma(e.im, cm ? a.re : -a.im, s));
      }
    s += __shfl_xor_sync(0xffffffffu, s, 2);
    s += __shfl_xor_sync(0xffffffffu, s, 4);
    if (p < k && q == 0) reinterpret_cast<float *>(rf)[2 * p + cm] = (float)((cm ? w1[p].im : w1[p].re) - s);
  }
  __syncthreads();
#pragma unroll 2
  for (int i = wp; i < k - r; i += NW) {      // X = (Ur^H R) ./ (d_j - w)
    cx<float> s = mk<float>(0.f, 0.f);
    const cx<float> *u = Uf + (size_t)(r + i) * k;
    for (int p = lane; p < k; p += 32) fmac_(s, u[p], rf[p]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      s.re += __shfl_xor_sync(0xffffffffu, s.re, o);
      s.im += __shfl_xor_sync(0xffffffffu, s.im, o);
    }
    if (lane == 0) x[i] = (fabsf(den[i]) > 1e-30f) ? mk<float>(s.re / den[i], s.im / den[i]) : mk<float>(0.f, 0.f);
  }
  __syncthreads();
  {                                           // D = Ur X, in four parts
    const int c = t / (NEWTON_THREADS / 4), n4 = (k - r + 3) / 4, i1 = min(k - r, (c + 1) * n4);
    for (int p = t % (NEWTON_THREADS / 4); p < k; p += NEWTON_THREADS / 4) {
      cx<float> s = mk<float>(0.f, 0.f);
#pragma unroll 8
      for (int i = c * n4; i < i1; ++i) fma_(s, Uf[(size_t)(r + i) * k + p], x[i]);
      pd[c * k + p] = s;
    }
  }
  __syncthreads();
  for (int p = t; p < k; p += NEWTON_THREADS) d2[p] = (pd[p] + pd[k + p]) + (pd[2 * k + p] + pd[3 * k + p]);
  __syncthreads();
  for (int i = wp; i < r; i += NW) {          // g = E^H D
    cx<float> s = mk<float>(0.f, 0.f);
    for (int p = lane; p < k; p += 32) fmac_(s, Ef[(size_t)i * k + p], d2[p]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      s.re += __shfl_xor_sync(0xffffffffu, s.re, o);
      s.im += __shfl_xor_sync(0xffffffffu, s.im, o);
    }
    if (lane == 0) g1[i] = s;
  }
  __syncthreads();
  unsigned big = 0;
  for (int p = t; p < k; p += NEWTON_THREADS) {   // Enew = E + D - E g
    cx<float> s = d2[p];
#pragma unroll 8
    for (int i = 0; i < r; ++i) s = s - Ef[(size_t)i * k + p] * g1[i];
    const zd e = E[(size_t)j * k + p];
    Enew[(size_t)j * k + p] = mk<double>(e.re + (double)s.re, e.im + (double)s.im);
    big = max(big, max(__float_as_uint(fabsf(s.re)), __float_as_uint(fabsf(s.im))));
  }
  big = __reduce_max_sync(0xffffffffu, big);
  if (lane == 0 && big) atomicMax(reinterpret_cast<unsigned *>(meta + META_D + pass - 1), big);
}

size_t newton_chain_smem(int k, int r) {
  return (size_t)r * sizeof(zd) + (size_t)(7 * k + r) * sizeof(cx<float>) + (size_t)k * sizeof(float);
}

// Column j of E T for T = (15/8) I - (5/4) G + (3/8) G^2, G = E^H E = I + d: E (E^H E)^{-1/2} + O(d^3), the orthonormal polar
// factor of E (same span); Ein itself when the pass needs no orthonormalisation.  Also in FP32.
// Eight lanes (4 parts x re, im) per entry of T and of the product; 32 rows per CTA, r columns.  (T by one kernel,
// E T by another: 5.5 + 4.7 us at r = 8.)
__global__ void __launch_bounds__(256) polar_kernel(const zd *__restrict__ G, const zd *__restrict__ Ein, int k, int r,
                                                    zd *__restrict__ Eout, cx<float> *__restrict__ Eoutf, const int *meta,
                                                    int pass) {
  if (pass && newton_done(meta, pass - 1)) return;
  __shared__ zd T[MAX_R];
  const int j = blockIdx.x, t = threadIdx.x, cm = t & 1, q = (t >> 1) & 3, row = t >> 3;
  const int p = blockIdx.y * 32 + row;
  double s = 0.0;
  if (!pass || newton_orth(meta, pass)) {
    if (row < r)
      for (int m = q; m < r; m += 4) {
        const zd a = G[(size_t)m * r + row], b = G[(size_t)j * r + m];
        s = fma(a.re, cm ? b.im : b.re, fma(a.im, cm ? b.re : -b.im, s));
      }
    s += __shfl_xor_sync(0xffffffffu, s, 2);
    s += __shfl_xor_sync(0xffffffffu, s, 4);
    if (row < r && q == 0) {
      const double g = reinterpret_cast<const double *>(G + (size_t)j * r + row)[cm];
      reinterpret_cast<double *>(T)[2 * row + cm] = fma(0.375, s, fma(-1.25, g, (row == j && !cm) ? 1.875 : 0.0));
    }
    __syncthreads();
    s = 0.0;
    if (p < k)
      for (int m = q; m < r; m += 4) {
        const zd a = Ein[(size_t)m * k + p], b = T[m];
        s = fma(a.re, cm ? b.im : b.re, fma(a.im, cm ? b.re : -b.im, s));
      }
    s += __shfl_xor_sync(0xffffffffu, s, 2);
    s += __shfl_xor_sync(0xffffffffu, s, 4);
  } else if (p < k) {
    s = reinterpret_cast<const double *>(Ein + (size_t)j * k + p)[cm];
  }
  if (p < k && q == 0) {
    reinterpret_cast<double *>(Eout + (size_t)j * k + p)[cm] = s;
    reinterpret_cast<float *>(Eoutf + (size_t)j * k + p)[cm] = (float)s;
  }
}

// G = E^H E for polar_kernel, where the pass needs it: a warp per entry of the upper triangle.
__global__ void __launch_bounds__(128) polar_gram_kernel(const zd *__restrict__ E, int k, int r, zd *__restrict__ G,
                                                         const int *meta, int pass) {
  if (pass && (newton_done(meta, pass - 1) || !newton_orth(meta, pass))) return;
  const int e = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (e >= r * (r + 1) / 2) return;
  int i, j;
  tri_item(e, &i, &j, 1);
  zd s = mk<double>(0, 0);
  for (int p = lane; p < k; p += 32) fmac_(s, E[(size_t)i * k + p], E[(size_t)j * k + p]);
  s = warp_sum(s);
  if (lane == 0) {
    if (i == j) s.im = 0.0;
    G[(size_t)j * r + i] = s;
    if (i != j) G[(size_t)i * r + j] = conj(s);
  }
}

// Y = E Wr (column j: blockIdx.x, 32 rows per CTA, eight lanes per entry), the residual M Y - Y diag(mu) from ME = M E, and its check:
// an entry that may exceed tol * max |mu|, or is not finite, sets ST_EIG_RESID.
__global__ void __launch_bounds__(256) eig_finish_kernel(const zd *__restrict__ E, const zd *__restrict__ ME,
                                                         const zd *__restrict__ Wr, const double *__restrict__ mu, int k, int r,
                                                         zd *__restrict__ Y, int ldy, double tol, int *status) {
  const int j = blockIdx.x, t = threadIdx.x, cm = t & 1, q = (t >> 1) & 3, p = blockIdx.y * 32 + (t >> 3);
  double y = 0.0, z = 0.0;
  if (p < k)
    for (int m = q; m < r; m += 4) {
      const zd a = E[(size_t)m * k + p], c = ME[(size_t)m * k + p], b = Wr[(size_t)j * r + m];
      const double bs = cm ? b.im : b.re, bo = cm ? b.re : -b.im;
      y = fma(a.re, bs, fma(a.im, bo, y));
      z = fma(c.re, bs, fma(c.im, bo, z));
    }
#pragma unroll
  for (int o = 2; o <= 4; o <<= 1) {
    y += __shfl_xor_sync(0xffffffffu, y, o);
    z += __shfl_xor_sync(0xffffffffu, z, o);
  }
  if (p < k && q == 0) {
    reinterpret_cast<double *>(Y + (size_t)j * ldy + p)[cm] = y;
    double mm = 1e-300;
    for (int i = 0; i < r; ++i) mm = fmax(mm, fabs(mu[i]));
    if (!(fabs(fma(-mu[j], y, z)) <= 0.70710678 * tol * mm)) atomicOr(status, ST_EIG_RESID);
  }
}

static size_t rots_bytes(int k) {
  const int kp = std::min(k + (k & 1), J32_KMAX);
  return (size_t)J32_SWEEPS * (kp - 1) * (kp / 2) * sizeof(float4);
}

size_t sm_eig_ws_bytes(int kmax, int rmax) {
  size_t z = sizeof(zd);
  size_t b = 0;
  b += (size_t)kmax * 8;                                  // w
  b += 3 * (size_t)kmax * rmax * z;                       // W1, E1, W2
  b += 3 * (size_t)rmax * rmax * z;                       // G, Ar, Wr
  b += (size_t)kmax * (kmax + rmax) * sizeof(cx<float>);  // FP32 eigenvectors, FP32 copy of E
  b += (size_t)kmax * sizeof(int) + META_INTS * sizeof(int) + rots_bytes(kmax);
  return b + 4096;
}

void sm_eig_topr(const zd *M, int ldm, int k, int r, zd *Y, int ldy, double *mu, void *ws, int *status,
                 cudaStream_t st, int max_sweeps) {
  unsigned char *p = reinterpret_cast<unsigned char *>(ws);
  auto take = [&](size_t bytes) { unsigned char *q = p; p += (bytes + 255) & ~(size_t)255; return q; };
  double *w = (double *)take((size_t)k * 8);
  zd *W1 = (zd *)take((size_t)k * r * sizeof(zd));
  zd *E1 = (zd *)take((size_t)k * r * sizeof(zd));
  zd *W2 = (zd *)take((size_t)k * r * sizeof(zd));
  zd *G = (zd *)take((size_t)r * r * sizeof(zd));
  zd *Ar = (zd *)take((size_t)r * r * sizeof(zd));
  zd *Wr = (zd *)take((size_t)r * r * sizeof(zd));
  cx<float> *U32 = (cx<float> *)take((size_t)k * k * sizeof(cx<float>));
  cx<float> *E32 = (cx<float> *)take((size_t)k * r * sizeof(cx<float>));
  int *order = (int *)take((size_t)k * sizeof(int));
  int *meta = (int *)take(META_INTS * sizeof(int));
  float4 *rots = (float4 *)take(rots_bytes(k));
  const zd one = mk<double>(1, 0), zero = mk<double>(0, 0);
  // 1. FP32 eigendecomposition of the whole k x k matrix: all eigenvectors in FP32 (U32), the
  //    top r also in FP64 (E1), eigenvalues in FP64 (w).  Threads: a block each while the CTA has them.
  const int np = (k + 1) / 2, nt = std::min(512, std::max(64, (np * (np + 1) / 2 + 31) / 32 * 32));
  ::lrei::count_launch();
  jacobi32_kernel<<<1, nt, j32_smem(k), st>>>(M, ldm, k, w, order, rots, meta, 1e-5f);
  ::lrei::count_launch();
  auto replay = [&](auto kern) { kern<<<(k + 7) / 8, 256, replay_smem(k), st>>>(k, rots, meta, order, U32, E1, k, r); };
  if (np <= 32) replay(replay_kernel<1>);
  else if (np <= 64) replay(replay_kernel<2>);
  else replay(replay_kernel<3>);
  // 2.-3. block-Newton corrections of the top-r invariant subspace and polar re-orthonormalisations, each pass
  //       returning at once when the ones before it have converged
  const dim3 rows(r, (k + 31) / 32);
  const int grams = (r * (r + 1) / 2 + 3) / 4;
  auto polar = [&](const zd *in, zd *out, int pass) {
    ::lrei::count_launch();
    polar_gram_kernel<<<grams, 128, 0, st>>>(in, k, r, G, meta, pass);
    ::lrei::count_launch();
    polar_kernel<<<rows, 256, 0, st>>>(G, in, k, r, out, E32, meta, pass);
  };
  zd *E = E1;
  if (k > r) {
    for (int pass = 1; pass <= NEWTON_PASSES; ++pass) {
      gemm_launch('N', 'N', k, r, k, one, M, ldm, E1, k, zero, W1, k, W1, k, 0, st, meta, pass - 1);   // W1 = M E
      ::lrei::count_launch();
      newton_chain_kernel<<<r, NEWTON_THREADS, newton_chain_smem(k, r), st>>>(W1, E1, pass == 1 ? U32 : E32, U32, w, k, r, W2,
                                                                             meta, pass);
      polar(W2, E1, pass);
    }
  } else {
    polar(E1, W2, 0);
    E = W2;
  }
  // 4. Rayleigh-Ritz on span(E) in FP64
  sm_gemm('N', 'N', k, r, k, one, M, ldm, E, k, zero, W1, k, st);
  sm_gemm_herm('C', 'N', r, k, one, E, k, W1, k, zero, Ar, r, Ar, r, st);
  sm_jacobi64(Ar, r, r, Wr, r, mu, max_sweeps, 1e-14, status, st);
  // 5. the returned vectors and the residual check of the pairs
  ::lrei::count_launch();
  eig_finish_kernel<<<rows, 256, 0, st>>>(E, W1, Wr, mu, k, r, Y, ldy, 1e-9, status);
}

// ------------------------------------------------------------ elementwise
__global__ void copy_kernel(const zd *A, int lda, int M, int N, zd *B, int ldb, int mode) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < M * N; e += gridDim.x * blockDim.x) {
    const int i = e % M, j = e / M;
    if (mode == 0) B[(size_t)j * ldb + i] = A[(size_t)j * lda + i];
    else if (mode == 2) B[(size_t)j * ldb + i] = mk<double>(0, 0);
    else B[(size_t)j * ldb + i] = mk<double>(i == j ? 1 : 0, 0);
  }
}
static int grid_for(long long n) { long long g = (n + 255) / 256; return (int)(g < 1 ? 1 : (g > 1024 ? 1024 : g)); }
void sm_copy(const zd *A, int lda, int M, int N, zd *B, int ldb, cudaStream_t st) {
  ::lrei::count_launch(); copy_kernel<<<grid_for((long long)M * N), 256, 0, st>>>(A, lda, M, N, B, ldb, 0);
}
void sm_zero(zd *A, int lda, int M, int N, cudaStream_t st) {
  ::lrei::count_launch(); copy_kernel<<<grid_for((long long)M * N), 256, 0, st>>>(nullptr, 0, M, N, A, lda, 2);
}
void sm_set_identity(zd *A, int lda, int M, int N, cudaStream_t st) {
  ::lrei::count_launch(); copy_kernel<<<grid_for((long long)M * N), 256, 0, st>>>(nullptr, 0, M, N, A, lda, 3);
}

__global__ void hermitize_kernel(zd *A, int lda, int k) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < k * k; e += gridDim.x * blockDim.x) {
    const int i = e % k, j = e / k;
    if (i > j) continue;
    const zd a = A[(size_t)j * lda + i], b = A[(size_t)i * lda + j];
    const zd h = mk<double>(0.5 * (a.re + b.re), 0.5 * (a.im - b.im));
    A[(size_t)j * lda + i] = h;
    A[(size_t)i * lda + j] = conj(h);
    if (i == j) A[(size_t)j * lda + i] = mk<double>(h.re, 0);
  }
}
void sm_hermitize(zd *A, int lda, int k, cudaStream_t st) { ::lrei::count_launch(); hermitize_kernel<<<grid_for((long long)k * k), 256, 0, st>>>(A, lda, k); }

// B = (A + A^H)/2, k x k.
__global__ void herm_copy_kernel(const zd *__restrict__ A, int lda, int k, zd *__restrict__ B, int ldb) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < k * k; e += gridDim.x * blockDim.x) {
    const int i = e % k, j = e / k;
    const zd a = A[(size_t)j * lda + i], b = A[(size_t)i * lda + j];
    B[(size_t)j * ldb + i] = mk<double>(0.5 * (a.re + b.re), i == j ? 0.0 : 0.5 * (a.im - b.im));
  }
}
void sm_herm_copy(const zd *A, int lda, int k, zd *B, int ldb, cudaStream_t st) {
  ::lrei::count_launch(); herm_copy_kernel<<<grid_for((long long)k * k), 256, 0, st>>>(A, lda, k, B, ldb);
}

}  // namespace lrei

namespace lrei {
int sm_init() {
  const int lim = 210 * 1024;
  cudaFuncSetAttribute(chol_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
  cudaError_t a = cudaFuncSetAttribute(jacobi32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
  return a == cudaSuccess ? 0 : -1;
}
}  // namespace lrei

namespace lrei {
int sm_read_counters(unsigned long long *out) {
  return cudaMemcpyFromSymbol(out, g_jacobi_counters, sizeof(unsigned long long) * 4) == cudaSuccess ? 0 : -1;
}
}  // namespace lrei
