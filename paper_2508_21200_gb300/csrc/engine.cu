// LREI step engine and C ABI (include/lrei.h).
//
// One RK_s step (paper Sec. 3.7, eqs. rk:sstageform, K-expand, rho-expand)
// is computed exactly as the paper's scheme, but organised for the GPU:
//
//  * Every stage matrix K_{j+1} = K_1 + h sum_l a_{j+1,l} (Z_l V_l^* + V_l W_l^*)
//    has its range inside span{V_1, W_1, ..., W_j}, and since W_l lies in
//    span{V_l, H V_l} and V_l in range(K_l), that span is the block Krylov
//    space K_{j+1}(H, V_1).  The engine therefore builds one block-Krylov
//    basis Q = [Q_0 = V_1, Q_1, ..., Q_s] per step (one H application and two
//    tall-skinny passes per block, measured Gram Gamma = Q^*Q) and evaluates
//    every stage -- G_j = V_j^* H V_j, the X blocks of eqs. X-blocks-sol /
//    X-blocks-sol-qLL, W_j, Z_j, the stage matrix and its partial
//    eigendecomposition -- in the (s+1) r dimensional coordinates of Q.
//  * The partial eigendecomposition of each K_{j+1} (the paper's IRLM on
//    g(x), eq. g-func) is an exact Rayleigh-Ritz on that space, so the result
//    equals the projected EI scheme up to rounding.
//  * The complement product W = V^ X12^* (Sec. 3.4-3.5) is applied in
//    coordinates as (I - V V^*) H V diag(conj c), which equals the Householder
//    form for any orthonormal complement.
//  * The new factor V_{k+1} = Q Y is formed in one pass at the end of the step.
// All small algebra is FP64; the N-length passes run in the context's
// precision.  A whole step is captured once in a CUDA graph and replayed.
#include "lrei.h"
#include "common.cuh"
#include "small.cuh"
#include "small_dev.cuh"
#include "tsk.cuh"

namespace lrei { int sm_read_counters(unsigned long long *out); }
namespace lrei {
int launch_rdm(bool fp64, const void *V, long long N, int r, const double *lam, const int *pairs, int npairs,
               double *partial, int ncta, cudaStream_t st);
void launch_rdm_final(const double *partial, int nparts, int npairs, double p_werner, double *out, cudaStream_t st);
}  // namespace lrei
// controller network inference on a given stream (mlp.cu)
int lrei_mlp_forward_on(lrei_mlp *net, const float *X, int B, float *Y, cudaStream_t st);

#include <nvtx3/nvToolsExt.h>

#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <algorithm>
#include <cstdlib>
#include <vector>

namespace lrei {

static std::atomic<long long> g_launches{0};
long long launch_counter() { return g_launches.load(); }
void count_launch(int n) { g_launches += n; }

// A named NVTX range for the duration of one ABI call (shows in Nsight timelines; no cost when
// no tool is attached).  Work inside a captured step graph is not split into ranges: the graph
// replays without host code.
struct NvtxScope {
  explicit NvtxScope(const char *name) { nvtxRangePushA(name); }
  ~NvtxScope() { nvtxRangePop(); }
  NvtxScope(const NvtxScope &) = delete;
  NvtxScope &operator=(const NvtxScope &) = delete;
};

int cuda_fail(cudaError_t e, const char *what) {
  (void)what;
  if (e == cudaErrorMemoryAllocation) return LREI_ERR_OOM;
  return LREI_ERR_CUDA;
}

struct Tableau {
  int s;
  double a[4][4];
  double b[4];
};
// Butcher tableaus: forward Euler, the paper's RK2 example (a21 = 1, b = 1/2, 1/2),
// Kutta's third-order method, classic RK4.
static const Tableau kRK[4] = {
    {1, {{0}}, {1.0}},
    {2, {{0, 0}, {1.0, 0}}, {0.5, 0.5}},
    {3, {{0, 0, 0}, {0.5, 0, 0}, {-1.0, 2.0, 0}}, {1.0 / 6, 4.0 / 6, 1.0 / 6}},
    {4, {{0, 0, 0, 0}, {0.5, 0, 0, 0}, {0, 0.5, 0, 0}, {0, 0, 1.0, 0}}, {1.0 / 6, 2.0 / 6, 2.0 / 6, 1.0 / 6}},
};

// Adams-Bashforth weights b_1..b_m (most recent first).  The 2-step weights are
// (3/2, -1/2); the printed -3/2 would not be consistent (weights must sum to 1).
static const double kAB[3][4] = {
    {1.5, -0.5, 0, 0},
    {23.0 / 12, -16.0 / 12, 5.0 / 12, 0},
    {55.0 / 24, -59.0 / 24, 37.0 / 24, -9.0 / 24},
};

// ----------------------------------------------------------- stage kernels
// Column j of the X11 block, the complement coefficient c_j, and the W, Z
// coordinates of one stage (eqs. X-blocks-sol and X-blocks-sol-qLL, hbar = 1):
//   q-LLG: X11_ij = i (l_i - l_j) G_ij / (1 - i kappa (l_i - l_j)),  c_i = i l_i / (1 - i kappa l_i)
//   q-LL:  X11_ij = (i (l_i - l_j) - kappa (l_i - l_j)^2) G_ij,       c_i = (i - kappa l_i) l_i
//   W = (H V - V G) diag(conj c),  Z = V X11 + W.
__device__ __forceinline__ zd x11_factor(double li, double lj, double kappa, int model) {
  const double d = li - lj;
  if (model == LREI_QLLG) {
    // i d / (1 - i kappa d) = i d (1 + i kappa d) / (1 + kappa^2 d^2)
    const double den = 1.0 + kappa * kappa * d * d;
    return mk<double>(-kappa * d * d / den, d / den);
  }
  return mk<double>(-kappa * d * d, d);
}
__device__ __forceinline__ zd c_factor(double l, double kappa, int model) {
  if (model == LREI_QLLG) {
    const double den = 1.0 + kappa * kappa * l * l;
    return mk<double>(-kappa * l * l / den, l / den);
  }
  return mk<double>(-kappa * l * l, l);
}

__global__ void stage_xwz_kernel(const zd *__restrict__ G, int r, const double *__restrict__ lam, double kappa,
                                 int model, const zd *__restrict__ Y, const zd *__restrict__ T, int K, int ld,
                                 zd *__restrict__ X11, zd *__restrict__ Z, zd *__restrict__ W, zd *__restrict__ Gh) {
  const int j = blockIdx.x;
  extern __shared__ zd sh[];
  zd *gcol = sh;        // hermitised column j of G
  zd *xcol = sh + r;    // column j of X11
  for (int i = threadIdx.x; i < r; i += blockDim.x) {
    const zd a = G[(size_t)j * r + i], b = G[(size_t)i * r + j];
    zd g = mk<double>(0.5 * (a.re + b.re), 0.5 * (a.im - b.im));
    if (i == j) g.im = 0.0;
    gcol[i] = g;
    xcol[i] = x11_factor(lam[i], lam[j], kappa, model) * g;
    if (blockIdx.y) continue;
    X11[(size_t)j * r + i] = xcol[i];
    if (Gh) Gh[(size_t)j * r + i] = g;
  }
  __syncthreads();
  const zd cc = conj(c_factor(lam[j], kappa, model));
  // eight lanes (4 parts x re, im) per row, 32 rows per CTA: the sums are chains of FP64 instructions of 64 cycles
  const int row = blockIdx.y * 32 + (threadIdx.x >> 3), cm = threadIdx.x & 1, q = (threadIdx.x >> 1) & 3;
  double yg = 0.0, yx = 0.0;
  if (row < K)
    for (int i = q; i < r; i += 4) {
      const zd y = Y[(size_t)i * ld + row], g = gcol[i], x = xcol[i];
      yg = fma(y.re, cm ? g.im : g.re, fma(cm ? y.im : -y.im, cm ? g.re : g.im, yg));
      yx = fma(y.re, cm ? x.im : x.re, fma(cm ? y.im : -y.im, cm ? x.re : x.im, yx));
    }
#pragma unroll
  for (int o = 2; o <= 4; o <<= 1) {
    yg += __shfl_xor_sync(0xffffffffu, yg, o);
    yx += __shfl_xor_sync(0xffffffffu, yx, o);
  }
  double d = 0.0;
  if (row < K) d = reinterpret_cast<const double *>(T + (size_t)j * ld + row)[cm] - yg;
  const double od = __shfl_xor_sync(0xffffffffu, d, 1);   // the other component
  if (row < K && q == 0) {
    const double w = cm ? fma(od, cc.im, d * cc.re) : fma(d, cc.re, -od * cc.im);
    reinterpret_cast<double *>(W + (size_t)j * ld + row)[cm] = w;
    reinterpret_cast<double *>(Z + (size_t)j * ld + row)[cm] = yx + w;
  }
}

struct StageCoefs {
  int nterms;
  double c[4];
};

// Factor matrices of a stage matrix: M = sum_b U_b V_b^H with
//   U = [Y_0 Lambda_0 | h c_0 Z_0 | h c_0 Y_0 | h c_1 Z_1 | h c_1 Y_1 | ...]
//   V = [Y_0          | Y_0       | W_0       | Y_1       | W_1       | ...]
// i.e. K_1 + h sum_l c_l (Z_l V_l^* + V_l W_l^*) in the Krylov coordinates (eqs. K-expand, rho-expand).
struct StagePtrs {
  const zd *y[5];
  const zd *z[4];
  const zd *w[4];
};
__global__ void stage_factors_kernel(StagePtrs P, StageCoefs C, const double *__restrict__ lam,
                                     const double *__restrict__ dt, int r, int K, int ld, zd *__restrict__ U,
                                     zd *__restrict__ V) {
  const int nb = 1 + 2 * C.nterms;
  const double h = *dt;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < nb * r * K; e += gridDim.x * blockDim.x) {
    const int row = e % K, col = e / K, blk = col / r, j = col % r;
    zd u, v;
    if (blk == 0) {
      const zd y = P.y[0][(size_t)j * ld + row];
      u = lam[j] * y;
      v = y;
    } else {
      const int l = (blk - 1) / 2;
      const double a = h * C.c[l];
      if ((blk - 1) % 2 == 0) {
        u = a * P.z[l][(size_t)j * ld + row];
        v = P.y[l][(size_t)j * ld + row];
      } else {
        u = a * P.y[l][(size_t)j * ld + row];
        v = P.w[l][(size_t)j * ld + row];
      }
    }
    U[(size_t)col * ld + row] = u;
    V[(size_t)col * ld + row] = v;
  }
}

// The part of the new rows k..k+r-1 of the Cholesky factor of Gamma left of their diagonal block (which the
// Cholesky kernel writes): Bs^H.  A dead column (numerically dependent on the earlier ones) is decoupled from the later
// columns; with keep_dead its row keeps the projections onto the earlier frame vectors, else it is zeroed too.  dead_frame (may be NULL)
// receives the dead flags of the new columns.
__global__ void store_lrows_kernel(const zd *__restrict__ Bs, int ldb, int r, int k,
                                   const int *__restrict__ dead, zd *__restrict__ L, int ldl, int keep_dead,
                                   int *__restrict__ dead_frame) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < r * k; e += gridDim.x * blockDim.x) {
    const int j = e % r, m = e / r;   // row k + j, column m
    L[(size_t)m * ldl + (k + j)] = (dead[j] && !keep_dead) ? mk<double>(0, 0) : conj(Bs[(size_t)j * ldb + m]);
  }
  if (dead_frame && blockIdx.x == 0)
    for (int j = threadIdx.x; j < r; j += blockDim.x) dead_frame[k + j] = dead[j];
}

// Rows of A (M x N) whose frame column is dead are set to zero.
__global__ void zero_dead_rows_kernel(zd *__restrict__ A, int lda, int M, int N, const int *__restrict__ dead_frame) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < M * N; e += gridDim.x * blockDim.x) {
    const int i = e % M, j = e / M;
    if (dead_frame[i]) A[(size_t)j * lda + i] = mk<double>(0, 0);
  }
}

__global__ void check_small_kernel(const double *mu, int r, const zd *G, int ldg, int *status) {
  bool bad = false;
  for (int i = threadIdx.x; i < r; i += blockDim.x) bad |= !isfinite(mu[i]);
  for (int e = threadIdx.x; e < r * r; e += blockDim.x) {
    const zd v = G[(size_t)(e / r) * ldg + (e % r)];
    bad |= !isfinite(v.re) || !isfinite(v.im);
  }
  if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(status, ST_NONFINITE);
}

// Diagonal matrix of conj(c) (for the explicit right-hand side) and -G diag(conj c).
__global__ void rhs_coef_kernel(const zd *__restrict__ G, int r, const double *__restrict__ lam, double kappa,
                                int model, zd *__restrict__ Dc, zd *__restrict__ Gc, zd *__restrict__ X11) {
  for (int e = threadIdx.x; e < r * r; e += blockDim.x) {
    const int i = e % r, j = e / r;
    const zd a = G[(size_t)j * r + i], b = G[(size_t)i * r + j];
    zd g = mk<double>(0.5 * (a.re + b.re), 0.5 * (a.im - b.im));
    const zd cc = conj(c_factor(lam[j], kappa, model));
    Dc[e] = (i == j) ? cc : mk<double>(0, 0);
    Gc[e] = mk<double>(-1, 0) * (g * cc);
    X11[e] = x11_factor(lam[i], lam[j], kappa, model) * g;
  }
}

// B = L^H diag(lam) L (r x r) for set_state: eight lanes per entry.
__global__ void lhl_kernel(const zd *__restrict__ L, int r, const double *__restrict__ lam, zd *__restrict__ B) {
  const int e = (blockIdx.x * blockDim.x + threadIdx.x) / 8, q = threadIdx.x & 7;
  const int i = e % r, j = e / r;
  zd s = mk<double>(0, 0);
  if (e < r * r)
    for (int m = q; m < r; m += 8) fma_(s, conj(L[(size_t)i * r + m]), lam[m] * L[(size_t)j * r + m]);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) {
    s.re += __shfl_xor_sync(0xffffffffu, s.re, o);
    s.im += __shfl_xor_sync(0xffffffffu, s.im, o);
  }
  if (e < r * r && q == 0) B[e] = s;
}

// Observables from the Gram blocks of the observable pass (one CTA, r <= 32).
// The stored factor V is orthonormalised implicitly: with V^*V = L L^H and X = L^{-1},
// Tr(rho A) = Tr(Lambda X (V^*AV) X^H) = Tr(W V^*AV), W = X^H Lambda X: the products by X are done once (W, and
// W2 = X^H Lambda^2 X for Tr(rho^2 H^2)) and each observable is a sum over r^2 entries.  Tr(rho H rho H) takes
// Gbar = X V^*HV X^H itself, sum lambda_i lambda_j |Gbar_ij|^2: as the trace of P P, P = W V^*HV (similar to Lambda Gbar by X^H), it
// would lose another condition number of V (of which the allocation-free call takes any).  FP64 instructions bound it (an SM issues
// one per 19 cycles): an entry's sum is split over four lanes.
// (With X A X^H formed per observable and square roots in the factor's chain: 179 us at r = 8, 2310 us at r = 32.)
// With Werner weight p (Sec. 5, eq. werner-sol) the state is rho = p I/N + (1 - p) rho_hat, rho_hat the
// stored low-rank state: H and the magnetisations are traceless, so their expectations and [rho, H] scale
// by q = 1 - p; Tr rho = p + q Tr rho_hat; Tr rho^2 = p^2/N + 2 p q Tr(rho_hat)/N + q^2 Tr rho_hat^2; each
// eigenvalue mu of rho_hat becomes p/N + q mu.  When mu is given, out[16 + i] receives the mapped Ritz
// values and out[48 + i] the mapped spectrum.
__device__ __forceinline__ zd quad_sum(zd v) {
#pragma unroll
  for (int o = 1; o <= 2; o <<= 1) {
    v.re += __shfl_xor_sync(0xffffffffu, v.re, o);
    v.im += __shfl_xor_sync(0xffffffffu, v.im, o);
  }
  return v;
}
__global__ void __launch_bounds__(512) obs_final_kernel(const double *__restrict__ red, int r, const double *__restrict__ lam,
                                                        double *__restrict__ out, double p, double inv_n,
                                                        const double *__restrict__ mu) {
  // blocks: 0 V^*HV, 1 (HV)^*(HV), 2 V^*V, 3 V^*MxV, 4 V^*MyV, 5 V^*MzV
  extern __shared__ zd s[];
  const int rr = r * r;
  zd *P = s, *X = s + rr, *W = s + 2 * rr, *W2 = s + 3 * rr;
  constexpr int NSUM = 8, NMAX = 3;
  __shared__ double part[NSUM][16];
  __shared__ unsigned long long pmax[NMAX][16];
  __shared__ double tot[NSUM], lams[MAX_R];
  const zd *B = reinterpret_cast<const zd *>(red);
  const zd *Gam = B + 2 * rr;
  const int t = threadIdx.x, nt = blockDim.x, lane = t & 31, wp = t >> 5, q4 = t & 3;
  for (int i = t; i < r; i += nt) lams[i] = lam[i];
  chol_inv_cta(Gam, r, r, P, X);
  for (int base = 0; base < rr; base += nt / 4) {      // W and W2, i <= j: sums over m >= j (X is lower triangular)
    const int e = base + (t >> 2), i = e % r, j = e / r;
    zd w = mk<double>(0, 0), w2 = w;
    if (e < rr && i <= j)
      for (int m = j + q4; m < r; m += 4) {
        const zd a = conj(X[i * r + m]), b = lams[m] * X[j * r + m];
        fma_(w, a, b);
        fma_(w2, a, lams[m] * b);
      }
    w = quad_sum(w);
    w2 = quad_sum(w2);
    if (e < rr && i <= j && q4 == 0) {
      W[j * r + i] = w;
      W[i * r + j] = conj(w);
      W2[j * r + i] = w2;
      W2[i * r + j] = conj(w2);
    }
  }
  __syncthreads();
  for (int base = 0; base < rr; base += nt / 4) {      // P = X V^*HV: sums over m <= i
    const int e = base + (t >> 2), i = e % r, j = e / r;
    zd v = mk<double>(0, 0);
    if (e < rr)
      for (int m = q4; m <= i; m += 4) fma_(v, X[m * r + i], B[j * r + m]);
    v = quad_sum(v);
    if (e < rr && q4 == 0) P[e] = v;
  }
  __syncthreads();
  // sums: 0 Tr(W A0), 1 Tr(W2 A1), 2..4 Tr(W A3..5), 5 sum lambda_i lambda_j |Gbar_ij|^2, 6 trace, 7 purity; maxima
  // (squares): V^*V - I, V^*HV - its conjugate transpose, V^*HV
  double acc[NSUM] = {0, 0, 0, 0, 0, 0, 0, 0};
  double mx[NMAX] = {0, 0, 0};
  for (int base = 0; base < rr; base += nt / 4) {      // Gbar = P X^H: sums over m <= j
    const int e = base + (t >> 2), i = e % r, j = e / r;
    zd g = mk<double>(0, 0);
    if (e < rr)
      for (int m = q4; m <= j; m += 4) fma_(g, P[m * r + i], conj(X[m * r + j]));
    g = quad_sum(g);
    if (e < rr && q4 == 0) acc[5] = fma(lams[i] * lams[j], norm2(g), acc[5]);
  }
  auto dot = [](double &a, zd x, zd y) { a = fma(x.re, y.re, fma(-x.im, y.im, a)); };   // a += Re(x y)
  for (int e = t; e < rr; e += nt) {
    const int i = e % r, j = e / r, et = i * r + j;
    const zd w = W[et], g = Gam[e], h = B[e], ht = B[et];
    dot(acc[0], w, h);
    dot(acc[1], W2[et], B[rr + e]);
    dot(acc[2], w, B[3 * rr + e]);
    dot(acc[3], w, B[4 * rr + e]);
    dot(acc[4], w, B[5 * rr + e]);
    acc[7] = fma(lams[i] * lams[j], norm2(g), acc[7]);
    if (i == j) acc[6] = fma(lams[i], g.re, acc[6]);
    mx[0] = fmax(mx[0], norm2(i == j ? mk<double>(g.re - 1.0, g.im) : g));
    mx[1] = fmax(mx[1], norm2(h - conj(ht)));
    mx[2] = fmax(mx[2], norm2(h));
  }
#pragma unroll
  for (int x = 0; x < NSUM; ++x) {
    double v = acc[x];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) part[x][wp] = v;
  }
#pragma unroll
  for (int x = 0; x < NMAX; ++x) {   // not negative: ordered as integers, which run at full rate
    unsigned long long v = __double_as_longlong(mx[x]);
    for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
    if (lane == 0) pmax[x][wp] = v;
  }
  __syncthreads();
  if (t < NSUM) {
    double v = 0.0;
    for (int w = 0; w < nt / 32; ++w) v += part[t][w];
    tot[t] = v;
  }
  __syncthreads();
  if (t < 9) {
    const double q = 1.0 - p;
    double v = 0.0;
    if (t == 0) v = q * tot[0];
    else if (t <= 3) v = q * tot[t + 1];
    else if (t == 4) v = p * p * inv_n + 2.0 * p * q * inv_n * tot[6] + q * q * tot[7];
    else if (t == 5) v = p + q * tot[6];
    else {
      unsigned long long m[NMAX] = {0, 0, 0};
      for (int w = 0; w < nt / 32; ++w)
        for (int x = 0; x < NMAX; ++x) m[x] = max(m[x], pmax[x][w]);
      const double orth = __longlong_as_double(m[0]), herm = __longlong_as_double(m[1]), g = __longlong_as_double(m[2]);
      v = sqrt(t == 6 ? orth : (t == 7 ? (g > 0 ? herm / g : 0.0) : fmax(0.0, 2.0 * tot[1] - 2.0 * tot[5])));
      if (t == 8) v *= q;
    }
    out[t] = v;
  }
  if (mu)
    for (int i = t; i < r; i += nt) {
      out[16 + i] = p * inv_n + (1.0 - p) * mu[i];
      out[48 + i] = p * inv_n + (1.0 - p) * lams[i];
    }
}
static int obs_final_threads(int r) { return std::max(64, eliminate_threads(r)); }

// ----------------------------------------------------------- controller features
// ||[rho, H]||_F^2 = 2 Tr(Lambda^2 V^*H^2V) - 2 Tr(Lambda G Lambda G); in the Krylov frame H V_1 has
// coordinates t_0 = Tbar e, so V^*H^2V = t_0^H t_0 and only its diagonal is needed.
__global__ void feat_comm_kernel(const zd *__restrict__ T, int K, int ld, const zd *__restrict__ G, int r,
                                 const double *__restrict__ lam, double *__restrict__ feat) {
  __shared__ double red[8];
  double s = 0.0;
  for (int e = threadIdx.x; e < K * r; e += blockDim.x) s += 2.0 * lam[e / K] * lam[e / K] * norm2(T[(size_t)(e / K) * ld + (e % K)]);
  for (int e = threadIdx.x; e < r * r; e += blockDim.x) s -= 2.0 * lam[e % r] * lam[e / r] * norm2(G[e]);
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0;
    for (int w = 0; w < (int)(blockDim.x + 31) / 32; ++w) a += red[w];
    feat[0] = fmax(a, 0.0);
  }
}

// feat[1] = ||G_last - G_0||_F / ||G_0||_F (stage spread), feat[2] = max_i |mu_i - lambda_i| / lambda_max
// (spectral drift of the unprojected rho_{k+1}).
__global__ void feat_final_kernel(const double *__restrict__ mu, const double *__restrict__ lam, int r,
                                  const zd *__restrict__ G0, const zd *__restrict__ Gl, double *__restrict__ feat) {
  // one entry per thread (FP64 issues slowly on this part: a one-thread loop over r^2 entries
  // takes ~0.1 ms), then a block reduction
  __shared__ double red[3][8];
  const int t = threadIdx.x;
  double d = 0, n0 = 0, dr = 0;
  for (int e = t; e < r * r; e += blockDim.x) {
    const int i = e % r, j = e / r;
    const zd a = Gl[e], b = Gl[(size_t)i * r + j];
    const zd h = mk<double>(0.5 * (a.re + b.re), 0.5 * (a.im - b.im));
    d += norm2(h - G0[e]);
    n0 += norm2(G0[e]);
  }
  double lm = 0;
  for (int i = t; i < r; i += blockDim.x) {
    dr = fmax(dr, fabs(mu[i] - lam[i]));
    lm = fmax(lm, lam[i]);
  }
  for (int o = 16; o > 0; o >>= 1) {
    d += __shfl_xor_sync(0xffffffffu, d, o);
    n0 += __shfl_xor_sync(0xffffffffu, n0, o);
    dr = fmax(dr, __shfl_xor_sync(0xffffffffu, dr, o));
    lm = fmax(lm, __shfl_xor_sync(0xffffffffu, lm, o));
  }
  __shared__ double lmax[8];
  if ((t & 31) == 0) { red[0][t >> 5] = d; red[1][t >> 5] = n0; red[2][t >> 5] = dr; lmax[t >> 5] = lm; }
  __syncthreads();
  if (t == 0) {
    double D = 0, N0 = 0, DR = 0, LM = 0;
    for (int w = 0; w < (int)(blockDim.x + 31) / 32; ++w) {
      D += red[0][w]; N0 += red[1][w]; DR = fmax(DR, red[2][w]); LM = fmax(LM, lmax[w]);
    }
    feat[1] = N0 > 0 ? sqrt(D / N0) : 0.0;
    feat[2] = LM > 0 ? DR / LM : 0.0;
  }
}

// Frobenius distance between two states rho_a = Va La Va^*, rho_b (same spectrum Lambda), from
// C = Va^*Vb and the Grams of the stored factors (implicit Cholesky orthonormalisation):
// ||rho_a - rho_b||_F^2 = 2 sum lam^2 - 2 sum_ij lam_i lam_j |Cbar_ij|^2, Cbar = La^{-1} C Lb^{-H}.
__global__ void dist_kernel(const zd *__restrict__ red, int r, const zd *__restrict__ Ga, int lda_,
                            const double *__restrict__ lam, double *__restrict__ out) {
  extern __shared__ zd sd[];
  zd *La = sd, *Xa = sd + r * r, *Lb = sd + 2 * r * r, *Xb = sd + 3 * r * r, *T = sd + 4 * r * r;
  const int t = threadIdx.x;
  const int ldr = 2 * r;   // red: rows 0..r-1 = Va^*Vb, rows r..2r-1 = Vb^*Vb (column-major)
  chol_inv_cta(Ga, lda_, r, La, Xa);
  chol_inv_cta(red + r, ldr, r, Lb, Xb);
  for (int e = t; e < r * r; e += blockDim.x) {   // T = Xa C
    const int i = e % r, j = e / r;
    zd v = mk<double>(0, 0);
    for (int m = 0; m <= i; ++m) fma_(v, Xa[m * r + i], red[(size_t)j * ldr + m]);
    T[e] = v;
  }
  __syncthreads();
  __shared__ double acc[32];
  double s = 0.0;
  for (int e = t; e < r * r; e += blockDim.x) {   // Cbar = T Xb^H
    const int i = e % r, j = e / r;
    zd v = mk<double>(0, 0);
    for (int m = 0; m <= j; ++m) v = v + T[m * r + i] * conj(Xb[m * r + j]);
    s += lam[i] * lam[j] * norm2(v);
  }
  const double a = cta_sum(s, acc);
  if (t == 0) {
    double l2 = 0;
    for (int i = 0; i < r; ++i) l2 += lam[i] * lam[i];
    out[0] = sqrt(fmax(2.0 * l2 - 2.0 * a, 0.0));
    out[1] = sqrt(l2);
  }
}

// Step-doubling distance without cancellation.  With Vbar = V L^{-H}, Vbar_b = V_b L_b^{-H} and
// C = Vbar_b^H Vbar, write Vbar = Vbar_b C + P (P orthogonal to V_b).  Then to second order
//   ||rho - rho_b||_F^2 = ||offdiag(C Lambda C^H)||_F^2 + 2 sum_i lambda_i^2 ||P e_i||^2,
// where the off-diagonal entries are first-order small (no cancellation) and P is formed
// explicitly in N-space by one fused pass (coefficients written here).
__global__ void dist_prep_kernel(const zd *__restrict__ red, int r, const zd *__restrict__ Gb,
                                 const zd *__restrict__ Lcur, int ldl, const double *__restrict__ lam,
                                 zd *__restrict__ coef, double *__restrict__ out) {
  extern __shared__ zd sd[];
  zd *Lb = sd, *Xb = sd + r * r, *Xc = sd + 2 * r * r, *T = sd + 3 * r * r, *C = sd + 4 * r * r, *Lc = sd + 5 * r * r;
  const int t = threadIdx.x;
  const int ldr = 2 * r;   // red rows 0..r-1: V_b^* V
  for (int e = t; e < r * r; e += blockDim.x) Lc[e] = Lcur[(size_t)(e / r) * ldl + (e % r)];
  __syncthreads();
  chol_inv_cta(Gb, r, r, Lb, Xb);
  tri_inv_cta(Lc, r, Xc);   // Xc = Lc^{-1} from the current factor's Cholesky factor
  for (int e = t; e < r * r; e += blockDim.x) {   // T = Xb (V_b^* V)
    const int i = e % r, j = e / r;
    zd v = mk<double>(0, 0);
    for (int m = 0; m <= i; ++m) fma_(v, Xb[m * r + i], red[(size_t)j * ldr + m]);
    T[e] = v;
  }
  __syncthreads();
  for (int e = t; e < r * r; e += blockDim.x) {   // C = T Xc^H
    const int i = e % r, j = e / r;
    zd v = mk<double>(0, 0);
    for (int m = 0; m <= j; ++m) v = v + T[m * r + i] * conj(Xc[m * r + j]);
    C[e] = v;
  }
  __syncthreads();
  // coefficients of P = V Xc^H - V_b (Xb^H C), column-major (2r x r, ld 2r)
  for (int e = t; e < r * r; e += blockDim.x) {
    const int i = e % r, j = e / r;
    coef[(size_t)j * 2 * r + i] = conj(Xc[i * r + j]);                  // (Xc^H)_{ij}
    zd v = mk<double>(0, 0);
    for (int m = i; m < r; ++m) v = v + conj(Xb[i * r + m]) * C[j * r + m];   // (Xb^H)_{im} C_{mj}
    coef[(size_t)j * 2 * r + r + i] = mk<double>(-v.re, -v.im);
  }
  // off-diagonal part of C Lambda C^H
  __shared__ double acc[32];
  double s = 0.0;
  for (int e = t; e < r * r; e += blockDim.x) {
    const int i = e % r, j = e / r;
    if (i == j) continue;
    zd v = mk<double>(0, 0);
    for (int m = 0; m < r; ++m) v = v + lam[m] * (C[m * r + i] * conj(C[m * r + j]));
    s += norm2(v);
  }
  const double a = cta_sum(s, acc);
  if (t == 0) {
    double l2 = 0;
    for (int i = 0; i < r; ++i) l2 += lam[i] * lam[i];
    out[0] = a;
    out[1] = l2;
  }
}

__global__ void dist_final_kernel(const zd *__restrict__ PP, int r, const double *__restrict__ lam, double *__restrict__ out) {
  if (threadIdx.x != 0) return;
  double s = out[0];
  for (int i = 0; i < r; ++i) s += 2.0 * lam[i] * lam[i] * PP[(size_t)i * r + i].re;
  out[2] = sqrt(fmax(s, 0.0));
  out[3] = sqrt(out[1]);
}

// ---------------------------------------------------------- rank truncation
// dst (N x k, row-major) = the first k columns of src (N x r, row-major).
template <typename T>
__global__ void keep_cols_kernel(const cx<T> *__restrict__ src, int r, cx<T> *__restrict__ dst, int k, long long N) {
  const long long total = N * k;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total; e += (long long)gridDim.x * blockDim.x)
    dst[e] = src[(e / k) * r + e % k];
}

// ---------------------------------------------------------- Householder route
// Compact-WY form Q = I - U T U^H of the r Householder reflectors that triangularise the
// orthonormal factor V (Sec. 3.4, eq. Householder-mat), reconstructed from V itself: with
// D = diag(d), d_i = -conj(V_ii)/|V_ii| (so no cancellation on the diagonal), the top block
// B = I - V_top D has an unpivoted LU factorisation B = L_u R_u, and
//   U = ([I; 0] - V D) R_u^{-1} (unit lower trapezoidal, U_top = L_u),  T = R_u L_u^{-H},
// which gives Q[:, :r] = V D and Q^H V = [D^{-1}; 0].  The complement V^ is Q[:, r:].
template <typename T>
__global__ void top_block_kernel(const cx<T> *__restrict__ V, int r, zd *__restrict__ Vt) {
  for (int e = threadIdx.x; e < r * r; e += blockDim.x) {
    const int b = e / r, c = e % r;   // row b, column c of V (rows < r only)
    const cx<T> v = V[(size_t)b * r + c];
    Vt[(size_t)c * r + b] = mk<double>((double)v.re, (double)v.im);
  }
}

// One CTA, r <= 32: D, L_u, R_u, R_u^{-1}, T and the coefficient -D R_u^{-1} of the U pass.
__global__ void hh_setup_kernel(const zd *__restrict__ Vt, int r, zd *__restrict__ D, zd *__restrict__ Rinv,
                                zd *__restrict__ T, zd *__restrict__ Cu, int *status) {
  extern __shared__ zd sh[];
  zd *B = sh, *Lu = sh + r * r, *Ru = sh + 2 * r * r, *Li = sh + 3 * r * r;   // Li = L_u^{-1}
  const int t = threadIdx.x;
  if (t < r) {
    const zd v = Vt[(size_t)t * r + t];
    const double a = sqrt(norm2(v));
    D[t] = a > 0 ? mk<double>(-v.re / a, v.im / a) : mk<double>(-1, 0);
  }
  __syncthreads();
  for (int e = t; e < r * r; e += blockDim.x) {
    const int i = e % r, j = e / r;
    B[e] = mk<double>(i == j ? 1.0 : 0.0, 0) - Vt[(size_t)j * r + i] * D[j];
  }
  __syncthreads();
  if (t == 0) {
    // Doolittle LU without pivoting: B = Lu Ru, Lu unit lower
    bool bad = false;
    for (int k = 0; k < r; ++k) {
      for (int j = k; j < r; ++j) {
        zd s = B[(size_t)j * r + k];
        for (int m = 0; m < k; ++m) s = s - Lu[(size_t)m * r + k] * Ru[(size_t)j * r + m];
        Ru[(size_t)j * r + k] = s;
      }
      const zd piv = Ru[(size_t)k * r + k];
      const double pn = norm2(piv);
      if (!(pn > 1e-300)) bad = true;
      for (int i = 0; i < r; ++i) {
        if (i < k) { Lu[(size_t)k * r + i] = mk<double>(0, 0); continue; }
        if (i == k) { Lu[(size_t)k * r + i] = mk<double>(1, 0); continue; }
        zd s = B[(size_t)k * r + i];
        for (int m = 0; m < k; ++m) s = s - Lu[(size_t)m * r + i] * Ru[(size_t)k * r + m];
        Lu[(size_t)k * r + i] = mk<double>((s.re * piv.re + s.im * piv.im) / pn, (s.im * piv.re - s.re * piv.im) / pn);
      }
      for (int i = k + 1; i < r; ++i) Ru[(size_t)k * r + i] = mk<double>(0, 0);
    }
    if (bad && status) atomicOr(status, ST_RANK);
    // Rinv = Ru^{-1} (upper): column j by back substitution
    for (int j = 0; j < r; ++j)
      for (int i = r - 1; i >= 0; --i) {
        zd s = mk<double>(i == j ? 1.0 : 0.0, 0);
        for (int m = i + 1; m < r; ++m) s = s - Ru[(size_t)m * r + i] * Rinv[(size_t)j * r + m];
        const zd d = Ru[(size_t)i * r + i];
        const double dn = norm2(d);
        Rinv[(size_t)j * r + i] = (i > j) ? mk<double>(0, 0)
                                          : mk<double>((s.re * d.re + s.im * d.im) / dn, (s.im * d.re - s.re * d.im) / dn);
      }
    // Li = Lu^{-1} (unit lower): column j by forward substitution
    for (int j = 0; j < r; ++j)
      for (int i = 0; i < r; ++i) {
        if (i < j) { Li[(size_t)j * r + i] = mk<double>(0, 0); continue; }
        zd s = mk<double>(i == j ? 1.0 : 0.0, 0);
        for (int m = j; m < i; ++m) s = s - Lu[(size_t)m * r + i] * Li[(size_t)j * r + m];
        Li[(size_t)j * r + i] = s;
      }
  }
  __syncthreads();
  // T = Ru Lu^{-H} = Ru Li^H;  Cu = -D Rinv (row i of Rinv scaled by d_i)
  for (int e = t; e < r * r; e += blockDim.x) {
    const int i = e % r, j = e / r;
    zd s = mk<double>(0, 0);
    for (int m = 0; m < r; ++m) s = s + Ru[(size_t)m * r + i] * conj(Li[(size_t)m * r + j]);
    T[e] = s;
    Cu[e] = mk<double>(-1, 0) * (D[i] * Rinv[e]);
  }
}

// U[0:r, :] += Rinv (rows of the N x r row-major block)
template <typename T>
__global__ void add_top_kernel(cx<T> *__restrict__ U, int r, const zd *__restrict__ Rinv) {
  for (int e = threadIdx.x; e < r * r; e += blockDim.x) {
    const int b = e / r, c = e % r;
    const zd a = Rinv[(size_t)c * r + b];
    U[(size_t)b * r + c] = U[(size_t)b * r + c] + mk<T>((T)a.re, (T)a.im);
  }
}

__global__ void diag_conj_c_kernel(const double *__restrict__ lam, int r, double kappa, int model, zd *__restrict__ Dc,
                                   const zd *__restrict__ K1, zd *__restrict__ Cq) {
  // Dc = diag(conj c), Cq = -K1 diag(conj c)
  for (int e = threadIdx.x; e < r * r; e += blockDim.x) {
    const int i = e % r, j = e / r;
    const zd cc = conj(c_factor(lam[j], kappa, model));
    Dc[e] = (i == j) ? cc : mk<double>(0, 0);
    Cq[e] = mk<double>(-1, 0) * (K1[e] * cc);
  }
}

__global__ void x11_from_g_kernel(const zd *__restrict__ G, int ldg, int r, const double *__restrict__ lam,
                                  double kappa, int model, zd *__restrict__ X11, zd *__restrict__ Gh) {
  for (int e = threadIdx.x; e < r * r; e += blockDim.x) {
    const int i = e % r, j = e / r;
    const zd a = G[(size_t)j * ldg + i], b = G[(size_t)i * ldg + j];
    zd g = mk<double>(0.5 * (a.re + b.re), 0.5 * (a.im - b.im));
    if (i == j) g.im = 0;
    Gh[e] = g;
    X11[e] = x11_factor(lam[i], lam[j], kappa, model) * g;
  }
}

// The six observable Grams (column-major r x r each, in the order obs_final_kernel reads them:
// V^*HV, (HV)^*(HV), V^*V, V^*M_xV, V^*M_yV, V^*M_zV) from the two measured blocks
//   R1 = [HV, CV, ZV, V]^* V  (4r x r, C = M_x + i M_y, Z = M_z) and  R2 = (HV)^*(HV),
// using that H, M_z and V^*V are Hermitian: V^*AV = (A V)^*V conjugate-transposed, and
// V^*M_xV = (K + K^*)/2, V^*M_yV = (K - K^*)/(2i) for K = V^*CV.
__global__ void obs_assemble_kernel(const zd *__restrict__ R1, const zd *__restrict__ R2, int r, zd *__restrict__ out) {
  const int ld = 4 * r;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < r * r; e += gridDim.x * blockDim.x) {
    const int i = e % r, j = e / r;   // entry (i, j) of every block
    auto blkT = [&](int m, int a, int b) { return conj(R1[(size_t)a * ld + m * r + b]); };   // (block m)^*: entry (a, b)
    const zd K = blkT(1, i, j), Kt = blkT(1, j, i);
    out[0 * r * r + e] = blkT(0, i, j);
    out[1 * r * r + e] = R2[(size_t)j * r + i];
    out[2 * r * r + e] = R1[(size_t)j * ld + 3 * r + i];
    out[3 * r * r + e] = mk<double>(0.5 * (K.re + Kt.re), 0.5 * (K.im - Kt.im));
    // (K - K^*)/(2i): K - conj(K^T) = (K.re - Kt.re) + i (K.im + Kt.im); divided by 2i
    out[4 * r * r + e] = mk<double>(0.5 * (K.im + Kt.im), -0.5 * (K.re - Kt.re));
    out[5 * r * r + e] = blkT(2, i, j);
  }
}

void launch_obs_final(const double *red, int r, const double *lam, double *out, cudaStream_t st) {
  ::lrei::count_launch();
  obs_final_kernel<<<1, obs_final_threads(r), 4 * r * r * sizeof(zd), st>>>(red, r, lam, out, 0.0, 0.0, nullptr);
}

}  // namespace lrei

using namespace lrei;

struct lrei_ctx {
  int dev = 0, nsm = 0;
  int n = 0;
  long long N = 0;
  int r_max = 0, r = 0;
  int model = 0, prec = 0;
  double kappa = 0.0;      // damping of the stored low-rank state: (1 - werner_p) kappa0
  double kappa0 = 0.0;     // damping of the equation (lrei_create)
  double werner_p = 0.0;   // weight of the identity part of rho (lrei_set_werner)
  bool fp64 = true;
  size_t elem = 16;
  cudaStream_t user = nullptr, st = nullptr;
  cudaEvent_t ev_in = nullptr, ev_out = nullptr;
  // second stream of the RK step: the stage algebra of stage j runs on it while the N-length
  // passes of the later Krylov blocks run on st (events: fork, Krylov block j done, join)
  cudaStream_t st2 = nullptr;
  cudaEvent_t ev_fork = nullptr, ev_join = nullptr, ev_inv = nullptr, ev_kry[4] = {};
  int nsm_pass = 0;   // SMs the N-length passes of the RK step use (the rest serve the stage algebra)
  int eig_sweeps = 30;   // FP64 Jacobi sweep limit of each partial eigendecomposition
  ModelArgs M;
  int KM = 0;   // leading dimension / capacity of the small k x k arrays
  // N x r blocks
  void *V = nullptr;
  void *blk[MAXB] = {};
  int nblk = 0;
  void *Sbuf = nullptr;   // S = H Q_l of the current Krylov block
  // device workspace
  double *partial = nullptr;
  double *red = nullptr;
  void *coef_scratch = nullptr;
  zd *Gam = nullptr, *L = nullptr, *Li = nullptr, *Tr = nullptr, *Chat = nullptr, *Tbar = nullptr, *Cc = nullptr, *GR = nullptr,
     *Lr = nullptr, *Ainv = nullptr, *coefQ = nullptr, *Bs = nullptr, *Dm = nullptr, *L22 = nullptr, *Mm = nullptr,
     *Uf = nullptr, *Vf = nullptr, *Yc = nullptr, *ts = nullptr, *G = nullptr, *X11 = nullptr, *Gh = nullptr;
  zd *ys[5] = {}, *zs[4] = {}, *wsv[4] = {};
  zd *yfin = nullptr;
  double *lam0_dev = nullptr, *mu_dev = nullptr, *dt_dev = nullptr, *obs_dev = nullptr, *feat_dev = nullptr;
  int *status_dev = nullptr, *dead_dev = nullptr;
  void *eig_ws = nullptr;
  int *status_host = nullptr;
  double *obs_host = nullptr;
  std::vector<double> lam0;
  double t = 0.0;
  double dt_cur = 0.0;
  bool has_state = false;
  // graph cache for one step of a given scheme (the captured graph and its instance)
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t gexec = nullptr;
  int nsm_use = 0;   // SMs the N-length passes spread over (all of them unless a batch shares the GPU)
  int g_scheme = -1, g_r = -1;
  long long g_nodes = 0;
  long long launches = 0, cnt0 = 0;
  int last_status = 0;
  // allocation list
  std::vector<void *> allocs;
  // Adams-Bashforth state: history of raw (V_l, Y_l = H V_l) pairs, most recent first
  int ab_m = 0;            // steps of the scheme whose history is held (0 = none)
  double ab_dt = 0.0;
  std::vector<void *> ab_free;
  std::vector<std::pair<void *, void *>> ab_hist;
  void *abQ[8] = {};       // Q_1 .. Q_{2m-1} of the AB basis (Q_0 = V)
  zd *Rraw = nullptr, *Bbar = nullptr, *tys[4] = {};
  int *dead_frame = nullptr;   // frame columns decoupled as numerically dependent (AB basis)
  // two-spin reduced density matrices: pair bit positions and per-pair results (device)
  int *rdm_pairs = nullptr;
  double *rdm_out = nullptr;
  size_t partial_doubles = 0;   // capacity of `partial`
  bool ab_alloc = false;
  // adaptive step controller
  int ctrl_judge_every = 8, ctrl_judge_learned = 32, ctrl_record = 0;
  double ctrl_h = 0.0, ctrl_safety = 1.0, ctrl_calib = -1.0;
  long long st_accepted = 0, st_rejected = 0, st_judged = 0, st_rk4 = 0;
  double st_err_judged = 0.0;
  void *Vsave = nullptr, *Vbig = nullptr;
  zd *Gsave = nullptr, *Lsave = nullptr, *Gbig = nullptr;
  double *dist_dev = nullptr, *host_small = nullptr;
  std::vector<double> records;
  lrei_mlp *net = nullptr;
  float *net_x = nullptr, *net_y = nullptr, *net_host = nullptr;
  int learned_fallback = 0;
  double learn_corr = -1.0;   // judged error / network estimate at the last judge (learned rule)
};

namespace {

int dalloc(lrei_ctx *c, void **p, size_t bytes) {
  cudaError_t e = cudaMalloc(p, bytes ? bytes : 16);
  if (e != cudaSuccess) return LREI_ERR_OOM;
  c->allocs.push_back(*p);
  // zeroed on the context's stream, so the zeros land before any later work of the context
  // (a memset on the legacy stream is not ordered with a non-blocking stream)
  if (cudaMemsetAsync(*p, 0, bytes ? bytes : 16, c->st) != cudaSuccess) return LREI_ERR_CUDA;
  return LREI_OK;
}
template <typename P>
int dalloc_t(lrei_ctx *c, P **p, size_t bytes) {
  void *q = nullptr;
  int rc = dalloc(c, &q, bytes);
  *p = reinterpret_cast<P *>(q);
  return rc;
}

int status_to_code(int st) {
  if (st & ST_NONFINITE) return LREI_ERR_NONFINITE;
  if (st & ST_TIMEOUT) return LREI_ERR_TIMEOUT;
  if (st & ST_RANK) return LREI_ERR_RANK;
  if (st & (ST_EIG_NOCONV | ST_EIG_RESID)) return LREI_ERR_EIG_NOCONV;
  if (st & ST_TRACE) return LREI_ERR_TRACE;
  return LREI_OK;
}

// Order the internal stream after the caller's stream, and back.
void enter(lrei_ctx *c) {
  c->cnt0 = launch_counter();
  cudaEventRecord(c->ev_in, c->user);
  cudaStreamWaitEvent(c->st, c->ev_in, 0);
}
void leave(lrei_ctx *c) {
  c->launches += launch_counter() - c->cnt0;
  c->cnt0 = launch_counter();
  cudaEventRecord(c->ev_out, c->st);
  cudaStreamWaitEvent(c->user, c->ev_out, 0);
}

const zd ONE = {1.0, 0.0}, ZERO = {0.0, 0.0}, MONE = {-1.0, 0.0};

double tol_rc(const lrei_ctx *c) { return c->fp64 ? 1e-26 : 1e-13; }
const double TOL_GAM = 1e-6;

// One tall-skinny pass + deterministic reduction of its Gram into c->red.
int ts_pass(lrei_ctx *c, TSArgs a, int nsm = 0) {
  a.N = c->N;
  a.r = c->r;
  a.partial = c->partial;
  a.coef_scratch = c->coef_scratch;
  a.status = c->status_dev;
  a.red = c->red;
  int g = launch_ts(c->fp64, c->M, a, nsm > 0 ? nsm : c->nsm_use, c->st);
  if (g < 0) return LREI_ERR_ARG;
  if (g > 0) launch_reduce(c->partial, g, (int)ts_partial_doubles(a.gram_left, c->r), c->red, c->st);
  return LREI_OK;
}

void *qblock(lrei_ctx *c, int m) { return m == 0 ? c->V : c->blk[m - 1]; }

// Gamma[0:r,0:r] <- red (V^*V), L[0:r,0:r] <- chol.
void set_gamma00(lrei_ctx *c) {
  const int r = c->r, KM = c->KM;
  sm_herm_copy(reinterpret_cast<zd *>(c->red), r, r, c->Gam, KM, c->st);
  sm_chol(c->Gam, KM, r, c->L, KM, TOL_GAM, 1, c->dead_dev, c->status_dev, 1, c->st);
}

// Li[0:r,0:r] <- L[0:r,0:r]^{-1}, on stream st.  Li is the inverse of the frame's Cholesky factor L (lower triangular,
// well conditioned: the frame's blocks are normalised or their columns scaled by L itself), kept block by block, so that
// a triangular solve is a product spread over the GPU (about 4 us) instead of a chain of k steps in
// one warp (24 us at k = 16..64).  Recomputed from L in every step, so a step depends on the stored L only.
void start_inverse(lrei_ctx *c, cudaStream_t st) {
  const int r = c->r, KM = c->KM;
  sm_set_identity(c->Li, KM, r, r, st);
  sm_trsv('N', c->L, KM, r, c->Li, KM, r, st);
}

// The frame extended by block Q_i (k = i r earlier columns), from its measured Gram column in red: the new rows of L
// and of its inverse.  ref: the squared norms the pivots are judged against (NULL: the largest diagonal entry).
void extend_frame(lrei_ctx *c, int k, bool keep_dead, int *dead_frame, const zd *ref, int ldref) {
  const int r = c->r, KM = c->KM, ldr = k + r;
  cudaStream_t st = c->st;
  const zd *red = reinterpret_cast<const zd *>(c->red);
  zd *L22 = c->L + (size_t)k * KM + k, *I22 = c->Li + (size_t)k * KM + k;
  sm_gemm('N', 'N', k, r, k, ONE, c->Li, KM, red, ldr, ZERO, c->Bs, KM, st);                       // Bs = L^{-1} Gamma_col
  sm_gemm_herm('C', 'N', r, k, MONE, c->Bs, KM, c->Bs, KM, ONE, red + k, ldr, c->Dm, r, st);       // Schur complement
  sm_chol(c->Dm, r, r, L22, KM, TOL_GAM, keep_dead ? 0 : 1, c->dead_dev, c->status_dev, 0, st, ref, ldref, I22, KM);
  ::lrei::count_launch();
  store_lrows_kernel<<<8, 256, 0, st>>>(c->Bs, KM, r, k, c->dead_dev, c->L, KM, keep_dead ? 1 : 0, dead_frame);
  // rows k.. of the inverse: -L22^{-1} (L21 L11^{-1})
  sm_gemm('N', 'N', r, k, k, ONE, c->L + k, KM, c->Li, KM, ZERO, c->Tr, r, st);
  sm_gemm('N', 'N', r, k, r, MONE, I22, KM, c->Tr, r, ZERO, c->Li + k, KM, st);
}

// Stage j of an RK step, on stream st2: the stage quantities in the orthonormal frame (G_j, X11,
// W_j, Z_j), the stage matrix of K_{j+2} (or of rho_{k+1} for the last stage) and its top-r
// eigenpairs.  It needs the frame of Q_0..Q_{j+1} only: with a = (j+2) r and b = (j+1) r,
// Tbar[0:a, 0:b] = L_a^H Chat[0:a, 0:b] L_b^{-H}, because L is lower triangular and H Q_m lies
// in span(Q_0..Q_{m+1}); for the same reason stage j adds the last r columns only (the entries below them
// are zero, set at the step's start).
void enqueue_stage(lrei_ctx *c, const Tableau &tb, int j, cudaStream_t st2) {
  const int s = tb.s, r = c->r, KM = c->KM, K = (s + 1) * r;
  const int a = (j + 2) * r, b = (j + 1) * r;
  sm_gemm('N', 'C', a, r, b, ONE, c->Chat, KM, c->Li + (size_t)j * r, KM, ZERO, c->Yc, KM, st2);
  sm_gemm('C', 'N', a, r, a, ONE, c->L, KM, c->Yc, KM, ZERO, c->Tbar + (size_t)j * r * KM, KM, st2);
  sm_hermitize(c->Tbar, KM, b, st2);
  // H V_j in the frame (ys[j] has no rows beyond b)
  sm_gemm('N', 'N', K, r, b, ONE, c->Tbar, KM, c->ys[j], KM, ZERO, c->ts, KM, st2);
  sm_gemm('C', 'N', r, r, b, ONE, c->ys[j], KM, c->ts, KM, ZERO, c->G, r, st2);
  ::lrei::count_launch();
  stage_xwz_kernel<<<dim3(r, (K + 31) / 32), 256, 2 * r * sizeof(zd), st2>>>(
      c->G, r, c->lam0_dev, c->kappa, c->model, c->ys[j], c->ts, K, KM, c->X11, c->zs[j], c->wsv[j], j == 0 ? c->Gh : nullptr);
  if (j == 0) {
    ::lrei::count_launch();
    feat_comm_kernel<<<1, 256, 0, st2>>>(c->ts, K, KM, c->Gh, r, c->lam0_dev, c->feat_dev);
  }
  StageCoefs C{};
  C.nterms = j + 1;
  const bool last = (j + 1 == s);
  for (int l = 0; l <= j; ++l) C.c[l] = last ? tb.b[l] : tb.a[j + 1][l];
  StagePtrs P{};
  for (int l = 0; l <= j; ++l) {
    P.y[l] = c->ys[l];
    P.z[l] = c->zs[l];
    P.w[l] = c->wsv[l];
  }
  const int nf = r * (1 + 2 * (j + 1));
  const int kk = last ? K : (j + 2) * r;
  ::lrei::count_launch();
  stage_factors_kernel<<<64, 256, 0, st2>>>(P, C, c->lam0_dev, c->dt_dev, r, K, KM, c->Uf, c->Vf);
  sm_gemm_herm('N', 'C', kk, nf, ONE, c->Uf, KM, c->Vf, KM, ZERO, c->Mm, KM, c->Mm, KM, st2);
  zd *dst = last ? c->yfin : c->ys[j + 1];   // rows beyond kk: zero, set at the step's start
  sm_eig_topr(c->Mm, KM, kk, r, dst, KM, c->mu_dev, c->eig_ws, c->status_dev, st2, c->eig_sweeps);
}

// Enqueue one RK step (scheme 0..3) on c->st.  Precondition: Gam/L leading r x r hold V^*V.
// Krylov block l+1 (H.V, the Gram pass, the coefficients, the extension pass, the Cholesky
// extension) runs on st; once it is done, stage l runs on st2 alongside Krylov block l+2.  The
// N-length passes of the Krylov chain leave some SMs to the stage algebra (nsm_pass).  After the
// last stage the streams join and st forms the new factor.
int enqueue_rk_step(lrei_ctx *c, int scheme) {
  const Tableau &tb = kRK[scheme];
  const int s = tb.s, r = c->r, KM = c->KM, K = (s + 1) * r;
  cudaStream_t st = c->st, st2 = c->st2;
  zd *red = reinterpret_cast<zd *>(c->red);
  LREI_CUDA_TRY(cudaEventRecord(c->ev_fork, st));
  LREI_CUDA_TRY(cudaStreamWaitEvent(st2, c->ev_fork, 0));
  // beside the first Krylov block: the inverse of L_00, and the zeros the stages count on
  start_inverse(c, st2);
  LREI_CUDA_TRY(cudaEventRecord(c->ev_inv, st2));
  sm_set_identity(c->ys[0], KM, K, r, st2);
  for (int j = 1; j < s; ++j) sm_zero(c->ys[j], KM, K, r, st2);
  sm_zero(c->yfin, KM, K, r, st2);
  sm_zero(c->Tbar, KM, K, K, st2);
  for (int l = 0; l < s; ++l) {
    const int k = (l + 1) * r, ldr = (l + 2) * r;
    // pass A: S = H Q_l (formed once by the H.V kernel; both passes read it), then
    // P = [Q_0..Q_l]^* S and S^*S
    TSArgs a{};
    a.nq = l + 1;
    a.gram_left = l + 1;
    for (int m = 0; m <= l; ++m) a.q[m] = qblock(c, m);
    launch_hv(c->fp64, c->M, qblock(c, l), c->Sbuf, c->N, r, c->nsm_pass, st, c->status_dev);
    a.src = c->Sbuf;
    a.apply_h = 0;
    a.mode = 0;
    int rc = ts_pass(c, a, c->nsm_pass);
    if (rc) return rc;
    if (l == 0) LREI_CUDA_TRY(cudaStreamWaitEvent(st, c->ev_inv, 0));
    // T = L^{-1} P; the Gram of the projected residual GR = S^*S - P^* Gamma^{-1} P = S^*S - T^*T = Lr Lr^H;
    // A = (Lr^H)^{-1}; Chat column block l = [C; Lr^H], C = Gamma^{-1} P = L^{-H} T; coefQ = -C A
    zd *Cl = c->Chat + (size_t)l * r * KM;
    sm_gemm('N', 'N', k, r, k, ONE, c->Li, KM, red, ldr, ZERO, c->Cc, KM, st);
    sm_gemm_herm('C', 'N', r, k, MONE, c->Cc, KM, c->Cc, KM, ONE, red + k, ldr, c->GR, r, st);
    sm_chol(c->GR, r, r, nullptr, 0, tol_rc(c), 0, c->dead_dev, c->status_dev, 0, st, red + k, ldr, c->Ainv, r, 1,
            Cl + k, KM);
    sm_gemm('C', 'N', k, r, k, ONE, c->Li, KM, c->Cc, KM, ZERO, Cl, KM, st);
    sm_gemm('N', 'N', k, r, r, MONE, Cl, KM, c->Ainv, r, ZERO, c->coefQ, k, st);
    // pass B: Q_{l+1} = S A - Q C A, Gram column [Q_0..Q_l, Q_{l+1}]^* Q_{l+1}
    TSArgs b = a;
    b.mode = 1;
    b.coefS = c->Ainv;
    b.coefQ = c->coefQ;
    b.out = qblock(c, l + 1);
    rc = ts_pass(c, b, c->nsm_pass);
    if (rc) return rc;
    extend_frame(c, k, false, nullptr, nullptr, 0);
    // the frame of Q_0..Q_{l+1} is complete: stage l can run
    LREI_CUDA_TRY(cudaEventRecord(c->ev_kry[l], st));
    LREI_CUDA_TRY(cudaStreamWaitEvent(st2, c->ev_kry[l], 0));
    enqueue_stage(c, tb, l, st2);
  }
  LREI_CUDA_TRY(cudaEventRecord(c->ev_join, st2));
  LREI_CUDA_TRY(cudaStreamWaitEvent(st, c->ev_join, 0));
  // V_{k+1} = Qbar Yfin = Q (L^{-H} Yfin), formed in place over Q_0 = V
  sm_gemm('C', 'N', K, r, K, ONE, c->Li, KM, c->yfin, KM, ZERO, c->coefQ, K, st);
  TSArgs cmb{};
  cmb.nq = s + 1;
  cmb.gram_left = 0;
  for (int m = 0; m <= s; ++m) cmb.q[m] = qblock(c, m);
  cmb.coefQ = c->coefQ;
  cmb.mode = 2;
  cmb.out = c->V;
  int rc = ts_pass(c, cmb);
  if (rc) return rc;
  set_gamma00(c);
  ::lrei::count_launch(); check_small_kernel<<<1, 256, 0, st>>>(c->mu_dev, r, c->Gam, KM, c->status_dev);
  ::lrei::count_launch(); feat_final_kernel<<<1, 256, 0, st>>>(c->mu_dev, c->lam0_dev, r, c->Gh, c->G, c->feat_dev);
  return LREI_OK;
}

int count_kernel_nodes(cudaGraph_t g) {
  size_t n = 0;
  cudaGraphGetNodes(g, nullptr, &n);
  std::vector<cudaGraphNode_t> nodes(n);
  cudaGraphGetNodes(g, nodes.data(), &n);
  int k = 0;
  for (size_t i = 0; i < n; ++i) {
    cudaGraphNodeType t;
    cudaGraphNodeGetType(nodes[i], &t);
    if (t == cudaGraphNodeTypeKernel) ++k;
  }
  return k;
}

int build_graph(lrei_ctx *c, int scheme) {
  if (c->gexec && c->g_scheme == scheme && c->g_r == c->r) return LREI_OK;
  if (c->gexec) {
    cudaGraphExecDestroy(c->gexec);
    c->gexec = nullptr;
  }
  if (c->graph) {
    cudaGraphDestroy(c->graph);
    c->graph = nullptr;
  }
  cudaGraph_t g = nullptr;
  const long long before = launch_counter();
  LREI_CUDA_TRY(cudaStreamBeginCapture(c->st, cudaStreamCaptureModeThreadLocal));
  int rc = enqueue_rk_step(c, scheme);
  cudaError_t e = cudaStreamEndCapture(c->st, &g);
  c->cnt0 += launch_counter() - before;   // recorded into the graph, not launched
  if (rc) {
    if (g) cudaGraphDestroy(g);
    return rc;
  }
  if (e != cudaSuccess) return cuda_fail(e, "capture");
  c->g_nodes = count_kernel_nodes(g);
  e = cudaGraphInstantiate(&c->gexec, g, 0);
  c->graph = g;   // kept: a batch of contexts runs it as a child graph
  if (e != cudaSuccess) return cuda_fail(e, "instantiate");
  c->g_scheme = scheme;
  c->g_r = c->r;
  return LREI_OK;
}

int read_status(lrei_ctx *c) {
  LREI_CUDA_TRY(cudaMemcpyAsync(c->status_host, c->status_dev, sizeof(int), cudaMemcpyDeviceToHost, c->st));
  LREI_CUDA_TRY(cudaStreamSynchronize(c->st));
  int s = *c->status_host;
  c->last_status = s;
  LREI_CUDA_TRY(cudaMemsetAsync(c->status_dev, 0, sizeof(int), c->st));
  return s;
}


// ------------------------------------------------------------ Adams-Bashforth
// LREI-AB_m (paper Sec. 3.8): rho_{k+1} = rho_k + h sum_l b_l f(rho_{k-l}), whose range lies in
// span{V_k, W_k, V_{k-1}, W_{k-1}, ...} = span of the raw blocks [V_k, H V_k, V_{k-1}, H V_{k-1}, ...].
// Those blocks are nearly dependent (consecutive V's differ by O(h)), so they are orthonormalised
// explicitly, block by block, with the same fused passes as the Krylov basis (a Gram of the raw
// block against the basis, then the projected, normalised block with its measured Gram column);
// every history term is then evaluated in the orthonormal frame and one exact Rayleigh-Ritz step
// gives V_{k+1}.
int ab_prepare(lrei_ctx *c) {
  if (c->ab_alloc) return LREI_OK;
  const size_t blk_bytes = (size_t)c->N * c->r_max * c->elem;
  int rc;
  for (int i = 0; i < 8; ++i) {
    void *p = nullptr;
    if ((rc = dalloc(c, &p, blk_bytes))) return rc;
    c->ab_free.push_back(p);
  }
  for (int i = 0; i < 7; ++i)
    if ((rc = dalloc(c, &c->abQ[i], blk_bytes))) return rc;
  const size_t zs = sizeof(zd);
  if ((rc = dalloc_t(c, &c->Rraw, (size_t)c->KM * c->KM * zs))) return rc;
  if ((rc = dalloc_t(c, &c->Bbar, (size_t)c->KM * c->KM * zs))) return rc;
  if ((rc = dalloc_t(c, &c->dead_frame, (size_t)c->KM * sizeof(int)))) return rc;
  for (int i = 0; i < 4; ++i)
    if ((rc = dalloc_t(c, &c->tys[i], (size_t)c->KM * c->r_max * zs))) return rc;
  c->ab_alloc = true;
  return LREI_OK;
}

void ab_clear(lrei_ctx *c) {
  for (auto &e : c->ab_hist) {
    c->ab_free.push_back(e.first);
    c->ab_free.push_back(e.second);
  }
  c->ab_hist.clear();
  c->ab_m = 0;
}

void ab_trim(lrei_ctx *c, int keep) {
  while ((int)c->ab_hist.size() > keep) {
    c->ab_free.push_back(c->ab_hist.back().first);
    c->ab_free.push_back(c->ab_hist.back().second);
    c->ab_hist.pop_back();
  }
}

void *ab_take(lrei_ctx *c) {
  void *p = c->ab_free.back();
  c->ab_free.pop_back();
  return p;
}

// Record (V, H V) of the current state at the front of the history (used by the RK4 start-up).
int ab_push_current(lrei_ctx *c) {
  void *vk = ab_take(c), *yk = ab_take(c);
  LREI_CUDA_TRY(cudaMemcpyAsync(vk, c->V, (size_t)c->N * c->r * c->elem, cudaMemcpyDeviceToDevice, c->st));
  launch_hv(c->fp64, c->M, c->V, yk, c->N, c->r, c->nsm, c->st, c->status_dev);
  c->ab_hist.insert(c->ab_hist.begin(), {vk, yk});
  return LREI_OK;
}

// One block of explicit Gram-Schmidt: raw block i against Q_0..Q_{i-1} (measured Gram), giving
// Q_i = raw_i - Q C (the residual, not normalised: its measured Gram column normalises it in the
// frame), the extended Cholesky factor of Gamma, and the coordinates raw_i = Q [C; I] in R.
// The history blocks are nearly dependent (consecutive states differ by O(h)), so their residuals
// are small; normalising them by a residual Gram formed as S^*S - P^*C would cancel to the
// rounding level of the complex64 Grams, while the Gram of the written residual is measured
// directly.  A residual column that is numerically dependent on the earlier frame (Schur pivot
// below TOL_GAM times its own squared norm) is decoupled: it keeps its projections in L and is
// flagged in dead_frame so that the stage coordinates drop its leftover part.
int orth_block(lrei_ctx *c, int i, const void *src, void *const *qb, zd *R) {
  const int r = c->r, KM = c->KM, k = i * r, ldr = (i + 1) * r;
  cudaStream_t st = c->st;
  zd *red = reinterpret_cast<zd *>(c->red);
  TSArgs a{};
  a.nq = i;
  a.gram_left = i;
  for (int m = 0; m < i; ++m) a.q[m] = qb[m];
  a.src = src;
  a.apply_h = 0;
  a.mode = 0;
  int rc = ts_pass(c, a);
  if (rc) return rc;
  // C = Gamma^{-1} P = L^{-H} L^{-1} P; Q_i = raw_i - Q C
  sm_gemm('N', 'N', k, r, k, ONE, c->Li, KM, red, ldr, ZERO, c->Cc, KM, st);
  sm_gemm('C', 'N', k, r, k, ONE, c->Li, KM, c->Cc, KM, ZERO, R + (size_t)i * r * KM, KM, st);
  sm_gemm('C', 'N', k, r, k, MONE, c->Li, KM, c->Cc, KM, ZERO, c->coefQ, k, st);
  sm_set_identity(c->Ainv, r, r, r, st);
  sm_set_identity(R + (size_t)i * r * KM + k, KM, r, r, st);
  TSArgs b = a;
  b.mode = 1;
  b.out = qb[i];
  b.coefS = c->Ainv;
  b.coefQ = c->coefQ;
  if ((rc = ts_pass(c, b))) return rc;
  // extend the Cholesky factor of Gamma: pivots judged against each column's own squared norm
  extend_frame(c, k, true, c->dead_frame, red + k, ldr);
  return LREI_OK;
}

// One AB_m step.  Precondition: m-1 previous (V, H V) pairs in the history, Gamma_00 = V^*V.
int enqueue_ab_step(lrei_ctx *c, int m) {
  const double *bw = kAB[m - 2];
  const int r = c->r, KM = c->KM, nb = 2 * m, K = nb * r;
  cudaStream_t st = c->st;
  void *vk = ab_take(c), *yk = ab_take(c);
  LREI_CUDA_TRY(cudaMemcpyAsync(vk, c->V, (size_t)c->N * r * c->elem, cudaMemcpyDeviceToDevice, st));
  const void *raw[8];
  raw[0] = c->V;
  raw[1] = yk;
  for (int l = 1; l < m; ++l) {
    raw[2 * l] = c->ab_hist[l - 1].first;
    raw[2 * l + 1] = c->ab_hist[l - 1].second;
  }
  void *qb[8];
  qb[0] = c->V;
  for (int i = 1; i < nb; ++i) qb[i] = c->abQ[i - 1];
  sm_zero(c->Rraw, KM, K, K, st);
  sm_set_identity(c->Rraw, KM, r, r, st);
  LREI_CUDA_TRY(cudaMemsetAsync(c->dead_frame, 0, (size_t)K * sizeof(int), st));
  start_inverse(c, st);
  for (int i = 1; i < nb; ++i) {
    if (i == 1) launch_hv(c->fp64, c->M, c->V, yk, c->N, r, c->nsm, st, c->status_dev);
    const int rc = orth_block(c, i, raw[i], qb, c->Rraw);
    if (rc) return rc;
  }
  // coordinates of the raw blocks in the orthonormal frame Qbar = Q L^{-H}: Bbar = L^H Rraw, without
  // the leftover parts of dead columns
  sm_gemm('C', 'N', K, K, K, ONE, c->L, KM, c->Rraw, KM, ZERO, c->Bbar, KM, st);
  ::lrei::count_launch();
  zero_dead_rows_kernel<<<8, 256, 0, st>>>(c->Bbar, KM, K, K, c->dead_frame);
  for (int l = 0; l < m; ++l) {
    // the state of step k-l is V_l orthonormalised: vbar = v Lv^{-H}, H vbar = y Lv^{-H}
    const zd *vb = c->Bbar + (size_t)(2 * l) * r * KM, *yb = vb + (size_t)r * KM;
    sm_gemm_herm('C', 'N', r, K, ONE, vb, KM, vb, KM, ZERO, c->G, r, c->G, r, st);
    sm_chol(c->G, r, r, nullptr, 0, 0.0, 0, nullptr, nullptr, 0, st, nullptr, 0, c->Ainv, r, 1);
    sm_gemm('N', 'N', K, r, r, ONE, vb, KM, c->Ainv, r, ZERO, c->ys[l], KM, st);
    sm_gemm('N', 'N', K, r, r, ONE, yb, KM, c->Ainv, r, ZERO, c->tys[l], KM, st);
    sm_gemm('C', 'N', r, r, K, ONE, c->ys[l], KM, c->tys[l], KM, ZERO, c->G, r, st);
    ::lrei::count_launch(); stage_xwz_kernel<<<dim3(r, (K + 31) / 32), 256, 2 * r * sizeof(zd), st>>>(c->G, r, c->lam0_dev, c->kappa, c->model, c->ys[l],
                                                         c->tys[l], K, KM, c->X11, c->zs[l], c->wsv[l],
                                                         l == 0 ? c->Gh : nullptr);
  }
  StageCoefs C{};
  C.nterms = m;
  StagePtrs P{};
  for (int l = 0; l < m; ++l) {
    C.c[l] = bw[l];
    P.y[l] = c->ys[l];
    P.z[l] = c->zs[l];
    P.w[l] = c->wsv[l];
  }
  ::lrei::count_launch(); stage_factors_kernel<<<64, 256, 0, st>>>(P, C, c->lam0_dev, c->dt_dev, r, K, KM, c->Uf, c->Vf);
  sm_gemm_herm('N', 'C', K, r * (1 + 2 * m), ONE, c->Uf, KM, c->Vf, KM, ZERO, c->Mm, KM, c->Mm, KM, st);
  sm_zero(c->yfin, KM, K, r, st);
  sm_eig_topr(c->Mm, KM, K, r, c->yfin, KM, c->mu_dev, c->eig_ws, c->status_dev, st, c->eig_sweeps);
  sm_gemm('C', 'N', K, r, K, ONE, c->Li, KM, c->yfin, KM, ZERO, c->coefQ, K, st);
  TSArgs cmb{};
  cmb.nq = nb;
  cmb.gram_left = 0;
  for (int i = 0; i < nb; ++i) cmb.q[i] = qb[i];
  cmb.coefQ = c->coefQ;
  cmb.mode = 2;
  cmb.out = c->V;
  int rc = ts_pass(c, cmb);
  if (rc) return rc;
  set_gamma00(c);
  ::lrei::count_launch(); check_small_kernel<<<1, 256, 0, st>>>(c->mu_dev, r, c->Gam, KM, c->status_dev);
  c->ab_hist.insert(c->ab_hist.begin(), {vk, yk});
  ab_trim(c, m - 1);
  return LREI_OK;
}


// ----------------------------------------------------------- adaptive stepping
// Plain rule (the adaptive stepping the paper proposes as future work, Sec. 6): the local error
// of an RK4 step is estimated from the spectral drift of the unprojected rho_{k+1} (free, a
// by-product of the final Rayleigh-Ritz step) times a calibration factor; every judge_every-th
// step, and after any rejection, the estimate is replaced by step doubling (one step of h
// against two of h/2, error = 16/15 ||rho_h - rho_{h/2,h/2}||_F / ||rho||_F), which also
// recalibrates the drift factor.  h_new = h clip(0.9 (tol/err)^(1/5), 0.2, 5); a step whose
// error exceeds tol is rejected and retried.  The learned rule replaces the calibrated drift by
// the controller network's estimate of the step's local error (from the step's features: the
// spectrum, the drift, h, ||[rho,H]||^2, the stage spread, kappa, the model, tol, r), so it needs
// the step-doubling judge four times less often (every 4 judge_every steps, after a rejection,
// and when no estimate is available).  Its estimate is scaled by a correction factor refitted at
// every judge (judged error / network estimate), so a shift of the whole error scale (another
// system size, another tolerance) is absorbed at the first judge and the network only has to
// follow the variation between judges.  The same formula turns either estimate into the next h.
// A judge that finds the error more than 3x above the corrected estimate hands control to the
// plain rule for the next 16 steps; an estimate more than 10x below the calibrated drift is
// judged before it is used.
constexpr int NFEAT = 40;

int ctrl_prepare(lrei_ctx *c) {
  if (c->Vsave) return LREI_OK;
  const size_t blk = (size_t)c->N * c->r_max * c->elem;
  int rc;
  if ((rc = dalloc(c, &c->Vsave, blk)) || (rc = dalloc(c, &c->Vbig, blk))) return rc;
  const size_t rr = (size_t)c->r_max * c->r_max * sizeof(zd);
  if ((rc = dalloc_t(c, &c->Gsave, rr)) || (rc = dalloc_t(c, &c->Lsave, rr)) || (rc = dalloc_t(c, &c->Gbig, rr)))
    return rc;
  if ((rc = dalloc_t(c, &c->dist_dev, 4 * sizeof(double)))) return rc;
  if ((rc = dalloc_t(c, &c->net_x, NFEAT * sizeof(float))) || (rc = dalloc_t(c, &c->net_y, 64 * sizeof(float))))
    return rc;
  if (cudaMallocHost(&c->host_small, 64 * sizeof(double)) != cudaSuccess) return LREI_ERR_OOM;
  if (cudaMallocHost(&c->net_host, 64 * sizeof(float)) != cudaSuccess) return LREI_ERR_OOM;
  return LREI_OK;
}

void save_state(lrei_ctx *c, void *dst, zd *G, zd *L) {
  const int r = c->r, KM = c->KM;
  cudaMemcpyAsync(dst, c->V, (size_t)c->N * r * c->elem, cudaMemcpyDeviceToDevice, c->st);
  sm_copy(c->Gam, KM, r, r, G, r, c->st);
  if (L) sm_copy(c->L, KM, r, r, L, r, c->st);
}

void restore_state(lrei_ctx *c, const void *src, const zd *G, const zd *L) {
  const int r = c->r, KM = c->KM;
  cudaMemcpyAsync(c->V, src, (size_t)c->N * r * c->elem, cudaMemcpyDeviceToDevice, c->st);
  sm_copy(G, r, r, r, c->Gam, KM, c->st);
  sm_copy(L, r, r, r, c->L, KM, c->st);
}

int set_dt(lrei_ctx *c, double h) {
  c->host_small[32] = h;
  LREI_CUDA_TRY(cudaMemcpyAsync(c->dt_dev, &c->host_small[32], sizeof(double), cudaMemcpyHostToDevice, c->st));
  c->dt_cur = h;
  return LREI_OK;
}

// Reads feat[0..2] (commutator^2, stage spread, drift) and the status word; syncs.
int read_feats(lrei_ctx *c, double *f) {
  LREI_CUDA_TRY(cudaMemcpyAsync(c->host_small, c->feat_dev, 3 * sizeof(double), cudaMemcpyDeviceToHost, c->st));
  const int s = read_status(c);
  for (int i = 0; i < 3; ++i) f[i] = c->host_small[i];
  return s;
}

void build_features(lrei_ctx *c, const double *f, double h, double tol, float *x) {
  for (int i = 0; i < 32; ++i) x[i] = (float)std::log10(i < c->r ? std::fmax(c->lam0[i], 1e-12) : 1e-12) / 12.0f;
  x[32] = (float)(std::log10(std::fmax(f[2], 1e-300)) / 16.0);
  x[33] = (float)(std::log10(h) / 4.0);
  x[34] = (float)(std::log10(std::fmax(f[0], 1e-300)) / 8.0);
  x[35] = (float)(std::log10(std::fmax(f[1], 1e-300)) / 8.0);
  x[36] = (float)c->kappa;
  x[37] = (float)c->model;
  x[38] = (float)(std::log10(tol) / 16.0);
  x[39] = (float)c->r / 32.0f;
}

// Step doubling from the saved state: returns the relative error estimate of the h step and
// leaves the state at the result of the two h/2 steps.
int judge(lrei_ctx *c, double h, double *err) {
  const int r = c->r;
  save_state(c, c->Vbig, c->Gbig, nullptr);
  restore_state(c, c->Vsave, c->Gsave, c->Lsave);
  set_dt(c, 0.5 * h);
  LREI_CUDA_TRY(cudaGraphLaunch(c->gexec, c->st));
  LREI_CUDA_TRY(cudaGraphLaunch(c->gexec, c->st));
  c->launches += 2 * c->g_nodes;
  TSArgs a{};
  a.nq = 1;
  a.gram_left = 1;
  a.q[0] = c->Vbig;
  a.src = c->V;
  a.apply_h = 0;
  a.mode = 0;
  int rc = ts_pass(c, a);
  if (rc) return rc;
  ::lrei::count_launch();
  dist_prep_kernel<<<1, 256, 6 * r * r * sizeof(zd), c->st>>>(reinterpret_cast<zd *>(c->red), r, c->Gbig, c->L, c->KM,
                                                              c->lam0_dev, c->coefQ, c->dist_dev);
  TSArgs p{};
  p.nq = 2;
  p.gram_left = 0;
  p.q[0] = c->V;
  p.q[1] = c->Vbig;
  p.coefQ = c->coefQ;
  p.mode = 2;
  p.out = c->Sbuf;
  if ((rc = ts_pass(c, p))) return rc;
  ::lrei::count_launch();
  dist_final_kernel<<<1, 32, 0, c->st>>>(reinterpret_cast<zd *>(c->red), r, c->lam0_dev, c->dist_dev);
  LREI_CUDA_TRY(cudaMemcpyAsync(c->host_small + 8, c->dist_dev + 2, 2 * sizeof(double), cudaMemcpyDeviceToHost, c->st));
  LREI_CUDA_TRY(cudaStreamSynchronize(c->st));
  *err = (16.0 / 15.0) * c->host_small[8] / std::fmax(c->host_small[9], 1e-300);
  return LREI_OK;
}

// Local error estimate of the learned rule for the step just taken: the network maps the step's
// features to log(err / drift), the ratio of the local error to the spectral drift of the
// unprojected rho_{k+1}.  Returns a negative value when no estimate is available.
int learned_estimate(lrei_ctx *c, const double *f, double hs, double tol, double *err) {
  float x[NFEAT];
  build_features(c, f, hs, tol, x);
  std::memcpy(c->net_host, x, sizeof(x));
  LREI_CUDA_TRY(cudaMemcpyAsync(c->net_x, c->net_host, sizeof(x), cudaMemcpyHostToDevice, c->st));
  int rc = lrei_mlp_forward_on(c->net, c->net_x, 1, c->net_y, c->st);   // on the context's stream
  if (rc) return rc;
  LREI_CUDA_TRY(cudaMemcpyAsync(c->net_host, c->net_y, sizeof(float), cudaMemcpyDeviceToHost, c->st));
  LREI_CUDA_TRY(cudaStreamSynchronize(c->st));
  const double e = std::exp((double)c->net_host[0]) * f[2];
  *err = (std::isfinite(e) && f[2] > 0) ? e : -1.0;
  return LREI_OK;
}

int run_adaptive(lrei_ctx *c, double t_end, double tol, int controller) {
  int rc = build_graph(c, (int)LREI_RK4);
  if (rc) return rc;
  double h = c->ctrl_h > 0 ? c->ctrl_h : 1e-2;
  // below the rounding floor of the stored factor the judged error is noise: never ask for less
  tol = std::fmax(tol, c->fp64 ? LREI_TOL_FLOOR_FP64 : LREI_TOL_FLOOR_MIXED);
  const double h_min = 1e-12 * std::fmax(1.0, std::fabs(t_end));
  int rejected_in_row = 0;
  int since_judge = 1 << 30;   // the first step is judged
  bool last_rejected = false;
  double f[3];
  while (c->t < t_end - 1e-12 * std::fmax(1.0, std::fabs(t_end))) {
    const double hs = std::fmin(h, t_end - c->t);
    save_state(c, c->Vsave, c->Gsave, c->Lsave);
    set_dt(c, hs);
    LREI_CUDA_TRY(cudaGraphLaunch(c->gexec, c->st));
    c->launches += c->g_nodes;
    int sbits = read_feats(c, f);
    if (sbits & (ST_NONFINITE | ST_RANK)) return status_to_code(sbits);
    const double drift = f[2];
    ++since_judge;
    // the learned rule is in charge unless a judged step caught it underestimating the error
    const bool learned = controller == 1 && c->net && c->learned_fallback <= 0;
    double err_net = -1.0;
    if (learned && (rc = learned_estimate(c, f, hs, tol, &err_net))) return rc;
    const int period = learned ? c->ctrl_judge_learned : c->ctrl_judge_every;
    const double err_plain = (c->ctrl_calib > 0 ? c->ctrl_calib : 1.0) * drift;
    // the network's estimate times its correction factor (refitted at every judge)
    const double err_learn = err_net >= 0 ? (c->learn_corr > 0 ? c->learn_corr : 1.0) * err_net : -1.0;
    // an estimate far below the calibrated drift is checked by a judge before it is used
    const bool doubtful = learned && (err_learn < 0 || err_learn < 0.1 * err_plain);
    const bool do_judge = since_judge >= period || last_rejected || c->ctrl_calib < 0 || doubtful;
    double err;
    c->st_rk4 += 1;
    if (do_judge) {
      if ((rc = judge(c, hs, &err))) return rc;
      c->st_rk4 += 2;
      c->st_judged += 1;
      c->st_err_judged = err;
      since_judge = 0;
      if (drift > 0) c->ctrl_calib = err / drift;
      if (learned && err_net > 0) {
        // an estimate more than 3x below the judged error sends control to the plain rule
        if (err_learn > 0 && c->learn_corr > 0 && err > 3.0 * err_learn) c->learned_fallback = 16;
        c->learn_corr = err / err_net;
      }
    } else {
      err = learned ? err_learn : err_plain;
    }
    if (c->ctrl_record) {
      float x[NFEAT];
      build_features(c, f, hs, tol, x);
      for (int i = 0; i < NFEAT; ++i) c->records.push_back(x[i]);
      c->records.push_back(hs);
      c->records.push_back(drift);
      c->records.push_back(do_judge ? err : -1.0);
      c->records.push_back(err <= tol ? 1.0 : 0.0);
    }
    if (c->learned_fallback > 0) --c->learned_fallback;
    const double ratio = std::fmin(5.0, std::fmax(0.2, 0.9 * std::pow(tol / std::fmax(err, 1e-300), 0.2)));
    if (!(err <= tol)) {
      restore_state(c, c->Vsave, c->Gsave, c->Lsave);
      c->st_rejected += 1;
      h = hs * std::fmin(ratio, 0.9);
      last_rejected = true;
      if (++rejected_in_row >= 64 || h < h_min) {
        c->ctrl_h = h;
        return LREI_ERR_STEP;
      }
      continue;
    }
    c->t += hs;
    c->st_accepted += 1;
    rejected_in_row = 0;
    last_rejected = false;
    h = hs * ratio;
    if (h < h_min) {
      c->ctrl_h = h;
      return LREI_ERR_STEP;
    }
  }
  c->ctrl_h = h;
  return LREI_OK;
}

}  // namespace

namespace lrei {
int build_model_args(int n, const void *bonds, const double B[3], ModelArgs *M) {
  const lrei_bonds *J = static_cast<const lrei_bonds *>(bonds);
  if (n < 1 || n > MAX_SPINS) return LREI_ERR_ARG;
  double Bv[3] = {0, 0, 0};
  if (B) for (int i = 0; i < 3; ++i) Bv[i] = B[i];
  for (int i = 0; i < 3; ++i)
    if (!std::isfinite(Bv[i])) return LREI_ERR_NONFINITE;
  const int nb = J ? J->nbonds : 0;
  if (nb < 0 || nb > MAX_BONDS) return LREI_ERR_ARG;
  if (nb > 0 && (!J->site_i || !J->site_j || !J->jxy || !J->jz)) return LREI_ERR_ARG;
  std::memset(M, 0, sizeof(*M));
  M->n = n;
  M->nb = nb;
  M->bx = Bv[0];
  M->by = Bv[1];
  M->bz = Bv[2];
  M->cplx = (Bv[0] != 0.0 || Bv[1] != 0.0) ? 1 : 0;
  double c0 = 0.0;
  for (int b = 0; b < nb; ++b) {
    const int i = J->site_i[b], j = J->site_j[b];
    if (i < 0 || i >= n || j < 0 || j >= n || i == j) return LREI_ERR_ARG;
    if (!std::isfinite(J->jxy[b]) || !std::isfinite(J->jz[b])) return LREI_ERR_NONFINITE;
    // site i is bit n-1-i of the basis index (site 0 = most significant bit)
    M->bi[b] = (uint8_t)(n - 1 - i);
    M->bj[b] = (uint8_t)(n - 1 - j);
    M->mask[b] = (1u << (n - 1 - i)) | (1u << (n - 1 - j));
    M->jxy[b] = J->jxy[b];
    M->jz[b] = J->jz[b];
    c0 += 0.5 * J->jz[b];
  }
  M->c0 = c0;
  return LREI_OK;
}
}  // namespace lrei

extern "C" {

const char *lrei_error_string(int code) {
  switch (code) {
    case LREI_OK: return "ok";
    case LREI_ERR_ARG: return "invalid argument";
    case LREI_ERR_UNSUPPORTED: return "unsupported in this build";
    case LREI_ERR_NONFINITE: return "non-finite value in input or state";
    case LREI_ERR_TRACE: return "spectrum must be >= 0 and sum to 1";
    case LREI_ERR_RANK: return "rank-deficient factor";
    case LREI_ERR_EIG_NOCONV: return "small eigensolver did not converge";
    case LREI_ERR_OOM: return "device allocation failed";
    case LREI_ERR_CUDA: return "CUDA runtime error";
    case LREI_ERR_STATE: return "call out of order";
    case LREI_ERR_TIMEOUT: return "bounded device wait ran out";
    case LREI_ERR_STEP: return "adaptive step size underflow";
    default: return "unknown error";
  }
}

int lrei_create(int n, const lrei_bonds *J, const double B[3], double lambda, lrei_model model,
                lrei_precision prec, int r_max, void *cuda_stream, lrei_ctx **out) {
  if (!out) return LREI_ERR_ARG;
  *out = nullptr;
  if (n < 1 || n > MAX_SPINS || r_max < 1 || r_max > MAX_R || !(lambda >= 0.0) || !std::isfinite(lambda))
    return LREI_ERR_ARG;
  if (model != LREI_QLL && model != LREI_QLLG) return LREI_ERR_ARG;
  if (prec == LREI_MIXED_BF16X) return LREI_ERR_UNSUPPORTED;
  if (prec != LREI_FP64 && prec != LREI_MIXED_C64) return LREI_ERR_ARG;
  if ((long long)r_max > (1LL << n)) return LREI_ERR_ARG;
  ModelArgs Mk;
  const int mrc = build_model_args(n, J, B, &Mk);
  if (mrc != LREI_OK) return mrc;
  lrei_ctx *c = new (std::nothrow) lrei_ctx();
  if (!c) return LREI_ERR_OOM;
  c->M = Mk;
  c->n = n;
  c->N = 1LL << n;
  c->r_max = r_max;
  c->model = model;
  c->prec = prec;
  c->kappa = lambda;
  c->kappa0 = lambda;
  c->fp64 = (prec == LREI_FP64);
  c->elem = c->fp64 ? 16 : 8;
  c->user = reinterpret_cast<cudaStream_t>(cuda_stream);
  int rc = LREI_OK;
  auto fail = [&](int code) {
    lrei_destroy(c);
    return code;
  };
  if (cudaGetDevice(&c->dev) != cudaSuccess) return fail(LREI_ERR_CUDA);
  cudaDeviceGetAttribute(&c->nsm, cudaDevAttrMultiProcessorCount, c->dev);
  if (cudaStreamCreateWithFlags(&c->st, cudaStreamNonBlocking) != cudaSuccess) return fail(LREI_ERR_CUDA);
  if (cudaStreamCreateWithFlags(&c->st2, cudaStreamNonBlocking) != cudaSuccess) return fail(LREI_ERR_CUDA);
  cudaEventCreateWithFlags(&c->ev_in, cudaEventDisableTiming);
  cudaEventCreateWithFlags(&c->ev_out, cudaEventDisableTiming);
  cudaEventCreateWithFlags(&c->ev_fork, cudaEventDisableTiming);
  cudaEventCreateWithFlags(&c->ev_join, cudaEventDisableTiming);
  cudaEventCreateWithFlags(&c->ev_inv, cudaEventDisableTiming);
  for (int i = 0; i < 4; ++i) cudaEventCreateWithFlags(&c->ev_kry[i], cudaEventDisableTiming);
  c->nsm_use = c->nsm;
  // the complex64 N-length passes of the RK step leave one SM in 32 to the stage algebra running
  // beside them (measured at n=20, r=16: 5.55 ms per step against 5.61 with one in 16, 5.88 with
  // one in 8 and 6.25 with none); the FP64 passes are long enough that the stage algebra hides
  // behind them without a reserve
  c->nsm_pass = c->fp64 ? c->nsm_use : c->nsm_use - std::max(1, c->nsm_use / 32);
  if (ts_init() || sm_init()) return fail(LREI_ERR_CUDA);
  {
    const int lim = 100 * 1024;
    if (cudaFuncSetAttribute(hh_setup_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, lim) != cudaSuccess ||
        cudaFuncSetAttribute(dist_prep_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, lim) != cudaSuccess ||
        cudaFuncSetAttribute(dist_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, lim) != cudaSuccess ||
        cudaFuncSetAttribute(obs_final_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, lim) != cudaSuccess)
      return fail(LREI_ERR_CUDA);
  }
  const size_t blk_bytes = (size_t)c->N * r_max * c->elem;
  c->nblk = 4;
  if ((rc = dalloc(c, &c->V, blk_bytes))) return fail(rc);
  for (int i = 0; i < c->nblk; ++i)
    if ((rc = dalloc(c, &c->blk[i], blk_bytes))) return fail(rc);
  if ((rc = dalloc(c, &c->Sbuf, blk_bytes))) return fail(rc);
  c->KM = 8 * r_max;   // RK_s needs (s+1) r <= 5 r, AB_m needs 2 m r <= 8 r
  const int KM = c->KM, R = r_max;
  const size_t zs = sizeof(zd);
  c->partial_doubles = (size_t)(ts_max_grid(c->nsm) + 16) * (MAXB + 1) * R * R * 2;
  if ((rc = dalloc_t(c, &c->partial, c->partial_doubles * sizeof(double)))) return fail(rc);
  if ((rc = dalloc_t(c, &c->rdm_pairs, 2 * LREI_RDM_MAX_PAIRS * sizeof(int)))) return fail(rc);
  if ((rc = dalloc_t(c, &c->rdm_out, (size_t)34 * LREI_RDM_MAX_PAIRS * sizeof(double)))) return fail(rc);
  if ((rc = dalloc_t(c, &c->red, (size_t)(MAXB + 1) * R * R * 2 * sizeof(double)))) return fail(rc);
  if ((rc = dalloc(c, &c->coef_scratch, (size_t)(MAXB + 1) * MAX_R * MAX_R * zs))) return fail(rc);
  zd **kk[] = {&c->Gam, &c->L, &c->Li, &c->Chat, &c->Tbar, &c->Mm};
  for (auto p : kk)
    if ((rc = dalloc_t(c, p, (size_t)KM * KM * zs))) return fail(rc);
  zd **kr[] = {&c->Cc, &c->coefQ, &c->Bs, &c->Yc, &c->Tr, &c->ts, &c->yfin};
  for (auto p : kr)
    if ((rc = dalloc_t(c, p, (size_t)KM * R * zs))) return fail(rc);
  for (int i = 0; i < 5; ++i)
    if ((rc = dalloc_t(c, &c->ys[i], (size_t)KM * R * zs))) return fail(rc);
  for (int i = 0; i < 4; ++i) {
    if ((rc = dalloc_t(c, &c->zs[i], (size_t)KM * R * zs))) return fail(rc);
    if ((rc = dalloc_t(c, &c->wsv[i], (size_t)KM * R * zs))) return fail(rc);
  }
  if ((rc = dalloc_t(c, &c->Uf, (size_t)KM * 9 * R * zs))) return fail(rc);
  if ((rc = dalloc_t(c, &c->Vf, (size_t)KM * 9 * R * zs))) return fail(rc);
  zd **rr[] = {&c->GR, &c->Lr, &c->Ainv, &c->Dm, &c->L22, &c->G, &c->X11, &c->Gh};
  for (auto p : rr)
    if ((rc = dalloc_t(c, p, (size_t)R * R * zs))) return fail(rc);
  if ((rc = dalloc_t(c, &c->lam0_dev, R * sizeof(double)))) return fail(rc);
  if ((rc = dalloc_t(c, &c->mu_dev, R * sizeof(double)))) return fail(rc);
  if ((rc = dalloc_t(c, &c->dt_dev, sizeof(double)))) return fail(rc);
  if ((rc = dalloc_t(c, &c->obs_dev, 128 * sizeof(double)))) return fail(rc);
  if ((rc = dalloc_t(c, &c->feat_dev, 16 * sizeof(double)))) return fail(rc);
  if ((rc = dalloc_t(c, &c->status_dev, sizeof(int)))) return fail(rc);
  if ((rc = dalloc_t(c, &c->dead_dev, R * sizeof(int)))) return fail(rc);
  if ((rc = dalloc(c, &c->eig_ws, sm_eig_ws_bytes(KM, R)))) return fail(rc);
  if (cudaMallocHost(&c->status_host, sizeof(int)) != cudaSuccess) return fail(LREI_ERR_OOM);
  if (cudaMallocHost(&c->obs_host, 128 * sizeof(double)) != cudaSuccess) return fail(LREI_ERR_OOM);
  if (cudaDeviceSynchronize() != cudaSuccess) return fail(LREI_ERR_CUDA);
  *out = c;
  return LREI_OK;
}

int lrei_destroy(lrei_ctx *c) {
  if (!c) return LREI_OK;
  if (c->st) cudaStreamSynchronize(c->st);
  if (c->st2) cudaStreamSynchronize(c->st2);
  if (c->gexec) cudaGraphExecDestroy(c->gexec);
  if (c->graph) cudaGraphDestroy(c->graph);
  for (void *p : c->allocs) cudaFree(p);
  if (c->status_host) cudaFreeHost(c->status_host);
  if (c->obs_host) cudaFreeHost(c->obs_host);
  if (c->ev_in) cudaEventDestroy(c->ev_in);
  if (c->ev_out) cudaEventDestroy(c->ev_out);
  if (c->ev_fork) cudaEventDestroy(c->ev_fork);
  if (c->ev_join) cudaEventDestroy(c->ev_join);
  if (c->ev_inv) cudaEventDestroy(c->ev_inv);
  for (int i = 0; i < 4; ++i)
    if (c->ev_kry[i]) cudaEventDestroy(c->ev_kry[i]);
  if (c->st2) cudaStreamDestroy(c->st2);
  if (c->st) cudaStreamDestroy(c->st);
  delete c;
  return LREI_OK;
}

int lrei_set_state(lrei_ctx *c, const void *V_dev, int r, int ld, int dtype, const double *Lambda_host) {
  NvtxScope nvtx_scope("lrei_set_state");
  if (!c || !V_dev || !Lambda_host) return LREI_ERR_ARG;
  if (r < 1 || r > c->r_max || ld < r || (dtype != LREI_C128 && dtype != LREI_C64)) return LREI_ERR_ARG;
  double sum = 0.0;
  for (int i = 0; i < r; ++i) {
    if (!std::isfinite(Lambda_host[i])) return LREI_ERR_NONFINITE;
    if (Lambda_host[i] < 0.0) return LREI_ERR_TRACE;
    sum += Lambda_host[i];
  }
  if (std::fabs(sum - 1.0) > 1e-12) return LREI_ERR_TRACE;
  enter(c);
  c->r = r;
  c->has_state = false;
  if (c->ab_alloc) ab_clear(c);
  const int KM = c->KM;
  std::vector<double> lam_in(Lambda_host, Lambda_host + r);
  LREI_CUDA_TRY(cudaMemsetAsync(c->status_dev, 0, sizeof(int), c->st));
  LREI_CUDA_TRY(cudaMemsetAsync(c->L, 0, (size_t)KM * KM * sizeof(zd), c->st));
  LREI_CUDA_TRY(cudaMemsetAsync(c->Gam, 0, (size_t)KM * KM * sizeof(zd), c->st));
  LREI_CUDA_TRY(cudaMemsetAsync(c->Chat, 0, (size_t)KM * KM * sizeof(zd), c->st));   // its zero blocks depend on r
  launch_convert(V_dev, dtype == LREI_C64, ld, c->V, c->fp64, c->N, r, c->st);
  launch_check_finite(c->fp64, c->V, c->N, r, c->status_dev, c->st);
  // R^H R = V^*V (Cholesky), rho_0 = Q (R Lambda R^H) Q^*, Q = V R^{-1}
  TSArgs a{};
  a.nq = 0;
  a.gram_left = 0;
  a.src = c->V;
  a.apply_h = 0;
  a.mode = 0;
  int rc = ts_pass(c, a);
  if (rc) { leave(c); return rc; }
  zd *red = reinterpret_cast<zd *>(c->red);
  sm_hermitize(red, r, r, c->st);
  sm_chol(red, r, r, c->L22, r, 1e-24, 1, c->dead_dev, c->status_dev, 1, c->st);
  LREI_CUDA_TRY(cudaMemcpyAsync(c->lam0_dev, lam_in.data(), r * sizeof(double), cudaMemcpyHostToDevice, c->st));
  ::lrei::count_launch(); lhl_kernel<<<(r * r + 31) / 32, 256, 0, c->st>>>(c->L22, r, c->lam0_dev, c->Dm);
  sm_jacobi64(c->Dm, r, r, c->Lr, r, c->mu_dev, 60, 1e-15, c->status_dev, c->st);
  // coefficients R^{-1} E = L^{-H} E
  sm_copy(c->Lr, r, r, r, c->coefQ, r, c->st);
  sm_trsv('C', c->L22, r, r, c->coefQ, r, r, c->st);
  TSArgs cmb{};
  cmb.nq = 1;
  cmb.gram_left = 0;
  cmb.q[0] = c->V;
  cmb.coefQ = c->coefQ;
  cmb.mode = 2;
  cmb.out = c->V;
  rc = ts_pass(c, cmb);
  if (rc) { leave(c); return rc; }
  set_gamma00(c);
  LREI_CUDA_TRY(cudaMemcpyAsync(c->lam0_dev, c->mu_dev, r * sizeof(double), cudaMemcpyDeviceToDevice, c->st));
  c->lam0.assign(r, 0.0);
  LREI_CUDA_TRY(cudaMemcpyAsync(c->lam0.data(), c->mu_dev, r * sizeof(double), cudaMemcpyDeviceToHost, c->st));
  const int s = read_status(c);
  leave(c);
  if (s) return status_to_code(s);
  for (int i = 0; i < r; ++i) {
    if (!std::isfinite(c->lam0[i])) return LREI_ERR_NONFINITE;
    if (c->lam0[i] < -1e-12) return LREI_ERR_TRACE;
    if (c->lam0[i] < 0.0) c->lam0[i] = 0.0;
  }
  // on the context's stream: a plain copy from pageable memory may return before the data lands
  LREI_CUDA_TRY(cudaMemcpyAsync(c->lam0_dev, c->lam0.data(), r * sizeof(double), cudaMemcpyHostToDevice, c->st));
  LREI_CUDA_TRY(cudaStreamSynchronize(c->st));
  c->t = 0.0;
  c->has_state = true;
  return LREI_OK;
}

int lrei_get_state(lrei_ctx *c, void *V_dev_out, double *Lambda_host_out, double *t_out) {
  if (!c) return LREI_ERR_ARG;
  if (!c->has_state) return LREI_ERR_STATE;
  enter(c);
  if (V_dev_out)
    LREI_CUDA_TRY(cudaMemcpyAsync(V_dev_out, c->V, (size_t)c->N * c->r * c->elem, cudaMemcpyDeviceToDevice, c->st));
  leave(c);
  LREI_CUDA_TRY(cudaStreamSynchronize(c->st));
  if (Lambda_host_out) std::memcpy(Lambda_host_out, c->lam0.data(), c->r * sizeof(double));
  if (t_out) *t_out = c->t;
  return LREI_OK;
}

int lrei_step(lrei_ctx *c, double dt, lrei_scheme scheme, int nsteps) {
  NvtxScope nvtx_scope("lrei_step");
  if (!c) return LREI_ERR_ARG;
  if (!c->has_state) return LREI_ERR_STATE;
  if (!std::isfinite(dt) || nsteps < 0) return LREI_ERR_ARG;
  if (scheme < LREI_RK1 || scheme > LREI_AB4) return LREI_ERR_ARG;
  const bool ab = scheme >= LREI_AB2;
  const int m = ab ? (int)scheme - (int)LREI_AB2 + 2 : 0;
  if (ab && 2 * m * c->r > 160) return LREI_ERR_UNSUPPORTED;   // k x k eigensolver limit
  if (nsteps == 0) return LREI_OK;
  enter(c);
  if (dt != c->dt_cur) {
    LREI_CUDA_TRY(cudaMemcpyAsync(c->dt_dev, &dt, sizeof(double), cudaMemcpyHostToDevice, c->st));
    LREI_CUDA_TRY(cudaStreamSynchronize(c->st));
    c->dt_cur = dt;
  }
  int rc = build_graph(c, ab ? (int)LREI_RK4 : (int)scheme);
  if (rc) { leave(c); return rc; }
  if (!ab) {
    for (int i = 0; i < nsteps; ++i) {
      LREI_CUDA_TRY(cudaGraphLaunch(c->gexec, c->st));
      c->launches += c->g_nodes;
    }
  } else {
    if ((rc = ab_prepare(c))) { leave(c); return rc; }
    if (c->ab_m != m || c->ab_dt != dt) {
      ab_clear(c);
      c->ab_m = m;
      c->ab_dt = dt;
    }
    for (int i = 0; i < nsteps; ++i) {
      if ((int)c->ab_hist.size() < m - 1) {
        // start-up: RK4 steps (global order 4 >= m - 1), recording the history they pass through
        if ((rc = ab_push_current(c))) { leave(c); return rc; }
        LREI_CUDA_TRY(cudaGraphLaunch(c->gexec, c->st));
        c->launches += c->g_nodes;
      } else {
        if ((rc = enqueue_ab_step(c, m))) { leave(c); return rc; }
      }
    }
  }
  const int s = read_status(c);
  leave(c);
  c->t += dt * nsteps;
  return status_to_code(s);
}

int lrei_step_adaptive(lrei_ctx *c, double t_end, double tol, int controller) {
  NvtxScope nvtx_scope("lrei_step_adaptive");
  if (!c) return LREI_ERR_ARG;
  if (!c->has_state) return LREI_ERR_STATE;
  if (!std::isfinite(t_end) || !(tol > 0) || (controller != 0 && controller != 1)) return LREI_ERR_ARG;
  if (controller == 1 && !c->net) return LREI_ERR_STATE;
  if (t_end <= c->t) return LREI_OK;
  enter(c);
  int rc = ctrl_prepare(c);
  if (!rc) rc = run_adaptive(c, t_end, tol, controller);
  leave(c);
  return rc;
}

int lrei_controller_config(lrei_ctx *c, int judge_every, int record, double h0) {
  if (!c || judge_every < 1) return LREI_ERR_ARG;
  c->ctrl_judge_every = judge_every;
  c->ctrl_judge_learned = judge_every < (1 << 26) ? 4 * judge_every : judge_every;
  c->ctrl_record = record ? 1 : 0;
  if (h0 > 0) c->ctrl_h = h0;
  c->ctrl_calib = -1.0;
  c->learn_corr = -1.0;
  c->records.clear();
  c->st_accepted = c->st_rejected = c->st_judged = c->st_rk4 = 0;
  return LREI_OK;
}

int lrei_controller_attach(lrei_ctx *c, lrei_mlp *net) {
  if (!c) return LREI_ERR_ARG;
  c->net = net;
  c->learned_fallback = 0;
  return LREI_OK;
}

int lrei_controller_stats(lrei_ctx *c, lrei_ctrl_stats *out) {
  if (!c || !out) return LREI_ERR_ARG;
  out->accepted = c->st_accepted;
  out->rejected = c->st_rejected;
  out->judged = c->st_judged;
  out->rk4_steps = c->st_rk4;
  out->h = c->ctrl_h;
  out->err_judged = c->st_err_judged;
  out->calib = c->ctrl_calib;
  return LREI_OK;
}

int lrei_controller_records(lrei_ctx *c, double *rows, int max_rows, int *n_rows) {
  if (!c || !n_rows) return LREI_ERR_ARG;
  const int w = LREI_CTRL_NFEAT + 4;
  const int n = (int)(c->records.size() / w);
  *n_rows = n;
  if (rows) std::memcpy(rows, c->records.data(), (size_t)std::min(n, max_rows) * w * sizeof(double));
  return LREI_OK;
}

int lrei_observables(lrei_ctx *c, lrei_obs *out) {
  NvtxScope nvtx_scope("lrei_observables");
  if (!c || !out) return LREI_ERR_ARG;
  if (!c->has_state) return LREI_ERR_STATE;
  const int r = c->r;
  enter(c);
  // H V, (M_x + i M_y) V and M_z V on full rows into the idle Krylov blocks, then two measured
  // Gram passes; where the full-row kernels do not apply, one fused gather pass
  void *S = c->Sbuf, *CV = c->blk[0], *ZV = c->blk[1];
  const bool tiled = launch_hv_tiled(c->fp64, c->M, c->V, S, c->N, r, c->nsm, c->st, c->status_dev) &&
                     launch_magnetization(c->fp64, 1, c->n, c->V, CV, c->N, r, c->nsm, c->st, c->status_dev) &&
                     launch_magnetization(c->fp64, 0, c->n, c->V, ZV, c->N, r, c->nsm, c->st, c->status_dev);
  if (tiled) {
    TSArgs a{};
    a.nq = 3;
    a.gram_left = 3;
    a.q[0] = S;
    a.q[1] = CV;
    a.q[2] = ZV;
    a.src = c->V;
    int rc = ts_pass(c, a, c->nsm);
    if (rc) { leave(c); return rc; }
    zd *R1 = reinterpret_cast<zd *>(c->Uf), *R2 = R1 + 4 * r * r;   // small scratch, idle outside a step
    LREI_CUDA_TRY(cudaMemcpyAsync(R1, c->red, (size_t)4 * r * r * sizeof(zd), cudaMemcpyDeviceToDevice, c->st));
    TSArgs b{};
    b.nq = 0;
    b.gram_left = 0;
    b.src = S;
    if ((rc = ts_pass(c, b, c->nsm))) { leave(c); return rc; }
    LREI_CUDA_TRY(cudaMemcpyAsync(R2, c->red, (size_t)r * r * sizeof(zd), cudaMemcpyDeviceToDevice, c->st));
    ::lrei::count_launch();
    obs_assemble_kernel<<<1, 256, 0, c->st>>>(R1, R2, r, reinterpret_cast<zd *>(c->red));
  } else {
    const int g = launch_obs(c->fp64, c->M, c->V, c->N, r, c->partial, c->nsm, c->st);
    launch_reduce(c->partial, g, 6 * r * r * 2, c->red, c->st);
  }
  ::lrei::count_launch();
  obs_final_kernel<<<1, obs_final_threads(r), 4 * r * r * sizeof(zd), c->st>>>(c->red, r, c->lam0_dev, c->obs_dev, c->werner_p,
                                                               1.0 / (double)c->N, c->mu_dev);
  LREI_CUDA_TRY(cudaMemcpyAsync(c->obs_host, c->obs_dev, 80 * sizeof(double), cudaMemcpyDeviceToHost, c->st));
  leave(c);
  LREI_CUDA_TRY(cudaStreamSynchronize(c->st));
  std::memset(out, 0, sizeof(*out));
  out->t = c->t;
  out->energy = c->obs_host[0];
  out->mx = c->obs_host[1];
  out->my = c->obs_host[2];
  out->mz = c->obs_host[3];
  out->purity = c->obs_host[4];
  out->trace = c->obs_host[5];
  out->orth_err = c->obs_host[6];
  out->herm_err = c->obs_host[7];
  out->comm_norm = c->obs_host[8];
  out->r = r;
  for (int i = 0; i < r && i < 32; ++i) {
    out->ritz[i] = c->obs_host[16 + i];
    out->lambda0[i] = c->obs_host[48 + i];
  }
  return LREI_OK;
}

int lrei_set_eig_sweeps(lrei_ctx *c, int max_sweeps) {
  if (!c || max_sweeps < 1 || max_sweeps > 100) return LREI_ERR_ARG;
  c->eig_sweeps = max_sweeps;
  if (c->gexec) {   // the limit is a kernel argument of the captured step
    cudaGraphExecDestroy(c->gexec);
    c->gexec = nullptr;
    c->g_scheme = -1;
  }
  return LREI_OK;
}

int lrei_set_dmi(lrei_ctx *c, int nbonds, const double *dz) {
  if (!c || nbonds != c->M.nb || (nbonds > 0 && !dz)) return LREI_ERR_ARG;
  for (int k = 0; k < nbonds; ++k)
    if (!std::isfinite(dz[k])) return LREI_ERR_NONFINITE;
  bool any = c->M.bx != 0.0 || c->M.by != 0.0;
  for (int k = 0; k < nbonds; ++k) {
    c->M.dz[k] = dz[k];
    any = any || dz[k] != 0.0;
  }
  c->M.cplx = any ? 1 : 0;
  // the model is a kernel argument of the captured step and of the multistep history
  if (c->gexec) {
    cudaGraphExecDestroy(c->gexec);
    c->gexec = nullptr;
    c->g_scheme = -1;
  }
  if (c->ab_alloc) ab_clear(c);
  return LREI_OK;
}

int lrei_set_werner(lrei_ctx *c, double p) {
  if (!c || !std::isfinite(p) || p < 0.0 || p >= 1.0) return LREI_ERR_ARG;
  c->werner_p = p;
  c->kappa = (1.0 - p) * c->kappa0;
  // the damping is a kernel argument of the captured step and of the multistep history
  if (c->gexec) {
    cudaGraphExecDestroy(c->gexec);
    c->gexec = nullptr;
    c->g_scheme = -1;
  }
  if (c->ab_alloc) ab_clear(c);
  return LREI_OK;
}

int lrei_apply_h(lrei_ctx *c, const void *V_dev, void *Y_dev, int r) {
  if (!c || !V_dev || !Y_dev || V_dev == Y_dev || r < 1 || r > MAX_R) return LREI_ERR_ARG;
  enter(c);
  launch_hv(c->fp64, c->M, V_dev, Y_dev, c->N, r, c->nsm, c->st, c->status_dev);
  leave(c);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? LREI_OK : cuda_fail(e, "apply_h");
}

int lrei_gram(lrei_ctx *c, const void *const *blocks_dev, int nblocks, void *G_dev) {
  if (!c || !blocks_dev || !G_dev || nblocks < 1 || nblocks > MAXB + 1) return LREI_ERR_ARG;
  for (int i = 0; i < nblocks; ++i)
    if (!blocks_dev[i]) return LREI_ERR_ARG;
  const int r = c->r;
  if (r < 1) return LREI_ERR_STATE;
  enter(c);
  TSArgs a{};
  a.nq = nblocks - 1;
  a.gram_left = nblocks - 1;
  for (int i = 0; i + 1 < nblocks; ++i) a.q[i] = const_cast<void *>(blocks_dev[i]);
  a.src = const_cast<void *>(blocks_dev[nblocks - 1]);
  a.apply_h = 0;
  a.mode = 0;
  int rc = ts_pass(c, a);
  if (!rc) {
    const size_t bytes = (size_t)nblocks * r * r * sizeof(zd);
    cudaError_t e = cudaMemcpyAsync(G_dev, c->red, bytes, cudaMemcpyDeviceToDevice, c->st);
    if (e != cudaSuccess) rc = cuda_fail(e, "gram");
  }
  leave(c);
  if (!rc) {
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) rc = cuda_fail(e, "gram");
  }
  return rc;
}

// Householder compact-WY factors of the current factor (U into U_dev, T and D to the host).
static int householder_factors(lrei_ctx *c, void *U_dev) {
  const int r = c->r;
  cudaStream_t st = c->st;
  ::lrei::count_launch(2);
  if (c->fp64) top_block_kernel<double><<<1, 256, 0, st>>>((const cx<double> *)c->V, r, c->Dm);
  else top_block_kernel<float><<<1, 256, 0, st>>>((const cx<float> *)c->V, r, c->Dm);
  hh_setup_kernel<<<1, 256, 4 * r * r * sizeof(zd), st>>>(c->Dm, r, c->X11, c->Ainv, c->L22, c->GR, c->status_dev);
  // U = -V D Rinv (all rows), then U_top += Rinv
  TSArgs u{};
  u.nq = 1;
  u.gram_left = 0;
  u.q[0] = c->V;
  u.coefQ = c->GR;
  u.mode = 2;
  u.out = U_dev;
  int rc = ts_pass(c, u);
  if (rc) return rc;
  ::lrei::count_launch();
  if (c->fp64) add_top_kernel<double><<<1, 256, 0, st>>>((cx<double> *)U_dev, r, c->Ainv);
  else add_top_kernel<float><<<1, 256, 0, st>>>((cx<float> *)U_dev, r, c->Ainv);
  return LREI_OK;
}

int lrei_rhs(lrei_ctx *c, void *Z_dev, void *W_dev, double *G_host, int complement) {
  if (!c || !Z_dev || !W_dev || (complement != 0 && complement != 1)) return LREI_ERR_ARG;
  if (!c->has_state) return LREI_ERR_STATE;
  const int r = c->r;
  if ((long long)r >= c->N && complement == 1) return LREI_ERR_ARG;
  enter(c);
  zd *red = reinterpret_cast<zd *>(c->red);
  int rc = LREI_OK;
  if (complement == 0) {
    // pass 1: Y = H V written to W, G = V^* Y
    TSArgs a{};
    a.nq = 1;
    a.gram_left = 1;
    a.q[0] = c->V;
    a.src = c->V;
    a.apply_h = 1;
    a.mode = 0;
    a.out = W_dev;
    if ((rc = ts_pass(c, a))) { leave(c); return rc; }
    sm_copy(red, 2 * r, r, r, c->G, r, c->st);
    ::lrei::count_launch();
    rhs_coef_kernel<<<1, 256, 0, c->st>>>(c->G, r, c->lam0_dev, c->kappa, c->model, c->Dm, c->GR, c->X11);
    // pass 2: W = Y diag(conj c) - V (G diag(conj c))   (in place over Y: row-local)
    TSArgs b{};
    b.nq = 1;
    b.gram_left = 0;
    b.q[0] = c->V;
    b.src = W_dev;
    b.apply_h = 0;
    b.mode = 1;
    b.coefS = c->Dm;
    b.coefQ = c->GR;
    b.out = W_dev;
    if ((rc = ts_pass(c, b))) { leave(c); return rc; }
  } else {
    // Householder route (Sec. 3.4-3.5): A = V^*H, A V^ = tail of A Q, X12 = diag(c) A V^,
    // W = V^ X12^* = Q [0; X12^*], with Q = I - U T U^H.
    void *U = c->blk[0], *Xh = c->blk[1];
    if ((rc = householder_factors(c, U))) { leave(c); return rc; }
    // P1: Y = H V (into W_dev), Grams [U, V]^* Y
    TSArgs a{};
    a.nq = 2;
    a.gram_left = 2;
    a.q[0] = U;
    a.q[1] = c->V;
    a.src = c->V;
    a.apply_h = 1;
    a.mode = 0;
    a.out = W_dev;
    if ((rc = ts_pass(c, a))) { leave(c); return rc; }
    // G = V^*Y (rows r..2r-1 of the Gram), X11; K1 = T^H (U^*Y)
    ::lrei::count_launch();
    x11_from_g_kernel<<<1, 256, 0, c->st>>>(red + r, 3 * r, r, c->lam0_dev, c->kappa, c->model, c->X11, c->G);
    sm_gemm('C', 'N', r, r, r, ONE, c->L22, r, red, 3 * r, ZERO, c->Bs, r, c->st);
    ::lrei::count_launch();
    diag_conj_c_kernel<<<1, 256, 0, c->st>>>(c->lam0_dev, r, c->kappa, c->model, c->Dm, c->Bs, c->coefQ);
    // P2: Xh = (Y - U K1) diag(conj c), rows < r zero (= [0; X12^*]); Gram U^* Xh
    TSArgs b{};
    b.nq = 1;
    b.gram_left = 1;
    b.q[0] = U;
    b.src = W_dev;
    b.apply_h = 0;
    b.mode = 1;
    b.coefS = c->Dm;
    b.coefQ = c->coefQ;
    b.out = Xh;
    b.zero_rows = r;
    if ((rc = ts_pass(c, b))) { leave(c); return rc; }
    // K2 = T (U^* Xh); P3: W = Xh - U K2
    sm_gemm('N', 'N', r, r, r, MONE, c->L22, r, red, 2 * r, ZERO, c->Bs, r, c->st);
    sm_set_identity(c->Lr, r, r, r, c->st);
    TSArgs w3{};
    w3.nq = 1;
    w3.gram_left = 0;
    w3.q[0] = U;
    w3.src = Xh;
    w3.apply_h = 0;
    w3.mode = 1;
    w3.coefS = c->Lr;
    w3.coefQ = c->Bs;
    w3.out = W_dev;
    if ((rc = ts_pass(c, w3))) { leave(c); return rc; }
  }
  // Z = V X11 + W
  sm_set_identity(c->Ainv, r, r, r, c->st);
  TSArgs z{};
  z.nq = 1;
  z.gram_left = 0;
  z.q[0] = c->V;
  z.src = W_dev;
  z.apply_h = 0;
  z.mode = 1;
  z.coefS = c->Ainv;
  z.coefQ = c->X11;
  z.out = Z_dev;
  if ((rc = ts_pass(c, z))) { leave(c); return rc; }
  if (G_host) {
    sm_hermitize(c->G, r, r, c->st);
    LREI_CUDA_TRY(cudaMemcpyAsync(G_host, c->G, (size_t)r * r * sizeof(zd), cudaMemcpyDeviceToHost, c->st));
  }
  leave(c);
  LREI_CUDA_TRY(cudaStreamSynchronize(c->st));
  const int s = read_status(c);
  return status_to_code(s);
}

int lrei_householder(lrei_ctx *c, void *U_dev, double *T_host, double *D_host) {
  if (!c || !U_dev) return LREI_ERR_ARG;
  if (!c->has_state) return LREI_ERR_STATE;
  const int r = c->r;
  if ((long long)r >= c->N) return LREI_ERR_ARG;
  enter(c);
  int rc = householder_factors(c, U_dev);
  if (rc) { leave(c); return rc; }
  if (T_host) LREI_CUDA_TRY(cudaMemcpyAsync(T_host, c->L22, (size_t)r * r * sizeof(zd), cudaMemcpyDeviceToHost, c->st));
  if (D_host) LREI_CUDA_TRY(cudaMemcpyAsync(D_host, c->X11, (size_t)r * sizeof(zd), cudaMemcpyDeviceToHost, c->st));
  leave(c);
  LREI_CUDA_TRY(cudaStreamSynchronize(c->st));
  return status_to_code(read_status(c));
}

int lrei_two_spin_rdm(lrei_ctx *c, int npairs, const int *site_k, const int *site_l, double *R_host,
                      double *concurrence_host, double *negativity_host) {
  NvtxScope nvtx_scope("lrei_two_spin_rdm");
  if (!c || npairs < 1 || npairs > LREI_RDM_MAX_PAIRS || !site_k || !site_l) return LREI_ERR_ARG;
  if (!c->has_state) return LREI_ERR_STATE;
  if (c->n < 2) return LREI_ERR_ARG;
  std::vector<int> bits(2 * (size_t)npairs);
  for (int q = 0; q < npairs; ++q) {
    const int k = site_k[q], l = site_l[q];
    if (k < 0 || k >= c->n || l < 0 || l >= c->n || k == l) return LREI_ERR_ARG;
    bits[2 * q] = c->n - 1 - k;   // site i is bit n-1-i of the basis index
    bits[2 * q + 1] = c->n - 1 - l;
  }
  const int r = c->r;
  enter(c);
  // the orthonormalised factor Vb = V L^{-H} (V^*V = L L^H) into the scratch block
  sm_set_identity(c->Ainv, r, r, r, c->st);
  sm_trsv('C', c->L, c->KM, r, c->Ainv, r, r, c->st);
  TSArgs cmb{};
  cmb.nq = 1;
  cmb.gram_left = 0;
  cmb.q[0] = c->V;
  cmb.coefQ = c->Ainv;
  cmb.mode = 2;
  cmb.out = c->Sbuf;
  int rc = ts_pass(c, cmb);
  if (rc) { leave(c); return rc; }
  LREI_CUDA_TRY(cudaMemcpyAsync(c->rdm_pairs, bits.data(), bits.size() * sizeof(int), cudaMemcpyHostToDevice, c->st));
  // CTAs per pair: enough to fill the GPU for a few pairs, bounded by the partial-sum buffer
  const long long groups = c->N / 4;
  const long long per_cta = 256 / r;
  int ncta = (int)std::min<long long>(64, std::max<long long>(1, (groups + per_cta - 1) / per_cta));
  int chunk = (int)std::min<size_t>((size_t)npairs, c->partial_doubles / ((size_t)ncta * 16));
  while (chunk < 1 && ncta > 1) {
    ncta /= 2;
    chunk = (int)std::min<size_t>((size_t)npairs, c->partial_doubles / ((size_t)ncta * 16));
  }
  for (int q0 = 0; q0 < npairs && !rc; q0 += chunk) {
    const int nq = std::min(chunk, npairs - q0);
    if (launch_rdm(c->fp64, c->Sbuf, c->N, r, c->lam0_dev, c->rdm_pairs + 2 * q0, nq, c->partial, ncta, c->st))
      rc = LREI_ERR_ARG;
    else
      launch_rdm_final(c->partial, ncta, nq, c->werner_p, c->rdm_out + (size_t)34 * q0, c->st);
  }
  std::vector<double> res((size_t)34 * npairs);
  if (!rc)
    LREI_CUDA_TRY(cudaMemcpyAsync(res.data(), c->rdm_out, res.size() * sizeof(double), cudaMemcpyDeviceToHost, c->st));
  leave(c);
  LREI_CUDA_TRY(cudaStreamSynchronize(c->st));
  if (rc) return rc;
  for (int q = 0; q < npairs; ++q) {
    if (R_host) std::memcpy(R_host + (size_t)32 * q, res.data() + (size_t)34 * q, 32 * sizeof(double));
    if (concurrence_host) concurrence_host[q] = res[(size_t)34 * q + 32];
    if (negativity_host) negativity_host[q] = res[(size_t)34 * q + 33];
  }
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? LREI_OK : cuda_fail(e, "two_spin_rdm");
}

int lrei_truncate_rank(lrei_ctx *c, double tol_r, int *r_out, double *dropped_out) {
  NvtxScope nvtx_scope("lrei_truncate_rank");
  if (!c || !std::isfinite(tol_r) || tol_r < 0.0) return LREI_ERR_ARG;
  if (!c->has_state) return LREI_ERR_STATE;
  const int r = c->r;
  // keep the leading k eigenvalues: the trailing ones (smallest, Lambda_0 is decreasing) go while
  // their cumulative weight stays within tol_r; at least one is kept
  int k = r;
  double w = 0.0;
  while (k > 1 && w + c->lam0[k - 1] <= tol_r) w += c->lam0[--k];
  if (r_out) *r_out = k;
  if (dropped_out) *dropped_out = w;
  if (k == r) return LREI_OK;
  enter(c);
  const long long total = c->N * k;
  const int grid = (int)((total + 255) / 256 < 4096 ? (total + 255) / 256 : 4096);
  ::lrei::count_launch();
  if (c->fp64) keep_cols_kernel<double><<<grid, 256, 0, c->st>>>((const cx<double> *)c->V, r, (cx<double> *)c->Sbuf, k, c->N);
  else keep_cols_kernel<float><<<grid, 256, 0, c->st>>>((const cx<float> *)c->V, r, (cx<float> *)c->Sbuf, k, c->N);
  LREI_CUDA_TRY(cudaMemcpyAsync(c->V, c->Sbuf, (size_t)total * c->elem, cudaMemcpyDeviceToDevice, c->st));
  c->r = k;
  // the kept weights are renormalised to trace one
  for (int i = 0; i < k; ++i) c->lam0[i] /= (1.0 - w);
  c->lam0.resize(k);
  LREI_CUDA_TRY(cudaMemcpyAsync(c->lam0_dev, c->lam0.data(), k * sizeof(double), cudaMemcpyHostToDevice, c->st));
  LREI_CUDA_TRY(cudaMemcpyAsync(c->mu_dev, c->lam0.data(), k * sizeof(double), cudaMemcpyHostToDevice, c->st));
  // the Gram of the kept columns is the leading block of the old one; measured again all the same
  TSArgs a{};
  a.nq = 0;
  a.gram_left = 0;
  a.src = c->V;
  a.apply_h = 0;
  a.mode = 0;
  int rc = ts_pass(c, a);
  if (!rc) {
    LREI_CUDA_TRY(cudaMemsetAsync(c->L, 0, (size_t)c->KM * c->KM * sizeof(zd), c->st));
    LREI_CUDA_TRY(cudaMemsetAsync(c->Chat, 0, (size_t)c->KM * c->KM * sizeof(zd), c->st));
    set_gamma00(c);
  }
  if (c->ab_alloc) ab_clear(c);
  const int s = read_status(c);
  leave(c);
  if (rc) return rc;
  return status_to_code(s);
}

// ---- checkpoint: everything the next steps read, byte for byte
namespace {
struct CkptHeader {
  char magic[8];
  int version, n, r, prec, model, ab_m, nhist, pad;
  double t, ab_dt, kappa0, werner_p, ctrl_h, ctrl_calib;
};
size_t ckpt_bytes(const lrei_ctx *c) {
  const size_t blk = (size_t)c->N * c->r * c->elem;
  const size_t nh = c->ab_alloc ? c->ab_hist.size() : 0;
  return sizeof(CkptHeader) + 2 * (size_t)c->r * sizeof(double) + 2 * (size_t)c->r * c->r * sizeof(zd) + blk +
         2 * nh * blk;
}
}  // namespace

long long lrei_checkpoint_bytes(lrei_ctx *c) {
  if (!c || !c->has_state) return 0;
  return (long long)ckpt_bytes(c);
}

int lrei_checkpoint_save(lrei_ctx *c, void *buf, long long bytes) {
  NvtxScope nvtx_scope("lrei_checkpoint_save");
  if (!c || !buf) return LREI_ERR_ARG;
  if (!c->has_state) return LREI_ERR_STATE;
  if (bytes < (long long)ckpt_bytes(c)) return LREI_ERR_ARG;
  const int r = c->r, KM = c->KM;
  const size_t blk = (size_t)c->N * r * c->elem;
  CkptHeader h;
  std::memset(&h, 0, sizeof(h));
  std::memcpy(h.magic, "LREICKP", 8);
  h.version = 1;
  h.n = c->n;
  h.r = r;
  h.prec = c->prec;
  h.model = c->model;
  h.ab_m = c->ab_alloc ? c->ab_m : 0;
  h.nhist = c->ab_alloc ? (int)c->ab_hist.size() : 0;
  h.t = c->t;
  h.ab_dt = c->ab_dt;
  h.kappa0 = c->kappa0;
  h.werner_p = c->werner_p;
  h.ctrl_h = c->ctrl_h;
  h.ctrl_calib = c->ctrl_calib;
  unsigned char *p = static_cast<unsigned char *>(buf);
  std::memcpy(p, &h, sizeof(h));
  p += sizeof(h);
  std::memcpy(p, c->lam0.data(), r * sizeof(double));
  p += r * sizeof(double);
  enter(c);
  LREI_CUDA_TRY(cudaMemcpyAsync(p, c->mu_dev, r * sizeof(double), cudaMemcpyDeviceToHost, c->st));
  p += r * sizeof(double);
  LREI_CUDA_TRY(cudaMemcpy2DAsync(p, r * sizeof(zd), c->Gam, KM * sizeof(zd), r * sizeof(zd), r, cudaMemcpyDeviceToHost, c->st));
  p += (size_t)r * r * sizeof(zd);
  LREI_CUDA_TRY(cudaMemcpy2DAsync(p, r * sizeof(zd), c->L, KM * sizeof(zd), r * sizeof(zd), r, cudaMemcpyDeviceToHost, c->st));
  p += (size_t)r * r * sizeof(zd);
  LREI_CUDA_TRY(cudaMemcpyAsync(p, c->V, blk, cudaMemcpyDeviceToHost, c->st));
  p += blk;
  for (int i = 0; i < h.nhist; ++i) {
    LREI_CUDA_TRY(cudaMemcpyAsync(p, c->ab_hist[i].first, blk, cudaMemcpyDeviceToHost, c->st));
    p += blk;
    LREI_CUDA_TRY(cudaMemcpyAsync(p, c->ab_hist[i].second, blk, cudaMemcpyDeviceToHost, c->st));
    p += blk;
  }
  leave(c);
  LREI_CUDA_TRY(cudaStreamSynchronize(c->st));
  return LREI_OK;
}

int lrei_checkpoint_load(lrei_ctx *c, const void *buf, long long bytes) {
  NvtxScope nvtx_scope("lrei_checkpoint_load");
  if (!c || !buf || bytes < (long long)sizeof(CkptHeader)) return LREI_ERR_ARG;
  CkptHeader h;
  std::memcpy(&h, buf, sizeof(h));
  if (std::memcmp(h.magic, "LREICKP", 8) != 0 || h.version != 1) return LREI_ERR_ARG;
  if (h.n != c->n || h.prec != c->prec || h.model != c->model || h.r < 1 || h.r > c->r_max || h.nhist < 0 ||
      h.nhist > 3 || h.kappa0 != c->kappa0)
    return LREI_ERR_ARG;
  const int r = h.r, KM = c->KM;
  const size_t blk = (size_t)c->N * r * c->elem;
  const size_t need = sizeof(h) + 2 * (size_t)r * sizeof(double) + 2 * (size_t)r * r * sizeof(zd) + blk +
                      2 * (size_t)h.nhist * blk;
  if ((size_t)bytes < need) return LREI_ERR_ARG;
  int rc;
  if (h.nhist > 0 && (rc = ab_prepare(c))) return rc;
  const unsigned char *p = static_cast<const unsigned char *>(buf) + sizeof(h);
  c->r = r;
  c->lam0.assign(reinterpret_cast<const double *>(p), reinterpret_cast<const double *>(p) + r);
  p += r * sizeof(double);
  enter(c);
  LREI_CUDA_TRY(cudaMemcpyAsync(c->lam0_dev, c->lam0.data(), r * sizeof(double), cudaMemcpyHostToDevice, c->st));
  LREI_CUDA_TRY(cudaMemcpyAsync(c->mu_dev, p, r * sizeof(double), cudaMemcpyHostToDevice, c->st));
  p += r * sizeof(double);
  LREI_CUDA_TRY(cudaMemsetAsync(c->Gam, 0, (size_t)KM * KM * sizeof(zd), c->st));
  LREI_CUDA_TRY(cudaMemsetAsync(c->L, 0, (size_t)KM * KM * sizeof(zd), c->st));
  LREI_CUDA_TRY(cudaMemsetAsync(c->Chat, 0, (size_t)KM * KM * sizeof(zd), c->st));
  LREI_CUDA_TRY(cudaMemcpy2DAsync(c->Gam, KM * sizeof(zd), p, r * sizeof(zd), r * sizeof(zd), r, cudaMemcpyHostToDevice, c->st));
  p += (size_t)r * r * sizeof(zd);
  LREI_CUDA_TRY(cudaMemcpy2DAsync(c->L, KM * sizeof(zd), p, r * sizeof(zd), r * sizeof(zd), r, cudaMemcpyHostToDevice, c->st));
  p += (size_t)r * r * sizeof(zd);
  LREI_CUDA_TRY(cudaMemcpyAsync(c->V, p, blk, cudaMemcpyHostToDevice, c->st));
  p += blk;
  if (c->ab_alloc) ab_clear(c);
  for (int i = 0; i < h.nhist; ++i) {
    void *vk = ab_take(c), *yk = ab_take(c);
    LREI_CUDA_TRY(cudaMemcpyAsync(vk, p, blk, cudaMemcpyHostToDevice, c->st));
    p += blk;
    LREI_CUDA_TRY(cudaMemcpyAsync(yk, p, blk, cudaMemcpyHostToDevice, c->st));
    p += blk;
    c->ab_hist.push_back({vk, yk});
  }
  c->ab_m = h.nhist > 0 ? h.ab_m : 0;
  c->ab_dt = h.ab_dt;
  leave(c);
  LREI_CUDA_TRY(cudaStreamSynchronize(c->st));
  c->t = h.t;
  c->ctrl_h = h.ctrl_h;
  c->ctrl_calib = h.ctrl_calib;
  c->has_state = true;
  if (h.werner_p != c->werner_p) return lrei_set_werner(c, h.werner_p);
  return LREI_OK;
}

// ---- many trajectories side by side: one graph launch per RK4 step of the whole batch
struct lrei_batch {
  std::vector<lrei_ctx *> ctx;
  cudaStream_t st = nullptr;
  cudaEvent_t ev = nullptr;
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  double dt = 0.0;
  int nsm_use = 0;
};

namespace {
void set_sm_share(lrei_ctx *c, int nsm) {
  nsm = std::max(1, std::min(nsm, c->nsm));
  if (nsm == c->nsm_use) return;
  c->nsm_use = nsm;
  c->nsm_pass = c->fp64 ? nsm : std::max(1, nsm - (nsm >= 16 ? nsm / 16 : 0));
  if (c->gexec) {   // grid sizes are baked into the captured step
    cudaGraphExecDestroy(c->gexec);
    c->gexec = nullptr;
    c->g_scheme = -1;
  }
}

int batch_build(lrei_batch *b) {
  if (b->exec) { cudaGraphExecDestroy(b->exec); b->exec = nullptr; }
  if (b->graph) { cudaGraphDestroy(b->graph); b->graph = nullptr; }
  for (lrei_ctx *c : b->ctx) {
    int rc = build_graph(c, (int)LREI_RK4);
    if (rc) return rc;
  }
  LREI_CUDA_TRY(cudaGraphCreate(&b->graph, 0));
  // independent child graphs: the trajectories have no edges between them
  for (lrei_ctx *c : b->ctx) {
    cudaGraphNode_t node;
    LREI_CUDA_TRY(cudaGraphAddChildGraphNode(&node, b->graph, nullptr, 0, c->graph));
  }
  LREI_CUDA_TRY(cudaGraphInstantiate(&b->exec, b->graph, 0));
  return LREI_OK;
}

int batch_run(lrei_batch *b, double dt, int nsteps) {
  // order the batch after the contexts' own streams
  for (lrei_ctx *c : b->ctx) {
    LREI_CUDA_TRY(cudaEventRecord(c->ev_out, c->st));
    LREI_CUDA_TRY(cudaStreamWaitEvent(b->st, c->ev_out, 0));
  }
  if (dt != b->dt) {
    for (lrei_ctx *c : b->ctx) {
      LREI_CUDA_TRY(cudaMemcpyAsync(c->dt_dev, &dt, sizeof(double), cudaMemcpyHostToDevice, b->st));
      c->dt_cur = dt;
    }
    LREI_CUDA_TRY(cudaStreamSynchronize(b->st));
    b->dt = dt;
  }
  for (int i = 0; i < nsteps; ++i) LREI_CUDA_TRY(cudaGraphLaunch(b->exec, b->st));
  LREI_CUDA_TRY(cudaEventRecord(b->ev, b->st));
  LREI_CUDA_TRY(cudaEventSynchronize(b->ev));
  int code = LREI_OK;
  for (lrei_ctx *c : b->ctx) {
    LREI_CUDA_TRY(cudaStreamWaitEvent(c->st, b->ev, 0));
    c->t += dt * nsteps;
    c->launches += c->g_nodes * nsteps;
    const int s = read_status(c);
    if (s && code == LREI_OK) code = status_to_code(s);
  }
  return code;
}
}  // namespace

int lrei_batch_create(int nctx, lrei_ctx *const *ctxs, void *cuda_stream, lrei_batch **out) {
  if (!out || nctx < 1 || !ctxs) return LREI_ERR_ARG;
  *out = nullptr;
  int dev = -1;
  for (int i = 0; i < nctx; ++i) {
    if (!ctxs[i]) return LREI_ERR_ARG;
    if (!ctxs[i]->has_state) return LREI_ERR_STATE;
    if (dev < 0) dev = ctxs[i]->dev;
    if (ctxs[i]->dev != dev) return LREI_ERR_ARG;
    for (int j = 0; j < i; ++j)
      if (ctxs[j] == ctxs[i]) return LREI_ERR_ARG;
  }
  lrei_batch *b = new (std::nothrow) lrei_batch();
  if (!b) return LREI_ERR_OOM;
  b->ctx.assign(ctxs, ctxs + nctx);
  b->st = reinterpret_cast<cudaStream_t>(cuda_stream);
  b->nsm_use = ctxs[0]->nsm;
  if (cudaEventCreateWithFlags(&b->ev, cudaEventDisableTiming) != cudaSuccess) {
    delete b;
    return LREI_ERR_CUDA;
  }
  const int rc = batch_build(b);
  if (rc) {
    lrei_batch_destroy(b);
    return rc;
  }
  *out = b;
  return LREI_OK;
}

int lrei_batch_step(lrei_batch *b, double dt, int nsteps) {
  NvtxScope nvtx_scope("lrei_batch_step");
  if (!b || !std::isfinite(dt) || nsteps < 0) return LREI_ERR_ARG;
  if (nsteps == 0) return LREI_OK;
  return batch_run(b, dt, nsteps);
}

int lrei_batch_autotune(lrei_batch *b, double dt, int steps, int *nsm_out, double *ms_out) {
  NvtxScope nvtx_scope("lrei_batch_autotune");
  if (!b || !std::isfinite(dt) || steps < 1) return LREI_ERR_ARG;
  const int nsm = b->ctx[0]->nsm;
  int best = nsm;
  double best_ms = 1e300;
  cudaEvent_t e0, e1;
  LREI_CUDA_TRY(cudaEventCreate(&e0));
  LREI_CUDA_TRY(cudaEventCreate(&e1));
  int rc = LREI_OK;
  for (int share = nsm; share >= 1 && !rc; share = (share > 1 ? share / 2 : 0)) {
    for (lrei_ctx *c : b->ctx) set_sm_share(c, share);
    if ((rc = batch_build(b))) break;
    if ((rc = batch_run(b, dt, 1))) break;   // warm-up
    cudaEventRecord(e0, b->st);
    for (int i = 0; i < steps; ++i) cudaGraphLaunch(b->exec, b->st);
    cudaEventRecord(e1, b->st);
    if (cudaEventSynchronize(e1) != cudaSuccess) { rc = LREI_ERR_CUDA; break; }
    float ms = 0.f;
    cudaEventElapsedTime(&ms, e0, e1);
    for (lrei_ctx *c : b->ctx) {
      c->t += dt * steps;
      c->launches += c->g_nodes * steps;
      const int s = read_status(c);
      if (s && !rc) rc = status_to_code(s);
    }
    if (ms / steps < best_ms) {
      best_ms = ms / steps;
      best = share;
    }
    if (share < 8) break;   // candidates: nsm, nsm/2, ..., down to a few SMs per trajectory
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (rc) return rc;
  for (lrei_ctx *c : b->ctx) set_sm_share(c, best);
  b->nsm_use = best;
  if ((rc = batch_build(b))) return rc;
  if (nsm_out) *nsm_out = best;
  if (ms_out) *ms_out = best_ms;
  return LREI_OK;
}

int lrei_batch_destroy(lrei_batch *b) {
  if (!b) return LREI_OK;
  if (b->st) cudaStreamSynchronize(b->st);
  if (b->exec) cudaGraphExecDestroy(b->exec);
  if (b->graph) cudaGraphDestroy(b->graph);
  if (b->ev) cudaEventDestroy(b->ev);
  delete b;
  return LREI_OK;
}

int lrei_last_status(lrei_ctx *c) { return c ? c->last_status : 0; }

int lrei_debug_counters(unsigned long long *out4) {
  if (!out4) return LREI_ERR_ARG;
  cudaDeviceSynchronize();
  return sm_read_counters(out4) == 0 ? LREI_OK : LREI_ERR_CUDA;
}

long long lrei_kernel_launches(lrei_ctx *c) {
  if (!c) return 0;
  long long n = c->launches;
  c->launches = 0;
  return n;
}

}  // extern "C"
