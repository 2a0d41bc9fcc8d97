// Tall-skinny tile passes of complex128 blocks on the tensor cores (the contract of tsk.cuh, without H.V).
//
// FP64 arithmetic runs at 1.0 TFLOP/s on this part (a DFMA takes a scheduler 64 cycles), FP16 tensor
// instructions at 600 TFLOP/s (mma.sync, 953 multiply-adds per clock and SM, both measured), so a Gram or a
// projection in FP64 costs less as 28 exact integer products.  The operands are cut into integer digits
// (the error-free slicing of Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59, 2012): a column of a tile is
//     x = 2^(e - 7) sum_{s < 7} d_s 2^(-8 s),   |d_s| <= 128,
// with one exponent e per column (55 bits below 2^e, so an entry of the column's top binade is exact), the
// digits held exactly in FP16.  The product of two digit planes is an integer sum, exact in the tensor core's
// FP32 accumulator while it stays below 2^24.  Of the 49 digit products the 28 with s + t <= 6 are formed (the
// others are below 2^-55 of the largest); those of equal s + t share an accumulator (a "class").  Every 128 complex summands
// (the rows of a Gram, the columns of a projection: 2 x 128 x 4 x 2^14 = 2^24 for the first four classes; a class beyond
// the fourth carries less than 2^-32 of the result) the classes go into two 64-bit integers per entry, without rounding.
// In a Gram a column keeps its exponent from tile to tile while the tile's largest entry stays within ten bits below it.
// Above it, the column's exponent rises and the sums so far are shifted down; further below, they are flushed to the CTA's
// FP64 partial at the old exponents and the column gets a new one.  A value is off by 2^-56 of the power of two above the largest of its column so far, an entry of the Gram by
// some 2^-55 of its columns' norms: a value beside a larger one keeps fewer bits, which the sum over the rows does not see.
// A projection does: each of its rows is a result.  There the exponents are those of the rows, after the columns are
// weighted: with 2^(g_k) the largest coefficient of input column k,
//     new_rj = sum_k (x_rk 2^(g_k)) (c_kj 2^(-g_k)),
// the entries of row r share the exponent e_r of the largest weighted one and the coefficients of output j the exponent f_j, and
// the result is off by 2^-52 K max_k |x_rk| max_j |c_kj| whatever the other rows of the tile hold (a column exponent per
// tile lost as many bits of a row as it was smaller than the largest of 16 or 32 rows).  g and the digits of the
// coefficients are made once per CTA.
// A tile with infinities, NaN or entries near the ends of the exponent range takes a direct path in FP64 FMAs.
//
// Layout.  A column group is 8 complex columns of one block (ranks that are not a multiple of 8 are padded by
// repeating the last column), a chunk is 16 rows.  A thread (g = lane / 4, q = lane % 4) of a cutting warp
// takes column g of its unit (group, chunk) at rows q, q+4, q+8, q+12, which are the elements an m16n8k16 fragment
// wants of it, and stores the digit planes as four 8 x 8 FP16 matrices (re / im x first / last 8 rows), so that
// ldmatrix gives a Gram operand (columns x rows) and ldmatrix.trans a projection operand (rows x columns) from the
// same bytes.
//
// The work of a CTA is split by warp: the cutting warps wait for a tile's bulk copies and make its planes while the
// multiplying warps work on the planes of the tile before (two buffers, named barriers).  What bounds the kernels
// is the two together: a tile of 32 rows of five 16-column blocks costs 4700 cycles of tensor pipe and 2500 cycles
// of integer ALU per scheduler.
#include "tsk.cuh"

#include <cuda_fp16.h>

#include <algorithm>

namespace lrei {

// What one launch does, worked out on the host (tsx_plan).
struct XPlan {
  int cpb;        // column groups per block, ceil(r / 8)
  int kt, nkc;    // rows and chunks per tile
  int rpb;        // Gram row blocks per blockIdx.y
  int npb;        // column groups of the new block per blockIdx.y
  int wm, wc;     // warps that multiply, warps that cut
  int ksplit;     // multiplying warps sharing one Gram item over the chunks
  int gpw;        // groups of a cutting warp (at most CUT_UNITS / nkc)
  int items;      // Gram items (16 left columns x 8 right columns)
  int ldnv;       // reals per row of the new tile
  int o_raw, o_sums, o_coef, o_nv, o_int, bytes;   // shared memory offsets
};

namespace {

constexpr int NS = 7;                 // digits
constexpr int CUT_UNITS = 4;          // units a cutting warp holds in registers
constexpr int X_THREADS = 512;        // most threads of a CTA (128 registers)
constexpr int X_DRAIN = 128;          // complex summands between drains
// Gram: bits that a column's tiles may stay below its exponent, and what tells the multiplying warps that one changed.  H V of a
// spin chain varies by 2^7 from tile to tile (the diagonal and the number of flips do): with 2 bits 60 to 97 of 100 tiles flushed
// the sums of their CTA, 7 us each.  With 10, and a tile above the largest so far shifting the sums in shared memory, hardly any does.
// A column's first exponent is a bit above its tile's, which spares most columns without structure any shift (6 random blocks at
// n = 14, r = 16: 66 us against 73), later ones are the tile's own.
constexpr int X_SLACK = 10, X_RAISED = 1, X_LOWERED = 2;
constexpr int X_EMIN = 530, X_EMAX = 1510;   // exponent fields that are cut; others take the direct path
constexpr int E_UNSET = -100000;
// projections: exponents of the rows that are cut, of the coefficients' largest (either side); a zero coefficient row; the
// bias of a row's key (0: a zero row)
constexpr int X_RMIN = -450, X_RMAX = 480, X_GMAX = 400, G_ZERO = -3000, X_BIAS = 8192;
// named barriers: planes b full (BAR_FULL + b), free again (BAR_FREE + b), the multiplying and the cutting warps
constexpr int BAR_FULL = 1, BAR_FREE = 3, BAR_MUL = 5, BAR_CUT = 6;

__device__ __forceinline__ void bar_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;\n" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id, int threads) {
  asm volatile("bar.arrive %0, %1;\n" ::"r"(id), "r"(threads) : "memory");
}
// bounded wait on an mbarrier phase (2^16 suspending polls of up to 2 us)
__device__ __forceinline__ bool wait_phase(uint32_t bar, uint32_t parity) {
  for (int it = 0; it < (1 << 16); ++it) {
    uint32_t done;
    asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\nselp.u32 %0, 1, 0, p;\n}\n"
                 : "=r"(done) : "r"(bar), "r"(parity), "r"(2000u) : "memory");
    if (done) return true;
  }
  return false;
}
__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldsm4(uint32_t (&v)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldsm4t(uint32_t (&v)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]) : "r"(addr) : "memory");
}
constexpr uint32_t NEG2 = 0x80008000u;   // flips the sign of a pair of FP16 digits

// a magnitude key: larger |x| gives a larger key (NaN the largest); key >> 20 is the exponent field
__device__ __forceinline__ uint32_t mag_key(double x) { return (uint32_t)__double2hiint(x) & 0x7fffffffu; }

// rint(x 2^(55-e)) + 0x80..80 (a byte per digit) for |x| < 2^e, in 32-bit integer operations
__device__ __forceinline__ unsigned long long fixed_biased(double x, int e) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const int E = (int)((hi << 1) >> 21);
  const uint32_t sg = (uint32_t)((int)hi >> 31);
  // the significand 2^3 too large and signed, then down by s, leaving one bit to round with (a zero or
  // denormal has s > 63 and vanishes)
  unsigned long long m = ((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32 | lo) << 3;
  m = (m ^ ((unsigned long long)sg << 32 | sg)) - (long long)(int)sg;
  const int s = min(e + 1022 - E, 63);
  const long long t = (long long)m >> s;
  return (unsigned long long)(t + 0x0101010101010101ll) >> 1;
}
// the same for any x and scale: rint(x 2^k) + 0x80..80, |x 2^k| < 2^55 (used for the few coefficients)
__device__ __forceinline__ unsigned long long fixed_biased_k(double x, int k) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int E = (int)(b >> 52) & 0x7ff;
  unsigned long long m = (b & 0xfffffffffffffull) | (E ? 0x10000000000000ull : 0ull);
  const int sh = k + (E ? E : 1) - 1075;
  if (sh >= 0) m <<= min(sh, 63);   // a zero may come with any scale
  else if (sh > -56) m = (m + (1ull << (-sh - 1))) >> (-sh);
  else m = 0;
  return ((long long)b < 0 ? 0ull - m : m) + 0x80808080808080ull;
}
// Digit planes of a pair of biased integers: the bytes (the first digit: the top 16 bits) minus 128, as FP16.
__device__ __forceinline__ void digit_planes(unsigned long long a, unsigned long long b, uint32_t (&d)[NS]) {
  const uint32_t al = (uint32_t)a, ah = (uint32_t)(a >> 32), bl = (uint32_t)b, bh = (uint32_t)(b >> 32);
  auto minus = [](uint32_t v) {   // FP16 pair 1024 + byte -> byte - 128
    const __half2 h = __hadd2(*reinterpret_cast<__half2 *>(&v), __float2half2_rn(-1152.f));
    return *reinterpret_cast<const uint32_t *>(&h);
  };
  auto byte_pair = [&](uint32_t x, uint32_t y, uint32_t sel) {
    return minus((__byte_perm(x, y, sel) & 0x00ff00ffu) | 0x64006400u);
  };
  d[0] = minus(__byte_perm(ah, bh, 0x7632) | 0x64006400u);
  d[1] = byte_pair(ah, bh, 0x0501);
  d[2] = byte_pair(ah, bh, 0x0400);
  d[3] = byte_pair(al, bl, 0x0703);
  d[4] = byte_pair(al, bl, 0x0602);
  d[5] = byte_pair(al, bl, 0x0501);
  d[6] = byte_pair(al, bl, 0x0400);
}

// The classes as integers (first three, last four): x = h 2^-16 + l 2^-48.
__device__ __forceinline__ void class_ints(const float (&a)[NS], long long &h, long long &l) {
  h = ((long long)__float2int_rn(a[0]) << 16) + ((long long)__float2int_rn(a[1]) << 8) + __float2int_rn(a[2]);
  l = ((long long)__float2int_rn(a[3]) << 24) + ((long long)__float2int_rn(a[4]) << 16) +
      ((long long)__float2int_rn(a[5]) << 8) + __float2int_rn(a[6]);
}
// (h 2^-16 + l 2^-48) 2^k, rounded once, by integer operations (an FP64 conversion or multiply takes a scheduler
// 64 cycles; this is about 30 integer instructions).
__device__ __forceinline__ double ints_value(long long h, long long l, int k) {
  const long long t = h + (l >> 32), sg = t >> 63;      // h 2^32 + l = t 2^32 + (low word of l)
  unsigned long long H = (unsigned long long)(t ^ sg), L = (unsigned long long)((uint32_t)l ^ (uint32_t)sg) << 32;
  if (sg) {                                             // two's complement of the 96 bits
    L += 1ull << 32;
    H += L == 0;
  }
  int e = 1023 + 63 + 32 - 48 + k;
  if (H == 0) {
    if (L == 0) return 0.0;
    H = L;
    L = 0;
    e -= 64;
  }
  const int z = __clzll((long long)H);
  const unsigned long long m = z ? (H << z) | (L >> (64 - z)) : H;   // the leading 64 bits
  e -= z;
  const unsigned long long f = (m >> 11) + ((m >> 10) & 1);          // 53 bits, rounded
  if (e <= 0 || e >= 2046) return scalbn((sg ? -(double)f : (double)f), e - 1023 - 52);
  return __longlong_as_double((long long)((unsigned long long)sg << 63 | (((unsigned long long)(e - 1) << 52) + f)));
}
// A running sum of an accumulator entry between flushes, in shared memory.
struct Sum {
  long long h, l;
  __device__ __forceinline__ void load(uint32_t at) {
    asm volatile("ld.shared.v2.s64 {%0, %1}, [%2];\n" : "=l"(h), "=l"(l) : "r"(at));
  }
  __device__ __forceinline__ void store(uint32_t at) const {
    asm volatile("st.shared.v2.s64 [%0], {%1, %2};\n" ::"r"(at), "l"(h), "l"(l));
  }
  __device__ __forceinline__ void down(int k) {   // h 2^32 + l, k > 0 bits down
    if (k >= 32) {
      l = h + (l >> 32);
      h = 0;
      k -= 32;
    }
    if (k >= 32) {
      l >>= min(k, 63);
      return;
    }
    l = (l >> k) + ((h & ((1ll << k) - 1)) << (32 - k));
    h >>= k;
  }
};

extern __shared__ __align__(128) unsigned char tsx_smem[];

// Sizes and shared memory of a CTA, from the launch arguments.
template <bool PROJ>
struct Geo {
  int nt;                 // threads that multiply
  int rb0, rb1, nleft, nload, ncg, mt, ncl;
  int n0, np;             // the new block's column groups n0 .. n0 + np - 1 are this CTA's
  unsigned char *dig;     // [buffer][chunk][group][digit][4][128]: digit planes
  zd *raw;                // [block][kt][r] the loaded tile
  unsigned char *sums;    // [entry][nt] the threads' sums
  uint32_t *coef;         // [group][column group][digit][re, im][32]
  double *nv;             // [kt][ldnv] the new tile
  int *rowkey;            // projection: [4][kt] biased exponents of the weighted rows (tile & 3)
  int *gam;               // projection: [ncl] exponents g of the input columns
  uint32_t *key;          // Gram: [4][ncl] magnitude keys of the columns (tile & 3)
  int *ecol;              // [4][ncl] exponents of the columns in a tile (tile & 3)
  int *eacc;              // [ncl] exponents of the sums since the last flush
  int *fcol;              // [npb * 8] exponents of the coefficient columns
  int *flags;             // 0: non-finite coefficients, 1: a wait ran out; 4 + 2 (tile & 3), 5 + 2 (tile & 3): an
                          // exponent changes, a column cannot be cut
  double2 *outp;          // the CTA's partial
  __device__ __forceinline__ Geo(const TSArgs &a, const XPlan &p) {
    const int ng = a.gram_left + 1;
    nt = p.wm * 32;
    // Gram row blocks of this CTA ([q_rb0 ..] and, when it is the last, G) and the blocks it loads
    rb0 = PROJ ? 0 : blockIdx.y * p.rpb;
    rb1 = PROJ ? 0 : min(ng, rb0 + p.rpb);
    nleft = min(rb1, a.gram_left) - rb0;
    nload = PROJ ? a.nq + (a.mode == 1 ? 1 : 0) : nleft + 1;
    ncg = nload * p.cpb;
    mt = (rb1 - rb0) * p.cpb;
    n0 = PROJ ? blockIdx.y * p.npb : 0;
    np = PROJ ? min(p.npb, p.cpb - n0) : p.cpb;
    ncl = ncg * 8;
    dig = tsx_smem;
    raw = reinterpret_cast<zd *>(tsx_smem + p.o_raw);
    sums = tsx_smem + p.o_sums;
    coef = reinterpret_cast<uint32_t *>(tsx_smem + p.o_coef);
    nv = reinterpret_cast<double *>(tsx_smem + p.o_nv);
    int *at = reinterpret_cast<int *>(tsx_smem + p.o_int);
    rowkey = at;
    gam = rowkey + 4 * p.kt;
    key = reinterpret_cast<uint32_t *>(at);
    ecol = at + 4 * ncl;
    eacc = ecol + 4 * ncl;
    fcol = PROJ ? gam + ncl : eacc + ncl;
    flags = fcol + p.npb * 8;
    outp = reinterpret_cast<double2 *>(a.partial + (size_t)blockIdx.x * ng * a.r * a.r * 2);
  }
  __device__ __forceinline__ const zd *block(const TSArgs &a, int b) const {
    const bool left = PROJ ? b < a.nq : b < nleft;
    return reinterpret_cast<const zd *>(left ? a.q[rb0 + b] : a.src);
  }
};

__device__ __forceinline__ zd coef_at(const TSArgs &a, int b, int i, int j) {
  const int r = a.r;
  if (i >= r || j >= r) return mk<double>(0, 0);
  if (b < a.nq) return a.coefQ ? a.coefQ[(size_t)j * a.nq * r + b * r + i] : mk<double>(0, 0);
  return a.coefS ? a.coefS[(size_t)j * r + i] : mk<double>(0, 0);
}

// Exponents g of the coefficient rows of this CTA's columns; by the multiplying warps.
__device__ __forceinline__ void weigh_columns(const TSArgs &a, const XPlan &p, const Geo<true> &G) {
  const int c0 = G.n0 * 8, rc = min(G.np * 8, a.r - c0), tid = threadIdx.x;
  for (int k = tid; k < G.ncl; k += G.nt) G.gam[k] = 0;
  bar_sync(BAR_MUL, G.nt);
#pragma unroll 4
  for (int e = tid; e < G.ncl * rc; e += G.nt) {
    const int k = e % G.ncl, j = e / G.ncl;
    const zd v = coef_at(a, k / (p.cpb * 8), k % (p.cpb * 8), c0 + j);
    atomicMax(&G.gam[k], (int)max(mag_key(v.re), mag_key(v.im)));
  }
  bar_sync(BAR_MUL, G.nt);
  for (int k = tid; k < G.ncl; k += G.nt) {
    const int m = G.gam[k], g = (m >> 20) - 1022;
    G.gam[k] = m ? g : G_ZERO;
    if (m && abs(g) > X_GMAX) G.flags[0] = 1;   // also infinities and NaN: every tile directly
  }
}

// Digit planes of the weighted coefficients; by the multiplying warps.
__device__ __forceinline__ void slice_coefs(const TSArgs &a, const XPlan &p, const Geo<true> &G) {
  const int tid = threadIdx.x, cpb = p.cpb, np = G.np, c0 = G.n0 * 8;
  for (int j = tid; j < np * 8; j += G.nt) G.fcol[j] = E_UNSET;
  bar_sync(BAR_MUL, G.nt);
  for (int e = tid; e < G.ncg * 8 * np * 8; e += G.nt) {
    const int j = e / (G.ncg * 8), k = e % (G.ncg * 8), b = k / (cpb * 8), i = k % (cpb * 8);
    const zd v = coef_at(a, b, i, c0 + j);
    const uint32_t m = max(mag_key(v.re), mag_key(v.im));
    if (m >= (1u << 20)) atomicMax(&G.fcol[j], (int)(m >> 20) - 1022 - G.gam[k]);
  }
  bar_sync(BAR_MUL, G.nt);
  // word (group, column group, lane): rows 2q, 2q+1 of the group, output column g
  for (int e = tid; e < G.ncg * np * 32; e += G.nt) {
    const int l = e & 31, gn = e >> 5, n = gn % np, cg = gn / np;
    const int j = n * 8 + (l >> 2), b = cg / cpb, i = (cg % cpb) * 8 + 2 * (l & 3);
    const int f = G.fcol[j];
    uint32_t dr[NS], di[NS];
#pragma unroll
    for (int s = 0; s < NS; ++s) dr[s] = di[s] = 0;
    if (f != E_UNSET && !G.flags[0]) {
      const zd v0 = coef_at(a, b, i, c0 + j), v1 = coef_at(a, b, i + 1, c0 + j);
      const int k0 = 55 - f - G.gam[cg * 8 + 2 * (l & 3)], k1 = 55 - f - G.gam[cg * 8 + 2 * (l & 3) + 1];
      digit_planes(fixed_biased_k(v0.re, k0), fixed_biased_k(v1.re, k1), dr);
      digit_planes(fixed_biased_k(v0.im, k0), fixed_biased_k(v1.im, k1), di);
    }
    uint32_t *w = G.coef + (size_t)gn * NS * 64;
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      w[s * 64 + l] = dr[s];
      w[s * 64 + 32 + l] = di[s];
    }
  }
  bar_sync(BAR_MUL, G.nt);
}

// Direct path of an irregular tile in FP64 FMAs, by the multiplying warps.
__device__ __forceinline__ void direct_new(const TSArgs &a, const XPlan &p, const Geo<true> &G, long long row0) {
  const int r = a.r, c0 = G.n0 * 8, rc = min(G.np * 8, r - c0);
  for (int e = threadIdx.x; e < p.kt * rc; e += G.nt) {
    const int lr = e / rc, j = e % rc;
    const long long row = row0 + lr;
    zd s = mk<double>(0, 0);
    if (row >= a.zero_rows)
      for (int b = G.nload - 1; b >= 0; --b)
        for (int i = 0; i < r; ++i) fma_(s, G.block(a, b)[(size_t)row * r + i], coef_at(a, b, i, c0 + j));
    G.nv[lr * p.ldnv + 2 * j] = s.re;
    G.nv[lr * p.ldnv + 2 * j + 1] = s.im;
  }
}
__device__ __forceinline__ void direct_gram(const TSArgs &a, const XPlan &p, const Geo<false> &G, long long row0) {
  const int r = a.r, nr = (G.rb1 - G.rb0) * r;
  const zd *src = reinterpret_cast<const zd *>(a.src);
  for (int e = threadIdx.x; e < nr * r; e += G.nt) {
    const int j = e / nr, row = e % nr, b = row / r, i = row % r;
    const zd *left = b < G.nleft ? G.block(a, b) : src;
    zd s = mk<double>(0, 0);
    for (int lr = 0; lr < p.kt; ++lr) {
      const size_t at = (size_t)(row0 + lr) * r;
      fmac_(s, left[at + i], src[at + j]);
    }
    double2 *o = G.outp + (size_t)j * (a.gram_left + 1) * r + G.rb0 * r + row;
    double2 x = *o;
    x.x += s.re;
    x.y += s.im;
    *o = x;
  }
}

}  // namespace

// PROJ: new = [Q, S] coef, written.  Else: the partial Gram [q_0 .. q_{gl-1}, S]^* S.
template <bool PROJ>
__global__ void __launch_bounds__(X_THREADS, 1) tsx_kernel(const __grid_constant__ TSArgs a,
                                                           const __grid_constant__ XPlan p) {
  const Geo<PROJ> G(a, p);
  const int r = a.r, cpb = p.cpb, np = G.np, nkc = p.nkc, nt = G.nt, all = (p.wm + p.wc) * 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = lane >> 2, q = lane & 3;
  const int ncg = G.ncg, ncl = G.ncl;
  const uint32_t dig_a = (uint32_t)__cvta_generic_to_shared(G.dig);
  const int dig_words = nkc * ncg * NS * 128;   // of one buffer

  __shared__ __align__(8) unsigned long long full;   // the bulk copies of a tile
  const uint32_t full_a = (uint32_t)__cvta_generic_to_shared(&full);
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(full_a));
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  // thread nt (the first that cuts): the blocks' tiles by one bulk copy each
  const uint32_t tile_bytes = (uint32_t)p.kt * r * 16u;
  auto fetch = [&](long long tile) {
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(G.raw);
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(full_a), "r"(tile_bytes * G.nload) : "memory");
    for (int b = 0; b < G.nload; ++b)
      asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
                       dst + (uint32_t)(b * p.kt * r) * 16u),
                   "l"(G.block(a, b) + (size_t)tile * p.kt * r), "r"(tile_bytes), "r"(full_a)
                   : "memory");
  };
  if (tid < 12) G.flags[tid] = 0;
  if constexpr (PROJ) {
    for (int i = tid; i < 4 * p.kt; i += all) G.rowkey[i] = 0;
    __syncthreads();   // the flags and the barrier are set
    if (tid == nt) fetch(blockIdx.x);
    if (warp < p.wm) weigh_columns(a, p, G);
  } else {
    for (int i = tid; i < 4 * ncl; i += all) {
      G.key[i] = 0;
      G.ecol[i] = E_UNSET;
    }
    for (int i = tid; i < ncl; i += all) G.eacc[i] = E_UNSET;
    const int nr = (G.rb1 - G.rb0) * r;   // the partial: zero until the first flush
    for (int e = tid; e < nr * r; e += all)
      G.outp[(size_t)(e / nr) * (a.gram_left + 1) * r + G.rb0 * r + e % nr] = make_double2(0.0, 0.0);
  }
  __syncthreads();

  const long long ntiles = a.N / p.kt;
  const int mine = (int)((ntiles - blockIdx.x + gridDim.x - 1) / gridDim.x);   // tiles of this CTA

  if (warp >= p.wm) {
    // ==== cutting warps: tile i into digit planes i & 1, while the others multiply tile i - 1
    const int cw = warp - p.wm, ct = tid - nt, ncut = p.wc * 32;
    // units (group, chunk), worked out once so that the loop has no divisions: groups cw, cw + wc, .., all chunks
    const int nu = min(p.gpw, (ncg - cw + p.wc - 1) / p.wc) * nkc;
    int usrc[CUT_UNITS];   // the thread's first value in the tile (a padding column repeats the last one)
    int ucol[CUT_UNITS];   // its column
    int udig[CUT_UNITS];   // its word of the first digit plane
#pragma unroll
    for (int x = 0; x < CUT_UNITS; ++x) {
      const int cg = cw + (x / nkc) * p.wc, kc = x % nkc, b = cg / cpb, c = (cg - b * cpb) * 8 + g;
      ucol[x] = cg * 8 + g;
      usrc[x] = (b * p.kt + kc * 16 + q) * r + min(c, r - 1);
      udig[x] = (kc * ncg + cg) * NS * 128 + lane;
    }
    const int rs = 4 * r;
    uint32_t *const dig32 = reinterpret_cast<uint32_t *>(G.dig);
    if (!PROJ && ct == 0) fetch(blockIdx.x);
    for (int i = 0; i < mine; ++i) {
      uint32_t *key = G.key + (i & 3) * ncl;   // Gram
      // after a copy that never landed nothing more is fetched or waited for; the loop runs on for its barriers
      if (!G.flags[1] && !wait_phase(full_a, (uint32_t)(i & 1))) G.flags[1] = 1;
      zd raw[CUT_UNITS][4];
#pragma unroll
      for (int x = 0; x < CUT_UNITS; ++x)
        if (x < nu) {
          const zd *v = G.raw + usrc[x];
#pragma unroll
          for (int k = 0; k < 4; ++k) raw[x][k] = v[k * rs];
        }
      if constexpr (PROJ) {
        // the rows' largest weighted exponents over this warp's columns: per chunk, rows q + 4 k
        int rv[2][4] = {{0, 0, 0, 0}, {0, 0, 0, 0}};
#pragma unroll
        for (int x = 0; x < CUT_UNITS; ++x)
          if (x < nu) {
            const int gk = G.gam[ucol[x]];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const uint32_t m = max(mag_key(raw[x][k].re), mag_key(raw[x][k].im));
              const int E = (int)(m >> 20);
              // infinities and NaN count whatever their coefficients
              const int v = E == 0x7ff ? 1 << 20 : (m == 0 || gk == G_ZERO ? 0 : E + gk + X_BIAS);
              if (nkc == 1 || (x & 1) == 0) rv[0][k] = max(rv[0][k], v);
              else rv[1][k] = max(rv[1][k], v);
            }
          }
        int *rk = G.rowkey + (i & 3) * p.kt;
#pragma unroll
        for (int c = 0; c < 2; ++c)
          if (c < nkc) {   // over the columns (lane bits 2..4): halving the rows twice
            const bool u4 = lane & 16, u3 = lane & 8;
            const int s0 = u4 ? rv[c][0] : rv[c][2], s1 = u4 ? rv[c][1] : rv[c][3];
            const int a0 = max(u4 ? rv[c][2] : rv[c][0], __shfl_xor_sync(0xffffffffu, s0, 16));
            const int a1 = max(u4 ? rv[c][3] : rv[c][1], __shfl_xor_sync(0xffffffffu, s1, 16));
            int v = max(u3 ? a1 : a0, __shfl_xor_sync(0xffffffffu, u3 ? a0 : a1, 8));
            v = max(v, __shfl_xor_sync(0xffffffffu, v, 4));
            if (!(lane & 4) && v) atomicMax(&rk[c * 16 + q + (u4 ? 8 : 0) + (u3 ? 4 : 0)], v);
          }
        // the keys of tile i - 3 become those of tile i + 1 (they were last read before its planes were released)
        if (ct < p.kt) G.rowkey[((i + 1) & 3) * p.kt + ct] = 0;
      } else {
        uint32_t m = 0;
#pragma unroll
        for (int x = 0; x < CUT_UNITS; ++x)
          if (x < nu) {
#pragma unroll
            for (int k = 0; k < 4; ++k) m = max(m, max(mag_key(raw[x][k].re), mag_key(raw[x][k].im)));
            if (((x + 1) & (nkc - 1)) == 0) {   // the group's last chunk (nkc is 1 or 2): over the lanes of a column
              m = max(m, __shfl_xor_sync(0xffffffffu, m, 1));
              m = max(m, __shfl_xor_sync(0xffffffffu, m, 2));
              if (q == 0) key[ucol[x]] = m;
              m = 0;
            }
          }
      }
      bar_sync(BAR_CUT, ncut);   // the raw tile is in registers: the next one goes out behind the arithmetic
      if (ct == 0 && i + 1 < mine && !G.flags[1]) fetch(blockIdx.x + (long long)(i + 1) * gridDim.x);
      // planes i & 1 are free once tile i - 2 is multiplied; its flags go with them
      if (i >= 2) bar_sync(BAR_FREE + (i & 1), all);
      int *flag = G.flags + 4 + 2 * (i & 3);
      const int *el = G.ecol + ((i + 3) & 3) * ncl;   // Gram, before this tile: those of tile i - 1
      uint32_t *cut = dig32 + (i & 1) * dig_words;
      int e = 0;
#pragma unroll
      for (int x = 0; x < CUT_UNITS; ++x)
        if (x < nu) {
          int er[4];   // the exponents of the four values
          if constexpr (PROJ) {
            const int *rk = G.rowkey + (i & 3) * p.kt + (x & (nkc - 1)) * 16 + q, gk = G.gam[ucol[x]];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const int v = rk[4 * k], ex = v - X_BIAS - 1022;
              if (v && (ex < X_RMIN || ex > X_RMAX)) flag[1] = 1;
              er[k] = (v ? ex : 0) - gk;
            }
          } else {
            if ((x & (nkc - 1)) == 0) {
              const uint32_t k = key[ucol[x]];
              const int E = (int)(k >> 20), ex = E - 1022;   // |x| < 2^ex
              e = el[ucol[x]];
              if (k != 0 && (E < X_EMIN || E > X_EMAX)) {
                flag[1] = 1;
              } else if (k != 0 && (ex > e || ex < e - X_SLACK)) {
                atomicOr(flag, ex > e ? X_RAISED : X_LOWERED);
                e = e == E_UNSET ? ex + 1 : ex;
              }
              G.ecol[(i & 3) * ncl + ucol[x]] = e;
              if (e == E_UNSET) e = 0;   // zero so far: any exponent gives zero digits
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) er[k] = e;
          }
          uint32_t *w = cut + udig[x];
#pragma unroll
          for (int h = 0; h < 2; ++h) {   // rows q, q+4 and rows q+8, q+12; matrices re, re, im, im
            uint32_t dr[NS], di[NS];
            const zd u = raw[x][2 * h], v = raw[x][2 * h + 1];
            digit_planes(fixed_biased(u.re, er[2 * h]), fixed_biased(v.re, er[2 * h + 1]), dr);
            digit_planes(fixed_biased(u.im, er[2 * h]), fixed_biased(v.im, er[2 * h + 1]), di);
#pragma unroll
            for (int s = 0; s < NS; ++s) {
              w[s * 128 + h * 32] = dr[s];
              w[s * 128 + 64 + h * 32] = di[s];
            }
          }
        }
      if (ct == 0) G.flags[4 + 2 * ((i + 2) & 3)] = G.flags[5 + 2 * ((i + 2) & 3)] = 0;   // tile i - 2's
      bar_arrive(BAR_FULL + (i & 1), all);
    }
    // the last planes' releases, so that every barrier completes
    for (int i = max(mine, 2); i < mine + 2; ++i) bar_sync(BAR_FREE + (i & 1), all);
    if (ct == 0 && G.flags[1] && a.status) atomicOr(a.status, ST_TIMEOUT);
    return;
  }

  // ==== multiplying warps
  if constexpr (PROJ) {
    slice_coefs(a, p, G);
    zd *out = reinterpret_cast<zd *>(a.out);
    const int c0 = G.n0 * 8, rc = min(np * 8, r - c0);
    for (int i = 0; i < mine; ++i) {
      const long long row0 = (blockIdx.x + (long long)i * gridDim.x) * p.kt;
      const int *rk = G.rowkey + (i & 3) * p.kt;
      bar_sync(BAR_FULL + (i & 1), all);
      const bool direct = G.flags[5 + 2 * (i & 3)] != 0 || G.flags[0] != 0;
      if (direct) {
        direct_new(a, p, G, row0);
      } else {
        // item (16 rows, 8 columns, re or im)
        for (int t = warp; t < nkc * np * 2; t += p.wm) {
          const int h = t & 1, n = (t >> 1) % np, kc = (t >> 1) / np;
          float pa[NS][4];
#pragma unroll
          for (int w = 0; w < NS; ++w)
#pragma unroll
            for (int k = 0; k < 4; ++k) pa[w][k] = 0.f;
          long long hh[4] = {0, 0, 0, 0}, ll[4] = {0, 0, 0, 0};
          auto drain = [&]() {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              float c[NS];
#pragma unroll
              for (int w2 = 0; w2 < NS; ++w2) {
                c[w2] = pa[w2][k];
                pa[w2][k] = 0.f;
              }
              long long x, y;
              class_ints(c, x, y);
              hh[k] += x;
              ll[k] += y;
            }
          };
          const uint32_t *w = G.coef + (size_t)n * NS * 64 + lane;
          uint32_t ad = dig_a + (uint32_t)((i & 1) * dig_words) * 4u + (uint32_t)(kc * ncg * NS) * 512u + lane * 16u;
#pragma unroll 2
          for (int cg = 0; cg < ncg; ++cg, w += np * NS * 64, ad += NS * 512u) {
            uint32_t b0[NS], b1[NS];
#pragma unroll
            for (int s = 0; s < NS; ++s) {
              const uint32_t cr = w[s * 64], ci = w[s * 64 + 32];
              b0[s] = h ? ci : cr;
              b1[s] = h ? cr : ci ^ NEG2;   // re: re.re - im.im, im: re.im + im.re
            }
#pragma unroll
            for (int s = 0; s < NS; ++s) {
              uint32_t av[4];
              ldsm4t(av, ad + s * 512u);
#pragma unroll
              for (int u = 0; u + s < NS; ++u) mma16816(pa[s + u], av, b0[u], b1[u]);
            }
            if ((cg + 1) % (X_DRAIN / 8) == 0) drain();
          }
          drain();
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            // fragment row k of a chunk is row (k & 8) + 4 (k & 1) + (k & 7) / 2
            const int lr = kc * 16 + (k >= 2 ? 8 : 0) + (g & 1) * 4 + (g >> 1), j = n * 8 + 2 * q + (k & 1);
            if (c0 + j >= r) continue;
            const long long row = row0 + lr;
            const int f = G.fcol[j];
            double v = 0.0;
            if (f != E_UNSET && row >= a.zero_rows) v = ints_value(hh[k], ll[k], rk[lr] - X_BIAS - 1022 + f - 14);
            G.nv[lr * p.ldnv + 2 * j + h] = v;
          }
        }
      }
      bar_arrive(BAR_FREE + (i & 1), all);
      bar_sync(BAR_MUL, nt);
      for (int e = tid; e < p.kt * rc; e += nt) {
        const int lr = e / rc, j = e - lr * rc;
        out[(size_t)(row0 + lr) * r + c0 + j] = mk<double>(G.nv[lr * p.ldnv + 2 * j], G.nv[lr * p.ldnv + 2 * j + 1]);
      }
    }
  } else {
    // Gram item of this warp: row groups mg0, mg0 + 1 against column group in0
    const int item = warp % p.items, kg = warp / p.items;
    const bool has_item = kg < p.ksplit;
    const int mg0 = 2 * (item / np), in0 = item % np, nl = G.nleft * cpb;
    // the group in the planes of Gram row group m (m >= nl: G's column group m - nl)
    auto group = [&](int m) { return m < nl ? m : (G.nload - 1) * cpb + (m - nl); };
    const int ga = group(min(mg0, G.mt - 1)), gb = group(min(mg0 + 1, G.mt - 1)), gg = group(nl);
    // left operand: (group 0, group 1) x (rows 0-7, rows 8-15) of one part, one matrix per 8 lanes
    const uint32_t a_at = dig_a + (uint32_t)((lane & 8 ? gb : ga) * NS) * 512u + (lane >> 4) * 128u + (lane & 7) * 16u;
    const uint32_t b_at = dig_a + (uint32_t)((gg + in0) * NS) * 512u + lane * 16u;
    float acc[2][NS][4];
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int w = 0; w < NS; ++w)
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[h][w][k] = 0.f;
    const uint32_t sums = (uint32_t)__cvta_generic_to_shared(G.sums) + tid * 16u, sum_step = nt * 16u;
    auto clear_sums = [&]() {
      const Sum z{0, 0};
#pragma unroll
      for (int e = 0; e < 8; ++e) z.store(sums + e * sum_step);
    };
    clear_sums();
    auto drain = [&]() {
      if (!has_item) return;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        Sum s[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) s[k].load(sums + (h * 4 + k) * sum_step);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          float c[NS];
#pragma unroll
          for (int w = 0; w < NS; ++w) {
            c[w] = acc[h][w][k];
            acc[h][w][k] = 0.f;
          }
          long long x, y;
          class_ints(c, x, y);
          s[k].h += x;
          s[k].l += y;
          s[k].store(sums + (h * 4 + k) * sum_step);
        }
      }
    };
    // the sums into the FP64 partial, at the exponents they were made with; then cleared, for the exponents el.
    // Called by every multiplying thread; warps that share an item take turns.
    const int ldg_ = (a.gram_left + 1) * r;
    auto flush = [&](const int *el) {
      for (int k = 0; k < p.ksplit; ++k) {
        bar_sync(BAR_MUL, nt);
        if (!has_item || kg != k) continue;
#pragma unroll
        for (int x = 0; x < 4; ++x) {
          const int mg = mg0 + (x >> 1);
          if (mg >= G.mt) continue;
          const int col = (mg % cpb) * 8 + g, j = in0 * 8 + 2 * q + (x & 1);
          if (col >= r || j >= r) continue;
          const int e0 = G.eacc[(x < 2 ? ga : gb) * 8 + g], e1 = G.eacc[gg * 8 + j];
          if (e0 == E_UNSET || e1 == E_UNSET) continue;      // a column that has been zero so far
          double2 *o = G.outp + (size_t)j * ldg_ + (G.rb0 + mg / cpb) * r + col;
          double2 v = *o;
          Sum re, im;
          re.load(sums + x * sum_step);
          im.load(sums + (4 + x) * sum_step);
          v.x += ints_value(re.h, re.l, e0 + e1 - 14);
          v.y += ints_value(im.h, im.l, e0 + e1 - 14);
          *o = v;
        }
      }
      bar_sync(BAR_MUL, nt);
      for (int c = tid; c < ncl; c += nt) G.eacc[c] = el[c];
      clear_sums();
    };
    // the sums for larger exponents el: down by the bits that an entry's two columns rose
    auto shift = [&](const int *el) {
      bar_sync(BAR_MUL, nt);
      if (has_item)
#pragma unroll
        for (int x = 0; x < 4; ++x) {
          const int c0 = (x < 2 ? ga : gb) * 8 + g, c1 = gg * 8 + in0 * 8 + 2 * q + (x & 1);
          if (G.eacc[c0] == E_UNSET || G.eacc[c1] == E_UNSET) continue;   // zero so far
          const int k = el[c0] - G.eacc[c0] + el[c1] - G.eacc[c1];
          if (k == 0) continue;
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            Sum v;
            v.load(sums + (h * 4 + x) * sum_step);
            v.down(k);
            v.store(sums + (h * 4 + x) * sum_step);
          }
        }
      bar_sync(BAR_MUL, nt);
      for (int c = tid; c < ncl; c += nt) G.eacc[c] = el[c];
    };
    int since = 0;                // rows in the accumulators since the last drain or flush
    for (int i = 0; i < mine; ++i) {
      bar_sync(BAR_FULL + (i & 1), all);
      const int changed = G.flags[4 + 2 * (i & 3)];
      const bool direct = G.flags[5 + 2 * (i & 3)] != 0;
      if (changed) {
        if (since > 0) drain();
        if (changed & X_LOWERED) flush(G.ecol + (i & 3) * ncl);
        else shift(G.ecol + (i & 3) * ncl);
        since = 0;
      }
      if (direct) {
        direct_gram(a, p, *reinterpret_cast<const Geo<false> *>(&G), (blockIdx.x + (long long)i * gridDim.x) * p.kt);
      } else {
        if (has_item)
          for (int kc = kg; kc < nkc; kc += p.ksplit) {
            const uint32_t off = (uint32_t)(((i & 1) * nkc + kc) * ncg * NS) * 512u;
            uint32_t bd[NS][4];   // re rows 0-7, 8-15, im rows 0-7, 8-15
#pragma unroll
            for (int s = 0; s < NS; ++s) ldsm4(bd[s], b_at + off + s * 512u);
#pragma unroll
            for (int s = 0; s < NS; ++s) {
              uint32_t are[4], aim[4];
              ldsm4(are, a_at + off + s * 512u);
              ldsm4(aim, a_at + off + s * 512u + 256u);
#pragma unroll
              for (int u = 0; u + s < NS; ++u) {   // re: re.re + im.im, im: re.im - im.re
                const uint32_t(&b)[4] = bd[u];
                mma16816(acc[0][s + u], are, b[0], b[1]);
                mma16816(acc[0][s + u], aim, b[2], b[3]);
                mma16816(acc[1][s + u], are, b[2], b[3]);
                mma16816(acc[1][s + u], aim, b[0] ^ NEG2, b[1] ^ NEG2);
              }
            }
          }
        since += p.kt;
      }
      bar_arrive(BAR_FREE + (i & 1), all);
      if (since == X_DRAIN) {
        drain();
        since = 0;
      }
    }
    drain();
    flush(G.ecol);
  }
}

// ---------------------------------------------------------------- launch
namespace {

constexpr int TSX_SMEM = 227 * 1024 - 128;   // dynamic; the barrier is static

// Shapes of one launch: false when it does not fit a CTA.
bool tsx_plan(const TSArgs &a, bool proj, XPlan *out) {
  const int maxw = X_THREADS / 32, r = a.r, ng = a.gram_left + 1, cpb = (r + 7) / 8;
  auto items_of = [&](int blocks) { return ((blocks * cpb + 1) / 2) * cpb; };
  int rpb = ng;
  if (!proj)
    while (rpb > 1 && items_of(rpb) > 10) --rpb;
  const int items = proj ? 0 : items_of(rpb);
  if (items > 10) return false;
  const int nload = proj ? a.nq + (a.mode == 1 ? 1 : 0) : rpb + (rpb > a.gram_left ? 0 : 1);
  const int ncg = nload * cpb;
  if (nload < 1) return false;
  // a projection in place must read a tile's rows before any of its columns are written: no split by columns
  bool in_place = proj && a.mode == 1 && a.src == a.out;
  for (int m = 0; m < a.nq; ++m) in_place = in_place || (proj && a.q[m] == a.out);
  for (int split = 1; split <= (proj && !in_place ? cpb : 1); ++split)
    for (int kt = 32; kt >= 16; kt /= 2) {
      XPlan p{};
      p.cpb = cpb;
      p.kt = kt;
      p.nkc = kt / 16;
      p.rpb = rpb;
      p.npb = (cpb + split - 1) / split;
      p.items = std::max(1, items);
      p.ksplit = 1;
      while (!proj && p.ksplit * 2 <= p.nkc && items * p.ksplit * 2 <= 8) p.ksplit *= 2;
      // multiplying warps: one per Gram item and chunk share, or one per 16 x 8 tile of the product
      p.wm = std::max(2, proj ? std::min(8, p.nkc * p.npb * 2) : items * p.ksplit);
      p.wc = std::min(ncg, maxw - p.wm);
      p.gpw = (ncg + p.wc - 1) / p.wc;
      if (p.gpw * p.nkc > CUT_UNITS) continue;
      p.ldnv = 2 * p.npb * 8 + 2;
      int b = 2 * p.nkc * ncg * NS * 512;
      p.o_raw = b;
      b += nload * kt * r * 16;   // a multiple of 128 bytes
      p.o_sums = b;
      b += proj ? 0 : p.wm * 32 * 8 * 16;
      p.o_coef = b;
      b += proj ? ncg * p.npb * NS * 256 : 0;
      p.o_nv = b;
      b += proj ? kt * p.ldnv * 8 : 0;
      b = (b + 15) & ~15;
      p.o_int = b;
      b += ((proj ? 4 * kt + ncg * 8 : 9 * ncg * 8) + p.npb * 8 + 12) * 4;
      p.bytes = b;
      if (b > TSX_SMEM) continue;
      *out = p;
      return true;
    }
  return false;
}

int tsx_run(const TSArgs &a, bool proj, const XPlan &p, int nsm, cudaStream_t st) {
  const int ng = a.gram_left + 1, gy = proj ? (p.cpb + p.npb - 1) / p.npb : (ng + p.rpb - 1) / p.rpb, w = p.wm + p.wc;
  // persistent: as many CTAs as fit an SM by registers (128 a thread: 16 warps) and shared memory
  const int occ = std::max(1, std::min(16 / w, 228 * 1024 / (p.bytes + 2048)));
  const long long ntiles = a.N / p.kt;
  long long gx = (long long)occ * nsm / gy;
  // the caller's buffer holds at least 2 nsm partials of MAXB + 1 blocks
  if (!proj) gx = std::min(gx, 2LL * nsm * (MAXB + 1) / ng);
  gx = std::max(1LL, std::min(gx, ntiles));
  const dim3 grid((unsigned)gx, (unsigned)gy);
  ::lrei::count_launch();
  if (proj) tsx_kernel<true><<<grid, w * 32, p.bytes, st>>>(a, p);
  else tsx_kernel<false><<<grid, w * 32, p.bytes, st>>>(a, p);
  return (int)gx;
}
}  // namespace

// The pass by tsx_kernel: the number of partials, or 0 when it does not apply (H.V fused, an operand that a bulk
// copy cannot read, too wide for a CTA's shared memory, or fewer than 256 rows: there the general kernel's FMAs are
// as fast (about 20 us, all latency) and its sums a little closer).  Modes 1 and 2 are a projection and the Gram of what it
// wrote: in one kernel the projection's planes, the coefficients' and the Gram's sums leave shared memory for
// 16-row tiles only, and the pass was slower than the two (n = 20, r = 16, five blocks: 7.1 ms against 2.6 + 1.9).
// Measured against the general kernel (ts2_kernel) at n = 20, r = 16: Gram of 1 / 2 / 3 / 5 Krylov blocks 1.83 / 3.66 / 5.55 /
// 10.96 ms there and 0.24 / 0.47 / 0.62 / 0.91 ms here (the five blocks' tensor work alone is 0.47 ms), an RK4 step 96.0 and
// 15.1 ms.
int launch_tsx(const TSArgs &a, int nsm, cudaStream_t st) {
  if ((a.mode == 0 && a.out) || (a.mode != 0 && !a.out) || a.r > MAX_R || a.N < 256) return 0;
  auto off = [](const void *x) { return (reinterpret_cast<uintptr_t>(x) & 15) != 0; };
  for (int m = 0; m < a.nq; ++m)
    if (off(a.q[m])) return 0;
  if ((a.mode != 2 && off(a.src)) || (a.mode != 0 && off(a.out))) return 0;
  XPlan p, pg;
  TSArgs b = a;
  // projections of ranks 1 and 2 from 2^16 rows on: eight columns are cut for one or two, and the FMAs of so few cost less (r = 1, five
  // blocks at n = 18: 150 us there, 218 here; at n = 14 29 and 28)
  if (a.mode != 0 && a.r <= 2 && a.N >= 65536) return 0;
  if (a.mode != 0) {
    b.mode = 0;
    b.src = a.out;
    b.out = nullptr;
    b.nq = a.gram_left;
    for (int m = 0; m < a.gram_left; ++m)
      if (a.q[m] == a.out) return 0;   // the Gram would read the new block in the left one's place
    if (!tsx_plan(a, true, &p)) return 0;
  }
  if (!tsx_plan(b, false, &pg)) return 0;
  if (a.mode != 0) tsx_run(a, true, p, nsm, st);
  return tsx_run(b, false, pg, nsm, st);
}

int tsx_init() {
  for (const void *f : {(const void *)tsx_kernel<true>, (const void *)tsx_kernel<false>})
    if (cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, TSX_SMEM) != cudaSuccess) return -1;
  return 0;
}

}  // namespace lrei
