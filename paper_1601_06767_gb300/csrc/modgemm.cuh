// FP64 complex products on the 16-bit tensor cores by exact modular arithmetic.
//
//   C[m][n] = sum_k A[m][k] B[n][k]        (complex, FP64 accuracy)
//
// Every row of A and B is scaled by a power of two and rounded to complex
// integers of at most 2^57 (A) and 2^56 (B) in Euclidean norm, so that every
// component of C is an integer below 2^113 in magnitude (Cauchy-Schwarz).  It is
// then determined by its residues modulo the 13 pairwise coprime m_i below,
// whose product P has 2^113.36 < P / 2 (multi-modulus integer products: the
// residue number system with the Chinese remainder theorem).  All prime factors
// of every m_i are 1 mod 4, so an integer I with I^2 = -1 (mod m_i) exists and
//   x + i y  ->  (u, v) = (x + I y, x - I y)  (mod m_i)
// turns one complex product into two independent real ones: 26 real products for
// 13 moduli, where a digit split of 54 bits into six 9-bit terms needs 84.
// Residues are centred (|r| <= 255), exact in FP16, and a sum of 256 products is
// at most 255^2 256 < 2^24: exact in the tensor cores' FP32 accumulators, in any
// order and rounding.  The only error is the rounding to integers, about 0.08 x
// 2^-53 of |A_m| |B_n| (0.3 x 2^-53 for the same sum by FP64 fused multiply-adds
// over Gaussian rows).
//
// That is FP64 accuracy while S = sum_k |A[m][k]| |B[n][k]|, what FP64 sums are accurate
// to, is not far below |A_m| |B_n|; rows that live on different k have a smaller S.
// One more plane per operand (CHECK_PLANE) carries the elements' magnitudes, its
// product is S, and tiles with an S below CHECK_MIN of the norms are computed by
// FP64 multiply-adds instead (k_mod_check; dense Gaussian rows have 0.6, the largest
// error let through is 0.08 x 32 x 2^-53 of S).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace chi0 {
namespace mod {

constexpr int NM = 13;               // moduli
constexpr int NPL = 2 * NM;          // residue planes (u and v of every modulus)
constexpr int CHECK_PLANE = NPL;     // magnitudes, norm below 2^CHECK_BITS
constexpr int CPL = NPL + 1;         // planes of a checked product
constexpr int CHECK_BITS = 7;
constexpr int RPL = NPL + 8;         // planes of a product with the remainders (store_remainders)
enum Extra { PLAIN, CHECK, REST };   // what follows the residues
constexpr float CHECK_MIN = 1.0f / 32;
constexpr int BETA_A = 57, BETA_B = 56;   // bits of the rows' norms after scaling
constexpr int NO_SCALE = -(1 << 28);      // scale exponent of a row holding an infinity or a NaN

typedef unsigned __int128 u128;

constexpr int NL = 5, LB = 12;        // limbs of a scaled integer: 12 bits each, the last one signed

struct Tables {
  int m[NM] = {509, 505, 493, 481, 461, 457, 449, 433, 421, 409, 401, 397, 389};
  int c[NM][NL] = {}, ic[NM][NL] = {};            // 2^(12 j) and I 2^(12 j) (mod m), centred
  // C = sum_i s_i a_i (mod 1) in units of P, s = u + v for the real part and u - v for the
  // imaginary part: a 96-bit fraction in three words, the lower two balanced (signed)
  int re[NM][3] = {}, im[NM][3] = {};
  uint64_t p_top = 0;                             // P = p_top 2^p_exp, top bit set
  int p_exp = 0;
};

constexpr int cinv_mod(int a, int m) {            // by search: the moduli are small
  for (int x = 1; x < m; ++x)
    if ((int64_t)a * x % m == 1) return x;
  return 0;
}
constexpr int centred(int x, int m) { return x > m / 2 ? x - m : x; }

constexpr Tables make_tables() {
  Tables t;
  u128 P = 1;
  for (int i = 0; i < NM; ++i) P *= (unsigned)t.m[i];
  for (int i = 0; i < NM; ++i) {
    const int m = t.m[i];
    int I = 0;
    for (int x = 2; x < m && !I; ++x)
      if (x * x % m == m - 1) I = x;
    for (int j = 0, pw = 1; j < NL; ++j, pw = pw * ((1 << LB) % m) % m) {
      t.c[i][j] = centred(pw, m);
      t.ic[i][j] = centred(I * pw % m, m);
    }
    int q = 1;                                    // P / m (mod m)
    for (int j = 0; j < NM; ++j)
      if (j != i) q = q * (t.m[j] % m) % m;
    const int w = cinv_mod(q, m), half = cinv_mod(2, m);
    const int ar = w * half % m, ai = ar * cinv_mod(I, m) % m;
    for (int c = 0; c < 2; ++c) {
      const u128 f = (((u128)(unsigned)(c ? ai : ar) << 97) / (unsigned)m + 1) >> 1;   // rounded, below 2^96
      int* o = c ? t.im[i] : t.re[i];
      o[2] = (int)(uint32_t)f;
      const u128 f1 = (f >> 32) + (o[2] < 0 ? 1 : 0);
      o[1] = (int)(uint32_t)f1;
      o[0] = (int)(uint32_t)((f1 >> 32) + (o[1] < 0 ? 1 : 0));
    }
  }
  int top = 127;
  while (!(P >> top)) --top;
  t.p_exp = top - 63;
  t.p_top = (uint64_t)(P >> t.p_exp);
  return t;
}
constexpr Tables T = make_tables();
static_assert(T.p_exp + 64 == 115 && T.p_top >> 63, "P has 115 bits");
// P / 2 > 2^(BETA_A + BETA_B) with more than a quarter to spare for the rounding of the rows
static_assert((T.p_top >> 60) >= 10, "P / 2 covers the largest component");

// the constants of modulus I as compile-time scalars (device code takes them as immediates)
template <int I> struct Mod {
  static constexpr float m = (float)T.m[I], inv = 1.0f / (float)T.m[I];
  static constexpr float c1 = T.c[I][1], c2 = T.c[I][2], c3 = T.c[I][3], c4 = T.c[I][4];   // c[0] = 1
  static constexpr float i0 = T.ic[I][0], i1 = T.ic[I][1], i2 = T.ic[I][2], i3 = T.ic[I][3], i4 = T.ic[I][4];
  static constexpr int re0 = T.re[I][0], re1 = T.re[I][1], re2 = T.re[I][2];
  static constexpr int im0 = T.im[I][0], im1 = T.im[I][1], im2 = T.im[I][2];
};
constexpr uint64_t P_TOP = T.p_top;
constexpr int P_EXP = T.p_exp;

// ---------------------------------------------------------------------------
// scaling and rounding of a row
// ---------------------------------------------------------------------------
// high word of |x|: orders magnitudes, 0x7ff00000 and above for infinities and NaN
__device__ __forceinline__ uint32_t mag_word(double x) { return (uint32_t)__double2hiint(x) & 0x7fffffffu; }

// 2^k as a double for -1022 <= k <= 1023
__device__ __forceinline__ double pow2d(int k) { return __hiloint2double((k + 1023) << 20, 0); }

// exponent e with x < 2^(e + 1) for the largest magnitude word of a set (0 for zeros and subnormals)
__device__ __forceinline__ int word_exp(uint32_t w) { return (int)(w >> 20) - 1023; }

// scale exponent s with norm 2^s <= 2^beta, from norm^2 = n2 4^e (n2 > 0, to a relative 1e-5)
__device__ __forceinline__ int scale_exp(double n2, int e, int beta) {
  if (!(n2 > 0.0)) return 0;                      // a row of zeros
  int k;
  frexp(n2 * (1.0 + 2e-5), &k);                   // n2 < 2^k
  return beta - e - ((k + 1) >> 1);               // norm < 2^(e + k / 2)
}

// norm 2^(s - beta) in [0.5, 1), s the scale exponent of a row with norm^2 = n2 4^e (0 for zeros, NaN
// for non-finite rows)
__device__ __forceinline__ float scaled_norm(double n2, int s, int e, int beta) {
  if (s == NO_SCALE) return nanf("");
  return n2 > 0.0 ? (float)scalbn(sqrt(n2), s + e - beta) : 0.f;
}

// |x| 2^-e truncated to FP32, for |x| < 2^(e + 1) (integer operations; zero below 2^(e - 126))
__device__ __forceinline__ float scaled_abs(double x, int e) {
  const uint32_t hi = mag_word(x), lo = (uint32_t)__double2loint(x);
  const int ef = (int)(hi >> 20) - 1023 - e + 127;
  return ef > 0 ? __uint_as_float(((uint32_t)ef << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29)) : 0.f;
}

// round(x 2^s) for |x 2^s| < 2^58 (integer operations only: the FP64 pipe is narrow)
__device__ __forceinline__ int64_t quantise(double x, int s) {
  const int64_t b = __double_as_longlong(x);
  const int e = (int)((b >> 52) & 0x7ff);
  const uint64_t man = ((uint64_t)b & 0xfffffffffffffull) | 0x10000000000000ull;
  const int sh = e - 1075 + s;
  uint64_t q;
  if (sh >= 0) q = man << min(sh, 6);
  else q = sh < -54 ? 0ull : (man + (1ull << (-sh - 1))) >> -sh;
  if (e == 0) q = 0;
  return b < 0 ? -(int64_t)q : (int64_t)q;
}

// packed FP32 pairs
__device__ __forceinline__ uint64_t pack2(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ uint64_t both(float x) { return pack2(x, x); }

// limbs of two signed integers below 2^58 as packed FP32 numbers: a = sum_j l_j 2^(12 j)
struct Limbs {
  uint64_t l[NL];
};
__device__ __forceinline__ Limbs limbs(int64_t a, int64_t b) {
  const int al = (int)a, ah = (int)(a >> 32), bl = (int)b, bh = (int)(b >> 32);
  const int x[NL] = {al & 0xfff, (al >> 12) & 0xfff, (int)__funnelshift_r(al, ah, 24) & 0xfff, (ah >> 4) & 0xfff, ah >> 16};
  const int y[NL] = {bl & 0xfff, (bl >> 12) & 0xfff, (int)__funnelshift_r(bl, bh, 24) & 0xfff, (bh >> 4) & 0xfff, bh >> 16};
  Limbs r;
#pragma unroll
  for (int j = 0; j < NL; ++j)    // integers below 2^22 in magnitude
    r.l[j] = add2(pack2(__int_as_float(x[j] + 0x4b400000), __int_as_float(y[j] + 0x4b400000)), both(-12582912.f));
  return r;
}

// x - m round(x / m) for integers |x| < 2^24: |result| <= 255 (the quotient is within 2^-9 of exact)
template <int I>
__device__ __forceinline__ uint32_t residue2(uint64_t x) {
  const uint64_t q = add2(fma2(x, both(Mod<I>::inv), both(12582912.f)), both(-12582912.f));
  float lo, hi;
  unpack2(fma2(q, both(-Mod<I>::m), x), lo, hi);
  uint32_t r;
  asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}

// residues (u, v) modulo m_I of two complex integers (k and k + 1; limbs of the real and imaginary
// parts): a packed FP16 pair of each.  Packed FP32 multiply-adds on 12-bit limbs: every sum is an
// integer below 2 x 254 x (4 x 4095 + 512) < 2^23.04, exact.
template <int I>
__device__ __forceinline__ void residues2(const Limbs& x, const Limbs& y, uint32_t& u, uint32_t& v) {
  using C = Mod<I>;
  uint64_t a = fma2(both(C::c1), x.l[1], x.l[0]);
  a = fma2(both(C::c2), x.l[2], a);
  a = fma2(both(C::c3), x.l[3], a);
  a = fma2(both(C::c4), x.l[4], a);
  uint64_t b = mul2(both(C::i0), y.l[0]);
  b = fma2(both(C::i1), y.l[1], b);
  b = fma2(both(C::i2), y.l[2], b);
  b = fma2(both(C::i3), y.l[3], b);
  b = fma2(both(C::i4), y.l[4], b);
  u = residue2<I>(add2(a, b));
  v = residue2<I>(fma2(b, both(-1.f), a));
}

// all residues of two complex integers into planes of `plane` words each: u of modulus i at
// plane 2 i, v at 2 i + 1 (conj: of the conjugates, u and v exchanged)
template <int I = 0>
__device__ __forceinline__ void store_residues(const Limbs& x, const Limbs& y, bool conj, uint32_t* __restrict__ dst,
                                               size_t plane) {
  uint32_t u, v;
  residues2<I>(x, y, u, v);
  dst[(2 * I) * plane] = conj ? v : u;
  dst[(2 * I + 1) * plane] = conj ? u : v;
  if constexpr (I + 1 < NM) store_residues<I + 1>(x, y, conj, dst, plane);
}

// largest component of each of the two elements, scaled to norms of at most 2^CHECK_BITS (beta: BETA_A or
// BETA_B), into the plane after the residues: no more than the magnitude and 2^-21 of the norm, no
// less than 0.7 of it
__device__ __forceinline__ void store_magnitudes(const Limbs& x, const Limbs& y, int beta, uint32_t* __restrict__ dst,
                                                 size_t plane) {
  float a, b, c, d;
  unpack2(fma2(x.l[4], both(4096.f), x.l[3]), a, b);          // 2^-36 of the integers
  unpack2(fma2(y.l[4], both(4096.f), y.l[3]), c, d);
  const float s = __int_as_float((127 + 36 + CHECK_BITS - beta) << 23);
  uint32_t r;
  asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(s * fmaxf(fabsf(b), fabsf(d))), "f"(s * fmaxf(fabsf(a), fabsf(c))));
  dst[CHECK_PLANE * plane] = r;
}

// The first order of what the rounding to integers leaves out of A B: with A = Ah + Al and B = Bh + Bl (integers
// and remainders below 1/2), Al Bh + Ah Bl as eight real products in planes NPL .. RPL, to some 2^-7 of it.
// Remainders as they are, integers scaled to norms of at most 2^CHECK_BITS; the order of the parts gives
//   Re: + (0) - (1) + (4) - (5),   Im: + (2) + (3) + (6) + (7).
// The sums stay below 2^15: the remainders' norm is at most 2^7.5 for 2^16 elements.
__device__ __forceinline__ float rest_of(double x, int s, int64_t q) {
  return (float)(x * pow2d(s / 2) * pow2d(s - s / 2) - (double)q);      // exact: both are multiples of x's last bit
}
__device__ __forceinline__ void store_remainders(const Limbs& x, const Limbs& y, uint64_t rx, uint64_t ry, int beta,
                                                 uint32_t* __restrict__ dst, size_t plane) {
  const uint64_t s = both(__int_as_float((127 + 36 + CHECK_BITS - beta) << 23));
  const uint64_t v[4] = {rx, ry, mul2(s, fma2(x.l[4], both(4096.f), x.l[3])), mul2(s, fma2(y.l[4], both(4096.f), y.l[3]))};
  uint32_t h[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float a, b;
    unpack2(v[i], a, b);
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(h[i]) : "f"(b), "f"(a));
  }
  const bool A = beta == BETA_A;
  const uint32_t lr = h[0], li = h[1], hr = h[2], hi = h[3];
  const uint32_t o[8] = {A ? lr : hr, A ? li : hi, A ? lr : hi, A ? li : hr, A ? hr : lr, A ? hi : li, A ? hr : li, A ? hi : lr};
#pragma unroll
  for (int i = 0; i < 8; ++i) dst[(NPL + i) * plane] = o[i];
}

// ---------------------------------------------------------------------------
// reconstruction
// ---------------------------------------------------------------------------
// f += s a with a 96-bit fraction a (mod 1): three multiply-adds, the sums of the products with
// the three words kept apart (fraction = top 2^-32 + mid 2^-64 + lo 2^-96)
struct Frac {
  uint32_t top;
  int64_t mid, lo;
};
__device__ __forceinline__ void frac_add(Frac& f, int s, int a0, int a1, int a2) {
  f.lo += (int64_t)s * a2;
  f.mid += (int64_t)s * a1;
  f.top += (uint32_t)s * (uint32_t)a0;
}
// the residues (u, v) modulo m_I of a complex element
template <int I>
__device__ __forceinline__ void frac_add_uv(Frac& re, Frac& im, int u, int v) {
  frac_add(re, u + v, Mod<I>::re0, Mod<I>::re1, Mod<I>::re2);
  frac_add(im, u - v, Mod<I>::im0, Mod<I>::im1, Mod<I>::im2);
}

// the signed fraction f in [-1/2, 1/2) times P 2^k as a double (one rounding, to nearest).
// The fraction carries an error of 2^-84: what is below 2^-82 is zero.
__device__ __forceinline__ double frac_value(const Frac& f, int k) {
  uint64_t h = ((uint64_t)f.top << 32) + (uint64_t)f.mid + (uint64_t)(f.lo >> 32);
  uint32_t l = (uint32_t)f.lo;
  const bool neg = (int64_t)h < 0;
  if (neg) {
    l = ~l + 1u;
    h = ~h + (l == 0u ? 1ull : 0ull);
  }
  if (h == 0 && l < (1u << 14)) return 0.0;
  // normalise the 96-bit magnitude into 64 bits
  int z;
  uint64_t t;
  if (h) {
    z = __clzll((long long)h);
    t = z ? (h << z) | ((uint64_t)l << 32 >> (64 - z)) : h;
  } else {
    z = 64 + __clz((int)l);
    t = (uint64_t)l << (z - 32);
  }
  // t P_TOP / 2^64 without the product of the low words (2^-62): in [2^62 - 1, 2^64)
  const uint32_t th = (uint32_t)(t >> 32), tl = (uint32_t)t;
  constexpr uint32_t ph = (uint32_t)(P_TOP >> 32), pl = (uint32_t)P_TOP;
  uint64_t q = (uint64_t)th * ph + __umulhi(th, pl) + __umulhi(tl, ph);
  const int n = (int)(~q >> 63);                  // 1 when the top bit is clear
  q <<= n;
  uint64_t man = (q >> 11) + ((q >> 10) & 1u);    // 53 bits, rounded to nearest (a tie upwards)
  // value = q 2^(-64 - n - z + 64 + p_exp + k): t is the fraction times 2^(64 + z), q = t p_top / 2^64
  int e = 1023 + 63 - n - z + P_EXP + k;        // biased exponent of the leading bit of man at 2^52
  if (man >> 53) {
    man >>= 1;
    ++e;
  }
  const uint64_t sgn = neg ? 0x8000000000000000ull : 0ull;
  if (e >= 1 && e <= 2046)
    return __longlong_as_double((long long)(sgn | ((uint64_t)e << 52) | (man & 0xfffffffffffffull)));
  // beyond the normal numbers
  const double x = __longlong_as_double((long long)(sgn | (1023ull << 52) | (man & 0xfffffffffffffull)));
  return scalbn(x, e - 1023);
}

// Residues are kept in blocks of 32 rows x 8 columns (512 bytes): a warp, whose lanes
// hold 32 rows of the accumulator, writes whole blocks.  Index of (plane b, row, column).
__host__ __device__ __forceinline__ size_t res_plane(int rows, int ldR) { return (size_t)((rows + 31) / 32) * 32 * ldR; }
__device__ __forceinline__ size_t res_index(int rows, int ldR, int b, int row, int col) {
  return b * res_plane(rows, ldR) + ((size_t)(row >> 5) * (ldR >> 3) + (col >> 3)) * 256 + (row & 31) * 8 + (col & 7);
}

// Fractions of the real and imaginary parts of four elements: r points at eight columns of one row,
// the lane takes the even ones (sh = EVEN: sign-extended low halves) or the odd ones (sh = ODD)
constexpr uint32_t EVEN = 0x1110, ODD = 0x3332;   // byte selectors, the high byte replicated: residues are below 256
template <int I0, int I, int N>
__device__ __forceinline__ void add_words(const uint4 (&w)[2 * N], uint32_t sh, Frac (&re)[4], Frac (&im)[4]) {
  const uint4 u = w[2 * (I - I0)], v = w[2 * (I - I0) + 1];
  const uint32_t uw[4] = {u.x, u.y, u.z, u.w}, vw[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int c = 0; c < 4; ++c)
    frac_add_uv<I>(re[c], im[c], (int)__byte_perm(uw[c], 0, sh), (int)__byte_perm(vw[c], 0, sh));
  if constexpr (I + 1 < I0 + N) add_words<I0, I + 1, N>(w, sh, re, im);
}
// loads of N moduli first, then their sums: the loads of a thread are in flight together
template <int I0 = 0, int N = 7>
__device__ __forceinline__ void gather_fractions(const int16_t* __restrict__ r, size_t plane, uint32_t sh,
                                                 Frac (&re)[4], Frac (&im)[4]) {
  uint4 w[2 * N];
#pragma unroll
  for (int i = 0; i < 2 * N; ++i)    // volatile: kept together, ahead of the sums
    asm volatile("ld.global.cs.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(w[i].x), "=r"(w[i].y), "=r"(w[i].z), "=r"(w[i].w) : "l"(r + (2 * I0 + i) * plane));
  add_words<I0, I0, N>(w, sh, re, im);
  if constexpr (I0 + N < NM) gather_fractions<I0 + N, NM - N>(r, plane, sh, re, im);
}

}  // namespace mod
}  // namespace chi0
