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
// Residues are centred (|r| <= 254), exact in FP16, and a sum of 256 products is
// at most 254^2 256 < 2^24: exact in the tensor cores' FP32 accumulators, in any
// order and rounding.  The only error is the rounding to integers, about 0.08 x
// 2^-53 of |A_m| |B_n| (0.3 x 2^-53 for the same sum by FP64 fused multiply-adds
// over Gaussian rows).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace chi0 {
namespace mod {

constexpr int NM = 13;               // moduli
constexpr int NPL = 2 * NM;          // residue planes (u and v of every modulus)
constexpr int BETA_A = 57, BETA_B = 56;   // bits of the rows' norms after scaling
constexpr int NO_SCALE = -(1 << 28);      // scale exponent of a row holding an infinity or a NaN

typedef unsigned __int128 u128;

struct Tables {
  int m[NM] = {509, 505, 493, 481, 461, 457, 449, 433, 421, 409, 401, 397, 389};
  int c1[NM] = {}, c2[NM] = {};                   // 2^20, 2^40 (mod m), centred
  int i0[NM] = {}, i1[NM] = {}, i2[NM] = {};      // I, I 2^20, I 2^40 (mod m), centred
  uint32_t bias[NM] = {};                         // multiple of m above 2^30, plus (m - 1) / 2
  uint32_t mag[NM] = {};                          // ceil(2^40 / m): floor(t / m) = t mag >> 40 for t < 2^31
  // C = sum_i s_i a_i (mod 1) in units of P, s = u + v for the real part and u - v for the
  // imaginary part: a 96-bit fraction (hi, mid, lo)
  uint32_t re[NM][3] = {}, im[NM][3] = {};
  uint64_t p_top = 0;                             // P = p_top 2^p_exp, top bit set
  int p_exp = 0;
};

constexpr int cpow_mod(int b, int e, int m) {
  int64_t r = 1, x = ((b % m) + m) % m;
  for (; e > 0; --e) r = r * x % m;
  return (int)r;
}
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
    const int p20 = (1 << 20) % m, p40 = (int)((int64_t)p20 * p20 % m);
    t.c1[i] = centred(p20, m);
    t.c2[i] = centred(p40, m);
    t.i0[i] = centred(I, m);
    t.i1[i] = centred(I * p20 % m, m);
    t.i2[i] = centred(I * p40 % m, m);
    t.bias[i] = (uint32_t)(((1 << 30) / m + 1) * m + (m - 1) / 2);
    t.mag[i] = (uint32_t)(((uint64_t)1 << 40) / (unsigned)m + 1);
    int q = 1;                                    // P / m (mod m)
    for (int j = 0; j < NM; ++j)
      if (j != i) q = q * (t.m[j] % m) % m;
    const int w = cinv_mod(q, m), half = cinv_mod(2, m);
    const int ar = w * half % m, ai = ar * cinv_mod(I, m) % m;
    for (int c = 0; c < 2; ++c) {
      const u128 f = (((u128)(unsigned)(c ? ai : ar) << 97) / (unsigned)m + 1) >> 1;   // rounded, below 2^96
      uint32_t* o = c ? t.im[i] : t.re[i];
      o[0] = (uint32_t)(f >> 64);
      o[1] = (uint32_t)(f >> 32);
      o[2] = (uint32_t)f;
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
  static constexpr int m = T.m[I], c1 = T.c1[I], c2 = T.c2[I], i0 = T.i0[I], i1 = T.i1[I], i2 = T.i2[I];
  static constexpr int bias = (int)T.bias[I];
  static constexpr uint32_t mag = T.mag[I];
  static constexpr uint32_t re0 = T.re[I][0], re1 = T.re[I][1], re2 = T.re[I][2];
  static constexpr uint32_t im0 = T.im[I][0], im1 = T.im[I][1], im2 = T.im[I][2];
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

// scale exponent s with norm 2^s <= 2^beta, from norm^2 = n2 4^e (n2 > 0 an FP64 sum)
__device__ __forceinline__ int scale_exp(double n2, int e, int beta) {
  if (!(n2 > 0.0)) return 0;                      // a row of zeros
  int k;
  frexp(n2 * (1.0 + 1e-9), &k);                   // n2 < 2^k
  return beta - e - ((k + 1) >> 1);               // norm < 2^(e + k / 2)
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

// limbs of a signed integer below 2^58: a = l0 + l1 2^20 + l2 2^40
struct Limbs {
  int l0, l1, l2;
};
__device__ __forceinline__ Limbs limbs(int64_t a) {
  return Limbs{(int)(a & 0xfffff), (int)((a >> 20) & 0xfffff), (int)(a >> 40)};
}

// t >= 0 (below 2^31), returns the FP16 bits of 1536 + (t mod m) - (m - 1) / 2
template <int I>
__device__ __forceinline__ uint32_t residue_bits(uint32_t t) {
  const uint32_t q = __umulhi(t, Mod<I>::mag) >> 8;
  return t - q * (uint32_t)Mod<I>::m + (0x6600u - (uint32_t)((Mod<I>::m - 1) / 2));
}
// two biased residues to two FP16 numbers
__device__ __forceinline__ uint32_t unbias(uint32_t lo, uint32_t hi) {
  uint32_t r;
  asm("sub.f16x2 %0, %1, %2;" : "=r"(r) : "r"(lo | (hi << 16)), "r"(0x66006600u));
  return r;
}

// residues (u, v) modulo m_I of two complex integers (k and k + 1): a packed FP16
// pair of each
template <int I>
__device__ __forceinline__ void residues2(const Limbs& xr, const Limbs& xi, const Limbs& yr, const Limbs& yi,
                                          uint32_t& u, uint32_t& v) {
  const int ax = xr.l0 + Mod<I>::c1 * xr.l1 + Mod<I>::c2 * xr.l2 + Mod<I>::bias;
  const int bx = Mod<I>::i0 * xi.l0 + Mod<I>::i1 * xi.l1 + Mod<I>::i2 * xi.l2;
  const int ay = yr.l0 + Mod<I>::c1 * yr.l1 + Mod<I>::c2 * yr.l2 + Mod<I>::bias;
  const int by = Mod<I>::i0 * yi.l0 + Mod<I>::i1 * yi.l1 + Mod<I>::i2 * yi.l2;
  u = unbias(residue_bits<I>((uint32_t)(ax + bx)), residue_bits<I>((uint32_t)(ay + by)));
  v = unbias(residue_bits<I>((uint32_t)(ax - bx)), residue_bits<I>((uint32_t)(ay - by)));
}

// all residues of two complex integers into planes of `plane` words each: u of modulus i at
// plane 2 i, v at 2 i + 1 (conj: of the conjugates, u and v exchanged)
template <int I = 0>
__device__ __forceinline__ void store_residues(const Limbs& xr, const Limbs& xi, const Limbs& yr, const Limbs& yi,
                                               bool conj, uint32_t* __restrict__ dst, size_t plane) {
  uint32_t u, v;
  residues2<I>(xr, xi, yr, yi, u, v);
  dst[(2 * I) * plane] = conj ? v : u;
  dst[(2 * I + 1) * plane] = conj ? u : v;
  if constexpr (I + 1 < NM) store_residues<I + 1>(xr, xi, yr, yi, conj, dst, plane);
}

// ---------------------------------------------------------------------------
// reconstruction
// ---------------------------------------------------------------------------
// f += s a with a 96-bit fraction a (mod 1); hi holds the top 64 bits, lo a carry-save sum of
// the products with the low word
struct Frac {
  uint64_t hi;
  int64_t lo;
};
__device__ __forceinline__ void frac_add(Frac& f, int s, uint32_t a0, uint32_t a1, uint32_t a2) {
  f.lo += (int64_t)s * (int64_t)a2;
  f.hi += (uint64_t)((int64_t)s * (int64_t)a1) + ((uint64_t)((uint32_t)s * a0) << 32);
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
  uint64_t h = f.hi + (uint64_t)(f.lo >> 32);
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
  uint64_t q = __umul64hi(t, P_TOP);            // in [2^62, 2^64)
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

}  // namespace mod
}  // namespace chi0
