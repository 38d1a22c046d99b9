// Wavefunctions on the grid and pair matrix elements of FP64 plans in fixed point on
// the integer pipe.
//
// GB300's FP64 pipe does two multiply-adds per clock and SM, so the direct FP64
// sums (kern_pairs.cu) took 10.3 ms for the 8-atom workload's 3840 pairs.  Here
// every number is a signed integer in two limbs and a multiply-add is four 32 x
// 32 + 64-bit integer multiply-adds, thirty times the rate:
//
//   inputs    55 bits (limbs 28 + 28) relative to the largest one: of the plane's
//             products conj(psi_v) psi_c, which are formed in FP64, or of a column's
//             coefficients.  Each further transform rescales to the plane's largest
//             element (block floating point, one exponent per plane)
//   twiddles  55 bits; the sums are exact, one rounding per output
//
// The unit follows the products and not the bands, so bands that overlap little lose
// nothing: what a plane holds is rounded to 2^-56 of its own largest product, against
// 2^-53 of every partial sum in FP64.  Against quad precision (relative Frobenius,
// grids of 21 to 48 points): pairs 1.0-1.2e-16, FP64 sums 4.7-6.6e-16; wavefunctions
// 0.9e-16, FP64 sums 5.8-7.0e-16.
//
// A line of n points is transformed at the wanted frequencies only, with the
// symmetries of the twiddles folded out first: with h = n / 2 and a_i = x_i +
// x_{i+h}, b_i = x_i - x_{i+h},
//   even k:  X(+-k) = E +- i O,  E = sum_i (a_i + a_{h-i}) cos,  O = sum_i (a_i - a_{h-i}) sin
//   odd k:   the same with b_i - b_{h-i} and b_i + b_{h-i},
// about n / 2 real multiplications per component and pair +-k where the direct sum
// takes 4 n.  (Odd n: only the mirror i -> n - i.)  The folded values replace the
// line in place: E(i) at i, O(i) at h - i (even k), E at h + i, O at n - i (odd k).
#include <math.h>

#include <algorithm>
#include <vector>

#include "cplx.cuh"
#include "internal.h"
#include "modgemm.cuh"

namespace chi0 {
namespace {

constexpr int WBITS = 55, WL = 28;    // transform inputs and twiddles: bits and limb width
constexpr int FX_MAX_N = 128;         // the 64-bit sums hold n / 4 + 1 products of 2^57
constexpr int FX_MAX_W = 64;          // wavefunction sphere: 64 coefficients per column (4 products of 2^54 each)

// ---- doubles to fixed point ----
// biased exponent of a set's largest magnitude word; its integers are below 2^55 in units of
// 2^fx_unit(exponent)
__device__ __forceinline__ int fx_exp(uint32_t w) { return max((int)(w >> 20), 1); }
__device__ __forceinline__ int fx_unit(int emax) { return emax - 1023 - (WBITS - 1); }
// x in that unit, rounded (subnormal numbers included)
__device__ __forceinline__ int64_t fx_int(double x, int emax) {
  const int64_t b = __double_as_longlong(x);
  const int e = (int)((b >> 52) & 0x7ff);
  const uint64_t man = ((uint64_t)b & 0xfffffffffffffull) | (e ? 0x10000000000000ull : 0ull);
  const int64_t q = (int64_t)(((man << (WBITS - 52)) >> min(emax - max(e, 1), 63)) + 1) >> 1;
  return b < 0 ? -q : q;
}

// ---- line transforms ----
// x 2^-s, rounded to nearest (s may be negative)
__device__ __forceinline__ int64_t shift_round(int64_t x, int s) {
  if (s <= 0) return x << -s;
  return s > 62 ? 0 : (x + (1ll << (s - 1))) >> s;
}
__device__ __forceinline__ uint32_t abs_word(int64_t x) { return (uint32_t)((x ^ (x >> 63)) >> 32); }
// bits of the magnitudes whose largest high word is m
__device__ __forceinline__ int word_bits(uint32_t m) { return 64 - __clz((int)m); }

__device__ __forceinline__ int4 limbs_w(int64_t re, int64_t im) {
  const int r0 = ((int)re << (32 - WL)) >> (32 - WL), i0 = ((int)im << (32 - WL)) >> (32 - WL);
  return make_int4((int)((re - r0) >> WL), r0, (int)((im - i0) >> WL), i0);
}

// y 2^k as a double, rounded to nearest
__device__ __forceinline__ double to_double(int64_t y, int k) {
  if (y == 0) return 0.0;
  const uint64_t a = y < 0 ? 0ull - (uint64_t)y : (uint64_t)y;
  const int z = __clzll((long long)a);
  const uint64_t t = a << z;                              // top bit set
  uint64_t man = (t >> 11) + ((t >> 10) & 1u);
  int e = 1023 + 63 - z + k;
  if (man >> 53) {
    man >>= 1;
    ++e;
  }
  const uint64_t sgn = y < 0 ? 0x8000000000000000ull : 0ull;
  if (e >= 1 && e <= 2046) return __longlong_as_double((long long)(sgn | ((uint64_t)e << 52) | (man & 0xfffffffffffffull)));
  return scalbn(__longlong_as_double((long long)(sgn | (1023ull << 52) | (man & 0xfffffffffffffull))), e - 1023);
}

// units of one line's fold: i = 0 .. fold_units(n) - 1, each owns the slots it reads and writes
__host__ __device__ __forceinline__ int fold_units(int n) { return n & 1 ? (n + 1) / 2 : n / 4 + 1; }

// elements of a line as integers below 2^55: integers x 2^-s, doubles of a set with exponent s
__device__ __forceinline__ longlong2 line_int(longlong2 v, int s) {
  return make_longlong2(shift_round(v.x, s), shift_round(v.y, s));
}
__device__ __forceinline__ longlong2 line_int(double2 v, int s) { return make_longlong2(fx_int(v.x, s), fx_int(v.y, s)); }

template <class T>
__device__ __forceinline__ void fold_line(T* __restrict__ r, int n, int i, int s) {
  int4* w = reinterpret_cast<int4*>(r);
  auto ld = [&](int k) { return line_int(r[k], s); };
  if (n & 1) {
    const longlong2 x = ld(i);
    if (i == 0) {
      w[0] = limbs_w(x.x, x.y);
      return;
    }
    const longlong2 y = ld(n - i);
    w[i] = limbs_w(x.x + y.x, x.y + y.y);
    w[n - i] = limbs_w(x.x - y.x, x.y - y.y);
    return;
  }
  const int h = n >> 1;
  const longlong2 x1 = ld(i), x3 = ld(h + i);
  if (i == 0 || 2 * i == h) {      // E even at i, E odd (i = 0) or O odd (i = h / 2) at h + i
    w[i] = limbs_w(x1.x + x3.x, x1.y + x3.y);
    w[h + i] = limbs_w(x1.x - x3.x, x1.y - x3.y);
    return;
  }
  const longlong2 x2 = ld(h - i), x4 = ld(n - i);
  const longlong2 a = make_longlong2(x1.x + x3.x, x1.y + x3.y), c = make_longlong2(x2.x + x4.x, x2.y + x4.y);
  const longlong2 b = make_longlong2(x1.x - x3.x, x1.y - x3.y), d = make_longlong2(x2.x - x4.x, x2.y - x4.y);
  w[i] = limbs_w(a.x + c.x, a.y + c.y);
  w[h - i] = limbs_w(a.x - c.x, a.y - c.y);
  w[h + i] = limbs_w(b.x - d.x, b.y - d.y);
  w[n - i] = limbs_w(b.x + d.x, b.y + d.y);
}

struct Acc {
  int64_t hh = 0, cr = 0, ll = 0;
  __device__ __forceinline__ void add(int x1, int x0, int c1, int c0) {
    hh += (int64_t)x1 * c1;
    cr += (int64_t)x1 * c0;
    cr += (int64_t)x0 * c1;
    ll += (int64_t)x0 * c0;
  }
  // the sum over 2^55 (the twiddles' unit), rounded
  __device__ __forceinline__ int64_t value() const {
    return 2 * hh + ((cr + (ll >> WL) + (1ll << (WBITS - WL - 1))) >> (WBITS - WL));
  }
};

// X(+k) and X(-k) of a folded line at item `it` of the axis
__device__ __forceinline__ void line_pair(const int4* __restrict__ w, const FxAxis& ax, int it, int4 item,
                                          longlong2& pos, longlong2& neg) {
  const int n = ax.n, h = n >> 1;
  const bool odd_k = item.x != 0;     // never for odd n
  int ce, cb, oe, ob;                 // cosine terms w[cb + i], i < ce; sine terms w[ob - i], 1 <= i < oe
  if (n & 1) {
    ce = oe = (n + 1) / 2;
    cb = 0;
    ob = n;
  } else if (!odd_k) {
    ce = h / 2 + 1;
    oe = (h + 1) / 2;
    cb = 0;
    ob = h;
  } else {
    ce = (h + 1) / 2;
    oe = h / 2 + 1;
    cb = h;
    ob = n;
  }
  const int4* __restrict__ t = ax.coef + it * ax.units;     // (cos1, cos0, sin1, sin0)
  Acc er, ei, sr, si;
  for (int i = 0; i < ce; ++i) {
    const int4 x = w[cb + i], c = t[i];
    er.add(x.x, x.y, c.x, c.y);
    ei.add(x.z, x.w, c.x, c.y);
  }
  for (int i = 1; i < oe; ++i) {
    const int4 x = w[ob - i], c = t[i];
    sr.add(x.x, x.y, c.z, c.w);
    si.add(x.z, x.w, c.z, c.w);
  }
  const int64_t Er = er.value(), Ei = ei.value(), Or = sr.value(), Oi = si.value();
  pos = make_longlong2(Er - Oi, Ei + Or);
  neg = make_longlong2(Er + Oi, Ei - Or);
}

// largest magnitude word of the block: each thread gives its own, every thread gets the result
__device__ __forceinline__ uint32_t block_max(uint32_t m, uint32_t* __restrict__ slot) {
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) atomicMax(slot, m);
  __syncthreads();
  return *slot;
}

// Stages 1 and 2 of one plane i1: D[pair][i1][k2][k3] as 64-bit integers and their
// exponents ex[pair][i1] = (unit, top): value = D 2^unit, |value| < 2^top.  A CTA
// takes one valence band and a run of conduction bands.  The products run on the
// FP64 pipe (four operations per grid point), beside the integer multiplies of other
// CTAs' transforms (eight per folded point and frequency pair).
__global__ void k_fx_planes(const double2* __restrict__ psi_v, const int32_t* __restrict__ v_idx, int v_base,
                            const double2* __restrict__ psi_c, const int32_t* __restrict__ c_idx, int c_base, int nc,
                            int cpc, int n1, int n2, int n3, int nk2, int nk3, const __grid_constant__ FxAxis a3,
                            const __grid_constant__ FxAxis a2, longlong2* __restrict__ D, int2* __restrict__ ex) {
  extern __shared__ __align__(16) unsigned char smem_fx[];
  __shared__ uint32_t slot[3];
  const int ld3 = n3 | 1, ld2 = n2 | 1;
  double2* A = reinterpret_cast<double2*>(smem_fx);        // [n2][ld3]
  longlong2* X = reinterpret_cast<longlong2*>(A + (size_t)n2 * ld3);   // [nk3][ld2]
  const int i1 = blockIdx.x, jv = blockIdx.y, nt = blockDim.x, tid = threadIdx.x;
  const int plane = n2 * n3;
  const int64_t nr = (int64_t)n1 * plane, box = (int64_t)nk2 * nk3;
  const double2* v0 = psi_v + (v_idx ? v_idx[v_base + jv] : v_base + jv) * nr + (int64_t)i1 * plane;
  const int jc1 = min(nc, (int)(blockIdx.z + 1) * cpc);
  for (int jc = blockIdx.z * cpc; jc < jc1; ++jc) {
    const double2* c0 = psi_c + (c_idx ? c_idx[c_base + jc] : c_base + jc) * nr + (int64_t)i1 * plane;
    const int64_t pair = (int64_t)jv * nc + jc;
    __syncthreads();                                       // the previous pair's readers are done
    if (tid < 3) slot[tid] = 0;
    __syncthreads();
    uint32_t m = 0;
    for (int e = tid; e < plane; e += nt) {
      const int i2 = e / n3, i3 = e - i2 * n3;
      const double2 p = cconjmul(v0[e], c0[e]);
      A[i2 * ld3 + i3] = p;
      m = max(m, max(mod::mag_word(p.x), mod::mag_word(p.y)));
    }
    m = block_max(m, slot);                                // its barrier also orders A
    if (m >= 0x7ff00000u) {                                // an infinity or a NaN: the pair's elements are NaN
      if (tid == 0) ex[pair * n1 + i1] = make_int2(mod::NO_SCALE, 0);
      continue;
    }
    const int s0 = fx_exp(m);
    const int u3 = fold_units(n3);
    for (int e = tid; e < n2 * u3; e += nt) {
      const int i2 = e % n2, i = e / n2;
      fold_line(A + i2 * ld3, n3, i, s0);
    }
    __syncthreads();
    m = 0;
    for (int e = tid; e < n2 * a3.items; e += nt) {        // along i3
      const int i2 = e % n2, it = e / n2;
      const int4 item = a3.item[it];
      longlong2 p, q;
      line_pair(reinterpret_cast<const int4*>(A + i2 * ld3), a3, it, item, p, q);
      if (item.y >= 0) {
        X[item.y * ld2 + i2] = p;
        m = max(m, max(abs_word(p.x), abs_word(p.y)));
      }
      if (item.z >= 0) {
        X[item.z * ld2 + i2] = q;
        m = max(m, max(abs_word(q.x), abs_word(q.y)));
      }
    }
    const int s1 = word_bits(block_max(m, slot + 1)) - WBITS;
    const int u2 = fold_units(n2);
    for (int e = tid; e < nk3 * u2; e += nt) {
      const int k3 = e % nk3, i = e / nk3;
      fold_line(X + k3 * ld2, n2, i, s1);
    }
    __syncthreads();
    m = 0;
    longlong2* d = D + (pair * n1 + i1) * box;
    for (int e = tid; e < nk3 * a2.items; e += nt) {       // along i2
      const int k3 = e % nk3, it = e / nk3;
      const int4 item = a2.item[it];
      longlong2 p, q;
      line_pair(reinterpret_cast<const int4*>(X + k3 * ld2), a2, it, item, p, q);
      if (item.y >= 0) {
        d[(int64_t)item.y * nk3 + k3] = p;
        m = max(m, max(abs_word(p.x), abs_word(p.y)));
      }
      if (item.z >= 0) {
        d[(int64_t)item.z * nk3 + k3] = q;
        m = max(m, max(abs_word(q.x), abs_word(q.y)));
      }
    }
    m = block_max(m, slot + 2);
    if (tid == 0) {
      const int unit = fx_unit(s0) + s1;
      ex[pair * n1 + i1] = make_int2(unit, unit + word_bits(m));
    }
  }
}

// Stage 3: M[row][j] = (1/N_r) sum_i1 D(i1, k2_j, k3_j) e^{2 pi i k1_j i1 / n1} for a chunk of the
// (k2, k3) columns of one pair; colmap[column][k1 - k1min] = j, or -1 off the sphere
__global__ void __launch_bounds__(256) k_fx_gather(const longlong2* __restrict__ D, const int2* __restrict__ ex, int nc,
                                                   int64_t row0, int64_t ldv, int n1, int64_t box, int nG, int ncol,
                                                   int chunk, int nk1, const int* __restrict__ col_off,
                                                   const int* __restrict__ colmap, const __grid_constant__ FxAxis a1,
                                                   double scale, double2* __restrict__ M) {
  extern __shared__ __align__(16) unsigned char smem_fx[];
  __shared__ int unit[FX_MAX_N], s_top, s_bad;
  const int ld1 = n1 | 1, tid = threadIdx.x, nt = blockDim.x;
  longlong2* A = reinterpret_cast<longlong2*>(smem_fx);    // [chunk][ld1]
  const int pl = blockIdx.x, jv = pl / nc, jc = pl - jv * nc;
  const int c0 = blockIdx.y * chunk, cn = min(chunk, ncol - c0);
  if (tid == 0) {
    s_top = -(1 << 30);
    s_bad = 0;
  }
  __syncthreads();
  for (int i = tid; i < n1; i += nt) {
    const int2 e = ex[(int64_t)pl * n1 + i];
    unit[i] = e.x;
    atomicMax(&s_top, e.y);
    if (e.x == mod::NO_SCALE) s_bad = 1;
  }
  __syncthreads();
  const int base = s_top - WBITS;                          // common unit of the planes: 2^base
  const bool bad = s_bad != 0;
  for (int e = tid; e < cn * n1; e += nt) {
    const int c = e % cn, i = e / cn;
    const longlong2 v = D[((int64_t)pl * n1 + i) * box + col_off[c0 + c]];
    const int s = base - unit[i];
    A[c * ld1 + i] = make_longlong2(shift_round(v.x, s), shift_round(v.y, s));
  }
  __syncthreads();
  const int u1 = fold_units(n1);
  for (int e = tid; e < cn * u1; e += nt) {
    const int c = e % cn, i = e / cn;
    fold_line(A + c * ld1, n1, i, 0);
  }
  __syncthreads();
  double2* out = M + (row0 + (int64_t)jv * ldv + jc) * nG;
  auto put = [&](int j, longlong2 y) {
    out[j] = bad ? make_double2(nan(""), nan(""))
                 : make_double2(to_double(y.x, base) * scale, to_double(y.y, base) * scale);
  };
  for (int e = tid; e < cn * a1.items; e += nt) {
    const int c = e % cn, it = e / cn;
    const int4 item = a1.item[it];
    const int* cm = colmap + (int64_t)(c0 + c) * nk1;
    const int jp = item.y >= 0 ? cm[item.y] : -1, jn = item.z >= 0 ? cm[item.z] : -1;
    if (jp < 0 && jn < 0) continue;
    longlong2 p, q;
    line_pair(reinterpret_cast<const int4*>(A + c * ld1), a1, it, item, p, q);
    if (jp >= 0) put(jp, p);
    if (jn >= 0) put(jn, q);
  }
}

// ---- wavefunctions ----
// Synthesis of a line of n points from coefficients c(g), |g| <= G, with the same
// symmetries: P = c(g) + c(-g), M = c(g) - c(-g), sums over even and odd g apart,
//   X(i) = (Ee + Eo) + i (Oe + Oo),  X(n - i) = (Ee + Eo) - i (Oe + Oo),
//   X(i + h) = (Ee - Eo) + i (Oe - Oo),  X(h - i) = (Ee - Eo) - i (Oe - Oo),  h = n / 2,
// E = sum P cos, O = sum M sin, for i = 0 .. n / 4 (odd n: i = 0 .. (n - 1) / 2, the
// first row only).  The line is kept as slots G + g, folded in place (P at +g, M at -g).
// sp, sm: shifts of the slots at +g and -g.
__device__ __forceinline__ void fold_synth(longlong2* __restrict__ r, int G, int g, int sp, int sm) {
  int4* w = reinterpret_cast<int4*>(r);
  const longlong2 p = line_int(r[G + g], sp), m = line_int(r[G - g], sm);
  const int64_t px = p.x, py = p.y, mx = m.x, my = m.y;
  if (g == 0) {
    w[G] = limbs_w(px, py);
    return;
  }
  w[G + g] = limbs_w(px + mx, py + my);
  w[G - g] = limbs_w(px - mx, py - my);
}

// calls put(index, value) for the outputs of unit i
template <class Put>
__device__ __forceinline__ void synth_unit(const int4* __restrict__ w, const FxAxis& ax, int i, Put put) {
  const int n = ax.n, h = n >> 1, G = ax.items;
  const int4* __restrict__ t = ax.coef + i;            // [g][units]
  const bool even = !(n & 1);
  int64_t E[2][2] = {}, O[2][2] = {};                  // [parity of g][re, im]
#pragma unroll
  for (int par = 0; par < 2; ++par) {
    if (par && !even) break;
    Acc er, ei, sr, si;
    for (int g = par; g <= G; g += even ? 2 : 1) {
      const int4 p = w[G + g], c = t[g * ax.units];
      er.add(p.x, p.y, c.x, c.y);
      ei.add(p.z, p.w, c.x, c.y);
      if (g) {
        const int4 m = w[G - g];
        sr.add(m.x, m.y, c.z, c.w);
        si.add(m.z, m.w, c.z, c.w);
      }
    }
    E[par][0] = er.value();
    E[par][1] = ei.value();
    O[par][0] = sr.value();
    O[par][1] = si.value();
  }
  const int64_t er = E[0][0] + E[1][0], ei = E[0][1] + E[1][1], orr = O[0][0] + O[1][0], oi = O[0][1] + O[1][1];
  put(i, make_longlong2(er - oi, ei + orr));
  if (i) put(n - i, make_longlong2(er + oi, ei - orr));
  if (even) {
    const int64_t fr = E[0][0] - E[1][0], fi = E[0][1] - E[1][1], pr = O[0][0] - O[1][0], pi = O[0][1] - O[1][1];
    if (2 * i != h || i == 0) put(i + h, make_longlong2(fr - pi, fi + pr));
    if (i && 2 * i != h) put(h - i, make_longlong2(fr + pi, fi - pr));
  }
}

// q[band][k] = limbs of the coefficients in column order, each column in the unit of its own largest one:
// col_unit[band][column] (BAD_UNIT: an infinity or a NaN).  Eight lanes per column.
constexpr int BAD_UNIT = 1 << 20;
__global__ void __launch_bounds__(256) k_fx_cols(const double2* __restrict__ coeff, int npw, int ncols,
                                                 const int* __restrict__ col_start, const int* __restrict__ col_pw,
                                                 int4* __restrict__ q, int* __restrict__ col_unit) {
  const int c = blockIdx.x * 32 + (threadIdx.x >> 3), l = threadIdx.x & 7;
  const int64_t b = blockIdx.y;
  const double2* cb = coeff + b * npw;
  const int k0 = c < ncols ? col_start[c] : 0, k1 = c < ncols ? col_start[c + 1] : 0;
  uint32_t big = 0;
  for (int k = k0 + l; k < k1; k += 8) {
    const double2 v = cb[col_pw[k]];
    big = max(big, max(mod::mag_word(v.x), mod::mag_word(v.y)));
  }
  for (int o = 4; o; o >>= 1) big = max(big, __shfl_xor_sync(0xffffffffu, big, o));
  const int emax = fx_exp(big);
  for (int k = k0 + l; k < k1; k += 8) {
    const double2 v = cb[col_pw[k]];
    q[b * npw + k] = limbs_w(fx_int(v.x, emax), fx_int(v.y, emax));
  }
  if (l == 0 && c < ncols) col_unit[b * ncols + c] = big >= 0x7ff00000u ? BAD_UNIT : fx_unit(emax);
}

// psi[band][i1] for one plane and band: along g1 for every (g2, g3) column of the sphere (direct sums
// over its few coefficients), along g2 for every g3, along g3 for every i2.  The columns' sums join at the
// plane's exponent.
constexpr int TOP0 = 4096;                                 // exponents are compared as positive words, 0: none
constexpr int NO_UNIT = -(1 << 20);                        // of zeros: they stay zeros in any other unit
__global__ void k_fx_wfn(const int4* __restrict__ q, const int* __restrict__ col_unit, int npw, int n1, int n2, int n3,
                         int nw1, int w2min, int w3min, int nw2, int nw3, const int* __restrict__ col_start,
                         const int* __restrict__ col_g1, int w1min,
                         const int4* __restrict__ tw1, const __grid_constant__ FxAxis a2, const __grid_constant__ FxAxis a3,
                         double2* __restrict__ psi) {
  extern __shared__ __align__(16) unsigned char smem_fx[];
  __shared__ uint32_t slot[2];
  __shared__ int4 tws[FX_MAX_W];
  const int G2 = a2.items, G3 = a3.items, lda = 2 * G2 + 1, ldb = 2 * G3 + 1;   // odd
  longlong2* A = reinterpret_cast<longlong2*>(smem_fx);    // [2 G3 + 1][lda]: slot of g3, slot of g2
  longlong2* B = A + (size_t)(2 * G3 + 1) * lda;           // [n2][ldb]
  int* U = reinterpret_cast<int*>(B);                      // [2 G3 + 1][lda] units of A's values, before B is needed
  const int i1 = blockIdx.x, tid = threadIdx.x, nt = blockDim.x;
  const int64_t b = blockIdx.y;
  double2* out = psi + (b * n1 + i1) * (int64_t)n2 * n3;
  if (tid < 2) slot[tid] = 0;
  for (int g = tid; g < nw1; g += nt) {
    int k = (int)((int64_t)(w1min + g) * i1 % n1);
    tws[g] = tw1[k < 0 ? k + n1 : k];
  }
  for (int e = tid; e < (2 * G3 + 1) * lda; e += nt) {
    A[e] = make_longlong2(0, 0);
    U[e] = NO_UNIT;
  }
  __syncthreads();
  const int4* qb = q + b * npw;
  const int* ub = col_unit + b * (nw2 * nw3);
  uint32_t m = 0;
  for (int c = tid; c < nw2 * nw3; c += nt) {
    const int r = c / nw3, g3 = w3min + c - r * nw3, g2 = w2min + r;
    const int k0 = col_start[c], k1 = col_start[c + 1];
    const int unit = ub[c];
    Acc re, im;
    for (int k = k0; k < k1; ++k) {
      const int4 x = qb[k], t = tws[col_g1[k]];            // t = (cos, sin) in two limbs each
      re.add(x.x, x.y, t.x, t.y);
      re.add(-x.z, -x.w, t.z, t.w);
      im.add(x.z, x.w, t.x, t.y);
      im.add(x.x, x.y, t.z, t.w);
    }
    const longlong2 v = make_longlong2(re.value(), im.value());
    if (unit == BAD_UNIT) m = 0xffffffffu;
    const int at = (G3 + g3) * lda + G2 + g2;
    if (unit != BAD_UNIT && (v.x | v.y)) {
      A[at] = v;
      U[at] = unit;
      m = max(m, (uint32_t)(TOP0 + unit + word_bits(max(abs_word(v.x), abs_word(v.y)))));
    }
  }
  m = block_max(m, slot);
  if (m == 0xffffffffu) {
    for (int e = tid; e < n2 * n3; e += nt) out[e] = make_double2(nan(""), nan(""));
    return;
  }
  const int base = (int)m - TOP0 - WBITS;
  for (int e = tid; e < (2 * G3 + 1) * (G2 + 1); e += nt) {
    const int c = e % (2 * G3 + 1), g = e / (2 * G3 + 1), *u = U + c * lda + G2;
    fold_synth(A + c * lda, G2, g, base - u[g], base - u[-g]);
  }
  __syncthreads();
  m = 0;
  for (int e = tid; e < (2 * G3 + 1) * a2.units; e += nt) {    // along g2
    const int c = e % (2 * G3 + 1), i = e / (2 * G3 + 1);
    synth_unit(reinterpret_cast<const int4*>(A + c * lda), a2, i, [&](int i2, longlong2 v) {
      B[i2 * ldb + c] = v;
      m = max(m, max(abs_word(v.x), abs_word(v.y)));
    });
  }
  const int sb = word_bits(block_max(m, slot + 1)) - WBITS;
  for (int e = tid; e < n2 * (G3 + 1); e += nt) {
    const int i2 = e % n2, g = e / n2;
    fold_synth(B + i2 * ldb, G3, g, sb, sb);
  }
  __syncthreads();
  const int unit = base + sb;
  for (int e = tid; e < n2 * a3.units; e += nt) {              // along g3
    const int i = e % a3.units, i2 = e / a3.units;
    synth_unit(reinterpret_cast<const int4*>(B + i2 * ldb), a3, i, [&](int i3, longlong2 v) {
      out[i2 * n3 + i3] = make_double2(to_double(v.x, unit), to_double(v.y, unit));
    });
  }
}

size_t wfn_smem(const chi0_plan_s* p, const WfnSphere& w) {
  const size_t a = (size_t)(2 * w.fx[1].items + 1) * (2 * w.fx[0].items + 1), b = (size_t)p->n2 * (2 * w.fx[1].items + 1);
  return a * 16 + std::max(b * 16, a * 4);
}

size_t planes_smem(const chi0_plan_s* p, const SphereQ& s) {
  return ((size_t)p->n2 * (p->n3 | 1) + (size_t)s.nk3 * (p->n2 | 1)) * 16;
}
constexpr size_t SMEM_CAP = 220 * 1024;

// (cos, sin) of 2 pi m / n, m < n, in two limbs each; evaluated on the first octant only (long double
// is software on the Arm hosts)
std::vector<int4> twiddle_table(int n) {
  const long double two_pi = 2.0L * 3.14159265358979323846264338327950288L;
  std::vector<int64_t> c(n / 8 + 1), s(n / 8 + 1);
  for (int m = 0; m <= n / 8; ++m) {
    c[m] = llroundl(cosl(two_pi * m / n) * (long double)((int64_t)1 << WBITS));
    s[m] = llroundl(sinl(two_pi * m / n) * (long double)((int64_t)1 << WBITS));
  }
  std::vector<int4> t(n);
  for (int m = 0; m < n; ++m) {
    // angle 2 pi m / n = (quarter turns) + 2 pi r / (4 n): r = 4 m mod n quarters of a step
    const int quarter = 4 * m / n, r = 4 * m - quarter * n;
    int64_t co, si;
    if (r % 4 == 0 && 8 * (r / 4) <= n) {                    // r / 4 whole steps past the quarter turn
      co = c[r / 4];
      si = s[r / 4];
    } else if ((n - r) % 4 == 0 && 8 * ((n - r) / 4) <= n) { // before the next quarter turn
      co = s[(n - r) / 4];
      si = c[(n - r) / 4];
    } else {                                                 // n not a multiple of 4: no symmetric point
      co = llroundl(cosl(two_pi * r / (4.0L * n)) * (long double)((int64_t)1 << WBITS));
      si = llroundl(sinl(two_pi * r / (4.0L * n)) * (long double)((int64_t)1 << WBITS));
    }
    const int64_t re = quarter == 0 ? co : quarter == 1 ? -si : quarter == 2 ? -co : si;
    const int64_t im = quarter == 0 ? si : quarter == 1 ? co : quarter == 2 ? -si : -co;
    int l[4];
    for (int k = 0; k < 2; ++k) {
      const int64_t q = k ? im : re;
      int64_t q0 = q & (((int64_t)1 << WL) - 1);
      if (q0 >= (int64_t)1 << (WL - 1)) q0 -= (int64_t)1 << WL;
      l[2 * k] = (int)((q - q0) >> WL);
      l[2 * k + 1] = (int)q0;
    }
    t[m] = make_int4(l[0], l[1], l[2], l[3]);
  }
  return t;
}

// frequency pairs +-k of an axis (kmin .. kmin + nk - 1) and their twiddles
cudaError_t make_axis(int n, int kmin, int nk, FxAxis* a) {
  std::vector<int4> item, coef;
  const int units = fold_units(n);
  const std::vector<int4> tw = twiddle_table(n);
  for (int k = 0; k <= n / 2; ++k) {
    int pos = -1, neg = -1;
    for (int c = 0; c < nk; ++c) {
      int m = (kmin + c) % n;
      if (m < 0) m += n;
      if (m > n / 2) m -= n;
      if (m == k) pos = c;
      else if (m == -k) neg = c;
    }
    if (pos < 0 && neg < 0) continue;
    item.push_back(make_int4(n % 2 == 0 ? k & 1 : 0, pos, neg, 0));
    for (int i = 0; i < units; ++i) coef.push_back(tw[(int64_t)k * i % n]);
  }
  a->n = n;
  a->units = units;
  a->items = (int)item.size();
  int4 *di = nullptr, *dc = nullptr;
  cudaError_t e = cudaMalloc((void**)&di, item.size() * sizeof(int4));
  if (e == cudaSuccess) e = cudaMalloc((void**)&dc, coef.size() * sizeof(int4));
  if (e == cudaSuccess) e = cudaMemcpy(di, item.data(), item.size() * sizeof(int4), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(dc, coef.data(), coef.size() * sizeof(int4), cudaMemcpyHostToDevice);
  a->item = di;
  a->coef = dc;
  return e;
}

}  // namespace

static cudaError_t upload4(const int4** dst, const std::vector<int4>& v) {
  int4* d = nullptr;
  cudaError_t e = cudaMalloc((void**)&d, v.size() * sizeof(int4));
  if (e == cudaSuccess) e = cudaMemcpy(d, v.data(), v.size() * sizeof(int4), cudaMemcpyHostToDevice);
  *dst = d;
  return e;
}

// tables of the wavefunction sphere where the fixed-point synthesis fits (else w->fx_tw stays NULL and the
// direct FP64 sums run): axis g2 in fx[0], g3 in fx[1] (items = largest |g|), plane twiddles
cudaError_t fx_setup_wfn(const chi0_plan_s* p, WfnSphere* w) {
  if (w->npw <= 0 || p->n1 > FX_MAX_N || p->n2 > FX_MAX_N || p->n3 > FX_MAX_N || w->nw1 > FX_MAX_W) return cudaSuccess;
  const int n[2] = {p->n2, p->n3}, lo[2] = {w->w2min, w->w3min}, cnt[2] = {w->nw2, w->nw3};
  for (int a = 0; a < 2; ++a) {
    const int G = std::max(std::abs(lo[a]), std::abs(lo[a] + cnt[a] - 1));
    if (G > FX_MAX_W) return cudaSuccess;                   // a sphere far from the origin
    w->fx[a].n = n[a];
    w->fx[a].units = fold_units(n[a]);
    w->fx[a].items = G;
  }
  if (wfn_smem(p, *w) > SMEM_CAP) return cudaSuccess;
  std::vector<int> start((size_t)w->nw2 * w->nw3 + 1);
  cudaError_t e = cudaMemcpy(start.data(), w->col_start, start.size() * sizeof(int), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return e;
  for (size_t c = 0; c + 1 < start.size(); ++c)             // (a vector listed twice counts twice)
    if (start[c + 1] - start[c] > FX_MAX_W) return cudaSuccess;
  for (int a = 0; a < 2 && e == cudaSuccess; ++a) {
    const std::vector<int4> tw = twiddle_table(n[a]);
    std::vector<int4> t;
    for (int g = 0; g <= w->fx[a].items; ++g)
      for (int i = 0; i < w->fx[a].units; ++i) t.push_back(tw[(int64_t)g * i % n[a]]);
    e = upload4(&w->fx[a].coef, t);
  }
  if (e == cudaSuccess) e = upload4(&w->fx_tw, twiddle_table(p->n1));
  return e;
}

// scratch per band: limbs of its coefficients and units of its columns
size_t fx_wfn_ws_bytes(const chi0_plan_s* p, int64_t bands) {
  return (size_t)bands * ((size_t)p->w.npw * sizeof(int4) + (size_t)p->w.nw2 * p->w.nw3 * sizeof(int));
}

// nb bands (at most 65535: grid y)
cudaError_t launch_fx_wfn(const chi0_plan_s* p, const double2* coeff, int nb, double2* psi, void* ws, cudaStream_t s) {
  const WfnSphere& w = p->w;
  const size_t sm = wfn_smem(p, w);
  cudaError_t e = cudaFuncSetAttribute(k_fx_wfn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  const int nt = sm <= 32 * 1024 ? 128 : (sm <= 72 * 1024 ? 256 : 512), ncols = w.nw2 * w.nw3;
  int4* q = reinterpret_cast<int4*>(ws);
  int* unit = reinterpret_cast<int*>(q + (size_t)nb * w.npw);
  k_fx_cols<<<dim3((ncols + 31) / 32, nb), 256, 0, s>>>(coeff, w.npw, ncols, w.col_start, w.col_pw, q, unit);
  k_fx_wfn<<<dim3(p->n1, nb), nt, sm, s>>>(q, unit, w.npw, p->n1, p->n2, p->n3, w.nw1, w.w2min, w.w3min, w.nw2, w.nw3,
                                           w.col_start, w.col_g1, w.w1min, w.fx_tw, w.fx[0], w.fx[1], psi);
  return cudaGetLastError();
}

// whether the plan's grid and a sphere fit the kernels (else the direct FP64 sums run)
bool fx_fits(const chi0_plan_s* p, const SphereQ& s) {
  return p->n1 <= FX_MAX_N && p->n2 <= FX_MAX_N && p->n3 <= FX_MAX_N && planes_smem(p, s) <= SMEM_CAP;
}

cudaError_t fx_setup(const chi0_plan_s* p, SphereQ* s) {
  std::vector<int> map((size_t)s->ncol * s->nk1, -1), col((size_t)s->nk2 * s->nk3, -1);
  int nc = 0;
  for (int t = 0; t < s->nG; ++t) {         // columns in (k2, k3) order, as col_off lists them
    const int32_t* g = &s->g_host[3 * t];
    col[(size_t)(g[1] - s->k2min) * s->nk3 + (g[2] - s->k3min)] = 0;
  }
  for (int& c : col)
    if (c == 0) c = nc++;
  for (int t = 0; t < s->nG; ++t) {
    const int32_t* g = &s->g_host[3 * t];
    int& slot = map[(size_t)col[(size_t)(g[1] - s->k2min) * s->nk3 + (g[2] - s->k3min)] * s->nk1 + (g[0] - s->k1min)];
    if (slot >= 0) return cudaSuccess;      // a G vector listed twice: the direct sums run (fx_map stays NULL)
    slot = t;
  }
  cudaError_t e = cudaMalloc((void**)&s->fx_map, map.size() * sizeof(int));
  if (e == cudaSuccess) e = cudaMemcpy(s->fx_map, map.data(), map.size() * sizeof(int), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = make_axis(p->n1, s->k1min, s->nk1, &s->fx[0]);
  if (e == cudaSuccess) e = make_axis(p->n2, s->k2min, s->nk2, &s->fx[1]);
  if (e == cudaSuccess) e = make_axis(p->n3, s->k3min, s->nk3, &s->fx[2]);
  return e;
}

// workspace of the exponents of D for `pairs` pairs at a time
size_t fx_ws_bytes(const chi0_plan_s* p, int64_t pairs) { return (size_t)pairs * p->n1 * sizeof(int2); }

// stages 1 and 2 of the pairs of valence rows v0 .. v0 + nv and conduction columns c0 .. c0 + nc into D, and
// their exponents
cudaError_t launch_fx_planes(const chi0_plan_s* p, int iq, const double2* psi_v, const int32_t* v_idx, int v0, int nv,
                             const double2* psi_c, const int32_t* c_idx, int c0, int nc, void* D, void* ex,
                             cudaStream_t st) {
  const SphereQ& s = p->q[iq];
  const size_t sm = planes_smem(p, s);
  cudaError_t e = cudaFuncSetAttribute(k_fx_planes, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  // threads: a line and frequency pair each; conduction bands in runs that leave enough CTAs
  const int items = std::max(p->n2 * s.fx[2].items, s.nk3 * s.fx[1].items);
  const int nt = items <= 128 ? 128 : (items <= 512 || sm <= 72 * 1024 ? 256 : 512);
  int cpc = 8;
  while (cpc > 1 && (int64_t)p->n1 * nv * ((nc + cpc - 1) / cpc) < 16 * 152) cpc >>= 1;
  k_fx_planes<<<dim3(p->n1, nv, (nc + cpc - 1) / cpc), nt, sm, st>>>(psi_v, v_idx, v0, psi_c, c_idx, c0, nc, cpc, p->n1,
                                                                    p->n2, p->n3, s.nk2, s.nk3, s.fx[2], s.fx[1],
                                                                    (longlong2*)D, (int2*)ex);
  return cudaGetLastError();
}

// stage 3: M rows row0 + iv ldv + ic
cudaError_t launch_fx_gather(const chi0_plan_s* p, int iq, int nv, int nc, const void* D, const void* ex, int64_t row0,
                             int64_t ldv, double2* M, cudaStream_t st) {
  const SphereQ& s = p->q[iq];
  const int ld1 = p->n1 | 1;
  const int chunk = std::min(s.ncol, std::max(1, 40 * 1024 / (ld1 * 16)));
  k_fx_gather<<<dim3((unsigned)(nv * nc), (s.ncol + chunk - 1) / chunk), 256, (size_t)chunk * ld1 * 16, st>>>(
      (const longlong2*)D, (const int2*)ex, nc, row0, ldv, p->n1, (int64_t)s.nk2 * s.nk3, s.nG, s.ncol, chunk,
      s.nk1, s.col_off, s.fx_map, s.fx[0], 1.0 / (double)p->nr, M);
  return cudaGetLastError();
}

}  // namespace chi0
