// Adjoint of the contraction of Eq. 1.  With upstream Gamma_w = dL/dRe chi0_w
// + i dL/dIm chi0_w and chi0_w = sum_p f_p(w) M_p M_p^H:
//   grad M_p  = sum_w conj(f_p(w)) Gamma_w M_p + f_p(w) Gamma_w^H M_p
//   grad dE_p = sum_w Re( f'_p(w) conj(M_p^H Gamma_w M_p) ),
//   f'_p(w)   = -(w_p/2) [ (dE_p - w + i d)^-2 + (dE_p + w + i d)^-2 ],
// and dE_p = E_v[iv] - E_col[ic] gives grad E_v = sum_ic grad dE, grad E_col = -sum_iv grad dE.
//
// Diagonal upstream (Gamma_w = diag(g_w), g real): one fused bandwidth-bound pass
//   grad M_p(G) = sum_w 2 Re f_p(w) g_w(G) M_p(G),  grad dE_p = sum_w Re f'_p(w) sum_G g_w(G) |M_p(G)|^2.
// Dense upstream: two FP64 complex products per frequency, Y = M Gamma^T and
// Z = M conj(Gamma), as modular products on the tensor cores (modgemm.cuh) combined
// by k_bwd_mod, or as FP64 multiply-adds combined in the epilogue (k_bwd_dense).
#include <algorithm>

#include "cplx.cuh"
#include "internal.h"
#include "modgemm.cuh"

namespace chi0 {
namespace {

__device__ __forceinline__ double2 cinv_d(double a, double b) {
  const double d = a * a + b * b;
  return make_double2(a / d, -b / d);
}

// f and f' of pair p at frequency om
__device__ __forceinline__ void factors(double dE, double w, double2 om, double delta, double2* f, double2* fp) {
  const double2 a = cinv_d(dE - om.x, delta - om.y);
  const double2 b = cinv_d(dE + om.x, delta + om.y);
  *f = make_double2(0.5 * w * (a.x + b.x), 0.5 * w * (a.y + b.y));
  const double2 a2 = cmul(a, a), b2 = cmul(b, b);
  *fp = make_double2(-0.5 * w * (a2.x + b2.x), -0.5 * w * (a2.y + b2.y));
}

__device__ __forceinline__ double2 ld_d(const float2* p, int64_t i) {
  const float2 v = p[i];
  return make_double2(v.x, v.y);
}
__device__ __forceinline__ double2 ld_d(const double2* p, int64_t i) { return p[i]; }
__device__ __forceinline__ void st_c(float2* p, int64_t i, double2 v) { p[i] = make_float2((float)v.x, (float)v.y); }
__device__ __forceinline__ void st_c(double2* p, int64_t i, double2 v) { p[i] = v; }

constexpr int kMaxFreqBwd = 64;

// x^2 as a double, exact: from the mantissa's integer square (the FP64 pipe, two operations per clock
// and SM, is what bounds the diagonal adjoint)
__device__ __forceinline__ double square(float x) {
  const uint32_t u = __float_as_uint(x) & 0x7fffffffu, e = u >> 23;
  if (e - 1u >= 254u) return (double)x * (double)x;       // zero, subnormal, infinity, NaN
  const uint32_t m = (u & 0x7fffffu) | 0x800000u;
  const uint64_t p = (uint64_t)m * m;                     // in [2^46, 2^48)
  const int t = (int)(p >> 47);
  return __longlong_as_double((long long)(((uint64_t)(2 * e + (1023 - 254) + t) << 52) | ((p << (6 - t)) & 0xfffffffffffffull)));
}
__device__ __forceinline__ double square(double x) { return x * x; }

// s m rounded to the output type, s = c g.  FP32: c and g as sums of two FP32 numbers (48 bits), the
// product rounded once to within 2^-22 of half a unit, like the FP64 product rounded to FP32; `wide`
// (c or g outside the range where that holds) takes the FP64 product.
struct Split {
  float hi, lo;
  bool ok;
};
__device__ __forceinline__ Split split_of(double x) {     // integer operations: no FP64 subtraction
  const uint32_t h = (uint32_t)__double2hiint(x), l = (uint32_t)__double2loint(x);
  const int e = (int)((h >> 20) & 0x7ff);
  Split r;
  r.ok = (e >= 1023 - 40 && e <= 1023 + 40) || x == 0.0;
  const uint32_t sgn = h & 0x80000000u;
  r.hi = __uint_as_float(sgn | ((uint32_t)(e - 1023 + 127) << 23) | ((h & 0xfffffu) << 3) | (l >> 29));
  r.lo = (float)(l & 0x1fffffffu) * __uint_as_float(sgn | ((uint32_t)(e - 1023 - 52 + 127) << 23));
  if (x == 0.0) r.hi = r.lo = 0.f;
  return r;
}
__device__ __forceinline__ float2 scaled(double c, Split cs, double g, Split gs, float2 m) {
  if (cs.ok && gs.ok) {
    const float h = cs.hi * gs.hi;
    const float l = fmaf(cs.hi, gs.hi, -h) + fmaf(cs.hi, gs.lo, cs.lo * gs.hi);
    const float2 r = make_float2(fmaf(h, m.x, l * m.x), fmaf(h, m.y, l * m.y));
    if (fabsf(r.x) < INFINITY && fabsf(r.y) < INFINITY) return r;   // not 0 x infinity
  }
  const double s = c * g;
  return make_float2((float)(s * (double)m.x), (float)(s * (double)m.y));
}
__device__ __forceinline__ double2 scaled(double c, Split, double g, Split, double2 m) {
  const double s = c * g;
  return make_double2(s * m.x, s * m.y);
}

// fac[w][k] = (2 Re f, Re f') of pair p0 + k
__global__ void __launch_bounds__(128) k_bwd_factors(int64_t p0, int64_t K, int n_c, const double* __restrict__ E_v,
                                                     const double* __restrict__ E_col, const double* __restrict__ w_col,
                                                     const double2* __restrict__ omega, double delta,
                                                     double2* __restrict__ fac) {
  const int64_t k = (int64_t)blockIdx.x * 128 + threadIdx.x;
  if (k >= K) return;
  const int64_t p = p0 + k, iv = p / n_c, ic = p - iv * n_c;
  double2 f, fp;
  factors(E_v[iv] - E_col[ic], w_col ? w_col[ic] : 1.0, omega[blockIdx.y], delta, &f, &fp);
  fac[blockIdx.y * K + k] = make_double2(2.0 * f.x, fp.x);
}

// A CTA per P pairs of the block p0..p0+K, g [n_freq][nG] real, read once for
// them:  gM = sum_w 2 Re f_w g_w M,  gdE = sum_w Re f'_w sum_G g_w |M|^2.
// ONE: a single frequency, its factors out of the loop: two FP64 operations per
// element in FP32 plans.  Bound by the FP64 pipe and the integer squares: 1.01 ms
// for 128,000 pairs, N_G 1200 (2.4 TB/s); 3.97 ms with the square, both products,
// the conversions and every CTA's own factors on the FP64 pipe, and 2.2 ms more for
// the row sums by one thread per row.
//
// P = 4 pairs by 128 threads.  Up to BD_FEW pairs that leaves most of the GPU idle
// (64 pairs, N_G 2000, nine frequencies: 146 us a call): P = 1 by 256 threads, with
// several frequencies 512, which take the pair's factors themselves (60 us; 75 by the
// kernel before the grouping).  The line, six CTAs per SM: 1216 pairs, N_G 1200, one
// frequency 68 us by fours and 75 one by one, at 532 67 and 62; with nine they meet there.
constexpr int64_t BD_FEW = 912;
template <typename C, bool ONE, int P, int NT>
__global__ void __launch_bounds__(NT)
k_bwd_diag(const C* __restrict__ M, int nG, int64_t p0, int64_t K, int n_c, const double* __restrict__ E_v,
           const double* __restrict__ E_col, const double* __restrict__ w_col, const double2* __restrict__ omega,
           double delta, const double2* __restrict__ fac, int n_freq, const double* __restrict__ g, C* __restrict__ gM,
           double* __restrict__ gdE) {
  __shared__ double s_fr2[P][kMaxFreqBwd];   // 2 Re f
  __shared__ double s_fpr[P][kMaxFreqBwd];   // Re f'
  __shared__ double s_red[NT / 32][P];
  const int64_t k0 = (int64_t)blockIdx.x * P;
  const int np = (int)min((int64_t)P, K - k0);
  for (int e = threadIdx.x; e < np * n_freq; e += NT) {
    const int j = e / n_freq, iw = e - j * n_freq;
    double2 f;
    if (P == 1) {
      const int64_t p = p0 + k0, iv = p / n_c, ic = p - iv * n_c;
      double2 d;
      factors(E_v[iv] - E_col[ic], w_col ? w_col[ic] : 1.0, omega[iw], delta, &f, &d);
      f = make_double2(2.0 * f.x, d.x);
    } else {
      f = fac[iw * K + k0 + j];
    }
    s_fr2[j][iw] = f.x;
    s_fpr[j][iw] = f.y;
  }
  __syncthreads();
  double t[P] = {}, c[P];
  Split cs[P];
  if (ONE)
#pragma unroll
    for (int j = 0; j < P; ++j) {
      c[j] = j < np ? s_fr2[j][0] : 0.0;
      cs[j] = split_of(c[j]);
    }
  for (int G = threadIdx.x; G < nG; G += NT) {
    C m[P];
#pragma unroll
    for (int j = 0; j < P; ++j)
      if (j < np) m[j] = M[(k0 + j) * nG + G];
    if constexpr (ONE) {
      const double gw = g[G];
      const Split gs = split_of(gw);
#pragma unroll
      for (int j = 0; j < P; ++j)
        if (j < np) {
          gM[(k0 + j) * nG + G] = scaled(c[j], cs[j], gw, gs, m[j]);
          t[j] = fma(gw, square(m[j].x), t[j]);
          t[j] = fma(gw, square(m[j].y), t[j]);
        }
    } else if constexpr (P == 1) {
      const double2 d = make_double2((double)m[0].x, (double)m[0].y);
      const double m2 = d.x * d.x + d.y * d.y;
      double s = 0.0, s2 = 0.0;
      for (int iw = 0; iw < n_freq; ++iw) {
        const double gw = g[(int64_t)iw * nG + G];
        s = fma(s_fr2[0][iw], gw, s);
        s2 = fma(s_fpr[0][iw], gw, s2);
      }
      t[0] = fma(s2, m2, t[0]);
      st_c(gM, k0 * nG + G, make_double2(s * d.x, s * d.y));
    } else {
      double s[P] = {}, s2[P] = {};
      for (int iw = 0; iw < n_freq; ++iw) {
        const double gw = g[(int64_t)iw * nG + G];
#pragma unroll
        for (int j = 0; j < P; ++j)
          if (j < np) {
            s[j] = fma(s_fr2[j][iw], gw, s[j]);
            s2[j] = fma(s_fpr[j][iw], gw, s2[j]);
          }
      }
#pragma unroll
      for (int j = 0; j < P; ++j)
        if (j < np) {
          st_c(gM, (k0 + j) * nG + G, make_double2(s[j] * (double)m[j].x, s[j] * (double)m[j].y));
          t[j] = fma(s2[j], square(m[j].x), t[j]);
          t[j] = fma(s2[j], square(m[j].y), t[j]);
        }
    }
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if constexpr (P == 4) {
    // four sums over the warp in six additions: lanes keep two, then one of them
    const bool hi = lane & 16, hi2 = lane & 8;
    const double a0 = hi ? t[2] : t[0], a1 = hi ? t[3] : t[1], b0 = hi ? t[0] : t[2], b1 = hi ? t[1] : t[3];
    const double u0 = a0 + __shfl_xor_sync(0xffffffffu, b0, 16), u1 = a1 + __shfl_xor_sync(0xffffffffu, b1, 16);
    double r = (hi2 ? u1 : u0) + __shfl_xor_sync(0xffffffffu, hi2 ? u0 : u1, 8);
    for (int o = 4; o; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
    if ((lane & 7) == 0) s_red[warp][(hi ? 2 : 0) + (hi2 ? 1 : 0)] = r;
  } else {
    static_assert(P == 1, "reduction of one or four sums");
    for (int o = 16; o; o >>= 1) t[0] += __shfl_xor_sync(0xffffffffu, t[0], o);
    if (lane == 0) s_red[warp][0] = t[0];
  }
  __syncthreads();
  if (threadIdx.x < np) {
    double sum = 0.0;
    for (int w = 0; w < NT / 32; ++w) sum += s_red[w][threadIdx.x];
    gdE[k0 + threadIdx.x] = ONE ? s_fpr[threadIdx.x][0] * sum : sum;
  }
}

// dense upstream, one frequency after the other: tile of 32 pairs x 64 sphere points, K loop over H
//   Y[p][G] = sum_H M[p][H] Gam[G][H],  Z[p][G] = sum_H M[p][H] conj(Gam[H][G])
//   gM[p][G] += conj(f_p) Y + f_p Z;  part[p][gt] += Re( f'_p conj(sum_{G in tile} conj(M[p][G]) Y[p][G]) )
// (= at the first frequency).  flags (or NULL): [pairs / 64][ntile], only the tiles that are not 0 (mostly none, so one
// launch and not one per frequency to find that out).
template <typename C>
__global__ void __launch_bounds__(256)
k_bwd_dense(const C* __restrict__ M, int nG, int64_t p0, int64_t K, int n_c, const double* __restrict__ E_v,
            const double* __restrict__ E_col, const double* __restrict__ w_col, const double2* __restrict__ omega,
            int n_freq, double delta, const double2* __restrict__ Gam, C* __restrict__ gM, double* __restrict__ part,
            int ntile, const int* __restrict__ flags) {
  if (flags && flags[(blockIdx.y >> 1) * ntile + blockIdx.x] == 0) return;
  constexpr int TP = 32, TG = 64, TH = 16;
  __shared__ double2 Ms[TP][TH + 1];
  __shared__ double2 Gs[TG][TH + 1];     // Gam[G][H]
  __shared__ double2 Gt[TH][TG + 1];     // conj(Gam[H][G])
  __shared__ double2 sf[TP], sfp[TP];
  __shared__ double sq[TP][17];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;   // 16 x 16 threads: 2 pairs x 4 points each
  const int64_t kp0 = (int64_t)blockIdx.y * TP;
  const int G0 = blockIdx.x * TG;
  for (int iw = 0; iw < n_freq; ++iw, Gam += (int64_t)nG * nG) {
    __syncthreads();                       // the previous frequency's readers are done
    if (threadIdx.x < TP) {
      const int64_t k = kp0 + threadIdx.x;
      double2 f = make_double2(0, 0), fp = make_double2(0, 0);
      if (k < K) {
        const int64_t p = p0 + k, iv = p / n_c, ic = p - iv * n_c;
        factors(E_v[iv] - E_col[ic], w_col ? w_col[ic] : 1.0, omega[iw], delta, &f, &fp);
      }
      sf[threadIdx.x] = f;
      sfp[threadIdx.x] = fp;
    }
    double2 y[2][4], z[2][4];
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
      for (int c = 0; c < 4; ++c) y[r][c] = z[r][c] = make_double2(0, 0);
    for (int H0 = 0; H0 < nG; H0 += TH) {
      for (int e = threadIdx.x; e < TP * TH; e += blockDim.x) {
        const int r = e / TH, h = e - r * TH;
        const int64_t k = kp0 + r;
        Ms[r][h] = (k < K && H0 + h < nG) ? ld_d(M, k * nG + H0 + h) : make_double2(0, 0);
      }
      for (int e = threadIdx.x; e < TG * TH; e += blockDim.x) {
        const int gg = e / TH, h = e - gg * TH;
        const int G = G0 + gg, H = H0 + h;
        Gs[gg][h] = (G < nG && H < nG) ? Gam[(int64_t)G * nG + H] : make_double2(0, 0);
        const int hh = e / TG, g2 = e - hh * TG;
        const int Gb = G0 + g2, Hb = H0 + hh;
        double2 v = (Gb < nG && Hb < nG) ? Gam[(int64_t)Hb * nG + Gb] : make_double2(0, 0);
        v.y = -v.y;
        Gt[hh][g2] = v;
      }
      __syncthreads();
#pragma unroll 4
      for (int h = 0; h < TH; ++h) {
        double2 m[2];
#pragma unroll
        for (int r = 0; r < 2; ++r) m[r] = Ms[ty + 16 * r][h];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const double2 a = Gs[tx + 16 * c][h], b = Gt[h][tx + 16 * c];
#pragma unroll
          for (int r = 0; r < 2; ++r) {
            cfma(y[r][c], m[r], a);
            cfma(z[r][c], m[r], b);
          }
        }
      }
      __syncthreads();
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int rr = ty + 16 * r;
      const int64_t k = kp0 + rr;
      double2 qs = make_double2(0, 0);
      if (k < K) {
        const double2 f = sf[rr];
        const double2 fc = make_double2(f.x, -f.y);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int G = G0 + tx + 16 * c;
          if (G >= nG) continue;
          double2 gv = iw == 0 ? make_double2(0, 0) : ld_d(gM, k * nG + G);
          const double2 t1 = cmul(fc, y[r][c]), t2 = cmul(f, z[r][c]);
          gv.x += t1.x + t2.x;
          gv.y += t1.y + t2.y;
          st_c(gM, k * nG + G, gv);
          const double2 m = ld_d(M, k * nG + G);
          cfma(qs, make_double2(m.x, -m.y), y[r][c]);
        }
      }
      sq[rr][tx] = 0.0;
      if (k < K) {
        const double2 fp = sfp[rr];
        sq[rr][tx] = fp.x * qs.x + fp.y * qs.y;     // Re(f' conj(q))
      }
    }
    __syncthreads();
    if (threadIdx.x < TP) {
      const int64_t k = kp0 + threadIdx.x;
      if (k < K) {
        double sum = 0.0;
        for (int t = 0; t < 16; ++t) sum += sq[threadIdx.x][t];
        double* o = part + k * ntile + blockIdx.x;
        *o = iw == 0 ? sum : *o + sum;
      }
    }
  }
}

// Dense upstream from the residues of Y and Z (modgemm.cuh), frequencies w0 .. w0 + nw: plane set
// 2 w holds Y, 2 w + 1 holds Z of the block's pairs.  (Tiles that k_mod_check flagged for any of them are
// overwritten by k_bwd_dense.)
//   gM[k][G] (+)= sum_w conj(f) Y + f Z;  part[k][tile] (+)= Re( f' conj(sum_{G in tile} conj(M) Y) )
// A CTA takes 16 pairs x 64 sphere points, a warp 16 x 8 of them (half a residue block): two
// neighbouring lanes share a pair and take its even and odd points.  Bound by the integer pipe
// (reconstruction of two values from 52 residues), the FP64 pipe a third of it: 356 us for 4096
// pairs, N_G 1200, one frequency (530 us with one CTA per SM, before its registers were bounded).
// The whole adjoint of that size: 77.0 -> 1.02 ms (0.98 without the check of the products' S).
constexpr int BM_PAIRS = 16;
template <typename C>
__global__ void __launch_bounds__(256, 2)
k_bwd_mod(const int16_t* __restrict__ R, int rows, int ldR, const int* __restrict__ sA, const int* __restrict__ sB,
          const C* __restrict__ M, int nG, int64_t p0, int n_c, const double* __restrict__ E_v,
          const double* __restrict__ E_col, const double* __restrict__ w_col, const double2* __restrict__ omega, int w0,
          int nw, double delta, C* __restrict__ gM, double* __restrict__ part, int ntile) {
  __shared__ double2 sf[16], sfp[16];
  __shared__ double red[8][16];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, odd = lane & 1, r = lane >> 1;
  const int i = blockIdx.y * 16 + r, j0 = blockIdx.x * 64 + warp * 8;     // pair of the block, first point
  const int64_t k = i;
  const bool in = i < rows && j0 < nG;
  const size_t plane = mod::res_plane(rows, ldR);
  double2 g[4], m[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const int G = j0 + 2 * c + odd;
    g[c] = m[c] = make_double2(0.0, 0.0);
    if (in && G < nG) {
      m[c] = ld_d(M, k * nG + G);
      if (w0 > 0) g[c] = ld_d(gM, k * nG + G);
    }
  }
  double t = 0.0;
  for (int w = 0; w < nw; ++w) {
    __syncthreads();
    if (threadIdx.x < 16 && blockIdx.y * 16 + threadIdx.x < rows) {
      const int64_t p = p0 + blockIdx.y * 16 + threadIdx.x, iv = p / n_c, ic = p - iv * n_c;
      factors(E_v[iv] - E_col[ic], w_col ? w_col[ic] : 1.0, omega[w0 + w], delta, &sf[threadIdx.x], &sfp[threadIdx.x]);
    }
    __syncthreads();
    if (!in) continue;
    double2 y[4], z[4];
#pragma unroll
    for (int part2 = 0; part2 < 2; ++part2) {
      mod::Frac re[4] = {}, im[4] = {};
      mod::gather_fractions(R + mod::res_index(rows, ldR, (2 * w + part2) * mod::CPL, i, j0), plane, odd ? mod::ODD : mod::EVEN, re, im);
      const int sa = sA[k];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int G = min(j0 + 2 * c + odd, nG - 1), sb = sB[(size_t)(2 * w + part2) * nG + G];
        double2 v;
        if (sa == mod::NO_SCALE || sb == mod::NO_SCALE) v = make_double2(nan(""), nan(""));
        else v = make_double2(mod::frac_value(re[c], -sa - sb), mod::frac_value(im[c], -sa - sb));
        if (part2) z[c] = v; else y[c] = v;
      }
    }
    const double2 f = sf[r], fc = make_double2(f.x, -f.y), fp = sfp[r];
    double2 q = make_double2(0.0, 0.0);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      cfma(g[c], fc, y[c]);
      cfma(g[c], f, z[c]);
      if (j0 + 2 * c + odd < nG) cfma(q, make_double2(m[c].x, -m[c].y), y[c]);
    }
    t += fp.x * q.x + fp.y * q.y;     // Re(f' conj(q))
  }
#pragma unroll
  for (int c = 0; c < 4; ++c)
    if (in && j0 + 2 * c + odd < nG) st_c(gM, k * nG + j0 + 2 * c + odd, g[c]);
  t += __shfl_xor_sync(0xffffffffu, t, 1);
  if (!odd) red[warp][r] = t;
  __syncthreads();
  if (threadIdx.x < 16 && blockIdx.y * 16 + threadIdx.x < rows) {
    double s = 0.0;
    for (int w = 0; w < 8; ++w) s += red[w][threadIdx.x];
    double* o = part + (int64_t)(blockIdx.y * 16 + threadIdx.x) * ntile + blockIdx.x;
    *o = w0 > 0 ? *o + s : s;
  }
}

// gdE[k] = sum_t part[k][t]
__global__ void k_rowsum(const double* __restrict__ part, int64_t K, int ntile, double* __restrict__ gdE) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= K) return;
  double s = 0.0;
  for (int t = 0; t < ntile; ++t) s += part[k * ntile + t];
  gdE[k] = s;
}

// grad E_v[iv] += sum of gdE over the block's pairs in row iv; grad E_col[ic] -= column sums.  A CTA
// per row, 32 x 32 threads per 32 columns, sums in a fixed order (one thread per row took 135 us for a
// block of 8192 pairs in rows of 2000).
__global__ void __launch_bounds__(128) k_reduce_rows(const double* __restrict__ gdE, int64_t p0, int64_t K, int n_c,
                                                     double* __restrict__ gEv) {
  __shared__ double red[4];
  const int64_t iv = p0 / n_c + blockIdx.x;
  const int64_t a = max(p0, iv * n_c), b = min(p0 + K, (iv + 1) * n_c);
  double s = 0.0;
  for (int64_t p = a + threadIdx.x; p < b; p += 128) s += gdE[p - p0];
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) gEv[iv] += (red[0] + red[1]) + (red[2] + red[3]);
}
__global__ void __launch_bounds__(1024) k_reduce_cols(const double* __restrict__ gdE, int64_t p0, int64_t K, int n_c,
                                                      double* __restrict__ gEc) {
  __shared__ double red[32][33];
  const int64_t ic = (int64_t)blockIdx.x * 32 + threadIdx.x;
  double s = 0.0;
  if (ic < n_c)
    for (int64_t iv = p0 / n_c + threadIdx.y; iv * n_c + ic < p0 + K; iv += 32) {
      const int64_t p = iv * n_c + ic;
      if (p >= p0) s += gdE[p - p0];
    }
  red[threadIdx.y][threadIdx.x] = s;
  __syncthreads();
  // thread row y sums column y of the tile over the 32 partial rows
  s = red[threadIdx.x][threadIdx.y];
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  const int64_t c = (int64_t)blockIdx.x * 32 + threadIdx.y;
  if (threadIdx.x == 0 && c < n_c) gEc[c] -= s;
}

// Eq. 4 step edge e_k = min(E_0 + k dE, E_max), rounded as written (no fused multiply-add, so the
// value is the same as the host selection's)
__device__ __forceinline__ double step_edge(double E0, double dE, int k, double E_max) {
  return fmin(__dadd_rn(E0, __dmul_rn(dE, (double)k)), E_max);
}

// First-order estimate of the energy substitution of Eq. 3/4: every band c >= N0 takes the
// midpoint E_i of the Eq. 4 step [e_k, e_k+1) holding E_c (the last step closed, energies outside
// [E_0, E_max] to the end steps), and the estimate is sum_c sens_c (E_i(c) - E_c).  One block:
// each thread sums a fixed stride of bands, then a fixed tree in shared memory (deterministic).
constexpr int kEstThreads = 1024;
__global__ void __launch_bounds__(kEstThreads)
k_energy_substitution(const double* __restrict__ E_c, const double* __restrict__ sens, int n_c, int N0, double dE,
                      double E_max, double* __restrict__ E_sub, double* __restrict__ out) {
  __shared__ double red[kEstThreads];
  // E_0 = E_c of band N0 and N_E = ceil((E_max - E_0) / dE) steps, as the host selection has them
  const bool grid = N0 > 0 && N0 < n_c;
  const double E0 = grid ? E_c[N0 - 1] : 0.0;
  const int NE = grid ? (int)fmax(ceil((E_max - E0) / dE - 1e-12), 0.0) : 0;
  double acc = 0.0;
  for (int c = threadIdx.x; c < n_c; c += kEstThreads) {
    const double E = E_c[c];
    double Ei = E;
    if (c >= N0 && NE > 0) {
      // last k in [0, NE-1] with e_k <= E: start from the quotient, then step to the exact edge
      int k = (int)fmin(fmax(floor((E - E0) / dE), 0.0), (double)(NE - 1));
      while (k + 1 <= NE - 1 && step_edge(E0, dE, k + 1, E_max) <= E) ++k;
      while (k > 0 && step_edge(E0, dE, k, E_max) > E) --k;
      const double lo = step_edge(E0, dE, k, E_max), hi = step_edge(E0, dE, k + 1, E_max);
      Ei = __dmul_rn(0.5, __dadd_rn(lo, hi));
      acc = __dadd_rn(acc, __dmul_rn(sens[c], __dadd_rn(Ei, -E)));
    }
    if (E_sub) E_sub[c] = Ei;
  }
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int h = kEstThreads / 2; h > 0; h >>= 1) {
    if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = red[0];
}

}  // namespace

cudaError_t launch_energy_substitution(const double* E_c, const double* sens, int n_c, int N0, double dE, double E_max,
                                       double* E_sub, double* out, cudaStream_t s) {
  k_energy_substitution<<<1, kEstThreads, 0, s>>>(E_c, sens, n_c, N0, dE, E_max, E_sub, out);
  return cudaGetLastError();
}

int bwd_max_freq() { return kMaxFreqBwd; }
// doubles of work for K pairs at a time: grad dE, then per-tile sums (dense) or factors (diagonal)
size_t bwd_work_doubles(int nG, int n_freq, int64_t K) {
  return (size_t)(K + 1) / 2 * 2 + (size_t)K * std::max((nG + 63) / 64, 2 * std::min(n_freq, kMaxFreqBwd));
}

// all frequencies of the pairs' dense adjoint (flags: the flagged tiles') by FP64 multiply-adds
template <typename C>
static void dense_direct(chi0_plan_s* p, int nG, const C* M, int64_t p0, int64_t K, int n_c, const double* E_v,
                         const double* E_col, const double* w_col, const double2* gamma, C* gM, double* part,
                         const int* flags, cudaStream_t s) {
  const int ntile = (nG + 63) / 64;
  k_bwd_dense<C><<<dim3(ntile, (unsigned)((K + 31) / 32)), 256, 0, s>>>(
      M, nG, p0, K, n_c, E_v, E_col, w_col, p->d_omega, p->n_freq, p->delta, gamma, gM, part, ntile, flags);
}

template <typename C>
static cudaError_t bwd_impl(chi0_plan_s* p, int nG, const C* M, int64_t p0, int64_t K, int n_c, const double* E_v,
                            const double* E_col, const double* w_col, const double2* gamma, const double* diag,
                            C* gM, double* gEv, double* gEc, double* work, cudaStream_t s) {
  double* gdE = work;
  if (diag) {
    double2* fac = reinterpret_cast<double2*>(work + (K + 1) / 2 * 2);
    const bool one = p->n_freq == 1, few = K <= BD_FEW;
    if (!few)
      k_bwd_factors<<<dim3((unsigned)((K + 127) / 128), p->n_freq), 128, 0, s>>>(p0, K, n_c, E_v, E_col, w_col, p->d_omega,
                                                                                p->delta, fac);
    auto* kern = few ? (one ? k_bwd_diag<C, true, 1, 256> : k_bwd_diag<C, false, 1, 512>)
                     : (one ? k_bwd_diag<C, true, 4, 128> : k_bwd_diag<C, false, 4, 128>);
    kern<<<(unsigned)(few ? K : (K + 3) / 4), few ? (one ? 256 : 512) : 128, 0, s>>>(
        M, nG, p0, K, n_c, E_v, E_col, w_col, p->d_omega, p->delta, fac, p->n_freq, diag, gM, gdE);
  } else {
    const int ntile = (nG + 63) / 64;
    double* part = work + K;
    dense_direct<C>(p, nG, M, p0, K, n_c, E_v, E_col, w_col, gamma, gM, part, nullptr, s);
    k_rowsum<<<(unsigned)((K + 255) / 256), 256, 0, s>>>(part, K, ntile, gdE);
  }
  const int64_t rows = (p0 + K - 1) / n_c - p0 / n_c + 1;
  k_reduce_rows<<<(unsigned)rows, 128, 0, s>>>(gdE, p0, K, n_c, gEv);
  k_reduce_cols<<<(unsigned)((n_c + 31) / 32), dim3(32, 32), 0, s>>>(gdE, p0, K, n_c, gEc);
  return cudaGetLastError();
}

// Where the tensor-core form of the dense adjoint pays: estimates in microseconds.  A tile of
// k_bwd_dense takes 4.1 us per sphere point of the contraction (FP64 pipe), so even one pair costs that
// times N_G per frequency; the modular form costs its launches, the planes of Gamma and the products.
bool bwd_mod_pays(const chi0_plan_s* p, int nG, int64_t n_pairs) {
  const double n2 = (double)nG * nG, K = (double)n_pairs;
  const double direct = p->n_freq * std::max(4.1 * nG, 16.0 * n2 * K / 1.1e6);
  const double modular = 80.0 + p->n_freq * (20.0 + 6e-5 * n2 + 7e-5 * K * nG + 9e-8 * n2 * K);
  return modular < direct;
}

// Memory of a pass over the pairs: planes of Gamma and Gamma^H for nw frequencies, planes of M and
// residues of Y and Z for kc pairs, scales
struct BwdMod {
  int Kp, ldR, nw, kc;
  size_t off_a, off_r, off_sa, off_sb, off_na, off_nb, off_flag, off_ws, bytes;
};
static BwdMod bwd_mod_sizes(const chi0_plan_s* p, int nG, int64_t n_pairs) {
  constexpr int64_t kMem = (int64_t)4 << 30;
  auto al = [](size_t x) { return (x + 255) / 256 * 256; };
  BwdMod z;
  z.Kp = (nG + 63) / 64 * 64;
  z.ldR = (nG + 7) / 8 * 8;
  const int64_t gam = (int64_t)2 * mod::CPL * 2 * nG * z.Kp;                  // one frequency's planes
  z.nw = (int)std::max<int64_t>(1, std::min<int64_t>(p->n_freq, kMem / gam));
  const int64_t per_pair = (int64_t)2 * z.nw * mod::CPL * 2 * z.ldR;           // residues of one pair
  z.kc = (int)std::min<int64_t>({n_pairs, p->max_pairs, std::max<int64_t>(256, kMem / per_pair / 256 * 256),
                                 (int64_t)65535 * BM_PAIRS});   // grid y of k_bwd_mod
  z.off_a = al((size_t)gam * z.nw);
  z.off_r = z.off_a + al((size_t)mod::CPL * 2 * z.kc * z.Kp);
  z.off_sa = z.off_r + al((size_t)2 * z.nw * mod::CPL * 2 * mod::res_plane(z.kc, z.ldR));
  z.off_sb = z.off_sa + al(sizeof(int) * (size_t)z.kc);
  z.off_na = z.off_sb + al(sizeof(int) * (size_t)2 * z.nw * nG);
  z.off_nb = z.off_na + al(sizeof(float) * (size_t)z.kc);
  z.off_flag = z.off_nb + al(sizeof(float) * (size_t)2 * z.nw * nG);
  z.off_ws = z.off_flag + al(sizeof(int) * (size_t)((z.kc + 63) / 64) * ((nG + 63) / 64));
  z.bytes = z.off_ws + al(mod_cols_ws_bytes(nG, nG));
  return z;
}
size_t bwd_mod_ws_bytes(const chi0_plan_s* p, int nG, int64_t n_pairs) { return bwd_mod_sizes(p, nG, n_pairs).bytes; }

template <typename C>
static cudaError_t bwd_mod_impl(chi0_plan_s* p, int nG, const C* M, int64_t n_pairs, int n_c, const double* E_v,
                                const double* E_col, const double* w_col, const double2* gamma, C* gM, double* gEv,
                                double* gEc, double* work, void* ws, cudaStream_t s) {
  const BwdMod z = bwd_mod_sizes(p, nG, n_pairs);
  unsigned char* b = reinterpret_cast<unsigned char*>(ws);
  uint16_t* Bp = reinterpret_cast<uint16_t*>(b);
  uint16_t* Ap = reinterpret_cast<uint16_t*>(b + z.off_a);
  int16_t* R = reinterpret_cast<int16_t*>(b + z.off_r);
  int* sA = reinterpret_cast<int*>(b + z.off_sa);
  int* sB = reinterpret_cast<int*>(b + z.off_sb);
  float* nA = reinterpret_cast<float*>(b + z.off_na);
  float* nB = reinterpret_cast<float*>(b + z.off_nb);
  int* flags = reinterpret_cast<int*>(b + z.off_flag);
  const size_t set = (size_t)mod::CPL * nG * z.Kp;       // 16-bit words of one operand's planes
  const int ntile = (nG + 63) / 64;
  cudaError_t e;
  // every pair block keeps its sums over the frequencies in gM and part: with several groups of
  // frequencies the groups run inside the block and the planes of Gamma are made again for each
  for (int64_t p0 = 0; p0 < n_pairs; p0 += z.kc) {
    const int K = (int)std::min<int64_t>(z.kc, n_pairs - p0);
    double* gdE = work;
    double* part = work + K;
    e = cudaMemsetAsync(flags, 0, sizeof(int) * (size_t)((K + 63) / 64) * ntile, s);
    if (e == cudaSuccess) e = launch_mod_pack_rows(M + p0 * nG, K, nG, nG, z.Kp, true, sA, nA, Ap, s);
    if (e != cudaSuccess) return e;
    for (int w0 = 0; w0 < p->n_freq; w0 += z.nw) {
      const int nw = std::min(z.nw, p->n_freq - w0);
      if (p0 == 0 || z.nw < p->n_freq)
        for (int w = 0; w < nw; ++w) {
          const double2* G = gamma + (size_t)(w0 + w) * nG * nG;
          e = launch_mod_pack_rows(G, nG, nG, nG, z.Kp, false, sB + (size_t)2 * w * nG,
                                   nB + (size_t)2 * w * nG, Bp + 2 * w * set, s);
          if (e == cudaSuccess)
            e = launch_mod_pack_cols(G, nG, nG, z.Kp, true, sB + (size_t)(2 * w + 1) * nG, nB + (size_t)(2 * w + 1) * nG,
                                     Bp + (2 * w + 1) * set, b + z.off_ws, s);
          if (e != cudaSuccess) return e;
        }
      ModGemm g{Ap, Bp, R, K, 0, K, nG, z.ldR, z.Kp, 2 * nw * mod::CPL, mod::CPL, 2 * nw * mod::CPL, mod::CPL, nullptr};
      e = launch_mod_gemm(p, g, s);
      if (e == cudaSuccess) e = launch_mod_check(R, K, nG, z.ldR, 0, nA, 0, nB, nG, flags, 0, 2 * nw, s);
      if (e != cudaSuccess) return e;
      k_bwd_mod<C><<<dim3(ntile, (K + BM_PAIRS - 1) / BM_PAIRS), 256, 0, s>>>(R, K, z.ldR, sA, sB, M + p0 * nG, nG, p0, n_c, E_v, E_col,
                                                              w_col, p->d_omega, w0, nw, p->delta, gM + p0 * nG, part,
                                                              ntile);
    }
    dense_direct<C>(p, nG, M + p0 * nG, p0, K, n_c, E_v, E_col, w_col, gamma, gM + p0 * nG, part, flags, s);
    k_rowsum<<<(unsigned)((K + 255) / 256), 256, 0, s>>>(part, K, ntile, gdE);
    const int64_t rows = (p0 + K - 1) / n_c - p0 / n_c + 1;
    k_reduce_rows<<<(unsigned)rows, 128, 0, s>>>(gdE, p0, K, n_c, gEv);
    k_reduce_cols<<<(unsigned)((n_c + 31) / 32), dim3(32, 32), 0, s>>>(gdE, p0, K, n_c, gEc);
  }
  return cudaGetLastError();
}

cudaError_t launch_backward_mod(chi0_plan_s* p, int nG, const void* M, int64_t n_pairs, int n_c, const double* E_v,
                                const double* E_col, const double* w_col, const double2* gamma, void* gM, double* gEv,
                                double* gEc, double* work, void* ws, cudaStream_t s) {
  if (is_split(p))
    return bwd_mod_impl<float2>(p, nG, (const float2*)M, n_pairs, n_c, E_v, E_col, w_col, gamma, (float2*)gM, gEv, gEc,
                                work, ws, s);
  return bwd_mod_impl<double2>(p, nG, (const double2*)M, n_pairs, n_c, E_v, E_col, w_col, gamma, (double2*)gM, gEv, gEc,
                               work, ws, s);
}

cudaError_t launch_backward(chi0_plan_s* p, int nG, const void* M, int64_t p0, int64_t K, int n_c, const double* E_v,
                            const double* E_col, const double* w_col, const double2* gamma, const double* diag,
                            void* gM, double* gEv, double* gEc, double* work, cudaStream_t s) {
  if (is_split(p))
    return bwd_impl<float2>(p, nG, (const float2*)M + p0 * nG, p0, K, n_c, E_v, E_col, w_col, gamma, diag,
                            (float2*)gM + p0 * nG, gEv, gEc, work, s);
  return bwd_impl<double2>(p, nG, (const double2*)M + p0 * nG, p0, K, n_c, E_v, E_col, w_col, gamma, diag,
                           (double2*)gM + p0 * nG, gEv, gEc, work, s);
}

}  // namespace chi0
