// FP64 contraction of Eq. 1 on the tensor cores (CHI0_FP64 plans):
//   chi0[w][G][H] += sum_p f_p(w) M_p(G) conj(M_p(H))
// as exact modular products (modgemm.cuh): FP64 accuracy from 26 FP16 products.
//
// Steps of a block of K pairs: row norms and scales (k_mod_fmax, k_mod_rowmax,
// k_mod_norms, k_mod_scales), residue planes of conj(M) and of W_w = f(w) M
// (k_mod_pack), 26 products per frequency with their sums reduced modulo m and one
// of the magnitudes (k_mod_gemm), tiles that want FP64 sums (k_mod_check),
// reconstruction and addition into chi0 (k_mod_add), those tiles (k_contract_f64).
//
// The CUDA-core contraction ran at the FP64 pipe's rate (two multiply-adds per clock
// and SM): 790 ms for 2048 pairs, N_G 2500, nine frequencies.  This form takes
// 6.4 ms: 4.05 ms of products (the 16-bit tensor pipe 67 % busy at 1.9 GHz, 1.6
// PFLOP/s executed), 1.15 ms reconstruction, 0.71 ms planes, 0.19 ms norms; the check
// of S (k_mod_check, its plane in all the steps) is 0.25 ms of it.  The static 8-atom
// contraction (3840 pairs, N_G 350): 15.97 ms -> 0.20 ms.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <string>

#include "cplx.cuh"
#include "internal.h"
#include "modgemm.cuh"
#include "tc_ptx.cuh"

namespace chi0 {
namespace {

using mod::NM;
using mod::NPL;
using mod::CPL;
using mod::gather_fractions;
using mod::res_index;
using mod::res_plane;
using mod::add2;
using mod::fma2;
using mod::pack2;
using mod::unpack2;

// ---------------------------------------------------------------------------
// scales
// ---------------------------------------------------------------------------
// ef[w] = largest magnitude word of the factors f[w][0..K)
__global__ void __launch_bounds__(256) k_mod_fmax(const double2* __restrict__ f, int64_t K, uint32_t* __restrict__ ef) {
  __shared__ uint32_t red[8];
  uint32_t m = 0;
  for (int64_t k = threadIdx.x; k < K; k += blockDim.x) {
    const double2 v = f[(int64_t)blockIdx.x * K + k];
    m = max(m, max(mod::mag_word(v.x), mod::mag_word(v.y)));
  }
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < 8; ++i) m = max(m, red[i]);
    ef[blockIdx.x] = m;
  }
}

constexpr int ST_COLS = 64, ST_ROWS = 128;   // a statistics block: 64 sphere points x 128 pairs

// eg[G] = largest magnitude word of M[0..K)[G] (eg cleared by the caller)
__global__ void __launch_bounds__(256) k_mod_rowmax(const double2* __restrict__ M, int nG, int64_t K,
                                                    uint32_t* __restrict__ eg, const int* __restrict__ todo) {
  if (todo && *todo == 0) return;
  const int G = blockIdx.x * ST_COLS + (threadIdx.x & 63);
  if (G >= nG) return;
  const int64_t k1 = min(K, (int64_t)(blockIdx.y + 1) * ST_ROWS);
  uint32_t m = 0;
  for (int64_t k = (int64_t)blockIdx.y * ST_ROWS + (threadIdx.x >> 6); k < k1; k += 4) {
    const double2 v = M[k * nG + G];
    m = max(m, max(mod::mag_word(v.x), mod::mag_word(v.y)));
  }
  atomicMax(eg + G, m);
}

// part[block of pairs][slot][G] = sum over the block of |M|^2 4^-eg (slot 0) and of
// |f(w)|^2 |M|^2 4^-(eg + ef) (slot 1 + w): FP64 sums in a fixed order (a scale that
// depended on the order could move a result by its rounding from run to run)
__global__ void __launch_bounds__(256) k_mod_norms(const double2* __restrict__ M, int nG, int64_t K,
                                                   const double2* __restrict__ f, int n_freq,
                                                   const uint32_t* __restrict__ eg, const uint32_t* __restrict__ ef,
                                                   double* __restrict__ part) {
  __shared__ double f2[ST_ROWS];
  __shared__ double red[4][ST_COLS];
  const int g = threadIdx.x & 63, r = threadIdx.x >> 6, G = blockIdx.x * ST_COLS + g;
  const int64_t k0 = (int64_t)blockIdx.y * ST_ROWS;
  double m2[ST_ROWS / 4];
  const uint32_t wg = G < nG ? eg[G] : 0;
  const bool use = wg >= 0x00100000u && wg < 0x7ff00000u;
  // 2^-eg in two steps: its exponent may leave the normal range
  const int e = mod::word_exp(wg);
  const double s1 = use ? mod::pow2d(-(e / 2)) : 0.0, s2 = use ? mod::pow2d(-(e - e / 2)) : 0.0;
#pragma unroll
  for (int j = 0; j < ST_ROWS / 4; ++j) {
    const int64_t k = k0 + r + 4 * j;
    m2[j] = 0.0;
    if (use && k < K) {
      const double2 v = M[k * nG + G];
      const double x = v.x * s1 * s2, y = v.y * s1 * s2;
      m2[j] = fma(x, x, y * y);
    }
  }
  for (int slot = 0; slot <= n_freq; ++slot) {
    __syncthreads();
    if (slot > 0 && threadIdx.x < ST_ROWS) {
      const int64_t k = k0 + threadIdx.x;
      double v = 0.0;
      const uint32_t wf = ef[slot - 1];
      if (k < K && wf >= 0x00100000u && wf < 0x7ff00000u) {
        const double2 d = f[(int64_t)(slot - 1) * K + k];
        const int q = mod::word_exp(wf);
        const double t1 = mod::pow2d(-(q / 2)), t2 = mod::pow2d(-(q - q / 2));
        const double x = d.x * t1 * t2, y = d.y * t1 * t2;
        v = fma(x, x, y * y);
      }
      f2[threadIdx.x] = v;
    }
    __syncthreads();
    double s = 0.0;
#pragma unroll
    for (int j = 0; j < ST_ROWS / 4; ++j) s = slot ? fma(m2[j], f2[r + 4 * j], s) : s + m2[j];
    red[r][g] = s;
    __syncthreads();
    if (r == 0 && G < nG)
      part[((size_t)blockIdx.y * (n_freq + 1) + slot) * nG + G] = (red[0][g] + red[1][g]) + (red[2][g] + red[3][g]);
  }
}

// slot 0 alone, relative to the column's own largest element: FP32 sums do (what underflows is below
// 2^-126 of the norm), without the FP64 pipe
__global__ void __launch_bounds__(256) k_mod_col_norms(const double2* __restrict__ M, int nG, int64_t K,
                                                       const uint32_t* __restrict__ eg, double* __restrict__ part,
                                                       const int* __restrict__ todo) {
  if (todo && *todo == 0) return;
  __shared__ float red[4][ST_COLS];
  const int g = threadIdx.x & 63, r = threadIdx.x >> 6, G = blockIdx.x * ST_COLS + g;
  const int64_t k0 = (int64_t)blockIdx.y * ST_ROWS;
  const uint32_t wg = G < nG ? eg[G] : 0;
  float s = 0.f;
  if (wg >= 0x00100000u && wg < 0x7ff00000u) {
    const int e = mod::word_exp(wg);
    for (int j = r; j < ST_ROWS && k0 + j < K; j += 4) {
      const double2 v = M[(k0 + j) * nG + G];
      const float x = mod::scaled_abs(v.x, e), y = mod::scaled_abs(v.y, e);
      s = fmaf(x, x, fmaf(y, y, s));
    }
  }
  red[r][g] = s;
  __syncthreads();
  if (r == 0 && G < nG) part[(size_t)blockIdx.y * nG + G] = (double)((red[0][g] + red[1][g]) + (red[2][g] + red[3][g]));
}

// scale exponents and, where norm is not NULL, scaled norms: slot 0 (conj(M), operand B) and 1 + w (W_w, operand A)
__global__ void __launch_bounds__(256) k_mod_scales(const double* __restrict__ part, int n_part, int nG, int n_freq,
                                                    const uint32_t* __restrict__ eg, const uint32_t* __restrict__ ef,
                                                    int* __restrict__ scale, float* __restrict__ norm) {
  const int G = blockIdx.x * blockDim.x + threadIdx.x, slot = blockIdx.y;
  if (G >= nG) return;
  double s = 0.0;
  for (int b = 0; b < n_part; ++b) s += part[((size_t)b * (n_freq + 1) + slot) * nG + G];
  const uint32_t wg = eg[G], wf = slot ? ef[slot - 1] : 0x3ff00000u;
  int r;
  const int e = mod::word_exp(wg) + (slot ? mod::word_exp(wf) : 0), beta = slot ? mod::BETA_A : mod::BETA_B;
  if (wg >= 0x7ff00000u || wf >= 0x7ff00000u) r = mod::NO_SCALE;   // the result row is NaN
  else r = mod::scale_exp(s, e, beta);
  scale[(size_t)slot * nG + G] = r;
  if (norm) norm[(size_t)slot * nG + G] = mod::scaled_norm(s, r, e, beta);
}

// ---------------------------------------------------------------------------
// residue planes
// ---------------------------------------------------------------------------
constexpr int PK_G = 16, PK_K = 64;   // tile: 16 sphere points x 64 pairs, transposed through shared memory

// Planes [26][nG][Kp] (FP16) of conj(M) (of M: conj = false) into Bp (when not NULL) and of W_w = f(w) M,
// w = w0 .. w0 + nw, into Ap (26 planes per frequency; CHECK: 27, with the
// magnitudes; REST: 34, with the remainders).  A warp holds one sphere point, a lane two neighbouring pairs:
// 128-byte stores per plane.
template <mod::Extra X>
__global__ void __launch_bounds__(256) k_mod_pack(const double2* __restrict__ M, int nG, int64_t K, int Kp,
                                                  const double2* __restrict__ f, int w0, int nw,
                                                  const int* __restrict__ scale, bool conj, uint32_t* __restrict__ Bp,
                                                  uint32_t* __restrict__ Ap, const int* __restrict__ todo) {
  if (todo && *todo == 0) return;
  __shared__ double2 tile[PK_K][PK_G + 1];
  __shared__ double2 fs[PK_K];
  const int G0 = blockIdx.x * PK_G;
  const int64_t p0 = (int64_t)blockIdx.y * PK_K;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int e = threadIdx.x; e < PK_K * PK_G; e += blockDim.x) {
    const int pp = e / PK_G, g = e - pp * PK_G;
    double2 v = make_double2(0.0, 0.0);
    if (p0 + pp < K && G0 + g < nG) v = M[(p0 + pp) * nG + G0 + g];
    tile[pp][g] = v;
  }
  const size_t plane = (size_t)nG * (Kp / 2);
  for (int slot = Bp ? -1 : 0; slot < nw; ++slot) {
    __syncthreads();
    if (slot >= 0 && threadIdx.x < PK_K) {
      const int64_t p = p0 + threadIdx.x;
      fs[threadIdx.x] = p < K ? f[(int64_t)(w0 + slot) * K + p] : make_double2(0.0, 0.0);
    }
    __syncthreads();
    const int* sc = scale + (size_t)(slot < 0 ? 0 : 1 + w0 + slot) * nG;
    uint32_t* dst = slot < 0 ? Bp : Ap + (size_t)slot * (X == mod::CHECK ? CPL : NPL) * plane;
    for (int g = warp; g < PK_G; g += 8) {
      const int G = G0 + g;
      if (G >= nG) break;
      const int s = sc[G];
      double2 a = tile[2 * lane][g], b = tile[2 * lane + 1][g];
      if (slot >= 0) {
        a = cmul(fs[2 * lane], a);
        b = cmul(fs[2 * lane + 1], b);
      }
      const int64_t ax = mod::quantise(a.x, s), bx = mod::quantise(b.x, s), ay = mod::quantise(a.y, s), by = mod::quantise(b.y, s);
      const mod::Limbs x = mod::limbs(ax, bx), y = mod::limbs(ay, by);
      uint32_t* o = dst + (size_t)G * (Kp / 2) + p0 / 2 + lane;
      mod::store_residues(x, y, slot < 0 && conj, o, plane);
      if (X == mod::CHECK) mod::store_magnitudes(x, y, slot < 0 ? mod::BETA_B : mod::BETA_A, o, plane);
      if (X == mod::REST)
        mod::store_remainders(x, y, mod::pack2(mod::rest_of(a.x, s, ax), mod::rest_of(b.x, s, bx)),
                              mod::pack2(mod::rest_of(a.y, s, ay), mod::rest_of(b.y, s, by)), mod::BETA_B, o, plane);
    }
  }
}

// Rows whose contraction index is contiguous: X [rows][n] with row stride ld.
__device__ __forceinline__ double2 ld_wide(const float2* p, size_t i) { return make_double2(p[i].x, p[i].y); }
__device__ __forceinline__ double2 ld_wide(const double2* p, size_t i) { return p[i]; }

// scale[row]: a CTA per row, the largest magnitude and then the norm (FP32, relative to the
// largest: what underflows there does not count), summed in a fixed order
template <typename C>
__global__ void __launch_bounds__(128) k_mod_row_scales(const C* __restrict__ X, int n, size_t ld, int beta,
                                                        int* __restrict__ scale, float* __restrict__ norm,
                                                        const int* __restrict__ todo) {
  if (todo && *todo == 0) return;
  __shared__ uint32_t mx[4];
  __shared__ float sm[4];
  const C* x = X + blockIdx.x * ld;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint32_t m = 0;
  for (int i = threadIdx.x; i < n; i += 128) {
    const double2 v = ld_wide(x, i);
    m = max(m, max(mod::mag_word(v.x), mod::mag_word(v.y)));
  }
  m = __reduce_max_sync(0xffffffffu, m);
  if (lane == 0) mx[warp] = m;
  __syncthreads();
  m = max(max(mx[0], mx[1]), max(mx[2], mx[3]));
  const int e = mod::word_exp(m);
  float s = 0.f;
  if (m >= 0x00100000u && m < 0x7ff00000u)
    for (int i = threadIdx.x; i < n; i += 128) {
      const double2 v = ld_wide(x, i);
      const float a = mod::scaled_abs(v.x, e), b = mod::scaled_abs(v.y, e);
      s = fmaf(a, a, fmaf(b, b, s));
    }
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) sm[warp] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    const double n2 = (double)((sm[0] + sm[1]) + (sm[2] + sm[3]));
    const int r = m >= 0x7ff00000u ? mod::NO_SCALE : mod::scale_exp(n2, e, beta);
    scale[blockIdx.x] = r;
    if (norm) norm[blockIdx.x] = mod::scaled_norm(n2, r, e, beta);
  }
}

// planes [26][rows][Kp] of X (CHECK: 27, with the magnitudes, REST: 34, with the remainders); a warp takes 64
// elements of a row
template <typename C, mod::Extra E>
__global__ void __launch_bounds__(256) k_mod_pack_rows(const C* __restrict__ X, int rows, int n, size_t ld, int Kp,
                                                       const int* __restrict__ scale, int beta,
                                                       uint32_t* __restrict__ dst, const int* __restrict__ todo) {
  if (todo && *todo == 0) return;
  const int lane = threadIdx.x & 31, segs = Kp / 64;
  const int64_t unit = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  if (unit >= (int64_t)rows * segs) return;
  const int r = (int)(unit / segs), k = (int)(unit - (int64_t)r * segs) * 64 + 2 * lane;
  const C* x = X + r * ld;
  const int s = scale[r];
  const double2 a = k < n ? ld_wide(x, k) : make_double2(0.0, 0.0);
  const double2 b = k + 1 < n ? ld_wide(x, k + 1) : make_double2(0.0, 0.0);
  const int64_t ax = mod::quantise(a.x, s), bx = mod::quantise(b.x, s), ay = mod::quantise(a.y, s), by = mod::quantise(b.y, s);
  const mod::Limbs u = mod::limbs(ax, bx), v = mod::limbs(ay, by);
  uint32_t* o = dst + (size_t)r * (Kp / 2) + k / 2;
  mod::store_residues(u, v, false, o, (size_t)rows * (Kp / 2));
  if (E == mod::CHECK) mod::store_magnitudes(u, v, beta, o, (size_t)rows * (Kp / 2));
  if (E == mod::REST)
    mod::store_remainders(u, v, mod::pack2(mod::rest_of(a.x, s, ax), mod::rest_of(b.x, s, bx)),
                          mod::pack2(mod::rest_of(a.y, s, ay), mod::rest_of(b.y, s, by)), beta, o, (size_t)rows * (Kp / 2));
}

// ---------------------------------------------------------------------------
// modular products
// ---------------------------------------------------------------------------
// R[b][i][j] = sum_k A[b][i][k] B[b][j][k] (mod m of plane b), |R| <= 255; of the planes after the
// residues the sum itself, rounded.
// A CTA pair computes a 256 x 256 tile with tcgen05.mma.cta_group::2 (each CTA
// holds 128 rows of A and 128 of B: 32 KB per 512 MMA cycles, half the operand
// traffic per flop of two single-CTA 128 x 128 tiles).  Warp 0 issues the TMA
// loads (128-byte rows of 64 k) into a ring, warp 1 of the first CTA the MMAs into
// two 256-column accumulators, warps 4..11 drain them: a chain is 256 k (the
// longest whose sums are exact), 2048 MMA cycles, against 128 elements per thread
// of four FP32 operations each (in packed pairs), so the reductions hide behind
// the MMAs.  The register split is the contraction kernels' (kern_tc.cu).
constexpr int GM = 256, GN = 256, GK = 64;
constexpr int CHAIN = 256 / GK;                    // stages per accumulation chain
constexpr int A_BYTES = (GM / 2) * GK * 2, B_BYTES = (GN / 2) * GK * 2;
constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
constexpr int STAGES = 6;
constexpr int EPI_WARP0 = 4, EPI_WARPS = 8, THREADS = (EPI_WARP0 + EPI_WARPS) * 32;
constexpr int REG_LAUNCH = 168, REG_LOW = 72, REG_HIGH = 216;
static_assert(EPI_WARP0 * 32 * REG_LOW + EPI_WARPS * 32 * REG_HIGH <= THREADS * REG_LAUNCH,
              "register split exceeds the launch's registers");
constexpr size_t SMEM_BYTES = (size_t)STAGES * STAGE_BYTES + 1024 + 256;
static_assert(SMEM_BYTES <= 227 * 1024, "shared memory above the per-block limit");
constexpr uint64_t WAIT_BUDGET_NS = 2000000000ull;

struct GemmArgs {
  CUtensorMap tmA, tmB;
  int16_t* R;
  int rows, cols, ldR;         // output of one plane: rows x cols, ldR = cols rounded up to 8
  int row0;                    // first row of A
  int tiles_m, tiles_n, n_b;   // tiles and planes
  int a_planes, b_planes;      // planes of A and B (a plane index is taken modulo these)
  int set;                     // planes of a product: NPL, CPL with the magnitudes, RPL with the remainders
  int nK;                      // stages of GK
  const int* todo;             // not NULL: nothing is done where it points at 0
};

struct GemmBars {
  uint64_t full[STAGES], empty[STAGES], tfull[2], tempty[2], done;
  uint32_t tmem_base;
};
static_assert(sizeof(GemmBars) <= 256, "barriers");

// K-major tile of 128-byte rows written by TMA with 128-byte swizzling; 8-row groups 1024 bytes apart
__device__ __forceinline__ uint64_t sdesc_sw128(const void* tile) {
  const uint64_t addr = tc::smem_u32(tile);
  return ((addr >> 4) & 0x3FFFull) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) | ((uint64_t)1 << 46) |
         ((uint64_t)2 << 61);
}

// item -> (plane, tile row, tile column): planes outermost (both operand planes stay in L2), inside
// a plane groups of 8 tile rows, column by column
__device__ __forceinline__ void gemm_item(const GemmArgs& P, int item, int& b, int& tm, int& tn) {
  const int tiles = P.tiles_m * P.tiles_n;
  b = item / tiles;
  const int t = item - b * tiles;
  const int grp = t / (8 * P.tiles_n), first = grp * 8, rows = min(8, P.tiles_m - first);
  const int within = t - grp * 8 * P.tiles_n;
  tm = first + within % rows;
  tn = within / rows;
}

// the moduli; for the planes after the residues one that their sums (below 2^15) never reach
__constant__ float c_mod[mod::RPL / 2] = {509.f, 505.f, 493.f, 481.f, 461.f, 457.f, 449.f, 433.f, 421.f,
                                          409.f, 401.f, 397.f, 389.f, 0x1p20f, 0x1p20f, 0x1p20f, 0x1p20f};

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(THREADS, 1)
k_mod_gemm(const __grid_constant__ GemmArgs P, int* __restrict__ status) {
  if (P.todo && *P.todo == 0) return;   // the same for both CTAs of a pair
  extern __shared__ __align__(1024) unsigned char smem_mod[];
  unsigned char* tiles = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_mod) + 1023) & ~uintptr_t(1023));
  GemmBars* bar = reinterpret_cast<GemmBars*>(tiles + STAGES * STAGE_BYTES);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = tc::cluster_rank();
  const bool leader = rank == 0;
  const int pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
  const int nK = P.nK, n_items = P.tiles_m * P.tiles_n * P.n_b;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      tc::mbar_init(&bar->full[s], 1);
      tc::mbar_init(&bar->empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      tc::mbar_init(&bar->tfull[b], 1);
      tc::mbar_init(&bar->tempty[b], 2 * EPI_WARPS);
    }
    tc::mbar_init(&bar->done, 1);
    tc::fence_mbar_init();
    tc::prefetch_tmap(&P.tmA);
    tc::prefetch_tmap(&P.tmB);
  }
  if (warp == 1) {
    tc::tmem_alloc_pair(&bar->tmem_base, 512);
    tc::tmem_relinquish_pair();
  }
  tc::fence_before();
  __syncthreads();
  tc::cluster_sync();      // barriers of both CTAs initialised before any remote use
  tc::fence_after();
  const uint32_t tbase = bar->tmem_base;

  if (warp < EPI_WARP0) {
    tc::setmaxnreg_dec<REG_LOW>();
    if (warp == 0) {
      if (lane == 0) {
        // ---------------- TMA producer (both CTAs) ----------------
        int64_t gs = 0;
        int slot = 0;
        uint32_t ph = 0;
        bool ok = true;
        for (int item = pair; item < n_items && ok; item += npairs) {
          int b, tm, tn;
          gemm_item(P, item, b, tm, tn);
          const int arow = P.row0 + tm * GM + (int)rank * (GM / 2), brow = tn * GN + (int)rank * (GN / 2);
          const int pa = b % P.a_planes, pb = b % P.b_planes;
          for (int kc = 0; kc < nK; ++kc, ++gs) {
            const int s = slot;
            if (!tc::mbar_wait(&bar->empty[s], ph ^ 1u, status, 1, WAIT_BUDGET_NS)) { ok = false; break; }
            if (++slot == STAGES) {
              slot = 0;
              ph ^= 1u;
            }
            // the first CTA's barrier counts the loads of both CTAs
            if (leader) tc::mbar_arrive_expect_tx(&bar->full[s], 2 * STAGE_BYTES);
            const uint32_t fb = tc::mapa(&bar->full[s], 0);
            unsigned char* st = tiles + (size_t)s * STAGE_BYTES;
            tc::tma_load_3d_pair(st, &P.tmA, fb, kc * GK, arow, pa);
            tc::tma_load_3d_pair(st + A_BYTES, &P.tmB, fb, kc * GK, brow, pb);
          }
        }
        // copies of this CTA still in flight land before it may exit
        for (int64_t g = max((int64_t)0, gs - STAGES); g < gs; ++g)
          tc::mbar_wait(&bar->empty[g % STAGES], (uint32_t)((g / STAGES) & 1), status, 1, WAIT_BUDGET_NS);
      }
    } else if (warp == 1) {
      if (lane == 0 && leader) {
        // ---------------- MMA issuer (first CTA of the pair) ----------------
        int64_t gc = 0;
        int slot = 0;
        uint32_t ph = 0;
        bool ok = true;
        constexpr uint32_t idesc = tc::idesc_f16(false, false, GM, GN);
        for (int item = pair; item < n_items && ok; item += npairs) {
          for (int kc = 0, pos = 0; kc < nK; ++kc) {
            const int buf = (int)(gc & 1);
            if (pos == 0) {
              if (!tc::mbar_wait(&bar->tempty[buf], (uint32_t)(((gc >> 1) & 1) ^ 1), status, 1, WAIT_BUDGET_NS)) {
                ok = false;
                break;
              }
              tc::fence_after();
            }
            const int s = slot;
            if (!tc::mbar_wait(&bar->full[s], ph, status, 1, WAIT_BUDGET_NS)) {
              ok = false;
              break;
            }
            if (++slot == STAGES) {
              slot = 0;
              ph ^= 1u;
            }
            tc::fence_after();
            const unsigned char* st = tiles + (size_t)s * STAGE_BYTES;
            const uint64_t da = sdesc_sw128(st), db = sdesc_sw128(st + A_BYTES);
            const uint32_t d = tbase + buf * GN;
#pragma unroll
            for (int ks = 0; ks < GK / 16; ++ks)   // a K step of 16 is 32 bytes of the row
              tc::mma_f16_pair(d, da + ks * 2, db + ks * 2, idesc, (pos > 0 || ks > 0) ? 1u : 0u);
            tc::mma_commit_pair(&bar->empty[s], 0x3);
            if (++pos == CHAIN || kc == nK - 1) {
              tc::mma_commit_pair(&bar->tfull[buf], 0x3);
              ++gc;
              pos = 0;
            }
          }
        }
        tc::mma_commit_pair(&bar->done, 0x1);
        tc::mbar_wait(&bar->done, 0, status, 1, WAIT_BUDGET_NS);
      }
    }
  } else {
    tc::setmaxnreg_inc<REG_HIGH>();
    // ---------------- epilogue (both CTAs, own 128 rows) ----------------
    const int ew = warp - EPI_WARP0, quad = warp & 3, half = ew >> 2;
    const int nch = (nK + CHAIN - 1) / CHAIN;
    int64_t gc = 0;
    bool ok = true;
    for (int item = pair; item < n_items && ok; item += npairs) {
      int b, tm, tn;
      gemm_item(P, item, b, tm, tn);
      const float m = c_mod[(b % P.set) >> 1], im = 1.0f / m;
      const uint64_t inv2 = pack2(im, im), neg2 = pack2(-m, -m);
      const uint64_t magic = pack2(12582912.f, 12582912.f), nmagic = pack2(-12582912.f, -12582912.f);
      uint64_t acc[64];
#pragma unroll
      for (int i = 0; i < 64; ++i) acc[i] = 0ull;
      for (int c = 0; c < nch; ++c, ++gc) {
        const int buf = (int)(gc & 1);
        if (!tc::mbar_wait(&bar->tfull[buf], (uint32_t)((gc >> 1) & 1), status, 1, WAIT_BUDGET_NS)) { ok = false; break; }
        tc::fence_after();
        const uint32_t ta = tbase + ((uint32_t)(quad * 32) << 16) + buf * GN + half * 128;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          float v[32];
          tc::tmem_ld32(ta + 32 * j, v);
          tc::tmem_ld_wait();
          tc::reg_after_wait(v);
          if (j == 3) {
            tc::fence_before();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive_cluster(tc::mapa(&bar->tempty[buf], 0));
          }
          // acc = (acc + x) - m round((acc + x) / m): |acc + x| <= 255^2 256 + 257 < 2^24, every step exact
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const uint64_t y = add2(acc[16 * j + i], pack2(v[2 * i], v[2 * i + 1]));
            const uint64_t t = add2(fma2(y, inv2, magic), nmagic);
            acc[16 * j + i] = fma2(t, neg2, y);
          }
        }
      }
      if (!ok) break;
      const int row = tm * GM + (int)rank * (GM / 2) + quad * 32 + lane, col = tn * GN + half * 128;
      if (row < (P.rows + 31) / 32 * 32) {
        int16_t* o = P.R + res_index(P.rows, P.ldR, b, row, col);
        // the low 16 bits of 1.5 2^23 + r are r in two's complement
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          if (col + 8 * i < P.ldR) {
            uint32_t w[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              float x, y;
              unpack2(add2(acc[4 * i + k], magic), x, y);
              w[k] = __byte_perm(__float_as_uint(x), __float_as_uint(y), 0x5410);
            }
            *reinterpret_cast<uint4*>(o + 256 * i) = make_uint4(w[0], w[1], w[2], w[3]);
          }
        }
      }
    }
  }
  tc::fence_before();
  __syncthreads();
  tc::cluster_sync();      // neither CTA leaves while the pair's MMAs may still read its operands
  tc::fence_after();
  if (warp == 1) tc::tmem_dealloc_pair(tbase, 512);
}

// ---------------------------------------------------------------------------
// reconstruction
// ---------------------------------------------------------------------------
// flags[z flag_step + tile] = 1 for the 64 x 64 tiles with an element whose S (modgemm.cuh) is below CHECK_MIN of its
// rows' norms; R holds the products z = 0 .. gridDim.z of CPL planes each.  Grid (column tiles, row tiles, products);
// tile row0 / 64 is the first of flag_cols tiles a row.  Zeros and non-finite rows raise no flag.
__global__ void __launch_bounds__(128) k_mod_check(const int16_t* __restrict__ R, int rows, int cols, int ldR, int row0,
                                                   const float* __restrict__ nA, size_t stepA,
                                                   const float* __restrict__ nB, size_t stepB, int* __restrict__ flags,
                                                   size_t flag_step) {
  const int z = blockIdx.z, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int16_t* S = R + (size_t)z * CPL * res_plane(rows, ldR);
  const float t = mod::CHECK_MIN * (float)(1 << 2 * mod::CHECK_BITS);
  bool low = false;
#pragma unroll
  for (int q = 0; q < 4; ++q) {                     // a warp reads blocks of 32 rows x 8 columns
    const int i = blockIdx.y * 64 + (q & 1) * 32 + lane, j0 = blockIdx.x * 64 + (warp + 4 * (q >> 1)) * 8;
    if (i >= rows || j0 >= cols) continue;
    const uint4 v = *reinterpret_cast<const uint4*>(S + res_index(rows, ldR, mod::CHECK_PLANE, i, j0));
    const uint32_t u[4] = {v.x, v.y, v.z, v.w};
    const float ta = t * nA[z * stepA + row0 + i];
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const float s = (float)(int16_t)(u[c >> 1] >> 16 * (c & 1));
      if (j0 + c < cols && s < ta * nB[z * stepB + j0 + c]) low = true;
    }
  }
  if (__syncthreads_or(low) && threadIdx.x == 0)
    flags[z * flag_step + (size_t)(row0 / 64 + blockIdx.y) * gridDim.x + blockIdx.x] = 1;
}

// chi[w][row0 + i][j] += the value of R's planes (w, i, j).  A warp takes 16 rows x 8
// columns (half a residue block); two neighbouring lanes share a row and take its
// even and odd columns, so that each access to chi covers whole 32-byte sectors.
// Grid (column blocks / 4, half row blocks, frequencies).  Flagged tiles are left out.
__global__ void __launch_bounds__(128) k_mod_add(const int16_t* __restrict__ R, int rows, int row0, int nG, int ldR,
                                                 const int* __restrict__ scale, int w0, const int* __restrict__ flags,
                                                 double2* __restrict__ chi) {
  const int lane = threadIdx.x & 31, w = blockIdx.z;
  const int j0 = 8 * (blockIdx.x * 4 + (threadIdx.x >> 5)), i = blockIdx.y * 16 + (lane >> 1);
  if (j0 >= nG || i >= rows) return;
  const int G = row0 + i, sa = scale[(size_t)(1 + w0 + w) * nG + G], nt = (nG + 63) / 64;
  if (flags[((size_t)(w0 + w) * nt + (G >> 6)) * nt + (j0 >> 6)]) return;
  double2* o = chi + ((size_t)(w0 + w) * nG + G) * nG + j0 + (lane & 1);
  double2 v[4];                                  // read early: the loads run beside those of the residues
#pragma unroll
  for (int c = 0; c < 4; ++c)
    if (j0 + 2 * c + (lane & 1) < nG) v[c] = o[2 * c];
  mod::Frac re[4] = {}, im[4] = {};
  gather_fractions(R + res_index(rows, ldR, w * CPL, i, j0), res_plane(rows, ldR), lane & 1 ? mod::ODD : mod::EVEN, re, im);
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const int j = j0 + 2 * c + (lane & 1);
    if (j >= nG) break;
    const int sb = scale[j];
    const bool bad = sa == mod::NO_SCALE || sb == mod::NO_SCALE;
    v[c].x += bad ? nan("") : mod::frac_value(re[c], -sa - sb);
    v[c].y += bad ? nan("") : mod::frac_value(im[c], -sa - sb);
    o[2 * c] = v[c];
  }
}

// ---------------------------------------------------------------------------
// host
// ---------------------------------------------------------------------------
PFN_cuTensorMapEncodeTiled_v12000 encoder() {
  static const PFN_cuTensorMapEncodeTiled_v12000 fn = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess) {
      cudaGetLastError();
      f = nullptr;
    }
    return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(f);
  }();
  return fn;
}

bool encode(CUtensorMap* tm, const void* base, int Kp, int rows, int planes) {
  cuuint64_t dims[3] = {(cuuint64_t)Kp, (cuuint64_t)rows, (cuuint64_t)planes};
  cuuint64_t strides[2] = {(cuuint64_t)Kp * 2, (cuuint64_t)Kp * 2 * rows};
  cuuint32_t box[3] = {GK, 128, 1}, estr[3] = {1, 1, 1};
  return encoder()(tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int64_t round64(int64_t x) { return (x + 63) / 64 * 64; }
size_t al256(size_t x) { return (x + 255) / 256 * 256; }

}  // namespace

// The register split of the kernel adds up to REG_LAUNCH per thread (see kern_tc.cu): a build with
// another count is never launched.
bool mod_gemm_usable() {
  static const bool ok = [] {
    cudaFuncAttributes a;
    if (!encoder() || cudaFuncGetAttributes(&a, k_mod_gemm) != cudaSuccess || a.numRegs != REG_LAUNCH) {
      cudaGetLastError();
      return false;
    }
    return true;
  }();
  return ok;
}

cudaError_t launch_mod_gemm(chi0_plan_s* p, const ModGemm& g, cudaStream_t s) {
  // before every launch: the attribute belongs to the current device
  const cudaError_t ea = cudaFuncSetAttribute(k_mod_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_BYTES);
  if (ea != cudaSuccess) return ea;
  GemmArgs P{};
  if (!encode(&P.tmA, g.A, g.Kp, g.rows_a, g.a_planes) || !encode(&P.tmB, g.B, g.Kp, g.cols, g.b_planes))
    return cudaErrorInvalidValue;
  P.R = g.R;
  P.rows = g.rows;
  P.cols = g.cols;
  P.ldR = g.ldR;
  P.row0 = g.row0;
  P.tiles_m = (g.rows + GM - 1) / GM;
  P.tiles_n = (g.cols + GN - 1) / GN;
  P.n_b = g.planes;
  P.a_planes = g.a_planes;
  P.b_planes = g.b_planes;
  P.set = g.set;
  P.nK = g.Kp / GK;
  P.todo = g.todo;
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const int pairs = (int)std::min<int64_t>((int64_t)P.tiles_m * P.tiles_n * P.n_b, std::max(1, nsm / 2));
  k_mod_gemm<<<2 * pairs, THREADS, SMEM_BYTES, s>>>(P, p->d_status);
  return cudaGetLastError();
}

cudaError_t launch_mod_check(const int16_t* R, int rows, int cols, int ldR, int row0, const float* nA, size_t stepA,
                             const float* nB, size_t stepB, int* flags, size_t flag_step, int products, cudaStream_t s) {
  k_mod_check<<<dim3((cols + 63) / 64, (rows + 63) / 64, products), 128, 0, s>>>(R, rows, cols, ldR, row0, nA, stepA, nB,
                                                                               stepB, flags, flag_step);
  return cudaGetLastError();
}

// Workspace of the contraction: pairs and frequencies held at a time, rows of chi0 per product
ModSizes mod_sizes(const chi0_plan_s* p, int nG) {
  constexpr int64_t kPlanes = (int64_t)4 << 30, kRes = (int64_t)4 << 30;   // operand planes, residues
  ModSizes z;
  z.ldR = (nG + 7) / 8 * 8;
  const int64_t per_pair = (int64_t)CPL * 2 * nG;
  z.Kc = (int)std::min<int64_t>({round64(p->max_pairs), std::max<int64_t>(64, kPlanes / per_pair / 64 * 64),
                                 (int64_t)65535 * PK_K});   // grid y of k_mod_pack
  // enough frequencies per launch for 40 waves of CTA pairs, within the same memory
  const int64_t tiles = (int64_t)((nG + GM - 1) / GM) * ((nG + GN - 1) / GN) * CPL;
  int64_t nw = std::min<int64_t>(p->n_freq, std::max<int64_t>(1, (40 * 76 + tiles - 1) / tiles));
  nw = std::max<int64_t>(1, std::min(nw, kPlanes / (per_pair * z.Kc)));
  nw = std::max<int64_t>(1, std::min(nw, kRes / ((int64_t)CPL * 2 * nG * z.ldR)));
  z.nw = (int)nw;
  z.rows = (int)std::min<int64_t>(nG, std::max<int64_t>(GM, kRes / ((int64_t)CPL * 2 * z.ldR * nw) / GM * GM));
  z.n_part = (z.Kc + ST_ROWS - 1) / ST_ROWS;
  const size_t nf1 = (size_t)p->n_freq + 1;
  z.off_a = al256((size_t)per_pair * z.Kc);
  z.off_r = z.off_a + al256((size_t)per_pair * z.Kc * nw);
  z.off_part = z.off_r + al256((size_t)CPL * 2 * nw * res_plane(z.rows, z.ldR));
  z.off_scale = z.off_part + al256(nf1 * z.n_part * nG * sizeof(double));
  z.off_exp = z.off_scale + al256(nf1 * nG * sizeof(int));
  z.off_norm = z.off_exp + al256((nG + nf1) * sizeof(uint32_t));
  z.off_flag = z.off_norm + al256(nf1 * nG * sizeof(float));
  const size_t nt = (nG + 63) / 64;
  z.bytes_flag = (size_t)p->n_freq * nt * nt * sizeof(int);
  z.bytes = z.off_flag + al256(z.bytes_flag);
  return z;
}

template <typename C>
static cudaError_t pack_rows(const C* X, int rows, int n, size_t ld, int Kp, int beta, int* scale, float* norm,
                             bool rest, uint16_t* planes, const int* todo, cudaStream_t s) {
  k_mod_row_scales<C><<<rows, 128, 0, s>>>(X, n, ld, beta, scale, norm, todo);
  const int64_t units = (int64_t)rows * (Kp / 64);
  auto* pack = rest ? k_mod_pack_rows<C, mod::REST> : norm ? k_mod_pack_rows<C, mod::CHECK> : k_mod_pack_rows<C, mod::PLAIN>;
  pack<<<(unsigned)((units + 7) / 8), 256, 0, s>>>(X, rows, n, ld, Kp, scale, beta, (uint32_t*)planes, todo);
  return cudaGetLastError();
}
cudaError_t launch_mod_pack_rows(const double2* X, int rows, int n, size_t ld, int Kp, bool a, int* scale, float* norm,
                                 uint16_t* planes, cudaStream_t s, const int* todo, bool rest) {
  return pack_rows(X, rows, n, ld, Kp, a ? mod::BETA_A : mod::BETA_B, scale, norm, rest, planes, todo, s);
}
cudaError_t launch_mod_pack_rows(const float2* X, int rows, int n, size_t ld, int Kp, bool a, int* scale, float* norm,
                                 uint16_t* planes, cudaStream_t s, const int* todo, bool rest) {
  return pack_rows(X, rows, n, ld, Kp, a ? mod::BETA_A : mod::BETA_B, scale, norm, rest, planes, todo, s);
}
size_t mod_cols_ws_bytes(int n, int rows) {
  return al256(sizeof(uint32_t) * rows) + sizeof(double) * ((n + ST_ROWS - 1) / ST_ROWS) * (size_t)rows;
}
cudaError_t launch_mod_pack_cols(const double2* X, int n, int rows, int Kp, bool conj, int* scale, float* norm,
                                 uint16_t* planes, void* ws, cudaStream_t s, const int* todo, bool rest) {
  uint32_t* eg = reinterpret_cast<uint32_t*>(ws);
  double* part = reinterpret_cast<double*>(reinterpret_cast<unsigned char*>(ws) + al256(sizeof(uint32_t) * rows));
  cudaError_t e = cudaMemsetAsync(eg, 0, sizeof(uint32_t) * rows, s);
  if (e != cudaSuccess) return e;
  const int n_part = (n + ST_ROWS - 1) / ST_ROWS;
  const dim3 gst((rows + ST_COLS - 1) / ST_COLS, n_part);
  k_mod_rowmax<<<gst, 256, 0, s>>>(X, rows, n, eg, todo);
  k_mod_col_norms<<<gst, 256, 0, s>>>(X, rows, n, eg, part, todo);
  k_mod_scales<<<dim3((rows + 255) / 256, 1), 256, 0, s>>>(part, n_part, rows, 0, eg, nullptr, scale, norm);
  auto* pack = rest ? k_mod_pack<mod::REST> : norm ? k_mod_pack<mod::CHECK> : k_mod_pack<mod::PLAIN>;
  pack<<<dim3((rows + PK_G - 1) / PK_G, Kp / PK_K), 256, 0, s>>>(X, rows, n, Kp, nullptr, 0, 0, scale, conj,
                                                               (uint32_t*)planes, nullptr, todo);
  return cudaGetLastError();
}

int mod_launches(const chi0_plan_s* p, int nG) {
  const ModSizes z = mod_sizes(p, nG);
  const int groups = (p->n_freq + z.nw - 1) / z.nw, panels = (nG + z.rows - 1) / z.rows;
  return 5 + groups * (1 + 3 * panels);
}

// K <= mod_sizes().Kc pairs of M with factors f [n_freq][K]
cudaError_t launch_contract_mod(chi0_plan_s* p, int nG, const double2* M, int64_t K, const double2* f, double2* chi,
                                void* ws, cudaStream_t s) {
  const ModSizes z = mod_sizes(p, nG);
  unsigned char* b = reinterpret_cast<unsigned char*>(ws);
  uint16_t* Bp = reinterpret_cast<uint16_t*>(b);
  uint16_t* Ap = reinterpret_cast<uint16_t*>(b + z.off_a);
  int16_t* R = reinterpret_cast<int16_t*>(b + z.off_r);
  double* part = reinterpret_cast<double*>(b + z.off_part);
  int* scale = reinterpret_cast<int*>(b + z.off_scale);
  uint32_t* eg = reinterpret_cast<uint32_t*>(b + z.off_exp);
  uint32_t* ef = eg + nG;
  float* norm = reinterpret_cast<float*>(b + z.off_norm);
  int* flags = reinterpret_cast<int*>(b + z.off_flag);
  const int nf = p->n_freq, Kp = (int)round64(K);
  cudaError_t e = cudaMemsetAsync(eg, 0, sizeof(uint32_t) * nG, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(flags, 0, z.bytes_flag, s);
  if (e != cudaSuccess) return e;
  const int n_part = (int)((K + ST_ROWS - 1) / ST_ROWS), nt = (nG + 63) / 64;
  const dim3 gst((nG + ST_COLS - 1) / ST_COLS, n_part);
  k_mod_fmax<<<nf, 256, 0, s>>>(f, K, ef);
  k_mod_rowmax<<<gst, 256, 0, s>>>(M, nG, K, eg, nullptr);
  k_mod_norms<<<gst, 256, 0, s>>>(M, nG, K, f, nf, eg, ef, part);
  k_mod_scales<<<dim3((nG + 255) / 256, nf + 1), 256, 0, s>>>(part, n_part, nG, nf, eg, ef, scale, norm);
  for (int w0 = 0; w0 < nf; w0 += z.nw) {
    const int nw = std::min(z.nw, nf - w0);
    k_mod_pack<mod::CHECK><<<dim3((nG + PK_G - 1) / PK_G, Kp / PK_K), 256, 0, s>>>(
        M, nG, K, Kp, f, w0, nw, scale, true, w0 == 0 ? (uint32_t*)Bp : nullptr, (uint32_t*)Ap, nullptr);
    for (int r0 = 0; r0 < nG; r0 += z.rows) {
      const int rows = std::min(z.rows, nG - r0);
      ModGemm g{Ap, Bp, R, nG, r0, rows, nG, z.ldR, Kp, CPL * nw, CPL * nw, CPL, CPL, nullptr};
      e = launch_mod_gemm(p, g, s);
      if (e != cudaSuccess) return e;
      e = launch_mod_check(R, rows, nG, z.ldR, r0, norm + (size_t)(1 + w0) * nG, nG, norm, 0,
                           flags + (size_t)w0 * nt * nt, (size_t)nt * nt, nw, s);
      if (e != cudaSuccess) return e;
      k_mod_add<<<dim3((z.ldR / 8 + 3) / 4, (rows + 15) / 16, nw), 128, 0, s>>>(R, rows, r0, nG, z.ldR, scale, w0, flags,
                                                                               chi);
    }
  }
  e = cudaGetLastError();
  return e == cudaSuccess ? launch_contract_f64(p, nG, M, K, f, chi, s, flags) : e;
}

}  // namespace chi0
