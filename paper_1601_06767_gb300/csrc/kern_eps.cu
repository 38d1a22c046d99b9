// RPA dielectric matrix from chi0 and its inverse (section II: eps = 1 - v chi0,
// W = eps^-1 v; Table III: eps_inf = 1 / [eps^-1]_00).
//
// eps[w] = I - diag(v) chi0[w]  or the symmetrised  I - diag(v^1/2) chi0[w] diag(v^1/2).
//
// Inverse: blocked Gauss-Jordan elimination with partial pivoting, in place, on
// all n_freq matrices at once (grid dimension z / x = frequency).  For each
// panel of NB columns C1 = [k0, k0 + kb):
//   1. pivot rows among rows >= k0 by tournament pivoting (k_tp_select: GEPP
//      on blocks of candidate rows in shared memory, winners merged level by
//      level); k_tp_final moves the winners to R1 = [k0, k0 + kb) (recorded as
//      a swap sequence), copies the panel columns of every row to Z and forms
//      T = A11^-1 by Gauss-Jordan with partial pivoting on the pivot block;
//   2. k_gj_rows: apply the row swaps to the other columns and replace the
//      pivot rows R1 = [k0, k0 + kb) there by T A10;
//   3. k_gj_update: every other row i: A[i][j] = A[i][j] - Z[i] . R[:, j] for
//      j outside C1 and -Z[i] . T[:, j] inside C1 (R = the new pivot rows),
//      the block sweep  A00 -= A01 T A10,  A01 = -A01 T,  A10 = T A10,  A11 = T.
// After the last panel the in-place result is (P A)^-1; k_gj_colperm applies
// the column swaps in reverse order to give A^-1.
#include <cuda_runtime.h>

#include <algorithm>

#include "cplx.cuh"
#include "internal.h"
#include "modgemm.cuh"

namespace chi0 {
namespace {

constexpr int NB = 32;          // panel width
constexpr int SINGULAR_BIT = 0x100;

template <typename C> __device__ __forceinline__ C csub(C a, C b) {
  a.x -= b.x;
  a.y -= b.y;
  return a;
}
template <typename C> __device__ __forceinline__ C crecip(C a) {
  const auto d = fma(a.x, a.x, a.y * a.y);
  C r;
  r.x = a.x / d;
  r.y = -a.y / d;
  return r;
}
template <typename C> __device__ __forceinline__ auto cabs1(C a) -> decltype(a.x) { return fabs(a.x) + fabs(a.y); }

// A CTA takes 256 columns of EPS_ROWS rows of one matrix; the square roots of its rows
// and columns are taken once (per element they and a 64-bit division cost 1.95 ms for
// 9 x 2500^2 on the FP64 pipe, against 0.27 ms for the bytes).
constexpr int EPS_ROWS = 32;
__global__ void __launch_bounds__(256) k_epsilon(const double2* __restrict__ chi, const double* __restrict__ v,
                                                 int symmetric, int nG, double2* __restrict__ eps) {
  __shared__ double vr[EPS_ROWS];
  const int j = blockIdx.x * 256 + threadIdx.x, i0 = blockIdx.y * EPS_ROWS, rows = min(EPS_ROWS, nG - i0);
  if (threadIdx.x < rows) vr[threadIdx.x] = symmetric ? sqrt(v[i0 + threadIdx.x]) : v[i0 + threadIdx.x];
  __syncthreads();
  if (j >= nG) return;
  const double vj = symmetric ? sqrt(v[j]) : 1.0;
  const size_t base = ((size_t)blockIdx.z * nG + i0) * nG + j;
#pragma unroll 4
  for (int r = 0; r < rows; ++r) {
    const double s = vr[r] * vj;
    const double2 c = chi[base + (size_t)r * nG];
    eps[base + (size_t)r * nG] = make_double2((i0 + r == j ? 1.0 : 0.0) - s * c.x, -s * c.y);
  }
}

__global__ void k_to_c64(const double2* __restrict__ a, int64_t n, float2* __restrict__ b) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
    b[e] = make_float2((float)a[e].x, (float)a[e].y);
}
__global__ void k_from_c64(const float2* __restrict__ b, int64_t n, double2* __restrict__ a) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
    a[e] = make_double2((double)b[e].x, (double)b[e].y);
}

// ---------------------------------------------------------------------------
// 1. panel: pivot rows by tournament (communication-avoiding) pivoting, then
//    the swaps, the Z copy and T = A11^-1
// ---------------------------------------------------------------------------
// rows of one selection block: 128 (FP32) or 64 (FP64) candidate rows in shared memory
template <typename R> struct SelRows { static constexpr int V = sizeof(R) == 4 ? 128 : 64; };

// Gaussian elimination with partial pivoting on up to ROWS candidate rows of
// the panel (their current values); the first kb pivot rows are the block's
// winners.  Leaf level (cand_in == NULL): block c holds rows k0 + c*ROWS ...;
// merge levels: block c holds entries c*ROWS ... of the previous level's list
// (NB slots per set, -1 = empty).  Writes NB slots per block to cand_out.
//
// Rows are not moved, each has a position instead (ties go to the lowest one).  Two
// barriers per column (FP64: three) and several threads per row; latency bound (33
// us a level of 128 FP32 rows with one thread per row, moved rows and four barriers;
// 61 us with the rows in registers, whose straight-line code missed the
// instruction cache).
constexpr int SEL_THREADS = 256;
template <typename R>
__global__ void __launch_bounds__(SEL_THREADS)
k_tp_select(const typename Cx<R>::T* __restrict__ A, int N, int k0, int kb, const int* __restrict__ cand_in,
            int n_in, int* __restrict__ cand_out, int ld, const int* __restrict__ skip) {
  using C = typename Cx<R>::T;
  constexpr int ROWS = SelRows<R>::V, TPR = SEL_THREADS / ROWS, NW = SEL_THREADS / 32;
  const int w = blockIdx.y, c = blockIdx.x, tid = threadIdx.x, warp = tid >> 5;
  if (skip && skip[w] == 0) return;
  const C* a = A + (size_t)w * N * N;
  __shared__ C S[ROWS][NB + 2];
  __shared__ int idx[ROWS], win[NB], wcnt[ROWS / 32];
  __shared__ ulonglong2 w_best[2][NW];             // a warp's largest key and the complement of its position
  __shared__ C s_inv[ROWS];                        // reciprocals of the candidates
  // valid rows to the front, keeping their order (deterministic ties)
  int g = -1;
  if (tid < ROWS) {
    const int e = c * ROWS + tid;
    if (cand_in == nullptr) g = k0 + e < N ? k0 + e : -1;
    else g = e < n_in ? cand_in[(size_t)w * ld + e] : -1;
  }
  const unsigned bal = __ballot_sync(0xffffffffu, g >= 0);
  if (tid < ROWS && (tid & 31) == 0) wcnt[warp] = __popc(bal);
  __syncthreads();
  int nr = 0, at = __popc(bal & ((1u << (tid & 31)) - 1u));
#pragma unroll
  for (int q = 0; q < ROWS / 32; ++q) {
    if (q < warp) at += wcnt[q];
    nr += wcnt[q];
  }
  if (g >= 0) idx[at] = g;
  __syncthreads();
#pragma unroll
  for (int q = 0; q < ROWS * NB / SEL_THREADS; ++q) {   // all loads in flight
    const int e = tid + q * SEL_THREADS, r = e / NB, t = e - r * NB;
    if (r < nr) S[r][t] = t < kb ? a[(size_t)idx[r] * N + k0 + t] : cz(C{});
  }
  __syncthreads();
  const int row = tid / TPR, sub = tid - row * TPR, steps = min(kb, nr);
  int pos = row;
  for (int j = 0; j < steps; ++j) {
    const int b = j & 1;
    // largest |re| + |im| among positions >= j, ties to the lowest position: the value's bits order
    // non-negative numbers; 0 marks a row that is no candidate
    unsigned long long key = 0;
    const bool cand = pos >= j && pos < nr;
    if (cand) {
      const C d = S[row][j];
      if constexpr (sizeof(R) == 4) key = (unsigned long long)__float_as_uint(cabs1(d)) + 1;
      else key = (unsigned long long)__double_as_longlong(cabs1(d)) + 1;
      // FP32: every candidate's reciprocal, beside the search (FP64: the pivot's alone, by one thread, after it)
      if (sizeof(R) == 4 && sub == 0) s_inv[row] = crecip(d);
    }
    unsigned long long best = key;
    if constexpr (sizeof(R) == 4) best = __reduce_max_sync(0xffffffffu, (unsigned)key);
    else
      for (int o = 16; o; o >>= 1) best = max(best, __shfl_xor_sync(0xffffffffu, best, o));
    const unsigned mp = __reduce_min_sync(0xffffffffu, (key == best && key) ? (unsigned)(pos << 8 | row) : 0xffffffffu);
    if ((tid & 31) == 0) w_best[b][warp] = make_ulonglong2(best, ~mp);
    __syncthreads();
    // the warps' answers, one per lane
    ulonglong2 top = w_best[b][tid & (NW - 1)];
    if constexpr (sizeof(R) == 4) {
      const unsigned k = (unsigned)top.x, m = __reduce_max_sync(0xffffffffu, k);
      top.y = __reduce_max_sync(0xffffffffu, k == m ? (unsigned)top.y : 0u);
    } else {
      for (int o = NW / 2; o; o >>= 1) {
        const unsigned long long ox = __shfl_xor_sync(0xffffffffu, top.x, o), oy = __shfl_xor_sync(0xffffffffu, top.y, o);
        if (ox > top.x || (ox == top.x && oy > top.y)) top = make_ulonglong2(ox, oy);
      }
    }
    // the pivot row goes to position j, the row there to the pivot's
    const unsigned pm = ~(unsigned)top.y;
    const int p = (int)(pm >> 8), pr = (int)(pm & 255u);
    if (row == pr) {
      if (sub == 0) {
        win[j] = idx[row];
        if (sizeof(R) == 8) s_inv[row] = crecip(S[row][j]);
      }
      pos = j;
    } else if (pos == j) {
      pos = p;
    }
    if (sizeof(R) == 8) __syncthreads();
    if (pos > j && pos < nr) {
      const C piv = S[pr][j];
      if (piv.x != (R)0 || piv.y != (R)0) {
        const C l = cmul(S[row][j], s_inv[pr]);
#pragma unroll 4
        for (int t = j + 1 + sub; t < kb; t += TPR) S[row][t] = csub(S[row][t], cmul(l, S[pr][t]));
      }
    }
    __syncthreads();
  }
  if (tid < NB) cand_out[(size_t)w * ld + (size_t)c * NB + tid] = (tid < steps) ? win[tid] : -1;
}

// Move the winners to rows k0..k0+kb-1 of the panel (recorded as a swap sequence in
// piv, and for k_gj_rows as the moves themselves: mv[t] = the row that comes to k0 + t,
// mv[NB + t] = where row k0 + t goes to, -1 = within the pivot rows) and invert the pivot block by Gauss-Jordan with partial pivoting in shared
// memory: T = A11^-1 (also written over the pivot block).  One CTA per matrix,
// latency bound: three barriers per column, the reciprocals taken beside the pivot
// search, the moved rows (64 at most) read and written once each, the copy of the
// panel left to k_copy_panel (2500^2 FP32: 91 us with a barrier and two memory
// round trips per swap, six barriers of 1024 threads per column and the copy by
// this one CTA; 33 us with four barriers of 1024 threads).
constexpr int FIN_THREADS = 256;
template <typename R>
__global__ void __launch_bounds__(FIN_THREADS)
k_tp_final(typename Cx<R>::T* __restrict__ A, int N, int k0, int kb, const int* __restrict__ win, int ld,
           typename Cx<R>::T* __restrict__ Tb, int* __restrict__ piv, int* __restrict__ moves,
           int* __restrict__ status, const int* __restrict__ skip) {
  using C = typename Cx<R>::T;
  const int w = blockIdx.x, tid = threadIdx.x;
  if (skip && skip[w] == 0) return;
  C* a = A + (size_t)w * N * N;
  int* pv = piv + (size_t)w * N;
  __shared__ int orig[2 * NB], cur[2 * NB], s_n;
  __shared__ C B[NB][2 * NB + 1];
  __shared__ int s_p;
  __shared__ C s_inv;
  if (tid < 32) {
    // swap sequence: step t exchanges row k0+t with the current row of winner t; (orig, cur) lists the
    // rows moved so far and where each is now, two entries per lane
    int n = 0, o0 = -1, o1 = -1, c0 = -1, c1 = -1;
    const int mywin = tid < kb ? win[(size_t)w * ld + tid] : -1;
    for (int t = 0; t < kb; ++t) {
      const int x = __shfl_sync(0xffffffffu, mywin, t), y = k0 + t;
      // position of original row x, original row at position y (each in at most one entry)
      const int px_l = (o0 == x && tid < n) ? c0 : ((o1 == x && tid + 32 < n) ? c1 : -1);
      const int oy_l = (c0 == y && tid < n) ? o0 : ((c1 == y && tid + 32 < n) ? o1 : -1);
      int px = (int)__reduce_max_sync(0xffffffffu, (unsigned)(px_l + 1)) - 1;
      int oy = (int)__reduce_max_sync(0xffffffffu, (unsigned)(oy_l + 1)) - 1;
      if (px < 0) px = x;
      if (oy < 0) oy = y;
      if (x < 0) px = y;      // fewer candidates than columns (cannot happen for kb <= N - k0)
      if (tid == 0) pv[y] = px;
      if (px != y) {
        // the row now at y (original oy) moves to px, winner x moves to y
        const bool fo = __any_sync(0xffffffffu, (o0 == oy && tid < n) || (o1 == oy && tid + 32 < n));
        const bool fx = __any_sync(0xffffffffu, (o0 == x && tid < n) || (o1 == x && tid + 32 < n));
        if (tid < n) {
          if (o0 == oy) c0 = px;
          else if (o0 == x) c0 = y;
        }
        if (tid + 32 < n) {
          if (o1 == oy) c1 = px;
          else if (o1 == x) c1 = y;
        }
        if (!fo) {
          if (n == tid) { o0 = oy; c0 = px; }
          if (n == tid + 32) { o1 = oy; c1 = px; }
          ++n;
        }
        if (!fx) {
          if (n == tid) { o0 = x; c0 = y; }
          if (n == tid + 32) { o1 = x; c1 = y; }
          ++n;
        }
      }
    }
    orig[tid] = o0;
    orig[tid + 32] = o1;
    cur[tid] = c0;
    cur[tid + 32] = c1;
    if (tid == 0) s_n = n;
  }
  __syncthreads();
  {
    // all moves at once: row orig[q] to cur[q], 32 columns each
    C u[2 * NB * 32 / FIN_THREADS];
    int* mv = moves + (size_t)w * 2 * NB;
    if (tid < 2 * NB) mv[tid] = tid < NB ? k0 + tid : -1;
#pragma unroll
    for (int x = 0; x < 2 * NB * 32 / FIN_THREADS; ++x) {
      const int q = (tid >> 5) + x * (FIN_THREADS / 32), t = tid & 31;
      u[x] = q < s_n && t < kb ? a[(size_t)orig[q] * N + k0 + t] : cz(C{});
    }
    __syncthreads();
#pragma unroll
    for (int x = 0; x < 2 * NB * 32 / FIN_THREADS; ++x) {
      const int q = (tid >> 5) + x * (FIN_THREADS / 32), t = tid & 31;
      if (q < s_n && t < kb) a[(size_t)cur[q] * N + k0 + t] = u[x];
    }
    if (tid < s_n) {
      const int o = orig[tid] - k0, c = cur[tid] - k0;
      if (c < kb) mv[c] = orig[tid];
      else if (o < kb) mv[NB + o] = cur[tid];
    }
  }
  __syncthreads();
  // [A11 | I] -> [I | A11^-1]
  for (int e = tid; e < NB * 2 * NB; e += blockDim.x) {
    const int i = e / (2 * NB), c = e - i * 2 * NB;
    C v = cz(C{});
    if (i < kb && c < kb) v = a[(size_t)(k0 + i) * N + k0 + c];
    else if (i < kb && c >= NB && c - NB == i) v.x = (R)1;
    B[i][c] = v;
  }
  __syncthreads();
  for (int j = 0; j < kb; ++j) {
    if (tid < 32) {
      const bool in = tid >= j && tid < kb;
      const C d = in ? B[tid][j] : cz(C{});
      const C inv = crecip(d);                     // of every candidate, beside the search
      int bi;
      bool none;                                   // no candidate above zero (or not a number)
      if constexpr (sizeof(R) == 4) {
        const unsigned key = in ? __float_as_uint(cabs1(d)) + 1u : 0u, m = __reduce_max_sync(0xffffffffu, key);
        bi = __ffs(__ballot_sync(0xffffffffu, key == m)) - 1;
        none = m <= 1u || m > 0x7f800001u;
      } else {
        R best = in ? cabs1(d) : (R)-1;
        bi = in ? tid : NB;
        for (int o = 16; o; o >>= 1) {
          const R ob = __shfl_xor_sync(0xffffffffu, best, o);
          const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
          if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
        }
        none = __shfl_sync(0xffffffffu, !(best > (R)0) || bi >= kb, 0);
        bi = __shfl_sync(0xffffffffu, bi, 0);
      }
      if (none) bi = j;
      if (tid == 0) {
        if (none && status) atomicOr(status, SINGULAR_BIT);
        s_p = bi;
      }
      if (tid == bi) s_inv = inv;
    }
    __syncthreads();
    const int p = s_p;
    if (tid < 2 * NB) {                            // a thread per column: swap rows j and p, scale row j
      const C u = B[j][tid], v = B[p][tid];
      if (p != j) B[p][tid] = u;
      B[j][tid] = cmul(v, s_inv);
    }
    __syncthreads();
    // eliminate column j from every other row: thread (i, c); columns up to j of the left half are
    // not read again
#pragma unroll
    for (int x = 0; x < NB * 2 * NB / FIN_THREADS; ++x) {
      const int e = tid + x * FIN_THREADS, i = e / (2 * NB), c = e - i * 2 * NB;
      if (i != j && i < kb && c > j) B[i][c] = csub(B[i][c], cmul(B[i][j], B[j][c]));
    }
    __syncthreads();
  }
  for (int e = tid; e < kb * kb; e += blockDim.x) {
    const int i = e / kb, c = e - i * kb;
    const C t = B[i][NB + c];
    Tb[(size_t)w * NB * NB + i * NB + c] = t;
    a[(size_t)(k0 + i) * N + k0 + c] = t;
  }
}

// Z = the panel's columns k0..k0+kb of every row outside the pivot rows (those are not read)
template <typename R>
__global__ void __launch_bounds__(256) k_copy_panel(const typename Cx<R>::T* __restrict__ A, int N, int k0, int kb,
                                                    typename Cx<R>::T* __restrict__ Z, const int* __restrict__ skip) {
  const int w = blockIdx.y;
  if (skip && skip[w] == 0) return;
  const int e = blockIdx.x * 256 + threadIdx.x, i = e / NB, t = e - i * NB;
  if (i < N && t < kb) Z[((size_t)w * N + i) * NB + t] = A[((size_t)w * N + i) * N + k0 + t];
}

// ---------------------------------------------------------------------------
// 2. row swaps outside the panel, pivot rows := T A10
// ---------------------------------------------------------------------------
// A CTA takes 32 columns: the pivot rows and the rows that come to them are read at
// once, the moved pivot rows written out, and four threads per column form eight
// rows of the product each (38 panels of 1200^2 FP32: 443 us with a thread per
// column doing one swap after another).
constexpr int GR_COLS = 32;
template <typename R>
__global__ void __launch_bounds__(128)
k_gj_rows(typename Cx<R>::T* __restrict__ A, int N, int k0, int kb, const typename Cx<R>::T* __restrict__ Tb,
          const int* __restrict__ moves, const int* __restrict__ skip) {
  using C = typename Cx<R>::T;
  const int w = blockIdx.y;
  if (skip && skip[w] == 0) return;
  C* a = A + (size_t)w * N * N;
  const int* mv = moves + (size_t)w * 2 * NB;
  __shared__ C ts[NB][NB];
  __shared__ C xs[NB][GR_COLS + 1];
  const int c = threadIdx.x & 31, g = threadIdx.x >> 5;
  const int j = blockIdx.x * GR_COLS + c;
  const bool in = j < N && !(j >= k0 && j < k0 + kb);
  // entries outside the kb x kb block are never written by the panel kernel: use zeros
  for (int e = threadIdx.x; e < NB * NB; e += 128) {
    const int r = e / NB, t = e - r * NB;
    ts[r][t] = (r < kb && t < kb) ? Tb[(size_t)w * NB * NB + e] : cz(C{});
  }
  C old[NB / 4], nw[NB / 4];
#pragma unroll
  for (int q = 0; q < NB / 4; ++q) {
    const int t = g + 4 * q;
    old[q] = nw[q] = cz(C{});
    if (in && t < kb) {
      old[q] = a[(size_t)(k0 + t) * N + j];
      nw[q] = a[(size_t)mv[t] * N + j];
    }
  }
#pragma unroll
  for (int q = 0; q < NB / 4; ++q) xs[g + 4 * q][c] = nw[q];
  __syncthreads();                                 // every row that moves has been read
#pragma unroll
  for (int q = 0; q < NB / 4; ++q) {
    const int t = g + 4 * q;
    if (in && t < kb) {
      const int d = mv[NB + t];
      if (d >= 0) a[(size_t)d * N + j] = old[q];
    }
  }
  if (!in) return;
#pragma unroll 2
  for (int q = 0; q < NB / 4; ++q) {
    const int i = g + 4 * q;
    if (i >= kb) break;
    C s = cz(C{});
#pragma unroll
    for (int t = 0; t < NB; ++t) cfma(s, ts[i][t], xs[t][c]);
    a[(size_t)(k0 + i) * N + j] = s;
  }
}

// ---------------------------------------------------------------------------
// 3. trailing update of all rows outside R1, columns [c0, c1) without [x0, x1)
// ---------------------------------------------------------------------------
template <int BYTES>
__device__ __forceinline__ void cp_async(void* dst, const void* src, bool ok) {
  const int n = ok ? BYTES : 0;                   // 0: fill with zeros
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
               "n"(BYTES), "r"(n)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

__device__ __forceinline__ float4 ld_early(const float2* p) {   // volatile: not moved past the products
  float4 v;
  asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
  return v;
}

// FP32 with even N (every row starts on 16 bytes): 64 x 64 output tiles, 256
// threads, four consecutive rows x two pairs of columns each.  A CTA takes one tile
// of rows and a run of `run` column tiles: Z's tile is loaded once, the pivot rows
// of the next tile are copied (asynchronously, double buffered) and the tile's own
// elements read while the products run.  Issue bound: 64 multiply-adds per step and
// thread against four 16-byte shared loads.  9 x 2500^2, 79 panels: 24.3 ms; 32.0
// ms with a CTA per tile, scalar loads and the tile's elements read after the
// products.  (Packed f32x2 multiply-adds, with operands doubled in shared memory:
// 33.4 ms, the shared-memory loads bound it.)
constexpr int UT = 64, ULD = UT + 2;
constexpr size_t UPD32_SMEM = (size_t)(NB * ULD + 2 * NB * UT) * sizeof(float2);
__global__ void __launch_bounds__(256, 2)
k_gj_update32(float2* __restrict__ A, int N, int k0, int kb, int c0, int c1, int x0, int x1, int run,
              const float2* __restrict__ Z, const int* __restrict__ skip) {
  extern __shared__ __align__(16) unsigned char smem_upd[];
  float2* rs = reinterpret_cast<float2*>(smem_upd);    // [2][NB][UT]  rs[t][col]
  float2* zs = rs + 2 * NB * UT;                       // [NB][ULD]  zs[t][row]
  const int w = blockIdx.z, tid = threadIdx.x;
  if (skip && skip[w] == 0) return;
  float2* a = A + (size_t)w * N * N;
  const float2* z = Z + (size_t)w * N * NB;
  const int i0 = blockIdx.y * UT, jt0 = blockIdx.x * run;
  const int ntile = (c1 - c0 + UT - 1) / UT, jt1 = min(ntile, jt0 + run);
  // pivot rows: a thread copies column pair 2 (tid mod 32) of rows tid / 32 + 8 q (c0 and c1 are even)
  const int pc = 2 * (tid & 31), pt = tid >> 5;
  auto load_rows = [&](int jt) {
    float2* dst = rs + (jt & 1) * NB * UT;
    const int j = c0 + jt * UT + pc;
#pragma unroll
    for (int q = 0; q < NB / 8; ++q) {
      const int t = pt + 8 * q;
      const bool ok = j < c1 && t < kb;
      cp_async<16>(dst + t * UT + pc, a + (ok ? (size_t)(k0 + t) * N + j : 0), ok);
    }
    cp_async_commit();
  };
  if (jt0 < jt1) load_rows(jt0);
  for (int e = tid; e < UT * NB; e += 256) {
    const int r = e / NB, t = e - r * NB, i = i0 + r;
    zs[t * ULD + r] = (i < N && t < kb) ? z[(size_t)i * NB + t] : make_float2(0.f, 0.f);
  }
  const int tx = tid & 15, ty = tid >> 4;
  float2* arow = a + (size_t)(i0 + 4 * ty) * N + 2 * tx;
  for (int jt = jt0; jt < jt1; ++jt) {
    const int j0 = c0 + jt * UT;
    cp_async_wait<0>();
    __syncthreads();                                   // this tile's pivot rows are there, the other buffer is free
    if (jt + 1 < jt1) load_rows(jt + 1);
    float4 base[4][2];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const int j = j0 + 2 * tx + 32 * c;
        base[r][c] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (i0 + 4 * ty + r < N && j < c1 && !(j >= k0 && j < k0 + kb)) base[r][c] = ld_early(arow + (size_t)r * N + j0 + 32 * c);
      }
    const float2* rt = rs + (jt & 1) * NB * UT + 2 * tx;
    float2 acc[4][4];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[r][c] = make_float2(0.f, 0.f);
#pragma unroll 4
    for (int t = 0; t < NB; ++t) {                     // rows t >= kb are zero
      const float4 r0 = *reinterpret_cast<const float4*>(rt + t * UT);
      const float4 r1 = *reinterpret_cast<const float4*>(rt + t * UT + 32);
      const float4 z0 = *reinterpret_cast<const float4*>(zs + t * ULD + 4 * ty);
      const float4 z1 = *reinterpret_cast<const float4*>(zs + t * ULD + 4 * ty + 2);
      const float2 rc[4] = {make_float2(r0.x, r0.y), make_float2(r0.z, r0.w), make_float2(r1.x, r1.y), make_float2(r1.z, r1.w)};
      const float2 zr[4] = {make_float2(z0.x, z0.y), make_float2(z0.z, z0.w), make_float2(z1.x, z1.y), make_float2(z1.z, z1.w)};
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) cfma(acc[r][c], zr[r], rc[c]);
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int i = i0 + 4 * ty + r;
      if (i >= N || (i >= k0 && i < k0 + kb)) continue;
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const int j = j0 + 2 * tx + 32 * c;            // x0, x1 and the panel's edges are even
        if (j >= c1 || (j >= x0 && j < x1)) continue;
        const float2 u = csub(make_float2(base[r][c].x, base[r][c].y), acc[r][2 * c]);
        const float2 v = csub(make_float2(base[r][c].z, base[r][c].w), acc[r][2 * c + 1]);
        *reinterpret_cast<float4*>(arow + (size_t)r * N + j0 + 32 * c) = make_float4(u.x, u.y, v.x, v.y);
      }
    }
  }
}

// FP64 (bound by the FP64 pipe) and FP32 with odd N: a CTA per 32 x 32 output tile, 256 threads, 2 x 2
// elements each
constexpr int UTG = 32;
template <typename C>
__global__ void __launch_bounds__(256)
k_gj_update_tile(C* __restrict__ A, int N, int k0, int kb, int c0, int c1, int x0, int x1, const C* __restrict__ Z,
                 const int* __restrict__ skip) {
  const int w = blockIdx.z;
  if (skip && skip[w] == 0) return;
  C* a = A + (size_t)w * N * N;
  const C* z = Z + (size_t)w * N * NB;
  __shared__ C zs[NB][UTG + 1];     // zs[t][row]
  __shared__ C rs[NB][UTG + 1];     // rs[t][col]
  const int i0 = blockIdx.y * UTG, j0 = c0 + blockIdx.x * UTG;
  for (int e = threadIdx.x; e < UTG * NB; e += blockDim.x) {
    const int r = e / NB, t = e - r * NB, i = i0 + r;
    zs[t][r] = (i < N && t < kb) ? z[(size_t)i * NB + t] : cz(C{});
    const int tt = e / UTG, c = e - tt * UTG, j = j0 + c;
    rs[tt][c] = (j < c1 && tt < kb) ? a[(size_t)(k0 + tt) * N + j] : cz(C{});
  }
  __syncthreads();
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  C acc[2][2] = {{cz(C{}), cz(C{})}, {cz(C{}), cz(C{})}};
  for (int t = 0; t < kb; ++t) {
    C zr[2], rc[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) zr[r] = zs[t][ty + 16 * r];
#pragma unroll
    for (int c = 0; c < 2; ++c) rc[c] = rs[t][tx + 16 * c];
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
      for (int c = 0; c < 2; ++c) cfma(acc[r][c], zr[r], rc[c]);
  }
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int i = i0 + ty + 16 * r;
    if (i >= N || (i >= k0 && i < k0 + kb)) continue;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int j = j0 + tx + 16 * c;
      if (j >= c1 || (j >= x0 && j < x1)) continue;
      C* o = a + (size_t)i * N + j;
      *o = csub((j >= k0 && j < k0 + kb) ? cz(C{}) : *o, acc[r][c]);
    }
  }
}

// ---------------------------------------------------------------------------
// 4. column swaps in reverse order: (P A)^-1 P = A^-1
// ---------------------------------------------------------------------------
template <typename R>
__global__ void k_gj_colperm(typename Cx<R>::T* __restrict__ A, int N, const int* __restrict__ piv,
                             const int* __restrict__ skip) {
  using C = typename Cx<R>::T;
  const int w = blockIdx.y;
  if (skip && skip[w] == 0) return;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  C* row = A + (size_t)w * N * N + (size_t)i * N;
  const int* pv = piv + (size_t)w * N;
  for (int k = N - 1; k >= 0; --k) {
    const int p = pv[k];
    if (p != k) {
      const C u = row[k];
      row[k] = row[p];
      row[p] = u;
    }
  }
}

// side stream and events of the look-ahead, made on first use; false inside a stream capture
bool inv_streams(chi0_plan_s* p, cudaStream_t s) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone) {
    cudaGetLastError();
    return false;
  }
  if (p->inv_state != 0) return p->inv_state > 0;
  p->inv_state = -1;
  int least = 0, greatest = 0;
  if (cudaDeviceGetStreamPriorityRange(&least, &greatest) != cudaSuccess ||
      cudaStreamCreateWithPriority(&p->inv_side, cudaStreamNonBlocking, greatest) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  for (cudaEvent_t& e : p->inv_ev)
    if (cudaEventCreateWithFlags(&e, cudaEventDisableTiming) != cudaSuccess) {
      cudaGetLastError();
      return false;
    }
  p->inv_state = 1;
  return true;
}

// candidate-list slots per matrix for an N-row panel (ping-pong pair)
template <typename R> int64_t tp_ld(int N) { return (int64_t)((N + SelRows<R>::V - 1) / SelRows<R>::V) * NB; }

// pivot search and pivot block of panel k0: Z (copy of its columns), T, piv
template <typename R>
void gj_panel(chi0_plan_s* p, typename Cx<R>::T* A, int N, int nf, int k0, void* Z, void* Tb, int* piv, int* cand,
              int* moves, int* status, const int* skip, cudaStream_t s) {
  using C = typename Cx<R>::T;
  constexpr int ROWS = SelRows<R>::V;
  const int ld = (int)tp_ld<R>(N), kb = min(NB, N - k0);
  int* cbuf[2] = {cand, cand + (size_t)nf * ld};
  // tournament: leaf blocks of ROWS rows, then merges of ROWS / NB sets until one is left
  int nblk = (N - k0 + ROWS - 1) / ROWS, levels = 1, cur = 0;
  for (int b = nblk; b > 1; b = (b * NB + ROWS - 1) / ROWS) ++levels;
  ProfScope ps(p, CHI0_K_INV_PANEL, s, levels + 2);
  k_tp_select<R><<<dim3(nblk, nf), SEL_THREADS, 0, s>>>(A, N, k0, kb, nullptr, 0, cbuf[0], ld, skip);
  while (nblk > 1) {
    const int n_in = nblk * NB;
    nblk = (n_in + ROWS - 1) / ROWS;
    k_tp_select<R><<<dim3(nblk, nf), SEL_THREADS, 0, s>>>(A, N, k0, kb, cbuf[cur], n_in, cbuf[cur ^ 1], ld, skip);
    cur ^= 1;
  }
  k_tp_final<R><<<nf, FIN_THREADS, 0, s>>>(A, N, k0, kb, cbuf[cur], ld, (C*)Tb, piv, moves, status, skip);
  k_copy_panel<R><<<dim3((N * NB + 255) / 256, nf), 256, 0, s>>>(A, N, k0, kb, (C*)Z, skip);
}

// columns [c0, c1) without [x0, x1)
template <typename R>
cudaError_t gj_update(chi0_plan_s* p, typename Cx<R>::T* A, int N, int nf, int k0, int c0, int c1, int x0, int x1,
                      const void* Z, const int* skip, cudaStream_t s) {
  using C = typename Cx<R>::T;
  const int kb = min(NB, N - k0);
  ProfScope ps(p, CHI0_K_INV_UPDATE, s, 1);
  bool wide = false;
  if constexpr (sizeof(R) == 4) {
    if (N % 2 == 0) {
      cudaError_t e = cudaFuncSetAttribute(k_gj_update32, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)UPD32_SMEM);
      if (e != cudaSuccess) return e;
      // runs of column tiles as long as eight CTAs per SM are left (two run at a time); short ones, so
      // that the panel kernels beside them find room soon
      const int rows = (N + UT - 1) / UT, cols = (c1 - c0 + UT - 1) / UT;
      int run = 4;
      while (run > 1 && (int64_t)rows * ((cols + run - 1) / run) * nf < 8 * 152) run >>= 1;
      k_gj_update32<<<dim3((cols + run - 1) / run, rows, nf), 256, UPD32_SMEM, s>>>(A, N, k0, kb, c0, c1, x0, x1, run,
                                                                                  (const C*)Z, skip);
      wide = true;
    }
  }
  if (!wide) {
    const dim3 grid((c1 - c0 + UTG - 1) / UTG, (N + UTG - 1) / UTG, nf);
    k_gj_update_tile<C><<<grid, 256, 0, s>>>(A, N, k0, kb, c0, c1, x0, x1, (const C*)Z, skip);
  }
  return cudaGetLastError();
}

// The panel of the next columns needs only their update, so that is done first and
// the panel's latency-bound kernels (pivot search, pivot block) run on a stream of
// the plan beside the update of all other columns; Z and T are double buffered.
// 9 x 2500^2 in FP32, with the copies and eps = 1 - v chi0: 49.7 -> 34.4 ms.
// Inside a stream capture everything stays on one stream.
// skip (or NULL): matrices whose entry is 0 are left alone.  status: NULL = zero pivots not recorded.
template <typename R>
cudaError_t gj_invert(chi0_plan_s* p, typename Cx<R>::T* A, int N, int nf, void* Z, void* Tb, int* piv,
                      int* cand, int* status, const int* skip, cudaStream_t s) {
  using C = typename Cx<R>::T;
  C* Zb[2] = {(C*)Z, (C*)Z + (size_t)nf * N * NB};
  C* Tbb[2] = {(C*)Tb, (C*)Tb + (size_t)nf * NB * NB};
  int* mvb[2] = {cand + (size_t)2 * nf * tp_ld<R>(N), cand + (size_t)2 * nf * tp_ld<R>(N) + (size_t)nf * 2 * NB};
  const bool look = !skip && inv_streams(p, s);
  cudaError_t e = cudaSuccess;
  gj_panel<R>(p, A, N, nf, 0, Zb[0], Tbb[0], piv, cand, mvb[0], status, skip, s);
  for (int k0 = 0, b = 0; k0 < N && e == cudaSuccess; k0 += NB, b ^= 1) {
    const int kb = min(NB, N - k0), n0 = k0 + NB, n1 = min(N, n0 + NB);
    {
      ProfScope ps(p, CHI0_K_INV_PANEL, s, 1);
      k_gj_rows<R><<<dim3((N + GR_COLS - 1) / GR_COLS, nf), 128, 0, s>>>(A, N, k0, kb, Tbb[b], mvb[b], skip);
    }
    if (n0 >= N) {
      e = gj_update<R>(p, A, N, nf, k0, 0, N, 0, 0, Zb[b], skip, s);
    } else if (!look) {
      e = gj_update<R>(p, A, N, nf, k0, 0, N, 0, 0, Zb[b], skip, s);
      if (e == cudaSuccess) gj_panel<R>(p, A, N, nf, n0, Zb[b ^ 1], Tbb[b ^ 1], piv, cand, mvb[b ^ 1], status, skip, s);
    } else {
      e = gj_update<R>(p, A, N, nf, k0, n0, n1, 0, 0, Zb[b], skip, s);
      if (e == cudaSuccess) e = cudaEventRecord(p->inv_ev[0], s);
      if (e == cudaSuccess) e = cudaStreamWaitEvent(p->inv_side, p->inv_ev[0], 0);
      if (e == cudaSuccess) gj_panel<R>(p, A, N, nf, n0, Zb[b ^ 1], Tbb[b ^ 1], piv, cand, mvb[b ^ 1], status, skip, p->inv_side);
      // joined whatever happens
      cudaEventRecord(p->inv_ev[1], p->inv_side);
      if (e == cudaSuccess) e = gj_update<R>(p, A, N, nf, k0, 0, N, n0, n1, Zb[b], skip, s);
      cudaStreamWaitEvent(s, p->inv_ev[1], 0);
    }
    if (e == cudaSuccess) e = cudaGetLastError();
  }
  if (e != cudaSuccess) return e;
  ProfScope ps(p, CHI0_K_INV_PANEL, s, 1);
  k_gj_colperm<R><<<dim3((N + 127) / 128, nf), 128, 0, s>>>(A, N, piv, skip);
  return cudaGetLastError();
}

}  // namespace

int eps_panel_width() { return NB; }

cudaError_t launch_epsilon(chi0_plan_s* p, int nG, const double2* chi, const double* v, int symmetric,
                           double2* eps, cudaStream_t s) {
  ProfScope ps(p, CHI0_K_EPS, s, 1);
  for (int w = 0; w < p->n_freq; w += 65535) {     // grid z limit
    const int nw = std::min(65535, p->n_freq - w);
    const size_t off = (size_t)w * nG * nG;
    k_epsilon<<<dim3((nG + 255) / 256, (nG + EPS_ROWS - 1) / EPS_ROWS, nw), 256, 0, s>>>(chi + off, v, symmetric, nG,
                                                                                       eps + off);
  }
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// FP64 plans: FP32 inverse refined in FP64
// ---------------------------------------------------------------------------
// The FP64 elimination is bound by the FP64 pipe (two multiply-adds per clock and SM):
// 42 ms for one 1200^2.  Here X is the FP32 inverse and every step takes
//   R = I - A X,  X += X R   (Newton; the error is squared)
// with both products exact modular ones on the tensor cores (modgemm.cuh).  A step
// with |R| <= 2^-26.5 in the Frobenius norm is a matrix's last: the error left, X R^2,
// is at most 2^-53 of X.  (A bound on the largest element alone leaves up to N^2
// times its square.)  From the second step on, the first one that may be the last, A X
// includes the first order of what its integers leave out (store_remainders): equal
// small elements of a row are all rounded one way, and a nearly singular A would
// amplify their sum (I - (1 - e) / N 11^T, N 1000, cond 40: 3.0e-14, 9.0e-16 by the
// elimination).  A matrix that has no such step within STEPS (ill conditioned
// beyond FP32, out of its range, singular, not finite) is inverted by the FP64
// elimination from A, whose kernels skip the others.
//
// All of this is done on A with its columns scaled to the same power of two, and the
// rows of the result scaled back: both exact.  The products are rounded relative to
// |row of A| |column of X|, where a graded A would lose the ratio of its columns (an
// elimination does not: it gives the same digits for any column scaling).
//
// 1200^2: 42.6 -> 7.6 ms (FP32 inverse 6.2, one matrix's latency; two steps 0.8,
// skipped kernels 0.6); 9 x 2500^2: 1047 -> 75 ms.  Against quad precision 5e-17
// (relative Frobenius, eps-like matrices; 1.8e-16 before the remainders, at 71 ms),
// 3.3e-16 by the elimination.
namespace {
constexpr int STEPS = 3;
constexpr double LAST_STEP = 1.1102230246251565e-16;            // |R|^2 = 2^-53

// cmax[w][j] = largest magnitude word of column j (cleared by the caller); a CTA takes 64 columns x 128 rows
__global__ void __launch_bounds__(256) k_ref_colmax(const double2* __restrict__ A, int N, uint32_t* __restrict__ cmax) {
  const int j = blockIdx.x * 64 + (threadIdx.x & 63), w = blockIdx.z;
  if (j >= N) return;
  const double2* a = A + (size_t)w * N * N;
  const int i1 = min(N, (int)(blockIdx.y + 1) * 128);
  uint32_t m = 0;
  for (int i = blockIdx.y * 128 + (threadIdx.x >> 6); i < i1; i += 4) {
    const double2 v = a[(size_t)i * N + j];
    m = max(m, max(mod::mag_word(v.x), mod::mag_word(v.y)));
  }
  atomicMax(cmax + (size_t)w * N + j, m);
}
// 2^-e of a column: e the exponent of its largest component (0 for zeros, subnormal and non-finite columns)
__device__ __forceinline__ double col_scale(uint32_t w) {
  return w >= 0x00100000u && w < 0x7ff00000u ? mod::pow2d(-min(mod::word_exp(w), 1022)) : 1.0;
}
// A = A diag(2^-e) in place, and its complex64 copy
__global__ void __launch_bounds__(256) k_ref_scale_cols(double2* __restrict__ A, int N, const uint32_t* __restrict__ cmax,
                                                        float2* __restrict__ a32) {
  const int j = blockIdx.x * 256 + threadIdx.x, w = blockIdx.z;
  if (j >= N) return;
  const double s = col_scale(cmax[(size_t)w * N + j]);
  const int i1 = min(N, (int)(blockIdx.y + 1) * 16);
  for (int i = blockIdx.y * 16; i < i1; ++i) {
    const size_t o = ((size_t)w * N + i) * N + j;
    const double2 v = make_double2(A[o].x * s, A[o].y * s);
    A[o] = v;
    a32[o] = make_float2((float)v.x, (float)v.y);
  }
}

__global__ void k_ref_init(int* __restrict__ todo, int nf) {
  for (int w = threadIdx.x; w < nf; w += blockDim.x) todo[w] = 1;
}

// values of the residue planes of one N x N product.  ADD = false: R = I - value and the sum of
// |R|^2 over the block's elements; true: X += value.  REST: with the remainders' planes.  A warp takes 16 rows
// x 8 columns (as k_mod_add).
template <bool ADD, bool REST = false>
__global__ void __launch_bounds__(128) k_ref_value(const int16_t* __restrict__ P, int N, int ldR,
                                                   const int* __restrict__ sA, const int* __restrict__ sB,
                                                   double2* __restrict__ out, float* __restrict__ part,
                                                   const int* __restrict__ todo) {
  if (*todo == 0) return;
  __shared__ float red[4];
  const int lane = threadIdx.x & 31;
  const int j0 = 8 * (blockIdx.x * 4 + (threadIdx.x >> 5)), i = blockIdx.y * 16 + (lane >> 1);
  float sq = 0.f;
  if (j0 < N && i < N) {
    double2* o = out + (size_t)i * N + j0 + (lane & 1);
    double2 v[4];
#pragma unroll
    for (int c = 0; c < 4; ++c)
      if (ADD && j0 + 2 * c + (lane & 1) < N) v[c] = o[2 * c];
    mod::Frac re[4] = {}, im[4] = {};
    mod::gather_fractions(P + mod::res_index(N, ldR, 0, i, j0), mod::res_plane(N, ldR), lane & 1 ? mod::ODD : mod::EVEN, re, im);
    const int sa = sA[i];
    int lr[4] = {}, li[4] = {};                    // remainders, in units of 2^(BETA_B - CHECK_BITS)
    if (REST) {
      const int16_t* r = P + mod::res_index(N, ldR, mod::NPL, i, j0);
      const int sh = (lane & 1) * 16;
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const uint4 u = *reinterpret_cast<const uint4*>(r + k * mod::res_plane(N, ldR));
        const uint32_t w[4] = {u.x, u.y, u.z, u.w};
        const int f = (k < 4 ? 1 : mod::BETA_A == mod::BETA_B + 1 ? 2 : 0) * (k == 1 || k == 5 ? -1 : 1);
#pragma unroll
        for (int c = 0; c < 4; ++c) ((k & 2) ? li : lr)[c] += f * (int16_t)(w[c] >> sh);
      }
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int j = j0 + 2 * c + (lane & 1);
      if (j >= N) break;
      const int sb = sB[j];
      const bool bad = sa == mod::NO_SCALE || sb == mod::NO_SCALE;
      const double x = bad ? nan("") : mod::frac_value(re[c], -sa - sb), y = bad ? nan("") : mod::frac_value(im[c], -sa - sb);
      double2 r = ADD ? make_double2(v[c].x + x, v[c].y + y) : make_double2((i == j ? 1.0 : 0.0) - x, -y);
      if (REST && !bad) {
        const int k = mod::BETA_B - mod::CHECK_BITS - sa - sb;
        r.x -= scalbn((double)lr[c], k);
        r.y -= scalbn((double)li[c], k);
      }
      if (!ADD) sq = fmaf((float)r.x, (float)r.x, fmaf((float)r.y, (float)r.y, sq));
      o[2 * c] = r;
    }
  }
  if (!ADD) {
    for (int o = 16; o; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
    if (lane == 0) red[threadIdx.x >> 5] = sq;
    __syncthreads();
    if (threadIdx.x == 0) part[blockIdx.y * gridDim.x + blockIdx.x] = (red[0] + red[1]) + (red[2] + red[3]);
  }
}

// after a step: the matrix is done when its R was small enough (sums in a fixed order; an infinity or a
// NaN is not small)
__global__ void __launch_bounds__(256) k_ref_decide(const float* __restrict__ part, int n, int* __restrict__ todo) {
  __shared__ double red[8];
  if (*todo == 0) return;
  double s = 0.0;
  for (int i = threadIdx.x; i < n; i += 256) s += (double)part[i];
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) s += red[w];
    if (s <= LAST_STEP) *todo = 0;
  }
}

// eps = diag(2^-e) Y of matrix blockIdx.y, Y = X where the matrix is done (todo 0), else the elimination's result in eps itself
__global__ void __launch_bounds__(256) k_ref_store(const double2* X, int N, const uint32_t* __restrict__ cmax,
                                                   double2* eps, const int* __restrict__ todo, int if_todo) {
  if ((todo[blockIdx.y] != 0) != (if_todo != 0)) return;
  X += (size_t)blockIdx.y * N * N;
  eps += (size_t)blockIdx.y * N * N;
  cmax += (size_t)blockIdx.y * N;
  for (int i = blockIdx.x; i < N; i += gridDim.x) {
    const double s = col_scale(cmax[i]);
    for (int j = threadIdx.x; j < N; j += 256) {
      const double2 v = X[(size_t)i * N + j];
      eps[(size_t)i * N + j] = make_double2(v.x * s, v.y * s);
    }
  }
}

// offsets of the refinement's workspace: FP32 copies of all matrices, then for one matrix at a time X, R,
// planes of A, planes of X rows, planes of a transposed operand, residues, scales
struct RefSizes {
  int Kp, ldR;
  size_t x, r, pa, px, pt, res, sa, sx, st, cols, todo, part, cmax, bytes;
};
dim3 ref_grid(int N) { return dim3(((N + 7) / 8 + 3) / 4, (N + 15) / 16); }   // k_ref_value
RefSizes ref_sizes(int N, int nf) {
  auto al = [](size_t v) { return (v + 255) / 256 * 256; };
  RefSizes z;
  z.Kp = (N + 63) / 64 * 64;
  z.ldR = (N + 7) / 8 * 8;
  const size_t planes = al((size_t)mod::RPL * 2 * N * z.Kp), mat = al((size_t)N * N * sizeof(double2)), sc = al((size_t)N * sizeof(int));
  z.x = al((size_t)nf * N * N * sizeof(float2));
  z.r = z.x + mat;
  z.pa = z.r + mat;
  z.px = z.pa + planes;
  z.pt = z.px + planes;
  z.res = z.pt + planes;
  z.sa = z.res + al((size_t)mod::RPL * 2 * mod::res_plane(N, z.ldR));
  z.sx = z.sa + sc;
  z.st = z.sx + sc;
  z.cols = z.st + sc;
  z.todo = z.cols + al(mod_cols_ws_bytes(N, N));
  z.part = z.todo + al((size_t)nf * sizeof(int));
  const dim3 g = ref_grid(N);
  z.cmax = z.part + al((size_t)g.x * g.y * sizeof(float));
  z.bytes = z.cmax + al((size_t)nf * N * sizeof(uint32_t));
  return z;
}

cudaError_t refined_inverse(chi0_plan_s* p, double2* eps, int N, int nf, void* Z, void* Tb, int* piv, int* cand, void* ws,
                            cudaStream_t s) {
  const RefSizes z = ref_sizes(N, nf);
  unsigned char* b = reinterpret_cast<unsigned char*>(ws);
  float2* a32 = reinterpret_cast<float2*>(b);
  double2 *X = reinterpret_cast<double2*>(b + z.x), *R = reinterpret_cast<double2*>(b + z.r);
  uint16_t *PA = (uint16_t*)(b + z.pa), *PX = (uint16_t*)(b + z.px), *PT = (uint16_t*)(b + z.pt);
  int16_t* res = (int16_t*)(b + z.res);
  int *sA = (int*)(b + z.sa), *sX = (int*)(b + z.sx), *sT = (int*)(b + z.st), *todo = (int*)(b + z.todo);
  float* part = (float*)(b + z.part);
  uint32_t* cmax = (uint32_t*)(b + z.cmax);
  const int64_t n2 = (int64_t)N * N;
  {
    ProfScope ps(p, CHI0_K_EPS, s, 3);
    k_ref_init<<<1, 128, 0, s>>>(todo, nf);
    const cudaError_t em = cudaMemsetAsync(cmax, 0, (size_t)nf * N * sizeof(uint32_t), s);
    if (em != cudaSuccess) return em;
    k_ref_colmax<<<dim3((N + 63) / 64, (N + 127) / 128, nf), 256, 0, s>>>(eps, N, cmax);
    k_ref_scale_cols<<<dim3((N + 255) / 256, (N + 15) / 16, nf), 256, 0, s>>>(eps, N, cmax, a32);
  }
  cudaError_t e = gj_invert<float>(p, a32, N, nf, Z, Tb, piv, cand, nullptr, nullptr, s);
  const dim3 gv = ref_grid(N);
  for (int w = 0; w < nf && e == cudaSuccess; ++w) {
    ProfScope ps(p, CHI0_K_INV_UPDATE, s, 4 + STEPS * 15);
    const double2* A = eps + w * n2;
    k_from_c64<<<4 * 152, 256, 0, s>>>(a32 + w * n2, n2, X);
    e = launch_mod_pack_rows(A, N, N, N, z.Kp, true, sA, nullptr, PA, s, nullptr, true);
    for (int it = 0; it < STEPS && e == cudaSuccess; ++it) {
      e = launch_mod_pack_cols(X, N, N, z.Kp, false, sT, nullptr, PT, b + z.cols, s, todo + w, it > 0);
      const int np = it ? mod::RPL : mod::NPL;
      if (e == cudaSuccess)
        e = launch_mod_gemm(p, ModGemm{PA, PT, res, N, 0, N, N, z.ldR, z.Kp, np, mod::RPL, np, np, todo + w}, s);
      auto* value = it ? k_ref_value<false, true> : k_ref_value<false, false>;
      value<<<gv, 128, 0, s>>>(res, N, z.ldR, sA, sT, R, part, todo + w);
      if (e == cudaSuccess) e = launch_mod_pack_rows(X, N, N, N, z.Kp, true, sX, nullptr, PX, s, todo + w);
      if (e == cudaSuccess) e = launch_mod_pack_cols(R, N, N, z.Kp, false, sT, nullptr, PT, b + z.cols, s, todo + w);
      if (e == cudaSuccess)
        e = launch_mod_gemm(p, ModGemm{PX, PT, res, N, 0, N, N, z.ldR, z.Kp, mod::NPL, mod::NPL, mod::NPL, mod::NPL, todo + w}, s);
      k_ref_value<true><<<gv, 128, 0, s>>>(res, N, z.ldR, sX, sT, X, nullptr, todo + w);
      if (it) k_ref_decide<<<1, 256, 0, s>>>(part, (int)(gv.x * gv.y), todo + w);
    }
    k_ref_store<<<4 * 152, 256, 0, s>>>(X, N, cmax + (size_t)w * N, eps + w * n2, todo + w, 0);
    if (e == cudaSuccess) e = cudaGetLastError();
  }
  if (e != cudaSuccess) return e;
  e = gj_invert<double>(p, eps, N, nf, Z, Tb, piv, cand, p->d_status, todo, s);
  if (e != cudaSuccess) return e;
  ProfScope ps(p, CHI0_K_EPS, s, 1);
  k_ref_store<<<dim3(4 * 152, nf), 256, 0, s>>>(eps, N, cmax, eps, todo, 1);
  return cudaGetLastError();
}
}  // namespace

// Where the refined inverse runs: FP64 plans from REF_MIN_N on, two panels (128^2: 2.5 ms by the
// elimination, 0.7 ms refined; a single panel has nothing to gain)
constexpr int REF_MIN_N = 64;
bool eps_inverse_refines(const chi0_plan_s* p, int nG) { return !is_split(p) && nG >= REF_MIN_N && mod_gemm_usable(); }

// Workspace (bytes): complex64 copy of the matrices (split plans), Z [2][nf][N][NB], T [2][nf][NB][NB],
// piv [nf][N], two candidate lists [nf][tp_ld], two lists of row moves [nf][2 NB].
size_t eps_inverse_ws_bytes(const chi0_plan_s* p, int nG, bool refined) {
  const size_t nf = (size_t)p->n_freq, c = is_split(p) ? sizeof(float2) : sizeof(double2);
  const size_t copy = is_split(p) ? nf * nG * nG * sizeof(float2) : 0;
  const size_t ld = (size_t)(is_split(p) ? tp_ld<float>(nG) : tp_ld<double>(nG));
  auto al = [](size_t x) { return (x + 255) / 256 * 256; };
  return al(copy) + al(2 * nf * nG * NB * c) + al(2 * nf * NB * NB * c) + al(nf * nG * sizeof(int)) +
         al((2 * nf * ld + 4 * NB * nf) * sizeof(int)) + (refined ? ref_sizes(nG, (int)nf).bytes : 0);
}

cudaError_t launch_epsilon_inverse(chi0_plan_s* p, int nG, double2* eps, void* ws, bool refined, cudaStream_t s) {
  const size_t nf = (size_t)p->n_freq;
  auto al = [](size_t x) { return (x + 255) / 256 * 256; };
  unsigned char* b = reinterpret_cast<unsigned char*>(ws);
  if (is_split(p)) {
    float2* a32 = reinterpret_cast<float2*>(b);
    b += al(nf * nG * nG * sizeof(float2));
    void* Z = b;
    b += al(2 * nf * nG * NB * sizeof(float2));
    void* Tb = b;
    b += al(2 * nf * NB * NB * sizeof(float2));
    int* piv = reinterpret_cast<int*>(b);
    b += al(nf * nG * sizeof(int));
    int* cand = reinterpret_cast<int*>(b);
    const int64_t n = (int64_t)nf * nG * nG;
    {
      ProfScope ps(p, CHI0_K_EPS, s, 1);
      k_to_c64<<<4 * 152, 256, 0, s>>>(eps, n, a32);
    }
    cudaError_t e = gj_invert<float>(p, a32, nG, (int)nf, Z, Tb, piv, cand, p->d_status, nullptr, s);
    if (e != cudaSuccess) return e;
    ProfScope ps(p, CHI0_K_EPS, s, 1);
    k_from_c64<<<4 * 152, 256, 0, s>>>(a32, n, eps);
    return cudaGetLastError();
  }
  void* Z = b;
  b += al(2 * nf * nG * NB * sizeof(double2));
  void* Tb = b;
  b += al(2 * nf * NB * NB * sizeof(double2));
  int* piv = reinterpret_cast<int*>(b);
  b += al(nf * nG * sizeof(int));
  int* cand = reinterpret_cast<int*>(b);
  b += al((2 * nf * tp_ld<double>(nG) + 4 * NB * nf) * sizeof(int));
  if (refined) return refined_inverse(p, eps, nG, (int)nf, Z, Tb, piv, cand, b, s);
  return gj_invert<double>(p, eps, nG, (int)nf, Z, Tb, piv, cand, p->d_status, nullptr, s);
}

}  // namespace chi0
