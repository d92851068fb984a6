// FP32 local factorizations with FP64 iterative refinement of K^+.
//
// In the FETI_MIXED_F32FACTOR form the dense local elimination of Sec. 4.3 /
// 4.4 (K_rr = L L^T with the interior columns first, the Schur complement S_i
// as its trailing block, F_i = (S_i[b',b'])^-1 through an identity
// augmentation) runs in FP32 (the batched Cholesky kernels instantiated for
// float).  The FP32 explicit operators F_i and S_i drive the inner PCG as in
// the mixed form; every FP64-accurate use of the generalized inverse (the
// dual right-hand side d~, the outer dual residual, the recovery of u_i)
// goes through K^+ refined in FP64 (classical mixed-precision iterative
// refinement, Moler 1967):
//   x = L^-T L^-1 g (FP32);  repeat: r = g - K_rr x (FP64, from the element
//   matrices);  x += L^-T L^-1 r,
// with zero on the fixing DOFs, which is K^+ g of the fixing-DOF generalized
// inverse of Sec. 5.2 ("regularization by fixing nodes").  Each FP32
// correction sweeps only the interior block of L and reaches the boundary
// block through the explicit F_i (k_kp_fwd_* / k_kp_bwd_*); the FP64
// residual is an element pass and a row pass (k_elem_kx / k_row_resid).
#include "feti_internal.h"
#include "feti_smem.h"

#include <algorithm>

namespace feti {
namespace {

constexpr int kT = 256;

// The dense local operators out of the eliminated workspace in one pass, one
// CTA per 32 x 32 tile (I, J), J <= I, of one subdomain's lower triangle: read
// once into shared memory, converted once, and written to (I, J) and mirrored to
// (J, I) of each requested layout: FP64 row-major (out64, stride m), the FP32
// copy with rows padded to 4 (out32), and the FP32 32-row lower panels of the
// symmetric apply (sym32; zero beyond the matrix).  which 0: the preconditioner
// block S_i (m = n_b' + k), which 1: F_i = minus the eliminated augmentation
// block (m = n_b').
//
// Bound by memory: 4 m^2 bytes read and 8 + 4 + 2 m^2 written per subdomain,
// with one FP64-pipe instruction (the conversion) per entry of the lower
// triangle; the sign is an integer operation.  A CTA per output tile, which
// read every tile twice and multiplied and converted every entry, took 8.4 ms
// for both operators of 1024 subdomains; this 4.8.
__device__ __forceinline__ double flip(double v, unsigned s) {
  return __hiloint2double(__double2hiint(v) ^ (int)s, __double2loint(v));
}
__device__ __forceinline__ float flip(float v, unsigned s) { return __int_as_float(__float_as_int(v) ^ (int)s); }

template <typename TS>
__global__ void __launch_bounds__(256) k_extract_tiles(const SubLayout* __restrict__ lay, int which,
                                                       const TS* __restrict__ Abase, double* __restrict__ out64,
                                                       float* __restrict__ out32, float* __restrict__ sym32) {
  const SubLayout& L = lay[blockIdx.y];
  const int m = which == 0 ? L.nbp + L.k : L.nbp;
  const int nT = (m + 31) / 32;
  int I = (int)((sqrtf(8.0f * blockIdx.x + 1.0f) - 1.0f) * 0.5f);  // row of the triangular index
  while (I * (I + 1) / 2 > (int)blockIdx.x) --I;
  while ((I + 1) * (I + 2) / 2 <= (int)blockIdx.x) ++I;
  const int J = (int)blockIdx.x - I * (I + 1) / 2;
  if (I >= nT) return;
  const size_t ld = L.ld;
  const int base = which == 0 ? L.nI : L.n;
  const unsigned sgn = which == 0 ? 0u : 0x80000000u;
  const TS* A = Abase + L.aoff + (size_t)base * ld + base;
  __shared__ TS T[32][33];
  __shared__ float T32[32][33];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;  // 8 rows per pass
  TS a[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int gr = 32 * I + ty + 8 * q, gc = 32 * J + tx;
    a[q] = (gr < m && gc < m && gc <= gr) ? A[(size_t)gr * ld + gc] : (TS)0;
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int r = ty + 8 * q;
    const TS v = flip(a[q], sgn);
    const float f = (float)v;
    if (I != J || tx <= r) {
      T[r][tx] = v;
      T32[r][tx] = f;
    }
    if (I == J && tx < r) {  // the diagonal tile is symmetric
      T[tx][r] = v;
      T32[tx][r] = f;
    }
  }
  __syncthreads();
  const int ldo = (m + 3) & ~3;
  double* o64 = out64 ? out64 + (which == 0 ? L.soff : L.foff) : nullptr;
  float* o32 = out32 ? out32 + (which == 0 ? L.soff32 : L.foff32) : nullptr;
  float* sp = sym32 ? sym32 + (which == 0 ? L.ssym32 : L.fsym32) + (size_t)512 * I * (I + 1) : nullptr;
  const int w = 32 * (I + 1);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int r = ty + 8 * q;
    const int gr = 32 * I + r, gc = 32 * J + tx;
    if (o64 && gr < m && gc < m) o64[(size_t)gr * m + gc] = (double)T[r][tx];
    if (o32 && gr < m && gc < ldo) o32[(size_t)gr * ldo + gc] = gc < m ? T32[r][tx] : 0.0f;
    if (sp) sp[(size_t)r * w + gc] = gr < m && gc < m ? T32[r][tx] : 0.0f;
  }
  if (I == J) return;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int r = ty + 8 * q;
    const int gr = 32 * J + r, gc = 32 * I + tx;
    if (o64 && gc < m) o64[(size_t)gr * m + gc] = (double)T[tx][r];
    if (o32 && gc < ldo) o32[(size_t)gr * ldo + gc] = gc < m ? T32[tx][r] : 0.0f;
  }
}

// Zeroes the part of the workspace that the assembly, the elimination and the
// extraction touch: the lower triangle, and of the augmentation rows the columns
// from n_I on.  A fill of the whole squares took 5.2 ms for 1024 subdomains,
// this 2.5.
template <typename T>
__global__ void __launch_bounds__(256) k_clear_lower(const SubLayout* __restrict__ lay, T* __restrict__ Abase) {
  const SubLayout& L = lay[blockIdx.y];
  const int i = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (i >= L.ld) return;
  T* row = Abase + L.aoff + (size_t)i * L.ld;
  for (int c = (i < L.n ? 0 : L.nI) + (threadIdx.x & 31); c <= i; c += 32) row[c] = (T)0;
}

// One FP32 correction x (+)= L^-T L^-1 r on the rows [0, n_I + n_b'), with
// the triangular sweeps confined to the interior: with K_rr = L L^T and L = [[L_II, 0], [L_bI, L_bb]] (interior rows first,
// then the boundary rows b' that are not fixing DOFs),
//   y_I = L_II^-1 r_I,   z_b = r_b - L_bI y_I,   x_b = (L_bb L_bb^T)^-1 z_b = F_i z_b,
//   x_I = L_II^-T (y_I - L_bI^T x_b),
// and F_i = S_i[b',b']^-1 is the explicit FP32 operator the PCG already
// applies.  The dependent 64-row block chains shrink from n_I + n_b' rows to
// n_I rows; the boundary panel products carry no chain.
// The sweeps in four kernels: the two triangular chains over L_II run one
// CTA per subdomain (k_kp_fwd_interior, k_kp_bwd_interior: 64-row blocks one
// after another), and the two products with L_bI, which carry no chain and
// hold most of the factor's bytes, run many CTAs per subdomain
// (k_kp_fwd_boundary: 32 boundary rows per CTA; k_kp_bwd_boundary: 32
// interior columns per CTA).  T is the factor's precision; every kernel reads
// the compact interior factor (rows [0, n_I + n_b') x columns [0, n_I) at
// L.loff, row stride kp_ld).
template <typename T>
__device__ __forceinline__ T kp_warp_sum(T v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// The diagonal blocks of the compact factor are stored inverted: rows and
// columns [64 b, 64 b + 64) of L_II hold W_b = L_bb^-1 (k_tcc_diag), so a block's
// solve is a product over all threads.  A substitution by one warp costs a
// division and a product in a row for each of its columns, every one of them
// some 65 clocks of issue in FP64: 27 us per 32 columns, 0.55 ms for the 640
// interior DOFs of a sub-cube, where the whole sweep is 0.05 ms of FP64 issue.
constexpr int kKB = kCholPanel;  // block of the sweeps

// Sixteen consecutive entries at p (16-byte aligned), the first n of them.
__device__ __forceinline__ void load16(const float* __restrict__ p, int n, float (&a)[16]) {
  if (n >= 16) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const float4 v = __ldg(reinterpret_cast<const float4*>(p) + u);
      a[4 * u] = v.x, a[4 * u + 1] = v.y, a[4 * u + 2] = v.z, a[4 * u + 3] = v.w;
    }
  } else {
#pragma unroll
    for (int u = 0; u < 16; ++u) a[u] = u < n ? __ldg(p + u) : 0.0f;
  }
}
__device__ __forceinline__ void load16(const double* __restrict__ p, int n, double (&a)[16]) {
  if (n >= 16) {
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const double2 v = __ldg(reinterpret_cast<const double2*>(p) + u);
      a[2 * u] = v.x, a[2 * u + 1] = v.y;
    }
  } else {
#pragma unroll
    for (int u = 0; u < 16; ++u) a[u] = u < n ? __ldg(p + u) : 0.0;
  }
}
// sum over the four lanes of a row
template <typename T>
__device__ __forceinline__ T quad_sum(T v) {
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  return v + __shfl_xor_sync(0xffffffffu, v, 2);
}

// y_I = L_II^-1 r_I (into yI at the subdomain's local offset), right-looking
// by 64-column blocks, four threads per row (16 columns each): y_b = W_b r_b,
// then the rows below are updated with it.  The next block's W and the first
// rows to update are fetched before they are needed.
template <typename T>
__global__ void __launch_bounds__(kT, sizeof(T) == 4 ? 5 : 3)
    k_kp_fwd_interior(const SubLayout* __restrict__ lay, const T* __restrict__ Lbase, const double* __restrict__ rbase,
                      T* __restrict__ yIbase) {
  extern __shared__ __align__(16) unsigned char kp_smem[];
  T* ys = reinterpret_cast<T*>(kp_smem);  // [nI rounded up to 64], zero beyond nI
  const SubLayout L = lay[blockIdx.x];
  const T* A = Lbase + L.loff;
  const size_t ld = kp_ld(L);
  const double* r = rbase + L.voff;
  const int nI = L.nI;
  const int tid = threadIdx.x, row = tid >> 2, c = 16 * (tid & 3);
  T w[16], a[16];
  // entries [row i, columns I0 + c ..), the columns up to `end`
  auto fetch = [&](T (&v)[16], int i, int I0, int end) {
    load16(A + (size_t)min(i, nI - 1) * ld + I0 + c, i < nI ? end - I0 - c : 0, v);
  };
  if (nI > 0) fetch(w, row, 0, nI);
  for (int i = tid; i < (nI + kKB - 1) / kKB * kKB; i += kT) ys[i] = i < nI ? (T)r[i] : (T)0;
  __syncthreads();
  for (int I0 = 0; I0 < nI; I0 += kKB) {
    const int I1 = I0 + kKB;
    T acc = 0;
#pragma unroll
    for (int u = 0; u < 16; ++u) acc += w[u] * ys[I0 + c + u];
    acc = quad_sum(acc);
    const bool more = I1 < nI;  // then the block is whole
    if (more) fetch(a, I1 + row, I0, I1);
    __syncthreads();
    if (c == 0) ys[I0 + row] = acc;  // rows beyond nI: zero
    if (more) fetch(w, I1 + row, I1, nI);
    __syncthreads();
    if (!more) break;
    const T* xs = ys + I0 + c;
    for (int i = I1 + row;; i += kKB) {
      T t = 0;
#pragma unroll
      for (int u = 0; u < 16; ++u) t += a[u] * xs[u];
      t = quad_sum(t);
      if (c == 0 && i < nI) ys[i] -= t;
      if (i - row + kKB >= nI) break;
      fetch(a, i + kKB, I0, I1);
    }
    __syncthreads();
  }
  T* yI = yIbase + L.voff;
  for (int i = tid; i < nI; i += kT) yI[i] = ys[i];
}

// z_b = r_b - L_bI y_I for 32 boundary rows per CTA (grid.x over row blocks,
// grid.y over subdomains; warp w takes rows w, w + 8, w + 16, w + 24 of the
// block, four column strides at a time); the CTA with block 0 also zeros z on
// the fixing positions.
template <typename T>
__global__ void __launch_bounds__(kT, sizeof(T) == 4 ? 8 : 4)
    k_kp_fwd_boundary(const SubLayout* __restrict__ lay, const T* __restrict__ Lbase, const double* __restrict__ rbase,
                      const T* __restrict__ yIbase, T* __restrict__ zb) {
  extern __shared__ __align__(16) unsigned char kp_smem[];
  T* ys = reinterpret_cast<T*>(kp_smem);
  const SubLayout L = lay[blockIdx.y];
  const int nI = L.nI, nbp = L.nbp;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int kW = kT / 32;
  if (blockIdx.x == 0)
    for (int p = nbp + tid; p < nbp + L.k; p += kT) zb[L.boff + p] = (T)0;
  const int p0 = blockIdx.x * 32;
  if (p0 >= nbp) return;
  const T* yI = yIbase + L.voff;
  for (int i = tid; i < nI; i += kT) ys[i] = yI[i];
  __syncthreads();
  const size_t ld = kp_ld(L);
  const T* rp = Lbase + L.loff + (size_t)(nI + p0) * ld;
  const double* r = rbase + L.voff;
  int ro[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) ro[q] = min(warp + kW * q, nbp - 1 - p0) * (int)ld;
  T acc[4] = {0, 0, 0, 0};
  int j = lane;
  for (; j + 96 < nI; j += 128) {
    T a[4][4];
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int u = 0; u < 4; ++u) a[q][u] = __ldg(rp + ro[q] + j + 32 * u);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const T yv = ys[j + 32 * u];
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[q] += a[q][u] * yv;
    }
  }
  for (; j < nI; j += 32) {
    const T yv = ys[j];
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[q] += __ldg(rp + ro[q] + j) * yv;
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const T v = kp_warp_sum(acc[q]);
    const int p = p0 + warp + kW * q;
    if (lane == 0 && p < min(nbp, p0 + 32)) zb[L.boff + p] = (T)(r[nI + p] - (double)v);
  }
}

// t_I = y_I - L_bI^T x_b in place in yI, 32 interior columns per CTA: lane =
// column, warp w = boundary rows w, w + 8, ..., eight rows in flight per
// thread, the eight warps' partial sums added in a fixed order.
template <typename T>
__global__ void __launch_bounds__(kT, sizeof(T) == 4 ? 8 : 4)
    k_kp_bwd_boundary(const SubLayout* __restrict__ lay, const T* __restrict__ Lbase, const double* __restrict__ xb,
                      T* __restrict__ yIbase) {
  extern __shared__ __align__(16) unsigned char kp_smem[];
  T* xbs = reinterpret_cast<T*>(kp_smem);
  const SubLayout L = lay[blockIdx.y];
  const int nI = L.nI, nbp = L.nbp;
  const int c0 = blockIdx.x * 32;
  if (c0 >= nI) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int kW = kT / 32;
  __shared__ T part[kW][32];
  for (int p = tid; p < nbp; p += kT) xbs[p] = (T)xb[L.boff + p];
  __syncthreads();
  const size_t ld = kp_ld(L);
  const int c = c0 + lane;
  const T* col = Lbase + L.loff + (size_t)nI * ld + min(c, nI - 1);
  T acc = 0;
  int p = warp;
  for (; p + 7 * kW < nbp; p += 8 * kW) {
    T a[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) a[u] = __ldg(col + (size_t)(p + kW * u) * ld);
#pragma unroll
    for (int u = 0; u < 8; ++u) acc += a[u] * xbs[p + kW * u];
  }
  for (; p < nbp; p += kW) acc += __ldg(col + (size_t)p * ld) * xbs[p];
  part[warp][lane] = acc;
  __syncthreads();
  if (warp == 0 && c < nI) {
    T s = part[0][lane];
#pragma unroll
    for (int w = 1; w < kW; ++w) s += part[w][lane];
    T* yI = yIbase + L.voff;
    yI[c] -= s;
  }
}

// x_I = L_II^-T t_I (t_I in yI after k_kp_bwd_boundary), by 64-column blocks
// from the last: x_b = W_b^T t_b, then L[b, j]^T x_b is taken from every column j
// before the block; then x (+)= x on rows [0, n_I + n_b') (x_b from the F_i
// apply, FP64 at the boundary offset), and with init x = that correction,
// zero on the fixing rows.  Four threads (parts = 4) share a column, each with
// 16 of a block's rows and its own copy of the subtracted sums, added in a fixed
// order when the block is reached.  Where five interior vectors do not fit shared
// memory (parts = 0) a thread owns whole columns and subtracts from the one vector.
template <typename T>
__global__ void __launch_bounds__(kT, sizeof(T) == 4 ? 5 : 3)
    k_kp_bwd_interior(const SubLayout* __restrict__ lay, const T* __restrict__ Lbase, const T* __restrict__ yIbase,
                      const double* __restrict__ xb, double* __restrict__ xbase, int init, int parts) {
  extern __shared__ __align__(16) unsigned char kp_smem[];
  T* ys = reinterpret_cast<T*>(kp_smem);
  const SubLayout L = lay[blockIdx.x];
  const T* A = Lbase + L.loff;
  const size_t ld = kp_ld(L);
  double* x = xbase + L.voff;
  const int nI = L.nI, nbp = L.nbp;
  const int nIp = (nI + kKB - 1) / kKB * kKB;
  T* sub = ys + nIp;  // [parts][nIp]
  const int np = max(parts, 1);
  const int tid = threadIdx.x;
  __shared__ T ts[kKB], ps[4][kKB];
  const int wj = tid & 63, wi = 16 * (tid >> 6);
  T w[16];
  auto fetch_w = [&](int I0) {  // rows wi .., column wj of W_b
#pragma unroll
    for (int u = 0; u < 16; ++u) {
      const int i = I0 + wi + u;
      w[u] = (i < nI && wj <= wi + u) ? __ldg(A + (size_t)i * ld + I0 + wj) : (T)0;
    }
  };
  if (nI > 0) fetch_w(nIp - kKB);
  const T* yI = yIbase + L.voff;
  for (int i = tid; i < nIp; i += kT) ys[i] = i < nI ? yI[i] : (T)0;
  for (int i = tid; i < parts * nIp; i += kT) sub[i] = (T)0;
  __syncthreads();
  const int per = kT / np, col = tid % per, rows = kKB / np, i0 = (tid / per) * rows;
  T* mine = sub + (size_t)(tid / per) * nIp;
  for (int I0 = nIp - kKB; I0 >= 0; I0 -= kKB) {
    if (tid < kKB) {
      T t = ys[I0 + tid];
      for (int k = 0; k < parts; ++k) t -= sub[(size_t)k * nIp + I0 + tid];
      ts[tid] = t;
    }
    __syncthreads();
    T acc = 0;
#pragma unroll
    for (int u = 0; u < 16; ++u) acc += w[u] * ts[wi + u];
    ps[tid >> 6][wj] = acc;
    if (I0 > 0) fetch_w(I0 - kKB);
    __syncthreads();
    if (tid < kKB) ys[I0 + tid] = (ps[0][tid] + ps[1][tid]) + (ps[2][tid] + ps[3][tid]);
    __syncthreads();
    const T* blk = A + (size_t)I0 * ld;
    for (int j = col; j < I0; j += per) {
      T t = 0;
      for (int h = i0; h < i0 + rows; h += 16) {
        T a[16];
#pragma unroll
        for (int u = 0; u < 16; ++u) a[u] = I0 + h + u < nI ? __ldg(blk + (size_t)(h + u) * ld + j) : (T)0;
#pragma unroll
        for (int u = 0; u < 16; ++u) t += a[u] * ys[I0 + h + u];
      }
      if (parts)
        mine[j] += t;
      else
        ys[j] -= t;
    }
    __syncthreads();
  }
  for (int i = tid; i < nI; i += kT) x[i] = (init ? 0.0 : x[i]) + (double)ys[i];
  for (int p = tid; p < nbp; p += kT) x[nI + p] = (init ? 0.0 : x[nI + p]) + xb[L.boff + p];
  if (init)
    for (int i = nI + nbp + tid; i < L.n; i += kT) x[i] = 0.0;
}

// Compact interior factor: one CTA per 32 rows of one subdomain, a warp per
// row, lanes along the columns (coalesced on both sides).
template <typename T>
__global__ void __launch_bounds__(256) k_compact_factor(const SubLayout* __restrict__ lay, const T* __restrict__ Abase,
                                                        T* __restrict__ Lbase) {
  const SubLayout L = lay[blockIdx.y];
  const int rows = L.nI + L.nbp;
  const int r0 = blockIdx.x * 32;
  if (r0 >= rows) return;
  const int ldo = kp_ld(L);
  const size_t ld = L.ld;
  const T* A = Abase + L.aoff;
  T* out = Lbase + L.loff;
  for (int r = r0 + (threadIdx.x >> 5); r < min(r0 + 32, rows); r += 8) {
    const int cmax = r < L.nI ? r : L.nI - 1;  // L_II lower triangle, L_bI whole rows
    for (int c = threadIdx.x & 31; c < ldo; c += 32)
      out[(size_t)r * ldo + c] = c <= cmax ? A[(size_t)r * ld + c] : (T)0;
  }
}

// r = g - K_rr x in FP64 on the rows [0, n_I + n_b') (zero on the fixing
// rows), in two deterministic passes: ye[nde e + a] = (K_e x_e)_a
// for every element (its dense map and the local vector of its subdomain,
// columns of eliminated DOFs skipped), then per local row r = g - the sum of
// its (element, row) entries in the order of its incidence list.
template <int NDE>
__global__ void __launch_bounds__(128) k_elem_kx(int n_el, const int32_t* __restrict__ elem_sub,
                                                 const SubLayout* __restrict__ lay,
                                                 const int32_t* __restrict__ elem_dense, const double* __restrict__ Ke,
                                                 const double* __restrict__ xbase, double* __restrict__ ye) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n_el) return;
  const double* x = xbase + lay[elem_sub[e]].voff;
  const int32_t* dm = elem_dense + (size_t)NDE * e;
  const double* ke = Ke + (size_t)e * ke_packed(NDE);
  double xe[NDE];
#pragma unroll
  for (int b = 0; b < NDE; ++b) {
    const int c = dm[b];
    xe[b] = c >= 0 ? x[c] : 0.0;
  }
  // K_e maps a translation to zero, so node 0's value is taken from the others
  // (9 x 9 of the 12 x 12 products, 45 of the 78 entries read: the packed tail)
  // and its rows are minus the sums of theirs.  Bound by the FP64 pipe: solve of
  // 1024 subdomains with FP32 factors (28 calls) 177.1 -> 174.2 ms.
  double y0[3] = {0.0, 0.0, 0.0};
#pragma unroll
  for (int b = 3; b < NDE; ++b) xe[b] -= xe[b % 3];
#pragma unroll
  for (int a = 3; a < NDE; ++a) {
    double t = 0.0;
#pragma unroll
    for (int b = 3; b < NDE; ++b) t += ke[ke_idx(NDE, a, b)] * xe[b];
    ye[(size_t)NDE * e + a] = t;
    y0[a % 3] -= t;
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) ye[(size_t)NDE * e + a] = y0[a];
}

__global__ void k_row_resid(int n, const int32_t* __restrict__ row_sub, const SubLayout* __restrict__ lay,
                            const int32_t* __restrict__ kinc_ptr, const int32_t* __restrict__ kinc,
                            const double* __restrict__ ye, const double* __restrict__ g, double* __restrict__ r) {
  for (int gi = blockIdx.x * blockDim.x + threadIdx.x; gi < n; gi += gridDim.x * blockDim.x) {
    const SubLayout L = lay[row_sub[gi]];
    double acc = 0.0;
    if (gi - L.voff < L.nI + L.nbp) {
      acc = g[gi];
      const int q1 = kinc_ptr[gi + 1];
      int q = kinc_ptr[gi];
      for (; q + 4 <= q1; q += 4) {
        const int e0 = kinc[q], e1 = kinc[q + 1], e2 = kinc[q + 2], e3 = kinc[q + 3];
        const double v0 = ye[e0], v1 = ye[e1], v2 = ye[e2], v3 = ye[e3];
        acc -= v0;
        acc -= v1;
        acc -= v2;
        acc -= v3;
      }
      for (; q < q1; ++q) acc -= ye[kinc[q]];
    }
    r[gi] = acc;
  }
}

// out (full local vectors) = the boundary vector loc at the boundary
// positions [nI, n), zero on the interior.
__global__ void k_place(const SubLayout* __restrict__ lay, const double* __restrict__ loc, double* __restrict__ out,
                        const int* __restrict__ done) {
  if (done && *done) return;
  const SubLayout L = lay[blockIdx.x];
  for (int i = threadIdx.x; i < L.n; i += blockDim.x)
    out[L.voff + i] = i < L.nI ? 0.0 : loc[L.boff + i - L.nI];
}

// Per subdomain: out[2 s] = sum of r_i^2, out[2 s + 1] = sum of g_i^2 over [0, nr).
__global__ void k_sub_norm2(const SubLayout* __restrict__ lay, const double* __restrict__ r,
                            const double* __restrict__ g, double* __restrict__ out) {
  const SubLayout L = lay[blockIdx.x];
  const int nr = L.nI + L.nbp;
  __shared__ double sr[kT / 32], sg[kT / 32];
  double a = 0.0, b = 0.0;
  for (int i = threadIdx.x; i < nr; i += kT) {
    a += r[L.voff + i] * r[L.voff + i];
    b += g[L.voff + i] * g[L.voff + i];
  }
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
  }
  if ((threadIdx.x & 31) == 0) {
    sr[threadIdx.x >> 5] = a;
    sg[threadIdx.x >> 5] = b;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double ta = 0.0, tb = 0.0;
    for (int w = 0; w < kT / 32; ++w) {
      ta += sr[w];
      tb += sg[w];
    }
    out[2 * blockIdx.x] = ta;
    out[2 * blockIdx.x + 1] = tb;
  }
}

// Deterministic test vector in [-1, 1) from a 64-bit mix of the index
// (splitmix64 finaliser).
__global__ void k_fill_mix(long n, double* __restrict__ x) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
    unsigned long long z = (unsigned long long)i + 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    x[i] = (double)(z >> 11) * (2.0 / 9007199254740992.0) - 1.0;
  }
}

}  // namespace

void launch_clear_lower(int P, int max_ld, const SubLayout* lay, double* A, cudaStream_t st) {
  if (P > 0 && max_ld > 0) k_clear_lower<double><<<dim3((max_ld + 7) / 8, P), 256, 0, st>>>(lay, A);
}

void launch_clear_lower(int P, int max_ld, const SubLayout* lay, float* A, cudaStream_t st) {
  if (P > 0 && max_ld > 0) k_clear_lower<float><<<dim3((max_ld + 7) / 8, P), 256, 0, st>>>(lay, A);
}

void launch_extract_tiles(int P, int max_m, const SubLayout* lay, int which, const float* A, double* out64, float* out32,
                          float* sym32, cudaStream_t st) {
  const int nT = (max_m + 31) / 32;
  if (P > 0 && nT > 0) k_extract_tiles<float><<<dim3(nT * (nT + 1) / 2, P), 256, 0, st>>>(lay, which, A, out64, out32, sym32);
}

void launch_extract_tiles(int P, int max_m, const SubLayout* lay, int which, const double* A, double* out64,
                          float* out32, float* sym32, cudaStream_t st) {
  const int nT = (max_m + 31) / 32;
  if (P > 0 && nT > 0) k_extract_tiles<double><<<dim3(nT * (nT + 1) / 2, P), 256, 0, st>>>(lay, which, A, out64, out32, sym32);
}

template <typename T>
void kp_forward(int P, const SubLayout* lay, const T* Lc, const double* r, T* yI, T* zb, int max_nr, int max_nI, cudaStream_t st) {
  if (P <= 0) return;
  const size_t smem = (size_t)std::max(max_nr, 1) * sizeof(T);
  const size_t smem_int = (size_t)(std::max(max_nI, 1) + kKB - 1) / kKB * kKB * sizeof(T);
  (void)allow_smem(k_kp_fwd_interior<T>, smem_int);
  (void)allow_smem(k_kp_fwd_boundary<T>, smem);
  k_kp_fwd_interior<T><<<P, kT, smem_int, st>>>(lay, Lc, r, yI);
  const int nblk = std::max(1, (max_nr + 31) / 32);
  k_kp_fwd_boundary<T><<<dim3(nblk, P), kT, smem, st>>>(lay, Lc, r, yI, zb);
}

template <typename T>
void kp_backward(int P, const SubLayout* lay, const T* Lc, T* yI, const double* xb, double* x, int init,
                 int max_nr, int max_nI, cudaStream_t st) {
  if (P <= 0) return;
  const size_t smem = (size_t)std::max(max_nr, 1) * sizeof(T);
  const size_t row = (size_t)(std::max(max_nI, 1) + kKB - 1) / kKB * kKB * sizeof(T);
  const int parts = 5 * row <= 200 * 1024 ? 4 : 0;
  (void)allow_smem(k_kp_bwd_boundary<T>, smem);
  (void)allow_smem(k_kp_bwd_interior<T>, (1 + parts) * row);
  const int nblk = std::max(1, (max_nr + 31) / 32);
  k_kp_bwd_boundary<T><<<dim3(nblk, P), kT, smem, st>>>(lay, Lc, xb, yI);
  k_kp_bwd_interior<T><<<P, kT, (1 + parts) * row, st>>>(lay, Lc, yI, xb, x, init, parts);
}

void launch_kp_forward(int P, const SubLayout* lay, const float* Lc, const double* r, float* yI, float* zb, int max_nr,
                       int max_nI, cudaStream_t st) {
  kp_forward<float>(P, lay, Lc, r, yI, zb, max_nr, max_nI, st);
}

void launch_kp_backward(int P, const SubLayout* lay, const float* Lc, float* yI, const double* xb, double* x,
                        int init, int max_nr, int max_nI, cudaStream_t st) {
  kp_backward<float>(P, lay, Lc, yI, xb, x, init, max_nr, max_nI, st);
}

void launch_kp_forward(int P, const SubLayout* lay, const double* Lc, const double* r, double* yI, double* zb,
                       int max_nr, int max_nI, cudaStream_t st) {
  kp_forward<double>(P, lay, Lc, r, yI, zb, max_nr, max_nI, st);
}

void launch_kp_backward(int P, const SubLayout* lay, const double* Lc, double* yI, const double* xb, double* x,
                        int init, int max_nr, int max_nI, cudaStream_t st) {
  kp_backward<double>(P, lay, Lc, yI, xb, x, init, max_nr, max_nI, st);
}

void launch_compact_factor(int P, int max_rows, const SubLayout* lay, const double* A, double* Lc, cudaStream_t st) {
  const int nt = (max_rows + 31) / 32;
  if (P > 0 && nt > 0) k_compact_factor<double><<<dim3(nt, P), 256, 0, st>>>(lay, A, Lc);
}

void launch_compact_factor(int P, int max_rows, const SubLayout* lay, const float* A, float* Lc, cudaStream_t st) {
  const int nt = (max_rows + 31) / 32;
  if (P > 0 && nt > 0) k_compact_factor<float><<<dim3(nt, P), 256, 0, st>>>(lay, A, Lc);
}

void launch_kresid2(int n_el, int nde, const int32_t* elem_sub, const int32_t* row_sub, int n_rows, const SubLayout* lay,
                    const int32_t* kinc_ptr, const int32_t* kinc, const int32_t* elem_dense, const double* Ke,
                    const double* g, const double* x, double* ye, double* r, cudaStream_t st) {
  if (n_el > 0) {
    if (nde == 30)
      k_elem_kx<30><<<(n_el + 127) / 128, 128, 0, st>>>(n_el, elem_sub, lay, elem_dense, Ke, x, ye);
    else
      k_elem_kx<12><<<(n_el + 127) / 128, 128, 0, st>>>(n_el, elem_sub, lay, elem_dense, Ke, x, ye);
  }
  long b = ((long)n_rows + kT - 1) / kT;
  if (b > 65535) b = 65535;
  if (n_rows > 0) k_row_resid<<<(int)b, kT, 0, st>>>(n_rows, row_sub, lay, kinc_ptr, kinc, ye, g, r);
}

void launch_place(int P, const SubLayout* lay, const double* loc, double* out, cudaStream_t st, const int* done) {
  k_place<<<P, kT, 0, st>>>(lay, loc, out, done);
}

void launch_sub_norm2(int P, const SubLayout* lay, const double* r, const double* g, double* out, cudaStream_t st) {
  k_sub_norm2<<<P, kT, 0, st>>>(lay, r, g, out);
}

void launch_fill_mix(long n, double* x, cudaStream_t st) {
  if (n <= 0) return;
  k_fill_mix<<<(unsigned)std::min<long>((n + kT - 1) / kT, 4096), kT, 0, st>>>(n, x);
}

}  // namespace feti
