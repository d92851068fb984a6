// FP64 local apply y = M v of the symmetric operators F_i and S_i (Sec. 4.3 /
// 4.4) from 56-bit fixed-point copies, in 64-bit integer arithmetic.
//
// What bounds it: a dense FP64 matvec issues one FMA per entry, two per clock
// and SM here (1.21 ms for the 0.67 G entries of F on the 1024-subdomain tube,
// 86 % of that pipe), while its 2.65 GB lower triangle takes 0.39 ms from
// HBM.  Integer multiply-adds issue many times faster, so the entries are
// stored as A_ij = round(a_ij 2^(56 - e_i - e_j)), e_i half the exponent of
// row i's largest entry (|a_ij| <= sqrt(max_i max_j), so |A_ij| <= 2^56), as
// two signed 28-bit limbs; v is scaled by 2^e_j and rounded to 56 bits of the
// subdomain's largest entry.  An entry then costs three 32 x 32 + 64-bit
// multiply-adds for the row and three for the column (high x high, and the two
// cross products in a second accumulator; the low x low product is below
// 2^-58).  Integer sums are exact: the result carries the roundings of the
// operands and of the partial sums, at most (1.3 m + 80) 2^-56 2^(e_i) w with
// w = max_j 2^(e_j) |v_j|, whatever row i adds up to.  That is less than the
// error of an FP64 sum where the row meets large entries of v, and more where it
// does not (S_i with 858 rows and a vector that falls by 1e-8 across the
// subdomain: 2e-9 of |M| |v|, FP64 sums 8e-16).  So a row is kept only where
// |M| |v| is known to reach 2^-8 2^(e_i) w: by its diagonal product, by its result,
// or by the sum of |A_ij| |V_j| over its diagonal block and the 64 to 112 columns
// before it, taken from the high limbs for the tenth of the rows of S_i (a
// fortieth of F_i) that the first two leave.  The others, one row of S_i in a
// thousand in the iterations and none of F_i, are taken again as FP64 sums of
// the full matrix, like all rows of a subdomain whose vector or matrix has an
// infinite, NaN or nearly underflowing entry.  The error is then at most
// (1.3 m + 80) 2^-48 |M| |v|; the largest seen over random vectors, vectors that
// fall by 1e-8, 1e-16 and 1e-300, unit vectors and vectors of one component is 8e-14
// (m = 1125; an FP64 sum is bounded by m 2^-53 = 1.2e-13), the median 5e-16.
// The checks cost 0.7 ms of 47 on the 64-subdomain tube (187 iterations), with 2^-7
// 3 ms; without the check of the columns a solve took 142 ms instead of 74.
//
// Layout: lower block triangle in panels of 16 rows (panel I: columns
// 0 .. 16 (I + 1) - 1), a panel in tiles of 16 x 64 entries of 8 bytes, row-major
// and whole, so that a lane's loads of a tile differ by constants; zero beyond
// the matrix, the diagonal block full; what lies right of it in the last tile
// is never read.
//
// One cluster of C CTAs per subdomain (largest first), its 8 C warps take the
// panels in a snake order.  A warp sweeps its panel in tiles of 64 columns (16
// bytes a lane per row, 16 rows in flight): it keeps the 16 row sums, and adds
// each tile's column sums, the transposed products of the blocks left of the
// diagonal, to its own FP64 column buffer in shared memory.  After a cluster
// barrier every CTA adds the 8 C buffers of a share of the rows in a fixed
// order (distributed shared memory): no atomics, no second pass.  C = 1 fills
// the chip from about 300 subdomains on, 2 to 8 split fewer; the set-up
// autotuner times them.
#include "feti_internal.h"
#include "feti_fixed.cuh"
#include "feti_launch.cuh"
#include "feti_smem.h"

#include <cooperative_groups.h>

namespace feti {
namespace {

namespace cg = cooperative_groups;

constexpr int PR = kFixRows;  // panel rows
constexpr int SW = 8;         // warps per CTA of the set-up kernels
constexpr int kPoison = -1000000;  // far below any exponent
constexpr int kEmptyRow = -4000;   // exponent of a row of zeros: below any other
constexpr int kPoorList = 64;      // rows that the warps of a CTA share out
constexpr int kWeak = 8;           // bits |M| |v| of a row may stay below 2^(e_i) w

// Entry offset of panel I: panel J holds (J >> 2) + 1 tiles.
__host__ __device__ inline int64_t fix_panel(int64_t I) { return 1024 * ((I >> 2) + 1) * (2 * (I >> 2) + (I & 3)); }

// Row exponents: x = ceil(log2(row's largest entry) / 2), kPoison for a row
// whose largest entry is infinite, NaN or below 2^-895 (so that no rounding unit
// underflows); y: a_ii >= 2^(2 x - y).
__global__ void __launch_bounds__(256) k_fix_exp(const SubLayout* __restrict__ lay, int which,
                                                 const double* __restrict__ M, int2* __restrict__ ex) {
  const SubLayout L = lay[blockIdx.y];
  const int m = which == 0 ? L.nbp : L.nbp + L.k;
  const int row = blockIdx.x * SW + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (row >= m) return;
  const double* a = M + (which == 0 ? L.foff : L.soff) + (size_t)row * m;
  int e = 0;
  bool any = false;
#pragma unroll 4
  for (int c = lane; c < m; c += 32) {
    const double x = a[c];
    e = max(e, bexp64(x));
    any = any || x != 0.0;
  }
  e = __reduce_max_sync(0xffffffffu, e);
  any = __any_sync(0xffffffffu, any);
  // |a| < 2^(e - 1022)
  if (lane) return;
  const int x = !any ? kEmptyRow : e == 2047 || e < 128 ? kPoison : (e - 1022 + 1) >> 1;
  const double d = a[row];
  ex[L.boff + row] = make_int2(x, d > 0.0 ? min(max(2 * x - (bexp64(d) - 1023), 0), 100) : 100);
}

// Panels from the full FP64 matrix, one CTA per panel.
__global__ void __launch_bounds__(256) k_fix_pack(const SubLayout* __restrict__ lay, int which,
                                                  const double* __restrict__ M, const int2* __restrict__ ex,
                                                  int2* __restrict__ out) {
  const SubLayout L = lay[blockIdx.y];
  const int m = which == 0 ? L.nbp : L.nbp + L.k;
  const int I = blockIdx.x;
  if (I * PR >= m) return;
  const double* a = M + (which == 0 ? L.foff : L.soff);
  const int w = PR * (I + 1);
  int2* o = out + (which == 0 ? L.ffix : L.sfix) + fix_panel(I);
  const int2* e = ex + L.boff;
  for (int r = threadIdx.x >> 5; r < PR; r += SW) {
    const int gr = PR * I + r;
    const int er = gr < m ? e[gr].x : 0;
    for (int c = threadIdx.x & 31; c < w; c += 32) {
      int2 q = make_int2(0, 0);
      if (gr < m && c < m) {
        const int ec = e[c].x;
        const double x = a[(size_t)gr * m + c];
        if (er != kPoison && ec != kPoison) {
          // x 2^(56 - er - ec): mantissa << 3 is x 2^(56 - (bexp - 1022))
          const long long v = fixed64<3>(x, er + ec - (bexp64(x) - 1022));
          q.x = (int)((v + (1 << 27)) >> 28);
          q.y = (int)(v - ((long long)q.x << 28));
        }
      }
      o[(size_t)(c >> 6) * 1024 + 64 * r + (c & 63)] = q;
    }
  }
}

// A warp's place in its panels: panel of rows r0 .. and w columns, tile at
// column c0, the lane's two entries of its first row at p.
struct Place {
  int k, r0, w, c0;
  const int4* p;
  // panel of round k, snake order over G warps, longest first; false past the last
  __device__ __forceinline__ bool panel(int k_, int G, int g, int nP, const int2* M, int lane) {
    for (k = k_; k * G < nP; ++k) {
      const int pos = k * G + ((k & 1) ? G - 1 - g : g);
      if (pos >= nP) continue;
      const int I = nP - 1 - pos;
      r0 = PR * I;
      w = r0 + PR;
      c0 = 0;
      p = reinterpret_cast<const int4*>(M + fix_panel(I)) + lane;
      return true;
    }
    return false;
  }
};

constexpr int GR = 8;  // rows per load group: one group in flight while the other is multiplied

// Lanes right of the panel keep what they hold: their entries of v are zero and
// their column sums are dropped.
__device__ __forceinline__ void load_group(int4 (&a)[GR], const Place& q, int g, int lane) {
  if (q.c0 + 2 * lane < q.w) {
#pragma unroll
    for (int r = 0; r < GR; ++r) a[r] = __ldg(q.p + 32 * (GR * g + r));
  }
}

__device__ __forceinline__ void mul_group(const int4 (&a)[GR], const int2* __restrict__ vr, const int4& vc, long long* rh,
                                          long long* rc, long long (&col)[4]) {
#pragma unroll
  for (int r = 0; r < GR; r += 4) {  // four rows at a time: independent accumulators side by side
#pragma unroll
    for (int i = r; i < r + 4; ++i) rh[i] = mad_wide(a[i].x, vc.x, rh[i]);
#pragma unroll
    for (int i = r; i < r + 4; ++i) rc[i] = mad_wide(a[i].x, vc.y, rc[i]);
    int2 v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = vr[r + i];
#pragma unroll
    for (int i = r; i < r + 4; ++i) rh[i] = mad_wide(a[i].z, vc.z, rh[i]);
#pragma unroll
    for (int i = r; i < r + 4; ++i) rc[i] = mad_wide(a[i].y, vc.x, rc[i]);
#pragma unroll
    for (int i = r; i < r + 4; ++i) {
      col[0] = mad_wide(a[i].x, v[i - r].x, col[0]);
      col[1] = mad_wide(a[i].x, v[i - r].y, col[1]);
      col[2] = mad_wide(a[i].z, v[i - r].x, col[2]);
      col[3] = mad_wide(a[i].z, v[i - r].y, col[3]);
      rc[i] = mad_wide(a[i].z, vc.w, rc[i]);
    }
#pragma unroll
    for (int i = r; i < r + 4; ++i) {
      rc[i] = mad_wide(a[i].w, vc.z, rc[i]);
      col[1] = mad_wide(a[i].y, v[i - r].x, col[1]);
      col[3] = mad_wide(a[i].w, v[i - r].x, col[3]);
    }
  }
}

// y_i as an FP64 sum by one warp.
__device__ __forceinline__ void row_fp64(const double* __restrict__ a, const double* __restrict__ v, int m, double* y) {
  const int lane = threadIdx.x & 31;
  double s = 0.0;
#pragma unroll 16
  for (int c = lane; c < m; c += 32) s += a[c] * v[c];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) *y = s;
}

template <int W>
__global__ void __launch_bounds__(32 * W, W == 6 ? 2 : 1) k_symv_fix64(const int32_t* __restrict__ order, int C, int early,
                                                          const SubLayout* __restrict__ lay, int which,
                                                          const int2* __restrict__ M, const int2* __restrict__ ex,
                                                          const double* __restrict__ M64,
                                                          const double* __restrict__ vloc, double* __restrict__ y,
                                                          const int* __restrict__ done) {
  dep_wait();
  if (early) dep_go();
  M = fresh(M);
  ex = fresh(ex);
  vloc = fresh(vloc);
  y = fresh(y);
  done = fresh(done);
  if (*done) return;
  extern __shared__ __align__(16) unsigned char sm_fix[];
  __shared__ int s_emax, s_poor[kPoorList], n_poor;
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = C > 1 ? (int)cluster.block_rank() : 0;
  const SubLayout L = lay[order[blockIdx.x / C]];
  const int m = which == 0 ? L.nbp : L.nbp + L.k;
  const int nP = (m + PR - 1) / PR, mp = nP * PR;
  int2* vs = reinterpret_cast<int2*>(sm_fix);          // [mp] limbs of v
  double* cols = reinterpret_cast<double*>(vs + mp);   // [W][mp] sums by row, one buffer per warp
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const double* v = vloc + L.boff;
  const int2* e = ex + L.boff;
  const int2* Mb = M + (which == 0 ? L.ffix : L.sfix);
  const int G = W * C, g = W * rank + warp;
  Place cur;
  const bool any = cur.panel(0, G, g, nP, Mb, lane);
  int4 a0[GR], a1[GR];
#pragma unroll
  for (int r = 0; r < GR; ++r) a0[r] = a1[r] = make_int4(0, 0, 0, 0);
  if (any) load_group(a0, cur, 0, lane);  // the first tile travels while v is scaled
  if (which == 0 && rank == 0)
    for (int p = tid; p < L.k; p += 32 * W) y[L.boff + L.nbp + p] = 0.0;
  // largest scaled entry: biased exponent of v_j plus e_j
  if (tid == 0) {
    s_emax = kPoison;
    n_poor = 0;
  }
  __syncthreads();
  int em = kPoison, sub = kPoison - 100;
  bool bad = false;
  for (int j = tid; j < m; j += 32 * W) {
    const double x = v[j];
    const int b = bexp64(x), ej = e[j].x;
    bad = bad || b == 2047 || ej == kPoison;
    if (b)
      em = max(em, b + ej);
    else if (x != 0.0)
      sub = max(sub, ej + 1);  // a subnormal entry counts as zero below
  }
  em = __reduce_max_sync(0xffffffffu, em);
  if (lane == 0) atomicMax(&s_emax, em);
  __syncthreads();
  em = s_emax;
  bad = __syncthreads_or(bad || sub > em - 57);
  for (int j = tid; j < mp; j += 32 * W) {
    int2 q = make_int2(0, 0);
    if (j < m) {
      const long long x = fixed64<3>(v[j], em - bexp64(v[j]) - e[j].x);
      q.x = (int)((x + (1 << 27)) >> 28);
      q.y = (int)(x - ((long long)q.x << 28));
    }
    vs[j] = q;
  }
  for (int j = tid; j < W * mp; j += 32 * W) cols[j] = 0.0;
  __syncthreads();
  double* cw = cols + (size_t)warp * mp;
  long long rh[PR], rc[PR];
#pragma unroll
  for (int r = 0; r < PR; ++r) rh[r] = rc[r] = 0;
  bool more = any;
  while (more) {
    const int c = cur.c0 + 2 * lane, r0 = cur.r0;
    const int4 vc = c < cur.w ? *reinterpret_cast<const int4*>(vs + c) : make_int4(0, 0, 0, 0);
    long long col[4] = {0, 0, 0, 0};
    load_group(a1, cur, 1, lane);
    mul_group(a0, vs + r0, vc, rh, rc, col);
    const bool last = cur.c0 + 64 >= cur.w;  // of this panel
    if (last)
      more = cur.panel(cur.k + 1, G, g, nP, Mb, lane);
    else
      cur.c0 += 64, cur.p += 512;
    if (more) load_group(a0, cur, 0, lane);
    mul_group(a1, vs + r0 + GR, vc, rh + GR, rc + GR, col);
    if (c < r0) {  // left of the diagonal block: the transposed products
      double2* d = reinterpret_cast<double2*>(cw + c);
      double2 t = *d;
      t.x += (double)(col[0] + ((col[1] + (1 << 27)) >> 28));
      t.y += (double)(col[2] + ((col[3] + (1 << 27)) >> 28));
      *d = t;
    }
    if (!last) continue;
    // row sums over the lanes, half of the rows handed over per step; two
    // steps in integers (units of 4), three in FP64
    long long u[PR];
#pragma unroll
    for (int r = 0; r < PR; ++r) {
      u[r] = (rh[r] + ((rc[r] + (1 << 27)) >> 28) + 2) >> 2;
      rh[r] = rc[r] = 0;
    }
    const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4, b1 = lane & 2;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const long long o = __shfl_xor_sync(0xffffffffu, b4 ? u[r] : u[r + 8], 16);
      u[r] = (b4 ? u[r + 8] : u[r]) + o;
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const long long o = __shfl_xor_sync(0xffffffffu, b3 ? u[r] : u[r + 4], 8);
      u[r] = (b3 ? u[r + 4] : u[r]) + o;
    }
    double d[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) d[r] = (double)u[r];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const double o = __shfl_xor_sync(0xffffffffu, b2 ? d[r] : d[r + 2], 4);
      d[r] = (b2 ? d[r + 2] : d[r]) + o;
    }
    {
      const double o = __shfl_xor_sync(0xffffffffu, b1 ? d[0] : d[1], 2);
      d[0] = (b1 ? d[1] : d[0]) + o;
    }
    d[0] += __shfl_xor_sync(0xffffffffu, d[0], 1);
    __syncwarp();
    if (!(lane & 1)) cw[r0 + ((lane >> 1) & 1) + ((lane >> 2) & 1) * 2 + ((lane >> 3) & 1) * 4 + ((lane >> 4) & 1) * 8] +=
        4.0 * d[0];
    __syncwarp();
  }
  if (C > 1)
    cluster.sync();
  else
    __syncthreads();
  const int per = (m + C - 1) / C;
  const int i1 = min(m, (rank + 1) * per);
  const double* Mr = fresh(M64) + (which == 0 ? L.foff : L.soff);
  // rows of this warp, then the weak ones of all of them at once
  const int lo = rank * per + 32 * warp;
  unsigned weak_mask = 0;  // lane k: rows of the warp's k-th group of 32
  int n_weak = 0;
  for (int i0 = lo, k = 0; i0 < i1; i0 += 32 * W, ++k) {
    const int i = i0 + lane;
    bool weak = false;
    if (i < i1) {
      double t = 0.0;
      for (int q = 0; q < C; ++q) {
        const double* b = C > 1 ? cluster.map_shared_rank(cols, q) : cols;
#pragma unroll
        for (int k = 0; k < W; ++k) t += b[(size_t)k * mp + i];
      }
      const int2 ei = e[i];
      weak = bad || (em != kPoison && abs(vs[i].x) < 1 << min(28 - kWeak + ei.y, 30) && bexp64(t) < 1023 + 56 - kWeak);
      y[L.boff + i] = em == kPoison ? 0.0 : scalbn(t, ei.x + em - 1022 - 56);
    }
    const unsigned mask = __ballot_sync(0xffffffffu, weak);
    if (lane == k) weak_mask = mask;
    n_weak += __popc(mask);
  }
  __syncwarp();
  int below = 0;  // weak rows of the groups before the lane's
  {
    int inc = __popc(weak_mask);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += u;
    }
    below = inc - __popc(weak_mask);
  }
  for (int r0 = 0; r0 < n_weak; r0 += 8) {
    const int want = r0 + (lane >> 2);
    int row = -1;
    // the group that holds row `want` of the list: the last with below <= want
    int g2 = 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
      if (__shfl_sync(0xffffffffu, below, g2 + o) <= want) g2 += o;
    const unsigned gm = __shfl_sync(0xffffffffu, weak_mask, g2);
    const int gb = __shfl_sync(0xffffffffu, below, g2);
    if (want < n_weak) row = lo + 32 * W * g2 + (int)__fns(gm, 0, want - gb + 1);
    long long sum = 0;
    if (row >= 0 && !bad) {
      const int I = row / PR, w = PR * (I + 1), t1 = (w - 1) >> 6;
      const int4* p = reinterpret_cast<const int4*>(Mb + fix_panel(I)) + 32 * (row % PR);
      for (int tile = max(t1 - 1, 0); tile <= t1; ++tile) {
        int4 a[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int q = (lane & 3) + 4 * u;
          a[u] = 64 * tile + 2 * q < w ? __ldg(p + 512 * tile + q) : make_int4(0, 0, 0, 0);
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int c = min(64 * tile + 2 * ((lane & 3) + 4 * u), mp - 2);
          const int4 vc = *reinterpret_cast<const int4*>(vs + c);
          sum = mad_wide(abs(a[u].x), abs(vc.x), sum);
          sum = mad_wide(abs(a[u].z), abs(vc.z), sum);
        }
      }
    }
    sum += __shfl_xor_sync(0xffffffffu, sum, 2);
    sum += __shfl_xor_sync(0xffffffffu, sum, 1);
    unsigned poor = __ballot_sync(0xffffffffu, row >= 0 && !(lane & 3) && (bad || sum < 1ll << (56 - kWeak)));
    for (; poor; poor &= poor - 1) {
      const int i = __shfl_sync(0xffffffffu, row, __ffs(poor) - 1);
      int k = 0;
      if (lane == 0) {
        k = atomicAdd(&n_poor, 1);
        if (k < kPoorList) s_poor[k] = i;
      }
      if (__shfl_sync(0xffffffffu, k, 0) >= kPoorList) row_fp64(Mr + (size_t)i * m, v, m, y + L.boff + i);
    }
  }
  __syncthreads();
  for (int k = warp; k < min(n_poor, kPoorList); k += W)
    row_fp64(Mr + (size_t)s_poor[k] * m, v, m, y + L.boff + s_poor[k]);
  if (C > 1) cluster.sync();  // the buffers stay until every CTA has read them
}

size_t fix_smem(int max_m, int W) {
  const size_t mp = (size_t)(max_m + PR - 1) / PR * PR;
  return mp * sizeof(int2) + W * mp * sizeof(double);
}
constexpr size_t kFixSmem = 226 * 1024;

template <int W>
cudaError_t launch_fix(int C, int P, const int32_t* order, int max_m, const SubLayout* lay, int which, const int2* M,
                       const int2* ex, const double* M64, const double* vloc, double* y, const int* done,
                       cudaStream_t st) {
  const size_t sm = fix_smem(max_m, W);
  (void)allow_smem(k_symv_fix64<W>, sm);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(P * C));
  cfg.blockDim = dim3(32 * W);
  cfg.dynamicSmemBytes = sm;
  cfg.stream = st;
  cudaLaunchAttribute at[2]{};
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)C;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  // operators that stay in the second-level cache (a few 10 us) are placed while
  // the gather before them runs, and let the scatter be placed beside them
  // (quadratic cube, 52 MB, 14.0 -> 12.6 ms a solve); larger ones are not:
  // beside the gather their CTAs spread unevenly over the SMs (64-subdomain
  // tube, 334 MB, 82.9 -> 85.8 ms)
  const int early = (int64_t)P * max_m * max_m * 4 <= (int64_t)128 << 20 ? 1 : 0;
  cfg.numAttrs = 1 + early;
  return cudaLaunchKernelEx(&cfg, k_symv_fix64<W>, order, C, early, lay, which, M, ex, M64, vloc, y, done);
}

}  // namespace

int64_t fix_entries(int m) { return fix_panel((m + PR - 1) / PR); }

// Shared memory of the largest operator: up to 3,200 rows.  The row sums would
// hold in 64 bits up to 64 tiles (2^63 / 2^56 / 2 columns a lane).
static_assert(kFixSmem / (sizeof(int2) + 8 * sizeof(double)) < 64 * 64 - PR, "row sums of one row's tiles in 64 bits");
bool symv_fixed_fits(int max_m) { return fix_smem(max_m, 8) <= kFixSmem; }

void launch_fix_operator(int P, int max_m, const SubLayout* lay, int which, const double* M, int2* ex, int2* out,
                         cudaStream_t st) {
  if (max_m <= 0) return;
  k_fix_exp<<<dim3((max_m + SW - 1) / SW, P), 256, 0, st>>>(lay, which, M, ex);
  k_fix_pack<<<dim3((max_m + PR - 1) / PR, P), 256, 0, st>>>(lay, which, M, ex, out);
}

cudaError_t launch_symv_fixed(int C, int P, const int32_t* order, int max_m, const SubLayout* lay, int which,
                              const int2* M, const int2* ex, const double* M64, const double* vloc, double* y,
                              const int* done, cudaStream_t st) {
  // six warps and two CTAs per SM, so that one CTA's start and end run beside
  // the other's stream, while two sets of buffers fit
  if (2 * fix_smem(max_m, 6) <= kFixSmem)
    return launch_fix<6>(C, P, order, max_m, lay, which, M, ex, M64, vloc, y, done, st);
  return launch_fix<8>(C, P, order, max_m, lay, which, M, ex, M64, vloc, y, done, st);
}

}  // namespace feti
