// Topology tables of the vector kernels: signed rows of a boundary position,
// signed positions of a row, R row of a position.
//
// The vector kernels of an iteration are chains of dependent loads (pointer,
// row, value) around a few FP64 operations.  The topology comes from tables of
// one 8- or 16-byte entry per row and position, read before the wait for the
// previous kernel; the values are then loaded at once, and the stop flag after
// them, so that one memory latency is left.  Newton load step on 32
// subdomains (6,256 iterations of 14 launches): 600 -> 470 ms; quadratic cube
// 13.0 -> 12.0 ms.
#pragma once
#include "feti_internal.h"

namespace feti {
namespace {

// Positions: rows 2 row + (sign < 0) in x, y, z (-1: none), w further rows in
// the lists.  Rows: the same code for their two positions.
__device__ __forceinline__ int4 pos_rows(const Maps& mp, int gp) {
  return gp < mp.nb_total ? __ldg(mp.bt_tab + gp) : make_int4(-1, -1, -1, 0);
}
__device__ __forceinline__ int2 row_poss(const Maps& mp, int r) {
  return r < mp.n_lambda ? __ldg(mp.row_tab + r) : make_int2(-1, -1);
}
__device__ __forceinline__ double signed_val(int t, double v) {  // the sign as an integer operation
  return __hiloint2double(__double2hiint(v) ^ (int)((unsigned)t << 31), __double2loint(v));
}

// The stop flag, loaded after the loads that precede it in the program.
__device__ __forceinline__ int flag_now(const int* done) {
  int d;
  asm volatile("ld.global.s32 %0, [%1];" : "=r"(d) : "l"(done) : "memory");
  return d;
}

// Signed sum of the rows beyond the third, continued on v.
template <typename F>
__device__ __forceinline__ double more_rows(const Maps& mp, int gp, int n, double v, F x) {
  const int end = mp.bt_ptr[gp + 1];
  for (int e = end - n; e < end; e += 4) {
    double t[4], sg[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int ei = min(e + i, end - 1);
      sg[i] = mp.bt_sgn[ei];
      t[i] = x(mp.bt_row[ei]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (e + i < end) v += sg[i] * t[i];
  }
  return v;
}

// Offset of the R row in the last two words of a table entry.
__device__ __forceinline__ int64_t pos_roff(const int4& t) {
  return (int64_t)(((uint64_t)(uint32_t)t.w << 32) | (uint32_t)t.z);
}

}  // namespace
}  // namespace feti
