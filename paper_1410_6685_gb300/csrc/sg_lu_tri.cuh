// sg_lu_tri.cuh -- small triangular solves shared by the elimination kernels
// (k_lu.cu, k_lu_diag.cu).
#pragma once
#include <cuda_runtime.h>

#include "sg_lu.h"

namespace sgk {

// x := L^-1 x for one column x of 32 entries (stride xs) and the unit lower
// triangle of L (row stride ls, a multiple of 4; L 16-byte aligned), by
// forward substitution in registers: row i subtracts L[i][0] x[0], L[i][1]
// x[1], ... in that order, reading L's row four entries per shared-memory
// load.
__device__ __forceinline__ void unit_lower_solve_col4(const float* L, int ls, float* x, int xs) {
  float v[kLuPanel];
#pragma unroll
  for (int i = 0; i < kLuPanel; ++i) v[i] = x[i * xs];
#pragma unroll
  for (int i = 1; i < kLuPanel; ++i) {
    float acc = v[i];
    const float4* Li = reinterpret_cast<const float4*>(L + i * ls);
#pragma unroll
    for (int g = 0; g < i / 4; ++g) {
      const float4 l = Li[g];
      acc = fmaf(-l.x, v[4 * g], acc);
      acc = fmaf(-l.y, v[4 * g + 1], acc);
      acc = fmaf(-l.z, v[4 * g + 2], acc);
      acc = fmaf(-l.w, v[4 * g + 3], acc);
    }
#pragma unroll
    for (int q = (i / 4) * 4; q < i; ++q) acc = fmaf(-L[i * ls + q], v[q], acc);
    v[i] = acc;
  }
#pragma unroll
  for (int i = 1; i < kLuPanel; ++i) x[i * xs] = v[i];
}

}  // namespace sgk
