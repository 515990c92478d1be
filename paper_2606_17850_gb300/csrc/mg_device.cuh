// Device code of the multigrid V-cycle shared by the single-grid kernels
// (multigrid.cu) and the batched persistent solve (batched.cu): level descriptors and
// the coarsest dense solve (the passes of a level: mg_tile.cuh).
//
// One V-cycle applies M^-1 (see multigrid.cu): x/y aggregation of 2 x 2 columns,
// piecewise-constant P, R = P^T, Galerkin coarse operators, damped z-line Jacobi
// x <- x + omega T^-1 (b - A x) with T the tridiagonal block of a column, exact
// coarsest solve.
#pragma once

#include "common.cuh"

constexpr float kMGOmega = 0.8f;  // damping of the z-line Jacobi smoother

struct MGDev {  // one level, by value into kernels
  int nx, ny, L;
  const float *gx, *gy, *gz, *s, *m, *w;
};

// A layer-uniform level: the coefficients and the Thomas factors depend only on the
// layer and on which in-plane neighbours exist (case nxf + 3 nyf, nxf/nyf = number
// of x/y neighbours), so they come from this table (kernel parameters) instead of
// per-cell arrays.
template <int LMAX>
struct MGUni {
  float s[LMAX], gx[LMAX], gy[LMAX], gz[LMAX];  // gz: face to the layer above (0 on top)
  float m[9][LMAX], w[9][LMAX];
};

// coarsest level: x = C b with the dense inverse C (n x n, FP32), one warp per row;
// warps `warp0`, `warp0 + nwarps`, ... of the caller take the rows
__device__ __forceinline__ void mg_coarsest_rows(int n, const float* __restrict__ C, const float* __restrict__ b,
                                                 float* __restrict__ x, int warp0, int nwarps) {
  const int lane = threadIdx.x & 31;
  for (int row = warp0; row < n; row += nwarps) {
    float acc = 0.f;
    for (int j = lane; j < n; j += 32) acc += C[(long long)row * n + j] * b[j];
    acc = warp_sum(acc);
    if (lane == 0) x[row] = acc;
  }
}
