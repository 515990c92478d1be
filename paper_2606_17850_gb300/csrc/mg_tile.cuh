// The two halves of a multigrid level on a tile of columns, one thread per column.
//
// A block of 32 x EY threads covers a grown tile: its inner (32 - 2) x (EY - 2) columns
// are results, the ring around them supplies their neighbours.  Every thread brings its
// own column (all layers) into registers once, with independent loads, and the in-plane
// neighbours are read from shared memory, so a cell costs one global load per vector
// instead of five, and the two passes of a level's way down (smoothing from zero, residual
// and restriction) need b only once: the ring's columns are smoothed again, which is local
// to a column.  Both halves work on any nx, ny (aggregates at an odd edge are incomplete)
// and on either coefficient source.  CG: the vectors were written by other blocks of
// the running kernel (loads that bypass L1).
//
// Order of a cell's product: s x, then the x, y and z faces (+ before -); an aggregate is
// summed x pairs first: the operations of the kernels that read every neighbour from global
// memory, in their order.  A V-cycle's error against 64 bits over 24 right-hand sides on four
// grids (5e-8 to 1.2e-7 of ||z||) is 0.53 to 1.43 of theirs, 0.94 in the mean: which way FP32
// rounds, not how much.
#pragma once

#include "mg_device.cuh"

#define MGT_EX 32

template <bool CG>
__device__ __forceinline__ float mgt_ld(const float* p) {
  return CG ? __ldcg(p) : *p;
}

// tiles of a level
template <int EY>
__host__ __device__ __forceinline__ int mgt_tiles(int nx, int ny) {
  return ((nx + MGT_EX - 3) / (MGT_EX - 2)) * ((ny + EY - 3) / (EY - 2));
}

// Coefficients of one column (layers z < LMAX, in registers' reach): the level's table,
// zero beyond the stack's layers, or the per-cell arrays, zero where there is no cell.  No
// loop over layers leaves early: a branch per layer would keep the loads of one layer
// from being issued before the arithmetic of the one before.
template <int LMAX, bool UNI>
struct MGTCol {
  const MGDev& v;
  const MGUni<LMAX>& U;
  long long i0, pxy;
  int cs;
  bool on, hasL, hasD;
  __device__ __forceinline__ float cell(const float* a, int z, long long off, bool ok) const {
    return (ok && z >= 0 && z < v.L) ? __ldg(a + i0 + pxy * z + off) : 0.f;
  }
  __device__ __forceinline__ float s(int z) const { return UNI ? U.s[z] : cell(v.s, z, 0, on); }
  __device__ __forceinline__ float gxr(int z) const { return UNI ? U.gx[z] : cell(v.gx, z, 0, on); }
  __device__ __forceinline__ float gxl(int z) const { return UNI ? U.gx[z] : cell(v.gx, z, -1, on && hasL); }
  __device__ __forceinline__ float gyu(int z) const { return UNI ? U.gy[z] : cell(v.gy, z, 0, on); }
  __device__ __forceinline__ float gyd(int z) const { return UNI ? U.gy[z] : cell(v.gy, z, -v.nx, on && hasD); }
  __device__ __forceinline__ float gz(int z) const {  // face above layer z
    return z < 0 ? 0.f : (UNI ? U.gz[z] : cell(v.gz, z, 0, on));
  }
  __device__ __forceinline__ float m(int z) const { return UNI ? U.m[cs][z] : cell(v.m, z, 0, on); }
  __device__ __forceinline__ float w(int z) const { return UNI ? U.w[cs][z] : cell(v.w, z, 0, on); }
};

// where this thread stands in the grown tile
template <int EY>
struct MGTPos {
  int x, y, tid, oR, oL, oU, oD;  // column; shared-memory places of it and its neighbours
  bool inside, inner;
  long long i0, pxy;
  int cs;
  __device__ __forceinline__ MGTPos(const MGDev& v, int bx, int by) {
    const int ex = threadIdx.x, ey = threadIdx.y;
    tid = ex + MGT_EX * ey;
    x = bx * (MGT_EX - 2) - 1 + ex;
    y = by * (EY - 2) - 1 + ey;
    inside = x >= 0 && x < v.nx && y >= 0 && y < v.ny;
    inner = inside && ex > 0 && ex < MGT_EX - 1 && ey > 0 && ey < EY - 1;
    pxy = (long long)v.nx * v.ny;
    i0 = inside ? (long long)x + (long long)v.nx * y : 0;
    const bool r = x + 1 < v.nx, l = x > 0, u = y + 1 < v.ny, d = y > 0;
    cs = inside ? (int)r + (int)l + 3 * ((int)u + (int)d) : 0;
    // an absent neighbour is the column itself (difference 0); only inner columns look
    oR = inner && r ? tid + 1 : tid;
    oL = inner && l ? tid - 1 : tid;
    oU = inner && u ? tid + MGT_EX : tid;
    oD = inner && d ? tid - MGT_EX : tid;
  }
};

// residual of layer z: b_z - (A x)_z, x in registers and (in-plane neighbours) in xs
template <int LMAX, bool UNI, int EY>
__device__ __forceinline__ float mgt_residual(const MGTCol<LMAX, UNI>& C, const MGTPos<EY>& p, const float* xs, int z,
                                              float bz, const float (&xv)[LMAX]) {
  const float* q = xs + z * (MGT_EX * EY);
  const float xi = xv[z];
  float a = C.s(z) * xi;
  a += C.gxr(z) * (xi - q[p.oR]);
  a += C.gxl(z) * (xi - q[p.oL]);
  a += C.gyu(z) * (xi - q[p.oU]);
  a += C.gyd(z) * (xi - q[p.oD]);
  if (z + 1 < LMAX) a += C.gz(z) * (xi - xv[z + 1 < LMAX ? z + 1 : z]);
  if (z > 0) a += C.gz(z - 1) * (xi - xv[z > 0 ? z - 1 : 0]);
  return bz - a;
}

// Way down: x = omega T^-1 b, b_c = P^T (b - A x).  xs: LMAX x (32 EY) floats.
template <int LMAX, bool UNI, int EY, bool CG>
__device__ __forceinline__ void mgt_down(const MGDev& v, const MGUni<LMAX>& U, int bx, int by, const float* b,
                                         float* xout, int nxc, int nyc, float* bc, float* xs) {
  constexpr int NT = MGT_EX * EY;
  const MGTPos<EY> p(v, bx, by);
  const MGTCol<LMAX, UNI> C{v, U, p.i0, p.pxy, p.cs, p.inside, p.x > 0, p.y > 0};
  const int L = v.L, tid = p.tid;
  float bv[LMAX], xv[LMAX];
#pragma unroll
  for (int z = 0; z < LMAX; ++z) bv[z] = (p.inside && z < L) ? mgt_ld<CG>(b + p.i0 + p.pxy * z) : 0.f;
  float dprev = 0.f;
#pragma unroll
  for (int z = 0; z < LMAX; ++z) xv[z] = dprev = (bv[z] + C.gz(z - 1) * dprev) * C.m(z);
  float dn = 0.f;
#pragma unroll
  for (int z = LMAX - 1; z >= 0; --z) {
    dn = xv[z] + C.w(z) * dn;
    xv[z] = kMGOmega * dn;
    xs[z * NT + tid] = xv[z];
    if (p.inner && z < L) xout[p.i0 + p.pxy * z] = xv[z];
  }
  __syncthreads();
#pragma unroll
  for (int z = 0; z < LMAX; ++z) {
    const float r = mgt_residual<LMAX, UNI, EY>(C, p, xs, z, bv[z], xv);
    bv[z] = p.inner ? r : 0.f;
    bv[z] += __shfl_down_sync(0xffffffffu, bv[z], 1);  // x pair (x even in odd lanes)
  }
  __syncthreads();
#pragma unroll
  for (int z = 0; z < LMAX; ++z) xs[z * NT + tid] = bv[z];
  __syncthreads();
  if (p.inner && (threadIdx.x & 1) && (threadIdx.y & 1)) {  // y even in odd rows
    const long long ic = (long long)(p.x >> 1) + (long long)nxc * (p.y >> 1), pc = (long long)nxc * nyc;
#pragma unroll
    for (int z = 0; z < LMAX; ++z)
      if (z < L) bc[ic + pc * z] = xs[z * NT + tid] + xs[z * NT + tid + MGT_EX];
  }
}

// Way up: x = x_in + P x_c, x_out = x + omega T^-1 (b - A x).  With RZ it returns this
// thread's part of b^T x_out (b read again, so that the sweep can reuse its registers): four
// layers in two sums of two, the fours one after the other, so that the product of an
// 8-layer column meets three additions and that of a 32-layer one nine.  (The V-cycle at
// 1024^2 x 10 took 215.6 us with one sum over the layers, 215.5 so, 222 with four sums side
// by side: the pass has no registers to spare.)
template <int LMAX, bool UNI, int EY, bool CG, bool RZ>
__device__ __forceinline__ float mgt_up(const MGDev& v, const MGUni<LMAX>& U, int bx, int by, const float* b,
                                        const float* xin, const float* xc, int nxc, int nyc, float* xout, float* xs) {
  constexpr int NT = MGT_EX * EY;
  const MGTPos<EY> p(v, bx, by);
  const MGTCol<LMAX, UNI> C{v, U, p.i0, p.pxy, p.cs, p.inside, p.x > 0, p.y > 0};
  const int L = v.L, tid = p.tid;
  const long long ic = p.inside ? (long long)(p.x >> 1) + (long long)nxc * (p.y >> 1) : 0, pc = (long long)nxc * nyc;
  float bv[LMAX], xv[LMAX];
#pragma unroll
  for (int z = 0; z < LMAX; ++z) {
    const bool on = p.inside && z < L;
    xv[z] = on ? mgt_ld<CG>(xin + p.i0 + p.pxy * z) : 0.f;
    bv[z] = on ? mgt_ld<CG>(xc + ic + pc * z) : 0.f;
  }
#pragma unroll
  for (int z = 0; z < LMAX; ++z) {
    xv[z] += bv[z];
    xs[z * NT + tid] = xv[z];
  }
#pragma unroll
  for (int z = 0; z < LMAX; ++z) bv[z] = (p.inner && z < L) ? mgt_ld<CG>(b + p.i0 + p.pxy * z) : 0.f;
  __syncthreads();
  float rz = 0.f, two[2] = {0.f, 0.f}, dprev = 0.f;
#pragma unroll
  for (int z = 0; z < LMAX; ++z) {
    const float res = mgt_residual<LMAX, UNI, EY>(C, p, xs, z, bv[z], xv);
    bv[z] = dprev = (res + C.gz(z - 1) * dprev) * C.m(z);
  }
  float dn = 0.f;
#pragma unroll
  for (int z = LMAX - 1; z >= 0; --z) {
    dn = bv[z] + C.w(z) * dn;
    const float o = xv[z] + kMGOmega * dn;
    const bool on = p.inner && z < L;
    if (on) xout[p.i0 + p.pxy * z] = o;
    if (RZ) {
      const float q = on ? mgt_ld<CG>(b + p.i0 + p.pxy * z) : 0.f;
      two[z % 2] = z % 4 > 1 ? q * o : two[z % 2] + q * o;
      if (z % 4 == 0) rz += two[0] + two[1];
    }
  }
  return rz;
}
