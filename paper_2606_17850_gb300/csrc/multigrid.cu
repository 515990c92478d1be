// Geometric multigrid preconditioner (one V-cycle per application), FP32.
//
// Not in the paper: the robust alternative to the Chebyshev preconditioner when
// layers are in-plane dominated (Si, Cu) and vertically dominated (BEOL, TIM,
// bonds) in the same stack.
//
// * Semi-coarsening in x and y only (every level keeps all layers): a coarse cell
//   aggregates the 2 x 2 fine columns (2X..2X+1, 2Y..2Y+1) of its layer (fewer on an
//   odd edge).  Piecewise-constant prolongation P, restriction P^T, Galerkin coarse
//   operator P^T A P, which is again a 7-point operator: a coarse face sums the fine
//   faces crossing the aggregate boundary, the coarse per-cell term sums the fine
//   sink/capacity terms.  Levels are added while max(nx, ny) > 8.
// * Smoother: damped z-line Jacobi, x <- x + omega T^-1 (b - A x), T the tridiagonal
//   block of A over each (x, y) column (Thomas factors precomputed per level), one
//   sweep before and one after the coarse correction; omega = 0.8.
// * Coarsest level (at most 8 x 8 columns): exact solve with a dense inverse
//   computed once on the device in FP64 (banded factorisation).
// The cycle starts from zero on every level and pre/post sweeps match, so M^-1 is
// symmetric, as PCG requires.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <memory>
#include <vector>

#include "internal.h"
#include "mg_device.cuh"
#include "mg_tile.cuh"

namespace {

constexpr int MG_COARSEST = 8;

__device__ __forceinline__ long long idx3(int nx, int ny, int x, int y, int z) {
  return (long long)x + (long long)nx * ((long long)y + (long long)ny * z);
}

// per-cell sink + capacity term of the finest level from the layer table
__global__ void k_mg_s0(Dims d, const LayerTab* tab, float* __restrict__ s) {
  const Cell c = cell_of(d);
  if (!c.valid) return;
  s[c.i] = __ldg(&tab->s32[c.z]);
}

// Galerkin coarse operator of the 2 x 2-column aggregation (one thread per coarse cell)
__global__ void k_mg_coarsen(int nxf, int nyf, int nxc, int nyc, int L, const float* __restrict__ gxf,
                             const float* __restrict__ gyf, const float* __restrict__ gzf,
                             const float* __restrict__ sf, float* __restrict__ gxc, float* __restrict__ gyc,
                             float* __restrict__ gzc, float* __restrict__ sc) {
  const int X = blockIdx.x * blockDim.x + threadIdx.x;
  const int Y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = blockIdx.z;
  if (X >= nxc || Y >= nyc) return;
  const int x0 = 2 * X, y0 = 2 * Y;
  const bool hx = x0 + 1 < nxf, hy = y0 + 1 < nyf;  // second fine column / row exists
  float s = 0.f, gz = 0.f, gx = 0.f, gy = 0.f;
  for (int b = 0; b < (hy ? 2 : 1); ++b)
    for (int a = 0; a < (hx ? 2 : 1); ++a) {
      const long long i = idx3(nxf, nyf, x0 + a, y0 + b, z);
      s += sf[i];
      gz += gzf[i];
    }
  if (hx) {  // faces between fine x0+1 and x0+2, i.e. between aggregates X and X+1
    gx = gxf[idx3(nxf, nyf, x0 + 1, y0, z)];
    if (hy) gx += gxf[idx3(nxf, nyf, x0 + 1, y0 + 1, z)];
  }
  if (hy) {
    gy = gyf[idx3(nxf, nyf, x0, y0 + 1, z)];
    if (hx) gy += gyf[idx3(nxf, nyf, x0 + 1, y0 + 1, z)];
  }
  const long long ic = idx3(nxc, nyc, X, Y, z);
  sc[ic] = s;
  gzc[ic] = gz;
  gxc[ic] = (X + 1 < nxc) ? gx : 0.f;
  gyc[ic] = (Y + 1 < nyc) ? gy : 0.f;
}

// Thomas factors of every column's tridiagonal block T: b_z = A_zz, a_z = -gz_{z-1},
// c_z = -gz_z; m_z = 1 / (b_z - a_z c'_{z-1}), c'_z = c_z m_z; stored m_z and
// w_z = gz_z m_z (= -c'_z).
__global__ void k_mg_zfactors(int nx, int ny, int L, const float* __restrict__ gx, const float* __restrict__ gy,
                              const float* __restrict__ gz, const float* __restrict__ s, float* __restrict__ m,
                              float* __restrict__ w) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  if (x >= nx || y >= ny) return;
  const long long pxy = (long long)nx * ny;
  double wprev = 0.0;  // -c'_{z-1}
  for (int z = 0; z < L; ++z) {
    const long long i = idx3(nx, ny, x, y, z);
    double b = s[i];
    if (x + 1 < nx) b += gx[i];
    if (x > 0) b += gx[i - 1];
    if (y + 1 < ny) b += gy[i];
    if (y > 0) b += gy[i - nx];
    if (z + 1 < L) b += gz[i];
    const double gb = (z > 0) ? (double)gz[i - pxy] : 0.0;
    if (z > 0) b += gb;
    const double mz = 1.0 / (b - gb * wprev);  // a_z c'_{z-1} = (-gb)(-wprev)
    const double wz = (z + 1 < L) ? (double)gz[i] * mz : 0.0;
    m[i] = (float)mz;
    w[i] = (float)wz;
    wprev = wz;
  }
}

// ---------------------------------------------------------------- the cycle's kernels
// A level is two passes (mg_tile.cuh): smoothing from zero + residual + restriction on the
// way down, prolongation + smoothing on the way up, each reading its vectors once.  Levels
// with more tiles than a cluster has blocks run them as launches of their own; the levels
// below run, way down, coarsest solve and way up, in one launch of a single cluster whose
// blocks meet at its hardware barrier: they are bound by the latency of a pass, not by
// work, and a grid has two or three of them.  Measured V-cycles with r^T z, before (two
// launches down and one up per level, r^T z apart) and now: 64^2 x 4 42 -> 18.8 us, 128^2 x
// 8 69 -> 29, 357 x 301 x 8 168 -> 61, 512^2 x 8 126 -> 60, 1024^2 x 8 225 -> 126, 1024^2 x
// 10 287 -> 181.  (All these levels in one cooperative grid with a barrier in memory: 84 ->
// 108 us at 512^2; a phase there costs 5 us.)  The finest level is bound by the latency of
// a tile's load - solve - store chain at 32 warps an SM (2.3 to 2.5 TB/s).

// Rows of a block's grown tile, and blocks per SM that the registers allow.  Measured
// V-cycles (us, 512^2 x 8 / 357 x 301 x 8 / 1024^2 x 8 / 1024^2 x 10): 16 rows at 2 blocks
// 64.0 / 76.8 / 134.7 / 180.7, at 3 blocks 64.1 / 91.2 / 133.2 / 189.8; 8 rows at 4 blocks
// 60.4 / 60.7 / 131.9 / 181.3, at 6 blocks 62.3 / 74.9 / 131.1 / 183.6.
constexpr int MG_EY = 8;
constexpr unsigned MG_MINB = 4;
// blocks of the cluster (8 where 16 cannot be scheduled; 1 on a stream that has only part of
// the SMs, whose clusters may be smaller: slow, but any SM takes it)
constexpr int MG_CLUSTER = 16;

template <int LMAX>
struct MGCLev {
  int nx, ny, uni, pad;
  const float *gx, *gy, *gz, *s, *m, *w;
  float *x, *xt, *b;
  MGUni<LMAX> t;
};

template <int LMAX>
constexpr size_t mg_xs_bytes() {
  return sizeof(float) * LMAX * MGT_EX * MG_EY;
}

// Row of tiles: more than 65535 of them (ny from 393211) continue in z; those past the last
// hold no column.  (Tiles in one grid dimension, with a division, cost a 1024^2 x 10 cycle 2 %.)
__device__ __forceinline__ int mg_tile_y() { return (int)(blockIdx.y + gridDim.y * blockIdx.z); }
dim3 mg_tile_grid(int nx, int ny) {
  const unsigned rows = (ny + MG_EY - 3) / (MG_EY - 2), z = (rows + 65534) / 65535;
  return dim3((nx + MGT_EX - 3) / (MGT_EX - 2), (rows + z - 1) / z, z);
}

template <int LMAX, bool UNI>
__global__ void __launch_bounds__(MGT_EX* MG_EY, LMAX <= 12 ? MG_MINB : 1)
    k_mg_down(const Ctl* ctl, MGDev v, const __grid_constant__ MGUni<LMAX> U, const float* __restrict__ b,
              float* __restrict__ x, int nxc, int nyc, float* __restrict__ bc) {
  grid_dep_enter();
  if (ld_int(&ctl->done)) return;
  extern __shared__ __align__(16) float mg_xs[];
  mgt_down<LMAX, UNI, MG_EY, false>(v, U, blockIdx.x, mg_tile_y(), b, x, nxc, nyc, bc, mg_xs);
}

// way up; on the finest level (RZ) with r^T z and beta (b is r)
template <int LMAX, bool UNI, bool RZ>
__global__ void __launch_bounds__(MGT_EX* MG_EY, LMAX <= 12 ? MG_MINB : 1)
    k_mg_up(Ctl* ctl, MGDev v, const __grid_constant__ MGUni<LMAX> U, const float* __restrict__ b,
            const float* __restrict__ xin, const float* __restrict__ xc, int nxc, int nyc, float* __restrict__ xout,
            double* partials, int stride, unsigned* counter) {
  grid_dep_enter();
  if (ld_int(&ctl->done)) return;
  extern __shared__ __align__(16) float mg_xs[];
  if (!RZ) {
    mgt_up<LMAX, UNI, MG_EY, false, RZ>(v, U, blockIdx.x, mg_tile_y(), b, xin, xc, nxc, nyc, xout, mg_xs);
    return;
  }
  // the tiles over the blocks that are resident at once, so that the reduction's tail (7 us
  // of 19 with one tile per block at 512 x 512 x 8) is paid once per block; a thread's sum
  // over its tiles keeps its rounding errors
  Sum2 part[1] = {{0.f, 0.f}};
  const int tx = (v.nx + MGT_EX - 3) / (MGT_EX - 2);
  for (int q = blockIdx.x; q < mgt_tiles<MG_EY>(v.nx, v.ny); q += gridDim.x) {
    sum2_add(part[0], mgt_up<LMAX, UNI, MG_EY, false, RZ>(v, U, q % tx, q / tx, b, xin, xc, nxc, nyc, xout, mg_xs));
    __syncthreads();
  }
  double tot[1];
  if (!grid_reduce<Sum2, 1>(part, partials, stride, counter, tot)) return;
  ctl->rz_next = tot[0];
  ctl_set_beta(ctl);
}

__device__ __forceinline__ void mg_cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Levels k0 .. nl - 1 of one cycle by one cluster.  b0: right-hand side of level k0
// (level 0: r); z: where level 0's result goes (k0 = 0), with r^T z and beta.
template <int LMAX>
__global__ void __launch_bounds__(MGT_EX* MG_EY, 1)
    k_mg_levels(Ctl* ctl, const MGCLev<LMAX>* lv, int L, int k0, int nl, int nc, const float* __restrict__ cinv,
                const float* b0, float* z, double* partials, int stride, unsigned* counter) {
  grid_dep_enter();
  extern __shared__ __align__(16) float mg_xs[];
  static_assert(alignof(MGCLev<LMAX>) <= 16 && mg_xs_bytes<LMAX>() % 16 == 0, "descriptors behind the tile");
  MGCLev<LMAX>* sl = reinterpret_cast<MGCLev<LMAX>*>(mg_xs + LMAX * MGT_EX * MG_EY);  // levels k0 ..
  const int t = thread_linear_id();
  {
    const int* src = reinterpret_cast<const int*>(lv + k0);
    int* dst = reinterpret_cast<int*>(sl);
    for (int i = t; i < (int)(sizeof(MGCLev<LMAX>) / 4) * (nl - k0); i += MGT_EX * MG_EY) dst[i] = __ldg(src + i);
  }
  if (__syncthreads_or(t == 0 && ld_int(&ctl->done))) return;  // set by an earlier kernel: every block sees it
  Sum2 part[1] = {{0.f, 0.f}};
  for (int k = k0; k + 1 < nl; ++k) {
    const MGCLev<LMAX>& l = sl[k - k0];
    const int nxc = (l.nx + 1) / 2, nyc = (l.ny + 1) / 2, tx = (l.nx + MGT_EX - 3) / (MGT_EX - 2);
    const MGDev v{l.nx, l.ny, L, l.gx, l.gy, l.gz, l.s, l.m, l.w};
    const float* b = k == k0 ? b0 : l.b;
    float* bc = sl[k + 1 - k0].b;
    for (int q = blockIdx.x; q < mgt_tiles<MG_EY>(l.nx, l.ny); q += gridDim.x) {
      __syncthreads();
      if (l.uni) mgt_down<LMAX, true, MG_EY, true>(v, l.t, q % tx, q / tx, b, l.x, nxc, nyc, bc, mg_xs);
      else mgt_down<LMAX, false, MG_EY, true>(v, l.t, q % tx, q / tx, b, l.x, nxc, nyc, bc, mg_xs);
    }
    mg_cluster_sync();
  }
  {  // coarsest: x = C b, a warp per row, b in shared memory (at most LMAX x 64 values)
    const float* b = k0 == nl - 1 ? b0 : sl[nl - 1 - k0].b;
    float* x = sl[nl - 1 - k0].x;
    for (int j = t; j < nc; j += MGT_EX * MG_EY) mg_xs[j] = __ldcg(b + j);
    __syncthreads();
    const int nw = MGT_EX * MG_EY / 32, lane = t & 31;
    for (int row = blockIdx.x * nw + (t >> 5); row < nc; row += nw * gridDim.x) {
      float acc = 0.f;
#pragma unroll 8
      for (int j = lane; j < nc; j += 32) acc += __ldg(cinv + (long long)row * nc + j) * mg_xs[j];
      acc = warp_sum(acc);
      if (lane == 0) x[row] = acc;
    }
    if (nl - 1 > k0) mg_cluster_sync();
  }
  for (int k = nl - 2; k >= k0; --k) {
    const MGCLev<LMAX>& l = sl[k - k0];
    const int nxc = (l.nx + 1) / 2, nyc = (l.ny + 1) / 2, tx = (l.nx + MGT_EX - 3) / (MGT_EX - 2);
    const MGDev v{l.nx, l.ny, L, l.gx, l.gy, l.gz, l.s, l.m, l.w};
    const MGCLev<LMAX>& c = sl[k + 1 - k0];
    const float *b = k == k0 ? b0 : l.b, *xc = k + 1 == nl - 1 ? c.x : c.xt;
    float* out = k == 0 ? z : l.xt;
    for (int q = blockIdx.x; q < mgt_tiles<MG_EY>(l.nx, l.ny); q += gridDim.x) {
      __syncthreads();
      float rz;
      if (l.uni) rz = mgt_up<LMAX, true, MG_EY, true, true>(v, l.t, q % tx, q / tx, b, l.x, xc, nxc, nyc, out, mg_xs);
      else rz = mgt_up<LMAX, false, MG_EY, true, true>(v, l.t, q % tx, q / tx, b, l.x, xc, nxc, nyc, out, mg_xs);
      if (k == 0) sum2_add(part[0], rz);
    }
    if (k > k0) mg_cluster_sync();
  }
  if (k0 != 0) return;
  double tot[1];
  if (!grid_reduce<Sum2, 1>(part, partials, stride, counter, tot)) return;
  ctl->rz_next = tot[0];
  ctl_set_beta(ctl);
}

// coarsest level: x = C b with the dense inverse C (n x n, FP32), a warp per row
__global__ void __launch_bounds__(256) k_mg_coarsest(const Ctl* ctl, int n, const float* __restrict__ C,
                                                     const float* __restrict__ b, float* __restrict__ x) {
  grid_dep_enter();
  if (ld_int(&ctl->done)) return;
  const int nw = blockDim.x >> 5;
  mg_coarsest_rows(n, C, b, x, blockIdx.x * nw + (threadIdx.x >> 5), nw * gridDim.x);
}

// r^T z with FP32 products and FP64 sums, then beta (the preconditioner's dot
// product); grid-stride over a few resident blocks per SM, so that the last-block
// reduction sums few partials
__global__ void __launch_bounds__(256) k_mg_rz(long long n, Ctl* ctl, const float* __restrict__ r,
                                               const float* __restrict__ z, double* partials, int stride,
                                               unsigned* counter) {
  grid_dep_enter();
  if (ld_int(&ctl->done)) return;
  const long long step = (long long)gridDim.x * blockDim.x, t0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long n4 = n / 4;
  const float4* r4 = reinterpret_cast<const float4*>(r);
  const float4* z4p = reinterpret_cast<const float4*>(z);
  float v[1] = {0.f};
  for (long long q = t0; q < n4; q += step) {
    const float4 a = __ldcg(r4 + q), b = __ldcg(z4p + q);
    v[0] += a.x * b.x + a.y * b.y + a.z * b.z + a.w * b.w;
  }
  for (long long i = 4 * n4 + t0; i < n; i += step) v[0] += r[i] * z[i];
  double tot[1];
  if (!grid_reduce<float, 1>(v, partials, stride, counter, tot)) return;
  ctl->rz_next = tot[0];
  ctl_set_beta(ctl);
}

// ---------------------------------------------------------------- coarsest inverse
// The coarsest operator's dense inverse, in FP64 on the device.  Unknowns are ordered
// layer fastest, then the shorter in-plane side, so the matrix is a band of half width
// bw = L min(nx, ny) <= 8 L: A = Lu D Lu^T costs n bw^2 / 2 instead of a dense
// factorisation's n^3 / 3, and a column of the inverse 2 n bw.  A hierarchy is rebuilt
// whenever the conductivities change, as every pass of a conductivity gradient does:
// dense Cholesky and inversion on the host made such a pass (1024 x 1024 x 10, solve and
// gradient) 346 ms, with this pair of kernels it takes 75.8 ms; the first call on a batch
// of 32 stacks went from 2.47 to 0.23 s.
__device__ __forceinline__ int mg_band_index(int nx, int ny, int L, int x, int y, int z) {
  return z + L * (nx <= ny ? x + nx * y : y + ny * x);
}

// Right-looking L D L^T by one block: column j's update of its bw x bw window is spread
// over the block.  lr[i][k - i + bw] and lt[k][i - k] hold the unit lower factor by rows
// and by columns, rinv the inverse pivots; *bad is set when a pivot is not positive.
__global__ void __launch_bounds__(1024)
    k_mg_band_factor(int nx, int ny, int L, int bw, const float* __restrict__ gx, const float* __restrict__ gy,
                     const float* __restrict__ gz, const float* __restrict__ s, double* lr, double* lt, double* rinv,
                     int* bad) {
  __shared__ double col[TH_MAXL * MG_COARSEST];
  __shared__ double piv;
  const int n = nx * ny * L, w = bw + 1, t = threadIdx.x, nt = blockDim.x;
  for (int i = t; i < n * w; i += nt) {
    lr[i] = 0.0;
    lt[i] = 0.0;
  }
  if (t == 0) *bad = 0;
  __syncthreads();
  for (int c = t; c < n; c += nt) {
    const int x = c % nx, y = (c / nx) % ny, z = c / (nx * ny);
    const int q = mg_band_index(nx, ny, L, x, y, z);
    double dg = s[c];
    auto couple = [&](int xx, int yy, int zz, double g) {
      dg += g;
      const int k = mg_band_index(nx, ny, L, xx, yy, zz);
      if (k < q) lr[q * w + (k - q + bw)] = -g;
    };
    if (x + 1 < nx) couple(x + 1, y, z, gx[c]);
    if (x > 0) couple(x - 1, y, z, gx[c - 1]);
    if (y + 1 < ny) couple(x, y + 1, z, gy[c]);
    if (y > 0) couple(x, y - 1, z, gy[c - nx]);
    if (z + 1 < L) couple(x, y, z + 1, gz[c]);
    if (z > 0) couple(x, y, z - 1, gz[c - nx * ny]);
    lr[q * w + bw] = dg;
  }
  __syncthreads();
  const int tx = t & 31, ty = t >> 5, ny32 = nt >> 5;
  for (int j = 0; j < n; ++j) {
    const int m = min(bw, n - 1 - j);  // rows below the pivot inside the band
    for (int i = t; i < m; i += nt) col[i] = lr[(j + 1 + i) * w + (bw - 1 - i)];
    if (t == nt - 1) {
      const double d = lr[j * w + bw];
      if (!(d > 0.0)) *bad = 1;
      piv = 1.0 / d;
      rinv[j] = piv;
    }
    __syncthreads();
    const double p = piv;
    for (int i = ty; i < m; i += ny32) {
      const double li = col[i] * p;
      double* row = lr + (j + 1 + i) * w + (bw - 1 - i);  // entries (j+1+i, j), (j+1+i, j+1), ...
      if (tx == 0) {
        row[0] = li;
        lt[j * w + (i + 1)] = li;
      }
      for (int k = tx; k <= i; k += 32) row[1 + k] -= li * col[k];
    }
    __syncthreads();
  }
}

// One warp per column of the inverse: forward and backward substitution through the
// band (lanes split a row's bw products), the column in shared memory.
__global__ void k_mg_band_inverse(int nx, int ny, int L, int bw, const double* __restrict__ lr,
                                  const double* __restrict__ lt, const double* __restrict__ rinv,
                                  float* __restrict__ cinv) {
  extern __shared__ double mg_cols[];
  const int n = nx * ny * L, w = bw + 1, lane = threadIdx.x & 31;
  const int c = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);  // cell of the right-hand side
  if (c >= n) return;
  double* y = mg_cols + (size_t)(threadIdx.x >> 5) * n;
  const int q = mg_band_index(nx, ny, L, c % nx, (c / nx) % ny, c / (nx * ny));
  for (int i = lane; i < n; i += 32) y[i] = i == q ? 1.0 : 0.0;
  __syncwarp();
  for (int i = q + 1; i < n; ++i) {
    double a = 0.0;
    for (int k = max(q, i - bw) + lane; k < i; k += 32) a += lr[i * w + (k - i + bw)] * y[k];
    a = warp_sum(a);
    if (lane == 0) y[i] = -a;
    __syncwarp();
  }
  for (int i = lane; i < n; i += 32) y[i] *= rinv[i];
  __syncwarp();
  for (int i = n - 2; i >= 0; --i) {
    double a = 0.0;
    const int m = min(bw, n - 1 - i);
    for (int k = 1 + lane; k <= m; k += 32) a += lt[i * w + k] * y[i + k];
    a = warp_sum(a);
    if (lane == 0) y[i] -= a;
    __syncwarp();
  }
  for (int i = lane; i < n; i += 32)  // the inverse is symmetric: column c stored as row c
    cinv[(size_t)c * n + i] = (float)y[mg_band_index(nx, ny, L, i % nx, (i / nx) % ny, i / (nx * ny))];
}

dim3 col_grid(int nx, int ny) { return dim3((nx + 31) / 32, (ny + 7) / 8, 1); }

}  // namespace

struct MGLevelH {
  int nx = 0, ny = 0;
  long long n = 0;
  const float *gx = nullptr, *gy = nullptr, *gz = nullptr;  // level 0: the grid's FP32 faces
  float *own_gx = nullptr, *own_gy = nullptr, *own_gz = nullptr;
  float *s = nullptr;
  float *m = nullptr, *w = nullptr;  // Thomas factors, from the first time the level is not layer-uniform
  float *x = nullptr, *xt = nullptr, *b = nullptr;
};

struct MGHier {
  double dt = -1.0;
  std::vector<MGLevelH> lv;
  int cluster = 0;    // blocks of k_mg_levels' cluster (0: not looked up yet)
  bool whole = true;  // the current call's stream has all SMs
  // Levels whose coefficients depend only on the layer (and on which in-plane
  // neighbours exist): the finest level of a layer-uniform grid and every coarser
  // level reached through complete 2 x 2 aggregates (even nx, ny above it).  Their
  // tables replace the per-cell arrays in the smoother and the restriction.
  std::vector<char> luni;
  std::vector<MGUni<32>> ltab;
  float* cinv = nullptr;  // dense inverse of the coarsest operator
  void* dlv = nullptr;       // levels for k_mg_levels (MGCLev<LMAX> of the stack's layer capacity)
  double* band = nullptr;  // its banded factor (rows, columns, 1/d) and the factorisation's flag
  int nc = 0;
  ~MGHier() {
    for (auto& l : lv) {
      for (float* p : {l.own_gx, l.own_gy, l.own_gz, l.s, l.m, l.w, l.x, l.xt, l.b})
        if (p) cudaFree(p);
    }
    if (cinv) cudaFree(cinv);
    if (band) cudaFree(band);
    if (dlv) cudaFree(dlv);
  }
};

void mg_free(MGHier* h) { delete h; }

static th_status mg_alloc(float** p, long long n) {
  if (cudaMalloc((void**)p, sizeof(float) * (size_t)std::max(n, 1LL)) != cudaSuccess) {
    cudaGetLastError();
    return th_fail(TH_ENOMEM, "multigrid level allocation failed");
  }
  return TH_OK;
}

static MGDev dev_of(const MGLevelH& l, int L) { return MGDev{l.nx, l.ny, L, l.gx, l.gy, l.gz, l.s, l.m, l.w}; }

// layer capacity of the kernels
static int mg_lmax(int L) { return L <= 4 ? 4 : (L <= 6 ? 6 : (L <= 8 ? 8 : (L <= 12 ? 12 : (L <= 16 ? 16 : 32)))); }
#define MG_LMAX(L, STMT)                                                                             \
  switch (mg_lmax(L)) {                                                                              \
    case 4: { constexpr int LM = 4; STMT; break; }                                                   \
    case 6: { constexpr int LM = 6; STMT; break; }                                                   \
    case 8: { constexpr int LM = 8; STMT; break; }                                                   \
    case 12: { constexpr int LM = 12; STMT; break; }                                                 \
    case 16: { constexpr int LM = 16; STMT; break; }                                                 \
    default: { constexpr int LM = 32; STMT; break; }                                                 \
  }

template <int LMAX>
static th_status mg_upload(thermal_grid* g, cudaStream_t s);

th_status grid_ensure_mg(thermal_grid* g, double dt, cudaStream_t s) {
  TH_TRY(grid_ensure_tab(g, dt, s));
  const double key = dt > 0.0 ? dt : 0.0;
  if (g->mg && g->mg_valid && g->mg->dt == key) return TH_OK;
  if (g->L > 32) return th_fail(TH_EINVAL, "multigrid supports at most 32 layers");
  g->mg_valid = false;  // until the rebuild below is complete
  if (!g->mg) {
    auto h = std::make_unique<MGHier>();  // the grid's once every level has its memory
    int nx = g->nx, ny = g->ny;
    while (true) {
      MGLevelH l;
      l.nx = nx;
      l.ny = ny;
      l.n = (long long)nx * ny * g->L;
      h->lv.push_back(l);
      if (std::max(nx, ny) <= MG_COARSEST) break;
      nx = (nx + 1) / 2;
      ny = (ny + 1) / 2;
    }
    for (size_t k = 0; k < h->lv.size(); ++k) {
      MGLevelH& l = h->lv[k];
      TH_TRY(mg_alloc(&l.s, l.n));
      TH_TRY(mg_alloc(&l.xt, l.n));
      if (k == 0) {
        l.gx = g->f32.gx;
        l.gy = g->f32.gy;
        l.gz = g->f32.gz;
      } else {
        TH_TRY(mg_alloc(&l.own_gx, l.n));
        TH_TRY(mg_alloc(&l.own_gy, l.n));
        TH_TRY(mg_alloc(&l.own_gz, l.n));
        l.gx = l.own_gx;
        l.gy = l.own_gy;
        l.gz = l.own_gz;
        TH_TRY(mg_alloc(&l.x, l.n));
        TH_TRY(mg_alloc(&l.b, l.n));
      }
    }
    g->mg = h.release();
  }
  MGHier* h = g->mg;
  const int L = g->L;
  k_mg_s0<<<grid_blocks(g), dim3(TH_BX, TH_BY), 0, s>>>(grid_dims(g), g->tab, h->lv[0].s);
  TH_CHECK_LAUNCH();
  for (size_t k = 0; k + 1 < h->lv.size(); ++k) {
    const MGLevelH& f = h->lv[k];
    MGLevelH& c = h->lv[k + 1];
    const dim3 gr((c.nx + 31) / 32, (c.ny + 7) / 8, L);
    k_mg_coarsen<<<gr, dim3(32, 8), 0, s>>>(f.nx, f.ny, c.nx, c.ny, L, f.gx, f.gy, f.gz, f.s, c.own_gx, c.own_gy,
                                            c.own_gz, c.s);
    TH_CHECK_LAUNCH();
  }
  // layer-uniform levels: coefficients and Thomas factors per in-plane case
  const size_t nlv = h->lv.size();
  h->luni.assign(nlv, 0);
  h->ltab.assign(nlv, MGUni<32>{});
  auto factors = [&](MGUni<32>& t) {
    for (int nyf = 0; nyf < 3; ++nyf)
      for (int nxf = 0; nxf < 3; ++nxf) {
        const int c = nxf + 3 * nyf;
        double wprev = 0.0;
        for (int z = 0; z < L; ++z) {  // the order of k_mg_zfactors: s, x faces, y faces, z faces
          double b = t.s[z];
          for (int q = 0; q < nxf; ++q) b += t.gx[z];
          for (int q = 0; q < nyf; ++q) b += t.gy[z];
          if (z + 1 < L) b += t.gz[z];
          const double gb = (z > 0) ? (double)t.gz[z - 1] : 0.0;
          if (z > 0) b += gb;
          const double mz = 1.0 / (b - gb * wprev);
          const double wz = (z + 1 < L) ? (double)t.gz[z] * mz : 0.0;
          t.m[c][z] = (float)mz;
          t.w[c][z] = (float)wz;
          wprev = wz;
        }
      }
  };
  if (g->uniform) {
    const LayerTab& T = g->tab_host;
    MGUni<32>& t0 = h->ltab[0];
    std::memset(&t0, 0, sizeof(t0));
    for (int z = 0; z < L; ++z) {
      t0.s[z] = T.s32[z];
      t0.gx[z] = T.gxl[z];
      t0.gy[z] = T.gyl[z];
      t0.gz[z] = (z + 1 < L) ? T.gzl[z] : 0.f;
    }
    factors(t0);
    h->luni[0] = 1;
    // a coarse level of complete 2 x 2 aggregates: per-cell term and vertical face
    // summed over the 4 fine cells, in-plane faces over the 2 crossing ones (FP32, in
    // k_mg_coarsen's order, so the table equals the per-cell arrays)
    for (size_t k = 0; k + 1 < nlv; ++k) {
      if (!h->luni[k] || h->lv[k].nx % 2 != 0 || h->lv[k].ny % 2 != 0) break;
      const MGUni<32>& f = h->ltab[k];
      MGUni<32>& t = h->ltab[k + 1];
      std::memset(&t, 0, sizeof(t));
      for (int z = 0; z < L; ++z) {
        float sz = 0.f, gz = 0.f;
        for (int q = 0; q < 4; ++q) {
          sz += f.s[z];
          gz += f.gz[z];
        }
        t.s[z] = sz;
        t.gz[z] = gz;
        t.gx[z] = f.gx[z] + f.gx[z];
        t.gy[z] = f.gy[z] + f.gy[z];
      }
      factors(t);
      h->luni[k + 1] = 1;
    }
  }
  for (size_t k = 0; k < nlv; ++k) {  // a layer-uniform level's factors are in its table
    MGLevelH& l = h->lv[k];
    if (h->luni[k]) continue;
    if (!l.m) TH_TRY(mg_alloc(&l.m, l.n));
    if (!l.w) TH_TRY(mg_alloc(&l.w, l.n));
    k_mg_zfactors<<<col_grid(l.nx, l.ny), dim3(32, 8), 0, s>>>(l.nx, l.ny, L, l.gx, l.gy, l.gz, l.s, l.m, l.w);
    TH_CHECK_LAUNCH();
  }
  // dense inverse of the coarsest operator (at most MG_COARSEST^2 columns x L layers)
  const MGLevelH& c = h->lv.back();
  const int nc = (int)c.n, bw = L * std::min(c.nx, c.ny);
  if (!h->cinv) TH_TRY(mg_alloc(&h->cinv, (long long)nc * nc));
  if (!h->band) {
    if (cudaMalloc((void**)&h->band, sizeof(double) * ((size_t)2 * nc * (bw + 1) + nc) + sizeof(int)) != cudaSuccess) {
      cudaGetLastError();
      h->band = nullptr;
      return th_fail(TH_ENOMEM, "multigrid coarsest factor allocation failed");
    }
  }
  h->nc = nc;
  double* lt = h->band + (size_t)nc * (bw + 1);
  double* rinv = lt + (size_t)nc * (bw + 1);
  int* bad = (int*)(rinv + nc);
  k_mg_band_factor<<<1, 1024, 0, s>>>(c.nx, c.ny, L, bw, c.gx, c.gy, c.gz, c.s, h->band, lt, rinv, bad);
  TH_CHECK_LAUNCH();
  const size_t ysm = sizeof(double) * (size_t)nc;
  const int warps = (int)std::max<size_t>(1, std::min<size_t>(4, (size_t)(48 << 10) / ysm));
  k_mg_band_inverse<<<(nc + warps - 1) / warps, 32 * warps, warps * ysm, s>>>(c.nx, c.ny, L, bw, h->band, lt, rinv,
                                                                             h->cinv);
  TH_CHECK_LAUNCH();
  int hbad = 0;
  TH_CUDA(cudaMemcpyAsync(&hbad, bad, sizeof(int), cudaMemcpyDeviceToHost, s));
  TH_CUDA(cudaStreamSynchronize(s));
  if (hbad) return th_fail(TH_ENOCONV, "coarsest multigrid operator is not positive definite");
  MG_LMAX(L, TH_TRY(mg_upload<LM>(g, s)));
  h->dt = key;
  g->mg_valid = true;
  return TH_OK;
}

bool mg_set_stream(thermal_grid* g, cudaStream_t s) {
  g->mg->whole = stream_sms(s) >= device_sms();
  return g->mg->whole;
}

// the table of level k (layer-uniform levels only)
template <int LMAX>
static MGUni<LMAX> uni_of(const MGHier* h, int k) {
  MGUni<LMAX> u;
  std::memset(&u, 0, sizeof(u));
  const MGUni<32>& t = h->ltab[k];
  for (int z = 0; z < LMAX; ++z) {
    u.s[z] = t.s[z];
    u.gx[z] = t.gx[z];
    u.gy[z] = t.gy[z];
    u.gz[z] = t.gz[z];
    for (int c = 0; c < 9; ++c) {
      u.m[c][z] = t.m[c][z];
      u.w[c][z] = t.w[c][z];
    }
  }
  return u;
}

static bool mg_uni(const MGHier* h, int k) { return k < (int)h->luni.size() && h->luni[k]; }

// level descriptors and tables for k_mg_levels
template <int LMAX>
static th_status mg_upload(thermal_grid* g, cudaStream_t s) {
  MGHier* h = g->mg;
  const int nl = (int)h->lv.size();
  std::vector<MGCLev<LMAX>> d(nl);
  std::memset((void*)d.data(), 0, sizeof(MGCLev<LMAX>) * nl);
  for (int k = 0; k < nl; ++k) {
    const MGLevelH& l = h->lv[k];
    MGCLev<LMAX>& o = d[k];
    o.nx = l.nx;
    o.ny = l.ny;
    o.uni = mg_uni(h, k);
    o.gx = l.gx;
    o.gy = l.gy;
    o.gz = l.gz;
    o.s = l.s;
    o.m = l.m;
    o.w = l.w;
    o.x = k == 0 ? l.xt : l.x;  // the pre-smoothed iterate
    o.xt = l.xt;
    o.b = l.b;
    if (o.uni) o.t = uni_of<LMAX>(h, k);
  }
  auto al = [](void** p, size_t bytes) -> th_status {
    if (*p || cudaMalloc(p, bytes) == cudaSuccess) return TH_OK;
    cudaGetLastError();
    *p = nullptr;
    return th_fail(TH_ENOMEM, "multigrid level table allocation failed");
  };
  TH_TRY(al(&h->dlv, sizeof(MGCLev<LMAX>) * nl));
  TH_CUDA(cudaMemcpyAsync(h->dlv, d.data(), sizeof(MGCLev<LMAX>) * nl, cudaMemcpyHostToDevice, s));
  TH_CUDA(cudaStreamSynchronize(s));
  return TH_OK;
}

// levels k0 .. of the cycle by one cluster
template <int LMAX>
static th_status mg_levels(thermal_grid* g, int k0, const float* b0, float* z, cudaStream_t s) {
  MGHier* h = g->mg;
  const int nl = (int)h->lv.size();
  auto* kern = k_mg_levels<LMAX>;
  cudaLaunchConfig_t c{};
  c.blockDim = dim3(MGT_EX, MG_EY);
  c.dynamicSmemBytes = mg_xs_bytes<LMAX>() + sizeof(MGCLev<LMAX>) * (nl - k0);
  c.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  c.attrs = &at;
  c.numAttrs = 1;
  TH_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)c.dynamicSmemBytes));
  TH_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  auto blocks = [&](int n) {
    c.gridDim = dim3(n);
    at.val.clusterDim.x = n;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
  };
  blocks(MG_CLUSTER);
  if (!h->cluster) {  // once per hierarchy
    int fits = 0;
    if (cudaOccupancyMaxActiveClusters(&fits, kern, &c) != cudaSuccess) cudaGetLastError();
    h->cluster = fits > 0 ? MG_CLUSTER : 8;
  }
  blocks(h->whole ? h->cluster : 1);
  TH_CUDA(cudaLaunchKernelEx(&c, kern, g->ctl, (const MGCLev<LMAX>*)h->dlv, g->L, k0, nl, h->nc, (const float*)h->cinv,
                             b0, z, g->partials, g->partials_stride, g->counters));
  return TH_OK;
}

// one half of level k as a launch of its own
template <int LMAX, bool UNI>
static th_status mg_half(thermal_grid* g, int k, bool up, const float* b, float* x, const float* xc, float* z,
                         cudaStream_t s) {
  const MGHier* h = g->mg;
  const MGLevelH &l = h->lv[k], &c = h->lv[k + 1];
  const MGUni<LMAX> U = uni_of<LMAX>(h, k);
  const dim3 gr = mg_tile_grid(l.nx, l.ny), bl(MGT_EX, MG_EY);
  constexpr size_t sm = mg_xs_bytes<LMAX>();
  static_assert(sm <= (40u << 10), "a tile needs the opt-in for larger shared memory");
  auto launch = [&](auto* kern, dim3 blocks, auto... a) -> th_status {
    th_launch(kern, blocks, bl, sm, s, a...);
    TH_CHECK_LAUNCH();
    return TH_OK;
  };
  if (!up) return launch(k_mg_down<LMAX, UNI>, gr, g->ctl, dev_of(l, g->L), U, b, x, c.nx, c.ny, c.b);
  if (k == 0)
    return launch(k_mg_up<LMAX, UNI, true>,
                  std::min(mgt_tiles<MG_EY>(l.nx, l.ny), (LMAX <= 12 ? (int)MG_MINB : 1) * device_sms()), g->ctl,
                  dev_of(l, g->L), U, b, x, xc, c.nx, c.ny, z, g->partials, g->partials_stride, g->counters);
  return launch(k_mg_up<LMAX, UNI, false>, gr, g->ctl, dev_of(l, g->L), U, b, x, xc, c.nx, c.ny, z, g->partials,
                g->partials_stride, g->counters);
}

template <int LMAX>
static th_status mg_cycle(thermal_grid* g, const float* r, float* z, cudaStream_t s) {
  MGHier* h = g->mg;
  const int nl = (int)h->lv.size();
  auto half = [&](int k, bool up) -> th_status {
    const MGLevelH& l = h->lv[k];
    const float* b = k == 0 ? r : l.b;
    float* x = k == 0 ? l.xt : l.x;  // the pre-smoothed iterate
    const float* xc = k + 1 == nl - 1 ? h->lv[k + 1].x : h->lv[k + 1].xt;
    float* out = k == 0 ? z : l.xt;
    return mg_uni(h, k) ? mg_half<LMAX, true>(g, k, up, b, x, xc, out, s)
                        : mg_half<LMAX, false>(g, k, up, b, x, xc, out, s);
  };
  // first level of the cluster's: at most two tiles a block (so a 64 x 64 level, of 33 tiles,
  // is not).  V-cycles (us) at two / three / four / eight: 64^2 x 4 18.8 / 20.5 / 20.5 / 20.5,
  // 200 x 150 x 8 38.9 / 38.9 / 45.1 / 45.1, 512^2 x 8 60.1 / 63.2 / 63.3 / 77.9, 1024^2 x 10
  // 180.7 / 186.4 / 186.5 / 205.3
  int k0 = 0;
  while (k0 < nl - 1 && mgt_tiles<MG_EY>(h->lv[k0].nx, h->lv[k0].ny) > 2 * MG_CLUSTER) ++k0;
  for (int k = 0; k < k0; ++k) TH_TRY(half(k, false));
  TH_TRY(mg_levels<LMAX>(g, k0, k0 == 0 ? r : h->lv[k0].b, z, s));
  for (int k = k0 - 1; k >= 0; --k) TH_TRY(half(k, true));
  return TH_OK;
}

static th_status mg_rz(thermal_grid* g, const float* r, const float* z, cudaStream_t s);

// z = M^-1 r: one V-cycle (see the file comment), r^T z and beta.
th_status mg_vcycle(thermal_grid* g, const float* r, float* z, cudaStream_t s) {
  MGHier* h = g->mg;
  if (!h || !g->mg_valid) return th_fail(TH_ESTATE, "multigrid hierarchy not built");
  if (h->lv.size() == 1) {
    th_launch(k_mg_coarsest, (h->nc + 7) / 8, 256, 0, s, g->ctl, h->nc, h->cinv, r, z);
    TH_CHECK_LAUNCH();
    return mg_rz(g, r, z, s);
  }
  MG_LMAX(g->L, return mg_cycle<LM>(g, r, z, s));
  return TH_OK;
}

// r^T z of a single-level grid's exact solve
static th_status mg_rz(thermal_grid* g, const float* r, const float* z, cudaStream_t s) {
  const long long n = g->n;
  static int sms[64] = {0};
  int dev = 0;
  TH_CUDA(cudaGetDevice(&dev));
  if (dev >= 0 && dev < 64 && sms[dev] == 0) TH_CUDA(cudaDeviceGetAttribute(&sms[dev], cudaDevAttrMultiProcessorCount, dev));
  const long long want = (n / 4 + 255) / 256;
  const int per = (dev >= 0 && dev < 64 && sms[dev] > 0) ? 4 * sms[dev] : 608;
  const unsigned nb = (unsigned)std::max(1LL, std::min<long long>(want, std::min(per, g->partials_stride)));
  th_launch(k_mg_rz, nb, 256, 0, s, n, g->ctl, r, z, g->partials, g->partials_stride, g->counters);
  TH_CHECK_LAUNCH();
  return TH_OK;
}

th_status mg_batch_levels(thermal_grid* g, MGBDesc* out, cudaStream_t s) {
  TH_TRY(grid_ensure_mg(g, 0.0, s));
  const MGHier* h = g->mg;
  const int nl = (int)h->lv.size();
  if (nl > MG_BMAXL) return th_fail(TH_EINVAL, "multigrid hierarchy deeper than %d levels", MG_BMAXL);
  std::memset(out, 0, sizeof(*out));
  out->nl = nl;
  out->nc = h->nc;
  out->cinv = h->cinv;
  for (int k = 0; k < nl; ++k) {
    const MGLevelH& l = h->lv[k];
    MGBLevel& d = out->lv[k];
    d.nx = l.nx;
    d.ny = l.ny;
    d.gx = l.gx;
    d.gy = l.gy;
    d.gz = l.gz;
    d.s = l.s;
    d.m = l.m;
    d.w = l.w;
    d.x = l.x;
    d.xt = l.xt;
    d.b = l.b;
    d.uni = (g->L <= 8 && mg_uni(h, k)) ? 1 : 0;
    if (d.uni) d.t = uni_of<8>(h, k);
  }
  return TH_OK;
}
