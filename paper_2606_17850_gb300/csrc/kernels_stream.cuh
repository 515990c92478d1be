// Fused Chebyshev steps of large layer-uniform grids as register streams along y.
//
// S <= TB_H steps of the polynomial run in one launch.  A warp owns a strip of 64 columns
// (a lane two neighbouring ones, as one operand of the paired FP32 instructions; the inner
// ST_TX columns are results, ST_X0 on either side are halo that is recomputed) and marches
// along y.  At row t it takes in row t of z_m and, as a pipeline, forms row t - s of z_{m+s}
// for s = 1..S: step s needs rows t - s - 1, t - s and t - s + 1 of z_{m+s-1}, and the last
// of these was formed by step s - 1 in the same iteration.  So each level keeps two rows in
// registers (all layers): the y and z neighbours are the thread's own, and only two values
// per layer and row cross lanes, as warp shuffles.  No block barrier and no shared-memory
// plane; the halo in y is only the 2 S rows that a strip starts with.
//
// The product is taken in expanded form, r - A v = r - d v + gx (v_E + v_W) + gy (v_N + v_S)
// + gzu v_U + gzd v_D, with d the diagonal of a cell that has all four in-plane faces; an
// absent neighbour counts as the cell itself.  Columns, rows and layers outside the grid
// hold zeros: their inverse diagonal is 0, so a step leaves them 0.
//
// Rows arrive in a shared-memory ring ST_PF rows ahead by the tensor memory accelerator:
// one lane issues a 64 x 1 x L box per vector and row, completion on an mbarrier per ring
// slot, cells outside the grid filled with zeros (nx % 4 == 0 gives the row pitch it needs).
// A block is one warp, so that everything about the march is uniform.  The rows' registers
// are shifted by moves: rotating them by name over three unrolled rows (no moves) made the
// loop 30 KB of code and stalled on its fetch (45.0 instead of 38.3 us).
//
// Measured, four steps on 1024^2 x 8 / x 6 / x 4 and 2048^2 x 8: 55.5 / 53.5 / 50.6 / 198 us
// with 24 x 24-column tiles (shared-memory bound, k_cheb_tb), 38.3 / 32.9 / 23.2 / 115 us
// here.  One column a lane, layers paired: 50 us (twice the shuffles and a third of a
// strip halo).  Bound by issue and, at 16 rows a strip, by the 8 rows a strip starts with;
// at 2048^2 it moves 168 MB x 4 in 115 us, 5.8 TB/s.
#pragma once

#include <cuda.h>

#include "kernels_tb.cuh"

#define ST_PF 1     // rows in flight ahead of the current one (2: one warp less fits an SM, 39.5 us)
#define ST_X0 4     // halo columns on either side (a 16-byte boundary for the tensor copies)
#define ST_TX 56    // result columns of a strip
#define ST_BW 64    // columns of a strip

template <int LMAX>
struct __align__(8) STParams {
  float2 c1[TB_H], c2[TB_H];       // step coefficients of this chunk, (c, c)
  float2 nd[LMAX];                 // -(diagonal of a cell with all four in-plane faces)
  float2 gx[LMAX], gy[LMAX];       // in-plane face conductances
  float2 gzu[LMAX], gzd[LMAX];     // face to the layer above / below, 0 at the ends
  float invd[9][LMAX];             // 1 / diagonal for (x faces present) + 3 (y faces present)
  float z1s;                       // first chunk: z_1 = z1s D^-1 r
  int expire_test;                 // test hook: the first wait of each warp runs out
};

// ring slots: z_m and z_{m-1} live two rows (the current and the one before), r lives
// until step S has used it
constexpr int st_nz() { return ST_PF + 2; }
template <int S> constexpr int st_nr() { return ST_PF + 1 + S; }
template <int LMAX, int S, bool FIRST>
constexpr size_t st_smem_bytes() {
  return (size_t)LMAX * ST_BW * (st_nr<S>() + (FIRST ? 0 : 2 * st_nz())) * sizeof(float) + 8 * (1 + st_nz()) + 128;
}

template <int V> struct StInt { static constexpr int v = V; };

// STEPS of k_cheb_tb: inner chunk (z_m, z_{m-1}, r in; z_{m+S}, z_{m+S-1} out); FIRST: the
// chunk starts the polynomial, z_1 = z1s D^-1 r and z_0 = 0 formed from r; LAST: no z_{m+S-1},
// r^T z reduced.
template <int LMAX, int S, bool LAST, bool FIRST>
__global__ void __launch_bounds__(32, LMAX <= 4 ? 14 : (LMAX <= 6 ? 10 : 8))
    k_cheb_st(Dims d, int nsx, int R, Ctl* ctl, const __grid_constant__ CUtensorMap m_cur,
              const __grid_constant__ CUtensorMap m_prev, const __grid_constant__ CUtensorMap m_r,
              float* __restrict__ out_cur, float* __restrict__ out_prev, const __grid_constant__ STParams<LMAX> P,
              double* partials, int stride, unsigned* counter) {
  grid_dep_enter();
  constexpr int NZ = st_nz(), NR = st_nr<S>(), ROW = LMAX * ST_BW;
  extern __shared__ __align__(128) float tb_dyn[];
  const int lane = threadIdx.x;
  float* rr_ring = tb_dyn + (((128u - (tb_smem(tb_dyn) & 127u)) & 127u) >> 2);  // [NR][LMAX][64]
  float* zc_ring = rr_ring + NR * ROW;                                          // [NZ][LMAX][64]
  float* zp_ring = zc_ring + (FIRST ? 0 : NZ * ROW);
  unsigned long long* bars = (unsigned long long*)(zp_ring + (FIRST ? 0 : NZ * ROW));
  unsigned long long* bar = bars + 1;  // bars[0]: the test hook's, never completed
  const int L = d.L, nx = d.nx, ny = d.ny;
  Sum2 part[1] = {{0.f, 0.f}};  // r^T z: a row's products as a tree, the rows with their rounding errors
  if (lane == 0) {
    for (int i = 0; i < 1 + NZ; ++i) tb_mbar_init(bars + i, 1);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  __syncthreads();
  const int sx = (int)blockIdx.x % nsx, sy = (int)blockIdx.x / nsx;
  const int xb = sx * ST_TX - ST_X0, gx = xb + 2 * lane;  // this lane: columns gx, gx + 1
  const int y0 = sy * R, y1 = min(y0 + R, ny);
  const int nit = (y1 - y0) + 2 * S;  // rows y0 - S .. y1 - 1 + S
  const bool inx = gx >= 0 && gx < nx;  // nx is even: both columns or none
  const unsigned row_bytes = (unsigned)(L * ST_BW * sizeof(float)) * (FIRST ? 1u : 3u);
  if (L < LMAX) {  // never written by the copies
    for (int i = lane; i < (LMAX - L) * ST_BW; i += 32) {
      for (int q = 0; q < NR; ++q) rr_ring[q * ROW + L * ST_BW + i] = 0.f;
      if (!FIRST)
        for (int q = 0; q < NZ; ++q) zc_ring[q * ROW + L * ST_BW + i] = zp_ring[q * ROW + L * ST_BW + i] = 0.f;
    }
  }
  int izs = 0, irs = 0, ii = 0;  // next row to fetch: its ring slots and its number
  auto fetch = [&]() {
    if (lane == 0 && ii < nit) {
      const int y = y0 - S + ii;
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      tb_mbar_expect(bar + izs, row_bytes);
      tb_tma_3d(rr_ring + irs * ROW, &m_r, xb, y, 0, bar + izs);
      if (!FIRST) {
        tb_tma_3d(zc_ring + izs * ROW, &m_cur, xb, y, 0, bar + izs);
        tb_tma_3d(zp_ring + izs * ROW, &m_prev, xb, y, 0, bar + izs);
      }
    }
    ++ii;
    if (++izs == NZ) izs = 0;
    if (++irs == NR) irs = 0;
  };
  for (int q = 0; q < ST_PF; ++q) fetch();
  // the first rows are on their way meanwhile
  const bool done = __shfl_sync(0xffffffffu, ld_int(&ctl->done), 0) != 0;

  // the columns' inverse diagonals; 0 outside the grid
  const int nxa = (gx > 0) + 1, nxb = 1 + (gx + 2 < nx);
  auto invd_of = [&](int nyf, int z) {
    return inx ? make_float2(P.invd[nxa + 3 * nyf][z], P.invd[nxb + 3 * nyf][z]) : make_float2(0.f, 0.f);
  };
  float2 iv[LMAX];
#pragma unroll
  for (int z = 0; z < LMAX; ++z) iv[z] = invd_of(2, z);
  const bool xe = xb < 0 || xb + ST_BW > nx;  // the strip holds an end of the rows (uniform)
  const bool endL = gx == 0, endR = gx + 2 == nx;
  const int le = min(lane + 1, 31), lw = max(lane - 1, 0);
  const float2 m1 = make_float2(-1.f, -1.f);
  const bool store_lane = lane >= ST_X0 / 2 && lane < (ST_X0 + ST_TX) / 2 && gx < nx;

  float2 Z[S][3][LMAX];
#pragma unroll
  for (int l = 0; l < S; ++l)
#pragma unroll
    for (int q = 0; q < 3; ++q)
#pragma unroll
      for (int z = 0; z < LMAX; ++z) Z[l][q][z] = make_float2(0.f, 0.f);

  bool ok = __all_sync(0xffffffffu, !P.expire_test || tb_mbar_wait(bars, 0u, TB_TEST_WAIT_NS));
  int lost = 0;  // the row whose wait ran out
  int it = 0, zs = 0, rs = 0;
  unsigned par = 0;
  unsigned off = 4u * (unsigned)(gx + nx * (y0 - 2 * S));  // bytes to the cell of the row that step S forms, in its layer

  // one row: GEN handles rows at and outside the y edges and the strip's first rows
  auto row = [&](auto gen) {
    constexpr int O = 0, M = 1, N = 2;  // older, middle and new row of a level
    constexpr bool GEN = decltype(gen)::v != 0;
    const int t = y0 - S + it;
    __syncwarp();  // every lane is done with the ring slots that the next fetch reuses
    if (ok) fetch();
    if (ok && !__all_sync(0xffffffffu, tb_mbar_wait(bar + zs, par))) {
      ok = false;
      lost = it;
    }
    const float2* rrow = reinterpret_cast<const float2*>(rr_ring + rs * ROW) + lane;
    const float2* zrow = reinterpret_cast<const float2*>(zc_ring + zs * ROW) + lane;
    const float2* prow = reinterpret_cast<const float2*>(zp_ring + (zs == 0 ? NZ - 1 : zs - 1) * ROW) + lane;  // row t - 1
#pragma unroll
    for (int z = 0; z < LMAX; ++z) {
      if (FIRST) {
        float2 i0 = iv[z];
        if (GEN) {
          const int ym = (t <= 0) + (t >= ny - 1);
          if (ym) i0 = (t < 0 || t >= ny) ? make_float2(0.f, 0.f) : invd_of(2 - ym, z);
        }
        Z[0][N][z] = __fmul2_rn(__fmul2_rn(rrow[z * (ST_BW / 2)], i0), make_float2(P.z1s, P.z1s));
      } else {
        Z[0][N][z] = zrow[z * (ST_BW / 2)];
      }
    }
#pragma unroll
    for (int s = 1; s <= S; ++s) {
      const int y = t - s;
      const int q = rs >= s ? rs - s : rs - s + NR;
      const float2* rq = reinterpret_cast<const float2*>(rr_ring + q * ROW) + lane;
      const bool inside = !GEN || (y >= 0 && y < ny && it >= 2 * s);
      float2 out[LMAX];
      if (inside) {
        const int ym = GEN ? (y == 0) + (y == ny - 1) : 0;  // absent y neighbours of this row
        const float2 ym2 = make_float2((float)ym, (float)ym);
#pragma unroll
        for (int z = 0; z < LMAX; ++z) {
          const float2 v = Z[s - 1][M][z];
          float w = __shfl_sync(0xffffffffu, v.y, lw), e = __shfl_sync(0xffffffffu, v.x, le);
          if (xe) {
            w = endL ? v.x : w;
            e = endR ? v.y : e;
          }
          float2 xs, ys = __fadd2_rn(Z[s - 1][O][z], Z[s - 1][N][z]);
          xs.x = w + v.y;
          xs.y = v.x + e;
          float2 i0 = iv[z];
          if (GEN && ym) {
            ys = __ffma2_rn(ym2, v, ys);
            i0 = invd_of(2 - ym, z);
          }
          float2 a = __ffma2_rn(P.nd[z], v, rq[z * (ST_BW / 2)]);
          a = __ffma2_rn(P.gx[z], xs, a);
          a = __ffma2_rn(P.gy[z], ys, a);
          if (z + 1 < LMAX) a = __ffma2_rn(P.gzu[z], Z[s - 1][M][z + 1 < LMAX ? z + 1 : z], a);
          if (z > 0) a = __ffma2_rn(P.gzd[z], Z[s - 1][M][z > 0 ? z - 1 : z], a);
          float2 dz;  // z_m - z_{m-1}
          if (s == 1) {
            if (FIRST) dz = v;
            else dz = __ffma2_rn(prow[z * (ST_BW / 2)], m1, v);
          } else {
            dz = __ffma2_rn(Z[s > 1 ? s - 2 : 0][O][z], m1, v);
          }
          out[z] = __ffma2_rn(P.c2[s - 1], __fmul2_rn(a, i0), __ffma2_rn(P.c1[s - 1], dz, v));
        }
      } else {
#pragma unroll
        for (int z = 0; z < LMAX; ++z) out[z] = make_float2(0.f, 0.f);
      }
      if (s < S) {
#pragma unroll
        for (int z = 0; z < LMAX; ++z) Z[s < S ? s : 0][N][z] = out[z];
      } else if ((!GEN || it >= 2 * S) && store_lane) {
#pragma unroll
        for (int z = 0; z < LMAX; ++z) {
          if (z < L) {
            *(float2*)((char*)(out_cur + d.pxy * z) + off) = out[z];
            if (!LAST) *(float2*)((char*)(out_prev + d.pxy * z) + off) = Z[S - 1][M][z];
          }
        }
        if (LAST) {  // (layers beyond the stack's are zeros)
#pragma unroll
          for (int z = 0; z < LMAX; ++z) out[z] = __fmul2_rn(rq[z * (ST_BW / 2)], out[z]);
          sum2_add(part[0], pair_sum(out));
        }
      }
    }
    off += 4u * (unsigned)nx;
    ++it;
    if (++zs == NZ) {
      zs = 0;
      par ^= 1u;
    }
    if (++rs == NR) rs = 0;
  };
  auto shift = [&]() {
#pragma unroll
    for (int l = 0; l < S; ++l)
#pragma unroll
      for (int z = 0; z < LMAX; ++z) {
        Z[l][0][z] = Z[l][1][z];
        Z[l][1][z] = Z[l][2][z];
      }
  };
  // rows in whose iteration every step works strictly inside the grid
  const int lo = max(2 * S, 2 * S + 1 - y0), hi = min(nit, ny - (y0 - S) - (FIRST ? 1 : 0));
  if (ok && !done) {
#pragma unroll 1
    while (it < nit && ok) {
      if (it >= lo && it < hi) row(StInt<0>{});
      else row(StInt<1>{});
      shift();
    }
  }
  if (!ok && lane == 0) ctl_wait_lost(ctl);
  // never leave while copies into this block's shared memory are in flight
  for (int q = ok ? it : lost; q < min(ii, nit); ++q) tb_mbar_wait(bar + q % NZ, (unsigned)(q / NZ) & 1u);
  if (!LAST || done) return;
  double tot[1];
  if (!grid_reduce<Sum2, 1>(part, partials, stride, counter, tot)) return;
  ctl->rz_next = tot[0];
  ctl_set_beta(ctl);
}
