// Host side of the on-chip inner PCG (kernels_oc.cuh).
#include <algorithm>
#include <cstring>

#include "internal.h"
#include "kernels_oc.cuh"

// Rows of the grown tile and halo width, {0, 0} where the kernel does not apply: the tiles
// have to fit the `sms` that the launch may use, one each, and a tile has to hold its neighbour's halo.  Among the
// shapes that do, the one with the least time for the k - 1 steps.  Measured over 64^2 to
// 301 x 203 columns, 16 / 24 / 32 rows and halos of 2 to 8: a step takes 5.2 ns per row and
// layer pair of the grown tile (0.17 us at 16 rows of 4 layers, 0.67 us at 32 rows of 8),
// an exchange 1.3 to 1.9 us whatever its width.
OCShape oc_shape(int nx, int ny, int L, int k, int sms) {
  OCShape best{0, 0};
  if (L > 12 || k < 2 || k > OC_MAXK) return best;
  const int lp = L <= 4 ? 2 : (L <= 6 ? 3 : (L <= 8 ? 4 : 6));
  double least = 1e30;
  for (int ey : {16, 24, 32}) {
    if (L > 8 && ey == 32) continue;  // 12 layers: at most 768 threads' registers
    for (int h = 2; h <= 8 && 3 * h <= ey; ++h) {
      const long long tx = TB_EX - 2 * h, ty = ey - 2 * h;
      if (((nx + tx - 1) / tx) * ((ny + ty - 1) / ty) > sms) continue;
      const double t = (k - 1) * 0.0052 * lp * ey + 1.6 * ((k - 1 + h - 1) / h);
      if (t < least) {
        least = t;
        best = OCShape{ey, h};
      }
    }
  }
  return best;
}

bool oc_cannot_launch(cudaError_t e) {
  return e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorNotSupported || e == cudaErrorLaunchOutOfResources;
}

template <int LMAX, int EY, bool DIFF>
static th_status oc_launch(thermal_grid* g, const OCRun& o, cudaStream_t s) {
  const Dims d = grid_dims(g);
  OCParams<LMAX> prm;
  std::memset(&prm, 0, sizeof(prm));
  for (int m = 1; m < o.k; ++m) {
    prm.c1[m] = (float)o.c1[m];
    prm.c2[m] = (float)o.c2[m];
  }
  prm.z1s = (float)o.inv_theta;
  prm.k = o.k;
  prm.expire_test = o.expire_test;
  const LayerTab& T = g->tab_host;
  const int L = d.L;
  // layer z is component (z < LMAX/2 ? x : y) of pair z % (LMAX/2)
  auto at = [](float2* a, int z) -> float& { return z < LMAX / 2 ? a[z].x : a[z - LMAX / 2].y; };
  for (int z = 0; z < L; ++z) {
    const LayerCoefs c = layer_coefs(T, L, z);
    at(prm.gx, z) = c.gx;
    at(prm.gy, z) = c.gy;
    at(prm.gzu, z) = c.gzu;
    at(prm.gzd, z) = c.gzd;
    at(prm.s, z) = c.s;
    at(prm.nd, z) = -c.d;
    for (int q = 0; q < 9; ++q) prm.invd[q][z] = c.invd[q];
  }
  const int tx = TB_EX - 2 * o.shape.halo, ty = EY - 2 * o.shape.halo;
  const int ntx = (d.nx + tx - 1) / tx, nblk = ntx * ((d.ny + ty - 1) / ty), cap = device_sms();
  constexpr size_t smem = oc_smem_bytes<LMAX, EY>();
  auto* kern = k_pcg_oc<LMAX, EY, DIFF>;
  TH_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  cudaLaunchAttribute at1{};
  at1.id = cudaLaunchAttributeCooperative;  // every CTA resident: they wait for one another
  at1.val.cooperative = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = dim3(nblk);
  c.blockDim = dim3(TB_EX, EY);
  c.dynamicSmemBytes = smem;
  c.stream = s;
  c.attrs = &at1;
  c.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&c, kern, d, ntx, o.shape.halo, o.solve, g->ctl, o.r, g->d32, o.z, prm,
                                           (OCWord*)g->oc_sync, cap);
  if (e == cudaSuccess) return TH_OK;
  g->oc_refused = oc_cannot_launch(e);
  cudaGetLastError();
  return th_fail(TH_ECUDA, "launch of the on-chip inner solve failed: %s", cudaGetErrorString(e));
}

template <int LMAX, bool DIFF>
static th_status oc_rows(thermal_grid* g, const OCRun& o, cudaStream_t s) {
  if (o.shape.rows == 16) return oc_launch<LMAX, 16, DIFF>(g, o, s);
  if (o.shape.rows == 24) return oc_launch<LMAX, 24, DIFF>(g, o, s);
  if constexpr (LMAX <= 8) return oc_launch<LMAX, 32, DIFF>(g, o, s);
  return th_fail(TH_ESTATE, "on-chip tile of %d rows", o.shape.rows);
}

template <bool DIFF>
static th_status oc_layers(thermal_grid* g, const OCRun& o, cudaStream_t s) {
  if (g->L <= 4) return oc_rows<4, DIFF>(g, o, s);
  if (g->L <= 6) return oc_rows<6, DIFF>(g, o, s);
  if (g->L <= 8) return oc_rows<8, DIFF>(g, o, s);
  return oc_rows<12, DIFF>(g, o, s);
}

static size_t oc_bytes(const thermal_grid* g) {
  const int lmax = g->L <= 4 ? 4 : (g->L <= 6 ? 6 : (g->L <= 8 ? 8 : 12));
  return sizeof(OCWord) * (2 * (size_t)device_sms() + 1 + 2 * (size_t)oc_column_words(lmax) * g->nx * g->ny);
}

// workspace of oc_run, before any graph capture; ready for any stream when this returns
th_status oc_prepare(thermal_grid* g, cudaStream_t s) {
  if (g->oc_sync) return TH_OK;
  if (cudaMalloc(&g->oc_sync, oc_bytes(g)) != cudaSuccess) {
    cudaGetLastError();
    g->oc_sync = nullptr;
    return th_fail(TH_ENOMEM, "exchange allocation failed");
  }
  cudaError_t e = cudaMemsetAsync(g->oc_sync, 0, oc_bytes(g), s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e == cudaSuccess) return TH_OK;
  cudaFree(g->oc_sync);  // not cleared: not the grid's
  g->oc_sync = nullptr;
  return th_fail(TH_ECUDA, "clearing the exchange words failed: %s", cudaGetErrorString(e));
}

th_status oc_run(thermal_grid* g, const OCRun& o, cudaStream_t s) {
  return g->nx % 4 == 0 ? oc_layers<false>(g, o, s) : oc_layers<true>(g, o, s);
}
