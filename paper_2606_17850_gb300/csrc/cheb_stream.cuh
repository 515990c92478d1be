// Launch of the streaming Chebyshev kernel for one layer capacity (LMAX); each
// cheb_stream_*.cu instantiates one, so they compile in parallel.
#pragma once

#include <algorithm>
#include <cstring>

#include "internal.h"
#include "kernels_stream.cuh"

template <int LMAX, int S, bool LAST, bool FIRST>
static th_status st_launch(thermal_grid* g, const Dims& d, const StreamChunk& c, cudaStream_t st) {
  STParams<LMAX> prm;
  std::memset(&prm, 0, sizeof(prm));
  auto two = [](float v) { return make_float2(v, v); };
  for (int j = 0; j < S; ++j) {
    prm.c1[j] = two(c.c1[j]);
    prm.c2[j] = two(c.c2[j]);
  }
  prm.z1s = c.z1s;
  prm.expire_test = c.expire_test;
  const LayerTab& T = g->tab_host;
  const int L = d.L;
  for (int z = 0; z < L; ++z) {
    const LayerCoefs q = layer_coefs(T, L, z);
    prm.gx[z] = two(q.gx);
    prm.gy[z] = two(q.gy);
    prm.gzu[z] = two(q.gzu);
    prm.gzd[z] = two(q.gzd);
    prm.nd[z] = two(-q.d);
    for (int k = 0; k < 9; ++k) prm.invd[k][z] = q.invd[k];
  }
  CUtensorMap mc, mp, mr;
  std::memset(&mc, 0, sizeof(mc));
  mp = mc;
  TH_TRY(tensor_map_3d(&mr, d, c.r, ST_BW, 1));
  if (!FIRST) {
    TH_TRY(tensor_map_3d(&mc, d, c.in_cur, ST_BW, 1));
    TH_TRY(tensor_map_3d(&mp, d, c.in_prev, ST_BW, 1));
  }
  auto* kern = k_cheb_st<LMAX, S, LAST, FIRST>;
  constexpr size_t smem = st_smem_bytes<LMAX, S, FIRST>();
  TH_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  const StreamCut cut = cheb_stream_cut(d.nx, d.ny, LMAX);
  const int nsx = cut.strips, R = cut.rows, ntask = cut.warps;
  if (LAST && ntask > g->partials_stride)
    return th_fail(TH_ESTATE, "partials buffer smaller than the streaming grid");
  th_launch(kern, ntask, 32, smem, st, d, nsx, R, g->ctl, mc, mp, mr, c.out_cur, c.out_prev, prm, g->partials,
            g->partials_stride, g->counters);
  TH_CHECK_LAUNCH();
  return TH_OK;
}

template <int LMAX, bool LAST, bool FIRST>
static th_status st_steps(thermal_grid* g, const Dims& d, const StreamChunk& c, cudaStream_t st) {
  switch (c.steps) {
    case 1: return st_launch<LMAX, 1, LAST, FIRST>(g, d, c, st);
    case 2: return st_launch<LMAX, 2, LAST, FIRST>(g, d, c, st);
    case 3: return st_launch<LMAX, 3, LAST, FIRST>(g, d, c, st);
    case 4: return st_launch<LMAX, 4, LAST, FIRST>(g, d, c, st);
    default: return th_fail(TH_ESTATE, "streaming chunk with %d steps", c.steps);
  }
}

template <int LMAX>
static th_status st_chunk(thermal_grid* g, const Dims& d, const StreamChunk& c, cudaStream_t st) {
  if (c.first) return c.last ? st_steps<LMAX, true, true>(g, d, c, st) : st_steps<LMAX, false, true>(g, d, c, st);
  return c.last ? st_steps<LMAX, true, false>(g, d, c, st) : st_steps<LMAX, false, false>(g, d, c, st);
}
