// The FP32 inner PCG of a small layer-uniform grid in one launch, on chip.
//
// A grid whose columns fit one tile per SM is bound by latency, not by work: an
// iteration with a degree-30 polynomial was ten launches of 6 to 8 us each, of which a
// fused chunk computes for about 3.  Here one cooperative kernel runs the whole inner
// solve.  Every CTA owns one tile of (32 - 2H) x (EY - 2H) columns (all layers) grown by
// H cells; a thread keeps its column's z_m, z_{m-1}, r and 1/D in registers (layer pairs, as
// in kernels_tb.cuh) and r, x, p in its own shared-memory slots.  H Chebyshev steps run between two exchanges, in which the tile's
// H outermost cells go to the neighbours' halo columns.  With fewer tiles than SMs the
// halo that is recomputed costs nothing; oc_shape picks EY and H from what a step and an
// exchange cost.  No tensor copies, so any nx.
//
// Measured (before: one launch per chunk of four steps where nx % 4 == 0, else per step):
// steady 64 x 64 x 4, degree 30, in a graph 2.24 -> 0.76 ms; steady 301 x 203 x 8 36.4 ->
// 5.8 ms; one 130 x 70 x 4 time step 0.86 -> 0.30 ms.  What bounds it now is shared memory
// and issue inside a step (32 rows x 8 layers: 0.67 us for 1280 wavefronts) and the
// latency of 1.5 us per exchange or sum.
//
// Everything that crosses CTAs goes through global memory (L2) as 128-bit words of three
// 32-bit values beside the exchange's number, each word written and read whole: a reader
// polls the very words it needs, so there is no flag, no fence and no barrier, and an
// exchange costs one store and one load latency.  (Words of one value and the number made
// an exchange 8 us: the instructions of all its threads, not the latency.)  A dot product
// is summed the same way: each CTA writes its FP64 partial as one word into a slot of its
// own, warp 0 of every CTA reads all slots and adds them in slot order, so all CTAs hold
// the same total, deterministically.  Two sets of words alternate, and exchanges and sums
// are numbered apart: a CTA writes a set again only after it has read its neighbours' words
// of the exchange in between (everybody's of the sum in between), which they wrote after
// they had read the earlier ones.  Waits are bounded (one second), after which the error is
// recorded and every CTA leaves; the cooperative launch starts no CTA before all of them have
// a place, however long other work holds the SMs.
#pragma once

#include "kernels_tb.cuh"

#define OC_MAXK 128  // highest polynomial degree (its coefficients are kernel parameters)

template <int LMAX>
struct __align__(8) OCParams {
  float c1[OC_MAXK], c2[OC_MAXK];         // three-term coefficients of step m
  float2 nd[LMAX / 2];                    // -(diagonal of a cell with all four in-plane faces)
  float2 gx[LMAX / 2], gy[LMAX / 2];      // in-plane faces
  float2 gzu[LMAX / 2], gzd[LMAX / 2];    // face to the layer above / below, 0 at the ends
  float2 s[LMAX / 2];                     // sink + capacity term
  float invd[9][LMAX];                    // 1 / diagonal for (x faces present) + 3 (y faces present)
  float z1s;                              // z_1 = z1s D^-1 r
  int k;                                  // polynomial degree
  int expire_test;                        // test hook: the first barrier runs out
};

// 2 sets x cap sum slots, the numbers of the last exchange and sum, then 2 sets of
// exchanged words: [word of a column][column]
__host__ __device__ constexpr int oc_column_words(int lmax) { return (2 * lmax + 2) / 3; }

struct OCWord { unsigned long long lo, hi; };
__device__ __forceinline__ void oc_put(OCWord* p, unsigned long long lo, unsigned long long hi) {
  asm volatile("{\n\t.reg .b128 q;\n\tmov.b128 q, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], q;\n\t}"
               ::"l"(p), "l"(lo), "l"(hi) : "memory");
}
__device__ __forceinline__ OCWord oc_get(const OCWord* p) {
  OCWord w;
  asm volatile("{\n\t.reg .b128 q;\n\tld.relaxed.gpu.global.b128 q, [%2];\n\tmov.b128 {%0, %1}, q;\n\t}"
               : "=l"(w.lo), "=l"(w.hi) : "l"(p) : "memory");
  return w;
}

// true once a poll that started with t0 = 0 has lasted TB_WAIT_NS
__device__ __forceinline__ bool oc_late(unsigned long long& t0) {
  const unsigned long long now = tb_clock_ns();
  if (t0 == 0) t0 = now;
  return now - t0 > TB_WAIT_NS;
}

// A column's message of NP layer pairs (a, or a then b) as words of three values and the
// exchange's number, `stride` words apart.
template <int NP, int LP>
__device__ __forceinline__ void oc_send(OCWord* w, long long stride, const float2 (&a)[LP], const float2 (&b)[LP],
                                        unsigned epoch) {
  constexpr int NF = 2 * NP, NJ = (NF + 2) / 3;
  unsigned f[3 * NJ];
#pragma unroll
  for (int i = 0; i < 3 * NJ; ++i) f[i] = 0u;
#pragma unroll
  for (int k = 0; k < LP; ++k) {
    f[2 * k] = __float_as_uint(a[k].x);
    f[2 * k + 1] = __float_as_uint(a[k].y);
    if (NP > LP) {
      f[2 * (NP > LP ? LP : 0) + 2 * k] = __float_as_uint(b[k].x);
      f[2 * (NP > LP ? LP : 0) + 2 * k + 1] = __float_as_uint(b[k].y);
    }
  }
#pragma unroll
  for (int j = 0; j < NJ; ++j)
    oc_put(w + j * stride, ((unsigned long long)f[3 * j + 1] << 32) | f[3 * j],
           ((unsigned long long)epoch << 32) | f[3 * j + 2]);
}

// polls the message until every word carries the number; false when the wait ran out
template <int NP, int LP>
__device__ __forceinline__ bool oc_recv(const OCWord* w, long long stride, float2 (&a)[LP], float2 (&b)[LP],
                                        unsigned epoch) {
  constexpr int NF = 2 * NP, NJ = (NF + 2) / 3;
  unsigned f[3 * NJ];
  unsigned long long t0 = 0;
  bool all = false, late = false;
  while (!all && !late) {
    unsigned off = 0;
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
      const OCWord q = oc_get(w + j * stride);
      f[3 * j] = (unsigned)q.lo;
      f[3 * j + 1] = (unsigned)(q.lo >> 32);
      f[3 * j + 2] = (unsigned)q.hi;
      off |= (unsigned)(q.hi >> 32) ^ epoch;
    }
    all = off == 0;
    if (!all) late = oc_late(t0);
  }
#pragma unroll
  for (int k = 0; k < LP; ++k) {
    a[k] = make_float2(__uint_as_float(f[2 * k]), __uint_as_float(f[2 * k + 1]));
    if (NP > LP)
      b[k] = make_float2(__uint_as_float(f[2 * (NP > LP ? LP : 0) + 2 * k]),
                         __uint_as_float(f[2 * (NP > LP ? LP : 0) + 2 * k + 1]));
  }
  return all;
}

// scalars of the iteration, decided by thread 0 of every CTA from the same totals
struct OCShared {
  float red[32 * 16];
  double rz, rr0, tgt;
  float alpha, beta;
  int it, status, stop, ok;
};

template <int LMAX, int EY>
constexpr size_t oc_smem_bytes() {
  return (size_t)(2 + 3) * (LMAX / 2) * EY * TB_EX * sizeof(float2);
}

// A float per thread, the sum of a column's LP layer pairs, summed over the grid and handed
// to fin(total) in thread 0 of every CTA.  False when the wait ran out.  A product meets at
// most five FP32 additions, those of its column among them, as in the one-step kernels
// (one cell a thread, 32 lanes); the rest keeps its rounding errors.  As fast as a plain
// FP32 sum of column and lanes (steady 64 x 64 x 4 757 us with it, 755 now); all five lane
// steps with their errors kept took 791.
template <int LP, typename F>
__device__ __forceinline__ bool oc_sum(OCShared& sh, OCWord* sync, int cap, unsigned& sums, float v, F fin) {
  constexpr int FP = 5 - (tree_depth(LP) + 1), G = 32 >> FP;  // lane steps in FP32, values left of a warp
  static_assert(FP >= 1 && G <= 16, "lane groups of a column sum");
  const int t = thread_linear_id(), nw = block_threads() >> 5, nblk = gridDim.x;
  const unsigned epoch = ++sums;
#pragma unroll
  for (int o = 1; o < (1 << FP); o *= 2) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((t & ((1 << FP) - 1)) == 0) sh.red[t >> FP] = v;
  __syncthreads();
  if (t < 32) {
    Sum2 part{0.f, 0.f};
#pragma unroll
    for (int i = 0; i < G; ++i)
      if (t + 32 * i < nw * G) sum2_add(part, sh.red[t + 32 * i]);
    const double mine = warp_sum(sum2_value(part));
    OCWord* set = sync + (size_t)(epoch & 1u) * cap;
    if (t == 0) oc_put(set + blockIdx.x, (unsigned long long)__double_as_longlong(mine), epoch);
    double tot = 0.0;
    bool ok = true;
    unsigned long long t0 = 0;
    for (int j0 = t; j0 < nblk && ok; j0 += 32 * 5) {  // a lane reads its slots together
      OCWord w[5];
      bool behind = true;
      while (behind && ok) {
        behind = false;
#pragma unroll
        for (int i = 0; i < 5; ++i)
          if (j0 + 32 * i < nblk) w[i] = oc_get(set + j0 + 32 * i);
          else w[i] = OCWord{0ull, epoch};
#pragma unroll
        for (int i = 0; i < 5; ++i) behind = behind || (unsigned)w[i].hi != epoch;
        if (behind) ok = !oc_late(t0);
      }
#pragma unroll
      for (int i = 0; i < 5; ++i) tot += __longlong_as_double((long long)w[i].lo);
    }
    ok = __all_sync(0xffffffffu, ok);
    tot = warp_sum(tot);
    if (t == 0) {
      sh.ok = ok;
      if (ok) fin(tot);
    }
  }
  __syncthreads();
  return sh.ok != 0;
}

// solve = 1: the inner PCG on r (x = 0 on entry; ctl holds its start, see fin_update);
// x_out receives the correction.  solve = 0: z_out = M^-1 r only.
//
// DIFF takes the steps' product in difference form, sum_f g_f (v_f - v), instead of the
// expanded form: six more additions per cell, for grids that had no fused chunks before
// (nx % 4 != 0, one difference-form launch per step), so that their vectors are as
// accurate as they were.  The residual r - A v is formed before it is scaled: with D^-1 r
// kept in r's place (one instruction less in difference form, 0.8 % of an iteration) the
// error against 64 bits was 1.08 times the one-step kernels' in the mean over 1700 grids,
// degrees and stacks with nx % 4 != 0, and 1.01 times the tiles' elsewhere; it is 1.016 and
// 0.79 times (what is left of the former: they divide by the diagonal).
template <int LMAX, int EY, bool DIFF>
__global__ void __launch_bounds__(TB_EX * EY, 1)
    k_pcg_oc(Dims d, int ntx, int H, int solve, Ctl* ctl, const float* __restrict__ r, float* __restrict__ x_out,
             float* __restrict__ z_out, const __grid_constant__ OCParams<LMAX> P, OCWord* sync, int cap) {
  grid_dep_enter();
  constexpr int LP = LMAX / 2, PL = EY * TB_EX;
  extern __shared__ __align__(16) float2 oc_dyn[];
  __shared__ OCShared sh;
  const int tid = thread_linear_id();
  float2* plane = oc_dyn;                    // [2][LP][PL]
  float2* rs_ = oc_dyn + 2 * LP * PL + tid;  // this thread's slots, stride PL: r, x, p
  float2* xs_ = rs_ + LP * PL;
  float2* ps_ = xs_ + LP * PL;
  if (solve && ld_int(&ctl->done)) return;
  const int L = d.L, ex = threadIdx.x, ey = threadIdx.y;
  const int TX = TB_EX - 2 * H, TY = EY - 2 * H;
  const int tx = (int)blockIdx.x % ntx, ty = (int)blockIdx.x / ntx;
  const int gx = tx * TX - H + ex, gy = ty * TY - H + ey;
  const bool inside = gx >= 0 && gx < d.nx && gy >= 0 && gy < d.ny;
  const bool interior = inside && ex >= H && ex < TB_EX - H && ey >= H && ey < EY - H;
  const bool halo = inside && !interior;
  // steps a column can take before a cell it needs is no longer valid
  const int depth = inside ? min(min(ex, TB_EX - 1 - ex), min(ey, EY - 1 - ey)) : 0;
  // interior cells that a neighbour's halo (H wide) or first ring (1 wide) covers
  const bool pubH = interior && (ex < 2 * H || ex >= TB_EX - 2 * H || ey < 2 * H || ey >= EY - 2 * H);
  const bool pub1 = interior && (ex == H || ex == TB_EX - 1 - H || ey == H || ey == EY - 1 - H);
  const bool ring1 = halo && ex >= H - 1 && ex <= TB_EX - H && ey >= H - 1 && ey <= EY - H;
  const long long base = inside ? (long long)gx + (long long)d.nx * gy : 0;
  const int nxf = (gx + 1 < d.nx) + (gx > 0), nyf = (gy + 1 < d.ny) + (gy > 0);
  const int oR = tid + ((gx + 1 < d.nx) ? 1 : 0), oL = tid - ((gx > 0) ? 1 : 0);
  const int oU = tid + ((gy + 1 < d.ny) ? TB_EX : 0), oD = tid - ((gy > 0) ? TB_EX : 0);
  const float2 m1 = make_float2(-1.f, -1.f);
  // numbers of the last exchange and the last sum of the launch before
  const OCWord last = oc_get(sync + 2 * cap);
  unsigned epoch = (unsigned)last.lo, sums = (unsigned)last.hi;
  const unsigned epoch0 = epoch, sums0 = sums;

  // this column's words of the current exchange's set
  OCWord* const col0 = sync + 2 * cap + 1 + (inside ? gx + (long long)d.nx * gy : 0);
  const long long set1 = (long long)oc_column_words(LMAX) * d.pxy;
  float2 za[LP], zb[LP], iv[LP], rs[LP];  // iv = 1/D, rs = r
#pragma unroll
  for (int k = 0; k < LP; ++k) {
    float2 rv = make_float2(0.f, 0.f);
    if (inside && k < L) rv.x = __ldg(r + base + d.pxy * k);
    if (inside && k + LP < L) rv.y = __ldg(r + base + d.pxy * (k + LP));
    rs_[k * PL] = rv;
    xs_[k * PL] = make_float2(0.f, 0.f);
    ps_[k * PL] = make_float2(0.f, 0.f);
    const int c = nxf + 3 * nyf;
    iv[k] = inside ? make_float2(P.invd[c][k], P.invd[c][k + LP]) : make_float2(0.f, 0.f);
  }
  if (tid == 0) {
    sh.rr0 = ld_dbl(&ctl->rr0);
    const double rel = ld_dbl(&ctl->inner_rel);
    sh.tgt = rel * rel * sh.rr0;
    sh.rz = 0.0;
    sh.beta = 0.f;
    sh.it = 0;
    sh.status = 0;
    sh.stop = 0;
  }
  const int max_inner = ld_int(&ctl->max_inner);
  auto step = [&](const float2 (&C)[LP], float2 (&N)[LP], const int j, const float c1s, const float c2s) {
    float2* pl = plane + (j & 1) * LP * PL;
#pragma unroll
    for (int k = 0; k < LP; ++k) pl[k * PL + tid] = C[k];
    __syncthreads();
    if (depth > j) {
      const float2 c1 = make_float2(c1s, c1s), c2 = make_float2(c2s, c2s);
#pragma unroll
      for (int k = 0; k < LP; ++k) {
        const float2 v = C[k];
        const float2* q = pl + k * PL;
        float2 a;  // -(A v)
        if (DIFF) {  // the operation order of the one-step kernels
          const float2 nv = __fmul2_rn(v, m1);
          a = __fmul2_rn(P.s[k], nv);
          a = __ffma2_rn(P.gx[k], __fadd2_rn(q[oR], nv), a);
          a = __ffma2_rn(P.gx[k], __fadd2_rn(q[oL], nv), a);
          a = __ffma2_rn(P.gy[k], __fadd2_rn(q[oU], nv), a);
          a = __ffma2_rn(P.gy[k], __fadd2_rn(q[oD], nv), a);
          const float2 up = k + 1 < LP ? C[k + 1 < LP ? k + 1 : k] : make_float2(C[0].y, 0.f);
          const float2 dn = k > 0 ? C[k > 0 ? k - 1 : k] : make_float2(0.f, C[LP - 1].x);
          a = __ffma2_rn(P.gzu[k], __fadd2_rn(up, nv), a);  // the faces at the ends are 0
          a = __ffma2_rn(P.gzd[k], __fadd2_rn(dn, nv), a);
          a = __fadd2_rn(rs[k], a);
        } else {  // the operation order of k_cheb_tb with every sign turned, from r on
          a = __ffma2_rn(P.nd[k], v, rs[k]);
          a = __ffma2_rn(P.gx[k], __fadd2_rn(q[oR], q[oL]), a);
          a = __ffma2_rn(P.gy[k], __fadd2_rn(q[oU], q[oD]), a);
          if (k + 1 < LP) a = __ffma2_rn(P.gzu[k], C[k + 1 < LP ? k + 1 : k], a);
          else a.x = fmaf(P.gzu[k].x, C[0].y, a.x);
          if (k > 0) a = __ffma2_rn(P.gzd[k], C[k > 0 ? k - 1 : k], a);
          else a.y = fmaf(P.gzd[0].y, C[LP - 1].x, a.y);
        }
        const float2 res = __fmul2_rn(a, iv[k]);
        N[k] = __ffma2_rn(c2, res, __ffma2_rn(c1, __ffma2_rn(N[k], m1, v), v));
      }
    }
  };
  bool ok = true;
  if (P.expire_test) {  // wait for a number that nothing writes
    bool dead = true;
    if (tid == 0) {
      const unsigned long long t0 = tb_clock_ns();
      while (dead && tb_clock_ns() - t0 <= TB_TEST_WAIT_NS) dead = oc_get(sync + 2 * cap).hi != ~0ull;
    }
    ok = !__syncthreads_or(tid == 0 && dead);
  }
  bool got = true;  // this thread's polls since the last block-wide check
  while (ok) {
    // ---- z = M^-1 r on the interior
#pragma unroll
    for (int k = 0; k < LP; ++k) {
      rs[k] = rs_[k * PL];
      za[k] = __fmul2_rn(__fmul2_rn(rs[k], iv[k]), make_float2(P.z1s, P.z1s));
      zb[k] = make_float2(0.f, 0.f);
    }
    int m = 1;
    while (true) {
      const int S = min(H, P.k - m);
      // the planes are free, every halo column has arrived
      if (!(ok = !__syncthreads_or(!got))) break;
      for (int j = 0; j + 1 < S; j += 2) {
        step(za, zb, j, P.c1[m + j], P.c2[m + j]);
        step(zb, za, j + 1, P.c1[m + j + 1], P.c2[m + j + 1]);
      }
      if (S & 1) {
        step(za, zb, S - 1, P.c1[m + S - 1], P.c2[m + S - 1]);
#pragma unroll
        for (int k = 0; k < LP; ++k) {
          const float2 v = za[k];
          za[k] = zb[k];
          zb[k] = v;
        }
      }
      m += S;
      if (m >= P.k) break;
      ++epoch;
      if (pubH) oc_send<2 * LP>(col0 + (epoch & 1u) * set1, d.pxy, za, zb, epoch);
      if (halo) got = oc_recv<2 * LP>(col0 + (epoch & 1u) * set1, d.pxy, za, zb, epoch);
    }
    if (!ok) break;
    if (!solve) {
      if (interior) {
#pragma unroll
        for (int k = 0; k < LP; ++k) {
          if (k < L) z_out[base + d.pxy * k] = za[k].x;
          if (k + LP < L) z_out[base + d.pxy * (k + LP)] = za[k].y;
        }
      }
      // nobody may record the last number before everybody has read the first
      if (epoch != epoch0) ok = oc_sum<LP>(sh, sync, cap, sums, 0.f, [](double) {});
      break;
    }
    // ---- r^T z, beta, p = z + beta p on the interior and the ring around it
    float part = 0.f;
    ++epoch;
    if (interior) {
      float2 t[LP];
#pragma unroll
      for (int k = 0; k < LP; ++k) t[k] = __fmul2_rn(rs_[k * PL], za[k]);
      part = pair_sum(t);
      if (pub1) oc_send<LP>(col0 + (epoch & 1u) * set1, d.pxy, za, za, epoch);
    }
    ok = oc_sum<LP>(sh, sync, cap, sums, part, [&](double t) {
      sh.beta = (sh.it == 0 || !(sh.rz != 0.0)) ? 0.f : (float)(t / sh.rz);
      sh.rz = t;
    });
    if (!ok) break;
    if (ring1) got = oc_recv<LP>(col0 + (epoch & 1u) * set1, d.pxy, za, zb, epoch);
    const float beta = sh.beta;
    float2* pl = plane;
    if (interior || ring1) {
#pragma unroll
      for (int k = 0; k < LP; ++k) {
        const float2 z = za[k], po = ps_[k * PL];
        const float2 pn = sh.it == 0 ? z : make_float2(z.x + beta * po.x, z.y + beta * po.y);
        ps_[k * PL] = pn;
        pl[k * PL + tid] = pn;
      }
    }
    if (!(ok = !__syncthreads_or(!got))) break;
    // ---- mu = A p in difference form (kept in zb), p^T mu
    part = 0.f;
    if (interior) {
      float2 t[LP];
#pragma unroll
      for (int k = 0; k < LP; ++k) {
        const float2* q = pl + k * PL;
        const float2 v = q[tid];
        auto dif = [&](const float2& o) { return __ffma2_rn(o, m1, v); };
        float2 a = __fmul2_rn(P.s[k], v);
        a = __ffma2_rn(P.gx[k], dif(q[oR]), a);
        a = __ffma2_rn(P.gx[k], dif(q[oL]), a);
        a = __ffma2_rn(P.gy[k], dif(q[oU]), a);
        a = __ffma2_rn(P.gy[k], dif(q[oD]), a);
        const float2 up = k + 1 < LP ? pl[(k + 1 < LP ? k + 1 : k) * PL + tid] : make_float2(pl[tid].y, 0.f);
        const float2 dn = k > 0 ? pl[(k > 0 ? k - 1 : k) * PL + tid] : make_float2(0.f, pl[(LP - 1) * PL + tid].x);
        a = __ffma2_rn(P.gzu[k], dif(up), a);  // the faces at the ends are 0
        a = __ffma2_rn(P.gzd[k], dif(dn), a);
        zb[k] = a;
        t[k] = __fmul2_rn(v, a);
      }
      part = pair_sum(t);
    }
    ok = oc_sum<LP>(sh, sync, cap, sums, part, [&](double pAp) {
      const bool fine = pAp > 0.0 && sh.rz > 0.0;
      sh.alpha = fine ? (float)(sh.rz / pAp) : 0.f;
      if (!fine) {  // breakdown (see fin_pap)
        sh.status = (isfinite(pAp) && isfinite(sh.rz)) ? 5 : 6;
        sh.stop = 1;
      }
    });
    if (!ok || sh.stop) break;
    // ---- x += alpha p, r -= alpha mu, ||r||^2
    const float alpha = sh.alpha;
    part = 0.f;
    ++epoch;
    if (interior) {
      float2 t[LP];
#pragma unroll
      for (int k = 0; k < LP; ++k) {
        const float2 p = ps_[k * PL], x = xs_[k * PL], mu = zb[k];
        float2 rv = rs_[k * PL];
        xs_[k * PL] = make_float2(x.x + alpha * p.x, x.y + alpha * p.y);
        rv.x -= alpha * mu.x;
        rv.y -= alpha * mu.y;
        rs_[k * PL] = rv;
        za[k] = rv;
        t[k] = __fmul2_rn(rv, rv);
      }
      part = pair_sum(t);
      if (pubH) oc_send<LP>(col0 + (epoch & 1u) * set1, d.pxy, za, za, epoch);
    }
    ok = oc_sum<LP>(sh, sync, cap, sums, part, [&](double rr) {
      sh.it += 1;
      sh.rr0 = rr;  // from here on the current ||r||^2
      if (!isfinite(rr)) {
        sh.status = 6;
        sh.stop = 1;
      } else if (rr <= sh.tgt || sh.it >= max_inner) {
        sh.stop = 1;
      }
    });
    if (!ok || sh.stop) break;
    if (halo) {
      got = oc_recv<LP>(col0 + (epoch & 1u) * set1, d.pxy, za, zb, epoch);
#pragma unroll
      for (int k = 0; k < LP; ++k) rs_[k * PL] = za[k];
    }
  }
  if (!ok) {  // a wait ran out
    if (tid == 0) {
      ctl_wait_lost(ctl);
      // numbers that this launch cannot have used, so that no later one meets its words
      oc_put(sync + 2 * cap, epoch0 + 0x40000000u, sums0 + 0x40000000u);
    }
    return;
  }
  if (solve && interior) {
#pragma unroll
    for (int k = 0; k < LP; ++k) {
      const float2 x = xs_[k * PL];
      if (k < L) x_out[base + d.pxy * k] = x.x;
      if (k + LP < L) x_out[base + d.pxy * (k + LP)] = x.y;
    }
  }
  if (blockIdx.x == 0 && tid == 0) {
    // (every CTA has taken part in a sum by now, so has read the word before)
    if (solve || epoch != epoch0) oc_put(sync + 2 * cap, epoch, sums);
    if (solve) {
      ctl->it = sh.it;
      ctl->it_total += sh.it;
      ctl->rr = sh.rr0;
      ctl->rz = ctl->rz_next = sh.rz;
      ctl->first = 0;
      if (sh.status) {
        ctl->status = sh.status;
        ctl->outer_done = 1;
      }
      ctl->done = 1;
    }
  }
}
