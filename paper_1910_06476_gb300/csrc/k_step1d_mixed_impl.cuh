#pragma once
// 1D DSEM-SL step, mixed precision, shared operator (uniform mesh, constant velocity).
//
// State: double-float, a hi plane and a lo plane of floats (phi = hi + lo, about 48 bits).
// Every element of a CTA tile is advanced by one thread, two elements (half a tile apart) per thread, one in
// each lane of the paired FP32 operations: the kernel is bound by instruction issue before HBM, and a pair
// costs the instructions of one element:
//   - its values are read relative to a per-element reference ref = hi of its first node:
//     psi = (hi - ref) + lo, in float.  The step operator reproduces constants, so phi^{n+1} = ref + G psi
//     and the float rounding scales with the variation inside the stencil rather than with |phi|;
//   - the linear step (remap eq. 4.9, upwinded boundary values eq. 4.12a, mass target
//     eq. remap_mass, constrained fit eq. matrix_a) is one shared operator applied in float.  The upwind
//     neighbour enters it through two numbers only, its outflow trace and its outflow flux (and through the
//     flux's stage values in the energy target); each element forms its own, relative to its own reference,
//     and leaves them in shared memory for its downstream neighbour;
//   - the energy constraint (eq. remap_energy) is solved per element; its mismatch is formed
//     from increments only, so that the decision to apply it is free of float cancellation;
//   - the result is written back exactly as ref + psi by TwoSum (Knuth), hi = fl(ref + psi),
//     lo = (ref + psi) - hi;
//   - with the mass row (hard fit), the element's mass target is also formed in float-float,
//     M^n - lam (F_own - F_up), where F is the outflow-flux functional applied to an element's hi + lo
//     (each element's F is computed bit for bit alike by the element itself and by its downstream
//     neighbour, so global mass telescopes); after the fit, the float-float miss of the written
//     element mass is moved along the pseudo-inverse column of the mass row into the lo words, so
//     that the element mass meets its target to about 1e-16 relative.
// Measured (one GB300): K = 2^20, n = 9, every constraint: 41.0 -> 36.8 us per step (16 bytes per node take
// 22 us at the measured copy rate); 34.5 M -> 23 M warp instructions, issue 60 %, FMA pipe 56 % busy.  Five
// CTAs per SM spill registers (42.9 us); from n = 14 on three CTAs with a few spills beat two without (n = 14: 58
// against 72 us).  The operators stand in the parameter bank as single floats, duplicated into both lanes where
// they are used: stored twice they cost every launch a cold read of up to 8 KB more (K = 4096, n = 12: 6.0 / 5.6
// us; K = 2^20, n = 17: 79.5 / 69.3).
// The kernel is persistent: a CTA advances tiles of TILE elements, one thread per two elements.  A
// tile's rows (its elements and the upwind halo element) are one contiguous run of each plane;
// one thread moves both runs into shared memory with bulk asynchronous copies (TMA) that complete
// on an mbarrier, into one of two stages, so the next tile's load overlaps this tile's
// arithmetic.  Results are written back into the stage and stored with bulk copies.  The kernel
// reads 8 and writes 8 bytes per node from HBM.  Every wait on a copy is bounded: on a timeout
// the CTA stops, reports SL_ST_TIMEOUT, and drains its stores.
#include <algorithm>
#include <type_traits>

#include "ffloat.cuh"
#include "sl_internal.h"

namespace sl {
namespace k1m {

constexpr int TILE = 256;                  // elements per tile
constexpr int NT = TILE / 2;               // threads: thread t advances elements t and t + NT of the tile
constexpr int WAIT_LIMIT = 1 << 22;        // polls of an mbarrier before a wait gives up

__device__ __forceinline__ int wrap_elem(int e, int K, bool periodic) {
  if (e >= 0 && e < K) return e;
  if (!periodic) return -1;
  e %= K;
  return e < 0 ? e + K : e;
}

// ---- bulk asynchronous copies (PTX cp.async.bulk) and mbarriers
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_init_fence() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
               : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, unsigned parity) {
  unsigned done;
  asm volatile(
      "{\n"
      "  .reg .pred p;\n"
      "  mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      "  selp.u32 %0, 1, 0, p;\n"
      "}\n"
      : "=r"(done)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return done != 0;
}

// global -> shared, completion counted in bytes on bar; addresses and size multiples of 16 bytes
__device__ __forceinline__ void bulk_load(void* dst, const void* src, unsigned bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_addr(dst)),
               "l"(src), "r"(bytes), "r"(smem_addr(bar))
               : "memory");
}

// shared -> global in the thread's bulk group; addresses and size multiples of 16 bytes
__device__ __forceinline__ void bulk_store(void* dst, const void* src, unsigned bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(smem_addr(src)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read_all() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
// this thread's shared-memory writes become visible to later bulk copies (async proxy)
__device__ __forceinline__ void fence_to_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// floats of one plane of one stage: TILE + 1 rows, up to 3 floats of alignment shift, and the
// rounding of the copied run to 16 bytes at both ends
template <int NN>
__host__ __device__ constexpr int stage_floats() { return ((TILE + 1) * NN + 16 + 3) & ~3; }

// Where tile t's rows sit: rows r in [r_lo, r_hi) are elements first + r inside [0, K), one
// contiguous run of floats [g0, g1) of each plane, copied as the 16-byte-aligned window [a0, a1)
// to shared offset sbase; row r starts at shared offset sh + r NN.  sh in [0, 4) makes sbase a
// multiple of 4 floats.
struct TileGeo {
  int e0, first, r_lo, r_hi, sh, sbase, nvec;
  int64_t a0;
};

template <int NN>
__device__ __forceinline__ TileGeo tile_geo(int K, int left_up, int t) {
  TileGeo g;
  g.e0 = t * TILE;
  g.first = left_up ? g.e0 - 1 : g.e0;
  g.r_lo = max(0, -g.first);
  g.r_hi = min(TILE + 1, K - g.first);
  const int64_t g0 = (int64_t)(g.first + g.r_lo) * NN, g1 = (int64_t)(g.first + g.r_hi) * NN;
  g.a0 = g0 & ~int64_t(3);
  const int64_t a1 = (g1 + 3) & ~int64_t(3);   // within the plane: planes are padded to 64 floats
  const int d = (int)(g0 - g.a0);
  g.sh = (d - g.r_lo * NN) & 3;
  g.sbase = g.sh + g.r_lo * NN - d;
  g.nvec = (int)((a1 - g.a0) >> 2);
  return g;
}

// Operators applied with the same entry by every thread (duplicated into both lanes at their use), and the scalars
template <int NN>
struct Par {
  fdup Gs[NN * NN], rout[NN], ui[NN], um[NN];
  fdup w[NN], E[3][NN], C[MMAX1D * NN], Cp[NN * MMAX1D], Ff[NN], wh[NN], nwh[NN], wl[NN], cmass[NN];   // nwh = -wh
  float fb[3];
  int K, left_up, periodic, m, mass_on, energy_on, nst, refine, picard_cap;
  int64_t plane;
  float ghost, ghost_lo;                     // the inflow value as float-float
  float lam, lam_lo, sumf, picard_rtol;
};

// What an element leaves for its downstream neighbour, relative to its own reference: the trace of its
// remapped polynomial at the outflow face, its outflow flux functional sum f_i psi_i (the same float
// operations whichever CTA evaluates it, so that both elements see the same number and global mass
// telescopes), the values at the flux's stage feet, the largest |psi|.  One array per quantity over the
// tile's rows.
struct Exch {
  float T[TILE + 1], F[TILE + 1], E[3][TILE + 1], mx[TILE + 1];
};

// Functionals of one row by one thread (the halo row): the scalar form of those in element_step
template <int NN>
__device__ __forceinline__ void halo_row(const Par<NN>& P, const float* hi, const float* lo, int row, Exch& X) {
  const float ref = hi[0];
  float t = 0.0f, f = 0.0f, e[3] = {0.0f, 0.0f, 0.0f}, mx = 0.0f;
#pragma unroll
  for (int i = 0; i < NN; ++i) {
    const float v = __fadd_rn(__fadd_rn(hi[i], -ref), lo[i]);
    t = fmaf(P.rout[i].v, v, t);
    f = fmaf(P.Ff[i].v, v, f);
#pragma unroll
    for (int s = 0; s < 3; ++s)
      if (s < P.nst) e[s] = fmaf(P.E[s][i].v, v, e[s]);
    mx = fmaxf(mx, fabsf(v));
  }
  X.T[row] = t;
  X.F[row] = f;
#pragma unroll
  for (int s = 0; s < 3; ++s) X.E[s][row] = e[s];
  X.mx[row] = mx;
}

// Two elements: rows (of the staged tile) row and urow, their shared offsets own and up; writes
// res = phi^{n+1} - ref and the mass target.  has_up, act: per lane, whether there is an upwind element and
// whether the lane holds an element.  halo: the row that thread 0 also evaluates.  Every thread of the CTA
// calls it (a barrier separates what the elements leave from what they read).  Returns per lane whether the
// energy iteration converged (else the linear solution is kept).
template <int NN>
__device__ __forceinline__ void element_step(const Par<NN>& P, Exch& X, const float* shi, const float* slo, int sh,
                                             const int (&row)[2], const int (&urow)[2], const bool (&has_up)[2],
                                             const bool (&act)[2], int halo, float2& ref, float2 (&res)[NN], ff2& target,
                                             bool (&ok)[2]) {
  const int own[2] = {sh + row[0] * NN, sh + row[1] * NN};
  ref = make_float2(shi[own[0]], shi[own[1]]);
  const float2 mref = neg2(ref);
  float2 ps[NN], eo[3];
  float2 t = dup(0.0f), f = dup(0.0f);
  float mxx = 0.0f, mxy = 0.0f;
  cdot2n mn;
#pragma unroll
  for (int s = 0; s < 3; ++s) eo[s] = dup(0.0f);
#pragma unroll
  for (int i = 0; i < NN; ++i) {
    const float2 h = make_float2(shi[own[0] + i], shi[own[1] + i]), l = make_float2(slo[own[0] + i], slo[own[1] + i]);
    ps[i] = __fadd2_rn(__fadd2_rn(h, mref), l);
    if (P.refine) mn.add(P.wh[i], P.nwh[i], P.wl[i], h, l);
    t = __ffma2_rn(P.rout[i], ps[i], t);
    f = __ffma2_rn(P.Ff[i], ps[i], f);
    if (P.energy_on) {
#pragma unroll
      for (int s = 0; s < 3; ++s)
        if (s < P.nst) eo[s] = __ffma2_rn(P.E[s][i], ps[i], eo[s]);
      mxx = fmaxf(mxx, fabsf(ps[i].x));
      mxy = fmaxf(mxy, fabsf(ps[i].y));
    }
  }
  if (act[0]) {
    X.T[row[0]] = t.x;
    X.F[row[0]] = f.x;
    X.mx[row[0]] = mxx;
#pragma unroll
    for (int s = 0; s < 3; ++s) X.E[s][row[0]] = eo[s].x;
  }
  if (act[1]) {
    X.T[row[1]] = t.y;
    X.F[row[1]] = f.y;
    X.mx[row[1]] = mxy;
#pragma unroll
    for (int s = 0; s < 3; ++s) X.E[s][row[1]] = eo[s].y;
  }
  if (threadIdx.x == 0) halo_row<NN>(P, shi + sh + halo * NN, slo + sh + halo * NN, halo, X);
  __syncthreads();
  ok[0] = ok[1] = true;
  if (!act[0]) return;                       // (the second element comes after the first)
  // upwind values relative to the own reference; at an inflow domain face the ghost
  const float2 refu = make_float2(shi[sh + urow[0] * NN], shi[sh + urow[1] * NN]), dref = sub2(refu, ref);
  float2 Tu = __fadd2_rn(make_float2(X.T[urow[0]], X.T[urow[1]]), dref);
  const float2 fu0 = make_float2(X.F[urow[0]], X.F[urow[1]]);
  float2 Fu = __ffma2_rn(dref, dup(P.sumf), fu0), fu = __ffma2_rn(refu, dup(P.sumf), fu0);
  const float2 fo = __ffma2_rn(ref, dup(P.sumf), f);
  const float2 gh = __fadd2_rn(__fadd2_rn(dup(P.ghost), mref), dup(P.ghost_lo));
  if (!has_up[0]) {
    Tu.x = gh.x;
    Fu.x = gh.x * P.sumf;
    fu.x = P.ghost * P.sumf;
  }
  if (!has_up[1]) {
    Tu.y = gh.y;
    Fu.y = gh.y * P.sumf;
    fu.y = P.ghost * P.sumf;
  }
  if (P.refine) {
    // M^{n+1} = M^n - lam (F_own - F_up) in float-float; the fluxes are exact floats by definition
    const ff2 net = two_sum2(fu, neg2(fo)), m = ff_mul2(net, dup(P.lam), dup(P.lam_lo)), mm = mn.get();
    target = ff_add2(ff2{neg2(mm.hi), neg2(mm.lo)}, m);
  }
  // shared linear operator
  float2 pl[NN];
#pragma unroll
  for (int j = 0; j < NN; ++j) {
    float2 acc = dup(0.0f);
#pragma unroll
    for (int i = 0; i < NN; ++i) acc = __ffma2_rn(P.Gs[j * NN + i], ps[i], acc);
    acc = __ffma2_rn(P.ui[j], Tu, acc);
    acc = __ffma2_rn(P.um[j], Fu, acc);
    pl[j] = acc;
    res[j] = acc;
  }
  if (!P.energy_on) return;
  // The energy iteration is covariant under phi -> c phi (gamma, alpha, beta scale by c^2, q by c, s is
  // invariant), so it runs on values scaled by a power of two to order one; elements whose values lie below
  // the normal float range carry no energy correction.  The decision whether to run it is the same for
  // every power of two as long as nothing over- or underflows, so values of ordinary size skip the scaling.
  const float sx = fmaxf(fmaxf(fabsf(ref.x), mxx), has_up[0] ? fmaxf(fabsf(dref.x), X.mx[urow[0]]) : fabsf(gh.x));
  const float sy = fmaxf(fmaxf(fabsf(ref.y), mxy), has_up[1] ? fmaxf(fabsf(dref.y), X.mx[urow[1]]) : fabsf(gh.y));
  // energy mismatch from increments: variance part, plus 2 ref x mass residual when the mass row is not
  // enforced (with it, that bracket vanishes identically)
  float2 gamma, escale;
  auto mismatch = [&](auto scaled, float2 sc) {
    constexpr bool SC = decltype(scaled)::value;
    float2 gv = dup(0.0f), gm = dup(0.0f), es = dup(0.0f);
    const float2 rf = SC ? __fmul2_rn(ref, sc) : ref;
#pragma unroll
    for (int i = 0; i < NN; ++i) {
      const float2 qs = SC ? __fmul2_rn(ps[i], sc) : ps[i];
      const float2 ql = SC ? __fmul2_rn(pl[i], sc) : pl[i];
      const float2 d = sub2(ql, qs), v = __fadd2_rn(rf, qs);
      gv = __ffma2_rn(P.w[i], __fmul2_rn(d, __fadd2_rn(ql, qs)), gv);
      if (!P.mass_on) gm = __ffma2_rn(P.w[i], d, gm);
      es = __ffma2_rn(P.w[i], __fmul2_rn(v, v), es);
    }
#pragma unroll
    for (int s = 0; s < 3; ++s)
      if (s < P.nst) {
        const float2 fs = dup(P.lam * P.fb[s]);
        float2 eu = __fadd2_rn(make_float2(X.E[s][urow[0]], X.E[s][urow[1]]), dref);
        if (!has_up[0]) eu.x = gh.x;
        if (!has_up[1]) eu.y = gh.y;
        const float2 a = SC ? __fmul2_rn(eo[s], sc) : eo[s], b = SC ? __fmul2_rn(eu, sc) : eu;
        gv = __ffma2_rn(fs, sub2(__fmul2_rn(a, a), __fmul2_rn(b, b)), gv);
        if (!P.mass_on) gm = __ffma2_rn(fs, sub2(a, b), gm);
      }
    gamma = P.mass_on ? gv : __ffma2_rn(__fmul2_rn(dup(2.0f), rf), gm, gv);
    escale = es;
  };
  // powers of two that bring the lanes to order one (1 for values of ordinary size)
  auto pow2 = [](float v, int& ex) {
    frexpf(v, &ex);
    return ldexpf(1.0f, -ex);
  };
  const bool plain = fminf(sx, sy) >= 1e-8f && fmaxf(sx, sy) <= 1e8f;
  int exx = 0, exy = 0;
  float2 sc = dup(1.0f);
  if (plain) {
    mismatch(std::false_type{}, sc);
  } else {
    sc = make_float2(pow2(sx, exx), pow2(sy, exy));
    mismatch(std::true_type{}, sc);
  }
  bool on[2] = {act[0] && sx >= 1e-30f && fabsf(gamma.x) > (float)ENERGY_SKIP_RTOL_MIXED * escale.x,
                act[1] && sy >= 1e-30f && fabsf(gamma.y) > (float)ENERGY_SKIP_RTOL_MIXED * escale.y};
  if (!(on[0] || on[1])) return;
  if (plain) {
    sc = make_float2(pow2(sx, exx), pow2(sy, exy));
    gamma = __fmul2_rn(gamma, __fmul2_rn(sc, sc));
  }
  const float2 rf = __fmul2_rn(ref, sc);
  float2 ql[NN], cur[NN];
  float pmx = 0.0f, pmy = 0.0f;
#pragma unroll
  for (int i = 0; i < NN; ++i) {
    ql[i] = __fmul2_rn(pl[i], sc);
    cur[i] = ql[i];
    pmx = fmaxf(pmx, fabsf(ql[i].x));
    pmy = fmaxf(pmy, fabsf(ql[i].y));
  }
  const float tolx = fmaxf(P.picard_rtol * fabsf(rf.x), 2.4e-7f * pmx) + 1e-30f;
  const float toly = fmaxf(P.picard_rtol * fabsf(rf.y), 2.4e-7f * pmy) + 1e-30f;
  const bool ran[2] = {on[0], on[1]};
  ok[0] = !on[0];
  ok[1] = !on[1];
  // the exact solution of the energy equation along q for one lane
  auto root = [](float alpha, float beta, float g, bool& feasible) {
    if (beta <= 0.0f) {
      feasible = g <= 0.0f;
      return 0.0f;
    }
    const float disc = alpha * alpha - beta * g;
    feasible = !(disc < 0.0f);
    if (disc < 0.0f) return -alpha / beta;
    const float r = sqrtf(disc);
    const float den = alpha + (alpha >= 0.0f ? r : -r);
    return den == 0.0f ? 0.0f : -g / den;
  };
  for (int it = 0; it < P.picard_cap && (on[0] || on[1]); ++it) {
    float2 q[NN], ca[MMAX1D];
#pragma unroll
    for (int i = 0; i < NN; ++i) q[i] = __fmul2_rn(P.w[i], P.mass_on ? cur[i] : __fadd2_rn(rf, cur[i]));
#pragma unroll
    for (int k = 0; k < MMAX1D; ++k)
      if (k < P.m) {
        float2 acc = dup(0.0f);
#pragma unroll
        for (int i = 0; i < NN; ++i) acc = __ffma2_rn(P.C[k * NN + i], q[i], acc);
        ca[k] = neg2(acc);
      }
    float2 alpha = dup(0.0f), beta = dup(0.0f), wq = dup(0.0f);
#pragma unroll
    for (int j = 0; j < NN; ++j) {
#pragma unroll
      for (int k = 0; k < MMAX1D; ++k)
        if (k < P.m) q[j] = __ffma2_rn(P.Cp[j * MMAX1D + k], ca[k], q[j]);
      const float2 wj = __fmul2_rn(P.w[j], q[j]);
      alpha = __ffma2_rn(ql[j], wj, alpha);
      beta = __ffma2_rn(q[j], wj, beta);
      if (!P.mass_on) wq = __fadd2_rn(wj, wq);
    }
    if (!P.mass_on) alpha = __ffma2_rn(rf, wq, alpha);
    bool fx, fy;
    const float2 s = make_float2(root(alpha.x, beta.x, gamma.x, fx), root(alpha.y, beta.y, gamma.y, fy));
    float dx = 0.0f, dy = 0.0f;
#pragma unroll
    for (int i = 0; i < NN; ++i) {
      const float2 nv = __ffma2_rn(s, q[i], ql[i]), d = sub2(nv, cur[i]);
      dx = fmaxf(dx, fabsf(d.x));
      dy = fmaxf(dy, fabsf(d.y));
      if (on[0]) cur[i].x = nv.x;
      if (on[1]) cur[i].y = nv.y;
    }
    if (on[0] && dx <= tolx) { ok[0] = fx; on[0] = false; }
    if (on[1] && dy <= toly) { ok[1] = fy; on[1] = false; }
  }
  const float ux = ldexpf(1.0f, exx), uy = ldexpf(1.0f, exy);
#pragma unroll
  for (int i = 0; i < NN; ++i) {              // else: keep the linear-constraint solution
    if (ran[0] && ok[0]) res[i].x = cur[i].x * ux;
    if (ran[1] && ok[1]) res[i].y = cur[i].y * uy;
  }
}

template <int NN>
__global__ void __launch_bounds__(NT, NN <= 9 ? 4 : 3)
    k_step1d_mixed(const __grid_constant__ Par<NN> P, const float* __restrict__ in, float* __restrict__ out,
                   unsigned* status) {
  constexpr int SF = stage_floats<NN>();
  extern __shared__ __align__(16) float sm[];     // [stage][hi | lo][SF]
  __shared__ Exch X;
  __shared__ __align__(8) uint64_t bar[2];
  const int tid = threadIdx.x;
  const int K = P.K;
  const int64_t plane = P.plane;                  // float offset of the lo plane (multiple of 64)
  const int ntiles = (K + TILE - 1) / TILE;
  if (tid == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    mbar_init_fence();
  }
  __syncthreads();
  // thread 0: both planes of tile t into stage st
  auto issue = [&](int t, int st) {
    const TileGeo g = tile_geo<NN>(P.K, P.left_up, t);
    float* hi = sm + st * 2 * SF;
    const unsigned bytes = (unsigned)g.nvec * 16u;
    mbar_expect_tx(&bar[st], 2u * bytes);
    bulk_load(hi + g.sbase, in + g.a0, bytes, &bar[st]);
    bulk_load(hi + SF + g.sbase, in + plane + g.a0, bytes, &bar[st]);
  };
  if (tid == 0 && (int)blockIdx.x < ntiles) issue(blockIdx.x, 0);
  unsigned parity = 0;                            // bit st: phase parity awaited on stage st
  unsigned bits = 0;
  int st = 0;
  for (int t = blockIdx.x; t < ntiles; t += gridDim.x, st ^= 1) {
    // prefetch the next tile into the other stage once the stores that read it are done
    const int tn = t + (int)gridDim.x;
    if (tid == 0 && tn < ntiles) {
      bulk_wait_read_all();
      issue(tn, st ^ 1);
    }
    bool arrived = false;
    for (int it = 0; it < WAIT_LIMIT && !arrived; ++it) arrived = mbar_try_wait(&bar[st], (parity >> st) & 1u);
    if (__syncthreads_or(!arrived)) {             // every thread leaves together
      bits |= SL_ST_TIMEOUT;
      // the loads still in flight into this stage and into the prefetched one must land before
      // the CTA's shared memory is released: one more bounded wait on each (the output is left
      // incomplete either way)
      if (tid == 0) {
        bool done = false;
        for (int it = 0; it < WAIT_LIMIT && !done; ++it) done = mbar_try_wait(&bar[st], (parity >> st) & 1u);
        done = tn >= ntiles;
        for (int it = 0; it < WAIT_LIMIT && !done; ++it) done = mbar_try_wait(&bar[st ^ 1], (parity >> (st ^ 1)) & 1u);
      }
      __syncthreads();
      break;
    }
    parity ^= 1u << st;
    const TileGeo g = tile_geo<NN>(P.K, P.left_up, t);
    float* shi = sm + st * 2 * SF;
    float* slo = shi + SF;
    // the one halo row outside [0, K): periodic wrap, or zero at an inflow face (unused there)
    const int hrow = P.left_up ? 0 : g.r_hi;
    const bool hfix = P.left_up ? (g.r_lo == 1) : (g.r_hi <= TILE);
    if (hfix && tid < NN) {
      const int eh = wrap_elem(g.first + hrow, K, P.periodic != 0);
      shi[g.sh + hrow * NN + tid] = eh >= 0 ? in[(int64_t)eh * NN + tid] : 0.0f;
      slo[g.sh + hrow * NN + tid] = eh >= 0 ? in[plane + (int64_t)eh * NN + tid] : 0.0f;
    }
    __syncthreads();
    const int e[2] = {g.e0 + tid, g.e0 + NT + tid};
    const bool act[2] = {e[0] < K, e[1] < K};
    float2 res[NN];
    float2 ref = dup(0.0f);
    ff2 target = {dup(0.0f), dup(0.0f)};
    {
      int row[2], urow[2];
      bool has_up[2], ok[2];
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        // a lane without an element repeats the first one's rows (a thread without any, row 0's neighbour), so
        // that it reads staged values only
        const int r = act[c] ? tid + c * NT : act[0] ? tid : 0, ee = g.e0 + r;
        row[c] = P.left_up ? r + 1 : r;
        urow[c] = P.left_up ? r : r + 1;
        has_up[c] = wrap_elem(P.left_up ? ee - 1 : ee + 1, K, P.periodic != 0) >= 0;
      }
      const int halo = P.left_up ? 0 : min(TILE, K - g.e0);
      element_step<NN>(P, X, shi, slo, g.sh, row, urow, has_up, act, halo, ref, res, target, ok);
      if (!ok[0] || !ok[1]) bits |= SL_ST_PICARD_NOCONV;
    }
    __syncthreads();                              // the stage's rows are rewritten below
    if (act[0]) {
      bool finite = true;
      // TwoSum: hi + lo == ref + res exactly
      float2 vh[NN], vl[NN];
      cdot2n mv;
#pragma unroll
      for (int j = 0; j < NN; ++j) {
        const ff2 v = two_sum2(ref, res[j]);
        vh[j] = v.hi;
        vl[j] = v.lo;
        if (P.refine) mv.add(P.wh[j], P.nwh[j], P.wl[j], v.hi, v.lo);
      }
      if (P.refine) {
        // float-float miss of the element mass, moved along the mass column into the lo words
        const ff2 d = ff_add2(target, mv.get());     // (minus the written mass)
        const float2 miss = __fadd2_rn(d.hi, d.lo);
#pragma unroll
        for (int j = 0; j < NN; ++j) {
          const ff2 v = fast_two_sum2(vh[j], __ffma2_rn(miss, P.cmass[j], vl[j]));
          vh[j] = v.hi;
          vl[j] = v.lo;
        }
      }
#pragma unroll
      for (int j = 0; j < NN; ++j) {
        shi[tid * NN + j] = vh[j].x;
        slo[tid * NN + j] = vl[j].x;
        finite = finite && isfinite(vh[j].x);
      }
      if (act[1]) {
#pragma unroll
        for (int j = 0; j < NN; ++j) {
          shi[(tid + NT) * NN + j] = vh[j].y;
          slo[(tid + NT) * NN + j] = vl[j].y;
          finite = finite && isfinite(vh[j].y);
        }
      }
      if (!finite) bits |= SL_ST_NONFINITE;
      fence_to_async();
    }
    __syncthreads();
    // the tile's own elements are one run starting at e0 NN (a multiple of 4 floats)
    const int nout = min(TILE, K - g.e0) * NN, nv = nout >> 2;
    if (tid == 0 && nv > 0) {
      bulk_store(out + (int64_t)g.e0 * NN, shi, (unsigned)nv * 16u);
      bulk_store(out + plane + (int64_t)g.e0 * NN, slo, (unsigned)nv * 16u);
      bulk_commit();
    }
    for (int idx = 4 * nv + tid; idx < nout; idx += NT) {
      out[(int64_t)g.e0 * NN + idx] = shi[idx];
      out[plane + (int64_t)g.e0 * NN + idx] = slo[idx];
    }
    __syncthreads();                              // the stage is free once its stores have read it
  }
  if (tid == 0) bulk_wait_all();
  if (bits) atomicOr(status, bits);
}

template <int NN>
void launch_n(const Mixed1DParams& p, const float* in, float* out, unsigned* st, cudaStream_t s) {
  // persistent grid: resident CTAs per SM times the SM count (cached per device and kernel)
  constexpr size_t smem = (size_t)2 * 2 * stage_floats<NN>() * sizeof(float);
  const int cached_grid = persistent_grid((const void*)k_step1d_mixed<NN>, NT, smem);
  const int ntiles = (p.K + TILE - 1) / TILE;
  Par<NN> P;
  auto two = [](fdup* dst, const float* src, int n) {
    for (int i = 0; i < n; ++i) dst[i] = fdup{src[i]};
  };
  two(P.Gs, p.Gs, NN * NN);
  two(P.rout, p.rout, NN);
  two(P.ui, p.ui, NN);
  two(P.um, p.um, NN);
  two(P.w, p.w, NN);
  for (int k = 0; k < 3; ++k) {
    two(P.E[k], p.E[k], NN);
    P.fb[k] = p.fb[k];
  }
  two(P.C, p.C, MMAX1D * NN);
  for (int j = 0; j < NN; ++j)                 // rows of the pseudo-inverse at a fixed stride
    for (int k = 0; k < MMAX1D; ++k) P.Cp[j * MMAX1D + k] = fdup{k < p.m ? p.Cp[j * p.m + k] : 0.0f};
  two(P.Ff, p.Ff, NN);
  two(P.wh, p.wh, NN);
  two(P.wl, p.wl, NN);
  for (int i = 0; i < NN; ++i) P.nwh[i] = fdup{-p.wh[i]};
  two(P.cmass, p.cmass, NN);
  P.K = p.K;
  P.left_up = p.left_up;
  P.periodic = p.periodic;
  P.m = p.m;
  P.mass_on = p.mass_on;
  P.energy_on = p.energy_on;
  P.nst = p.nst;
  P.refine = p.refine;
  P.picard_cap = p.picard_cap;
  P.plane = p.plane;
  P.ghost = (float)p.ghost;
  P.ghost_lo = (float)(p.ghost - (double)P.ghost);
  P.lam = p.lam;
  P.lam_lo = p.lam_lo;
  P.sumf = p.sumf;
  P.picard_rtol = p.picard_rtol;
  k_step1d_mixed<NN><<<std::min(ntiles, cached_grid), NT, smem, s>>>(P, in, out, st);
}

}  // namespace k1m
}  // namespace sl
