#pragma once
// 2D DSEM-SL step, mixed precision, shared operator: uniform mesh and constant velocity (a, b), so
// every element sees the same advected geometry (Sec. 5.3).  Operators are built once on the host
// (ops_mixed2d.cpp) and applied here in structured form:
//   row phase (thread j owns row j): x-remap of the row, x-outflow trace, the row's share of the mass and
//     outflow-flux functionals                                      (eq. 5.4, 4.12a, remap_mass)
//   column phase (thread j owns column j): y-remap of the column, y-outflow trace, inflow residuals
//   fit: s = (C C^T)^+ r over the inflow-face and mass rows, phi_L = psihat + C^T s   (eq. matrix_a)
// C^T s is separable (face rows are l0/l1 along one index and a unit vector along the other, the
// mass row is w (x) w), so the constrained fit costs O(n) per node instead of O(n) per constraint.
// State is double-float (hi plane, lo plane); all arithmetic is in float on increments relative to
// the element's first hi value and the result is written back exactly (TwoSum).
//
// A CTA owns a TX x TY tile of elements.  Each staged tile row (the TX elements plus the x-upwind
// halo element) is one contiguous run of global memory; it is copied in aligned 16-byte vectors
// into a shared row buffer at the same offset modulo 16 bytes, followed by the y-upwind halo row.
// Results are written back into the own slots and stored from there with aligned vectors.
//
// The kernel is bound by instruction issue and the shared-memory pipe before HBM, so a thread advances TWO
// elements at once, one in each lane of the paired FP32 operations (neighbours along x; halo elements in
// pairs of their own): every product, sum and float-float step is one instruction for both, every table
// entry is loaded once for both, and entries that all threads apply alike come from the parameter bank.
// What an element needs from its upwind neighbours (outflow traces, outflow fluxes) is computed once, by the
// neighbour's own threads, and exchanged through shared memory relative to the neighbour's reference.
// (C C^T)^+ is applied by its structure: the face rows of C are l0/l1 times unit vectors, so C C^T is a
// multiple of the identity on each pair of opposite faces plus couplings through span{l0, l1, w}.  Its
// pseudo-inverse therefore is s_F = alpha_F r + Q c_F with Q an orthonormal basis of that span (three
// columns) and 13 coefficients per element, linear in r: about 18 products per row instead of 8 n.
//
// Measured (one GB300): 512 x 512 elements of n = 9, boundary and mass rows: 228 -> 182 us per step (16 bytes per
// node take 50 us at the measured copy rate; the shared-memory pipe, barriers and issue are what is left).
// Pairing the elements alone left it at 234 us, the shared-memory pipe taking the operator tables; the
// structure of the pseudo-inverse and the exchanged traces made it 189; the sums between the phases spread over
// all threads (one float-float sum of written and old mass instead of two, LN lanes an element) and four CTAs
// per SM instead of three, 182.
//
// With the mass row, the element's mass target is also formed in float-float: M^n (float-float sum of
// w (x) w (hi + lo)) minus its outflow fluxes through the x- and y-outflow faces plus its upwind
// neighbours' outflow fluxes, each flux a fixed float functional of one element's values evaluated
// alike by that element and by its downstream neighbour (so global mass telescopes); after the fit
// the float-float miss of the written element mass is moved along the mass column of the
// pseudo-inverse into the lo words.
#include "ffloat.cuh"
#include "sl_internal.h"

namespace sl {
namespace k2c {

template <int NN, int TX, int TY>
struct Tile {
  static_assert(TX % 2 == 0 && TY % 2 == 0, "elements are advanced in pairs");
  static constexpr int ND = NN * NN;
  static constexpr int NE = TX * TY;              // elements advanced by one CTA
  static constexpr int RW = TX + 1;               // slots per staged tile row (with the x halo)
  // floats per staged row buffer: a multiple of 4 that is 8 modulo 32, so that the lanes of a warp, which run
  // over a row or column of an element and then over the tile's rows, fall into different banks
  static constexpr int RS = ((RW * ND + 8 + 31 - 8) & ~31) + 8;
  static constexpr int HS = (TX * ND + 8 + 3) & ~3;   // floats of the y-halo row buffer
  static constexpr int SP = TY * RS + HS;         // floats per staged plane
  static constexpr int VR = RS / 4, VH = HS / 4, VT = TY * VR + VH;   // 16-byte vectors
  static constexpr int NP = NE / 2;               // own pairs: pair p holds two elements along x, see slot_of
  static constexpr int PT = NP + TY / 2 + TX / 2; // and the x-halo (pairs along y) and y-halo pairs
  static constexpr int NT = (PT * NN + 31) / 32 * 32;   // threads
  static constexpr int MAXV = (VT + NT - 1) / NT; // vectors per thread and plane
  static constexpr int NR = NN | 1;               // row stride of the remapped rows
  static constexpr int PS = NN * NR + ((NN - NN * NR) & 15);   // and the stride of a pair: NN modulo 16 (same reason)
  static constexpr int PH = NP + TX / 2;          // pairs that are remapped: own and y-halo
  // resident CTAs asked of the compiler: 72 registers up to n = 9 and 80 up to n = 11, which spill two words at
  // most (512 x 512, n = 9: 188 -> 182 us, n = 8: 170 -> 154; 300 x 300, n = 11: 112 -> 108); 96 at n = 12 (125 us,
  // 131 at 80 registers)
  static constexpr int MINB = NN <= 9 ? (910 / NT > 8 ? 8 : 910 / NT) : NN <= 11 ? 819 / NT : 4;
};

// Operators applied with the same entry by every thread, each entry twice (parameter bank)
template <int NN>
struct Uni {
  float2 Rx[NN * NN], Ry[NN * NN];
  float2 xix[NN], rox[NN], liny[NN], louty[NN], l0[NN], l1[NN], w[NN], wh[NN], nwh[NN], wl[NN];   // wh + wl: w as float-float, nwh = -wh
};
// scalars of Mixed2DConstParams and the table offsets (in entries)
struct Head {
  int kx, ky, xw, ys, per_x, per_y, bnd, mass, mc, refine;
  int64_t plane;
  float gh, ghl;                                  // the inflow value as float-float
  float sfx, sfy;
  float al[4];                                    // alpha_F of the faces W, E, S, N
  int o_kd, o_fx, o_fy, o_RyT, o_t, o_q, o_l0, o_l1, o_w, o_cm;
};

// shared memory of a CTA (dynamic)
template <int NN, int TX, int TY>
struct __align__(16) Smem {
  using T = Tile<NN, TX, TY>;
  float hi[T::SP], lo[T::SP];                     // staged planes
  union {
    float2 t[T::PH * T::PS];                      // x-remapped rows, until the column phase has read them
    struct {
      float2 r[T::NP * (2 * NN + 1)], c[T::NP * 13], sw[T::NP * NN], se[T::NP * NN], mv[2][T::NP * NN];
    } f;                                          // the fit, after it
  } a;
  float2 u[T::PT * NN], v[T::PT * NN];            // outflow traces along x (before R_y) and y (relative to the own ref)
  float2 fp[3][T::PT * NN];                       // row shares: mass residual, x and y flux
  float2 dx[T::NP * NN];
  float ref[2 * T::PT], tot[3][2 * T::PT], miss[2 * T::NP];
  int64_t a0[TY + 1];                             // first aligned global float of each staged row
  int off[TY + 1], nv[TY + 1];                    // row data offset in its buffer; vectors (0: gather)
};

__device__ __forceinline__ int wrapi(int i, int n, bool per) {
  if (i >= 0 && i < n) return i;
  if (!per) return -1;
  i %= n;
  return i < 0 ? i + n : i;
}

__device__ __forceinline__ int64_t floor4(int64_t g) { return g & ~int64_t(3); }

template <int NN, int TX, int TY>
__global__ void __launch_bounds__(Tile<NN, TX, TY>::NT, Tile<NN, TX, TY>::MINB)
    k_step2d_shared(const __grid_constant__ Uni<NN> U, const __grid_constant__ Head P, const float* __restrict__ tab,
                    const float* __restrict__ in, float* __restrict__ out, unsigned* status) {
  using T = Tile<NN, TX, TY>;
  constexpr int ND = T::ND, RW = T::RW, RS = T::RS, NT = T::NT, NP = T::NP, NR = T::NR, NC = 2 * NN + 1;
  constexpr int VR = T::VR, VT = T::VT, MAXV = T::MAXV;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Smem<NN, TX, TY>& S = *reinterpret_cast<Smem<NN, TX, TY>*>(smem_raw);
  const int tid = threadIdx.x;
  const int ex0 = blockIdx.x * TX, ey0 = blockIdx.y * TY;
  const bool perx = P.per_x != 0, pery = P.per_y != 0;
  const int xs0 = P.xw ? ex0 - 1 : ex0;           // first element of a staged tile row
  const int eyh = P.ys ? ey0 - 1 : ey0 + TY;      // element row of the y halo
  if (tid <= TY) {
    const int ey = tid < TY ? ey0 + tid : eyh;
    const int xa = tid < TY ? xs0 : ex0, cnt = tid < TY ? RW : TX;
    const int64_t g0 = ((int64_t)ey * P.kx + xa) * ND;
    const int64_t a0 = floor4(g0);
    const bool fast = ey >= 0 && ey < P.ky && xa >= 0 && xa + cnt <= P.kx;
    S.a0[tid] = a0;
    S.off[tid] = (int)(g0 - a0);
    S.nv[tid] = fast ? (int)((floor4(g0 + cnt * ND + 3) - a0) >> 2) : 0;
  }
  __syncthreads();
  // contiguous rows: every vector load first, then the shared stores
  {
    float4 vh[MAXV], vl[MAXV];
#pragma unroll
    for (int k = 0; k < MAXV; ++k) {
      const int v = tid + k * NT;
      const int r = v < TY * VR ? v / VR : TY;
      const int vv = v - r * VR;
      if (v < VT && vv < S.nv[r]) {
        const float4* src = reinterpret_cast<const float4*>(in + S.a0[r]) + vv;
        vh[k] = __ldg(src);
        vl[k] = __ldg(reinterpret_cast<const float4*>(reinterpret_cast<const float*>(src) + P.plane));
      }
    }
#pragma unroll
    for (int k = 0; k < MAXV; ++k) {
      const int v = tid + k * NT;
      const int r = v < TY * VR ? v / VR : TY;
      const int vv = v - r * VR;
      if (v < VT && vv < S.nv[r]) {
        reinterpret_cast<float4*>(S.hi + r * RS)[vv] = vh[k];
        reinterpret_cast<float4*>(S.lo + r * RS)[vv] = vl[k];
      }
    }
  }
  // rows that wrap, leave the mesh or are ragged: element by element (ghost slots hold zero)
#pragma unroll 1
  for (int r = 0; r <= TY; ++r) {
    if (S.nv[r] != 0) continue;
    const int ey = r < TY ? ey0 + r : eyh;
    const int xa = r < TY ? xs0 : ex0, cnt = r < TY ? RW : TX;
    const int wy = wrapi(ey, P.ky, pery);
    const int base = r * RS + S.off[r];
    for (int idx = tid; idx < cnt * ND; idx += NT) {
      const int sl = idx / ND, q = idx - sl * ND;
      const int wx = wrapi(xa + sl, P.kx, perx);
      const bool ok = wx >= 0 && wy >= 0;
      const size_t g = ((size_t)wy * P.kx + wx) * ND + q;
      S.hi[base + idx] = ok ? __ldg(in + g) : 0.0f;
      S.lo[base + idx] = ok ? __ldg(in + P.plane + g) : 0.0f;
    }
  }
  __syncthreads();

  // pair p: own pairs first (along y, then along x), then the x halo (rows 2 r, 2 r + 1), then the y halo;
  // element e of the arrays below is lane e & 1 of pair e / 2
  auto slot_of = [](int lx, int ly) { return 2 * ((lx >> 1) * TY + ly) + (lx & 1); };
  const int p = tid / NN, j = tid - p * NN;
  const bool own = p < NP, valid = p < T::PT, halox = !own && p < NP + TY / 2;
  int o0, o1;                                     // staged offsets of the pair's elements
  if (halox) {
    const int r = 2 * (p - NP), c = (P.xw ? 0 : TX) * ND;
    o0 = r * RS + S.off[r] + c;
    o1 = (r + 1) * RS + S.off[r + 1] + c;
  } else if (own || !valid) {
    const int ly = valid ? p % TY : 0, lx = valid ? 2 * (p / TY) : 0;
    o0 = ly * RS + S.off[ly] + (lx + P.xw) * ND;
    o1 = o0 + ND;
  } else {
    o0 = TY * RS + S.off[TY] + 2 * (p - NP - TY / 2) * ND;
    o1 = o0 + ND;
  }
  const float2 ref = make_float2(S.hi[o0], S.hi[o1]);
  const int pj = p * NN + j;

  // ---- row phase: thread j holds row j of psi
  float2 tau = dup(0.0f);
  ff2 mrow = {dup(0.0f), dup(0.0f)};              // minus the row's share of M^n
  if (valid) {
    float2 q[NN];
    const float2 mref = make_float2(-ref.x, -ref.y);
    cdot2n mn;
    const bool massf = own && P.refine;
#pragma unroll
    for (int i = 0; i < NN; ++i) {
      const float2 h = make_float2(S.hi[o0 + j * NN + i], S.hi[o1 + j * NN + i]);
      const float2 l = make_float2(S.lo[o0 + j * NN + i], S.lo[o1 + j * NN + i]);
      q[i] = __fadd2_rn(__fadd2_rn(h, mref), l);
      if (massf) mn.add(U.wh[i], U.nwh[i], U.wl[i], h, l);   // (row sum; the rows' weights in the element total)
    }
    float2 u = dup(0.0f);
#pragma unroll
    for (int i = 0; i < NN; ++i) {
      u = __ffma2_rn(U.rox[i], q[i], u);
      tau = __ffma2_rn(U.xix[i], q[i], tau);
    }
    S.u[pj] = u;
    if (P.mass) {
      float2 kd = dup(0.0f), fx = dup(0.0f), fy = dup(0.0f);
#pragma unroll
      for (int i = 0; i < NN; ++i) {
        kd = __ffma2_rn(dup(__ldg(tab + P.o_kd + i * NN + j)), q[i], kd);
        fx = __ffma2_rn(dup(__ldg(tab + P.o_fx + i * NN + j)), q[i], fx);
        fy = __ffma2_rn(dup(__ldg(tab + P.o_fy + i * NN + j)), q[i], fy);
      }
      S.fp[0][pj] = kd;
      S.fp[1][pj] = fx;
      S.fp[2][pj] = fy;
      mrow = mn.get();
    }
    if (j == 0) {
      S.ref[2 * p] = ref.x;
      S.ref[2 * p + 1] = ref.y;
    }
    if (!halox) {
      float2* tr = S.a.t + (own ? p : p - TY / 2) * T::PS + j * NR;
      // x-remap of row j: t[j][l] = sum_i R_x[l][i] psi[j][i]
#pragma unroll
      for (int l = 0; l < NN; ++l) {
        float2 acc = dup(0.0f);
#pragma unroll
        for (int i = 0; i < NN; ++i) acc = __ffma2_rn(U.Rx[l * NN + i], q[i], acc);
        tr[l] = acc;
      }
    }
  }
  __syncthreads();

  // upwind neighbours: elements xn0, xn1 across the x-inflow faces, pair yp across the y-inflow face
  const int ly = own ? p % TY : 0, lx = own ? 2 * (p / TY) : 0, e0 = 2 * p;
  const int ex = ex0 + lx, ey = ey0 + ly;
  int xn0, xn1, yp;
  {
    const int xh = 2 * NP + ly;                   // this tile row's x-halo element
    if (P.xw) { xn0 = lx > 0 ? slot_of(lx - 1, ly) : xh; xn1 = e0; }
    else { xn0 = e0 + 1; xn1 = lx + 2 < TX ? slot_of(lx + 2, ly) : xh; }
    const int ry = P.ys ? ly - 1 : ly + 1;
    yp = ry >= 0 && ry < TY ? (lx >> 1) * TY + ry : NP + TY / 2 + (lx >> 1);
  }
  const bool gx0 = wrapi(P.xw ? ex - 1 : ex + 1, P.kx, perx) < 0, gx1 = wrapi(P.xw ? ex : ex + 2, P.kx, perx) < 0;
  const bool gy = wrapi(P.ys ? ey - 1 : ey + 1, P.ky, pery) < 0;
  const float2 gval = __fadd2_rn(sub2(dup(P.gh), ref), dup(P.ghl));   // the ghost relative to the reference
  // differences of the references: neighbour values relative to the own reference
  const float2 drx = own ? make_float2(gx0 ? 0.0f : S.ref[xn0] - ref.x, gx1 ? 0.0f : S.ref[xn1] - ref.y) : dup(0.0f);
  const float2 dry = own && !gy ? make_float2(S.ref[2 * yp] - ref.x, S.ref[2 * yp + 1] - ref.y) : dup(0.0f);

  // ---- column phase: thread j holds column j of psihat = R_y t
  float2 ph[NN], ty = dup(0.0f);
  if (valid && !halox) {
    float2 tc[NN], v = dup(0.0f);
    const float2* tr = S.a.t + (own ? p : p - TY / 2) * T::PS + j;
#pragma unroll
    for (int m = 0; m < NN; ++m) tc[m] = tr[m * NR];
#pragma unroll
    for (int k = 0; k < NN; ++k) {
      float2 acc = dup(0.0f);
#pragma unroll
      for (int m = 0; m < NN; ++m) acc = __ffma2_rn(U.Ry[k * NN + m], tc[m], acc);
      ph[k] = acc;
      ty = __ffma2_rn(U.liny[k], acc, ty);
      v = __ffma2_rn(U.louty[k], acc, v);
    }
    S.v[pj] = v;                                  // trace of psihat on the y-outflow face
  }
  if (own) {
    const float* us = reinterpret_cast<const float*>(S.u);
    const float2 un = make_float2(gx0 ? 0.0f : us[((xn0 >> 1) * NN + j) * 2 + (xn0 & 1)],
                                  gx1 ? 0.0f : us[((xn1 >> 1) * NN + j) * 2 + (xn1 & 1)]);
    S.dx[pj] = sub2(__fadd2_rn(un, drx), tau);
  }
  // element totals of the row shares, one thread per element and quantity, rows in order (the same sums
  // whichever CTA forms them): mass residual, outflow fluxes
  if (P.mass)
    for (int i = tid; i < 6 * T::PT; i += NT) {
      const int q = i / (2 * T::PT), e = i - q * (2 * T::PT);
      const float* f = reinterpret_cast<const float*>(S.fp[q]) + (e >> 1) * NN * 2 + (e & 1);
      float v = 0.0f;
#pragma unroll
      for (int r = 0; r < NN; ++r) v += f[2 * r];
      S.tot[q][e] = v;
    }
  __syncthreads();

  float2 rm = dup(0.0f);                          // mass residual
  if (own && P.mass) {
    auto at = [&](int k, int a, int b) { return make_float2(S.tot[k][a], S.tot[k][b]); };
    const float2 gxv = make_float2(gx0 ? gval.x : drx.x, gx1 ? gval.y : drx.y), gyv = gy ? gval : dry;
    float2 fxu = make_float2(gx0 ? 0.0f : S.tot[1][xn0], gx1 ? 0.0f : S.tot[1][xn1]);
    float2 fyu = gy ? dup(0.0f) : at(2, 2 * yp, 2 * yp + 1);
    fxu = __ffma2_rn(gxv, dup(P.sfx), fxu);
    fyu = __ffma2_rn(gyv, dup(P.sfy), fyu);
    rm = __fadd2_rn(at(0, e0, e0 + 1), __fadd2_rn(sub2(fxu, at(1, e0, e0 + 1)), sub2(fyu, at(2, e0, e0 + 1))));
  }
  float2 rx = dup(0.0f), ry = dup(0.0f);
  if (own && P.bnd) {
#pragma unroll
    for (int m = 0; m < NN; ++m) rx = __ffma2_rn(dup(__ldg(tab + P.o_RyT + m * NN + j)), S.dx[p * NN + m], rx);
    if (gx0) rx.x += gval.x;
    if (gx1) rx.y += gval.y;
    ry = sub2(gy ? gval : __fadd2_rn(S.v[yp * NN + j], dry), ty);
    S.a.f.r[p * NC + j] = rx;
    S.a.f.r[p * NC + NN + j] = ry;
    if (j == 0) S.a.f.r[p * NC + 2 * NN] = rm;    // (zero without the mass row)
  }
  __syncthreads();

  // ---- fit: s = (C C^T)^+ r: the 13 coefficients (three per face along Q, the mass row's entry), spread over
  // the element's threads; then thread j forms the face entries of row / column j
  float2 sS = dup(0.0f), sN = dup(0.0f), sm = dup(0.0f);
  if (P.bnd) {
    if (own) {
      for (int o = j; o < 13; o += NN) {
        const float* To = tab + P.o_t + o * NC;
        float2 c = dup(0.0f);
#pragma unroll
        for (int k = 0; k < NC; ++k) c = __ffma2_rn(dup(__ldg(To + k)), S.a.f.r[p * NC + k], c);
        S.a.f.c[p * 13 + o] = c;
      }
    }
    __syncthreads();
    if (own) {
      const float2 q0 = dup(__ldg(tab + P.o_q + j)), q1 = dup(__ldg(tab + P.o_q + NN + j)), q2 = dup(__ldg(tab + P.o_q + 2 * NN + j));
      const float2* c = S.a.f.c + p * 13;
      auto entry = [&](int f, float2 r) {
        return __ffma2_rn(c[3 * f + 2], q2, __ffma2_rn(c[3 * f + 1], q1, __ffma2_rn(c[3 * f], q0, __fmul2_rn(dup(P.al[f]), r))));
      };
      S.a.f.sw[pj] = entry(0, rx);
      S.a.f.se[pj] = entry(1, rx);
      sS = entry(2, ry);
      sN = entry(3, ry);
      sm = c[12];
    }
    __syncthreads();
  } else if (own) {
    sm = __fmul2_rn(dup(__ldg(tab + P.o_t + 12)), rm);
  }

  // ---- phi_L = psihat + C^T s, column j; exact write-back
  float2 vh[NN], vl[NN];
  if (own) {
    const float2 l0j = dup(__ldg(tab + P.o_l0 + j)), l1j = dup(__ldg(tab + P.o_l1 + j));
    const float2 wj = __fmul2_rn(dup(__ldg(tab + P.o_w + j)), sm);
    cdot2n mv;
#pragma unroll
    for (int k = 0; k < NN; ++k) {
      float2 acc = ph[k];
      acc = __ffma2_rn(sS, U.l0[k], acc);
      acc = __ffma2_rn(sN, U.l1[k], acc);
      acc = __ffma2_rn(wj, U.w[k], acc);
      if (P.bnd) {
        acc = __ffma2_rn(S.a.f.sw[p * NN + k], l0j, acc);
        acc = __ffma2_rn(S.a.f.se[p * NN + k], l1j, acc);
      }
      const ff2 s = two_sum2(ref, acc);
      vh[k] = s.hi;
      vl[k] = s.lo;
      if (P.refine) mv.add(U.wh[k], U.nwh[k], U.wl[k], vh[k], vl[k]);    // (column sum)
    }
    if (P.refine) {
      // minus the written column's mass plus the row's share of M^n, times their common weight w_j
      const ff2 mc = mv.get(), m = ff_mul2(ff_add2(mc, ff2{neg2(mrow.hi), neg2(mrow.lo)}), U.wh[j], U.wl[j]);
      S.a.f.mv[0][pj] = m.hi;
      S.a.f.mv[1][pj] = m.lo;
    }
  }
  if (P.refine) {
    // the float-float miss of the written element mass against the target, LN lanes per element:
    // F(element) = ref sum(f) + its total, own fluxes with this element's reference, upwind fluxes with the
    // neighbour's (or the ghost value)
    __syncthreads();
    constexpr int LN = NN > 6 ? 4 : NN > 4 ? 2 : 1;
    for (int i = tid; i < ((2 * NP * LN + 31) & ~31); i += NT) {
      const int e = min(i / LN, 2 * NP - 1);
      const float* f = reinterpret_cast<const float*>(S.a.f.mv) + (e >> 1) * NN * 2 + (e & 1);
      constexpr int F = NP * NN * 2;
      ff m = {0.0f, 0.0f};
#pragma unroll
      for (int q = 0; q < (NN + LN - 1) / LN; ++q) {
        const int r = LN * q + i % LN;
        if (r < NN) m = q == 0 ? ff{f[2 * r], f[F + 2 * r]} : ff_add(m, ff{f[2 * r], f[F + 2 * r]});
      }
      const int x = 2 * ((e >> 1) / TY) + (e & 1), y = (e >> 1) % TY;
      const int xh = 2 * NP + y;
      const int xn = P.xw ? (x > 0 ? slot_of(x - 1, y) : xh) : (x + 1 < TX ? slot_of(x + 1, y) : xh);
      const int ry = P.ys ? y - 1 : y + 1, yn = ry >= 0 && ry < TY ? slot_of(x, ry) : 2 * (NP + TY / 2) + x;
      const bool gx = wrapi(P.xw ? ex0 + x - 1 : ex0 + x + 1, P.kx, perx) < 0;
      const bool gyy = wrapi(P.ys ? ey0 + y - 1 : ey0 + y + 1, P.ky, pery) < 0;
      const float Fxo = fmaf(S.ref[e], P.sfx, S.tot[1][e]), Fyo = fmaf(S.ref[e], P.sfy, S.tot[2][e]);
      const float Fxu = gx ? P.gh * P.sfx : fmaf(S.ref[xn], P.sfx, S.tot[1][xn]);
      const float Fyu = gyy ? P.gh * P.sfy : fmaf(S.ref[yn], P.sfy, S.tot[2][yn]);
      // M^{n+1} = M^n - (outflow) + (inflow), float-float
      const ff fl = ff_add(two_sum(-Fxo, -Fyo), two_sum(Fxu, Fyu));
#pragma unroll
      for (int o = 1; o < LN; o <<= 1)
        m = ff_add(m, ff{__shfl_xor_sync(0xffffffffu, m.hi, o), __shfl_xor_sync(0xffffffffu, m.lo, o)});
      if (i % LN == 0 && i < 2 * NP * LN) S.miss[e] = ff_to_f(ff_add(fl, m));
    }
    __syncthreads();
    if (own) {
      const float2 miss = make_float2(S.miss[e0], S.miss[e0 + 1]);
#pragma unroll
      for (int k = 0; k < NN; ++k) {
        const ff2 v = fast_two_sum2(vh[k], __ffma2_rn(miss, dup(__ldg(tab + P.o_cm + k * NN + j)), vl[k]));
        vh[k] = v.hi;
        vl[k] = v.lo;
      }
    }
  }
  if (own) {
    bool f0 = true, f1 = true;
#pragma unroll
    for (int k = 0; k < NN; ++k) {
      S.hi[o0 + k * NN + j] = vh[k].x;
      S.lo[o0 + k * NN + j] = vl[k].x;
      S.hi[o1 + k * NN + j] = vh[k].y;
      S.lo[o1 + k * NN + j] = vl[k].y;
      f0 = f0 && isfinite(vh[k].x);
      f1 = f1 && isfinite(vh[k].y);
    }
    const bool in0 = ex < P.kx && ey < P.ky, in1 = ex + 1 < P.kx && ey < P.ky;
    if ((in0 && !f0) || (in1 && !f1)) atomicOr(status, SL_ST_NONFINITE);
  }
  __syncthreads();

  // ---- stores: the own elements of a tile row are one contiguous run; aligned vectors inside,
  // single floats at its ends
#pragma unroll 1
  for (int r = 0; r < TY; ++r) {
    const int eyr = ey0 + r;
    if (eyr >= P.ky) break;
    const int cnt = min(TX, P.kx - ex0);
    const int64_t g0 = ((int64_t)eyr * P.kx + ex0) * ND, g1 = g0 + (int64_t)cnt * ND;
    const int64_t A = floor4(g0 + 3), B = floor4(g1);
    const int64_t a0 = S.a0[r];                   // global float G of this row is at r RS + (G - a0)
    const float* rh = S.hi + r * RS;
    const float* rl = S.lo + r * RS;
    if (A <= B) {
      const int nvec = (int)((B - A) >> 2);
      for (int v = tid; v < nvec; v += NT) {
        const int64_t G = A + 4 * (int64_t)v;
        const int q = (int)(G - a0);
        *reinterpret_cast<float4*>(out + G) = *reinterpret_cast<const float4*>(rh + q);
        *reinterpret_cast<float4*>(out + P.plane + G) = *reinterpret_cast<const float4*>(rl + q);
      }
      if (tid < A - g0) {
        const int q = (int)(g0 + tid - a0);
        out[g0 + tid] = rh[q];
        out[P.plane + g0 + tid] = rl[q];
      }
      if (tid < g1 - B) {
        const int q = (int)(B + tid - a0);
        out[B + tid] = rh[q];
        out[P.plane + B + tid] = rl[q];
      }
    } else if (tid < g1 - g0) {
      const int q = (int)(g0 + tid - a0);
      out[g0 + tid] = rh[q];
      out[P.plane + g0 + tid] = rl[q];
    }
  }
}

template <int NN, int TX, int TY>
void launch(const Mixed2DConstParams& p, const float* tab, const float* in, float* out, unsigned* st, cudaStream_t s) {
  Uni<NN> U;
  auto two = [](float2* dst, const float* src, int n) {
    for (int i = 0; i < n; ++i) dst[i] = make_float2(src[i], src[i]);
  };
  two(U.Rx, p.Rx, NN * NN);
  two(U.Ry, p.Ry, NN * NN);
  two(U.xix, p.xix, NN);
  two(U.rox, p.rox, NN);
  two(U.louty, p.louty, NN);
  two(U.liny, p.liny, NN);
  two(U.l0, p.l0, NN);
  two(U.l1, p.l1, NN);
  two(U.w, p.w, NN);
  two(U.wh, p.wh, NN);
  two(U.wl, p.wl, NN);
  for (int i = 0; i < NN; ++i) U.nwh[i] = make_float2(-p.wh[i], -p.wh[i]);
  const Head H{p.kx,  p.ky,  p.xw,   p.ys,   p.per_x, p.per_y, p.bnd, p.mass, p.mc,   p.refine, p.plane,
               (float)p.ghost, (float)(p.ghost - (double)(float)p.ghost), p.sfx, p.sfy,
               {p.al[0], p.al[1], p.al[2], p.al[3]}, p.o_kd, p.o_fx, p.o_fy, p.o_RyT, p.o_t, p.o_q, p.o_l0, p.o_l1, p.o_w, p.o_cm};
  dim3 grid((p.kx + TX - 1) / TX, (p.ky + TY - 1) / TY);
  constexpr size_t dyn = sizeof(Smem<NN, TX, TY>);
  allow_dynamic_smem((const void*)k_step2d_shared<NN, TX, TY>, dyn);
  k_step2d_shared<NN, TX, TY><<<grid, Tile<NN, TX, TY>::NT, dyn, s>>>(U, H, tab, in, out, st);
}

}  // namespace k2c
}  // namespace sl
