#pragma once
// 1D DSEM-SL step in double precision, one thread per element (Sec. 4, steps a-d).
//
// A CTA of b threads owns b-2 consecutive elements plus one halo element on each side.  Phase 1 (every
// thread, halo included): seed particles at the Gauss nodes, integrate them with explicit RK (eq. 4.4a,
// 4.8), remap by interpolation through the advected nodes (eq. 4.9), take the two face traces (eq.
// remap_bnd, or eq. 4.11 when backtracking), and integrate the outflow mass/energy flux through each face
// over the step.  These six numbers go to shared memory.  Phase 2 (core threads): upwind the interface
// values (eq. 4.12a), form the mass/energy targets (eq. remap_mass, remap_energy), apply the constrained
// fit (eq. matrix_a) and the energy iteration, and store phi^{n+1}.  Nothing but the state is read from or
// written to global memory; halo elements are recomputed.
//
// Bound by the FP64 pipe (one FP64 warp instruction per 16 cycles and SM), so each velocity takes the form
// with the fewest FP64 instructions:
//   - constant (k_step1d_shift): the displacement is the same for every element, so the remap and the flux
//     feet are matrices built once on the host and applied as DFMAs whose matrix entry comes from the
//     parameter bank;
//   - u = -sin x (k_step1d_f64<n, true>): one sincos per element, at its centre; node and face sines follow
//     by angle addition with offsets common to all elements, displaced ones with a Taylor series of the
//     small angle;
//   - a velocity given at the nodes: k_step1d_f64<n, false>.
// Measured (one GB300): constant velocity, K = 2^20, n = 9, every constraint: 2.69 -> 0.53 ms (FP64 pipe 86 %
// busy, 8.7 M FP64 warp instructions); K = 16: 41 -> 8.2 us, launch bound; u = -sin x, K = 30011, n = 7:
// 148 -> 70 us (1.77 -> 0.96 M FP64 warp instructions).
#include <algorithm>
#include <cfloat>
#include <cmath>

#include "sl_internal.h"

namespace sl {
namespace k1d {

constexpr int BLOCK = 128;                // threads of a CTA at most

static __constant__ int c_rk_s[5] = {0, 1, 2, 3, 4};
static __constant__ double c_rk_a[5][4][4] = {
    {},
    {{0}},
    {{0, 0}, {1.0, 0}},
    {{0, 0, 0}, {0.5, 0, 0}, {-1.0, 2.0, 0}},
    {{0, 0, 0, 0}, {0.5, 0, 0, 0}, {0, 0.5, 0, 0}, {0, 0, 1.0, 0}}};
static __constant__ double c_rk_b[5][4] = {
    {}, {1.0}, {0.5, 0.5}, {1.0 / 6, 2.0 / 3, 1.0 / 6}, {1.0 / 6, 1.0 / 3, 1.0 / 3, 1.0 / 6}};
static __constant__ double c_rk_c[5][4] = {{}, {0.0}, {0.0, 1.0}, {0.0, 0.5, 1.0}, {0.0, 0.5, 0.5, 1.0}};

// value at reference point z of the polynomial with nodal values v on nodes xn (barycentric
// weights lam): sum_j lam_j prod_{m != j} (z - xn_m) v_j, by prefix/suffix products
template <int NN>
__device__ __forceinline__ double eval_poly(const double* xn, const double* lam, const double* v, double z) {
  double d[NN], pre[NN];
#pragma unroll
  for (int m = 0; m < NN; ++m) d[m] = z - xn[m];
  double acc = 1.0;
#pragma unroll
  for (int m = 0; m < NN; ++m) { pre[m] = acc; acc *= d[m]; }
  double suf = 1.0, out = 0.0;
#pragma unroll
  for (int j = NN - 1; j >= 0; --j) {
    out += lam[j] * pre[j] * suf * v[j];
    suf *= d[j];
  }
  return out;
}

// the same polynomial and its derivative in z: the prefix and suffix products carry their
// derivatives along (product rule), so nodes need no special case
template <int NN>
__device__ __forceinline__ void eval_poly_d(const double* xn, const double* lam, const double* v, double z,
                                            double& val, double& der) {
  double d[NN], pre[NN], dpre[NN];
#pragma unroll
  for (int m = 0; m < NN; ++m) d[m] = z - xn[m];
  double acc = 1.0, dacc = 0.0;
#pragma unroll
  for (int m = 0; m < NN; ++m) {
    pre[m] = acc;
    dpre[m] = dacc;
    dacc = dacc * d[m] + acc;
    acc *= d[m];
  }
  double suf = 1.0, dsuf = 0.0, out = 0.0, dout = 0.0;
#pragma unroll
  for (int j = NN - 1; j >= 0; --j) {
    const double c = lam[j] * v[j];
    out += c * pre[j] * suf;
    dout += c * (dpre[j] * suf + pre[j] * dsuf);
    dsuf = dsuf * d[j] + suf;
    suf *= d[j];
  }
  val = out;
  der = dout;
}

// SL_VEL_NODAL in 1D: the node velocities of element k at time t (linear between the step's
// two arrays), evaluated with their derivative at reference point z
template <int NN>
__device__ __forceinline__ void nodal_elem1d(const StepParams& P, const double* xi, const double* lam, int k,
                                             double z, double th, double& u, double& du) {
  const double* U0 = P.nodal + (size_t)k * NN;
  const double* U1 = U0 + P.nvals;
  double v[NN];
#pragma unroll
  for (int j = 0; j < NN; ++j) v[j] = (1.0 - th) * U0[j] + th * U1[j];
  eval_poly_d<NN>(xi, lam, v, z, u, du);
}

// the nodal field at physical x: the containing element's interpolant (the boundary element's
// beyond a non-periodic face, wrapped across a periodic one); on a face the average over the
// elements that share it
template <int NN>
__device__ void nodal1d(const StepParams& P, const double* xi, const double* lam, double x, double t, double& u,
                        double& dv) {
  const double h = P.hx, x1 = P.x0 + P.K * h;
  const double th = (t - P.t) / P.dt;
  const double s = (x - P.x0) / h;
  const double r = rint(s);
  const bool perW = P.bc[0] == SL_BC_PERIODIC, perE = P.bc[1] == SL_BC_PERIODIC;
  u = 0.0;
  dv = 0.0;
  if (fabs(x - (P.x0 + r * h)) <= FACE_RTOL * (fabs(P.x0) + fabs(x1))) {
    int ks[2];
    double zs[2];
    int cnt = 0;
    const long long ri = (long long)r;
#pragma unroll
    for (int side = 0; side < 2; ++side) {
      long long k = side ? ri : ri - 1;
      if (k < 0 || k >= P.K) {
        if (!(k < 0 ? perW : perE)) continue;
        k %= P.K;
        if (k < 0) k += P.K;
      }
      ks[cnt] = (int)k;
      zs[cnt] = side ? 0.0 : 1.0;
      ++cnt;
    }
    for (int q = 0; q < cnt; ++q) {
      double uq, dq;
      nodal_elem1d<NN>(P, xi, lam, ks[q], zs[q], th, uq, dq);
      u += uq / cnt;
      dv += dq / h / cnt;
    }
    return;
  }
  const double fk = floor(s);
  long long k = (long long)fk;
  double z = s - fk;
  if (k < 0 || k >= P.K) {
    if (k < 0 ? perW : perE) {
      k %= P.K;
      if (k < 0) k += P.K;
    } else {
      k = k < 0 ? 0 : P.K - 1;
      z = s - (double)k;
    }
  }
  double du;
  nodal_elem1d<NN>(P, xi, lam, (int)k, z, th, u, du);
  dv = du / h;
}

// one explicit RK step of dx/dt = u, dphi/dt = -phi div u through the nodal velocity, size h (h < 0 runs
// backward)
template <int NN>
__device__ __forceinline__ void rk_step(const StepParams& P, const double* xi, const double* lam, double& x,
                                        double& ph, double t, double h) {
  const int S = c_rk_s[P.rk];
  double kx[4], kp[4];
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    if (s < S) {
      double xs = x, ps = ph;
#pragma unroll
      for (int j = 0; j < s; ++j) {
        xs += h * c_rk_a[P.rk][s][j] * kx[j];
        ps += h * c_rk_a[P.rk][s][j] * kp[j];
      }
      double u, dv;
      nodal1d<NN>(P, xi, lam, xs, t + c_rk_c[P.rk][s] * h, u, dv);
      kx[s] = u;
      kp[s] = -ps * dv;
    }
  }
  double sx = 0.0, sp = 0.0;
#pragma unroll
  for (int s = 0; s < 4; ++s)
    if (s < S) {
      sx += c_rk_b[P.rk][s] * kx[s];
      sp += c_rk_b[P.rk][s] * kp[s];
    }
  x += h * sx;
  ph += h * sp;
}

// ------------------------------------------------------------------ u = -sin x
// sine and cosine of A + x from those of A by the Taylor series of the small angle (ser 0: |x| <= 0.0039,
// 1: |x| <= 0.05; remainders below 1e-17 and 1e-19), or directly at the point z = A + x (ser 2)
__device__ __forceinline__ void add_angle(int ser, double x, double A, double S, double C, double& s, double& c) {
  if (ser == 2) {
    sincos(A + x, &s, &c);
    return;
  }
  const double x2 = x * x;
  double ps = fma(x2, 1.0 / 120, -1.0 / 6), pc = fma(x2, 1.0 / 24, -0.5);
  if (ser) {
    ps = fma(x2, fma(x2, fma(x2, 1.0 / 362880, -1.0 / 5040), 1.0 / 120), -1.0 / 6);
    pc = fma(x2, fma(x2, fma(x2, 1.0 / 40320, -1.0 / 720), 1.0 / 24), -0.5);
  }
  const double sn = fma(x * x2, ps, x), cm = x2 * pc;
  s = fma(S, cm, fma(C, sn, S));
  c = fma(C, cm, fma(-S, sn, C));
}

template <int RK>
struct Tab {
  __device__ static constexpr double a(int s, int j) {
    return RK == 2 ? (s == 1 && j == 0 ? 1.0 : 0.0)
         : RK == 3 ? (s == 1 && j == 0 ? 0.5 : s == 2 && j == 0 ? -1.0 : s == 2 && j == 1 ? 2.0 : 0.0)
         : RK == 4 ? ((s == 1 && j == 0) || (s == 2 && j == 1) ? 0.5 : s == 3 && j == 2 ? 1.0 : 0.0)
                   : 0.0;
  }
  __device__ static constexpr double b(int s) {
    return RK == 1 ? 1.0 : RK == 2 ? 0.5 : RK == 3 ? (s == 1 ? 2.0 / 3 : 1.0 / 6) : (s == 0 || s == 3 ? 1.0 / 6 : 1.0 / 3);
  }
};

// one RK step of size h through u = -sin x from the point A (sine S, cosine C) with value v: the
// displacement and the new value (D phi / Dt = -phi div u = phi cos x)
template <int RK>
__device__ __noinline__ double2 rk_sinx_t(int ser, double A, double S, double C, double v, double h) {
  using T = Tab<RK>;
  double kx[RK], kp[RK];
#pragma unroll
  for (int s = 0; s < RK; ++s) {
    double ss = S, cc = C, vs = v;
    if (s > 0) {
      double xs = 0.0;
#pragma unroll
      for (int j = 0; j < s; ++j)
        if (T::a(s, j) != 0.0) {
          xs = fma(h * T::a(s, j), kx[j], xs);
          vs = fma(h * T::a(s, j), kp[j], vs);
        }
      add_angle(ser, xs, A, S, C, ss, cc);
    }
    kx[s] = -ss;
    kp[s] = vs * cc;
  }
  double sx = T::b(0) * kx[0], sp = T::b(0) * kp[0];
#pragma unroll
  for (int s = 1; s < RK; ++s) {
    sx = fma(T::b(s), kx[s], sx);
    sp = fma(T::b(s), kp[s], sp);
  }
  return make_double2(h * sx, fma(h, sp, v));
}

__device__ __forceinline__ double2 rk_sinx(int rk, int ser, double A, double S, double C, double v, double h) {
  switch (rk) {
    case 4: return rk_sinx_t<4>(ser, A, S, C, v, h);
    case 3: return rk_sinx_t<3>(ser, A, S, C, v, h);
    case 2: return rk_sinx_t<2>(ser, A, S, C, v, h);
    default: return rk_sinx_t<1>(ser, A, S, C, v, h);
  }
}

static __constant__ int c_ds_n[5] = {0, 1, 2, 3, 3};        // distinct stage times, summed weights
static __constant__ double c_ds_c[5][3] = {{}, {0.0}, {0.0, 1.0}, {0.0, 0.5, 1.0}, {0.0, 0.5, 1.0}};
static __constant__ double c_ds_b[5][3] = {
    {}, {1.0}, {0.5, 0.5}, {1.0 / 6, 2.0 / 3, 1.0 / 6}, {1.0 / 6, 2.0 / 3, 1.0 / 6}};

// sum_j c_j prod_{m != j} d_m by prefix and suffix products
template <int NN>
__device__ __forceinline__ double sum_products(const double (&d)[NN], const double (&c)[NN]) {
  double pre[NN];
  pre[0] = 1.0;
#pragma unroll
  for (int m = 1; m < NN; ++m) pre[m] = m == 1 ? d[0] : pre[m - 1] * d[m - 1];
  double suf = d[NN - 1], out = c[NN - 1] * pre[NN - 1];
#pragma unroll
  for (int j = NN - 2; j >= 0; --j) {
    out = fma(c[j], j == 0 ? suf : pre[j] * suf, out);
    suf *= d[j];
  }
  return out;
}

struct Smem1D {
  double xi[NMAX], w[NMAX], lam[NMAX], l0[NMAX], l1[NMAX];
  double Cp[3][NMAX], SCt[3][NMAX];   // columns of the rows left, right, mass (as many as are active)
  double S[NMAX * NMAX];
  double tr[2][BLOCK];       // face traces at t^{n+1}
  double fm[2][BLOCK];       // outflow mass flux per face
  double fe[2][BLOCK];       // outflow energy flux per face
};

__device__ __forceinline__ int wrap_elem(int e, int K, bool periodic) {
  if (e >= 0 && e < K) return e;
  if (!periodic) return -1;
  e %= K;
  return e < 0 ? e + K : e;
}

template <int NN>
__device__ __forceinline__ void load_tables(const StepParams& P, const Tables1D& tb, Smem1D& sm) {
  const int tid = threadIdx.x, nt = blockDim.x, m = P.m;
  const int col0 = P.cons & SL_C_BOUNDARY ? 0 : 2;           // first column of an active row
  for (int i = tid; i < NN; i += nt) {
    sm.xi[i] = tb.xi[i]; sm.w[i] = tb.w[i]; sm.lam[i] = tb.lam[i];
    sm.l0[i] = tb.l0[i]; sm.l1[i] = tb.l1[i];
  }
  if (P.fit == SL_FIT_HARD) {
    for (int i = tid; i < NN * m; i += nt) sm.Cp[col0 + i % m][i / m] = tb.Cpinv[i];
  } else {
    for (int i = tid; i < NN * m; i += nt) sm.SCt[col0 + i % m][i / m] = tb.SCt[i];
    for (int i = tid; i < NN * NN; i += nt) sm.S[i] = tb.S[i];
  }
}

// whether a double is finite, from its high word (an integer test)
__device__ __forceinline__ bool finite64(double v) { return (__double2hiint(v) & 0x7ff00000) != 0x7ff00000; }

// Phase 2 of element e (eraw before the periodic wrap): phi its values, ph its remap, dm the mass of phi less
// that of ph (read by the hard fit with the mass row); uface(side, c): the velocity at a face at t + c dt
template <int NN, typename UF>
__device__ __forceinline__ void phase2(const StepParams& P, const Smem1D& sm, int e, int eraw, const double (&phi)[NN],
                                       const double (&ph)[NN], double dm, UF uface, double* __restrict__ out,
                                       unsigned* status) {
  const int tid = threadIdx.x, K = P.K;
  const double lam = P.lam;              // dt / h
  const bool perW = P.bc[0] == SL_BC_PERIODIC, perE = P.bc[1] == SL_BC_PERIODIC;
  const bool bnd = (P.cons & SL_C_BOUNDARY) != 0, mass = (P.cons & SL_C_MASS) != 0;
  double d[3] = {0.0, 0.0, 0.0};        // right-hand sides of the rows left, right, mass
  double netm = 0.0, nete = 0.0;        // net outward flux (mass, energy) through both faces
#pragma unroll
  for (int side = 0; side < 2; ++side) {
    const int nbraw = side ? eraw + 1 : eraw - 1;
    const bool onbnd = nbraw < 0 || nbraw >= K;
    const bool per = side ? perE : perW;
    const bool ghostface = onbnd && !per;
    const int nbt = side ? tid + 1 : tid - 1;     // neighbour's thread in this CTA
    if (bnd) {
      const double u = uface(side, 1.0);
      const double un = side ? u : -u;
      const double own = sm.tr[side][tid];
      const double other = ghostface ? (P.gtab ? P.gtab[side * 5] : P.ghost) : sm.tr[1 - side][nbt];
      double val;
      if (un > TIE) val = own;
      else if (un < -TIE) val = other;
      else val = ghostface ? own : 0.5 * (own + other);
      d[side] = val;
    }
    if (P.cons & (SL_C_MASS | SL_C_ENERGY)) {
      netm += sm.fm[side][tid];
      nete += sm.fe[side][tid];
      if (!ghostface) {
        netm -= sm.fm[1 - side][nbt];
        nete -= sm.fe[1 - side][nbt];
      } else {
        const int S = c_rk_s[P.rk];
        for (int s = 0; s < S; ++s) {
          const double u = uface(side, c_rk_c[P.rk][s]);
          const double un = side ? u : -u;
          if (un < -TIE) {
            const double g = P.gtab ? P.gtab[side * 5 + 1 + s] : P.ghost;
            netm += c_rk_b[P.rk][s] * un * g;
            nete += c_rk_b[P.rk][s] * un * g * g;
          }
        }
      }
    }
  }
  // linear constrained fit; rows are skipped where their residual vanishes (an outflow face's own trace)
  double phL[NN];
  if (P.fit == SL_FIT_HARD) {
    double r0 = 0.0, r1 = 0.0, r2 = 0.0;
    if (bnd) {
      // with interpolated interface values the stored traces are those of phihat
      double c0 = sm.tr[0][tid], c1 = sm.tr[1][tid];
      if (P.bvalue == SL_BV_BACKTRACK) {
        c0 = c1 = 0.0;
#pragma unroll
        for (int j = 0; j < NN; ++j) { c0 += sm.l0[j] * ph[j]; c1 += sm.l1[j] * ph[j]; }
      }
      r0 = d[0] - c0;
      r1 = d[1] - c1;
    }
    if (mass) r2 = dm - lam * netm;       // reference-measure target (eq. remap_mass) less the mass of ph
#pragma unroll
    for (int j = 0; j < NN; ++j) phL[j] = ph[j];
    if (r0 != 0.0) {
#pragma unroll
      for (int j = 0; j < NN; ++j) phL[j] += sm.Cp[0][j] * r0;
    }
    if (r1 != 0.0) {
#pragma unroll
      for (int j = 0; j < NN; ++j) phL[j] += sm.Cp[1][j] * r1;
    }
    if (mass) {
#pragma unroll
      for (int j = 0; j < NN; ++j) phL[j] += sm.Cp[2][j] * r2;
    }
  } else {
    if (mass) {
      double Mn = 0.0;
#pragma unroll
      for (int i = 0; i < NN; ++i) Mn += sm.w[i] * phi[i];
      d[2] = Mn - lam * netm;
    }
#pragma unroll
    for (int j = 0; j < NN; ++j) {
      double acc = 0.0;
#pragma unroll
      for (int k = 0; k < NN; ++k) acc += sm.S[j * NN + k] * ph[k];
      if (bnd) acc += sm.SCt[0][j] * d[0] + sm.SCt[1][j] * d[1];
      if (mass) acc += sm.SCt[2][j] * d[2];
      phL[j] = acc;
    }
  }
  double res_phi[NN];
#pragma unroll
  for (int j = 0; j < NN; ++j) res_phi[j] = phL[j];

  bool ok = true;
  if (P.cons & SL_C_ENERGY) {
    double En = 0.0;
#pragma unroll
    for (int i = 0; i < NN; ++i) En += sm.w[i] * phi[i] * phi[i];
    const double Et = En - lam * nete;
    double EL = 0.0;
#pragma unroll
    for (int i = 0; i < NN; ++i) EL += sm.w[i] * phL[i] * phL[i];
    const double gamma = EL - Et;
    // energy row only when the linear fit misses its target beyond rounding level
    const bool apply = fabs(gamma) > ENERGY_SKIP_RTOL * fmax(fabs(Et), EL);
    bool conv = !apply, feasible = true;
    double tol = 0.0;
    if (apply) {
      double pmax = 0.0;
#pragma unroll
      for (int i = 0; i < NN; ++i) pmax = fmax(pmax, fabs(ph[i]));
      tol = P.picard_rtol * fmax(pmax, 1e-300);
    }
    for (int it = 0; apply && it < P.picard_cap; ++it) {
      double a[NN], qv[NN];
#pragma unroll
      for (int i = 0; i < NN; ++i) a[i] = sm.w[i] * res_phi[i];
      if (P.fit == SL_FIT_HARD) {
        double c0 = 0.0, c1 = 0.0, cm = 0.0;
#pragma unroll
        for (int j = 0; j < NN; ++j) {
          if (bnd) { c0 += sm.l0[j] * a[j]; c1 += sm.l1[j] * a[j]; }
          if (mass) cm += sm.w[j] * a[j];
        }
#pragma unroll
        for (int j = 0; j < NN; ++j) {
          double acc = a[j];
          if (bnd) acc -= sm.Cp[0][j] * c0 + sm.Cp[1][j] * c1;
          if (mass) acc -= sm.Cp[2][j] * cm;
          qv[j] = acc;
        }
        double alpha = 0.0, beta = 0.0;
#pragma unroll
        for (int i = 0; i < NN; ++i) { alpha += sm.w[i] * phL[i] * qv[i]; beta += sm.w[i] * qv[i] * qv[i]; }
        double s;
        if (beta <= 0.0) { s = 0.0; feasible = gamma <= 0.0; }
        else {
          const double disc = alpha * alpha - beta * gamma;
          if (disc < 0.0) { s = -alpha / beta; feasible = false; }
          else {
            const double root = sqrt(disc);
            const double den = alpha + (alpha >= 0.0 ? root : -root);
            s = den == 0.0 ? 0.0 : -gamma / den;
            feasible = true;
          }
        }
        double delta = 0.0;
#pragma unroll
        for (int i = 0; i < NN; ++i) {
          const double nv = phL[i] + s * qv[i];
          delta = fmax(delta, fabs(nv - res_phi[i]));
          res_phi[i] = nv;
        }
        if (delta < tol) { conv = feasible; break; }
      } else {
#pragma unroll
        for (int j = 0; j < NN; ++j) {
          double acc = 0.0;
#pragma unroll
          for (int k = 0; k < NN; ++k) acc += sm.S[j * NN + k] * a[k];
          qv[j] = acc;
        }
        double aphi = 0.0, aq = 0.0;
#pragma unroll
        for (int i = 0; i < NN; ++i) { aphi += a[i] * phL[i]; aq += a[i] * qv[i]; }
        const double s = (Et - aphi) / (1.0 + aq);
        double delta = 0.0;
#pragma unroll
        for (int i = 0; i < NN; ++i) {
          const double nv = phL[i] + s * qv[i];
          delta = fmax(delta, fabs(nv - res_phi[i]));
          res_phi[i] = nv;
        }
        if (delta < tol) { conv = true; break; }
      }
    }
    if (!conv) {                          // keep the linear-constraint solution
      ok = false;
#pragma unroll
      for (int i = 0; i < NN; ++i) res_phi[i] = phL[i];
    }
  }
  bool finite = true;
#pragma unroll
  for (int i = 0; i < NN; ++i) {
    out[(size_t)e * NN + i] = res_phi[i];
    finite = finite && finite64(res_phi[i]);
  }
  unsigned bits = (finite ? 0u : SL_ST_NONFINITE) | (ok ? 0u : SL_ST_PICARD_NOCONV);
  if (bits) atomicOr(status, bits);
}

// offsets from an element's centre to its nodes [0, NN) and faces NN, NN + 1: sines and cosines (u = -sin x)
struct Sinx1D {
  double so[NMAX + 2], co[NMAX + 2];
  int ser;
};

template <int NN, bool SINX>
__global__ void __launch_bounds__(BLOCK) k_step1d_f64(StepParams P, Tables1D tb, const __grid_constant__ Sinx1D O,
                                                     const double* __restrict__ in, double* __restrict__ out,
                                                     unsigned* status) {
  __shared__ Smem1D sm;
  __shared__ double s_dx[SINX ? NN * NN : 1];               // xi_i - xi_q
  const int tid = threadIdx.x;
  load_tables<NN>(P, tb, sm);
  if (SINX)
    for (int i = tid; i < NN * NN; i += blockDim.x) s_dx[i] = tb.xi[i / NN] - tb.xi[i % NN];
  __syncthreads();

  const int K = P.K, own = (int)blockDim.x - 2;
  const bool perW = P.bc[0] == SL_BC_PERIODIC, perE = P.bc[1] == SL_BC_PERIODIC;
  const int eraw = (int)blockIdx.x * own + tid - 1;
  const int e = wrap_elem(eraw, K, eraw < 0 ? perW : perE);
  const bool core = tid >= 1 && tid <= own && eraw < K;
  const double h = P.hx;
  const double tn1 = P.t + P.dt;

  // ---------------- phase 1 --------------------------------------------------------------
  double phi[NN], ph[NN];
  double S0 = 0.0, C0 = 0.0, S1 = 0.0, C1 = 0.0;            // sines and cosines at the two faces
  if (SINX && e >= 0) {
    const double xk = P.x0 + e * h, ih = 1.0 / h;
    double Sc, Cc;
    sincos(P.x0 + (e + 0.5) * h, &Sc, &Cc);
    auto at = [&](int i, double& S, double& C) {
      S = fma(Sc, O.co[i], Cc * O.so[i]);
      C = fma(Cc, O.co[i], -Sc * O.so[i]);
    };
    at(NN, S0, C0);
    at(NN + 1, S1, C1);
#pragma unroll
    for (int i = 0; i < NN; ++i) phi[i] = in[(size_t)e * NN + i];
    // (a)-(b) seed at the Gauss nodes and advect: displacements D (reference units), values ps
    double D[NN], ps[NN];
#pragma unroll
    for (int i = 0; i < NN; ++i) {
      double S, C;
      at(i, S, C);
      const double2 r = rk_sinx(P.rk, O.ser, xk + h * sm.xi[i], S, C, phi[i], P.dt);
      D[i] = r.x * ih;
      ps[i] = r.y;
    }
    // (c) remap: phihat_j = sum_i phi*_i h*_i(xi_j), barycentric weights of the advected nodes; each
    // difference serves two products
    double pr[NN];
#pragma unroll
    for (int i = 0; i < NN; ++i) pr[i] = 1.0;
#pragma unroll
    for (int i = 0; i < NN; ++i)
#pragma unroll
      for (int q = i + 1; q < NN; ++q) {
        const double t = s_dx[i * NN + q] + (D[i] - D[q]);
        pr[i] *= t;
        pr[q] *= -t;
      }
#pragma unroll
    for (int i = 0; i < NN; ++i) ps[i] /= pr[i];
#pragma unroll
    for (int j = 0; j < NN; ++j) {
      double d[NN];
#pragma unroll
      for (int m = 0; m < NN; ++m) d[m] = s_dx[j * NN + m] - D[m];
      ph[j] = sum_products<NN>(d, ps);
    }
    // face traces at t^{n+1}, outflow fluxes over the step by the RK quadrature (face value from phi^n at
    // the foot of each distinct stage time; at t^n the trace of phi^n)
    double tr[2], fm[2] = {0.0, 0.0}, fe[2] = {0.0, 0.0}, c[NN];
    const bool back = P.bvalue == SL_BV_BACKTRACK;
    const bool flux = (P.cons & (SL_C_MASS | SL_C_ENERGY)) != 0;
#pragma unroll
    for (int i = 0; i < NN; ++i) c[i] = sm.lam[i] * phi[i];
    auto foot = [&](int side, double cs) {
      const double2 r = rk_sinx(P.rk, O.ser, xk + (side ? h : 0.0), side ? S1 : S0, side ? C1 : C0, 1.0, -cs * P.dt);
      const double z = r.x * ih;
      double d[NN];
#pragma unroll
      for (int m = 0; m < NN; ++m) d[m] = ((side ? 1.0 : 0.0) - sm.xi[m]) + z;
      return sum_products<NN>(d, c) / r.y;
    };
#pragma unroll
    for (int side = 0; side < 2; ++side) {
      const double* L = side ? sm.l1 : sm.l0;
      double acc = 0.0;
      if (back) {
        acc = foot(side, 1.0);
      } else {
#pragma unroll
        for (int j = 0; j < NN; ++j) acc += L[j] * ph[j];
      }
      tr[side] = acc;
      const double un = side ? -S1 : S0;                     // u = -sin x, the same at every stage
      if (flux && un > TIE) {
        for (int s = 0; s < c_ds_n[P.rk]; ++s) {
          double val = 0.0;
          if (s == 0) {
#pragma unroll
            for (int j = 0; j < NN; ++j) val += L[j] * phi[j];
          } else {
            val = foot(side, c_ds_c[P.rk][s]);
          }
          const double bv = c_ds_b[P.rk][s] * un * val;
          fm[side] += bv;
          fe[side] += bv * val;
        }
      }
    }
    sm.tr[0][tid] = tr[0]; sm.tr[1][tid] = tr[1];
    sm.fm[0][tid] = fm[0]; sm.fm[1][tid] = fm[1];
    sm.fe[0][tid] = fe[0]; sm.fe[1][tid] = fe[1];
  }
  if (!SINX && e >= 0) {
    const double xk = P.x0 + e * h;
#pragma unroll
    for (int i = 0; i < NN; ++i) phi[i] = in[(size_t)e * NN + i];
    // (a)-(b) seed at the Gauss nodes and advect
    double xs[NN], ps[NN];
#pragma unroll
    for (int i = 0; i < NN; ++i) {
      double x = xk + h * sm.xi[i], p = phi[i];
      rk_step<NN>(P, sm.xi, sm.lam, x, p, P.t, P.dt);
      xs[i] = (x - xk) / h;
      ps[i] = p;
    }
    // (c) remap: phihat_j = sum_i phi*_i h*_i(xi_j) with barycentric weights of the advected nodes
    double lams[NN];
#pragma unroll
    for (int i = 0; i < NN; ++i) {
      double prod = 1.0;
#pragma unroll
      for (int q = 0; q < NN; ++q)
        if (q != i) prod *= (xs[i] - xs[q]);
      lams[i] = 1.0 / prod;
    }
#pragma unroll
    for (int j = 0; j < NN; ++j) ph[j] = eval_poly<NN>(xs, lams, ps, sm.xi[j]);
    // face traces at t^{n+1}
    double T0, T1;
    if (P.bvalue == SL_BV_BACKTRACK) {
      double f0 = xk, f1 = xk + h, g0 = 1.0, g1 = 1.0;
      rk_step<NN>(P, sm.xi, sm.lam, f0, g0, tn1, -P.dt);
      rk_step<NN>(P, sm.xi, sm.lam, f1, g1, tn1, -P.dt);
      T0 = eval_poly<NN>(sm.xi, sm.lam, phi, (f0 - xk) / h) / g0;
      T1 = eval_poly<NN>(sm.xi, sm.lam, phi, (f1 - xk) / h) / g1;
    } else {
      T0 = 0.0; T1 = 0.0;
#pragma unroll
      for (int j = 0; j < NN; ++j) { T0 += sm.l0[j] * ph[j]; T1 += sm.l1[j] * ph[j]; }
    }
    // outflow fluxes over the step by the RK quadrature, face value from phi^n at the foot
    double fm0 = 0.0, fm1 = 0.0, fe0 = 0.0, fe1 = 0.0;
    if (P.cons & (SL_C_MASS | SL_C_ENERGY)) {
      const int S = c_rk_s[P.rk];
      for (int s = 0; s < S; ++s) {
        const double cs = c_rk_c[P.rk][s], bs = c_rk_b[P.rk][s];
        const double tau = P.t + cs * P.dt;
#pragma unroll
        for (int side = 0; side < 2; ++side) {
          const double xf = xk + (side ? h : 0.0);
          double u, dv;
          nodal1d<NN>(P, sm.xi, sm.lam, xf, tau, u, dv);
          const double un = side ? u : -u;
          if (un > TIE) {
            double fx = xf, g = 1.0;
            if (cs != 0.0) rk_step<NN>(P, sm.xi, sm.lam, fx, g, tau, -cs * P.dt);
            const double val = eval_poly<NN>(sm.xi, sm.lam, phi, (fx - xk) / h) / g;
            if (side) { fm1 += bs * un * val; fe1 += bs * un * val * val; }
            else { fm0 += bs * un * val; fe0 += bs * un * val * val; }
          }
        }
      }
    }
    sm.tr[0][tid] = T0; sm.tr[1][tid] = T1;
    sm.fm[0][tid] = fm0; sm.fm[1][tid] = fm1;
    sm.fe[0][tid] = fe0; sm.fe[1][tid] = fe1;
  }
  __syncthreads();
  if (!core) return;
  const double xk = P.x0 + e * h;
  auto uface = [&](int side, double c) {
    if (SINX) return side ? -S1 : -S0;
    double u, dv;
    nodal1d<NN>(P, sm.xi, sm.lam, xk + (side ? h : 0.0), P.t + c * P.dt, u, dv);
    return u;
  };
  double dm = 0.0;
  if ((P.cons & SL_C_MASS) && P.fit == SL_FIT_HARD) {
#pragma unroll
    for (int i = 0; i < NN; ++i) dm += sm.w[i] * (phi[i] - ph[i]);
  }
  phase2<NN>(P, sm, e, eraw, phi, ph, dm, uface, out, status);
}

// Constant velocity: phihat = R phi^n and the outflow face's values at the feet E_s phi^n, the same matrices
// for every element (ops_shift.cpp), entries from the parameter bank.  About 2 n + 20 FP64 instructions per
// node with every constraint.
template <int NN>
struct Shift1DOps {
  double R[NN * NN], E[3][NN], bs[3];
  double L[2][NN];                          // interface values: of phihat at the faces, or (eq. 4.11) of phi^n at
  double Km[NN];                            // w - R^T w: the mass of phi^n less that of phihat
  int nst, back;                            // the faces' feet when backtracked
};

template <int NN>
__global__ void __launch_bounds__(BLOCK, NN <= 6 ? 4 : NN <= 9 ? 3 : 2) k_step1d_shift(const __grid_constant__ Shift1DOps<NN> O, StepParams P,
                                                       Tables1D tb, const double* __restrict__ in,
                                                       double* __restrict__ out, unsigned* status) {
  __shared__ Smem1D sm;
  const int tid = threadIdx.x;
  load_tables<NN>(P, tb, sm);
  const int K = P.K, own = (int)blockDim.x - 2;
  const bool perW = P.bc[0] == SL_BC_PERIODIC, perE = P.bc[1] == SL_BC_PERIODIC;
  const int eraw = (int)blockIdx.x * own + tid - 1;
  const int e = wrap_elem(eraw, K, eraw < 0 ? perW : perE);
  const bool core = tid >= 1 && tid <= own && eraw < K;
  double phi[NN], ph[NN];
  if (e >= 0) {
#pragma unroll
    for (int i = 0; i < NN; ++i) phi[i] = in[(size_t)e * NN + i];
  }
  __syncthreads();
  const double a = P.vp[0];
  if (e >= 0) {
    double T0 = 0.0, T1 = 0.0;
#pragma unroll
    for (int j = 0; j < NN; ++j) {
      double t = 0.0;
#pragma unroll
      for (int i = 0; i < NN; ++i) t = fma(O.R[j * NN + i], phi[i], t);
      ph[j] = t;
      const double v = O.back ? phi[j] : t;
      T0 = fma(O.L[0][j], v, T0);
      T1 = fma(O.L[1][j], v, T1);
    }
    double fm = 0.0, fe = 0.0;
    if ((P.cons & (SL_C_MASS | SL_C_ENERGY)) && fabs(a) > TIE) {
#pragma unroll
      for (int s = 0; s < 3; ++s)
        if (s < O.nst) {
          double v = 0.0;
#pragma unroll
          for (int i = 0; i < NN; ++i) v = fma(O.E[s][i], phi[i], v);
          const double bv = O.bs[s] * v;
          fm += bv;
          fe = fma(bv, v, fe);
        }
      fm *= fabs(a);
      fe *= fabs(a);
    }
    const int so = a > 0.0;                                  // outflow side
    sm.tr[0][tid] = T0; sm.tr[1][tid] = T1;
    sm.fm[so][tid] = fm; sm.fm[1 - so][tid] = 0.0;
    sm.fe[so][tid] = fe; sm.fe[1 - so][tid] = 0.0;
  }
  __syncthreads();
  if (!core) return;
  double dm = 0.0;
  if (P.cons & SL_C_MASS) {
#pragma unroll
    for (int i = 0; i < NN; ++i) dm = fma(O.Km[i], phi[i], dm);
  }
  phase2<NN>(P, sm, e, eraw, phi, ph, dm, [&](int, double) { return a; }, out, status);
}

// Threads per CTA: the size whose CTAs leave the busiest SM the fewest warps (a short mesh is spread over
// the chip in small CTAs); between equals the larger, whose halo recomputes less
inline int block_for(int K) {
  int best = BLOCK;
  int64_t least = INT64_MAX;
  for (int b = BLOCK; b >= 32; b /= 2) {
    const int64_t ctas = (K + b - 3) / (b - 2), per = (ctas + sm_count() - 1) / sm_count() * (b / 32);
    if (per < least) {
      least = per;
      best = b;
    }
  }
  return best;
}

template <int NN>
void launch_n(const StepParams& p, const Tables1D& tb, const Shift1D* h, const double* xi, const double* in, double* out,
              unsigned* st, cudaStream_t s) {
  const int b = block_for(p.K), grid = (p.K + b - 3) / (b - 2);
  if (h) {
    Shift1DOps<NN> O;
    std::copy(h->R, h->R + NN * NN, O.R);
    for (int k = 0; k < 3; ++k) {
      std::copy(h->E[k], h->E[k] + NN, O.E[k]);
      O.bs[k] = h->bs[k];
    }
    std::copy(h->Km, h->Km + NN, O.Km);
    O.nst = h->nst;
    O.back = p.bvalue == SL_BV_BACKTRACK;
    for (int k = 0; k < 2; ++k) std::copy(O.back ? h->B[k] : h->L[k], (O.back ? h->B[k] : h->L[k]) + NN, O.L[k]);
    k_step1d_shift<NN><<<grid, b, 0, s>>>(O, p, tb, in, out, st);
    return;
  }
  Sinx1D O{};
  if (p.vel_kind == SL_VEL_SINX) {
    for (int i = 0; i < NN + 2; ++i) {
      const double o = p.hx * ((i < NN ? xi[i] : i == NN ? 0.0 : 1.0) - 0.5);
      O.so[i] = std::sin(o);
      O.co[i] = std::cos(o);
    }
    // |u| <= 1: a stage's displacement is at most 3 dt (Kutta's third stage)
    O.ser = 3.0 * p.dt <= 0.0039 ? 0 : 3.0 * p.dt <= 0.05 ? 1 : 2;
    k_step1d_f64<NN, true><<<grid, b, 0, s>>>(p, tb, O, in, out, st);
  } else {
    k_step1d_f64<NN, false><<<grid, b, 0, s>>>(p, tb, O, in, out, st);
  }
}

}  // namespace k1d
}  // namespace sl
