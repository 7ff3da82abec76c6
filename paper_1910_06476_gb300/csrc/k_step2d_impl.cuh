#pragma once
// 2D DSEM-SL step in double precision for any prescribed velocity (Sec. 4, two-dimensional scheme), in
// two kernels with one thread per particle / node and several elements (slots) per CTA.
//
// Phase 1 (k_p1): seed particles at the tensor Gauss nodes, integrate them with explicit RK (eq. 4.4a with
// u and v), solve the collocation system of eq. 5.4,
//     sum_{l,m} phihat_{ml} h_l(xi*_p) h_m(eta*_p) = phi*_p   for every particle p,
// take the face traces of phihat (eq. 2dx_bnd_interpolate, 2dy_bnd_interpolate), the upwind side of every
// face point at t^{n+1} and the mass/energy flux through each face over the step (RK quadrature; outflow:
// this element's phi^n at the backward characteristic foot, inflow through a domain face: the ghost value).
// phihat, traces, upwind sides and fluxes go to workspace in global memory.
// Phase 2 (k_p2): upwind the interface values per face point (eq. 4.12a), form the mass and energy targets
// (eq. remap_mass, remap_energy) from own and neighbour fluxes, apply the constrained least-squares fit
// (eq. matrix_a; 4n boundary rows + mass) and the energy iteration, and store phi^{n+1}.
//
// What bounds these kernels: the FP64 pipe, which runs at 1/64 of the FP32 rate (one FP64 warp instruction
// per 16 cycles and SM).  So the layout and the algorithms save FP64 instructions and spend FP32, integer
// and shared-memory ones freely:
//   - elements are packed side by side into a CTA (thread = slot * n^2 + node), so that idle lanes, which
//     cost as much as busy ones, are only those of the CTA's last warp;
//   - the collocation system is solved by iterative refinement: residuals in FP64 (n^2 + n DFMA per
//     particle), the correction from an inner FP32 iteration on the residual scaled to order one
//     (preconditioner: the exact inverse R_y (x) R_x of the element's mean shift).  The first guess comes
//     from the inner iteration too, so a solve takes two FP64 residuals: each outer pass shrinks the
//     residual by the float accuracy, about 1e-7;
//   - particles are integrated as displacements in reference units; the swirl's sines at displaced points
//     follow from per-element tables by angle addition, with the sine and cosine of the small angle from
//     their Taylor series, exact to 1e-17 over the range each form is chosen for;
//   - stage times that coincide (RK4's two c = 1/2 stages) share one foot, the feet are compacted over the
//     CTA's slots, the flux at stage time t^n is a plain trace;
//   - sums over an element go through shared memory, one thread per row, instead of a butterfly in which
//     every lane adds; maxima compare the high words of the values as integers.
// Measured (one GB300): swirl, 128 x 96 elements of n = 8, every constraint: 4.99 -> 1.29 ms per step against
// one element per CTA with FP64 sines, a FP64 preconditioner and 5-6 FP64 residuals per solve (3030 -> 530
// FP64 instructions per node in phase 1, pipe 84 % busy; phase 2 waits on the few elements whose energy
// iteration runs to its cap); rotation, 66 x 61, n = 8: 0.87 -> 0.30 ms.
#include <cfloat>

#include "k_map2d.cuh"

namespace sl {
namespace k2d {

constexpr int SOLVE_CAP = 60;
constexpr double SOLVE_RTOL = 1e-15;        // target, relative to max |phi*|
constexpr double SOLVE_STALL = 1e-13;       // a residual that stops improving below this is the floor
constexpr int SOLVE_NEXT = 53;              // a correction whose predicted residual is below 2^-53 is the last
constexpr int HI_TINY = 52 << 20;           // high word of DBL_MIN / DBL_EPSILON = 2^-970
constexpr int INNER_CAP = 12;
constexpr float INNER_RTOL = 4e-7f;         // inner (FP32) residual, relative to the outer one

// RK tableaux of orders 1-4 (forward Euler, Heun, Kutta's third order, classical) as compile-time values;
// c2 = 2 c, and the distinct stage times of each order with their summed weights
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
  __device__ static constexpr int c2(int s) {
    return RK == 2 ? 2 * s : RK == 3 ? s : RK == 4 ? (s == 0 ? 0 : s == 3 ? 2 : 1) : 0;
  }
};
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
static __constant__ int c_ds_n[5] = {0, 1, 2, 3, 3};
static __constant__ int c_ds_q[5][3] = {{}, {0}, {0, 4}, {0, 2, 4}, {0, 2, 4}};   // stage time in quarter steps
static __constant__ double c_ds_b[5][3] = {
    {}, {1.0}, {0.5, 0.5}, {1.0 / 6, 2.0 / 3, 1.0 / 6}, {1.0 / 6, 2.0 / 3, 1.0 / 6}};

// ------------------------------------------------------------------ an element of a CTA
struct Geo {
  int64_t g, gb, base;                      // global index, first element of its problem, first value
  int ex, ey, valid;
  int ser;                                  // swirl: 0 short series, 1 long series, 2 direct evaluation
  int nb[4], nq[4];                         // neighbour (within the problem, -1: none), points per face
  double x0, y0, hx, hy, t, dt, ghost, lam; // lam = dt / (hx hy)
  double pihx, pihy, ckx[5], cky[5];        // swirl: 2 cos(pi tau / T) / h at quarter steps of the step
  double kx, ky;                            // rotation: gradients of the reference velocity
};

__device__ __forceinline__ int nb_index(int kx, int ky, const int* bc, int ex, int ey, int face) {
  int jx = ex + (face == 0 ? -1 : face == 1 ? 1 : 0);
  int jy = ey + (face == 2 ? -1 : face == 3 ? 1 : 0);
  if (jx >= 0 && jx < kx && jy >= 0 && jy < ky) return jy * kx + jx;
  if (bc[face] != SL_BC_PERIODIC) return -1;
  jx = (jx + kx) % kx;
  jy = (jy + ky) % ky;
  return jy * kx + jx;
}

// PHASE 2 needs neither positions nor velocities: one thread sets up a slot, and each of its FP64
// instructions holds a scheduler's pipe for 64 cycles
template <int NN, int PHASE>
__device__ __forceinline__ void geo_setup(const StepParams& P, const Map2D& M, int64_t k, int64_t count, Geo& G) {
  G.valid = k < count;
  for (int f = 0; f < 4; ++f) { G.nb[f] = -1; G.nq[f] = 0; }
  G.ser = 0;
  if (!G.valid) return;
  G.g = M.list ? (int64_t)M.list[k] : k;
  G.gb = 0;
  int kx = P.kx, ky = P.ky, bc[4] = {P.bc[0], P.bc[1], P.bc[2], P.bc[3]};
  double X0 = P.x0, Y0 = P.y0;
  G.hx = P.hx; G.hy = P.hy; G.t = P.t; G.dt = P.dt; G.ghost = P.ghost;
  G.lam = P.lam;
  if (M.geo) {
    const ProbGeom& Q = M.geo[M.prob[G.g]];
    kx = Q.kx; ky = Q.ky;
    for (int f = 0; f < 4; ++f) bc[f] = Q.bc[f];
    X0 = Q.x0; Y0 = Q.y0;
    G.hx = Q.hx; G.hy = Q.hy; G.t = Q.t; G.dt = Q.dt; G.ghost = Q.ghost;
    G.gb = Q.gbase;
    G.lam = G.dt / (G.hx * G.hy);
  }
  const int e = (int)(G.g - G.gb);
  G.ex = e % kx;
  G.ey = e / kx;
  G.base = M.off ? M.off[G.g] : G.g * (NN * NN);
  if (PHASE == 1) {
    G.x0 = X0 + G.ex * G.hx;
    G.y0 = Y0 + G.ey * G.hy;
  }
  for (int f = 0; f < 4; ++f) {
    G.nb[f] = nb_index(kx, ky, bc, G.ex, G.ey, f);
    // a face shared with an element of more nodes takes the rule of the finer side, so that both
    // elements integrate the same points (the flux telescopes)
    G.nq[f] = G.nb[f] < 0 ? NN : max(NN, order_of<NN>(M, G.gb + G.nb[f]));
  }
  if (PHASE == 2) return;
  if (P.vel_kind == SL_VEL_ROTATION) {
    G.kx = -P.vp[0] * G.hy / G.hx;
    G.ky = P.vp[0] * G.hx / G.hy;
  } else if (P.vel_kind == SL_VEL_SWIRL) {
    const double pi = 3.14159265358979323846;
    G.pihx = pi * G.hx;
    G.pihy = pi * G.hy;
    // |u|, |v| <= 1, so a stage's displacement times pi is at most 3 pi dt (Kutta's third stage).  Series
    // remainders relative to 1: 5e-18 for the short one up to 0.0039, 3e-20 for the long one up to 0.05
    const double ang = 3.0 * pi * G.dt;
    G.ser = ang <= 0.0039 ? 0 : ang <= 0.05 ? 1 : 2;
  }
}

// ------------------------------------------------------------------ velocity
// A base point is b[4]: its velocity in reference units (constant, rotation); sin pi x, cos pi x, sin pi y,
// cos pi y (swirl); the physical coordinates (swirl, direct evaluation).
__device__ __forceinline__ void swirl_uv(double sx, double cx, double sy, double cy, double ckx, double cky, double& u,
                                         double& v) {
  const double p = sx * sy;                 // sin(2 pi y) = 2 sin cos
  u = (p * ckx) * (sx * cy);
  v = (p * cky) * (sy * cx);
}

// angle addition: sine and cosine of A + x from those of A, |x| small
__device__ __forceinline__ void add_angle(int ser, double x, double S, double C, double& s, double& c) {
  const double x2 = x * x;
  double ps = fma(x2, 1.0 / 120, -1.0 / 6), pc = fma(x2, 1.0 / 24, -0.5);
  if (ser) {
    ps = fma(x2, fma(x2, fma(x2, 1.0 / 362880, -1.0 / 5040), 1.0 / 120), -1.0 / 6);
    pc = fma(x2, fma(x2, fma(x2, 1.0 / 40320, -1.0 / 720), 1.0 / 24), -0.5);
  }
  const double sn = fma(x * x2, ps, x), cm = x2 * pc;        // sin x, cos x - 1
  s = fma(S, cm, fma(C, sn, S));
  c = fma(C, cm, fma(-S, sn, C));
}

// velocity in reference units at the base point displaced by (dx, dy); q: stage time in quarter steps
__device__ __forceinline__ void vel_at(const Geo& G, int kind, double b0, double b1, double b2, double b3, double dx,
                                       double dy, int q, double& u, double& v) {
  if (kind == SL_VEL_ROTATION) {
    u = fma(G.kx, dy, b0);
    v = fma(G.ky, dx, b1);
  } else if (kind == SL_VEL_SWIRL) {
    double sx, cx, sy, cy;
    if (G.ser == 2) {
      sincospi(fma(G.hx, dx, b0), &sx, &cx);
      sincospi(fma(G.hy, dy, b1), &sy, &cy);
    } else {
      add_angle(G.ser, G.pihx * dx, b0, b1, sx, cx);
      add_angle(G.ser, G.pihy * dy, b2, b3, sy, cy);
    }
    swirl_uv(sx, cx, sy, cy, G.ckx[q], G.cky[q], u, v);
  } else {
    u = b0;
    v = b1;
  }
}

// Displacement, in reference units, of one explicit RK step of size h (negative: backward) from the base
// point; stage s is at q0 + c_s qstep quarter steps.  Not inlined: one copy per order serves the particles
// and the feet, and the call costs nothing beside the FP64 work.
template <int RK>
__device__ __noinline__ double2 rk_disp_t(const Geo& G, int kind, double b0, double b1, double b2, double b3, double h,
                                          int q0, int qstep) {
  using T = Tab<RK>;
  double kx[RK], ky[RK];
#pragma unroll
  for (int s = 0; s < RK; ++s) {
    double xs = 0.0, ys = 0.0;
#pragma unroll
    for (int j = 0; j < s; ++j)
      if (T::a(s, j) != 0.0) {
        const double ha = h * T::a(s, j);
        xs = fma(ha, kx[j], xs);
        ys = fma(ha, ky[j], ys);
      }
    const int q = q0 + (T::c2(s) * qstep) / 2;
    if (s == 0 && kind == SL_VEL_SWIRL && G.ser != 2) swirl_uv(b0, b1, b2, b3, G.ckx[q], G.cky[q], kx[0], ky[0]);
    else vel_at(G, kind, b0, b1, b2, b3, xs, ys, q, kx[s], ky[s]);
  }
  double sx = T::b(0) * kx[0], sy = T::b(0) * ky[0];
#pragma unroll
  for (int s = 1; s < RK; ++s) {
    sx = fma(T::b(s), kx[s], sx);
    sy = fma(T::b(s), ky[s], sy);
  }
  return make_double2(h * sx, h * sy);
}

__device__ __forceinline__ double2 rk_disp(const Geo& G, int kind, int rk, const double (&b)[4], double h, int q0,
                                           int qstep) {
  if (kind == SL_VEL_CONST) return make_double2(h * b[0], h * b[1]);
  switch (rk) {
    case 4: return rk_disp_t<4>(G, kind, b[0], b[1], b[2], b[3], h, q0, qstep);
    case 3: return rk_disp_t<3>(G, kind, b[0], b[1], b[2], b[3], h, q0, qstep);
    case 2: return rk_disp_t<2>(G, kind, b[0], b[1], b[2], b[3], h, q0, qstep);
    default: return rk_disp_t<1>(G, kind, b[0], b[1], b[2], b[3], h, q0, qstep);
  }
}

// ------------------------------------------------------------------ bases
// Products prod_{k != l} (z - xi_k) at z = z0 + dz, without the barycentric weights; the differences are
// formed as (z0 - xi_k) + dz, exact for the node z0 itself
template <int NN, typename R>
__device__ __forceinline__ void basis_raw(const R* xi, R z0, R dz, R* out) {
  R d[NN], pre[NN];
#pragma unroll
  for (int k = 0; k < NN; ++k) d[k] = (z0 - xi[k]) + dz;
  pre[0] = R(1);
#pragma unroll
  for (int k = 1; k < NN; ++k) pre[k] = k == 1 ? d[0] : pre[k - 1] * d[k - 1];
  R suf = R(1);
#pragma unroll
  for (int l = NN - 1; l >= 0; --l) {
    out[l] = l == NN - 1 ? pre[l] : l == 0 ? suf : pre[l] * suf;
    suf = l == NN - 1 ? d[l] : suf * d[l];
  }
}

// the Lagrange basis itself
template <int NN, typename R>
__device__ __forceinline__ void basis_at(const R* xi, const R* lam, R z0, R dz, R* out) {
  basis_raw<NN, R>(xi, z0, dz, out);
#pragma unroll
  for (int l = 0; l < NN; ++l) out[l] *= lam[l];
}

// Lagrange basis and its derivative at z (prefix and suffix products carry their derivatives)
template <int NN>
__device__ __forceinline__ void basis_d(const double* xi, const double* lam, double z, double* L, double* D) {
  double d[NN], pre[NN], dpre[NN];
#pragma unroll
  for (int k = 0; k < NN; ++k) d[k] = z - xi[k];
  double acc = 1.0, dacc = 0.0;
#pragma unroll
  for (int k = 0; k < NN; ++k) {
    pre[k] = acc;
    dpre[k] = dacc;
    dacc = dacc * d[k] + acc;
    acc *= d[k];
  }
  double suf = 1.0, dsuf = 0.0;
#pragma unroll
  for (int l = NN - 1; l >= 0; --l) {
    L[l] = lam[l] * pre[l] * suf;
    D[l] = lam[l] * (dpre[l] * suf + pre[l] * dsuf);
    dsuf = dsuf * d[l] + suf;
    suf *= d[l];
  }
}

// sum_m bm[m] sum_l bl[l] v[m][l], rows of v NP values apart
template <int NN, int NP, typename R>
__device__ __forceinline__ R eval2(const R* v, const R (&bl)[NN], const R (&bm)[NN]) {
  R acc = R(0);
#pragma unroll
  for (int m = 0; m < NN; ++m) {
    R row = v[m * NP] * bl[0];
#pragma unroll
    for (int l = 1; l < NN; ++l) row += v[m * NP + l] * bl[l];
    acc += bm[m] * row;
  }
  return acc;
}

// ------------------------------------------------------------------ velocity given at the nodes
// SL_VEL_NODAL along one direction: the elements (index, reference coordinate) that give the field
// at coordinate x, two when x lies on a face (the elements sharing it), else the containing one
// (the boundary element beyond a non-periodic face, wrapped across a periodic one); returns the count
__device__ __forceinline__ int nodal_locate(double x, double lo, double h, int K, bool per, int* ks, double* zs) {
  const double hi = lo + K * h;
  const double s = (x - lo) / h;
  const double r = rint(s);
  if (fabs(x - (lo + r * h)) <= FACE_RTOL * (fabs(lo) + fabs(hi))) {
    const long long ri = (long long)r;
    int cnt = 0;
    for (int side = 0; side < 2; ++side) {
      long long k = side ? ri : ri - 1;
      if (k < 0 || k >= K) {
        if (!per) continue;
        k %= K;
        if (k < 0) k += K;
      }
      ks[cnt] = (int)k;
      zs[cnt] = side ? 0.0 : 1.0;
      ++cnt;
    }
    return cnt;
  }
  const double fk = floor(s);
  long long k = (long long)fk;
  double z = s - fk;
  if (k < 0 || k >= K) {
    if (per) {
      k %= K;
      if (k < 0) k += K;
    } else {
      k = k < 0 ? 0 : K - 1;
      z = s - (double)k;
    }
  }
  ks[0] = (int)k;
  zs[0] = z;
  return 1;
}

// u, v and div u at (x, y, t) from the node velocities of the step (linear in time), averaged over the
// elements that share a face or corner the point lies on
template <int NN>
__device__ __noinline__ void nodal2d(const StepParams& P, const double* xi, const double* lam, double x, double y,
                                     double t, double& u, double& v, double& dv) {
  constexpr int ND = NN * NN;
  const double th = (t - P.t) / P.dt;
  int kxs[2], kys[2];
  double zxs[2], zys[2];
  const int nx = nodal_locate(x, P.x0, P.hx, P.kx, P.bc[0] == SL_BC_PERIODIC, kxs, zxs);
  const int ny = nodal_locate(y, P.y0, P.hy, P.ky, P.bc[2] == SL_BC_PERIODIC, kys, zys);
  const double wt = 1.0 / (nx * ny);
  u = v = dv = 0.0;
  for (int a = 0; a < ny; ++a) {
    double Ly[NN], Dy[NN];
    basis_d<NN>(xi, lam, zys[a], Ly, Dy);
    for (int b = 0; b < nx; ++b) {
      double Lx[NN], Dx[NN];
      basis_d<NN>(xi, lam, zxs[b], Lx, Dx);
      const double* U0 = P.nodal + ((size_t)kys[a] * P.kx + kxs[b]) * ND;
      const double* V0 = U0 + P.nvals;
      const double* U1 = U0 + 2 * P.nvals;
      const double* V1 = U0 + 3 * P.nvals;
      double su = 0.0, sv = 0.0, sux = 0.0, svy = 0.0;
      for (int m = 0; m < NN; ++m) {
        double ru = 0.0, rv = 0.0, rux = 0.0;
#pragma unroll
        for (int l = 0; l < NN; ++l) {
          const double uu = (1.0 - th) * U0[m * NN + l] + th * U1[m * NN + l];
          const double vv = (1.0 - th) * V0[m * NN + l] + th * V1[m * NN + l];
          ru += Lx[l] * uu;
          rv += Lx[l] * vv;
          rux += Dx[l] * uu;
        }
        su += Ly[m] * ru;
        sv += Ly[m] * rv;
        sux += Ly[m] * rux;
        svy += Dy[m] * rv;
      }
      u += wt * su;
      v += wt * sv;
      dv += wt * (sux / P.hx + svy / P.hy);
    }
  }
}

// one explicit RK step of dx/dt = u, dy/dt = v and of the value factor dg/dt = -g div u (eq. 4.8) through
// the nodal velocity, size h (h < 0 runs the characteristic back)
template <int NN>
__device__ __noinline__ void rk_nodal(const StepParams& P, const double* xi, const double* lam, double& x, double& y,
                                      double& g, double t, double h) {
  const int S = c_rk_s[P.rk];
  double kx[4], ky[4], kg[4];
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    if (s < S) {
      double xs = x, ys = y, gs = g;
#pragma unroll
      for (int j = 0; j < s; ++j) {
        xs += h * c_rk_a[P.rk][s][j] * kx[j];
        ys += h * c_rk_a[P.rk][s][j] * ky[j];
        gs += h * c_rk_a[P.rk][s][j] * kg[j];
      }
      double dv;
      nodal2d<NN>(P, xi, lam, xs, ys, t + c_rk_c[P.rk][s] * h, kx[s], ky[s], dv);
      kg[s] = -gs * dv;
    }
  }
  double sx = 0.0, sy = 0.0, sg = 0.0;
#pragma unroll
  for (int s = 0; s < 4; ++s)
    if (s < S) {
      sx += c_rk_b[P.rk][s] * kx[s];
      sy += c_rk_b[P.rk][s] * ky[s];
      sg += c_rk_b[P.rk][s] * kg[s];
    }
  x += h * sx;
  y += h * sy;
  g += h * sg;
}

// ------------------------------------------------------------------ CTA shapes
template <int NN>
struct Shape {
  static constexpr int ND = NN * NN;
  // elements per CTA at most: whole 256 threads where several fit (16 caps the shared memory of tiny n)
  static constexpr int EPC = ND >= 256 ? 1 : (256 / ND < 16 ? 256 / ND : 16);
  static constexpr int NTMAX = (EPC * ND + 31) / 32 * 32;
  static constexpr int NPD = (NN + 1) & ~1;                // row stride of double tables (16-byte rows)
  static constexpr int NPF = (NN + 3) & ~3;                // row stride of float tables
  // resident CTAs asked of the compiler: one CTA's FP32 passes and barriers hide behind another's FP64 work
  static constexpr int MINB = NN <= 10 ? 2 : 1, MINB2 = NN <= 10 ? 4 : 3;
};

__device__ __forceinline__ double hi_value(int h) { return __hiloint2double(h, 0); }
__device__ __forceinline__ int hi_abs(double v) { return __double2hiint(v) & 0x7fffffff; }

template <int NN>
struct __align__(16) Slot1 {
  static constexpr int NPD = Shape<NN>::NPD, NPF = Shape<NN>::NPF;
  double phi[NN * NPD];                     // phi^n rows
  double ph[NN * NPD];                      // phihat rows (times the barycentric weights while solving)
  float r[NN * NPF], tt[NN * NPF], c[NN * NPF];   // inner iteration: residual, row pass, correction
  float Rx[NN * NPF], Ry[NN * NPF];
  double trig[4][NN];                       // swirl: sin, cos of pi x and of pi y at the nodes
  double corner[8];                         // and at x0, x0 + hx, y0, y0 + hy: sines, then cosines
  Geo G;
  int mx[3], fm[3];                         // rotating maxima of the outer and inner residuals
  float md[2];
};

// ------------------------------------------------------------------ phase 1
// dynamic shared memory: slots * Slot1, the face records [slots][4 fq][6] doubles (flux of the stage at t^n:
// mass, energy; weights and values of the later stages), the foot list [slots * 8 fq] ints
template <int NN>
inline size_t smem1(int slots, int fq) {
  return (size_t)slots * (sizeof(Slot1<NN>) + (size_t)4 * fq * 6 * sizeof(double) + (size_t)8 * fq * sizeof(int));
}

template <int NN, bool NOD>
__global__ void __launch_bounds__(Shape<NN>::NTMAX, NOD ? 1 : Shape<NN>::MINB)
    k_p1(StepParams P, Tables1D tb, Map2D M, int64_t count, int slots, int fq, const double* __restrict__ in, Work2D W,
         unsigned* status) {
  constexpr int ND = NN * NN, NPD = Shape<NN>::NPD, NPF = Shape<NN>::NPF;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Slot1<NN>* SL = reinterpret_cast<Slot1<NN>*>(smem_raw);
  double(*fr)[6] = reinterpret_cast<double(*)[6]>(SL + slots);
  int* items = reinterpret_cast<int*>(fr + slots * 4 * fq);
  __shared__ double s_xi[NN], s_lam[NN], s_w[NN], s_l0[NN], s_l1[NN];
  __shared__ float s_xif[NN], s_lamf[NN];
  __shared__ int s_items;
  const int tid = threadIdx.x, nt = blockDim.x;
  const int kind = P.vel_kind;
  if (tid < NN) {
    s_xi[tid] = tb.xi[tid]; s_lam[tid] = tb.lam[tid]; s_w[tid] = tb.w[tid];
    s_l0[tid] = tb.l0[tid]; s_l1[tid] = tb.l1[tid];
    s_xif[tid] = (float)tb.xi[tid];
    s_lamf[tid] = (float)tb.lam[tid];
  }
  if (tid < slots) {
    geo_setup<NN, 1>(P, M, (int64_t)blockIdx.x * slots + tid, count, SL[tid].G);
    for (int k = 0; k < 3; ++k) { SL[tid].mx[k] = 0; SL[tid].fm[k] = 0; }
  }
  if (tid == 0) s_items = 0;
  __syncthreads();
  const int slot = tid / ND < slots ? tid / ND : 0;
  Slot1<NN>& S = SL[slot];
  const bool part = tid < slots * ND && S.G.valid;
  const int nd = tid % ND, i = nd % NN, j = nd / NN;
  double phs = 0.0;
  if (part) {
    phs = in[S.G.base + nd];
    S.phi[j * NPD + i] = phs;
  }
  if (kind == SL_VEL_SWIRL && !NOD) {
    // sines and cosines at the node, corner and stage-time coordinates of every slot
    constexpr int NC = 2 * NN + 9;
    for (int idx = tid; idx < slots * NC; idx += nt) {
      Slot1<NN>& T = SL[idx / NC];
      const int c = idx % NC;
      if (!T.G.valid) continue;
      if (c < 2 * NN) {
        const int k = c < NN ? c : c - NN, d = c < NN ? 0 : 2;
        const double z = c < NN ? T.G.x0 + T.G.hx * s_xi[k] : T.G.y0 + T.G.hy * s_xi[k];
        sincospi(z, &T.trig[d][k], &T.trig[d + 1][k]);
      } else if (c < 2 * NN + 4) {
        const int k = c - 2 * NN;
        const double z = k < 2 ? T.G.x0 + (k == 1 ? T.G.hx : 0.0) : T.G.y0 + (k == 3 ? T.G.hy : 0.0);
        sincospi(z, &T.corner[k], &T.corner[4 + k]);
      } else {
        const int k = c - 2 * NN - 4;
        const double ct = cospi((T.G.t + (0.25 * k) * T.G.dt) / P.vp[0]);
        T.G.ckx[k] = 2.0 * ct / T.G.hx;
        T.G.cky[k] = -2.0 * ct / T.G.hy;
      }
    }
  }
  __syncthreads();

  // (a)-(b) seed and advect the particle of node (i, j): displacement (dx, dy) in reference units
  double dx = 0.0, dy = 0.0;
  if (part) {
    const Geo& G = S.G;
    if (NOD) {
      const double X = G.x0 + G.hx * s_xi[i], Y = G.y0 + G.hy * s_xi[j];
      double x = X, y = Y, g = 1.0;           // g: value factor of eq. 4.8
      rk_nodal<NN>(P, s_xi, s_lam, x, y, g, P.t, P.dt);
      dx = (x - X) / G.hx;
      dy = (y - Y) / G.hy;
      phs *= g;
    } else {
      double b[4];
      if (kind == SL_VEL_SWIRL && G.ser != 2) {
        b[0] = S.trig[0][i]; b[1] = S.trig[1][i]; b[2] = S.trig[2][j]; b[3] = S.trig[3][j];
      } else if (kind == SL_VEL_SWIRL) {
        b[0] = G.x0 + G.hx * s_xi[i]; b[1] = G.y0 + G.hy * s_xi[j]; b[2] = b[3] = 0.0;
      } else if (kind == SL_VEL_ROTATION) {
        b[0] = -P.vp[0] * (G.y0 + G.hy * s_xi[j] - P.vp[2]) / G.hx;
        b[1] = P.vp[0] * (G.x0 + G.hx * s_xi[i] - P.vp[1]) / G.hy;
        b[2] = b[3] = 0.0;
      } else {
        b[0] = P.vp[0] / G.hx; b[1] = P.vp[1] / G.hy; b[2] = b[3] = 0.0;
      }
      const double2 d = rk_disp(G, kind, P.rk, b, G.dt, 0, 4);
      dx = d.x;
      dy = d.y;
    }
    S.r[j * NPF + i] = (float)dx;
    S.tt[j * NPF + i] = (float)dy;
    atomicMax(&S.mx[0], hi_abs(phs));
  }
  __syncthreads();
  // mean displacement (float, fixed order: row sums, then their sum), the preconditioner's rows
  for (int idx = tid; idx < slots * 2 * NN; idx += nt) {
    Slot1<NN>& T = SL[idx / (2 * NN)];
    const int row = idx % NN;
    const float* v = ((idx / NN) & 1 ? T.tt : T.r) + row * NPF;
    float acc = 0.0f;
    if (T.G.valid)
      for (int q = 0; q < NN; ++q) acc += v[q];
    ((idx / NN) & 1 ? T.Ry : T.Rx)[row] = acc;
  }
  __syncthreads();
  for (int idx = tid; idx < 2 * slots; idx += nt) {
    Slot1<NN>& T = SL[idx >> 1];
    const float* v = idx & 1 ? T.Ry : T.Rx;
    float acc = 0.0f;
    for (int q = 0; q < NN; ++q) acc += v[q];
    T.md[idx & 1] = T.G.valid ? acc / ND : 0.0f;
  }
  __syncthreads();
  for (int idx = tid; idx < slots * 2 * NN; idx += nt) {
    Slot1<NN>& T = SL[idx / (2 * NN)];
    const int row = idx % NN, d = (idx / NN) & 1;
    float b[NN];
    basis_at<NN, float>(s_xif, s_lamf, s_xif[row], -T.md[d], b);
    float* R = (d ? T.Ry : T.Rx) + row * NPF;
#pragma unroll
    for (int q = 0; q < NN; ++q) R[q] = b[q];
  }
  // bases at the particle: FP64 without the barycentric weights (they go into the stored phihat), and FP32
  double Lx[NN], Ly[NN];
  float Fx[NN], Fy[NN];
  basis_raw<NN, double>(s_xi, s_xi[i], dx, Lx);
  basis_raw<NN, double>(s_xi, s_xi[j], dy, Ly);
  basis_at<NN, float>(s_xif, s_lamf, s_xif[i], (float)dx, Fx);
  basis_at<NN, float>(s_xif, s_lamf, s_xif[j], (float)dy, Fy);
  const double lam2 = s_lam[i] * s_lam[j];
  // (c) collocation solve
  // residual norms and their tests on the high words (sign cleared), which order like the values; the
  // exponent is hr >> 20
  const int hscale = S.mx[0];
  const int hrtol = hi_abs(SOLVE_RTOL * hi_value(hscale)), hstall = hi_abs(SOLVE_STALL * hi_value(hscale));
  double ph = 0.0, r = phs;
  int hr = hscale, hprev = hscale;
  bool live = part, solved = false;          // equal in every thread of a slot
  if (hscale >= 0x7ff00000) {                // not finite: one pass hands the value on, unconverged
    live = false;
    ph = phs + (hi_value(hscale) - hi_value(hscale));
  }
  __syncthreads();
  for (int it = 0; it < SOLVE_CAP; ++it) {
    if (it > 0) {
      if (live) {
        r = phs - eval2<NN, NPD, double>(S.ph, Lx, Ly);
        atomicMax(&S.mx[it % 3], hi_abs(r));
      }
      __syncthreads();
      hr = S.mx[it % 3];
      if (live) {
        // (data near the bottom of the double range carry no relative accuracy: a residual below
        // DBL_MIN / DBL_EPSILON, about 1e-292, is at the floor of the arithmetic; a residual that has
        // stopped improving at the rounding floor counts as converged)
        if (hr <= hrtol || hr <= HI_TINY || (hr > hprev - (1 << 20) && hr <= hstall)) {
          solved = true;
          live = false;
        } else if (hr >= 0x7ff00000) {       // diverged
          live = false;
        }
      }
    }
    if (nd == 0 && tid < slots * ND) S.mx[(it + 1) % 3] = 0;
    if (!__syncthreads_or(live)) break;
    // correction: H c = r in FP32, r scaled by a power of two to order one
    const int ef = min(max(2046 - (hr >> 20), 1), 2045);
    const double sc = __hiloint2double(ef << 20, 0), isc = __hiloint2double((2046 - ef) << 20, 0);
    const float rf = live ? (float)(r * sc) : 0.0f;
    if (live) S.r[j * NPF + i] = rf;
    __syncthreads();
    bool go = live;
    float c = 0.0f, pin = INFINITY;
    for (int k = 0; k < INNER_CAP; ++k) {
      if (go) {                              // tt[j][l] = sum_q Rx[l][q] r[j][q]
        float acc = 0.0f;
#pragma unroll
        for (int q = 0; q < NN; ++q) acc = fmaf(S.Rx[i * NPF + q], S.r[j * NPF + q], acc);
        S.tt[j * NPF + i] = acc;
      }
      if (nd == 0 && tid < slots * ND) S.fm[(k + 1) % 3] = 0;
      __syncthreads();
      if (go) {                              // c[m][l] += sum_q Ry[m][q] tt[q][l]
        float acc = 0.0f;
#pragma unroll
        for (int q = 0; q < NN; ++q) acc = fmaf(S.Ry[j * NPF + q], S.tt[q * NPF + i], acc);
        c += acc;
        S.c[j * NPF + i] = c;
      }
      __syncthreads();
      if (go) {
        const float rr = rf - eval2<NN, NPF, float>(S.c, Fx, Fy);
        S.r[j * NPF + i] = rr;
        atomicMax(&S.fm[k % 3], __float_as_int(fabsf(rr)));
      }
      __syncthreads();
      const float fm = __int_as_float(S.fm[k % 3]);
      go = go && fm > INNER_RTOL && fm <= 0.5f * pin;
      pin = fm;
      if (!__syncthreads_or(go)) break;
    }
    if (nd == 0 && tid < slots * ND) { S.fm[0] = 0; S.fm[1] = 0; S.fm[2] = 0; }
    if (live) {
      ph = fma((double)c, isc, ph);
      S.ph[j * NPD + i] = ph * lam2;
      // the next residual shrinks at least as this one did: nothing left to see below round-off
      if (it > 0 && 2 * (hr >> 20) - (hprev >> 20) + 4 <= (hscale >> 20) - SOLVE_NEXT) {
        solved = true;
        live = false;
      }
      hprev = hr;
    }
    __syncthreads();
  }
  if (part && !solved && nd == 0) atomicOr(status, SL_ST_SOLVE_NOCONV);
  if (part) {
    W.phihat[S.G.base + nd] = ph;
    S.ph[j * NPD + i] = ph;
  }
  __syncthreads();

  // base point of face point (f, q) of a face rule with nq points: sin, cos of pi x and pi y (swirl), the
  // reference velocity (constant, rotation); x, y physical
  auto face_base = [&](const Slot1<NN>& T, int f, int q, int nq, double (&b)[4], double& x, double& y, double& zq) {
    const Geo& G = T.G;
    zq = nq == NN ? s_xi[q] : tb.rules[(size_t)nq * 3 * NMAX + q];
    x = f == 0 ? G.x0 : f == 1 ? G.x0 + G.hx : G.x0 + G.hx * zq;
    y = f == 2 ? G.y0 : f == 3 ? G.y0 + G.hy : G.y0 + G.hy * zq;
    if (NOD) return;
    if (kind == SL_VEL_SWIRL) {
      if (f < 2) {
        b[0] = T.corner[f]; b[1] = T.corner[4 + f];
        if (nq == NN) { b[2] = T.trig[2][q]; b[3] = T.trig[3][q]; }
        else sincospi(y, &b[2], &b[3]);
      } else {
        b[2] = T.corner[f]; b[3] = T.corner[4 + f];
        if (nq == NN) { b[0] = T.trig[0][q]; b[1] = T.trig[1][q]; }
        else sincospi(x, &b[0], &b[1]);
      }
    } else if (kind == SL_VEL_ROTATION) {
      b[0] = -P.vp[0] * (y - P.vp[2]) / G.hx;
      b[1] = P.vp[0] * (x - P.vp[1]) / G.hy;
    } else {
      b[0] = P.vp[0] / G.hx;
      b[1] = P.vp[1] / G.hy;
    }
  };
  // outward normal velocity (physical) at a face point, q quarter steps into the step
  auto face_un = [&](const Slot1<NN>& T, int f, const double (&b)[4], double x, double y, int qt) {
    const Geo& G = T.G;
    double u, v;
    if (NOD) {
      double dv;
      nodal2d<NN>(P, s_xi, s_lam, x, y, P.t + (0.25 * qt) * P.dt, u, v, dv);
    } else if (kind == SL_VEL_SWIRL) {
      swirl_uv(b[0], b[1], b[2], b[3], G.ckx[qt] * G.hx, G.cky[qt] * G.hy, u, v);
    } else if (kind == SL_VEL_ROTATION) {
      u = -P.vp[0] * (y - P.vp[2]);
      v = P.vp[0] * (x - P.vp[1]);
    } else {
      u = P.vp[0];
      v = P.vp[1];
    }
    return f == 0 ? -u : f == 1 ? u : f == 2 ? -v : v;
  };
  // value factor and foot: phi^n of the element at the backward foot of a face point, from qt quarter steps
  auto foot_value = [&](const Slot1<NN>& T, int f, double (&b)[4], double x, double y, double zq, int qt) {
    const Geo& G = T.G;
    const double zx = f == 0 ? 0.0 : f == 1 ? 1.0 : zq, zy = f == 2 ? 0.0 : f == 3 ? 1.0 : zq;
    double fx, fy, gf = 1.0;
    if (NOD) {
      double X = x, Y = y;
      const double c = 0.25 * qt;
      rk_nodal<NN>(P, s_xi, s_lam, X, Y, gf, P.t + c * P.dt, -c * P.dt);
      fx = (X - x) / G.hx;
      fy = (Y - y) / G.hy;
    } else {
      if (kind == SL_VEL_SWIRL && G.ser == 2) { b[0] = x; b[1] = y; }
      const double2 d = rk_disp(G, kind, P.rk, b, -(0.25 * qt) * G.dt, qt, -qt);
      fx = d.x;
      fy = d.y;
    }
    double bx[NN], by[NN];
    basis_at<NN, double>(s_xi, s_lam, zx, fx, bx);
    basis_at<NN, double>(s_xi, s_lam, zy, fy, by);
    double val = eval2<NN, NPD, double>(T.phi, bx, by);
    if (NOD) val /= gf;
    return val;
  };

  // interface values at the element's own face points: traces of phihat (eq. 2dx/2dy_bnd_interpolate), or
  // phi^n at the backward characteristic foot from t^{n+1} (eq. 4.11); the upwind side at t^{n+1}
  // (0 own, 1 the neighbour's or the ghost, 2 tie)
  for (int idx = tid; idx < slots * 4 * NN; idx += nt) {
    const Slot1<NN>& T = SL[idx / (4 * NN)];
    if (!T.G.valid) continue;
    const int t = idx % (4 * NN), f = t / NN, q = t % NN;
    double b[4], x, y, zq;
    face_base(T, f, q, NN, b, x, y, zq);
    if (P.cons & SL_C_BOUNDARY) {
      const double un = face_un(T, f, b, x, y, 4);
      W.side[T.G.g * M.tstride + t] = un > TIE ? 0 : un < -TIE ? 1 : 2;
    }
    double acc = 0.0;
    if (P.bvalue == SL_BV_BACKTRACK) {
      acc = foot_value(T, f, b, x, y, zq, 4);
    } else {
      const double* L = (f == 1 || f == 3) ? s_l1 : s_l0;
#pragma unroll
      for (int k = 0; k < NN; ++k) acc += (f < 2 ? T.ph[q * NPD + k] : T.ph[k * NPD + q]) * L[k];
    }
    W.traces[T.G.g * M.tstride + t] = acc;
  }
  // fluxes: per face point and distinct stage time the normal velocity; at t^n the outflow value is the
  // trace of phi^n; later outflow points are listed for their feet; inflow through a domain face brings
  // the ghost value
  if (P.cons & (SL_C_MASS | SL_C_ENERGY)) {
    const int nst = c_ds_n[P.rk];
    for (int idx = tid; idx < slots * 4 * fq; idx += nt) {
      const Slot1<NN>& T = SL[idx / (4 * fq)];
      const int t = idx % (4 * fq), f = t / fq, q = t % fq;
      const int nq = T.G.nq[f];
      if (q >= nq) continue;
      double b[4], x, y, zq;
      face_base(T, f, q, nq, b, x, y, zq);
      const double Wq = (f < 2 ? T.G.hy : T.G.hx) * (nq == NN ? s_w[q] : tb.rules[(size_t)nq * 3 * NMAX + 2 * NMAX + q]);
      double fm = 0.0, fe = 0.0;
      for (int s = 0; s < nst; ++s) {
        const int qt = c_ds_q[P.rk][s];
        const double un = face_un(T, f, b, x, y, qt);
        const double bw = c_ds_b[P.rk][s] * Wq * un;
        const bool out = un > TIE;
        if (s == 0) {
          if (out) {
            double val = 0.0;
            if (nq == NN) {
              const double* L = (f == 1 || f == 3) ? s_l1 : s_l0;
#pragma unroll
              for (int k = 0; k < NN; ++k) val += (f < 2 ? T.phi[q * NPD + k] : T.phi[k * NPD + q]) * L[k];
            } else {                           // the face is refined: the trace at another rule's point
              double bt[NN];
              basis_at<NN, double>(s_xi, s_lam, zq, 0.0, bt);
              const double* L = (f == 1 || f == 3) ? s_l1 : s_l0;
#pragma unroll
              for (int m = 0; m < NN; ++m) {
                double row = 0.0;
#pragma unroll
                for (int k = 0; k < NN; ++k) row += (f < 2 ? T.phi[m * NPD + k] : T.phi[k * NPD + m]) * L[k];
                val += bt[m] * row;
              }
            }
            fm = bw * val;
            fe = fm * val;
          }
        } else {
          fr[idx][1 + s] = out ? bw : 0.0;
          if (out) items[atomicAdd(&s_items, 1)] = idx * 4 + s;
        }
        if (un < -TIE && T.G.nb[f] < 0) {
          fm += bw * T.G.ghost;
          fe += bw * T.G.ghost * T.G.ghost;
        }
      }
      fr[idx][0] = fm;
      fr[idx][1] = fe;
    }
    __syncthreads();
    const int ni = s_items;
    for (int it = tid; it < ni; it += nt) {
      const int idx = items[it] >> 2, s = items[it] & 3;
      const Slot1<NN>& T = SL[idx / (4 * fq)];
      const int t = idx % (4 * fq), f = t / fq, q = t % fq;
      double b[4], x, y, zq;
      face_base(T, f, q, T.G.nq[f], b, x, y, zq);
      fr[idx][3 + s] = foot_value(T, f, b, x, y, zq, c_ds_q[P.rk][s]);
    }
    __syncthreads();
    for (int idx = tid; idx < slots * 8; idx += nt) {          // per face, the points in index order
      const Slot1<NN>& T = SL[idx >> 3];
      if (!T.G.valid) continue;
      const int f = (idx >> 1) & 3, k = idx & 1;
      const double(*F)[6] = fr + ((idx >> 3) * 4 + f) * fq;
      double acc = 0.0;
      for (int q = 0; q < T.G.nq[f]; ++q) {
        acc += F[q][k];
        for (int s = 1; s < nst; ++s)
          if (F[q][1 + s] != 0.0) acc += F[q][1 + s] * (k ? F[q][3 + s] * F[q][3 + s] : F[q][3 + s]);
      }
      W.fluxes[T.G.g * 8 + 2 * f + k] = acc;
    }
  }
}

// ------------------------------------------------------------------ phase 2
template <int NN>
struct __align__(16) Slot2 {
  static constexpr int MMAX = 4 * NN + 1;
  double ph[NN * NN], a[NN * NN];           // phihat; energy iteration: w o phi
  double r[MMAX], d[MMAX], ca[MMAX];
  double rs[2][NN], tot[2];                 // sums over the element: rows, totals
  double netm, nete, Et, gamma, s;          // net fluxes; energy target, miss and step along q
  Geo G;
  int rows[4];                              // faces with a non-zero residual
  int on, feasible, mx, ht;                 // energy iteration: running, maximum (high word), tolerance
};

template <int NN>
inline size_t smem2(int slots) {
  return (size_t)slots * (sizeof(Slot2<NN>) + (size_t)3 * NN * NN * sizeof(double));
}

// the neighbour's trace across a p-nonconforming face, out of line: its 2 x 17 products in registers would
// set the register count of the whole kernel
static __device__ __noinline__ double interp_far(const double* rules, int nn, const double* tr, double z) {
  return interp_rule(rules, nn, tr, z);
}

// sum of NN values a stride apart, in two interleaved chains (fixed order)
template <int NN>
__device__ __forceinline__ double chain_sum(const double* v) {
  double a = v[0], b = NN > 1 ? v[1] : 0.0;
#pragma unroll
  for (int k = 2; k < NN; ++k) (k & 1 ? b : a) += v[k];
  return a + b;
}

// Sums of nq quantities buf[slot][quantity][node] over the elements that are on, in a fixed order: one thread
// per row, then one per quantity.  Called by every thread of the CTA; not inlined, it is used several times.
template <int NN>
__device__ __noinline__ void slot_sums(const double* buf, Slot2<NN>* SL, int slots, int nq) {
  constexpr int ND = NN * NN;
  const int tid = threadIdx.x, nt = blockDim.x;
  __syncthreads();
  for (int idx = tid; idx < slots * nq * NN; idx += nt) {
    const int s = idx / (nq * NN), q = (idx / NN) % nq, row = idx % NN;
    if (SL[s].on) SL[s].rs[q][row] = chain_sum<NN>(buf + ((size_t)s * 3 + q) * ND + row * NN);
  }
  __syncthreads();
  for (int idx = tid; idx < slots * nq; idx += nt) {
    const int s = idx / nq, q = idx % nq;
    if (SL[s].on) SL[s].tot[q] = chain_sum<NN>(SL[s].rs[q]);
  }
  __syncthreads();
}

template <int NN>
__global__ void __launch_bounds__(Shape<NN>::NTMAX, Shape<NN>::MINB2)
    k_p2(StepParams P, Tables1D tb, Map2D M, int64_t count, int slots, const double* __restrict__ in, Work2D W,
         double* __restrict__ out, unsigned* status) {
  constexpr int ND = NN * NN;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Slot2<NN>* SL = reinterpret_cast<Slot2<NN>*>(smem_raw);
  double* buf = reinterpret_cast<double*>(SL + slots);         // [slots][3][ND]
  __shared__ double s_xi[NN], s_w[NN], s_l0[NN], s_l1[NN];
  const int tid = threadIdx.x, nt = blockDim.x;
  if (tid < NN) {
    s_xi[tid] = tb.xi[tid]; s_w[tid] = tb.w[tid];
    s_l0[tid] = tb.l0[tid]; s_l1[tid] = tb.l1[tid];
  }
  if (tid < slots) {
    geo_setup<NN, 2>(P, M, (int64_t)blockIdx.x * slots + tid, count, SL[tid].G);
    for (int f = 0; f < 4; ++f) SL[tid].rows[f] = 0;
    SL[tid].on = SL[tid].G.valid;
    SL[tid].mx = 0;
    SL[tid].feasible = 0;
  }
  __syncthreads();
  const int slot = tid / ND < slots ? tid / ND : 0;
  Slot2<NN>& S = SL[slot];
  const bool part = tid < slots * ND && S.G.valid;
  const int nd = tid % ND, i = nd % NN, j = nd / NN;
  double phn = 0.0, ph = 0.0;
  if (part) {
    phn = in[S.G.base + nd];
    ph = W.phihat[S.G.base + nd];
    S.ph[nd] = ph;
  }
  __syncthreads();
  const double w2 = part ? s_w[i] * s_w[j] : 0.0;
  const bool bnd = (P.cons & SL_C_BOUNDARY) != 0;
  const bool mass = (P.cons & SL_C_MASS) != 0, energy = (P.cons & SL_C_ENERGY) != 0;
  const bool hard = P.fit == SL_FIT_HARD;
  const int nb_rows = bnd ? 4 * NN : 0, m = P.m;
  double* mine = buf + (size_t)slot * 3 * ND;
  auto put = [&](int q, double v) { if (part) mine[q * ND + nd] = v; };
  // upwinded interface values (rows W, E, S, N at the tangential nodes); residual d - C phihat
  if (bnd)
    for (int idx = tid; idx < slots * 4 * NN; idx += nt) {
      Slot2<NN>& T = SL[idx / (4 * NN)];
      if (!T.G.valid) continue;
      const int t = idx % (4 * NN), f = t / NN, q = t % NN;
      const int nb = T.G.nb[f];
      const double own = W.traces[T.G.g * M.tstride + t];
      const int side = W.side[T.G.g * M.tstride + t];
      double val = own;
      if (side != 0) {
        double other = T.G.ghost;
        if (nb >= 0) {                         // the neighbour's trace (opposite face) at this face point
          const int nn = order_of<NN>(M, T.G.gb + nb);
          const double* tr = W.traces + (T.G.gb + nb) * M.tstride + (f ^ 1) * nn;
          other = nn == NN ? tr[q] : interp_far(tb.rules, nn, tr, s_xi[q]);
        }
        if (side == 1) val = other;
        else if (nb >= 0) val = 0.5 * (own + other);
      }
      // the row's value at phihat: the own trace when the interface values are traces of phihat, else
      // the trace formed here
      double trh = own;
      if (P.bvalue == SL_BV_BACKTRACK) {
        const double* L = (f == 1 || f == 3) ? s_l1 : s_l0;
        trh = 0.0;
#pragma unroll
        for (int k = 0; k < NN; ++k) trh += (f < 2 ? T.ph[q * NN + k] : T.ph[k * NN + q]) * L[k];
      }
      T.d[t] = val;
      const double rr = val - trh;
      T.r[t] = rr;
      if (!(rr == 0.0)) T.rows[f] = 1;         // (any thread: the same value)
    }
  // mass and energy targets (reference measure): net flux from the faces in order; scalars by one thread per
  // slot (an instruction of every thread costs the pipe eight times as much)
  if (mass || energy) {
    for (int idx = tid; idx < 2 * slots; idx += nt) {
      Slot2<NN>& T = SL[idx >> 1];
      if (!T.G.valid) continue;
      const int k = idx & 1;
      double net = 0.0;
      for (int f = 0; f < 4; ++f) {
        net += W.fluxes[T.G.g * 8 + 2 * f + k];
        if (T.G.nb[f] >= 0) net -= W.fluxes[(T.G.gb + T.G.nb[f]) * 8 + 2 * (f ^ 1) + k];
      }
      (k ? T.nete : T.netm) = net;
    }
    put(0, hard ? w2 * (phn - ph) : w2 * phn); // hard: M^n - M(phihat)
    if (energy) put(1, w2 * phn * phn);
    slot_sums<NN>(buf, SL, slots, energy ? 2 : 1);
    if (tid < slots && SL[tid].G.valid) {
      Slot2<NN>& T = SL[tid];
      if (mass) T.r[nb_rows] = T.d[nb_rows] = T.tot[0] - T.G.lam * T.netm;   // residual (hard), target (soft)
      if (energy) T.Et = T.tot[1] - T.G.lam * T.nete;
    }
  }
  __syncthreads();
  // linear constrained fit; a face whose rows all vanish (outflow: own trace) adds nothing
  double phL = ph;
  if (part) {
    if (hard) {
      if (bnd)
        for (int f = 0; f < 4; ++f) {
          if (!S.rows[f]) continue;
          const double* c = tb.Cpinv + (size_t)f * NN * ND + nd;
#pragma unroll
          for (int k = 0; k < NN; ++k) phL += c[(size_t)k * ND] * S.r[f * NN + k];
        }
      if (mass) phL += tb.Cpinv[(size_t)nb_rows * ND + nd] * S.r[nb_rows];
    } else {
      double acc = 0.0;
      for (int k = 0; k < ND; ++k) acc += tb.S[(size_t)nd * ND + k] * S.ph[k];
      for (int k = 0; k < m; ++k) acc += tb.SCt[(size_t)nd * m + k] * S.d[k];
      phL = acc;
    }
  }
  double cur = phL;
  bool ok = true;
  if (energy) {
    put(0, w2 * phL * phL);
    slot_sums<NN>(buf, SL, slots, 1);
    bool run = false;
    if (tid < slots) {
      Slot2<NN>& T = SL[tid];
      const double EL = T.tot[0];
      T.gamma = EL - T.Et;
      run = T.G.valid && fabs(T.gamma) > ENERGY_SKIP_RTOL * fmax(fabs(T.Et), EL);
      T.on = run;
    }
    if (__syncthreads_or(run)) {
      // Few elements of a CTA iterate, some of them up to the cap, and set the tail of the launch: only their
      // threads work, and the scalars (a square root and a division) are formed by one thread per slot.
      // Equal in every thread of a slot:
      bool on = part && S.on, conv = false;
      const bool apply = on;
      if (on) {
        atomicMax(&S.mx, hi_abs(ph));
        if (ph != 0.0) S.feasible = 1;
      }
      __syncthreads();
      // where phihat vanishes identically the tolerance is zero and no change is below it: the linear fit
      // stays, without the sixty iterations that find that out
      if (tid < slots) {
        Slot2<NN>& T = SL[tid];
        T.ht = hi_abs(P.picard_rtol * fmax(hi_value(T.mx), 1e-300));
        T.on = T.on && T.feasible;
      }
      __syncthreads();
      on = on && S.on;
      for (int it = 0; it < P.picard_cap; ++it) {
        double a = 0.0, q = 0.0;
        if (on) {
          a = w2 * cur;
          S.a[nd] = a;
          if (mass) put(0, w2 * a);
        }
        __syncthreads();
        if (hard) {
          // C a: boundary rows (traces of a), the mass row's row sums
          for (int idx = tid; idx < slots * 5 * NN; idx += nt) {
            Slot2<NN>& T = SL[idx / (5 * NN)];
            if (!T.on) continue;
            const int t = idx % (5 * NN), f = t / NN, qq = t % NN;
            if (f == 4) {
              if (mass) T.rs[0][qq] = chain_sum<NN>(buf + (size_t)(idx / (5 * NN)) * 3 * ND + qq * NN);
            } else if (bnd) {
              const double* L = (f == 1 || f == 3) ? s_l1 : s_l0;
              double acc = 0.0;
#pragma unroll
              for (int k = 0; k < NN; ++k) acc += (f < 2 ? T.a[qq * NN + k] : T.a[k * NN + qq]) * L[k];
              T.ca[t] = acc;
            }
          }
          __syncthreads();
          // q = a - C+ (C a), the rows in order (where the two roots of the energy equation meet, whether the
          // iteration settles below the tolerance hangs on the rounding of this sum)
          if (on) {
            double acc = a;
#pragma unroll 8
            for (int k = 0; k < nb_rows; ++k) acc -= tb.Cpinv[(size_t)k * ND + nd] * S.ca[k];
            if (mass) acc -= tb.Cpinv[(size_t)nb_rows * ND + nd] * chain_sum<NN>(S.rs[0]);
            q = acc;
            put(0, w2 * phL * q);
            put(1, w2 * q * q);
          }
        } else if (on) {
          double acc = 0.0;
          for (int k = 0; k < ND; ++k) acc += tb.S[(size_t)nd * ND + k] * S.a[k];
          q = acc;
          put(0, a * phL);
          put(1, a * q);
        }
        slot_sums<NN>(buf, SL, slots, 2);
        if (tid < slots && SL[tid].on) {
          Slot2<NN>& T = SL[tid];
          const double alpha = T.tot[0], beta = T.tot[1], gamma = T.gamma;
          T.mx = 0;
          T.feasible = 1;
          if (!hard) {
            T.s = (T.Et - alpha) / (1.0 + beta);
          } else if (beta <= 0.0) {
            T.s = 0.0;
            T.feasible = gamma <= 0.0;
          } else {
            const double disc = alpha * alpha - beta * gamma;
            if (disc < 0.0) {
              T.s = -alpha / beta;
              T.feasible = 0;
            } else {
              const double root = sqrt(disc);
              const double den = alpha + (alpha >= 0.0 ? root : -root);
              T.s = den == 0.0 ? 0.0 : -gamma / den;
            }
          }
        }
        __syncthreads();
        if (on) {
          const double nv = phL + S.s * q;
          atomicMax(&S.mx, hi_abs(nv - cur));
          cur = nv;
        }
        __syncthreads();
        if (on && S.mx < S.ht) {               // (high words: below the tolerance for certain)
          conv = S.feasible;
          on = false;
          if (nd == 0) S.on = 0;
        }
        if (!__syncthreads_or(on)) break;
      }
      if (apply && !conv) {                    // keep the linear-constraint solution
        cur = phL;
        ok = false;
      }
    }
  }
  if (part) {
    out[S.G.base + nd] = cur;
    if (hi_abs(cur) >= 0x7ff00000) atomicOr(status, SL_ST_NONFINITE);
    if (!ok && nd == 0) atomicOr(status, SL_ST_PICARD_NOCONV);
  }
}

// Elements per CTA: as many as a CTA packs, but no more than leave two CTAs for every SM (a small mesh is
// spread over the chip: the FP64 pipe of each SM is what there is to share)
inline int slots_for(int epc, int64_t count) {
  const int64_t spread = count / (2 * (int64_t)sm_count());
  return (int)std::max<int64_t>(1, std::min<int64_t>(epc, spread));
}

template <int NN>
void launch_n(int phase, const StepParams& p, const Tables1D& tb, const Map2D& m, int64_t count, const double* in,
              double* out, const Work2D& w, unsigned* st, cudaStream_t s) {
  if (count <= 0) return;
  const int slots = slots_for(Shape<NN>::EPC, count);
  const int nt = (slots * NN * NN + 31) / 32 * 32;
  const unsigned grid = (unsigned)((count + slots - 1) / slots);
  const int fq = m.ord ? NMAX : NN;           // face points of the finest rule a face may take
  if (phase == 1) {
    const size_t sm = smem1<NN>(slots, fq);
    if (p.vel_kind == SL_VEL_NODAL) {
      allow_dynamic_smem((const void*)k_p1<NN, true>, smem1<NN>(Shape<NN>::EPC, NMAX));
      k_p1<NN, true><<<grid, nt, sm, s>>>(p, tb, m, count, slots, fq, in, w, st);
    } else {
      allow_dynamic_smem((const void*)k_p1<NN, false>, smem1<NN>(Shape<NN>::EPC, NMAX));
      k_p1<NN, false><<<grid, nt, sm, s>>>(p, tb, m, count, slots, fq, in, w, st);
    }
  } else {
    allow_dynamic_smem((const void*)k_p2<NN>, smem2<NN>(Shape<NN>::EPC));
    k_p2<NN><<<grid, nt, smem2<NN>(slots), s>>>(p, tb, m, count, slots, in, w, out, st);
  }
}

// ------------------------------------------------------------------ phase 1, one displacement
// Constant velocity on a mesh of one node count: every element sees the same displacement, phase 1 is a set
// of operators built once on the host (ops_shift.cpp) and applied in separable form, n threads per element:
// thread j takes row j of phi^n through R_x, then column j of the result through R_y.  Operator entries are
// the same for every thread, so they come from the parameter bank as DFMA operands; entries that differ by
// thread sit in shared memory.  About 2 n + 10 FP64 instructions per node, where the per-element solve takes
// a few hundred: 512 x 512 elements of n = 9 with the mass row, both phases, 52.2 -> 2.77 ms per step (this
// kernel: 29 FP64 instructions per node, pipe 79 % busy; phase 2: 31, 72 %).
template <int NN>
struct ShiftOps {
  double Rx[NN * NN], Ry[NN * NN];          // remap: R[l][q] = h_q(xi_l - shift)
  double bx[3][NN], by[3][NN];              // basis at the feet of the outflow face, per distinct stage
  double wx[3][NN], wy[3][NN];              // b_s times the face weights through the feet's tangential shift
  double Bx[2][NN * NN], By[2][NN * NN];    // basis at the tangential feet of the later stages
  double bs[3];
  double l0[NN], l1[NN], w[NN];
};

template <int NN>
struct SlotC {
  static constexpr int NR = NN | 1;
  double phi[NN * NR], tt[NN * NR];
  double v[2][NN];                          // W and E traces before R_y
  double X[3][NN], Y[3][NN];                // phi^n at the feet across the face, per stage, along the face
  double p[4][NN];                          // flux pieces: mass x, mass y, energy x, energy y
};

template <int NN>
struct ShapeC {
  static constexpr int EPC = 256 / NN < 32 ? 256 / NN : 32;
  static constexpr int NTMAX = (EPC * NN + 31) / 32 * 32;
};

template <int NN>
__global__ void __launch_bounds__(ShapeC<NN>::NTMAX)
    k_p1c(const __grid_constant__ ShiftOps<NN> O, StepParams P, int64_t count, int slots, int nst,
          const double* __restrict__ in, Work2D W) {
  constexpr int ND = NN * NN, NR = SlotC<NN>::NR;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  SlotC<NN>* SL = reinterpret_cast<SlotC<NN>*>(smem_raw);
  __shared__ double s_Ry[ND], s_wx[3][NN], s_wy[3][NN], s_w[NN];
  const int tid = threadIdx.x, nt = blockDim.x;
  const int64_t k0 = (int64_t)blockIdx.x * slots;
  const int here = (int)(count - k0 < slots ? count - k0 : slots);
  const bool mass = (P.cons & SL_C_MASS) != 0, energy = (P.cons & SL_C_ENERGY) != 0;
  for (int idx = tid; idx < ND; idx += nt) s_Ry[idx] = O.Ry[idx];
  for (int idx = tid; idx < 3 * NN; idx += nt) {
    s_wx[idx / NN][idx % NN] = O.wx[idx / NN][idx % NN];
    s_wy[idx / NN][idx % NN] = O.wy[idx / NN][idx % NN];
  }
  if (tid < NN) s_w[tid] = O.w[tid];
  const double* src = in + k0 * ND;
  for (int idx = tid; idx < here * ND; idx += nt) {
    const int s = idx / ND, nd = idx % ND;
    SL[s].phi[(nd / NN) * NR + nd % NN] = src[idx];
  }
  __syncthreads();
  const int slot = tid / NN < slots ? tid / NN : 0, j = tid % NN;
  SlotC<NN>& S = SL[slot];
  const bool act = tid < here * NN;
  if (act) {
    double row[NN], v0 = 0.0, v1 = 0.0;
#pragma unroll
    for (int i = 0; i < NN; ++i) row[i] = S.phi[j * NR + i];
#pragma unroll
    for (int l = 0; l < NN; ++l) {
      double t = 0.0;
#pragma unroll
      for (int i = 0; i < NN; ++i) t = fma(O.Rx[l * NN + i], row[i], t);
      S.tt[j * NR + l] = t;
      v0 = fma(O.l0[l], t, v0);
      v1 = fma(O.l1[l], t, v1);
    }
    S.v[0][j] = v0;
    S.v[1][j] = v1;
    if (mass || energy) {
      double p = 0.0;
#pragma unroll
      for (int s = 0; s < 3; ++s)
        if (s < nst) {
          double x = 0.0;
#pragma unroll
          for (int l = 0; l < NN; ++l) x = fma(O.bx[s][l], row[l], x);
          S.X[s][j] = x;
          p = fma(s_wy[s][j], x, p);
        }
      S.p[0][j] = p;
    }
  }
  __syncthreads();
  double ph[NN];
  if (act) {
    const int64_t g = k0 + slot;
    double* tr = W.traces + g * (4 * NN);
    double col[NN];
#pragma unroll
    for (int m = 0; m < NN; ++m) col[m] = S.tt[m * NR + j];
    double ts = 0.0, tn = 0.0;
#pragma unroll
    for (int k = 0; k < NN; ++k) {
      double t = 0.0;
#pragma unroll
      for (int m = 0; m < NN; ++m) t = fma(O.Ry[k * NN + m], col[m], t);
      ph[k] = t;
      ts = fma(O.l0[k], t, ts);
      tn = fma(O.l1[k], t, tn);
    }
    double tw = 0.0, te = 0.0;
#pragma unroll
    for (int q = 0; q < NN; ++q) {
      tw = fma(s_Ry[j * NN + q], S.v[0][q], tw);
      te = fma(s_Ry[j * NN + q], S.v[1][q], te);
    }
    tr[j] = tw;
    tr[NN + j] = te;
    tr[2 * NN + j] = ts;
    tr[3 * NN + j] = tn;
    if (P.cons & SL_C_BOUNDARY) {
      uint8_t* sd = W.side + g * (4 * NN);
      const double a = P.vp[0], b = P.vp[1];
      sd[j] = -a > TIE ? 0 : -a < -TIE ? 1 : 2;
      sd[NN + j] = a > TIE ? 0 : a < -TIE ? 1 : 2;
      sd[2 * NN + j] = -b > TIE ? 0 : -b < -TIE ? 1 : 2;
      sd[3 * NN + j] = b > TIE ? 0 : b < -TIE ? 1 : 2;
    }
    if (mass || energy) {
#pragma unroll
      for (int m = 0; m < NN; ++m) col[m] = S.phi[m * NR + j];
      double p = 0.0;
#pragma unroll
      for (int s = 0; s < 3; ++s)
        if (s < nst) {
          double y = 0.0;
#pragma unroll
          for (int m = 0; m < NN; ++m) y = fma(O.by[s][m], col[m], y);
          S.Y[s][j] = y;
          p = fma(s_wx[s][j], y, p);
        }
      S.p[1][j] = p;
    }
  }
  __syncthreads();
  if (act) {
#pragma unroll
    for (int k = 0; k < NN; ++k) S.phi[k * NR + j] = ph[k];
    if (energy) {                             // the energy flux needs the values at the face points
      double ex = 0.0, ey = 0.0;
      for (int s = 0; s < nst; ++s) {
        double vx = S.X[s][j], vy = S.Y[s][j];
        if (s > 0) {
          vx = 0.0;
          vy = 0.0;
#pragma unroll
          for (int m = 0; m < NN; ++m) {
            vx = fma(O.By[s - 1][j * NN + m], S.X[s][m], vx);
            vy = fma(O.Bx[s - 1][j * NN + m], S.Y[s][m], vy);
          }
        }
        ex = fma(O.bs[s] * vx, vx, ex);
        ey = fma(O.bs[s] * vy, vy, ey);
      }
      S.p[2][j] = s_w[j] * ex;
      S.p[3][j] = s_w[j] * ey;
    }
  }
  __syncthreads();
  for (int idx = tid; idx < here * ND; idx += nt) {
    const int s = idx / ND, nd = idx % ND;
    W.phihat[k0 * ND + idx] = SL[s].phi[(nd / NN) * NR + nd % NN];
  }
  if (mass || energy) {
    for (int idx = tid; idx < here * 4; idx += nt) {
      const int s = idx >> 2, c = idx & 3, d = c & 1;          // quantity c: direction d, mass or energy
      const int64_t g = k0 + s;
      double acc = 0.0;
      if (c < 2 || energy)
        for (int q = 0; q < NN; ++q) acc += SL[s].p[c][q];
      const double un = d ? P.vp[1] : P.vp[0], Wn = (d ? P.hx : P.hy) * fabs(un);
      const int fo = 2 * d + (un > 0.0), fi = fo ^ 1;          // outflow and inflow face
      const int ex = (int)(g % P.kx), ey = (int)(g / P.kx), at = d ? ey : ex, last = (d ? P.ky : P.kx) - 1;
      const int bc = d ? (fi == 2 ? P.bc[2] : P.bc[3]) : (fi == 0 ? P.bc[0] : P.bc[1]);
      const bool wall = bc != SL_BC_PERIODIC && at == (fi & 1 ? last : 0);
      const bool flows = fabs(un) > TIE;
      double* F = W.fluxes + g * 8 + (c >> 1);
      F[2 * fo] = flows ? Wn * acc : 0.0;
      F[2 * fi] = flows && wall ? -Wn * (c >> 1 ? P.ghost * P.ghost : P.ghost) : 0.0;
    }
  }
}

template <int NN>
void launch_shift(const Shift2D& h, const StepParams& p, int64_t count, const double* in, const Work2D& w,
                  cudaStream_t s) {
  ShiftOps<NN> O;
  auto cp = [](double* dst, const double* src, int n) { std::copy(src, src + n, dst); };
  cp(O.Rx, h.Rx, NN * NN);
  cp(O.Ry, h.Ry, NN * NN);
  for (int k = 0; k < 3; ++k) {
    cp(O.bx[k], h.bx[k], NN);
    cp(O.by[k], h.by[k], NN);
    cp(O.wx[k], h.wx[k], NN);
    cp(O.wy[k], h.wy[k], NN);
    O.bs[k] = h.bs[k];
  }
  for (int k = 0; k < 2; ++k) {
    cp(O.Bx[k], h.Bx[k], NN * NN);
    cp(O.By[k], h.By[k], NN * NN);
  }
  cp(O.l0, h.l0, NN);
  cp(O.l1, h.l1, NN);
  cp(O.w, h.w, NN);
  const int64_t spread = count / (2 * (int64_t)sm_count());
  const int slots = (int)std::max<int64_t>(1, std::min<int64_t>(ShapeC<NN>::EPC, spread));
  const int nt = (slots * NN + 31) / 32 * 32;
  allow_dynamic_smem((const void*)k_p1c<NN>, ShapeC<NN>::EPC * sizeof(SlotC<NN>));
  k_p1c<NN><<<(unsigned)((count + slots - 1) / slots), nt, slots * sizeof(SlotC<NN>), s>>>(O, p, count, slots, h.nst, in,
                                                                                         w);
}

}  // namespace k2d
}  // namespace sl
