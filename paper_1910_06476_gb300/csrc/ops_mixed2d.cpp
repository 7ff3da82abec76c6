// Host construction (double; the tables are floats) of the shared 2D step operator for a uniform mesh under a
// constant velocity (a, b): every element then sees the same advected geometry (Sec. 5.3), so the
// remap (eq. 5.4, separable: A_y (x) A_x), the face traces (eq. 2dx/2dy_bnd_interpolate), the
// upwind values (eq. 4.12a), the mass target (eq. remap_mass with the RK quadrature of the face
// flux) and the constrained fit (eq. matrix_a) reduce to a few small operators applied per
// element in structured form (psi: the element's n x n values, rows j = y index):
//   psihat = R_y psi R_x^T                        (separable remap, R = A^{-1} of a uniform shift)
//   x inflow residual, row q = sum_m R_y[q][m] (psi_X[m][.] . r_ox - psi[m][.] . R_x^T l_in,x)
//   y inflow residual, col i = sum_p R_x[i][p] (r_oy . psi_Y[.][p]) - l_in,y . psihat[.][i]
//   mass residual            = K_s . psi + K_x . psi_X + K_y . psi_Y  (target minus mass of psihat)
//   phi_L = psihat + C+ r = psihat + C^T s,  s = (C C^T)^+ r over the inflow-face and mass rows
// (the outflow-face rows meet their targets exactly: they are this element's own traces).  C^T s
// is separable: face rows are l0/l1 along one index and a unit vector along the other, the mass
// row is w (x) w, so the correction costs five products per node.
#include <algorithm>
#include <cmath>

#include "sl_internal.h"

namespace sl {
namespace {

using vec = std::vector<double>;

// distinct stage times of the RK orders 1-4 and their summed weights
const int ds_n[5] = {0, 1, 2, 3, 3};
const double ds_c[5][3] = {{}, {0.0}, {0.0, 1.0}, {0.0, 0.5, 1.0}, {0.0, 0.5, 1.0}};
const double ds_b[5][3] = {{}, {1.0}, {0.5, 0.5}, {1.0 / 6, 2.0 / 3, 1.0 / 6}, {1.0 / 6, 2.0 / 3, 1.0 / 6}};

}  // namespace

// A first step pays for this construction, so it is O(n^3): the outflow-flux functionals are sums of a few
// outer products, and (C C^T)^+ comes with the fit operators.
bool build_mixed2d_const(const sl_ctx* c, double a, double b, double dt, unsigned cons, int rk,
                         std::vector<float>& buf, Mixed2DConstParams& P, std::string& err) {
  const int n = c->n, nd = n * n;
  const Basis1D& B = c->b;
  const double hx = (c->mesh.x1 - c->mesh.x0) / c->mesh.kx, hy = (c->mesh.y1 - c->mesh.y0) / c->mesh.ky;
  if (a == 0.0 || b == 0.0) { err = "the 2D shared-operator path needs both velocity components non-zero"; return false; }
  if (cons & SL_C_ENERGY) { err = "energy is applied by the general 2D mixed path"; return false; }
  const vec& w = B.w;
  const double dx = a * dt / hx, dy = b * dt / hy;
  // remap matrices R[l][q] = l_q(xi_l - shift)
  vec Rx(nd), Ry(nd);
  for (int l = 0; l < n; ++l) {
    basis_row(B, B.xi[l], -dx, Rx.data() + l * n);
    basis_row(B, B.xi[l], -dy, Ry.data() + l * n);
  }
  const bool xw = a > 0.0, ys = b > 0.0;       // x-upwind neighbour is W (else E); y-upwind is S (else N)
  const vec &l0 = B.l0, &l1 = B.l1;
  const vec& lin_x = xw ? l0 : l1;
  const vec& lout_x = xw ? l1 : l0;
  const vec& lin_y = ys ? l0 : l1;
  const vec& lout_y = ys ? l1 : l0;
  vec r_ox(n, 0.0), r_oy(n, 0.0);
  for (int q = 0; q < n; ++q)
    for (int i = 0; i < n; ++i) {
      r_ox[q] += Rx[i * n + q] * lout_x[i];
      r_oy[q] += Ry[i * n + q] * lout_y[i];
    }
  // outflow-face flux functionals (mass): Kx[m][l] = |a| hy sum_s b_s sum_q w_q l_m(eta_q - c dy) l_l(xo - c dx)
  vec Kx(nd, 0.0), Ky(nd, 0.0);
  const double xo = xw ? 1.0 : 0.0, yo = ys ? 1.0 : 0.0;
  for (int s = 0; s < ds_n[rk]; ++s) {
    const double cs = ds_c[rk][s], bs = ds_b[rk][s];
    vec ex(n), ey(n), t(n), wx(n, 0.0), wy(n, 0.0);
    basis_row(B, xo, -cs * dx, ex.data());
    basis_row(B, yo, -cs * dy, ey.data());
    for (int q = 0; q < n; ++q) {
      basis_row(B, B.xi[q], -cs * dy, t.data());
      for (int m = 0; m < n; ++m) wy[m] += w[q] * t[m];
      basis_row(B, B.xi[q], -cs * dx, t.data());
      for (int m = 0; m < n; ++m) wx[m] += w[q] * t[m];
    }
    for (int m = 0; m < n; ++m)
      for (int l = 0; l < n; ++l) {
        Kx[m * n + l] += std::fabs(a) * hy * bs * wy[m] * ex[l];
        Ky[m * n + l] += std::fabs(b) * hx * bs * ey[m] * wx[l];
      }
  }
  const double lam = dt / (hx * hy);
  // rows of the hard fit: W (n), E (n), S (n), N (n), mass (1) -- see make_fit_2d
  const FitOps& F = c->fit[cons & 3u][0];
  const int m = F.m;
  const bool bnd = cons & SL_C_BOUNDARY, mass = cons & SL_C_MASS;
  std::vector<int> cols;                         // residuals kept: inflow x rows, inflow y rows, mass
  if (bnd) {
    const int fx = xw ? 0 : 1, fy = ys ? 2 : 3;
    for (int q = 0; q < n; ++q) cols.push_back(fx * n + q);
    for (int q = 0; q < n; ++q) cols.push_back(fy * n + q);
  }
  if (mass) cols.push_back(bnd ? 4 * n : 0);
  const int mc = (int)cols.size();
  // (C C^T)^+ restricted to the kept columns: G[r][k]
  vec G((size_t)m * mc, 0.0);
  for (int r = 0; r < m; ++r)
    for (int k = 0; k < mc; ++k) G[(size_t)r * mc + k] = F.Gp[(size_t)r * m + cols[k]];
  P = Mixed2DConstParams{};
  P.n = n;
  P.kx = c->mesh.kx;
  P.ky = c->mesh.ky;
  P.xw = xw ? 1 : 0;
  P.ys = ys ? 1 : 0;
  P.per_x = c->mesh.bc[0] == SL_BC_PERIODIC ? 1 : 0;
  P.per_y = c->mesh.bc[2] == SL_BC_PERIODIC ? 1 : 0;
  P.ghost = c->mesh.ghost;
  P.bnd = bnd ? 1 : 0;
  P.mass = mass ? 1 : 0;
  P.mc = mc;
  for (int l = 0; l < n; ++l)
    for (int q = 0; q < n; ++q) {
      P.Rx[l * n + q] = (float)Rx[l * n + q];
      P.Ry[l * n + q] = (float)Ry[l * n + q];
    }
  for (int q = 0; q < n / 2; ++q)
    for (int i = 0; i < n; ++i) {
      P.Rxp[q][i] = make_float2(P.Rx[2 * q * n + i], P.Rx[(2 * q + 1) * n + i]);
      P.Ryp[q][i] = make_float2(P.Ry[2 * q * n + i], P.Ry[(2 * q + 1) * n + i]);
    }
  vec wxr(n, 0.0), wyr(n, 0.0);   // R_x^T w, R_y^T w: mass of psihat is wyr^T psi wxr
  for (int p = 0; p < n; ++p) {
    double xi_in = 0.0;
    for (int l = 0; l < n; ++l) {
      xi_in += Rx[l * n + p] * lin_x[l];
      wxr[p] += Rx[l * n + p] * w[l];
      wyr[p] += Ry[l * n + p] * w[l];
    }
    P.xix[p] = (float)xi_in;
    P.rox[p] = (float)r_ox[p];
    P.roy[p] = (float)r_oy[p];
    P.liny[p] = (float)lin_y[p];
    P.l0[p] = (float)l0[p];
    P.l1[p] = (float)l1[p];
    P.w[p] = (float)w[p];
  }
  if (mass) {
    const int rm = bnd ? 4 * n : 0;
    for (int k = 0; k < mc; ++k) P.gm[k] = (float)G[(size_t)rm * mc + k];
  }
  buf.clear();
  auto put = [&](const vec& v) {
    size_t off = buf.size();
    for (double x : v) buf.push_back((float)x);
    return (int)off;
  };
  // tables a thread reads by its own row j are stored [other index][j], so that the n threads of
  // an element read n consecutive floats
  auto transpose = [n](const vec& M) {
    vec T(M.size());
    for (int r = 0; r < n; ++r)
      for (int q = 0; q < n; ++q) T[q * n + r] = M[r * n + q];
    return T;
  };
  // mass residual functionals (reference measure): own psi, x-neighbour psi_X (row j of each) and
  // y-neighbour psi_Y (column j); the mass of psihat is folded into the own functional
  vec Ks(nd), Kxl(nd), Kyl(nd), Kd(nd);
  for (int j = 0; j < n; ++j)
    for (int i = 0; i < n; ++i) {
      const int k = j * n + i;
      Ks[k] = w[j] * w[i] - lam * (Kx[k] + Ky[k]) - wyr[j] * wxr[i];
      Kd[k] = w[j] * w[i] - wyr[j] * wxr[i];
      Kxl[k] = lam * Kx[k];
      Kyl[k] = lam * Ky[k];
    }
  P.o_ks = put(transpose(Ks));
  P.o_kx = put(transpose(Kxl));
  P.o_ky = put(Kyl);                             // column j of psi_Y: entry [m][j]
  P.o_kd = put(transpose(Kd));
  P.o_RxT = put(transpose(Rx));
  P.o_RyT = put(transpose(Ry));
  // face rows of G as Gt[(f * mc + k) * n + j] = G[f n + j][k], f = W, E, S, N
  if (bnd) {
    vec Gt((size_t)4 * mc * n);
    for (int f = 0; f < 4; ++f)
      for (int k = 0; k < mc; ++k)
        for (int j = 0; j < n; ++j) Gt[((size_t)f * mc + k) * n + j] = G[(size_t)(f * n + j) * mc + k];
    P.o_g = put(Gt);
  }
  {
    // orthonormal basis Q of span{l0, l1, w} (twice orthogonalised; a dependent vector leaves a zero column)
    vec Q(3 * n, 0.0), T((size_t)13 * (2 * n + 1), 0.0);
    const vec* span[3] = {&l0, &l1, &w};
    for (int c = 0; c < 3; ++c) {
      vec v = *span[c];
      double v0 = 0.0, v1 = 0.0;
      for (double x : v) v0 += x * x;
      for (int pass = 0; pass < 2; ++pass)
        for (int e = 0; e < c; ++e) {
          double d = 0.0;
          for (int i = 0; i < n; ++i) d += Q[e * n + i] * v[i];
          for (int i = 0; i < n; ++i) v[i] -= d * Q[e * n + i];
        }
      for (double x : v) v1 += x * x;
      if (v1 > 1e-20 * v0)
        for (int i = 0; i < n; ++i) Q[c * n + i] = v[i] / std::sqrt(v1);
    }
    // on the complement of the span opposite faces couple by [a b; b a]
    double a2 = 0.0, b2 = 0.0;
    for (int i = 0; i < n; ++i) {
      a2 += l0[i] * l0[i];
      b2 += l0[i] * l1[i];
    }
    const int fx = xw ? 0 : 1, fy = ys ? 2 : 3, W2 = 2 * n + 1;
    for (int f = 0; f < 4; ++f) {
      const bool in = f == fx || f == fy;
      const double al = bnd ? (in ? a2 : -b2) / (a2 * a2 - b2 * b2) : 0.0;
      P.al[f] = (float)al;
      for (int c = 0; c < 3 && bnd; ++c)
        for (int k = 0; k < mc; ++k) {
          double t = 0.0;
          for (int j = 0; j < n; ++j)
            t += Q[c * n + j] * (G[(size_t)(f * n + j) * mc + k] - (k == (f < 2 ? j : n + j) ? al : 0.0));
          T[(size_t)(3 * f + c) * W2 + k] = t;
        }
    }
    if (mass && bnd)
      for (int k = 0; k < mc; ++k) T[(size_t)12 * W2 + k] = G[(size_t)4 * n * mc + k];
    if (mass && !bnd) T[12] = G[0];
    P.o_t = put(T);
    P.o_q = put(Q);
    for (int i = 0; i < n; ++i) {
      P.louty[i] = (float)lout_y[i];
      P.wh[i] = (float)w[i];
      P.wl[i] = (float)(w[i] - (double)P.wh[i]);
    }
  }
  P.o_l0 = put(l0);
  P.o_l1 = put(l1);
  P.o_w = put(w);
  // mass refinement: each element's outflow flux through its x- and y-outflow faces is a fixed
  // float functional of its own values (lam Kx, lam Ky), evaluated alike by the element and by its
  // downstream neighbour; w (x) w in float-float; the mass column of C+
  // the refinement moves mass along C+ e_m, which keeps the face rows only when C C+ e_m = e_m
  const bool indep = mass && F.last_free;
  P.refine = indep ? 1 : 0;
  if (mass) {
    vec fx(nd), fy(nd);
    float sfx = 0.0f, sfy = 0.0f;
    for (int k = 0; k < nd; ++k) {
      fx[k] = (double)(float)(lam * Kx[k]);
      fy[k] = (double)(float)(lam * Ky[k]);
    }
    // the sums in the order the kernel forms a row's partial sums and then adds the rows
    for (int j = 0; j < n; ++j) {
      float rx = 0.0f, ry = 0.0f;
      for (int i = 0; i < n; ++i) {
        rx += (float)fx[j * n + i];
        ry += (float)fy[j * n + i];
      }
      sfx += rx;
      sfy += ry;
    }
    P.sfx = sfx;
    P.sfy = sfy;
    P.o_fx = put(transpose(fx));
    P.o_fy = put(transpose(fy));
  }
  if (indep) {
    vec wh(nd), wl(nd), cm(nd);
    const int rmass = bnd ? 4 * n : 0;
    for (int j = 0; j < n; ++j)
      for (int i = 0; i < n; ++i) {
        const double v = B.w[i] * B.w[j];
        wh[j * n + i] = (double)(float)v;
        wl[j * n + i] = (double)(float)(v - (double)(float)v);
        cm[j * n + i] = (double)F.Cpinv[(size_t)(j * n + i) * m + rmass];
      }
    P.o_wh = put(transpose(wh));
    P.o_wl = put(transpose(wl));
    P.o_cm = put(cm);                          // [k][j]: node (j, k) of column j at k n + j
  }
  buf.resize((buf.size() + 3) & ~size_t(3), 0.0f);
  return true;
}

}  // namespace sl
