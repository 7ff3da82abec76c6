// Host operators of the constant-velocity FP64 steps: every element of a uniform mesh sees the same particle
// displacement, so the remap (eq. 4.9, 5.4) and the flux feet (eq. remap_mass, remap_energy) are fixed
// matrices.  Differences are formed as (z0 - xi_k) + dz in reference coordinates, so the displacement is
// not rounded to the element's physical position.  Double arithmetic, O(n^3) operations (microseconds).
#include <algorithm>
#include <cmath>

#include "sl_internal.h"

namespace sl {

namespace {

// distinct stage times of the RK orders 1-4 and their summed weights (RK4's two c = 1/2 stages coincide)
const int ds_n[5] = {0, 1, 2, 3, 3};
const double ds_c[5][3] = {{}, {0.0}, {0.0, 1.0}, {0.0, 0.5, 1.0}, {0.0, 0.5, 1.0}};
const double ds_b[5][3] = {{}, {1.0}, {0.5, 0.5}, {1.0 / 6, 2.0 / 3, 1.0 / 6}, {1.0 / 6, 2.0 / 3, 1.0 / 6}};

}  // namespace

void build_shift1d(const Basis1D& B, double a, double dt, double h, int rk, Shift1D& S) {
  const double sx = dt * a / h;                         // displacement in reference units
  S.nst = ds_n[rk];
  for (int j = 0; j < B.n; ++j) basis_row(B, B.xi[j], -sx, S.R + j * B.n);
  for (int s = 0; s < 3; ++s) {
    S.bs[s] = s < S.nst ? ds_b[rk][s] : 0.0;
    basis_row(B, a > 0.0 ? 1.0 : 0.0, s < S.nst ? -ds_c[rk][s] * sx : 0.0, S.E[s]);
  }
  for (int i = 0; i < B.n; ++i) {
    double m = B.w[i];
    for (int j = 0; j < B.n; ++j) m -= B.w[j] * S.R[j * B.n + i];
    S.Km[i] = m;
  }
  for (int f = 0; f < 2; ++f) {
    const std::vector<double>& l = f ? B.l1 : B.l0;
    std::copy(l.begin(), l.end(), S.L[f]);
    basis_row(B, f, -sx, S.B[f]);
  }
  S.a = a;
  S.dt = dt;
  S.rk = rk;
  S.valid = true;
}

void build_shift2d(const Basis1D& B, double a, double b, double dt, double hx, double hy, int rk, Shift2D& S) {
  const int n = B.n;
  const double sx = dt * a / hx, sy = dt * b / hy;      // displacement in reference units
  S.nst = ds_n[rk];
  for (int l = 0; l < n; ++l) {
    basis_row(B, B.xi[l], -sx, S.Rx + l * n);
    basis_row(B, B.xi[l], -sy, S.Ry + l * n);
  }
  for (int s = 0; s < 3; ++s) {
    S.bs[s] = s < S.nst ? ds_b[rk][s] : 0.0;
    const double c = s < S.nst ? ds_c[rk][s] : 0.0;
    basis_row(B, a > 0.0 ? 1.0 : 0.0, -c * sx, S.bx[s]);
    basis_row(B, b > 0.0 ? 1.0 : 0.0, -c * sy, S.by[s]);
    double Bx[NMAX * NMAX], By[NMAX * NMAX];
    for (int q = 0; q < n; ++q) {
      basis_row(B, B.xi[q], -c * sx, Bx + q * n);
      basis_row(B, B.xi[q], -c * sy, By + q * n);
    }
    for (int m = 0; m < n; ++m) {
      double x = 0.0, y = 0.0;
      for (int q = 0; q < n; ++q) {
        x += B.w[q] * Bx[q * n + m];
        y += B.w[q] * By[q * n + m];
      }
      S.wx[s][m] = S.bs[s] * x;
      S.wy[s][m] = S.bs[s] * y;
    }
    if (s > 0) {
      std::copy(Bx, Bx + n * n, S.Bx[s - 1]);
      std::copy(By, By + n * n, S.By[s - 1]);
    }
  }
  for (int l = 0; l < n; ++l) {
    S.l0[l] = B.l0[l];
    S.l1[l] = B.l1[l];
    S.w[l] = B.w[l];
  }
  S.a = a;
  S.b = b;
  S.dt = dt;
  S.rk = rk;
  S.valid = true;
}

}  // namespace sl
