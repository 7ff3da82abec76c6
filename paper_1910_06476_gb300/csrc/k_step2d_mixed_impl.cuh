#pragma once
// 2D DSEM-SL step in mixed precision for any prescribed velocity (Sec. 4, two-dimensional scheme):
// particles seeded at the Gauss nodes and advected (eq. 4.4a), the collocation system eq. 5.4 solved for
// the remapped values, face traces (eq. 2dx/2dy_bnd_interpolate), upwinded interface values (eq. 4.12a),
// mass and energy targets (eq. 4.14, remap_mass, remap_energy) and the constrained fit (eq. matrix_a).
//
// State: double-float (hi + lo floats).  The bulk arithmetic is float on increments psi = phi - L
// relative to an element reference L, written back exactly, so float rounding scales with the
// variation inside the element:
//   - without the energy row L = r0 + gx (xi - 1/2) + gy (eta - 1/2) from the corner values, with the
//     energy row the constant r0.  L at a point is an exact float-float value (two-sum of r0 and the
//     once-rounded linear part), psi = (hi - L_hi) + (lo - L_lo) is therefore accurate relative to psi,
//     and the write-back L + psi is a float-float sum.  No FP64 instruction is used: this GPU's FP64
//     pipe runs at about 1/64 of the FP32 rate.
//   - Particles keep phi (divergence-free velocity), so the collocation data of psihat = phihat - L at a
//     particle displaced by d are psi - grad L . d.
//   - Mass: the element mass M^n = sum w (x) w (hi + lo) and each face's outflow flux G_f (outflow points
//     of the element, RK/Gauss quadrature at the backward characteristic feet, plus the ghost inflow on a
//     domain face) are float-float values.  An element's net outflow is its own G_f minus its
//     neighbours' G through the shared faces: every face flux enters two elements with opposite signs
//     as the same number, so global mass telescopes.  The fit itself works on float increments; one
//     refinement step then measures the element mass of the result in float-float and moves the
//     remaining miss along the pseudo-inverse column of the mass row into the lo word, which brings the
//     element mass to its target to about 1e-16 relative.
//   - Energy: target and mismatch from float increments (the energy row is decided at a 1e-9 relative
//     miss, its float resolution).
//
// Work layout: a group of G warps advances one element at a time (G = 1 up to n = 8, 5 at n = 17), two
// particles per thread (p0 = t, p1 = t + 32 G) with paired float operations across them where they
// share operands, several groups per CTA, each synchronising on its own named barrier (one warp:
// __syncwarp).  Reductions are butterflies (every lane gets the same bits) and, across the warps of a
// group, a fixed-order sum.  The kernels are persistent: group k of the grid walks the launch's elements
// k, k + groups, ...; per-group counters (solve and energy iterations, elements that stopped at the
// float floor or did not converge) are added to the context's counters once per group.
// Swirl velocity without transcendentals in the RK stages: sin and cos of pi x at the element's node
// and corner coordinates are taken once per element; at a displaced point they follow from the angle
// addition formulas, with the sine and cosine of the small angle pi h d from their Taylor series (used
// while h <= 1/4, so that |pi h d| <= pi / 4 where ten terms are exact to 1e-9; coarser meshes evaluate
// sinpi and cospi directly).  cos(pi t / T) is taken once per element at the stage-time fractions 0,
// 1/4, 1/2, 3/4, 1 of the step, which cover the RK schemes and their backward feet.
// Bound by instruction issue (60 % / 73 % of the issue slots in the two phases; FMA pipe 51 % / 32 %, HBM 4 %).
// Measured (one GB300), 512 x 512 elements of n = 8, swirl, every constraint: phase 1 757 -> 651 us (607 -> 473 M
// warp instructions), phase 2 597 -> 357 us (353 -> 225 M).  What that took: no FP64 instruction (element corners
// in float-float, per-problem parameters from the host), the upwind side of each face point formed once in
// phase 1 from the tabulated sines, the pseudo-inverse read as pairs with a thread's two nodes side by side and
// skipped for faces whose residual vanishes, one evaluation for all tabulated sines, maxima by one integer
// reduction, reductions that share a barrier merged, the preconditioner's passes as dot products of rows in
// 16-byte vectors at a conflict-free stride, the traces and the face fluxes in one pass over the face points.
#include <type_traits>

#include "k_map2d.cuh"
#include "ffloat.cuh"

namespace sl {
namespace k2m {

// distinct stage times of the face-flux quadrature and their summed weights (RK4's two c = 1/2
// stages see the same face velocity and the same foot)
static __constant__ int c_ds_n[5] = {0, 1, 2, 3, 3};
static __constant__ float c_ds_c[5][3] = {{}, {0.0f}, {0.0f, 1.0f}, {0.0f, 0.5f, 1.0f}, {0.0f, 0.5f, 1.0f}};
static __constant__ float c_ds_b[5][3] = {
    {}, {1.0f}, {0.5f, 0.5f}, {1.0f / 6, 2.0f / 3, 1.0f / 6}, {1.0f / 6, 1.0f / 3 + 1.0f / 3, 1.0f / 6}};

constexpr int SOLVE_CAP = 40;
constexpr float SOLVE_RTOL = 3e-7f;          // target, relative to max |psi*|
constexpr float SOLVE_STALL = 4e-6f;         // a residual that stops improving below this is the float floor
constexpr float SOLVE_FLOOR = 1e-4f;         // best residual accepted (SL_ST_SOLVE_FLOOR) above the floor

// asynchronous 4-byte global-to-shared copies (the next element's inputs are staged while the current
// one is computed); a thread waits for its own copies, a group barrier then publishes them
__device__ __forceinline__ void cp_async4(float* smem, const float* gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait1() { asm volatile("cp.async.wait_group 1;\n" ::: "memory"); }

// element reference L at reference coordinates given as (a, b) = (xi - 1/2, eta - 1/2): the linear
// part is rounded once, L = r0 + t exactly as a float-float value.  Every use runs this same
// instruction sequence, so both kernels agree on L bit for bit.
__device__ __forceinline__ ff lref(float r0, float gx, float gy, float a, float b) {
  const float t = fmaf(gx, a, __fmul_rn(gy, b));
  return two_sum(r0, t);
}
// the same at two points at once
__device__ __forceinline__ ff2 lref2(float r0, float gx, float gy, float2 a, float2 b) {
  return two_sum2(dup(r0), __ffma2_rn(dup(gx), a, __fmul2_rn(dup(gy), b)));
}

// ------------------------------------------------------------------ groups of warps
template <int NN>
struct Shape {
  static constexpr int ND = NN * NN;
  static constexpr int G = (ND + 63) / 64;                 // warps per element
  static constexpr int GT = 32 * G;                        // threads per element
  static constexpr int EPC = G == 1 ? 8 : G == 2 ? 4 : G <= 4 ? 2 : 1;   // element groups per CTA
  static constexpr int NT = GT * EPC;
  static constexpr int NP = (NN + 3) & ~3;                 // row stride of psihat and psi^n (16 bytes)
  // row stride of the preconditioner tables: the rows that lanes read side by side, as 16-byte vectors, start
  // in different banks
  static constexpr int RP = NP + (NP % 8 == 0 ? 4 : 0);
  // resident CTAs asked of the compiler.  Phase 1 at three (80 registers) fits up to n = 5 (558 / 504 us at n = 4,
  // 4.2 M nodes) and spills above (179 / 191 us at n = 8); four CTAs of five warps at n = 17 (474 / 420 us); below
  // two, n >= 13 ran 6-8 warps per SM.  Phase 2 fits four since the far-neighbour interpolation is out of line
  static constexpr int MINB = NN <= 5 ? 3 : G <= 4 ? 2 : 4;
  static constexpr int MINB2 = NN <= 16 ? 4 : 3;
};

template <int G>
struct Grp {
  int t, lane, w, slot;
  float* red;                                              // 8 G floats: two buffers of four values per warp
  int rb;
  __device__ __forceinline__ void sync() const {
    if (G == 1) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(1 + slot), "r"(32 * G) : "memory");
  }
  // Cross-warp sums alternate between two scratch buffers: a buffer is rewritten two reductions
  // later, after every warp has passed the barrier of the reduction in between.
  __device__ __forceinline__ float sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (G == 1) return v;
    float* r = red + rb * 4 * G;
    rb ^= 1;
    if (lane == 0) r[w] = v;
    sync();
    float s = 0.0f;
#pragma unroll
    for (int k = 0; k < G; ++k) s += r[k];
    return s;
  }
  __device__ __forceinline__ float2 sum2(float a, float b) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float2 v = __fadd2_rn(make_float2(a, b), make_float2(__shfl_xor_sync(0xffffffffu, a, o),
                                                                 __shfl_xor_sync(0xffffffffu, b, o)));
      a = v.x;
      b = v.y;
    }
    if (G == 1) return make_float2(a, b);
    float* r = red + rb * 4 * G;
    rb ^= 1;
    if (lane == 0) { r[w] = a; r[G + w] = b; }
    sync();
    float sa = 0.0f, sb = 0.0f;
#pragma unroll
    for (int k = 0; k < G; ++k) { sa += r[k]; sb += r[G + k]; }
    return make_float2(sa, sb);
  }
  // maximum of non-negative values: their bits order like the values (one warp instruction); NaN, whose bits
  // are above infinity's, wins
  __device__ __forceinline__ float max(float v) {
    v = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(v)));
    if (G == 1) return v;
    float* r = red + rb * 4 * G;
    rb ^= 1;
    if (lane == 0) r[w] = v;
    sync();
    unsigned s = 0u;
#pragma unroll
    for (int k = 0; k < G; ++k) s = ::max(s, __float_as_uint(r[k]));
    return __uint_as_float(s);
  }
  // two or three sums and a maximum of non-negative values in one pass (one barrier between the warps)
  __device__ __forceinline__ void sum3max(float& a, float& b, float& c, float& m, bool three) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float2 v = __fadd2_rn(make_float2(a, b), make_float2(__shfl_xor_sync(0xffffffffu, a, o),
                                                                 __shfl_xor_sync(0xffffffffu, b, o)));
      a = v.x;
      b = v.y;
      if (three) c += __shfl_xor_sync(0xffffffffu, c, o);
    }
    m = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(m)));
    if (G == 1) return;
    float* r = red + rb * 4 * G;
    rb ^= 1;
    if (lane == 0) { r[w] = a; r[G + w] = b; r[2 * G + w] = c; r[3 * G + w] = m; }
    sync();
    a = b = c = 0.0f;
    unsigned mx = 0u;
#pragma unroll
    for (int k = 0; k < G; ++k) {
      a += r[k];
      b += r[G + k];
      if (three) c += r[2 * G + k];
      mx = ::max(mx, __float_as_uint(r[3 * G + k]));
    }
    m = __uint_as_float(mx);
  }
  // float-float sum: the high parts by two-sums, their errors and the low parts in one float (symmetric at
  // every level, so every lane gets the same bits), renormalised once
  __device__ __forceinline__ ff ffsum(ff v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float uh = __shfl_xor_sync(0xffffffffu, v.hi, o), ul = __shfl_xor_sync(0xffffffffu, v.lo, o);
      const ff s = two_sum(v.hi, uh);
      v.hi = s.hi;
      v.lo = __fadd_rn(__fadd_rn(v.lo, ul), s.lo);
    }
    v = fast_two_sum(v.hi, v.lo);
    if (G == 1) return v;
    float* r = red + rb * 4 * G;
    rb ^= 1;
    if (lane == 0) { r[w] = v.hi; r[G + w] = v.lo; }
    sync();
    return ffjoin(r);
  }
  // the same, with two plain sums in the same pass
  __device__ __forceinline__ ff ffsum_sum2(ff v, float& a, float& b) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float uh = __shfl_xor_sync(0xffffffffu, v.hi, o), ul = __shfl_xor_sync(0xffffffffu, v.lo, o);
      const ff s = two_sum(v.hi, uh);
      v.hi = s.hi;
      v.lo = __fadd_rn(__fadd_rn(v.lo, ul), s.lo);
      const float2 u = __fadd2_rn(make_float2(a, b), make_float2(__shfl_xor_sync(0xffffffffu, a, o),
                                                                 __shfl_xor_sync(0xffffffffu, b, o)));
      a = u.x;
      b = u.y;
    }
    v = fast_two_sum(v.hi, v.lo);
    if (G == 1) return v;
    float* r = red + rb * 4 * G;
    rb ^= 1;
    if (lane == 0) { r[w] = v.hi; r[G + w] = v.lo; r[2 * G + w] = a; r[3 * G + w] = b; }
    sync();
    a = b = 0.0f;
#pragma unroll
    for (int k = 0; k < G; ++k) {
      a += r[2 * G + k];
      b += r[3 * G + k];
    }
    return ffjoin(r);
  }
  __device__ __forceinline__ ff ffjoin(const float* r) const {
    ff s = {r[0], r[G]};
#pragma unroll
    for (int k = 1; k < G; ++k) s = ff_add(s, ff{r[k], r[G + k]});
    return s;
  }
};

// ------------------------------------------------------------------ velocity
// sine and cosine of a small angle by their Taylor series: five terms each (exact to 1e-9 for
// |x| <= pi / 4), or three when |x| <= 0.02 (the remainders x^7 / 7! and x^6 / 6! are then below
// 1e-13)
__device__ __forceinline__ void small_sincos(float x, bool shortser, float& s, float& c) {
  const float x2 = x * x;
  if (shortser) {
    s = fmaf(x * x2, fmaf(x2, 1.0f / 120.0f, -1.0f / 6.0f), x);
    c = fmaf(x2, fmaf(x2, 1.0f / 24.0f, -0.5f), 1.0f);
    return;
  }
  float ps = fmaf(x2, 1.0f / 362880.0f, -1.0f / 5040.0f);
  ps = fmaf(x2, ps, 1.0f / 120.0f);
  ps = fmaf(x2, ps, -1.0f / 6.0f);
  s = fmaf(x * x2, ps, x);
  float pc = fmaf(x2, -1.0f / 3628800.0f, 1.0f / 40320.0f);
  pc = fmaf(x2, pc, -1.0f / 720.0f);
  pc = fmaf(x2, pc, 1.0f / 24.0f);
  pc = fmaf(x2, pc, -0.5f);
  c = fmaf(x2, pc, 1.0f);
}

// paired float operations
__device__ __forceinline__ float2 bc2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }

__device__ __forceinline__ void small_sincos2(float2 x, bool shortser, float2& s, float2& c) {
  const float2 x2 = mul2(x, x);
  if (shortser) {
    s = fma2(mul2(x, x2), fma2(x2, bc2(1.0f / 120.0f), bc2(-1.0f / 6.0f)), x);
    c = fma2(x2, fma2(x2, bc2(1.0f / 24.0f), bc2(-0.5f)), bc2(1.0f));
    return;
  }
  float2 ps = fma2(x2, bc2(1.0f / 362880.0f), bc2(-1.0f / 5040.0f));
  ps = fma2(x2, ps, bc2(1.0f / 120.0f));
  ps = fma2(x2, ps, bc2(-1.0f / 6.0f));
  s = fma2(mul2(x, x2), ps, x);
  float2 pc = fma2(x2, bc2(-1.0f / 3628800.0f), bc2(1.0f / 40320.0f));
  pc = fma2(x2, pc, bc2(-1.0f / 720.0f));
  pc = fma2(x2, pc, bc2(1.0f / 24.0f));
  pc = fma2(x2, pc, bc2(-0.5f));
  c = fma2(x2, pc, bc2(1.0f));
}

// The velocity of one element divided by its size (the time derivative of the reference
// coordinates).  A point is given by its base reference coordinates (bx, by), the sine and cosine of
// pi times the base's physical coordinates (swirl), and a displacement (dx, dy) in reference units;
// ct = cos(pi tau / T) at the stage time.
struct VelElem {
  int kind;
  bool direct;                   // evaluate sinpi/cospi at the point itself (coarse meshes)
  bool shortser;                 // pi h <= 0.02: three-term series for the small angle
  float x0, y0, hx, hy, ihx, ihy, pihx, pihy;
  float a, b, om, cx, cy;
};

__device__ __forceinline__ void vel_at(const VelElem& V, float bx, float by, float Sx, float Cx, float Sy, float Cy,
                                       float dx, float dy, float ct, float& u, float& v) {
  switch (V.kind) {
    case SL_VEL_ROTATION: {
      const float x = fmaf(V.hx, bx + dx, V.x0), y = fmaf(V.hy, by + dy, V.y0);
      u = -V.om * (y - V.cy) * V.ihx;
      v = V.om * (x - V.cx) * V.ihy;
      break;
    }
    case SL_VEL_SWIRL: {
      float sx, cx, sy, cy;
      if (V.direct) {
        sincospif(fmaf(V.hx, bx + dx, V.x0), &sx, &cx);
        sincospif(fmaf(V.hy, by + dy, V.y0), &sy, &cy);
      } else {
        float st, ctt;
        small_sincos(V.pihx * dx, V.shortser, st, ctt);
        sx = fmaf(Sx, ctt, Cx * st);
        cx = fmaf(Cx, ctt, -Sx * st);
        small_sincos(V.pihy * dy, V.shortser, st, ctt);
        sy = fmaf(Sy, ctt, Cy * st);
        cy = fmaf(Cy, ctt, -Sy * st);
      }
      // sin(2 pi y) = 2 sin(pi y) cos(pi y)
      u = sx * sx * (2.0f * sy * cy) * ct * V.ihx;
      v = -sy * sy * (2.0f * sx * cx) * ct * V.ihy;
      break;
    }
    default:
      u = V.a * V.ihx;
      v = V.b * V.ihy;
  }
}

// Butcher tableaux of the explicit RK schemes of orders 1-4 (forward Euler, Heun, Kutta's third
// order, classical), as compile-time functions so that the coefficients become immediates
template <int RK>
struct Tab {
  static constexpr int S = RK;
  __device__ static constexpr float a(int s, int j) {
    return RK == 2 ? (s == 1 && j == 0 ? 1.0f : 0.0f)
         : RK == 3 ? (s == 1 && j == 0 ? 0.5f : s == 2 && j == 0 ? -1.0f : s == 2 && j == 1 ? 2.0f : 0.0f)
         : RK == 4 ? ((s == 1 && j == 0) || (s == 2 && j == 1) ? 0.5f : s == 3 && j == 2 ? 1.0f : 0.0f)
                   : 0.0f;
  }
  __device__ static constexpr float b(int s) {
    return RK == 1 ? 1.0f
         : RK == 2 ? 0.5f
         : RK == 3 ? (s == 1 ? 2.0f / 3.0f : 1.0f / 6.0f)
                   : (s == 0 || s == 3 ? 1.0f / 6.0f : 1.0f / 3.0f);
  }
  __device__ static constexpr float c(int s) {
    return RK == 2 ? (s == 1 ? 1.0f : 0.0f)
         : RK == 3 ? (s == 1 ? 0.5f : s == 2 ? 1.0f : 0.0f)
         : RK == 4 ? (s == 1 || s == 2 ? 0.5f : s == 3 ? 1.0f : 0.0f)
                   : 0.0f;
  }
};

// One RK step of the displacement (dx, dy) of a point over a time step h (negative: backward), the
// stage time of stage s being the step fraction f0 + c_s fstep (one of 0, 1/4, 1/2, 3/4, 1, whose
// cos(pi tau / T) are ctab[0..4]).  The displacement is integrated by itself (not the position), so
// that its float rounding is relative to the displacement.
// velocity of the swirl at a displaced point from the tabulated sines (angle addition)
__device__ __forceinline__ void vel_swirl_tab(const VelElem& V, float Sx, float Cx, float Sy, float Cy, float dx,
                                              float dy, float ct, float& u, float& v) {
  float st, ctt;
  small_sincos(V.pihx * dx, V.shortser, st, ctt);
  const float sx = fmaf(Sx, ctt, Cx * st), cx = fmaf(Cx, ctt, -Sx * st);
  small_sincos(V.pihy * dy, V.shortser, st, ctt);
  const float sy = fmaf(Sy, ctt, Cy * st), cy = fmaf(Cy, ctt, -Sy * st);
  const float p = sx * sy;
  u = (p * (sx * cy)) * (2.0f * ct * V.ihx);
  v = (p * (sy * cx)) * (-2.0f * ct * V.ihy);
}

// The displacement starts at zero, so the first stage is the base point itself.
// TAB: the velocity is the swirl from the tabulated sines (chosen once per element)
template <int RK, bool TAB>
__device__ __forceinline__ void rk_disp_t(const VelElem& V, float bx, float by, float Sx, float Cx, float Sy, float Cy,
                                          float& dx, float& dy, float h, float f0, float fstep, const float* ctab) {
  using T = Tab<RK>;
  float kx[T::S], ky[T::S];
#pragma unroll
  for (int s = 0; s < T::S; ++s) {
    float xs = 0.0f, ys = 0.0f;
#pragma unroll
    for (int j = 0; j < s; ++j)
      if (T::a(s, j) != 0.0f) {
        xs = fmaf(h * T::a(s, j), kx[j], xs);
        ys = fmaf(h * T::a(s, j), ky[j], ys);
      }
    const int ci = __float2int_rn(4.0f * fmaf(T::c(s), fstep, f0));
    if (TAB && s == 0) {
      const float p = Sx * Sy;
      kx[0] = (p * (Sx * Cy)) * (2.0f * ctab[ci] * V.ihx);
      ky[0] = (p * (Sy * Cx)) * (-2.0f * ctab[ci] * V.ihy);
    } else if (TAB) vel_swirl_tab(V, Sx, Cx, Sy, Cy, xs, ys, ctab[ci], kx[s], ky[s]);
    else vel_at(V, bx, by, Sx, Cx, Sy, Cy, xs, ys, ctab[ci], kx[s], ky[s]);
  }
  float sx = 0.0f, sy = 0.0f;
#pragma unroll
  for (int s = 0; s < T::S; ++s) {
    sx = fmaf(T::b(s), kx[s], sx);
    sy = fmaf(T::b(s), ky[s], sy);
  }
  dx = h * sx;
  dy = h * sy;
}

__device__ __forceinline__ void rk_disp(const VelElem& V, int rk, float bx, float by, float Sx, float Cx, float Sy,
                                        float Cy, float& dx, float& dy, float h, float f0, float fstep,
                                        const float* ctab) {
  if (rk == 4 && V.kind == SL_VEL_SWIRL && !V.direct) {
    rk_disp_t<4, true>(V, bx, by, Sx, Cx, Sy, Cy, dx, dy, h, f0, fstep, ctab);
    return;
  }
  switch (rk) {
    case 4: rk_disp_t<4, false>(V, bx, by, Sx, Cx, Sy, Cy, dx, dy, h, f0, fstep, ctab); break;
    case 3: rk_disp_t<3, false>(V, bx, by, Sx, Cx, Sy, Cy, dx, dy, h, f0, fstep, ctab); break;
    case 2: rk_disp_t<2, false>(V, bx, by, Sx, Cx, Sy, Cy, dx, dy, h, f0, fstep, ctab); break;
    default: rk_disp_t<1, false>(V, bx, by, Sx, Cx, Sy, Cy, dx, dy, h, f0, fstep, ctab);
  }
}

// vel_at at two points at once (paired float operations; the direct evaluation per component)
__device__ __forceinline__ void vel_at2(const VelElem& V, float2 bx, float2 by, float2 Sx, float2 Cx, float2 Sy,
                                        float2 Cy, float2 dx, float2 dy, float2 ct, float2& u, float2& v) {
  switch (V.kind) {
    case SL_VEL_ROTATION: {
      const float2 x = fma2(bc2(V.hx), add2(bx, dx), bc2(V.x0)), y = fma2(bc2(V.hy), add2(by, dy), bc2(V.y0));
      u = mul2(bc2(-V.om * V.ihx), add2(y, bc2(-V.cy)));
      v = mul2(bc2(V.om * V.ihy), add2(x, bc2(-V.cx)));
      break;
    }
    case SL_VEL_SWIRL: {
      float2 sx, cx, sy, cy;
      if (V.direct) {
        sincospif(fmaf(V.hx, bx.x + dx.x, V.x0), &sx.x, &cx.x);
        sincospif(fmaf(V.hx, bx.y + dx.y, V.x0), &sx.y, &cx.y);
        sincospif(fmaf(V.hy, by.x + dy.x, V.y0), &sy.x, &cy.x);
        sincospif(fmaf(V.hy, by.y + dy.y, V.y0), &sy.y, &cy.y);
      } else {
        float2 st, ctt;
        small_sincos2(mul2(bc2(V.pihx), dx), V.shortser, st, ctt);
        sx = fma2(Sx, ctt, mul2(Cx, st));
        cx = fma2(Cx, ctt, mul2(neg2(Sx), st));
        small_sincos2(mul2(bc2(V.pihy), dy), V.shortser, st, ctt);
        sy = fma2(Sy, ctt, mul2(Cy, st));
        cy = fma2(Cy, ctt, mul2(neg2(Sy), st));
      }
      u = mul2(mul2(sx, sx), mul2(mul2(sy, cy), mul2(ct, bc2(2.0f * V.ihx))));
      v = mul2(mul2(sy, sy), mul2(mul2(sx, cx), mul2(ct, bc2(-2.0f * V.ihy))));
      break;
    }
    default:
      u = bc2(V.a * V.ihx);
      v = bc2(V.b * V.ihy);
  }
}

// rk_disp for two points at once (paired float operations); cts(c) gives cos(pi tau / T) at the step fraction c of
// each point's own step h
template <int RK, bool TAB, class CT>
__device__ __forceinline__ void rk_disp2_t(const VelElem& V, float2 bx, float2 by, float2 Sx, float2 Cx, float2 Sy,
                                           float2 Cy, float2& dx, float2& dy, float2 h, CT cts) {
  using T = Tab<RK>;
  float2 kx[T::S], ky[T::S];
#pragma unroll
  for (int s = 0; s < T::S; ++s) {
    float2 xs = bc2(0.0f), ys = bc2(0.0f);
#pragma unroll
    for (int j = 0; j < s; ++j)
      if (T::a(s, j) != 0.0f) {
        const float2 hj = mul2(h, bc2(T::a(s, j)));
        xs = fma2(hj, kx[j], xs);
        ys = fma2(hj, ky[j], ys);
      }
    const float2 ct = cts(T::c(s));
    if (TAB && s == 0) {
      const float2 p = mul2(Sx, Sy);
      kx[0] = mul2(mul2(p, mul2(ct, bc2(2.0f * V.ihx))), mul2(Sx, Cy));
      ky[0] = mul2(mul2(p, mul2(ct, bc2(-2.0f * V.ihy))), mul2(Sy, Cx));
    } else if (TAB) {
      float2 st, ctt;
      small_sincos2(mul2(bc2(V.pihx), xs), V.shortser, st, ctt);
      const float2 sx = fma2(Sx, ctt, mul2(Cx, st)), cx = fma2(Cx, ctt, mul2(neg2(Sx), st));
      small_sincos2(mul2(bc2(V.pihy), ys), V.shortser, st, ctt);
      const float2 sy = fma2(Sy, ctt, mul2(Cy, st)), cy = fma2(Cy, ctt, mul2(neg2(Sy), st));
      const float2 p = mul2(sx, sy);
      kx[s] = mul2(mul2(p, mul2(ct, bc2(2.0f * V.ihx))), mul2(sx, cy));
      ky[s] = mul2(mul2(p, mul2(ct, bc2(-2.0f * V.ihy))), mul2(sy, cx));
    } else {
      vel_at2(V, bx, by, Sx, Cx, Sy, Cy, xs, ys, ct, kx[s], ky[s]);
    }
  }
  float2 sx = bc2(0.0f), sy = bc2(0.0f);
#pragma unroll
  for (int s = 0; s < T::S; ++s) {
    sx = fma2(bc2(T::b(s)), kx[s], sx);
    sy = fma2(bc2(T::b(s)), ky[s], sy);
  }
  dx = mul2(h, sx);
  dy = mul2(h, sy);
}

template <class CT>
__device__ __forceinline__ void rk_disp2(const VelElem& V, int rk, float2 bx, float2 by, float2 Sx, float2 Cx,
                                         float2 Sy, float2 Cy, float2& dx, float2& dy, float2 h, CT cts) {
  if (rk == 4 && V.kind == SL_VEL_SWIRL && !V.direct) {
    rk_disp2_t<4, true>(V, bx, by, Sx, Cx, Sy, Cy, dx, dy, h, cts);
    return;
  }
  switch (rk) {
    case 4: rk_disp2_t<4, false>(V, bx, by, Sx, Cx, Sy, Cy, dx, dy, h, cts); break;
    case 3: rk_disp2_t<3, false>(V, bx, by, Sx, Cx, Sy, Cy, dx, dy, h, cts); break;
    case 2: rk_disp2_t<2, false>(V, bx, by, Sx, Cx, Sy, Cy, dx, dy, h, cts); break;
    default: rk_disp2_t<1, false>(V, bx, by, Sx, Cx, Sy, Cy, dx, dy, h, cts);
  }
}

// velocity at a base point itself (no displacement): the tabulated sines and cosines directly
__device__ __forceinline__ void vel_base(const VelElem& V, float bx, float by, float Sx, float Cx, float Sy, float Cy,
                                         float ct, float& u, float& v) {
  if (V.kind == SL_VEL_SWIRL && !V.direct) {
    u = Sx * Sx * (2.0f * Sy * Cy) * ct * V.ihx;
    v = -Sy * Sy * (2.0f * Sx * Cx) * ct * V.ihy;
  } else {
    vel_at(V, bx, by, Sx, Cx, Sy, Cy, 0.0f, 0.0f, ct, u, v);
  }
}

// Lagrange basis at z = z0 + dz with the differences formed as (z0 - xi_k) + dz: when z0 is a
// node, its own difference is dz exactly
template <int NN>
__device__ __forceinline__ void basis_at(const float* xi, const float* lam, float z0, float dz, float* out) {
  float d[NN], pre[NN];
#pragma unroll
  for (int k = 0; k < NN; ++k) d[k] = (z0 - xi[k]) + dz;
  float acc = 1.0f;
#pragma unroll
  for (int k = 0; k < NN; ++k) { pre[k] = acc; acc *= d[k]; }
  float suf = 1.0f;
#pragma unroll
  for (int l = NN - 1; l >= 0; --l) {
    out[l] = lam[l] * pre[l] * suf;
    suf *= d[l];
  }
}

// the same at two points at once, in paired float operations (same rounding per point)
template <int NN>
__device__ __forceinline__ void basis_at2(const float* xi, const float* lam, float z0a, float z0b, float dza, float dzb,
                                          float2* out) {
  float2 d[NN], pre[NN];
  const float2 dz = make_float2(dza, dzb);
#pragma unroll
  for (int k = 0; k < NN; ++k) d[k] = __fadd2_rn(make_float2(z0a - xi[k], z0b - xi[k]), dz);
  float2 acc = make_float2(1.0f, 1.0f);
#pragma unroll
  for (int k = 0; k < NN; ++k) { pre[k] = acc; acc = __fmul2_rn(acc, d[k]); }
  float2 suf = make_float2(1.0f, 1.0f);
#pragma unroll
  for (int l = NN - 1; l >= 0; --l) {
    out[l] = __fmul2_rn(__fmul2_rn(make_float2(lam[l], lam[l]), pre[l]), suf);
    suf = __fmul2_rn(suf, d[l]);
  }
}

// sum_l row[l] b[l] for two vectors b at once (paired FMAs), row 16-byte aligned with NN values
template <int NN>
__device__ __forceinline__ float2 row_dot2(const float* row, const float2 (&b)[NN]) {
  const float4* rowp = reinterpret_cast<const float4*>(row);
  float2 r = make_float2(0.0f, 0.0f);
#pragma unroll
  for (int q = 0; q < (NN + 3) / 4; ++q) {
    const float4 v = rowp[q];
    if (4 * q + 0 < NN) r = __ffma2_rn(make_float2(v.x, v.x), b[(4 * q + 0) % NN], r);
    if (4 * q + 1 < NN) r = __ffma2_rn(make_float2(v.y, v.y), b[(4 * q + 1) % NN], r);
    if (4 * q + 2 < NN) r = __ffma2_rn(make_float2(v.z, v.z), b[(4 * q + 2) % NN], r);
    if (4 * q + 3 < NN) r = __ffma2_rn(make_float2(v.w, v.w), b[(4 * q + 3) % NN], r);
  }
  return r;
}

// sum_l row[l] b[l] for one vector b: even and odd columns in the two lanes of paired FMAs
template <int NN>
__device__ __forceinline__ float row_dot(const float* row, const float (&b)[NN]) {
  const float4* rowp = reinterpret_cast<const float4*>(row);
  float2 r2 = make_float2(0.0f, 0.0f);
#pragma unroll
  for (int q = 0; q < NN / 4; ++q) {
    const float4 v = rowp[q];
    r2 = __ffma2_rn(make_float2(v.x, v.y), make_float2(b[4 * q], b[4 * q + 1]), r2);
    r2 = __ffma2_rn(make_float2(v.z, v.w), make_float2(b[4 * q + 2], b[4 * q + 3]), r2);
  }
  float r = r2.x + r2.y;
  if (NN % 4 != 0) {
    const float4 v = rowp[NN / 4];
    constexpr int l0 = NN & ~3;
    r = fmaf(v.x, b[l0], r);
    if (NN % 4 > 1) r = fmaf(v.y, b[(l0 + 1) % NN], r);
    if (NN % 4 > 2) r = fmaf(v.z, b[(l0 + 2) % NN], r);
  }
  return r;
}

__device__ __forceinline__ int nb_index(const StepParams& P, int ex, int ey, int face) {
  int jx = ex + (face == 0 ? -1 : face == 1 ? 1 : 0);
  int jy = ey + (face == 2 ? -1 : face == 3 ? 1 : 0);
  if (jx >= 0 && jx < P.kx && jy >= 0 && jy < P.ky) return jy * P.kx + jx;
  // the face's boundary condition by selection (a dynamic index would put P in local memory)
  const int bc = face == 0 ? P.bc[0] : face == 1 ? P.bc[1] : face == 2 ? P.bc[2] : P.bc[3];
  if (bc != SL_BC_PERIODIC) return -1;
  jx = (jx + P.kx) % P.kx;
  jy = (jy + P.ky) % P.ky;
  return jy * P.kx + jx;
}

// sum_q a[q] b[q] of two shared rows (16-byte aligned, padded to 4): even and odd terms in the lanes of paired FMAs
template <int NN>
__device__ __forceinline__ float dot_rows(const float* a, const float* b) {
  const float4* ap = reinterpret_cast<const float4*>(a);
  const float4* bp = reinterpret_cast<const float4*>(b);
  float2 r2 = make_float2(0.0f, 0.0f);
#pragma unroll
  for (int q = 0; q < NN / 4; ++q) {
    const float4 u = ap[q], v = bp[q];
    r2 = __ffma2_rn(make_float2(u.x, u.y), make_float2(v.x, v.y), r2);
    r2 = __ffma2_rn(make_float2(u.z, u.w), make_float2(v.z, v.w), r2);
  }
  float r = r2.x + r2.y;
  if (NN % 4 != 0) {
    const float4 u = ap[NN / 4], v = bp[NN / 4];
    r = fmaf(u.x, v.x, r);
    if (NN % 4 > 1) r = fmaf(u.y, v.y, r);
    if (NN % 4 > 2) r = fmaf(u.z, v.z, r);
  }
  return r;
}

// the element of launch-list index k, and its problem's record (GEO: batches, else null)
template <int NN, bool GEO>
__device__ __forceinline__ Elem elem_at(const StepParams& P, const Map2D& M, int64_t k, const ProbGeom*& geo) {
  Elem E;
  E.g = M.list ? (int64_t)M.list[k] : k;
  E.gb = 0;
  geo = nullptr;
  int kx = P.kx;
  if (GEO) {
    geo = M.geo + M.prob[E.g];
    kx = geo->kx;
    E.gb = geo->gbase;
  }
  E.e = (int)(E.g - E.gb);
  E.ey = E.e / kx;
  E.ex = E.e - E.ey * kx;
  E.base = M.off ? M.off[E.g] : E.g * (NN * NN);
  return E;
}

// a problem's mesh and float parameters into P and X (batches)
__device__ __forceinline__ void use_problem(const ProbGeom* G, StepParams& P, Mixed2DExtra& X) {
  P.kx = G->kx;
  P.ky = G->ky;
  for (int f = 0; f < 4; ++f) P.bc[f] = G->bc[f];
  P.ghost = G->ghost;
  X.f = G->f;
}

// corner of element e along one direction, x0 + e h rounded to float, in float-float arithmetic (FP64
// instructions would stall the element on the FP64 pipe); e < 2^24 or rounded once
__device__ __forceinline__ float corner_of(float x0, float x0l, float h, float hl, int e) {
  const float ef = (float)e, el = (float)(e - (int)ef);
  const ff p = two_prod(ef, h);
  const ff s = two_sum(x0, p.hi);
  return __fadd_rn(s.hi, __fadd_rn(s.lo, __fadd_rn(fmaf(ef, hl, fmaf(el, h, p.lo)), x0l)));
}

__device__ __forceinline__ VelElem make_vel(const StepParams& P, const Mixed2DExtra& X, float x0, float y0) {
  VelElem V;
  V.kind = P.vel_kind;
  V.x0 = x0;
  V.y0 = y0;
  V.hx = X.f.hx;
  V.hy = X.f.hy;
  V.ihx = X.f.ihx;
  V.ihy = X.f.ihy;
  V.pihx = 3.14159265358979f * X.f.hx;
  V.pihy = 3.14159265358979f * X.f.hy;
  V.direct = !(X.f.hx <= 0.25f && X.f.hy <= 0.25f);
  V.shortser = V.pihx <= 0.02f && V.pihy <= 0.02f;
  V.a = X.a;
  V.b = X.b;
  V.om = X.om;
  V.cx = X.cx;
  V.cy = X.cy;
  return V;
}

// Per-element sines and cosines of the swirl: sin and cos of pi x at the node x-coordinates n[0],
// n[1], y-coordinates n[2], n[3]; at the corner coordinates x0, x0 + hx, y0, y0 + hy (sines in
// corner[0..3], cosines in corner[4..7]); ct[k] = cos(pi (t + k dt / 4) / T).
template <int NN>
struct Trig {
  float n[4][NN];
  float corner[8];
  float ct[5];
};

template <int NN, int G>
__device__ __forceinline__ void trig_setup(const Grp<G>& g, const VelElem& V, const Mixed2DExtra& X, const float* xi,
                                           Trig<NN>& T) {
  // every lane evaluates one coordinate (a branch per kind of coordinate would run the evaluation four times)
  if (V.kind == SL_VEL_SWIRL) {
    for (int t = g.t; t < 2 * NN + 9; t += 32 * G) {
      const int c = t - 2 * NN;                              // corner, then stage-time index
      const bool y = t < 2 * NN ? t >= NN : c >= 2;
      const float h = y ? V.hy : V.hx, z0 = y ? V.y0 : V.x0;
      float z = c < 0 ? fmaf(h, xi[y ? t - NN : t], z0) : z0 + ((c & 1) ? h : 0.0f);
      if (c >= 4) z = fmaf(0.25f * (float)(c - 4), X.f.dtT, X.f.tT);
      float sn, cs;
      sincospif(z, &sn, &cs);
      if (c < 0) {
        T.n[y ? 2 : 0][y ? t - NN : t] = sn;
        T.n[y ? 3 : 1][y ? t - NN : t] = cs;
      } else if (c < 4) {
        T.corner[c] = sn;
        T.corner[4 + c] = cs;
      } else {
        T.ct[c - 4] = cs;
      }
    }
  } else if (g.t < 5) {
    T.ct[g.t] = 1.0f;
  }
}

// ------------------------------------------------------------------ phase 1
template <int NN>
struct Smem1 {
  static constexpr int ND = Shape<NN>::ND, NP = Shape<NN>::NP, RP = Shape<NN>::RP, G = Shape<NN>::G;
  __align__(16) float ph[NN * NP];             // psihat rows
  __align__(16) float psi[NN * NP];            // psi^n rows
  union {
    struct {                                   // the collocation solve
      __align__(16) float r[NN * NP], tt[NN * RP], Rx[NN * RP], Ry[NN * RP];   // residual rows, columns of the row pass
      float best[ND];
    } sv;
    struct {                                   // the face outflow, after the solve
      float fbo[4][NMAX][3];                   // per face point and distinct stage: outflow weight
      float fv[4][NMAX][3];                    //   and the outflow value (phi - r0)
      float pt[4][NMAX][4];                    // per face point: U_out, U_in, P1, P2 over the step
      float fs[4][4];                          // per face: the same summed over its points
      int items[4 * NMAX * 2];                 // outflow (point, stage) pairs that need a foot
    } fc;
  } u;
  float red[8 * G];
  float trp[4 * NN];                           // traces of psi^n at the own face points
  int cum[5];
  int nitems;
  Trig<NN> T;
  Elem el[2];                                  // this and the next element, its problem's record
  const ProbGeom* geo[2];
  float sth[2][ND], stl[2][ND];                // staged input state (hi, lo) of this and the next element
};

template <int NN, bool GEO>
__global__ void __launch_bounds__(Shape<NN>::NT, Shape<NN>::MINB)
    k_p1(StepParams P0, const __grid_constant__ Mixed2DExtra X0, Map2D M, int64_t count, const float* __restrict__ in,
         Work2M W, unsigned* status) {
  using S = Shape<NN>;
  constexpr int ND = S::ND, NP = S::NP, RP = S::RP, G = S::G, GT = S::GT, EPC = S::EPC;
  __shared__ float s_xi[NN], s_lam[NN], s_w[NN], s_l0[NN], s_l1[NN];
  __shared__ Smem1<NN> sm_all[EPC];
  if (threadIdx.x < NN) {
    s_xi[threadIdx.x] = X0.xi[threadIdx.x];
    s_lam[threadIdx.x] = X0.lam[threadIdx.x];
    s_w[threadIdx.x] = X0.w[threadIdx.x];
    s_l0[threadIdx.x] = X0.l0[threadIdx.x];
    s_l1[threadIdx.x] = X0.l1[threadIdx.x];
  }
  __syncthreads();
  Grp<G> g;
  g.slot = threadIdx.x / GT;
  g.t = threadIdx.x % GT;
  g.lane = threadIdx.x & 31;
  g.w = g.t >> 5;
  Smem1<NN>& sm = sm_all[g.slot];
  g.red = sm.red;
  g.rb = 0;
  const int t = g.t;
  const int p0 = t, p1 = t + GT;
  const bool v0 = p0 < ND, v1 = p1 < ND;
  const int i0 = p0 % NN, j0 = (p0 / NN) % NN, i1 = p1 % NN, j1 = (p1 / NN) % NN;
  // w (x) w at the thread's nodes as float-float
  const float2 w2h = make_float2(v0 ? X0.w2h[p0] : 0.0f, v1 ? X0.w2h[p1] : 0.0f);
  const float2 w2l = make_float2(v0 ? X0.w2l[p0] : 0.0f, v1 ? X0.w2l[p1] : 0.0f);
  unsigned c_it = 0, c_floor = 0, c_nc = 0, c_feet = 0;
  unsigned bits = 0;
  const int64_t ngroups = (int64_t)gridDim.x * EPC;
  // asynchronous copies of element kk's input state into staging buffer b (one group per call); the element
  // is resolved here, one iteration ahead
  auto stage = [&](int64_t kk, int b) {
    if (kk < count) {
      const ProbGeom* gn;
      const Elem En = elem_at<NN, GEO>(P0, M, kk, gn);
      if (t == 0) {
        sm.el[b] = En;
        sm.geo[b] = gn;
      }
      if (v0) { cp_async4(&sm.sth[b][p0], in + En.base + p0); cp_async4(&sm.stl[b][p0], in + X0.plane + En.base + p0); }
      if (v1) { cp_async4(&sm.sth[b][p1], in + En.base + p1); cp_async4(&sm.stl[b][p1], in + X0.plane + En.base + p1); }
    }
    cp_async_commit();
  };
  int64_t k = (int64_t)blockIdx.x * EPC + g.slot;
  stage(k, 0);
  for (int b = 0; k < count; k += ngroups, b ^= 1) {
    g.sync();                                    // the previous element's shared data is consumed
    const Elem E = sm.el[b];
    StepParams P = P0;
    Mixed2DExtra X = X0;
    if (GEO) use_problem(sm.geo[b], P, X);
    stage(k + ngroups, b ^ 1);
    cp_async_wait1();
    const int ex = E.ex, ey = E.ey;
    const VelElem V = make_vel(P, X, corner_of(X.f.x0, X.f.x0l, X.f.hx, X.f.hxl, ex),
                               corner_of(X.f.y0, X.f.y0l, X.f.hy, X.f.hyl, ey));
    trig_setup<NN>(g, V, X, s_xi, sm.T);
    g.sync();                                    // this element's staged state is visible
    const float* sh = sm.sth[b];
    const float* sl = sm.stl[b];
    // element reference: linear from the four corner values, or the first node value
    const float c00 = sh[0], c01 = sh[NN - 1], c10 = sh[(NN - 1) * NN], c11 = sh[ND - 1];
    float r0 = c00, gx = 0.0f, gy = 0.0f;
    if (X.linref) {
      r0 = 0.25f * ((c00 + c01) + (c10 + c11));
      gx = ((c01 + c11) - (c00 + c10)) * X.span;
      gy = ((c10 + c11) - (c00 + c01)) * X.span;
    }
    // psi^n at the own nodes, and the element mass in float-float
    const float2 hi2 = make_float2(v0 ? sh[p0] : 0.0f, v1 ? sh[p1] : 0.0f);
    const float2 lo2 = make_float2(v0 ? sl[p0] : 0.0f, v1 ? sl[p1] : 0.0f);
    const float2 ha = make_float2(s_xi[i0] - 0.5f, s_xi[i1] - 0.5f), hb = make_float2(s_xi[j0] - 0.5f, s_xi[j1] - 0.5f);
    const ff2 L2 = lref2(r0, gx, gy, ha, hb);
    const float2 pn2 = add2(sub2(hi2, L2.hi), sub2(lo2, L2.lo));
    const float pn0 = v0 ? pn2.x : 0.0f, pn1 = v1 ? pn2.y : 0.0f;
    if (v0) sm.psi[j0 * NP + i0] = pn0;
    if (v1) sm.psi[j1 * NP + i1] = pn1;
    const ff2 mn2 = ff_mul2(ff2{hi2, lo2}, w2h, w2l);
    const ff mn = ff_add(ff{mn2.hi.x, mn2.lo.x}, ff{mn2.hi.y, mn2.lo.y});
    // element sums of psi^n (reference measure) and the float-float element mass
    const float w20 = v0 ? s_w[i0] * s_w[j0] : 0.0f, w21 = v1 ? s_w[i1] * s_w[j1] : 0.0f;
    float m1 = fmaf(w20, pn0, w21 * pn1), m2 = fmaf(w20 * pn0, pn0, w21 * pn1 * pn1);
    g.sync();
    const ff Mn = g.ffsum_sum2(mn, m1, m2);
    float* el = W.elem + E.g * 8;
    if (t == 0) {
      el[0] = r0;
      el[1] = gx;
      el[2] = gy;
      el[3] = m1;
      el[4] = m2;
      el[5] = Mn.hi;
      el[6] = Mn.lo;
    }
    // advect the particles of nodes p0, p1 in reference coordinates
    float2 d2x = bc2(0.0f), d2y = bc2(0.0f);
    rk_disp2(V, P.rk, make_float2(s_xi[i0], s_xi[i1]), make_float2(s_xi[j0], s_xi[j1]),
             make_float2(sm.T.n[0][i0], sm.T.n[0][i1]), make_float2(sm.T.n[1][i0], sm.T.n[1][i1]),
             make_float2(sm.T.n[2][j0], sm.T.n[2][j1]), make_float2(sm.T.n[3][j0], sm.T.n[3][j1]), d2x, d2y, bc2(X.f.dt),
             [&](float c) { return bc2(sm.T.ct[__float2int_rn(4.0f * c)]); });
    const float dx0 = v0 ? d2x.x : 0.0f, dy0 = v0 ? d2y.x : 0.0f, dx1 = v1 ? d2x.y : 0.0f, dy1 = v1 ? d2y.y : 0.0f;
    float2 Lx[NN], Ly[NN];
    basis_at2<NN>(s_xi, s_lam, s_xi[i0], s_xi[i1], dx0, dx1, Lx);
    basis_at2<NN>(s_xi, s_lam, s_xi[j0], s_xi[j1], dy0, dy1, Ly);
    // collocation data of psihat = phihat - L
    const float ps0 = v0 ? pn0 - fmaf(gx, dx0, gy * dy0) : 0.0f;
    const float ps1 = v1 ? pn1 - fmaf(gx, dx1, gy * dy1) : 0.0f;
    float sdx = dx0 + dx1, sdy = dy0 + dy1, unused = 0.0f, scale = fmaxf(fabsf(ps0), fabsf(ps1));
    g.sum3max(sdx, sdy, unused, scale, false);
    const float mdx = sdx / ND, mdy = sdy / ND;
    // preconditioner: interpolation back over the mean displacement, Rx[i][q] = l_q(xi_i - mdx)
    if (t < 2 * NN) {
      float b[NN];
      const int row = t < NN ? t : t - NN;
      basis_at<NN>(s_xi, s_lam, s_xi[row], t < NN ? -mdx : -mdy, b);
      float* R = (t < NN ? sm.u.sv.Rx : sm.u.sv.Ry) + row * RP;
#pragma unroll
      for (int q = 0; q < NN; ++q) R[q] = b[q];
    }
    if (v0) sm.u.sv.r[j0 * NP + i0] = ps0;
    if (v1) sm.u.sv.r[j1 * NP + i1] = ps1;
    g.sync();
    // psihat (+)= Ry r Rx^T: the row pass leaves its result by columns, so that both passes read rows
    auto precond = [&](bool first) {
      if (v0) sm.u.sv.tt[i0 * RP + j0] = dot_rows<NN>(sm.u.sv.Rx + i0 * RP, sm.u.sv.r + j0 * NP);
      if (v1) sm.u.sv.tt[i1 * RP + j1] = dot_rows<NN>(sm.u.sv.Rx + i1 * RP, sm.u.sv.r + j1 * NP);
      g.sync();
      if (v0) {
        const float acc = dot_rows<NN>(sm.u.sv.Ry + j0 * RP, sm.u.sv.tt + i0 * RP);
        sm.ph[j0 * NP + i0] = first ? acc : sm.ph[j0 * NP + i0] + acc;
      }
      if (v1) {
        const float acc = dot_rows<NN>(sm.u.sv.Ry + j1 * RP, sm.u.sv.tt + i1 * RP);
        sm.ph[j1 * NP + i1] = first ? acc : sm.ph[j1 * NP + i1] + acc;
      }
      g.sync();
    };
    precond(true);
    // iterate to the tolerance; a residual that stalls at the float floor is accepted; the best
    // iterate is kept against divergence, and accepting it above the floor is reported
    float prev = INFINITY, best = INFINITY, rmax = INFINITY;
    int it = 0;
    bool done = false;
    for (; it < SOLVE_CAP; ++it) {
      float2 acc = make_float2(0.0f, 0.0f);
#pragma unroll
      for (int mm = 0; mm < NN; ++mm) {
        const float2 row = row_dot2<NN>(sm.ph + mm * NP, Lx);
        acc = __ffma2_rn(Ly[mm], row, acc);
      }
      const float r0v = ps0 - acc.x, r1v = ps1 - acc.y;
      rmax = g.max(fmaxf(v0 ? fabsf(r0v) : 0.0f, v1 ? fabsf(r1v) : 0.0f));
      // values below the normal float range carry no accuracy to refine
      if (rmax <= SOLVE_RTOL * scale || rmax == 0.0f || scale < 1e-30f) { done = true; break; }
      const bool stalled = rmax > 0.5f * prev && rmax <= SOLVE_STALL * scale;
      const bool diverging = !(rmax <= 4.0f * best);                             // or not finite
      if (stalled || diverging) break;
      if (rmax < best) {
        best = rmax;
        if (v0) sm.u.sv.best[p0] = sm.ph[j0 * NP + i0];
        if (v1) sm.u.sv.best[p1] = sm.ph[j1 * NP + i1];
      }
      prev = rmax;
      if (v0) sm.u.sv.r[j0 * NP + i0] = r0v;
      if (v1) sm.u.sv.r[j1 * NP + i1] = r1v;
      g.sync();
      precond(false);
    }
    c_it += it < SOLVE_CAP ? it + 1 : SOLVE_CAP;
    if (!done) {
      // stalled, diverging or at the cap: the better of the last and the best iterate
      float acc_r = rmax;
      if (!(rmax <= best)) {
        if (v0) sm.ph[j0 * NP + i0] = sm.u.sv.best[p0];
        if (v1) sm.ph[j1 * NP + i1] = sm.u.sv.best[p1];
        acc_r = best;
        g.sync();
      }
      if (acc_r <= SOLVE_STALL * scale) {
        // the float floor of the residual: the solve is as accurate as float allows
      } else if (acc_r <= SOLVE_FLOOR * scale) {
        ++c_floor;
        bits |= SL_ST_SOLVE_FLOOR;
      } else {
        ++c_nc;
        bits |= SL_ST_SOLVE_NOCONV;
      }
    }
    if (v0) W.psihat[E.base + p0] = sm.ph[j0 * NP + i0];
    if (v1) W.psihat[E.base + p1] = sm.ph[j1 * NP + i1];
    // interface values at the face points (relative to L): traces of psihat, or phi^n at the
    // backward characteristic foot of the face point from t^{n+1} (eq. 4.11; meshes of one node
    // count), L(foot) - L(face point) being the linear part over the foot's displacement
    float ub = 0.0f, tr0 = 0.0f;                 // own face point: u.n at ct = 1, the trace of psi^n
    const bool flux = (P.cons & (SL_C_MASS | SL_C_ENERGY)) != 0;
    static_assert(4 * NN <= GT, "a thread per own face point");
    if (t < 4 * NN) {
      const int f = t / NN, q = t % NN;
      const float xr = f == 0 ? 0.0f : f == 1 ? 1.0f : s_xi[q];
      const float yr = f == 2 ? 0.0f : f == 3 ? 1.0f : s_xi[q];
      float Sx = 0.0f, Cx = 0.0f, Sy = 0.0f, Cy = 0.0f;
      if (V.kind == SL_VEL_SWIRL && !V.direct) {
        Sx = f < 2 ? sm.T.corner[f] : sm.T.n[0][q];
        Cx = f < 2 ? sm.T.corner[4 + f] : sm.T.n[1][q];
        Sy = f < 2 ? sm.T.n[2][q] : sm.T.corner[f];
        Cy = f < 2 ? sm.T.n[3][q] : sm.T.corner[4 + f];
      }
      float ur, vr;
      vel_base(V, xr, yr, Sx, Cx, Sy, Cy, 1.0f, ur, vr);
      ub = (f == 0 || f == 2 ? -1.0f : 1.0f) * (f < 2 ? ur * X.f.hx : vr * X.f.hy);
      const float* Lb = (f == 1 || f == 3) ? s_l1 : s_l0;
      const int at = f < 2 ? q * NP : q, st = f < 2 ? 1 : NP;
      float acc = 0.0f;
      if (P.bvalue == SL_BV_BACKTRACK) {
        float fdx = 0.0f, fdy = 0.0f;
        rk_disp(V, P.rk, xr, yr, Sx, Cx, Sy, Cy, fdx, fdy, -X.f.dt, 1.0f, -1.0f, sm.T.ct);
        float bx[NN], by[NN];
        basis_at<NN>(s_xi, s_lam, xr, fdx, bx);
        basis_at<NN>(s_xi, s_lam, yr, fdy, by);
#pragma unroll
        for (int mm = 0; mm < NN; ++mm) acc = fmaf(by[mm], row_dot<NN>(sm.psi + mm * NP, bx), acc);
        acc += fmaf(gx, fdx, gy * fdy);
      } else {
        float a2 = 0.0f;
#pragma unroll
        for (int kk = 0; kk < NN; ++kk) {
          acc = fmaf(sm.ph[at + kk * st], Lb[kk], acc);
          a2 = fmaf(sm.psi[at + kk * st], Lb[kk], a2);
        }
        tr0 = a2;
        sm.trp[t] = a2;
      }
      W.traces[E.g * M.tstride + t] = acc;
      // the upwind side of the face point at t^{n+1} (eq. 4.12a): 0 own, 1 the neighbour's or the ghost, 2 tie
      if (P.cons & SL_C_BOUNDARY) {
        const float un = ub * sm.T.ct[4];
        W.side[E.g * M.tstride + t] = un > (float)TIE ? 0 : un < -(float)TIE ? 1 : 2;
      }
    }
    // outflow over each face and step; a face shared with a neighbour of another node count takes
    // the rule of the finer side, so that both elements integrate the same points.  Pass 1 (one face
    // point per thread): the sign of u.n at each distinct stage time, the quadrature weights, and at
    // the stage time t^n the outflow value itself (the trace of psi^n, no foot).  Pass 2: the outflow
    // (point, stage) pairs of later stage times, compacted into a list, one backward characteristic
    // foot each.  Every pair writes its own slot; the face sums add the slots in a fixed order.
    // Conforming elements of at most 13 nodes under the swirl take both later feet (at most two) of a face point
    // at once in paired operations instead, with no list: a list of more than 32 pairs cost a second round, and
    // the list its atomics and the values' way through shared memory (phase 1 with the list / with this, 4.2 M
    // nodes: 505 / 476 us at n = 4, 290 / 276 at n = 6, 179 / 172 at n = 8, 334 / 320 at n = 12, but 376 / 398 at
    // n = 14, where the paired bases no longer fit the registers).
    if (flux) {
      if (t < 4) {
        // points of face t and their prefix sum (lanes 0-3 of the first warp)
        const int nb = nb_index(P, ex, ey, t);
        const int nq = nb < 0 ? NN : max(NN, order_of<NN>(M, E.gb + nb));
        int acc = nq;
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
          const int v = __shfl_up_sync(0xfu, acc, o);
          if (t >= o) acc += v;
        }
        sm.cum[t + 1] = acc;
        if (t == 0) {
          sm.cum[0] = 0;
          sm.nitems = 0;
        }
      }
      g.sync();
      const int S = c_ds_n[P.rk];
      const int total = sm.cum[4];
      // Geometry of face point idx: face, point, rule, reference coordinates, sines and cosines.
      // CONF: every face takes the element's own rule (conforming neighbours), so that no lane
      // carries the general rule's branches.
      auto face_point = [&](auto conf, int idx, int& f, int& q, int& nq, float& zq, float& xr, float& yr, float& Sx,
                            float& Cx, float& Sy, float& Cy) {
        constexpr bool CONF = decltype(conf)::value;
        if (CONF) {
          f = idx / NN;
          q = idx % NN;
          nq = NN;
        } else {
          f = (idx >= sm.cum[1]) + (idx >= sm.cum[2]) + (idx >= sm.cum[3]);
          q = idx - sm.cum[f];
          nq = sm.cum[f + 1] - sm.cum[f];
        }
        zq = (CONF || nq == NN) ? s_xi[q] : X.rules[(size_t)nq * 3 * NMAX + q];
        xr = f == 0 ? 0.0f : f == 1 ? 1.0f : zq;
        yr = f == 2 ? 0.0f : f == 3 ? 1.0f : zq;
        Sx = Cx = Sy = Cy = 0.0f;
        if (V.kind == SL_VEL_SWIRL && !V.direct) {
          if (f < 2) {
            Sx = sm.T.corner[f];
            Cx = sm.T.corner[4 + f];
            if (CONF || nq == NN) { Sy = sm.T.n[2][q]; Cy = sm.T.n[3][q]; }
            else sincospif(fmaf(V.hy, zq, V.y0), &Sy, &Cy);
          } else {
            Sy = sm.T.corner[f];
            Cy = sm.T.corner[4 + f];
            if (CONF || nq == NN) { Sx = sm.T.n[0][q]; Cx = sm.T.n[1][q]; }
            else sincospif(fmaf(V.hx, zq, V.x0), &Sx, &Cx);
          }
        }
      };
      constexpr bool PAIRED = NN <= 13;
      const bool conforming = total == 4 * NN;
      const bool tab = V.kind == SL_VEL_SWIRL && !V.direct;
      // CONF: conforming faces; TAB: the swirl from the tabulated sines (both known per element)
      auto pass1 = [&](auto conf, auto tabc) {
      constexpr bool CONF = decltype(conf)::value;
      constexpr bool PAIR = CONF && decltype(tabc)::value && PAIRED;
      for (int idx = t; idx < total; idx += GT) {
        int f, q, nq;
        float zq, xr, yr, Sx, Cx, Sy, Cy;
        face_point(conf, idx, f, q, nq, zq, xr, yr, Sx, Cx, Sy, Cy);
        const float hn = f < 2 ? X.f.hx : X.f.hy;            // velocity in reference units times this = u.n
        const float sg = (f == 0 || f == 2) ? -1.0f : 1.0f;
        const float Wq = (f < 2 ? X.f.hy : X.f.hx) *
                         ((CONF || nq == NN) ? s_w[q] : X.rules[(size_t)nq * 3 * NMAX + 2 * NMAX + q]);
        // phi - r0 at the face point itself (stage time t^n): the trace of psi^n plus (L - r0); u.n at ct = 1
        float val0, ubase;
        if (CONF && P.bvalue != SL_BV_BACKTRACK) {
          val0 = tr0;                              // this thread's own face point, formed with the traces
        } else if (CONF || nq == NN) {
          const float* Lb = (f == 1 || f == 3) ? s_l1 : s_l0;
          float acc = 0.0f;
#pragma unroll
          for (int kk = 0; kk < NN; ++kk) acc = fmaf(f < 2 ? sm.psi[q * NP + kk] : sm.psi[kk * NP + q], Lb[kk], acc);
          val0 = acc;
        } else {
          // a point of another rule: the own traces interpolated along the face (with backtracked values the
          // mesh has one node count)
          float bt[NN];
          basis_at<NN>(s_xi, s_lam, zq, 0.0f, bt);
          float acc = 0.0f;
#pragma unroll
          for (int mm = 0; mm < NN; ++mm) acc = fmaf(bt[mm], sm.trp[f * NN + mm], acc);
          val0 = acc;
        }
        val0 += fmaf(gx, xr - 0.5f, gy * (yr - 0.5f));
        if (CONF) {
          ubase = ub;
        } else {
          float ur, vr;
          vel_base(V, xr, yr, Sx, Cx, Sy, Cy, 1.0f, ur, vr);
          ubase = sg * (f < 2 ? ur : vr) * hn;
        }
        // per distinct stage time: the sign of u.n, the weight; later stage times that flow out
        // are queued for their backward foot (their weight kept in fbo, 0 otherwise)
        float uo = 0.0f, ui = 0.0f, q1 = 0.0f, q2 = 0.0f;
        float2 bo = bc2(0.0f);                     // PAIR: outflow weights of the later stage times
        for (int s = 0; s < S; ++s) {
          const float cs = c_ds_c[P.rk][s];
          const float un = ubase * sm.T.ct[__float2int_rn(4.0f * cs)];
          const float bw = c_ds_b[P.rk][s] * Wq * un;
          const bool out = un > (float)TIE;
          if (out) uo += bw;
          if (un < -(float)TIE) ui += bw;
          if (cs == 0.0f) {
            if (out) {
              q1 = fmaf(bw, val0, q1);
              q2 = fmaf(bw * val0, val0, q2);
            }
          } else if (PAIR) {
            if (s == S - 1) bo.y = out ? bw : 0.0f;          // t^{n+1} is the last one,
            else bo.x = out ? bw : 0.0f;                     // t^{n+1/2} any other
          } else {
            sm.u.fc.fbo[f][q][s] = out ? bw : 0.0f;
            // queue the pair: one shared atomic per warp (lane order within the warp)
            const unsigned act = __activemask();
            const unsigned want = __ballot_sync(act, out);
            if (want) {
              const int leader = __ffs(act) - 1;
              int base = 0;
              if (g.lane == leader) base = atomicAdd(&sm.nitems, __popc(want));
              base = __shfl_sync(act, base, leader);
              if (out) sm.u.fc.items[base + __popc(want & ((1u << g.lane) - 1u))] = idx * 4 + s;
            }
          }
        }
        if (PAIR && (bo.x != 0.0f || bo.y != 0.0f)) {
          c_feet += (bo.x != 0.0f) + (bo.y != 0.0f);
          float2 fdx, fdy;
          const float2 h = make_float2(-0.5f * X.f.dt, -X.f.dt);
          rk_disp2(V, P.rk, bc2(xr), bc2(yr), bc2(Sx), bc2(Cx), bc2(Sy), bc2(Cy), fdx, fdy, h, [&](float c) {
            return make_float2(sm.T.ct[2 - __float2int_rn(2.0f * c)], sm.T.ct[4 - __float2int_rn(4.0f * c)]);
          });
          float2 bx[NN], by[NN];
          basis_at2<NN>(s_xi, s_lam, xr, xr, fdx.x, fdx.y, bx);
          basis_at2<NN>(s_xi, s_lam, yr, yr, fdy.x, fdy.y, by);
          float2 val = bc2(0.0f);
#pragma unroll
          for (int mm = 0; mm < NN; ++mm) val = fma2(by[mm], row_dot2<NN>(sm.psi + mm * NP, bx), val);
          // phi - r0 = (L - r0) + psi
          val = add2(val, fma2(bc2(gx), add2(bc2(xr - 0.5f), fdx), mul2(bc2(gy), add2(bc2(yr - 0.5f), fdy))));
          if (bo.x != 0.0f) {
            q1 = fmaf(bo.x, val.x, q1);
            q2 = fmaf(bo.x * val.x, val.x, q2);
          }
          if (bo.y != 0.0f) {
            q1 = fmaf(bo.y, val.y, q1);
            q2 = fmaf(bo.y * val.y, val.y, q2);
          }
        }
        sm.u.fc.pt[f][q][0] = uo;
        sm.u.fc.pt[f][q][1] = ui;
        sm.u.fc.pt[f][q][2] = q1;
        sm.u.fc.pt[f][q][3] = q2;
      }
      };
      if (conforming && tab) pass1(std::true_type{}, std::true_type{});
      else pass1(std::false_type{}, std::false_type{});
      g.sync();
      if (!(PAIRED && conforming && tab)) {
        const int nitems = sm.nitems;
        if (t == 0) c_feet += nitems;
        for (int it2 = t; it2 < nitems; it2 += GT) {
          const int code = sm.u.fc.items[it2];
          const int idx = code >> 2, s = code & 3;
          int f, q, nq;
          float zq, xr, yr, Sx, Cx, Sy, Cy;
          if (conforming) face_point(std::true_type{}, idx, f, q, nq, zq, xr, yr, Sx, Cx, Sy, Cy);
          else face_point(std::false_type{}, idx, f, q, nq, zq, xr, yr, Sx, Cx, Sy, Cy);
          const float cs = c_ds_c[P.rk][s];
          float fdx = 0.0f, fdy = 0.0f;
          rk_disp(V, P.rk, xr, yr, Sx, Cx, Sy, Cy, fdx, fdy, -cs * X.f.dt, cs, -cs, sm.T.ct);
          float bx[NN], by[NN];
          basis_at<NN>(s_xi, s_lam, xr, fdx, bx);
          basis_at<NN>(s_xi, s_lam, yr, fdy, by);
          float val = 0.0f;
  #pragma unroll
          for (int mm = 0; mm < NN; ++mm) val = fmaf(by[mm], row_dot<NN>(sm.psi + mm * NP, bx), val);
          val += fmaf(gx, (xr - 0.5f) + fdx, gy * ((yr - 0.5f) + fdy));   // phi - r0 = (L - r0) + psi
          sm.u.fc.fv[f][q][s] = val;
        }
        g.sync();
        // per face point: the outflow of the later stage times, added in stage order
        if (S > 1)
          for (int idx = t; idx < total; idx += GT) {
            const int f = (idx >= sm.cum[1]) + (idx >= sm.cum[2]) + (idx >= sm.cum[3]);
            const int q = idx - sm.cum[f];
            float q1 = sm.u.fc.pt[f][q][2], q2 = sm.u.fc.pt[f][q][3];
            for (int s = 1; s < S; ++s) {
              const float bo = sm.u.fc.fbo[f][q][s];
              if (bo != 0.0f) {
                const float v = sm.u.fc.fv[f][q][s];
                q1 = fmaf(bo, v, q1);
                q2 = fmaf(bo * v, v, q2);
              }
            }
            sm.u.fc.pt[f][q][2] = q1;
            sm.u.fc.pt[f][q][3] = q2;
          }
        g.sync();
      }
      // per face and quantity (16 threads): the sum over the face's points in point order
      if (t < 16) {
        const int f = t >> 2, c = t & 3;
        const int nq = sm.cum[f + 1] - sm.cum[f];
        float acc = 0.0f;
        if (conforming) {
#pragma unroll
          for (int q = 0; q < NN; ++q) acc += sm.u.fc.pt[f][q][c];
        } else {
          for (int q = 0; q < nq; ++q) acc += sm.u.fc.pt[f][q][c];
        }
        sm.u.fc.fs[f][c] = acc;
      }
      g.sync();
      if (t < 4) {
        const int f = t;
        const float uo = sm.u.fc.fs[f][0], ui = sm.u.fc.fs[f][1], q1 = sm.u.fc.fs[f][2], q2 = sm.u.fc.fs[f][3];
        // the face's outflow flux of phi as a float-float value: r0 U_out + sum bw (phi - r0), plus
        // the inflow of the ghost value through a domain face
        ff Gf = ff_add(two_prod(r0, uo), ff{q1, 0.0f});
        if (nb_index(P, ex, ey, f) < 0) Gf = ff_add(Gf, two_prod((float)P.ghost, ui));
        float* F = W.faces + E.g * 24 + 6 * f;
        F[0] = Gf.hi;
        F[1] = Gf.lo;
        F[2] = uo;
        F[3] = ui;
        F[4] = q1;
        F[5] = q2;
      }
    }
  }
  if (t == 0 && X0.counts) {
    atomicAdd(X0.counts + SL_CNT_SOLVE_ITERS, (unsigned long long)c_it);
    if (c_floor) atomicAdd(X0.counts + SL_CNT_SOLVE_FLOOR, (unsigned long long)c_floor);
    if (c_nc) atomicAdd(X0.counts + SL_CNT_SOLVE_NOCONV, (unsigned long long)c_nc);
  }
  c_feet = __reduce_add_sync(0xffffffffu, c_feet);
  if (g.lane == 0 && c_feet && X0.counts) atomicAdd(X0.counts + SL_CNT_FEET, (unsigned long long)c_feet);
  if (bits) atomicOr(status, bits);
}

// ------------------------------------------------------------------ phase 2
// the neighbour's trace across a p-nonconforming face, out of line: its 2 x 17 products in registers would set
// the register count of the whole kernel
static __device__ __noinline__ float interp_far(const float* rules, int nn, const float* tr, float z) {
  return interp_rule(rules, nn, tr, z);
}

template <int NN>
struct Smem2 {
  static constexpr int ND = Shape<NN>::ND, G = Shape<NN>::G;
  static constexpr int MMAX = 4 * NN + 1;
  __align__(16) float2 r[(MMAX + 1) & ~1];     // residuals, each twice (operands of the paired products)
  __align__(16) float2 ca[(MMAX + 1) & ~1];
  float a[ND];
  int rows[G];                                 // per warp: faces with a non-zero residual among its points
  float red[8 * G];
  float scal[8];
};

template <int NN, bool GEO>
__global__ void __launch_bounds__(Shape<NN>::NT, Shape<NN>::MINB2)
    k_p2(StepParams P0, const __grid_constant__ Mixed2DExtra X0, Map2D M, int64_t count, const float* __restrict__ in,
         Work2M W, float* __restrict__ out, unsigned* status) {
  using S = Shape<NN>;
  constexpr int ND = S::ND, G = S::G, GT = S::GT, EPC = S::EPC;
  __shared__ float s_xi[NN], s_w[NN], s_l0[NN], s_l1[NN];
  __shared__ Smem2<NN> sm_all[EPC];
  // the pseudo-inverse of the fit by row, a thread's two nodes side by side (zero where it has none), staged
  // once per CTA (dynamic shared memory): one 8-byte load and one paired FMA per row and thread
  extern __shared__ __align__(16) float2 s_Cp[];               // [m][GT]
  if (threadIdx.x < NN) {
    s_xi[threadIdx.x] = X0.xi[threadIdx.x];
    s_w[threadIdx.x] = X0.w[threadIdx.x];
    s_l0[threadIdx.x] = X0.l0[threadIdx.x];
    s_l1[threadIdx.x] = X0.l1[threadIdx.x];
  }
  for (int i = threadIdx.x; i < P0.m * GT; i += blockDim.x) {
    const int kk = i / GT, c = i % GT;
    s_Cp[i] = make_float2(c < ND ? X0.Cp[kk * ND + c] : 0.0f, c + GT < ND ? X0.Cp[kk * ND + c + GT] : 0.0f);
  }
  __syncthreads();
  Grp<G> g;
  g.slot = threadIdx.x / GT;
  g.t = threadIdx.x % GT;
  g.lane = threadIdx.x & 31;
  g.w = g.t >> 5;
  Smem2<NN>& sm = sm_all[g.slot];
  g.red = sm.red;
  g.rb = 0;
  const int t = g.t;
  const int p0 = t, p1 = t + GT;
  const bool v0 = p0 < ND, v1 = p1 < ND;
  const int i0 = p0 % NN, j0 = (p0 / NN) % NN, i1 = p1 % NN, j1 = (p1 / NN) % NN;
  const float w20 = v0 ? s_w[i0] * s_w[j0] : 0.0f, w21 = v1 ? s_w[i1] * s_w[j1] : 0.0f;
  unsigned c_el = 0, c_eapp = 0, c_pit = 0, c_pnc = 0;
  unsigned bits = 0;
  const int64_t ngroups = (int64_t)gridDim.x * EPC;
  for (int64_t k = (int64_t)blockIdx.x * EPC + g.slot; k < count; k += ngroups) {
    g.sync();
    StepParams P = P0;
    const ProbGeom* geo;
    const Elem E = elem_at<NN, GEO>(P0, M, k, geo);
    Mixed2DExtra X = X0;
    if (GEO) use_problem(geo, P, X);
    const int ex = E.ex, ey = E.ey;
    // every global read of the element first, so that they share one memory round trip: own
    // record, psihat, input (energy), face-point traces and the neighbours' records and faces
    const bool bnd = (P.cons & SL_C_BOUNDARY) != 0;
    const bool mass = (P.cons & SL_C_MASS) != 0, energy = (P.cons & SL_C_ENERGY) != 0;
    const int nb_rows = bnd ? 4 * NN : 0;
    const float* el = W.elem + E.g * 8;
    const float r0 = el[0], gx = el[1], gy = el[2], m1 = el[3], mn_hi = el[5], mn_lo = el[6];
    const float ph0 = v0 ? W.psihat[E.base + p0] : 0.0f;
    const float ph1 = v1 ? W.psihat[E.base + p1] : 0.0f;
    float in_hi0 = 0.0f, in_lo0 = 0.0f, in_hi1 = 0.0f, in_lo1 = 0.0f;
    if (energy) {
      if (v0) { in_hi0 = in[E.base + p0]; in_lo0 = in[X.plane + E.base + p0]; }
      if (v1) { in_hi1 = in[E.base + p1]; in_lo1 = in[X.plane + E.base + p1]; }
    }
    // boundary lanes: face point (f, q), own trace, neighbour's trace at this point and record
    int bf = 0, bq = 0, bnb = -1, bside = 0;
    float own = 0.0f, trn = 0.0f, en0 = 0.0f, en1 = 0.0f, en2 = 0.0f;
    if (bnd && t < 4 * NN) {
      bf = t / NN;
      bq = t % NN;
      bnb = nb_index(P, ex, ey, bf);
      own = W.traces[E.g * M.tstride + t];
      bside = W.side[E.g * M.tstride + t];
      if (bnb >= 0) {
        const int64_t gn = E.gb + bnb;
        const int nn = order_of<NN>(M, gn);
        const float* tr = W.traces + gn * M.tstride + (bf ^ 1) * nn;
        const float* en = W.elem + gn * 8;
        en0 = en[0];
        en1 = en[1];
        en2 = en[2];
        trn = nn == NN ? tr[bq] : interp_far(X.rules, nn, tr, s_xi[bq]);
      }
    }
    // face lanes (0-3): own face record, the neighbour's record of the shared face and its r0
    int fnb = -1;
    float F[6] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f}, Gn[6] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f}, rnb = 0.0f;
    if ((mass || energy) && t < 4) {
      fnb = nb_index(P, ex, ey, t);
      const float* Fp = W.faces + E.g * 24 + 6 * t;
#pragma unroll
      for (int c = 0; c < 6; ++c) F[c] = Fp[c];
      if (fnb >= 0) {
        const float* Gp = W.faces + (E.gb + fnb) * 24 + 6 * (t ^ 1);
#pragma unroll
        for (int c = 0; c < 6; ++c) Gn[c] = Gp[c];
        rnb = W.elem[(E.gb + fnb) * 8];
      }
    }
    float rr = 0.0f;
    if (bnd && t < 4 * NN) {
      const int f = bf, q = bq, nb = bnb;
      // neighbour's value at this element's face point relative to this element's L: the difference
      // of the two references (float-float, of the size of psi when both fit the same data) plus the
      // neighbour's trace of its own psihat
      const float aq = s_xi[q] - 0.5f;
      const float fa = f == 0 ? -0.5f : f == 1 ? 0.5f : aq, fb = f == 2 ? -0.5f : f == 3 ? 0.5f : aq;
      const ff lown = lref(r0, gx, gy, fa, fb);
      float other;
      if (nb >= 0) {
        const ff lnb = lref(en0, en1, en2, f == 0 ? 0.5f : f == 1 ? -0.5f : fa, f == 2 ? 0.5f : f == 3 ? -0.5f : fb);
        const float dl = __fadd_rn(__fsub_rn(lnb.hi, lown.hi), __fsub_rn(lnb.lo, lown.lo));
        other = dl + trn;
      } else {
        other = __fsub_rn(__fsub_rn((float)P.ghost, lown.hi), lown.lo);
      }
      float val;
      if (bside == 0) val = own;
      else if (bside == 1) val = other;
      else val = nb < 0 ? own : 0.5f * (own + other);
      // the row's value at psihat: the own trace when the interface values are traces of psihat,
      // else the trace formed here from the stored psihat
      float trh = own;
      if (P.bvalue == SL_BV_BACKTRACK) {
        const float* Lb = (f == 1 || f == 3) ? s_l1 : s_l0;
        const float* ps = W.psihat + E.base;
        trh = 0.0f;
#pragma unroll
        for (int kk = 0; kk < NN; ++kk) trh = fmaf(f < 2 ? ps[q * NN + kk] : ps[kk * NN + q], Lb[kk], trh);
      }
      rr = val - trh;
      sm.r[t] = bc2(rr);
    }
    // faces whose rows all vanish (outflow faces: the own trace) add nothing to the fit
    if (bnd && 32 * g.w < 4 * NN) {
      const unsigned nz = __ballot_sync(0xffffffffu, !(rr == 0.0f));
      int rows = 0;
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        const int lo = f * NN - 32 * g.w, hi = lo + NN;        // lanes of face f in this warp
        const unsigned a = lo <= 0 ? 0xffffffffu : lo >= 32 ? 0u : 0xffffffffu << lo;
        const unsigned b = hi >= 32 ? 0xffffffffu : hi <= 0 ? 0u : (1u << hi) - 1u;
        rows |= (nz & a & b) ? 1 << f : 0;
      }
      if (g.lane == 0) sm.rows[g.w] = rows;
    } else if (g.lane == 0) {
      sm.rows[g.w] = 0;
    }
    // net outflow of mass (increments), of the squared increments and of the velocity, lanes 0-3 of
    // the first warp one face each, summed in face order; the float-float mass target
    if ((mass || energy) && t < 32) {
      float cu = 0.0f, cm = 0.0f, cd = 0.0f;
      ff net = {0.0f, 0.0f};
      if (t < 4) {
        cu = F[2] + F[3];
        net = ff{F[0], F[1]};
        if (fnb >= 0) {
          const float dref = rnb - r0;
          // inflow part: u.n (dref + psi_nb) with the neighbour's u.n = -ours
          cm = F[4] + (dref * F[3] - Gn[4]);
          cd = F[5] + (dref * dref * F[3] - 2.0f * dref * Gn[4] - Gn[5]);
          net = ff_add(net, ff_neg(ff{Gn[0], Gn[1]}));
        } else {
          const float gg = (float)P.ghost - r0;
          cm = F[4] + gg * F[3];
          cd = F[5] + gg * gg * F[3];
        }
      }
      float su = 0.0f, smm = 0.0f, sd = 0.0f;
      ff sn = {0.0f, 0.0f};
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        su += __shfl_sync(0xffffffffu, cu, f);
        smm += __shfl_sync(0xffffffffu, cm, f);
        sd += __shfl_sync(0xffffffffu, cd, f);
        sn = ff_add(sn, ff{__shfl_sync(0xffffffffu, net.hi, f), __shfl_sync(0xffffffffu, net.lo, f)});
      }
      if (t == 0) {
        // M^{n+1} = M^n - dt / (hx hy) (net outflow), in float-float
        const ff ln = ff_mul(sn, ff{X.f.lam_hi, X.f.lam_lo});
        const ff target = ff_add(ff{mn_hi, mn_lo}, ff_neg(ln));
        sm.scal[0] = smm;
        sm.scal[1] = sd;
        sm.scal[2] = su;
        sm.scal[3] = target.hi;
        sm.scal[4] = target.lo;
      }
    }
    g.sync();
    const float netm = sm.scal[0], netd2 = sm.scal[1];
    const ff target = {sm.scal[3], sm.scal[4]};
    const float lam = X.f.lam_hi;                 // dt / (hx hy)
    if (mass) {
      const float mh = g.sum(fmaf(w20, ph0, w21 * ph1));
      // target (increments): sum w psi^n - lam (net increment outflow + ref * closed-surface u.n);
      // ref * (closed-surface integral of u.n) is dropped: every 2D velocity here is divergence free
      // and the face quadrature integrates it to rounding (the refinement below meets the float-float
      // target whatever this residual leaves)
      if (t == 0) sm.r[nb_rows] = bc2((m1 - lam * netm) - mh);
    }
    g.sync();
    const int m = P.m;
    float2 L2 = make_float2(ph0, ph1);
    int rows = 0;
#pragma unroll
    for (int w = 0; w < G; ++w) rows |= sm.rows[w];
#pragma unroll
    for (int f = 0; f < 4; ++f)
      if (rows & (1 << f)) {
        const float2* c = s_Cp + f * NN * GT + t;
#pragma unroll
        for (int kk = 0; kk < NN; ++kk) L2 = fma2(c[kk * GT], sm.r[f * NN + kk], L2);
      }
    if (mass) L2 = fma2(s_Cp[nb_rows * GT + t], sm.r[nb_rows], L2);
    const float phL0 = L2.x, phL1 = L2.y;
    float cur0 = phL0, cur1 = phL1;
    bool ok = true;
    if (energy) {
      // energy mismatch from increments (mass enforced): sum w (psiL - psi)(psiL + psi) + lam net(delta^2);
      // without the mass row, add 2 ref times the mass residual (closed-surface u.n taken as zero)
      float psin0 = 0.0f, psin1 = 0.0f;
      if (v0) {
        const ff L = lref(r0, gx, gy, s_xi[i0] - 0.5f, s_xi[j0] - 0.5f);
        psin0 = __fadd_rn(__fsub_rn(in_hi0, L.hi), __fsub_rn(in_lo0, L.lo));
      }
      if (v1) {
        const ff L = lref(r0, gx, gy, s_xi[i1] - 0.5f, s_xi[j1] - 0.5f);
        psin1 = __fadd_rn(__fsub_rn(in_hi1, L.hi), __fsub_rn(in_lo1, L.lo));
      }
      const float dp0 = phL0 - psin0, dp1 = phL1 - psin1;
      float ev = fmaf(w20 * dp0, phL0 + (phL0 - dp0), w21 * dp1 * (phL1 + (phL1 - dp1)));
      float ml = fmaf(w20, phL0, w21 * phL1);
      float escale = fmaf(w20 * (r0 + cur0), r0 + cur0, w21 * (r0 + cur1) * (r0 + cur1));
      float smax = fmaxf(fmaxf(fabsf(phL0), fabsf(phL1)), fabsf(r0));
      g.sum3max(ev, ml, escale, smax, true);
      float gamma;
      if (mass) gamma = ev + lam * netd2;
      else gamma = fmaf(2.0f * r0, (ml - m1) + lam * netm, ev + lam * netd2);
      if (smax >= 1e-30f && fabsf(gamma) > (float)ENERGY_SKIP_RTOL_MIXED * escale) {
        ++c_eapp;
        int exn;
        frexpf(smax, &exn);
        const float sc = ldexpf(1.0f, -exn), usc = ldexpf(1.0f, exn);
        const float rf = r0 * sc, gm = gamma * sc * sc;
        const float ql0 = phL0 * sc, ql1 = phL1 * sc;
        float c20 = ql0, c21 = ql1;
        const float tol = 2.4e-7f + 1e-30f;         // scaled units: values are of order one
        bool conv = false, feasible = true;
        int it = 0;
        for (; it < P.picard_cap; ++it) {
          const float a0 = w20 * (mass ? c20 : rf + c20), a1 = w21 * (mass ? c21 : rf + c21);
          if (v0) sm.a[p0] = a0;
          if (v1) sm.a[p1] = a1;
          g.sync();
          if (bnd && t < 4 * NN) {
            const int f = t / NN, qq = t % NN;
            const float* Lb = (f == 1 || f == 3) ? s_l1 : s_l0;
            float acc = 0.0f;
            for (int kk = 0; kk < NN; ++kk) acc = fmaf(f < 2 ? sm.a[qq * NN + kk] : sm.a[kk * NN + qq], Lb[kk], acc);
            sm.ca[t] = bc2(-acc);
          }
          if (mass) {
            const float cmm = g.sum(fmaf(w20, a0, w21 * a1));
            if (t == 0) sm.ca[nb_rows] = bc2(-cmm);
          }
          g.sync();
          float2 q2 = make_float2(a0, a1);
#pragma unroll 4
          for (int kk = 0; kk < m; ++kk) q2 = fma2(s_Cp[kk * GT + t], sm.ca[kk], q2);
          const float q0 = q2.x, q1 = q2.y;
          const float2 ab = g.sum2(fmaf(w20 * ql0, q0, w21 * ql1 * q1), fmaf(w20 * q0, q0, w21 * q1 * q1));
          float alpha = ab.x;
          if (!mass) alpha = fmaf(rf, g.sum(fmaf(w20, q0, w21 * q1)), alpha);
          const float beta = ab.y;
          float s;
          if (beta <= 0.0f) { s = 0.0f; feasible = gm <= 0.0f; }
          else {
            const float disc = alpha * alpha - beta * gm;
            if (disc < 0.0f) { s = -alpha / beta; feasible = false; }
            else {
              const float root = sqrtf(disc);
              const float den = alpha + (alpha >= 0.0f ? root : -root);
              s = den == 0.0f ? 0.0f : -gm / den;
              feasible = true;
            }
          }
          const float nv0 = v0 ? fmaf(s, q0, ql0) : 0.0f, nv1 = v1 ? fmaf(s, q1, ql1) : 0.0f;
          const float delta = g.max(fmaxf(fabsf(nv0 - c20), fabsf(nv1 - c21)));
          c20 = nv0;
          c21 = nv1;
          if (delta <= tol) { conv = feasible; break; }
        }
        c_pit += it < P.picard_cap ? it + 1 : P.picard_cap;
        if (conv) {                                 // else keep the linear-constraint solution
          cur0 = c20 * usc;
          cur1 = c21 * usc;
        }
        ok = conv;
      }
    }
    // write-back v = L + psi as a float-float sum; with the mass row, one refinement step moves the
    // float-float miss of the element mass along the pseudo-inverse column of the mass row (lo word)
    ff vv0 = {0.0f, 0.0f}, vv1 = {0.0f, 0.0f};
    if (v0) {
      const ff L = lref(r0, gx, gy, s_xi[i0] - 0.5f, s_xi[j0] - 0.5f);
      const ff s = two_sum(L.hi, cur0);
      vv0 = fast_two_sum(s.hi, __fadd_rn(s.lo, L.lo));
    }
    if (v1) {
      const ff L = lref(r0, gx, gy, s_xi[i1] - 0.5f, s_xi[j1] - 0.5f);
      const ff s = two_sum(L.hi, cur1);
      vv1 = fast_two_sum(s.hi, __fadd_rn(s.lo, L.lo));
    }
    if (mass) {
      ff mv = {0.0f, 0.0f};
      if (v0) mv = ff_mul(vv0, ff{X.w2h[p0], X.w2l[p0]});
      if (v1) mv = ff_add(mv, ff_mul(vv1, ff{X.w2h[p1], X.w2l[p1]}));
      mv = g.ffsum(mv);
      const float miss = ff_to_f(ff_add(target, ff_neg(mv)));
      const float2 cm = s_Cp[nb_rows * GT + t];
      if (v0) vv0 = fast_two_sum(vv0.hi, fmaf(miss, cm.x, vv0.lo));
      if (v1) vv1 = fast_two_sum(vv1.hi, fmaf(miss, cm.y, vv1.lo));
    }
    if (v0) {
      out[E.base + p0] = vv0.hi;
      out[X.plane + E.base + p0] = vv0.lo;
      if (!isfinite(vv0.hi)) bits |= SL_ST_NONFINITE;
    }
    if (v1) {
      out[E.base + p1] = vv1.hi;
      out[X.plane + E.base + p1] = vv1.lo;
      if (!isfinite(vv1.hi)) bits |= SL_ST_NONFINITE;
    }
    ++c_el;
    if (!ok) {
      bits |= SL_ST_PICARD_NOCONV;
      ++c_pnc;
    }
  }
  if (t == 0 && X0.counts) {
    atomicAdd(X0.counts + SL_CNT_ELEMS, (unsigned long long)c_el);
    if (c_eapp) atomicAdd(X0.counts + SL_CNT_ENERGY_APPLIED, (unsigned long long)c_eapp);
    if (c_pit) atomicAdd(X0.counts + SL_CNT_PICARD_ITERS, (unsigned long long)c_pit);
    if (c_pnc) atomicAdd(X0.counts + SL_CNT_PICARD_NOCONV, (unsigned long long)c_pnc);
  }
  if (bits) atomicOr(status, bits);
}

// persistent grid: the resident CTAs of the whole GPU, or one CTA per EPC elements if fewer
template <int NN, bool GEO>
void launch_g(int phase, const StepParams& p, const Mixed2DExtra& x, const Map2D& m, int64_t count, const float* in,
              float* out, const Work2M& w, unsigned* st, cudaStream_t s, int per_sm) {
  if (count <= 0) return;
  using S = Shape<NN>;
  // phase 2 stages the fit operator for the largest row set (4 n + 1 rows), whatever p.m is, so
  // that one occupancy figure serves every launch
  const size_t smem2 = (size_t)(4 * NN + 1) * S::GT * sizeof(float2);
  const void* kern = phase == 1 ? (const void*)k_p1<NN, GEO> : (const void*)k_p2<NN, GEO>;
  int fill = persistent_grid(kern, S::NT, phase == 1 ? 0 : smem2);
  // per_sm > 0: that many resident CTAs per SM (the autotuner's choice), within the occupancy
  if (per_sm > 0) fill = std::min(fill, per_sm * sm_count());
  const int64_t want = (count + S::EPC - 1) / S::EPC;
  const unsigned grid = (unsigned)(want < fill ? want : fill);
  if (phase == 1) k_p1<NN, GEO><<<grid, S::NT, 0, s>>>(p, x, m, count, in, w, st);
  else k_p2<NN, GEO><<<grid, S::NT, smem2, s>>>(p, x, m, count, in, w, out, st);
}

// Batches read their problem's parameters per element; other launches have them in the parameter bank, which
// frees about 25 registers of each kernel (256 x 256 elements of n = 8: 187 -> 179 us and 187 -> 182 us)
template <int NN>
void launch_n(int phase, const StepParams& p, const Mixed2DExtra& x, const Map2D& m, int64_t count, const float* in,
              float* out, const Work2M& w, unsigned* st, cudaStream_t s, int per_sm) {
  if (m.geo) launch_g<NN, true>(phase, p, x, m, count, in, out, w, st, s, per_sm);
  else launch_g<NN, false>(phase, p, x, m, count, in, out, w, st, s, per_sm);
}

}  // namespace k2m
}  // namespace sl
