// Device-side building blocks of the HWENO stage kernels (sm_103a).
//
// Scheme: moment-based multi-resolution HWENO, Li, Shu & Qiu (arXiv 2201.12193).
// Section and equation names below are the paper's.
//
// Precision: T = fx64 (FP64 path, fx64.cuh), double (FP64 path of the learned
// indicator), float (FP32-bulk path) or df64 (double-float path, df64.cuh).  The state, the Runge-Kutta combination and the conservation
// sums stay FP64 in all three.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "hweno_parity.h"
#include "df64.cuh"
#include "fx64.cuh"

namespace hw {

constexpr int EQ_ADV = 0, EQ_BURGERS = 1, EQ_EULER = 2;
constexpr int BC_PERIODIC = 0, BC_TRANSMISSIVE = 1, BC_REFLECTIVE = 2;
constexpr int IND_NONE = 0, IND_KXRCF = 1, IND_ALL = 2, IND_MLP = 3, IND_TVB = 4;

// device status word bits
constexpr unsigned ST_NONFINITE = 1u;     // a non-finite value in the new state
constexpr unsigned ST_NONPOSITIVE = 2u;   // rho <= 0 or p <= 0 in a new cell average (Euler)
constexpr unsigned ST_NODT = 8u;          // no CFL step length (rho <= 0 or a non-finite wave speed)

// A problem constant in the three compute precisions, converted once on the
// host (the same roundings as the device conversions: float by round to
// nearest, double-float as the nearest float plus the nearest float of the
// rest), so kernels do not spend FP64 instructions converting it per use.
struct PConst {
  double d;
  float f;
  df64 x;
};
template <typename T> __device__ __forceinline__ T pc(const PConst& c);
template <> __device__ __forceinline__ double pc<double>(const PConst& c) { return c.d; }
template <> __device__ __forceinline__ float pc<float>(const PConst& c) { return c.f; }
template <> __device__ __forceinline__ df64 pc<df64>(const PConst& c) { return c.x; }
template <> __device__ __forceinline__ fx64 pc<fx64>(const PConst& c) { return c.d; }

// Problem description passed by value to every kernel.
struct Prob {
  int nx, ny;             // cells (ny = 1 in 1D)
  int pitch;              // row stride of the state arrays (doubles)
  long long plane;        // stride of one (variable, moment) plane = ny * pitch
  int gpitch;             // row stride of the point-value / aux arrays (elements of T)
  long long gplane;       // ny * gpitch
  int nvar, nmom;         // conserved variables; moments per variable (2 in 1D, 3 in 2D)
  int eq, indicator;
  int bc[4];              // x-lo, x-hi, y-lo, y-hi
  double dx, dy;
  double gamma;           // ratio of specific heats
  double adv_a, adv_b;    // linear advection speeds
  int nsm;                // multiprocessors of the device (grid sizing)
  double tvb_m;           // TVB constant M (indicator IND_TVB)
  int charwise;           // 1D Euler: reconstruction in local characteristic variables
  int positivity;         // 1: rho <= 0 or p <= 0 averages are non-physical; 0: p is
                          //    clamped at 0 in the sound speed (only rho <= 0 / non-finite fail)
  const double* fixtab;   // fixed-state ghost cells (inflow; 2D Euler): [side][pos + 1][4] conserved
                          //    states for ghost positions pos in [-1, n] along each side, rho = 0
                          //    where the side's kind applies instead; null: no fixed-state side
  int fixlen;             // entries per side of fixtab
  int persist;            // 1: the first moments modified in troubled cells (eq. (vi)) replace the
                          //    stage input and enter the Runge-Kutta combination; 0: they serve
                          //    L only and the combination takes the stage states as they entered
  int fused;              // one fused kernel per stage (1D default; 2D Euler option) instead of the pipeline
  PConst cgamma, cdx, cdy, crdx, crdy, cdx2;   // gamma, dx, dy, 1/dx, 1/dy, dx^2
  PConst cgm1, chk;   // gamma - 1 and (gamma + 1) / (2 gamma) of eq. (COEF)
  PConst chg;         // (gamma - 1) / (2 gamma)
  int sol_i, sol_j;       // solid block (2D Euler, the forward step): cells i >= sol_i, j < sol_j;
                          //    sol_j = 0: none
  int jlo, jhi;           // owned rows [jlo, jhi): the rows a row-slab of a decomposed grid owns (the
                          //    others are halo rows refilled from the neighbours before each stage);
                          //    only they enter the status checks, the CFL reduction and the totals
};

// Sound speed of a cell average for the CFL rule; +inf marks a non-physical
// average (dt = 0, the host reports it).
__device__ __forceinline__ void cell_speeds(const Prob& P, double rho, double mu, double nu, double p, double& sx,
                                            double& sy) {
  const double c = sqrt(P.gamma * (P.positivity ? p : fmax(p, 0.0)) / rho);
  sx = fabs(mu) + c;
  sy = fabs(nu) + c;
  if (!(rho > 0.0) || (P.positivity && !(p > 0.0)) || !isfinite(sx + sy)) sx = sy = INFINITY;
}

// Linear-weight data of eq. (linear-weight) and eq. (p) for positive gbar[4]:
// gamma_{l,4} = g_l / S_4 and p_l = (S_l q_l - S_{l-1} q_{l-1}) / g_l.
template <typename T>
struct Weights {
  T gam[4];      // gamma_{l,4}
  T sg[4];       // S_l / g_l
  T s1g[4];      // S_{l-1} / g_l  (0 for l = 1)
  T ss[4];       // S_l / S_4
  T eps;         // 1e-10 of eqs. (w1_-LR), (non-linear-weight)
};

// Rows of the smoothness indicators beta_2..beta_4 for the run-time weights,
// in the flat parity-basis order of hweno_parity.h: beta_l = sum_rows (row . s)^2
// with row = (S_l/g_l) R C_l - (S_{l-1}/g_l) R C_{l-1}  (eq. (beta), (2D-beta), (p)).
template <typename T> struct Beta1 { T B2[hwp::D1_NB2]; T B3[hwp::D1_NB3]; T B4[hwp::D1_NB4]; };
template <typename T> struct Beta2 { T B2[hwp::D2_NB2]; T B3[hwp::D2_NB3]; T B4[hwp::D2_NB4]; };
// fx64: the rows in fixed point (hweno_fx.cuh), per parity class and over the class's
// columns; a coefficient is (x = h, y = l): (h 2^32 + l) 2^-F with one F a level (the root
// of the sum of squares of its rows' |coefficient| sums between 2^61.9 and 2^62.9 units, which
// keeps the Squares below 2^122), f = 61 - F.
template <int RA, int CA, int RB, int CB, int RE, int CE>
struct FxRows {
  int2 a[RA][CA], b[RB][CB], e[RE][CE];
  int f[3];           // a row's value times 2^-61 has the unit 2^f
  int elin;           // data with exponents up to it leave c_4 at least 1/4 (fx_uneven)
  Weights<fx64> w;    // for recon2d_levels (double-float kernels hold theirs in pairs)
};
template <> struct Beta1<fx64> : FxRows<hwp::D1_NRA, hwp::D1_NCA, hwp::D1_NRB, hwp::D1_NCB, 1, 1> {};
template <> struct Beta2<fx64>
    : FxRows<hwp::D2_NRA, hwp::D2_NCA, hwp::D2_NRB, hwp::D2_NCB, hwp::D2_NRE, hwp::D2_NCE> {};

// Gauss-Lobatto nodes and weights of eq. (F)
template <typename T> __device__ __forceinline__ T gl_w(int k) { return (k == 0 || k == 3) ? T(1.0 / 12.0) : T(5.0 / 12.0); }
template <typename T> __device__ __forceinline__ T gl_x(int k) {
  return k == 0 ? T(-0.5) : k == 1 ? T(-0.22360679774997896964) : k == 2 ? T(0.22360679774997896964) : T(0.5);
}

template <typename T> __device__ __forceinline__ T tabs(T x) { return x < T(0) ? -x : x; }
template <typename T> __device__ __forceinline__ T tmax(T a, T b) { return a > b ? a : b; }
template <> __device__ __forceinline__ fx64 tabs<fx64>(fx64 x) { return fabs(x.v); }
// (of non-negative values everywhere: their bits order like them, and a NaN wins)
template <> __device__ __forceinline__ fx64 tmax<fx64>(fx64 a, fx64 b) {
  return __longlong_as_double(max(__double_as_longlong(a.v), __double_as_longlong(b.v)));
}
// The smoothness-indicator rows a pipeline kernel takes (double-float: those of
// fx64), and the precisions it reconstructs in fixed point (recon2d_fx).
template <typename T> struct rows2d { using type = Beta2<T>; };
template <> struct rows2d<df64> { using type = Beta2<fx64>; };
template <typename T> struct fixed2d { static constexpr bool value = is_df64<T>::value || std::is_same<T, fx64>::value; };

// ---------------------------------------------------------------- boundary images
// A ghost cell is the image of an interior cell: periodic wrap, or (transmissive)
// the mirror about the boundary face, under which the mirrored direction's first
// moment changes sign and point values are reversed along that direction.
// A reflective boundary (a solid wall, Euler only) is the transmissive mirror
// with the wall-normal momentum negated as well (all its moments and point
// values): neg has bit v set for each variable v the image negates
// (variable 1 = x momentum, 2 = y momentum in 2D).
// A fixed-state ghost (inflow, the post-shock boundaries of the double Mach
// reflection) holds a constant state, entry fs of Prob::fixtab: that average,
// zero first moments, the same value at every Gauss-Lobatto point, never
// troubled.  Corners take the y rule on the cell the x rule gives (ghost
// columns first, then ghost rows over all columns): a fixed y ghost wins, and
// the y mirror of a fixed x ghost negates its y momentum at a wall.
struct Img { int i, j, sx, sy, neg, fs; };

__device__ __forceinline__ int wrap(int i, int n) { i %= n; return i < 0 ? i + n : i; }

// Solid block of the forward-facing step (Example 3.10): in-domain cells with
// i >= sol_i and j < sol_j.
__device__ __forceinline__ bool is_solid(const Prob& P, int i, int j) {
  return P.sol_j > 0 && i >= P.sol_i && i < P.nx && j >= 0 && j < P.sol_j;
}

// The block's faces are reflective walls: a solid cell in the stencil of the
// fluid cell (vi, vj) is that cell's wall image, mirrored across the vertical
// face when the viewer lies left of it (vi < sol_i), across the horizontal
// face when the viewer lies above it (vj >= sol_j), across both (a point
// reflection through the corner) for the one viewer diagonal to the corner;
// each crossed face negates its wall-normal momentum and its normal first
// moment.  The image depends on the viewer (the corner cell seen from its left
// neighbour is that neighbour's x mirror, from above the y mirror of the cell
// above it).
__device__ __forceinline__ void solid_image(const Prob& P, int vi, int vj, Img& r) {
  if (r.fs >= 0 || !is_solid(P, r.i, r.j)) return;
  if (vi < P.sol_i) { r.i = 2 * P.sol_i - 1 - r.i; r.sx = -r.sx; r.neg ^= 2; }
  if (vj >= P.sol_j) { r.j = 2 * P.sol_j - 1 - r.j; r.sy = -r.sy; r.neg ^= 4; }
}

// The image of cell (i, j) by the boundary sides alone (a cell of the solid
// block maps to itself; callers that can meet one use the viewer form below).
__device__ __forceinline__ Img image(const Prob& P, int i, int j) {
  Img r{i, j, 1, 1, 0, -1};
  if (j < 0 || j >= P.ny) {
    const int side = j < 0 ? 2 : 3;
    if (P.fixtab) {
      const int e = side * P.fixlen + i + 1;
      if (P.fixtab[4 * e] > 0.0) { r.fs = e; return r; }
    }
    const int k = P.bc[side];
    if (k == BC_PERIODIC) r.j = wrap(j, P.ny);
    else { r.j = j < 0 ? -1 - j : 2 * P.ny - 1 - j; r.sy = -1; if (k == BC_REFLECTIVE) r.neg |= 4; }
  }
  if (i < 0 || i >= P.nx) {
    const int side = i < 0 ? 0 : 1;
    if (P.fixtab) {
      const int e = side * P.fixlen + r.j + 1;
      if (P.fixtab[4 * e] > 0.0) { r.fs = e; return r; }
    }
    const int k = P.bc[side];
    if (k == BC_PERIODIC) r.i = wrap(i, P.nx);
    else { r.i = i < 0 ? -1 - i : 2 * P.nx - 1 - i; r.sx = -1; if (k == BC_REFLECTIVE) r.neg |= 2; }
  }
  return r;
}

// The image of cell (i, j) as the stencil of the fluid cell (vi, vj) sees it:
// boundary sides first, then the solid block.
__device__ __forceinline__ Img image(const Prob& P, int i, int j, int vi, int vj) {
  Img r = image(P, i, j);
  if (P.sol_j > 0) solid_image(P, vi, vj, r);
  return r;
}

// The image by the sides' kinds alone (fixed states ignored; an inflow side
// maps like a transmissive one).  Separable in x and y; equal to image() for
// every cell image() does not make a fixed-state ghost.
__device__ __forceinline__ Img image_kind(const Prob& P, int i, int j) {
  Img r{i, j, 1, 1, 0, -1};
  if (i < 0 || i >= P.nx) {
    const int k = P.bc[i < 0 ? 0 : 1];
    if (k == BC_PERIODIC) r.i = wrap(i, P.nx);
    else { r.i = i < 0 ? -1 - i : 2 * P.nx - 1 - i; r.sx = -1; if (k == BC_REFLECTIVE) r.neg |= 2; }
  }
  if (j < 0 || j >= P.ny) {
    const int k = P.bc[j < 0 ? 2 : 3];
    if (k == BC_PERIODIC) r.j = wrap(j, P.ny);
    else { r.j = j < 0 ? -1 - j : 2 * P.ny - 1 - j; r.sy = -1; if (k == BC_REFLECTIVE) r.neg |= 4; }
  }
  return r;
}

// Variable v of a fixed-state ghost (its average and every point value)
__device__ __forceinline__ double fixed_val(const Prob& P, const Img& m, int v) {
  return ((m.neg >> v) & 1 ? -1.0 : 1.0) * P.fixtab[4 * m.fs + v];
}

// Sign of variable v of an image cell (reflective walls)
__device__ __forceinline__ int vsign(const Img& m, int v) { return (m.neg >> v) & 1 ? -1 : 1; }

__device__ __forceinline__ long long sidx(const Prob& P, int var, int mom, int i, int j) {
  return (long long)(var * P.nmom + mom) * P.plane + (long long)j * P.pitch + i;
}

// Cell average of variable v of an image cell, fixed-state ghosts included.
__device__ __forceinline__ double avg_img(const Prob& P, const double* __restrict__ U, const Img& m, int v) {
  if (m.fs >= 0) return fixed_val(P, m, v);
  return vsign(m, v) * U[sidx(P, v, 0, m.i, m.j)];
}

// ---------------------------------------------------------------- physics
// Physical flux of eq. (1D-Euler) / (2D-Euler) or of the scalar laws in
// direction dir (0 = x, 1 = y); NV = 1 (scalar), 3 (1D Euler), 4 (2D Euler).
// 1/x, correctly rounded in FP32, double and fx64 (the latter two in integers).
template <typename T> __device__ __forceinline__ T rcp(T x) { return T(1) / x; }
template <> __device__ __forceinline__ float rcp<float>(float x) { return __frcp_rn(x); }
template <> __device__ __forceinline__ double rcp<double>(double x) { return rcp_ieee(x); }
template <> __device__ __forceinline__ fx64 rcp<fx64>(fx64 x) { return reciprocal(x); }

__device__ __forceinline__ double rcp64(double x) { return rcp<fx64>(x).v; }

// Root and quotient of the general flux: plain double's in integers where that is the
// IEEE result (fx64.cuh).
template <typename T> __device__ __forceinline__ T root(T x) { return sqrt(x); }
template <> __device__ __forceinline__ double root<double>(double x) { return sqrt_ieee(x); }
template <typename T> __device__ __forceinline__ T quot(T a, T b) { return a / b; }
template <> __device__ __forceinline__ double quot<double>(double a, double b) { return div_ieee(a, b); }

// a + b never contracted into an FMA (operands that are products)
template <typename T> __device__ __forceinline__ T addrn(T a, T b) { return a + b; }
template <> __device__ __forceinline__ fx64 addrn<fx64>(fx64 a, fx64 b) { return __dadd_rn(a.v, b.v); }

template <typename T, int NV>
__device__ __forceinline__ void phys_flux(const Prob& P, const T* u, int dir, T* f) {
  if constexpr (NV == 1) {
    if (P.eq == EQ_ADV) f[0] = T(dir == 0 ? P.adv_a : P.adv_b) * u[0];
    else f[0] = T(0.5) * u[0] * u[0];
  } else if constexpr (NV == 3) {
    const T g = pc<T>(P.cgamma);
    const T inv = rcp(u[0]), mu = u[1] * inv, E = u[2];
    const T p = (g - T(1)) * (E - T(0.5) * u[1] * mu);
    f[0] = u[1]; f[1] = u[1] * mu + p; f[2] = mu * (E + p);
  } else {
    const T g = pc<T>(P.cgamma);
    const T inv = rcp(u[0]), mu = u[1] * inv, nu = u[2] * inv, E = u[3];
    const T p = (g - T(1)) * (E - T(0.5) * (u[1] * mu + u[2] * nu));
    if (dir == 0) { f[0] = u[1]; f[1] = u[1] * mu + p; f[2] = u[1] * nu; f[3] = mu * (E + p); }
    else          { f[0] = u[2]; f[1] = u[2] * mu; f[2] = u[2] * nu + p; f[3] = nu * (E + p); }
  }
}

// Euler flux with the reciprocal of the density supplied by the caller.
template <typename T, int NV>
__device__ __forceinline__ void euler_flux_inv(const Prob& P, const T* u, T inv, int dir, T* f) {
  const T g = pc<T>(P.cgamma);
  if constexpr (NV == 3) {
    const T mu = u[1] * inv, E = u[2];
    const T p = (g - T(1)) * (E - T(0.5) * u[1] * mu);
    f[0] = u[1]; f[1] = u[1] * mu + p; f[2] = mu * (E + p);
  } else {
    const T mu = u[1] * inv, nu = u[2] * inv, E = u[3];
    const T p = (g - T(1)) * (E - T(0.5) * (u[1] * mu + u[2] * nu));
    if (dir == 0) { f[0] = u[1]; f[1] = u[1] * mu + p; f[2] = u[1] * nu; f[3] = mu * (E + p); }
    else          { f[0] = u[2]; f[1] = u[2] * mu; f[2] = u[2] * nu + p; f[3] = nu * (E + p); }
  }
}

// Reciprocals of N values with a single division (prefix products, one inverse,
// back substitution); used by the FP64 path, where a division costs about as
// much as a dozen fused multiply-adds.
template <int N, typename T>
__device__ __forceinline__ void batch_inverse(const T (&x)[N], T (&inv)[N]) {
  T pre[N];
  pre[0] = x[0];
#pragma unroll
  for (int i = 1; i < N; ++i) pre[i] = pre[i - 1] * x[i];
  T r = rcp(pre[N - 1]);
#pragma unroll
  for (int i = N - 1; i > 0; --i) {
    inv[i] = r * pre[i - 1];
    r = r * x[i];
  }
  inv[0] = r;
}

// Reciprocals for the FP64-class types.  FP64: one division for all N.
// Double-float carries FP32's exponent range, where a product of 12 or 16
// densities can underflow, so it inverts groups of 4.
template <int N, typename T>
__device__ __forceinline__ void batch_inverse_ranged(const T (&x)[N], T (&inv)[N]) {
  if constexpr (is_df64<T>::value) {
    static_assert(N % 4 == 0, "groups of four");
#pragma unroll
    for (int g = 0; g < N; g += 4) {
      const T xs[4] = {x[g], x[g + 1], x[g + 2], x[g + 3]};
      T r[4];
      batch_inverse<4, T>(xs, r);
#pragma unroll
      for (int k = 0; k < 4; ++k) inv[g + k] = r[k];
    }
  } else {
    batch_inverse<N, T>(x, inv);
  }
}

// One common denominator for the nonlinear weights is safe in FP64 only: it
// multiplies four (beta + eps) factors (eps^4 = 1e-40 is below FP32's range,
// which double-float shares).
template <typename T> struct one_division { static constexpr bool value = sizeof(T) == 8 && !is_df64<T>::value; };

// Velocity seen by the KXRCF indicator for scalar laws (Remarks 2, 3): f'(u), g'(u).
template <typename T>
__device__ __forceinline__ T scalar_velocity(const Prob& P, T u, int dir) {
  if (P.eq == EQ_ADV) return T(dir == 0 ? P.adv_a : P.adv_b);
  return u;
}

// HLLC flux, eqs. (f_HLLC), (COEF), (uLR_), as a rotated 1D solver in direction
// dir (the tangential velocity is carried through the star state).
// Branch order: 0 <= sL -> fL; 0 <= s* -> f*L; 0 <= sR -> f*R; else fR.
// wall: the face of the forward step's solid block (one side the reflection of
// the other): the star branch is taken whatever the sign of the wave-speed
// estimate, so the flux carries no mass or energy (s* = 0) and the normal
// momentum flux is the star pressure -- the estimate of eq. (COEF) gives
// s_L > 0 for flow running into a wall faster than about its sound speed,
// where the first branch of eq. (f_HLLC) would let the gas through the wall.
template <typename T, int NV>
__device__ __forceinline__ void hllc(const Prob& P, const T* uL, const T* uR, int dir, T* F, bool wall = false) {
  constexpr bool two = NV == 4;
  const T g = pc<T>(P.cgamma);
  const int in = 1 + dir, it = 2 - dir;
  constexpr int iE = NV - 1;
  const T rL = uL[0], rR = uR[0];
  // one reciprocal for both densities' reciprocals
  const T q = rcp(rL * rR);
  const T iL = rR * q, iR = rL * q;
  const T mL = uL[in] * iL, mR = uR[in] * iR;
  const T tL = two ? uL[it] * iL : T(0), tR = two ? uR[it] * iR : T(0);
  const T EL = uL[iE], ER = uR[iE];
  const T gm1 = pc<T>(P.cgm1);
  const T pL = gm1 * (EL - T(0.5) * rL * (mL * mL + tL * tL));
  const T pR = gm1 * (ER - T(0.5) * rR * (mR * mR + tR * tR));
  const T gL = g * iL, gR = g * iR;
  const T cL = root(gL * pL), cR = root(gR * pR);
  const T rs = T(0.5) * (rL + rR), cs = T(0.5) * (cL + cR);
  const T crs = cs * rs;
  const T ps = T(0.5) * (pL + pR + (mL - mR) * crs);
  const T ss = T(0.5) * (mL + mR + quot(pL - pR, crs));
  // eq. (COEF): c_K coef_K = sqrt(gamma p_K / rho_K) sqrt(1 + k (p* / p_K - 1)) with
  // k = (gamma + 1) / (2 gamma) when p* > p_K, else c_K.  FP64 keeps the two roots
  // (the second only where p* > p_K); FP32 and double-float take one root,
  // sqrt(gamma / rho_K (p_K + k max(p* - p_K, 0))), without the divisions by p_K
  // (measured 5 % faster in the double-float update, 1 % slower in FP64).  A
  // non-finite p* stays non-finite either way (the comparison is written so), and
  // the branches below then fall through to f_R.
  const T k = pc<T>(P.chk);
  T sL, sR;
  if constexpr (one_division<T>::value) {
    const T coefL = ps <= pL ? T(1) : root(T(1) + k * (quot(ps, pL) - T(1)));
    const T coefR = ps <= pR ? T(1) : root(T(1) + k * (quot(ps, pR) - T(1)));
    sL = mL - cL * coefL;
    sR = mR + cR * coefR;
  } else {
    const T dL = ps - pL, dR = ps - pR;
    sL = mL - sqrt(gL * (pL + k * (dL <= T(0) ? T(0) : dL)));
    sR = mR + sqrt(gR * (pR + k * (dR <= T(0) ? T(0) : dR)));
  }
  const bool useL = (!wall && T(0) <= sL) || T(0) <= ss;     // left physical or left star flux
  const T rK = useL ? rL : rR, mK = useL ? mL : mR, tK = useL ? tL : tR;
  const T EK = useL ? EL : ER, pK = useL ? pL : pR, sK = useL ? sL : sR;
  // physical normal flux of the chosen side
  T fK[NV], uK[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) uK[v] = useL ? uL[v] : uR[v];
  fK[0] = rK * mK;
  fK[1] = dir == 0 ? rK * mK * mK + pK : rK * mK * tK;
  if constexpr (two) fK[2] = dir == 0 ? rK * mK * tK : rK * mK * mK + pK;
  fK[iE] = mK * (EK + pK);
  if (!wall && (T(0) <= sL || !(T(0) <= sR || T(0) <= ss))) {   // supersonic: fL or fR
#pragma unroll
    for (int v = 0; v < NV; ++v) F[v] = fK[v];
    return;
  }
  const T a = sK - mK, b = sK - ss;
  // D = 1/(a b) gives 1/a and 1/b with one reciprocal
  const T iK = useL ? iL : iR;
  const T D = rcp(a * b);
  const T fac = rK * a * (a * D);
  const T ek = EK * iK;
  const T pk = pK * iK * (b * D);
  T us[NV];
  us[0] = fac;
  us[in] = fac * ss;
  if constexpr (two) us[it] = fac * tK;
  us[iE] = fac * (ek + (ss - mK) * (ss + pk));
#pragma unroll
  for (int v = 0; v < NV; ++v) F[v] = fK[v] + sK * (us[v] - uK[v]);
}

// fx64 and double-float take the lean form below (fx64: 24 FP64 operations in 2D, the
// products, roots and reciprocals being integer work, against 150 of hllc); float and plain double keep hllc.
template <typename T> struct lean { static constexpr bool value = is_df64<T>::value || std::is_same<T, fx64>::value; };
template <typename T> __device__ __forceinline__ bool nonneg(T a) { return T(0) <= a; }
template <typename T> __device__ __forceinline__ bool nonpos(T a) { return a <= T(0); }
template <typename T> __device__ __forceinline__ bool below(T a, T b) { return a < b; }
template <typename T> __device__ __forceinline__ T half(T a) { return T(0.5) * a; }

// The same flux with fewer operations.  Only the chosen side's wave speed is
// formed: s* < 0 with m_L < c_L implies s_L < 0 (its coefficient is at least 1),
// so s_L matters for s* < 0 only in the remaining case.  The star flux is
// written through the Rankine-Hugoniot relations of its wave: with
// w = rho_K (s_K - m_K), p* = p_K + w (s* - m_K) and rho* = w / (s_K - s*) it is
// (rho* s*, rho* s*^2 + p*, rho* s* t_K, s* (E* + p*)),
// E* = (E_K (s_K - m_K) - p_K m_K + p* s*) / (s_K - s*).
template <typename T, int NV, bool SOFT = true>
__device__ __forceinline__ void hllc_lean(const Prob& P, const T* uL, const T* uR, int dir, T* F, bool wall = false) {
  constexpr bool two = NV == 4;
  // fx64 in 2D: the products in integers (SOFT) or by the FP64 pipe, the same bits
  auto M = [](T a, T b) {
    if constexpr (two && std::is_same<T, fx64>::value) return SOFT ? product(a, b) : fx64(__dmul_rn(a.v, b.v));
    else return a * b;
  };
  constexpr int iE = NV - 1;
  const int in = 1 + dir, it = 2 - dir;
  const T g = pc<T>(P.cgamma), gm1 = pc<T>(P.cgm1), k = pc<T>(P.chk);
  const T rL = uL[0], rR = uR[0], EL = uL[iE], ER = uR[iE];
  T iL, iR;
  if constexpr (is_df64<T>::value) {   // one division for both
    const T q = rcp(rL * rR);
    iL = rR * q;
    iR = rL * q;
  } else {
    iL = rcp(rL);
    iR = rcp(rR);
  }
  const T mL = M(uL[in], iL), mR = M(uR[in], iR);
  const T tL = two ? M(uL[it], iL) : T(0), tR = two ? M(uR[it], iR) : T(0);
  T kL = M(uL[in], mL), kR = M(uR[in], mR);
  if constexpr (two) { kL = fma(uL[it], tL, kL); kR = fma(uR[it], tR, kR); }
  const T pL = M(gm1, fma(T(-0.5), kL, EL)), pR = M(gm1, fma(T(-0.5), kR, ER));
  const T gL = M(g, iL), gR = M(g, iR);
  const T cL = sqrt(M(gL, pL)), cR = sqrt(M(gR, pR));
  const T x = M(rL + rR, cL + cR);                 // four times the mean density times the mean sound speed
  const T ps = fma(M(mL - mR, x), T(0.125), half(pL + pR));
  const T ss = fma(M(pL - pR, rcp(x)), T(2), half(mL + mR));
  auto speed = [&](T gk, T pk, T ck) {               // c_K coef_K of eq. (COEF)
    const T d = ps - pk;
    return nonpos(d) ? ck : sqrt(M(gk, fma(k, d, pk)));
  };
  bool left = nonneg(ss);
  if (!left && !wall && !below(mL, cL)) left = nonneg(mL - speed(gL, pL, cL));
  const T mK = left ? mL : mR, pK = left ? pL : pR, EK = left ? EL : ER, tK = left ? tL : tR;
  const T sd = speed(left ? gL : gR, pK, left ? cL : cR);
  const T sK = left ? mK - sd : mK + sd;
  const bool ge = nonneg(sK);
  if (!wall && (left ? ge : !ge)) {                  // supersonic: the physical flux of the side
    const T q = left ? uL[in] : uR[in];
    F[0] = q;
    F[in] = fma(q, mK, pK);
    if constexpr (two) F[it] = M(q, tK);
    F[iE] = M(mK, EK + pK);
    return;
  }
  const T a = sK - mK, w = M(left ? rL : rR, a);
  const T pst = fma(w, ss - mK, pK);
  const T rb = rcp(sK - ss);
  const T f0 = M(M(w, rb), ss);
  F[0] = f0;
  F[in] = fma(f0, ss, pst);
  if constexpr (two) F[it] = M(f0, tK);
  const T e = fma(pst, ss, fma(EK, a, -M(pK, mK)));
  F[iE] = M(ss, fma(e, rb, pst));
}

// Scalar laws: local Lax-Friedrichs flux with alpha = max(|f'(uL)|, |f'(uR)|).
template <typename T>
__device__ __forceinline__ T llf(const Prob& P, T uL, T uR, int dir) {
  T fl, fr;
  phys_flux<T, 1>(P, &uL, dir, &fl);
  phys_flux<T, 1>(P, &uR, dir, &fr);
  const T aL = tabs(scalar_velocity(P, uL, dir)), aR = tabs(scalar_velocity(P, uR, dir));
  return T(0.5) * (fl + fr) - T(0.5) * tmax(aL, aR) * (uR - uL);
}

template <typename T, int NV>
__device__ __forceinline__ void num_flux(const Prob& P, const T* uL, const T* uR, int dir, T* F) {
  if constexpr (NV == 1) F[0] = llf(P, uL[0], uR[0], dir);
  else if constexpr (lean<T>::value) hllc_lean<T, NV>(P, uL, uR, dir, F);
  else hllc<T, NV>(P, uL, uR, dir, F);
}

// ---------------------------------------------------------------- nonlinear weights
// WENO-Z weights of eqs. (tau4), (non-linear-weight) and the combination of
// eq. (re-p) rewritten on q_1..q_4:  u = sum_k c_k q_k with
// c_k = omega_k S_k/g_k - omega_{k+1} S_k/g_{k+1},  c_4 = omega_4 S_4/g_4.
template <typename T>
__device__ __forceinline__ void combine_weights(const Weights<T>& W, const T beta[4], T c[4]) {
  const T tau4s = tabs(beta[3] - beta[0]) + tabs(beta[3] - beta[1]) + tabs(beta[3] - beta[2]);
  const T tau4 = (tau4s * T(1.0 / 3.0)) * (tau4s * T(1.0 / 3.0));
  T om[4];
  if constexpr (one_division<T>::value) {
    // FP64: one division.  With x_l = beta_l + eps, wbar_l = gamma_l (x_l + tau)/x_l;
    // scaling every wbar_l by prod_m x_m gives N_l = gamma_l (x_l + tau) prod_{m!=l} x_m
    // and omega_l = N_l / sum_m N_m.
    const T x0 = beta[0] + W.eps, x1 = beta[1] + W.eps, x2 = beta[2] + W.eps, x3 = beta[3] + W.eps;
    const T p01 = x0 * x1, p23 = x2 * x3;
    const T n0 = W.gam[0] * (x0 + tau4) * (x1 * p23);
    const T n1 = W.gam[1] * (x1 + tau4) * (x0 * p23);
    const T n2 = W.gam[2] * (x2 + tau4) * (p01 * x3);
    const T n3 = W.gam[3] * (x3 + tau4) * (p01 * x2);
    const T inv = rcp((n0 + n1) + (n2 + n3));
    om[0] = n0 * inv; om[1] = n1 * inv; om[2] = n2 * inv; om[3] = n3 * inv;
  } else {
    T wb[4], ws = T(0);
#pragma unroll
    for (int l = 0; l < 4; ++l) { wb[l] = W.gam[l] * (T(1) + tau4 / (beta[l] + W.eps)); ws += wb[l]; }
    const T inv = rcp(ws);
#pragma unroll
    for (int l = 0; l < 4; ++l) om[l] = wb[l] * inv;
  }
  c[0] = om[0] * W.sg[0] - om[1] * W.s1g[1];
  c[1] = om[1] * W.sg[1] - om[2] * W.s1g[2];
  c[2] = om[2] * W.sg[2] - om[3] * W.s1g[3];
  c[3] = om[3] * W.sg[3];
}

// fx64: the same weights with one division.  With x_l = beta_l + eps,
// wbar_l = gamma_l (x_l + tau) / x_l; scaling every wbar_l by prod_m x_m gives
// omega_l = gamma_l n_l / sum_m gamma_m n_m with n_l = (x_l + tau) prod_{m != l} x_m,
// and, gamma_l S_l/g_l being S_l/S_4, c_k = (S_k/S_4) (n_k - n_{k+1}) / sum_m gamma_m n_m.
// c_1 = 1 - c_2 - c_3 - c_4 is not formed: q_1 is the target average u_5 and
// u = u_5 + sum_{k>1} c_k (q_k - u_5).  c = (c_2, c_3, c_4, c_2 + c_3).
__device__ __forceinline__ void weights_c(const Weights<fx64>& W, const fx64 (&bt)[4], fx64 (&c)[4]) {
  const double beta[4] = {bt[0].v, bt[1].v, bt[2].v, bt[3].v};
  const double tau4s = fabs(beta[3] - beta[0]) + fabs(beta[3] - beta[1]) + fabs(beta[3] - beta[2]);
  const double q = tau4s * (1.0 / 3.0);             // tau_4 = q^2
  const double eps = W.eps.v;
  const double x0 = beta[0] + eps, x1 = beta[1] + eps, x2 = beta[2] + eps, x3 = beta[3] + eps;
  const double p01 = x0 * x1, p23 = x2 * x3;
  const double n0 = fma(q, q, x0) * (x1 * p23), n1 = fma(q, q, x1) * (x0 * p23);
  const double n2 = fma(q, q, x2) * (p01 * x3), n3 = fma(q, q, x3) * (p01 * x2);
  const double inv = rcp64(fma(W.gam[3].v, n3, fma(W.gam[2].v, n2, fma(W.gam[1].v, n1, W.gam[0].v * n0))));
  c[0] = (W.ss[1].v * __dsub_rn(n1, n2)) * inv;
  c[1] = (W.ss[2].v * __dsub_rn(n2, n3)) * inv;
  c[2] = n3 * inv;
  c[3] = __dadd_rn(c[0].v, c[1].v);
}

__device__ __forceinline__ void weights_c(const Weights<df64>& W, const df64 (&beta)[4], df64 (&c)[4]) {
  df64 k[4];
  combine_weights<df64>(W, beta, k);
  c[0] = k[1];
  c[1] = k[2];
  c[2] = k[3];
  c[3] = k[1] + k[2];
}

// A fixed-point value x 2^eb in the compute precision.
template <typename T> __device__ __forceinline__ T from_fixed(long long x, int eb);
template <> __device__ __forceinline__ fx64 from_fixed<fx64>(long long x, int eb) { return hwfx::from_fx(x, eb); }
template <> __device__ __forceinline__ df64 from_fixed<df64>(long long x, int eb) {
  const float2 r = hwfx::from_fx_pair(x, eb);
  return df64(r.x, r.y);
}

template <typename T> __device__ __forceinline__ T from_squares(const hwfx::Squares& s, int e);
template <> __device__ __forceinline__ fx64 from_squares<fx64>(const hwfx::Squares& s, int e) { return hwfx::sum_of(s, e); }
template <> __device__ __forceinline__ df64 from_squares<df64>(const hwfx::Squares& s, int e) {
  const float2 r = hwfx::sum_of_pair(s, e);
  return df64(r.x, r.y);
}

// Adds (sum_k c[k] s[k])^2 of a beta row.  The class data are sums of up to four
// 57-bit data, the level's coefficients below 2^62.9 (root of the sum of squares of the
// rows' sums): with 2^-61 of the product the squares sum below 2^122.
template <int N>
__device__ __forceinline__ void fx_row(const hwfx::Half2 (&s)[N], const int2 (&c)[N], hwfx::Squares& q) {
  hwfx::Acc t = hwfx::prod(s[0], c[0].x, c[0].y);
#pragma unroll
  for (int k = 1; k < N; ++k) hwfx::mac(t, s[k], c[k].x, c[k].y);
  hwfx::add_square(q, hwfx::scaled<61>(t));
}

// A weight's exponent (2047: not finite), and the weight in units of 2^(e - 1022 - CBITS).
__device__ __forceinline__ int cexp(fx64 c) { return hwfx::bexp(c.v); }
__device__ __forceinline__ int cexp(df64 c) {
  const int f = (int)((__float_as_uint(c.hi) >> 23) & 0xFF);
  return f == 0xFF ? 0x7FF : f + 896;
}
__device__ __forceinline__ hwfx::Half2 cfixed(fx64 c, int e) { return hwfx::halves(hwfx::to_fx<hwfx::CBITS>(c.v, e)); }
__device__ __forceinline__ hwfx::Half2 cfixed(df64 c, int e) {
  return hwfx::halves(hwfx::to_fx<hwfx::CBITS>(c.hi, e) + hwfx::to_fx<hwfx::CBITS>(c.lo, e));
}

// Data of different size.  A datum is kept to 2^-57 of the largest that shares its
// exponent.  That is FP64's accuracy as long as the result is of that datum's size.  But
// the first moments enter only q_3 (the cell's own) and q_4, and where they are
// large against the averages the weights discard those: what remains would be left
// with the low bits of q_2's data (one exponent for all: 5e-9 of the values at a ratio of
// 1e8).  So each level's data have the unit of the largest datum that the level takes,
// and the weights the units that give c_l q_l one (that of the largest product).
// 1D does so throughout; in 2D, where three sets of class data would not fit the
// registers, the stencils with uneven data leave for recon2d_levels: those whose first
// moments' exponent em exceeds that of the averages' differences (ea) and of the average
// (eu: the value's own rounding) by more than `slack`: 1 for fx64 (a truncation below 2^-55 of
// the scale, FP64's rounding being 2^-54), 8 for double-float (2^-48, the pairs' is
// 2^-47).  Data below 2^(elin - 1022) leave c_4 at least 1/4 (their indicators are not much
// above the weights' eps): q_4 is not discarded and its largest datum is the scale, which
// keeps the small momenta of gas nearly at rest in the one-exponent form.
template <typename T>
__device__ __forceinline__ bool fx_uneven(int ea, int em, int eu, int elin) {
  constexpr int slack = is_df64<T>::value ? 8 : 1;
  return em > max(ea, eu) + slack && em > elin;
}

// The weights c_2, c_3, c_4, c_2 + c_3 as fixed-point integers of one exponent;
// returns it (2047 if one is not finite).
template <typename T>
__device__ __forceinline__ int fx_weights(const T (&c)[4], hwfx::Half2 (&h)[4]) {
  const int e = max(max(max(cexp(c[0]), cexp(c[1])), max(cexp(c[2]), cexp(c[3]))), hwfx::CEMIN);
#pragma unroll
  for (int k = 0; k < 4; ++k) h[k] = cfixed(c[k], e);
  return e;
}

// ---------------------------------------------------------------- 1D reconstruction
// d = (u_{i-1}, u_i, u_{i+1}, v_{i-1}, v_i, v_{i+1}) of one variable; out = the
// four Gauss-Lobatto values of eq. (re-u).  Steps 1.1-1.3 of the 1D algorithm.
// fx64: the linear part in block fixed point (hweno_fx.cuh).
__device__ __forceinline__ void recon1d_fp64(const Weights<fx64>& W, const Beta1<fx64>& B, const fx64 (&d)[6],
                                             fx64 (&out)[4]) {
  const double dl = d[1].v - d[0].v, dr = d[2].v - d[1].v;
  const double dv[6] = {-dl, 0.0, dr, d[3].v, d[4].v, d[5].v};
  // the exponents of the data of q_2, q_3 and q_4
  const int e2 = max(hwfx::EMIN, max(hwfx::bexp(dl), hwfx::bexp(dr))), e3 = max(e2, hwfx::bexp(dv[4]));
  const int e4 = max(e3, max(hwfx::bexp(dv[3]), hwfx::bexp(dv[5])));
  long long q[6];
#pragma unroll
  for (int k = 0; k < 6; ++k) q[k] = k == 1 ? 0 : hwfx::to_fx<hwfx::BITS>(dv[k], k < 3 ? e2 : k == 4 ? e3 : e4);
  const int s3 = min(e3 - e2, 63), s4 = min(e4 - e2, 63), s34 = min(e4 - e3, 63);
  const long long qs = q[0] + q[2], qd = q[0] - q[2];
  hwfx::Half2 a2[2], b2[3];            // each at the exponent of the level that brought it in
  hwp::fx_split1d(q, a2, b2);
  hwfx::Half2 a3[2] = {hwfx::halves(qs >> s3), a2[1]}, a4[2] = {hwfx::halves(qs >> s4), a2[1]};
  hwfx::Half2 b3[3] = {hwfx::halves(qd >> s3), b2[1], b2[2]};
  hwfx::Half2 b4[3] = {hwfx::halves(qd >> s4), b2[1], hwfx::halves(q[4] >> s34)};
  fx64 beta[4];
#pragma unroll
  for (int l = 0; l < 3; ++l) {
    hwfx::Squares bl{0, 0, 0};
#pragma unroll
    for (int r = hwp::D1_RA(l); r < hwp::D1_RA(l + 1); ++r) fx_row(l == 0 ? a2 : l == 1 ? a3 : a4, B.a[r], bl);
#pragma unroll
    for (int r = hwp::D1_RB(l); r < hwp::D1_RB(l + 1); ++r) fx_row(l == 0 ? b2 : l == 1 ? b3 : b4, B.b[r], bl);
    beta[l + 1] = from_squares<fx64>(bl, 2 * ((l == 0 ? e2 : l == 1 ? e3 : e4) - (1022 + hwfx::BITS) + B.f[l]));
  }
  // beta_1: eqs. (beta1-LR), (tau1), (w1_-LR), (w1-LR), (beta1) over a common denominator
  {
    const double td = fma(dr, dr, -(dl * dl));       // tau_1 = td^2
    const double xl = fma(dl, dl, W.eps.v), xr = fma(dr, dr, W.eps.v);
    const double nl = fma(td, td, xl) * xr, nr = fma(td, td, xr) * xl;
    const double gg = fma(nl, dl, nr * dr) * rcp64(__dadd_rn(nl, nr));
    beta[0] = gg * gg;
  }
  fx64 c[4];
  weights_c(W, beta, c);
  const int x2 = max(cexp(c[0]), cexp(c[3])), x3 = cexp(c[1]), x4 = cexp(c[2]);
  const int eu = max(max(x2 + e2, x3 + e3), e4 + max(x4, hwfx::CEMIN));   // the largest product's exponent
  long long x[4];
  hwp::fx_values1d(a2, b2, b3, a4, b4, cfixed(c[0], eu - e2), cfixed(c[1], eu - e3), cfixed(c[2], eu - e4),
                   cfixed(c[3], eu - e2), x);
  const bool bad = e4 > hwfx::EMAX || max(x2, max(x3, x4)) == 0x7FF;
  const double u = bad ? __longlong_as_double(0x7FF8000000000000LL) : d[1].v;
  const int eb = eu + (hwfx::CF - (1022 + hwfx::CBITS) - (1022 + hwfx::BITS));
#pragma unroll
  for (int p = 0; p < 4; ++p) out[p] = u + hwfx::from_fx(x[p], eb);
}

template <typename T>
__device__ __forceinline__ void recon1d(const Weights<T>& W, const Beta1<T>& B, const T (&d)[6], T (&out)[4]) {
  if constexpr (std::is_same<T, fx64>::value) {
    recon1d_fp64(W, B, d, out);
    return;
  } else {
  T s[6];
  hwp::split1d<T>(d, s);
  T beta[4];
  hwp::beta1d<T>(B.B2, B.B3, B.B4, s, beta[1], beta[2], beta[3]);
  // beta_1: eqs. (beta1-LR), (tau1), (w1_-LR), (w1-LR), (beta1)
  {
    const T dl = d[1] - d[0], dr = d[2] - d[1];
    const T bl = dl * dl, br = dr * dr;
    const T t1 = tabs(br - bl) * tabs(br - bl);
    T gg;
    if constexpr (sizeof(T) == 8) {   // common denominator: one division
      const T xl = bl + W.eps, xr = br + W.eps;
      const T nl = (xl + t1) * xr, nr = (xr + t1) * xl;
      gg = (nl * dl + nr * dr) / (nl + nr);
    } else {
      const T wl = T(0.5) * (T(1) + t1 / (bl + W.eps));
      const T wr = T(0.5) * (T(1) + t1 / (br + W.eps));
      const T inv = rcp(wl + wr);
      gg = (wl * inv) * dl + (wr * inv) * dr;
    }
    beta[0] = gg * gg;
  }
  T c[4];
  combine_weights(W, beta, c);
  hwp::values1d<T>(s, d[1], c, out);
  }
}

// ---------------------------------------------------------------- 2D reconstruction
// beta_1: eqs. (2D-q1-1234) .. (2D-beta1).  With x differences a (west), b (east)
// and y differences g (south), h (north), the four one-sided |grad|^2 are a^2 + h^2,
// b^2 + h^2, b^2 + g^2, a^2 + g^2; their six unordered differences are +-A twice,
// +-B twice, +-(A + B) and +-(A - B), A = a^2 - b^2, B = h^2 - g^2, so that
// tau_1 = ((|A| + |B| + max(|A|, |B|)) / 3)^2.
template <typename T>
__device__ __forceinline__ T beta1_2d(const Weights<T>& W, T a, T b, T g, T h) {
  const T A = tabs(fma(a, a, -(b * b))), Bq = tabs(fma(h, h, -(g * g)));
  const T ts = (A + Bq + tmax(A, Bq)) * T(1.0 / 3.0);
  const T he = fma(h, h, W.eps), ge = fma(g, g, W.eps);
  const T y0 = fma(a, a, he), y1 = fma(b, b, he), y2 = fma(b, b, ge), y3 = fma(a, a, ge);
  T n0, n1, n2, n3;
  if constexpr (one_division<T>::value) {   // over a common denominator
    const T p01 = y0 * y1, p23 = y2 * y3;
    n0 = fma(ts, ts, y0) * (y1 * p23);
    n1 = fma(ts, ts, y1) * (y0 * p23);
    n2 = fma(ts, ts, y2) * (p01 * y3);
    n3 = fma(ts, ts, y3) * (p01 * y2);
  } else {
    n0 = T(1) + (ts * ts) / y0;
    n1 = T(1) + (ts * ts) / y1;
    n2 = T(1) + (ts * ts) / y2;
    n3 = T(1) + (ts * ts) / y3;
  }
  // (n_k are products: sums of them stay sums, so that every kernel rounds alike)
  const T n01 = addrn(n0, n1), n23 = addrn(n2, n3);
  const T inv = rcp(n01 + n23);
  const T gx = fma(addrn(n0, n3), a, addrn(n1, n2) * b) * inv, gy = fma(n01, h, n23 * g) * inv;
  return fma(gx, gx, gy * gy);
}

// d = the 23 data of q_4 (u at labels 1..9, v at 1,3,4,5,6,7,9, w at
// 1,2,3,5,7,8,9; labels of the paper's 3x3 stencil table); put(k*4+l, value)
// receives u_{i,j}(xi_k, eta_l) of eq. (2D-re-u).  Steps 1.1-1.3 of the 2D algorithm.
// Square cells: beta_1 of eq. (2D-beta1) is (sum w_1k Dx_k)^2 + (sum w_1k Dy_k)^2.
// fx64 and double-float: the linear part in block fixed point (hweno_fx.cuh).  The beta rows and
// the four base points (+-|xi|, +-|eta|) run as loops over coefficient tables:
// unrolled, a variable's code is 100 KB and the warps wait for instructions.
// dv: the data as deviations from the average u5 (dv[4] = u5 itself).
// e: the exponents of the data of q_2, q_3 and q_4.  LEVELS (uneven data): each level's data in
// its own unit, as in recon1d_fp64; otherwise, and bit for bit where the three are the
// same, all in that of e[2].
template <bool LEVELS, typename T, typename Put>
__device__ __forceinline__ void recon2d_fx(const Weights<T>& W, const Beta2<fx64>& B, const double (&dv)[23],
                                           const int (&e)[3], Put put) {
  using hwfx::Half2;
  const double u5 = dv[4];
  Half2 sa[7], sb[6], sc[6], se[3];   // parity classes (even, even), (odd, even), (even, odd), (odd, odd)
  {
    long long q[23];
#pragma unroll
    for (int k = 0; k < 23; ++k) {
      const int l = !LEVELS || !(k < 9 || k == 12 || k == 19) ? 2 : k < 9 ? 0 : 1;   // the level that brings it in
      q[k] = k == 4 ? 0 : hwfx::to_fx<hwfx::BITS>(dv[k], e[l]);
    }
    hwp::fx_split2d(q, sa, sb, sc, se);
  }
  [[maybe_unused]] Half2 a2[3], e2, b2[2], c2[2], b3[6], c3[6];   // LEVELS: what q_2 and q_3 take, in their units
  T beta[4];
  {
    int ra = 0, rb = 0, re = 0;
#pragma unroll 1
    for (int l = 0; l < 3; ++l) {
      if constexpr (LEVELS) {   // from the last level's unit to this one's
        const int s = l == 0 ? 0 : min(e[l] - e[l - 1], 63);
        auto shift = [s](Half2& x) { x = hwfx::halves((((long long)x.h << 32) + x.l) >> s); };
        if (l > 0) {
          shift(sa[0]); shift(sa[1]); shift(sa[2]); shift(sb[0]); shift(sb[1]); shift(sc[0]); shift(sc[1]); shift(se[0]);
          if (l == 2) { shift(sb[4]); shift(sc[4]); }
        }
      }
      const int na = l == 0 ? hwp::D2_RA(1) : l == 1 ? hwp::D2_RA(2) : hwp::D2_RA(3);
      const int nb = l == 0 ? hwp::D2_RB(1) : l == 1 ? hwp::D2_RB(2) : hwp::D2_RB(3);
      const int ne = l == 0 ? hwp::D2_RE(1) : l == 1 ? hwp::D2_RE(2) : hwp::D2_RE(3);
      hwfx::Squares q{0, 0, 0};
#pragma unroll 1
      for (; ra < na; ++ra) fx_row(sa, B.a[ra], q);   // (a lower level's rows are zero where a higher one's data are)
#pragma unroll 1
      for (; rb < nb; ++rb) {   // the same rows for both odd classes (x <-> y images)
        fx_row(sb, B.b[rb], q);
        fx_row(sc, B.b[rb], q);
      }
#pragma unroll 1
      for (; re < ne; ++re) fx_row(se, B.e[re], q);
      const T bl = from_squares<T>(q, 2 * (e[LEVELS ? l : 2] - (1022 + hwfx::BITS) + B.f[l]));
      if (l == 0) beta[1] = bl; else if (l == 1) beta[2] = bl; else beta[3] = bl;
      if constexpr (LEVELS) {
        if (l == 0) {
          a2[0] = sa[0]; a2[1] = sa[1]; a2[2] = sa[2]; e2 = se[0];
          b2[0] = sb[0]; b2[1] = sb[1]; c2[0] = sc[0]; c2[1] = sc[1];
        } else if (l == 1) {
          b3[0] = sb[0]; b3[1] = sb[1]; b3[4] = sb[4];
          c3[0] = sc[0]; c3[1] = sc[1]; c3[4] = sc[4];
        }
      }
    }
  }
  beta[0] = beta1_2d<T>(W, from_double<T>(-dv[3]), from_double<T>(dv[5]), from_double<T>(-dv[1]), from_double<T>(dv[7]));
  T c[4];
  weights_c(W, beta, c);
  Half2 hc[4];
  int ec, eu;                          // the largest exponent of a weight, of a product
  if constexpr (LEVELS) {
    const int x2 = max(cexp(c[0]), cexp(c[3])), x3 = cexp(c[1]), x4 = cexp(c[2]);
    ec = max(x2, max(x3, x4));
    eu = max(max(x2 + e[0], x3 + e[1]), max(x4, hwfx::CEMIN) + e[2]);
    hc[0] = cfixed(c[0], eu - e[0]); hc[1] = cfixed(c[1], eu - e[1]);
    hc[2] = cfixed(c[2], eu - e[2]); hc[3] = cfixed(c[3], eu - e[0]);
  } else {
    ec = fx_weights(c, hc);
    eu = ec + e[2];
  }
  const T u = from_double<T>(e[2] > hwfx::EMAX || ec == 0x7FF ? __longlong_as_double(0x7FF8000000000000LL) : u5);
  const int eb = eu + (hwfx::CF - (1022 + hwfx::CBITS) - (1022 + hwfx::BITS));
  using namespace hwp;
#pragma unroll 1
  for (int b = 0; b < 4; ++b) {
    const int bt = ((b & 1) << 1) | (b >> 1);     // the point with |xi| and |eta| exchanged
    auto dot = [](const int2& c0, const Half2& s0) { return hwfx::prod(s0, c0.x, c0.y); };
    auto add = [](hwfx::Acc& t, const int2& ck, const Half2& sk) { hwfx::mac(t, sk, ck.x, ck.y); };
    auto fin = [](const hwfx::Acc& t) { return hwfx::halves(hwfx::scaled<60>(t)); };
    long long E[4];
    // c_2 q_2 + c_3 q_3 + c_4 q_4 of one class
    auto comb = [&](const Half2& q2, const Half2& q3, const Half2& q4) {
      hwfx::Acc t = hwfx::prod(q2, hc[0].h, hc[0].l);
      hwfx::mac(t, q3, hc[1].h, hc[1].l);
      hwfx::mac(t, q4, hc[2].h, hc[2].l);
      return hwfx::scaled<hwfx::CF>(t);
    };
    auto comb_a = [&](const Half2& q23, const Half2& q4) {   // q_2 = q_3
      hwfx::Acc t = hwfx::prod(q23, hc[3].h, hc[3].l);
      hwfx::mac(t, q4, hc[2].h, hc[2].l);
      return hwfx::scaled<hwfx::CF>(t);
    };
    {
      auto x2 = [&](int k) -> const Half2& { if constexpr (LEVELS) return a2[k]; else return sa[k]; };
      hwfx::Acc t = dot(D2_VA2[b][0], x2(0));
      add(t, D2_VA2[b][1], x2(1)); add(t, D2_VA2[b][2], x2(2));
      hwfx::Acc r = dot(D2_VA4[b][0], sa[0]);
#pragma unroll
      for (int k = 1; k < 7; ++k) add(r, D2_VA4[b][k], sa[k]);
      E[0] = comb_a(fin(t), fin(r));
    }
    auto odd = [&](int p, const Half2* x2, const Half2* x3, const Half2 (&x)[6]) {
      hwfx::Acc t = dot(D2_VB2[p][0], x2[0]);
      add(t, D2_VB2[p][1], x2[1]);
      hwfx::Acc r = dot(D2_VB3[p][0], x3[0]);
      add(r, D2_VB3[p][1], x3[1]); add(r, D2_VB3[p][2], x3[4]);
      hwfx::Acc z = dot(D2_VB4[p][0], x[0]);
#pragma unroll
      for (int k = 1; k < 6; ++k) add(z, D2_VB4[p][k], x[k]);
      return comb(fin(t), fin(r), fin(z));
    };
    E[1] = odd(b, LEVELS ? b2 : sb, LEVELS ? b3 : sb, sb);
    E[2] = odd(bt, LEVELS ? c2 : sc, LEVELS ? c3 : sc, sc);
    {
      hwfx::Acc t = dot(D2_VE2[b][0], LEVELS ? e2 : se[0]);
      hwfx::Acc r = dot(D2_VE4[b][0], se[0]);
      add(r, D2_VE4[b][1], se[1]); add(r, D2_VE4[b][2], se[2]);
      E[3] = comb_a(fin(t), fin(r));
    }
    const int k = 2 + (b >> 1), l = 2 + (b & 1);
    const long long p = E[0] + E[2], q = E[1] + E[3], r = E[0] - E[2], t = E[1] - E[3];
    put(k * 4 + l, u + from_fixed<T>(p + q, eb));
    put((3 - k) * 4 + l, u + from_fixed<T>(p - q, eb));
    put(k * 4 + 3 - l, u + from_fixed<T>(r + t, eb));
    put((3 - k) * 4 + 3 - l, u + from_fixed<T>(r - t, eb));
  }
}

// The form for stencils of uneven data, as a call: the common one keeps its registers.
static __device__ __noinline__ void recon2d_levels(const Beta2<fx64>& B, const double (&dv)[23], int ea, int eo, int em,
                                                   double (&out)[16]) {
  const int e[3] = {ea, eo, em};
  recon2d_fx<true, fx64>(B.w, B, dv, e, [&](int p, fx64 x) { out[p] = x.v; });
}

// Either.  fx64: for a whole warp, since with one exponent the two agree bit for bit and a
// warp that held both kinds would run one after the other (double Mach 800 x 200, two steps:
// 3.03 ms with one exponent for all, 3.10 so, 3.17 by the stencil, 3.20 in plain FP64).
// Double-float, whose common form has its weights in pairs: by the stencil.
template <typename T, typename Put>
__device__ __forceinline__ void recon2d_fixed(const Weights<T>& W, const Beta2<fx64>& B, const double (&d)[23], Put put) {
  const double u5 = d[4];
  double dv[23];
  int ea = hwfx::EMIN, em = 0;
#pragma unroll
  for (int k = 0; k < 23; ++k) {
    dv[k] = k < 9 && k != 4 ? d[k] - u5 : d[k];
    if (k < 9 && k != 4) ea = max(ea, hwfx::bexp(dv[k]));
    else if (k > 8) em = max(em, hwfx::bexp(dv[k]));
  }
  const bool uneven = fx_uneven<T>(ea, em, hwfx::bexp(u5), B.elin);
  const int eo = max(ea, max(hwfx::bexp(dv[12]), hwfx::bexp(dv[19])));   // (the cell's own first moments)
  em = max(ea, em);
  bool levels = uneven;
  if constexpr (std::is_same<T, fx64>::value) levels = __any_sync(__activemask(), uneven);
  double x[23];
  if (levels) {                        // (kept apart from the call: there the data need no registers)
#pragma unroll
    for (int k = 0; k < 23; ++k) x[k] = dv[k];
  } else {
    const int e[3] = {em, em, em};
    recon2d_fx<false, T>(W, B, dv, e, put);
  }
  asm volatile("" ::: "memory");
  if (levels) {
    double y[16];
    recon2d_levels(B, x, uneven ? ea : em, uneven ? eo : em, em, y);
#pragma unroll 1
    for (int p = 0; p < 16; ++p) put(p, from_double<T>(y[p]));
  }
}

template <typename T, typename Put>
__device__ __forceinline__ void recon2d(const Weights<T>& W, const Beta2<T>& B, const T (&d)[23], Put put) {
  if constexpr (std::is_same<T, fx64>::value) {
    double x[23];
#pragma unroll
    for (int k = 0; k < 23; ++k) x[k] = d[k].v;
    recon2d_fixed<T>(W, B, x, put);
    return;
  } else {
  T s[23];
  hwp::split2d<T>(d, s);
  T beta[4];
  hwp::beta2d<T>(B.B2, B.B3, B.B4, s, beta[1], beta[2], beta[3]);
  // beta_1: eqs. (2D-q1-1234) .. (2D-beta1); tau_1 over the 6 unordered pairs
  {
    const T u2 = d[1], u4 = d[3], u5 = d[4], u6 = d[5], u8 = d[7];
    const T bx[4] = {u5 - u4, u6 - u5, u6 - u5, u5 - u4};
    const T by[4] = {u8 - u5, u8 - u5, u5 - u2, u5 - u2};
    T b1[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) b1[k] = bx[k] * bx[k] + by[k] * by[k];
    T ts = T(0);
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int l = k + 1; l < 4; ++l) ts += tabs(b1[k] - b1[l]);
    const T t1 = (ts * T(1.0 / 6.0)) * (ts * T(1.0 / 6.0));
    T gx = T(0), gy = T(0);
    if constexpr (one_division<T>::value) {   // common denominator: one division
      const T y0 = b1[0] + W.eps, y1 = b1[1] + W.eps, y2 = b1[2] + W.eps, y3 = b1[3] + W.eps;
      const T p01 = y0 * y1, p23 = y2 * y3;
      const T n[4] = {(y0 + t1) * (y1 * p23), (y1 + t1) * (y0 * p23), (y2 + t1) * (p01 * y3), (y3 + t1) * (p01 * y2)};
      const T inv = rcp((n[0] + n[1]) + (n[2] + n[3]));
#pragma unroll
      for (int k = 0; k < 4; ++k) { gx = fma(n[k], bx[k], gx); gy = fma(n[k], by[k], gy); }
      gx *= inv;
      gy *= inv;
    } else {
      T w[4], wsum = T(0);
#pragma unroll
      for (int k = 0; k < 4; ++k) { w[k] = T(0.25) * (T(1) + t1 / (b1[k] + W.eps)); wsum += w[k]; }
      const T inv = rcp(wsum);
#pragma unroll
      for (int k = 0; k < 4; ++k) { gx = fma(w[k] * inv, bx[k], gx); gy = fma(w[k] * inv, by[k], gy); }
    }
    beta[0] = gx * gx + gy * gy;
  }
  T c[4];
  combine_weights(W, beta, c);
  T out[16];
  hwp::values2d<T>(s, d[4], c, out);
#pragma unroll
  for (int p = 0; p < 16; ++p) put(p, out[p]);
  }
}

// Positions (ox, oy, kind) of the 23 data of q_4 in gather order.
__device__ __forceinline__ void d4_slot(int c, int& kind, int& ox, int& oy) {
  // u at labels 1..9 (bottom row first), v at 1,3,4,5,6,7,9, w at 1,2,3,5,7,8,9
  const int vl[7] = {1, 3, 4, 5, 6, 7, 9};
  const int wl[7] = {1, 2, 3, 5, 7, 8, 9};
  int lbl;
  if (c < 9) { kind = 0; lbl = c + 1; }
  else if (c < 16) { kind = 1; lbl = vl[c - 9]; }
  else { kind = 2; lbl = wl[c - 16]; }
  ox = (lbl - 1) % 3 - 1;
  oy = (lbl - 1) / 3 - 1;
}

// A face counts as inflow in KXRCF when its velocity exceeds this (absolute,
// in the problem's velocity units): rounding noise around a fluid exactly at
// rest must not decide the indicator.
constexpr double KX_VDEAD = 1e-12;

// Modification weights of eq. (vi) (quartic p_0 of eq. (p0)):
// vbar_i <- -5/76 u_{i-1} + 5/76 u_{i+1} - 11/38 v_{i-1} - 11/38 v_{i+1}.
constexpr double MOD_WU = 5.0 / 76.0;
constexpr double MOD_WV = -11.0 / 38.0;

// ---------------------------------------------------------------- 2D point values and KXRCF
// Point-value arrays G[var][16][j][gpitch]; point (k, l) of a possibly mirrored image cell.
__device__ __forceinline__ int mpt(const Img& m, int k, int l) {
  if (m.sx < 0) k = 3 - k;
  if (m.sy < 0) l = 3 - l;
  return k * 4 + l;
}

__device__ __forceinline__ long long goff(const Prob& P, int i, int j) { return (long long)j * P.gpitch + i; }

// KXRCF decision (and, where asked for, the value) of eq. (KXRCF_) with eq. (line-integral-average_): inflow faces by
// the sign of the GL-weighted face velocity (average of both sides), jumps of
// the indicator variable (variable 0) weighted by dy w_l or dx w_k.
template <typename T>
__device__ __forceinline__ bool kxrcf2d(const Prob& P, const T* __restrict__ G, const T* __restrict__ aux, int i, int j,
                                        double* __restrict__ aleph) {
  const long long o = goff(P, i, j);
  const Img L = image(P, i - 1, j, i, j), R = image(P, i + 1, j, i, j), Bo = image(P, i, j - 1, i, j),
            Tp = image(P, i, j + 1, i, j);
  const long long oL = goff(P, L.i, L.j), oR = goff(P, R.i, R.j), oB = goff(P, Bo.i, Bo.j), oT = goff(P, Tp.i, Tp.j);
  // the neighbours' face velocities (the x ones negated through an x wall, the y
  // ones through a y wall); a fixed-state ghost's is its own state's velocity
  const T axl = L.fs >= 0 ? from_double<T>(P.fixtab[4 * L.fs + 1] / P.fixtab[4 * L.fs]) : aux[(L.sx < 0 ? 0 : 1) * P.gplane + oL];
  const T axr = R.fs >= 0 ? from_double<T>(P.fixtab[4 * R.fs + 1] / P.fixtab[4 * R.fs]) : aux[(R.sx < 0 ? 1 : 0) * P.gplane + oR];
  const T ayb = Bo.fs >= 0 ? from_double<T>(P.fixtab[4 * Bo.fs + 2] / P.fixtab[4 * Bo.fs]) : aux[(Bo.sy < 0 ? 2 : 3) * P.gplane + oB];
  const T ayt = Tp.fs >= 0 ? from_double<T>(P.fixtab[4 * Tp.fs + 2] / P.fixtab[4 * Tp.fs]) : aux[(Tp.sy < 0 ? 3 : 2) * P.gplane + oT];
  // the indicator variable (density) of a neighbour at its point (k, l)
  auto rho_at = [&](const Img& m, long long om, int k, int l) -> T {
    return m.fs >= 0 ? from_double<T>(P.fixtab[4 * m.fs]) : G[(long long)mpt(m, k, l) * P.gplane + om];
  };
  const T dx = pc<T>(P.cdx), dy = pc<T>(P.cdy);
  T s = T(0), len = T(0);
  // a face shared with a solid cell (the forward step's block) is a wall, never an inflow face
  const bool wl = P.sol_j > 0 && is_solid(P, i - 1, j), wr = P.sol_j > 0 && is_solid(P, i + 1, j);
  const bool wb = P.sol_j > 0 && is_solid(P, i, j - 1), wt = P.sol_j > 0 && is_solid(P, i, j + 1);
  const T nrm = aux[4 * P.gplane + o];
  if constexpr (std::is_same<T, fx64>::value) {
    // FP64: no halving, halves of the weights, division or compare on the FP64 pipe
    // (about 50 operations against 90)
    auto inflow = [](fx64 a, fx64 b) {               // (a + b) / 2 > KX_VDEAD (positive doubles order like
      const long long x = __double_as_longlong(a.v + b.v);   //    their bits; not a NaN)
      return x > __double_as_longlong(2.0 * KX_VDEAD) && x < 0x7FF0000000000000LL;
    };
    const bool il = inflow(L.neg & 2 ? -axl : axl, aux[0 * P.gplane + o]) && !wl;
    const bool ir = inflow(-aux[1 * P.gplane + o], R.neg & 2 ? axr : -axr) && !wr;
    const bool ib = inflow(Bo.neg & 4 ? -ayb : ayb, aux[2 * P.gplane + o]) && !wb;
    const bool it = inflow(-aux[3 * P.gplane + o], Tp.neg & 4 ? ayt : -ayt) && !wt;
    auto jump = [&](int p0, int dp, const Img& m, long long om, bool xd, int e) {
      T q[4];
#pragma unroll
      for (int l = 0; l < 4; ++l)
        q[l] = G[(long long)(p0 + l * dp) * P.gplane + o] - (xd ? rho_at(m, om, e, l) : rho_at(m, om, l, e));
      return fma(T(5.0 / 12.0), addrn(q[1], q[2]), T(1.0 / 12.0) * addrn(q[0], q[3]));
    };
    if (il) { s = dy * jump(0, 1, L, oL, true, 3); len = dy; }
    if (ir) { s = fma(dy, jump(12, 1, R, oR, true, 0), s); len += dy; }
    if (ib) { s = fma(dx, jump(0, 4, Bo, oB, false, 3), s); len += dx; }
    if (it) { s = fma(dx, jump(3, 4, Tp, oT, false, 0), s); len += dx; }
    const T d = len * (pc<T>(P.cdx2) * nrm);
    if (aleph) *aleph = d == T(0) ? 0.0 : double(tabs(s) / d);
    const long long bs = __double_as_longlong(tabs(s).v), bd = __double_as_longlong(d.v);
    return bs > bd && bd > 0 && bs <= 0x7FF0000000000000LL;
  }
  const T vxl = T(0.5) * ((L.neg & 2 ? -axl : axl) + aux[0 * P.gplane + o]);
  const T vxr = T(0.5) * (aux[1 * P.gplane + o] + (R.neg & 2 ? -axr : axr));
  const T vyb = T(0.5) * ((Bo.neg & 4 ? -ayb : ayb) + aux[2 * P.gplane + o]);
  const T vyt = T(0.5) * (aux[3 * P.gplane + o] + (Tp.neg & 4 ? -ayt : ayt));
  if (vxl > T(KX_VDEAD) && !wl) {
#pragma unroll
    for (int l = 0; l < 4; ++l) s += dy * gl_w<T>(l) * (G[(long long)(l)*P.gplane + o] - rho_at(L, oL, 3, l));
    len += dy;
  }
  if (-vxr > T(KX_VDEAD) && !wr) {
#pragma unroll
    for (int l = 0; l < 4; ++l) s += dy * gl_w<T>(l) * (G[(long long)(12 + l) * P.gplane + o] - rho_at(R, oR, 0, l));
    len += dy;
  }
  if (vyb > T(KX_VDEAD) && !wb) {
#pragma unroll
    for (int k = 0; k < 4; ++k) s += dx * gl_w<T>(k) * (G[(long long)(k * 4) * P.gplane + o] - rho_at(Bo, oB, k, 3));
    len += dx;
  }
  if (-vyt > T(KX_VDEAD) && !wt) {
#pragma unroll
    for (int k = 0; k < 4; ++k) s += dx * gl_w<T>(k) * (G[(long long)(k * 4 + 3) * P.gplane + o] - rho_at(Tp, oT, k, 0));
    len += dx;
  }
  const T a = len == T(0) || nrm == T(0) ? T(0) : tabs(s) / len / (pc<T>(P.cdx2) * nrm);   // h^{(l+1)/3}, l = 5, h = dx
  if (aleph) *aleph = double(a);
  return a > T(1);
}

// ---------------------------------------------------------------- step checks
// A double truncated to FP32 by integer work, magnitudes outside its normal range as 0 or infinity.
__device__ __forceinline__ float f32_trunc(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const int e = (int)((hi >> 20) & 0x7FFu) - (1023 - 127);
  if (e <= 0) return 0.0f;
  if (e >= 255) return __uint_as_float((hi & 0x80000000u) | 0x7F800000u);
  return __uint_as_float((hi & 0x80000000u) | ((unsigned)e << 23) | ((hi & 0xFFFFFu) << 3) | (lo >> 29));
}

// Whether an Euler cell average is outside the physical set: not rho > 0, or not
// p = (gamma - 1)(E - |m|^2 / (2 rho)) > 0, i.e. 2 E rho > |m|^2 (no division).
// Cells that are inside by more than FP32's rounding are passed on FP32 copies;
// only the others take the FP64 test.
__device__ __forceinline__ bool nonphysical(double rho, double m, double n, double E) {
  const float r = f32_trunc(rho), a = f32_trunc(m), b = f32_trunc(n), e = f32_trunc(E);
  const float x = 2.0f * e * r, y = a * a + b * b;
  if (r > 0.0f && x > 1.00001f * y && x > 1e-30f && x < 1e30f) return false;
  const double m2 = m * m + n * n;
  return !(rho > 0.0) || !(2.0 * E * rho > m2);
}

// Bounds of an Euler average's |velocity| + sound speed per direction from FP32
// copies: lo <= exact <= hi.  Truncating the conserved values and the FP32
// arithmetic err by less than 2^-20 relative, the pressure by 2^-20 of E + kinetic
// energy (gamma - 1 is rounded from FP64: in FP32 it cancels near 1).  What falls
// below FP32's normal range (a momentum, its product with the velocity) is below
// 1e-38 absolute, which density, E and the squared sound speed inside the limits leave
// far below those margins.  Outside them, and for a non-physical or barely physical
// average, hi = infinity and lo = 0: the cell takes the exact speed.
__device__ __forceinline__ void speed_bounds(const Prob& P, const double* __restrict__ U, int i, int j, float (&lo)[2],
                                             float (&hi)[2]) {
  const float r = f32_trunc(U[sidx(P, 0, 0, i, j)]), m = f32_trunc(U[sidx(P, 1, 0, i, j)]);
  const float n = P.nvar == 4 ? f32_trunc(U[sidx(P, 2, 0, i, j)]) : 0.0f, E = f32_trunc(U[sidx(P, P.nvar - 1, 0, i, j)]);
  const float ri = 1.0f / r, u = fabsf(m) * ri, w = fabsf(n) * ri, ke = 0.5f * (fabsf(m) * u + fabsf(n) * w);
  const float p = E - ke, d = 1e-6f * (E + ke), gg = P.cgamma.f * P.cgm1.f * ri, c2 = gg * (p + d);
  const float cl = sqrtf(gg * (p - d)) * 0.999998f, ch = sqrtf(c2) * 1.000002f;
  const bool ok = r > 1e-15f && r < 1e15f && E > 1e-15f && E < 1e15f && p > d && c2 > 1e-30f && c2 < 1e30f;
  lo[0] = ok ? u * 0.999998f + cl : 0.0f;
  lo[1] = ok ? w * 0.999998f + cl : 0.0f;
  hi[0] = ok ? u * 1.000002f + ch : INFINITY;
  hi[1] = ok ? w * 1.000002f + ch : INFINITY;
}

// ---------------------------------------------------------------- TVB indicator
// The minmod-based TVB indicator named in Remark 2 (Cockburn & Shu's TVB
// limiter used as a troubled-cell indicator) on the indicator variable
// (variable 0), acting on the cell's linear polynomial fixed by its moments:
// its face deviations are +-6 vbar (x) and +-6 wbar (y).  The cell is troubled
// when the modified minmod m(a, b, c) = a if |a| <= M h^2, else minmod(a, b, c)
// changes a = 6 vbar (6 wbar) against the forward and backward differences of
// the averages in that direction.  FP64: it reads only the FP64 state.
__device__ __forceinline__ bool tvb_changes(double a, double b, double c, double bound) {
  if (!(fabs(a) > bound)) return false;
  double mm = 0.0;
  if (a > 0.0 && b > 0.0 && c > 0.0) mm = fmin(a, fmin(b, c));
  else if (a < 0.0 && b < 0.0 && c < 0.0) mm = fmax(a, fmax(b, c));
  return mm != a;
}

__device__ __forceinline__ bool tvb_cell(const Prob& P, const double* __restrict__ U, int i, int j) {
  const double bound = P.tvb_m * P.dx * P.dx;
  const double u0 = U[sidx(P, 0, 0, i, j)];
  const Img L = image(P, i - 1, j, i, j), R = image(P, i + 1, j, i, j);
  const double ax = 6.0 * U[sidx(P, 0, 1, i, j)];
  if (tvb_changes(ax, avg_img(P, U, R, 0) - u0, u0 - avg_img(P, U, L, 0), bound)) return true;
  if (P.nmom == 2) return false;
  const Img Bo = image(P, i, j - 1, i, j), Tp = image(P, i, j + 1, i, j);
  const double ay = 6.0 * U[sidx(P, 0, 2, i, j)];
  return tvb_changes(ay, avg_img(P, U, Tp, 0) - u0, u0 - avg_img(P, U, Bo, 0), bound);
}

}  // namespace hw
