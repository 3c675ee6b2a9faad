// Kernels of the two-dimensional stage pipeline and of the batched stage (shared
// by the per-precision translation units; internal linkage).
#pragma once
#include <algorithm>
#include <type_traits>

#include "hweno_internal.h"

namespace hw {
namespace {


constexpr int TX = 32, TY = 4;   // update tile (one warp per row)
constexpr int RB = 128;          // threads per block of the per-cell kernels

// Images of the 3x3 block around (i,j); the boundary map is separable, so
// three x-images and three y-images describe all nine cells.
struct Nbr {
  int xi[3], xs[3];     // image column and sign of the x first moment, for ox = -1, 0, 1
  int yj[3], ys[3];     // image row and sign of the y first moment, for oy = -1, 0, 1
  int neg[3][3];        // variables negated by reflective walls, [oy + 1][ox + 1]
  int fs[3][3];         // fixed-state ghost entry (-1: none), set when FIX
  int ci[3][3], cj[3][3], csx[3][3], csy[3][3];   // FIX: the full image of each cell
};

template <bool FIX>
__device__ __forceinline__ Nbr neighbours(const Prob& P, int i, int j) {
  Nbr n;
  int nx[3], ny[3];
#pragma unroll
  for (int o = -1; o <= 1; ++o) {
    // by the kinds alone: a fixed ghost in the separable x or y image does
    // not make its row or column fixed for the diagonal cells
    const Img a = image_kind(P, i + o, j), b = image_kind(P, i, j + o);
    n.xi[o + 1] = a.i; n.xs[o + 1] = a.sx; nx[o + 1] = a.neg;
    n.yj[o + 1] = b.j; n.ys[o + 1] = b.sy; ny[o + 1] = b.neg;
  }
#pragma unroll
  for (int oy = 0; oy < 3; ++oy)
#pragma unroll
    for (int ox = 0; ox < 3; ++ox) n.neg[oy][ox] = nx[ox] | ny[oy];
  if constexpr (FIX) {
    // fixed-state ghosts and the solid block break the separable form: the full
    // image of each cell (equal to the separable one wherever neither applies)
#pragma unroll
    for (int oy = 0; oy < 3; ++oy)
#pragma unroll
      for (int ox = 0; ox < 3; ++ox) {
        const Img m = image(P, i + ox - 1, j + oy - 1, i, j);
        n.fs[oy][ox] = m.fs;
        n.neg[oy][ox] = m.fs >= 0 ? m.neg : (P.sol_j > 0 ? m.neg : n.neg[oy][ox]);
        n.ci[oy][ox] = m.fs >= 0 ? n.xi[ox] : m.i;
        n.cj[oy][ox] = m.fs >= 0 ? n.yj[oy] : m.j;
        n.csx[oy][ox] = m.fs >= 0 ? n.xs[ox] : m.sx;
        n.csy[oy][ox] = m.fs >= 0 ? n.ys[oy] : m.sy;
      }
  }
  return n;
}

// Reconstruction passes: every cell from the stage input (PLAIN); the listed
// troubled cells from the modified moments (FLAGGED, Step 2.3); or every cell,
// those already flagged (mask 1) from the modified moments (MIXED: the learned
// indicator decides before Step 1).
enum RecMode { REC_PLAIN = 0, REC_FLAGGED = 1, REC_MIXED = 2 };

// Moment of kind 0 (average), 1 (x first moment) or 2 (y first moment) of
// the stencil cell (ox, oy); when usemod, first moments of flagged stencil
// cells come from the modified copy (eq. (vi) applied before Step 2.3).
template <int MODE, bool FIX>
__device__ __forceinline__ double load_mom(const Prob& P, const double* __restrict__ U, const uint8_t* __restrict__ mask,
                                           const double* __restrict__ Mod, const Nbr& n, int var, int kind, int ox,
                                           int oy, bool usemod) {
  if constexpr (FIX) {
    const int fs = n.fs[oy + 1][ox + 1];
    if (fs >= 0) return kind == 0 ? ((n.neg[oy + 1][ox + 1] >> var) & 1 ? -1.0 : 1.0) * P.fixtab[4 * fs + var] : 0.0;
  }
  const int ci = FIX ? n.ci[oy + 1][ox + 1] : n.xi[ox + 1], cj = FIX ? n.cj[oy + 1][ox + 1] : n.yj[oy + 1];
  const int sxm = FIX ? n.csx[oy + 1][ox + 1] : n.xs[ox + 1], sym = FIX ? n.csy[oy + 1][ox + 1] : n.ys[oy + 1];
  const long long so = (long long)cj * P.pitch + ci;
  // the sign bit flipped by integer work (no FP64 instruction; bitwise the same
  // as negation), measured 6 % faster in FP64
  unsigned long long flip = ((n.neg[oy + 1][ox + 1] >> var) & 1) ? 1ull : 0ull;
  double v;
  if (kind == 0) {
    v = U[(long long)(var * 3) * P.plane + so];
  } else {
    if (MODE != REC_PLAIN && usemod && mask[(long long)cj * P.nx + ci] == 1)
      v = Mod[(long long)(var * 2 + kind - 1) * P.plane + so];
    else
      v = U[(long long)(var * 3 + kind) * P.plane + so];
    if (kind == 1 && sxm < 0) flip ^= 1ull;
    if (kind == 2 && sym < 0) flip ^= 1ull;
  }
  return __longlong_as_double(__double_as_longlong(v) ^ (long long)(flip << 63));
}

// FP32 form: the moment from the float copy of the state the update kernel
// writes beside it (the state rounded to nearest), signs flipped by integer
// work; modified first moments of flagged cells still come from the FP64 copy.
template <int MODE>
__device__ __forceinline__ float load_mom32(const Prob& P, const float* __restrict__ U32,
                                            const uint8_t* __restrict__ mask, const double* __restrict__ Mod,
                                            const Nbr& n, int var, int kind, int ox, int oy, bool usemod) {
  const int ci = n.xi[ox + 1], cj = n.yj[oy + 1];
  const long long so = (long long)cj * P.pitch + ci;
  unsigned flip = (n.neg[oy + 1][ox + 1] >> var) & 1u;
  float v;
  if (kind == 0) {
    v = U32[(long long)(var * 3) * P.plane + so];
  } else {
    if (MODE != REC_PLAIN && usemod && mask[(long long)cj * P.nx + ci] == 1)
      v = float(Mod[(long long)(var * 2 + kind - 1) * P.plane + so]);
    else
      v = U32[(long long)(var * 3 + kind) * P.plane + so];
    if (kind == 1 && n.xs[ox + 1] < 0) flip ^= 1u;
    if (kind == 2 && n.ys[oy + 1] < 0) flip ^= 1u;
  }
  return __uint_as_float(__float_as_uint(v) ^ (flip << 31));
}

// KXRCF face-velocity partials of faces [f0, f1) (x-lo, x-hi, y-lo, y-hi) of the cell
// at offset o from its point values: point indices p0 + q dp, velocity
// (rho mu)/rho, (rho nu)/rho or u.  (G was written by this block: no read-only loads.)
template <typename T, int NV>
__device__ __forceinline__ void face_partials(const Prob& P, T* G, T* aux, long long o, int f0, int f1) {
#pragma unroll 1
  for (int f = f0; f < f1; ++f) {
    const int p0 = f == 1 ? 12 : f == 3 ? 3 : 0, dp = f < 2 ? 1 : 4, v = NV == 4 ? (f < 2 ? 1 : 2) : 0;
    T s = T(0);
    if (P.eq == EQ_ADV) {
      s = T(f < 2 ? P.adv_a : P.adv_b);
    } else {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const T m = G[(long long)(v * 16 + p0 + q * dp) * P.gplane + o];
        s = fma(gl_w<T>(q), NV == 4 ? m * rcp(G[(long long)(p0 + q * dp) * P.gplane + o]) : m, s);
      }
    }
    aux[(long long)f * P.gplane + o] = s;
  }
}

// Variables [v0, v1) of cell (i, j).  The fixed-point precisions leave the face
// partials to face_partials.
template <typename T, int NV, int MODE, bool FIX = false, bool S32 = false>
__device__ __forceinline__ void rec2d_cell(const Prob& P, const Weights<T>& W,
                                           const typename rows2d<T>::type& B, const double* __restrict__ U,
                                           const uint8_t* __restrict__ mask,
                                           const double* __restrict__ Mod, int i, int j, T* __restrict__ G,
                                           T* __restrict__ aux, const float* __restrict__ U32 = nullptr, int v0 = 0,
                                           int v1 = NV) {
  constexpr bool FLAGGED = MODE == REC_FLAGGED;
  const bool usemod = MODE == REC_FLAGGED || (MODE == REC_MIXED && mask[(long long)j * P.nx + i] == 1);
  const Nbr nb = neighbours<FIX>(P, i, j);
  const long long o = goff(P, i, j);
  // FP32 from the float copy and fx64, plain pass, all 3 x 3 cells inside the grid: no image to apply,
  // the moments are read at fixed offsets from the cell's own
  constexpr bool DIRECT = (S32 || (fixed2d<T>::value && !FIX)) && MODE == REC_PLAIN;
  const bool inner = DIRECT && i > 0 && i < P.nx - 1 && j > 0 && j < P.ny - 1;
  using Src = std::conditional_t<S32, float, double>;
  const Src* __restrict__ Uc;
  if constexpr (S32) Uc = U32 + ((long long)j * P.pitch + i);
  else Uc = U + ((long long)j * P.pitch + i);
  constexpr bool FXD = fixed2d<T>::value;
  using D = std::conditional_t<FXD, double, T>;   // the data's type
  T rinv[16];
  T pxl = T(0), pxr = T(0), pyb = T(0), pyt = T(0), nrm = T(0);
  [[maybe_unused]] long long nrmb = 0;   // fx64: the norm's bits (non-negative doubles order like them)
#pragma unroll 1
  for (int v = v0; v < v1; ++v) {
    D d[23];
    if (inner) {
#pragma unroll
      for (int c = 0; c < 23; ++c) {
        int kind, ox, oy;
        d4_slot(c, kind, ox, oy);
        if constexpr (DIRECT) d[c] = D(Uc[(long long)(v * 3 + kind) * P.plane + (long long)oy * P.pitch + ox]);
      }
    } else {
#pragma unroll
      for (int c = 0; c < 23; ++c) {
        int kind, ox, oy;
        d4_slot(c, kind, ox, oy);
        if constexpr (S32)
          d[c] = load_mom32<MODE>(P, U32, mask, Mod, nb, v, kind, ox, oy, usemod);
        else
          d[c] = from_double<D>(load_mom<MODE, FIX>(P, U, mask, Mod, nb, v, kind, ox, oy, usemod));
      }
    }
    T out[16];
    if constexpr (FXD) {
      // the point values go out as they are formed (four base points in turn);
      // the partials read them back below
      T* __restrict__ Gv = G + (long long)(v * 16) * P.gplane + o;
      recon2d_fixed<T>(W, B, d, [&](int p, T x) {
        Gv[p * P.gplane] = x;
        if (!FLAGGED && v == 0) {
          if constexpr (is_df64<T>::value) nrm = tmax(nrm, tabs(x));
          else nrmb = max(nrmb, __double_as_longlong(x.v) & 0x7FFFFFFFFFFFFFFFLL);
        }
      });
      if (!FLAGGED && v == 0) {
        if constexpr (!is_df64<T>::value) nrm = __longlong_as_double(nrmb);
        aux[4 * P.gplane + o] = nrm;
      }
    } else {
      recon2d<T>(W, B, d, [&](int p, T x) { out[p] = x; });
#pragma unroll
      for (int p = 0; p < 16; ++p) G[(long long)(v * 16 + p) * P.gplane + o] = out[p];
    }
    if (!FLAGGED && !FXD) {
      if (v == 0) {
#pragma unroll
        for (int p = 0; p < 16; ++p) nrm = tmax(nrm, tabs(out[p]));
        if (P.eq == EQ_EULER) {
          // 1/rho at the 12 boundary points (the face velocities need only those)
          constexpr int bp[12] = {0, 1, 2, 3, 4, 7, 8, 11, 12, 13, 14, 15};
          if constexpr (sizeof(T) == 8) {
            T x[12], r[12];
#pragma unroll
            for (int q = 0; q < 12; ++q) x[q] = out[bp[q]];
            batch_inverse_ranged<12, T>(x, r);
#pragma unroll
            for (int q = 0; q < 12; ++q) rinv[bp[q]] = r[q];
          } else {
#pragma unroll
            for (int q = 0; q < 12; ++q) rinv[bp[q]] = rcp(out[bp[q]]);
          }
        } else if (P.eq == EQ_BURGERS) {
#pragma unroll
          for (int l = 0; l < 4; ++l) {
            pxl += gl_w<T>(l) * out[l];
            pxr += gl_w<T>(l) * out[12 + l];
            pyb += gl_w<T>(l) * out[l * 4];
            pyt += gl_w<T>(l) * out[l * 4 + 3];
          }
        } else {
          pxl = pxr = T(P.adv_a);
          pyb = pyt = T(P.adv_b);
        }
      } else if (P.eq == EQ_EULER && v == 1) {
#pragma unroll
        for (int l = 0; l < 4; ++l) {
          pxl += gl_w<T>(l) * (out[l] * rinv[l]);
          pxr += gl_w<T>(l) * (out[12 + l] * rinv[12 + l]);
        }
      } else if (P.eq == EQ_EULER && v == 2) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          pyb += gl_w<T>(k) * (out[k * 4] * rinv[k * 4]);
          pyt += gl_w<T>(k) * (out[k * 4 + 3] * rinv[k * 4 + 3]);
        }
      }
    }
  }
  if (!FLAGGED && !FXD) {
    aux[0 * P.gplane + o] = pxl;
    aux[1 * P.gplane + o] = pxr;
    aux[2 * P.gplane + o] = pyb;
    aux[3 * P.gplane + o] = pyt;
    aux[4 * P.gplane + o] = nrm;
  }
}

// rerec (REC_FLAGGED only, may be null) accumulates the number of cells
// reconstructed a second time.  A thread per cell: FP32, plain double and the
// scalar laws.  FP32 with the float copy: 8 blocks (64 registers, 164 B of spills)
// measured 0.545 ms per 2048^2 launch against 0.685 at 4 blocks (119 registers).
template <typename T, int NV, int MODE, bool S32 = false>
__global__ void __launch_bounds__(RB, (std::is_same<T, float>::value ? 8 : fixed2d<T>::value ? 4 : 1)) rec2d_kernel(
    const __grid_constant__ Prob P, const __grid_constant__ Weights<T> W,
    const __grid_constant__ typename rows2d<T>::type B, const double* __restrict__ U,
                                                  const uint8_t* __restrict__ mask, const double* __restrict__ Mod,
                                                  const int* __restrict__ list, const int* __restrict__ count,
                                                  T* __restrict__ G, T* __restrict__ aux,
                                                  unsigned long long* __restrict__ rerec,
                                                  const float* __restrict__ U32 = nullptr) {
  constexpr bool FLAGGED = MODE == REC_FLAGGED;
  const long long ncell = (long long)P.nx * P.ny;
  const long long n = FLAGGED ? (long long)*count : ncell;
  if (FLAGGED && rerec && blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(rerec, (unsigned long long)n);
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
    const int cell = FLAGGED ? list[t] : (int)t;
    rec2d_cell<T, NV, MODE, false, S32>(P, W, B, U, mask, Mod, cell % P.nx, cell / P.nx, G, aux, U32);
    if constexpr (fixed2d<T>::value && !FLAGGED) face_partials<T, NV>(P, G, aux, goff(P, cell % P.nx, cell / P.nx), 0, 4);
  }
}

// 2D Euler in the fixed-point precisions: 32 cells a block, a warp per variable and
// then per face, so that a thread's chain is a quarter of the cell's and the code
// between the barriers is shared by the block.  Measured against a thread per cell
// (ms per launch, FP64): 64^2 0.065 -> 0.021, 256^2 0.123 -> 0.105, 2048^2
// 5.67 -> 5.52 (18.1 with the linear part in FP64), troubled cells 0.13 -> 0.11;
// double-float 2048^2 5.44 -> 5.24 (7.6 in pairs); with the reciprocals and the
// indicators' squares in integers 4.39 and 4.67; with the stencils of uneven data
// and the reciprocals rounded to nearest 4.51 and 4.72.  FP64: 5 resident blocks per
// SM; 504 FP64 operations per cell (2330 before), that pipe 74 % busy, 20.4 k
// instructions.  Double-float: 25.1 k instructions per cell, issue 56 %, the ALU
// 37 % busy (1.2 % faster at 5 blocks than at 4 with 120 registers); weights in FP64
// beside the integers measured alike.
template <typename T, int MODE, bool FIX = false>
__global__ void __launch_bounds__(RB, 5) rec2d_split_kernel(
    const __grid_constant__ Prob P, const __grid_constant__ Weights<T> W,
    const __grid_constant__ typename rows2d<T>::type B, const double* __restrict__ U,
    const uint8_t* __restrict__ mask, const double* __restrict__ Mod, const int* __restrict__ list,
    const int* __restrict__ count, T* __restrict__ G, T* __restrict__ aux, unsigned long long* __restrict__ rerec) {
  constexpr bool FLAGGED = MODE == REC_FLAGGED;
  const int n = FLAGGED ? *count : P.nx * P.ny;
  if (FLAGGED && rerec && blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(rerec, (unsigned long long)n);
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int t0 = blockIdx.x * 32; t0 < n; t0 += gridDim.x * 32) {   // (block-uniform)
    const int t = t0 + lane, cell = t < n ? (FLAGGED ? list[t] : t) : -1;
    const int i = cell % P.nx, j = cell / P.nx;
    const bool take = cell >= 0 && !(FIX && is_solid(P, i, j));
    if (take) rec2d_cell<T, 4, MODE, FIX>(P, W, B, U, mask, Mod, i, j, G, aux, nullptr, w, w + 1);
    if constexpr (!FLAGGED) {
      __syncthreads();
      if (take) face_partials<T, 4>(P, G, aux, goff(P, i, j), w, w + 1);
    }
  }
}

// Step 2.1 for one cell: the troubled-cell decision of the configured indicator.
template <typename T>
__device__ __forceinline__ bool flag2d_cell(const Prob& P, const double* __restrict__ U,
                                            const T* __restrict__ G, const T* __restrict__ aux, int i, int j,
                                            double* __restrict__ aleph) {
  if (P.sol_j > 0 && is_solid(P, i, j)) {
    if (aleph) aleph[(long long)j * P.nx + i] = 0.0;
    return false;
  }
  if (P.indicator == IND_ALL) return true;
  if (P.indicator == IND_TVB) return tvb_cell(P, U, i, j);
  if (P.indicator != IND_KXRCF) return false;
  return kxrcf2d<T>(P, G, aux, i, j, aleph ? aleph + ((long long)j * P.nx + i) : nullptr);
}

// Step 2.2 for one troubled cell (dimension by dimension): modified first
// moments from the pre-modification moments of the x and y neighbours.
template <int NV>
__device__ __forceinline__ void modify2d_cell(const Prob& P, const double* __restrict__ U, double* __restrict__ Mod,
                                              int i, int j) {
  const Img L = image(P, i - 1, j, i, j), R = image(P, i + 1, j, i, j), Bo = image(P, i, j - 1, i, j),
            Tp = image(P, i, j + 1, i, j);
  const long long o = (long long)j * P.pitch + i;
  // moment (kind 1: x, 2: y first moment) of an edge neighbour; a fixed-state
  // ghost has its state as average and zero first moments
  auto mom = [&](const Img& m, int v, int kind) -> double {
    if (m.fs >= 0) return kind == 0 ? fixed_val(P, m, v) : 0.0;
    // the image's sign as a bit (a product with an integer sign is a conversion and
    // a multiplication on the FP64 pipe: 70 % of this kernel's cycles in FP32)
    const int neg = ((m.neg >> v) ^ ((kind == 1 ? m.sx : kind == 2 ? m.sy : 1) >> 31)) & 1;
    return __longlong_as_double(__double_as_longlong(U[sidx(P, v, kind, m.i, m.j)]) ^ ((long long)neg << 63));
  };
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const double uL = mom(L, v, 0), uR = mom(R, v, 0), vL = mom(L, v, 1), vR = mom(R, v, 1);
    const double uB = mom(Bo, v, 0), uT = mom(Tp, v, 0), wB = mom(Bo, v, 2), wT = mom(Tp, v, 2);
    Mod[(long long)(v * 2 + 0) * P.plane + o] = MOD_WU * (uR - uL) + MOD_WV * (vL + vR);
    Mod[(long long)(v * 2 + 1) * P.plane + o] = MOD_WU * (uT - uB) + MOD_WV * (wB + wT);
  }
}

// Warp-aggregated append of flagged entries to a list (all 32 lanes take part).
template <typename E>
__device__ __forceinline__ void warp_append(bool flag, E entry, E* __restrict__ list, int* __restrict__ count) {
  const unsigned act = __ballot_sync(0xffffffffu, flag);
  if (!act) return;
  const int lane = threadIdx.x & 31;
  const int leader = __ffs(act) - 1;
  int base = 0;
  if (lane == leader) base = atomicAdd(count, __popc(act));
  base = __shfl_sync(0xffffffffu, base, leader);
  if (flag) list[base + __popc(act & ((1u << lane) - 1u))] = entry;
}

template <typename T, int NV>
__global__ void __launch_bounds__(TX * TY) flag2d_kernel(const __grid_constant__ Prob P, const double* __restrict__ U,
                                                        const T* __restrict__ G, const T* __restrict__ aux,
                                                        uint8_t* __restrict__ mask, double* __restrict__ Mod,
                                                        int* __restrict__ list, int* __restrict__ count,
                                                        double* __restrict__ aleph) {
  const int i = blockIdx.x * TX + threadIdx.x, j = blockIdx.y * TY + threadIdx.y;
  const bool valid = i < P.nx && j < P.ny;
  const bool flag = valid && flag2d_cell<T>(P, U, G, aux, i, j, aleph);
  warp_append<int>(flag, j * P.nx + i, list, count);   // a warp is one tile row
  if (!valid) return;
  mask[(long long)j * P.nx + i] = flag ? 1 : 0;
  if (flag) modify2d_cell<NV>(P, U, Mod, i, j);
}

// KXRCF for the cells the learned indicator left undecided (mask 2): the
// decision, eq. (vi) for the troubled ones and their list for Step 2.3.
template <typename T, int NV>
__global__ void __launch_bounds__(RB) fallback2d_kernel(const __grid_constant__ Prob P, const double* __restrict__ U,
                                                       const T* __restrict__ G, const T* __restrict__ aux,
                                                       const int* __restrict__ und, const int* __restrict__ und_count,
                                                       uint8_t* __restrict__ mask, double* __restrict__ Mod,
                                                       int* __restrict__ list, int* __restrict__ count,
                                                       double* __restrict__ aleph) {
  const long long n = *und_count;
  const long long stride = (long long)gridDim.x * blockDim.x;
  // warp-uniform trip count: every lane of a warp takes part in the append
  for (long long b = (long long)blockIdx.x * blockDim.x + (threadIdx.x & ~31); b < n; b += stride) {
    const long long t = b + (threadIdx.x & 31);
    bool flag = false;
    int cell = 0;
    if (t < n) {
      cell = und[t];
      const int i = cell % P.nx, j = cell / P.nx;
      flag = kxrcf2d<T>(P, G, aux, i, j, aleph ? aleph + cell : nullptr);
      mask[cell] = flag ? 1 : 0;
      if (flag) modify2d_cell<NV>(P, U, Mod, i, j);
    }
    warp_append<int>(flag, cell, list, count);
  }
}

template <typename T, int NV>
__device__ __forceinline__ void gl_state(const Prob& P, const T* __restrict__ G, const Img& m, int k, int l, T (&u)[NV]) {
  if (m.fs >= 0) {   // fixed-state ghost: its state at every point
#pragma unroll
    for (int v = 0; v < NV; ++v) u[v] = from_double<T>(fixed_val(P, m, v));
    return;
  }
  const long long o = goff(P, m.i, m.j);
  const int p = mpt(m, k, l);
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const T x = G[(long long)(v * 16 + p) * P.gplane + o];
    u[v] = (m.neg >> v) & 1 ? -x : x;
  }
}

// The numerical flux of one face point, one inlined solver for both
// directions: a y face is an x face with the two momentum components
// exchanged (the HLLC expressions are the same, term for term); at a wall
// face the star branch is taken.
template <typename T, int NV, bool SOFT = true>
__device__ __forceinline__ void face_flux(const Prob& P, T (&uL)[NV], T (&uR)[NV], bool xd, bool wall, T* out) {
  if constexpr (NV == 4) {
    if (!xd) {
      const T a = uL[1], b = uR[1];
      uL[1] = uL[2]; uL[2] = a;
      uR[1] = uR[2]; uR[2] = b;
    }
    T F[4];
    if constexpr (lean<T>::value) hllc_lean<T, 4, SOFT>(P, uL, uR, 0, F, wall);
    else hllc<T, 4>(P, uL, uR, 0, F, wall);
    out[0] = F[0];
    out[1] = xd ? F[1] : F[2];
    out[2] = xd ? F[2] : F[1];
    out[3] = F[3];
  } else {
    num_flux<T, NV>(P, uL, uR, xd ? 0 : 1, out);
  }
}

struct Rk {
  const double* Uin; const double* Un; double* Uout;
  const uint8_t* mask; const double* Mod; const uint8_t* maskN; const double* ModN;
  double dt, cA, cB;
  double* Lout; double* Umod;
  unsigned* status;
  const double* dtp;     // dt on the device (overrides dt); < 0: skip, Uout = Uin
  float* U32out = nullptr;   // FP32 form: the float copy of Uout (the next stage's reconstruction input)
};

// Where update2d_tile reads point values and stage states: global memory (any
// tile) or, for an interior tile of the FP32 TMA kernel, the boxes staged in
// shared memory.  The arithmetic is the same template either way, so both give
// bitwise the same results.
template <typename T>
struct GlobalSrc {
  static constexpr bool staged = false;
  const T* __restrict__ G;
  __device__ __forceinline__ T g(const Prob& P, int v, int p, int i, int j) const {
    return G[(long long)(v * 16 + p) * P.gplane + goff(P, i, j)];
  }
  __device__ __forceinline__ double uin(const Prob& P, const Rk& S, int q, int i, int j) const {
    return S.Uin[(long long)q * P.plane + (long long)j * P.pitch + i];
  }
  __device__ __forceinline__ double un(const Prob& P, const Rk& S, int q, int i, int j) const {
    return S.Un[(long long)q * P.plane + (long long)j * P.pitch + i];
  }
};

// The TMA kernel's shared-memory box (FP32): the tile's own point values,
// [64 planes][4 rows][32 columns] from cell (i0, j0); the one-cell halo the face
// fluxes need and the stage states come from global memory.
constexpr int GBX = 32, GBY = 4;
struct StagedSrc {
  static constexpr bool staged = true;
  const float* gs;
  const float* __restrict__ G;
  int i0, j0;
  __device__ __forceinline__ float g(const Prob& P, int v, int p, int i, int j) const {
    const int x = i - i0, y = j - j0;
    if ((unsigned)x < (unsigned)GBX && (unsigned)y < (unsigned)GBY) return gs[((v * 16 + p) * GBY + y) * GBX + x];
    return G[(long long)(v * 16 + p) * P.gplane + goff(P, i, j)];
  }
  __device__ __forceinline__ double uin(const Prob& P, const Rk& S, int q, int i, int j) const {
    return S.Uin[(long long)q * P.plane + (long long)j * P.pitch + i];
  }
  __device__ __forceinline__ double un(const Prob& P, const Rk& S, int q, int i, int j) const {
    return S.Un[(long long)q * P.plane + (long long)j * P.pitch + i];
  }
};

// Quadrature of one cell (2D Euler, the lean precisions).  The 16 points fall into
// three groups of one weight (corners 1, edges 5, centre 25, over 144), summed
// without weights.  With the kinetic terms A = sum w m^2/rho and
// S = sum w (m^2 + n^2)/rho the momentum fluxes need no pressure per point:
// sum w p = (gamma - 1)(E - S/2), and the sums of m, n and E are the cell's averages
// (every q_l has them, and the quadrature is exact for degree 5).
template <typename T> struct Quad { T A, C, K, X, Y; };

template <typename T, typename Src>
__device__ __forceinline__ Quad<T> quad_lean(const Prob& P, const Src& src, int i, int j) {
  const T kap = pc<T>(P.chg);
  T A, C, K, X, Y;
  A = C = K = X = Y = T(0);
#pragma unroll
  for (int grp = 2; grp >= 0; --grp) {               // 25 centre + 5 edges + corners (Horner in 5)
    if (grp < 2) { A *= T(5); C *= T(5); K *= T(5); X *= T(5); Y *= T(5); }
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int l = 0; l < 4; ++l) {
        const bool ki = k == 1 || k == 2, li = l == 1 || l == 2;
        if ((int)ki + (int)li != grp) continue;
        const int p = k * 4 + l;
        const T m = src.g(P, 1, p, i, j), n = src.g(P, 2, p, i, j), E = src.g(P, 3, p, i, j);
        const T inv = rcp(src.g(P, 0, p, i, j));
        const T mu = m * inv, nu = n * inv;
        const T s = fma(m, mu, n * nu);
        A = fma(m, mu, A);
        C = fma(m, nu, C);
        K = K + s;
        const T H = fma(-kap, s, E);                 // (E + p) / gamma
        X = fma(mu, H, X);
        Y = fma(nu, H, Y);
      }
  }
  return Quad<T>{A, C, K, X, Y};
}

// L(U) and the Runge-Kutta combination of variables [v0, v1) of one cell, from its
// quadrature and the integrals of its faces (slot 0 the mean, 1 the first moment; xm
// left, xp right, ym below, yp above).  The new averages go to newavg; returns
// whether every new moment is finite.
template <typename T, typename Src>
__device__ __forceinline__ bool combine_lean(const Prob& P, const Src& src, const Rk& S, int i, int j, const Quad<T>& q,
                                             const T (&xm)[4][4], const T (&xp)[4][4], const T (&ym)[4][4],
                                             const T (&yp)[4][4], int v0, int v1, double* newavg) {
  const long long so = (long long)j * P.pitch + i;
  const long long cell = (long long)j * P.nx + i;
  const T g = pc<T>(P.cgamma), gm1 = pc<T>(P.cgm1);
  const T A = q.A, C = q.C, K = q.K, X = q.X, Y = q.Y;
  // (every product that meets a sum is a written fma: what the compiler would
  // contract could differ between the kernels that share this, which agree bit for bit)
  const T w = T(1.0 / 144.0);
  const T mbar = from_double<T>(src.uin(P, S, 3, i, j)), nbar = from_double<T>(src.uin(P, S, 6, i, j)),
          Ebar = from_double<T>(src.uin(P, S, 9, i, j));
  const T pbar = gm1 * fma(T(-0.5) * w, K, Ebar);
  const T Fc[4] = {mbar, fma(w, A, pbar), w * C, w * g * X}, Gc[4] = {nbar, w * C, fma(w, K - A, pbar), w * g * Y};
  // eq. (2D-equ-int-approximation); the average equation in FP64 (its flux differences telescope)
  const double idx = P.crdx.d, idy = P.crdy.d;
  const T tidx = pc<T>(P.crdx), tidy = pc<T>(P.crdy);
  const bool fk = S.mask[cell] != 0 && (P.persist || S.Lout);
  const bool fn = P.persist && S.maskN && S.maskN[cell] != 0;
  const bool first = S.cA == 0.0;                    // U^(1) = U' + dt L: no U^n term
  bool finite = true;
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    if (v < v0 || v >= v1) continue;
    double L[3];
    const T Fp = xp[0][v], Fm = xm[0][v], Gp = yp[0][v], Gm = ym[0][v];
    L[0] = -fma(to_f64(Fp) - to_f64(Fm), idx, (to_f64(Gp) - to_f64(Gm)) * idy);
    L[1] = to_f64(fma(fma(T(-0.5), Fp + Fm, Fc[v]), tidx, (ym[1][v] - yp[1][v]) * tidy));
    L[2] = to_f64(fma(fma(T(-0.5), Gp + Gm, Gc[v]), tidy, (xm[1][v] - xp[1][v]) * tidx));
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      const long long si = (long long)(v * 3 + m) * P.plane + so;
      const double uin = (m > 0 && fk) ? S.Mod[(long long)(v * 2 + m - 1) * P.plane + so] : src.uin(P, S, v * 3 + m, i, j);
      if (S.Lout) {
        S.Lout[si] = L[m];
        if (S.Umod) S.Umod[si] = uin;
        continue;
      }
      double r;
      if (first) {
        r = fma(S.dt, L[m], uin);
      } else {
        const double un = (m > 0 && fn) ? S.ModN[(long long)(v * 2 + m - 1) * P.plane + so] : src.un(P, S, v * 3 + m, i, j);
        r = fma(S.cA, un, S.cB * fma(S.dt, L[m], uin));
      }
      S.Uout[si] = r;
      if (m == 0) newavg[v] = r;
      finite = finite && ((__double_as_longlong(r) >> 52) & 0x7FF) != 0x7FF;
    }
  }
  return finite;
}

template <typename T, typename Src>
__device__ __forceinline__ void update_cell_lean(const Prob& P, const Src& src, const Rk& S, int i, int j,
                                                 const T (&xm)[4][4], const T (&xp)[4][4], const T (&ym)[4][4],
                                                 const T (&yp)[4][4]) {
  double newavg[4];
  const bool finite = combine_lean<T>(P, src, S, i, j, quad_lean<T>(P, src, i, j), xm, xp, ym, yp, 0, 4, newavg);
  if (S.Lout || j < P.jlo || j >= P.jhi) return;
  if (!finite) atomicOr(S.status, ST_NONFINITE);
  if (nonphysical(newavg[0], newavg[1], newavg[2], newavg[3])) atomicOr(S.status, ST_NONPOSITIVE);
}

// Face fluxes of the TXV x TYV tile at (i0, j0) into shared memory, points t0,
// t0 + step, ... below t1 of tile_points.
// A face flux at one Gauss-Lobatto point per iteration, by one
// call site, so that a face shared by two tiles gets bitwise the same flux
// from both (the flux differences then telescope exactly in FP64).
// xf[r][c] is the face left of cell (i0 + c, j0 + r); yf[r][c] the face below it.
template <int TXV, int TYV>
__host__ __device__ constexpr int tile_points(bool above) { return (TXV + 1) * TYV * 4 + TXV * (TYV + 1) * 4 - (above ? TXV * 4 : 0); }

template <typename T, int NV, int TXV, int TYV, bool SOLID, bool SOFT, typename Src>
__device__ __forceinline__ void tile_fluxes(const Prob& P, const Src& src, int i0, int j0, int t0, int t1, int step,
                                            T (&xf)[TYV][TXV + 1][4][NV], T (&yf)[TYV + 1][TXV][4][NV], bool above) {
  constexpr int NXP = (TXV + 1) * TYV * 4;
  // a tile whose faces all join cells inside the grid (no image, no solid cell):
  // the point values at fixed offsets
  const bool tin = Src::staged || ((!SOLID || P.sol_j == 0) && i0 >= 1 && i0 + TXV < P.nx && j0 >= 1 && j0 + TYV < P.ny);
  for (int t = t0; t < t1; t += step) {
    const int f = above && t >= NXP ? t + TXV * 4 : t;
    // the face's GL point q, its slot (c, r) in the tile, its two cells a
    // (left / below) and b (right / above) and their point indices
    const bool xd = f < NXP;
    const int g = xd ? f : f - NXP, q = g & 3, face = g >> 2;
    const int c = xd ? face % (TXV + 1) : face % TXV, r = xd ? face / (TXV + 1) : face / TXV;
    const int aI = xd ? i0 + c - 1 : i0 + c, aJ = xd ? j0 + r : j0 + r - 1;
    const int bI = xd ? aI + 1 : aI, bJ = xd ? aJ : aJ + 1;
    const int ka = xd ? 3 : q, la = xd ? q : 3, kb = xd ? 0 : q, lb = xd ? q : 0;
    T uL[NV], uR[NV];
    bool wall = false;
    if (tin) {
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        uL[v] = src.g(P, v, ka * 4 + la, aI, aJ);
        uR[v] = src.g(P, v, kb * 4 + lb, bI, bJ);
      }
    } else if constexpr (!Src::staged) {
      const T* __restrict__ G = src.G;
      if (aJ >= P.ny || aI >= P.nx) continue;
      const bool sa = SOLID && P.sol_j > 0 && is_solid(P, aI, aJ), sb = SOLID && P.sol_j > 0 && is_solid(P, bI, bJ);
      // a face no fluid cell uses (solid on one side, solid or outside on the
      // other) is skipped: only solid cells would read it, and they are not updated
      if (SOLID && P.sol_j > 0 && (sa || aI < 0 || aJ < 0) && (sb || bI >= P.nx || bJ >= P.ny)) continue;
      if (!sa) gl_state<T, NV>(P, G, image(P, aI, aJ), ka, la, uL);
      if (!sb) gl_state<T, NV>(P, G, image(P, bI, bJ), kb, lb, uR);
      // a face shared with a solid cell: the outer state is the reflection of
      // the fluid side's own (the wall-normal momentum negated)
      const int wn = xd ? 1 : 2;
      if (sb && !sa) {
#pragma unroll
        for (int v = 0; v < NV; ++v) uR[v] = v == wn ? -uL[v] : uL[v];
      }
      if (sa && !sb) {
#pragma unroll
        for (int v = 0; v < NV; ++v) uL[v] = v == wn ? -uR[v] : uR[v];
      }
      wall = sa || sb;
    }
    face_flux<T, NV, SOFT>(P, uL, uR, xd, wall, xd ? xf[r][c][q] : yf[r][c][q]);
  }
}

// Face integrals (eq. (integral2), (integral3)), once per face: point slots 0 and 1
// become the mean and the first moment along the face.
template <typename T, int TXV, int TYV>
__device__ __forceinline__ void tile_integrals(int tid, int step, T (&xf)[TYV][TXV + 1][4][4],
                                               T (&yf)[TYV + 1][TXV][4][4], bool above) {
  constexpr int NXF = (TXV + 1) * TYV * 4;
  for (int t = tid; t < NXF + TXV * (TYV + 1) * 4 - (above ? TXV * 4 : 0); t += step) {
    const int f = above && t >= NXF ? t + TXV * 4 : t;
    const int g = (f < NXF ? f : f - NXF) >> 2, v = f & 3;
    T* q = f < NXF ? &xf[0][0][0][0] + g * 16 + v : &yf[0][0][0][0] + g * 16 + v;
    const T f0 = q[0], f1 = q[4], f2 = q[8], f3 = q[12];
    q[0] = fma(T(5.0 / 12.0), f1 + f2, T(1.0 / 12.0) * (f0 + f3));
    q[4] = fma(T(5.0 / 12.0 * 0.22360679774997896964), f2 - f1, T(1.0 / 24.0) * (f3 - f0));
  }
}

// Step 3 for the TXV x TYV tile at (i0, j0): face fluxes into shared memory, then
// quadrature, L(U) and the Runge-Kutta combination per cell.  tid = ty*TXV + tx.
// above: the block has just done the tile below (its top faces are reused).
// SOLID: the handle may have a solid block (FP64 2D Euler only); without it the
// wall-face code is not compiled in (the batched kernel runs at the register limit).
template <typename T, int NV, int TXV, int TYV, bool SOLID = false, typename Src = GlobalSrc<T>>
__device__ __forceinline__ void update2d_tile(const Prob& P, const Src& src, const Rk& S, int i0, int j0,
                                              int tid, T (&xf)[TYV][TXV + 1][4][NV], T (&yf)[TYV + 1][TXV][4][NV],
                                              bool above = false) {
  const int tx = tid % TXV, ty = tid / TXV;
  const int i = i0 + tx, j = j0 + ty;
  const bool live = i < P.nx && j < P.ny;
  __syncthreads();   // the shared arrays may still be read for a previous tile
  if (above) {       // the tile below was this block's last: its top faces are this one's bottom faces
    for (int q = tid; q < TXV * 4 * NV; q += TXV * TYV) (&yf[0][0][0][0])[q] = (&yf[TYV][0][0][0])[q];
    __syncthreads();
  }
  tile_fluxes<T, NV, TXV, TYV, SOLID, true>(P, src, i0, j0, tid, tile_points<TXV, TYV>(above), TXV * TYV, xf, yf, above);
  __syncthreads();
  if constexpr (NV == 4 && lean<T>::value) {
    tile_integrals<T, TXV, TYV>(tid, TXV * TYV, xf, yf, above);
    __syncthreads();
  }
  if (!live) return;
  if (SOLID && P.sol_j > 0 && is_solid(P, i, j)) {   // solid cells are not updated: the state passes through
    if (!S.Lout) {
#pragma unroll 1
      for (int q = 0; q < NV * 3; ++q) {
        const long long si = (long long)q * P.plane + (long long)j * P.pitch + i;
        S.Uout[si] = S.Uin[si];
        if (S.U32out) S.U32out[si] = f32_rn(S.Uin[si]);
      }
    } else {
#pragma unroll 1
      for (int q = 0; q < NV * 3; ++q) {
        const long long si = (long long)q * P.plane + (long long)j * P.pitch + i;
        S.Lout[si] = 0.0;
        if (S.Umod) S.Umod[si] = S.Uin[si];
      }
    }
    return;
  }
  if constexpr (NV == 4 && lean<T>::value) {
    update_cell_lean<T>(P, src, S, i, j, xf[ty][tx], xf[ty][tx + 1], yf[ty][tx], yf[ty + 1][tx]);
  } else {
  // face integrals (eq. (integral2), (integral3)) and the cell quadrature (eq. (integral1))
  T Fp[NV], Fm[NV], Fpe[NV], Fme[NV], Gp[NV], Gm[NV], Gpx[NV], Gmx[NV], Fc[NV], Gc[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) Fp[v] = Fm[v] = Fpe[v] = Fme[v] = Gp[v] = Gm[v] = Gpx[v] = Gmx[v] = Fc[v] = Gc[v] = T(0);
#pragma unroll
  for (int l = 0; l < 4; ++l) {
    const T w = gl_w<T>(l), we = gl_w<T>(l) * gl_x<T>(l);
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      Fp[v] += w * xf[ty][tx + 1][l][v];
      Fpe[v] += we * xf[ty][tx + 1][l][v];
      Fm[v] += w * xf[ty][tx][l][v];
      Fme[v] += we * xf[ty][tx][l][v];
      Gp[v] += w * yf[ty + 1][tx][l][v];
      Gpx[v] += we * yf[ty + 1][tx][l][v];
      Gm[v] += w * yf[ty][tx][l][v];
      Gmx[v] += we * yf[ty][tx][l][v];
    }
  }
  if constexpr (NV == 4 && sizeof(T) == 8) {
    // Euler, FP64: the 16 reciprocal densities with one division
    T rho[16], inv[16];
#pragma unroll
    for (int p = 0; p < 16; ++p) rho[p] = src.g(P, 0, p, i, j);
    batch_inverse_ranged<16, T>(rho, inv);
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int l = 0; l < 4; ++l) {
        T u[NV], fx[NV], gy[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) u[v] = src.g(P, v, k * 4 + l, i, j);
        euler_flux_inv<T, NV>(P, u, inv[k * 4 + l], 0, fx);
        euler_flux_inv<T, NV>(P, u, inv[k * 4 + l], 1, gy);
        const T w = gl_w<T>(k) * gl_w<T>(l);
#pragma unroll
        for (int v = 0; v < NV; ++v) { Fc[v] += w * fx[v]; Gc[v] += w * gy[v]; }
      }
  } else {
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int l = 0; l < 4; ++l) {
        T u[NV], fx[NV], gy[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) u[v] = src.g(P, v, k * 4 + l, i, j);
        phys_flux<T, NV>(P, u, 0, fx);
        phys_flux<T, NV>(P, u, 1, gy);
        const T w = gl_w<T>(k) * gl_w<T>(l);
#pragma unroll
        for (int v = 0; v < NV; ++v) { Fc[v] += w * fx[v]; Gc[v] += w * gy[v]; }
      }
  }
  // eq. (2D-equ-int-approximation); the average equation in FP64 from the
  // face integrals so that the flux differences telescope in every precision
  // (FP32 values widened by integer work: the FP64 pipe keeps only the sums)
  const double idx = P.crdx.d, idy = P.crdy.d;
  const T tidx = pc<T>(P.crdx), tidy = pc<T>(P.crdy);
  const long long so = (long long)j * P.pitch + i;
  const long long cell = (long long)j * P.nx + i;
  // modified first moments in the combination (persist), and always in the Umod output of Lout
  const bool fk = S.mask[cell] != 0 && (P.persist || S.Lout);
  const bool fn = P.persist && S.maskN && S.maskN[cell] != 0;
  // the first stage has no U^n term (cA = 0, cB = 1): U^(1) = U' + dt L
  const bool first = S.cA == 0.0;
  const bool owned = j >= P.jlo && j < P.jhi;
  double newavg[NV];
  bool finite = true;
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    double L[3];
    L[0] = -(to_f64(Fp[v]) - to_f64(Fm[v])) * idx - (to_f64(Gp[v]) - to_f64(Gm[v])) * idy;
    L[1] = to_f64(-(Fp[v] + Fm[v]) * T(0.5) * tidx + Fc[v] * tidx - (Gpx[v] - Gmx[v]) * tidy);
    L[2] = to_f64(-(Fpe[v] - Fme[v]) * tidx - (Gp[v] + Gm[v]) * T(0.5) * tidy + Gc[v] * tidy);
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      const long long si = (long long)(v * 3 + m) * P.plane + so;
      const double uin = (m > 0 && fk) ? S.Mod[(long long)(v * 2 + m - 1) * P.plane + so] : src.uin(P, S, v * 3 + m, i, j);
      if (S.Lout) {
        S.Lout[si] = L[m];
        if (S.Umod) S.Umod[si] = uin;
        continue;
      }
      double r;
      if (first) {
        r = fma(S.dt, L[m], uin);
      } else {
        const double un = (m > 0 && fn) ? S.ModN[(long long)(v * 2 + m - 1) * P.plane + so] : src.un(P, S, v * 3 + m, i, j);
        r = S.cA * un + S.cB * (uin + S.dt * L[m]);
      }
      S.Uout[si] = r;
      if (S.U32out) S.U32out[si] = f32_rn(r);
      if (m == 0) newavg[v] = r;
      // non-finite by the exponent field (integer work, no FP64 compare)
      finite = finite && ((__double_as_longlong(r) >> 52) & 0x7FF) != 0x7FF;
    }
  }
  if (!S.Lout && !finite && owned) atomicOr(S.status, ST_NONFINITE);
  if constexpr (NV == 4) {
    if (!S.Lout && P.eq == EQ_EULER && owned && nonphysical(newavg[0], newavg[1], newavg[2], newavg[3]))
      atomicOr(S.status, ST_NONPOSITIVE);
  }
  }
}

// fx64 and double-float: a block does `sweep` tiles, one above the other, and the
// faces between them once (8.1 instead of 9.1 fluxes per cell at 16 tiles; float,
// which waits for loads rather than for its arithmetic, measured 9 % slower so).
// fx64 at 2048^2: 15.2 ms per launch with hllc and the quadrature per point, 9.6
// with hllc_lean and update_cell_lean, 8.07 with the integer compares, the 5-operation
// root and the sweep, 5.8 with roots and reciprocals and 4.7 with the flux's products
// in integers (4.8 at 4 blocks per SM): 540 FP64 operations per cell of 1915 (mean of
// the three stages), the FP64 pipe still 80 % busy, 0.92 of the rate that chains of
// independent FMAs reach.  Double-float 5.2 -> 2.9 ms; at 1024^2 0.78 -> 0.74 with
// 5 blocks per SM for 4.
template <typename T, int NV, bool SOLID = false>
__global__ void __launch_bounds__(TX * TY, (std::is_same<T, float>::value ? 8
                                         : lean<T>::value ? (NV == 4 && !SOLID ? 5 : 4) : 3))
    update2d_kernel(const __grid_constant__ Prob P, const T* __restrict__ G, Rk S, int sweep) {
  __shared__ T xf[TY][TX + 1][4][NV];
  __shared__ T yf[TY + 1][TX][4][NV];
  const int i0 = blockIdx.x * TX, ja = blockIdx.y * sweep * TY, jb = min(ja + sweep * TY, P.ny);
  if (S.dtp) {
    S.dt = *S.dtp;
    if (S.dt < 0.0) {   // a skipped step (block-uniform): the state passes through unchanged
      const int i = i0 + threadIdx.x;
      for (int j = ja + threadIdx.y; j < jb; j += TY)
        if (i < P.nx && !S.Lout)
          for (int q = 0; q < NV * 3; ++q) {
            const long long si = (long long)q * P.plane + (long long)j * P.pitch + i;
            S.Uout[si] = S.Uin[si];
            if (S.U32out) S.U32out[si] = f32_rn(S.Uin[si]);
          }
      return;
    }
  }
  const int tid = threadIdx.y * TX + threadIdx.x;
  if constexpr (!std::is_same<T, float>::value) {
#pragma unroll 1
    for (int j0 = ja; j0 < jb; j0 += TY)
      update2d_tile<T, NV, TX, TY, SOLID>(P, GlobalSrc<T>{G}, S, i0, j0, tid, xf, yf, j0 > ja);
  } else {
    update2d_tile<T, NV, TX, TY, SOLID>(P, GlobalSrc<T>{G}, S, i0, ja, tid, xf, yf);
  }
}

// Few tiles (at most WIDE_TILES per SM): 256 threads a tile.  A tile's time is
// then one warp's chain of FP64 operations (64 clocks each, one warp per
// scheduler), not the pipe's rate, so the second half of the block takes the
// quadrature while the first does face fluxes, then the rest of these, and a cell's
// variables are shared by two threads.  The flux's products stay on the FP64
// pipe: it has room, and an integer product is the longer chain.  Bit for bit
// update2d_kernel's results.  Per launch, against update2d_kernel: 64^2 55 -> 39 us,
// 128^2 57 -> 39, 192^2 (1.9 tiles per SM) 72 -> 68; 224^2 (2.6) 89 -> 98, so the
// line is at two.
constexpr int WIDE_TILES = 2;
template <typename T>
__global__ void __launch_bounds__(2 * TX * TY, 2)
    update2d_wide_kernel(const __grid_constant__ Prob P, const T* __restrict__ G, Rk S) {
  constexpr int N = TX * TY;
  __shared__ T xf[TY][TX + 1][4][4];
  __shared__ T yf[TY + 1][TX][4][4];
  __shared__ Quad<T> qs[N];
  __shared__ double avg[4][N];
  __shared__ int bad[N];
  const int tid = threadIdx.x, c = tid % N, part = tid / N;
  const int i0 = blockIdx.x * TX, j0 = blockIdx.y * TY, i = i0 + c % TX, j = j0 + c / TX;
  const bool live = i < P.nx && j < P.ny;
  if (S.dtp) {
    S.dt = *S.dtp;
    if (S.dt < 0.0) {   // a skipped step (block-uniform): the state passes through unchanged
      if (live && !S.Lout)
        for (int q = part * 6; q < part * 6 + 6; ++q) {
          const long long si = (long long)q * P.plane + (long long)j * P.pitch + i;
          S.Uout[si] = S.Uin[si];
        }
      return;
    }
  }
  const GlobalSrc<T> src{G};
  // 9.1 flux points per cell, of which the half with the quadrature takes 3.1
  constexpr int first = 6 * N;
  if (part == 1 && live) qs[c] = quad_lean<T>(P, src, i, j);
  tile_fluxes<T, 4, TX, TY, false, false>(P, src, i0, j0, part * first + c, part ? tile_points<TX, TY>(false) : first, N,
                                          xf, yf, false);
  __syncthreads();
  tile_integrals<T, TX, TY>(tid, 2 * N, xf, yf, false);
  __syncthreads();
  bool finite = true;
  const int x = c % TX, y = c / TX;
  if (live) {
    double a[4];
    finite = combine_lean<T>(P, src, S, i, j, qs[c], xf[y][x], xf[y][x + 1], yf[y][x], yf[y + 1][x], 2 * part,
                             2 * part + 2, a);
    if (part) { avg[2][c] = a[2]; avg[3][c] = a[3]; bad[c] = !finite; }
    else { avg[0][c] = a[0]; avg[1][c] = a[1]; }
  }
  __syncthreads();
  if (part || !live || S.Lout || j < P.jlo || j >= P.jhi) return;
  if (!finite || bad[c]) atomicOr(S.status, ST_NONFINITE);
  if (nonphysical(avg[0][c], avg[1][c], avg[2][c], avg[3][c])) atomicOr(S.status, ST_NONPOSITIVE);
}

// Tiles per block: as many as leave six waves of 4 blocks per SM (the kernels hold
// 3 in plain double, 4 with the solid block, 5 in fx64 and double-float: five waves or
// more), at most 16; small grids keep one, their blocks must reach every SM first.
template <typename T>
inline int update_sweep(const Prob& P) {
  if (std::is_same<T, float>::value) return 1;
  const long long tiles = (long long)((P.nx + TX - 1) / TX) * ((P.ny + TY - 1) / TY);
  return (int)std::max<long long>(1, std::min<long long>(16, tiles / (6LL * P.nsm * 4)));
}

// ---------------------------------------------------------------- TMA-staged update (FP32 form)
// An interior tile loads its own point values (a 32 x 4 x 64-plane box from
// cell (i0, j0), 32 KB) with one cp.async.bulk.tensor into shared memory,
// completing on an mbarrier; the halo points and the stage states come from
// global memory, and tiles at the grid's edges take the global-memory path
// (boundary images).  An option (hweno_set_tma): with 52 KB of shared memory a
// block, 4 blocks fit an SM against the global kernel's 8, and the global
// kernel measured faster (1.07 against 1.46 ms per 2048^2 launch; a 40 x 6 box
// with the halo and both stage states in shared memory, 2 blocks per SM: 1.63).
constexpr unsigned GBOX_BYTES = GBX * GBY * 64 * 4;
constexpr unsigned TMA_SMEM = GBOX_BYTES + 128;
constexpr unsigned long long MBAR_POLL_LIMIT = 1ull << 22;
static_assert(GBX == TX && GBY == TY, "the box covers one update tile");

__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void tma_load3d(void* dst, const CUtensorMap* map, int x, int y, int z, unsigned bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
      :: "r"(smem_u32(dst)), "l"((unsigned long long)map), "r"(x), "r"(y), "r"(z), "r"(bar) : "memory");
}

// Phase `parity` of the mbarrier at `bar` completed; at most `limit` polls, false if the wait gave up.
__device__ __forceinline__ bool mbar_wait(unsigned bar, unsigned parity, unsigned long long limit) {
  for (unsigned long long k = 0; k < limit; ++k) {
    unsigned done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(done) : "r"(bar), "r"(parity) : "memory");
    if (done) return true;
  }
  return false;
}

__global__ void __launch_bounds__(TX * TY, 4) update2d_tma_kernel(Prob P, const float* __restrict__ G, Rk S,
                                                                  const __grid_constant__ CUtensorMap tmG) {
  __shared__ float xf[TY][TX + 1][4][4];
  __shared__ float yf[TY + 1][TX][4][4];
  extern __shared__ __align__(128) unsigned char dsm[];
  const int tid = threadIdx.y * TX + threadIdx.x;
  const int i0 = blockIdx.x * TX, j0 = blockIdx.y * TY;
  if (S.dtp) {
    S.dt = *S.dtp;
    if (S.dt < 0.0) {   // a skipped step (block-uniform): the state passes through unchanged
      const int i = i0 + threadIdx.x, j = j0 + threadIdx.y;
      if (i < P.nx && j < P.ny)
        for (int q = 0; q < 12; ++q) {
          const long long si = (long long)q * P.plane + (long long)j * P.pitch + i;
          S.Uout[si] = S.Uin[si];
          if (S.U32out) S.U32out[si] = f32_rn(S.Uin[si]);
        }
      return;
    }
  }
  if (!(i0 >= 1 && i0 + TX < P.nx && j0 >= 1 && j0 + TY < P.ny)) {
    update2d_tile<float, 4, TX, TY>(P, GlobalSrc<float>{G}, S, i0, j0, tid, xf, yf);
    return;
  }
  float* gs = reinterpret_cast<float*>(dsm);
  const unsigned bar = smem_u32(dsm + GBOX_BYTES);
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(bar) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (tid == 0) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(bar), "r"(GBOX_BYTES) : "memory");
    tma_load3d(gs, &tmG, i0, j0, 0, bar);   // i0 is a multiple of 32 floats (16-byte aligned)
  }
  if (!mbar_wait(bar, 0, MBAR_POLL_LIMIT)) {
    // gave up: report, wait (bounded) for the copies still in flight, skip the tile
    if (tid == 0) atomicOr(S.status, ST_TIMEOUT);
    mbar_wait(bar, 0, MBAR_POLL_LIMIT);
    return;
  }
  update2d_tile<float, 4, TX, TY, false, StagedSrc>(P, StagedSrc{gs, G, i0, j0}, S, i0, j0, tid, xf, yf);
}

// The TMA update kernel needs more than 48 KB of dynamic shared memory.
[[maybe_unused]] bool set_update_tma_attribute() {
  return cudaFuncSetAttribute(update2d_tma_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TMA_SMEM) ==
         cudaSuccess;
}

}  // namespace
}  // namespace hw

#include "hweno_fused.cuh"

namespace hw {
namespace {

// Fixed-state ghosts and the solid block are supported for 2D Euler in FP64 without the
// learned indicator (the library rejects other combinations), so only fx64's split kernel
// carries the FIX variant.
template <typename T, int NV, int MODE>
void launch_rec2d(int blocks, cudaStream_t st, const Prob& P, const Weights<T>& W, const typename rows2d<T>::type& Bt,
                  const double* U, const uint8_t* mask, const double* Mod, const int* list, const int* count, T* G,
                  T* aux, unsigned long long* rerec, const float* U32 = nullptr) {
  if constexpr (std::is_same<T, float>::value) {
    if (U32) {   // FP32 form with the float copy of the state: no per-moment conversion
      rec2d_kernel<T, NV, MODE, true><<<blocks, RB, 0, st>>>(P, W, Bt, U, mask, Mod, list, count, G, aux, rerec, U32);
      return;
    }
  }
  if constexpr (NV == 4 && fixed2d<T>::value) {
    const int sb = MODE == REC_FLAGGED ? blocks : (int)(((long long)P.nx * P.ny + 31) / 32);
    if constexpr (std::is_same<T, fx64>::value && MODE != REC_MIXED) {
      if (P.fixtab || P.sol_j > 0) {
        rec2d_split_kernel<T, MODE, true><<<sb, RB, 0, st>>>(P, W, Bt, U, mask, Mod, list, count, G, aux, rerec);
        return;
      }
    }
    rec2d_split_kernel<T, MODE><<<sb, RB, 0, st>>>(P, W, Bt, U, mask, Mod, list, count, G, aux, rerec);
  } else {
    rec2d_kernel<T, NV, MODE><<<blocks, RB, 0, st>>>(P, W, Bt, U, mask, Mod, list, count, G, aux, rerec);
  }
}

template <typename T, int NV>
void stage_t(const Prob& P, const HostTabs& HT, const Weights<T>& W, const Beta2<T>& Btf, const Bufs& B,
             const StageCall& S, cudaStream_t st) {
  const typename rows2d<T>::type* rows;   // Btf serves the fused kernel, rows the pipeline's
  if constexpr (is_df64<T>::value) rows = &HT.b2d;
  else rows = &Btf;
  const typename rows2d<T>::type& Bt = *rows;
  if constexpr (NV == 4 && !std::is_same<T, double>::value) {
    if (fused_applies(P, NV)) {   // the whole stage in one launch
      Rk r{S.Uin, S.Un, S.Uout, S.mask, S.Mod, S.maskN, S.ModN, S.dt, S.cA, S.cB, S.Lout, S.Umod, B.status, S.dtp};
      FzOut o{S.mask, S.Mod, S.aleph, B.rerec};
      if (B.prof) B.prof->begin(5, st);
      launch_fused2d<T>(P, W, Btf, r, o, st);
      if (B.prof) B.prof->end(st);
      return;
    }
  }
  const long long ncell = (long long)P.nx * P.ny;
  int* cnt = B.count + S.stage;
  cudaMemsetAsync(cnt, 0, sizeof(int), st);
  const int rblocks = (int)((ncell + RB - 1) / RB);
  const int fblocks = (int)std::min<long long>(rblocks, (long long)P.nsm * 8);
  const dim3 blk(TX, TY), grd((P.nx + TX - 1) / TX, (P.ny + TY - 1) / TY);
  bool learned = false;
  if constexpr (NV == 4) {
    learned = P.indicator == IND_MLP;
    if (learned) {
      // Learned indicator first (moments only): confident cells are decided and
      // modified before Step 1, which then reconstructs them from the modified
      // moments; KXRCF decides the rest from the Step-1 point values, and only
      // the cells it flags are reconstructed again.
      int* ucnt = B.und_count + S.stage;
      cudaMemsetAsync(ucnt, 0, sizeof(int), st);
      if (B.prof) B.prof->begin(4, st);
      run_mlpre2d(P, B.mlp, B.mlp_conf, S.Uin, S.mask, S.Mod, B.und, ucnt, B.mlp_stats, B.mlp_prob, st);
      if (B.prof) B.prof->end(st);
      if (B.prof) B.prof->begin(0, st);
      launch_rec2d<T, NV, REC_MIXED>(rblocks, st, P, W, Bt, S.Uin, S.mask, S.Mod, nullptr, nullptr, (T*)B.G,
                                     (T*)B.aux, nullptr);
      if (B.prof) B.prof->end(st);
      if (B.prof) B.prof->begin(1, st);
      fallback2d_kernel<T, NV><<<fblocks, RB, 0, st>>>(P, S.Uin, (const T*)B.G, (const T*)B.aux, B.und, ucnt,
                                                       S.mask, S.Mod, B.list, cnt, S.aleph);
      if (B.prof) B.prof->end(st);
    }
  }
  if (!learned) {
    if (B.prof) B.prof->begin(0, st);
    launch_rec2d<T, NV, REC_PLAIN>(rblocks, st, P, W, Bt, S.Uin, nullptr, nullptr, nullptr, nullptr, (T*)B.G,
                                   (T*)B.aux, nullptr, S.U32in);
    if (B.prof) B.prof->end(st);
    if (B.prof) B.prof->begin(1, st);
    flag2d_kernel<T, NV><<<grd, blk, 0, st>>>(P, S.Uin, (const T*)B.G, (const T*)B.aux, S.mask, S.Mod, B.list,
                                              cnt, S.aleph);
    if (B.prof) B.prof->end(st);
  }
  if (P.indicator != IND_NONE) {
    if (B.prof) B.prof->begin(2, st);
    launch_rec2d<T, NV, REC_FLAGGED>(fblocks, st, P, W, Bt, S.Uin, S.mask, S.Mod, B.list, cnt, (T*)B.G, nullptr,
                                     B.rerec, S.U32in);
    if (B.prof) B.prof->end(st);
  }
  Rk r{S.Uin, S.Un, S.Uout, S.mask, S.Mod, S.maskN, S.ModN, S.dt, S.cA, S.cB, S.Lout, S.Umod, B.status, S.dtp,
       std::is_same<T, float>::value ? S.U32out : nullptr};
  if (B.prof) B.prof->begin(3, st);
  const int sweep = update_sweep<T>(P);
  const dim3 sgrd(grd.x, (grd.y + sweep - 1) / sweep);
  if constexpr (NV == 4 && std::is_same<T, fx64>::value) {
    if (P.sol_j == 0 && (long long)grd.x * grd.y <= (long long)WIDE_TILES * P.nsm)
      update2d_wide_kernel<T><<<grd, 2 * TX * TY, 0, st>>>(P, (const T*)B.G, r);
    else if (P.sol_j > 0) update2d_kernel<T, NV, true><<<sgrd, blk, 0, st>>>(P, (const T*)B.G, r, sweep);
    else update2d_kernel<T, NV><<<sgrd, blk, 0, st>>>(P, (const T*)B.G, r, sweep);
  } else if constexpr (NV == 4 && std::is_same<T, float>::value) {
    if (B.tmG && !S.Lout)
      update2d_tma_kernel<<<grd, blk, TMA_SMEM, st>>>(P, (const float*)B.G, r, *B.tmG);
    else
      update2d_kernel<T, NV><<<sgrd, blk, 0, st>>>(P, (const T*)B.G, r, sweep);
  } else {
    update2d_kernel<T, NV><<<sgrd, blk, 0, st>>>(P, (const T*)B.G, r, sweep);
  }
  if (B.prof) B.prof->end(st);
}

// ---------------------------------------------------------------- batched problems
//
// Work items of all problems form one list per phase (128-cell rows for the
// per-cell phases, update tiles for the flux phase).  A stage runs a launch per
// phase, or one persistent cooperative launch whose resident blocks stride over
// the lists, phases separated by a grid barrier.  The barrier's wait is bounded:
// past the limit the block records ST_TIMEOUT and continues (the host reports
// HWENO_ETIMEOUT), so no wait can hang the GPU.

// nblocks: arrivals that release the barrier; limit: polls before the wait gives up.
__device__ __forceinline__ void grid_barrier(unsigned* bar, unsigned nblocks, unsigned* status,
                                             unsigned long long limit) {
  __syncthreads();
  if (threadIdx.x == 0) {
    volatile unsigned* vgen = bar + 1;
    const unsigned gen = *vgen;
    __threadfence();
    const unsigned arrived = atomicAdd(bar, 1u);
    if (arrived == nblocks - 1) {
      atomicExch(bar, 0u);
      __threadfence();
      atomicAdd(bar + 1, 1u);
    } else {
      unsigned long long spins = 0;
      while (*vgen == gen) {
        if (++spins > limit) {
          atomicOr(status, ST_TIMEOUT);
          break;
        }
        __nanosleep(64);
      }
    }
    __threadfence();
  }
  __syncthreads();
}

// One work item of each phase; tid 0 .. RB - 1.  P: the problem's description
// (shared memory), Q its entry.
__device__ __forceinline__ void batch_speeds_item(const BatchStage& A, const Prob& P, const BProb& Q, int p, int it,
                                                  int tid, bool filter) {
  const double* U = A.Uin + Q.uoff;
  const int cell = (it - Q.rec_first) * RB + tid;
  double sx = 0.0, sy = 0.0;
  bool take = cell < P.nx * P.ny;
  const int i = cell % P.nx, j = cell / P.nx;
  if (take && filter) {   // only cells whose FP32 upper bound reaches the largest lower bound
    float lo[2], hi[2];
    speed_bounds(P, U, i, j, lo, hi);
    take = !(hi[0] < __uint_as_float(A.bounds[2 * p]) && hi[1] < __uint_as_float(A.bounds[2 * p + 1]));
  }
  if (take) {
    const double rho = U[sidx(P, 0, 0, i, j)];
    const double mu = U[sidx(P, 1, 0, i, j)] / rho, nu = U[sidx(P, 2, 0, i, j)] / rho;
    const double pr = (P.gamma - 1.0) * (U[sidx(P, 3, 0, i, j)] - 0.5 * rho * (mu * mu + nu * nu));
    cell_speeds(P, rho, mu, nu, pr, sx, sy);
  }
  if (!__any_sync(0xffffffffu, take)) return;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    sx = fmax(sx, __shfl_down_sync(0xffffffffu, sx, o));
    sy = fmax(sy, __shfl_down_sync(0xffffffffu, sy, o));
  }
  if ((tid & 31) == 0) {   // non-negative doubles order like their bit patterns
    atomicMax(A.speeds + 2 * p, (unsigned long long)__double_as_longlong(sx));
    atomicMax(A.speeds + 2 * p + 1, (unsigned long long)__double_as_longlong(sy));
  }
}

__device__ __forceinline__ double batch_dt(const BatchStage& A, const Prob& P, int p) {
  if (A.dt_in) return A.dt_in[p];
  const double ax = __longlong_as_double((long long)A.speeds[2 * p]);
  const double ay = __longlong_as_double((long long)A.speeds[2 * p + 1]);
  const double r = ax / P.dx + ay / P.dy;
  return (r > 0.0 && isfinite(r)) ? A.cfl / r : 0.0;
}

// Quarters [q0, q1) of the item's 128 cells (fixed-point precisions: 32 cells at a
// time, a warp per variable and then per face).  S32: from the float copy of the state.
template <typename T, bool S32>
__device__ __forceinline__ void batch_rec_item(const BatchStage& A, const Prob& P, const BProb& Q, int it, int tid,
                                               const Weights<T>& W, const typename rows2d<T>::type& B, int q0 = 0,
                                               int q1 = 4) {
  T* G = (T*)A.G + Q.goff;
  T* aux = (T*)A.aux + Q.aoff;
  if constexpr (fixed2d<T>::value) {
    const int w = tid >> 5;
    for (int q = q0; q < q1; ++q) {
      const int cell = (it - Q.rec_first) * RB + q * 32 + (tid & 31), i = cell % P.nx, j = cell / P.nx;
      if (cell < P.nx * P.ny)
        rec2d_cell<T, 4, REC_PLAIN>(P, W, B, A.Uin + Q.uoff, nullptr, nullptr, i, j, G, aux, nullptr, w, w + 1);
      __syncthreads();
      if (cell < P.nx * P.ny) face_partials<T, 4>(P, G, aux, goff(P, i, j), w, w + 1);
    }
  } else {
    const int cell = (it - Q.rec_first) * RB + tid;
    if (cell < P.nx * P.ny)
      rec2d_cell<T, 4, REC_PLAIN, false, S32>(P, W, B, A.Uin + Q.uoff, nullptr, nullptr, cell % P.nx, cell / P.nx, G,
                                              aux, S32 ? A.U32in + Q.uoff : nullptr);
  }
}

template <typename T>
__device__ __forceinline__ void batch_flag_item(const BatchStage& A, const Prob& P, const BProb& Q, int p, int it,
                                                int tid) {
  const int cell = (it - Q.rec_first) * RB + tid;
  const bool valid = cell < P.nx * P.ny;
  const int i = cell % P.nx, j = cell / P.nx;
  const bool flag =
      valid && flag2d_cell<T>(P, A.Uin + Q.uoff, (const T*)A.G + Q.goff, (const T*)A.aux + Q.aoff, i, j, nullptr);
  warp_append<unsigned long long>(flag, ((unsigned long long)p << 32) | (unsigned)cell, A.list, A.count);
  if (valid) {
    A.mask[Q.coff + cell] = flag ? 1 : 0;
    if (flag) modify2d_cell<4>(P, A.Uin + Q.uoff, A.Mod + Q.moff, i, j);
  }
}

template <typename T, bool S32>
__device__ __forceinline__ void batch_rerec(const BatchStage& A, const Weights<T>& W,
                                            const typename rows2d<T>::type& B) {
  constexpr bool FXD = fixed2d<T>::value;
  const int n = *(volatile int*)A.count;
  // a thread per cell, or (fixed-point precisions) a warp per variable of 32 cells
  const int per = FXD ? 32 : RB, w = threadIdx.x >> 5;
  for (int t = blockIdx.x * per + (FXD ? threadIdx.x & 31 : threadIdx.x); t < n; t += gridDim.x * per) {
    const unsigned long long e = A.list[t];
    const int p = (int)(e >> 32), cell = (int)(e & 0xffffffffu);
    // after a barrier wait that gave up, an entry may not be written yet
    if (p < 0 || p >= A.nprob || cell < 0 || cell >= A.probs[p].P.nx * A.probs[p].P.ny) continue;
    const BProb& Q = A.probs[p];
    rec2d_cell<T, 4, REC_FLAGGED, false, S32>(Q.P, W, B, A.Uin + Q.uoff, A.mask + Q.coff, A.Mod + Q.moff,
                                              cell % Q.P.nx, cell / Q.P.nx, (T*)A.G + Q.goff, nullptr,
                                              S32 ? A.U32in + Q.uoff : nullptr, FXD ? w : 0, FXD ? w + 1 : 4);
  }
}

template <typename T, int TXV, int TYV>
__device__ __forceinline__ void batch_update_item(const BatchStage& A, const Prob& P, const BProb& Q, int p, int it,
                                                  int tid, double dt, T (&xf)[TYV][TXV + 1][4][4],
                                                  T (&yf)[TYV + 1][TXV][4][4]) {
  const int t = it - Q.upd_first;
  Rk S{A.Uin + Q.uoff, A.Un + Q.uoff, A.Uout + Q.uoff, A.mask + Q.coff, A.Mod + Q.moff,
       A.maskN ? A.maskN + Q.coff : nullptr, A.ModN ? A.ModN + Q.moff : nullptr, dt, A.cA, A.cB,
       nullptr, nullptr, A.pstatus + p, nullptr, std::is_same<T, float>::value && A.U32out ? A.U32out + Q.uoff : nullptr};
  update2d_tile<T, 4, TXV, TYV>(P, GlobalSrc<T>{(const T*)A.G + Q.goff}, S, (t % Q.tiles_x) * TXV,
                                (t / Q.tiles_x) * TYV, tid, xf, yf);
}

// The block's problem description in shared memory (the kernels' stores could
// alias a description in global memory, so its fields would be loaded again and again).
__device__ __forceinline__ void stage_prob(const BProb& Q, Prob* sp, int tid) {
  static_assert(sizeof(Prob) % 4 == 0, "copied by words");
  const int* src = reinterpret_cast<const int*>(&Q.P);
  for (int k = tid; k < (int)(sizeof(Prob) / 4); k += RB) reinterpret_cast<int*>(sp)[k] = src[k];
  __syncthreads();
}

// ---- a launch per phase
__global__ void __launch_bounds__(RB) batch_bounds_kernel(const __grid_constant__ BatchStage A) {
  const int it = blockIdx.x, p = A.rec_owner[it], tid = threadIdx.x;
  const BProb& Q = A.probs[p];
  const Prob& P = Q.P;
  const int cell = (it - Q.rec_first) * RB + tid;
  float lo[2] = {0.0f, 0.0f}, hi[2];
  if (cell < P.nx * P.ny) speed_bounds(P, A.Uin + Q.uoff, cell % P.nx, cell / P.nx, lo, hi);
#pragma unroll
  for (int k = 0; k < 2; ++k) {   // non-negative floats order like their bit patterns
    const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(lo[k]));
    if ((tid & 31) == 0) atomicMax(A.bounds + 2 * p + k, m);
  }
}

__global__ void __launch_bounds__(RB) batch_speeds_kernel(const __grid_constant__ BatchStage A) {
  const int it = blockIdx.x, p = A.rec_owner[it];
  batch_speeds_item(A, A.probs[p].P, A.probs[p], p, it, threadIdx.x, true);
}

__global__ void batch_dt_kernel(const __grid_constant__ BatchStage A) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p < A.nprob) A.dt_out[p] = batch_dt(A, A.probs[p].P, p);
}

template <typename T, bool S32>
__global__ void __launch_bounds__(RB, (is_df64<T>::value ? 4 : std::is_same<T, float>::value ? 8 : 5))
    batch_rec_kernel(const __grid_constant__ BatchStage A, const __grid_constant__ Weights<T> W,
                     const __grid_constant__ typename rows2d<T>::type B) {
  __shared__ Prob sp;
  const int it = fixed2d<T>::value ? blockIdx.x >> 2 : blockIdx.x, q = blockIdx.x & 3;
  const BProb& Q = A.probs[A.rec_owner[it]];
  stage_prob(Q, &sp, threadIdx.x);
  batch_rec_item<T, S32>(A, sp, Q, it, threadIdx.x, W, B, q, q + 1);
}

template <typename T>
__global__ void __launch_bounds__(RB) batch_flag_kernel(const __grid_constant__ BatchStage A) {
  __shared__ Prob sp;
  const int it = blockIdx.x, p = A.rec_owner[it];
  const BProb& Q = A.probs[p];
  stage_prob(Q, &sp, threadIdx.x);
  batch_flag_item<T>(A, sp, Q, p, it, threadIdx.x);
}

template <typename T, bool S32>
__global__ void __launch_bounds__(RB) batch_rerec_kernel(const __grid_constant__ BatchStage A,
                                                         const __grid_constant__ Weights<T> W,
                                                         const __grid_constant__ typename rows2d<T>::type B) {
  batch_rerec<T, S32>(A, W, B);
}

template <typename T, int TXV, int TYV>
__global__ void __launch_bounds__(TXV * TYV, (std::is_same<T, float>::value ? 7 : 4))
    batch_update_kernel(const __grid_constant__ BatchStage A) {
  __shared__ T xf[TYV][TXV + 1][4][4];
  __shared__ T yf[TYV + 1][TXV][4][4];
  __shared__ Prob sp;
  const int it = blockIdx.x, p = A.upd_owner[it];
  const BProb& Q = A.probs[p];
  stage_prob(Q, &sp, threadIdx.x);
  batch_update_item<T, TXV, TYV>(A, sp, Q, p, it, threadIdx.x, A.dt_out[p], xf, yf);
}

// ---- one persistent launch
template <typename T, int TXV, int TYV>
__global__ void __launch_bounds__(TXV * TYV) batch_stage_kernel(const __grid_constant__ BatchStage A,
                                                                const __grid_constant__ Weights<T> W,
                                                                const __grid_constant__ typename rows2d<T>::type B) {
  static_assert(TXV * TYV == RB, "tiles and rows use the same block");
  constexpr bool FP32 = std::is_same<T, float>::value;
  __shared__ T xf[TYV][TXV + 1][4][4];
  __shared__ T yf[TYV + 1][TXV][4][4];
  const int tid = threadIdx.x;
  const unsigned nb = gridDim.x;
  // CFL wave speeds of U^n (first stage, when the caller gives no dt)
  if (A.stage == 0 && !A.dt_in) {
    for (int it = blockIdx.x; it < A.n_rec; it += nb) {
      const int p = A.rec_owner[it];
      batch_speeds_item(A, A.probs[p].P, A.probs[p], p, it, tid, false);
    }
    grid_barrier(A.bar, nb + A.bar_extra, A.status, A.spin_limit);
  }
  // Step 1: every cell
  for (int it = blockIdx.x; it < A.n_rec; it += nb) {
    const BProb& Q = A.probs[A.rec_owner[it]];
    if (FP32 && A.U32in) batch_rec_item<T, FP32>(A, Q.P, Q, it, tid, W, B);
    else batch_rec_item<T, false>(A, Q.P, Q, it, tid, W, B);
  }
  grid_barrier(A.bar, nb + A.bar_extra, A.status, A.spin_limit);
  // Steps 2.1-2.2
  for (int it = blockIdx.x; it < A.n_rec; it += nb) {
    const int p = A.rec_owner[it];
    batch_flag_item<T>(A, A.probs[p].P, A.probs[p], p, it, tid);
  }
  grid_barrier(A.bar, nb + A.bar_extra, A.status, A.spin_limit);
  // Step 2.3: troubled cells
  if (FP32 && A.U32in) batch_rerec<T, FP32>(A, W, B);
  else batch_rerec<T, false>(A, W, B);
  grid_barrier(A.bar, nb + A.bar_extra, A.status, A.spin_limit);
  // Step 3: fluxes, quadrature, L, Runge-Kutta
  for (int it = blockIdx.x; it < A.n_upd; it += nb) {
    const int p = A.upd_owner[it];
    const BProb& Q = A.probs[p];
    const double dt = batch_dt(A, Q.P, p);
    if (A.stage == 0 && it == Q.upd_first && tid == 0) A.dt_out[p] = dt;
    batch_update_item<T, TXV, TYV>(A, Q.P, Q, p, it, tid, dt, xf, yf);
  }
}

// The persistent kernel holds every phase to the registers and shared memory of the
// largest and pays four grid barriers; a launch per phase measured faster at every
// size (ms per step, persistent / per phase: 4 problems of 13 k cells FP32
// 0.29 / 0.20, FP64 1.03 / 0.57; 64 problems of 3.8 M cells FP32 8.3 / 5.5, FP64
// 44 / 41; FP32 9.0 with its moments converted per gather).  The persistent form
// runs where the caller sets its barrier up (hweno_batch_set_barrier).
template <typename T, int TXV, int TYV>
cudaError_t launch_batch(const Weights<T>& W, const typename rows2d<T>::type& Bt, const BatchStage& S, int nsm,
                         cudaStream_t st) {
  if (!S.persistent) {
    if (S.stage == 0) {
      if (!S.dt_in) {
        batch_bounds_kernel<<<S.n_rec, RB, 0, st>>>(S);
        batch_speeds_kernel<<<S.n_rec, RB, 0, st>>>(S);
      }
      batch_dt_kernel<<<(S.nprob + 127) / 128, 128, 0, st>>>(S);
    }
    constexpr bool FP32 = std::is_same<T, float>::value;
    const bool copy = FP32 && S.U32in;
    if (copy) batch_rec_kernel<T, FP32><<<S.n_rec, RB, 0, st>>>(S, W, Bt);
    else batch_rec_kernel<T, false><<<fixed2d<T>::value ? 4 * S.n_rec : S.n_rec, RB, 0, st>>>(S, W, Bt);
    batch_flag_kernel<T><<<S.n_rec, RB, 0, st>>>(S);
    if (copy) batch_rerec_kernel<T, FP32><<<nsm * 8, RB, 0, st>>>(S, W, Bt);
    else batch_rerec_kernel<T, false><<<nsm * 8, RB, 0, st>>>(S, W, Bt);
    batch_update_kernel<T, TXV, TYV><<<S.n_upd, RB, 0, st>>>(S);
    return cudaGetLastError();
  }
  auto kern = batch_stage_kernel<T, TXV, TYV>;
  int per_sm = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, RB, 0);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(nsm * per_sm);
  cfg.blockDim = dim3(RB);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, S, W, Bt);
}

}  // namespace
}  // namespace hw
