// Reductions over the cell averages (FP64): the CFL wave speeds and the
// conservation totals.  Warp shuffles inside a block, one partial per block,
// then a single-block pass in a fixed order (deterministic for a given grid).
#include <math.h>

#include <algorithm>

#include "hweno_internal.h"

namespace hw {
namespace {

constexpr int RT = 256;       // threads per block (128 in the wave speeds of small grids)
constexpr int MAXB = 1024;    // blocks of the first pass (partials per quantity)

template <int K, int NT = RT>
__device__ __forceinline__ void block_reduce(double (&v)[K], bool is_max, double (*sm)[NT / 32]) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < K; ++k)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double w = __shfl_down_sync(0xffffffffu, v[k], o);
      v[k] = is_max ? fmax(v[k], w) : v[k] + w;
    }
  if (lane == 0)
#pragma unroll
    for (int k = 0; k < K; ++k) sm[k][wid] = v[k];
  __syncthreads();
  if (wid == 0) {
#pragma unroll
    for (int k = 0; k < K; ++k) {
      double x = lane < NT / 32 ? sm[k][lane] : 0.0;   // 0 is neutral for sums and for max of speeds
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const double w = __shfl_down_sync(0xffffffffu, x, o);
        x = is_max ? fmax(x, w) : x + w;
      }
      v[k] = x;
    }
  }
}

// The step length of hweno_advance on the device, from the wave-speed maxima:
// the CFL rule of the host's hweno_max_dt (same expressions), clipped to the
// remaining time; st[0] = t, st[1] = dt, st[2] = steps taken, st[3] = the time at
// the start of the step, par = {T, cfl, max_steps}.  dt = -1 marks a step to skip
// (done, step budget spent, or a non-physical average, which also sets
// ST_NONPOSITIVE and ST_NODT; the latter fails the call whatever the positivity switch).
__device__ __forceinline__ void advance_dt(const Prob& P, double ax, double ay, const double* __restrict__ par,
                                           double* __restrict__ st, unsigned* __restrict__ status) {
  const double T = par[0], cfl = par[1], maxs = par[2];
  double dtc;
  if (P.nmom == 2) dtc = ax > 0.0 ? cfl * P.dx / ax : INFINITY;
  else {
    const double r = ax / P.dx + ay / P.dy;
    dtc = r > 0.0 ? cfl / r : INFINITY;
  }
  const double t = st[0], rem = T - t;
  st[3] = t;
  double dt = -1.0;
  if (!(dtc > 0.0) || isnan(dtc)) {
    atomicOr(status, ST_NONPOSITIVE | ST_NODT);
  } else if (st[2] < maxs && rem > 1e-14 * fmax(1.0, fabs(T))) {
    dt = fmin(dtc, rem);
    st[0] = dtc >= rem ? T : t + dt;
    st[2] += 1.0;
  }
  st[1] = dt;
}

// The exact speeds of one cell average: |f'| (scalars) or |velocity| + sound speed
// (Euler) per direction.  A non-physical average yields +inf (dt = 0).  With the
// positivity check off the sound speed uses max(p, 0).
__device__ __forceinline__ void speeds_of(const Prob& P, const double* __restrict__ U, int i, int j, double& sx, double& sy) {
  if (P.eq == EQ_ADV) { sx = fabs(P.adv_a); sy = fabs(P.adv_b); }
  else if (P.eq == EQ_BURGERS) { sx = sy = fabs(U[sidx(P, 0, 0, i, j)]); }
  else {
    const double rho = U[sidx(P, 0, 0, i, j)];
    const double mu = U[sidx(P, 1, 0, i, j)] / rho;
    const double nu = P.nvar == 4 ? U[sidx(P, 2, 0, i, j)] / rho : 0.0;
    const double E = U[sidx(P, P.nvar - 1, 0, i, j)];
    const double p = (P.gamma - 1.0) * (E - 0.5 * rho * (mu * mu + nu * nu));
    cell_speeds(P, rho, mu, nu, p, sx, sy);
  }
}

// The largest speeds over the cells.  The last block to arrive (part[4 MAXB] counts them and returns to 0) reduces the
// blocks' partials to out[0..1], copies the status word to out[2] (the host then reads
// speeds and status at once) and, with par set, forms hweno_advance's step
// length: one launch where the partials, their reduction and the step length took
// three (each about 2 us of a small grid's step; a maximum is the same in any order).
// FILTER (Euler, large grids): a block first takes the largest lower bound of its
// cells from FP32 copies and then the exact FP64 speed, about 55 operations of the
// scarce pipe, only of cells whose upper bound reaches it: the same maximum (2^22
// cells in 1D: hweno_max_dt 0.44 -> 0.13 ms, of which 0.03 the host).
template <int NT, bool FILTER>
__global__ void __launch_bounds__(NT) wavespeed_kernel(const __grid_constant__ Prob P, const double* __restrict__ U,
                                                       double* __restrict__ part, double* __restrict__ out,
                                                       const double* __restrict__ par, double* __restrict__ st,
                                                       unsigned* __restrict__ status) {
  __shared__ double sm[2][NT / 32];
  __shared__ float fm[2][NT / 32];
  __shared__ bool last;
  double v[2] = {0.0, 0.0};
  const unsigned n = (unsigned)P.nx * (unsigned)(P.jhi - P.jlo), nx = P.nx;   // owned cells (below 2^31)
  const unsigned per = (n + gridDim.x - 1) / gridDim.x, t0 = min(n, per * blockIdx.x), t1 = min(n, t0 + per);
  [[maybe_unused]] float thr[2] = {0.0f, 0.0f};
  if constexpr (FILTER) {
    for (unsigned t = t0 + threadIdx.x; t < t1; t += NT) {
      const int i = t % nx, j = P.jlo + t / nx;
      if (P.sol_j > 0 && is_solid(P, i, j)) continue;
      float lo[2], hi[2];
      speed_bounds(P, U, i, j, lo, hi);
      thr[0] = fmaxf(thr[0], lo[0]);
      thr[1] = fmaxf(thr[1], lo[1]);
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) thr[k] = fmaxf(thr[k], __shfl_xor_sync(0xffffffffu, thr[k], o));
      if ((threadIdx.x & 31) == 0) fm[k][threadIdx.x >> 5] = thr[k];
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 2; ++k)
      for (int q = 0; q < NT / 32; ++q) thr[k] = fmaxf(thr[k], fm[k][q]);
  }
  for (unsigned t = t0 + threadIdx.x; t < t1; t += NT) {
    const int i = t % nx, j = P.jlo + t / nx;
    if (P.sol_j > 0 && is_solid(P, i, j)) continue;    // the step's block takes no part
    if constexpr (FILTER) {
      float lo[2], hi[2];
      speed_bounds(P, U, i, j, lo, hi);
      if (hi[0] < thr[0] && hi[1] < thr[1]) continue;
    }
    double sx, sy;
    speeds_of(P, U, i, j, sx, sy);
    v[0] = fmax(v[0], sx);
    v[1] = fmax(v[1], sy);
  }
  block_reduce<2, NT>(v, true, sm);
  if (threadIdx.x == 0) {
    part[blockIdx.x] = v[0];
    part[MAXB + blockIdx.x] = v[1];
    __threadfence();
    last = atomicInc(reinterpret_cast<unsigned*>(part + 4 * MAXB), gridDim.x - 1) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double w[2] = {0.0, 0.0};
  for (int b = threadIdx.x; b < gridDim.x; b += NT) {
    w[0] = fmax(w[0], __ldcg(part + b));
    w[1] = fmax(w[1], __ldcg(part + MAXB + b));
  }
  __syncthreads();   // sm is free again
  block_reduce<2, NT>(w, true, sm);
  if (threadIdx.x == 0) {
    out[0] = w[0];
    out[1] = w[1];
    out[2] = (double)*status;
    if (par) advance_dt(P, w[0], w[1], par, st, status);
  }
}

__global__ void __launch_bounds__(RT) totals_kernel(Prob P, const double* __restrict__ U, double* __restrict__ part) {
  __shared__ double sm[4][RT / 32];
  double v[4] = {0.0, 0.0, 0.0, 0.0};
  const long long n = (long long)P.nx * (P.jhi - P.jlo);   // owned rows
  for (long long t = (long long)blockIdx.x * RT + threadIdx.x; t < n; t += (long long)gridDim.x * RT) {
    const int i = (int)(t % P.nx), j = P.jlo + (int)(t / P.nx);
    if (P.sol_j > 0 && is_solid(P, i, j)) continue;
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (k < P.nvar) v[k] += U[sidx(P, k, 0, i, j)];
  }
  block_reduce<4>(v, false, sm);
  if (threadIdx.x == 0)
#pragma unroll
    for (int k = 0; k < 4; ++k) part[k * MAXB + blockIdx.x] = v[k];
}

// Single block: sum K rows of nb partials each into out[K].
template <int K>
__global__ void __launch_bounds__(RT) finish_kernel(const double* __restrict__ part, int nb, double* __restrict__ out) {
  __shared__ double sm[K][RT / 32];
  double v[K];
#pragma unroll
  for (int k = 0; k < K; ++k) {
    v[k] = 0.0;
    for (int b = threadIdx.x; b < nb; b += RT) v[k] += part[k * MAXB + b];
  }
  block_reduce<K>(v, false, sm);
  if (threadIdx.x == 0)
#pragma unroll
    for (int k = 0; k < K; ++k) out[k] = v[k];
}

int first_pass_blocks(const Prob& P) {
  const long long n = (long long)P.nx * (P.jhi - P.jlo);
  return (int)std::min<long long>(MAXB, (n + RT - 1) / RT);
}

// Fixed-state ghost table for the stage at time t (or, with dtp set, at
// *tn + c * *dtp read on the device; a skipped step, *dtp < 0, leaves it).
// Products and sums are rounded separately (no fused multiply-add), as the
// host computes the same positions and times.
__global__ void fixfill_kernel(FixSpec F, double* __restrict__ tab, double t, const double* __restrict__ tn,
                               const double* __restrict__ dtp, double c) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= 4 * F.fixlen) return;
  if (dtp) {
    const double dt = *dtp;
    if (dt < 0.0) return;
    t = __dadd_rn(*tn, __dmul_rn(c, dt));
  }
  const int side = q / F.fixlen, pos = q % F.fixlen - 1;
  const double at = __dmul_rn((double)pos + 0.5, side < 2 ? F.dy : F.dx);
  const double pc = __dadd_rn(side < 2 ? F.y0 : F.x0, at);
  const double* src = nullptr;
  if (pos <= F.n[side]) {
    if (F.seg[side] && pc < __dadd_rn(F.c0[side], __dmul_rn(F.speed[side], t))) src = F.a[side];
    else if (F.inflow[side]) src = F.b[side];
  }
#pragma unroll
  for (int v = 0; v < 4; ++v) tab[4 * (long long)q + v] = src ? src[v] : 0.0;
}

// The float copy of rows [j0, j0 + nrows) of every moment plane (FP32 form):
// each state value rounded to nearest by integer work, as the update kernel
// rounds the values it writes.
__global__ void shadow32_kernel(Prob P, const double* __restrict__ U, float* __restrict__ U32, int j0, int nrows) {
  const long long per = (long long)nrows * P.nx, n = (long long)P.nvar * P.nmom * per;
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
    const long long q = t / per, r = t % per;
    const long long si = q * P.plane + (long long)(j0 + r / P.nx) * P.pitch + r % P.nx;
    U32[si] = f32_rn(U[si]);
  }
}

}  // namespace

void run_shadow32(const Prob& P, const double* U, float* U32, int j0, int nrows, cudaStream_t st) {
  const long long n = (long long)P.nvar * P.nmom * nrows * P.nx;
  if (n <= 0) return;
  const int nb = (int)std::min<long long>((n + RT - 1) / RT, (long long)P.nsm * 16);
  shadow32_kernel<<<nb, RT, 0, st>>>(P, U, U32, j0, nrows);
}

void run_fixfill(const FixSpec& F, double* tab, double t, const double* tn, const double* dtp, double c,
                 cudaStream_t st) {
  const int n = 4 * F.fixlen;
  fixfill_kernel<<<(n + 127) / 128, 128, 0, st>>>(F, tab, t, tn, dtp, c);
}

int reduce_partials_len(const Prob&) { return 4 * MAXB + 1; }

void run_wavespeed(const Prob& P, const double* U, double* partials, double* out, const double* par, double* st,
                   unsigned* status, cudaStream_t s) {
  const long long n = (long long)P.nx * (P.jhi - P.jlo);
  // few cells: 128-thread blocks, one warp per scheduler of more SMs (the cells' FP64
  // divisions and roots issue at 2 per clock and SM); 64 threads doubled the blocks the
  // last one waits for (2D Burgers 161^2, 12 steps: 2.11 -> 2.09 ms)
  if (n <= 256LL * P.nsm)
    wavespeed_kernel<128, false><<<(int)std::min<long long>(MAXB, (n + 127) / 128), 128, 0, s>>>(P, U, partials, out, par,
                                                                                                st, status);
  else if (P.eq == EQ_EULER)
    wavespeed_kernel<RT, true><<<first_pass_blocks(P), RT, 0, s>>>(P, U, partials, out, par, st, status);
  else
    wavespeed_kernel<RT, false><<<first_pass_blocks(P), RT, 0, s>>>(P, U, partials, out, par, st, status);
}

void run_totals(const Prob& P, const double* U, double* partials, double* out, cudaStream_t st) {
  const int nb = first_pass_blocks(P);
  totals_kernel<<<nb, RT, 0, st>>>(P, U, partials);
  finish_kernel<4><<<1, RT, 0, st>>>(partials, nb, out);
}

}  // namespace hw
