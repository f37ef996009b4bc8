// Cell-wise kernels of the solver: ghost layers, conservative <-> primitive
// conversion, the CFL reduction, the flux-divergence + SSP-RK3 update and the
// MOOD counters.  Built with -fmad=false: every FP64 operation rounds once,
// in the order written, so that the FP64 path reproduces a plain IEEE
// evaluation of the same formulas bit for bit.
#include <cuda_runtime.h>

#include "fp64_pipes.cuh"
#include "ws_internal.h"

namespace ws {

namespace {

using fp64::divide;
using fp64::root;

constexpr int BS = 256;

inline int blocks_for(int64_t n, int bs = BS) {
  int64_t b = (n + bs - 1) / bs;
  if (b > (1LL << 30)) b = 1LL << 30;
  return (int)(b < 1 ? 1 : b);
}

// Sec. 2, Eq. (eos): rho e = Gamma p + Pi.
__device__ __forceinline__ void cons_to_prim(int ndim, const double* U, double* q) {
  double rho = U[0];
  double usq = 0.0;
  q[0] = rho;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    if (d < ndim) {
      double u = divide(U[1 + d], rho);
      q[1 + d] = u;
      usq = usq + u * u;
    }
  }
  double ke = (0.5 * rho) * usq;
  double E = U[1 + ndim], Gam = U[2 + ndim], Pi = U[3 + ndim];
  q[1 + ndim] = divide((E - ke) - Pi, Gam);
  q[2 + ndim] = Gam;
  q[3 + ndim] = Pi;
}

__device__ __forceinline__ double sound_speed2(double rho, double p, double Gam, double Pi) {
  return divide(((Gam + 1.0) * p) + Pi, Gam * rho);
}

__device__ __forceinline__ bool admissible(double rho, double p, double Gam, double Pi) {
  return (rho > 0.0) && (Gam > 0.0) && ((((Gam + 1.0) * p) + Pi) > 0.0);
}

// coordinates of linear index i in extents e0, e1 (x fastest), in 32-bit
// arithmetic where the index allows (a 64-bit division takes about 70
// instructions)
__device__ __forceinline__ void coords(int64_t i, int64_t e0, int64_t e1, int64_t c[3]) {
  if (i < (1LL << 31)) {
    const unsigned u = (unsigned)i, r = u / (unsigned)e0, z = r / (unsigned)e1;
    c[0] = u - r * (unsigned)e0;
    c[1] = r - z * (unsigned)e1;
    c[2] = z;
  } else {
    c[0] = i % e0;
    const int64_t r = i / e0;
    c[1] = r % e1;
    c[2] = r / e1;
  }
}

// atomicMax of the threads' values
__device__ __forceinline__ void block_max(unsigned long long b, unsigned long long* out) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    unsigned long long v = __shfl_xor_sync(0xffffffffu, b, o);
    b = v > b ? v : b;
  }
  __shared__ unsigned long long sm[32];
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0) sm[w] = b;
  __syncthreads();
  if (w == 0) {
    b = lane < (int)(blockDim.x >> 5) ? sm[lane] : 0ULL;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      unsigned long long v = __shfl_xor_sync(0xffffffffu, b, o);
      b = v > b ? v : b;
    }
    if (lane == 0) atomicMax(out, b);
  }
}

// The start of an RHS evaluation in one launch: ghost layers of U (of the
// cells with one coordinate outside the interior: the others are never read),
// primitives and sound speed of every cell the sweeps read and, with lmax,
// the CFL rate: max over the interior cells of sum_d (|u_d| + c)/dx_d.
// Non-negative doubles order like their bit patterns, so the maximum is an
// integer atomicMax; a NaN orders above +inf.  clear: a counter set to zero.
template <int NDIM>
__global__ void __launch_bounds__(BS) k_prep(const __grid_constant__ GridDev g, double* U, double* __restrict__ Q,
                                             unsigned long long* lmax, unsigned long long* clear) {
  constexpr int NV = NDIM + 4;
  follow_previous();
  if (clear && blockIdx.x == 0 && threadIdx.x == 0) *clear = 0ULL;
  unsigned long long best = 0ULL;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < g.N; i += (int64_t)gridDim.x * blockDim.x) {
    int64_t c[3];
    coords(i, g.P[0], g.P[1], c);
    int out = 0, flip = -1;
    int64_t src = i;
#pragma unroll
    for (int d = 0; d < NDIM; ++d) {
      const int64_t x = c[d] - NG;
      if (x >= 0 && x < g.n[d]) continue;
      ++out;
      const int kind = g.bc[d][x < 0 ? 0 : 1];
      int64_t m = x < 0 ? 0 : g.n[d] - 1;
      if (kind == WS_BC_PERIODIC) m = x < 0 ? x + g.n[d] : x - g.n[d];
      if (kind == WS_BC_REFLECTIVE) {
        m = x < 0 ? -1 - x : 2 * (int64_t)g.n[d] - 1 - x;
        flip = 1 + d;
      }
      src += (m - x) * g.st[d];
    }
    if (out > 1) continue;
    double u[NV], q[NV];
#pragma unroll
    for (int f = 0; f < NV; ++f) {
      u[f] = U[f * g.N + src];
      if (f == flip) u[f] = -u[f];
      if (out) U[f * g.N + i] = u[f];
    }
    cons_to_prim(NDIM, u, q);
    const double cs = root(sound_speed2(q[0], q[1 + NDIM], q[2 + NDIM], q[3 + NDIM]));
#pragma unroll
    for (int f = 0; f < NV; ++f) Q[f * g.N + i] = q[f];
    Q[NV * g.N + i] = cs;
    if (lmax && !out) {
      double lam = 0.0;
#pragma unroll
      for (int d = 0; d < NDIM; ++d) lam = lam + divide(fabs(q[1 + d]) + cs, g.dx[d]);
      const unsigned long long b = lam <= 0.0 ? 0ULL : (unsigned long long)__double_as_longlong(lam);
      best = b > best ? b : best;
    }
  }
  if (lmax) block_max(best, lmax);
}

__global__ void k_prim_to_cons(GridDev g, const double* __restrict__ Q, double* __restrict__ U) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < g.N; i += (int64_t)gridDim.x * blockDim.x) {
    int nd = g.ndim;
    double rho = Q[i];
    double usq = 0.0;
    U[i] = rho;
    for (int d = 0; d < nd; ++d) {
      double u = Q[(1 + d) * g.N + i];
      U[(1 + d) * g.N + i] = rho * u;
      usq = usq + u * u;
    }
    double ke = (0.5 * rho) * usq;
    double p = Q[(1 + nd) * g.N + i], Gam = Q[(2 + nd) * g.N + i], Pi = Q[(3 + nd) * g.N + i];
    U[(1 + nd) * g.N + i] = ((Gam * p) + Pi) + ke;
    U[(2 + nd) * g.N + i] = Gam;
    U[(3 + nd) * g.N + i] = Pi;
  }
}

__global__ void k_cons_to_prim_all(GridDev g, const double* __restrict__ U, double* __restrict__ Q) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < g.N; i += (int64_t)gridDim.x * blockDim.x) {
    double u[MAXV], q[MAXV];
    for (int f = 0; f < g.nv; ++f) u[f] = U[f * g.N + i];
    cons_to_prim(g.ndim, u, q);
    for (int f = 0; f < g.nv; ++f) Q[f * g.N + i] = q[f];
  }
}

__global__ void k_set_dt(double dt_fixed, double cfl, const unsigned long long* __restrict__ lmax,
                         double* __restrict__ dt, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    if (dt_fixed > 0.0)
      dt[i] = dt_fixed;
    else
      dt[i] = cfl / __longlong_as_double((long long)lmax[i]);
  }
}

// Sec. 3.1: L(U) summed over x, y, z, then the SSP-RK3 stage.
// stage -1: write L itself; 0, 1, 2: the three Shu-Osher stages.  Stage 0
// derives the step (dt_fixed, or cfl / *lmax) and leaves it in *dtp for the
// others.  Uout may alias Un or Us (each thread reads its cell before writing
// it).
struct UpdateArgs {
  GridDev g;
  int stage;
  const double *Un, *Us;
  double* Uout;
  const double* F[3];
  const double* u[3];
  double dt_fixed, cfl;
  const unsigned long long* lmax;
  double* dtp;
  double* dt_host;  // nullable, mapped host memory: receives the step, too
  unsigned long long* nbad;
};

template <int NDIM>
__global__ void __launch_bounds__(BS) k_update(const __grid_constant__ UpdateArgs a) {
  constexpr int NV = NDIM + 4;
  follow_previous();
  const GridDev& g = a.g;
  const double c13 = 1.0 / 3.0, c23 = 2.0 / 3.0;
  double dt = 0.0;
  if (a.stage == 0) {
    dt = a.dt_fixed > 0.0 ? a.dt_fixed : divide(a.cfl, __longlong_as_double((long long)*a.lmax));
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      *a.dtp = dt;
      if (a.dt_host) *a.dt_host = dt;
    }
  } else if (a.stage > 0) {
    dt = *a.dtp;
  }
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < g.ncell; t += (int64_t)gridDim.x * blockDim.x) {
    int64_t c[3];
    coords(t, g.n[0], g.n[1], c);
    const int64_t i = (g.G[0] + c[0]) * g.st[0] + (g.G[1] + c[1]) * g.st[1] + (g.G[2] + c[2]) * g.st[2];
    int64_t fl[NDIM], fr[NDIM];
    double du[NDIM];
#pragma unroll
    for (int d = 0; d < NDIM; ++d) {
      fl[d] = (c[2] * g.fe[d][1] + c[1]) * g.fe[d][0] + c[0];
      fr[d] = fl[d] + (d == 0 ? 1 : (d == 1 ? g.fe[d][0] : g.fe[d][0] * g.fe[d][1]));
      du[d] = divide(a.u[d][fr[d]] - a.u[d][fl[d]], g.dx[d]);
    }
    double out[NV];
#pragma unroll
    for (int f = 0; f < NV; ++f) {
      double L = 0.0;
      const double phi = a.Us[f * g.N + i];
#pragma unroll
      for (int d = 0; d < NDIM; ++d) {
        const int64_t nf = g.nfaces[d];
        const double dF = a.F[d][f * nf + fr[d]] - a.F[d][f * nf + fl[d]];
        double term = -divide(dF, g.dx[d]);
        if (f >= 2 + NDIM) term = term + phi * du[d];
        L = L + term;
      }
      double o;
      if (a.stage < 0) {
        o = L;
      } else {
        const double un = a.Un[f * g.N + i];
        if (a.stage == 0)
          o = un + dt * L;
        else if (a.stage == 1)
          o = (0.75 * un) + (0.25 * (phi + dt * L));
        else
          o = (c13 * un) + (c23 * (phi + dt * L));
      }
      out[f] = o;
    }
#pragma unroll
    for (int f = 0; f < NV; ++f) a.Uout[f * g.N + i] = out[f];
    if (a.stage == 2) {
      double q[NV];
      cons_to_prim(NDIM, out, q);
      if (!admissible(q[0], q[1 + NDIM], q[2 + NDIM], q[3 + NDIM])) atomicAdd(a.nbad, 1ULL);
    }
  }
}

__global__ void k_mood_count(const uint8_t* __restrict__ mask, int64_t n, int64_t nstage,
                             const int64_t* __restrict__ dir_off, int ndim, unsigned long long* counts) {
  __shared__ unsigned long long sc[9];
  if (threadIdx.x < 9) sc[threadIdx.x] = 0;
  __syncthreads();
  unsigned long long loc[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
  int64_t total = n * nstage;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
    int64_t k = t % n;
    int d = 0;
    for (int e = 1; e < ndim; ++e)
      if (k >= dir_off[e]) d = e;
    uint8_t m = mask[t];
    int cl = m & 3, cr = (m >> 2) & 3;
    if (cl < 3) loc[3 * d + cl]++;
    if (cr < 3) loc[3 * d + cr]++;
  }
  for (int j = 0; j < 9; ++j)
    if (loc[j]) atomicAdd(&sc[j], loc[j]);
  __syncthreads();
  if (threadIdx.x < 9 && sc[threadIdx.x]) atomicAdd(&counts[threadIdx.x], sc[threadIdx.x]);
}

}  // namespace

void launch_prep(const GridDev& g, double* U, double* Q, unsigned long long* lmax, unsigned long long* clear,
                 cudaStream_t s) {
  const int b = blocks_for(g.N);
  switch (g.ndim) {
    case 1: launch_following(k_prep<1>, b, BS, s, g, U, Q, lmax, clear); break;
    case 2: launch_following(k_prep<2>, b, BS, s, g, U, Q, lmax, clear); break;
    default: launch_following(k_prep<3>, b, BS, s, g, U, Q, lmax, clear); break;
  }
}

void launch_prim_to_cons(const GridDev& g, const double* Q, double* U, cudaStream_t s) {
  k_prim_to_cons<<<blocks_for(g.N), BS, 0, s>>>(g, Q, U);
}

void launch_cons_to_prim_all(const GridDev& g, const double* U, double* Q, cudaStream_t s) {
  k_cons_to_prim_all<<<blocks_for(g.N), BS, 0, s>>>(g, U, Q);
}

void launch_set_dt(const double*, double dt_fixed, double cfl, const unsigned long long* lmax, double* dt_dev,
                   int64_t n, cudaStream_t s) {
  k_set_dt<<<blocks_for(n), BS, 0, s>>>(dt_fixed, cfl, lmax, dt_dev, n);
}

void launch_update(const GridDev& g, int stage, const double* Un, const double* Us, double* Uout,
                   double* const Fh[3], double* const us[3], double dt_fixed, double cfl,
                   const unsigned long long* lmax, double* dt_dev, double* dt_host, unsigned long long* nbad,
                   cudaStream_t s) {
  UpdateArgs a{g, stage, Un, Us, Uout, {Fh[0], Fh[1], Fh[2]}, {us[0], us[1], us[2]}, dt_fixed, cfl, lmax, dt_dev, dt_host, nbad};
  const int b = blocks_for(g.ncell);
  switch (g.ndim) {
    case 1: launch_following(k_update<1>, b, BS, s, a); break;
    case 2: launch_following(k_update<2>, b, BS, s, a); break;
    default: launch_following(k_update<3>, b, BS, s, a); break;
  }
}

void launch_mood_count(const uint8_t* mask, int64_t n, int64_t nstage, const int64_t* dir_off, int ndim,
                       unsigned long long* counts, cudaStream_t s) {
  int b = blocks_for(n * nstage);
  if (b > 152 * 4) b = 152 * 4;
  k_mood_count<<<b, BS, 0, s>>>(mask, n, nstage, dir_off, ndim, counts);
}

}  // namespace ws
