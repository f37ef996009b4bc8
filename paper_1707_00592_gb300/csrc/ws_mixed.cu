// Mixed-precision sweep: FP32 projection, WENO-IS and HLLC (face_fp32.cuh),
// FP64 where accuracy needs it -- the pressure recovery's E - Pi
// cancellation, the sign of the MOOD admissibility test, and the
// conservative SSP-RK3 accumulation of the FP64 state.
//
// Generic form (any dimension): ghost layers and the primitive cache in FP32
// (k_prep32), one face sweep (k_face32) writing FP32 fluxes, and the update
// (k_update_mixed) that forms L(U) in FP32 and accumulates the RK stage in
// FP64.  1D steps take k_line32.
#include <cuda_runtime.h>

#include "face_fp32.cuh"
#include "fp64_pipes.cuh"
#include "ws_internal.h"

namespace ws {

namespace {

using namespace fp32;

constexpr int BS = 256;

inline int blocks_for(int64_t n, int bs = BS) {
  int64_t b = (n + bs - 1) / bs;
  if (b > (1LL << 30)) b = 1LL << 30;
  return (int)(b < 1 ? 1 : b);
}

// Conservative FP64 -> FP32 primitives: the internal energy E - Pi is formed
// in FP64 (for water Pi ~ 7.8e8 dwarfs Gamma p at p ~ 1e5), the rest in FP32.
template <int NDIM>
__device__ __forceinline__ void cons_to_prim32(const double* U, float* q, float& c) {
  float rho = (float)U[0];
  float irho = frcp(rho);
  float usq = 0.0f;
  q[0] = rho;
#pragma unroll
  for (int d = 0; d < NDIM; ++d) {
    float u = (float)U[1 + d] * irho;
    q[1 + d] = u;
    usq = fmaf(u, u, usq);
  }
  float Gam = (float)U[2 + NDIM], Pi = (float)U[3 + NDIM];
  float eint = (float)(U[1 + NDIM] - U[3 + NDIM]);  // E - Pi in FP64
  float p = fmaf(-0.5f * rho, usq, eint) * frcp(Gam);
  q[1 + NDIM] = p;
  q[2 + NDIM] = Gam;
  q[3 + NDIM] = Pi;
  c = fsqrt(sound_speed2(rho, p, Gam, Pi));
}

// coordinates of linear index i in extents e0, e1 (x fastest), in 32-bit
// arithmetic where the index allows
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

// atomicMax of the threads' wave rates (as doubles: non-negative ones order
// like their bit patterns, a NaN above +inf)
__device__ __forceinline__ void block_max(float best, unsigned long long* lmax) {
  unsigned long long b = (unsigned long long)__double_as_longlong((double)best);
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
    if (lane == 0) atomicMax(lmax, b);
  }
}

// The start of an RHS evaluation in one launch: ghost layers of U (of the
// cells with one coordinate outside the interior: the others are never read),
// FP32 primitives and sound speed of every cell the sweeps read and, with lmax,
// the CFL rate: max over the interior cells of sum_d (|u_d| + c)/dx_d.
// clear: a counter set to zero.
template <int NDIM>
__global__ void __launch_bounds__(BS) k_prep32(const __grid_constant__ GridDev g, double* U, float* __restrict__ Q,
                                               unsigned long long* lmax, unsigned long long* clear) {
  constexpr int NV = NDIM + 4;
  follow_previous();
  if (clear && blockIdx.x == 0 && threadIdx.x == 0) *clear = 0ULL;
  float idx_[3];
#pragma unroll
  for (int d = 0; d < NDIM; ++d) idx_[d] = lmax ? (float)(1.0 / g.dx[d]) : 0.0f;
  float best = 0.0f;
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
    double u[NV];
#pragma unroll
    for (int f = 0; f < NV; ++f) {
      u[f] = U[f * g.N + src];
      if (f == flip) u[f] = -u[f];
      if (out) U[f * g.N + i] = u[f];
    }
    float q[NV], cs;
    cons_to_prim32<NDIM>(u, q, cs);
#pragma unroll
    for (int f = 0; f < NV; ++f) Q[f * g.N + i] = q[f];
    Q[NV * g.N + i] = cs;
    if (lmax && !out) {
      float lam = 0.0f;
#pragma unroll
      for (int d = 0; d < NDIM; ++d) lam = fmaf(fabsf(q[1 + d]) + cs, idx_[d], lam);
      if (!(lam <= best)) best = lam;  // NaN propagates
    }
  }
  if (lmax) block_max(best, lmax);
}

struct FaceArgs {
  GridDev g;
  const float* Q;
  float* Fh[3];
  float* us[3];
  uint8_t* mask[3];
  unsigned first[3];  // first CTA of each direction
  WenoParams P;
  int mood;
};

// a thread to a face, the CTAs of one direction after another
template <int NDIM>
__global__ void __launch_bounds__(128) k_face32(const __grid_constant__ FaceArgs a) {
  constexpr int NQ = NDIM + 4;
  follow_previous();
  const GridDev& g = a.g;
  int d = 0;
#pragma unroll
  for (int e = 1; e < NDIM; ++e)
    if (blockIdx.x >= a.first[e]) d = e;
  const int64_t nf = g.nfaces[d], N = g.N;
  const int64_t f = (int64_t)(blockIdx.x - a.first[d]) * 128 + threadIdx.x;
  if (f >= nf) return;
  int fld[NQ];
  fld[0] = 0;
  fld[1] = 1 + d;
#pragma unroll
  for (int m = 2; m < NQ - 3; ++m) fld[m] = m - 2 < d ? m - 1 : m;  // tangential velocities in increasing axis order
  fld[NQ - 3] = 1 + NDIM;
  fld[NQ - 2] = 2 + NDIM;
  fld[NQ - 1] = 3 + NDIM;
  int64_t c[3];
  coords(f, g.fe[d][0], g.fe[d][1], c);
  c[d] -= 1;
  const int64_t sd = g.st[d];
  const float* q = a.Q + (g.G[0] + c[0]) * g.st[0] + (g.G[1] + c[1]) * g.st[1] + (g.G[2] + c[2]) * g.st[2] - 2 * sd;
  float qc[6][NQ], cc[6];
#pragma unroll
  for (int j = 0; j < 6; ++j) {
#pragma unroll
    for (int m = 0; m < NQ; ++m) qc[j][m] = __ldg(q + fld[m] * N + j * sd);
    cc[j] = __ldg(q + NQ * N + j * sd);
  }
  float Fhat[NQ], ustar;
  int cl, cr;
  face<NQ>(qc, cc, a.P, a.mood, Fhat, ustar, cl, cr);
#pragma unroll
  for (int m = 0; m < NQ; ++m) a.Fh[d][fld[m] * nf + f] = Fhat[m];
  a.us[d][f] = ustar;
  if (a.mask[d]) a.mask[d][f] = (uint8_t)(cl | (cr << 2));
}

// RK stage of one cell from its L in FP32: FP64 accumulation.
__device__ __forceinline__ double rk_stage(int stage, double un, double us, float incr) {
  double di = (double)incr;
  if (stage == 0) return un + di;
  if (stage == 1) return fma(0.75, un, 0.25 * (us + di));
  return fma(1.0 / 3.0, un, (2.0 / 3.0) * (us + di));
}

// division-free FP64 admissibility of a conservative state:
// rho > 0, Gamma > 0 and (Gamma+1)(rho E - |m|^2/2) - rho Pi > 0
template <int NDIM>
__device__ __forceinline__ bool admissible_cons(const double* o) {
  double rho = o[0], Gam = o[2 + NDIM], Pi = o[3 + NDIM];
  double m2 = 0.0;
#pragma unroll
  for (int d = 0; d < NDIM; ++d) m2 = fma(o[1 + d], o[1 + d], m2);
  double t = fma(rho, o[1 + NDIM], -0.5 * m2);
  return rho > 0.0 && Gam > 0.0 && fma(Gam + 1.0, t, -rho * Pi) > 0.0;
}

// Stage 0 derives the step (dt_fixed, or cfl / *lmax) and leaves it in *dtp for
// the others; stage -1 writes L itself.
struct UpdateArgs {
  GridDev g;
  int stage;
  const double *Un, *Us;
  double* Uout;
  const float* F[3];
  const float* u[3];
  const float* Q;
  double dt_fixed, cfl;
  const unsigned long long* lmax;
  double* dtp;
  double* dt_host;  // nullable, mapped host memory: receives the step, too
  unsigned long long* nbad;
};

template <int NDIM>
__global__ void __launch_bounds__(BS) k_update_mixed(const __grid_constant__ UpdateArgs a) {
  constexpr int NV = NDIM + 4;
  follow_previous();
  const GridDev& g = a.g;
  float idx_[3];
#pragma unroll
  for (int d = 0; d < NDIM; ++d) idx_[d] = (float)(1.0 / g.dx[d]);
  float dt = 1.0f;
  if (a.stage == 0) {
    const double s = a.dt_fixed > 0.0 ? a.dt_fixed : fp64::divide(a.cfl, __longlong_as_double((long long)*a.lmax));
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      *a.dtp = s;
      if (a.dt_host) *a.dt_host = s;
    }
    dt = (float)s;
  } else if (a.stage > 0) {
    dt = (float)*a.dtp;
  }
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < g.ncell; t += (int64_t)gridDim.x * blockDim.x) {
    int64_t c[3];
    coords(t, g.n[0], g.n[1], c);
    const int64_t i = (g.G[0] + c[0]) * g.st[0] + (g.G[1] + c[1]) * g.st[1] + (g.G[2] + c[2]) * g.st[2];
    int64_t fl[NDIM], fr[NDIM];
    float du[NDIM];
#pragma unroll
    for (int d = 0; d < NDIM; ++d) {
      fl[d] = (c[2] * g.fe[d][1] + c[1]) * g.fe[d][0] + c[0];
      fr[d] = fl[d] + (d == 0 ? 1 : (d == 1 ? g.fe[d][0] : g.fe[d][0] * g.fe[d][1]));
      du[d] = (a.u[d][fr[d]] - a.u[d][fl[d]]) * idx_[d];
    }
    double out[NV];
#pragma unroll
    for (int f = 0; f < NV; ++f) {
      float L = 0.0f;
#pragma unroll
      for (int d = 0; d < NDIM; ++d) {
        const int64_t nf = g.nfaces[d];
        L = fmaf(-(a.F[d][f * nf + fr[d]] - a.F[d][f * nf + fl[d]]), idx_[d], L);
      }
      if (f >= 2 + NDIM) {
        float phi = a.Q[f * g.N + i];
        float s = 0.0f;
#pragma unroll
        for (int d = 0; d < NDIM; ++d) s += du[d];
        L = fmaf(phi, s, L);
      }
      if (a.stage < 0)
        out[f] = (double)L;
      else
        out[f] = rk_stage(a.stage, a.Un[f * g.N + i], a.Us[f * g.N + i], dt * L);
    }
#pragma unroll
    for (int f = 0; f < NV; ++f) a.Uout[f * g.N + i] = out[f];
    if (a.stage == 2 && !admissible_cons<NDIM>(out)) atomicAdd(a.nbad, 1ULL);
  }
}

// One RK stage of a 1D grid in one launch: primitives, faces and update of
// LF faces and the LF - 1 cells between them (neighbouring CTAs share a face),
// with the arithmetic of the general kernels above.  Boundary conditions are
// applied on load.  Stage 0 leaves L(U) and the CFL rate, stage 1 forms
// U1 = U + dt L from them on load and leaves U2, stage 2 updates U.  Three
// launches per step instead of the 14 and two memsets of the general path.
constexpr int LF = 128;

struct LineArgs {
  int n, stage;
  int64_t N;                 // padded cells of a field
  int bc[2];
  double dx, cfl, dt_fixed;
  WenoParams P;
  int mood;
  double* U;
  float* L;                  // n values per field
  double* U2;                // laid out like U
  uint8_t* mask;             // nullable
  unsigned long long* lmax;  // zero before stage 0; stage 2 leaves it zero
  double* dt;
  double* dt_host;           // nullable, mapped host memory: receives the step, too
  unsigned long long* nbad;  // stage 0 sets it to zero
};

__global__ void __launch_bounds__(LF) k_line32(const __grid_constant__ LineArgs a) {
  constexpr int C = LF + 5;
  __shared__ float prim[6][C], flux[6][LF];  // cell c of the CTA is cell f0 - 3 + c
  __shared__ double cons[5][C];
  __shared__ double dt_sh;
  __shared__ unsigned red[LF / 32];
  follow_previous();
  const int tid = threadIdx.x, n = a.n;
  const int f0 = blockIdx.x * (LF - 1);
  if (tid == 0) {
    if (a.stage == 1) {
      dt_sh = a.dt_fixed > 0.0 ? a.dt_fixed : fp64::divide(a.cfl, __longlong_as_double((long long)*a.lmax));
      if (blockIdx.x == 0) {
        *a.dt = dt_sh;
        if (a.dt_host) *a.dt_host = dt_sh;
      }
    } else if (a.stage == 2) {
      dt_sh = *a.dt;
      if (blockIdx.x == 0) *a.lmax = 0ULL;
    } else if (blockIdx.x == 0) {
      *a.nbad = 0ULL;
    }
  }
  if (a.stage != 0) __syncthreads();
  const float idx = (float)(1.0 / a.dx), dt = a.stage != 0 ? (float)dt_sh : 0.0f;
  unsigned best = 0u;  // the wave rate's bits: non-negative values order like them, a NaN above +inf
  for (int c = tid; c < C && f0 - 3 + c < n + NG; c += LF) {
    const int x = f0 - 3 + c;
    int m = x;
    bool flip = false;
    if (x < 0 || x >= n) {
      const int kind = a.bc[x < 0 ? 0 : 1];
      m = x < 0 ? 0 : n - 1;
      if (kind == WS_BC_PERIODIC) m = x < 0 ? x + n : x - n;
      if (kind == WS_BC_REFLECTIVE) {
        m = x < 0 ? -1 - x : n - 1 - (x - n);
        flip = true;
      }
    }
    double u[5];
#pragma unroll
    for (int f = 0; f < 5; ++f) {
      u[f] = (a.stage == 2 ? a.U2 : a.U)[f * a.N + NG + m];
      if (a.stage == 1) u[f] = rk_stage(0, u[f], u[f], dt * a.L[(int64_t)f * n + m]);
      if (flip && f == 1) u[f] = -u[f];
      cons[f][c] = u[f];
    }
    float q[5], cs;
    cons_to_prim32<1>(u, q, cs);
#pragma unroll
    for (int f = 0; f < 5; ++f) prim[f][c] = q[f];
    prim[5][c] = cs;
    if (a.stage == 0 && x >= 0 && x < n) {
      best = max(best, __float_as_uint(fmaf(fabsf(q[1]) + cs, idx, 0.0f)));
    }
  }
  if (a.stage == 0 && a.dt_fixed <= 0.0) {
    best = __reduce_max_sync(0xffffffffu, best);
    if ((tid & 31) == 0) red[tid >> 5] = best;
  }
  __syncthreads();
  if (a.stage == 0 && a.dt_fixed <= 0.0 && tid == 0) {
    for (int w = 1; w < LF / 32; ++w) best = max(best, red[w]);
    atomicMax(a.lmax, (unsigned long long)__double_as_longlong((double)__uint_as_float(best)));
  }
  if (f0 + tid <= n) {
    float qc[6][5], cc[6];
#pragma unroll
    for (int j = 0; j < 6; ++j) {
#pragma unroll
      for (int m = 0; m < 5; ++m) qc[j][m] = prim[m][tid + j];
      cc[j] = prim[5][tid + j];
    }
    float Fhat[5], ustar;
    int cl, cr;
    face<5>(qc, cc, a.P, a.mood, Fhat, ustar, cl, cr);
#pragma unroll
    for (int m = 0; m < 5; ++m) flux[m][tid] = Fhat[m];
    flux[5][tid] = ustar;
    if (a.mask) a.mask[f0 + tid] = (uint8_t)(cl | (cr << 2));
  }
  __syncthreads();
  if (tid == LF - 1 || f0 + tid >= n) return;
  const int64_t x = f0 + tid;
  const float du = (flux[5][tid + 1] - flux[5][tid]) * idx;
  double out[5];
#pragma unroll
  for (int f = 0; f < 5; ++f) {
    float L = fmaf(-(flux[f][tid + 1] - flux[f][tid]), idx, 0.0f);
    if (f >= 3) L = fmaf(prim[f][tid + 3], 0.0f + du, L);
    if (a.stage == 0)
      a.L[(int64_t)f * n + x] = L;
    else
      out[f] = rk_stage(a.stage, a.U[f * a.N + NG + x], cons[f][tid + 3], dt * L);
  }
  if (a.stage == 0) return;
#pragma unroll
  for (int f = 0; f < 5; ++f) (a.stage == 1 ? a.U2 : a.U)[f * a.N + NG + x] = out[f];
  if (a.stage == 2 && !admissible_cons<1>(out)) atomicAdd(a.nbad, 1ULL);
}

}  // namespace

void launch_prep32(const GridDev& g, double* U, float* Q, unsigned long long* lmax, unsigned long long* clear,
                   cudaStream_t s) {
  const int b = blocks_for(g.N);
  switch (g.ndim) {
    case 1: launch_following(k_prep32<1>, b, BS, s, g, U, Q, lmax, clear); break;
    case 2: launch_following(k_prep32<2>, b, BS, s, g, U, Q, lmax, clear); break;
    default: launch_following(k_prep32<3>, b, BS, s, g, U, Q, lmax, clear); break;
  }
}

void launch_face_mixed(const GridDev& g, const float* Q, float* const Fh[3], float* const us[3], uint8_t* const mask[3],
                       float eps_rel, int mood, int weights, cudaStream_t s) {
  FaceArgs a;
  a.g = g;
  a.Q = Q;
  a.P = weno_params(eps_rel, weights);
  a.mood = mood;
  unsigned b = 0;
  for (int d = 0; d < 3; ++d) {
    a.Fh[d] = Fh[d];
    a.us[d] = us[d];
    a.mask[d] = mask[d];
    a.first[d] = b;
    if (d < g.ndim) b += (unsigned)((g.nfaces[d] + 127) / 128);
  }
  switch (g.ndim) {
    case 1: launch_following(k_face32<1>, b, 128, s, a); break;
    case 2: launch_following(k_face32<2>, b, 128, s, a); break;
    default: launch_following(k_face32<3>, b, 128, s, a); break;
  }
}

void launch_update_mixed(const GridDev& g, int stage, const double* Un, const double* Us, double* Uout,
                         float* const Fh[3], float* const us[3], const float* Q, double dt_fixed, double cfl,
                         const unsigned long long* lmax, double* dt_dev, double* dt_host, unsigned long long* nbad,
                         cudaStream_t s) {
  const UpdateArgs a{g, stage, Un, Us, Uout, {Fh[0], Fh[1], Fh[2]}, {us[0], us[1], us[2]}, Q, dt_fixed, cfl, lmax, dt_dev,
                     dt_host, nbad};
  const int b = blocks_for(g.ncell);
  switch (g.ndim) {
    case 1: launch_following(k_update_mixed<1>, b, BS, s, a); break;
    case 2: launch_following(k_update_mixed<2>, b, BS, s, a); break;
    default: launch_following(k_update_mixed<3>, b, BS, s, a); break;
  }
}

void launch_line_mixed(const GridDev& g, int stage, double* U, float* L, double* U2, uint8_t* mask, float eps_rel, int mood,
                       int weights, double dt_fixed, double cfl, unsigned long long* lmax, double* dt, double* dt_host,
                       unsigned long long* nbad, cudaStream_t s) {
  const LineArgs a{g.n[0], stage, g.N, {g.bc[0][0], g.bc[0][1]}, g.dx[0], cfl, dt_fixed, weno_params(eps_rel, weights),
                   mood, U, L, U2, mask, lmax, dt, dt_host, nbad};
  launch_following(k_line32, (unsigned)((a.n + LF - 2) / (LF - 1)), LF, s, a);
}

}  // namespace ws
