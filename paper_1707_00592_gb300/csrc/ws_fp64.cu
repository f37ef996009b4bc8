// FP64 sweep over the grid: the faces of all directions in one launch
// (face_fp64.cuh), and for 1D grids a whole RK stage in one launch.  Built
// with -fmad=false.
#include <cuda_runtime.h>

#include "face_fp64.cuh"
#include "ws_internal.h"

namespace ws {

namespace {

using namespace fp64;

struct FaceArgs {
  GridDev g;
  const double* Q;
  double* Fh[3];
  double* us[3];
  uint8_t* mask[3];
  unsigned first[3];  // first CTA of each direction
  double eps;
  int mood, weights;
};

// One CTA: CH chunks of FPW consecutive faces of one direction.  24 warps per
// SM (80 registers): enough to cover the FP64 pipe's latency (96 registers and
// 18 warps, or 64 registers with spills, measured 2 % slower).  The FP64 pipe
// runs at 95 % of its rate of one instruction in 76 cycles: on the 512^2
// shock-bubble a sweep takes 0.57 ms against 2.4 ms for one thread per face and
// native operations.
template <int NDIM, int CH, Scheme SC, int PI>
__global__ void __launch_bounds__(32 * (NDIM + 4), 24 / (NDIM + 4)) k_face(const __grid_constant__ FaceArgs a) {
  constexpr int NQ = NDIM + 4, H = (NQ + 2) / 2;
  __shared__ FaceSmem<NQ, CH> sm;
  follow_previous();
  int d = 0;
#pragma unroll
  for (int e = 1; e < NDIM; ++e)
    if (blockIdx.x >= a.first[e]) d = e;
  const GridDev& g = a.g;
  const int64_t nf = g.nfaces[d];
  const int lane = threadIdx.x & 31, side = lane & 1;
  const int64_t f0 = (int64_t)(blockIdx.x - a.first[d]) * (CH * FPW) + (lane >> 1);
  auto at = [&](int k) {
    int64_t f = f0 + k * FPW;
    if (f >= nf) f = nf - 1;  // past the end: a face worked out for nothing
    int64_t c[3];
    if (nf < (1LL << 31)) {
      const unsigned u = (unsigned)f, fe0 = (unsigned)g.fe[d][0], fe1 = (unsigned)g.fe[d][1];
      const unsigned r = u / fe0, z = r / fe1;
      c[0] = u - r * fe0;
      c[1] = r - z * fe1;
      c[2] = z;
    } else {
      c[0] = f % g.fe[d][0];
      const int64_t r = f / g.fe[d][0];
      c[1] = r % g.fe[d][1];
      c[2] = r / g.fe[d][1];
    }
    // face i+1/2 with i = f_d - 1: stencil cell 0 is i - 2 = f_d - 3
    Faces<NQ> fc;
    fc.q = a.Q;
    fc.N = g.N;
    fc.d = d;
    fc.st = g.st[d];
    fc.base = (g.G[0] + c[0]) * g.st[0] + (g.G[1] + c[1]) * g.st[1] + (g.G[2] + c[2]) * g.st[2] - 3 * fc.st;
    return fc;
  };
  cta_faces<NQ, CH, SC, PI>(sm, a.eps, a.mood, a.weights, at,
                            [&](int k, const Faces<NQ>& fc, const double (&out)[H], int code) {
    const int other = __shfl_xor_sync(ALL, code, 1);
    const int64_t f = f0 + k * FPW;
    if (f >= nf) return;
    // fluxes stored in the global field order (rho, rho u_1.., E, Gamma, Pi)
#pragma unroll
    for (int j = 0; j < H; ++j) {
      const int m = (side ? H : 0) + j;
      if (m < NQ)
        a.Fh[d][fc.fld(m) * nf + f] = out[j];
      else if (m == NQ)
        a.us[d][f] = out[j];
    }
    if (a.mask[d] && side == 0) a.mask[d][f] = (uint8_t)(code | (other << 2));
  });
}

// Chunks of a direction and CTAs of a launch with CH chunks each.
unsigned ctas_of(const FaceArgs& a, int ch, unsigned (&first)[3]) {
  unsigned n = 0;
  for (int d = 0; d < 3; ++d) {
    first[d] = n;
    if (d < a.g.ndim) n += (unsigned)((a.g.nfaces[d] + ch * FPW - 1) / (ch * FPW));
  }
  return n;
}

template <int NDIM, Scheme SC>
void launch_faces(FaceArgs a, cudaStream_t s) {
  constexpr int NQ = NDIM + 4;
  unsigned ctas = ctas_of(a, NQ, a.first);
  if (SC != LITERAL && large_sweep(ctas)) {
    launch_following(k_face<NDIM, NQ, SC, PIPES>, ctas, 32 * NQ, s, a);
  } else {
    ctas = ctas_of(a, 1, a.first);
    launch_following(k_face<NDIM, 1, SC, CHAIN>, ctas, 32 * NQ, s, a);
  }
}

template <int NDIM>
void launch_faces(const FaceArgs& a, cudaStream_t s) {
  switch (scheme_of(a.eps, a.weights)) {
    case JS: launch_faces<NDIM, JS>(a, s); break;
    case LITERAL: launch_faces<NDIM, LITERAL>(a, s); break;
    default: launch_faces<NDIM, IS>(a, s); break;
  }
}

// One RK stage of a 1D grid: primitives, faces and update of CH FPW faces and
// the CH FPW - 1 cells between them in a CTA (neighbouring CTAs share a face).
// Boundary conditions are applied on load; U's ghost cells stay as they are.
// Stage 0 leaves L(U) and the CFL rate, stage 1 forms U1 = U + dt L from them
// on load and leaves U2, stage 2 updates U: no stage needs a value that another
// CTA of its launch writes.  A 200-cell step is bound by launches and the
// length of its chains: 3 launches instead of the 9 of the general path.
struct LineArgs {
  int n, stage;
  int64_t N;                 // padded cells of a field
  int bc[2];
  double dx, eps, cfl, dt_fixed;
  int mood, weights;
  double *U, *L, *U2;        // L: n values per field; U2: laid out like U
  uint8_t* mask;             // nullable
  unsigned long long* lmax;  // zero before stage 0; stage 2 leaves it zero
  double* dt;
  double* dt_host;           // nullable, mapped host memory: receives the step, too
  unsigned long long* nbad;  // stage 0 sets it to zero
};

template <int CH, Scheme SC, int PI>
__global__ void __launch_bounds__(160) k_line(const __grid_constant__ LineArgs a) {
  constexpr int F = CH * FPW, C = F + 5, H = 3;
  __shared__ FaceSmem<5, CH> sm;
  __shared__ double prim[6][C], cons[5][C], flux[6][F];  // cell c of the CTA is cell f0 - 3 + c
  __shared__ double dt_sh;
  __shared__ unsigned long long red[5];
  follow_previous();
  const int tid = threadIdx.x, n = a.n;
  const int f0 = blockIdx.x * (F - 1);
  if (tid == 0) {
    if (a.stage == 1) {
      dt_sh = a.dt_fixed > 0.0 ? a.dt_fixed : divide_call(a.cfl, __longlong_as_double((long long)*a.lmax));
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
  unsigned long long best = 0ULL;
  for (int c = tid; c < C && f0 - 3 + c < n + NG; c += 160) {
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
      if (a.stage == 1) u[f] = u[f] + dt_sh * a.L[(int64_t)f * n + m];
      if (flip && f == 1) u[f] = -u[f];
      cons[f][c] = u[f];
    }
    const double rho = u[0], v = divide_call(u[1], rho);
    const double ke = (0.5 * rho) * (0.0 + v * v);
    const double p = divide_call((u[2] - ke) - u[4], u[3]);
    const double cs = root_call(divide_call(((u[3] + 1.0) * p) + u[4], u[3] * rho));
    prim[0][c] = rho;
    prim[1][c] = v;
    prim[2][c] = p;
    prim[3][c] = u[3];
    prim[4][c] = u[4];
    prim[5][c] = cs;
    if (a.stage == 0 && a.dt_fixed <= 0.0 && x >= 0 && x < n) {
      const double lam = 0.0 + divide_call(fabs(v) + cs, a.dx);
      const unsigned long long b = lam <= 0.0 ? 0ULL : (unsigned long long)__double_as_longlong(lam);
      best = b > best ? b : best;
    }
  }
  if (a.stage == 0 && a.dt_fixed <= 0.0) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long v = __shfl_xor_sync(ALL, best, o);
      best = v > best ? v : best;
    }
    if ((tid & 31) == 0) red[tid >> 5] = best;
  }
  __syncthreads();
  if (a.stage == 0 && a.dt_fixed <= 0.0 && tid == 0) {
    for (int w = 1; w < 5; ++w) best = red[w] > best ? red[w] : best;
    atomicMax(a.lmax, best);
  }
  const int lane = tid & 31, side = lane & 1;
  auto at = [&](int k) {
    Faces<5, true> fc;
    fc.q = &prim[0][0];
    fc.N = C;
    fc.d = 0;
    fc.st = 1;
    fc.base = min(k * FPW + (lane >> 1), n - f0);  // past the end: the last face again
    return fc;
  };
  cta_faces<5, CH, SC, PI>(sm, a.eps, a.mood, a.weights, at,
                           [&](int k, const Faces<5, true>&, const double (&out)[H], int code) {
    const int other = __shfl_xor_sync(ALL, code, 1);
    const int i = k * FPW + (lane >> 1);
#pragma unroll
    for (int j = 0; j < H; ++j) flux[(side ? H : 0) + j][i] = out[j];
    if (a.mask && side == 0 && f0 + i <= n) a.mask[f0 + i] = (uint8_t)(code | (other << 2));
  });
  __syncthreads();
  const double c13 = 1.0 / 3.0, c23 = 2.0 / 3.0;
  for (int t = tid; t < F - 1 && f0 + t < n; t += 160) {
    const int64_t x = f0 + t;
    const double du = divide_call(flux[5][t + 1] - flux[5][t], a.dx);
    double out[5];
#pragma unroll
    for (int f = 0; f < 5; ++f) {
      const double phi = cons[f][t + 3];
      double term = -divide_call(flux[f][t + 1] - flux[f][t], a.dx);
      if (f >= 3) term = term + phi * du;
      const double L = 0.0 + term;
      if (a.stage == 0) {
        a.L[(int64_t)f * n + x] = L;
        continue;
      }
      const double un = a.U[f * a.N + NG + x];
      out[f] = a.stage == 1 ? (0.75 * un) + (0.25 * (phi + dt_sh * L)) : (c13 * un) + (c23 * (phi + dt_sh * L));
    }
    if (a.stage == 0) continue;
#pragma unroll
    for (int f = 0; f < 5; ++f) (a.stage == 1 ? a.U2 : a.U)[f * a.N + NG + x] = out[f];
    if (a.stage == 2) {
      const double v = divide_call(out[1], out[0]);
      const double ke = (0.5 * out[0]) * (0.0 + v * v);
      const double p = divide_call((out[2] - ke) - out[4], out[3]);
      if (!(out[0] > 0.0 && out[3] > 0.0 && (((out[3] + 1.0) * p) + out[4]) > 0.0)) atomicAdd(a.nbad, 1ULL);
    }
  }
}

template <Scheme SC>
void launch_line(const LineArgs& a, cudaStream_t s) {
  const unsigned b = (unsigned)((a.n + 5 * FPW - 2) / (5 * FPW - 1)), b1 = (unsigned)((a.n + FPW - 2) / (FPW - 1));
  if (SC != LITERAL && large_sweep(b))
    launch_following(k_line<5, SC, PIPES>, b, 160, s, a);
  else
    launch_following(k_line<1, SC, CHAIN>, b1, 160, s, a);
}

}  // namespace

void launch_face_fp64(const GridDev& g, const double* Q, double* const Fh[3], double* const us[3],
                      uint8_t* const mask[3], double eps, int mood, int weights, cudaStream_t s) {
  FaceArgs a;
  a.g = g;
  a.Q = Q;
  a.eps = eps;
  a.mood = mood;
  a.weights = weights;
  for (int d = 0; d < 3; ++d) {
    a.Fh[d] = Fh[d];
    a.us[d] = us[d];
    a.mask[d] = mask ? mask[d] : nullptr;
  }
  switch (g.ndim) {
    case 1: launch_faces<1>(a, s); break;
    case 2: launch_faces<2>(a, s); break;
    default: launch_faces<3>(a, s); break;
  }
}

void launch_line_fp64(const GridDev& g, int stage, double* U, double* L, double* U2, uint8_t* mask, double eps, int mood,
                      int weights, double dt_fixed, double cfl, unsigned long long* lmax, double* dt, double* dt_host,
                      unsigned long long* nbad, cudaStream_t s) {
  const LineArgs a{g.n[0], stage, g.N, {g.bc[0][0], g.bc[0][1]}, g.dx[0], eps, cfl, dt_fixed, mood, weights, U, L, U2,
                   mask, lmax, dt, dt_host, nbad};
  switch (scheme_of(eps, weights)) {
    case JS: launch_line<JS>(a, s); break;
    case LITERAL: launch_line<LITERAL>(a, s); break;
    default: launch_line<IS>(a, s); break;
  }
}

}  // namespace ws
