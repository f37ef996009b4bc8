// FP64 sweep over the grid: primitives and ghost layers in one launch, then
// the faces of all directions in one launch (face_fp64.cuh).  Built with
// -fmad=false.
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
// 18 warps, or 64 registers with spills, measured 2 % slower).  On the 512^2
// shock-bubble a sweep takes 0.60 ms, the FP64 pipe 80 % busy, against 2.4 ms
// for one thread per face and native operations.
template <int NDIM, int CH, Scheme SC, int PI>
__global__ void __launch_bounds__(32 * (NDIM + 4), 24 / (NDIM + 4)) k_face(const __grid_constant__ FaceArgs a) {
  constexpr int NQ = NDIM + 4, H = (NQ + 2) / 2;
  __shared__ FaceSmem<NQ, CH> sm;
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
    k_face<NDIM, NQ, SC, PIPES><<<ctas, 32 * NQ, 0, s>>>(a);
  } else {
    ctas = ctas_of(a, 1, a.first);
    k_face<NDIM, 1, SC, CHAIN><<<ctas, 32 * NQ, 0, s>>>(a);
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

}  // namespace ws
