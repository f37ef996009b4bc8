// Learned smooth-face gate: training-data sampling and the MLP's training
// kernels (forward, backward, Adam), hand-written in FP32.
//
// The gate is a 24 -> 32 -> 32 -> 1 MLP (ReLU, ReLU, sigmoid) that reads, for
// one face i+1/2, the characteristic variables w1 (u-c), w2 (entropy), w6
// (u+c) and w_Gamma of the six stencil cells i-2..i+3, each normalised over
// the stencil as (w - mean)/(max - min + 1e-30), or zero when the stencil is
// flat to 1e-6 of its magnitude (below FP32 resolution of the variable).  A
// face is labelled "needs WENO-IS" (1) when MOOD lowers either side below 5th
// order or when, for any characteristic variable with a non-flat stencil and
// either side, the WENO-IS value differs from the 5th-order linear-weight
// value by more than 1e-6 (max - min); faces labelled 0 may take the linear
// weights d = (4,2,3,1)/10 for w1, w2, w6, w_Gamma and w_Pi (Pi is affine in
// Gamma across a two-material interface, so w_Gamma's inputs speak for it);
// shear variables always keep WENO-IS and are not part of the label.
// Parameter layout (FP32, WS_MLP_NPARAM floats): W1[32][24], b1[32],
// W2[32][32], b2[32], W3[32], b3.
#include <cuda_runtime.h>

#include "face_fp32.cuh"
#include "ws_internal.h"

namespace ws {

namespace {

using namespace fp32;

constexpr int NIN = 24, NH = 32;
constexpr int OW1 = 0, OB1 = OW1 + NH * NIN, OW2 = OB1 + NH, OB2 = OW2 + NH * NH, OW3 = OB2 + NH,
              OB3 = OW3 + NH, NPARAM = OB3 + 1;
static_assert(NPARAM == WS_MLP_NPARAM, "parameter count");

inline int blocks_for(int64_t n, int bs) {
  int64_t b = (n + bs - 1) / bs;
  if (b > (1LL << 30)) b = 1LL << 30;
  return (int)(b < 1 ? 1 : b);
}

// features and label of one face from sweep-frame FP32 primitives
template <int NQ>
__device__ void face_features(const float (&qc)[6][NQ], const float (&cc)[6], const WenoParams& P, float* feat,
                              uint8_t& label) {
  constexpr int NT = NQ - 5, IP = 2 + NT;
  float rho_bar = 0.5f * (qc[2][0] + qc[3][0]);
  float c_bar = 0.5f * (cc[2] + cc[3]);
  float rc = rho_bar * c_bar, hrc = 0.5f * rc;
  float ic2 = frcp(c_bar * c_bar), irc = frcp(rc);
  bool rough = false;
  bool flat_gamma = false;
  float wt5[2][NQ];
#pragma unroll
  for (int r = 0; r < NQ; ++r) {
    float w[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) w[k] = project<NQ>(qc[k], r, hrc, ic2);
    float mn = w[0], mx = w[0], sum = w[0];
#pragma unroll
    for (int k = 1; k < 6; ++k) {
      mn = fminf(mn, w[k]);
      mx = fmaxf(mx, w[k]);
      sum += w[k];
    }
    float range = (mx - mn) + 1e-30f;
    // features: w1 (r = 0), w2 (r = 1), w6 (r = NQ-1), w_Gamma (r = IP); a
    // stencil flat to 1e-6 of its magnitude gives zero features
    int slot = r == 0 ? 0 : (r == 1 ? 1 : (r == NQ - 1 ? 2 : (r == IP ? 3 : -1)));
    if (slot >= 0) {
      float mean = sum * (1.0f / 6.0f);
      float inv = (mx - mn) > 1e-6f * fmaxf(fabsf(mx), fabsf(mn)) ? frcp(range) : 0.0f;
#pragma unroll
      for (int k = 0; k < 6; ++k) feat[slot * 6 + k] = (w[k] - mean) * inv;
    }
#pragma unroll
    for (int side = 0; side < 2; ++side) {
      float v0 = side == 0 ? w[0] : w[5], v1 = side == 0 ? w[1] : w[4], v2 = side == 0 ? w[2] : w[3];
      float v3 = side == 0 ? w[3] : w[2], v4 = side == 0 ? w[4] : w[1];
      float full = weno_is(v0, v1, v2, v3, v4, P, 5);
      float lin = linear5(v0, v1, v2, v3, v4);
      // a stencil flat to 1e-6 of its magnitude (FP32 noise level) counts as
      // smooth; shear variables always keep WENO-IS, so they do not count
      bool flat = (mx - mn) <= 1e-6f * fmaxf(fabsf(mx), fabsf(mn));
      if (r == IP) flat_gamma = flat;
      if (r == IP + 1) flat = flat || flat_gamma;  // Pi follows Gamma (affine across the interface)
      bool shear = r >= 2 && r < IP;
      if (!shear && !flat && fabsf(full - lin) > 1e-6f * range) rough = true;
      wt5[side][r] = full;
    }
  }
#pragma unroll
  for (int side = 0; side < 2; ++side) {
    float q[NQ];
    back_project<NQ>(wt5[side], ic2, irc, q);
    if (!admissible<NQ>(q)) rough = true;
  }
  label = rough ? 1 : 0;
}

template <int NDIM>
__global__ void k_face_samples(GridDev g, int d, const float* __restrict__ Q, int64_t stride, int64_t out0,
                               int64_t max_out, float* __restrict__ feats, uint8_t* __restrict__ labels,
                               WenoParams P) {
  constexpr int NQ = NDIM + 4;
  const int64_t nf = g.nfaces[d];
  const int64_t ns = (nf + stride - 1) / stride;
  const int64_t fe0 = g.fe[d][0], fe1 = g.fe[d][1];
  const int64_t N = g.N;
  int fld[NQ];
  fld[0] = 0;
  fld[1] = 1 + d;
  {
    int k = 2;
#pragma unroll
    for (int e = 0; e < NDIM; ++e)
      if (e != d) fld[k++] = 1 + e;
  }
  fld[NQ - 3] = 1 + NDIM;
  fld[NQ - 2] = 2 + NDIM;
  fld[NQ - 1] = 3 + NDIM;
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < ns; s += (int64_t)gridDim.x * blockDim.x) {
    int64_t o = out0 + s;
    if (o >= max_out) break;
    int64_t f = s * stride;
    int64_t c[3];
    c[0] = f % fe0;
    int64_t r = f / fe0;
    c[1] = r % fe1;
    c[2] = r / fe1;
    c[d] -= 1;
    int64_t base = (g.G[0] + c[0]) * g.st[0] + (g.G[1] + c[1]) * g.st[1] + (g.G[2] + c[2]) * g.st[2];
    float qc[6][NQ], cc[6];
#pragma unroll
    for (int j = 0; j < 6; ++j) {
      int64_t idx = base + (j - 2) * g.st[d];
#pragma unroll
      for (int m = 0; m < NQ; ++m) qc[j][m] = Q[fld[m] * N + idx];
      cc[j] = Q[NQ * N + idx];
    }
    float feat[NIN];
    uint8_t lab;
    face_features<NQ>(qc, cc, P, feat, lab);
#pragma unroll
    for (int k = 0; k < NIN; ++k) feats[o * NIN + k] = feat[k];
    labels[o] = lab;
  }
}

// ---- MLP in FP32 ----
__device__ __forceinline__ void mlp_forward(const float* __restrict__ W, const float* x, float* h1, float* h2,
                                            float& z) {
#pragma unroll 4
  for (int j = 0; j < NH; ++j) {
    float a = W[OB1 + j];
#pragma unroll
    for (int k = 0; k < NIN; ++k) a = fmaf(W[OW1 + j * NIN + k], x[k], a);
    h1[j] = fmaxf(a, 0.0f);
  }
#pragma unroll 4
  for (int j = 0; j < NH; ++j) {
    float a = W[OB2 + j];
#pragma unroll
    for (int k = 0; k < NH; ++k) a = fmaf(W[OW2 + j * NH + k], h1[k], a);
    h2[j] = fmaxf(a, 0.0f);
  }
  float a = W[OB3];
#pragma unroll
  for (int k = 0; k < NH; ++k) a = fmaf(W[OW3 + k], h2[k], a);
  z = a;
}

__global__ void k_mlp_forward(const float* __restrict__ params, const float* __restrict__ X, int64_t n,
                              float* __restrict__ logits) {
  __shared__ float W[NPARAM];
  for (int i = threadIdx.x; i < NPARAM; i += blockDim.x) W[i] = params[i];
  __syncthreads();
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < n; s += (int64_t)gridDim.x * blockDim.x) {
    float x[NIN], h1[NH], h2[NH], z;
#pragma unroll
    for (int k = 0; k < NIN; ++k) x[k] = X[s * NIN + k];
    mlp_forward(W, x, h1, h2, z);
    logits[s] = z;
  }
}

// The gradient is summed in 64-bit fixed point (units of 2^-48): integer
// additions commute, so the sums do not depend on the order in which samples
// and blocks come in, and a gradient is the same on every run.  Each
// contribution is rounded to the unit once (|contributions| < 3e4).
constexpr float kFixScale = 281474976710656.0f;  // 2^48
// the sums; [NPARAM]: the loss.  Each call sets them to zero first
__device__ unsigned long long g_mlp_acc[NPARAM + 1];

__global__ void k_mlp_acc_zero() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");  // k_mlp_grad, which waits before it adds
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i <= NPARAM; i += gridDim.x * blockDim.x) g_mlp_acc[i] = 0ULL;
}

__device__ __forceinline__ long long fix(float v) {
  float s = fminf(fmaxf(v * kFixScale, -9.0e18f), 9.0e18f);  // exact scaling by a power of two
  return __float2ll_rn(s);
}

__global__ void k_mlp_acc_out(float* __restrict__ grad, float* __restrict__ loss) {
  follow_previous();
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i <= NPARAM; i += gridDim.x * blockDim.x) {
    float v = (float)((double)(long long)g_mlp_acc[i] * (1.0 / 281474976710656.0));
    if (i < NPARAM)
      grad[i] = v;
    else
      *loss = v;
  }
}

// fix(a b) for |a b| < 2^-3, b given times 2^48, without a conversion
// instruction: adding 1.5 2^46 rounds the product s to a multiple of 2^23,
// which the sum's low bits hold, and adding 1.5 2^23 rounds the exact rest
// (at most 2^22) to an integer.  The two parts are summed apart, as 32-bit
// integers that hold a tile's 128 samples.
__device__ __forceinline__ void fix_add(float a, float b, int& hi, int& lo) {
  const float M = 105553116266496.0f, m = 12582912.0f;
  const float s = __fmul_rn(a, b);
  const float t = __fadd_rn(s, M);
  const float rest = __fsub_rn(s, __fsub_rn(t, M));
  hi += __float_as_int(t) - 0x56c00000;
  lo += __float_as_int(__fadd_rn(rest, m)) - 0x4b400000;
}

// Mean binary cross-entropy (positives weighted by pos_weight) and its
// gradient over n samples, into g_mlp_acc.  A CTA takes tiles of GT samples
// through two parts.  First a sample to a thread: forward and backward, with
// activations and their gradients left in shared memory.  Then the
// parameters to the threads: a warp owns GR rows of W1 and of W2, a lane a
// column, and each adds up its parameters' contributions over the tile's
// samples in registers, which reach global memory once per CTA.  (One thread per
// sample adding 1889 shared-memory atomics to the same addresses as its
// neighbours took 2.71 ms for 65536 samples; this takes 0.09 ms.  Its warps are
// few: 150 registers and 93 KB of shared memory a CTA leave 11 % of them on an SM,
// which issues in 46 % of its cycles.)
constexpr int GT = 128, GR = NH / (GT / 32), GP = NH + 1;  // GP: row pitch without bank conflicts
struct GradSmem {
  float W[(NPARAM + 3) / 4 * 4];
  float x[GT][GP];   // inputs, then 1 (for b1) and zeros
  float h1[GT][GP], h2[GT][GP], g1[GT][GP], g2[GT][GP];
  float dz[GT], loss[GT];
};

// out[j] = max(b[j] + sum_k W[j][k] in[k], 0), j < NH, summed in the order of k
template <int K>
__device__ __forceinline__ void dense_relu(const float* W, const float* b, const float (&in)[K], float* out) {
#pragma unroll 4
  for (int j = 0; j < NH; ++j) {
    float a = b[j];
#pragma unroll
    for (int k = 0; k < K; k += 4) {
      const float4 w = *reinterpret_cast<const float4*>(W + j * K + k);
      a = fmaf(w.x, in[k], a);
      a = fmaf(w.y, in[k + 1], a);
      a = fmaf(w.z, in[k + 2], a);
      a = fmaf(w.w, in[k + 3], a);
    }
    out[j] = fmaxf(a, 0.0f);
  }
}

__global__ void __launch_bounds__(GT, 2) k_mlp_grad(const float* __restrict__ params, const float* __restrict__ X,
                                                    const uint8_t* __restrict__ y, int64_t n, float pos_weight,
                                                    float inv_n) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");  // k_mlp_acc_out, which waits
  extern __shared__ __align__(16) unsigned char grad_raw[];
  GradSmem& S = *reinterpret_cast<GradSmem*>(grad_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  static_assert(OW2 % 4 == 0 && OW1 % 4 == 0 && NIN % 4 == 0, "weight rows are read four at a time");
  for (int i = tid; i < NPARAM; i += GT) S.W[i] = params[i];
  for (int k = NIN; k < NH; ++k) S.x[tid][k] = k == NIN ? 1.0f : 0.0f;
  long long a1[GR], a2[GR], a3 = 0;  // W1 and b1 rows, W2 rows; warp 0: W3, warp 1: b2, warp 2: b3 and the loss
#pragma unroll
  for (int r = 0; r < GR; ++r) a1[r] = a2[r] = 0;
  __syncthreads();
  for (int64_t t0 = blockIdx.x * (int64_t)GT; t0 < n; t0 += (int64_t)gridDim.x * GT) {
    const int ns = (int)(n - t0 < GT ? n - t0 : GT);
    float most = 0.0f;  // bound of this sample's contributions
    if (tid < ns) {
      const int64_t s = t0 + tid;
      float act = 1.0f, gr = 0.0f;  // largest activation (or input) and gradient
      {
        float x[NIN];
#pragma unroll
        for (int k = 0; k < NIN; ++k) {
          S.x[tid][k] = x[k] = X[s * NIN + k];
          act = fmaxf(act, fabsf(x[k]));
        }
        dense_relu<NIN>(S.W + OW1, S.W + OB1, x, S.h1[tid]);
      }
      float z = S.W[OB3], h1[NH];
#pragma unroll
      for (int k = 0; k < NH; ++k) {
        h1[k] = S.h1[tid][k];
        act = fmaxf(act, h1[k]);
      }
      dense_relu<NH>(S.W + OW2, S.W + OB2, h1, S.h2[tid]);
#pragma unroll 8
      for (int k = 0; k < NH; ++k) {
        z = fmaf(S.W[OW3 + k], S.h2[tid][k], z);
        act = fmaxf(act, S.h2[tid][k]);
      }
      const bool pos = y[s] != 0;
      const float t = pos ? 1.0f : 0.0f;
      const float wgt = (pos ? pos_weight : 1.0f) * inv_n;
      // BCE with logits: softplus(z) - t z, computed stably
      const float sp = fmaxf(z, 0.0f) + log1pf(expf(-fabsf(z)));
      S.loss[tid] = wgt * (sp - t * z);
      const float p = 1.0f / (1.0f + expf(-z));
      const float dz = wgt * (p - t);
      S.dz[tid] = dz;
      float dh1[NH];
#pragma unroll
      for (int k = 0; k < NH; ++k) dh1[k] = 0.0f;
#pragma unroll 2
      for (int j = 0; j < NH; ++j) {
        const float g2 = S.h2[tid][j] > 0.0f ? dz * S.W[OW3 + j] : 0.0f;
        S.g2[tid][j] = g2;
        gr = fmaxf(gr, fabsf(g2));
        if (g2 == 0.0f) continue;
#pragma unroll
        for (int k = 0; k < NH; k += 4) {
          const float4 w = *reinterpret_cast<const float4*>(&S.W[OW2 + j * NH + k]);
          dh1[k] = fmaf(w.x, g2, dh1[k]);
          dh1[k + 1] = fmaf(w.y, g2, dh1[k + 1]);
          dh1[k + 2] = fmaf(w.z, g2, dh1[k + 2]);
          dh1[k + 3] = fmaf(w.w, g2, dh1[k + 3]);
        }
      }
#pragma unroll
      for (int k = 0; k < NH; ++k) {
        const float g1 = S.h1[tid][k] > 0.0f ? dh1[k] : 0.0f;
        S.g1[tid][k] = g1;
        gr = fmaxf(gr, fabsf(g1));
      }
      most = fmaxf(act * fmaxf(gr, fabsf(dz)), fabsf(S.loss[tid]));
      // maxima pass over a NaN; whatever holds one shows it in z or in a gradient's sum
      if (!(fabsf(z) < 1e30f) || !(act < 1e18f)) most = 1.0f;
    }
    const bool large = __syncthreads_or(tid < ns && !(most < 0.125f));  // (NaN counts as large)
    // a row's gradient is zero for the samples whose unit is off
    if (!large) {
      int hi1[GR], lo1[GR], hi2[GR], lo2[GR], hi3 = 0, lo3 = 0;
#pragma unroll
      for (int r = 0; r < GR; ++r) hi1[r] = lo1[r] = hi2[r] = lo2[r] = 0;
#pragma unroll 2
      for (int s = 0; s < ns; ++s) {
        const float h = S.h1[s][lane] * kFixScale, x = S.x[s][lane] * kFixScale;
#pragma unroll
        for (int r = 0; r < GR; ++r) {
          const float g = S.g2[s][warp * GR + r];
          if (g != 0.0f) fix_add(g, h, hi2[r], lo2[r]);
        }
#pragma unroll
        for (int r = 0; r < GR; ++r) {
          const float g = S.g1[s][warp * GR + r];
          if (g != 0.0f) fix_add(g, x, hi1[r], lo1[r]);
        }
        if (warp == 0) fix_add(S.dz[s], S.h2[s][lane] * kFixScale, hi3, lo3);
        if (warp == 1) fix_add(S.g2[s][lane], kFixScale, hi3, lo3);
        if (warp == 2) fix_add(lane == 0 ? S.dz[s] : S.loss[s], kFixScale, hi3, lo3);
      }
#pragma unroll
      for (int r = 0; r < GR; ++r) {
        a1[r] += (long long)hi1[r] * (1 << 23) + lo1[r];
        a2[r] += (long long)hi2[r] * (1 << 23) + lo2[r];
      }
      a3 += (long long)hi3 * (1 << 23) + lo3;
    } else {
#pragma unroll 1
      for (int s = 0; s < ns; ++s) {
        const float h = S.h1[s][lane], x = S.x[s][lane];
#pragma unroll
        for (int r = 0; r < GR; ++r) {
          const float u = S.g2[s][warp * GR + r], v = S.g1[s][warp * GR + r];
          if (u != 0.0f) a2[r] += fix(u * h);
          if (v != 0.0f) a1[r] += fix(v * x);
        }
        if (warp == 0) a3 += fix(S.dz[s] * S.h2[s][lane]);
        if (warp == 1) a3 += fix(S.g2[s][lane]);
        if (warp == 2) a3 += fix(lane == 0 ? S.dz[s] : S.loss[s]);
      }
    }
    __syncthreads();  // the next tile takes the arrays
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");  // the sums are zero
  auto add = [](int i, long long v) {
    if (v != 0) atomicAdd(&g_mlp_acc[i], (unsigned long long)v);
  };
#pragma unroll
  for (int r = 0; r < GR; ++r) {
    const int j = warp * GR + r;
    add(OW2 + j * NH + lane, a2[r]);
    if (lane < NIN) add(OW1 + j * NIN + lane, a1[r]);
    if (lane == NIN) add(OB1 + j, a1[r]);
  }
  if (warp == 0) add(OW3 + lane, a3);
  if (warp == 1) add(OB2 + lane, a3);
  if (warp == 2 && lane < 2) add(lane == 0 ? OB3 : NPARAM, a3);
}

__global__ void k_adam(float* __restrict__ p, float* __restrict__ m, float* __restrict__ v,
                       const float* __restrict__ g, float lr, float b1, float b2, float eps, float c1, float c2) {
  follow_previous();
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= NPARAM) return;
  float gi = g[i];
  float mi = fmaf(b1, m[i], (1.0f - b1) * gi);
  float vi = fmaf(b2, v[i], (1.0f - b2) * gi * gi);
  m[i] = mi;
  v[i] = vi;
  p[i] -= lr * (mi * c1) / (sqrtf(vi * c2) + eps);
}

}  // namespace

void launch_face_samples(const GridDev& g, int d, const float* Q, int64_t stride, int64_t out0, int64_t max_out,
                         float* feats, uint8_t* labels, float eps_rel, int weights, cudaStream_t s) {
  WenoParams P = weno_params(eps_rel, weights);
  int64_t ns = (g.nfaces[d] + stride - 1) / stride;
  int b = blocks_for(ns, 128);
  switch (g.ndim) {
    case 1: k_face_samples<1><<<b, 128, 0, s>>>(g, d, Q, stride, out0, max_out, feats, labels, P); break;
    case 2: k_face_samples<2><<<b, 128, 0, s>>>(g, d, Q, stride, out0, max_out, feats, labels, P); break;
    default: k_face_samples<3><<<b, 128, 0, s>>>(g, d, Q, stride, out0, max_out, feats, labels, P); break;
  }
}

}  // namespace ws

using namespace ws;

extern "C" WS_API int ws_mlp_forward(const float* params, const float* X, int64_t n, float* logits, void* stream) {
  if (n < 0 || !params || (n > 0 && (!X || !logits))) return WS_EINVAL;
  if (n == 0) return WS_OK;
  int b = blocks_for(n, 256);
  if (b > 152 * 16) b = 152 * 16;
  k_mlp_forward<<<b, 256, 0, (cudaStream_t)stream>>>(params, X, n, logits);
  return cudaGetLastError() == cudaSuccess ? WS_OK : WS_ECUDA;
}

extern "C" WS_API int ws_mlp_grad(const float* params, const float* X, const uint8_t* y, int64_t n, float pos_weight,
                                  float* grad, float* loss, void* stream) {
  if (n <= 0 || !params || !X || !y || !grad || !loss) return WS_EINVAL;
  cudaStream_t s = (cudaStream_t)stream;
  int b = blocks_for(n, GT);
  if (b > 152 * 2) b = 152 * 2;  // two CTAs per SM
  if (cudaFuncSetAttribute(k_mlp_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(GradSmem)) != cudaSuccess)
    return WS_ECUDA;
  // (k_mlp_acc_zero begins when everything before it has ended, so k_mlp_grad
  // may read its inputs while that one runs)
  k_mlp_acc_zero<<<(NPARAM + 256) / 256, 256, 0, s>>>();
  launch_following_smem(k_mlp_grad, b, GT, sizeof(GradSmem), s, params, X, y, n, pos_weight, 1.0f / (float)n);
  launch_following(k_mlp_acc_out, (NPARAM + 256) / 256, 256, s, grad, loss);
  return cudaGetLastError() == cudaSuccess ? WS_OK : WS_ECUDA;
}

extern "C" WS_API int ws_mlp_adam(float* params, float* m, float* v, const float* grad, int64_t step, float lr,
                                  void* stream) {
  if (!params || !m || !v || !grad || step < 1) return WS_EINVAL;
  const float b1 = 0.9f, b2 = 0.999f;
  float c1 = 1.0f / (1.0f - powf(b1, (float)step)), c2 = 1.0f / (1.0f - powf(b2, (float)step));
  launch_following(k_adam, (NPARAM + 255) / 256, 256, (cudaStream_t)stream, params, m, v, grad, lr, b1, b2, 1e-8f, c1,
                   c2);
  return cudaGetLastError() == cudaSuccess ? WS_OK : WS_ECUDA;
}
