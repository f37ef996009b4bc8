// Batched independent 1D tubes, mixed precision, one persistent launch per RK
// stage.  Work items are chunks of CH cells of one tube; CTAs (a few per SM,
// for the whole launch) pull items from an atomic counter until none is left,
// so tubes of very different lengths balance across the GPU.  Per chunk the
// phases mirror the 2D fused stage: FP32 primitives of the chunk plus a
// 3-cell halo in shared memory (transmissive tube ends applied on load, E - Pi
// in FP64); one loop over the faces, each thread taking a face through
// WENO-IS of its characteristic variables (the linear weights for stencils
// flat to 1e-6), back-projection, MOOD and HLLC; and the increment-form
// SSP-RK3 with FP64 accumulation (see ws_fused.cu).  A chunk of CH = 2^k - 1
// cells has 2^k faces, a whole number per thread.
// Stage 0 also reduces each tube's CFL rate (atomicMax per tube); stages 1
// and 2 take dt = CFL / max per tube.
//
// Quiet chunks.  Until a tube's waves arrive a chunk and its halo hold one
// state (half of all cells over a 1000-step run), its fluxes are equal and its
// increments zero.  Stage 0 finds these chunks, writes their zero increments
// of both stages and their MOOD bytes of all three, and lists the others:
// stage 1 works through the chunks that move and those beside them, stage 2
// also through the next ones, and neither touches the rest (a chunk's halo
// lies in the chunks beside it).  The results are those of evaluating
// everything, bit for bit; the chunks of a tube whose step is not finite are
// all worked through (list_tube).
//
// While a CTA works on an item, its first thread fetches the next one's
// description and CFL rate step by step with asynchronous copies, so that no
// item starts with a chain of dependent loads.  4096 tubes (9.4 M cells, half
// of them quiet): 1034 -> 593 us per step.
#include <cuda_runtime.h>

#include "face_fp32.cuh"
#include "fp64_pipes.cuh"
#include "ws_internal.h"

namespace ws {

namespace {

using namespace fp32;

constexpr int NQ = 5;  // rho, u, p, Gamma, Pi

template <int CH>
struct TSmem {
  float q[NQ + 1][CH + 2 * NG];  // primitives + sound speed
  float F[NQ + 1][CH + 1];       // face fluxes + face velocity
  alignas(16) TubeItem next;     // the next item, copied in while this one is worked on
  double rate;                   // and its tube's CFL rate
  TubeItem now;
  int more;                      // now holds an item
  float dt;
  unsigned red[32];
};

struct TubeArgs {
  TubesDev t;
  int stage;
  double* U;
  float* U32;
  const float* Kin;
  float* Kout;
  float* Knext;              // stage 0: the increments of stage 1 (zeros of quiet chunks)
  double dt_fixed;
  float cfl;
  unsigned long long* lmax;  // per tube
  double* dt_out;            // per tube (written in stage 1)
  TubeWork w;
  uint8_t* mask;             // per padded cell, nullable; stages follow at nmask
  int64_t nmask;
  WenoParams P;
  int mood;
  unsigned long long* nbad;
};

__device__ __forceinline__ void copy16(void* dst, const void* src) {
  unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void copy8(void* dst, const void* src) {
  unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void copies_wait() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// A uniform state (rho, u, p, Gamma, Pi, c) that is admissible with a margin no
// reconstruction of it uses up, and whose flux is finite.
__device__ __forceinline__ bool quiet_state(float rho, float u, float p, float G, float Pi, float c) {
  return rho > 1e-20f && rho < 1e20f && G > 1e-6f && G < 1e6f && c > 1e-6f && fabsf(u) + c < 1e9f && fabsf(p) < 1e18f &&
         fabsf(Pi) < 1e18f &&
         fmaf(G + 1.0f, p, Pi) > 1e-4f * ((G + 1.0f) * (fabsf(p) + rho * c * fabsf(u)) + fabsf(Pi));
}

// Stage 1 of tube t with a step that is not finite: the step reaches every
// cell, those of chunks that stage 0 left out too.  In stage 1 their states are
// not numbers (0 times the step): both sides of their faces take the last resort
// of the MOOD cascade, and the increments don't matter any more; stage 2 works
// through them.
__device__ __noinline__ void list_tube(const TubeArgs& a, int64_t t, int chunk) {
  int64_t lo = 0, hi = a.w.nitems;  // the tube's first item
  while (lo < hi) {
    const int64_t m = (lo + hi) / 2;
    if (a.w.items[m].tube < t)
      lo = m + 1;
    else
      hi = m;
  }
  for (int64_t j = lo; j < a.w.nitems && a.w.items[j].tube == t; ++j) {
    const TubeItem it = a.w.items[j];
    if (a.mask && a.w.listed[j] == 0)
      for (int f = 0; f <= min(chunk, it.len - it.c0); ++f) a.mask[it.off + NG + it.c0 + f - 1] = a.mood ? 2 | (2 << 2) : 0;
    if (atomicExch(&a.w.listed[a.w.nitems + j], 1) == 0) a.w.list[a.w.nitems + atomicAdd(&a.w.counters[4], 1u)] = it;
  }
}

template <int CH, int NTH>
__global__ void __launch_bounds__(NTH, 1024 / NTH) k_tube_stage(const __grid_constant__ TubeArgs a) {  // 64 registers
  extern __shared__ __align__(16) unsigned char smem_raw[];
  TSmem<CH>& S = *reinterpret_cast<TSmem<CH>*>(smem_raw);
  constexpr int HW = CH + 2 * NG;
  const int tid = threadIdx.x;
  const int64_t N = a.t.total;
  // this stage's items: all of them, or the list that stage 0 left
  const TubeItem* items = a.stage == 0 ? a.w.items : a.w.list + (a.stage - 1) * a.w.nitems;
  const unsigned nitems = a.stage == 0 ? (unsigned)a.w.nitems : a.w.counters[2 + a.stage];
  unsigned* counter = a.w.counters + a.stage;
  if (a.stage == 1)  // the steps of all tubes
    for (int64_t t = blockIdx.x * (int64_t)NTH + tid; t < a.t.ntubes; t += (int64_t)gridDim.x * NTH) {
      const double d = a.dt_fixed > 0.0 ? a.dt_fixed : (double)a.cfl / __longlong_as_double((long long)a.lmax[t]);
      a.dt_out[t] = d;
      if (!(fabsf(f64_to_f32(d)) < INFINITY)) list_tube(a, t, CH);
    }
  // thread 0: makes the item in S.next the current one
  auto take = [&](unsigned k) {
    S.more = k < nitems;
    if (k >= nitems) return;
    copies_wait();
    S.now = S.next;
    if (a.stage > 0) S.dt = f64_to_f32(a.dt_fixed > 0.0 ? a.dt_fixed : fp64::divide((double)a.cfl, S.rate));
  };
  auto fetch_item = [&](unsigned k) {
    if (k >= nitems) return;
    copy16(&S.next, items + k);
    copy16(reinterpret_cast<char*>(&S.next) + 16, reinterpret_cast<const char*>(items + k) + 16);
  };
  auto fetch_rate = [&](unsigned k) {
    if (k >= nitems || a.stage == 0) return;
    copies_wait();
    copy8(&S.rate, &a.lmax[S.next.tube]);
  };
  unsigned nxt = 0;
  if (tid == 0) {
    nxt = blockIdx.x;  // the first item is the CTA's own, the counter hands out those after the first wave
    fetch_item(nxt);
    fetch_rate(nxt);
    take(nxt);
  }
  for (;;) {
    __syncthreads();
    if (!S.more) break;
    if (tid == 0) nxt = gridDim.x + atomicAdd(counter, 1u);
    const int64_t tube = S.now.tube;
    const int64_t off = S.now.off;
    const int len = S.now.len;
    const int c0 = S.now.c0;
    const int nc = min(CH, len - c0);  // cells of this chunk
    const float idx = (float)len;      // 1/dx, dx = 1/len
    // ---- phase A ----
    float p_own = -1.0f;
    unsigned lam = 0u;  // the wave rate's bits: non-negative values order like them, a NaN above +inf
    for (int h = tid; h < nc + 2 * NG; h += NTH) {
      int gc = c0 + h - NG;  // tube-local interior index
      int mc = gc < 0 ? 0 : (gc >= len ? len - 1 : gc);
      int64_t i = off + NG + mc;
      float rho, mu, eint, Gam, Pi;
      if (a.stage == 0) {
        rho = f64_to_f32(a.U[i]);
        mu = f64_to_f32(a.U[N + i]);
        eint = f64_to_f32(a.U[2 * N + i] - a.U[4 * N + i]);
        Gam = f64_to_f32(a.U[3 * N + i]);
        Pi = f64_to_f32(a.U[4 * N + i]);
        if (h >= NG && h < NG + nc) {
          a.U32[i] = rho;
          a.U32[N + i] = mu;
          a.U32[2 * N + i] = eint;
          a.U32[3 * N + i] = Gam;
          a.U32[4 * N + i] = Pi;
        }
      } else {
        float coef = a.stage == 1 ? S.dt : 0.25f * S.dt;
        const float* V = a.U32;
        const float* K = a.Kin;
        rho = fmaf(coef, K[i], V[i]);
        mu = fmaf(coef, K[N + i], V[N + i]);
        eint = fmaf(coef, K[2 * N + i] - K[4 * N + i], V[2 * N + i]);
        Gam = fmaf(coef, K[3 * N + i], V[3 * N + i]);
        Pi = fmaf(coef, K[4 * N + i], V[4 * N + i]);
      }
      float u = mu * frcp(rho);
      float p = fmaf(-0.5f * rho, u * u, eint) * frcp(Gam);
      float c = fsqrt(sound_speed2(rho, p, Gam, Pi));
      S.q[0][h] = rho;
      S.q[1][h] = u;
      S.q[2][h] = p;
      S.q[3][h] = Gam;
      S.q[4][h] = Pi;
      S.q[5][h] = c;
      p_own = p;
      if (a.stage == 0 && h >= NG && h < NG + nc) {
        lam = max(lam, __float_as_uint((fabsf(u) + c) * idx));
      }
    }
    if (a.stage == 0) {
      lam = __reduce_max_sync(0xffffffffu, lam);
      if ((tid & 31) == 0) S.red[tid >> 5] = lam;
      // one pressure in every warp: worth a look at all cells
      bool quiet = __syncthreads_and(p_own == __shfl_sync(0xffffffffu, p_own, 0) || p_own == -1.0f);
      if (tid == 0) {
        unsigned r = 0;
        for (int w = 0; w < NTH / 32; ++w) r = max(r, S.red[w]);
        if (r) atomicMax(&a.lmax[tube], (unsigned long long)__double_as_longlong(f32_to_f64(__uint_as_float(r))));
        fetch_item(nxt);
      }
      if (quiet) {
        bool eq = true;
        for (int h = tid; h < nc + 2 * NG; h += NTH)
#pragma unroll
          for (int m = 0; m < NQ; ++m) eq = eq && S.q[m][h] == S.q[m][0];
        quiet = __syncthreads_and(eq && quiet_state(S.q[0][0], S.q[1][0], S.q[2][0], S.q[3][0], S.q[4][0], S.q[5][0]));
      }
      if (quiet) {
        for (int cc_ = tid; cc_ < nc; cc_ += NTH) {
          const int64_t gi = off + NG + c0 + cc_;
#pragma unroll
          for (int m = 0; m < NQ; ++m) a.Kout[m * N + gi] = a.Knext[m * N + gi] = 0.0f;
        }
        if (a.mask)
          for (int f = tid; f <= nc; f += NTH)
#pragma unroll
            for (int s = 0; s < 3; ++s) a.mask[s * a.nmask + off + NG + c0 + f - 1] = 0;
        if (tid == 0) take(nxt);
        continue;
      }
      // this chunk and the ones beside it for stage 1, two on each side for stage 2
      if (tid < 8) {
        const int st = tid < 3 ? 0 : 1, d = st == 0 ? tid - 1 : tid - 5;
        const int cn = c0 + d * CH;
        if (cn >= 0 && cn < len) {
          const int64_t j = S.now.index + d;
          if (atomicExch(&a.w.listed[st * a.w.nitems + j], 1) == 0)
            a.w.list[st * a.w.nitems + atomicAdd(&a.w.counters[3 + st], 1u)] = TubeItem{off, (int)tube, len, cn, (int)j, 0, 0};
        }
      }
    } else {
      __syncthreads();
      if (tid == 0) fetch_item(nxt);
    }
    // ---- phase B: faces f = 0..nc (face f between chunk cells f-1 and f) ----
    const int nf = nc + 1;
    for (int f = tid; f < nf; f += NTH) {
      const int ha = f + 2, hb = f + 3, h0 = f;  // stencil cell 0 = chunk cell f-3 -> halo index f
      float rho_bar = 0.5f * (S.q[0][ha] + S.q[0][hb]);
      float c_bar = 0.5f * (S.q[5][ha] + S.q[5][hb]);
      float c2 = c_bar * c_bar, rc = rho_bar * c_bar;
      float inv = frcp(c2 * rc);
      float ic2 = rc * inv, irc = c2 * inv;
      const float mic2 = -frcp(c2);
      float2 W[NQ], Q[NQ];  // (left, right) characteristics, then primitives
#pragma unroll
      for (int r = 0; r < NQ; ++r) {
        float w[6];
        if (r == 0 || r == NQ - 1) {
          const float rcs = r == 0 ? -rc : rc;
#pragma unroll
          for (int k = 0; k < 6; ++k) w[k] = 0.5f * fmaf(rcs, S.q[1][h0 + k], S.q[2][h0 + k]);
        } else if (r == 1) {
#pragma unroll
          for (int k = 0; k < 6; ++k) w[k] = fmaf(mic2, S.q[2][h0 + k], S.q[0][h0 + k]);
        } else {
#pragma unroll
          for (int k = 0; k < 6; ++k) w[k] = S.q[r + 1][h0 + k];  // Gamma (r = 2), Pi (r = 3)
        }
        float mn = fminf(fmin3(w[0], w[1], w[2]), fmin3(w[3], w[4], w[5]));
        float mx = fmaxf(fmax3(w[0], w[1], w[2]), fmax3(w[3], w[4], w[5]));
        // both sides at once: lanes (left, right) of the mirrored stencils
        float2 p0 = make_float2(w[0], w[5]), p1 = make_float2(w[1], w[4]), p2 = make_float2(w[2], w[3]);
        float2 p3 = make_float2(w[3], w[2]), p4 = make_float2(w[4], w[1]);
        if (mx - mn <= 1e-6f * fmaxf(fabsf(mx), fabsf(mn)))
          W[r] = linear5_pair(p0, p1, p2, p3, p4);
        else
          W[r] = weno5_pair(p0, p1, p2, p3, p4, a.P);
      }
      back_project_pair<NQ>(W, ic2, irc, Q);
      int code[2] = {0, 0};
      if (a.mood) {
        float qs[2][NQ];
#pragma unroll
        for (int r = 0; r < NQ; ++r) {
          qs[0][r] = Q[r].x;
          qs[1][r] = Q[r].y;
        }
        const bool ok0 = admissible<NQ>(qs[0]), ok1 = admissible<NQ>(qs[1]);
        if (!ok0 || !ok1) {  // MOOD cascade of the failing side(s): rare
#pragma unroll 1
          for (int side = 0; side < 2; ++side) {
            if (side == 0 ? ok0 : ok1) continue;
            // 3rd-order retry (d3 = d4 = 0) of this side
            float qc[6][NQ];
#pragma unroll
            for (int k = 0; k < 6; ++k) {
#pragma unroll
              for (int m = 0; m < NQ; ++m) qc[k][m] = S.q[m][f + k];
            }
            float hrc = 0.5f * rc, wt[NQ], q3[NQ];
#pragma unroll
            for (int r = 0; r < NQ; ++r) {
              float v[5];
#pragma unroll
              for (int k = 0; k < 5; ++k) v[k] = project<NQ>(qc[side == 0 ? k : 5 - k], r, hrc, ic2);
              wt[r] = weno_is(v[0], v[1], v[2], v[3], v[4], a.P, 3);
            }
            back_project<NQ>(wt, ic2, irc, q3);
            code[side] = 1;
            if (!admissible<NQ>(q3)) {
              int hh = side == 0 ? ha : hb;
#pragma unroll
              for (int m = 0; m < NQ; ++m) q3[m] = S.q[m][hh];
              code[side] = 2;
            }
#pragma unroll
            for (int r = 0; r < NQ; ++r) {
              if (side == 0)
                Q[r].x = q3[r];
              else
                Q[r].y = q3[r];
            }
          }
        }
      }
      float Fh[NQ], us;
      hllc_pair<NQ>(Q, Fh, us);
#pragma unroll
      for (int m = 0; m < NQ; ++m) S.F[m][f] = Fh[m];
      S.F[NQ][f] = us;
      // face f sits at padded cell off + NG + c0 + f - 1 (faces -1/2 .. len-1/2 on cells off+2 .. off+len+2)
      if (a.mask) a.mask[off + NG + c0 + f - 1] = (uint8_t)(code[0] | (code[1] << 2));
    }
    if (tid == 0) fetch_rate(nxt);
    __syncthreads();
    // ---- phase C ----
    const float dt = S.dt;
    for (int cc_ = tid; cc_ < nc; cc_ += NTH) {
      int64_t gi = off + NG + c0 + cc_;
      float du = (S.F[NQ][cc_ + 1] - S.F[NQ][cc_]) * idx;
      float inc[NQ];
#pragma unroll
      for (int m = 0; m < NQ; ++m) {
        float L = -(S.F[m][cc_ + 1] - S.F[m][cc_]) * idx;
        if (m >= 3) L = fmaf(S.q[m][cc_ + NG], du, L);
        inc[m] = L;
      }
      if (a.stage == 0) {
#pragma unroll
        for (int m = 0; m < NQ; ++m) a.Kout[m * N + gi] = inc[m];
      } else if (a.stage == 1) {
#pragma unroll
        for (int m = 0; m < NQ; ++m) a.Kout[m * N + gi] = a.Kin[m * N + gi] + inc[m];
      } else {
        float d[NQ];
        bool moves = false;
#pragma unroll
        for (int m = 0; m < NQ; ++m) {
          d[m] = dt * fmaf(1.0f / 6.0f, a.Kin[m * N + gi], (2.0f / 3.0f) * inc[m]);
          moves = moves || d[m] != 0.0f;
        }
        if (moves) {  // (a cell of the chunks beside the waves often does not)
#pragma unroll
          for (int m = 0; m < NQ; ++m) a.U[m * N + gi] = a.U[m * N + gi] + f32_to_f64(d[m]);
        }
        const float* V = a.U32;
        float rho = V[gi] + d[0], mu = V[N + gi] + d[1];
        float eint = V[2 * N + gi] + (d[2] - d[4]), Gam = V[3 * N + gi] + d[3], Pi = V[4 * N + gi] + d[4];
        float pe = fmaf(-0.5f, mu * mu * frcp(rho), eint);
        bool ok = rho > 0.0f && Gam > 0.0f && fmaf(Gam + 1.0f, pe * frcp(Gam), Pi) > 0.0f;
        if (!ok) atomicAdd(a.nbad, 1ULL);
      }
    }
    __syncthreads();  // shared memory is reused by the next item
    if (tid == 0) take(nxt);
  }
}

template <int CH, int NTH>
void launch_one(const TubeArgs& a, int ctas_per_sm, cudaStream_t s) {
  static bool prepared = false;
  if (!prepared) {
    cudaFuncSetAttribute(k_tube_stage<CH, NTH>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)sizeof(TSmem<CH>));
    prepared = true;
  }
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  int64_t grid = (int64_t)sms * ctas_per_sm;
  if (grid > a.w.nitems) grid = a.w.nitems > 0 ? a.w.nitems : 1;
  k_tube_stage<CH, NTH><<<(int)grid, NTH, sizeof(TSmem<CH>), s>>>(a);
}

}  // namespace

// configurations the autotuner chooses from: chunk size x threads (a chunk of
// 2^k - 1 cells has 2^k faces)
const int kTubeConfigs[][2] = {{255, 128}, {255, 256}, {511, 256}, {511, 512}, {1023, 512}};
const int kNumTubeConfigs = 5;

int tube_chunk_size(int config) { return kTubeConfigs[config][0]; }

// The configuration of a new context, for `cells` cells: the smallest chunks
// leave the most cells out where the tubes are quiet (4096 tubes, half of their
// cells quiet: 607 us per step, against 643, 674, 839 and 864 us for the
// others in turn; none quiet: 1378 against 1363 and 1344).  A batch that does
// not fill the GPU with them takes a face to a thread (32 tubes of 100 to 1000
// cells: 29 us against 36).
int tube_default_config(int64_t cells) { return cells >= 255LL * 152 * 8 ? 0 : 1; }

void launch_tubes_stage_mixed(const TubesDev& t, int config, int stage, double* U, float* U32, float* Ka, float* Kb,
                              double dt_fixed, double cfl, unsigned long long* lmax, double* dt_out,
                              const TubeWork& work, uint8_t* mask, int64_t nmask, float eps_rel, int mood, int weights,
                              unsigned long long* nbad, cudaStream_t s) {
  TubeArgs a;
  a.t = t;
  a.stage = stage;
  a.U = U;
  a.U32 = U32;
  a.Kin = stage == 1 ? Ka : Kb;
  a.Kout = stage == 0 ? Ka : Kb;
  a.Knext = Kb;
  a.dt_fixed = dt_fixed;
  a.cfl = (float)cfl;
  a.lmax = lmax;
  a.dt_out = dt_out;
  a.w = work;
  a.mask = mask ? mask + stage * nmask : nullptr;
  a.nmask = nmask;
  a.P = weno_params(eps_rel, weights);
  a.mood = mood;
  a.nbad = nbad;
  switch (config) {
    case 0: launch_one<255, 128>(a, 8, s); break;
    case 1: launch_one<255, 256>(a, 4, s); break;
    case 2: launch_one<511, 256>(a, 4, s); break;
    case 3: launch_one<511, 512>(a, 2, s); break;
    default: launch_one<1023, 512>(a, 2, s); break;
  }
}

}  // namespace ws
