// FP64 arithmetic of the faces i+1/2 (shared by the grid sweep and the
// batched-tube sweep; both translation units are built with -fmad=false):
// characteristic projection (Sec. 3.2), WENO-IS reconstruction of both sides
// (Secs. 3.3.1, 3.3.2), back-projection, MOOD positivity cascade (Sec. 3.4)
// and the stiffened-gas HLLC flux and face velocity (Sec. 3.2.1).
//
// Every value is the one that a plain evaluation of the formulas gives, one
// IEEE binary64 operation at a time in the order written there, bit for bit
// (up to the sign of a zero flux).  The FP64 pipe takes 76 cycles per warp
// instruction and is what bounds these kernels, so the evaluation spends as
// few instructions on it as that allows:
//  - divisions run on the integer and FP32 pipes (fp64_pipes.cuh), in large
//    launches the products too;
//  - products by powers of two are exact, so they fold into the next addition
//    (a fused multiply-add of an exact product rounds once, like the
//    addition alone) or move out of a product;
//  - an epsilon that cannot change a smoothness indicator is not added;
//  - a warp whose stencils are constant to the last bit skips the
//    reconstruction, whose increments are zeros;
//  - of HLLC's two star fluxes only the one the contact speed selects is
//    formed (both where the other could contribute: S* = 0, or a value that
//    is not finite).
// The characteristic matrices are applied through their non-zero entries.
//
// A face belongs to a pair of lanes, one per side, and a characteristic
// variable to a warp; the reconstructed values meet in shared memory, where one
// warp of the CTA solves the Riemann problems.  Even the 200 faces of a short
// tube then spread over the GPU, and a warp runs one variable's code.
#pragma once

#include "fp64_pipes.cuh"
#include "ws_internal.h"

namespace ws {
namespace fp64 {

constexpr int FPW = 16;                 // faces per CTA (a warp's 32 lanes are 16 pairs)
constexpr unsigned ALL = 0xffffffffu;

// weights and epsilon of a launch: modified or basic (IS), or JS.  LITERAL:
// modified or basic weights with an unusual epsilon; every operation as
// written.  IS needs eps >= 1e-50 (2^-166): a smoothness indicator or tau_5
// below 2^-400 then changes no weight, and no weight overflows.
enum Scheme { IS = 0, JS = 1, LITERAL = 2 };
inline Scheme scheme_of(double eps, int weights) {
  if (weights == WS_W_JS) return eps >= 1e-50 && eps <= 1e50 ? JS : LITERAL;
  return eps >= 1e-50 && eps <= 1e50 ? IS : LITERAL;
}

// Where a launch runs what is not an addition.  NATIVE: everything by the
// compiler's FP64 instructions.  CHAIN: divisions and roots on the integer
// pipe.  PIPES: products there too.
enum Pipes { NATIVE = 0, CHAIN = 1, PIPES = 2 };
template <int PI>
__device__ __forceinline__ double square(double a, uint32_t& rg) {  // zero below 2^-510 with PIPES
  return PI == PIPES ? isquare(a, rg) : __dmul_rn(a, a);
}
template <int PI>
__device__ __forceinline__ double coef(double c, double a, uint32_t& rg) {  // c: a constant
  return PI == PIPES ? imul_const(c, a, rg) : __dmul_rn(c, a);
}
template <int PI>
__device__ __forceinline__ double mul(double a, double b, uint32_t& rg) {
  return PI == PIPES ? imul(a, b, rg) : __dmul_rn(a, b);
}
template <int PI>
__device__ __forceinline__ double sqroot(double x, uint32_t& rg) {
  return PI == NATIVE ? sqrt(x) : (PI == CHAIN ? root_call(x) : isqrt(x, rg));
}
// The divisions are calls: inlined, the code of a large sweep is a fifth longer
// and its warps wait for instructions (512^2 shock-bubble, us per step: 2278
// inlined, 2159 with those of the Riemann problem called, 2045 with all; the
// 48^3 drop 1794, 1790, 1789).  Roots or products as calls gained nothing.
template <int PI>
__device__ __forceinline__ double quot(double a, double b) {
  return PI == NATIVE ? a / b : divide_call(a, b);
}
// A launch of many CTAs (NQ chunks of faces each) is bound by the pipes, and
// its products go to the integer pipe; one of few CTAs is bound by the length
// of its dependency chains: one chunk to a CTA, and products on the FP64 pipe,
// where their latency is shorter.  The line lies at two CTAs per SM; us per step
// as small and as large launch: 108^2 (246 CTAs) 234, 241; 122^2 (314) 270, 292;
// 140^2 (412) 320, 306; 19^3 (195) 282, 324; 22^3 (300) 371, 332; 24^3 (387) 447,
// 360.
inline bool large_sweep(unsigned ctas) { return ctas >= 152 * 2; }

__device__ __forceinline__ double fma_exact(double two_k, double a, double b) { return __fma_rn(two_k, a, b); }
__device__ __forceinline__ double partner(double x) { return __shfl_xor_sync(ALL, x, 1); }

// WENO-JS (Jiang & Shu 1996) as written, the paper's comparison scheme:
// candidates on S_0 = {i-2,i-1,i}, S_1 = {i-1,i,i+1}, S_2 = {i,i+1,i+2} (the
// paper's S_4, S_12, S_3), d = (1,6,3)/10, alpha_k = d_k/(eps+beta_k)^2.
static __device__ __noinline__ double weno_js_literal(double qm2, double qm1, double q0, double qp1, double qp2,
                                                      double eps) {
  const double c13_12 = 13.0 / 12.0;
  double delta3 = ((5.0 / 6.0) * (qp1 - q0)) - ((1.0 / 6.0) * (qp2 - q0));
  double delta4 = ((1.0 / 3.0) * (qm2 - q0)) - ((7.0 / 6.0) * (qm1 - q0));
  double deltaC = ((1.0 / 3.0) * (qp1 - q0)) - ((1.0 / 6.0) * (qm1 - q0));
  double a, b;
  a = (q0 - 2.0 * qp1) + qp2;
  b = ((3.0 * q0) - (4.0 * qp1)) + qp2;
  double beta3 = (c13_12 * (a * a)) + (0.25 * (b * b));
  a = (qm2 - 2.0 * qm1) + q0;
  b = (qm2 - (4.0 * qm1)) + (3.0 * q0);
  double beta4 = (c13_12 * (a * a)) + (0.25 * (b * b));
  a = (qm1 - 2.0 * q0) + qp1;
  b = qm1 - qp1;
  double beta12 = (c13_12 * (a * a)) + (0.25 * (b * b));
  double e0 = eps + beta4, e1 = eps + beta12, e2 = eps + beta3;
  double a0 = 1.0 / (e0 * e0);
  double a1 = 6.0 / (e1 * e1);
  double a2 = 3.0 / (e2 * e2);
  double num = ((a0 * delta4) + (a1 * deltaC)) + (a2 * delta3);
  double den = (a0 + a1) + a2;
  return q0 + num / den;
}

// Sec. 3.3.1-3.3.2 as written: left value at x_{i+1/2} from q_{i-2..i+2};
// order 5: all four candidates; order 3: d3 = d4 = 0.  The MOOD retry, the
// LITERAL scheme and operands outside the range of fp64_pipes.cuh.  WENO-JS
// has no 3rd order of its own: it takes the modified weights there.
static __device__ __noinline__ double weno_literal(double qm2, double qm1, double q0, double qp1, double qp2, double eps,
                                            int order, int weights) {
  if (weights == WS_W_JS && order == 5) return weno_js_literal(qm2, qm1, q0, qp1, qp2, eps);
  const double c13_12 = 13.0 / 12.0;
  // Eq. (candidates) as increments about q_i
  double delta1 = 0.5 * (qp1 - q0);
  double delta2 = 0.5 * (q0 - qm1);
  double delta3 = ((5.0 / 6.0) * (qp1 - q0)) - ((1.0 / 6.0) * (qp2 - q0));
  double delta4 = ((1.0 / 3.0) * (qm2 - q0)) - ((7.0 / 6.0) * (qm1 - q0));
  // Eq. (smoothness-indicator), beta_12 and Eq. (tau-5)
  double a, b;
  a = qp1 - q0;
  double beta1 = a * a;
  a = q0 - qm1;
  double beta2 = a * a;
  a = (qm1 - 2.0 * q0) + qp1;
  b = qm1 - qp1;
  double beta12 = (c13_12 * (a * a)) + (0.25 * (b * b));
  a = ((qp2 - 2.0 * qp1) + 2.0 * qm1) - qm2;
  b = ((((qp2 - 4.0 * qp1) + 6.0 * q0) - 4.0 * qm1) + qm2);
  double tau5 = (0.25 * (a * a)) + (c13_12 * (b * b));
  // Eq. (weighting-modification) / Eq. (weight-new) with q = 1
  double r1 = tau5 / (beta1 + eps);
  double r2 = tau5 / (beta2 + eps);
  double alpha1, alpha2;
  if (weights != WS_W_BASIC) {
    double r12 = tau5 / (beta12 + eps);
    alpha1 = 4.0 * (1.0 + r1 * r12);
    alpha2 = 2.0 * (1.0 + r2 * r12);
  } else {
    alpha1 = 4.0 * (1.0 + r1);
    alpha2 = 2.0 * (1.0 + r2);
  }
  double num = (alpha1 * delta1) + (alpha2 * delta2);
  double den = alpha1 + alpha2;
  if (order == 5) {
    a = (q0 - 2.0 * qp1) + qp2;
    b = ((3.0 * q0) - (4.0 * qp1)) + qp2;
    double beta3 = (c13_12 * (a * a)) + (0.25 * (b * b));
    a = (qm2 - 2.0 * qm1) + q0;
    b = (qm2 - (4.0 * qm1)) + (3.0 * q0);
    double beta4 = (c13_12 * (a * a)) + (0.25 * (b * b));
    double alpha3 = 3.0 * (1.0 + tau5 / (beta3 + eps));
    double alpha4 = 1.0 * (1.0 + tau5 / (beta4 + eps));
    num = (num + (alpha3 * delta3)) + (alpha4 * delta4);
    den = (den + alpha3) + alpha4;
  }
  // Eq. (final-weighting) with omega_k = alpha_k / sum(alpha)
  return q0 + num / den;
}

// The 5th-order value, the same operations with exact products folded (of
// the 139 FP64-pipe instructions of the plain form about 70 remain).  thr: the
// high word above which a smoothness indicator is at least 2^54 eps, so that
// adding eps leaves it.
template <Scheme SC, int PI>
__device__ __forceinline__ double weno5(double qm2, double qm1, double q0, double qp1, double qp2, double eps, int thr,
                                        int weights) {
  if (SC == LITERAL) return weno_literal(qm2, qm1, q0, qp1, qp2, eps, 5, weights);
  // values below 2^150 (twice the high word leaves out the sign): no overflow anywhere
  const uint32_t most = max(max(max(hi_of(qm2) << 1, hi_of(qm1) << 1), max(hi_of(qp1) << 1, hi_of(qp2) << 1)), hi_of(q0) << 1);
  uint32_t rg = most < ((1023u + 150u) << 21) ? kInRange : 0u;
  const double c13_12 = 13.0 / 12.0;
  const double dp = qp1 - q0, dm = q0 - qm1;
  const double t3 = coef<PI>(3.0, q0, rg);
  // (13/12) a^2 + b^2/4
  auto beta_of = [&](double a, double b) {
    return fma_exact(0.25, square<PI>(b, rg), coef<PI>(c13_12, square<PI>(a, rg), rg));
  };
  double beta3 = beta_of(fma_exact(-2.0, qp1, q0) + qp2, fma_exact(-4.0, qp1, t3) + qp2);
  double beta4 = beta_of(fma_exact(-2.0, qm1, qm2) + q0, fma_exact(-4.0, qm1, qm2) + t3);
  double num, den;
  if (SC == JS) {  // WENO-JS: candidates on S_4, S_12, S_3 with d = (1,6,3)/10
    const double delta3 = coef<PI>(5.0 / 6.0, dp, rg) - coef<PI>(1.0 / 6.0, qp2 - q0, rg);
    const double delta4 = coef<PI>(1.0 / 3.0, qm2 - q0, rg) + coef<PI>(7.0 / 6.0, dm, rg);
    const double deltaC = coef<PI>(1.0 / 3.0, dp, rg) + coef<PI>(1.0 / 6.0, dm, rg);
    const double beta12 = beta_of(fma_exact(-2.0, q0, qm1) + qp1, qm1 - qp1);
    const double e0 = eps + beta4, e1 = eps + beta12, e2 = eps + beta3;
    const double a0 = quot<PI>(1.0, mul<PI>(e0, e0, rg)), a1 = quot<PI>(6.0, mul<PI>(e1, e1, rg)),
                 a2 = quot<PI>(3.0, mul<PI>(e2, e2, rg));
    num = (mul<PI>(a0, delta4, rg) + mul<PI>(a1, deltaC, rg)) + mul<PI>(a2, delta3, rg);
    den = (a0 + a1) + a2;
  } else {
    double beta1 = square<PI>(dp, rg), beta2 = square<PI>(dm, rg);
    double beta12 = 1.0;
    if (weights != WS_W_BASIC) beta12 = beta_of(fma_exact(-2.0, q0, qm1) + qp1, qm1 - qp1);
    const double ta = fma_exact(2.0, qm1, fma_exact(-2.0, qp1, qp2)) - qm2;
    const double tb = fma_exact(-4.0, qm1, fma_exact(2.0, t3, fma_exact(-4.0, qp1, qp2))) + qm2;
    double tau5 = beta_of(tb, ta);
    if (hi_of(tau5) < ((1023u - 400u) << 20)) tau5 = 0.0;
    int least = min((int)hi_of(beta1), (int)hi_of(beta2));
    least = min(min((int)hi_of(beta12), least), min((int)hi_of(beta3), (int)hi_of(beta4)));
    if (least < thr) {
      beta1 = beta1 + eps;
      beta2 = beta2 + eps;
      beta12 = beta12 + eps;
      beta3 = beta3 + eps;
      beta4 = beta4 + eps;
    }
    const double r1 = quot<PI>(tau5, beta1), r2 = quot<PI>(tau5, beta2);
    double A, B;  // alpha1 / 4, alpha2 / 2
    if (weights != WS_W_BASIC) {
      const double r12 = quot<PI>(tau5, beta12);
      A = 1.0 + mul<PI>(r1, r12, rg);
      B = 1.0 + mul<PI>(r2, r12, rg);
    } else {
      A = 1.0 + r1;
      B = 1.0 + r2;
    }
    const double alpha3 = coef<PI>(3.0, 1.0 + quot<PI>(tau5, beta3), rg), alpha4 = 1.0 + quot<PI>(tau5, beta4);
    check_or_zero(rg, hi_of(dp), is_zero(dp));  // far from the subnormal range: halves are exact
    check_or_zero(rg, hi_of(dm), is_zero(dm));
    num = fma_exact(2.0, mul<PI>(A, dp, rg), mul<PI>(B, dm, rg));  // alpha1 delta1 + alpha2 delta2
    den = fma_exact(2.0, fma_exact(2.0, A, B), alpha3) + alpha4;   // (alpha1 + alpha2) / 2 first
    const double delta3 = coef<PI>(5.0 / 6.0, dp, rg) - coef<PI>(1.0 / 6.0, qp2 - q0, rg);
    const double delta4 = coef<PI>(1.0 / 3.0, qm2 - q0, rg) + coef<PI>(7.0 / 6.0, dm, rg);
    num = (num + mul<PI>(alpha3, delta3, rg)) + mul<PI>(alpha4, delta4, rg);
  }
  const double v = q0 + quot<PI>(num, den);
  if (!in_range(rg)) return weno_literal(qm2, qm1, q0, qp1, qp2, eps, 5, SC == JS ? WS_W_JS : weights);
  return v;
}

__device__ __forceinline__ double sound_speed2(double rho, double p, double Gam, double Pi) {
  return divide(((Gam + 1.0) * p) + Pi, Gam * rho);
}

// Characteristic variable r of the sweep-frame primitive q
// (rho, u_n, u_t.., p, Gamma, Pi): row r of L_{i+1/2} in Eq. (eigen-vectors).
template <int NQ>
__device__ __forceinline__ double project(const double* q, int r, double L01, double L1p, double L51) {
  constexpr int NT = NQ - 5, IP = 2 + NT;
  if (r == 0) return (L01 * q[1]) + (0.5 * q[IP]);
  if (r == 1) return q[0] + (L1p * q[IP]);
  if (r == NQ - 1) return (L51 * q[1]) + (0.5 * q[IP]);
  if (r < IP) return q[r];      // shear
  return q[r + 1];              // Gamma, Pi
}

// q = R_{i+1/2} w (Eq. back-projected), with R00 = 1/c^2, irc = 1/(rho c)
template <int NQ>
__device__ __forceinline__ void back_project(const double* w, double R00, double irc, double* q) {
  constexpr int NT = NQ - 5, IP = 2 + NT;
  q[0] = ((R00 * w[0]) + w[1]) + (R00 * w[NQ - 1]);
  q[1] = (irc * w[NQ - 1]) - (irc * w[0]);
#pragma unroll
  for (int t = 0; t < NT; ++t) q[2 + t] = w[2 + t];
  q[IP] = w[0] + w[NQ - 1];
  q[IP + 1] = w[IP];
  q[IP + 2] = w[IP + 1];
}

template <int NQ>
__device__ __forceinline__ bool admissible(const double* q) {
  return positive(q[0]) && positive(q[NQ - 2]) && positive(((q[NQ - 2] + 1.0) * q[NQ - 3]) + q[NQ - 1]);
}

// Where the six cells of a lane pair's face lie: cell i-2+j at base + j st of
// every primitive field; field m of the sweep frame (rho, u_n, u_t.., p,
// Gamma, Pi) starts at q + fld(m) N, the sound speed at q + NQ N.
// SH: the fields lie in shared memory.
template <int NQ_, bool SH_ = false>
struct Faces {
  static constexpr int NQ = NQ_;
  const double* q;
  int64_t N, base, st;
  int d;
  __device__ __forceinline__ int fld(int m) const {  // global field of sweep-frame field m
    if (m == 0 || m >= NQ - 3) return m;
    if (m == 1) return 1 + d;
    return m - 2 < d ? m - 1 : m;  // tangential velocities in increasing axis order
  }
  __device__ __forceinline__ double at(int f, int j) const {
    const double* p = q + (int64_t)f * N + base + j * st;
    return SH_ ? *p : __ldg(p);
  }
};

// The MOOD retry of one side: 3rd order, then the cell's own state.  Rare.
template <int NQ, bool SH>
__device__ __noinline__ int retry(const Faces<NQ, SH> fc, int side, double eps, int weights, double* q) {
  double qc[6][NQ];
#pragma unroll 1
  for (int j = 0; j < 6; ++j)
    for (int m = 0; m < NQ; ++m) qc[j][m] = fc.at(fc.fld(m), j);
  const double rho_bar = 0.5 * (qc[2][0] + qc[3][0]);
  const double c_bar = 0.5 * (fc.at(NQ, 2) + fc.at(NQ, 3));
  const double rc = rho_bar * c_bar, c2 = c_bar * c_bar;
  const double L01 = -rc / 2.0, L51 = rc / 2.0, L1p = -1.0 / c2;
  double wt[NQ];
#pragma unroll 1
  for (int r = 0; r < NQ; ++r) {
    double v[5];
    for (int k = 0; k < 5; ++k) v[k] = project<NQ>(qc[side == 0 ? k : 5 - k], r, L01, L1p, L51);
    wt[r] = weno_literal(v[0], v[1], v[2], v[3], v[4], eps, 3, weights == WS_W_JS ? WS_W_MODIFIED : weights);
  }
  back_project<NQ>(wt, 1.0 / c2, 1.0 / rc, q);
  if (admissible<NQ>(q)) return 1;
  for (int r = 0; r < NQ; ++r) q[r] = qc[2 + side][r];  // Eq. (upwind)
  return 2;
}

// Sec. 3.2.1: HLLC flux and face velocity of a lane pair's face from the
// state q of each lane's side.  The lanes of a pair end with half of the
// results each: out[j] is component (side ? H : 0) + j, where components
// 0..NQ-1 are the fluxes and component NQ the face velocity.
template <int NQ, int PI>
__device__ __forceinline__ bool hllc_pair(const double (&q)[NQ], int side, double (&out)[(NQ + 2) / 2]) {
  constexpr int NT = NQ - 5, IP = 2 + NT, H = (NQ + 2) / 2;
  uint32_t rg = kInRange;
  const double rho = q[0], un = q[1], p = q[IP], Gam = q[IP + 1], Pi = q[IP + 2];
  // |q| < 2^150: no overflow below
  uint32_t most = hi_of(q[0]) << 1;
#pragma unroll
  for (int m = 1; m < NQ; ++m) most = max(most, hi_of(q[m]) << 1);
  const bool moderate = most < ((1023u + 150u) << 21);
  if (!moderate) rg = 0u;
  // a sum that a square below 2^-510 times 2^150 (taken as zero) cannot change
  auto covers = [&](double x) { if ((hi_of(x) & 0x7fffffffu) < ((1023u - 250u) << 20)) rg = 0u; };
  double usq = square<PI>(un, rg);
#pragma unroll
  for (int t = 0; t < NT; ++t) usq = usq + square<PI>(q[2 + t], rg);
  const double ei = mul<PI>(Gam, p, rg) + Pi;
  covers(ei);
  const double E = PI == NATIVE ? ei + (0.5 * rho) * usq : fma_exact(0.5, mul<PI>(rho, usq, rg), ei);
  const double mn = mul<PI>(rho, un, rg);
  // conserved state and flux; component NQ: the face velocity as S 1 - un
  double U[2 * H], F[2 * H];
  U[0] = rho;
  F[0] = mn;
  U[1] = mn;
  F[1] = mul<PI>(mn, un, rg) + p;
#pragma unroll
  for (int t = 0; t < NT; ++t) {
    U[2 + t] = mul<PI>(rho, q[2 + t], rg);
    F[2 + t] = mul<PI>(mn, q[2 + t], rg);
  }
  U[IP] = E;
  F[IP] = mul<PI>(E + p, un, rg);
  U[IP + 1] = Gam;
  F[IP + 1] = mul<PI>(Gam, un, rg);
  U[IP + 2] = Pi;
  F[IP + 2] = mul<PI>(Pi, un, rg);
#pragma unroll
  for (int m = NQ; m < 2 * H; ++m) {
    U[m] = 1.0;
    F[m] = un;
  }
  const double c2 = quot<PI>(mul<PI>(Gam + 1.0, p, rg) + Pi, mul<PI>(Gam, rho, rg));
  const double cc = sqroot<PI>(c2, rg), s = sqroot<PI>(rho, rg);
  // Eq. (wave-speeds): lane 0 divides for u_bar, lane 1 for the averaged c^2
  const double so = partner(s), den = s + so;
  const double pu = mul<PI>(s, un, rg), pc = mul<PI>(s, c2, rg);
  const double avg = quot<PI>((side ? pc : pu) + partner(side ? pu : pc), den);
  const double avgo = partner(avg);
  const double ubar = side ? avgo : avg, c2avg = side ? avg : avgo;
  const double du = un - partner(un);
  covers(c2avg);
  const double ss = mul<PI>(s, so, rg), dd = mul<PI>(den, den, rg), duu = square<PI>(du, rg);
  const double c2bar =
      PI == NATIVE ? c2avg + ((0.5 * ss) / dd) * duu : fma_exact(0.5, mul<PI>(quot<PI>(ss, dd), duu, rg), c2avg);
  const double cbar = sqroot<PI>(c2bar, rg);
  // S_l = min(u_bar - c_bar, u_l - c_l, 0); S_r as minus the minimum of the negatives
  const double sg = side ? -1.0 : 1.0;
  const double ux = side ? -ubar : ubar, uy = side ? -un : un;
  const double S = sg * fmin(fmin(ux - cbar, uy - cc), 0.0);
  // Eq. (wave-speed)
  const double Sm = S - un, ms = mul<PI>(rho, Sm, rg), ks = mul<PI>(mn, Sm, rg);
  const double po = partner(p), ko = partner(ks), mo = partner(ms);
  const double num = (((side ? p - po : po - p)) + (side ? ko : ks)) - (side ? ks : ko);
  const double Ss = quot<PI>(num, side ? mo - ms : ms - mo);
  auto small = [](double x) { return (hi_of(x) & 0x7fffffffu) < ((1023u + 150u) << 20); };
  if (!(small(S) && small(Ss))) rg = 0u;  // no product below exceeds 2^700
  // Eq. (flux-function), D* = (0, 1, 0.., S*, 0, 0), and Eq. (velocities)
  const double SP = mul<PI>(S, p + mul<PI>(ms, Ss - un, rg), rg), SPS = mul<PI>(SP, Ss, rg);
  const double dS = S - Ss;
  // only the side that S* selects contributes if the other's flux is finite
  const bool ok = moderate && small(S) && small(Ss) && small(E) && small(dS) && (hi_of(dS) & 0x7fffffffu) > ((1023u - 150u) << 20) &&
            !is_zero(Ss);
  const unsigned b = __ballot_sync(ALL, ok);
  const unsigned pair = 3u << (threadIdx.x & 30u);
  const bool one = (b & pair) == pair;
  const unsigned ones = __ballot_sync(ALL, one), act = one ? ones : ~ones;  // the lanes of this branch
  if (one) {
    const bool right = (int)hi_of(Ss) < 0;  // S* < 0 selects the right side (lane 1)
    const bool own = right == (side != 0);
    const int src = (threadIdx.x & 30) + (right ? 1 : 0);
    const double Sk = __shfl_sync(act, S, src), dk = __shfl_sync(act, dS, src);
    const double SPk = __shfl_sync(act, SP, src), SPSk = __shfl_sync(act, SPS, src);
#pragma unroll
    for (int j = 0; j < H; ++j) {
      const double xu = __shfl_xor_sync(act, side ? U[j] : U[H + j], 1), xf = __shfl_xor_sync(act, side ? F[j] : F[H + j], 1);
      const double u = own ? (side ? U[H + j] : U[j]) : xu, f = own ? (side ? F[H + j] : F[j]) : xf;
      double t = mul<PI>(Ss, mul<PI>(Sk, u, rg) - f, rg);
      // -0.0 leaves t as it is
      if (j == 1) t = t + (side ? (IP == H + 1 ? SPSk : -0.0) : SPk);
      if (j == IP || (j + H == IP && j != 1)) t = t + ((side ? H + j : j) == IP ? SPSk : -0.0);
      out[j] = quot<PI>(t, dk);
    }
  } else {
    const double w = Ss > 0.0 ? (side ? 0.0 : 1.0) : (Ss < 0.0 ? (side ? 1.0 : 0.0) : 0.5);
    double c[2 * H];
#pragma unroll
    for (int m = 0; m < 2 * H; ++m) {
      double t = Ss * ((S * U[m]) - F[m]);
      if (m == 1) t = t + SP;
      if (m == IP) t = t + SPS;
      t = S == Ss ? F[m] : quot<PI>(t, dS);
      c[m] = w * t;
    }
    // Eq. (hllc-flux)
#pragma unroll
    for (int j = 0; j < H; ++j) {
      const double x = __shfl_xor_sync(act, side ? c[j] : c[H + j], 1);
      out[j] = (side ? c[H + j] : c[j]) + x;
    }
  }
  return PI == NATIVE || in_range(rg);
}

template <int NQ>
__device__ __noinline__ void hllc_native(const double (&q)[NQ], int side, double (&out)[(NQ + 2) / 2]) {
  hllc_pair<NQ, NATIVE>(q, side, out);
}

template <int NQ, int CH>
struct FaceSmem {
  double w[CH][NQ][32];  // reconstructed characteristics of the lane pairs of CH chunks
  int next;              // the first (variable, chunk) no warp has taken yet
};

// The reconstruction of characteristic variable r on a warp's lane pairs.
template <int NQ, Scheme SC, int PI, bool SH>
__device__ __forceinline__ double reconstruct(const Faces<NQ, SH>& fc, int r, double eps, int weights) {
  constexpr int IP = NQ - 3;
  const int side = threadIdx.x & 1;
  auto cell = [&](int k) { return side ? 5 - k : k; };  // this side's stencil cell k
  double v[5];
  if (r < 2 || r == NQ - 1) {
    const int s1 = fc.fld(1);
    const double c = fc.at(NQ, cell(2)), s2 = c + partner(c);  // 2 c_bar
    if (r == 1) {
      const double L1p = quot<PI>(-4.0, __dmul_rn(s2, s2));  // -1/c_bar^2
#pragma unroll
      for (int k = 0; k < 3; ++k) v[k] = fc.at(0, cell(k)) + __dmul_rn(L1p, fc.at(IP, cell(k)));
    } else {
      const double rho = fc.at(0, cell(2));
      const double hrc = 0.125 * __dmul_rn(rho + partner(rho), s2);  // rho_bar c_bar / 2
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const double x = __dmul_rn(hrc, fc.at(s1, cell(k)));
        v[k] = fma_exact(0.5, fc.at(IP, cell(k)), r == 0 ? -x : x);
      }
    }
  } else {  // shear, Gamma, Pi
    const int f = fc.fld(r < IP ? r : r + 1);
#pragma unroll
    for (int k = 0; k < 3; ++k) v[k] = fc.at(f, cell(k));
  }
  v[3] = partner(v[2]);
  v[4] = partner(v[1]);
  // a constant stencil (the increments are zeros and the weights finite)
  const long long b0 = __double_as_longlong(v[0]);
  const bool flat = SC != LITERAL && b0 == __double_as_longlong(v[1]) && b0 == __double_as_longlong(v[2]) &&
                    b0 == __double_as_longlong(v[3]) && b0 == __double_as_longlong(v[4]) &&
                    (hi_of(v[0]) & 0x7fffffffu) < ((1023u + 150u) << 20);
  if (__all_sync(ALL, flat)) return v[2] + 0.0;
  return weno5<SC, PI>(v[0], v[1], v[2], v[3], v[4], eps, (int)hi_of(eps) + (55 << 20), weights);
}

// The Riemann problem of a warp's lane pairs from the reconstructed
// characteristics w; code: this side's MOOD level.
template <int NQ, int PI, bool SH>
__device__ __forceinline__ void solve(const Faces<NQ, SH>& fc, const double (&w)[NQ], double eps, int mood, int weights,
                                      double (&out)[(NQ + 2) / 2], int& code) {
  const int side = threadIdx.x & 1, own = 2 + side;
  double q[NQ];
  {
    const double c = fc.at(NQ, own), s2 = c + partner(c);
    const double rho = fc.at(0, own), s1 = rho + partner(rho);
    const double cc = __dmul_rn(s2, s2), rc = __dmul_rn(s1, s2);
    back_project<NQ>(w, quot<PI>(4.0, cc), quot<PI>(4.0, rc), q);
  }
  code = 0;
  if (mood && !admissible<NQ>(q)) {
    double q3[NQ];
    code = retry(fc, side, eps, weights, q3);
#pragma unroll
    for (int m = 0; m < NQ; ++m) q[m] = q3[m];
  }
  __syncwarp();
  const bool fine = hllc_pair<NQ, PI>(q, side, out);
  if (!__all_sync(ALL, fine)) hllc_native<NQ>(q, side, out);
}

// The faces of one CTA of NQ warps: CH chunks of FPW faces, first a variable of
// a chunk to a warp, then a chunk to a warp.  at(k) places chunk k, done(k, fc,
// out, code) takes its results (called by the warps that hold them).  With CH =
// NQ every warp works in both parts; CH = 1 spreads a short sweep over more SMs.
// Variables differ in work (constant ones have none), so warps take the next
// (variable, chunk) as they become free; with a fixed variable to each a quarter
// of their time went into the barrier (512^2 shock-bubble, us per step: 2096
// fixed, 2035 taken chunk by chunk, 2006 variable by variable, which keeps the
// warps in the same code; the 48^3 drop 1790, 1747, 1722.  2, 3, 4, 8 and 12
// warps and chunks to a CTA: 2101, 2089, 2018, 2002, 2064).
template <int NQ, int CH, Scheme SC, int PI, class At, class Done>
__device__ __forceinline__ void cta_faces(FaceSmem<NQ, CH>& sm, double eps, int mood, int weights, At at, Done done) {
  const int lane = threadIdx.x & 31, r = threadIdx.x >> 5;
  if (CH > 1) {
    if (threadIdx.x == 0) sm.next = CH;
    __syncthreads();
#pragma unroll 1
    for (int i = r; i < CH * NQ;) {
      const int m = i / CH, k = i - m * CH;
      sm.w[k][m][lane] = reconstruct<NQ, SC, PI>(at(k), m, eps, weights);
      if (lane == 0) i = atomicAdd(&sm.next, 1);
      i = __shfl_sync(ALL, i, 0);
    }
  } else {
    sm.w[0][r][lane] = reconstruct<NQ, SC, PI>(at(0), r, eps, weights);
  }
  __syncthreads();
  // (CH = 1: a different warp from CTA to CTA, so that the SM's sub-partitions share the work)
  const int k = CH == 1 ? (r + (int)(blockIdx.x % NQ)) % NQ : r;
  if (k >= CH) return;
  double w[NQ], out[(NQ + 2) / 2];
  int code;
#pragma unroll
  for (int m = 0; m < NQ; ++m) w[m] = sm.w[k][m][lane];
  const auto fc = at(k);
  solve<NQ, PI>(fc, w, eps, mood, weights, out, code);
  done(k, fc, out, code);
}

}  // namespace fp64
}  // namespace ws
