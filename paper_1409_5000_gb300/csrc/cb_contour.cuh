// FP64 building blocks for functions of the small Lanczos tridiagonal T.
//
//  * lambda_max: the largest eigenvalue of T, bracketed in FP32 by a warp-wide
//    multisection on the signs of the pivots of xI - T, then the FP64 Rayleigh
//    quotient of an eigenvector from inverse iteration.
//  * lambda_max_laguerre: the same by Laguerre's iteration on det(xI - T),
//    started above the Gershgorin bound.  For a polynomial with only real
//    roots, Laguerre's method started above the largest root decreases
//    monotonically to it and converges cubically.
//  * contour nodes: exp(x) on (-inf, 0] as the trapezoid rule for the
//    Cauchy integral over the cotangent contour of Trefethen, Weideman &
//    Schmelzer ("Talbot quadratures and rational approximations", BIT 46,
//    2006): z(t) = N (a t cot(b t) - c + i d t), N = 24, error ~2e-14.
//    Nodes come in conjugate pairs; only the 12 in the upper half plane are
//    evaluated and the real result is 2 Re of their sum.
//  * continuants: (z I - (T - theta I))^{-1} e1 for the 12 nodes z at once.
#pragma once

#include <cmath>

#include "cb_internal.cuh"

namespace cb {
namespace contour {

constexpr int kNodes = 24;
constexpr int kHalf = kNodes / 2;
constexpr long double kA = 0.5017L, kB = 0.6407L, kC = 0.6122L, kD = 0.2645L;

struct cplx {
  double re, im;
};
__device__ __forceinline__ cplx cmul(cplx a, cplx b) {
  return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re};
}
__device__ __forceinline__ cplx cinv(cplx a) {
  const double d = 1.0 / (a.re * a.re + a.im * a.im);
  return {a.re * d, -a.im * d};
}

// 1 / r for r in the normal FP32 range: an FP32 reciprocal refined by two
// Newton-Raphson steps y <- y + y (1 - r y), which double the correct bits
// each (23 -> 46 -> all).
__device__ __forceinline__ double rcp_nr(double r) {
  double y = (double)__frcp_rn((float)r);
  y = fma(y, fma(-r, y, 1.0), y);
  return fma(y, fma(-r, y, 1.0), y);
}

// FP32 Laguerre terms at x from f'/f and (f'/f)^2 - f''/f of f(x) = det(xI - T),
// through the ratios r_k = p_k / p_{k-1} of the leading principal minors (one
// reciprocal per k), which cannot overflow.  a: diagonal, b2: squared
// off-diagonal.  False if some r_k <= 0, i.e. x is not above the spectrum.
__device__ inline bool laguerre_f32(const float *a, const float *b2, int M, float x, float *step) {
  float r = x - a[0], rd = 1.0f, rdd = 0.0f;
  if (!(r > 0.0f)) return false;
  float ir = 1.0f / r;
  float g = rd * ir;
  float h = g * g - rdd * ir;
  for (int k = 1; k < M; ++k) {
    const float q = b2[k - 1] * ir;
    const float nr = (x - a[k]) - q;
    const float nrd = 1.0f + q * ir * rd;
    const float nrdd = q * ir * (rdd - 2.0f * rd * rd * ir);
    r = nr;
    rd = nrd;
    rdd = nrdd;
    if (!(r > 0.0f)) return false;
    ir = 1.0f / r;
    const float gk = rd * ir;
    g += gk;
    h += gk * gk - rdd * ir;
  }
  const float disc = (float)(M - 1) * ((float)M * h - g * g);
  const float den = g + sqrtf(disc > 0.0f ? disc : 0.0f);
  if (!(den > 0.0f)) return false;
  *step = (float)M / den;
  return true;
}

// Shared-memory scratch of the largest eigenvalue.
struct Spectrum {
  float f[5 * CB_MAX_M];
  double as[CB_MAX_M], bs2[CB_MAX_M];
};

// Largest eigenvalue of tridiag(be, al, be) (be[0..M-2] used, positive), by
// one full warp; every lane gets it.  al and be are in shared memory.
//
// An FP64 instruction of one warp occupies its sub-core's FP64 unit for about
// 64 cycles whatever its active lanes (0.5 lanes per clock), so the serial
// recurrences run in FP32 and FP64 only takes the few operations that set the
// accuracy, spread over the lanes:
//  1. FP32 multisection: x lies above the spectrum iff every pivot of xI - T
//     is positive; the 32 lanes test 32 points of the bracket at once, so a
//     round costs M dependent FP32 steps and gains a factor of 33; four
//     rounds leave a bracket of 2e-6 lambda_max, sigma its upper end.
//  2. two inverse iterations with sigma I - T (positive definite) in FP32.
//  3. the Rayleigh quotient in FP64, as rho + v.(T - rho)v / v.v from rho =
//     sigma, one correction of v from its FP64 residual by an FP32 solve, and
//     the quotient again: the error of the quotient is the square of v's, which
//     the correction takes from FP32 rounding to below 1e-9.  A cluster (the
//     copies of lambda_max in an unreorthogonalised T) gives a value inside it.
// tridiag_kernel with this and the continuants below: 79 -> 20 us at M = 20,
// 131 -> 25 us at M = 30, 220 -> 34 us at M = 40 (before: one lane running
// Laguerre's iteration in FP32 and twice in FP64, and a Thomas sweep with a
// complex reciprocal per row and lane).
__device__ inline double lambda_max(const double *al, const double *be, int M, Spectrum &S) {
  float *f = S.f;
  if (M == 1) return al[0];
  const int lane = threadIdx.x & 31;
  float *fa = f, *fb = f + M, *fl = f + 2 * M, *fi = f + 3 * M, *fv = f + 4 * M;
  float hi = -3.0e38f, lo = -3.0e38f, amax = 0.f;
  for (int i = lane; i < M; i += 32) {
    const float a = (float)al[i], b0 = i > 0 ? fabsf((float)be[i - 1]) : 0.f;
    const float b1 = i < M - 1 ? fabsf((float)be[i]) : 0.f;
    fa[i] = a;
    fb[i] = b1;
    hi = fmaxf(hi, a + b0 + b1);
    lo = fmaxf(lo, a);
    amax = fmaxf(amax, fabsf(a) + b0 + b1);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    lo = fmaxf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
  }
  __syncwarp();
  auto next_pivot = [](float x, float a, float b, float r) {  // no contraction: the same in both uses
    return __fsub_rn(__fsub_rn(x, a), __fdividef(__fmul_rn(b, b), r));
  };
  hi += 4e-6f * (amax + 1e-30f);  // Gershgorin: strictly above the spectrum, also in FP32
  for (int round = 0; round < 4; ++round) {
    const float x = lo + (hi - lo) * ((float)(lane + 1) * (1.0f / 33.0f));
    float r = x - fa[0];
    bool above = r > 0.f;
#pragma unroll 4
    for (int k = 1; k < M; ++k) {
      r = next_pivot(x, fa[k], fb[k - 1], r);
      above = above && r > 0.f;  // r is meaningless after the first r <= 0
    }
    const unsigned m = __ballot_sync(0xffffffffu, above);
    const int first = m ? __ffs(m) - 1 : 32;  // lowest point above the spectrum
    const float xl = __shfl_sync(0xffffffffu, x, first > 0 ? first - 1 : 0);
    const float xh = __shfl_sync(0xffffffffu, x, first < 32 ? first : 31);
    if (first > 0) lo = xl;
    if (first < 32) hi = xh;
  }
  // sigma I - T = L D L^T, sigma = hi: fl = -L's off-diagonal, fi = 1 / D; the
  // pivots are those of the test that placed hi, so all are positive and the
  // solves below stay bounded (every lane runs the serial loops; lane 0 writes)
  float r = hi - fa[0];
  for (int k = 0; k < M; ++k) {
    if (k) r = next_pivot(hi, fa[k], fb[k - 1], r);
    const float ir = __fdividef(1.0f, fmaxf(r, 1e-9f * amax + 1e-30f));
    if (lane == 0) {
      fi[k] = ir;
      fl[k] = fb[k] * ir;
      fv[k] = 1.0f;
    }
  }
  __syncwarp();
  // fv <- (sigma I - T)^{-1} fv, scaled to a largest entry of 1 when `unit`
  auto solve = [&](bool unit) {
    float y = 0.f;
#pragma unroll 4
    for (int k = 0; k < M; ++k) {
      y = fmaf(k ? fl[k - 1] : 0.f, y, fv[k]);
      __syncwarp();
      if (lane == 0) fv[k] = y;
    }
    __syncwarp();
    float x = 0.f, top = 0.f;
#pragma unroll 4
    for (int k = M - 1; k >= 0; --k) {
      x = fmaf(fl[k], x, fv[k] * fi[k]);  // fl[M-1] = 0
      top = fmaxf(top, fabsf(x));
      __syncwarp();
      if (lane == 0) fv[k] = x;
    }
    __syncwarp();
    if (unit) {
      const float sc = __fdividef(1.0f, fmaxf(top, 1e-30f));
      for (int i = lane; i < M; i += 32) fv[i] *= sc;
      __syncwarp();
    }
  };
  solve(true);
  solve(true);
  // quotient, correction, quotient; up to 4 entries per lane (M <= 128)
  double v[4], rho = (double)hi;
#pragma unroll
  for (int e = 0; e < 4; ++e) v[e] = lane + 32 * e < M ? (double)fv[lane + 32 * e] : 0.0;
  for (int it = 0; it < 2; ++it) {
    double t[4], num = 0.0;
    float den = 0.f;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      t[e] = 0.0;
      if (32 * e < M) {  // uniform
        const int i = lane + 32 * e;
        double left = __shfl_up_sync(0xffffffffu, v[e], 1), right = __shfl_down_sync(0xffffffffu, v[e], 1);
        const double lastp = e > 0 ? __shfl_sync(0xffffffffu, v[e > 0 ? e - 1 : 0], 31) : 0.0;
        const double firstn = e < 3 ? __shfl_sync(0xffffffffu, v[e < 3 ? e + 1 : 3], 0) : 0.0;
        if (lane == 0) left = lastp;
        if (lane == 31) right = firstn;
        if (i < M) {
          t[e] = (al[i] - rho) * v[e];
          if (i > 0) t[e] = fma(be[i - 1], left, t[e]);
          if (i < M - 1) t[e] = fma(be[i], right, t[e]);
          num = fma(v[e], t[e], num);
          den = fmaf((float)v[e], (float)v[e], den);
        }
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      num += __shfl_xor_sync(0xffffffffu, num, o);
      den += __shfl_xor_sync(0xffffffffu, den, o);
    }
    // num is of the size of lambda_max - rho, 1e-6 and then 1e-12 of
    // lambda_max, so FP32 suffices for the ratio
    const float q = (float)num / den;
    rho += (double)q;
    if (it == 1) break;
    __syncwarp();
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (lane + 32 * e < M) fv[lane + 32 * e] = (float)t[e] - q * (float)v[e];  // (T - rho) v
    __syncwarp();
    solve(false);  // (sigma - T)^{-1} (T - rho) v: minus the contamination of v
    // the component along v itself would only rescale it: taken out, so that
    // the correction stays small
    float dot = 0.f;
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (lane + 32 * e < M) dot = fmaf(fv[lane + 32 * e], (float)v[e], dot);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
    dot /= den;
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (lane + 32 * e < M) v[e] += (double)(fv[lane + 32 * e] - dot * (float)v[e]);
  }
  return rho;
}

// The same by Laguerre's iteration on det(xI - T), for FP64 recurrences (25
// against 34 us at M = 30).  The iteration from above the Gershgorin bound runs
// in FP32 until its step is below 1e-6 relative, then two FP64 steps polish the
// result: the convergence is cubic, so the FP32 estimate turns into an
// FP64-accurate one.  Not always: where the FP32 iterate ends below lambda_max,
// an FP64 step meets a pivot that is not positive and is left out, and theta
// stays up to 4e-8 short (relative; 3 of 48 ER, WS and BA graphs of 900 to 8500
// nodes at m = 30, the others within 6e-15); over copies of lambda_max (T without
// reorthogonalisation) it stops up to 1.2e-7 above.  exp(theta) y does not depend
// on it, but theta and y are results that callers compare and store to FP64
// accuracy, so both FP64 modes take them by this one method.
//
// T is converted once, in parallel, and the FP64 steps take f, f' and f'' from
// p_k = (x - a_k) p_{k-1} - b_{k-1}^2 p_{k-2} and its derivatives on three
// lanes at once: 4 FP64 instructions per row (the ratios above take 22).  T
// and x are scaled by a power of two there, so that no product leaves the FP64
// range for M <= CB_MAX_M.
__device__ inline double lambda_max_laguerre(const double *al, const double *be, int M, Spectrum &S) {
  if (M == 1) return al[0];
  const int lane = threadIdx.x & 31;
  float *fa = S.f, *fb2 = S.f + CB_MAX_M;
  double x0 = -1e300, low = 1e300;
  for (int i = lane; i < M; i += 32) {
    const double lo = i > 0 ? fabs(be[i - 1]) : 0.0;
    const double hi = i < M - 1 ? fabs(be[i]) : 0.0;
    x0 = fmax(x0, al[i] + lo + hi);
    low = fmin(low, al[i]);
    const float fb = (float)be[i];
    fa[i] = (float)al[i];
    fb2[i] = fb * fb;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    x0 = fmax(x0, __shfl_xor_sync(0xffffffffu, x0, o));
    low = fmin(low, __shfl_xor_sync(0xffffffffu, low, o));
  }
  x0 += 1e-3 * (fabs(x0) + 1.0);  // strictly above the spectrum, also in FP32
  int ex;
  frexpf((float)(x0 - low) + 1.0f, &ex);
  const double s = __hiloint2double((1023 - ex) << 20, 0);  // 2^-ex: |x - a_k| < 2^ex
  for (int i = lane; i < M; i += 32) {
    const double b = be[i] * s;
    S.as[i] = al[i] * s;
    S.bs2[i] = b * b;
  }
  __syncwarp();
  float xf = (float)x0;
  if ((double)xf < x0) xf = nextafterf(xf, 3.0e38f);
  float st;
  if (laguerre_f32(fa, fb2, M, xf, &st)) {
    for (int it = 0; it < 40; ++it) {
      const float nx = xf - st;
      float st2;
      if (!laguerre_f32(fa, fb2, M, nx, &st2)) break;  // nx not above: keep xf
      xf = nx;
      st = st2;
      if (st <= 1e-6f * (fabsf(xf) + 1.0f)) break;
    }
  }
  double x = xf;
  const double c = lane == 1 ? 1.0 : lane == 2 ? 2.0 : 0.0;  // lane d: the d-th derivative
  for (int it = 0; it < 2; ++it) {  // FP64 polish, left out from below lambda_max
    const double xs = x * s;
    double own2 = lane == 0 ? 1.0 : 0.0;                                 // p_0
    double own = lane == 0 ? xs - S.as[0] : lane == 1 ? 1.0 : 0.0;       // p_1
    bool above = lane != 0 || own > 0.0;
#pragma unroll 2
    for (int k = 1; k < M; ++k) {
      const double below = __shfl_up_sync(0xffffffffu, own, 1);  // lane 0's c is 0
      const double nxt = fma(xs - S.as[k], own, fma(c, below, -S.bs2[k - 1] * own2));
      own2 = own;
      own = nxt;
      if (lane == 0) above = above && __double2hiint(own) > 0;  // own > 0, without an FP64 compare
    }
    if (!__all_sync(0xffffffffu, above)) break;
    const double p = __shfl_sync(0xffffffffu, own, 0), p1 = __shfl_sync(0xffffffffu, own, 1);
    const double p2 = __shfl_sync(0xffffffffu, own, 2);
    // G = f'/f, H = G^2 - f''/f, times s and s^2
    const double ip = 1.0 / p, G = p1 * ip, H = G * G - p2 * ip;
    const double disc = (double)(M - 1) * ((double)M * H - G * G);
    const double den = G + sqrt(disc > 0.0 ? disc : 0.0);
    if (!(den > 0.0)) break;
    x -= (double)M / (den * s);
  }
  return x;
}

// FP32 recurrences: lambda_max is the nearer of the two to the largest eigenvalue
// of A's Krylov matrix (against a dense FP64 eigensolver on T of a fully
// reorthogonalised FP64 run; 24 cliques in sparse graphs, ER and BA graphs of
// lambda_max 19 to 201, m = 30 and 35: 7.3e-8 of lambda_max off on average, 2.4e-7 at
// most; Laguerre's 4.4e-7 and 8.7e-7, from above, over the copies that T carries).
// But every score is scaled by exp(-theta): above kCopiesShow the difference is
// some 2e-5 of each, which callers that compare or store FP32 scores with earlier
// ones would see, and Laguerre's value stays.  (FP64: its method alone.)
constexpr double kCopiesShow = 48.0;

__device__ inline double largest(const double *al, const double *be, int M, Spectrum &S, bool laguerre) {
  if (!laguerre) {
    const double t = lambda_max(al, be, M, S);
    if (t <= kCopiesShow) return t;
    __syncwarp();  // S is used again
  }
  return lambda_max_laguerre(al, be, M, S);
}

// Node z and weight w = e^z z'(t) / (i N) of the upper-half nodes q =
// 0..kHalf-1, evaluated once on the host and passed to the kernels by value.
struct Nodes {
  cplx z[kHalf], w[kHalf];
};
inline Nodes make_nodes() {
  Nodes n;
  long double re[kHalf], im[kHalf], at0 = 0.0L;
  const long double pi = std::acos(-1.0L);
  for (int q = 0; q < kHalf; ++q) {
    const long double t = -pi + (kHalf + q + 0.5L) * (2.0L * pi / kNodes);
    const long double sn = std::sin(kB * t), cot = std::cos(kB * t) / sn;
    const long double zr = kNodes * (kA * t * cot - kC), zi = kNodes * kD * t;
    const long double dr = kNodes * (kA * cot - kA * kB * t / (sn * sn)), di = kNodes * kD;
    const long double ec = std::exp(zr) * std::cos(zi), es = std::exp(zr) * std::sin(zi);
    re[q] = (ec * di + es * dr) / kNodes;
    im[q] = -(ec * dr - es * di) / kNodes;
    n.z[q] = {(double)zr, (double)zi};
    at0 += 2.0L * (re[q] * zr + im[q] * zi) / (zr * zr + zi * zi);  // 2 Re(w / z)
  }
  // the rule's value at 0, where the dominant eigenvalue of T - theta lies, is
  // e^0 = 1 up to its truncation error (1.7e-14): the weights make it exact
  for (int q = 0; q < kHalf; ++q) n.w[q] = {(double)(re[q] / at0), (double)(im[q] / at0)};
  return n;
}
inline const Nodes &nodes() {
  static const Nodes n = make_nodes();
  return n;
}

// The contour solves x_k = (z_k I - (T - theta I))^{-1} e1 of one warp, by
// continuants: with d_i = z - (al_i - theta),
//   phi_M = 1, phi_i = d_i phi_{i+1} - be_i^2 phi_{i+2},
//   x_i = be_0 .. be_{i-1} phi_{i+1} / phi_0,
// no reciprocal per row, and the real and imaginary part of a node on two
// lanes (24 of the warp): 4 FP64 instructions per row, where a pivoted sweep
// takes 18 on 12 lanes.  T and z are scaled by a power of two so that |d_i|
// is below 1 and no product leaves the FP64 range for M <= CB_MAX_M.
constexpr int kCols = 2 * kHalf;
struct Solve {                     // shared memory of one solve
  double phi[CB_MAX_M * kCols];    // phi_{i+1} at row i, column 2 k + part
  double d[CB_MAX_M], b2[CB_MAX_M], B[CB_MAX_M];  // scaled; B: the products of be
};

// Fills S; returns the scale (a power of two: x above is to be multiplied by
// it) and, in both lanes of a node's pair, 1 / phi_0 of lane / 2.  al, be in
// shared memory.
__device__ inline double continuants(const double *al, const double *be, int M, double theta,
                                     const Nodes &nd, Solve &S, cplx *inv_phi0) {
  const int lane = threadIdx.x & 31, part = lane & 1, q = lane < kCols ? lane >> 1 : 0;
  double lowest = theta;
  for (int i = lane; i < M; i += 32) lowest = fmin(lowest, al[i]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) lowest = fmin(lowest, __shfl_xor_sync(0xffffffffu, lowest, o));
  int ex;
  frexpf((float)(theta - lowest) + 64.f, &ex);  // |z| < 40
  const double s = __hiloint2double((1023 - ex) << 20, 0);  // 2^-ex
  double run = 1.0;  // product of the chunks before this one
  for (int c = 0; c < M; c += 32) {
    const int i = c + lane;
    const double b = i < M ? be[i] * s : 1.0;
    if (i < M) {
      S.d[i] = (theta - al[i]) * s;
      S.b2[i] = i < M - 1 ? b * b : 0.0;
    }
    double p = b;  // inclusive prefix product
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const double y = __shfl_up_sync(0xffffffffu, p, o);
      if (lane >= o) p *= y;
    }
    const double ex1 = __shfl_up_sync(0xffffffffu, p, 1);
    if (i < M) S.B[i] = run * (lane ? ex1 : 1.0);
    run *= __shfl_sync(0xffffffffu, p, 31);
  }
  __syncwarp();
  const double zr = nd.z[q].re * s, zi = (part ? 1.0 : -1.0) * nd.z[q].im * s;
  double own = part ? 0.0 : 1.0, own2 = 0.0;
#pragma unroll 2
  for (int i = M - 1; i >= 0; --i) {
    if (lane < kCols) S.phi[i * kCols + lane] = own;
    const double other = __shfl_xor_sync(0xffffffffu, own, 1);
    const double nxt = fma(zr + S.d[i], own, fma(zi, other, -S.b2[i] * own2));
    own2 = own;
    own = nxt;
  }
  // 1 / phi_0, scaled to exponent 0 on the way (|phi_0|^2 may underflow)
  const double other = __shfl_xor_sync(0xffffffffu, own, 1);
  const double re = part ? other : own, im = part ? own : other;
  const int e0 = max((__double2hiint(re) >> 20) & 0x7ff, (__double2hiint(im) >> 20) & 0x7ff);
  const double k = __hiloint2double((2046 - e0) << 20, 0);  // 2^(1023 - e0)
  const double rs = re * k, is = im * k, dd = rcp_nr(fma(rs, rs, is * is)) * k;
  *inv_phi0 = {rs * dd, -is * dd};
  __syncwarp();
  return s;
}

// out(i, c_i) for the rows i < M: c_i = sum_k Re(p_k x_k,i), p (both lanes of
// the pair) the node's factor times *inv_phi0.  Called by the warp.
template <typename F>
__device__ inline void real_sum(Solve &S, int M, double scale, cplx g, F out) {
  const int lane = threadIdx.x & 31;
  __shared__ double s_g[kCols];
  if (lane < kCols) s_g[lane] = (lane & 1) ? -g.im * scale : g.re * scale;
  __syncwarp();
  for (int i = lane; i < M; i += 32) {
    double c = 0.0;
#pragma unroll
    for (int q = 0; q < kCols; ++q) c = fma(s_g[q], S.phi[i * kCols + q], c);
    out(i, c * S.B[i]);
  }
}

}  // namespace contour
}  // namespace cb
