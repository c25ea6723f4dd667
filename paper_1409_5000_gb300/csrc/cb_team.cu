// The whole Lanczos recurrence of on-chip problems in one launch.
//
// Where the CSR arrays and vectors of a call stay on the chip (L2 and shared
// memory), a step's arithmetic takes a few microseconds and three launches a
// step (SpMV, finalize, beta) cost more than it: 19 + 4.5 + 5.7 us a step on
// one graph of 1e5 nodes and 1e6 entries.  Here a team of CTAs, all resident,
// runs every step of one realisation; a realisation small enough has a team
// of one.  Per CTA:
//  * a run of consecutive rows, cut so that entries + (mean degree) x rows is
//    equal over the team (found at the start by a 32-way search of row_ptr);
//  * in shared memory: the rows' offsets, W_j, W_{j-1} and the new vector on
//    its rows, and the columns when they fit; W_j of the whole realisation too
//    when copying it each step is cheaper than gathering from L2 (teams of one
//    always);
//  * each row summed by as many lanes as there are threads per row, eight
//    gathers of a lane in flight; rows of more than kMedRun entries per lane by
//    a warp, of more than kLongRun by the CTA;
//  * alpha and beta: per-CTA partials in FP64, added by every CTA in the same
//    order after a barrier of the team: each CTA stores its partial and adds
//    to the team's counter (release), one thread per CTA polls the counter
//    (acquire).  Measured at 152 CTAs: 2200 cycles a barrier; 3200 to 4500 when
//    every CTA writes into an inbox of every other, and 8000 to 18000 when all
//    poll one array of partials.  The beta barrier also publishes the new vector.
// With CB_REORTH the two Gram-Schmidt passes run in the same launch, their
// dot products exchanged with the norms.
//
// Measured, us per step before (one CTA with its rows' chains of global loads up
// to 8192 nodes, three launches a step above) and now: 10 x 500 nodes FP32 7.0 ->
// 3.8; 40 x 4000 36 -> 6.8; 8 x 30000 32 -> 12; FP64 with reorthogonalisation,
// one graph of 1e5 nodes: 118 -> 43.  An FP64 instruction takes its sub-core 65
// cycles per warp, so scalars and splits are formed by one warp.
//
// The recurrence, its scalars and breakdown test are those of spmv_kernel +
// finalize_kernel + finalize_beta_kernel (cb_lanczos.cu); scale, beta scale
// and alpha scale enter the FP32 arithmetic as a two-float sum instead of one
// rounded factor, which would shift every entry of a vector the same way.
#include <algorithm>
#include <type_traits>

#include "cb_contour.cuh"
#include "cb_grid.cuh"
#include "cb_internal.cuh"
#include "cb_reduce.cuh"
#include "cb_step.cuh"
#include "cb_team.cuh"

namespace cb {

namespace {

constexpr int kTeamThreads = 1024;
constexpr uint32_t kMedRun = 32;     // entries per lane beyond which a warp sums the row
constexpr uint32_t kLongRun = 2048;  // entries beyond which the CTA does
constexpr uint32_t kLists = 64;      // longest lists of such rows (else: as the short ones)

__device__ __forceinline__ double ld_relaxed(const double *p) {
  double v;
  asm volatile("ld.relaxed.gpu.global.f64 %0, [%1];" : "=d"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ bool finite(double v) {
  return (__double2hiint(v) & 0x7ff00000) != 0x7ff00000;
}

// A double as the sum of two floats, or itself (T = double).  Formed once per
// step by one warp: a conversion by every warp costs its sub-core 64 cycles
// of the FP64 unit each.
template <typename T>
struct Split;
template <>
struct Split<float> {
  float hi, lo;
  __device__ void set(double v) {
    hi = (float)v;
    lo = (float)(v - (double)hi);
  }
  __device__ float times(float x) const { return fmaf(hi, x, lo * x); }
  // c - this * x
  __device__ float from(float c, float x) const { return fmaf(-hi, x, fmaf(-lo, x, c)); }
};
template <>
struct Split<double> {
  double hi;
  __device__ void set(double v) { hi = v; }
  __device__ double times(double x) const { return hi * x; }
  __device__ double from(double c, double x) const { return fma(-hi, x, c); }
};

// Smallest i in [0, n] with rp[i] + c i >= target, by one warp (32 probes a round).
__device__ uint32_t row_split(const uint32_t *rp, uint32_t n, uint32_t c, uint64_t target) {
  const uint32_t lane = threadIdx.x & 31;
  uint32_t lo = 0, hi = n;  // the answer is in [lo, hi]
  while (lo < hi) {
    const uint32_t step = (hi - lo + 31) / 32;
    const uint32_t at = min(hi, lo + step * lane);  // lane 0 probes lo
    const bool ge = (uint64_t)rp[at] + (uint64_t)c * at >= target;
    const uint32_t m = __ballot_sync(0xffffffffu, ge);
    if (m == 0) {  // beyond the last probe
      lo = min(hi, lo + step * 31) + 1;
      if (lo > hi) lo = hi;
      continue;
    }
    const uint32_t f = __ffs(m) - 1;
    hi = min(hi, lo + step * f);
    lo = f == 0 ? hi : min(hi, lo + step * (f - 1) + 1);
  }
  return lo;
}

// hi + lo: a sum over a warp to about twice the precision of FP32 (two-sum: lo
// holds what the additions into hi round away), taken for alpha, whose error every
// entry of the result shares: with plain FP32 warp sums the scores of 10 graphs of
// 500 nodes were 1.9e-7 off on average (16 seeds; 8.7e-8 by the per-step
// kernels, whose rows have more lanes), so 7.9e-8.  For beta it made no difference.
template <typename T>
struct Pair {
  T hi, lo;
  __device__ double value() const { return to_double(hi) + to_double(lo); }
};
__device__ __forceinline__ Pair<float> exact_warp_sum(float v) {
  Pair<float> p{v, 0.f};
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float h = __shfl_xor_sync(0xffffffffu, p.hi, o), l = __shfl_xor_sync(0xffffffffu, p.lo, o);
    const float s = __fadd_rn(p.hi, h), b = __fsub_rn(s, p.hi);
    const float e = __fadd_rn(__fsub_rn(p.hi, __fsub_rn(s, b)), __fsub_rn(h, b));
    p = {s, __fadd_rn(__fadd_rn(p.lo, l), e)};
  }
  return p;
}

template <typename T>
struct Shared {
  T red[kTeamThreads / 32];
  Pair<float> ared[kTeamThreads / 32];
  Split<T> scj, bpj, coef;  // scale_j, beta_{j-1} scale_{j-1}, alpha_j scale_j
  double scale, alpha, beta;  // of this step; beta: of the one before
  float alpha32, beta32;      // the same in FP32
  double h[CB_MAX_M + 1], sc[CB_MAX_M + 1];  // Gram-Schmidt coefficients; scale_i so far
  uint32_t split[2];
  uint32_t nmed, nlong;
  uint16_t med[kLists], lng[kLists];  // local rows summed by a warp, by the CTA
  T lsum[kTeamThreads / 32];
  int stop;
};

// The breakdown test where FP32 does not decide it (a call: four FP64 operations of
// 65 cycles that must not be issued on the way of every step).
__device__ __noinline__ bool breaks_down(double beta, double tau, double alpha, double bprev) {
  return beta <= tau * (fabs(alpha) + bprev) || beta == 0.0;
}

template <typename T>
__device__ __forceinline__ double cta_partial(T v, Shared<T> &sh) {  // valid in warp 0
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  v = warp_sum<T>(v);
  if (lane == 0) sh.red[warp] = v;
  __syncthreads();
  return warp == 0 ? warp_sum_d(to_double(sh.red[lane])) : 0.0;
}

template <typename T>
__device__ __forceinline__ double cta_alpha(T v, Shared<T> &sh) {  // valid in warp 0
  if constexpr (sizeof(T) == 8) {
    return cta_partial<T>(v, sh);
  } else {
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const Pair<float> p = exact_warp_sum(v);
    if (lane == 0) sh.ared[warp] = p;
    __syncthreads();
    return warp == 0 ? warp_sum_d(sh.ared[lane].value()) : 0.0;
  }
}

// Warp 0: the team's sum of `mine` (equal in all lanes); the same bits in
// every CTA.  part: the team's partials, two sets that alternate (a CTA writes
// a set again only after a barrier that every other reached having read it);
// ctr: 0 before the launch; ex: the exchange's number, from 1.  What the CTA's
// threads stored before the barrier in front of this call is visible to the
// team after it.  *ok turns false when the wait gave up.
__device__ double team_sum(double *part, uint32_t *ctr, uint32_t rank, uint32_t size, uint32_t ex, double mine,
                           uint64_t wait_ns, bool *ok) {
  if (size == 1) return mine;
  const uint32_t lane = threadIdx.x & 31;
  part += (ex & 1u) * kMaxTeamCtas;
  if (lane == 0) {
    part[rank] = mine;
    red_release(ctr, 1u);
    if (!grid_wait(ctr, ex * size, wait_ns)) *ok = false;
  }
  __syncwarp();  // orders the other lanes' loads after lane 0's acquire
  *ok = __all_sync(0xffffffffu, *ok);
  constexpr uint32_t kPer = kMaxTeamCtas / 32;
  double v[kPer];
#pragma unroll
  for (uint32_t u = 0; u < kPer; ++u) v[u] = 32 * u + lane < size ? ld_relaxed(part + 32 * u + lane) : 0.0;
  double acc = v[0];
#pragma unroll
  for (uint32_t u = 1; u < kPer; ++u)
    if (32 * u < size) acc += v[u];
  return warp_sum_d(acc);
}

}  // namespace

template <typename T>
__global__ void __launch_bounds__(kTeamThreads, 1) team_lanczos_kernel(const __grid_constant__ LArgs a,
                                                                       const __grid_constant__ TeamArgs t,
                                                                       uint32_t r0, uint32_t m) {
  extern __shared__ float4 s_dyn4[];
  __shared__ Shared<T> sh;
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint32_t q = blockIdx.x, rank = 0, size = 1;
  if (t.nteams) {
    q = 0;
    while (q + 1 < t.nteams && t.first[q + 1] <= blockIdx.x) ++q;
    rank = blockIdx.x - t.first[q];
    size = t.first[q + 1] - t.first[q];
  }
  const uint32_t r = r0 + q;
  const InstDesc &I = a.inst[r];
  const uint32_t n = I.n, nnz = I.nnz, ms = a.sc.ms;
  const uint32_t mr = min(a.sc.meff[r], m);  // 0: no start vector (no CTA has changed it yet)
  if (mr == 0 || (t.stall && size > 1 && rank + 1 == size)) return;
  const uint32_t *rpg = a.row_ptr + I.rp_base;
  const uint32_t *cg = a.col + I.edge_base;
  const uint32_t rc = max(1u, (uint32_t)(((uint64_t)nnz + (uint64_t)n * t.rowdiv - 1) / ((uint64_t)n * t.rowdiv)));
  if (warp < 2 && size > 1) {
    const uint64_t F = (uint64_t)nnz + (uint64_t)rc * n;
    const uint32_t at = rank + warp;
    const uint32_t s = at == 0 ? 0u : at == size ? n : row_split(rpg, n, rc, F * at / size);
    if (lane == 0) sh.split[warp] = s;
  }
  if (tid == 0) {
    sh.scale = sh.sc[0] = a.sc.scale[r * ms];
    sh.beta = 0.0;
    sh.beta32 = 0.f;
    sh.scj.set(sh.scale);
    sh.bpj.set(0.0);
    sh.stop = 0;
    sh.nmed = sh.nlong = 0;
  }
  __syncthreads();
  const uint32_t row0 = size > 1 ? sh.split[0] : 0u, row1 = size > 1 ? sh.split[1] : n;
  const uint32_t rows = row1 - row0;
  const uint32_t e0 = rpg[row0], ne = rpg[row1] - e0;

  // shared memory: x (whole or own rows), W_{j-1}, u (own rows), row offsets,
  // then the columns if they fit
  const bool xs = size == 1 || (q < 64 && (t.whole_x >> q & 1ull));
  const uint32_t rows4 = (rows + 3) & ~3u, n4 = (n + 3) & ~3u;
  T *xw = reinterpret_cast<T *>(s_dyn4);
  T *xp = xw + (xs ? n4 : rows4);
  T *us = xp + rows4;
  uint32_t *rp = reinterpret_cast<uint32_t *>(us + rows4);
  uint8_t *rest = reinterpret_cast<uint8_t *>(rp + ((rows + 1 + 3) & ~3u));
  const size_t used = (size_t)(rest - reinterpret_cast<uint8_t *>(s_dyn4));
  if (used > t.smem) return;  // cannot happen: the plan bounds the rows of a CTA
  const size_t room = t.smem - used;
  // 0: columns from global memory, 1: u16 in shared memory, 2: u32
  const int cmode = n <= 65536 && (size_t)ne * 2 <= room ? 1 : !xs && (size_t)ne * 4 <= room ? 2 : 0;
  uint16_t *c16 = reinterpret_cast<uint16_t *>(rest);
  uint32_t *c32 = reinterpret_cast<uint32_t *>(rest);
  for (uint32_t i = tid; i <= rows; i += kTeamThreads) rp[i] = rpg[row0 + i] - e0;
  if (cmode == 1)
    for (uint32_t e = tid; e < ne; e += kTeamThreads) c16[e] = (uint16_t)ld_stream(cg + e0 + e);
  if (cmode == 2)
    for (uint32_t e = tid; e < ne; e += kTeamThreads) c32[e] = ld_stream(cg + e0 + e);
  T *Vb = reinterpret_cast<T *>(a.V) + I.node_base;
  if (xs)
    for (uint32_t i = tid; i < n; i += kTeamThreads) xw[i] = Vb[i];
  else
    for (uint32_t i = tid; i < rows; i += kTeamThreads) xw[i] = Vb[row0 + i];
  __syncthreads();

  // lanes per row, and the rows too long for them
  uint32_t G = 1;
  while (G < 32 && 2 * G * rows <= kTeamThreads) G *= 2;
  bool any = false;
  for (uint32_t i = tid; i < rows; i += kTeamThreads) any |= rp[i + 1] - rp[i] > kMedRun * G;
  if (__syncthreads_or(any) && warp == 0) {  // lists in row order: every sum has one order
    uint32_t nm = 0, nl = 0;
    for (uint32_t b = 0; b < rows; b += 32) {
      const uint32_t i = b + lane, len = i < rows ? rp[i + 1] - rp[i] : 0u;
      const bool l = len > kLongRun, md = !l && len > kMedRun * G;
      const uint32_t bl = __ballot_sync(0xffffffffu, l), bm = __ballot_sync(0xffffffffu, md);
      const uint32_t below = (1u << lane) - 1u, al = nl + __popc(bl & below), am = nm + __popc(bm & below);
      if (l && al < kLists) sh.lng[al] = (uint16_t)i;
      if (md && am < kLists) sh.med[am] = (uint16_t)i;
      nl += __popc(bl);
      nm += __popc(bm);
    }
    // lists that overflow (or rows beyond 16 bits) are not used: all rows go the short way
    if (lane == 0 && nm <= kLists && nl <= kLists && rows <= 65536) {
      sh.nmed = nm;
      sh.nlong = nl;
    }
  }
  __syncthreads();
  const uint32_t nmed = sh.nmed, nlong = sh.nlong;
  const uint32_t long_from = nlong ? kLongRun : 0xffffffffu;
  const uint32_t med_from = nmed ? kMedRun * G : long_from;
  const uint32_t first = t.nteams ? t.first[q] : blockIdx.x;
  double *parts = t.parts + first;  // two sets, kMaxTeamCtas apart
  uint32_t *ctr = t.ctr + q * kCtrStride;
  uint32_t ex = 0;
  bool ok = true;
  // sum of x over the entries lo, lo + step, ... < hi; CM: the column mode, U
  // gathers of a lane in flight
  auto run_sum = [&](auto CM, auto U, const T *from, uint32_t lo, uint32_t hi, uint32_t step) -> T {
    T sum = T(0);
    for (uint32_t e = lo; e < hi; e += U * step) {
      T v[U];
#pragma unroll
      for (uint32_t u = 0; u < U; ++u) {
        v[u] = T(0);
        if (e + u * step < hi) {
          const uint32_t at = e + u * step;
          const uint32_t c = CM == 1 ? (uint32_t)c16[at] : CM == 2 ? c32[at] : ld_stream(cg + e0 + at);
          if (CB_DCHECK(c < n, kDbgCsrCol, c)) v[u] = from[c];
        }
      }
#pragma unroll
      for (uint32_t u = 0; u < U; ++u) sum += v[u];
    }
    return sum;
  };
  for (uint32_t j = 0; j < mr; ++j) {
    const T *x = Vb + (uint64_t)j * a.vs;  // W_j, whole (global)
    T *out = Vb + (uint64_t)(j + 1) * a.vs + row0;
    T *xo = xs ? xw + row0 : xw;  // W_j on this CTA's rows
    const Split<T> scj = sh.scj, bpj = sh.bpj;
    T acc = T(0);
    // u = scale_j (A W_j) - beta_{j-1} scale_{j-1} W_{j-1} of one row, and its alpha term
    auto finish_row = [&](uint32_t i, T sum) {
      T u = scj.times(sum);
      if (j > 0) u = bpj.from(u, xp[i]);
      us[i] = u;
      acc += xo[i] * u;
    };
    auto spmv = [&](auto CM, auto U, const T *from) {
      for (uint32_t k = 0; k < nlong; ++k) {
        const uint32_t i = sh.lng[k];
        const T p = warp_sum<T>(run_sum(CM, U, from, rp[i] + tid, rp[i + 1], kTeamThreads));
        if (lane == 0) sh.lsum[warp] = p;
        __syncthreads();
        if (warp == 0) {
          const T sum = warp_sum<T>(sh.lsum[lane]);
          if (lane == 0) finish_row(i, sum);
        }
        __syncthreads();
      }
      for (uint32_t k = warp; k < nmed; k += kTeamThreads / 32) {
        const uint32_t i = sh.med[k];
        const T sum = warp_sum<T>(run_sum(CM, U, from, rp[i] + lane, rp[i + 1], 32));
        if (lane == 0) finish_row(i, sum);
      }
      const uint32_t lg = tid & (G - 1);
      for (uint32_t b = 0; b < rows; b += kTeamThreads / G) {  // uniform: the shuffles see all lanes
        const uint32_t i = b + tid / G;
        uint32_t lo = 0, hi = 0;
        if (i < rows) {
          lo = rp[i];
          hi = rp[i + 1];
        }
        const bool mine = i < rows && hi - lo <= med_from;
        T sum = mine ? run_sum(CM, U, from, lo + lg, hi, G) : T(0);
        for (uint32_t o = G / 2; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if (mine && lg == 0) finish_row(i, sum);
      }
    };
    using std::integral_constant;
    constexpr integral_constant<uint32_t, 4> kNear;  // shared memory: short latency
    constexpr integral_constant<uint32_t, 8> kFar;   // L2
    if (xs && cmode == 1)
      spmv(integral_constant<int, 1>(), kNear, xw);
    else if (xs)
      spmv(integral_constant<int, 0>(), kFar, xw);
    else if (cmode == 1)
      spmv(integral_constant<int, 1>(), kFar, x);
    else if (cmode == 2)
      spmv(integral_constant<int, 2>(), kFar, x);
    else
      spmv(integral_constant<int, 0>(), kFar, x);
    double part = cta_alpha<T>(acc, sh);
    if (warp == 0) {
      const double total = team_sum(parts, ctr, rank, size, ex + 1, part, t.wait_ns, &ok);
      const double scale = sh.scale, alpha = scale * total;
      if (lane == 0) {
        sh.alpha = alpha;
        sh.alpha32 = (float)alpha;
        sh.coef.set(alpha * scale);
        if (!ok || !finite(alpha)) {
          sh.stop = 1;
          if (rank == 0 || !ok) {
            if (a.sc.status[r] == CB_OK) a.sc.status[r] = ok ? CB_ERR_NONFINITE : CB_ERR_TIMEOUT;
            a.sc.meff[r] = j;
          }
        }
        if (rank == 0) a.sc.alpha[r * ms + j] = alpha;
      }
    }
    __syncthreads();
    if (sh.stop) break;
    // ---- w = u - alpha_j scale_j W_j
    const Split<T> coef = sh.coef;
    T acc2 = T(0);
    for (uint32_t i = tid; i < rows; i += kTeamThreads) {
      const T w = coef.from(us[i], xo[i]);
      us[i] = w;
      if (!t.reorth) out[i] = w;
      acc2 += w * w;
      if (xs) xp[i] = xo[i];
    }
    // beta_j, the breakdown test and scale_{j+1} from the team's ||w||^2
    auto finish = [&](double total, bool last) {
      double beta, inv;
      float beta32;
      const int te = (__double2hiint(total) >> 20) - 1023;  // exponent (sign set: negative)
      if (te > -100 && te < 100) {
        // 1 / sqrt(x) = y (1 - 2 r)^(-1/2), r = (1 - x y^2) / 2 of 2^-23: the series to
        // r^2, to 2^-68; six FP64 operations
        const float y = rsqrtf((float)total);
        beta32 = (float)total * y;
        const double yd = to_double(y), z = total * yd, r = fma(-z, to_double(0.5f * y), 0.5);
        const double c = r * fma(1.5, r, 1.0);
        inv = fma(yd, c, yd);
        beta = fma(z, c, z);
      } else {
        beta = sqrt(total);
        inv = 1.0 / beta;
        beta32 = (float)beta;
      }
      // the next step's two factors, split side by side on two lanes
      if (last && lane < 2) (lane ? sh.bpj : sh.scj).set(lane ? beta * sh.scale : inv);
      __syncwarp();
      if (lane != 0) return;
      const bool bad = !ok || !finite(beta);
      const bool broke = !(beta32 > 1.01f * (float)a.tau * (fabsf(sh.alpha32) + sh.beta32)) &&
                         breaks_down(beta, a.tau, sh.alpha, sh.beta);
      if (rank == 0 || !ok) {
        a.sc.beta[r * ms + j] = beta;
        if (bad) a.sc.status[r] = ok ? CB_ERR_NONFINITE : CB_ERR_TIMEOUT;
        if (bad || broke) a.sc.meff[r] = j + 1;
        else if (last) a.sc.scale[r * ms + j + 1] = inv;
      }
      if (bad || broke) sh.stop = 1;
      if (last) {
        sh.scale = sh.sc[j + 1] = inv;
        sh.beta = beta;
        sh.beta32 = beta32;
      }
    };
    if (t.reorth) {
      // two classical Gram-Schmidt passes against v_i = scale_i W_i, i <= j; the
      // norm of the vector before each pass is exchanged with its dot products
      for (uint32_t pass = 0; pass < 2 && !sh.stop; ++pass) {
        __syncthreads();  // us is complete
        double *xd = t.xd + (uint64_t)pass * kMaxTeamCtas * ms;
        for (uint32_t i = warp; i <= j; i += kTeamThreads / 32) {
          const T *wi = Vb + (uint64_t)i * a.vs + row0;
          T d = T(0);
          for (uint32_t k = lane; k < rows; k += 32) d += wi[k] * us[k];
          const double s = warp_sum_d((double)d) * sh.sc[i];
          if (lane == 0) {
            if (size > 1) xd[(uint64_t)blockIdx.x * ms + i] = s;
            sh.h[i] = s;
          }
        }
        part = cta_partial<T>(acc2, sh);
        if (warp == 0) finish(team_sum(parts, ctr, rank, size, ex + 2 + pass, part, t.wait_ns, &ok), false);
        __syncthreads();
        if (sh.stop) break;
        if (size > 1) {  // h_i over the team, in rank order
          for (uint32_t i = warp; i <= j; i += kTeamThreads / 32) {
            double s = 0.0;
            for (uint32_t k = lane; k < size; k += 32)
              s += ld_relaxed(xd + (uint64_t)(blockIdx.x - rank + k) * ms + i);
            s = warp_sum_d(s);
            if (lane == 0) sh.h[i] = s;
          }
        }
        __syncthreads();
        if (tid <= j) sh.h[tid] *= sh.sc[tid];
        __syncthreads();
        acc2 = T(0);
        for (uint32_t k = tid; k < rows; k += kTeamThreads) {
          T w = us[k];
          for (uint32_t i = 0; i <= j; ++i) w -= (T)sh.h[i] * Vb[(uint64_t)i * a.vs + row0 + k];
          us[k] = w;
          acc2 += w * w;
          if (pass == 1) out[k] = w;
        }
      }
      if (sh.stop) break;
    }
    part = cta_partial<T>(acc2, sh);
    if (warp == 0) finish(team_sum(parts, ctr, rank, size, ex + (t.reorth ? 4 : 2), part, t.wait_ns, &ok), true);
    __syncthreads();
    if (sh.stop) break;
    ex += t.reorth ? 4 : 2;
    // ---- W_{j+1} becomes W_j
    if (!xs) {
      T *old = xp;
      xp = xw;
      xw = us;
      us = old;
    } else if (size == 1) {
      for (uint32_t i = tid; i < n; i += kTeamThreads) xw[i] = us[i];
    } else if (j + 1 < mr) {
      const T *nx = Vb + (uint64_t)(j + 1) * a.vs;
      uint32_t i = 4 * tid;
      for (; i + 4 <= n; i += 4 * kTeamThreads) {  // 16-byte loads: node_base is a multiple of 32
#pragma unroll
        for (int b = 0; b < (int)sizeof(T) / 4; ++b)
          reinterpret_cast<float4 *>(xw + i)[b] = __ldcg(reinterpret_cast<const float4 *>(nx + i) + b);
      }
      if (tid < (n & 3u)) xw[(n & ~3u) + tid] = __ldcg(nx + (n & ~3u) + tid);
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// Plan: team sizes, what each keeps in shared memory, and whether the launch
// pays at all.
// ---------------------------------------------------------------------------
namespace {

constexpr size_t kTeamSmem = 222 * 1024;  // of 227 KB; the kernel's static part is below 3 KB
// Cost of a step in ns.  Measured at m = 20 on ER graphs of mean degree 4 to 150,
// 1 to 2000 of them, 500 to 800 000 nodes; within 30% of what the chosen route
// takes, and where two are nearer than that either will do.  What does not depend
// on the size; entries per ns of a CTA whose columns are in shared memory, the
// vector there too or in L2; bytes per ns of a CTA copying the vector from L2.
constexpr double kOneNs = 2000.0, kManyNs = 6000.0;
constexpr double kSmemPerNs = 8.0, kL2PerNs = 1.0, kCopyPerNs = 60.0;
// Columns that do not fit stay in global memory, and as a lane then walks rows of its
// own, 4 bytes of a sector at a time, long rows thrash the L1: 100 graphs of 8000
// nodes at degree 10 ran at 2.9 entries per ns, 150 of 8000 at 18 at 1.9, 100 of
// 4000 at 50 at 0.67, 140 of 1000 at 150 at 0.5 (299 us a step where the per-step
// kernels take 61 and one CTA each 34).  In FP64 0.6 (150 of 2000 at 60), and with
// the vector in L2 too 0.3 to 0.5 (1 to 8 of 30 000 to 300 000 at 24 to 120).
constexpr double kFarLeast = 0.5, kFarMost = 2.9, kFarRow = 40.0, kFar64 = 0.6, kFarL2 = 0.35;
// Reorthogonalisation, per node (of the realisation, of the call) and flat.
constexpr double kOneGs = 30.0, kManyGs = 0.18, kManyGsNs = 24000.0;

// The per-step kernels over realisations [r0, r1), ns a step: launches, tiles that
// realisations do not fill, nodes, and entries, which find the vector of a small
// graph in the L1, or are summed by the column-blocked kernel.
double steps_ns(const cb_graph *h, uint32_t r0, uint32_t r1, size_t esz, bool reorth) {
  double t = 20000.0 + 50.0 * (r1 - r0);
  const bool blocked = h->total_btiles >= h->n_sm;
  for (uint32_t r = r0; r < r1; ++r) {
    const InstDesc &I = h->inst[r];
    t += 0.02 * I.n + (esz == 8 ? 0.0065 : blocked ? 0.0011 : I.n <= 16384 ? 0.0022 : 0.0035) * I.nnz;
    if (reorth) t += 0.22 * I.n;
  }
  return t + (reorth ? 60000.0 : 0.0);
}

}  // namespace

bool small_launch_pays(const cb_graph *h, uint32_t r0, uint32_t r1) {
  double one = 0.0;
  for (uint32_t r = r0; r < r1; ++r)
    one = std::max(one, 10.0 * h->inst[r].n + 0.17 * h->inst[r].nnz);
  one *= std::max(1.0, (double)(r1 - r0) / h->n_sm);
  return 1.3 * one < steps_ns(h, r0, r1, sizeof(float), false);
}

bool team_plan(const cb_graph *h, uint32_t r0, uint32_t r1, size_t esz, bool reorth, TeamArgs *out,
               uint32_t *grid, bool *cooperative) {
  const uint32_t N = r1 - r0;
  if (h->plan_of) {  // the teams of the whole handle's plan, renumbered
    const uint32_t p0 = h->plan_r0 + r0;
    if (!team_plan(h->plan_of, 0, h->plan_of->n_inst, esz, reorth, out, grid, cooperative)) return false;
    if (!out->nteams) {
      *grid = N;
      return true;
    }
    const uint32_t base = out->first[p0];
    out->whole_x = p0 < 64 ? out->whole_x >> p0 : 0;
    for (uint32_t q = 0; q <= N; ++q) out->first[q] = (uint16_t)(out->first[p0 + q] - base);
    out->nteams = N;
    *grid = out->first[N];
    *cooperative = *grid > N;
    return true;
  }
  uint64_t nodes = 0, work = 0;
  for (uint32_t r = r0; r < r1; ++r) {
    if (h->inst[r].pb && esz == 4) return false;  // the two-phase kernels take it
    nodes += h->inst[r].n;
    work += (uint64_t)h->inst[r].nnz + h->inst[r].n;
  }
  TeamArgs &t = *out;
  t.whole_x = 0;
  t.reorth = reorth ? 1u : 0u;
  t.smem = (uint32_t)kTeamSmem;
  auto bytes = [&](const InstDesc &I, uint64_t rows, bool whole) -> size_t {
    return esz * ((whole ? (I.n + 3ull) : rows + 3) + 2 * (rows + 3)) + 4 * (rows + 4);
  };
  // ns a CTA takes for the sums of `entries` entries in `rows` rows, of which a
  // team's CTA expects that many and must have room for a tenth more (the kernel
  // looks for itself)
  auto sum_ns = [&](const InstDesc &I, double entries, double rows, bool whole) -> double {
    const double room = (rows < I.n ? 1.1 : 1.0) * entries * (I.n <= 65536 ? 2 : 4);
    if ((!whole || I.n <= 65536) && bytes(I, (uint64_t)rows, whole) + room <= (double)kTeamSmem)
      return entries / (whole ? kSmemPerNs : kL2PerNs);
    if (!whole) return entries / kFarL2;
    if (esz == 8) return entries / kFar64;
    return entries / std::min(kFarMost, std::max(kFarLeast, kFarRow * I.n / std::max(I.nnz, 1u)));
  };
  // teams of one, in waves over the SMs
  double one = 0.0;
  for (uint32_t r = r0; r < r1; ++r) {
    const InstDesc &I = h->inst[r];
    if (bytes(I, I.n, true) > kTeamSmem) one = 1e30;
    one = std::max(one, kOneNs + 2.0 * I.n / kSmemPerNs + sum_ns(I, I.nnz, I.n, true) + (reorth ? kOneGs * I.n : 0.0));
  }
  one *= (N + h->n_sm - 1) / h->n_sm;
  // teams sharing the SMs by work
  double many = 1e30;
  uint32_t total = 0;
  const uint32_t G = std::min<uint32_t>(h->n_sm, kMaxTeamCtas);
  t.rowdiv = 4;
  if (N <= G && N <= kMaxTeams) {
    for (; t.rowdiv >= 1; t.rowdiv /= 2) {
      many = 0.0;
      total = 0;
      t.whole_x = 0;
      for (uint32_t q = 0; q < N; ++q) {
        const InstDesc &I = h->inst[r0 + q];
        const uint64_t w = (uint64_t)I.nnz + I.n;
        uint64_t g = std::max<uint64_t>(1, (G - N) * w / std::max<uint64_t>(work, 1) + 1);
        g = std::min<uint64_t>(g, std::max<uint64_t>(1, w / 1024));  // enough work per CTA
        t.first[q] = (uint16_t)total;
        total += (uint32_t)g;
        // entries + rc x rows is equal over the team, rc rowdiv n >= nnz: at most
        // (rowdiv + 1) n / g + 2 rows
        const uint64_t rows = std::min<uint64_t>(I.n, (t.rowdiv + 1) * (I.n / g + 2) + 2);
        const double per = (double)I.nnz / g;
        // the whole vector each step, or gathers from L2
        const double own = (double)I.n / g, copy = I.n * esz / kCopyPerNs;
        const bool whole = g == 1 || (q < 64 && copy + sum_ns(I, per, own, true) < sum_ns(I, per, own, false) &&
                                      bytes(I, rows, true) <= kTeamSmem);
        if (whole && q < 64) t.whole_x |= 1ull << q;
        if (bytes(I, rows, whole) > kTeamSmem) many = 1e30;
        many = std::max(many, sum_ns(I, per, own, whole) +
                                  (g == 1 ? kOneNs + 2.0 * I.n / kSmemPerNs : kManyNs + (whole ? copy : 0.0)));
      }
      if (many < 1e30 || t.rowdiv == 1) break;
    }
    t.first[N] = (uint16_t)total;
    if (total > kMaxTeamCtas) many = 1e30;
    if (reorth) many += kManyGsNs + kManyGs * nodes;
  }
  const double steps = steps_ns(h, r0, r1, esz, reorth);
  if (one <= many && one <= steps) {
    t.nteams = 0;
    t.first[0] = 0;
    *grid = N;
    *cooperative = false;
    return true;
  }
  if (many <= steps) {
    t.nteams = N;
    *grid = total;
    *cooperative = total > N;
    return true;
  }
  return false;
}

template <typename T>
int team_launch(const LArgs &a, TeamArgs t, uint32_t r0, uint32_t m, uint32_t grid, bool cooperative,
                cudaStream_t s) {
  auto k = team_lanczos_kernel<T>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTeamSmem);
  if (e != cudaSuccess) return cuda_error(e, "lanczos launch");
  if (cooperative) {
    LArgs av = a;
    void *args[] = {&av, &t, &r0, &m};
    e = cudaLaunchCooperativeKernel(reinterpret_cast<const void *>(k), dim3(grid), dim3(kTeamThreads), args,
                                    kTeamSmem, s);
  } else {
    k<<<grid, kTeamThreads, kTeamSmem, s>>>(a, t, r0, m);
  }
  if (e == cudaSuccess) e = cudaGetLastError();
  return cuda_error(e, "lanczos launch");
}
template int team_launch<float>(const LArgs &, TeamArgs, uint32_t, uint32_t, uint32_t, bool, cudaStream_t);
template int team_launch<double>(const LArgs &, TeamArgs, uint32_t, uint32_t, uint32_t, bool, cudaStream_t);

CB_DEBUG_READER(team)

}  // namespace cb
