// Sub-graph centrality SC(i) = (e^A)_ii (eq. 3) of a set of nodes of one
// realisation, by Gauss quadrature.
//
// e_i^T e^A e_i is the integral of exp against the spectral measure of A
// seen from e_i; m Lanczos steps from e_i (beta0 = ||e_i|| = 1) give the
// m-point Gauss rule e1^T exp(T_m) e1 (Golub & Meurant, "Matrices, Moments
// and Quadrature with Applications", 2010).  Every derivative of exp is
// positive, so the rule is a lower bound that increases with m, exact once
// the Krylov space is invariant.  The paper calls SC expensive for large
// graphs ("Identification algorithm"); restricted to candidate nodes it
// costs one Lanczos run per node, all run together here.
//
// The recurrences of kSC start nodes run side by side over the one graph,
// their vectors stored node-major: a warp sums a row with lane q holding vector
// q, so an entry is one coalesced read of a node's kSC values and the columns
// are read once for all vectors.  Only alpha and beta are kept, so three
// vectors rotate.  Per step sc_spmv_kernel, sc_alpha_kernel, sc_axpy_kernel,
// sc_beta_kernel, launched as dependent kernels; kSC start nodes at a time.
// (k copies of the graph as k realisations, uploaded and formatted per call,
// take 3.2 ms for 30 nodes of a graph of 1e5 nodes at m = 20, half of it
// copies, formats and host scans: 1.1 ms so.)  Where a few start nodes would not
// fill the kSC vectors, or one row outlasts all others (few_pay), and with
// CB_REORTH, which needs the bases, the k start nodes become k realisations of a
// temporary handle (device-to-device copies through cb_graph_upload).  Only
// e1^T exp(T - theta) e1 is needed: no basis combine.
#include <algorithm>

#include "cb_contour.cuh"
#include "cb_reduce.cuh"
#include "cb_step.cuh"

namespace cb {
namespace {

constexpr uint32_t kSC = 32;           // recurrences side by side
constexpr uint32_t kScNodes = 256;     // nodes per CTA of the axpy
constexpr uint32_t kScLong = 256;      // longer rows are summed by the whole CTA
constexpr uint32_t kScEnd = 1u << 31;  // mark of a row's last entry

struct ScArgs {
  const uint32_t *row_ptr, *col;
  const uint2 *tiles;   // [first, last) rows
  uint32_t n, n_tiles, n_axpy, k;
  void *v[3];           // vectors j mod 3, [n][kSC]
  Scalars sc;           // per vector
  void *fac;            // [3][kSC] factors of the step: scale_j, beta_{j-1} scale_{j-1}, alpha_j scale_j
  double *part;         // [kSC][max(n_tiles, n_axpy)] partials
  uint32_t pstride;
  double tau;
};

// A factor as the vectors' arithmetic takes it, formed once per step and vector:
// in FP32 the sum of two floats (one rounded factor would shift every entry of a
// vector the same way).
template <typename T>
struct ScFac;
template <>
struct ScFac<float> {
  float hi, lo;
  __device__ static ScFac of(double v) { return {(float)v, (float)(v - (double)(float)v)}; }
  __device__ float times(float x) const { return fmaf(hi, x, lo * x); }
  __device__ float from(float c, float x) const { return fmaf(-hi, x, fmaf(-lo, x, c)); }  // c - this x
};
template <>
struct ScFac<double> {
  double hi;
  __device__ static ScFac of(double v) { return {v}; }
  __device__ double times(double x) const { return hi * x; }
  __device__ double from(double c, double x) const { return fma(-hi, x, c); }
};
template <typename T>
__device__ __forceinline__ ScFac<T> *fac_of(const ScArgs &a, int which) {
  return reinterpret_cast<ScFac<T> *>(a.fac) + which * kSC;
}

// W_0 = e_i per vector, and the scalars (vectors past k: nothing to do)
template <typename T>
__global__ void __launch_bounds__(256) sc_init_kernel(ScArgs a, const uint32_t *nodes, uint32_t m) {
  T *x = reinterpret_cast<T *>(a.v[0]);
  if (threadIdx.x < kSC) {
    const uint32_t q = threadIdx.x, ms = a.sc.ms;
    for (uint32_t j = 0; j < ms; ++j) {
      a.sc.alpha[q * ms + j] = a.sc.beta[q * ms + j] = a.sc.gamma[q * ms + j] = 0.0;
      a.sc.scale[q * ms + j] = j == 0 && q < a.k ? 1.0 : 0.0;
    }
    a.sc.meff[q] = q < a.k ? m : 0u;
    a.sc.status[q] = CB_OK;
    a.sc.theta[q] = 0.0;
    fac_of<T>(a, 0)[q] = ScFac<T>::of(q < a.k ? 1.0 : 0.0);
    fac_of<T>(a, 1)[q] = fac_of<T>(a, 2)[q] = ScFac<T>::of(0.0);
    if (q < a.k) x[(uint64_t)nodes[q] * kSC + q] = T(1);
  }
}

// u = scale_j (A W_j) - beta_{j-1} scale_{j-1} W_{j-1} for one tile of rows and
// all vectors (lane q: vector q), and the tile's alpha terms.
template <typename T>
__global__ void __launch_bounds__(kThreads) sc_spmv_kernel(ScArgs a, uint32_t j) {
  constexpr uint32_t kW = kThreads / 32;
  __shared__ uint32_t s_rp[kTileRows + 1];
  __shared__ uint32_t s_col[kTileNnz];
  __shared__ T s_sum[kW][kSC];
  __shared__ double s_part[kW][kSC];
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint2 tr = a.tiles[blockIdx.x];
  const uint32_t nrows = tr.y - tr.x;
  // The tile's row offsets and columns, while the kernel before ends.  A column
  // is kept as its offset in the vectors, the last one of a row marked, so that
  // a warp walks its rows' entries as one stream (below).  A tile with long rows
  // takes its columns from global memory.
  for (uint32_t q = threadIdx.x; q <= nrows; q += kThreads) s_rp[q] = a.row_ptr[tr.x + q];
  __syncthreads();
  const uint32_t t0 = s_rp[0], te = s_rp[nrows] - t0;
  bool over = te > kTileNnz || a.n > (kScEnd - 1) / kSC;
  for (uint32_t q = threadIdx.x; q < nrows; q += kThreads) over |= s_rp[q + 1] - s_rp[q] > kScLong;
  const bool stream = !__syncthreads_or(over);
  if (stream) {
    for (uint32_t q = threadIdx.x; q < te; q += kThreads) {
      const uint32_t c = ld_stream(a.col + t0 + q);
      s_col[q] = CB_DCHECK(c < a.n, kDbgCsrCol, c) ? c * kSC : 0u;
    }
    __syncthreads();
    for (uint32_t q = threadIdx.x; q < nrows; q += kThreads)
      if (s_rp[q + 1] > s_rp[q]) s_col[s_rp[q + 1] - 1 - t0] |= kScEnd;
  }
  // the warp's rows: as many entries each
  auto row_at = [&](uint32_t target) -> uint32_t {  // first row that starts at or after it
    uint32_t lo = 0, hi = nrows;
    while (lo < hi) {
      const uint32_t mid = (lo + hi) >> 1;
      if (s_rp[mid] - t0 >= target) hi = mid; else lo = mid + 1;
    }
    return lo;
  };
  const uint32_t w0 = warp == 0 ? 0u : row_at(te * warp / kW), w1 = warp + 1 == kW ? nrows : row_at(te * (warp + 1) / kW);
  dep_wait();
  dep_trigger();
  __syncthreads();
  const T *x = reinterpret_cast<const T *>(a.v[j % 3]) + lane;
  const T *xp = reinterpret_cast<const T *>(a.v[(j + 2) % 3]) + lane;
  T *out = reinterpret_cast<T *>(a.v[(j + 1) % 3]) + lane;
  const ScFac<T> sj = fac_of<T>(a, 0)[lane], bp = fac_of<T>(a, 1)[lane];
  double acc = 0.0;
  T acct = T(0);  // this warp's short rows
  // entries [e0, e1) of one row: eight reads of kSC values in flight
  auto run_sum = [&](uint32_t e0, uint32_t e1) -> T {
    T s = T(0);
    for (uint32_t e = e0; e < e1; e += 8) {
      T v[8];
#pragma unroll
      for (uint32_t u = 0; u < 8; ++u) {
        v[u] = T(0);
        if (e + u < e1) {
          const uint32_t c = __ldg(a.col + e + u);
          if (CB_DCHECK(c < a.n, kDbgCsrCol, c)) v[u] = x[(uint64_t)c * kSC];
        }
      }
#pragma unroll
      for (uint32_t u = 0; u < 8; ++u) s += v[u];
    }
    return s;
  };
  auto finish = [&](uint32_t row, T sum, T xr, T xpr) {
    T u = sj.times(sum);
    if (j) u = bp.from(u, xpr);
    out[(uint64_t)row * kSC] = u;
    acct += xr * u;
  };
  if (stream) {
    // the entries of rows [w0, w1) as one stream, kFly reads in flight, the sum
    // closed at each row's last entry; every branch is the same for all lanes
    constexpr uint32_t kFly = 16;
    uint32_t lr = w0;
    T sum = T(0), xr = T(0), xpr = T(0);
    auto open = [&] {  // the next row with entries; rows without end at once
      for (; lr < w1; ++lr) {
        const uint64_t o = (uint64_t)(tr.x + lr) * kSC;
        xr = x[o];
        if (j) xpr = xp[o];
        if (s_rp[lr + 1] > s_rp[lr]) break;
        finish(tr.x + lr, T(0), xr, xpr);
      }
    };
    open();
    const uint32_t eend = s_rp[w1] - t0;
    for (uint32_t e = s_rp[w0] - t0; e < eend; e += kFly) {
      T v[kFly];
      uint32_t c[kFly];
#pragma unroll
      for (uint32_t u = 0; u < kFly; ++u) {
        c[u] = s_col[min(e + u, eend - 1)];  // past the end: the last one again, not added
        v[u] = x[c[u] & (kScEnd - 1)];
      }
#pragma unroll
      for (uint32_t u = 0; u < kFly; ++u) {
        if (e + u >= eend) break;
        sum += v[u];
        if (c[u] & kScEnd) {
          finish(tr.x + lr, sum, xr, xpr);
          sum = T(0);
          ++lr;
          open();
        }
      }
    }
    acc = (double)acct;
  } else {
    for (uint32_t lr = warp; lr < nrows; lr += kW) {
      const uint32_t e0 = s_rp[lr], e1 = s_rp[lr + 1], row = tr.x + lr;
      if (e1 - e0 > kScLong) continue;
      const T xr = x[(uint64_t)row * kSC], xpr = j ? xp[(uint64_t)row * kSC] : T(0);
      finish(row, run_sum(e0, e1), xr, xpr);
    }
    acc = (double)acct;
    // long rows: a part per warp, added in warp order
    for (uint32_t lr = 0; lr < nrows; ++lr) {
      const uint32_t e0 = s_rp[lr], e1 = s_rp[lr + 1], row = tr.x + lr;
      if (e1 - e0 <= kScLong) continue;  // uniform
      const uint32_t per = (e1 - e0 + kW - 1) / kW;
      const uint32_t b0 = min(e1, e0 + warp * per), b1 = min(e1, b0 + per);
      s_sum[warp][lane] = run_sum(b0, b1);
      __syncthreads();
      if (warp == 0) {
        T sum = T(0);
        for (uint32_t w = 0; w < kW; ++w) sum += s_sum[w][lane];
        acct = T(0);
        finish(row, sum, x[(uint64_t)row * kSC], j ? xp[(uint64_t)row * kSC] : T(0));
        acc += (double)acct;
      }
      __syncthreads();
    }
  }
  s_part[warp][lane] = acc;
  __syncthreads();
  if (warp == 0) {
    double t = 0.0;
    for (uint32_t w = 0; w < kW; ++w) t += s_part[w][lane];
    a.part[(uint64_t)lane * a.pstride + blockIdx.x] = t;
  }
}

// Sum of a vector's partials: threads strided, then warps in order (one CTA of
// 128 threads per vector; valid in thread 0).
__device__ __forceinline__ double sc_total(const double *p, uint32_t count) {
  __shared__ double s_w[4];
  double acc = 0.0;
  for (uint32_t q = threadIdx.x; q < count; q += 128) acc += p[q];
  acc = warp_sum_d(acc);
  if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = acc;
  __syncthreads();
  return threadIdx.x == 0 ? ((s_w[0] + s_w[1]) + s_w[2]) + s_w[3] : 0.0;
}

template <typename T>
__global__ void __launch_bounds__(128) sc_alpha_kernel(ScArgs a, uint32_t j) {
  const uint32_t q = blockIdx.x, ms = a.sc.ms;
  dep_wait();
  dep_trigger();
  if (j >= a.sc.meff[q]) return;
  const double total = sc_total(a.part + (uint64_t)q * a.pstride, a.n_tiles);
  if (threadIdx.x) return;
  const double alpha = a.sc.scale[q * ms + j] * total;
  a.sc.alpha[q * ms + j] = alpha;
  fac_of<T>(a, 2)[q] = ScFac<T>::of(alpha * a.sc.scale[q * ms + j]);
  if (!isfinite(alpha)) {
    if (a.sc.status[q] == CB_OK) a.sc.status[q] = CB_ERR_NONFINITE;
    a.sc.meff[q] = j;
    fac_of<T>(a, 0)[q] = fac_of<T>(a, 1)[q] = fac_of<T>(a, 2)[q] = ScFac<T>::of(0.0);
  }
}

// w = u - alpha_j scale_j W_j in place and the partials of ||w||^2: kScNodes
// nodes per CTA, 4 consecutive vectors of a node per thread.
template <typename T>
__global__ void __launch_bounds__(256) sc_axpy_kernel(ScArgs a, uint32_t j) {
  __shared__ double s_part[8][kSC];
  const uint32_t q0 = 4 * (threadIdx.x & 7), warp = threadIdx.x >> 5;
  const T *x = reinterpret_cast<const T *>(a.v[j % 3]);
  T *w = reinterpret_cast<T *>(a.v[(j + 1) % 3]);
  dep_wait();
  dep_trigger();
  ScFac<T> c[4];
  T acc[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    c[u] = fac_of<T>(a, 2)[q0 + u];
    acc[u] = T(0);
  }
  const uint32_t i1 = min(a.n, (blockIdx.x + 1) * kScNodes);
#pragma unroll 2
  for (uint32_t i = blockIdx.x * kScNodes + threadIdx.x / 8; i < i1; i += 32) {
    T *wr = w + (uint64_t)i * kSC + q0;
    const T *xr = x + (uint64_t)i * kSC + q0;
    T a4[4], b4[4];
#pragma unroll
    for (int u = 0; u < 4; u += 16 / (int)sizeof(T)) {
      *reinterpret_cast<float4 *>(a4 + u) = *reinterpret_cast<const float4 *>(wr + u);
      *reinterpret_cast<float4 *>(b4 + u) = *reinterpret_cast<const float4 *>(xr + u);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      a4[u] = c[u].from(a4[u], b4[u]);
      acc[u] += a4[u] * a4[u];
    }
#pragma unroll
    for (int u = 0; u < 4; u += 16 / (int)sizeof(T))
      *reinterpret_cast<float4 *>(wr + u) = *reinterpret_cast<const float4 *>(a4 + u);
  }
  // over the four nodes of a warp's pass, then the warps in order
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    acc[u] += __shfl_xor_sync(0xffffffffu, acc[u], 8);
    acc[u] += __shfl_xor_sync(0xffffffffu, acc[u], 16);
    if ((threadIdx.x & 31) < 8) s_part[warp][q0 + u] = (double)acc[u];
  }
  __syncthreads();
  if (threadIdx.x < kSC) {
    double t = 0.0;
    for (int v = 0; v < 8; ++v) t += s_part[v][threadIdx.x];
    a.part[(uint64_t)threadIdx.x * a.pstride + blockIdx.x] = t;
  }
}

template <typename T>
__global__ void __launch_bounds__(128) sc_beta_kernel(ScArgs a, uint32_t j) {
  const uint32_t q = blockIdx.x, ms = a.sc.ms;
  dep_wait();
  dep_trigger();
  if (j >= a.sc.meff[q]) return;
  const double total = sc_total(a.part + (uint64_t)q * a.pstride, a.n_axpy);
  if (threadIdx.x) return;
  const double beta = sqrt(total), alpha = a.sc.alpha[q * ms + j];
  const double bprev = j ? a.sc.beta[q * ms + j - 1] : 0.0;
  a.sc.beta[q * ms + j] = beta;
  ScFac<T> sj = ScFac<T>::of(0.0), bp = sj;  // a vector that stops: nothing more
  if (!isfinite(beta)) {
    a.sc.status[q] = CB_ERR_NONFINITE;
    a.sc.meff[q] = j + 1;
  } else if (beta <= a.tau * (fabs(alpha) + bprev) || beta == 0.0) {
    a.sc.meff[q] = j + 1;  // exact breakdown
  } else {
    const double scale = 1.0 / beta;
    a.sc.scale[q * ms + j + 1] = scale;
    sj = ScFac<T>::of(scale);
    bp = ScFac<T>::of(beta * a.sc.scale[q * ms + j]);
  }
  fac_of<T>(a, 0)[q] = sj;
  fac_of<T>(a, 1)[q] = bp;
  if (a.sc.meff[q] == j + 1) fac_of<T>(a, 2)[q] = ScFac<T>::of(0.0);
}

// One warp per start node: theta_q = lambda_max(T), c0_q = [exp(T - theta) e1]_0
// via the contour rule (theta in sc.theta[q], c0 in sc.gamma[q * ms]).
__global__ void __launch_bounds__(32) sc_tridiag_kernel(Scalars sc, contour::Nodes nd, bool laguerre) {
  using namespace contour;
  __shared__ double s_al[CB_MAX_M], s_be[CB_MAX_M];
  __shared__ Solve s_s;
  __shared__ Spectrum s_sp;
  const uint32_t q = blockIdx.x, lane = threadIdx.x, ms = sc.ms;
  const int M = (int)sc.meff[q];
  if (sc.status[q] != CB_OK || M < 1) {
    if (lane == 0) {
      sc.theta[q] = 0.0;
      sc.gamma[q * ms] = M < 1 && sc.status[q] == CB_OK ? 0.0 : __longlong_as_double(0x7ff8000000000000ll);
    }
    return;
  }
  for (int i = lane; i < M; i += 32) {
    s_al[i] = sc.alpha[q * ms + i];
    s_be[i] = sc.beta[q * ms + i];
  }
  __syncwarp();
  const double theta = largest(s_al, s_be, M, s_sp, laguerre);
  __syncwarp();
  cplx inv0;
  const double scale = continuants(s_al, s_be, M, theta, nd, s_s, &inv0);
  real_sum(s_s, 1, 2.0 * scale, cmul(nd.w[lane < kCols ? lane >> 1 : 0], inv0), [&](int, double c0) {
    sc.theta[q] = theta;
    sc.gamma[q * ms] = c0;
  });
}

// Common shift theta* = max_q theta_q; out[q] = exp(theta_q - theta*) c0_q.
__global__ void __launch_bounds__(256) sc_finish_kernel(Scalars sc, uint32_t k, double *out,
                                                        double *log_scale) {
  __shared__ double s_max[8];
  double tm = -1e308;
  for (uint32_t q = threadIdx.x; q < k; q += blockDim.x)
    if (sc.status[q] == CB_OK) tm = fmax(tm, sc.theta[q]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) tm = fmax(tm, __shfl_xor_sync(0xffffffffu, tm, o));
  if ((threadIdx.x & 31) == 0) s_max[threadIdx.x >> 5] = tm;
  __syncthreads();
  double tmax = s_max[0];
  for (int w = 1; w < 8; ++w) tmax = fmax(tmax, s_max[w]);
  if (tmax < -1e307) tmax = 0.0;
  for (uint32_t q = threadIdx.x; q < k; q += blockDim.x)
    out[q] = sc.status[q] == CB_OK ? exp(sc.theta[q] - tmax) * sc.gamma[q * sc.ms]
                                   : __longlong_as_double(0x7ff8000000000000ll);
  if (threadIdx.x == 0) *log_scale = tmax;
}

}  // namespace
CB_DEBUG_READER(subgraph)

}  // namespace cb

using namespace cb;

// Whether k copies of the graph are the better route for k start nodes.  kSC
// vectors cost the same whatever k; m = 20, by copies / by kSC vectors, ms:
//   FP32  1e5 nodes, degree 10: k = 1 1.08 / 1.13, 2 1.26 / 1.13; degree 40: 1 1.5 /
//         2.8, 4 2.8 / 2.8; 1e6, degree 16: 1 5.9 / 10.7, 4 10.2 / 10.8, 8 14.7 / 10.7;
//         1e7: 1 52 / 109, 4 100 / 109, 8 158 / 109
//   FP64  1e4, degree 10: 4 1.04 / 1.22, 8 1.22 / 1.22; 1e5: 1 1.2 / 2.7, 4 2.0 / 2.7,
//         8 2.8 / 2.7; degree 40: 8 6.7 / 7.3; 1e6: 1 7 / 28, 8 24 / 29, 16 42 / 29
// And one CTA sums each row there, 16 ns an entry (FP64: 21), where the copies'
// kernels cut rows of more than kHeavyDeg entries over the chip: a row of 300 000
// among 1e6 nodes 95 ms at any k, by copies 5 at k = 1, 17 at 16; of 9000 among 1e5
// 2.5 ms, 1.1 at 1, 2.2 at 8, 3.3 at 30.
static bool few_pay(const InstDesc &I, uint32_t k, int prec) {
  const bool f64 = prec == CB_FP64;
  const uint64_t nnz = I.nnz;
  if (k <= (f64 ? (nnz >= 4000000u ? 8u : 6u) : nnz >= 4000000u ? 4u : nnz >= 2000000u ? 2u : 1u)) return true;
  const double row_ns = (f64 ? 21.0 : 16.0) * I.longest * ((k + kSC - 1) / kSC);
  return 50000.0 + (f64 ? 0.0107 : 0.0055) * nnz * k < row_ns;
}

// k copies of the graph as realisations of a temporary handle.
static int sc_copies(cb_graph *h, uint32_t inst, uint32_t m, int prec, bool reorth, uint32_t k,
                     const uint32_t *d_nodes, double *sc_scaled, double *log_scale, cudaStream_t s) {
  const InstDesc I = h->inst[inst];
  const uint64_t nnz = (inst + 1 < h->n_inst ? h->inst[inst + 1].edge_base : h->total_nnz) - I.edge_base;
  // k copies of realisation inst, one per start node
  std::vector<uint32_t> vn(k, I.n);
  std::vector<uint64_t> vnnz(k, nnz);
  std::vector<const uint32_t *> vrp(k, h->row_ptr + I.rp_base), vcol(k, h->col + I.edge_base);
  cb_graph *v = nullptr;
  int rc = cb_graph_upload(k, vn.data(), vnnz.data(), vrp.data(), vcol.data(), CB_DEVICE_PTRS,
                           s, &v);
  if (rc != CB_OK) return rc;
  v->reorth = reorth;
  rc = ensure_workspace(v, v->ws, m, prec, s);
  if (rc == CB_OK) rc = lanczos_run(v, v->ws, 0, k, m, prec, s, d_nodes, k, true);
  if (rc == CB_OK) {
    sc_tridiag_kernel<<<k, 32, 0, s>>>(v->ws.sc, contour::nodes(), prec == CB_FP64);
    sc_finish_kernel<<<1, 256, 0, s>>>(v->ws.sc, k, sc_scaled, log_scale);
    rc = cuda_error(cudaGetLastError(), "cb_subgraph_centrality: launch");
  }
  if (rc == CB_OK) rc = cuda_error(cudaStreamSynchronize(s), "cb_subgraph_centrality");
  const int rf = cb_graph_free(v);
  return rc != CB_OK ? rc : rf;
}

// kSC start nodes at a time over the one graph.
template <typename T>
static int sc_batches(cb_graph *h, uint32_t inst, uint32_t m, uint32_t k, const uint32_t *d_nodes,
                      double *sc_scaled, double *log_scale, cudaStream_t s) {
  const InstDesc &I = h->inst[inst];
  const uint32_t ms = m + 1, kp = (k + kSC - 1) / kSC * kSC;
  ScArgs a;
  a.row_ptr = h->row_ptr + I.rp_base;
  a.col = h->col + I.edge_base;
  a.tiles = h->d_tile_rows + I.tile_base;
  a.n = I.n;
  a.n_tiles = I.n_tiles;
  a.n_axpy = (I.n + kScNodes - 1) / kScNodes;
  a.pstride = std::max(a.n_tiles, a.n_axpy);
  a.tau = sizeof(T) == 4 ? 1e-5 : 1e-12;
  const uint64_t vec = (uint64_t)I.n * kSC;
  const uint64_t nd = 4ull * kp * ms + kp + (uint64_t)kSC * a.pstride + 3 * kSC;
  const size_t bytes = 3 * vec * sizeof(T) + nd * 8 + 2ull * kp * 4;
  void *blob = nullptr;
  cudaError_t e = dev_alloc(&blob, bytes);
  if (e != cudaSuccess) return cuda_error(e, "cb_subgraph_centrality: vectors");
  for (int q = 0; q < 3; ++q) a.v[q] = reinterpret_cast<T *>(blob) + q * vec;
  double *d = reinterpret_cast<double *>(reinterpret_cast<T *>(blob) + 3 * vec);  // n kSC T: a multiple of 8 bytes
  Scalars all;
  all.alpha = d; d += (uint64_t)kp * ms;
  all.beta = d; d += (uint64_t)kp * ms;
  all.scale = d; d += (uint64_t)kp * ms;
  all.gamma = d; d += (uint64_t)kp * ms;
  all.theta = d; d += kp;
  a.part = d; d += (uint64_t)kSC * a.pstride;
  a.fac = d; d += 3 * kSC;
  static_assert(sizeof(ScFac<T>) == 8, "a factor takes 8 bytes");
  all.meff = reinterpret_cast<uint32_t *>(d);
  all.status = reinterpret_cast<int32_t *>(all.meff + kp);
  all.ms = ms;
  for (uint32_t b = 0; b < k && e == cudaSuccess; b += kSC) {
    a.k = std::min(kSC, k - b);
    a.sc = all;
    a.sc.alpha += (uint64_t)b * ms;
    a.sc.beta += (uint64_t)b * ms;
    a.sc.scale += (uint64_t)b * ms;
    a.sc.gamma += (uint64_t)b * ms;
    a.sc.theta += b;
    a.sc.meff += b;
    a.sc.status += b;
    e = cudaMemsetAsync(a.v[0], 0, vec * sizeof(T), s);
    sc_init_kernel<T><<<1, 256, 0, s>>>(a, d_nodes + b, m);
    for (uint32_t j = 0; j < m; ++j) {
      launch_dep(sc_spmv_kernel<T>, a.n_tiles, kThreads, 0, s, a, j);
      launch_dep(sc_alpha_kernel<T>, kSC, 128, 0, s, a, j);
      launch_dep(sc_axpy_kernel<T>, a.n_axpy, 256, 0, s, a, j);
      launch_dep(sc_beta_kernel<T>, kSC, 128, 0, s, a, j);
    }
  }
  if (e == cudaSuccess) {
    sc_tridiag_kernel<<<k, 32, 0, s>>>(all, contour::nodes(), sizeof(T) == 8);
    sc_finish_kernel<<<1, 256, 0, s>>>(all, k, sc_scaled, log_scale);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  dev_free(blob);
  return cuda_error(e, "cb_subgraph_centrality");
}

CB_API int cb_subgraph_centrality(cb_graph *h, uint32_t inst, uint32_t m, int prec, uint32_t k,
                                  const uint32_t *nodes, double *sc_scaled, double *log_scale,
                                  void *stream) {
  NvtxRange nvtx_range("cb_subgraph_centrality");
  if (!h || !nodes || !sc_scaled || !log_scale)
    return set_error(CB_ERR_ARG, "cb_subgraph_centrality: null argument");
  if (inst >= h->n_inst) return set_error(CB_ERR_ARG, "cb_subgraph_centrality: realisation out of range");
  if (m < 1 || m > CB_MAX_M) return set_error(CB_ERR_ARG, "cb_subgraph_centrality: need 1 <= m <= CB_MAX_M");
  const bool reorth = split_prec(prec);
  if (prec != CB_FP32 && prec != CB_FP64) return set_error(CB_ERR_ARG, "cb_subgraph_centrality: bad precision");
  if (k < 1 || k > CB_MAX_SC_NODES)
    return set_error(CB_ERR_ARG, "cb_subgraph_centrality: need 1 <= k <= CB_MAX_SC_NODES");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const InstDesc I = h->inst[inst];
  // the node indices are read back once to reject out-of-range entries
  std::vector<uint32_t> hn(k);
  cudaError_t e = cudaMemcpyAsync(hn.data(), nodes, k * 4ull, cudaMemcpyDefault, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return cuda_error(e, "cb_subgraph_centrality: read nodes");
  for (uint32_t q = 0; q < k; ++q)
    if (hn[q] >= I.n) return set_error(CB_ERR_ARG, "cb_subgraph_centrality: node index >= n");
  const uint32_t *d_nodes = nodes;
  uint32_t *tmp = nullptr;
  cudaPointerAttributes pa{};
  if (cudaPointerGetAttributes(&pa, nodes) != cudaSuccess || pa.type != cudaMemoryTypeDevice) {
    cudaGetLastError();  // host pointer: stage the indices on the device
    e = dev_alloc_n(&tmp, k);
    if (e == cudaSuccess) e = cudaMemcpyAsync(tmp, hn.data(), k * 4ull, cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) {
      dev_free(tmp);
      return cuda_error(e, "cb_subgraph_centrality: stage nodes");
    }
    d_nodes = tmp;
  }
  const bool few = reorth || few_pay(I, k, prec);
  int rc = CB_OK;
  for (int route = 0; route < 2; ++route) {  // out of memory: the other route may fit
    rc = few == (route == 0) ? sc_copies(h, inst, m, prec, reorth, k, d_nodes, sc_scaled, log_scale, s)
         : prec == CB_FP64   ? sc_batches<double>(h, inst, m, k, d_nodes, sc_scaled, log_scale, s)
                             : sc_batches<float>(h, inst, m, k, d_nodes, sc_scaled, log_scale, s);
    if (rc != CB_ERR_OOM || reorth) break;
  }
  dev_free(tmp);
  return rc;
}
