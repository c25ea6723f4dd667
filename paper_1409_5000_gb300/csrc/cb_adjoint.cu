// Adjoint: edge gradient of the summed top-k total communicability.
//
// The paper has no gradient; this differentiates its score.  With w the
// indicator of a fixed node set S (the recovered top-k of eq. 5), the loss is
//     L = sum_r sum_{i in S, i < n_r} (e^{A_r} 1)_i = sum_r w_r^T e^{A_r} 1,
// and for the undirected weight a_ij = a_ji of an existing edge of A_r
//     dL/da_ij = G_ij + G_ji,   G = int_0^1 e^{sA} w 1^T e^{(1-s)A} ds
// (the Frechet derivative of e^A, contracted with w and 1).
//
// Krylov form.  With Lanczos bases V_w (from w) and V_1 (from 1) and their
// tridiagonals T_w, T_1, e^{sA} w ~ ||w|| V_w e^{s T_w} e1 and
// e^{(1-s)A} 1 ~ sqrt(n) V_1 e^{(1-s) T_1} e1, so G ~ V_w M V_1^T with
//     M = ||w|| sqrt(n) int_0^1 (e^{s T_w} e1)(e^{(1-s) T_1} e1)^T ds.
// M is the upper-right block of exp([[T_w, e1 e1^T], [0, T_1]]) (Van Loan's
// block formula).  The resolvent of that block-triangular matrix has
// upper-right block R_w(z) e1 e1^T R_1(z), so the contour rule of the
// forward step (cb_contour.cuh) gives, with the shift theta,
//     M = ||w|| sqrt(n) 2 Re sum_k w_k x_k y_k^T,
//     x_k = (z_k I - (T_w - theta))^{-1} e1,  y_k = (z_k I - (T_1 - theta))^{-1} e1:
// 24 complex tridiagonal solves and 12 rank-1 terms, no eigendecomposition.
//
// Then P = V_w M and U = V_1 are written node-major (m contiguous values per
// node) and every CSR entry (i, j) gets g = P_i . U_j + P_j . U_i, computed
// in the basis precision (FP32 or FP64).  Realisations share one shift theta* =
// max_r theta_r; dL/da_e = exp(theta*) * grad[e].
#include <algorithm>
#include <cstdlib>

#include "cb_contour.cuh"
#include "cb_reduce.cuh"

namespace cb {

CB_DEBUG_STATE()

constexpr uint32_t kMaxAdjM = 64;  // adjoint depth limit (shared-memory staging)

void free_backwork(BackWork &B) {
  dev_free(B.P);
  dev_free(B.U);
  dev_free(B.blob);
  B = BackWork{};
}

static int ensure_backwork(cb_graph *h, uint32_t m, int prec, cudaStream_t s) {
  BackWork &B = h->bw;
  if (B.P && B.prec == prec && B.m == m) return CB_OK;
  free_backwork(B);
  const uint32_t mpad = (m + 3) / 4 * 4;
  const size_t esz = prec == CB_FP64 ? sizeof(double) : sizeof(float);
  const size_t vb = h->total_nodes_padded * mpad * esz + 16;
  cudaError_t e = dev_alloc(&B.P, vb);
  if (e == cudaSuccess) e = dev_alloc(&B.U, vb);
  const uint32_t N = h->n_inst;
  const size_t bytes = ((size_t)N * m * m + N) * sizeof(double) + (size_t)N * sizeof(uint32_t) + 64;
  if (e == cudaSuccess) e = dev_alloc(&B.blob, bytes);
  if (e != cudaSuccess) {
    free_backwork(B);
    return cuda_error(e, "adjoint workspace");
  }
  B.K = reinterpret_cast<double *>(B.blob);
  B.theta = B.K + (size_t)N * m * m;
  B.cnt = reinterpret_cast<uint32_t *>(B.theta + N);
  B.prec = prec;
  B.m = m;
  B.mpad = mpad;
  return cuda_error(cudaMemsetAsync(B.blob, 0, bytes, s), "adjoint workspace clear");
}

// Two warps per realisation: theta_r and the coefficient matrix K_r = M_r.
// Warp 0 solves for the basis from w, warp 1 for the one from 1 (on sub-cores
// of their own: each has its FP64 unit).
__global__ void __launch_bounds__(64) bw_tridiag_kernel(Scalars s1, Scalars sw,
                                                        const InstDesc *inst, double *K,
                                                        uint32_t kdim, double *theta_out,
                                                        uint32_t *cnt_out, contour::Nodes nd,
                                                        bool laguerre) {
  using namespace contour;
  extern __shared__ double s_dyn[];
  Solve *s_s = reinterpret_cast<Solve *>(s_dyn);  // [2]
  __shared__ double s_al[2][kMaxAdjM], s_be[2][kMaxAdjM];
  __shared__ double s_th[2], s_scale[2];
  __shared__ cplx s_inv0[2][kHalf];
  __shared__ Spectrum s_sp[2];
  const uint32_t r = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
  const int M1 = (int)s1.meff[r], Mw = (int)sw.meff[r];
  const bool ok = M1 > 0 && Mw > 0 && s1.status[r] == CB_OK && sw.status[r] == CB_OK;
  if (!ok) {
    if (tid == 0) {
      theta_out[r] = -1e308;
      cnt_out[r] = 0;
    }
    return;
  }
  const Scalars &sc = wp ? s1 : sw;
  const int M = wp ? M1 : Mw;
  for (int i = lane; i < M; i += 32) {
    s_al[wp][i] = sc.alpha[r * sc.ms + i];
    s_be[wp][i] = sc.beta[r * sc.ms + i];
  }
  __syncwarp();
  const double th = largest(s_al[wp], s_be[wp], M, s_sp[wp], laguerre);
  if (lane == 0) s_th[wp] = th;
  __syncthreads();
  const double theta = fmax(s_th[0], s_th[1]);
  cplx inv0;
  const double scale = continuants(s_al[wp], s_be[wp], M, theta, nd, s_s[wp], &inv0);
  if (lane < kCols && !(lane & 1)) s_inv0[wp][lane >> 1] = inv0;
  if (lane == 0) s_scale[wp] = scale;
  __syncthreads();
  // x_k of the basis from w in place of its continuants, with the node's weight
  // and both 1 / phi_0 folded in
  for (int t = tid; t < Mw * kHalf; t += 64) {
    const int i = t / kHalf, k = t % kHalf;
    double *x = s_s[0].phi + i * kCols + 2 * k;
    const cplx v = cmul(cmul(cmul(nd.w[k], s_inv0[0][k]), s_inv0[1][k]), {x[0], x[1]});
    x[0] = v.re;
    x[1] = -v.im;  // the product below takes the real part
  }
  __syncthreads();
  // ||w|| = 1 / scale_w[0], sqrt(n) = 1 / scale_1[0]
  const double c = 2.0 * s_scale[0] * s_scale[1] / (sw.scale[r * sw.ms] * s1.scale[r * s1.ms]);
  double *Kr = K + (size_t)r * kdim * kdim;
  for (int q = tid; q < Mw * M1; q += 64) {
    const int a = q / M1, b = q % M1;
    const double *x = s_s[0].phi + a * kCols, *y = s_s[1].phi + b * kCols;
    double acc = 0.0;
#pragma unroll
    for (int k = 0; k < kCols; ++k) acc = fma(x[k], y[k], acc);
    Kr[a * kdim + b] = c * (s_s[0].B[a] * s_s[1].B[b]) * acc;
  }
  if (tid == 0) {
    theta_out[r] = theta;
    const double sw0 = sw.scale[r * sw.ms];
    cnt_out[r] = (uint32_t)llrint(1.0 / (sw0 * sw0));
  }
}

// 16 bytes of consecutive values
__device__ __forceinline__ void ld16(const float *p, float (&v)[4]) {
  const float4 x = *reinterpret_cast<const float4 *>(p);
  v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
}
__device__ __forceinline__ void ld16(const double *p, double (&v)[2]) {
  const double2 x = *reinterpret_cast<const double2 *>(p);
  v[0] = x.x; v[1] = x.y;
}

// B-byte asynchronous copy global -> shared (both addresses B-byte aligned)
template <int B>
__device__ __forceinline__ void cp_async(void *smem, const void *gmem) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(smem);
  if constexpr (B == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(gmem) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(d), "l"(gmem), "n"(B) : "memory");
}

// Node-major P = exp(theta_r - theta*) V_w K_r and U = V_1 (scales applied).
// One CTA per finalize tile (kFinRows nodes of one realisation), 4 warps.  A
// warp copies 32 nodes' basis values to shared memory asynchronously (all 2 m
// lines in flight; the scales go into K and into the stored U); lane b then holds
// P_q,b of all 32 nodes q in registers, so that a step of the sum over a takes
// one load of K and 32 values of V_w by 16-byte broadcasts for 32 products
// (2.3 ms on 64 graphs of 1e5 nodes at m = 30 when every product loaded both of
// its operands, and U was read back through one bank; now 0.72), and writes
// the node-major rows with lanes over the row index (coalesced).  All
// per-node arithmetic runs in T: the FP64 scalars are converted once per CTA
// (FP64 instructions are scarce on GB300).
template <typename T>
__global__ void __launch_bounds__(128) bw_node_kernel(const T *V1, const T *Vw, uint64_t vs,
                                                      Scalars s1, Scalars sw,
                                                      const InstDesc *inst, const uint32_t *fin_inst,
                                                      uint32_t n_inst, const double *K,
                                                      uint32_t kdim, const double *theta_in,
                                                      uint32_t mpad, T *P, T *U,
                                                      double *log_scale) {
  extern __shared__ float4 s_raw4[];
  T *sV = reinterpret_cast<T *>(s_raw4);             // 4 warps x kdim x 32 (V_w values)
  T *sW = sV + 4 * kdim * 32;                        // 4 warps x kdim x 33 (V_1 values)
  T *sK = sW + 4 * kdim * 33;                        // kdim * kdim
  __shared__ T s_sc1[kMaxAdjM];
  __shared__ double s_wmax[4];
  const uint32_t t = blockIdx.x;
  const uint32_t r = fin_inst[t];
  const InstDesc I = inst[r];
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double tm = -1e308;
  for (uint32_t q = threadIdx.x; q < n_inst; q += blockDim.x) tm = fmax(tm, theta_in[q]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) tm = fmax(tm, __shfl_xor_sync(0xffffffffu, tm, o));
  if (lane == 0) s_wmax[warp] = tm;
  const double th = theta_in[r];
  const bool active = th > -1e307;
  const int M1 = active ? (int)s1.meff[r] : 0, Mw = active ? (int)sw.meff[r] : 0;
  for (int q = threadIdx.x; q < M1; q += blockDim.x) s_sc1[q] = (T)s1.scale[r * s1.ms + q];
  __syncthreads();
  const double tmax = fmax(fmax(s_wmax[0], s_wmax[1]), fmax(s_wmax[2], s_wmax[3]));
  if (t == 0 && threadIdx.x == 0) *log_scale = tmax > -1e307 ? tmax : 0.0;
  const double f = active ? exp(th - tmax) : 0.0;
  for (uint32_t q = threadIdx.x; q < (uint32_t)(Mw * M1); q += blockDim.x) {
    const uint32_t a = q / M1, b = q % M1;
    sK[a * kdim + b] = (T)(f * sw.scale[r * sw.ms + a] * K[(size_t)r * kdim * kdim + a * kdim + b]);
  }
  __syncthreads();
  T *myV = sV + warp * kdim * 32, *myW = sW + warp * kdim * 33;
  const uint32_t i0 = (t - I.fin_base) * kFinRows, i1 = min(i0 + kFinRows, I.n);
  for (uint32_t base = i0 + warp * 32; base < i1; base += 4 * 32) {
    // whole groups of 32 nodes: the node ranges are padded to them
    const T *gw = Vw + I.node_base + base, *g1 = V1 + I.node_base + base + lane;
    constexpr uint32_t kV = 16 / sizeof(T), kParts = 32 / kV;  // 16-byte parts of a vector's 32 values
    for (uint32_t q = lane; q < Mw * kParts; q += 32) {
      const uint32_t a = q / kParts, part = (q % kParts) * kV;
      cp_async<16>(myV + a * 32 + part, gw + (uint64_t)a * vs + part);
    }
    for (int b = 0; b < M1; ++b) cp_async<sizeof(T)>(myW + b * 33 + lane, g1 + (uint64_t)b * vs);
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncwarp();
    const uint32_t nn = min(32u, i1 - base);
    for (uint32_t b = lane; b < ((mpad + 31) & ~31u); b += 32) {  // uniform trip count
      const bool in = (int)b < M1;
      T p[32];
#pragma unroll
      for (int q = 0; q < 32; ++q) p[q] = T(0);
      for (int a = 0; a < Mw; ++a) {
        const T k = in ? sK[a * kdim + b] : T(0);
#pragma unroll
        for (int q = 0; q < 32; q += (int)kV) {
          T v[kV];
          ld16(myV + a * 32 + q, v);
#pragma unroll
          for (int u = 0; u < (int)kV; ++u) p[q + u] += v[u] * k;
        }
      }
      if (b < mpad) {
        T *Pr = P + (I.node_base + base) * (uint64_t)mpad + b, *Ur = U + (I.node_base + base) * (uint64_t)mpad + b;
#pragma unroll
        for (uint32_t q = 0; q < 32; ++q)
          if (q < nn) {
            Pr[(uint64_t)q * mpad] = p[q];
            Ur[(uint64_t)q * mpad] = in ? s_sc1[b] * myW[b * 33 + q] : T(0);
          }
      }
    }
    __syncwarp();
  }
}

// mirror[e] for every CSR entry e = (i, j) of one SpMV tile: the position of
// (j, i) in row j (rows are sorted; binary search).  An entry without a
// mirror (asymmetric input) points at itself.
__global__ void __launch_bounds__(256) bw_mirror_kernel(const InstDesc *inst,
                                                        const uint32_t *tile_inst,
                                                        const uint2 *tile_rows,
                                                        const uint32_t *row_ptr, const uint32_t *col,
                                                        uint32_t *mirror) {
  __shared__ uint32_t s_rp[kTileRows + 1];
  const uint32_t t = blockIdx.x;
  const InstDesc I = inst[tile_inst[t]];
  const uint32_t *rp = row_ptr + I.rp_base;
  const uint32_t *cl = col + I.edge_base;
  const uint2 tr = tile_rows[t];
  const uint32_t row0 = tr.x, nrows = tr.y - tr.x;
  for (uint32_t q = threadIdx.x; q <= nrows; q += blockDim.x) s_rp[q] = rp[row0 + q];
  __syncthreads();
  for (uint32_t e = s_rp[0] + threadIdx.x; e < s_rp[nrows]; e += blockDim.x) {
    uint32_t lo = 0, hi = nrows;  // last lr with s_rp[lr] <= e
    while (hi - lo > 1) {
      const uint32_t mid = (lo + hi) >> 1;
      if (s_rp[mid] <= e) lo = mid; else hi = mid;
    }
    const uint32_t i = row0 + lo, j = __ldg(cl + e);
    if (!CB_DCHECK(j < I.n, kDbgAdjointCol, j)) {
      mirror[I.edge_base + e] = e;
      continue;
    }
    uint32_t a = rp[j], b = rp[j + 1];  // first position in row j with col >= i
    while (a < b) {
      const uint32_t mid = (a + b) >> 1;
      if (__ldg(cl + mid) < i) a = mid + 1; else b = mid;
    }
    mirror[I.edge_base + e] = (a < rp[j + 1] && __ldg(cl + a) == i) ? a : e;
  }
}

// 4 consecutive values (16- or 32-byte aligned)
template <typename T>
struct Quad {
  T v[4];
};
__device__ __forceinline__ Quad<float> ld_quad(const float *p) {
  const float4 x = *reinterpret_cast<const float4 *>(p);
  return {{x.x, x.y, x.z, x.w}};
}
__device__ __forceinline__ Quad<double> ld_quad(const double *p) {
  const double2 x = *reinterpret_cast<const double2 *>(p), y = *reinterpret_cast<const double2 *>(p + 2);
  return {{x.x, x.y, y.x, y.y}};
}
template <typename T>
__device__ __forceinline__ T dot4(const Quad<T> &a, const Quad<T> &b) {
  return a.v[0] * b.v[0] + a.v[1] * b.v[1] + a.v[2] * b.v[2] + a.v[3] * b.v[3];
}

// The gradient is symmetric: g(i, j) = P_i . U_j + P_j . U_i = g(j, i).  Each
// undirected edge is computed once, from its upper entry (j >= i, a suffix
// of the sorted row i), and written to both CSR entries (the lower one
// through mirror).  A warp takes an equal run of the tile's upper entries, 32
// at a time: each lane finds the row, column and mirror of one entry, and the
// result is stored by that lane; the dot products go four entries at a time,
// kEdgeLanes lanes each, lane c reading the 4-value chunks c, c + kEdgeLanes of
// the four node-major rows as whole 128-byte lines, two such steps in flight,
// and a shuffle tree sums the partials.  Entries of one row meet in one load
// instruction, so P_i and U_i cost little.  Latency bounds it (L2 at a quarter
// of its throughput): 64 graphs of 1e5 nodes, 8e5 edges each, at m = 30 took
// 3.62 ms with one dependent chain (row, column, rows, stores) per edge and
// group, 3.98 ms with P_i and U_i kept in registers per group (few warps, groups
// of a warp in rows of different lengths), 2.44 ms now.  Arithmetic in T (FP32
// in CB_FP32 mode): FP64 instructions are scarce on GB300 and would bound this
// kernel.
constexpr uint32_t kEdgeLanes = 8;
template <typename T, int NC>  // NC: chunks of a lane (rows of up to 32 NC values)
__global__ void __launch_bounds__(256) bw_edge_kernel(const T *P, const T *U, uint32_t mpad,
                                                      const InstDesc *inst,
                                                      const uint32_t *tile_inst,
                                                      const uint2 *tile_rows,
                                                      const uint32_t *row_ptr, const uint32_t *col,
                                                      const uint32_t *mirror,
                                                      const double *theta_in, float *grad) {
  __shared__ uint32_t s_rp[kTileRows + 1];
  __shared__ uint32_t s_first[kTileRows];   // first upper entry of each row
  __shared__ uint32_t s_up[kTileRows + 1];  // prefix of upper-entry counts
  const uint32_t t = blockIdx.x;
  const uint32_t r = tile_inst[t];
  const InstDesc I = inst[r];
  const uint32_t *rp = row_ptr + I.rp_base;
  const uint32_t *cl = col + I.edge_base;
  const uint2 tr = tile_rows[t];
  const uint32_t row0 = tr.x;
  const uint32_t nrows = tr.y - tr.x;
  for (uint32_t q = threadIdx.x; q <= nrows; q += blockDim.x) s_rp[q] = rp[row0 + q];
  __syncthreads();
  for (uint32_t lr = threadIdx.x; lr < nrows; lr += blockDim.x) {
    uint32_t a = s_rp[lr], b = s_rp[lr + 1];
    const uint32_t row = row0 + lr;
    while (a < b) {
      const uint32_t mid = (a + b) >> 1;
      if (__ldg(cl + mid) < row) a = mid + 1; else b = mid;
    }
    s_first[lr] = a;
  }
  __syncthreads();
  if (threadIdx.x < 32) {  // warp 0: prefix over up to 32 x 8 rows
    constexpr uint32_t kPer = kTileRows / 32;
    const uint32_t lane = threadIdx.x, base = lane * kPer;
    uint32_t c[kPer], sum = 0;
#pragma unroll
    for (uint32_t q = 0; q < kPer; ++q) {
      const uint32_t lr = base + q;
      c[q] = lr < nrows ? s_rp[lr + 1] - s_first[lr] : 0u;
      sum += c[q];
    }
    uint32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
      if ((int)lane >= o) incl += y;
    }
    uint32_t run = incl - sum;
#pragma unroll
    for (uint32_t q = 0; q < kPer; ++q) {
      if (base + q <= nrows) s_up[base + q] = run;
      run += c[q];
    }
    if (lane == 31 && nrows == kTileRows) s_up[kTileRows] = run;
  }
  __syncthreads();
  const uint32_t nup = s_up[nrows];
  const bool active = theta_in[r] > -1e307;
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t c0 = lane % kEdgeLanes, grp = lane / kEdgeLanes;
  constexpr uint32_t kStep = 32 / kEdgeLanes;  // entries of a step
  constexpr uint32_t kFly = NC == 1 && sizeof(T) == 4 ? 2 : 1;  // steps in flight
  const uint32_t u1 = (uint32_t)((uint64_t)nup * (warp + 1) / 8);
  for (uint32_t ub = (uint32_t)((uint64_t)nup * warp / 8); ub < u1; ub += 32) {
    const uint32_t u = ub + lane;
    uint32_t row = row0, j = row0, e = 0, mi = 0;
    if (u < u1) {
      uint32_t lo = 0, hi = nrows;  // s_up[lo] <= u < s_up[hi]
      while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (s_up[mid] <= u) lo = mid; else hi = mid;
      }
      e = s_first[lo] + (u - s_up[lo]);
      row = row0 + lo;
      j = __ldg(cl + e);
      mi = __ldg(mirror + I.edge_base + e);
      if (!CB_DCHECK(j < I.n, kDbgAdjointCol, j)) j = row;
    }
    T res = T(0);
    const uint32_t cnt = min(32u, u1 - ub);
    for (uint32_t k0 = 0; k0 * kStep < cnt; k0 += kFly) {  // uniform over the warp
      Quad<T> x[kFly][NC][4];
#pragma unroll
      for (uint32_t f = 0; f < kFly; ++f) {
        const uint32_t src = (k0 + f) * kStep + grp;  // lanes past the run: row0 with itself
        const uint64_t oi = (I.node_base + __shfl_sync(0xffffffffu, row, src)) * (uint64_t)mpad;
        const uint64_t oj = (I.node_base + __shfl_sync(0xffffffffu, j, src)) * (uint64_t)mpad;
#pragma unroll
        for (int q = 0; q < NC; ++q) {
          const uint32_t c = 4 * (c0 + q * kEdgeLanes);
          if (c < mpad) {
            x[f][q][0] = ld_quad(P + oi + c);
            x[f][q][1] = ld_quad(U + oj + c);
            x[f][q][2] = ld_quad(P + oj + c);
            x[f][q][3] = ld_quad(U + oi + c);
          } else {
            x[f][q][0] = x[f][q][1] = x[f][q][2] = x[f][q][3] = Quad<T>{};
          }
        }
      }
#pragma unroll
      for (uint32_t f = 0; f < kFly; ++f) {
        T g = T(0);
#pragma unroll
        for (int q = 0; q < NC; ++q) g += dot4(x[f][q][0], x[f][q][1]) + dot4(x[f][q][2], x[f][q][3]);
#pragma unroll
        for (uint32_t off = kEdgeLanes / 2; off > 0; off >>= 1) g += __shfl_xor_sync(0xffffffffu, g, off, kEdgeLanes);
        const T mine = __shfl_sync(0xffffffffu, g, (lane % kStep) * kEdgeLanes);
        if (lane / kStep == k0 + f) res = mine;
      }
    }
    if (u < u1) {
      const float v = active ? (float)res : 0.f;
      grad[I.edge_base + e] = v;
      grad[I.edge_base + mi] = v;
    }
  }
}

template <typename T>
static int backward_t(cb_graph *h, uint32_t m, const uint32_t *idx, uint32_t k, float *grad,
                      double *log_scale, cudaStream_t s) {
  BackWork &B = h->bw;
  const uint32_t N = h->n_inst;
  prefer_shared(bw_tridiag_kernel);
  prefer_shared(bw_node_kernel<T>);
  prefer_shared(bw_edge_kernel<T, 1>);
  prefer_shared(bw_edge_kernel<T, 2>);
  const int tok = prof_begin(CB_K_BACKWARD, s);
  const size_t shm_tri = 2 * sizeof(contour::Solve);
  cudaFuncSetAttribute(bw_tridiag_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm_tri);
  bw_tridiag_kernel<<<N, 64, shm_tri, s>>>(h->ws.sc, h->ws2.sc, h->d_inst, B.K, m, B.theta, B.cnt,
                                           contour::nodes(), sizeof(T) == 8);
  const size_t shm = (size_t)(m * m + 4 * m * 65) * sizeof(T);
  auto nk = bw_node_kernel<T>;
  if (shm > 48 * 1024) cudaFuncSetAttribute(nk, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm);
  nk<<<h->total_fin, 128, shm, s>>>((const T *)h->ws.V, (const T *)h->ws2.V, h->ws.vec_stride,
                                    h->ws.sc, h->ws2.sc, h->d_inst, h->d_fin_inst, N, B.K, m,
                                    B.theta, B.mpad, (T *)B.P, (T *)B.U, log_scale);
  auto ek = B.mpad <= 4 * kEdgeLanes ? bw_edge_kernel<T, 1> : bw_edge_kernel<T, 2>;
  ek<<<h->total_tiles, 256, 0, s>>>((const T *)B.P, (const T *)B.U, B.mpad, h->d_inst, h->d_tile_inst,
                                    h->d_tile_rows, h->row_ptr, h->col, h->d_mirror, B.theta, grad);
  prof_end(tok, s);
  (void)idx;
  (void)k;
  return cuda_error(cudaGetLastError(), "adjoint launch");
}

CB_DEBUG_READER(adjoint)

}  // namespace cb

using namespace cb;

CB_API int cb_scores_backward(cb_graph *h, uint32_t m, int prec, const uint32_t *topk_idx,
                              uint32_t k, float *grad, double *log_scale, void *stream) {
  NvtxRange nvtx_range("cb_scores_backward");
  if (!h || !topk_idx || !grad || !log_scale)
    return set_error(CB_ERR_ARG, "cb_scores_backward: null argument");
  if (m < 1 || m > kMaxAdjM)
    return set_error(CB_ERR_ARG, "cb_scores_backward: need 1 <= m <= 64");
  if (k < 1 || k > CB_MAX_TOPK)
    return set_error(CB_ERR_ARG, "cb_scores_backward: need 1 <= k <= CB_MAX_TOPK");
  const bool reorth = split_prec(prec);
  if (prec != CB_FP32 && prec != CB_FP64)
    return set_error(CB_ERR_ARG, "cb_scores_backward: bad precision");
  h->reorth = reorth;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  int rc = ensure_workspace(h, h->ws, m, prec, s);
  if (rc == CB_OK) rc = ensure_workspace(h, h->ws2, m, prec, s);
  if (rc == CB_OK) rc = ensure_backwork(h, m, prec, s);
  if (rc == CB_OK && !h->d_mirror) {  // once per handle: the position of each entry's mirror
    cudaError_t e = dev_alloc_n(&h->d_mirror, std::max<uint64_t>(h->total_nnz, 1));
    if (e == cudaSuccess && h->total_tiles) {
      bw_mirror_kernel<<<h->total_tiles, 256, 0, s>>>(h->d_inst, h->d_tile_inst, h->d_tile_rows,
                                                      h->row_ptr, h->col, h->d_mirror);
      e = cudaGetLastError();
    }
    if (e != cudaSuccess) {
      dev_free(h->d_mirror);
      h->d_mirror = nullptr;
      rc = cuda_error(e, "adjoint: mirror index");
    }
  }
  // the basis from 1 is the forward pass's when an ensemble pass at this m
  // and precision ran last on the handle (same stream order assumed)
  const bool reuse = rc == CB_OK && h->basis_m == m && h->basis_prec == prec &&
                     h->basis_reorth == reorth && h->basis_gen == h->ws.gen;
  if (rc == CB_OK && !reuse) {
    h->basis_m = 0;
    rc = lanczos_run(h, h->ws, 0, h->n_inst, m, prec, s);
    if (rc == CB_OK) {
      h->basis_m = m;
      h->basis_prec = prec;
      h->basis_reorth = reorth;
      h->basis_gen = h->ws.gen;
    }
  }
  if (rc == CB_OK) rc = lanczos_run(h, h->ws2, 0, h->n_inst, m, prec, s, topk_idx, k);
  if (rc == CB_OK)
    rc = prec == CB_FP64 ? backward_t<double>(h, m, topk_idx, k, grad, log_scale, s)
                         : backward_t<float>(h, m, topk_idx, k, grad, log_scale, s);
  return rc;
}

namespace cb {
namespace {

// loss = sum over q of S[nodes[q]] for the nodes inside [0, n), FP64: lane l
// sums q = l, l + 32, ... in order, then a fixed shuffle tree (deterministic).
__global__ void __launch_bounds__(32) score_sum_kernel(const double *S, uint32_t n,
                                                       const uint32_t *nodes, uint32_t k,
                                                       double *out) {
  double acc = 0.0;
  for (uint32_t q = threadIdx.x; q < k; q += 32) {
    const uint32_t i = nodes[q];
    if (i < n) acc += S[i];
  }
  acc = warp_sum_d(acc);
  if (threadIdx.x == 0) *out = acc;
}

// grad *= exp(ls_grad - ls_ref) * (grad_out ? *grad_out : 1), the factor
// formed once in FP64 and applied in FP32.
__global__ void __launch_bounds__(256) grad_rescale_kernel(float *g, uint64_t n,
                                                           const double *ls_grad,
                                                           const double *ls_ref,
                                                           const double *grad_out) {
  const double f64 = exp(*ls_grad - *ls_ref) * (grad_out ? *grad_out : 1.0);
  const float f = (float)f64;
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n;
       i += (uint64_t)gridDim.x * blockDim.x)
    g[i] *= f;
}

__global__ void scale_grad_kernel(float *g, uint64_t n, const double *ls_group,
                                  const double *ls_all) {
  const float f = (float)exp(*ls_group - *ls_all);
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n;
       i += (uint64_t)gridDim.x * blockDim.x)
    g[i] *= f;
}

__global__ void max_shift_kernel(const double *ls, uint32_t n, double *out) {
  if (threadIdx.x == 0) {
    double t = ls[0];
    for (uint32_t q = 1; q < n; ++q) t = fmax(t, ls[q]);
    *out = t;
  }
}

}  // namespace
}  // namespace cb

// Working set of the adjoint for realisation r: two (m + 1)-vector bases and
// the node-major P and U, plus the copy of its graph and format in a group
// handle (about 12 bytes per CSR entry).
static uint64_t adjoint_bytes(const cb::InstDesc &I, uint64_t nnz, uint32_t m, int prec) {
  const uint64_t esz = prec == CB_FP64 ? 8 : 4;
  const uint64_t npad = (I.n + cb::kNodeAlign - 1) / cb::kNodeAlign * cb::kNodeAlign;
  const uint64_t mpad = (m + 3) / 4 * 4;
  return esz * npad * (2 * (uint64_t)(m + 1) + 2 * mpad) + 12 * nnz + 8ull * I.n;
}

CB_API int cb_scores_backward_budget(cb_graph *h, uint32_t m, int prec, const uint32_t *topk_idx,
                                     uint32_t k, float *grad, double *log_scale,
                                     size_t mem_budget, void *stream) {
  NvtxRange nvtx_range("cb_scores_backward_budget");
  if (!h || !topk_idx || !grad || !log_scale)
    return set_error(CB_ERR_ARG, "cb_scores_backward_budget: null argument");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const uint32_t N = h->n_inst;
  std::vector<uint64_t> nnz(N), need(N);
  uint64_t total = 0;
  for (uint32_t r = 0; r < N; ++r) {
    nnz[r] = (r + 1 < N ? h->inst[r + 1].edge_base : h->total_nnz) - h->inst[r].edge_base;
    need[r] = adjoint_bytes(h->inst[r], nnz[r], m, prec & ~CB_REORTH);
    total += need[r];
  }
  if (total <= mem_budget || N == 1)
    return cb_scores_backward(h, m, prec, topk_idx, k, grad, log_scale, stream);
  // groups of consecutive realisations whose working set fits (at least one each)
  std::vector<uint32_t> starts;
  uint64_t acc = 0;
  for (uint32_t r = 0; r < N; ++r) {
    if (starts.empty() || acc + need[r] > mem_budget) {
      starts.push_back(r);
      acc = 0;
    }
    acc += need[r];
  }
  starts.push_back(N);
  const uint32_t G = (uint32_t)starts.size() - 1;
  double *d_ls = nullptr;  // per-group shift, then the common one
  cudaError_t e = dev_alloc_n(&d_ls, G + 1);
  if (e != cudaSuccess) return cuda_error(e, "cb_scores_backward_budget: allocate");
  int rc = CB_OK;
  for (uint32_t g = 0; g < G && rc == CB_OK; ++g) {
    const uint32_t r0 = starts[g], r1 = starts[g + 1];
    std::vector<uint32_t> vn(r1 - r0);
    std::vector<const uint32_t *> vrp(r1 - r0), vcol(r1 - r0);
    for (uint32_t r = r0; r < r1; ++r) {
      vn[r - r0] = h->inst[r].n;
      vrp[r - r0] = h->row_ptr + h->inst[r].rp_base;
      vcol[r - r0] = h->col + h->inst[r].edge_base;
    }
    cb_graph *v = nullptr;
    rc = cb_graph_upload(r1 - r0, vn.data(), nnz.data() + r0, vrp.data(), vcol.data(),
                         CB_DEVICE_PTRS, stream, &v);
    if (rc != CB_OK) break;
    v->plan_of = h;
    v->plan_r0 = r0;
    rc = cb_scores_backward(v, m, prec, topk_idx, k, grad + h->inst[r0].edge_base, d_ls + g, stream);
    if (rc == CB_OK) rc = cuda_error(cudaStreamSynchronize(s), "cb_scores_backward_budget");
    const int rf = cb_graph_free(v);
    if (rc == CB_OK) rc = rf;
  }
  if (rc == CB_OK) {
    max_shift_kernel<<<1, 32, 0, s>>>(d_ls, G, d_ls + G);
    for (uint32_t g = 0; g < G; ++g) {
      const uint64_t e0 = h->inst[starts[g]].edge_base;
      const uint64_t e1 = starts[g + 1] < N ? h->inst[starts[g + 1]].edge_base : h->total_nnz;
      if (e1 > e0)
        scale_grad_kernel<<<(uint32_t)std::min<uint64_t>((e1 - e0 + 255) / 256, 152 * 8), 256, 0, s>>>(
            grad + e0, e1 - e0, d_ls + g, d_ls + G);
    }
    e = cudaMemcpyAsync(log_scale, d_ls + G, 8, cudaMemcpyDeviceToDevice, s);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    rc = cuda_error(e, "cb_scores_backward_budget: combine");
  }
  dev_free(d_ls);
  return rc;
}

CB_API int cb_score_sum(const double *S, uint32_t n, const uint32_t *nodes, uint32_t k,
                        double *loss, void *stream) {
  NvtxRange nvtx_range("cb_score_sum");
  if (!S || !nodes || !loss) return set_error(CB_ERR_ARG, "cb_score_sum: null argument");
  if (k < 1 || k > CB_MAX_TOPK)
    return set_error(CB_ERR_ARG, "cb_score_sum: need 1 <= k <= CB_MAX_TOPK");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  score_sum_kernel<<<1, 32, 0, s>>>(S, n, nodes, k, loss);
  return cuda_error(cudaGetLastError(), "cb_score_sum");
}

CB_API int cb_grad_rescale(float *grad, uint64_t count, const double *log_scale_grad,
                           const double *log_scale_ref, const double *grad_out, void *stream) {
  NvtxRange nvtx_range("cb_grad_rescale");
  if (!grad || !log_scale_grad || !log_scale_ref)
    return set_error(CB_ERR_ARG, "cb_grad_rescale: null argument");
  if (count == 0) return CB_OK;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const uint64_t blocks = std::min<uint64_t>((count + 255) / 256, 152ull * 8);
  grad_rescale_kernel<<<(uint32_t)blocks, 256, 0, s>>>(grad, count, log_scale_grad, log_scale_ref,
                                                       grad_out);
  return cuda_error(cudaGetLastError(), "cb_grad_rescale");
}
