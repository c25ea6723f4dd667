// Batched Lanczos recurrence for e^A 1 on pattern-only CSR (sm_103a).
//
// The paper evaluates the total communicability e^A 1 (eq. 4) with a Krylov
// method ("Identification algorithm").  This file runs the m-step Lanczos
// recurrence that builds the Krylov basis of K_m(A, 1) and the tridiagonal
// coefficients, for every realisation of a handle at once (eq. 5 sums
// independent realisations, so they advance in lock step: one launch per
// phase covers all of them).
//
// Basis storage.  Vector j of realisation r is kept unnormalised as W_j with
// an FP64 scale, v_j = scale_j * W_j, in one array of (m+1) vectors; the
// realisations' node ranges are concatenated with kNodeAlign padding.
// W_0 = 1, scale_0 = 1/sqrt(n).
//
// Step j (0-based), three kernels:
//   spmv:     u = scale_j (A W_j) - beta_{j-1} scale_{j-1} W_{j-1}
//             alpha_j = scale_j (W_j . u);   W_{j+1} <- u
//   finalize: w = W_{j+1} - alpha_j scale_j W_j;  W_{j+1} <- w, and the
//             per-tile partials of ||w||^2
//   beta:     beta_j = ||w||; scale_{j+1} = 1/beta_j, or stop at an exact
//             breakdown beta_j <= tau (|alpha_j| + beta_{j-1}).
// Deterministic reductions: the SpMV's alpha uses the last CTA to arrive
// (cb_reduce.cuh); beta sums the finalize partials in the same groups and
// order in its own kernel, so finalize CTAs retire without waiting.
// No reorthogonalisation: the Lanczos approximation of f(A)b stays accurate
// in finite precision after orthogonality is lost (Greenbaum; Musco, Musco &
// Sidford 2018), which the parity tests check against the FP64 oracle that
// reorthogonalises fully.
//
// SpMV work split.  A CTA owns a tile of consecutive rows (at most kTileRows,
// closed before kTileNnz entries, so hub regions get short tiles).  Rows with at
// most 8*G entries are summed by G-lane groups; longer rows up to kLongDeg
// by one warp each; rows up to kHeavyDeg by the whole CTA; rows above
// kHeavyDeg are cut into kChunk-edge chunks, one CTA per chunk, and the last
// chunk to finish completes the row.  Column indices are streamed with an
// evict-first hint; the gathered vector stays cache-resident.
#include <algorithm>

#include "cb_internal.cuh"
#include "cb_reduce.cuh"
#include "cb_step.cuh"
#include "cb_team.cuh"

namespace cb {


template <typename T>
__global__ void __launch_bounds__(kThreads) init_vec_kernel(T *w0, uint64_t n8, T fill) {
  // W_0 = fill (1 for the start vector 1, 0 before an indicator is set), 8
  // nodes at a time over the realisations' range, the alignment gaps between
  // them (which nothing reads) included: a loop over the realisations, its
  // grid sized for one, took 155 us for 256 of them, 58 now.
  T v[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) v[q] = fill;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n8;
       i += (uint64_t)gridDim.x * blockDim.x)
    Vec8<T>::store(w0 + 8 * i, v);
}

// W_0[idx[q]] = 1 for the start indices inside each realisation's range
// (per_inst: realisation r0 + q starts from the single node idx[q]).
template <typename T>
__global__ void __launch_bounds__(kThreads) init_indicator_kernel(LArgs a, uint32_t r0,
                                                                  const uint32_t *idx, uint32_t k,
                                                                  bool per_inst) {
  const uint32_t r = r0 + blockIdx.x;
  const InstDesc I = a.inst[r];
  T *w0 = reinterpret_cast<T *>(a.V) + I.node_base;
  if (per_inst) {
    if (threadIdx.x == 0 && idx[blockIdx.x] < I.n) w0[idx[blockIdx.x]] = T(1);
    return;
  }
  for (uint32_t q = threadIdx.x; q < k; q += blockDim.x) {
    const uint32_t i = idx[q];
    if (i < I.n) w0[i] = T(1);
  }
}

// rscale (restart): W_0 already holds the start vector and scale_0 =
// rscale[r]; 0 marks a realisation that has nothing left to do.
__global__ void __launch_bounds__(kThreads) init_scalars_kernel(LArgs a, uint32_t r0, uint32_t r1,
                                                                uint32_t m, const uint32_t *idx,
                                                                uint32_t k, bool per_inst,
                                                                const double *rscale,
                                                                uint32_t *tctr) {
  const uint32_t ms = a.sc.ms;
  // the team kernel's barrier counters
  if (blockIdx.x == 0)
    for (uint32_t q = threadIdx.x; q < kMaxTeams; q += blockDim.x) tctr[q * kCtrStride] = 0u;
  const uint64_t total = (uint64_t)(r1 - r0) * ms;
  for (uint64_t q = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; q < total;
       q += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t r = r0 + (uint32_t)(q / ms), jj = (uint32_t)(q % ms);
    const uint64_t o = (uint64_t)r * ms + jj;
    a.sc.alpha[o] = 0.0;
    a.sc.beta[o] = 0.0;
    a.sc.gamma[o] = 0.0;
    uint32_t cnt = a.inst[r].n;  // ||start||^2
    if (idx && jj == 0) {
      cnt = 0;
      if (per_inst)
        cnt = idx[r - r0] < a.inst[r].n ? 1u : 0u;
      else
        for (uint32_t q = 0; q < k; ++q) cnt += (idx[q] < a.inst[r].n);
    }
    double s0 = cnt ? 1.0 / sqrt((double)cnt) : 0.0;
    if (rscale) {
      s0 = rscale[r];
      cnt = s0 > 0.0 ? 1u : 0u;
    }
    a.sc.scale[o] = jj == 0 ? s0 : 0.0;
    if (jj == 0) {
      a.sc.meff[r] = cnt ? m : 0u;  // no start vector: nothing to do
      a.sc.status[r] = CB_OK;
      a.sc.theta[r] = 0.0;
    }
  }
}


// Sums of B values per lane over groups of G lanes (B <= G, powers of two), in
// the order of group_sum's tree: at each of the first steps a lane sends half
// of its values and keeps the sums of the other half, B - 1 additions for
// B values where B separate sums take B log2(B).  Lane l of a group gets the sum
// of value l / (G / B).
template <int B, int G>
__device__ __forceinline__ double batch_sum(double (&v)[B]) {
  const int l = threadIdx.x % G;
  int o = G / 2;
#pragma unroll
  for (int half = B / 2; half >= 1; half >>= 1, o >>= 1) {
    const bool up = (l & o) != 0;
#pragma unroll
    for (int q = 0; q < half; ++q) {
      const double keep = up ? v[q + half] : v[q], send = up ? v[q] : v[q + half];
      v[q] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  for (; o >= 1; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
  return v[0];
}

// One Lanczos SpMV step over a range of realisations.  FP64 is bound by the
// FP64 pipe, 65 cycles of a sub-core per warp instruction however many lanes
// are active: there the sums of several rows (kSide short ones per group, kSideLong
// longer ones per warp or CTA) are formed side by side (batch_sum), a row's
// result by a lane of its own, and a first entry is not added to 0; the
// sums' orders, alpha's included, are those of one row at a time.
// How many rows, and CTAs per SM, follows the group width, because more of one
// leaves registers for fewer of the other, and the gathers in flight count as much:
// with 8 short and 4 longer rows and five CTAs at every width, widths 1, 8, 16
// and 32 spilled 260 to 340 bytes a thread.  m = 16, one row at a time / that /
// now, ms: width 1, 8 graphs of 1.5e5 nodes, degree 2.5, 1.28 / 1.32 / 1.22; width 2,
// degree 5, 1.68 / 1.54 / 1.43; width 8, degree 60, 9.04 / 10.8 / 8.89, degree 40,
// 5.09 / 5.46 / 4.58; width 16, 6 of 1e5, degree 120, 7.38 / 11.9 / 7.20; width 32,
// 6 of 3e4, degree 300, 5.38 / 5.65 / 4.45.  Width 4 has both (SIDE): few entries a
// row gain from rows side by side, BA(1e5, 5) 0.76 / 0.65 / 0.63 (0.70 as the other
// widths); from degree kSideDeg on from the sixth CTA, degree 20, one graph of
// 2.3e5 nodes, m = 10, 0.53 / 0.56 / 0.49 (0.56 with rows side by side).  FP32: six
// CTAs, one row at a time (five: up to 20% slower where six hold all tiles at once).
constexpr uint32_t kSideDeg = 16;
template <typename T, int G, bool SIDE>
struct SpmvShape {
  static constexpr int kCtas = SIDE ? 5 : 6;
  static constexpr int kSide = SIDE ? 4 : G < 2 ? G : 2, kSideLong = SIDE ? 2 : 1;
};
// Blocks [0, n_chunks) are heavy-row chunks starting at chunk_off; blocks
// [n_chunks, ...) are normal tiles starting at tile_off.
template <typename T, int G, bool SIDE>
__global__ void __launch_bounds__(kThreads, SpmvShape<T, G, SIDE>::kCtas)
    spmv_kernel(LArgs a, uint32_t j, uint32_t chunk_off, uint32_t n_chunks, uint32_t tile_off) {
  __shared__ double s_red[32];
  __shared__ uint32_t s_rp[kTileRows + 1];
  __shared__ uint16_t s_med[kTileRows], s_long[kTileRows];
  __shared__ uint32_t s_wcnt[kThreads / 32][2];
  __shared__ uint32_t s_nmed, s_nlong;
  __shared__ T s_rowsum[32];

  const uint32_t ms = a.sc.ms;
  static_assert(kTileRows == kThreads, "one tile row per thread in the row classification");
  const bool is_chunk = blockIdx.x < n_chunks;
  uint32_t r;
  uint32_t hid = 0, cidx = 0, tile = 0;
  if (is_chunk) {
    cidx = chunk_off + blockIdx.x;
    hid = a.chunk_heavy[cidx];
    r = a.heavy[hid].inst;
  } else {
    tile = tile_off + (blockIdx.x - n_chunks);
    r = a.tile_inst[tile];
    // the tile's row offsets, staged once (coalesced); fixed by the upload
    const uint2 tr = a.tile_rows[tile];
    const uint32_t *rp = a.row_ptr + a.inst[r].rp_base + tr.x;
    for (uint32_t q = threadIdx.x; q <= tr.y - tr.x; q += kThreads) s_rp[q] = rp[q];
  }
  dep_wait();
  dep_trigger();
  if (j >= a.sc.meff[r]) return;  // realisation stopped (uniform per CTA)
  if (a.skip_blocked && a.inst[r].blocked) return;  // the column-blocked kernel owns it
  if (a.skip_pb && a.inst[r].pb) return;            // the two-phase kernels own it

  const InstDesc &I = a.inst[r];
  const uint32_t *col = a.col + I.edge_base;
  T *Vb = reinterpret_cast<T *>(a.V);
  const T *x = Vb + (uint64_t)j * a.vs + I.node_base;
  const bool has_prev = j > 0;
  const T *xp = has_prev ? Vb + (uint64_t)(j - 1) * a.vs + I.node_base : x;
  T *out = Vb + (uint64_t)(j + 1) * a.vs + I.node_base;
  const T sj = (T)a.sc.scale[r * ms + j];
  const T bp = has_prev ? (T)(a.sc.beta[r * ms + j - 1] * a.sc.scale[r * ms + j - 1]) : T(0);

  if (is_chunk) {
    heavy_chunk<T>(a, j, cidx, hid, r, I.spmv, I.n_tiles + (hid - I.heavy_base));
    return;
  }

  // ---- normal tile ----
  const uint2 tr = a.tile_rows[tile];
  const uint32_t row0 = tr.x;
  const uint32_t nrows = tr.y - tr.x;  // <= kTileRows
  __syncthreads();  // s_rp

  T acc = T(0);
  const uint32_t lane_g = threadIdx.x % G;
  const uint32_t grp = threadIdx.x / G;
  constexpr uint32_t kGroups = kThreads / G;
  constexpr uint32_t kShort = 8 * G;
  // Short rows: G lanes per row.  The trip count depends only on the tile,
  // so every lane of a warp runs every iteration and the full-mask group
  // shuffles are always converged.
  if constexpr (sizeof(T) == 8) {
    constexpr int B = SpmvShape<T, G, SIDE>::kSide, kDup = G / B;
    for (uint32_t it0 = 0; it0 < (uint32_t)G && it0 * kGroups < nrows; it0 += B) {
      // this lane's row of the batch, its operands loaded before the sums
      const uint32_t mine = (it0 + lane_g / kDup) * kGroups + grp;
      const bool short_row = mine < nrows && s_rp[mine + 1] - s_rp[mine] <= kShort;
      const uint32_t shorts = __ballot_sync(0xffffffffu, short_row);
      if (!shorts) continue;
      double xr = 0.0, xpr = 0.0;
      if (short_row) {
        xr = x[row0 + mine];
        if (has_prev) xpr = xp[row0 + mine];
      }
      double v[B];
#pragma unroll
      for (int q = 0; q < B; ++q) {
        const uint32_t lr = (it0 + q) * kGroups + grp;
        uint32_t e0 = 0, len = 0;
        if (lr < nrows) {
          e0 = s_rp[lr];
          len = s_rp[lr + 1] - e0;
        }
        if (len > kShort) len = 0;
        double g[kShort / G];
#pragma unroll
        for (uint32_t i = 0; i < kShort / G; ++i) {
          const uint32_t t = lane_g + i * G;
          g[i] = 0.0;
          if (t < len) {
            const uint32_t c = ld_stream(col + e0 + t);
            if (CB_DCHECK(c < I.n, kDbgCsrCol, c)) g[i] = ld_vec(x + c);
          }
        }
        const uint32_t most = __reduce_max_sync(0xffffffffu, len);
        v[q] = g[0];
#pragma unroll
        for (uint32_t i = 1; i < kShort / G; ++i)
          if (i * G < most) v[q] += g[i];  // adding a 0 past a row's end changes no bit
      }
      const double sum = batch_sum<B, G>(v);
      double u = sj * sum;
      if (has_prev) u -= bp * xpr;
      if (short_row && lane_g % kDup == 0) out[row0 + mine] = u;
      // the group's first lane takes the rows' alpha terms in row order
#pragma unroll
      for (int q = 0; q < B; ++q) {
        const int src = (threadIdx.x & 31 & ~(G - 1)) + q * kDup;
        const double xq = __shfl_sync(0xffffffffu, xr, src), uq = __shfl_sync(0xffffffffu, u, src);
        if (lane_g == 0 && (shorts >> src & 1u)) acc += xq * uq;
      }
    }
  } else {
    for (uint32_t base = 0; base < nrows; base += kGroups) {
      const uint32_t lr = base + grp;
      const bool valid = lr < nrows;
      uint32_t e0 = 0, e1 = 0;
      if (valid) { e0 = s_rp[lr]; e1 = s_rp[lr + 1]; }
      const bool is_short = valid && (e1 - e0) <= kShort;
      T s = T(0);
      if (is_short) {
        // at most kShort / G entries per lane: a fixed, predicated trip count
        // puts all of the lane's index loads, then all of its gathers, in
        // flight at once (a counted loop of 2-4 trips runs its remainder
        // path one load pair at a time); the summation order is unchanged
        const uint32_t len = e1 - e0;
#pragma unroll
        for (uint32_t i = 0; i < kShort / G; ++i) {
          const uint32_t t = lane_g + i * G;
          if (t < len) {
            const uint32_t c = ld_stream(col + e0 + t);
            if (CB_DCHECK(c < I.n, kDbgCsrCol, c)) s += ld_vec(x + c);
          }
        }
      }
      s = group_sum<G, T>(s);
      if (is_short && lane_g == 0) acc += row_epilogue<T>(s, row0 + lr, x, xp, out, sj, bp, has_prev);
    }
  }

  // Medium (kShort < deg <= kLongDeg) and long (kLongDeg < deg <= kHeavyDeg)
  // rows: lists in row order, built with one ballot per warp (thread q
  // classifies row q of the tile), so the processing order is fixed.
  {
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t lr = threadIdx.x;  // kTileRows == kThreads
    uint32_t deg = 0;
    if (lr < nrows) deg = s_rp[lr + 1] - s_rp[lr];
    const bool med = deg > kShort && deg <= kLongDeg;
    const bool lng = deg > kLongDeg && deg <= kHeavyDeg;
    const uint32_t bm = __ballot_sync(0xffffffffu, med), bl = __ballot_sync(0xffffffffu, lng);
    if (lane == 0) { s_wcnt[warp][0] = __popc(bm); s_wcnt[warp][1] = __popc(bl); }
    __syncthreads();
    uint32_t om = 0, ol = 0, nm = 0, nl = 0;
    for (uint32_t w = 0; w < kThreads / 32; ++w) {
      if (w < warp) { om += s_wcnt[w][0]; ol += s_wcnt[w][1]; }
      nm += s_wcnt[w][0];
      nl += s_wcnt[w][1];
    }
    const uint32_t below = (1u << lane) - 1u;
    if (med) s_med[om + __popc(bm & below)] = lr;
    if (lng) s_long[ol + __popc(bl & below)] = lr;
    if (threadIdx.x == 0) { s_nmed = nm; s_nlong = nl; }
  }
  __syncthreads();

  // x over the entries e, e + step, ... < e1 in order (FP32): four gathers in
  // flight, also in the last round (a counted loop runs its remainder one by
  // one): 31.4 -> 25.6 us a step on BA(1e5, 5).
  auto run_sum = [&](uint32_t e, uint32_t e1, uint32_t step) -> T {
    T s = T(0);
    for (; e < e1; e += 4 * step) {
      T v[4];
#pragma unroll
      for (uint32_t u = 0; u < 4; ++u) {
        v[u] = T(0);  // adding the 0 past the end changes no bit
        if (e + u * step < e1) {
          const uint32_t c = ld_stream(col + e + u * step);
          if (CB_DCHECK(c < I.n, kDbgCsrCol, c)) v[u] = ld_vec(x + c);
        }
      }
#pragma unroll
      for (uint32_t u = 0; u < 4; ++u) s += v[u];
    }
    return s;
  };
  // u = sj * sum - bp * W_{j-1}[row], stored; the row's alpha term.  The row's
  // operands are loaded before its sum.
  auto finish_row = [&](T sum, uint32_t row, T xr, T xpr) {
    T u = sj * sum;
    if (has_prev) u -= bp * xpr;
    out[row] = u;
    acc += xr * u;
  };

  // R rows (entries e0 .. e1 of each) side by side, kU gathers of each in
  // flight, entry `first` on by `step`; a round past a row's end is skipped by
  // the whole warp, and adding a 0 past it changes no bit
  auto run_sums = [&](auto &v, const uint32_t *e0, const uint32_t *e1, uint32_t first, uint32_t step) {
    constexpr int R = sizeof(v) / sizeof(v[0]), kU = 4;
    uint32_t most = 0;
#pragma unroll
    for (int q = 0; q < R; ++q) most = max(most, e1[q] - e0[q]);
    for (uint32_t base = 0; base < most; base += kU * step) {
      double g[R][kU];
#pragma unroll
      for (int q = 0; q < R; ++q)
#pragma unroll
        for (int i = 0; i < kU; ++i) {
          const uint32_t e = e0[q] + base + i * step + first;
          g[q][i] = 0.0;
          if (e < e1[q]) {
            const uint32_t c = ld_stream(col + e);
            if (CB_DCHECK(c < I.n, kDbgCsrCol, c)) g[q][i] = ld_vec(x + c);
          }
        }
#pragma unroll
      for (int q = 0; q < R; ++q)
#pragma unroll
        for (int i = 0; i < kU; ++i)
          if (base + i == 0)
            v[q] = g[q][i];
          else if (e0[q] + base + i * step < e1[q])
            v[q] += g[q][i];
    }
  };

  if constexpr (sizeof(T) == 8) {
    // medium rows: warp w takes list entries w, w+8, ..., kR at a time
    constexpr int kR = SpmvShape<T, G, SIDE>::kSideLong;
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t nmed = s_nmed;
    for (uint32_t q0 = warp; q0 < nmed; q0 += kR * (kThreads / 32)) {
      uint32_t e0[kR], e1[kR];
      double v[kR];
#pragma unroll
      for (int q = 0; q < kR; ++q) {
        const uint32_t at = q0 + q * (kThreads / 32);
        e0[q] = e1[q] = 0;
        v[q] = 0.0;
        if (at < nmed) {
          e0[q] = s_rp[s_med[at]];
          e1[q] = s_rp[s_med[at] + 1];
        }
      }
      const uint32_t my = q0 + (lane / (32 / kR)) * (kThreads / 32);  // this lane's row
      double xr = 0.0, xpr = 0.0;
      const uint32_t row = my < nmed ? row0 + s_med[my] : row0;
      if (my < nmed) {
        xr = x[row];
        if (has_prev) xpr = xp[row];
      }
      run_sums(v, e0, e1, lane, 32);
      const double sum = batch_sum<kR, 32>(v);
      double u = sj * sum;
      if (has_prev) u -= bp * xpr;
      if (my < nmed && lane % (32 / kR) == 0) out[row] = u;
#pragma unroll
      for (int q = 0; q < kR; ++q) {
        const double xq = __shfl_sync(0xffffffffu, xr, q * (32 / kR)), uq = __shfl_sync(0xffffffffu, u, q * (32 / kR));
        if (lane == 0 && q0 + q * (kThreads / 32) < nmed) acc += xq * uq;
      }
    }
    // long rows: the whole CTA, kL rows at a time, in row order
    constexpr int kL = SpmvShape<T, G, SIDE>::kSideLong;
    __shared__ double s_sums[kL][kThreads / 32];
    const uint32_t nlong = s_nlong;
    for (uint32_t q0 = 0; q0 < nlong; q0 += kL) {
      uint32_t e0[kL], e1[kL];
      double v[kL];
#pragma unroll
      for (int q = 0; q < kL; ++q) {
        e0[q] = e1[q] = 0;
        v[q] = 0.0;
        if (q0 + q < nlong) {
          e0[q] = s_rp[s_long[q0 + q]];
          e1[q] = s_rp[s_long[q0 + q] + 1];
        }
      }
      run_sums(v, e0, e1, threadIdx.x, kThreads);
      const double sum = batch_sum<kL, 32>(v);
      if (lane % (32 / kL) == 0) s_sums[lane / (32 / kL)][warp] = sum;
      __syncthreads();
      if (warp == 0) {
        const bool on = lane < kL && q0 + lane < nlong;
        const uint32_t row = on ? row0 + s_long[q0 + lane] : row0;
        double xr = 0.0, xpr = 0.0, tot = 0.0;
        if (on) {
          xr = x[row];
          if (has_prev) xpr = xp[row];
          for (uint32_t w = 0; w < kThreads / 32; ++w) tot += s_sums[lane][w];
        }
        double u = sj * tot;
        if (has_prev) u -= bp * xpr;
        if (on) out[row] = u;
#pragma unroll
        for (int q = 0; q < kL; ++q) {
          const double xq = __shfl_sync(0xffffffffu, xr, q), uq = __shfl_sync(0xffffffffu, u, q);
          if (lane == 0 && q0 + q < nlong) acc += xq * uq;
        }
      }
      __syncthreads();
    }
  } else {
    // medium rows: warp w takes list entries w, w+8, ...
    {
      const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
      const uint32_t nmed = s_nmed;
      for (uint32_t q = warp; q < nmed; q += kThreads / 32) {
        const uint32_t lr = s_med[q], row = row0 + lr;
        T xr = T(0), xpr = T(0);
        if (lane == 0) {
          xr = x[row];
          if (has_prev) xpr = xp[row];
        }
        const T s = warp_sum<T>(run_sum(s_rp[lr] + lane, s_rp[lr + 1], 32));
        if (lane == 0) finish_row(s, row, xr, xpr);
      }
    }

    // long rows: the whole CTA per row, in row order
    const uint32_t nlong = s_nlong;
    for (uint32_t q = 0; q < nlong; ++q) {
      const uint32_t lr = s_long[q], row = row0 + lr;
      const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
      T xr = T(0), xpr = T(0);
      if (threadIdx.x == 0) {
        xr = x[row];
        if (has_prev) xpr = xp[row];
      }
      const T s = warp_sum<T>(run_sum(s_rp[lr] + threadIdx.x, s_rp[lr + 1], kThreads));
      if (lane == 0) s_rowsum[warp] = s;
      __syncthreads();
      if (threadIdx.x == 0) {
        T tot = T(0);
        for (int w = 0; w < kThreads / 32; ++w) tot += s_rowsum[w];
        finish_row(tot, row, xr, xpr);
      }
      __syncthreads();
    }
  }

  const double part = block_sum_to_double<T>(acc, s_red);
  double total;
  if (arrive_and_reduce(I.spmv, tile - I.tile_base, r, part, a.red, &total))
    finish_alpha<T>(a, r, j, total);
}

// ---------------------------------------------------------------------------
// Column-blocked SpMV step (FP32).  Same arithmetic as spmv_kernel
// (u = scale_j A W_j - beta_{j-1} scale_{j-1} W_{j-1}, alpha_j partial), but
// every gather of W_j is a shared-memory load: the CTA walks the column
// blocks of its tile, double-buffering each block of W_j into shared memory
// with one bulk copy (cp.async.bulk, completion on an mbarrier) while the
// previous block is consumed.  Thread i owns rows
// i + kBThreads k (k = 0..15) of the tile and accumulates them in shared memory;
// every row has a single writer, so the result is deterministic.
//
// Bound by the shared-memory pipe: a step of 32 elements is about 2.9
// wavefronts for the gathers (4.1 before the elements of a round were ordered
// by bank), 1.4 to read and 1.4 to write the sums (1.6), 0.85 for its share of the
// staged blocks.  175 M entries in 40 graphs: 325 us with a round's gathers
// after the previous sums, elements decoded by shifts (29 instructions a
// step, 56% of the pipe); 293 with byte offsets and the gathers of a round
// together (18); 277 with the loads two rounds ahead; 263 with the
// prologue's and epilogue's loads together (17); 242 with the rounds ordered
// by bank, 236 with the lanes dealt most and fewest in turn, 224 with the
// longest tiles first (562 tiles on 152 SMs).
// ---------------------------------------------------------------------------

// two column blocks of W_j, then kBRowsPerThread row sums per thread and
// one spare per thread (the padding elements add into it)
constexpr size_t kBSmemBytes = (2 * kBBuf + (kBRowsPerThread + 1) * kBThreads) * sizeof(float);
static_assert(kBSmemBytes + 1024 <= 227 * 1024, "column-blocked CTA shared memory");

__global__ void __launch_bounds__(kBThreads, 1) bspmv_kernel(LArgs a, uint32_t j,
                                                             uint32_t btile_off) {
  extern __shared__ float4 s_dyn4[];
  float *xs = reinterpret_cast<float *>(s_dyn4);  // two column blocks of W_j
  float *sacc = xs + 2 * kBBuf;                   // [warp][slot][lane] row sums
  __shared__ uint32_t s_long[kBTileRows / 32];    // bitmap of long rows
  __shared__ double s_red[32];
  __shared__ float s_rowsum[32];
  __shared__ __align__(8) uint64_t s_full[2];     // block of W_j landed in buffer p
  __shared__ uint32_t s_done[2];                  // warps finished with buffer p
  __shared__ uint32_t s_issued[2];                // copies issued into buffer p
  __shared__ int s_abort;
  __shared__ uint64_t s_seg[kBMaxBlocks + 1];     // stream offset of each column block's segment
  __shared__ float s_coef[2];                     // scale_j, beta_{j-1} scale_{j-1}
  __shared__ __align__(8) uint64_t s_coef_ok;     // s_coef written
  // One CTA per SM: nothing hides what a CTA does before its first and after
  // its last element (13k and 18k of 149k cycles when each load waited for
  // the one before), so the loads go out together, the static ones and the
  // first rounds of the streams before the wait for the previous kernel, and
  // the copies of W_j before it is known whether the realisation goes on.
  const uint32_t t = a.border ? a.border[blockIdx.x] : btile_off + blockIdx.x;
  const uint32_t r = a.btile_inst[t];
  const uint64_t sbase = a.bseg_base[t];
  const uint32_t lp0 = a.blong_ptr[t], lp1 = a.blong_ptr[t + 1];
  const InstDesc &I = a.inst[r];
  const uint32_t nb = I.nb, n = I.n, row0 = (t - I.btile_base) * kBTileRows;
  const uint64_t node_base = I.node_base;
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // lane b holds the warp's stream of block b: its first element and its pairs
  // of steps
  static_assert(kBMaxBlocks <= 32, "one lane per column block");
  uint64_t st = 0;
  uint32_t np = 0;
  if (lane < nb) {
    st = a.bwstart[(sbase + lane) * 32 + warp];
    np = a.bwlen[(sbase + lane) * 32 + warp] >> 1;
  }
  float *sw = sacc + warp * kBWarpSums;  // this warp's row sums: sw[32 * slot + lane]
#pragma unroll
  for (int k = 0; k <= kBRowsPerThread; ++k) sw[32 * k + lane] = 0.f;
  for (uint32_t q = tid; q < kBTileRows / 32; q += kBThreads) s_long[q] = 0u;
  if (tid == 0) {
    mbar_init(&s_full[0], 1);
    mbar_init(&s_full[1], 1);
    mbar_init(&s_coef_ok, 1);
    s_done[0] = s_done[1] = 0;
    s_issued[0] = s_issued[1] = 0;
    s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0 && lane < nb) s_seg[lane] = st;
  if (warp == 31 && lane == nb - 1) s_seg[nb] = st + 64ull * np;

  // A warp's stream of block b has T_b steps, read as T_b / 2 pairs (two
  // elements per lane per 8-byte load) in rounds of up to 4 pairs that do not
  // cross a block (an empty block is one empty round).  The loads run two
  // rounds ahead of the sums, across the ends of blocks.
  const uint32_t *fp = a.belem + __shfl_sync(0xffffffffu, st, 0) + 2 * lane;  // next round to load
  uint32_t fb = 0, frem = __shfl_sync(0xffffffffu, np, 0);  // its block, the pairs left there
  uint32_t b = 0, rem = frem;                               // the same of the round summed
  auto fetch = [&](uint2 (&e)[4]) {
    if (fb >= nb) return;
    if (frem >= 4) {
#pragma unroll
      for (int u = 0; u < 4; ++u) e[u] = __ldcs(reinterpret_cast<const uint2 *>(fp + 64 * u));
    } else {
#pragma unroll
      for (int u = 0; u < 3; ++u)
        if ((uint32_t)u < frem) e[u] = __ldcs(reinterpret_cast<const uint2 *>(fp + 64 * u));
    }
    if (frem > 4) {
      frem -= 4;
      fp += 256;
    } else if (++fb < nb) {
      fp = a.belem + __shfl_sync(0xffffffffu, st, fb) + 2 * lane;
      frem = __shfl_sync(0xffffffffu, np, fb);
    }
  };
  uint2 eA[4], eB[4], eC[4];
  fetch(eA);
  fetch(eB);

  dep_wait();
  dep_trigger();
  const uint32_t meff = a.sc.meff[r];
  const uint32_t ms = a.sc.ms;
  float *Vb = reinterpret_cast<float *>(a.V);
  const float *x = Vb + (uint64_t)j * a.vs + node_base;
  const bool has_prev = j > 0;
  const float *xp = has_prev ? Vb + (uint64_t)(j - 1) * a.vs + node_base : x;
  float *out = Vb + (uint64_t)(j + 1) * a.vs + node_base;
  // Column block b of W_j goes to buffer b & 1 by one bulk copy that
  // completes on s_full[b & 1].  No CTA-wide barrier per block: each warp
  // waits only for the block it needs, and the last warp to finish with a
  // buffer issues the copy of block b + 2 into it, so warps drift apart by up
  // to a block instead of all waiting for the slowest at every block.  After
  // the last block the tile's rows of W_{j-1} follow as block nb, for the
  // epilogue.  The edge streams of block b + 1 are prefetched into L2 when
  // block b is staged, so the warps' stream loads find them there.
  auto issue = [&](uint32_t b) {
    if (b > nb || (b == nb && !has_prev)) return;
    const float *src = b < nb ? x + (uint64_t)b * kBCol : xp + row0;
    const uint32_t len = b < nb ? min(kBCol, n - b * kBCol) : min((uint32_t)kBTileRows, n - row0);
    const uint32_t bytes = ((len + 3u) & ~3u) * 4u;  // whole 16-byte units (reads up to 3 floats of padding)
    const uint32_t p = b & 1;
    mbar_expect_tx(&s_full[p], bytes);
    if (b == 0 && t == a.stall_btile) return;  // test hook: block 0 never arrives
    bulk_g2s(xs + p * kBBuf, src, bytes, &s_full[p]);
    s_issued[p] += 1;
  };
  auto prefetch_seg = [&](uint32_t b) {
    if (b < nb && s_seg[b + 1] > s_seg[b])
      l2_prefetch(a.belem + s_seg[b], (uint32_t)(4 * (s_seg[b + 1] - s_seg[b])));
  };
  // every copy issued into a buffer has landed before the CTA ends (bounded)
  auto drain = [&]() {
    for (int p = 0; p < 2; ++p)
      if (s_issued[p]) mbar_wait(&s_full[p], (s_issued[p] - 1) & 1u);
  };
  if (tid == 0) {
    issue(0);
    issue(1);
  }
  __syncthreads();
  if (j >= meff) {
    if (tid == 0) drain();
    return;
  }
  if (tid == 0) {
    prefetch_seg(1);
    prefetch_seg(2);
  }
  if (tid == kBThreads - 1) {  // one thread: an FP64 instruction holds its sub-core for 65 cycles
    s_coef[0] = (float)a.sc.scale[r * ms + j];
    s_coef[1] = has_prev ? (float)(a.sc.beta[r * ms + j - 1] * a.sc.scale[r * ms + j - 1]) : 0.f;
    mbar_arrive(&s_coef_ok);
  }
  if (lp1 > lp0) {
    for (uint32_t q = lp0 + tid; q < lp1; q += kBThreads) {
      const uint32_t lr = a.blong_rows[q];
      atomicOr(&s_long[lr >> 5], 1u << (lr & 31));
    }
    __syncthreads();
  }

  const char *cur = reinterpret_cast<const char *>(xs);
  char *swc = reinterpret_cast<char *>(sw);
  auto gather = [&](uint32_t v) -> float {
    if (!CB_DCHECK((v >> 18) < kBWarpSums && (v & 3u) == 0, kDbgBlockedElem, v)) return 0.f;
    return *reinterpret_cast<const float *>(cur + (v & 0xffffu));
  };
  auto add = [&](uint32_t v, float g) {
    if (!CB_DCHECK((v >> 18) < kBWarpSums, kDbgBlockedElem, v)) return;
    *reinterpret_cast<float *>(swc + (v >> 16)) += g;
  };
  // One round: the gathers of all its elements, then the sums, in step order
  // (no two lanes of a step add into one row sum).  False once the tile's
  // streams are done or a copy never landed.
  bool aborted = false;
  auto round = [&](const uint2 (&e)[4]) -> bool {
    if (rem >= 4) {
      float g[8];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        g[2 * u] = gather(e[u].x);
        g[2 * u + 1] = gather(e[u].y);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        add(e[u].x, g[2 * u]);
        add(e[u].y, g[2 * u + 1]);
      }
    } else {
#pragma unroll
      for (int u = 0; u < 3; ++u)
        if ((uint32_t)u < rem) {
          const float g0 = gather(e[u].x), g1 = gather(e[u].y);
          add(e[u].x, g0);
          add(e[u].y, g1);
        }
    }
    if (rem > 4) {
      rem -= 4;
      return true;
    }
    // this warp is done with buffer b & 1; the last warp refills it
    __syncwarp();
    if (lane == 0) {
      __threadfence_block();
      if (atomicAdd(&s_done[b & 1], 1u) == kBThreads / 32 - 1) {
        s_done[b & 1] = 0;
        __threadfence_block();
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        issue(b + 2);
        prefetch_seg(b + 3);
      }
    }
    if (++b == nb) return false;
    rem = __shfl_sync(0xffffffffu, np, b);
    cur = reinterpret_cast<const char *>(xs + (b & 1) * kBBuf);
    aborted = !mbar_wait_sleep(&s_full[b & 1], (b >> 1) & 1u);  // the copy never landed: give up
    return !aborted;
  };
  aborted = !mbar_wait_sleep(&s_full[0], 0);
  if (!aborted)
    while (true) {
      fetch(eC);
      if (!round(eA)) break;
      fetch(eA);
      if (!round(eB)) break;
      fetch(eB);
      if (!round(eC)) break;
    }

  // the warp's rows: their sums are complete, nobody else adds into them.
  // Row slot k of this thread is row tid + kBThreads k of the tile.
  float xr[kBRowsPerThread];
#pragma unroll
  for (int k = 0; k < kBRowsPerThread; ++k) {
    const uint32_t row = row0 + tid + kBThreads * k;
    xr[k] = row < n ? x[row] : 0.f;
  }
  if (has_prev && !aborted) aborted = !mbar_wait_sleep(&s_full[nb & 1], (nb >> 1) & 1u);
  if (!mbar_wait_sleep(&s_coef_ok, 0)) aborted = true;
  const float sj = s_coef[0], bp = s_coef[1];
  const float *xpt = xs + (nb & 1) * kBBuf;  // W_{j-1} of the tile
  float acc = 0.f;
#pragma unroll
  for (int k = 0; k < kBRowsPerThread; ++k) {
    const uint32_t lr = tid + kBThreads * k, row = row0 + lr;
    if (row < n && !((s_long[lr >> 5] >> (lr & 31)) & 1u)) {
      float u = sj * sw[32 * k + lane];
      if (has_prev) u -= bp * xpt[lr];
      out[row] = u;
      acc += u * xr[k];
    }
  }
  if (aborted) s_abort = 1;  // read after the sum's barrier
  // long rows: whole CTA per row from the CSR, in row order
  const uint32_t *rp = a.row_ptr + I.rp_base;
  const uint32_t *col = a.col + I.edge_base;
  for (uint32_t q = lp0; q < lp1; ++q) {
    const uint32_t row = row0 + a.blong_rows[q];
    const uint32_t e0 = rp[row], e1 = rp[row + 1];
    float sum = 0.f;
    for (uint32_t e = e0 + tid; e < e1; e += kBThreads) {
      const uint32_t c = ld_stream(col + e);
      if (CB_DCHECK(c < I.n, kDbgCsrCol, c)) sum += __ldg(x + c);
    }
    sum = warp_sum<float>(sum);
    if ((tid & 31) == 0) s_rowsum[tid >> 5] = sum;
    __syncthreads();
    if (tid == 0) {
      float tot = 0.f;
      for (int w = 0; w < kBThreads / 32; ++w) tot += s_rowsum[w];
      acc += row_epilogue<float>(tot, row, x, xp, out, sj, bp, has_prev);
    }
    __syncthreads();
  }
  acc = warp_sum<float>(acc);
  if (lane == 0) s_red[warp] = (double)acc;
  __syncthreads();
  double part = 0.0;
  if (warp == 0) part = warp_sum_d(s_red[lane]);
  if (tid == 0) {
    if (s_abort) {  // a block never arrived: this step of the realisation fails
      a.sc.status[r] = CB_ERR_TIMEOUT;
      part = __longlong_as_double(0x7ff8000000000000ll);
    }
    drain();
  }
  double total;
  if (arrive_and_reduce(I.bspmv, t - I.btile_base, r, part, a.red, &total))
    finish_alpha<float>(a, r, j, total);
}

// w = W_{j+1} - alpha_j scale_j W_j, in place; beta_j = ||w||.  Each thread
// owns 8 consecutive nodes of the tile (16- or 32-byte aligned vectors).
template <typename T>
__global__ void __launch_bounds__(kThreads) finalize_kernel(LArgs a, uint32_t j, uint32_t fin_off) {
  static_assert(kFinRows == 8 * kThreads, "8 nodes per thread");
  __shared__ double s_red[32];
  const uint32_t t = fin_off + blockIdx.x;
  const uint32_t r = a.fin_inst[t];
  const InstDesc &I = a.inst[r];
  const uint32_t ms = a.sc.ms;
  T *Vb = reinterpret_cast<T *>(a.V);
  const T *x = Vb + (uint64_t)j * a.vs + I.node_base;
  T *out = Vb + (uint64_t)(j + 1) * a.vs + I.node_base;
  const uint32_t i0 = (t - I.fin_base) * kFinRows + 8 * threadIdx.x;
  const bool full = i0 + 8 <= I.n;
  // the vector loads go out before the scalars they do not depend on (the
  // CTA's latency chain is most of its lifetime); a finished realisation
  // only reads them
  T u[8], v[8];
  if (full) Vec8<T>::load(x + i0, v);  // W_j: complete before the SpMV began
  dep_wait();
  dep_trigger();
  if (full) Vec8<T>::load(out + i0, u);
  if (j >= a.sc.meff[r]) return;
  const T coef = (T)(a.sc.alpha[r * ms + j] * a.sc.scale[r * ms + j]);
  T acc = T(0);
  if (full) {
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      u[q] -= coef * v[q];
      acc += u[q] * u[q];
    }
    Vec8<T>::store(out + i0, u);
  } else {
    for (uint32_t i = i0; i < I.n; ++i) {
      const T w = out[i] - coef * x[i];
      out[i] = w;
      acc += w * w;
    }
  }
  // the tile's partial of ||w||^2 goes to its slot; beta_j follows in
  // finalize_beta_kernel, so no CTA waits on an arrival counter
  const double part = block_sum_to_double<T>(acc, s_red);
  if (threadIdx.x == 0) a.red.part[I.fin.slot_base + (t - I.fin_base)] = part;
}

// beta_j = ||w|| per realisation from the finalize partials, one CTA of
// kThreads per realisation: group sums over kGroup slots by one warp each,
// then the sum over groups, in the same order and shapes as the
// last-arriving reduction of arrive_and_reduce (so beta is bit-identical to
// it); then the breakdown test and scale_{j+1} = 1 / beta.
__global__ void __launch_bounds__(kThreads) finalize_beta_kernel(LArgs a, uint32_t j, uint32_t r0) {
  __shared__ double s_red[kThreads / 32];
  const uint32_t r = r0 + blockIdx.x;
  const RedPlan P = a.inst[r].fin;
  dep_wait();
  dep_trigger();
  if (j >= a.sc.meff[r]) return;
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // Many groups: one lane per group, its 32 slots added in the order of the
  // warp sum's tree.  A warp then issues 31 FP64 additions for 32 groups, not
  // 5 for each (an addition holds its sub-core for 65 cycles however many lanes
  // are active): 4883 partials (1e7 nodes) 20.3 -> 8.4 us; from about 24 groups
  // on it is the shorter chain.
  static_assert(kGroup == 32, "one lane per slot of a group");
  if (P.n_groups >= 24) {
    for (uint32_t g = threadIdx.x; g < P.n_groups; g += kThreads) {
      const uint32_t gsize = min((uint32_t)kGroup, P.n_slots - g * kGroup);
      const double *p = a.red.part + P.slot_base + g * kGroup;
      double v[32];
#pragma unroll
      for (uint32_t q = 0; q < 32; ++q) v[q] = q < gsize ? p[q] : 0.0;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int q = 0; q < o; ++q) v[q] += v[q + o];
      a.red.gpart[P.group_base + g] = v[0];
    }
  } else {
    for (uint32_t g = warp; g < P.n_groups; g += kThreads / 32) {
      const uint32_t gsize = min((uint32_t)kGroup, P.n_slots - g * kGroup);
      double v = lane < gsize ? a.red.part[P.slot_base + g * kGroup + lane] : 0.0;
      v = warp_sum_d(v);
      if (lane == 0) a.red.gpart[P.group_base + g] = v;
    }
  }
  __syncthreads();
  double acc = 0.0;
  for (uint32_t q = threadIdx.x; q < P.n_groups; q += kThreads) acc += a.red.gpart[P.group_base + q];
  acc = warp_sum_d(acc);
  if (lane == 0) s_red[warp] = acc;
  __syncthreads();
  if (threadIdx.x != 0) return;
  double total = 0.0;
  for (int w = 0; w < kThreads / 32; ++w) total += s_red[w];
  const uint32_t ms = a.sc.ms;
  const double beta = sqrt(total);
  const double alpha = a.sc.alpha[r * ms + j];
  const double bprev = j > 0 ? a.sc.beta[r * ms + j - 1] : 0.0;
  a.sc.beta[r * ms + j] = beta;
  if (!isfinite(beta)) {
    a.sc.status[r] = CB_ERR_NONFINITE;
    a.sc.meff[r] = j + 1;
  } else if (beta <= a.tau * (fabs(alpha) + bprev) || beta == 0.0) {
    a.sc.meff[r] = j + 1;  // exact breakdown: K_{j+1}(A,1) is invariant
  } else {
    a.sc.scale[r * ms + j + 1] = 1.0 / beta;
  }
}

// ---------------------------------------------------------------------------
// Small realisations (n <= kSmallN, at most kSmallNnz entries) without
// reorthogonalisation, in FP64 and, with hubs, in FP32 (here the order of the
// sums stays, which decides the trailing part of T once orthogonality is lost,
// and theta's last FP32 digits with hubs); in FP32 without hubs those too dense
// for the team kernel (cb_team.cu) and too few entries in all for the per-step
// kernels (140 graphs of 1000 nodes, degree 150: 34 us a step, 61 per step,
// 299 by teams): one CTA per realisation runs all m Lanczos steps in one launch -- SpMV with the row
// epilogue, alpha, the axpy w = u - alpha_j scale_j W_j, beta_j and the
// breakdown test, the same arithmetic as spmv_kernel + finalize_kernel +
// finalize_beta_kernel -- with W_j, W_{j-1} and the new vector resident in
// shared memory (each new vector is also written to the basis) and the
// reductions CTA-wide (no grid-wide one is needed), so a pass of m steps is
// one launch instead of 3m.  Rows are summed by groups of 8 lanes.
// ---------------------------------------------------------------------------
constexpr int kSmallThreads = 512;

template <typename T>
__global__ void __launch_bounds__(kSmallThreads) lanczos_small_kernel(LArgs a, uint32_t r0, uint32_t m) {
  // three vectors of the realisation rotate through shared memory: W_j, W_{j-1}
  // and the new one (u, then w); each new vector is also stored to the basis
  extern __shared__ float4 s_dyn4[];
  const uint32_t r = r0 + blockIdx.x;
  const InstDesc &I = a.inst[r];
  const uint32_t n = I.n, ms = a.sc.ms;
  T *xs = reinterpret_cast<T *>(s_dyn4);  // W_j
  T *xps = xs + ((n + 3) & ~3u);          // W_{j-1}
  T *us = xps + ((n + 3) & ~3u);          // u, then W_{j+1}
  __shared__ double s_red[32];
  const uint32_t *rp = a.row_ptr + I.rp_base;
  const uint32_t *cl = a.col + I.edge_base;
  T *Vb = reinterpret_cast<T *>(a.V);
  const uint32_t tid = threadIdx.x, l8 = tid & 7u, grp = tid >> 3;
  const unsigned gmask = 0xffu << (tid & 24u);  // the 8 lanes of this thread's group
  constexpr uint32_t kGroups = kSmallThreads / 8;
  {
    const T *x0 = Vb + I.node_base;
    for (uint32_t i = tid; i < n; i += kSmallThreads) xs[i] = x0[i];
  }
  // the recurrence scalars stay in shared memory between steps (thread 0
  // writes them to the Scalars arrays as it forms them, never reads them back)
  __shared__ double s_scale, s_beta_prev, s_alpha;
  __shared__ int s_stop;
  if (tid == 0) {
    s_scale = a.sc.scale[r * ms];
    s_beta_prev = 0.0;
    s_stop = a.sc.meff[r] == 0u;
  }
  const uint32_t mr = a.sc.meff[r] < m ? a.sc.meff[r] : m;  // steps allowed from the start
  __syncthreads();
  double scale_prev = 0.0;  // scale_{j-1} (all threads)
  for (uint32_t j = 0; j < mr; ++j) {
    if (s_stop) break;  // uniform: set by thread 0 before a CTA barrier
    T *out = Vb + (uint64_t)(j + 1) * a.vs + I.node_base;
    const double scale_j = s_scale;
    const T sj = (T)scale_j;
    const T bp = j > 0 ? (T)(s_beta_prev * scale_prev) : T(0);
    T acc = T(0);
    for (uint32_t i = grp; i < n; i += kGroups) {
      T sum = T(0);
      for (uint32_t e = rp[i] + l8; e < rp[i + 1]; e += 8) {
        const uint32_t c = cl[e];
        if (CB_DCHECK(c < n, kDbgCsrCol, c)) sum += xs[c];
      }
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) sum += __shfl_xor_sync(gmask, sum, o, 8);
      if (l8 == 0) {
        T u = sj * sum;
        if (j > 0) u -= bp * xps[i];
        us[i] = u;
        acc += xs[i] * u;
      }
    }
    const double dot = block_sum_to_double<T>(acc, s_red);  // also orders `us` for the CTA
    if (tid == 0) {  // alpha_j, as finish_alpha
      const double alpha = scale_j * dot;
      a.sc.alpha[r * ms + j] = alpha;
      s_alpha = alpha;
      if (!isfinite(alpha)) {
        if (a.sc.status[r] == CB_OK) a.sc.status[r] = CB_ERR_NONFINITE;
        a.sc.meff[r] = j;
        s_stop = 1;
      }
    }
    __syncthreads();
    if (s_stop) break;  // alpha was not finite
    const T coef = (T)(s_alpha * scale_j);
    T acc2 = T(0);
    for (uint32_t i = tid; i < n; i += kSmallThreads) {
      const T w = us[i] - coef * xs[i];
      us[i] = w;
      out[i] = w;
      acc2 += w * w;
    }
    const double total = block_sum_to_double<T>(acc2, s_red);
    if (tid == 0) {  // beta_j, the breakdown test and scale_{j+1}, as finalize_beta_kernel
      const double beta = sqrt(total);
      const double alpha = s_alpha, bprev = s_beta_prev;
      a.sc.beta[r * ms + j] = beta;
      if (!isfinite(beta)) {
        a.sc.status[r] = CB_ERR_NONFINITE;
        a.sc.meff[r] = j + 1;
        s_stop = 1;
      } else if (beta <= a.tau * (fabs(alpha) + bprev) || beta == 0.0) {
        a.sc.meff[r] = j + 1;
        s_stop = 1;
      } else {
        a.sc.scale[r * ms + j + 1] = 1.0 / beta;
        s_scale = 1.0 / beta;
      }
      s_beta_prev = beta;
    }
    scale_prev = scale_j;
    __syncthreads();
    T *t = xps;  // rotate: W_{j-1} <- W_j, W_j <- W_{j+1}
    xps = xs;
    xs = us;
    us = t;
  }
}

// ---------------------------------------------------------------------------
// Full reorthogonalisation (CB_REORTH), after the finalize of step j: the new
// vector w (basis slot j + 1, unnormalised) is orthogonalised against
// v_i = scale_i W_i, i = 0..j, by classical Gram-Schmidt,
//   h_i = v_i . w,   w <- w - sum_i h_i v_i,   beta_j = ||w||,
// run twice, as the oracle does.  Per pass: partial dots per finalize tile,
// their ordered sum per realisation, then the update with the norm reduced
// as in finalize (deterministic throughout).  A step that has stopped
// (breakdown in finalize or in an earlier pass: scale_{j+1} = 0) is left
// alone.
// ---------------------------------------------------------------------------
__device__ __forceinline__ bool reorth_active(const LArgs &a, uint32_t r, uint32_t j) {
  return j < a.sc.meff[r] && a.sc.scale[r * a.sc.ms + j + 1] != 0.0;
}

template <typename T>
__global__ void __launch_bounds__(kThreads) reorth_dot_kernel(LArgs a, uint32_t j, uint32_t fin_off,
                                                              double *rpart) {
  __shared__ double s_w[kThreads / 32][CB_MAX_M + 1];
  const uint32_t t = fin_off + blockIdx.x;
  const uint32_t r = a.fin_inst[t];
  if (!reorth_active(a, r, j)) return;
  const InstDesc &I = a.inst[r];
  const uint32_t ms = a.sc.ms;
  const T *Vb = reinterpret_cast<const T *>(a.V);
  const T *w = Vb + (uint64_t)(j + 1) * a.vs + I.node_base;
  const uint32_t i0 = (t - I.fin_base) * kFinRows + 8 * threadIdx.x;
  const uint32_t cnt = i0 < I.n ? min(8u, I.n - i0) : 0u;
  T wv[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) wv[q] = T(0);
  if (cnt == 8) {
    Vec8<T>::load(w + i0, wv);
  } else {
    for (uint32_t q = 0; q < cnt; ++q) wv[q] = w[i0 + q];
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (uint32_t i = 0; i <= j; ++i) {
    const T *x = Vb + (uint64_t)i * a.vs + I.node_base;
    T xv[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) xv[q] = T(0);
    if (cnt == 8) {
      Vec8<T>::load(x + i0, xv);
    } else {
      for (uint32_t q = 0; q < cnt; ++q) xv[q] = x[i0 + q];
    }
    T acc = T(0);
#pragma unroll
    for (int q = 0; q < 8; ++q) acc += xv[q] * wv[q];
    acc = warp_sum<T>(acc);
    if (lane == 0) s_w[warp][i] = (double)acc;
  }
  __syncthreads();
  for (uint32_t i = threadIdx.x; i <= j; i += blockDim.x) {
    double sum = 0.0;
    for (int q = 0; q < kThreads / 32; ++q) sum += s_w[q][i];
    rpart[(uint64_t)t * ms + i] = a.sc.scale[r * ms + i] * sum;
  }
}

__global__ void __launch_bounds__(128) reorth_sum_kernel(LArgs a, uint32_t j, uint32_t r0,
                                                         const double *rpart, double *rh) {
  const uint32_t r = r0 + blockIdx.x;
  if (!reorth_active(a, r, j)) return;
  const InstDesc &I = a.inst[r];
  const uint32_t ms = a.sc.ms;
  for (uint32_t i = threadIdx.x; i <= j; i += blockDim.x) {
    double sum = 0.0;  // tile order: deterministic
    for (uint32_t q = 0; q < I.n_fin; ++q) sum += rpart[(uint64_t)(I.fin_base + q) * ms + i];
    rh[r * ms + i] = sum;
  }
}

template <typename T>
__global__ void __launch_bounds__(kThreads) reorth_update_kernel(LArgs a, uint32_t j,
                                                                 uint32_t fin_off, const double *rh) {
  __shared__ double s_red[32];
  __shared__ T s_c[CB_MAX_M + 1];
  const uint32_t t = fin_off + blockIdx.x;
  const uint32_t r = a.fin_inst[t];
  if (!reorth_active(a, r, j)) return;
  const InstDesc &I = a.inst[r];
  const uint32_t ms = a.sc.ms;
  for (uint32_t i = threadIdx.x; i <= j; i += blockDim.x)
    s_c[i] = (T)(rh[r * ms + i] * a.sc.scale[r * ms + i]);
  __syncthreads();
  T *Vb = reinterpret_cast<T *>(a.V);
  T *w = Vb + (uint64_t)(j + 1) * a.vs + I.node_base;
  const uint32_t i0 = (t - I.fin_base) * kFinRows + 8 * threadIdx.x;
  const uint32_t cnt = i0 < I.n ? min(8u, I.n - i0) : 0u;
  T wv[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) wv[q] = T(0);
  if (cnt == 8) {
    Vec8<T>::load(w + i0, wv);
  } else {
    for (uint32_t q = 0; q < cnt; ++q) wv[q] = w[i0 + q];
  }
  for (uint32_t i = 0; i <= j; ++i) {
    const T *x = Vb + (uint64_t)i * a.vs + I.node_base;
    const T c = s_c[i];
    T xv[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) xv[q] = T(0);
    if (cnt == 8) {
      Vec8<T>::load(x + i0, xv);
    } else {
      for (uint32_t q = 0; q < cnt; ++q) xv[q] = x[i0 + q];
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) wv[q] -= c * xv[q];
  }
  T acc = T(0);
  if (cnt == 8) {
    Vec8<T>::store(w + i0, wv);
  } else {
    for (uint32_t q = 0; q < cnt; ++q) w[i0 + q] = wv[q];
  }
#pragma unroll
  for (int q = 0; q < 8; ++q) acc += wv[q] * wv[q];  // entries past cnt are 0
  const double part = block_sum_to_double<T>(acc, s_red);
  double total;
  if (arrive_and_reduce(I.fin, t - I.fin_base, r, part, a.red, &total)) {
    const double beta = sqrt(total);
    const double alpha = a.sc.alpha[r * ms + j];
    const double bprev = j > 0 ? a.sc.beta[r * ms + j - 1] : 0.0;
    a.sc.beta[r * ms + j] = beta;
    if (!isfinite(beta)) {
      a.sc.status[r] = CB_ERR_NONFINITE;
      a.sc.meff[r] = j + 1;
      a.sc.scale[r * ms + j + 1] = 0.0;
    } else if (beta <= a.tau * (fabs(alpha) + bprev) || beta == 0.0) {
      a.sc.meff[r] = j + 1;  // exact breakdown once the lost orthogonality is removed
      a.sc.scale[r * ms + j + 1] = 0.0;
    } else {
      a.sc.scale[r * ms + j + 1] = 1.0 / beta;
    }
  }
}

template <typename T, int G, bool SIDE = false>
static void launch_spmv(const LArgs &a, uint32_t j, uint32_t chunk_off, uint32_t n_chunks,
                        uint32_t tile_off, uint32_t n_tiles, cudaStream_t s) {
  const uint32_t grid = n_chunks + n_tiles;
  if (grid) launch_dep(spmv_kernel<T, G, SIDE>, grid, kThreads, 0, s, a, j, chunk_off, n_chunks, tile_off);
}

template <typename T>
static void launch_spmv_lanes(int lanes, bool side, const LArgs &a, uint32_t j, uint32_t co, uint32_t nc,
                              uint32_t to, uint32_t nt, cudaStream_t s) {
  if constexpr (sizeof(T) == 8) {
    if (lanes == 4 && side) return launch_spmv<T, 4, true>(a, j, co, nc, to, nt, s);
  }
  switch (lanes) {
    case 1: launch_spmv<T, 1>(a, j, co, nc, to, nt, s); break;
    case 2: launch_spmv<T, 2>(a, j, co, nc, to, nt, s); break;
    case 4: launch_spmv<T, 4>(a, j, co, nc, to, nt, s); break;
    case 8: launch_spmv<T, 8>(a, j, co, nc, to, nt, s); break;
    case 16: launch_spmv<T, 16>(a, j, co, nc, to, nt, s); break;
    default: launch_spmv<T, 32>(a, j, co, nc, to, nt, s); break;
  }
}

// The route of the recurrence over realisations [r0, r1) on the automatic path,
// and the plan of the first: on-chip problems take one launch.  A team sums in an
// order of its own: taken where that cannot show, FP64 with reorthogonalisation
// and FP32 ensembles and small graphs without hubs.  One larger graph in FP32 keeps
// the order of the per-step kernels (a planted clique's scores differ by less
// than FP32 rounding), as does FP64 without it (T's trailing part).
enum Route { kPerStep, kTeam, kOneCta };
template <typename T>
static Route one_launch_route(const cb_graph *h, uint32_t r0, uint32_t r1, bool reorth, TeamArgs *ta, uint32_t *grid,
                              bool *cooperative) {
  const cb_graph *hp = h->plan_of ? h->plan_of : h;  // a group handle decides as the whole one
  const uint32_t p0 = h->plan_of ? 0u : r0, p1 = h->plan_of ? hp->n_inst : r1;
  bool small = true, hubs = false;
  for (uint32_t r = p0; r < p1; ++r) {
    small &= hp->inst[r].n <= kSmallN && hp->inst[r].nnz <= kSmallNnz;
    hubs |= hp->inst[r].hubs != 0;
  }
  if ((sizeof(T) == 8 ? reorth : !reorth && !hubs && (small || p1 - p0 > 1)) &&
      team_plan(h, r0, r1, sizeof(T), reorth, ta, grid, cooperative))
    return kTeam;
  return small && !reorth && (sizeof(T) == 8 || hubs || small_launch_pays(hp, p0, p1)) ? kOneCta : kPerStep;
}

bool lanczos_one_launch(const cb_graph *h, int prec) {
  TeamArgs ta;
  uint32_t grid;
  bool coop;
  return (prec == CB_FP64 ? one_launch_route<double>(h, 0, h->n_inst, false, &ta, &grid, &coop)
                          : one_launch_route<float>(h, 0, h->n_inst, false, &ta, &grid, &coop)) != kPerStep;
}

template <typename T>
static int run_t(cb_graph *h, Workspace &W, uint32_t r0, uint32_t r1, uint32_t m, cudaStream_t s,
                 const uint32_t *start_idx, uint32_t k, bool per_inst, const double *rscale) {
  LArgs a;
  a.inst = h->d_inst;
  a.tile_inst = h->d_tile_inst;
  a.tile_rows = h->d_tile_rows;
  a.heavy = h->d_heavy;
  a.chunk_heavy = h->d_chunk_heavy;
  a.fin_inst = h->d_fin_inst;
  a.row_ptr = h->row_ptr;
  a.col = h->col;
  a.V = W.V;
  a.vs = W.vec_stride;
  a.sc = W.sc;
  a.red = RedBufs{W.part, W.gpart, W.gcnt, W.icnt};
  a.cpart = W.cpart;
  a.hcnt = W.hcnt;
  a.tau = sizeof(T) == 4 ? 1e-5 : 1e-12;
  a.btile_inst = h->d_btile_inst;
  a.bseg_base = h->d_bseg_base;
  a.bwstart = h->d_bwstart;
  a.bwlen = h->d_bwlen;
  a.belem = h->d_belem;
  a.blong_ptr = h->d_blong_ptr;
  a.blong_rows = h->d_blong_rows;
  // FP32 path: the column-blocked kernel needs about one 16384-row tile per
  // SM to fill the GPU (a single 1e5-node graph has 7), so the automatic
  // choice takes it only from one tile per SM on; the test hook forces it
  const bool blocked_auto = h->total_btiles >= h->n_sm || h->stall_btile != UINT32_MAX;
  const bool use_blocked = sizeof(T) == 4 && h->total_btiles > 0 && h->path != CB_PATH_CSR &&
                           (h->path == CB_PATH_FORMATS || blocked_auto);
  a.skip_blocked = use_blocked ? 1u : 0u;
  a.stall_btile = h->stall_btile;
  a.pbin = h->d_pbin;
  a.ptbase = h->d_ptbase;
  a.ptile_inst = h->d_ptile_inst;
  a.pxbase = h->d_pxbase;
  a.psrc = h->d_psrc;
  a.pgdst = h->d_pgdst;
  a.pX = h->d_pX;
  a.psl = h->d_psl;
  a.pdesc = h->d_pdesc;
  a.pgroups = h->total_pgroups;
  const bool use_pb = sizeof(T) == 4 && h->total_ptiles > 0 && h->path != CB_PATH_CSR;
  a.skip_pb = use_pb ? 1u : 0u;

  const InstDesc &A0 = h->inst[r0], &A1 = h->inst[r1 - 1];
  const uint32_t chunk_off = A0.chunk_base;
  const uint32_t n_chunks = A1.chunk_base + A1.n_chunks - chunk_off;
  const uint32_t tile_off = A0.tile_base;
  const uint32_t n_tiles = A1.tile_base + A1.n_tiles - tile_off;
  const uint32_t fin_off = A0.fin_base;
  const uint32_t n_fin = A1.fin_base + A1.n_fin - fin_off;
  const uint32_t btile_off = A0.btile_base;
  const uint32_t n_btiles = use_blocked ? A1.btile_base + A1.n_btiles - btile_off : 0u;
  a.border = n_btiles == h->total_btiles ? h->d_border : nullptr;  // part of them: in their own order
  const uint32_t ptile_lo = A0.ptile_base, ptile_hi = A1.ptile_base + A1.pns;
  const uint64_t pg_lo = use_pb ? h->ptbase[ptile_lo] : 0, pg_hi = use_pb ? h->ptbase[ptile_hi] : 0;
  const uint32_t bin_off = A0.pbin_base;
  const uint32_t n_bins = use_pb ? A1.pbin_base + A1.n_pbin - bin_off : 0u;
  bool any_pb = false;  // two-phase realisations in the range (their heavy rows too)
  for (uint32_t r = r0; r < r1 && use_pb; ++r) any_pb |= h->inst[r].pb != 0;
  // does the tiled-CSR kernel have work in the range?
  bool any_csr = false;
  for (uint32_t r = r0; r < r1 && !any_csr; ++r)
    any_csr = !(use_blocked && h->inst[r].blocked) && !(use_pb && h->inst[r].pb);
  if (n_btiles) {
    static bool attr_set = false;  // one-time opt-in to > 48 KB of shared memory
    if (!attr_set) {
      cudaFuncSetAttribute(bspmv_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)kBSmemBytes);
      cudaFuncSetAttribute(bspmv_kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                           cudaSharedmemCarveoutMaxShared);
      attr_set = true;
    }
  }

  uint32_t nmax = 0;
  for (uint32_t r = r0; r < r1; ++r) nmax = h->inst[r].n > nmax ? h->inst[r].n : nmax;
  const uint64_t init_n8 = (A1.node_base + A1.n - A0.node_base + 7) / 8;
  static_assert(kNodeAlign % 8 == 0, "a realisation's last 8 nodes lie in its own range");
  const uint32_t init_grid = (uint32_t)std::min<uint64_t>((init_n8 + kThreads - 1) / kThreads, 8 * h->n_sm);
  prefer_shared(init_vec_kernel<T>);
  prefer_shared(init_indicator_kernel<T>);
  prefer_shared(init_scalars_kernel);
  prefer_shared(finalize_kernel<T>);
  int tok = prof_begin(CB_K_INIT, s);
  if (!rscale)
    init_vec_kernel<T><<<init_grid ? init_grid : 1, kThreads, 0, s>>>(
        reinterpret_cast<T *>(a.V) + A0.node_base, init_n8, start_idx ? T(0) : T(1));
  if (start_idx && !rscale)
    init_indicator_kernel<T><<<r1 - r0, kThreads, 0, s>>>(a, r0, start_idx, k, per_inst);
  TeamArgs ta;
  uint32_t team_grid = 0;
  bool team_coop = false;
  Route route = kPerStep;
  if ((h->path == CB_PATH_AUTO || (h->tuned && sizeof(T) == 8 && h->reorth)) && h->stall_btile == UINT32_MAX)
    route = one_launch_route<T>(h, r0, r1, h->reorth, &ta, &team_grid, &team_coop);
  const uint64_t nsc = (uint64_t)(r1 - r0) * W.sc.ms;
  init_scalars_kernel<<<(uint32_t)((nsc + kThreads - 1) / kThreads), kThreads, 0, s>>>(
      a, r0, r1, m, start_idx, k, per_inst, rscale, W.tctr);
  prof_end(tok, s);
  if (route == kTeam) {
    ta.parts = W.tparts;
    ta.ctr = W.tctr;
    ta.xd = W.xd;
    ta.wait_ns = barrier_wait_ns();
    ta.stall = barrier_stall_ms() != 0;
    tok = prof_begin(CB_K_SPMV, s);
    const int rc = team_launch<T>(a, ta, r0, m, team_grid, team_coop, s);
    prof_end(tok, s);
    return rc;
  }
  if (route == kOneCta) {
    cudaFuncSetAttribute(lanczos_small_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)(3 * kSmallN * sizeof(T)));
    tok = prof_begin(CB_K_SPMV, s);
    lanczos_small_kernel<T><<<r1 - r0, kSmallThreads, 3 * (size_t)((nmax + 3) & ~3u) * sizeof(T), s>>>(a, r0, m);
    prof_end(tok, s);
    return cuda_error(cudaGetLastError(), "lanczos launch");
  }
  const bool side = h->total_nnz < kSideDeg * h->total_nodes_padded;
  for (uint32_t j = 0; j < m; ++j) {
    tok = prof_begin(CB_K_SPMV, s);
    if (any_csr) launch_spmv_lanes<T>(h->lanes, side, a, j, chunk_off, n_chunks, tile_off, n_tiles, s);
    if (n_btiles) launch_dep(bspmv_kernel, n_btiles, kBThreads, kBSmemBytes, s, a, j, btile_off);
    if (any_pb)
      launch_twophase(a, h->lanes, j, ptile_lo, ptile_hi, pg_lo, pg_hi, chunk_off, n_chunks,
                      bin_off, n_bins, s);
    prof_end(tok, s);
    tok = prof_begin(CB_K_FINALIZE, s);
    if (n_fin) {
      launch_dep(finalize_kernel<T>, n_fin, kThreads, 0, s, a, j, fin_off);
      launch_dep(finalize_beta_kernel, r1 - r0, kThreads, 0, s, a, j, r0);
    }
    if (n_fin && h->reorth)
      for (int pass = 0; pass < 2; ++pass) {
        reorth_dot_kernel<T><<<n_fin, kThreads, 0, s>>>(a, j, fin_off, W.rpart);
        reorth_sum_kernel<<<r1 - r0, 128, 0, s>>>(a, j, r0, W.rpart, W.rh);
        reorth_update_kernel<T><<<n_fin, kThreads, 0, s>>>(a, j, fin_off, W.rh);
      }
    prof_end(tok, s);
  }
  return cuda_error(cudaGetLastError(), "lanczos launch");
}

int lanczos_run(cb_graph *h, Workspace &W, uint32_t r0, uint32_t r1, uint32_t m, int prec,
                cudaStream_t s, const uint32_t *start_idx, uint32_t k, bool per_inst,
                const double *restart_scale) {
  NvtxRange nvtx_range("lanczos");
  return prec == CB_FP64 ? run_t<double>(h, W, r0, r1, m, s, start_idx, k, per_inst, restart_scale)
                         : run_t<float>(h, W, r0, r1, m, s, start_idx, k, per_inst, restart_scale);
}

CB_DEBUG_READER(lanczos)

}  // namespace cb
