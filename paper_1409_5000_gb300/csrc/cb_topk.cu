// Top-k selection of the summed scores of eq. 5 (section "Identification
// algorithm": the recovered target is the k nodes of largest summed EBTC).
//
// The paper sorts all n scores (Introsort, O(n log n)).  Only the k largest
// are needed, so one kernel selects a few candidates and sorts those:
//
//  * each score maps to an order-preserving 64-bit key (NaN lowest, -0 = +0),
//    extended by the complemented node index: the 96-bit composite keys are
//    distinct and larger composite = larger score, ties to the smaller index;
//  * every thread takes the largest key of its own elements.  The k-th largest
//    of these maxima bounds the k-th largest element from below, so a radix
//    select over one key per thread (11 bits a pass, histograms merged over
//    the grid) gives a threshold that at least k and usually few more elements
//    reach: the scores are read twice in all, whatever their digits;
//  * the elements at or above the threshold are collected and sorted by one
//    CTA (bitonic).  If more than kCand reach it (ties), or k is too large for
//    the maxima to bound it well, the radix select runs over the composite
//    keys of all elements instead, until at most kCand remain.
//
// The passes are separated by grid barriers of one cooperative launch (up to
// one CTA per SM; a single CTA with everything in shared memory for small n).
// Up to 4096 scores one bitonic sort of all took 17 us at n = 500 and 100 us
// at n = 4000 (now 12 and 16 us), and above that 12 histogram passes with a
// launch each 67 us at n = 1e5 and 250 us at n = 1e7 (now 17 and 93 us): the
// launches, and in the first passes, where all scores share a digit, the
// histogram's same-address atomics.
#include <algorithm>

#include "cb_grid.cuh"
#include "cb_internal.cuh"

namespace cb {

namespace {

constexpr uint32_t kTopkThreads = 1024;
constexpr uint32_t kBins = 2048;   // 11-bit digits
constexpr uint32_t kLevels = 9;    // 64 key bits as 5 x 11 + 9, then 32 index bits as 11 + 11 + 10
constexpr uint32_t kKeyLevels = 6;
constexpr uint32_t kCand = CB_MAX_TOPK;  // most candidates one CTA sorts
constexpr uint32_t kFew = 1024;          // candidates after which no further pass pays
constexpr uint32_t kOneCta = 4096;       // up to this many scores: one CTA

struct TopkState {
  uint32_t bar;      // grid barrier
  uint32_t ncol;     // candidates collected
  uint32_t pad[62];
  uint32_t hist[3][kBins];  // pass p adds into hist[p % 3]; cleared two barriers later
};

struct Cand {
  unsigned long long key;
  uint32_t idx;
  uint32_t pad;
};

// order-preserving key, integer arithmetic only (FP64 compares are scarce)
__device__ __forceinline__ unsigned long long order_key(double v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  const unsigned long long mag = b & 0x7fffffffffffffffull;
  if (mag > 0x7ff0000000000000ull) return 0ull;        // NaN ranks below every number
  if (mag == 0ull) return 0x8000000000000000ull;       // -0.0 -> +0.0
  return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}

// bits fixed before level L, and the digit of level L
__device__ __forceinline__ uint32_t bits_before(uint32_t L) {
  return L <= 5 ? 11 * L : (L == 6 ? 64u : (L == 7 ? 75u : (L == 8 ? 86u : 96u)));
}
__device__ __forceinline__ unsigned long long mask_hi(uint32_t L) {
  const uint32_t b = bits_before(L);
  return b == 0 ? 0ull : (b >= 64 ? ~0ull : (~0ull << (64 - b)));
}
__device__ __forceinline__ uint32_t mask_lo(uint32_t L) {
  const uint32_t b = bits_before(L);
  return b <= 64 ? 0u : (b >= 96 ? ~0u : (~0u << (96 - b)));
}
__device__ __forceinline__ uint32_t digit(unsigned long long hi, uint32_t lo, uint32_t L) {
  if (L < 5) return (uint32_t)(hi >> (53 - 11 * L)) & 2047u;
  if (L == 5) return (uint32_t)hi & 511u;
  return L == 6 ? lo >> 21 : (L == 7 ? (lo >> 10) & 2047u : lo & 1023u);
}
__device__ __forceinline__ unsigned long long put_hi(uint32_t d, uint32_t L) {
  return L < 5 ? (unsigned long long)d << (53 - 11 * L) : (L == 5 ? (unsigned long long)d : 0ull);
}
__device__ __forceinline__ uint32_t put_lo(uint32_t d, uint32_t L) {
  return L < 6 ? 0u : (L == 6 ? d << 21 : (L == 7 ? d << 10 : d));
}

// (key desc, idx asc) ordering: a goes before b
__device__ __forceinline__ bool before(unsigned long long ka, uint32_t ia, unsigned long long kb,
                                       uint32_t ib) {
  return ka > kb || (ka == kb && ia < ib);
}

// The prefix found so far and what is still needed inside it.
struct Select {
  unsigned long long phi;
  uint32_t plo, krem, above;  // above: elements in higher buckets (taken already)
};

// The CTAs that select together (all of the grid, or one alone), and their scratch.
struct Team {
  uint32_t ctas, rank;
  uint64_t wait_ns;
  TopkState *st;  // zeroed; unused by a CTA alone, as is the candidates' global buffer
};

// What the passes share within a CTA.
struct TopkShared {
  uint32_t hist[kBins];
  uint32_t warp[kTopkThreads / 32];
  uint32_t digit, need, bucket, ncol;
};

// End of pass L: the histograms of the grid merged, the digit where the count
// from the top reaches sel.krem chosen, the prefix extended.  Returns the
// elements of the chosen bucket.  pass: passes done so far (selects the merged
// histogram).  *ok turns false when a barrier gave up.
__device__ uint32_t pass_end(TopkShared &sh, const Team &t, Select &sel, uint32_t L, uint32_t &pass,
                             uint32_t &epoch, bool *ok) {
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  __syncthreads();
  uint32_t h0 = sh.hist[kBins - 1 - 2 * tid], h1 = sh.hist[kBins - 2 - 2 * tid];  // from the top
  if (t.ctas > 1) {
    uint32_t *g = t.st->hist[pass % 3];
    if (h0) atomicAdd(&g[kBins - 1 - 2 * tid], h0);
    if (h1) atomicAdd(&g[kBins - 2 - 2 * tid], h1);
    if (!grid_sync(&t.st->bar, epoch, t.ctas, t.wait_ns)) *ok = false;
    h0 = __ldcg(&g[kBins - 1 - 2 * tid]);
    h1 = __ldcg(&g[kBins - 2 - 2 * tid]);
    // the buffer of the previous pass: every CTA read it before this barrier,
    // and its next use is two passes on
    if (pass > 0)
      for (uint32_t q = t.rank * kTopkThreads + tid; q < kBins; q += t.ctas * kTopkThreads)
        t.st->hist[(pass - 1) % 3][q] = 0u;
  }
  ++pass;
  const uint32_t mine = h0 + h1;
  uint32_t incl = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= (uint32_t)o) incl += y;
  }
  if (lane == 31) sh.warp[warp] = incl;
  __syncthreads();
  uint32_t base = 0;
  for (uint32_t w = 0; w < warp; ++w) base += sh.warp[w];
  const uint32_t c0 = base + incl - mine;  // count in higher bins
  if (c0 < sel.krem && c0 + mine >= sel.krem) {  // exactly one thread
    const bool first = c0 + h0 >= sel.krem;
    sh.digit = kBins - 1 - 2 * tid - (first ? 0u : 1u);
    sh.need = sel.krem - (first ? c0 : c0 + h0);
    sh.bucket = first ? h0 : h1;
  }
  __syncthreads();
  sel.phi |= put_hi(sh.digit, L);
  sel.plo |= put_lo(sh.digit, L);
  sel.above += sel.krem - sh.need;
  sel.krem = sh.need;
  const uint32_t bucket = sh.bucket;
  __syncthreads();
  sh.hist[2 * tid] = sh.hist[2 * tid + 1] = 0u;
  __syncthreads();
  return bucket;
}

// Elements whose composite key reaches the prefix (phi, plo) go to buf, in any
// order; their number (which may exceed kCand) is returned.
__device__ uint32_t collect(const double *__restrict__ S, uint32_t n, unsigned long long phi,
                            uint32_t plo, TopkShared &sh, const Team &t, Cand *buf, uint32_t &epoch,
                            bool *ok) {
  uint32_t *ctr = t.ctas > 1 ? &t.st->ncol : &sh.ncol;
  const uint64_t stride = (uint64_t)t.ctas * kTopkThreads;
  uint64_t i = t.rank * kTopkThreads + threadIdx.x;
  auto take = [&](double v, uint32_t at) {
    const unsigned long long key = order_key(v);
    if (key > phi || (key == phi && ~at >= plo)) {
      const uint32_t pos = atomicAdd(ctr, 1u);
      if (pos < kCand) buf[pos] = Cand{key, at, 0u};
    }
  };
  for (; i + 3 * stride < n; i += 4 * stride) {
    double v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = __ldg(S + i + u * stride);
#pragma unroll
    for (int u = 0; u < 4; ++u) take(v[u], (uint32_t)(i + u * stride));
  }
  for (; i < n; i += stride) take(__ldg(S + i), (uint32_t)i);
  if (!grid_sync(t.ctas > 1 ? &t.st->bar : nullptr, epoch, t.ctas, t.wait_ns)) *ok = false;
  const uint32_t c = t.ctas > 1 ? __ldcg(&t.st->ncol) : sh.ncol;
  __syncthreads();  // a second collection clears the count
  return c;
}

// buf[0, C) sorted, the first k out.  One CTA.
__device__ void sort_out(const double *__restrict__ S, const Cand *buf, uint32_t C, uint32_t k,
                         unsigned char *s_raw, uint32_t *idx, double *val) {
  uint32_t P = 32;
  while (P < C) P <<= 1;
  unsigned long long *sk = reinterpret_cast<unsigned long long *>(s_raw);
  uint32_t *si = reinterpret_cast<uint32_t *>(sk + P);
  const uint32_t q = threadIdx.x;
  if (P <= kTopkThreads) {  // one element per thread: strides below 32 by shuffle
    unsigned long long key = 0ull;
    uint32_t ix = 0xffffffffu;  // after every element, NaN included
    if (q < C) {
      key = buf[q].key;
      ix = buf[q].idx;
    }
    for (uint32_t size = 2; size <= P; size <<= 1) {
      for (uint32_t stride = size >> 1; stride > 0; stride >>= 1) {
        unsigned long long ok2;
        uint32_t oi;
        if (stride >= 32) {
          __syncthreads();
          if (q < P) { sk[q] = key; si[q] = ix; }
          __syncthreads();
          ok2 = q < P ? sk[q ^ stride] : 0ull;
          oi = q < P ? si[q ^ stride] : 0u;
        } else {
          ok2 = __shfl_xor_sync(0xffffffffu, key, stride);
          oi = __shfl_xor_sync(0xffffffffu, ix, stride);
        }
        const bool low = (q & stride) == 0, desc = (q & size) == 0;
        if (before(ok2, oi, key, ix) == (low == desc)) { key = ok2; ix = oi; }
      }
    }
    if (q < k) {
      idx[q] = ix;
      val[q] = S[ix];
    }
    return;
  }
  for (uint32_t p = q; p < P; p += kTopkThreads) {
    if (p < C) { sk[p] = buf[p].key; si[p] = buf[p].idx; }
    else { sk[p] = 0ull; si[p] = 0xffffffffu; }
  }
  __syncthreads();
  for (uint32_t size = 2; size <= P; size <<= 1) {
    for (uint32_t stride = size >> 1; stride > 0; stride >>= 1) {
      for (uint32_t a = q; a < P; a += kTopkThreads) {
        const uint32_t p = a ^ stride;
        if (p > a) {
          const bool desc = (a & size) == 0;  // first half of each block in final order
          const bool swap = desc ? before(sk[p], si[p], sk[a], si[a])
                                 : before(sk[a], si[a], sk[p], si[p]);
          if (swap) {
            const unsigned long long tk = sk[a]; sk[a] = sk[p]; sk[p] = tk;
            const uint32_t ti = si[a]; si[a] = si[p]; si[p] = ti;
          }
        }
      }
      __syncthreads();
    }
  }
  for (uint32_t p = q; p < k; p += kTopkThreads) {
    idx[p] = si[p];
    val[p] = S[si[p]];
  }
}

// The candidates, at least k and at most kCand, in buf; their number, or 0 when a
// barrier gave up.
__device__ uint32_t select(const double *__restrict__ S, uint32_t n, uint32_t k, const Team &t, TopkShared &sh,
                           Cand *buf) {
  const uint32_t tid = threadIdx.x;
  const uint64_t stride = (uint64_t)t.ctas * kTopkThreads, i0 = t.rank * kTopkThreads + tid;
  uint32_t epoch = 0, pass = 0, C = kCand + 1;
  bool ok = true;
  sh.hist[2 * tid] = sh.hist[2 * tid + 1] = 0u;
  if (tid == 0) sh.ncol = 0u;
  __syncthreads();
  const uint32_t maxima = (uint32_t)min((uint64_t)n, stride);  // threads that hold an element
  if (k <= maxima / 4 || maxima == n) {
    // threshold: the k-th largest of the threads' maxima, to kFew candidates
    unsigned long long my = 0ull;
    uint64_t i = i0;
    for (; i + 3 * stride < n; i += 4 * stride) {
      double v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) v[u] = __ldg(S + i + u * stride);
#pragma unroll
      for (int u = 0; u < 4; ++u) my = max(my, order_key(v[u]));
    }
    for (; i < n; i += stride) my = max(my, order_key(__ldg(S + i)));
    Select sel{0ull, 0u, k, 0u};
    for (uint32_t L = 0; L < kKeyLevels && ok; ++L) {
      if (i0 < n && (my & mask_hi(L)) == sel.phi) atomicAdd(&sh.hist[digit(my, 0u, L)], 1u);
      const uint32_t bucket = pass_end(sh, t, sel, L, pass, epoch, &ok);
      if (sel.above + bucket <= max(kFew, k) || sel.krem == bucket) break;
    }
    if (ok) C = collect(S, n, sel.phi, 0u, sh, t, buf, epoch, &ok);
  }
  if (C > kCand && ok) {  // uniform over the CTAs: the composite keys of all elements
    if (tid == 0 && t.ctas == 1) sh.ncol = 0u;
    Select sel{0ull, 0u, k, 0u};
    for (uint32_t L = 0; L < kLevels && ok; ++L) {
      const unsigned long long mh = mask_hi(L);
      const uint32_t ml = mask_lo(L);
      for (uint64_t i = i0; i < n; i += stride) {
        const unsigned long long key = order_key(__ldg(S + i));
        const uint32_t lo = ~(uint32_t)i;
        if ((key & mh) == sel.phi && (lo & ml) == sel.plo) atomicAdd(&sh.hist[digit(key, lo, L)], 1u);
      }
      // no CTA still reads the count of the first collection after the first barrier
      const uint32_t bucket = pass_end(sh, t, sel, L, pass, epoch, &ok);
      if (L == 0 && t.ctas > 1 && t.rank == 0 && tid == 0) t.st->ncol = 0u;
      if (L > 0 && (sel.above + bucket <= max(kFew, k) || sel.krem == bucket)) break;
    }
    if (ok) C = collect(S, n, sel.phi, sel.plo, sh, t, buf, epoch, &ok);
  }
  return ok ? C : 0u;
}

// Every wait is bounded (a GPU that suspends a CTA for seconds must not hang the
// others).  Should one give up, the first CTA selects alone: what it then reads
// and writes is its own, so CTAs that come late disturb nothing, and the result is
// the same.  Its candidates stay in shared memory, beside the sort's arrays.
__global__ void __launch_bounds__(kTopkThreads, 1) topk_kernel(const double *__restrict__ S, uint32_t n,
                                                               uint32_t k, TopkState *st, Cand *gbuf,
                                                               uint32_t *idx, double *val, uint64_t wait_ns,
                                                               uint32_t stall) {
  extern __shared__ __align__(16) unsigned char s_raw[];
  __shared__ TopkShared sh;
  Cand *own = reinterpret_cast<Cand *>(s_raw + kCand * 12), *buf = gridDim.x > 1 ? gbuf : own;
  if (stall && blockIdx.x > 0 && blockIdx.x + 1 == gridDim.x) return;  // test hook
  uint32_t C = select(S, n, k, Team{gridDim.x, blockIdx.x, wait_ns, st}, sh, buf);
  if (blockIdx.x != 0) return;
  if (C == 0) {
    buf = own;
    __syncthreads();
    C = select(S, n, k, Team{1u, 0u, wait_ns, nullptr}, sh, buf);
  }
  sort_out(S, buf, C, k, s_raw, idx, val);
}

}  // namespace

int topk_launch(const double *S, uint32_t n, uint32_t k, uint32_t *idx, double *val,
                void *scratch, cudaStream_t s) {
  // shared memory: the sort's arrays and the candidates of a CTA that selects alone
  constexpr size_t kSort = (size_t)kCand * 12, kAll = kSort + (size_t)kCand * sizeof(Cand);
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(topk_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kAll);
  if (e != cudaSuccess) return cuda_error(e, "topk launch");
  const int tok = prof_begin(CB_K_TOPK, s);
  if (n <= kOneCta) {
    topk_kernel<<<1, kTopkThreads, kAll, s>>>(S, n, k, nullptr, nullptr, idx, val, 0, 0);
  } else {
    TopkState *st = reinterpret_cast<TopkState *>(scratch);
    Cand *buf = reinterpret_cast<Cand *>(st + 1);
    // four scores per thread up to one CTA per SM: a barrier over fewer CTAs is cheaper
    const uint32_t grid = std::min<uint32_t>((uint32_t)sms, (n + 4 * kTopkThreads - 1) / (4 * kTopkThreads));
    e = cudaMemsetAsync(st, 0, sizeof(TopkState), s);
    uint64_t wait_ns = barrier_wait_ns();
    uint32_t stall = barrier_stall_ms() != 0;
    void *args[] = {&S, &n, &k, &st, &buf, &idx, &val, &wait_ns, &stall};
    if (e == cudaSuccess)
      e = cudaLaunchCooperativeKernel(reinterpret_cast<const void *>(topk_kernel), dim3(grid),
                                      dim3(kTopkThreads), args, kAll, s);
  }
  prof_end(tok, s);
  if (e == cudaSuccess) e = cudaGetLastError();
  return cuda_error(e, "topk launch");
}

size_t topk_scratch_bytes(uint32_t /*k*/) { return sizeof(TopkState) + (size_t)kCand * sizeof(Cand); }

}  // namespace cb

CB_API int cb_topk(const double *S, uint32_t n, uint32_t k, uint32_t *idx, double *val,
                   void *stream) {
  cb::NvtxRange nvtx_range("cb_topk");
  using namespace cb;
  if (!S || !idx || !val) return set_error(CB_ERR_ARG, "cb_topk: null pointer");
  if (n == 0 || k == 0 || k > n || k > CB_MAX_TOPK)
    return set_error(CB_ERR_ARG, "cb_topk: need 1 <= k <= min(n, CB_MAX_TOPK)");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  void *scratch = nullptr;
  cudaError_t e = cudaMallocAsync(&scratch, topk_scratch_bytes(k), s);
  if (e != cudaSuccess) return cuda_error(e, "cb_topk: cudaMallocAsync");
  int rc = topk_launch(S, n, k, idx, val, scratch, s);
  e = cudaFreeAsync(scratch, s);
  if (rc != CB_OK) return rc;
  return cuda_error(e, "cb_topk: cudaFreeAsync");
}

// ---------------------------------------------------------------------------
// Top-k without allocation.
//
// cb_topk takes its scratch from the stream-ordered allocator.  Some callers
// cannot allocate device memory at all: a host application that has
// reserved the whole GPU for its own pool and rejects any further cudaMalloc
// / cudaMallocAsync, a plug-in whose host forbids CUDA allocation calls, or a
// latency-critical loop where an allocation could stall on the device.  This
// variant uses a fixed file-scope device array instead, sized for the
// largest k the library accepts (CB_MAX_TOPK), about 90 KB per device.  It
// runs the same kernels as cb_topk.
// ---------------------------------------------------------------------------
#include <mutex>

namespace cb {
namespace {

constexpr size_t kNoAllocScratchBytes = sizeof(TopkState) + (size_t)kCand * sizeof(Cand);

// Shared by every cb_topk_noalloc call on a device; resident until exit.
__device__ __align__(256) unsigned char g_topk_noalloc_scratch[kNoAllocScratchBytes];

// The array's device address belongs to the CUDA context that loaded the
// module, so it is cached per context: keyed by the context's process-unique
// id (cuCtxGetId), which a context created after cudaDeviceReset, or another
// context made current on the same device, does not share.  The driver
// functions come through the runtime's entry-point query, so the library
// needs no link against the driver library.
typedef int (*CtxGetCurrentFn)(void **ctx);
typedef int (*CtxGetIdFn)(void *ctx, unsigned long long *id);
constexpr int kMaxContexts = 64;
std::mutex g_noalloc_mu;
unsigned long long g_noalloc_ctx[kMaxContexts] = {};
void *g_noalloc_ptr[kMaxContexts] = {};
int g_noalloc_used = 0;
CtxGetCurrentFn g_ctx_get_current = nullptr;
CtxGetIdFn g_ctx_get_id = nullptr;

// Device address of the scratch array in the current context.  The host-side
// symbol is only a stand-in, so the address is looked up (with the context
// current) the first time a context calls, and cached.
int noalloc_scratch(void **out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_error(e, "cb_topk_noalloc: cudaGetDevice");
  std::lock_guard<std::mutex> lk(g_noalloc_mu);
  if (!g_ctx_get_current || !g_ctx_get_id) {
    cudaDriverEntryPointQueryResult q1, q2;
    e = cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", (void **)&g_ctx_get_current, 12000,
                                         cudaEnableDefault, &q1);
    if (e == cudaSuccess)
      e = cudaGetDriverEntryPointByVersion("cuCtxGetId", (void **)&g_ctx_get_id, 12000,
                                           cudaEnableDefault, &q2);
    if (e != cudaSuccess || q1 != cudaDriverEntryPointSuccess || q2 != cudaDriverEntryPointSuccess) {
      g_ctx_get_current = nullptr;
      g_ctx_get_id = nullptr;
      return set_error(CB_ERR_CUDA, "cb_topk_noalloc: driver context query unavailable");
    }
  }
  void *ctx = nullptr;
  if (g_ctx_get_current(&ctx) != 0 || !ctx) {
    // no context current on this thread yet: make the device's primary
    // context current (cudaSetDevice initialises it; no allocation)
    e = cudaSetDevice(dev);
    if (e != cudaSuccess) return cuda_error(e, "cb_topk_noalloc: cudaSetDevice");
    if (g_ctx_get_current(&ctx) != 0 || !ctx)
      return set_error(CB_ERR_CUDA, "cb_topk_noalloc: no current CUDA context");
  }
  unsigned long long id = 0;
  if (g_ctx_get_id(ctx, &id) != 0) return set_error(CB_ERR_CUDA, "cb_topk_noalloc: cuCtxGetId failed");
  for (int q = 0; q < g_noalloc_used; ++q)
    if (g_noalloc_ctx[q] == id) {
      *out = g_noalloc_ptr[q];
      return CB_OK;
    }
  void *p = nullptr;
  e = cudaGetSymbolAddress(&p, g_topk_noalloc_scratch);
  if (e != cudaSuccess) return cuda_error(e, "cb_topk_noalloc: cudaGetSymbolAddress");
  if (g_noalloc_used < kMaxContexts) {  // beyond that many contexts: looked up every call
    g_noalloc_ctx[g_noalloc_used] = id;
    g_noalloc_ptr[g_noalloc_used] = p;
    ++g_noalloc_used;
  }
  *out = p;
  return CB_OK;
}

}  // namespace
}  // namespace cb

CB_API int cb_topk_noalloc(const double *S, uint32_t n, uint32_t k, uint32_t *idx, double *val,
                           void *stream) {
  cb::NvtxRange nvtx_range("cb_topk_noalloc");
  using namespace cb;
  if (!S || !idx || !val) return set_error(CB_ERR_ARG, "cb_topk_noalloc: null pointer");
  if (n == 0 || k == 0 || k > n)
    return set_error(CB_ERR_ARG, "cb_topk_noalloc: need 1 <= k <= n");
  if (k > CB_MAX_TOPK || topk_scratch_bytes(k) > kNoAllocScratchBytes)
    return set_error(CB_ERR_ARG,
                     "cb_topk_noalloc: k exceeds the fixed scratch capacity (CB_MAX_TOPK = 4096)");
  void *scratch = nullptr;
  int rc = noalloc_scratch(&scratch);
  if (rc != CB_OK) return rc;
  // topk_launch clears every counter and histogram in the scratch first, so
  // the previous call's contents need no clearing here.
  return topk_launch(S, n, k, idx, val, scratch, reinterpret_cast<cudaStream_t>(stream));
}
