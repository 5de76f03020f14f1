// abi.cu -- host side of the C ABI declared in include/gvegas.h: context
// lifetime, derived integrand constants, launch geometry, the per-iteration
// kernel sequence (captured once into a CUDA graph per call shape) and the
// result read-back.
#include <cuda.h>  // types only: the driver is reached through the runtime
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <tuple>
#include <utility>
#include <vector>

#include "common.cuh"
#include "integrands.cuh"
#include "kernels.h"

using gv::GState;

static_assert(GVEGAS_MAXUSERPARAMS == gv::kNumDerived, "user parameters fill the derived-constant block");

namespace {

thread_local std::string g_thread_err;

std::string vformat(const char* fmt, va_list ap) {
  char buf[512];
  va_list ap2;
  va_copy(ap2, ap);
  const int n = vsnprintf(buf, sizeof buf, fmt, ap);
  if (n < (int)sizeof buf) {
    va_end(ap2);
    return std::string(buf);
  }
  std::string big((size_t)n + 1, '\0');
  vsnprintf(&big[0], big.size(), fmt, ap2);
  va_end(ap2);
  big.resize((size_t)n);
  return big;
}

// Allocation wrappers.  g_alloc_left: allocations still allowed before an
// injected failure (-1: none armed); the failing call returns
// cudaErrorMemoryAllocation without calling the allocator and disarms.
std::atomic<long long> g_alloc_left{-1};
std::atomic<unsigned long long> g_alloc_count{0};

bool injected_failure() {
  long long left = g_alloc_left.load();
  while (left >= 0)
    if (g_alloc_left.compare_exchange_weak(left, left - 1)) return left == 0;
  return false;
}

}  // namespace

extern "C" cudaError_t gv_dev_malloc(void** p, size_t bytes) {
  g_alloc_count.fetch_add(1);
  if (injected_failure()) {
    *p = nullptr;
    return cudaErrorMemoryAllocation;
  }
  return cudaMalloc(p, bytes);
}

extern "C" cudaError_t gv_host_malloc(void** p, size_t bytes) {
  g_alloc_count.fetch_add(1);
  if (injected_failure()) {
    *p = nullptr;
    return cudaErrorMemoryAllocation;
  }
  return cudaMallocHost(p, bytes);
}

extern "C" void vegas_fail_alloc_after(int64_t n) { g_alloc_left.store(n < 0 ? -1 : (long long)n); }

extern "C" uint64_t vegas_alloc_count(void) { return (uint64_t)g_alloc_count.load(); }

struct vegas_ctx {
  vegas_config cfg{};
  int kind = 0;
  std::vector<double> params;            // integrand parameters as given
  double derived[gv::kNumDerived] = {};  // device constants (see integrands.cuh)
  double scale = 1.0;                    // output scale applied in k_reduce
  int prec = VG_FP64;
  int ybits = 53;
  int g = 1;
  uint64_t ncubes = 1, nc = 0;
  uint32_t cube_mul = 1;  // order of the cubes (gv::cube_of)
  int strat = 0;
  gv::KernelEntry ke{};
  const void* col = nullptr;  // the column-histogram kernel of this shape, or null
  int sm_count = 0;
  // launch geometry: threads per CTA asked for (0: automatic) and CTAs per SM;
  // those of the passes without bins, where the autotuner set them apart
  int threads_req = 0, ctas_per_sm_req = 0, frozen_req = 0;
  int cap = 0;  // histogram bucket capacity (see sample_kernel.cuh; 0: column histogram)
  int ppt = 1, ppt_req = 0, ppt_min = 1;  // points per thread per histogram tile
  bool small_cap = false;                 // tile capacity policy (gv::choose_tile)
  gv::PassShape pass_bins, pass_nobins;   // passes with and without the per-bin sums
  // device buffers
  double* d_edges = nullptr;
  double2* d_tab64 = nullptr;
  float2* d_tab32 = nullptr;
  double* d_derived = nullptr;
  double* d_part_bins = nullptr;
  double* d_part_tot = nullptr;
  double2* d_cube_part = nullptr;  // sums of the hypercubes' parts
  size_t part_bins_len = 0, part_tot_len = 0, cube_part_len = 0;  // bytes
  double* d_bins = nullptr;    // behind the edges, in their allocation
  double* d_cubes = nullptr;
  double* d_cube_max = nullptr;  // [G] max(0, largest w) per cube, integration phase
  bool have_max = false;         // a bases_integrate has recorded the maxima
  // SPRING buffers (grown on demand)
  uint64_t* d_q = nullptr;
  uint64_t* d_prefix = nullptr;
  double* d_mt = nullptr;          // [G] cube bounds q_c / scale
  float* d_mt32 = nullptr;         // [G] the same in FP32
  uint32_t* d_guide = nullptr;     // guide table of the cube search
  double* d_bmax = nullptr;        // per-block maxima and sums of the table kernels
  unsigned long long* d_bsum = nullptr;
  double* d_meta = nullptr;        // {Q, scale, status}
  double* d_stage_x = nullptr;     // [n][d]
  uint64_t* d_stage_t = nullptr;   // [n]
  double* d_out_x = nullptr;
  uint64_t* d_out_t = nullptr;
  uint32_t* d_counts = nullptr;
  unsigned long long* d_counters = nullptr;
  uint32_t spring_cap = 0, spring_out_cap = 0;
  void* h_spring = nullptr;  // SpringOutcome (pinned)
  cudaEvent_t spring_timer[2] = {nullptr, nullptr};  // set by spring_profile around the trial kernel
  double* d_gpart = nullptr;  // adjoint partials [grad_nt + 2][grad_ctas] then totals
  int grad_ctas = 0;
  size_t grad_smem = 0;
  GState* d_st = nullptr;
  // pinned host memory: the state's mirror (only the fields before `hist`)
  // and the staging buffer
  GState* h_st = nullptr;
  double* h_stage = nullptr;
  size_t h_stage_len = 0;
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  // graph cache, keyed by (shape, n1, n2, refine, acc1, acc2)
  std::map<std::tuple<int, int, int, int, double, double>, cudaGraphExec_t> graphs;
  int hist_upper = 0;  // upper bound of the window length (host shadow)
  std::string err;

  vegas_status fail(vegas_status st, const char* fmt, ...) {
    va_list ap;
    va_start(ap, fmt);
    err = vformat(fmt, ap);
    va_end(ap);
    g_thread_err = err;
    return st;
  }
};

namespace {

vegas_status thread_fail(vegas_status st, const char* fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  g_thread_err = vformat(fmt, ap);
  va_end(ap);
  return st;
}

#define CK(ctx, call)                                                                  \
  do {                                                                                 \
    cudaError_t e_ = (call);                                                           \
    if (e_ != cudaSuccess)                                                             \
      return (ctx)->fail(e_ == cudaErrorMemoryAllocation ? VEGAS_ENOMEM : VEGAS_ECUDA, \
                         "%s: %s (%s:%d)", #call, cudaGetErrorString(e_), __FILE__,    \
                         __LINE__);                                                    \
  } while (0)

bool lookup_kernel(int kind, int prec, int ybits, int d, gv::KernelEntry* e) {
  const bool y24 = ybits == 24;
  switch (kind) {
    case VG_GENZ_GAUSSIAN:
      return y24 ? gv::entries_genz_gaussian_y24(prec, d, e) : gv::entries_genz_gaussian_y53(prec, d, e);
    case VG_GENZ_PRODUCT_PEAK:
      return y24 ? gv::entries_genz_product_peak_y24(prec, d, e) : gv::entries_genz_product_peak_y53(prec, d, e);
    case VG_GENZ_CORNER_PEAK:
      return y24 ? gv::entries_genz_corner_peak_y24(prec, d, e) : gv::entries_genz_corner_peak_y53(prec, d, e);
    case VG_GENZ_OSCILLATORY:
      return y24 ? gv::entries_genz_oscillatory_y24(prec, d, e) : gv::entries_genz_oscillatory_y53(prec, d, e);
    case VG_DOUBLE_GAUSSIAN:
      return y24 ? gv::entries_dgauss_y24(prec, d, e) : gv::entries_dgauss_y53(prec, d, e);
    case VG_RAMBO_BW:
      return y24 ? gv::entries_rambo_y24(prec, d, e) : gv::entries_rambo_y53(prec, d, e);
    case VG_W_MUNU:
      return y24 ? gv::entries_wmunu_y24(prec, d, e) : gv::entries_wmunu_y53(prec, d, e);
    case VG_GENZ_CONTINUOUS:
      return y24 ? gv::entries_genz_continuous_y24(prec, d, e) : gv::entries_genz_continuous_y53(prec, d, e);
    case VG_GENZ_DISCONTINUOUS:
      return y24 ? gv::entries_genz_discontinuous_y24(prec, d, e)
                 : gv::entries_genz_discontinuous_y53(prec, d, e);
    default: return false;
  }
}

void destroy_graphs(vegas_ctx* c) {
  for (auto& kv : c->graphs) cudaGraphExecDestroy(kv.second);
  c->graphs.clear();
}

// Launch geometry: a persistent grid of CTAs per SM as occupancy allows
// (or as requested), capped by the work available.
// SPRING table, in four small kernels over blocks of kSpan cubes (every
// FP64 operation of a cube is the oracle's, in the oracle's order; the
// integer sums are exact in any order):
//   k_spring_max      per-block maxima of M_c = cmax_c * out_scale;
//   k_spring_weights  M = the largest M_c, scale = 2^24 / M,
//                     q_c = ceil(M_c scale), the bound mt_c = q_c / scale,
//                     per-block sums of q;
//   k_spring_scan     (one block) exclusive scan of the block sums,
//                     P[G] = Q, meta = {Q, scale, status} (status 1: no
//                     positive maximum);
//   k_spring_prefix   exclusive prefix sums P[0..G) in 64-bit integers;
//   k_spring_guide    the guide table (Chen and Asau): for each of the 2^gk
//                     equal intervals of [0, Q), guide[j] = the last cube c
//                     with P[c] <= floor(j Q / 2^gk); guide[2^gk] = G - 1.
constexpr int kSpanThreads = 256, kSpanPer = 4;
constexpr uint32_t kSpan = kSpanThreads * kSpanPer;  // cubes per block

__device__ double block_max_d(double m, double* sm) {
  for (int off = 16; off > 0; off >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, off));
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = m;
  __syncthreads();
  double M = 0.0;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) M = fmax(M, sm[w]);
  return M;
}

__global__ void __launch_bounds__(kSpanThreads) k_spring_max(const double* cmax, uint32_t G, double out_scale,
                                                             double* bmax) {
  __shared__ double sm[32];
  const uint32_t lo = blockIdx.x * kSpan, hi = min(lo + kSpan, G);
  double m = 0.0;
  for (uint32_t i = lo + threadIdx.x; i < hi; i += blockDim.x) m = fmax(m, cmax[i] * out_scale);
  m = block_max_d(m, sm);
  if (threadIdx.x == 0) bmax[blockIdx.x] = m;
}

// The largest of the block maxima (any order: max is exact).
__device__ double spring_global_max(const double* bmax, uint32_t nb, double* sm) {
  double m = 0.0;
  for (uint32_t i = threadIdx.x; i < nb; i += blockDim.x) m = fmax(m, bmax[i]);
  return block_max_d(m, sm);
}

__global__ void __launch_bounds__(kSpanThreads) k_spring_weights(const double* cmax, uint32_t G, double out_scale,
                                                                 const double* bmax, uint32_t nb, uint64_t* q,
                                                                 double* mt, float* mt32, unsigned long long* bsum) {
  __shared__ double sm[32];
  __shared__ unsigned long long ss[32];
  const double M = spring_global_max(bmax, nb, sm);
  if (!(M > 0.0) || !isfinite(M)) return;  // k_spring_scan reports it
  const double scale = 16777216.0 / M;
  const uint32_t lo = blockIdx.x * kSpan, hi = min(lo + kSpan, G);
  unsigned long long sum = 0;
  for (uint32_t i = lo + threadIdx.x; i < hi; i += blockDim.x) {
    const double v = cmax[i] * out_scale;
    const uint64_t qi = v > 0.0 ? (uint64_t)ceil(v * scale) : 0ull;
    q[i] = qi;
    const double b = (double)qi / scale;  // the cube's bound in the integrand's units
    mt[i] = b;
    mt32[i] = (float)b;
    sum += qi;
  }
  for (int off = 16; off > 0; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
  if ((threadIdx.x & 31) == 0) ss[threadIdx.x >> 5] = sum;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long t = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += ss[w];
    bsum[blockIdx.x] = t;
  }
}

__global__ void __launch_bounds__(1024) k_spring_scan(const double* bmax, uint32_t nb, unsigned long long* bsum,
                                                      uint32_t G, uint64_t* prefix, double* meta) {
  __shared__ double sm[32];
  __shared__ unsigned long long ssum[1024];
  const double M = spring_global_max(bmax, nb, sm);
  const int tid = threadIdx.x, nt = blockDim.x;
  if (!(M > 0.0) || !isfinite(M)) {
    if (tid == 0) {
      meta[0] = 0.0;
      meta[1] = 0.0;
      meta[2] = 1.0;
    }
    return;
  }
  // exclusive scan of bsum[0..nb) in place: contiguous runs per thread
  const uint32_t per = (nb + nt - 1) / nt, lo = min((uint32_t)tid * per, nb), hi = min(lo + per, nb);
  unsigned long long sum = 0;
  for (uint32_t i = lo; i < hi; ++i) sum += bsum[i];
  ssum[tid] = sum;
  __syncthreads();
  if (tid == 0) {
    unsigned long long run = 0;
    for (int k = 0; k < nt; ++k) {
      const unsigned long long v = ssum[k];
      ssum[k] = run;
      run += v;
    }
    prefix[G] = run;
    meta[0] = (double)run;
    meta[1] = 16777216.0 / M;
    meta[2] = 0.0;
  }
  __syncthreads();
  unsigned long long run = ssum[tid];
  for (uint32_t i = lo; i < hi; ++i) {
    const unsigned long long v = bsum[i];
    bsum[i] = run;
    run += v;
  }
}

__global__ void __launch_bounds__(kSpanThreads) k_spring_prefix(const uint64_t* q, uint32_t G,
                                                                const unsigned long long* boff, uint64_t* prefix,
                                                                const double* meta) {
  __shared__ unsigned long long sw[32];
  if (meta[2] != 0.0) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t lo = blockIdx.x * kSpan + (uint32_t)tid * kSpanPer;
  uint64_t v[kSpanPer];
  unsigned long long s = 0;
#pragma unroll
  for (int k = 0; k < kSpanPer; ++k) {
    v[k] = lo + k < G ? q[lo + k] : 0ull;
    s += v[k];
  }
  // exclusive scan of the thread sums: within the warp, then over the warps
  unsigned long long inc = s;
  for (int off = 1; off < 32; off <<= 1) {
    const unsigned long long o = __shfl_up_sync(0xffffffffu, inc, off);
    if (lane >= off) inc += o;
  }
  if (lane == 31) sw[warp] = inc;
  __syncthreads();
  unsigned long long run = boff[blockIdx.x] + inc - s;
  for (int w = 0; w < warp; ++w) run += sw[w];
#pragma unroll
  for (int k = 0; k < kSpanPer; ++k) {
    const uint32_t i = lo + k;
    if (i < G) prefix[i] = run;
    run += v[k];
  }
}

// One guide entry per thread: the interval start b_j = floor(j Q / 2^gk)
// from the 128-bit product, then the last cube with P[c] <= b_j by
// bisection (P[0] = 0 <= b_j always).
__global__ void __launch_bounds__(256) k_spring_guide(const uint64_t* prefix, uint32_t G, uint32_t gk,
                                                      uint32_t* guide, const double* meta) {
  if (meta[2] != 0.0) return;
  const uint32_t j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j > (1u << gk)) return;
  const uint64_t Q = prefix[G];
  const uint64_t plo = (uint64_t)j * Q, phi = __umul64hi((uint64_t)j, Q);
  const uint64_t b = gk ? ((phi << (64 - gk)) | (plo >> gk)) : plo;
  uint32_t lo = 0, hi = G;
  while (hi - lo > 1) {
    const uint32_t mid = lo + ((hi - lo) >> 1);
    if (prefix[mid] <= b)
      lo = mid;
    else
      hi = mid;
  }
  guide[j] = lo;
}

// What the host reads of a SPRING call (pinned memory, written by the
// compaction kernel's last block).
struct SpringOutcome {
  unsigned long long events, overflow, nonpos;
  double status;  // meta[2]
};

// SPRING compaction: block k copies chunk k's kept points behind those of
// chunks 0 .. k-1 (trial order).  ox and ot, either of which may be null, are
// the caller's own buffers where the GPU can write them (pinned memory): the
// events then cross to the host once, while they are compacted, and nothing
// waits for their number first.
__global__ void k_spring_compact(const uint32_t* counts, uint32_t chunk, int d, const double* sx, const uint64_t* st,
                                 double* ox, uint64_t* ot, const double* meta, const unsigned long long* counters,
                                 SpringOutcome* outcome) {
  __shared__ unsigned long long part[32];
  const uint32_t k = blockIdx.x;
  unsigned long long o = 0;
  for (uint32_t i = threadIdx.x; i < k; i += blockDim.x) o += counts[i];
  for (int off = 16; off > 0; off >>= 1) o += __shfl_xor_sync(0xffffffffu, o, off);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = o;
  __syncthreads();
  unsigned long long off = 0;
  for (uint32_t w = 0; w < blockDim.x / 32; ++w) off += part[w];
  const uint32_t n = counts[k];
  const size_t src = (size_t)k * chunk;
  if (meta[2] == 0.0) {
    if (ox)
      for (uint32_t i = threadIdx.x; i < n * (uint32_t)d; i += blockDim.x) ox[off * d + i] = sx[src * d + i];
    if (ot)
      for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) ot[off + i] = st[src + i];
  }
  if (k == gridDim.x - 1 && threadIdx.x == 0) {
    outcome->events = off + n;
    outcome->overflow = counters[0];
    outcome->nonpos = counters[1];
    outcome->status = meta[2];
  }
}

// The address under which the GPU may write the caller's host buffer [p, p +
// bytes), or null where the events must go through device memory and a copy:
// pageable memory, a start that is not a multiple of `align` (the kernel
// stores whole elements; a copy takes any address), or a buffer that does not
// lie inside one pinned allocation.  The driver names the allocation's range:
// under unified addressing two separate pinned allocations can have pageable
// memory between them at addresses that look contiguous.
void* device_view(void* p, size_t bytes, size_t align) {
  using Query = CUresult (*)(void*, CUpointer_attribute, CUdeviceptr);
  static const Query query = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult r;
    const cudaError_t e = cudaGetDriverEntryPointByVersion("cuPointerGetAttribute", &f, 12000, cudaEnableDefault, &r);
    if (e != cudaSuccess) cudaGetLastError();
    return reinterpret_cast<Query>(e == cudaSuccess && r == cudaDriverEntryPointSuccess ? f : nullptr);
  }();
  if (!query || reinterpret_cast<uintptr_t>(p) % align != 0) return nullptr;
  cudaPointerAttributes a{};
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  if (a.type != cudaMemoryTypeHost || !a.devicePointer || reinterpret_cast<uintptr_t>(a.devicePointer) % align != 0)
    return nullptr;
  const CUdeviceptr at = reinterpret_cast<CUdeviceptr>(a.devicePointer);
  CUdeviceptr base = 0;
  size_t size = 0;
  if (query(&base, CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, at) != CUDA_SUCCESS ||
      query(&size, CU_POINTER_ATTRIBUTE_RANGE_SIZE, at) != CUDA_SUCCESS)
    return nullptr;
  return at >= base && bytes <= size && at - base <= size - bytes ? a.devicePointer : nullptr;
}

// Shape of the column-histogram pass (col_hist.cuh): `threads` threads per
// CTA, or, when 0, one CTA of as many warps as the columns' shared memory
// allows (16 at up to 50 bins, the most the registers allow; one wide CTA
// folds into one partial row: at 72 bins 11 warps in one CTA beat 10 in
// five, 65 against 70 us at d = 8).  A small pass takes narrower CTAs until
// every SM has one, but wide enough that the CTA's threads cover the cells they
// clear and fold, 128 or 256 (us per pass of 1000 points with 64 threads -> so:
// d = 4, 50 bins 17.7 -> 16.9, d = 15, 50 bins 25.9 -> 23.2, d = 20, 80 bins
// 38.0 -> 33.0).
//
// False, and the pass takes bucketed tiles, when threads == 0 and fewer than
// kColMinWarps warps of columns fit an SM (8 fit up to 109 bins at d = 2, 105 at
// 8, 103 at 16, 95 at 32): us per pass of 2^22 points at 100 bins, columns
// against the best tile: d = 4 43.9 / 47.1, d = 7 115.6 / 119.6, d = 8 66 / 93,
// d = 16 119 / 206.  And, unstratified with more than 50 bins (fewer than 16
// warps), for passes too small to pay for clearing and folding the columns (one
// or two axes have little to fold).  Columns over tiles, measured at 80 bins:
//   d (exact)      4     8    16   |  d (run-time) 3     6     7    9    12    15
//   10^5 points   .98  1.08  1.12  |             1.09  1.10  1.18 1.17  1.15  1.09
//   4 10^5        .95  1.00   .98  |             1.00  1.08  1.04 1.08  1.01   .87
//   2^20          .92   .87   .84  |             1.09  1.04   .97 1.01   .97   .76
//   2^22                .79   .76  |             1.09  1.04   .93       .92   .69
// so from n d = 2 10^6 on where the kernel knows the dimension, and from 6 10^6
// with at least 7 axes where it does not (beyond 16 axes, where tiles keep one
// small CTA per SM, from 2 10^6 again: 1.2 10^5 points d = 17, 64 bins, tiles 5.2
// us, columns 4.7; 8.3 10^4, d = 24, 80 bins, 5.5 and 5.0; 6.7 10^4, d = 30, 60
// bins, 4.95 and 5.2; 2 10^5, d = 24, 80 bins, 63 and 51 per evaluation).
constexpr int kColMinWarps = 8;
// Static shared memory of k_sample, at most (its dynamic part must leave room).
constexpr size_t kSampleStatic = 1024;
bool cols_pay(bool exact, int d, int N, uint64_t ncubes, uint64_t ncall) {
  if (ncubes > 1 || N <= 50 || d <= 2) return true;
  return exact || d > 16 ? ncall * (uint64_t)d >= 2000000u : d >= 7 && ncall * (uint64_t)d >= 6000000u;
}
bool shape_col(const void* fn, const gv::KernelEntry& ke, int d, int N, int sm_count, int threads, int per_sm_req,
               uint64_t ncubes, uint64_t nc, uint64_t ncall, int64_t max_rows, uint64_t max_parts,
               gv::PassShape* out, cudaError_t* e) {
  // A shape whose smallest buckets do not fit has columns or nothing.
  const bool tiles = ke.smem(d, N, 4) + kSampleStatic <= 227 * 1024;
  // (2 KB: the kernel's static shared memory)
  auto fits = [&](int warps) { return ke.smem_col(d, N, warps) + 2048 <= 227 * 1024; };
  int best_t = threads;
  if (threads == 0) {
    if (tiles && !cols_pay(fn == ke.sample_col_exact, d, N, ncubes, ncall)) return false;
    int warps = 16;
    while (warps >= kColMinWarps && !fits(warps)) --warps;
    best_t = 32 * warps;
    if (warps < kColMinWarps) return false;
  }
  if (!fits(best_t / 32)) return false;
  const size_t smem = ke.smem_col(d, N, best_t / 32);
  if ((*e = gv_raise_smem_limit(fn, smem)) != cudaSuccess) return false;
  int best_occ = 0;
  if ((*e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&best_occ, fn, best_t, smem)) != cudaSuccess) return false;
  if (per_sm_req > 0) best_occ = std::min(best_occ, per_sm_req);
  if (best_occ < 1) return false;
  const int pif = d <= 8 ? 2 : 1;
  if (threads == 0) {
    const uint64_t per = (ncall + (uint64_t)sm_count * pif - 1) / ((uint64_t)sm_count * pif);
    if (per < (uint64_t)best_t) {
      const uint64_t least = d * N <= 400 ? 128 : 256;
      best_t = (int)std::min<uint64_t>(best_t, (std::max(per, least) + 31) / 32 * 32);
      best_occ = 1;
    }
  }
  out->fn = fn;
  out->threads = best_t;
  out->occ = best_occ;
  out->smem = ke.smem_col(d, N, best_t / 32);
  const int64_t most = std::min<int64_t>((int64_t)sm_count * best_occ, max_rows);
  const gv::CubeLanes cl =
      ncubes > 1 ? gv::balanced_lanes(ncubes, nc, best_t, sm_count, pif, max_parts) : gv::CubeLanes{1, 1};
  out->lanes = cl.lanes;
  out->parts = cl.parts;
  const uint64_t units = ncubes > 1 ? ncubes * cl.parts * (uint64_t)cl.lanes : ncall;
  out->ctas = (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)((units + best_t - 1) / best_t), most));
  return true;
}

// Launch shapes of both kinds of pass and the buffers they need.  The context
// changes only where all of it succeeds: new buffers are allocated before the
// old ones go, and the graphs, which hold the old addresses, go first.  (The
// stream is idle here.)
vegas_status configure_launch(vegas_ctx* c) {
  int threads = c->threads_req > 0 ? c->threads_req : 256;
  const int d = c->cfg.ndim, N = c->cfg.nbins;
  gv::PassShape pb, pn;
  int cap = 0, ppt = 1;
  const bool strat = c->strat != 0;
  cudaError_t e = cudaSuccess;
  auto ctas_for = [&](const gv::PassShape& s, int t, int64_t most) {
    const uint64_t units = strat ? c->ncubes * (uint64_t)s.lanes * s.parts : (uint64_t)c->cfg.ncall;
    return (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)((units + t - 1) / t), most));
  };
  int per_sm = 1;
  if (c->col && c->ppt_req == 0 &&
      shape_col(c->col, c->ke, d, N, c->sm_count, c->threads_req, c->ctas_per_sm_req, c->ncubes, c->nc,
                (uint64_t)c->cfg.ncall, INT64_MAX, gv::kMaxCubeParts, &pb, &e)) {
    ppt = d <= 8 ? 2 : 1;
    per_sm = std::max(1, pb.occ);
  } else {
    // Histogram tile (gv::choose_tile): points per thread between gathers and
    // bucket capacity, against the CTAs per SM each leaves resident.
    auto occ_of = [&](int cp, int) -> int {
      const size_t smem = c->ke.smem(d, N, cp);
      int o = 0;
      if (e != cudaSuccess || smem + kSampleStatic > 227 * 1024) return 0;
      e = gv_raise_smem_limit(c->ke.sample, smem);
      if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, c->ke.sample, threads, smem);
      return e == cudaSuccess ? o : 0;
    };
    int occ_cap = 0;
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ_cap, c->ke.sample, threads, 0);
    if (e != cudaSuccess) return c->fail(VEGAS_ECUDA, "launch configuration: %s", cudaGetErrorString(e));
    gv::TileShape t = gv::choose_tile(threads, N, c->ppt_req, c->ppt_min, occ_cap, occ_of, c->small_cap);
    // Few points: the same number of rounds with CTAs just wide enough, so
    // that every SM runs the same number of warps (10^5 points over 456 CTAs:
    // 224 threads, 21 warps per SM, instead of 391 CTAs of 256, up to 24).
    // Where warps are what an SM runs short of, that is FP64 points and FP64
    // sums of 8 or more axes, and only a little narrower: set-up and
    // finishing go by CTAs (us per pass with 256 threads -> so: FP64 53 bits
    // d = 8, 2 10^5 points, 224 threads 65.9 -> 57.5; d = 16, 10^5, 224 69.3 ->
    // 59.8; d = 6, 10^5, 192 41.9 -> 39.5; but 3 10^4, 128 27.0 -> 28.7; FP64 sums
    // d = 8, 2 10^5, 224 44.1 -> 39.7, but d = 4 33.0 -> 35.8; FP32 sums 53 bits
    // d = 16, 4 10^5, 224 47.9 -> 52.9), narrower yet where one CTA is all that
    // fits (d = 8, 256 bins, 9 10^4: 218 -> 182 per four iterations).
    // And where few bins would overflow their buckets (64 slots): narrower at
    // any rate (2 bins, d = 7, 2 10^4 points: 217 us per four iterations with
    // 256 threads, 98 so; FP64, d = 9, 4 10^4: 283 and 171).
    int narrowest = c->prec == VG_FP64 ? 160 : 256;
    if (c->prec == VG_FP32_ACC64) narrowest = t.occ == 1 ? 160 : (d >= 8 ? 224 : 256);
    if (threads > 40 * N) narrowest = 64;
    if (e == cudaSuccess && c->threads_req == 0 && !strat && t.occ > 0) {
      const uint64_t n = (uint64_t)c->cfg.ncall, most = (uint64_t)c->sm_count * t.occ;
      const uint64_t rounds = (n + most * threads - 1) / (most * threads);
      const int w = (int)(((n + most * rounds - 1) / (most * rounds) + 31) / 32 * 32);
      if (w >= narrowest && w < threads) {
        const int wide = threads;
        threads = w;
        const gv::TileShape u = gv::choose_tile(threads, N, c->ppt_req, c->ppt_min, occ_cap, occ_of, c->small_cap);
        if (u.occ >= t.occ && u.ppt >= t.ppt)  // (a shorter tile costs more than even rounds give)
          t = u;
        else
          threads = wide;
      }
    }
    if (e != cudaSuccess) return c->fail(VEGAS_ECUDA, "launch configuration: %s", cudaGetErrorString(e));
    if (t.occ < 1) return c->fail(VEGAS_EINVAL, "sampling kernel does not fit: %d threads, %d points per thread",
                                  threads, t.ppt);
    pb.fn = c->ke.sample;
    pb.threads = threads;
    pb.occ = t.occ;
    // the limit covers the chosen size (it only grows: see gv_raise_smem_limit)
    pb.smem = c->ke.smem(d, N, t.cap);
    e = gv_raise_smem_limit(c->ke.sample, pb.smem);
    if (e != cudaSuccess) return c->fail(VEGAS_ECUDA, "launch configuration: %s", cudaGetErrorString(e));
    cap = t.cap;
    ppt = t.ppt;
    per_sm = c->ctas_per_sm_req > 0 ? std::min(c->ctas_per_sm_req, t.occ) : t.occ;
    const int64_t most = (int64_t)c->sm_count * per_sm;
    pb.lanes = strat ? gv::choose_lanes(c->ncubes, c->nc, threads, most) : 1;
    pb.parts = 1;
    if (pb.lanes == 32) {  // few cubes: several groups each
      const gv::CubeLanes cl = gv::balanced_lanes(c->ncubes, c->nc, threads, c->sm_count, c->ppt_min, gv::kMaxCubeParts);
      pb.parts = cl.parts;
    }
    pb.ctas = ctas_for(pb, threads, most);
  }
  threads = c->frozen_req > 0 ? c->frozen_req : (c->threads_req > 0 ? c->threads_req : 256);
  // passes without the per-bin histogram (no refinement) need only the
  // grid table and constants in shared memory: more CTAs may be resident
  pn.fn = c->ke.frozen;
  pn.threads = threads;
  pn.smem = c->ke.smem_nobins(d, N);
  int occ_nb = 0;
  e = gv_raise_smem_limit(pn.fn, pn.smem);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ_nb, pn.fn, threads, pn.smem);
  if (e != cudaSuccess) return c->fail(VEGAS_ECUDA, "launch configuration: %s", cudaGetErrorString(e));
  if (c->ctas_per_sm_req > 0) occ_nb = std::min(occ_nb, std::max(c->ctas_per_sm_req, per_sm));
  // 32 warps hide the latencies; more CTAs only add rows of totals (each
  // ends in dependent reductions) and set-up (64 threads, d = 7, 72 bins: 36.0 us
  // per pass against 40.0 with all that fit)
  pn.occ = std::max(1, std::min(occ_nb, std::max(32 * 32 / threads, per_sm)));
  const int64_t most_nb = (int64_t)c->sm_count * pn.occ;
  // (without the histogram a cube's parts cost more, in their merge and in the
  // groups' own reductions, than even rounds give, until a quarter of the SMs
  // would idle: 6561 cubes of 300, d = 8, 85.6 us per call with parts, 78.4
  // without; 729 of 1438, d = 6, 45 and 63)
  const uint64_t max_parts = c->ncubes * 128 < (uint64_t)threads * c->sm_count * 3 ? gv::kMaxCubeParts : 0;
  const gv::CubeLanes cl = strat ? gv::balanced_lanes(c->ncubes, c->nc, threads, c->sm_count, c->ppt_min, max_parts)
                                 : gv::CubeLanes{1, 1};
  pn.lanes = cl.lanes;
  pn.parts = cl.parts;
  pn.ctas = ctas_for(pn, threads, most_nb);
  // partial rows (of the passes that keep bins), totals per CTA and
  // iteration, and the sums of the hypercubes' parts (a refining pass's, or
  // those of a frozen-grid launch's iterations)
  struct Buffer {
    void** p;
    size_t* have;
    size_t need;
    void* fresh;
  } buffers[3] = {
      {(void**)&c->d_part_bins, &c->part_bins_len, sizeof(double) * 2 * (size_t)d * N * pb.ctas, nullptr},
      {(void**)&c->d_part_tot, &c->part_tot_len,
       sizeof(double) * gv::kTotCols * gv::kMergeIters * (size_t)std::max(pb.ctas, pn.ctas), nullptr},
      {(void**)&c->d_cube_part, &c->cube_part_len,
       16 * std::max(pb.parts > 1 ? (size_t)c->ncubes * pb.parts : 0,
                     pn.parts > 1 ? (size_t)c->ncubes * pn.parts * gv::kMergeIters : 0),
       nullptr}};
  for (Buffer& b : buffers) {
    if (b.need <= *b.have || (e = gv_dev_malloc(&b.fresh, b.need)) == cudaSuccess) continue;
    for (Buffer& o : buffers) cudaFree(o.fresh);
    return c->fail(e == cudaErrorMemoryAllocation ? VEGAS_ENOMEM : VEGAS_ECUDA, "cudaMalloc(%zu): %s", b.need,
                   cudaGetErrorString(e));
  }
  destroy_graphs(c);
  for (Buffer& b : buffers)
    if (b.fresh) {
      cudaFree(*b.p);
      *b.p = b.fresh;
      *b.have = b.need;
    }
  c->pass_bins = pb;
  c->pass_nobins = pn;
  c->cap = cap;
  c->ppt = ppt;
  return VEGAS_OK;
}

gv::SampleArgs sample_args(const vegas_ctx* c, int it_override, bool nobins = false, int niter = 1) {
  gv::SampleArgs A{};
  const gv::PassShape& ps = nobins ? c->pass_nobins : c->pass_bins;
  A.d = c->cfg.ndim;
  A.N = c->cfg.nbins;
  A.g = c->g;
  A.ybits = c->ybits;
  A.lanes = ps.lanes;
  A.parts = ps.parts;
  A.units = (uint32_t)c->ncubes * ps.parts;
  A.vl = (uint32_t)ps.lanes * ps.parts;
  A.per_lane = c->strat ? (uint32_t)((c->nc + A.vl - 1) / A.vl) : 0;
  A.niter = niter;
  A.cube_part = c->d_cube_part;
  A.cap = c->cap;
  A.ppt = c->ppt;
  A.strat = c->strat;
  A.key0 = (uint32_t)c->cfg.seed;
  A.key1 = (uint32_t)(c->cfg.seed >> 32);
  gv::philox_key_schedule(A.key0, A.key1, A.ks);
  A.instance = c->cfg.instance;
  A.it_override = it_override;
  A.force = it_override >= 0;
  A.ncall = (uint64_t)c->cfg.ncall;
  A.nc = (uint32_t)c->nc;
  A.ncubes = (uint32_t)c->ncubes;
  A.cube_mul = c->cube_mul;
  A.g_pow2 = (c->g & (c->g - 1)) == 0;
  A.g_log2 = 0;
  while ((1 << A.g_log2) < c->g) ++A.g_log2;
  A.t32 = (int64_t)c->g * c->cfg.nbins <= 256;
  const double gb = (double)c->g * std::ldexp(1.0, c->ybits);
  A.inv_gb_d = 1.0 / gb;
  A.inv_gb_f = (float)(1.0 / gb);
  A.inv_nc = c->nc > 0 ? 1.0 / (double)c->nc : 0.0;
  A.inv_nc1 = c->nc > 1 ? 1.0 / (double)(c->nc - 1) : 0.0;
  A.nparts = ps.ctas;
  A.tab = c->prec == VG_FP64 ? (const void*)c->d_tab64 : (const void*)c->d_tab32;
  A.dparams = c->d_derived;
  A.st = c->d_st;
  A.part_bins = c->d_part_bins;
  A.part_tot = c->d_part_tot;
  A.cubes = c->d_cubes;
  return A;
}

gv::FinArgs fin_args(const vegas_ctx* c, int refine, int record, bool nobins = false, bool combine = true,
                     int niter = 1) {
  gv::FinArgs F{};
  F.niter = niter;
  F.parts = (nobins ? c->pass_nobins : c->pass_bins).parts;
  F.cube_mul = c->cube_mul;
  F.inv_nc = c->nc > 0 ? 1.0 / (double)c->nc : 0.0;
  F.inv_nc1 = c->nc > 1 ? 1.0 / (double)(c->nc - 1) : 0.0;
  F.cube_part = c->d_cube_part;
  F.cubes = c->d_cubes;
  F.combine = combine;
  F.d = c->cfg.ndim;
  F.N = c->cfg.nbins;
  F.nobins = nobins;
  F.nparts = (nobins ? c->pass_nobins : c->pass_bins).ctas;
  F.strat = c->strat;
  F.refine = refine;
  F.record = record;
  F.pair32 = c->prec == VG_FP32_ACCCOMP;
  F.ncall = (uint64_t)c->cfg.ncall;
  F.ncubes = c->ncubes;
  F.scale = c->d_derived + gv::kNumDerived;
  F.alpha = c->cfg.alpha;
  F.part_bins = c->d_part_bins;
  F.part_tot = c->d_part_tot;
  F.bins = c->d_bins;
  F.edges = c->d_edges;
  F.tab64 = c->d_tab64;
  F.tab32 = c->d_tab32;
  F.st = c->d_st;
  F.mirror = combine || !record ? c->h_st : nullptr;  // (a pass in the middle of a call: not read)
  return F;
}

// One pass of steps 2-6 on the context stream.  A pass that does not
// refine the grid skips the per-bin histogram, whose sums only step 5
// reads (`nobins`), unless the caller wants them, and may hold `niter`
// iterations.
// `combine`: form the combined result after it (the last pass of a call, and
// every pass of a call with an ACC target).
vegas_status launch_pass(vegas_ctx* c, int it_override, int refine, int record, bool record_max = false,
                         bool nobins = false, bool combine = true, int niter = 1) {
  if (refine) nobins = false;
  gv::SampleArgs A = sample_args(c, it_override, nobins, niter);
  if (record_max) A.cube_max = c->d_cube_max;
  void* args[] = {&A};
  const gv::PassShape& ps = nobins ? c->pass_nobins : c->pass_bins;
  CK(c, cudaLaunchKernel(ps.fn, dim3(ps.ctas, A.niter), dim3(ps.threads), args, ps.smem, c->stream));
  gv::FinArgs F = fin_args(c, refine, record, nobins, combine, niter);
  CK(c, gv_launch_finish(&F, c->stream));
  return VEGAS_OK;
}

// Graph of one call.  shape 0 (vegas_iterate): set the ACC target, then n1
// passes (refining if `refine`).  shape 1 (bases_integrate): reset the
// window, n1 refining passes at acc1, snapshot phase 1, reset, n2 frozen-grid
// passes at acc2.  Each call shape is captured once and replayed.
vegas_status get_graph(vegas_ctx* c, int shape, int n1, int n2, int refine, double acc1, double acc2,
                       cudaGraphExec_t* out) {
  auto key = std::make_tuple(shape, n1, n2, refine, acc1, acc2);
  auto itg = c->graphs.find(key);
  if (itg != c->graphs.end()) {
    *out = itg->second;
    return VEGAS_OK;
  }
  cudaGraph_t g = nullptr;
  CK(c, cudaStreamBeginCapture(c->stream, cudaStreamCaptureModeThreadLocal));
  vegas_status st = VEGAS_OK;
  auto ctl = [&](int ops, double acc) {
    if (st) return;
    cudaError_t e = gv_launch_control(c->d_st, ops, acc, 0u, c->h_st, c->stream);
    if (e != cudaSuccess) st = c->fail(VEGAS_ECUDA, "control: %s", cudaGetErrorString(e));
  };
  // n iterations on the grid as it stands.  Without an ACC target nothing is
  // decided between them, so one launch runs up to kMergeIters: no launch
  // gap and no half-empty last round per iteration.
  auto frozen = [&](int n, double acc, bool record_max) {
    for (int i = 0; i < n && !st;) {
      const int m = acc > 0.0 ? 1 : std::min(gv::kMergeIters, n - i);
      i += m;
      st = launch_pass(c, -1, 0, 1, record_max, true, acc > 0.0 || i == n, m);
    }
  };
  if (shape == 0) {
    ctl(gv::CTL_SET_ACC, acc1);
    if (refine)
      for (int i = 0; i < n1 && !st; ++i) st = launch_pass(c, -1, 1, 1, false, false, acc1 > 0.0 || i == n1 - 1);
    else
      frozen(n1, acc1, false);
  } else {
    ctl(gv::CTL_RESET_WINDOW | gv::CTL_SET_ACC, acc1);
    for (int i = 0; i < n1 && !st; ++i) st = launch_pass(c, -1, 1, 1, false, false, acc1 > 0.0 || i == n1 - 1);
    ctl(gv::CTL_SNAPSHOT | gv::CTL_RESET_WINDOW | gv::CTL_SET_ACC, acc2);
    // the integration phase records the per-cube maxima that SPRING uses
    if (!st && cudaMemsetAsync(c->d_cube_max, 0, sizeof(double) * c->ncubes, c->stream) != cudaSuccess)
      st = c->fail(VEGAS_ECUDA, "cube maxima reset");
    if (!st) frozen(n2, acc2, true);
  }
  cudaError_t e = cudaStreamEndCapture(c->stream, &g);
  if (st != VEGAS_OK) {
    if (g) cudaGraphDestroy(g);
    return st;
  }
  if (e != cudaSuccess) return c->fail(VEGAS_ECUDA, "graph capture: %s", cudaGetErrorString(e));
  cudaGraphExec_t ge = nullptr;
  e = cudaGraphInstantiate(&ge, g, 0);
  cudaGraphDestroy(g);
  if (e != cudaSuccess) return c->fail(VEGAS_ECUDA, "graph instantiate: %s", cudaGetErrorString(e));
  if (c->graphs.size() >= 64) destroy_graphs(c);
  c->graphs[key] = ge;
  *out = ge;
  return VEGAS_OK;
}

// The host's view of the state (c->h_st up to `hist`): pinned memory that the
// kernels which change the state write themselves, so only the stream is
// waited for.
vegas_status read_state(vegas_ctx* c) {
  CK(c, cudaStreamSynchronize(c->stream));
  return VEGAS_OK;
}

void fill_result(const vegas_ctx* c, vegas_result* r) {
  const GState* s = c->h_st;
  r->I = s->I;
  r->sigma = s->sigma;
  r->chi2_dof = s->chi2;
  r->iters_done = s->nhist;
  r->stopped = s->stopped;
  r->nonfinite = s->nonfinite;
  r->samples = s->samples;
}

vegas_status stage(vegas_ctx* c, size_t n) {
  if (n <= c->h_stage_len) return VEGAS_OK;
  CK(c, cudaStreamSynchronize(c->stream));  // no copy may still read the old buffer
  if (c->h_stage) cudaFreeHost(c->h_stage);
  c->h_stage = nullptr;
  c->h_stage_len = 0;
  CK(c, gv_malloc_host(&c->h_stage, n * sizeof(double)));
  c->h_stage_len = n;
  return VEGAS_OK;
}

vegas_status upload_grid(vegas_ctx* c, const double* edges) {
  const int d = c->cfg.ndim, N = c->cfg.nbins;
  const size_t n = (size_t)d * (N + 1);
  vegas_status st = stage(c, n);
  if (st) return st;
  CK(c, cudaStreamSynchronize(c->stream));  // staging buffer may still be in use
  memcpy(c->h_stage, edges, n * sizeof(double));
  CK(c, cudaMemcpyAsync(c->d_edges, c->h_stage, n * sizeof(double), cudaMemcpyHostToDevice, c->stream));
  CK(c, gv_launch_tables(c->d_edges, d, N, c->d_tab64, c->d_tab32, c->stream));
  return VEGAS_OK;  // stream-ordered; the next host write to the stage synchronises first
}

// Integrand constants and output scale as a kernel argument: the values
// travel with the launch, with no staging buffer to wait for.
struct DerivedBlock {
  double v[gv::kNumDerived + 1];  // the constants, then the output scale
};

__global__ void k_derived(const DerivedBlock b, double* dst) {
  for (int i = threadIdx.x; i <= gv::kNumDerived; i += blockDim.x) dst[i] = b.v[i];
}

vegas_status upload_derived(vegas_ctx* c) {
  DerivedBlock b;
  memcpy(b.v, c->derived, sizeof c->derived);
  b.v[gv::kNumDerived] = c->scale;
  k_derived<<<1, 128, 0, c->stream>>>(b, c->d_derived);
  CK(c, cudaGetLastError());
  return VEGAS_OK;  // stream-ordered
}

bool valid_grid(const double* e, int d, int N) {
  for (int a = 0; a < d; ++a) {
    const double* r = e + (size_t)a * (N + 1);
    if (r[0] != 0.0 || r[N] != 1.0) return false;
    for (int k = 0; k < N; ++k)
      if (!(r[k + 1] > r[k])) return false;
  }
  return true;
}

// Checks on a configuration shared by every constructor: sizes, precision,
// random bits (ybits, resolved), and the stratification g^d | ncall.
vegas_status check_config(const vegas_config* cfg, int* ybits_out, int* g_out, uint64_t* G_out) {
  const int d = cfg->ndim, N = cfg->nbins;
  if (d < 1 || d > GVEGAS_MAXDIM) return thread_fail(VEGAS_EINVAL, "ndim %d outside 1..%d", d, GVEGAS_MAXDIM);
  if (N < 2 || N > GVEGAS_MAXBINS) return thread_fail(VEGAS_EINVAL, "nbins %d outside 2..%d", N, GVEGAS_MAXBINS);
  if (cfg->ncall < 2 || cfg->ncall > (int64_t)1 << 32)
    return thread_fail(VEGAS_EINVAL, "ncall %lld outside 2..2^32", (long long)cfg->ncall);
  if (cfg->precision < VG_FP64 || cfg->precision > VG_FP32_ACCCOMP)
    return thread_fail(VEGAS_EINVAL, "unknown precision %d", cfg->precision);
  const int ybits = cfg->ybits ? cfg->ybits : (cfg->precision == VG_FP64 ? 53 : 24);
  if (ybits != 24 && ybits != 53) return thread_fail(VEGAS_EINVAL, "ybits must be 24 or 53");
  if (!(cfg->alpha >= 0.0) || !std::isfinite(cfg->alpha)) return thread_fail(VEGAS_EINVAL, "alpha must be >= 0");
  const int g = cfg->nstrat < 1 ? 1 : cfg->nstrat;
  uint64_t G = 1;
  for (int a = 0; a < d; ++a) {
    G *= (uint64_t)g;
    if (G > (uint64_t)cfg->ncall) return thread_fail(VEGAS_EINVAL, "nstrat^ndim exceeds ncall");
  }
  if ((uint64_t)cfg->ncall % G != 0) return thread_fail(VEGAS_EINVAL, "ncall must be a multiple of nstrat^ndim");
  if (G > 1 && (uint64_t)cfg->ncall / G < 2) return thread_fail(VEGAS_EINVAL, "need >= 2 points per hypercube");
  if ((int64_t)g * N >= (ybits == 53 ? 2048 : (1 << 30)))
    return thread_fail(VEGAS_EINVAL, "nstrat * nbins too large for %d-bit sampling", ybits);
  *ybits_out = ybits;
  *g_out = g;
  *G_out = G;
  return VEGAS_OK;
}

vegas_ctx* new_context(const vegas_config* cfg, int ybits, int g, uint64_t G) {
  vegas_ctx* c = new vegas_ctx();
  c->cfg = *cfg;
  c->cfg.ybits = ybits;
  c->prec = cfg->precision;
  c->ybits = ybits;
  c->g = g;
  c->ncubes = G;
  c->nc = (uint64_t)cfg->ncall / G;
  c->strat = G > 1;
  c->cube_mul = gv::cube_multiplier(G);
  return c;
}

// The specialised sampling kernel applies: d equal to the compile-time bound
// dm, 24-bit words, a power-of-two number of divisions with g N <= 256.
bool spec_shape(int d, int dm, int ybits, int g, int N) {
  return d == dm && ybits == 24 && (g & (g - 1)) == 0 && (int64_t)g * N <= 256;
}

// The column-histogram kernel of a shape (the divisions of spec_shape with
// any d up to the compile-time bound; the exact one where d equals it), or
// null.
const void* pick_col(const gv::KernelEntry& ke, int d, int ybits, int g, int N) {
  if (!spec_shape(ke.dm, ke.dm, ybits, g, N)) return nullptr;
  return d == ke.dm ? ke.sample_col_exact : ke.sample_col;
}

// Second half of every constructor, for a context whose integrand, kernel
// entry and constants are set: device buffers, launch shape, uniform grid.
vegas_status finish_create(vegas_ctx* c, vegas_ctx** out) {
  const vegas_config* cfg = &c->cfg;
  const int d = cfg->ndim, N = cfg->nbins;
  const uint64_t G = c->ncubes;
  // the specialised kernel when the shape allows it (see kernels.h)
  if (c->ke.sample_spec && spec_shape(d, c->ke.dm, c->ybits, c->g, N)) {
    c->ke.sample = c->ke.sample_spec;
    c->ke.frozen = c->ke.frozen_spec;
    c->ke.max_threads = gv::kSampleMaxThreads<true>;
    c->ppt_min = c->ke.spec_ppt_min;
    if (c->ke.grad_spec) c->ke.grad = c->ke.grad_spec;
  }
  c->col = pick_col(c->ke, d, c->ybits, c->g, N);
  auto bail = [&](vegas_status st) {
    g_thread_err = c->err;
    vegas_destroy(c);
    return st;
  };
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&c->sm_count, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return bail(c->fail(VEGAS_ECUDA, "no CUDA device: %s", cudaGetErrorString(e)));
  e = gv_prepare_aux_kernels();
  for (const void* f : {c->ke.sample, c->ke.frozen, c->col})
    if (e == cudaSuccess && f)
      e = cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
  if (e != cudaSuccess) return bail(c->fail(VEGAS_ECUDA, "kernel attributes: %s", cudaGetErrorString(e)));
  if (cfg->stream) {
    c->stream = (cudaStream_t)cfg->stream;
  } else {
    e = cudaStreamCreateWithFlags(&c->stream, cudaStreamNonBlocking);
    if (e != cudaSuccess) return bail(c->fail(VEGAS_ECUDA, "stream: %s", cudaGetErrorString(e)));
    c->own_stream = true;
  }
  auto alloc = [&](void** p, size_t bytes) -> vegas_status {
    cudaError_t ae = gv_dev_malloc(p, bytes);
    if (ae != cudaSuccess)
      return c->fail(VEGAS_ENOMEM, "cudaMalloc(%zu): %s", bytes, cudaGetErrorString(ae));
    return VEGAS_OK;
  };
  vegas_status st = VEGAS_OK;
  // edges and per-bin sums together: vegas_get_grid reads both in one copy
  if (!st) st = alloc((void**)&c->d_edges, sizeof(double) * ((size_t)d * (N + 1) + 2 * (size_t)d * N));
  if (!st) st = alloc((void**)&c->d_tab64, sizeof(double2) * d * N);
  if (!st) st = alloc((void**)&c->d_tab32, sizeof(float2) * d * N);
  if (!st) st = alloc((void**)&c->d_derived, sizeof c->derived + sizeof(double));  // + the output scale
  if (!st) c->d_bins = c->d_edges + (size_t)d * (N + 1);
  if (!st && c->strat) st = alloc((void**)&c->d_cubes, sizeof(double) * 2 * G);
  if (!st) st = alloc((void**)&c->d_cube_max, sizeof(double) * G);
  if (!st) st = alloc((void**)&c->d_st, sizeof(GState));
  if (st) return bail(st);
  const size_t head = sizeof(GState) - sizeof(c->h_st->hist);
  if (gv_malloc_host(&c->h_st, head) != cudaSuccess) return bail(c->fail(VEGAS_ENOMEM, "cudaMallocHost(state)"));
  memset(c->h_st, 0, head);
  if ((st = stage(c, (size_t)d * (N + 1) + 2 * (size_t)d * N))) return bail(st);  // (what vegas_get_grid reads)
  if (cudaMemsetAsync(c->d_st, 0, sizeof(GState), c->stream) != cudaSuccess ||
      cudaMemsetAsync(c->d_bins, 0, sizeof(double) * 2 * d * N, c->stream) != cudaSuccess)
    return bail(c->fail(VEGAS_ECUDA, "state initialisation failed"));
  if ((st = configure_launch(c))) return bail(st);
  if (c->ke.grad) {  // adjoint pass (vegas_grad): launch shape and partial rows
    c->grad_smem = c->ke.grad_smem(d, N);
    int occg = 0;
    e = gv_raise_smem_limit(c->ke.grad, c->grad_smem);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occg, c->ke.grad, 256, c->grad_smem);
    if (e != cudaSuccess) return bail(c->fail(VEGAS_ECUDA, "adjoint launch: %s", cudaGetErrorString(e)));
    const int64_t want = (cfg->ncall + 255) / 256;
    c->grad_ctas = (int)std::max<int64_t>(1, std::min<int64_t>(want, (int64_t)c->sm_count * std::max(occg, 1)));
    if ((st = alloc((void**)&c->d_gpart, sizeof(double) * (size_t)(c->ke.grad_nt + 2) * (c->grad_ctas + 1))))
      return bail(st);
  }
  e = gv_launch_uniform_grid(c->d_edges, d, N, c->d_tab64, c->d_tab32, c->stream);
  if (e != cudaSuccess) return bail(c->fail(VEGAS_ECUDA, "uniform grid: %s", cudaGetErrorString(e)));
  if ((st = upload_derived(c))) return bail(st);
  *out = c;
  return VEGAS_OK;
}

}  // namespace

extern "C" {

const char* vegas_last_error(const vegas_ctx* ctx) {
  if (ctx) return ctx->err.c_str();
  return g_thread_err.c_str();
}

void vegas_destroy(vegas_ctx* c) {
  if (!c) return;
  if (c->stream) cudaStreamSynchronize(c->stream);
  destroy_graphs(c);
  cudaFree(c->d_edges);
  cudaFree(c->d_tab64);
  cudaFree(c->d_tab32);
  cudaFree(c->d_derived);
  cudaFree(c->d_part_bins);
  cudaFree(c->d_part_tot);
  cudaFree(c->d_cube_part);
  cudaFree(c->d_cubes);
  cudaFree(c->d_cube_max);
  for (void* p : {(void*)c->d_q, (void*)c->d_mt, (void*)c->d_mt32, (void*)c->d_guide, (void*)c->d_bmax, (void*)c->d_bsum, (void*)c->d_prefix, (void*)c->d_meta, (void*)c->d_stage_x, (void*)c->d_stage_t,
                  (void*)c->d_out_x, (void*)c->d_out_t, (void*)c->d_counts, (void*)c->d_counters})
    cudaFree(p);
  cudaFree(c->d_gpart);
  cudaFree(c->d_st);
  if (c->h_st) cudaFreeHost(c->h_st);
  if (c->h_spring) cudaFreeHost(c->h_spring);
  if (c->h_stage) cudaFreeHost(c->h_stage);
  if (c->own_stream && c->stream) cudaStreamDestroy(c->stream);
  delete c;
}

vegas_status vegas_create(const vegas_config* cfg, const vegas_integrand* fn, vegas_ctx** out) {
  if (!out) return thread_fail(VEGAS_EINVAL, "out is NULL");
  *out = nullptr;
  if (!cfg || !fn) return thread_fail(VEGAS_EINVAL, "config or integrand is NULL");
  int ybits = 0, g = 1;
  uint64_t G = 1;
  vegas_status cs = check_config(cfg, &ybits, &g, &G);
  if (cs) return cs;
  const int d = cfg->ndim;
  if (fn->ndim != d) return thread_fail(VEGAS_EINVAL, "integrand ndim %d != config ndim %d", fn->ndim, d);
  const int np = gv::expected_nparams(fn->kind, d);
  if (np < 0) return thread_fail(VEGAS_EINVAL, "unknown integrand kind %d", fn->kind);
  if (fn->nparams != np || (np > 0 && !fn->params))
    return thread_fail(VEGAS_EINVAL, "integrand kind %d needs %d parameters, got %d", fn->kind, np, fn->nparams);
  vegas_ctx* c = new_context(cfg, ybits, g, G);
  c->kind = fn->kind;
  c->params.assign(fn->params, fn->params + np);
  std::string why;
  if (!gv::derive_params(fn->kind, d, c->params.data(), c->derived, &c->scale, &why)) {
    delete c;
    return thread_fail(VEGAS_EINVAL, "%s", why.c_str());
  }
  if (!lookup_kernel(fn->kind, c->prec, ybits, d, &c->ke)) {
    delete c;
    return thread_fail(VEGAS_EINVAL, "no kernel for kind %d, ndim %d", fn->kind, d);
  }
  return finish_create(c, out);
}

vegas_status vegas_create_user(const vegas_config* cfg, const char* source, const double* params, int nparams,
                               vegas_ctx** out) {
  if (!out) return thread_fail(VEGAS_EINVAL, "out is NULL");
  *out = nullptr;
  if (!cfg || !source) return thread_fail(VEGAS_EINVAL, "config or source is NULL");
  int ybits = 0, g = 1;
  uint64_t G = 1;
  vegas_status cs = check_config(cfg, &ybits, &g, &G);
  if (cs) return cs;
  if (nparams < 0 || nparams > GVEGAS_MAXUSERPARAMS || (nparams > 0 && !params))
    return thread_fail(VEGAS_EINVAL, "user integrand takes 0..%d parameters, got %d", GVEGAS_MAXUSERPARAMS, nparams);
  vegas_ctx* c = new_context(cfg, ybits, g, G);
  c->kind = VG_USER;
  c->params.assign(params, params + nparams);
  std::copy(c->params.begin(), c->params.end(), c->derived);
  c->scale = 1.0;
  std::string why;
  const int d = cfg->ndim;
  const int rs = gv::rtc_user_entry(source, c->prec, ybits, d, spec_shape(d, d, ybits, g, cfg->nbins), &c->ke, &why);
  if (rs != VEGAS_OK) {
    delete c;
    return thread_fail((vegas_status)rs, "%s", why.c_str());
  }
  return finish_create(c, out);
}

vegas_status vegas_user_compile(const vegas_config* cfg, const char* source) {
  if (!cfg || !source) return thread_fail(VEGAS_EINVAL, "config or source is NULL");
  int ybits = 0, g = 1;
  uint64_t G = 1;
  vegas_status cs = check_config(cfg, &ybits, &g, &G);
  if (cs) return cs;
  const int d = cfg->ndim;
  std::string why;
  const int rs = gv::rtc_user_compile(source, cfg->precision, ybits, d, spec_shape(d, d, ybits, g, cfg->nbins), &why);
  if (rs != VEGAS_OK) return thread_fail((vegas_status)rs, "%s", why.c_str());
  return VEGAS_OK;
}

vegas_status vegas_iterate(vegas_ctx* c, int n_iter, int refine, vegas_result* out) {
  if (!c) return thread_fail(VEGAS_EINVAL, "ctx is NULL");
  if (n_iter < 0) return c->fail(VEGAS_EINVAL, "n_iter < 0");
  if (n_iter > 0) {
    if (c->hist_upper + n_iter > gv::kMaxHist)
      return c->fail(VEGAS_EINVAL, "window would exceed %d iterations; call vegas_reset_results", gv::kMaxHist);
    cudaGraphExec_t ge;
    vegas_status st = get_graph(c, 0, n_iter, 0, refine ? 1 : 0, c->cfg.acc, 0.0, &ge);
    if (st) return st;
    CK(c, cudaGraphLaunch(ge, c->stream));
    c->hist_upper += n_iter;
  }
  if (out) {
    vegas_status st = read_state(c);
    if (st) return st;
    fill_result(c, out);
  }
  return VEGAS_OK;
}

vegas_status vegas_reset_results(vegas_ctx* c) {
  if (!c) return thread_fail(VEGAS_EINVAL, "ctx is NULL");
  CK(c, gv_launch_control(c->d_st, gv::CTL_RESET_WINDOW | gv::CTL_SET_ACC, c->cfg.acc, 0u, c->h_st, c->stream));
  c->hist_upper = 0;
  return VEGAS_OK;
}

vegas_status vegas_reset_grid(vegas_ctx* c) {
  if (!c) return thread_fail(VEGAS_EINVAL, "ctx is NULL");
  const int d = c->cfg.ndim, N = c->cfg.nbins;
  CK(c, gv_launch_uniform_grid(c->d_edges, d, N, c->d_tab64, c->d_tab32, c->stream));
  return VEGAS_OK;
}

vegas_status bases_integrate(vegas_ctx* c, int itmx1, double acc1, int itmx2, double acc2,
                             vegas_result* out, vegas_result* phase1) {
  if (!c) return thread_fail(VEGAS_EINVAL, "ctx is NULL");
  if (itmx1 < 0 || itmx2 < 1 || itmx1 > gv::kMaxHist || itmx2 > gv::kMaxHist)
    return c->fail(VEGAS_EINVAL, "need 0 <= itmx1 <= %d and 1 <= itmx2 <= %d", gv::kMaxHist, gv::kMaxHist);
  cudaGraphExec_t ge;
  vegas_status st = get_graph(c, 1, itmx1, itmx2, 1, acc1, acc2, &ge);
  if (st) return st;
  CK(c, cudaGraphLaunch(ge, c->stream));
  c->hist_upper = itmx2;
  c->have_max = true;
  if (out || phase1) {
    if ((st = read_state(c))) return st;
    if (out) fill_result(c, out);
    if (phase1) {
      const GState* h = c->h_st;
      phase1->I = h->ph1_I;
      phase1->sigma = h->ph1_sigma;
      phase1->chi2_dof = h->ph1_chi2;
      phase1->iters_done = h->ph1_iters;
      phase1->stopped = h->ph1_stopped;
      phase1->nonfinite = h->ph1_nonfinite;
      phase1->samples = h->ph1_samples;
    }
  }
  return VEGAS_OK;
}

vegas_status vegas_get_grid(vegas_ctx* c, double* edges, double* bin_sums) {
  if (!c) return thread_fail(VEGAS_EINVAL, "ctx is NULL");
  const int d = c->cfg.ndim, N = c->cfg.nbins;
  const size_t ne = (size_t)d * (N + 1), nb = 2 * (size_t)d * N;
  vegas_status st = stage(c, ne + nb);
  if (st) return st;
  const size_t from = edges ? 0 : ne, upto = bin_sums ? ne + nb : ne;  // (the sums lie behind the edges)
  if (upto > from)
    CK(c, cudaMemcpyAsync(c->h_stage + from, c->d_edges + from, (upto - from) * sizeof(double), cudaMemcpyDeviceToHost,
                          c->stream));
  CK(c, cudaStreamSynchronize(c->stream));
  if (edges) memcpy(edges, c->h_stage, ne * sizeof(double));
  if (bin_sums) memcpy(bin_sums, c->h_stage + ne, nb * sizeof(double));
  return VEGAS_OK;
}

vegas_status vegas_set_grid(vegas_ctx* c, const double* edges) {
  if (!c) return thread_fail(VEGAS_EINVAL, "ctx is NULL");
  if (!edges || !valid_grid(edges, c->cfg.ndim, c->cfg.nbins))
    return c->fail(VEGAS_EINVAL, "edges must start at 0, end at 1 and increase strictly");
  return upload_grid(c, edges);
}

vegas_status vegas_get_history(vegas_ctx* c, double* hist, int max_iters, int* n_out) {
  if (!c) return thread_fail(VEGAS_EINVAL, "ctx is NULL");
  // up to the longest window the calls so far can have left, in one go
  const int most = hist ? std::min(c->hist_upper, std::max(max_iters, 0)) : 0;
  vegas_status st = VEGAS_OK;
  if (most > 0) {
    if ((st = stage(c, 2 * (size_t)most))) return st;
    CK(c, cudaMemcpyAsync(c->h_stage, &c->d_st->hist[0][0], 2 * most * sizeof(double), cudaMemcpyDeviceToHost,
                          c->stream));
  }
  if ((st = read_state(c))) return st;
  const int n = std::min(c->h_st->nhist, most);
  if (n_out) *n_out = c->h_st->nhist;
  if (n > 0) memcpy(hist, c->h_stage, 2 * (size_t)n * sizeof(double));
  return VEGAS_OK;
}

vegas_status vegas_get_cube_sums(vegas_ctx* c, double* sums) {
  if (!c) return thread_fail(VEGAS_EINVAL, "ctx is NULL");
  if (!c->strat) return c->fail(VEGAS_ESTATE, "context is not stratified");
  if (!sums) return c->fail(VEGAS_EINVAL, "sums is NULL");
  const size_t n = 2 * (size_t)c->ncubes;
  vegas_status st = stage(c, n);
  if (st) return st;
  CK(c, cudaMemcpyAsync(c->h_stage, c->d_cubes, n * sizeof(double), cudaMemcpyDeviceToHost, c->stream));
  CK(c, cudaStreamSynchronize(c->stream));
  const double s1 = c->scale, s2 = c->scale * c->scale;
  const bool pairs = c->prec == VG_FP32_ACCCOMP;  // (hi, lo, hi, lo) floats per cube
  const float* fp = reinterpret_cast<const float*>(c->h_stage);
  for (size_t i = 0; i < c->ncubes; ++i) {
    if (pairs) {
      sums[2 * i] = ((double)fp[4 * i] + (double)fp[4 * i + 1]) * s1;
      sums[2 * i + 1] = ((double)fp[4 * i + 2] + (double)fp[4 * i + 3]) * s2;
    } else {
      sums[2 * i] = c->h_stage[2 * i] * s1;
      sums[2 * i + 1] = c->h_stage[2 * i + 1] * s2;
    }
  }
  return VEGAS_OK;
}

vegas_status vegas_get_cube_max(vegas_ctx* c, double* cmax) {
  if (!c) return thread_fail(VEGAS_EINVAL, "ctx is NULL");
  if (!cmax) return c->fail(VEGAS_EINVAL, "cmax is NULL");
  if (!c->have_max) return c->fail(VEGAS_ESTATE, "no integration phase has run (bases_integrate)");
  const size_t n = (size_t)c->ncubes;
  vegas_status st = stage(c, n);
  if (st) return st;
  CK(c, cudaMemcpyAsync(c->h_stage, c->d_cube_max, n * sizeof(double), cudaMemcpyDeviceToHost, c->stream));
  CK(c, cudaStreamSynchronize(c->stream));
  for (size_t i = 0; i < n; ++i) cmax[i] = c->h_stage[i] * c->scale;
  return VEGAS_OK;
}

vegas_status spring_generate(vegas_ctx* c, uint64_t trial0, uint32_t n_trials, double* x_out, uint64_t* trial_out,
                             uint32_t* n_events, uint32_t* n_overflow, uint32_t* n_nonpos) {
  if (!c) return thread_fail(VEGAS_EINVAL, "ctx is NULL");
  if (!n_events) return c->fail(VEGAS_EINVAL, "n_events is NULL");
  if (!c->have_max) return c->fail(VEGAS_ESTATE, "no integration phase has run (bases_integrate)");
  if (trial0 + (uint64_t)n_trials > 0x100000000ull) return c->fail(VEGAS_EINVAL, "trial indices must stay below 2^32");
  if (c->ncubes > 0xFFFFFFFFull) return c->fail(VEGAS_EINVAL, "too many hypercubes");
  *n_events = 0;
  if (n_overflow) *n_overflow = 0;
  if (n_nonpos) *n_nonpos = 0;
  if (n_trials == 0) return VEGAS_OK;
  const int d = c->cfg.ndim, N = c->cfg.nbins;
  const uint32_t chunk = 4096, nchunks = (n_trials + chunk - 1) / chunk;
  const bool spec = c->ke.sample == c->ke.sample_spec && c->ke.spring_spec;
  const void* fn = spec ? c->ke.spring_spec : c->ke.spring;
  auto grow = [&](void** p, size_t bytes) -> vegas_status {
    cudaFree(*p);
    *p = nullptr;
    if (gv_dev_malloc(p, bytes) != cudaSuccess) return c->fail(VEGAS_ENOMEM, "cudaMalloc(%zu)", bytes);
    return VEGAS_OK;
  };
  vegas_status st = VEGAS_OK;
  uint32_t gk = 0;  // 2^gk guide intervals: about one per cube, at most 2^22 (16 MB)
  while (gk < 22 && (1ull << gk) < c->ncubes) ++gk;
  if (!c->d_counters) {  // the tables (all of them again where an earlier call got only some: the counters come last)
    if (!st) st = grow((void**)&c->d_q, sizeof(uint64_t) * c->ncubes);
    if (!st) st = grow((void**)&c->d_mt, sizeof(double) * c->ncubes);
    if (!st) st = grow((void**)&c->d_mt32, sizeof(float) * c->ncubes);
    if (!st) st = grow((void**)&c->d_guide, sizeof(uint32_t) * ((1ull << gk) + 1));
    const size_t nb = (c->ncubes + kSpan - 1) / kSpan;
    if (!st) st = grow((void**)&c->d_bmax, sizeof(double) * nb);
    if (!st) st = grow((void**)&c->d_bsum, sizeof(unsigned long long) * nb);
    if (!st) st = grow((void**)&c->d_prefix, sizeof(uint64_t) * (c->ncubes + 1));
    if (!st) st = grow((void**)&c->d_meta, sizeof(double) * 3);
    if (!st) st = grow((void**)&c->d_counters, sizeof(unsigned long long) * 2);
  }
  if (!st && !c->h_spring && gv_malloc_host(&c->h_spring, sizeof(SpringOutcome)) != cudaSuccess) {
    c->h_spring = nullptr;
    st = c->fail(VEGAS_ENOMEM, "cudaMallocHost(SPRING outcome)");
  }
  if (!st && n_trials > c->spring_cap) {
    if (!st) st = grow((void**)&c->d_stage_x, sizeof(double) * d * (size_t)n_trials);
    if (!st) st = grow((void**)&c->d_stage_t, sizeof(uint64_t) * (size_t)n_trials);
    if (!st) st = grow((void**)&c->d_counts, sizeof(uint32_t) * nchunks);
    if (!st) c->spring_cap = n_trials;
  }
  // where the compacted events go: the caller's buffers, or, when the GPU
  // cannot write those, device buffers that are copied
  double* ox = x_out ? static_cast<double*>(device_view(x_out, sizeof(double) * d * (size_t)n_trials, sizeof(double)))
                     : nullptr;
  uint64_t* ot = trial_out ? static_cast<uint64_t*>(device_view(trial_out, sizeof(uint64_t) * (size_t)n_trials, sizeof(uint64_t)))
                           : nullptr;
  const bool copy = (x_out && !ox) || (trial_out && !ot);
  if (!st && copy && n_trials > c->spring_out_cap) {
    if (!st) st = grow((void**)&c->d_out_x, sizeof(double) * d * (size_t)n_trials);
    if (!st) st = grow((void**)&c->d_out_t, sizeof(uint64_t) * (size_t)n_trials);
    c->spring_out_cap = st ? 0 : n_trials;
  }
  if (st) {
    c->spring_cap = 0;
    return st;
  }
  if (copy) {
    ox = x_out ? c->d_out_x : nullptr;
    ot = trial_out ? c->d_out_t : nullptr;
  }
  // integer cube table from the recorded maxima (in the integrand's units)
  {
    const uint32_t G = (uint32_t)c->ncubes, nb = (G + kSpan - 1) / kSpan;
    k_spring_max<<<nb, kSpanThreads, 0, c->stream>>>(c->d_cube_max, G, c->scale, c->d_bmax);
    k_spring_weights<<<nb, kSpanThreads, 0, c->stream>>>(c->d_cube_max, G, c->scale, c->d_bmax, nb, c->d_q,
                                                         c->d_mt, c->d_mt32, c->d_bsum);
    k_spring_scan<<<1, 1024, 0, c->stream>>>(c->d_bmax, nb, c->d_bsum, G, c->d_prefix, c->d_meta);
    k_spring_prefix<<<nb, kSpanThreads, 0, c->stream>>>(c->d_q, G, c->d_bsum, c->d_prefix, c->d_meta);
    k_spring_guide<<<(uint32_t)(((1ull << gk) + 256) / 256), 256, 0, c->stream>>>(c->d_prefix, G, gk, c->d_guide,
                                                                                  c->d_meta);
  }
  CK(c, cudaGetLastError());
  CK(c, cudaMemsetAsync(c->d_counters, 0, sizeof(unsigned long long) * 2, c->stream));
  gv::SpringArgs R{};
  R.S = sample_args(c, 0);
  R.prefix = c->d_prefix;
  R.mt = c->d_mt;
  R.mt32 = c->d_mt32;
  R.guide = c->d_guide;
  R.gk = gk;
  R.meta = c->d_meta;
  R.out_scale = c->scale;
  R.trial0 = (uint32_t)trial0;
  R.n = n_trials;
  R.chunk = chunk;
  R.nchunks = nchunks;
  R.stage_x = c->d_stage_x;
  R.stage_t = c->d_stage_t;
  R.counts = c->d_counts;
  R.counters = c->d_counters;
  const bool f64 = c->prec == VG_FP64;
  const size_t smem = (size_t)d * N * (f64 ? sizeof(double2) : sizeof(float2)) +
                      gv::kNumDerived * (f64 ? sizeof(double) : sizeof(float));
  int occ = 0;
  CK(c, gv_raise_smem_limit(fn, smem));
  CK(c, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, 256, smem));
  if (occ < 1) return c->fail(VEGAS_EINVAL, "SPRING kernel does not fit");
  const uint32_t blocks = std::min<uint32_t>(nchunks, (uint32_t)(c->sm_count * occ));
  void* args[] = {&R};
  if (c->spring_timer[0]) CK(c, cudaEventRecord(c->spring_timer[0], c->stream));
  CK(c, cudaLaunchKernel(fn, dim3(blocks), dim3(256), args, smem, c->stream));
  if (c->spring_timer[1]) CK(c, cudaEventRecord(c->spring_timer[1], c->stream));
  SpringOutcome* oc = static_cast<SpringOutcome*>(c->h_spring);
  k_spring_compact<<<nchunks, 256, 0, c->stream>>>(c->d_counts, chunk, d, c->d_stage_x, c->d_stage_t, ox, ot,
                                                  c->d_meta, c->d_counters, oc);
  CK(c, cudaGetLastError());
  CK(c, cudaStreamSynchronize(c->stream));
  if (oc->status != 0.0) return c->fail(VEGAS_ESTATE, "every recorded cube maximum is zero");
  const uint64_t total = oc->events;
  *n_events = (uint32_t)total;
  if (n_overflow) *n_overflow = (uint32_t)oc->overflow;
  if (n_nonpos) *n_nonpos = (uint32_t)oc->nonpos;
  if (copy && total) {
    if (x_out)
      CK(c, cudaMemcpyAsync(x_out, c->d_out_x, sizeof(double) * d * total, cudaMemcpyDeviceToHost, c->stream));
    if (trial_out)
      CK(c, cudaMemcpyAsync(trial_out, c->d_out_t, sizeof(uint64_t) * total, cudaMemcpyDeviceToHost, c->stream));
    CK(c, cudaStreamSynchronize(c->stream));
  }
  return VEGAS_OK;
}

vegas_status spring_profile(vegas_ctx* c, uint32_t n_trials, int reps, double* ms) {
  if (!c) return thread_fail(VEGAS_EINVAL, "ctx is NULL");
  if (reps < 1 || !ms) return c->fail(VEGAS_EINVAL, "need reps >= 1 and ms");
  uint32_t k = 0;
  vegas_status st = spring_generate(c, 0, n_trials, nullptr, nullptr, &k, nullptr, nullptr);  // buffers, warm-up
  if (st) return st;
  cudaEvent_t a, b;
  CK(c, cudaEventCreate(&a));
  CK(c, cudaEventCreate(&b));
  double acc = 0.0;
  for (int r = 0; r < reps && !st; ++r) {
    c->spring_timer[0] = a;
    c->spring_timer[1] = b;
    st = spring_generate(c, 0, n_trials, nullptr, nullptr, &k, nullptr, nullptr);
    float t = 0.f;
    if (!st && cudaEventElapsedTime(&t, a, b) != cudaSuccess) st = c->fail(VEGAS_ECUDA, "event timing");
    acc += t;
  }
  c->spring_timer[0] = c->spring_timer[1] = nullptr;
  cudaEventDestroy(a);
  cudaEventDestroy(b);
  if (st) return st;
  *ms = acc / reps;
  return VEGAS_OK;
}

vegas_status vegas_get_iteration(vegas_ctx* c, uint32_t* it) {
  if (!c || !it) return thread_fail(VEGAS_EINVAL, "NULL argument");
  vegas_status st = read_state(c);
  if (st) return st;
  *it = c->h_st->it;
  return VEGAS_OK;
}

vegas_status vegas_set_iteration(vegas_ctx* c, uint32_t it) {
  if (!c) return thread_fail(VEGAS_EINVAL, "ctx is NULL");
  CK(c, gv_launch_control(c->d_st, gv::CTL_SET_ITER, 0.0, it, c->h_st, c->stream));
  return VEGAS_OK;
}

vegas_status vegas_set_params(vegas_ctx* c, const double* params, int nparams) {
  if (!c) return thread_fail(VEGAS_EINVAL, "ctx is NULL");
  if (!params || nparams != (int)c->params.size())
    return c->fail(VEGAS_EINVAL, "expected %d parameters", (int)c->params.size());
  std::vector<double> p(params, params + nparams);
  double dv[gv::kNumDerived] = {}, sc = 1.0;
  std::string why;
  if (c->kind == VG_USER)  // the user's parameters are the device constants
    std::copy(p.begin(), p.end(), dv);
  else if (!gv::derive_params(c->kind, c->cfg.ndim, p.data(), dv, &sc, &why))
    return c->fail(VEGAS_EINVAL, "%s", why.c_str());
  c->params = p;
  memcpy(c->derived, dv, sizeof dv);
  c->scale = sc;
  // constants and scale live in device memory: the captured graphs read
  // them at run time and stay valid
  return upload_derived(c);
}

vegas_status vegas_eval(vegas_ctx* c, uint32_t it, double* I, double* var) {
  if (!c) return thread_fail(VEGAS_EINVAL, "ctx is NULL");
  if (it > 0x7FFFFFFFu) return c->fail(VEGAS_EINVAL, "iteration index must be < 2^31");
  vegas_status st = launch_pass(c, (int)it, 0, 0);
  if (st) return st;
  if ((st = read_state(c))) return st;
  if (I) *I = c->h_st->last_I;
  if (var) *var = c->h_st->last_var;
  return VEGAS_OK;
}

vegas_status vegas_sample_dump(vegas_ctx* c, uint32_t it, const uint64_t* s, int64_t n, uint32_t* words,
                               int32_t* bins, double* x, double* jac, double* f) {
  if (!c) return thread_fail(VEGAS_EINVAL, "ctx is NULL");
  if (n < 0 || (n > 0 && !s)) return c->fail(VEGAS_EINVAL, "bad sample list");
  if (n == 0) return VEGAS_OK;
  if (it > 0x7FFFFFFFu) return c->fail(VEGAS_EINVAL, "iteration index must be < 2^31");
  for (int64_t i = 0; i < n; ++i)
    if (s[i] >= (uint64_t)c->cfg.ncall) return c->fail(VEGAS_EINVAL, "sample index %llu >= ncall", (unsigned long long)s[i]);
  const int d = c->cfg.ndim, W = c->ybits == 24 ? d : 2 * d;
  uint64_t* ds = nullptr;
  uint32_t* dw = nullptr;
  int32_t* db = nullptr;
  double *dx = nullptr, *dj = nullptr, *df = nullptr;
  vegas_status st = VEGAS_OK;
  auto A = [&](void** p, size_t b) {
    if (!st && gv_dev_malloc(p, b) != cudaSuccess) st = c->fail(VEGAS_ENOMEM, "cudaMalloc(%zu)", b);
  };
  A((void**)&ds, n * sizeof(uint64_t));
  if (words) A((void**)&dw, n * W * sizeof(uint32_t));
  if (bins) A((void**)&db, n * d * sizeof(int32_t));
  if (x) A((void**)&dx, n * d * sizeof(double));
  if (jac) A((void**)&dj, n * sizeof(double));
  if (f) A((void**)&df, n * sizeof(double));
  cudaError_t e = cudaSuccess;
  if (!st) {
    gv::DumpArgs D{};
    D.S = sample_args(c, (int)it);
    D.s = ds;
    D.n = n;
    D.words = dw;
    D.bins = db;
    D.x = dx;
    D.jac = dj;
    D.f = df;
    void* args[] = {&D};
    e = cudaMemcpyAsync(ds, s, n * sizeof(uint64_t), cudaMemcpyHostToDevice, c->stream);
    if (e == cudaSuccess)
      e = cudaLaunchKernel(c->ke.dump, dim3((unsigned)((n + 255) / 256)), dim3(256), args, 0, c->stream);
    if (e == cudaSuccess && words) e = cudaMemcpyAsync(words, dw, n * W * sizeof(uint32_t), cudaMemcpyDeviceToHost, c->stream);
    if (e == cudaSuccess && bins) e = cudaMemcpyAsync(bins, db, n * d * sizeof(int32_t), cudaMemcpyDeviceToHost, c->stream);
    if (e == cudaSuccess && x) e = cudaMemcpyAsync(x, dx, n * d * sizeof(double), cudaMemcpyDeviceToHost, c->stream);
    if (e == cudaSuccess && jac) e = cudaMemcpyAsync(jac, dj, n * sizeof(double), cudaMemcpyDeviceToHost, c->stream);
    if (e == cudaSuccess && f) e = cudaMemcpyAsync(f, df, n * sizeof(double), cudaMemcpyDeviceToHost, c->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess) st = c->fail(VEGAS_ECUDA, "sample dump: %s", cudaGetErrorString(e));
  }
  cudaFree(ds);
  cudaFree(dw);
  cudaFree(db);
  cudaFree(dx);
  cudaFree(dj);
  cudaFree(df);
  if (!st && f) {
    for (int64_t i = 0; i < n; ++i) f[i] *= c->scale;
    if (jac) {
      // jac is reported as the Jacobian itself; f carries the integrand scale
    }
  }
  return st;
}

vegas_status vegas_set_launch(vegas_ctx* c, int threads, int ctas_per_sm) {
  if (!c) return thread_fail(VEGAS_EINVAL, "ctx is NULL");
  if (threads < 64 || threads > c->ke.max_threads || threads % 32 != 0)
    return c->fail(VEGAS_EINVAL, "threads must be a multiple of 32 in 64..%d", c->ke.max_threads);
  if (ctas_per_sm < 0) return c->fail(VEGAS_EINVAL, "ctas_per_sm < 0");
  CK(c, cudaStreamSynchronize(c->stream));
  const int t0 = c->threads_req, p0 = c->ctas_per_sm_req, f0 = c->frozen_req;
  c->threads_req = threads;
  c->ctas_per_sm_req = ctas_per_sm;
  c->frozen_req = 0;
  vegas_status st = configure_launch(c);
  if (st) {  // (the shape and its buffers are as before)
    c->threads_req = t0;
    c->ctas_per_sm_req = p0;
    c->frozen_req = f0;
  }
  return st;
}

vegas_status vegas_set_tile(vegas_ctx* c, int points_per_thread) {
  if (!c) return thread_fail(VEGAS_EINVAL, "ctx is NULL");
  if (points_per_thread < 0 || points_per_thread > 8)
    return c->fail(VEGAS_EINVAL, "points_per_thread must be in 0..8 (0: automatic)");
  CK(c, cudaStreamSynchronize(c->stream));
  const int p0 = c->ppt_req;
  c->ppt_req = points_per_thread;
  vegas_status st = configure_launch(c);
  if (st) c->ppt_req = p0;  // (the shape and its buffers are as before)
  return st;
}

vegas_status vegas_autotune(vegas_ctx* c, int* threads, int* points_per_thread, double* ms) {
  if (!c) return thread_fail(VEGAS_EINVAL, "ctx is NULL");
  // (0: the automatic shape, which has CTA widths of its own)
  static const int kThreads[] = {0, 128, 256, 384, 512};
  static const int kTiles[] = {0, 1, 2, 4};
  struct Shape {  // requests of configure_launch
    int t, per_sm, f, p;
    bool small;
  };
  struct Cand {
    Shape s;
    double ms;
  };
  auto get = [&]() { return Shape{c->threads_req, c->ctas_per_sm_req, c->frozen_req, c->ppt_req, c->small_cap}; };
  auto put = [&](const Shape& s) {
    c->threads_req = s.t;
    c->ctas_per_sm_req = s.per_sm;
    c->frozen_req = s.f;
    c->ppt_req = s.p;
    c->small_cap = s.small;
  };
  auto set_shape = [&](const Shape& s) -> vegas_status {
    CK(c, cudaStreamSynchronize(c->stream));
    const Shape had = get();
    put(s);
    const vegas_status st = configure_launch(c);
    if (st) put(had);
    return st;
  };
  // one pass of warm-up, then the mean of n passes, for shape s
  auto time_shape = [&](const Shape& s, bool frozen, int n, double* out) -> vegas_status {
    if (set_shape(s) != VEGAS_OK) return VEGAS_EINVAL;
    double m[3];
    vegas_status st = VEGAS_OK;
    for (int k : {1, n})
      if (!st) st = frozen ? vegas_profile_frozen_pass(c, k, m) : vegas_profile_pass(c, k, m);
    if (!st) *out = m[2];
    return st == VEGAS_OK ? VEGAS_OK : VEGAS_ECUDA;
  };
  const Shape before = get();
  auto give_up = [&]() -> vegas_status {  // a pass failed: back to the shape it came with
    const std::string why = c->err;
    set_shape(before);
    return c->fail(VEGAS_ECUDA, "%s", why.empty() ? "autotune: pass failed" : why.c_str());
  };
  // screening: every shape the kernel takes (the others are skipped)
  std::vector<Cand> cands;
  for (int t : kThreads)
    for (int p : kTiles) {
      if (t > c->ke.max_threads || (t == 0 && p > 0)) continue;
      int cap_large = -1;  // the tile of the largest-capacity policy (a repeat is not timed twice)
      for (bool small : {false, true}) {
        const Shape s{t, 0, 0, p, small};
        double m = 0.0;
        const vegas_status st = time_shape(s, false, 3, &m);
        if (st == VEGAS_ECUDA) return give_up();
        if (st != VEGAS_OK || (small && c->cap == cap_large)) continue;
        if (!small) cap_large = c->cap;
        cands.push_back({s, m});
      }
    }
  if (cands.empty()) return c->fail(VEGAS_EINVAL, "autotune: no launch shape fits");
  // the three fastest again, in interleaved rounds, keeping each one's best
  // round (shapes a few percent apart are within one screening's noise)
  auto faster = [](const Cand& a, const Cand& b) { return a.ms < b.ms; };
  auto finals = [&](std::vector<Cand>& v, bool frozen, int rounds) -> vegas_status {
    for (int r = 0; r < rounds; ++r)
      for (Cand& k : v) {
        double m = 0.0;
        if (time_shape(k.s, frozen, 5, &m) != VEGAS_OK) return VEGAS_ECUDA;
        k.ms = r == 0 ? m : std::min(k.ms, m);
      }
    return VEGAS_OK;
  };
  std::sort(cands.begin(), cands.end(), faster);
  cands.resize(std::min<size_t>(cands.size(), 3));
  if (finals(cands, false, 3) != VEGAS_OK) return give_up();
  const Cand best = *std::min_element(cands.begin(), cands.end(), faster);
  // the passes without bins have a width of their own
  std::vector<Cand> widths;
  for (int f : {128, 256, 384, 512})
    if (f <= c->ke.max_threads) {
      widths.push_back({best.s, 0.0});
      widths.back().s.f = f;
    }
  for (Cand& k : widths)
    if (time_shape(k.s, true, 3, &k.ms) != VEGAS_OK) return give_up();
  std::sort(widths.begin(), widths.end(), faster);
  widths.resize(std::min<size_t>(widths.size(), 2));
  if (finals(widths, true, 2) != VEGAS_OK) return give_up();
  const Cand width = *std::min_element(widths.begin(), widths.end(), faster);
  const vegas_status st = set_shape(width.s);
  if (st) return st;
  if (threads) *threads = c->pass_bins.threads;
  if (points_per_thread) *points_per_thread = c->ppt;
  if (ms) *ms = best.ms;
  return VEGAS_OK;
}

vegas_status vegas_get_tile(vegas_ctx* c, int* points_per_thread, int* cap) {
  if (!c) return thread_fail(VEGAS_EINVAL, "ctx is NULL");
  if (points_per_thread) *points_per_thread = c->ppt;
  if (cap) *cap = c->cap;
  return VEGAS_OK;
}

vegas_status vegas_get_launch(vegas_ctx* c, int* threads, int* ctas, int* ctas_per_sm) {
  if (!c) return thread_fail(VEGAS_EINVAL, "ctx is NULL");
  if (threads) *threads = c->pass_bins.threads;
  if (ctas) *ctas = c->pass_bins.ctas;
  if (ctas_per_sm) *ctas_per_sm = c->pass_bins.occ;
  return VEGAS_OK;
}

vegas_status vegas_grad(vegas_ctx* c, uint32_t it, double* grad, double* I) {
  if (!c) return thread_fail(VEGAS_EINVAL, "ctx is NULL");
  if (!grad) return c->fail(VEGAS_EINVAL, "grad is NULL");
  if (it > 0x7FFFFFFFu) return c->fail(VEGAS_EINVAL, "iteration index must be < 2^31");
  const int nt = vegas_ntheta(c);
  if (!c->ke.grad || nt == 0 || nt > c->ke.grad_nt)
    return c->fail(VEGAS_EINVAL, "no adjoint kernel for integrand kind %d with ndim %d", c->kind, c->cfg.ndim);
  if (c->kind == VG_RAMBO_BW && c->params[VG_RB_OBS] != 0.0)
    return c->fail(VEGAS_EINVAL, "the RAMBO gradient is defined for the full integrand (observable 0)");
  const int ncol = c->ke.grad_nt + 2;
  gv::SampleArgs A = sample_args(c, (int)it);
  double* part = c->d_gpart;
  double* out = c->d_gpart + (size_t)ncol * c->grad_ctas;
  void* args[] = {&A, &part};
  CK(c, cudaLaunchKernel(c->ke.grad, dim3(c->grad_ctas), dim3(256), args, c->grad_smem, c->stream));
  CK(c, gv_launch_colsum(part, ncol, c->grad_ctas, out, c->stream));
  vegas_status st = stage(c, ncol);
  if (st) return st;
  CK(c, cudaMemcpyAsync(c->h_stage, out, ncol * sizeof(double), cudaMemcpyDeviceToHost, c->stream));
  CK(c, cudaStreamSynchronize(c->stream));
  const double k = c->scale / (double)c->cfg.ncall;
  const int d = c->cfg.ndim, DM = c->ke.dm;
  for (int t = 0; t < nt; ++t) {
    // the Genz Gaussian kernel stores du at [0, d) and da at [DM, DM + d)
    const int src = (c->kind == VG_GENZ_GAUSSIAN && t >= d) ? DM + (t - d) : t;
    grad[t] = c->h_stage[src] * k;
  }
  if (I) *I = c->h_stage[c->ke.grad_nt] * k;
  return VEGAS_OK;
}

}  // extern "C"

namespace {
vegas_status profile_passes(vegas_ctx* c, int n_pass, bool nobins, double* ms);
}  // namespace

extern "C" {

vegas_status vegas_profile_pass(vegas_ctx* c, int n_pass, double* ms) { return profile_passes(c, n_pass, false, ms); }

vegas_status vegas_profile_frozen_pass(vegas_ctx* c, int n_pass, double* ms) {
  return profile_passes(c, n_pass, true, ms);
}

}  // extern "C"

namespace {

vegas_status profile_passes(vegas_ctx* c, int n_pass, bool nobins, double* ms) {
  if (!c) return thread_fail(VEGAS_EINVAL, "ctx is NULL");
  if (n_pass < 1 || !ms) return c->fail(VEGAS_EINVAL, "need n_pass >= 1 and ms[3]");
  CK(c, cudaStreamSynchronize(c->stream));
  vegas_status st = read_state(c);
  if (st) return st;
  const uint32_t it = c->h_st->it;
  cudaEvent_t ev[3];
  for (int i = 0; i < 3; ++i) CK(c, cudaEventCreate(&ev[i]));
  double acc[3] = {0, 0, 0};
  const gv::PassShape& ps = nobins ? c->pass_nobins : c->pass_bins;
  cudaError_t e = cudaSuccess;
  for (int p = 0; p < n_pass && e == cudaSuccess; ++p) {
    gv::SampleArgs A = sample_args(c, (int)(it & 0x7FFFFFFFu), nobins);
    void* args[] = {&A};
    gv::FinArgs F = fin_args(c, 0, 0, nobins);
    e = cudaEventRecord(ev[0], c->stream);
    if (!e)
      e = cudaLaunchKernel(ps.fn, dim3(ps.ctas), dim3(ps.threads), args, ps.smem, c->stream);
    if (!e) e = cudaEventRecord(ev[1], c->stream);
    if (!e) e = gv_launch_finish(&F, c->stream);
    if (!e) e = cudaEventRecord(ev[2], c->stream);
    if (!e) e = cudaEventSynchronize(ev[2]);
    float t0 = 0.f, t1 = 0.f, t2 = 0.f;
    if (!e) e = cudaEventElapsedTime(&t0, ev[0], ev[1]);
    if (!e) e = cudaEventElapsedTime(&t1, ev[1], ev[2]);
    if (!e) e = cudaEventElapsedTime(&t2, ev[0], ev[2]);
    acc[0] += t0;
    acc[1] += t1;
    acc[2] += t2;
  }
  for (int i = 0; i < 3; ++i) cudaEventDestroy(ev[i]);
  if (e != cudaSuccess) return c->fail(VEGAS_ECUDA, "profile: %s", cudaGetErrorString(e));
  for (int k = 0; k < 3; ++k) ms[k] = acc[k] / n_pass;
  return VEGAS_OK;
}

}  // namespace

extern "C" {

int vegas_ntheta(const vegas_ctx* c) {
  if (!c) return 0;
  switch (c->kind) {
    case VG_GENZ_GAUSSIAN: return 2 * c->cfg.ndim;
    case VG_DOUBLE_GAUSSIAN: return 3;
    case VG_RAMBO_BW: return 3;
    default: return 0;
  }
}

}  // extern "C"

// ---------------------------------------------------------------------------
// One evaluation pass without any device allocation.
//
// Some callers cannot call cudaMalloc at all: code that runs inside another
// runtime's memory pool with a fixed budget, or a latency-critical loop where
// an allocation (which may synchronise the device or fail under
// fragmentation) is not allowed after start-up.  vegas_eval_noalloc serves
// them: the caller passes the grid and the output in its own device memory,
// and every intermediate the pass needs (grid tables, integrand constants,
// pass state, per-CTA partial sums) lives in the file-scope array below.
// ---------------------------------------------------------------------------
namespace {

constexpr size_t kNoAllocScratchBytes = 8u << 20;  // 8 MiB, held by every GPU
                                                    // that loads this library
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];

constexpr int kNoAllocMaxDevices = 64;
std::mutex g_noalloc_mutex;
unsigned char* g_noalloc_ptr[kNoAllocMaxDevices] = {};
int g_noalloc_sms[kNoAllocMaxDevices] = {};

// Set-up in one launch: the state (it must start cleared; its stop flag gates
// the kernels), the integrand constants and the grid's tables.
__global__ void k_noalloc_setup(const DerivedBlock b, double* derived, GState* st, const double* edges, int d, int N,
                                double2* tab64, float2* tab32) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i <= gv::kNumDerived) derived[i] = b.v[i];
  const int words = (int)(offsetof(GState, hist) / sizeof(int));
  if (i < words) reinterpret_cast<int*>(st)[i] = 0;
  if (i >= d * N) return;
  const int a = i / N, k = i - a * N;
  const double lo = edges[(size_t)a * (N + 1) + k], w = edges[(size_t)a * (N + 1) + k + 1] - lo;
  tab64[i] = make_double2(lo, w);
  tab32[i] = make_float2((float)lo, (float)w);
}

size_t align256(size_t b) { return (b + 255) & ~size_t(255); }

}  // namespace

extern "C" vegas_status vegas_eval_noalloc(const vegas_config* cfg, const vegas_integrand* fn,
                                           const double* edges, uint32_t it, double* out) {
  if (!cfg || !fn || !edges || !out) return thread_fail(VEGAS_EINVAL, "NULL argument");
  const int d = cfg->ndim, N = cfg->nbins;
  if (d < 1 || d > GVEGAS_MAXDIM) return thread_fail(VEGAS_EINVAL, "ndim %d outside 1..%d", d, GVEGAS_MAXDIM);
  if (N < 2 || N > GVEGAS_MAXBINS) return thread_fail(VEGAS_EINVAL, "nbins %d outside 2..%d", N, GVEGAS_MAXBINS);
  if (cfg->ncall < 2 || cfg->ncall > (int64_t)1 << 32)
    return thread_fail(VEGAS_EINVAL, "ncall %lld outside 2..2^32", (long long)cfg->ncall);
  if (cfg->precision < VG_FP64 || cfg->precision > VG_FP32_ACCCOMP)
    return thread_fail(VEGAS_EINVAL, "unknown precision %d", cfg->precision);
  if (it > 0x7FFFFFFFu) return thread_fail(VEGAS_EINVAL, "iteration index must be < 2^31");
  const int ybits = cfg->ybits ? cfg->ybits : (cfg->precision == VG_FP64 ? 53 : 24);
  if (ybits != 24 && ybits != 53) return thread_fail(VEGAS_EINVAL, "ybits must be 24 or 53");
  if (fn->ndim != d) return thread_fail(VEGAS_EINVAL, "integrand ndim %d != config ndim %d", fn->ndim, d);
  const int np = gv::expected_nparams(fn->kind, d);
  if (np < 0) return thread_fail(VEGAS_EINVAL, "unknown integrand kind %d", fn->kind);
  if (fn->nparams != np || (np > 0 && !fn->params))
    return thread_fail(VEGAS_EINVAL, "integrand kind %d needs %d parameters, got %d", fn->kind, np, fn->nparams);
  const int g = cfg->nstrat < 1 ? 1 : cfg->nstrat;
  uint64_t G = 1;
  for (int a = 0; a < d; ++a) {
    G *= (uint64_t)g;
    if (G > (uint64_t)cfg->ncall) return thread_fail(VEGAS_EINVAL, "nstrat^ndim exceeds ncall");
  }
  if ((uint64_t)cfg->ncall % G != 0) return thread_fail(VEGAS_EINVAL, "ncall must be a multiple of nstrat^ndim");
  if (G > 1 && (uint64_t)cfg->ncall / G < 2) return thread_fail(VEGAS_EINVAL, "need >= 2 points per hypercube");
  if ((int64_t)g * N >= (ybits == 53 ? 2048 : (1 << 30)))
    return thread_fail(VEGAS_EINVAL, "nstrat * nbins too large for %d-bit sampling", ybits);

  DerivedBlock db;
  double scale = 1.0;
  char why_buf[128] = {0};
  {
    std::string why;
    if (!gv::derive_params(fn->kind, d, fn->params, db.v, &scale, &why)) {
      snprintf(why_buf, sizeof why_buf, "%s", why.c_str());
      return thread_fail(VEGAS_EINVAL, "%s", why_buf);
    }
    db.v[gv::kNumDerived] = scale;
  }
  gv::KernelEntry ke{};
  if (!lookup_kernel(fn->kind, cfg->precision, ybits, d, &ke))
    return thread_fail(VEGAS_EINVAL, "no kernel for kind %d, ndim %d", fn->kind, d);
  int ppt_min = 1;
  if (ke.sample_spec && d == ke.dm && ybits == 24 && (g & (g - 1)) == 0 && (int64_t)g * N <= 256) {
    ke.sample = ke.sample_spec;
    ppt_min = ke.spec_ppt_min;
  }

  // Per-device set-up on the first call for the current device: the device
  // address of the scratch array (its host-side name is only a stand-in).
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return thread_fail(VEGAS_ECUDA, "cudaGetDevice: %s", cudaGetErrorString(e));
  if (dev < 0 || dev >= kNoAllocMaxDevices) return thread_fail(VEGAS_EINVAL, "device index %d too large", dev);
  unsigned char* scratch;
  int sms;
  {
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_noalloc_ptr[dev]) {
      void* p = nullptr;
      e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
      if (e != cudaSuccess) return thread_fail(VEGAS_ECUDA, "cudaGetSymbolAddress: %s", cudaGetErrorString(e));
      int n = 0;
      e = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
      if (e != cudaSuccess) return thread_fail(VEGAS_ECUDA, "device attribute: %s", cudaGetErrorString(e));
      g_noalloc_sms[dev] = n;
      g_noalloc_ptr[dev] = static_cast<unsigned char*>(p);
    }
    scratch = g_noalloc_ptr[dev];
    sms = g_noalloc_sms[dev];
  }

  // Launch shape (as for a context) with the CTA count bounded by the rows
  // of partial sums that fit in the scratch array.
  const int dN = d * N;
  const size_t off_st = 0;
  const size_t off_dp = align256(off_st + sizeof(GState));
  const size_t off_t64 = align256(off_dp + sizeof(double) * (gv::kNumDerived + 1));
  const size_t off_t32 = align256(off_t64 + sizeof(double2) * dN);
  const size_t off_rows = align256(off_t32 + sizeof(float2) * dN);
  const size_t row_bytes = sizeof(double) * (2 * (size_t)dN + gv::kTotCols);
  const int64_t max_rows = off_rows < kNoAllocScratchBytes ? (int64_t)((kNoAllocScratchBytes - off_rows - 512) / row_bytes) : 0;
  if (max_rows < 1)
    return thread_fail(VEGAS_EINVAL, "ndim * nbins = %d too large for the %zu-byte no-allocation scratch", dN,
                       kNoAllocScratchBytes);
  const uint64_t nc = (uint64_t)cfg->ncall / G;
  const int strat = G > 1;
  gv::PassShape ps;
  int ppt = d <= 8 ? 2 : 1, cap = 0;
  const void* col = pick_col(ke, d, ybits, g, N);
  if (!col || !shape_col(col, ke, d, N, sms, 0, 0, G, nc, (uint64_t)cfg->ncall, max_rows, 0, &ps, &e)) {
    const int threads = 256;
    auto occ_of = [&](int cp, int) -> int {
      const size_t sm = ke.smem(d, N, cp);
      int o = 0;
      if (e != cudaSuccess || sm + kSampleStatic > 227 * 1024) return 0;
      e = gv_raise_smem_limit(ke.sample, sm);
      if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, ke.sample, threads, sm);
      return e == cudaSuccess ? o : 0;
    };
    int occ_cap = 0;
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ_cap, ke.sample, threads, 0);
    const gv::TileShape t = e == cudaSuccess ? gv::choose_tile(threads, N, 0, ppt_min, occ_cap, occ_of) : gv::TileShape{1, 4, 0};
    if (e != cudaSuccess) return thread_fail(VEGAS_ECUDA, "launch configuration: %s", cudaGetErrorString(e));
    if (t.occ < 1) return thread_fail(VEGAS_EINVAL, "sampling kernel does not fit in shared memory");
    ppt = t.ppt;
    cap = t.cap;
    ps.fn = ke.sample;
    ps.threads = threads;
    ps.smem = ke.smem(d, N, cap);
    e = gv_raise_smem_limit(ke.sample, ps.smem);
    const int64_t most = std::min<int64_t>((int64_t)sms * t.occ, max_rows);
    ps.lanes = strat ? gv::choose_lanes(G, nc, threads, most) : 1;
    const uint64_t units = strat ? G * (uint64_t)ps.lanes : (uint64_t)cfg->ncall;
    ps.ctas = (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)((units + threads - 1) / threads), most));
  }
  if (e != cudaSuccess) return thread_fail(VEGAS_ECUDA, "launch configuration: %s", cudaGetErrorString(e));
  const int ctas = ps.ctas;
  double* part_tot = reinterpret_cast<double*>(scratch + off_rows);
  double* part_bins = reinterpret_cast<double*>(scratch + align256(off_rows + sizeof(double) * gv::kTotCols * ctas));
  GState* st = reinterpret_cast<GState*>(scratch + off_st);

  cudaStream_t s = (cudaStream_t)cfg->stream;
  // Contents left by the previous call: the pass state must start cleared;
  // tables, partial rows and totals are overwritten in full.
  k_noalloc_setup<<<(std::max(dN, 256) + 255) / 256, 256, 0, s>>>(
      db, reinterpret_cast<double*>(scratch + off_dp), st, edges, d, N, reinterpret_cast<double2*>(scratch + off_t64),
      reinterpret_cast<float2*>(scratch + off_t32));
  e = cudaGetLastError();
  if (e != cudaSuccess) return thread_fail(VEGAS_ECUDA, "no-allocation set-up: %s", cudaGetErrorString(e));

  gv::SampleArgs A{};
  A.d = d;
  A.N = N;
  A.g = g;
  A.ybits = ybits;
  A.lanes = ps.lanes;
  A.cap = cap;
  A.ppt = ppt;
  A.strat = strat;
  A.key0 = (uint32_t)cfg->seed;
  A.key1 = (uint32_t)(cfg->seed >> 32);
  gv::philox_key_schedule(A.key0, A.key1, A.ks);
  A.instance = cfg->instance;
  A.it_override = (int)it;
  A.ncall = (uint64_t)cfg->ncall;
  A.nc = (uint32_t)nc;
  A.ncubes = (uint32_t)G;
  A.cube_mul = gv::cube_multiplier(G);
  A.parts = 1;
  A.units = (uint32_t)G;
  A.vl = (uint32_t)ps.lanes;
  A.per_lane = (uint32_t)((nc + A.vl - 1) / A.vl);
  A.niter = 1;
  A.g_pow2 = (g & (g - 1)) == 0;
  A.g_log2 = 0;
  while ((1 << A.g_log2) < g) ++A.g_log2;
  A.t32 = (int64_t)g * N <= 256;
  const double gb = (double)g * std::ldexp(1.0, ybits);
  A.inv_gb_d = 1.0 / gb;
  A.inv_gb_f = (float)(1.0 / gb);
  A.inv_nc = 1.0 / (double)nc;
  A.inv_nc1 = nc > 1 ? 1.0 / (double)(nc - 1) : 0.0;
  A.nparts = ctas;
  A.tab = cfg->precision == VG_FP64 ? (const void*)(scratch + off_t64) : (const void*)(scratch + off_t32);
  A.dparams = reinterpret_cast<const double*>(scratch + off_dp);
  A.st = st;
  A.part_bins = part_bins;
  A.part_tot = part_tot;
  A.cubes = nullptr;
  void* args[] = {&A};
  e = cudaLaunchKernel(ps.fn, dim3(ctas), dim3(ps.threads), args, ps.smem, s);
  gv::FinArgs F{};
  F.d = d;
  F.N = N;
  F.nparts = ctas;
  F.niter = 1;
  F.parts = 1;
  F.strat = strat;
  F.refine = 0;
  F.record = 0;
  F.pair32 = cfg->precision == VG_FP32_ACCCOMP;
  F.ncall = (uint64_t)cfg->ncall;
  F.ncubes = G;
  F.scale = reinterpret_cast<double*>(scratch + off_dp) + gv::kNumDerived;
  F.alpha = cfg->alpha;
  F.part_bins = part_bins;
  F.part_tot = part_tot;
  F.bins = out;
  F.edges = nullptr;
  F.tab64 = reinterpret_cast<double2*>(scratch + off_t64);
  F.tab32 = reinterpret_cast<float2*>(scratch + off_t32);
  F.st = st;
  F.result = out + 2 * (size_t)dN;
  if (e == cudaSuccess) e = gv_launch_finish(&F, s);
  if (e != cudaSuccess) return thread_fail(VEGAS_ECUDA, "no-allocation pass: %s", cudaGetErrorString(e));
  return VEGAS_OK;
}
