// finalize.cu -- steps 4-6 of Sec. 2.1 after the sampling pass, all on the
// GPU in FP64 (the paper ran them on the host, Sec. 2.2), in one launch:
//   k_finish    fixed-order reduction of the per-CTA partial rows into the
//               per-bin sums S1, S2 and the iteration totals; one cluster of
//               CTAs per axis, whose first CTA then runs the grid
//               optimisation (Lepage 1978: smoothing, log-compression with
//               exponent alpha, rebinning to equal weight), and one CTA that
//               forms the iteration estimate, the inverse-variance
//               combination, chi^2 and the ACC test.
#include <cooperative_groups.h>

#include <map>
#include <mutex>
#include <utility>

#include "common.cuh"
#include "kernels.h"
#include "refine.cuh"

namespace gv {

// CTAs per cluster of k_finish: an axis's partial rows are shared out over
// this many SMs.
constexpr int kFinishCluster = 8;
// Thread slices per column within a CTA, at most.
constexpr int kFinishSlices = 8;

// Sum of one per-CTA totals column by one warp (lanes stride the rows, eight
// loads in flight, then a fixed xor butterfly); every lane gets the sum.
__device__ double total_column(const double* src, int np, int lane) {
  double acc = 0.0;
  int r = lane;
  for (; r + 7 * 32 < np; r += 8 * 32) {
    double v[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = __ldcg(src + r + 32 * j);
#pragma unroll
    for (int j = 0; j < 8; ++j) acc += v[j];
  }
  for (; r < np; r += 32) acc += __ldcg(src + r);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
  return acc;
}

// A partial sum of the rows: a compensated FP32 pair or a double.
__device__ __forceinline__ void psum_add(fpair& a, const float2& v) { comp_merge(a, fpair{v.x, v.y}); }
__device__ __forceinline__ void psum_add(double& a, const double& v) { a += v; }
__device__ __forceinline__ void psum_merge(fpair& a, const fpair& b) { comp_merge(a, b); }
__device__ __forceinline__ void psum_merge(double& a, const double& b) { a += b; }
__device__ __forceinline__ double psum_value(const fpair& a) { return comp_value(a); }
__device__ __forceinline__ double psum_value(const double& a) { return a; }
__device__ __forceinline__ void psum_zero(fpair& a) { a = fpair{0.f, 0.f}; }
__device__ __forceinline__ void psum_zero(double& a) { a = 0.0; }

// The 2N columns (S1 then S2) of axis a over the rows of this cluster: CTA
// `rank` takes rows rank, rank + 8, ..., its threads the columns, in
// nsl slices of those rows; the slices, then the CTAs, are merged in order
// by the cluster's first CTA.  The rows are stored [CTA][2 d N], so a warp
// reads consecutive columns of a row.  V: stored element, S: running sum.
// Returns in the first CTA's s2[] the scaled S2 sums.
template <int T, typename V, typename S>
__device__ __forceinline__ void reduce_axis(const FinArgs& F, int a, unsigned rank, S* buf, double* s2) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const int N = F.N, dN = F.d * N, C = 2 * N, np = F.nparts;
  const int nsl = min(kFinishSlices, max(1, T / C));
  const int j = threadIdx.x % C, sl = threadIdx.x / C;  // column and slice (C <= T: one column per thread)
  const size_t stride = 2 * (size_t)dN;
  for (int c = C <= T ? j : (int)threadIdx.x; c < C && sl < nsl; c += C <= T ? C : T) {
    const int slice = C <= T ? sl : 0;
    const V* src = reinterpret_cast<const V*>(F.part_bins) + (c < N ? a * N + c : dN + a * N + (c - N));
    const int step = kFinishCluster * nsl;
    int r = (int)rank + kFinishCluster * slice;
    S acc;
    psum_zero(acc);
    for (; r + 7 * step < np; r += 8 * step) {
      V v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = __ldcg(src + (size_t)(r + u * step) * stride);
#pragma unroll
      for (int u = 0; u < 8; ++u) psum_add(acc, v[u]);
    }
    V v[8];
    int m = 0;
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (r + u * step < np) {
        v[u] = __ldcg(src + (size_t)(r + u * step) * stride);
        m = u + 1;
      }
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (u < m) psum_add(acc, v[u]);
    buf[slice * C + c] = acc;
  }
  __syncthreads();
  for (int c = threadIdx.x; c < C && nsl > 1; c += T) {
    S acc = buf[c];
    for (int q = 1; q < nsl; ++q) psum_merge(acc, buf[q * C + c]);
    buf[c] = acc;
  }
  cl.sync();
  if (rank == 0) {
    const double sc = *F.scale;
    for (int c = threadIdx.x; c < C; c += T) {
      S q[kFinishCluster];
#pragma unroll
      for (int k = 0; k < kFinishCluster; ++k) q[k] = cl.map_shared_rank(buf, k)[c];
#pragma unroll
      for (int k = 1; k < kFinishCluster; ++k) psum_merge(q[0], q[k]);
      const double v = psum_value(q[0]) * (c < N ? sc : sc * sc);
      F.bins[c < N ? a * N + c : dN + a * N + (c - N)] = v;
      if (c >= N) s2[c - N] = v;
    }
  }
  cl.sync();  // the first CTA has read the others' sums; s2 is complete
}

// The totals of iteration j from the hypercubes' part sums, by the whole
// cluster: each thread adds the parts of its cubes in order, forms their
// means and variances and writes the last iteration's cube sums; the threads
// of a warp, the warps and the CTAs are merged in fixed order.  V: a part's
// two sums (16 bytes), S: running sum.
__device__ __forceinline__ void cube_load(const float4& v, fpair& c1, fpair& c2) {
  c1 = fpair{v.x, v.y};
  c2 = fpair{v.z, v.w};
}
__device__ __forceinline__ void cube_load(const double2& v, double& c1, double& c2) {
  c1 = v.x;
  c2 = v.y;
}
__device__ __forceinline__ fpair psum_xor(const fpair& a, int off) {
  return fpair{__shfl_xor_sync(0xffffffffu, a.hi, off), __shfl_xor_sync(0xffffffffu, a.lo, off)};
}
__device__ __forceinline__ double psum_xor(const double& a, int off) { return __shfl_xor_sync(0xffffffffu, a, off); }

template <int T, typename V, typename S>
__device__ __forceinline__ void reduce_cubes(const FinArgs& F, int j, unsigned rank, S (*buf)[4], double* tot) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const uint32_t G = (uint32_t)F.ncubes;
  const V* src = reinterpret_cast<const V*>(F.cube_part) + (size_t)j * F.parts * G;
  S t[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) psum_zero(t[q]);
  const bool store = F.cubes && j == F.niter - 1;
  for (uint32_t i = rank * T + threadIdx.x; i < G; i += kFinishCluster * T) {
    S c1, c2;
    psum_zero(c1);
    psum_zero(c2);
    for (uint32_t p = 0; p < F.parts; p += 4) {  // (a power of two above one: 2, or fours)
      V v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (p + u < F.parts) v[u] = __ldcg(src + (size_t)(p + u) * G + i);
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (p + u < F.parts) {
          S a1, a2;
          cube_load(v[u], a1, a2);
          psum_merge(c1, a1);
          psum_merge(c2, a2);
        }
    }
    cube_totals(F.inv_nc, F.inv_nc1, c1, c2, t);
    if (store) cube_store(F.cubes, cube_of(G, F.cube_mul, i), c1, c2);
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = T / 32;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) psum_merge(t[q], psum_xor(t[q], off));
    if (lane == 0) buf[warp][q] = t[q];
  }
  __syncthreads();
  if (threadIdx.x < 4) {
    S a = buf[0][threadIdx.x];
    for (int w = 1; w < nw; ++w) psum_merge(a, buf[w][threadIdx.x]);
    buf[0][threadIdx.x] = a;
  }
  cl.sync();
  if (rank == 0 && threadIdx.x < 4) {
    S a = buf[0][threadIdx.x];
    for (int r = 1; r < kFinishCluster; ++r) psum_merge(a, cl.map_shared_rank(&buf[0][0], r)[threadIdx.x]);
    tot[threadIdx.x] = psum_value(a);
  }
  cl.sync();  // the others' sums have been read; buf may be used again
}

// Step 6 for the pass, by one full warp (lane 0 writes the state).
__device__ void record_iteration(const FinArgs& F, const double* t, bool combine) {
  GState* st = F.st;
  const int lane = threadIdx.x & 31;
  double I, var;
  if (F.strat) {
    const double G = (double)F.ncubes;
    I = t[TOT_SI] / G;
    var = t[TOT_SV] / (G * G);
  } else {
    const double n = (double)F.ncall;
    I = t[TOT_SW] / n;
    var = (t[TOT_SW2] / n - I * I) / (n - 1.0);
    if (var < 0.0) var = 0.0;
  }
  if (lane == 0) {
    st->last_I = I;
    st->last_var = var;
    st->last_sw = t[TOT_SW];
    st->last_sw2 = t[TOT_SW2];
    st->last_nonfinite = (long long)t[TOT_NONFINITE];
  }
  if (F.result && lane == 0) {
    F.result[0] = I;
    F.result[1] = var;
    F.result[2] = t[TOT_SW];
    F.result[3] = t[TOT_SW2];
    F.result[4] = t[TOT_NONFINITE];
  }
  if (!F.record) {
    if (F.mirror) mirror_state(F.mirror, st);
    return;
  }
  int h = st->nhist;
  if (h < kMaxHist) {
    if (lane == 0) {
      st->hist[h][0] = I;
      st->hist[h][1] = var;
      st->nhist = h + 1;
    }
    ++h;
  }
  __syncwarp();
  if (lane == 0) {
    st->nonfinite += (long long)t[TOT_NONFINITE];
    st->samples += (long long)F.ncall;
    st->it += 1;
  }
  // Inverse-variance combination over the window (Lepage): in a call without
  // an ACC target only the last pass's combination can be read.
  if (!combine) return;
  double Ib, sg, chi;
  combine_history(st->hist, h, &Ib, &sg, &chi);
  if (lane == 0) {
    st->I = Ib;
    st->sigma = sg;
    st->chi2 = chi;
    if (st->acc > 0.0 && sg < st->acc * fabs(Ib)) {
      st->done = 1;
      st->stopped = 1;
    }
  }
  if (F.mirror) mirror_state(F.mirror, st);
}

// Steps 4-6 after a sampling pass in one launch.  Cluster a < d reduces the
// 2N columns (S1, S2) of axis a and its first CTA refines the axis; the last
// cluster's first CTA reduces the iteration totals and records the
// iteration.  No block waits for another cluster.  `live` was latched by the
// sampling kernel of this pass and the ACC test below writes only `done`.
//
// Bound by latency: the rows are read once (dgauss8: 152 rows of 6.4 KB)
// with every load of a thread in flight, the merge crosses the SMs through
// distributed shared memory, without a memory fence and an arrival counter,
// and what remains is the dependent FP64 chain of the refinement.
//
// T threads: two to eight slices of an axis's 2 N columns, so 256 up to 64 bins
// and 512 beyond (one column each at 256 bins), two CTAs of which fit an SM, as
// the clusters of 16 and more axes need (d = 4, us of this kernel, 256 threads ->
// 512: 160 bins, 456 rows 15.0 -> 11.9; 256 bins, 304 rows 13.9 -> 11.65; d = 8, 200
// bins 11.9 -> 9.85).
template <int T>
__global__ void __cluster_dims__(kFinishCluster, 1, 1) __launch_bounds__(T, T > kFinishThreads ? 2 : 0) k_finish(const FinArgs F) {
  // (the slices' partial sums, 8 bytes per thread, or the cubes', 64 per warp)
  __shared__ __align__(16) unsigned char buf[T * 16];
  __shared__ double s2[kMaxBins];
  __shared__ double tot[kMergeIters][kTotCols];
  GState* st = F.st;
  if (!st->live) return;  // (uniform over the launch)
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned rank = blockIdx.x % kFinishCluster;
  const int group = F.nobins ? F.d : (int)(blockIdx.x / kFinishCluster);
  if (group < F.d) {
    if (F.pair32)
      reduce_axis<T, float2, fpair>(F, group, rank, reinterpret_cast<fpair*>(buf), s2);
    else
      reduce_axis<T, double, double>(F, group, rank, reinterpret_cast<double*>(buf), s2);
    if (rank != 0 || !F.refine) return;
    // one thread per bin (whole warps) refines; the other warps leave
    const int N = F.N, a = group;
    const Team t{min(T, (N + 31) / 32 * 32)};
    if ((int)threadIdx.x >= t.n) return;
    refine_axis_core(s2, F.edges + (size_t)a * (N + 1), F.tab64 + (size_t)a * N, F.tab32 + (size_t)a * N, N,
                     F.alpha, t);
    return;
  }
  // The totals of each iteration: the columns over the partial rows, or,
  // where several groups share a hypercube, the cubes' own sums over the
  // cluster (and only the non-finite count from the rows).
  if (F.parts > 1u) {
    for (int j = 0; j < F.niter; ++j) {
      if (F.pair32)
        reduce_cubes<T, float4, fpair>(F, j, rank, reinterpret_cast<fpair(*)[4]>(buf), tot[j]);
      else
        reduce_cubes<T, double2, double>(F, j, rank, reinterpret_cast<double(*)[4]>(buf), tot[j]);
    }
  }
  if (rank != 0) return;
  const double s1 = *F.scale;
  for (int i = warp; i < 5 * F.niter; i += T / 32) {
    const int j = i / 5, q = i - 5 * j;
    if (F.parts > 1u && q != TOT_NONFINITE) continue;
    const double v = total_column(F.part_tot + ((size_t)j * kTotCols + q) * F.nparts, F.nparts, lane);
    if (lane == 0) tot[j][q] = v;
  }
  __syncthreads();
  if (threadIdx.x < 5 * F.niter) {
    const int j = threadIdx.x / 5, q = threadIdx.x - 5 * j;
    tot[j][q] *= (q == TOT_SW || q == TOT_SI) ? s1 : (q == TOT_NONFINITE ? 1.0 : s1 * s1);
  }
  __syncthreads();
  if (warp == 0)
    for (int j = 0; j < F.niter; ++j) record_iteration(F, tot[j], F.combine && j == F.niter - 1);
}

// Column sums of a [ncols][nrows] partial block (one warp per column,
// lanes stride the rows, fixed xor butterfly).
__global__ void __launch_bounds__(256) k_colsum(const double* part, int ncols, int nrows, double* out) {
  const int lane = threadIdx.x & 31;
  const int col = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (col >= ncols) return;
  double acc = 0.0;
  for (int r = lane; r < nrows; r += 32) acc += part[(size_t)col * nrows + r];
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
  if (lane == 0) out[col] = acc;
}

// Window / stop-flag bookkeeping between passes (one warp; its first lane);
// CTL_SET_ITER sets the Philox iteration counter.
__device__ __forceinline__ void control(GState* st, int ops, double acc, uint32_t it) {
  if (ops & CTL_SET_ITER) st->it = it;
  if (ops & CTL_SNAPSHOT) {
    st->ph1_I = st->I;
    st->ph1_sigma = st->sigma;
    st->ph1_chi2 = st->chi2;
    st->ph1_iters = st->nhist;
    st->ph1_stopped = st->stopped;
    st->ph1_nonfinite = st->nonfinite;
    st->ph1_samples = st->samples;
  }
  if (ops & CTL_RESET_WINDOW) {
    st->nhist = 0;
    st->nonfinite = 0;
    st->samples = 0;
    st->I = st->sigma = st->chi2 = 0.0;
  }
  if (ops & CTL_SET_ACC) {
    st->acc = acc;
    st->done = 0;
    st->stopped = 0;
  }
}

__global__ void k_control(GState* st, int ops, double acc, uint32_t it, GState* mirror) {
  if (threadIdx.x == 0) control(st, ops, acc, it);
  mirror_state(mirror, st);
}

// Uniform grid e_a[k] = k / N (step 1) and its tables.
__global__ void k_uniform_grid(double* edges, int d, int N, double2* tab64, float2* tab32) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= d * (N + 1)) return;
  const int a = i / (N + 1), k = i - a * (N + 1);
  const double lo = (double)k / (double)N;
  edges[i] = lo;
  if (k < N) {
    const double w = (double)(k + 1) / (double)N - lo;
    tab64[a * N + k] = make_double2(lo, w);
    tab32[a * N + k] = make_float2((float)lo, (float)w);
  }
}

// Pure table rebuild (after vegas_set_grid): tab64 / tab32 from edges.
__global__ void k_tables(const double* edges, int d, int N, double2* tab64, float2* tab32) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= d * N) return;
  const int a = i / N, k = i % N;
  const double lo = edges[(size_t)a * (N + 1) + k], w = edges[(size_t)a * (N + 1) + k + 1] - lo;
  tab64[i] = make_double2(lo, w);
  tab32[i] = make_float2((float)lo, (float)w);
}

}  // namespace gv

extern "C" {

// The sampling kernels run with most of the unified L1 / shared memory as
// shared memory; the small kernels between them ask for the same split, so
// that an SM need not change its partition (and drain) at every boundary.
cudaError_t gv_prepare_aux_kernels(void) {
  const void* fns[] = {(const void*)gv::k_finish<gv::kFinishThreads>, (const void*)gv::k_finish<gv::kMaxFinishThreads>, (const void*)gv::k_colsum,
                       (const void*)gv::k_control, (const void*)gv::k_uniform_grid, (const void*)gv::k_tables};
  for (const void* f : fns) {
    const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout,
                                               (int)cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// Dynamic shared-memory limit of a kernel on the current device, raised to
// at least `bytes` and never lowered.  Contexts, batches and the
// no-allocation pass share compiled kernels with different tile shapes;
// captured graphs and later launches of each keep needing the size it
// asked for, so the limit only grows (mutex: any host thread may call).
cudaError_t gv_raise_smem_limit(const void* fn, size_t bytes) {
  static std::mutex mu;
  static std::map<std::pair<int, const void*>, size_t> limit;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lock(mu);
  size_t& cur = limit[std::make_pair(dev, fn)];
  if (bytes <= cur) return cudaSuccess;
  e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e == cudaSuccess) cur = bytes;
  return e;
}

cudaError_t gv_launch_finish(const gv::FinArgs* F, cudaStream_t s) {
  const int blocks = gv::kFinishCluster * (F->nobins ? 1 : F->d + 1);
  if (F->N <= 64 || F->nobins)
    gv::k_finish<gv::kFinishThreads><<<blocks, gv::kFinishThreads, 0, s>>>(*F);
  else
    gv::k_finish<gv::kMaxFinishThreads><<<blocks, gv::kMaxFinishThreads, 0, s>>>(*F);
  return cudaGetLastError();
}

cudaError_t gv_launch_colsum(const double* part, int ncols, int nrows, double* out, cudaStream_t s) {
  gv::k_colsum<<<(ncols + 7) / 8, 256, 0, s>>>(part, ncols, nrows, out);
  return cudaGetLastError();
}

cudaError_t gv_launch_control(gv::GState* st, int ops, double acc, uint32_t it, gv::GState* mirror, cudaStream_t s) {
  gv::k_control<<<1, 32, 0, s>>>(st, ops, acc, it, mirror);
  return cudaGetLastError();
}

cudaError_t gv_launch_uniform_grid(double* edges, int d, int N, double2* t64, float2* t32, cudaStream_t s) {
  const int n = d * (N + 1);
  gv::k_uniform_grid<<<(n + 255) / 256, 256, 0, s>>>(edges, d, N, t64, t32);
  return cudaGetLastError();
}

cudaError_t gv_launch_tables(const double* edges, int d, int N, double2* t64, float2* t32,
                             cudaStream_t s) {
  const int n = d * N;
  gv::k_tables<<<(n + 255) / 256, 256, 0, s>>>(edges, d, N, t64, t32);
  return cudaGetLastError();
}
}
