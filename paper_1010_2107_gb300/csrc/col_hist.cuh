// col_hist.cuh -- step 4's per-bin sums without atomics: the column histogram
// of the FP32 form (compensated sums), shared by the sampling kernels.
//
// Shared-memory float atomics are compare-and-swap loops on this GPU (1.15
// updates per SM-clock, measured), so the sums need another way to keep two
// lanes off one cell.  Here the lanes of a warp own the cells: after a warp
// has evaluated its points (one lane per point), their weights and bins are
// handed over through a small per-warp staging area, and lane l then works
// for axis l mod d on the points l div d, l div d + P, ... (P = 32 div d
// points at a time).  Each lane has a private column of N cells (S1, S2), so
// its read-modify-write races with nobody, needs no atomic, no barrier and
// no overflow path, and the 32 columns sit side by side (row k holds bin k
// of all lanes), so every access is free of bank conflicts.
//
// The updates of one hand-over run as short steps between the axes of the
// next points' evaluation (EXACT: where the dimension is a compile-time
// constant): a step finishes the previous read-modify-write and starts the
// next one, so the load's latency lies under the evaluation's arithmetic
// (two-peak Gaussian, d = 8, 2^22 points: 70.5 -> 61.4 us per pass; with a
// run-time dimension the steps' own bookkeeping costs more than it hides,
// 78.7 -> 85.2 us at d = 7, so there they run together after it).
//
// The cells are accessed through volatile inline assembly without a memory
// clobber: these accesses keep their order among themselves, while the table
// lookups and constants around them stay free to move.  Ordinary accesses to
// the cells (bind clears them, col_sum folds and clears) are not ordered
// against them by the compiler, so a barrier has to stand wherever the two meet:
// bind ends in __syncwarp, a fold begins and ends in __syncthreads.
//
// What it costs per 32 point-axes, in shared-memory wavefronts: bin byte 1,
// cell load 2, cell store 2, weight 1/4, about 5.5 with the staging writes
// (6.9 measured with the folds, d = 8), against 11.2 for bucketed tiles (claim
// atomic 3.8, slot store 3.6, gather);
// and about 6 issue slots against 16.  The price is memory: 256 N bytes per
// warp (12.8 KB at 50 bins), which bounds the warps per SM (16 at 50 bins).
#pragma once

#include "common.cuh"

namespace gv {

// Additions a lane may make to its column in plain FP32 before the CTA's
// columns are folded into compensated pairs.  A cell then holds the sum of
// at most this many terms (of this many div N in a grid that spreads them).
constexpr int kColFoldAdds = 1024;

// DM bounds the dimension d (equal to it when EXACT); PIF points per lane are
// handed over at a time.
template <int DM, bool EXACT, int PIF>
struct ColHist {
  static constexpr int NPT = 32 * PIF;     // points of a warp per hand-over
  static constexpr int KW = (DM + 3) / 4;  // words of packed bins
  static constexpr int BS = 4 * KW;        // bytes of a point's bins

  static __host__ __device__ constexpr int points_per_step(int d) { return 32 / d; }
  static __host__ __device__ constexpr int steps(int d) { return (NPT + points_per_step(d) - 1) / points_per_step(d); }
  // EXACT: a lane's weights lie together and are read four steps at a time
  static __host__ __device__ constexpr int steps4(int d) { return (steps(d) + 3) / 4 * 4; }
  static __host__ __device__ constexpr int slots(int d) { return points_per_step(d) * steps4(d); }
  static __host__ __device__ constexpr size_t stage_bytes(int d) {
    return (size_t)((slots(d) * 4 + slots(d) * BS + 15) & ~15);
  }
  static __host__ __device__ constexpr size_t cell_bytes(int N) { return (size_t)N * 32 * sizeof(float2); }
  static __host__ __device__ constexpr size_t warp_bytes(int d, int N) { return stage_bytes(d) + cell_bytes(N); }

  int P, S;              // points per step, steps per hand-over
  uint32_t cells;        // this lane's column (shared-memory address): cells + 256 k
  float* put_w[PIF];     // where this lane stages its points: weights
  unsigned char* put_b;  // ... and bins (the first point's)
  const float* get_w;    // the weights of this lane's steps
  const unsigned char* get_b;  // the bin bytes of this lane's steps, P * BS apart

  // EXACT: the read-modify-write under way, and the bins and weights of a
  // group of four steps and the next
  float2 v;
  float w;
  uint32_t addr;
  uint32_t kq[2][4];
  float4 wq[2];

  // base: the warp's area (16-byte aligned; cells first, then the staging)
  __device__ __forceinline__ void bind(unsigned char* base, int d_, int N, int lane) {
    const int d = EXACT ? DM : d_;
    P = points_per_step(d);
    S = steps(d);
    const int S4 = steps4(d), W = slots(d);
    cells = (uint32_t)__cvta_generic_to_shared(base) + 8u * (uint32_t)lane;
    float* sw = reinterpret_cast<float*>(base + cell_bytes(N));
    unsigned char* sb = base + cell_bytes(N) + 4 * W;
#pragma unroll
    for (int q = 0; q < PIF; ++q) {  // point p = 32 q + lane belongs to lanes (p mod P) d .., step p div P
      const int p = 32 * q + lane;
      put_w[q] = sw + (EXACT ? (p % P) * S4 + p / P : p);
    }
    put_b = sb + lane * BS;
    // lanes past P d repeat the last point's axes into columns nobody reads
    const int sub = min(lane / d, P - 1), ax = lane % d;
    get_w = sw + (EXACT ? sub * S4 : sub);
    get_b = sb + sub * BS + ax;
    // clear the columns and the staging area (the first hand-over taken over
    // is empty, and the slots no point fills keep the weight zero)
    for (int i = lane; i < N * 16; i += 32) reinterpret_cast<float4*>(base)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int i = lane; i < W * (4 + BS) / 4; i += 32) reinterpret_cast<uint32_t*>(sw)[i] = 0u;
    __syncwarp();
  }

  // Stage point q of this lane: weight and packed bins.
  __device__ __forceinline__ void put(int q, float wt, const uint32_t (&kb)[KW]) {
    *put_w[q] = wt;
    uint32_t* b = reinterpret_cast<uint32_t*>(put_b + 32 * BS * q);
    if constexpr (KW % 4 == 0) {
#pragma unroll
      for (int i = 0; i < KW; i += 4) *reinterpret_cast<uint4*>(b + i) = make_uint4(kb[i], kb[i + 1], kb[i + 2], kb[i + 3]);
    } else if constexpr (KW % 2 == 0) {
#pragma unroll
      for (int i = 0; i < KW; i += 2) *reinterpret_cast<uint2*>(b + i) = make_uint2(kb[i], kb[i + 1]);
    } else {  // an odd stride in words: free of bank conflicts
#pragma unroll
      for (int i = 0; i < KW; ++i) b[i] = kb[i];
    }
  }

  static __device__ __forceinline__ float2 load(uint32_t at) {
    float2 r;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(r.x), "=f"(r.y) : "r"(at));
    return r;
  }
  static __device__ __forceinline__ void add(uint32_t at, float2 r, float wt) {
    r.x += wt;
    r.y = fmaf(wt, wt, r.y);
    asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(at), "f"(r.x), "f"(r.y));
  }
  __device__ __forceinline__ void group(int j, uint32_t (&k)[4], float4& wt) const {
    wt = *reinterpret_cast<const float4*>(get_w + j);
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (j + u < steps(DM)) k[u] = get_b[(j + u) * points_per_step(DM) * BS];
  }

  // Take over what the warp has staged (after a __syncwarp).
  __device__ __forceinline__ void begin() {
    if constexpr (EXACT) group(0, kq[0], wq[0]);
  }
  // Step i of the hand-over (a compile-time constant in unrolled code):
  // finish step i - 1, start step i, read the operands ahead.
  __device__ __forceinline__ void step(int i) {
    const int g = (i >> 2) & 1, u = i & 3;
    if (i > 0) add(addr, v, w);
    w = u == 0 ? wq[g].x : (u == 1 ? wq[g].y : (u == 2 ? wq[g].z : wq[g].w));
    addr = cells + 256u * kq[g][u];
    v = load(addr);
    if (u == 1 && i + 3 < steps(DM)) group(i + 3, kq[g ^ 1], wq[g ^ 1]);
  }
  // The share of the hand-over's steps that goes with evaluation slot e of
  // `total` (the axes of the points under evaluation, in order).
  __device__ __forceinline__ void advance(int e, int total) {
    if constexpr (EXACT) {
#pragma unroll
      for (int i = e * steps(DM) / total; i < (e + 1) * steps(DM) / total; ++i) step(i);
    }
  }
  // Every step done: nothing is under way.
  __device__ __forceinline__ void end() {
    if constexpr (EXACT) {
      add(addr, v, w);
    } else {
      for (int j = 0; j < S; j += 4) {  // (slots past the last point hold zero weights)
        uint32_t k[4];
        float wt[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          k[u] = get_b[(j + u) * P * BS];
          wt[u] = get_w[(j + u) * P];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const uint32_t at = cells + 256u * k[u];
          add(at, load(at), wt[u]);
        }
      }
    }
  }
  // The whole hand-over at once; its slots are left empty.
  __device__ __forceinline__ void drain() {
    begin();
    if constexpr (EXACT) {
#pragma unroll
      for (int i = 0; i < steps(DM); ++i) step(i);
    }
    end();
    __syncwarp();
#pragma unroll
    for (int q = 0; q < PIF; ++q) *put_w[q] = 0.f;
    __syncwarp();
  }
};

// Sum of cell (axis a, bin k) over the columns of all warps of the CTA, as
// compensated pairs of S1 and S2; the columns are cleared.  Copies of one
// warp are added in FP32, the warps compensated.  `base` is the first warp's
// cells; the copy order rotates with k so that neighbouring threads (a
// fastest) read different banks.
__device__ __forceinline__ void col_sum(unsigned char* base, size_t warp_bytes, int nw, int d, int P, int a, int k,
                                        fpair& s1, fpair& s2) {
  s1 = s2 = fpair{0.f, 0.f};
  const int r = k % P;
  for (int w = 0; w < nw; ++w) {
    float2* row = reinterpret_cast<float2*>(base + w * warp_bytes) + 32 * k + a;
    float2 t = make_float2(0.f, 0.f);
#pragma unroll 4
    for (int c = 0; c < P; ++c) {
      int q = c + r;
      q = q >= P ? q - P : q;
      t = __fadd2_rn(t, row[q * d]);
      row[q * d] = make_float2(0.f, 0.f);
    }
    comp_add(s1, t.x);
    comp_add(s2, t.y);
  }
}

}  // namespace gv
