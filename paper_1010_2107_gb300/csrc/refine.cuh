// refine.cuh -- step 5 (grid optimisation, Lepage 1978) and the step-6
// combination of iterations as device functions shared by the single-context
// and the batched finalisation kernels.  All FP64.
#pragma once

#include "common.cuh"

namespace gv {

// Error-free sum of two doubles (Knuth TwoSum): s + e == a + b exactly.
__device__ __forceinline__ void two_sum_d(double a, double b, double& s, double& e) {
  s = a + b;
  const double bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}

// The first n threads of a block (n a multiple of 32) working as one team
// with a barrier of its own (named barrier 1), so that a step needing few
// threads leaves the other warps idle: scalar FP64 is slow on this GPU and
// even idle lanes of a warp that issues an FP64 instruction cost its pipe.
struct Team {
  int n;
  __device__ __forceinline__ void sync() const { asm volatile("bar.sync 1, %0;" ::"r"(n) : "memory"); }
};

// Exact sum over the team of 64-bit integers below 2^62 in total: three
// 22-bit digits per value through the warp's integer reduction, then the
// warps in order.  `buf`: one entry per warp; all team threads must call.
__device__ __forceinline__ unsigned long long team_sum(unsigned long long v, unsigned long long* buf, Team t) {
  constexpr unsigned M = (1u << 22) - 1u;
  const unsigned d0 = __reduce_add_sync(0xffffffffu, (unsigned)v & M);
  const unsigned d1 = __reduce_add_sync(0xffffffffu, (unsigned)(v >> 22) & M);
  const unsigned d2 = __reduce_add_sync(0xffffffffu, (unsigned)(v >> 44));
  const unsigned long long w = (unsigned long long)d0 + ((unsigned long long)d1 << 22) + ((unsigned long long)d2 << 44);
  if (t.n == 32) return w;
  if ((threadIdx.x & 31) == 0) buf[threadIdx.x >> 5] = w;
  t.sync();
  unsigned long long S = buf[0];
  for (int i = 1; i < t.n >> 5; ++i) S += buf[i];
  return S;
}

// One axis, one team of threads (one per bin, N <= t.n): smooth the per-bin
// sums of w^2 over neighbours, compress them with r_k = ((1 - d_k/D) /
// ln(D/d_k))^alpha, and move the edges so that every new bin holds an equal
// share of sum r, with r spread uniformly inside each old bin.  dd: S2 of the
// axis (N values); ea: its N+1 edges (updated in place); t64 / t32: its (e_k,
// Delta_k) cells.  An axis whose smoothed sum is zero or not finite is left
// unchanged.
//
// This runs once per refining pass with nothing beside it, so what counts is
// the length of its dependent chain, and the FP64 pipe (1.65 operations per
// SM-clock: 19 clocks for a warp's instruction) is all of it.  The sums D
// and R and the prefix sums C_k = r_0 + ... + r_{k-1} are therefore 64-bit
// integers: a value enters as a multiple of 2^-58 or less of the largest one
// (of 1 for r), and the integer sums are exact, so they carry less error
// than FP64 sums would and cost no FP64 instruction.  Divisions by a common
// divisor are products with its reciprocal.
//
// New edge j is found by each thread on its own: old bin k_j is the first k
// with C_{k+1} >= tau_j = j R / N (or the last bin), and the new edge sits at
// the fraction (tau_j - C_k) / r_k of it.  This is the sequential rebinning
// walk of Lepage written without its loop-carried dependence.
__device__ inline void refine_axis_core(const double* dd, double* ea, double2* t64, float2* t32, int N,
                                        double alpha, Team t) {
  __shared__ double e[kMaxBins + 1], enew[kMaxBins + 1];
  __shared__ unsigned long long C[kMaxBins + 1], buf[2][8];
  __shared__ int ibuf[16];
  const int k = threadIdx.x, lane = k & 31, warp = k >> 5, nw = t.n >> 5;
  const bool in = k < N;
  // fixed-point position of the largest value: N values below 2^top sum below 2^62
  const int top = 62 - (32 - __clz(N - 1));
  double x = 0.0;
  if (in) {
    e[k] = ea[k];
    if (k == 0) {
      e[N] = ea[N];
      enew[0] = 0.0;
      enew[N] = 1.0;
    }
    if (N == 2 || k == 0)
      x = (dd[0] + dd[1]) * 0.5;
    else if (k == N - 1)
      x = (dd[N - 2] + dd[N - 1]) * 0.5;
    else
      x = (dd[k - 1] + dd[k] + dd[k + 1]) * (1.0 / 3.0);
  }
  // the largest exponent (finite non-negative doubles order as their bits)
  int hi = __reduce_max_sync(0xffffffffu, __double2hiint(x) & 0x7FFFFFFF);
  if (nw > 1) {
    if (lane == 0) ibuf[warp] = hi;
    t.sync();
    hi = ibuf[0];
    for (int i = 1; i < nw; ++i) hi = max(hi, ibuf[i]);
  }
  const int ex = hi >> 20;  // values below 2^(ex - 1022)
  if (ex >= 0x7FF) return;  // not finite (uniform across the team)
  // scale = 2^(top - (ex - 1022)) in two factors, each within range
  const int sh = top + 1022 - max(ex, 1), h1 = sh / 2, h2 = sh - h1;
  const double f1 = __hiloint2double((1023 + h1) << 20, 0), f2 = __hiloint2double((1023 + h2) << 20, 0);
  const unsigned long long Di = team_sum(x > 0.0 ? (unsigned long long)__double2ll_rn(x * f1 * f2) : 0ull, buf[0], t);
  if (Di == 0ull) return;  // every sum zero (uniform across the team)
  if (64 - __clzll((long long)Di) - sh > 1024) return;  // D = Di 2^-sh not finite, though its terms are
  // q = x / D and r = ((1 - q) / -ln q)^alpha
  double rk = 0.0;
  if (x > 0.0) {
    const double q = (x * f1 * f2) * (1.0 / (double)Di);
    rk = 1.0;
    if (q < 1.0) {
      // (D / x overflows, and ln with it, for q up to 2^-1024: then y = 0)
      const double y = q > 0x1p-1024 ? (1.0 - q) / -log(q) : 0.0;
      // the default alpha = 3/2 as y sqrt(y) (a few FP64 instructions
      // instead of a general power)
      rk = alpha == 1.5 ? y * sqrt(y) : pow(y, alpha);
    }
  }
  // inclusive prefix sums of r 2^top.  With alpha = 3/2 the largest r lies in
  // [0.06, 1] (q >= 1/N there, N <= 256); for another alpha the values are
  // scaled by the largest one's exponent first.
  int re = 0;
  if (alpha != 1.5) {
    re = __reduce_max_sync(0xffffffffu, __double2hiint(rk));
    if (nw > 1) {
      if (lane == 0) ibuf[8 + warp] = re;
      t.sync();
      re = ibuf[8];
      for (int i = 1; i < nw; ++i) re = max(re, ibuf[8 + i]);
    }
    re = max(re >> 20, 64) - 1022;  // r below 2^re
    if (re < 0) rk *= __hiloint2double((1023 - re) << 20, 0);
  }
  const double f = __hiloint2double((1023 + top) << 20, 0);
  const unsigned long long ri = (unsigned long long)__double2ll_rn(rk * f);
  unsigned long long run = ri;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const unsigned long long o = __shfl_up_sync(0xffffffffu, run, off);
    if (lane >= off) run += o;
  }
  if (nw > 1) {
    if (lane == 31) buf[1][warp] = run;
    t.sync();
    for (int i = 0; i < warp; ++i) run += buf[1][i];
  }
  if (in) C[k + 1] = run;
  if (k == 0) C[0] = 0ull;
  t.sync();
  const double share = (double)C[N] * (1.0 / (double)N);
  const int j = k;
  if (j > 0 && in) {
    const unsigned long long tau = (unsigned long long)__double2ll_rn((double)j * share);
    // first b in [0, N-1) with C[b + 1] >= tau, else N - 1 (C is nondecreasing)
    int lo = 0, up = N - 1;
    while (lo < up) {
      const int mid = (lo + up) >> 1;
      if (C[mid + 1] >= tau)
        up = mid;
      else
        lo = mid + 1;
    }
    const unsigned long long c0 = C[lo], w = C[lo + 1] - c0;
    enew[j] = e[lo] + (double)(long long)(tau - c0) / (double)w * (e[lo + 1] - e[lo]);
  }
  t.sync();
  if (in) {
    const double lo = enew[k], w = enew[k + 1] - enew[k];
    if (k > 0) ea[k] = lo;
    t64[k] = make_double2(lo, w);
    t32[k] = make_float2((float)lo, (float)w);
  }
}

// Inverse-variance combination of h iteration estimates (Lepage):
// weighted mean, its standard error and chi^2 per degree of freedom; any
// zero-variance estimate makes the result the mean of those, with sigma 0.
// Compensated xor-butterfly sum of the lanes' (s, c) pairs.
__device__ inline double warp_sum_comp(double s, double c) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const double os = __shfl_xor_sync(0xffffffffu, s, off), oc = __shfl_xor_sync(0xffffffffu, c, off);
    double t, e;
    two_sum_d(s, os, t, e);
    s = t;
    c = c + oc + e;
  }
  return s + c;
}

// Called by a full warp: lane j takes estimates j, j + 32, ... (divisions in
// parallel, a compensated running sum per lane), then a compensated xor
// butterfly merges the lanes; every lane returns the same result.
__device__ inline void combine_history(const double (*hist)[2], int h, double* Ib, double* sg, double* chi) {
  const int lane = threadIdx.x & 31;
  double zs = 0.0, zc = 0.0, ws = 0.0, wc = 0.0, qs = 0.0, qc = 0.0;
  int nz = 0;
  for (int j = lane; j < h; j += 32) {
    const double I = hist[j][0], v = hist[j][1];
    double t, e;
    if (!(v > 0.0)) {
      two_sum_d(zs, I, t, e);
      zs = t;
      zc += e;
      ++nz;
    } else {
      const double iv = 1.0 / v;
      two_sum_d(ws, iv, t, e);
      ws = t;
      wc += e;
      two_sum_d(qs, I * iv, t, e);
      qs = t;
      qc += e;
    }
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) nz += __shfl_xor_sync(0xffffffffu, nz, off);
  const double Z = warp_sum_comp(zs, zc);
  const double W = warp_sum_comp(ws, wc);
  const double Q = warp_sum_comp(qs, qc);
  double I = 0.0, s = 0.0, x2 = 0.0;
  if (nz > 0) {
    I = Z / (double)nz;
  } else if (h > 0) {
    I = Q / W;
    s = 1.0 / sqrt(W);
    if (h > 1) {
      double cs = 0.0, cc = 0.0;
      for (int j = lane; j < h; j += 32) {
        const double dv = hist[j][0] - I;
        double t, e;
        two_sum_d(cs, dv * dv / hist[j][1], t, e);
        cs = t;
        cc += e;
      }
      x2 = warp_sum_comp(cs, cc) / (double)(h - 1);
    }
  }
  *Ib = I;
  *sg = s;
  *chi = x2;
}

}  // namespace gv
