// common.cuh -- device-side building blocks of the sm_103a VEGAS / BASES path:
// Philox4x32-10 in registers, compensated FP32 sums, precision-generic math,
// and the argument blocks of the kernels.
#pragma once

#ifdef __CUDACC_RTC__
// Run-time compilation (user integrands, see rtc.cu): no host headers, so
// the fixed-width types are spelled out (LP64, as on the host side).
typedef signed char int8_t;
typedef unsigned char uint8_t;
typedef int int32_t;
typedef unsigned int uint32_t;
typedef long int64_t;
typedef unsigned long uint64_t;
#else
#include <cuda_runtime.h>
#include <stdint.h>
#endif

#include "../../include/gvegas.h"

namespace gv {

constexpr int kMaxDim = GVEGAS_MAXDIM;
constexpr int kMaxBins = GVEGAS_MAXBINS;
constexpr int kMaxHist = GVEGAS_MAXHIST;
constexpr int kNumDerived = 3 * kMaxDim + 24;  // derived integrand constants
constexpr int kTotCols = 8;                     // per-CTA totals columns

// Columns of the per-CTA totals block.
enum { TOT_SW = 0, TOT_SW2 = 1, TOT_SI = 2, TOT_SV = 3, TOT_NONFINITE = 4 };

// ---------------------------------------------------------------------------
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): the counter-based
// generator that replaces the per-thread xorshift state of Appendix A.
// Stateless: any thread can produce the words of any sample.
// ---------------------------------------------------------------------------
// The 64-bit product a b as (lo, hi) through one widening multiply (the
// batched kernels' bin and fraction).  The Philox rounds keep a low and a
// high multiply, which measured faster there (dgauss8 passes 2-3 %).
__device__ __forceinline__ void mul_wide(uint32_t a, uint32_t b, uint32_t& lo, uint32_t& hi) {
  const uint64_t p = (uint64_t)a * (uint64_t)b;
  lo = (uint32_t)p;
  hi = (uint32_t)(p >> 32);
}

__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r > 0) {
      k0 += 0x9E3779B9u;
      k1 += 0xBB67AE85u;
    }
    const uint32_t lo0 = 0xD2511F53u * c.x, hi0 = __umulhi(0xD2511F53u, c.x);
    const uint32_t lo1 = 0xCD9E8D57u * c.z, hi1 = __umulhi(0xCD9E8D57u, c.z);
    c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
  }
  return c;
}

// Round keys of Philox4x32-10 for key (k0, k1): ks[2 r], ks[2 r + 1] are
// the two key words of round r (Weyl increments 0x9E3779B9, 0xBB67AE85).
// Kernels receive them precomputed in their arguments, so every round reads
// its key from the constant bank instead of adding it on the fly.
constexpr int kPhiloxKeyWords = 20;
__host__ __device__ inline void philox_key_schedule(uint32_t k0, uint32_t k1, uint32_t* ks) {
  for (int r = 0; r < 10; ++r) {
    ks[2 * r] = k0;
    ks[2 * r + 1] = k1;
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
}

__device__ __forceinline__ uint4 philox4x32_10(uint4 c, const uint32_t (&ks)[kPhiloxKeyWords]) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint32_t lo0 = 0xD2511F53u * c.x, hi0 = __umulhi(0xD2511F53u, c.x);
    const uint32_t lo1 = 0xCD9E8D57u * c.z, hi1 = __umulhi(0xCD9E8D57u, c.z);
    c = make_uint4(hi1 ^ c.y ^ ks[2 * r], lo1, hi0 ^ c.w ^ ks[2 * r + 1], lo0);
  }
  return c;
}

__device__ __forceinline__ uint32_t pick(const uint4& v, int i) {
  return i == 0 ? v.x : (i == 1 ? v.y : (i == 2 ? v.z : v.w));
}

// ---------------------------------------------------------------------------
// Error-free transformation (Knuth TwoSum) and compensated pairs.
// ---------------------------------------------------------------------------
struct fpair {
  float hi, lo;
};

__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

__device__ __forceinline__ void comp_add(fpair& p, float v) {
  float s, e;
  two_sum(p.hi, v, s, e);
  p.hi = s;
  p.lo = __fadd_rn(p.lo, e);
}

__device__ __forceinline__ void comp_merge(fpair& p, const fpair& q) {
  float s, e;
  two_sum(p.hi, q.hi, s, e);
  p.hi = s;
  p.lo = __fadd_rn(__fadd_rn(p.lo, q.lo), e);
}

__device__ __forceinline__ double comp_value(const fpair& p) {
  return (double)p.hi + (double)p.lo;
}

// ---------------------------------------------------------------------------
// Precision-generic math.
// ---------------------------------------------------------------------------
__device__ __forceinline__ double vexp(double x) { return exp(x); }
__device__ __forceinline__ float vexp(float x) { return expf(x); }
__device__ __forceinline__ double vlog(double x) { return log(x); }
__device__ __forceinline__ float vlog(float x) { return logf(x); }
__device__ __forceinline__ double vsqrt(double x) { return sqrt(x); }
__device__ __forceinline__ float vsqrt(float x) { return sqrtf(x); }
__device__ __forceinline__ double vatan2(double y, double x) { return atan2(y, x); }
__device__ __forceinline__ float vatan2(float y, float x) { return atan2f(y, x); }
__device__ __forceinline__ double vcos(double x) { return cos(x); }
__device__ __forceinline__ float vcos(float x) { return cosf(x); }
__device__ __forceinline__ double vsin(double x) { return sin(x); }
__device__ __forceinline__ float vsin(float x) { return sinf(x); }
__device__ __forceinline__ void vsincospi(double x, double* s, double* c) { sincospi(x, s, c); }
__device__ __forceinline__ void vsincospi(float x, float* s, float* c) { sincospif(x, s, c); }
__device__ __forceinline__ double vpow(double x, double y) { return pow(x, y); }
__device__ __forceinline__ float vpow(float x, float y) { return powf(x, y); }
__device__ __forceinline__ double vcopysign(double x, double y) { return copysign(x, y); }
__device__ __forceinline__ float vcopysign(float x, float y) { return copysignf(x, y); }
__device__ __forceinline__ double vfma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float vfma(float a, float b, float c) { return fmaf(a, b, c); }
// (FP64 by the exponent's bits: an FP64 comparison costs the slow FP64 pipe)
__device__ __forceinline__ bool vfinite(double x) { return (__double2hiint(x) & 0x7FF00000) != 0x7FF00000; }
__device__ __forceinline__ bool vfinite(float x) { return isfinite(x); }

// r 2^-bits rounded to nearest (exact below 2^53, as a conversion and a power
// of two would give it), without the FP64 pipe (1.65 operations per SM-clock
// on this GPU, against 128 integer ones): the leading bit moved to bit 52 and
// the exponent put above it.
__device__ __forceinline__ double scaled_u64(uint64_t r, int bits) {
  const int lz = __clzll((long long)r);  // 0..64
  uint64_t m;
  if (lz >= 11) {
    m = r << (lz - 11);
  } else {  // 54 to 64 bits: round to nearest, ties to even
    const int s = 11 - lz;
    const uint64_t rem = r & ((1ull << s) - 1ull), half = 1ull << (s - 1);
    m = r >> s;
    m += rem > half || (rem == half && (m & 1ull)) ? 1ull : 0ull;  // (a carry moves into the exponent)
  }
  return r == 0 ? 0.0 : __longlong_as_double((long long)(((uint64_t)(1023 + 62 - lz - bits) << 52) + m));
}

// exp in FP64 for the integrands: Tang's table method (Tang, ACM TOMS 15,
// 1989): x = (64 m + j) ln2 / 64 + r, |r| <= ln2 / 128, exp x = 2^m 2^(j/64)
// (1 + p(r)) with a degree-5 polynomial and the table 2^(j/64) in two
// doubles.  The error stays below 0.84 ulp: half from the last rounding, up to
// 0.31 from the polynomial's end (r^6 / 720 <= 3.5e-17 of a value below 2), the
// rest from the roundings of p (largest measured 0.80, mean 0.254; CUDA's exp
// 0.85 and 0.258).  11 FP64 operations instead of the library's 16 or so:
// the FP64 kernels are bound by that pipe.  Arguments whose result is not a
// normal number go to the library.
static __device__ const double2 kExpTable[64] = {
    {0x1.0000000000000p+0, 0x0.0p+0}, {0x1.02c9a3e778061p+0, -0x1.19083535b085dp-56},
    {0x1.059b0d3158574p+0, 0x1.d73e2a475b465p-55}, {0x1.0874518759bc8p+0, 0x1.186be4bb284ffp-57},
    {0x1.0b5586cf9890fp+0, 0x1.8a62e4adc610bp-54}, {0x1.0e3ec32d3d1a2p+0, 0x1.03a1727c57b53p-59},
    {0x1.11301d0125b51p+0, -0x1.6c51039449b3ap-54}, {0x1.1429aaea92de0p+0, -0x1.32fbf9af1369ep-54},
    {0x1.172b83c7d517bp+0, -0x1.19041b9d78a76p-55}, {0x1.1a35beb6fcb75p+0, 0x1.e5b4c7b4968e4p-55},
    {0x1.1d4873168b9aap+0, 0x1.e016e00a2643cp-54}, {0x1.2063b88628cd6p+0, 0x1.dc775814a8495p-55},
    {0x1.2387a6e756238p+0, 0x1.9b07eb6c70573p-54}, {0x1.26b4565e27cddp+0, 0x1.2bd339940e9d9p-55},
    {0x1.29e9df51fdee1p+0, 0x1.612e8afad1255p-55}, {0x1.2d285a6e4030bp+0, 0x1.0024754db41d5p-54},
    {0x1.306fe0a31b715p+0, 0x1.6f46ad23182e4p-55}, {0x1.33c08b26416ffp+0, 0x1.32721843659a6p-54},
    {0x1.371a7373aa9cbp+0, -0x1.63aeabf42eae2p-54}, {0x1.3a7db34e59ff7p+0, -0x1.5e436d661f5e3p-56},
    {0x1.3dea64c123422p+0, 0x1.ada0911f09ebcp-55}, {0x1.4160a21f72e2ap+0, -0x1.ef3691c309278p-58},
    {0x1.44e086061892dp+0, 0x1.89b7a04ef80d0p-59}, {0x1.486a2b5c13cd0p+0, 0x1.3c1a3b69062f0p-56},
    {0x1.4bfdad5362a27p+0, 0x1.d4397afec42e2p-56}, {0x1.4f9b2769d2ca7p+0, -0x1.4b309d25957e3p-54},
    {0x1.5342b569d4f82p+0, -0x1.07abe1db13cadp-55}, {0x1.56f4736b527dap+0, 0x1.9bb2c011d93adp-54},
    {0x1.5ab07dd485429p+0, 0x1.6324c054647adp-54}, {0x1.5e76f15ad2148p+0, 0x1.ba6f93080e65ep-54},
    {0x1.6247eb03a5585p+0, -0x1.383c17e40b497p-54}, {0x1.6623882552225p+0, -0x1.bb60987591c34p-54},
    {0x1.6a09e667f3bcdp+0, -0x1.bdd3413b26456p-54}, {0x1.6dfb23c651a2fp+0, -0x1.bbe3a683c88abp-57},
    {0x1.71f75e8ec5f74p+0, -0x1.16e4786887a99p-55}, {0x1.75feb564267c9p+0, -0x1.0245957316dd3p-54},
    {0x1.7a11473eb0187p+0, -0x1.41577ee04992fp-55}, {0x1.7e2f336cf4e62p+0, 0x1.05d02ba15797ep-56},
    {0x1.82589994cce13p+0, -0x1.d4c1dd41532d8p-54}, {0x1.868d99b4492edp+0, -0x1.fc6f89bd4f6bap-54},
    {0x1.8ace5422aa0dbp+0, 0x1.6e9f156864b27p-54}, {0x1.8f1ae99157736p+0, 0x1.5cc13a2e3976cp-55},
    {0x1.93737b0cdc5e5p+0, -0x1.75fc781b57ebcp-57}, {0x1.97d829fde4e50p+0, -0x1.d185b7c1b85d1p-54},
    {0x1.9c49182a3f090p+0, 0x1.c7c46b071f2bep-56}, {0x1.a0c667b5de565p+0, -0x1.359495d1cd533p-54},
    {0x1.a5503b23e255dp+0, -0x1.d2f6edb8d41e1p-54}, {0x1.a9e6b5579fdbfp+0, 0x1.0fac90ef7fd31p-54},
    {0x1.ae89f995ad3adp+0, 0x1.7a1cd345dcc81p-54}, {0x1.b33a2b84f15fbp+0, -0x1.2805e3084d708p-57},
    {0x1.b7f76f2fb5e47p+0, -0x1.5584f7e54ac3bp-56}, {0x1.bcc1e904bc1d2p+0, 0x1.23dd07a2d9e84p-55},
    {0x1.c199bdd85529cp+0, 0x1.11065895048ddp-55}, {0x1.c67f12e57d14bp+0, 0x1.2884dff483cadp-54},
    {0x1.cb720dcef9069p+0, 0x1.503cbd1e949dbp-56}, {0x1.d072d4a07897cp+0, -0x1.cbc3743797a9cp-54},
    {0x1.d5818dcfba487p+0, 0x1.2ed02d75b3707p-55}, {0x1.da9e603db3285p+0, 0x1.c2300696db532p-54},
    {0x1.dfc97337b9b5fp+0, -0x1.1a5cd4f184b5cp-54}, {0x1.e502ee78b3ff6p+0, 0x1.39e8980a9cc8fp-55},
    {0x1.ea4afa2a490dap+0, -0x1.e9c23179c2893p-54}, {0x1.efa1bee615a27p+0, 0x1.dc7f486a4b6b0p-54},
    {0x1.f50765b6e4540p+0, 0x1.9d3e12dd8a18bp-54}, {0x1.fa7c1819e90d8p+0, 0x1.74853f3a5931ep-55},
};
__device__ __forceinline__ double exp64(double x) {
  // |x| < 708: by the high word (NaN and infinity fail too)
  if ((__double2hiint(x) & 0x7FFFFFFF) >= 0x40862000) return exp(x);
  const double t = fma(x, 64.0 * 1.4426950408889634074, 6755399441055744.0);  // 1.5 2^52: n in the low bits
  const int n = __double2loint(t);
  const double nd = t - 6755399441055744.0;
  // ln2 / 64 in two parts, the first with 20 trailing zero bits (n nd exact)
  double r = fma(nd, -0x1.62e42fee00000p-7, x);
  r = fma(nd, -0x1.a39ef35793c76p-39, r);
  const double2 T = __ldg(&kExpTable[n & 63]);
  double q = fma(r, 1.0 / 120.0, 1.0 / 24.0);
  q = fma(r, q, 1.0 / 6.0);
  q = fma(r, q, 0.5);
  const double p = fma(r * r, q, r);
  const double y = T.x + fma(T.x, p, T.y);
  return __hiloint2double(__double2hiint(y) + ((n >> 6) << 20), __double2loint(y));
}

// Quick FP32 forms for the FP32 integrands: the special-function unit's
// approximations (__logf, __expf, __sincosf, __fdividef, sqrt.approx),
// a few parts in 2^22 on the ranges used; arguments of the trigonometric
// forms are kept in [-pi, pi] by their callers.  The FP64 overloads are CUDA's
// library functions, except for exp, which is exp64.
__device__ __forceinline__ float qlog(float x) { return __logf(x); }
__device__ __forceinline__ double qlog(double x) { return log(x); }
// ln x with a small relative error also near x = 1, where __logf's
// absolute error would dominate a small result: 2 atanh(s),
// s = (x - 1)/(x + 1), by its odd series through s^9 on [0.75, 1.25]
// (|s| <= 1/7, truncation below 1e-8 relative), __logf elsewhere.
__device__ __forceinline__ float qlog_rel(float x) {
  const float s = __fdividef(x - 1.0f, x + 1.0f), s2 = s * s;
  const float series =
      2.0f * s * fmaf(s2, fmaf(s2, fmaf(s2, fmaf(s2, 1.0f / 9.0f, 1.0f / 7.0f), 1.0f / 5.0f), 1.0f / 3.0f), 1.0f);
  return (x > 0.75f && x < 1.25f) ? series : __logf(x);
}
__device__ __forceinline__ double qlog_rel(double x) { return log(x); }
__device__ __forceinline__ float qexp(float x) { return __expf(x); }
__device__ __forceinline__ double qexp(double x) { return exp64(x); }
__device__ __forceinline__ float qdiv(float a, float b) { return __fdividef(a, b); }
__device__ __forceinline__ double qdiv(double a, double b) { return a / b; }
__device__ __forceinline__ float qsqrt(float x) {
  float r;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ double qsqrt(double x) { return sqrt(x); }
__device__ __forceinline__ float qsin(float x) { return __sinf(x); }
__device__ __forceinline__ double qsin(double x) { return sin(x); }
__device__ __forceinline__ float qcos(float x) { return __cosf(x); }
__device__ __forceinline__ double qcos(double x) { return cos(x); }
// sin and cos of 2 pi u for u in [0, 1): evaluated at 2 pi (u - 1/2) in
// [-pi, pi) and negated
__device__ __forceinline__ void qsincos2pi(float u, float* s, float* c) {
  float sn, cs;
  __sincosf(6.28318530717958648f * (u - 0.5f), &sn, &cs);
  *s = -sn;
  *c = -cs;
}
__device__ __forceinline__ void qsincos2pi(double u, double* s, double* c) { sincospi(2.0 * u, s, c); }

// A compile-time flag as a type (selects a code path of a generic lambda).
template <bool V> struct BoolTag {
  static constexpr bool value = V;
};

template <typename T> struct Vec2;
template <> struct Vec2<double> { using type = double2; };
template <> struct Vec2<float> { using type = float2; };

// ---------------------------------------------------------------------------
// Device-resident iteration state (one per context).
// ---------------------------------------------------------------------------
struct GState {
  uint32_t it;          // Philox iteration counter: iterations run so far
  int done;             // set when the ACC test stops the current call
  int live;             // latched per pass by the sampling kernel: 1 if it ran
  int nhist;            // iterations in the combination window
  int stopped;
  long long nonfinite;  // non-finite weights in the window
  long long samples;    // points in the window
  double acc;           // relative accuracy target of the current call
  double I, sigma, chi2;
  double last_I, last_var, last_sw, last_sw2;
  long long last_nonfinite;
  // snapshot of the first BASES phase
  double ph1_I, ph1_sigma, ph1_chi2;
  int ph1_iters, ph1_stopped;
  long long ph1_nonfinite, ph1_samples;
  double hist[kMaxHist][2];
};

// The state's fields up to the history into its host-visible copy, by one
// warp (after its writes): the host reads them once the stream has got here,
// without a copy of its own.
__device__ __forceinline__ void mirror_state(GState* mirror, const GState* st) {
  __syncwarp();
  const int n = (int)((sizeof(GState) - sizeof(st->hist)) / sizeof(int));
  const int* src = reinterpret_cast<const int*>(st);
  int* dst = reinterpret_cast<int*>(mirror);
  for (int i = threadIdx.x & 31; i < n; i += 32) dst[i] = src[i];
}

// Threads per block of k_finish: up to 64 bins (and in passes without bins), and beyond.
constexpr int kFinishThreads = 256, kMaxFinishThreads = 512;

// Device-side control operations captured into the iteration graphs.
enum { CTL_RESET_WINDOW = 1, CTL_SET_ACC = 2, CTL_SNAPSHOT = 4, CTL_SET_ITER = 8 };

// Iterations on a frozen grid one sampling launch can run (their points need
// nothing from one another unless an ACC test may stop between them).
constexpr int kMergeIters = 8;

// The hypercube in place `slot` of the processing order: an odd or coprime
// multiplier permutes the n cubes, so that the groups of a CTA sit in
// unrelated cubes and spread over the bins.
__host__ __device__ __forceinline__ uint32_t cube_of(uint32_t n, uint32_t mul, uint32_t slot) {
  return (n & (n - 1u)) == 0u ? (slot * mul) & (n - 1u) : (uint32_t)(((uint64_t)slot * mul) % n);
}

// Step 4 of one hypercube from its sums (n_c points): the cube mean m = C1 /
// n_c and variance (C2 / n_c - m^2) / (n_c - 1) into the totals t = (sum w,
// sum w^2, sum of means, sum of variances).
// Compensated form: FP32 with the square formed exactly (FMA), pairs kept.
__device__ __forceinline__ void cube_totals(double inv_nc, double inv_nc1, const fpair& c1, const fpair& c2,
                                            fpair (&t)[4]) {
  const float inv = (float)inv_nc, inv1 = (float)inv_nc1;
  const float mh = c1.hi * inv, ml = c1.lo * inv;
  const float sq = mh * mh;
  const float sqe = fmaf(mh, mh, -sq) + 2.0f * mh * ml;
  const float e2h = c2.hi * inv, e2l = c2.lo * inv;
  float v = ((e2h - sq) + (e2l - sqe)) * inv1;
  if (!(v > 0.f)) v = 0.f;
  comp_merge(t[0], c1);
  comp_merge(t[1], c2);
  comp_add(t[2], mh);
  comp_add(t[2], ml);
  comp_add(t[3], v);
}
__device__ __forceinline__ void cube_totals(double inv_nc, double inv_nc1, double c1, double c2, double (&t)[4]) {
  const double m = c1 * inv_nc;
  double v = (c2 * inv_nc - m * m) * inv_nc1;
  if (v < 0.0) v = 0.0;
  t[0] += c1;
  t[1] += c2;
  t[2] += m;
  t[3] += v;
}
// A hypercube's sums (or a part of them) in memory: (hi, lo, hi, lo) floats
// or two doubles, 16 bytes.
__device__ __forceinline__ void cube_store(void* p, size_t i, const fpair& c1, const fpair& c2) {
  reinterpret_cast<float4*>(p)[i] = make_float4(c1.hi, c1.lo, c2.hi, c2.lo);
}
__device__ __forceinline__ void cube_store(void* p, size_t i, double c1, double c2) {
  reinterpret_cast<double2*>(p)[i] = make_double2(c1, c2);
}

// Arguments of the sampling kernel (steps 2-4).
struct SampleArgs {
  int d, N, g, ybits;
  int lanes;               // lanes per group (stratified mode), power of two <= 32
  int cap;                 // bucket capacity per (axis, bin) and tile
  int ppt;                 // points per thread per tile (>= 1)
  int strat;
  uint32_t key0, key1, instance;
  // Philox round keys of (key0, key1).  On a 16-byte boundary: off it the
  // compiler reads them word by word (k_spring, d = 8: 52 registers, not 48)
  alignas(16) uint32_t ks[kPhiloxKeyWords];
  int it_override;         // >= 0: use this iteration index
  uint64_t ncall;
  uint32_t nc;             // points per hypercube
  uint32_t ncubes;         // number of hypercubes
  uint32_t cube_mul;       // multiplier permuting the cube order (cube_of)
  int g_pow2, g_log2;
  int t32;                 // 24-bit bins fit 32-bit integers (g N <= 256)
  float inv_gb_f;          // 1 / (g 2^ybits)
  double inv_gb_d;
  double inv_nc, inv_nc1;  // 1 / nc, 1 / (nc - 1)
  int nparts;              // number of CTAs == partial rows
  const void* tab;         // [d][N] (e_k, Delta_k) in the kernel precision
  const double* dparams;   // derived integrand constants
  GState* st;              // the sampling kernel latches st->live
  void* part_bins;         // [nparts][2 d N]: double, or float (hi, lo) pairs (FP32 forms)
  double* part_tot;        // [niter][kTotCols][nparts]
  void* cubes;             // [ncubes]: double (sum w, sum w^2), or float (hi, lo, hi, lo)
  double* cube_max;        // [ncubes] running max(0, largest w) (integration phase), or null
  void* cube_part;         // [niter][parts][ncubes] sums of the parts (parts > 1), as `cubes`
  uint32_t parts;          // groups per hypercube, each with its share of the cube's points
  uint32_t units, vl, per_lane;  // groups of a pass (hypercubes x parts), lanes of a cube, points per lane
  int niter;               // iterations this launch runs, one per blockIdx.y (frozen grid; 1 with the histogram)
  int force;               // 1: run even if the ACC test has stopped the last call (evaluation passes)
};

// Arguments of the reduction and finalisation kernels (steps 4-6).
struct FinArgs {
  int d, N, nparts, strat, refine, record;
  int combine;             // 1: form the combined result (and the ACC test)
  int nobins;              // the pass kept no per-bin histogram: totals only, no refinement
  int pair32;              // part_bins hold float (hi, lo) pairs
  uint64_t ncall;
  uint64_t ncubes;
  const double* scale;     // integrand output scale (RAMBO units), in device memory so
                           // that captured graphs follow vegas_set_params
  double alpha;
  const void* part_bins;
  const double* part_tot;
  uint32_t units, vl, per_lane;  // groups of a pass (hypercubes x parts), lanes of a cube, points per lane
  int niter;               // iterations of the pass (frozen grid)
  uint32_t parts;          // groups per hypercube; > 1: the totals come from cube_part
  uint32_t cube_mul;
  double inv_nc, inv_nc1;  // 1 / nc, 1 / (nc - 1)
  const void* cube_part;
  void* cubes;             // per-cube sums of the last iteration (parts > 1), or null
  double* bins;            // [2][d][N] reduced, scaled
  double* edges;           // [d][N+1]
  double2* tab64;          // [d][N]
  float2* tab32;           // [d][N]
  GState* st;
  GState* mirror;          // host-visible copy of the state up to `hist`, or null
  double* result;          // (I, variance, sum w, sum w^2, non-finite count), or null
};

}  // namespace gv
