// Toy datasets on the device (Sec. 1: RooStats toy Monte Carlo) and their
// 64-bin histograms.
//
// Random numbers: Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11), a
// counter-based generator, so every event of every set is addressable on its
// own: key = (seed, seed >> 32), counter = (event, attempt, set, factor); the
// size draw uses counter (iteration, 0, set, 0xFFFFFFFF).  Uniforms take the
// top 53 bits of two words.  Set sizes: Poisson by inversion below mean 10,
// else by PTRS (W. Hoermann, "The transformed rejection method for generating
// Poisson random variables", 1993).  Events: accept-reject, independently for
// each factor of a product at the root, against 1.2 x the largest density on
// 4096 midpoints of the factor's range.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "api_internal.h"
#include "expr.cuh"
#include "nll_kernels.cuh"

namespace rf {

namespace {

constexpr int kMaxFactors = 8;
constexpr uint32_t kMaxAttempts = 100000u;
constexpr int kMaxTerms = 24, kMaxFactorTerms = 16, kMaxPath = 6;  // float filter: terms in all, of a factor, SUM depth

__device__ __forceinline__ void philox4x32_10(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, uint32_t k0,
                                              uint32_t k1, uint32_t out[4]) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r > 0) {
      k0 += 0x9E3779B9u;
      k1 += 0xBB67AE85u;
    }
    const uint32_t lo0 = 0xD2511F53u * c0, hi0 = __umulhi(0xD2511F53u, c0);
    const uint32_t lo1 = 0xCD9E8D57u * c2, hi1 = __umulhi(0xCD9E8D57u, c2);
    const uint32_t n0 = hi1 ^ c1 ^ k0, n2 = hi0 ^ c3 ^ k1;
    c0 = n0;
    c1 = lo1;
    c2 = n2;
    c3 = lo0;
  }
  out[0] = c0; out[1] = c1; out[2] = c2; out[3] = c3;
}

__device__ __forceinline__ double u53(uint32_t hi, uint32_t lo) {
  return (double)(((uint64_t)hi << 21) | (lo >> 11)) * 0x1.0p-53;
}
__device__ __forceinline__ double u53_open(uint32_t hi, uint32_t lo) {
  return __dmul_rn(__dadd_rn((double)(((uint64_t)hi << 21) | (lo >> 11)), 0.5), 0x1.0p-53);
}

// Density of one generation factor at x in FP64 (the full-precision formulas
// of the event kernel, without the adjoint): the nodes of `mask`, the
// factor's own node `root` last.  Out of line: the filter below decides
// almost every point, so the FP64 code stays out of the hot loop.
__device__ __noinline__ double factor_value(const Program& P, const double* __restrict__ C, uint32_t mask, int root,
                                            double xc) {
  double v[kMaxPdf];
  for (int n = 0; n <= root; ++n) {
    if (!(mask >> n & 1u)) continue;
    const PNode& q = P.node[n];
    const double* c = C + q.cofs;
    switch (q.kind) {
      case GAUSS: {
        const double u = (xc - c[0]) * c[1];
        v[n] = exp(-0.5 * u * u) * c[2];
        break;
      }
      case EXPO: v[n] = exp(c[0] * (xc - c[1])) * c[2]; break;
      case GAUSSEXP: {
        const double u = (xc - c[0]) * c[1], s = c[2];
        const double z = (s - u) * 0.70710678118654752440;
        const double f = z > 0.0 ? 0.5 * exp(-0.5 * u * u) * erfcx(z) : 0.5 * exp(s * (0.5 * s - u)) * erfc(z);
        v[n] = f * c[4];
        break;
      }
      case CHEB: {
        const int np = q.n_par;
        const double xp = xc * c[0] - c[1];
        double t0 = 1.0, t1 = xp, sh = 1.0;
        for (int k = 1; k <= np; ++k) {
          sh += c[3 + np + k - 1] * t1;
          const double t2 = 2.0 * xp * t1 - t0;
          t0 = t1;
          t1 = t2;
        }
        v[n] = sh * c[2];
        break;
      }
      case POLY: {
        const int np = q.n_par;
        const double xv = xc;
        double sh = 0.0;
        for (int k = np; k >= 1; --k) sh = (sh + c[1 + np + k - 1]) * xv;
        v[n] = (1.0 + sh) * c[0];
        break;
      }
      case POISSON: {
        const double k = fmin(floor(xc), q.hi - 1.0);
        v[n] = exp(k * c[1] - c[0] - lgamma(k + 1.0)) * c[3];
        break;
      }
      case EXPR: {
        double f;
        v[n] = expr_eval<false>(P, q, c + 1 + q.n_par, xc, &f, nullptr) == 0 ? f * c[0] : NAN;
        break;
      }
      case SUM: {
        double r = 0.0;
        for (int j = 0; j < q.n_child; ++j) r += c[j] * v[q.child[j]];
        v[n] = r;
        break;
      }
      case PROD: {
        double r = 1.0;
        for (int j = 0; j < q.n_child; ++j) r *= v[q.child[j]];
        v[n] = r;
        break;
      }
      default: v[n] = 0.0;
    }
  }
  return v[root];
}

struct GenArgs {
  int32_t n_factors;
  int32_t factor[kMaxFactors];  // program index of each factor
  int32_t fcol[kMaxFactors];    // its observable column
  uint32_t mask[kMaxFactors];   // the nodes it is computed from (itself included)
  double lo[kMaxFactors], hi[kMaxFactors];
  // The float filter's terms: factor j is the sum over terms t in [term0[j],
  // term0[j + 1]) of weight times leaf, the weight being the product of the
  // SUM fractions on the way down (path: SUM nodes and child numbers).  No
  // term: the factor has no float form and is always compared in FP64.
  int32_t term0[kMaxFactors + 1];
  int8_t leaf[kMaxTerms], kind[kMaxTerms], n_par[kMaxTerms], n_path[kMaxTerms];
  int8_t path[kMaxTerms][2 * kMaxPath];
};

// ------------------------------------------------------------- float filter
//
// Accept-reject compares y = M u' with the density v in FP64, and on this GPU
// an FP64 warp instruction occupies a sub-partition for 64 cycles: a decay
// density costs about 150 of them, three tries an event, and taken literally
// the generation of 2.4e7 decay events (1024 sets) is FP64-bound at 44 ms.
// Almost every comparison is far from a tie, so a float value with a bound on
// its error decides it (Shewchuk 1997, "Adaptive precision floating-point
// arithmetic": a filter, then the exact test where the bound leaves the sign
// open).  The decision is always the one that FP64 takes, so the events keep
// every bit.  The same events now take 0.63 ms, bound by instruction issue
// (Philox and the float density; 70 % of the issue slots, FP64 25 %).
//
// A draw is x = lo + W U, U in [0, 1).  The terms work on U, not on x: the
// standardised coordinate (x - mu)/sigma = A + B U, A = (lo - mu)/sigma, B =
// W/sigma as float pairs, keeps full float precision however narrow the peak
// is beside x itself.  The bound on |float value - FP64 value| is absolute and
// uniform in U, so it costs nothing per attempt: e.g. a Gaussian's relative
// error grows as w^2 2^-24, but w^2 exp(-w^2/2) <= 0.74.  In units of 2^-24,
// with the documented errors of __expf (2 + 1.17 |x| ulp) and erfcxf (4 ulp),
// the roundings add up to at most 8 N for GAUSS and EXP, 28 N for GAUSSEXP,
// |c_k| (4 k^2 + 4) N for CHEB and |a_k| X^k (3 k + 4) N for POLY; 64 N and 16
// (k^2 + 2), 16 (k + 2) are used.  Error e0 of the coordinate itself (the pair
// arithmetic, the bits of U left out, the rounding of x in the FP64 value)
// moves these by at most 1.4 N e0; 4 N e0 is used.  A bound that is not
// finite, or a value that is NaN, leaves the decision to FP64.
constexpr int kFilt = 12;  // floats per term; N = weight / I, err = its error bound
// GAUSS    [A, A lo, B, B lo, N, err]              N exp(-w^2/2), w = A + B U
// EXP      [A, A lo, B, B lo, N, err]              N exp(A + B U)
// GAUSSEXP [A, A lo, B, B lo, N, err, s]
// CHEB     [N, err, c_1..c_7]                      in y = 2 U - 1
// POLY     [N, err, lo, W, a_1..a_7]

__device__ __forceinline__ void put_pair(float* o, double v) {
  o[0] = (float)v;
  o[1] = (float)(v - (double)o[0]);
}

// The filter constants of every term of every set: a thread per (set, term).
__global__ void filter_kernel(const __grid_constant__ Program P, const __grid_constant__ GenArgs g,
                              const double* __restrict__ consts, int n_sets, float* __restrict__ out) {
  const int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int n_terms = g.term0[g.n_factors];
  if (id >= (int64_t)n_sets * n_terms) return;
  const int t = (int)(id % n_terms);
  const double* C = consts + (size_t)(id / n_terms) * P.n_const;
  const PNode& q = P.node[g.leaf[t]];
  const double* c = C + q.cofs;
  double N = 1.0;
  for (int i = 0; i < g.n_path[t]; ++i) N *= C[P.node[g.path[t][2 * i]].cofs + g.path[t][2 * i + 1]];
  float k[kFilt];
  for (int i = 0; i < kFilt; ++i) k[i] = 0.0f;
  const double lo = q.lo, W = q.hi - q.lo, X = fmax(fabs(q.lo), fabs(q.hi));
  const float inf = __int_as_float(0x7f800000);
  int at_n = 4, at_e = 5;  // where N and err go
  double err = 0.0;        // over |N|
  switch (q.kind) {
    case GAUSS:
    case GAUSSEXP: {
      const double A = (lo - c[0]) * c[1], B = W * c[1];
      put_pair(k, A);
      put_pair(k + 2, B);
      N *= q.kind == GAUSS ? c[2] : c[4];
      const double e0 = (fabs(A) + fabs(B)) * 0x1p-43 + fabs(B) * 0x1p-32 + (2.0 * X + fabs(c[0])) * c[1] * 0x1p-50;
      err = 0x1p-18 + 4.0 * e0;
      if (q.kind == GAUSSEXP) k[6] = (float)c[2];
      break;
    }
    case EXPO: {
      const double A = c[0] * (lo - c[1]), B = c[0] * W;
      put_pair(k, A);
      put_pair(k + 2, B);
      N *= c[2];
      const double e0 =
          (fabs(A) + fabs(B)) * 0x1p-43 + fabs(B) * 0x1p-32 + (2.0 * X + fabs(c[1])) * fabs(c[0]) * 0x1p-50;
      err = 0x1p-18 + 4.0 * e0;
      break;
    }
    case CHEB: {
      at_n = 0;
      at_e = 1;
      N *= c[2];
      err = 0x1p-20;
      for (int j = 1; j <= q.n_par; ++j) {
        const double a = c[3 + q.n_par + j - 1];
        k[1 + j] = (float)a;
        err += fabs(a) * (j * j + 2) * (0x1p-20 + X / W * 0x1p-48);
      }
      break;
    }
    default: {  // POLY
      at_n = 0;
      at_e = 1;
      N *= c[0];
      err = 0x1p-20;
      double Xk = 1.0;
      for (int j = 1; j <= q.n_par; ++j) {
        const double a = c[1 + q.n_par + j - 1];
        k[3 + j] = (float)a;
        Xk *= X;
        err += fabs(a) * Xk * (j + 2) * 0x1p-20;
      }
      k[2] = (float)lo;
      k[3] = (float)W;
    }
  }
  // Numbers beyond an ordinary float's range leave no bound.  N = 0 (a
  // fraction of exactly 0 or 1) is a term of exactly 0.
  for (int i = 0; i < kFilt; ++i)
    if (!(fabsf(k[i]) < 1e15f)) err = INFINITY;
  if (N != 0.0 && (!(fabs(N) > 1e-25) || !(fabs(N) < 1e25))) err = INFINITY;
  // (the float exponentials flush results below 2^-126; err < 0.01 keeps the
  // linear bounds above valid)
  k[at_n] = (float)N;
  k[at_e] = err < 0.01 ? (float)(fabs(N) * (err + 1e-30)) : inf;
  float4* o = reinterpret_cast<float4*>(out + id * kFilt);
  for (int i = 0; i < kFilt / 4; ++i) o[i] = make_float4(k[4 * i], k[4 * i + 1], k[4 * i + 2], k[4 * i + 3]);
}

// U of a draw's word r0 (r1's bits are below 2^-32 and left out): 23 bits in
// uh, 9 in ul, by bit patterns and exact subtractions (the integer-to-float
// conversions run on a quarter-rate pipe).
__device__ __forceinline__ void filter_u(uint32_t r0, float* uh, float* ul) {
  *uh = __fsub_rn(__uint_as_float((r0 >> 9) | 0x3f800000u), 1.0f);
  *ul = __fmul_rn(__fsub_rn(__uint_as_float((r0 & 0x1ffu) | 0x4b000000u), 8388608.0f), 0x1p-32f);
}

// A + B (uh + ul) with the pairs' products and sums carried to the last
// rounding: error <= 2^-24 |w| + e0.
__device__ __forceinline__ float filter_arg(const float4 ab, float uh, float ul) {
  const float p = __fmul_rn(ab.z, uh), e = __fmaf_rn(ab.z, uh, -p);
  const float s = __fadd_rn(ab.x, p), bb = __fsub_rn(s, ab.x);
  const float r = __fadd_rn(__fsub_rn(ab.x, __fsub_rn(s, bb)), __fsub_rn(p, bb));
  return __fadd_rn(s, __fadd_rn(r, __fadd_rn(e, __fmaf_rn(ab.z, ul, __fmaf_rn(ab.w, uh, ab.y)))));
}

// Factor j's density at U = uh + ul; k: the set's filter constants.
__device__ __forceinline__ float filter_value(const GenArgs& g, int j, const float* __restrict__ k, float uh,
                                              float ul) {
  float sum = 0.0f;
  const int t1 = g.term0[j + 1];
#pragma unroll 1
  for (int t = g.term0[j]; t < t1; ++t) {
    const float4* k4 = reinterpret_cast<const float4*>(k + t * kFilt);
    const float4 ka = __ldg(k4), kb = __ldg(k4 + 1);
    switch (g.kind[t]) {
      case GAUSS: {
        const float w = filter_arg(ka, uh, ul);
        sum = __fmaf_rn(__expf(-0.5f * w * w), kb.x, sum);
        break;
      }
      case EXPO: {
        const float w = filter_arg(ka, uh, ul);
        sum = __fmaf_rn(__expf(w), kb.x, sum);
        break;
      }
      case GAUSSEXP: {
        // z <= 0: exp(A) erfc(z)/2 = exp(A) - exp(-u^2/2) erfcx(-z)/2, A = s (s/2 - u)
        const float u = filter_arg(ka, uh, ul), s = kb.z;
        const float z = (s - u) * 0.70710678f;
        float f = __expf(s * __fmaf_rn(0.5f, s, -u));
        if (!(z < -6.0f)) {  // beyond, the other term is below 1e-16
          const float y = fabsf(z);
          float ex;
          if (z > 1.0f) {
            ex = erfcxf(z);
          } else {
            // Abramowitz & Stegun 7.1.26: erfc(y) to 1.5e-7, absolute
            const float r = __fdividef(1.0f, __fmaf_rn(0.3275911f, y, 1.0f));
            ex = r * __fmaf_rn(r, __fmaf_rn(r, __fmaf_rn(r, __fmaf_rn(r, 1.061405429f, -1.453152027f), 1.421413741f),
                                            -0.284496736f), 0.254829592f);
          }
          const float h = 0.5f * __expf(-0.5f * u * u) * ex;
          f = z > 0.0f ? h : f - h;
        }
        sum = __fmaf_rn(f, kb.x, sum);
        break;
      }
      case CHEB: {
        const float y = __fmaf_rn(2.0f, uh, -1.0f) + 2.0f * ul;
        const int np = g.n_par[t];
        // c_1, c_2 of the record's first vector, then the others
        float t0 = y, t1 = __fmaf_rn(2.0f * y, y, -1.0f), sh = __fmaf_rn(ka.w, t1, __fmaf_rn(ka.z, y, 1.0f));
        for (int i = 3; i <= np; ++i) {
          const float t2 = __fmaf_rn(2.0f * y, t1, -t0);
          t0 = t1;
          t1 = t2;
          sh = __fmaf_rn(__ldg(k + t * kFilt + 1 + i), t1, sh);
        }
        sum = __fmaf_rn(sh, ka.x, sum);
        break;
      }
      default: {  // POLY
        const float xv = __fmaf_rn(ka.w, uh + ul, ka.z);
        float sh = 0.0f;
        for (int i = g.n_par[t]; i >= 1; --i) sh = (sh + __ldg(k + t * kFilt + 3 + i)) * xv;
        sum = __fmaf_rn(sh + 1.0f, ka.x, sum);
      }
    }
  }
  return sum;
}

// The terms' error bounds summed.  The factor 1.25 and the reserve in each
// bound (64 for 28 above, ...) cover the roundings of the terms' sum, at most
// 2^-24 of the sum of the terms' largest values for each of up to 16 terms.
__device__ __forceinline__ float filter_err(const GenArgs& g, int j, const float* __restrict__ k) {
  float e = 0.0f;
  for (int t = g.term0[j]; t < g.term0[j + 1]; ++t)
    e += k[t * kFilt + (g.kind[t] == CHEB || g.kind[t] == POLY ? 1 : 5)];
  return 1.25f * e;
}

// Accept-reject bound M of (set, factor): 1.2 x the largest FP64 density on
// 4096 midpoints, one block per pair; limits: M in float and the distance
// beyond which the float comparison decides.  The float filter leaves the points that
// could be the largest, and only those are evaluated in FP64 (1024 sets of
// the decay model: a few thousand densities instead of 4.2e6; 33 us).
constexpr int kBoundThreads = 256, kBoundPoints = 4096, kBoundPer = kBoundPoints / kBoundThreads;
__global__ void __launch_bounds__(kBoundThreads) bounds_kernel(const __grid_constant__ Program P,
                                                               const __grid_constant__ GenArgs g,
                                                               const double* __restrict__ consts,
                                                               const float* __restrict__ filt,
                                                               double* __restrict__ bounds,
                                                               float2* __restrict__ limits) {
  const int s = blockIdx.x / g.n_factors, j = blockIdx.x % g.n_factors;
  const double* C = consts + (size_t)s * P.n_const;
  const uint32_t mask = g.mask[j];
  const int root = g.factor[j], tid = threadIdx.x;
  const int n_terms = g.term0[g.n_factors];
  const bool filter = g.term0[j + 1] > g.term0[j];
  __shared__ double red[kBoundThreads];
  __shared__ float least[kBoundThreads];
  const double width = g.hi[j] - g.lo[j];
  const float* k = filt + (size_t)s * n_terms * kFilt;
  const float e = filter ? filter_err(g, j, k) : __int_as_float(0x7f800000);
  float up[kBoundPer], low = 0.0f;
  if (filter) {
#pragma unroll 1
    for (int i = 0; i < kBoundPer; ++i) {
      const float uh = ((float)(tid + i * kBoundThreads) + 0.5f) * (1.0f / kBoundPoints);
      const float v = filter_value(g, j, k, uh, 0.0f);
      up[i] = v + e;
      low = fmaxf(low, v - e);
    }
  }
  least[tid] = low;
  __syncthreads();
  for (int o = kBoundThreads / 2; o > 0; o >>= 1) {
    if (tid < o) least[tid] = fmaxf(least[tid], least[tid + o]);
    __syncthreads();
  }
  low = least[0];
  double mx = 0.0;
#pragma unroll 1
  for (int i = 0; i < kBoundPer; ++i) {
    if (filter && up[i] < low) continue;
    const int p = tid + i * kBoundThreads;
    const double d = factor_value(P, C, mask, root, __dadd_rn(g.lo[j], __dmul_rn(width, (p + 0.5) / 4096.0)));
    if (d > mx) mx = d;
  }
  red[tid] = mx;
  __syncthreads();
  for (int o = kBoundThreads / 2; o > 0; o >>= 1) {
    if (tid < o) red[tid] = fmax(red[tid], red[tid + o]);
    __syncthreads();
  }
  if (tid == 0) {
    const double M = 1.2 * red[0];
    bounds[(size_t)s * kMaxFactors + j] = M;
    // the events' comparison: y = M u' to 23 bits of u', four roundings
    limits[(size_t)s * kMaxFactors + j] = make_float2((float)M, e + (float)M * 0x1p-20f);
  }
}

// Set sizes: Poisson(mean) (or round(mean) when poisson == 0), one thread per set.
__global__ void sizes_kernel(const double* __restrict__ mean_n, int n_sets, int poisson, uint32_t k0, uint32_t k1,
                             int64_t* __restrict__ sizes) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= n_sets) return;
  const double mu = mean_n[s];
  if (!poisson) {
    sizes[s] = (mu > 0.0) ? (int64_t)llrint(mu) : 0;
    return;
  }
  if (!(mu > 0.0)) {
    sizes[s] = 0;
    return;
  }
  uint32_t r[4];
  if (mu < 10.0) {
    philox4x32_10(0u, 0u, (uint32_t)s, 0xFFFFFFFFu, k0, k1, r);
    const double u = u53(r[0], r[1]);
    double p = exp(-mu), F = p;
    int64_t k = 0;
    while (u > F && k < 1000) {
      ++k;
      p = __dmul_rn(p, __ddiv_rn(mu, (double)k));
      F = __dadd_rn(F, p);
    }
    sizes[s] = k;
    return;
  }
  const double smu = sqrt(mu);
  const double b = __dadd_rn(0.931, __dmul_rn(2.53, smu));
  const double a = __dadd_rn(-0.059, __dmul_rn(0.02483, b));
  const double inv_alpha = __dadd_rn(1.1239, __ddiv_rn(1.1328, __dsub_rn(b, 3.4)));
  const double vr = __dsub_rn(0.9277, __ddiv_rn(3.6224, __dsub_rn(b, 2.0)));
  const double log_mu = log(mu);
  for (uint32_t j = 0; j < 100000u; ++j) {
    philox4x32_10(j, 0u, (uint32_t)s, 0xFFFFFFFFu, k0, k1, r);
    const double U = __dsub_rn(u53_open(r[0], r[1]), 0.5);
    const double V = u53_open(r[2], r[3]);
    const double us = __dsub_rn(0.5, fabs(U));
    const double kd =
        floor(__dadd_rn(__dadd_rn(__dmul_rn(__dadd_rn(__ddiv_rn(__dmul_rn(2.0, a), us), b), U), mu), 0.43));
    if (us >= 0.07 && V <= vr) {
      sizes[s] = (int64_t)kd;
      return;
    }
    if (kd < 0.0 || (us < 0.013 && V > us)) continue;
    const double lhs = __dsub_rn(__dadd_rn(log(V), log(inv_alpha)), log(__dadd_rn(__ddiv_rn(a, __dmul_rn(us, us)), b)));
    const double rhs = __dsub_rn(__dadd_rn(-mu, __dmul_rn(kd, log_mu)), lgamma(__dadd_rn(kd, 1.0)));
    if (lhs <= rhs) {
      sizes[s] = (int64_t)kd;
      return;
    }
  }
  sizes[s] = -1;
}

// Events, at 7 blocks an SM (72 registers: 632 us for 2.4e7 decay events; 5
// blocks without spills 688, 6 640, 8 670).  A warp takes a pool of consecutive events (over set boundaries)
// and draws one factor's observable for all of them: every lane tries its
// event's next attempt, and a lane whose event is accepted takes the pool's
// next one, so lanes with few attempts do not wait for those with many (a
// lane per event leaves two thirds of the lanes idle at 30 % acceptance).
// An accepted draw is kept as its 53 bits; the pool's observables are then
// computed in FP64 and stored densely, one FP64 sequence per 32 events
// instead of one per loop turn.  The decision is the float filter's where it
// can take one, else FP64 (of the order of 1e-4 of the attempts).
constexpr int kGenWarps = 4, kPoolMax = 512;
__global__ void __launch_bounds__(32 * kGenWarps, 7) events_kernel(
    const __grid_constant__ Program P, const __grid_constant__ GenArgs g, const double* __restrict__ consts,
    const float* __restrict__ filt, const double* __restrict__ bounds, const float2* __restrict__ limits,
    const int64_t* __restrict__ offsets, int n_sets, int64_t n_events, int pool, uint32_t k0, uint32_t k1,
    const __grid_constant__ Columns out, int32_t* __restrict__ error) {
  __shared__ uint64_t kept[kGenWarps][kPoolMax];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t first = ((int64_t)blockIdx.x * kGenWarps + warp) * pool;
  if (first >= n_events) return;
  const int n = (int)(n_events - first < pool ? n_events - first : pool);
  uint64_t* keep = kept[warp];
  int lo = 0, hi = n_sets - 1;  // last set with offsets[set] <= first
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (offsets[mid] <= first) lo = mid;
    else hi = mid - 1;
  }
  const int set0 = lo, n_terms = g.term0[g.n_factors];
  for (int j = 0; j < g.n_factors; ++j) {
    const uint32_t mask = g.mask[j];
    const int root = g.factor[j], col = g.fcol[j];
    const bool filter = g.term0[j + 1] > g.term0[j];
    const double width = __dsub_rn(g.hi[j], g.lo[j]);
    int i = lane, s = set0, next = min(32, n);  // the lane's event, its set; the pool's next event
    // the set's events as pool indices [s_beg, s_end), and the attempt
    int64_t s_beg = offsets[s] - first, s_end = offsets[s + 1] - first;
    uint32_t a = 0;
    float2 lim = __ldg(limits + (size_t)s * kMaxFactors + j);  // M and the filter's reach
    const float* fk = filt + (size_t)s * n_terms * kFilt;
    bool live = i < n;
    while (__any_sync(0xffffffffu, live)) {
      bool done = false;
      if (live) {
        if (i >= s_end) {
          do s_end = offsets[++s + 1] - first;
          while (i >= s_end);
          s_beg = offsets[s] - first;
          lim = __ldg(limits + (size_t)s * kMaxFactors + j);
          fk = filt + (size_t)s * n_terms * kFilt;
        }
        uint32_t r[4];
        philox4x32_10((uint32_t)(i - s_beg), a, (uint32_t)s, (uint32_t)j, k0, k1, r);
        float uh, ul, d = 0.0f;
        filter_u(r[0], &uh, &ul);
        const float u2 = __fsub_rn(__uint_as_float((r[2] >> 9) | 0x3f800000u), 1.0f);
        if (filter) d = __fmaf_rn(-lim.x, u2, filter_value(g, j, fk, uh, ul));
        bool accept = d > lim.y;
        if (!accept && !(d < -lim.y)) {  // too near, or no bound: the FP64 comparison itself
          const double xv = __dadd_rn(g.lo[j], __dmul_rn(width, u53(r[0], r[1])));
          accept = __dmul_rn(bounds[(size_t)s * kMaxFactors + j], u53(r[2], r[3])) <
                   factor_value(P, consts + (size_t)s * P.n_const, mask, root, xv);
        }
        ++a;
        if (accept) keep[i] = ((uint64_t)r[0] << 21) | (r[1] >> 11);
        done = accept;
        if (!accept && a == kMaxAttempts) {
          atomicExch(error, 1);
          keep[i] = 0;
          done = true;
        }
      }
      const unsigned m = __ballot_sync(0xffffffffu, done);
      if (done) {
        i = next + __popc(m & ((1u << lane) - 1u));
        a = 0;
        live = i < n;
      }
      next += __popc(m);
    }
    __syncwarp();
    for (int t = lane; t < n; t += 32) {
      const double xv = __dadd_rn(g.lo[j], __dmul_rn(width, (double)keep[t] * 0x1p-53));
      if (out.is_f32[col]) ((float*)out.ptr[col])[first + t] = (float)xv;
      else ((double*)out.ptr[col])[first + t] = xv;
    }
    __syncwarp();
  }
}

// Per-set 64-bin histogram: bin = floor((x - lo) scale) in FP64, clamped to
// [0, 63].  Bound by the FP64 unit when taken literally (a conversion, a
// subtraction, a product and a floor per event, 64 cycles each), so the bin is
// taken in float where the float coordinate is further than `reach` (in bins)
// from the next bin edge, which is its largest distance from the FP64 one for
// an x in [lo - span, hi + span]; other x, NaN and infinities among them, take
// the FP64 expression (1024 sets, 2.4e7 events: 305 -> 72 us).  `split` blocks share a set's events; with several,
// they add their counts to the integers that the caller's output holds in the
// meantime (hist64_norm_kernel turns them into fractions).
constexpr int kHistThreads = 256, kHistLogCopies = 4, kHistCopies = 1 << kHistLogCopies, kHistSmall = 1024;
// Out of line: inlined, the compiler would compute the FP64 bin of every
// event and select.
__device__ __noinline__ int hist_bin_fp64(double x, double lo, double scale) {
  return (int)floor(__dmul_rn(__dsub_rn(x, lo), scale));
}
__device__ __forceinline__ int hist_bin(double x, float xf, double lo, double scale, float lof, float scalef,
                                        float reach) {
  const float t = __fmul_rn(__fsub_rn(xf, lof), scalef);
  const float b = floorf(t), f = __fsub_rn(t, b);
  int bin;
  if (f > reach && f < 1.0f - reach && t > -64.0f && t < 128.0f) bin = (int)b;
  else bin = hist_bin_fp64(x, lo, scale);
  return min(63, max(0, bin));
}
// The float nearest below |x| (from the bits: the FP64-to-float conversion
// runs on the FP64 unit); zero for what is below the float range, infinite above.
__device__ __forceinline__ float hist_float(double x) {
  const uint32_t h = (uint32_t)__double2hiint(x), l = (uint32_t)__double2loint(x);
  const int ex = (int)((h >> 20) & 0x7ffu) - 896;
  const uint32_t mag = ex <= 0 ? 0u : ex >= 255 ? 0x7f800000u : ((uint32_t)ex << 23) | ((h & 0xfffffu) << 3) | (l >> 29);
  return __uint_as_float((h & 0x80000000u) | mag);
}
template <bool kF32, int kThreads>
__global__ void __launch_bounds__(kThreads) hist64_kernel(const void* __restrict__ colp,
                                                          const int64_t* __restrict__ offsets, double lo,
                                                          double scale, float lof, float scalef, float reach,
                                                          int split, float* __restrict__ out) {
  // 16 copies of the 64 counters, a lane's copy interleaved over the banks:
  // a peaked column puts many of a warp's events into one bin.  A small set
  // has one copy: clearing and adding up 16 takes longer than its events.
  __shared__ int bins[64 * kHistCopies];
  const int s = split == 1 ? blockIdx.x : blockIdx.x / split, part = blockIdx.x - s * split, tid = threadIdx.x;
  const int64_t b0 = offsets[s], b1 = offsets[s + 1], n = b1 - b0;
  const int log_copies = n < kHistSmall ? 0 : kHistLogCopies, copies = 1 << log_copies;
  for (int i = tid; i < 64 * copies; i += kThreads) bins[i] = 0;
  __syncthreads();
  const int64_t e1 = split == 1 ? b1 : b0 + n * (part + 1) / split;
  int* mine = bins + (tid & (copies - 1));
  int64_t e = (split == 1 ? b0 : b0 + n * part / split) + tid;
  constexpr int kU = 8;  // loads in flight per thread
  for (; e + (kU - 1) * kThreads < e1; e += kU * kThreads) {
    if constexpr (kF32) {  // (an FP32 column widens only where FP64 decides)
      float x[kU];
#pragma unroll
      for (int i = 0; i < kU; ++i) x[i] = __ldg((const float*)colp + e + i * kThreads);
#pragma unroll
      for (int i = 0; i < kU; ++i)
        atomicAdd(mine + (hist_bin((double)x[i], x[i], lo, scale, lof, scalef, reach) << log_copies), 1);
    } else {
      double x[kU];
#pragma unroll
      for (int i = 0; i < kU; ++i) x[i] = __ldg((const double*)colp + e + i * kThreads);
#pragma unroll
      for (int i = 0; i < kU; ++i)
        atomicAdd(mine + (hist_bin(x[i], hist_float(x[i]), lo, scale, lof, scalef, reach) << log_copies), 1);
    }
  }
  for (; e < e1; e += kThreads) {
    const double x = kF32 ? (double)__ldg((const float*)colp + e) : __ldg((const double*)colp + e);
    const float xf = kF32 ? __ldg((const float*)colp + e) : hist_float(x);
    atomicAdd(mine + (hist_bin(x, xf, lo, scale, lof, scalef, reach) << log_copies), 1);
  }
  __syncthreads();
  if (tid < 64) {
    int c = 0;
    for (int i = 0; i < copies; ++i) c += bins[(tid << log_copies) + ((i + tid) & (copies - 1))];
    float* o = out + (size_t)s * 64 + tid;
    if (split == 1) *o = n > 0 ? (float)((double)c / (double)n) : 0.0f;
    else if (c) atomicAdd(reinterpret_cast<int*>(o), c);
  }
}
__global__ void hist64_norm_kernel(const int64_t* __restrict__ offsets, int n_sets, float* __restrict__ out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)n_sets * 64) return;
  const int64_t n = offsets[i / 64 + 1] - offsets[i / 64];
  out[i] = n > 0 ? (float)((double)__float_as_int(out[i]) / (double)n) : 0.0f;
}

// Appends the float filter's terms of the factor at node `root`, from term
// `t0` on, to g; returns the end (t0 if the factor has no float form: a
// Poisson leaf needs the exact floor of x, a program is interpreted in FP64,
// a product is no sum of leaves, or too many terms).
int filter_terms(const Program& P, int root, GenArgs& g, int t0) {
  struct Item {
    int node, n_path;
    int8_t path[2 * kMaxPath];
  };
  std::vector<Item> todo(1);
  todo[0] = Item{};
  todo[0].node = root;
  int t = t0;
  while (!todo.empty()) {
    const Item it = todo.back();
    todo.pop_back();
    const PNode& q = P.node[it.node];
    if (q.kind == SUM) {
      if (it.n_path == kMaxPath || todo.size() > kMaxTerms) return t0;
      for (int c = q.n_child - 1; c >= 0; --c) {
        Item next = it;
        next.node = q.child[c];
        next.path[2 * it.n_path] = (int8_t)it.node;
        next.path[2 * it.n_path + 1] = (int8_t)c;
        next.n_path = it.n_path + 1;
        todo.push_back(next);
      }
      continue;
    }
    if (t == kMaxTerms || t - t0 == kMaxFactorTerms ||
        (q.kind != GAUSS && q.kind != EXPO && q.kind != GAUSSEXP && q.kind != CHEB && q.kind != POLY))
      return t0;
    g.leaf[t] = (int8_t)it.node;
    g.kind[t] = q.kind;
    g.n_par[t] = q.n_par;
    g.n_path[t] = (int8_t)it.n_path;
    std::memcpy(g.path[t], it.path, sizeof it.path);
    ++t;
  }
  return t;
}

}  // namespace

}  // namespace rf

using namespace rf;

extern "C" {

rf_status rf_generate_toys(const rf_model* m, const double* theta, int32_t theta_per_set, uint64_t seed,
                           int32_t n_sets, const double* mean_n, int32_t poisson, const int32_t* dtype,
                           rf_data** out) {
  if (!m || !out || n_sets < 1 || !mean_n) {
    set_error("rf_generate_toys: bad argument");
    return RF_E_INVALID;
  }
  *out = nullptr;
  const Model& mm = m->m;
  const Program& P = mm.prog;
  if (mm.gen_factors.empty() || (int)mm.gen_factors.size() > kMaxFactors) {
    set_error("rf_generate_toys: the model must be a product of 1-D factors (or one 1-D pdf)");
    return RF_E_INVALID;
  }
  for (int s = 0; s < n_sets; ++s)
    if (!(mean_n[s] >= 0.0) || mean_n[s] > 2e9) {
      set_error("rf_generate_toys: mean sizes must be in [0, 2e9]");
      return RF_E_INVALID;
    }
  const int nf = P.n_free;
  std::vector<double> th((size_t)n_sets * nf);
  for (int s = 0; s < n_sets; ++s)
    for (int k = 0; k < nf; ++k)
      th[(size_t)s * nf + k] = theta ? theta[(theta_per_set ? (size_t)s * nf : 0) + k] : mm.theta_default[k];

  GenArgs g{};
  g.n_factors = (int)mm.gen_factors.size();  // (term0[0] = 0)
  for (int j = 0; j < g.n_factors; ++j) {
    g.factor[j] = mm.gen_factors[j];
    // the factor's observable: the column of its first leaf
    int n = mm.gen_factors[j];
    while (P.node[n].kind == SUM || P.node[n].kind == PROD) n = P.node[n].child[0];
    g.fcol[j] = P.node[n].col;
    g.lo[j] = mm.obs_lo[g.fcol[j]];
    g.hi[j] = mm.obs_hi[g.fcol[j]];
    g.mask[j] = 1u << g.factor[j];  // children come before their parents
    for (int i = g.factor[j]; i >= 0; --i)
      if (g.mask[j] >> i & 1u)
        for (int c = 0; c < P.node[i].n_child; ++c) g.mask[j] |= 1u << P.node[i].child[c];
    g.term0[j + 1] = filter_terms(P, g.factor[j], g, g.term0[j]);
  }
  const uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);

  const int n_terms = g.term0[g.n_factors];

  // Constants of the generating parameters (the parameter-point kernel).
  DevBuf d_theta, d_consts, d_sets, d_flags, d_out, d_counter, d_bounds, d_limits, d_filt, d_mean, d_sizes, d_err;
  std::vector<int32_t> sets(n_sets);
  for (int s = 0; s < n_sets; ++s) sets[s] = s;
  if (!d_theta.ensure(sizeof(double) * std::max<size_t>(1, th.size())) ||
      !d_consts.ensure(sizeof(double) * n_sets * std::max(1, P.n_const)) || !d_sets.ensure(sizeof(int32_t) * n_sets) ||
      !d_flags.ensure(sizeof(int32_t) * n_sets) || !d_out.ensure(sizeof(double) * n_sets * (1 + nf)) ||
      !d_counter.ensure(sizeof(int32_t)) || !d_bounds.ensure(sizeof(double) * n_sets * kMaxFactors) ||
      !d_limits.ensure(sizeof(float2) * n_sets * kMaxFactors) ||
      !d_filt.ensure(sizeof(float) * kFilt * (size_t)n_sets * std::max(1, n_terms)) || !d_mean.ensure(sizeof(double) * n_sets) || !d_sizes.ensure(sizeof(int64_t) * n_sets) || !d_err.ensure(sizeof(int32_t)))
    return RF_E_OOM;
  std::vector<int64_t> zero_off(n_sets + 1, 1);  // every set "non-empty" for the parameter-point pass
  DevBuf d_zoff;
  for (int s = 0; s <= n_sets; ++s) zero_off[s] = s;
  if (!d_zoff.ensure(sizeof(int64_t) * (n_sets + 1))) return RF_E_OOM;
  bool ok = cuda_ok(cudaMemcpy(d_theta.p, th.data(), sizeof(double) * th.size(), cudaMemcpyHostToDevice), "theta") &&
            cuda_ok(cudaMemcpy(d_sets.p, sets.data(), sizeof(int32_t) * n_sets, cudaMemcpyHostToDevice), "sets") &&
            cuda_ok(cudaMemcpy(d_mean.p, mean_n, sizeof(double) * n_sets, cudaMemcpyHostToDevice), "mean") &&
            cuda_ok(cudaMemcpy(d_zoff.p, zero_off.data(), sizeof(int64_t) * (n_sets + 1), cudaMemcpyHostToDevice), "off") &&
            cuda_ok(cudaMemset(d_err.p, 0, sizeof(int32_t)), "memset");
  if (!ok) return RF_E_CUDA;
  Pass pass{};
  pass.offsets = (const int64_t*)d_zoff.p;
  pass.sets = (const int32_t*)d_sets.p;
  pass.n_active = n_sets;
  pass.theta = (const double*)d_theta.p;
  pass.consts = (double*)d_consts.p;
  pass.counter = (int32_t*)d_counter.p;
  pass.out = (double*)d_out.p;
  pass.flags = (int32_t*)d_flags.p;
  pass.Q = 1;
  launch_param_point(P, pass, 0);
  std::vector<int32_t> flags(n_sets);
  if (!cuda_ok(cudaMemcpy(flags.data(), d_flags.p, sizeof(int32_t) * n_sets, cudaMemcpyDeviceToHost), "flags"))
    return RF_E_CUDA;
  for (int s = 0; s < n_sets; ++s)
    if (flags[s]) {
      set_error("rf_generate_toys: generating parameters outside the pdf's domain");
      return RF_E_DOMAIN;
    }
  if (n_terms > 0) {
    note_launches(1, nullptr);
    filter_kernel<<<(unsigned)(((int64_t)n_sets * n_terms + 127) / 128), 128>>>(P, g, (const double*)d_consts.p, n_sets,
                                                                                (float*)d_filt.p);
  }
  note_launches(1, nullptr);
  bounds_kernel<<<n_sets * g.n_factors, kBoundThreads>>>(P, g, (const double*)d_consts.p, (const float*)d_filt.p,
                                                         (double*)d_bounds.p, (float2*)d_limits.p);
  note_launches(1, nullptr);
  sizes_kernel<<<(n_sets + 127) / 128, 128>>>((const double*)d_mean.p, n_sets, poisson, k0, k1,
                                              (int64_t*)d_sizes.p);
  std::vector<int64_t> sizes(n_sets);
  if (!cuda_ok(cudaGetLastError(), "launch") ||
      !cuda_ok(cudaMemcpy(sizes.data(), d_sizes.p, sizeof(int64_t) * n_sets, cudaMemcpyDeviceToHost), "sizes"))
    return RF_E_CUDA;
  std::vector<int64_t> off(n_sets + 1, 0);
  for (int s = 0; s < n_sets; ++s) {
    if (sizes[s] < 0) {
      set_error("rf_generate_toys: Poisson draw did not terminate");
      return RF_E_TIMEOUT;
    }
    off[s + 1] = off[s] + sizes[s];
  }
  rf_data* d = new (std::nothrow) rf_data();
  if (!d) return RF_E_OOM;
  d->n_obs = P.n_obs;
  d->n_sets = n_sets;
  d->n_events = off[n_sets];
  d->offsets = off;
  d->owns_cols = true;
  Columns outc{};
  for (int c = 0; c < P.n_obs; ++c) {
    d->dtype[c] = dtype ? dtype[c] : RF_F64;
    if (d->dtype[c] != RF_F64 && d->dtype[c] != RF_F32) {
      delete d;
      set_error("rf_generate_toys: dtype must be RF_F64 or RF_F32");
      return RF_E_INVALID;
    }
    if (!d->col_bufs[c].ensure((size_t)std::max<int64_t>(1, d->n_events) * (d->dtype[c] == RF_F32 ? 4 : 8))) {
      delete d;
      return RF_E_OOM;
    }
    d->cols[c] = d->col_bufs[c].p;
    outc.ptr[c] = d->cols[c];
    outc.is_f32[c] = d->dtype[c] == RF_F32;
  }
  rf_status st = finish_data(d);
  if (st != RF_OK) {
    delete d;
    return st;
  }
  if (d->n_events > 0) {
    // A pool ends with idle lanes, so large ones are better (512: 26 of 32
    // lanes active over the whole kernel); few events take smaller pools, down
    // to one event a lane, so that all SMs (at 32 warps each) have work.
    int pool = kPoolMax;
    while (pool > 32 && d->n_events < (int64_t)pool * 32 * sm_count()) pool /= 2;
    const int64_t blocks = (d->n_events + (int64_t)pool * kGenWarps - 1) / ((int64_t)pool * kGenWarps);
    note_launches(1, nullptr);
    events_kernel<<<(unsigned)blocks, 32 * kGenWarps>>>(P, g, (const double*)d_consts.p, (const float*)d_filt.p,
                                                        (const double*)d_bounds.p, (const float2*)d_limits.p,
                                                        (const int64_t*)d->offsets_dev.p, n_sets, d->n_events, pool, k0, k1, outc, (int32_t*)d_err.p);
  }
  int32_t err = 0;
  if (!cuda_ok(cudaGetLastError(), "launch") ||
      !cuda_ok(cudaMemcpy(&err, d_err.p, sizeof(int32_t), cudaMemcpyDeviceToHost), "generation")) {
    delete d;
    return RF_E_CUDA;
  }
  if (err) {
    delete d;
    set_error("rf_generate_toys: an event needed more than 100000 accept-reject attempts");
    return RF_E_TIMEOUT;
  }
  *out = d;
  return RF_OK;
}

rf_status rf_hist64(const rf_model* m, const rf_data* d, int32_t col, float* d_out, void* stream) {
  if (!m || !d || !d_out || col < 0 || col >= d->n_obs || d->n_obs != m->m.prog.n_obs) {
    set_error("rf_hist64: bad argument");
    return RF_E_INVALID;
  }
  const cudaStream_t st = (cudaStream_t)stream;
  const double lo = m->m.obs_lo[col], hi = m->m.obs_hi[col], scale = 64.0 / (hi - lo);
  // x, lo and scale as floats, the difference and the product: at most 2^-23
  // of |x| + |lo| and, for an x that is no normal float, 2^-126 (hist_float
  // takes it as zero), in bins, and 2^-22 of the coordinate (below 128); four
  // times that (beyond 0.5, every event takes the FP64 expression).
  const double far = std::max(std::fabs(lo), std::fabs(hi)) + (hi - lo);
  const float reach = (float)std::min(1.0, 4.0 * ((2.0 * far * 0x1p-23 + 0x1p-126) * scale + 128.0 * 0x1p-22));
  // Blocks per set: 8 resident blocks an SM fill the GPU; a block takes at
  // least 16384 events (64 a thread), below which a second one gains nothing.
  const int64_t per_set = (d->n_events + d->n_sets - 1) / d->n_sets;
  const int64_t most = std::max<int64_t>(1, 8 * (int64_t)sm_count() / d->n_sets);
  const int split = (int)std::max<int64_t>(1, std::min(most, per_set / 16384));
  const int64_t* off = (const int64_t*)d->offsets_dev.p;
  if (split > 1 &&
      !cuda_ok(cudaMemsetAsync(d_out, 0, sizeof(float) * 64 * (size_t)d->n_sets, st), "rf_hist64 reset"))
    return RF_E_CUDA;
  note_launches(1, st);
  // Sets that all have fewer than 512 events take blocks of 64 threads: 20000
  // sets of 50 events 80 -> 67 us (88 with 256 threads and 16 copies of the
  // counters), 3000 of 300 27 -> 22; at 512 the two are equal.
  const bool small = d->max_set < 512, f32 = d->dtype[col] == RF_F32;
  const auto kernel = small ? (f32 ? hist64_kernel<true, 64> : hist64_kernel<false, 64>)
                            : (f32 ? hist64_kernel<true, kHistThreads> : hist64_kernel<false, kHistThreads>);
  kernel<<<d->n_sets * split, small ? 64 : kHistThreads, 0, st>>>(d->cols[col], off, lo, scale, (float)lo, (float)scale,
                                                                 reach, split, d_out);
  if (split > 1) {
    note_launches(1, st);
    hist64_norm_kernel<<<(d->n_sets * 64 + 255) / 256, 256, 0, st>>>(off, d->n_sets, d_out);
  }
  return cuda_ok(cudaGetLastError(), "rf_hist64 launch") ? RF_OK : RF_E_CUDA;
}

}  // extern "C"
