// Binned (HistFactory-style) likelihood: NLL and gradient of many datasets
// of bin counts at once (paper Sec. 3: models built from histograms --
// channels of samples with +-1 sigma systematic variations).
//
// nu_s[i] = prod(normfactors) prod(normsys eta) (h_s[i] + sum histosys
// delta), eta = exp(a alpha + b g(alpha)) with a, b = (log k_hi -+ log
// k_lo)/2, delta_i = a_i alpha + b_i g(alpha) with a_i = (h_hi - h_lo)/2,
// b_i = (h_hi + h_lo)/2 - h, g = alpha^2 inside +-1 and 2|alpha| - 1
// beyond (quadratic interpolation, linear extrapolation: continuous with a
// continuous derivative, so quasi-Newton fits see no kink); nu_b = sum over
// the samples on bin b; NLL = sum_b (nu_b - n_b log nu_b) + sum over
// constrained parameters theta^2/2.  d NLL / d theta_k = sum_b w_b d nu_b /
// d theta_k + [constrained] theta_k, w_b = 1 - n_b / nu_b; per modifier of
// parameter k: a normfactor or normsys on sample s contributes dlog(factor)
// / dtheta_k sum_i w nu_s[i], a histosys F_s sum_i w (a_i + b_i g').
//
// (One block per dataset, each reading every coefficient for itself and waiting
// for it, took 490 us for one dataset of the 28-channel model and 1500 us for
// 1024; this takes 58 and 834 us a call: the float-float loops 0.29 ms each, at
// about 60 % of the FP32 pipe's rate, the bins' FP64 division and logarithm
// 0.13 ms.)
// A pass is five chained kernels over (dataset, work) grids -- parameters and
// sample factors, entry rates, bins, weighted sums, gradient and NLL -- so one
// dataset fills as many SMs as its work can, and many datasets share every
// coefficient load (four datasets a thread).  Every sum has a fixed order
// (samples, bins and modifiers in index order, fixed trees), so results do not
// depend on the launch or on the other datasets.  The two
// loops that carry nearly all the multiply-adds -- the entries' histosys
// sums and the histosys modifiers' weighted coefficient sums -- and the
// samples' weighted sums run in float-float on the FP32 pipe (ff.cuh: FP64
// issues at 1/58 of the FP32 rate); the sample factors, the bins' Poisson
// terms and weights, the gradient's assembly and the expected counts stay
// in FP64.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "api_internal.h"
#include "ff.cuh"

namespace rf {

namespace {

constexpr int kBinnedThreads = 256;
constexpr int kMaxBinnedBins = 8192, kMaxBinnedSamples = 2048;

// The largest model: this many bytes have to fit a block's shared memory (the
// expected-counts kernel's theta, g, g' and F fit in them too).
size_t binned_smem(int n_params, int n_samples, int n_bins) {
  return sizeof(double) * (5 * (size_t)n_params + 3 * (size_t)n_samples + (size_t)n_bins + kBinnedThreads);
}

enum ModKind : int32_t { MOD_NORMFACTOR = 0, MOD_NORMSYS = 1, MOD_HISTOSYS = 2 };

// A factor modifier of a sample and a modifier of a parameter (normsys: a, b of
// log eta = a alpha + b g(alpha)).
struct FactorRec {
  int32_t param, kind;
  double a, b;
};
struct GradRec {
  int32_t kind, sample, hs, pad;
  double a, b;
};

struct BinnedDev {
  int32_t n_bins, n_samples, n_params, n_mods, n_entries, n_hs;
  const int32_t* bin0;        // per sample: first bin
  const int32_t* nb;          // per sample: bins
  const int32_t* eofs;        // per sample: its first (sample, bin) entry; entries run sample by sample
  const int32_t* esample;     // per entry: its sample
  const double* nominal;      // per entry
  const int32_t* smod_start;  // per sample: its normfactor / normsys modifiers (CSR, modifier order; `factor`)
  const int32_t* shs_start;   // per sample: its histosys modifiers (CSR, modifier order), as indices
  const int32_t* shs;         //   into the histosys arrays below
  const double* coef;         // per histosys: a_i then b_i, nb each (at shs_ofs)
  // The same coefficients transposed per sample for the weighted sums:
  // sample s's histosys j (its j-th in shs order) at local bin i sits at
  // tbase[s] + i * (histosys of s) + j, in coef_af and coef_bf.
  const int64_t* tbase;
  const int32_t* g_sample;    // per position in shs: its sample
  // The nominal rates and the histosys coefficients again as float pairs
  // (same indexing), for the float-float loops.
  const float2* nominal_f;
  const float2* coef_f;
  const int32_t* shs_k;       // per position in shs: the histosys's parameter and
  const int64_t* shs_ofs;     //   coefficient offset (one load level instead of two)
  const float2* coef_af;
  const float2* coef_bf;
  const int32_t* bin_start;   // per bin: its entries (CSR, sample order)
  const int32_t* bin_entry;
  const int32_t* pmod_start;  // per parameter: its modifiers (CSR, normfactors first, modifier order; `grad`)
  const int32_t* pmod_norm;   // per parameter: the end of its normfactors
  const int32_t* constrained;
  // The modifiers as records in the order they are summed.
  const FactorRec* factor;
  const GradRec* grad;
};

// The intermediate results of a pass for up to rf_binned::cap datasets,
// dataset-major.
struct BinnedScratch {
  float4* pt;      // per parameter: theta and g as float pairs
  double* dgk;     // g'
  double* F;       // per sample: its factor, the same as a pair, sum_i w nu_s[i]
  float2* Ff;
  double* Ssum;
  float2* nu_e;    // per entry
  float2* W;       // per bin: weight, Poisson term
  double* term;
  double* T;       // per histosys: sum_i w (a_i + b_i g')
};

__device__ __forceinline__ ff ld_pair(const float2* p) {
  const float2 v = __ldg(p);
  return {v.x, v.y};
}
__device__ __forceinline__ ff as_ff(double v) { return ff_from_double(v); }

// theta and g(theta) into smem (once per parameter and dataset:
// an FP64 comparison per term would occupy the FP64 unit as long as the
// multiply-add itself), then the sample factors F: the normfactors times
// one exponential of the normsys exponents' sum.
__device__ __forceinline__ void sample_factors(const BinnedDev& m, const double* th_g, double* th, double* gk,
                                               double* F) {
  for (int k = threadIdx.x; k < m.n_params; k += kBinnedThreads) {
    const double a = th_g[k];
    th[k] = a;
    const bool in = fabs(a) <= 1.0;
    gk[k] = in ? a * a : 2.0 * fabs(a) - 1.0;
  }
  __syncthreads();
  for (int s = threadIdx.x; s < m.n_samples; s += kBinnedThreads) {
    double f = 1.0, le = 0.0;
    for (int j = m.smod_start[s]; j < m.smod_start[s + 1]; ++j) {
      const FactorRec r = m.factor[j];
      if (r.kind == MOD_NORMFACTOR) f *= th[r.param];
      else le = fma(r.b, gk[r.param], fma(r.a, th[r.param], le));
    }
    F[s] = le != 0.0 ? f * exp(le) : f;
  }
  __syncthreads();
}

// nu of every (sample, bin) entry in FP64 (for the expected counts).  A block
// waits for its chain of loads (a histosys's parameter and offset, then its
// coefficients), so these are two levels, four at a time: one dataset of the
// 28-channel model 355 -> 213 us, 1024 995 -> 894.
__device__ __forceinline__ void entry_rates(const BinnedDev& m, const double* th, const double* gk, const double* F,
                                            double* nu_e) {
  for (int e = threadIdx.x; e < m.n_entries; e += kBinnedThreads) {
    const int s = m.esample[e], i = e - m.eofs[s], n = m.nb[s];
    double shape = m.nominal[e];
    const int j1 = m.shs_start[s + 1];
#pragma unroll 4
    for (int j = m.shs_start[s]; j < j1; ++j) {
      const int k = __ldg(m.shs_k + j);
      const double* c = m.coef + __ldg(m.shs_ofs + j) + i;
      shape = fma(__ldg(c + n), gk[k], fma(__ldg(c), th[k], shape));
    }
    nu_e[e] = F[s] * shape;
  }
}

// Each kernel of a pass is a programmatic dependent of the one before: it is
// scheduled while that runs and waits here for its results (which it then
// reads with plain loads: the read-only path may not see them).
__device__ __forceinline__ void chain_wait() {
  asm volatile("griddepcontrol.launch_dependents;");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Step 1: block (set, chunk of samples).  theta, g, g' of the set (all blocks
// need them, chunk 0 stores them), then the chunk's sample factors: the
// normfactors times one exponential of the normsys exponents' sum.
constexpr int kPrepThreads = 128;
__global__ void __launch_bounds__(kPrepThreads) binned_prep_kernel(const BinnedDev m, const BinnedScratch w,
                                                                   const double* theta, int per_block,
                                                                   int32_t* flags) {
  extern __shared__ double smem[];
  double* th = smem;
  double* gk = th + m.n_params;
  chain_wait();
  const int set = blockIdx.y;
  const double* th_g = theta + (size_t)set * m.n_params;
  for (int k = threadIdx.x; k < m.n_params; k += kPrepThreads) {
    const double a = th_g[k];
    const bool in = fabs(a) <= 1.0;
    const double g = in ? a * a : 2.0 * fabs(a) - 1.0;
    th[k] = a;
    gk[k] = g;
    if (blockIdx.x == 0) {
      const ff t = as_ff(a), u = as_ff(g);
      w.pt[(size_t)set * m.n_params + k] = make_float4(t.hi, t.lo, u.hi, u.lo);
      w.dgk[(size_t)set * m.n_params + k] = in ? 2.0 * a : (a > 0.0 ? 2.0 : -2.0);
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) flags[set] = 0;
  __syncthreads();
  const int s1 = min(m.n_samples, (int)(blockIdx.x + 1) * per_block);
  for (int s = blockIdx.x * per_block + threadIdx.x; s < s1; s += kPrepThreads) {
    double f = 1.0, le = 0.0;
    const int j1 = m.smod_start[s + 1];
#pragma unroll 4
    for (int j = m.smod_start[s]; j < j1; ++j) {
      const FactorRec r = m.factor[j];
      if (r.kind == MOD_NORMFACTOR) f *= th[r.param];
      else le = fma(r.b, gk[r.param], fma(r.a, th[r.param], le));
    }
    const double F = le != 0.0 ? f * exp(le) : f;
    w.F[(size_t)set * m.n_samples + s] = F;
    const ff p = as_ff(F);
    w.Ff[(size_t)set * m.n_samples + s] = make_float2(p.hi, p.lo);
  }
}

// Step 2: nu of every (sample, bin) entry, a thread per entry for kSets
// datasets: consecutive threads take consecutive bins of a sample, so its
// histosys coefficients are read coalesced, once for the kSets datasets.
constexpr int kBinnedThreads2 = 128;
template <int kSets>
__global__ void __launch_bounds__(kBinnedThreads2) binned_rates_kernel(const BinnedDev m, const BinnedScratch w,
                                                                       int n_sets) {
  chain_wait();
  const int e = blockIdx.x * kBinnedThreads2 + threadIdx.x;
  if (e >= m.n_entries) return;
  const int set0 = blockIdx.y * kSets;
  const float4* pt[kSets];
#pragma unroll
  for (int t = 0; t < kSets; ++t) pt[t] = w.pt + (size_t)min(set0 + t, n_sets - 1) * m.n_params;
  const int s = m.esample[e], i = e - m.eofs[s], n = m.nb[s], j1 = m.shs_start[s + 1];
  ff shape[kSets];
  const ff nom = ld_pair(m.nominal_f + e);
#pragma unroll
  for (int t = 0; t < kSets; ++t) shape[t] = nom;
#pragma unroll 4
  for (int j = m.shs_start[s]; j < j1; ++j) {
    const int k = __ldg(m.shs_k + j);
    const float2* c = m.coef_f + __ldg(m.shs_ofs + j) + i;
    const ff c0 = ld_pair(c), c1 = ld_pair(c + n);
#pragma unroll
    for (int t = 0; t < kSets; ++t) {
      const float4 q = pt[t][k];
      shape[t] = ff_fma(c1, ff{q.z, q.w}, ff_fma(c0, ff{q.x, q.y}, shape[t]));
    }
  }
#pragma unroll
  for (int t = 0; t < kSets; ++t)
    if (set0 + t < n_sets) {
      const float2 f = w.Ff[(size_t)(set0 + t) * m.n_samples + s];
      const ff v = ff_mul(ff{f.x, f.y}, shape[t]);
      w.nu_e[(size_t)(set0 + t) * m.n_entries + e] = make_float2(v.hi, v.lo);
    }
}

// Step 3: per bin the expected count (samples in order), the weight 1 - n/nu
// and the Poisson term.  sets: null, or the row of counts of each dataset.
__global__ void __launch_bounds__(kBinnedThreads2) binned_bins_kernel(const BinnedDev m, const BinnedScratch w,
                                                                      const int32_t* sets, const double* counts,
                                                                      int32_t* flags) {
  chain_wait();
  const int b = blockIdx.x * kBinnedThreads2 + threadIdx.x, set = blockIdx.y;
  if (b >= m.n_bins) return;
  const double n = counts[(size_t)(sets ? sets[set] : set) * m.n_bins + b];
  const float2* nu_e = w.nu_e + (size_t)set * m.n_entries;
  ff nf = {0.0f, 0.0f};
  const int j1 = m.bin_start[b + 1];
#pragma unroll 4
  for (int j = m.bin_start[b]; j < j1; ++j) {
    const float2 v = nu_e[__ldg(m.bin_entry + j)];
    nf = ff_add(nf, ff{v.x, v.y});
  }
  const double nu = ff_to_double(nf);
  float2 wt = make_float2(0.0f, 0.0f);
  double term = 0.0;
  if (!(nu > 0.0) || !isfinite(nu)) {
    flags[set] = 1;
  } else {
    const ff p = as_ff(1.0 - n / nu);
    wt = make_float2(p.hi, p.lo);
    term = nu - (n != 0.0 ? n * log(nu) : 0.0);
  }
  w.W[(size_t)set * m.n_bins + b] = wt;
  w.term[(size_t)set * m.n_bins + b] = term;
}

// Step 4: per histosys sum_i w (a_i + b_i g') and per sample sum_i w nu_s[i],
// for kSets datasets.  A block takes 32 of them (threads along them, so
// consecutive threads read consecutive coefficients of the transposed layout)
// times four quarters of the sample's bins (one chain of dependent
// multiply-adds a quarter as long), added in order at the end; a warp's
// weights are those of one or two samples.
constexpr int kQuarters = kBinnedThreads2 / 32;
template <int kSets>
__global__ void __launch_bounds__(kBinnedThreads2) binned_sums_kernel(const BinnedDev m, const BinnedScratch w,
                                                                      int n_sets) {
  __shared__ float4 part[kQuarters - 1][kSets][32];
  chain_wait();
  const int lane = threadIdx.x & 31, quarter = threadIdx.x >> 5, set0 = blockIdx.y * kSets;
  const int id = blockIdx.x * 32 + lane, s = id < m.n_hs ? m.g_sample[id] : id - m.n_hs;
  const bool hs = id < m.n_hs, any = s < m.n_samples;
  ff ta[kSets], tb[kSets];
#pragma unroll
  for (int t = 0; t < kSets; ++t) ta[t] = tb[t] = {0.0f, 0.0f};
  if (any) {
    const int nbs = m.nb[s], i0 = nbs * quarter / kQuarters, i1 = nbs * (quarter + 1) / kQuarters;
    const float2* W[kSets];
#pragma unroll
    for (int t = 0; t < kSets; ++t) W[t] = w.W + (size_t)min(set0 + t, n_sets - 1) * m.n_bins + m.bin0[s];
    if (hs) {
      const int j0 = m.shs_start[s], nh = m.shs_start[s + 1] - j0;
      const float2* ca = m.coef_af + m.tbase[s] + (id - j0);
      const float2* cb = m.coef_bf + m.tbase[s] + (id - j0);
#pragma unroll 4
      for (int i = i0; i < i1; ++i) {
        const ff a = ld_pair(ca + (size_t)i * nh), b = ld_pair(cb + (size_t)i * nh);
#pragma unroll
        for (int t = 0; t < kSets; ++t) {
          const float2 v = W[t][i];
          ff_acc_mul(ta[t], ff{v.x, v.y}, a);
          ff_acc_mul(tb[t], ff{v.x, v.y}, b);
        }
      }
    } else {
      const float2* nu[kSets];
#pragma unroll
      for (int t = 0; t < kSets; ++t) nu[t] = w.nu_e + (size_t)min(set0 + t, n_sets - 1) * m.n_entries + m.eofs[s];
#pragma unroll 4
      for (int i = i0; i < i1; ++i)
#pragma unroll
        for (int t = 0; t < kSets; ++t) {
          const float2 v = W[t][i], e = nu[t][i];
          ff_acc_mul(ta[t], ff{v.x, v.y}, ff{e.x, e.y});
        }
    }
  }
  if (quarter > 0)
#pragma unroll
    for (int t = 0; t < kSets; ++t) part[quarter - 1][t][lane] = make_float4(ta[t].hi, ta[t].lo, tb[t].hi, tb[t].lo);
  __syncthreads();
  if (quarter > 0 || !any) return;
#pragma unroll
  for (int t = 0; t < kSets; ++t) {
    if (set0 + t >= n_sets) break;
    for (int q = 0; q < kQuarters - 1; ++q) {
      const float4 v = part[q][t][lane];
      ta[t] = ff_add(ta[t], ff{v.x, v.y});
      tb[t] = ff_add(tb[t], ff{v.z, v.w});
    }
    if (hs)
      w.T[(size_t)(set0 + t) * m.n_hs + m.shs[id]] =
          fma(w.dgk[(size_t)(set0 + t) * m.n_params + m.shs_k[id]], ff_to_double(tb[t]), ff_to_double(ta[t]));
    else
      w.Ssum[(size_t)(set0 + t) * m.n_samples + s] = ff_to_double(ta[t]);
  }
}

// Step 5: out[set] = NLL, then gradient.  Block (0, set): the bins' terms and
// the constraints summed, each by thread-strided sums and a fixed tree; the
// others 16 parameters each, eight lanes a parameter: its modifiers lane by
// lane, the lanes by butterfly, then its constraint.
constexpr int kGradThreads = 128, kGradLanes = 8, kGradPer = kGradThreads / kGradLanes;
// Out of line: inlined, every warp would divide (an FP64 division on each of
// them takes as long as the kernel) and select.
__device__ __noinline__ double divided(double x, double a) { return x / a; }
__global__ void __launch_bounds__(kGradThreads) binned_grad_kernel(const BinnedDev m, const BinnedScratch w,
                                                                   const double* theta, double* out,
                                                                   const int32_t* flags) {
  chain_wait();
  const int set = blockIdx.y, tid = threadIdx.x;
  const double* th = theta + (size_t)set * m.n_params;
  double* o = out + (size_t)set * (1 + m.n_params);
  if (blockIdx.x == 0) {
    __shared__ double red[kGradThreads];
    const double* term = w.term + (size_t)set * m.n_bins;
    double t = 0.0, c = 0.0;
#pragma unroll 4
    for (int b = tid; b < m.n_bins; b += kGradThreads) t += term[b];
    for (int k = tid; k < m.n_params; k += kGradThreads)
      if (m.constrained[k]) c = fma(0.5 * th[k], th[k], c);
    red[tid] = t + c;
    for (int d = kGradThreads / 2; d > 0; d >>= 1) {
      __syncthreads();
      if (tid < d) red[tid] += red[tid + d];
    }
    if (tid == 0) o[0] = flags[set] ? INFINITY : red[0];
    return;
  }
  const int k = (blockIdx.x - 1) * kGradPer + tid / kGradLanes, l = tid % kGradLanes;
  double g = 0.0, a = 0.0;
  if (k < m.n_params) {
    const double* F = w.F + (size_t)set * m.n_samples;
    const double* S = w.Ssum + (size_t)set * m.n_samples;
    const double* T = w.T + (size_t)set * m.n_hs;
    a = th[k];
    const double dg = w.dgk[(size_t)set * m.n_params + k];
    const int j0 = m.pmod_norm[k], j1 = m.pmod_start[k + 1];
    // the normfactors' sums, divided by a once
    for (int j = m.pmod_start[k] + l; j < j0; j += kGradLanes) g += S[m.grad[j].sample];
    if (m.pmod_start[k] + l < j0) g = divided(g, a);
#pragma unroll 4
    for (int j = j0 + l; j < j1; j += kGradLanes) {
      const GradRec r = m.grad[j];
      const bool hs = r.kind == MOD_HISTOSYS;
      g = fma(hs ? F[r.sample] : S[r.sample], hs ? T[r.hs] : fma(r.b, dg, r.a), g);
    }
  }
#pragma unroll
  for (int d = kGradLanes / 2; d > 0; d >>= 1) g += __shfl_xor_sync(0xffffffffu, g, d);
  if (k < m.n_params && l == 0) o[1 + k] = m.constrained[k] ? g + a : g;
}

// Expected counts nu_b per dataset (for generating toys).
__global__ void __launch_bounds__(kBinnedThreads) binned_expected_kernel(const BinnedDev m, int n_sets,
                                                                          const double* theta, double* nu_out,
                                                                          double* scratch) {
  extern __shared__ double smem[];
  double* th = smem;
  double* F = th + m.n_params;
  double* gk = F + m.n_samples;
  double* nu_e = scratch + (size_t)blockIdx.x * m.n_entries;
  for (int set = blockIdx.x; set < n_sets; set += gridDim.x) {
    sample_factors(m, theta + (size_t)set * m.n_params, th, gk, F);
    entry_rates(m, th, gk, F, nu_e);
    __syncthreads();
    for (int b = threadIdx.x; b < m.n_bins; b += kBinnedThreads) {
      double nu = 0.0;
      for (int j = m.bin_start[b]; j < m.bin_start[b + 1]; ++j) nu += nu_e[m.bin_entry[j]];
      nu_out[(size_t)set * m.n_bins + b] = nu;
    }
    __syncthreads();
  }
}

}  // namespace

}  // namespace rf

// ---------------------------------------------------------------- handle

struct rf_binned {
  int32_t n_bins = 0, n_samples = 0, n_params = 0, n_mods = 0, n_entries = 0, n_hs = 0;
  rf::DevBuf bin0, nb, eofs, esample, nominal, smod_start, shs_start, shs, coef, tbase, g_sample,
      bin_start, bin_entry, pmod_start, pmod_norm, constrained, nominal_f, coef_f, coef_af, coef_bf, shs_k, shs_ofs, factor, grad;
  rf::DevBuf counts, theta, out, flags, sets, io;
  rf::GrowBuf work, scratch;  // intermediate results of the passes, of the expected counts
  rf::HostBuf h_out, h_flags, h_theta, h_sets, h_io;
  rf::BinnedDev dev{};
  rf::BinnedScratch ws{};
  int grid = 0;  // most blocks of the expected-counts kernel
  int cap = 0;   // datasets a pass takes at once: those that `work` has room for
  size_t smem = 0;
};

using namespace rf;

namespace {

template <class T>
bool upload(DevBuf& b, const std::vector<T>& v) {
  if (!b.ensure(sizeof(T) * std::max<size_t>(1, v.size()))) return false;
  return v.empty() || cuda_ok(cudaMemcpy(b.p, v.data(), sizeof(T) * v.size(), cudaMemcpyHostToDevice), "binned upload");
}

// Launches a kernel that begins with chain_wait(), as a programmatic dependent
// of the stream's previous kernel.
template <class... Params, class... Args>
void launch_chained(void (*kernel)(Params...), dim3 grid, int threads, size_t smem, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  note_launches(1, st);
  cudaLaunchKernelEx(&cfg, kernel, args...);
}

// Bytes of a dataset's intermediate results.
size_t work_per_set(const rf_binned* m) {
  return 24 * (size_t)std::max(1, m->n_params) + 24 * (size_t)m->n_samples + 8 * (size_t)m->n_entries +
         16 * (size_t)m->n_bins + 8 * (size_t)std::max(1, m->n_hs);
}

// Room for the intermediate results of n datasets, of 256 MB or 32768 (a
// grid's second dimension) at most, one at least (n <= 0: of the datasets that
// 8 MB hold).  A group costs five launches: 4096 datasets of a one-channel
// model in four groups 461 us, in one 293.  A model starts with
// 8 MB (50 datasets of the 28-channel model, whose 160 MB for 1024 would lie
// idle beside models that only see a few) and grows to what a call has, at
// least twofold.  Without memory a call goes on in groups of `cap`.
bool reserve_sets(rf_binned* m, int n) {
  const size_t per_set = work_per_set(m);
  const auto held = [&](size_t bytes) { return (int)std::max<size_t>(1, std::min<size_t>(32768, bytes / per_set)); };
  const int most = held((size_t)256 << 20);
  if (m->cap > 0 && std::min(n, most) <= m->cap) return true;
  const int cap = std::min(most, n > 0 ? std::max(n, 2 * m->cap) : held((size_t)8 << 20));
  if (!m->work.ensure(per_set * (size_t)cap)) return false;
  m->cap = cap;
  char* p = (char*)m->work.p;  // (16-byte items first)
  auto take = [&](size_t bytes) {
    char* q = p;
    p += bytes * (size_t)cap;
    return (void*)q;
  };
  const size_t P = (size_t)std::max(1, m->n_params), S = (size_t)m->n_samples, E = (size_t)m->n_entries,
               B = (size_t)m->n_bins, H = (size_t)std::max(1, m->n_hs);
  m->ws.pt = (float4*)take(16 * P);
  m->ws.dgk = (double*)take(8 * P);
  m->ws.F = (double*)take(8 * S);
  m->ws.Ssum = (double*)take(8 * S);
  m->ws.Ff = (float2*)take(8 * S);
  m->ws.nu_e = (float2*)take(8 * E);
  m->ws.W = (float2*)take(8 * B);
  m->ws.term = (double*)take(8 * B);
  m->ws.T = (double*)take(8 * H);
  return true;
}

rf_status launch_binned(rf_binned* m, int32_t n_sets, const double* d_counts, const double* d_theta, double* d_out,
                        int32_t* d_flags, cudaStream_t st, const int32_t* d_sets = nullptr) {
  const BinnedDev& D = m->dev;
  const int P = D.n_params;
  reserve_sets(m, n_sets);
  for (int s0 = 0; s0 < n_sets; s0 += m->cap) {
    const int n = std::min(n_sets - s0, m->cap);
    const double* th = d_theta + (size_t)s0 * P;
    const double* counts = d_sets ? d_counts : d_counts + (size_t)s0 * D.n_bins;
    const int32_t* sets = d_sets ? d_sets + s0 : nullptr;
    double* out = d_out + (size_t)s0 * (1 + P);
    int32_t* flags = d_flags + s0;
    // samples per block of step 1: 32 while that leaves SMs free (each block
    // repeats the parameters' part), else a block per dataset
    const int per_block = (int64_t)n * ((D.n_samples + 31) / 32) <= 2 * sm_count() ? 32 : D.n_samples;
    auto blocks = [](int work, int threads) { return (unsigned)((work + threads - 1) / threads); };
    launch_chained(binned_prep_kernel, dim3(blocks(D.n_samples, per_block), n), kPrepThreads,
                   2 * sizeof(double) * (size_t)P, st, D, m->ws, th, per_block, flags);
    // four datasets a thread (one load of a coefficient for the four) once the
    // blocks still fill the GPU at that; one at a time else
    const dim3 ge(blocks(D.n_entries, kBinnedThreads2)), gs(blocks(D.n_hs + D.n_samples, 32));
    const bool four = (int64_t)ge.x * n >= 32 * (int64_t)sm_count();
    const unsigned ny = four ? blocks(n, 4) : (unsigned)n;
    launch_chained(four ? binned_rates_kernel<4> : binned_rates_kernel<1>, dim3(ge.x, ny), kBinnedThreads2, 0, st, D,
                   m->ws, n);
    launch_chained(binned_bins_kernel, dim3(blocks(D.n_bins, kBinnedThreads2), n), kBinnedThreads2, 0, st, D, m->ws,
                   sets, counts, flags);
    launch_chained(four ? binned_sums_kernel<4> : binned_sums_kernel<1>, dim3(gs.x, ny), kBinnedThreads2, 0, st, D,
                   m->ws, n);
    launch_chained(binned_grad_kernel, dim3(1 + blocks(P, kGradPer), n), kGradThreads, 0, st, D, m->ws, th, out,
                   (const int32_t*)flags);
  }
  return cuda_ok(cudaGetLastError(), "binned launch") ? RF_OK : RF_E_CUDA;
}

}  // namespace

extern "C" {

rf_status rf_binned_create(int32_t n_bins, int32_t n_samples, const int32_t* bin0, const int32_t* nbins,
                           const double* nominal, int32_t n_params, const int32_t* constrained, int32_t n_mods,
                           const rf_modifier* mods, const double* hist_data, rf_binned** out) {
  if (!out || n_bins < 1 || n_bins > kMaxBinnedBins || n_samples < 1 || n_samples > kMaxBinnedSamples ||
      n_params < 0 || n_mods < 0 || !bin0 || !nbins || !nominal || (n_params > 0 && !constrained) ||
      (n_mods > 0 && !mods)) {
    set_error("rf_binned_create: bad argument (1 <= bins <= 8192, 1 <= samples <= 2048)");
    return RF_E_INVALID;
  }
  *out = nullptr;
  std::vector<int32_t> eofs(n_samples), esample;
  int64_t total = 0;
  for (int s = 0; s < n_samples; ++s) {
    if (nbins[s] < 1 || bin0[s] < 0 || bin0[s] + nbins[s] > n_bins) {
      set_error("rf_binned_create: a sample's bins lie outside the model's bins");
      return RF_E_INVALID;
    }
    eofs[s] = (int32_t)total;
    total += nbins[s];
    for (int i = 0; i < nbins[s]; ++i) esample.push_back(s);
  }
  if (total > (int64_t)1 << 30) {
    set_error("rf_binned_create: too many (sample, bin) entries");
    return RF_E_INVALID;
  }
  std::vector<int32_t> kind(n_mods), param(n_mods), msample(n_mods), mhs(n_mods, -1);
  std::vector<double> ns_a(n_mods, 0.0), ns_b(n_mods, 0.0);
  std::vector<int32_t> hs_param;
  std::vector<int64_t> hs_ofs;
  std::vector<double> coef;
  int64_t hd = 0;
  for (int j = 0; j < n_mods; ++j) {
    const rf_modifier& md = mods[j];
    if (md.sample < 0 || md.sample >= n_samples || md.param < 0 || md.param >= n_params || md.kind < 0 ||
        md.kind > 2) {
      set_error("rf_binned_create: bad modifier");
      return RF_E_INVALID;
    }
    if (md.kind == RF_MOD_NORMSYS && !(md.k_lo > 0.0 && md.k_hi > 0.0)) {
      set_error("rf_binned_create: normsys factors must be positive");
      return RF_E_INVALID;
    }
    kind[j] = md.kind;
    param[j] = md.param;
    msample[j] = md.sample;
    if (md.kind == RF_MOD_NORMSYS) {
      ns_a[j] = 0.5 * (std::log(md.k_hi) - std::log(md.k_lo));
      ns_b[j] = 0.5 * (std::log(md.k_hi) + std::log(md.k_lo));
    }
    if (md.kind == RF_MOD_HISTOSYS) {
      if (!hist_data) {
        set_error("rf_binned_create: histosys modifiers need hist_data");
        return RF_E_INVALID;
      }
      const int n = nbins[md.sample];
      const double* h = nominal + eofs[md.sample];
      const double *lo = hist_data + hd, *hi = hist_data + hd + n;
      mhs[j] = (int32_t)hs_param.size();
      hs_param.push_back(md.param);
      hs_ofs.push_back((int64_t)coef.size());
      for (int i = 0; i < n; ++i) coef.push_back(0.5 * (hi[i] - lo[i]));
      for (int i = 0; i < n; ++i) coef.push_back(0.5 * (hi[i] + lo[i]) - h[i]);
      hd += 2 * (int64_t)n;
    }
  }
  const int n_hs = (int)hs_param.size();
  // CSR lists: factor modifiers and histosys per sample, modifiers per
  // parameter (modifier order), the entries of each bin (sample order).
  std::vector<int32_t> smod_start(n_samples + 1, 0), shs_start(n_samples + 1, 0), pmod_start(n_params + 1, 0),
      pmod_norm(n_params);
  for (int j = 0; j < n_mods; ++j) {
    (kind[j] == RF_MOD_HISTOSYS ? shs_start : smod_start)[msample[j] + 1]++;
    pmod_start[param[j] + 1]++;
  }
  for (int s = 0; s < n_samples; ++s) {
    smod_start[s + 1] += smod_start[s];
    shs_start[s + 1] += shs_start[s];
  }
  for (int k = 0; k < n_params; ++k) pmod_start[k + 1] += pmod_start[k];
  std::vector<int32_t> smod(smod_start[n_samples]), shs(shs_start[n_samples]), pmod(n_mods);
  std::vector<int32_t> sfill(smod_start.begin(), smod_start.end() - 1), hfill(shs_start.begin(), shs_start.end() - 1),
      pfill(pmod_start.begin(), pmod_start.end() - 1);
  for (int j = 0; j < n_mods; ++j) {
    if (kind[j] == RF_MOD_HISTOSYS) shs[hfill[msample[j]]++] = mhs[j];
    else smod[sfill[msample[j]]++] = j;
    pmod[pfill[param[j]]++] = j;
  }
  for (int k = 0; k < n_params; ++k)
    pmod_norm[k] = (int32_t)(std::stable_partition(pmod.begin() + pmod_start[k], pmod.begin() + pmod_start[k + 1],
                                                   [&](int32_t j) { return kind[j] == RF_MOD_NORMFACTOR; }) -
                             pmod.begin());
  // transposed coefficients per sample
  std::vector<int64_t> tbase(n_samples);
  std::vector<int32_t> g_sample(shs.size());
  std::vector<double> coef_a, coef_b;
  for (int s = 0; s < n_samples; ++s) {
    const int nh = shs_start[s + 1] - shs_start[s], n = nbins[s];
    tbase[s] = (int64_t)coef_a.size();
    for (int g = shs_start[s]; g < shs_start[s + 1]; ++g) g_sample[g] = s;
    for (int i = 0; i < n; ++i)
      for (int j = 0; j < nh; ++j) {
        const int h = shs[shs_start[s] + j];
        coef_a.push_back(coef[hs_ofs[h] + i]);
        coef_b.push_back(coef[hs_ofs[h] + n + i]);
      }
  }
  std::vector<int32_t> bin_start(n_bins + 1, 0);
  for (int s = 0; s < n_samples; ++s)
    for (int i = 0; i < nbins[s]; ++i) bin_start[bin0[s] + i + 1]++;
  for (int b = 0; b < n_bins; ++b) bin_start[b + 1] += bin_start[b];
  std::vector<int32_t> bin_entry(bin_start[n_bins]);
  std::vector<int32_t> bfill(bin_start.begin(), bin_start.end() - 1);
  for (int s = 0; s < n_samples; ++s)
    for (int i = 0; i < nbins[s]; ++i) bin_entry[bfill[bin0[s] + i]++] = eofs[s] + i;

  rf_binned* m = new (std::nothrow) rf_binned();
  if (!m) return RF_E_OOM;
  m->n_bins = n_bins;
  m->n_samples = n_samples;
  m->n_params = n_params;
  m->n_mods = n_mods;
  m->n_entries = (int32_t)total;
  m->n_hs = n_hs;
  const std::vector<int32_t> vb0(bin0, bin0 + n_samples), vnb(nbins, nbins + n_samples);
  const std::vector<double> vnom(nominal, nominal + total);
  std::vector<int32_t> vcon(n_params);
  for (int k = 0; k < n_params; ++k) vcon[k] = constrained[k] ? 1 : 0;
  std::vector<int32_t> shs_k(shs.size());
  std::vector<int64_t> shs_ofs(shs.size());
  for (size_t j = 0; j < shs.size(); ++j) {
    shs_k[j] = hs_param[shs[j]];
    shs_ofs[j] = hs_ofs[shs[j]];
  }
  // float-pair copies: hi = the float nearest v, lo = the float nearest v - hi
  std::vector<FactorRec> factor(smod.size());
  for (size_t j = 0; j < smod.size(); ++j) factor[j] = FactorRec{param[smod[j]], kind[smod[j]], ns_a[smod[j]], ns_b[smod[j]]};
  std::vector<GradRec> grad(pmod.size());
  for (size_t j = 0; j < pmod.size(); ++j) {
    const int md = pmod[j];
    grad[j] = GradRec{kind[md], msample[md], mhs[md], 0, ns_a[md], ns_b[md]};
  }
  auto pairs = [](const std::vector<double>& v) {
    std::vector<float2> f(v.size());
    for (size_t i = 0; i < v.size(); ++i) {
      const float h = (float)v[i];
      f[i] = make_float2(h, (float)(v[i] - (double)h));
    }
    return f;
  };
  const bool ok = upload(m->factor, factor) && upload(m->grad, grad) && upload(m->shs_k, shs_k) &&
                  upload(m->shs_ofs, shs_ofs) && upload(m->nominal_f, pairs(vnom)) && upload(m->coef_f, pairs(coef)) &&
                  upload(m->coef_af, pairs(coef_a)) && upload(m->coef_bf, pairs(coef_b)) &&
                  upload(m->bin0, vb0) && upload(m->nb, vnb) && upload(m->eofs, eofs) && upload(m->esample, esample) &&
                  upload(m->nominal, vnom) && upload(m->smod_start, smod_start) && upload(m->shs_start, shs_start) &&
                  upload(m->shs, shs) &&
                  upload(m->coef, coef) && upload(m->tbase, tbase) && upload(m->g_sample, g_sample) &&
                  upload(m->bin_start, bin_start) && upload(m->bin_entry, bin_entry) &&
                  upload(m->pmod_start, pmod_start) && upload(m->pmod_norm, pmod_norm) && upload(m->constrained, vcon);
  m->smem = binned_smem(n_params, n_samples, n_bins);
  int dev_id = 0, max_optin = 0;
  cudaGetDevice(&dev_id);
  cudaDeviceGetAttribute(&max_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev_id);
  // The attribute is the kernel's, for every model in the process: once the
  // device's maximum, not this model's size (a smaller model created later
  // took a larger one's launches away).
  if (m->smem > (size_t)max_optin ||
      !cuda_ok(cudaFuncSetAttribute(binned_prep_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, max_optin),
               "binned smem") ||
      !cuda_ok(cudaFuncSetAttribute(binned_expected_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, max_optin),
               "binned smem")) {
    delete m;
    set_error("rf_binned_create: the model needs more shared memory than a block has");
    return RF_E_INVALID;
  }
  int per_sm = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, binned_expected_kernel, kBinnedThreads, m->smem);
  m->grid = sm_count() * std::max(1, per_sm);
  if (!ok || !m->scratch.ensure(sizeof(double) * (size_t)total) || !reserve_sets(m, 0)) {
    delete m;
    return RF_E_OOM;
  }
  BinnedDev& D = m->dev;
  D.n_bins = n_bins;
  D.n_samples = n_samples;
  D.n_params = n_params;
  D.n_mods = n_mods;
  D.n_entries = m->n_entries;
  D.n_hs = n_hs;
  D.bin0 = (const int32_t*)m->bin0.p;
  D.nb = (const int32_t*)m->nb.p;
  D.eofs = (const int32_t*)m->eofs.p;
  D.esample = (const int32_t*)m->esample.p;
  D.nominal = (const double*)m->nominal.p;
  D.smod_start = (const int32_t*)m->smod_start.p;
  D.shs_start = (const int32_t*)m->shs_start.p;
  D.shs = (const int32_t*)m->shs.p;
  D.coef = (const double*)m->coef.p;
  D.tbase = (const int64_t*)m->tbase.p;
  D.g_sample = (const int32_t*)m->g_sample.p;
  D.nominal_f = (const float2*)m->nominal_f.p;
  D.shs_k = (const int32_t*)m->shs_k.p;
  D.shs_ofs = (const int64_t*)m->shs_ofs.p;
  D.coef_f = (const float2*)m->coef_f.p;
  D.coef_af = (const float2*)m->coef_af.p;
  D.coef_bf = (const float2*)m->coef_bf.p;
  D.bin_start = (const int32_t*)m->bin_start.p;
  D.bin_entry = (const int32_t*)m->bin_entry.p;
  D.pmod_start = (const int32_t*)m->pmod_start.p;
  D.pmod_norm = (const int32_t*)m->pmod_norm.p;
  D.constrained = (const int32_t*)m->constrained.p;
  D.factor = (const FactorRec*)m->factor.p;
  D.grad = (const GradRec*)m->grad.p;
  *out = m;
  return RF_OK;
}

void rf_binned_destroy(rf_binned* m) { delete m; }

int32_t rf_binned_n_params(const rf_binned* m) { return m ? m->n_params : 0; }

rf_status rf_binned_nll_grad_async(rf_binned* m, int32_t n_sets, const double* d_counts, const double* d_theta,
                                   double* d_out, int32_t* d_flags, void* stream) {
  if (!m || n_sets < 0 || (n_sets > 0 && (!d_counts || !d_theta || !d_out || !d_flags))) {
    set_error("rf_binned_nll_grad_async: bad argument");
    return RF_E_INVALID;
  }
  return launch_binned(m, n_sets, d_counts, d_theta, d_out, d_flags, (cudaStream_t)stream);
}

// Up to this many bytes of counts, parameters and results (17 datasets of 1400
// bins and 256 parameters) a host call goes through one pinned buffer: one dataset of
// 1400 bins and 256 parameters 76 -> 58 us.
constexpr size_t kStagedBytes = size_t(256) << 10;

// A host call's results: NLL and gradient by dataset from `o`, the status
// from the datasets' flags.
static rf_status read_results(int32_t n_sets, int P, const double* o, const int32_t* f, double* nll, double* grad) {
  rf_status st = RF_OK;
  for (int t = 0; t < n_sets; ++t) {
    nll[t] = o[(size_t)t * (1 + P)];
    for (int k = 0; k < P; ++k) grad[(size_t)t * P + k] = o[(size_t)t * (1 + P) + 1 + k];
    if (f[t]) st = RF_E_DOMAIN;
  }
  if (st == RF_E_DOMAIN) set_error("expected count <= 0 in some bin");
  return st;
}

rf_status rf_binned_nll_grad(rf_binned* m, int32_t n_sets, const double* counts, const double* theta, double* nll,
                             double* grad) {
  if (!m || n_sets < 0 || (n_sets > 0 && (!counts || !theta || !nll || !grad))) {
    set_error("rf_binned_nll_grad: bad argument");
    return RF_E_INVALID;
  }
  if (n_sets == 0) return RF_OK;
  const int P = m->n_params, B = m->n_bins;
  const size_t n_in = (size_t)n_sets * (B + P), n_out = (size_t)n_sets * (1 + P);
  if (sizeof(double) * (n_in + n_out) <= kStagedBytes) {
    // Small calls: inputs and results side by side in pinned and in device
    // memory, one copy each way on the stream and one wait, where the four
    // copies of the larger ones wait each for themselves.
    const size_t bytes_in = sizeof(double) * n_in, bytes_out = sizeof(double) * n_out + sizeof(int32_t) * n_sets;
    if (!m->io.ensure(bytes_in + bytes_out) || !m->h_io.ensure(bytes_in + bytes_out)) return RF_E_OOM;
    double *h = (double*)m->h_io.p, *dev = (double*)m->io.p;
    std::memcpy(h, counts, sizeof(double) * (size_t)n_sets * B);
    std::memcpy(h + (size_t)n_sets * B, theta, sizeof(double) * (size_t)n_sets * P);
    if (!cuda_ok(cudaMemcpyAsync(dev, h, bytes_in, cudaMemcpyHostToDevice, nullptr), "binned")) return RF_E_CUDA;
    const rf_status s = launch_binned(m, n_sets, dev, dev + (size_t)n_sets * B, dev + n_in, (int32_t*)(dev + n_in + n_out), nullptr);
    if (s != RF_OK) return s;
    if (!cuda_ok(cudaMemcpyAsync(h + n_in, dev + n_in, bytes_out, cudaMemcpyDeviceToHost, nullptr), "binned") ||
        !cuda_ok(cudaStreamSynchronize(nullptr), "binned"))
      return RF_E_CUDA;
    return read_results(n_sets, P, h + n_in, (const int32_t*)(h + n_in + n_out), nll, grad);
  }
  if (!m->counts.ensure(sizeof(double) * (size_t)n_sets * B) ||
      !m->theta.ensure(sizeof(double) * (size_t)n_sets * std::max(P, 1)) ||
      !m->out.ensure(sizeof(double) * (size_t)n_sets * (1 + P)) || !m->flags.ensure(sizeof(int32_t) * n_sets) ||
      !m->h_out.ensure(sizeof(double) * (size_t)n_sets * (1 + P)) || !m->h_flags.ensure(sizeof(int32_t) * n_sets))
    return RF_E_OOM;
  if (!cuda_ok(cudaMemcpy(m->counts.p, counts, sizeof(double) * (size_t)n_sets * B, cudaMemcpyHostToDevice), "binned") ||
      (P > 0 && !cuda_ok(cudaMemcpy(m->theta.p, theta, sizeof(double) * (size_t)n_sets * P, cudaMemcpyHostToDevice),
                         "binned")))
    return RF_E_CUDA;
  rf_status s = launch_binned(m, n_sets, (const double*)m->counts.p, (const double*)m->theta.p, (double*)m->out.p,
                              (int32_t*)m->flags.p, nullptr);
  if (s != RF_OK) return s;
  if (!cuda_ok(cudaMemcpy(m->h_out.p, m->out.p, sizeof(double) * (size_t)n_sets * (1 + P), cudaMemcpyDeviceToHost),
               "binned") ||
      !cuda_ok(cudaMemcpy(m->h_flags.p, m->flags.p, sizeof(int32_t) * n_sets, cudaMemcpyDeviceToHost), "binned"))
    return RF_E_CUDA;
  return read_results(n_sets, P, (const double*)m->h_out.p, (const int32_t*)m->h_flags.p, nll, grad);
}

rf_status rf_binned_expected(rf_binned* m, int32_t n_sets, const double* d_theta, double* d_nu, void* stream) {
  if (!m || n_sets < 0 || (n_sets > 0 && (!d_theta || !d_nu))) {
    set_error("rf_binned_expected: bad argument");
    return RF_E_INVALID;
  }
  if (n_sets == 0) return RF_OK;
  // A block's entry rates are n_entries doubles; without memory for all blocks,
  // as many as there is room for.
  const size_t per_block = sizeof(double) * (size_t)m->n_entries;
  int grid = std::min(n_sets, m->grid);
  if (m->scratch.bytes < per_block * (size_t)grid)
    m->scratch.ensure(per_block * std::min((size_t)m->grid, std::max((size_t)grid, 2 * m->scratch.bytes / per_block)));
  grid = (int)std::min((size_t)grid, m->scratch.bytes / per_block);
  note_launches(1, (cudaStream_t)stream);
  binned_expected_kernel<<<grid, kBinnedThreads, m->smem, (cudaStream_t)stream>>>(m->dev, n_sets, d_theta, d_nu,
                                                                                  (double*)m->scratch.p);
  return cuda_ok(cudaGetLastError(), "binned launch") ? RF_OK : RF_E_CUDA;
}

rf_status rf_binned_fit(rf_binned* m, int32_t n_sets, const double* counts, const double* theta0, const double* lo,
                        const double* hi, const rf_fit_opts* opts, double* theta_hat, double* nll_min, double* cov,
                        int32_t* n_evals, int32_t* fit_status) {
  if (!m || n_sets < 0 || (n_sets > 0 && (!counts || !theta0 || !lo || !hi || !theta_hat || !nll_min || !n_evals ||
                                          !fit_status))) {
    set_error("rf_binned_fit: bad argument");
    return RF_E_INVALID;
  }
  if (n_sets == 0) return RF_OK;
  const int P = m->n_params, B = m->n_bins, S = n_sets;
  const double tol = (opts && opts->tol_edm > 0.0) ? opts->tol_edm : 1e-7;
  const int max_evals = (opts && opts->max_evals > 0) ? opts->max_evals : 1000;
  const bool want_cov = opts && opts->want_cov && cov;
  if (!m->counts.ensure(sizeof(double) * (size_t)S * B) || !m->theta.ensure(sizeof(double) * (size_t)S * std::max(P, 1)) ||
      !m->out.ensure(sizeof(double) * (size_t)S * (1 + P)) || !m->flags.ensure(sizeof(int32_t) * S) ||
      !m->sets.ensure(sizeof(int32_t) * S) || !m->h_out.ensure(sizeof(double) * (size_t)S * (1 + P)) ||
      !m->h_theta.ensure(sizeof(double) * (size_t)S * std::max(P, 1)) || !m->h_sets.ensure(sizeof(int32_t) * S))
    return RF_E_OOM;
  if (!cuda_ok(cudaMemcpy(m->counts.p, counts, sizeof(double) * (size_t)S * B, cudaMemcpyHostToDevice), "binned fit"))
    return RF_E_CUDA;
  cudaStream_t st = nullptr;
  // One round: the active sets' points packed, one launch, results scattered.
  auto eval = [&](const std::vector<int32_t>& active, std::vector<double>& th, std::vector<double>& nll,
                  std::vector<double>& grad) -> rf_status {
    const int n = (int)active.size();
    double* ht = (double*)m->h_theta.p;
    int32_t* hs = (int32_t*)m->h_sets.p;
    for (int a = 0; a < n; ++a) {
      hs[a] = active[a];
      std::memcpy(ht + (size_t)a * P, &th[(size_t)active[a] * P], sizeof(double) * P);
    }
    if (!cuda_ok(cudaMemcpyAsync(m->theta.p, ht, sizeof(double) * (size_t)n * P, cudaMemcpyHostToDevice, st),
                 "binned fit") ||
        !cuda_ok(cudaMemcpyAsync(m->sets.p, hs, sizeof(int32_t) * n, cudaMemcpyHostToDevice, st), "binned fit"))
      return RF_E_CUDA;
    const rf_status r = launch_binned(m, n, (const double*)m->counts.p, (const double*)m->theta.p, (double*)m->out.p,
                                      (int32_t*)m->flags.p, st, (const int32_t*)m->sets.p);
    if (r != RF_OK) return r;
    if (!cuda_ok(cudaMemcpyAsync(m->h_out.p, m->out.p, sizeof(double) * (size_t)n * (1 + P), cudaMemcpyDeviceToHost,
                                 st),
                 "binned fit") ||
        !cuda_ok(cudaStreamSynchronize(st), "binned fit"))
      return RF_E_CUDA;
    const double* o = (const double*)m->h_out.p;
    for (int a = 0; a < n; ++a) {
      const int s = active[a];
      nll[s] = o[(size_t)a * (1 + P)];
      for (int k = 0; k < P; ++k) grad[(size_t)s * P + k] = o[(size_t)a * (1 + P) + 1 + k];
    }
    return RF_OK;
  };
  return fit_batch(S, P, lo, hi, theta0, tol, max_evals, want_cov, eval, nullptr, theta_hat, nll_min,
                   want_cov ? cov : nullptr, n_evals, fit_status);
}

}  // extern "C"
