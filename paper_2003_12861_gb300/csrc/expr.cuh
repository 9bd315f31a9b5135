// RF_EXPR leaves on the device: a density given as a short postfix program
// over the observable x, the node's parameters and constants, for PDFs that
// have no built-in kind (Sec. 5: a fall-back implementation for PDFs that
// have not been given batch code).  The generic graph interpreter evaluates
// it per event; its normalisation integral and the integral's parameter
// derivatives are computed per parameter point by adaptive Gauss-Kronrod
// quadrature, cooperatively by the parameter-point kernel's block.
#pragma once

#include <cuda_runtime.h>

#include "fp64_math.cuh"
#include "rf_internal.h"

namespace rf {

__device__ __forceinline__ bool not_finite(double v) {
  return (__double2hiint(v) & 0x7ff00000) == 0x7ff00000;
}

// Quotients t / b by one reciprocal: q = t y corrected by its residual
// (Markstein, IBM J. Res. Dev. 34 (1990)), y = 1 / b rounded.  Operands whose
// quotient or residual could leave the normal range are divided as they are.
struct Divisor {
  double b, y;
  bool plain;
};
__device__ __forceinline__ Divisor divisor(double b) {
  const int e = (__double2hiint(b) >> 20) & 0x7ff;
  Divisor d{b, 0.0, e < 1023 - 400 || e > 1023 + 400};
  if (!d.plain) d.y = 1.0 / b;
  return d;
}
__device__ __forceinline__ double quotient(double t, const Divisor& d) {
  const int e = (__double2hiint(t) >> 20) & 0x7ff;
  if (d.plain || e < 1023 - 400 || e > 1023 + 400) return t / d.b;
  const double q = t * d.y;
  return fma(fma(-q, d.b, t), d.y, q);
}

// The program's value at x and, for kDeriv, its derivatives in the node's
// parameters (forward mode), df[0..n_par).  par: the node's parameter values.
// Returns 0 if the value is finite and in the program's domain (no log or pow
// of a value <= 0, no division by 0), with kDeriv 2 if some derivative is not
// finite; 1 otherwise (df not written).
//
// An FP64 warp instruction occupies its sub-partition's unit for some 64
// cycles, an integer one for 1, so the interpretation is free and only the
// FP64 operations count: each stack entry carries a mask of the parameters
// that it depends on, and only their tangents are computed.  The others'
// are zero; where arithmetic with that zero would give NaN (times an
// infinity), all derivatives are NaN all the same.  One that leaves the finite
// range by itself leaves the others as they are.
template <bool kDeriv, class M = LibMath>
__device__ __forceinline__ int expr_eval(const Program& P, const PNode& q, const double* par, double x, double* f,
                                         double* df, const M& mt = M()) {
  double v[kExprStack], d[kDeriv ? kExprStack : 1][kMaxPar];
  unsigned act[kDeriv ? kExprStack : 1];
  bool wild = false;  // a value that tangents are multiplied with left the finite range
  int sp = 0;
  const int32_t* ops = P.ex_ops + q.ex_op0;
  const double* cs = P.ex_consts + q.ex_c0;
  for (int i = 0; i < q.ex_nops; ++i) {
    const int code = ops[i] & 0xff, arg = ops[i] >> 8;
    if (code <= RF_EX_CONST) {
      v[sp] = code == RF_EX_X ? x : code == RF_EX_PAR ? par[arg] : cs[arg];
      if constexpr (kDeriv) {
        act[sp] = code == RF_EX_PAR ? 1u << arg : 0u;
        if (code == RF_EX_PAR) d[sp][arg] = 1.0;
      }
      ++sp;
      continue;
    }
    const bool unary = code >= RF_EX_NEG && code <= RF_EX_LOG;
    const int a = sp - (unary ? 1 : 2), b = a + 1;
    const double va = v[a], vb = unary ? 0.0 : v[b];
    unsigned ma = 0, mb = 0;
    if constexpr (kDeriv) {
      ma = act[a];
      mb = unary ? 0u : act[b];
      act[a] = ma | mb;
    }
    switch (code) {
      case RF_EX_NEG:
        v[a] = -va;
        for (unsigned m = ma; m; m &= m - 1) d[a][__ffs(m) - 1] = -d[a][__ffs(m) - 1];
        break;
      case RF_EX_EXP: {
        const double r = mt.exp_(va);
        v[a] = r;
        if constexpr (kDeriv) wild |= not_finite(r);
        for (unsigned m = ma; m; m &= m - 1) d[a][__ffs(m) - 1] *= r;
        break;
      }
      case RF_EX_LOG:
        if (!(va > 0.0)) return 1;
        for (unsigned m = ma; m; m &= m - 1) d[a][__ffs(m) - 1] /= va;
        v[a] = log(va);
        break;
      case RF_EX_ADD:
      case RF_EX_SUB: {
        const double sg = code == RF_EX_ADD ? 1.0 : -1.0;
        v[a] = fma(sg, vb, va);
        for (unsigned m = mb; m; m &= m - 1) {
          const int k = __ffs(m) - 1;
          const double t = code == RF_EX_ADD ? d[b][k] : -d[b][k];
          d[a][k] = (ma >> k & 1u) ? d[a][k] + t : t;
        }
        break;
      }
      case RF_EX_MUL:
        v[a] = va * vb;
        if constexpr (kDeriv) wild |= not_finite(va) || not_finite(vb);
        for (unsigned m = ma | mb; m; m &= m - 1) {
          const int k = __ffs(m) - 1;
          const bool ia = ma >> k & 1u, ib = mb >> k & 1u;
          const double t = ib ? va * d[b][k] : 0.0;
          d[a][k] = ia ? fma(d[a][k], vb, t) : t;
        }
        break;
      case RF_EX_DIV: {
        if (vb == 0.0) return 1;
        if (!kDeriv || (ma | mb) == 0) {
          v[a] = va / vb;
          if constexpr (kDeriv) wild |= not_finite(v[a]);
          break;
        }
        const Divisor D = divisor(vb);
        const double r = quotient(va, D);
        v[a] = r;
        if constexpr (kDeriv) wild |= not_finite(r);
        for (unsigned m = ma | mb; m; m &= m - 1) {
          const int k = __ffs(m) - 1;
          const bool ia = ma >> k & 1u, ib = mb >> k & 1u;
          const double da = ia ? d[a][k] : 0.0;
          d[a][k] = quotient(ib ? fma(-r, d[b][k], da) : da, D);
        }
        break;
      }
      default: {  // RF_EX_POW: a^b = exp(b log a), a > 0
        if (!(va > 0.0)) return 1;
        const double la = log(va), r = mt.exp_(vb * la);
        v[a] = r;
        if constexpr (kDeriv) wild |= not_finite(r) || not_finite(la) || not_finite(vb);
        for (unsigned m = ma | mb; m; m &= m - 1) {
          const int k = __ffs(m) - 1;
          const bool ia = ma >> k & 1u, ib = mb >> k & 1u;
          const double t = ia ? vb * d[a][k] / va : 0.0;
          d[a][k] = r * (ib ? fma(d[b][k], la, t) : t);
        }
      }
    }
    sp = a + 1;
  }
  *f = v[0];
  if (not_finite(v[0])) return 1;
  if constexpr (kDeriv) {
    if (wild && q.n_par > 0) {
      for (int k = 0; k < q.n_par; ++k) df[k] = NAN;
      return 2;
    }
    for (int k = 0; k < q.n_par; ++k) {
      df[k] = (act[0] >> k & 1u) ? d[0][k] : 0.0;
      wild |= not_finite(df[k]);
    }
    if (wild && q.n_par > 0) return 2;
  }
  return 0;
}

// 15-point Gauss-Kronrod rule and its embedded 7-point Gauss rule on
// [-1, 1] (Kronrod 1965; the abscissae and weights as tabulated with
// QUADPACK's qk15): nodes +-kGK15x[i] with Kronrod weights kGK15w[i], the
// Gauss nodes being kGK15x[1], kGK15x[3], kGK15x[5] and 0 with weights kG7w.
__device__ __constant__ const double kGK15x[8] = {
    0.991455371120812639206854697526329, 0.949107912342758524526189684047851, 0.864864423359769072789712788640926,
    0.741531185599394439863864773280788, 0.586087235467691130294144845693013, 0.405845151377397166906606412076961,
    0.207784955007898467600689403773245, 0.0};
__device__ __constant__ const double kGK15w[8] = {
    0.022935322010529224963732008058970, 0.063092092629978553290700663189204, 0.104790010322250183839876322541518,
    0.140653259715525918745189590510238, 0.169004726639267902826583426598550, 0.190350578064785409913256402421014,
    0.204432940075298892414161999234649, 0.209482141084727828012999174891714};
__device__ __constant__ const double kG7w[4] = {0.129484966168869693270611432679082, 0.279705391489276667901467771423780,
                                                0.381830050505118944950369775488975, 0.417959183673469387755102040816327};

constexpr int kQuadPanels = 256;   // panels per refinement level (one per thread of the block)
constexpr int kQuadLevels = 16;    // refinement levels at most
constexpr double kQuadRel = 1e-14; // target error, relative to the integral
constexpr int kQuadBatch = 16;     // panels evaluated together: 16 threads for a panel's 15 points

// Shared-memory workspace of the block-cooperative quadrature.
struct QuadSmem {
  double a[2][kQuadPanels], b[2][kQuadPanels];
  double pt[kQuadBatch][1 + kMaxPar][15];  // the batch's values and derivatives by point
  double sum[kQuadBatch][2 + kMaxPar];     // its Kronrod sums, then the Gauss sum
  double red[kQuadPanels / 32][1 + kMaxPar];
  int split[kQuadPanels / 32];
  int bad;
};

// Sum of val[0..nv) over the block's first n threads (the others' are zero)
// in a fixed order (lanes by butterfly, then warps in order): the same bits
// for the same inputs.  Block-wide, every thread gets the result.
__device__ inline void quad_block_sum(QuadSmem& s, double* val, int nv, int n) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (n + 31) >> 5;
  if (warp < nw)
    for (int k = 0; k < nv; ++k) {
      double x = val[k];
      for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
      if (lane == 0) s.red[warp][k] = x;
    }
  __syncthreads();
  for (int k = 0; k < nv; ++k) {
    double x = 0.0;
    for (int w = 0; w < nw; ++w) x += s.red[w][k];
    val[k] = x;
  }
  __syncthreads();
}

// Integral of node q's program over [q.lo, q.hi] (out[0]) and its
// derivatives in the node's parameters (out[1..n_par]), by the whole block
// (blockDim.x == kQuadPanels).  Start: 16 equal panels.  At each level
// the 15-point Kronrod sum and the embedded 7-point Gauss sum of every panel
// are taken; a panel whose two sums differ by at most
// kQuadRel |I| times its share of the range is accepted (its Kronrod sums are
// added), the others are halved for the next level, in order; when the next
// level would exceed kQuadPanels panels, or at the last level, all are
// accepted.  |I| is first estimated by the 16 panels' Kronrod sum.  Every
// sum has a fixed order, so the result depends only on the parameters.
// Returns false (on every thread) outside the program's domain or for I <= 0.
//
// A level has a few dozen panels, and what it takes is the FP64 unit's time
// for the program, once per warp that runs it however few of its lanes do:
// the 15 points of 16 panels go to 240 threads (one evaluation on each of
// the block's 8 warps instead of 15 in a row on one), then one thread per
// sum adds them in the order of the points.  Thread t keeps panel t's sums.
// The parameter-point kernel of a line shape and a power times an
// exponential: 500 us -> 68 us (100 from cold caches).
__device__ inline bool expr_integrate_block(const Program& P, const PNode& q, const double* par, QuadSmem& s,
                                            double* out) {
  const int t = threadIdx.x, np = q.n_par, lane = t & 31, warp = t >> 5;
  const double lo = q.lo, hi = q.hi, span = hi - lo;
  if (t == 0) s.bad = 0;
  for (int k = 0; k <= np; ++k) out[k] = 0.0;
  int cur = 0, n_pan = 16;
  if (t < n_pan) {
    s.a[0][t] = lo + span * t / 16.0;
    s.b[0][t] = t == 15 ? hi : lo + span * (t + 1) / 16.0;
  }
  __syncthreads();
  double tol = 0.0;
  for (int level = 0; level < kQuadLevels && n_pan > 0; ++level) {
    double kr[1 + kMaxPar], g7 = 0.0;
    for (int k = 0; k <= np; ++k) kr[k] = 0.0;
    double width = 0.0;
    for (int p0 = 0; p0 < n_pan; p0 += kQuadBatch) {
      const int g = t / kQuadBatch, i = t % kQuadBatch, p = p0 + g;
      if (p < n_pan && i < 15) {
        const double a = s.a[cur][p], b = s.b[cur][p];
        const double c = 0.5 * (a + b), h = 0.5 * (b - a);
        const int j = i < 7 ? i : i < 14 ? i - 7 : 7;
        const double x = i < 7 ? c - h * kGK15x[j] : i < 14 ? c + h * kGK15x[j] : c;
        double f = 0.0, df[kMaxPar];
        if (expr_eval<true>(P, q, par, x, &f, df) != 0) {
          s.bad = 1;
        } else {
          s.pt[g][0][i] = f;
          for (int k = 0; k < np; ++k) s.pt[g][1 + k][i] = df[k];
        }
      }
      __syncthreads();
      if (s.bad) return false;
      if (p < n_pan && i <= np + 1) {  // i: the sum's index, np + 1 the Gauss sum
        const double* v = s.pt[g][i <= np ? i : 0];
        double x = 0.0;
        if (i <= np) {
          for (int n = 0; n < 15; ++n) x += kGK15w[n < 7 ? n : n < 14 ? n - 7 : 7] * v[n];
        } else {
          for (int n = 1; n < 14; n += n == 5 ? 3 : 2) x += kG7w[(n < 7 ? n : n - 7) >> 1] * v[n];
          x += kG7w[3] * v[14];
        }
        s.sum[g][i] = x;
      }
      __syncthreads();
      if (t >= p0 && t < p0 + kQuadBatch && t < n_pan) {
        const double a = s.a[cur][t], b = s.b[cur][t], h = 0.5 * (b - a);
        width = b - a;
        for (int k = 0; k <= np; ++k) kr[k] = s.sum[t - p0][k] * h;
        g7 = s.sum[t - p0][np + 1] * h;
      }
    }
    if (level == 0) {  // the tolerance from the first estimate of |I|
      double e = fabs(kr[0]);
      quad_block_sum(s, &e, 1, n_pan);
      tol = kQuadRel * e;
    }
    int split = (t < n_pan && fabs(kr[0] - g7) > tol * (width / span)) ? 1 : 0;
    // exclusive prefix sum of the split flags
    const unsigned flags = __ballot_sync(0xffffffffu, split);
    if (lane == 0) s.split[warp] = __popc(flags);
    __syncthreads();
    int n_split = 0, pref = __popc(flags & ((1u << lane) - 1u));
    for (int w = 0; w < kQuadPanels / 32; ++w) {
      if (w < warp) pref += s.split[w];
      n_split += s.split[w];
    }
    if (2 * n_split > kQuadPanels || level == kQuadLevels - 1) split = 0;  // accept all
    double contrib[1 + kMaxPar];
    for (int k = 0; k <= np; ++k) contrib[k] = (t < n_pan && !split) ? kr[k] : 0.0;
    quad_block_sum(s, contrib, 1 + np, n_pan);
    for (int k = 0; k <= np; ++k) out[k] += contrib[k];
    if (2 * n_split > kQuadPanels || level == kQuadLevels - 1) break;
    if (split) {
      const double a = s.a[cur][t], b = s.b[cur][t], m = 0.5 * (a + b);
      s.a[cur ^ 1][2 * pref] = a;
      s.b[cur ^ 1][2 * pref] = m;
      s.a[cur ^ 1][2 * pref + 1] = m;
      s.b[cur ^ 1][2 * pref + 1] = b;
    }
    __syncthreads();
    cur ^= 1;
    n_pan = 2 * n_split;
  }
  return out[0] > 0.0 && isfinite(out[0]);
}

}  // namespace rf
