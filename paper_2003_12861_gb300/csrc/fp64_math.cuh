// FP64 functions of the generic event kernel.  Its events are bound by the
// FP64 unit, where a warp instruction takes some 64 cycles, so what counts is
// the number of FP64 operations: a table look-up (integer and shared-memory
// work, free beside them) takes the place of most of a polynomial.  Decay
// model on 4e6 events 705 -> 601 us, program model on 1e6 355 -> 329.
// Largest and mean error in units in the last place, here (from the tables) /
// CUDA's: exp 0.58, 0.25 / 0.76, 0.25; erfc on [-7, 0] 0.55, 0.21 / 1.36, 0.21;
// erfcx on [0, 8] 0.61, 0.25 / on [0, 9.5] 1.96, 0.38.
#pragma once

#include <cuda_runtime.h>

#include "fp64_tables.h"

namespace rf {

// CUDA's own functions.
struct LibMath {
  static constexpr bool kTables = false;
  __device__ __forceinline__ double exp_(double x) const { return exp(x); }
  __device__ __forceinline__ double tail(double z, bool right) const { return right ? erfcx(z) : erfc(z); }
};

// T: kExp64 staged in shared memory (lanes read different entries).
struct TableMath {
  static constexpr bool kTables = true;
  const double2* T;
  // exp x = 2^(k/256) e^r, k the nearest integer to 256 x / ln 2 and
  // |r| <= ln2/512 (P. T. P. Tang, ACM TOMS 15 (1989)): 10 FP64 operations.
  // Both parts of the table entry are added, so the error stays near half a
  // unit in the last place.  Beyond +-708 (and NaN) CUDA's exp, out of line.
  __device__ __forceinline__ double exp_(double x) const {
    if ((unsigned)(__double2hiint(x) & 0x7fffffff) >= 0x40862000u) return far(x);
    const double magic = 6755399441055744.0;  // 1.5 * 2^52
    const double t = fma(x, kExp64_K, magic);
    const int k = __double2loint(t);
    const double kf = t - magic;
    const double r = fma(-kf, kExp64_C2, fma(-kf, kExp64_C1, x));
    const double p = fma(fma(fma(kExp64_4, r, kExp64_3), r, kExp64_2), r * r, r);
    const double2 e = T[k & 255];
    const double y = e.x + fma(e.x, p, e.y);
    return __hiloint2double(__double2hiint(y) + (k >> 8) * (1 << 20), __double2loint(y));
  }
  static __device__ __noinline__ double far(double x) { return exp(x); }
  // erfc(z) for z <= 0, erfcx(z) for z > 0 (right): the interpolant about the
  // nearest multiple of 1/8, 14 FP64 operations on both sides alike, where
  // erfcx and erfc take several times that each and a warp with both signs
  // ran both.  Beyond its ends: erfc rounds to 2 below -7, CUDA's erfcx from 8.
  __device__ __forceinline__ double tail(double z, bool right) const {
    if ((unsigned)(__double2hiint(z) & 0x7fffffff) >= 0x40200000u) return far_tail(z);
    const double magic = 6755399441055744.0;
    const double t = fma(z, 8.0, magic);
    const int i = __double2loint(t);
    if (i < -56) return 2.0;
    const double d = fma(t - magic, -0.125, z);
    const double* c = kTail64 + (i + (right ? 57 : 56)) * kTailRow;
    double y = __ldg(c + 10);
#pragma unroll
    for (int n = 9; n >= 1; --n) y = fma(y, d, __ldg(c + n));
    return __ldg(c) + fma(y, d, __ldg(c + 11));
  }
  static __device__ __noinline__ double far_tail(double z) { return z < 0.0 ? 2.0 : erfcx(z); }
};

}  // namespace rf
