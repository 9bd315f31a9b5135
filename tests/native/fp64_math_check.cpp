// The generic event kernel's table-driven functions (fp64_math.cuh), compiled
// for the host with stand-ins for the device's bit functions.  Reads lines
// "e x", "l z" (erfc, z <= 0) and "r z" (erfcx, z > 0), prints the results.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>

#include <cuda_runtime.h>

static inline uint64_t bits(double x) {
  uint64_t u;
  std::memcpy(&u, &x, 8);
  return u;
}
static inline int __double2hiint(double x) { return (int)(bits(x) >> 32); }
static inline int __double2loint(double x) { return (int)bits(x); }
static inline double __hiloint2double(int hi, int lo) {
  const uint64_t u = ((uint64_t)(uint32_t)hi << 32) | (uint32_t)lo;
  double x;
  std::memcpy(&x, &u, 8);
  return x;
}
static inline double __ldg(const double* p) { return *p; }
static inline double erfcx(double) { return NAN; }  // beyond the table: not checked here
using std::exp;
using std::fma;
#undef __noinline__
#undef __forceinline__
#define __noinline__
#define __forceinline__ inline

#include "fp64_math.cuh"

int main() {
  const rf::TableMath mt{(const double2*)rf::kExp64};
  char f;
  double x;
  while (std::scanf(" %c %lf", &f, &x) == 2) std::printf("%a\n", f == 'e' ? mt.exp_(x) : mt.tail(x, f == 'r'));
  return 0;
}
