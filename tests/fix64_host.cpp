// The fixed-point arithmetic of the device (csrc/fix64.cuh) compiled for the
// host, with the device's intrinsics written out, for tests/test_fix64.py.
#include <math.h>
#include <stdint.h>
#include <string.h>

static inline int64_t bits_of(double x) { int64_t b; memcpy(&b, &x, 8); return b; }
static inline int __double2hiint(double x) { return (int)(bits_of(x) >> 32); }
static inline int __double2loint(double x) { return (int)bits_of(x); }
static inline double __hiloint2double(int hi, int lo) {
  const uint64_t b = ((uint64_t)(uint32_t)hi << 32) | (uint32_t)lo;
  double x;
  memcpy(&x, &b, 8);
  return x;
}
static inline int __clzll(long long v) { return v ? __builtin_clzll((unsigned long long)v) : 64; }
static inline int __clz(int v) { return v ? __builtin_clz((unsigned)v) : 32; }
template <typename T> static inline T min(T a, T b) { return b < a ? b : a; }
template <typename T> static inline T max(T a, T b) { return a < b ? b : a; }

#include <cuda_runtime.h>
#undef __noinline__
#define __noinline__
#include "fix64.cuh"

// n rows of nine entries (low, high) on the scales ek times n vectors
extern "C" void rows9(int n, const int* K, const int* ek, const double* p, double* out) {
  for (int i = 0; i < n; ++i) {
    fix64::Vec9 f;
    fix64::vec9(p + 9 * i, f);
    out[i] = fix64::row9(reinterpret_cast<const int2*>(K) + 9 * i, 1, f, ek[i]);
  }
}
