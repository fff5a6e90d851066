// 64-bit fixed-point arithmetic for the FP64 transforms and stencils.
//
// One FP64 instruction of a warp occupies an SM of this GPU for 16 or more
// cycles (2 lanes per clock; measured 1.7 additions and 2.0 FMAs), a 64-bit
// integer addition (two 32-bit ones) or a 32 x 32 + 64-bit multiply-add half
// a cycle (64 lanes per clock).  Sums of doubles of one tile are therefore
// formed as integers on a common power-of-two scale taken from the tile's
// largest magnitude: a value keeps every bit above 2^-B of that magnitude
// (B >= 52, more than the 2^-53 relative rounding of each FP64 operation it
// replaces leaves in a sum of the tile's values), and integer additions are
// exact.
//
// A tile that holds an infinity or a NaN gives NaN throughout.  Scales go down to
// that of values of 2^-959: smaller ones keep the bits above 2^-1016 (FP64 itself
// keeps those above 2^-1074).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace fix64 {

typedef long long i64;

constexpr int EXP_MIN = 64;           // smallest common exponent field used (zeros and denormals are shifted out)
constexpr int EXP_SLOW = 1930;        // output exponent bases above this, or negative, take the checked path
constexpr int EXP_BAD = 1 << 20;      // scale of values that an infinity or a NaN went into
constexpr int EXP_ZERO = -(1 << 20);  // scale of exact zeros

// magnitude key of a double: its high word without the sign (the exponent
// field on top), to be maximised over a tile
__device__ __forceinline__ unsigned mag(double x) { return (unsigned)__double2hiint(x) & 0x7fffffffu; }

// exponent field of a tile's largest magnitude key (0x7ff: infinity or NaN)
__device__ __forceinline__ int tile_exp(unsigned key) {
  const int e = (int)(key >> 20);
  return e < EXP_MIN ? EXP_MIN : e;
}

// x as an integer on the scale of exponent field e: |result| < 2^B for every
// |x| of that exponent or a smaller one (truncated toward zero); s0 = e + 63 - B
__device__ __forceinline__ i64 to_fix(double x, int s0) {
  const int hi = __double2hiint(x), lo = __double2loint(x);
  // the significand with its leading bit at 2^62, moved down by d: below 2^(63 - d)
  const unsigned mh = (((unsigned)hi & 0xfffffu) | 0x100000u) << 10 | ((unsigned)lo >> 22);
  const unsigned ml = (unsigned)lo << 10;
  const unsigned d = min((unsigned)(s0 - ((hi >> 20) & 0x7ff)), 63u);
  const uint64_t m = (((uint64_t)mh << 32) | ml) >> d;
  const i64 s = (i64)(hi >> 31);
  return ((i64)m ^ s) - s;
}

static __device__ __noinline__ double from_fix_checked(i64 v, int eb) {
  if (eb >= EXP_BAD / 2) return __hiloint2double(0x7ff80000, 0);    // an infinity or NaN went in
  return v ? scalbn((double)v, eb - 1016) : 0.0;                    // may overflow to infinity or underflow
}

// v on the scale given by eb (70 less than the exponent field of 2^63 on that scale, so that
// a result of a base of zero is still a normal number) as a double, rounded to nearest (ties away from zero)
__device__ __forceinline__ double from_fix(i64 v, int eb) {
  if ((unsigned)eb > (unsigned)EXP_SLOW) return from_fix_checked(v, eb);
  const i64 s = v >> 63;
  const uint64_t a = (uint64_t)((v ^ s) - s);
  const int lz = __clzll((i64)a);
  const uint64_t n = a << (lz & 63);
  const uint64_t t = (n >> 11) + ((n >> 10) & 1u);                   // implicit bit at 2^52
  int hi = (int)(t >> 32) + ((eb + 69 - lz) << 20);
  hi = a ? (hi | ((int)s & (int)0x80000000)) : 0;
  return __hiloint2double(hi, (int)t);
}
// exponent base of from_fix for integers on the scale to_fix(., e + 63 - B) gave, times 2^sh
__device__ __forceinline__ int out_base(int e, int B, int sh = 0) {
  return e == 0x7ff ? EXP_BAD : e - 6 - B + sh;
}
// s0 of to_fix for the scale eb
__device__ __forceinline__ int fix_shift(int eb) { return eb + 69; }

// ---- integers already on a scale eb (v 2^(eb - 1016), |v| < 2^63) ----
// |v| < 2^(33 + top_bit(high(v)))
__device__ __forceinline__ int abs_hi(i64 v) { const int h = (int)(v >> 32); return h ^ (h >> 31); }
__device__ __forceinline__ int top_bit(int h) { return 31 - __clz(h); }
// Key of values on the scale ex whose magnitudes' high words or to h: maximised
// over the values that are to share a scale, key_scale() of it is the scale on which
// all of them just fit B bits.
__device__ __forceinline__ int fit_key(int h, int ex) { return ex + top_bit(h); }
__device__ __forceinline__ int key_scale(int key, int B) { return key + 33 - B; }
// v from the scale ex to the scale E (up only as far as the key allowed)
__device__ __forceinline__ i64 rescale(i64 v, int ex, int E) {
  const int d = E - ex;
  return (v << min(max(-d, 0), 63)) >> min(max(d, 0), 63);
}

// ---- multiplication by Q62 factors (|w| <= 1) ----
// w = wh 2^32 + wl with wl in (-2^31, 2^31): signed 32 x 32 products only
struct Sp { int h, l; };
__device__ __forceinline__ Sp split(i64 a) {
  Sp s;
  s.l = (int)a;
  s.h = (int)(a >> 32) - (s.l >> 31);
  return s;
}
__device__ __forceinline__ i64 wide(int a, int b) { return (i64)a * (i64)b; }
// a w for a real factor, rounded (the product of the low words is dropped)
__device__ __forceinline__ i64 mulq(i64 a, int wh, int wl) {
  const Sp s = split(a);
  const i64 mid = wide(s.h, wl) + wide(s.l, wh) + (1LL << 29);
  return (wide(s.h, wh) << 2) + (mid >> 30);
}
// (x u + y v) / 4, rounded, for |x|, |y| < 2^62 and u^2 + v^2 = 1: the high
// words of the products as they are, no shift
__device__ __forceinline__ i64 mulq2(Sp x, int uh, int ul, Sp y, int vh, int vl) {
  const i64 mid = wide(x.h, ul) + wide(x.l, uh) + wide(y.h, vl) + wide(y.l, vh) + (1LL << 31);
  return wide(x.h, uh) + wide(y.h, vh) + (mid >> 32);
}

// a Q62 factor in the split form (F: long double on the host, double on the device)
template <typename F>
__host__ __device__ inline void split_q62(F w, int* h, int* l) {
  int64_t v = (int64_t)(w * (F)4611686018427387904.0 + (w < 0 ? (F)-0.5 : (F)0.5));
  if ((int32_t)(uint32_t)(uint64_t)v == INT32_MIN) v += 1;   // wl in (-2^31, 2^31): its negation stays in range
  const int64_t lo = (int32_t)(uint32_t)(uint64_t)v;
  *l = (int)lo;
  *h = (int)((v - lo) >> 32);
}

// ---- rows of K : p ----
// K: 60-bit integers on the voxel's scale (the largest entry at 2^58 or more), each as a signed low word
// and a high word.  p: 56 bits on the scale of its largest component, as h 2^29 + l 2^-3, so that
// three 32 x 32 multiply-adds per entry give the high and the mixed products exactly and the low
// ones, which are dropped, are below 2^59: 2^-55 of max|K| max|p| at the usual 2^59 and 2^55.  (Split at
// 32 bits they reached 2^62, and the row erred by more than nine FP64 FMAs; kept by a fourth
// multiply-add the apply of 64^3 took 44.8 us for 43.4.)  Sums: 9 (2^28 2^31 + 2^31 2^27) < 2^63.
constexpr int P_BITS = 56, ROW_SHIFT = 4;
struct Vec9 { int h[9], l[9], e; };
__device__ __forceinline__ void vec9(const double* p, Vec9& f) {
  unsigned m = 0u;
#pragma unroll
  for (int c = 0; c < 9; ++c) m = max(m, mag(p[c]));
  const int e = tile_exp(m);
#pragma unroll
  for (int c = 0; c < 9; ++c) {
    const i64 v = to_fix(p[c], e + 63 - P_BITS);
    f.l[c] = (int)((unsigned)v << 3);
    f.h[c] = (int)(v >> 29) - (f.l[c] >> 31);
  }
  f.e = out_base(e, P_BITS);
}
// one row of K (entries `stride` apart, on the scale ek) times p
__device__ __forceinline__ double row9(const int2* K, size_t stride, const Vec9& p, int ek) {
  i64 hi = 0, mid = 0;
#pragma unroll
  for (int j = 0; j < 9; ++j) {
    const int2 k = K[j * stride];                          // low (signed), high
    hi += wide(k.y, p.h[j]);
    mid += wide(k.y, p.l[j]) + wide(k.x, p.h[j]);
  }
  const int eb = max(ek, p.e) >= EXP_BAD / 2 ? EXP_BAD : ek + p.e - 959;
  return from_fix((hi << ROW_SHIFT) + (mid >> (32 - ROW_SHIFT)), eb);
}

}  // namespace fix64
