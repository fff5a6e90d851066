// Hand-written batched 3-D real FFT of tensor-component fields (FP64 data, and
// FP32 for the mixed-precision conjugate gradients), with the frequency-space operators of the method fused between the
// forward and inverse transforms along z:
//   - the Galerkin projection with mixed control (Sec. 2.2, Eqs. weakarbi,
//     eql_discrete2) built from the rotated-scheme frequencies (App. A, Eq. kas);
//   - the Nye tensor G_ij = -eps_jkl d_k Fp_il (App. B, Eq. nyeindexfourier)
//     with the same rotated-scheme derivative.
//
// Layout.  Real fields: [c][z][y][x] (x fastest).  Half spectrum:
// [c][z][y][kx], kx = 0..n0/2.  Passes (each a kernel):
//   X  (R2C): two real rows y, y+1 packed as one complex row, one length-n0
//             FFT, then the two half spectra are separated;
//   Y  (C2C): consecutive columns (z, kx), length-n1 FFTs;
//   Z  (C2C + operator + C2C): pencils of consecutive (ky, kx), forward z
//             FFT, operator, inverse z FFT;
//   Y^-1, X^-1 (C2R).  The 1/nvox scaling is folded into the operator.
// Of small grids the X and Y passes of the three-field transforms run in one kernel each way
// (k_fft_xy, k_fft_yx).
//
// A transform is held by T = n / R0 threads (R0: its first, largest radix), one
// butterfly of R0 points per thread and pass.  The first butterfly takes its
// points from global memory straight into registers, the last one of a Y or Z
// transform stores to global memory, and only the passes between exchange
// through shared memory (double-buffered: one barrier per pass).
//
// Arithmetic.  FP32 fields are transformed in FP32.  FP64 fields are
// transformed in 64-bit fixed point (fix64.cuh): the FP64 pipe of this GPU
// does 2 lanes per clock and SM and held every FP64 pass of a 64^3 grid to
// 24-50 us, where the bytes need about 2.  A block takes the
// largest magnitude of each transform's values, converts them to integers on that
// scale with 56 or more bits (57 to 61 at every length but 288, 384 and 512; one less in the
// inverse X pass; so that no sum of the transform can overflow),
// and converts back on the way out.  Twiddles are Q62; a twiddled pass leaves the
// values a factor 4 down (the high words of the products, no shift), which is about what its
// sums grow by.  The rounding errors of a pass are 0.3 units of 2^-55 ...
// 2^-53 of the transform's largest value, below the 2^-53 of each
// intermediate value that every FP64 operation of a butterfly would leave.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "common.cuh"
#include "fix64.cuh"
#include "rve_internal.h"

namespace {

using fix64::i64;

// storage pair, arithmetic type and twiddle type of a field type R
template <typename R> struct FT;
template <> struct FT<double> { typedef double2 pair; typedef i64 w; typedef int4 tw; };
template <> struct FT<float> { typedef float2 pair; typedef float w; typedef float2 tw; };
template <typename R> using V2 = typename FT<R>::pair;
template <typename W> struct CX { W x, y; };
template <typename R> using C = CX<typename FT<R>::w>;
template <typename R> using TW = typename FT<R>::tw;

template <typename W> __device__ __forceinline__ CX<W> mk(W a, W b) { CX<W> c; c.x = a; c.y = b; return c; }
template <typename W> __device__ __forceinline__ CX<W> add(CX<W> a, CX<W> b) { return mk<W>(a.x + b.x, a.y + b.y); }
template <typename W> __device__ __forceinline__ CX<W> sub(CX<W> a, CX<W> b) { return mk<W>(a.x - b.x, a.y - b.y); }
template <int SIGN, typename W>
__device__ __forceinline__ CX<W> mul_i(CX<W> a) { return SIGN > 0 ? mk<W>(-a.y, a.x) : mk<W>(a.y, -a.x); }

// x / sqrt 2, x sqrt(3) / 2, x / 2
__device__ __forceinline__ float by_r2(float x) { return 0.70710678f * x; }
__device__ __forceinline__ float by_s3(float x) { return 0.86602540f * x; }
__device__ __forceinline__ float by_half(float x) { return 0.5f * x; }
constexpr i64 Q62_R2 = 3260954456333195553LL, Q62_S3 = 3993837246235628775LL;   // round(2^62 /sqrt 2), round(2^62 sqrt 3 /2)
__host__ __device__ constexpr int q62_lo(i64 v) { return (int)(uint32_t)(uint64_t)v; }
__host__ __device__ constexpr int q62_hi(i64 v) { return (int)((v - (i64)q62_lo(v)) >> 32); }
__device__ __forceinline__ i64 by_r2(i64 x) { return fix64::mulq(x, q62_hi(Q62_R2), q62_lo(Q62_R2)); }
__device__ __forceinline__ i64 by_s3(i64 x) { return fix64::mulq(x, q62_hi(Q62_S3), q62_lo(Q62_S3)); }
__device__ __forceinline__ i64 by_half(i64 x) { return x >> 1; }

// a * w (SIGN < 0) or a * conj(w) with w from the forward table
template <int SIGN>
__device__ __forceinline__ CX<float> twiddle(CX<float> a, const float2* tw, int idx) {
  const float2 w = __ldg(tw + idx);
  if (SIGN < 0) return mk<float>(fmaf(a.x, w.x, -a.y * w.y), fmaf(a.x, w.y, a.y * w.x));
  return mk<float>(fmaf(a.x, w.x, a.y * w.y), fmaf(a.y, w.x, -a.x * w.y));
}
template <int SIGN>
__device__ __forceinline__ CX<i64> twiddle(CX<i64> a, const int4* tw, int idx) {
  const int4 w = __ldg(tw + idx);              // cosine (high, low), sine of the forward factor
  const fix64::Sp x = fix64::split(a.x), y = fix64::split(a.y);
  // (the result is a factor 4 down)
  if (SIGN < 0) return mk<i64>(fix64::mulq2(x, w.x, w.y, y, -w.z, -w.w), fix64::mulq2(x, w.z, w.w, y, w.x, w.y));
  return mk<i64>(fix64::mulq2(x, w.x, w.y, y, w.z, w.w), fix64::mulq2(y, w.x, w.y, x, -w.z, -w.w));
}

// ---- DFTs of RAD points in registers, natural order in and out ----
template <int SIGN, typename W>
__device__ __forceinline__ void dft3(CX<W>& a0, CX<W>& a1, CX<W>& a2) {
  const CX<W> t = add(a1, a2), d = mul_i<SIGN, W>(sub(a1, a2));
  const CX<W> u = mk<W>(by_s3(d.x), by_s3(d.y));
  const CX<W> m = mk<W>(a0.x - by_half(t.x), a0.y - by_half(t.y));
  a0 = add(a0, t);
  a1 = add(m, u);
  a2 = sub(m, u);
}
template <int SIGN, typename W>
__device__ __forceinline__ void dft4(CX<W>& a0, CX<W>& a1, CX<W>& a2, CX<W>& a3) {
  const CX<W> t0 = add(a0, a2), t1 = sub(a0, a2), t2 = add(a1, a3), t3 = mul_i<SIGN, W>(sub(a1, a3));
  a0 = add(t0, t2);
  a1 = add(t1, t3);
  a2 = sub(t0, t2);
  a3 = sub(t1, t3);
}
template <int SIGN, int RAD, typename W>
__device__ __forceinline__ void dft(CX<W>* a) {
  if (RAD == 2) {
    const CX<W> t = a[0];
    a[0] = add(t, a[1]);
    a[1] = sub(t, a[1]);
  } else if (RAD == 3) {
    dft3<SIGN, W>(a[0], a[1], a[2]);
  } else if (RAD == 4) {
    dft4<SIGN, W>(a[0], a[1], a[2], a[3]);
  } else if (RAD == 6) {
    // Good-Thomas 2 x 3: input 3 i + 2 l, output 3 k1 + 4 k2 (mod 6), no factors between
    CX<W> b0 = a[0], b1 = a[2], b2 = a[4], c0 = a[3], c1 = a[5], c2 = a[1];
    dft3<SIGN, W>(b0, b1, b2);
    dft3<SIGN, W>(c0, c1, c2);
    a[0] = add(b0, c0); a[3] = sub(b0, c0);
    a[4] = add(b1, c1); a[1] = sub(b1, c1);
    a[2] = add(b2, c2); a[5] = sub(b2, c2);
  } else {
    // radix 8: a radix-2 step (a_m +/- a_{m+4}), the factors W8^m on the
    // differences, then two radix-4 DFTs (even and odd outputs)
    CX<W> b[4], c[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) { b[m] = add(a[m], a[m + 4]); c[m] = sub(a[m], a[m + 4]); }
    const CX<W> c1 = c[1], c3 = c[3];
    if (SIGN < 0) {
      c[1] = mk<W>(by_r2(c1.x + c1.y), by_r2(c1.y - c1.x));
      c[3] = mk<W>(by_r2(c3.y - c3.x), -by_r2(c3.x + c3.y));
    } else {
      c[1] = mk<W>(by_r2(c1.x - c1.y), by_r2(c1.x + c1.y));
      c[3] = mk<W>(-by_r2(c3.x + c3.y), by_r2(c3.x - c3.y));
    }
    c[2] = mul_i<SIGN, W>(c[2]);
    dft4<SIGN, W>(b[0], b[1], b[2], b[3]);
    dft4<SIGN, W>(c[0], c[1], c[2], c[3]);
#pragma unroll
    for (int m = 0; m < 4; ++m) { a[2 * m] = b[m]; a[2 * m + 1] = c[m]; }
  }
}

constexpr int RMAX = 8;                 // largest radix

// plan of one axis as the kernels take it
struct PlanDev {
  int n, npass, r0, T;                  // length, passes, first radix, threads per transform (n / r0)
  int bits;                             // B: bits of a converted input (fixed point)
  int down;                             // bits a fixed-point transform's values have moved down at its end
  unsigned tdiv;                        // ceil(2^20 / T)
  int radix[RVE_MAX_RADIX_PASSES], ns[RVE_MAX_RADIX_PASSES], step[RVE_MAX_RADIX_PASSES];
  unsigned nsdiv[RVE_MAX_RADIX_PASSES]; // ceil(2^20 / ns)
};

// j / d for 0 <= j < 512 and 1 <= d <= 512 with m = ceil(2^20 / d): the
// error j (m d - 2^20) / (2^20 d) stays below 1 / d
__device__ __forceinline__ int fdiv(int j, unsigned m) { return (int)(((unsigned)j * m) >> 20); }
unsigned div_magic(int d) { return ((1u << 20) + (unsigned)d - 1u) / (unsigned)d; }

// n / d for 0 <= n < 2^31 and 1 <= d < 2^31 by one multiplication: with s = ceil(log2 d) and m = ceil(2^(31 + s) / d)
// the error n (m d - 2^(31 + s)) / (2^(31 + s) d) stays below 1 / d.  (A division by a run-time
// number is a call of 30 to 100 instructions at the start of every block.)
struct Div {
  unsigned m;
  int s, d;
  __device__ __forceinline__ int operator()(int n) const {
    return s ? (int)(__umulhi((unsigned)n, m) >> (s - 1)) : n;
  }
};
Div make_div(int d) {
  Div r{0u, 0, d};
  while ((1LL << r.s) < d) ++r.s;
  r.m = (unsigned)(((1ULL << (31 + r.s)) + (unsigned)d - 1ULL) / (unsigned)d);
  return r;
}

PlanDev to_dev(const FFTPlan& p) {
  PlanDev d{};
  d.n = p.n;
  d.npass = p.npass;
  d.T = p.npass > 0 ? p.n / p.radix[0] : 1;
  d.r0 = p.npass > 0 ? p.radix[0] : 1;
  d.tdiv = div_magic(d.T);
  // A component below 2^B has |z| < 2^(B + 1/2) and a pass of radix r grows it
  // by at most r; a twiddled pass (all but the first) takes values below
  // 2^62 and moves them 2 bits down; the results stay below 2^61.5, so that
  // the sums of the X passes' split fit
  double grown = 0.5, bits = 61.0;
  for (int i = 0; i < p.npass; ++i) {
    if (i) {
      bits = std::fmin(bits, 62.0 - grown);
      grown -= 2.0;
    }
    grown += std::log2((double)p.radix[i]);
  }
  bits = std::fmin(bits, 61.5 - grown);
  d.bits = (int)std::floor(bits + 1e-9);
  d.down = p.npass > 1 ? 2 * (p.npass - 1) : 0;
  int ns = 1;
  for (int i = 0; i < p.npass; ++i) {
    d.radix[i] = p.radix[i];
    d.ns[i] = ns;
    d.nsdiv[i] = div_magic(ns);
    d.step[i] = p.n / (ns * p.radix[i]);
    ns *= p.radix[i];
  }
  return d;
}

// the untwiddled point of a twiddled pass, on the scale of the others
__device__ __forceinline__ CX<float> untwiddled(CX<float> a) { return a; }
__device__ __forceinline__ CX<i64> untwiddled(CX<i64> a) { return mk<i64>((a.x + 2) >> 2, (a.y + 2) >> 2); }

// Pass p of radix RAD of one transform: points ld(pos), results st(pos, value); the FIRST
// pass has no twiddles
template <int SIGN, typename R, int RAD, bool FIRST = false, class Ld, class St>
__device__ __forceinline__ void pass_r(const PlanDev& pl, int p, int tj, const TW<R>* __restrict__ tw, Ld ld, St st) {
  const int nb = pl.n / RAD, ns = pl.ns[p];
  for (int j = tj; j < nb; j += pl.T) {
    C<R> a[RAD];
#pragma unroll
    for (int m = 0; m < RAD; ++m) a[m] = ld(j + m * nb);
    const int q = fdiv(j, pl.nsdiv[p]), k = j - q * ns;
    if (!FIRST) {
      a[0] = untwiddled(a[0]);
#pragma unroll
      for (int m = 1; m < RAD; ++m) a[m] = twiddle<SIGN>(a[m], tw, m * k * pl.step[p]);
    }
    dft<SIGN, RAD>(a);
    const int d = q * ns * RAD + k;
#pragma unroll
    for (int m = 0; m < RAD; ++m) st(d + m * ns, a[m]);
  }
}

// The transform whose first butterfly's points (tj + m T) are in a[]: the
// first pass writes b0, the others alternate b1, b0, ..., the last one hands
// its results to st(pos, value); with `shared`, st is not used and the last pass
// goes to a buffer as well, which last_buffer() names.  idx maps a position of
// this thread's transform to its shared-memory element.  All threads of the
// block call it (barriers); `on`: this thread holds a transform.
//
// st only stores: conversions belong into a rolled loop over a shared result.
// Inlined into every radix they made the code a warp runs once so long that
// fetching it was the largest stall (6-8 cycles per instruction issued).
template <int SIGN, typename R, class Idx, class St>
__device__ __forceinline__ void transform(C<R>* a, C<R>* b0, C<R>* b1, const PlanDev& pl, int tj, bool on, Idx idx,
                                          const TW<R>* __restrict__ tw, bool shared, St st) {
  const int last = shared ? -1 : pl.npass - 1;        // the pass that goes to st
  if (on) {
    auto put = [&](int pos, C<R> v) {
      if (last >= 0 && last == 0) st(pos, v);
      else b0[idx(pos)] = v;
    };
    auto first = [&](auto rad) {
      constexpr int RAD = decltype(rad)::value;
      dft<SIGN, RAD>(a);
#pragma unroll
      for (int m = 0; m < RAD; ++m) put(tj * RAD + m, a[m]);
    };
    switch (pl.radix[0]) {
      case 8: first(std::integral_constant<int, 8>()); break;
      case 6: first(std::integral_constant<int, 6>()); break;
      case 4: first(std::integral_constant<int, 4>()); break;
      case 3: first(std::integral_constant<int, 3>()); break;
      case 2: first(std::integral_constant<int, 2>()); break;
      default:                                        // length 1
        if (shared) b0[idx(0)] = a[0];
        else st(0, a[0]);
        break;
    }
  }
  for (int p = 1; p < pl.npass; ++p) {
    __syncthreads();
    if (on) {
      C<R>* src = (p & 1) ? b0 : b1;
      C<R>* dst = (p & 1) ? b1 : b0;
      auto ld = [&](int pos) { return src[idx(pos)]; };
      auto put = [&](int pos, C<R> v) {
        if (p == last) st(pos, v);
        else dst[idx(pos)] = v;
      };
      switch (pl.radix[p]) {
        case 8: pass_r<SIGN, R, 8>(pl, p, tj, tw, ld, put); break;
        case 6: pass_r<SIGN, R, 6>(pl, p, tj, tw, ld, put); break;
        case 4: pass_r<SIGN, R, 4>(pl, p, tj, tw, ld, put); break;
        case 3: pass_r<SIGN, R, 3>(pl, p, tj, tw, ld, put); break;
        default: pass_r<SIGN, R, 2>(pl, p, tj, tw, ld, put); break;
      }
    }
  }
}
template <typename W>
__device__ __forceinline__ CX<W>* last_buffer(const PlanDev& pl, CX<W>* b0, CX<W>* b1) {
  return (pl.npass > 1 && !(pl.npass & 1)) ? b1 : b0;
}
struct NoStore { template <typename Z> __device__ void operator()(int, Z) const {} };

// ---- the common scale of a transform's points (FP64; all threads call it) ----
// Each transform has its own: the spectra of neighbouring
// columns differ by orders of magnitude (the divergence has almost nothing
// near the Nyquist frequencies, where the inverse Laplacian is largest), and a
// column on a larger scale than its own would lose what FP64 keeps.
// Columns (Y, Z): the transform of column c is held by the threads c, c + cpb, ...
// (cpb a power of two <= 32): shuffles within the warps, one word per warp and
// column across them.
constexpr int MAX_WARPS = 8;
template <typename R>
__device__ __forceinline__ int column_max(int key, int cpb, int* red) {
  if (sizeof(R) == 4) return 0;
  for (int o = cpb; o < 32; o <<= 1) key = max(key, __shfl_xor_sync(0xffffffffu, key, o));
  const int nw = blockDim.x >> 5;
  if (nw > 1) {
    const int lane = threadIdx.x & 31, c = lane & (cpb - 1);
    if (lane < cpb) red[(threadIdx.x >> 5) * 32 + lane] = key;
    __syncthreads();
    for (int w = 0; w < nw; ++w) key = max(key, red[w * 32 + c]);
  }
  return key;
}
// Rows (X): row pair `row` of the block is held by T consecutive threads.  T a power of two up
// to 32: shuffles; other lengths by shared-memory atomics.  (Not the block's largest key: the
// rows of a block can belong to two tensor rows of very different size.)
constexpr int MAX_ROWS = 256;
template <typename R>
__device__ __forceinline__ int row_max(int key, int T, int row, int tj, int* red) {
  if (sizeof(R) == 4) return 0;
  if (T <= 32 && (T & (T - 1)) == 0) {
    for (int o = 1; o < T; o <<= 1) key = max(key, __shfl_xor_sync(0xffffffffu, key, o));
    return key;
  }
  if (tj == 0) red[row] = key;
  __syncthreads();
  atomicMax(&red[row], key);
  __syncthreads();
  return red[row];
}

// Points as they lie in memory, their key and their conversion to a transform's
// scale.  Three storages:
//   Plain<float>:  floats, no scale;
//   Plain<double>: doubles, scaled by the exponent of the largest (to_fix);
//   Fixed:         64-bit integers with a scale of their own per row or column
//                  (the ex arrays), as the three-field transforms of the
//                  projection keep them between their passes: no conversion, only shifts.
__device__ __forceinline__ double2 st2(double a, double b) { return make_double2(a, b); }
__device__ __forceinline__ float2 st2(float a, float b) { return make_float2(a, b); }
template <typename R> struct Plain {
  typedef V2<R> pair;
  typedef R real;
  static constexpr bool FIX = false;
  static constexpr bool direct = sizeof(R) == 4;      // the last pass stores its results itself
  __device__ static int key(pair v, int) { return max(key(v.x, 0), key(v.y, 0)); }
  __device__ static int key(double v, int) { return (int)fix64::mag(v); }
  __device__ static int key(float, int) { return 0; }
  // the scale as an output exponent base (see fix64::from_fix)
  __device__ static int scale(int key, int B) { return sizeof(R) == 4 ? 0 : fix64::out_base(fix64::tile_exp((unsigned)key), B); }
  __device__ static i64 work(double x, int, int E, int B) {
    // (NaN tiles: any shift; their results are marked by E)
    return fix64::to_fix(x, E >= fix64::EXP_BAD ? 0x7ff : fix64::fix_shift(E));
  }
  __device__ static float work(float x, int, int, int) { return x; }
  // a result on the scale eb
  __device__ static pair store(C<R> z, int eb) {
    if constexpr (sizeof(R) == 4) return st2(z.x, z.y);
    else return st2(fix64::from_fix(z.x, eb), fix64::from_fix(z.y, eb));
  }
};
struct Fixed {
  typedef longlong2 pair;
  typedef i64 real;
  static constexpr bool FIX = true;
  static constexpr bool direct = true;
  __device__ static int key(pair v, int ex) { return fix64::fit_key(fix64::abs_hi(v.x) | fix64::abs_hi(v.y), ex); }
  __device__ static int key(i64 v, int ex) { return fix64::fit_key(fix64::abs_hi(v), ex); }
  __device__ static int scale(int key, int B) { return fix64::key_scale(key, B); }
  __device__ static i64 work(i64 v, int ex, int E, int) { return fix64::rescale(v, ex, E); }
  __device__ static pair store(CX<i64> z, int) { return make_longlong2(z.x, z.y); }
};
template <class S> __device__ __forceinline__ typename S::pair zero_pair() {
  typename S::pair z;
  z.x = z.y = (typename S::real)0;
  return z;
}
extern __shared__ __align__(16) unsigned char fft_smem[];

// element of position p of row `row` in the X passes (one pad element every
// eight: the strided writes of a radix-8 pass spread over the banks)
__device__ __forceinline__ int row_elem(int row, int n, int p) { return row * (n + (n >> 3) + 1) + p + (p >> 3); }

// Scales of the three-field transforms, one int each: of the divergence's rows
// (tensor row, z, y), of the row pairs of both X passes (field, z, y / 2), and of the columns
// (field, z, kx) after the Y passes and (field, ky, kx) after the Z pass.  Unused by the other storages.

// ---------------------------------------------------------------- pass X (R2C)
// in: real fields; spec: half spectrum.  rows: number of row pairs over all
// fields; rpb of them per block, T threads each.
template <typename R, class In, class Out>
__global__ void __launch_bounds__(256) k_fft_x_r2c(const typename In::real* __restrict__ in, const int* __restrict__ exin,
                                                   typename Out::pair* __restrict__ spec, int* __restrict__ exout,
                                                   int rows, int nkx, int rpb, PlanDev pl,
                                                   const TW<R>* __restrict__ tw, const double* __restrict__ done) {
  chain_wait();
  __shared__ int red[MAX_ROWS];
  __shared__ int ebs[MAX_ROWS];             // output scale of each row pair
  const int n0 = pl.n;
  C<R>* b0 = reinterpret_cast<C<R>*>(fft_smem);
  C<R>* b1 = b0 + rpb * (n0 + (n0 >> 3) + 1);
  const int row = fdiv(threadIdx.x, pl.tdiv), tj = threadIdx.x - row * pl.T;
  const long g0 = (long)blockIdx.x * rpb, g = g0 + row;
  const bool on = row < rpb && g < rows;
  const typename In::real* src = in + (size_t)(on ? g : 0) * 2 * n0;
  const int eu = In::FIX && on ? exin[2 * g] : 0, ev = In::FIX && on ? exin[2 * g + 1] : 0;
  typename In::real u[RMAX], v[RMAX];
#pragma unroll
  for (int m = 0; m < RMAX; ++m) {
    u[m] = v[m] = 0;
    if (on && m < pl.r0) {
      u[m] = src[tj + m * pl.T];
      v[m] = src[n0 + tj + m * pl.T];
    }
  }
  if (done && *done != 0.0) return;
  int key = In::FIX ? 2 * fix64::EXP_ZERO : 0;
#pragma unroll
  for (int m = 0; m < RMAX; ++m)
    if (on && m < pl.r0) key = max(key, max(In::key(u[m], eu), In::key(v[m], ev)));
  const int E = In::scale(row_max<R>(key, pl.T, row, tj, red), pl.bits), eb = E + pl.down;
  C<R> a[RMAX];
#pragma unroll
  for (int m = 0; m < RMAX; ++m) a[m] = mk(In::work(u[m], eu, E, pl.bits), In::work(v[m], ev, E, pl.bits));
  transform<-1, R>(a, b0, b1, pl, tj, on, [&](int p) { return row_elem(row, n0, p); }, tw, true, NoStore());
  const C<R>* res = last_buffer(pl, b0, b1);
  if (tj == 0 && on) {
    ebs[row] = eb;
    if (Out::FIX) exout[g] = eb;
  }
  __syncthreads();
  // the two half spectra are Z(k) +/- conj(Z(n0 - k)) without the factor 1/2
  // of the split: every operator applied between the z passes carries it in
  // its 1/nvox (SPEC_SCALE), exactly, as a power of two
  const int live = (int)min((long)rpb, rows - g0);
#pragma unroll 1
  for (int q = threadIdx.x; q < live * nkx; q += blockDim.x) {
    const int jj = q / nkx, k = q - jj * nkx;
    const C<R> zk = res[row_elem(jj, n0, k)];
    const C<R> zc = res[row_elem(jj, n0, k == 0 ? 0 : n0 - k)];
    const int ej = ebs[jj];
    typename Out::pair* dst = spec + (size_t)(g0 + jj) * 2 * nkx + k;
    dst[0] = Out::store(mk(zk.x + zc.x, zk.y - zc.y), ej);
    dst[nkx] = Out::store(mk(zk.y + zc.y, zc.x - zk.x), ej);
  }
}

// ---------------------------------------------------------------- pass X^-1 (C2R)
// S: storage of the spectrum (In) and of the real fields (Out)
template <typename R, class In, class Out>
__global__ void __launch_bounds__(256) k_fft_x_c2r(const typename In::pair* __restrict__ spec, const int* __restrict__ exin,
                                                   typename Out::real* __restrict__ out, int* __restrict__ exout,
                                                   int rows, int rows_per_plane, int nkx, int rpb, PlanDev pl,
                                                   const TW<R>* __restrict__ tw, const double* __restrict__ done) {
  chain_wait();
  __shared__ int red[MAX_ROWS];
  const int n0 = pl.n;
  C<R>* b0 = reinterpret_cast<C<R>*>(fft_smem);
  C<R>* b1 = b0 + rpb * (n0 + (n0 >> 3) + 1);
  const int row = fdiv(threadIdx.x, pl.tdiv), tj = threadIdx.x - row * pl.T;
  const long g = (long)blockIdx.x * rpb + row;
  const bool on = row < rpb && g < rows;
  const typename In::pair* src = spec + (size_t)(on ? g : 0) * 2 * nkx;
  const int* exs = In::FIX ? exin + (size_t)(on ? g / rows_per_plane : 0) * nkx : nullptr;
  // the row pair's spectra A, B at k = tj + m T <= n0 / 2 (at most RMAX / 2
  // + 1 of them) give Z(k) = A + i B and Z(n0 - k) = conj(A) + i conj(B)
  constexpr int HM = RMAX / 2 + 1;
  typename In::pair A[HM], B[HM];
  int ex[HM];
  const int bits = pl.bits - 1;          // (the sums A + i B double the components: one bit less)
#pragma unroll
  for (int m = 0; m < HM; ++m) {
    A[m] = B[m] = zero_pair<In>();
    ex[m] = 0;
    if (on && tj + m * pl.T < nkx) {
      A[m] = src[tj + m * pl.T];
      B[m] = src[nkx + tj + m * pl.T];
      if (In::FIX) ex[m] = exs[tj + m * pl.T];
    }
  }
  if (done && *done != 0.0) return;
  int key = In::FIX ? 2 * fix64::EXP_ZERO : 0;
#pragma unroll
  for (int m = 0; m < HM; ++m)
    if (on && tj + m * pl.T < nkx) key = max(key, max(In::key(A[m], ex[m]), In::key(B[m], ex[m])));
  const int E = In::scale(row_max<R>(key, pl.T, row, tj, red), bits), eb = E + pl.down;
  if (on) {
    if (Out::FIX && tj == 0) exout[g] = eb;
#pragma unroll
    for (int m = 0; m < HM; ++m) {
      const int k = tj + m * pl.T;
      if (k < nkx) {
        const C<R> z = mk(In::work(A[m].x, ex[m], E, bits), In::work(A[m].y, ex[m], E, bits));
        const C<R> w = mk(In::work(B[m].x, ex[m], E, bits), In::work(B[m].y, ex[m], E, bits));
        b1[row_elem(row, n0, k)] = mk(z.x - w.y, z.y + w.x);
        if (k > 0 && 2 * k < n0) b1[row_elem(row, n0, n0 - k)] = mk(z.x + w.y, w.x - z.y);
      }
    }
  }
  __syncthreads();
  C<R> a[RMAX];
#pragma unroll
  for (int m = 0; m < RMAX; ++m)
    if (on && m < pl.r0) a[m] = b1[row_elem(row, n0, tj + m * pl.T)];
  typename Out::real* dst = out + (size_t)(on ? g : 0) * 2 * n0;
  transform<+1, R>(a, b0, b1, pl, tj, on, [&](int p) { return row_elem(row, n0, p); }, tw, !Out::direct,
                   [&](int p, C<R> z) {
                     if constexpr (Out::direct) {
                       dst[p] = (typename Out::real)z.x;
                       dst[n0 + p] = (typename Out::real)z.y;
                     }
                   });
  if constexpr (!Out::direct) {
    __syncthreads();
    if (!on) return;
    const C<R>* res = last_buffer(pl, b0, b1);
#pragma unroll 1
    for (int p = tj; p < n0; p += pl.T) {
      const typename Out::pair v = Out::store(res[row_elem(row, n0, p)], eb);
      dst[p] = v.x;
      dst[n0 + p] = v.y;
    }
  }
}

// ---------------------------------------------------------------- pass Y (C2C)
// ncol columns (field, z, kx), cpb consecutive ones per block, kx fastest.
// Scales of stored integers, in: forward, of the row pairs (plane, y / 2); inverse,
// of the columns (field, y, kx) of the Z pass.  Out: of the columns (plane, kx).
// With fold.mean_blocks the first FOLD_BLOCKS blocks add up the divergence's and the tangent apply's
// block sums instead (see Fold).
template <int SIGN, typename R, class S>
__global__ void __launch_bounds__(256) k_fft_y(typename S::pair* __restrict__ spec, const int* __restrict__ exin,
                                               int* __restrict__ exout, int ncol, int n2, int nkx, int cpb, PlanDev pl,
                                               const TW<R>* __restrict__ tw, const double* __restrict__ done, Fold fold) {
  chain_wait();
  if (SIGN < 0 && fold.mean_blocks && blockIdx.x < FOLD_BLOCKS) {
    __shared__ double fsh[MAX_WARPS];
    if (!(done && *done != 0.0)) fold_block(fold, blockIdx.x, fsh);
    return;
  }
  const int block = (int)blockIdx.x - (SIGN < 0 && fold.mean_blocks ? FOLD_BLOCKS : 0);
  __shared__ int red[MAX_WARPS * 32];
  C<R>* b0 = reinterpret_cast<C<R>*>(fft_smem);
  C<R>* b1 = b0 + cpb * pl.n;
  const int tj = threadIdx.x / cpb, c = threadIdx.x - tj * cpb;     // cpb: a power of two
  const long col = (long)block * cpb + c;
  const bool on = tj < pl.T && col < ncol;
  const int plane = on ? (int)(col / nkx) : 0, kx = on ? (int)(col - (long)plane * nkx) : 0;
  typename S::pair* base = spec + (size_t)plane * pl.n * nkx + kx;
  const int* exs = nullptr;
  if (S::FIX) exs = SIGN < 0 ? exin + (size_t)plane * (pl.n / 2) : exin + (size_t)(plane / n2) * pl.n * nkx + kx;
  typename S::pair u[RMAX];
  int ex[RMAX];
#pragma unroll
  for (int m = 0; m < RMAX; ++m) {
    u[m] = zero_pair<S>();
    ex[m] = 0;
    if (on && m < pl.r0) {
      const int y = tj + m * pl.T;
      u[m] = base[(size_t)y * nkx];
      if (S::FIX) ex[m] = SIGN < 0 ? exs[y >> 1] : exs[(size_t)y * nkx];
    }
  }
  if (done && *done != 0.0) return;
  int key = S::FIX ? 2 * fix64::EXP_ZERO : 0;
#pragma unroll
  for (int m = 0; m < RMAX; ++m)
    if (on && m < pl.r0) key = max(key, S::key(u[m], ex[m]));
  const int E = S::scale(column_max<R>(key, cpb, red), pl.bits), eb = E + pl.down;
  C<R> a[RMAX];
#pragma unroll
  for (int m = 0; m < RMAX; ++m) a[m] = mk(S::work(u[m].x, ex[m], E, pl.bits), S::work(u[m].y, ex[m], E, pl.bits));
  if (S::FIX && on && tj == 0) exout[col] = eb;
  transform<SIGN, R>(a, b0, b1, pl, tj, on, [&](int p) { return p * cpb + c; }, tw, !S::direct, [&](int p, C<R> z) {
    if constexpr (S::direct) base[(size_t)p * nkx] = S::store(z, 0);
  });
  if constexpr (!S::direct) {
    __syncthreads();
    if (!on) return;
    const C<R>* res = last_buffer(pl, b0, b1);
#pragma unroll 1
    for (int p = tj; p < pl.n; p += pl.T) base[(size_t)p * nkx] = S::store(res[p * cpb + c], eb);
  }
}

// ---------------------------------------------------------------- planes
// The X and Y passes of one (field, z) plane in one kernel, the plane in shared
// memory in between.  On small grids a Laplace solve is bound by its chain of
// launches (about 2 us each, dependent launches included), not by their work: two of five
// go (planes_fit has the line and both sides measured).  The transforms and scales are
// those of the separate passes; a transform's threads find its largest value by
// shared-memory atomics, since a plane's transforms need not fill whole warps.
// Buffers: two of Plane::cap complex values; X transforms in row_elem's layout, Y transforms as [y][kx].

// one pass of every transform: slot q is thread tj of transform t
template <int SIGN, typename R, bool FIRST, class Slot, class Ld, class St>
__device__ __forceinline__ void plane_pass(const PlanDev& pl, int p, int slots, const TW<R>* __restrict__ tw, Slot slot, Ld ld,
                                           St st) {
#pragma unroll 1
  for (int q = threadIdx.x; q < slots; q += blockDim.x) {
    int t, tj;
    slot(q, t, tj);
    auto l = [&](int pos) { return ld(t, pos); };
    auto w = [&](int pos, C<R> v) { st(t, pos, v); };
    switch (pl.radix[p]) {
      case 8: pass_r<SIGN, R, 8, FIRST>(pl, p, tj, tw, l, w); break;
      case 6: pass_r<SIGN, R, 6, FIRST>(pl, p, tj, tw, l, w); break;
      case 4: pass_r<SIGN, R, 4, FIRST>(pl, p, tj, tw, l, w); break;
      case 3: pass_r<SIGN, R, 3, FIRST>(pl, p, tj, tw, l, w); break;
      default: pass_r<SIGN, R, 2, FIRST>(pl, p, tj, tw, l, w); break;
    }
  }
}

// sizes of one plane kernel, for its launch and its pointers
struct Plane {
  int n0, n1, nkx, rows, cap;            // rows: line pairs; cap: complex values per buffer
  Div dkx, dTx;
  PlanDev x, y;
};
template <typename R>
size_t plane_bytes(const Plane& g, bool inverse) {
  return 2 * (size_t)g.cap * sizeof(C<R>) +
         (sizeof(R) == 8 ? (2 * (size_t)g.rows + 2 * (size_t)g.nkx + (inverse ? (size_t)g.n1 * g.nkx : 0)) * sizeof(int) : 0);
}

template <typename R, class S>
__global__ void __launch_bounds__(512) k_fft_xy(const typename S::real* __restrict__ in, const int* __restrict__ exin,
                                                typename S::pair* __restrict__ spec, int* __restrict__ exout, Plane g,
                                                const TW<R>* __restrict__ twx, const TW<R>* __restrict__ twy,
                                                const double* __restrict__ done, Fold fold) {
  chain_wait();
  if (done && *done != 0.0) return;
  if (fold.mean_blocks && blockIdx.x < FOLD_BLOCKS) {
    __shared__ double fsh[32];
    fold_block(fold, blockIdx.x, fsh);
    return;
  }
  const int plane = (int)blockIdx.x - (fold.mean_blocks ? FOLD_BLOCKS : 0);
  C<R>* A = reinterpret_cast<C<R>*>(fft_smem);
  C<R>* B = A + g.cap;
  int* rowkey = reinterpret_cast<int*>(B + g.cap);   // largest key, then output scale, of each line pair
  int* rowex = rowkey + g.rows;
  int* colkey = rowex + g.rows;
  const int n0 = g.n0, nkx = g.nkx;
  if (S::FIX) {
    for (int i = threadIdx.x; i < g.rows; i += blockDim.x) rowkey[i] = 2 * fix64::EXP_ZERO;
    for (int i = threadIdx.x; i < nkx; i += blockDim.x) colkey[i] = 2 * fix64::EXP_ZERO;
    __syncthreads();
  }
  auto xslot = [&](int q, int& t, int& tj) { t = g.dTx(q); tj = q - t * g.x.T; };
  const typename S::real* src = in + (size_t)plane * g.n1 * n0;
  const int* exr = exin + (size_t)plane * g.n1;
#pragma unroll 1
  for (int q = threadIdx.x; q < g.rows * g.x.T; q += blockDim.x) {
    int row, tj;
    xslot(q, row, tj);
    typename S::real u[RMAX], v[RMAX];
#pragma unroll
    for (int m = 0; m < RMAX; ++m)
      if (m < g.x.r0) {
        u[m] = src[(size_t)2 * row * n0 + tj + m * g.x.T];
        v[m] = src[(size_t)(2 * row + 1) * n0 + tj + m * g.x.T];
      }
    int hu = 0, hv = 0;
#pragma unroll
    for (int m = 0; m < RMAX; ++m)
      if (m < g.x.r0) {
        if constexpr (S::FIX) { hu |= fix64::abs_hi(u[m]); hv |= fix64::abs_hi(v[m]); }
        B[row_elem(row, n0, tj + m * g.x.T)] = mk((typename FT<R>::w)u[m], (typename FT<R>::w)v[m]);
      }
    if constexpr (S::FIX)
      atomicMax(&rowkey[row], max(fix64::fit_key(hu, exr[2 * row]), fix64::fit_key(hv, exr[2 * row + 1])));
  }
  __syncthreads();
  C<R>* from = B;
  C<R>* to = A;
  plane_pass<-1, R, true>(g.x, 0, g.rows * g.x.T, twx, xslot,
                          [&](int row, int pos) {
                            C<R> z = from[row_elem(row, n0, pos)];
                            if constexpr (S::FIX) {
                              const int E = S::scale(rowkey[row], g.x.bits);
                              z = mk(S::work(z.x, exr[2 * row], E, 0), S::work(z.y, exr[2 * row + 1], E, 0));
                            }
                            return z;
                          },
                          [&](int row, int pos, C<R> v) { to[row_elem(row, n0, pos)] = v; });
  for (int p = 1; p < g.x.npass; ++p) {
    __syncthreads();
    C<R>* o = from; from = to; to = o;
    plane_pass<-1, R, false>(g.x, p, g.rows * g.x.T, twx, xslot, [&](int row, int pos) { return from[row_elem(row, n0, pos)]; },
                             [&](int row, int pos, C<R> v) { to[row_elem(row, n0, pos)] = v; });
  }
  if constexpr (S::FIX) {
    for (int i = threadIdx.x; i < g.rows; i += blockDim.x) rowex[i] = S::scale(rowkey[i], g.x.bits) + g.x.down;
  }
  __syncthreads();
  { C<R>* o = from; from = to; to = o; }
  // the two half spectra of each pair (without the factor 1/2, as in k_fft_x_r2c)
#pragma unroll 1
  for (int q = threadIdx.x; q < g.rows * nkx; q += blockDim.x) {
    const int row = g.dkx(q), k = q - row * nkx;
    const C<R> zk = from[row_elem(row, n0, k)], zc = from[row_elem(row, n0, k == 0 ? 0 : n0 - k)];
    const C<R> a = mk(zk.x + zc.x, zk.y - zc.y), b = mk(zk.y + zc.y, zc.x - zk.x);
    to[2 * row * nkx + k] = a;
    to[(2 * row + 1) * nkx + k] = b;
    if constexpr (S::FIX)
      atomicMax(&colkey[k], fix64::fit_key(fix64::abs_hi(a.x) | fix64::abs_hi(a.y) | fix64::abs_hi(b.x) | fix64::abs_hi(b.y),
                                           rowex[row]));
  }
  __syncthreads();
  typename S::pair* dst = spec + (size_t)plane * g.n1 * nkx;
  auto yslot = [&](int q, int& t, int& tj) { tj = g.dkx(q); t = q - tj * nkx; };
  if constexpr (S::FIX) {
    for (int k = threadIdx.x; k < nkx; k += blockDim.x)
      exout[(size_t)plane * nkx + k] = S::scale(colkey[k], g.y.bits) + g.y.down;
  }
  { C<R>* o = from; from = to; to = o; }
  plane_pass<-1, R, true>(g.y, 0, nkx * g.y.T, twy, yslot,
                          [&](int k, int pos) {
                            C<R> z = from[pos * nkx + k];
                            if constexpr (S::FIX) {
                              const int E = S::scale(colkey[k], g.y.bits);
                              z = mk(S::work(z.x, rowex[pos >> 1], E, 0), S::work(z.y, rowex[pos >> 1], E, 0));
                            }
                            return z;
                          },
                          [&](int k, int pos, C<R> v) {
                            if (g.y.npass == 1) dst[pos * nkx + k] = S::store(v, 0);
                            else to[pos * nkx + k] = v;
                          });
  for (int p = 1; p < g.y.npass; ++p) {
    __syncthreads();
    C<R>* o = from; from = to; to = o;
    plane_pass<-1, R, false>(g.y, p, nkx * g.y.T, twy, yslot, [&](int k, int pos) { return from[pos * nkx + k]; },
                             [&](int k, int pos, C<R> v) {
                               if (p + 1 == g.y.npass) dst[pos * nkx + k] = S::store(v, 0);
                               else to[pos * nkx + k] = v;
                             });
  }
}

template <typename R, class S>
__global__ void __launch_bounds__(512) k_fft_yx(const typename S::pair* __restrict__ spec, const int* __restrict__ exin,
                                                typename S::real* __restrict__ out, int* __restrict__ exout, int n2, Plane g,
                                                const TW<R>* __restrict__ twx, const TW<R>* __restrict__ twy,
                                                const double* __restrict__ done) {
  chain_wait();
  if (done && *done != 0.0) return;
  const int plane = blockIdx.x, n0 = g.n0, nkx = g.nkx;
  C<R>* A = reinterpret_cast<C<R>*>(fft_smem);
  C<R>* B = A + g.cap;
  int* rowkey = reinterpret_cast<int*>(B + g.cap);
  int* colkey = rowkey + 2 * g.rows;
  int* colex = colkey + nkx;             // scale of each column after its inverse
  int* ex = colex + nkx;                 // scale of each value of the plane as it comes in
  if (S::FIX) {
    for (int i = threadIdx.x; i < g.rows; i += blockDim.x) rowkey[i] = 2 * fix64::EXP_ZERO;
    for (int i = threadIdx.x; i < nkx; i += blockDim.x) colkey[i] = 2 * fix64::EXP_ZERO;
    __syncthreads();
  }
  const typename S::pair* src = spec + (size_t)plane * g.n1 * nkx;
  const int* exs = exin + (size_t)((unsigned)plane / (unsigned)n2) * g.n1 * nkx;
#pragma unroll 4
  for (int q = threadIdx.x; q < g.n1 * nkx; q += blockDim.x) {
    const typename S::pair v = src[q];
    B[q] = mk((typename FT<R>::w)v.x, (typename FT<R>::w)v.y);
    if constexpr (S::FIX) {
      const int e = exs[q];
      ex[q] = e;
      atomicMax(&colkey[q - g.dkx(q) * nkx], S::key(v, e));
    }
  }
  __syncthreads();
  auto yslot = [&](int q, int& t, int& tj) { tj = g.dkx(q); t = q - tj * nkx; };
  C<R>* from = B;
  C<R>* to = A;
  plane_pass<+1, R, true>(g.y, 0, nkx * g.y.T, twy, yslot,
                          [&](int k, int pos) {
                            C<R> z = from[pos * nkx + k];
                            if constexpr (S::FIX) {
                              const int E = S::scale(colkey[k], g.y.bits);
                              z = mk(S::work(z.x, ex[pos * nkx + k], E, 0), S::work(z.y, ex[pos * nkx + k], E, 0));
                            }
                            return z;
                          },
                          [&](int k, int pos, C<R> v) { to[pos * nkx + k] = v; });
  for (int p = 1; p < g.y.npass; ++p) {
    __syncthreads();
    C<R>* o = from; from = to; to = o;
    plane_pass<+1, R, false>(g.y, p, nkx * g.y.T, twy, yslot, [&](int k, int pos) { return from[pos * nkx + k]; },
                             [&](int k, int pos, C<R> v) { to[pos * nkx + k] = v; });
  }
  if constexpr (S::FIX) {
    for (int k = threadIdx.x; k < nkx; k += blockDim.x) colex[k] = S::scale(colkey[k], g.y.bits) + g.y.down;
  }
  __syncthreads();
  { C<R>* o = from; from = to; to = o; }
  const int bits = g.x.bits - 1;         // (the sums A + i B double the components: one bit less)
  if constexpr (S::FIX) {
#pragma unroll 1
    for (int q = threadIdx.x; q < g.rows * nkx; q += blockDim.x) {
      const int row = g.dkx(q), k = q - row * nkx;
      const C<R> a = from[2 * row * nkx + k], b = from[(2 * row + 1) * nkx + k];
      atomicMax(&rowkey[row], fix64::fit_key(fix64::abs_hi(a.x) | fix64::abs_hi(a.y) | fix64::abs_hi(b.x) | fix64::abs_hi(b.y),
                                             colex[k]));
    }
    __syncthreads();
    for (int i = threadIdx.x; i < g.rows; i += blockDim.x)
      exout[(size_t)plane * g.rows + i] = S::scale(rowkey[i], bits) + g.x.down;
  }
  // Z(k) = A + i B and Z(n0 - k) = conj(A) + i conj(B)
#pragma unroll 1
  for (int q = threadIdx.x; q < g.rows * nkx; q += blockDim.x) {
    const int row = g.dkx(q), k = q - row * nkx;
    C<R> a = from[2 * row * nkx + k], b = from[(2 * row + 1) * nkx + k];
    if constexpr (S::FIX) {
      const int E = S::scale(rowkey[row], bits), e = colex[k];
      a = mk(S::work(a.x, e, E, 0), S::work(a.y, e, E, 0));
      b = mk(S::work(b.x, e, E, 0), S::work(b.y, e, E, 0));
    }
    to[row_elem(row, n0, k)] = mk(a.x - b.y, a.y + b.x);
    if (k > 0 && 2 * k < n0) to[row_elem(row, n0, n0 - k)] = mk(a.x + b.y, b.x - a.y);
  }
  __syncthreads();
  auto xslot = [&](int q, int& t, int& tj) { t = g.dTx(q); tj = q - t * g.x.T; };
  typename S::real* dst = out + (size_t)plane * g.n1 * n0;
  auto put = [&](int row, int pos, C<R> v) {
    dst[2 * row * n0 + pos] = (typename S::real)v.x;
    dst[(2 * row + 1) * n0 + pos] = (typename S::real)v.y;
  };
  { C<R>* o = from; from = to; to = o; }
  plane_pass<+1, R, true>(g.x, 0, g.rows * g.x.T, twx, xslot, [&](int row, int pos) { return from[row_elem(row, n0, pos)]; },
                          [&](int row, int pos, C<R> v) {
                            if (g.x.npass == 1) put(row, pos, v);
                            else to[row_elem(row, n0, pos)] = v;
                          });
  for (int p = 1; p < g.x.npass; ++p) {
    __syncthreads();
    C<R>* o = from; from = to; to = o;
    plane_pass<+1, R, false>(g.x, p, g.rows * g.x.T, twx, xslot, [&](int row, int pos) { return from[row_elem(row, n0, pos)]; },
                             [&](int row, int pos, C<R> v) {
                               if (p + 1 == g.x.npass) put(row, pos, v);
                               else to[row_elem(row, n0, pos)] = v;
                             });
  }
}

struct OpTables {
  const double* s20; const double* s21; const double* s22;
  const double* c20; const double* c21; const double* c22;
  const double* tan0; const double* tan1; const double* tan2;
  const int8_t* nyq0; const int8_t* nyq1; const int8_t* nyq2;
  const double2* ph0; const double2* ph1; const double2* ph2;
  const double* xi0; const double* xi1; const double* xi2;
};

// The forward transform leaves the spectrum at 1 / SPEC_SCALE = 2 times its
// value (see the X pass); the operators scale by SPEC_SCALE / nvox.
constexpr double SPEC_SCALE = 0.5;

// Inverse-Laplacian weight at one frequency, with SPEC_SCALE:
// SPEC_SCALE / (64 nvox sum_m s2_m prod_{j!=m} c2_j), 0 where it vanishes
__device__ __forceinline__ double lapinv_weight(const OpTables& T, double inv_nvox, int kx, int ky, int kz) {
  const double sx = T.s20[kx], sy = T.s21[ky], sz = T.s22[kz];
  const double cx = T.c20[kx], cy = T.c21[ky], cz = T.c22[kz];
  const double lap = fma(sx, cy * cz, fma(cx, sy * cz, cx * cy * sz));
  return lap > 0.0 ? (SPEC_SCALE * inv_nvox) / (64.0 * lap) : 0.0;
}

// Operator at one frequency on the three fields of a tensor row (in double).
__device__ __forceinline__ void apply_op(const OpTables& T, const SpecParams& sp, int i, int kx, int ky, int kz,
                                         cplx& X0, cplx& X1, cplx& X2) {
  cplx Y0, Y1, Y2;
  const double sc = SPEC_SCALE * sp.inv_nvox;
  if (sp.op == OP_PROJECT) {
    if (kx == 0 && ky == 0 && kz == 0) {
      if (sp.mean_out) {
        sp.mean_out[3 * i + 0] = X0.x * sc;
        sp.mean_out[3 * i + 1] = X1.x * sc;
        sp.mean_out[3 * i + 2] = X2.x * sc;
      }
      const double nv = 1.0 / sp.inv_nvox;
      Y0 = sp.keep[3 * i + 0] ? cmk((SPEC_SCALE * X0.x - nv * sp.shift[3 * i + 0]) * sp.inv_nvox, X0.y * sc) : cmk(0.0, 0.0);
      Y1 = sp.keep[3 * i + 1] ? cmk((SPEC_SCALE * X1.x - nv * sp.shift[3 * i + 1]) * sp.inv_nvox, X1.y * sc) : cmk(0.0, 0.0);
      Y2 = sp.keep[3 * i + 2] ? cmk((SPEC_SCALE * X2.x - nv * sp.shift[3 * i + 2]) * sp.inv_nvox, X2.y * sc) : cmk(0.0, 0.0);
    } else {
      const int q0 = T.nyq0[kx], q1 = T.nyq1[ky], q2 = T.nyq2[kz];
      double u0, u1, u2;
      if (q0 + q1 + q2 >= 2) {
        u0 = u1 = u2 = 0.0;
      } else if (q0 + q1 + q2 == 1) {
        u0 = q0; u1 = q1; u2 = q2;
      } else {
        const double t0 = T.tan0[kx], t1 = T.tan1[ky], t2 = T.tan2[kz];
        const double inv = rsqrt(fma(t0, t0, fma(t1, t1, t2 * t2)));
        u0 = t0 * inv; u1 = t1 * inv; u2 = t2 * inv;
      }
      // (G X)_ij = u_j sum_l X_il u_l  (scaled by SPEC_SCALE / nvox)
      cplx s = cmk(fma(X0.x, u0, fma(X1.x, u1, X2.x * u2)), fma(X0.y, u0, fma(X1.y, u1, X2.y * u2)));
      s = cscale(s, sc);
      Y0 = cscale(s, u0); Y1 = cscale(s, u1); Y2 = cscale(s, u2);
    }
  } else if (sp.op == OP_CURL_STD) {
    // the standard spectral derivative i xi_k / h (no rotated stencil)
    const double scd = 4.0 * sp.inv4h * sc;
    const cplx D0 = cmk(0.0, T.xi0[kx] * scd), D1 = cmk(0.0, T.xi1[ky] * scd), D2 = cmk(0.0, T.xi2[kz] * scd);
    Y0 = csub(cmul(D2, X1), cmul(D1, X2));
    Y1 = csub(cmul(D0, X2), cmul(D2, X0));
    Y2 = csub(cmul(D1, X0), cmul(D0, X1));
  } else {  // OP_CURL: G_ij = -eps_jkl D_k Fp_il
    const double2 e0 = T.ph0[kx], e1 = T.ph1[ky], e2 = T.ph2[kz];
    const cplx p0 = cmk(1.0 + e0.x, e0.y), p1 = cmk(1.0 + e1.x, e1.y), p2 = cmk(1.0 + e2.x, e2.y);
    const cplx m0 = cmk(e0.x - 1.0, e0.y), m1 = cmk(e1.x - 1.0, e1.y), m2 = cmk(e2.x - 1.0, e2.y);
    const double scd = sp.inv4h * sc;
    const cplx D0 = cscale(cmul(m0, cmul(p1, p2)), scd);
    const cplx D1 = cscale(cmul(p0, cmul(m1, p2)), scd);
    const cplx D2 = cscale(cmul(p0, cmul(p1, m2)), scd);
    Y0 = csub(cmul(D2, X1), cmul(D1, X2));
    Y1 = csub(cmul(D0, X2), cmul(D2, X0));
    Y2 = csub(cmul(D1, X0), cmul(D0, X1));
  }
  X0 = Y0; X1 = Y1; X2 = Y2;
}

// the inverse-Laplacian weight of every spectrum point (layout of one field's half
// spectrum, [kz][ky][kx]), built once per handle; w32: its rounding to float
// for the FP32 transforms (nullable)
__global__ void k_lapinv_table(double* __restrict__ w, float* __restrict__ w32, OpTables T, int nkx, int n1, int n2,
                               double inv_nvox) {
  const size_t n = (size_t)nkx * n1 * n2;
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
    const int kx = (int)(e % nkx), ky = (int)((e / nkx) % n1), kz = (int)(e / ((size_t)nkx * n1));
    const double v = lapinv_weight(T, inv_nvox, kx, ky, kz);
    w[e] = v;
    if (w32) w32[e] = (float)v;
  }
}

// ---------------------------------------------------------------- pass Z + operator
// np pencils (ky, kx) of every field, cpb consecutive ones per block; the
// inverse Laplacian treats each field by itself (blockIdx.y: the field)
__device__ __forceinline__ CX<float> weighted(CX<float> z, float w, int, int&) {
  return mk<float>(z.x * w, z.y * w);
}
// the weight's significand as a Q62 factor, its exponent into the scale
__device__ __forceinline__ CX<i64> weighted(CX<i64> z, double w, int eb, int& ex) {
  const int hi = __double2hiint(w), lo = __double2loint(w);
  const fix64::Sp m = fix64::split(((i64)((((hi & 0xfffff) | 0x100000) << 9) | (int)((unsigned)lo >> 23)) << 32) |
                                   (i64)((unsigned)lo << 9));
  ex = hi ? eb + (hi >> 20) - 1022 : fix64::EXP_ZERO;
  return hi ? mk<i64>(fix64::mulq(z.x, m.h, m.l), fix64::mulq(z.y, m.h, m.l)) : mk<i64>(0, 0);
}

template <typename R, class S>
__global__ void __launch_bounds__(256) k_fft_z_lap(typename S::pair* __restrict__ spec, const int* __restrict__ exin,
                                                   int* __restrict__ exout, int np, int nkx, int cpb, PlanDev pl,
                                                   const TW<R>* __restrict__ tw, const R* __restrict__ weight,
                                                   const double* __restrict__ done) {
  chain_wait();
  __shared__ int red[2][MAX_WARPS * 32];
  C<R>* b0 = reinterpret_cast<C<R>*>(fft_smem);
  C<R>* b1 = b0 + cpb * pl.n;
  const int tj = threadIdx.x / cpb, c = threadIdx.x - tj * cpb;
  const int pc = blockIdx.x * cpb + c;
  const bool on = tj < pl.T && pc < np;
  typename S::pair* base = spec + (size_t)blockIdx.y * pl.n * np + (on ? pc : 0);
  const int* exs = S::FIX ? exin + (size_t)blockIdx.y * pl.n * nkx + (on ? pc % nkx : 0) : nullptr;
  typename S::pair u[RMAX];
  R w[RMAX];
  int ex[RMAX];
#pragma unroll
  for (int m = 0; m < RMAX; ++m) {
    u[m] = zero_pair<S>();
    w[m] = (R)0;
    ex[m] = 0;
    if (on && m < pl.r0) {
      const int z = tj + m * pl.T;
      u[m] = base[(size_t)z * np];
      if (S::FIX) ex[m] = exs[(size_t)z * nkx];
      w[m] = __ldg(weight + (size_t)z * np + pc);
    }
  }
  if (done && *done != 0.0) return;
  int key = S::FIX ? 2 * fix64::EXP_ZERO : 0;
#pragma unroll
  for (int m = 0; m < RMAX; ++m)
    if (on && m < pl.r0) key = max(key, S::key(u[m], ex[m]));
  int E = S::scale(column_max<R>(key, cpb, red[0]), pl.bits), eb = E + pl.down;
  C<R> a[RMAX];
#pragma unroll
  for (int m = 0; m < RMAX; ++m) a[m] = mk(S::work(u[m].x, ex[m], E, pl.bits), S::work(u[m].y, ex[m], E, pl.bits));
  auto idx = [&](int p) { return p * cpb + c; };
  transform<-1, R>(a, b0, b1, pl, tj, on, idx, tw, true, NoStore());
  C<R>* res = last_buffer(pl, b0, b1);
  __syncthreads();
  key = S::FIX ? 2 * fix64::EXP_ZERO : 0;
#pragma unroll
  for (int m = 0; m < RMAX; ++m) {
    a[m] = mk((typename FT<R>::w)0, (typename FT<R>::w)0);
    if (on && m < pl.r0) {
      a[m] = weighted(res[idx(tj + m * pl.T)], w[m], eb, ex[m]);
      if constexpr (S::FIX) key = max(key, S::key(make_longlong2(a[m].x, a[m].y), ex[m]));
    }
  }
  E = S::scale(column_max<R>(key, cpb, red[1]), pl.bits);
  eb = E + pl.down;
  if constexpr (S::FIX) {
#pragma unroll
    for (int m = 0; m < RMAX; ++m) a[m] = mk(S::work(a[m].x, ex[m], E, pl.bits), S::work(a[m].y, ex[m], E, pl.bits));
    if (on && tj == 0) exout[(size_t)blockIdx.y * np + pc] = eb;
  }
  // the inverse starts in the other buffer: this one may still be read
  transform<+1, R>(a, res == b0 ? b1 : b0, res, pl, tj, on, idx, tw, false, [&](int p, C<R> z) {
    base[(size_t)p * np] = S::store(z, 0);
  });
}

// The operators that couple the three fields of a tensor row (projection and
// curls; blockIdx.y: the row): each thread carries its points of all three
// through the forward transforms, applies the operator in FP64 and goes back.
__global__ void __launch_bounds__(128) k_fft_z_op(double2* __restrict__ spec, int np, int nkx, int cpb, PlanDev pl,
                                                  const int4* __restrict__ tw, OpTables T, SpecParams sp) {
  chain_wait();
  typedef double R;
  __shared__ int red[6][MAX_WARPS * 32];
  typedef Plain<double> S;
  C<R>* b0 = reinterpret_cast<C<R>*>(fft_smem);
  C<R>* b1 = b0 + cpb * pl.n;
  const int tj = threadIdx.x / cpb, c = threadIdx.x - tj * cpb;
  const int pc = blockIdx.x * cpb + c, row = blockIdx.y;
  const bool on = tj < pl.T && pc < np;
  const size_t fstride = (size_t)pl.n * np;
  double2* base = spec + (size_t)row * 3 * fstride + (on ? pc : 0);
  auto idx = [&](int p) { return p * cpb + c; };
  double2 u[3][RMAX];
#pragma unroll
  for (int f = 0; f < 3; ++f)
#pragma unroll
    for (int m = 0; m < RMAX; ++m) {
      u[f][m] = st2(0.0, 0.0);
      if (on && m < pl.r0) u[f][m] = base[f * fstride + (size_t)(tj + m * pl.T) * np];
    }
#pragma unroll
  for (int f = 0; f < 3; ++f) {
    int key = 0;
#pragma unroll
    for (int m = 0; m < RMAX; ++m) key = max(key, S::key(u[f][m], 0));
    if (f) __syncthreads();                       // the previous field's results are read
    const int E = S::scale(column_max<R>(key, cpb, red[f]), pl.bits), eb = E + pl.down;
    C<R> a[RMAX];
#pragma unroll
    for (int m = 0; m < RMAX; ++m) a[m] = mk(S::work(u[f][m].x, 0, E, pl.bits), S::work(u[f][m].y, 0, E, pl.bits));
    transform<-1, R>(a, b0, b1, pl, tj, on, idx, tw, true, NoStore());
    const C<R>* res = last_buffer(pl, b0, b1);
    __syncthreads();
#pragma unroll
    for (int m = 0; m < RMAX; ++m)
      if (on && m < pl.r0) {
        const C<R> z = res[idx(tj + m * pl.T)];
        u[f][m] = S::store(z, eb);
      }
  }
  int key[3] = {0, 0, 0};                         // (a scale per field: a component of a curl does not depend on all three)
  if (on) {
    const int ky = pc / nkx, kx = pc - ky * nkx;
#pragma unroll
    for (int m = 0; m < RMAX; ++m)
      if (m < pl.r0) {
        cplx X0 = cmk(u[0][m].x, u[0][m].y), X1 = cmk(u[1][m].x, u[1][m].y), X2 = cmk(u[2][m].x, u[2][m].y);
        apply_op(T, sp, row, kx, ky, tj + m * pl.T, X0, X1, X2);
        u[0][m] = st2(X0.x, X0.y); u[1][m] = st2(X1.x, X1.y); u[2][m] = st2(X2.x, X2.y);
#pragma unroll
        for (int f = 0; f < 3; ++f) key[f] = max(key[f], S::key(u[f][m], 0));
      }
  }
#pragma unroll
  for (int f = 0; f < 3; ++f) {
    __syncthreads();                              // the previous results are read
    const int E = S::scale(column_max<R>(key[f], cpb, red[3 + f]), pl.bits), eb = E + pl.down;
    C<R> a[RMAX];
#pragma unroll
    for (int m = 0; m < RMAX; ++m) a[m] = mk(S::work(u[f][m].x, 0, E, pl.bits), S::work(u[f][m].y, 0, E, pl.bits));
    transform<+1, R>(a, b0, b1, pl, tj, on, idx, tw, true, NoStore());
    const C<R>* res = last_buffer(pl, b0, b1);
    __syncthreads();
    if (on) {
#pragma unroll 1
      for (int p = tj; p < pl.n; p += pl.T) base[f * fstride + (size_t)p * np] = S::store(res[idx(p)], eb);
    }
  }
}

// Transforms per block.  Small blocks keep the barriers cheap and the common
// scale local; the tile starts at 1024 values (a block's shared memory is two
// tiles) and halves while the grid has fewer blocks than `fill` or the block
// more than 256 threads, down to one warp.
int rows_per_block(const PlanDev& pl, long rows, int fill) {
  int r = 1024 / pl.n;
  if (r < 1) r = 1;
  while (r > 1 && (r * pl.T > 256 || (r * pl.T > 32 && (rows + r - 1) / r < fill))) r /= 2;
  return r;
}
// columns per block of the y and z passes: a power of two, at least 8 where
// the shared memory allows it (128 bytes of consecutive FP64 columns)
int cols_per_block(const PlanDev& pl, long cols, int fill, int max_threads) {
  int c = 1;
  while (2 * c * pl.n <= 1024 && 2 * c * pl.T <= max_threads && c < 32) c *= 2;
  while (c > 8 && c * pl.T > 32 && (cols + c - 1) / c < fill) c /= 2;
  return c;
}
int round32(int t) { return (t + 31) / 32 * 32; }

OpTables op_tables(const rve_s* h) {
  OpTables T;
  T.tan0 = h->ax[0].tanh_; T.tan1 = h->ax[1].tanh_; T.tan2 = h->ax[2].tanh_;
  T.nyq0 = h->ax[0].nyq; T.nyq1 = h->ax[1].nyq; T.nyq2 = h->ax[2].nyq;
  T.ph0 = h->ax[0].ph; T.ph1 = h->ax[1].ph; T.ph2 = h->ax[2].ph;
  T.xi0 = h->ax[0].xi; T.xi1 = h->ax[1].xi; T.xi2 = h->ax[2].xi;
  T.s20 = h->ax[0].s2; T.s21 = h->ax[1].s2; T.s22 = h->ax[2].s2;
  T.c20 = h->ax[0].c2; T.c21 = h->ax[1].c2; T.c22 = h->ax[2].c2;
  return T;
}

template <typename R> const TW<R>* twt(const rve_s* h, int a);
template <> const int4* twt<double>(const rve_s* h, int a) { return h->ax[a].twq; }
template <> const float2* twt<float>(const rve_s* h, int a) { return h->ax[a].tw32; }
template <typename R> const R* lap_weight(const rve_s* h);
template <> const double* lap_weight<double>(const rve_s* h) { return h->lapw; }
template <> const float* lap_weight<float>(const rve_s* h) { return h->lapw32; }
template <class S> typename S::pair* spect(const rve_s* h);
template <> double2* spect<Plain<double>>(const rve_s* h) { return h->spec; }
template <> longlong2* spect<Fixed>(const rve_s* h) { return reinterpret_cast<longlong2*>(h->spec); }
template <> float2* spect<Plain<float>>(const rve_s* h) { return h->spec32; }

template <typename R>
size_t row_smem(int rpb, int n) { return 2 * (size_t)rpb * (n + (n >> 3) + 1) * sizeof(C<R>); }

int fft_category(const rve_s* h, int cat) { return h->fft_cat >= 0 ? h->fft_cat : cat; }

template <typename R, class In, class S>
void launch_r2c(const rve_s* h, const typename In::real* in, cudaStream_t s, const double* done, int nf) {
  const PlanDev pl = to_dev(h->plan[0]);
  const long rows = (long)nf * h->n2 * (h->n1 / 2);
  const int rpb = rows_per_block(pl, rows, h->fft_fill);
  ProfScope ps_(h, fft_category(h, RVE_K_FFT_X_R2C), s);
  launch_chained(h, k_fft_x_r2c<R, In, S>, (unsigned)((rows + rpb - 1) / rpb), round32(rpb * pl.T), row_smem<R>(rpb,
                 pl.n), s, in, h->ex.div, spect<S>(h), h->ex.x, (int)rows, h->nkx, rpb, pl, twt<R>(h, 0), done);
}

template <int SIGN, typename R, class S>
void launch_y(const rve_s* h, cudaStream_t s, const double* done, int nf, const Fold& fold = Fold{}) {
  const PlanDev pl = to_dev(h->plan[1]);
  const long cols = (long)nf * h->n2 * h->nkx;
  const int c = cols_per_block(pl, cols, h->fft_fill_y, 256);
  ProfScope ps_(h, fft_category(h, SIGN < 0 ? RVE_K_FFT_Y : RVE_K_FFT_Y_INV), s);
  const unsigned blocks = (unsigned)((cols + c - 1) / c) + (fold.mean_blocks ? (unsigned)FOLD_BLOCKS : 0u);
  launch_chained(h, k_fft_y<SIGN, R, S>, blocks, round32(c * pl.T), 2 * (size_t)c * pl.n * sizeof(C<R>), s,
                 spect<S>(h), SIGN < 0 ? h->ex.x : h->ex.z, h->ex.y, (int)cols, h->n2, h->nkx, c, pl, twt<R>(h, 1),
                 done, fold);
}

template <typename R, class S>
void launch_lap(const rve_s* h, cudaStream_t s, const double* done) {
  const PlanDev pl = to_dev(h->plan[2]);
  const int np = h->n1 * h->nkx;
  const int c = cols_per_block(pl, 3L * np, h->fft_fill_z, 256);
  ProfScope ps_(h, RVE_K_FFT_Z_OP, s);
  launch_chained(h, k_fft_z_lap<R, S>, dim3((np + c - 1) / c, 3), round32(c * pl.T), 2 * (size_t)c * pl.n *
                 sizeof(C<R>), s, spect<S>(h), h->ex.y, h->ex.z, np, h->nkx, c, pl, twt<R>(h, 2), lap_weight<R>(h),
                 done);
}

void zop(const rve_s* h, const SpecParams& sp, cudaStream_t s) {
  const PlanDev pl = to_dev(h->plan[2]);
  const int np = h->n1 * h->nkx;
  const int c = cols_per_block(pl, 3L * np, h->fft_fill_z, 128);
  ProfScope ps_(h, fft_category(h, RVE_K_FFT_Z_OP), s);
  launch_chained(h, k_fft_z_op, dim3((np + c - 1) / c, 3), round32(c * pl.T), 2 * (size_t)c * pl.n *
                 sizeof(C<double>), s, h->spec, np, h->nkx, c, pl, h->ax[2].twq, op_tables(h), sp);
}

template <typename R, class S, class Out>
void launch_c2r(const rve_s* h, typename Out::real* out, cudaStream_t s, const double* done, int nf) {
  const PlanDev pl = to_dev(h->plan[0]);
  const long rows = (long)nf * h->n2 * (h->n1 / 2);
  const int rpb = rows_per_block(pl, rows, h->fft_fill);
  ProfScope ps_(h, fft_category(h, RVE_K_FFT_X_C2R), s);
  launch_chained(h, k_fft_x_c2r<R, S, Out>, (unsigned)((rows + rpb - 1) / rpb), round32(rpb * pl.T), row_smem<R>(rpb,
                 pl.n), s, spect<S>(h), h->ex.y, out, h->ex.u, (int)rows, h->n1 / 2, h->nkx, rpb, pl, twt<R>(h, 0),
                 done);
}

}  // namespace

cudaError_t launch_lapinv_table(const rve_s* h, cudaStream_t s) {
  if (!h->lapw) return cudaSuccess;
  k_lapinv_table<<<RVE_RED_BLOCKS, 256, 0, s>>>(h->lapw, h->lapw32, op_tables(h), h->nkx, h->n1, h->n2,
                                                1.0 / (double)h->nvox);
  return cudaGetLastError();
}

// Radices of a length 2^a 3^b, the largest first (a transform has n / radix[0]
// threads): 8s, and what is left of the 2s as a 6 (with a 3), as 4 4 instead of 8 2
// (four radix-2 butterflies per thread would follow one of radix 8), or as a 4;
// then 3s.
void make_plan(int n, FFTPlan* p) {
  p->n = n;
  p->npass = 0;
  int a = 0, b = 0, m = n;
  while (m % 2 == 0) { ++a; m /= 2; }
  while (m % 3 == 0) { ++b; m /= 3; }
  if (m != 1) { p->npass = -1; return; }     // unsupported length
  auto add = [&](int r) { p->radix[p->npass++] = r; };
  const bool fours = a % 3 == 1 && a > 1 && b == 0;
  for (int q = a / 3 - (fours ? 1 : 0); q > 0; --q) add(8);
  if (fours) { add(4); add(4); }
  else if (a % 3 == 1 && b > 0) { add(6); --b; }
  else if (a % 3 == 1) add(2);
  else if (a % 3 == 2 && b > 1) { add(6); add(6); b -= 2; }
  else if (a % 3 == 2) add(4);
  for (; b > 0; --b) add(3);
}

Plane plane_of(const rve_s* h) {
  Plane g;
  g.n0 = h->n0; g.n1 = h->n1; g.nkx = h->nkx; g.rows = h->n1 / 2;
  g.cap = std::max(g.rows * (h->n0 + (h->n0 >> 3) + 1), h->n1 * h->nkx);
  g.x = to_dev(h->plan[0]);
  g.y = to_dev(h->plan[1]);
  g.dkx = make_div(h->nkx);
  g.dTx = make_div(g.x.T);
  return g;
}
// Whole planes per block where two buffers fit 47 KB (with the static part the 48 KB a launch
// gets unasked): 48 x 48 in FP64, 64 x 64 in FP32.  Faster on every grid below the
// line that was measured, by what two launches cost: an FP64 projection of 8^3 40.3 -> 36.6 us,
// 16^3 44.0 -> 39.9, 32^3 54.3 -> 50.5, 36 x 54 x 27 58.6 -> 56.8, 48^3 67.9 -> 65.9,
// 16 x 16 x 256 62.3 -> 58.0; a mixed increment of 32^3 12.25 -> 11.88 ms, of 64^3 80.5 -> 79.6 ms.
// Above it few blocks share an SM and the passes within a block wait for each other: FP64
// at 64^3 (84 KB) 79.6 -> 81.8 us.
constexpr size_t PLANE_SMEM = 47 * 1024;
template <typename R>
bool planes_fit(const rve_s* h) { return plane_bytes<R>(plane_of(h), true) <= PLANE_SMEM; }
template <typename R>
int plane_threads(const Plane& g) {
  return std::min(512, round32(std::max(g.rows * g.x.T, g.nkx * g.y.T)));
}

template <typename R, class S>
void launch_xy(const rve_s* h, const typename S::real* in, cudaStream_t s, const double* done, const Fold& fold) {
  const Plane g = plane_of(h);
  ProfScope ps_(h, RVE_K_FFT_X_R2C, s);
  launch_chained(h, k_fft_xy<R, S>, 3 * h->n2 + (fold.mean_blocks ? FOLD_BLOCKS : 0), plane_threads<R>(g),
                 plane_bytes<R>(g, false), s, in, h->ex.div, spect<S>(h), h->ex.y, g, twt<R>(h, 0), twt<R>(h, 1), done, fold);
}
template <typename R, class S>
void launch_yx(const rve_s* h, typename S::real* out, cudaStream_t s, const double* done) {
  const Plane g = plane_of(h);
  ProfScope ps_(h, RVE_K_FFT_X_C2R, s);
  launch_chained(h, k_fft_yx<R, S>, 3 * h->n2, plane_threads<R>(g), plane_bytes<R>(g, true), s, spect<S>(h), h->ex.z, out,
                 h->ex.u, h->n2, g, twt<R>(h, 0), twt<R>(h, 1), done);
}

// the block sums waiting to be added up, taken by the caller's Y pass
Fold take_fold(const rve_s* h) {
  Fold f{};
  f.mean = h->partial;
  f.mean_blocks = h->fold.mean_blocks;
  f.mean_mask = h->fold.mean_mask;
  f.inv_nvox = 1.0 / (double)h->nvox;
  f.pkp = h->partial_pkp();
  f.pkp_blocks = h->fold.pkp_blocks;
  f.xmean = h->dscal + DS_XMEAN;
  f.rr_pkp_alpha = h->dscal + DS_RR;
  static_assert(DS_PKP == DS_RR + 1 && DS_ALPHA == DS_RR + 2, "Fold writes these scalars in a row");
  h->fold.mean_blocks = h->fold.pkp_blocks = 0;
  return f;
}

// nine fields (double spectra) around the operators that couple a tensor row
cudaError_t launch_fft9(const rve_s* h, const double* in, double* out, const SpecParams& sp, cudaStream_t s) {
  typedef Plain<double> S;
  launch_r2c<double, S, S>(h, in, s, nullptr, 9);
  launch_y<-1, double, S>(h, s, nullptr, 9);
  zop(h, sp, s);
  launch_y<+1, double, S>(h, s, nullptr, 9);
  launch_c2r<double, S, S>(h, out, s, nullptr, 9);
  return cudaGetLastError();
}
// three fields around the inverse Laplacian.  FP64: the divergence comes and the
// solution goes as integers with a scale per row (h->ex), or as doubles where the
// stencils of this grid work on doubles
cudaError_t launch_laplace_solve(const rve_s* h, const double* d, double* u, bool fixed, cudaStream_t s,
                                 const double* done) {
  if (fixed && planes_fit<double>(h)) {
    launch_xy<double, Fixed>(h, reinterpret_cast<const i64*>(d), s, done, take_fold(h));
    launch_lap<double, Fixed>(h, s, done);
    launch_yx<double, Fixed>(h, reinterpret_cast<i64*>(u), s, done);
    return cudaGetLastError();
  }
  if (fixed) launch_r2c<double, Fixed, Fixed>(h, reinterpret_cast<const i64*>(d), s, done, 3);
  else launch_r2c<double, Plain<double>, Fixed>(h, d, s, done, 3);
  launch_y<-1, double, Fixed>(h, s, done, 3, take_fold(h));
  launch_lap<double, Fixed>(h, s, done);
  launch_y<+1, double, Fixed>(h, s, done, 3);
  if (fixed) launch_c2r<double, Fixed, Fixed>(h, reinterpret_cast<i64*>(u), s, done, 3);
  else launch_c2r<double, Fixed, Plain<double>>(h, u, s, done, 3);
  return cudaGetLastError();
}
cudaError_t launch_laplace_solve32(const rve_s* h, const float* d, float* u, cudaStream_t s, const double* done) {
  typedef Plain<float> S;
  if (planes_fit<float>(h)) {
    launch_xy<float, S>(h, d, s, done, take_fold(h));
    launch_lap<float, S>(h, s, done);
    launch_yx<float, S>(h, u, s, done);
    return cudaGetLastError();
  }
  launch_r2c<float, S, S>(h, d, s, done, 3);
  launch_y<-1, float, S>(h, s, done, 3, take_fold(h));
  launch_lap<float, S>(h, s, done);
  launch_y<+1, float, S>(h, s, done, 3);
  launch_c2r<float, S, S>(h, u, s, done, 3);
  return cudaGetLastError();
}
