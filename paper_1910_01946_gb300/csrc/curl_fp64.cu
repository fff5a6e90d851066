// The Nye curl of a mixed-precision handle's rve_eval_constitutive, in FP64 floating
// point.
//
// That call returns the consistent tangent rounded to FP32 (the storage of
// the mixed-precision conjugate gradients).  Rounding turns a difference of one part in 1e13
// of what goes in into one of 6e-8 wherever it crosses a rounding boundary: with the curl in
// fixed point (fft.cu) and the local update of constitutive.cu about 40 of a million
// entries came out as the other neighbouring float.  So this entry point keeps the
// floating-point arithmetic, operation for operation, from the curl to the tangent (here, k_local_fp64
// and k_tangent_fp64 in constitutive.cu): its tangents are the same bits as before the
// fixed-point transforms.  Everything that is not rounded to FP32 takes the
// fast path, whose results agree to the last digits (64^3: curl 92 us per pass here,
// 38 there).
//
// Layout and passes as in fft.cu: X (two real rows packed as one complex row), Y, Z with the
// curl between the transforms, Y^-1, X^-1; mixed-radix 8/4/2/3 Stockham passes in
// shared memory.
#include "common.cuh"
#include "rve_internal.h"

namespace {

// complex value and storage pair type of a real type R
template <typename R> struct CX { R x, y; };
template <typename R> struct V2T;
template <> struct V2T<double> { typedef double2 t; };
template <typename R> using V2 = typename V2T<R>::t;

template <typename R> __device__ __forceinline__ CX<R> mk(R a, R b) { CX<R> c; c.x = a; c.y = b; return c; }
template <typename R> __device__ __forceinline__ CX<R> add(CX<R> a, CX<R> b) { return mk<R>(a.x + b.x, a.y + b.y); }
template <typename R> __device__ __forceinline__ CX<R> sub(CX<R> a, CX<R> b) { return mk<R>(a.x - b.x, a.y - b.y); }
template <typename R> __device__ __forceinline__ CX<R> scl(CX<R> a, R s) { return mk<R>(a.x * s, a.y * s); }
template <typename R> __device__ __forceinline__ V2<R> st2(R a, R b) { V2<R> v; v.x = a; v.y = b; return v; }

struct PlanDev {
  int n, npass;
  int radix[RVE_MAX_RADIX_PASSES];
};

PlanDev to_dev(const FFTPlan& p) {
  PlanDev d;
  d.n = p.n;
  d.npass = p.npass;
  for (int i = 0; i < RVE_MAX_RADIX_PASSES; ++i) d.radix[i] = p.radix[i];
  return d;
}

// a * w or a * conj(w) (w from the forward table) with the sign fixed at
// compile time, so the negation folds into the FMA operands; float
// transforms read the float table
template <int SIGN, typename R>
__device__ __forceinline__ CX<R> twiddle(CX<R> a, const V2<R>* tw, int idx) {
  const V2<R> w = __ldg(tw + idx);
  if (SIGN < 0) return mk<R>(fma(a.x, w.x, -a.y * w.y), fma(a.x, w.y, a.y * w.x));
  return mk<R>(fma(a.x, w.x, a.y * w.y), fma(a.y, w.x, -a.x * w.y));
}

template <int SIGN, typename R>
__device__ __forceinline__ CX<R> mul_i(CX<R> a) { return SIGN > 0 ? mk<R>(-a.y, a.x) : mk<R>(a.y, -a.x); }

// One Stockham pass of radix R over `howmany` contiguous transforms of length
// N from src to dst (both shared memory).
template <int SIGN, typename RT>
__device__ void stockham_pass(const CX<RT>* __restrict__ src, CX<RT>* __restrict__ dst, int N, int howmany,
                              int R, int Ns, const V2<RT>* tw) {
  typedef CX<RT> cplx;
  const int nb = N / R;
  const int total = nb * howmany;
  const int twstep = N / (Ns * R);
  for (int b = threadIdx.x; b < total; b += blockDim.x) {
    const int tr = b / nb;
    const int j = b - tr * nb;
    const int k = j % Ns;
    const cplx* X = src + tr * N;
    cplx* Y = dst + tr * N;
    const int d = (j / Ns) * Ns * R + k;
    if (R == 8) {
      // radix 8 as a radix-2 step (a_m +/- a_{m+4}), the factors W8^m on the
      // differences, then two radix-4 DFTs (even and odd outputs)
      cplx a[8];
#pragma unroll
      for (int m = 0; m < 8; ++m) a[m] = X[j + m * nb];
      if (k) {
#pragma unroll
        for (int m = 1; m < 8; ++m) a[m] = twiddle<SIGN, RT>(a[m], tw, m * k * twstep);
      }
      const RT r2 = (RT)0.70710678118654752440;    // 1/sqrt(2)
      cplx b[4], c[4];
#pragma unroll
      for (int m = 0; m < 4; ++m) { b[m] = add(a[m], a[m + 4]); c[m] = sub(a[m], a[m + 4]); }
      // c1 *= W8^(sign), c2 *= -/+ i, c3 *= W8^(3 sign)
      {
        const cplx c1 = c[1], c3 = c[3];
        if (SIGN < 0) {
          c[1] = mk<RT>(r2 * (c1.x + c1.y), r2 * (c1.y - c1.x));
          c[3] = mk<RT>(r2 * (c3.y - c3.x), -r2 * (c3.x + c3.y));
        } else {
          c[1] = mk<RT>(r2 * (c1.x - c1.y), r2 * (c1.x + c1.y));
          c[3] = mk<RT>(-r2 * (c3.x + c3.y), r2 * (c3.x - c3.y));
        }
        c[2] = mul_i<SIGN, RT>(c[2]);
      }
      const cplx t0 = add(b[0], b[2]), t1 = sub(b[0], b[2]), t2 = add(b[1], b[3]), t3 = mul_i<SIGN, RT>(sub(b[1], b[3]));
      const cplx u0 = add(c[0], c[2]), u1 = sub(c[0], c[2]), u2 = add(c[1], c[3]), u3 = mul_i<SIGN, RT>(sub(c[1], c[3]));
      Y[d] = add(t0, t2);
      Y[d + 4 * Ns] = sub(t0, t2);
      Y[d + 2 * Ns] = add(t1, t3);
      Y[d + 6 * Ns] = sub(t1, t3);
      Y[d + Ns] = add(u0, u2);
      Y[d + 5 * Ns] = sub(u0, u2);
      Y[d + 3 * Ns] = add(u1, u3);
      Y[d + 7 * Ns] = sub(u1, u3);
    } else if (R == 4) {
      cplx a0 = X[j], a1 = X[j + nb], a2 = X[j + 2 * nb], a3 = X[j + 3 * nb];
      if (k) {
        a1 = twiddle<SIGN, RT>(a1, tw, k * twstep);
        a2 = twiddle<SIGN, RT>(a2, tw, 2 * k * twstep);
        a3 = twiddle<SIGN, RT>(a3, tw, 3 * k * twstep);
      }
      cplx t0 = add(a0, a2), t1 = sub(a0, a2), t2 = add(a1, a3), t3 = mul_i<SIGN, RT>(sub(a1, a3));
      Y[d] = add(t0, t2);
      Y[d + Ns] = add(t1, t3);
      Y[d + 2 * Ns] = sub(t0, t2);
      Y[d + 3 * Ns] = sub(t1, t3);
    } else if (R == 2) {
      cplx a0 = X[j], a1 = X[j + nb];
      if (k) a1 = twiddle<SIGN, RT>(a1, tw, k * twstep);
      Y[d] = add(a0, a1);
      Y[d + Ns] = sub(a0, a1);
    } else {  // R == 3
      cplx a0 = X[j], a1 = X[j + nb], a2 = X[j + 2 * nb];
      if (k) {
        a1 = twiddle<SIGN, RT>(a1, tw, k * twstep);
        a2 = twiddle<SIGN, RT>(a2, tw, 2 * k * twstep);
      }
      const RT s3 = (RT)0.86602540378443864676;  // sqrt(3)/2
      cplx t = add(a1, a2);
      cplx u = scl(mul_i<SIGN, RT>(sub(a1, a2)), s3);
      cplx m = mk<RT>(fma((RT)-0.5, t.x, a0.x), fma((RT)-0.5, t.y, a0.y));
      Y[d] = add(a0, t);
      Y[d + Ns] = add(m, u);
      Y[d + 2 * Ns] = sub(m, u);
    }
  }
}

// Full transform of `howmany` contiguous length-N sequences; the caller has
// synchronised after filling `a`.  Returns the buffer that holds the result.
template <int SIGN, typename RT>
__device__ CX<RT>* block_fft(CX<RT>* a, CX<RT>* b, const PlanDev& pl, int howmany, const V2<RT>* tw) {
  int Ns = 1;
  for (int p = 0; p < pl.npass; ++p) {
    const int R = pl.radix[p];
    stockham_pass<SIGN, RT>(a, b, pl.n, howmany, R, Ns, tw);
    __syncthreads();
    CX<RT>* t = a; a = b; b = t;
    Ns *= R;
  }
  return a;
}

// ---------------------------------------------------------------- pass X (R2C)
// in: real fields (type R); spec: half spectrum (pairs of R)
template <typename R>
__global__ void __launch_bounds__(256) k_fft_x_r2c(const R* __restrict__ in, V2<R>* __restrict__ spec,
                                                   int n0, int n1, int n2, int nkx, int rpb, PlanDev pl,
                                                   const V2<R>* __restrict__ tw) {
  typedef CX<R> cplx;
  extern __shared__ __align__(16) unsigned char smraw[];
  cplx* a = reinterpret_cast<cplx*>(smraw);
  cplx* b = a + rpb * n0;
  const int f = blockIdx.z, z = blockIdx.y, j0 = blockIdx.x * rpb;
  const size_t nvox = (size_t)n0 * n1 * n2;
  const R* src = in + f * nvox + (size_t)z * n1 * n0;
  for (int e = threadIdx.x; e < rpb * n0; e += blockDim.x) {
    const int jj = e / n0, x = e - jj * n0;
    const int y0 = 2 * (j0 + jj);
    a[e] = mk<R>(src[(size_t)y0 * n0 + x], src[(size_t)(y0 + 1) * n0 + x]);
  }
  __syncthreads();
  cplx* res = block_fft<-1, R>(a, b, pl, rpb, tw);
  V2<R>* dst = spec + ((size_t)f * n2 + z) * n1 * nkx;
  // the two half spectra are Z(k) +/- conj(Z(n0 - k)) without the factor 1/2
  // of the split, which the curl carries in its 1/nvox (SPEC_SCALE), exactly
  for (int e = threadIdx.x; e < rpb * nkx; e += blockDim.x) {
    const int jj = e / nkx, k = e - jj * nkx;
    const cplx zk = res[jj * n0 + k];
    const cplx zc = res[jj * n0 + (k == 0 ? 0 : n0 - k)];
    const cplx zm = mk<R>(zc.x, -zc.y);
    const cplx s = add(zk, zm), d = sub(zk, zm);
    const int y0 = 2 * (j0 + jj);
    dst[(size_t)y0 * nkx + k] = st2<R>(s.x, s.y);
    dst[(size_t)(y0 + 1) * nkx + k] = st2<R>(d.y, -d.x);
  }
}

// ---------------------------------------------------------------- pass X^-1 (C2R)
template <typename R>
__global__ void __launch_bounds__(256) k_fft_x_c2r(const V2<R>* __restrict__ spec, R* __restrict__ out,
                                                   int n0, int n1, int n2, int nkx, int rpb, PlanDev pl,
                                                   const V2<R>* __restrict__ tw) {
  typedef CX<R> cplx;
  extern __shared__ __align__(16) unsigned char smraw[];
  cplx* a = reinterpret_cast<cplx*>(smraw);
  cplx* b = a + rpb * n0;
  const int f = blockIdx.z, z = blockIdx.y, j0 = blockIdx.x * rpb;
  const size_t nvox = (size_t)n0 * n1 * n2;
  const V2<R>* src = spec + ((size_t)f * n2 + z) * n1 * nkx;
  for (int e = threadIdx.x; e < rpb * n0; e += blockDim.x) {
    const int jj = e / n0, k = e - jj * n0;
    const int y0 = 2 * (j0 + jj);
    cplx A, B;
    if (k < nkx) {
      V2<R> u = src[(size_t)y0 * nkx + k], v = src[(size_t)(y0 + 1) * nkx + k];
      A = mk<R>(u.x, u.y); B = mk<R>(v.x, v.y);
    } else {
      V2<R> u = src[(size_t)y0 * nkx + (n0 - k)], v = src[(size_t)(y0 + 1) * nkx + (n0 - k)];
      A = mk<R>(u.x, -u.y); B = mk<R>(v.x, -v.y);
    }
    a[e] = mk<R>(A.x - B.y, A.y + B.x);  // A + i B
  }
  __syncthreads();
  cplx* res = block_fft<+1, R>(a, b, pl, rpb, tw);
  R* dst = out + f * nvox + (size_t)z * n1 * n0;
  for (int e = threadIdx.x; e < rpb * n0; e += blockDim.x) {
    const int jj = e / n0, x = e - jj * n0;
    const int y0 = 2 * (j0 + jj);
    dst[(size_t)y0 * n0 + x] = res[e].x;
    dst[(size_t)(y0 + 1) * n0 + x] = res[e].y;
  }
}

// ---------------------------------------------------------------- pass Y (C2C)
template <int SIGN, typename R>
__global__ void __launch_bounds__(256) k_fft_y(V2<R>* __restrict__ spec, int n1, int n2, int nkx, int tx,
                                               PlanDev pl, const V2<R>* __restrict__ tw) {
  typedef CX<R> cplx;
  extern __shared__ __align__(16) unsigned char smraw[];
  cplx* a = reinterpret_cast<cplx*>(smraw);
  cplx* b = a + tx * n1;
  const int f = blockIdx.z, z = blockIdx.y, kx0 = blockIdx.x * tx;
  V2<R>* base = spec + ((size_t)f * n2 + z) * n1 * nkx;
  for (int e = threadIdx.x; e < tx * n1; e += blockDim.x) {
    const int y = e / tx, t = e - y * tx;
    const int kx = kx0 + t;
    V2<R> v = kx < nkx ? base[(size_t)y * nkx + kx] : st2<R>((R)0, (R)0);
    a[t * n1 + y] = mk<R>(v.x, v.y);
  }
  __syncthreads();
  cplx* res = block_fft<SIGN, R>(a, b, pl, tx, tw);
  for (int e = threadIdx.x; e < tx * n1; e += blockDim.x) {
    const int y = e / tx, t = e - y * tx;
    const int kx = kx0 + t;
    if (kx < nkx) {
      cplx v = res[t * n1 + y];
      base[(size_t)y * nkx + kx] = st2<R>(v.x, v.y);
    }
  }
}

constexpr double SPEC_SCALE = 0.5;

// G_ij = -eps_jkl D_k Fp_il at one frequency, on the three fields of a tensor row
__device__ __forceinline__ void apply_curl(const double2* ph0, const double2* ph1, const double2* ph2, double inv_nvox,
                                           double inv4h, int kx, int ky, int kz, cplx& X0, cplx& X1, cplx& X2) {
  cplx Y0, Y1, Y2;
  const double sc = SPEC_SCALE * inv_nvox;
  const double2 e0 = ph0[kx], e1 = ph1[ky], e2 = ph2[kz];
  const cplx p0 = cmk(1.0 + e0.x, e0.y), p1 = cmk(1.0 + e1.x, e1.y), p2 = cmk(1.0 + e2.x, e2.y);
  const cplx m0 = cmk(e0.x - 1.0, e0.y), m1 = cmk(e1.x - 1.0, e1.y), m2 = cmk(e2.x - 1.0, e2.y);
  const double scd = inv4h * sc;
  const cplx D0 = cscale(cmul(m0, cmul(p1, p2)), scd);
  const cplx D1 = cscale(cmul(p0, cmul(m1, p2)), scd);
  const cplx D2 = cscale(cmul(p0, cmul(p1, m2)), scd);
  Y0 = csub(cmul(D2, X1), cmul(D1, X2));
  Y1 = csub(cmul(D0, X2), cmul(D2, X0));
  Y2 = csub(cmul(D1, X0), cmul(D0, X1));
  X0 = Y0; X1 = Y1; X2 = Y2;
}

// ---------------------------------------------------------------- pass Z + operator
template <typename R>
__global__ void __launch_bounds__(256) k_fft_z_op(V2<R>* __restrict__ spec, int n1, int n2, int nkx, int tx,
                                                  PlanDev pl, const V2<R>* __restrict__ tw, const double2* ph0,
                                                  const double2* ph1, const double2* ph2, double inv_nvox,
                                                  double inv4h) {
  typedef CX<R> cx;
  extern __shared__ __align__(16) unsigned char smraw[];
  const int cnt = 3 * tx * n2;
  cx* a = reinterpret_cast<cx*>(smraw);
  cx* b = a + cnt;
  const int i = blockIdx.z, ky = blockIdx.y, kx0 = blockIdx.x * tx;
  const size_t zstride = (size_t)n1 * nkx;
  for (int e = threadIdx.x; e < cnt; e += blockDim.x) {
    const int c = e / (tx * n2);
    const int rem = e - c * tx * n2;
    const int z = rem / tx, t = rem - z * tx;
    const int kx = kx0 + t;
    const size_t f = 3 * i + c;
    V2<R> v = kx < nkx ? spec[(f * n2 + z) * zstride + (size_t)ky * nkx + kx] : st2<R>((R)0, (R)0);
    a[(c * tx + t) * n2 + z] = mk<R>(v.x, v.y);
  }
  __syncthreads();
  cx* res = block_fft<-1, R>(a, b, pl, 3 * tx, tw);
  cx* oth = (res == a) ? b : a;
  for (int e = threadIdx.x; e < tx * n2; e += blockDim.x) {
    const int t = e / n2, z = e - t * n2;
    const int kx = kx0 + t;
    cx Y0 = res[(0 * tx + t) * n2 + z], Y1 = res[(1 * tx + t) * n2 + z], Y2 = res[(2 * tx + t) * n2 + z];
    if (kx >= nkx) {
      Y0 = Y1 = Y2 = mk<R>((R)0, (R)0);
    } else {
      cplx X0 = cmk((double)Y0.x, (double)Y0.y), X1 = cmk((double)Y1.x, (double)Y1.y),
           X2 = cmk((double)Y2.x, (double)Y2.y);
      apply_curl(ph0, ph1, ph2, inv_nvox, inv4h, kx, ky, z, X0, X1, X2);
      Y0 = mk<R>((R)X0.x, (R)X0.y); Y1 = mk<R>((R)X1.x, (R)X1.y); Y2 = mk<R>((R)X2.x, (R)X2.y);
    }
    oth[(0 * tx + t) * n2 + z] = Y0;
    oth[(1 * tx + t) * n2 + z] = Y1;
    oth[(2 * tx + t) * n2 + z] = Y2;
  }
  __syncthreads();
  cx* res2 = block_fft<+1, R>(oth, res, pl, 3 * tx, tw);
  for (int e = threadIdx.x; e < cnt; e += blockDim.x) {
    const int c = e / (tx * n2);
    const int rem = e - c * tx * n2;
    const int z = rem / tx, t = rem - z * tx;
    const int kx = kx0 + t;
    if (kx < nkx) {
      const size_t f = 3 * i + c;
      cx v = res2[(c * tx + t) * n2 + z];
      spec[(f * n2 + z) * zstride + (size_t)ky * nkx + kx] = st2<R>(v.x, v.y);
    }
  }
}

// Tile sizes: as large as shared memory allows (up to 1024 complex per
// transform batch, 512 in the z pass that holds three fields), shrunk while
// the grid would fill less than four blocks per SM, down to 256 elements.

int rows_per_block(int n0, int n1, int n2, int nf, int fill) {
  int r = 1024 / n0;
  if (r < 1) r = 1;
  if (r > n1 / 2) r = n1 / 2;
  while (r > 1 && (n1 / 2) % r) --r;
  while (r > 1 && (long)(n1 / 2 / r) * n2 * nf < fill && r * n0 > 256) {
    int q = r / 2;
    while (q > 1 && (n1 / 2) % q) --q;
    r = q;
  }
  return r;
}
int tile_y(int n1, int n2, int nkx, int nf, int fill) {
  int t = 1024 / n1;
  if (t > 16) t = 16;
  if (t < 1) t = 1;
  while (t > 1 && (long)((nkx + t - 1) / t) * n2 * nf < fill && t * n1 > 256) t /= 2;
  return t;
}
int tile_z(int n1, int n2, int nkx, int nf, int fill) {
  int t = 512 / n2;
  if (t > 16) t = 16;
  if (t < 1) t = 1;
  while (t > 1 && (long)((nkx + t - 1) / t) * n1 * (nf / 3) < fill && 3 * t * n2 > 256) t /= 2;
  return t;
}
// threads for a block holding `elems` complex values: one per `per` values
// (the x and y passes: one butterfly of the plan's largest radix, its first
// pass, per thread; the z pass, whose tiles are narrow and few per SM, keeps
// one thread per four values for the warps that hide its latency)
int threads_for(int elems, int per) {
  int t = (elems / per + 31) / 32 * 32;
  return t < 64 ? 64 : (t > 256 ? 256 : t);
}
int first_radix(const FFTPlan& pl) { return pl.npass > 0 ? pl.radix[0] : 4; }

// radix passes 8 (X and Y), 4, 2, 3
FFTPlan plan_of(int n, int max_radix) {
  FFTPlan plan, *p = &plan;
  p->n = n;
  p->npass = 0;
  int m = n;
  while (max_radix >= 8 && m % 8 == 0) { p->radix[p->npass++] = 8; m /= 8; }
  while (m % 4 == 0) { p->radix[p->npass++] = 4; m /= 4; }
  if (m % 2 == 0) { p->radix[p->npass++] = 2; m /= 2; }
  while (m % 3 == 0) { p->radix[p->npass++] = 3; m /= 3; }
  return plan;
}


}  // namespace

cudaError_t launch_curl_fp64(const rve_s* h, const double* in, double* out, cudaStream_t s) {
  const FFTPlan px = plan_of(h->n0, 8), py = plan_of(h->n1, 8), pz = plan_of(h->n2, 4);
  const int nf = 9, fill = 8 * h->num_sms;
  const int rpb = rows_per_block(h->n0, h->n1, h->n2, nf, fill);
  const dim3 gx(h->n1 / 2 / rpb, h->n2, nf);
  const size_t shx = 2 * (size_t)rpb * h->n0 * sizeof(CX<double>);
  const int tx = threads_for(rpb * h->n0, first_radix(px));
  const int ty = tile_y(h->n1, h->n2, h->nkx, nf, fill);
  const dim3 gy((h->nkx + ty - 1) / ty, h->n2, nf);
  const size_t shy = 2 * (size_t)ty * h->n1 * sizeof(CX<double>);
  const int tyt = threads_for(ty * h->n1, first_radix(py));
  const int tz = tile_z(h->n1, h->n2, h->nkx, nf, 4 * h->num_sms);
  const dim3 gz((h->nkx + tz - 1) / tz, h->n1, nf / 3);
  const size_t shz = 2 * 3 * (size_t)tz * h->n2 * sizeof(CX<double>);
  {
    ProfScope ps_(h, RVE_K_FFT_CURL, s);
    k_fft_x_r2c<double><<<gx, tx, shx, s>>>(in, h->spec, h->n0, h->n1, h->n2, h->nkx, rpb, to_dev(px), h->ax[0].tw64);
  }
  {
    ProfScope ps_(h, RVE_K_FFT_CURL, s);
    k_fft_y<-1, double><<<gy, tyt, shy, s>>>(h->spec, h->n1, h->n2, h->nkx, ty, to_dev(py), h->ax[1].tw64);
  }
  {
    ProfScope ps_(h, RVE_K_FFT_CURL, s);
    k_fft_z_op<double><<<gz, threads_for(3 * tz * h->n2, 4), shz, s>>>(h->spec, h->n1, h->n2, h->nkx, tz, to_dev(pz),
                                                                      h->ax[2].tw64, h->ax[0].ph, h->ax[1].ph,
                                                                      h->ax[2].ph, 1.0 / (double)h->nvox, 0.25 / h->h);
  }
  {
    ProfScope ps_(h, RVE_K_FFT_CURL, s);
    k_fft_y<+1, double><<<gy, tyt, shy, s>>>(h->spec, h->n1, h->n2, h->nkx, ty, to_dev(py), h->ax[1].tw64);
  }
  {
    ProfScope ps_(h, RVE_K_FFT_CURL, s);
    k_fft_x_c2r<double><<<gx, tx, shx, s>>>(h->spec, out, h->n0, h->n1, h->n2, h->nkx, rpb, to_dev(px), h->ax[0].tw64);
  }
  return cudaGetLastError();
}
