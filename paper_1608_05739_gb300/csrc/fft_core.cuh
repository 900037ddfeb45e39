// fft_core.cuh -- register/shared-memory Stockham FFT building blocks for sm_103a.
//
// A length-L transform is computed by T = L/EPT threads; thread t holds the EPT
// elements x[t + T*m], m < EPT, in registers before and after the transform
// (natural order in both domains).  Lengths: powers of two 8..4096 with 8 or
// 16 elements per thread (a radix-2/4/8 first stage, then radix-EPT stages),
// 3 * 2^k, 48..3072, with 24 (radix 3, 6 or 12, then 8) or 12 (radix 12, then 2,
// then 4), or 5 * 2^k, 80..1280, with 20 (radix 10 or 20, then 4) -- FFTPlan
// below.  Between stages the data go
// through shared memory in rows of 16 elements whose columns are XOR-swizzled
// per exchange (free of bank conflicts for each stage's write pattern).
//
// Forward = Stockham decimation in time: stage (radix R, span Ns) multiplies
// input r of butterfly j by w^(r*k), w = exp(-2 pi i/(Ns R)), k = j mod Ns,
// applies the radix-R DFT and writes output r to (j - k) R + k + r Ns.
// Inverse = the exact adjoint of the forward (stages in reverse order, adjoint
// butterflies, conjugated twiddles), i.e. the unnormalised inverse DFT.  With
// the adjoint, a forward/inverse round trip deviates from N*I only through
// |w| != 1; in FP32 the twiddles and the sqrt(1/2) constant are therefore
// applied in compensated form (hi + lo parts, FMA), which keeps the round
// trip free of systematic gain over thousands of steps.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <utility>

#include "tc_dft.cuh"

namespace psatd {

// First statement of a pass launched with launch_pass (launch.h): wait for the passes
// before it (everything they wrote is visible then), and let the next one be scheduled.
// Before any allocation of tensor memory, so that a waiting pass holds none.
__device__ __forceinline__ void pass_begin() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <typename R> struct Types;
template <> struct Types<float> {
  typedef float2 C;   // complex value
  typedef float4 W;   // twiddle: (re_hi, im_hi, re_lo, im_lo)
  static constexpr bool kComp = true;
};
template <> struct Types<double> {
  typedef double2 C;
  typedef double2 W;  // twiddle: (re, im)
  static constexpr bool kComp = false;
};

// Two floats that go through the same arithmetic (the same element of two
// transforms), computed with the packed FP32 instructions: one instruction for
// both, each half rounded as the scalar operation, so a transform's bits do not
// depend on whether it ran in a pair.
struct alignas(8) F2 {
  float a, b;
};
struct alignas(16) C2 {  // complex pair: (re, re), (im, im)
  F2 x, y;
};
template <> struct Types<F2> {
  typedef C2 C;
  typedef float4 W;  // one twiddle serves both halves
  static constexpr bool kComp = true;
};
__device__ __forceinline__ float2 f2v(F2 v) { return make_float2(v.a, v.b); }
__device__ __forceinline__ F2 f2(float2 v) { return F2{v.x, v.y}; }
__device__ __forceinline__ F2 operator+(F2 a, F2 b) { return f2(__fadd2_rn(f2v(a), f2v(b))); }
// a - b as fma(b, -1, a): the product is exact, so this is the one rounding of a - b
__device__ __forceinline__ F2 operator-(F2 a, F2 b) {
  return f2(__ffma2_rn(f2v(b), make_float2(-1.f, -1.f), f2v(a)));
}
__device__ __forceinline__ F2 operator*(float s, F2 v) { return f2(__fmul2_rn(make_float2(s, s), f2v(v))); }
__device__ __forceinline__ F2 fma_s(F2 v, float s, F2 c) {
  return f2(__ffma2_rn(f2v(v), make_float2(s, s), f2v(c)));
}
__device__ __forceinline__ float fma_s(float v, float s, float c) { return fmaf(v, s, c); }
__device__ __forceinline__ double fma_s(double v, float s, double c) { return fma(v, (double)s, c); }

__device__ __forceinline__ float2 mkc(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ double2 mkc(double a, double b) { return make_double2(a, b); }
__device__ __forceinline__ C2 mkc(F2 a, F2 b) { return C2{a, b}; }

template <class C> __device__ __forceinline__ C cadd(C a, C b) { return mkc(a.x + b.x, a.y + b.y); }
template <class C> __device__ __forceinline__ C csub(C a, C b) { return mkc(a.x - b.x, a.y - b.y); }
template <class C> __device__ __forceinline__ C cmul_pi(C a) { return mkc(-a.y, a.x); }  // * (+i)
template <class C> __device__ __forceinline__ C cconj(C a) { return mkc(a.x, -a.y); }
// a +- i b (the rotation costs no operation, also in the packed type)
template <class C> __device__ __forceinline__ C add_i(C a, C b) { return mkc(a.x - b.y, a.y + b.x); }
template <class C> __device__ __forceinline__ C sub_i(C a, C b) { return mkc(a.x + b.y, a.y - b.x); }

// x * w, compensated: the low parts enter first, the leading product last.
__device__ __forceinline__ float2 twmul(float2 x, float4 w) {
  float re = fmaf(x.x, w.z, -x.y * w.w);
  float im = fmaf(x.x, w.w, x.y * w.z);
  re = fmaf(-x.y, w.y, re);
  im = fmaf(x.y, w.x, im);
  re = fmaf(x.x, w.x, re);
  im = fmaf(x.x, w.y, im);
  return make_float2(re, im);
}
// x * conj(w), compensated.
__device__ __forceinline__ float2 twmul_conj(float2 x, float4 w) {
  float re = fmaf(x.x, w.z, x.y * w.w);
  float im = fmaf(x.y, w.z, -x.x * w.w);
  re = fmaf(x.y, w.y, re);
  im = fmaf(-x.x, w.y, im);
  re = fmaf(x.x, w.x, re);
  im = fmaf(x.y, w.x, im);
  return make_float2(re, im);
}
// the same products in the packed type (term by term as above)
__device__ __forceinline__ C2 twmul(C2 x, float4 w) {
  F2 re = fma_s(x.x, w.z, -w.w * x.y);
  F2 im = fma_s(x.x, w.w, w.z * x.y);
  re = fma_s(x.y, -w.y, re);
  im = fma_s(x.y, w.x, im);
  re = fma_s(x.x, w.x, re);
  im = fma_s(x.x, w.y, im);
  return C2{re, im};
}
__device__ __forceinline__ C2 twmul_conj(C2 x, float4 w) {
  F2 re = fma_s(x.x, w.z, w.w * x.y);
  F2 im = fma_s(x.y, w.z, -w.w * x.x);
  re = fma_s(x.y, w.y, re);
  im = fma_s(x.x, -w.y, im);
  re = fma_s(x.x, w.x, re);
  im = fma_s(x.y, w.x, im);
  return C2{re, im};
}
__device__ __forceinline__ double2 twmul(double2 x, double2 w) {
  return make_double2(fma(x.x, w.x, -x.y * w.y), fma(x.x, w.y, x.y * w.x));
}
__device__ __forceinline__ double2 twmul_conj(double2 x, double2 w) {
  return make_double2(fma(x.x, w.x, x.y * w.y), fma(x.y, w.x, -x.x * w.y));
}

// v * sqrt(1/2); in float as hi + lo (0.70710677f + 1.2101617e-8f).
__device__ __forceinline__ float rsqrt2_mul(float v) { return fmaf(v, 0.70710677f, v * 1.2101617e-08f); }
__device__ __forceinline__ double rsqrt2_mul(double v) { return v * 0.70710678118654752440; }
__device__ __forceinline__ F2 rsqrt2_mul(F2 v) { return fma_s(v, 0.70710677f, 1.2101617e-08f * v); }
// v * -sqrt(1/2)
__device__ __forceinline__ float rsqrt2_mul_n(float v) { return fmaf(v, -0.70710677f, v * -1.2101617e-08f); }
__device__ __forceinline__ double rsqrt2_mul_n(double v) { return v * -0.70710678118654752440; }
__device__ __forceinline__ F2 rsqrt2_mul_n(F2 v) { return fma_s(v, -0.70710677f, -1.2101617e-08f * v); }

// ---------------------------------------------------------------- butterflies
// Radix-4 DFT in place (forward: exp(-2 pi i/4) = -i; adjoint: +i).  Exact
// operations apart from the additions, so the adjoint is exact.
template <bool ADJ, class C>
__device__ __forceinline__ void dft4_tail(C s0, C d0, C s1, C t, C& x0, C& x1, C& x2, C& x3) {
  x0 = cadd(s0, s1);
  x1 = ADJ ? add_i(d0, t) : sub_i(d0, t);
  x2 = csub(s0, s1);
  x3 = ADJ ? sub_i(d0, t) : add_i(d0, t);
}
template <bool ADJ, class C>
__device__ __forceinline__ void dft4(C& x0, C& x1, C& x2, C& x3) {
  dft4_tail<ADJ>(cadd(x0, x2), csub(x0, x2), cadd(x1, x3), csub(x1, x3), x0, x1, x2, x3);
}
// dft4 of (x0, x1, -+ i x2, x3) (forward -i, adjoint +i)
template <bool ADJ, class C>
__device__ __forceinline__ void dft4_r2(C& x0, C& x1, C& x2, C& x3) {
  dft4_tail<ADJ>(ADJ ? add_i(x0, x2) : sub_i(x0, x2), ADJ ? sub_i(x0, x2) : add_i(x0, x2), cadd(x1, x3),
                 csub(x1, x3), x0, x1, x2, x3);
}

// Radix-8 forward DFT, natural order in and out: split a_r +- a_(r+4), rotate
// the difference half by w8^r, two radix-4 DFTs interleaved.
template <class C>
__device__ __forceinline__ void dft8_fwd(C* a) {
  C b0 = cadd(a[0], a[4]), b1 = cadd(a[1], a[5]), b2 = cadd(a[2], a[6]), b3 = cadd(a[3], a[7]);
  C c0 = csub(a[0], a[4]), c1 = csub(a[1], a[5]), c2 = csub(a[2], a[6]), c3 = csub(a[3], a[7]);
  // c1 *= s(1 - i); c2 *= -i; c3 *= s(-1 - i) = (p, -q)
  c1 = mkc(rsqrt2_mul(c1.x + c1.y), rsqrt2_mul(c1.y - c1.x));
  const auto p = rsqrt2_mul(c3.y - c3.x), q = rsqrt2_mul(c3.x + c3.y);
  dft4<false>(b0, b1, b2, b3);
  dft4_tail<false>(sub_i(c0, c2), add_i(c0, c2), mkc(c1.x + p, c1.y - q), mkc(c1.x - p, c1.y + q), c0, c1, c2, c3);
  a[0] = b0; a[1] = c0; a[2] = b1; a[3] = c1;
  a[4] = b2; a[5] = c2; a[6] = b3; a[7] = c3;
}

// Exact adjoint of dft8_fwd (reverse order of its steps, conjugate constants).
template <class C>
__device__ __forceinline__ void dft8_adj(C* a) {
  C b0 = a[0], b1 = a[2], b2 = a[4], b3 = a[6];
  C c0 = a[1], c1 = a[3], c2 = a[5], c3 = a[7];
  dft4<true>(b0, b1, b2, b3);
  dft4<true>(c0, c1, c2, c3);
  // c1 *= s(1 + i); c2 *= +i; c3 *= s(-1 + i) = (-q, p)
  c1 = mkc(rsqrt2_mul(c1.x - c1.y), rsqrt2_mul(c1.x + c1.y));
  const auto q = rsqrt2_mul(c3.x + c3.y), p = rsqrt2_mul(c3.x - c3.y);
  a[0] = cadd(b0, c0); a[1] = cadd(b1, c1); a[2] = add_i(b2, c2); a[3] = mkc(b3.x - q, b3.y + p);
  a[4] = csub(b0, c0); a[5] = csub(b1, c1); a[6] = sub_i(b2, c2); a[7] = mkc(b3.x + q, b3.y - p);
}

// Multiplication by constants of the radix-16 DFT: z (p + i q) with p, q the
// double-precision values, applied as hi + lo pairs in float.
template <class C> struct KMul;
template <> struct KMul<float2> {
  template <int P_NUM>
  static __device__ __forceinline__ float2 mul(float2 z, double p, double q) {
    const float ph = (float)p, pl = (float)(p - (double)ph), qh = (float)q, ql = (float)(q - (double)qh);
    float re = z.x * pl;
    re = fmaf(-z.y, ql, re);
    re = fmaf(-z.y, qh, re);
    re = fmaf(z.x, ph, re);
    float im = z.x * ql;
    im = fmaf(z.y, pl, im);
    im = fmaf(z.y, ph, im);
    im = fmaf(z.x, qh, im);
    return make_float2(re, im);
  }
};
template <> struct KMul<C2> {
  template <int P_NUM>
  static __device__ __forceinline__ C2 mul(C2 z, double p, double q) {
    const float ph = (float)p, pl = (float)(p - (double)ph), qh = (float)q, ql = (float)(q - (double)qh);
    F2 re = pl * z.x;
    re = fma_s(z.y, -ql, re);
    re = fma_s(z.y, -qh, re);
    re = fma_s(z.x, ph, re);
    F2 im = ql * z.x;
    im = fma_s(z.y, pl, im);
    im = fma_s(z.y, ph, im);
    im = fma_s(z.x, qh, im);
    return C2{re, im};
  }
};
template <> struct KMul<double2> {
  template <int P_NUM>
  static __device__ __forceinline__ double2 mul(double2 z, double p, double q) {
    return make_double2(fma(z.x, p, -z.y * q), fma(z.x, q, z.y * p));
  }
};
constexpr double kCos8 = 0.92387953251128675613;  // cos(pi/8)
constexpr double kSin8 = 0.38268343236508977173;  // sin(pi/8)

// z * w16^e (forward, w16 = exp(-2 pi i/16)) or z * conj(w16^e) (adjoint), e in {1,2,3,6,9}
// (e = 4, the rotation by -+i, is part of dft4_r2)
template <int E, bool ADJ, class C>
__device__ __forceinline__ C w16mul(C z) {
  constexpr double sg = ADJ ? 1.0 : -1.0;  // sign of the imaginary part of the constant
  if constexpr (E == 1) return KMul<C>::template mul<1>(z, kCos8, sg * kSin8);
  else if constexpr (E == 3) return KMul<C>::template mul<3>(z, kSin8, sg * kCos8);
  else if constexpr (E == 9) return KMul<C>::template mul<1>(z, -kCos8, -sg * kSin8);
  else if constexpr (E == 2) {
    if constexpr (ADJ) return mkc(rsqrt2_mul(z.x - z.y), rsqrt2_mul(z.x + z.y));
    else return mkc(rsqrt2_mul(z.x + z.y), rsqrt2_mul(z.y - z.x));
  } else {  // E == 6
    if constexpr (ADJ) return mkc(rsqrt2_mul_n(z.x + z.y), rsqrt2_mul(z.x - z.y));
    else return mkc(rsqrt2_mul(z.y - z.x), rsqrt2_mul_n(z.x + z.y));
  }
}

// Radix-16 forward DFT, natural order in and out: 4 x 4 decomposition
// (radix-4 DFTs over the stride-4 columns, twiddles w16^(r1 k2), radix-4 DFTs
// over the rows, transposed read-out).
template <class C>
__device__ __forceinline__ void dft16_fwd(C* a) {
#pragma unroll
  for (int r1 = 0; r1 < 4; ++r1) dft4<false>(a[r1], a[r1 + 4], a[r1 + 8], a[r1 + 12]);
  a[5] = w16mul<1, false>(a[5]);
  a[9] = w16mul<2, false>(a[9]);
  a[13] = w16mul<3, false>(a[13]);
  a[6] = w16mul<2, false>(a[6]);
  a[14] = w16mul<6, false>(a[14]);
  a[7] = w16mul<3, false>(a[7]);
  a[11] = w16mul<6, false>(a[11]);
  a[15] = w16mul<9, false>(a[15]);
#pragma unroll
  for (int k2 = 0; k2 < 4; ++k2) {
    if (k2 == 2) dft4_r2<false>(a[8], a[9], a[10], a[11]);
    else dft4<false>(a[4 * k2], a[4 * k2 + 1], a[4 * k2 + 2], a[4 * k2 + 3]);
  }
  C y[16];
#pragma unroll
  for (int k2 = 0; k2 < 4; ++k2)
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) y[k2 + 4 * k1] = a[4 * k2 + k1];
#pragma unroll
  for (int i = 0; i < 16; ++i) a[i] = y[i];
}

// Exact adjoint of dft16_fwd.
template <class C>
__device__ __forceinline__ void dft16_adj(C* a) {
  C x[16];
#pragma unroll
  for (int k2 = 0; k2 < 4; ++k2)
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) x[4 * k2 + k1] = a[k2 + 4 * k1];
#pragma unroll
  for (int k2 = 0; k2 < 4; ++k2) dft4<true>(x[4 * k2], x[4 * k2 + 1], x[4 * k2 + 2], x[4 * k2 + 3]);
  x[5] = w16mul<1, true>(x[5]);
  x[9] = w16mul<2, true>(x[9]);
  x[13] = w16mul<3, true>(x[13]);
  x[6] = w16mul<2, true>(x[6]);
  x[14] = w16mul<6, true>(x[14]);
  x[7] = w16mul<3, true>(x[7]);
  x[11] = w16mul<6, true>(x[11]);
  x[15] = w16mul<9, true>(x[15]);
#pragma unroll
  for (int r1 = 0; r1 < 4; ++r1) {
    if (r1 == 2) dft4_r2<true>(x[2], x[6], x[10], x[14]);
    else dft4<true>(x[r1], x[r1 + 4], x[r1 + 8], x[r1 + 12]);
  }
#pragma unroll
  for (int i = 0; i < 16; ++i) a[i] = x[i];
}

// v * sqrt(3)/2; in float as hi + lo
constexpr double kHalfSqrt3 = 0.86602540378443864676;
__device__ __forceinline__ float r3_mul(float v) {
  constexpr float h = (float)kHalfSqrt3, l = (float)(kHalfSqrt3 - (double)(float)kHalfSqrt3);
  return fmaf(v, h, v * l);
}
__device__ __forceinline__ double r3_mul(double v) { return v * kHalfSqrt3; }
__device__ __forceinline__ F2 r3_mul(F2 v) {
  constexpr float h = (float)kHalfSqrt3, l = (float)(kHalfSqrt3 - (double)(float)kHalfSqrt3);
  return fma_s(v, h, l * v);
}

// Radix-3 DFT in place (forward: exp(-2 pi i/3) = -1/2 - i sqrt3/2; adjoint:
// the conjugate constant): X0 = a0 + (a1 + a2), X1,2 = a0 - (a1 + a2)/2 -+ i
// sqrt3/2 (a1 - a2) (forward), +- (adjoint).
template <bool ADJ, class C>
__device__ __forceinline__ void dft3(C& a0, C& a1, C& a2) {
  const C t = cadd(a1, a2), d = csub(a1, a2);
  const C m = mkc(fma_s(t.x, -0.5f, a0.x), fma_s(t.y, -0.5f, a0.y));
  const C s = mkc(r3_mul(d.x), r3_mul(d.y));
  a0 = cadd(a0, t);
  a1 = ADJ ? add_i(m, s) : sub_i(m, s);
  a2 = ADJ ? sub_i(m, s) : add_i(m, s);
}

// Radix-5 DFT in place.  With t1 = a1 + a4, t2 = a2 + a3, t3 = a1 - a4,
// t4 = a2 - a3 and c_j = cos(2 pi j/5), s_j = sin(2 pi j/5):
//   X0 = a0 + t1 + t2,  m1 = a0 + c1 t1 + c2 t2,  m2 = a0 + c2 t1 + c1 t2,
//   n1 = s1 t3 + s2 t4,  n2 = s2 t3 - s1 t4,
//   forward (W = exp(-2 pi i/5)): X1,4 = m1 -+ i n1, X2,3 = m2 -+ i n2;
//   adjoint (the conjugate constants): X1,4 = m1 +- i n1, X2,3 = m2 +- i n2.
// The four constants multiply as hi + lo pairs in float.
constexpr double kC51 = 0.30901699437494742410;   // cos(2 pi/5)
constexpr double kC52 = -0.80901699437494742410;  // cos(4 pi/5)
constexpr double kS51 = 0.95105651629515357212;   // sin(2 pi/5)
constexpr double kS52 = 0.58778525229247312917;   // sin(4 pi/5)
template <int K> __device__ __forceinline__ float k5_mul(float v) {
  constexpr double c = K == 0 ? kC51 : K == 1 ? kC52 : K == 2 ? kS51 : kS52;
  constexpr float h = (float)c, l = (float)(c - (double)(float)c);
  return fmaf(v, h, v * l);
}
template <int K> __device__ __forceinline__ F2 k5_mul(F2 v) {
  constexpr double c = K == 0 ? kC51 : K == 1 ? kC52 : K == 2 ? kS51 : kS52;
  constexpr float h = (float)c, l = (float)(c - (double)(float)c);
  return fma_s(v, h, l * v);
}
template <int K> __device__ __forceinline__ double k5_mul(double v) {
  return v * (K == 0 ? kC51 : K == 1 ? kC52 : K == 2 ? kS51 : kS52);
}
template <bool ADJ, class C>
__device__ __forceinline__ void dft5(C* a) {
  const C t1 = cadd(a[1], a[4]), t2 = cadd(a[2], a[3]), t3 = csub(a[1], a[4]), t4 = csub(a[2], a[3]);
  const C m1 = mkc(a[0].x + k5_mul<0>(t1.x) + k5_mul<1>(t2.x), a[0].y + k5_mul<0>(t1.y) + k5_mul<1>(t2.y));
  const C m2 = mkc(a[0].x + k5_mul<1>(t1.x) + k5_mul<0>(t2.x), a[0].y + k5_mul<1>(t1.y) + k5_mul<0>(t2.y));
  const C n1 = mkc(k5_mul<2>(t3.x) + k5_mul<3>(t4.x), k5_mul<2>(t3.y) + k5_mul<3>(t4.y));
  const C n2 = mkc(k5_mul<3>(t3.x) - k5_mul<2>(t4.x), k5_mul<3>(t3.y) - k5_mul<2>(t4.y));
  a[0] = cadd(a[0], cadd(t1, t2));
  a[1] = ADJ ? add_i(m1, n1) : sub_i(m1, n1);
  a[4] = ADJ ? sub_i(m1, n1) : add_i(m1, n1);
  a[2] = ADJ ? add_i(m2, n2) : sub_i(m2, n2);
  a[3] = ADJ ? sub_i(m2, n2) : add_i(m2, n2);
}

// DFT of N1 * N2 points in place, natural order in and out, N1 and N2 coprime, as the
// prime-factor (Good-Thomas) split: with n = (N2 n1 + N1 n2) mod N and k the residue
// with k = k1 mod N1, k = k2 mod N2, W_N^(n k) = W_N1^(n1 k1) W_N2^(n2 k2) where N2 k1 =
// k mod N1 and N1 k2 = k mod N2 fold into the index maps below, so the DFTs over n1 and
// n2 need no twiddles between them.  k = (K1 k1 + K2 k2) mod N with K1 = 1 mod N1, 0 mod
// N2 and K2 = 0 mod N1, 1 mod N2, for (N1, N2): (2, 3), (4, 3), (2, 5), (4, 5).  The adjoint
// runs the same steps in reverse order with the conjugate DFTs.
template <int N, bool ADJ, class C>
__device__ __forceinline__ void dft_small(C* a) {
  if constexpr (N == 2) {
    const C s = cadd(a[0], a[1]), d = csub(a[0], a[1]);
    a[0] = s;
    a[1] = d;
  } else if constexpr (N == 3) {
    dft3<ADJ>(a[0], a[1], a[2]);
  } else if constexpr (N == 4) {
    dft4<ADJ>(a[0], a[1], a[2], a[3]);
  } else {
    dft5<ADJ>(a);
  }
}
template <int N1, int N2, bool ADJ, class C>
__device__ __forceinline__ void dft_pfa(C* a) {
  constexpr int N = N1 * N2;
  constexpr int K1 = N2 == 3 ? (N1 == 2 ? 3 : 9) : 5;             // 1 mod N1, 0 mod N2
  constexpr int K2 = N2 == 3 ? 4 : (N1 == 2 ? 6 : 16);            // 0 mod N1, 1 mod N2
  static_assert(K1 % N1 == 1 && K1 % N2 == 0 && K2 % N1 == 0 && K2 % N2 == 1, "index maps");
  C y[N];  // y[n1 * N2 + k2]
  if constexpr (!ADJ) {
#pragma unroll
    for (int n1 = 0; n1 < N1; ++n1) {
      C c[N2];
#pragma unroll
      for (int n2 = 0; n2 < N2; ++n2) c[n2] = a[(N2 * n1 + N1 * n2) % N];
      dft_small<N2, false>(c);
#pragma unroll
      for (int k2 = 0; k2 < N2; ++k2) y[n1 * N2 + k2] = c[k2];
    }
#pragma unroll
    for (int k2 = 0; k2 < N2; ++k2) {
      C d[N1];
#pragma unroll
      for (int n1 = 0; n1 < N1; ++n1) d[n1] = y[n1 * N2 + k2];
      dft_small<N1, false>(d);
#pragma unroll
      for (int k1 = 0; k1 < N1; ++k1) a[(K1 * k1 + K2 * k2) % N] = d[k1];
    }
  } else {
#pragma unroll
    for (int k2 = 0; k2 < N2; ++k2) {
      C d[N1];
#pragma unroll
      for (int k1 = 0; k1 < N1; ++k1) d[k1] = a[(K1 * k1 + K2 * k2) % N];
      dft_small<N1, true>(d);
#pragma unroll
      for (int n1 = 0; n1 < N1; ++n1) y[n1 * N2 + k2] = d[n1];
    }
#pragma unroll
    for (int n1 = 0; n1 < N1; ++n1) {
      C c[N2];
#pragma unroll
      for (int k2 = 0; k2 < N2; ++k2) c[k2] = y[n1 * N2 + k2];
      dft_small<N2, true>(c);
#pragma unroll
      for (int n2 = 0; n2 < N2; ++n2) a[(N2 * n1 + N1 * n2) % N] = c[n2];
    }
  }
}

template <int RS, bool ADJ, class C>
__device__ __forceinline__ void butterfly(C* a) {
  if constexpr (RS == 3) {
    dft3<ADJ>(a[0], a[1], a[2]);
  } else if constexpr (RS == 5) {
    dft5<ADJ>(a);
  } else if constexpr (RS == 6) {
    dft_pfa<2, 3, ADJ>(a);
  } else if constexpr (RS == 12) {
    dft_pfa<4, 3, ADJ>(a);
  } else if constexpr (RS == 10) {
    dft_pfa<2, 5, ADJ>(a);
  } else if constexpr (RS == 20) {
    dft_pfa<4, 5, ADJ>(a);
  } else if constexpr (RS == 2) {
    dft_small<2, ADJ>(a);
  } else if constexpr (RS == 4) {
    dft4<ADJ>(a[0], a[1], a[2], a[3]);
  } else if constexpr (RS == 8) {
    if constexpr (ADJ) dft8_adj(a); else dft8_fwd(a);
  } else {
    if constexpr (ADJ) dft16_adj(a); else dft16_fwd(a);
  }
}

// ---------------------------------------------------------------- stage plan
__host__ __device__ constexpr int ilog2(int v) { return v <= 1 ? 0 : 1 + ilog2(v >> 1); }

__host__ __device__ constexpr bool is_pow2(int v) { return v > 0 && (v & (v - 1)) == 0; }

// Transposing passes: 16 elements per thread; 5 * 2^k lengths 20; 3 * 2^k lengths 12 up
// to 384 points, where 24 (one exchange fewer, but half the warps: 230 registers a
// thread) measured slower (192^3 y forward 121 -> 109 us, inverse 72.1 -> 66.1; the FP32
// batch of 512 patches 10.1 -> 9.4 ms per four steps), and 24 beyond (1536 points: 121
// us, with 12 131; 768 points: 19.0, with 12 20.6).  The fused pass takes 12 for 3 * 2^k.
__host__ __device__ constexpr int odd_factor(int v) { return is_pow2(v) ? 1 : (v % 3 == 0 ? 3 : 5); }
// FP64 takes as few as fit its threads, 4 up to 1024 points: radix-4 butterflies need no more
// operations per level than radix 16 (their twiddle products come on top), and at 2 FP64 operations per cycle and SM (half an
// operation per scheduler, so 64 cycles per warp instruction) a small grid's time is
// the instructions of one thread (x forward of 128^2, 6 components: 22.6 us with 16
// elements per thread); the extra exchanges cost a tenth of that.  Large 3D grids, whose
// passes keep the FP64 units busy, run 128- and 256-point rows with 16 all the same (row_wide;
// a third of the twiddle products: 256 x 128 x 128 J-form, x forward 1072 -> 980 us, y forward
// 833 -> 737, y inverse 552 -> 487, x inverse 748 -> 639).
__host__ __device__ constexpr int row_ept(int L, bool f32) {
  return !f32 ? (L <= 1024 ? 4 : L / 256) : odd_factor(L) == 3 ? (L <= 384 ? 12 : 24) : odd_factor(L) == 5 ? 20 : L >= 16 ? 16 : 8;
}
// lengths that also have a 16-element variant
__host__ __device__ constexpr bool row_wide(int L, bool f32) { return !f32 && (L == 128 || L == 256); }
template <int L, typename R = float>
struct RowEPT { static constexpr int value = row_ept(L, sizeof(R) == 4); };
// Elements per thread of the fused pass by default.  8 (radix-8 stages) up to 512
// points; 16 (radix-16 stages) from 1024 points on in FP32, where they save an
// exchange and a quarter of the shared-memory traffic and component groups make
// up for the threads (2048 points TE: 75.7 us with 8, 73.1 us with 16 and two
// groups; 1024 points, eleven components: 0.968 / 0.884 ms; 512 points: 12.2 /
// 18.5 us), and in the tensor-core variant (TC), whose stages are radix-16
// DFT-matrix contractions.
__host__ __device__ constexpr int push_ept(int L, bool tc, bool f32) {
  return odd_factor(L) == 3 ? 12 : odd_factor(L) == 5 ? 20 : (tc || (f32 && L >= 1024)) ? 16 : 8;
}
// Elements per thread that the fused pass's kernel runs for a plan's choice `ept` on grids of
// nlines lines: in FP64 the radix-8 schedule runs as radix-4 stages of 4 elements up to 128
// points (as many operations per level, half of them per thread: see row_ept; a step of 128^2
// TE 59 -> 31 us, six components 47 -> 31), while a line stays one warp (256^2 TE 60 -> 69 us)
// and, at 128 points, the grid leaves the schedulers idle (128^3 1902 -> 1918 us; 64 points,
// 128 x 128 x 64: 956 -> 931 us).
__host__ __device__ constexpr int push_kernel_ept(int L, int ept, bool f32, int64_t nlines) {
  return !f32 && ept == 8 && (L <= 64 || (L == 128 && nlines * (L / 8) < 256 * 152)) ? 4 : ept;
}

// Whether the fused pass takes the six 2D components as two sets, each a block of its own
// (pair_push.cuh): FP32 always; FP64, bound by its units, while every block has an SM to
// itself (128^2 30.7 -> 26.7 us a step; 2048 x 256 479 -> 497).
constexpr bool push_sets(bool f32, int64_t blocks) { return f32 || 2 * blocks <= 152; }

// Power-of-two L: a radix-2/4/8 first stage when log2 L is not a multiple of
// log2 EPT, then radix-EPT stages.  Mixed lengths take the odd factor and a power of
// two in a prime-factor first stage (no twiddles inside it).  L = 3 * 2^k: with EPT =
// 24 radix 3, 6 or 12, then radix-8 stages (two exchanges at 384 and 768 points, one
// at 48 and 96; as radix 3, (2 | 4), 8, .. they had one more); with EPT = 12 radix 12,
// a radix-2 stage when k is odd, then radix-4 stages.  L = 5 * 2^k (EPT = 20): radix
// 10 or 20, then radix-4 stages.  Every radix divides EPT.
template <int L, int EPT = 8>
struct FFTPlan {
  static constexpr int kEPT = EPT;
  static constexpr int kF = odd_factor(L);  // 1, 3 or 5
  static constexpr bool kMixed = kF > 1;
  static constexpr int kLog = ilog2(L / kF);  // log2 of the power-of-two part
  static constexpr int kB = kF == 5 ? 2 : kMixed ? (EPT == 12 ? 2 : 3) : ilog2(EPT);
  // power of two taken by the first stage of a mixed length (prime-factor DFTs: 3 * 2^h, 5 * 2^h)
  static constexpr int kHeadLog = !kMixed ? 0 : EPT == 12 ? 2 : kF == 5 ? (kLog % 2 ? 1 : 2) : kLog % 3;
  static constexpr int kRem = (kLog - kHeadLog) % kB;
  static constexpr int kR0 = kMixed ? kF << kHeadLog : kRem ? (1 << kRem) : EPT;
  static constexpr int kStages = kMixed ? 1 + (kRem ? 1 : 0) + (kLog - kHeadLog) / kB
                                        : kRem ? kLog / kB + 1 : kLog / kB;
  static constexpr int kT = L / EPT;
  static constexpr int kBuf = L;  // exchange buffer (XOR-swizzled, no padding)
  __host__ __device__ static constexpr int radix(int s) {
    if (kMixed) return s == 0 ? kR0 : (s == 1 && kRem) ? (1 << kRem) : (1 << kB);
    return s == 0 ? kR0 : EPT;
  }
  __host__ __device__ static constexpr int span(int s) {  // Ns of stage s
    int ns = 1;
    for (int i = 0; i < s; ++i) ns *= radix(i);
    return ns;
  }
  // offset of stage s's twiddle block in the stage table (stages s >= 1)
  __host__ __device__ static constexpr int tw_off(int s) {
    int o = 0;
    for (int i = 1; i < s; ++i) o += (radix(i) - 1) * span(i);
    return o;
  }
  // entries of the stage table: sum over s >= 1 of (R_s - 1) Ns_s = L - R_0
  static constexpr int kTwEntries = L - kR0;
  // XOR multiplier of the exchange written by stage s (bank-conflict free for
  // the Stockham write pattern of that stage and the contiguous reads after it)
  __host__ __device__ static constexpr int swz(int s) {
    return (kMixed || EPT == 16) ? 1 : (span(s) == 1 ? 1 : 10);
  }
  // swizzle of the last exchange: forward output / inverse input positions
  // sw<kLastCX>(t + T m) are each touched by their own thread only
  static constexpr int kLastCX = (kStages >= 2) ? swz(kStages - 2) : 0;
  static_assert(kF == 3   ? (L == 3 * (1 << kLog) && (EPT == 24 || EPT == 12) && kLog >= 4)
                : kF == 5 ? (L == 5 * (1 << kLog) && EPT == 20 && kLog >= 4)
                          : (L >= EPT && EPT != 24 && EPT != 12 && EPT != 20),
                "L must be a power of two >= EPT, 3 * 2^k (k >= 4) with EPT = 12 or 24, or 5 * 2^k with EPT 20");
};

// element i of an exchange buffer, rows of 16 elements (128 B) XOR-swizzled
template <int CX>
__device__ __forceinline__ int sw(int i) { return i ^ (((i >> 4) * CX) & 15); }

// Two exchange buffers used alternately: consecutive exchanges never share a
// buffer, so one barrier per exchange suffices.  `twslot` is a shared-memory
// word holding the twiddle table's address (written before the kernel's first
// barrier): each stage reads it back, which ties that stage's twiddle loads to
// the stage (the compiler cannot prefetch every stage's twiddles of every
// transform in a kernel into registers).
// With b[0] == b[1] (one buffer, `single`), next() adds the barrier that lets
// the previous exchange's reads finish before the buffer is overwritten.
// The exchange barrier: the whole CTA (bar_n == 0), or, when each line's
// transform is private to its own warps, the named barrier bar_id over the
// line's bar_n threads (a multiple of 32), so that lines do not wait for one
// another between stages.
template <class C>
struct ExBuf {
  C* b[2];
  int cur;
  const void* const* twslot;
  bool single;
  int bar_id = 0;
  int bar_n = 0;
  __device__ __forceinline__ void sync() const {
    if (bar_n) asm volatile("bar.sync %0, %1;" ::"r"(bar_id), "r"(bar_n) : "memory");
    else __syncthreads();
  }
  __device__ __forceinline__ C* next() {
    C* p = b[cur];
    cur ^= 1;
    if (single) sync();
    return p;
  }
};

template <typename R, class C>
__device__ __forceinline__ const typename Types<R>::W* stage_tw(const ExBuf<C>& ex) {
  return reinterpret_cast<const typename Types<R>::W*>(
      const_cast<const void*>(*reinterpret_cast<const void* const volatile*>(ex.twslot)));
}

// Twiddle tables of a length-L transform (built in tables.cu): stage s >= 1
// keeps W_L^(r k L/(Ns R)) at [tw_off(s) + (r-1) Ns + k], k < Ns, 1 <= r < R,
// so the threads of a warp read consecutive entries.

// One forward stage.
template <typename R, int L, int EPT, int S, int TC>
__device__ __forceinline__ void fwd_stage(typename Types<R>::C (&v)[EPT], ExBuf<typename Types<R>::C>& ex,
                                          const typename Types<R>::W* __restrict__ tw, int t, TcCtx* tc) {
  typedef typename Types<R>::C C;
  typedef FFTPlan<L, EPT> P;
  constexpr int RS = P::radix(S), NS = P::span(S), Q = EPT / RS, T = P::kT;
  constexpr bool LAST = (S == P::kStages - 1);
  constexpr int CX = P::swz(S);
  C* buf = nullptr;
  if constexpr (!LAST) buf = ex.next();
  asm volatile("" : "+r"(t)::"memory");  // stage boundary for the front end
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const int j = t + q * T;
    const int k = is_pow2(NS) ? (j & (NS - 1)) : (int)((unsigned)j % (unsigned)NS);
    C a[RS];
#pragma unroll
    for (int r = 0; r < RS; ++r) a[r] = v[q + r * Q];
    if constexpr (NS > 1) {
      const typename Types<R>::W* tws = stage_tw<R>(ex) + P::tw_off(S) + k;
#pragma unroll
      for (int r = 1; r < RS; ++r) a[r] = twmul(a[r], __ldg(&tws[(r - 1) * NS]));
    }
    if constexpr (TC && RS == 16) tc_dft<16, false, TC == 2>(a, *tc);
    else butterfly<RS, false>(a);
    if constexpr (LAST) {
#pragma unroll
      for (int r = 0; r < RS; ++r) v[q + r * Q] = a[r];
    } else {
      const int base = (j - k) * RS + k;
#pragma unroll
      for (int r = 0; r < RS; ++r) buf[sw<CX>(base + r * NS)] = a[r];
    }
  }
  if constexpr (!LAST) {
    ex.sync();
#pragma unroll
    for (int m = 0; m < EPT; ++m) v[m] = buf[sw<CX>(t + T * m)];
  }
}

// Adjoint of fwd_stage<S>.
template <typename R, int L, int EPT, int S, int TC>
__device__ __forceinline__ void inv_stage(typename Types<R>::C (&v)[EPT], ExBuf<typename Types<R>::C>& ex,
                                          const typename Types<R>::W* __restrict__ tw, int t, TcCtx* tc) {
  typedef typename Types<R>::C C;
  typedef FFTPlan<L, EPT> P;
  constexpr int RS = P::radix(S), NS = P::span(S), Q = EPT / RS, T = P::kT;
  constexpr bool FIRST = (S == P::kStages - 1);
  constexpr int CX = P::swz(S);
  C* buf = nullptr;
  if constexpr (!FIRST) {
    buf = ex.next();
#pragma unroll
    for (int m = 0; m < EPT; ++m) buf[sw<CX>(t + T * m)] = v[m];
    ex.sync();
  }
  asm volatile("" : "+r"(t)::"memory");  // stage boundary (see fwd_stage)
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const int j = t + q * T;
    const int k = is_pow2(NS) ? (j & (NS - 1)) : (int)((unsigned)j % (unsigned)NS);
    C a[RS];
    if constexpr (FIRST) {
#pragma unroll
      for (int r = 0; r < RS; ++r) a[r] = v[q + r * Q];
    } else {
      const int base = (j - k) * RS + k;
#pragma unroll
      for (int r = 0; r < RS; ++r) a[r] = buf[sw<CX>(base + r * NS)];
    }
    if constexpr (TC && RS == 16) tc_dft<16, true, TC == 2>(a, *tc);
    else butterfly<RS, true>(a);
    if constexpr (NS > 1) {
      const typename Types<R>::W* tws = stage_tw<R>(ex) + P::tw_off(S) + k;
#pragma unroll
      for (int r = 1; r < RS; ++r) a[r] = twmul_conj(a[r], __ldg(&tws[(r - 1) * NS]));
    }
#pragma unroll
    for (int r = 0; r < RS; ++r) v[q + r * Q] = a[r];
  }
}

// Twiddles of one stage per thread (fft_line.cuh): the most over the stages.
template <int L, int EPT>
struct PFCount {
  typedef FFTPlan<L, EPT> P;
  static constexpr int at(int s) { return s >= 1 && s < P::kStages ? (EPT / P::radix(s)) * (P::radix(s) - 1) : 0; }
  static constexpr int max_from(int s) { return s >= P::kStages ? 1 : (at(s) > max_from(s + 1) ? at(s) : max_from(s + 1)); }
  static constexpr int value = max_from(1);
};

template <typename R, int L, int EPT, int TC, int... S>
__device__ __forceinline__ void fft_fwd_seq(typename Types<R>::C (&v)[EPT], ExBuf<typename Types<R>::C>& ex,
                                            const typename Types<R>::W* tw, int t, TcCtx* tc,
                                            std::integer_sequence<int, S...>) {
  (fwd_stage<R, L, EPT, S, TC>(v, ex, tw, t, tc), ...);
}
template <typename R, int L, int EPT, int TC, int... S>
__device__ __forceinline__ void fft_inv_seq(typename Types<R>::C (&v)[EPT], ExBuf<typename Types<R>::C>& ex,
                                            const typename Types<R>::W* tw, int t, TcCtx* tc,
                                            std::integer_sequence<int, S...>) {
  (inv_stage<R, L, EPT, FFTPlan<L, EPT>::kStages - 1 - S, TC>(v, ex, tw, t, tc), ...);
}

// Forward DFT of length L: v holds x[t + T m] on entry, X[t + T m] on exit
// (T = L/EPT, m < EPT).  Every thread of the block must call it (block-wide
// barriers inside); the exchanges alternate between the two buffers of `ex`.
// TC: the radix-16 stages run on the tensor cores (tc_dft.cuh, context *tc):
// 1 split-FP16, 2 split-BF16.
template <typename R, int L, int EPT, int TC = 0>
__device__ __forceinline__ void block_fft_fwd(typename Types<R>::C (&v)[EPT], ExBuf<typename Types<R>::C>& ex,
                                              const typename Types<R>::W* tw, int t, TcCtx* tc = nullptr) {
  static_assert(!TC || sizeof(R) == 4, "tensor-core stages take float data");
  fft_fwd_seq<R, L, EPT, TC>(v, ex, tw, t, tc, std::make_integer_sequence<int, FFTPlan<L, EPT>::kStages>{});
}
// Unnormalised inverse DFT (adjoint of block_fft_fwd).
template <typename R, int L, int EPT, int TC = 0>
__device__ __forceinline__ void block_fft_inv(typename Types<R>::C (&v)[EPT], ExBuf<typename Types<R>::C>& ex,
                                              const typename Types<R>::W* tw, int t, TcCtx* tc = nullptr) {
  static_assert(!TC || sizeof(R) == 4, "tensor-core stages take float data");
  fft_inv_seq<R, L, EPT, TC>(v, ex, tw, t, tc, std::make_integer_sequence<int, FFTPlan<L, EPT>::kStages>{});
}

}  // namespace psatd
