// gp_split.cuh -- FP64 increments on the FP32 pipe.
//
// GB300 retires 2 FP64 lane operations per clock and SM and 128 FP32 ones (measured: a
// DADD, a DFMA and every conversion between FP64 and FP32 or integers take 1.7-2.0
// lanes per clock; FADD / FFMA / IADD about 121-124).  Each substep of a time step
// changes a value by a small increment, u = v + c with |c| << |v|, so the FP64 sweeps
// form c as an unevaluated sum of two FP32 numbers (about 48 bits of c) and add it to
// the FP64 v with one DADD.  Everything here works on two values at a time (f32x2
// instructions: one issue slot for two lanes' arithmetic).
//
// Increments are carried times 2^kSplitShift, so that FP32's exponent range covers
// values from 2^-150 (below: the increments lose bits, and vanish under 2^-182) up to 2^67 in
// modulus.  Larger or non-finite values are the caller's to detect (split3's tmax), and so are
// fields that are small as a whole (kIncTiny in gp_sweeps64.cu); both go through FP64.
//
// The error-free transformations are the published ones: TwoSum (Knuth, The Art of
// Computer Programming 2, 4.2.2) and the FMA product residual; every operation is an
// explicitly rounded one, so no contraction changes them.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define GP_HD __host__ __device__ __forceinline__
#else
#include <cmath>
#include <cstring>
#define GP_HD inline
struct float2 {
  float x, y;
};
#endif

namespace gpk {

constexpr int kSplitShift = 56;
// FP64 exponent field minus kSplitOff is the FP32 exponent field of v 2^kSplitShift
constexpr int kSplitOff = (1023 - 127 - kSplitShift) << 20;
constexpr int kSplitOff1 = (1023 - 127) << 20;   // of v itself
// split3's tmax from which the value is too large (FP32 exponent field 250)
constexpr int kSplitTooBig = 250 << 20;

// ------------------------------------------------------------ two-lane FP32

GP_HD float2 f2(float a) {
  float2 r;
  r.x = a;
  r.y = a;
  return r;
}
GP_HD float2 f2(float a, float b) {
  float2 r;
  r.x = a;
  r.y = b;
  return r;
}
GP_HD float2 add2(float2 a, float2 b) {
#ifdef __CUDA_ARCH__
  return __fadd2_rn(a, b);
#else
  return f2(a.x + b.x, a.y + b.y);
#endif
}
GP_HD float2 mul2(float2 a, float2 b) {
#ifdef __CUDA_ARCH__
  return __fmul2_rn(a, b);
#else
  return f2(a.x * b.x, a.y * b.y);
#endif
}
GP_HD float2 fma2(float2 a, float2 b, float2 c) {
#ifdef __CUDA_ARCH__
  return __ffma2_rn(a, b, c);
#else
  return f2(std::fma(a.x, b.x, c.x), std::fma(a.y, b.y, c.y));
#endif
}
GP_HD float2 neg2(float2 a) { return f2(-a.x, -a.y); }
// a - b as b (-1) + a, the same rounding: a negated operand of a two-lane add costs two
// extra instructions, the constant -1 none
GP_HD float2 sub2(float2 a, float2 b) { return fma2(b, f2(-1.f), a); }

GP_HD float bits_f(uint32_t u) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(u);
#else
  float f;
  memcpy(&f, &u, 4);
  return f;
#endif
}
GP_HD uint32_t f_bits(float f) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(f);
#else
  uint32_t u;
  memcpy(&u, &f, 4);
  return u;
#endif
}
GP_HD void words(double v, uint32_t* hi, uint32_t* lo) {
#ifdef __CUDA_ARCH__
  *hi = (uint32_t)__double2hiint(v);
  *lo = (uint32_t)__double2loint(v);
#else
  uint64_t w;
  memcpy(&w, &v, 8);
  *hi = (uint32_t)(w >> 32);
  *lo = (uint32_t)w;
#endif
}
GP_HD double from_words(uint32_t hi, uint32_t lo) {
#ifdef __CUDA_ARCH__
  return __hiloint2double((int)hi, (int)lo);
#else
  const uint64_t w = ((uint64_t)hi << 32) | lo;
  double v;
  memcpy(&v, &w, 8);
  return v;
#endif
}
GP_HD int round_int(float x) {
#ifdef __CUDA_ARCH__
  return __float2int_rn(x);
#else
  return (int)std::nearbyint(x);
#endif
}
GP_HD int addmax0(int a, int b) {   // max(a + b, 0)
#ifdef __CUDA_ARCH__
  return __viaddmax_s32_relu(a, b, 0);
#else
  return a + b > 0 ? a + b : 0;
#endif
}
GP_HD int imax(int a, int b) { return a > b ? a : b; }

// ------------------------------------------------------- two-part numbers

// Two values, each the unevaluated sum h + l.
struct Two {
  float2 h, l;
};
GP_HD Two two_zero() {
  Two t;
  t.h = f2(0.f);
  t.l = f2(0.f);
  return t;
}
GP_HD Two two_neg(Two a) {
  Two t;
  t.h = neg2(a.h);
  t.l = neg2(a.l);
  return t;
}
// a + b = s + e exactly
GP_HD void two_sum(float2 a, float2 b, float2* s, float2* e) {
  const float2 t = add2(a, b);
  const float2 m = sub2(a, t);   // minus the part of b that arrived in t
  *e = add2(sub2(a, add2(t, m)), add2(b, m));
  *s = t;
}
// a + b, the high parts' sum error-free
GP_HD Two two_add(Two a, Two b) {
  Two r;
  float2 e;
  two_sum(a.h, b.h, &r.h, &e);
  r.l = add2(add2(a.l, b.l), e);
  return r;
}
// A product h - nl (its low part with the sign turned: no negated operands).
struct Prod {
  float2 h, nl;
};
GP_HD Prod prod_zero() {
  Prod t;
  t.h = f2(0.f);
  t.nl = f2(0.f);
  return t;
}
// A constant h + l and its negative.
struct Coef {
  float2 h, nh, nl;
};
GP_HD Coef coef_pair(float2 h, float2 l) {
  Coef c;
  c.h = h;
  c.nh = neg2(h);
  c.nl = neg2(l);
  return c;
}
GP_HD Prod two_mul(const Coef& c, const Two& x) {
  Prod r;
  r.h = mul2(c.h, x.h);
  r.nl = fma2(c.nh, x.l, fma2(c.nl, x.h, fma2(c.nh, x.h, r.h)));
  return r;
}
GP_HD Two two_add(const Two& a, const Prod& b) {
  Two r;
  float2 e;
  two_sum(a.h, b.h, &r.h, &e);
  r.l = add2(sub2(a.l, b.nl), e);
  return r;
}
GP_HD Prod prod_add(const Prod& a, const Prod& b) {
  Prod r;
  float2 e;
  two_sum(a.h, b.h, &r.h, &e);
  r.nl = sub2(add2(a.nl, b.nl), e);
  return r;
}
GP_HD Two prod_two(const Prod& a) {
  Two r;
  r.h = a.h;
  r.l = neg2(a.nl);
  return r;
}
// a + b rounded towards zero
GP_HD float2 add2_rz(float2 a, float2 b) {
#ifdef __CUDA_ARCH__
  return __fadd2_rz(a, b);
#else
  const double x = (double)a.x + b.x, y = (double)a.y + b.y;
  float fx = (float)x, fy = (float)y;
  if (std::fabs((double)fx) > std::fabs(x)) fx = std::nextafter(fx, 0.f);
  if (std::fabs((double)fy) > std::fabs(y)) fy = std::nextafter(fy, 0.f);
  return f2(fx, fy);
#endif
}
// high part = the value truncated to FP32, low part the rest (same sign, below ulp(h)),
// for a low part not above the high one by much
GP_HD Two two_norm(const Prod& x) {
  Two r;
  const float2 n = f2(-1.f);
  r.h = add2_rz(x.h, mul2(x.nl, n));
  r.l = sub2(sub2(x.h, r.h), x.nl);
  return r;
}

GP_HD Two two_norm(const Two& x) {
  Two r;
  r.h = add2_rz(x.h, x.l);
  r.l = add2(sub2(x.h, r.h), x.l);
  return r;
}
GP_HD Two two_mul(const Two& a, const Two& b) {
  Two r;
  r.h = mul2(a.h, b.h);
  const float2 e = fma2(a.h, b.h, mul2(r.h, f2(-1.f)));
  r.l = fma2(a.l, b.h, fma2(a.h, b.l, e));
  return r;
}
GP_HD Two two_scalar(float2 h, float2 l) {
  Two r;
  r.h = h;
  r.l = l;
  return r;
}
// c + y a for a constant c = ch + cl and an FP32 a
GP_HD Two two_const_fma(float2 ch, float2 cl, const Two& y, float2 a) {
  Two p;
  p.h = mul2(y.h, a);
  p.l = fma2(y.l, a, fma2(y.h, a, mul2(p.h, f2(-1.f))));
  return two_add(two_scalar(ch, cl), p);
}
// (exp(-y) - 1 + y) / y^2 (Taylor; FP32 from the y^5 term of exp on, in the long form from y^6:
// an error of 2^-32 y^5, 2^-35 y^6 of exp, which the sizes of y it is taken for keep below 2^-56)
template <bool LONG> GP_HD Two two_exp_series(const Two& y) {
  const float2 y1 = y.h;
  float2 a = fma2(y1, f2(1.f / 40320.f), f2(-1.f / 5040.f));
  a = fma2(y1, a, f2(1.f / 720.f));
  Two w;   // 1/24, 1/6 and, long, 1/120 as an FP32 pair
  if constexpr (LONG) {
    w = two_const_fma(f2(-1.f / 120.f), f2((float)(-(1.0 / 120.0 - (double)(1.f / 120.f)))), y, a);
    w = two_add(two_scalar(f2(1.f / 24.f), f2((float)(1.0 / 24.0 - (double)(1.f / 24.f)))), two_mul(y, w));
  } else {
    a = fma2(y1, a, f2(-1.f / 120.f));
    w = two_const_fma(f2(1.f / 24.f), f2((float)(1.0 / 24.0 - (double)(1.f / 24.f))), y, a);
  }
  w = two_add(two_scalar(f2(-1.f / 6.f), f2((float)(-(1.0 / 6.0 - (double)(1.f / 6.f))))), two_mul(y, w));
  return two_add(two_scalar(f2(0.5f), f2(0.f)), two_mul(y, w));
}
// exp(-y) - 1 for |y| <= 1/64, and the same without its leading term, exp(-y) - 1 + y, for |y| <= 1/16
GP_HD Two two_expm1_neg(const Two& y) {
  return two_mul(y, two_add(two_scalar(f2(-1.f), f2(0.f)), two_mul(y, two_exp_series<false>(y))));
}
GP_HD Two two_expm1_neg_rest(const Two& y) { return two_mul(y, two_mul(y, two_exp_series<true>(y))); }
// exp(-y) - 1 for |y| <= 2^-9: y^3 and higher terms (below 2^-29) in FP32
GP_HD Two two_expm1_neg_small(const Two& y) {
  const float2 y1 = y.h, y2 = mul2(y1, y1);
  const float2 a = fma2(y1, fma2(y1, f2(-1.f / 120.f), f2(1.f / 24.f)), f2(-1.f / 6.f));
  Two r = two_mul(y, y);
  r.h = mul2(r.h, f2(0.5f));
  r.l = fma2(mul2(y1, y2), a, mul2(r.l, f2(0.5f)));
  Two n;
  n.h = mul2(y.h, f2(-1.f));
  n.l = mul2(y.l, f2(-1.f));
  return two_add(n, r);
}
// Complex numbers: lanes (re, im).
GP_HD Two two_swap(const Two& a) { return two_scalar(f2(a.h.y, a.h.x), f2(a.l.y, a.l.x)); }
GP_HD Two two_cmul(const Two& a, const Two& b) {
  const Two ar = two_scalar(f2(a.h.x), f2(a.l.x));
  const Two ai = two_scalar(f2(-a.h.y, a.h.y), f2(-a.l.y, a.l.y));
  return two_add(two_mul(ar, b), two_mul(ai, two_swap(b)));
}
// (cos y - 1, 1 - sin y / y) for |y| <= 1/16, both lanes of y the same (Taylor in z = y^2; the
// terms from z^3 / 720 and y z^3 / 5040 on in FP32)
GP_HD Two two_cis_series(const Two& y) {
  const Two z = two_mul(y, y);
  const float2 a = fma2(z.h, f2(1.f / 40320.f, 0.f), f2(-1.f / 720.f, 1.f / 5040.f));
  Two w = two_const_fma(f2(1.f / 24.f, -1.f / 120.f),
                        f2((float)(1.0 / 24.0 - (double)(1.f / 24.f)), (float)(-(1.0 / 120.0 - (double)(1.f / 120.f)))),
                        z, a);
  w = two_add(two_scalar(f2(-0.5f, 1.f / 6.f), f2(0.f, (float)(1.0 / 6.0 - (double)(1.f / 6.f)))), two_mul(z, w));
  return two_mul(z, w);
}
// (cos y - 1, -sin y), and the same without its leading term, (cos y - 1, y - sin y)
GP_HD Two two_cis_neg_m1(const Two& y) {
  const Two c = two_cis_series(y), m = two_mul(y, two_add(two_scalar(f2(-1.f), f2(0.f)), c));
  return two_scalar(f2(c.h.x, m.h.y), f2(c.l.x, m.l.y));
}
GP_HD Two two_cis_neg_rest(const Two& y) {
  const Two c = two_cis_series(y), m = two_mul(y, c);
  return two_scalar(f2(c.h.x, m.h.y), f2(c.l.x, m.l.y));
}
// (cos y - 1, -sin y) for |y| <= 2^-10: z^2 and y z terms (below 2^-32) in FP32
GP_HD Two two_cis_neg_m1_small(const Two& y) {
  const Two z = two_mul(y, y);
  const float re = z.h.x, rel = z.l.x;
  const float c = -0.5f * re, cl = -0.5f * rel + re * re * (1.f / 24.f);
  const float m = -y.h.y, ml = -y.l.y + y.h.y * re * (1.f / 6.f);
  return two_scalar(f2(c, m), f2(cl, ml));
}
// Two FP64 values times 2^kSplitShift as h + m + l exactly: h the leading 21 bits, m and
// l the next 16 and 16.  Sums of a few m (or l) of neighbouring values are exact (16-bit
// integers times nearby powers of two).  *tmax receives the larger of itself and the
// values' exponent fields (kSplitTooBig: out of range or non-finite).  With off = kSplitOff1 the
// values themselves (FP32's range and no more).
struct Three {
  float2 h, m, l;
};
GP_HD Three split3(double a, double b, int* tmax, int off = kSplitOff) {
  uint32_t h[2], o[2];
  words(a, &h[0], &o[0]);
  words(b, &h[1], &o[1]);
  float hf[2], p[2], mf[2], lf[2];
  for (int q = 0; q < 2; ++q) {
    const int t = addmax0((int)(h[q] & 0x7fffffffu), -off);
    *tmax = imax(*tmax, t);
    const uint32_t w = ((uint32_t)t << 3) | (h[q] & 0x80000000u);
    hf[q] = bits_f(w);
    p[q] = bits_f(w & 0xff800000u);                     // +- 2^E
    mf[q] = bits_f(0x4b000000u | (o[q] >> 16));         // 2^23 + high half of the low word
    lf[q] = bits_f(0x4b000000u | (o[q] & 0xffffu));     // 2^23 + low half
  }
  Three r;
  r.h = f2(hf[0], hf[1]);
  const float2 P = f2(p[0], p[1]);
  const float2 bias = f2(-8388608.f);
  r.m = mul2(add2(f2(mf[0], mf[1]), bias), mul2(P, f2(0x1p-36f)));
  r.l = mul2(add2(f2(lf[0], lf[1]), bias), mul2(P, f2(0x1p-52f)));
  return r;
}

// Two FP64 values times 2^kSplitShift as h + l, each part rounded to nearest: 48 bits.
GP_HD Two split2(double a, double b, int* tmax) {
  uint32_t h[2], o[2];
  words(a, &h[0], &o[0]);
  words(b, &h[1], &o[1]);
  float hf[2], p[2], lf[2];
  for (int q = 0; q < 2; ++q) {
    const int t = addmax0((int)(h[q] & 0x7fffffffu), -kSplitOff);
    *tmax = imax(*tmax, t);
    const uint32_t w = ((((uint32_t)t << 3) | (o[q] >> 29)) & 0x7fffffffu) | (h[q] & 0x80000000u);
    // the low 29 bits as a signed remainder (times 8); its sign rounds the high part
    const int r = (int)(o[q] << 3);
    hf[q] = bits_f(w + ((uint32_t)r >> 31));
    p[q] = bits_f(w & 0xff800000u);
    lf[q] = (float)r;
  }
  Two r;
  r.h = f2(hf[0], hf[1]);
  r.l = mul2(mul2(f2(lf[0], lf[1]), f2(0x1p-55f)), f2(p[0], p[1]));
  return r;
}

// Second difference a - 2 b + c: exact for neighbouring values of similar size (smooth
// fields), within about 2^-48 of the largest of them otherwise.
GP_HD Two second_difference(const Three& a, const Three& b, const Three& c) {
  float2 t, e1, sh, e2;
  two_sum(a.h, c.h, &t, &e1);
  two_sum(t, mul2(f2(-2.f), b.h), &sh, &e2);
  const float2 sm = fma2(f2(-2.f), b.m, add2(a.m, c.m));
  const float2 sl = add2(fma2(f2(-2.f), b.l, add2(a.l, c.l)), add2(e1, e2));
  Two r;
  float2 e;
  two_sum(sh, sm, &r.h, &e);
  r.l = add2(e, sl);
  return r;
}

// (h + l) 2^(k - kSplitShift) as an FP64 number, of a two_norm'ed number: l is added to
// the significand of h in units of its FP64 ulp, and because it never points back below
// h the unit is right at powers of two as well.  A subnormal h counts as zero.
GP_HD double to_double(float h, float l, int k) {
  const uint32_t a = f_bits(h);
  // |l| in units of 2^(E - 52), E the exponent of h
  const float q = bits_f(0x7f000000u - (a & 0x7f800000u));
  const uint32_t ci = (uint32_t)round_int(fabsf((l * q) * 0x1p52f));
  const uint32_t off = (a & 0x7f800000u) == 0u ? 0u : (uint32_t)(kSplitOff + (k << 20));
  const uint32_t top = (uint32_t)((int32_t)a >> 3) & 0x8fffffffu;   // sign, exponent and leading significand
  const uint64_t w = (((uint64_t)top << 32) | (uint64_t)(a << 29)) + (((uint64_t)off << 32) | ci);
  return from_words((uint32_t)(w >> 32), (uint32_t)w);
}

#ifdef __CUDACC__
// The banded operator (gp_sweeps.cu) on two lanes at a time: two points of a real line, or
// the parts of one complex point, its products as two real sums, A = sum w.re s and
// B = sum w.im s, joined at the end (4 W + 5 instructions; 8 W + 6 as complex products).
template <bool CPLX, int W> struct BandTaps {
  float2 wr[W + 1], wi[CPLX ? W + 1 : 1];
  __device__ __forceinline__ explicit BandTaps(const float* wt) {   // centre first
#pragma unroll
    for (int k = 0; k <= W; ++k) {
      wr[k] = f2(CPLX ? wt[2 * (W + k)] : wt[W + k]);
      if constexpr (CPLX) wi[k] = f2(wt[2 * (W + k) + 1]);
    }
  }
  // at(k): the value k points along the line (a float2 of the vector)
  template <class AT> __device__ __forceinline__ float2 operator()(AT at) const {
    const float2 c = at(0);
    float2 a = mul2(wr[0], c);
    if constexpr (CPLX) {
      float2 b = mul2(wi[0], c);
#pragma unroll
      for (int k = 1; k <= W; ++k) {
        const float2 s = add2(at(-k), at(k));
        a = fma2(wr[k], s, a);
        b = fma2(wi[k], s, b);
      }
      return add2(c, f2(a.x - b.y, a.y + b.x));
    } else {
#pragma unroll
      for (int k = 1; k <= W; ++k) a = fma2(wr[k], add2(at(-k), at(k)), a);
      return add2(c, a);
    }
  }
};
// The same operator with the complex products' roundings of Field::chain (gp_device.cuh),
// each tap added to the result before it; real lines: as BandTaps.
template <bool CPLX, int W> struct BandChain : BandTaps<CPLX, W> {
  using BandTaps<CPLX, W>::wr;
  using BandTaps<CPLX, W>::wi;
  __device__ __forceinline__ explicit BandChain(const float* wt) : BandTaps<CPLX, W>(wt) {
    if constexpr (CPLX)
#pragma unroll
      for (int k = 0; k <= W; ++k) wi[k].x = -wi[k].x;
  }
  template <class AT> __device__ __forceinline__ float2 operator()(AT at) const {
    if constexpr (CPLX) {
      const float2 c = at(0);
      float2 a = fma2(wr[0], c, mul2(wi[0], f2(c.y, c.x)));
#pragma unroll
      for (int k = 1; k <= W; ++k) {
        const float2 s = add2(at(-k), at(k));
        a = fma2(wr[k], s, fma2(wi[k], f2(s.y, s.x), a));
      }
      return add2(c, a);
    } else {
      return BandTaps<CPLX, W>::operator()(at);
    }
  }
};
#endif

}  // namespace gpk
