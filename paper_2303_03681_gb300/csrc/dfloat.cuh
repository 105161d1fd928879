// Double-float arithmetic for the FP64-accurate SVD and the contractions of
// complex128 states.
//
// This part executes FP64 at two fused multiply-adds per clock per SM and
// FP32 at 128: a value held as the unevaluated sum of two floats (h + l,
// |l| <= ulp(h) / 2, about 48 significant bits) and handled with the
// error-free transformations of Knuth (two-sum: the rounding error of a + b
// recovered exactly from three more additions) and of the fused multiply-add
// (two-product: a b - rn(a b) = fma(a, b, -rn(a b)) exactly) runs the sweeps
// on the FP32 pipes several times faster than FP64, at a unit roundoff of
// about 2^-46.  The exponent range is FP32's: the kernels that use it keep
// squared norms above the rounding floor, far from 1e-38.
//
// Complex values keep (re, im) pairs of heads and of error terms, so that both
// parts go through the packed FP32 instructions (add / mul / fma .f32x2).
#pragma once

#include <cuda_runtime.h>

namespace mpsv {

struct ff {
  float h, l;
};

__device__ __forceinline__ ff ff_make(float h, float l) {
  ff r;
  r.h = h;
  r.l = l;
  return r;
}

// exact: s + e = a + b (Knuth's two-sum)
__device__ __forceinline__ ff two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return ff_make(s, e);
}

// exact when |a| >= |b| or a = 0
__device__ __forceinline__ ff quick_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  return ff_make(s, __fsub_rn(b, __fsub_rn(s, a)));
}

__device__ __forceinline__ ff ff_add(ff a, ff b) {
  ff s = two_sum(a.h, b.h);
  s.l = __fadd_rn(s.l, __fadd_rn(a.l, b.l));
  return quick_two_sum(s.h, s.l);
}

__device__ __forceinline__ ff ff_neg(ff a) { return ff_make(-a.h, -a.l); }

__device__ __forceinline__ ff ff_sub(ff a, ff b) { return ff_add(a, ff_neg(b)); }

// a b with the exact product of the heads (two-product by fma)
__device__ __forceinline__ ff ff_mul(ff a, ff b) {
  const float p = __fmul_rn(a.h, b.h);
  float e = __fmaf_rn(a.h, b.h, -p);
  e = __fmaf_rn(a.h, b.l, e);
  e = __fmaf_rn(a.l, b.h, e);
  return quick_two_sum(p, e);
}

// acc + a b
__device__ __forceinline__ ff ff_fma(ff a, ff b, ff acc) { return ff_add(ff_mul(a, b), acc); }

// exact: h + l = a b (the fma two-product)
__device__ __forceinline__ ff two_prod(float a, float b) {
  const float p = __fmul_rn(a, b);
  return ff_make(p, __fmaf_rn(a, b, -p));
}

__device__ __forceinline__ ff ff_shfl_xor(ff a, int o) {
  return ff_make(__shfl_xor_sync(0xffffffffu, a.h, o), __shfl_xor_sync(0xffffffffu, a.l, o));
}

// Sums of double-float products (the per-lane Gram sums of the Jacobi SVD,
// the multiply-adds of the complex128 contractions): a running FP32 head h,
// summed exactly (two_sum), and an FP32 error term e collecting the two_sum
// errors and each product's exact error (fma) and cross terms a_h b_l +
// a_l b_h; 12 FP32 operations a product against 18 for a double-float fma.
// e holds about 2^-23 of the sum of |products|, so after K additions its
// own rounding is about K 2^-47 of that sum (1e-12 at K = 128).
struct GramAcc {
  float h = 0.f, e = 0.f;
  __device__ __forceinline__ void add(ff a, ff b) {
    const float p = __fmul_rn(a.h, b.h);
    float pe = __fmaf_rn(a.h, b.h, -p);
    pe = __fmaf_rn(a.h, b.l, pe);
    pe = __fmaf_rn(a.l, b.h, pe);
    const ff s = two_sum(h, p);
    h = s.h;
    e = __fadd_rn(e, __fadd_rn(s.l, pe));
  }
  __device__ __forceinline__ ff value() const { return quick_two_sum(h, e); }
};

// ---- packed FP32 pairs --------------------------------------------------
__device__ __forceinline__ float2 mk2(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ float2 swap2(float2 a) { return make_float2(a.y, a.x); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
// a - b, exactly rounded (the product with -1 is exact)
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, mk2(-1.f, -1.f), a); }
// s + e = a + b exactly (Knuth's two-sum)
__device__ __forceinline__ void two_sum2(float2 a, float2 b, float2& s, float2& e) {
  s = add2(a, b);
  const float2 bb = sub2(s, a);
  e = add2(sub2(a, sub2(s, bb)), sub2(b, bb));
}
// (h, l) <- h + l renormalised, |h| >= |l|
__device__ __forceinline__ void renorm2(float2& h, float2& l) {
  const float2 s = add2(h, l);
  l = sub2(l, sub2(s, h));
  h = s;
}
// A pair of running sums of double-float products: exact heads h, error
// terms e (the GramAcc of dfloat.cuh, two at a time).
struct Acc2 {
  float2 h = {0.f, 0.f}, e = {0.f, 0.f};
  // += a b for a = (ah, al) given with its negatives
  __device__ __forceinline__ void add(float2 ah, float2 nah, float2 nal, float2 bh, float2 bl) {
    const float2 p = mul2(ah, bh);
    float2 ne = fma2(nah, bh, p);  // minus the product's rounding error
    ne = fma2(nah, bl, ne);
    ne = fma2(nal, bh, ne);
    float2 t;
    two_sum2(h, p, h, t);
    e = add2(e, sub2(t, ne));
  }
  __device__ __forceinline__ ff x() const { return quick_two_sum(h.x, e.x); }
  __device__ __forceinline__ ff y() const { return quick_two_sum(h.y, e.y); }
};

// A double as a float pair by integer operations: FP64 conversions and
// subtractions run at 1/64 of the FP32 rate here (three of them per value took
// longer than reading the theta).  h is the value rounded to 24 bits (half up
// in magnitude), l the signed rest rounded to 24 bits: 2^-49 relative, as
// rounding by conversions.  Values below 2^-126 give 0; infinities and NaN
// stay.
__device__ __forceinline__ ff ff_split(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
  const int e = (int)(b >> 52) - 1023;
  const float sign = (__double2hiint(x) < 0) ? -1.f : 1.f;
  if (e < -126) return ff_make(0.f, 0.f);
  if (e > 126) return ff_make((float)x, 0.f);  // inf, NaN, and values that may overflow
  const unsigned long long hb = (b + (1ull << 28)) >> 29;  // exponent and 23 mantissa bits, rounded
  const int rest = (int)(long long)(b - (hb << 29));       // |rest| <= 2^28, units of 2^(e - 52)
  const float h = __int_as_float((int)((unsigned)hb - (896u << 23)));
  const float l = e > -75 ? (float)rest * __int_as_float((e - 52 + 127) << 23) : 0.f;
  return ff_make(sign * h, sign * l);
}

// The double nearest to h + l, by integer operations for the same reason.
__device__ __forceinline__ double ff_join(ff a) {
  const unsigned hb = (unsigned)__float_as_int(a.h) & 0x7fffffffu;
  const int e = (int)(hb >> 23);  // biased
  if (e == 0 || e == 255) return (double)a.h;
  // l in units of 2^(e - 127 - 52), |l| <= 2^28 of them; two exact factors
  // keep 2^(179 - e) inside the FP32 range
  const int up = 179 - e;
  const float u = a.l * __int_as_float((min(up, 100) + 127) << 23) * __int_as_float((max(up - 100, 0) + 127) << 23);
  // below a power of two the spacing halves
  const float l = a.h < 0.f ? -u : u;
  const int li = __float2int_rn((hb & 0x7fffffu) == 0 && l < 0.f ? 2.f * l : l);
  const long long m = (((long long)hb + (896ll << 23)) << 29) + li;
  return __longlong_as_double(m | (a.h < 0.f ? (long long)0x8000000000000000ull : 0ll));
}

// A complex double-float value as the contraction tiles hold it: (re, im) of
// the heads and of the error terms.
struct Cff {
  float2 h, l;
};
__device__ __forceinline__ Cff cff_split(double2 z) {
  const ff a = ff_split(z.x), b = ff_split(z.y);
  Cff c;
  c.h = mk2(a.h, b.h);
  c.l = mk2(a.l, b.l);
  return c;
}

// Sums of complex double-float products, re and im packed: a += (xr, xi) o
// (yr, yi) and b += (xr, xi) o (yi, yr), from which x y and conj(x) y both
// follow.  26 packed instructions a product, two of them the negatives of x,
// which products with the same x share; the scalar form took 48 (the pipe
// rate is the same, the issue slots halve).
struct CAcc {
  Acc2 a, b;
  __device__ __forceinline__ void add(const Cff& x, const Cff& y) {
    const float2 m1 = mk2(-1.f, -1.f);
    const float2 nh = mul2(x.h, m1), nl = mul2(x.l, m1);
    a.add(x.h, nh, nl, y.h, y.l);
    b.add(x.h, nh, nl, swap2(y.h), swap2(y.l));
  }
  static __device__ __forceinline__ ff sum(const Acc2& p, float s) {  // p.x + s p.y, s = +-1
    ff t = two_sum(p.h.x, s * p.h.y);
    t.l = __fadd_rn(t.l, __fadd_rn(p.e.x, s * p.e.y));
    return quick_two_sum(t.h, t.l);
  }
  __device__ __forceinline__ double2 value() const {  // sum of x y
    return make_double2(ff_join(sum(a, -1.f)), ff_join(sum(b, 1.f)));
  }
  __device__ __forceinline__ double2 value_conj() const {  // sum of conj(x) y
    return make_double2(ff_join(sum(a, 1.f)), ff_join(sum(b, -1.f)));
  }
};

}  // namespace mpsv
