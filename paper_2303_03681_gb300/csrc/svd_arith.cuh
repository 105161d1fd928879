// Arithmetic of the FP64-accurate truncation SVD (svd_jacobi.cuh): how a complex column
// entry is stored, and the few operations on it that the factorisation and
// the Jacobi sweeps are made of.
//
//  * ArDF: double-float (dfloat.cuh), heads and error terms in two planes of a
//    column.  Re and im of an entry go through the packed FP32 instructions
//    (add / mul / fma .f32x2: two lanes' worth of FP32 work per issue slot;
//    the pipe rate is the same 128 FMA/clk/SM, so the gain is in issue slots
//    for the loads).  A rotation of one entry pair costs 62 packed
//    instructions (12 real products, each 4, summed with exact heads) against
//    172 scalar ones for products and sums taken one by one; a Gram term
//    costs 26.  Early sweeps take the Gram term from the heads alone (2).
//  * ArF64: complex128 columns in FP64 (2 FMA/clk/SM on this part).
#pragma once

#include "common.cuh"
#include "dfloat.cuh"

namespace mpsv {

// 1 / sqrt(a) in double-float: FP32 seed and one Newton step whose residual
// 1 - a y^2 is formed with the exact square of the seed
__device__ __forceinline__ ff ff_rsqrt(ff a) {
  const float y = rsqrtf(a.h);
  const ff p = ff_mul(a, two_prod(y, y));
  const float d = __fadd_rn(__fsub_rn(1.f, p.h), -p.l);
  return quick_two_sum(y, y * fmaf(0.375f * d, d, 0.5f * d));
}

// ---- rotations -----------------------------------------------------------
// x' = c x - conj(s) y, y' = c y + s x; dn = t |g|: |x'|^2 = |x|^2 - dn,
// |y'|^2 = |y|^2 + dn.
template <typename S> struct Rot {
  S c, sr, si, dn;
};

__device__ __forceinline__ int exp_of(float x) { return ((__float_as_int(x) >> 23) & 0xff) - 127; }
__device__ __forceinline__ float pow2f(int e) { return __int_as_float((e + 127) << 23); }  // -126 <= e <= 127

// |g|^2 / (a b) for squared column norms a, b (0 when either is zero).  g is
// scaled by the power of two nearest sqrt(a b), so nothing underflows while
// the ratio is above 1e-36 (norms are scaled: 1e-12 is a zero column, see
// kScaleExp); no square root or division on this path, which
// every pair takes.
__device__ __forceinline__ float pair_off2(float a, float b, float gr, float gi) {
  if (!(fminf(a, b) > 1e-12f)) return 0.f;
  const int ea = exp_of(a), eb = exp_of(b), h = (ea + eb) >> 1;
  const float s = pow2f(-h);
  const float xr = gr * s, xi = gi * s;
  const float ab = (a * pow2f(-ea)) * (b * pow2f(ea - 2 * h));  // a b 2^(-2h), in [1, 8)
  return __fdividef(fmaf(xr, xr, xi * xi), ab);
}

// The FP32 angle of a pair: d = (b - a) / 2 and g scaled to max(a, b) in
// [1, 2).  With r = sqrt(d^2 + |g|^2) and q = |d| + r: t = |g| / q, c =
// sqrt(q / 2r), s e^{i phi} = sign(d) (c / q) g, dn = sign(d) |g|^2 / q - two
// dependent special-function steps, no hypot and no tangent.
struct Angle32 {
  float c, sf, dn;
};
__device__ __forceinline__ Angle32 angle32(float d, float xr, float xi) {
  const float g2 = fmaf(xr, xr, xi * xi);
  const float w = fmaf(d, d, g2);
  const float rw = rsqrtf(w);
  const float q = fmaf(w, rw, fabsf(d));
  const float h = 0.5f * q * rw;  // c^2, in [1/2, 1]
  const float rh = rsqrtf(h);
  const float iq = __fdividef(copysignf(1.f, d), q);
  Angle32 o;
  o.c = h * rh;
  o.sf = o.c * iq;
  o.dn = g2 * iq;
  // unit norm to FP32 rounding (the approximate functions leave about 4e-7)
  const float s2 = o.sf * o.sf * g2;
  const float f = -0.5f * (fmaf(o.c, o.c, -1.f) + s2);
  o.c = fmaf(o.c, f, o.c);
  o.sf = fmaf(o.sf, f, o.sf);
  return o;
}

// The rotation of a pair from its squared norms a, b and Gram entry g, on the
// FP32 pipes.  b - a is formed from heads and error terms, so a nearly
// degenerate pair's angle is not rounding noise.  The FP32 (c, s e^{i phi})
// has c^2 + |s|^2 = 1 + d, |d| ~ 2^-24; d is evaluated with exact products and
// sums and the rotation is scaled by 1 - d/2 + 3 d^2 / 8 (the binomial series
// of (1 + d)^(-1/2)).  The angle itself is FP32-accurate: a pair left with
// 1e-7 of its Gram entry is rotated again in the next sweep.
__device__ __forceinline__ bool df_angle(ff a, ff b, ff gr, ff gi, Rot<ff>& o) {
  const int e = exp_of(fmaxf(a.h, b.h));
  const float scl = pow2f(-e);
  const float xr = gr.h * scl, xi = gi.h * scl;
  const float dd = 0.5f * scl * __fadd_rn(__fsub_rn(b.h, a.h), __fsub_rn(b.l, a.l));
  const Angle32 t = angle32(dd, xr, xi);
  if (!(t.c <= 2.f)) return false;  // NaN
  const float cf = t.c;
  const ff s_r = two_prod(t.sf, xr), s_i = two_prod(t.sf, xi);
  const ff c2 = two_prod(cf, cf), r2 = two_prod(s_r.h, s_r.h), i2 = two_prod(s_i.h, s_i.h);
  const ff u0 = two_sum(c2.h, -1.f);
  const ff u1 = two_sum(u0.h, r2.h);
  const ff u2 = two_sum(u1.h, i2.h);
  const float tail = __fadd_rn(__fadd_rn(__fadd_rn(u0.l, u1.l), u2.l), __fadd_rn(c2.l, __fadd_rn(r2.l, i2.l)));
  const float cross = 2.f * __fmaf_rn(s_r.h, s_r.l, __fmul_rn(s_i.h, s_i.l));
  const float d = __fadd_rn(u2.h, __fadd_rn(tail, cross));
  const float fl = __fmaf_rn(0.375f * d, d, -0.5f * d);
  o.c = quick_two_sum(cf, __fmul_rn(cf, fl));
  o.sr = quick_two_sum(s_r.h, __fmaf_rn(s_r.h, fl, s_r.l));
  o.si = quick_two_sum(s_i.h, __fmaf_rn(s_i.h, fl, s_i.l));
  o.dn = ff_make(t.dn * pow2f(e), 0.f);
  return true;
}

// ---- column memory ---------------------------------------------------------
// Columns in this CTA's dynamic shared memory are named by their byte offset
// (shared-space instructions with 32-bit addresses), columns in the global
// workspace by pointer (shared between CTAs, so they bypass L1).
extern __shared__ __align__(16) unsigned char svd_smem[];
template <bool kG> struct Mem;
template <> struct Mem<false> {
  using H = unsigned;
  template <typename T> __device__ static __forceinline__ T ld(H c, int i) {
    return reinterpret_cast<const T*>(svd_smem + c)[i];
  }
  template <typename T> __device__ static __forceinline__ void st(H c, int i, T v) {
    reinterpret_cast<T*>(svd_smem + c)[i] = v;
  }
};
template <> struct Mem<true> {
  using H = char*;
  template <typename T> __device__ static __forceinline__ T ld(H c, int i) {
    return __ldcg(reinterpret_cast<const T*>(c) + i);
  }
  template <typename T> __device__ static __forceinline__ void st(H c, int i, T v) {
    __stcg(reinterpret_cast<T*>(c) + i, v);
  }
};

// ---- the arithmetics ------------------------------------------------
// Every one provides: V (an entry in registers), S (a real sum), kBytes per
// stored entry, ld(len) (the padded column length: strides that put the
// columns of neighbouring pairs in different halves of the banks), load /
// store of row r of a column, and the operations below.  A dot product is
// summed over a group's lanes by dot_sum.

struct ArDF {
  using S = ff;
  struct V {
    float2 h, l;
  };
  struct Acc {  // sums of x^H y: re in a.h.x + a.h.y, im in b.h.x - b.h.y
    Acc2 a, b;
  };
  static constexpr int kBytes = 16;
  static constexpr bool kRough = true;  // Gram terms of early sweeps from the heads
  __host__ __device__ static int ld(int len) { return (len + 3) / 8 * 8 + 4; }
  __device__ static __forceinline__ double unit() { return 1.4210854715202004e-14; }  // 2^-46
  template <bool kG> __device__ static __forceinline__ V load(typename Mem<kG>::H col, int ld, int r) {
    V v;
    v.h = Mem<kG>::template ld<float2>(col, r);
    v.l = Mem<kG>::template ld<float2>(col, ld + r);
    return v;
  }
  template <bool kG> __device__ static __forceinline__ void store(typename Mem<kG>::H col, int ld, int r, V v) {
    Mem<kG>::template st<float2>(col, r, v.h);
    Mem<kG>::template st<float2>(col, ld + r, v.l);
  }
  __device__ static __forceinline__ V zero_entry() { return cval(zero(), zero()); }
  __device__ static __forceinline__ float2 head(V v) { return v.h; }
  __device__ static __forceinline__ V make(double re, double im) {
    const ff a = ff_split(re), b = ff_split(im);
    V v;
    v.h = mk2(a.h, b.h);
    v.l = mk2(a.l, b.l);
    return v;
  }
  __device__ static __forceinline__ S from_double(double x) { return ff_split(x); }
  __device__ static __forceinline__ double to_double(S x) { return ff_join(x); }
  __device__ static __forceinline__ float to_float(S x) { return x.h; }
  __device__ static __forceinline__ S zero() { return ff_make(0.f, 0.f); }
  __device__ static __forceinline__ S shfl_add(S x, int o) { return ff_add(x, ff_shfl_xor(x, o)); }
  __device__ static __forceinline__ float head_norm2(V v) { return fmaf(v.h.x, v.h.x, v.h.y * v.h.y); }
  __device__ static __forceinline__ void dot(Acc& acc, V x, V y) {  // += conj(x) y
    const float2 m1 = mk2(-1.f, -1.f);
    const float2 nh = mul2(x.h, m1), nl = mul2(x.l, m1);
    acc.a.add(x.h, nh, nl, y.h, y.l);
    acc.b.add(x.h, nh, nl, swap2(y.h), swap2(y.l));
  }
  // the sum over the G lanes of a group, re and im packed: one exact two-sum
  // of the heads and two additions of the error terms a stage, renormalised
  // once at the end (the same bits in every lane: each step is symmetric)
  __device__ static __forceinline__ void dot_sum(const Acc& a, int G, S& re, S& im) {
    float2 h, t;
    two_sum2(mk2(a.a.h.x, a.b.h.x), mk2(a.a.h.y, -a.b.h.y), h, t);
    float2 e = add2(add2(mk2(a.a.e.x, a.b.e.x), mk2(a.a.e.y, -a.b.e.y)), t);
    for (int o = G >> 1; o > 0; o >>= 1) {
      const float2 h2 = mk2(__shfl_xor_sync(0xffffffffu, h.x, o), __shfl_xor_sync(0xffffffffu, h.y, o));
      const float2 e2 = mk2(__shfl_xor_sync(0xffffffffu, e.x, o), __shfl_xor_sync(0xffffffffu, e.y, o));
      two_sum2(h, h2, h, t);
      e = add2(add2(e, e2), t);
    }
    re = quick_two_sum(h.x, e.x);
    im = quick_two_sum(h.y, e.y);
  }
  // dot_sum and the sum of a squared norm in one run of stages
  __device__ static __forceinline__ void dot_norm_sum(const Acc& a, const Acc2& q, int G, S& re, S& im, S& nn) {
    float2 h, t;
    two_sum2(mk2(a.a.h.x, a.b.h.x), mk2(a.a.h.y, -a.b.h.y), h, t);
    float2 e = add2(add2(mk2(a.a.e.x, a.b.e.x), mk2(a.a.e.y, -a.b.e.y)), t);
    ff u = two_sum(q.h.x, q.h.y);
    u.l = __fadd_rn(__fadd_rn(q.e.x, q.e.y), u.l);
    for (int o = G >> 1; o > 0; o >>= 1) {
      const float2 h2 = mk2(__shfl_xor_sync(0xffffffffu, h.x, o), __shfl_xor_sync(0xffffffffu, h.y, o));
      const float2 e2 = mk2(__shfl_xor_sync(0xffffffffu, e.x, o), __shfl_xor_sync(0xffffffffu, e.y, o));
      const ff u2 = ff_shfl_xor(u, o);
      two_sum2(h, h2, h, t);
      e = add2(add2(e, e2), t);
      const ff s = two_sum(u.h, u2.h);
      u = ff_make(s.h, __fadd_rn(__fadd_rn(u.l, u2.l), s.l));
    }
    re = quick_two_sum(h.x, e.x);
    im = quick_two_sum(h.y, e.y);
    nn = quick_two_sum(u.h, u.l);
  }
  // the sums of two squared norms
  __device__ static __forceinline__ void norm2_sum(const Acc2& p, const Acc2& q, int G, S& a, S& b) {
    float2 h, t;
    two_sum2(mk2(p.h.x, q.h.x), mk2(p.h.y, q.h.y), h, t);
    float2 e = add2(add2(mk2(p.e.x, q.e.x), mk2(p.e.y, q.e.y)), t);
    for (int o = G >> 1; o > 0; o >>= 1) {
      const float2 h2 = mk2(__shfl_xor_sync(0xffffffffu, h.x, o), __shfl_xor_sync(0xffffffffu, h.y, o));
      const float2 e2 = mk2(__shfl_xor_sync(0xffffffffu, e.x, o), __shfl_xor_sync(0xffffffffu, e.y, o));
      two_sum2(h, h2, h, t);
      e = add2(add2(e, e2), t);
    }
    a = quick_two_sum(h.x, e.x);
    b = quick_two_sum(h.y, e.y);
  }
  using NAcc = Acc2;
  __device__ static __forceinline__ void nrm(NAcc& acc, V x) {
    const float2 m1 = mk2(-1.f, -1.f);
    acc.add(x.h, mul2(x.h, m1), mul2(x.l, m1), x.h, x.l);
  }
  __device__ static __forceinline__ S nrm_value(const NAcc& a) { return ff_add(a.x(), a.y()); }
  __device__ static __forceinline__ S rsqrt(S a) { return ff_rsqrt(a); }
  __device__ static __forceinline__ S mul(S a, S b) { return ff_mul(a, b); }
  __device__ static __forceinline__ S sub(S a, S b) { return ff_sub(a, b); }
  __device__ static __forceinline__ S add(S a, S b) { return ff_add(a, b); }
  __device__ static __forceinline__ V cval(S re, S im) {
    V v;
    v.h = mk2(re.h, im.h);
    v.l = mk2(re.l, im.l);
    return v;
  }
  // constants of y <- y - x w
  struct Axpy {
    float2 ah, nah, nal, bh, nbh, nbl;
  };
  __device__ static __forceinline__ Axpy axpy_const(S wr, S wi) {
    Axpy k;
    k.ah = mk2(-wr.h, -wr.h);
    k.nah = mk2(wr.h, wr.h);
    k.nal = mk2(wr.l, wr.l);
    k.bh = mk2(wi.h, -wi.h);
    k.nbh = mk2(-wi.h, wi.h);
    k.nbl = mk2(-wi.l, wi.l);
    return k;
  }
  __device__ static __forceinline__ V axpy(const Axpy& k, V x, V y) {
    Acc2 s;
    s.h = y.h;
    s.e = y.l;
    s.add(k.ah, k.nah, k.nal, x.h, x.l);
    s.add(k.bh, k.nbh, k.nbl, swap2(x.h), swap2(x.l));
    renorm2(s.h, s.e);
    V v;
    v.h = s.h;
    v.l = s.e;
    return v;
  }
  struct RotK {
    float2 c, nc, ncl, s, ns, sl, nsl, i, ni, nil;
  };
  __device__ static __forceinline__ RotK rot_const(const Rot<S>& r) {
    RotK k;
    k.c = mk2(r.c.h, r.c.h);
    k.nc = mk2(-r.c.h, -r.c.h);
    k.ncl = mk2(-r.c.l, -r.c.l);
    k.s = mk2(r.sr.h, r.sr.h);
    k.ns = mk2(-r.sr.h, -r.sr.h);
    k.sl = mk2(r.sr.l, r.sr.l);
    k.nsl = mk2(-r.sr.l, -r.sr.l);
    k.i = mk2(-r.si.h, r.si.h);
    k.ni = mk2(r.si.h, -r.si.h);
    k.nil = mk2(r.si.l, -r.si.l);
    return k;
  }
  // a complex sum of three products with exact heads: c u + a1 v1 + a2 v2
  __device__ static __forceinline__ V sum3(float2 c, float2 nc, float2 ncl, V u, float2 a, float2 na, float2 nal, V v,
                                           float2 b, float2 nb, float2 nbl, float2 wh, float2 wl) {
    Acc2 s;
    s.h = mul2(c, u.h);
    float2 ne = fma2(nc, u.h, s.h);
    ne = fma2(nc, u.l, ne);
    ne = fma2(ncl, u.h, ne);
    s.e = mul2(ne, mk2(-1.f, -1.f));
    s.add(a, na, nal, v.h, v.l);
    s.add(b, nb, nbl, wh, wl);
    renorm2(s.h, s.e);
    V o;
    o.h = s.h;
    o.l = s.e;
    return o;
  }
  __device__ static __forceinline__ void rotate(const RotK& k, V& x, V& y) {
    // x' = c x - sr (yr, yi) + (-si, si) (yi, yr);  y' = c y + sr (xr, xi) + (-si, si) (xi, xr)
    const V nx = sum3(k.c, k.nc, k.ncl, x, k.ns, k.s, k.sl, y, k.i, k.ni, k.nil, swap2(y.h), swap2(y.l));
    const V ny = sum3(k.c, k.nc, k.ncl, y, k.s, k.ns, k.nsl, x, k.i, k.ni, k.nil, swap2(x.h), swap2(x.l));
    x = nx;
    y = ny;
  }
  __device__ static __forceinline__ float off2(S a, S b, S gr, S gi) { return pair_off2(a.h, b.h, gr.h, gi.h); }
  __device__ static __forceinline__ bool angle(S a, S b, S gr, S gi, Rot<S>& o) { return df_angle(a, b, gr, gi, o); }
  __device__ static __forceinline__ V scale(V x, S f) {
    return cval(ff_mul(ff_make(x.h.x, x.l.x), f), ff_mul(ff_make(x.h.y, x.l.y), f));
  }
  __device__ static __forceinline__ V times(V x, float pow2) {  // exact
    x.h = mul2(x.h, mk2(pow2, pow2));
    x.l = mul2(x.l, mk2(pow2, pow2));
    return x;
  }
  __device__ static __forceinline__ double2 value(V x) {
    return make_double2(ff_join(ff_make(x.h.x, x.l.x)), ff_join(ff_make(x.h.y, x.l.y)));
  }
  __device__ static __forceinline__ float2 value32(V x) { return x.h; }
};

struct ArF64 {
  using S = double;
  using V = double2;
  struct Acc {
    double re = 0.0, im = 0.0;
  };
  static constexpr int kBytes = 16;
  static constexpr bool kRough = false;
  __host__ __device__ static int ld(int len) { return len; }
  __device__ static __forceinline__ double unit() { return 1.1102230246251565e-16; }
  template <bool kG> __device__ static __forceinline__ V load(typename Mem<kG>::H col, int, int r) {
    return Mem<kG>::template ld<double2>(col, r);
  }
  template <bool kG> __device__ static __forceinline__ void store(typename Mem<kG>::H col, int, int r, V v) {
    Mem<kG>::template st<double2>(col, r, v);
  }
  __device__ static __forceinline__ V zero_entry() { return cval(zero(), zero()); }
  __device__ static __forceinline__ float2 head(V v) { return mk2((float)v.x, (float)v.y); }
  __device__ static __forceinline__ V make(double re, double im) { return make_double2(re, im); }
  __device__ static __forceinline__ S from_double(double x) { return x; }
  __device__ static __forceinline__ double to_double(S x) { return x; }
  __device__ static __forceinline__ float to_float(S x) { return (float)x; }
  __device__ static __forceinline__ S zero() { return 0.0; }
  __device__ static __forceinline__ S shfl_add(S x, int o) { return x + __shfl_xor_sync(0xffffffffu, x, o); }
  __device__ static __forceinline__ float head_norm2(V v) {
    const float a = (float)v.x, b = (float)v.y;
    return fmaf(a, a, b * b);
  }
  __device__ static __forceinline__ void dot(Acc& a, V x, V y) {
    a.re = fma(x.x, y.x, fma(x.y, y.y, a.re));
    a.im = fma(x.x, y.y, fma(-x.y, y.x, a.im));
  }
  __device__ static __forceinline__ void dot_sum(const Acc& a, int G, S& re, S& im) {
    re = a.re;
    im = a.im;
    for (int o = G >> 1; o > 0; o >>= 1) {
      re += __shfl_xor_sync(0xffffffffu, re, o);
      im += __shfl_xor_sync(0xffffffffu, im, o);
    }
  }
  struct NAcc {
    double v = 0.0;
  };
  __device__ static __forceinline__ void dot_norm_sum(const Acc& a, const NAcc& q, int G, S& re, S& im, S& nn) {
    re = a.re;
    im = a.im;
    nn = q.v;
    for (int o = G >> 1; o > 0; o >>= 1) {
      re += __shfl_xor_sync(0xffffffffu, re, o);
      im += __shfl_xor_sync(0xffffffffu, im, o);
      nn += __shfl_xor_sync(0xffffffffu, nn, o);
    }
  }
  __device__ static __forceinline__ void norm2_sum(const NAcc& p, const NAcc& q, int G, S& a, S& b) {
    a = p.v;
    b = q.v;
    for (int o = G >> 1; o > 0; o >>= 1) {
      a += __shfl_xor_sync(0xffffffffu, a, o);
      b += __shfl_xor_sync(0xffffffffu, b, o);
    }
  }
  __device__ static __forceinline__ void nrm(NAcc& a, V x) { a.v = fma(x.x, x.x, fma(x.y, x.y, a.v)); }
  __device__ static __forceinline__ S nrm_value(const NAcc& a) { return a.v; }
  // FP32 seed and two Newton steps (1e-7 -> 1e-14 -> rounding); a within the FP32 range
  __device__ static __forceinline__ S rsqrt(S a) {
    double y = (double)rsqrtf((float)a);
    const double h = 0.5 * a;
    y = y * fma(-h * y, y, 1.5);
    return y * fma(-h * y, y, 1.5);
  }
  __device__ static __forceinline__ S mul(S a, S b) { return a * b; }
  __device__ static __forceinline__ S sub(S a, S b) { return a - b; }
  __device__ static __forceinline__ S add(S a, S b) { return a + b; }
  __device__ static __forceinline__ V cval(S re, S im) { return make_double2(re, im); }
  struct Axpy {
    double wr, wi;
  };
  __device__ static __forceinline__ Axpy axpy_const(S wr, S wi) { return Axpy{wr, wi}; }
  __device__ static __forceinline__ V axpy(const Axpy& k, V x, V y) {
    return make_double2(fma(-x.x, k.wr, fma(x.y, k.wi, y.x)), fma(-x.x, k.wi, fma(-x.y, k.wr, y.y)));
  }
  using RotK = Rot<S>;
  __device__ static __forceinline__ RotK rot_const(const Rot<S>& r) { return r; }
  __device__ static __forceinline__ void rotate(const RotK& k, V& x, V& y) {
    const V nx = make_double2(fma(k.c, x.x, fma(-k.sr, y.x, -k.si * y.y)), fma(k.c, x.y, fma(-k.sr, y.y, k.si * y.x)));
    const V ny = make_double2(fma(k.c, y.x, fma(k.sr, x.x, -k.si * x.y)), fma(k.c, y.y, fma(k.sr, x.y, k.si * x.x)));
    x = nx;
    y = ny;
  }
  __device__ static __forceinline__ float off2(S a, S b, S gr, S gi) {
    return pair_off2((float)a, (float)b, (float)gr, (float)gi);
  }
  // FP32 angle brought to unit norm in FP64 (as the double-float form, with
  // the same binomial correction)
  __device__ static __forceinline__ bool angle(S a, S b, S gr, S gi, Rot<S>& o) {
    const int e = exp_of(fmaxf((float)a, (float)b));
    const double scl = pow2f(-e);
    const float xr = (float)(gr * scl), xi = (float)(gi * scl);
    const Angle32 t = angle32((float)(0.5 * (b - a) * scl), xr, xi);
    if (!(t.c <= 2.f)) return false;  // NaN
    const double cd = t.c, sr = double(t.sf) * double(xr), si = double(t.sf) * double(xi);
    const double d = fma(cd, cd, fma(sr, sr, fma(si, si, -1.0)));
    const double f = fma(d, fma(0.375, d, -0.5), 1.0);
    o.c = cd * f;
    o.sr = sr * f;
    o.si = si * f;
    o.dn = (double)t.dn * pow2f(e);
    return true;
  }
  __device__ static __forceinline__ V scale(V x, S f) { return make_double2(x.x * f, x.y * f); }
  __device__ static __forceinline__ V times(V x, float pow2) { return make_double2(x.x * pow2, x.y * pow2); }
  __device__ static __forceinline__ double2 value(V x) { return x; }
  __device__ static __forceinline__ float2 value32(V x) { return mk2((float)x.x, (float)x.y); }
};

}  // namespace mpsv
