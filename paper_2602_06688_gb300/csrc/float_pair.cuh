// Numbers as unevaluated sums h + l of two float32 (about 48 bits; Dekker 1971,
// Knuth's two-sum), for float64-grade sums whose results are rounded to float32.
// float64 runs at 2 fused multiply-adds per clock and SM here, float32 at 128: a
// pair product-and-sum of about 20 float32 instructions is six times faster than
// its float64 form.
//
// Sums are left unnormalised (|l| up to a few units in the last place of h):
// the next product renormalises, and what it leaves out, l times a normalised
// operand's l, is below 2^-45 of the result.
#pragma once
#include <stdint.h>

namespace specula {

struct __align__(8) fpair {
  float h, l;
};
struct __align__(16) cpair {
  fpair re, im;
};

__device__ __forceinline__ fpair fp_from(double v) {
  const float h = (float)v;
  return fpair{h, (float)(v - (double)h)};
}
__device__ __forceinline__ fpair fp_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b), v = __fsub_rn(s, a);
  return fpair{s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, v)), __fsub_rn(b, v))};
}
__device__ __forceinline__ fpair fp_norm(float h, float l) {
  const float s = __fadd_rn(h, l);
  return fpair{s, __fsub_rn(l, __fsub_rn(s, h))};
}
__device__ __forceinline__ fpair fp_add(fpair a, fpair b) {
  const fpair s = fp_two_sum(a.h, b.h);
  return fpair{s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l))};
}
__device__ __forceinline__ fpair fp_neg(fpair a) { return fpair{-a.h, -a.l}; }
__device__ __forceinline__ fpair fp_sub(fpair a, fpair b) { return fp_add(a, fp_neg(b)); }
__device__ __forceinline__ fpair fp_mul(fpair a, fpair b) {
  const float p = __fmul_rn(a.h, b.h);
  float e = __fmaf_rn(a.h, b.h, -p);
  e = __fmaf_rn(a.h, b.l, e);
  return fp_norm(p, __fmaf_rn(a.l, b.h, e));
}
// a b + c d, normalised
__device__ __forceinline__ fpair fp_dot(fpair a, fpair b, fpair c, fpair d) {
  const float p = __fmul_rn(a.h, b.h), q = __fmul_rn(c.h, d.h);
  float e = __fadd_rn(__fmaf_rn(a.h, b.h, -p), __fmaf_rn(c.h, d.h, -q));
  e = __fmaf_rn(a.h, b.l, e);
  e = __fmaf_rn(a.l, b.h, e);
  e = __fmaf_rn(c.h, d.l, e);
  e = __fmaf_rn(c.l, d.h, e);
  const fpair s = fp_two_sum(p, q);
  return fp_norm(s.h, __fadd_rn(s.l, e));
}

__device__ __forceinline__ cpair cp_add(cpair a, cpair b) {
  return cpair{fp_add(a.re, b.re), fp_add(a.im, b.im)};
}
__device__ __forceinline__ cpair cp_sub(cpair a, cpair b) {
  return cpair{fp_sub(a.re, b.re), fp_sub(a.im, b.im)};
}
__device__ __forceinline__ cpair cp_mul(cpair a, cpair w) {
  return cpair{fp_dot(a.re, w.re, fp_neg(a.im), w.im), fp_dot(a.re, w.im, a.im, w.re)};
}

// ---- Box-Muller ----------------------------------------------------------------
// (r cos 2 pi v, r sin 2 pi v), r = sqrt(-2 ln u), u, v = (x + 1/2) 2^-32 of two
// Philox words: integer range reduction, tables and short polynomials (the
// table-driven method of Tang, ACM TOMS 16, 378, 1990, for the logarithm; addition
// theorems for sine and cosine; one Newton step for the square root).  Errors
// on the CPU over 20 million arguments, the ends of the range among them, with a
// reciprocal square root off by up to 2 units: radius (relative) 2^-40.4 at most,
// r.m.s. 2^-44.6; cosine and sine 2^-42.9 at most, r.m.s. 2^-46.3.

// c: a 12-bit reciprocal of j / 128, so that f c is exact in a pair; 2 ln c
struct __align__(16) BmLog {
  float c, h, l, pad;
};

// sqrt(-2 ln((x + 1/2) 2^-32)).  With m = 2 x + 1 = f 2^k, f in [1, 2) or, from
// 181/128 on, halved: -2 ln u = 2 n ln 2 + 2 ln c - 2 ln(1 + r), n = 33 - k (32 - k
// where halved), r = f c - 1, |r| < 2^-7.3.  log_tab[j - kBmFirst], exp_tab[n] =
// 2 n ln 2; near u = 1 both are zero, so small results keep their relative accuracy.
constexpr int kBmFirst = 90, kBmCount = 91;   // j = 90 .. 180
__device__ __forceinline__ fpair bm_radius(uint32_t x, const BmLog *__restrict__ log_tab,
                                           const fpair *__restrict__ exp_tab) {
  const int k = 32 - __clz(x);   // bit length of x: m has its top bit there
  const uint64_t m = 2ull * x + 1ull;
  const uint64_t f33 = m << (32 - k);                // f 2^32, bit 32 set
  const int j1 = 128 + (((int)(f33 >> 24) - 256 + 1) >> 1);
  const bool half = j1 > 180;
  const int j = half ? 64 + (((int)(f33 >> 25) - 128 + 1) >> 1) : j1;
  const float unit = half ? 0x1p-33f : 0x1p-32f;
  const float fh = (float)(uint32_t)(f33 >> 9) * (512.f * unit);   // 24 bits
  const float fl = (float)(uint32_t)(f33 & 511u) * unit;
  const float4 g = __ldg(reinterpret_cast<const float4 *>(log_tab + (j - kBmFirst)));
  const float2 en = __ldg(reinterpret_cast<const float2 *>(exp_tab + (33 - k - (half ? 1 : 0))));
  // r = f c - 1: every step exact
  const float p = __fmul_rn(fh, g.x);
  const float e = __fadd_rn(__fmaf_rn(fh, g.x, -p), __fmul_rn(fl, g.x));
  const fpair r = fp_two_sum(__fsub_rn(p, 1.f), e);
  const float q = __fmul_rn(r.h, r.h);
  const float ql = __fmaf_rn(2.f * r.h, r.l, __fmaf_rn(r.h, r.h, -q));
  float s = __fmaf_rn(r.h, 1.f / 3.f, -2.f / 5.f);
  s = __fmaf_rn(r.h, s, 0.5f);
  s = __fmaf_rn(r.h, s, -2.f / 3.f);
  s = __fmul_rn(__fmul_rn(r.h, q), s);
  fpair t = fp_add(fpair{en.x, en.y}, fpair{g.y, g.z});
  t = fp_add(t, fpair{-2.f * r.h, -2.f * r.l});
  t = fp_add(t, fpair{q, __fadd_rn(ql, s)});
  t = fp_norm(t.h, t.l);
  const float y = rsqrtf(t.h), w = __fmul_rn(t.h, y);
  const float d = __fadd_rn(__fmaf_rn(-w, w, t.h), t.l);
  return fp_norm(w, __fmul_rn(d, 0.5f * y));
}

// (cos, sin) of 2 pi (x + 1/2) 2^-32: the nearest k / 256 of a turn from
// trig_tab, the rest |theta| <= pi / 256 by Taylor polynomials
__device__ __forceinline__ cpair bm_angle(uint32_t x, const cpair *__restrict__ trig_tab) {
  const uint32_t k = (uint32_t)(((uint64_t)x + (1u << 23)) >> 24);
  const float q = (float)(int)(2ll * x + 1ll - ((long long)k << 25));   // |q| <= 2^24: exact
  constexpr double unit = 2.0 * 3.14159265358979323846 / 8589934592.0;
  constexpr float uh = (float)unit, ul = (float)(unit - (double)(float)unit);
  const float th = __fmul_rn(q, uh);
  const float tl = __fmaf_rn(q, ul, __fmaf_rn(q, uh, -th));
  const float4 t = __ldg(reinterpret_cast<const float4 *>(trig_tab + k));
  const fpair C{t.x, t.y}, S{t.z, t.w};
  const float a = __fmul_rn(th, th);
  const float al = __fmaf_rn(2.f * th, tl, __fmaf_rn(th, th, -a));
  const float s3 = __fmul_rn(__fmul_rn(th, a), __fmaf_rn(a, 1.f / 120.f, -1.f / 6.f));
  const fpair sn = fp_norm(th, __fadd_rn(tl, s3));
  const float c4 = __fmul_rn(__fmul_rn(a, a), __fmaf_rn(a, -1.f / 720.f, 1.f / 24.f));
  const fpair c1 = fp_norm(-0.5f * a, __fmaf_rn(-0.5f, al, c4));   // cos - 1
  const fpair u = fp_dot(C, c1, fp_neg(S), sn), v = fp_dot(S, c1, C, sn);
  const fpair c = fp_add(C, u), d = fp_add(S, v);
  return cpair{fp_norm(c.h, c.l), fp_norm(d.h, d.l)};
}

}  // namespace specula
