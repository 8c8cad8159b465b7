// kbc_fix.cuh -- 64-bit fixed-point arithmetic and the FP64 KBC collision built on it.
//
// GB300 executes 2 FP64 lanes per SM and cycle (conversions to and from FP64 included), but 62
// 64-bit integer additions, 64 shifts and logic operations, ~30 32 x 32 -> 64 bit multiplies and
// 128 FP32 FMAs (measured). An FP64 collision in FP64 instructions (571 of them per node) is
// bound by that pipe at 6 % of the memory roof. Here the shifts f - W, their moments and the
// equilibrium are integers of unit 2^-60 instead: |f - W| < 1/4 then has at least the
// resolution that f itself has in FP64 (f >= 2^-8), sums are exact and products are rounded
// once, so that the absolute error of the result is a few 2^-60 where FP64 arithmetic leaves
// ~2^-53 W_i (its sqrt(1 + 3u^2) alone is rounded at 2^-53).
//   * everything linear in f (moments, deviations, relaxation, back transform) is done on the
//     27 natural moments with integer additions; the relaxation multiplies 23 moments, not
//     2 x 27 populations;
//   * u = j / rho and R - 1 = sqrt(1 + 3u^2) - 1 start from FP32 approximations and are
//     corrected by Newton's method with integer residuals;
//   * only the entropic products, of which a ratio is taken, need a floating format: FP32 pairs
//     (hi + lo, two-product and two-sum arithmetic after Dekker and Knuth), with the integer
//     deviations of a node scaled by a common power of two, about 2^-45 relative.
// Nodes outside the range of the format (|f - W| >= 1/4, rho or u far from a lattice state,
// NaN, |beta gamma| >= 512) are reported and left to the FP64 collision.
//
// The functions are host code as well (no CUDA intrinsics there), so that they can be checked
// without a GPU.
#pragma once

#include <stdint.h>
#include <string.h>

#include <cmath>

#define KBC_HD __host__ __device__ __forceinline__

namespace kbc {
namespace fix {

typedef long long fx;  // value * 2^60
constexpr int kFrac = 60;
constexpr fx kOne = 1ll << kFrac;
// round(2^60 / 3), / 9, / 27
constexpr fx kThird = 384307168202282325ll, kNinth = 128102389400760775ll,
             k27th = 42700796466920258ll;
// high word of 0.25: the bound on |f - W| under which no sum of 27 shifts leaves the range
constexpr uint32_t kTopF64 = 0x3fd00000u;
constexpr uint32_t kTopF32 = 0x3e800000u;

KBC_HD uint64_t bits_of(double d) {
#ifdef __CUDA_ARCH__
  return (uint64_t)__double_as_longlong(d);
#else
  uint64_t b;
  memcpy(&b, &d, 8);
  return b;
#endif
}
KBC_HD double f64_of(uint64_t b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double d;
  memcpy(&d, &b, 8);
  return d;
#endif
}
KBC_HD uint32_t bits_of(float d) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(d);
#else
  uint32_t b;
  memcpy(&b, &d, 4);
  return b;
#endif
}
KBC_HD float f32_of(uint32_t b) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(b);
#else
  float d;
  memcpy(&d, &b, 4);
  return d;
#endif
}
// right shift by any amount (PTX clamps; 0 from 64 on)
KBC_HD uint64_t shr(uint64_t x, uint32_t n) {
#ifdef __CUDA_ARCH__
  uint64_t r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));
  return r;
#else
  return n > 63 ? 0 : x >> n;
#endif
}
KBC_HD float rcpf(float x) {
#ifdef __CUDA_ARCH__
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
#else
  return 1.0f / x;
#endif
}
KBC_HD float sqrtf_fast(float x) {
#ifdef __CUDA_ARCH__
  float r;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
#else
  return sqrtf(x);
#endif
}
KBC_HD float fmaf_(float a, float b, float c) {
#ifdef __CUDA_ARCH__
  return __fmaf_rn(a, b, c);
#else
  return fmaf(a, b, c);
#endif
}
KBC_HD float mulf(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fmul_rn(a, b);
#else
  volatile float r = a * b;
  return r;
#endif
}
KBC_HD float addf(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fadd_rn(a, b);
#else
  volatile float r = a + b;
  return r;
#endif
}
KBC_HD int f2i(float x) {
#ifdef __CUDA_ARCH__
  return __float2int_rn(x);
#else
  return (int)lrintf(x);
#endif
}
KBC_HD int clz64(uint64_t x) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)x);
#else
  return x ? __builtin_clzll(x) : 64;
#endif
}

// d as a fixed-point number, truncated; *top collects the largest high word of |d|, by which
// the caller sees values (and NaN) outside the range
KBC_HD fx from_f64(double d, uint32_t* top) {
  const uint64_t b = bits_of(d);
  const uint32_t hi = (uint32_t)(b >> 32), ah = hi & 0x7fffffffu;
  *top = ah > *top ? ah : *top;
  const uint64_t m = (b << 11) | 0x8000000000000000ull;  // 1.mantissa, leading bit at 63
  const fx x = (fx)shr(m, 1026u - (ah >> 20));           // 0 for |d| < 2^-61, zero included
  return (int32_t)hi < 0 ? -x : x;
}
KBC_HD fx from_f32(float d, uint32_t* top) {
  const uint32_t b = bits_of(d), ah = b & 0x7fffffffu;
  *top = ah > *top ? ah : *top;
  const uint64_t m = (uint64_t)((b << 8) | 0x80000000u) << 32;
  const fx x = (fx)shr(m, 130u - (ah >> 23));
  return (int32_t)b < 0 ? -x : x;
}
// v * 2^-(60 + n), rounded to nearest even: one conversion and an exponent shift (|v| < 2^63;
// the result is normal or zero)
template <int N> KBC_HD double to_f64(fx v) {
  const uint64_t b = bits_of((double)v);
  return f64_of(v == 0 ? b : b - ((uint64_t)(kFrac + N) << 52));
}

// ------------------------------------------------------------------ products
// v = h 2^32 + l with both halves signed, for the product below
struct Split {
  int32_t h, l;
};
KBC_HD Split split(fx v) {
  const uint32_t lo = (uint32_t)v;
  Split s;
  s.l = (int32_t)lo;
  s.h = (int32_t)((uint32_t)((uint64_t)v >> 32) + (lo >> 31));
  return s;
}
// a b / 2^64, rounded, to within 3/4 of a unit (l x l, less than 1/4 unit, is dropped): three
// 32 x 32 -> 64 bit multiplies. |a| < 2^62.9 and |b| < 2^63 - 2^31 keep the middle sum in range.
KBC_HD fx mul(Split a, Split b) {
  long long mid = (long long)a.h * b.l + 0x80000000ll;
  mid += (long long)a.l * b.h;
  return (long long)a.h * b.h + (mid >> 32);
}
// a factor below 1/2 in magnitude, scaled by 2^4 so that mul() gives a product of unit 2^-60
KBC_HD Split factor(fx v) { return split((fx)((uint64_t)v << 4)); }

// 1 / rho for 1/2 < rho < 2: FP32 reciprocal r0 in units of 2^-28, then r0 (1 + E + E^2) with
// E = 1 - rho r0 exact to 2^-60 (|E| < 2^-21, so E^3 < 2^-63)
KBC_HD fx reciprocal(fx rho) {
  const float rf = mulf((float)(int32_t)(rho >> 32), 1.0f / 268435456.0f);  // 2^-28 (rho 2^28)
  const int32_t r0 = f2i(mulf(rcpf(rf), 268435456.0f));
  const int32_t rh = (int32_t)(rho >> 32);
  const uint32_t rl = (uint32_t)rho;
  // rho r0 2^-28: high part exactly, low part truncated (below one unit)
  const fx p = (((long long)rh * r0) << 4) + (fx)(((uint64_t)rl * (uint32_t)r0) >> 28);
  const fx E = kOne - p;
  const int32_t Es = (int32_t)(E >> 16);
  const fx F = E + (((long long)Es * Es) >> 28);
  // r0 F 2^-28
  const int32_t Fh = (int32_t)(F >> 24);
  const int32_t Fl = (int32_t)(F & 0xffffff);
  return ((fx)r0 << 32) + ((((long long)Fh * r0) + (((long long)Fl * r0) >> 24)) >> 4);
}

// e = sqrt(1 + 3u^2) - 1, the root of e^2 + 2e = t = 3u^2, for |u| < 1/4 (e < 0.09): an FP32
// value e0 (unit 2^-32), then two Newton corrections r / (2 (1 + e0)) with the residual exact in
// integers; they leave ~2^-51 and below one unit of 2^-60
KBC_HD fx axis_e(Split u4, fx u) {
  const fx uu = mul(split(u), u4);
  const fx t = uu + uu + uu;
  const float tf = mulf((float)(int32_t)(t >> 29), 1.0f / 2147483648.0f);
  const float R1 = addf(1.0f, sqrtf_fast(addf(1.0f, tf)));
  const float ef = mulf(tf, rcpf(R1));
  const int32_t e0 = f2i(mulf(ef, 4294967296.0f));
  const fx r0 = t - ((fx)e0 << 29) - (((long long)e0 * e0) >> 4);
  const float gf = mulf(0.5f, rcpf(addf(1.0f, ef)));
  const int32_t g = f2i(mulf(gf, 1073741824.0f));  // unit 2^-30
  const fx e1 = ((fx)e0 << 28) + (((long long)(int32_t)(r0 >> 6) * g) >> 24);
  const Split e1s = split(e1);
  const fx r1 = t - e1 - e1 - mul(e1s, factor(e1));
  return e1 + (fx)(((long long)(int32_t)r1 * g) >> 30);
}

// ------------------------------------------------------------------ FP32 pairs
struct df {
  float h, l;
};
// an integer of the entropic products' scale in units of 2^32: its top 24 significant bits in h
// (the sum of two exactly converted halves), the rest, to 24 bits, in l
KBC_HD df df_of(fx v) {
  const int32_t hi = (int32_t)((uint64_t)v >> 32);
  const float f1 = (float)(hi & ~0xffff), f0 = (float)(hi & 0xffff);
  df r;
  r.h = addf(f1, f0);
  r.l = fmaf_((float)(uint32_t)v, 1.0f / 4294967296.0f, addf(f0, -addf(r.h, -f1)));
  return r;
}
// a value of unit 2^-60 and below 4 (|v| < 2^62), as its value: the top 24 bits in h
KBC_HD df df_value(fx v) {
  df r;
  r.h = mulf((float)((int32_t)((uint64_t)v >> 32) >> 8), 1.0f / 1048576.0f);  // 2^-20
  r.l = mulf((float)(int32_t)((uint32_t)((uint64_t)v >> 9) & 0x7fffffffu),
             1.0f / 2251799813685248.0f);  // 2^-51
  return r;
}
// 1 / a (a away from 0): FP32 reciprocal and one correction
KBC_HD df df_rcp(df a) {
  const float r0 = rcpf(a.h);
  float e = fmaf_(-a.h, r0, 1.0f);
  e = fmaf_(-a.l, r0, e);
  df r;
  r.h = r0;
  r.l = mulf(r0, fmaf_(e, e, e));
  return r;
}
KBC_HD df df_mul(df a, df b) {
  df r;
  r.h = mulf(a.h, b.h);
  const float e = fmaf_(a.h, b.h, -r.h);
  const float l = fmaf_(a.h, b.l, fmaf_(a.l, b.h, fmaf_(a.l, b.l, e)));
  const float h = addf(r.h, l);  // renormalised: without it the low parts grow and lose two bits
  r.l = addf(l, -addf(h, -r.h));
  r.h = h;
  return r;
}
KBC_HD df df_add(df a, df b) {  // two-sum of the high parts
  df r;
  r.h = addf(a.h, b.h);
  const float bb = addf(r.h, -a.h);
  const float e = addf(addf(a.h, -addf(r.h, -bb)), addf(b.h, -bb));
  r.l = addf(addf(a.l, b.l), e);
  return r;
}
KBC_HD double df_f64(df a) { return (double)a.h + (double)a.l; }

// ------------------------------------------------------------------ transforms
// natural moments M[p + 3q + 9r] = sum_i f_i vx^p vy^q vz^r (eq:natmoments), in place: per axis
// (f-, f0, f+) -> (sum, difference, sum of the outer two)
KBC_HD void to_moments(fx (&m)[27]) {
#pragma unroll
  for (int s = 1; s < 27; s *= 3)
#pragma unroll
    for (int k = 0; k < 27; ++k) {
      if ((k / s) % 3) continue;
      const fx a = m[k], z = m[k + s], p = m[k + 2 * s];
      m[k + 2 * s] = p + a;
      m[k + s] = p - a;
      m[k] = p + a + z;
    }
}
// the inverse, in place, population i times 2^(number of non-zero components of v_i): per axis
// f0 = m0 - m2, 2 f+- = m2 +- m1
KBC_HD void to_populations(fx (&m)[27]) {
#pragma unroll
  for (int s = 1; s < 27; s *= 3)
#pragma unroll
    for (int k = 0; k < 27; ++k) {
      if ((k / s) % 3) continue;
      const fx m0 = m[k], m1 = m[k + s], m2 = m[k + 2 * s];
      m[k] = m2 - m1;
      m[k + s] = m0 - m2;
      m[k + 2 * s] = m2 + m1;
    }
}
KBC_HD constexpr int nonzero(int i) {
  return (i % 3 != 1) + ((i / 3) % 3 != 1) + (i / 9 != 1);
}
KBC_HD constexpr int mi(int p, int q, int r) { return p + 3 * q + 9 * r; }

KBC_HD uint64_t magnitude(fx v) { return (uint64_t)(v ^ (v >> 63)); }
KBC_HD fx shl(fx v, int n) { return (fx)((uint64_t)v << n); }

struct Relax {
  double beta, inv_beta;  // eq:Egeneral's beta and 1 / beta
  int with_t, with_q, gamma_mode;
};

// One KBC collision (Sec. KBC, natural moments, product-form equilibrium) of the shifts d,
// |d_i| < 1/4, in place; the result d_i is f'_i - W_i times 2^nonzero(i) (to_f64<nonzero(i)>).
// Returns gamma; *guarded is set when <dh|dh> is 0 (gamma = 2), *bad when the node is outside
// the format's range (d is then not a result).
KBC_HD double collide(fx (&d)[27], const Relax& rx, int* guarded, bool* bad) {
  to_moments(d);
  const fx jx = d[mi(1, 0, 0)], jy = d[mi(0, 1, 0)], jz = d[mi(0, 0, 1)];
  const fx rho = kOne + d[0];
  const uint64_t jm = magnitude(jx) | magnitude(jy) | magnitude(jz);
  *bad = rho <= (kOne >> 1) || rho >= 2 * kOne || (jm >> 58) != 0;
  *guarded = 0;
  const fx ir = reciprocal(rho);
  const Split irs = split(ir);
  const fx ux = mul(irs, factor(jx)), uy = mul(irs, factor(jy)), uz = mul(irs, factor(jz));
  *bad = *bad || ((magnitude(ux) | magnitude(uy) | magnitude(uz)) >> 58) != 0;
  const Split ux4 = factor(ux), uy4 = factor(uy), uz4 = factor(uz);
  const fx ex = axis_e(ux4, ux), ey = axis_e(uy4, uy), ez = axis_e(uz4, uz);
  // second moments of the axis factors, m_2(u) = 1/3 + 2e/3
  const Split third = split((fx)((uint64_t)kThird << 4));
  const Split wx4 = factor(kThird + mul(split(ex + ex), third));
  const Split wy4 = factor(kThird + mul(split(ey + ey), third));
  const Split wz4 = factor(kThird + mul(split(ez + ez), third));

  // deviations A = M - rho M_eq (the moments of f - f_eq), all but the conserved four
  fx A[27];
  A[0] = A[mi(1, 0, 0)] = A[mi(0, 1, 0)] = A[mi(0, 0, 1)] = 0;
  const Split rs = split(rho), jxs = split(jx), jys = split(jy), jzs = split(jz);
  const fx rwx = mul(rs, wx4), rwy = mul(rs, wy4), rwz = mul(rs, wz4);
  const fx pxy = mul(jxs, uy4), pxz = mul(jxs, uz4), pyz = mul(jys, uz4);
  const fx jxwy = mul(jxs, wy4), jxwz = mul(jxs, wz4), jywx = mul(jys, wx4);
  const fx jywz = mul(jys, wz4), jzwx = mul(jzs, wx4), jzwy = mul(jzs, wy4);
  const Split rwxs = split(rwx);
  const fx rwxwy = mul(rwxs, wy4);
  const Split pxys = split(pxy);
  A[mi(2, 0, 0)] = d[mi(2, 0, 0)] + kThird - rwx;
  A[mi(0, 2, 0)] = d[mi(0, 2, 0)] + kThird - rwy;
  A[mi(0, 0, 2)] = d[mi(0, 0, 2)] + kThird - rwz;
  A[mi(1, 1, 0)] = d[mi(1, 1, 0)] - pxy;
  A[mi(1, 0, 1)] = d[mi(1, 0, 1)] - pxz;
  A[mi(0, 1, 1)] = d[mi(0, 1, 1)] - pyz;
  A[mi(1, 2, 0)] = d[mi(1, 2, 0)] - jxwy;
  A[mi(1, 0, 2)] = d[mi(1, 0, 2)] - jxwz;
  A[mi(2, 1, 0)] = d[mi(2, 1, 0)] - jywx;
  A[mi(0, 1, 2)] = d[mi(0, 1, 2)] - jywz;
  A[mi(2, 0, 1)] = d[mi(2, 0, 1)] - jzwx;
  A[mi(0, 2, 1)] = d[mi(0, 2, 1)] - jzwy;
  A[mi(1, 1, 1)] = d[mi(1, 1, 1)] - mul(pxys, uz4);
  A[mi(2, 2, 0)] = d[mi(2, 2, 0)] + kNinth - rwxwy;
  A[mi(2, 0, 2)] = d[mi(2, 0, 2)] + kNinth - mul(rwxs, wz4);
  A[mi(0, 2, 2)] = d[mi(0, 2, 2)] + kNinth - mul(split(rwy), wz4);
  A[mi(2, 1, 1)] = d[mi(2, 1, 1)] - mul(split(pyz), wx4);
  A[mi(1, 2, 1)] = d[mi(1, 2, 1)] - mul(split(pxz), wy4);
  A[mi(1, 1, 2)] = d[mi(1, 1, 2)] - mul(pxys, wz4);
  A[mi(2, 2, 1)] = d[mi(2, 2, 1)] - mul(split(jzwx), wy4);
  A[mi(2, 1, 2)] = d[mi(2, 1, 2)] - mul(split(jywx), wz4);
  A[mi(1, 2, 2)] = d[mi(1, 2, 2)] - mul(split(jxwy), wz4);
  A[mi(2, 2, 2)] = d[mi(2, 2, 2)] + k27th - mul(split(rwxwy), wz4);

  // the trace belongs to s (with_t) or, spread over the three diagonal moments, to h
  const fx tr = A[mi(2, 0, 0)] + A[mi(0, 2, 0)] + A[mi(0, 0, 2)];
  const fx ht = rx.with_t ? 0 : mul(split(tr), third);
  // s is relaxed by 2 beta = 8 (beta / 4)
  const Split bs = split((fx)(rx.beta * 4611686018427387904.0));  // beta / 4 of 2^64
  double gamma = 2.0;
  int k = 3;       // beta gamma = 2^k x (factor cs of 2^64)
  Split cs = bs;
  uint64_t hm = 0, sm = 0;  // bits of the largest deviations of h and of s
  if (rx.gamma_mode == 2) {  // gamma = 1 / beta
    gamma = rx.inv_beta;
    cs = split(1ll << 61);   // 1 = 8 x 1/8
  }
  if (rx.gamma_mode == 0) {
    // ---- gamma by eq:result21: ds and dh as populations, population i times 2^nonzero(i) (the
    // factors 4 of a product are taken up by the weights), from the moments scaled to below 2^58
    fx h[27];
#pragma unroll
    for (int i = 0; i < 27; ++i) h[i] = A[i];
    h[mi(0, 0, 0)] = h[mi(1, 0, 0)] = h[mi(0, 1, 0)] = h[mi(0, 0, 1)] = 0;
    h[mi(1, 1, 0)] = h[mi(1, 0, 1)] = h[mi(0, 1, 1)] = 0;
    h[mi(2, 0, 0)] = h[mi(0, 2, 0)] = h[mi(0, 0, 2)] = ht;
    const fx qm = rx.with_q ? -1ll : 0ll;  // the seven third moments: in s or in h
    const int third_of[7] = {mi(1, 2, 0), mi(1, 0, 2), mi(2, 1, 0), mi(0, 1, 2),
                             mi(2, 0, 1), mi(0, 2, 1), mi(1, 1, 1)};
    fx q[7];
#pragma unroll
    for (int n = 0; n < 7; ++n) {
      q[n] = A[third_of[n]] & qm;
      h[third_of[n]] = A[third_of[n]] & ~qm;
    }
    fx sx = A[mi(2, 0, 0)] - ht, sy = A[mi(0, 2, 0)] - ht, sz = A[mi(0, 0, 2)] - ht;
    fx sxy = A[mi(1, 1, 0)], sxz = A[mi(1, 0, 1)], syz = A[mi(0, 1, 1)];
    sm = magnitude(sx) | magnitude(sy) | magnitude(sz) | magnitude(sxy) | magnitude(sxz) |
         magnitude(syz);
#pragma unroll
    for (int n = 0; n < 7; ++n) sm |= magnitude(q[n]);
#pragma unroll
    for (int i = 0; i < 27; ++i)
      if (i % 3 + (i / 3) % 3 + i / 9 >= 2) hm |= magnitude(h[i]);
    int hs = clz64(hm) - 6, ss = clz64(sm) - 6;
    *bad = *bad || hs < 0 || ss < 0;
    hs = hs < 0 ? 0 : hs;
    ss = ss < 0 ? 0 : ss;
#pragma unroll
    for (int i = 0; i < 27; ++i) h[i] = shl(h[i], hs);
    to_populations(h);
    sx = shl(sx, ss), sy = shl(sy, ss), sz = shl(sz, ss);
    sxy = shl(sxy, ss), sxz = shl(sxz, ss), syz = shl(syz, ss);
#pragma unroll
    for (int n = 0; n < 7; ++n) q[n] = shl(q[n], ss);
    // Table 1 by class: centre -(sx + sy + sz), faces 2 ds = s -+ (Q + Q'), edges
    // 4 ds = +-P +- Q +- Q', corners 8 ds = +-Q_xyz
    const fx s0 = sx + sy + sz;
    const fx Gx = q[0] + q[1], Gy = q[2] + q[3], Gz = q[4] + q[5];
    // per-axis factors of f_eq / rho and their reciprocals (the weights of the entropic
    // products; the common factor 1 / rho drops out of the ratio): phi_+- = (1 + 2e +- 3u)/6 and
    // phi_0 = 4 (1 - e)/6, so with the factor 4 of the +- populations 1/(1 + 2e +- 3u) and
    // 1/(1 - e)
    df w[3][3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const fx e = a == 0 ? ex : (a == 1 ? ey : ez), u = a == 0 ? ux : (a == 1 ? uy : uz);
      const fx b = kOne + e + e, u3 = u + u + u;
      w[a][0] = df_rcp(df_value(b - u3));
      w[a][1] = df_rcp(df_value(kOne - e));
      w[a][2] = df_rcp(df_value(b + u3));
    }
    df num = {0.0f, 0.0f}, den = {0.0f, 0.0f};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      df cn, cd;
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        df rn, rd;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          const int i = a + 3 * b + 9 * c, va = a - 1, vb = b - 1, vc = c - 1;
          fx s;
          const int nz = nonzero(i);
          if (nz == 0) s = -s0;
          else if (nz == 1)
            s = va ? (va > 0 ? sx - Gx : sx + Gx)
                   : vb ? (vb > 0 ? sy - Gy : sy + Gy) : (vc > 0 ? sz - Gz : sz + Gz);
          else if (nz == 2) {
            // xy: P_xy, Q_xxy with the sign of vy, Q_xyy with that of vx; and so on
            const fx P = vc == 0 ? sxy : (vb == 0 ? sxz : syz);
            const int sp = vc == 0 ? va * vb : (vb == 0 ? va * vc : vb * vc);
            const fx Q1 = vc == 0 ? q[2] : (vb == 0 ? q[4] : q[5]);
            const int s1 = vc == 0 ? vb : vc;
            const fx Q2 = vc == 0 ? q[0] : (vb == 0 ? q[1] : q[3]);
            const int s2 = vc == 0 ? va : (vb == 0 ? va : vb);
            s = sp > 0 ? P : -P;
            s = s1 > 0 ? s + Q1 : s - Q1;
            s = s2 > 0 ? s + Q2 : s - Q2;
          } else {
            s = va * vb * vc > 0 ? q[6] : -q[6];
          }
          const df hd = df_of(h[i]), sd = df_of(s);
          const df t = df_mul(w[0][a], hd);
          const df tn = df_mul(t, sd), td = df_mul(t, hd);
          rn = a == 0 ? tn : df_add(rn, tn);
          rd = a == 0 ? td : df_add(rd, td);
        }
        rn = df_mul(w[1][b], rn);
        rd = df_mul(w[1][b], rd);
        cn = b == 0 ? rn : df_add(cn, rn);
        cd = b == 0 ? rd : df_add(cd, rd);
      }
      cn = df_mul(w[2][c], cn);
      cd = df_mul(w[2][c], cd);
      num = c == 0 ? cn : df_add(num, cn);
      den = c == 0 ? cd : df_add(den, cd);
    }
    double bg = 2.0 * rx.beta;
    if (hm != 0) {
      // num / den of the unscaled deviations: num carries 2^(hs + ss), den 2^(2 hs)
      const double qd = df_f64(num) / df_f64(den);
      const double qs = qd * f64_of((uint64_t)(1023 + hs - ss) << 52);
      gamma = rx.inv_beta - (2.0 - rx.inv_beta) * qs;
      bg = rx.beta * gamma;
    } else {
      *guarded = 1;
    }
    const uint32_t be = (uint32_t)(bits_of(bg) >> 52) & 0x7ffu;  // |bg| < 2^(be - 1022)
    k = be <= 1023 ? 3 : (int)be - 1020;
    *bad = *bad || k > 10 || clz64(hm) < k + 2;
    k = k > 10 ? 10 : k;
    cs = split((fx)(bg * f64_of((uint64_t)(1023 + 64 - k) << 52)));
  }
  if (rx.gamma_mode != 0) {
#pragma unroll
    for (int i = 0; i < 27; ++i)
      if (i % 3 + (i / 3) % 3 + i / 9 >= 2) hm |= magnitude(A[i]);
    *bad = *bad || clz64(hm) < 6;
  }
  // relaxation: M - 2 beta A for the moments of s, M - beta gamma A for the others
#pragma unroll
  for (int i = 0; i < 27; ++i) {
    const int order = i % 3 + (i / 3) % 3 + i / 9;
    if (order < 2) continue;
    if (order == 2 && (i % 3 == 2 || (i / 3) % 3 == 2 || i / 9 == 2)) {
      d[i] -= mul(split(shl(A[i] - ht, 3)), bs);
      if (!rx.with_t) d[i] -= mul(split(shl(ht, k)), cs);
    } else if (order == 2 || (order == 3 && rx.with_q)) {
      d[i] -= mul(split(shl(A[i], 3)), bs);
    } else {
      d[i] -= mul(split(shl(A[i], k)), cs);
    }
  }
  to_populations(d);
  return gamma;
}

}  // namespace fix
}  // namespace kbc
