// kbc_fix.cuh -- 64-bit fixed-point arithmetic and the FP64 KBC collision built on it.
//
// GB300 executes 2 FP64 lanes per SM and cycle (conversions to and from FP64 included), but 64
// integer additions, shifts and logic operations (a 64-bit addition of two or three terms is
// two instructions) and 64 32-bit multiplies (measured). An FP64 collision in FP64 instructions
// (571 of them per node) is bound by that pipe at 6 % of the memory roof. Here the shifts f - W,
// their moments and the equilibrium are integers instead, of a unit that follows the node: its
// largest shift has 55 bits (a unit of 2^-60 for shifts above 2^-6), so that nothing is lost at
// small amplitudes either. Sums are exact, products good to 3/4 of a unit. FP64 storage adds the
// change f' - f, whose conserved moments are exactly 0, to the stored shift: what a shift has below
// the unit stays with it, and mass and momentum drift by the rounding of that addition only.
// Against extended precision, relative to the node's largest shift, rms over nodes of amplitudes
// 0.12 to 1e-17: 4e-17..7e-17, FP64 instructions 1.0e-16..1.5e-16; 10^4 collisions of a uniform flow
// change its mass and momentum by 5e-16..1.1e-14 of it, FP64 instructions by 1e-15..2.6e-13. gamma
// is good to 4e-16..7e-16 far from equilibrium (FP64 2e-16..3e-16) and to less than FP64's error
// nearer to it.
//   * everything linear in f (moments, deviations, relaxation, back transform) is done on the
//     27 natural moments with integer additions; the relaxation multiplies 23 moments, not
//     2 x 27 populations;
//   * u = j / rho and R - 1 = sqrt(1 + 3u^2) - 1 start from FP32 approximations and are
//     corrected by Newton's method with integer residuals;
//   * the entropic products, of which a ratio is taken, are integer products too, of deviations
//     scaled by a common power of two to about 2^59, with integer weights that need no
//     reciprocal.
// About 4000 instructions per node, of which 54 (the conversions of the changes and the additions)
// are the FP64 pipe's, which they fill for nearly half of the time; 16 warps per SM.
// Measured at 256^3 (FP64 pull): FP64 instructions 17.4 ms a step, this 3.27; 432 B a node take
// 1.08 ms. A fixed unit of 2^-60, without the change and with products rounded down took 2.85 ms (32^3
// 8.7 us, now 11.3) but lost momentum one-sidedly, and small shifts their bits. With the last sum
// in integers instead of FP64 a step is 9 % slower.
// Nodes outside the range of the format (|f - W| >= 1/4 or all below 2^-70, rho or u far from a
// lattice state, NaN, |beta gamma| >= 128) are reported and left to the FP64 collision.
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
KBC_HD fx sar(fx x, uint32_t n) {
#ifdef __CUDA_ARCH__
  fx r;
  asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));
  return r;
#else
  return x >> (n > 63 ? 63 : n);
#endif
}
KBC_HD int32_t sar32(int32_t x, uint32_t n) {
#ifdef __CUDA_ARCH__
  int32_t r;
  asm("shr.s32 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(n));
  return r;
#else
  return x >> (n > 31 ? 31 : n);
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

// The high word of |d| (FP32: |d|); its largest over a node tells the caller whether the values
// (NaN among them) are in the range, and the node's scale.
KBC_HD uint32_t top_of(double d) { return (uint32_t)(bits_of(d) >> 32) & 0x7fffffffu; }
KBC_HD uint32_t top_of(float d) { return bits_of(d) & 0x7fffffffu; }

// A node's scale s: its numbers are integers of unit 2^-(60 + s), so that small shifts keep their
// bits. s puts the largest shift into [1/2, 1) 2^-5 (the room to 1/4 is for the moments, sums of
// many shifts), and is 0 where it is larger than that. False for shifts that are all below
// 2^-6 2^-kMaxScale but not zero.
constexpr uint32_t kMaxScale = 64;
template <typename T, uint32_t EXP> KBC_HD bool scale_to(uint32_t top, uint32_t* s) {
  const uint32_t bias = sizeof(T) == 8 ? 1023 : 127, e = top >> (sizeof(T) == 8 ? 20 : 23);
  const uint32_t want = bias - EXP - 1;  // biased exponent of the values in [1/2, 1) 2^-EXP
  *s = e < want && top != 0 ? want - e : 0;
  return *s <= kMaxScale;
}
template <typename T> KBC_HD bool scale_of(uint32_t top, uint32_t* s) {
  return scale_to<T, 5>(top, s);
}

// d 2^s as a fixed-point number, truncated
KBC_HD fx scaled(double d, uint32_t s) {
  const uint64_t b = bits_of(d);
  const uint64_t m = (b << 11) | 0x8000000000000000ull;  // 1.mantissa, leading bit at 63
  // 0 for |d| < 2^-61, zero included
  const fx x = (fx)shr(m, 1026u - s - ((uint32_t)(b >> 52) & 0x7ffu));
  return (int64_t)b < 0 ? -x : x;
}
KBC_HD fx scaled(float d, uint32_t s) {
  const uint32_t b = bits_of(d);
  const uint64_t m = (uint64_t)((b << 8) | 0x80000000u) << 32;
  const fx x = (fx)shr(m, 130u - s - ((b >> 23) & 0xffu));
  return (int32_t)b < 0 ? -x : x;
}
// the same for s = 0; *top collects the largest top_of()
KBC_HD fx from_f64(double d, uint32_t* top) {
  const uint32_t ah = top_of(d);
  *top = ah > *top ? ah : *top;
  return scaled(d, 0);
}
KBC_HD fx from_f32(float d, uint32_t* top) {
  const uint32_t ah = top_of(d);
  *top = ah > *top ? ah : *top;
  return scaled(d, 0);
}
// v * 2^-(60 + n + s), rounded to nearest even: one conversion and an exponent shift (|v| < 2^63;
// the result is normal or zero)
template <int N> KBC_HD double to_f64(fx v, uint32_t s = 0) {
  const uint64_t b = bits_of((double)v);
  uint32_t hi = (uint32_t)(b >> 32);
  hi = hi == 0 ? 0 : hi - ((kFrac + N + s) << 20);
  return f64_of((uint64_t)hi << 32 | (uint32_t)b);
}

// a 2^-n + b, n < 64, rounded to nearest or towards zero (a and b exact)
template <int N> KBC_HD float add_rn(float a, float b) {
  constexpr float c = 1.0f / (float)(1ull << N);
#ifdef __CUDA_ARCH__
  return __fmaf_rn(a, c, b);
#else
  return fmaf(a, c, b);
#endif
}
template <int N> KBC_HD float add_rz(float a, float b) {
  constexpr float c = 1.0f / (float)(1ull << N);
#ifdef __CUDA_ARCH__
  return __fmaf_rz(a, c, b);
#else
  const double s = (double)a * c + (double)b;  // exact: 48 bits
  const float f = (float)s;
  return fabs((double)f) > fabs(s) ? f32_of(bits_of(f) - 1) : f;
#endif
}
// 24 bits of v from bit S on, as a float
template <int S> KBC_HD float window(fx v, uint32_t sticky) {
  return (float)(int32_t)(((uint32_t)((uint64_t)v >> S) & 0xffffffu) | sticky);
}

// v * 2^-(60 + N) in FP32, rounded to nearest even. The short way, for 2^38 <= |v| < 2^60: the sum
// of bits 36 and above and of the 24 below, both exact in FP32, is rounded once; the last 12 bits
// count as a sticky bit, two places below the rounding one. Less than that is normalised first
// (that way for every value took 36 of the 57 instructions a population of an FP32
// initialisation: 256^3 1.00 -> 0.77 ms).
KBC_HD bool short_way(fx v) { return (uint32_t)((int32_t)((uint64_t)v >> 32) + 64) >= 128u; }
template <int N> KBC_HD float to_f32_short(fx v) {
  return add_rn<24 + N>((float)((int32_t)((uint64_t)v >> 32) >> 4),
                        mulf(window<12>(v, ((uint32_t)v & 0xfffu) != 0),
                             1.0f / (float)(1ull << (48 + N))));
}
template <int N> KBC_HD float to_f32(fx v) {
  if (short_way(v)) return to_f32_short<N>(v);
  const uint64_t a = v < 0 ? 0 - (uint64_t)v : (uint64_t)v;
  const int lz = clz64(a);
  const uint64_t q = lz == 64 ? 0 : a << lz;
  // the leading 32 bits, the rest as a sticky bit: the conversion rounds at bit 24
  const uint32_t t = (uint32_t)(q >> 32) | ((uint32_t)q != 0 ? 1u : 0u);
  const uint32_t b = bits_of((float)t);  // t 2^(32 - lz) of the units
  const uint32_t r = t == 0 ? 0 : b + ((uint32_t)(32 - kFrac - N - lz) << 23);
  return f32_of(r | ((uint32_t)((uint64_t)v >> 32) & 0x80000000u));
}
// The same rounded to odd: towards zero, with the last bit set where that is not exact, for a
// further rounding to a shorter type, which then rounds v itself, ties to even, as long as it has at
// most 22 bits of v from 2^16 units, 2^-44, on. |v| < 2^63. FP16 initialisation of 256^3: 1.08 ->
// 0.87 ms.
template <int N> KBC_HD float to_f32_odd(fx v) {
  const float a = (float)((int32_t)((uint64_t)v >> 32) >> 8);
  const float b = mulf(window<16>(v, ((uint32_t)v & 0xffffu) != 0), 1.0f / (float)(1ull << (44 + N)));
  const float f = add_rz<20 + N>(a, b);
  const float part = add_rn<20 + N>(-a, f);  // exact: what f holds of b
  return f32_of(bits_of(f) | (part != b ? 1u : 0u));
}

// ------------------------------------------------------------------ products
// v = h 2^32 + l with both halves signed, for the product below
struct Split {
  int32_t h, l;
};
KBC_HD constexpr Split split(fx v) {
  const uint32_t lo = (uint32_t)(uint64_t)v;
  return Split{(int32_t)((uint32_t)((uint64_t)v >> 32) + (lo >> 31)), (int32_t)lo};
}
KBC_HD constexpr int32_t mul_high(int32_t a, int32_t b) {
#ifdef __CUDA_ARCH__
  return __mulhi(a, b);
#else
  return (int32_t)(((long long)a * b) >> 32);
#endif
}
// a b / 2^64 to nearest, but for l x l (less than 1/4 unit, of either sign), which is dropped:
// within 3/4 of a unit, 0 for a factor 0. |a| < 2^62.9 and |b| < 2^63 - 2^31 keep the cross terms'
// sum in 64 bits.
KBC_HD fx mul(Split a, Split b) {
#ifdef __CUDA_ARCH__
  long long c, r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(c) : "r"(a.l), "r"(b.h), "l"(0x80000000ll));
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(c) : "r"(a.h), "r"(b.l), "l"(c));
  asm("mad.wide.s32 %0, %1, %2, %3;"
      : "=l"(r)
      : "r"(a.h), "r"(b.h), "l"((long long)(int32_t)(c >> 32)));
  return r;
#else
  const long long c = (long long)a.h * b.l + ((long long)a.l * b.h + 0x80000000ll);
  return (long long)a.h * b.h + (int32_t)(c >> 32);
#endif
}
// The same with each cross term rounded down, a unit low on average unless a factor is 0: two high
// halves instead of two wide multiplies, which take twice as long (256^3 FP64 pull with every product
// to nearest is 8 % slower than with the 81 innermost entropic ones by this). For sums that start with
// what they will lose.
KBC_HD fx mul_down(Split a, Split b) {
  return (long long)a.h * b.h + (mul_high(a.h, b.l) + mul_high(a.l, b.h));
}
// a factor below 1/2 in magnitude, scaled by 2^4 so that mul() gives a product of unit 2^-60
KBC_HD constexpr Split factor(fx v) { return split((fx)((uint64_t)v << 4)); }

// 1/3 (rounded)
constexpr fx kThird = 384307168202282325ll;

// 1 / rho for 0.4 < rho < 2: FP32 reciprocal r0 in units of 2^-28, then r0 (1 + E + E^2) with
// E = 1 - rho r0 to 2^-58 (|E| < 2^-21, so E^3 < 2^-63)
KBC_HD fx reciprocal(fx rho) {
  const int32_t rh = (int32_t)((uint64_t)rho >> 32);
  const int32_t r0 = f2i(mulf(rcpf((float)rh), 72057594037927936.0f));  // (2^28 / 2^-28) / rh
  const uint32_t rl = (uint32_t)(((uint64_t)(uint32_t)rho * (uint32_t)(r0 << 2)) >> 32);
  const fx E = kOne - (fx)((uint64_t)((((long long)rh * r0) << 2) + rl) << 2);
  const int32_t Eh = (int32_t)(E >> 16);
  // the low 16 bits of E, and E^2
  const int32_t El = (int32_t)((uint32_t)E & 0xffffu) + (int32_t)(((long long)Eh * Eh) >> 28);
  return ((fx)r0 << 32) + (((long long)r0 * Eh) >> 12) + mul_high(r0, El << 4);
}

// e 2^s with e = sqrt(1 + 3u^2) - 1, the root of e^2 + 2e = t = 3u^2, for |u| 2^s < 1/4 (us is
// u 2^s, u4 the factor of u; ps = 2^-s): an FP32 value e0 of e 2^s (unit 2^-32, good to 2^-24), then
// x = d - g d^2 2^-s with d = g r, r = t 2^s - 2 e0 - e0^2 2^-s exact in integers and
// g = 1 / (2 + 2e) to 2^-30 (one Newton step on the FP32 reciprocal)
KBC_HD fx axis_e(Split u4, fx us, uint32_t s, float ps) {
  const fx uu = mul(split(us), u4);
  const fx t = uu + uu + uu;
  const float tf = mulf((float)(int32_t)(t >> 29), 1.0f / 2147483648.0f);
  const float ef = mulf(tf, rcpf(addf(1.0f, sqrtf_fast(addf(1.0f, mulf(tf, ps))))));
  const int32_t e0 = f2i(mulf(ef, 4294967296.0f));
  const fx r = t - ((fx)e0 << 29) - sar(((long long)e0 * e0) >> 4, s);  // |r| < 2^37
  int32_t g = f2i(mulf(rcpf(addf(1.0f, mulf(ef, ps))), 1073741824.0f));  // 1 / (1 + e) of 2^30
  // g (1 + e) of 2^60, less 1, over 2^30
  const int32_t off =
      (int32_t)((((long long)g << 30) + sar(((long long)g * e0) >> 2, s) - kOne) >> 30);
  g -= off;
  // r / (2 (1 + e)) of 2^63
  const long long d =
      ((long long)(int32_t)(r >> 6) * g + (mul_high((int32_t)(r & 63) << 25, g) << 1)) >> 22;
  const int32_t ds = (int32_t)(d >> 9);                 // of 2^54, below 2^31
  const int32_t x2 = mul_high(mul_high(ds, ds), g);     // d^2 / (1 + e) of 2^74
  return ((fx)e0 << 28) + ((d - sar32(x2, s + 12)) >> 3);
}
// 2^-s
KBC_HD float pow2_of(uint32_t s) { return f32_of((127 - s) << 23); }

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
KBC_HD uint32_t high(fx v) {
  const int32_t h = (int32_t)((uint64_t)v >> 32);
  return (uint32_t)(h ^ (h >> 31));
}
KBC_HD uint32_t magnitude_low(fx v) { return (uint32_t)magnitude(v); }
KBC_HD int clz32(uint32_t x) {
#ifdef __CUDA_ARCH__
  return __clz((int)x);
#else
  return x ? __builtin_clz(x) : 32;
#endif
}
KBC_HD fx shl(fx v, int n) { return (fx)((uint64_t)v << n); }

// f_eq(1 + drho, u) - W, times 2^s, for drho 2^s and u 2^s below 1/4: its moments, transformed
// back; population i times 2^nonzero(i). The sum of the populations is drho exactly. The moments are
// built from what they deviate by from those of the weights, which scales like the shifts:
// rho m_2 - 1/3 = drho m_2 + (m_2 - 1/3), and so on.
KBC_HD void equilibrium(fx drho, fx ux, fx uy, fx uz, fx (&m)[27], uint32_t s = 0) {
  const float ps = pow2_of(s);
  const Split ux4 = factor(sar(ux, s)), uy4 = factor(sar(uy, s)), uz4 = factor(sar(uz, s));
  const Split third = factor(kThird);
  const fx ex = axis_e(ux4, ux, s, ps), ey = axis_e(uy4, uy, s, ps), ez = axis_e(uz4, uz, s, ps);
  // second moments of the axis factors less 1/3: 2e/3
  const fx vx = mul(split(ex + ex), third), vy = mul(split(ey + ey), third),
           vz = mul(split(ez + ez), third);
  const Split wx4 = factor(kThird + sar(vx, s)), wy4 = factor(kThird + sar(vy, s)),
              wz4 = factor(kThird + sar(vz, s));
  const Split rs = split(drho);
  m[mi(0, 0, 0)] = drho;
  m[mi(1, 0, 0)] = ux + mul(rs, ux4);
  m[mi(0, 1, 0)] = uy + mul(rs, uy4);
  m[mi(0, 0, 1)] = uz + mul(rs, uz4);
  const Split jxs = split(m[mi(1, 0, 0)]), jys = split(m[mi(0, 1, 0)]);
  const Split jzs = split(m[mi(0, 0, 1)]);
  m[mi(1, 1, 0)] = mul(jxs, uy4);
  m[mi(1, 0, 1)] = mul(jxs, uz4);
  m[mi(0, 1, 1)] = mul(jys, uz4);
  const Split pxys = split(m[mi(1, 1, 0)]);
  m[mi(1, 2, 0)] = mul(jxs, wy4);
  m[mi(1, 0, 2)] = mul(jxs, wz4);
  m[mi(2, 1, 0)] = mul(jys, wx4);
  m[mi(0, 1, 2)] = mul(jys, wz4);
  m[mi(2, 0, 1)] = mul(jzs, wx4);
  m[mi(0, 2, 1)] = mul(jzs, wy4);
  m[mi(1, 1, 1)] = mul(pxys, uz4);
  m[mi(2, 1, 1)] = mul(split(m[mi(0, 1, 1)]), wx4);
  m[mi(1, 2, 1)] = mul(split(m[mi(1, 0, 1)]), wy4);
  m[mi(1, 1, 2)] = mul(pxys, wz4);
  m[mi(2, 2, 1)] = mul(split(m[mi(2, 0, 1)]), wy4);
  m[mi(2, 1, 2)] = mul(split(m[mi(2, 1, 0)]), wz4);
  m[mi(1, 2, 2)] = mul(split(m[mi(1, 2, 0)]), wz4);
  m[mi(2, 0, 0)] = mul(rs, wx4) + vx;
  m[mi(0, 2, 0)] = mul(rs, wy4) + vy;
  m[mi(0, 0, 2)] = mul(rs, wz4) + vz;
  const fx ty = mul(split(vy), third), tz = mul(split(vz), third);
  const Split rxs = split(m[mi(2, 0, 0)]);
  m[mi(2, 2, 0)] = mul(rxs, wy4) + ty;
  m[mi(2, 0, 2)] = mul(rxs, wz4) + tz;
  m[mi(0, 2, 2)] = mul(split(m[mi(0, 2, 0)]), wz4) + tz;
  m[mi(2, 2, 2)] = mul(split(m[mi(2, 2, 0)]), wz4) + mul(split(tz), third);
  to_populations(m);
}

// the parameters of the collision as integers
struct Relax {
  fx quarter_beta;     // beta / 4 of 2^64: 2 beta = 8 x this
  fx two_beta_1;       // 2 beta - 1 of 2^62
  double inv_beta;     // for the value of gamma that is recorded
  int with_t, with_q, gamma_mode;
};
inline __host__ __device__ fx quarter_beta(double beta) {
  return (fx)(beta * 4611686018427387904.0);
}
inline __host__ __device__ fx two_beta_1(double beta) {
  return (fx)((2.0 * beta - 1.0) * 4611686018427387904.0);
}

// beta gamma = 1 - (2 beta - 1) q, q = num / den 2^e, as factor 2^k (k >= 3): the result is
// (beta gamma) 2^(64 - k), |result| < 2^62.6; num = 0 gives 1
KBC_HD fx relax_factor(fx num, fx den, int e, fx two_beta_1, int* k) {
  const int ld = clz64((uint64_t)den), ln = clz64(magnitude(num) | 1);
  const fx r = reciprocal(shl(den, ld - 1) >> 3);        // den in [1/2, 1): 1 / den in (1, 2]
  const fx n = shl(num, ln - 1) >> 3;                    // |num| in [1/2, 1)
  const fx q = mul(split(shl(n, 2)), split(shl(r, 1)));  // of 2^59, |q| < 2
  const fx t = mul(split(shl(q, 2)), split(two_beta_1));  // of 2^59, |t| < 2
  e += ld - ln;
  const int up = e > 0 ? (e > 60 ? 60 : e) : 0, down = e < 0 ? (e < -63 ? 63 : -e) : 0;
  *k = 3 + up;
  return shl(((1ll << 59) >> up) - (t >> down), 2);
}

// One KBC collision (Sec. KBC, natural moments, product-form equilibrium) of the shifts d 2^s,
// |d_i| 2^s < 1/4, in place; the result d_i is f'_i - W_i, or with CHANGE f'_i - f_i, times
// 2^(s + nonzero(i)) (to_f64<nonzero(i)>). The conserved moments of a change are exactly 0.
// Returns gamma; *guarded is set when <dh|dh> is 0 (gamma = 2), *bad when the node is outside
// the format's range (d is then not a result).
template <bool CHANGE = false>
KBC_HD double collide(fx (&d)[27], const Relax& rx, int* guarded, bool* bad, uint32_t s = 0) {
  // FP32 results need no products to nearest (all nodes of 256^3: 4.7 -> 4.2 ms)
  auto times = [](Split a, Split b) { return CHANGE ? mul(a, b) : mul_down(a, b); };
  to_moments(d);
  const fx dr = d[0], jx = d[mi(1, 0, 0)], jy = d[mi(0, 1, 0)], jz = d[mi(0, 0, 1)];
  const fx rho = kOne + sar(dr, s);
  const float ps = pow2_of(s);
  // 1/2 < rho < 2, |rho u| < 1/4, |u| < 1/4, the velocities times 2^s
  *bad = rho <= (kOne >> 1) || rho >= 2 * kOne ||
         ((magnitude(jx) | magnitude(jy) | magnitude(jz)) >> 58) != 0;
  *guarded = 0;
  const Split ir = split(reciprocal(rho));
  const fx usx = times(ir, factor(jx)), usy = times(ir, factor(jy)), usz = times(ir, factor(jz));
  *bad = *bad || ((magnitude(usx) | magnitude(usy) | magnitude(usz)) >> 58) != 0;
  const fx ux = sar(usx, s), uy = sar(usy, s), uz = sar(usz, s);
  const Split ux4 = factor(ux), uy4 = factor(uy), uz4 = factor(uz);
  const fx esx = axis_e(ux4, usx, s, ps), esy = axis_e(uy4, usy, s, ps),
           esz = axis_e(uz4, usz, s, ps);
  const fx ex = sar(esx, s), ey = sar(esy, s), ez = sar(esz, s);
  // second moments of the axis factors, m_2(u) = 1/3 + 2e/3: less 1/3 and times 2^s, and as factors
  const Split third = factor(kThird);
  const fx vx = times(split(esx + esx), third), vy = times(split(esy + esy), third),
           vz = times(split(esz + esz), third);
  const Split wx4 = factor(kThird + sar(vx, s)), wy4 = factor(kThird + sar(vy, s)),
              wz4 = factor(kThird + sar(vz, s));

  // deviations A = M - rho M_eq (the moments of f - f_eq), times 2^s; M and rho M_eq are both less
  // the weights' moments, as in equilibrium(). s is relaxed by 2 beta at once, the moments of h
  // (and the third ones, which are in s or in h) are kept in H
  const Split bs = split(rx.quarter_beta);
  auto relax_s = [&](int m, fx a) { d[m] -= times(split(shl(a, 3)), bs); };
  const Split rs = split(dr), jxs = split(jx), jys = split(jy), jzs = split(jz);
  const fx rwx = times(rs, wx4) + vx, rwy = times(rs, wy4) + vy, rwz = times(rs, wz4) + vz;
  const Split rwxs = split(rwx);
  const fx pxy = times(jxs, uy4), pxz = times(jxs, uz4), pyz = times(jys, uz4);
  const Split pxys = split(pxy);
  const fx jxwy = times(jxs, wy4), jywx = times(jys, wx4), jzwx = times(jzs, wx4);
  const fx ty = times(split(vy), third), tz = times(split(vz), third);
  const fx rwxwy = times(rwxs, wy4) + ty;
  fx H[27];
  H[mi(2, 2, 0)] = d[mi(2, 2, 0)] - rwxwy;
  H[mi(2, 0, 2)] = d[mi(2, 0, 2)] - (times(rwxs, wz4) + tz);
  H[mi(0, 2, 2)] = d[mi(0, 2, 2)] - (times(split(rwy), wz4) + tz);
  H[mi(2, 1, 1)] = d[mi(2, 1, 1)] - times(split(pyz), wx4);
  H[mi(1, 2, 1)] = d[mi(1, 2, 1)] - times(split(pxz), wy4);
  H[mi(1, 1, 2)] = d[mi(1, 1, 2)] - times(pxys, wz4);
  H[mi(2, 2, 1)] = d[mi(2, 2, 1)] - times(split(jzwx), wy4);
  H[mi(2, 1, 2)] = d[mi(2, 1, 2)] - times(split(jywx), wz4);
  H[mi(1, 2, 2)] = d[mi(1, 2, 2)] - times(split(jxwy), wz4);
  H[mi(2, 2, 2)] = d[mi(2, 2, 2)] - (times(split(rwxwy), wz4) + times(split(tz), third));
  fx q[7];  // 120, 102, 210, 012, 201, 021, 111
  q[0] = d[mi(1, 2, 0)] - jxwy;
  q[1] = d[mi(1, 0, 2)] - times(jxs, wz4);
  q[2] = d[mi(2, 1, 0)] - jywx;
  q[3] = d[mi(0, 1, 2)] - times(jys, wz4);
  q[4] = d[mi(2, 0, 1)] - jzwx;
  q[5] = d[mi(0, 2, 1)] - times(jzs, wy4);
  q[6] = d[mi(1, 1, 1)] - times(pxys, uz4);
  fx sxy = d[mi(1, 1, 0)] - pxy, sxz = d[mi(1, 0, 1)] - pxz, syz = d[mi(0, 1, 1)] - pyz;
  fx sx = d[mi(2, 0, 0)] - rwx, sy = d[mi(0, 2, 0)] - rwy, sz = d[mi(0, 0, 2)] - rwz;
  if constexpr (CHANGE) {
#pragma unroll
    for (int i = 0; i < 27; ++i) d[i] = 0;
  }
  // the trace belongs to s (with_t) or, spread over the three diagonal moments, to h
  const fx ht = rx.with_t ? 0 : times(split(sx + sy + sz), third);
  sx -= ht, sy -= ht, sz -= ht;
  H[mi(2, 0, 0)] = H[mi(0, 2, 0)] = H[mi(0, 0, 2)] = ht;
  H[mi(0, 0, 0)] = H[mi(1, 0, 0)] = H[mi(0, 1, 0)] = H[mi(0, 0, 1)] = 0;
  H[mi(1, 1, 0)] = H[mi(1, 0, 1)] = H[mi(0, 1, 1)] = 0;
  const int qm[7] = {mi(1, 2, 0), mi(1, 0, 2), mi(2, 1, 0), mi(0, 1, 2),
                     mi(2, 0, 1), mi(0, 2, 1), mi(1, 1, 1)};
  const fx keep = rx.with_q ? -1ll : 0ll;
  relax_s(mi(2, 0, 0), sx);
  relax_s(mi(0, 2, 0), sy);
  relax_s(mi(0, 0, 2), sz);
  relax_s(mi(1, 1, 0), sxy);
  relax_s(mi(1, 0, 1), sxz);
  relax_s(mi(0, 1, 1), syz);
  uint32_t smh = high(sx) | high(sy) | high(sz) | high(sxy) | high(sxz) | high(syz);
#pragma unroll
  for (int n = 0; n < 7; ++n) {
    H[qm[n]] = q[n] & ~keep;
    q[n] &= keep;
    relax_s(qm[n], q[n]);
    smh |= high(q[n]);
  }
  // scaling to below 2^59: a scaled population is a sum of at most 8 moments
  uint32_t hmh = high(ht);
#pragma unroll
  for (int i = 0; i < 27; ++i)
    if (i % 3 + (i / 3) % 3 + i / 9 >= 3) hmh |= high(H[i]);
  int hs = clz32(hmh) - 5, ss = clz32(smh) - 5;
  bool none = false;  // nothing in h
  if (hmh == 0 || smh == 0) {  // deviations below 2^-28: look at the low words too
    uint32_t hl = magnitude_low(ht), sl = magnitude_low(sx) | magnitude_low(sy) |
             magnitude_low(sz) | magnitude_low(sxy) | magnitude_low(sxz) | magnitude_low(syz);
    for (int i = 0; i < 27; ++i) hl |= magnitude_low(H[i]);
    for (int n = 0; n < 7; ++n) sl |= magnitude_low(q[n]);
    if (hmh == 0) hs = 32 + clz32(hl) - 5;
    if (smh == 0) ss = 32 + clz32(sl) - 5;
    none = hmh == 0 && hl == 0;
  }
  *bad = *bad || hs < 0 || ss < 0;  // deviations of 1/2 or more
  const int hz = hs + 5;
  hs = hs < 0 ? 0 : hs;
  ss = ss < 0 ? 0 : ss;

  double gamma = 2.0;
  int k = 3;                 // beta gamma = 2^k x (factor cs of 2^64)
  fx cf = rx.quarter_beta;   // gamma = 2
  if (rx.gamma_mode == 2) {  // gamma = 1 / beta
    gamma = rx.inv_beta;
    cf = 1ll << 61;          // 1 = 8 x 1/8
  } else if (rx.gamma_mode == 0) {
    // ---- gamma by eq:result21: ds and dh as populations, population i times 2^nonzero(i) (the
    // factors 4 of a product are taken up by the weights)
#pragma unroll
    for (int i = 0; i < 27; ++i) H[i] = shl(H[i], hs);
    sx = shl(sx, ss), sy = shl(sy, ss), sz = shl(sz, ss);
    sxy = shl(sxy, ss), sxz = shl(sxz, ss), syz = shl(syz, ss);
#pragma unroll
    for (int n = 0; n < 7; ++n) q[n] = shl(q[n], ss);
    // Table 1 by class: centre -(sx + sy + sz), faces 2 ds = s -+ (Q + Q'), edges
    // 4 ds = +-P +- Q +- Q', corners 8 ds = +-Q_xyz
    const fx s0 = sx + sy + sz;
    const fx Gx = q[0] + q[1], Gy = q[2] + q[3], Gz = q[4] + q[5];
    // the weights 1 / f_eq of the entropic products, per axis and but for common factors, which
    // drop out of the ratio: 1 / phi_+- = 6 / (1 + 2e +- 3u) and 1 / phi_0 = 6 / (4 (1 - e)). As
    // e^2 + 2e = 3u^2, (1 + 2e + 3u)(1 + 2e - 3u) = (1 - e)^2, so that with the factor 4 of the +-
    // populations they are (1 + 2e -+ 3u) : (1 - e) : no reciprocal is needed. An eighth of them
    // as factors of 2^64.
    Split w[3][3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const fx e = a == 0 ? ex : (a == 1 ? ey : ez), u = a == 0 ? ux : (a == 1 ? uy : uz);
      const fx b = kOne + e + e, u3 = u + u + u;
      w[a][0] = split(shl(b + u3, 1));
      w[a][1] = split(shl(kOne - e, 1));
      w[a][2] = split(shl(b - u3, 1));
    }
    const fx lost = CHANGE ? 0 : 3;
    fx num = lost, den = lost;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      fx L[9], cn = lost, cd = lost;  // the level's moments in x and y
#pragma unroll
      for (int m = 0; m < 9; ++m)
        L[m] = c == 1 ? H[m] - H[m + 18] : (c == 2 ? H[m + 18] + H[m + 9] : H[m + 18] - H[m + 9]);
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        // the row's moments in x; the sums start with the unit that each product loses
        fx R[3], rn = b != 1 && c != 1 ? 1 - 2 * keep : 3, rd = 3;
#pragma unroll
        for (int m = 0; m < 3; ++m)
          R[m] = b == 1 ? L[m] - L[m + 6] : (b == 2 ? L[m + 6] + L[m + 3] : L[m + 6] - L[m + 3]);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          const int va = a - 1, vb = b - 1, vc = c - 1;
          const int nz = nonzero(a + 3 * b + 9 * c);
          const fx h = a == 1 ? R[0] - R[2] : (a == 2 ? R[2] + R[1] : R[2] - R[1]);
          fx s;
          if (nz == 0) {
            s = -s0;
          } else if (nz == 1) {
            s = va ? (va > 0 ? sx - Gx : sx + Gx)
                   : vb ? (vb > 0 ? sy - Gy : sy + Gy) : (vc > 0 ? sz - Gz : sz + Gz);
          } else if (nz == 2) {
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
          const Split hh = split(h), t = split(mul_down(hh, w[0][a]));  // below 2^62, 2^60.3
          rn += mul_down(split(s), t);
          rd += mul_down(hh, t);  // below 2^58.3 each
        }
        cn += times(split(shl(rn, 2)), w[1][b]);  // a row below 2^62, half of its weighted sum
        cd += times(split(shl(rd, 2)), w[1][b]);
      }
      num += times(split(shl(cn, 1)), w[2][c]);
      den += times(split(shl(cd, 1)), w[2][c]);
    }
    if (!none) {
      // the unscaled deviations: num carries 2^(hs + ss), den 2^(2 hs)
      cf = relax_factor(num, den, hs - ss, rx.two_beta_1, &k);
      *bad = *bad || den <= 0 || k > 10 || hz < k + 2;
      gamma = rx.inv_beta * ((double)cf * f64_of((uint64_t)(1023 - 64 + k) << 52));
      k = k > 10 ? 10 : k;
    } else {
      *guarded = 1;  // every moment of h is 0 or -1 unit
    }
#pragma unroll
    for (int i = 0; i < 27; ++i) H[i] = H[i] >> hs;
  }
  // the moments of h: M - beta gamma A
  const Split cs = split(cf);
#pragma unroll
  for (int i = 0; i < 27; ++i) {
    const int order = i % 3 + (i / 3) % 3 + i / 9;
    if (order >= 3 || (order == 2 && (i == mi(2, 0, 0) || i == mi(0, 2, 0) || i == mi(0, 0, 2))))
      d[i] -= times(split(shl(H[i], k)), cs);
  }
  to_populations(d);
  return gamma;
}

// ------------------------------------------------------------------ density pre-solve
// rho - 1 of the shifts d, for the pre-solve and the measure of its change, which both take it from
// here. In fixed point: v receives the shifts (times 2^s), *sum their sum, *in_range says that they
// fit (the sum below 1/4, which that of a density shift is: 27/8 of the largest); FP64 sums otherwise.
KBC_HD double presolve_density(const double (&d)[27], fx (&v)[27], fx* sum, uint32_t* s,
                               uint32_t* top, bool* in_range) {
  *top = 0;
#pragma unroll
  for (int i = 0; i < 27; ++i) *top = top_of(d[i]) > *top ? top_of(d[i]) : *top;
  *in_range = scale_to<double, 4>(*top, s) && *top < kTopF64;
#pragma unroll
  for (int i = 0; i < 27; ++i) v[i] = scaled(d[i], *s);
  fx a = 0;
#pragma unroll
  for (int i = 0; i < 27; ++i) a += v[i];
  *sum = a;
  *in_range = *in_range && a > -(kOne >> 2) && a < (kOne >> 2);
  if (*in_range) return to_f64<0>(a, *s);
  double t = 0.0;
#pragma unroll
  for (int i = 0; i < 27; ++i) t += d[i];
  return t;
}

// One node of the pre-solve: p = f - beta2 (f - f_eq(rho(f), u)), times 2^(s + nonzero(i)); FULL:
// beta2 = 1, so that p is f_eq. What is stored is what the next iteration reads: the populations
// are rounded to units of the grid that it reads the shifts in, or to 53 bits of their class's
// largest and of the one at rest, so that the conversion to FP64 is exact, and the one at rest takes
// what that leaves of the density: the sum of what is read is the density again, to the bit. Otherwise the residues of the
// roundings, the same in every iteration of a settled node, add up in the density. *drho receives
// rho - 1 of d. False: not in the range.
template <bool FULL>
KBC_HD bool presolve(const double (&d)[27], double ux, double uy, double uz, double beta2,
                     fx (&p)[27], uint32_t* s, double* drho) {
  fx v[27], dr;
  uint32_t top, sd;
  bool ok;
  *drho = presolve_density(d, v, &dr, &sd, &top, &ok);
  // the velocity's scale, if smaller: |u| 2^s < 1/4
  const uint32_t tx = top_of(ux), ty = top_of(uy), tz = top_of(uz);
  uint32_t tu = tx > ty ? tx : ty, su;
  tu = tz > tu ? tz : tu;
  scale_to<double, 2>(tu, &su);
  *s = top == 0 || (su < sd && tu != 0) ? su : sd;
  ok = ok && tu < kTopF64 && *s <= kMaxScale;
  if (!ok) return false;
  const uint32_t less = sd > *s ? sd - *s : 0;
  dr = sar(dr, less);
  equilibrium(dr, scaled(ux, *s), scaled(uy, *s), scaled(uz, *s), p, *s);
  if constexpr (!FULL) {
    // f - beta2 (f - f_eq): beta2 / 8 < 1/4 as a factor of 2^64
    const Split b = split((fx)(beta2 * 2305843009213693952.0));
    uint32_t far = 0;
#pragma unroll
    for (int i = 0; i < 27; ++i) {
      v[i] = shl(sar(v[i], less), nonzero(i));
      p[i] = v[i] - p[i];
      far |= high(p[i]);
    }
    ok = (far >> 27) == 0;  // |f - f_eq| 2^N < 1/2
#pragma unroll
    for (int i = 0; i < 27; ++i) p[i] = v[i] - mul(split(shl(p[i], 3)), b);
  }
  uint32_t most[4] = {0, 0, 0, 0};
#pragma unroll
  for (int i = 0; i < 27; ++i) most[nonzero(i)] |= high(p[i]);
#pragma unroll
  for (int i = 0; i < 27; ++i) {
    const int N = nonzero(i);
    if (N == 0) continue;
    // bits above 53
    const int rest = 11 - clz32(most[0]), own = 11 - clz32(most[N]) - N;
    const int over = own > rest ? own : rest;
    const uint32_t n = N + (over > 0 ? over : 0);
    const fx q = sar(p[i] + (fx)(1ull << (n - 1)), n);  // to nearest
    dr -= shl(q, n - N);
    p[i] = shl(q, n);
  }
  p[13] = dr;
  return ok;
}

}  // namespace fix
}  // namespace kbc
