// pp_hx.cuh -- block-scaled integer + float arithmetic of the FP64-class line transforms.
//
// A line's values share one power-of-two scale; a value is h + l in units of it, h a 32-bit integer and l
// a float of a few units.  A sum is one integer add and one float add (the integer part is exact as long
// as it does not overflow, which the scale excludes), where a double-float sum takes eight FP32
// instructions (TwoSum and two adds): a butterfly of eight points with its seven twiddles takes 430
// issue slots a warp instead of 780 (measured in registers, GB300), and 63 registers instead of 80.  A
// product with a twiddle takes one 32 x 32 -> 64-bit multiply-add per real product for the integer parts
// and float FMAs for the rest.
//
// Scale.  The transforms are sums of unit-modulus multiples of a line's values, so the modulus of every
// intermediate is bounded by the sum of magnitudes l1 of the line, and after s stages by (product of their
// radices) x sqrt 2 x the largest magnitude.  The butterflies also form re + im and re - im (hrot8), which reach
// sqrt 2 times the modulus; hx_bounds says where that counts.  Every twiddle product is scaled by 1/4, which
// leaves room for most of a stage's growth.  The scale is the largest power of two that keeps every stage's
// integers within 0.95 2^31 by one of the two bounds; random lines then start near 2^26 and end near 2^25, a line with a single
// coefficient starts near 2^30, and the rounding of l (2^-25 of a unit) is 2^-49 to 2^-51 of the values;
// the unnormalised double-float pairs round their low parts at 2^-47.
//
// A line with a non-finite value becomes NaN as a whole (every output of a transform depends on every
// input).
#pragma once
#include <algorithm>
#include <cmath>

#include "pp_arith.cuh"

namespace pp {

struct hx {
  int h;
  float l;
};
__device__ __forceinline__ hx operator+(hx a, hx b) { return hx{a.h + b.h, a.l + b.l}; }
__device__ __forceinline__ hx operator-(hx a, hx b) { return hx{a.h - b.h, a.l - b.l}; }
__device__ __forceinline__ hx operator-(hx a) { return hx{-a.h, -a.l}; }

struct alignas(16) hcx {
  hx re, im;
};
__device__ __forceinline__ hcx operator+(hcx a, hcx b) { return hcx{a.re + b.re, a.im + b.im}; }
__device__ __forceinline__ hcx operator-(hcx a, hcx b) { return hcx{a.re - b.re, a.im - b.im}; }
__device__ __forceinline__ hcx hconj(hcx a) { return hcx{a.re, -a.im}; }

// A twiddle c + i s: the integers round(c 2^30), round(s 2^30), the floats c/4, s/4 (for l), and what the
// integers leave, (c - ci 2^-30) / 4, in a second array.
struct alignas(16) htwa {
  int c, s;
  float c0, s0;
};
struct alignas(8) htwb {
  float c1, s1;
};

// (host) +-1 as +-(2^30 - 1): products with 2^30 would end in ties, whose remainders have a mean (hquarter)
inline void hx_twiddle(double c, double s, htwa& a, htwb& b) {
  auto ints = [](double x) { return (int)std::max(-1073741823LL, std::min(1073741823LL, std::llround(x * 0x1p30))); };
  a = htwa{ints(c), ints(s), (float)(0.25 * c), (float)(0.25 * s)};
  b = htwb{(float)(0.25 * (c - a.c * 0x1p-30)), (float)(0.25 * (s - a.s * 0x1p-30))};
}

// The 64-bit sum rounded to its top word, and the signed remainder beside the float terms u.
__device__ __forceinline__ hx hx_fin(long long s, float u) {
  return hx{(int)(s >> 32) + (int)((unsigned)s >> 31), __fmaf_rn(__int2float_rn((int)s), 0x1p-32f, u)};
}
// x w / 4, or x conj(w) / 4
template <bool CONJ> __device__ __forceinline__ hcx hmul(hcx x, htwa w, htwb r) {
  const int s = CONJ ? -w.s : w.s;
  const float s0 = CONJ ? -w.s0 : w.s0, s1 = CONJ ? -r.s1 : r.s1;
  const float fr = __int2float_rn(x.re.h), fi = __int2float_rn(x.im.h);
  long long p = (long long)x.re.h * w.c;
  p += (long long)x.im.h * -s;
  float u = __fmul_rn(x.re.l, w.c0);
  u = __fmaf_rn(-x.im.l, s0, u);
  u = __fmaf_rn(fr, r.c1, u);
  u = __fmaf_rn(-fi, s1, u);
  long long q = (long long)x.re.h * s;
  q += (long long)x.im.h * w.c;
  float v = __fmul_rn(x.re.l, s0);
  v = __fmaf_rn(x.im.l, w.c0, v);
  v = __fmaf_rn(fr, s1, v);
  v = __fmaf_rn(fi, r.c1, v);
  return hcx{hx_fin(p, u), hx_fin(q, v)};
}
// x / 4 (the untwiddled partner of such a product), ties to even: the remainders must have no mean, or
// the rounding of the float twiddles c0 turns it into a constant error of the lowest modes
__device__ __forceinline__ hx hquarter(hx x) {
  const int q = (x.h + 1 + ((x.h >> 2) & 1)) >> 2;
  return hx{q, __fmul_rn(__fadd_rn(x.l, __int2float_rn(x.h - 4 * q)), 0.25f)};
}
__device__ __forceinline__ hcx hquarter(hcx x) { return hcx{hquarter(x.re), hquarter(x.im)}; }
// x / sqrt 2 = x + x (1/sqrt 2 - 1)
__device__ __forceinline__ hx hsqrt1_2(hx x) {
  constexpr double w = 0.70710678118654752440 - 1.0;
  constexpr int wi = -1257966796;  // round(w 2^32)
  constexpr float w1 = (float)(w - (double)wi * 0x1p-32);
  long long s = ((long long)x.h << 32);
  s += (long long)x.h * wi;
  float u = __fmul_rn(x.l, 0.70710678118654752f);
  u = __fmaf_rn(__int2float_rn(x.h), w1, u);
  return hx_fin(s, u);
}
// x exp(-i pi/4) (INV: exp(+i pi/4))
template <bool INV> __device__ __forceinline__ hcx hrot8(hcx x) {
  return INV ? hcx{hsqrt1_2(x.re - x.im), hsqrt1_2(x.im + x.re)} : hcx{hsqrt1_2(x.re + x.im), hsqrt1_2(x.im - x.re)};
}

// r-point DFTs in registers (forward kernel exp(-2 pi i / r); INV the conjugate).
template <bool INV> __device__ __forceinline__ void hdft2(hcx* a) {
  const hcx t = a[0];
  a[0] = t + a[1];
  a[1] = t - a[1];
}
template <bool INV> __device__ __forceinline__ void hdft4(hcx* a) {
  const hcx t0 = a[0] + a[2], t1 = a[0] - a[2], t2 = a[1] + a[3], d = a[1] - a[3];
  a[0] = t0 + t2;
  a[2] = t0 - t2;
  // t1 -+ i d
  const hcx m{t1.re + d.im, t1.im - d.re}, p{t1.re - d.im, t1.im + d.re};
  a[1] = INV ? p : m;
  a[3] = INV ? m : p;
}
template <bool INV> __device__ __forceinline__ void hdft8(hcx* a) {
  hcx e[4] = {a[0], a[2], a[4], a[6]}, o[4] = {a[1], a[3], a[5], a[7]};
  hdft4<INV>(e);
  hdft4<INV>(o);
  a[0] = e[0] + o[0];
  a[4] = e[0] - o[0];
  const hcx o1 = hrot8<INV>(o[1]);
  a[1] = e[1] + o1;
  a[5] = e[1] - o1;
  // o2 times -+i
  const hcx m{e[2].re + o[2].im, e[2].im - o[2].re}, p{e[2].re - o[2].im, e[2].im + o[2].re};
  a[2] = INV ? p : m;
  a[6] = INV ? m : p;
  // o3 times exp(-+3 i pi/4) = -+i exp(-+i pi/4): with r = exp(-+i pi/4) o3
  const hcx r = hrot8<INV>(o[3]);
  const hcx m3{e[3].re + r.im, e[3].im - r.re}, p3{e[3].re - r.im, e[3].im + r.re};
  a[3] = INV ? p3 : m3;
  a[7] = INV ? m3 : p3;
}
template <int RAD, bool INV> __device__ __forceinline__ void hdft(hcx* a) {
  if constexpr (RAD == 8) hdft8<INV>(a);
  else if constexpr (RAD == 4) hdft4<INV>(a);
  else hdft2<INV>(a);
}

// double-float <-> hx at scale S (a power of two); back with f = 1/S times what the products took off
__device__ __forceinline__ hx hx_from(df v, float S) {
  const float a = __fmul_rn(v.hi, S);
  const int h = __float2int_rn(a);
  const float r = __fmaf_rn(v.lo, S, __fsub_rn(a, __int2float_rn(h)));
  // r reaches 2^7 where h is large: its integer part joins h (round to nearest by adding 1.5 2^23)
  const float t = __fadd_rn(r, 12582912.0f);
  return hx{h + (__float_as_int(t) - 0x4b400000), __fsub_rn(r, __fsub_rn(t, 12582912.0f))};
}
__device__ __forceinline__ df hx_to(hx v, float f) {
  const float a = __int2float_rn(v.h);
  const float r = __int2float_rn(v.h - __float2int_rn(a));
  return df{__fmul_rn(a, f), __fmul_rn(__fadd_rn(r, v.l), f)};
}

// (h + l) 2^E as FP64, by integer operations (an FP64 add runs at 1/67 of the FP32 rate): the sum in units of
// 2^-22, where the rounding of l lies, shifted to an FP64 significand.  Values below 2^10 units (or zero)
// take the FP64 unit.
static __device__ __noinline__ double hx_to_double_small(long long m, int E) {
  return __dmul_rn(__ll2double_rn(m), __longlong_as_double((long long)(E - 22 + 1023) << 52));
}
__device__ __forceinline__ double hx_to_double(hx v, int E) {
  const int t = __float2int_rn(__fmul_rn(v.l, 0x1p22f));
  const long long m = (long long)v.h * (1 << 22) + t;
  const long long a = m < 0 ? -m : m;
  const int hi = (int)(a >> 32);
  if (hi == 0) return hx_to_double_small(m, E);
  const int sh = __clz(hi) - 11;  // leading bit to bit 20 of the high word (a < 2^53)
  const unsigned long long b = (unsigned long long)a << sh;
  // exponent field: 1023 + E - 22 + (position of the leading bit, 52 - sh); the leading bit itself adds one
  const unsigned top = (unsigned)(b >> 32) + ((unsigned)(1023 + E - 22 + 52 - 1 - sh) << 20);
  return __hiloint2double((int)(top | ((unsigned)(m >> 32) & 0x80000000u)), (int)(unsigned)b);
}

// Scale of a line from its largest magnitude and its sum of magnitudes: the largest power of two with
// S <= max(am_e / mx, as_e / l1) for every bound e.  l1 is summed in units of 2^12, so that the up to 2052 magnitudes
// of a line stay within FP32's range; it is infinite or NaN for non-finite values only.
constexpr float kHxSum = 0x1p-12f;
struct HScale {
  float am[6], as[6];  // limit / (bound per unit of the largest magnitude, of the sum in units of 2^12)
  int n;
  int out;             // exponent of the scale that the products took off
};
// (host) Bounds of one transform: every intermediate, per unit of the line's largest magnitude and of its sum
// of magnitudes, and the factors of 1/4 that the products take off.  iv: type IV; inv: C2R, DCT-III, DST-III;
// c2c; none of them: R2C, DCT-II, DST-II.  rad: the radices of the nst stages.
inline HScale hx_bounds(bool iv, bool inv, bool c2c, const int* rad, int nst) {
  HScale b = {};
  auto add = [&](double per_max, double per_sum) {
    b.am[b.n] = (float)(0.95 * 0x1p31 / per_max);
    b.as[b.n] = (float)(0.95 * 0x1p31 * kHxSum / per_sum);
    b.n++;
  };
  // before the first stage: the values themselves (type IV), sums of two pairs (inverse kinds)
  if (iv) add(1.0, 1.0);
  if (inv) add(2.5, 1.0);
  // In stage s: complex sums of R values of modulus <= sqrt 2 (after the pre-products / 4: type IV), and re +- im of
  // sums of R/2 of them.  By the sum of magnitudes: l1 bounds |re| + |im| of any sum of a line's own values, so
  // re +- im too (first stage of C2C and the forward kinds); once a twiddle has turned them it bounds the modulus,
  // and re +- im reach sqrt 2 l1.  (The pre-products of the inverse kinds turn theirs as well, but with
  // |E|^2 + |O|^2 = (|A|^2 + |B|^2) / 8 the two values of an item, E +- iO, have moduli of (|A| + |B|) / sqrt 2 at most
  // together.)
  double R = 1.0, off = iv ? 0.25 : 1.0;
  for (int s = 0; s < nst; s++) {
    R *= rad[s];
    // (the Hermitian split of the forward kinds adds two of the last stage's results)
    const double two = (s + 1 == nst && !iv && !inv && !c2c) ? 2.0 : 1.0;
    const double turned = (iv || (s > 0 && !inv)) ? std::sqrt(2.0) : 1.0;
    add(two * std::sqrt(2.0) * R * off, std::max(two, turned) * off);
    if (s + 1 < nst) off *= 0.25;
  }
  // products by 1/4: nst - 1 twiddled stages; the pre- and post-products; the forward split works with
  // twice the even and odd parts
  b.out = 2 * (nst - 1) + (iv ? 4 : inv ? 2 : c2c ? 0 : 1);
  return b;
}
__device__ __forceinline__ void hx_stat(float& mx, float& l1, float v) {
  mx = fmaxf(mx, fabsf(v));
  l1 = __fmaf_rn(fabsf(v), kHxSum, l1);
}
__device__ __forceinline__ float hx_scale(const HScale& b, float mx, float l1) {
  const float rm = __frcp_rn(mx), rl = __frcp_rn(l1);
  float s = 0x1p126f;
  for (int e = 0; e < b.n; e++) s = fminf(s, fmaxf(b.am[e] * rm, b.as[e] * rl));
  s = __uint_as_float(__float_as_uint(s) & 0x7f800000u);
  return l1 <= 3.4028234e38f ? s : __uint_as_float(0x7fc00000u);
}
__device__ __forceinline__ float hx_unscale(const HScale& b, float S) {
  return __uint_as_float((254u << 23) - (__float_as_uint(S) & 0x7f800000u) + ((unsigned)b.out << 23));
}

}  // namespace pp
