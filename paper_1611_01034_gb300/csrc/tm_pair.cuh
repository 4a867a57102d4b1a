// Arithmetic on unevaluated sums h + l of two FP32 numbers ("pairs").
//
// GB300 runs FP64 at 1/64 of its FP32 rate.  Where a result must be
// FP64-accurate but the arithmetic is heavy, every real is carried as a pair
// (Dekker's double-length arithmetic, Numer. Math. 18 (1971) 224, with
// Knuth's two-sum): the product a.h * b.h is made exact with an FMA, the cross
// terms and all rounding errors gather in l.  A pair holds about 47 bits of
// significand; products and sums lose a few bits more.
//
// Conversions go through integer operations on the bit patterns, so that no
// FP64 instruction is issued per element where it can be avoided:
//   d2pair: FP64 -> pair, h the FP64 value truncated to 24 significant bits, l
//           the remainder truncated to 24 bits (47 bits in all);
//   f2d_bits: FP32 -> FP64 exactly (normal numbers).
#pragma once
#include "tm_internal.cuh"
#include "tm_lane.cuh"

namespace tmamg {

// a value h + l
struct dfl {
  float h, l;
};

// error-free transforms (the _rn intrinsics are never contracted into FMAs)
__device__ __forceinline__ dfl two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return {s, e};
}
__device__ __forceinline__ void add_to(dfl& acc, dfl a) {
  const dfl s = two_sum(acc.h, a.h);
  acc.h = s.h;
  acc.l = __fadd_rn(acc.l, __fadd_rn(s.l, a.l));
}

// A complex pair number with its real and imaginary parts as the lanes of packed
// FP32 arithmetic: h = (re.h, im.h), l = (re.l, im.l).
struct pk2 {
  f2 h, l;
};

__device__ __forceinline__ pk2 two_sum2(f2 a, f2 b) {
  const f2 s = a + b;
  const f2 bb = s - a;
  return {s, (a - (s - bb)) + (b - bb)};
}
__device__ __forceinline__ void add_to(pk2& acc, pk2 a) {
  const pk2 s = two_sum2(acc.h, a.h);
  acc.h = s.h;
  acc.l = acc.l + (s.l + a.l);
}
// a factor as fma_px wants it: h, -h and -l
struct pn2 {
  f2 h, nh, nl;
};
// a pair broadcast to both lanes
__device__ __forceinline__ pn2 bc_pair(float h, float l) {
  return {f2_pack(h, h), f2_pack(-h, -h), f2_pack(-l, -l)};
}
// each lane its own factor
__device__ __forceinline__ pn2 lane_pair(pk2 a) {
  const float2 h = f2_unpack(a.h), l = f2_unpack(a.l);
  return {a.h, f2_pack(-h.x, -h.y), f2_pack(-l.x, -l.y)};
}
// acc += a x per lane, for x exact in FP32, and for x a pair (l l, 2^-48 relative, is dropped);
// ne = minus the rounding error of a.h x.h and the cross terms
__device__ __forceinline__ void fma_px(pk2& acc, pn2 a, f2 x) {
  const f2 p = a.h * x;
  f2 ne = lfma(a.nh, x, p);
  ne = lfma(a.nl, x, ne);
  const pk2 s = two_sum2(acc.h, p);
  acc.h = s.h;
  acc.l = acc.l + (s.l - ne);
}
__device__ __forceinline__ void fma_px(pk2& acc, pn2 a, pk2 x) {
  const f2 p = a.h * x.h;
  f2 ne = lfma(a.nh, x.h, p);
  ne = lfma(a.nh, x.l, ne);
  ne = lfma(a.nl, x.h, ne);
  const pk2 s = two_sum2(acc.h, p);
  acc.h = s.h;
  acc.l = acc.l + (s.l - ne);
}
// i x
__device__ __forceinline__ f2 times_i(f2 x) {
  const float2 v = f2_unpack(x);
  return f2_pack(-v.y, v.x);
}
__device__ __forceinline__ pk2 times_i(pk2 x) { return {times_i(x.h), times_i(x.l)}; }
// FP32 bits -> FP64 with integer operations (exact for normal numbers; FP32
// subnormals, below 1.2e-38, become zero)
__device__ __forceinline__ double f2d_bits(float f) {
  const unsigned u = __float_as_uint(f);
  const unsigned long long sgn = (unsigned long long)(u & 0x80000000u) << 32;
  const unsigned mag = u & 0x7fffffffu;
  if (mag < 0x00800000u) return __longlong_as_double((long long)sgn);
  if (mag >= 0x7f800000u) return (double)f;  // Inf, NaN
  const unsigned long long bits = sgn | (((unsigned long long)mag << 29) + (896ull << 52));
  return __longlong_as_double((long long)bits);
}

// FP64 -> pair by bit operations.  x = (-1)^s 2^E (1 + m / 2^52): h keeps the
// top 23 bits of m; the remaining 29 bits r give x - h = (-1)^s 2^(E-23) r / 2^29,
// formed exactly as the difference of the FP32 numbers 2^(E-23) (1 + (r >> 6) / 2^23)
// and 2^(E-23) (Sterbenz) after dropping r's lowest 6 bits.  Magnitudes below
// 2^-103 (where 2^(E-23) leaves the FP32 normal range) become 0; above the FP32
// range the ordinary conversion applies.
__device__ __forceinline__ dfl d2pair(double x) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const unsigned top = (unsigned)(u >> 32);
  const unsigned sgn = top & 0x80000000u;
  const int e = (int)((top >> 20) & 0x7ffu) - 1023;  // unbiased exponent
  if (e < -103) return dfl{__uint_as_float(sgn), 0.f};
  if (e > 127) return dfl{__double2float_rn(x), 0.f};
  const unsigned E = (unsigned)(e + 127);
  const float h = __uint_as_float(sgn | (E << 23) | ((unsigned)(u >> 29) & 0x7fffffu));
  const unsigned r = (unsigned)u & 0x1fffffffu;
  const unsigned El = (E - 23u) << 23;
  const float l = __fsub_rn(__uint_as_float(El | (r >> 6)), __uint_as_float(El));
  return dfl{h, sgn ? -l : l};
}

// pair -> FP64 (one FP64 addition)
__device__ __forceinline__ double pair2d(dfl a) { return f2d_bits(a.h) + f2d_bits(a.l); }

// both parts of a complex FP64 number, with fewer instructions where both are in range: shifted left
// by three, the high word has the FP32 mantissa in place and the exponent short of its bias; the
// sign goes with both numbers whose difference is l
__device__ __forceinline__ pk2 cx2pair(double re, double im) {
  const unsigned hr = (unsigned)__double2hiint(re), lr = (unsigned)__double2loint(re);
  const unsigned hm = (unsigned)__double2hiint(im), lm = (unsigned)__double2loint(im);
  const unsigned er = ((hr >> 20) & 0x7ffu) - 920u, ei = ((hm >> 20) & 0x7ffu) - 920u;
  if (max(er, ei) > 230u) {  // exponents beyond -103 .. 127, zeros too
    const dfl a = d2pair(re), b = d2pair(im);
    return {f2_pack(a.h, b.h), f2_pack(a.l, b.l)};
  }
  const unsigned ar = ((__funnelshift_l(lr, hr, 3) + 0x40000000u) & 0x7fffffffu) | (hr & 0x80000000u);
  const unsigned ai = ((__funnelshift_l(lm, hm, 3) + 0x40000000u) & 0x7fffffffu) | (hm & 0x80000000u);
  const unsigned br = (ar & 0xff800000u) - (23u << 23), bi = (ai & 0xff800000u) - (23u << 23);
  const unsigned cr = br | ((lr >> 6) & 0x7fffffu), ci = bi | ((lm >> 6) & 0x7fffffu);
  return {f2_pack(__uint_as_float(ar), __uint_as_float(ai)),
          f2_pack(__uint_as_float(cr), __uint_as_float(ci)) - f2_pack(__uint_as_float(br), __uint_as_float(bi))};
}

}  // namespace tmamg
