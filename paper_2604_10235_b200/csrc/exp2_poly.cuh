// 2^x helpers shared by the score kernel, the chunk-scoring kernel and the throughput probe:
// the special-function instruction, the FMA-pipe polynomial, and the packed f32x2 arithmetic
// that the inner loops are written in.
#pragma once

#include <stdint.h>

namespace cc {

constexpr float kEx2Magic = 12582912.0f;         // 1.5 * 2^23: adding it rounds to the nearest integer
// 2^f on [-0.5, 0.5] by the cubic with the least mean error among those within 7.8e-5 of it (relative; a linear program over
// 2001 points).  The mean is what stays in a row's sum: 2.6e-6, against 5.8e-6 of an earlier fit and 8e-5 as the
// least maximum with a mean of zero.
constexpr float kEx2C3 = 0.05528990179300308f;
constexpr float kEx2C2 = 0.24261438846588135f;
constexpr float kEx2C1 = 0.6932293772697449f;
constexpr float kEx2C0 = 0.9999241828918457f;

__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// 2^x on the FMA pipe: x = n + f with n = round(x) taken from the low mantissa bits of
// x + 1.5 * 2^23, 2^f by the polynomial, n added into the exponent field.  Arguments are
// clamped at -125 so that the exponent never wraps (2^-125 is far below anything a score or a
// likelihood can resolve); the caller keeps x below 127.
__device__ __forceinline__ float ex2_poly(float x) {
  x = fmaxf(x, -125.0f);
  const float t = x + kEx2Magic;
  const float f = x - (t - kEx2Magic);
  float p = fmaf(f, kEx2C3, kEx2C2);
  p = fmaf(p, f, kEx2C1);
  p = fmaf(p, f, kEx2C0);
  return __int_as_float(__float_as_int(p) + (__float_as_int(t) << 23));
}

// packed f32x2 arithmetic (two values in a 64-bit register pair per instruction)
__device__ __forceinline__ uint64_t pack2(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
// 2^x for a pair on the special-function unit
__device__ __forceinline__ uint64_t ex2_pair_sfu(uint64_t x) {
  float a, b;
  unpack2(x, a, b);
  return pack2(ex2(a), ex2(b));
}
__device__ __forceinline__ uint64_t ex2_cubic(uint64_t f) {
  uint64_t p = fma2(f, pack2(kEx2C3, kEx2C3), pack2(kEx2C2, kEx2C2));
  p = fma2(p, f, pack2(kEx2C1, kEx2C1));
  return fma2(p, f, pack2(kEx2C0, kEx2C0));
}
// p * 2^n: n (low mantissa bits of t) shifted into the exponent field by one multiply-add
__device__ __forceinline__ uint64_t ex2_insert(uint64_t p, uint64_t t) {
  float p0, p1, t0, t1;
  unpack2(p, p0, p1);
  unpack2(t, t0, t1);
  int r0, r1;
  asm("mad.lo.s32 %0, %1, 8388608, %2;" : "=r"(r0) : "r"(__float_as_int(t0)), "r"(__float_as_int(p0)));
  asm("mad.lo.s32 %0, %1, 8388608, %2;" : "=r"(r1) : "r"(__float_as_int(t1)), "r"(__float_as_int(p1)));
  return pack2(__int_as_float(r0), __int_as_float(r1));
}
// 2^x for a pair on the FMA pipe (packed form of ex2_poly, same clamp)
__device__ __forceinline__ uint64_t ex2_pair_fma(uint64_t x) {
  float a, b;
  unpack2(x, a, b);
  x = pack2(fmaxf(a, -125.0f), fmaxf(b, -125.0f));
  const uint64_t magic = pack2(kEx2Magic, kEx2Magic);
  const uint64_t t = add2(x, magic);
  return ex2_insert(ex2_cubic(sub2(x, sub2(t, magic))), t);
}

constexpr float kScale = 0.12751743f;            // log2(e) / sqrt(128)
__device__ __forceinline__ float fma_sat(float a, float b, float c) {
  float d;
  asm("fma.rn.ftz.sat.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
// Two forms of 2^x for a pair on the FMA pipe, x given by the product v, for the two passes of the score kernel.  An argument
// rounded at its own size is good to 2^-20 between -16 and -32; its place on one scale of 248 powers of two, from a saturating
// multiply-add that clamps on both sides, is good to 2^-18 only and has a bias per reference, which is why neither form computes with one.
// Against 64 bits, geometric means over 17 shapes x 4 inputs: log-sums of rows 1.45e-6 with arguments of their own size, 1.47e-6
// from that scale, 1.14e-6 now; scores 3.70e-6, 3.71e-6, 3.66e-6 in norm.  The calls take 0 to 0.4 % more than with that scale, 1 % at the
// power limit; with arguments of their own size in pass 1 1.5 %, with the clamps as minima and maxima 0.7 %.
//
// Pass 1: acc + 2^(v * kScale - m), m an integer of at most kMaxRef in size.  n comes from the place of the argument on a scale that
// ends at -127 and 124 (the rounding there, 2^-10 at most and 2^-16 for references below 64, moves the border between one n and the next and nothing else).  The remainder takes the
// unrounded product and is rounded once, to 2^-25, since kEx2Magic - m is exact.  2^n is a factor of its own, 0 for n = -127:
// whatever the cubic makes of a remainder outside [-1/2, 1/2], where the scale has saturated, counts nothing below and is 2^124
// or more above.  (Only where the cubic overflows, below -2^43, the product with 0 is no number; the caller looks for that.)
constexpr float kMaxRef = 4096.0f;
constexpr float kPlaceLow = 127.0f, kPlaceSpan = 251.0f;
struct PolyRef { float bias, place; };
__device__ __forceinline__ PolyRef poly_ref(float m) { return PolyRef{kEx2Magic - m, (kPlaceLow - m) * (1.0f / kPlaceSpan)}; }
__device__ __forceinline__ uint64_t ex2_pair_scaled(float v0, float v1, const PolyRef& r, uint64_t acc) {
  const uint64_t y = pack2(fma_sat(v0, kScale / kPlaceSpan, r.place), fma_sat(v1, kScale / kPlaceSpan, r.place));
  const uint64_t t = fma2(y, pack2(kPlaceSpan, kPlaceSpan), pack2(kEx2Magic - kPlaceLow, kEx2Magic - kPlaceLow));    // magic + n
  const uint64_t p = ex2_cubic(fma2(pack2(v0, v1), pack2(kScale, kScale), sub2(pack2(r.bias, r.bias), t)));
  float t0, t1;
  unpack2(t, t0, t1);
  int s0, s1;                                      // n in the exponent field, 127 + n
  asm("mad.lo.s32 %0, %1, 8388608, 1065353216;" : "=r"(s0) : "r"(__float_as_int(t0)));
  asm("mad.lo.s32 %0, %1, 8388608, 1065353216;" : "=r"(s1) : "r"(__float_as_int(t1)));
  return fma2(p, pack2(__int_as_float(s0), __int_as_float(s1)), acc);
}
// Pass 2: 2^(v * kScale) for arguments of at most 0 (taken as 0 above).  The scale ends at -124 and 0 and is counted from its upper end,
// so the place is the argument rounded at its own size (kScale / kDepth is exact in f32).
constexpr float kDepth = 124.0f;
__device__ __forceinline__ uint64_t ex2_pair_below(float v0, float v1) {
  const uint64_t y = pack2(fma_sat(v0, -kScale / kDepth, 0.0f), fma_sat(v1, -kScale / kDepth, 0.0f)), span = pack2(-kDepth, -kDepth);
  const uint64_t magic = pack2(kEx2Magic, kEx2Magic), t = fma2(y, span, magic);
  return ex2_insert(ex2_cubic(fma2(y, span, sub2(magic, t))), t);
}

// Of every three pairs one takes the polynomial path, and the two paths have a sum each: the special-function unit is the
// fuller pipe (one pair in four: +3 to 5 % on the score kernel, six of sixteen: +5 %), and the order of the source decides how
// well it stays fed (polynomials bunched together: +3 to 7 %).  Which pairs they are decides which values carry the
// polynomial's error: another choice is as good, but moves scores by 2e-6 and with them some ties at the cut-off.
__device__ __forceinline__ constexpr bool poly_pair(int pair) { return pair % 3 == 2; }

// acc += 2^(v * kScale + off) over the first kWidth of 32 values; off per value from shared memory (off_col: shared-space address of
// the first one, so that the loads need no address arithmetic).  Arguments up to 64.
template <int kWidth>
__device__ __forceinline__ void exp_accumulate_columns(const uint32_t (&v)[32], uint32_t off_col, uint64_t (&acc)[2]) {
  const uint64_t c2 = pack2(kScale, kScale);
#pragma unroll
  for (int i = 0; i < kWidth; i += 4) {
    float4 L;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(L.x), "=f"(L.y), "=f"(L.z), "=f"(L.w)
                 : "r"(off_col + (uint32_t)(i * 4)));
    const uint64_t o[2] = {pack2(L.x, L.y), pack2(L.z, L.w)};
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const uint64_t x = fma2(pack2(__uint_as_float(v[i + 2 * k]), __uint_as_float(v[i + 2 * k + 1])), c2, o[k]);
      if (poly_pair((i >> 1) + k)) acc[1] = add2(acc[1], ex2_pair_fma(x));
      else acc[0] = add2(acc[0], ex2_pair_sfu(x));
    }
  }
}
// The same with one offset for all values, any number.
__device__ __forceinline__ void exp_accumulate_any(const uint32_t (&v)[32], float off, uint64_t (&acc)[2]) {
  const uint64_t c2 = pack2(kScale, kScale), off2 = pack2(off, off);
#pragma unroll
  for (int pair = 0; pair < 16; ++pair) {
    const uint64_t x = fma2(pack2(__uint_as_float(v[2 * pair]), __uint_as_float(v[2 * pair + 1])), c2, off2);
    if (poly_pair(pair)) acc[1] = add2(acc[1], ex2_pair_fma(x));
    else acc[0] = add2(acc[0], ex2_pair_sfu(x));
  }
}
// acc += 2^(v * kScale - m) over 32 values, m an integer of at most kMaxRef in size, r = poly_ref(m).
__device__ __forceinline__ void exp_accumulate(const uint32_t (&v)[32], float m, const PolyRef& r, uint64_t (&acc)[2]) {
  const uint64_t c2 = pack2(kScale, kScale), off2 = pack2(-m, -m);
#pragma unroll
  for (int pair = 0; pair < 16; ++pair) {
    const float a = __uint_as_float(v[2 * pair]), b = __uint_as_float(v[2 * pair + 1]);
    if (poly_pair(pair)) acc[1] = ex2_pair_scaled(a, b, r, acc[1]);
    else acc[0] = add2(acc[0], ex2_pair_sfu(fma2(pack2(a, b), c2, off2)));
  }
}
// acc += 2^(v * kScale) over the first kWidth of 32 values, arguments of at most 0.
template <int kWidth>
__device__ __forceinline__ void exp_accumulate_below(const uint32_t (&v)[32], uint64_t (&acc)[2]) {
  const uint64_t c2 = pack2(kScale, kScale);
#pragma unroll
  for (int pair = 0; pair < kWidth / 2; ++pair) {
    const float a = __uint_as_float(v[2 * pair]), b = __uint_as_float(v[2 * pair + 1]);
    if (poly_pair(pair)) acc[1] = add2(acc[1], ex2_pair_below(a, b));
    else acc[0] = add2(acc[0], ex2_pair_sfu(mul2(pack2(a, b), c2)));
  }
}
// The largest size of the values that take the polynomial path.
__device__ __forceinline__ float poly_reach(const uint32_t (&v)[32]) {
  float reach = 0.0f;
#pragma unroll
  for (int pair = 0; pair < 16; ++pair)
    if (poly_pair(pair))
      asm("max.f32 %0, %0, %1, %2;" : "+f"(reach) : "f"(fabsf(__uint_as_float(v[2 * pair]))), "f"(fabsf(__uint_as_float(v[2 * pair + 1]))));
  return reach;
}
__device__ __forceinline__ float acc_total(const uint64_t (&acc)[2]) {
  float a, b;
  unpack2(add2(acc[0], acc[1]), a, b);
  return a + b;
}

}  // namespace cc
