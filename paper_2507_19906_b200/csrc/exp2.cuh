// exp2 on two pipes.  The special-function unit gives one ex2 per 8 cycles and scheduler for a warp; a softmax
// over logits that the tensor cores deliver needs nothing else as much, so that unit is what the scoring
// kernels wait for.  A share of the exponentials is therefore evaluated on the FMA pipe, on PAIRS of values
// (the packed fp32 instructions do two per issue slot): 2^x = 2^n 2^f with n = round(x), f in [-1/2, 1/2], the
// second factor a polynomial of degree 6, the first put together in the exponent field.
// The coefficients are the minimax polynomial of 2^f on [-1/2, 1/2] in relative error (Remez exchange), rounded to fp32
// one after the other from 1 upwards with the rest fitted again: 3e-9; evaluated in fp32 6.5e-8 at most, 2.6e-8 rms and
// no bias, where ex2.approx has 1.4e-7, 6e-8 rms and a bias of -5e-8 (measured on [-30, 0]).  Degree 5 has 7.5e-8
// before any rounding and 6.5e-8 rms after it, and sums of exponentials were less exact with it than with ex2.
// Measured in a bare loop over accumulators in tensor memory, four warps per scheduler, cycles per warp-wide
// exponential and scheduler (degree 5): ex2 on scalars 8.8, on packed arguments 8.6; with 2, 4, 5, 6, 8, 16 pairs of 16 on
// the polynomial 7.6, 6.9, 6.6, 6.7, 7.7, 12.0.  Whole calls, us, with 0, 2, 3, 4 pairs of 16 (degree 6): 32 units x
// 256 rows x 32768 keys 379, 376, 371, 373; 4 x 448 x 131072 337, 332, 327, 328; accumulated scores of 32 heads x 8192
// tokens 728, 716, 708, 719; 8 x 128 x 8192 46.7, 46.2, 44.7, 44.5.  Hence 3.  (With unpacked arithmetic the
// polynomial costs ten issue slots per value, and any share of it loses.)
#pragma once

#include "common.cuh"

namespace calidrop {

using f32x2 = unsigned long long;   // two fp32 in one 64-bit register pair

__device__ __forceinline__ f32x2 pack2(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ f32x2 pack2(uint32_t a, uint32_t b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(a), "r"(b));
  return r;
}
__device__ __forceinline__ f32x2 pack2(float a) { return pack2(a, a); }
__device__ __forceinline__ float2 unpack2(f32x2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 d;
  asm("fma.rn.ftz.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("add.rn.ftz.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("mul.rn.ftz.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// fmaxf and fminf return the other operand for a NaN, and a NaN logit would leave no trace
__device__ __forceinline__ float max_nan(float a, float b) {
  float r;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float min_nan(float a, float b) {
  float r;
  asm("min.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}

// 2^x as a product of two factors, the second a power of two.  The argument is held at -127 from below, where the power
// of two is 0: like ex2.approx.ftz, the result underflows to 0 below -126, so that a sum over masked or far smaller
// logits is 0 and not a count of them.  kAbove: the argument may exceed 127 (it is then held at 128, and the result is
// infinite from 127.5 on); for logits relative to their own row's maximum or sum it cannot.
struct Exp2Factors {
  f32x2 p, pow2;
};
template <bool kAbove>
__device__ __forceinline__ Exp2Factors exp2_factors(f32x2 x) {
  constexpr float kRound = 12582912.f;   // 1.5 * 2^23: adding it rounds to an integer in the low mantissa bits
  constexpr float kExp2Poly[7] = {1.f, 0.6931471824645996f, 0.24022647738456726f, 0.05550359934568405f,
                                  0.009618505835533142f, 0.0013390806270763278f, 0.00015326471475418657f};
  float2 v = unpack2(x);
  v.x = max_nan(v.x, -127.f); v.y = max_nan(v.y, -127.f);
  if (kAbove) { v.x = min_nan(v.x, 128.f); v.y = min_nan(v.y, 128.f); }
  x = pack2(v.x, v.y);
  const f32x2 t = add2(x, pack2(kRound));
  const f32x2 f = fma2(add2(t, pack2(-kRound)), pack2(-1.f), x);
  f32x2 p = fma2(pack2(kExp2Poly[6]), f, pack2(kExp2Poly[5]));
  p = fma2(p, f, pack2(kExp2Poly[4]));
  p = fma2(p, f, pack2(kExp2Poly[3]));
  p = fma2(p, f, pack2(kExp2Poly[2]));
  p = fma2(p, f, pack2(kExp2Poly[1]));
  p = fma2(p, f, pack2(kExp2Poly[0]));
  const float2 tv = unpack2(t);
  return {p, pack2((__float_as_uint(tv.x) << 23) + 0x3f800000u, (__float_as_uint(tv.y) << 23) + 0x3f800000u)};
}

__device__ __forceinline__ f32x2 exp2_unit2(f32x2 x) {
  const float2 v = unpack2(x);
  return pack2(ex2_approx(v.x), ex2_approx(v.y));
}

// 2^x of one value on the FMA pipe, for the few factors by which partial sums are brought to a common maximum: they
// multiply whole sums, and the unit's bias of -5e-8 would add up from step to step.
__device__ __forceinline__ float exp2_unbiased(float x) {
  const Exp2Factors e = exp2_factors<false>(pack2(x));
  return unpack2(mul2(e.p, e.pow2)).x;
}

// Pair i of every 16 goes to the polynomial for kPolyPairs of them, evenly spread.
constexpr int kPolyPairs = 3;
__host__ __device__ constexpr bool exp2_pair_on_poly(int i) {
  return ((i % 16 + 1) * kPolyPairs) / 16 > ((i % 16) * kPolyPairs) / 16;
}

// 2^x and acc + 2^x of pair i (the addition costs the polynomial's pairs nothing: it takes the place of the product).
template <bool kAbove>
__device__ __forceinline__ f32x2 exp2_pair(f32x2 x, int i) {
  if (!exp2_pair_on_poly(i)) return exp2_unit2(x);
  const Exp2Factors e = exp2_factors<kAbove>(x);
  return mul2(e.p, e.pow2);
}
template <bool kAbove>
__device__ __forceinline__ f32x2 add_exp2_pair(f32x2 acc, f32x2 x, int i) {
  if (!exp2_pair_on_poly(i)) return add2(acc, exp2_unit2(x));
  const Exp2Factors e = exp2_factors<kAbove>(x);
  return fma2(e.p, e.pow2, acc);
}

}  // namespace calidrop
