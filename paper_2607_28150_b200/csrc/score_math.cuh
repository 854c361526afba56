// Arithmetic that the two forms of the scoring kernel share: exponentials on the SFU and on the FMA pipe, and the sums over
// the columns of a chunk of scores.
#pragma once

#include "common.cuh"

namespace sg {

constexpr float kLog2e = 1.4426950408889634f;

// ---------------------------------------------------------------- exponentials
// The SFU gives 16 exp2 per clock and SM and is the first unit to fill up: a 128 x 128 block is 1024 clocks of it, while
// the FMA pipe has 256 clocks of work (scale and sum, two at a time).  So a share of the exponentials is computed on the
// FMA pipe with packed fp32 instructions.
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.ftz.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
__device__ __forceinline__ uint64_t pair_of(const uint32_t* v) { return pack2(__uint_as_float(v[0]), __uint_as_float(v[1])); }
__device__ __forceinline__ uint64_t exp2_sfu2(uint64_t x) {
  float x0, x1;
  unpack2(x, x0, x1);
  return pack2(exp2f(x0), exp2f(x1));
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
// Bounds that let a NaN through (fmaxf and fminf return the bound in its place).
__device__ __forceinline__ float max_nan(float a, float b) {
  float r;
  asm("max.ftz.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float min_nan(float a, float b) {
  float r;
  asm("min.ftz.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}
// Two exp2 on the FMA pipe: x = n + f with n an integer and |f| <= 1/2, 2^f by a polynomial of degree 5 (minimax fit of
// 2^f by iterated weighted least squares, constant term 1; relative error at most 1.7e-7 including the fp32 evaluation),
// times 2^n put together from its exponent field.  x is clamped to -127, where that field is 0 and so is the factor, and,
// where x may be large (pass 1, against a stale reference), to 127: a huge finite number, which trips the range test of
// pass 1 as the SFU's inf does.  A NaN passes the clamps and the polynomial and is a NaN behind the product, as the
// SFU's is: a non-finite score shows in the sums whatever column it stands in.
template <bool kAbove>
__device__ __forceinline__ uint64_t exp2_fma2(uint64_t x) {
  float x0, x1;
  unpack2(x, x0, x1);
  x0 = max_nan(x0, -127.f);
  x1 = max_nan(x1, -127.f);
  if (kAbove) { x0 = min_nan(x0, 127.f); x1 = min_nan(x1, 127.f); }
  x = pack2(x0, x1);
  const uint64_t t = add2(x, pack2(12582912.f, 12582912.f));                 // 1.5 * 2^23: the low bits of t are round(x)
  const uint64_t f = fma2(add2(t, pack2(-12582912.f, -12582912.f)), pack2(-1.f, -1.f), x);
  uint64_t q = fma2(pack2(0.001326472731307149f, 0.001326472731307149f), f, pack2(0.009671512991189957f, 0.009671512991189957f));
  q = fma2(q, f, pack2(0.05550733581185341f, 0.05550733581185341f));
  q = fma2(q, f, pack2(0.24022242426872253f, 0.24022242426872253f));
  q = fma2(q, f, pack2(0.6931470036506653f, 0.6931470036506653f));
  q = fma2(q, f, pack2(1.f, 1.f));
  float t0, t1;
  unpack2(t, t0, t1);
  return mul2(q, pack2(__int_as_float((__float_as_int(t0) << 23) + 0x3f800000), __int_as_float((__float_as_int(t1) << 23) + 0x3f800000)));
}
// Pairs of a 32-column chunk's sixteen whose exponentials run on the FMA pipe, spread evenly.
constexpr int kFmaPairs1 = 4, kFmaPairs2 = 4;
__device__ __forceinline__ constexpr bool on_fma(int pair, int share) { return ((pair + 1) * share) / 16 != (pair * share) / 16; }
// Pass 1: adds exp2(score * scale - m) of a chunk's 32 (or 16) columns to two pairs of accumulators (nm2 = {-m, -m}).
template <int kCols>
__device__ __forceinline__ void chunk_rows(uint32_t (&cur)[kCols], uint64_t scale2, uint64_t nm2, uint64_t& s0, uint64_t& s1) {
#pragma unroll
  for (int i = 0; i < kCols / 2; i += 2) {
    const uint64_t x0 = fma2(pair_of(cur + 2 * i), scale2, nm2), x1 = fma2(pair_of(cur + 2 * i + 2), scale2, nm2);
    s0 = add2(s0, on_fma(i, kFmaPairs1) ? exp2_fma2<true>(x0) : exp2_sfu2(x0));
    s1 = add2(s1, on_fma(i + 1, kFmaPairs1) ? exp2_fma2<true>(x1) : exp2_sfu2(x1));
  }
}
// Pass 2: adds exp2(score * scale + nl[column]) of a chunk's 32 (or 16) columns (nl = negated log-sum-exps).
template <int kCols>
__device__ __forceinline__ void chunk_cols(uint32_t (&cur)[kCols], uint64_t scale2, const float* nl, uint64_t& s0, uint64_t& s1) {
#pragma unroll
  for (int i = 0; i < kCols / 2; i += 2) {
    const float4 l4 = *reinterpret_cast<const float4*>(nl + 2 * i);
    const uint64_t x0 = fma2(pair_of(cur + 2 * i), scale2, pack2(l4.x, l4.y));
    const uint64_t x1 = fma2(pair_of(cur + 2 * i + 2), scale2, pack2(l4.z, l4.w));
    s0 = add2(s0, on_fma(i, kFmaPairs2) ? exp2_fma2<false>(x0) : exp2_sfu2(x0));
    s1 = add2(s1, on_fma(i + 1, kFmaPairs2) ? exp2_fma2<false>(x1) : exp2_sfu2(x1));
  }
}
}  // namespace sg
