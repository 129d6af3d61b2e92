// Float-float arithmetic (Dekker 1971; Knuth, TAOCP vol. 2, 4.2.2) on the FP32 pipes: a
// value is the unevaluated sum hi + lo of two floats, |lo| <= ulp(hi) / 2, about 48
// significant bits. Products use the exact FMA residual of hi * hi; sums use TwoSum. Every
// operation uses the explicitly rounded intrinsics, so no multiply-add contraction alters
// them. On GB300 the FP32 pipes issue ~60x the FP64 rate, which makes these 10-15 instruction
// sequences several times faster than FP64 arithmetic.
#pragma once
#include <cuda_runtime.h>

namespace mrd {

struct FF {
  float hi, lo;
};

__device__ __forceinline__ FF ff_from(double x) {
  const float h = __double2float_rn(x);
  return {h, __double2float_rn(x - (double)h)};
}

// The same from the bits of x, without the FP64 pipe (64 cycles per warp instruction and SM quarter, four of
// them above): hi rounds half away from zero, and the rest is the exact remainder of the mantissa.
__device__ __forceinline__ FF ff_from_bits(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x), m = b & 0x7fffffffffffffffull;
  const int f = (int)(m >> 52) - 896;   // x's FP32 exponent field
  if (m == 0) return {0.f, 0.f};
  if (f < 53 || f > 253) return ff_from(x);   // (below 2^-74 lo may be subnormal)
  const unsigned sign = (unsigned)(b >> 32) & 0x80000000u;
  const unsigned hi = (unsigned)(((m + (1ull << 28)) >> 29) - (896ull << 23));
  const int rest = (int)((unsigned)m << 3) >> 3;   // of 2^(exponent - 52): the low 29 bits, signed
  const float lo = __fmul_rn(__fmul_rn(__int2float_rn(rest), 0x1p-52f), __uint_as_float((unsigned)f << 23));
  return {__uint_as_float(hi | sign), __uint_as_float(__float_as_uint(lo) ^ sign)};
}

// accumulator s + c: s collects the rounded partial sums, c their TwoSum errors and the
// low-order parts of the products
struct FFAcc {
  float s, c;
};

// acc += x * y
__device__ __forceinline__ void ff_mac(FFAcc& a, FF x, FF y) {
  const float p = __fmul_rn(x.hi, y.hi);
  float e = __fmaf_rn(x.hi, y.hi, -p);         // x.hi * y.hi = p + e exactly
  e = __fmaf_rn(x.hi, y.lo, e);
  e = __fmaf_rn(x.lo, y.hi, e);
  const float s = __fadd_rn(a.s, p);           // TwoSum(a.s, p)
  const float bp = __fsub_rn(s, a.s);
  const float err = __fadd_rn(__fsub_rn(a.s, __fsub_rn(s, bp)), __fsub_rn(p, bp));
  a.s = s;
  a.c = __fadd_rn(a.c, __fadd_rn(err, e));
}

// acc += x * c for an FP32 coefficient c (exact product of c with both parts of x)
__device__ __forceinline__ void ff_mac1(FFAcc& a, FF x, float c) {
  const float p = __fmul_rn(c, x.hi);
  float e = __fmaf_rn(c, x.hi, -p);
  e = __fmaf_rn(c, x.lo, e);
  const float s = __fadd_rn(a.s, p);
  const float bp = __fsub_rn(s, a.s);
  const float err = __fadd_rn(__fsub_rn(a.s, __fsub_rn(s, bp)), __fsub_rn(p, bp));
  a.s = s;
  a.c = __fadd_rn(a.c, __fadd_rn(err, e));
}

// x * c for an FP32 coefficient c as an accumulator (the exact product: no sum to form yet)
__device__ __forceinline__ FFAcc ff_prod1(FF x, float c) {
  const float p = __fmul_rn(c, x.hi);
  float e = __fmaf_rn(c, x.hi, -p);
  e = __fmaf_rn(c, x.lo, e);
  return {p, e};
}

// a * b of two FP32 numbers, exactly, as a float-float value
__device__ __forceinline__ FF ff_two_prod(float a, float b) {
  const float p = __fmul_rn(a, b);
  return {p, __fmaf_rn(a, b, -p)};
}

__device__ __forceinline__ FF ff_norm(FFAcc a) {  // FastTwoSum(s, c)
  const float h = __fadd_rn(a.s, a.c);
  return {h, __fsub_rn(a.c, __fsub_rn(h, a.s))};
}

__device__ __forceinline__ FF ff_neg(FF a) { return {-a.hi, -a.lo}; }

// a + b (TwoSum of the high parts, low parts added to the error)
__device__ __forceinline__ FF ff_add(FF a, FF b) {
  const float s = __fadd_rn(a.hi, b.hi);
  const float bp = __fsub_rn(s, a.hi);
  float e = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, bp)), __fsub_rn(b.hi, bp));
  e = __fadd_rn(e, __fadd_rn(a.lo, b.lo));
  const float h = __fadd_rn(s, e);
  return {h, __fsub_rn(e, __fsub_rn(h, s))};
}

__device__ __forceinline__ FF ff_warp_sum(FF v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const FF w = {__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)};
    v = ff_add(v, w);
  }
  return v;
}

// ---------------------------------------------------------------- complex values

// complex float-float value (re, im), staged as float4 {re.hi, im.hi, re.lo, im.lo}
__device__ __forceinline__ float4 cff_from(double2 v) {
  const FF r = ff_from(v.x), i = ff_from(v.y);
  return make_float4(r.hi, i.hi, r.lo, i.lo);
}

// Complex products by three real ones (Gauss): rr = sum a_r b_r, ii = sum a_i b_i,
// ss = sum (a_r + a_i)(b_r + b_i); then Re = rr - ii, Im = ss - rr - ii. The operand sums are
// formed once per staged element, so a complex multiply-add costs 3 float-float products (36
// FP32 instructions) instead of 4 (48). Every product still carries ~2^-48 |a||b| absolute
// error, as in the four-product form, so the result's error against the output's scale is
// unchanged in order.
struct CAcc {
  FFAcc rr, ii, ss;
};

// (Re, Im) of an accumulated product as float-float values
__device__ __forceinline__ void cff_result(const CAcc& a, FF& re, FF& im) {
  const FF rr = ff_norm(a.rr), ii = ff_norm(a.ii), ss = ff_norm(a.ss);
  re = ff_add(rr, ff_neg(ii));
  im = ff_add(ss, ff_neg(ff_add(rr, ii)));
}

// a_r + a_i of a staged element (float-float), for the third product
__device__ __forceinline__ float2 cff_sum(float4 a) {
  const FF s = ff_add(FF{a.x, a.z}, FF{a.y, a.w});
  return make_float2(s.hi, s.lo);
}

// c += a * b (complex), sa = a_r + a_i, sb = b_r + b_i
__device__ __forceinline__ void cff_mac(CAcc& c, float4 a, float2 sa, float4 b, float2 sb) {
  ff_mac(c.rr, FF{a.x, a.z}, FF{b.x, b.z});
  ff_mac(c.ii, FF{a.y, a.w}, FF{b.y, b.w});
  ff_mac(c.ss, FF{sa.x, sa.y}, FF{sb.x, sb.y});
}

__device__ __forceinline__ FFAcc ff_renorm(FFAcc a) {
  const FF r = ff_norm(a);
  return {r.hi, r.lo};
}

}  // namespace mrd
