// Pairs of floats: h + l with 48 bits and more, on the FP32 pipe.  This GPU issues FP64 instructions
// at 1/64 of the FP32 rate, a pair's sum takes 8 FP32 instructions and its product 4.
#pragma once
#include <cuda_runtime.h>

namespace apd {

// h + l, |l| small against the operands it came from (not always against h).
struct F2 { float h, l; };

__device__ __forceinline__ F2 f2(float h, float l) { F2 r; r.h = h; r.l = l; return r; }

// a + k b for k = 1, -1, 2, -2: the error of the leading sum kept exactly (Knuth's two-sum).
template <int K>
__device__ __forceinline__ F2 f2_addk(F2 a, F2 b) {
  const float k = float(K);
  const float s = __fmaf_rn(k, b.h, a.h), bb = __fsub_rn(s, a.h);
  const float e = __fadd_rn(__fsub_rn(a.h, __fsub_rn(s, bb)), __fmaf_rn(k, b.h, -bb));
  return f2(s, __fadd_rn(e, __fmaf_rn(k, b.l, a.l)));
}
__device__ __forceinline__ F2 f2_add(F2 a, F2 b) { return f2_addk<1>(a, b); }
__device__ __forceinline__ F2 f2_sub(F2 a, F2 b) { return f2_addk<-1>(a, b); }
// a + k b for k = 1 or -1 given at run time.
__device__ __forceinline__ F2 f2_addr(F2 a, F2 b, float k) {
  const float s = __fmaf_rn(k, b.h, a.h), bb = __fsub_rn(s, a.h);
  const float e = __fadd_rn(__fsub_rn(a.h, __fsub_rn(s, bb)), __fmaf_rn(k, b.h, -bb));
  return f2(s, __fadd_rn(e, __fmaf_rn(k, b.l, a.l)));
}
// The same value with |l| <= ulp(h)/2.
__device__ __forceinline__ F2 f2_norm(F2 a) {
  const float h = __fadd_rn(a.h, a.l);
  return f2(h, __fsub_rn(a.l, __fsub_rn(h, a.h)));
}
__device__ __forceinline__ F2 f2_mul(F2 a, F2 b) {
  const float p = __fmul_rn(a.h, b.h);
  return f2(p, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.l, __fmaf_rn(a.h, b.h, -p))));
}
__device__ __forceinline__ F2 f2_sqr(F2 a) {
  const float p = __fmul_rn(a.h, a.h);
  return f2(p, __fmaf_rn(a.h, a.l, __fmaf_rn(a.h, a.l, __fmaf_rn(a.h, a.h, -p))));
}
// k a for an integer k that is a float.
__device__ __forceinline__ F2 f2_scale(F2 a, float k) {
  const float p = __fmul_rn(k, a.h);
  return f2(p, __fmaf_rn(k, a.l, __fmaf_rn(k, a.h, -p)));
}
// n / d: one approximate quotient and the remainder's, with the same reciprocal.
__device__ __forceinline__ F2 f2_div(F2 n, F2 d) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d.h));
  const float q = __fmul_rn(n.h, r);
  const float rem = __fadd_rn(__fmaf_rn(-q, d.h, n.h), __fmaf_rn(-q, d.l, n.l));
  return f2(q, __fmul_rn(rem, r));
}
// 2^-(exponent of x) for 0 < x finite (0, infinity and NaN give something harmless or not finite).
__device__ __forceinline__ float inv_pow2(float x) {
  return __uint_as_float(0x7f000000u - (__float_as_uint(x) & 0x7f800000u));
}

// An FP64 increment as a pair, by integer operations (a conversion instruction takes a
// slot of the FP64 pipe): h the leading 24 bits truncated, l the other 29 rounded to 24.
__device__ __forceinline__ F2 f2_from_double(double d) {
  const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
  const unsigned ea = (hi >> 20) & 0x7ffu;
  if (ea - 949u <= 1150u - 949u) {   // 2^-74 <= |d| < 2^128
    const unsigned s = hi & 0x80000000u;
    const float h = __uint_as_float((__funnelshift_l(lo, hi, 3) - (384u << 23)) | s);   // 896 mod 512
    const float m = __uint2float_rn(lo & 0x1fffffffu);
    return f2(h, __fmul_rn(m, __uint_as_float(((ea - 948u) << 23) | s)));
  }
  if ((hi << 1 | lo) == 0u) return f2(0.f, 0.f);
  const float h = __double2float_rn(d);
  return f2(h, __double2float_rn(d - (double)h));
}

// FP32 to FP64 on the integer pipe, exact: a normal value's exponent rebiased, its fraction extended
// (subnormal values, infinities and NaN by the instruction).
__device__ __forceinline__ double widen_f32(float x) {
  const unsigned u = __float_as_uint(x);
  if (((u >> 23) & 0xffu) - 1u < 254u)
    return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + (896u << 20))), (int)(u << 29));
  if ((u << 1) == 0u) return __hiloint2double((int)u, 0);
  return (double)x;
}
// h + l in FP64 (one FP64 operation).
__device__ __forceinline__ double f2_to_double(F2 a) { return widen_f32(a.h) + widen_f32(a.l); }

// a float times a pair of constants, and two floats' sum and difference, exact up to the pair's rounding.
__device__ __forceinline__ F2 f2_mulf(F2 c, float x) {
  const float p = __fmul_rn(c.h, x);
  return f2(p, __fmaf_rn(c.l, x, __fmaf_rn(c.h, x, -p)));
}
__device__ __forceinline__ F2 f2_sum(float a, float b) {
  const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
  return f2(s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb)));
}

}  // namespace apd
