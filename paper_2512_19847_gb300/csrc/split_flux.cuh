// FP64 WENO fluxes with their nonlinear part on the FP32 pipe.
//
// This GPU issues FP64 instructions at 1/64 of the FP32 rate, and a WENO5 flux
// in FP64 takes about 55 of them per interface.  Here the flux is taken apart
// into a part that is linear in the data, which stays in FP64, and the weights'
// correction, which is a sum of products (nonlinear weight) x (third difference)
// and is evaluated in pairs of floats (h + l, 48 bits and more).  The differences
// it starts from are taken in FP64, so that the pair's relative rounding (2^-48)
// applies to increments between neighbouring cells and not to the values.
//
// With g+- = g +- U (twice the Lax-Friedrichs split), interface i + 1/2, increments
// D_k = f_{k+1} - f_k, second differences c_k = D_k - D_{k-1} and third differences
// T_k = c_{k+1} - c_k, the two reconstructions are (WENO5, about the centred candidate)
//   6 L(g+) = 3 (g+_i + g+_{i+1}) - [c_i + 2 w0 T_{i-1} + w2 T_i](g+),
//   6 R(g-) = 3 (g-_i + g-_{i+1}) - [c_{i+1} - 2 w0 T_{i+1} - w2 T_i](g-),
// so that the flux difference of cell i is 1/(12 h) times
//   6 (g_{i+1} - g_{i-1}) + N_{i+1/2} - N_{i-1/2},
// N the two brackets, negated: the only term that is linear in the values and not in their
// increments is a central difference of g, one FP64 operation.  The smoothness indicators (times 4,
// plus 4 eps_W) are sums of squares of increments: (13/3) c_k^2 + l^2 + 4 eps_W with
// l = 3 D_k - D_{k-1}, D_{k-1} + D_k or D_k - 3 D_{k-1} for the three candidates.
// WENO3: the brackets are 3 w0 c_i (g+) and 3 w0 c_{i+1} (g-), taken as (1 + 3 (w0 - 1/3)) c.
//
// Where this holds.  The pairs' rounding is relative to the increments, and the weights amplify it: on data
// that is rough at the mesh scale a bracket is off by up to 2^-42 of its increments (2000 random
// stencils), where the whole FP64 form is off by 2^-53 of the values.  So an interface takes its pairs
// only while the third differences it uses (WENO3: the second) are below a limit, a fixed part of
// the largest value in the field (SplitLimits); its bracket is a NaN otherwise, and the cells beside it take
// their flux difference from the whole FP64 form.  The limit is zero or negative, and every
// interface rough, where the squares or products could leave the float range.
#pragma once
#include "pairs.cuh"

namespace apd {

// Part of the field's largest value up to which an interface's third differences (WENO5) or second
// differences (WENO3) may reach.  Errors of flux differences, split against whole (rms over a field, and
// largest), measured with 113-bit arithmetic for smooth fields, jumps, and noise of 0.001 to 0.5 on a
// smooth field: WENO5 with 1/32 at most 1.00 and 1.20 times the whole form's (without a limit 70 and 147
// times on noise, the largest 32 times at a jump), with 1/8 1.44 and 2.9.  WENO3 with 3/128 at most 1.25 and
// 1.23 (random field of wavenumbers up to 16, 256 cells a side; 1.05 at 300, 0.76 at 360), with 1/16 1.28 and
// 1.72; with 1/64 1.17 and 1.23, but then the shoulders of the 256^2 layer, where the split errs least, are rough:
// ten steps 2324 us instead of 1619.  A 1024^2 step takes 1.32 ms (WENO5; WENO3 1.26) with no interface rough and
// 3.83 (3.07) with all.
#ifndef APD_SPLIT_ROUGH5
#define APD_SPLIT_ROUGH5 (1.f / 32.f)
#endif
#ifndef APD_SPLIT_ROUGH3
#define APD_SPLIT_ROUGH3 (3.f / 128.f)
#endif

// Limits on an interface's differences for the pair (q; v) of E and for the pairs (v; u) of D_LF . B, from
// the largest |u|, |v|, |q| of the state a step starts from, given as high words of doubles (field_max),
// and w, the eps_W the indicators hold.  The scale of E holds u as well as q and v, as E adds (tau/4) D_0 . u
// to tau eps^2 times the flux difference (cu = their ratio 1/(4 eps^2), at most 1).  Zero (only zero
// differences pass) for values below 2^-80, whose pairs would lose their low parts; negative for values from
// 2^50 on, infinities and NaN, and where eps_W is out of proportion.
struct SplitLimits { float e, b; };
__device__ __forceinline__ float field_scale(unsigned hi) {
  if (hi < (943u << 20)) return 0.f;
  if (hi >= (1073u << 20)) return __uint_as_float(0x7f800000u);
  return __uint_as_float((hi - (896u << 20)) << 3);
}
__device__ __forceinline__ SplitLimits split_limits(unsigned mu, unsigned mv, unsigned mq, float cu, float w, float rough) {
  const float su = field_scale(mu), sv = field_scale(mv), sq = field_scale(mq);
  const float s = fmaxf(fmaxf(su, sv), sq);
  SplitLimits r;
  r.b = rough * fmaxf(su, sv);
  r.e = rough * fmaxf(fmaxf(sv, sq), su * cu);
  if (!(s < 1.1259e15f && w >= s * s * 7.8886e-31f && w <= 1.2677e30f)) r.e = r.b = -1.f;   // 2^50, 2^-100, 2^100
  return r;
}
__device__ __forceinline__ float rough_mark() { return __uint_as_float(0x7fffffffu); }
__device__ __forceinline__ bool is_rough(float h) { return !(fabsf(h) <= 3.4028235e38f); }

// The bracket of one WENO5 reconstruction for each of KR neighbouring interfaces:
// q[m] = c + 2 w0 T_{out} + w2 T_{in} from the increments D[m .. m + 3] of its stencil (upwind
// to downwind; T_out = D[m+2] - 2 D[m+1] + D[m], T_in one further), w = 16 eps_W (the
// indicators times 4, the doubled split).  With the e_k scaled by a power of two so that the
// largest is about 1, and their products likewise where even the largest is small, every step stays in
// the float range for the values and eps_W that SplitLimits admits: what underflows is below 2^-60 of the
// sum it belongs to.  rough[m]: a third difference exceeds lim.
template <int KR>
__device__ __forceinline__ void w5_split(const F2* D, F2 w, float lim, F2* q, bool* rough) {
  F2 c[KR + 3], C[KR + 3];
#pragma unroll
  for (int k = 1; k < KR + 3; ++k) {
    c[k] = f2_sub(D[k], D[k - 1]);
    const F2 s = f2_sqr(c[k]);
    const float kh = 4.3333335f, kl = -1.5894572e-07f;   // 13/3
    const float p = __fmul_rn(kh, s.h);
    const float pl = __fmaf_rn(kl, s.h, __fmaf_rn(kh, s.l, __fmaf_rn(kh, s.h, -p)));
    C[k] = f2_add(w, f2(p, pl));
  }
  F2 to = f2_sub(c[2], c[1]);
#pragma unroll
  for (int m = 0; m < KR; ++m) {
    F2 e0 = f2_add(C[m + 1], f2_sqr(f2_addk<2>(c[m + 1], D[m + 1])));
    F2 e1 = f2_add(C[m + 2], f2_sqr(f2_add(D[m + 1], D[m + 2])));
    F2 e2 = f2_add(C[m + 3], f2_sqr(f2_addk<-2>(c[m + 3], D[m + 2])));
    const float se = inv_pow2(fmaxf(fmaxf(e0.h, e1.h), e2.h));
    e0 = f2(e0.h * se, e0.l * se);
    e1 = f2(e1.h * se, e1.l * se);
    e2 = f2(e2.h * se, e2.l * se);
    F2 pa = f2_mul(e1, e2), pb = f2_mul(e0, e2), pc = f2_mul(e0, e1);
    const float pm = fmaxf(fmaxf(pa.h, pb.h), pc.h);
    if (pm < 9.09e-13f) {   // 2^-40
      const float sp = inv_pow2(pm);
      pa = f2(pa.h * sp, pa.l * sp);
      pb = f2(pb.h * sp, pb.l * sp);
      pc = f2(pc.h * sp, pc.l * sp);
    }
    const F2 A = f2_sqr(pa), B = f2_scale(f2_sqr(pb), 6.f), E = f2_scale(f2_sqr(pc), 3.f);
    const F2 den = f2_add(f2_add(A, E), B);
    const F2 ti = f2_sub(c[m + 3], c[m + 2]);
    q[m] = f2_add(c[m + 2], f2_div(f2_addk<2>(f2_mul(E, ti), f2_mul(A, to)), den));
    rough[m] = fmaxf(fabsf(to.h), fabsf(ti.h)) > lim;
    to = ti;
  }
}

// The same for WENO3: q[m] = c + 3 (w0 - 1/3) c with c = D[m+1] - D[m] (upwind, then downwind increment),
// w = 4 eps_W, indicators e_k = D_k^2 + w: w0 = e1^2 / (e1^2 + 2 e0^2) and
// 3 (w0 - 1/3) = 2 (e1 - e0)(e1 + e0) / (e1^2 + 2 e0^2), e1 - e0 = c (D[m] + D[m+1]); rough[m]: |c| exceeds lim.
template <int KR>
__device__ __forceinline__ void w3_split(const F2* D, F2 w, float lim, F2* q, bool* rough) {
  F2 e[KR + 1];
#pragma unroll
  for (int k = 0; k < KR + 1; ++k) e[k] = f2_add(w, f2_sqr(D[k]));
#pragma unroll
  for (int m = 0; m < KR; ++m) {
    const float se = inv_pow2(fmaxf(e[m].h, e[m + 1].h));
    const F2 e0 = f2(e[m].h * se, e[m].l * se), e1 = f2(e[m + 1].h * se, e[m + 1].l * se);
    const F2 c = f2_sub(D[m + 1], D[m]), d = f2_add(D[m + 1], D[m]);
    const F2 n = f2_mul(f2_mul(f2_mul(c, f2(d.h * se, d.l * se)), f2_add(e0, e1)), c);
    const F2 r = f2_div(n, f2_addk<2>(f2_sqr(e1), f2_sqr(e0)));
    q[m] = f2_addk<2>(c, r);
    rough[m] = fabsf(c.h) > lim;
  }
}

}  // namespace apd
