// Periodic Helmholtz solve of Algorithm 1, step 2:
//     (D_Delta - kappa_i) theta^(i) = R_i
// by diagonalisation in the discrete Fourier basis (the operator is periodic
// with constant coefficients, so every DFT mode is an eigenvector with
// eigenvalue lam_x(kx) + lam_y(ky) - kappa_i).  Three passes:
//   k_fft_rows_fwd : real row DFTs of R (two rows packed as one complex row),
//                    written as the half spectrum S[y][0..nx/2];
//   k_fft_cols     : per spectral column, DFT along y, division by the
//                    symbol (mode k = 0 set to mean(theta^n): every other term of R has zero mean),
//                    inverse DFT along y, scaled by 1/(nx ny);
//   k_fft_rows_inv : inverse real row DFTs into theta^(i).
// Power-of-two lengths: radix-2^3 passes in shared memory, from bit-reversed to natural
// order (fft_dit) or from natural to bit-reversed (fft_rev), so no permutation pass
// is needed.  Other lengths that factor into 2, 3, 5 and 7: a self-sorting
// mixed-radix transform (below).  Any other length n is transformed by
// Bluestein's chirp-z identity (L. I. Bluestein, 1970): with
// w_m = exp(i pi m^2 / n) and
// jk = (j^2 + k^2 - (k - j)^2) / 2,
//     sum_j x_j exp(-2 pi i jk / n) = conj(w_k) sum_j (x_j conj(w_j)) w_{k-j},
// a circular convolution of length M, the power of two >= 2n - 1, taken with
// two radix-2 transforms of length M and the precomputed DFT of the filter
// (w_m for |m| < n); the inverse transform conjugates chirp and filter.  A
// row or spectral column then occupies M complex values in shared memory.
// Each pass has a power-of-two kernel and a kernel for the other lengths
// (suffix _bs: mixed radix or Bluestein); each takes the work items of its
// kind and skips the others, and a step launches only the kinds its batch
// holds.  When ny is odd, the last row pair
// holds one row (its partner is zero).
#pragma once
#include "common.cuh"

namespace apd {

template <typename T> struct Cplx;
template <> struct Cplx<double> { using type = double2; };
template <> struct Cplx<float> { using type = float2; };

// Twiddles in the transform's own type (no conversion per butterfly).
template <typename T> __device__ __forceinline__ const typename Cplx<T>::type* twiddles(const BatchDev& b);
template <> __device__ __forceinline__ const double2* twiddles<double>(const BatchDev& b) { return b.tw; }
template <> __device__ __forceinline__ const float2* twiddles<float>(const BatchDev& b) { return b.tw32; }

__device__ __forceinline__ int brev(int k, int ln) { return (int)(__brev((unsigned)k) >> (32 - ln)); }

// Complex helpers.  mul_j(z, inv) multiplies by -i (forward) or +i (inverse):
// the twiddle W_{4h}^h of the second stage of a radix-2^2 step.
template <typename C>
__device__ __forceinline__ C cadd(C a, C b) { C r; r.x = a.x + b.x; r.y = a.y + b.y; return r; }
template <typename C>
__device__ __forceinline__ C csub(C a, C b) { C r; r.x = a.x - b.x; r.y = a.y - b.y; return r; }
template <typename C>
__device__ __forceinline__ C cmul_tw(C w, C b, bool inv) {   // w (conjugated when inv) times b
  C r;
  if (inv) { r.x = w.x * b.x + w.y * b.y; r.y = w.x * b.y - w.y * b.x; }
  else { r.x = w.x * b.x - w.y * b.y; r.y = w.x * b.y + w.y * b.x; }
  return r;
}
template <typename C>
__device__ __forceinline__ C mul_j(C a, bool inv) {
  C r;
  if (inv) { r.x = -a.y; r.y = a.x; } else { r.x = a.y; r.y = -a.x; }
  return r;
}

// Butterfly with the twiddle on the second input: (a, b) -> (a + w b, a - w b) in six FMAs, the
// difference as 2 a - (a + w b).  Multiplying first and adding after takes eight operations.
template <typename C>
__device__ __forceinline__ void bfly(C& a, C& b, C w) {
  using T = decltype(a.x);
  const T sx = fma(-w.y, b.y, fma(w.x, b.x, a.x)), sy = fma(w.y, b.x, fma(w.x, b.y, a.y));
  b.x = fma(T(2), a.x, -sx);
  b.y = fma(T(2), a.y, -sy);
  a.x = sx;
  a.y = sy;
}
template <typename C>
__device__ __forceinline__ void bfly1(C& a, C& b) {   // w = 1
  const C s = cadd(a, b), d = csub(a, b);
  a = s;
  b = d;
}
template <typename C>
__device__ __forceinline__ void bflyj(C& a, C& b, bool inv) {   // w = W_4
  b = mul_j(b, inv);
  bfly1(a, b);
}
// Twiddle of a table, conjugated for the inverse transform, and times W_4 (likewise).
template <typename C>
__device__ __forceinline__ C tw_of(C w, bool inv) { if (inv) w.y = -w.y; return w; }
template <typename C>
__device__ __forceinline__ C tw_j(C w, bool inv) { return mul_j(w, inv); }
template <typename C>
__device__ __forceinline__ C tw_8(bool inv) {
  using T = decltype(C().x);
  C w;
  w.x = T(0.70710678118654752440);
  w.y = inv ? T(0.70710678118654752440) : T(-0.70710678118654752440);
  return w;
}

// Shared-memory index with padding: one spare element after every 2^PS
// elements (PS = 31: none), so that the strided accesses of the butterfly
// passes spread over the 32 banks: with 8-byte (FP32) complex values PS = 4,
// with 16-byte (FP64) values PS = 3, every radix-2^3 pass below reads and
// writes with the minimum number of shared-memory wavefronts.
template <int PS>
__device__ __forceinline__ int pidx(int i) { return PS >= 31 ? i : i + (i >> PS); }
template <typename T>
__host__ __device__ constexpr int pad_shift() { return sizeof(T) == 4 ? 4 : 3; }
// Complex elements a padded region of n values occupies.
__host__ __device__ constexpr int padded_len(int n, int ps) { return ps >= 31 ? n : n + (n >> ps) + 1; }

// ntr transforms of length n = 2^ln held back to back in x[] (element i at
// x[pidx<PS>(i)]), input in bit-reversed order, output natural.  Twiddle
// W_m^p = tw[p * nmax/m].  Stages are taken three at a time (radix-2^3): each
// thread loads eight elements p0 + k h (k = 0..7, h = 2^(s-1)), applies stage s
// (half h, twiddle W_{2h}^pos), stage s+1 (half 2h, W_{4h}^pos times 1 and W_4)
// and stage s+2 (half 4h, W_{8h}^pos times 1, W_8, W_4, W_4 W_8) in registers, and stores
// them: every butterfly takes its whole twiddle (bfly), read from the table or that times W_4,
// which exchanges its parts.  One or two stages left over take a radix-2^2 or radix-2 step; the
// first step has only constant twiddles.
// FP64 transforms are bound by the FP64 pipe: 72 operations per eight elements and step against
// 104 with twiddles and constant roots multiplied separately.  2048^2, FP64, ms per step: columns
// 0.944 -> 0.652, rows 0.417 -> 0.312 (forward) and 0.406 -> 0.290 (inverse); FP32, which is not: 0.098
// -> 0.095, 0.050 -> 0.052 and 0.049 -> 0.047.
//
// The eight elements of one step in registers: dit8 three stages from stage s (half h), dit8_first the same
// at s = 1.
template <typename C>
__device__ __forceinline__ void dit8(C (&v)[8], const C* __restrict__ tw, int lnmax, int s, int pos, int h, bool inv) {
  const C w1 = tw_of(tw[pos << (lnmax - s)], inv), w2 = tw_of(tw[pos << (lnmax - s - 1)], inv);
  const C w3 = tw_of(tw[pos << (lnmax - s - 2)], inv), w4 = tw_of(tw[(pos + h) << (lnmax - s - 2)], inv);
  bfly(v[0], v[1], w1); bfly(v[2], v[3], w1); bfly(v[4], v[5], w1); bfly(v[6], v[7], w1);
  const C w2j = tw_j(w2, inv);
  bfly(v[0], v[2], w2); bfly(v[1], v[3], w2j); bfly(v[4], v[6], w2); bfly(v[5], v[7], w2j);
  bfly(v[0], v[4], w3); bfly(v[1], v[5], w4); bfly(v[2], v[6], tw_j(w3, inv)); bfly(v[3], v[7], tw_j(w4, inv));
}
template <typename C>
__device__ __forceinline__ void dit8_first(C (&v)[8], bool inv) {
  bfly1(v[0], v[1]); bfly1(v[2], v[3]); bfly1(v[4], v[5]); bfly1(v[6], v[7]);
  bfly1(v[0], v[2]); bflyj(v[1], v[3], inv); bfly1(v[4], v[6]); bflyj(v[5], v[7], inv);
  const C w8 = tw_8<C>(inv);
  bfly1(v[0], v[4]); bfly(v[1], v[5], w8); bflyj(v[2], v[6], inv); bfly(v[3], v[7], tw_j(w8, inv));
}
template <int PS, typename C>
__device__ __forceinline__ void load8(C (&v)[8], const C* x, int q, int h) {
#pragma unroll
  for (int m = 0; m < 8; ++m) v[m] = x[pidx<PS>(q + m * h)];
}
template <int PS, typename C>
__device__ __forceinline__ void store8(const C (&v)[8], C* x, int q, int h) {
#pragma unroll
  for (int m = 0; m < 8; ++m) x[pidx<PS>(q + m * h)] = v[m];
}

template <typename T, int PS = 31>
__device__ __forceinline__ void fft_dit(typename Cplx<T>::type* x, int ln, int ntr,
                                        const typename Cplx<T>::type* __restrict__ tw, int lnmax,
                                        bool inv, int tid, int nthr) {
  using C = typename Cplx<T>::type;
  const int n = 1 << ln;
  int s = 1;
  for (; s + 2 <= ln; s += 3) {
    const int h = 1 << (s - 1), ne = n >> 3, nb = ntr * ne;
    for (int k = tid; k < nb; k += nthr) {
      const int t = k >> (ln - 3), bi = k & (ne - 1);
      const int pos = bi & (h - 1), grp = bi >> (s - 1);
      const int q = t * n + grp * 8 * h + pos;
      C v[8];
      load8<PS>(v, x, q, h);
      if (s == 1) dit8_first(v, inv);
      else dit8(v, tw, lnmax, s, pos, h, inv);
      store8<PS>(v, x, q, h);
    }
    __syncthreads();
  }
  if (s + 1 == ln) {   // two stages left: radix-2^2
    const int h = 1 << (s - 1), nq = n >> 2, nb = ntr * nq;
    for (int k = tid; k < nb; k += nthr) {
      const int t = k >> (ln - 2), pos = k & (nq - 1);   // one group: h = n / 4
      const int p0 = t * n + pos;
      C x0 = x[pidx<PS>(p0)], x1 = x[pidx<PS>(p0 + h)], x2 = x[pidx<PS>(p0 + 2 * h)], x3 = x[pidx<PS>(p0 + 3 * h)];
      const C w1 = tw_of(tw[pos << (lnmax - s)], inv), w2 = tw_of(tw[pos << (lnmax - s - 1)], inv);
      bfly(x0, x1, w1); bfly(x2, x3, w1);
      bfly(x0, x2, w2); bfly(x1, x3, tw_j(w2, inv));
      x[pidx<PS>(p0)] = x0; x[pidx<PS>(p0 + h)] = x1; x[pidx<PS>(p0 + 2 * h)] = x2; x[pidx<PS>(p0 + 3 * h)] = x3;
    }
    __syncthreads();
  } else if (s == ln) {   // one stage left: radix-2
    const int half = 1 << (s - 1), sh = lnmax - s, nb = ntr * (n >> 1);
    for (int k = tid; k < nb; k += nthr) {
      const int t = k >> (ln - 1), pos = k & ((n >> 1) - 1);
      const int i0 = t * n + pos, i1 = i0 + half;
      C a = x[pidx<PS>(i0)], c = x[pidx<PS>(i1)];
      bfly(a, c, tw_of(tw[pos << sh], inv));
      x[pidx<PS>(i0)] = a;
      x[pidx<PS>(i1)] = c;
    }
    __syncthreads();
  }
}

// Natural-order input, bit-reversed output, with the same butterflies: splitting the polynomial
// sum_i x_i z^i modulo z^n - 1 into its remainders modulo z^t - c and z^t + c, level by level, block j
// of a level of m blocks takes c = W_{2m}^{rev(j)} (rev: j's log2 m bits reversed) for all its pairs.
// rev(j) / (2m) is half the fraction with j's bits after the point in reverse, for every m, so
// one table in that order, tr[j] = exp(-pi i 0.b0 b1 b2 ...), serves all levels: block j of three
// successive levels takes tr[j], tr[2j] (times 1 and W_4) and tr[4j], tr[4j + 2] = W_8 tr[4j].
// tr follows the nmax / 2 values of tw.
//
// rev8 takes three levels of block j in registers, rev8_first those of the only block of the first levels.
template <typename C>
__device__ __forceinline__ void rev8(C (&v)[8], const C* __restrict__ tr, int j, bool inv) {
  const C w1 = tw_of(tr[j], inv), w2 = tw_of(tr[2 * j], inv), w3 = tw_of(tr[4 * j], inv), w4 = tw_of(tr[4 * j + 2], inv);
  bfly(v[0], v[4], w1); bfly(v[1], v[5], w1); bfly(v[2], v[6], w1); bfly(v[3], v[7], w1);
  const C w2j = tw_j(w2, inv);
  bfly(v[0], v[2], w2); bfly(v[1], v[3], w2); bfly(v[4], v[6], w2j); bfly(v[5], v[7], w2j);
  bfly(v[0], v[1], w3); bfly(v[2], v[3], tw_j(w3, inv)); bfly(v[4], v[5], w4); bfly(v[6], v[7], tw_j(w4, inv));
}
template <typename C>
__device__ __forceinline__ void rev8_first(C (&v)[8], bool inv) {
  bfly1(v[0], v[4]); bfly1(v[1], v[5]); bfly1(v[2], v[6]); bfly1(v[3], v[7]);
  bfly1(v[0], v[2]); bfly1(v[1], v[3]); bflyj(v[4], v[6], inv); bflyj(v[5], v[7], inv);
  const C w8 = tw_8<C>(inv);
  bfly1(v[0], v[1]); bflyj(v[2], v[3], inv); bfly(v[4], v[5], w8); bfly(v[6], v[7], tw_j(w8, inv));
}

// The first step takes element i of transform t from load(t, i), so that a kernel's input passes
// from global memory to the butterflies without a pass of its own through shared memory; n >= 8.
// Row passes at 2048^2, FP32, bound by these passes: 0.050 -> 0.038 (forward) and 0.046 -> 0.037 ms
// (inverse) per step; FP64 forward 0.308 -> 0.291.
template <typename T, int PS = 31, typename Load>
__device__ __forceinline__ void fft_rev_from(typename Cplx<T>::type* x, int ln, int ntr,
                                             const typename Cplx<T>::type* __restrict__ tw, int lnmax,
                                             bool inv, int tid, int nthr, Load load) {
  using C = typename Cplx<T>::type;
  const C* __restrict__ tr = tw + (1 << (lnmax - 1));
  const int n = 1 << ln, ne = n >> 3, nb = ntr * ne;
  for (int k = tid; k < nb; k += nthr) {
    const int t = k >> (ln - 3), pos = k & (ne - 1);
    C v[8];
#pragma unroll
    for (int m = 0; m < 8; ++m) v[m] = load(t, pos + m * ne);
    rev8_first(v, inv);
    store8<PS>(v, x, t * n + pos, ne);
  }
  __syncthreads();
  int s = ln - 3;   // levels of size 2^s and below are left
  for (; s >= 3; s -= 3) {
    const int h = 1 << (s - 3);
    for (int k = tid; k < nb; k += nthr) {
      const int t = k >> (ln - 3), bi = k & (ne - 1);
      const int pos = bi & (h - 1), j = bi >> (s - 3);
      const int q = t * n + j * 8 * h + pos;
      C v[8];
      load8<PS>(v, x, q, h);
      rev8(v, tr, j, inv);
      store8<PS>(v, x, q, h);
    }
    __syncthreads();
  }
  if (s == 2) {   // two levels left: radix-2^2
    const int nq = n >> 2, nb = ntr * nq;
    for (int k = tid; k < nb; k += nthr) {
      const int j = k & (nq - 1), p0 = 4 * k;
      C x0 = x[pidx<PS>(p0)], x1 = x[pidx<PS>(p0 + 1)], x2 = x[pidx<PS>(p0 + 2)], x3 = x[pidx<PS>(p0 + 3)];
      const C w1 = tw_of(tr[j], inv), w2 = tw_of(tr[2 * j], inv);
      bfly(x0, x2, w1); bfly(x1, x3, w1);
      bfly(x0, x1, w2); bfly(x2, x3, tw_j(w2, inv));
      x[pidx<PS>(p0)] = x0; x[pidx<PS>(p0 + 1)] = x1; x[pidx<PS>(p0 + 2)] = x2; x[pidx<PS>(p0 + 3)] = x3;
    }
    __syncthreads();
  } else if (s == 1) {   // one level left
    const int nb = ntr * (n >> 1);
    for (int k = tid; k < nb; k += nthr) {
      const int i0 = 2 * k, i1 = i0 + 1;
      C a = x[pidx<PS>(i0)], c = x[pidx<PS>(i1)];
      bfly(a, c, tw_of(tr[k & ((n >> 1) - 1)], inv));
      x[pidx<PS>(i0)] = a;
      x[pidx<PS>(i1)] = c;
    }
    __syncthreads();
  }
}

template <typename T, int PS = 31>
__device__ __forceinline__ void fft_rev(typename Cplx<T>::type* x, int ln, int ntr,
                                        const typename Cplx<T>::type* __restrict__ tw, int lnmax,
                                        bool inv, int tid, int nthr) {
  const int n = 1 << ln;
  fft_rev_from<T, PS>(x, ln, ntr, tw, lnmax, inv, tid, nthr, [=](int t, int i) { return x[pidx<PS>(t * n + i)]; });
}

// Forward transform, an operation on the spectrum and inverse transform of ntr <= 2^lg sequences of length
// n = 2^ln >= 8, from load(t, i) to store(t, i, v); op(t, ky, v) changes value ky of the spectrum.  The levels
// are taken so that those which do not fill a step of three come first forwards and last
// backwards: the last forward and the first backward step then hold the same eight elements,
// and with op between them they stay in registers.  The first step reads load() and the last one
// writes store(); in these two adjacent threads take the same element of adjacent sequences.  Length 2048 passes
// through shared memory 6 times instead of 9 (in, 4, op, 4, out before, the first and the last a half).
// Column pass, ms per step: FP32 2048^2 (bound by these passes) 0.094 -> 0.070, FP64 2048^2 (bound by the
// FP64 pipe) 0.650 -> 0.637.  In FP64 op is a pass of its own (spread) where a step does not fill the
// block: a warp instruction costs the FP64 pipe the same with few lanes as with all, and eight
// reciprocals one after the other in few warps cost more than the exchange (64^2 and 256^2, ten
// steps: 378 and 422 us together, 335 and 406 apart).
template <typename T, int PS, typename Load, typename Op, typename Store>
__device__ __forceinline__ void fft_there_and_back(typename Cplx<T>::type* x, int ln, int lg, int ntr,
                                                   const typename Cplx<T>::type* __restrict__ tw, int lnmax,
                                                   int tid, int nthr, Load load, Op op, Store store) {
  using C = typename Cplx<T>::type;
  const C* __restrict__ tr = tw + (1 << (lnmax - 1));
  const int n = 1 << ln, ne = n >> 3, nb = ntr * ne, G = 1 << lg;
  if (ln == 3) {   // one step each way: nothing to exchange
    for (int t = tid; t < ntr; t += nthr) {
      C v[8];
#pragma unroll
      for (int m = 0; m < 8; ++m) v[m] = load(t, m);
      rev8_first(v, false);
#pragma unroll
      for (int m = 0; m < 8; ++m) op(t, brev(m, 3), v[m]);
      dit8_first(v, true);
#pragma unroll
      for (int m = 0; m < 8; ++m) store(t, m, v[m]);
    }
    return;
  }
  const int left = ln % 3;
  int s = ln - (left ? left : 3);   // levels of size 2^s and below are left
  if (left == 0) {
    for (int k = tid; k < (ne << lg); k += nthr) {
      const int t = k & (G - 1), pos = k >> lg;
      if (t >= ntr) continue;
      C v[8];
#pragma unroll
      for (int m = 0; m < 8; ++m) v[m] = load(t, pos + m * ne);
      rev8_first(v, false);
      store8<PS>(v, x, t * n + pos, ne);
    }
  } else if (left == 2) {
    const int h = n >> 2;
#pragma unroll 2
    for (int k = tid; k < (h << lg); k += nthr) {
      const int t = k & (G - 1), pos = k >> lg, q = t * n + pos;
      if (t >= ntr) continue;
      C x0 = load(t, pos), x1 = load(t, pos + h), x2 = load(t, pos + 2 * h), x3 = load(t, pos + 3 * h);
      bfly1(x0, x2); bfly1(x1, x3);
      bfly1(x0, x1); bflyj(x2, x3, false);
      x[pidx<PS>(q)] = x0; x[pidx<PS>(q + h)] = x1; x[pidx<PS>(q + 2 * h)] = x2; x[pidx<PS>(q + 3 * h)] = x3;
    }
  } else {
    const int h = n >> 1;
#pragma unroll 4
    for (int k = tid; k < (h << lg); k += nthr) {
      const int t = k & (G - 1), pos = k >> lg, q = t * n + pos;
      if (t >= ntr) continue;
      C a = load(t, pos), c = load(t, pos + h);
      bfly1(a, c);
      x[pidx<PS>(q)] = a; x[pidx<PS>(q + h)] = c;
    }
  }
  __syncthreads();
  for (; s > 3; s -= 3) {
    const int h = 1 << (s - 3);
    for (int k = tid; k < nb; k += nthr) {
      const int t = k >> (ln - 3), bi = k & (ne - 1);
      const int pos = bi & (h - 1), j = bi >> (s - 3);
      const int q = t * n + j * 8 * h + pos;
      C v[8];
      load8<PS>(v, x, q, h);
      rev8(v, tr, j, false);
      store8<PS>(v, x, q, h);
    }
    __syncthreads();
  }
  // Element 8 j + m holds the value at the reversed bits.
  const bool spread = sizeof(T) == 8 && nb < nthr;
  for (int k = tid; k < nb; k += nthr) {
    const int t = k >> (ln - 3), j = k & (ne - 1), ky = brev(j, ln - 3);
    C v[8];
    load8<PS>(v, x, 8 * k, 1);
    rev8(v, tr, j, false);
    if (!spread) {
#pragma unroll
      for (int m = 0; m < 8; ++m) op(t, ky + (brev(m, 3) << (ln - 3)), v[m]);
      dit8_first(v, true);
    }
    store8<PS>(v, x, 8 * k, 1);
  }
  __syncthreads();
  if (spread) {
    for (int e = tid; e < ntr * n; e += nthr) op(e >> ln, brev(e & (n - 1), ln), x[pidx<PS>(e)]);
    __syncthreads();
    for (int k = tid; k < nb; k += nthr) {
      C v[8];
      load8<PS>(v, x, 8 * k, 1);
      dit8_first(v, true);
      store8<PS>(v, x, 8 * k, 1);
    }
    __syncthreads();
  }
  for (s = 4; s + 2 < ln; s += 3) {
    const int h = 1 << (s - 1);
    for (int k = tid; k < nb; k += nthr) {
      const int t = k >> (ln - 3), bi = k & (ne - 1);
      const int pos = bi & (h - 1), grp = bi >> (s - 1);
      const int q = t * n + grp * 8 * h + pos;
      C v[8];
      load8<PS>(v, x, q, h);
      dit8(v, tw, lnmax, s, pos, h, true);
      store8<PS>(v, x, q, h);
    }
    __syncthreads();
  }
  if (left == 0) {
    for (int k = tid; k < (ne << lg); k += nthr) {
      const int t = k & (G - 1), pos = k >> lg;
      if (t >= ntr) continue;
      C v[8];
      load8<PS>(v, x, t * n + pos, ne);
      dit8(v, tw, lnmax, s, pos, ne, true);
#pragma unroll
      for (int m = 0; m < 8; ++m) store(t, pos + m * ne, v[m]);
    }
  } else if (left == 2) {
    const int h = n >> 2;
#pragma unroll 2
    for (int k = tid; k < (h << lg); k += nthr) {
      const int t = k & (G - 1), pos = k >> lg, q = t * n + pos;
      if (t >= ntr) continue;
      C x0 = x[pidx<PS>(q)], x1 = x[pidx<PS>(q + h)], x2 = x[pidx<PS>(q + 2 * h)], x3 = x[pidx<PS>(q + 3 * h)];
      const C w1 = tw_of(tw[pos << (lnmax - s)], true), w2 = tw_of(tw[pos << (lnmax - s - 1)], true);
      bfly(x0, x1, w1); bfly(x2, x3, w1);
      bfly(x0, x2, w2); bfly(x1, x3, tw_j(w2, true));
      store(t, pos, x0); store(t, pos + h, x1); store(t, pos + 2 * h, x2); store(t, pos + 3 * h, x3);
    }
  } else {
    const int h = n >> 1;
#pragma unroll 4
    for (int k = tid; k < (h << lg); k += nthr) {
      const int t = k & (G - 1), pos = k >> lg, q = t * n + pos;
      if (t >= ntr) continue;
      C a = x[pidx<PS>(q)], c = x[pidx<PS>(q + h)];
      bfly(a, c, tw_of(tw[pos << (lnmax - s)], true));
      store(t, pos, a); store(t, pos + h, c);
    }
  }
}

// Circular convolution of ntr sequences of length M = 2^lm held back to back
// in x[] (natural order, zero beyond n) with the Bluestein filter whose DFT is
// filt (bit-reversed order, scaled by 1/M; conjugated when inv): forward
// radix-2 DFT (natural in, bit-reversed out), product with the filter,
// inverse DFT (bit-reversed in, natural out).  Shared memory padded as in the power-of-two kernels:
// without it the passes of small distance read many lanes from one bank pair (FP32 509x251, four
// steps: 485 us unpadded, 448 us padded).
template <typename T>
__device__ __forceinline__ void bluestein_conv(typename Cplx<T>::type* x, int lm, int ntr,
                                               const typename Cplx<T>::type* __restrict__ filt,
                                               const typename Cplx<T>::type* __restrict__ tw, int lnmax, bool inv,
                                               int tid, int nthr) {
  using C = typename Cplx<T>::type;
  constexpr int PS = pad_shift<T>();
  fft_rev<T, PS>(x, lm, ntr, tw, lnmax, false, tid, nthr);
  const int m = 1 << lm;
  for (int e = tid; e < ntr * m; e += nthr) {
    C& v = x[pidx<PS>(e)];
    v = cmul_tw(filt[e & (m - 1)], v, inv);
  }
  __syncthreads();
  fft_dit<T, PS>(x, lm, ntr, tw, lnmax, true, tid, nthr);
}

// mean(theta^n) of instance I from its nt partial sums (one per item of the first
// stage's right-hand side kernel), in a fixed order, into *mean (shared); every thread of the
// block calls it; red holds one value per warp of the block.
__device__ __forceinline__ void theta_mean(const InstDev& I, int nt, double* red, double* mean, int tid, int nthr) {
  // four independent partial sums per thread (their loads in flight together)
  double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
  int k = tid;
  for (; k + 3 * nthr < nt; k += 4 * nthr) {
    a0 += I.th_part[k];
    a1 += I.th_part[k + nthr];
    a2 += I.th_part[k + 2 * nthr];
    a3 += I.th_part[k + 3 * nthr];
  }
  for (; k < nt; k += nthr) a0 += I.th_part[k];
  double acc = (a0 + a1) + (a2 + a3);
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if ((tid & 31) == 0) red[tid >> 5] = acc;
  __syncthreads();
  if (tid == 0) {
    double sum = 0.0;
    for (int w = 0; w < (nthr + 31) / 32; ++w) sum += red[w];
    *mean = sum * I.hscale;
  }
  __syncthreads();
}

// ---- power-of-two axes (shared memory padded, pidx<pad_shift<T>()>)

// Threads per block of the power-of-two row passes (FP32 configurable; 1024 / threads
// resident blocks per SM in FP32, three in FP64).
#ifndef APD_ROWS_THREADS32
#define APD_ROWS_THREADS32 256
#endif
template <typename T>
__host__ __device__ constexpr int rows_threads() { return sizeof(T) == 4 ? APD_ROWS_THREADS32 : 256; }
template <typename T>
__host__ __device__ constexpr int rows_min_blocks() { return sizeof(T) == 4 ? 1024 / APD_ROWS_THREADS32 : 3; }

template <typename T>
__global__ void __launch_bounds__(rows_threads<T>(), rows_min_blocks<T>()) k_fft_rows_fwd(const __grid_constant__ BatchDev b) {
  grid_dependency();
  using C = typename Cplx<T>::type;
  constexpr int PS = pad_shift<T>();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* x = reinterpret_cast<C*>(smem_raw);
  const int nitems = b.counts[1], tid = threadIdx.x, nthr = blockDim.x;
  for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
    const int k_inst = find_inst(b.row_start, b.counts[3], it);
    const InstDev& I = b.inst[k_inst];
    if (I.chirp[0] || I.mr_npass[0]) continue;      // an item of another length
    const int n = I.nx, ny = I.ny, ln = I.lnx, ss = I.sstride;
    const int pair0 = (it - b.row_start[k_inst]) * I.row_pairs;
    const int ntr = min(I.row_pairs, ((ny + 1) >> 1) - pair0);
    const T* R = reinterpret_cast<const T*>(I.R);
    fft_rev_from<T, PS>(x, ln, ntr, twiddles<T>(b), b.lnmax, false, tid, nthr, [=](int p, int k) {
      const size_t row = (size_t)(2 * (pair0 + p));
      C z;
      z.x = R[row * n + k];
      z.y = row + 1 < (size_t)ny ? R[(row + 1) * n + k] : T(0);
      return z;
    });
    C* S = reinterpret_cast<C*>(I.S);
    const int nh = (n >> 1) + 1;
    for (int e = tid; e < ntr * nh; e += nthr) {
      const int p = e / nh, k = e - p * nh;
      const C zk = x[pidx<PS>(p * n + brev(k, ln))], zm = x[pidx<PS>(p * n + brev((n - k) & (n - 1), ln))];
      const size_t row = (size_t)(2 * (pair0 + p));
      C A, B;
      A.x = T(0.5) * (zk.x + zm.x); A.y = T(0.5) * (zk.y - zm.y);
      B.x = T(0.5) * (zk.y + zm.y); B.y = T(-0.5) * (zk.x - zm.x);
      S[row * ss + k] = A;
      if (row + 1 < (size_t)ny) S[(row + 1) * ss + k] = B;
    }
    __syncthreads();
  }
}

// Column pass: a work item is a group of col_group (a power of two) adjacent
// spectral columns, loaded and stored row by row (adjacent threads take
// adjacent columns of one row); the forward transform runs from natural to
// bit-reversed order and the inverse back, so the symbol division takes the
// spectrum in bit-reversed order and no permutation pass is needed
// (fft_there_and_back).  The FP32
// form runs it with blocks of 512 threads, two per SM (cols_threads<T>; at 2048^2
// its 257 items of four columns then run in one wave: 0.098 ms per step, with a pass more for input,
// symbol and output each, against 0.120 with one block of 1024 and 0.143 with 256), the FP64 form with 256 (its
// butterflies keep the FP64 pipe busy either way); the load and store loops are
// unrolled so that several global accesses per thread are in flight.
#ifndef APD_COLS_THREADS32
#define APD_COLS_THREADS32 512
#endif
template <typename T>
__host__ __device__ constexpr int cols_threads() { return sizeof(T) == 4 ? APD_COLS_THREADS32 : 256; }

template <typename T>
__global__ void __launch_bounds__(cols_threads<T>(), sizeof(T) == 4 ? 1024 / APD_COLS_THREADS32 : 2)
    k_fft_cols(const __grid_constant__ BatchDev b, int i) {
  grid_dependency();
  using C = typename Cplx<T>::type;
  constexpr int PS = pad_shift<T>();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* x = reinterpret_cast<C*>(smem_raw);
  __shared__ double red[32];
  __shared__ double s_mean;
  const int nitems = b.counts[2], tid = threadIdx.x, nthr = blockDim.x;
  for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
    const int k_inst = find_inst(b.col_start, b.counts[3], it);
    const InstDev& I = b.inst[k_inst];
    if (I.chirp[1] || I.mr_npass[1]) continue;      // an item of another length
    const int n = I.ny, ln = I.lny, ss = I.sstride, nh = (I.nx >> 1) + 1;
    const int G = I.col_group, lg = __ffs(G) - 1;
    const int col0 = (it - b.col_start[k_inst]) * G;
    const int ntr = min(G, nh - col0);
    if (col0 == 0) theta_mean(I, b.rhs_start[k_inst + 1] - b.rhs_start[k_inst], red, &s_mean, tid, nthr);
    C* S = reinterpret_cast<C*>(I.S);
    const double kap = I.kappa[i], scale = I.hscale;
    fft_there_and_back<T, PS>(
        x, ln, lg, ntr, twiddles<T>(b), b.lnmax, tid, nthr,
        [=](int g, int y) { return S[(size_t)y * ss + col0 + g]; },
        [&](int g, int ky, C& v) {
          const int kx = col0 + g;
          if (kx == 0 && ky == 0) {
            v.x = T(s_mean); v.y = T(0);
          } else if (sizeof(T) == 8) {
            const double f = scale * rcp_newton(I.lamx[kx] + I.lamy[ky] - kap);
            v.x = T(double(v.x) * f); v.y = T(double(v.y) * f);
          } else {
            // FP32 form: the symbol in FP32 from the tables rounded once on the host
            const float f = I.hscale32 * __frcp_rn(I.lamx32[kx] + I.lamy32[ky] - I.k32.kappa[i]);
            v.x *= T(f); v.y *= T(f);
          }
        },
        [=](int g, int y, C v) { S[(size_t)y * ss + col0 + g] = v; });
    __syncthreads();
  }
}

template <typename T>
__global__ void __launch_bounds__(rows_threads<T>(), rows_min_blocks<T>()) k_fft_rows_inv(const __grid_constant__ BatchDev b, int i) {
  grid_dependency();
  using C = typename Cplx<T>::type;
  constexpr int PS = pad_shift<T>();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* x = reinterpret_cast<C*>(smem_raw);
  const int nitems = b.counts[1], tid = threadIdx.x, nthr = blockDim.x;
  for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
    const int k_inst = find_inst(b.row_start, b.counts[3], it);
    const InstDev& I = b.inst[k_inst];
    if (I.chirp[0] || I.mr_npass[0]) continue;      // an item of another length
    const int n = I.nx, ny = I.ny, ln = I.lnx, ss = I.sstride;
    const int pair0 = (it - b.row_start[k_inst]) * I.row_pairs;
    const int ntr = min(I.row_pairs, ((ny + 1) >> 1) - pair0);
    const C* S = reinterpret_cast<const C*>(I.S);
    auto load = [=](int p, int k) {
      const size_t row = (size_t)(2 * (pair0 + p));
      const int kk = k <= (n >> 1) ? k : n - k;
      C A = S[row * ss + kk], B;
      B.x = B.y = T(0);
      if (row + 1 < (size_t)ny) B = S[(row + 1) * ss + kk];
      if (kk != k) { A.y = -A.y; B.y = -B.y; }
      C z;
      z.x = A.x - B.y; z.y = A.y + B.x;
      return z;
    };
    if constexpr (sizeof(T) == 4) {
      fft_rev_from<T, PS>(x, ln, ntr, twiddles<T>(b), b.lnmax, true, tid, nthr, load);
    } else {
      // FP64: the two sums of load() on all threads, not on the n/8 of a step (256^2, ten steps: 244 us
      // against 278; 2048^2: no difference)
#pragma unroll 4
      for (int e = tid; e < ntr * n; e += nthr) x[pidx<PS>(e)] = load(e >> ln, e & (n - 1));
      __syncthreads();
      fft_rev<T, PS>(x, ln, ntr, twiddles<T>(b), b.lnmax, true, tid, nthr);
    }
    T* th = reinterpret_cast<T*>(I.Xs[i]) + 2 * (size_t)I.nx * I.ny;
    for (int e = tid; e < ntr * n; e += nthr) {
      const int p = e >> ln, m = e & (n - 1);
      const size_t row = (size_t)(2 * (pair0 + p));
      const C z = x[pidx<PS>(p * n + brev(m, ln))];
      th[row * n + m] = z.x;
      if (row + 1 < (size_t)ny) th[(row + 1) * n + m] = z.y;
    }
    __syncthreads();
  }
}

// ---- mixed radix: lengths 2^a 3^b 5^c 7^d that are not powers of two, by
// Stockham's self-sorting formulation (natural order in and out, ping-pong
// between two buffers of n values).  With Ns the product of the radices of
// the passes before, a pass of radix R takes, for each j < n/R with k = j mod Ns,
// the R values src[j + r n/R] times W_{Ns R}^{k r}, transforms them with an
// R-point DFT and writes them to dst[(j - k) R + k + r Ns].

// cos and sin of 2 pi q / R, q = 1 .. (R-1)/2, for the odd radices.
__device__ __forceinline__ constexpr double root_cos(int R, int q) {
  return R == 3 ? -0.5
       : R == 5 ? (q == 1 ? 0.3090169943749474241022934 : -0.8090169943749474241022934)
       : (q == 1 ? 0.6234898018587335305250049 : q == 2 ? -0.2225209339563144042889026 : -0.9009688679024191262361023);
}
__device__ __forceinline__ constexpr double root_sin(int R, int q) {
  return R == 3 ? 0.8660254037844386467637232
       : R == 5 ? (q == 1 ? 0.9510565162951535721164393 : 0.5877852522924731291687060)
       : (q == 1 ? 0.7818314824680298087084445 : q == 2 ? 0.9749279121818236070181317 : 0.4338837391175581204757683);
}

// R-point DFT of v in place, R odd (exp(-2 pi i ab/R); conjugate roots when inv):
// opposite inputs are paired, y_a = v_0 + sum_b [(v_b + v_{R-b}) cos - i (v_b - v_{R-b}) sin](2 pi ab/R).
template <int R, typename C>
__device__ __forceinline__ void small_dft(C* v, bool inv) {
  using T = decltype(v[0].x);
  constexpr int H = (R - 1) / 2;
  C sp[H], dm[H], out[R];
  C y0 = v[0];
#pragma unroll
  for (int b = 1; b <= H; ++b) {
    sp[b - 1] = cadd(v[b], v[R - b]);
    dm[b - 1] = csub(v[b], v[R - b]);
    y0 = cadd(y0, sp[b - 1]);
  }
  out[0] = y0;
#pragma unroll
  for (int a = 1; a <= H; ++a) {
    C re = v[0], im;
    im.x = T(0); im.y = T(0);
#pragma unroll
    for (int b = 1; b <= H; ++b) {
      const int q = (a * b) % R, qq = q <= H ? q : R - q;
      const T c = T(root_cos(R, qq)), sn = q <= H ? T(root_sin(R, qq)) : -T(root_sin(R, qq));
      re.x += c * sp[b - 1].x; re.y += c * sp[b - 1].y;
      im.x += sn * dm[b - 1].x; im.y += sn * dm[b - 1].y;
    }
    C ya, yb;   // re -+ i im (forward), re +- i im (inverse)
    if (!inv) { ya.x = re.x + im.y; ya.y = re.y - im.x; yb.x = re.x - im.y; yb.y = re.y + im.x; }
    else { ya.x = re.x - im.y; ya.y = re.y + im.x; yb.x = re.x + im.y; yb.y = re.y - im.x; }
    out[a] = ya;
    out[R - a] = yb;
  }
#pragma unroll
  for (int a = 0; a < R; ++a) v[a] = out[a];
}

template <typename T, int R>
__device__ __forceinline__ void stockham_pass(typename Cplx<T>::type* x, int m, int n, int ntr, int Ns, int src_off,
                                              const typename Cplx<T>::type* __restrict__ tw, bool inv, int tid,
                                              int nthr) {
  using C = typename Cplx<T>::type;
  const int nr = n / R, dst_off = n - src_off, tws = n / (Ns * R);
  for (int e = tid; e < ntr * nr; e += nthr) {
    const int p = e / nr, j = e - p * nr, k = j % Ns;
    const C* src = x + p * m + src_off;
    C* dst = x + p * m + dst_off;
    C v[R];
    v[0] = src[j];
    if constexpr (R == 4) {
      // two levels of butterflies with their whole twiddles: W^{2k}, then W^k times 1 and W_4
      v[1] = src[j + nr];
      v[2] = src[j + 2 * nr];
      v[3] = src[j + 3 * nr];
      const C w1 = tw_of(tw[k * tws], inv), w2 = tw_of(tw[2 * k * tws], inv);
      bfly(v[0], v[2], w2);
      bfly(v[1], v[3], w2);
      bfly(v[0], v[1], w1);
      bfly(v[2], v[3], tw_j(w1, inv));
      const C y1 = v[2];
      v[2] = v[1];
      v[1] = y1;
    } else if constexpr (R == 2) {
      v[1] = src[j + nr];
      bfly(v[0], v[1], tw_of(tw[k * tws], inv));
    } else {
#pragma unroll
      for (int r = 1; r < R; ++r) v[r] = cmul_tw(tw[k * r * tws], src[j + r * nr], inv);
      small_dft<R>(v, inv);
    }
    const int d0 = (j - k) * R + k;
#pragma unroll
    for (int r = 0; r < R; ++r) dst[d0 + r * Ns] = v[r];
  }
  __syncthreads();
}

// ntr transforms of length n (plan: npass radices, 4 bits each, first pass in the
// low bits), transform p in x + p m, starting in the buffer at offset off (0 or n);
// returns the offset of the buffer that holds the result.  tw[q] = W_n^q, q < n.
template <typename T>
__device__ __forceinline__ int stockham(typename Cplx<T>::type* x, int m, int n, int ntr, unsigned plan, int npass,
                                        const typename Cplx<T>::type* __restrict__ tw, bool inv, int off, int tid,
                                        int nthr) {
  int Ns = 1;
  for (int q = 0; q < npass; ++q) {
    const int R = (int)((plan >> (4 * q)) & 15u);
    if (R == 4) stockham_pass<T, 4>(x, m, n, ntr, Ns, off, tw, inv, tid, nthr);
    else if (R == 2) stockham_pass<T, 2>(x, m, n, ntr, Ns, off, tw, inv, tid, nthr);
    else if (R == 3) stockham_pass<T, 3>(x, m, n, ntr, Ns, off, tw, inv, tid, nthr);
    else if (R == 5) stockham_pass<T, 5>(x, m, n, ntr, Ns, off, tw, inv, tid, nthr);
    else stockham_pass<T, 7>(x, m, n, ntr, Ns, off, tw, inv, tid, nthr);
    off = n - off;
    Ns *= R;
  }
  return off;
}

// ---- axes whose length is not a power of two: mixed radix where the length
// factors into 2, 3, 5 and 7, else Bluestein; x holds ntr regions of m = 2^ln
// values (the Bluestein convolution length, >= 2n: room for the two mixed-radix
// buffers as well) back to back

template <typename T>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 4 : 3) k_fft_rows_fwd_bs(const __grid_constant__ BatchDev b) {
  constexpr int PS = pad_shift<T>();   // Bluestein's regions; the mixed-radix buffers are not padded
  grid_dependency();
  using C = typename Cplx<T>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* x = reinterpret_cast<C*>(smem_raw);
  const int nitems = b.counts[1], tid = threadIdx.x, nthr = blockDim.x;
  for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
    const int k_inst = find_inst(b.row_start, b.counts[3], it);
    const InstDev& I = b.inst[k_inst];
    const C* ch = reinterpret_cast<const C*>(I.chirp[0]);
    if (!ch && !I.mr_npass[0]) continue;            // a power-of-two item
    const int n = I.nx, ny = I.ny, ln = I.lnx, m = 1 << ln, ss = I.sstride;
    const int pair0 = (it - b.row_start[k_inst]) * I.row_pairs;
    const int ntr = min(I.row_pairs, ((ny + 1) >> 1) - pair0);
    const T* R = reinterpret_cast<const T*>(I.R);
    if (I.mr_npass[0]) {
      for (int e = tid; e < ntr * n; e += nthr) {
        const int p = e / n, k = e - p * n;
        const size_t row = (size_t)(2 * (pair0 + p));
        C z;
        z.x = R[row * n + k];
        z.y = row + 1 < (size_t)ny ? R[(row + 1) * n + k] : T(0);
        x[p * m + k] = z;
      }
      __syncthreads();
      const int off = stockham<T>(x, m, n, ntr, I.mr_plan[0], I.mr_npass[0], reinterpret_cast<const C*>(I.mr_tw[0]),
                                  false, 0, tid, nthr);
      C* S = reinterpret_cast<C*>(I.S);
      const int nh = (n >> 1) + 1;
      for (int e = tid; e < ntr * nh; e += nthr) {
        const int p = e / nh, k = e - p * nh, km = k == 0 ? 0 : n - k;
        const C zk = x[p * m + off + k], zm = x[p * m + off + km];
        const size_t row = (size_t)(2 * (pair0 + p));
        C A, B;
        A.x = T(0.5) * (zk.x + zm.x); A.y = T(0.5) * (zk.y - zm.y);
        B.x = T(0.5) * (zk.y + zm.y); B.y = T(-0.5) * (zk.x - zm.x);
        S[row * ss + k] = A;
        if (row + 1 < (size_t)ny) S[(row + 1) * ss + k] = B;
      }
      __syncthreads();
      continue;
    }
    for (int e = tid; e < ntr * m; e += nthr) {
      const int p = e >> ln, k = e & (m - 1);
      const size_t row = (size_t)(2 * (pair0 + p));
      C z;
      z.x = T(0); z.y = T(0);
      if (k < n) {
        z.x = R[row * n + k];
        if (row + 1 < (size_t)ny) z.y = R[(row + 1) * n + k];
        z = cmul_tw(ch[k], z, false);
      }
      x[pidx<PS>(e)] = z;
    }
    __syncthreads();
    bluestein_conv<T>(x, ln, ntr, reinterpret_cast<const C*>(I.filt[0]), twiddles<T>(b), b.lnmax, false, tid, nthr);
    C* S = reinterpret_cast<C*>(I.S);
    const int nh = (n >> 1) + 1;
    for (int e = tid; e < ntr * nh; e += nthr) {
      const int p = e / nh, k = e - p * nh, km = k == 0 ? 0 : n - k;
      const C zk = cmul_tw(ch[k], x[pidx<PS>(p * m + k)], false), zm = cmul_tw(ch[km], x[pidx<PS>(p * m + km)], false);
      const size_t row = (size_t)(2 * (pair0 + p));
      C A, B;
      A.x = T(0.5) * (zk.x + zm.x); A.y = T(0.5) * (zk.y - zm.y);
      B.x = T(0.5) * (zk.y + zm.y); B.y = T(-0.5) * (zk.x - zm.x);
      S[row * ss + k] = A;
      if (row + 1 < (size_t)ny) S[(row + 1) * ss + k] = B;
    }
    __syncthreads();
  }
}

// v times a real factor given in FP64, rounded once: FP32 values by the factor as a pair of floats.
__device__ __forceinline__ void apply_factor(double2& v, double f) { v.x *= f; v.y *= f; }
__device__ __forceinline__ void apply_factor(float2& v, double f) {
  const F2 p = f2_from_double(f), a = f2_mulf(p, v.x), c = f2_mulf(p, v.y);
  v.x = a.h + a.l;
  v.y = c.h + c.l;
}

// The forward Bluestein convolution differs from the spectrum along y by the
// factor conj(w_ky), which the inverse transform's input chirp w_ky cancels,
// so the division by the symbol applies to the convolution directly.
template <typename T>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 4 : 3) k_fft_cols_bs(const __grid_constant__ BatchDev b, int i) {
  constexpr int PS = pad_shift<T>();   // Bluestein's regions; the mixed-radix buffers are not padded
  grid_dependency();
  using C = typename Cplx<T>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* x = reinterpret_cast<C*>(smem_raw);
  __shared__ double red[8];
  __shared__ double s_mean;
  const int nitems = b.counts[2], tid = threadIdx.x, nthr = blockDim.x;
  for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
    const int k_inst = find_inst(b.col_start, b.counts[3], it);
    const InstDev& I = b.inst[k_inst];
    const C* ch = reinterpret_cast<const C*>(I.chirp[1]);
    if (!ch && !I.mr_npass[1]) continue;            // a power-of-two item
    const C* filt = reinterpret_cast<const C*>(I.filt[1]);
    const int n = I.ny, ln = I.lny, m = 1 << ln, ss = I.sstride, nh = (I.nx >> 1) + 1;
    const int col0 = (it - b.col_start[k_inst]) * I.col_group;
    const int ntr = min(I.col_group, nh - col0);
    if (col0 == 0) theta_mean(I, b.rhs_start[k_inst + 1] - b.rhs_start[k_inst], red, &s_mean, tid, nthr);
    C* S = reinterpret_cast<C*>(I.S);
    if (I.mr_npass[1]) {
      const C* tw = reinterpret_cast<const C*>(I.mr_tw[1]);
      for (int e = tid; e < ntr * n; e += nthr) {
        const int g = e / n, y = e - g * n;
        x[g * m + y] = S[(size_t)y * ss + col0 + g];
      }
      __syncthreads();
      const int off = stockham<T>(x, m, n, ntr, I.mr_plan[1], I.mr_npass[1], tw, false, 0, tid, nthr);
      const double kap = I.kappa[i];
      const double scale = I.hscale;
      for (int e = tid; e < ntr * n; e += nthr) {
        const int g = e / n, ky = e - g * n, kx = col0 + g;
        C v = x[g * m + off + ky];
        if (kx == 0 && ky == 0) {
          v.x = T(s_mean); v.y = T(0);
        } else {
          const double f = scale * rcp_newton(I.lamx[kx] + I.lamy[ky] - kap);
          apply_factor(v, f);
        }
        x[g * m + off + ky] = v;
      }
      __syncthreads();
      const int off2 = stockham<T>(x, m, n, ntr, I.mr_plan[1], I.mr_npass[1], tw, true, off, tid, nthr);
      for (int e = tid; e < ntr * n; e += nthr) {
        const int g = e / n, y = e - g * n;
        S[(size_t)y * ss + col0 + g] = x[g * m + off2 + y];
      }
      __syncthreads();
      continue;
    }
    for (int e = tid; e < ntr * m; e += nthr) {
      const int g = e >> ln, y = e & (m - 1);
      C z;
      z.x = T(0); z.y = T(0);
      if (y < n) z = cmul_tw(ch[y], S[(size_t)y * ss + col0 + g], false);
      x[pidx<PS>(e)] = z;
    }
    __syncthreads();
    bluestein_conv<T>(x, ln, ntr, filt, twiddles<T>(b), b.lnmax, false, tid, nthr);
    const double kap = I.kappa[i];
    const double scale = I.hscale;
    for (int e = tid; e < ntr * m; e += nthr) {
      const int g = e >> ln, ky = e & (m - 1), kx = col0 + g;
      C v = x[pidx<PS>(e)];
      if (ky >= n) {
        v.x = T(0); v.y = T(0);
      } else if (kx == 0 && ky == 0) {
        v.x = T(s_mean); v.y = T(0);
      } else {
        const double f = scale * rcp_newton(I.lamx[kx] + I.lamy[ky] - kap);
        apply_factor(v, f);
      }
      x[pidx<PS>(e)] = v;
    }
    __syncthreads();
    bluestein_conv<T>(x, ln, ntr, filt, twiddles<T>(b), b.lnmax, true, tid, nthr);
    for (int e = tid; e < ntr * m; e += nthr) {
      const int g = e >> ln, y = e & (m - 1);
      if (y < n) S[(size_t)y * ss + col0 + g] = cmul_tw(ch[y], x[pidx<PS>(e)], true);
    }
    __syncthreads();
  }
}

template <typename T>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 4 : 3) k_fft_rows_inv_bs(const __grid_constant__ BatchDev b, int i) {
  constexpr int PS = pad_shift<T>();   // Bluestein's regions; the mixed-radix buffers are not padded
  grid_dependency();
  using C = typename Cplx<T>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* x = reinterpret_cast<C*>(smem_raw);
  const int nitems = b.counts[1], tid = threadIdx.x, nthr = blockDim.x;
  for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
    const int k_inst = find_inst(b.row_start, b.counts[3], it);
    const InstDev& I = b.inst[k_inst];
    const C* ch = reinterpret_cast<const C*>(I.chirp[0]);
    if (!ch && !I.mr_npass[0]) continue;            // a power-of-two item
    const int n = I.nx, ny = I.ny, ln = I.lnx, m = 1 << ln, ss = I.sstride;
    const int pair0 = (it - b.row_start[k_inst]) * I.row_pairs;
    const int ntr = min(I.row_pairs, ((ny + 1) >> 1) - pair0);
    const C* S = reinterpret_cast<const C*>(I.S);
    if (I.mr_npass[0]) {
      for (int e = tid; e < ntr * n; e += nthr) {
        const int p = e / n, k = e - p * n;
        const size_t row = (size_t)(2 * (pair0 + p));
        const bool two = row + 1 < (size_t)ny;
        const int kk = k <= (n >> 1) ? k : n - k;   // Hermitian symmetry of a real row
        C A = S[row * ss + kk], B;
        B.x = B.y = T(0);
        if (two) B = S[(row + 1) * ss + kk];
        if (kk != k) { A.y = -A.y; B.y = -B.y; }
        C z;
        z.x = A.x - B.y; z.y = A.y + B.x;
        x[p * m + k] = z;
      }
      __syncthreads();
      const int off = stockham<T>(x, m, n, ntr, I.mr_plan[0], I.mr_npass[0], reinterpret_cast<const C*>(I.mr_tw[0]),
                                  true, 0, tid, nthr);
      T* th = reinterpret_cast<T*>(I.Xs[i]) + 2 * (size_t)I.nx * I.ny;
      for (int e = tid; e < ntr * n; e += nthr) {
        const int p = e / n, mm = e - p * n;
        const size_t row = (size_t)(2 * (pair0 + p));
        const C z = x[p * m + off + mm];
        th[row * n + mm] = z.x;
        if (row + 1 < (size_t)ny) th[(row + 1) * n + mm] = z.y;
      }
      __syncthreads();
      continue;
    }
    for (int e = tid; e < ntr * m; e += nthr) {
      const int p = e >> ln, k = e & (m - 1);
      const size_t row = (size_t)(2 * (pair0 + p));
      const bool two = row + 1 < (size_t)ny;
      C A, B, z;
      A.x = A.y = B.x = B.y = z.x = z.y = T(0);
      if (k < n) {
        const int kk = k <= (n >> 1) ? k : n - k;   // Hermitian symmetry of a real row
        A = S[row * ss + kk];
        if (two) B = S[(row + 1) * ss + kk];
        if (kk != k) { A.y = -A.y; B.y = -B.y; }
        z.x = A.x - B.y; z.y = A.y + B.x;
        z = cmul_tw(ch[k], z, true);
      }
      x[pidx<PS>(e)] = z;
    }
    __syncthreads();
    bluestein_conv<T>(x, ln, ntr, reinterpret_cast<const C*>(I.filt[0]), twiddles<T>(b), b.lnmax, true, tid, nthr);
    T* th = reinterpret_cast<T*>(I.Xs[i]) + 2 * (size_t)I.nx * I.ny;
    for (int e = tid; e < ntr * m; e += nthr) {
      const int p = e >> ln, mm = e & (m - 1);
      if (mm >= n) continue;
      const size_t row = (size_t)(2 * (pair0 + p));
      const C z = cmul_tw(ch[mm], x[pidx<PS>(e)], true);
      th[row * n + mm] = z.x;
      if (row + 1 < (size_t)ny) th[(row + 1) * n + mm] = z.y;
    }
    __syncthreads();
  }
}

}  // namespace apd
