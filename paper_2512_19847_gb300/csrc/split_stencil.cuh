// The FP64 explicit and update kernels of the WENO schemes with the split fluxes of
// split_flux.cuh: three passes over a staged tile,
//   1. FP64 increments along both axes, kept as pairs of floats (one FP64 operation each),
//   2. the nonlinear interface terms N, on the FP32 pipe, in runs of neighbouring interfaces,
//   3. per cell: the linear parts and the closed forms in FP64, with the differences of N.
// Where an interface of the tile is rough (split_flux.cuh), the whole FP64 fluxes are taken too, pair by pair
// in the space of the increments (w5_fluxes_xy, axis_fluxes), for the cells beside such an interface:
// which form a cell takes depends on its stencil and the field's largest values alone, not on tile
// or batch.  The test of every interface costs 0.3 to 0.9 % of a step on smooth data.
// What bounds them is still the FP64 pipe (2 operations per clock and SM), with 100 (explicit, all
// terms) and 74 (update) FP64 operations per cell instead of 510 and 370, beside about 450 FP32
// instructions per interface.  WENO5 at 2048^2, ms per step (32x8 tiles): explicit
// 6.17 -> 1.65, update 6.06 -> 1.55; WENO3 at 256^2, 10 steps: 0.98 -> 0.44 and 1.00 -> 0.41.  Measured choices
// (explicit + update, ms per step): WENO5 at 2048^2 768 threads per SM (80 registers) 1.65 + 1.55, 512 (128
// registers) 1.77 + 1.71; runs of 3 interfaces 1.65 + 1.55, of 2 1.78 + 1.69, of 4 1.73 + 1.86.  WENO3 512
// threads 0.044 + 0.041 at 256^2 and 1.48 + 1.41 at 2048^2, 768 0.050 + 0.045 and 1.40 + 1.31: a choice for
// the sizes the paper runs WENO3 at, 6 % against the largest.
#pragma once
#include "split_flux.cuh"
#include "stencil_kernels.cuh"

namespace apd {

#ifndef APD_SPLIT_RUN
#define APD_SPLIT_RUN 3   // interfaces per run of pass 2
#endif
#ifndef APD_SPLIT_THREADS5
#define APD_SPLIT_THREADS5 768   // threads per SM the split kernels are compiled for, WENO5
#endif
#ifndef APD_SPLIT_THREADS3
#define APD_SPLIT_THREADS3 512   // ... and WENO3
#endif

template <int SCHEME, int TX, int TY>
struct SplitGeo {
  using G = Geo<double, SCHEME, TX, TY>;
  static constexpr int NS = SCHEME == WENO5_C4 ? 4 : 2;                    // increments of one reconstruction
  static constexpr int LX = G::W - 1, LY = G::HH - 1;                      // increments per line
  static constexpr int LIX = TY * LX, LIY = LY * TX;                       // per field
  // elements of 8 bytes: increments of F fields per axis, N of P pairs per axis
  static constexpr int inc(int F) { return F * (LIX + LIY); }
  static constexpr int nl(int P) { return P * (G::NX + G::NY); }
  // scratch of the whole fluxes of one pair, and with these fluxes
  static constexpr int WSCR = SCHEME == WENO5_C4 ? 4 * (G::LSX + G::LSY) : 4 * G::LS;
  static constexpr int WHOLE = WSCR + G::NX + G::NY;
  static_assert(WHOLE <= inc(5), "the whole fluxes of a pair take the place of the increments");
  static constexpr size_t explicit_bytes = 128 + 8 * (size_t)(6 * G::PL + inc(5) + nl(3));
  // Update: what lies before N, behind n staged planes: the increments, or (whole fluxes) from
  // plane 5 on, the partner being in planes 3 and 4.
  static __host__ __device__ constexpr int update_front(int n) {
    const int a = n * G::PL + inc(4), b = 5 * G::PL + WHOLE;
    return a > b ? a : b;
  }
  static constexpr size_t update_bytes(int n) { return 128 + 8 * (size_t)(update_front(n) + nl(2)); }
};

template <int SCHEME, int THREADS>
__host__ __device__ constexpr int split_min_blocks() {
  const int n = (SCHEME == WENO5_C4 ? APD_SPLIT_THREADS5 : APD_SPLIT_THREADS3) / THREADS;
  return n > 0 ? n : 1;
}

// The limits of the tile's instance, by one thread, once for the tiles of an instance in turn.
template <int SCHEME>
__device__ __forceinline__ void load_limits(const InstDev& I, const InstDev** of, SplitLimits* lim, F2 w, int tid) {
  if (tid != 32 || *of == &I) return;
  *of = &I;
  *lim = split_limits(I.mag[0], I.mag[1], I.mag[2], fminf(1.f, __fdividef(I.k32.qtau, I.k32.te2)), w.h,
                      SCHEME == WENO5_C4 ? APD_SPLIT_ROUGH5 : APD_SPLIT_ROUGH3);
}

// Pass 1: increments of NF staged planes along x (fx) and NF along y (fy).
template <int SCHEME, int TX, int TY, int NF>
__device__ __forceinline__ void split_increments(const double* const* fx, const double* const* fy, F2* ix, F2* iy, int tid) {
  using S = SplitGeo<SCHEME, TX, TY>;
  using G = typename S::G;
  for (int k = tid; k < S::LIX + S::LIY; k += G::NT) {
    if (k < S::LIX) {
      const int line = k / S::LX, o = (G::H + line) * G::BW + G::XO + (k - line * S::LX);
#pragma unroll
      for (int f = 0; f < NF; ++f) ix[f * S::LIX + k] = f2_from_double(fx[f][o + 1] - fx[f][o]);
    } else {
      const int r = k - S::LIX, pt = r / TX, o = pt * G::BW + G::XO + G::H + (r - pt * TX);
#pragma unroll
      for (int f = 0; f < NF; ++f) iy[f * S::LIY + r] = f2_from_double(fy[f][o + G::BW] - fy[f][o]);
    }
  }
}

// Pass 1 of the update: increments of v1, v2 and of the dissipation partner
// P = sum over the earlier stages' staged u planes (from plane 3 on) of weight (wh + wl) times u,
// formed from the planes' increments.
template <int SCHEME, int TX, int TY>
__device__ __forceinline__ void split_increments_update(const double* s, int nw, const F2* wt, F2* ix, F2* iy, int tid) {
  using S = SplitGeo<SCHEME, TX, TY>;
  using G = typename S::G;
  constexpr int PL = G::PL;
  for (int k = tid; k < S::LIX + S::LIY; k += G::NT) {
    const bool ax = k < S::LIX;
    const int r = ax ? k : k - S::LIX, line = ax ? r / S::LX : r % TX, pt = ax ? r - line * S::LX : r / TX;
    const int o = ax ? (G::H + line) * G::BW + G::XO + pt : pt * G::BW + G::XO + G::H + line, st = ax ? 1 : G::BW;
    F2* out = (ax ? ix : iy) + r;
    const int fs = ax ? S::LIX : S::LIY;
    const double* v = s + PL + o;
    const F2 d1 = f2_from_double(v[st] - v[0]), d2 = f2_from_double(v[PL + st] - v[PL]);
    out[0] = ax ? d1 : d2;
    out[fs] = ax ? d2 : d1;
    F2 p1 = f2(0.f, 0.f), p2 = p1;
    const double* u = s + 3 * PL + o;
    for (int m = 0; m < nw; ++m, u += 2 * PL) {
      const F2 a1 = f2_mul(wt[m], f2_from_double(u[st] - u[0])), a2 = f2_mul(wt[m], f2_from_double(u[PL + st] - u[PL]));
      p1 = m ? f2_add(p1, a1) : a1;
      p2 = m ? f2_add(p2, a2) : a2;
    }
    out[2 * fs] = p1;
    out[3 * fs] = p2;
  }
}

// Pass 2, one run: the increments of g and U at ig, iu (stride st between points); N of interfaces
// m0 .. m0 + KR - 1 into out (stride so), those from skip on.  sg = -1 negates g, by
// exchanging the two reconstructions (-g + U = -(g - U)).  Returns whether any is rough.
template <int SCHEME, int KR>
__device__ __forceinline__ bool split_run(const F2* ig, const F2* iu, float sg, int st, F2 w, float lim, F2* out, int so,
                                          int m0, int skip) {
  constexpr int NS = SCHEME == WENO5_C4 ? 4 : 2, ND = KR + NS;
  F2 D[ND], q[KR], qm[KR];
  bool b[KR], bm[KR];
#pragma unroll
  for (int j = 0; j < ND - 1; ++j) D[j] = f2_norm(f2_addr(ig[(m0 + j) * st], iu[(m0 + j) * st], sg));
  if constexpr (SCHEME == WENO5_C4) w5_split<KR>(D, w, lim, q, b);
  else w3_split<KR>(D, w, lim, q, b);
  // from the right: the same with the increments in reverse
#pragma unroll
  for (int j = 1; j < ND; ++j) D[ND - 1 - j] = f2_norm(f2_addr(ig[(m0 + j) * st], iu[(m0 + j) * st], -sg));
  if constexpr (SCHEME == WENO5_C4) w5_split<KR>(D, w, lim, qm, bm);
  else w3_split<KR>(D, w, lim, qm, bm);
  bool rough = false;
#pragma unroll
  for (int i = 0; i < KR; ++i)
    if (i >= skip) {
      F2 r = f2_norm(f2_sub(qm[KR - 1 - i], q[i]));
      if (b[i] || bm[KR - 1 - i]) r.h = rough_mark();
      rough |= is_rough(r.h);
      out[(m0 + i) * so] = f2(sg * r.h, sg * r.l);
    }
  return rough;
}

// Pass 2: NP pairs per axis.  Pair p takes the fields gi(p) and ui(p) of the increments
// (NP = 3: g 0 1 2, U 1 3 4; NP = 2: g 0 1, U 2 3; NP = 1: g 0, U 1); the x pair NEGX is negated.
// A line's last run ends at its last interface and leaves out what the one before it has.
// rough is set where any interface is.
template <int SCHEME, int TX, int TY, int NP, int NEGX>
__device__ __forceinline__ void split_interfaces(const F2* ix, const F2* iy, F2* nx, F2* ny, F2 w, const SplitLimits& lim, int* rough,
                                                 int tid) {
  using S = SplitGeo<SCHEME, TX, TY>;
  using G = typename S::G;
  constexpr int KR = APD_SPLIT_RUN;
  static_assert(TX + 1 >= KR && TY + 1 >= KR, "a run fits a line");
  constexpr int RX = (TX + 1 + KR - 1) / KR, RY = (TY + 1 + KR - 1) / KR;
  constexpr int IX = NP * TY * RX, IY = NP * TX * RY;
  const float le = lim.e, lb = lim.b;
  for (int k = tid; k < IX + IY; k += G::NT) {
    const bool ax = k < IX;
    const int kk = ax ? k : k - IX, nl = ax ? TY : TX, per = ax ? TY * RX : TX * RY;
    const int p = kk / per, r = kk - p * per, run = r / nl, line = r - run * nl;
    const int gi = p, ui = NP == 1 ? 1 : (NP == 2 ? 2 + p : (p == 0 ? 1 : 2 + p));
    const F2* base = ax ? ix + line * S::LX : iy + line;
    const int fs = ax ? S::LIX : S::LIY;
    const int over = (TX + 1) % KR == 0 && (TY + 1) % KR == 0 ? 0 : max(0, (run + 1) * KR - (ax ? TX + 1 : TY + 1));
    if (split_run<SCHEME, KR>(base + gi * fs, base + ui * fs, (ax && p == NEGX) ? -1.f : 1.f, ax ? 1 : TX, w,
                              NP == 1 || (NP == 3 && p == 0) ? le : lb,
                              ax ? nx + p * G::NX + line * (TX + 1) : ny + p * G::NY + line, ax ? 1 : TX, run * KR - over, over))
      *rough = 1;
  }
}

// The whole FP64 fluxes of one pair per axis into wx [TY][TX+1] and wy [TY+1][TX], behind the scratch at scr;
// every thread of the block calls it, and it ends with a barrier.
template <int SCHEME, int TX, int TY, bool NEGX>
__device__ __forceinline__ void whole_pair(const double* gx, const double* ux, const double* gy, const double* uy, double* scr,
                                           double weno_eps, int tid) {
  using S = SplitGeo<SCHEME, TX, TY>;
  double* wx = scr + S::WSCR;
  both_axes<double, SCHEME, TX, TY, 1, NEGX ? 1u : 0u, 0u, SCHEME == WENO5_C4>(&gx, &ux, &gy, &uy, scr, wx, wx + S::G::NX, weno_eps, tid);
  __syncthreads();
}

// 8 (f_1 - f_-1) - (f_2 - f_-2) and the fourth difference along a line.
__device__ __forceinline__ double cd12(const double* f, int st) { return fma(8.0, f[st] - f[-st], f[-2 * st] - f[2 * st]); }
// The same in the order of the whole form (cdiff): D_0 . u, a difference of nearly opposite sums that
// the right-hand side divides by dt, keeps its rounding (theta of a 2048^2 Taylor-Green step against
// plain FP64: 5e-15 as the whole form's 1.2e-14; 3.6e-14 with the differences first).
__device__ __forceinline__ double cd12s(const double* f, int st) {
  return fma(-8.0, f[-st], fma(8.0, f[st], -f[2 * st])) + f[-2 * st];
}
// 12 h times the flux difference of g: 6 (g_1 - g_-1) and the difference of N.
__device__ __forceinline__ double fd12(double dg, double sg6, const F2* n, int a, int b) {
  return fma(sg6, dg, f2_to_double(f2_sub(n[b], n[a])));
}
// The same, or (a rough interface beside the cell) from the whole fluxes w (flux_scale: 1/6 or 1/2 of 1/h).
template <int SCHEME>
__device__ __forceinline__ double fd12(double dg, double sg6, const F2* n, int a, int b, const double* w) {
  const F2 d = f2_sub(n[b], n[a]);
  return is_rough(d.h) ? (SCHEME == WENO5_C4 ? 2.0 : 6.0) * (w[b] - w[a]) : fma(sg6, dg, f2_to_double(d));
}

__device__ __forceinline__ F2 f2_of(double x) {
  const float h = (float)x;
  return f2(h, (float)(x - (double)h));
}

// ---------------------------------------------------------------------------
// k_explicit (stencil_kernels.cuh) with split fluxes.
template <int SCHEME, int TX, int TY>
__global__ void __launch_bounds__(SplitGeo<SCHEME, TX, TY>::G::NT, split_min_blocks<SCHEME, SplitGeo<SCHEME, TX, TY>::G::NT>()) k_explicit_split(const __grid_constant__ BatchDev b, int j, unsigned need,
                                                                                double weno_eps) {
  grid_dependency();
  using S = SplitGeo<SCHEME, TX, TY>;
  using G = typename S::G;
  constexpr int BW = G::BW, PL = G::PL, NX = G::NX, NY = G::NY;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ uint64_t bars[2];
  __shared__ SplitLimits s_lim;
  __shared__ const InstDev* lim_of;   // the instance s_lim is of
  __shared__ int s_rough;      // the tile holds a rough interface
  double* stage = aligned_smem<double>(smem_raw);
  F2* ix = reinterpret_cast<F2*>(stage + 6 * PL);
  F2* iy = ix + 5 * S::LIX;
  F2* nxs = iy + 5 * S::LIY;   // [3][NX]: (q;v1), (-v1;u1), (v2;u2)
  F2* nys = nxs + 3 * NX;      // [3][NY]: (q;v2), (v2;u1), (v1;u2)
  double* scr = reinterpret_cast<double*>(ix);
  const double* wx = scr + S::WSCR;
  const double* wy = wx + NX;
  const int tx = threadIdx.x, ty = threadIdx.y, tid = tx + ty * TX + threadIdx.z * TX * TY;
  const F2 w = f2_of((SCHEME == WENO5_C4 ? 16.0 : 4.0) * weno_eps);
  const bool needB = (need & NEED_DLFB) != 0, needE = (need & NEED_E) != 0;
  if (tid == 32) lim_of = nullptr;
  PlaneList pr;
  for (int k = 0; k < 6; ++k) pr.add(j, k);
  tile_loop<double, G, TX, TY, 1, true>(b, pr, stage, bars, tid, [&](const InstDev& I, const TileRef& t, double* s) {
    const double* su1 = s;
    const double* su2 = s + PL;
    const double* sth = s + 2 * PL;
    const double* sv1 = s + 3 * PL;
    const double* sv2 = s + 4 * PL;
    const double* sq = s + 5 * PL;
    const int nx = I.nx;
    const size_t pl = (size_t)nx * I.ny;
    if (tid == 0) {
      s_rough = 0;
      if (j == 1 && t.tile == 0) I.magnext[0] = I.magnext[1] = I.magnext[2] = 0u;   // the last stage's update raises them
    }
    load_limits<SCHEME>(I, &lim_of, &s_lim, w, tid);
    if (needE && needB) {
      const double* fx[5] = {sq, sv1, sv2, su1, su2};
      const double* fy[5] = {sq, sv2, sv1, su1, su2};
      split_increments<SCHEME, TX, TY, 5>(fx, fy, ix, iy, tid);
      __syncthreads();
      split_interfaces<SCHEME, TX, TY, 3, 1>(ix, iy, nxs, nys, w, s_lim, &s_rough, tid);
    } else if (needE) {
      const double* fx[2] = {sq, sv1};
      const double* fy[2] = {sq, sv2};
      split_increments<SCHEME, TX, TY, 2>(fx, fy, ix, iy, tid);
      __syncthreads();
      split_interfaces<SCHEME, TX, TY, 1, -1>(ix, iy, nxs, nys, w, s_lim, &s_rough, tid);
    } else if (needB) {
      const double* fx[4] = {sv1, sv2, su1, su2};
      const double* fy[4] = {sv2, sv1, su1, su2};
      split_increments<SCHEME, TX, TY, 4>(fx, fy, ix, iy, tid);
      __syncthreads();
      split_interfaces<SCHEME, TX, TY, 2, 0>(ix, iy, nxs + NX, nys + NY, w, s_lim, &s_rough, tid);
    }
    __syncthreads();
    const bool any = s_rough != 0;
    const bool cell = threadIdx.z == 0 && t.x0 + tx < nx && t.y0 + ty < I.ny;   // not beyond the grid (ragged edge tile)
    const Coef<double>& K = I.k64;
    const double cx = K.cdx, cy = K.cdy;                // 1/(12 h)
    const int c = G::C00 + ty * BW + tx;
    const int fa = ty * (TX + 1) + tx, fb = ty * TX + tx;   // this cell's lower interfaces
    const size_t o = (size_t)(t.y0 + ty) * nx + (t.x0 + tx);
    double e1 = 0.0, e2 = 0.0;
    double gx = 0.0, gy = 0.0;
    if (needE) {
      const double dx = sq[c + 1] - sq[c - 1], dy = sq[c + BW] - sq[c - BW];
      if (any) {
        whole_pair<SCHEME, TX, TY, false>(sq, sv1, sq, sv2, scr, weno_eps, tid);
        gx = fd12<SCHEME>(dx, 6.0, nxs, fa, fa + 1, wx);
        gy = fd12<SCHEME>(dy, 6.0, nys, fb, fb + TX, wy);
      } else if (cell) {
        gx = fd12(dx, 6.0, nxs, fa, fa + 1);
        gy = fd12(dy, 6.0, nys, fb, fb + TX);
      }
    }
    if (cell && (needE || (need & NEED_DU))) {
      const double u1x = cd12s(su1 + c, 1), u2y = cd12s(su2 + c, BW);
      if (need & NEED_DU) reinterpret_cast<double*>(I.Du[j])[o] = fma(cx, u1x, cy * u2y);
      if (needE) {
        const double u2x = cd12(su2 + c, 1), u1y = cd12(su1 + c, BW);
        const double a1 = su1[c], a2 = su2[c];
        // (tau/4) (D0_y u2 - D0_x u1) + tau eps^2 D_x q - (u2^2 - u1^2)/2, and the second component
        e1 = fma(K.qcy, u2y, fma(-K.qcx, u1x, fma(0.5 * (a1 - a2), a1 + a2, K.tcx * gx)));
        e2 = fma(K.qcx, u2x, fma(K.qcy, u1y, fma(-a1, a2, K.tcy * gy)));
        double* e = reinterpret_cast<double*>(I.E[j]);
        e[o] = e1;
        e[o + pl] = e2;
      }
    }
    if (cell && (need & NEED_LTH)) {
      const double* f = sth + c;
      const double lx = fma(-30.0, f[0], fma(16.0, f[1] + f[-1], -(f[2] + f[-2])));
      const double ly = fma(-30.0, f[0], fma(16.0, f[BW] + f[-BW], -(f[2 * BW] + f[-2 * BW])));
      reinterpret_cast<double*>(I.Lth[j])[o] = fma(K.ldx, lx, K.ldy * ly);
    }
    if (needB) {
      double v1x = 0.0, v2y = 0.0, v2x = 0.0, v1y = 0.0;
      if (any) {
        __syncthreads();   // the fluxes of the pair before have been read
        whole_pair<SCHEME, TX, TY, true>(sv1, su1, sv2, su1, scr, weno_eps, tid);
        v1x = fd12<SCHEME>(sv1[c + 1] - sv1[c - 1], -6.0, nxs + NX, fa, fa + 1, wx);
        v2y = fd12<SCHEME>(sv2[c + BW] - sv2[c - BW], 6.0, nys + NY, fb, fb + TX, wy);
        __syncthreads();
        whole_pair<SCHEME, TX, TY, false>(sv2, su2, sv1, su2, scr, weno_eps, tid);
        v2x = fd12<SCHEME>(sv2[c + 1] - sv2[c - 1], 6.0, nxs + 2 * NX, fa, fa + 1, wx);
        v1y = fd12<SCHEME>(sv1[c + BW] - sv1[c - BW], 6.0, nys + 2 * NY, fb, fb + TX, wy);
      } else if (cell) {
        v1x = fd12(sv1[c + 1] - sv1[c - 1], -6.0, nxs + NX, fa, fa + 1);
        v2y = fd12(sv2[c + BW] - sv2[c - BW], 6.0, nys + NY, fb, fb + TX);
        v2x = fd12(sv2[c + 1] - sv2[c - 1], 6.0, nxs + 2 * NX, fa, fa + 1);
        v1y = fd12(sv1[c + BW] - sv1[c - BW], 6.0, nys + 2 * NY, fb, fb + TX);
      }
      if (cell) {
        // D_LF . B(v^(j)) + D_0 theta^(j), the only form later stages use them in
        double* db = reinterpret_cast<double*>(I.DLFB[j]);
        db[o] = fma(cx, v1x + cd12(sth + c, 1), cy * v2y);
        db[o + pl] = fma(cy, v1y + cd12(sth + c, BW), cx * v2x);
      }
    }
    if (cell && (need & NEED_V)) {
      double r1, r2;   // step 1 of stage i = j + 1 at this cell
      relax_v_cell<false, double>(b, I, j + 1, o, pl, j, e1, e2, sv1[c], sv2[c], r1, r2);
      double* vi = reinterpret_cast<double*>(I.Xs[j + 1]);
      vi[o + 3 * pl] = r1;
      vi[o + 4 * pl] = r2;
    }
  });
}

// k_update (stencil_kernels.cuh) with split fluxes.
template <int SCHEME, int TX, int TY>
__global__ void __launch_bounds__(SplitGeo<SCHEME, TX, TY>::G::NT, split_min_blocks<SCHEME, SplitGeo<SCHEME, TX, TY>::G::NT>()) k_update_split(const __grid_constant__ BatchDev b, int i, double weno_eps,
                                                                              int close_step, int form) {
  grid_dependency();
  using S = SplitGeo<SCHEME, TX, TY>;
  using G = typename S::G;
  constexpr int BW = G::BW, PL = G::PL, NX = G::NX, NY = G::NY;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ uint64_t bars[2];
  __shared__ SplitLimits s_lim;
  __shared__ const InstDev* lim_of;   // the instance s_lim is of
  __shared__ int s_rough;      // the tile holds a rough interface
  __shared__ unsigned s_mag[3];   // largest |u|, |v|, |q| that this block has closed of the instance of mag_of
  __shared__ unsigned* mag_of;
  const PlaneList pr = update_planes(b, i);
  double* stage = aligned_smem<double>(smem_raw);
  F2* ix = reinterpret_cast<F2*>(stage + pr.n * PL);
  F2* iy = ix + 4 * S::LIX;
  F2* nxs = reinterpret_cast<F2*>(stage + S::update_front(pr.n));   // [2][NX]: (-v1;p1), (v2;p2)
  F2* nys = nxs + 2 * NX;      // [2][NY]: (v2;p1), (v1;p2)
  double* scr = stage + 5 * PL;
  const double* wx = scr + S::WSCR;
  const double* wy = wx + NX;
  const int tx = threadIdx.x, ty = threadIdx.y, tid = tx + ty * TX + threadIdx.z * TX * TY;
  const F2 w = f2_of((SCHEME == WENO5_C4 ? 16.0 : 4.0) * weno_eps);
  const unsigned mwp = b.m_wp[i], mim = b.m_im[i];
  if (tid == 0) mag_of = nullptr;
  if (tid == 32) lim_of = nullptr;
  auto raise = [&]() {
    if (mag_of)
      for (int k = 0; k < 3; ++k) atomicMax(mag_of + k, s_mag[k]);
  };
  tile_loop<double, G, TX, TY, 1, true>(b, pr, stage, bars, tid, [&](const InstDev& I, const TileRef& t, double* s) {
    const double* sth = s;
    const double* sv1 = s + PL;
    const double* sv2 = s + 2 * PL;
    const int nx = I.nx;
    const size_t pl = (size_t)nx * I.ny;
    const Coef<double>& K = I.k64;
    if (tid == 0) {
      s_rough = 0;
      if (close_step && mag_of != I.magnext) {
        raise();
        mag_of = I.magnext;
        s_mag[0] = s_mag[1] = s_mag[2] = 0u;
      }
    }
    load_limits<SCHEME>(I, &lim_of, &s_lim, w, tid);
    // weights of the dissipation partner of D_LF . B(v^(i)), the explicit-weight predictor
    // (1/a_ii) sum_{j<i} (atilde_ij - a_ij) u^(j), as pairs (k32 and k32lo)
    F2 wt[APD_MAXS - 1];
    int nw = 0;
#pragma unroll
    for (int jj = 1; jj < APD_MAXS; ++jj)
      if (jj < i && has(mwp, jj)) {
        const F2 a = f2(I.k32.wp[i][jj], I.k32lo.wp[i][jj]);
        if (nw == 0) wt[0] = a; else if (nw == 1) wt[1] = a; else wt[2] = a;
        ++nw;
      }
    split_increments_update<SCHEME, TX, TY>(s, nw, wt, ix, iy, tid);
    __syncthreads();
    split_interfaces<SCHEME, TX, TY, 2, 0>(ix, iy, nxs, nys, w, s_lim, &s_rough, tid);
    __syncthreads();
    const bool any = s_rough != 0;
    const bool cell = threadIdx.z == 0 && t.x0 + tx < nx && t.y0 + ty < I.ny;   // not beyond the grid (ragged edge tile)
    const double cx = K.cdx, cy = K.cdy;
    const int c = G::C00 + ty * BW + tx;
    const int fa = ty * (TX + 1) + tx, fb = ty * TX + tx;
    const size_t o = (size_t)(t.y0 + ty) * nx + (t.x0 + tx);
    const double dv1 = sv1[c + 1] - sv1[c - 1], dv2 = sv2[c + BW] - sv2[c - BW];
    const double dv2x = sv2[c + 1] - sv2[c - 1], dv1y = sv1[c + BW] - sv1[c - BW];
    double v1x = 0.0, v2y = 0.0, v2x = 0.0, v1y = 0.0;
    if (any) {
      // the partner in FP64, in place of the staged planes 3 and 4
      double* p1 = s + 3 * PL;
      double* p2 = s + 4 * PL;
      for (int e = tid; e < BW * G::BH; e += G::NT) {
        double a1 = 0.0, a2 = 0.0;
        const double* u = p1 + e;
        for (int jj = 1; jj < i; ++jj)
          if (has(mwp, jj)) {
            a1 = fma(K.wp[i][jj], u[0], a1);
            a2 = fma(K.wp[i][jj], u[PL], a2);
            u += 2 * PL;
          }
        p1[e] = a1;
        p2[e] = a2;
      }
      __syncthreads();
      whole_pair<SCHEME, TX, TY, true>(sv1, p1, sv2, p1, scr, weno_eps, tid);
      v1x = fd12<SCHEME>(dv1, -6.0, nxs, fa, fa + 1, wx);
      v2y = fd12<SCHEME>(dv2, 6.0, nys, fb, fb + TX, wy);
      __syncthreads();
      whole_pair<SCHEME, TX, TY, false>(sv2, p2, sv1, p2, scr, weno_eps, tid);
      v2x = fd12<SCHEME>(dv2x, 6.0, nxs + NX, fa, fa + 1, wx);
      v1y = fd12<SCHEME>(dv1y, 6.0, nys + NY, fb, fb + TX, wy);
    } else if (cell) {
      v1x = fd12(dv1, -6.0, nxs, fa, fa + 1);
      v2y = fd12(dv2, 6.0, nys, fb, fb + TX);
      v2x = fd12(dv2x, 6.0, nxs + NX, fa, fa + 1);
      v1y = fd12(dv1y, 6.0, nys + NY, fb, fb + TX);
    }
    unsigned mu = 0u, mv = 0u, mq = 0u;
    if (cell) {
      const double dv1x = fma(8.0, dv1, sv1[c - 2] - sv1[c + 2]), dv2y = fma(8.0, dv2, sv2[c - 2 * BW] - sv2[c + 2 * BW]);
      const double dg1 = fma(cx, v1x + cd12(sth + c, 1), cy * v2y);    // D_LF . B(v^(i)) + D_0 theta^(i)
      const double dg2 = fma(cy, v1y + cd12(sth + c, BW), cx * v2x);
      const double dvi = fma(cx, dv1x, cy * dv2y);
      // step 3
      double s1 = K.aim[i][i] * dg1, s2 = K.aim[i][i] * dg2;
      for (int jj = 1; jj < i; ++jj) {
        if (has(mim, jj)) {
          const double* bg = reinterpret_cast<const double*>(I.DLFB[jj]);
          s1 = fma(K.aim[i][jj], bg[o], s1);
          s2 = fma(K.aim[i][jj], bg[o + pl], s2);
        }
      }
      const double* Xn = reinterpret_cast<const double*>(I.X);
      double* out = reinterpret_cast<double*>(I.Xs[i]);
      const double u1 = fma(-K.dt, s1, Xn[o]), u2 = fma(-K.dt, s2, Xn[o + pl]);
      if (!close_step) {
        out[o] = u1;
        out[o + pl] = u2;
        reinterpret_cast<double*>(I.Dv[i])[o] = dvi;   // D0 . v^(i) for the q steps of later stages
      }
      // step 4
      double qi = K.r_n[i] * Xn[o + 5 * pl];
      for (int jj = 1; jj <= i; ++jj) {
        if (!has(mim, jj)) continue;
        const double dv = (jj == i) ? dvi : reinterpret_cast<const double*>(I.Dv[jj])[o];
        qi = fma(K.rq_d[i][jj], dv, qi);
        if (jj < i) qi = fma(K.rv_v[i][jj], reinterpret_cast<const double*>(I.Xs[jj])[o + 5 * pl], qi);
      }
      if (!close_step) {
        out[o + 5 * pl] = qi;
      } else {
        const double m[6] = {u1, u2, sth[c], sv1[c], sv2[c], qi};
        if (close_step_cell<double>(I, o, pl, m, form, reinterpret_cast<double*>(I.Xnext))) atomicOr(b.err, 1u);
        field_max(m, mu, mv, mq);
      }
    }
    if (close_step) field_max_to(s_mag, mu, mv, mq, tid);
  });
  if (tid == 0) raise();
}

}  // namespace apd
