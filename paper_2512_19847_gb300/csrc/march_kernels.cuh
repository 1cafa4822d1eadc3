// The FP32 explicit and update kernels for large grids, by marching warps.
//
// A warp takes MARCH_OUT columns (its 32 lanes hold them and 3 halo columns on each side) and a
// segment of rows, and walks down the rows: the fluxes along y come from a register window of six
// rows, each interface evaluated once, those along x from the neighbouring lanes by shuffles.
// No shared memory, no barrier, no staged halo; a row is read once per warp (the 6 halo
// columns and rows again by the neighbours, from L1 and L2).  Same flux arithmetic as the
// tile kernels (w5_rec_f32, weno3, LF1); the narrower schemes keep the same window and columns.
//
// What bounds the tile kernels here (figures of WENO5) is the instruction issue (60 % active) and the latency
// of their phases: 1314 (explicit) and 1463 (update) thread instructions per cell, half of
// them not flux arithmetic (indices, staging, the runs' overlap).  2048^2, ms per step: explicit
// 0.359 -> 0.235, update 0.458 -> 0.254 (WENO3 0.399 -> 0.240 and 0.489 -> 0.224, LF1 0.261 -> 0.184 and
// 0.343 -> 0.199).  What the closed forms read beside the window is loaded at
// the head of a row, before its fluxes: with those loads where they are used (and their pointers
// read from the descriptor each row) 0.295 and 0.456.  Measured choices: explicit 3 blocks per SM
// and 3 rows per loop body 0.235 (1 row 0.240, 6 rows 0.273, 4 blocks 0.241, 5 blocks 0.39);
// update 4 blocks and 2 rows 0.253 (1 row 0.257, 3 blocks 0.28, 5 blocks 0.38).
#pragma once
#include "stencil_kernels.cuh"

namespace apd {

// Resident blocks per SM (128 threads: 3 take 168 registers, 4 take 128) and rows per loop body of the
// explicit and update kernels.
#ifndef APD_MARCH_MINB_E
#define APD_MARCH_MINB_E 3
#endif
#ifndef APD_MARCH_MINB_U
#define APD_MARCH_MINB_U 4
#endif
#ifndef APD_MARCH_UNROLL_E
#define APD_MARCH_UNROLL_E 3
#endif
#ifndef APD_MARCH_UNROLL_U
#define APD_MARCH_UNROLL_U 2
#endif
constexpr int kMarchUnrollE = APD_MARCH_UNROLL_E, kMarchUnrollU = APD_MARCH_UNROLL_U;
constexpr int MARCH_WARPS = 4, MARCH_THREADS = 32 * MARCH_WARPS;

struct MarchTask { int inst, x0, y0, y1; };

__device__ __forceinline__ MarchTask march_task(const BatchDev& b, int which, int task) {
  MarchTask t;
  t.inst = find_inst(b.march_start[which], b.counts[3], task);
  const InstDev& I = b.inst[t.inst];
  const int rows = b.counts[6 + which], groups = (I.nx + MARCH_OUT - 1) / MARCH_OUT;
  const int local = task - b.march_start[which][t.inst], s = local / groups;
  t.x0 = (local - s * groups) * MARCH_OUT;
  t.y0 = s * rows;
  t.y1 = min(t.y0 + rows, I.ny);
  return t;
}

constexpr unsigned MARCH_ALL = 0xffffffffu;
__device__ __forceinline__ float lane_up(float v, int k) { return __shfl_up_sync(MARCH_ALL, v, k); }
__device__ __forceinline__ float lane_dn(float v, int k) { return __shfl_down_sync(MARCH_ALL, v, k); }

// (13/3) (a - 2 b + c)^2 + 16 eps_W, as in w5_runs_item
__device__ __forceinline__ float march_curv(float a, float b, float c, float ew4) {
  const float d = fmaf(-2.f, b, a) + c;
  return fmaf(13.f / 3.f * d, d, ew4);
}

// One pair (g, U) along y, in the window's rows: its flux at the interface between rows 2 and 3.
// WENO5 carries the curvature terms, of g+ at rows 1, 2, 3 and of g- at rows 2, 3, 4, from row to row.
template <int SCHEME>
struct MarchPair {
  __device__ __forceinline__ void init(const float*, const float*, float) {}
  __device__ __forceinline__ void next(const float*, const float*, float) {}
  __device__ __forceinline__ float flux(const float* g, const float* u, float ew4) const {
    if (SCHEME == LF1_C2) return cell_lf1(g[2], g[3], u[2], u[3]);
    return add_rn(weno3<float>(g[1] + u[1], g[2] + u[2], g[3] + u[3], ew4), weno3<float>(g[4] - u[4], g[3] - u[3], g[2] - u[2], ew4));
  }
};
template <>
struct MarchPair<WENO5_C4> {
  float p[3], m[3];
  __device__ __forceinline__ void init(const float* g, const float* u, float ew4) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      p[k] = march_curv(g[k] + u[k], g[k + 1] + u[k + 1], g[k + 2] + u[k + 2], ew4);
      m[k] = march_curv(g[k + 1] - u[k + 1], g[k + 2] - u[k + 2], g[k + 3] - u[k + 3], ew4);
    }
  }
  // after the window has moved on by a row
  __device__ __forceinline__ void next(const float* g, const float* u, float ew4) {
    p[0] = p[1];
    p[1] = p[2];
    p[2] = march_curv(g[2] + u[2], g[3] + u[3], g[4] + u[4], ew4);
    m[0] = m[1];
    m[1] = m[2];
    m[2] = march_curv(g[3] - u[3], g[4] - u[4], g[5] - u[5], ew4);
  }
  __device__ __forceinline__ float flux(const float* g, const float* u, float) const {
    return w5_flux_f32(w5_rec_f32(g[0] + u[0], g[1] + u[1], g[2] + u[2], g[3] + u[3], g[4] + u[4], p[0], p[1], p[2]),
                       w5_rec_f32(g[5] - u[5], g[4] - u[4], g[3] - u[3], g[2] - u[2], g[1] - u[1], m[2], m[1], m[0]));
  }
};

// Difference of the x fluxes at this lane's cell (its right interface minus its left one).
template <int SCHEME>
__device__ __forceinline__ float march_dx(float g, float u, float ew4) {
  float f;
  if constexpr (SCHEME == LF1_C2) {
    f = cell_lf1(g, lane_dn(g, 1), u, lane_dn(u, 1));
  } else {
    const float P = g + u, M = g - u;
    const float pb = lane_up(P, 1), pd = lane_dn(P, 1), mc = lane_dn(M, 1), md = lane_dn(M, 2);
    if constexpr (SCHEME == WENO3_C4) {
      f = add_rn(weno3<float>(pb, P, pd, ew4), weno3<float>(md, mc, M, ew4));
    } else {
      const float pa = lane_up(P, 2), pe = lane_dn(P, 2);
      const float cp = march_curv(pb, P, pd, ew4);
      const float2 l = w5_rec_f32(pa, pb, P, pd, pe, lane_up(cp, 1), cp, lane_dn(cp, 1));
      const float ma = lane_up(M, 1), me = lane_dn(M, 3);
      const float cm = march_curv(ma, M, mc, ew4);
      f = w5_flux_f32(l, w5_rec_f32(me, md, mc, M, ma, lane_dn(cm, 2), lane_dn(cm, 1), cm));
    }
  }
  return f - lane_up(f, 1);
}

// The scheme's central differences along x (lanes) and along y (window rows 0 .. 4).
template <int SCHEME>
__device__ __forceinline__ float march_c1x(float a) {
  if (SCHEME == LF1_C2) return cell_c1<float, SCHEME>(0.f, lane_up(a, 1), lane_dn(a, 1), 0.f);
  return cell_c1<float, SCHEME>(lane_up(a, 2), lane_up(a, 1), lane_dn(a, 1), lane_dn(a, 2));
}
template <int SCHEME>
__device__ __forceinline__ float march_c1y(const float* w) { return cell_c1<float, SCHEME>(w[0], w[1], w[3], w[4]); }

__device__ __forceinline__ void march_push(float* w, float v) {
#pragma unroll
  for (int k = 0; k < 5; ++k) w[k] = w[k + 1];
  w[5] = v;
}

__device__ __forceinline__ int march_row(int r, int ny) { return r < 0 ? r + ny : (r >= ny ? r - ny : r); }

// The planes of earlier stages that a kernel's closed forms add at a cell, as (offset in floats from the
// state X, coefficient as a pair), collected once per task and loaded at the head of each row, before
// its fluxes, so that their latency is hidden.  MAXT: exact for the second-order tableau's stages, the
// most any tableau has otherwise (GENERIC: n of them, tested per term).
template <int MAXT, bool GENERIC>
struct MarchTerms {
  static constexpr int M = MAXT > 0 ? MAXT : 1;
  int off[M], n = 0;
  float c[M], lo[M];
  __device__ __forceinline__ MarchTerms() {
#pragma unroll
    for (int k = 0; k < M; ++k) {
      off[k] = 0;
      c[k] = lo[k] = 0.f;
    }
  }
  __device__ __forceinline__ void add(const void* base, const void* p, float cc, float ll) {
    const int d = (int)(reinterpret_cast<const float*>(p) - reinterpret_cast<const float*>(base));
#pragma unroll
    for (int k = 0; k < MAXT; ++k)
      if (k == n) {
        off[k] = d;
        c[k] = cc;
        lo[k] = ll;
      }
    ++n;
  }
  __device__ __forceinline__ bool on(int k) const { return !GENERIC || k < n; }
};

// ---------------------------------------------------------------------------
// k_explicit (stencil_kernels.cuh) for stage j; E and B: whether its E^(j) and its
// D_LF . B(v^(j)) + D_0 theta^(j) are needed; NT: terms of v^(j+1) read from memory
// (v^n and the earlier stages' E and v; 5: up to that many).
template <int SCHEME, bool E, bool B, int NT>
__global__ void __launch_bounds__(MARCH_THREADS, APD_MARCH_MINB_E) k_explicit_march(const __grid_constant__ BatchDev b, int j, unsigned need,
                                                                                  double weno_eps) {
  grid_dependency();
  const int lane = threadIdx.x & 31;
  const int ntasks = b.march_start[0][b.counts[3]];
  const float ew4 = (SCHEME == WENO5_C4 ? 16.f : 4.f) * float(weno_eps);   // of the doubled split
  const int i = j + 1;
  const bool curE = has(b.m_ex[i], j), curV = has(b.m_im[i], j);
  for (int task = blockIdx.x * MARCH_WARPS + (threadIdx.x >> 5); task < ntasks; task += gridDim.x * MARCH_WARPS) {
    const MarchTask t = march_task(b, 0, task);
    const InstDev& I = b.inst[t.inst];
    const Coef<float>& K = I.k32;
    const int nx = I.nx, ny = I.ny;
    const int pl = nx * ny;
    const int xs = t.x0 + lane - 3;
    const int x = xs < 0 ? xs + nx : xs % nx;
    const bool out = lane >= 3 && lane < 3 + MARCH_OUT && xs < nx;
    const float* X = reinterpret_cast<const float*>(I.Xs[j]);
    const float* base = reinterpret_cast<const float*>(I.X);
    const float cx = c1_scale<SCHEME>(K.inv_dx, K.cdx), cy = c1_scale<SCHEME>(K.inv_dy, K.cdy);
    const float fx = flux_scale<float, SCHEME>(K.inv_dx), fy = flux_scale<float, SCHEME>(K.inv_dy);
    const float qt = K.qtau, te2 = K.te2;
    MarchTerms<NT, (NT > 2)> tm;
    tm.add(base, base + 3 * (size_t)pl, K.r_n[i], I.k32lo.r_n[i]);
    for (int jj = 1; jj < j; ++jj) {
      if (has(b.m_ex[i], jj)) tm.add(base, I.E[jj], K.rv_e[i][jj], I.k32lo.rv_e[i][jj]);
      if (has(b.m_im[i], jj)) tm.add(base, reinterpret_cast<const float*>(I.Xs[jj]) + 3 * (size_t)pl, K.rv_v[i][jj], I.k32lo.rv_v[i][jj]);
    }
    const float ce = K.rv_e[i][j], cel = I.k32lo.rv_e[i][j], cv = K.rv_v[i][j], cvl = I.k32lo.rv_v[i][j];
    const bool pairs = I.relax64 != 0;
    float* oE = reinterpret_cast<float*>(I.E[j]);
    float* oDu = reinterpret_cast<float*>(I.Du[j]);
    float* oL = reinterpret_cast<float*>(I.Lth[j]);
    float* oB = reinterpret_cast<float*>(I.DLFB[j]);
    float* oV = reinterpret_cast<float*>(I.Xs[i]) + 3 * (size_t)pl;
    float u1[6], u2[6], th[6], v1[6], v2[6], q[6];   // rows r - 2 .. r + 3
    auto load = [&](int row, float& a, float& bb, float& c, float& d, float& e, float& f) {
      const float* p = X + (size_t)(march_row(row, ny) * nx + x);
      a = p[0];
      bb = p[pl];
      if (B || (need & NEED_LTH)) c = p[2 * (size_t)pl];
      d = p[3 * (size_t)pl];
      e = p[4 * (size_t)pl];
      if (E) f = p[5 * (size_t)pl];
    };
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      th[k] = q[k] = 0.f;
      load(t.y0 - 3 + k, u1[k], u2[k], th[k], v1[k], v2[k], q[k]);
    }
    MarchPair<SCHEME> a, bu, bv;   // along y: (q;v2), (v2;u1), (v1;u2)
    if (E) a.init(q, v2, ew4);
    if (B) {
      bu.init(v2, u1, ew4);
      bv.init(v1, u2, ew4);
    }
    float fq = 0.f, fu = 0.f, fv = 0.f;   // the fluxes of the interface below row r
#pragma unroll kMarchUnrollE
    for (int r = t.y0 - 1; r < t.y1; ++r) {
      float nu1 = 0.f, nu2 = 0.f, nth = 0.f, nv1 = 0.f, nv2 = 0.f, nq = 0.f;
      const bool more = r + 1 < t.y1, put = out && r >= t.y0;
      if (more) load(r + 4, nu1, nu2, nth, nv1, nv2, nq);
      const int o = r * nx + x;
      float x1[MarchTerms<NT, (NT > 2)>::M], x2[MarchTerms<NT, (NT > 2)>::M];
#pragma unroll
      for (int k = 0; k < NT; ++k) {
        x1[k] = x2[k] = 0.f;
        if (put && tm.on(k)) {
          const float* p = base + (ptrdiff_t)(tm.off[k] + o);
          x1[k] = p[0];
          x2[k] = p[pl];
        }
      }
      const float gq = E ? a.flux(q, v2, ew4) : 0.f, gu = B ? bu.flux(v2, u1, ew4) : 0.f, gv = B ? bv.flux(v1, u2, ew4) : 0.f;
      if (r >= t.y0) {
        float e1 = 0.f, e2 = 0.f;
        const float u1x = march_c1x<SCHEME>(u1[2]), u2y = march_c1y<SCHEME>(u2);
        if ((need & NEED_DU) && out) oDu[o] = cell_sum(cx, u1x, cy, u2y);
        if (E) {
          const float u2x = march_c1x<SCHEME>(u2[2]), u1y = march_c1y<SCHEME>(u1);
          const float g1 = march_dx<SCHEME>(q[2], v1[2], ew4) * fx, g2 = (gq - fq) * fy;
          cell_e<float>(qt, te2, cx, cy, u1x, u2y, u2x, u1y, g1, g2, u1[2], u2[2], e1, e2);
          if (out) {
            oE[o] = e1;
            oE[o + (size_t)pl] = e2;
          }
        }
        if (need & NEED_LTH) {
          const float lx = cell_c2<float, SCHEME>(lane_up(th[2], 2), lane_up(th[2], 1), th[2], lane_dn(th[2], 1), lane_dn(th[2], 2));
          const float ly = cell_c2<float, SCHEME>(th[0], th[1], th[2], th[3], th[4]);
          if (out) oL[o] = cell_sum(d2_scale<float, SCHEME>(K.inv_dx), lx, d2_scale<float, SCHEME>(K.inv_dy), ly);
        }
        if (B) {
          const float d1 = cell_sum(march_dx<SCHEME>(-v1[2], u1[2], ew4), fx, gu - fu, fy);
          const float d2 = cell_sum(march_dx<SCHEME>(v2[2], u2[2], ew4), fx, gv - fv, fy);
          const float t1 = march_c1x<SCHEME>(th[2]), t2 = march_c1y<SCHEME>(th);
          if (out) {
            oB[o] = fmaf(cx, t1, d1);
            oB[o + (size_t)pl] = fmaf(cy, t2, d2);
          }
        }
        if ((need & NEED_V) && out) {   // step 1 of stage j + 1
          auto step1 = [&](auto s1, auto s2) {
            s1.start(tm.c[0], tm.lo[0], x1[0]);
            s2.start(tm.c[0], tm.lo[0], x2[0]);
#pragma unroll
            for (int k = 1; k < NT; ++k)
              if (tm.on(k)) {
                s1.add(tm.c[k], tm.lo[k], x1[k]);
                s2.add(tm.c[k], tm.lo[k], x2[k]);
              }
            if (curE) {
              s1.add(ce, cel, e1);
              s2.add(ce, cel, e2);
            }
            if (curV) {
              s1.add(cv, cvl, v1[2]);
              s2.add(cv, cvl, v2[2]);
            }
            oV[o] = s1.value();
            oV[o + (size_t)pl] = s2.value();
          };
          if (pairs) step1(RelaxSum<true, float>(), RelaxSum<true, float>());
          else step1(RelaxSum<false, float>(), RelaxSum<false, float>());
        }
      }
      fq = gq;
      fu = gu;
      fv = gv;
      march_push(u1, nu1);
      march_push(u2, nu2);
      march_push(th, nth);
      march_push(v1, nv1);
      march_push(v2, nv2);
      march_push(q, nq);
      if (E) a.next(q, v2, ew4);
      if (B) {
        bu.next(v2, u1, ew4);
        bv.next(v1, u2, ew4);
      }
    }
  }
}

// ---------------------------------------------------------------------------
// k_update (stencil_kernels.cuh) for stage i.  NW: stages in the dissipation partner, NT: earlier
// stages in the sums of steps 3 and 4 (NT = 3: up to NW and NT of them).
template <int SCHEME, int NW, int NT>
__global__ void __launch_bounds__(MARCH_THREADS, APD_MARCH_MINB_U) k_update_march(const __grid_constant__ BatchDev b, int i, double weno_eps,
                                                                                int close_step, int form) {
  grid_dependency();
  constexpr bool GEN = NT == 3;
  constexpr int MT = NT > 0 ? NT : 1;
  const int lane = threadIdx.x & 31;
  const int ntasks = b.march_start[1][b.counts[3]];
  const float ew4 = (SCHEME == WENO5_C4 ? 16.f : 4.f) * float(weno_eps);   // of the doubled split
  const unsigned mwp = b.m_wp[i], mim = b.m_im[i];
  for (int task = blockIdx.x * MARCH_WARPS + (threadIdx.x >> 5); task < ntasks; task += gridDim.x * MARCH_WARPS) {
    const MarchTask t = march_task(b, 1, task);
    const InstDev& I = b.inst[t.inst];
    const Coef<float>& K = I.k32;
    const int nx = I.nx, ny = I.ny;
    const int pl = nx * ny;
    const int xs = t.x0 + lane - 3;
    const int x = xs < 0 ? xs + nx : xs % nx;
    const bool out = lane >= 3 && lane < 3 + MARCH_OUT && xs < nx;
    const float cx = c1_scale<SCHEME>(K.inv_dx, K.cdx), cy = c1_scale<SCHEME>(K.inv_dy, K.cdy);
    const float fx = flux_scale<float, SCHEME>(K.inv_dx), fy = flux_scale<float, SCHEME>(K.inv_dy);
    const float dt = K.dt, aii = K.aim[i][i], rn = K.r_n[i], rnl = I.k32lo.r_n[i], rd = K.rq_d[i][i], rdl = I.k32lo.rq_d[i][i];
    const bool pairs = I.relax64 != 0;
    float* Xi = reinterpret_cast<float*>(I.Xs[i]);
    float* oD = reinterpret_cast<float*>(I.Dv[i]);
    const float* base = reinterpret_cast<const float*>(I.X);
    MarchTerms<NW, GEN> pw;                      // dissipation partner: u1, u2 planes and weights
    MarchTerms<NT, GEN> ts, td, tq;              // D_LF . B(v) + D_0 theta (2 planes), D0 . v and q of the earlier stages
    for (int jj = 1; jj < i; ++jj) {
      if (has(mwp, jj)) pw.add(base, I.Xs[jj], K.wp[i][jj], 0.f);
      if (NT > 0 && has(mim, jj)) {
        ts.add(base, I.DLFB[jj], K.aim[i][jj], 0.f);
        td.add(base, I.Dv[jj], K.rq_d[i][jj], I.k32lo.rq_d[i][jj]);
        tq.add(base, reinterpret_cast<const float*>(I.Xs[jj]) + 5 * (size_t)pl, K.rv_v[i][jj], I.k32lo.rv_v[i][jj]);
      }
    }
    float th[6], v1[6], v2[6], p1[6], p2[6];   // rows r - 2 .. r + 3
    auto load = [&](int row, float& c, float& d, float& e, float* f, float* g) {
      const int o = march_row(row, ny) * nx + x;
      const float* p = Xi + (size_t)o;
      c = p[2 * (size_t)pl];
      d = p[3 * (size_t)pl];
      e = p[4 * (size_t)pl];
#pragma unroll
      for (int k = 0; k < NW; ++k) {
        f[k] = g[k] = 0.f;
        if (pw.on(k)) {
          const float* u = base + (ptrdiff_t)(pw.off[k] + o);
          f[k] = u[0];
          g[k] = u[pl];
        }
      }
    };
    auto partner = [&](const float* f) {
      float s = 0.f;
#pragma unroll
      for (int k = 0; k < NW; ++k)
        if (pw.on(k)) s = fmaf(pw.c[k], f[k], s);
      return s;
    };
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      float f[NW], g[NW];
      load(t.y0 - 3 + k, th[k], v1[k], v2[k], f, g);
      p1[k] = partner(f);
      p2[k] = partner(g);
    }
    MarchPair<SCHEME> a, c;   // along y: (v2;p1), (v1;p2)
    a.init(v2, p1, ew4);
    c.init(v1, p2, ew4);
    float fa = 0.f, fc = 0.f;
#pragma unroll kMarchUnrollU
    for (int r = t.y0 - 1; r < t.y1; ++r) {
      float nth = 0.f, nv1 = 0.f, nv2 = 0.f, nf[NW], ng[NW];
#pragma unroll
      for (int k = 0; k < NW; ++k) nf[k] = ng[k] = 0.f;
      const bool more = r + 1 < t.y1, put = out && r >= t.y0;
      if (more) load(r + 4, nth, nv1, nv2, nf, ng);
      const int o = r * nx + x;
      float n1 = 0.f, n2 = 0.f, n3 = 0.f, b1[MT], b2[MT], xd[MT], xq[MT];
#pragma unroll
      for (int k = 0; k < NT; ++k) b1[k] = b2[k] = xd[k] = xq[k] = 0.f;
      if (put) {
        n1 = base[o];
        n2 = base[o + (size_t)pl];
        n3 = base[o + 5 * (size_t)pl];
#pragma unroll
        for (int k = 0; k < NT; ++k)
          if (ts.on(k)) {
            const float* p = base + (ptrdiff_t)(ts.off[k] + o);
            b1[k] = p[0];
            b2[k] = p[pl];
            xd[k] = base[(ptrdiff_t)(td.off[k] + o)];
            xq[k] = base[(ptrdiff_t)(tq.off[k] + o)];
          }
      }
      const float ga = a.flux(v2, p1, ew4), gc = c.flux(v1, p2, ew4);
      if (r >= t.y0) {
        const float d1 = cell_sum(march_dx<SCHEME>(-v1[2], p1[2], ew4), fx, ga - fa, fy);
        const float d2 = cell_sum(march_dx<SCHEME>(v2[2], p2[2], ew4), fx, gc - fc, fy);
        const float t1 = march_c1x<SCHEME>(th[2]), t2 = march_c1y<SCHEME>(th);
        const float dvi = cell_sum(cx, march_c1x<SCHEME>(v1[2]), cy, march_c1y<SCHEME>(v2));
        if (out) {
          // step 3
          float s1 = 0.f, s2 = 0.f;
#pragma unroll
          for (int k = 0; k < NT; ++k)
            if (ts.on(k)) {
              s1 = fmaf(ts.c[k], b1[k], s1);
              s2 = fmaf(ts.c[k], b2[k], s2);
            }
          s1 = fmaf(aii, fmaf(cx, t1, d1), s1);
          s2 = fmaf(aii, fmaf(cy, t2, d2), s2);
          const float w1 = fmaf(-dt, s1, n1), w2 = fmaf(-dt, s2, n2);
          // step 4
          auto step4 = [&](auto sum) {
            sum.start(rn, rnl, n3);
#pragma unroll
            for (int k = 0; k < NT; ++k)
              if (td.on(k)) {
                sum.add(td.c[k], td.lo[k], xd[k]);
                sum.add(tq.c[k], tq.lo[k], xq[k]);
              }
            sum.add(rd, rdl, dvi);
            return sum.value();
          };
          const float qi = pairs ? step4(RelaxSum<true, float>()) : step4(RelaxSum<false, float>());
          if (!close_step) {
            Xi[o] = w1;
            Xi[o + (size_t)pl] = w2;
            oD[o] = dvi;   // D0 . v^(i) for the q steps of later stages
            Xi[o + 5 * (size_t)pl] = qi;
          } else {
            const float m[6] = {w1, w2, th[2], v1[2], v2[2], qi};
            if (close_step_cell<float>(I, o, pl, m, form, reinterpret_cast<float*>(I.Xnext))) atomicOr(b.err, 1u);
          }
        }
      }
      fa = ga;
      fc = gc;
      march_push(th, nth);
      march_push(v1, nv1);
      march_push(v2, nv2);
      march_push(p1, partner(nf));
      march_push(p2, partner(ng));
      a.next(v2, p1, ew4);
      c.next(v1, p2, ew4);
    }
  }
}

}  // namespace apd
