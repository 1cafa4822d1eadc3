// The launch sequence of one IMEX step (Algorithm 1, CK/ARS tableau with
// stage 1 = X^n, GSA close), shared by the handle path and the
// no-allocation entry point.
#pragma once
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdlib>

#include "../../include/ap_dvm.h"
#include "common.cuh"
#include "dispatch.h"

namespace apd {

enum KernelKind { KK_EXPLICIT, KK_RHS, KK_ROWS_FWD, KK_COLS, KK_ROWS_INV, KK_UPDATE, KK_FINISH, KK_STAGE1 };

// Kinds of stencil work a batch holds (bits of StepKernels::stencil_kinds): instances taken by the tile
// kernels with whole fluxes, those with split fluxes (FP64, split_flux.cuh), and those taken by the
// marching kernels (FP32, march_kernels.cuh).
enum StencilKinds { STENCIL_WHOLE = 1, STENCIL_SPLIT = 2, STENCIL_MARCH = 4 };

// Kinds of Helmholtz transform work a batch holds (bits of StepKernels::fft_kinds).
enum FftKinds { FFT_X_POW2 = 1, FFT_X_BS = 2, FFT_Y_POW2 = 4, FFT_Y_BS = 8 };

// Transform launches of one implicit stage for the given kinds.
inline int fft_launches(unsigned kinds) {
  return 2 * (((kinds & FFT_X_POW2) ? 1 : 0) + ((kinds & FFT_X_BS) ? 1 : 0)) + ((kinds & FFT_Y_POW2) ? 1 : 0) +
         ((kinds & FFT_Y_BS) ? 1 : 0);
}

struct StepKernels {
  StencilSet ks;
  MiscSet km;
  int g_explicit, g_rhs, g_update, g_finish, g_fft, g_cols, cols_threads;
  size_t fft_smem, cols_smem;   // the power-of-two column pass has its own (wider) work items
  size_t smem_update;
  unsigned fft_kinds;   // FftKinds present among the attached solves
  int g_rows;           // grid of the power-of-two row passes (km.rows_threads threads per block)
  unsigned stencil_kinds = STENCIL_WHOLE;   // StencilKinds present among the attached solves
  int g_explicit_split = 0, g_update_split = 0;
  size_t smem_update_split = 0;
  int g_explicit_march = 0, g_update_march = 0;
};

// Planes k_update stages at its largest stage: theta, v1, v2 and u1, u2 of every
// earlier stage entering the dissipation partner (the explicit-weight predictor
// (1/a_ii) sum_{j<i} (atilde_ij - a_ij) u^(j)).
inline int update_planes_max(const ap_dvm_params& t) {
  int best = 0;
  for (int i = 1; i <= t.s; ++i) {
    int np = 3;
    for (int j = 1; j < i; ++j)
      if (t.A_ex[(i - 1) * AP_DVM_MAX_STAGES + (j - 1)] - t.A_im[(i - 1) * AP_DVM_MAX_STAGES + (j - 1)] != 0.0) np += 2;
    if (np > best) best = np;
  }
  return best;
}

// Shared memory of the transform kernels: every pass of a batch takes work items of
// at most eblk complex values (eblk_cols for the power-of-two column pass), padded in
// the power-of-two kernels (one spare value per 16 FP32 or 8 FP64 complex values).
inline size_t fft_block_bytes(int elems, bool f32) {
  const int ps = f32 ? 4 : 3;
  return (size_t)(elems + (elems >> ps) + 1) * (f32 ? 8 : 16);
}
// Complex values per work item: rows and the other-length kernels eblk (at least
// one transform of the longest length), the power-of-two column pass a few
// adjacent columns (coalesced loads): 8192 values (64 KB) in FP32, 4096 in FP64.
inline int fft_eblk(int nmax) { return nmax > 2048 ? nmax : 2048; }
inline int fft_eblk_cols(int nmax, bool f32) {
  const int e = f32 ? 8192 : 4096;
  return nmax > e ? nmax : e;
}

inline size_t update_smem_split(const StencilSet& ks, const ap_dvm_params& t) {
  return ks.smem_update_split(update_planes_max(t));
}

// Whether the fluxes of a solve are split (split_flux.cuh): FP64 with a WENO scheme and at least
// kSplitMinCells cells on each side.  Where its data are rough, the split kernels themselves fall back on the
// whole form; the line keeps grids that are rough all over off them.
// Why the line lies there: the pairs of floats round second and third differences to about 2^-47 of
// the increments, FP64 rounds the whole flux to 2^-52 of its own size.  For fields of wavenumbers up
// to 16 (the workloads') the rms error of a flux difference against 113-bit arithmetic, split and
// whole, in units of 1e-17: WENO5 at 2048 cells a side 0.4 and 5.3, 512: 1.6 and 5.3, 256: 3.2 and
// 5.3, 128: 9.2 and 5.4; WENO3 at 512: 1.9 and 5.3, 256: 6.0 and 5.5, 128: 21 and 5.7 (WENO3's meet near 300
// cells for these fields; the layers it is run on, smooth along x, stay below to 256: a fifth of the whole form's).
// Whole steps against 64-bit-mantissa arithmetic (relative; u1, theta, v1): 512^2 Taylor-Green 0.90e-16, 8.5e-15,
// 1.30e-16 split, 1.15e-16, 7.0e-15, 1.43e-16 whole; 256^2 WENO3 layer 0.93e-16, 4.6e-15, 1.7e-16 and
// 1.55e-16, 3.3e-15, 2.5e-16; 256^2 random field, WENO5 1.19e-16, 3.6e-15, 2.7e-16 and 1.15e-16, 2.9e-15,
// 2.8e-16, WENO3 1.69e-16, 3.3e-15, 2.9e-16 and 1.43e-16, 3.1e-15, 2.9e-16; 300^2 WENO3 1.46e-16, 2.7e-15, 1.7e-16
// and 1.44e-16, 2.7e-15, 1.7e-16.  (Theta's is the sum of a few low modes' roundings: it varies by a third
// with the draw, for both forms alike.)
constexpr int kSplitMinCells = 256;
inline bool split_fluxes(const ap_dvm_params& p) {
  return p.precision == AP_DVM_FP64 && p.space_scheme != AP_DVM_LF1_C2 && p.nx >= kSplitMinCells && p.ny >= kSplitMinCells;
}

// Whether a solve is taken by the marching kernels: FP32, a width that does not leave over a quarter of
// their warps' columns (26 each) beyond the grid, and enough cells, of its own or of its batch, for
// these warps to fill the chip.  Explicit + update, us per step, marching against tiles: WENO5 256^2 54
// and 45, 384^2 58 and 61, 512^2 66 and 78, 1024^2 147 and 216, 2048^2 477 and 774; WENO3 56 and 51, 59
// and 68, 66 and 85, 141 and 240, 464 and 888; LF1 47 and 41, 49 and 55, 52 and 65, 110 and 169, 383 and
// 605.  24 uneven solves of 64 to 512 cells a side, 5 steps: 3.01 ms against 3.23 with those below
// 384^2 by tiles.  Both kinds give the same bits
// (cell_c1 and what follows it in stencil_kernels.cuh), so that a batch does not change a solve's result.
constexpr long long kMarchMinCells = 384LL * 384, kMarchMinBatchCells = 2 * kMarchMinCells;
inline bool march_wide(const ap_dvm_params& p) {
  const int covered = (p.nx + MARCH_OUT - 1) / MARCH_OUT * MARCH_OUT;
  return p.precision != AP_DVM_FP64 && 4LL * covered <= 5LL * p.nx;
}
inline unsigned stencil_kind(const ap_dvm_params& p, bool march_all) {
  if (split_fluxes(p)) return STENCIL_SPLIT;
  return march_wide(p) && (march_all || (long long)p.nx * p.ny >= kMarchMinCells) ? STENCIL_MARCH : STENCIL_WHOLE;
}
inline int march_tasks(int nx, int ny, int rows) { return ((nx + MARCH_OUT - 1) / MARCH_OUT) * ((ny + rows - 1) / rows); }

inline size_t update_smem(const StencilSet& ks, const ap_dvm_params& t) {
  return ks.update_fixed + (size_t)ks.nbuf * update_planes_max(t) * ks.plane_bytes;
}

// Tensor maps of the stage buffers of one instance for TMA staging: map j
// (j = 1: the state X, j >= 2: X^(j)) describes 6 planes of nx x ny values as a
// 3D tensor (x, y, plane) with a box of bw x bh x 1.  Writes s+1 maps to out
// (64-byte aligned) and returns 1, or 0 when TMA is not used for this
// instance (grid smaller than the box, no driver entry point, or the
// environment variable AP_DVM_NO_TMA set).
inline int encode_stage_maps(const ap_dvm_params& p, const InstDev& d, int bw, int bh, CUtensorMap* out) {
  if (std::getenv("AP_DVM_NO_TMA")) return 0;
  if (p.nx < bw || p.ny < bh) return 0;
  // a tensor map's row stride must be a multiple of 16 bytes: other widths stage with plain loads
  if ((size_t)p.nx * (p.precision == AP_DVM_FP64 ? 8 : 4) % 16 != 0) return 0;
  static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
  if (!encode) {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess || !fn)
      return 0;
    encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
  }
  const bool f64 = p.precision == AP_DVM_FP64;
  const size_t es = f64 ? 8 : 4;
  const cuuint64_t dims[3] = {(cuuint64_t)p.nx, (cuuint64_t)p.ny, 6};
  const cuuint64_t strides[2] = {(cuuint64_t)p.nx * es, (cuuint64_t)p.nx * p.ny * es};
  const cuuint32_t box[3] = {(cuuint32_t)bw, (cuuint32_t)bh, 1};
  const cuuint32_t estr[3] = {1, 1, 1};
  for (int j = 1; j <= p.s; ++j) {
    void* base = d.Xs[j];
    const CUresult r = encode(&out[j], f64 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT64 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, base, dims,
                              strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                              CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return 0;
  }
  return 1;
}

// Launch of a kernel of a step as a programmatic dependent of the work before it on the stream
// (grid_dependency in common.cuh): the launch's own latency then overlaps the end of that work.  Taken
// by single solves of at most kDependentMaxCells cells, whose kernels run for a few microseconds
// each: 64^2 FP64, 10 steps, 2.15 -> 1.88 ms, 384x192 LF1 1.115 -> 0.936, 509x251 FP32 0.665 ->
// 0.565, 512^2 FP64 1.96 -> 1.88, 1000^2 FP64 3.13 -> 3.08; beyond, it costs 0.2-0.7 % (2048^2 FP64
// 5.85 -> 5.87, 24 uneven FP32 solves 4.67 -> 4.70).
constexpr long long kDependentMaxCells = 3LL << 19;
inline cudaError_t launch_dependent(const void* fn, int grid, dim3 block, size_t smem, void** args, cudaStream_t stream) {
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelExC(&cfg, fn, args);
}

// launch(fn, grid, block, smem, args, kind) -> int status (0 = success); form = the precision form
// (AP_DVM_FP64, AP_DVM_FP32_DEV, AP_DVM_FP32_DEV_TH), passed to the finish kernel
// fused: the last stage's update closes the step into the other state buffer
// (I.Xnext; the handle path's double-buffered state), else a finish kernel
// closes it in place.
template <class Launch>
int enqueue_imex_step(const ap_dvm_params& t, const StepKernels& K, const BatchDev& batch, int form, Launch&& launch,
                      bool fused = false) {
  const int s = t.s;
  void* bp = const_cast<BatchDev*>(&batch);   // copied into each launch's parameters
  const dim3 blk(K.ks.tx, K.ks.ty, K.ks.tz), cells(K.ks.tx, K.ks.ty);
  double weno_eps = t.weno_eps;
  int st;
  auto AEX = [&](int i, int j) { return t.A_ex[(i - 1) * AP_DVM_MAX_STAGES + (j - 1)]; };
  auto AIM = [&](int i, int j) { return t.A_im[(i - 1) * AP_DVM_MAX_STAGES + (j - 1)]; };
  // type-A tableaux (a_11 != 0) compute stage 1 with the four steps; CK/ARS take X^(1) = X^n
  const bool type_a = AIM(1, 1) != 0.0;
  if (type_a) {
    int c4 = t.space_scheme != AP_DVM_LF1_C2;
    void* a[] = {bp, &c4};
    if ((st = launch(K.km.k_stage1, K.g_finish, cells, 0, a, KK_STAGE1))) return st;
  }
  for (int i = type_a ? 1 : 2; i <= s; ++i) {
    int j = i - 1;
    unsigned need = 32u;                                   // v^(i), step 1 of stage i
    for (int k = j + 1; k <= s; ++k) {
      if (AEX(k, j) != 0.0) need |= 1u;                    // E^(j)
      if (AIM(k, j) != 0.0) need |= 2u | 4u | 16u;        // D0.u, D_Delta theta, D_LF.B(v) + D0 theta of stage j
    }
    if (j == 1 && !type_a) need |= 2u;                     // D0 . u^n (= D0 . u^(1)) enters every right-hand side
    if (j >= 1) {
      void* a[] = {bp, &j, &need, &weno_eps};
      if ((K.stencil_kinds & STENCIL_WHOLE) && (st = launch(K.ks.k_explicit, K.g_explicit, blk, K.ks.smem_explicit, a, KK_EXPLICIT))) return st;
      if ((K.stencil_kinds & STENCIL_SPLIT) &&
          (st = launch(K.ks.k_explicit_split, K.g_explicit_split, blk, K.ks.smem_explicit_split, a, KK_EXPLICIT)))
        return st;
      if (K.stencil_kinds & STENCIL_MARCH) {
        int terms = 1;   // of v^(i): v^n and the stages before j
        for (int k = 1; k < j; ++k) terms += (AEX(i, k) != 0.0) + (AIM(i, k) != 0.0);
        const void* fn = K.ks.k_explicit_march[std::min(terms, 3) - 1][(need & 1u) | ((need & 16u) >> 3)];
        if ((st = launch(fn, K.g_explicit_march, dim3(K.ks.march_threads), 0, a, KK_EXPLICIT))) return st;
      }
    }
    double sign = -1.0;   // theta-history term with a minus sign (the stage equations of Sec. 3.1)
    int first = (i == (type_a ? 1 : 2)) ? 1 : 0;           // the first right-hand side also sums theta^n
    {
      void* a[] = {bp, &i, &sign, &first};
      int terms = 1;   // D_0 . u^n, and three planes of every earlier stage with a_ij
      for (int k = 1; k < i; ++k) terms += AIM(i, k) != 0.0 ? 3 : 0;
      const void* fn = K.ks.k_rhs[terms == 1 ? 0 : (terms == 4 ? 1 : 2)];
      if ((st = launch(fn, K.g_rhs, dim3(K.ks.rhs_threads), 0, a, KK_RHS))) return st;
    }
    {
      // each pass: the power-of-two kernel and/or the Bluestein kernel, as the batch needs
      void* a[] = {bp};
      void* b[] = {bp, &i};
      const unsigned kk = K.fft_kinds;
      if ((kk & FFT_X_POW2) && (st = launch(K.km.k_rows_fwd, K.g_rows, dim3(K.km.rows_threads), K.fft_smem, a, KK_ROWS_FWD))) return st;
      if ((kk & FFT_X_BS) && (st = launch(K.km.k_rows_fwd_bs, K.g_fft, dim3(256), K.fft_smem, a, KK_ROWS_FWD))) return st;
      if ((kk & FFT_Y_POW2) && (st = launch(K.km.k_cols, K.g_cols, dim3(K.cols_threads), K.cols_smem, b, KK_COLS))) return st;
      if ((kk & FFT_Y_BS) && (st = launch(K.km.k_cols_bs, K.g_fft, dim3(256), K.fft_smem, b, KK_COLS))) return st;
      if ((kk & FFT_X_POW2) && (st = launch(K.km.k_rows_inv, K.g_rows, dim3(K.km.rows_threads), K.fft_smem, b, KK_ROWS_INV))) return st;
      if ((kk & FFT_X_BS) && (st = launch(K.km.k_rows_inv_bs, K.g_fft, dim3(256), K.fft_smem, b, KK_ROWS_INV))) return st;
    }
    {
      int close = (fused && i == s) ? 1 : 0;
      void* a[] = {bp, &i, &weno_eps, &close, &form};
      if ((K.stencil_kinds & STENCIL_WHOLE) && (st = launch(K.ks.k_update, K.g_update, blk, K.smem_update, a, KK_UPDATE))) return st;
      if ((K.stencil_kinds & STENCIL_SPLIT) &&
          (st = launch(K.ks.k_update_split, K.g_update_split, blk, K.smem_update_split, a, KK_UPDATE)))
        return st;
      if (K.stencil_kinds & STENCIL_MARCH) {
        int nw = 0, nt = 0;
        for (int k = 1; k < i; ++k) {
          nw += AEX(i, k) - AIM(i, k) != 0.0;
          nt += AIM(i, k) != 0.0;
        }
        const void* fn = K.ks.k_update_march[nw == 1 && nt == 0 ? 0 : (nw == 2 && nt == 1 ? 1 : 2)];
        if ((st = launch(fn, K.g_update_march, dim3(K.ks.march_threads), 0, a, KK_UPDATE))) return st;
      }
    }
  }
  if (fused) return 0;
  void* a[] = {bp, &form};
  return launch(K.km.k_finish, K.g_finish, cells, 0, a, KK_FINISH);
}

// Fill the derived per-instance constants of a descriptor from its parameters.
// Stage coefficients of one instance, computed in FP64 and rounded once to T.
template <typename T>
inline void fill_coef(const ap_dvm_params& p, const InstDev& d, Coef<T>& k) {
  k = Coef<T>{};
  k.dt = T(d.dt);
  k.te2 = T(d.te2);
  k.qtau = T(0.25) * T(d.tau);
  k.htau = T(0.5 * d.tau);
  k.inv_dx = T(d.inv_dx);
  k.inv_dy = T(d.inv_dy);
  k.cdx = T(d.inv_dx / 12.0);
  k.cdy = T(d.inv_dy / 12.0);
  k.qcx = T(0.25 * d.tau * d.inv_dx / 12.0);
  k.qcy = T(0.25 * d.tau * d.inv_dy / 12.0);
  k.tcx = T(d.te2 * d.inv_dx / 12.0);
  k.tcy = T(d.te2 * d.inv_dy / 12.0);
  k.ldx = T(d.inv_dx * d.inv_dx / 12.0);
  k.ldy = T(d.inv_dy * d.inv_dy / 12.0);
  for (int i = 1; i <= p.s; ++i)
    for (int j = 1; j <= p.s; ++j) {
      k.aex[i][j] = T(p.A_ex[(i - 1) * AP_DVM_MAX_STAGES + (j - 1)]);
      k.aim[i][j] = T(p.A_im[(i - 1) * AP_DVM_MAX_STAGES + (j - 1)]);
    }
  for (int i = 1; i <= p.s; ++i) {
    const double aii = p.A_im[(i - 1) * AP_DVM_MAX_STAGES + (i - 1)];
    if (aii == 0.0) continue;                     // stage 1 of a CK/ARS tableau is X^n
    k.kappa[i] = T(d.kappa[i]);
    k.r_n[i] = T(d.te2 * d.inv_den[i]);
    k.c_dun[i] = T(1.0 / (p.dt * aii));
    for (int j = 1; j <= i; ++j) {
      const double a = p.A_im[(i - 1) * AP_DVM_MAX_STAGES + (j - 1)];
      const double ae = p.A_ex[(i - 1) * AP_DVM_MAX_STAGES + (j - 1)];
      k.c_du[i][j] = T(a / (p.dt * aii * aii));
      k.c_db[i][j] = T(a / aii);
      k.c_lth[i][j] = T(-1.0 * (a / aii));
      k.wp[i][j] = T((ae - a) * d.inv_aii[i]);
      k.rv_e[i][j] = T(-p.dt * ae * d.inv_den[i]);
      k.rv_v[i][j] = T(-p.dt * a * d.inv_den[i]);
      k.rq_d[i][j] = T(-p.dt * a * (0.5 * d.tau) * d.inv_den[i]);
    }
  }
}

// Tableau of a batch and the nonzero patterns of its rows.
inline void fill_tableau(const ap_dvm_params& p, BatchDev& b) {
  for (int k = 0; k < APD_MAXS * APD_MAXS; ++k) {
    b.A_ex[k] = p.A_ex[k];
    b.A_im[k] = p.A_im[k];
  }
  for (int i = 1; i <= APD_MAXS; ++i) {
    b.m_ex[i] = b.m_im[i] = b.m_wp[i] = 0u;
    for (int j = 1; j <= APD_MAXS; ++j) {
      const double ae = p.A_ex[(i - 1) * AP_DVM_MAX_STAGES + (j - 1)];
      const double ai = p.A_im[(i - 1) * AP_DVM_MAX_STAGES + (j - 1)];
      if (ae != 0.0) b.m_ex[i] |= 1u << j;
      if (ai != 0.0 && j <= i) b.m_im[i] |= 1u << j;
      if (ae - ai != 0.0 && j < i) b.m_wp[i] |= 1u << j;
    }
  }
  b.m_ex[0] = b.m_im[0] = b.m_wp[0] = 0u;
}

inline void fill_constants(const ap_dvm_params& p, InstDev& d) {
  d.dx = p.Lx / p.nx;
  d.dy = p.Ly / p.ny;
  d.dt = p.dt;
  d.eps = p.eps;
  d.tau = p.tau < 0 ? 4.0 * p.eps / p.mach : p.tau;
  d.te2 = d.tau * p.eps * p.eps;
  d.rho0 = p.rho0;
  d.amp = p.mach;
  d.eps32 = (float)p.eps;
  d.rho032 = (float)p.rho0;
  d.amp32 = (float)p.mach;
  for (int i = 1; i <= p.s; ++i) {
    const double a = p.A_im[(i - 1) * AP_DVM_MAX_STAGES + (i - 1)];
    if (a == 0.0) continue;
    d.kappa[i] = 2.0 * p.eps * p.eps / (p.dt * p.dt * a * a);
    d.den[i] = d.te2 + p.dt * a;
    d.inv_den[i] = 1.0 / d.den[i];
  }
  d.inv_dx = 1.0 / d.dx;
  d.inv_dy = 1.0 / d.dy;
  d.hscale = 1.0 / ((double)p.nx * (double)p.ny);
  d.hscale32 = (float)d.hscale;
  for (int i = 1; i <= p.s; ++i) {
    const double a = p.A_im[(i - 1) * AP_DVM_MAX_STAGES + (i - 1)];
    d.inv_aii[i] = a != 0.0 ? 1.0 / a : 0.0;
  }
  fill_coef(p, d, d.k64);
  fill_coef(p, d, d.k32);
  // every member of Coef is a T
  const double* c64 = reinterpret_cast<const double*>(&d.k64);
  const float* c32 = reinterpret_cast<const float*>(&d.k32);
  float* lo = reinterpret_cast<float*>(&d.k32lo);
  static_assert(sizeof(Coef<double>) == 2 * sizeof(Coef<float>), "Coef holds values of its type only");
  for (size_t k = 0; k < sizeof(Coef<float>) / sizeof(float); ++k) lo[k] = (float)(c64[k] - (double)c32[k]);
  const double ra = 1.0 / (p.rho0 * p.mach);
  d.sc_u = ra;
  d.sc_th = p.eps > 0 ? ra / (2.0 * p.eps) : 0.0;
  d.sc_v = p.eps > 0 ? ra / p.eps : 0.0;
  d.sc_q = p.eps > 0 ? ra / (p.eps * p.eps) : 0.0;
  const double sq3 = 1.7320508075688772935;
  d.pmc[0] = d.sc_u;
  d.pmc[1] = 0.5 * d.sc_u;
  d.pmc[2] = 0.5 * sq3 * d.sc_u;
  d.pmc[3] = d.sc_th;
  d.pmc[4] = -0.5 * d.sc_v;
  d.pmc[5] = 0.25 * d.sc_v;
  d.pmc[6] = 0.25 * sq3 * d.sc_v;
  d.pmc[7] = 0.25 * d.sc_q;
  const double pm[6] = {d.pmc[0], d.pmc[2], d.pmc[3], d.pmc[4], d.pmc[6], d.pmc[7]};
  for (int k = 0; k < 6; ++k) {
    int e = 0;
    const double m = 2.0 * std::frexp(pm[k], &e);   // pm = m 2^(e - 1), |m| in [1, 2) (or 0)
    d.pmp_h[k] = (float)m;
    d.pmp_l[k] = (float)(m - (double)d.pmp_h[k]);
    // two powers of two in the float range; a constant beyond it overflows as its narrowed result would
    const int ea = std::max(-120, std::min(120, e - 1)), eb = std::max(-120, std::min(120, e - 1 - ea));
    d.pms_a[k] = (float)std::ldexp(1.0, ea);
    d.pms_b[k] = (float)std::ldexp(1.0, eb);
  }
}

}  // namespace apd
