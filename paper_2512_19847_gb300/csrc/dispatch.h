// Kernel tables shared between the instantiation units and the host API.
#pragma once
#include <cstddef>
#include <cuda_runtime.h>

namespace apd {

// Tile shapes of the stencil kernels (index = ap_dvm_set_tile argument).
constexpr int kNumTiles = 6;
constexpr int kTileX[kNumTiles] = {32, 32, 16, 8, 64, 32};
constexpr int kTileY[kNumTiles] = {8, 4, 8, 8, 4, 16};

// The automatic tile shape for grids of at least minx x miny cells.  tiles(t) is the number of
// tiles of shape t over all of them, num_sms 0 when it is not to be looked at (a batch, whose
// tiles come and go).
//   FP32: 16x8 (7 blocks of 128 threads per SM); 2048^2, 4 steps, explicit + update: 1.55 + 2.00 ms
//   against 1.82 + 2.65 with 32x8 and 1.99 + 2.31 with 8x8; 509x251: 0.14 + 0.16 against 0.20 +
//   0.23 and 0.16 + 0.18; 24 uneven solves: 1.33 + 1.66 against 1.58 + 2.23 and 1.69 + 1.91.
//   FP64: 32x8 while it gives two tiles per SM (2048^2: 2.16 + 2.18 against 2.12 + 2.31 with 16x8
//   and 2.33 + 2.51 with 8x8), else the next smaller: a grid of fewer tiles leaves SMs, and with
//   them FP64 pipes, idle (64^2, 10 steps: 0.78 + 0.78 ms with 16 tiles of 32x8, 0.55 + 0.57 with
//   64 of 8x8; 384x192 LF1: 0.29 + 0.26 with 288 of 32x8, 0.26 + 0.24 with 576 of 16x8).
template <class Tiles>
inline int pick_tile(bool f32, int minx, int miny, int num_sms, Tiles&& tiles) {
  static constexpr int order64[4] = {0, 1, 2, 3}, order32[2] = {2, 3}, small64[3] = {0, 2, 3};
  auto fits = [&](int t) { return kTileX[t] <= minx && kTileY[t] <= miny; };
  if (f32) {
    for (int t : order32)
      if (fits(t)) return t;
  } else if (num_sms > 0) {
    for (int t : small64)
      if (fits(t) && tiles(t) >= 2LL * num_sms) return t;
  } else {
    for (int t : order64)
      if (fits(t)) return t;
  }
  return 3;
}

struct StencilSet {
  const void* k_explicit;
  const void* k_rhs[3];                // 1, 4, or up to the most terms of earlier stages
  const void* k_update;
  const void* k_explicit_split;        // FP64 WENO: the same with split fluxes (null otherwise)
  const void* k_update_split;
  size_t smem_explicit_split;
  size_t (*smem_update_split)(int planes);   // with so many staged planes
  // FP32: by marching warps (null otherwise).  Explicit: [terms of v read from memory: 1, 2, up to
  // 5][bit 0: E, bit 1: D_LF . B(v)]; update: [(stages in the partner, earlier stages in the sums):
  // (1, 0), (2, 1), up to (3, 3)]
  const void* k_explicit_march[3][4];
  const void* k_update_march[3];
  int march_threads;
  size_t smem_explicit;
  int rhs_threads;                     // k_rhs: threads per block (no dynamic shared memory)
  size_t plane_bytes, update_fixed;   // k_update: update_fixed + nbuf * (planes staged) * plane_bytes
  int nbuf;                            // staged plane buffers of k_update (1 or 2)
  int tx, ty, tz;                      // tile, and threads per cell (explicit and update kernels)
  int bw, bh;                          // staged box: (tx + 8) x (ty + 2 * halo)
};

struct MiscSet {
  const void* k_finish;    // per tile shape
  const void* k_stage1;    // per tile shape; type-A tableaux only
  const void* k_rows_fwd;    // Helmholtz transforms, power-of-two axes ...
  const void* k_cols;
  int cols_threads;        // threads per block of k_cols
  int rows_threads;        // threads per block of k_rows_fwd and k_rows_inv
  const void* k_rows_inv;
  const void* k_rows_fwd_bs; // ... and axes of other lengths (Bluestein)
  const void* k_cols_bs;
  const void* k_rows_inv_bs;
  const void* k_set_state;
  const void* k_get_state;
  const void* k_diagnostics;
};

StencilSet stencil_f64_lf1(int tile);
StencilSet stencil_f64_w3(int tile);
StencilSet stencil_f64_w5(int tile);
StencilSet stencil_f32_lf1(int tile);
StencilSet stencil_f32_w3(int tile);
StencilSet stencil_f32_w5(int tile);
MiscSet misc_set(int f32form, int tile);
// One kernel whose bounded wait expires after limit_ns (sets the timeout bit of err).
cudaError_t launch_wait_timeout(unsigned* err, unsigned long long limit_ns, cudaStream_t stream);
// The integer-pipe FP32 <-> FP64 conversions against the instructions (ap_dvm_check_conversions).
cudaError_t launch_check_conversions(const double* in, int n, unsigned* bad, cudaStream_t stream);

}  // namespace apd
