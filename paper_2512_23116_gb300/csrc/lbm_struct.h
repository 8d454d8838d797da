// Host interface of the structure-function kernels (lbm_struct.cu).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace lbm {

constexpr int kMaxStructSeps = 24;

// How the pencils of one axis are cut into tiles.
struct StructAxis {
  int64_t first;    // first tile of the axis
  int64_t pencils;  // pencils along the axis
  int64_t stride;   // values between neighbours along the axis
  int n;            // cells of a pencil
  int segs, len;    // segments of a pencil and their length (the last may be shorter)
  int halo;         // largest wrapped separation
};

// One launch of k_struct_tiles (kernel parameter).
struct StructPlan {
  StructAxis ax[3];
  int64_t tiles, ncell, plane;
  int nx, nr;
  int rows_max;                 // longest tile: segment plus halo
  int r[3][kMaxStructSeps];     // separations wrapped to each extent
  int grid, threads, smem;
};

// Plan the structure functions of nr <= 24 separations r[k] >= 1 on a lattice:
// exact = false in FP32 powers, exact = true with the accuracy of FP64 sums.  At
// most max_blocks blocks.  Returns false when a separation, wrapped, is too long
// for a tile in shared memory (*err = cudaSuccess) or on a CUDA error (*err).
bool plan_struct(int nx, int ny, int nz, const int* r, int nr, bool exact, int max_blocks, StructPlan* out,
                 cudaError_t* err);

// partials[pl.grid][nr][6]: sums over a block's cells and the three axes of
// (u_a(x + r e_a) - u_a(x))^p, p = 1..6, for the velocity u [3][nz][ny][nx] FP32.
cudaError_t launch_struct_plan(const float* u, const StructPlan& pl, bool exact, double* partials, cudaStream_t st);

// The same sums of one separation of any length in FP64: per block b,
// partials[b * block_stride + p - 1].
cudaError_t launch_struct(const float* u, int nx, int ny, int nz, int r, double* partials,
                          int blocks, cudaStream_t st, int64_t block_stride);

uint32_t bounds_word_struct();

}  // namespace lbm
