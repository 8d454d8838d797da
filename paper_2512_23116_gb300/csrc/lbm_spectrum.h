// Host interface of the energy-spectrum kernels (lbm_spectrum.cu).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace lbm {

constexpr int kMaxStages = 12;
// Shells of a spectrum: the block totals of k_bin_lines and of the last transform
// pass are FP64 values in shared memory.
constexpr int kMaxShells = 6144;

// A transform of length n as radix[0] x radix[1] x ... (stages in that order).  Stage
// i works on sub-transforms of radix[i] x m[i] rows; a butterfly's number b splits
// into b = blk m + j by a multiplication with inv_m, and the step from one butterfly of a
// thread to its next into dj, db (integer divisions cost a thread as much as a butterfly).
struct FftAxis {
  int n, stages;
  int radix[kMaxStages], m[kMaxStages], dj[kMaxStages], db[kMaxStages];
  float inv_m[kMaxStages];
};

// Plan of the framework's own three-dimensional transform of a velocity component.
struct FftPlan {
  FftAxis ax[3];              // x, y, z
  int64_t half;               // complex values of a component's half spectrum [nz/2 + 1][ny][nx]
  int width[3], tile[3], threads[3], smem[3], blocks[3];  // per pass (x, y, z): columns and values of a tile, launch
};

// True when every extent has prime factors up to 13 only and its columns fit shared
// memory: the plan for `kmax` shells.  False otherwise, or on a CUDA error (*err).
bool plan_fft(int nx, int ny, int nz, int kmax, FftPlan* out, cudaError_t* err);
// exp(-2 pi i k / n) for k < n: x table, then y, then z (nx + ny + nz values).
void fft_twiddles(const FftPlan& pl, float2* host);
// Shell sums of |u_hat|^2 (not normalised) of `comps` components of u
// [3][nz][ny][nx] starting at component `first`, added to partials
// [pl.blocks[0]][kmax + 1]; work holds comps x pl.half values, tw the tables.
cudaError_t launch_fft_shells(const float* u, const FftPlan& pl, int first, int comps, int kmax, const float2* tw,
                              float2* work, double* partials, cudaStream_t st);

// Shell sums of |u_hat|^2 (not normalised) of a kx-half spectrum [nz][ny][nx/2 + 1],
// added to partials [blocks][kmax + 1].
int bin_lines_blocks(int nx, int ny, int nz, int kmax, int num_sms);
cudaError_t launch_bin_lines(const float2* c, int nx, int ny, int nz, int kmax, double* partials, int blocks,
                             cudaStream_t st);

uint32_t bounds_word_spectrum();

}  // namespace lbm
