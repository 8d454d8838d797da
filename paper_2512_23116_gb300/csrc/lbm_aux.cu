// Auxiliary kernels: initial equilibrium, canonical population access in the
// AA layout, parity re-layout and the FP64 reduction finishers.
#include <cuda_runtime.h>

#include <algorithm>
#include <cfloat>

#include "lbm_device.cuh"
#include "lbm_kernels.h"

namespace lbm {

namespace {

constexpr int kAuxThreads = 256;

__device__ __forceinline__ void cell_xyz(int64_t c, int nx, int ny, int& x, int& y, int& z) {
  if (c < (int64_t)0x7fffffff) {  // 32-bit division for lattices below 2^31 cells
    const uint32_t cu = (uint32_t)c, row = cu / (uint32_t)nx;
    x = (int)(cu - row * (uint32_t)nx);
    z = (int)(row / (uint32_t)ny);
    y = (int)(row - (uint32_t)z * (uint32_t)ny);
    return;
  }
  const int64_t row = c / nx;
  x = (int)(c - row * nx);
  z = (int)(row / ny);
  y = (int)(row - (int64_t)z * ny);
}

// Where canonical population a of cell (x, y, z) lives at the given parity:
// even time: slot a of x; odd time: slot opp(a) of x - c_a.
__device__ __forceinline__ int64_t canon_index(const InstDesc& d, int a, bool odd, int x, int y,
                                               int z) {
  if (!odd) return pop_off(d, a, x, y, z);
  int xs = x - cx(a), ys = y - cy(a), zs = z - cz(a);
  xs = xs < 0 ? xs + d.nx : (xs >= d.nx ? xs - d.nx : xs);
  ys = ys < 0 ? ys + d.ny : (ys >= d.ny ? ys - d.ny : ys);
  zs = zs < 0 ? zs + d.nz : (zs >= d.nz ? zs - d.nz : zs);
  return pop_off(d, opp(a), xs, ys, zs);
}

// U: type of the given velocity (mode 3), FP64 or FP32; the equilibrium is
// computed from its FP32 rounding either way.
template <typename T, typename U>
__global__ void k_init(InstDesc d, bool odd, int mode, double amp, const U* __restrict__ u,
                       int64_t ustride, int64_t c0, int64_t n) {
  T* fb = static_cast<T*>(d.f);
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n;
       k += (int64_t)gridDim.x * blockDim.x) {
    int x, y, z;
    cell_xyz(c0 + k, d.nx, d.ny, x, y, z);
    double ux = 0.0, uy = 0.0, uz = 0.0, drho = 0.0;
    if (mode == 1 || mode == 2) {
      double sX, cX, sY, cY, sZ, cZ;
      sincospi(2.0 * x / d.nx, &sX, &cX);
      sincospi(2.0 * y / d.ny, &sY, &cY);
      sincospi(2.0 * z / d.nz, &sZ, &cZ);
      if (mode == 1) {
        ux = amp * sX * cY * cZ;
        uy = -amp * cX * sY * cZ;
      } else {
        ux = amp * sX * cY;
        uy = -amp * cX * sY;
        // pressure of the 2-D vortex: p = (A^2/4)(cos 2X + cos 2Y), drho = 3 p
        drho = 0.75 * amp * amp * ((cX * cX - sX * sX) + (cY * cY - sY * sY));
      }
    } else if (mode == 3) {
      ux = u[k];
      uy = u[ustride + k];
      uz = u[2 * ustride + k];
    }
    float f[19];
    equilibrium((float)drho, (float)ux, (float)uy, (float)uz, f);
#pragma unroll
    for (int a = 0; a < 19; ++a) {
      const int64_t i = canon_index(d, a, odd, x, y, z);
      if (in_bounds(i >= 0 && i < d.f_elems)) fb[i] = Storage<T>::pack(f[a]);
    }
  }
}

template <typename T>
__global__ void k_get_pop(InstDesc d, bool odd, int a, double* __restrict__ out, int shifted,
                          int64_t c0, int64_t n) {
  const T* fb = static_cast<const T*>(d.f);
  const double w = shifted ? 0.0 : weight(a);
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n;
       k += (int64_t)gridDim.x * blockDim.x) {
    int x, y, z;
    cell_xyz(c0 + k, d.nx, d.ny, x, y, z);
    const int64_t i = canon_index(d, a, odd, x, y, z);
    out[k] = (in_bounds(i >= 0 && i < d.f_elems) ? (double)Storage<T>::cvt(fb[i]) : 0.0) + w;
  }
}

template <typename T>
__global__ void k_set_pop(InstDesc d, bool odd, int a, const double* __restrict__ in, int shifted,
                          int64_t c0, int64_t n) {
  T* fb = static_cast<T*>(d.f);
  const double w = shifted ? 0.0 : weight(a);
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n;
       k += (int64_t)gridDim.x * blockDim.x) {
    int x, y, z;
    cell_xyz(c0 + k, d.nx, d.ny, x, y, z);
    const int64_t i = canon_index(d, a, odd, x, y, z);
    if (in_bounds(i >= 0 && i < d.f_elems)) fb[i] = Storage<T>::pack((float)(in[k] - w));
  }
}

__global__ void k_widen(const float* __restrict__ in, int64_t n, double* __restrict__ out) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
    out[k] = (double)in[k];
}

// sa, sb: dense [nz][ny][nxp] copies of slots a and opp(a) taken at the old parity.
template <typename T>
__global__ void k_relayout(InstDesc d, bool from_odd, int a, const T* __restrict__ sa,
                           const T* __restrict__ sb) {
  T* fb = static_cast<T*>(d.f);
  const int b = opp(a);
  const int64_t n = (int64_t)d.nx * d.ny * d.nz;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n;
       k += (int64_t)gridDim.x * blockDim.x) {
    int x, y, z;
    cell_xyz(k, d.nx, d.ny, x, y, z);
    const int64_t o = cell_off(x, y, z, d.ny, d.nxp);
    // canonical values at this cell, from the old layout
    double fa, fbv;
    if (!from_odd) {
      fa = Storage<T>::cvt(sa[o]);
      fbv = Storage<T>::cvt(sb[o]);
    } else {
      // f_a(x) = slot b of x - c_a ; f_b(x) = slot a of x + c_a
      int xs = x - cx(a), ys = y - cy(a), zs = z - cz(a);
      xs = (xs + d.nx) % d.nx;
      ys = (ys + d.ny) % d.ny;
      zs = (zs + d.nz) % d.nz;
      int xq = x + cx(a), yq = y + cy(a), zq = z + cz(a);
      xq = (xq + d.nx) % d.nx;
      yq = (yq + d.ny) % d.ny;
      zq = (zq + d.nz) % d.nz;
      fa = Storage<T>::cvt(sb[cell_off(xs, ys, zs, d.ny, d.nxp)]);
      fbv = Storage<T>::cvt(sa[cell_off(xq, yq, zq, d.ny, d.nxp)]);
    }
    const bool to_odd = !from_odd;
    const int64_t ia = canon_index(d, a, to_odd, x, y, z), ib = canon_index(d, b, to_odd, x, y, z);
    if (in_bounds(ia >= 0 && ia < d.f_elems)) fb[ia] = Storage<T>::pack((float)fa);
    if (in_bounds(ib >= 0 && ib < d.f_elems)) fb[ib] = Storage<T>::pack((float)fbv);
  }
}

// One warp per output value: lane l folds blocks l, l + 32, ... in that order,
// then a fixed shuffle tree combines the lanes, so a result depends only on
// the partials and the grid size, never on scheduling.  seq[0] counts the
// records in the ring; seq[1] counts the blocks of a launch that are done, and
// the last of them advances seq[0] (every block has read it by then).
__global__ void k_finish(const double* __restrict__ partials, int ninst, int grid,
                         double* __restrict__ results, double* ring, unsigned long long* seq,
                         int cap, uint32_t* err) {
  const unsigned long long slot = ring ? (__ldcg(seq) % (unsigned long long)cap) : 0ull;
  const int lane = threadIdx.x & 31;
  const int warps = (int)((gridDim.x * blockDim.x) >> 5);
  for (int idx = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); idx < ninst * kNP; idx += warps) {
    const int i = idx / kNP, k = idx - i * kNP;
    const bool lo = k == P_THMIN, hi = k == P_THMAX;
    double r = lo ? DBL_MAX : (hi ? -DBL_MAX : 0.0);
#pragma unroll 4
    for (int b = lane; b < grid; b += 32) {  // unrolled: the loads of four blocks in flight together
      const double* p = partials + ((int64_t)i * grid + b) * kNP;
      const double v = p[k], n = p[P_CELLS];
      if (n != 0.0) r = lo ? fmin(r, v) : (hi ? fmax(r, v) : r + v);  // else the block saw no cell of instance i
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      const double o = __shfl_down_sync(0xffffffffu, r, off);
      r = lo ? fmin(r, o) : (hi ? fmax(r, o) : r + o);
    }
    if (lane == 0) {
      results[idx] = r;
      if (k == P_BAD && r > 0.0) atomicOr(err, ERR_NONFINITE);
      if (ring) ring[slot * (unsigned long long)(ninst * kNP) + idx] = r;
    }
  }
  if (!ring) return;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(seq + 1, 1ull) == (unsigned long long)gridDim.x - 1ull) {
      seq[0] += 1ull;
      seq[1] = 0ull;
    }
  }
}

// Column sums of a [rows][cols] table times `scale`, one warp per column in the fixed order
// of k_finish (lane l adds rows l, l + 32, ...; then a shuffle tree).
__global__ void k_sum_cols(const double* __restrict__ p, int rows, int cols, double scale,
                           double* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  const int warps = (int)((gridDim.x * blockDim.x) >> 5);
  for (int c = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); c < cols; c += warps) {
    double r = 0.0;
#pragma unroll 4
    for (int b = lane; b < rows; b += 32) r += p[(int64_t)b * cols + c];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) r += __shfl_down_sync(0xffffffffu, r, off);
    if (lane == 0) out[c] = r * scale;
  }
}

int grid_for(int64_t n) {
  int64_t b = (n + kAuxThreads - 1) / kAuxThreads;
  if (b < 1) b = 1;
  if (b > 4096) b = 4096;
  return (int)b;
}

template <typename T, typename U>
cudaError_t init_t(const InstDesc& d, bool odd, int mode, double amp, const U* u,
                   int64_t ustride, int64_t c0, int64_t n, cudaStream_t st) {
  return launch_kernel(k_init<T, U>, grid_for(n), kAuxThreads, 0, st, d, odd, mode, amp, u, ustride, c0, n);
}

template <typename U>
cudaError_t launch_init_u(const InstDesc& d, int precision, bool odd, int mode, double amp,
                          const U* u, int64_t ustride, int64_t c0, int64_t n, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  switch (precision) {
    case 0: return init_t<float, U>(d, odd, mode, amp, u, ustride, c0, n, st);
    case 1: return init_t<__half, U>(d, odd, mode, amp, u, ustride, c0, n, st);
    case 2: return init_t<__nv_bfloat16, U>(d, odd, mode, amp, u, ustride, c0, n, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_init(const InstDesc& d, int precision, bool odd, int mode, double amp,
                        const double* u, int64_t ustride, int64_t c0, int64_t n, cudaStream_t st) {
  return launch_init_u<double>(d, precision, odd, mode, amp, u, ustride, c0, n, st);
}

cudaError_t launch_init(const InstDesc& d, int precision, bool odd, const float* u, int64_t ustride,
                        int64_t c0, int64_t n, cudaStream_t st) {
  return launch_init_u<float>(d, precision, odd, 3, 0.0, u, ustride, c0, n, st);
}

cudaError_t launch_get_pop(const InstDesc& d, int precision, bool odd, int a, double* out,
                           int shifted, int64_t c0, int64_t n, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  const int g = grid_for(n);
  switch (precision) {
    case 0: return launch_kernel(k_get_pop<float>, g, kAuxThreads, 0, st, d, odd, a, out, shifted, c0, n);
    case 1: return launch_kernel(k_get_pop<__half>, g, kAuxThreads, 0, st, d, odd, a, out, shifted, c0, n);
    case 2: return launch_kernel(k_get_pop<__nv_bfloat16>, g, kAuxThreads, 0, st, d, odd, a, out, shifted, c0, n);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_set_pop(const InstDesc& d, int precision, bool odd, int a, const double* in,
                           int shifted, int64_t c0, int64_t n, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  const int g = grid_for(n);
  switch (precision) {
    case 0: return launch_kernel(k_set_pop<float>, g, kAuxThreads, 0, st, d, odd, a, in, shifted, c0, n);
    case 1: return launch_kernel(k_set_pop<__half>, g, kAuxThreads, 0, st, d, odd, a, in, shifted, c0, n);
    case 2: return launch_kernel(k_set_pop<__nv_bfloat16>, g, kAuxThreads, 0, st, d, odd, a, in, shifted, c0, n);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_widen(const float* in, int64_t n, double* out, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  return launch_kernel(k_widen, grid_for(n), kAuxThreads, 0, st, in, n, out);
}

cudaError_t launch_relayout_pair(const InstDesc& d, int precision, bool from_odd, int a,
                                 void* scratch, cudaStream_t st) {
  const size_t es = precision == 0 ? 4 : 2;
  const size_t row = (size_t)d.nxp * es;
  const size_t rows = (size_t)d.nz * d.ny;
  const size_t plane = row * rows;
  char* s = static_cast<char*>(scratch);
  const char* base = static_cast<const char*>(d.f);
  const size_t pa = d.slot_grouped ? gpos(a) : a, pb = d.slot_grouped ? gpos(opp(a)) : opp(a);
  // slots a and opp(a), x-line by x-line (row_stride apart in either layout), into dense planes
  cudaError_t e = cudaMemcpy2DAsync(s, row, base + pa * d.slot_stride * es, (size_t)d.row_stride * es,
                                    row, rows, cudaMemcpyDeviceToDevice, st);
  if (e != cudaSuccess) return e;
  e = cudaMemcpy2DAsync(s + plane, row, base + pb * d.slot_stride * es, (size_t)d.row_stride * es,
                        row, rows, cudaMemcpyDeviceToDevice, st);
  if (e != cudaSuccess) return e;
  const int g = grid_for((int64_t)d.nx * d.ny * d.nz);
  switch (precision) {
    case 0:
      return launch_kernel(k_relayout<float>, g, kAuxThreads, 0, st, d, from_odd, a, (const float*)s,
                           (const float*)(s + plane));
    case 1:
      return launch_kernel(k_relayout<__half>, g, kAuxThreads, 0, st, d, from_odd, a, (const __half*)s,
                           (const __half*)(s + plane));
    case 2:
      return launch_kernel(k_relayout<__nv_bfloat16>, g, kAuxThreads, 0, st, d, from_odd, a,
                           (const __nv_bfloat16*)s, (const __nv_bfloat16*)(s + plane));
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_finish(const double* partials, int ninst, int grid, double* results,
                          double* ring, unsigned long long* seq, int cap, uint32_t* err,
                          cudaStream_t st) {
  const int warps_per_block = 256 / 32;
  const int blocks = std::max(1, std::min(1024, (ninst * kNP + warps_per_block - 1) / warps_per_block));
  return launch_kernel(k_finish, blocks, 256, 0, st, partials, ninst, grid, results, ring, seq, cap, err);
}

cudaError_t launch_sum_cols(const double* partials, int rows, int cols, double* out,
                            cudaStream_t st, double scale) {
  const int blocks = std::max(1, std::min(1024, (cols + 7) / 8));  // 8 warps per block, a warp per column
  return launch_kernel(k_sum_cols, blocks, 256, 0, st, partials, rows, cols, scale, out);
}

uint32_t bounds_word_aux() { return take_bounds_word(); }

}  // namespace lbm
