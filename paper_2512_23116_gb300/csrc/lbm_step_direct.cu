// Direct-load stream + collide kernel (AA pattern, one population array).
//
// Even step: cell x reads f_a from its own slot a and writes f*_a to its own
// slot opp(a).  Odd step: cell x reads f_a from slot opp(a) of x - c_a and
// writes f*_a to slot a of x + c_a.  Each cell reads exactly the locations it
// writes, so all cells of a step are independent (Eq. mrt_les_guo, with
// periodic streaming of Sec. 3.1).  One thread per cell, plain coalesced
// loads and stores.
//
// Work is dealt out in chunks of blockDim.x consecutive cells (x fastest, rows and
// planes running on), so no thread idles at the end of a row or a tile; the
// coordinates advance from chunk to chunk by additions.  The location that f*_a goes to
// is the one f_opp(a) came from, so 19 offsets serve loads and stores; they are
// 32-bit for arrays below 4 GB (WIDE = false).
//
// What bounds it: the L2 cache.  With the collision taken out a step of 64^3 takes
// 5.7 of its 6.2 us and one of 100^3 18.5 of 19.9 (9 TB/s; the odd step's x-shifted
// slots cost 2-3 us of that in partly written sectors); prefetching the next
// cell, into registers or by asynchronous copies, made it slower.  Below that it is
// latency: launches and the first loads, which the launch parameter `one`, 32-bit
// divisions and dependent launches shorten.  A step of 16^3 takes 1.5 us, 32^3 2.1 (the TMA
// kernel 5.2), 48^3 3.7 (6.2), 64^3 6.2 (8.6), 80^3 10.5 (12.4); beyond ~100^3 the TMA
// kernel is ahead (128^3: 54 against 61), but for boxes of small planes.
#include <cuda_runtime.h>

#include <type_traits>

#include "lbm_device.cuh"
#include "lbm_kernels.h"
#include "lbm_reduce.cuh"

namespace lbm {

constexpr int kSmemHistBins = 12000;  // (bins + 1) * 4 bytes below 48 KB

namespace {

// Index of the instance that owns chunk t, `from` or a later one (a block's chunks
// increase).  The instances of a batch are mostly alike: the chunks ahead over those
// of `from` guess it, and a wrong guess bounds a bisection.  Going through them one by one
// cost a dependent load each: 300 instances of 8^3 took 40 us a step, 1000 of 6^3 148; now
// 4.5 and 8.3.
__device__ __forceinline__ int find_chunk_instance(const InstDesc* __restrict__ insts, int ninst, int64_t t, int from) {
  const int64_t begin = insts[from].chunk_begin, end = insts[from].chunk_end;
  if (t < end || from + 1 >= ninst) return from;
  int lo = from + 1, hi = ninst - 1;
  int i = min(hi, from + (int)fminf((float)(t - begin) / (float)(end - begin), (float)ninst));
  while (lo < hi) {
    if (t < insts[i].chunk_begin) {
      hi = i - 1;
    } else if (t >= insts[i].chunk_end) {
      lo = i + 1;
    } else {
      return i;
    }
    i = (lo + hi) >> 1;
  }
  return lo;
}

// What a thread keeps of the instance it is in.
template <typename I>
struct CellWalk {
  int64_t end;             // one past the instance's last chunk
  int nx, ny, nz;
  int x, y, z;             // the thread's cell
  int dx, dy, dz;          // from one of the block's chunks to its next
  I slot, row, plane;      // strides (values)
  bool grouped;
  __device__ __forceinline__ void enter(const InstDesc& d, int64_t t, int64_t stride) {
    end = d.chunk_end;
    nx = d.nx;
    ny = d.ny;
    nz = d.nz;
    slot = (I)d.slot_stride;
    row = (I)d.row_stride;
    plane = (I)d.plane_stride;
    grouped = d.slot_grouped != 0;
    // cells and strides fit 32 bits with 32-bit offsets
    using U = typename std::conditional<sizeof(I) == 4, uint32_t, int64_t>::type;
    const U plane_cells = (U)nx * (U)ny;
    const U c = (U)(t - d.chunk_begin) * blockDim.x + threadIdx.x, s = (U)stride * blockDim.x;
    z = (int)(c / plane_cells);
    const U r = c - (U)z * plane_cells;
    y = (int)(r / (U)nx);
    x = (int)(r - (U)y * (U)nx);
    dz = (int)(s / plane_cells);
    const U q = s - (U)dz * plane_cells;
    dy = (int)(q / (U)nx);
    dx = (int)(q - (U)dy * (U)nx);
  }
  __device__ __forceinline__ void next() {
    x += dx;
    y += dy;
    z += dz;
    if (x >= nx) {
      x -= nx;
      ++y;
    }
    if (y >= ny) {
      y -= ny;
      ++z;
    }
  }
};

// Offset of what the cell reads as f_a (values): the even step's slot a of the cell, the
// odd step's slot opp(a) of the cell at -c_a.  f*_a goes to the location of opp(a).
template <typename I, bool ODD>
__device__ __forceinline__ void offsets(const CellWalk<I>& w, I (&o)[19]) {
  if (!ODD) {
    const I c = (I)w.z * w.plane + (I)w.y * w.row + (I)w.x;
#pragma unroll
    for (int a = 0; a < 19; ++a) o[a] = c + (I)(w.grouped ? gpos(a) : a) * w.slot;
  } else {
    const I xs[3] = {(I)wrap_inc(w.x, w.nx), (I)w.x, (I)wrap_dec(w.x, w.nx)};  // by cx + 1
    const I ys[3] = {(I)wrap_inc(w.y, w.ny) * w.row, (I)w.y * w.row, (I)wrap_dec(w.y, w.ny) * w.row};
    const I zs[3] = {(I)wrap_inc(w.z, w.nz) * w.plane, (I)w.z * w.plane, (I)wrap_dec(w.z, w.nz) * w.plane};
#pragma unroll
    for (int a = 0; a < 19; ++a)
      o[a] = (zs[cz(a) + 1] + ys[cy(a) + 1]) + (xs[cx(a) + 1] + (I)(w.grouped ? gpos(opp(a)) : opp(a)) * w.slot);
  }
}

}  // namespace

// Dependent launches: the next step's blocks may start, and read their launch
// parameters, while this step's last blocks still run; nothing of the populations is
// touched before dependency_wait, which returns when the step before has completed
// and its writes are visible.
__device__ __forceinline__ void dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void dependents_may_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// ONE: a single instance, described by the launch parameter `one` (the table costs a chain of
// dependent loads before the first population can be read).
template <typename T, bool ODD, int MODE, bool WIDE, bool ONE>
__global__ void __launch_bounds__(256, 2)
k_step_direct(const InstDesc* __restrict__ insts, int ninst, int64_t chunk_lo, int64_t chunk_hi,
              StatsArgs sa, DiagOut dout, const __grid_constant__ InstDesc one) {
  using S = Storage<T>;
  using I = typename std::conditional<WIDE, int64_t, uint32_t>::type;
  extern __shared__ uint32_t shist[];
  // theta histogram in shared memory when it fits the default 48 KB, else
  // straight into the global counts
  const bool use_hist = (MODE == MODE_DIAG) && dout.hist != nullptr && dout.hist_bins < kSmemHistBins;
  if (use_hist) {
    for (int i = threadIdx.x; i <= dout.hist_bins; i += blockDim.x) shist[i] = 0u;
    __syncthreads();
  }
  Acc acc;
  acc.reset();
  HistRun run;
  uint32_t* const hist_sm = use_hist ? shist : nullptr;
  const int hist_win = use_hist ? dout.hist_bins + 1 : 0;
  uint32_t* const hist_gl = use_hist ? nullptr : dout.hist;
  int cur = -1;
  CellWalk<I> w;
  w.end = -1;
  T* __restrict__ fb = nullptr;
  const float *fx = nullptr, *fy = nullptr, *fz = nullptr;
  float cfx = 0.f, cfy = 0.f, cfz = 0.f, nu0 = 0.f, s_nu0 = 0.f, C = 0.f;
  int smode = 0;
  if (MODE == MODE_STEP) dependents_may_start();
  bool waited = MODE != MODE_STEP;
  for (int64_t t = chunk_lo + blockIdx.x; t < chunk_hi; t += gridDim.x) {
    if (t >= w.end) {
      const int ii = ONE ? 0 : find_chunk_instance(insts, ninst, t, cur < 0 ? 0 : cur);
      if (MODE != MODE_STEP) {
        if (cur >= 0 && sa.partials)
          block_flush(acc, sa.partials + ((int64_t)cur * sa.grid + blockIdx.x) * kNP, blockDim.x, 0);
        acc.reset();
      }
      cur = ii;
      const InstDesc& d = ONE ? one : insts[ii];
      w.enter(d, t, gridDim.x);
      fb = static_cast<T*>(d.f);
      fx = d.fx_of_y;
      fy = d.fy_of_z;
      fz = d.fz_of_x;
      cfx = d.fconst[0];
      cfy = d.fconst[1];
      cfz = d.fconst[2];
      nu0 = d.nu0;
      s_nu0 = d.s_nu0;
      C = d.C;
      smode = d.strain_mode;
    } else {
      w.next();
    }
    if (!waited) {
      dependency_wait();
      waited = true;
    }
    // one copy of the cell's work per strain mode, a constant in each, as in the TMA
    // kernel: the compiler then contracts the same operations, and the two kernels give
    // the same bits
    auto cell = [&](auto mode) __attribute__((always_inline)) {
      I o[19];
      offsets<I, ODD>(w, o);
      float f[19];
#pragma unroll
      for (int a = 0; a < 19; ++a)
        f[a] = in_bounds((int64_t)o[a] >= 0 && (int64_t)o[a] < (ONE ? one : insts[cur]).f_elems) ? S::load(fb + o[a]) : 0.f;
      const bool cell_ok = in_bounds(w.x >= 0 && w.x < w.nx && w.y >= 0 && w.y < w.ny && w.z >= 0 && w.z < w.nz);
      const float Fx = (cell_ok ? fx[w.y] : 0.f) + cfx, Fy = (cell_ok ? fy[w.z] : 0.f) + cfy,
                  Fz = (cell_ok ? fz[w.x] : 0.f) + cfz;
      CellDiag g;
      mrt_collide(f, Fx, Fy, Fz, nu0, s_nu0, C, g, decltype(mode)::value);
      if (MODE != MODE_DIAG) {
#pragma unroll
        for (int a = 0; a < 19; ++a)
          if (in_bounds((int64_t)o[opp(a)] >= 0 && (int64_t)o[opp(a)] < (ONE ? one : insts[cur]).f_elems))
            fb[o[opp(a)]] = S::pack(f[a]);
      }
      if (MODE != MODE_STEP) acc.add(g, Fx, Fy, Fz, C);
      if (MODE == MODE_DIAG)
        diag_write(dout, g, w.x, w.y, w.z, w.nx, w.ny, w.nz, hist_sm, 0, hist_win, hist_gl, run);
    };
    if (w.z < w.nz) {  // the last chunk of an instance may run past its cells
      if (smode == 1)
        cell(std::integral_constant<int, 1>{});
      else
        cell(std::integral_constant<int, 0>{});
    }
    if (MODE != MODE_STEP) acc.fold_if_full();
  }
  if (MODE != MODE_STEP) {
    if (cur >= 0 && sa.partials)
      block_flush(acc, sa.partials + ((int64_t)cur * sa.grid + blockIdx.x) * kNP, blockDim.x, 0);
  }
  if (MODE == MODE_DIAG && dout.hist) run.flush(hist_sm, 0, hist_win, hist_gl);
  if (use_hist) {
    __syncthreads();
    for (int i = threadIdx.x; i <= dout.hist_bins; i += blockDim.x)
      if (shist[i]) atomicAdd(&dout.hist[i], shist[i]);
  }
}

template <typename T, bool ODD, int MODE>
static cudaError_t launch_direct_t(const LaunchArgs& la, cudaStream_t st) {
  if constexpr (MODE == MODE_STEP) {
    if (la.ninst == 1 && !la.wide)
      return launch_dependent(k_step_direct<T, ODD, MODE, false, true>, la.grid, la.threads, 0, st, la.insts, la.ninst,
                              la.tile_lo, la.tile_hi, la.sa, la.dout, la.one);
    return launch_dependent(la.wide ? k_step_direct<T, ODD, MODE, true, false> : k_step_direct<T, ODD, MODE, false, false>,
                            la.grid, la.threads, 0, st, la.insts, la.ninst, la.tile_lo, la.tile_hi, la.sa, la.dout, la.one);
  }
  const size_t smem = (MODE == MODE_DIAG && la.dout.hist && la.dout.hist_bins < kSmemHistBins)
                          ? (size_t)(la.dout.hist_bins + 1) * 4
                          : 0;
  return launch_kernel(la.wide ? k_step_direct<T, ODD, MODE, true, false> : k_step_direct<T, ODD, MODE, false, false>,
                       la.grid, la.threads, smem, st, la.insts, la.ninst, la.tile_lo, la.tile_hi, la.sa, la.dout, la.one);
}

template <typename T>
static cudaError_t dispatch_direct(const LaunchArgs& la, cudaStream_t st) {
  if (la.odd) {
    if (la.mode == MODE_STEP) return launch_direct_t<T, true, MODE_STEP>(la, st);
    if (la.mode == MODE_STEP_STATS) return launch_direct_t<T, true, MODE_STEP_STATS>(la, st);
    return launch_direct_t<T, true, MODE_DIAG>(la, st);
  }
  if (la.mode == MODE_STEP) return launch_direct_t<T, false, MODE_STEP>(la, st);
  if (la.mode == MODE_STEP_STATS) return launch_direct_t<T, false, MODE_STEP_STATS>(la, st);
  return launch_direct_t<T, false, MODE_DIAG>(la, st);
}

cudaError_t launch_step_direct(const LaunchArgs& la, cudaStream_t st) {
  switch (la.precision) {
    case 0: return dispatch_direct<float>(la, st);
    case 1: return dispatch_direct<__half>(la, st);
    case 2: return dispatch_direct<__nv_bfloat16>(la, st);
    default: return cudaErrorInvalidValue;
  }
}

int direct_max_blocks_per_sm(int precision, int threads) {
  int n = 0;
  cudaError_t e = cudaErrorInvalidValue;
  switch (precision) {
    case 0: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_step_direct<float, true, MODE_STEP, false, false>, threads, 0); break;
    case 1: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_step_direct<__half, true, MODE_STEP, false, false>, threads, 0); break;
    case 2: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_step_direct<__nv_bfloat16, true, MODE_STEP, false, false>, threads, 0); break;
  }
  return e == cudaSuccess ? n : 0;
}

uint32_t bounds_word_direct() { return take_bounds_word(); }

}  // namespace lbm
