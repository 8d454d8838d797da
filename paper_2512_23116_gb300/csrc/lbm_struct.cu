// Structure functions S_p(r) = <(u_a(x + r e_a) - u_a(x))^p>, p = 1..6, pooled
// over the three axes a (Eqs. velocity_increment, structure_function), for up to
// 24 separations in one launch.
//
// Layout of the work.  Component a only ever meets itself along axis a, so the
// field falls into pencils: 32 pencils by L cells along the axis (plus the
// largest separation, wrapped) are staged in shared memory once and serve every
// separation; element i of pencil c is at i x 33 + c, so that staging x-lines
// (lanes along i) and walking pencils (lanes along c) are both free of bank
// conflicts.  A warp walks a run of cells with one lane per pencil; a cell's own
// value and its partners are one shared-memory load each at a fixed offset.
// Reading every partner from global memory instead was bound by the latency of
// the shifted loads (9 % of the DRAM peak at 256^3).
//
// Two accuracies share that skeleton:
//  - k_struct_tiles<SUMS_4> and <SUMS_1>, for lbm_stats: FP32 increments and powers as
//    the FP32 velocity allows.  Plain FP32 sums span 4 cells; over a lane's run those of
//    the odd powers, and over the warp all of them, are kept in two words, then added in
//    FP64.  Lattices up to kSmallCells have few cells for roundings to average over, and
//    time to spare: no plain sums at all.  Two separations share a register pair (f32x2
//    operations).  Against FP64 sums of random solenoidal fields S_1 to S_6 are off by
//    2e-11 to 6e-10 of <|d|^p> at 100^3 and 7e-12 to 2e-9 at 404^3; plain sums of 64 cells
//    and the warp left S_1, S_3 and S_5 2-20 times that.  Bound by the FP32 pipe: 13
//    operations an increment (9 with plain sums).  A call of lbm_stats with them
//    takes 84 us more than one without at 100^3 (11 separations), 1.74 ms at 400^3 (15), 3.42
//    ms at 512^3 (16); 125 us, 3.34 and 7.03 ms with partners read from global memory.
//  - k_struct_tiles<SUMS_EXACT>, for lbm_structure_functions_noalloc: the FP64 sums of
//    the exact increments.  This part executes 2 FP64 operations per clock and
//    SM against 128 in FP32, so increments, powers and running sums are kept as
//    unevaluated sums of FP32 words (Dekker 1971; Knuth's two-sum, products with
//    an FMA for the remainder).  Against quadruple-precision sums it is off by at most
//    6e-16 of <|d|^p> for every p, on random, Taylor-Green, sinusoidal and ramp fields of
//    5e2 to 1e6 cells (2e-16 typically), where the FP64 loop left 0.1-1.2e-14.  Each tile
//    scales its increments by a power of two so that neither the sixth power nor its low
//    words leave the FP32 range; a tile whose values do not allow that (infinities, NaN,
//    extreme exponents) is summed in FP64.  Bound by issue: ~215 FP32 operations an
//    increment.  12 separations at 160^3: 4.50 ms (one FP64 pass over global memory
//    per separation, at the FP64 rate) -> 1.15 ms.
#include <cuda_runtime.h>

#include <algorithm>
#include <cfloat>
#include <climits>

#include "lbm_check.cuh"
#include "lbm_kernels.h"
#include "lbm_struct.h"
#include "lbm_words.cuh"

namespace lbm {

namespace {

constexpr int kCols = 32;       // pencils of a tile: one per lane
constexpr int kPitch = 33;      // values between consecutive cells of a pencil
constexpr int kRunMax = 64;     // cells a lane sums before the warp reduces
constexpr int kRunMin = 4;      // fewer are not worth the reduction
constexpr int64_t kSmallCells = 1 << 20;  // lattices up to 101^3: SUMS_1
constexpr int kWarpsMax = 8;
constexpr int kSmemMax = 225 * 1024;  // dynamic shared memory of a block, beside the few static words

// Arithmetic of the sums: FP32 with plain sums of 4 cells, with none, or exact.
enum { SUMS_4 = 0, SUMS_1 = 1, SUMS_EXACT = 2 };
// Separations of one pass over a tile: its sums stay in registers (24 two-word sums
// of 4 separations, or 12 three-word sums of 2).
template <int SUMS> constexpr int chunk_len() { return SUMS == SUMS_EXACT ? 2 : 4; }

__device__ __forceinline__ void stage4(uint32_t dst, const float* src, bool live) {
  // 4-byte asynchronous copy; a pencil past the end reads as zeros
  const int n = live ? 4 : 0;
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}

// a b to three words, every term down to second order.  None may be left out, and no
// remainder of a running sum: a low word rounds what is dropped at 2^-48 of a term, and
// fields whose pencils repeat do so alike in every lane and run (sums of d^4 and d^6
// were off by 1-2e-14 of a sinusoid or a ramp, where FP64 loops leave 0.5-1e-14).
__device__ __forceinline__ Words mul_full(const Words& a, const Words& b) {
  Words c;
  c.h = __fmul_rn(a.h, b.h);
  const float t = __fmaf_rn(a.h, b.h, -c.h);
  const float x1 = __fmul_rn(a.h, b.l), x2 = __fmul_rn(a.l, b.h);
  const float r1 = __fmaf_rn(a.h, b.l, -x1), r2 = __fmaf_rn(a.l, b.h, -x2);
  float y1, y2;
  const float w = two_sum(x1, x2, y1);
  c.l = two_sum(t, w, y2);
  c.m = __fmaf_rn(a.l, b.l, __fmaf_rn(a.h, b.m, __fmaf_rn(a.m, b.h, __fadd_rn(__fadd_rn(r1, r2), __fadd_rn(y1, y2)))));
  return c;
}
__device__ __forceinline__ Words sqr_two(const Words& a) {  // a.m = 0
  Words c;
  c.h = __fmul_rn(a.h, a.h);
  const float t = __fmaf_rn(a.h, a.h, -c.h), a2 = __fadd_rn(a.h, a.h);
  const float x = __fmul_rn(a2, a.l), r = __fmaf_rn(a2, a.l, -x);
  float y;
  c.l = two_sum(t, x, y);
  c.m = __fmaf_rn(a.l, a.l, __fadd_rn(r, y));
  return c;
}
__device__ __forceinline__ Words sqr_full(const Words& a) {
  Words c = sqr_two(a);
  c.m = __fmaf_rn(__fadd_rn(a.h, a.h), a.m, c.m);
  return c;
}

// Running sums of (d, d^2, ..., d^6) of one separation.
struct PowerSums {
  Words s[6];
  __device__ __forceinline__ void reset() {
#pragma unroll
    for (int k = 0; k < 6; ++k) s[k] = {0.f, 0.f, 0.f};
  }
  // d = (a - b) times `scale`, a power of two: exact in two words
  __device__ __forceinline__ void add(float a, float b, float scale) {
    float e;
    const float r = two_sum(a, -b, e);
    const Words d = {__fmul_rn(r, scale), __fmul_rn(e, scale), 0.f};
    const Words q = sqr_two(d), c = mul_full(q, d);
    add_full(s[0], d);
    add_full(s[1], q);
    add_full(s[2], c);
    add_full(s[3], sqr_full(q));
    add_full(s[4], mul_full(c, q));
    add_full(s[5], sqr_full(c));
  }
};

// Sum 24 values over the warp's 32 lanes, value i ending in lane i: each step
// halves the values a lane holds (31 additions instead of 120).  A value is h + l, l
// of run_f32<K>; every remainder is kept, as FP64 additions (slow on this part) would.
template <int K>
__device__ __forceinline__ double warp_sums(const float (&h)[24], const float (&l)[24], int lane) {
  float a[32], b[32];
#pragma unroll
  for (int i = 0; i < 32; ++i) {
    a[i] = i < 24 ? h[i] : 0.f;
    b[i] = i < 24 ? l[i] : 0.f;
  }
#pragma unroll
  for (int s = 16; s > 0; s >>= 1) {
    const bool up = (lane & s) != 0;
#pragma unroll
    for (int i = 0; i < s; ++i) {
      const float send = up ? a[i] : a[i + s], keep = up ? a[i + s] : a[i];
      float e, lo = 0.f;
      a[i] = two_sum(keep, __shfl_xor_sync(0xffffffffu, send, s), e);
      if (s < 16 || K == 1 || i % 2 == 0) lo = (up ? b[i + s] : b[i]) + __shfl_xor_sync(0xffffffffu, up ? b[i] : b[i + s], s);
      b[i] = lo + e;
    }
  }
  // a sum that has left the FP32 range is infinite (or NaN), its remainder NaN
  return fabsf(a[0]) <= FLT_MAX ? (double)a[0] + (double)b[0] : (double)a[0];
}

// The same for the 12 three-word sums of two separations, value i ending in lanes
// 2 i and 2 i + 1, as FP64 (which adds them up only here: 5 slow FP64 operations
// a warp instead of 76).
__device__ __forceinline__ double warp_sums(const PowerSums (&v)[2], int lane) {
  Words a[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) a[i] = i < 12 ? v[i / 6].s[i % 6] : Words{0.f, 0.f, 0.f};
  return to_double(warp_sum16(a, lane));
}
__device__ __forceinline__ double warp_sums(const double (&v)[12], int lane) {
  double a[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) a[i] = i < 12 ? v[i] : 0.0;
  return warp_sum16(a, lane);
}

// Two FP32 values in one 64-bit register, operated on together (add / mul / fma.f32x2:
// one issue slot for two operations, each rounded as the scalar one).
using Pair = unsigned long long;
__device__ __forceinline__ Pair pack2(float x, float y) {
  Pair r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ void unpack2(Pair a, float& x, float& y) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a));
}
__device__ __forceinline__ Pair add2(Pair a, Pair b) {
  Pair r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ Pair mul2(Pair a, Pair b) {
  Pair r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ Pair fma2(Pair a, Pair b, Pair c) {
  Pair r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// Plain FP32 sums span K cells; theirs, hi, keep what an addition rounds away in lo: of
// the odd powers, whose terms cancel over a pencil but not within a run (neighbouring
// increments are alike, so a running sum grows far beyond what is left of it), and with
// K = 1 of the even ones too.  The remainder is exact while |hi| >= |s|, as it is after the
// first of alike increments, and off by no more than the rounding of s itself otherwise.
template <int K>
struct PairSums {
  Pair hi[2][6], lo[2][6];
  static __device__ __forceinline__ constexpr bool keeps(int k) { return K == 1 || k % 2 == 0; }
  __device__ __forceinline__ void reset() {
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int k = 0; k < 6; ++k) hi[j][k] = lo[j][k] = 0ull;
  }
  // The C cells from p on.
  template <int C>
  __device__ __forceinline__ void add(const float* p, const int (&off)[4]) {
    const Pair minus = pack2(-1.f, -1.f);
    Pair s[2][6];
#pragma unroll
    for (int i = 0; i < C; ++i, p += kPitch) {
      const float own = -p[0];
      const Pair own2 = pack2(own, own);
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const Pair d = add2(pack2(p[off[2 * j]], p[off[2 * j + 1]]), own2);
        const Pair q = mul2(d, d), c = mul2(q, d);
        if (i == 0) {
          s[j][0] = d;
          s[j][1] = q;
          s[j][2] = c;
          s[j][3] = mul2(q, q);
          s[j][4] = mul2(c, q);
          s[j][5] = mul2(c, c);
        } else {
          s[j][0] = add2(s[j][0], d);
          s[j][1] = add2(s[j][1], q);
          s[j][2] = fma2(q, d, s[j][2]);
          s[j][3] = fma2(q, q, s[j][3]);
          s[j][4] = fma2(c, q, s[j][4]);
          s[j][5] = fma2(c, c, s[j][5]);
        }
      }
    }
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        const Pair t = add2(hi[j][k], s[j][k]);
        if (keeps(k)) lo[j][k] = add2(lo[j][k], fma2(fma2(hi[j][k], minus, t), minus, s[j][k]));
        hi[j][k] = t;
      }
  }
};

// Sums h + l of one chunk over the run of n cells that starts at p (lane's pencil), two
// separations to a register pair.
template <int K>
__device__ __forceinline__ void run_f32(const float* p, const int (&off)[4], int n, float (&h)[24], float (&l)[24]) {
  PairSums<K> t;
  t.reset();
#pragma unroll (8 / K)
  for (int g = n / K; g > 0; --g, p += K * kPitch) t.template add<K>(p, off);
  for (int i = n % K; i > 0; --i, p += kPitch) t.template add<1>(p, off);
#pragma unroll
  for (int j = 0; j < 2; ++j)
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      unpack2(t.hi[j][k], h[12 * j + k], h[12 * j + 6 + k]);
      if (PairSums<K>::keeps(k)) {
        unpack2(t.lo[j][k], l[12 * j + k], l[12 * j + 6 + k]);
      } else {
        l[12 * j + k] = l[12 * j + 6 + k] = 0.f;
      }
    }
}

// The same in three-word arithmetic, increments times `scale` (a power of two).
__device__ __forceinline__ void run_words(const float* p, const int (&off)[2], int n, float scale, PowerSums (&t)[2]) {
  t[0].reset();
  t[1].reset();
  for (int i = 0; i < n; ++i, p += kPitch) {
    const float own = p[0];
#pragma unroll
    for (int j = 0; j < 2; ++j) t[j].add(p[off[j]], own, scale);
  }
}

// The same in FP64, for tiles outside the range of the three-word arithmetic.
__device__ __noinline__ void run_f64(const float* p, int off0, int off1, int n, double* t) {
  for (int i = 0; i < n; ++i, p += kPitch) {
    const double own = p[0];
    for (int j = 0; j < 2; ++j) {
      const double d = (double)p[j ? off1 : off0] - own;
      double q = d;
      for (int k = 0; k < 6; ++k) {
        t[6 * j + k] += q;
        q *= d;
      }
    }
  }
}

// The exponent k of the tile's scale 2^k: the largest difference of adjacent
// cells times 2^k lies in [2^7, 2^8), so an increment over at most 2^11 cells
// stays below 2^19, its sixth power below 2^114 and a run's sum below 2^120; its
// low parts keep all their bits down to increments 2^-20 of that largest one,
// whose share of a sum is below the FP64 rounding.  INT_MIN when the
// values do not allow it.  adj is zero only when every pencil is constant bit by bit
// (cells_differ): differences below the normal range flush to zero in FP32, not in FP64.
__device__ __forceinline__ int tile_exponent(float adj, float top) {
  if (adj == 0.f && top < 1e30f) return 0;  // every increment is zero
  if (!(adj >= 0x1p-60f && adj < 0x1p60f && top < 0x1p60f)) return INT_MIN;
  const int e = (int)(__float_as_uint(adj) >> 23) - 127;
  const int k = 7 - e;
  const int et = (int)(__float_as_uint(top) >> 23) - 127;
  return et + k < 120 ? k : INT_MIN;
}

// The values differ (zeros of either sign are alike).
__device__ __forceinline__ bool cells_differ(float a, float b) {
  const uint32_t x = __float_as_uint(a), y = __float_as_uint(b);
  return x != y && ((x | y) << 1) != 0u;
}

// Tiles of the three axes in one numbering; a block takes tiles b, b + grid, ...
// partials[block][nr][6].
template <int SUMS>
__global__ void __launch_bounds__(kWarpsMax * 32, 2)
k_struct_tiles(const float* __restrict__ u, StructPlan pl, double* __restrict__ partials) {
  extern __shared__ __align__(16) float tile[];  // [rows][33], then [warps][nr][6] doubles
  __shared__ float s_adj[kWarpsMax], s_top[kWarpsMax];
  constexpr bool EXACT = SUMS == SUMS_EXACT;
  constexpr int CH = chunk_len<SUMS>();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const int nv = 6 * pl.nr;
  double* tot = reinterpret_cast<double*>(tile + pl.rows_max * kPitch);
  double* mine = tot + warp * nv;
  for (int i = lane; i < nv; i += 32) mine[i] = 0.0;
  const uint32_t tile_s = static_cast<uint32_t>(__cvta_generic_to_shared(tile));
  for (int64_t t = blockIdx.x; t < pl.tiles; t += gridDim.x) {
    const int a = t < pl.ax[1].first ? 0 : (t < pl.ax[2].first ? 1 : 2);
    const StructAxis& ax = pl.ax[a];
    const int64_t local = t - ax.first;
    const int64_t ct = local / ax.segs;
    const int i0 = (int)(local - ct * ax.segs) * ax.len;
    const int64_t c0 = ct * kCols;
    const int len = min(ax.len, ax.n - i0), rows = len + ax.halo;
    const float* ua = u + a * pl.ncell;
    __syncthreads();  // the previous tile has been read
    if (a == 0) {     // x-lines: lanes along the line
      for (int c = warp; c < kCols; c += nwarps) {
        const bool live = c0 + c < ax.pencils;
        const float* line = ua + (live ? c0 + c : 0) * ax.n;
        for (int i = lane; i < rows; i += 32) {
          const int x = i0 + i < ax.n ? i0 + i : i0 + i - ax.n;
          if (in_bounds(x >= 0 && x < ax.n && i < pl.rows_max)) stage4(tile_s + 4u * (i * kPitch + c), line + x, live);
        }
      }
    } else {  // pencils across x-lines: lanes along x
      const int64_t c = c0 + lane;
      const bool live = c < ax.pencils;
      // y: pencil (z, x) starts at z ny nx + x; z: pencil (y, x) at its own index
      int64_t base = live ? c : 0;
      if (a == 1) base += base / pl.nx * (pl.plane - pl.nx);
      for (int i = warp; i < rows; i += nwarps) {
        const int k = i0 + i < ax.n ? i0 + i : i0 + i - ax.n;
        const int64_t o = base + k * ax.stride;
        if (in_bounds(o >= 0 && o < pl.ncell && i < pl.rows_max)) stage4(tile_s + 4u * (i * kPitch + lane), ua + o, live);
      }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    int kexp = 0;
    if (EXACT) {
      float adj = 0.f, top = 0.f;
      bool odd = false, moved = false;  // odd: NaN, which fmaxf would drop
      for (int i = warp; i < rows; i += nwarps) {
        const float v = tile[i * kPitch + lane];
        top = fmaxf(top, fabsf(v));
        odd |= !(fabsf(v) < 0x1p60f);
        if (i + 1 < rows) {
          const float w = tile[(i + 1) * kPitch + lane];
          adj = fmaxf(adj, fabsf(w - v));
          moved |= cells_differ(v, w);
        }
      }
      if (odd) top = 0x1p100f;
      if (moved) adj = fmaxf(adj, 0x1p-126f);
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) {
        adj = fmaxf(adj, __shfl_xor_sync(0xffffffffu, adj, off));
        top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, off));
      }
      if (lane == 0) {
        s_adj[warp] = adj;
        s_top[warp] = top;
      }
      __syncthreads();
      for (int w = 0; w < nwarps; ++w) {
        adj = fmaxf(adj, s_adj[w]);
        top = fmaxf(top, s_top[w]);
      }
      kexp = tile_exponent(adj, top);
    }
    const int q = (len + nwarps - 1) / nwarps;
    int n = max(0, min(q, len - warp * q));
    if (!in_bounds(n == 0 || (warp * q + n + ax.halo <= rows && rows <= pl.rows_max))) n = 0;
    const float* p = tile + warp * q * kPitch + lane;
    for (int k0 = 0; k0 < pl.nr; k0 += CH) {
      int off[CH];  // a chunk past the last separation is padded with r = 0: zero increments
#pragma unroll
      for (int j = 0; j < CH; ++j) {
        const int r = k0 + j < pl.nr ? pl.r[a][k0 + j] : 0;
        off[j] = (in_bounds(r >= 0 && r <= ax.halo) ? r : 0) * kPitch;
      }
      if constexpr (EXACT) {
        double v;
        if (kexp == INT_MIN) {
          double d[12];
#pragma unroll
          for (int i = 0; i < 12; ++i) d[i] = 0.0;
          run_f64(p, off[0], off[1], n, d);
          v = warp_sums(d, lane);
        } else {
          PowerSums s[2];
          run_words(p, off, n, __uint_as_float((uint32_t)(kexp + 127) << 23), s);
          v = warp_sums(s, lane);
          // sum of (2^k d)^p: times 2^(-k p)
          if (kexp != 0) v *= __longlong_as_double((long long)(1023 - kexp * ((lane >> 1) % 6 + 1)) << 52);
        }
        const int i = k0 * 6 + (lane >> 1);
        if (!(lane & 1) && lane < 24 && i < nv) mine[i] += v;
      } else {
        float h[24], l[24];
        constexpr int K = SUMS == SUMS_1 ? 1 : 4;
        run_f32<K>(p, off, n, h, l);
        const double v = warp_sums<K>(h, l, lane);
        const int i = k0 * 6 + lane;
        if (lane < 24 && i < nv) mine[i] += v;
      }
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < nv; i += blockDim.x) {
    double s = 0.0;
    for (int w = 0; w < nwarps; ++w) s += tot[w * nv + i];
    partials[(int64_t)blockIdx.x * nv + i] = s;
  }
}

// S_p(r) of one separation in FP64, one cell per thread and pass, partners read
// from global memory: separations whose wrapped distance does not fit a tile.
__global__ void k_struct(const float* __restrict__ u, int nx, int ny, int nz, int r,
                         double* __restrict__ partials, int64_t block_stride) {
  const int64_t n = (int64_t)nx * ny * nz;
  double acc[6] = {0, 0, 0, 0, 0, 0};
  const int rx = r % nx, ry = r % ny, rz = r % nz;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    int x, y, z;
    if (n < (int64_t)0x7fffffff) {  // 32-bit division for lattices below 2^31 cells
      const uint32_t row = (uint32_t)i / (uint32_t)nx;
      x = (int)((uint32_t)i - row * (uint32_t)nx);
      z = (int)(row / (uint32_t)ny);
      y = (int)(row - (uint32_t)z * (uint32_t)ny);
    } else {
      const int64_t row = i / nx;
      x = (int)(i - row * nx);
      z = (int)(row / ny);
      y = (int)(row - (int64_t)z * ny);
    }
    const int xr = x + rx >= nx ? x + rx - nx : x + rx;
    const int yr = y + ry >= ny ? y + ry - ny : y + ry;
    const int zr = z + rz >= nz ? z + rz - nz : z + rz;
    if (!in_bounds(xr >= 0 && xr < nx && yr >= 0 && yr < ny && zr >= 0 && zr < nz)) continue;
    const double d3[3] = {
        (double)u[((int64_t)z * ny + y) * nx + xr] - (double)u[i],
        (double)u[n + ((int64_t)z * ny + yr) * nx + x] - (double)u[n + i],
        (double)u[2 * n + ((int64_t)zr * ny + y) * nx + x] - (double)u[2 * n + i]};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      double p = d3[a];
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        acc[k] += p;
        p *= d3[a];
      }
    }
  }
  __shared__ double red[32][6];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    double v = acc[k];
    for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
    if (lane == 0) red[warp][k] = v;
  }
  __syncthreads();
  if (threadIdx.x < 6) {
    double v = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) v += red[w][threadIdx.x];
    partials[(int64_t)blockIdx.x * block_stride + threadIdx.x] = v;
  }
}

using TilesFn = void (*)(const float*, StructPlan, double*);
TilesFn tiles_fn(const StructPlan& pl, bool exact) {
  if (exact) return k_struct_tiles<SUMS_EXACT>;
  return pl.ncell <= kSmallCells ? k_struct_tiles<SUMS_1> : k_struct_tiles<SUMS_4>;
}

cudaError_t finish_plan(StructPlan& pl, bool exact, int max_blocks, int sms) {
  const TilesFn fn = tiles_fn(pl, exact);
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax);
  int per_sm = 0;
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, pl.threads, pl.smem);
  if (e == cudaSuccess && per_sm < 1) e = cudaErrorInvalidConfiguration;
  if (e == cudaSuccess)
    pl.grid = (int)std::max<int64_t>(1, std::min<int64_t>({pl.tiles, (int64_t)per_sm * sms, (int64_t)max_blocks}));
  return e;
}

}  // namespace

bool plan_struct(int nx, int ny, int nz, const int* r, int nr, bool exact, int max_blocks, StructPlan* out,
                 cudaError_t* err) {
  *err = cudaErrorInvalidValue;
  if (nr < 1 || nr > kMaxStructSeps) return false;
  StructPlan pl{};
  const int n[3] = {nx, ny, nz};
  pl.nr = nr;
  pl.nx = nx;
  pl.plane = (int64_t)nx * ny;
  pl.ncell = pl.plane * nz;
  int longest = 0, halo = 0;
  for (int a = 0; a < 3; ++a) {
    for (int k = 0; k < nr; ++k) {
      pl.r[a][k] = r[k] % n[a];
      pl.ax[a].halo = std::max(pl.ax[a].halo, pl.r[a][k]);
    }
    longest = std::max(longest, n[a]);
    halo = std::max(halo, pl.ax[a].halo);
  }
  const size_t sums = sizeof(double) * 6 * nr;
  // Blocks of 4 warps where six or more of them fit an SM (its pencils up to
  // ~250 cells with their halo): a lane's run is then long against the warp
  // reduction that ends it.  Longer pencils get 8 warps, so that the two
  // blocks an SM has room for still fill it.  A pencil is cut into segments of
  // at most kRunMax cells per warp.
  const int short_rows = std::min(longest, 4 * kRunMax) + halo;
  const int warps = longest <= 4 * kRunMax && (size_t)short_rows * kPitch * 4 + 4 * sums <= 36 * 1024 ? 4 : kWarpsMax;
  auto cut = [&](int64_t least) {  // into `least` tiles an axis or more, runs of kRunMin cells or more
    int64_t tiles = 0;
    pl.rows_max = 0;
    for (int a = 0; a < 3; ++a) {
      StructAxis& ax = pl.ax[a];
      ax.n = n[a];
      ax.stride = a == 0 ? 1 : (a == 1 ? (int64_t)nx : pl.plane);
      ax.pencils = pl.ncell / n[a];
      const int64_t cols = (ax.pencils + kCols - 1) / kCols;
      ax.segs = std::max((n[a] + warps * kRunMax - 1) / (warps * kRunMax),
                         (int)std::min<int64_t>(least / cols, n[a] / (warps * kRunMin)));
      ax.len = (n[a] + ax.segs - 1) / ax.segs;
      ax.segs = (n[a] + ax.len - 1) / ax.len;
      ax.first = tiles;
      tiles += cols * ax.segs;
      pl.rows_max = std::max(pl.rows_max, ax.len + ax.halo);
    }
    pl.rows_max += pl.rows_max & 1;  // the FP64 sums behind the tile start on 8 bytes
    pl.tiles = tiles;
    return (size_t)pl.rows_max * kPitch * 4 + warps * sums;
  };
  size_t smem = cut(0);
  pl.threads = 32 * warps;
  *err = cudaSuccess;
  // an increment spans at most 2^11 cells (tile_exponent)
  if (smem > (size_t)kSmemMax || pl.rows_max > 2048) return false;
  int dev = 0, sms = 0;
  *err = cudaGetDevice(&dev);
  if (*err == cudaSuccess) *err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (*err != cudaSuccess) return false;
  // Exact sums: a long box has few pencils along its length, whose tiles of 8 x 64 cells
  // would keep a few SMs busy for long (2000 x 2 x 2, 24 separations: 456 us in 4 tiles).
  // Shorter segments give every SM one.
  if (exact) smem = cut(sms);
  pl.smem = (int)smem;
  *err = finish_plan(pl, exact, max_blocks, sms);
  *out = pl;
  return *err == cudaSuccess;
}

cudaError_t launch_struct_plan(const float* u, const StructPlan& pl, bool exact, double* partials, cudaStream_t st) {
  return launch_kernel(tiles_fn(pl, exact), pl.grid, pl.threads, pl.smem, st, u, pl, partials);
}

cudaError_t launch_struct(const float* u, int nx, int ny, int nz, int r, double* partials,
                          int blocks, cudaStream_t st, int64_t block_stride) {
  return launch_kernel(k_struct, blocks, 256, 0, st, u, nx, ny, nz, r, partials, block_stride);
}

uint32_t bounds_word_struct() { return take_bounds_word(); }

}  // namespace lbm
