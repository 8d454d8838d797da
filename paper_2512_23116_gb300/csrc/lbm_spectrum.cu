// Energy spectrum: transform of the velocity and shell sums of |u_hat|^2
// (Eq. integral_length_scale, integer shells s - 1/2 <= |k| < s + 1/2).
//
// The transform is done here, not by a library, because only the shell sums are
// wanted: three passes, z (real to half spectrum), y (in place), x, and the last
// adds its modes to the shells straight from shared memory instead of writing
// them.  20 bytes of traffic per cell and component; the library's transform
// followed by a binning pass moves 28.  Three components, transform and shells:
// 100^3 73 -> 38 us, 400^3 3.68 -> 1.40 ms, 800^3 37.6 -> 11.6 ms.  A pass is bound
// by issue (67 % of the issue slots at 320^3: ~90 instructions a point, two thirds of them the
// stages) with its DRAM traffic at 60 % of the copy bandwidth.
//
// A tile is W columns by the whole extent in shared memory.  The z pass packs two
// neighbouring real columns into one complex column (their spectra separate by
// Hermitian symmetry), so a row of a tile is W x 8 contiguous bytes in every
// strided pass; the x pass comes last because it reads contiguous lines and
// writes nothing.  Stages are decimation in frequency, in place: a butterfly
// of radix R reads R rows into registers, multiplies by the twiddles (a table in
// shared memory, rounded from FP64) and writes the same rows back, one
// barrier per stage; the frequency order that leaves is undone by a table of row
// numbers when the rows are used.  Radices 10, 8, 6, 5, 4, 3, 2 in 64 registers (16
// would need 120 and halve the warps that hide the loads), and 13, 11, 7 by the definition in
// kernels of their own, chosen for the fewest stages.  Extents with larger prime
// factors go to cuFFT and k_bin_lines.
//
// Shells: along a line the shell of a mode never falls and never skips one, so a
// thread walks a run of modes of one line and stores the running sum of the
// current shell at its place in a table [shell][line] in shared memory: no search, no
// atomics, every mode read once; the table's rows then add up to the block's FP64
// totals.  In k_bin_lines 132 us per component at 404^3 for 265 MB of modes (40 us at
// the copy bandwidth); adding to shells with FP64 atomics in shared memory took 443 us at
// 400^3, a lane per shell gathering its intervals of modes by their square roots 170-200.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "lbm_check.cuh"
#include "lbm_kernels.h"
#include "lbm_spectrum.h"
#include "lbm_words.cuh"

namespace lbm {

namespace {

constexpr int kFftThreads = 512, kBinThreads = 256;
constexpr int kEnergies = 16;  // modes |kx| a thread of the x pass holds at once
constexpr int kSmemLimit = 225 * 1024;
constexpr int kBinWidth = 16, kBinChunk = 512;  // lines and modes of a line in a k_bin_lines tile

enum { PASS_X = 0, PASS_Y = 1, PASS_Z = 2 };

// ---- butterflies: forward DFT of R values, natural order in and out ---------------

__device__ __forceinline__ float2 operator+(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 operator-(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 mul_mi(float2 a) { return make_float2(a.y, -a.x); }  // -i a

template <int R> struct Dft;
template <> struct Dft<2> {
  static __device__ __forceinline__ void run(float2 (&x)[2]) {
    const float2 a = x[0], b = x[1];
    x[0] = a + b;
    x[1] = a - b;
  }
};
template <> struct Dft<3> {
  static __device__ __forceinline__ void run(float2 (&x)[3]) {
    constexpr float s = 0.866025403784438647f;  // sin 60
    const float2 t = x[1] + x[2], d = x[1] - x[2];
    const float2 m = make_float2(fmaf(-0.5f, t.x, x[0].x), fmaf(-0.5f, t.y, x[0].y));
    x[0] = x[0] + t;
    x[1] = make_float2(fmaf(s, d.y, m.x), fmaf(-s, d.x, m.y));
    x[2] = make_float2(fmaf(-s, d.y, m.x), fmaf(s, d.x, m.y));
  }
};
template <> struct Dft<4> {
  static __device__ __forceinline__ void run(float2 (&x)[4]) {
    const float2 a = x[0] + x[2], b = x[0] - x[2], c = x[1] + x[3], d = mul_mi(x[1] - x[3]);
    x[0] = a + c;
    x[1] = b + d;
    x[2] = a - c;
    x[3] = b - d;
  }
};
template <> struct Dft<5> {
  static __device__ __forceinline__ void run(float2 (&x)[5]) {
    constexpr float c1 = 0.309016994374947424f, c2 = -0.809016994374947424f;  // cos 72, cos 144
    constexpr float s1 = 0.951056516295153572f, s2 = 0.587785252292473129f;   // sin 72, sin 144
    const float2 t1 = x[1] + x[4], t2 = x[2] + x[3], d1 = x[1] - x[4], d2 = x[2] - x[3];
    const float2 a = make_float2(fmaf(c1, t1.x, fmaf(c2, t2.x, x[0].x)), fmaf(c1, t1.y, fmaf(c2, t2.y, x[0].y)));
    const float2 b = make_float2(fmaf(c2, t1.x, fmaf(c1, t2.x, x[0].x)), fmaf(c2, t1.y, fmaf(c1, t2.y, x[0].y)));
    const float2 e = make_float2(fmaf(s1, d1.x, s2 * d2.x), fmaf(s1, d1.y, s2 * d2.y));
    const float2 f = make_float2(fmaf(s2, d1.x, -s1 * d2.x), fmaf(s2, d1.y, -s1 * d2.y));
    x[0] = x[0] + (t1 + t2);
    x[1] = a + mul_mi(e);
    x[2] = b + mul_mi(f);
    x[3] = b - mul_mi(f);
    x[4] = a - mul_mi(e);
  }
};
// coprime factors (Good-Thomas): n = N2 n1 + N1 n2, k by the remainders, no twiddles
template <> struct Dft<6> {
  static __device__ __forceinline__ void run(float2 (&x)[6]) {
    float2 y[2][3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const float2 a = x[(2 * j) % 6], b = x[(2 * j + 3) % 6];
      y[0][j] = a + b;
      y[1][j] = a - b;
    }
    Dft<3>::run(y[0]);
    Dft<3>::run(y[1]);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      x[(4 * j) % 6] = y[0][j];
      x[(4 * j + 3) % 6] = y[1][j];
    }
  }
};
template <> struct Dft<10> {
  static __device__ __forceinline__ void run(float2 (&x)[10]) {
    float2 y[2][5];
#pragma unroll
    for (int j = 0; j < 5; ++j) {
      const float2 a = x[(2 * j) % 10], b = x[(2 * j + 5) % 10];
      y[0][j] = a + b;
      y[1][j] = a - b;
    }
    Dft<5>::run(y[0]);
    Dft<5>::run(y[1]);
#pragma unroll
    for (int j = 0; j < 5; ++j) {
      x[(6 * j) % 10] = y[0][j];
      x[(6 * j + 5) % 10] = y[1][j];
    }
  }
};
template <> struct Dft<8> {
  static __device__ __forceinline__ void run(float2 (&x)[8]) {
    constexpr float h = 0.707106781186547524f;
    float2 e[4] = {x[0], x[2], x[4], x[6]}, o[4] = {x[1], x[3], x[5], x[7]};
    Dft<4>::run(e);
    Dft<4>::run(o);
    o[1] = make_float2(h * (o[1].x + o[1].y), h * (o[1].y - o[1].x));
    o[2] = mul_mi(o[2]);
    o[3] = make_float2(h * (o[3].y - o[3].x), -h * (o[3].x + o[3].y));
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      x[k] = e[k] + o[k];
      x[k + 4] = e[k] - o[k];
    }
  }
};
// One decimation-in-frequency stage i: rows base + j + q m, q < R, of sub-transforms of
// R m rows.  tw: exp(-2 pi i k / n).
template <int R, int P>
__device__ __forceinline__ void stage(float2* s, const float2* tw, const FftAxis& ax, int i, int done, int col, int g,
                                      int groups) {
  const int m = ax.m[i], count = m * done, dj = ax.dj[i], db = ax.db[i];
  int blk = (int)(((float)g + 0.5f) * ax.inv_m[i]), j = g - blk * m;
  for (int b = g; b < count; b += groups) {
    if (in_bounds(blk >= 0 && j >= 0 && blk * R * m + j + (R - 1) * m < ax.n && (R - 1) * j * done < ax.n)) {
      float2* p = s + (blk * R * m + j) * P + col;
      float2 x[R];
#pragma unroll
      for (int q = 0; q < R; ++q) x[q] = p[q * m * P];
      Dft<R>::run(x);
      p[0] = x[0];
      if (m > 1) {
        const int step = j * done;
#pragma unroll
        for (int q = 1; q < R; ++q) p[q * m * P] = cmul(x[q], tw[q * step]);
      } else {
#pragma unroll
        for (int q = 1; q < R; ++q) p[q * P] = x[q];
      }
    }
    j += dj;
    blk += db;
    if (j >= m) {
      j -= m;
      ++blk;
    }
  }
}

// The same for an odd prime R by the definition, real and imaginary parts of the
// pairs x_m, x_{R-m} sharing their products; cos and sin of 2 pi k / R from the table.
template <int R, int P>
__device__ __forceinline__ void stage_prime(float2* s, const float2* tw, const FftAxis& ax, int i, int done, int col,
                                            int g, int groups) {
  const int m = ax.m[i], count = m * done, n = ax.n;
  for (int b = g; b < count; b += groups) {
    const int blk = b / m, j = b - blk * m;
    if (!in_bounds(blk * R * m + j + (R - 1) * m < n && (R - 1) * j * done < n)) continue;
    float2* p = s + (blk * R * m + j) * P + col;
    const float2 x0 = p[0];
    float2 t[R / 2], d[R / 2];
    float2 sum = x0;
#pragma unroll
    for (int q = 1; q <= R / 2; ++q) {
      const float2 a = p[q * m * P], c = p[(R - q) * m * P];
      t[q - 1] = a + c;
      d[q - 1] = a - c;
      sum = sum + t[q - 1];
    }
    p[0] = sum;
#pragma unroll
    for (int k = 1; k <= R / 2; ++k) {
      float2 a = x0, e = make_float2(0.f, 0.f);
#pragma unroll
      for (int q = 1; q <= R / 2; ++q) {
        const float2 w = tw[(q * k % R) * (n / R)];  // cos, -sin
        a = make_float2(fmaf(w.x, t[q - 1].x, a.x), fmaf(w.x, t[q - 1].y, a.y));
        e = make_float2(fmaf(-w.y, d[q - 1].x, e.x), fmaf(-w.y, d[q - 1].y, e.y));
      }
      const float2 f = mul_mi(e);
      p[k * m * P] = cmul(a + f, tw[j * k * done]);
      p[(R - k) * m * P] = cmul(a - f, tw[j * (R - k) * done]);
    }
  }
}

template <int P, bool PRIMES>
__device__ __forceinline__ void transform(float2* s, const float2* tw, const FftAxis& ax, int col, int g, int groups) {
  int done = 1;  // product of the earlier radices
  for (int i = 0; i < ax.stages; ++i) {
    const int R = ax.radix[i];
    if constexpr (PRIMES) {
      switch (R) {
        case 7: stage_prime<7, P>(s, tw, ax, i, done, col, g, groups); break;
        case 11: stage_prime<11, P>(s, tw, ax, i, done, col, g, groups); break;
        case 13: stage_prime<13, P>(s, tw, ax, i, done, col, g, groups); break;
      }
    }
    switch (R) {
      case 2: stage<2, P>(s, tw, ax, i, done, col, g, groups); break;
      case 3: stage<3, P>(s, tw, ax, i, done, col, g, groups); break;
      case 4: stage<4, P>(s, tw, ax, i, done, col, g, groups); break;
      case 5: stage<5, P>(s, tw, ax, i, done, col, g, groups); break;
      case 6: stage<6, P>(s, tw, ax, i, done, col, g, groups); break;
      case 8: stage<8, P>(s, tw, ax, i, done, col, g, groups); break;
      case 10: stage<10, P>(s, tw, ax, i, done, col, g, groups); break;
    }
    done *= R;
    __syncthreads();
  }
}

// Row that holds frequency k after the stages: its digits in the radices, the first
// stage's digit the slowest.
__device__ __forceinline__ int row_of(const FftAxis& ax, int k) {
  int len = ax.n, row = 0;
  for (int i = 0; i < ax.stages; ++i) {
    const int R = ax.radix[i], q = k % R;
    k /= R;
    len /= R;
    row += q * len;
  }
  return row;
}

__device__ __forceinline__ void copy_async8(uint32_t dst, const void* src, bool live) {
  const int n = live ? 8 : 0;
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void copy_async4(uint32_t dst, const void* src, bool live) {
  const int n = live ? 4 : 0;
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void copies_landed() { asm volatile("cp.async.wait_all;" ::: "memory"); }

__device__ __forceinline__ int floor_sqrt(int v) {  // v >= 0; sqrtf is within one of the integer root
  int r = (int)sqrtf((float)v);
  if (r * r > v) --r;
  if ((r + 1) * (r + 1) <= v) ++r;
  return r;
}

// k_1^2 + k_2^2 of a line, clamped where it exceeds every counted shell.
__device__ __forceinline__ int line_p(int64_t a, int64_t b, int kmax) {
  const int64_t p = a * a + b * b, top = (int64_t)(kmax + 1) * (kmax + 1);
  return (int)(p < top ? p : top);
}

// Exact integer shell of K: s with s^2 - s < K <= s^2 + s (s = 0 for K = 0).
__device__ __forceinline__ int shell_of(int K) {
  const int r = floor_sqrt(K);
  return K > r * r + r ? r + 1 : r;
}

// Shared-memory scratch of add_shells for W lines of at most nk modes.
template <int W>
struct ShellTile {
  float* run;    // [nk][W + 1]: a line's shells, from its first one
  float* carry;  // [threads]
  int* carry_at; // [threads]
  int* first;    // [W], [W]: a line's first and last shell
  int* last;
  static __host__ __device__ constexpr size_t bytes(int nk, int threads) {
    return sizeof(float) * ((size_t)nk * (W + 1) + 2 * (size_t)threads + 2 * W);
  }
  __device__ __forceinline__ ShellTile(float* at, int nk)
      : run(at),
        carry(at + nk * (W + 1)),
        carry_at(reinterpret_cast<int*>(carry + blockDim.x)),
        first(carry_at + blockDim.x),
        last(first + W) {}
};

// Add the modes |kx| in [k0, k0 + nk) of W lines to the shells 0..kmax; lp[c], lw[c]:
// line c's p (INT32_MAX: no line) and weight.  Thread (col, g) walks the L modes from k0
// + g L of line col with the energies e(i).  sqrt(p + k^2) grows by less than one
// per mode, so a line's shells follow one another without a gap: the running sum of the
// current shell is simply stored at its place.  A shell that began in the run of
// the thread before goes through `carry`.  Sums keep their remainders: what a line
// gives a shell is rounded to FP32 once where it is stored (and once more with a
// carry), the lines of a tile add up in two words.  Ends without a barrier.
template <int W, int L, typename E>
__device__ __forceinline__ void add_shells(const E& e, int k0, int nk, int per, int col, int g, int groups, const int* lp,
                                           const float* lw, const ShellTile<W>& t, int kmax, double* shells) {
  const int p = lp[col], kb = k0 + g * per, ke = min(kb + per, k0 + nk);
  int at = -1;
  if (p != INT32_MAX && kb < ke) {
    const int base = shell_of(p + k0 * k0);
    int K = p + kb * kb, s = shell_of(K), top = s * s + s;
    bool first = kb > k0 && shell_of(K - 2 * kb + 1) == s;
    if (first) at = s - base;
    float run = 0.f, low = 0.f, held = 0.f;
    float* r = t.run + (s - base) * (W + 1) + col;
#pragma unroll
    for (int i = 0; i < L; ++i) {
      const int k = kb + i;
      if (k < ke) {
        if (K > top) {
          if (first) held = run + low;
          first = false;
          run = low = 0.f;
          ++s;
          top += 2 * s;
          r += W + 1;
        }
        float err;
        run = two_sum(run, e(i), err);
        low += err;
        if (!first && in_bounds(s >= base && s - base < nk)) *r = run + low;
        K += 2 * k + 1;
      }
    }
    t.carry[g * W + col] = first ? run + low : held;
  }
  t.carry_at[g * W + col] = at;
  if (g == 0) {
    t.first[col] = p == INT32_MAX ? INT32_MAX : shell_of(p + k0 * k0);
    t.last[col] = p == INT32_MAX ? -1 : shell_of(p + (k0 + nk - 1) * (k0 + nk - 1));
  }
  __syncthreads();
  // carries: the first of those that go to one shell adds them all
  if (at >= 0 && in_bounds(at < nk) && (g == 1 || t.carry_at[(g - 1) * W + col] != at)) {
    float v = t.carry[g * W + col], low = 0.f, err;
    for (int h = g + 1; h < groups && t.carry_at[h * W + col] == at; ++h) {
      v = two_sum(v, t.carry[h * W + col], err);
      low += err;
    }
    t.run[at * (W + 1) + col] += v + low;
  }
  __syncthreads();
  int s0 = INT32_MAX, s1 = -1;
#pragma unroll
  for (int c = 0; c < W; ++c) {
    s0 = min(s0, t.first[c]);
    s1 = max(s1, t.last[c]);
  }
  s1 = min(s1, kmax);
  for (int s = s0 + (int)threadIdx.x; s <= s1; s += blockDim.x) {
    float acc = 0.f, low = 0.f, err;
#pragma unroll
    for (int c = 0; c < W; ++c)
      if (s >= t.first[c] && s <= t.last[c] && in_bounds(s - t.first[c] < nk)) {
        acc = two_sum(acc, lw[c] * t.run[(s - t.first[c]) * (W + 1) + c], err);  // lw is 0, 1 or 2: exact
        low += err;
      }
    shells[s] += (double)acc + (double)low;
  }
}

struct FftArgs {
  const float* u;      // PASS_Z: real input, `comps` components
  float2* work;        // [comps][nz/2 + 1][ny][nx]
  const float2* tw;    // this axis's table
  FftAxis ax;
  int nx, ny, nz, comps, kmax;
  int tile;            // complex values of the tile (or of the scratch it becomes)
  int64_t ncell, half, cols, tiles_per_comp;  // cols: columns of a component in this pass
  double* partials;    // PASS_X
};

template <int PASS, int W, bool PRIMES>
__global__ void __launch_bounds__(kFftThreads, PRIMES ? 1 : 2) k_fft_pass(FftArgs a) {
  constexpr int P = PASS == PASS_X ? W + 1 : W;  // x: lanes along a line store without conflicts
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int n = a.ax.n;
  // shells first (8-byte values), then the tile, the twiddles, the row numbers, the lines' p and weight
  double* shells = reinterpret_cast<double*>(smem_raw);
  float2* s = reinterpret_cast<float2*>(smem_raw + (PASS == PASS_X ? sizeof(double) * (size_t)(a.kmax + 1) : 0));
  float2* tw = s + a.tile;
  int* lp = reinterpret_cast<int*>(tw + n);
  float* lw = reinterpret_cast<float*>(lp + W);
  uint16_t* row = reinterpret_cast<uint16_t*>(lw + W);
  const uint32_t s_addr = static_cast<uint32_t>(__cvta_generic_to_shared(s));
  const int tid = threadIdx.x, col = tid % W, g = tid / W, groups = blockDim.x / W;
  for (int k = tid; k < n; k += blockDim.x) {
    tw[k] = a.tw[k];
    const int r = row_of(a.ax, k);
    row[k] = (uint16_t)(in_bounds(r >= 0 && r < n) ? r : 0);
  }
  if (PASS == PASS_X)
    for (int k = tid; k <= a.kmax; k += blockDim.x) shells[k] = 0.0;
  const int64_t plane = (int64_t)a.nx * a.ny;
  for (int64_t t = blockIdx.x; t < a.tiles_per_comp * a.comps; t += gridDim.x) {
    const int64_t comp = t / a.tiles_per_comp, c0 = (t - comp * a.tiles_per_comp) * W;
    float2* work = a.work + comp * a.half;
    __syncthreads();  // the previous tile has been used
    const int64_t c = c0 + col;
    const bool live = c < a.cols;
    int64_t base = 0;
    if (PASS == PASS_X) {  // lines (kz, ky); lanes along a line
      const int lane = tid & 31;
      for (int l = tid >> 5; l < W; l += blockDim.x >> 5) {
        const bool ok = c0 + l < a.cols;
        const float2* src = work + (ok ? c0 + l : 0) * n;
        for (int x = lane; x < n; x += 32)
          if (in_bounds(src + x >= work && src + x < work + a.half)) copy_async8(s_addr + 8u * (uint32_t)(x * P + l), src + x, ok);
      }
      if (tid < W) {
        const int kz = (int)(c / a.ny), ky = (int)(c - (int64_t)kz * a.ny);
        lp[tid] = live ? line_p(min(ky, a.ny - ky), kz, a.kmax) : INT32_MAX;
        lw[tid] = !live ? 0.f : (kz == 0 || 2 * kz == a.nz ? 1.f : 2.f);
      }
    } else if (PASS == PASS_Y) {  // columns (kz, x)
      const int64_t kz = live ? c / a.nx : 0;
      base = live ? kz * plane + (c - kz * a.nx) : 0;
      for (int i = g; i < n; i += groups) {
        const int64_t o = base + (int64_t)i * a.nx;
        if (in_bounds(o >= 0 && o < a.half)) copy_async8(s_addr + 8u * (uint32_t)(i * P + col), work + o, live);
      }
    } else {  // pairs of columns 2 c, 2 c + 1 of the plane
      base = live ? 2 * c : 0;
      const float* u = a.u + comp * a.ncell;
      if ((plane & 1) == 0) {
        for (int i = g; i < n; i += groups) {
          const int64_t o = base + i * plane;
          if (in_bounds(o >= 0 && o + 1 < a.ncell)) copy_async8(s_addr + 8u * (uint32_t)(i * P + col), u + o, live);
        }
      } else {  // planes start at odd offsets, and the last column has no partner
        const bool two = live && base + 1 < plane;
        for (int i = g; i < n; i += groups) {
          const int64_t o = base + i * plane;
          if (in_bounds(o >= 0 && o < a.ncell)) {
            copy_async4(s_addr + 8u * (uint32_t)(i * P + col), u + o, live);
            copy_async4(s_addr + 8u * (uint32_t)(i * P + col) + 4u, u + (two ? o + 1 : o), two);
          }
        }
      }
    }
    copies_landed();
    __syncthreads();
    transform<P, PRIMES>(s, tw, a.ax, col, g, groups);
    if (PASS == PASS_X) {
      // energies of kx and -kx together, taken from the tile before it becomes scratch
      float e[kEnergies];
      const int nk = n / 2 + 1, per = (nk + groups - 1) / groups;
#pragma unroll
      for (int i = 0; i < kEnergies; ++i) {
        const int k = g * per + i;
        if (i < per && k < nk) {
          const float2 v = s[row[k] * P + col];
          e[i] = fmaf(v.x, v.x, v.y * v.y);
          if (k > 0 && 2 * k != n) {
            const float2 w = s[row[n - k] * P + col];
            e[i] = fmaf(w.x, w.x, fmaf(w.y, w.y, e[i]));
          }
        }
      }
      __syncthreads();
      add_shells<W, kEnergies>([&](int i) { return e[i]; }, 0, nk, per, col, g, groups, lp, lw,
                               ShellTile<W>(reinterpret_cast<float*>(s), nk), a.kmax, shells);
    } else if (PASS == PASS_Y) {
      if (live)
        for (int k = g; k < n; k += groups) {
          const int64_t o = base + (int64_t)k * a.nx;
          if (in_bounds(o >= 0 && o < a.half)) work[o] = s[row[k] * P + col];
        }
    } else if (live) {
      // A = (Z_k + conj Z_-k) / 2, B = (Z_k - conj Z_-k) / 2i
      const bool even = (plane & 1) == 0, two = base + 1 < plane;
      for (int k = g; k <= n / 2; k += groups) {
        const float2 z = s[row[k] * P + col], w = s[row[k == 0 ? 0 : n - k] * P + col];
        const float2 A = make_float2(0.5f * (z.x + w.x), 0.5f * (z.y - w.y));
        const float2 B = make_float2(0.5f * (z.y + w.y), 0.5f * (w.x - z.x));
        const int64_t o = base + k * plane;
        if (!in_bounds(o >= 0 && o + (two ? 1 : 0) < a.half)) continue;
        if (even) {
          *reinterpret_cast<float4*>(work + o) = make_float4(A.x, A.y, B.x, B.y);
        } else {
          work[o] = A;
          if (two) work[o + 1] = B;
        }
      }
    }
  }
  if (PASS == PASS_X) {
    __syncthreads();
    for (int k = tid; k <= a.kmax; k += blockDim.x) a.partials[(int64_t)blockIdx.x * (a.kmax + 1) + k] += shells[k];
  }
}

// Shell sums of a kx-half spectrum [nz][ny][nx/2 + 1] (cuFFT's order): tiles of
// kBinWidth lines by at most kBinChunk modes.
__global__ void __launch_bounds__(kBinThreads, 4)
k_bin_lines(const float2* __restrict__ c, int nx, int ny, int nz, int kmax, double* __restrict__ partials) {
  constexpr int W = kBinWidth;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int nxh = nx / 2 + 1, chunk = min(nxh, kBinChunk);
  double* shells = reinterpret_cast<double*>(smem_raw);
  float* e = reinterpret_cast<float*>(shells + kmax + 1);
  const ShellTile<W> scratch(e + chunk * (W + 1), chunk);
  int* lp = scratch.last + W;
  float* lw = reinterpret_cast<float*>(lp + W);
  const int tid = threadIdx.x, lane = tid & 31;
  for (int k = tid; k <= kmax; k += blockDim.x) shells[k] = 0.0;
  const int64_t lines = (int64_t)ny * nz, tiles = (lines + W - 1) / W;
  for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
    for (int k0 = 0; k0 < nxh; k0 += chunk) {
      const int m = min(chunk, nxh - k0);
      __syncthreads();
      for (int l = tid >> 5; l < W; l += blockDim.x >> 5) {
        const bool ok = t * W + l < lines;
        const float2* src = c + (ok ? t * W + l : 0) * nxh + k0;
#pragma unroll 4
        for (int x = lane; x < m; x += 32) {
          const float2 v = in_bounds(src + x >= c && src + x < c + lines * nxh) ? src[x] : make_float2(0.f, 0.f);
          const float w = k0 + x == 0 || 2 * (k0 + x) == nx ? 1.f : 2.f;  // kx and -kx
          e[x * (W + 1) + l] = w * fmaf(v.x, v.x, v.y * v.y);
        }
      }
      if (tid < W) {
        const int64_t l = t * W + tid;
        const int64_t kz = l / ny, ky = l - kz * ny;
        const bool ok = l < lines;
        lp[tid] = ok ? line_p(min(ky, ny - ky), min(kz, nz - kz), kmax) : INT32_MAX;
        lw[tid] = ok ? 1.f : 0.f;
      }
      __syncthreads();
      const int groups = blockDim.x / W, col = tid % W, g = tid / W, per = (m + groups - 1) / groups;
      const float* mine = e + g * per * (W + 1) + col;
      add_shells<W, kBinChunk * W / kBinThreads>([&](int i) { return mine[i * (W + 1)]; }, k0, m, per, col, g, groups, lp,
                                                 lw, scratch, kmax, shells);
    }
  }
  __syncthreads();
  for (int k = tid; k <= kmax; k += blockDim.x) partials[(int64_t)blockIdx.x * (kmax + 1) + k] += shells[k];
}

size_t bin_smem(int nx, int kmax) {
  return sizeof(double) * (size_t)(kmax + 1) + sizeof(float) * (size_t)std::min(nx / 2 + 1, kBinChunk) * (kBinWidth + 1) +
         ShellTile<kBinWidth>::bytes(std::min(nx / 2 + 1, kBinChunk), kBinThreads) + 8 * kBinWidth;
}

// Fewest stages, then the smallest sum of radices.
bool factor(int n, FftAxis* out) {
  static const int radices[] = {13, 11, 10, 8, 7, 6, 5, 4, 3, 2};
  FftAxis best{}, cur{};
  best.stages = kMaxStages + 1;
  int best_sum = 0;
  auto rec = [&](auto&& self, int m, int at, int sum) -> void {
    if (m == 1) {
      if (cur.stages < best.stages || (cur.stages == best.stages && sum < best_sum)) {
        best = cur;
        best_sum = sum;
      }
      return;
    }
    if (cur.stages >= kMaxStages || cur.stages + 1 > best.stages) return;
    for (int i = at; i < (int)(sizeof radices / sizeof *radices); ++i)
      if (m % radices[i] == 0) {
        cur.radix[cur.stages++] = radices[i];
        self(self, m / radices[i], i, sum + radices[i]);
        --cur.stages;
      }
  };
  rec(rec, n, 0, 0);
  if (best.stages > kMaxStages) return false;
  *out = best;
  out->n = n;
  return true;
}

using PassFn = void (*)(FftArgs);
template <int PASS>
PassFn pass_fn(int width, bool primes) {
  if (primes) return width == 16 ? k_fft_pass<PASS, 16, true> : k_fft_pass<PASS, 8, true>;
  return width == 16 ? k_fft_pass<PASS, 16, false> : k_fft_pass<PASS, 8, false>;
}
PassFn pass_fn(int pass, const FftPlan& pl) {
  const FftAxis& ax = pl.ax[pass];
  bool primes = false;
  for (int i = 0; i < ax.stages; ++i) primes |= ax.radix[i] == 7 || ax.radix[i] > 10;
  const int w = pl.width[pass];
  return pass == PASS_X ? pass_fn<PASS_X>(w, primes) : (pass == PASS_Y ? pass_fn<PASS_Y>(w, primes) : pass_fn<PASS_Z>(w, primes));
}

}  // namespace

bool plan_fft(int nx, int ny, int nz, int kmax, FftPlan* out, cudaError_t* err) {
  *err = cudaSuccess;
  FftPlan pl{};
  const int n[3] = {nx, ny, nz};
  if (kmax >= kMaxShells) return false;
  pl.half = (int64_t)(nz / 2 + 1) * ny * nx;
  int dev = 0, sms = 0;
  for (int a = 0; a < 3; ++a) {
    if (n[a] > 65535 || !factor(n[a], &pl.ax[a])) return false;
    // 16 columns (rows of 128 bytes) while two blocks of them fit an SM, else 8
    auto tile = [&](int w) {
      return std::max((size_t)n[a] * (w + (a == PASS_X)),
                      a == PASS_X ? (ShellTile<16>::bytes(n[a] / 2 + 1, kFftThreads) + 7) / 8 : (size_t)0);
    };
    auto bytes = [&](int w) {
      return (size_t)(a == PASS_X ? sizeof(double) * (kmax + 1) : 0) + sizeof(float2) * tile(w) +
             sizeof(float2) * (size_t)n[a] + 8 * w + 2 * (size_t)n[a];
    };
    pl.width[a] = bytes(16) <= 113 * 1024 ? 16 : 8;
    const size_t smem = bytes(pl.width[a]);
    if (smem > (size_t)kSmemLimit) return false;
    pl.smem[a] = (int)smem;
    pl.tile[a] = (int)tile(pl.width[a]);
    // as many threads as a stage has butterflies, in whole warps, and no more than
    // fill the SM with the blocks that its shared memory takes
    int most = 1;
    for (int i = 0; i < pl.ax[a].stages; ++i) most = std::max(most, n[a] / pl.ax[a].radix[i]);
    const int want = (most * pl.width[a] + 31) / 32 * 32, per_block = smem > 56 * 1024 ? kFftThreads : kFftThreads / 2;
    pl.threads[a] = std::min(per_block, std::max(64, want));
    const int groups = pl.threads[a] / pl.width[a];
    for (int i = 0, len = n[a]; i < pl.ax[a].stages; ++i) {
      len /= pl.ax[a].radix[i];
      pl.ax[a].m[i] = len;
      pl.ax[a].inv_m[i] = 1.f / (float)len;
      pl.ax[a].dj[i] = groups % len;
      pl.ax[a].db[i] = groups / len;
    }
    if (a == PASS_X && (int64_t)(n[a] / 2 + 1) * pl.width[a] > (int64_t)kEnergies * pl.threads[a]) return false;
  }
  *err = cudaGetDevice(&dev);
  if (*err == cudaSuccess) *err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  for (int a = 0; a < 3 && *err == cudaSuccess; ++a) {
    const PassFn fn = pass_fn(a, pl);
    int per_sm = 0;
    *err = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit);
    if (*err == cudaSuccess)
      *err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, pl.threads[a], pl.smem[a]);
    if (*err == cudaSuccess && per_sm < 1) *err = cudaErrorInvalidConfiguration;
    pl.blocks[a] = per_sm * sms;
  }
  *out = pl;
  return *err == cudaSuccess;
}

void fft_twiddles(const FftPlan& pl, float2* host) {
  for (int a = 0; a < 3; ++a)
    for (int k = 0; k < pl.ax[a].n; ++k) {
      const double t = -2.0 * 3.14159265358979323846 * k / pl.ax[a].n;
      *host++ = make_float2((float)std::cos(t), (float)std::sin(t));
    }
}

cudaError_t launch_fft_shells(const float* u, const FftPlan& pl, int first, int comps, int kmax, const float2* tw,
                              float2* work, double* partials, cudaStream_t st) {
  const int nx = pl.ax[0].n, ny = pl.ax[1].n, nz = pl.ax[2].n;
  const int64_t plane = (int64_t)nx * ny, nh = nz / 2 + 1;
  const int64_t cols[3] = {nh * ny, nh * nx, (plane + 1) / 2};
  const float2* table[3] = {tw, tw + nx, tw + nx + ny};
  for (int a = 2; a >= 0; --a) {
    FftArgs fa{};
    fa.u = u + (int64_t)first * plane * nz;
    fa.work = work;
    fa.tw = table[a];
    fa.ax = pl.ax[a];
    fa.nx = nx;
    fa.ny = ny;
    fa.nz = nz;
    fa.comps = comps;
    fa.kmax = kmax;
    fa.tile = pl.tile[a];
    fa.ncell = plane * nz;
    fa.half = pl.half;
    fa.cols = cols[a];
    fa.tiles_per_comp = (cols[a] + pl.width[a] - 1) / pl.width[a];
    fa.partials = partials;
    // the x pass always has pl.blocks[0] blocks or fewer rows of partials in use
    const int grid = (int)std::min<int64_t>(pl.blocks[a], fa.tiles_per_comp * comps);
    const cudaError_t e = launch_kernel(pass_fn(a, pl), grid, pl.threads[a], pl.smem[a], st, fa);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

int bin_lines_blocks(int nx, int ny, int nz, int kmax, int num_sms) {
  int per_sm = 0;
  const size_t smem = bin_smem(nx, kmax);
  if (cudaFuncSetAttribute(k_bin_lines, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_bin_lines, kBinThreads, smem) != cudaSuccess)
    return num_sms;
  const int64_t tiles = ((int64_t)ny * nz + kBinWidth - 1) / kBinWidth;
  return (int)std::min<int64_t>(tiles, (int64_t)num_sms * std::max(1, per_sm));
}

cudaError_t launch_bin_lines(const float2* c, int nx, int ny, int nz, int kmax, double* partials, int blocks,
                             cudaStream_t st) {
  if (kmax >= kMaxShells) return cudaErrorInvalidValue;
  return launch_kernel(k_bin_lines, blocks, kBinThreads, bin_smem(nx, kmax), st, c, nx, ny, nz, kmax, partials);
}

uint32_t bounds_word_spectrum() { return take_bounds_word(); }

}  // namespace lbm
