// Diagnostics reduction over five device moment fields rho, ux, uy, bx, by [ny][nx] (periodic), for
// lbmhd_diagnostics_fields_noalloc and binary64 states, and its parts, which binary32 and binary16
// states apply to moments taken straight from the populations (diag_pops_kernel, lbmhd_aux.cu).
//
// Slots of a record: 0 sum rho, 1 sum Jx, 2 sum Jy, 3 sum Bx, 4 sum By, 5 sum rho |u|^2 / 2,
// 6 sum |B|^2 / 2, 7 max |div B| (isotropic), 8 max |div B| (central), 9 max |d_beta B_alpha|
// (isotropic), 10 instability flag.  Maxima skip NaN (the flag reports it), as fmax does.
//
// Bound by GB300's binary64 rate (528 G instructions/s; the 40 bytes per cell would take 25 us at
// 2048^2), so the work is arranged for few binary64 instructions, 25 per cell against about 60
// with each derivative summed from its six neighbours: a thread marches down one column of a
// 128-column tile and forms each row's x-difference D = a(x+1) - a(x-1) and weighted sum
// S = a(x) + (a(x-1) + a(x+1)) / 4 once, from which the isotropic derivatives of row y are
// 3 d_x = D(y) + (D(y-1) + D(y+1)) / 4 and 3 d_y = S(y+1) - S(y-1); scales are applied once at the
// end; maxima and the stability tests compare bit patterns with integer instructions.
// 2048^2, cold caches: 444 us and 42 us for the final record before, 224 and 13 us now.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "lbmhd_internal.cuh"

namespace lbmhd_gpu {

constexpr int kDiagThreads = 128;  // columns of a tile
constexpr int kDiagMinRows = 4;    // rows of a tile, at least (halo rows are formed twice)

// Tiles of kDiagThreads columns x `rows` rows: as few rows as keep the tiles within max_blocks.
// `grouped`: on grids of up to half as many columns a tile is `groups` pieces of `cols` = nx columns, one
// below the other, so that few lanes idle.  Fields to values, threads over consecutive cells / one
// piece / now: 3 x 65536 82 / 164 / 30 us, 16 x 65536 170 / 164 / 80, 64 x 65536 581 / 269 / 236.
struct DiagTiles {
  int strips, rows, blocks;
  int cols, groups;
  long tiles;
};
inline DiagTiles diag_tiles(int nx, int ny, int max_blocks, bool grouped, int min_rows) {
  DiagTiles t;
  t.strips = (nx + kDiagThreads - 1) / kDiagThreads;
  t.groups = grouped && nx <= kDiagThreads / 2 ? kDiagThreads / nx : 1;
  t.cols = t.groups > 1 ? nx : kDiagThreads;
  const long pieces = (long)max_blocks * t.groups;
  const long rows = ((long)t.strips * ny + pieces - 1) / pieces;
  // a tile's rows are a serial chain: fewer of them while that leaves fewer than sixteen tiles (fields of 4 x 4 and
  // 8 x 8 14.4 us with a thread per cell, 16.4 in rows of four, 13.4 and 12.4 now; lbmhd_diagnostics of 64^2 binary64
  // 55 -> 51)
  const long spread = ((long)t.strips * ny + 16L * t.groups - 1) / (16L * t.groups);
  if (spread < min_rows) min_rows = (int)spread;
  t.rows = (int)(rows < min_rows ? min_rows : (rows > ny ? ny : rows));
  t.tiles = (long)t.strips * ((ny + (long)t.rows * t.groups - 1) / ((long)t.rows * t.groups));
  t.blocks = (int)(t.tiles < max_blocks ? t.tiles : max_blocks);
  return t;
}

namespace {

// Bits of |v|, ordered like the values; NaN (a quiet one, as arithmetic gives) as 0.  On the two
// words: written on the 64-bit pattern, the compiler turns the test back into a binary64 compare.
__device__ __forceinline__ unsigned long long abs_bits(double v) {
  const unsigned hi = (unsigned)__double2hiint(v) & 0x7fffffffu, lo = (unsigned)__double2loint(v);
  return hi >= 0x7ff80000u ? 0ull : ((unsigned long long)hi << 32) | lo;
}
__device__ __forceinline__ bool not_finite(double v) { return (__double2hiint(v) & 0x7ff00000) == 0x7ff00000; }

// Combine two records' slot k (max for the non-negative maxima and the flag).
__device__ __forceinline__ double diag_combine(int k, double a, double b) { return k <= 6 ? a + b : (b > a ? b : a); }

// A thread's part of a record: sums of its cells, maxima (bits) and flag.
struct DiagAcc {
  double sum[7];
  unsigned long long mx[3];
  bool bad;
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int k = 0; k < 7; ++k) sum[k] = 0.0;
#pragma unroll
    for (int k = 0; k < 3; ++k) mx[k] = 0;
    bad = false;
  }
  __device__ __forceinline__ void add_cell(double r, double u, double v, double b, double d) {
    const double q = fma(u, u, v * v);
    sum[0] += r;
    sum[1] = fma(r, u, sum[1]);
    sum[2] = fma(r, v, sum[2]);
    sum[3] += b;
    sum[4] += d;
    sum[5] = fma(r, q, sum[5]);
    sum[6] = fma(b, b, fma(d, d, sum[6]));
    // not (rho > 0 and |u|^2 <= 0.16), or anything not finite
    bad = bad || not_finite(r) || not_finite(u) || not_finite(v) || not_finite(b) || not_finite(d) ||
          __double_as_longlong(r) <= 0 || __double_as_longlong(q) > __double_as_longlong(0.16);
  }
};

// Rows y - 1, y, y + 1 of one column in slots 0, 1, 2: value, D and S of B_x and B_y.
struct DiagRows {
  double a[2][3], D[2][3], S[2][3];
  __device__ __forceinline__ void set(int f, int k, double v, double e, double w) {
    a[f][k] = v;
    D[f][k] = e - w;
    S[f][k] = fma(0.25, e + w, v);
  }
  // the derivatives of row y
  __device__ __forceinline__ void add_to(DiagAcc& acc) const {
    double dx[2], dy[2];  // three times the isotropic derivatives
#pragma unroll
    for (int f = 0; f < 2; ++f) {
      dx[f] = fma(0.25, D[f][0] + D[f][2], D[f][1]);
      dy[f] = S[f][2] - S[f][0];
    }
    acc.mx[0] = max(acc.mx[0], abs_bits(dx[0] + dy[1]));
    acc.mx[1] = max(acc.mx[1], abs_bits(D[0][1] + (a[1][2] - a[1][0])));
    acc.mx[2] =
        max(max(acc.mx[2], max(abs_bits(dx[0]), abs_bits(dy[0]))), max(abs_bits(dx[1]), abs_bits(dy[1])));
  }
  __device__ __forceinline__ void advance() {
#pragma unroll
    for (int f = 0; f < 2; ++f)
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        a[f][k] = a[f][k + 1];
        D[f][k] = D[f][k + 1];
        S[f][k] = S[f][k + 1];
      }
  }
};

// The block's record: its threads' parts by halves.
__device__ __forceinline__ void diag_record(const DiagAcc& acc, double (&sh)[kDiagSlots][kDiagThreads],
                                            double* __restrict__ rec) {
#pragma unroll
  for (int k = 0; k < 7; ++k) sh[k][threadIdx.x] = (k >= 5 ? 0.5 : 1.0) * acc.sum[k];
#pragma unroll
  for (int k = 0; k < 3; ++k)
    sh[7 + k][threadIdx.x] = (k == 1 ? 0.5 : 1.0 / 3.0) * __longlong_as_double((long long)acc.mx[k]);
  sh[10][threadIdx.x] = acc.bad ? 1.0 : 0.0;
  __syncthreads();
  for (int w = kDiagThreads / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) {
#pragma unroll
      for (int k = 0; k < kDiagSlots; ++k)
        sh[k][threadIdx.x] = diag_combine(k, sh[k][threadIdx.x], sh[k][threadIdx.x + w]);
    }
    __syncthreads();
  }
  if (threadIdx.x < kDiagSlots) rec[threadIdx.x] = sh[threadIdx.x][0];
}

// One record per block into partials[blockIdx.x].  GROUPED: tiles of several pieces (else a block's rows
// are the same in all threads, and their addresses not per thread: 2048^2 234 us, 239 without the
// distinction).
template <bool GROUPED>
__global__ void __launch_bounds__(kDiagThreads)
    diag_partial_kernel(const double* __restrict__ rho, const double* __restrict__ ux, const double* __restrict__ uy,
                        const double* __restrict__ bx, const double* __restrict__ by, int nx, int ny, DiagTiles t,
                        double* __restrict__ partials) {
  DiagAcc acc;
  acc.clear();
  const int group = GROUPED ? (int)threadIdx.x / t.cols : 0;
  const int col = GROUPED ? (int)threadIdx.x - group * t.cols : (int)threadIdx.x;
  for (long tile = blockIdx.x; tile < t.tiles; tile += gridDim.x) {
    const int x = (int)(tile % t.strips) * kDiagThreads + col;
    const long top = (GROUPED ? tile / t.strips * t.groups + group : tile / t.strips) * t.rows;
    if (x >= nx || (GROUPED && (group >= t.groups || top >= ny))) continue;
    const int y0 = (int)top, y1 = (int)min(top + t.rows, (long)ny);
    const int xe = x + 1 == nx ? 0 : x + 1, xw = x == 0 ? nx - 1 : x - 1;
    DiagRows rows;
    auto row = [&](int y, int k) {
      const size_t o = (size_t)(y < 0 ? y + ny : (y >= ny ? y - ny : y)) * nx;
#pragma unroll
      for (int f = 0; f < 2; ++f) {
        const double* p = (f ? by : bx) + o;
        rows.set(f, k, p[x], p[xe], p[xw]);
      }
    };
    row(y0 - 1, 0);
    row(y0, 1);
    for (int y = y0; y < y1; ++y) {
      row(y + 1, 2);
      const size_t c = (size_t)y * nx + x;
      acc.add_cell(rho[c], ux[c], uy[c], rows.a[0][1], rows.a[1][1]);
      rows.add_to(acc);
      rows.advance();
    }
  }
  __shared__ double sh[kDiagSlots][kDiagThreads];
  diag_record(acc, sh, partials + (size_t)blockIdx.x * kDiagSlots);
}

inline void launch_diag_partials(const double* rho, const double* ux, const double* uy, const double* bx,
                                 const double* by, int nx, int ny, const DiagTiles& t, double* partials,
                                 cudaStream_t s) {
  const auto kernel = t.groups > 1 ? diag_partial_kernel<true> : diag_partial_kernel<false>;
  kernel<<<t.blocks, kDiagThreads, 0, s>>>(rho, ux, uy, bx, by, nx, ny, t, partials);
}

// out[k] = records combined in a fixed order: warp k takes slot k, each lane every 32nd record,
// then the lanes by halves.  (One thread per slot took 42 us for 304 records.)
__global__ void __launch_bounds__(32 * kDiagSlots)
    diag_final_kernel(const double* __restrict__ partials, int nblocks, double* __restrict__ out) {
  const int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double a = 0.0;
#pragma unroll 4
  for (int b = lane; b < nblocks; b += 32) a = diag_combine(k, a, partials[(size_t)b * kDiagSlots + k]);
  for (int w = 16; w > 0; w >>= 1) a = diag_combine(k, a, __shfl_down_sync(0xffffffffu, a, w));
  if (lane == 0) out[k] = a;
}

}  // namespace
}  // namespace lbmhd_gpu
