// Analysis kernels for comparing filtered DNS with LES: the box filter with downsampling, and
// shell-summed kinetic and magnetic energy spectra.  Off the time-step path.
//
// Box filter: out(i, j) = r^-2 sum of the r x r block of `in` starting at (r i, r j) -- the
// discrete top-hat filter of width r (Sec. 1, Eq. VelFilter, with a top-hat G) sampled at
// every r-th cell.
//
// Spectra: with Z = FFT(u_x + i u_y), |u_x^(k)|^2 + |u_y^(k)|^2 = (|Z(k)|^2 + |Z(-k)|^2) / 2, and a
// shell holds -k whenever it holds k, so E_kin(s) = n^-4 / 2 sum_{k in shell s} |Z(k)|^2 with ONE
// complex transform for the two fields (likewise E_mag from B_x + i B_y).  Shell s holds the
// integer wavevectors with (2s-1)^2 < 4|k|^2 < (2s+1)^2.  Each thread adds a shell's cells of one
// column in a fixed order and the column sums are combined in a fixed order, so results are
// bitwise reproducible.
//
// What bounds it: GB300's binary64 rate (528 G instructions/s, 1/74 of binary32), not memory, so
// the transform is arranged for few binary64 instructions -- about 32 per point and dimension
// with radix-8 stages and twiddles from a table -- and spends integer instructions (digit
// reversal, shell limits) freely.  Lines stay in shared memory: one kernel transforms the rows,
// one the columns and adds up the shells, so the n x n spectrum is never stored.  Every n <= 4096
// takes O(n^2 log n): radices 8, 4, 2, 3, 5, 7, 11, 13 when they factor n, Bluestein's chirp
// convolution of power-of-two length >= 2n - 1 otherwise.  Four fields at n = 1024 took 60.1 ms with
// direct O(n^3) sums, 0.40 ms with tests
// for unit twiddles and for Bluestein around single products (predicated, these take binary64 time
// all the same), now 0.35: rows 147, columns and shells 186, shell totals 7 us.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdio>
#include <type_traits>

#include "lbmhd.h"
#include "lbmhd_internal.cuh"

namespace lbmhd_gpu {
namespace {

// s 2^-k, by its exponent where that is exact; the product is a call, so that it is branched
// around (predicated, it would take its time on the binary64 pipe in every thread).
__device__ __noinline__ double scaled_product(double s, double inv) { return s * inv; }
__device__ __forceinline__ double scale_down(double s, int k, double inv) {
  const int hi = __double2hiint(s), ex = (hi >> 20) & 0x7ff;
  if (ex > k && ex < 0x7ff) return __hiloint2double(hi - (k << 20), __double2loint(s));
  if (((hi & 0x7fffffff) | __double2loint(s)) == 0) return s;
  return scaled_product(s, inv);  // subnormal results, infinities, NaN
}

// Bound by memory (8 bytes in per cell) and, nearly as much, by binary64 instructions (at r = 2 the
// three additions of a coarse cell take 6 us for 2048^2, its bytes as long): a thread adds up one
// coarse cell, row by row from the left, with the loads of a row independent of one another; a
// warp reads whole rows of the fine field.  VEC: 16-byte loads (r even, rows and field on 16-byte
// boundaries).  log2sq: 2 log2 r, or -1 when r is no power of two and the mean takes a product.
// 2048^2, r = 2, cold caches: 24.5 us with 64-bit divisions per cell and a grid-stride loop (a division
// by r^2 in every thread cost another binary64 dozen), 13.9 with a first addition to zero and a
// product in every thread, now 10.1 us.
// UNROLL: loads in flight; few additions wait on one another in small cells and the remainder of a row
// costs more (1300^2, r = 10: 4 12.3 us, 8 14.4; r = 26: 46, 55), in large ones the loads do (2048^2,
// r = 32: 72, 57; r = 1024: 58 and 46 ms).
// ROWS: several rows of means to a block (else its row is the same in all threads).
template <bool VEC, int UNROLL, bool ROWS>
__global__ void __launch_bounds__(128)
    block_mean_kernel(const double* __restrict__ in, int nx, int mx, int my, int r, int log2sq, double inv,
                      double* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= mx) return;
  const int rows = ROWS ? blockDim.y : 1;
  for (int j = blockIdx.y * rows + (ROWS ? threadIdx.y : 0); j < my; j += gridDim.y * rows) {
    const double* row = in + (size_t)j * r * nx + (size_t)i * r;
    double s;
    if constexpr (VEC) {
      const double2 v = *reinterpret_cast<const double2*>(row);
      s = v.x + v.y;
    } else {
      s = row[0];
    }
    int first = VEC ? 2 : 1;  // of this row
#pragma unroll 2
    for (int yy = 0; yy < r; ++yy, row += nx, first = 0) {
      if constexpr (VEC) {
#pragma unroll UNROLL
        for (int xx = first; xx < r; xx += 2) {
          const double2 v = *reinterpret_cast<const double2*>(row + xx);
          s += v.x;
          s += v.y;
        }
      } else {
#pragma unroll UNROLL
        for (int xx = first; xx < r; ++xx) s += row[xx];
      }
    }
    out[(size_t)j * mx + i] = log2sq >= 0 ? scale_down(s, log2sq, inv) : scaled_product(s, inv);
  }
}

// ---- in-place FFT of lines in shared memory -----------------------------------------------------
constexpr int kMaxRadices = 16;

// Transform of lines of n points: n itself factored into `rad` (len = n), or Bluestein's
// convolution of power-of-two length len >= 2n - 1.
struct FftPlan {
  int n, len, nrad;
  int lines;    // lines per block
  int threads;  // threads per block
  unsigned char rad[kMaxRadices];
  __host__ __device__ bool chirp() const { return len != n; }
};

// Device tables of a plan: tw[len] = exp(-2 pi i j / len); for Bluestein also chirp[n] =
// exp(-pi i j^2 / n) and the transform of the conjugate chirp, over len, in digit-reversed order.
struct FftTables {
  double2* tw;
  double2* chirp;
  double2* filter;
};

__device__ __forceinline__ double2 operator+(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 operator-(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 swap_ri(double2 a) { return make_double2(a.y, a.x); }
__device__ __forceinline__ double2 mul_mi(double2 a) { return make_double2(a.y, -a.x); }  // -i a

__device__ __forceinline__ void dft4(double2& a, double2& b, double2& c, double2& d) {
  const double2 s = a + c, t = a - c, u = b + d, v = mul_mi(b - d);
  a = s + u;
  b = t + v;
  c = s - u;
  d = t - v;
}

// x <- R-point DFT of x (natural order).  Odd R: cosines and sines are tw[k len / R].
template <int R>
__device__ __forceinline__ void dft(double2 (&x)[R], const double2* __restrict__ tw, int len) {
  if constexpr (R == 2) {
    const double2 t = x[0] - x[1];
    x[0] = x[0] + x[1];
    x[1] = t;
  } else if constexpr (R == 4) {
    dft4(x[0], x[1], x[2], x[3]);
  } else if constexpr (R == 8) {
    dft4(x[0], x[2], x[4], x[6]);
    dft4(x[1], x[3], x[5], x[7]);
    const double h = 0.70710678118654752440;  // sqrt(1/2)
    const double2 o0 = x[1], o2 = mul_mi(x[5]);
    const double2 o1 = make_double2(h * (x[3].x + x[3].y), h * (x[3].y - x[3].x));
    const double2 o3 = make_double2(h * (x[7].y - x[7].x), -h * (x[7].x + x[7].y));
    const double2 e0 = x[0], e1 = x[2], e2 = x[4], e3 = x[6];
    x[0] = e0 + o0;
    x[1] = e1 + o1;
    x[2] = e2 + o2;
    x[3] = e3 + o3;
    x[4] = e0 - o0;
    x[5] = e1 - o1;
    x[6] = e2 - o2;
    x[7] = e3 - o3;
  } else {
    // odd prime: X_k = x_0 + sum_j cos(jk) (x_j + x_-j) - i sin(jk) (x_j - x_-j), j = 1 .. (R-1)/2
    constexpr int H = (R - 1) / 2;
    double2 s[H], d[H], w[H];
    double2 dc = x[0];
#pragma unroll
    for (int j = 0; j < H; ++j) {
      s[j] = x[j + 1] + x[R - 1 - j];
      d[j] = x[j + 1] - x[R - 1 - j];
      w[j] = tw[(j + 1) * (len / R)];  // (cos, -sin)
      dc = dc + s[j];
    }
#pragma unroll
    for (int k = 1; k <= H; ++k) {
      double2 a = x[0], b = make_double2(0.0, 0.0);
#pragma unroll
      for (int j = 1; j <= H; ++j) {
        constexpr int RR = R;
        const int jk = j * k % RR;
        const double c = w[(jk <= H ? jk : RR - jk) - 1].x;
        const double sn = jk <= H ? w[jk - 1].y : -w[RR - jk - 1].y;  // -sin(2 pi jk / R)
        a.x += c * s[j - 1].x;
        a.y += c * s[j - 1].y;
        b.x += sn * d[j - 1].x;
        b.y += sn * d[j - 1].y;
      }
      // i b = (-b.y, b.x)
      x[k] = make_double2(a.x - b.y, a.y + b.x);
      x[R - k] = make_double2(a.x + b.y, a.y - b.x);
    }
    x[0] = dc;
  }
}

// One radix-R stage over sub-blocks of ns points, in place.  Forward (decimation in frequency):
// R-point DFT, then twiddles; natural order in, digit-reversed order out after the last stage.
// Inverse undoes it: conjugate twiddles, then the conjugate DFT.  UNIT: ns = R, all twiddles one (a
// test of m in the loop would be predicated, and the products take binary64 pipe time all the same).
template <int R, bool INVERSE, bool UNIT>
__device__ __forceinline__ void fft_stage_of(double2* buf, int lines, int len, int ns, const double2* __restrict__ tw) {
  const int m = UNIT ? 1 : ns / R, per_line = len / R, tstep = len / ns;
  for (int q = threadIdx.x; q < lines * per_line; q += blockDim.x) {
    const int line = q / per_line, r = q - line * per_line;
    const int blk = r / m, j = r - blk * m;
    double2* a = buf + line * len + blk * ns + j;
    double2 x[R];
#pragma unroll
    for (int k = 0; k < R; ++k) x[k] = a[k * m];
    if constexpr (INVERSE) {
#pragma unroll
      for (int k = 0; k < R; ++k) {
        if (k > 0 && !UNIT) {
          const double2 w = tw[j * k * tstep];
          x[k] = cmul(x[k], make_double2(w.x, -w.y));
        }
        x[k] = swap_ri(x[k]);
      }
      dft<R>(x, tw, len);
#pragma unroll
      for (int k = 0; k < R; ++k) a[k * m] = swap_ri(x[k]);
    } else {
      dft<R>(x, tw, len);
#pragma unroll
      for (int k = 0; k < R; ++k) {
        if (k > 0 && !UNIT) x[k] = cmul(x[k], tw[j * k * tstep]);
        a[k * m] = x[k];
      }
    }
  }
  __syncthreads();
}

template <int R, bool INVERSE>
__device__ __forceinline__ void fft_stage(double2* buf, int lines, int len, int ns, const double2* __restrict__ tw) {
  if (ns == R) fft_stage_of<R, INVERSE, true>(buf, lines, len, ns, tw);
  else fft_stage_of<R, INVERSE, false>(buf, lines, len, ns, tw);
}

// Forward transform of the block's lines (buf[line * len + j], complete before the call).
__device__ __forceinline__ void fft_forward(double2* buf, const FftPlan& p, const double2* __restrict__ tw) {
  int ns = p.len;
  for (int st = 0; st < p.nrad; ++st) {
    const int R = p.rad[st];
    switch (R) {
      case 8: fft_stage<8, false>(buf, p.lines, p.len, ns, tw); break;
      case 4: fft_stage<4, false>(buf, p.lines, p.len, ns, tw); break;
      case 2: fft_stage<2, false>(buf, p.lines, p.len, ns, tw); break;
      case 3: fft_stage<3, false>(buf, p.lines, p.len, ns, tw); break;
      case 5: fft_stage<5, false>(buf, p.lines, p.len, ns, tw); break;
      case 7: fft_stage<7, false>(buf, p.lines, p.len, ns, tw); break;
      case 11: fft_stage<11, false>(buf, p.lines, p.len, ns, tw); break;
      default: fft_stage<13, false>(buf, p.lines, p.len, ns, tw); break;
    }
    ns /= R;
  }
}

// Inverse (unscaled) of fft_forward for power-of-two lengths: digit-reversed in, natural out.
__device__ __forceinline__ void fft_inverse_pow2(double2* buf, const FftPlan& p, const double2* __restrict__ tw) {
  int ns = 1;
  for (int st = p.nrad - 1; st >= 0; --st) {
    const int R = p.rad[st];
    ns *= R;
    if (R == 8) fft_stage<8, true>(buf, p.lines, p.len, ns, tw);
    else if (R == 4) fft_stage<4, true>(buf, p.lines, p.len, ns, tw);
    else fft_stage<2, true>(buf, p.lines, p.len, ns, tw);
  }
}

// Position of output k in a digit-reversed line.
__device__ __forceinline__ int digit_reversed(const FftPlan& p, int k) {
  int pos = 0, ns = p.len;
  for (int st = 0; st < p.nrad; ++st) {
    const int R = p.rad[st], q = k / R;
    ns /= R;
    pos += (k - q * R) * ns;
    k = q;
  }
  return pos;
}

// DFT of the block's lines; buf[line * len + j] holds point j (times chirp[j] for Bluestein, zero
// from n on), complete before the call.  Afterwards fft_result reads the outputs.
template <bool CHIRP>
__device__ __forceinline__ void transform_lines(double2* buf, const FftPlan& p, const FftTables& t) {
  fft_forward(buf, p, t.tw);
  if constexpr (CHIRP) {
    for (int q = threadIdx.x; q < p.lines * p.len; q += blockDim.x) buf[q] = cmul(buf[q], t.filter[q % p.len]);
    __syncthreads();
    fft_inverse_pow2(buf, p, t.tw);
  }
}

// Output k of a transformed line up to a unit factor (Bluestein leaves out the last chirp
// product): exact for |X_k|, which is all that the columns need; `full` puts it in (the rows).
template <bool CHIRP>
__device__ __forceinline__ double2 fft_result(const double2* line, const FftPlan& p, const FftTables& t, int k,
                                              bool full) {
  if constexpr (!CHIRP) return line[digit_reversed(p, k)];
  else return full ? cmul(line[k], t.chirp[k]) : line[k];
}

__global__ void fft_tables_kernel(FftPlan p, FftTables t) {
  const int total = p.len + (p.chirp() ? p.n : 0);
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < total; j += gridDim.x * blockDim.x) {
    double s, c;
    if (j < p.len) {
      sincospi(2.0 * (double)j / (double)p.len, &s, &c);
      t.tw[j] = make_double2(c, -s);
    } else {
      const long i = j - p.len;
      sincospi((double)(i * i % (2L * p.n)) / (double)p.n, &s, &c);  // period 2n in j^2
      t.chirp[i] = make_double2(c, -s);
    }
  }
}

// Bluestein: transform of the periodic conjugate chirp b_j = conj(chirp[|j|]), |j| < n, over len.
__global__ void fft_filter_kernel(FftPlan p, FftTables t) {
  extern __shared__ double2 fft_buf[];
  p.lines = 1;
  for (int j = threadIdx.x; j < p.len; j += blockDim.x) {
    const int i = j < p.n ? j : p.len - j;
    double2 v = make_double2(0.0, 0.0);
    if (i < p.n) v = make_double2(t.chirp[i].x, -t.chirp[i].y);
    fft_buf[j] = v;
  }
  __syncthreads();
  fft_forward(fft_buf, p, t.tw);
  const double inv = 1.0 / p.len;
  for (int j = threadIdx.x; j < p.len; j += blockDim.x)
    t.filter[j] = make_double2(inv * fft_buf[j].x, inv * fft_buf[j].y);
}

// G[pair][y][kx]: row transforms of u_x + i u_y (pair 0) and B_x + i B_y (pair 1).  CHIRP: Bluestein
// (compiled apart: its products, predicated off, would take an eighth of the binary64 issue).
template <bool CHIRP>
__global__ void __launch_bounds__(256)
    fft_rows_kernel(const double* __restrict__ ux, const double* __restrict__ uy, const double* __restrict__ bx,
                    const double* __restrict__ by, FftPlan p, FftTables t, double2* __restrict__ G) {
  extern __shared__ double2 fft_buf[];
  const int n = p.n, y0 = blockIdx.x * p.lines;
  const double* re = blockIdx.y ? bx : ux;
  const double* im = blockIdx.y ? by : uy;
  p.lines = min(p.lines, n - y0);
  for (int q = threadIdx.x; q < p.lines * p.len; q += blockDim.x) {
    const int line = q / p.len, j = q - line * p.len;
    double2 v = make_double2(0.0, 0.0);
    if (j < n) {
      const size_t c = (size_t)(y0 + line) * n + j;
      v = make_double2(re[c], im[c]);
      if constexpr (CHIRP) v = cmul(v, t.chirp[j]);
    }
    fft_buf[q] = v;
  }
  __syncthreads();
  transform_lines<CHIRP>(fft_buf, p, t);
  double2* g = G + (size_t)blockIdx.y * n * n + (size_t)y0 * n;
  for (int q = threadIdx.x; q < p.lines * n; q += blockDim.x) {
    const int line = q / n, k = q - line * n;
    g[q] = fft_result<CHIRP>(fft_buf + (size_t)line * p.len, p, t, k, true);
  }
}

// Largest integer r >= 0 with 4 r^2 <= v (v >= 0, v < 2^28): binary32 estimate, then exact.
__device__ __forceinline__ int half_isqrt(int v) {
  int r = (int)(0.5f * sqrtf((float)v));
  while (4 * r * r > v) --r;
  while (4 * (r + 1) * (r + 1) <= v) ++r;
  return r;
}

// Column transforms of pair blockIdx.y and the shell sums of this block's columns:
// part[pair][column group][s] = sum over the group's columns kx and the ky of shell s of
// |Z(kx, ky)|^2.  In one column a shell is two runs of consecutive ky, which one thread adds.
template <bool CHIRP>
__global__ void __launch_bounds__(256)
    fft_cols_kernel(const double2* __restrict__ G, FftPlan p, FftTables t, int nbins, double* __restrict__ part) {
  extern __shared__ double2 fft_buf[];
  const int n = p.n, x0 = blockIdx.x * p.lines;
  p.lines = min(p.lines, n - x0);
  const int kneg = n / 2, kpos = (n - 1) / 2;  // wavenumbers -kneg .. kpos
  double* out = part + ((size_t)blockIdx.y * gridDim.x + blockIdx.x) * nbins;
  // a column beyond the outermost shell contributes nothing
  const long top4 = (long)(2 * nbins - 1) * (2 * nbins - 1);
  bool any = false;
  for (int c = 0; c < p.lines; ++c) {
    const long kx = x0 + c <= kpos ? x0 + c : x0 + c - n;
    any = any || 4 * kx * kx < top4;
  }
  if (!any) {
    for (int s = threadIdx.x; s < nbins; s += blockDim.x) out[s] = 0.0;
    return;
  }
  const double2* g = G + (size_t)blockIdx.y * n * n;
  // consecutive threads take consecutive columns of a row; p.lines columns per row
  const int lines = p.lines, len = p.len;
  for (int q = threadIdx.x; q < lines * len; q += blockDim.x) {
    const int j = q / lines, line = q - j * lines;
    double2 v = make_double2(0.0, 0.0);
    if (j < n) {
      v = g[(size_t)j * n + x0 + line];
      if constexpr (CHIRP) v = cmul(v, t.chirp[j]);
    }
    fft_buf[line * len + j] = v;
  }
  __syncthreads();
  transform_lines<CHIRP>(fft_buf, p, t);
  // |Z|^2 in natural order first: the runs below are then consecutive (a thread that added up to 45
  // digit-reversed cells of its run held its block up)
  double* power = reinterpret_cast<double*>(fft_buf + (size_t)lines * len);  // [lines][n]
  for (int q = threadIdx.x; q < lines * n; q += blockDim.x) {
    const int c = q / n, k = q - c * n;
    const double2 z = fft_result<CHIRP>(fft_buf + (size_t)c * len, p, t, k, false);
    power[q] = z.x * z.x + z.y * z.y;
  }
  __syncthreads();
  for (int s = threadIdx.x; s < nbins; s += blockDim.x) {
    const int lo4 = (2 * s - 1) * (2 * s - 1), hi4 = (2 * s + 1) * (2 * s + 1);
    double sum = 0.0;
    for (int c = 0; c < lines; ++c) {
      const int kx = x0 + c <= kpos ? x0 + c : x0 + c - n;
      const int k4 = 4 * kx * kx;
      if (k4 >= hi4) continue;
      // 4 ky^2 in (lo4 - k4, hi4 - k4); the limits are odd squares less a multiple of 4, never met.
      // Shell 0 holds the zero wavevector only.
      const int a = s == 0 || k4 > lo4 ? 0 : half_isqrt(lo4 - k4) + 1;
      const int b = half_isqrt(hi4 - k4);
      const double* line = power + (size_t)c * n;
      for (int k = a; k <= min(b, kpos); ++k) sum += line[k];
      for (int k = max(a, 1); k <= min(b, kneg); ++k) sum += line[n - k];
    }
    out[s] = sum;
  }
}

// E[s] = norm * sum over the column groups of part[pair][group][s]: 32 threads per shell take every
// 32nd group in order, then are added in order.
constexpr int kTotalShells = 8;
__global__ void __launch_bounds__(32 * kTotalShells)
    shell_total_kernel(const double* __restrict__ part, int groups, int nbins, double norm, double* __restrict__ ek,
                       double* __restrict__ em) {
  __shared__ double sh[32][kTotalShells + 1];
  const int s = blockIdx.x * kTotalShells + threadIdx.x;
  const double* p = part + (size_t)blockIdx.y * groups * nbins;
  double sum = 0.0;
  if (s < nbins) {
#pragma unroll 4
    for (int g = threadIdx.y; g < groups; g += 32) sum += p[(size_t)g * nbins + s];
  }
  sh[threadIdx.y][threadIdx.x] = sum;
  __syncthreads();
  if (threadIdx.y == 0 && s < nbins) {
    double tot = 0.0;
#pragma unroll
    for (int i = 0; i < 32; ++i) tot += sh[i][threadIdx.x];
    (blockIdx.y ? em : ek)[s] = norm * tot;
  }
}

// Shared memory of a block, at most: one line of 8192 points (Bluestein, n > 2048), and in the columns
// its n <= 4096 squared magnitudes.
constexpr int kMaxRowBytes = 8192 * (int)sizeof(double2);
constexpr int kMaxColBytes = kMaxRowBytes + 4096 * (int)sizeof(double);

// Lines per block: up to 32 KB of points (binary64 work hides everything else, so small blocks
// that fill the last wave evenly are worth more than reuse), 256 threads when a radix-8 stage
// has that many butterflies.
FftPlan make_plan(int n) {
  FftPlan p{};
  p.n = p.len = n;
  // Radix 8 first, so that what is left over comes last, without twiddles -- but a radix 2, whose
  // stage has the fewest, comes first: spectra of 1024^2 fields 387 -> 378 us (2048^2 with its radix 4
  // first 1447 -> 1457, so that stays behind).
  static const int radices[] = {8, 4, 2, 3, 5, 7, 11, 13};
  auto factor = [&](int v) {
    p.nrad = 0;
    int twos = 0;
    while (v >> twos > 0 && (v >> twos) % 2 == 0) ++twos;
    if (twos % 3 == 1) {
      p.rad[p.nrad++] = 2;
      v /= 2;
    }
    for (int r : radices)
      while (v % r == 0) {
        p.rad[p.nrad++] = (unsigned char)r;
        v /= r;
      }
    return v == 1;
  };
  if (!factor(n)) {
    p.len = 1;
    while (p.len < 2 * n - 1) p.len *= 2;
    factor(p.len);
  }
  p.lines = 2048 / p.len < 1 ? 1 : (2048 / p.len > 8 ? 8 : 2048 / p.len);
  p.threads = p.lines * p.len >= 2048 ? 256 : 128;
  return p;
}

}  // namespace

size_t spectrum_work_bytes(int n) {
  const size_t nn = (size_t)n * n;
  return ((size_t)n * sizeof(double2) + 255) / 256 * 256 + 4 * nn * sizeof(double2) + 2 * nn * sizeof(double);
}

cudaError_t launch_energy_spectrum(const double* ux, const double* uy, const double* bx,
                                   const double* by, int n, int nbins, double* ek, double* em,
                                   void* work, cudaStream_t s, int* launches) {
  const size_t nn = (size_t)n * n;
  const FftPlan p = make_plan(n);
  if (launches) *launches = p.chirp() ? 5 : 4;
  // work: tables (len < 4n: at most 9n points), two complex planes, the column groups' shells
  // (at most n x nbins per pair): 144 n + 32 n^2 + 16 n^2 bytes within spectrum_work_bytes(n)
  FftTables t{};
  t.tw = static_cast<double2*>(work);
  double2* G = t.tw + p.len;
  if (p.chirp()) {
    t.chirp = G;
    t.filter = t.chirp + n;
    G = t.filter + p.len;
  }
  double* part = reinterpret_cast<double*>(G + 2 * nn);
  const size_t smem = (size_t)p.lines * p.len * sizeof(double2);
  const size_t smem_cols = smem + (size_t)p.lines * n * sizeof(double);  // and the power of the lines
  const auto rows = p.chirp() ? fft_rows_kernel<true> : fft_rows_kernel<false>;
  const auto cols = p.chirp() ? fft_cols_kernel<true> : fft_cols_kernel<false>;
  if (smem_cols > 48 * 1024) {
    // The limit belongs to the kernel, not to this call: every call sets the same value, the largest
    // that any n needs, so that threads with spectra of different sizes never lower it for one another.
    const auto limit = cudaFuncAttributeMaxDynamicSharedMemorySize;
    cudaError_t e = cudaFuncSetAttribute(rows, limit, kMaxRowBytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(cols, limit, kMaxColBytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fft_filter_kernel, limit, kMaxRowBytes);
    if (e != cudaSuccess) return e;
  }
  const int groups = (n + p.lines - 1) / p.lines;
  fft_tables_kernel<<<(p.len + n + 127) / 128, 128, 0, s>>>(p, t);
  if (p.chirp()) fft_filter_kernel<<<1, 256, p.len * sizeof(double2), s>>>(p, t);
  rows<<<dim3(groups, 2), p.threads, smem, s>>>(ux, uy, bx, by, p, t, G);
  cols<<<dim3(groups, 2), p.threads, smem_cols, s>>>(G, p, t, nbins, part);
  shell_total_kernel<<<dim3((nbins + kTotalShells - 1) / kTotalShells, 2), dim3(kTotalShells, 32), 0, s>>>(part, groups, nbins,
                                                                       0.5 / ((double)nn * (double)nn), ek, em);
  return cudaGetLastError();
}

cudaError_t launch_block_mean(const double* in, int nx, int ny, int r, double* out, cudaStream_t s) {
  const int mx = nx / r, my = ny / r;
  const double inv = 1.0 / ((double)r * r);  // a binary64 division per thread would outweigh the sums
  int log2sq = -1;
  if ((r & (r - 1)) == 0)
    for (log2sq = 0; (1 << (log2sq / 2)) < r;) log2sq += 2;
  // several whole rows of means to a block (but four blocks on every SM) where they are short: with one
  // row to a block 4 x 262144, r = 4, took 86 us and 64 x 65536, r = 8, 39; now 7 and 14
  dim3 nt(mx < 128 ? mx : 128, 1);
  if (mx < 128) {
    const int fit = 128 / mx, spread = my / (4 * 152);
    nt.y = fit < spread ? fit : (spread > 1 ? spread : 1);
  }
  const int rows = (my + (int)nt.y - 1) / (int)nt.y;
  const dim3 grid((mx + nt.x - 1) / nt.x, rows < 65535 ? rows : 65535);
  const bool vec = r % 2 == 0 && nx % 2 == 0 && reinterpret_cast<uintptr_t>(in) % 16 == 0;
  const auto pick = [&](auto rows_tag) {
    constexpr bool R = decltype(rows_tag)::value;
    return r < 32 ? (vec ? block_mean_kernel<true, 4, R> : block_mean_kernel<false, 4, R>)
                  : (vec ? block_mean_kernel<true, 8, R> : block_mean_kernel<false, 8, R>);
  };
  const auto kernel = nt.y > 1 ? pick(std::true_type{}) : pick(std::false_type{});
  kernel<<<grid, nt, 0, s>>>(in, nx, mx, my, r, log2sq, inv, out);
  return cudaGetLastError();
}

}  // namespace lbmhd_gpu

namespace {
int analysis_error(int code, const char* msg) {
  lbmhd_gpu::set_thread_error(msg);
  return code;
}
}  // namespace

extern "C" int lbmhd_block_mean_device(const double* in, int nx, int ny, int r, double* out,
                                       void* stream) {
  if (!in || !out) return analysis_error(LBMHD_ERR_INVALID, "NULL field pointer");
  if (nx < 1 || ny < 1 || r < 1 || nx % r || ny % r)
    return analysis_error(LBMHD_ERR_INVALID, "block mean: r must divide both grid sides");
  cudaError_t e = lbmhd_gpu::launch_block_mean(in, nx, ny, r, out, static_cast<cudaStream_t>(stream));
  if (e != cudaSuccess) return analysis_error(LBMHD_ERR_CUDA, cudaGetErrorString(e));
  return LBMHD_OK;
}

extern "C" size_t lbmhd_energy_spectrum_work_bytes(int n) {
  return n >= 1 ? lbmhd_gpu::spectrum_work_bytes(n) : 0;
}

extern "C" int lbmhd_energy_spectrum_device(const double* ux, const double* uy, const double* bx,
                                            const double* by, int n, int nbins, double* e_kin,
                                            double* e_mag, void* work, size_t work_bytes,
                                            void* stream) {
  if (!ux || !uy || !bx || !by || !e_kin || !e_mag || !work)
    return analysis_error(LBMHD_ERR_INVALID, "NULL pointer");
  if (n < 1 || n > 4096) return analysis_error(LBMHD_ERR_INVALID, "spectrum: n must be in [1, 4096]");
  if (nbins < 1 || nbins > n) return analysis_error(LBMHD_ERR_INVALID, "spectrum: nbins must be in [1, n]");
  if (work_bytes < lbmhd_gpu::spectrum_work_bytes(n))
    return analysis_error(LBMHD_ERR_INVALID, "spectrum: work buffer too small");
  cudaError_t e = lbmhd_gpu::launch_energy_spectrum(ux, uy, bx, by, n, nbins, e_kin, e_mag, work,
                                                    static_cast<cudaStream_t>(stream));
  if (e != cudaSuccess) return analysis_error(LBMHD_ERR_CUDA, cudaGetErrorString(e));
  return LBMHD_OK;
}
