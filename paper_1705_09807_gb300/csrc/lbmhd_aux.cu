// Auxiliary kernels: equilibrium initialisation, macroscopic moments, canonical population
// export and double-precision diagnostics.  None of them is on the per-step path.
#include <algorithm>
#include <type_traits>

#include "lbmhd_diag.cuh"
#include "lbmhd_internal.cuh"
#include "lbmhd_quotient.cuh"

namespace lbmhd_gpu {
namespace {

__host__ __device__ constexpr int vx(int i) { return vel_x(i); }
__host__ __device__ constexpr int vy(int i) { return vel_y(i); }
__host__ __device__ constexpr double wt(int i) { return lattice_w(i); }

__device__ __forceinline__ int wrapi(int i, int n) { return i < 0 ? i + n : (i >= n ? i - n : i); }

// Stored (post-collision) populations whose pull gives the equilibria of the fields:
// stored f*_i(x) = f_i^eq(fields(x + c_i)), so that f_i(x) = f*_i(x - c_i) = f_i^eq(x).
// Eq. feq, written as the deviation f_i^eq - w_i; Eq. geq.  Ghost columns written too.
// REL (relative binary16 storage, LBMHD_FP16_REL): the cell's velocity reference U is its own
// initial u rounded to binary16 (planes kQ, kQ + 1), and each stored f value is taken relative
// to w_i (1 + 3 c_i . U).  The equilibria are evaluated in the storage's arithmetic type A:
// binary64 for binary64 storage, binary32 otherwise (the stored value is rounded to binary32 or
// binary16 anyway, and GB300's binary64 rate is about 1/60 of its binary32 rate).
//
// One block per strip of kInitCols columns and band of kInitRows rows.  The fields of rows
// y - 1, y, y + 1 sit in a ring of three shared-memory rows (columns x0 - 1 .. x0 + kInitCols,
// periodic), each value read and converted to A once, with |u|^2 and |B|^2 formed once per cell:
// the nine equilibria of a cell then read only shared memory.  Only the two halo rows of each
// band are read twice, so the input arrays may be page-locked host memory read over the host
// link.  (Converting every binary64 input nine times, once per direction, took 0.45 ms at 2048^2
// on GB300's binary64 conversion rate.)
constexpr int kInitCols = 128, kInitRows = 32;

template <typename T, bool REL = false>
__global__ void __launch_bounds__(kInitCols)
    init_eq_kernel(T* __restrict__ pops, StepGeom g, const double* __restrict__ rho,
                   const double* __restrict__ ux, const double* __restrict__ uy,
                   const double* __restrict__ bx, const double* __restrict__ by) {
  using A = typename std::conditional<sizeof(T) == 8, double, float>::type;
  constexpr int W = kInitCols + 2;
  constexpr int NV = REL ? 9 : 7;  // rho, ux, uy, bx, by, |u|^2, |B|^2 (REL: U_x, U_y in binary16)
  __shared__ A ring[3][NV][W];
  const int x0 = blockIdx.x * kInitCols;
  const int cols = min(kInitCols, g.nx - x0);
  const int nbands = (g.ny + kInitRows - 1) / kInitRows;
  for (int band = blockIdx.y; band < nbands; band += gridDim.y) {
    const int y0 = band * kInitRows, y1 = min(y0 + kInitRows, g.ny);
    // field row yy (in [-1, ny], periodic) into ring slot (yy + 3) mod 3
    auto load_row = [&](int yy) {
      const int slot = (yy + 3) % 3;
      const size_t row = (size_t)wrapi(yy, g.ny) * g.nx;
      for (int j = threadIdx.x; j < cols + 2; j += blockDim.x) {
        const size_t c = row + wrapi(x0 - 1 + j, g.nx);
        const double du = ux[c], dv = uy[c];
        const A r = (A)rho[c], u = (A)du, v = (A)dv, bb = (A)bx[c], d = (A)by[c];
        A* e = &ring[slot][0][j];
        e[0 * W] = r;
        e[1 * W] = u;
        e[2 * W] = v;
        e[3 * W] = bb;
        e[4 * W] = d;
        e[5 * W] = u * u + v * v;
        e[6 * W] = bb * bb + d * d;
        if constexpr (REL) {
          e[7 * W] = (A)__half2float(__double2half(du));
          e[8 * W] = (A)__half2float(__double2half(dv));
        }
      }
    };
    // (the previous band ended with a block barrier: its readers of the ring are done)
    load_row(y0 - 1);
    load_row(y0);
    for (int y = y0; y < y1; ++y) {
      load_row(y + 1);
      __syncthreads();
      const int jx = threadIdx.x + 1;
      const int x = x0 + threadIdx.x;
      if (threadIdx.x < cols) {
        const size_t o = (size_t)y * g.pitch + kXOff + x;
        A Ux = A(0), Uy = A(0);
        if constexpr (REL) {
          const A* e = &ring[y % 3][0][jx];
          Ux = e[7 * W];
          Uy = e[8 * W];
          const T u2[2] = {store_as<T>(Ux), store_as<T>(Uy)};  // exact: Ux, Uy are binary16 values
#pragma unroll
          for (int comp = 0; comp < 2; ++comp) {
            T* pl = pops + (size_t)(kQ + comp) * g.plane + o;
            pl[0] = u2[comp];
            if (x < 2) pl[g.nx] = u2[comp];
            if (x >= g.nx - 2) pl[-g.nx] = u2[comp];
          }
        }
#pragma unroll
        for (int i = 0; i < 9; ++i) {
          const A* e = &ring[(y + vy(i) + 3) % 3][0][jx + vx(i)];
          const A r = e[0 * W], u = e[1 * W], v = e[2 * W], b = e[3 * W], d = e[4 * W];
          const A usq = e[5 * W], bsq = e[6 * W];
          const A cu = vx(i) * u + vy(i) * v;
          const A cb = vx(i) * b + vy(i) * d;
          const A csq = (A)(vx(i) * vx(i) + vy(i) * vy(i));
          const A w = (A)wt(i);
          A fdev = w * (r - A(1)) + w * r * (A(3) * cu + A(4.5) * cu * cu - A(1.5) * usq) +
                   A(4.5) * w * (A(0.5) * bsq * csq - cb * cb);
          if (REL) fdev -= A(3) * w * (vx(i) * Ux + vy(i) * Uy);
          const A gx = w * (b + A(3) * (cu * b - cb * u));
          const A gy = w * (d + A(3) * (cu * d - cb * v));
          const T vals[3] = {store_as<T>(fdev), store_as<T>(gx), store_as<T>(gy)};
#pragma unroll
          for (int comp = 0; comp < 3; ++comp) {
            T* pl = pops + (size_t)plane_of(9 * comp + i) * g.plane + o;
            pl[0] = vals[comp];
            if (x < 2) pl[g.nx] = vals[comp];          // ghosts of columns 0, 1 at nx, nx + 1
            if (x >= g.nx - 2) pl[-g.nx] = vals[comp];  // ghosts of columns nx-2, nx-1 at -2, -1
          }
        }
      }
      __syncthreads();
    }
  }
}

// Pull the 27 current populations of cell (x, y) in binary64, f as deviations (for REL, each f
// value plus 3 w_i c_i . U of the source cell that stored it).
template <typename T, bool REL = false>
__device__ __forceinline__ void pull_cell(const T* __restrict__ pops, const StepGeom& g, int x,
                                          int y, double v[27]) {
#pragma unroll
  for (int q = 0; q < 27; ++q) {
    const int i = q % 9;
    const int sx = wrapi(x - vx(i), g.nx), sy = wrapi(y - vy(i), g.ny);
    const size_t src = (size_t)sy * g.pitch + kXOff + sx;
    v[q] = load_as<double>(pops[(size_t)plane_of(q) * g.plane + src]);
    if (REL && q >= 1 && q < 9) {
      const double Ux = load_as<double>(pops[(size_t)kQ * g.plane + src]);
      const double Uy = load_as<double>(pops[(size_t)(kQ + 1) * g.plane + src]);
      v[q] += 3.0 * wt(i) * (vx(i) * Ux + vy(i) * Uy);
    }
  }
}

// Exact binary64 value of a binary32 number, by integer operations alone: GB300 converts binary32
// to binary64 at its binary64 rate (1/74 of its integer rate), and a conversion kept for the rare
// forms is predicated, not branched around, and so takes its time on the binary64 pipe all the same.
__device__ __forceinline__ double widen(float f) {
  const uint32_t b = __float_as_uint(f), a = b & 0x7fffffffu;
  uint32_t m = a, e = 0x38000000u;  // significand with its exponent field, exponent offset
  if (a - 0x00800000u >= 0x7f000000u) {
    if (a >= 0x7f800000u) {  // infinity, NaN (made quiet)
      e = 0x70000000u;
      m = a > 0x7f800000u ? a | 0x00400000u : a;
    } else if (a != 0u) {  // subnormal: normalise
      const int shift = __clz(a) - 8;
      m = a << shift;
      e = 0x38000000u - (uint32_t)(shift << 20);
    } else {
      e = 0u;
    }
  }
  return __hiloint2double((int)((b & 0x80000000u) | ((m >> 3) + e)), (int)(m << 29));
}

// Sum of binary32 values kept exactly as the unevaluated pair hi + lo (Knuth's TwoSum: the
// rounding error of each binary32 addition is itself a binary32 value).  Nine stored binary32 or
// binary16 values sum to the binary64 result up to one rounding of lo, with binary32 arithmetic
// only.  EXACT: the caller knows that hi + v never rounds, so lo stays zero.
struct PairSum {
  float hi = 0.f, lo = 0.f;
  template <bool EXACT = false>
  __device__ __forceinline__ void add(float v) {
    const float s = hi + v;
    if constexpr (!EXACT) {
      const float bv = s - hi;
      lo += (hi - (s - bv)) + (v - bv);
    }
    hi = s;
  }
  template <bool EXACT = false>
  __device__ __forceinline__ double value() const {
    return EXACT ? widen(hi) : widen(hi) + widen(lo);
  }
  __device__ __forceinline__ float rounded() const { return hi + lo; }
  // hi + lo + n / 12 rounded to binary32 (n a pair): quotient and remainder, then one TwoSum
  __device__ __forceinline__ float plus_twelfth(const PairSum& n) const {
    const float r12 = 1.f / 12.f, q = __fmul_rn(n.hi, r12);  // rounded: TwoSum needs the value
    const float ql = (fmaf(-12.f, q, n.hi) + n.lo) * r12;
    PairSum t = *this;
    t.add(q);
    return t.hi + (t.lo + ql);
  }
};

// rho, u, B of one cell from its 27 pulled binary32 values (f as stored deviations; REL: relative
// to w_i (1 + 3 c_i . U), with U[k] = {U_x, U_y} of the source cell of f_(k+1)).  False if a value is
// infinite or NaN: one of f makes rho and then u NaN (TwoSum subtracts infinities), one of g a sum.
template <bool EXACT, bool REL>
__device__ __forceinline__ bool moments_of(const float (&v)[27], const float (&U)[8][2], double (&out)[5]) {
  PairSum r, px, py, qx, qy;
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    r.add<EXACT>(v[i]);
    if (vx(i)) px.add<EXACT>(vx(i) > 0 ? v[i] : -v[i]);
    if (vy(i)) py.add<EXACT>(vy(i) > 0 ? v[i] : -v[i]);
    qx.add<EXACT>(v[9 + i]);
    qy.add<EXACT>(v[18 + i]);
  }
  float jx, jy;
  if constexpr (REL) {
    // sum_i (1, c_i) 3 w_i c_i . U(x - c_i) = n / 12 with integer coefficients: 3 w_i is 4/12 on
    // the axes and 1/12 on the diagonals
    PairSum nr, nx, ny;
#pragma unroll
    for (int i = 1; i < 9; ++i) {
      const float k = i < 5 ? 4.f : 1.f;
#pragma unroll
      for (int comp = 0; comp < 2; ++comp) {
        const int c = comp ? vy(i) : vx(i);
        if (c == 0) continue;
        const float t = k * (c > 0 ? U[i - 1][comp] : -U[i - 1][comp]);
        nr.add(t);
        if (vx(i)) nx.add(vx(i) > 0 ? t : -t);
        if (vy(i)) ny.add(vy(i) > 0 ? t : -t);
      }
    }
    out[0] = 1.0 + fma(nr.value(), 1.0 / 12.0, r.value<EXACT>());
    jx = px.plus_twelfth(nx);
    jy = py.plus_twelfth(ny);
    const float q = __fmul_rn(nr.hi, 1.f / 12.f);  // for the binary32 division below
    r.add(q);
    r.lo += (fmaf(-12.f, q, nr.hi) + nr.lo) * (1.f / 12.f);
  } else {
    out[0] = 1.0 + r.value<EXACT>();
    jx = px.rounded();
    jy = py.rounded();
  }
  PairSum rr;
  rr.hi = 1.f;
  rr.add(r.hi);
  rr.lo += r.lo;
  const float ir = 1.f / rr.rounded();  // binary32: GB300's binary64 divide is slow
  out[1] = widen(jx * ir);
  out[2] = widen(jy * ir);
  out[3] = qx.value<EXACT>();
  out[4] = qy.value<EXACT>();
  return isfinite(jx * ir + (qx.hi + qy.hi));
}

// Macroscopic fields.  One cell per thread, rows of a block's columns; the ghost columns hold the
// periodic x-neighbours, so a cell's 27 values are at fixed offsets from its three rows.  For
// binary32 and binary16 storage the sums are exact binary32 pairs, and only what a result
// cannot do without is binary64 (four additions per cell, one for binary16): with conversions and
// additions of every sum in binary64 the binary64 units set the time.  Binary16 values are
// multiples of 2^-24, so while a sum's magnitudes add up to at most 1 (|f_i - w_i|, |g_i| ~ 0.1
// in any flow this model is valid for) plain binary32 additions are exact and the pairs are not
// needed; other cells take them.  Cold caches, conversions and sums in binary64 -> now: binary32
// 2048^2 125 -> 91 us (memory: 92), binary16 4096^2 436 -> 268, relative binary16 2048^2 844 -> 88.
// The values that a cell pulls, as stored.
template <typename T, bool REL>
struct CellValues {
  T v[27];
  T U[REL ? 8 : 1][2];  // of the source cell of f_(k+1): U_x where c_x != 0, U_y where c_y != 0
  // WRAP: west of column 0 its original instead of the ghost copy, whose sector holds nothing else of a
  // narrow row (the offsets are no constants then: 2000^2 binary32 107 -> 141 us; the copies in the east
  // share sectors: 16 x 65536 binary32 54 -> 61 us without them).
  template <bool WRAP = false>
  __device__ __forceinline__ void load(const T* __restrict__ pops, const StepGeom& g, int x, int y) {
    const T* rows[3];  // rows y - 1, y, y + 1 (sources of c_y = 1, 0, -1) at column x
#pragma unroll
    for (int k = 0; k < 3; ++k) rows[k] = pops + (size_t)wrapi(y - 1 + k, g.ny) * g.pitch + kXOff + x;
    const int west = WRAP && x == 0 ? g.nx - 1 : -1;
    auto at = [&](int plane, int i) {
      const T* p = rows[1 - vy(i)] + (size_t)plane * g.plane;
      if constexpr (WRAP) return p[vx(i) > 0 ? west : -vx(i)];
      else return p[-vx(i)];
    };
#pragma unroll
    for (int q = 0; q < 27; ++q) v[q] = at(plane_of(q), q % 9);
    if constexpr (REL) {
#pragma unroll
      for (int i = 1; i < 9; ++i) {
        if (vx(i)) U[i - 1][0] = at(kQ, i);
        if (vy(i)) U[i - 1][1] = at(kQ + 1, i);
      }
    }
  }
  // (false: moments_of's, for the relative form only)
  __device__ __forceinline__ bool moments(double (&out)[5]) const {
    if constexpr (sizeof(T) == 8) {
      // with the terms of zero c left out and one reciprocal for both velocities 46 binary64
      // instructions a cell instead of 62: 2048^2 497 -> 363 us
      double r = v[0], jx = v[1], jy = v[2], sbx = v[9], sby = v[18];
#pragma unroll
      for (int i = 1; i < 9; ++i) {
        r += v[i];
        if (i > 1 && vx(i)) jx += vx(i) * v[i];
        if (i > 2 && vy(i)) jy += vy(i) * v[i];
        sbx += v[9 + i];
        sby += v[18 + i];
      }
      out[0] = 1.0 + r;
      out[3] = sbx;
      out[4] = sby;
      if (quotient_in_range(jx, out[0]) && quotient_in_range(jy, out[0])) {
        const double y = __drcp_rn(out[0]);
        out[1] = quotient(jx, out[0], y);
        out[2] = quotient(jy, out[0], y);
      } else {  // extreme values, infinities and NaN
        jx = jy = 0.0;
#pragma unroll
        for (int i = 0; i < 9; ++i) {
          jx += vx(i) * v[i];
          jy += vy(i) * v[i];
        }
        out[1] = jx / out[0];
        out[2] = jy / out[0];
      }
      return true;
    } else {
      float w[27], W[8][2] = {};
#pragma unroll
      for (int q = 0; q < 27; ++q) w[q] = load_as<float>(v[q]);
      if constexpr (REL) {
#pragma unroll
        for (int i = 1; i < 9; ++i) {
          if (vx(i)) W[i - 1][0] = load_as<float>(U[i - 1][0]);
          if (vy(i)) W[i - 1][1] = load_as<float>(U[i - 1][1]);
        }
      }
      if constexpr (sizeof(T) == 2) {
        float a[3] = {0.f, 0.f, 0.f};
#pragma unroll
        for (int q = 0; q < 27; ++q) a[q / 9] += fabsf(w[q]);
        if (a[0] <= 1.f && a[1] <= 1.f && a[2] <= 1.f) return moments_of<true, REL>(w, W, out);
        return moments_of<false, REL>(w, W, out);
      } else {
        return moments_of<false, REL>(w, W, out);
      }
    }
  }
};

// Moments of a cell of the relative binary16 form with infinities or NaN among its values, from
// binary64 sums: the pair sums make NaN of an infinite population, where rho is infinite.  For states that
// have diverged: a loop over the populations, so that it takes no registers from the others (1025 x 1024
// 27.9 us with a call, 27.6 now, 27.5 without).
template <typename T>
__device__ __forceinline__ void moments_diverged(const T* __restrict__ pops, const StepGeom& g, int x, int y,
                                                 double (&out)[5]) {
  double r = 0, jx = 0, jy = 0, sbx = 0, sby = 0;
#pragma unroll 1
  for (int i = 0; i < 9; ++i) {
    const int cx = vx(i), cy = vy(i);
    const T* p = pops + (size_t)wrapi(y - cy, g.ny) * g.pitch + kXOff + wrapi(x - cx, g.nx);
    double f = load_as<double>(p[(size_t)plane_of(i) * g.plane]);
    if (i > 0) {
      const double Ux = load_as<double>(p[(size_t)kQ * g.plane]), Uy = load_as<double>(p[(size_t)(kQ + 1) * g.plane]);
      f += 3.0 * wt(i) * (cx * Ux + cy * Uy);
    }
    r += f;
    jx += cx * f;
    jy += cy * f;
    sbx += load_as<double>(p[(size_t)plane_of(9 + i) * g.plane]);
    sby += load_as<double>(p[(size_t)plane_of(18 + i) * g.plane]);
  }
  out[0] = 1.0 + r;
  const float ir = 1.f / (float)out[0];
  out[1] = (double)((float)jx * ir);
  out[2] = (double)((float)jy * ir);
  out[3] = sbx;
  out[4] = sby;
}

// out <- moments of cell (x, y), whose values are loaded.
template <typename T, bool REL>
__device__ __forceinline__ void cell_moments(const CellValues<T, REL>& cell, const T* __restrict__ pops,
                                             const StepGeom& g, int x, int y, double (&out)[5]) {
  const bool finite = cell.moments(out);
  if constexpr (REL) {
    if (!finite) moments_diverged(pops, g, x, y, out);
  }
}

// ROWS: several rows per block.  WRAP: CellValues::load's, for grids of up to kWrapCols columns.
constexpr int kWrapCols = 16;
template <typename T, bool REL, bool ROWS, bool WRAP>
__global__ void __launch_bounds__(ROWS ? 256 : 128)
    moments_kernel(const T* __restrict__ pops, StepGeom g, double* __restrict__ rho, double* __restrict__ ux,
                   double* __restrict__ uy, double* __restrict__ bx, double* __restrict__ by) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= g.nx) return;
  // (a block's one row is known to be the same in all threads: with the row per thread 2048^2 binary32
  // took 113 instead of 99 us)
  const int rows = ROWS ? blockDim.y : 1, y0 = blockIdx.y * rows + (ROWS ? threadIdx.y : 0);
  for (int y = y0; y < g.ny; y += gridDim.y * rows) {
    const size_t c = (size_t)y * g.nx + x;
    double out[5];
    CellValues<T, REL> cell;
    cell.template load<WRAP>(pops, g, x, y);
    cell_moments(cell, pops, g, x, y, out);
    rho[c] = out[0];
    ux[c] = out[1];
    uy[c] = out[2];
    bx[c] = out[3];
    by[c] = out[4];
  }
}

// Diagnostics of a binary32 or binary16 state, one record per block (lbmhd_diag.cuh has the slots and
// the reduction's parts): the moments of a row are formed as moments_kernel forms them and used
// at once, so that reading the populations runs under the reduction's binary64 instructions,
// which bound it (30 per cell), and the moment fields are neither written nor read.  A block
// marches a 128-column tile down its rows.  B of a row passes through shared memory to the
// neighbouring columns; the columns beside the tile come in as single stored values, one per
// thread and two rows ahead, which four lanes of one warp, another one each row, add up.  One
// tile per block, four blocks per SM, tiles of at least one row: a small grid takes the time of
// three rows.  The next row's populations are loaded before this row's binary64 work where the
// registers allow it (not with REL's eight more values).  Cells of the relative form whose values are not
// finite make NaN of an infinite moment; lbmhd_diagnostics then takes the way through the fields.
// Kernels at 2048^2 binary32: moments 98 + reduction 224 -> 268 us.
// Call of lbmhd_diagnostics with moments and reduction apart -> now: binary32 64^2 57 -> 48, 256^2 59
// -> 58, 1024^2 146 -> 123, 2048^2 369 -> 307 us; binary16 2048^2 341 -> 281, relative 358 -> 330.
// Three, five or six blocks per SM: 439, 343, 383 (binary32, 2048^2); REL with the early loads 396.
constexpr int kDiagPopsBlocks = 4 * 152;
static_assert(kDiagPopsBlocks <= kDiagBlocks, "one record per block");
template <typename T, bool REL = false>
__global__ void __launch_bounds__(kDiagThreads, 4)
    diag_pops_kernel(const T* __restrict__ pops, StepGeom g, DiagTiles t, double* __restrict__ partials) {
  static_assert(sizeof(T) <= 4, "binary32 sums");
  constexpr bool kAhead = !REL;
  __shared__ double sh[kDiagSlots][kDiagThreads];
  __shared__ double sb[2][2][kDiagThreads + 2];  // [row parity][B_x, B_y][column x0 - 1 + .]
  __shared__ T hs[2][2][18];  // [row parity][west, east][stored g value]
  const int nx = g.nx, ny = g.ny, tid = threadIdx.x;
  DiagAcc acc;
  acc.clear();
  for (long tile = blockIdx.x; tile < t.tiles; tile += gridDim.x) {
    const int x0 = (int)(tile % t.strips) * kDiagThreads, cols = min(kDiagThreads, nx - x0);
    const int y0 = (int)(tile / t.strips) * t.rows, y1 = min(y0 + t.rows, ny);
    // threads 0 .. 35: one stored g value of the column west (0 .. 17) or east of the tile
    const bool halo = tid < 36;
    const int side = tid / 18, q = 9 + tid % 18, i = q % 9;
    const int hx = side ? (x0 + cols == nx ? 0 : x0 + cols) : (x0 == 0 ? nx - 1 : x0 - 1);
    auto load_halo = [&](int y) {  // y <= y1 + 2
      int yy = y - vel_y(i);
      yy = yy < 0 ? yy + ny : yy % ny;
      return pops[(size_t)yy * g.pitch + (size_t)plane_of(q) * g.plane + kXOff + hx - vel_x(i)];
    };
    T hv = T(0);
    if (halo) {
      hs[1][side][q - 9] = load_halo(y0 - 1);
      hv = load_halo(y0);
    }
    DiagRows rows;
    CellValues<T, REL> cell;
    if (kAhead && tid < cols) cell.load(pops, g, x0 + tid, wrapi(y0 - 1, ny));
    __syncthreads();
    for (int y = y0 - 1; y <= y1; ++y) {  // row y arrives in slot 2
      const int par = (y - y0) & 1;
      double m[5];
      if (halo) {
        hs[par ^ 1][side][q - 9] = hv;  // row y + 1
        if (y < y1) hv = load_halo(y + 2);
      }
      if (tid < cols) {
        if (!kAhead) cell.load(pops, g, x0 + tid, wrapi(y, ny));
        cell.moments(m);
        if (kAhead && y < y1) cell.load(pops, g, x0 + tid, wrapi(y + 1, ny));
        sb[par][0][tid + 1] = m[3];
        sb[par][1][tid + 1] = m[4];
        if (y >= y0 && y < y1) acc.add_cell(m[0], m[1], m[2], m[3], m[4]);
      }
      const int lane = tid - (((y - y0) & 3) << 5);
      if (lane >= 0 && lane < 4) {  // B_x, B_y beside the tile, summed as CellValues::moments does
        const T* h = hs[par][lane >> 1] + 9 * (lane & 1);
        PairSum p;
#pragma unroll
        for (int k = 0; k < 9; ++k) p.add(load_as<float>(h[k]));
        sb[par][lane & 1][lane >> 1 ? cols + 1 : 0] = p.value();
      }
      __syncthreads();  // the buffers of this parity are rewritten after the next row's barrier
      if (tid < cols) {
#pragma unroll
        for (int f = 0; f < 2; ++f) rows.set(f, 2, m[3 + f], sb[par][f][tid + 2], sb[par][f][tid]);
        if (y > y0) rows.add_to(acc);
        rows.advance();
      }
    }
    __syncthreads();
  }
  diag_record(acc, sh, partials + (size_t)blockIdx.x * kDiagSlots);
}

template <typename T, bool REL = false>
__global__ void populations_kernel(const T* __restrict__ pops, StepGeom g, double* __restrict__ out) {
  const long n = (long)g.nx * g.ny;
  for (long c = blockIdx.x * (long)blockDim.x + threadIdx.x; c < n; c += (long)gridDim.x * blockDim.x) {
    const int x = (int)(c % g.nx), y = (int)(c / g.nx);
    double v[27];
    pull_cell<T, REL>(pops, g, x, y, v);
#pragma unroll
    for (int q = 0; q < 27; ++q) out[(size_t)q * n + c] = q < 9 ? v[q] + wt(q) : v[q];
  }
}

int grid_for(long n, int threads) {
  long b = (n + threads - 1) / threads;
  if (b > 152L * 16) b = 152L * 16;
  if (b < 1) b = 1;
  return (int)b;
}

}  // namespace

cudaError_t launch_init_eq(int precision, void* pops, const StepGeom& g, const double* rho,
                           const double* ux, const double* uy, const double* bx, const double* by,
                           cudaStream_t s) {
  const dim3 grid((g.nx + kInitCols - 1) / kInitCols,
                  (unsigned)std::min((g.ny + kInitRows - 1) / kInitRows, 65535));
  if (precision == 0)
    init_eq_kernel<double><<<grid, kInitCols, 0, s>>>((double*)pops, g, rho, ux, uy, bx, by);
  else if (precision == 1)
    init_eq_kernel<float><<<grid, kInitCols, 0, s>>>((float*)pops, g, rho, ux, uy, bx, by);
  else if (precision == LBMHD_FP16)
    init_eq_kernel<__half><<<grid, kInitCols, 0, s>>>((__half*)pops, g, rho, ux, uy, bx, by);
  else
    init_eq_kernel<__half, true><<<grid, kInitCols, 0, s>>>((__half*)pops, g, rho, ux, uy, bx, by);
  return cudaGetLastError();
}

// Zero the row padding of both population copies: physical columns [0, kXOff - 2) and
// [nx + kXOff + 2, plane) of every plane row.  One thread per padding element; a warp covers a
// row's contiguous run.  (cudaMemset2DAsync over the same 110,592 row pieces at 2048^2 took
// 0.12 ms.)
template <typename W>
__global__ void zero_pads_kernel(W* __restrict__ p0, W* __restrict__ p1, StepGeom g, long rows) {
  const int left = kXOff - 2, right0 = g.nx + kXOff + 2, padw = left + (g.plane - right0);
  const long n = 2 * rows * padw;
  for (long k = blockIdx.x * (long)blockDim.x + threadIdx.x; k < n; k += (long)gridDim.x * blockDim.x) {
    const long rr = k / padw;
    const int j = (int)(k - rr * padw);
    const long row = rr < rows ? rr : rr - rows;
    W* base = rr < rows ? p0 : p1;
    base[(size_t)row * g.plane + (j < left ? j : right0 + (j - left))] = W(0);
  }
}

cudaError_t launch_zero_pads(void* pops0, void* pops1, const StepGeom& g, int nplanes, size_t elem,
                             cudaStream_t s) {
  const long rows = (long)nplanes * g.ny;
  const long n = 2 * rows * (kXOff - 2 + g.plane - (g.nx + kXOff + 2));
  const int grid = grid_for(n, 256);
  if (elem == 8)
    zero_pads_kernel<unsigned long long><<<grid, 256, 0, s>>>((unsigned long long*)pops0,
                                                             (unsigned long long*)pops1, g, rows);
  else if (elem == 4)
    zero_pads_kernel<unsigned><<<grid, 256, 0, s>>>((unsigned*)pops0, (unsigned*)pops1, g, rows);
  else
    zero_pads_kernel<unsigned short><<<grid, 256, 0, s>>>((unsigned short*)pops0,
                                                         (unsigned short*)pops1, g, rows);
  return cudaGetLastError();
}

template <typename T, bool REL = false>
cudaError_t launch_moments_of(const void* pops, const StepGeom& g, double* rho, double* ux, double* uy, double* bx,
                              double* by, cudaStream_t s) {
  // Blocks of several whole rows up to 127 columns, strips of equal width beyond: a block of one row
  // left most lanes idle on narrow grids.  Threads over consecutive cells without ghost columns / one
  // row a block / now: 3 x 262144 binary64 147 / 727 / 147 us, binary32 142 / 193 / 141; 16 x 65536
  // binary64 129 / 187 / 99, binary32 48 / 58 / 54; 65 x 16384 binary64 129 / 142 / 113.
  dim3 nt(g.nx, 1);
  if (g.nx < 128) {
    // (as few rows as keep four blocks on every SM: 64^2 in blocks of four rows leaves most SMs idle)
    nt.y = std::max(1, std::min(256 / g.nx, g.ny / (4 * 152)));
  } else {
    const int strips = (g.nx + 127) / 128;
    nt.x = ((g.nx + strips - 1) / strips + 31) / 32 * 32;
  }
  const dim3 grid((g.nx + nt.x - 1) / nt.x, std::min((g.ny + nt.y - 1) / nt.y, 65535u));
  const auto kernel = g.nx <= kWrapCols ? moments_kernel<T, REL, true, true>
                      : nt.y > 1        ? moments_kernel<T, REL, true, false>
                                        : moments_kernel<T, REL, false, false>;
  kernel<<<grid, nt, 0, s>>>(static_cast<const T*>(pops), g, rho, ux, uy, bx, by);
  return cudaGetLastError();
}

cudaError_t launch_moments(int precision, const void* pops, const StepGeom& g, double* rho,
                           double* ux, double* uy, double* bx, double* by, cudaStream_t s) {
  if (precision == 0) return launch_moments_of<double>(pops, g, rho, ux, uy, bx, by, s);
  if (precision == 1) return launch_moments_of<float>(pops, g, rho, ux, uy, bx, by, s);
  if (precision == LBMHD_FP16) return launch_moments_of<__half>(pops, g, rho, ux, uy, bx, by, s);
  return launch_moments_of<__half, true>(pops, g, rho, ux, uy, bx, by, s);
}

cudaError_t launch_populations(int precision, const void* pops, const StepGeom& g, double* out,
                               cudaStream_t s) {
  const int grid = grid_for((long)g.nx * g.ny, 256);
  if (precision == 0)
    populations_kernel<double><<<grid, 256, 0, s>>>((const double*)pops, g, out);
  else if (precision == 1)
    populations_kernel<float><<<grid, 256, 0, s>>>((const float*)pops, g, out);
  else if (precision == LBMHD_FP16)
    populations_kernel<__half><<<grid, 256, 0, s>>>((const __half*)pops, g, out);
  else
    populations_kernel<__half, true><<<grid, 256, 0, s>>>((const __half*)pops, g, out);
  return cudaGetLastError();
}

// Binary64 moments take 46 binary64 instructions a cell, too many to form them again in the tiles' halo
// rows: lbmhd_diagnostics at 256^2 57 us through the fields, 75 straight from the populations; 1024^2 205
// and 222; 2048^2 636 and 661 (below that 128^2 56.5 and 54.3).  The tiles of
// diag_pops_kernel are one grid wide, so on narrow grids most of their lanes idle: from three rows a
// block on the grouped pieces over the fields are faster (binary32, straight / through the fields: 16 x
// 256 48 / 50 us, 16 x 1024 53 / 53, 16 x 2048 62 / 56, 16 x 65536 388 / 163, 63 x 65536 448 / 379).
bool diagnostics_through_fields(int precision, int nx, int ny) {
  return precision == 0 || (nx <= kDiagThreads / 2 && ny > 2 * kDiagPopsBlocks);
}

cudaError_t launch_diagnostics(int precision, const void* pops, const StepGeom& g, double* fields, double* partials,
                               double* out, bool through_fields, cudaStream_t s) {
  const DiagTiles t = through_fields ? diag_tiles(g.nx, g.ny, kDiagBlocks, true, kDiagMinRows)
                                     : diag_tiles(g.nx, g.ny, kDiagPopsBlocks, false, 1);
  if (through_fields) {
    const size_t n = (size_t)g.nx * g.ny;
    cudaError_t e = launch_moments(precision, pops, g, fields, fields + n, fields + 2 * n, fields + 3 * n,
                                   fields + 4 * n, s);
    if (e != cudaSuccess) return e;
    launch_diag_partials(fields, fields + n, fields + 2 * n, fields + 3 * n, fields + 4 * n, g.nx, g.ny, t, partials, s);
  } else if (precision == 1) {
    diag_pops_kernel<float><<<t.blocks, kDiagThreads, 0, s>>>((const float*)pops, g, t, partials);
  } else if (precision == LBMHD_FP16) {
    diag_pops_kernel<__half><<<t.blocks, kDiagThreads, 0, s>>>((const __half*)pops, g, t, partials);
  } else {
    diag_pops_kernel<__half, true><<<t.blocks, kDiagThreads, 0, s>>>((const __half*)pops, g, t, partials);
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  diag_final_kernel<<<1, 32 * kDiagSlots, 0, s>>>(partials, t.blocks, out);
  return cudaGetLastError();
}

}  // namespace lbmhd_gpu
