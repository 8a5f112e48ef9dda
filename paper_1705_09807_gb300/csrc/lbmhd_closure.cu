// Learned subgrid correction: a 3-layer periodic 3x3 convolutional network (12 -> 32 -> 32 -> 4
// channels, tanh after the first two layers) that predicts the residual between the exact
// filtered subgrid terms and the analytic Delta^2/12 closure of Sec. 2.1 / Sec. 3.  This file
// holds its training kernels (binary32 forward, back-propagation, Adam), its inference kernel
// (all three layers fused in one kernel on the 5th-generation tensor cores: bf16 operands in
// shared memory, tcgen05.mma, fp32 accumulators in tensor memory), and the kernels that build
// features and training targets from filtered fine-grid fields.
//
// Conventions (shared with the C ABI): activations are [batch][channel][H][W] binary32 planes on
// a periodic H x W grid; parameters are one flat binary32 vector holding, per layer,
// W[co][ci][dy+1][dx+1] then b[co], with y[co](x) = b[co] + sum W[co][ci][dy+1][dx+1] a[ci](x+(dx,dy)).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "lbmhd.h"
#include "lbmhd_handle.h"
#include "lbmhd_internal.cuh"
#include "lbmhd_quotient.cuh"
#include "lbmhd_ptx.cuh"

namespace lbmhd_gpu {
namespace {

constexpr int kC0 = 12, kC1 = 32, kC2 = 32, kC3 = 4;
constexpr int kP1 = kC1 * kC0 * 9 + kC1;          // 3488
constexpr int kP2 = kC2 * kC1 * 9 + kC2;          // 9248
constexpr int kP3 = kC3 * kC2 * 9 + kC3;          // 1156
constexpr int kNumParams = kP1 + kP2 + kP3;       // 13892
constexpr int kThreads = 256;
constexpr int kMaxConvBlocks = 2 * 152;           // blocks of a convolution: two per SM
constexpr uint64_t kNetWaitNs = 2000000000ull;    // bound of every tensor-core completion wait

__device__ __forceinline__ int wrapi(int i, int n) { return i < 0 ? i + n : (i >= n ? i - n : i); }

// ---- binary32 convolutions (forward and data gradient) ----------------------------------------
// One kernel for y[o](x) = b[o] + sum_i sum_t w[o][i][t] in[i](x + d_t) (forward) and, BWD, for
// da[o](z) = sum_i sum_t W[i][o][t] dy[i](z - d_t) (W as the layer stores it).  Bound by binary32
// FMAs, so the operands have to reach registers by few instructions: a thread computes 4
// adjacent cells x 16 outputs (4 for the last layer), and one 16-byte shared-memory load of
// weights (all lanes the same address) feeds 16 FMAs, where one thread per cell needed a load per
// FMA.  Input channels arrive four at a time in two buffers (cp.async), the next four in flight
// while these are used; a block walks tiles with the weights kept in shared memory.  Each
// output's sum runs over channels, then taps, as with one thread per cell, so results are bitwise
// the same.  At 8 x 256^2: 32 -> 32 forward 567 -> 199 us (48 TFLOP/s; the FMA units reach about
// 75), its data gradient 425 -> 191 us, 12 -> 32 221 -> 86 us, 32 -> 4 with the loss 147 -> 53 us.
constexpr int kTileW = 32;        // tile width: 8 threads of 4 cells
constexpr int kConvThreads = 256;
constexpr int kConvChunk = 4;     // input channels per buffer
constexpr int kTilePitch = 36;    // floats per staged row: columns -1 .. 32, padded to 16 bytes

enum ConvEpilogue { kEpiNone, kEpiTanh, kEpiTanhGrad, kEpiLoss };

template <int CIN, int COUT>
struct ConvShape {
  static constexpr int kOuts = COUT < 16 ? COUT : 16;       // outputs per thread
  static constexpr int kGroups = COUT / kOuts;              // groups of warps over outputs
  static constexpr int kRows = 4 * kConvThreads / kGroups / kTileW;
  static constexpr int kRowElems = (kRows + 2) * kTilePitch;
  static constexpr int kLoads = ((kRows + 2) * (kTileW + 2) + kConvThreads - 1) / kConvThreads;
  static constexpr size_t kSmem = (CIN * 9 * COUT + 2 * kConvChunk * kRowElems) * sizeof(float);
  static_assert(CIN % kConvChunk == 0 && COUT % 4 == 0, "channel counts");
};

__device__ __forceinline__ int wrap_mod(int i, int n) {
  i %= n;
  return i < 0 ? i + n : i;
}

__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// aux: kEpiTanhGrad the activation a (result times 1 - a^2), kEpiLoss the target (result
// (y - target) / n_out, and the block's sum of (y - target)^2 into loss_part[blockIdx.x]).
template <int CIN, int COUT, int EPI, bool BWD>
__global__ void __launch_bounds__(kConvThreads, 2)
    conv_tile_kernel(const float* __restrict__ in, const float* __restrict__ params, const float* __restrict__ aux,
                     int batch, int H, int W, float* __restrict__ out, double* __restrict__ loss_part) {
  using Sh = ConvShape<CIN, COUT>;
  constexpr int NO = Sh::kOuts;
  extern __shared__ __align__(16) float conv_smem[];
  float* sw = conv_smem;                   // [ci][tap][co]
  float* st = conv_smem + CIN * 9 * COUT;  // [2][kConvChunk][row][kTilePitch]
  const int tid = threadIdx.x;
  for (int i = tid; i < CIN * 9 * COUT; i += kConvThreads) {
    const int co = i % COUT, ct = i / COUT, ci = ct / 9, t = ct % 9;
    sw[i] = params[BWD ? (ci * COUT + co) * 9 + t : (co * CIN + ci) * 9 + t];
  }
  const int o0 = tid / (kConvThreads / Sh::kGroups) * NO;
  const int xg = tid % 8, yy = tid % (kConvThreads / Sh::kGroups) / 8;
  const size_t plane = (size_t)H * W;
  const int tiles_x = (W + kTileW - 1) / kTileW, tiles_y = (H + Sh::kRows - 1) / Sh::kRows;
  const long ntiles = (long)batch * tiles_x * tiles_y;
  // 16-byte stores need rows of whole quads on 16-byte boundaries
  const bool vec = W % 4 == 0 && reinterpret_cast<uintptr_t>(out) % 16 == 0;
  const float inv_n = 1.f / (float)((long)batch * COUT * (long)plane);
  double loss = 0.0;

  for (long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int b = (int)(tile / ((long)tiles_x * tiles_y)), rem = (int)(tile % ((long)tiles_x * tiles_y));
    const int y0 = rem / tiles_x * Sh::kRows, x0 = rem % tiles_x * kTileW;
    const float* ib = in + (size_t)b * CIN * plane;
    // this thread's elements of a staged channel (rows y0 - 1 .., columns x0 - 1 .., periodic)
    size_t goff[Sh::kLoads];
    int soff[Sh::kLoads];
#pragma unroll
    for (int k = 0; k < Sh::kLoads; ++k) {
      const int e = tid + k * kConvThreads, r = e / (kTileW + 2), c = e % (kTileW + 2);
      soff[k] = r < Sh::kRows + 2 ? r * kTilePitch + c : -1;
      goff[k] = (size_t)wrap_mod(y0 - 1 + r, H) * W + wrap_mod(x0 - 1 + c, W);
    }
    auto stage = [&](int chunk) {
      float* d = st + (chunk & 1) * kConvChunk * Sh::kRowElems;
      const float* g = ib + (size_t)chunk * kConvChunk * plane;
#pragma unroll
      for (int c = 0; c < kConvChunk; ++c)
#pragma unroll
        for (int k = 0; k < Sh::kLoads; ++k)
          if (soff[k] >= 0) cp_async4(d + c * Sh::kRowElems + soff[k], g + c * plane + goff[k]);
      cp_async_commit();
    };
    float acc[4][NO];
#pragma unroll
    for (int o = 0; o < NO; ++o) {
      const float bv = BWD ? 0.f : params[COUT * CIN * 9 + o0 + o];
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[i][o] = bv;
    }
    stage(0);
    constexpr int kChunks = CIN / kConvChunk;
#pragma unroll 1
    for (int ch = 0; ch < kChunks; ++ch) {
      if (ch + 1 < kChunks) {
        stage(ch + 1);
        cp_async_wait<1>();
      } else {
        cp_async_wait<0>();
      }
      __syncthreads();
      const float* buf = st + (ch & 1) * kConvChunk * Sh::kRowElems + 4 * xg;
#pragma unroll 1
      for (int c = 0; c < kConvChunk; ++c) {
        const float* wc = sw + (size_t)(ch * kConvChunk + c) * 9 * COUT + o0;
#pragma unroll
        for (int r = 0; r < 3; ++r) {
          const float* row = buf + c * Sh::kRowElems + (yy + (BWD ? 2 - r : r)) * kTilePitch;
          const float4 lo4 = *reinterpret_cast<const float4*>(row);
          const float2 hi2 = *reinterpret_cast<const float2*>(row + 4);
          const float v[6] = {lo4.x, lo4.y, lo4.z, lo4.w, hi2.x, hi2.y};
#pragma unroll
          for (int dx = 0; dx < 3; ++dx) {
            float w[NO];
#pragma unroll
            for (int o = 0; o < NO; o += 4)
              *reinterpret_cast<float4*>(&w[o]) = *reinterpret_cast<const float4*>(wc + (r * 3 + dx) * COUT + o);
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
              for (int o = 0; o < NO; ++o) acc[i][o] = fmaf(w[o], v[i + (BWD ? 2 - dx : dx)], acc[i][o]);
          }
        }
      }
      __syncthreads();  // the buffer is refilled two chunks on
    }
    const int y = y0 + yy, x = x0 + 4 * xg;
    const int nv = y < H ? min(4, W - x) : 0;  // cells of this thread inside the grid
    if (nv > 0) {
#pragma unroll
      for (int o = 0; o < NO; ++o) {
        const size_t at = ((size_t)b * COUT + o0 + o) * plane + (size_t)y * W + x;
        float v[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          v[i] = acc[i][o];
          if (EPI == kEpiTanh) v[i] = tanhf(v[i]);
          if (i < nv) {
            if (EPI == kEpiTanhGrad) {
              const float a = aux[at + i];
              v[i] *= (1.f - a * a);
            }
            if (EPI == kEpiLoss) {
              const float d = v[i] - aux[at + i];
              v[i] = d * inv_n;
              loss += (double)d * d;
            }
          }
        }
        if (vec) {
          *reinterpret_cast<float4*>(out + at) = make_float4(v[0], v[1], v[2], v[3]);
        } else {
#pragma unroll
          for (int i = 0; i < 4; ++i)
            if (i < nv) out[at + i] = v[i];
        }
      }
    }
  }
  if constexpr (EPI == kEpiLoss) {
    __shared__ double sh[kConvThreads];
    sh[tid] = loss;
    __syncthreads();
    for (int w = kConvThreads / 2; w > 0; w >>= 1) {
      if (tid < w) sh[tid] += sh[tid + w];
      __syncthreads();
    }
    if (tid == 0) loss_part[blockIdx.x] = sh[0];
  }
}

// Forward convolution with one thread per cell (all outputs; weights a shared-memory load per FMA): for
// sets of narrow, low or small grids, whose tiles are mostly empty (conv).  Same order of sums, so
// the results are bitwise those of the tiles.
template <int CIN, int COUT, bool TANH>
__global__ void __launch_bounds__(kThreads)
    conv_cell_kernel(const float* __restrict__ in, const float* __restrict__ params, int batch, int H, int W,
                     float* __restrict__ out) {
  __shared__ float sw[COUT * CIN * 9 + COUT];
  for (int i = threadIdx.x; i < COUT * CIN * 9 + COUT; i += blockDim.x) sw[i] = params[i];
  __syncthreads();
  const long plane = (long)H * W, total = (long)batch * plane;
  for (long c = blockIdx.x * (long)blockDim.x + threadIdx.x; c < total; c += (long)gridDim.x * blockDim.x) {
    const int b = (int)(c / plane);
    const long cell = c % plane;
    const int y = (int)(cell / W), x = (int)(cell % W);
    long off[9];
#pragma unroll
    for (int t = 0; t < 9; ++t) off[t] = (long)wrapi(y + t / 3 - 1, H) * W + wrapi(x + t % 3 - 1, W);
    float acc[COUT];
#pragma unroll
    for (int co = 0; co < COUT; ++co) acc[co] = sw[COUT * CIN * 9 + co];
    const float* ib = in + (size_t)b * CIN * plane;
    for (int ci = 0; ci < CIN; ++ci) {
#pragma unroll
      for (int t = 0; t < 9; ++t) {
        const float v = ib[(size_t)ci * plane + off[t]];
#pragma unroll
        for (int co = 0; co < COUT; ++co) acc[co] = fmaf(sw[(co * CIN + ci) * 9 + t], v, acc[co]);
      }
    }
    float* ob = out + (size_t)b * COUT * plane + cell;
#pragma unroll
    for (int co = 0; co < COUT; ++co) ob[(size_t)co * plane] = TANH ? tanhf(acc[co]) : acc[co];
  }
}

// ---- weight gradients ----------------------------------------------------------------------------
// dW[co][ci][t] = sum_z dy[co](z) a[ci](z + d_t), db[co] = sum_z dy[co](z).  Bound by binary32 FMAs
// (18,432 flops per cell for the 32 x 32 layer).  Lane l of a warp holds channel l of the
// 32-channel operand ("lane": dy for layers 1 and 2, a for layer 3), a warp NW channels of the
// other ("window"), so a thread keeps NW x 9 sums in registers; per 8 cells it takes 2 16-byte
// loads of its lane's values and 3 loads per window row, the same address in every lane, for 72
// NW FMAs.  A block stages 32 x 8 cells of both operands in shared memory; its warps split the
// window channels, and the rows where there are fewer than eight groups of them.  Sums are
// kept per tile and then added to a running sum, so binary32 rounding grows with the tiles, not
// the cells; blocks write partial sums that sum_partials_kernel adds in block order
// (deterministic).  At 8 x 256^2 the three layers took 20.6 (32 x 32), 7.8 (12 x 32) and 2.6 ms
// (32 x 4) with one thread per weight reading both operands from global memory; now 236, 100 and
// 52 us.
constexpr int kWgThreads = 256;
constexpr int kWgRows = 8;
constexpr int kWgCells = kTileW * kWgRows;      // 256: one per thread when staging
constexpr int kWgLanePitch = kWgCells + 4;      // lanes 4 banks apart: conflict-free 16-byte loads
constexpr int kWgWinElems = (kWgRows + 2) * kTilePitch;
static_assert(kWgCells == kWgThreads, "one staged cell per thread and channel");

template <int NWIN>
__host__ __device__ constexpr size_t wgrad_smem() {
  return (32 * kWgLanePitch + NWIN * kWgWinElems) * sizeof(float);
}

// NWIN window channels in all, NW per warp.  LANE_DY: lane = dy [32 channels], window = a [NWIN];
// else lane = a, window = dy (its tap t offset is -d_t).  part: [block][kNumParams] with this
// layer's parameters from `base`.
template <int NWIN, int NW, bool LANE_DY>
__global__ void __launch_bounds__(kWgThreads, 2)
    conv_wgrad_kernel(const float* __restrict__ lane_op, const float* __restrict__ win_op, int batch, int H, int W,
                      float* __restrict__ part, int base) {
  constexpr int kGroups = NWIN / NW, kSplits = 8 / kGroups;
  static_assert(kGroups * NW == NWIN && kGroups * kSplits == 8, "eight warps");
  extern __shared__ __align__(16) float wg_smem[];
  float* sl = wg_smem;                       // [32][kWgLanePitch]
  float* sn = wg_smem + 32 * kWgLanePitch;   // [NWIN][row][kTilePitch]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int group = warp % kGroups, split = warp / kGroups;
  const size_t plane = (size_t)H * W;
  const int tiles_x = (W + kTileW - 1) / kTileW, tiles_y = (H + kWgRows - 1) / kWgRows;
  const long ntiles = (long)batch * tiles_x * tiles_y;
  float tot[NW * 9], tot_b[NW];
#pragma unroll
  for (int k = 0; k < NW * 9; ++k) tot[k] = 0.f;
#pragma unroll
  for (int k = 0; k < NW; ++k) tot_b[k] = 0.f;

  for (long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int b = (int)(tile / ((long)tiles_x * tiles_y)), rem = (int)(tile % ((long)tiles_x * tiles_y));
    const int y0 = rem / tiles_x * kWgRows, x0 = rem % tiles_x * kTileW;
    const float* lb = lane_op + (size_t)b * 32 * plane;
    const float* wb = win_op + (size_t)b * NWIN * plane;
    {  // lane operand: cell tid of every channel, zero outside the grid
      const int y = y0 + tid / kTileW, x = x0 + tid % kTileW;
      const bool in = y < H && x < W;
      const float* src = lb + (in ? (size_t)y * W + x : 0);
#pragma unroll 8
      for (int c = 0; c < 32; ++c) {
        if (in) cp_async4(sl + c * kWgLanePitch + tid, src + c * plane);
        else sl[c * kWgLanePitch + tid] = 0.f;
      }
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {  // window operand: rows y0 - 1 .., columns x0 - 1 .., periodic
      const int e = tid + k * kWgThreads, r = e / (kTileW + 2), c = e % (kTileW + 2);
      if (r < kWgRows + 2) {
        const float* src = wb + (size_t)wrap_mod(y0 - 1 + r, H) * W + wrap_mod(x0 - 1 + c, W);
        float* dst = sn + r * kTilePitch + c;
#pragma unroll 4
        for (int ch = 0; ch < NWIN; ++ch) cp_async4(dst + ch * kWgWinElems, src + ch * plane);
      }
    }
    cp_async_commit();
    cp_async_wait<0>();
    __syncthreads();
    float acc[NW * 9], acc_b[NW];
#pragma unroll
    for (int k = 0; k < NW * 9; ++k) acc[k] = 0.f;
#pragma unroll
    for (int k = 0; k < NW; ++k) acc_b[k] = 0.f;
#pragma unroll 1
    for (int q = split; q < kWgCells / 8; q += kSplits) {  // 8 cells of one row at a time
      const int row = q / (kTileW / 8), col = q % (kTileW / 8) * 8;
      float l[8];
      const float* lp = sl + lane * kWgLanePitch + row * kTileW + col;
      *reinterpret_cast<float4*>(&l[0]) = *reinterpret_cast<const float4*>(lp);
      *reinterpret_cast<float4*>(&l[4]) = *reinterpret_cast<const float4*>(lp + 4);
      const float* wp = sn + group * NW * kWgWinElems + row * kTilePitch + col;
#pragma unroll
      for (int n = 0; n < NW; ++n) {
#pragma unroll
        for (int r = 0; r < 3; ++r) {
          float w[10];
          const float* p = wp + n * kWgWinElems + r * kTilePitch;
          *reinterpret_cast<float4*>(&w[0]) = *reinterpret_cast<const float4*>(p);
          *reinterpret_cast<float4*>(&w[4]) = *reinterpret_cast<const float4*>(p + 4);
          *reinterpret_cast<float2*>(&w[8]) = *reinterpret_cast<const float2*>(p + 8);
#pragma unroll
          for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int dx = 0; dx < 3; ++dx) acc[n * 9 + r * 3 + dx] = fmaf(l[i], w[i + dx], acc[n * 9 + r * 3 + dx]);
          if (!LANE_DY && r == 1) {
            // db of window channel n: the cells' own values, those inside the grid (the lane
            // operand is zero outside, the window wraps)
            const int nc = y0 + row < H ? W - x0 - col : 0;
#pragma unroll
            for (int i = 0; i < 8; ++i) acc_b[n] += i < nc ? w[i + 1] : 0.f;
          }
        }
      }
      if (LANE_DY && group == 0) {
#pragma unroll
        for (int i = 0; i < 8; ++i) acc_b[0] += l[i];
      }
    }
#pragma unroll
    for (int k = 0; k < NW * 9; ++k) tot[k] += acc[k];
#pragma unroll
    for (int k = 0; k < NW; ++k) tot_b[k] += acc_b[k];
    __syncthreads();
  }
  // add the row splits in order (staging buffers free), then store this block's partial sums
  float* out = part + (size_t)blockIdx.x * kNumParams + base;
  float* red = wg_smem;  // [group][value][lane]
  constexpr int NV = NW * 9 + NW;
  static_assert(kGroups * NV * 32 * sizeof(float) <= wgrad_smem<NWIN>(), "reduction fits");
  for (int sidx = 1; sidx < kSplits; ++sidx) {
    if (split == sidx) {
#pragma unroll
      for (int k = 0; k < NW * 9; ++k) red[(group * NV + k) * 32 + lane] = tot[k];
#pragma unroll
      for (int k = 0; k < NW; ++k) red[(group * NV + NW * 9 + k) * 32 + lane] = tot_b[k];
    }
    __syncthreads();
    if (split == 0) {
#pragma unroll
      for (int k = 0; k < NW * 9; ++k) tot[k] += red[(group * NV + k) * 32 + lane];
#pragma unroll
      for (int k = 0; k < NW; ++k) tot_b[k] += red[(group * NV + NW * 9 + k) * 32 + lane];
    }
    __syncthreads();
  }
  if (split == 0) {
#pragma unroll
    for (int n = 0; n < NW; ++n) {
      const int wch = group * NW + n;
#pragma unroll
      for (int t = 0; t < 9; ++t) {
        if (LANE_DY) out[(lane * NWIN + wch) * 9 + t] = tot[n * 9 + t];
        else out[(wch * 32 + lane) * 9 + 8 - t] = tot[n * 9 + t];
      }
      if (!LANE_DY && lane == 0) out[NWIN * 32 * 9 + wch] = tot_b[n];
    }
    if (LANE_DY && group == 0) out[32 * NWIN * 9 + lane] = tot_b[0];
  }
}

// Sum the blocks' partial gradients and losses: eight threads per parameter take every eighth
// block in order and are added in order (deterministic).  Block 0 adds up the loss.
__global__ void sum_partials_kernel(const float* __restrict__ part, int nblocks, float* __restrict__ grad,
                                    const double* __restrict__ loss_part, int nloss, double* __restrict__ loss) {
  __shared__ float sh[8][32];
  const int w = blockIdx.x * 32 + threadIdx.x;
  float s = 0.f;
  if (w < kNumParams)
    for (int b = threadIdx.y; b < nblocks; b += 8) s += part[(size_t)b * kNumParams + w];
  sh[threadIdx.y][threadIdx.x] = s;
  __syncthreads();
  if (threadIdx.y == 0 && w < kNumParams) {
    float t = 0.f;
#pragma unroll
    for (int i = 0; i < 8; ++i) t += sh[i][threadIdx.x];
    grad[w] = t;
  }
  if (blockIdx.x == 0) {
    __shared__ double dl[256];
    const int tid = threadIdx.y * 32 + threadIdx.x;
    double d = 0.0;
    for (int b = tid; b < nloss; b += 256) d += loss_part[b];
    dl[tid] = d;
    __syncthreads();
    for (int h = 128; h > 0; h >>= 1) {
      if (tid < h) dl[tid] += dl[tid + h];
      __syncthreads();
    }
    if (tid == 0) *loss = dl[0];
  }
}

__global__ void adam_kernel(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                            float* __restrict__ v, int n, float lr, float b1, float b2, float eps,
                            float c1, float c2) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

// ---- bf16 tensor-core inference: the whole network in one kernel (tcgen05 + TMEM) --------------
// A CTA computes a kTT x kTT tile of the output from a kPS x kPS patch (3 cells of halo, one per
// layer) held in shared memory as bf16.  Each 3x3 layer is, per 128-cell M tile, nine shifted
// implicit GEMMs per 16-channel K chunk, D[cell][co] += A[cell + dy kPS + dx][k] W_tap[co][k],
// issued by one thread as tcgen05.mma (M = 128, N = 32, or 16 for the 4-channel last layer,
// K = 16) with the fp32 accumulators in tensor memory; the epilogue reads them back with
// tcgen05.ld (one cell per thread), adds the bias, applies tanh and stores the next layer's bf16
// input.  The patch is indexed linearly (cell = row kPS + col), so the shifts wrap across rows:
// the results wrapped that way lie in the halo, which shrinks by one cell per layer, and are
// never used by the kept outputs.
//
// Shared-memory operand layouts (no swizzle, K-major core matrices of 8 rows x 16 bytes):
//   activations: [8-channel chunk][cell] x 16 B; consecutive cells 16 B apart, so an 8-cell group
//     is one core matrix (stride byte offset 128 B), the next 8 channels one chunk further
//     (leading byte offset kChunkBytes), and a shift by s cells is a start address 16 s B later.
//   weights: per (tap, 16-channel K chunk) an N x 16 block with (n, k) at (n%8) 16 + (n/8) 256 +
//     (k/8) 128 + (k%8) 2 bytes (leading byte offset 128, stride byte offset 256).
constexpr int kTT = 16;                       // output tile side
constexpr int kPS = kTT + 6;                  // patch side: 22
constexpr int kPatch = kPS * kPS;             // 484 cells
constexpr int kMT = 4;                        // M tiles of every layer: cells 0 .. 511
constexpr int kPadCells = 24;                 // zero cells before and after each chunk (>= kPS + 1)
constexpr int kChunkCells = kPadCells + kMT * 128 + kPadCells;  // 560
constexpr int kChunkBytes = kChunkCells * 16;                   // 8960
constexpr int kW1Bytes = 9 * 1 * 32 * 32;     // taps x K chunks x (N rows x 32 B)
constexpr int kW2Bytes = 9 * 2 * 32 * 32;
// Layer 3 multiplies the unshifted activations once by all nine taps' weights: N = 48 rows
// n = 4 tap + co (36 used), per K chunk; the epilogue sums the nine shifted partial products.
constexpr int kN3 = 48;
constexpr int kW3Bytes = 2 * kN3 * 32;
// partial products P[4 tap + co][cell - kP3Lo] (binary32) for the cells that the kept outputs
// (patch rows / cols 3 .. 18) reach through a tap: 3 kPS + 3 - (kPS + 1) .. 18 kPS + 18 + kPS + 1
constexpr int kP3Lo = 3 * kPS + 3 - (kPS + 1);                  // 46
constexpr int kP3Rows = (18 * kPS + 18 + kPS + 1) - kP3Lo + 1;  // 392
constexpr int kP3Cols = 36;
constexpr int kWBytes = kW1Bytes + kW2Bytes + kW3Bytes;         // 36864
constexpr int kBiasFloats = 32 + 32 + 16;
constexpr int kPackedBytes = kWBytes + kBiasFloats * 4;         // weights then biases
// shared memory map (bytes from the 128-byte aligned base)
constexpr int kSmW = 0;
constexpr int kSmXA = kSmW + kWBytes;                 // features, then layer-2 output (4 chunks)
constexpr int kSmX1 = kSmXA + 4 * kChunkBytes;        // layer-1 output (4 chunks)
constexpr int kSmBias = kSmX1 + 4 * kChunkBytes;      // 80 biases, 4 output scales, 12 1/in_scale
constexpr int kSmBar = kSmBias + (kBiasFloats + 4 + 12) * 4;  // layer barrier, weight-copy barrier
constexpr int kSmSlot = kSmBar + 16;
constexpr int kNetSmemBytes = kSmSlot + 8 + 128;      // + alignment slack
constexpr int kMS = kPS + 2;                          // moment grid side for the features: 24
constexpr uint32_t kTmemCols = 256;  // layers 1, 2: 4 M tiles x 32 fp32 columns; layer 3: 4 x 48
constexpr int kNetThreads = 256;  // 8 warps: warps w and w + 4 share TMEM lanes 32 (w % 4) ..
static_assert(kSmBar % 8 == 0, "mbarrier alignment");
static_assert(5 * kMS * kMS * 4 <= 4 * kChunkBytes, "moments fit in the layer-1 output buffer");
static_assert(kPadCells >= kPS + 1, "shifted reads stay inside a chunk");
static_assert(kP3Lo >= 0 && kP3Lo + kP3Rows <= kMT * 128, "layer-3 partial products lie in the M tiles");
static_assert(kP3Cols * kP3Rows * 4 <= 8 * kChunkBytes, "layer-3 partial products fit in the activation buffers");
static_assert(kMT * kN3 <= (int)kTmemCols, "layer-3 accumulators fit in the TMEM allocation");

// Weights and biases of the three layers in the shared-memory layout above (bf16 weights,
// fp32 biases, zero padding for ci >= CI and co >= CO).
__global__ void pack_net_kernel(const float* __restrict__ params, unsigned char* __restrict__ packed) {
  __nv_bfloat16* w = reinterpret_cast<__nv_bfloat16*>(packed);
  float* bias = reinterpret_cast<float*>(packed + kWBytes);
  const int nw = kWBytes / 2;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nw + kBiasFloats; i += gridDim.x * blockDim.x) {
    if (i >= nw) {
      const int j = i - nw;
      const int layer = j < 32 ? 0 : (j < 64 ? 1 : 2);
      const int co = j - 32 * layer;
      const int CI = layer == 0 ? kC0 : kC1, CO = layer == 2 ? kC3 : kC1;
      const int base = layer == 0 ? 0 : (layer == 1 ? kP1 : kP1 + kP2);
      bias[j] = co < CO ? params[base + CO * CI * 9 + co] : 0.f;
      continue;
    }
    int byte = 2 * i;
    if (byte >= kW1Bytes + kW2Bytes) {
      // layer 3: per K chunk one N = 48 block, row n = 4 tap + co
      byte -= kW1Bytes + kW2Bytes;
      const int kc = byte / (kN3 * 32), in = byte % (kN3 * 32);
      const int n = (in / 256) * 8 + (in % 128) / 16;
      const int k = ((in % 256) / 128) * 8 + (in % 16) / 2;
      const int tap = n / kC3, co = n % kC3, ci = 16 * kc + k;
      w[i] = __float2bfloat16_rn(n < 9 * kC3 && ci < kC2 ? params[kP1 + kP2 + co * kC2 * 9 + ci * 9 + tap] : 0.f);
      continue;
    }
    int N, nkc, CI, CO, base;
    if (byte < kW1Bytes) {
      N = 32, nkc = 1, CI = kC0, CO = kC1, base = 0;
    } else {
      N = 32, nkc = 2, CI = kC1, CO = kC2, base = kP1, byte -= kW1Bytes;
    }
    const int blk = byte / (N * 32), in = byte % (N * 32);
    const int tap = blk / nkc, kc = blk % nkc;
    const int n = (in / 256) * 8 + (in % 128) / 16;
    const int k = ((in % 256) / 128) * 8 + (in % 16) / 2;
    const int ci = 16 * kc + k;
    w[i] = __float2bfloat16_rn(n < CO && ci < CI ? params[base + n * CI * 9 + ci * 9 + tap] : 0.f);
  }
}

__device__ __forceinline__ float tanh_approx(float x) {
  float y;
  asm("tanh.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ uint32_t bf16x2(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}

// Issue one layer: for each M tile, 9 taps x nkc K chunks into TMEM columns mt * n; then commit.
template <int N, int NKC, int FIRST, int NTILES>
__device__ __forceinline__ void issue_layer(uint32_t sbase, int act_off, int w_off, uint32_t tmem, uint64_t* bar) {
  // Descriptors of the layer's first A and B operands; every other operand differs only in its
  // start address, which the descriptor holds in 16-byte units in its low bits (no carry: all
  // addresses lie inside this CTA's shared memory), so it is the base plus a constant.
  constexpr uint32_t idesc = idesc_bf16_f32(128, N);
  const uint64_t a0 = smem_desc(sbase + act_off + (kPadCells + FIRST) * 16, kChunkBytes, 128);
  const uint64_t b0 = smem_desc(sbase + w_off, 128, 256);
#pragma unroll
  for (int mt = 0; mt < NTILES; ++mt) {
#pragma unroll
    for (int tap = 0; tap < 9; ++tap) {
      const int shift = (tap / 3 - 1) * kPS + (tap % 3 - 1);  // cells
#pragma unroll
      for (int kc = 0; kc < NKC; ++kc) {
        const uint64_t a = a0 + (uint64_t)(int64_t)(mt * 128 + shift + 2 * kc * (kChunkBytes / 16));
        const uint64_t b = b0 + (uint64_t)((tap * NKC + kc) * N * 2);
        tc_mma_bf16(tmem + mt * N, a, b, idesc, (tap | kc) != 0);
      }
    }
  }
  tc_commit(bar);
}

// Layer 3 (32 -> 4 channels): per M tile and K chunk ONE MMA of the unshifted activations by the
// N = 48 block of all nine taps' weights (row n = 4 tap + co), into TMEM columns mt * 48.  Column
// 4 t + co of row m then holds the tap-t partial product sum_k A[m][k] W_t[co][k]; the output at
// cell c is sum_t D[c + shift_t][4 t + co] (layer3_epilogue).  The nine shifted MMAs per chunk of
// the other layers re-read the activations nine times from shared memory, the bound of their
// phases; with four output channels that re-read cost layer 3 54 MMAs for 8 here.
__device__ __forceinline__ void issue_layer3(uint32_t sbase, int act_off, int w_off, uint32_t tmem, uint64_t* bar) {
  constexpr uint32_t idesc = idesc_bf16_f32(128, kN3);
  const uint64_t a0 = smem_desc(sbase + act_off + kPadCells * 16, kChunkBytes, 128);
  const uint64_t b0 = smem_desc(sbase + w_off, 128, 256);
#pragma unroll
  for (int mt = 0; mt < kMT; ++mt) {
#pragma unroll
    for (int kc = 0; kc < 2; ++kc) {
      const uint64_t a = a0 + (uint64_t)(mt * 128 + 2 * kc * (kChunkBytes / 16));
      const uint64_t b = b0 + (uint64_t)(kc * kN3 * 2);
      tc_mma_bf16(tmem + mt * kN3, a, b, idesc, kc != 0);
    }
  }
  tc_commit(bar);
}

// Layer-3 partial products TMEM -> shared memory P[col][cell - kP3Lo] (binary32, col = 4 tap +
// co < 36), for the cells kP3Lo .. kP3Lo + kP3Rows - 1.  Warp w reads the 32 lanes of quarter
// w % 4; warps 0-3 take columns 0-15 and 32-35, warps 4-7 columns 16-31.
__device__ __forceinline__ void layer3_partials(uint32_t tmem, float* __restrict__ P) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int quarter = warp & 3, half = warp >> 2;
#pragma unroll 1
  for (int mt = 0; mt < kMT; ++mt) {
    const uint32_t t = tmem + ((uint32_t)(32 * quarter) << 16) + mt * kN3;
    const int row = mt * 128 + 32 * quarter + lane - kP3Lo;
    const bool keep = row >= 0 && row < kP3Rows;
    uint32_t r[16];
    tmem_ld16(t + 16 * half, r);
    if (half == 0) {
      uint32_t q[4];
      tmem_ld4(t + 32, q);
      tmem_ld_wait();
      if (keep) {
#pragma unroll
        for (int j = 0; j < 4; ++j) P[(32 + j) * kP3Rows + row] = __uint_as_float(q[j]);
      }
    } else {
      tmem_ld_wait();
    }
    if (keep) {
#pragma unroll
      for (int j = 0; j < 16; ++j) P[(16 * half + j) * kP3Rows + row] = __uint_as_float(r[j]);
    }
  }
}

// Epilogue of a hidden layer: tanh(D + b) of this thread's cell in each M tile -> bf16 chunks.
// Warp w reads TMEM lanes 32 (w % 4) .. (its cells); warps 0-3 take channels 0-15, warps 4-7
// channels 16-31.
__device__ __forceinline__ void hidden_epilogue(uint32_t tmem, const float* __restrict__ bias,
                                                unsigned char* __restrict__ dst) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int quarter = warp & 3, half = warp >> 2;
#pragma unroll 1
  for (int mt = 0; mt < kMT; ++mt) {
    uint32_t r[16];
    tmem_ld16(tmem + ((uint32_t)(32 * quarter) << 16) + mt * 32 + 16 * half, r);
    tmem_ld_wait();
    const int cell = mt * 128 + 32 * quarter + lane;
    const float* b = bias + 16 * half;
    uint32_t pk[8];
#pragma unroll
    for (int j = 0; j < 8; ++j)
      pk[j] = bf16x2(tanh_approx(__uint_as_float(r[2 * j]) + b[2 * j]),
                     tanh_approx(__uint_as_float(r[2 * j + 1]) + b[2 * j + 1]));
#pragma unroll
    for (int c = 0; c < 2; ++c)
      *reinterpret_cast<uint4*>(dst + (2 * half + c) * kChunkBytes + (kPadCells + cell) * 16) =
          make_uint4(pk[4 * c], pk[4 * c + 1], pk[4 * c + 2], pk[4 * c + 3]);
  }
}

// All CTA threads wait for the layer's MMAs; false (uniformly) if a bounded wait ran out here or
// `mine` is false in some thread.
__device__ __forceinline__ bool wait_layer(uint64_t* bar, uint32_t& phase, bool mine) {
  const bool ok = mbar_wait_bounded(bar, phase, kNetWaitNs) && mine;
  phase ^= 1u;
  tc_fence_after();
  return !__syncthreads_or(!ok);
}

__device__ __forceinline__ void bulk_copy_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

// The 16 input channels (12 features, 4 zeros) of patch cell `cell` -> XA chunks 0, 1 (bf16).
__device__ __forceinline__ void put_features(unsigned char* sm, int cell, const float (&f)[12]) {
  uint32_t w8[8];
#pragma unroll
  for (int j = 0; j < 6; ++j) w8[j] = bf16x2(f[2 * j], f[2 * j + 1]);
  w8[6] = w8[7] = 0u;
  *reinterpret_cast<uint4*>(sm + kSmXA + (kPadCells + cell) * 16) = make_uint4(w8[0], w8[1], w8[2], w8[3]);
  *reinterpret_cast<uint4*>(sm + kSmXA + kChunkBytes + (kPadCells + cell) * 16) =
      make_uint4(w8[4], w8[5], w8[6], w8[7]);
}

// Patch input from feature planes [batch][12][H][W] (scaled already).
__device__ __forceinline__ void load_features(unsigned char* sm, const float* __restrict__ ib, long plane, int H,
                                              int W, int ty0, int tx0) {
  for (int cell = threadIdx.x; cell < kMT * 128; cell += kNetThreads) {
    float f[12];
    if (cell < kPatch) {
      const int gy = wrap_mod(ty0 - 3 + cell / kPS, H), gx = wrap_mod(tx0 - 3 + cell % kPS, W);
      const float* p = ib + (size_t)gy * W + gx;
#pragma unroll
      for (int k = 0; k < kC0; ++k) f[k] = p[k * plane];
    } else {
#pragma unroll
      for (int k = 0; k < kC0; ++k) f[k] = 0.f;
    }
    put_features(sm, cell, f);
  }
}

// Patch input from the populations of a square grid: pull the 27 populations of each cell of
// the 24 x 24 moment grid (origin ty0 - 4, tx0 - 4), form u = J / rho and B in binary32 (layer-1
// output buffer as scratch), then the features of the 22 x 22 patch: u_x, u_y, B_x, B_y and
// their central differences (d_x, d_y of each in turn), each times 1 / in_scale.
template <typename S>
__device__ __forceinline__ void load_from_pops(unsigned char* sm, const S* __restrict__ pops, const StepGeom& g,
                                               int ty0, int tx0, const float* __restrict__ inv_s) {
  float* mom = reinterpret_cast<float*>(sm + kSmX1);
  constexpr int MM = kMS * kMS;
#pragma unroll 2
  for (int cell = threadIdx.x; cell < MM; cell += kNetThreads) {
    const int y = wrap_mod(ty0 - 4 + cell / kMS, g.ny), x = wrap_mod(tx0 - 4 + cell % kMS, g.nx);
    float v[27];
#pragma unroll
    for (int q = 0; q < 27; ++q) {
      const int i = q % 9;
      const int sx = wrapi(x - vel_x(i), g.nx), sy = wrapi(y - vel_y(i), g.ny);
      v[q] = load_as<float>(pops[(size_t)plane_of(q) * g.plane + (size_t)sy * g.pitch + kXOff + sx]);
    }
    const float rho1 = (((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]))) + v[8];
    const float jx = (v[1] - v[3]) + (v[5] - v[6]) + (v[8] - v[7]);
    const float jy = (v[2] - v[4]) + (v[5] - v[8]) + (v[6] - v[7]);
    float bx = 0.f, by = 0.f;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      bx += v[9 + i];
      by += v[18 + i];
    }
    const float r = 1.f + rho1;
    mom[cell] = jx / r;
    mom[MM + cell] = jy / r;
    mom[2 * MM + cell] = bx;
    mom[3 * MM + cell] = by;
  }
  __syncthreads();
  for (int cell = threadIdx.x; cell < kMT * 128; cell += kNetThreads) {
    float f[12];
    if (cell < kPatch) {
      const int o = (cell / kPS + 1) * kMS + cell % kPS + 1;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float* a = mom + k * MM;
        f[k] = a[o] * inv_s[k];
        f[4 + 2 * k] = 0.5f * (a[o + 1] - a[o - 1]) * inv_s[4 + 2 * k];
        f[5 + 2 * k] = 0.5f * (a[o + kMS] - a[o - kMS]) * inv_s[5 + 2 * k];
      }
    } else {
#pragma unroll
      for (int k = 0; k < kC0; ++k) f[k] = 0.f;
    }
    put_features(sm, cell, f);
  }
}

// Persistent over tiles (batch x tiles_y x tiles_x).  SRC 0: src = features [batch][12][H][W]
// fp32; SRC 1 / 2: src = binary32 / binary64 populations of the square grid g (batch 1, H = ny,
// W = nx), features formed here with in_scale.  out: [batch][4][H][W] fp32 = (network output)
// x oscale[co] (oscale NULL: 1).
template <int SRC>
__global__ void __launch_bounds__(kNetThreads, 2)
    net_tc_kernel(const void* __restrict__ src, StepGeom g, const float* __restrict__ in_scale,
                  const unsigned char* __restrict__ packed, const float* __restrict__ oscale, int batch, int H,
                  int W, float* __restrict__ out, unsigned* __restrict__ err, int skip_mma) {
  extern __shared__ __align__(128) unsigned char net_smem_raw[];
  unsigned char* sm = net_smem_raw + ((128u - (smem_u32(net_smem_raw) & 127u)) & 127u);
  const uint32_t sbase = smem_u32(sm);
  float* bias = reinterpret_cast<float*>(sm + kSmBias);
  float* inv_s = bias + kBiasFloats + 4;
  uint64_t* bar = reinterpret_cast<uint64_t*>(sm + kSmBar);
  uint64_t* wbar = bar + 1;
  uint32_t* slot = reinterpret_cast<uint32_t*>(sm + kSmSlot);
  const int tid = threadIdx.x, warp = tid >> 5;

  if (tid == 0) {
    mbar_init(bar, 1);
    mbar_init(wbar, 1);
    fence_barrier_init();
  }
  // zero pad cells of the 8 activation chunks (shifted reads reach kPS + 1 cells beyond 0 .. 511)
  for (int i = tid; i < 8 * 2 * kPadCells; i += kNetThreads) {
    const int ch = i / (2 * kPadCells), j = i % (2 * kPadCells);
    const int cell = j < kPadCells ? j : kMT * 128 + j;
    *reinterpret_cast<uint4*>(sm + kSmXA + ch * kChunkBytes + cell * 16) = make_uint4(0, 0, 0, 0);
  }
  // global reads start here: with a programmatic launch the previous step may still be draining
  grid_dependency_wait();
  if (tid == 0) {
    mbar_arrive_expect_tx(wbar, kWBytes);
    bulk_copy_g2s(sm + kSmW, packed, kWBytes, wbar);
  }
  for (int i = tid; i < kBiasFloats + 4 + 12; i += kNetThreads) {
    float v;
    if (i < kBiasFloats) v = reinterpret_cast<const float*>(packed + kWBytes)[i];
    else if (i < kBiasFloats + 4) v = oscale ? oscale[i - kBiasFloats] : 1.f;
    else v = SRC ? 1.f / in_scale[i - kBiasFloats - 4] : 1.f;
    bias[i] = v;
  }
  if (warp == 0) {
    tmem_alloc(slot, kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *slot;

  const long plane = (long)H * W;
  const int tiles_x = (W + kTT - 1) / kTT, tiles_y = (H + kTT - 1) / kTT;
  const long ntiles = (long)batch * tiles_x * tiles_y;
  uint32_t phase = 0;
  bool ok = true, weights_ready = false;
  for (long tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
    const int b = (int)(tile / ((long)tiles_x * tiles_y));
    const int rem = (int)(tile % ((long)tiles_x * tiles_y));
    const int ty0 = (rem / tiles_x) * kTT, tx0 = (rem % tiles_x) * kTT;
    if (SRC == 0)
      load_features(sm, static_cast<const float*>(src) + (size_t)b * kC0 * plane, plane, H, W, ty0, tx0);
    else if (SRC == 1)
      load_from_pops<float>(sm, static_cast<const float*>(src), g, ty0, tx0, inv_s);
    else
      load_from_pops<double>(sm, static_cast<const double*>(src), g, ty0, tx0, inv_s);
    fence_proxy_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // layer 1: 12 (padded to 16) -> 32
    bool mine = true;
    if (tid == 0) {
      if (!weights_ready) mine = weights_ready = mbar_wait_bounded(wbar, 0, kNetWaitNs);
      // test hook: with skip_mma the first tile's layer-1 MMAs and their commit are left out,
      // so the completion wait below runs out (nothing is in flight when TMEM is freed)
      if (mine && !(skip_mma && tile == blockIdx.x)) issue_layer<32, 1, 0, kMT>(sbase, kSmXA, kSmW, tmem, bar);
      else if (!mine) tc_commit(bar);
    }
    if (!(ok = wait_layer(bar, phase, mine))) break;
    hidden_epilogue(tmem, bias, sm + kSmX1);
    fence_proxy_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // layer 2: 32 -> 32
    if (tid == 0) issue_layer<32, 2, 0, kMT>(sbase, kSmX1, kSmW + kW1Bytes, tmem, bar);
    if (!(ok = wait_layer(bar, phase, true))) break;
    hidden_epilogue(tmem, bias + 32, sm + kSmXA);
    fence_proxy_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // layer 3: 32 -> 4, one N = 48 MMA per M tile and K chunk, taps summed below
    if (tid == 0) issue_layer3(sbase, kSmXA, kSmW + kW1Bytes + kW2Bytes, tmem, bar);
    if (!(ok = wait_layer(bar, phase, true))) break;
    // the MMAs have read the activations: their buffers (XA, X1) now hold the partial products
    float* P = reinterpret_cast<float*>(sm + kSmXA);
    layer3_partials(tmem, P);
    __syncthreads();
    {  // one kept cell per thread: patch row / col 3 + tid / 16, 3 + tid % 16
      static_assert(kNetThreads == kTT * kTT, "one output cell per thread");
      const int pr = 3 + tid / kTT, pc = 3 + tid % kTT;
      const int gy = ty0 + pr - 3, gx = tx0 + pc - 3;
      if (gy < H && gx < W) {
        const int c = pr * kPS + pc - kP3Lo;
        float* ob = out + (size_t)b * kC3 * plane + (size_t)gy * W + gx;
#pragma unroll
        for (int co = 0; co < kC3; ++co) {
          float acc = 0.f;
#pragma unroll
          for (int tap = 0; tap < 9; ++tap) {
            const int shift = (tap / 3 - 1) * kPS + (tap % 3 - 1);
            acc += P[(kC3 * tap + co) * kP3Rows + c + shift];
          }
          ob[co * plane] = (acc + bias[64 + co]) * bias[kBiasFloats + co];
        }
      }
    }
    // TMEM reads and shared-memory operands of this tile are finished before the next tile
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
  }
  if (tid == 0) {
    if (!ok) {
      atomicOr(err, 1u);
      mbar_wait_bounded(bar, phase ^ 1u, kNetWaitNs);  // let outstanding MMAs drain
    }
    if (!weights_ready) mbar_wait_bounded(wbar, 0, kNetWaitNs);  // the weight copy has landed
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, kTmemCols);
}

int net_grid(int batch, int H, int W, int num_sms) {
  const long tiles = (long)batch * ((H + kTT - 1) / kTT) * ((W + kTT - 1) / kTT);
  const long cap = 2L * num_sms;
  return (int)(tiles < cap ? (tiles < 1 ? 1 : tiles) : cap);
}

template <int SRC>
cudaError_t set_net_attributes() {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  // per device, once; handles may be driven from several host threads (setting the attribute
  // twice is harmless, a plain flag read while another thread writes it is not)
  static std::atomic<bool> attr_set[64] = {};
  if (dev < 64 && attr_set[dev].load(std::memory_order_acquire)) return cudaSuccess;
  e = cudaFuncSetAttribute(net_tc_kernel<SRC>, cudaFuncAttributeMaxDynamicSharedMemorySize, kNetSmemBytes);
  if (e == cudaSuccess && dev < 64) attr_set[dev].store(true, std::memory_order_release);
  return e;
}

template <int SRC>
cudaError_t launch_net_impl(const void* src, const StepGeom& g, const float* in_scale, const unsigned char* packed,
                            const float* oscale, int batch, int H, int W, float* out, unsigned* err,
                            int skip_mma, cudaStream_t s) {
  cudaError_t e = set_net_attributes<SRC>();
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return launch_programmatic(net_tc_kernel<SRC>, dim3(net_grid(batch, H, W, sms)), kNetThreads, (size_t)kNetSmemBytes,
                             s, src, g, in_scale, packed, oscale, batch, H, W, out, err, skip_mma);
}

cudaError_t launch_net(const float* in, const unsigned char* packed, const float* oscale, int batch, int H,
                       int W, float* out, unsigned* err, int skip_mma, cudaStream_t s) {
  return launch_net_impl<0>(in, StepGeom{}, nullptr, packed, oscale, batch, H, W, out, err, skip_mma, s);
}

// ---- features and training targets ----------------------------------------------------------
// Coarse moments of a fine state by r x r box filter, including the filtered nonlinear products:
// out planes [0..4] = rho, Jx, Jy, Bx, By; [5] JxJy/rho - BxBy; [6] (Jx^2-Jy^2)/rho - (Bx^2-By^2);
// [7] (Jx^2+Jy^2)/rho; [8] (Jx By - Jy Bx)/rho.
//
// Bound by GB300's binary64 rate, not by the 40 bytes per fine cell: with J = rho u the quotients
// are products (J_x J_y / rho = J_x u_y, ...), 15 binary64 instructions per fine cell instead of
// about 57 with four divisions.  A thread adds up one fine column of a coarse row, so the loads
// are coalesced and a coarse cell occupies r threads; the r columns are then added in order, by
// one thread per sum and cell (one per cell, half a warp with nine sums each, cost a tenth of the
// binary64 issue).  2048^2, r = 8, cold caches: 481 us with quotients, 141 with one adding thread
// per cell, 129 with sums that began at zero, now 126.
constexpr int kFilterThreads = 128;
__global__ void __launch_bounds__(kFilterThreads)
    filter_products_kernel(const double* __restrict__ fine, int n, int r, double inv, double* __restrict__ coarse) {
  __shared__ double sh[9][kFilterThreads];
  const int m = n / r;
  const size_t mm = (size_t)m * m, nn = (size_t)n * n;
  // whole coarse cells per block; filters wider than the block take several passes of columns
  const int cells = r <= kFilterThreads ? kFilterThreads / r : 1;
  for (int j = blockIdx.y; j < m; j += gridDim.y) {
    const int i0 = blockIdx.x * cells;
    const int ncell = min(cells, m - i0), cols = ncell * r;
    double tot[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
    for (int c0 = 0; c0 < cols; c0 += kFilterThreads) {
      const int x = c0 + (int)threadIdx.x, w = min(kFilterThreads, cols - c0);
      double s[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
      if (x < cols) {
        const double* p = fine + (size_t)j * r * n + (size_t)i0 * r + x;
        double a, b, c, d;
        {  // the first row starts the sums: additions to zero are binary64 instructions too
          const double rho = p[0], ux = p[nn], uy = p[2 * nn], bx = p[3 * nn], by = p[4 * nn];
          const double jx = rho * ux, jy = rho * uy;
          s[0] = rho;
          s[1] = jx;
          s[2] = jy;
          s[3] = bx;
          s[4] = by;
          s[5] = fma(jx, uy, -bx * by);
          a = jx * ux;
          b = jy * uy;
          c = bx * bx;
          d = by * by;
          s[8] = fma(ux, by, -uy * bx);
        }
        for (int yy = 1; yy < r; ++yy) {
          p += n;
          const double rho = p[0], ux = p[nn], uy = p[2 * nn], bx = p[3 * nn], by = p[4 * nn];
          const double jx = rho * ux, jy = rho * uy;
          s[0] += rho;
          s[1] += jx;
          s[2] += jy;
          s[3] += bx;
          s[4] += by;
          s[5] = fma(jx, uy, fma(-bx, by, s[5]));
          a = fma(jx, ux, a);
          b = fma(jy, uy, b);
          c = fma(bx, bx, c);
          d = fma(by, by, d);
          s[8] = fma(ux, by, fma(-uy, bx, s[8]));
        }
        s[6] = (a - b) - (c - d);
        s[7] = a + b;
      }
#pragma unroll
      for (int k = 0; k < 9; ++k) sh[k][threadIdx.x] = s[k];
      __syncthreads();
      // the 9 sums of the block's coarse cells (one when r exceeds the block), one (sum, cell) pair per
      // thread and turn: its columns of this pass, in order
      const int num = r <= kFilterThreads ? r : w;
#pragma unroll
      for (int k = 0; k < 9; ++k) {
        const int e = k * kFilterThreads + (int)threadIdx.x;
        if (e < 9 * ncell) {
          const double* col = &sh[e / ncell][e % ncell * num];
          double t = c0 == 0 ? col[0] : tot[k] + col[0];
          for (int q = 1; q < num; ++q) t += col[q];
          tot[k] = t;
        }
      }
      __syncthreads();
    }
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      const int e = k * kFilterThreads + (int)threadIdx.x;
      if (e < 9 * ncell) coarse[e / ncell * mm + (size_t)j * m + i0 + e % ncell] = tot[k] * inv;
    }
  }
}

// Features (12 channels: u, B and their central differences, each over its scale) of a coarse
// state given as rho, Jx, Jy, Bx, By planes (J = rho u; u itself when `velocity`); optionally the
// analytic closure a0..a3 (kd = delta^2/12) into `analytic` (4 planes), and, when `products` is
// given (planes 5..8 of filter_products_kernel), the training target (c - a)/out_scale into
// `target`.
//
// Bound by binary64 divisions and their latency: a block forms u and J of its 32 x 4 cells and a
// ring of one cell once in shared memory (one reciprocal per cell instead of ten divisions), and
// scales by reciprocals formed once per block.  256^2, cold caches: 56 -> 24 with two divisions per
// cell -> 21 us.
__device__ __noinline__ double divided(double a, double b) { return a / b; }  // a call: branched around
constexpr int kFeatW = 32, kFeatH = 4, kFeatThreads = kFeatW * kFeatH;
__global__ void __launch_bounds__(kFeatThreads)
    features_kernel(const double* __restrict__ st, int m, int velocity, const float* __restrict__ in_scale,
                    const float* __restrict__ out_scale, double kd, float* __restrict__ x,
                    float* __restrict__ analytic, const double* __restrict__ products, float* __restrict__ target) {
  constexpr int PW = kFeatW + 2, PH = kFeatH + 2;
  __shared__ double u[4][PH][PW];  // u_x, u_y, B_x, B_y
  __shared__ double J[2][PH][PW];
  __shared__ double Ri[PH][PW];    // 1 / rho (not when `velocity`)
  __shared__ double inv[16];       // 1 / in_scale[12], 1 / out_scale[4]
  const size_t mm = (size_t)m * m;
  const int tid = threadIdx.x, lx = tid % kFeatW, ly = tid / kFeatW;
  if (tid < 16) inv[tid] = 1.0 / (double)(tid < 12 ? in_scale[tid] : out_scale[tid - 12]);
  const int x0 = blockIdx.x * kFeatW;
  const int bands = (m + kFeatH - 1) / kFeatH;
  for (int band = blockIdx.y; band < bands; band += gridDim.y) {
    const int y0 = band * kFeatH;
    for (int e = tid; e < PW * PH; e += kFeatThreads) {
      const int px = e % PW, py = e / PW;
      const size_t o = (size_t)wrap_mod(y0 - 1 + py, m) * m + wrap_mod(x0 - 1 + px, m);
      const double rho = st[o], v0 = st[mm + o], v1 = st[2 * mm + o];
      u[2][py][px] = st[3 * mm + o];
      u[3][py][px] = st[4 * mm + o];
      if (velocity) {
        J[0][py][px] = rho * v0;
        J[1][py][px] = rho * v1;
        u[0][py][px] = v0;
        u[1][py][px] = v1;
      } else {
        const double y = __drcp_rn(rho);
        const bool fast = quotient_in_range(v0, rho) && quotient_in_range(v1, rho);
        J[0][py][px] = v0;
        J[1][py][px] = v1;
        u[0][py][px] = fast ? quotient(v0, rho, y) : divided(v0, rho);
        u[1][py][px] = fast ? quotient(v1, rho, y) : divided(v1, rho);
        Ri[py][px] = y;
      }
    }
    __syncthreads();
    const int i = x0 + lx, j = y0 + ly;
    if (i < m && j < m) {
      const size_t c = (size_t)j * m + i;
      auto ddx = [&](const double (*a)[PW]) { return 0.5 * (a[ly + 1][lx + 2] - a[ly + 1][lx]); };
      auto ddy = [&](const double (*a)[PW]) { return 0.5 * (a[ly + 2][lx + 1] - a[ly][lx + 1]); };
      double gb[4];
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        const double dx = ddx(u[f]), dy = ddy(u[f]);
        x[f * mm + c] = (float)(u[f][ly + 1][lx + 1] * inv[f]);
        x[(4 + 2 * f) * mm + c] = (float)(dx * inv[4 + 2 * f]);
        x[(5 + 2 * f) * mm + c] = (float)(dy * inv[5 + 2 * f]);
        if (f >= 2) {
          gb[2 * (f - 2)] = dx;
          gb[2 * (f - 2) + 1] = dy;
        }
      }
      if (analytic || target) {
        const double gj[4] = {ddx(J[0]), ddy(J[0]), ddx(J[1]), ddy(J[1])};
        const double ir = velocity ? divided(1.0, st[c]) : Ri[ly + 1][lx + 1];
        const double Gxx = gj[0] * gj[0] + gj[1] * gj[1], Gyy = gj[2] * gj[2] + gj[3] * gj[3];
        const double Gxy = gj[0] * gj[2] + gj[1] * gj[3];
        const double Hxx = gb[0] * gb[0] + gb[1] * gb[1], Hyy = gb[2] * gb[2] + gb[3] * gb[3];
        const double Hxy = gb[0] * gb[2] + gb[1] * gb[3];
        const double Kxy = gj[0] * gb[2] + gj[1] * gb[3], Kyx = gj[2] * gb[0] + gj[3] * gb[1];
        const double a[4] = {kd * (Gxy * ir - Hxy), kd * ((Gxx - Gyy) * ir - Hxx + Hyy),
                             kd * (Gxx + Gyy) * ir, kd * (Kxy - Kyx) * ir};
        if (analytic)
          for (int f = 0; f < 4; ++f) analytic[f * mm + c] = (float)a[f];
        if (target && products) {
          const double jx = J[0][ly + 1][lx + 1], jy = J[1][ly + 1][lx + 1];
          const double ux = u[0][ly + 1][lx + 1], uy = u[1][ly + 1][lx + 1];
          const double b = u[2][ly + 1][lx + 1], d = u[3][ly + 1][lx + 1];
          const double cq[4] = {products[c] - (jx * uy - b * d),
                                products[mm + c] - ((jx * ux - jy * uy) - (b * b - d * d)),
                                products[2 * mm + c] - (jx * ux + jy * uy), products[3 * mm + c] - (ux * d - uy * b)};
          for (int f = 0; f < 4; ++f) target[f * mm + c] = (float)((cq[f] - a[f]) * inv[12 + f]);
        }
      }
    }
    __syncthreads();  // the tile is rewritten for the next band
  }
}

dim3 filter_grid(int m, int r) {
  const int cells = r <= kFilterThreads ? kFilterThreads / r : 1;
  return dim3((m + cells - 1) / cells, m < 65535 ? m : 65535);
}
dim3 features_grid(int m) {
  const int bands = (m + kFeatH - 1) / kFeatH;
  return dim3((m + kFeatW - 1) / kFeatW, bands < 65535 ? bands : 65535);
}

int grid_for(long n) {
  long b = (n + kThreads - 1) / kThreads;
  if (b > 152L * 16) b = 152L * 16;
  return b < 1 ? 1 : (int)b;
}

}  // namespace

int closure_num_params() { return kNumParams; }

cudaError_t prepare_closure_kernels() {
  cudaError_t e = set_net_attributes<1>();
  if (e == cudaSuccess) e = set_net_attributes<2>();
  return e;
}

// Correction planes [4][m][m] (physical units) for the current populations of a square
// binary64 / binary32 grid: one launch of the fused network kernel (pull, u and B, features,
// three tensor-core layers, output scale).
cudaError_t closure_correction(const lbmhd_closure_t* c, int precision, const void* pops, const StepGeom& g,
                               float* corr, unsigned* err, cudaStream_t s) {
  const float* sc = closure_device_scales(c);
  const unsigned char* pk = closure_device_packed(c);
  if (precision == 0) return launch_net_impl<2>(pops, g, sc, pk, sc + 12, 1, g.ny, g.nx, corr, err, 0, s);
  return launch_net_impl<1>(pops, g, sc, pk, sc + 12, 1, g.ny, g.nx, corr, err, 0, s);
}

}  // namespace lbmhd_gpu

// ---- the closure object and its C ABI -------------------------------------------------------
using namespace lbmhd_gpu;

struct lbmhd_closure {
  float* params = nullptr;  // device, binary32 master copy
  float* grad = nullptr;
  float* adam_m = nullptr;
  float* adam_v = nullptr;
  float* scales = nullptr;  // device: in_scale[12], out_scale[4]
  unsigned char* packed = nullptr;  // device: bf16 weights + fp32 biases for the tensor-core kernel
  unsigned* tc_err = nullptr;       // device: tensor-core wait timeout flag
  int test_skip_mma = 0;            // failure-detection test hook (lbmhd_closure_test_skip_mma)
  float host_scales[16];
  int adam_t = 0;
  // training scratch (grown on demand)
  size_t cap_cells = 0;
  float *a1 = nullptr, *a2 = nullptr, *d3 = nullptr, *d2 = nullptr, *d1 = nullptr;
  float* wpart = nullptr;   // [kMaxConvBlocks][kNumParams] partial weight gradients
  double* lpart = nullptr;  // kMaxConvBlocks partial losses, then their sum
  cudaStream_t stream = nullptr;
  std::string err;
};

namespace {
thread_local std::string g_cl_error;

int cfail(lbmhd_closure_t* c, int code, const char* msg) {
  if (c)
    c->err = msg;
  else
    g_cl_error = msg;
  return code;
}

#define CL_CUDA(c, call)                                                                         \
  do {                                                                                           \
    cudaError_t e_ = (call);                                                                     \
    if (e_ != cudaSuccess) {                                                                     \
      char b_[256];                                                                              \
      snprintf(b_, sizeof b_, "%s: %s", #call, cudaGetErrorString(e_));                         \
      return cfail(c, e_ == cudaErrorMemoryAllocation ? LBMHD_ERR_OOM : LBMHD_ERR_CUDA, b_);   \
    }                                                                                            \
  } while (0)

int ensure_scratch(lbmhd_closure_t* c, size_t cells) {
  if (cells <= c->cap_cells) return LBMHD_OK;
  c->cap_cells = 0;  // nothing usable until every buffer below has grown
  float** bufs[5] = {&c->a1, &c->a2, &c->d3, &c->d2, &c->d1};
  const int ch[5] = {kC1, kC2, kC3, kC2, kC1};
  for (int i = 0; i < 5; ++i) {
    if (*bufs[i]) cudaFree(*bufs[i]);
    *bufs[i] = nullptr;
    CL_CUDA(c, device_malloc(bufs[i], cells * ch[i] * sizeof(float)));
  }
  if (!c->wpart) CL_CUDA(c, device_malloc(&c->wpart, (size_t)kMaxConvBlocks * kNumParams * sizeof(float)));
  if (!c->lpart) CL_CUDA(c, device_malloc(&c->lpart, (kMaxConvBlocks + 1) * sizeof(double)));
  c->cap_cells = cells;
  return LBMHD_OK;
}

// Blocks for tiles of kTileW x rows cells.
int conv_grid(int batch, int H, int W, int rows) {
  const long tiles = (long)batch * ((H + rows - 1) / rows) * ((W + kTileW - 1) / kTileW);
  return (int)(tiles < kMaxConvBlocks ? tiles : kMaxConvBlocks);
}

template <int CIN, int COUT, int EPI, bool BWD = false>
cudaError_t conv(const float* in, const float* params, const float* aux, int batch, int H, int W, float* out,
                 double* loss_part, cudaStream_t s) {
  using Sh = ConvShape<CIN, COUT>;
  if constexpr (!BWD && (EPI == kEpiNone || EPI == kEpiTanh)) {
    // A full tile takes about a third of the time of as many cells with a thread each, an empty one
    // as long as a full one; up to one wave of tiles costs the same 80 us for the network.  Binary32 forward
    // pass by cells / by tiles: 65536 x 8 892 / 1234 us, 65536 x 16 1668 / 1227, 4 x 65536 505 / 687, 1024
    // grids of 8 x 8 147 / 362, 4096 of 4 x 4 151 / 1388; 64 of 4 x 4 97 / 82; 3 x 3 83 / 85, one cell 75 / 107.
    const long cells = (long)batch * H * W;
    const long tiles = (long)batch * ((H + Sh::kRows - 1) / Sh::kRows) * ((W + kTileW - 1) / kTileW);
    if (cells < 9 || (tiles > kMaxConvBlocks && 3 * cells < (long)Sh::kRows * kTileW * tiles)) {
      conv_cell_kernel<CIN, COUT, EPI == kEpiTanh><<<grid_for(cells), kThreads, 0, s>>>(in, params, batch, H, W, out);
      return cudaGetLastError();
    }
  }
  auto k = conv_tile_kernel<CIN, COUT, EPI, BWD>;
  if (Sh::kSmem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Sh::kSmem);
    if (e != cudaSuccess) return e;
  }
  k<<<conv_grid(batch, H, W, Sh::kRows), kConvThreads, Sh::kSmem, s>>>(in, params, aux, batch, H, W, out, loss_part);
  return cudaGetLastError();
}

template <int NWIN, int NW, bool LANE_DY>
cudaError_t wgrad(const float* lane_op, const float* win_op, int batch, int H, int W, float* part, int base,
                  cudaStream_t s) {
  auto k = conv_wgrad_kernel<NWIN, NW, LANE_DY>;
  constexpr size_t sm = wgrad_smem<NWIN>();
  if (sm > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
  }
  k<<<conv_grid(batch, H, W, kWgRows), kWgThreads, sm, s>>>(lane_op, win_op, batch, H, W, part, base);
  return cudaGetLastError();
}

// forward (binary32) + loss + back-propagation into c->grad; *loss = mean squared error / 2
int forward_backward(lbmhd_closure_t* c, const float* x, const float* t, int batch, int h, int w,
                     double* loss) {
  const size_t cells = (size_t)batch * h * w;
  int rc = ensure_scratch(c, cells);
  if (rc) return rc;
  cudaStream_t s = c->stream;
  const float* p1 = c->params;
  const float* p2 = c->params + kP1;
  const float* p3 = c->params + kP1 + kP2;
  CL_CUDA(c, (conv<kC0, kC1, kEpiTanh>(x, p1, nullptr, batch, h, w, c->a1, nullptr, s)));
  CL_CUDA(c, (conv<kC1, kC2, kEpiTanh>(c->a1, p2, nullptr, batch, h, w, c->a2, nullptr, s)));
  CL_CUDA(c, (conv<kC2, kC3, kEpiLoss>(c->a2, p3, t, batch, h, w, c->d3, c->lpart, s)));
  // data gradients of layers 3 and 2, weight gradients of all three
  CL_CUDA(c, (wgrad<kC3, 4, false>(c->a2, c->d3, batch, h, w, c->wpart, kP1 + kP2, s)));
  CL_CUDA(c, (conv<kC3, kC2, kEpiTanhGrad, true>(c->d3, p3, c->a2, batch, h, w, c->d2, nullptr, s)));
  CL_CUDA(c, (wgrad<kC1, 4, true>(c->d2, c->a1, batch, h, w, c->wpart, kP1, s)));
  CL_CUDA(c, (conv<kC2, kC1, kEpiTanhGrad, true>(c->d2, p2, c->a1, batch, h, w, c->d1, nullptr, s)));
  CL_CUDA(c, (wgrad<kC0, 3, true>(c->d1, x, batch, h, w, c->wpart, 0, s)));
  double* total = c->lpart + kMaxConvBlocks;
  sum_partials_kernel<<<(kNumParams + 31) / 32, dim3(32, 8), 0, s>>>(
      c->wpart, conv_grid(batch, h, w, kWgRows), c->grad, c->lpart,
      conv_grid(batch, h, w, ConvShape<kC2, kC3>::kRows), total);
  CL_CUDA(c, cudaGetLastError());
  double sum = 0.0;
  CL_CUDA(c, cudaMemcpyAsync(&sum, total, sizeof sum, cudaMemcpyDeviceToHost, s));
  CL_CUDA(c, cudaStreamSynchronize(s));
  if (loss) *loss = 0.5 * sum / (double)(cells * kC3);
  return LBMHD_OK;
}

// Refresh the tensor-core copy of the parameters (after any change of c->params).
int repack(lbmhd_closure_t* c) {
  pack_net_kernel<<<(kWBytes / 2 + kBiasFloats + 255) / 256, 256, 0, c->stream>>>(c->params, c->packed);
  CL_CUDA(c, cudaGetLastError());
  return LBMHD_OK;
}

void destroy_closure(lbmhd_closure_t* c) {
  if (!c) return;
  if (c->stream) cudaStreamSynchronize(c->stream);
  float* bufs[] = {c->params, c->grad, c->adam_m, c->adam_v, c->scales, c->a1, c->a2, c->d3, c->d2,
                   c->d1, c->wpart};
  for (float* b : bufs)
    if (b) cudaFree(b);
  if (c->lpart) cudaFree(c->lpart);
  if (c->packed) cudaFree(c->packed);
  if (c->tc_err) cudaFree(c->tc_err);
  if (c->stream) cudaStreamDestroy(c->stream);
  delete c;
}
}  // namespace

extern "C" {

int lbmhd_closure_num_params(void) { return kNumParams; }

int lbmhd_closure_create(lbmhd_closure_t** out, const float* params, const float* in_scale,
                         const float* out_scale) {
  if (!out) return cfail(nullptr, LBMHD_ERR_INVALID, "out is NULL");
  *out = nullptr;
  if (!params || !in_scale || !out_scale) return cfail(nullptr, LBMHD_ERR_INVALID, "NULL argument");
  for (int i = 0; i < 12; ++i)
    if (!(in_scale[i] > 0.f)) return cfail(nullptr, LBMHD_ERR_INVALID, "in_scale must be > 0");
  for (int i = 0; i < 4; ++i)
    if (!(out_scale[i] > 0.f)) return cfail(nullptr, LBMHD_ERR_INVALID, "out_scale must be > 0");
  lbmhd_closure_t* c = new (std::nothrow) lbmhd_closure();
  if (!c) return cfail(nullptr, LBMHD_ERR_OOM, "host allocation failed");
  std::memcpy(c->host_scales, in_scale, 12 * sizeof(float));
  std::memcpy(c->host_scales + 12, out_scale, 4 * sizeof(float));
  cudaError_t e = cudaStreamCreateWithFlags(&c->stream, cudaStreamNonBlocking);
  const size_t pb = kNumParams * sizeof(float);
  if (e == cudaSuccess) e = device_malloc(&c->params, pb);
  if (e == cudaSuccess) e = device_malloc(&c->grad, pb);
  if (e == cudaSuccess) e = device_malloc(&c->adam_m, pb);
  if (e == cudaSuccess) e = device_malloc(&c->adam_v, pb);
  if (e == cudaSuccess) e = device_malloc(&c->scales, 16 * sizeof(float));
  if (e == cudaSuccess) e = device_malloc(&c->packed, kPackedBytes);
  if (e == cudaSuccess) e = device_malloc(&c->tc_err, sizeof(unsigned));
  if (e == cudaSuccess) e = cudaMemset(c->tc_err, 0, sizeof(unsigned));
  if (e == cudaSuccess) e = cudaMemcpy(c->params, params, pb, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemset(c->adam_m, 0, pb);
  if (e == cudaSuccess) e = cudaMemset(c->adam_v, 0, pb);
  if (e == cudaSuccess) e = cudaMemcpy(c->scales, c->host_scales, 16 * sizeof(float), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    pack_net_kernel<<<(kWBytes / 2 + kBiasFloats + 255) / 256, 256, 0, c->stream>>>(c->params, c->packed);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
  if (e != cudaSuccess) {
    int rc = cfail(nullptr, e == cudaErrorMemoryAllocation ? LBMHD_ERR_OOM : LBMHD_ERR_CUDA,
                   cudaGetErrorString(e));
    destroy_closure(c);
    return rc;
  }
  *out = c;
  return LBMHD_OK;
}

int lbmhd_closure_get_params(lbmhd_closure_t* c, float* params) {
  if (!c || !params) return cfail(c, LBMHD_ERR_INVALID, "NULL argument");
  CL_CUDA(c, cudaStreamSynchronize(c->stream));
  CL_CUDA(c, cudaMemcpy(params, c->params, kNumParams * sizeof(float), cudaMemcpyDeviceToHost));
  return LBMHD_OK;
}

int lbmhd_closure_set_params(lbmhd_closure_t* c, const float* params) {
  if (!c || !params) return cfail(c, LBMHD_ERR_INVALID, "NULL argument");
  CL_CUDA(c, cudaStreamSynchronize(c->stream));
  CL_CUDA(c, cudaMemcpy(c->params, params, kNumParams * sizeof(float), cudaMemcpyHostToDevice));
  c->adam_t = 0;
  CL_CUDA(c, cudaMemset(c->adam_m, 0, kNumParams * sizeof(float)));
  CL_CUDA(c, cudaMemset(c->adam_v, 0, kNumParams * sizeof(float)));
  int rc = repack(c);
  if (rc) return rc;
  CL_CUDA(c, cudaStreamSynchronize(c->stream));
  return LBMHD_OK;
}

int lbmhd_closure_gradient(lbmhd_closure_t* c, const float* x, const float* t, int batch, int h,
                           int w, float* grad, double* loss) {
  if (!c || !x || !t) return cfail(c, LBMHD_ERR_INVALID, "NULL argument");
  if (batch < 1 || h < 1 || w < 1) return cfail(c, LBMHD_ERR_INVALID, "empty batch");
  int rc = forward_backward(c, x, t, batch, h, w, loss);
  if (rc) return rc;
  if (grad) CL_CUDA(c, cudaMemcpy(grad, c->grad, kNumParams * sizeof(float), cudaMemcpyDeviceToHost));
  return LBMHD_OK;
}

int lbmhd_closure_train_step(lbmhd_closure_t* c, const float* x, const float* t, int batch, int h,
                             int w, float lr, double* loss) {
  if (!c || !x || !t) return cfail(c, LBMHD_ERR_INVALID, "NULL argument");
  if (batch < 1 || h < 1 || w < 1 || !(lr > 0.f)) return cfail(c, LBMHD_ERR_INVALID, "bad batch or rate");
  int rc = forward_backward(c, x, t, batch, h, w, loss);
  if (rc) return rc;
  c->adam_t += 1;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - powf(b1, (float)c->adam_t), c2 = 1.f - powf(b2, (float)c->adam_t);
  adam_kernel<<<grid_for(kNumParams), kThreads, 0, c->stream>>>(c->params, c->grad, c->adam_m, c->adam_v,
                                                                kNumParams, lr, b1, b2, 1e-8f, c1, c2);
  CL_CUDA(c, cudaGetLastError());
  return repack(c);
}

int lbmhd_closure_forward(lbmhd_closure_t* c, const float* x, int batch, int h, int w, float* out,
                          int tensor_cores) {
  if (!c || !x || !out) return cfail(c, LBMHD_ERR_INVALID, "NULL argument");
  if (batch < 1 || h < 1 || w < 1) return cfail(c, LBMHD_ERR_INVALID, "empty batch");
  cudaStream_t s = c->stream;
  if (tensor_cores) {
    CL_CUDA(c, launch_net(x, c->packed, nullptr, batch, h, w, out, c->tc_err, c->test_skip_mma, s));
  } else {
    int rc = ensure_scratch(c, (size_t)batch * h * w);
    if (rc) return rc;
    const float* p = c->params;
    CL_CUDA(c, (conv<kC0, kC1, kEpiTanh>(x, p, nullptr, batch, h, w, c->a1, nullptr, s)));
    CL_CUDA(c, (conv<kC1, kC2, kEpiTanh>(c->a1, p + kP1, nullptr, batch, h, w, c->a2, nullptr, s)));
    CL_CUDA(c, (conv<kC2, kC3, kEpiNone>(c->a2, p + kP1 + kP2, nullptr, batch, h, w, out, nullptr, s)));
  }
  CL_CUDA(c, cudaGetLastError());
  CL_CUDA(c, cudaStreamSynchronize(s));
  if (tensor_cores) {
    unsigned v = 0;
    CL_CUDA(c, cudaMemcpy(&v, c->tc_err, sizeof v, cudaMemcpyDeviceToHost));
    if (v) {
      CL_CUDA(c, cudaMemset(c->tc_err, 0, sizeof v));
      return cfail(c, LBMHD_ERR_TIMEOUT, "a tensor-core completion wait timed out");
    }
  }
  return LBMHD_OK;
}

int lbmhd_closure_training_pair(lbmhd_closure_t* c, const double* fine, int n, int r, double delta,
                                float* x, float* t, double* work) {
  if (!c || !fine || !x || !t || !work) return cfail(c, LBMHD_ERR_INVALID, "NULL argument");
  if (n < 3 || r < 1 || n % r || n / r < 3 || !(delta >= 0.0))
    return cfail(c, LBMHD_ERR_INVALID, "need r | n, n/r >= 3, delta >= 0");
  const int m = n / r;
  const long mm = (long)m * m;
  cudaStream_t s = c->stream;
  filter_products_kernel<<<filter_grid(m, r), kFilterThreads, 0, s>>>(fine, n, r, 1.0 / ((double)r * r), work);
  features_kernel<<<features_grid(m), kFeatThreads, 0, s>>>(work, m, 0, c->scales, c->scales + 12,
                                                     delta * delta / 12.0, x, nullptr, work + 5 * mm, t);
  CL_CUDA(c, cudaGetLastError());
  CL_CUDA(c, cudaStreamSynchronize(s));
  return LBMHD_OK;
}

int lbmhd_closure_features(lbmhd_closure_t* c, const double* state, int m, double delta, float* x,
                           float* analytic) {
  if (!c || !state || !x) return cfail(c, LBMHD_ERR_INVALID, "NULL argument");
  if (m < 3) return cfail(c, LBMHD_ERR_INVALID, "m must be >= 3");
  features_kernel<<<features_grid(m), kFeatThreads, 0, c->stream>>>(
      state, m, 1, c->scales, c->scales + 12, delta * delta / 12.0, x, analytic, nullptr, nullptr);
  CL_CUDA(c, cudaGetLastError());
  CL_CUDA(c, cudaStreamSynchronize(c->stream));
  return LBMHD_OK;
}

int lbmhd_closure_test_skip_mma(lbmhd_closure_t* c, int enable) {
  if (!c) return cfail(nullptr, LBMHD_ERR_INVALID, "NULL argument");
  CL_CUDA(c, cudaStreamSynchronize(c->stream));
  c->test_skip_mma = enable ? 1 : 0;
  return LBMHD_OK;
}

const char* lbmhd_closure_last_error(const lbmhd_closure_t* c) {
  return c ? c->err.c_str() : g_cl_error.c_str();
}

void lbmhd_closure_free(lbmhd_closure_t* c) { destroy_closure(c); }

}  // extern "C"

namespace lbmhd_gpu {
// Device pointers of a closure's parameters and scales (for handles that attach it).
const float* closure_device_params(const lbmhd_closure_t* c) { return c->params; }
const float* closure_device_scales(const lbmhd_closure_t* c) { return c->scales; }
const unsigned char* closure_device_packed(const lbmhd_closure_t* c) { return c->packed; }
cudaStream_t closure_stream(const lbmhd_closure_t* c) { return c->stream; }
}  // namespace lbmhd_gpu
