// Learned start vector for rKS on a parametric operator family: a 4-level
// U-Net (32 channels, 3x3 convolutions, ReLU, 2x2 average pooling, 2x nearest
// upsampling, additive skips) maps the coefficient fields of an operator
// (log nu, bx / 50, by / 50 on the grid) to a start vector u_1, and is
// trained on the Schur vectors rKS itself computed, with the subspace-capture
// loss L = 1 - ||Q^T u||^2 / ||u||^2 (Q an orthonormal basis of the wanted
// invariant subspace).  The paper takes u_1 at random (Sec. 2.1); the random
// start stays the fallback and the residual of the solve is the judge.
//
// Arithmetic: FP32 master weights (Adam), copies rounded to FP16 (held as FP32)
// for the convolutions, FP32 activations and accumulation, FP64 for the loss sums.  Activations
// are channel-major (c x H x W) per level; every reduction is a fixed-order
// fold of per-CTA partial sums, so a training step gives the same bits on
// every run.
//
// Kernels:
//   k_conv3x3       32 x 8 output pixels per CTA, 4 pixels x 8 (or 4)
//                   outputs per thread, optional ReLU on the output and an optional mask
//                   on it (the ReLU derivative of the backward pass); the
//                   backward-data product is this kernel with the flipped,
//                   transposed weights.  k_conv3x3_one: the one-channel layer.
//   k_wgrad32 / k_wgrad3 / k_wgrad_one
//                   partial sums of dL/dW and dL/db per CTA, folded in a
//                   fixed order by k_fold_params.
//   k_pool, k_pool_back, k_up_add, k_up_back: level changes.
//   k_loss_dots, k_loss_grad: Q^T u and u^T u (FP64 partials), dL/du.
//   k_adam, k_pack_weights: the optimiser and the FP16 weight layouts.
//   k_two_norms, k_combine: the start vector u / ||u|| + eps g / ||g||.

#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "../../include/rks.h"
#include "rks_impl.h"

namespace {

constexpr int kCh = 32;          // channels of every hidden layer
constexpr int kConvs = 15;       // C1 .. C15
constexpr int kTile = 16;        // output tile side
constexpr int kHalo = kTile + 2;
constexpr int kHalo2 = kHalo * kHalo;

int conv_cin(int l) { return l == 0 ? 3 : kCh; }
int conv_cout(int l) { return l == kConvs - 1 ? 1 : kCh; }

// Two FP32 FMAs per lane and instruction (IEEE, round to nearest each): the
// FMA pipe then needs an issue slot only every other cycle, which leaves the
// others to the shared-memory loads.
__device__ __forceinline__ unsigned long long pack2(float lo, float hi) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack2(unsigned long long v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ void cp4_zfill(float* dst, const float* src, bool on) {
  const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(on ? 4 : 0) : "memory");
}

// out[o, y, x] = b[o] + sum_{c, dy, dx} W[o, c, dy, dx] z[c, y + dy - 1, x + dx - 1],
// zero outside the grid, for 32 output channels; W (the FP16 values as FP32)
// in layout [c][dy * 3 + dx][o]; optional ReLU on out; with omask, out is
// zero where omask <= 0 (the ReLU derivative of the layer that out is the
// gradient of).  FP32 FMAs in the order (c, dy, dx) from b.
//
// A CTA takes 32 x 8 pixels and four groups of OUTS outputs (grid.z the
// others), a thread 4 pixels of a row and one group: per channel 18 OUTS
// two-wide FMAs against 24 shared-memory loads (a group's weights are one
// broadcast address per warp), where one pixel x 32 outputs per thread needed
// 9 loads per 32 FMAs and ran at 27% of the FMA rate.  Channels come in
// stages of 8 with the next stage in flight (cp.async, zero fill at the
// border).  OUTS = 8 for large grids, 4 where its CTAs would not fill the
// SMs (half the chain per warp, twice the CTAs).
// Measured, 512 x 512, 32 -> 32 (2.4 GMAC): 89 us, 74% of the FMA rate (the
// pixel form 190 us); 8 pixels x 4 outputs per thread with doubled weights
// 125 us.  256 x 256: 31 us with OUTS = 4 (37 us with 8).
// On the tensor cores (bf16 splits of z) the sums would be truncated at
// every accumulation, always towards zero: layer after layer that shrinks
// the result by more than the rounding errors of these FMAs.
constexpr int kCvW = 32, kCvH = 8, kCvPitch = 36, kCvStage = 8;
constexpr int kCvPlane = (kCvH + 2) * kCvPitch;

// One channel's tile with its halo, by one warp: a lane a column, then the
// last two columns.
__device__ __forceinline__ void conv_stage_plane(const float* __restrict__ zc, int H, int W, int x0, int y0,
                                                 int lane, float* dst) {
  const int gx = x0 - 1 + lane;
  const bool okx = gx >= 0 && gx < W;
#pragma unroll
  for (int r = 0; r < kCvH + 2; ++r) {
    const int gy = y0 - 1 + r;
    const bool on = okx && gy >= 0 && gy < H;
    cp4_zfill(dst + r * kCvPitch + lane, on ? zc + (size_t)gy * W + gx : zc, on);
  }
  if (lane < 2 * (kCvH + 2)) {
    const int r = lane >> 1, hx = x0 + 31 + (lane & 1), gy = y0 - 1 + r;
    const bool on = hx < W && gy >= 0 && gy < H;
    cp4_zfill(dst + r * kCvPitch + 32 + (lane & 1), on ? zc + (size_t)gy * W + hx : zc, on);
  }
}

template <int OUTS>
__global__ void __launch_bounds__(256) k_conv3x3(const float* __restrict__ z, int cin, int H, int W,
                                                 const float* __restrict__ w, const float* __restrict__ bias,
                                                 int relu, const float* __restrict__ omask,
                                                 float* __restrict__ out) {
  extern __shared__ __align__(16) float sm[];
  constexpr int OP = OUTS / 2;                  // output pairs
  float* zs = sm;                               // two stages of kCvStage planes
  float* ws = sm + 2 * kCvStage * kCvPlane;     // (cin * 9) x 4 groups x OUTS
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int og = tid >> 6, xg = tid & 7, ty = (tid >> 3) & 7;
  const int tiles_x = (W + kCvW - 1) / kCvW;    // tiles in grid.x: a grid of 65 536 tile rows is legal
  const int x0 = blockIdx.x % tiles_x * kCvW, y0 = blockIdx.x / tiles_x * kCvH;
  const int o0 = (blockIdx.z * 4 + og) * OUTS;
  const size_t hw = (size_t)H * W;
  auto stage = [&](int c0, float* dst) {        // a warp a channel
    if (c0 + warp < cin) conv_stage_plane(z + (c0 + warp) * hw, H, W, x0, y0, lane, dst + warp * kCvPlane);
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  for (int i = tid; i < cin * 9 * OUTS; i += 256) {       // 16 bytes each
    const int r = i / OUTS, q = i % OUTS;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                     static_cast<uint32_t>(__cvta_generic_to_shared(ws + 4 * i))),
                 "l"(w + r * 32 + blockIdx.z * 4 * OUTS + 4 * q)
                 : "memory");
  }
  stage(0, zs);
  unsigned long long acc[4][OP];                // pixel, output pair
#pragma unroll
  for (int q = 0; q < OP; ++q) {
    const unsigned long long b = bias ? pack2(bias[o0 + 2 * q], bias[o0 + 2 * q + 1]) : 0ull;
#pragma unroll
    for (int p = 0; p < 4; ++p) acc[p][q] = b;
  }
  int buf = 0;
  for (int c0 = 0; c0 < cin; c0 += kCvStage, buf ^= 1) {
    const bool more = c0 + kCvStage < cin;
    if (more) stage(c0 + kCvStage, zs + (buf ^ 1) * kCvStage * kCvPlane);
    if (more) asm volatile("cp.async.wait_group 1;" ::: "memory");
    else asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    const int nc = min(kCvStage, cin - c0);
    const float* zc = zs + buf * kCvStage * kCvPlane + ty * kCvPitch + xg * 4;
    const float* wc = ws + c0 * 36 * OUTS + og * OUTS;
    for (int c = 0; c < nc; ++c, zc += kCvPlane, wc += 36 * OUTS) {
#pragma unroll
      for (int dy = 0; dy < 3; ++dy) {
        const float4 a = *reinterpret_cast<const float4*>(zc + dy * kCvPitch);
        const float2 b = *reinterpret_cast<const float2*>(zc + dy * kCvPitch + 4);
        const unsigned long long v[6] = {pack2(a.x, a.x), pack2(a.y, a.y), pack2(a.z, a.z),
                                         pack2(a.w, a.w), pack2(b.x, b.x), pack2(b.y, b.y)};
#pragma unroll
        for (int dx = 0; dx < 3; ++dx) {
#pragma unroll
          for (int h = 0; h < OP / 2; ++h) {
            const ulonglong2 wk = *reinterpret_cast<const ulonglong2*>(wc + (dy * 3 + dx) * 4 * OUTS + 4 * h);
#pragma unroll
            for (int p = 0; p < 4; ++p) {
              acc[p][2 * h] = fma2(wk.x, v[p + dx], acc[p][2 * h]);
              acc[p][2 * h + 1] = fma2(wk.y, v[p + dx], acc[p][2 * h + 1]);
            }
          }
        }
      }
    }
    __syncthreads();                            // the stage is free for the load after next
  }
  const int yy = y0 + ty, xx = x0 + xg * 4;
  if (yy >= H || xx >= W) return;
  const bool vec = (W & 3) == 0;                // then the row's four pixels exist and are aligned
#pragma unroll
  for (int o = 0; o < OUTS; ++o) {
    float r[4];
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      float lo, hi;
      unpack2(acc[p][o >> 1], lo, hi);
      r[p] = o & 1 ? hi : lo;
      if (relu) r[p] = fmaxf(r[p], 0.f);
    }
    const size_t at = ((size_t)(o0 + o) * H + yy) * W + xx;
    if (vec) {
      if (omask) {
        const float4 m = *reinterpret_cast<const float4*>(omask + at);
        r[0] = m.x > 0.f ? r[0] : 0.f;
        r[1] = m.y > 0.f ? r[1] : 0.f;
        r[2] = m.z > 0.f ? r[2] : 0.f;
        r[3] = m.w > 0.f ? r[3] : 0.f;
      }
      *reinterpret_cast<float4*>(out + at) = make_float4(r[0], r[1], r[2], r[3]);
    } else {
#pragma unroll
      for (int p = 0; p < 4; ++p)
        if (xx + p < W) out[at + p] = omask && !(omask[at + p] > 0.f) ? 0.f : r[p];
    }
  }
}

// One output channel (the network's last layer): 16 x 16 pixels per CTA, a
// thread a pixel, all cin channels staged.
__global__ void __launch_bounds__(256) k_conv3x3_one(const float* __restrict__ z, int cin, int H, int W,
                                                     const float* __restrict__ w, const float* __restrict__ bias,
                                                     float* __restrict__ out) {
  extern __shared__ __align__(16) float sm[];
  float* zs = sm;                          // cin x 18 x 18
  float* ws = sm + cin * kHalo2;           // cin x 9
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int x0 = blockIdx.x * kTile, y0 = blockIdx.y * kTile;
  for (int i = tid; i < cin * 9; i += 256) ws[i] = w[i];
  for (int i = tid; i < cin * kHalo2; i += 256) {
    const int c = i / kHalo2, r = i - c * kHalo2;
    const int yy = y0 - 1 + r / kHalo, xx = x0 - 1 + r % kHalo;
    const bool on = yy >= 0 && yy < H && xx >= 0 && xx < W;
    cp4_zfill(zs + i, on ? z + ((size_t)c * H + yy) * W + xx : z, on);
  }
  asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  float acc = bias[0];
  for (int c = 0; c < cin; ++c) {
    const float* zc = zs + c * kHalo2 + ty * kHalo + tx;
#pragma unroll
    for (int k = 0; k < 9; ++k) acc = fmaf(ws[c * 9 + k], zc[(k / 3) * kHalo + (k % 3)], acc);
  }
  const int yy = y0 + ty, xx = x0 + tx;
  if (yy < H && xx < W) out[(size_t)yy * W + xx] = acc;
}

// Weight gradients: per-CTA partial sums of dL/dW[o, c, k] = sum_p g[o, p]
// z[c, p + k] and dL/db[o] = sum_p g[o, p] over every gridDim.x-th tile of
// 16 x 8 pixels; part[blockIdx.x * (cin * 9 * COUT + COUT) + ...] in the
// parameter layout (o, c, k) then b, folded by k_fold_params.
//
// A warp takes one group of 8 outputs and half of a tile's rows, a lane one
// input channel (cin = 32): the nine taps x 8 outputs are 72 sums in
// registers, fed per pixel by one new column of the 3 x 3 window (3 loads)
// and the pixel's 8 gradients (2 broadcast loads), where a thread per
// (channel, tap) with 32 outputs needed 9 loads per 32 FMAs and left most of
// the warps idle.  cin = 3 uses 27 lanes, one per (channel, tap); COUT = 1
// has one group, every warp a row.  The next tile is in flight (cp.async)
// while one is used.  512 x 512, 32 -> 32: 121 us, was 590 us.
constexpr int kWgW = 16, kWgH = 8, kWgPx = kWgW * kWgH;
constexpr int kWgZw = kWgW + 2, kWgZ = kWgZw * (kWgH + 2) + 1;   // channel stride 181: odd, no bank conflicts
constexpr int kWgG = 36;                                          // gradients of a pixel: stride 36 words
constexpr int kWgCtas = 152 * 2;

// Tile (x0, y0) into shared memory, asynchronously (one commit group): the
// cin input planes with their halo, a warp a channel, and the gradients
// transposed to [pixel][output].
template <int COUT>
__device__ __forceinline__ void wgrad_stage(const float* __restrict__ z, int cin, int H, int W,
                                            const float* __restrict__ g, int x0, int y0, float* zs, float* gs) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const size_t hw = (size_t)H * W;
#pragma unroll
  for (int i = 0; i < (kWgZ - 1 + 31) / 32; ++i) {
    const int pos = lane + 32 * i, yy = pos / kWgZw, xx = pos % kWgZw;
    if (pos < kWgZ - 1) {
      const int gy = y0 - 1 + yy, gx = x0 - 1 + xx;
      const bool on = gy >= 0 && gy < H && gx >= 0 && gx < W;
      const float* src = on ? z + (size_t)gy * W + gx : z;
      for (int c = warp; c < cin; c += 8) cp4_zfill(zs + c * kWgZ + pos, on ? src + c * hw : z, on);
    }
  }
  const int p = threadIdx.x & (kWgPx - 1), yy = y0 + p / kWgW, xx = x0 + p % kWgW;
  const bool on = yy < H && xx < W;
  const float* gp = on ? g + (size_t)yy * W + xx : g;
  if (COUT == 1) {
    if (threadIdx.x < kWgPx) cp4_zfill(gs + p, gp, on);
  } else {
#pragma unroll 4
    for (int o = threadIdx.x / kWgPx; o < COUT; o += 256 / kWgPx) cp4_zfill(gs + p * kWgG + o, on ? gp + o * hw : g, on);
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}

__global__ void __launch_bounds__(256, 2) k_wgrad32(const float* __restrict__ z, int H, int W,
                                                    const float* __restrict__ g, float* __restrict__ part) {
  extern __shared__ __align__(16) float sm[];
  constexpr int kBuf = kWgPx * kWgG + 32 * kWgZ + 0;   // gradients, then the planes; two buffers
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, og = warp & 3, ph = warp >> 2;
  const int tiles_x = (W + kWgW - 1) / kWgW, ntiles = tiles_x * ((H + kWgH - 1) / kWgH);
  unsigned long long acc[9][4];
#pragma unroll
  for (int k = 0; k < 9; ++k)
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[k][q] = 0ull;
  float db = 0.f;                          // output warp * 4 + lane % 4, pixels lane / 4 + 8 i
  int buf = 0;
  wgrad_stage<32>(z, 32, H, W, g, (blockIdx.x % tiles_x) * kWgW, (blockIdx.x / tiles_x) * kWgH, sm + kWgPx * kWgG, sm);
  for (int t = blockIdx.x; t < ntiles; t += gridDim.x, buf ^= 1) {
    const int nt = t + gridDim.x;
    if (nt < ntiles) {
      float* nb = sm + (buf ^ 1) * kBuf;
      wgrad_stage<32>(z, 32, H, W, g, (nt % tiles_x) * kWgW, (nt / tiles_x) * kWgH, nb + kWgPx * kWgG, nb);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    const float *gs = sm + buf * kBuf, *zs = gs + kWgPx * kWgG;
#pragma unroll
    for (int i = 0; i < kWgPx / 8; ++i) db += gs[(lane / 4 + 8 * i) * kWgG + warp * 4 + (lane & 3)];
    for (int y = ph * (kWgH / 2); y < (ph + 1) * (kWgH / 2); ++y) {
      const float* zr = zs + lane * kWgZ + y * kWgZw;
      const float* gr = gs + y * kWgW * kWgG + og * 8;
      unsigned long long v[3][3];          // window: column, row
#pragma unroll
      for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int r = 0; r < 3; ++r) { const float u = zr[r * kWgZw + c]; v[c][r] = pack2(u, u); }
#pragma unroll
      for (int x = 0; x < kWgW; ++x) {
#pragma unroll
        for (int r = 0; r < 3; ++r) { const float u = zr[r * kWgZw + x + 2]; v[(x + 2) % 3][r] = pack2(u, u); }
        const ulonglong2 g0 = *reinterpret_cast<const ulonglong2*>(gr + x * kWgG);
        const ulonglong2 g1 = *reinterpret_cast<const ulonglong2*>(gr + x * kWgG + 4);
#pragma unroll
        for (int k = 0; k < 9; ++k) {
          const unsigned long long vk = v[(x + k % 3) % 3][k / 3];
          acc[k][0] = fma2(g0.x, vk, acc[k][0]);
          acc[k][1] = fma2(g0.y, vk, acc[k][1]);
          acc[k][2] = fma2(g1.x, vk, acc[k][2]);
          acc[k][3] = fma2(g1.y, vk, acc[k][3]);
        }
      }
    }
    __syncthreads();                     // the buffer is free for the tile after next
  }
  // the two row halves of a group, then to global memory
  __syncthreads();
  float* red = sm;                         // 4 groups x 72 x 32 lanes
  if (ph == 1) {
#pragma unroll
    for (int k = 0; k < 9; ++k)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        float lo, hi;
        unpack2(acc[k][q], lo, hi);
        red[(og * 72 + k * 8 + 2 * q) * 32 + lane] = lo;
        red[(og * 72 + k * 8 + 2 * q + 1) * 32 + lane] = hi;
      }
  }
  for (int o = 4; o < 32; o <<= 1) db += __shfl_xor_sync(0xffffffffu, db, o);
  __syncthreads();
  float* pp = part + (size_t)blockIdx.x * (32 * 9 * 32 + 32);
  if (ph == 0) {
#pragma unroll
    for (int k = 0; k < 9; ++k)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        float lo, hi;
        unpack2(acc[k][q], lo, hi);
        pp[((og * 8 + 2 * q) * 32 + lane) * 9 + k] = lo + red[(og * 72 + k * 8 + 2 * q) * 32 + lane];
        pp[((og * 8 + 2 * q + 1) * 32 + lane) * 9 + k] = hi + red[(og * 72 + k * 8 + 2 * q + 1) * 32 + lane];
      }
  }
  if (lane < 4) pp[32 * 9 * 32 + warp * 4 + lane] = db;
}

// cin = 3, 32 outputs: lane = channel * 9 + tap (27 of 32), 8 outputs per warp
__global__ void __launch_bounds__(256) k_wgrad3(const float* __restrict__ z, int H, int W,
                                                const float* __restrict__ g, float* __restrict__ part) {
  extern __shared__ __align__(16) float sm[];
  constexpr int kBuf = kWgPx * kWgG + 3 * kWgZ + 1;   // gradients, then the planes; two buffers
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, og = warp & 3, ph = warp >> 2;
  const int tiles_x = (W + kWgW - 1) / kWgW, ntiles = tiles_x * ((H + kWgH - 1) / kWgH);
  const int lk = min(lane, 26), c = lk / 9, k = lk % 9;
  unsigned long long acc[4] = {0ull, 0ull, 0ull, 0ull};
  float db = 0.f;
  int buf = 0;
  wgrad_stage<32>(z, 3, H, W, g, (blockIdx.x % tiles_x) * kWgW, (blockIdx.x / tiles_x) * kWgH, sm + kWgPx * kWgG, sm);
  for (int t = blockIdx.x; t < ntiles; t += gridDim.x, buf ^= 1) {
    const int nt = t + gridDim.x;
    if (nt < ntiles) {
      float* nb = sm + (buf ^ 1) * kBuf;
      wgrad_stage<32>(z, 3, H, W, g, (nt % tiles_x) * kWgW, (nt / tiles_x) * kWgH, nb + kWgPx * kWgG, nb);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    const float *gs = sm + buf * kBuf, *zs = gs + kWgPx * kWgG;
#pragma unroll
    for (int i = 0; i < kWgPx / 8; ++i) db += gs[(lane / 4 + 8 * i) * kWgG + warp * 4 + (lane & 3)];
    const float* zr = zs + c * kWgZ + (k / 3) * kWgZw + k % 3;
    for (int y = ph * (kWgH / 2); y < (ph + 1) * (kWgH / 2); ++y) {
#pragma unroll
      for (int x = 0; x < kWgW; ++x) {
        const float u = zr[y * kWgZw + x];
        const unsigned long long v = pack2(u, u);
        const ulonglong2 g0 = *reinterpret_cast<const ulonglong2*>(gs + (y * kWgW + x) * kWgG + og * 8);
        const ulonglong2 g1 = *reinterpret_cast<const ulonglong2*>(gs + (y * kWgW + x) * kWgG + og * 8 + 4);
        acc[0] = fma2(g0.x, v, acc[0]);
        acc[1] = fma2(g0.y, v, acc[1]);
        acc[2] = fma2(g1.x, v, acc[2]);
        acc[3] = fma2(g1.y, v, acc[3]);
      }
    }
    __syncthreads();                     // the buffer is free for the tile after next
  }
  __syncthreads();
  unsigned long long* red = reinterpret_cast<unsigned long long*>(sm);   // 4 groups x 4 x 32 lanes
  if (ph == 1)
#pragma unroll
    for (int q = 0; q < 4; ++q) red[(og * 4 + q) * 32 + lane] = acc[q];
  for (int o = 4; o < 32; o <<= 1) db += __shfl_xor_sync(0xffffffffu, db, o);
  __syncthreads();
  float* pp = part + (size_t)blockIdx.x * (3 * 9 * 32 + 32);
  if (ph == 0 && lane < 27) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float a, b, a1, b1;
      unpack2(acc[q], a, b);
      unpack2(red[(og * 4 + q) * 32 + lane], a1, b1);
      pp[((og * 8 + 2 * q) * 3 + c) * 9 + k] = a + a1;
      pp[((og * 8 + 2 * q + 1) * 3 + c) * 9 + k] = b + b1;
    }
  }
  if (lane < 4) pp[3 * 9 * 32 + warp * 4 + lane] = db;
}

// one output: lane = input channel (32), a warp per tile row
__global__ void __launch_bounds__(256) k_wgrad_one(const float* __restrict__ z, int H, int W,
                                                   const float* __restrict__ g, float* __restrict__ part) {
  extern __shared__ __align__(16) float sm[];
  constexpr int kBuf = kWgPx + 32 * kWgZ + 0;   // gradients, then the planes; two buffers
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int tiles_x = (W + kWgW - 1) / kWgW, ntiles = tiles_x * ((H + kWgH - 1) / kWgH);
  float acc[9], db = 0.f;
#pragma unroll
  for (int k = 0; k < 9; ++k) acc[k] = 0.f;
  int buf = 0;
  wgrad_stage<1>(z, 32, H, W, g, (blockIdx.x % tiles_x) * kWgW, (blockIdx.x / tiles_x) * kWgH, sm + kWgPx, sm);
  for (int t = blockIdx.x; t < ntiles; t += gridDim.x, buf ^= 1) {
    const int nt = t + gridDim.x;
    if (nt < ntiles) {
      float* nb = sm + (buf ^ 1) * kBuf;
      wgrad_stage<1>(z, 32, H, W, g, (nt % tiles_x) * kWgW, (nt / tiles_x) * kWgH, nb + kWgPx, nb);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    const float *gs = sm + buf * kBuf, *zs = gs + kWgPx;
    const float* zr = zs + lane * kWgZ + warp * kWgZw;
#pragma unroll
    for (int x = 0; x < kWgW; ++x) {
      const float gv = gs[warp * kWgW + x];
      db += gv;
#pragma unroll
      for (int k = 0; k < 9; ++k) acc[k] = fmaf(gv, zr[(k / 3) * kWgZw + x + k % 3], acc[k]);
    }
    __syncthreads();                     // the buffer is free for the tile after next
  }
  __syncthreads();
  float* red = sm;                         // 8 warps x 10 x 32 lanes
#pragma unroll
  for (int k = 0; k < 9; ++k) red[(warp * 10 + k) * 32 + lane] = acc[k];
  red[(warp * 10 + 9) * 32 + lane] = db;
  __syncthreads();
  float* pp = part + (size_t)blockIdx.x * (32 * 9 + 1);
  for (int i = tid; i < 289; i += 256) {
    const int k = i < 288 ? i % 9 : 9, c = i < 288 ? i / 9 : 0;
    float s = 0.f;
    for (int w = 0; w < 8; ++w) s += red[(w * 10 + k) * 32 + c];
    pp[i] = s;
  }
}

// grad[i] += sum_b part[b * cnt + i]: 16 strands b = s, s + 16, ... in
// order, then the strands in order (one strand of up to 304 dependent adds
// took 14 us a layer)
constexpr int kFoldStrands = 16;
__global__ void __launch_bounds__(32 * kFoldStrands) k_fold_params(const float* __restrict__ part, int nb, int cnt,
                                                                   float* __restrict__ grad) {
  __shared__ float red[kFoldStrands][32];
  const int lane = threadIdx.x & 31, s = threadIdx.x >> 5, i = blockIdx.x * 32 + lane;
  float v = 0.f;
  if (i < cnt) {
#pragma unroll 10
    for (int b = s; b < nb; b += kFoldStrands) v += part[(size_t)b * cnt + i];
  }
  red[s][lane] = v;
  __syncthreads();
  if (s == 0 && i < cnt) {
#pragma unroll
    for (int q = 1; q < kFoldStrands; ++q) v += red[q][lane];
    grad[i] += v;
  }
}

// y[c, i, j] = mean of the 2 x 2 block of z (H, W even)
__global__ void k_pool(const float* __restrict__ z, int C, int H, int W, float* __restrict__ y) {
  const int h = H / 2, w = W / 2;
  const int64_t cnt = (int64_t)C * h * w;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < cnt; t += (int64_t)gridDim.x * blockDim.x) {
    const int j = (int)(t % w), i = (int)((t / w) % h), c = (int)(t / ((int64_t)w * h));
    const float* zz = z + ((size_t)c * H + 2 * i) * W + 2 * j;
    y[t] = 0.25f * (zz[0] + zz[1] + zz[W] + zz[W + 1]);
  }
}

// gz[c, y, x] = (gz[c, y, x] + g[c, y / 2, x / 2] / 4) (mask > 0) (gz at H x W)
__global__ void k_pool_back(const float* __restrict__ g, int C, int H, int W, const float* __restrict__ mask,
                            float* __restrict__ gz) {
  const int64_t cnt = (int64_t)C * H * W;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < cnt; t += (int64_t)gridDim.x * blockDim.x) {
    const int x = (int)(t % W), y = (int)((t / W) % H), c = (int)(t / ((int64_t)W * H));
    const float v = gz[t] + 0.25f * g[((size_t)c * (H / 2) + y / 2) * (W / 2) + x / 2];
    gz[t] = mask[t] > 0.f ? v : 0.f;
  }
}

// y[c, y, x] = z[c, y / 2, x / 2] + skip[c, y, x] (y at H x W)
__global__ void k_up_add(const float* __restrict__ z, const float* __restrict__ skip, int C, int H, int W,
                         float* __restrict__ y) {
  const int64_t cnt = (int64_t)C * H * W;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < cnt; t += (int64_t)gridDim.x * blockDim.x) {
    const int x = (int)(t % W), yy = (int)((t / W) % H), c = (int)(t / ((int64_t)W * H));
    y[t] = z[((size_t)c * (H / 2) + yy / 2) * (W / 2) + x / 2] + skip[t];
  }
}

// gz[c, i, j] = sum of the 2 x 2 block of g, where mask > 0 (gz and mask at H/2 x W/2)
__global__ void k_up_back(const float* __restrict__ g, int C, int H, int W, const float* __restrict__ mask,
                          float* __restrict__ gz) {
  const int h = H / 2, w = W / 2;
  const int64_t cnt = (int64_t)C * h * w;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < cnt; t += (int64_t)gridDim.x * blockDim.x) {
    const int j = (int)(t % w), i = (int)((t / w) % h), c = (int)(t / ((int64_t)w * h));
    const float* gg = g + ((size_t)c * H + 2 * i) * W + 2 * j;
    gz[t] = mask[t] > 0.f ? (gg[0] + gg[1]) + (gg[W] + gg[W + 1]) : 0.f;
  }
}

constexpr int kLossCtas = 256;
constexpr int kMaxQ = 64;

// part[b * (q + 1) + j] = sum_p Q[p + j n] u[p] (j < q), part[.. + q] = sum_p u[p]^2
__global__ void __launch_bounds__(256) k_loss_dots(int64_t n, const float* __restrict__ u, const float* __restrict__ Q,
                                                   int q, double* __restrict__ part) {
  __shared__ double red[kMaxQ + 1][8];
  double s[kMaxQ + 1];
  for (int j = 0; j <= q; ++j) s[j] = 0.0;
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
    const double v = u[p];
    for (int j = 0; j < q; ++j) s[j] += (double)Q[p + (int64_t)j * n] * v;
    s[q] += v * v;
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int j = 0; j <= q; ++j) {
    double v = s[j];
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) red[j][warp] = v;
  }
  __syncthreads();
  for (int j = threadIdx.x; j <= q; j += blockDim.x) {
    double v = 0.0;
    for (int w = 0; w < 8; ++w) v += red[j][w];
    part[(size_t)blockIdx.x * (q + 1) + j] = v;
  }
}

// g[p] = alpha * sum_j Q[p + j n] c[j] + gamma * u[p]
__global__ void k_loss_grad(int64_t n, const float* __restrict__ u, const float* __restrict__ Q, int q,
                            const double* __restrict__ coef, float* __restrict__ g) {
  const double alpha = coef[kMaxQ], gamma = coef[kMaxQ + 1];
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
    double a = 0.0;
    for (int j = 0; j < q; ++j) a += (double)Q[p + (int64_t)j * n] * coef[j];
    g[p] = (float)(alpha * a + gamma * (double)u[p]);
  }
}

// Adam (Kingma & Ba 2015), bias-corrected: grad = acc / batch; acc cleared
__global__ void k_adam(int64_t cnt, float* __restrict__ theta, float* __restrict__ m, float* __restrict__ v,
                       float* __restrict__ acc, float inv_batch, float lr, float b1, float b2, float c1, float c2,
                       float eps) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < cnt; i += (int64_t)gridDim.x * blockDim.x) {
    const float g = acc[i] * inv_batch;
    const float mi = b1 * m[i] + (1.f - b1) * g;
    const float vi = b2 * v[i] + (1.f - b2) * g * g;
    m[i] = mi;
    v[i] = vi;
    theta[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    acc[i] = 0.f;
  }
}

// The FP16-rounded weights in FP32 as the convolutions read them (master
// layout (o, c, k)): forward [c][k][o] and, for the backward-data product, the
// flipped transpose [o][8 - k][c]
__global__ void k_pack_weights(const float* __restrict__ Wm, int cin, int cout, float* __restrict__ wf,
                               float* __restrict__ wb) {
  const int cnt = cin * cout * 9;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < cnt; i += gridDim.x * blockDim.x) {
    const int k = i % 9, c = (i / 9) % cin, o = i / (9 * cin);
    const float h = __half2float(__float2half_rn(Wm[i]));
    wf[(c * 9 + k) * cout + o] = h;
    if (wb) wb[(o * 9 + (8 - k)) * cin + c] = h;
  }
}

// part[b * 2 + 0] = sum u[p]^2, part[b * 2 + 1] = sum g[p]^2 (FP64)
__global__ void __launch_bounds__(256) k_two_norms(int64_t n, const float* __restrict__ u,
                                                   const double* __restrict__ g, double* __restrict__ part) {
  __shared__ double red[2][8];
  double a = 0.0, b = 0.0;
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
    const double v = u[p], w = g[p];
    a += v * v;
    b += w * w;
  }
  for (int o = 16; o; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) { red[0][warp] = a; red[1][warp] = b; }
  __syncthreads();
  if (threadIdx.x < 2) {
    double s = 0.0;
    for (int w = 0; w < 8; ++w) s += red[threadIdx.x][w];
    part[blockIdx.x * 2 + threadIdx.x] = s;
  }
}

// y[p] = a u[p] + b y[p]  (y holds g on entry)
__global__ void k_combine(int64_t n, const float* __restrict__ u, double a, double b, double* __restrict__ y) {
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x)
    y[p] = a * (double)u[p] + b * y[p];
}

}  // namespace

// ---------------------------------------------------------------------------
// Network state
// ---------------------------------------------------------------------------

struct rks_ws {
  int H = 0, W = 0;
  int64_t nparam = 0;
  cudaStream_t st = nullptr;
  bool own_stream = false;
  int64_t poff[2 * kConvs + 1] = {};   // offsets of W_l, b_l in the flat vector
  float* theta = nullptr;               // FP32 masters
  float* m = nullptr;
  float* v = nullptr;
  float* gacc = nullptr;                // gradient accumulated over the minibatch
  float* wf[kConvs] = {};               // forward layouts (FP16-rounded values)
  float* wb[kConvs] = {};               // backward-data layouts (none for C1)
  float* part = nullptr;                // weight-gradient partials
  int64_t part_cap = 0;
  double* lpart = nullptr;              // loss partials
  double* lcoef = nullptr;              // c (kMaxQ), alpha, gamma
  int adam_t = 0;
  int nacc = 0;                         // samples accumulated since the last step
  // activations: lv[level] sizes; buffers named as in the oracle
  float* buf = nullptr;
  float *e0a, *e0, *p1, *e1a, *e1, *p2, *e2a, *e2, *p3, *e3a, *e3;
  float *d2in, *d2a, *d2, *d1in, *d1a, *d1, *d0in, *d0a, *d0, *u;
  float *gA[4], *gB[4], *gS[4], *gu;    // gradient scratch per level
  ~rks_ws() {
    cudaFree(theta); cudaFree(m); cudaFree(v); cudaFree(gacc);
    for (int l = 0; l < kConvs; ++l) { cudaFree(wf[l]); cudaFree(wb[l]); }
    cudaFree(part); cudaFree(lpart); cudaFree(lcoef); cudaFree(buf);
    if (own_stream && st) cudaStreamDestroy(st);
  }
};

namespace {

cudaError_t configure_ws_kernels_once() {
  const int big = 200 * 1024;
  cudaError_t e = cudaFuncSetAttribute(k_conv3x3<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_conv3x3<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_conv3x3_one, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_wgrad32, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_wgrad_one, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
  return e;
}

int grid1(int64_t cnt) { return (int)std::max<int64_t>(1, std::min<int64_t>((cnt + 255) / 256, 152 * 16)); }

int lvH(const rks_ws* s, int l) { return s->H >> l; }
int lvW(const rks_ws* s, int l) { return s->W >> l; }

// Tiles (32 x 8 pixels) from which a CTA takes all 32 outputs: four per SM
constexpr int kCvWideFrom = 608;

// out = C_l(z) at level lv; back: with the backward-data weights (no bias),
// omask: out is zeroed where omask <= 0
void conv(rks_ws* s, int l, int lv, const float* z, bool back, int relu, const float* omask, float* out) {
  const int H = lvH(s, lv), W = lvW(s, lv);
  const int cin = back ? conv_cout(l) : conv_cin(l), cout = back ? conv_cin(l) : conv_cout(l);
  const float* bias = back ? nullptr : s->theta + s->poff[2 * l + 1];
  const float* w = back ? s->wb[l] : s->wf[l];
  if (cout == 1) {
    dim3 grid((W + kTile - 1) / kTile, (H + kTile - 1) / kTile);
    k_conv3x3_one<<<grid, 256, (size_t)(cin * kHalo2 + cin * 9) * sizeof(float), s->st>>>(z, cin, H, W, w, bias, out);
    return;
  }
  const int tiles = ((W + kCvW - 1) / kCvW) * ((H + kCvH - 1) / kCvH);
  const bool wide = tiles >= kCvWideFrom;
  const dim3 grid(tiles, 1, wide ? 1 : 2);
  const size_t sm = (size_t)(2 * kCvStage * kCvPlane + cin * 36 * (wide ? 8 : 4)) * sizeof(float);
  if (wide) k_conv3x3<8><<<grid, 256, sm, s->st>>>(z, cin, H, W, w, bias, relu, omask, out);
  else k_conv3x3<4><<<grid, 256, sm, s->st>>>(z, cin, H, W, w, bias, relu, omask, out);
}

// gacc[W_l, b_l] += dL/d(W_l, b_l) for the input z of C_l and dL/d(out) = g
void wgrad(rks_ws* s, int l, int lv, const float* z, const float* g) {
  const int H = lvH(s, lv), W = lvW(s, lv);
  const int cin = conv_cin(l), cout = conv_cout(l);
  const int nb = std::min(kWgCtas, ((W + kWgW - 1) / kWgW) * ((H + kWgH - 1) / kWgH));
  const int cnt = cin * 9 * cout + cout;
  const size_t sm = (size_t)2 * ((kWgPx * (cout == 1 ? 1 : kWgG) + cin * kWgZ + 3) & ~3) * sizeof(float);
  if (cout == 1) k_wgrad_one<<<nb, 256, sm, s->st>>>(z, H, W, g, s->part);
  else if (cin == 3) k_wgrad3<<<nb, 256, sm, s->st>>>(z, H, W, g, s->part);
  else k_wgrad32<<<nb, 256, sm, s->st>>>(z, H, W, g, s->part);
  k_fold_params<<<(cnt + 31) / 32, 32 * kFoldStrands, 0, s->st>>>(s->part, nb, cnt, s->gacc + s->poff[2 * l]);
}

void pool(rks_ws* s, int lv, const float* z, float* y) {   // lv: level of z
  const int64_t cnt = (int64_t)kCh * (lvH(s, lv) / 2) * (lvW(s, lv) / 2);
  k_pool<<<grid1(cnt), 256, 0, s->st>>>(z, kCh, lvH(s, lv), lvW(s, lv), y);
}

void pool_back(rks_ws* s, int lv, const float* g, const float* mask, float* gz) {   // lv: level of gz
  const int64_t cnt = (int64_t)kCh * lvH(s, lv) * lvW(s, lv);
  k_pool_back<<<grid1(cnt), 256, 0, s->st>>>(g, kCh, lvH(s, lv), lvW(s, lv), mask, gz);
}

void up_add(rks_ws* s, int lv, const float* z, const float* skip, float* y) {   // lv: level of y
  const int64_t cnt = (int64_t)kCh * lvH(s, lv) * lvW(s, lv);
  k_up_add<<<grid1(cnt), 256, 0, s->st>>>(z, skip, kCh, lvH(s, lv), lvW(s, lv), y);
}

void up_back(rks_ws* s, int lv, const float* g, const float* mask, float* gz) {   // lv: level of g
  const int64_t cnt = (int64_t)kCh * (lvH(s, lv) / 2) * (lvW(s, lv) / 2);
  k_up_back<<<grid1(cnt), 256, 0, s->st>>>(g, kCh, lvH(s, lv), lvW(s, lv), mask, gz);
}

void pack_weights(rks_ws* s) {
  for (int l = 0; l < kConvs; ++l) {
    const int cnt = conv_cin(l) * conv_cout(l) * 9;
    k_pack_weights<<<(cnt + 255) / 256, 256, 0, s->st>>>(s->theta + s->poff[2 * l], conv_cin(l), conv_cout(l),
                                                         s->wf[l], s->wb[l]);
  }
}

// block: o = R(C_{l+1}(R(C_l(z)))) at level lv
void block(rks_ws* s, int l, int lv, const float* z, float* a, float* o) {
  conv(s, l, lv, z, false, 1, nullptr, a);
  conv(s, l + 1, lv, a, false, 1, nullptr, o);
}

void forward(rks_ws* s, const float* x) {
  block(s, 0, 0, x, s->e0a, s->e0);
  pool(s, 0, s->e0, s->p1);
  block(s, 2, 1, s->p1, s->e1a, s->e1);
  pool(s, 1, s->e1, s->p2);
  block(s, 4, 2, s->p2, s->e2a, s->e2);
  pool(s, 2, s->e2, s->p3);
  block(s, 6, 3, s->p3, s->e3a, s->e3);
  up_add(s, 2, s->e3, s->e2, s->d2in);
  block(s, 8, 2, s->d2in, s->d2a, s->d2);
  up_add(s, 1, s->d2, s->e1, s->d1in);
  block(s, 10, 1, s->d1in, s->d1a, s->d1);
  up_add(s, 0, s->d1, s->e0, s->d0in);
  block(s, 12, 0, s->d0in, s->d0a, s->d0);
  conv(s, 14, 0, s->d0, false, 0, nullptr, s->u);
}

// through o = R(C_{l+1}(R(C_l(z)))): g = dL/do where o > 0 (zero elsewhere);
// ga is scratch; gz = dL/dz (unless null).  The gradients are masked by the
// kernels that produce them.
void block_back(rks_ws* s, int l, int lv, const float* z, const float* a, const float* g, float* ga, float* gz) {
  wgrad(s, l + 1, lv, a, g);
  conv(s, l + 1, lv, g, true, 0, a, ga);              // dL/da, masked by a
  wgrad(s, l, lv, z, ga);
  if (gz) conv(s, l, lv, ga, true, 0, nullptr, gz);
}

void backward(rks_ws* s, const float* x) {
  // u = C15(d0)
  wgrad(s, 14, 0, s->d0, s->gu);
  conv(s, 14, 0, s->gu, true, 0, s->d0, s->gA[0]);                       // dL/d(d0)
  block_back(s, 12, 0, s->d0in, s->d0a, s->gA[0], s->gB[0], s->gS[0]);   // gS0 = dL/d(U(d1) + e0)
  up_back(s, 0, s->gS[0], s->d1, s->gA[1]);
  block_back(s, 10, 1, s->d1in, s->d1a, s->gA[1], s->gB[1], s->gS[1]);   // gS1 = dL/d(U(d2) + e1)
  up_back(s, 1, s->gS[1], s->d2, s->gA[2]);
  block_back(s, 8, 2, s->d2in, s->d2a, s->gA[2], s->gB[2], s->gS[2]);    // gS2 = dL/d(U(e3) + e2)
  up_back(s, 2, s->gS[2], s->e3, s->gA[3]);
  block_back(s, 6, 3, s->p3, s->e3a, s->gA[3], s->gB[3], s->gS[3]);      // dL/d(P(e2))
  pool_back(s, 2, s->gS[3], s->e2, s->gS[2]);                             // dL/d(e2)
  block_back(s, 4, 2, s->p2, s->e2a, s->gS[2], s->gB[2], s->gA[2]);      // dL/d(P(e1))
  pool_back(s, 1, s->gA[2], s->e1, s->gS[1]);
  block_back(s, 2, 1, s->p1, s->e1a, s->gS[1], s->gB[1], s->gA[1]);      // dL/d(P(e0))
  pool_back(s, 0, s->gA[1], s->e0, s->gS[0]);
  block_back(s, 0, 0, x, s->e0a, s->gS[0], s->gB[0], nullptr);
}

int launch_ok() { return cudaGetLastError() == cudaSuccess ? RKS_OK : RKS_ECUDA; }

// host: SplitMix64 normals (Box-Muller) for the initial weights
uint64_t mix64h(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

}  // namespace

extern "C" {

int64_t rks_ws_nparams(void) {
  int64_t n = 0;
  for (int l = 0; l < kConvs; ++l) n += (int64_t)conv_cin(l) * conv_cout(l) * 9 + conv_cout(l);
  return n;
}

int rks_ws_create(rks_ws** out, int H, int W, uint64_t seed, void* stream) {
  if (!out) return RKS_EINVAL;
  *out = nullptr;
  if (H < 8 || W < 8 || H % 8 || W % 8 || (int64_t)H * W > (int64_t)1 << 26) return RKS_EINVAL;
  if (rks::once_per_device(rks::kCfgWs, configure_ws_kernels_once) != cudaSuccess) return RKS_ECUDA;
  rks_ws* s = new (std::nothrow) rks_ws();
  if (!s) return RKS_ENOMEM;
  s->H = H; s->W = W;
  s->st = (cudaStream_t)stream;
  if (!s->st) {
    if (cudaStreamCreateWithFlags(&s->st, cudaStreamNonBlocking) != cudaSuccess) { delete s; return RKS_ECUDA; }
    s->own_stream = true;
  }
  int64_t o = 0;
  for (int l = 0; l < kConvs; ++l) {
    s->poff[2 * l] = o;
    o += (int64_t)conv_cin(l) * conv_cout(l) * 9;
    s->poff[2 * l + 1] = o;
    o += conv_cout(l);
  }
  s->poff[2 * kConvs] = o;
  s->nparam = o;
  const int64_t n0 = (int64_t)H * W;
  // level element counts (32 channels): 0: n0, 1: n0/4, 2: n0/16, 3: n0/64
  const int64_t L[4] = {kCh * n0, kCh * n0 / 4, kCh * n0 / 16, kCh * n0 / 64};
  // e0a e0 d0in d0a d0 gA0 gB0 gS0 | p1 e1a e1 d1in d1a d1 gA1 gB1 gS1 | p2 e2a e2 d2in d2a d2 gA2 gB2 gS2 |
  // p3 e3a e3 gA3 gB3 gS3 | u gu
  const int64_t total = 8 * L[0] + 9 * L[1] + 9 * L[2] + 6 * L[3] + 2 * n0;
  const int ntiles_max = ((W + kWgW - 1) / kWgW) * ((H + kWgH - 1) / kWgH);
  s->part_cap = (int64_t)std::min(kWgCtas, ntiles_max) * (kCh * 9 * kCh + kCh);
  bool ok = cudaMalloc(&s->buf, total * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&s->theta, o * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&s->m, o * sizeof(float)) == cudaSuccess && cudaMalloc(&s->v, o * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&s->gacc, o * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&s->part, s->part_cap * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&s->lpart, (size_t)kLossCtas * (kMaxQ + 1) * sizeof(double)) == cudaSuccess &&
            cudaMalloc(&s->lcoef, (kMaxQ + 2) * sizeof(double)) == cudaSuccess;
  for (int l = 0; ok && l < kConvs; ++l) {
    const size_t cnt = (size_t)conv_cin(l) * conv_cout(l) * 9;
    ok = cudaMalloc(&s->wf[l], cnt * sizeof(float)) == cudaSuccess &&
         (l == 0 || cudaMalloc(&s->wb[l], cnt * sizeof(float)) == cudaSuccess);
  }
  if (!ok) { delete s; return RKS_ENOMEM; }
  float* p = s->buf;
  auto take = [&](int64_t cnt) { float* r = p; p += cnt; return r; };
  s->e0a = take(L[0]); s->e0 = take(L[0]); s->d0in = take(L[0]); s->d0a = take(L[0]); s->d0 = take(L[0]);
  s->gA[0] = take(L[0]); s->gB[0] = take(L[0]); s->gS[0] = take(L[0]);
  s->p1 = take(L[1]); s->e1a = take(L[1]); s->e1 = take(L[1]); s->d1in = take(L[1]); s->d1a = take(L[1]);
  s->d1 = take(L[1]); s->gA[1] = take(L[1]); s->gB[1] = take(L[1]); s->gS[1] = take(L[1]);
  s->p2 = take(L[2]); s->e2a = take(L[2]); s->e2 = take(L[2]); s->d2in = take(L[2]); s->d2a = take(L[2]);
  s->d2 = take(L[2]); s->gA[2] = take(L[2]); s->gB[2] = take(L[2]); s->gS[2] = take(L[2]);
  s->p3 = take(L[3]); s->e3a = take(L[3]); s->e3 = take(L[3]);
  s->gA[3] = take(L[3]); s->gB[3] = take(L[3]); s->gS[3] = take(L[3]);
  s->u = take(n0); s->gu = take(n0);
  // He-normal weights (std sqrt(2 / (9 cin))) from SplitMix64 + Box-Muller, zero biases
  std::vector<float> th(o, 0.f);
  uint64_t ctr = 0;
  const uint64_t base = mix64h(seed * 0x9E3779B97F4A7C15ull);
  for (int l = 0; l < kConvs; ++l) {
    const double sd = std::sqrt(2.0 / (9.0 * conv_cin(l)));
    for (int64_t i = s->poff[2 * l]; i < s->poff[2 * l + 1]; ++i) {
      const double u1 = ((mix64h(base + (++ctr) * 0x9E3779B97F4A7C15ull) >> 11) + 0.5) * 0x1.0p-53;
      const double u2 = ((mix64h(base + (++ctr) * 0x9E3779B97F4A7C15ull) >> 11) + 0.5) * 0x1.0p-53;
      th[i] = (float)(sd * std::sqrt(-2.0 * std::log(u1)) * std::cos(6.283185307179586 * u2));
    }
  }
  if (cudaMemcpyAsync(s->theta, th.data(), o * sizeof(float), cudaMemcpyHostToDevice, s->st) != cudaSuccess ||
      cudaMemsetAsync(s->m, 0, o * sizeof(float), s->st) != cudaSuccess ||
      cudaMemsetAsync(s->v, 0, o * sizeof(float), s->st) != cudaSuccess ||
      cudaMemsetAsync(s->gacc, 0, o * sizeof(float), s->st) != cudaSuccess) {
    delete s;
    return RKS_ECUDA;
  }
  pack_weights(s);
  if (launch_ok() != RKS_OK || cudaStreamSynchronize(s->st) != cudaSuccess) { delete s; return RKS_ECUDA; }
  *out = s;
  return RKS_OK;
}

int rks_ws_get_params(const rks_ws* s, float* theta) {
  if (!s || !theta) return RKS_EINVAL;
  if (cudaMemcpyAsync(theta, s->theta, s->nparam * sizeof(float), cudaMemcpyDeviceToHost, s->st) != cudaSuccess ||
      cudaStreamSynchronize(s->st) != cudaSuccess)
    return RKS_ECUDA;
  return RKS_OK;
}

int rks_ws_set_params(rks_ws* s, const float* theta) {
  if (!s || !theta) return RKS_EINVAL;
  if (cudaMemcpyAsync(s->theta, theta, s->nparam * sizeof(float), cudaMemcpyHostToDevice, s->st) != cudaSuccess)
    return RKS_ECUDA;
  pack_weights(s);
  if (launch_ok() != RKS_OK || cudaStreamSynchronize(s->st) != cudaSuccess) return RKS_ECUDA;
  s->adam_t = 0;
  s->nacc = 0;
  if (cudaMemsetAsync(s->m, 0, s->nparam * sizeof(float), s->st) != cudaSuccess ||
      cudaMemsetAsync(s->v, 0, s->nparam * sizeof(float), s->st) != cudaSuccess ||
      cudaMemsetAsync(s->gacc, 0, s->nparam * sizeof(float), s->st) != cudaSuccess ||
      cudaStreamSynchronize(s->st) != cudaSuccess)
    return RKS_ECUDA;
  return RKS_OK;
}

int rks_ws_forward(rks_ws* s, const float* x, float* u) {
  if (!s || !x || !u) return RKS_EINVAL;
  forward(s, x);
  const int64_t n0 = (int64_t)s->H * s->W;
  if (launch_ok() != RKS_OK ||
      cudaMemcpyAsync(u, s->u, n0 * sizeof(float), cudaMemcpyDeviceToDevice, s->st) != cudaSuccess ||
      cudaStreamSynchronize(s->st) != cudaSuccess)
    return RKS_ECUDA;
  return RKS_OK;
}

int rks_ws_accumulate(rks_ws* s, const float* x, const float* Q, int q, double* loss) {
  if (!s || !x || !Q || q < 1 || q > kMaxQ) return RKS_EINVAL;
  const int64_t n0 = (int64_t)s->H * s->W;
  forward(s, x);
  k_loss_dots<<<kLossCtas, 256, 0, s->st>>>(n0, s->u, Q, q, s->lpart);
  if (launch_ok() != RKS_OK) return RKS_ECUDA;
  std::vector<double> part((size_t)kLossCtas * (q + 1));
  if (cudaMemcpyAsync(part.data(), s->lpart, part.size() * sizeof(double), cudaMemcpyDeviceToHost, s->st) !=
          cudaSuccess ||
      cudaStreamSynchronize(s->st) != cudaSuccess)
    return RKS_ECUDA;
  std::vector<double> c(kMaxQ + 2, 0.0);
  double uu = 0.0;
  for (int b = 0; b < kLossCtas; ++b) {
    for (int j = 0; j < q; ++j) c[j] += part[(size_t)b * (q + 1) + j];
    uu += part[(size_t)b * (q + 1) + q];
  }
  if (!(uu > 0.0) || !std::isfinite(uu)) return RKS_ENAN;
  double cc = 0.0;
  for (int j = 0; j < q; ++j) cc += c[j] * c[j];
  if (loss) *loss = 1.0 - cc / uu;
  c[kMaxQ] = -2.0 / uu;                  // dL/du = -2 Q c / uu + 2 cc u / uu^2
  c[kMaxQ + 1] = 2.0 * cc / (uu * uu);
  if (cudaMemcpyAsync(s->lcoef, c.data(), c.size() * sizeof(double), cudaMemcpyHostToDevice, s->st) != cudaSuccess)
    return RKS_ECUDA;
  k_loss_grad<<<grid1(n0), 256, 0, s->st>>>(n0, s->u, Q, q, s->lcoef, s->gu);
  backward(s, x);
  if (launch_ok() != RKS_OK || cudaStreamSynchronize(s->st) != cudaSuccess) return RKS_ECUDA;
  ++s->nacc;
  return RKS_OK;
}

int rks_ws_get_grad(const rks_ws* s, float* grad) {
  if (!s || !grad) return RKS_EINVAL;
  if (cudaMemcpyAsync(grad, s->gacc, s->nparam * sizeof(float), cudaMemcpyDeviceToHost, s->st) != cudaSuccess ||
      cudaStreamSynchronize(s->st) != cudaSuccess)
    return RKS_ECUDA;
  return RKS_OK;
}

int rks_ws_zero_grad(rks_ws* s) {
  if (!s) return RKS_EINVAL;
  s->nacc = 0;
  if (cudaMemsetAsync(s->gacc, 0, s->nparam * sizeof(float), s->st) != cudaSuccess ||
      cudaStreamSynchronize(s->st) != cudaSuccess)
    return RKS_ECUDA;
  return RKS_OK;
}

int rks_ws_adam_step(rks_ws* s, float lr) {
  if (!s || !(lr > 0.f)) return RKS_EINVAL;
  if (s->nacc == 0) return RKS_ESTATE;
  ++s->adam_t;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - std::pow(b1, (float)s->adam_t), c2 = 1.f - std::pow(b2, (float)s->adam_t);
  k_adam<<<grid1(s->nparam), 256, 0, s->st>>>(s->nparam, s->theta, s->m, s->v, s->gacc, 1.f / (float)s->nacc, lr,
                                               b1, b2, c1, c2, 1e-8f);
  pack_weights(s);
  s->nacc = 0;
  if (launch_ok() != RKS_OK || cudaStreamSynchronize(s->st) != cudaSuccess) return RKS_ECUDA;
  return RKS_OK;
}

int rks_ws_start_vector(rks_ws* s, const float* x, double eps, uint64_t seed, double* u1) {
  if (!s || !x || !u1 || !(eps >= 0.0)) return RKS_EINVAL;
  const int64_t n0 = (int64_t)s->H * s->W;
  forward(s, x);
  rks::launch_start_vector(n0, seed, u1, s->st);   // g: N(0,1) from SplitMix64(seed), Box-Muller
  k_two_norms<<<kLossCtas, 256, 0, s->st>>>(n0, s->u, u1, s->lpart);
  if (launch_ok() != RKS_OK) return RKS_ECUDA;
  std::vector<double> part((size_t)kLossCtas * 2);
  if (cudaMemcpyAsync(part.data(), s->lpart, part.size() * sizeof(double), cudaMemcpyDeviceToHost, s->st) !=
          cudaSuccess ||
      cudaStreamSynchronize(s->st) != cudaSuccess)
    return RKS_ECUDA;
  double uu = 0.0, gg = 0.0;
  for (int b = 0; b < kLossCtas; ++b) { uu += part[2 * b]; gg += part[2 * b + 1]; }
  if (!(uu > 0.0) || !std::isfinite(uu) || !(gg > 0.0)) return RKS_ENAN;
  k_combine<<<grid1(n0), 256, 0, s->st>>>(n0, s->u, 1.0 / std::sqrt(uu), eps / std::sqrt(gg), u1);
  if (launch_ok() != RKS_OK || cudaStreamSynchronize(s->st) != cudaSuccess) return RKS_ECUDA;
  return RKS_OK;
}

void rks_ws_destroy(rks_ws* s) { delete s; }

}  // extern "C"
