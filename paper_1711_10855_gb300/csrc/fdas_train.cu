// fdas_train.cu -- the z-band network on windows, FP32 on the CUDA cores: forward (training and
// windowed inference), backward and Adam (the network itself is described in fdas_zband.cu).
//
// Only what the loss depends on is computed.  The pooled maximum runs over the central half of a
// window, so layer 3 is needed at n3 = W/2 positions, layer 2 at n2 = W/2 + 128 (its taps reach
// +-64) and layer 1 at n1 = W/2 + 160 (+-16 more); the activations are stored compactly at those
// positions.  The pooled gradient is one value per (window, channel), so layer 3's backward is a
// gather (weights) and a scatter (data) of those values.  At 256 windows of 1024 bins that leaves
// 5.8e9 multiply-adds of the 1.4e10 that every position in every layer would take.
//
// The convolutions are register-tiled: a thread owns 4 channels x 16 positions, the positions in
// four chunks of 4 spaced by the dilation D, so tap k of chunk c is chunk c + k and each 16-byte
// input load feeds up to 64 FMAs (one load per FMA without the tile: 8 times slower, bound by
// shared memory).  Rows are padded by one 16-byte chunk in five, which spreads a quarter-warp's
// loads over all banks for D = 4 and D = 16.  The next stage's operands are copied asynchronously while one
// is computed: with one buffer a fifth to a quarter of the warps' time went to waiting for them.
//
// A step on 256 windows of 1024 (Z = 201) takes 316 us, of which the four convolutions are about 260 at
// 60-65% of the FP32 pipe; with every position in every layer, dense gradients and untiled loops it
// took 3.46 ms.
//
// Every reduction has a fixed shape, which no device property enters, so one seed gives one network.
#include <cuda_fp16.h>
#include <cuda_pipeline.h>
#include <cuda_runtime.h>

#include "fdas_device.cuh"
#include "fdas_internal.h"

namespace fdas {
namespace {

constexpr int kC = kNetC, kK = kNetK;
constexpr int kTile = 128;               // positions per conv CTA
constexpr int kConvThreads = 64;         // 8 position threads x 8 channel groups of 4
constexpr int kStage = 8;                // input channels staged at a time (two stages in shared memory)
constexpr int kWgThreads = 256;          // layer-2 weight gradient: lane = input channel, warp = 4 output channels
constexpr int kWgUnit = 32;              // positions per unit of its work split
constexpr int kWgHalo = 32;              // 8 taps x dilation 4
constexpr int kWgPitch = kTile + kWgHalo + 4;   // floats; an odd number of 16-byte chunks
constexpr int kWgBuffer = kC * (kWgPitch + kTile);
// CTAs (and partial sums) of that gradient, at most: two for each of a GB300's 152 SMs, and as many on a device with
// another count, so that the sums' order and with it a training run's bits do not depend on the device.
constexpr int kWgCtas = 304;
// The splits below were chosen on 256 windows of 1024 and hold for any size: longer batches lengthen their chains
// of loads in proportion, as they do the convolutions, which stay most of a step (1024 windows: 1.09 ms, 256: 0.317).
constexpr int kScatter = 640;            // positions of the layer-2 gradient built at a time
constexpr int kL3Chunks = 32;            // window ranges of the layer-3 weight gradient
constexpr int kHeadChunks = 4;           // window ranges of the head's gradient
constexpr int kW1Chunks = 32;            // tile ranges layer 1's partials are summed over first
constexpr int kL3Part = kC * kC * kK + kC;
constexpr int kW1Part = kC * kK + kC;

__device__ __forceinline__ int padded(int pos) { return pos + (pos >> 4) * 4; }

// Adds 9 taps of one input channel to acc[chunk][element][channel]: x0 = the thread's first chunk,
// STEP floats between successive chunks (padding included where it is regular), w = 9 x 32 weights.
// Channels are paired (packed FP32x2): an FMA instruction then reads three register pairs in two cycles, where
// scalar FMAs with three different registers issue at about 60%.
template <int D>
__device__ __forceinline__ void conv_channel(float2 (&acc)[4][4][2], const float* __restrict__ x0,
                                             const float* __restrict__ w, int og) {
  float4 wk[kK];
#pragma unroll
  for (int k = 0; k < kK; ++k) wk[k] = *reinterpret_cast<const float4*>(w + k * kC + 4 * og);
#pragma unroll
  for (int j = 0; j < 12; ++j) {
    // chunk j is j*D positions further: 4j + 4(j/4) floats for D = 4 (the thread starts on a multiple
    // of 16), 20j for D = 16
    const float4 x = *reinterpret_cast<const float4*>(x0 + (D == 4 ? 4 * j + 4 * (j / 4) : 20 * j));
    const float2 xe[4] = {bc(x.x), bc(x.y), bc(x.z), bc(x.w)};
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int k = j - c;
      if (k < 0 || k >= kK) continue;
      const float2 w01 = make_float2(wk[k].x, wk[k].y), w23 = make_float2(wk[k].z, wk[k].w);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        acc[c][e][0] = fma2(w01, xe[e], acc[c][e][0]);
        acc[c][e][1] = fma2(w23, xe[e], acc[c][e][1]);
      }
    }
  }
}

enum { kConvL2 = 0, kConvL3 = 1, kConvBwd2 = 2 };

struct ConvArgs {
  const float* x;        // windows [B][W]
  const float* in;       // L3: h2, Bwd2: d2 ([B][32][W] rows, n2 used)
  const float* w;        // packed weights [32][9][32]
  const float* bias;     // L2, L3
  const float* w1;       // L2: layer-1 weights [32][9] and bias
  const float* b1;
  float* h1;             // L2 writes, Bwd2 reads its sign
  float* h2;             // L2 writes
  float* pool;           // L3: per (window, tile, channel) maximum
  int* arg;              // L3: its position (first on ties), 0 .. n3-1
  float* part1;          // Bwd2: per (window, tile): dW1 [32][9], db1 [32]
  int W;
};

// MODE kConvL2: h1 = relu(conv(x)) while staging, h2 = relu(conv_4(h1)).
// MODE kConvL3: conv_16(h2), its maximum over the tile per channel.
// MODE kConvBwd2: d1 = (h1 > 0) conv_4^T(d2), reduced at once to layer 1's weight gradient.
// Grid (tiles, windows).
template <int MODE>
__global__ void __launch_bounds__(kConvThreads) net_conv_kernel(const ConvArgs a) {
  constexpr int D = MODE == kConvL3 ? 16 : 4;
  constexpr int S = kTile + 8 * D;         // staged positions
  constexpr int SP = S / 4 * 5;            // padded row
  constexpr int XS = MODE == kConvL2 ? S + 8 : (MODE == kConvBwd2 ? kTile + 8 : 4);   // staged x
  __shared__ __align__(16) float sIn[2][kStage * SP];
  __shared__ __align__(16) float sW[2][kStage * kK * kC];
  __shared__ __align__(16) float sX[XS];
  __shared__ float sW1[kC * (kK + 1)];

  const int tid = threadIdx.x, pt = tid & 7, og = tid >> 3;
  const int b = blockIdx.y, p0 = blockIdx.x * kTile, W = a.W;
  const int n3 = W / 2, n2 = n3 + 128, n1 = n3 + 160;
  const size_t rows = (size_t)b * kC * W;
  // thread's first position within the tile and the float index of its first chunk
  const int pos0 = D == 4 ? 16 * pt : 64 * (pt >> 2) + 4 * (pt & 3);
  const int x0 = padded(pos0);

  if constexpr (MODE != kConvL3) {
    // x[u] = window position W/4 - 84 + p0 + u: taps of layer-1 position p0 + u - k (compact)
    const float* xw = a.x + (size_t)b * W + (W / 4 - 84);
    const int lim = n1 + 8 - p0;
    for (int u = tid; u < XS; u += kConvThreads) sX[u] = u < lim ? xw[p0 + u] : 0.f;
  }
  if constexpr (MODE == kConvL2) {
    for (int i = tid; i < kC * kK; i += kConvThreads) sW1[i] = a.w1[i];
    for (int i = tid; i < kC; i += kConvThreads) sW1[kC * kK + i] = a.b1[i];
  }

  float2 acc[4][4][2];   // [chunk][element][channel pair]
#pragma unroll
  for (int o = 0; o < 2; ++o) {
    const float2 v = MODE == kConvBwd2 ? bc(0.f) : make_float2(a.bias[4 * og + 2 * o], a.bias[4 * og + 2 * o + 1]);
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[c][e][o] = v;
  }
  auto at = [&](int c, int e, int o) { return o & 1 ? acc[c][e][o >> 1].y : acc[c][e][o >> 1].x; };

  // stage st's weights and (layers 3, 2 backward) input channels into buffer st & 1
  auto fetch = [&](int st) {
    const int c0 = st * kStage;
    const float* w = a.w + c0 * kK * kC;
    for (int i = tid; i < kStage * kK * kC / 4; i += kConvThreads)
      __pipeline_memcpy_async(sW[st & 1] + 4 * i, w + 4 * i, 16);
    if constexpr (MODE != kConvL2) {
      for (int i = tid; i < kStage * (S / 4); i += kConvThreads) {
        const int ch = i / (S / 4), u = 4 * (i - ch * (S / 4));
        const int t = MODE == kConvL3 ? p0 + u : p0 - 32 + u;   // a compact layer-2 position
        const bool in = t >= 0 && t < n2;
        const float* row = a.in + rows + (size_t)(c0 + ch) * W;
        __pipeline_memcpy_async(sIn[st & 1] + ch * SP + padded(u), row + (in ? t : 0), 16, in ? 0 : 16);
      }
    }
    __pipeline_commit();
  };
  constexpr int kStages = kC / kStage;
  fetch(0);
  __syncthreads();   // x and the layer-1 weights
#pragma unroll 1
  for (int st = 0; st < kStages; ++st) {
    const int c0 = st * kStage;
    if (st + 1 < kStages) fetch(st + 1);
    if constexpr (MODE == kConvL2) {
      for (int i = tid; i < kStage * (S / 4); i += kConvThreads) {
        const int ch = i / (S / 4), u = 4 * (i - ch * (S / 4));
        const float* w1 = sW1 + (c0 + ch) * kK;
        float xv[12], r[4];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          const float4 t = *reinterpret_cast<const float4*>(sX + u + 4 * q);
          xv[4 * q] = t.x, xv[4 * q + 1] = t.y, xv[4 * q + 2] = t.z, xv[4 * q + 3] = t.w;
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) r[e] = sW1[kC * kK + c0 + ch];
#pragma unroll
        for (int k = 0; k < kK; ++k) {
          const float w = w1[k];
#pragma unroll
          for (int e = 0; e < 4; ++e) r[e] = fmaf(w, xv[e + k], r[e]);
        }
        const float4 v = make_float4(fmaxf(r[0], 0.f), fmaxf(r[1], 0.f), fmaxf(r[2], 0.f), fmaxf(r[3], 0.f));
        // the tile keeps its own positions; the last one also the halo beyond layer 2's
        if ((u < kTile || p0 + kTile >= n2) && p0 + u < n1)
          *reinterpret_cast<float4*>(a.h1 + rows + (size_t)(c0 + ch) * W + p0 + u) = v;
        *reinterpret_cast<float4*>(sIn[st & 1] + ch * SP + padded(u)) = v;
      }
    }
    if (st + 1 < kStages) __pipeline_wait_prior(1);
    else __pipeline_wait_prior(0);
    __syncthreads();
#pragma unroll 1
    for (int i = 0; i < kStage; ++i) conv_channel<D>(acc, sIn[st & 1] + i * SP + x0, sW[st & 1] + i * kK * kC, og);
    __syncthreads();   // the buffer is free for stage st + 2
  }

  if constexpr (MODE == kConvL2) {
#pragma unroll
    for (int o = 0; o < 4; ++o)
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int p = p0 + pos0 + D * c;
        if (p < n2)
          *reinterpret_cast<float4*>(a.h2 + rows + (size_t)(4 * og + o) * W + p) =
              make_float4(fmaxf(at(c, 0, o), 0.f), fmaxf(at(c, 1, o), 0.f), fmaxf(at(c, 2, o), 0.f),
                          fmaxf(at(c, 3, o), 0.f));
      }
  } else if constexpr (MODE == kConvL3) {
#pragma unroll
    for (int o = 0; o < 4; ++o) {
      float best = -1.f;
      int where = 0;
#pragma unroll
      for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int e = 0; e < 4; ++e) {   // increasing positions
          const int p = p0 + pos0 + D * c + e;
          const float v = fmaxf(at(c, e, o), 0.f);
          if (p < n3 && v > best) {
            best = v;
            where = p;
          }
        }
#pragma unroll
      for (int off = 4; off > 0; off >>= 1) {
        const float ov = __shfl_down_sync(0xffffffffu, best, off, 8);
        const int oa = __shfl_down_sync(0xffffffffu, where, off, 8);
        if (ov > best || (ov == best && oa < where)) {
          best = ov;
          where = oa;
        }
      }
      if (pt == 0) {
        const size_t at_out = ((size_t)b * gridDim.x + blockIdx.x) * kC + 4 * og + o;
        a.pool[at_out] = best;
        a.arg[at_out] = where;
      }
    }
  } else {
    // dW1[i][k] = sum_t d1[i][t] x[t + k - 4], db1[i] = sum_t d1[i][t] over the tile
    float xv[24];
#pragma unroll
    for (int q = 0; q < 6; ++q) {
      const float4 t = *reinterpret_cast<const float4*>(sX + pos0 + 4 * q);
      xv[4 * q] = t.x, xv[4 * q + 1] = t.y, xv[4 * q + 2] = t.z, xv[4 * q + 3] = t.w;
    }
    float* out = a.part1 + ((size_t)b * gridDim.x + blockIdx.x) * kW1Part;
#pragma unroll
    for (int o = 0; o < 4; ++o) {
      float g[kK + 1];
#pragma unroll
      for (int k = 0; k <= kK; ++k) g[k] = 0.f;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int p = p0 + pos0 + 4 * c;
        float4 h = make_float4(0.f, 0.f, 0.f, 0.f);
        if (p < n1) h = *reinterpret_cast<const float4*>(a.h1 + rows + (size_t)(4 * og + o) * W + p);
        const float he[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float d = he[e] > 0.f ? at(c, e, o) : 0.f;
#pragma unroll
          for (int k = 0; k < kK; ++k) g[k] = fmaf(d, xv[4 * c + e + k], g[k]);
          g[kK] += d;
        }
      }
#pragma unroll
      for (int k = 0; k <= kK; ++k) {
#pragma unroll
        for (int off = 4; off > 0; off >>= 1) g[k] += __shfl_down_sync(0xffffffffu, g[k], off, 8);
        if (pt == 0) out[k < kK ? (4 * og + o) * kK + k : kC * kK + 4 * og + o] = g[k];
      }
    }
  }
}

struct HeadArgs {
  const float* pool;     // [B][tiles][32]
  const int* pool_arg;
  int tiles;
  const float* Wl;       // [Z][32], bl [Z]
  const float* bl;
  float* logits;         // [B][Z]
  int Z, W;
  // training
  const float* target;   // [B][Z]
  const float* w3b;      // packed [o][k][i]
  const float* h2;
  float* pooled;         // [B][32]
  float* seed;           // [B][32]: gradient of the pooled maximum (0 where the maximum is 0)
  int* arg;              // [B][32]: its position
  float* dlog;           // [B][Z]
  float* loss_part;      // [B]
  float* d2;             // [B][32] rows, n2 used: gradient of layer 2's pre-activations
  float* db2_part;       // [B][32]
  float count;           // B*Z
};

// One CTA per window: pooled maxima, head; in training also the loss, the pooled gradient, layer 3's
// data gradient scattered to layer 2's positions, and layer 2's bias gradient.  It waits on memory, not
// on arithmetic: the head's weights are staged 256 rows at a time (coalesced, used twice), the scatter
// covers all positions of a 1024-bin window at once and loads a channel's nine taps together.
template <bool TRAIN>
__global__ void __launch_bounds__(256) net_head_kernel(const HeadArgs a) {
  __shared__ float sM[kC], sS[kC], sRed[8][kC], sLoss[256], sDl[256];
  __shared__ int sA[kC];
  extern __shared__ __align__(16) float dyn[];   // head weights [256][33]; TRAIN, later: gradient [32][kScatter + 1]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, b = blockIdx.x, Z = a.Z;
  if (tid < kC) {
    float best = -1.f;
    int at = 0;
#pragma unroll 4
    for (int t = 0; t < a.tiles; ++t) {   // increasing positions: the first maximum
      const size_t i = ((size_t)b * a.tiles + t) * kC + tid;
      const float v = a.pool[i];
      const int where = a.pool_arg[i];
      if (v > best) {
        best = v;
        at = where;
      }
    }
    sM[tid] = best;
    sA[tid] = at;
  }
  float loss = 0.f, dm = 0.f;   // dm: warp w's share (j = w, w + 8, ...) of channel `lane`
  for (int j0 = 0; j0 < Z; j0 += 256) {
    const int nj = Z - j0 < 256 ? Z - j0 : 256;
    __syncthreads();
#pragma unroll 8
    for (int i = tid; i < nj * kC / 4; i += 256) {
      const float4 v = reinterpret_cast<const float4*>(a.Wl + (size_t)j0 * kC)[i];   // 16-byte aligned (NetLayout)
      float* d = dyn + (i >> 3) * (kC + 1) + 4 * (i & 7);
      d[0] = v.x, d[1] = v.y, d[2] = v.z, d[3] = v.w;
    }
    __syncthreads();
    if (tid < nj) {
      const float* w = dyn + tid * (kC + 1);
      float s = a.bl[j0 + tid];
#pragma unroll
      for (int c = 0; c < kC; ++c) s = fmaf(w[c], sM[c], s);
      const size_t at = (size_t)b * Z + j0 + tid;
      a.logits[at] = s;
      if constexpr (TRAIN) {
        const float t = a.target[at];
        const float d = (1.f / (1.f + expf(-s)) - t) / a.count;
        a.dlog[at] = d;
        sDl[tid] = d;
        loss += fmaxf(s, 0.f) - s * t + log1pf(expf(-fabsf(s)));
      }
    }
    if constexpr (TRAIN) {
      __syncthreads();
      for (int j = warp; j < nj; j += 8) dm = fmaf(sDl[j], dyn[j * (kC + 1) + lane], dm);
    }
  }
  if constexpr (TRAIN) {
    sRed[warp][lane] = dm;
    sLoss[tid] = loss;
    __syncthreads();
    for (int s = 128; s > 0; s >>= 1) {
      if (tid < s) sLoss[tid] += sLoss[tid + s];
      __syncthreads();
    }
    if (tid < kC) {
      float s = 0.f;
#pragma unroll
      for (int w = 0; w < 8; ++w) s += sRed[w][tid];
      s = sM[tid] > 0.f ? s : 0.f;
      sS[tid] = s;
      a.pooled[(size_t)b * kC + tid] = sM[tid];
      a.seed[(size_t)b * kC + tid] = s;
      a.arg[(size_t)b * kC + tid] = sA[tid];
    }
    if (tid == 0) a.loss_part[b] = sLoss[0] / a.count;
    // layer 3's data gradient at compact layer-2 position t = arg + 16k: sum over (o, k) of W3[o][i][k]
    // seed[o].  Warp w adds the channels o whose arg is 2w or 2w + 1 mod 16, so no two warps meet.
    const int n2 = a.W / 2 + 128;
    float* col = dyn + lane * (kScatter + 1);
    float db[4] = {0.f, 0.f, 0.f, 0.f};
    for (int t0 = 0; t0 < n2; t0 += kScatter) {
      const int nt = n2 - t0 < kScatter ? n2 - t0 : kScatter;
      __syncthreads();
      for (int i = tid; i < kC * (kScatter + 1) / 4; i += 256) reinterpret_cast<float4*>(dyn)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      __syncthreads();
      // this warp's channels, the next one's weights loaded before the current one's are used
      unsigned mine = __ballot_sync(0xffffffffu, ((sA[lane] & 15) >> 1) == warp && sS[lane] != 0.f);
      float w[kK];
      auto load = [&](int o) {
#pragma unroll
        for (int k = 0; k < kK; ++k) w[k] = a.w3b[(o * kK + k) * kC + lane];
      };
      if (mine) load(__ffs(mine) - 1);
      while (mine) {
        const int o = __ffs(mine) - 1, p = sA[o];
        const float s = sS[o];
        mine &= mine - 1;
        float v[kK], wc[kK];
#pragma unroll
        for (int k = 0; k < kK; ++k) wc[k] = w[k];
        if (mine) load(__ffs(mine) - 1);
#pragma unroll
        for (int k = 0; k < kK; ++k) {   // nine different positions
          const int t = p + 16 * k - t0;
          v[k] = t >= 0 && t < nt ? col[t] : 0.f;
        }
#pragma unroll
        for (int k = 0; k < kK; ++k) {
          const int t = p + 16 * k - t0;
          if (t >= 0 && t < nt) col[t] = fmaf(wc[k], s, v[k]);
        }
      }
      __syncthreads();
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int ch = warp + 8 * r;
        const size_t row = ((size_t)b * kC + ch) * a.W + t0;
        const float* src = dyn + ch * (kScatter + 1);
#pragma unroll
        for (int i = 0; i < kScatter / 128; ++i) {
          const int t = 128 * i + 4 * lane;   // nt is a multiple of 4
          if (t >= nt) continue;
          const float4 h = *reinterpret_cast<const float4*>(a.h2 + row + t);
          const float4 v = make_float4(h.x > 0.f ? src[t] : 0.f, h.y > 0.f ? src[t + 1] : 0.f,
                                       h.z > 0.f ? src[t + 2] : 0.f, h.w > 0.f ? src[t + 3] : 0.f);
          *reinterpret_cast<float4*>(a.d2 + row + t) = v;
          db[r] += (v.x + v.y) + (v.z + v.w);
        }
      }
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) db[r] += __shfl_down_sync(0xffffffffu, db[r], off);
      if (lane == 0) a.db2_part[(size_t)b * kC + warp + 8 * r] = db[r];
    }
  }
}

struct WgArgs {
  const float* h1;
  const float* d2;
  float* part2;          // [CTAs][32][9][32]
  int B, W;
};

// Layer 2's weight gradient dW2[o][i][k] = sum over windows and layer-2 positions t of d2[o][t] h1[i][t + 4k]
// (compact positions).  The positions are cut into equal contiguous ranges of 32-position units, one
// per CTA; lane = i, warp = 4 output channels, 36 sums per thread in registers over the CTA's whole range.
__global__ void __launch_bounds__(kWgThreads, 2) net_wgrad2_kernel(const WgArgs a) {
  extern __shared__ __align__(16) float wg_smem[];   // two buffers of h1 rows, then gradient rows
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, W = a.W;
  const int n2 = W / 2 + 128, per = n2 / kWgUnit;
  const int64_t U = (int64_t)a.B * per;
  int64_t u = (int64_t)blockIdx.x * U / gridDim.x;
  const int64_t u1 = ((int64_t)blockIdx.x + 1) * U / gridDim.x;
  float2 acc[4][kK];   // sums over even and odd positions (packed FP32x2)
#pragma unroll
  for (int o = 0; o < 4; ++o)
#pragma unroll
    for (int k = 0; k < kK; ++k) acc[o][k] = bc(0.f);
  // the next run of units within one window: its first element and length (0: none left)
  auto take = [&](size_t& rows) -> int {
    if (u >= u1) return 0;
    const int64_t b = u / per;
    const int q = (int)(u - b * per);
    int len = per - q;                                   // units to the end of the window
    if (len > kTile / kWgUnit) len = kTile / kWgUnit;
    if (len > u1 - u) len = (int)(u1 - u);
    u += len;
    rows = (size_t)b * kC * W + q * kWgUnit;
    return len * kWgUnit;
  };
  auto fetch = [&](int buf, size_t rows, int nt) {
    float* h = wg_smem + buf * kWgBuffer;
    float* d = h + kC * kWgPitch;
    const int hc = (nt + kWgHalo) / 4, dc = nt / 4;
    for (int i = tid; i < kC * hc; i += kWgThreads) {
      const int ch = i / hc, m = i - ch * hc;
      __pipeline_memcpy_async(h + ch * kWgPitch + 4 * m, a.h1 + rows + (size_t)ch * W + 4 * m, 16);
    }
    for (int i = tid; i < kC * dc; i += kWgThreads) {
      const int ch = i / dc, m = i - ch * dc;
      __pipeline_memcpy_async(d + ch * kTile + 4 * m, a.d2 + rows + (size_t)ch * W + 4 * m, 16);
    }
    __pipeline_commit();
  };
  size_t rows = 0;
  int nt = take(rows), buf = 0;
  if (nt) fetch(0, rows, nt);
  while (nt) {
    const int nt_next = take(rows);
    if (nt_next) {
      fetch(buf ^ 1, rows, nt_next);
      __pipeline_wait_prior(1);
    } else {
      __pipeline_wait_prior(0);
    }
    __syncthreads();
    const float* sH = wg_smem + buf * kWgBuffer;
    const float* sD = sH + kC * kWgPitch;
#pragma unroll 1
    for (int t = 0; t < nt; t += 8) {
      float4 d[4][2];
#pragma unroll
      for (int o = 0; o < 4; ++o)
#pragma unroll
        for (int c = 0; c < 2; ++c) d[o][c] = *reinterpret_cast<const float4*>(sD + (4 * warp + o) * kTile + t + 4 * c);
#pragma unroll
      for (int j = 0; j < 10; ++j) {
        const float4 h = *reinterpret_cast<const float4*>(sH + lane * kWgPitch + t + 4 * j);
        const float2 h01 = make_float2(h.x, h.y), h23 = make_float2(h.z, h.w);
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const int k = j - c;
          if (k < 0 || k >= kK) continue;
#pragma unroll
          for (int o = 0; o < 4; ++o) {
            acc[o][k] = fma2(make_float2(d[o][c].x, d[o][c].y), h01, acc[o][k]);
            acc[o][k] = fma2(make_float2(d[o][c].z, d[o][c].w), h23, acc[o][k]);
          }
        }
      }
    }
    __syncthreads();   // the buffer is free
    nt = nt_next;
    buf ^= 1;
  }
  float* out = a.part2 + (size_t)blockIdx.x * (kC * kC * kK);
#pragma unroll
  for (int o = 0; o < 4; ++o)
#pragma unroll
    for (int k = 0; k < kK; ++k) out[((4 * warp + o) * kK + k) * kC + lane] = acc[o][k].x + acc[o][k].y;
}

struct SparseArgs {
  const float* h2;
  const float* seed;
  const int* arg;
  const float* pooled;
  const float* dlog;
  const float* part1;    // [tiles1][kW1Part]
  float* sum1;           // [kW1Chunks][kW1Part]
  float* part3;          // [kL3Chunks][32][9][32] then [32]
  float* gl;             // [kHeadChunks] of dWl [Z][32], dbl [Z]
  int B, W, Z, tiles1;
};

// The small gradients, 288 threads a block: layer 3's weights from the pooled values (blocks o + 32 *
// chunk of windows), a first sum of layer 1's partials (kW1Chunks blocks), and the head's (8 outputs
// and a range of windows each).  All are chains of loads, so the ranges are short.
__global__ void __launch_bounds__(288) net_sparse_grad_kernel(const SparseArgs a) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int blk = blockIdx.x;
  if (blk < kC * kL3Chunks) {
    const int o = blk % kC, chunk = blk / kC;
    const int b0 = (int)((int64_t)chunk * a.B / kL3Chunks), b1 = (int)((int64_t)(chunk + 1) * a.B / kL3Chunks);
    float s = 0.f, sb = 0.f;   // warp = tap, lane = input channel
#pragma unroll 8
    for (int b = b0; b < b1; ++b) {
      const float g = a.seed[(size_t)b * kC + o];
      const int p = a.arg[(size_t)b * kC + o];
      s = fmaf(g, a.h2[((size_t)b * kC + lane) * a.W + p + 16 * warp], s);
      sb += g;
    }
    float* out = a.part3 + (size_t)chunk * kL3Part;
    out[(o * kK + warp) * kC + lane] = s;
    if (tid == 0) out[kC * kC * kK + o] = sb;
    return;
  }
  blk -= kC * kL3Chunks;
  if (blk < kW1Chunks) {
    const int t0 = (int)((int64_t)blk * a.tiles1 / kW1Chunks), t1 = (int)((int64_t)(blk + 1) * a.tiles1 / kW1Chunks);
    for (int e = tid; e < kW1Part; e += 288) {
      float s = 0.f;
#pragma unroll 16
      for (int t = t0; t < t1; ++t) s += a.part1[(size_t)t * kW1Part + e];
      a.sum1[(size_t)blk * kW1Part + e] = s;
    }
    return;
  }
  blk -= kW1Chunks;
  // dWl[j][c] = sum_b dlog[b][j] m[b][c], dbl[j] = sum_b dlog[b][j]
  const int chunk = blk % kHeadChunks, j = blk / kHeadChunks * 8 + tid / (kC + 1), c = tid % (kC + 1);
  if (tid >= 8 * (kC + 1) || j >= a.Z) return;
  const int b0 = (int)((int64_t)chunk * a.B / kHeadChunks), b1 = (int)((int64_t)(chunk + 1) * a.B / kHeadChunks);
  float s = 0.f;
#pragma unroll 16
  for (int b = b0; b < b1; ++b) {
    const float m = c < kC ? a.pooled[(size_t)b * kC + c] : 1.f;
    s = fmaf(a.dlog[(size_t)b * a.Z + j], m, s);
  }
  a.gl[(size_t)chunk * a.Z * (kC + 1) + (c < kC ? (size_t)j * kC + c : (size_t)a.Z * kC + j)] = s;
}

// Where a parameter's copies go (net layout: NetLayout in fdas_internal.h).
struct Copies {
  __half* ph;            // FP16 copy
  float* pr;             // its values as FP32
  __half* stack;         // layers 2 and 3 in the inference kernel's order
  float* packs;          // kNetPacks packed weight matrices
  int W2, W3;            // offsets of the two layers' weights in the parameter vector
};

__device__ __forceinline__ void publish(const Copies& c, int idx, float v) {
  const __half hv = __float2half_rn(v);
  const float r = __half2float(hv);
  c.ph[idx] = hv;
  c.pr[idx] = r;
  constexpr int n = kC * kC * kK;
  const bool l2 = idx >= c.W2 && idx < c.W2 + n, l3 = idx >= c.W3 && idx < c.W3 + n;
  if (!l2 && !l3) return;
  const int e = idx - (l2 ? c.W2 : c.W3), o = e / (kC * kK), i = e / kK % kC, k = e % kK;
  const int fwd = (i * kK + k) * kC + o;
  c.stack[stack_at(l3 ? 1 : 0, o, i, k)] = hv;
  c.packs[(l2 ? kPackW2 : kPackW3) * n + fwd] = v;
  c.packs[(l2 ? kPackW2Half : kPackW3Half) * n + fwd] = r;
  // layer 2's data gradient is a convolution with the taps reversed; layer 3's is scattered tap by tap
  if (l2) c.packs[kPackW2Back * n + (o * kK + kK - 1 - k) * kC + i] = v;
  else c.packs[kPackW3Back * n + (o * kK + k) * kC + i] = v;
}

__global__ void net_publish_kernel(const float* p, Copies c, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) publish(c, i, p[i]);
}

struct AdamArgs {
  struct Segment {
    const float* part;   // partial p of entry e: part[p * stride + e]
    int stride, parts, n, at, block0;   // `at`: first parameter; block0: first CTA
    bool oki;            // entries ordered (o, k, i) instead of the parameters' (o, i, k)
  } seg[8];
  float *p, *g, *m, *v;
  Copies copies;
  float lr, b1, b2, eps, c1, c2;
  const float* loss_part;
  int B;
  float* loss;
};

// Sums of the gradient partials (32 entries per CTA, 8 threads each, fixed order) and the Adam update
// of those parameters; the last CTA sums the loss.
__global__ void __launch_bounds__(256) net_adam_kernel(const AdamArgs a) {
  __shared__ float s[8][32];
  const int tid = threadIdx.x, lane = tid & 31, grp = tid >> 5, blk = blockIdx.x;
  if (blk == gridDim.x - 1) {
    float t = 0.f;
    for (int b = tid; b < a.B; b += 256) t += a.loss_part[b];
    s[grp][lane] = t;
    __syncthreads();
    if (tid == 0) {
      float sum = 0.f;
      for (int i = 0; i < 256; ++i) sum += s[i >> 5][i & 31];
      *a.loss = sum;
    }
    return;
  }
  int k = 0;
#pragma unroll
  for (int i = 1; i < 8; ++i)
    if (blk >= a.seg[i].block0) k = i;
  const auto& q = a.seg[k];
  const int e = (blk - q.block0) * 32 + lane;
  float t = 0.f;
  if (e < q.n) {
#pragma unroll 8
    for (int p = grp; p < q.parts; p += 8) t += q.part[(size_t)p * q.stride + e];
  }
  s[grp][lane] = t;
  __syncthreads();
  if (grp != 0 || e >= q.n) return;
  float gi = s[0][lane];
  const int used = q.parts < 8 ? q.parts : 8;
  for (int i = 1; i < used; ++i) gi += s[i][lane];
  int idx = q.at + e;
  if (q.oki) idx = q.at + (e / (kC * kK) * kC + e % kC) * kK + e / kC % kK;
  const float mi = a.b1 * a.m[idx] + (1.f - a.b1) * gi;
  const float vi = a.b2 * a.v[idx] + (1.f - a.b2) * gi * gi;
  const float pi = a.p[idx] - a.lr * (mi / a.c1) / (sqrtf(vi / a.c2) + a.eps);
  a.g[idx] = gi;
  a.m[idx] = mi;
  a.v[idx] = vi;
  a.p[idx] = pi;
  publish(a.copies, idx, pi);
}

int tiles_of(int n) { return (n + kTile - 1) / kTile; }
int wg_ctas(const NetState& s, int B) {
  const int64_t units = (int64_t)B * ((s.W / 2 + 128) / kWgUnit);
  return (int)(units < kWgCtas ? units : kWgCtas);
}
Copies copies_of(const NetState& s) { return Copies{s.ph, s.pr, s.stack, s.packs, s.lay.W2, s.lay.W3}; }

constexpr size_t kHeadTrainSmem = sizeof(float) * kC * (kScatter + 1);
constexpr size_t kHeadSmem = sizeof(float) * 256 * (kC + 1);
constexpr size_t kWgSmem = sizeof(float) * 2 * kWgBuffer;
static_assert(kHeadSmem <= kHeadTrainSmem, "the head's weights share the gradient's space");

void launch_forward(const NetState& s, const float* windows, int B, const float* params, int pack2, int pack3,
                    cudaStream_t st) {
  constexpr int n = kC * kC * kK;
  ConvArgs c{};
  c.x = windows;
  c.w = s.packs + pack2 * n;
  c.bias = params + s.lay.b2;
  c.w1 = params + s.lay.W1;
  c.b1 = params + s.lay.b1;
  c.h1 = s.h1;
  c.h2 = s.h2;
  c.W = s.W;
  net_conv_kernel<kConvL2><<<dim3(tiles_of(s.W / 2 + 128), B), kConvThreads, 0, st>>>(c);
  c.in = s.h2;
  c.w = s.packs + pack3 * n;
  c.bias = params + s.lay.b3;
  c.pool = s.pool;
  c.arg = s.pool_arg;
  net_conv_kernel<kConvL3><<<dim3(tiles_of(s.W / 2), B), kConvThreads, 0, st>>>(c);
}

HeadArgs head_args(const NetState& s, const float* params, float* logits) {
  HeadArgs h{};
  h.pool = s.pool;
  h.pool_arg = s.pool_arg;
  h.tiles = tiles_of(s.W / 2);
  h.Wl = params + s.lay.Wl;
  h.bl = params + s.lay.bl;
  h.logits = logits;
  h.Z = s.lay.Z;
  h.W = s.W;
  return h;
}

}  // namespace

NetSizes net_sizes(int W, int Z, int max_batch) {
  NetSizes z;
  const size_t B = (size_t)max_batch;
  z.act = B * kC * (size_t)W;
  z.pool = B * tiles_of(W / 2) * kC;
  z.part1 = B * tiles_of(W / 2 + 160) * kW1Part;
  z.part2 = (size_t)kWgCtas * kC * kC * kK;
  z.part3 = (size_t)kL3Chunks * kL3Part;
  z.sum1 = (size_t)kW1Chunks * kW1Part;
  z.gl = (size_t)kHeadChunks * Z * (kC + 1);
  z.packs = (size_t)kNetPacks * kC * kC * kK;
  return z;
}

cudaError_t net_prepare() {
  const cudaError_t e =
      cudaFuncSetAttribute(net_wgrad2_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWgSmem);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(net_head_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kHeadTrainSmem);
}

void net_publish(const NetState& s, cudaStream_t st) {
  net_publish_kernel<<<(s.lay.total + 255) / 256, 256, 0, st>>>(s.p, copies_of(s), s.lay.total);
}

cudaError_t net_predict(const NetState& s, const float* windows, int B, bool half_weights, float* logits,
                        cudaStream_t st) {
  const float* params = half_weights ? s.pr : s.p;
  launch_forward(s, windows, B, params, half_weights ? kPackW2Half : kPackW2, half_weights ? kPackW3Half : kPackW3, st);
  net_head_kernel<false><<<B, 256, kHeadSmem, st>>>(head_args(s, params, logits));
  return cudaGetLastError();
}

cudaError_t net_train_step(const NetState& s, const float* windows, const float* targets, int B, float lr, int step,
                           cudaStream_t st) {
  constexpr int n = kC * kC * kK;
  const int Z = s.lay.Z, W = s.W;
  launch_forward(s, windows, B, s.p, kPackW2, kPackW3, st);
  HeadArgs h = head_args(s, s.p, s.logits);
  h.target = targets;
  h.w3b = s.packs + kPackW3Back * n;
  h.h2 = s.h2;
  h.pooled = s.pooled;
  h.seed = s.seed;
  h.arg = s.arg;
  h.dlog = s.dlog;
  h.loss_part = s.loss_part;
  h.d2 = s.d2;
  h.db2_part = s.db2_part;
  h.count = (float)((int64_t)B * Z);
  net_head_kernel<true><<<B, 256, kHeadTrainSmem, st>>>(h);

  ConvArgs c{};
  c.x = windows;
  c.in = s.d2;
  c.w = s.packs + kPackW2Back * n;
  c.h1 = s.h1;
  c.part1 = s.part1;
  c.W = W;
  const int tiles1 = tiles_of(W / 2 + 160);
  net_conv_kernel<kConvBwd2><<<dim3(tiles1, B), kConvThreads, 0, st>>>(c);
  const int wg = wg_ctas(s, B);
  net_wgrad2_kernel<<<wg, kWgThreads, kWgSmem, st>>>(WgArgs{s.h1, s.d2, s.part2, B, W});
  net_sparse_grad_kernel<<<kC * kL3Chunks + kW1Chunks + kHeadChunks * ((Z + 7) / 8), 288, 0, st>>>(
      SparseArgs{s.h2, s.seed, s.arg, s.pooled, s.dlog, s.part1, s.sum1, s.part3, s.gl, B, W, Z, B * tiles1});

  AdamArgs a{};
  int blk = 0, k = 0;
  auto seg = [&](const float* part, int stride, int parts, int count, int at, bool oki) {
    a.seg[k++] = {part, stride, parts, count, at, blk, oki};
    blk += (count + 31) / 32;
  };
  seg(s.sum1, kW1Part, kW1Chunks, kC * kK, s.lay.W1, false);
  seg(s.sum1 + kC * kK, kW1Part, kW1Chunks, kC, s.lay.b1, false);
  seg(s.part2, n, wg, n, s.lay.W2, true);
  seg(s.db2_part, kC, B, kC, s.lay.b2, false);
  seg(s.part3, kL3Part, kL3Chunks, n, s.lay.W3, true);
  seg(s.part3 + n, kL3Part, kL3Chunks, kC, s.lay.b3, false);
  seg(s.gl, Z * (kC + 1), kHeadChunks, Z * kC, s.lay.Wl, false);
  seg(s.gl + Z * kC, Z * (kC + 1), kHeadChunks, Z, s.lay.bl, false);
  a.p = s.p;
  a.g = s.g;
  a.m = s.m;
  a.v = s.v;
  a.copies = copies_of(s);
  a.lr = lr;
  a.b1 = 0.9f;
  a.b2 = 0.999f;
  a.eps = 1e-8f;
  a.c1 = 1.f - powf(a.b1, (float)step);
  a.c2 = 1.f - powf(a.b2, (float)step);
  a.loss_part = s.loss_part;
  a.B = B;
  a.loss = s.loss;
  net_adam_kernel<<<blk + 1, 256, 0, st>>>(a);
  return cudaGetLastError();
}

}  // namespace fdas
