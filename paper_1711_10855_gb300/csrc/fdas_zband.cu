// fdas_zband.cu -- the learned z-band proposal (declared in include/fdas.h): a 1-D convolutional
// network over the z = 0 power spectrum that predicts which templates of the z grid are worth
// correlating near each block of bins, with hand-written training (FP32 forward, backward,
// Adam) and inference (a fused tcgen05 kernel: FP16 weights and activations, FP32
// accumulation), and the conversion of its proposals into a work list for the correlation
// kernel.  The paper has no counterpart; the full search stays the reference against which
// recall is measured.
//
// Network (window width Wd, hop Wd/2, C = 32 channels, k = 9, dilations 1, 4, 16, zero padding
// 4 x dilation):
//   x_r = min(|A_r|^2 ln 2 / median |A|^2, 64)   (one scale for the whole spectrum)
//   window w = x over bins [w*hop - Wd/4, w*hop + 3Wd/4), 0 outside [0, n)
//   a1 = conv_1(x; W1, b1), a2 = conv_4(relu(a1); W2, b2), a3 = conv_16(relu(a2); W3, b3)
//     conv_d(in; W, b)[o][t] = b[o] + sum_{i,k} W[o][i][k] in[i][t + (k - 4) d]
//   m[c] = max over t in [Wd/4, 3Wd/4) of relu(a3[c][t]),   logits = Wl m + bl  (Z outputs)
//   loss = mean BCE-with-logits(logits, target)
// The central positions' receptive field (+-84 = 4 (1 + 4 + 16)) stays inside the window
// (Wd >= 4 x 84), so the logits of window w are those of the layers run once over the
// zero-extended x and max-pooled over the block [w*hop, (w+1)*hop): the inference kernel
// computes that form, without the overlap.
#include <cmath>
#include <cstring>
#include <new>
#include <type_traits>

#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "fdas.h"
#include "fdas_internal.h"
#include "fdas_umma.cuh"

namespace {

using Layout = fdas::NetLayout;
constexpr int kC = fdas::kNetC;   // channels
constexpr int kK = fdas::kNetK;   // kernel taps
constexpr int kPad = 4;
constexpr int kWidthStep = 128;   // window widths are multiples of it
constexpr int kDil1 = 1, kDil2 = 4, kDil3 = 16;    // layer dilations
constexpr int kRF = kPad * (kDil1 + kDil2 + kDil3);   // receptive field of a layer-3 position

constexpr float kXCap = 64.f;   // input cap: x_r = min(|A_r|^2 ln 2 / median |A|^2, 64)
constexpr int kSelBlocks0 = 456;   // grid caps of the median's passes: 3 blocks of the first fit an SM of a GB300,
constexpr int kSelBlocks = 304;    // and the later ones flush their bins once per block

// Exact lower median of |A_r|^2 (rank (n-1)/2) by radix selection on the FP32 bit patterns
// (non-negative floats order as unsigned integers; the sign bit is 0): three passes over the spectrum
// histogram 8 bits (the exponent: most values share a few bins, so each thread counts into bytes of
// its own), then 10 bits of the values that match the digit found so far (a third of them, spread
// over every bin: few bins keep the blocks' flush short), then the last 13.  The block of a pass that finishes last
// finds the digit holding the rank; the last pass leaves scale = ln 2 / median.  The state is cleared
// before the first pass.
constexpr int kSelBins0 = 256, kSelBins1 = 1024, kSelBins2 = 8192;
constexpr int kSelPer = 8;   // complex values per thread and pass iteration (four 16-byte loads)
struct SelectState {
  long long k;                 // rank of the median among the values matching `prefix`
  unsigned prefix, done;       // bits fixed so far; blocks of the current pass that have finished
  unsigned hist0[kSelBins0];   // bits 30..23
  unsigned hist1[kSelBins1];   // bits 22..13 of the values matching digit 0
  unsigned hist2[kSelBins2];   // bits 12..0 of the values matching digits 0 and 1
};

__device__ __forceinline__ float power_of(const float2 a) { return fmaf(a.x, a.x, a.y * a.y); }

// PASS 0: bits 30..23 of every value, one byte per thread and bin (the four warps w, w + 1, ... of a
// 128-byte row of lanes use one byte of each word: no conflicts, no atomics), summed per block before a
// byte can overflow; PASS 1, 2: the next bits of the values whose higher bits equal st->prefix, by
// shared atomics.  Values are read in 16-byte pairs from the first 16-byte boundary (an 8-byte aligned
// spectrum's first value is counted on its own); the tail element by element.
template <int PASS>
__host__ __device__ constexpr size_t select_smem() {
  return PASS == 0 ? 256 * kSelBins0 : sizeof(unsigned) * (PASS == 1 ? kSelBins1 : kSelBins2);
}

template <int PASS>
__global__ void __launch_bounds__(256) select_pass_kernel(const float2* spec, int64_t n, SelectState* st,
                                                          float* scale) {
  constexpr int NB = PASS == 0 ? kSelBins0 : (PASS == 1 ? kSelBins1 : kSelBins2);
  constexpr int SHIFT = PASS == 0 ? 23 : (PASS == 1 ? 13 : 0);
  constexpr unsigned MASK = PASS == 0 ? 0u : (PASS == 1 ? 0xFF800000u : 0xFFFFE000u);
  extern __shared__ __align__(16) unsigned char sel_smem[];
  unsigned* h = reinterpret_cast<unsigned*>(sel_smem);
  __shared__ bool last;
  const int64_t total = n;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned char* mine = sel_smem + (warp >> 2) * 128 + lane * 4 + (warp & 3);   // + 256 * bin
  for (int i = threadIdx.x; i < (int)(select_smem<PASS>() / 16); i += 256)
    reinterpret_cast<uint4*>(sel_smem)[i] = make_uint4(0u, 0u, 0u, 0u);
  const unsigned prefix = PASS == 0 ? 0u : st->prefix;
  unsigned* hist = PASS == 0 ? st->hist0 : (PASS == 1 ? st->hist1 : st->hist2);
  __syncthreads();
  auto count = [&](float2 a, bool valid) {
    const unsigned bits = __float_as_uint(power_of(a)) & 0x7FFFFFFFu;
    const unsigned bucket = (bits >> SHIFT) & (unsigned)(NB - 1);
    if constexpr (PASS == 0) {
      if (valid) mine[256 * bucket] = (unsigned char)(mine[256 * bucket] + 1);
    } else {
      if (valid && (bits & MASK) == prefix) atomicAdd(&h[bucket], 1u);
    }
  };
  // PASS 0: the block's bytes of bin threadIdx.x added to the histogram and cleared (between barriers);
  // threads start at different words of their rows
  auto flush_bytes = [&]() {
    __syncthreads();
    unsigned c = 0u;
    unsigned* row = h + 64 * threadIdx.x;
    for (int i = 0; i < 64; ++i) {
      const unsigned w = row[(i + lane) & 63];
      row[(i + lane) & 63] = 0u;
      c += (w & 0xFFu) + ((w >> 8) & 0xFFu) + ((w >> 16) & 0xFFu) + (w >> 24);
    }
    if (c) atomicAdd(&hist[threadIdx.x], c);
    __syncthreads();
  };
  const int off = (reinterpret_cast<uintptr_t>(spec) & 15u) ? 1 : 0;
  if (off && blockIdx.x == 0 && threadIdx.x == 0 && n > 0) count(__ldg(spec), true);
  spec += off;
  n -= off;
  const int64_t step = (int64_t)gridDim.x * 256 * kSelPer;
  int held = 0;   // PASS 0: values counted since the last flush, per thread
  for (int64_t base = (int64_t)blockIdx.x * 256 * kSelPer; base < n; base += step) {
    if constexpr (PASS == 0) {
      if (held + kSelPer + 1 > 255) {   // uniform over the block
        flush_bytes();
        held = 0;
      }
      held += kSelPer;
    }
    // thread t reads the pairs (base + 2(t + 256 j), +1), j < kSelPer / 2: coalesced 16-byte loads
    float4 v[kSelPer / 2];
#pragma unroll
    for (int j = 0; j < kSelPer / 2; ++j) {
      const int64_t r = base + 2 * ((int64_t)threadIdx.x + 256 * j);
      v[j] = r + 1 < n ? __ldg(reinterpret_cast<const float4*>(spec + r))
                       : make_float4(r < n ? spec[r].x : 0.f, r < n ? spec[r].y : 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int j = 0; j < kSelPer / 2; ++j) {
      const int64_t r = base + 2 * ((int64_t)threadIdx.x + 256 * j);
      count(make_float2(v[j].x, v[j].y), r < n);
      count(make_float2(v[j].z, v[j].w), r + 1 < n);
    }
  }
  if constexpr (PASS == 0) {
    flush_bytes();
  } else {
    __syncthreads();
    for (int i = threadIdx.x; i < NB; i += 256)
      if (h[i]) atomicAdd(&hist[i], h[i]);
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(&st->done, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  // The last block: the digit of the histogram that holds rank st->k (thread t owns NB/256 bins; a block
  // scan of their sums leaves exactly one thread whose range holds the rank), appended to st->prefix.
  __threadfence();
  constexpr int per = NB / 256;
  __shared__ long long wsum[8];
  const int t = threadIdx.x, wid = t >> 5;
  // through shared memory: a thread's own bins straight from L2 are a line per lane and load (8192 bins that
  // way cost a proposal over 160,000 bins 4 us); threads start at different words of their bins
#pragma unroll
  for (int i = 0; i < per; ++i) h[t + 256 * i] = __ldcg(&hist[t + 256 * i]);
  __syncthreads();
  long long own = 0;
#pragma unroll
  for (int i = 0; i < per; ++i) own += h[t * per + ((i + lane) & (per - 1))];
  long long inc = own;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) wsum[wid] = inc;
  __syncthreads();
  long long excl = inc - own;
  for (int i = 0; i < wid; ++i) excl += wsum[i];
  const long long k = PASS == 0 ? (total - 1) / 2 : st->k;
  __syncthreads();   // st->k is read by every thread before one of them replaces it
  if (k >= excl && k < excl + own) {
    long long r = k - excl;
    int d = t * per;
#pragma unroll
    for (int i = 0; i < per - 1; ++i)
      if (d == t * per + i && r >= (long long)h[t * per + i]) {
        r -= h[t * per + i];
        ++d;
      }
    const unsigned found = prefix | ((unsigned)d << SHIFT);
    st->k = r;
    st->prefix = found;
    if (PASS == 2) {
      const float med = __uint_as_float(found);
      *scale = med > 0.f ? 0.69314718055994531f / med : 0.f;
    }
  }
  if (t == 0) st->done = 0u;
}

__device__ __forceinline__ float power_x(const float2* spec, int64_t n, int64_t r, float scale) {
  if (r < 0 || r >= n) return 0.f;
  return fminf(power_of(spec[r]) * scale, kXCap);
}

// Windows of x: window w covers bins [w*hop - Wd/4, w*hop + 3Wd/4), 0 outside [0, n).
__global__ void spectrum_windows_kernel(const float2* spec, int64_t n, const float* scale, int Wd, int hop,
                                        float* x) {
  const int64_t w = blockIdx.x;
  const int64_t r0 = w * hop - Wd / 4;
  const float sc = *scale;
  for (int t = threadIdx.x; t < Wd; t += blockDim.x) x[w * Wd + t] = power_x(spec, n, r0 + t, sc);
}

// Proposal -> correlation work list.  Segment j of group g (G segments of V bins: outputs
// [(gG+j)V, (gG+j+1)V)) is proposed for template z if any window whose central bins
// [w*hop, (w+1)*hop) meet the bins its outputs can draw on, [(gG+j)V - h, (gG+j+1)V + h), has
// sigmoid(logit_z) >= threshold; mask[g][z] holds those G bits and unit (g, z) is listed when
// any is set.
__global__ void group_flags_kernel(const float* logits, int n_win, int Z, float logit_thr, int hop, int64_t seg_bins,
                                   int G, int h, int n_groups, uint16_t* masks, int* counts) {
  const int g = blockIdx.x;
  const int64_t lo = (int64_t)g * G * seg_bins - h, hi = ((int64_t)g + 1) * G * seg_bins + h;
  int w0 = (int)((lo > 0 ? lo : 0) / hop);
  int w1 = (int)((hi + hop - 1) / hop);
  if (w1 > n_win) w1 = n_win;
  __shared__ int cnt;
  if (threadIdx.x == 0) cnt = 0;
  __syncthreads();
  for (int z = threadIdx.x; z < Z; z += blockDim.x) {
    unsigned m = 0u;
    for (int w = w0; w < w1; ++w) {
      if (!(logits[(size_t)w * Z + z] >= logit_thr)) continue;
      const int64_t b0 = (int64_t)w * hop, b1 = b0 + hop;   // the window's central bins
      for (int j = 0; j < G; ++j) {
        const int64_t s0 = ((int64_t)g * G + j) * seg_bins - h, s1 = ((int64_t)g * G + j + 1) * seg_bins + h;
        if (b0 < s1 && b1 > s0) m |= 1u << j;
      }
    }
    masks[(size_t)g * Z + z] = (uint16_t)m;
    if (m) atomicAdd(&cnt, 1);
  }
  __syncthreads();
  if (threadIdx.x == 0) counts[g] = cnt;
}

// Proposal -> pair list.  Segment s has the outputs [s*V, (s+1)*V) (seg_bins = V) and draws on
// the inputs [s*V - h, (s+1)*V + h).  A template q is proposed for it by a block w (central bins
// [w*hop, (w+1)*hop)) that meets its outputs with sigmoid(logit) >= threshold, or by a block that
// meets only the inputs beyond them with sigmoid(logit) >= reach_threshold (a signal there must be
// strong for its response to reach the segment's outputs); pair (s, z) is listed when a template
// within z_halo of z is proposed.  One block per segment: the two maxima per template, the
// proposed flags in shared memory (Z ints), then the dilation.  mask[s][z] = 1 for a listed pair.
__global__ void segment_flags_kernel(const float* logits, int n_win, int Z, float logit_thr, float logit_reach,
                                     int z_halo, int hop, int64_t seg_bins, int h, uint16_t* masks, int* counts) {
  extern __shared__ int sflag[];
  const int64_t s = blockIdx.x;
  const int64_t o0 = s * seg_bins, o1 = (s + 1) * seg_bins;   // outputs
  const int64_t r0 = o0 - h, r1 = o1 + h;                     // inputs
  auto clampw = [&](int64_t w) { return (int)(w < 0 ? 0 : (w > n_win ? n_win : w)); };
  const int wr0 = clampw((r0 > 0 ? r0 : 0) / hop), wr1 = clampw((r1 + hop - 1) / hop);
  const int wo0 = clampw(o0 / hop), wo1 = clampw((o1 + hop - 1) / hop);
  __shared__ int cnt;
  if (threadIdx.x == 0) cnt = 0;
  for (int z = threadIdx.x; z < Z; z += blockDim.x) {
    float own = -INFINITY, reach = -INFINITY;   // NaN logits never list
    for (int w = wr0; w < wr1; ++w) {
      const float v = logits[(size_t)w * Z + z];
      if (w >= wo0 && w < wo1) own = fmaxf(own, v);
      else reach = fmaxf(reach, v);
    }
    sflag[z] = (own >= logit_thr || reach >= logit_reach) ? 1 : 0;
  }
  __syncthreads();
  for (int z = threadIdx.x; z < Z; z += blockDim.x) {
    const int a = z - z_halo > 0 ? z - z_halo : 0, b = z + z_halo < Z - 1 ? z + z_halo : Z - 1;
    bool f = false;
    for (int q = a; q <= b && !f; ++q) f = sflag[q] != 0;
    masks[(size_t)s * Z + z] = f ? 1 : 0;
    if (f) atomicAdd(&cnt, 1);
  }
  __syncthreads();
  if (threadIdx.x == 0) counts[s] = cnt;
}

// Exclusive scan of per-group counts and the total: one block of 1024 threads, thread t owning
// the contiguous chunk [t c, (t+1) c) of the groups; chunk sums are scanned with warp shuffles.
__global__ void __launch_bounds__(1024) scan_counts_kernel(const int* counts, int n_groups, int64_t* offsets,
                                                           int64_t* total) {
  __shared__ int64_t warp_excl[32];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int chunk = (n_groups + 1023) / 1024;
  const int b = tid * chunk < n_groups ? tid * chunk : n_groups;
  const int e = b + chunk < n_groups ? b + chunk : n_groups;
  int64_t own = 0;
  for (int g = b; g < e; ++g) own += counts[g];
  int64_t incl = own;   // inclusive scan over the warp
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int64_t y = __shfl_up_sync(0xffffffffu, incl, off);
    if (lane >= off) incl += y;
  }
  if (lane == 31) warp_excl[wid] = incl;
  __syncthreads();
  if (wid == 0) {
    const int64_t ws = warp_excl[lane];
    int64_t wi = ws;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int64_t y = __shfl_up_sync(0xffffffffu, wi, off);
      if (lane >= off) wi += y;
    }
    warp_excl[lane] = wi - ws;
  }
  __syncthreads();
  int64_t run = warp_excl[wid] + incl - own;
  for (int g = b; g < e; ++g) {
    offsets[g] = run;
    run += counts[g];
  }
  if (tid == 1023) *total = run;
}

// units[offset_g + k] = g*Z + z for the k-th proposed z of group g (increasing z), and its
// segment mask when out_masks is set: one block of 256 threads per group, each unit placed by
// the popcount of the proposed templates before it.
__global__ void __launch_bounds__(256) write_units_kernel(const uint16_t* masks, const int64_t* offsets, int Z,
                                                          int32_t* units, uint16_t* out_masks) {
  __shared__ int warp_cnt[8];
  const int g = blockIdx.x, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int64_t base = offsets[g];
  for (int z0 = 0; z0 < Z; z0 += 256) {
    const int z = z0 + (int)threadIdx.x;
    const unsigned mz = z < Z ? masks[(size_t)g * Z + z] : 0u;
    const bool f = mz != 0u;
    const unsigned m = __ballot_sync(0xffffffffu, f);
    if (lane == 0) warp_cnt[wid] = __popc(m);
    __syncthreads();
    int before = 0, all = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      before += i < wid ? warp_cnt[i] : 0;
      all += warp_cnt[i];
    }
    if (f) {
      const int64_t at = base + before + __popc(m & ((1u << lane) - 1u));
      units[at] = (int32_t)((int64_t)g * Z + z);
      if (out_masks) out_masks[at] = (uint16_t)mz;
    }
    base += all;
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------------------
// Fused inference over a whole spectrum on the tensor cores (tcgen05.mma kind::f16: FP16
// weights and activations, FP32 accumulation in TMEM).  A CTA holds the weights once and runs
// two independent groups of 8 warps, each with its own activation slot, half of the TMEM
// allocation, mbarrier and named barriers, so one group's MMAs overlap the other's epilogues.
// Group g of CTA b walks blocks w = 2b + g, 2b + g + 2*gridDim.x, ...; block w owns output
// positions [w*hop, (w+1)*hop) and recomputes the +-84-position halo its three layers need
// (dilations 1, 4, 16):
//   x   at P0-84 + j, j < 128*T1 + 8     (prefetched into registers one block ahead)
//   h1  at P0-80 + r, r < hop + 160      (layer 1 as an im2col GEMM: K = 9 taps padded to 16, M = positions)
//   h2  at P0-64 + r, r < hop + 128      (layer 2)
//   h3  at P0 + r,    r < hop            (layer 3, max-pooled per channel)
// Layers 2 and 3 (dilation d) put the weights on the M side: row 32 i + c of the accumulator is channel c
// at the positions t = 4 d a + d i + b (phase i < 4, 0 <= b < d), column P = d a + b.  Tap k of phase i
// reads input position t + d k, which is phase (i + k) mod 4 of the same split, d ((i + k) div 4) columns
// further: for each of the 12 offsets o = i + k one MMA multiplies [W_o; W_{o-1}; W_{o-2}; W_{o-3}]
// (zero where o - i is no tap) by the input rows of phase o mod 4 from column d (o div 4) on.  The
// weight rows are kept once, as the stack [0 0 0 W_8 ... W_0 0 0 0]: offset o starts at its block 11 - o.
// N is (hop + 128)/4 and hop/4 columns instead of 32 channels, where an MMA's time no longer has
// its floor of about 50 cycles: 24 MMAs and a clear, of 80 and 64 cycles, per layer for 512 positions, against 90
// and 72 of 64 cycles with one tap, 128 positions and N = 32 each (kernel 330 to 176 us at 2^22
// bins).  The zero blocks are a quarter of the multiply-adds; their rows' lanes are switched off, since an
// activation that overflowed FP16 times zero would be NaN where no tap reaches.
// Activations sit in shared memory K-major "chunk-planar": channel chunk j (8 channels, 16 B) of row q at
// plane j, offset 16*q, rows ordered (phase, column) for the layer that reads them.  h2 overwrites
// h1 after the MMAs that read it.  While a group's layer-2 MMAs are issued (the issuing thread is held to
// their pace) its other seven warps do the previous block's head, and during layer 3 the next block's
// staging and im2col; what is left between MMAs is the conversion of the two activation layers.  The
// groups issue layers 2 and 3 one at a time (a token): left alone they fall into step, both in their MMAs
// at half speed and then both outside (14.0k cycles per block and group; 12.5k with the token, before the clears).
// ---------------------------------------------------------------------------------------
constexpr int kMaxHop = 512;
constexpr int kT1max = kMaxHop / 128 + 2;       // layer-1 M-tiles
constexpr int kNP1 = (kMaxHop + 160) / 4 + 4;   // h1 rows per phase (+4: a quarter-warp's rows on all banks)
constexpr int kNP2 = (kMaxHop + 128) / 4;       // h2 rows per phase
constexpr int kNA1 = 128 * kT1max;              // im2col rows of layer 1
constexpr int kNX = kNA1 + 8;                   // staged x values
constexpr int kGroupThreads = 256;             // two warps per TMEM quadrant share its columns
constexpr int kProposeThreads = 2 * kGroupThreads;
constexpr int kSideThreads = kGroupThreads - 32;   // a group without its issuing warp
constexpr int kXPer = (kNX + kSideThreads - 1) / kSideThreads;   // prefetched x per thread
constexpr int kZStage = 256;                    // head weights staged in shared memory up to this Z
constexpr uint32_t kPlaneH1 = 4 * kNP1 * 16, kPlaneA1 = kNA1 * 16;
constexpr uint32_t kPlaneH2 = 4 * kNP2 * 16 + 16;   // + 16: the four planes of a row on different banks
using fdas::kStackRows;                         // weight rows of layers 2 and 3
constexpr uint32_t kPlaneW = kStackRows * 16;
constexpr int kOffW1 = 0;                       // layer-1 weights: 2 K-chunks x 512 B
constexpr int kOffW2 = kOffW1 + 1024;           // 4 K-chunks x 480 rows
constexpr int kOffW3 = kOffW2 + 4 * kPlaneW;
constexpr int kOffWl = kOffW3 + 4 * kPlaneW;    // head weights [Z][32] FP16
constexpr int kOffBl = kOffWl + kZStage * kC * 2;
constexpr int kOffBias = kOffBl + kZStage * 4;  // b1, b2, b3 (FP32 values of the FP16 copy)
constexpr int kOffSlot = (kOffBias + 3 * kC * 4 + 127) / 128 * 128;   // two activation slots
constexpr int kSlotA1 = 4 * kPlaneH1;           // layer-1 im2col of the next block
constexpr int kSlotX = kSlotA1 + 2 * kPlaneA1;  // staged x
constexpr int kSlotBytes = (kSlotX + kNX * 4 + 127) / 128 * 128;
constexpr int kOffGroup = kOffSlot + 2 * kSlotBytes;   // per group: channel maxima, mbarrier
constexpr int kGroupMisc = 384;
constexpr int kOffTslot = kOffGroup + 2 * kGroupMisc;
constexpr int kProposeSmem = kOffTslot + 16;   // TMEM base, MMA token
constexpr uint32_t kIdesc1 = fdas::umma_idesc_f16(128, kC);
constexpr uint32_t kTmemCols = 512;             // 256 columns per group (<= 6 x 32 used)
static_assert(kDil1 == 1, "layer 1 is an im2col of adjacent x values");
static_assert(kPlaneH2 <= kPlaneH1, "h2 fits in the h1 planes");
static_assert(32 * kT1max <= (int)kTmemCols / 2 && kNP2 <= (int)kTmemCols / 2, "a group's TMEM half");
static_assert(kProposeSmem <= 227 * 1024, "shared memory");

struct ProposeParams {
  const float2* spec;
  int64_t n;
  const float* scale;       // ln 2 / median |A|^2 (device scalar)
  const __half* w;          // FP16 parameter vector (Layout order)
  const __half* stack;      // and its layers 2 and 3 as they lie in shared memory
  int oW1, ob1, ob2, ob3, oWl, obl;
  int Z, hop;
  int64_t n_blocks;
  float* logits;            // n_blocks x Z
  int* status;              // bit 0: a bounded wait gave up
};

// B operand (layer-1 weights) in the K-major no-swizzle layout: rows o (N = 32), K = tap.
__device__ __forceinline__ int wb_off(int o, int i) { return (i >> 3) * 512 + (o >> 3) * 128 + (o & 7) * 16 + (i & 7) * 2; }

// Named barrier of one group (ids 1, 2; id 0 is __syncthreads).
__device__ __forceinline__ void group_sync(int g) {
  asm volatile("bar.sync %0, %1;" ::"r"(g + 1), "n"(kGroupThreads) : "memory");
}
// The group without its first warp (ids 3, 4).
__device__ __forceinline__ void side_sync(int g) {
  asm volatile("bar.sync %0, %1;" ::"r"(g + 3), "n"(kSideThreads) : "memory");
}
// Bounded acquisition of the CTA's MMA token (0: free) by one thread; false if it gave up.
__device__ __forceinline__ bool take_token(int* token) {
  if (atomicCAS(token, 0, 1) == 0) return true;
  const unsigned long long t0 = fdas::globaltimer_ns();
  while (atomicCAS(token, 0, 1) != 0)
    if (fdas::globaltimer_ns() - t0 > fdas::kWaitLimitNs) return false;
  return true;
}
__device__ __forceinline__ int group_all(int g, int v) {
  int r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.s32 p, %1, 0;\n\tbar.red.and.pred q, %2, %3, p;\n\t"
      "selp.s32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"(v), "r"(g + 1), "n"(kGroupThreads)
      : "memory");
  return r;
}

template <int HOP>
__global__ void __launch_bounds__(kProposeThreads, 1) propose_kernel(const ProposeParams p) {
  static_assert(HOP % 128 == 0 && HOP <= kMaxHop, "hop");
  using namespace fdas;
  extern __shared__ __align__(1024) unsigned char sm[];
  __half* sW1 = reinterpret_cast<__half*>(sm + kOffW1);
  __half* sWl = reinterpret_cast<__half*>(sm + kOffWl);
  float* sBl = reinterpret_cast<float*>(sm + kOffBl);
  float* sBias = reinterpret_cast<float*>(sm + kOffBias);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(sm + kOffTslot);
  int* token = reinterpret_cast<int*>(sm + kOffTslot + 4);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = warp >> 3, q = warp & 3, half = (warp >> 2) & 1, gt = tid & (kGroupThreads - 1);
  unsigned char* slot = sm + kOffSlot + g * kSlotBytes;
  float* sX = reinterpret_cast<float*>(slot + kSlotX);
  unsigned* sMax = reinterpret_cast<unsigned*>(sm + kOffGroup + g * kGroupMisc);   // two blocks' channel maxima
  uint64_t* bar = reinterpret_cast<uint64_t*>(sm + kOffGroup + g * kGroupMisc + 256);
  const bool wl_staged = p.Z <= kZStage;

  // weights of layer 1 into the B layout, layers 2 and 3 and the head (FP16); biases as FP32 values of the FP16 copy
  for (int idx = tid; idx < kC * 16; idx += kProposeThreads) {
    const int o = idx >> 4, k = idx & 15;
    sW1[wb_off(o, k) / 2] = k < kK ? p.w[p.oW1 + o * kK + k] : __float2half_rn(0.f);
  }
  // The image is laid out when the weights are published: gathered here from the parameter vector by
  // scattered 2-byte loads, a proposal took 36.9 us over 65,536 bins at window 512 (now 32.8) and 212 over 2^22 at
  // 1024 (now 203).
  static_assert(kOffW3 == kOffW2 + 4 * kPlaneW && 8 * kPlaneW == 2 * fdas::kStackHalves, "the stack's image");
#pragma unroll
  for (int idx = tid; idx < (int)(8 * kPlaneW / 16); idx += kProposeThreads)
    reinterpret_cast<uint4*>(sm + kOffW2)[idx] = __ldg(reinterpret_cast<const uint4*>(p.stack) + idx);
  if (wl_staged) {
    for (int idx = tid; idx < p.Z * kC / 8; idx += kProposeThreads)   // 16-byte aligned (NetLayout)
      reinterpret_cast<uint4*>(sWl)[idx] = reinterpret_cast<const uint4*>(p.w + p.oWl)[idx];
    for (int j = tid; j < p.Z; j += kProposeThreads) sBl[j] = __half2float(p.w[p.obl + j]);
  }
  if (tid < kC) {
    sBias[tid] = __half2float(p.w[p.ob1 + tid]);
    sBias[kC + tid] = __half2float(p.w[p.ob2 + tid]);
    sBias[2 * kC + tid] = __half2float(p.w[p.ob3 + tid]);
  }
  if (gt == 0) {
    mbar_init(bar, 1);
    fence_barrier_init();
    *token = 0;
  }
  if (warp == 0) {
    tmem_alloc(tslot, kTmemCols);
    tmem_relinquish();
  }
  fence_proxy_async_smem();
  tmem_fence_before_sync();
  __syncthreads();
  tmem_fence_after_sync();
  const uint32_t tm = *tslot + 256u * g;
  const uint32_t tm_lane = tm + ((uint32_t)(32 * q) << 16);
  const uint32_t aW1 = smem_u32(sW1), aW2 = smem_u32(sm + kOffW2), aW3 = smem_u32(sm + kOffW3);
  const uint32_t aSlot = smem_u32(slot);
  const float sc = *p.scale;
  constexpr int T1 = HOP / 128 + 2, N2 = (HOP + 128) / 4, N3 = HOP / 4;
  constexpr int nx = 128 * T1 + 8;
  uint32_t phase = 0;
  bool ok = true, issued = true;   // issued: the issuing thread got the token

  const int st = gt - 32;   // the input and the head are the work of the warps that issue no MMAs
  // x values of block w's staging window into registers (all loads issued before any use)
  float2 xa[kXPer];
  auto load_x = [&](int64_t P0) {
#pragma unroll
    for (int e = 0; e < kXPer; ++e) {
      const int j = st + kSideThreads * e;
      const int64_t r = P0 - kRF + j;
      xa[e] = (st >= 0 && j < nx && r >= 0 && r < p.n) ? __ldg(p.spec + r) : make_float2(0.f, 0.f);
    }
  };
  // wait for this group's committed MMAs: one thread polls (bounded), the others sleep in the
  // group's hardware barrier
  auto wait_mma = [&]() -> bool {
    const int good = group_all(g, gt == 0 ? (issued && mbar_wait(bar, phase) ? 1 : 0) : 1);
    phase ^= 1u;
    tmem_fence_after_sync();
    return good != 0;
  };
  auto sync_for_mma = [&]() {
    fence_proxy_async_smem();
    tmem_fence_before_sync();
    group_sync(g);
    tmem_fence_after_sync();
  };
  const __half2 zero2 = __floats2half2_rn(0.f, 0.f);
  // layer 1's accumulator tiles (lanes = positions r = 128t + 32q + lane, columns = channels) + bias -> relu
  // -> FP16 rows of layer 2's input, r < HOP + 160.  The next tile's TMEM load is issued before this
  // tile is converted (tcgen05.wait::ld waits for every earlier load, so the wait comes first and the two
  // buffers alternate).
  auto store_h1 = [&]() {
    float a[2][16], b[2][16];
    const uint32_t src = tm_lane + 32 * half;   // this warp's tiles: half, half + 2, ...
    tmem_ld16(src, a[0]);
    tmem_ld16(src + 16, b[0]);
    unsigned char* dst =
        slot + (32 * half + ((lane >> 2) & 3) * kNP1 + 8 * q + 4 * (lane >> 4) + (lane & 3)) * 16;
    constexpr int NT = (T1 + 1) / 2;
    static_for<NT>([&](auto tt) {
      constexpr int t = decltype(tt)::value, cur = t & 1;
      tmem_wait_ld();
      if constexpr (t + 1 < NT) {
        tmem_ld16(src + 64 * (t + 1), a[cur ^ 1]);
        tmem_ld16(src + 64 * (t + 1) + 16, b[cur ^ 1]);
      }
      const int r = 128 * (2 * t + half) + 32 * q + lane;
      if (r < HOP + 160) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          __half2 h[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {   // rounding is monotonic: relu after it is the same
            const int c = 8 * j + 2 * e;
            const float2 v = c < 16 ? make_float2(a[cur][c], a[cur][c + 1]) : make_float2(b[cur][c - 16], b[cur][c - 15]);
            h[e] = __hmax2(__float22half2_rn(add2(v, *reinterpret_cast<const float2*>(sBias + c))), zero2);
          }
          *reinterpret_cast<uint4*>(dst + j * kPlaneH1 + t * (64 * 16)) = *reinterpret_cast<uint4*>(h);
        }
      }
    });
  };
  // layer 2's accumulator (lanes = channel `lane` of phase q, columns P = 4a + b: position 16a + 4q + b)
  // + bias -> relu -> FP16 rows of layer 3's input
  auto store_h2 = [&]() {
    float v[2][16];
    const uint32_t src = tm_lane + 16 * half;   // this warp's column chunks c' = 2c + half
    tmem_ld16(src, v[0]);
    const float2 bias = bc(sBias[kC + lane]);
    unsigned char* dst = slot + (lane >> 3) * kPlaneH2 + (lane & 7) * 2 + (16 * half + 4 * q) * 16;
    static_assert(N2 % 32 == 0, "two warps share the columns");
    static_for<N2 / 32>([&](auto cc) {
      constexpr int c = decltype(cc)::value, cur = c & 1;
      tmem_wait_ld();
      if constexpr (c + 1 < N2 / 32) tmem_ld16(src + 32 * (c + 1), v[cur ^ 1]);
#pragma unroll
      for (int e = 0; e < 16; e += 2) {   // a = 4c' + e/4: phase e/4, column 16c' + 4q + e%4 of dilation 16
        const __half2 h = __hmax2(__float22half2_rn(add2(make_float2(v[cur][e], v[cur][e + 1]), bias)), zero2);
        unsigned char* at = dst + ((e >> 2) * kNP2 + 32 * c + (e & 3)) * 16;
        *reinterpret_cast<__half*>(at) = __low2half(h);
        *reinterpret_cast<__half*>(at + 16) = __high2half(h);
      }
    });
  };
  // one k = 9 convolution layer with dilation D: 12 offsets x 2 halves of the input channels.  A
  // descriptor's start address is its low field, so every operand is a base descriptor plus a
  // constant.
  auto issue_conv = [&](auto dil, auto cols, uint32_t wts, uint32_t plane, uint32_t rows_per_phase) {
    constexpr int D = decltype(dil)::value, N = decltype(cols)::value;
    const uint64_t a0 = umma_desc(wts, kPlaneW, 128), b0 = umma_desc(aSlot, plane, 128);
    issued = take_token(token);
    if (!issued) return;
    // D = 0: from row 384 of the stack on, its last three blocks and the next plane's first three are zero
    const uint64_t zero = umma_desc(aW2 + 12 * kC * 16, kPlaneW, 128);
    static_assert(N <= 6 * kC, "rows of zeros");
    umma_f16(tm, zero, zero, umma_idesc_f16(128, N), 0u);
    static_for<12>([&](auto oo) {
      constexpr int o = decltype(oo)::value;
      static_for<2>([&](auto cc) {
        constexpr int c = decltype(cc)::value;
        const uint64_t ad = a0 + (uint64_t)((2u * c * kPlaneW + (11 - o) * kC * 16) >> 4);
        const uint64_t bd = b0 + (uint64_t)((2u * c * plane + ((o & 3) * rows_per_phase + D * (o >> 2)) * 16) >> 4);
        // the phases i for which o - i is no tap
        constexpr uint32_t off = o < 3 ? (0xEu << o) & 0xFu : (o > 8 ? (1u << (o - 8)) - 1u : 0u);
        umma_f16_lanes<off>(tm, ad, bd, umma_idesc_f16(128, N));
      });
    });
    umma_commit(bar);
    atomicExch(token, 0);
  };

  // x of the block in registers -> layer-1 im2col: row r (position P0-80+r) = x[r .. r+8], zero for K in [9, 16)
  unsigned char* sA1 = slot + kSlotA1;
  auto stage_x = [&]() {
#pragma unroll
    for (int e = 0; e < kXPer; ++e) {
      const int j = st + kSideThreads * e;
      if (st >= 0 && j < nx) sX[j] = fminf(power_of(xa[e]) * sc, kXCap);
    }
  };
  auto im2col = [&]() {
    for (int r = st; r < 128 * T1; r += kSideThreads) {
      __half2 h[8];
#pragma unroll
      for (int e = 0; e < 4; ++e) h[e] = __floats2half2_rn(sX[r + 2 * e], sX[r + 2 * e + 1]);
      h[4] = __floats2half2_rn(sX[r + 8], 0.f);
      h[5] = h[6] = h[7] = zero2;
      *reinterpret_cast<uint4*>(sA1 + r * 16) = *reinterpret_cast<uint4*>(&h[0]);
      *reinterpret_cast<uint4*>(sA1 + kPlaneA1 + r * 16) = *reinterpret_cast<uint4*>(&h[4]);
    }
  };
  // logits[w][j] = bl[j] + sum_c Wl[j][c] m[c]  (FP16 weights, FP32 sums)
  auto head = [&](int64_t w, const unsigned* smax) {
    float mc[kC];
#pragma unroll
    for (int c = 0; c < kC; ++c) mc[c] = __uint_as_float(smax[c]);
    for (int j = st; j < p.Z; j += kSideThreads) {
      const __half* wl = wl_staged ? sWl + j * kC : p.w + p.oWl + (size_t)j * kC;
      float s = wl_staged ? sBl[j] : __half2float(p.w[p.obl + j]);
#pragma unroll
      for (int c4 = 0; c4 < kC / 8; ++c4) {
        const uint4 u = *reinterpret_cast<const uint4*>(wl + 8 * c4);
        const __half2* h2 = reinterpret_cast<const __half2*>(&u);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float2 f = __half22float2(h2[e]);
          s = fmaf(f.x, mc[8 * c4 + 2 * e], s);
          s = fmaf(f.y, mc[8 * c4 + 2 * e + 1], s);
        }
      }
      p.logits[w * p.Z + j] = s;
    }
  };

  const int64_t wstep = 2 * (int64_t)gridDim.x;
  int64_t w = 2 * (int64_t)blockIdx.x + g, w_prev = -1;
  unsigned* max_cur = sMax;           // this block's maxima (zero when its layer 3 is read)
  unsigned* max_prev = sMax + kC;     // the previous block's
  if (w < p.n_blocks) {
    if (st >= 0) {
      load_x(w * HOP);
      stage_x();
      side_sync(g);
      if (w + wstep < p.n_blocks) load_x((w + wstep) * HOP);
      im2col();
    } else {
      max_cur[lane] = 0u;
    }
  }
  for (; w < p.n_blocks; w += wstep) {
    sync_for_mma();
    if (gt == 0) {
      const uint64_t bd = umma_desc(aW1, 512, 128), a0 = umma_desc(aSlot + kSlotA1, kPlaneA1, 128);
      static_for<T1>([&](auto tt) {
        constexpr int t = decltype(tt)::value;
        umma_f16(tm + 32 * t, a0 + (uint64_t)(128 * t), bd, kIdesc1, 0u);   // 128 rows x 16 B = 2048 B
      });
      umma_commit(bar);
    }
    if (!(ok = wait_mma())) break;
    store_h1();
    sync_for_mma();
    if (gt == 0)
      issue_conv(std::integral_constant<int, kDil2>{}, std::integral_constant<int, N2>{}, aW2, kPlaneH1, kNP1);
    if (st >= 0 && w_prev >= 0) head(w_prev, max_prev);
    if (!(ok = wait_mma())) break;
    store_h2();
    sync_for_mma();
    if (gt == 0)
      issue_conv(std::integral_constant<int, kDil3>{}, std::integral_constant<int, N3>{}, aW3, kPlaneH2, kNP2);
    // the next block's input (every thread has left the head that read max_prev)
    if (st < 0) {
      max_prev[lane] = 0u;
    } else if (w + wstep < p.n_blocks) {
      stage_x();
      side_sync(g);
      if (w + 2 * wstep < p.n_blocks) load_x((w + 2 * wstep) * HOP);
      im2col();
    }
    if (!(ok = wait_mma())) break;
    // layer 3: relu(acc + b3), channel maxima over the block: this lane's channel at its warp's phase,
    // then the four phases (adding the bias after the maximum changes nothing; non-negative floats
    // order as unsigned)
    {
      float mx = -INFINITY, v[2][16];
      const uint32_t src = tm_lane + 16 * half;
      static_assert(N3 % 32 == 0, "two warps share the columns");
      tmem_ld16(src, v[0]);
      static_for<N3 / 32>([&](auto cc) {
        constexpr int c = decltype(cc)::value, cur = c & 1;
        tmem_wait_ld();
        if constexpr (c + 1 < N3 / 32) tmem_ld16(src + 32 * (c + 1), v[cur ^ 1]);
#pragma unroll
        for (int e = 0; e < 16; ++e) mx = fmaxf(mx, v[cur][e]);
      });
      atomicMax(&max_cur[lane], __float_as_uint(fmaxf(mx + sBias[2 * kC + lane], 0.f)));
    }
    unsigned* const t = max_cur;
    max_cur = max_prev;
    max_prev = t;
    w_prev = w;
  }
  if (ok && w_prev >= 0) {
    group_sync(g);
    if (st >= 0) head(w_prev, max_prev);
  }
  if (!ok && gt == 0) {
    atomicOr(p.status, 1);
    (void)mbar_wait(bar, phase ^ 1u);   // bounded wait for this group's MMAs still in flight
  }
  tmem_fence_before_sync();
  __syncthreads();
  tmem_fence_after_sync();
  if (warp == 0) tmem_dealloc(*tslot, kTmemCols);
}

}  // namespace

struct fdas_zband {
  int Wd = 0, Z = 0, max_batch = 0, sm_count = 0;
  fdas::NetState net;
  SelectState* sel = nullptr; // median selection state
  float* scale = nullptr;    // ln 2 / median |A|^2
  int* status = nullptr;     // bit 0: a bounded wait of the inference kernel gave up
  int step = 0;
  // fdas_zband_propose as a CUDA graph of its launches, captured for these arguments
  cudaStream_t capture_stream = nullptr;
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t graph_exec = nullptr;
  const void* cap_spec = nullptr;
  int64_t cap_n = 0;
  const void* cap_logits = nullptr;
  // the synchronous host accessors run on `own`; `done` marks the last work enqueued on the net
  // (they and fdas_zband_destroy wait for it, not for the whole device)
  cudaStream_t own = nullptr;
  cudaEvent_t done = nullptr;
};

namespace {
void free_zband(fdas_zband* z) {
  const fdas::NetState& s = z->net;
  void* ptrs[] = {s.p,      s.ph,   s.pr,   s.stack, s.packs,  s.g,    s.m,         s.v,        s.h1,    s.h2,    s.d2,    s.pool,
                  s.pool_arg, s.pooled, s.seed, s.arg, s.logits, s.dlog, s.loss, s.loss_part, s.db2_part, s.part1, s.sum1, s.part2,
                  s.part3,  s.gl,   z->sel, z->scale, z->status};
  for (void* q : ptrs) cudaFree(q);
  if (z->graph_exec) cudaGraphExecDestroy(z->graph_exec);
  if (z->graph) cudaGraphDestroy(z->graph);
  if (z->capture_stream) cudaStreamDestroy(z->capture_stream);
  if (z->own) cudaStreamDestroy(z->own);
  if (z->done) cudaEventDestroy(z->done);
  delete z;
}

// Record the net's completion event after work enqueued on `st` (not while `st` is being captured
// into a CUDA graph: a captured record is no event the host can wait on).
int note_work(fdas_zband* z, cudaStream_t st, cudaError_t launch) {
  if (launch != cudaSuccess) return FDAS_ERR_CUDA;
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &cs) != cudaSuccess) return FDAS_ERR_CUDA;
  if (cs != cudaStreamCaptureStatusNone) return FDAS_OK;
  return cudaEventRecord(z->done, st) == cudaSuccess ? FDAS_OK : FDAS_ERR_CUDA;
}

// Host copy between the net's buffers and host memory on its own stream, after the net's last
// enqueued work; returns when the copy has completed.
int host_copy(fdas_zband* z, void* dst, const void* src, size_t bytes, cudaMemcpyKind kind) {
  if (cudaStreamWaitEvent(z->own, z->done, 0) != cudaSuccess ||
      cudaMemcpyAsync(dst, src, bytes, kind, z->own) != cudaSuccess || cudaStreamSynchronize(z->own) != cudaSuccess)
    return FDAS_ERR_CUDA;
  return FDAS_OK;
}

// scale = ln 2 / median |A|^2 into `scale`: a clear and three launches.
void launch_power_scale(const float2* spec, int64_t n, SelectState* sel, float* scale, cudaStream_t st) {
  const int64_t blocks = (n + 256 * kSelPer - 1) / (256 * kSelPer);
  auto grid = [&](int64_t cap) { return (unsigned)(blocks < cap ? blocks : cap); };
  cudaMemsetAsync(sel, 0, sizeof(SelectState), st);
  select_pass_kernel<0><<<grid(kSelBlocks0), 256, select_smem<0>(), st>>>(spec, n, sel, scale);
  select_pass_kernel<1><<<grid(kSelBlocks), 256, select_smem<1>(), st>>>(spec, n, sel, scale);
  select_pass_kernel<2><<<grid(kSelBlocks), 256, select_smem<2>(), st>>>(spec, n, sel, scale);
}
cudaError_t prepare_power_scale() {
  return cudaFuncSetAttribute(select_pass_kernel<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)select_smem<0>());
}
}  // namespace

extern "C" {

fdas_zband* fdas_zband_create(int window, int n_out, int max_batch) {
  // the window's quarter margins must hold the receptive field (the windowed and whole-sequence
  // forms then agree)
  if (window < 4 * kRF || window % kWidthStep != 0 || window > (1 << 16) || n_out < 1 || n_out > 65535 ||
      max_batch < 1 || max_batch > 65535)
    return nullptr;
  int dev = 0, major = 0, minor = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) ||
      cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev) ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) || major != 10 || minor != 3) {
    cudaGetLastError();
    return nullptr;
  }
  if (fdas::net_prepare() != cudaSuccess || prepare_power_scale() != cudaSuccess ||
      cudaFuncSetAttribute(propose_kernel<256>, cudaFuncAttributeMaxDynamicSharedMemorySize, kProposeSmem) !=
          cudaSuccess ||
      cudaFuncSetAttribute(propose_kernel<384>, cudaFuncAttributeMaxDynamicSharedMemorySize, kProposeSmem) !=
          cudaSuccess ||
      cudaFuncSetAttribute(propose_kernel<512>, cudaFuncAttributeMaxDynamicSharedMemorySize, kProposeSmem) !=
          cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  fdas_zband* z = new (std::nothrow) fdas_zband();
  if (!z) return nullptr;
  z->Wd = window;
  z->Z = n_out;
  z->max_batch = max_batch;
  z->sm_count = sms;
  fdas::NetState& s = z->net;
  s.lay = Layout(n_out);
  s.W = window;
  const size_t P = (size_t)s.lay.total, B = (size_t)max_batch;
  const fdas::NetSizes n = fdas::net_sizes(window, n_out, max_batch);
  bool ok = cudaMalloc(&s.p, P * 4) == cudaSuccess && cudaMalloc(&s.ph, P * 2) == cudaSuccess &&
            cudaMalloc(&s.pr, P * 4) == cudaSuccess && cudaMalloc(&s.packs, n.packs * 4) == cudaSuccess &&
            cudaMalloc(&s.stack, fdas::kStackHalves * 2) == cudaSuccess &&
            cudaMalloc(&s.g, P * 4) == cudaSuccess && cudaMalloc(&s.m, P * 4) == cudaSuccess &&
            cudaMalloc(&s.v, P * 4) == cudaSuccess && cudaMalloc(&s.h1, n.act * 4) == cudaSuccess &&
            cudaMalloc(&s.h2, n.act * 4) == cudaSuccess && cudaMalloc(&s.d2, n.act * 4) == cudaSuccess &&
            cudaMalloc(&s.pool, n.pool * 4) == cudaSuccess && cudaMalloc(&s.pool_arg, n.pool * 4) == cudaSuccess &&
            cudaMalloc(&s.pooled, B * kC * 4) == cudaSuccess && cudaMalloc(&s.seed, B * kC * 4) == cudaSuccess &&
            cudaMalloc(&s.arg, B * kC * 4) == cudaSuccess &&
            cudaMalloc(&s.logits, B * (size_t)n_out * 4) == cudaSuccess &&
            cudaMalloc(&s.dlog, B * (size_t)n_out * 4) == cudaSuccess && cudaMalloc(&s.loss, 4) == cudaSuccess &&
            cudaMalloc(&s.loss_part, B * 4) == cudaSuccess && cudaMalloc(&s.db2_part, B * kC * 4) == cudaSuccess &&
            cudaMalloc(&s.part1, n.part1 * 4) == cudaSuccess && cudaMalloc(&s.sum1, n.sum1 * 4) == cudaSuccess && cudaMalloc(&s.part2, n.part2 * 4) == cudaSuccess &&
            cudaMalloc(&s.part3, n.part3 * 4) == cudaSuccess && cudaMalloc(&s.gl, n.gl * 4) == cudaSuccess &&
            cudaMalloc(&z->sel, sizeof(SelectState)) == cudaSuccess &&
            cudaMalloc(&z->scale, 4) == cudaSuccess && cudaMalloc(&z->status, 4) == cudaSuccess &&
            cudaStreamCreateWithFlags(&z->own, cudaStreamNonBlocking) == cudaSuccess &&
            cudaEventCreateWithFlags(&z->done, cudaEventDisableTiming) == cudaSuccess;
  if (!ok || cudaMemsetAsync(s.p, 0, P * 4, z->own) != cudaSuccess ||
      cudaMemsetAsync(s.ph, 0, P * 2, z->own) != cudaSuccess || cudaMemsetAsync(s.pr, 0, P * 4, z->own) != cudaSuccess ||
      cudaMemsetAsync(s.packs, 0, n.packs * 4, z->own) != cudaSuccess ||
      cudaMemsetAsync(s.stack, 0, fdas::kStackHalves * 2, z->own) != cudaSuccess ||
      cudaMemsetAsync(s.m, 0, P * 4, z->own) != cudaSuccess || cudaMemsetAsync(s.v, 0, P * 4, z->own) != cudaSuccess ||
      cudaMemsetAsync(z->status, 0, 4, z->own) != cudaSuccess ||
      cudaEventRecord(z->done, z->own) != cudaSuccess || cudaStreamSynchronize(z->own) != cudaSuccess) {
    cudaGetLastError();
    free_zband(z);
    return nullptr;
  }
  return z;
}

int fdas_zband_param_count(const fdas_zband* z) { return z ? z->net.lay.total : FDAS_ERR_INVALID; }

int fdas_zband_set_params(fdas_zband* z, const float* host_params) {
  if (!z || !host_params) return FDAS_ERR_INVALID;
  const int P = z->net.lay.total;
  if (host_copy(z, z->net.p, host_params, (size_t)P * 4, cudaMemcpyHostToDevice) != FDAS_OK) return FDAS_ERR_CUDA;
  fdas::net_publish(z->net, z->own);
  cudaMemsetAsync(z->net.m, 0, (size_t)P * 4, z->own);
  cudaMemsetAsync(z->net.v, 0, (size_t)P * 4, z->own);
  z->step = 0;
  if (note_work(z, z->own, cudaGetLastError()) != FDAS_OK) return FDAS_ERR_CUDA;
  return cudaStreamSynchronize(z->own) == cudaSuccess ? FDAS_OK : FDAS_ERR_CUDA;
}

int fdas_zband_get_params(fdas_zband* z, float* host_params) {
  if (!z || !host_params) return FDAS_ERR_INVALID;
  return host_copy(z, host_params, z->net.p, (size_t)z->net.lay.total * 4, cudaMemcpyDeviceToHost);
}

int fdas_zband_get_adam(fdas_zband* z, float* host_m, float* host_v, int* host_step) {
  if (!z || !host_m || !host_v || !host_step) return FDAS_ERR_INVALID;
  const size_t bytes = (size_t)z->net.lay.total * 4;
  if (host_copy(z, host_m, z->net.m, bytes, cudaMemcpyDeviceToHost) != FDAS_OK ||
      host_copy(z, host_v, z->net.v, bytes, cudaMemcpyDeviceToHost) != FDAS_OK)
    return FDAS_ERR_CUDA;
  *host_step = z->step;
  return FDAS_OK;
}

int fdas_zband_set_adam(fdas_zband* z, const float* host_m, const float* host_v, int step) {
  if (!z || !host_m || !host_v || step < 0) return FDAS_ERR_INVALID;
  const size_t bytes = (size_t)z->net.lay.total * 4;
  if (host_copy(z, z->net.m, host_m, bytes, cudaMemcpyHostToDevice) != FDAS_OK ||
      host_copy(z, z->net.v, host_v, bytes, cudaMemcpyHostToDevice) != FDAS_OK)
    return FDAS_ERR_CUDA;
  z->step = step;
  return FDAS_OK;
}

int fdas_zband_train_step(fdas_zband* z, const float* d_windows, const float* d_targets, int batch, float lr,
                          float* host_loss, fdas_stream_t stream) {
  if (!z || !d_windows || !d_targets || batch < 1 || batch > z->max_batch || !(lr > 0.f)) return FDAS_ERR_INVALID;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  if (fdas::net_train_step(z->net, d_windows, d_targets, batch, lr, z->step + 1, st) != cudaSuccess)
    return FDAS_ERR_CUDA;
  z->step += 1;
  if (note_work(z, st, cudaGetLastError()) != FDAS_OK) return FDAS_ERR_CUDA;
  if (host_loss) {
    if (cudaMemcpyAsync(host_loss, z->net.loss, 4, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
      return FDAS_ERR_CUDA;
  }
  return FDAS_OK;
}

int fdas_zband_gradients(fdas_zband* z, float* host_grads) {
  if (!z || !host_grads) return FDAS_ERR_INVALID;
  return host_copy(z, host_grads, z->net.g, (size_t)z->net.lay.total * 4, cudaMemcpyDeviceToHost);
}

int fdas_zband_predict(fdas_zband* z, const float* d_windows, int batch, int half_weights, float* d_logits,
                       fdas_stream_t stream) {
  if (!z || !d_windows || !d_logits || batch < 1) return FDAS_ERR_INVALID;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  for (int b0 = 0; b0 < batch; b0 += z->max_batch) {
    const int B = batch - b0 < z->max_batch ? batch - b0 : z->max_batch;
    if (fdas::net_predict(z->net, d_windows + (size_t)b0 * z->Wd, B, half_weights != 0, d_logits + (size_t)b0 * z->Z,
                          st) != cudaSuccess)
      return FDAS_ERR_CUDA;
  }
  return note_work(z, st, cudaGetLastError());
}

// The launches of one proposal (median passes, then the fused inference) on `st`.
static cudaError_t launch_propose(fdas_zband* z, const float* d_spectrum, int64_t n_bins, float* d_logits,
                                  cudaStream_t st) {
  const int hop = z->Wd / 2;
  const int64_t nb = (n_bins + hop - 1) / hop;
  launch_power_scale(reinterpret_cast<const float2*>(d_spectrum), n_bins, z->sel, z->scale, st);
  ProposeParams q;
  q.spec = reinterpret_cast<const float2*>(d_spectrum);
  q.n = n_bins;
  q.scale = z->scale;
  q.w = z->net.ph;
  q.stack = z->net.stack;
  q.oW1 = z->net.lay.W1;
  q.ob1 = z->net.lay.b1;
  q.ob2 = z->net.lay.b2;
  q.ob3 = z->net.lay.b3;
  q.oWl = z->net.lay.Wl;
  q.obl = z->net.lay.bl;
  q.Z = z->Z;
  q.hop = hop;
  q.n_blocks = nb;
  q.logits = d_logits;
  q.status = z->status;
  const int64_t pairs = (nb + 1) / 2;
  const unsigned grid = (unsigned)(pairs < z->sm_count ? pairs : z->sm_count);
  switch (hop) {
    case 256: propose_kernel<256><<<grid, kProposeThreads, kProposeSmem, st>>>(q); break;
    case 384: propose_kernel<384><<<grid, kProposeThreads, kProposeSmem, st>>>(q); break;
    default: propose_kernel<512><<<grid, kProposeThreads, kProposeSmem, st>>>(q); break;
  }
  return cudaGetLastError();
}

int fdas_zband_propose(fdas_zband* z, const float* d_spectrum, int64_t n_bins, float* d_logits,
                       fdas_stream_t stream) {
  if (!z || !d_spectrum || !d_logits || n_bins < 1 || n_bins > (int64_t(1) << 30)) return FDAS_ERR_INVALID;
  const int hop = z->Wd / 2;
  if (hop % 128 != 0 || hop > kMaxHop) return FDAS_ERR_INVALID;
  if ((reinterpret_cast<uintptr_t>(d_spectrum) & 7u) || (reinterpret_cast<uintptr_t>(d_logits) & 3u))
    return FDAS_ERR_ALIGN;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  // a clear and four launches replayed as one graph: captured again when the spectrum, its length or the
  // logits buffer change (the weights are read through fixed pointers, so training needs none)
  if (!(z->graph_exec && z->cap_spec == d_spectrum && z->cap_n == n_bins && z->cap_logits == d_logits)) {
    if (z->graph_exec) cudaGraphExecDestroy(z->graph_exec);
    if (z->graph) cudaGraphDestroy(z->graph);
    z->graph_exec = nullptr;
    z->graph = nullptr;
    if (!z->capture_stream && cudaStreamCreateWithFlags(&z->capture_stream, cudaStreamNonBlocking) != cudaSuccess) {
      z->capture_stream = nullptr;
      return FDAS_ERR_CUDA;
    }
    if (cudaStreamBeginCapture(z->capture_stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess)
      return FDAS_ERR_CUDA;
    const cudaError_t le = launch_propose(z, d_spectrum, n_bins, d_logits, z->capture_stream);
    cudaGraph_t g = nullptr;
    const cudaError_t ce = cudaStreamEndCapture(z->capture_stream, &g);
    if (le != cudaSuccess || ce != cudaSuccess || !g) {
      if (g) cudaGraphDestroy(g);
      cudaGetLastError();
      return FDAS_ERR_CUDA;
    }
    if (cudaGraphInstantiate(&z->graph_exec, g, 0) != cudaSuccess) {
      cudaGraphDestroy(g);
      z->graph_exec = nullptr;
      cudaGetLastError();
      return FDAS_ERR_CUDA;
    }
    z->graph = g;
    z->cap_spec = d_spectrum;
    z->cap_n = n_bins;
    z->cap_logits = d_logits;
  }
  return note_work(z, st, cudaGraphLaunch(z->graph_exec, st));
}

int fdas_zband_check(fdas_zband* z, fdas_stream_t stream) {
  if (!z) return FDAS_ERR_INVALID;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  int status = 0;
  if (cudaMemcpyAsync(&status, z->status, 4, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    return FDAS_ERR_CUDA;
  if (status != 0) {
    if (cudaMemsetAsync(z->status, 0, 4, st) != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess)
      return FDAS_ERR_CUDA;
    return FDAS_ERR_TIMEOUT;
  }
  return FDAS_OK;
}

int fdas_zband_spectrum_windows(const float* d_spectrum, int64_t n_bins, int window, int hop, float* d_windows,
                                int64_t n_windows, fdas_stream_t stream) {
  if (!d_spectrum || !d_windows || n_bins < 1 || n_bins > (int64_t(1) << 30) || window < 4 || window % 4 != 0 ||
      window > (1 << 16) || hop < 1 || n_windows < 1 || n_windows > (1 << 30))
    return FDAS_ERR_INVALID;
  if (reinterpret_cast<uintptr_t>(d_spectrum) & 7u) return FDAS_ERR_ALIGN;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  SelectState* sel = nullptr;
  float* scale = nullptr;
  if (prepare_power_scale() != cudaSuccess) return FDAS_ERR_CUDA;
  if (cudaMallocAsync(&sel, sizeof(SelectState), st) != cudaSuccess) return FDAS_ERR_ALLOC;
  if (cudaMallocAsync(&scale, 4, st) != cudaSuccess) {
    cudaFreeAsync(sel, st);
    return FDAS_ERR_ALLOC;
  }
  launch_power_scale(reinterpret_cast<const float2*>(d_spectrum), n_bins, sel, scale, st);
  spectrum_windows_kernel<<<(unsigned)n_windows, 256, 0, st>>>(reinterpret_cast<const float2*>(d_spectrum), n_bins,
                                                               scale, window, hop, d_windows);
  const int rc = cudaGetLastError() == cudaSuccess ? FDAS_OK : FDAS_ERR_CUDA;
  cudaFreeAsync(sel, st);
  cudaFreeAsync(scale, st);
  return rc;
}

// Work-list scratch: offsets (int64, n_groups + 1), counts (int32, n_groups), segment masks
// (uint16, n_groups * Z), each 16-byte aligned.
static int64_t align16(int64_t x) { return (x + 15) & ~(int64_t)15; }
static int64_t units_scratch_bytes(int64_t n_groups, int Z) {
  return align16(8 * (n_groups + 1)) + align16(4 * n_groups) + align16(2 * n_groups * (int64_t)Z);
}

int64_t fdas_zband_work_units_scratch_bytes(int64_t n_groups, int Z) {
  if (n_groups < 1 || n_groups > (1 << 24) || Z < 1 || n_groups * (int64_t)Z > INT32_MAX) return FDAS_ERR_INVALID;
  return units_scratch_bytes(n_groups, Z);
}

int fdas_zband_work_units_masked(const float* d_logits, int64_t n_windows, int Z, float threshold, int hop,
                                 int64_t seg_bins, int G, int h, int64_t n_groups, int32_t* d_units,
                                 uint16_t* d_masks, void* d_scratch, int64_t* host_count, fdas_stream_t stream) {
  if (!d_logits || !d_units || (!host_count && !d_scratch) || n_windows < 1 || n_windows > (1 << 30) || Z < 1 ||
      !(threshold > 0.f && threshold < 1.f) || hop < 1 || seg_bins < 1 || G < 1 || G > 16 || h < 0 ||
      n_groups < 1 || n_groups > (1 << 24) || (int64_t)n_groups * Z > INT32_MAX ||
      seg_bins * G > (int64_t(1) << 40))
    return FDAS_ERR_INVALID;
  if ((reinterpret_cast<uintptr_t>(d_scratch) & 15u) || (reinterpret_cast<uintptr_t>(d_masks) & 1u))
    return FDAS_ERR_ALIGN;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const float logit_thr = logf(threshold / (1.f - threshold));
  const int64_t bytes = units_scratch_bytes(n_groups, Z);
  unsigned char* scratch = static_cast<unsigned char*>(d_scratch);
  const bool own = scratch == nullptr;
  if (own && cudaMallocAsync(reinterpret_cast<void**>(&scratch), (size_t)bytes, st) != cudaSuccess) {
    cudaGetLastError();
    return FDAS_ERR_ALLOC;
  }
  int64_t* offsets = reinterpret_cast<int64_t*>(scratch);
  int* counts = reinterpret_cast<int*>(scratch + align16(8 * (n_groups + 1)));
  uint16_t* masks = reinterpret_cast<uint16_t*>(scratch + align16(8 * (n_groups + 1)) + align16(4 * n_groups));
  group_flags_kernel<<<(unsigned)n_groups, 256, 0, st>>>(d_logits, (int)n_windows, Z, logit_thr, hop, seg_bins, G,
                                                        h, (int)n_groups, masks, counts);
  scan_counts_kernel<<<1, 1024, 0, st>>>(counts, (int)n_groups, offsets, offsets + n_groups);
  write_units_kernel<<<(unsigned)n_groups, 256, 0, st>>>(masks, offsets, Z, d_units, d_masks);
  int rc = FDAS_OK;
  if (cudaGetLastError() != cudaSuccess) rc = FDAS_ERR_CUDA;
  else if (host_count && (cudaMemcpyAsync(host_count, offsets + n_groups, 8, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
                          cudaStreamSynchronize(st) != cudaSuccess))
    rc = FDAS_ERR_CUDA;
  if (own) cudaFreeAsync(scratch, st);
  return rc;
}

int fdas_zband_work_units(const float* d_logits, int64_t n_windows, int Z, float threshold, int hop,
                          int64_t group_bins, int h, int64_t n_groups, int32_t* d_units, void* d_scratch,
                          int64_t* host_count, fdas_stream_t stream) {
  // one segment of group_bins per group: the group's flag
  return fdas_zband_work_units_masked(d_logits, n_windows, Z, threshold, hop, group_bins, 1, h, n_groups, d_units,
                                      nullptr, d_scratch, host_count, stream);
}

int fdas_zband_work_pairs(const float* d_logits, int64_t n_windows, int Z, float threshold, float reach_threshold,
                          int z_halo, int hop, int64_t seg_bins, int h, int64_t n_seg, int32_t* d_pairs,
                          void* d_scratch, int64_t* host_count, fdas_stream_t stream) {
  if (!d_logits || !d_pairs || !d_scratch || n_windows < 1 || n_windows > (1 << 30) || Z < 1 || Z > 8192 ||
      !(threshold > 0.f && threshold < 1.f) || !(reach_threshold >= threshold && reach_threshold <= 1.f) ||
      z_halo < 0 || z_halo > Z || hop < 1 || seg_bins < 1 || h < 0 ||
      n_seg < 1 || n_seg > (1 << 24) || n_seg * (int64_t)Z > INT32_MAX || seg_bins > (int64_t(1) << 40))
    return FDAS_ERR_INVALID;
  if ((reinterpret_cast<uintptr_t>(d_scratch) & 15u) || (reinterpret_cast<uintptr_t>(d_logits) & 3u) ||
      (reinterpret_cast<uintptr_t>(d_pairs) & 3u))
    return FDAS_ERR_ALIGN;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const float logit_thr = logf(threshold / (1.f - threshold));
  const float logit_reach = reach_threshold < 1.f ? logf(reach_threshold / (1.f - reach_threshold)) : INFINITY;
  unsigned char* scratch = static_cast<unsigned char*>(d_scratch);
  int64_t* offsets = reinterpret_cast<int64_t*>(scratch);
  int* counts = reinterpret_cast<int*>(scratch + align16(8 * (n_seg + 1)));
  uint16_t* masks = reinterpret_cast<uint16_t*>(scratch + align16(8 * (n_seg + 1)) + align16(4 * n_seg));
  segment_flags_kernel<<<(unsigned)n_seg, 256, sizeof(int) * (size_t)Z, st>>>(
      d_logits, (int)n_windows, Z, logit_thr, logit_reach, z_halo, hop, seg_bins, h, masks, counts);
  scan_counts_kernel<<<1, 1024, 0, st>>>(counts, (int)n_seg, offsets, offsets + n_seg);
  write_units_kernel<<<(unsigned)n_seg, 256, 0, st>>>(masks, offsets, Z, d_pairs, nullptr);
  if (cudaGetLastError() != cudaSuccess) return FDAS_ERR_CUDA;
  if (host_count && (cudaMemcpyAsync(host_count, offsets + n_seg, 8, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
                     cudaStreamSynchronize(st) != cudaSuccess))
    return FDAS_ERR_CUDA;
  return FDAS_OK;
}

int fdas_zband_destroy(fdas_zband* z) {
  if (!z) return FDAS_OK;
  if (z->done) cudaEventSynchronize(z->done);   // the net's last enqueued work, not the whole device
  free_zband(z);
  return FDAS_OK;
}

}  // extern "C"
