// fdas_internal.h -- declarations shared by the translation units of libfdas.
#pragma once

#include <cstdint>

#include <cuda_fp16.h>
#include <cuda_runtime.h>

namespace fdas {

// Bits of a device status word.
constexpr int kStatusTimeout = 1;   // a bounded device wait gave up
constexpr int kStatusBadList = 2;   // a work list failed its check and was not run

// Parameters of the fused correlation kernel (steps a2..a7).
struct ConvParams {
  const float2* spectrum;   // n_bins complex64 (read by bulk copies in the descriptor-driven kernel)
  const float2* templates;  // Z x L template spectra, per-template layout of the IFFT's first pass
  const float2* twist;      // L inter-pass twiddles exp(+i 2pi n2 k1 / L) (twist_re)
  float* plane;             // Z x n_bins output, row pitch n_bins
  int* status;              // device status word (kStatusTimeout | kStatusBadList)
  int64_t n_bins;
  int64_t nseg;             // ceil(n_bins / V)
  int Z, V, h;
  // work split (set by the launch): CTA k starts at unit k * span + min(k, span_extra) of a count in which
  // every segment group has group_cost units more than its templates
  int64_t span;
  int span_extra;
  int group_cost;
  int segs;                 // segments per group (set by the launch; fdas_convolve_wide.cu)
};

// One spectrum of a batch, as the persistent kernel reads it (device table or inline).
struct SpecDesc {
  const float2* spec;       // n_bins complex64, 16-byte aligned
  float* plane;             // Z x n_bins float32, row pitch n_bins
  int64_t n_bins;
  int64_t nseg;             // ceil(n_bins / V)
  int64_t unit_base;        // first flattened (segment group, template) unit of this spectrum
  int64_t ngroups;          // ceil(nseg / G), G = segments resident per CTA
  int Z;                    // templates of this spectrum
  int z_off;                // template-bank row of its first template
};

// Parameters of the descriptor-driven fused kernel (TMEM variant): one or many spectra.
struct BatchParams {
  const float2* templates;  // Z_bank x L template spectra (pair-major layout)
  const float2* twist;      // L inter-pass twiddles (twist_re)
  int* status;              // device status word (kStatusTimeout | kStatusBadList)
  const SpecDesc* descs;    // device table of `count` spectra, or nullptr: use `single`
  SpecDesc single;
  int count;
  int64_t units;            // total units over all spectra (or entries of unit_list)
  const int32_t* unit_list; // single spectrum only: ascending units g*Z + z to compute, or nullptr: all
  int V, h;
  // full planes (set by the launch): CTA k starts at unit k * span + min(k, span_extra) of a count in
  // which every segment group has group_cost units more than its templates
  int64_t span;
  int span_extra;
  int group_cost = 0;
  // with unit_list: per entry, bit j = segment j of the unit's group is computed (nullptr: all)
  const uint16_t* unit_mask = nullptr;
};

// The work-list instantiation's parameters: a BatchParams plus the list length in device memory
// (read by the kernel), or nullptr: `units` entries.  A separate type keeps the full-plane kernel's
// parameters, and so its code, free of the work-list fields.
struct ListParams : BatchParams {
  const int64_t* unit_count = nullptr;
};

// Parameters of the pair-list kernel: one spectrum restricted to a list of (segment s, template
// z) pairs, entries s*Z + z in ascending order, cut into equal contiguous ranges, one per warp.
struct PairParams {
  const float2* spec;       // n_bins complex64, 16-byte aligned
  float* plane;             // Z x n_bins float32, row pitch n_bins
  const float2* templates;  // Z x L template spectra (pair-major layout)
  const float2* twist;      // L inter-pass twiddles (twist_re)
  int* status;              // device status word (kStatusTimeout | kStatusBadList)
  const int32_t* pairs;     // ascending entries s*Z + z
  const int64_t* pair_count;  // list length in device memory (checked), or nullptr: n_pairs
  int64_t n_pairs;          // entries, or the list's capacity with pair_count
  int64_t n_bins;
  int64_t nseg;             // ceil(n_bins / V)
  int Z, V, h;
};

// Parameters of the forward-transform-only kernel (steps a2 + a3, for tests).
struct SegParams {
  const float2* twist;
  const float2* spectrum_in; // n_bins complex64 (read by bulk copies)
  float2* out;              // nseg x L, natural order
  int* status;
  int64_t n_bins;
  int64_t nseg;
  int V, h;
};

// Threads per transform group (N1) used for segment length L; the template bank is stored in the layout
// of that decomposition (element k = k1 + N1*k2 at ((k2/2)*N1 + k1)*2 + k2%2).
int conv_group_threads(int L);

// Segments per group of a full plane at 1024, 4096 and 8192, at most `most` (those a CTA has room for): while
// every unit has an SM of its own, halved, since a CTA's warps then share its four schedulers with fewer others.
inline int wide_segments(int64_t nseg, int Z, int most, int sm_count) {
  int segs = most;
  while (segs > 1 && (nseg + segs / 2 - 1) / (segs / 2) * Z <= sm_count) segs /= 2;
  return segs;
}

// group_cost of a full plane at 2048 whose units outnumber its CTAs: what a group's start,
// its segments' copy and forward transforms, counts in units (10,000 cycles against 7,600 per position at
// 2048), so that a CTA whose range enters a second group gets fewer templates.  2, unless that makes the
// longest range longer than 1 does; 0 where equal ranges end with the groups.  With 1 throughout, a CTA of
// two groups was the last one on planes of a few positions per CTA: 49,152 x 201 at 2048 30.2 us, now 28.7.
inline int group_cost_of(int64_t units, int64_t ngroups, int64_t grid) {
  if (units % grid == 0 && grid % ngroups == 0) return 0;
  const auto longest = [&](int cost) { return (units + cost * ngroups + grid - 1) / grid; };
  return longest(2) == longest(1) ? 2 : 1;
}
// a / b for a >= 0, in 32 bits where a fits.
__host__ __device__ __forceinline__ int64_t quotient(int64_t a, int b) {
  return (uint64_t)a <= 0xffffffffull ? (int64_t)((uint32_t)a / (uint32_t)b) : a / b;
}
// First unit of CTA k in that count, Z units per group; p: a struct with span, span_extra and group_cost
// (ConvParams, BatchParams).
template <class P>
__host__ __device__ __forceinline__ int64_t first_unit_of(const P& p, int Z, unsigned k) {
  const int64_t v = (int64_t)k * p.span + (k < (unsigned)p.span_extra ? k : (unsigned)p.span_extra);
  if (p.group_cost == 0) return v;
  const int per = Z + p.group_cost;
  const int64_t g = quotient(v, per);
  const int64_t r = v - g * per - p.group_cost;
  return g * Z + (r > 0 ? r : 0);
}

// Float offset of the real part of the twiddle exp(+i 2pi n2 k1 / L), n2 < N2 = 2*h2, k1 < n1, in the plan's
// table (the imaginary part is 2 floats further): a float4 (re, re, im, im) holds n2 = j and j + h2.  The
// kernels whose lanes own column pairs of the second pass (n1 <= h2: 256, 512 and 2048) read the pair of
// column j = r*n1 + t for one k1 at a time, lane t: entry (r*n1 + k1)*n1 + t.  The others read one k1 or
// one column per lane (the table is symmetric where n1 = N2): entry j*n1 + k1.  Either way a warp's load is
// one contiguous row; with the second order in all of them a warp touched 32 lines per load, which cost a
// CTA's start 3,400 cycles at 2048 and 11,500 at 4096 (4096 bins, one template: 14.4 us where it takes 12.3,
// and 20.5 us where it takes 12.4).
__host__ __device__ inline int twist_re(int n2, int k1, int n1, int h2) {
  const int j = n2 % h2, e = n1 <= h2 ? (j / n1 * n1 + k1) * n1 + j % n1 : j * n1 + k1;
  return 4 * e + n2 / h2;
}

// Segments resident per CTA of the descriptor-driven kernel for segment length L, or 0 if L has
// no descriptor-driven kernel (then only the single-spectrum plan path serves it).
int batch_segments_per_cta(int L);
// Descriptor-driven launch (L with batch_segments_per_cta(L) > 0).
cudaError_t launch_batch(int L, const BatchParams& p, int sm_count, cudaStream_t stream);
// Single spectrum restricted to a work list of units g*Z + z (ascending).
cudaError_t launch_units(int L, const ConvParams& p, const int32_t* units, const uint16_t* masks, int64_t n_units, int sm_count,
                         cudaStream_t stream, const int64_t* d_count = nullptr);

// Whether segment length L has the pair-list kernel (one transform per warp: L = 2048).
bool pairs_supported(int L);
// Single spectrum restricted to a list of pairs s*Z + z (checked on the device first).
cudaError_t launch_pairs(int L, const PairParams& p, int sm_count, cudaStream_t stream);

// Launch helpers (defined in fdas_convolve.cu).  Return a cudaError_t from the launch.  The segment length
// alone picks the kernel: 2048 and the short ones give every lane a pair of columns of the second pass
// (16-byte exchange entries); 1024, 4096 and 8192 have as many lanes as columns or more
// (fdas_convolve_wide.cu; 1024 with pairs of columns, 16 lanes and everything in shared memory took 611
// us where it now takes 482).
cudaError_t launch_convolve(int L, const ConvParams& p, int sm_count, cudaStream_t stream);
cudaError_t launch_segment_spectra(int L, const SegParams& p, int sm_count, cudaStream_t stream);
// Tensor-core variant for L = 2048 (fdas_tc.cu): inverse transforms as DFT-matrix contractions.
struct TcParams {
  const float2* seg;        // nseg x 2048 forward segment spectra, natural order (inverse pass)
  float2* seg_out;          // the same, written by the forward pass
  const float2* spectrum;   // n_bins complex64 (forward pass)
  const float2* bank;       // Z x 2048 template spectra, natural order
  const float2* twist;      // the plan's twist table
  const unsigned char* mats;  // DFT matrices of the precision and direction, operand layout (hi, lo)
  const unsigned* tmax;     // bits of max |Re|, |Im| over the bank
  float* plane;
  int* status;
  int64_t n_bins;
  int64_t nseg;
  int64_t units;            // inverse: nseg x ceil(Z / 4); forward: ceil(nseg / 4)
  int Z, V, h;
};
// Bytes of one set of DFT matrices; the workspace holds four sets: inverse BF16, inverse FP16,
// forward BF16, forward FP16.
int tc_matrices_bytes();
cudaError_t launch_tc_prepare(const float2* bank, int Z, float2* nat, unsigned* tmax, unsigned char* mats,
                              cudaStream_t stream);
// forward = true: the segment transforms (spectrum -> seg_out); false: the correlation (seg -> plane).
cudaError_t launch_tc(const TcParams& p, int precision, bool forward, int sm_count, cudaStream_t stream);

// Segment lengths 1024, 4096 and 8192 (fdas_convolve_wide.cu).
cudaError_t launch_convolve_wide(int L, const ConvParams& p, int sm_count, cudaStream_t stream);
cudaError_t launch_segment_spectra_wide(int L, const SegParams& p, int sm_count, cudaStream_t stream);

}  // namespace fdas

namespace fdas {
// Used by the allocation-free entry point (defined in fdas_api.cu).
int validate_geometry(int64_t n_bins, int zmax, int zstep, int seg_len, int tmpl_len);
// Step a1 (defined in fdas_templates.cu): taps, template spectra and twiddle table.
cudaError_t build_templates_into(double2* taps, float2* templates, float2* twist, int zmax, int zstep, int L,
                                 int m, cudaStream_t st);
// One thread waits, for at most limit_ns, on a barrier nothing completes and sets kStatusTimeout.
cudaError_t launch_wait_selftest(int* status, int64_t limit_ns, cudaStream_t st);
}  // namespace fdas

// ---------------------------------------------------------------------------------------
// The z-band network on windows (fdas_train.cu): FP32 forward, backward and Adam.
// ---------------------------------------------------------------------------------------
namespace fdas {

constexpr int kNetC = 32;   // channels
constexpr int kNetK = 9;    // kernel taps

// Flat parameter layout (floats).
struct NetLayout {
  int Z, W1, b1, W2, b2, W3, b3, Wl, bl, total;
  explicit NetLayout(int z) : Z(z) {
    W1 = 0;
    b1 = W1 + kNetC * 1 * kNetK;
    W2 = b1 + kNetC;
    b2 = W2 + kNetC * kNetC * kNetK;
    W3 = b2 + kNetC;
    b3 = W3 + kNetC * kNetC * kNetK;
    Wl = b3 + kNetC;
    bl = Wl + Z * kNetC;
    total = bl + Z;
  }
};

// Packed copies of the 32 x 32 x 9 weights, each [32 inputs of the pass][9 taps][32 outputs].
enum { kPackW2, kPackW3, kPackW2Back, kPackW3Back, kPackW2Half, kPackW3Half, kNetPacks };

// The inference kernel's FP16 image of the weights of layers 2 and 3: [layer][4 planes of 8 input
// channels][480 rows][8], row 32 b + o = output channel o of tap 11 - b, zero where that is no tap (the
// stack [0 0 0 W_8 ... W_0 0 0 0] of fdas_zband.cu).
constexpr int kStackRows = 15 * kNetC;
constexpr int kStackHalves = 2 * 4 * kStackRows * 8;
__host__ __device__ inline int stack_at(int layer, int o, int i, int k) {
  return ((layer * 4 + (i >> 3)) * kStackRows + (11 - k) * kNetC + o) * 8 + (i & 7);
}

struct NetState {
  NetLayout lay{0};
  int W = 0;
  float* p = nullptr;          // FP32 master parameters
  __half* ph = nullptr;        // FP16 copy for inference
  float* pr = nullptr;         // the FP16 copy's values as FP32
  __half* stack = nullptr;     // kStackHalves: layers 2 and 3 for the inference kernel (of ph)
  float* packs = nullptr;      // kNetPacks packed weight matrices (of p, and of pr: *Half)
  float* g = nullptr;          // gradients
  float* m = nullptr;          // Adam moments
  float* v = nullptr;
  float* h1 = nullptr;         // activations [B][32] rows of W: W/2 + 160 used,
  float* h2 = nullptr;         // W/2 + 128 used
  float* d2 = nullptr;         // gradient of layer 2's pre-activations, as h2
  float* pool = nullptr;       // per-tile maxima and positions of layer 3
  int* pool_arg = nullptr;
  float* pooled = nullptr;     // [B][32]
  float* seed = nullptr;       // [B][32] gradient of the pooled maxima
  int* arg = nullptr;          // [B][32]
  float* logits = nullptr;     // [B][Z]
  float* dlog = nullptr;       // [B][Z]
  float* loss = nullptr;       // device scalar
  float* loss_part = nullptr;  // [B]
  float* db2_part = nullptr;   // [B][32]
  float* part1 = nullptr;      // weight-gradient partials of the three layers (sum1: layer 1's, summed once)
  float* sum1 = nullptr;
  float* part2 = nullptr;
  float* part3 = nullptr;
  float* gl = nullptr;         // head gradients
};

// Element counts of the buffers whose size is not plain from their shape.
struct NetSizes {
  size_t act, pool, part1, sum1, part2, part3, gl, packs;
};
NetSizes net_sizes(int W, int Z, int max_batch);
cudaError_t net_prepare();   // function attributes, once per created net
// The copies (ph, pr, stack, packs) of the parameters p.
void net_publish(const NetState& s, cudaStream_t st);
cudaError_t net_predict(const NetState& s, const float* windows, int B, bool half_weights, float* logits,
                        cudaStream_t st);
// One step of Adam (`step` counts from 1); gradients in g, the loss in *loss.
cudaError_t net_train_step(const NetState& s, const float* windows, const float* targets, int B, float lr, int step,
                           cudaStream_t st);

}  // namespace fdas
