// fdas_api.cu -- the C ABI of libfdas (declared in include/fdas.h): plan life cycle, argument
// validation and the launch of the fused kernel.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>

#include <cuda_runtime.h>

#include "fdas.h"
#include "fdas_device.cuh"
#include "fdas_internal.h"

struct fdas_plan {
  int device = 0;
  int sm_count = 0;
  int64_t n_bins = 0;
  int zmax = 0, zstep = 1, L = 0, m = 0, h = 0, V = 0, Z = 0;
  int64_t nseg = 0;
  int n1 = 0;                        // lanes per transform group for this L
  void* memory = nullptr;            // one allocation holding the four buffers below
  float2* d_templates = nullptr;     // Z x L complex64, IFFT first-pass layout
  double2* d_taps = nullptr;         // Z x (m+1) complex128 normalised taps
  float2* d_twist = nullptr;         // L complex64 inter-pass twiddles (twist_re)
  int* d_status = nullptr;
  bool built = false;
  // tensor-core variant (fdas_convolve_power_tc), allocated on its first call
  float2* tc_bank = nullptr;         // Z x L natural-order template spectra
  float2* tc_seg = nullptr;          // nseg x L forward segment spectra of the current call
  unsigned char* tc_mats = nullptr;  // DFT matrices, BF16 then FP16
  unsigned* tc_tmax = nullptr;
  bool tc_ready = false;
  // completion of the last work this plan enqueued (fdas_destroy and the introspection calls wait
  // on it instead of on the whole device)
  cudaEvent_t done = nullptr;
};

namespace {

thread_local int g_last_error = FDAS_OK;

// Float offset of the real part of element k in the pair-major structure-of-arrays layout
// (lane k1 = k % n1, k2 = k / n1; pair p = k2/2 of lane k1 is the float4 at p*n1 + k1 holding
// re(2p), re(2p+1), im(2p), im(2p+1)); the imaginary part is 2 floats further.
int pair_layout_re(int k, int n1) {
  const int k1 = k % n1, k2 = k / n1;
  return ((k2 >> 1) * n1 + k1) * 4 + (k2 & 1);
}

// Failure-detection self test: one thread waits, with the given bound, on an mbarrier whose
// phase nothing completes, and records the timeout in the status word exactly as the fused
// kernel does.  The wait ends by itself; the context stays usable.
__global__ void wait_selftest_kernel(int* status, unsigned long long limit_ns) {
  __shared__ uint64_t bar;
  fdas::mbar_init(&bar, 1);
  fdas::fence_barrier_init();
  if (!fdas::mbar_wait(&bar, 0, limit_ns)) atomicOr(status, fdas::kStatusTimeout);
}

bool is_pow2(int x) { return x > 0 && (x & (x - 1)) == 0; }

int validate(int64_t n_bins, int zmax, int zstep, int seg_len, int tmpl_len) {
  if (n_bins < 4 || n_bins % 4 != 0 || n_bins > (int64_t(1) << 30)) return FDAS_ERR_INVALID;
  if (zstep < 1 || zmax < 0 || zmax % zstep != 0) return FDAS_ERR_INVALID;
  if (2 * (int64_t)(zmax / zstep) + 1 > 65535) return FDAS_ERR_INVALID;
  if (!is_pow2(seg_len) || seg_len < FDAS_MIN_SEG_LEN || seg_len > FDAS_MAX_SEG_LEN) return FDAS_ERR_INVALID;
  if (tmpl_len < 4 || tmpl_len % 4 != 0 || tmpl_len > seg_len / 2) return FDAS_ERR_INVALID;
  return FDAS_OK;
}

// Record the plan's completion event after work enqueued on `st` (skipped while the stream is
// being captured into a CUDA graph: a captured record is not an event the host can wait on).
int note_work(fdas_plan* p, cudaStream_t st) {
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &cs) != cudaSuccess) return FDAS_ERR_CUDA;
  if (cs != cudaStreamCaptureStatusNone) return FDAS_OK;
  return cudaEventRecord(p->done, st) == cudaSuccess ? FDAS_OK : FDAS_ERR_CUDA;
}
int enqueued(fdas_plan* p, cudaStream_t st, cudaError_t launch) {
  if (launch != cudaSuccess) return FDAS_ERR_CUDA;
  return note_work(p, st);
}

void free_tc_memory(fdas_plan* p) {
  cudaFree(p->tc_bank);
  cudaFree(p->tc_seg);
  cudaFree(p->tc_mats);
  cudaFree(p->tc_tmax);
  p->tc_bank = nullptr;
  p->tc_seg = nullptr;
  p->tc_mats = nullptr;
  p->tc_tmax = nullptr;
  p->tc_ready = false;
}

void free_plan_memory(fdas_plan* p) {
  free_tc_memory(p);
  if (p->done) cudaEventDestroy(p->done);
  p->done = nullptr;
  cudaFree(p->memory);
  p->memory = nullptr;
}

}  // namespace

extern "C" {

const char* fdas_error_string(int code) {
  switch (code) {
    case FDAS_OK: return "ok";
    case FDAS_ERR_INVALID: return "invalid argument";
    case FDAS_ERR_ALIGN: return "misaligned pointer";
    case FDAS_ERR_NOT_BUILT: return "templates not built (call fdas_templates_build first)";
    case FDAS_ERR_ALLOC: return "device allocation failed";
    case FDAS_ERR_CUDA: return "CUDA runtime or launch error";
    case FDAS_ERR_NO_DEVICE: return "no CUDA device";
    case FDAS_ERR_UNSUPPORTED: return "device is not compute capability 10.3 (GB300)";
    case FDAS_ERR_TIMEOUT: return "a bounded device-side wait gave up";
    default: return "unknown fdas status";
  }
}

int fdas_last_error(void) { return g_last_error; }

fdas_plan* fdas_plan_create(int64_t n_bins, int zmax, int zstep, int seg_len, int tmpl_len) {
  g_last_error = FDAS_OK;
  int rc = validate(n_bins, zmax, zstep, seg_len, tmpl_len);
  if (rc != FDAS_OK) {
    g_last_error = rc;
    return nullptr;
  }
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev < 1) {
    cudaGetLastError();
    g_last_error = FDAS_ERR_NO_DEVICE;
    return nullptr;
  }
  int dev = 0, major = 0, minor = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
    g_last_error = FDAS_ERR_CUDA;
    return nullptr;
  }
  if (major != 10 || minor != 3) {
    g_last_error = FDAS_ERR_UNSUPPORTED;
    return nullptr;
  }
  fdas_plan* p = new (std::nothrow) fdas_plan();
  if (!p) {
    g_last_error = FDAS_ERR_ALLOC;
    return nullptr;
  }
  p->device = dev;
  p->sm_count = sms;
  p->n_bins = n_bins;
  p->zmax = zmax;
  p->zstep = zstep;
  p->L = seg_len;
  p->m = tmpl_len;
  p->h = tmpl_len / 2;
  p->V = seg_len - tmpl_len;
  p->Z = 2 * (zmax / zstep) + 1;
  p->nseg = (n_bins + p->V - 1) / p->V;
  p->n1 = fdas::conv_group_threads(seg_len);
  const size_t ntap = (size_t)tmpl_len + 1;
  auto round256 = [](size_t x) { return (x + 255) / 256 * 256; };
  const size_t off_taps = round256(sizeof(float2) * (size_t)p->Z * p->L);
  const size_t off_twist = off_taps + round256(sizeof(double2) * (size_t)p->Z * ntap);
  const size_t off_status = off_twist + round256(sizeof(float2) * (size_t)p->L);
  if (cudaMalloc(&p->memory, off_status + sizeof(int)) != cudaSuccess ||
      cudaEventCreateWithFlags(&p->done, cudaEventDisableTiming) != cudaSuccess) {
    cudaGetLastError();
    free_plan_memory(p);
    delete p;
    g_last_error = FDAS_ERR_ALLOC;
    return nullptr;
  }
  unsigned char* base = static_cast<unsigned char*>(p->memory);
  p->d_templates = reinterpret_cast<float2*>(base);
  p->d_taps = reinterpret_cast<double2*>(base + off_taps);
  p->d_twist = reinterpret_cast<float2*>(base + off_twist);
  p->d_status = reinterpret_cast<int*>(base + off_status);
  // cleared before any stream can use the plan (a non-blocking stream is not ordered after
  // default-stream work)
  if (cudaMemsetAsync(p->d_status, 0, sizeof(int), 0) != cudaSuccess || cudaStreamSynchronize(0) != cudaSuccess) {
    free_plan_memory(p);
    delete p;
    g_last_error = FDAS_ERR_CUDA;
    return nullptr;
  }
  return p;
}

int fdas_templates_build(fdas_plan* p, fdas_stream_t stream) {
  if (!p) return FDAS_ERR_INVALID;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  if (fdas::build_templates_into(p->d_taps, p->d_templates, p->d_twist, p->zmax, p->zstep, p->L, p->m, st) !=
      cudaSuccess)
    return FDAS_ERR_CUDA;
  p->built = true;
  p->tc_ready = false;   // the tensor-core variant copies the bank again on its next call
  return note_work(p, st);
}

int fdas_convolve_power(fdas_plan* p, const float* d_spectrum, float* d_plane, fdas_stream_t stream) {
  if (!p || !d_spectrum || !d_plane) return FDAS_ERR_INVALID;
  if (!p->built) return FDAS_ERR_NOT_BUILT;
  if ((reinterpret_cast<uintptr_t>(d_spectrum) & 15u) || (reinterpret_cast<uintptr_t>(d_plane) & 15u))
    return FDAS_ERR_ALIGN;
  fdas::ConvParams q;
  q.spectrum = reinterpret_cast<const float2*>(d_spectrum);
  q.templates = p->d_templates;
  q.twist = p->d_twist;
  q.plane = d_plane;
  q.status = p->d_status;
  q.n_bins = p->n_bins;
  q.nseg = p->nseg;
  q.Z = p->Z;
  q.V = p->V;
  q.h = p->h;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  return enqueued(p, st, fdas::launch_convolve(p->L, q, p->sm_count, st));
}

int fdas_plan_group_segments(const fdas_plan* p) {
  if (!p) return FDAS_ERR_INVALID;
  const int G = fdas::batch_segments_per_cta(p->L);
  return G > 0 ? G : FDAS_ERR_INVALID;
}

int fdas_convolve_power_units_masked(fdas_plan* p, const float* d_spectrum, float* d_plane,
                                     const int32_t* d_units, const uint16_t* d_masks, int64_t n_units,
                                     fdas_stream_t stream) {
  if (!p || !d_spectrum || !d_plane || !d_units || n_units < 1) return FDAS_ERR_INVALID;
  if (!p->built) return FDAS_ERR_NOT_BUILT;
  if (fdas::batch_segments_per_cta(p->L) == 0) return FDAS_ERR_INVALID;
  if ((reinterpret_cast<uintptr_t>(d_spectrum) & 15u) || (reinterpret_cast<uintptr_t>(d_plane) & 15u) ||
      (reinterpret_cast<uintptr_t>(d_units) & 3u) || (reinterpret_cast<uintptr_t>(d_masks) & 1u))
    return FDAS_ERR_ALIGN;
  fdas::ConvParams q;
  q.spectrum = reinterpret_cast<const float2*>(d_spectrum);
  q.templates = p->d_templates;
  q.twist = p->d_twist;
  q.plane = d_plane;
  q.status = p->d_status;
  q.n_bins = p->n_bins;
  q.nseg = p->nseg;
  q.Z = p->Z;
  q.V = p->V;
  q.h = p->h;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  return enqueued(p, st, fdas::launch_units(p->L, q, d_units, d_masks, n_units, p->sm_count, st));
}

int fdas_convolve_power_units_device_count(fdas_plan* p, const float* d_spectrum, float* d_plane,
                                           const int32_t* d_units, const uint16_t* d_masks, const int64_t* d_count,
                                           int64_t max_units, fdas_stream_t stream) {
  if (!p || !d_spectrum || !d_plane || !d_units || !d_count || max_units < 1) return FDAS_ERR_INVALID;
  if (!p->built) return FDAS_ERR_NOT_BUILT;
  if (fdas::batch_segments_per_cta(p->L) == 0) return FDAS_ERR_INVALID;
  if ((reinterpret_cast<uintptr_t>(d_spectrum) & 15u) || (reinterpret_cast<uintptr_t>(d_plane) & 15u) ||
      (reinterpret_cast<uintptr_t>(d_units) & 3u) || (reinterpret_cast<uintptr_t>(d_masks) & 1u) ||
      (reinterpret_cast<uintptr_t>(d_count) & 7u))
    return FDAS_ERR_ALIGN;
  fdas::ConvParams q;
  q.spectrum = reinterpret_cast<const float2*>(d_spectrum);
  q.templates = p->d_templates;
  q.twist = p->d_twist;
  q.plane = d_plane;
  q.status = p->d_status;
  q.n_bins = p->n_bins;
  q.nseg = p->nseg;
  q.Z = p->Z;
  q.V = p->V;
  q.h = p->h;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  return enqueued(p, st, fdas::launch_units(p->L, q, d_units, d_masks, max_units, p->sm_count, st, d_count));
}

int fdas_convolve_power_units(fdas_plan* p, const float* d_spectrum, float* d_plane, const int32_t* d_units,
                              int64_t n_units, fdas_stream_t stream) {
  return fdas_convolve_power_units_masked(p, d_spectrum, d_plane, d_units, nullptr, n_units, stream);
}

namespace {
int convolve_pairs(fdas_plan* p, const float* d_spectrum, float* d_plane, const int32_t* d_pairs,
                   const int64_t* d_count, int64_t n_pairs, fdas_stream_t stream) {
  if (!p || !d_spectrum || !d_plane || !d_pairs || n_pairs < 1) return FDAS_ERR_INVALID;
  if (!p->built) return FDAS_ERR_NOT_BUILT;
  if (!fdas::pairs_supported(p->L)) return FDAS_ERR_INVALID;
  if ((reinterpret_cast<uintptr_t>(d_spectrum) & 15u) || (reinterpret_cast<uintptr_t>(d_plane) & 15u) ||
      (reinterpret_cast<uintptr_t>(d_pairs) & 3u) || (reinterpret_cast<uintptr_t>(d_count) & 7u))
    return FDAS_ERR_ALIGN;
  fdas::PairParams q;
  q.spec = reinterpret_cast<const float2*>(d_spectrum);
  q.plane = d_plane;
  q.templates = p->d_templates;
  q.twist = p->d_twist;
  q.status = p->d_status;
  q.pairs = d_pairs;
  q.pair_count = d_count;
  q.n_pairs = n_pairs;
  q.n_bins = p->n_bins;
  q.nseg = p->nseg;
  q.Z = p->Z;
  q.V = p->V;
  q.h = p->h;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  return enqueued(p, st, fdas::launch_pairs(p->L, q, p->sm_count, st));
}
}  // namespace

int fdas_convolve_power_pairs(fdas_plan* p, const float* d_spectrum, float* d_plane, const int32_t* d_pairs,
                              int64_t n_pairs, fdas_stream_t stream) {
  return convolve_pairs(p, d_spectrum, d_plane, d_pairs, nullptr, n_pairs, stream);
}

int fdas_convolve_power_pairs_device_count(fdas_plan* p, const float* d_spectrum, float* d_plane,
                                           const int32_t* d_pairs, const int64_t* d_count, int64_t max_pairs,
                                           fdas_stream_t stream) {
  if (!d_count) return FDAS_ERR_INVALID;
  return convolve_pairs(p, d_spectrum, d_plane, d_pairs, d_count, max_pairs, stream);
}

int fdas_segment_spectra(fdas_plan* p, const float* d_spectrum, float* d_out, fdas_stream_t stream) {
  if (!p || !d_spectrum || !d_out) return FDAS_ERR_INVALID;
  if (!p->built) return FDAS_ERR_NOT_BUILT;
  if ((reinterpret_cast<uintptr_t>(d_spectrum) & 15u) || (reinterpret_cast<uintptr_t>(d_out) & 15u))
    return FDAS_ERR_ALIGN;
  fdas::SegParams q;
  q.twist = p->d_twist;
  q.spectrum_in = reinterpret_cast<const float2*>(d_spectrum);
  q.out = reinterpret_cast<float2*>(d_out);
  q.status = p->d_status;
  q.n_bins = p->n_bins;
  q.nseg = p->nseg;
  q.V = p->V;
  q.h = p->h;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  return enqueued(p, st, fdas::launch_segment_spectra(p->L, q, p->sm_count, st));
}

namespace {

// The tensor-core variant's workspace, allocated and filled on the first call after a template
// build: natural-order bank, its max |Re|, |Im|, the four sets of DFT matrices, the segment
// spectra.
int tc_ensure_ready(fdas_plan* p, cudaStream_t st) {
  if (p->tc_ready) return FDAS_OK;
  free_tc_memory(p);
  const int mb = fdas::tc_matrices_bytes();
  if (cudaMalloc(&p->tc_bank, sizeof(float2) * (size_t)p->Z * p->L) != cudaSuccess ||
      cudaMalloc(&p->tc_seg, sizeof(float2) * (size_t)p->nseg * p->L) != cudaSuccess ||
      cudaMalloc(&p->tc_mats, 4 * (size_t)mb) != cudaSuccess ||
      cudaMalloc(&p->tc_tmax, sizeof(unsigned)) != cudaSuccess) {
    cudaGetLastError();
    free_tc_memory(p);
    return FDAS_ERR_ALLOC;
  }
  if (fdas::launch_tc_prepare(p->d_templates, p->Z, p->tc_bank, p->tc_tmax, p->tc_mats, st) != cudaSuccess)
    return FDAS_ERR_CUDA;
  p->tc_ready = true;
  return FDAS_OK;
}

fdas::TcParams tc_params(const fdas_plan* p, const float* d_spectrum, int precision, bool forward) {
  const int mb = fdas::tc_matrices_bytes();
  fdas::TcParams q;
  q.seg = p->tc_seg;
  q.seg_out = p->tc_seg;
  q.spectrum = reinterpret_cast<const float2*>(d_spectrum);
  q.bank = p->tc_bank;
  q.twist = p->d_twist;
  q.mats = p->tc_mats + (size_t)mb * ((forward ? 2 : 0) + (precision == FDAS_TC_FP16 ? 1 : 0));
  q.tmax = p->tc_tmax;
  q.plane = nullptr;
  q.status = p->d_status;
  q.n_bins = p->n_bins;
  q.nseg = p->nseg;
  q.units = forward ? (p->nseg + 3) / 4 : p->nseg * (int64_t)((p->Z + 3) / 4);
  q.Z = p->Z;
  q.V = p->V;
  q.h = p->h;
  return q;
}

int tc_validate(fdas_plan* p, const void* a, const void* b, int precision) {
  if (!p || !a || !b || (precision != FDAS_TC_BF16 && precision != FDAS_TC_FP16)) return FDAS_ERR_INVALID;
  if (!p->built) return FDAS_ERR_NOT_BUILT;
  if (p->L != 2048) return FDAS_ERR_INVALID;
  if ((reinterpret_cast<uintptr_t>(a) & 15u) || (reinterpret_cast<uintptr_t>(b) & 15u)) return FDAS_ERR_ALIGN;
  return FDAS_OK;
}

}  // namespace

int fdas_convolve_power_tc(fdas_plan* p, const float* d_spectrum, float* d_plane, int precision,
                           fdas_stream_t stream) {
  int rc = tc_validate(p, d_spectrum, d_plane, precision);
  if (rc != FDAS_OK) return rc;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  if ((rc = tc_ensure_ready(p, st)) != FDAS_OK) return rc;
  if (fdas::launch_tc(tc_params(p, d_spectrum, precision, true), precision, true, p->sm_count, st) != cudaSuccess)
    return FDAS_ERR_CUDA;
  fdas::TcParams q = tc_params(p, d_spectrum, precision, false);
  q.plane = d_plane;
  return enqueued(p, st, fdas::launch_tc(q, precision, false, p->sm_count, st));
}

int fdas_segment_spectra_tc(fdas_plan* p, const float* d_spectrum, float* d_out, int precision,
                            fdas_stream_t stream) {
  int rc = tc_validate(p, d_spectrum, d_out, precision);
  if (rc != FDAS_OK) return rc;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  if ((rc = tc_ensure_ready(p, st)) != FDAS_OK) return rc;
  fdas::TcParams q = tc_params(p, d_spectrum, precision, true);
  q.seg_out = reinterpret_cast<float2*>(d_out);
  return enqueued(p, st, fdas::launch_tc(q, precision, true, p->sm_count, st));
}

int fdas_check(fdas_plan* p, fdas_stream_t stream) {
  if (!p) return FDAS_ERR_INVALID;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  int status = 0;
  if (cudaMemcpyAsync(&status, p->d_status, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    return FDAS_ERR_CUDA;
  if (status != 0) {
    // cleared in the stream's order, before the call returns
    if (cudaMemsetAsync(p->d_status, 0, sizeof(int), st) != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess)
      return FDAS_ERR_CUDA;
    return (status & fdas::kStatusTimeout) ? FDAS_ERR_TIMEOUT : FDAS_ERR_INVALID;
  }
  return FDAS_OK;
}

int fdas_selftest_wait_timeout(fdas_plan* p, int64_t limit_ns, fdas_stream_t stream) {
  if (!p || limit_ns < 1000 || limit_ns > 2000000000LL) return FDAS_ERR_INVALID;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  return enqueued(p, st, fdas::launch_wait_selftest(p->d_status, limit_ns, st));
}

int fdas_destroy(fdas_plan* p) {
  if (!p) return FDAS_OK;
  if (p->done) cudaEventSynchronize(p->done);   // the plan's last enqueued work, not the whole device
  free_plan_memory(p);
  delete p;
  return FDAS_OK;
}

int fdas_plan_dims(const fdas_plan* p, int* Z, int* V, int64_t* nseg) {
  if (!p) return FDAS_ERR_INVALID;
  if (Z) *Z = p->Z;
  if (V) *V = p->V;
  if (nseg) *nseg = p->nseg;
  return FDAS_OK;
}

int fdas_template_taps(fdas_plan* p, int z_idx, double* host_out) {
  if (!p || !host_out || z_idx < 0 || z_idx >= p->Z) return FDAS_ERR_INVALID;
  if (!p->built) return FDAS_ERR_NOT_BUILT;
  const size_t ntap = (size_t)p->m + 1;
  if (cudaEventSynchronize(p->done) != cudaSuccess) return FDAS_ERR_CUDA;
  if (cudaMemcpy(host_out, p->d_taps + (size_t)z_idx * ntap, sizeof(double2) * ntap, cudaMemcpyDeviceToHost) !=
      cudaSuccess)
    return FDAS_ERR_CUDA;
  return FDAS_OK;
}

int fdas_template_spectrum(fdas_plan* p, int z_idx, float* host_out) {
  if (!p || !host_out || z_idx < 0 || z_idx >= p->Z) return FDAS_ERR_INVALID;
  if (!p->built) return FDAS_ERR_NOT_BUILT;
  if (cudaEventSynchronize(p->done) != cudaSuccess) return FDAS_ERR_CUDA;
  float2* tmp = static_cast<float2*>(std::malloc(sizeof(float2) * (size_t)p->L));
  if (!tmp) return FDAS_ERR_ALLOC;
  if (cudaMemcpy(tmp, p->d_templates + (size_t)z_idx * p->L, sizeof(float2) * (size_t)p->L,
                 cudaMemcpyDeviceToHost) != cudaSuccess) {
    std::free(tmp);
    return FDAS_ERR_CUDA;
  }
  const float* f = reinterpret_cast<const float*>(tmp);
  for (int k = 0; k < p->L; ++k) {
    const int off = pair_layout_re(k, p->n1);
    host_out[2 * k] = f[off];
    host_out[2 * k + 1] = f[off + 2];
  }
  std::free(tmp);
  return FDAS_OK;
}

}  // extern "C"

// ---------------------------------------------------------------------------------------
// Helpers for the allocation-free entry point (fdas_static.cu): the plan-based calls' validation and
// wait self test.
// ---------------------------------------------------------------------------------------
namespace fdas {

int validate_geometry(int64_t n_bins, int zmax, int zstep, int seg_len, int tmpl_len) {
  return validate(n_bins, zmax, zstep, seg_len, tmpl_len);
}

cudaError_t launch_wait_selftest(int* status, int64_t limit_ns, cudaStream_t st) {
  wait_selftest_kernel<<<1, 1, 0, st>>>(status, (unsigned long long)limit_ns);
  return cudaGetLastError();
}

}  // namespace fdas
