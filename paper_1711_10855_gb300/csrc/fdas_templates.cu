// fdas_templates.cu -- step a1: the FP64 template bank, once per plan.
//
// The raw response H_q(z) = int_0^1 exp(i pi (z u^2 - (z + 2q) u)) du is the q-th Fourier coefficient
// of the chirp f(u) = exp(-i pi z u (1 - u)) on [0, 1].  With [0, 1] cut into M equal panels and an
// n-point Gauss-Legendre rule (nodes xi_g, weights w_g on [0, 1]) in each,
//
//   H_q(z) = (1/M) sum_g w_g e^{-2 pi i q xi_g / M} F_g[q mod M],  F_g = DFT_M of f((p + xi_g) / M), p < M,
//
// so one M-point FFT per node gives every tap.  f(u) = f(1 - u) pairs node xi with 1 - xi (its F is
// e^{2 pi i q / M} F_g[-q]), so half of the nodes are sampled.  The symmetries H_q(z) = H_{-q}(z)
// and H_q(-z) = conj H_q(z) leave z >= 0, q >= 0 to compute.  The route is independent of the
// Fresnel closed form.
//
// The normalised, conjugated taps form an even sequence c_q, so the template spectrum is
//   T_z[k] = (1/L) e^{2 pi i k h / L} S[k],   S = DFT_L(c) (even in k),   T_{-z}[k] = (1/L) e^{2 pi i k h / L} conj S[k]
// (the conjugated template placed at circular index q + h: the correlation's valid outputs are the
// first V of each segment).
//
// One CTA per z >= 0 does all of it in shared memory.  It is bound by the FP64 units (2 lanes per SM
// and clock): about 2e5 FP64 operations per z at the survey geometry (Z = 201, m = 512, L = 2048).
// Measured there: 0.089 ms; a composite quadrature of every (z, q) by its own sincospi calls and a
// direct DFT of the taps (about 2e10 operations) took 62 ms.  L = 8192, m = 2048, Z = 401: 0.58 ms.
#include <cstdint>

#include <cuda_runtime.h>

#include "fdas_device.cuh"
#include "fdas_internal.h"

namespace {

constexpr int kNodes = 32;       // Gauss-Legendre points per panel
constexpr int kHalf = kNodes / 2;
constexpr int kThreads = 256;
constexpr int kTwistPer = 1024;  // twiddles per extra CTA
// Phase a panel may turn by, at most: the n-point rule's error for e^{i w x} on [-1, 1] is below
// 1e-24 at w = 20 (half the panel's phase) and n = 32.
constexpr double kPanelPhase = 40.0;
constexpr int kMaxPanels = 8192; // longer ones (zmax beyond about 1e5) are summed tap by tap
constexpr size_t kMaxSmem = 232448;

// Positive half of the rule on [0, 1]: x[g] = (1 + node)/2 of the negative nodes, by Newton iteration
// on the Legendre polynomial P_n (three-term recurrence), at compile time.
struct GaussRule {
  double x[kHalf], w[kHalf];
  constexpr GaussRule() : x(), w() {
    for (int i = 0; i < kHalf; ++i) {
      const double a = fdas::kPi * (i + 0.75) / (kNodes + 0.5);   // in (0, pi/2)
      double z = a <= fdas::kPi / 4 ? fdas::taylor_cos(a) : fdas::taylor_sin(fdas::kPi / 2 - a);
      double dp = 0.0;
      for (int it = 0; it < 12; ++it) {
        double p0 = 1.0, p1 = z;
        for (int k = 2; k <= kNodes; ++k) {
          const double p2 = ((2.0 * k - 1.0) * z * p1 - (k - 1.0) * p0) / k;
          p0 = p1;
          p1 = p2;
        }
        dp = kNodes * (z * p1 - p0) / (z * z - 1.0);
        z -= p1 / dp;
      }
      x[i] = 0.5 - 0.5 * z;
      w[i] = 1.0 / ((1.0 - z * z) * dp * dp);   // half of the weight on [-1, 1]
    }
  }
};
__constant__ constexpr GaussRule c_gauss{};

__device__ __forceinline__ double2 zmul(double2 a, double2 b) {
  return make_double2(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ double2 cispi(double t) {   // e^{i pi t}
  double s, c;
  sincospi(t, &s, &c);
  return make_double2(c, s);
}

// In-place radix-2 DIT stages on `count` transforms of M points (bit-reversed on entry), each at
// buf + t*M; W[k] = e^{-2 pi i k / N}, k < N/2.  All threads; ends with a barrier.
__device__ void fft_inplace(double2* buf, int M, int count, const double2* W, int N) {
  const int half = M / 2, total = count * half;
  for (int span = 1; span < M; span <<= 1) {
    const int stride = N / (2 * span);
    for (int i = threadIdx.x; i < total; i += kThreads) {
      const int t = i / half, r = i - t * half;
      const int k = r & (span - 1);
      double2* a = buf + t * M + ((r - k) << 1) + k;
      double2* b = a + span;
      const double2 va = *a, vb = *b;
      if (span == 1) {
        *a = make_double2(va.x + vb.x, va.y + vb.y);
        *b = make_double2(va.x - vb.x, va.y - vb.y);
      } else {
        const double2 w = W[k * stride];
        const double pr = fma(-w.y, vb.y, fma(w.x, vb.x, va.x));
        const double pi = fma(w.y, vb.x, fma(w.x, vb.y, va.y));
        *a = make_double2(pr, pi);
        *b = make_double2(fma(2.0, va.x, -pr), fma(2.0, va.y, -pi));
      }
    }
    __syncthreads();
  }
}

// Float offset of the real part of element k in the pair-major structure-of-arrays layout
// (lane k1 = k % n1, k2 = k / n1; pair p = k2/2 of lane k1 is the float4 at p*n1 + k1 holding
// re(2p), re(2p+1), im(2p), im(2p+1)); the imaginary part is 2 floats further.
__device__ __forceinline__ int layout_re(int k, int n1) {
  const int k1 = k % n1, k2 = k / n1;
  return ((k2 >> 1) * n1 + k1) * 4 + (k2 & 1);
}

struct BankShape {
  int zmax, zstep, L, h, n1;
  int M;      // panels, a power of two; 0: the taps are in `taps` already
  int N;      // twiddle period: max(L, M)
  int nbuf;   // entries of the work buffer
  int gc;     // nodes per chunk
};

// Inter-pass twiddles exp(+i 2pi n2 k1 / L), n2 < N2 = L/n1, k1 < n1, where twist_re puts them.
__device__ void write_twist(float2* tw, int idx, int L, int n1) {
  const int k1 = idx % n1, n2 = idx / n1;
  const double2 w = cispi(2.0 * (double)(((long long)n2 * k1) % L) / (double)L);
  float* dst = reinterpret_cast<float*>(tw);
  const int off = fdas::twist_re(n2, k1, n1, L / n1 / 2);
  dst[off] = (float)w.x;
  dst[off + 2] = (float)w.y;
}

// CTA j <= zmax/zstep: templates +-j*zstep (taps rows and spectra).  Further CTAs: twiddles.
// Shared memory: W[N/2] | buf[nbuf] | H[h + 1] | red[kThreads].
__global__ void __launch_bounds__(kThreads) template_bank_kernel(double2* taps, float2* templates, float2* twist,
                                                                 const BankShape b) {
  extern __shared__ double2 sm2[];
  const int tid = threadIdx.x, zc = b.zmax / b.zstep, j = blockIdx.x;
  const int L = b.L, h = b.h, N = b.N;
  if (j > zc) {
    for (int i = tid; i < kTwistPer; i += kThreads) {
      const int idx = (j - zc - 1) * kTwistPer + i;
      if (idx < L) write_twist(twist, idx, L, b.n1);
    }
    return;
  }
  double2* W = sm2;
  double2* buf = W + N / 2;
  double2* H = buf + b.nbuf;
  double* red = reinterpret_cast<double*>(H + h + 1);
  const int ntap = 2 * h + 1;
  double2* row_p = taps + (size_t)(zc + j) * ntap;
  double2* row_n = taps + (size_t)(zc - j) * ntap;

  // W[32a + f] = W[32a] W[f]: one sincospi per 32 entries and 32 more
  const int nf = N / 2 < 32 ? N / 2 : 32, na = N / 2 / nf;
  for (int i = tid; i < nf + na; i += kThreads) {
    const int k = i < nf ? i : (i - nf) * nf;
    buf[i] = cispi(-2.0 * (double)k / (double)N);
  }
  __syncthreads();
  for (int i = tid; i < N / 2; i += kThreads) W[i] = zmul(buf[i % nf], buf[nf + i / nf]);
  __syncthreads();

  if (b.M) {
    const int M = b.M, lg = 31 - __clz(M), na16 = h / 16 + 1;
    const double z = (double)j * (double)b.zstep, invM = 1.0 / (double)M;
    for (int q = tid; q <= h; q += kThreads) H[q] = make_double2(0.0, 0.0);
    for (int g0 = 0; g0 < kHalf; g0 += b.gc) {
      // samples of the chirp at (p + xi_g)/M, bit-reversed; e^{-2 pi i q xi_g / M} for q = 16a and q < 16
      double2* ea = buf + b.gc * M;
      double2* eb = ea + b.gc * na16;
      const int ns = b.gc * M, na_all = b.gc * na16;
      for (int i = tid; i < ns + na_all + b.gc * 16; i += kThreads) {
        if (i < ns) {
          const int g = i >> lg, p = i & (M - 1);
          const double u = ((double)p + c_gauss.x[g0 + g]) * invM;
          buf[(g << lg) + (M > 1 ? (int)(__brev((unsigned)p) >> (32 - lg)) : 0)] = cispi(-z * (u * (1.0 - u)));
        } else if (i < ns + na_all) {
          const int e = i - ns, g = e / na16, a = e - g * na16;
          ea[e] = cispi(-2.0 * (double)(16 * a) * c_gauss.x[g0 + g] * invM);
        } else {
          const int e = i - ns - na_all, g = e >> 4, f = e & 15;
          eb[e] = cispi(-2.0 * (double)f * c_gauss.x[g0 + g] * invM);
        }
      }
      __syncthreads();
      fft_inplace(buf, M, b.gc, W, N);
      for (int q = tid; q <= h; q += kThreads) {
        const int qp = q & (M - 1), qn = (M - qp) & (M - 1);
        double re = H[q].x, im = H[q].y;
        for (int g = 0; g < b.gc; ++g) {
          const double2 e = zmul(ea[g * na16 + (q >> 4)], eb[g * 16 + (q & 15)]);
          const double2 fp = buf[g * M + qp], fn = buf[g * M + qn];
          const double w = c_gauss.w[g0 + g];
          // e fp + conj(e) fn
          re = fma(w, fma(e.x, fp.x + fn.x, -e.y * (fp.y - fn.y)), re);
          im = fma(w, fma(e.x, fp.y + fn.y, e.y * (fp.x - fn.x)), im);
        }
        H[q] = make_double2(re, im);
      }
      __syncthreads();
    }
    // unit L2 norm over q = -h..h (the 1/M drops out)
    double part = 0.0;
    for (int q = tid; q <= h; q += kThreads)
      part += (q ? 2.0 : 1.0) * fma(H[q].x, H[q].x, H[q].y * H[q].y);
    red[tid] = part;
    __syncthreads();
    for (int s = kThreads / 2; s > 0; s >>= 1) {
      if (tid < s) red[tid] += red[tid + s];
      __syncthreads();
    }
    const double scale = 1.0 / sqrt(red[0]);
    for (int q = tid; q <= h; q += kThreads) {
      const double2 v = make_double2(H[q].x * scale, H[q].y * scale);
      H[q] = v;
      row_p[h + q] = row_p[h - q] = v;
      if (j) row_n[h + q] = row_n[h - q] = make_double2(v.x, -v.y);
    }
  } else {
    for (int q = tid; q <= h; q += kThreads) H[q] = row_p[h + q];
  }
  __syncthreads();

  // S = DFT_L of c_q = conj H_q (even), zero-extended; h <= L/4, so q and L - q do not meet
  const int lgL = 31 - __clz(L);
  for (int i = tid; i < L; i += kThreads) {
    const int q = i <= L / 2 ? i : L - i;
    double2 v = make_double2(0.0, 0.0);
    if (q <= h) v = make_double2(H[q].x, -H[q].y);
    buf[__brev((unsigned)i) >> (32 - lgL)] = v;
  }
  __syncthreads();
  fft_inplace(buf, L, 1, W, N);
  float* tp = reinterpret_cast<float*>(templates + (size_t)(zc + j) * L);
  float* tn = reinterpret_cast<float*>(templates + (size_t)(zc - j) * L);
  const double inv = 1.0 / (double)L;
  for (int k = tid; k < L; k += kThreads) {
    const int t = (int)(((long long)k * h) & (L - 1));            // e^{2 pi i t / L}
    double2 ph = W[(t & (L / 2 - 1)) * (N / L)];
    ph = t & (L / 2) ? make_double2(-ph.x, ph.y) : make_double2(ph.x, -ph.y);
    const double2 s = buf[k];
    const int off = layout_re(k, b.n1);
    tp[off] = (float)(fma(ph.x, s.x, -ph.y * s.y) * inv);
    tp[off + 2] = (float)(fma(ph.x, s.y, ph.y * s.x) * inv);
    if (j) {
      tn[off] = (float)(fma(ph.x, s.x, ph.y * s.y) * inv);
      tn[off + 2] = (float)(fma(-ph.x, s.y, ph.y * s.x) * inv);
    }
  }
}

// zmax so large that the panels of one node exceed kMaxPanels: every tap by its own composite
// quadrature, one CTA per z.
__global__ void __launch_bounds__(kThreads) taps_kernel(double2* taps, int zmax, int zstep, int h) {
  const int zi = blockIdx.x;
  const double z = (double)(-zmax + zi * zstep);
  const int ntap = 2 * h + 1;
  double2* row = taps + (size_t)zi * ntap;
  double part = 0.0;
  for (int j = threadIdx.x; j < ntap; j += blockDim.x) {
    const double q = (double)(j - h);
    const double bq = z + 2.0 * q;
    const int panels = (int)ceil(fdas::kPi * (fabs(z) + 2.0 * fabs(q) + 1.0) / 20.0) + 1;
    const double width = 1.0 / panels;
    double re = 0.0, im = 0.0;
    for (int k = 0; k < panels; ++k) {
      double pr = 0.0, pi = 0.0;
      for (int g = 0; g < kNodes; ++g) {
        const double xi = g < kHalf ? c_gauss.x[g] : 1.0 - c_gauss.x[g - kHalf];
        const double u = (k + xi) * width;
        const double2 e = cispi(z * u * u - bq * u);
        const double w = c_gauss.w[g < kHalf ? g : g - kHalf];
        pr = fma(w, e.x, pr);
        pi = fma(w, e.y, pi);
      }
      re += pr;
      im += pi;
    }
    re *= width;
    im *= width;
    row[j] = make_double2(re, im);
    part += re * re + im * im;
  }
  __shared__ double red[kThreads];
  red[threadIdx.x] = part;
  __syncthreads();
  for (int s = kThreads / 2; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
    __syncthreads();
  }
  const double scale = 1.0 / sqrt(red[0]);
  for (int j = threadIdx.x; j < ntap; j += blockDim.x) {
    const double2 v = row[j];
    row[j] = make_double2(v.x * scale, v.y * scale);
  }
}

}  // namespace

namespace fdas {

cudaError_t build_templates_into(double2* taps, float2* templates, float2* twist, int zmax, int zstep, int L, int m,
                                 cudaStream_t st) {
  BankShape b;
  b.zmax = zmax;
  b.zstep = zstep;
  b.L = L;
  b.h = m / 2;
  b.n1 = conv_group_threads(L);
  // the fastest phase of f(u) e^{-2 pi i q u} turns by 2 pi (z/2 + q) over [0, 1]
  const double turn = 2.0 * kPi * (0.5 * (double)zmax + (double)b.h);
  int64_t M = 8;
  while ((double)M * kPanelPhase < turn) M *= 2;
  const int extra = b.h / 16 + 17;   // e^{-2 pi i q xi / M} tables of one node
  size_t smem = 0;
  b.M = M <= kMaxPanels ? (int)M : 0;
  for (;; b.M = 0) {   // M = 0 always fits: L/2 + L + L/4 + 1 entries at most
    b.N = b.M > L ? b.M : L;
    b.nbuf = b.M + extra > L ? b.M + extra : L;
    smem = sizeof(double2) * ((size_t)b.N / 2 + b.nbuf + b.h + 1) + sizeof(double) * kThreads;
    if (smem <= kMaxSmem || !b.M) break;
  }
  b.gc = 1;
  while (b.M && b.gc < kHalf && 2 * b.gc * (b.M + extra) <= b.nbuf) b.gc *= 2;
  // the same limit whatever the shape: threads that build different banks at once do not undo each other's
  cudaError_t e =
      cudaFuncSetAttribute(template_bank_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem);
  if (e != cudaSuccess) return e;
  if (!b.M) taps_kernel<<<2 * (zmax / zstep) + 1, kThreads, 0, st>>>(taps, zmax, zstep, b.h);
  const int grid = zmax / zstep + 1 + (L + kTwistPer - 1) / kTwistPer;
  template_bank_kernel<<<grid, kThreads, smem, st>>>(taps, templates, twist, b);
  return cudaGetLastError();
}

}  // namespace fdas
