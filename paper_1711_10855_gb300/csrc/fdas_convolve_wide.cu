// fdas_convolve_wide.cu -- the fused correlation (steps a2..a7 of Eq. 2 by overlap-and-save, Section 2)
// with one column of the second pass per lane: segment lengths 1024 (one warp per transform), 4096
// (two warps) and 8192 (four warps).
//
// Transform of length L = N1 * N2 by N1 = 32 * WT lanes, N2 points per lane (four-step):
//   pass 1: lane k1 holds Y[k1 + N1*k2], k2 < N2, as N2/2 packed pairs: N2-point DFT in registers,
//   exchange: row n2 of a shared-memory tile holds the N1 values of that column, two neighbouring k1
//           per 16-byte entry (re, re, im, im), so that pass 2 reads packed pairs with 128-bit loads,
//   twist:  multiply by exp(SIGN i 2pi n2 k1 / L), joined with the first stage of
//   pass 2: lane (n2) runs the N1-point DFT of its column as a split pair; output n = n2 + N2*n1.
//   L = 8192 has N1 = 2*N2: the twist comes before the exchange, and lane (n2, c) first forms Z[a] + Z[a + N1/2] (c = 0) or
//           (Z[a] - Z[a + N1/2]) W^a (c = 1) and runs an N2-point DFT: the outputs n1 = 2 n' + c.
// In the exchange a lane writes single 4-byte words; the (re, im) halves of every second group of
// eight entries are swapped, which puts a warp's 32 words on 32 banks.
//
// Segment spectra and twiddles sit in tensor memory, templates stream through a ring of shared-memory
// slots (whole templates or halves of them) that every warp of the CTA reads, as in fdas_convolve.cu.
// The warps of a transform meet at a named barrier before and after the exchange.
//
// The FP32 pipe bounds the kernel: 32 points a lane let 1024 run 16 warps of 128 registers, 64 points
// a lane 4096 and 8192 only 8, which wait at barriers and on the exchange together.  Measured, before
// (1024: everything in shared memory; 4096, 8192: Stockham passes through it with a CTA barrier each)
// and now: 3,000,004 x 101 at L = 1024, m = 256: 611, 481 us; 2^21 x 401 at 4096, m = 1024: 2822, 1843 us (236
// registers); 1,500,012 x 401 at 8192, m = 2048: 3151, 1626 us (255 registers, 20 bytes spilled).
//
// A CTA has room for 16 (1024), 4 or 2 segments.  On planes of few units it takes fewer (wide_segments), and
// warps without a segment only keep the barriers and the ring going.  What remains of a single position is
// straight-line code run once, from cold instruction caches: one template at 4096 takes 8 us of device time,
// where a kernel of short loops with 256 threads per transform took 5 at twice the error.
#include <cuda_runtime.h>

#include "fdas_conv_common.cuh"
#include "fdas_internal.h"

namespace fdas {
namespace {

template <int L_, int WT_, int N2_, int W_, int PARTS_, int R_>
struct WideCfg {
  static constexpr int L = L_;
  static constexpr int WT = WT_;             // warps per transform
  static constexpr int N1 = 32 * WT;         // lanes per transform
  static constexpr int N2 = N2_;             // points per lane
  static constexpr int H2 = N2 / 2;
  static constexpr int W = W_;               // warps per CTA
  static constexpr int G = W / WT;           // segments resident per CTA
  static constexpr int PARTS = PARTS_;       // ring slots per template
  static constexpr int R = R_;               // ring slots
  static constexpr bool PIPE = true;         // see multiply_first_stage
  static constexpr int SPLIT = N1 / N2;      // lanes per column of pass 2
  static constexpr int M = N1 / SPLIT;       // points of a lane's pass-2 DFT (= N2)
  static constexpr int LOG_N2 = ilog2(N2);
  static constexpr int KP = N1 / 2;          // entries per tile row
  static constexpr int PITCH = KP + 1;       // odd: 128-bit column reads are conflict-free
  static constexpr int PART_PAIRS = H2 / PARTS;
  static constexpr size_t PART_BYTES = (size_t)L * 8 / PARTS;
  static constexpr size_t TILE = (size_t)N2 * PITCH * 16;
  static constexpr size_t REGION = align_up(TILE > (size_t)L * 8 ? TILE : (size_t)L * 8, 128);
  static constexpr size_t OFF_T = 0;
  static constexpr size_t OFF_REG = OFF_T + R * PART_BYTES;
  static constexpr size_t OFF_BAR = OFF_REG + G * REGION;
  static constexpr size_t SMEM = OFF_BAR + 256;
  static constexpr uint32_t COL_TW = 0;      // TMEM columns of each quadrant
  static constexpr uint32_t COL_X = 2 * N2;
  static constexpr uint32_t TMEM_COLS = 512;
  static_assert(N1 * N2 == L && (SPLIT == 1 || SPLIT == 2) && W % 4 == 0 && 4 % WT == 0, "bad decomposition");
  static_assert(2 * N2 * (1 + W / 4) <= (int)TMEM_COLS, "TMEM columns");
  static_assert(SMEM <= 232448, "shared memory budget");
  static_assert(R * 20 + 48 <= 256, "barrier area");
};

// Twist before the exchange (split columns) with the twiddle pairs held in this lane's TMEM row.
template <class Cfg, bool CONJ>
__device__ __forceinline__ void apply_twist_tmem(cp2 (&v)[Cfg::H2], uint32_t tw_addr) {
  static_assert(Cfg::H2 % 8 == 0, "twist chunking");
  static_for<Cfg::H2 / 8>([&](auto cc) {
    constexpr int c = decltype(cc)::value;
    float r0[16], r1[16];
    tmem_ld16(tw_addr + 32 * c, r0);
    tmem_ld16(tw_addr + 32 * c + 16, r1);
    tmem_wait_ld();
    static_for<4>([&](auto qq) {
      constexpr int q = decltype(qq)::value;
      const cp2 w0 = cp2{make_float2(r0[4 * q], r0[4 * q + 1]), make_float2(r0[4 * q + 2], r0[4 * q + 3])};
      const cp2 w1 = cp2{make_float2(r1[4 * q], r1[4 * q + 1]), make_float2(r1[4 * q + 2], r1[4 * q + 3])};
      v[8 * c + q] = CONJ ? cmul2_conj(v[8 * c + q], w0) : cmul2(v[8 * c + q], w0);
      v[8 * c + 4 + q] = CONJ ? cmul2_conj(v[8 * c + 4 + q], w1) : cmul2(v[8 * c + 4 + q], w1);
    });
  });
}

template <class Cfg>
__device__ __forceinline__ void transform_sync(int g) {
  if constexpr (Cfg::WT == 1) __syncwarp();
  else asm volatile("bar.sync %0, %1;" ::"r"(g + 1), "n"(32 * Cfg::WT) : "memory");
}

// W^a pairs of the split second pass: exp(SIGN i 2pi a / N1) for a = 2 kappa, 2 kappa + 1.
template <int N1, int SIGN, int A>
__device__ __forceinline__ cp2 split_twiddle() {
  constexpr CosSin a = cossin_2pi(A, N1), b = cossin_2pi(A + 1, N1);
  return cp2{make_float2((float)a.c, (float)b.c), make_float2((float)(SIGN * a.s), (float)(SIGN * b.s))};
}

// Exchange and pass 2.  On exit u[j] = (y[r0 + RS*j], y[r0 + RS*(j + M/2)]) in rows n1 of column n2,
// with RS = SPLIT and r0 = c.
template <class Cfg, int SIGN>
__device__ __forceinline__ void exchange_pass2(cp2 (&v)[Cfg::H2], cp2 (&u)[Cfg::M / 2], float4* tile, int g, int k1,
                                               int n2, int c, uint32_t tw_addr) {
  if constexpr (Cfg::SPLIT == 2) apply_twist_tmem<Cfg, (SIGN < 0)>(v, tw_addr);
  const int kappa = k1 >> 1, sw = (kappa >> 3) & 1;
  float* wr = reinterpret_cast<float*>(tile) + 4 * kappa + (k1 & 1);
  float* w_re = wr + 2 * sw;
  float* w_im = wr + 2 * (1 - sw);
  transform_sync<Cfg>(g);   // the tile's (or the staged segment's) earlier reads are done
  static_for<Cfg::H2>([&](auto jj) {
    constexpr int j = decltype(jj)::value;
    w_re[j * Cfg::PITCH * 4] = v[j].re.x;
    w_im[j * Cfg::PITCH * 4] = v[j].im.x;
    w_re[(j + Cfg::H2) * Cfg::PITCH * 4] = v[j].re.y;
    w_im[(j + Cfg::H2) * Cfg::PITCH * 4] = v[j].im.y;
  });
  transform_sync<Cfg>(g);
  const float4* row = tile + n2 * Cfg::PITCH;
  auto entry = [&](auto kk) -> cp2 {
    constexpr int k = decltype(kk)::value;
    const float4 e = row[k];
    if constexpr ((k >> 3) & 1) return cp2{make_float2(e.z, e.w), make_float2(e.x, e.y)};
    else return cp2{make_float2(e.x, e.y), make_float2(e.z, e.w)};
  };
  constexpr int LOGM = ilog2(Cfg::M);
  if constexpr (Cfg::SPLIT == 1) {
    twist_first_stage<Cfg::M / 2, 1, (SIGN < 0), false, Cfg::PIPE>(u, tw_addr, entry);
    fft_split_pairs<Cfg::M, SIGN, 1>(u);
    return;
  } else if (c == 0) {
    static_for<Cfg::M / 2>([&](auto kk) {
      constexpr int k = decltype(kk)::value;
      const cp2 a = entry(kk), b = entry(std::integral_constant<int, k + Cfg::M / 2>{});
      u[bitrev(2 * k, LOGM)] = cp2{add2(a.re, b.re), add2(a.im, b.im)};
    });
  } else {
    static_for<Cfg::M / 2>([&](auto kk) {
      constexpr int k = decltype(kk)::value;
      const cp2 a = entry(kk), b = entry(std::integral_constant<int, k + Cfg::M / 2>{});
      u[bitrev(2 * k, LOGM)] =
          cmul2(cp2{sub2(a.re, b.re), sub2(a.im, b.im)}, split_twiddle<Cfg::N1, SIGN, 2 * k>());
    });
  }
  fft_split_pairs<Cfg::M, SIGN>(u);
}

// Twiddle pairs of a lane (the plan's table holds exp(i 2pi n2 k1 / L) for n2 = j, j + H2 as pair j of
// lane k1, contiguous over the lanes).  Split columns: that pair j.  Otherwise the pairs of k1 = 2 kappa,
// 2 kappa + 1 of the lane's column n2, in slot order; N1 = N2 makes the table symmetric, so they are the
// lane's own pairs with n2 and k1 exchanged.
template <class Cfg>
__device__ __forceinline__ void load_lane_twiddles(float4 (&tw)[Cfg::H2], const float2* twist, int lane_k1) {
  float4 own[Cfg::H2];
  const float4* tw4 = reinterpret_cast<const float4*>(twist);
  static_for<Cfg::H2>([&](auto jj) { own[decltype(jj)::value] = __ldg(tw4 + decltype(jj)::value * Cfg::N1 + lane_k1); });
  static_for<Cfg::H2>([&](auto ii) {
    constexpr int i = decltype(ii)::value, k = 2 * slot_pair(i, Cfg::H2);
    if constexpr (Cfg::SPLIT == 2) {
      tw[i] = own[i];
    } else if constexpr (k < Cfg::H2) {
      tw[i] = make_float4(own[k].x, own[k + 1].x, own[k].z, own[k + 1].z);
    } else {
      const float4 a = own[k - Cfg::H2], b = own[k + 1 - Cfg::H2];
      tw[i] = make_float4(a.y, b.y, a.w, b.w);
    }
  });
}

// NV (eighths of the rows): pass-2 rows n1 >= NV*N1/8 hold no valid output and are dropped at compile
// time.  FWD: only the forward transforms, natural order, into p.plane (complex64).
template <class Cfg, int NV, bool FWD>
__global__ void __launch_bounds__(32 * Cfg::W, 1) fdas_convolve_wide_kernel(const ConvParams p) {
  constexpr int L = Cfg::L, N1 = Cfg::N1, N2 = Cfg::N2, H2 = Cfg::H2, R = Cfg::R, W = Cfg::W;
  constexpr int M = Cfg::M, PARTS = Cfg::PARTS, RS = Cfg::SPLIT;
  extern __shared__ __align__(1024) unsigned char smem[];
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + Cfg::OFF_BAR);
  uint64_t* segbar = full + R;
  int64_t* issued_pos = reinterpret_cast<int64_t*>(segbar + 1);   // [R] last ring position issued per slot
  unsigned* cnt = reinterpret_cast<unsigned*>(issued_pos + R);    // [R] consumer arrivals per slot
  volatile int* abort_flag = reinterpret_cast<volatile int*>(cnt + R);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(cnt + R + 1);
  int* next_z = reinterpret_cast<int*>(cnt + R + 2);              // template of the next part to issue

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = warp / Cfg::WT, k1 = 32 * (warp % Cfg::WT) + lane;
  const int n2 = k1 & (N2 - 1);
  const int c_fwd = k1 / N2;                          // 0 unless a column is split
  const int c_inv = RS == 2 ? c_fwd ^ (g & 1) : 0;    // the c = 1 lanes' extra multiply spread over the schedulers
  unsigned char* region = smem + Cfg::OFF_REG + (size_t)g * Cfg::REGION;
  float2* mySeg = reinterpret_cast<float2*>(region);
  float4* tile = reinterpret_cast<float4*>(region);

  const int Z = FWD ? 1 : p.Z;
  const int64_t u0 = first_unit_of(p, Z, blockIdx.x), u1 = first_unit_of(p, Z, blockIdx.x + 1);
  const int64_t npos = u1 - u0;
  if (npos <= 0) return;
  int64_t grp = quotient(u0, Z);
  int z = (int)(u0 - grp * Z);

  // a2: bulk copies of the in-range part of every segment of the group, one lane per segment
  auto fetch_segments = [&]() {   // a whole warp
    const int64_t x0 = (grp * p.segs + lane) * (int64_t)p.V - p.h;
    const int64_t c0 = x0 > 0 ? x0 : 0, c1 = x0 + L < p.n_bins ? x0 + L : p.n_bins;
    const uint32_t bytes = lane < p.segs && c1 > c0 ? (uint32_t)((c1 - c0) * 8) : 0u;
    const uint32_t total = __reduce_add_sync(0xffffffffu, bytes);
    if (lane == 0) mbar_arrive_expect_tx(segbar, total);
    __syncwarp();
    if (bytes) {
      float2* dst = reinterpret_cast<float2*>(smem + Cfg::OFF_REG + (size_t)lane * Cfg::REGION);
      bulk_g2s(dst + (c0 - x0), p.spectrum + c0, bytes, segbar);
    }
  };
  // The first group's segments, the first templates, the twiddles and the tensor memory are asked for at
  // once by different warps.
  if (warp == 0) {
    if (lane == 0) {
      mbar_init(segbar, 1);
      *abort_flag = 0;
      fence_barrier_init();
    }
    __syncwarp();
    fetch_segments();
  } else if (warp == 1) {
    if (lane < R) {
      mbar_init(&full[lane], 1);
      cnt[lane] = 0u;
      issued_pos[lane] = -1;
      fence_barrier_init();
    }
    __syncwarp();
  } else if (warp == 2) {
    tmem_alloc(tmem_slot, Cfg::TMEM_COLS);
    tmem_relinquish();
  }

  // ring position e = PARTS * (unit - u0) + part
  auto issue_part = [&](int64_t e) {
    const int slot = (int)(e % R);
    const int zr = *next_z;   // parts are issued in order, one thread at a time
    if (PARTS == 1 || e % PARTS == PARTS - 1) *next_z = zr + 1 == Z ? 0 : zr + 1;
    issued_pos[slot] = e;
    mbar_arrive_expect_tx(&full[slot], (uint32_t)Cfg::PART_BYTES);
    unsigned char* dst = smem + Cfg::OFF_T + slot * Cfg::PART_BYTES;
    const unsigned char* src = reinterpret_cast<const unsigned char*>(p.templates + (size_t)zr * L);
    if constexpr (PARTS == 1) {
      bulk_g2s(dst, src, (uint32_t)Cfg::PART_BYTES, &full[slot]);
    } else {   // the part's pairs, then their partners half a template further
      constexpr uint32_t half = (uint32_t)(Cfg::PART_BYTES / 2);
      src += (e % PARTS) * half;
      bulk_g2s(dst, src, half, &full[slot]);
      bulk_g2s(dst + half, src + (size_t)L * 4, half, &full[slot]);
    }
  };
  if (!FWD && tid == 32) {
    *next_z = z;
    const int64_t first = npos * PARTS < R ? npos * PARTS : R;
    for (int64_t e = 0; e < first; ++e) issue_part(e);
  }
  // warps w, w + 4, ... hold the same lanes of their transforms (WT divides 4): one copy of the twiddles
  // per quadrant (stored once the tensor memory is there)
  float4 tw[H2];
  if (warp >= 4 && warp < 8) load_lane_twiddles<Cfg>(tw, p.twist, k1);
  tmem_fence_before_sync();
  __syncthreads();
  tmem_fence_after_sync();
  const uint32_t tmem_row = *tmem_slot + ((uint32_t)(32 * (warp & 3)) << 16);
  const uint32_t tw_addr = tmem_row + Cfg::COL_TW;
  const uint32_t x_addr = tmem_row + Cfg::COL_X + (uint32_t)(warp >> 2) * (2 * N2);
  if (warp >= 4 && warp < 8) twiddles_to_tmem<H2>(tw, tw_addr);
  tmem_fence_before_sync();

  int alive = 1;
  uint32_t seg_phase = 0;
  bool seg_in_flight = false;
  int64_t u = u0;
  while (u < u1) {
    const int64_t a = u - u0;
    const int64_t bpos = (u + (Z - z) < u1 ? u + (Z - z) : u1) - u0;
    u = u0 + bpos;
    if (a > 0) {
      // every warp is done with its region (previous exchanges) before segments land in it
      fence_proxy_async_smem();
      alive = __syncthreads_and(alive && !*abort_flag);
      tmem_fence_after_sync();
      if (!alive) break;
      if (warp == 0) fetch_segments();
    }
    const int64_t s = grp * p.segs + g;
    const int64_t segbase = s * (int64_t)p.V;
    // the warps of a transform without a segment only keep the barriers and the ring going
    const bool on = g < p.segs && s < p.nseg;
    if (on) zero_outside<L>(mySeg, segbase - p.h, p.n_bins, k1, N1);
    seg_in_flight = true;
    alive = __syncthreads_and(mbar_wait(segbar, seg_phase) ? 1 : 0);
    tmem_fence_after_sync();   // the twiddles were stored by other warps
    if (!alive) {
      if (tid == 0) report_timeout(p.status, abort_flag);
      break;
    }
    seg_in_flight = false;
    seg_phase ^= 1u;

    // a3: forward FFT; lane k1's elements X[k1 + N1*k2] end in the lane itself: pairs (2q, 2q + 1) to TMEM
    if (on) {
      cp2 v[H2], x[M / 2];
      static_for<H2>([&](auto ii) {
        constexpr int i = decltype(ii)::value;
        constexpr int k2 = bitrev(i, Cfg::LOG_N2);
        const float2 e0 = mySeg[k1 + N1 * k2], e1 = mySeg[k1 + N1 * (k2 + 1)];
        v[i] = cp2{make_float2(e0.x, e1.x), make_float2(e0.y, e1.y)};
      });
      fft_split_pairs<N2, -1>(v);
      exchange_pass2<Cfg, -1>(v, x, tile, g, k1, n2, c_fwd, tw_addr);
      if constexpr (FWD) {
        float2* out = reinterpret_cast<float2*>(p.plane) + s * L;
        static_for<M / 2>([&](auto jj) {
          constexpr int j = decltype(jj)::value;
          out[k1 + N1 * j] = make_float2(x[j].re.x, x[j].im.x);
          out[k1 + N1 * (j + M / 2)] = make_float2(x[j].re.y, x[j].im.y);
        });
      } else spectrum_to_tmem<H2>(x_addr, [&](auto pp) {
        constexpr int k2 = 2 * decltype(pp)::value;   // members k2 and k2 + 1: both in .x or both in .y
        constexpr int j = k2 < M / 2 ? k2 : k2 - M / 2;
        if constexpr (k2 < M / 2)
          return cp2{make_float2(x[j].re.x, x[j + 1].re.x), make_float2(x[j].im.x, x[j + 1].im.x)};
        else
          return cp2{make_float2(x[j].re.y, x[j + 1].re.y), make_float2(x[j].im.y, x[j + 1].im.y)};
      });
    }

    if constexpr (FWD) {
      ++grp;
      tmem_fence_before_sync();
      continue;
    }

    const int64_t lim64 = p.n_bins - segbase < (int64_t)p.V ? p.n_bins - segbase : (int64_t)p.V;
    int lim = lim64 > 0 ? (int)lim64 : 0;   // outputs n < lim of this segment are stored
    // release the slot of ring position e; the last of the W consumers refills it R positions ahead
    auto release_part = [&](int64_t e, int slot, int ok) {
      __syncwarp();
      if (lane == 0) {
        const unsigned old = arrive_count(&cnt[slot]);
        if ((old + 1u) % (unsigned)W == 0u && e + R < npos * PARTS && ok) {
          fence_proxy_async_smem();
          issue_part(e + R);
        }
      }
    };
    if (!on) {
      for (int64_t e = a * PARTS; e < bpos * PARTS; ++e) {
        const int slot = (int)(e % R);
        const int ok = __all_sync(0xffffffffu, wait_slot(&full[slot], (uint32_t)((e / R) & 1), abort_flag));
        if (!ok && lane == 0) report_timeout(p.status, abort_flag);
        release_part(e, slot, ok);
      }
    } else for (int64_t i = a; i < bpos; ++i, ++z) {
      // a4: Y = X (TMEM) * T (shared ring), packed pairs in bit-reversed order.  A wait that gives up ends
      // the stores, not the loop: the warps of a transform keep meeting at their barriers until the
      // group ends.
      cp2 v[H2];
      static_for<PARTS>([&](auto pp) {
        constexpr int part = decltype(pp)::value;
        const int64_t e = i * PARTS + part;
        const int slot = (int)(e % R);
        const int ok = __all_sync(0xffffffffu, wait_slot(&full[slot], (uint32_t)((e / R) & 1), abort_flag));
        if (!ok) {
          if (lane == 0) report_timeout(p.status, abort_flag);
          lim = 0;
        }
        const float4* st4 = reinterpret_cast<const float4*>(smem + Cfg::OFF_T + slot * Cfg::PART_BYTES);
        // a part holds its pairs p and their partners p + H2/2
        multiply_first_stage<Cfg, part * Cfg::PART_PAIRS / 2, Cfg::PART_PAIRS / 2>(v, x_addr, [&](int q) {
          constexpr int first = part * Cfg::PART_PAIRS / 2;
          return st4[(q < H2 / 2 ? q - first : q - H2 / 2 - first + Cfg::PART_PAIRS / 2) * N1 + k1];
        });
        release_part(e, slot, ok);
      });
      // a5: inverse FFT
      fft_split_pairs<N2, +1, 1>(v);
      cp2 y[M / 2];
      exchange_pass2<Cfg, +1>(v, y, tile, g, k1, n2, c_inv, tw_addr);
      // a6 + a7: keep n < V (and inside the spectrum), store |y|^2
      float* row = p.plane + (int64_t)z * p.n_bins + segbase;
      const int nb = n2 + N2 * c_inv;
      static_for<M / 2>([&](auto jj) {
        constexpr int j = decltype(jj)::value;
        constexpr int n_lo = N2 * RS * j, n_hi = N2 * RS * (j + M / 2);
        const float2 pw = power2(y[j]);
        if (nb + n_lo < lim) __stcs(row + nb + n_lo, pw.x);
        if constexpr (n_hi < L / 8 * NV) {
          if (nb + n_hi < lim) __stcs(row + nb + n_hi, pw.y);
        }
      });
    }
    ++grp;
    z = 0;
    tmem_fence_before_sync();
  }

  // After a timeout, wait (bounded) for this CTA's copies still in flight; always free TMEM.
  tmem_fence_before_sync();
  __syncthreads();
  tmem_fence_after_sync();
  if (tid == 0 && (*abort_flag || !alive)) {
    for (int r = 0; r < R; ++r)
      if (issued_pos[r] >= 0) (void)mbar_wait(&full[r], (uint32_t)((issued_pos[r] / R) & 1));
    if (seg_in_flight) (void)mbar_wait(segbar, seg_phase);
  }
  if (warp == 2) tmem_dealloc(*tmem_slot, Cfg::TMEM_COLS);
}

using Wide1024 = WideCfg<1024, 1, 32, 16, 1, 4>;
using Wide4096 = WideCfg<4096, 2, 64, 8, 2, 5>;
using Wide8192 = WideCfg<8192, 4, 64, 8, 2, 3>;

template <class Cfg, int NV, bool FWD>
cudaError_t launch_wide(const ConvParams& p, int sm_count, cudaStream_t st) {
  auto kern = fdas_convolve_wide_kernel<Cfg, NV, FWD>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg::SMEM);
  if (e != cudaSuccess) return e;
  ConvParams q = p;
  // With G segments per CTA always, and transforms of segments that do not exist, 4096 bins took: one template
  // at 4096 12.4 us (now 9.3) and at 8192 16.4 us (10.3), 201 templates at 1024 14.4 us (10.3).
  q.segs = FWD ? Cfg::G : wide_segments(p.nseg, p.Z, Cfg::G, sm_count);
  const int64_t ngroups = (p.nseg + q.segs - 1) / q.segs;
  const int64_t units = FWD ? ngroups : ngroups * p.Z;
  const int64_t grid = units < sm_count ? units : sm_count;
  q.group_cost = !FWD && units > grid ? 1 : 0;   // about one position (2: 4096 and 8192 0.5% slower)
  const int64_t total = units + q.group_cost * ngroups;
  q.span = total / grid;
  q.span_extra = (int)(total % grid);
  kern<<<(unsigned)grid, 32 * Cfg::W, Cfg::SMEM, st>>>(q);
  return cudaGetLastError();
}

template <class Cfg>
cudaError_t launch_wide_len(const ConvParams& p, int sm_count, cudaStream_t st) {
  if (4 * p.V <= 3 * Cfg::L) return launch_wide<Cfg, 6, false>(p, sm_count, st);   // m >= L/4
  return launch_wide<Cfg, 8, false>(p, sm_count, st);
}

}  // namespace

cudaError_t launch_convolve_wide(int L, const ConvParams& p, int sm_count, cudaStream_t st) {
  switch (L) {
    case 1024: return launch_wide_len<Wide1024>(p, sm_count, st);
    case 4096: return launch_wide_len<Wide4096>(p, sm_count, st);
    case 8192: return launch_wide_len<Wide8192>(p, sm_count, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_segment_spectra_wide(int L, const SegParams& p, int sm_count, cudaStream_t st) {
  ConvParams q{};
  q.spectrum = p.spectrum_in;
  q.twist = p.twist;
  q.plane = reinterpret_cast<float*>(p.out);
  q.status = p.status;
  q.n_bins = p.n_bins;
  q.nseg = p.nseg;
  q.Z = 1;
  q.V = p.V;
  q.h = p.h;
  switch (L) {
    case 1024: return launch_wide<Wide1024, 8, true>(q, sm_count, st);
    case 4096: return launch_wide<Wide4096, 8, true>(q, sm_count, st);
    case 8192: return launch_wide<Wide8192, 8, true>(q, sm_count, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace fdas
