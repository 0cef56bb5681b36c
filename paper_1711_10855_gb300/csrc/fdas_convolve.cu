// fdas_convolve.cu -- the fused FDAS correlation kernel for sm_103a.
//
// One launch computes the whole f-fdot power plane (Adamek et al. 2017, Section 1 Eq. 2, by
// the overlap-and-save method of Section 2):
//
//   a2  bulk copies (cp.async.bulk) bring the part inside [0, n_bins) of each segment's L bins
//       A[s*V - h .. s*V - h + L) into shared memory, the rest is zero-filled,
//   a3  forward FFT of the segment, kept in tensor memory for all Z templates,
//   a4  for every template z: multiply by the template spectrum T_z (streamed from L2 into a
//       ring of shared-memory slots by bulk copies),
//   a5  inverse FFT,
//   a6  keep outputs n < V (the template is placed so that circular wrap-around lands in the
//       last m outputs),
//   a7  |y|^2 stored with streaming (evict-first) stores into plane[z][s*V + n].
//
// Transform of length L = N1 * N2 by a group of N1 lanes, N2 points per lane (four-step):
//   pass 1: lane k1 holds Y[k1 + N1*k2], k2 < N2, as N2/2 packed pairs and does its N2-point DFT
//           in registers (two N2/2-point DFTs in lockstep with packed f32x2 butterflies, then one
//           scalar stage joining them),
//   exchange: one shared-memory transposition of 16-byte pair entries through a padded tile,
//   twist:  multiply by exp(SIGN i 2pi n2 k1 / L), joined with the first stage of
//   pass 2: lane t holds two columns n2 (a packed pair) and runs two N1-point DFTs in lockstep;
//           output index n = n2 + N2*n1, so lane t ends with outputs n = t (mod N1).
// The paper's design (Section 2: shuffle stage for N <= 32, shared memory above, 4 elements per
// thread) is replaced by two register passes with compile-time FMA butterflies on packed pairs
// and a single shared-memory exchange per transform.
//
// Work decomposition: a CTA owns G consecutive segments at a time ("group"); the flattened (group,
// z) list is split into contiguous equal ranges, one per CTA (grid = #SMs).  The FP32 pipe bounds the kernel:
// 71.8k lane operations per 2048-point transform, 0.98 ms per 2^22 x 201 plane of which 1.31 ms is
// measured (1.36 with separate products; DRAM writes at 38% of their rate).  L = 2048 holds 64 points a
// lane (8 warps of 217 registers); L = 256 and 512 hold 32 (16 warps of 128, P = 2 warps per segment
// on alternate templates: 3e6 x 51 at L = 512 takes 198 us against 244 with 8 warps and separate products,
// 1e6 x 17 at 256 35 against 45 with everything in shared memory).
#include <cstdio>
#include <type_traits>

#include "fdas_conv_common.cuh"
#include "fdas_internal.h"

// The decoupled work-list instantiation leaves the shared-ring loop of the kernel unreachable.
#pragma nv_diag_suppress 128

namespace fdas {

// ---------------------------------------------------------------------------------------
// Shared per-lane pieces of the transform
//
// Buffer layout of a segment spectrum and a template spectrum (L complex values each), "pair-major structure of arrays": lane k1 of the first pass owns the pairs
// p = 0..H2-1; pair p of lane k1 is the float4 at index p*N1 + k1 holding
// (re(e0), re(e1), im(e0), im(e1)).  For spectra and templates e0, e1 are the elements
// k = k1 + N1*(2p) and k1 + N1*(2p+1); the twiddle table's order is twist_re's.  One 128-bit load gives
// a packed pair ready for f32x2 arithmetic.
// ---------------------------------------------------------------------------------------

struct NoHook {
  __device__ __forceinline__ void operator()() const {}
};

// Exchange, twist and pass 2 with the twiddles in TMEM: round r moves the rows of column pair r, each
// lane multiplies its column's entries (lane s wrote entry s) by their twiddles and runs two N1-point
// DFTs in lockstep; out(r, u) receives u[n1] = (y[t + N1*r + N2*n1], y[t + N1*(r+CP) + N2*n1]).
template <class Cfg, int SIGN, class Out, class AfterReads = NoHook>
__device__ __forceinline__ void exchange_twist_pass2(const cp2 (&v)[Cfg::H2], float4* xb, int k1, uint32_t tw_addr,
                                                     Out&& out, AfterReads&& after_reads = AfterReads{}) {
  constexpr int N1 = Cfg::N1;
  static_for<Cfg::CP>([&](auto rr) {
    constexpr int r = decltype(rr)::value;
    cp2 u[N1];
    __syncwarp();
    static_for<N1>([&](auto ii) {
      constexpr int i = decltype(ii)::value;
      xb[i * Cfg::XPITCH + k1] = cp2_to(v[r * N1 + i]);
    });
    __syncwarp();
    twist_first_stage<N1, 0, (SIGN < 0), true, Cfg::PIPE>(u, tw_addr + 4 * N1 * r, [&](auto ss) {
      return cp2_from(xb[k1 * Cfg::XPITCH + decltype(ss)::value]);
    });
    if constexpr (r == Cfg::CP - 1) after_reads();   // the tile is free once its last round is read
    fft_pair_columns<N1, SIGN, 1>(u);
    out(rr, u);
  });
}

// Forward FFT (Eq. 3) of one segment held in natural order (complex64) in sx; out as in
// exchange_twist_pass2: u[n1] = (X[t + N1*r + N2*n1], X[t + N1*(r+CP) + N2*n1]).
template <class Cfg, class Out>
__device__ __forceinline__ void forward_transform(const float2* sx, float4* xb, int k1, uint32_t tw_addr, Out&& out) {
  cp2 v[Cfg::H2];
  static_for<Cfg::H2>([&](auto ii) {
    constexpr int i = decltype(ii)::value;
    constexpr int k2 = bitrev(i, Cfg::LOG_N2);
    const float2 a = sx[k1 + Cfg::N1 * k2];
    const float2 b = sx[k1 + Cfg::N1 * (k2 + 1)];
    v[i] = cp2{make_float2(a.x, b.x), make_float2(a.y, b.y)};
  });
  fft_split_pairs<Cfg::N2, -1>(v);
  exchange_twist_pass2<Cfg, -1>(v, xb, k1, tw_addr, out);
}
// The same into this lane's TMEM slots: the pairs (k2 = 2p, 2p + 1) of the elements X[k1 + N1*k2].
template <class Cfg>
__device__ __forceinline__ void forward_to_tmem(const float2* sx, float4* xb, int k1, uint32_t tw_addr,
                                                uint32_t x_addr) {
  constexpr int N1 = Cfg::N1;
  cp2 first[Cfg::CP == 2 ? N1 : 1];   // two column pairs: round 0's, until round 1's complete the pairs
  forward_transform<Cfg>(sx, xb, k1, tw_addr, [&](auto rr, auto& x) {
    if constexpr (Cfg::CP == 1) {      // pair p = n1
      spectrum_to_tmem<Cfg::H2>(x_addr, [&](auto pp) { return x[decltype(pp)::value]; });
    } else if constexpr (decltype(rr)::value == 0) {   // elements k2 = 4 n1, 4 n1 + 2
      static_for<N1>([&](auto nn) { first[decltype(nn)::value] = x[decltype(nn)::value]; });
    } else {                                           // and 4 n1 + 1, 4 n1 + 3
      spectrum_to_tmem<Cfg::H2>(x_addr, [&](auto pp) {
        constexpr int n1 = decltype(pp)::value >> 1;
        if constexpr (decltype(pp)::value & 1)
          return cp2{make_float2(first[n1].re.y, x[n1].re.y), make_float2(first[n1].im.y, x[n1].im.y)};
        else
          return cp2{make_float2(first[n1].re.x, x[n1].re.x), make_float2(first[n1].im.x, x[n1].im.x)};
      });
    }
  });
}

// Twiddle pairs of lane k1's columns: entry r*N1 + slot = those of column pair r for the lane that
// slot stands for (contiguous over the lanes: twist_re).
template <class Cfg>
__device__ __forceinline__ void load_column_twiddles(float4 (&tw)[Cfg::H2], const float2* twist, int k1) {
  constexpr int N1 = Cfg::N1;
  const float4* tw4 = reinterpret_cast<const float4*>(twist);
  static_for<Cfg::H2>([&](auto ii) {
    constexpr int i = decltype(ii)::value, r = i / N1, src = slot_pair(i % N1, N1);
    tw[i] = __ldg(tw4 + (r * N1 + src) * N1 + k1);
  });
}

// ---------------------------------------------------------------------------------------
// The kernel: segment spectra and twiddle table in tensor memory (one column pair per lane at L = 512
// and 2048, two at 256).  Every warp holds its segment(s); the template of
// each position is read from the shared-memory ring by 8 warps.  Per inverse transform the
// shared-memory traffic is the template (L*8 bytes) and the exchange (2*L*8 bytes); the
// spectrum and the twiddles come from TMEM, a separate store, which relieves the shared-memory
// bandwidth that otherwise co-limits the kernel with the FP32 pipe.
// ---------------------------------------------------------------------------------------
template <int L_, int N1_, int W_ = 8, int P_ = 1>
struct TmemCfg {
  static constexpr int L = L_;
  static constexpr int N1 = N1_;
  static constexpr int N2 = L / N1;
  static constexpr int H2 = N2 / 2;
  static constexpr int F = 32 / N1;
  static constexpr int W = W_;             // warps per CTA
  static constexpr int P = P_;             // warps sharing a segment, taking alternate templates
  static constexpr int G = F * W / P;      // segments resident per CTA: one group of lanes each
  static constexpr int R = 4;
  static constexpr bool PIPE = false;      // see multiply_first_stage
  static constexpr int C = N2 / N1;        // pass-2 columns per lane
  static constexpr int CP = C / 2;         // and column pairs (exchange rounds)
  static constexpr int XPITCH = N1 + 1;
  static constexpr int XGROUP = N1 * XPITCH;
  static constexpr int XWARP = F * XGROUP;
  static constexpr int LOG_N1 = ilog2(N1);
  static constexpr int LOG_N2 = ilog2(N2);
  // per-warp shared region: staging of its segments, then its exchange tiles
  static constexpr size_t REGION = align_up(((size_t)F * L * 8 > (size_t)XWARP * 16) ? (size_t)F * L * 8
                                                                                     : (size_t)XWARP * 16, 128);
  static constexpr size_t OFF_T = 0;
  static constexpr size_t OFF_REG = OFF_T + (size_t)R * L * 8;
  static constexpr size_t OFF_BAR = align_up(OFF_REG + (size_t)W * REGION, 128);
  static constexpr size_t SMEM = OFF_BAR + 256;
  // TMEM columns of each quadrant: twiddles, then the spectra of its segments' warps
  static constexpr uint32_t TMEM_COLS = 512;
  static constexpr uint32_t COL_TW = 0;
  static constexpr uint32_t COL_X = 2 * N2;
  static_assert((C == 2 || C == 4) && 32 % N1 == 0, "one or two column pairs per lane");
  static_assert(W % (4 * P) == 0 && (P == 1 || P == 2), "warps sharing a segment share a TMEM quadrant");
  static_assert(2 * N2 * (1 + W / P / 4) <= (int)TMEM_COLS, "TMEM columns");
  static_assert(SMEM <= 232448, "shared memory budget");
};

// a6 + a7: |y|^2 of the outputs n < lim of column pair r; rows n1 >= NV hold none.
template <class Cfg, int NV, int r>
__device__ __forceinline__ void store_powers(const cp2 (&y)[Cfg::N1], float* row, int k1, int lim) {
  static_for<NV>([&](auto nn) {
    constexpr int n1 = decltype(nn)::value;
    const float2 pw = power2(y[n1]);
    const int n_lo = r * Cfg::N1 + k1 + Cfg::N2 * n1;
    const int n_hi = n_lo + Cfg::CP * Cfg::N1;
    if (n_lo < lim) __stcs(row + n_lo, pw.x);
    if (n_hi < lim) __stcs(row + n_hi, pw.y);
  });
}

// Spectrum b holding flattened unit u (largest b with unit_base <= u).
__device__ __forceinline__ int find_spectrum(const BatchParams& p, int64_t u) {
  if (p.descs == nullptr) return 0;
  int lo = 0, hi = p.count - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (p.descs[mid].unit_base <= u) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}
__device__ __forceinline__ SpecDesc spectrum_desc(const BatchParams& p, int b) {
  return p.descs == nullptr ? p.single : p.descs[b];
}

// Units to compute: all of them, or the list length (from device memory when the list was made on
// the device; the check kernel has bounded it by the list's capacity p.units).
__device__ __forceinline__ int64_t unit_total(const BatchParams& p) { return p.units; }
__device__ __forceinline__ int64_t unit_total(const ListParams& p) { return p.unit_count ? *p.unit_count : p.units; }

// First unit of CTA k.  The units are cut into equal ranges; one spectrum's groups count group_cost
// units more each.  A batch's do not: with a template count per spectrum the counted units would need a base of
// their own in every descriptor.
__device__ __forceinline__ int64_t first_unit(const BatchParams& p, unsigned k) {
  return first_unit_of(p, p.single.Z, k);
}

// NV: pass-2 output rows n1 < NV can hold valid outputs (NV >= ceil(V / N2)); rows n1 >= NV are
// dropped at compile time, which also removes the butterfly halves that only feed them.
//
// Work: units (spectrum b, segment group g, template z) flattened over all spectra; each CTA
// takes a contiguous equal range.  Segment s of spectrum b is brought in by one bulk copy of its
// part inside [0, n_b) (cp.async.bulk) and the rest of the L-bin window is zero-filled by the
// owning warp.
//
// DEC (work lists with segment masks only): the warps are decoupled.  Instead of the shared
// template ring, each warp walks only the positions where one of its segments is listed and
// brings that position's template into its own shared region by a bulk copy, issued as soon as
// the region's exchange tile has been read (so it lands while the warp finishes the previous
// transform).  The time of a group is then set by its busiest warp, not by the number of listed
// units: sparse masks cost about their share of (segment, template) pairs.
template <class Cfg, int NV, bool LIST, bool DEC = false>
__global__ void __launch_bounds__(32 * Cfg::W, 1)
    fdas_convolve_tmem_kernel(const std::conditional_t<LIST, ListParams, BatchParams> p) {
  static_assert(!DEC || LIST, "decoupled warps serve masked work lists");
  static_assert(!LIST || Cfg::P == 1, "work lists: every warp walks every position");
  constexpr int L = Cfg::L, N1 = Cfg::N1, R = Cfg::R, G = Cfg::G, H2 = Cfg::H2, W = Cfg::W, P = Cfg::P;
  extern __shared__ __align__(1024) unsigned char smem[];
  float2* sT = reinterpret_cast<float2*>(smem + Cfg::OFF_T);
  unsigned char* sReg = smem + Cfg::OFF_REG;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + Cfg::OFF_BAR);
  uint64_t* segbar = full + R;
  int64_t* issued_pos = reinterpret_cast<int64_t*>(segbar + 1);
  unsigned* cnt = reinterpret_cast<unsigned*>(issued_pos + R);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(cnt + R);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(cnt + R + 1);
  // template-refill cursor, one per position parity with P = 2 (the positions of one parity are issued in
  // increasing order, one thread at a time)
  struct IssueCursor {
    int64_t u;          // unit of the next position to issue
    int64_t spec_end;   // first unit of the next spectrum
    int b, z, Z, z_off; // its spectrum, template index within it, that spectrum's Z and bank offset
  };
  IssueCursor* cur = reinterpret_cast<IssueCursor*>(smem + Cfg::OFF_BAR + 128);
  uint64_t* wbar = reinterpret_cast<uint64_t*>(smem + Cfg::OFF_BAR + 192);   // [W] per-warp template copies (DEC)

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int gw = lane / N1, k1 = lane % N1;
  // P = 2: warps w and w + 4 (one TMEM quadrant) hold the same segments and take alternate templates
  const int par = P == 2 ? (warp >> 2) & 1 : 0;
  const int wseg = P == 2 ? (warp & 3) + 4 * (warp >> 3) : warp;
  float2* myRegion = reinterpret_cast<float2*>(sReg + (size_t)warp * Cfg::REGION);
  float2* mySeg = myRegion + (size_t)gw * L;
  float4* myXb = reinterpret_cast<float4*>(myRegion) + gw * Cfg::XGROUP;

  // a work list that failed its check (kStatusBadList, set by the preceding check kernel) is not
  // run
  if constexpr (LIST) {
    if (*reinterpret_cast<volatile const int*>(p.status) & kStatusBadList) return;
  }
  const int64_t U = unit_total(p);
  // flattened unit of list entry e (identity without a work list)
  auto unit_at = [&](int64_t e) -> int64_t {
    if constexpr (LIST) return (int64_t)__ldg(p.unit_list + e);
    else return e;
  };
  int64_t u0, u1;
  if constexpr (LIST) {
    u0 = (int64_t)blockIdx.x * U / gridDim.x;
    u1 = ((int64_t)blockIdx.x + 1) * U / gridDim.x;
  } else {
    u0 = first_unit(p, blockIdx.x);
    u1 = first_unit(p, blockIdx.x + 1);
  }
  const int64_t npos = u1 - u0;
  if (npos <= 0) return;

  // the segment group holding entry u0
  int b = find_spectrum(p, unit_at(u0));
  const SpecDesc d0 = spectrum_desc(p, b);
  int64_t grp = quotient(unit_at(u0) - d0.unit_base, d0.Z);
  int64_t z_first = unit_at(u0) - d0.unit_base - grp * d0.Z;

  // a2: bulk copies of the in-range part of every segment of the group, one lane per segment (issued one
  // after the other by a single thread they took 430 cycles each)
  static_assert(G <= 32, "one lane per segment");
  auto fetch_segments = [&](const SpecDesc& d) {   // a whole warp
    const int64_t x0 = (grp * G + lane) * (int64_t)p.V - p.h;
    const int64_t c0 = x0 > 0 ? x0 : 0;
    const int64_t c1 = x0 + L < d.n_bins ? x0 + L : d.n_bins;
    const uint32_t bytes = lane < G && c1 > c0 ? (uint32_t)((c1 - c0) * 8) : 0u;
    const uint32_t total = __reduce_add_sync(0xffffffffu, bytes);
    if (lane == 0) mbar_arrive_expect_tx(segbar, total);
    __syncwarp();
    if (bytes) {
      const int ws = lane / Cfg::F, wj = P == 2 ? (ws & 3) + 8 * (ws >> 2) : ws;   // the segment's first warp
      float2* dst = reinterpret_cast<float2*>(sReg + (size_t)wj * Cfg::REGION) + (size_t)(lane % Cfg::F) * L;
      bulk_g2s(dst + (c0 - x0), d.spec + c0, bytes, segbar);
    }
  };

  // The first group's segments, the first templates, the twiddles and the tensor memory are asked for at
  // once by different warps.
  if (warp == 0) {
    if (lane == 0) {
      mbar_init(segbar, 1);
      if constexpr (DEC)
        for (int w = 0; w < W; ++w) mbar_init(&wbar[w], 1);
      *abort_flag = 0;
      fence_barrier_init();
    }
    __syncwarp();
    fetch_segments(d0);
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

  // Move a cursor n units on (P = 2)
  [[maybe_unused]] auto advance = [&](IssueCursor* c, int n) {
    c->u += n;
    c->z += n;
    while (c->u >= c->spec_end && c->u < U) {   // into a later spectrum
      const SpecDesc dn = spectrum_desc(p, c->b + 1);
      c->z = (int)(c->u - c->spec_end);
      c->b += 1;
      c->Z = dn.Z;
      c->z_off = dn.z_off;
      c->spec_end = c->b + 1 < p.count ? spectrum_desc(p, c->b + 1).unit_base : U;
    }
    while (c->z >= c->Z) c->z -= c->Z;
  };
  // Template of CTA position i (unit u0 + i): bank row z_off_b + (u - unit_base_b) mod Z_b.  The
  // cursor walks units in order, so an issue costs a few shared-memory operations; a descriptor is
  // read from global memory only when the walk enters the next spectrum.
  auto issue_template = [&](int64_t i) {
    const int slot = (int)(i % R);
    issued_pos[slot] = i;
    int64_t zrow;
    IssueCursor* const cp = P == 2 ? cur + (i & 1) : cur;
    if constexpr (LIST) zrow = cur->z_off + unit_at(u0 + i) % cur->Z;
    else zrow = cp->z_off + cp->z;
    mbar_arrive_expect_tx(&full[slot], L * 8);
    bulk_g2s(sT + (size_t)slot * L, p.templates + (size_t)zrow * L, L * 8, &full[slot]);
    if constexpr (LIST) return;   // single spectrum: the cursor's spectrum never changes
    if constexpr (P == 2) {
      advance(cp, 2);
      return;
    }
    cur->u += 1;
    cur->z = cur->z + 1 == cur->Z ? 0 : cur->z + 1;
    if (cur->u == cur->spec_end && cur->u < U) {
      const int nb = cur->b + 1;
      const SpecDesc dn = spectrum_desc(p, nb);
      cur->b = nb;
      cur->z = 0;
      cur->Z = dn.Z;
      cur->z_off = dn.z_off;
      cur->spec_end = nb + 1 < p.count ? spectrum_desc(p, nb + 1).unit_base : U;
    }
  };
  if (tid == 32 && !DEC) {
    cur->u = u0;
    cur->b = b;
    cur->Z = d0.Z;
    cur->z_off = d0.z_off;
    cur->z = (int)z_first;
    cur->spec_end = b + 1 < p.count ? spectrum_desc(p, b + 1).unit_base : U;
    if constexpr (P == 2) {
      cur[1] = cur[0];
      advance(cur + 1, 1);
    }
    const int64_t first = npos < R ? npos : R;
    for (int64_t i = 0; i < first; ++i) issue_template(i);
  }
  // twiddle pairs of lane k1, one warp per quadrant (stored once the tensor memory is there)
  float4 tw[H2];
  if (warp >= 4 && warp < 8) load_column_twiddles<Cfg>(tw, p.twist, k1);
  tmem_fence_before_sync();
  __syncthreads();
  tmem_fence_after_sync();
  const uint32_t tmem_row = *tmem_slot + ((uint32_t)(32 * (warp & 3)) << 16);
  const uint32_t tw_addr = tmem_row + Cfg::COL_TW;
  const uint32_t x_addr = tmem_row + Cfg::COL_X + (uint32_t)(wseg >> 2) * (2 * Cfg::N2);
  if (warp >= 4 && warp < 8) twiddles_to_tmem<H2>(tw, tw_addr);
  // release template slot `slot` of position i; the last of the W / P consumers refills it R
  // positions ahead
  auto release_slot = [&](int64_t i, int slot) {
    __syncwarp();
    if (lane == 0) {
      const unsigned old = arrive_count(&cnt[slot]);
      if ((old + 1u) % (unsigned)(W / P) == 0u) {
        if (i + R < npos) {
          fence_proxy_async_smem();
          issue_template(i + R);
        }
      }
    }
  };
  // the group after the one whose positions end at entry e
  auto next_group = [&](int64_t e) {
    if (e >= u1) return;
    if constexpr (LIST) {
      grp = quotient(unit_at(e), p.single.Z);
      z_first = unit_at(e) - grp * p.single.Z;
    } else {
      z_first = 0;
      if (++grp == spectrum_desc(p, b).ngroups) {
        grp = 0;
        ++b;
      }
    }
  };
  tmem_fence_before_sync();
  int alive = 1;
  uint32_t seg_phase = 0;
  bool seg_in_flight = false;
  uint32_t w_phase = 0;        // DEC: parity of this warp's next template copy
  bool w_in_flight = false;    // DEC: a copy into this warp's region not yet waited for
  int64_t u = u0;
  while (u < u1) {
    const SpecDesc d = spectrum_desc(p, b);
    int64_t grp_end;
    if constexpr (LIST) {
      grp_end = u + 1;
      while (grp_end < u1 && unit_at(grp_end) < (grp + 1) * d.Z) ++grp_end;
    } else {
      grp_end = u + (d.Z - z_first);
    }
    const int64_t a = u - u0;
    const int64_t bpos = (grp_end < u1 ? grp_end : u1) - u0;
    u = u0 + bpos;
    if (a > 0) {
      // every warp is done with its region (previous exchanges) before segments land in it
      fence_proxy_async_smem();
      alive = __syncthreads_and(alive && !*abort_flag);
      tmem_fence_after_sync();
      if (!alive) break;
      if (warp == 0) fetch_segments(d);
    }
    if (P == 1 || par == 0) {
      // zeros outside [0, n_b) in this lane group's window
      const int64_t x0 = (grp * G + wseg * Cfg::F + gw) * (int64_t)p.V - p.h;
      const int64_t lo = x0 < 0 ? (-x0 < L ? -x0 : L) : 0;                           // [0, lo) below 0
      const int64_t hi = d.n_bins - x0 < L ? (d.n_bins - x0 > 0 ? d.n_bins - x0 : 0) : L;  // [hi, L) beyond n
      for (int e = k1; e < L; e += N1)
        if (e < lo || e >= hi) mySeg[e] = make_float2(0.f, 0.f);
    }
    seg_in_flight = true;
    alive = __syncthreads_and(mbar_wait(segbar, seg_phase) ? 1 : 0);
    tmem_fence_after_sync();   // the twiddles were stored by other warps
    if (!alive) {
      if (tid == 0) report_timeout(p.status, abort_flag);
      break;
    }
    seg_in_flight = false;
    seg_phase ^= 1u;

    // a3: forward FFT of this lane group's segment; X pairs (k2 = 2p, 2p+1) go to TMEM
    if (P == 1 || par == 0) forward_to_tmem<Cfg>(mySeg, myXb, k1, tw_addr, x_addr);
    if constexpr (P == 2) {   // the other warp of the segment reads the spectrum too
      tmem_fence_before_sync();
      __syncthreads();
      tmem_fence_after_sync();
    }

    const int64_t s = grp * G + wseg * Cfg::F + gw;
    const int64_t segbase = s * (int64_t)p.V;
    const int64_t lim64 = d.n_bins - segbase < (int64_t)p.V ? d.n_bins - segbase : (int64_t)p.V;
    const int lim = lim64 > 0 ? (int)lim64 : 0;
    if constexpr (DEC) {
      // this warp's segment bits of list position i (warp-uniform)
      auto warp_bits = [&](int64_t i) -> unsigned {
        return ((unsigned)__ldg(p.unit_mask + u0 + i) >> (warp * Cfg::F)) & ((1u << Cfg::F) - 1u);
      };
      auto next_active = [&](int64_t i) {
        while (i < bpos && warp_bits(i) == 0u) ++i;
        return i;
      };
      // template of position i into this warp's region (lane 0; the region's earlier generic
      // accesses are ordered before the asynchronous copy)
      auto fetch = [&](int64_t i) {
        __syncwarp();
        if (lane == 0) {
          fence_proxy_async_smem();
          const int64_t zrow = unit_at(u0 + i) % d.Z;
          mbar_arrive_expect_tx(&wbar[warp], L * 8);
          bulk_g2s(myRegion, p.templates + (size_t)zrow * L, L * 8, &wbar[warp]);
        }
        w_in_flight = true;
      };
      int64_t i = next_active(a);
      if (i < bpos) fetch(i);
      while (i < bpos) {
        const int ok = __all_sync(0xffffffffu, wait_slot(&wbar[warp], w_phase, abort_flag));
        if (!ok) {   // the copy stays in flight: the exit path waits for it (bounded)
          if (lane == 0) report_timeout(p.status, abort_flag);
          break;
        }
        w_in_flight = false;
        w_phase ^= 1u;
        const int64_t z = unit_at(u0 + i) % d.Z;
        const int lim_z = ((warp_bits(i) >> gw) & 1u) ? lim : 0;
        const float4* st4 = reinterpret_cast<const float4*>(myRegion);
        cp2 v[H2];
        multiply_first_stage<Cfg, 0, H2 / 2>(v, x_addr, [&](int q) { return st4[q * N1 + k1]; });
        const int64_t inext = next_active(i + 1);
        fft_split_pairs<Cfg::N2, +1, 1>(v);
        float* row = d.plane + z * d.n_bins + segbase;
        exchange_twist_pass2<Cfg, +1>(
            v, myXb, k1, tw_addr,
            [&](auto rr, auto& y) { store_powers<Cfg, NV, decltype(rr)::value>(y, row, k1, lim_z); },
            [&]() {
              if (inext < bpos) fetch(inext);
            });
        i = inext;
      }
      // after a timeout the abort flag is set: every warp leaves at the group barrier above
      next_group(u);
      tmem_fence_before_sync();
      continue;
    }
    for (int64_t i = P == 1 ? a : a + ((par - a) & 1); i < bpos; i += P) {
      const int slot = (int)(i % R);
      const int ok = __all_sync(0xffffffffu, wait_slot(&full[slot], (uint32_t)((i / R) & 1), abort_flag));
      if (!ok) {
        if (lane == 0) report_timeout(p.status, abort_flag);
        break;
      }
      // row of this position: consecutive templates without a list, the entry's own with one
      int64_t z;
      if constexpr (LIST) z = unit_at(u0 + i) % d.Z;
      else z = z_first + (int64_t)(i - a);
      const float4* st4 = reinterpret_cast<const float4*>(sT + (size_t)slot * L);
      // a masked list entry: a warp none of whose segments is listed skips the transform (it still
      // releases the slot); lanes of an unlisted segment store nothing
      bool warp_on = true, group_on = true;
      if constexpr (LIST) {
        if (p.unit_mask) {
          const unsigned wm = ((unsigned)__ldg(p.unit_mask + u0 + i) >> (warp * Cfg::F)) & ((1u << Cfg::F) - 1u);
          warp_on = wm != 0u;
          group_on = ((wm >> gw) & 1u) != 0u;
        }
      }

      if (!warp_on) {   // the slot is released unread
        release_slot(i, slot);
        continue;
      }
      const int lim_z = group_on ? lim : 0;

      // a4: Y = X (TMEM) * T (shared ring), packed pairs in bit-reversed order, with the first stage
      cp2 v[H2];
      multiply_first_stage<Cfg, 0, H2 / 2>(v, x_addr, [&](int q) { return st4[q * N1 + k1]; });
      release_slot(i, slot);
      // a5: inverse FFT; a6 + a7: keep n < V (and inside the spectrum), store |y|^2
      fft_split_pairs<Cfg::N2, +1, 1>(v);
      float* row = d.plane + z * d.n_bins + segbase;
      exchange_twist_pass2<Cfg, +1>(v, myXb, k1, tw_addr, [&](auto rr, auto& y) {
        store_powers<Cfg, NV, decltype(rr)::value>(y, row, k1, lim_z);
      });
    }
    next_group(u);
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
  if constexpr (DEC) {
    if (lane == 0 && w_in_flight) (void)mbar_wait(&wbar[warp], w_phase);   // bounded
  }
  if (warp == 2) tmem_dealloc(*tmem_slot, Cfg::TMEM_COLS);
}

// Pair-list kernel (one transform per warp, L = 2048).  The listed (segment s, template z) pairs,
// entries s*Z + z in ascending order, are cut into equal contiguous ranges, one per warp of the
// grid, so a sparse list costs about its share of the full plane's transforms whatever its
// layout.  The warps are independent: a warp whose range enters a new segment brings it into its
// shared region (bulk copy of the part inside [0, n), zero fill of the rest) and runs the forward
// transform (Eq. 3) into its TMEM columns; for every pair it brings the template into the same
// region (bulk copy, issued as soon as the previous transform's exchange tile has been read when
// the next pair has the same segment), multiplies, runs the inverse transform and stores |y|^2
// for the segment's valid outputs (Section 2, overlap-and-save).  One mbarrier per warp serves
// both kinds of copy, at most one of them in flight.
template <class Cfg, int NV>
__global__ void __launch_bounds__(256, 1) fdas_convolve_pairs_kernel(const PairParams p) {
  static_assert(Cfg::F == 1, "one transform per warp");
  constexpr int L = Cfg::L, N1 = Cfg::N1, H2 = Cfg::H2, W = Cfg::W;
  extern __shared__ __align__(1024) unsigned char smem[];
  uint64_t* wbar = reinterpret_cast<uint64_t*>(smem + (size_t)W * Cfg::REGION);   // [W]
  volatile int* abort_flag = reinterpret_cast<volatile int*>(wbar + W);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(wbar + W) + 1;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, k1 = lane;
  float2* myRegion = reinterpret_cast<float2*>(smem + (size_t)warp * Cfg::REGION);
  float4* myXb = reinterpret_cast<float4*>(myRegion);
  uint64_t* bar = &wbar[warp];

  // a list that failed its check (kStatusBadList, set by the preceding check kernel) is not run
  if (*reinterpret_cast<volatile const int*>(p.status) & kStatusBadList) return;
  const int64_t P = p.pair_count ? *p.pair_count : p.n_pairs;
  const int64_t NW = (int64_t)gridDim.x * W;
  const int64_t cta0 = (int64_t)blockIdx.x * W;
  if ((cta0 + W) * P / NW == cta0 * P / NW) return;   // no pair for this CTA (uniform)
  const int64_t e0 = (cta0 + warp) * P / NW, e1 = (cta0 + warp + 1) * P / NW;

  if (tid == 0) {
    for (int w = 0; w < W; ++w) mbar_init(&wbar[w], 1);
    *abort_flag = 0;
    fence_barrier_init();
  }
  if (warp == 2) {
    tmem_alloc(tmem_slot, Cfg::TMEM_COLS);
    tmem_relinquish();
  }
  // twiddle pairs of lane k1, one warp per quadrant (stored once the tensor memory is there)
  float4 tw[H2];
  if (warp >= 4) load_column_twiddles<Cfg>(tw, p.twist, k1);
  tmem_fence_before_sync();
  __syncthreads();
  tmem_fence_after_sync();
  const uint32_t tmem_row = *tmem_slot + ((uint32_t)(32 * (warp & 3)) << 16);
  const uint32_t tw_addr = tmem_row + Cfg::COL_TW;
  const uint32_t x_addr = tmem_row + Cfg::COL_X + (uint32_t)(warp >> 2) * (2 * Cfg::N2);
  if (warp >= 4) twiddles_to_tmem<H2>(tw, tw_addr);
  tmem_fence_before_sync();
  __syncthreads();
  tmem_fence_after_sync();

  uint32_t phase = 0;
  bool in_flight = false;   // a copy into this warp's region not yet waited for (warp-uniform)
  // bounded wait for the copy in flight; false after a timeout (the copy stays marked in flight)
  auto wait_copy = [&]() -> bool {
    const int ok = __all_sync(0xffffffffu, wait_slot(bar, phase, abort_flag));
    if (!ok) {
      if (lane == 0) report_timeout(p.status, abort_flag);
      return false;
    }
    in_flight = false;
    phase ^= 1u;
    return true;
  };
  // template z into the region (its earlier generic accesses are ordered before the copy)
  auto fetch_template = [&](int z) {
    __syncwarp();
    if (lane == 0) {
      fence_proxy_async_smem();
      mbar_arrive_expect_tx(bar, L * 8);
      bulk_g2s(myRegion, p.templates + (size_t)z * L, L * 8, bar);
    }
    in_flight = true;
  };

  int64_t cur_s = -1;
  for (int64_t e = e0; e < e1; ++e) {
    const int32_t u = __ldg(p.pairs + e);   // checked: 0 <= u < nseg*Z <= 2^31 - 1
    const int s32 = u / p.Z;                 // 32-bit division
    const int64_t s = s32;
    const int z = u - s32 * p.Z;
    if (s != cur_s) {
      // a2: the segment's window A[sV - h, sV - h + L): bulk copy of its part inside [0, n) (even
      // bounds: n and h are multiples of 4, so every copy is whole 16-byte units), zeros elsewhere
      const int64_t x0 = s * (int64_t)p.V - p.h;
      const int64_t c0 = x0 > 0 ? x0 : 0;
      const int64_t c1 = x0 + L < p.n_bins ? x0 + L : p.n_bins;
      __syncwarp();
      if (lane == 0) {
        fence_proxy_async_smem();
        mbar_arrive_expect_tx(bar, (uint32_t)((c1 - c0) * 8));
        bulk_g2s(myRegion + (c0 - x0), p.spec + c0, (uint32_t)((c1 - c0) * 8), bar);
      }
      in_flight = true;
      for (int i = k1; i < L; i += N1)
        if (x0 + i < c0 || x0 + i >= c1) myRegion[i] = make_float2(0.f, 0.f);
      if (!wait_copy()) break;
      __syncwarp();
      // a3: forward FFT of the segment
      forward_to_tmem<Cfg>(myRegion, myXb, k1, tw_addr, x_addr);
      cur_s = s;
      fetch_template(z);
    }
    if (!wait_copy()) break;
    // the next pair's template is fetched during this transform when it has the same segment
    int znext = -1;
    if (e + 1 < e1) {
      const int32_t un = __ldg(p.pairs + e + 1);
      if (un / p.Z == s32) znext = un - s32 * p.Z;
    }
    // a4: Y = X (TMEM) * T (this warp's region), packed pairs in bit-reversed order, with the first stage
    const float4* st4 = reinterpret_cast<const float4*>(myRegion);
    cp2 v[H2];
    multiply_first_stage<Cfg, 0, H2 / 2>(v, x_addr, [&](int q) { return st4[q * N1 + k1]; });
    // a5: inverse FFT; a6 + a7: keep n < V inside the spectrum, store |y|^2
    fft_split_pairs<Cfg::N2, +1, 1>(v);
    const int64_t segbase = s * (int64_t)p.V;
    const int64_t lim64 = p.n_bins - segbase < (int64_t)p.V ? p.n_bins - segbase : (int64_t)p.V;
    const int lim = (int)lim64;
    float* row = p.plane + (int64_t)z * p.n_bins + segbase;
    exchange_twist_pass2<Cfg, +1>(
        v, myXb, k1, tw_addr,
        [&](auto rr, auto& y) { store_powers<Cfg, NV, decltype(rr)::value>(y, row, k1, lim); },
        [&]() {
          if (znext >= 0) fetch_template(znext);
        });
  }

  // a copy still in flight after a timeout: wait for it (bounded); always free TMEM
  if (lane == 0 && in_flight) (void)mbar_wait(bar, phase);
  __syncwarp();
  tmem_fence_before_sync();
  __syncthreads();
  tmem_fence_after_sync();
  if (warp == 2) tmem_dealloc(*tmem_slot, Cfg::TMEM_COLS);
}

// Forward transforms only (steps a2 + a3), natural-order output, for tests of the FFT: the forward code of
// the kernels above, one CTA per segment group.
template <class Cfg>
constexpr size_t seg_smem() {
  return (size_t)Cfg::W * Cfg::REGION + 64;
}
template <class Cfg>
__global__ void __launch_bounds__(32 * Cfg::W, 1) fdas_segment_spectra_kernel(const SegParams p) {
  constexpr int L = Cfg::L, N1 = Cfg::N1, N2 = Cfg::N2, H2 = Cfg::H2, G = Cfg::G;
  static_assert(Cfg::P == 1 && Cfg::W == 8 && G <= 32, "one warp per segment set, one lane per segment");
  extern __shared__ __align__(1024) unsigned char smem[];
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem + (size_t)Cfg::W * Cfg::REGION);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bar + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int gw = lane / N1, k1 = lane % N1;
  float2* region = reinterpret_cast<float2*>(smem + (size_t)warp * Cfg::REGION);
  float2* mySeg = region + (size_t)gw * L;
  float4* myXb = reinterpret_cast<float4*>(region) + gw * Cfg::XGROUP;
  const int64_t s0 = (int64_t)blockIdx.x * G;
  if (warp == 0) {
    if (lane == 0) {
      mbar_init(bar, 1);
      fence_barrier_init();
    }
    __syncwarp();
    const int64_t x0 = (s0 + lane) * (int64_t)p.V - p.h;
    const int64_t c0 = x0 > 0 ? x0 : 0, c1 = x0 + L < p.n_bins ? x0 + L : p.n_bins;
    const uint32_t bytes = lane < G && c1 > c0 ? (uint32_t)((c1 - c0) * 8) : 0u;
    const uint32_t total = __reduce_add_sync(0xffffffffu, bytes);
    if (lane == 0) mbar_arrive_expect_tx(bar, total);
    __syncwarp();
    if (bytes) {
      float2* dst = reinterpret_cast<float2*>(smem + (size_t)(lane / Cfg::F) * Cfg::REGION) + (lane % Cfg::F) * L;
      bulk_g2s(dst + (c0 - x0), p.spectrum_in + c0, bytes, bar);
    }
  } else if (warp == 2) {
    tmem_alloc(tmem_slot, Cfg::TMEM_COLS);
    tmem_relinquish();
  }
  const int64_t s = s0 + warp * Cfg::F + gw;
  {
    // zeros outside [0, n) in this lane group's window
    const int64_t x0 = s * (int64_t)p.V - p.h;
    for (int e = k1; e < L; e += N1)
      if (x0 + e < 0 || x0 + e >= p.n_bins) mySeg[e] = make_float2(0.f, 0.f);
  }
  float4 tw[H2];
  if (warp >= 4) load_column_twiddles<Cfg>(tw, p.twist, k1);
  tmem_fence_before_sync();
  __syncthreads();
  tmem_fence_after_sync();
  const uint32_t tw_addr = *tmem_slot + ((uint32_t)(32 * (warp & 3)) << 16) + Cfg::COL_TW;
  if (warp >= 4) twiddles_to_tmem<H2>(tw, tw_addr);
  tmem_fence_before_sync();
  const int ok = __syncthreads_and(mbar_wait(bar, 0) ? 1 : 0);
  tmem_fence_after_sync();
  if (ok) {
    float2* dst = p.out + s * L;
    const bool valid = s < p.nseg;
    forward_transform<Cfg>(mySeg, myXb, k1, tw_addr, [&](auto rr, auto& x) {
      static_for<N1>([&](auto nn) {
        constexpr int n1 = decltype(nn)::value;
        const int n = decltype(rr)::value * N1 + k1 + N2 * n1;
        if (valid) {
          dst[n] = make_float2(x[n1].re.x, x[n1].im.x);
          dst[n + Cfg::CP * N1] = make_float2(x[n1].re.y, x[n1].im.y);
        }
      });
    });
  } else if (tid == 0) {
    atomicOr(p.status, kStatusTimeout);
    (void)mbar_wait(bar, 0);   // bounded wait for copies still in flight
  }
  tmem_fence_before_sync();
  __syncthreads();
  tmem_fence_after_sync();
  if (warp == 2) tmem_dealloc(*tmem_slot, Cfg::TMEM_COLS);
}

// ---------------------------------------------------------------------------------------
// Host dispatch
// ---------------------------------------------------------------------------------------
int conv_group_threads(int L) {
  switch (L) {
    case 256: return 8;
    case 512: return 16;
    case 1024:
    case 2048: return 32;
    case 4096: return 64;
    default: return 128;
  }
}

template <class Cfg>
static cudaError_t launch_seg_cfg(const SegParams& p, cudaStream_t st) {
  static_assert(seg_smem<Cfg>() <= 232448, "shared memory budget of the segment-spectra kernel");
  auto kern = fdas_segment_spectra_kernel<Cfg>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)seg_smem<Cfg>());
  if (e != cudaSuccess) return e;
  const int64_t grid = (p.nseg + Cfg::G - 1) / Cfg::G;
  kern<<<(unsigned)grid, 32 * Cfg::W, seg_smem<Cfg>(), st>>>(p);
  return cudaGetLastError();
}

// Full planes: PlaneCfg.  Work lists: ListCfg (the same segments per CTA; void: none), separate
// instantiations with their own parameter type, so that the full-plane code stays free of them.
template <class PlaneCfg, class ListCfg, int NV>
static cudaError_t launch_tmem_nv(const ListParams& p, int sm_count, cudaStream_t st) {
  const int64_t grid = p.units < sm_count ? p.units : sm_count;
  auto launch = [&](auto kern, int warps, size_t smem, const auto& params) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)grid, 32 * warps, smem, st>>>(params);
    return cudaGetLastError();
  };
  if constexpr (std::is_void_v<ListCfg>) {
    if (p.unit_list) return cudaErrorInvalidValue;
  } else {
    static_assert(PlaneCfg::G == ListCfg::G, "a unit is the same segments in both");
    if (p.unit_list && p.unit_mask)
      return launch(fdas_convolve_tmem_kernel<ListCfg, NV, true, true>, ListCfg::W, ListCfg::SMEM, p);
    if (p.unit_list) return launch(fdas_convolve_tmem_kernel<ListCfg, NV, true>, ListCfg::W, ListCfg::SMEM, p);
  }
  BatchParams q = p;
  // (P = 2: two positions, half of the warps run the forward transforms)
  if (q.descs == nullptr && q.units > grid)
    q.group_cost = PlaneCfg::P == 2 ? 2 : group_cost_of(q.units, q.single.ngroups, grid);
  const int64_t total = q.units + q.group_cost * q.single.ngroups;
  q.span = total / grid;
  q.span_extra = (int)(total % grid);
  return launch(fdas_convolve_tmem_kernel<PlaneCfg, NV, false>, PlaneCfg::W, PlaneCfg::SMEM, q);
}

// Smallest instantiated NV >= ceil(V / N2): N1*3/4, N1*7/8 or N1.
template <class PlaneCfg, class ListCfg>
static cudaError_t launch_tmem_cfg(const ListParams& p, int sm_count, cudaStream_t st) {
  constexpr int N1 = PlaneCfg::N1;
  const int rows = (p.V + PlaneCfg::N2 - 1) / PlaneCfg::N2;
  if (rows <= N1 * 3 / 4) return launch_tmem_nv<PlaneCfg, ListCfg, N1 * 3 / 4>(p, sm_count, st);
  if (rows <= N1 * 7 / 8) return launch_tmem_nv<PlaneCfg, ListCfg, N1 * 7 / 8>(p, sm_count, st);
  return launch_tmem_nv<PlaneCfg, ListCfg, N1>(p, sm_count, st);
}

using Tmem256 = TmemCfg<256, 8, 16, 2>;
using Tmem512 = TmemCfg<512, 16, 16, 2>;
using Tmem512List = TmemCfg<512, 16>;
using Tmem2048 = TmemCfg<2048, 32>;

// Lengths with work lists and with batches in one launch.  256 runs the same kernel but has no work-list form,
// which a non-zero count also promises: a batch there is one launch per spectrum, as at 1024, 4096 and 8192.
int batch_segments_per_cta(int L) {
  switch (L) {
    case 512: return Tmem512::G;
    case 2048: return Tmem2048::G;
    default: return 0;
  }
}

static cudaError_t launch_desc(int L, const ListParams& p, int sm_count, cudaStream_t st) {
  switch (L) {
    case 256: return launch_tmem_cfg<Tmem256, void>(p, sm_count, st);
    case 512: return launch_tmem_cfg<Tmem512, Tmem512List>(p, sm_count, st);
    case 2048: return launch_tmem_cfg<Tmem2048, Tmem2048>(p, sm_count, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_batch(int L, const BatchParams& p, int sm_count, cudaStream_t st) {
  ListParams q;
  static_cast<BatchParams&>(q) = p;
  return launch_desc(L, q, sm_count, st);
}

// Single spectrum: the descriptor-driven kernel with an inline one-entry table where it exists.
static cudaError_t launch_single_desc(int L, const ConvParams& p, int sm_count, cudaStream_t st) {
  const int G = L == 256 ? Tmem256::G : batch_segments_per_cta(L);
  BatchParams q;
  q.templates = p.templates;
  q.twist = p.twist;
  q.status = p.status;
  q.descs = nullptr;
  q.count = 1;
  q.single.spec = p.spectrum;
  q.single.plane = p.plane;
  q.single.n_bins = p.n_bins;
  q.single.nseg = p.nseg;
  q.single.unit_base = 0;
  q.single.ngroups = (p.nseg + G - 1) / G;
  q.single.Z = p.Z;
  q.single.z_off = 0;
  q.units = q.single.ngroups * p.Z;
  q.unit_list = nullptr;
  q.V = p.V;
  q.h = p.h;
  return launch_batch(L, q, sm_count, st);
}

// A work list is usable when its entries are strictly increasing and inside [0, limit): that
// bounds every template row, segment and plane row the kernel touches.  Otherwise kStatusBadList.
// With d_count the length is read from device memory and must lie in [0, n] (n = the list's capacity).
__global__ void check_units_kernel(const int32_t* units, int64_t n, int64_t limit, int* status,
                                   const int64_t* d_count) {
  if (d_count) {
    const int64_t c = *d_count;
    if (c < 0 || c > n) {
      if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(status, kStatusBadList);
      return;
    }
    n = c;
  }
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t u = units[e];
    if (u < 0 || u >= limit || (e > 0 && (int64_t)units[e - 1] >= u)) atomicOr(status, kStatusBadList);
  }
}

cudaError_t launch_units(int L, const ConvParams& p, const int32_t* units, const uint16_t* masks, int64_t n_units,
                         int sm_count, cudaStream_t st, const int64_t* d_count) {
  const int G = batch_segments_per_cta(L);
  if (G == 0 || n_units < 1) return cudaErrorInvalidValue;
  const int64_t ngroups = (p.nseg + G - 1) / G;
  {
    const int64_t blocks = (n_units + 255) / 256;
    const unsigned grid = (unsigned)(blocks < 4LL * sm_count ? blocks : 4LL * sm_count);
    check_units_kernel<<<grid, 256, 0, st>>>(units, n_units, ngroups * p.Z, p.status, d_count);
  }
  ListParams q;
  q.templates = p.templates;
  q.twist = p.twist;
  q.status = p.status;
  q.descs = nullptr;
  q.count = 1;
  q.single.spec = p.spectrum;
  q.single.plane = p.plane;
  q.single.n_bins = p.n_bins;
  q.single.nseg = p.nseg;
  q.single.unit_base = 0;
  q.single.ngroups = ngroups;
  q.single.Z = p.Z;
  q.single.z_off = 0;
  q.units = n_units;
  q.unit_list = units;
  q.unit_mask = masks;
  q.unit_count = d_count;   // with a device count, n_units is the list's capacity (grid: every SM)
  q.V = p.V;
  q.h = p.h;
  return launch_desc(L, q, sm_count, st);
}

bool pairs_supported(int L) { return L == 2048; }

template <class Cfg, int NV>
static cudaError_t launch_pairs_nv(const PairParams& p, int sm_count, cudaStream_t st) {
  constexpr size_t smem = (size_t)Cfg::W * Cfg::REGION + 128;
  static_assert(smem <= 232448, "shared memory budget of the pair-list kernel");
  auto kern = fdas_convolve_pairs_kernel<Cfg, NV>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  // every SM when the length is on the device; otherwise no more CTAs than W-pair shares
  const int64_t need = (p.n_pairs + Cfg::W - 1) / Cfg::W;
  const int64_t grid = p.pair_count || need > sm_count ? sm_count : need;
  kern<<<(unsigned)grid, 256, smem, st>>>(p);
  return cudaGetLastError();
}

cudaError_t launch_pairs(int L, const PairParams& p, int sm_count, cudaStream_t st) {
  if (!pairs_supported(L) || p.n_pairs < 1) return cudaErrorInvalidValue;
  {
    const int64_t blocks = (p.n_pairs + 255) / 256;
    const unsigned grid = (unsigned)(blocks < 4LL * sm_count ? blocks : 4LL * sm_count);
    check_units_kernel<<<grid, 256, 0, st>>>(p.pairs, p.n_pairs, p.nseg * p.Z, p.status, p.pair_count);
  }
  // two instantiations (compile time): rows pruned to 3/4 (m >= L/4), or none pruned
  using Cfg = TmemCfg<2048, 32>;
  const int rows = (p.V + Cfg::N2 - 1) / Cfg::N2;
  if (rows <= Cfg::N1 * 3 / 4) return launch_pairs_nv<Cfg, Cfg::N1 * 3 / 4>(p, sm_count, st);
  return launch_pairs_nv<Cfg, Cfg::N1>(p, sm_count, st);
}

cudaError_t launch_convolve(int L, const ConvParams& p, int sm_count, cudaStream_t st) {
  switch (L) {
    case 256:
    case 512:
    case 2048: return launch_single_desc(L, p, sm_count, st);
    default: return launch_convolve_wide(L, p, sm_count, st);
  }
}

cudaError_t launch_segment_spectra(int L, const SegParams& p, int sm_count, cudaStream_t st) {
  switch (L) {
    case 256: return launch_seg_cfg<TmemCfg<256, 8>>(p, st);
    case 512: return launch_seg_cfg<Tmem512List>(p, st);
    case 2048: return launch_seg_cfg<Tmem2048>(p, st);
    default: return launch_segment_spectra_wide(L, p, sm_count, st);
  }
}

}  // namespace fdas
