// fdas_conv_common.cuh -- pieces shared by the fused correlation kernels.
#pragma once

#include "fdas_device.cuh"
#include "fdas_internal.h"

namespace fdas {

__host__ __device__ constexpr size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Twist with the twiddle pairs held in this lane's TMEM row (4 columns per pair, chunks of 4 pairs).
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

// One arrival on a shared-memory consumer counter with acquire-release semantics at CTA scope: the
// caller's earlier reads of the slot (ordered within the warp by __syncwarp) happen before the
// arrival, and the last arriver's later refill of the slot happens after every other arrival.
// Returns the count before this arrival.
__device__ __forceinline__ unsigned arrive_count(unsigned* counter) {
  unsigned old;
  asm volatile("atom.acq_rel.cta.shared::cta.add.u32 %0, [%1], 1;" : "=r"(old) : "r"(smem_u32(counter)) : "memory");
  return old;
}

// Bounded wait for a template slot: the common case (already filled) costs one try_wait; the abort
// flag is read only when the slot is not ready, so one warp's timeout stops the others quickly.
__device__ __forceinline__ int wait_slot(uint64_t* bar, uint32_t parity, volatile int* abort_flag) {
  if (mbar_try_wait(bar, parity)) return 1;
  if (*abort_flag) return 0;
  return mbar_wait(bar, parity) ? 1 : 0;
}

// Device status word: set kStatusTimeout when a bounded wait gave up.
__device__ __forceinline__ void report_timeout(int* status, volatile int* abort_flag) {
  *abort_flag = 1;
  atomicOr(status, kStatusTimeout);
}

// Twiddle pairs of transform lane k1 (pair p at p*n1 + k1 of the plan's table) ...
template <int H2>
__device__ __forceinline__ void load_twiddles(float4 (&tw)[H2], const float2* twist, int n1, int k1) {
  const float4* tw4 = reinterpret_cast<const float4*>(twist);
  static_for<H2>([&](auto jj) { tw[decltype(jj)::value] = __ldg(tw4 + decltype(jj)::value * n1 + k1); });
}
// ... into this lane's TMEM columns from `addr`.
template <int H2>
__device__ __forceinline__ void twiddles_to_tmem(const float4 (&tw)[H2], uint32_t addr) {
  static_for<H2 / 4>([&](auto cc) {
    constexpr int c = decltype(cc)::value;
    float r[16];
    static_for<4>([&](auto qq) {
      constexpr int q = decltype(qq)::value;
      r[4 * q] = tw[4 * c + q].x;
      r[4 * q + 1] = tw[4 * c + q].y;
      r[4 * q + 2] = tw[4 * c + q].z;
      r[4 * q + 3] = tw[4 * c + q].w;
    });
    tmem_st16(addr + 16 * c, r);
  });
  tmem_wait_st();
}

// a / b for a >= 0, in 32 bits where a fits.
__device__ __forceinline__ int64_t quotient(int64_t a, int b) {
  return (uint64_t)a <= 0xffffffffull ? (int64_t)((uint32_t)a / (uint32_t)b) : a / b;
}

}  // namespace fdas
