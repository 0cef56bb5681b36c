// fdas_conv_common.cuh -- pieces shared by the fused correlation kernels.
#pragma once

#include "fdas_device.cuh"
#include "fdas_internal.h"

namespace fdas {

__host__ __device__ constexpr size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// The element-wise products with the templates (before pass 1) and with the twiddles (before pass 2)
// are joined with the radix-2 stage that follows them: a + b = t + B*b', a - b = 2t - (a + b) with
// t = A*a' take 10 packed instructions per butterfly where two products and the butterfly take 12.
// Operands whose pairs meet in that stage (p and p + n/2) therefore sit next to each other in tensor
// memory: slot 2p holds pair p, slot 2p + 1 pair p + n/2.
constexpr __host__ __device__ int slot_pair(int slot, int n) { return (slot >> 1) + (slot & 1) * (n / 2); }
__device__ __forceinline__ cp2 tmem_pair(const float (&r)[16], int q) {
  return cp2{make_float2(r[4 * q], r[4 * q + 1]), make_float2(r[4 * q + 2], r[4 * q + 3])};
}

// Both products go in chunks of two butterflies.  PIPE: a chunk's operands are fetched before the
// previous chunk is computed; the kernels with one column pair per lane and a ring shared by eight
// warps are faster without (2048: 1313 against 1366 us per survey plane), the others with it (4096: 1847
// against 1877 us, 8192: 1680 against 1713 us for their timed planes).

// Y = X (this lane's TMEM slots from x_addr) * T (load(p) = pair p) and the first stage of the
// N2-point DFT: v in bit-reversed order, pairs [P0, P0 + NP) and their partners.
template <class Cfg, int P0, int NP, class Load>
__device__ __forceinline__ void multiply_first_stage(cp2 (&v)[Cfg::H2], uint32_t x_addr, Load&& load) {
  constexpr int HALF = Cfg::H2 / 2, NC = NP / 2;
  float x[2][16];
  float4 t[2][4];
  auto fetch = [&](auto cc) {
    constexpr int b = decltype(cc)::value & 1, p0 = P0 + 2 * decltype(cc)::value;
    tmem_ld16(x_addr + 8 * p0, x[b]);
    t[b][0] = load(p0);
    t[b][1] = load(p0 + HALF);
    t[b][2] = load(p0 + 1);
    t[b][3] = load(p0 + 1 + HALF);
  };
  if constexpr (Cfg::PIPE) fetch(std::integral_constant<int, 0>{});
  static_for<NC>([&](auto cc) {
    constexpr int c = decltype(cc)::value, b = c & 1, p0 = P0 + 2 * c;
    if constexpr (!Cfg::PIPE) fetch(cc);
    tmem_wait_ld();
    if constexpr (Cfg::PIPE && c + 1 < NC) fetch(std::integral_constant<int, c + 1>{});
    constexpr int i0 = bitrev(2 * p0, Cfg::LOG_N2), i1 = bitrev(2 * p0 + 2, Cfg::LOG_N2);
    const cp2 t0 = cmul2(tmem_pair(x[b], 0), cp2_from(t[b][0])), t1 = cmul2(tmem_pair(x[b], 2), cp2_from(t[b][2]));
    v[i0] = cfma2(tmem_pair(x[b], 1), cp2_from(t[b][1]), t0);
    v[i1] = cfma2(tmem_pair(x[b], 3), cp2_from(t[b][3]), t1);
    v[i0 + 1] = twice_minus(t0, v[i0]);
    v[i1 + 1] = twice_minus(t1, v[i1]);
  });
}

// u = entries (load(s), s < N) times the twiddles of this lane's TMEM slots (conjugated for the forward
// transform), with the first stage done: N entries in bit-reversed order over log2(N) + SHIFT bits of
// (s << SHIFT).  The first pair's twiddle is 1 when UNIT0.
template <int N, int SHIFT, bool CONJ, bool UNIT0, bool PIPE, class Load>
__device__ __forceinline__ void twist_first_stage(cp2 (&u)[N], uint32_t tw_addr, Load&& load) {
  constexpr int HALF = N / 2, LOG = ilog2(N) + SHIFT, NC = N / 4;
  float w[2][16];
  cp2 e[2][4];
  auto fetch = [&](auto cc) {
    constexpr int b = decltype(cc)::value & 1, s0 = 2 * decltype(cc)::value;
    tmem_ld16(tw_addr + 8 * s0, w[b]);
    e[b][0] = load(std::integral_constant<int, s0>{});
    e[b][1] = load(std::integral_constant<int, s0 + HALF>{});
    e[b][2] = load(std::integral_constant<int, s0 + 1>{});
    e[b][3] = load(std::integral_constant<int, s0 + 1 + HALF>{});
  };
  auto times = [](const cp2& a, const cp2& t) { return CONJ ? cmul2_conj(a, t) : cmul2(a, t); };
  auto times_add = [](const cp2& a, const cp2& t, const cp2& c) { return CONJ ? cfma2_conj(a, t, c) : cfma2(a, t, c); };
  if constexpr (PIPE) fetch(std::integral_constant<int, 0>{});
  static_for<NC>([&](auto cc) {
    constexpr int c = decltype(cc)::value, b = c & 1, s0 = 2 * c;
    if constexpr (!PIPE) fetch(cc);
    tmem_wait_ld();
    if constexpr (PIPE && c + 1 < NC) fetch(std::integral_constant<int, c + 1>{});
    constexpr int i0 = bitrev(s0 << SHIFT, LOG), i1 = bitrev((s0 + 1) << SHIFT, LOG);
    const cp2 t0 = UNIT0 && s0 == 0 ? e[b][0] : times(e[b][0], tmem_pair(w[b], 0));
    const cp2 t1 = times(e[b][2], tmem_pair(w[b], 2));
    u[i0] = times_add(e[b][1], tmem_pair(w[b], 1), t0);
    u[i1] = times_add(e[b][3], tmem_pair(w[b], 3), t1);
    u[i0 + 1] = twice_minus(t0, u[i0]);
    u[i1 + 1] = twice_minus(t1, u[i1]);
  });
}

// This lane's spectrum pairs x(p), p < H2, to TMEM in slot order.
template <int H2, class Pair>
__device__ __forceinline__ void spectrum_to_tmem(uint32_t x_addr, Pair&& pair) {
  static_for<H2 / 4>([&](auto cc) {
    constexpr int c = decltype(cc)::value;
    float r[16];
    static_for<4>([&](auto qq) {
      constexpr int q = decltype(qq)::value;
      const cp2 x = pair(std::integral_constant<int, slot_pair(4 * c + q, H2)>{});
      r[4 * q] = x.re.x;
      r[4 * q + 1] = x.re.y;
      r[4 * q + 2] = x.im.x;
      r[4 * q + 3] = x.im.y;
    });
    tmem_st16(x_addr + 16 * c, r);
  });
  tmem_wait_st();
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

// Twiddle pairs into this lane's TMEM columns from `addr`, in order.
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

// Zeros outside [0, n) in a window of L bins from bin x0, by `lanes` lanes.  Only the missing ranges are
// walked: a test of every element cost an edge segment's CTA 1,700 cycles.
template <int L>
__device__ __forceinline__ void zero_outside(float2* seg, int64_t x0, int64_t n, int lane, int lanes) {
  const int lo = x0 < 0 ? (int)(-x0 < L ? -x0 : L) : 0;
  const int hi = n - x0 < L ? (int)(n - x0 > 0 ? n - x0 : 0) : L;
  for (int e = lane; e < lo; e += lanes) seg[e] = make_float2(0.f, 0.f);
  for (int e = (hi > lo ? hi : lo) + lane; e < L; e += lanes) seg[e] = make_float2(0.f, 0.f);
}

}  // namespace fdas
