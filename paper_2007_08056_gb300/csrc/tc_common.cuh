// Device helpers shared by the tensor-core GEMM kernels (gemm_tc.cu,
// gemm_tc10.cu): mbarrier, TMA and tcgen05 wrappers, the bounded waits, the
// integer-only float64 rounding and the map-back stores of the epilogues.
#pragma once

#include <cuda.h>
#include <cstdint>
#include <type_traits>
#include <utility>

#include "symctr_internal.h"

namespace symctr {

constexpr int32_t kExpBias = 4096;  // row exponents are stored biased (0 = all-zero row)
constexpr long long kTimeoutCycles = 4000000000ll;  // ~2 s per wait at 2 GHz

__device__ __forceinline__ uint32_t su32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(su32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.release.cta.shared::cta.b64 _, [%0], %1;" ::"r"(su32(bar)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];" ::"r"(su32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_test(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(ok)
      : "r"(su32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

struct Ctl {
  volatile int abort;
  unsigned* err;
  // the producer's copies, for the waits after an abort: how many, or (gemm_tc10.cu)
  // the stages used and the parities of their next use
  uint32_t copies, phases;
};

// Bounded wait: true when the phase completed; false on timeout or abort.
// The budget is counted in SM clock cycles (clock64 is cheap to read; about
// 2 s at the maximum SM clock, longer at lower clocks).
__device__ __forceinline__ bool wait_phase(uint64_t* bar, uint32_t parity, Ctl* ctl,
                                           long long limit = kTimeoutCycles) {
  if (mbar_test(bar, parity)) return true;
  const long long t0 = clock64();
  for (;;) {
    if (mbar_test(bar, parity)) return true;
    if (ctl->abort) return false;
    if (clock64() - t0 > limit) {
      atomicOr(ctl->err, (unsigned)DEVERR_TIMEOUT);
      ctl->abort = 1;
      return false;
    }
  }
}

// Same, for threads with nothing else to do: the hardware suspends them
// between polls (suspend-time hint), so they do not take issue slots from
// the producer and MMA threads.
__device__ __forceinline__ bool mbar_test_sleep(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(ok)
      : "r"(su32(bar)), "r"(parity), "r"(1000000u)
      : "memory");
  return ok != 0;
}

__device__ __forceinline__ bool wait_phase_sleep(uint64_t* bar, uint32_t parity, Ctl* ctl) {
  const long long t0 = clock64();
  for (;;) {
    if (mbar_test_sleep(bar, parity)) return true;
    if (ctl->abort) return false;
    if (clock64() - t0 > kTimeoutCycles) {
      atomicOr(ctl->err, (unsigned)DEVERR_TIMEOUT);
      ctl->abort = 1;
      return false;
    }
  }
}

// Before a CTA leaves after an abort: wait for its own copies or MMAs in flight
// (the waits above give up at once then), so that none writes to shared memory or
// TMEM that the next CTA holds.  Bounded by the limit alone.  The kernels do so
// behind their last barrier, when no thread can set the abort flag any more and
// all see the same; without an abort everything in flight has been consumed.  Out
// of line: within the kernels this code, though never run, cost the ladder in TF32
// 0.5% and the split GEMM 1.2% (40960 x 640 x 640 by 10 irreps).
static __device__ __noinline__ bool wait_landed(uint64_t* bar, uint32_t parity, Ctl* ctl,
                                                long long limit = kTimeoutCycles / 2) {
  const long long t0 = clock64();
  while (!mbar_test_sleep(bar, parity)) {
    if (clock64() - t0 > limit) {
      atomicOr(ctl->err, (unsigned)DEVERR_TIMEOUT);
      ctl->abort = 1;
      return false;
    }
  }
  return true;
}

// The same for a kernel whose producer made ctl->copies copies round the stages'
// barriers `full` and whose issuing thread (32) committed its MMAs to `mmas`.
__device__ __forceinline__ void land(uint64_t* full, int stages, uint64_t* mmas, Ctl* ctl) {
  const int i = threadIdx.x, last = (int)ctl->copies - 1 - i;   // thread i < stages: one of the last copies
  uint64_t* bar = i < stages && last >= 0 ? &full[last % stages] : i == 32 ? mmas : nullptr;
  if (bar) wait_landed(bar, i < stages ? (last / stages) & 1 : 0, ctl);
}

// Box of a [planes][batches][rows][k] map at (k = c0, row = c1, batch = c2, plane 0).
__device__ __forceinline__ void tma_load_4d(const CUtensorMap* map, uint64_t* bar, void* dst, int c0, int c1,
                                            int c2) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4, %5, %6}], [%2];" ::"r"(su32(dst)),
      "l"(map), "r"(su32(bar)), "r"(c0), "r"(c1), "r"(c2), "r"(0)
      : "memory");
}

__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                   su32(bar))
               : "memory");
}
// 4 consecutive 32-bit TMEM columns of this warp's 32 lanes.
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr));
}

// 16 consecutive 32-bit TMEM columns of this warp's 32 lanes.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
// 8 consecutive 32-bit TMEM columns of this warp's 32 lanes.
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
                 "=r"(r[7])
               : "r"(taddr));
}
// Registers that a TMEM load filled, after the wait for it: passing them through
// here keeps their uses behind the wait.
template <int W>
__device__ __forceinline__ void tmem_loaded(uint32_t* r) {
  static_assert(W == 4 || W == 16, "4 or 16 registers");
  if constexpr (W == 4) asm volatile("" : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]));
  else asm volatile("" : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]));
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
      "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}
template <int W>
__device__ __forceinline__ void tmem_ld_w(uint32_t taddr, uint32_t* r) {
  if constexpr (W == 16) tmem_ld16(taddr, r);
  else if constexpr (W == 8) tmem_ld8(taddr, r);
  else tmem_ld4(taddr, r);
}
// Zeros into W consecutive 32-bit TMEM columns of this warp's 32 lanes.
template <int W>
__device__ __forceinline__ void tmem_zero_w(uint32_t taddr) {
  const uint32_t z = 0u;
  if constexpr (W == 16) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
        "{%1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1};" ::"r"(taddr),
        "r"(z)
        : "memory");
  } else {
    static_assert(W == 8, "8 or 16 columns");
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %1, %1, %1, %1, %1, %1, %1};" ::"r"(taddr),
                 "r"(z)
                 : "memory");
  }
}
__device__ __forceinline__ void tmem_st4(uint32_t taddr, const uint32_t* r) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(taddr),
               "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3])
               : "memory");
}
__device__ __forceinline__ void tmem_wait_st() {
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_wait_ld() {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// RN(R * 2^e) as float64 using integer operations only (ties to even).
// Fast path: |R| < 2^53 and a normal result need no rounding, only a shift.
__device__ __forceinline__ double i64_scaled_slow(long long Rv, int e) {
  uint64_t sgn = Rv < 0 ? (1ull << 63) : 0ull;
  uint64_t m = Rv < 0 ? (uint64_t)(-Rv) : (uint64_t)Rv;
  int nb = 64 - __clzll((long long)m);
  int be = e + nb - 1 + 1023;  // biased exponent of the leading bit
  if (be >= 2047) return __longlong_as_double((long long)(sgn | 0x7FF0000000000000ull));
  if (be <= 0) {
    // subnormal: value / 2^-1074 = m * 2^(e + 1074)
    int k = -(e + 1074);
    uint64_t q;
    if (k <= 0) {
      q = m << (-k);
    } else if (k >= 64) {
      q = 0;
      if (k == 64 && m > (1ull << 63)) q = 1;
    } else {
      q = m >> k;
      uint64_t rem = m & ((1ull << k) - 1), half = 1ull << (k - 1);
      if (rem > half || (rem == half && (q & 1))) ++q;
    }
    return __longlong_as_double((long long)(sgn | q));
  }
  int shift = nb - 53;
  uint64_t q;
  if (shift > 0) {
    q = m >> shift;
    uint64_t rem = m & ((1ull << shift) - 1), half = 1ull << (shift - 1);
    if (rem > half || (rem == half && (q & 1))) ++q;
    if (q == (1ull << 53)) {
      q >>= 1;
      ++be;
      if (be >= 2047) return __longlong_as_double((long long)(sgn | 0x7FF0000000000000ull));
    }
  } else {
    q = m << (-shift);
  }
  return __longlong_as_double((long long)(sgn | ((uint64_t)be << 52) | (q & ((1ull << 52) - 1))));
}

__device__ __forceinline__ double i64_scaled(long long Rv, int e) {
  if (Rv == 0) return 0.0;
  const uint64_t m = Rv < 0 ? (uint64_t)(-Rv) : (uint64_t)Rv;
  if (m < (1ull << 53)) {
    const int nb = 64 - __clzll((long long)m);
    const int be = e + nb - 1 + 1023;
    if (be > 0 && be < 2047) {
      const uint64_t q = m << (53 - nb);
      const uint64_t sgn = Rv < 0 ? (1ull << 63) : 0ull;
      return __longlong_as_double((long long)(sgn | ((uint64_t)be << 52) | (q & ((1ull << 52) - 1))));
    }
  }
  return i64_scaled_slow(Rv, e);
}

// Out-of-line copies for the rare entries of a batch (keeps the batch code small).
static __device__ __noinline__ double i64_scaled_rare(long long Rv, int e) { return i64_scaled_slow(Rv, e); }

// The common case of i64_scaled without branches (selects only), so that a
// batch of conversions interleaves: exact for Rv = 0, or |Rv| < 2^53 with a
// normal result; `slow` is set for every other Rv.
__device__ __forceinline__ double i64_scaled_common(long long Rv, int e, bool& slow) {
  const uint64_t sm = (uint64_t)(Rv >> 63);   // all ones for Rv < 0
  const uint64_t m = ((uint64_t)Rv ^ sm) - sm;
  const int nb = 64 - __clzll((long long)m);
  const int be = e + nb - 1 + 1023;
  const uint64_t q = m << ((53 - nb) & 63);
  const uint64_t bits = (sm << 63) | ((uint64_t)(unsigned)be << 52) | (q & ((1ull << 52) - 1));
  slow = Rv != 0 && ((m >> 53) != 0 || (unsigned)(be - 1) >= 2046u);
  return Rv == 0 ? 0.0 : __longlong_as_double((long long)bits);
}

// RN(Rv[j] * 2^e[j]) for a batch: the common case for all, the general routine
// only for the entries that need it.
template <int B>
__device__ __forceinline__ void i64_scaled_batch(const long long (&Rv)[B], const int (&e)[B], double (&d)[B]) {
  unsigned slow_mask = 0;
#pragma unroll
  for (int j = 0; j < B; ++j) {
    bool sl;
    d[j] = i64_scaled_common(Rv[j], e[j], sl);
    slow_mask |= (unsigned)sl << j;
  }
  if (slow_mask) {
#pragma unroll
    for (int j = 0; j < B; ++j)
      if ((slow_mask >> j) & 1u) d[j] = i64_scaled_rare(Rv[j], e[j]);
  }
}

// Fire-and-forget 64-bit integer add in L2 (no value returned).
__device__ __forceinline__ void red_add_u64(unsigned long long* a, unsigned long long v) {
  asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(a), "l"(v) : "memory");
}

// Exact float32 -> float64 with integer operations.
__device__ __forceinline__ double f32_to_f64(uint32_t u) {
  uint64_t sgn = (uint64_t)(u >> 31) << 63;
  uint32_t e = (u >> 23) & 0xFF, m = u & 0x7FFFFF;
  if (e == 0) {
    if (m == 0) return __longlong_as_double((long long)sgn);
    double v = i64_scaled((long long)m, -149);
    return sgn ? -v : v;
  }
  if (e == 255) return __longlong_as_double((long long)(sgn | 0x7FF0000000000000ull | ((uint64_t)m << 29)));
  return __longlong_as_double((long long)(sgn | ((uint64_t)(e - 127 + 1023) << 52) | ((uint64_t)m << 29)));
}

static __device__ __noinline__ double f32_to_f64_rare(uint32_t u) { return f32_to_f64(u); }

// f32_to_f64 for a batch: normal numbers and zeros without branches, the
// general routine for subnormals, infinities and NaNs.
template <int B>
__device__ __forceinline__ void f32_to_f64_batch(const uint32_t (&u)[B], double (&d)[B]) {
  unsigned slow_mask = 0;
#pragma unroll
  for (int j = 0; j < B; ++j) {
    const uint32_t e = (u[j] >> 23) & 0xFFu;
    const uint64_t sgn = (uint64_t)(u[j] >> 31) << 63;
    const uint64_t bits = sgn | ((uint64_t)(e + 896u) << 52) | ((uint64_t)(u[j] & 0x7FFFFFu) << 29);
    const bool zero = (u[j] << 1) == 0;
    slow_mask |= (unsigned)(!zero && (e == 0 || e == 255)) << j;
    d[j] = __longlong_as_double((long long)(zero ? sgn : bits));
  }
  if (slow_mask) {
#pragma unroll
    for (int j = 0; j < B; ++j)
      if ((slow_mask >> j) & 1u) d[j] = f32_to_f64_rare(u[j]);
  }
}

// Map-back stores of a batch of results of one column (rows m_first, + rstep,
// ...): plain stores, or (complex products) adds, with the problem's sign; the
// output mode is uniform, so the plain path loads nothing from W.
// Rows or columns with offset -1 (general plans: absent from W) are not stored.
template <int B, bool GEN>
__device__ __forceinline__ void store_batch(const Problem& p, double* w, const int64_t (&ro)[B],
                                            int64_t co, const double (&d)[B], int64_t m_first,
                                            int rstep) {
  if (co < 0) return;
  if constexpr (!GEN) {
#pragma unroll
    for (int j = 0; j < B; ++j)
      if (m_first + rstep * j < p.M && ro[j] >= 0) w[ro[j] + co] = d[j];
  } else if (!p.accumulate) {
#pragma unroll
    for (int j = 0; j < B; ++j)
      if (m_first + rstep * j < p.M && ro[j] >= 0) w[(int64_t)p.es * (ro[j] + co)] = signed_result(p, d[j]);
  } else {
#pragma unroll
    for (int j = 0; j < B; ++j)
      if (m_first + rstep * j < p.M && ro[j] >= 0) w[(int64_t)p.es * (ro[j] + co)] += signed_result(p, d[j]);
  }
}

// Compile-time loop: f(std::integral_constant<int, 0>) ... f(..<N-1>).
template <typename F, int... Is>
__device__ __forceinline__ void static_for_impl(F&& f, std::integer_sequence<int, Is...>) {
  (f(std::integral_constant<int, Is>{}), ...);
}
template <int N, typename F>
__device__ __forceinline__ void static_for(F&& f) {
  static_for_impl(f, std::make_integer_sequence<int, N>{});
}


// ---- host side (gemm_tc.cu) ----
// Tensor map over [planes][batches][rows][kpad] elements, box (box_k, box_rows,
// 1, box_planes); 64- or 128-byte swizzle by the box row's bytes.
bool make_map(CUtensorMap* map, const void* base, CUtensorMapDataType type, int64_t kpad, int64_t rows,
              int64_t batches, int64_t planes, int box_k, int box_rows, int box_planes);

// Rounds the split-K sums wacc once to float64 and stores them through the
// tables (a programmatic dependent of the GEMM on `st`).
cudaError_t launch_splitk_round(const Problem& p, const unsigned long long* wacc, const int32_t* eu,
                                const int32_t* ev, const int64_t* wrow, const int64_t* wcol, double* w,
                                const unsigned* err, cudaStream_t st);

}  // namespace symctr
