// Default split form (n_slices = 5) of the aligned contraction on sm_103a:
// 40-bit operands as four FP16 digits of 10 bits, products on the tensor cores
// (TMA -> shared memory -> tcgen05.mma -> TMEM), W's reduced form written from
// the epilogue.
//
// Why FP16 and base 1024.  The operand keeps 39 bits and a sign whatever the
// digits are.  BF16 holds 8 significant bits, so it needs 5 digits and 15
// slice pairs (i + j <= 4); FP16 holds 11, and four balanced digits a_i in
// [-512, 512] need 10 pairs (i + j <= 3): two thirds of the tensor work, and
// four planes instead of five to write and read.  What bounds the digit is the
// FP32 accumulator: it adds integers exactly up to 2^24, i.e. 64 products of
// 2^18.  The dropped pairs (i + j = 4, three of them) weigh 3 x 2^-40 of the
// largest product, against 4 x 2^-40 (four pairs) with 8-bit digits.
//
// Diagonals d = i + j, each in its own TMEM accumulator:
//   d = 0  one pair, <= 2^18 per K: drained every 64 columns of K
//   d = 1  two pairs, <= 2^19 per K: drained every 32 columns (every stage)
//   d = 2  three pairs (weight 2^-20): its multiples of 2^13 move into the sum
//          of diagonal 1 every kFold stages (exact), the rest stays
//   d = 3  four pairs (weight 2^-30): rounded at 2^-24 of its sum, 2^-54 in all
// A drain moves the accumulator's multiple of 8 into an int32 and leaves the
// rest, so the sums are exact.  At the end they make one int64 in units of
// 2^-20 of the d = 0 unit, rounded once to float64 with the row and column
// exponents (integer arithmetic only: GB300 has little float64 throughput).
//
// CTA: 640 threads: warp 0 TMA, warps 1 and 2 MMA, warps 4-19 drains and
// epilogue; one 128 x 128 tile, 512 TMEM columns, three stages of 64 KB.  The
// tile is two halves of 64 columns with their own four accumulators side by
// side: one MMA per A digit takes all the B digits it pairs with (N = 256, 192,
// 128, 64).  Each half has its own issuing thread and its own 8 warps, so that
// its drain (TMEM loads, FP32 and integer adds) runs beside the other half's
// MMAs.  A half beyond N is neither loaded nor multiplied.  Where the wide tiles
// would leave SMs idle, a 128 x 64 tile is a CTA of its own, two to an SM.
//
// What bounds it: a stage's operands cross shared memory at 128 B/clk, 64 KB
// written by TMA and 144 KB read by the MMAs (1664 clocks; the MMAs alone would
// take 1344).  Measured on the CC ladder, clocks per stage: 1580 with drains
// left out, 1930 as it is; 2300 with one 128-column set of accumulators drained
// between MMAs, 2650 with both halves issued by one thread, whose waits leave
// the tensor pipe empty, 2970 for the five BF16 digits before.  Float-to-int
// conversions run at 16 per clock and SM here, so the drains use magic-number
// adds (3470 with conversions).  CC ladder step 6.68 -> 5.59 ms, (2,2,2) with
// D = 23 1.02 -> 0.85 ms, 40960 x 640 x 640 by 10 irreps 5.11 -> 4.44 ms.
// Every wait is bounded (see tc_common.cuh).
#include "tc_common.cuh"

namespace symctr {

namespace {

constexpr int TM = 128;
constexpr int HN = 64;            // columns of a half tile
constexpr int EPI_WARP0 = 4;
constexpr int P4 = 4;             // digit planes
constexpr int ROWB = 64;          // bytes per tile row and stage: 32 FP16, SWIZZLE_64B
constexpr int KSTAGE = 32;
constexpr int kFold = 16;         // stages between folds of diagonal 2 (even)
constexpr int A_BYTES = P4 * TM * ROWB;     // all digits of a stage's A tile
constexpr int B_BYTES = P4 * HN * ROWB;     // of one half's B tile

// H = 2: both halves, one CTA per SM; H = 1: a 128 x 64 tile, two CTAs per SM.
template <int H>
struct Cfg {
  static constexpr int TN = H * HN;
  static constexpr int EPI_WARPS = 8 * H;
  static constexpr int NTHREADS = 128 + 32 * EPI_WARPS;
  static constexpr int STAGES = H == 2 ? 3 : 2;
  static constexpr int STAGE_BYTES = A_BYTES + H * B_BYTES;
  static constexpr int LD = TN + 1;        // epilogue staging stride (doubles)
  static constexpr size_t REGION = (size_t)STAGES * STAGE_BYTES;
  static_assert(REGION >= (size_t)TM * LD * 8, "the epilogue staging fits the stages");
  static constexpr int BARS = 2 * STAGES + 6;
  static constexpr size_t SMEM = 1024 + REGION + 8 * BARS + 12 * (TN + TM) + 16 + 64;
};

// K-major rows of 64 bytes, SWIZZLE_64B, 8-row groups 512 bytes apart.
__device__ __forceinline__ uint64_t sdesc64(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)((8 * ROWB) >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)4 << 61;
  return d;
}

// FP16 operands, FP32 accumulate, K-major, M = 128.
template <int N>
__host__ __device__ constexpr uint32_t idesc() {
  return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(TM >> 4) << 24);
}

// A digit I times B digits 0 .. 3 - I of one half, both K steps of a stage:
// the accumulators of diagonals I .. 3 lie side by side from column 64 I on.
template <int I, int KK>
__device__ __forceinline__ void mma_step(uint32_t acc, uint64_t da, uint64_t db) {
  constexpr int N = (P4 - I) * HN;
  constexpr unsigned long long oa = (I * TM * ROWB + KK * 32) >> 4, ob = (KK * 32) >> 4;
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 a, b;\n\t"
      "add.u64 a, %1, %4;\n\tadd.u64 b, %2, %5;\n\t"
      "setp.ne.b32 p, 1, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, p;\n\t}\n" ::"r"(acc + HN * I),
      "l"(da), "l"(db), "r"(idesc<N>()), "n"(oa), "n"(ob)
      : "memory");
}
template <int I>
__device__ __forceinline__ void mma_digit(uint32_t acc, uint64_t da, uint64_t db) {
  mma_step<I, 0>(acc, da, db);
  mma_step<I, 1>(acc, da, db);
}

struct Tc10Args {
  Problem p;
  int n_kb;          // K stages
  const int32_t* eu; // row exponents of U
  const int32_t* ev; // row exponents of V
  double* w;
  unsigned* err;
  int ksplit;        // K ranges (grid.z = n_q * ksplit)
  int kb_per_split;  // stages per K range
  unsigned long long* wacc;  // [n_q][M][N] int64 partial sums when ksplit > 1 (zeroed)
  const int64_t* wrow;       // [n_q][M] offsets of W's rows in its reduced form
  const int64_t* wcol;       // [n_q][N] offsets of W's columns
  // Complex operands: the digits of real and imaginary parts are 2 n_q batches.
  // One launch multiplies part upart of U by the `parts` parts of V (grid.z =
  // parts * n_q * ksplit), part j into W + woff[j] with sign neg[j].
  int parts, upart;
  int woff[2], neg[2];
};

template <int H, bool GEN>
__global__ void __launch_bounds__(Cfg<H>::NTHREADS, 3 - H)
    gemm_tc10_kernel(const __grid_constant__ CUtensorMap tma_a, const __grid_constant__ CUtensorMap tma_b,
                     const __grid_constant__ Tc10Args args) {
  using C = Cfg<H>;
  constexpr int TN = C::TN, STAGES = C::STAGES, STAGE_BYTES = C::STAGE_BYTES, LD = C::LD;
  constexpr int EPI_WARPS = C::EPI_WARPS;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const Problem& p = args.p;
  uint8_t* tiles = smem;  // [STAGES][A digits, B digits of half 0, of half 1], later the epilogue staging
  uint64_t* full = (uint64_t*)(smem + C::REGION);
  uint64_t* empty = full + STAGES;
  uint64_t* go = empty + STAGES;         // [2] a half's MMAs of a stage are done: drain
  uint64_t* drained = go + 2;            // [2] its accumulators may be written again
  uint64_t* acc_full = drained + 2;
  uint64_t* zero_done = acc_full + 1;
  int64_t* coff = (int64_t*)(zero_done + 1);   // [TN] W column offsets
  int64_t* roffs = coff + TN;                  // [TM] W row offsets
  int32_t* cexp = (int32_t*)(roffs + TM);      // [TN] column exponents
  int32_t* rexps = cexp + TN;                  // [TM] row exponents
  uint32_t* tmem_slot = (uint32_t*)(rexps + TM);
  Ctl* ctl = (Ctl*)(tmem_slot + 4);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t n0 = (int64_t)blockIdx.x * TN, m0 = (int64_t)blockIdx.y * TM;
  const int zb = blockIdx.z / args.ksplit;       // part * n_q + irrep
  const int ks = blockIdx.z % args.ksplit;
  const int part_v = zb >= p.n_q ? 1 : 0, b = zb - part_v * p.n_q;
  const int ub = b + args.upart * p.n_q;         // U's batch (V's is zb)
  const int kb0 = ks * args.kb_per_split;
  const int n_kb = min(args.n_kb, kb0 + args.kb_per_split) - kb0;
  const int halves = H == 2 && p.N - n0 > HN ? 2 : 1;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], halves);
    }
    for (int h = 0; h < 2; ++h) {
      mbar_init(&go[h], 1);
      mbar_init(&drained[h], 8);
    }
    mbar_init(acc_full, halves);
    mbar_init(zero_done, 8 * halves);
    ctl->abort = 0;
    ctl->err = args.err;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tmem_slot)),
                 "n"(4 * TN)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  // W's offset tables are constants of the plan: read before the wait.
  const int et = (int)threadIdx.x - EPI_WARP0 * 32;   // epilogue thread
  if (et >= 0 && et < TM) {
    roffs[et] = m0 + et < p.M ? args.wrow[(int64_t)b * p.M + m0 + et] : -1;
    if (et < TN) coff[et] = n0 + et < p.N ? args.wcol[(int64_t)b * p.N + n0 + et] : -1;
  }
  // Launched as a programmatic dependent of the operand preparation: the setup
  // above overlaps its tail; everything below reads its outputs.
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (et >= 0 && et < TM) {
    rexps[et] = m0 + et < p.M ? args.eu[(int64_t)ub * p.M + m0 + et] - kExpBias : 0;
    if (et < TN) cexp[et] = n0 + et < p.N ? args.ev[(int64_t)zb * p.N + n0 + et] - kExpBias : 0;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  // registers: part of the producer warpgroup's share goes to the running sums
  // (H = 2: 56 x 128 + 104 x 512, less than the 96 x 640 of the launch; H = 1:
  // 32 x 128 + 104 x 256, the 80 x 384 of the launch)
  if (warp < EPI_WARP0) {
    if constexpr (H == 2) asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
    else asm volatile("setmaxnreg.dec.sync.aligned.u32 32;");
  }
  if (warp == 0) {
    // ------------------------------------------------------------ producer
    if (lane == 0) {
      int issued = 0;
      for (int kb = 0; kb < n_kb; ++kb) {
        const int st = kb % STAGES;
        if (!wait_phase(&empty[st], ((kb / STAGES) & 1) ^ 1, ctl)) break;
        mbar_expect_tx(&full[st], A_BYTES + halves * B_BYTES);
        uint8_t* sa = tiles + (size_t)st * STAGE_BYTES;
        // all four digit tiles of an operand in one copy
        const int kc = (kb0 + kb) * KSTAGE;
        tma_load_4d(&tma_a, &full[st], sa, kc, (int)m0, ub);
        tma_load_4d(&tma_b, &full[st], sa + A_BYTES, kc, (int)n0, zb);
        if (halves == 2) tma_load_4d(&tma_b, &full[st], sa + A_BYTES + B_BYTES, kc, (int)n0 + HN, zb);
        ++issued;
      }
      if (ctl->abort) {
        // let the copies this thread issued land before the CTA exits
        for (int kb = issued > STAGES ? issued - STAGES : 0; kb < issued; ++kb)
          wait_phase(&full[kb % STAGES], (kb / STAGES) & 1, ctl, kTimeoutCycles / 2);
      }
    }
  } else if (warp <= halves) {
    // ------------------------------------------------------------ MMA issuers
    // warp 1 + h issues half h: a thread that waits for one half's drain leaves
    // the other's MMAs flowing
    if (lane == 0) {
      const int h = warp - 1;
      const uint32_t ab = su32(tiles);
      const uint32_t acc = tmem + 4 * HN * h;
      // the epilogue warps have zeroed the accumulators
      bool ok = wait_phase(zero_done, 0, ctl);
      for (int kb = 0; ok && kb < n_kb; ++kb) {
        const int st = kb % STAGES;
        ok = wait_phase(&full[st], (kb / STAGES) & 1, ctl);
        if (!ok) break;
        tc_fence_after();
        const uint64_t da = sdesc64(ab + st * STAGE_BYTES);
        const uint64_t db = sdesc64(ab + st * STAGE_BYTES + A_BYTES + h * B_BYTES);
        // the digits that touch only diagonals 2 and 3 do not wait for the
        // half's drain (but the second does for a fold)
        const bool folding = kb % kFold == 0;
        mma_digit<3>(acc, da, db);
        if (!folding) mma_digit<2>(acc, da, db);
        if (kb > 0) {
          ok = wait_phase(&drained[h], (kb - 1) & 1, ctl);
          if (!ok) break;
          tc_fence_after();
        }
        if (folding) mma_digit<2>(acc, da, db);
        mma_digit<1>(acc, da, db);
        mma_digit<0>(acc, da, db);
        if (kb + 1 < n_kb) tc_commit(&go[h]);
        tc_commit(&empty[st]);
      }
      tc_commit(acc_full);
      // (also keeps the MMAs in flight from outliving the CTA after an abort)
      wait_phase(acc_full, 0, ctl, kTimeoutCycles / 2);
    }
  } else if (warp >= EPI_WARP0) {
    // ------------------------------------------------------------ epilogue
    // 8 warps to a half: a thread keeps 32 columns of one row
    asm volatile("setmaxnreg.inc.sync.aligned.u32 104;");
    const int ew = warp - EPI_WARP0;      // 0..15
    const int quad = warp & 3;            // TMEM lane quadrant this warp may access
    const int h = ew >> 3, part = (ew >> 2) & 1;   // half of the tile, half of its columns
    const int row = quad * 32 + lane;
    // accumulator of diagonal d: lane_base + 64 d
    const uint32_t lane_base = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(4 * HN * h + part * 32);
    // Running sums in units 8 (s0) and 8 x 2^-10 (s1): a drain moves the
    // accumulator's multiple of 8 and leaves |rest| <= 4 in TMEM.  Per column of
    // K they gain 2^15 and 2^16 + 3 x 2^5 at most, and every fold carries s1
    // into s0: int32 holds a K range of up to 32768 columns.
    int32_t s0[32], s1[32];
#pragma unroll
    for (int j = 0; j < 32; ++j) s0[j] = s1[j] = 0;
    const float M8 = 100663296.0f;             // 1.5 * 2^26: ulp 8, |x| <= 2^25
    const int32_t B8 = (int32_t)__float_as_uint(M8);
    const float M0 = 12582912.0f;              // 1.5 * 2^23: ulp 1
    const int32_t B0 = (int32_t)__float_as_uint(M0);
    // s += a's multiples of 8, a = what is left
    auto drain16 = [&](uint32_t* a, int32_t* s) {
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const float x = __uint_as_float(a[j]);
        const float r = x + M8;
        s[j] += (int32_t)__float_as_uint(r) - B8;
        a[j] = __float_as_uint(x - (r - M8));   // exact
      }
    };
    // The half after stage kb: its diagonal 1 (32 columns of this thread) and
    // every second stage, in turns, 16 of diagonal 0; all of diagonal 2 after
    // kFold stages.
    auto drain = [&](auto ODD, int kb) {
      constexpr int o = decltype(ODD)::value * 16;
      if (!wait_phase_sleep(&go[h], (uint32_t)kb & 1, ctl)) return false;
      tc_fence_after();
      uint32_t a[16];
      auto drain_at = [&](uint32_t at, int32_t* s) {
        tmem_ld16(at, a);
        tmem_wait_ld();
        tmem_loaded<16>(a);
        drain16(a, s);
        tmem_st16(at, a);
      };
      drain_at(lane_base + HN, s1);
      drain_at(lane_base + HN + 16, s1 + 16);
      drain_at(lane_base + o, s0 + o);
      if (o != 0 && (kb + 1) % kFold == 0) {
        // diagonal 2 (the MMAs that write it wait): multiples of 2^13 = 8 x 2^10
        // to s1, |rest| <= 2^12 stays
#pragma unroll
        for (int pc = 0; pc < 2; ++pc) {
          tmem_ld16(lane_base + 2 * HN + pc * 16, a);
          tmem_wait_ld();
          tmem_loaded<16>(a);
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const float x = __uint_as_float(a[j]);
            const float r = __fmaf_rn(x, 1.0f / 8192.0f, M0);   // round(x / 2^13) + 1.5 * 2^23
            int32_t& t = s1[pc * 16 + j];
            t += (int32_t)__float_as_uint(r) - B0;
            a[j] = __float_as_uint(__fmaf_rn(r - M0, -8192.0f, x));   // exact
            s0[pc * 16 + j] += t >> 10;
            t &= 1023;
          }
          tmem_st16(lane_base + 2 * HN + pc * 16, a);
        }
      }
      tmem_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&drained[h]);
      return true;
    };
    static_assert(kFold % 2 == 0, "folds follow odd stages");
    bool ok = true;
    if (h < halves) {
      // the accumulators start from zero (every MMA accumulates)
#pragma unroll
      for (int d = 0; d < 4; ++d)
#pragma unroll
        for (int pc = 0; pc < 2; ++pc) tmem_zero_w<16>(lane_base + HN * d + pc * 16);
      tmem_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(zero_done);
      // two stages a turn: the parts of diagonal 0 are compile-time
      for (int kb = 0; ok && kb + 1 < n_kb; kb += 2) {
        ok = drain(std::integral_constant<int, 0>{}, kb);
        if (ok && kb + 2 < n_kb) ok = drain(std::integral_constant<int, 1>{}, kb + 1);
      }
    }
    if (ok) ok = wait_phase_sleep(acc_full, 0, ctl);
    ok = ok && !ctl->abort;
    if (ok && h < halves) {
      tc_fence_after();
      // The last stages and the running sums as one int64 in units of 2^-20,
      // staged through shared memory (the operand stages are free by now).
      int64_t* st64 = (int64_t*)tiles + row * LD + h * HN + part * 32;
#pragma unroll
      for (int pc = 0; pc < 8; ++pc) {
        uint32_t a0[4], a1[4], a2[4], a3[4];
        const uint32_t at = lane_base + pc * 4;
        tmem_ld4(at, a0);
        tmem_ld4(at + HN, a1);
        tmem_ld4(at + 2 * HN, a2);
        tmem_ld4(at + 3 * HN, a3);
        tmem_wait_ld();
        tmem_loaded<4>(a0);
        tmem_loaded<4>(a1);
        tmem_loaded<4>(a2);
        tmem_loaded<4>(a3);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          // multiples of 8 of the exact diagonals by the magic number, as in the
          // drains, their rests (an integer below 2^13) likewise; diagonals 2 and 3
          // (|.| < 2^29) as one FP32 number and the only conversion
          const float x0 = __uint_as_float(a0[j]), x1 = __uint_as_float(a1[j]);
          const float r0 = x0 + M8, r1 = x1 + M8;
          const int32_t t0 = s0[pc * 4 + j] + ((int32_t)__float_as_uint(r0) - B8);
          const int32_t t1 = s1[pc * 4 + j] + ((int32_t)__float_as_uint(r1) - B8);
          const float low = __fmaf_rn(__uint_as_float(a3[j]), 1.0f / 1024.0f, __uint_as_float(a2[j]));
          const float rest = __fmaf_rn(x0 - (r0 - M8), 1024.0f, x1 - (r1 - M8));
          const int32_t l = (((int32_t)__float_as_uint(rest + M0) - B0) << 10) + __float2int_rn(low);
          st64[pc * 4 + j] = ((long long)t0 << 23) + ((long long)t1 << 13) + l;
        }
      }
    }
    tc_fence_before();
    // all epilogue threads meet here, whatever path they took
    asm volatile("bar.sync 1, %0;" ::"n"(EPI_WARPS * 32) : "memory");
    if (ok) {
      // a warp per row: lane l rounds and writes columns l, l + 32, ...; two rows
      // at a time (one was bound by the latency of its conversions)
      constexpr int NC = TN / 32;
      const int nrow = (int)min((int64_t)TM, p.M - m0), ncol = (int)min((int64_t)TN, p.N - n0);
      const long long* R0 = (const long long*)tiles + lane;
      if (args.ksplit > 1) {
        unsigned long long* acc = args.wacc + ((int64_t)zb * p.M + m0) * p.N + n0 + lane;
#pragma unroll 1
        for (int r = ew; r < nrow; r += EPI_WARPS) {
#pragma unroll
          for (int j = 0; j < NC; ++j)
            if (lane + 32 * j < ncol)
              red_add_u64(acc + (int64_t)r * p.N + 32 * j, (unsigned long long)R0[r * LD + 32 * j]);
        }
      } else {
        OutMode wp;
        wp.negate = args.neg[part_v];
        wp.accumulate = p.accumulate;
        int64_t co[NC];
        int ce[NC];
#pragma unroll
        for (int j = 0; j < NC; ++j) co[j] = coff[lane + 32 * j], ce[j] = cexp[lane + 32 * j] - 36;
#pragma unroll 2
        for (int r = ew; r < nrow; r += EPI_WARPS) {
          const int64_t ro = roffs[r];
          const int re = rexps[r];
          long long R[NC];
          int ex[NC];
          double d[NC];
#pragma unroll
          for (int j = 0; j < NC; ++j) R[j] = R0[r * LD + 32 * j], ex[j] = re + ce[j];
          i64_scaled_batch<NC>(R, ex, d);
          if (ro < 0) continue;   // general plans: a row absent from W
#pragma unroll
          for (int j = 0; j < NC; ++j) {
            if (co[j] < 0) continue;   // beyond N, or a column absent from W
            if constexpr (!GEN) {
              args.w[ro + co[j]] = d[j];
            } else {
              store_w(wp, args.w + args.woff[part_v] + (int64_t)p.es * (ro + co[j]), d[j]);
            }
          }
        }
      }
    }
  }
  // a split-K rounding kernel behind this one may start its launch now
  asm volatile("griddepcontrol.launch_dependents;");
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(4 * TN) : "memory");
  }
}

template <int H, bool GEN>
cudaError_t launch_mode(const Problem& p, const Tables& tab, const void* a, const void* bop, const int32_t* eu,
                        const int32_t* ev, int64_t kpad, double* w, unsigned* err, int ksplit,
                        unsigned long long* wacc, const ComplexParts* cx, cudaStream_t st) {
  using C = Cfg<H>;
  constexpr int TN = C::TN;
  const int64_t batches = cx ? 2 * p.n_q : p.n_q;
  CUtensorMap ma, mb;
  if (!make_map(&ma, a, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, kpad, p.M, batches, P4, KSTAGE, TM, P4) ||
      !make_map(&mb, bop, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, kpad, p.N, batches, P4, KSTAGE, HN, P4))
    return cudaErrorInvalidValue;
  Tc10Args args;
  args.p = p;
  args.n_kb = (int)(kpad / KSTAGE);
  args.eu = eu;
  args.ev = ev;
  args.w = w;
  args.err = err;
  if (ksplit < 1) ksplit = 1;
  args.kb_per_split = (args.n_kb + ksplit - 1) / ksplit;
  args.ksplit = (args.n_kb + args.kb_per_split - 1) / args.kb_per_split;
  args.wacc = wacc;
  args.wrow = tab.wrow;
  args.wcol = tab.wcol;
  args.parts = cx ? 2 : 1;
  args.upart = cx ? cx->upart : 0;
  for (int j = 0; j < 2; ++j) {
    args.woff[j] = cx ? cx->woff[j] : 0;
    args.neg[j] = cx ? cx->neg[j] : p.negate;
  }
  auto kern = gemm_tc10_kernel<H, GEN>;
  thread_local bool attr_set[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) dev = 0;
  if (!attr_set[dev]) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM);
    if (e != cudaSuccess) return e;
    attr_set[dev] = true;
  }
  const int64_t gx = (p.N + TN - 1) / TN, gy = (p.M + TM - 1) / TM;
  const int64_t gz = (int64_t)args.parts * p.n_q * args.ksplit;
  if (gx > 0x7FFFFFFF || gy > 65535 || gz > 65535) return cudaErrorInvalidConfiguration;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)gx, (unsigned)gy, (unsigned)gz);
  cfg.blockDim = dim3(C::NTHREADS);
  cfg.dynamicSmemBytes = C::SMEM;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaError_t le = cudaLaunchKernelEx(&cfg, kern, ma, mb, args);
  ++g_kernel_launches;
  if (le != cudaSuccess || args.ksplit == 1) return le;
  for (int j = 0; j < args.parts && le == cudaSuccess; ++j) {
    Problem pj = p;
    pj.negate = args.neg[j];
    le = launch_splitk_round(pj, wacc + (int64_t)j * p.n_q * p.M * p.N, eu + (int64_t)args.upart * p.n_q * p.M,
                             ev + (int64_t)j * p.n_q * p.N, tab.wrow, tab.wcol, w + args.woff[j], err, st);
  }
  return le;
}

template <int H>
cudaError_t launch_tile(const Problem& p, const Tables& tab, const void* a, const void* bop, const int32_t* eu,
                        const int32_t* ev, int64_t kpad, double* w, unsigned* err, int ksplit,
                        unsigned long long* wacc, const ComplexParts* cx, cudaStream_t st) {
  if (p.es == 1 && !p.negate && !p.accumulate)
    return launch_mode<H, false>(p, tab, a, bop, eu, ev, kpad, w, err, ksplit, wacc, cx, st);
  return launch_mode<H, true>(p, tab, a, bop, eu, ev, kpad, w, err, ksplit, wacc, cx, st);
}

}  // namespace

cudaError_t launch_gemm_split10(const Problem& p, const Tables& tab, const uint16_t* us, const uint16_t* vs,
                                const int32_t* eu, const int32_t* ev, int64_t kpad, double* w, unsigned* err,
                                int ksplit, unsigned long long* wacc, const ComplexParts* cx, cudaStream_t st) {
  // The narrower tile where it takes fewer rounds of the SMs.  Clocks measured
  // per stage and per tile: 1930 and 17000 for a 128 x 128 tile, 2270 and 20000
  // for two 128 x 64 tiles side by side (they load the A digits twice: 4650
  // against 4100 us for the CC ladder, but 1285 x 192 x 738 by 8 irreps, 176
  // wide or 264 narrow tiles, takes 103 us instead of 129, preparation included).
  const int sms = device_sms();
  const int64_t split = ksplit < 1 ? 1 : ksplit, blocks = ((p.M + TM - 1) / TM) * p.n_q * split * (cx ? 2 : 1);
  const int64_t n_kb = (kpad / KSTAGE + split - 1) / split;
  const int64_t wide = blocks * ((p.N + 2 * HN - 1) / (2 * HN)), narrow = blocks * ((p.N + HN - 1) / HN);
  const double t2 = (double)((wide + sms - 1) / sms) * (1930.0 * n_kb + 17000.0);
  const double t1 = (double)((narrow + 2 * sms - 1) / (2 * sms)) * (2270.0 * n_kb + 20000.0);
  if (t1 < 0.9 * t2) return launch_tile<1>(p, tab, us, vs, eu, ev, kpad, w, err, ksplit, wacc, cx, st);
  return launch_tile<2>(p, tab, us, vs, eu, ev, kpad, w, err, ksplit, wacc, cx, st);
}

}  // namespace symctr
