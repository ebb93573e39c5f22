// Default split form (n_slices = 5) of the aligned contraction on sm_103a:
// 40-bit operands as four FP16 digits of 10 bits, products on the tensor cores
// (TMA -> shared memory -> tcgen05.mma -> TMEM), W's reduced form written from
// the epilogue.
//
// Why FP16 and base 1024.  The operand keeps 39 bits and a sign whatever the
// digits are.  BF16 holds 8 significant bits, so it needs 5 digits and 15
// slice pairs (i + j <= 4); FP16 holds 11, and four balanced digits a_i in
// [-512, 511] need 10 pairs (i + j <= 3): two thirds of the tensor work, and
// four planes instead of five to write and read.  What bounds the digit is the
// FP32 accumulator: it adds integers exactly up to 2^24, i.e. 64 products of
// just below 2^18.  The dropped pairs (i + j = 4, three of them) weigh 3 x 2^-40
// of the largest product, against 4 x 2^-40 (four pairs) with 8-bit digits.
//
// Diagonals d = i + j, each in its own TMEM accumulator; the leading digit is at
// most 511 (row_exponent raises a row's scale where it would be 512):
//   d = 0  one pair, <= 511^2 per K: drained every 64 columns of K,
//          64 x 511^2 + 4 = 2^24 - 65468
//   d = 1  two pairs, <= 2 x 511 x 512 per K: drained every 32 columns (every
//          stage), 32 x 2 x 511 x 512 + 4 = 2^24 - 32764
//   d = 2  three pairs (weight 2^-20): an FP32 sum that reaches 3 x 2^27 in 17
//          stages and is then rounded to 2^5 in each MMA, 2^-37 of its 16
//          largest products at worst (lower digits all at their limits and of
//          one sign; random ones stay below 2^24 and exact); its multiples of
//          2^13 move into the sum of diagonal 1 every kFold stages, the rest stays
//   d = 3  four pairs (weight 2^-30): rounded at 2^-24 of its sum, 2^-54 in all
// A drain moves the accumulator's multiple of 8 into an int32 and leaves the
// rest of at most 4, so the sums of diagonals 0 and 1 are exact.  At the end all
// make one int64 in units of 2^-20 of the d = 0 unit, rounded once to float64
// with the row and column exponents (integer arithmetic only: GB300 has little
// float64 throughput).
//
// CTA: 640 threads: warp 0 TMA, warps 1 and 2 MMA, warps 4-19 drains and
// epilogue; 128 x 128 tiles, 512 TMEM columns, three stages of 64 KB.  The grid is
// resident as a whole and each CTA walks tiles one grid apart: the next tile's
// first loads and MMAs run beside the rounding and writing of the last one.  The
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
// adds (3470 with conversions).  CC ladder step 6.68 -> 5.49 ms, (2,2,2) with
// D = 23 1.02 -> 0.81 ms, 40960 x 640 x 640 by 10 irreps 5.11 -> 3.59 ms (3.99
// with a CTA to a tile and the longer writes, 3.70 with those alone).
// The drain loop leaves no register to spare: with 80 bytes of spills instead of
// 32 that last case takes 4.01 ms (the 128 x 64 tile, at 80 registers a thread for
// two CTAs, spills 108).
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
// Whether diagonal 2 is folded in the drain that has `left` drains behind it (only
// every second drain folds: the first in a pair asks nothing).  Counted from the
// end, so that a K range of kFold stages has none.
__device__ __forceinline__ bool folds_after(int left) { return (left / 2) % (kFold / 2) == kFold / 2 - 1; }
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
  static constexpr size_t REGION = (size_t)STAGES * STAGE_BYTES;
  // The epilogue staging (TM x TN 64-bit words) overlays the first stages; a tile
  // starts with stage FIRST, which at H = 2 lies behind it.
  static constexpr size_t STAGING = (size_t)TM * TN * 8;
  static_assert(REGION >= STAGING, "the epilogue staging fits the stages");
  static constexpr int FIRST = STAGES - 1;
  static constexpr bool EARLY = (size_t)FIRST * STAGE_BYTES >= STAGING;   // loads beside the epilogue
  static constexpr int BARS = 2 * STAGES + 9;
  static constexpr int TAB = 12 * (TN + TM);      // offsets and exponents of a tile
  static constexpr size_t SMEM = REGION + 8 * BARS + 2 * TAB + 16 + 64;
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
  int gx, gy;        // column and row blocks
  uint32_t tiles;    // gx * gy * parts * n_q * ksplit
};

// Rv[j] * 2^e[j] as float64 (exact) for |Rv| < 2^53 and results that are 0 or
// normal; false if an even entry is not in [-2^51, 2^51).  The selects and shifts of the integer way run at half rate and took
// most of a tile's write phase (11300 clocks); every second value goes through
// the float64 pipe instead, which is otherwise idle (one addition against
// 1.5 * 2^52, 2 per clock and SM, so not all of them: 16384 would take 8200).
// 40960 x 640 x 640 by 10 irreps 3.70 -> 3.59 ms (3.79 with all of them there),
// the CC ladder with 16 irreps and gradients 6.08 -> 5.90 ms.
template <int B>
__device__ __forceinline__ bool i64_scaled_small(const long long (&Rv)[B], const int (&e)[B], double (&d)[B]) {
  uint32_t out = 0;
#pragma unroll
  for (int j = 0; j < B; ++j) {
    const uint32_t lo = (uint32_t)Rv[j], hi = (uint32_t)((unsigned long long)Rv[j] >> 32);
    if (j % 2 == 0) {
      out |= (hi + 0x43380000u) ^ 0x43300000u;
      const double x = __hiloint2double((int)(hi + 0x43380000u), (int)lo) - 6755399441055744.0;
      const int h = __double2hiint(x);
      d[j] = __hiloint2double(h == 0 ? 0 : h + (e[j] << 20), __double2loint(x));
    } else {
      const uint64_t sm = (uint64_t)(Rv[j] >> 63);
      const uint64_t m = ((uint64_t)Rv[j] ^ sm) - sm;
      const int lz = __clzll((long long)m);
      const uint64_t q = m << ((lz - 11) & 63);     // the leading one at bit 52
      const uint32_t h = (uint32_t)(q >> 32) + ((uint32_t)(e[j] + 63 - lz + 1022) << 20);
      d[j] = __hiloint2double((int)(m == 0 ? 0u : h | ((uint32_t)sm & 0x80000000u)), (int)(uint32_t)q);
    }
  }
  return out >> 20 == 0;
}

// The thread's index, read again.
__device__ __forceinline__ int tid_again() {
  int t;
  asm volatile("mov.u32 %0, %%tid.x;" : "=r"(t));
  return t;
}

// Whether `ok` holds for all of the N threads that meet here (named barrier 1).
template <int N>
__device__ __forceinline__ bool all_ok(bool ok) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\t"
      "barrier.cta.red.and.pred.aligned q, 1, %2, p;\n\tselp.u32 %0, 1, 0, q;\n\t}\n"
      : "=r"(r)
      : "r"((uint32_t)ok), "n"(N)
      : "memory");
  return r != 0;
}

// After an abort, before the CTA gives its memory back (out of line: see wait_landed):
// thread i < STAGES waits for the last copy into stage i, the issuing threads for
// their MMAs.
template <int H>
__device__ __noinline__ void land10(uint64_t* full, uint64_t* issued, Ctl* ctl) {
  const int t = threadIdx.x, h = t / 32 - 1;
  uint64_t* bar = nullptr;
  if (t < Cfg<H>::STAGES && ((ctl->copies >> t) & 1)) bar = &full[t];
  if (t % 32 == 0 && h >= 0 && h < H) {
    bar = &issued[h];
    tc_commit(bar);
  }
  if (bar) wait_landed(bar, t < Cfg<H>::STAGES ? ((ctl->phases >> t) & 1) ^ 1 : 0, ctl);
}

template <int H, bool GEN>
__global__ void __launch_bounds__(Cfg<H>::NTHREADS, 3 - H)
    gemm_tc10_kernel(const __grid_constant__ CUtensorMap tma_a, const __grid_constant__ CUtensorMap tma_b,
                     const __grid_constant__ Tc10Args args) {
  using C = Cfg<H>;
  constexpr int TN = C::TN, STAGES = C::STAGES, STAGE_BYTES = C::STAGE_BYTES;
  constexpr int EPI_WARPS = C::EPI_WARPS;
  // (alignment by declaration: addresses within are constants, not registers)
  extern __shared__ __align__(1024) uint8_t smem[];
  const Problem& p = args.p;
  uint8_t* tiles = smem;  // [STAGES][A digits, B digits of half 0, of half 1], also the epilogue staging
  uint64_t* full = (uint64_t*)(smem + C::REGION);
  uint64_t* empty = full + STAGES;
  uint64_t* go = empty + STAGES;         // [2] a half's MMAs of a stage are done: drain
  uint64_t* drained = go + 2;            // [2] its accumulators may be written again
  uint64_t* acc_full = drained + 2;      // a tile's MMAs are done
  uint64_t* zero_done = acc_full + 1;    // its accumulators are read out and zeroed
  uint64_t* staged = zero_done + 1;      // its results have left the staging
  uint64_t* issued = staged + 1;         // [2] after an abort: all of an issuing thread's MMAs are done
  uint8_t* tabs = (uint8_t*)(issued + 2);      // [2] tables of this tile and the last one
  uint32_t* tmem_slot = (uint32_t*)(tabs + 2 * C::TAB);
  Ctl* ctl = (Ctl*)(tmem_slot + 4);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // Tile t: column block fastest (its neighbours share the rows of U).
  struct Tile {
    int n0, m0;
    int ub, vb, b, part;      // U's and V's batch, irrep, part of W (complex)
    int kb0, n_kb, halves;    // K range
  };
  auto tile_at = [&](uint32_t t) {
    Tile x;
    const uint32_t g = t / (uint32_t)args.gx, z = g / (uint32_t)args.gy;
    x.n0 = (int)(t - g * (uint32_t)args.gx) * TN;
    x.m0 = (int)(g - z * (uint32_t)args.gy) * TM;
    x.vb = (int)(z / (uint32_t)args.ksplit);      // part * n_q + irrep
    const int ks = (int)z - x.vb * args.ksplit;
    x.part = x.vb >= p.n_q ? 1 : 0;
    x.b = x.vb - x.part * p.n_q;
    x.ub = x.b + args.upart * p.n_q;
    x.kb0 = ks * args.kb_per_split;
    x.n_kb = min(args.n_kb, x.kb0 + args.kb_per_split) - x.kb0;
    x.halves = H == 2 && p.N - x.n0 > HN ? 2 : 1;
    return x;
  };

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], H);
    }
    for (int h = 0; h < 2; ++h) {
      mbar_init(&go[h], 1);
      mbar_init(&drained[h], 8);
      mbar_init(&issued[h], 1);
    }
    mbar_init(acc_full, H);
    mbar_init(zero_done, 8 * H);
    mbar_init(staged, 8 * H);
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
  // Launched as a programmatic dependent of the operand preparation: the setup
  // above overlaps its tail; everything below reads its outputs.
  asm volatile("griddepcontrol.wait;" ::: "memory");
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
      uint32_t ph = 0;          // bit s: parity of stage s's next use
      int n_tile = 0, st = 0;
      bool ok = true;
      uint32_t live = 0;        // stages with a copy issued
      for (uint32_t t = blockIdx.x; ok && t < args.tiles; t += gridDim.x, ++n_tile) {
        const Tile x = tile_at(t);
        st = C::FIRST;
        for (int kb = 0; kb < x.n_kb; ++kb) {
          // the stages under the last tile's staging wait until it is read out
          // (one phase a tile, waited for before this tile's last stage is loaded)
          const int under = C::EARLY && x.n_kb > 1 ? 1 : 0;
          if (n_tile > 0 && kb == under) ok = wait_phase(staged, (n_tile - 1) & 1, ctl);
          ok = ok && wait_phase(&empty[st], ((ph >> st) & 1) ^ 1, ctl);
          if (!ok) break;
          mbar_expect_tx(&full[st], A_BYTES + x.halves * B_BYTES);
          uint8_t* sa = tiles + (size_t)st * STAGE_BYTES;
          // all four digit tiles of an operand in one copy
          const int kc = (x.kb0 + kb) * KSTAGE;
          tma_load_4d(&tma_a, &full[st], sa, kc, x.m0, x.ub);
          tma_load_4d(&tma_b, &full[st], sa + A_BYTES, kc, x.n0, x.vb);
          if (x.halves == 2) tma_load_4d(&tma_b, &full[st], sa + A_BYTES + B_BYTES, kc, x.n0 + HN, x.vb);
          ph ^= 1u << st;
          live |= 1u << st;
          st = st + 1 == STAGES ? 0 : st + 1;
        }
      }
      ctl->copies = live;
      ctl->phases = ph;
    }
  } else if (warp <= H) {
    // ------------------------------------------------------------ MMA issuers
    // warp 1 + h issues half h: a thread that waits for one half's drain leaves
    // the other's MMAs flowing
    if (lane == 0) {
      const int h = warp - 1;
      const uint32_t ab = su32(tiles);
      const uint32_t acc = tmem + 4 * HN * h;
      uint32_t ph = 0, it = 0;  // bit s of ph: parity of stage s's next use
      bool ok = true;
      for (uint32_t t = blockIdx.x; ok && t < args.tiles; t += gridDim.x, ++it) {
        int n_kb;
        bool mine;
        {
          const Tile x = tile_at(t);
          n_kb = x.n_kb, mine = h < x.halves;
        }
        // the epilogue warps have read out the last tile and zeroed the accumulators
        ok = wait_phase(zero_done, it & 1, ctl);
        int st = C::FIRST;
        for (int kb = 0; ok && kb < n_kb; ++kb) {
          ok = wait_phase(&full[st], (ph >> st) & 1, ctl);
          if (!ok) break;
          ph ^= 1u << st;
          tc_fence_after();
          if (mine) {
            const uint64_t da = sdesc64(ab + st * STAGE_BYTES);
            const uint64_t db = sdesc64(ab + st * STAGE_BYTES + A_BYTES + h * B_BYTES);
            // the digits that touch only diagonals 2 and 3 do not wait for the
            // half's drain (but the second does for a fold)
            const bool folding = kb > 0 && !(kb & 1) && folds_after(n_kb - 1 - kb);
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
            // (an even number of phases a tile: the drains' parities start from 0)
            if (kb + 1 < n_kb || (kb & 1)) tc_commit(&go[h]);
          }
          tc_commit(&empty[st]);
          st = st + 1 == STAGES ? 0 : st + 1;
        }
        tc_commit(acc_full);
      }
    }
  } else if (warp >= EPI_WARP0) {
    // ------------------------------------------------------------ epilogue
    // 8 warps to a half: a thread keeps 32 columns of one row
    asm volatile("setmaxnreg.inc.sync.aligned.u32 104;");
    const int ew = warp - EPI_WARP0;      // 0..15
    const int quad = warp & 3;            // TMEM lane quadrant this warp may access
    const int h = ew >> 3, part = (ew >> 2) & 1;   // half of the tile, half of its columns
    // accumulator of diagonal d: lane_base + 64 d
    const uint32_t lane_base = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(4 * HN * h + part * 32);
    // Running sums in units 8 (s0) and 8 x 2^-10 (s1): a drain moves the
    // accumulator's multiple of 8 and leaves |rest| <= 4 in TMEM.  Per column of
    // K they gain 2^15 and 2^16 + 3 x 2^5 at most, and every fold carries s1
    // into s0: int32 holds a K range of up to 32768 columns.
    int32_t s0[32], s1[32];
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
    auto drain = [&](auto ODD, int left) {
      constexpr int o = decltype(ODD)::value * 16;
      if (!wait_phase_sleep(&go[h], decltype(ODD)::value, ctl)) return false;
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
      if (o != 0 && folds_after(left)) {
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
    // the accumulators start from zero (every MMA accumulates)
    auto zero = [&] {
#pragma unroll
      for (int d = 0; d < 4; ++d)
#pragma unroll
        for (int pc = 0; pc < 2; ++pc) tmem_zero_w<16>(lane_base + HN * d + pc * 16);
      tmem_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(zero_done);
    };
    zero();
    bool ok = true;
    // stages of tile t for the half of epilogue thread et
    auto my_stages = [&](uint32_t t, int et) {
      const Tile x = tile_at(t);
      return (et >> 8) < x.halves ? x.n_kb : 0;
    };
    for (uint32_t it = 0;; ++it) {
      int left;          // drains to come
      {
        const uint32_t t = blockIdx.x + it * gridDim.x;
        if (t >= args.tiles) break;
        const Tile x = tile_at(t);
        const int et = tid_again() - EPI_WARP0 * 32;
        left = my_stages(t, et) - 1;
        // this tile's offsets in W and exponents, beside the last one's, which other
        // warps may still read
        int64_t* coff = (int64_t*)(tabs + (it & 1) * C::TAB);
        int64_t* roffs = coff + TN;
        int32_t* cexp = (int32_t*)(roffs + TM);
        int32_t* rexps = cexp + TN;
        if (et < TM) {
          const bool rok = x.m0 + et < p.M;
          roffs[et] = rok ? args.wrow[(int64_t)x.b * p.M + x.m0 + et] : -1;
          rexps[et] = rok ? args.eu[(int64_t)x.ub * p.M + x.m0 + et] - kExpBias : 0;
          if (et < TN) {
            const bool cok = x.n0 + et < p.N;
            coff[et] = cok ? args.wcol[(int64_t)x.b * p.N + x.n0 + et] : -1;
            cexp[et] = cok ? args.ev[(int64_t)x.vb * p.N + x.n0 + et] - kExpBias : 0;
          }
        }
      }
#pragma unroll
      for (int j = 0; j < 32; ++j) s0[j] = s1[j] = 0;
      // two stages a turn: the parts of diagonal 0 are compile-time
#pragma unroll 1
      while (ok && left > 0) {
        ok = drain(std::integral_constant<int, 0>{}, --left);
        if (ok && left > 0) ok = drain(std::integral_constant<int, 1>{}, --left);
      }
      // the thread's place and its tile again: they would not fit the registers
      // beside the sums
      const int et = tid_again() - EPI_WARP0 * 32;
      const uint32_t t = blockIdx.x + it * gridDim.x;
      const int n_kb = my_stages(t, et);
      const bool extra = n_kb != 0 && !(n_kb & 1);   // the phase that makes them even
      if (ok && extra) ok = wait_phase_sleep(&go[h], 1, ctl);
      if (ok) ok = wait_phase_sleep(acc_full, it & 1, ctl);
      ok = ok && !ctl->abort;
      tc_fence_after();
      const int ew = et >> 5, lane = et & 31;
      if (ok && n_kb != 0) {
        // The last stages and the running sums as one int64 in units of 2^-20,
        // staged through shared memory (the operand stages are free by now): row r's
        // column c at word c ^ (r % 32), so that both walks spread over the banks.
        const int row = et & (TM - 1), part = (et >> 7) & 1;
        int64_t* st64 = (int64_t*)tiles + row * TN + (et >> 8) * HN + part * 32;
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
            st64[(pc * 4 + j) ^ lane] = ((long long)t0 << 23) + ((long long)t1 << 13) + l;
          }
        }
      }
      // the next tile's MMAs may start
      if (t + gridDim.x < args.tiles) {
        if (lane == 0 && extra) mbar_arrive(&drained[h]);
        zero();
      }
      ok = all_ok<EPI_WARPS * 32>(ok);
      if (ok) {
        const Tile x = tile_at(t);
        const int64_t* coff = (const int64_t*)(tabs + (it & 1) * C::TAB);
        const int64_t* roffs = coff + TN;
        const int32_t* cexp = (const int32_t*)(roffs + TM);
        const int32_t* rexps = cexp + TN;
        // a warp per row: lane l rounds and writes columns l, l + 32, ...; two rows
        // at a time (one was bound by the latency of its conversions)
        constexpr int NC = TN / 32;
        const int nrow = (int)min((int64_t)TM, p.M - x.m0), ncol = (int)min((int64_t)TN, p.N - x.n0);
        const long long* R0 = (const long long*)tiles;
        if (args.ksplit > 1) {
          unsigned long long* acc = args.wacc + ((int64_t)x.vb * p.M + x.m0) * p.N + x.n0 + lane;
#pragma unroll 1
          for (int r = ew; r < nrow; r += EPI_WARPS) {
#pragma unroll
            for (int j = 0; j < NC; ++j)
              if (lane + 32 * j < ncol)
                red_add_u64(acc + (int64_t)r * p.N + 32 * j, (unsigned long long)R0[r * TN + 32 * j + (lane ^ (r & 31))]);
          }
        } else {
          OutMode wp;
          wp.negate = args.neg[x.part];
          wp.accumulate = p.accumulate;
          int64_t co[NC];
          int ce[NC];
          int clo = INT32_MAX / 2, chi = INT32_MIN / 2;   // of the columns that are not all zero
#pragma unroll
          for (int j = 0; j < NC; ++j) {
            co[j] = coff[lane + 32 * j], ce[j] = cexp[lane + 32 * j] - 36;
            if (ce[j] > -kExpBias - 36) clo = min(clo, ce[j]), chi = max(chi, ce[j]);
          }
          // |R| <= 2^38 per column of K, and less than one more for what was dropped
          const bool small = args.kb_per_split * KSTAGE < 32768;
#pragma unroll 2
          for (int r = ew; r < nrow; r += EPI_WARPS) {
            const int64_t ro = roffs[r];
            const int re = rexps[r];
            long long R[NC];
            int ex[NC];
            double d[NC];
#pragma unroll
            for (int j = 0; j < NC; ++j) R[j] = R0[r * TN + 32 * j + (lane ^ (r & 31))], ex[j] = re + ce[j];
            // (an all-zero row's R are 0 whatever its exponent)
            const bool normal = re <= -kExpBias || (re + clo >= -1022 && re + chi <= 969);
            if (!(small && normal && i64_scaled_small<NC>(R, ex, d))) i64_scaled_batch<NC>(R, ex, d);
            if (ro < 0) continue;   // general plans: a row absent from W
#pragma unroll
            for (int j = 0; j < NC; ++j) {
              if (co[j] < 0) continue;   // beyond N, or a column absent from W
              if constexpr (!GEN) {
                args.w[ro + co[j]] = d[j];
              } else {
                store_w(wp, args.w + args.woff[x.part] + (int64_t)p.es * (ro + co[j]), d[j]);
              }
            }
          }
        }
      }
      if (!ok || t + gridDim.x >= args.tiles) break;
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // TMA writes there next
      __syncwarp();
      if (lane == 0) mbar_arrive(staged);
    }
  }
  // a split-K rounding kernel behind this one may start its launch now
  asm volatile("griddepcontrol.launch_dependents;");
  __syncthreads();
  if (ctl->abort) {
    land10<H>(full, issued, ctl);
    __syncthreads();
  }
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
  if (gx > 0x7FFFFFFF || gy > 65535 || gz > 65535 || gx * gy > 0x7FFFFFFFll / gz) return cudaErrorInvalidConfiguration;
  args.gx = (int)gx;
  args.gy = (int)gy;
  args.tiles = (uint32_t)(gx * gy * gz);
  // persistent CTAs, each walking the tiles one grid apart
  const int64_t resident = (int64_t)device_sms() * (3 - H);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(args.tiles < resident ? args.tiles : resident));
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
