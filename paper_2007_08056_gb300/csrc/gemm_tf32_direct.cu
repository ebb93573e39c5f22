// TF32 form for a long operand against a short one (at most 512 aligned rows),
// without the FP32 copy of the long one: its float64 entries are read from the
// reduced form once, rounded to TF32 on the way into shared memory, and
// multiplied by the whole short operand at once.
//
// The CC ladder (8192 x 512 x 8192 by 8 irreps) read 4.3 GB, wrote and read
// again 2.1 GB of FP32 (1.09 ms) and then ran its GEMM (0.75 ms): 1.85 ms.  Here
// the float64 entries cross HBM once: 1.27 ms in all (0.67 ms of copy bandwidth, 0.58
// of TF32 products; 512 tiles in four rounds of 152 SMs leave 16% of them idle).
// Measured on the way: 2.11 with float64 conversion instructions (narrow pipe),
// 1.70 with each stage's column offsets loaded in the loop, 1.34 without the
// 256-byte L2 fetches; sharing the short operand's copies between two CTAs of a
// cluster changed nothing (1.34), six stages of gathers in flight 1.38.
//
// CTA: 384 threads, a tile of 128 long rows by all short rows: one accumulator
// of up to 512 TMEM columns.  warp 0 copies the short operand's FP32 rows by
// TMA; warps 4-11 gather the long operand (16-byte loads, four stages in flight
// per thread), round it and store it in the swizzled K-major layout; warp 1
// issues the MMAs (M = 128, N up to 256 each, K = 8).  Five stages of 16 columns
// of K (64-byte rows, SWIZZLE_64B): the short operand's 32 KB a stage come from
// L2 and need more than two in flight.
// Every wait is bounded (see tc_common.cuh).
#include "tc_common.cuh"

namespace symctr {

namespace {

constexpr int TM = 128;
constexpr int NTHREADS = 384;
constexpr int W0 = 4;                 // first gathering (and epilogue) warp
constexpr int KST = 16;               // columns of K per stage
constexpr int ROWB = 4 * KST;         // bytes per tile row and stage
constexpr int A_BYTES = TM * ROWB;
constexpr int BH = 256;               // short rows per MMA and TMA copy
constexpr int B_BYTES = BH * ROWB;
constexpr int STAGES = 5;
constexpr int AHEAD = 4;              // stages of gathers in flight per thread
constexpr int CHUNK = 16;             // stages whose column offsets a warp fetches at once
constexpr int PASS = 128;             // columns of an epilogue pass
constexpr int LD = PASS + 1;

template <int NB>
struct Cfg {
  static constexpr int STAGE_BYTES = A_BYTES + NB * B_BYTES;
  static constexpr size_t REGION = (size_t)STAGES * STAGE_BYTES;
  static_assert(REGION >= (size_t)TM * LD * 4, "the epilogue staging fits the stages");
  static constexpr size_t SMEM = 1024 + REGION + 8 * (3 * STAGES + 1) + 8 * (TM + NB * BH) +
                                 8 * 8 * 2 * CHUNK * (KST / 2) + 16 + 64;
};

struct DirectArgs {
  Problem p;
  int n_kb;
  int64_t rows, short_rows;    // aligned rows of the long and of the short operand
  const double* src;           // long operand's reduced form
  const int64_t* rtab;         // [n_q][rows] its row offsets
  const int64_t* ctab;         // [n_q][K] its column offsets
  const int64_t* wl;           // [n_q][rows] W offsets along the long side
  const int64_t* ws;           // [n_q][short_rows] W offsets along the short side
  bool long_is_u;
  double* w;
  unsigned* err;
};

// Nearest TF32 value (ties to even) of a float64, through FP32: the general case.
__device__ __noinline__ uint32_t tf32_bits_rare(double x) {
  uint32_t u = __float_as_uint(__double2float_rn(x));
  if ((u & 0x7F800000u) != 0x7F800000u) u = (u + 0xFFFu + ((u >> 13) & 1u)) & ~0x1FFFu;
  return u;
}

// The same with integer operations for zeros and values normal in FP32 before
// and after rounding (`rare` is set for others): float64 conversions run on
// GB300's narrow float64 pipe.  The high word holds 20 mantissa bits, 10 are
// kept; a nonzero low word only breaks ties.
__device__ __forceinline__ uint32_t tf32_bits(double x, bool& rare) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const uint32_t m = (hi & 0x7FFFFFFFu) | min(lo, 1u);
  const uint32_t r = m + 0x1FFu + ((hi >> 10) & 1u) - (896u << 20);
  const uint32_t u = (hi & 0x80000000u) | ((r << 3) & 0x7FFFE000u);
  // exponents 897 .. 1149 (rounding up stays finite)
  const bool normal = m - (897u << 20) < (253u << 20);
  rare = !normal && m != 0u;
  return normal ? u : (hi & 0x80000000u);
}

// Two entries of a row, 256 bytes of it into L2: the next stage's 128 bytes come
// with them, and DRAM is read in longer pieces of the tile's 128 rows.
__device__ __forceinline__ double2 ld_pair(const double* a) {
  double2 d;
  asm("ld.global.L2::256B.v2.f64 {%0, %1}, [%2];" : "=d"(d.x), "=d"(d.y) : "l"(a));
  return d;
}

__device__ __forceinline__ uint64_t sdesc64(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)((8 * ROWB) >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)4 << 61;
  return d;
}

__device__ __forceinline__ void mma_tf32(uint32_t tacc, uint64_t da, uint64_t db, uint32_t id, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tacc),
      "l"(da), "l"(db), "r"(id), "r"(acc)
      : "memory");
}

template <int NB>
__global__ void __launch_bounds__(NTHREADS, 1)
    gemm_tf32_direct_kernel(const __grid_constant__ CUtensorMap tma_b, const __grid_constant__ DirectArgs args) {
  using C = Cfg<NB>;
  constexpr int STAGE_BYTES = C::STAGE_BYTES;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const Problem& p = args.p;
  uint64_t* a_full = (uint64_t*)(smem + C::REGION);
  uint64_t* b_full = a_full + STAGES;
  uint64_t* empty = b_full + STAGES;
  uint64_t* acc_full = empty + STAGES;
  int64_t* loff = (int64_t*)(acc_full + 1);   // [TM] W offsets of the tile's long rows
  int64_t* soff = loff + TM;                  // [NB * BH] W offsets of the short rows
  int64_t* coffs = soff + NB * BH;            // [8 warps][2][CHUNK * 8] column offsets of pairs
  uint32_t* tmem_slot = (uint32_t*)(coffs + 8 * 2 * CHUNK * (KST / 2));
  Ctl* ctl = (Ctl*)(tmem_slot + 4);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t r0 = (int64_t)blockIdx.x * TM;
  const int b = blockIdx.y;
  const int n_kb = args.n_kb;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&a_full[s], 8);
      mbar_init(&b_full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(acc_full, 1);
    ctl->abort = 0;
    ctl->err = args.err;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tmem_slot)),
                 "n"(NB * BH)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  for (int i = threadIdx.x; i < TM; i += NTHREADS)
    loff[i] = r0 + i < args.rows ? args.wl[(int64_t)b * args.rows + r0 + i] : -1;
  for (int i = threadIdx.x; i < NB * BH; i += NTHREADS)
    soff[i] = i < args.short_rows ? args.ws[(int64_t)b * args.short_rows + i] : -1;
  // programmatic dependent of the short operand's preparation
  asm volatile("griddepcontrol.wait;" ::: "memory");
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0) {
    // ------------------------------------------------------------ short operand
    if (lane == 0) {
      int issued = 0;
      for (int kb = 0; kb < n_kb; ++kb) {
        const int st = kb % STAGES;
        if (!wait_phase(&empty[st], ((kb / STAGES) & 1) ^ 1, ctl)) break;
        mbar_expect_tx(&b_full[st], NB * B_BYTES);
        uint8_t* sb = smem + (size_t)st * STAGE_BYTES + A_BYTES;
        for (int i = 0; i < NB; ++i) tma_load_4d(&tma_b, &b_full[st], sb + i * B_BYTES, kb * KST, i * BH, b);
        ++issued;
      }
      ctl->copies = (uint32_t)issued;
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    if (lane == 0) {
      const uint32_t base = su32(smem);
      // N of each MMA: the short rows, rounded to 16
      uint32_t id[NB];
      for (int i = 0; i < NB; ++i) {
        int n = (int)(args.short_rows - (int64_t)i * BH);
        n = n > BH ? BH : (n + 15) / 16 * 16;
        id[i] = (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(TM >> 4) << 24);
      }
      bool ok = true;
      for (int kb = 0; ok && kb < n_kb; ++kb) {
        const int st = kb % STAGES;
        ok = wait_phase(&b_full[st], (kb / STAGES) & 1, ctl) && wait_phase(&a_full[st], (kb / STAGES) & 1, ctl);
        if (!ok) break;
        tc_fence_after();
        const uint64_t da = sdesc64(base + st * STAGE_BYTES), db = sdesc64(base + st * STAGE_BYTES + A_BYTES);
#pragma unroll
        for (int kk = 0; kk < ROWB / 32; ++kk)
#pragma unroll
          for (int i = 0; i < NB; ++i)
            mma_tf32(tmem + i * BH, da + ((kk * 32) >> 4), db + ((i * B_BYTES + kk * 32) >> 4), id[i],
                     kb > 0 || kk > 0 ? 1u : 0u);
        tc_commit(&empty[st]);
      }
      tc_commit(acc_full);
      wait_phase(acc_full, 0, ctl, kTimeoutCycles / 2);
    }
  } else if (warp >= W0) {
    // ------------------------------------------------------------ long operand
    const int cw = warp - W0;
    // load i of a stage: 8 lanes per row (16 columns), 4 rows of the warp's 16
    const int pr = lane & 7, sub = lane >> 3;
    const double* rowp[4];
    uint32_t dst[4];
    bool rok[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = cw * 16 + i * 4 + sub;
      rok[i] = r0 + r < args.rows;
      rowp[i] = args.src + (rok[i] ? args.rtab[(int64_t)b * args.rows + r0 + r] : 0);
      dst[i] = (uint32_t)(r * ROWB + (((pr >> 1) ^ ((r >> 1) & 3)) << 4) + (pr & 1) * 8);
    }
    // Column offsets of the pairs of CHUNK stages, fetched a chunk ahead into this
    // warp's own ring: an offset loaded stage by stage would wait, in its shared
    // scoreboard, for the gathers queued behind it (one stage in flight, 2.7 TB/s).
    constexpr int PAIRS = CHUNK * (KST / 2);
    const int64_t* ctab = args.ctab + (int64_t)b * p.K;
    int64_t* ring = coffs + cw * 2 * PAIRS;
    int64_t fetched[PAIRS / 32];
    auto fetch = [&](int chunk) {
#pragma unroll
      for (int i = 0; i < PAIRS / 32; ++i) {
        const int64_t c = (int64_t)chunk * CHUNK * KST + 2 * (i * 32 + lane);
        fetched[i] = c < p.K ? ctab[c] : -1;
      }
    };
    auto publish = [&](int chunk) {
#pragma unroll
      for (int i = 0; i < PAIRS / 32; ++i) ring[(chunk & 1) * PAIRS + i * 32 + lane] = fetched[i];
      __syncwarp();
    };
    auto col = [&](int kb) { return ring[(kb / CHUNK & 1) * PAIRS + (kb % CHUNK) * (KST / 2) + pr]; };
    double2 x[AHEAD][4];
    auto gather = [&](double2 (&d)[4], int64_t co) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        d[i] = co >= 0 && rok[i] ? ld_pair(rowp[i] + co) : make_double2(0.0, 0.0);
    };
    fetch(0);
    publish(0);
    fetch(1);
#pragma unroll
    for (int j = 0; j < AHEAD; ++j) gather(x[j], col(j));
    bool ok = true;
    for (int kb0 = 0; ok && kb0 < n_kb; kb0 += AHEAD) {
#pragma unroll
      for (int j = 0; j < AHEAD; ++j) {
        const int kb = kb0 + j;
        if (!ok || kb >= n_kb) break;
        const int st = kb % STAGES;
        ok = wait_phase(&empty[st], ((kb / STAGES) & 1) ^ 1, ctl);
        if (!ok) break;
        uint8_t* sa = smem + (size_t)st * STAGE_BYTES;
        uint2 f[4];
        bool any = false;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          bool r0, r1;
          f[i] = make_uint2(tf32_bits(x[j][i].x, r0), tf32_bits(x[j][i].y, r1));
          any = any || r0 || r1;
        }
        if (any) {
#pragma unroll
          for (int i = 0; i < 4; ++i) f[i] = make_uint2(tf32_bits_rare(x[j][i].x), tf32_bits_rare(x[j][i].y));
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) *reinterpret_cast<uint2*>(sa + dst[i]) = f[i];
        if ((kb + AHEAD) % CHUNK == 0) {
          publish((kb + AHEAD) / CHUNK);
          fetch((kb + AHEAD) / CHUNK + 1);
        }
        gather(x[j], col(kb + AHEAD));
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(&a_full[st]);
      }
    }
    // ------------------------------------------------------------ epilogue
    if (ok) ok = wait_phase_sleep(acc_full, 0, ctl);
    ok = ok && !ctl->abort;
    tc_fence_after();
    const int quad = warp & 3, part = cw >> 2, row = quad * 32 + lane, t = threadIdx.x - W0 * 32;
    const uint32_t lane_base = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(part * (PASS / 2));
    uint32_t* stage = (uint32_t*)smem;   // [TM][LD]
    const int n_pass = (int)((args.short_rows + PASS - 1) / PASS);
    for (int ps = 0; ps < n_pass; ++ps) {
      if (ok) {
#pragma unroll
        for (int pc = 0; pc < PASS / 32; ++pc) {
          uint32_t a[16];
          tmem_ld16(lane_base + ps * PASS + pc * 16, a);
          tmem_wait_ld();
          tmem_loaded<16>(a);
#pragma unroll
          for (int j = 0; j < 16; ++j) stage[row * LD + part * (PASS / 2) + pc * 16 + j] = a[j];
        }
      }
      asm volatile("bar.sync 1, 256;" ::: "memory");
      if (ok) {
        // lanes along W's columns: the tile's columns, or (long operand V) its rows
        const int fix = t % 128;   // column of the pass, or row of the tile
        const int64_t fo = args.long_is_u ? soff[ps * PASS + fix] : loff[fix];
        if (fo >= 0) {
          constexpr int BATCH = 8;
#pragma unroll 1
          for (int o = t / 128; o < 128; o += 2 * BATCH) {
            uint32_t a[BATCH];
            int64_t oo[BATCH];
            double d[BATCH];
#pragma unroll
            for (int j = 0; j < BATCH; ++j) {
              const int q = o + 2 * j;
              a[j] = args.long_is_u ? stage[q * LD + fix] : stage[fix * LD + q];
              oo[j] = args.long_is_u ? loff[q] : soff[ps * PASS + q];
            }
            f32_to_f64_batch<BATCH>(a, d);
#pragma unroll
            for (int j = 0; j < BATCH; ++j)
              if (oo[j] >= 0) args.w[fo + oo[j]] = d[j];
          }
        }
      }
      asm volatile("bar.sync 1, 256;" ::: "memory");
    }
    tc_fence_before();
  }
  __syncthreads();
  if (ctl->abort) {
    land(b_full, STAGES, acc_full, ctl);
    __syncthreads();
  }
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(NB * BH) : "memory");
  }
}

template <int NB>
cudaError_t launch_nb(const CUtensorMap& mb, const DirectArgs& args, cudaStream_t st) {
  auto kern = gemm_tf32_direct_kernel<NB>;
  constexpr size_t smem = Cfg<NB>::SMEM;
  thread_local bool attr_set[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) dev = 0;
  if (!attr_set[dev]) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    attr_set[dev] = true;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((args.rows + TM - 1) / TM), (unsigned)args.p.n_q, 1);
  cfg.blockDim = dim3(NTHREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaError_t e = cudaLaunchKernelEx(&cfg, kern, mb, args);
  ++g_kernel_launches;
  return e;
}

}  // namespace

cudaError_t launch_gemm_tf32_direct(const Problem& p, const Tables& tab, int op, const double* src, const float* other,
                                    int64_t kpad, double* w, unsigned* err, cudaStream_t st) {
  DirectArgs a;
  a.p = p;
  a.n_kb = (int)((p.K + KST - 1) / KST);
  a.rows = op == 0 ? p.M : p.N;
  a.short_rows = op == 0 ? p.N : p.M;
  a.src = src;
  a.rtab = op == 0 ? tab.urow : tab.vrow;
  a.ctab = op == 0 ? tab.ucol : tab.vcol;
  a.wl = op == 0 ? tab.wrow : tab.wcol;
  a.ws = op == 0 ? tab.wcol : tab.wrow;
  a.long_is_u = op == 0;
  a.w = w;
  a.err = err;
  if (a.short_rows > kTf32DirectShort || p.n_q > 65535) return cudaErrorInvalidValue;
  CUtensorMap mb;
  if (!make_map(&mb, other, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, kpad, a.short_rows, p.n_q, 1, KST, BH, 1))
    return cudaErrorInvalidValue;
  return a.short_rows > BH ? launch_nb<2>(mb, a, st) : launch_nb<1>(mb, a, st);
}

}  // namespace symctr
