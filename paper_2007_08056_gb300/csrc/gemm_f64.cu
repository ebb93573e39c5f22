// Float64 form of the aligned contraction (Alg. 2, contraction step):
//   W_hat[Q, m, n] = sum_kappa U_hat[Q, m, kappa] V_hat[Q, n, kappa]
// with the input transformations fused into the operand loads (each tile
// element is gathered from the standard reduced form through the separable
// index maps) and the output step fused into the epilogue (each result is
// written straight to W's standard reduced form).  GB300 has very little
// float64 throughput, so the aligned operands are never materialised: the
// loads are free next to the FMAs.
//
// Three kernels: a 64x64 register-tiled kernel for GEMM-shaped problems, a
// warp-per-row dot-product kernel for skinny ones (a few rows or columns),
// both with optional split-K through atomicAdd into a zeroed output (or onto
// the existing output in accumulate mode), and a thread-per-row kernel for
// skinny problems with a short contracted extent (the adjoints of a GEMV:
// an outer product, K = 1, or K = 2), where lanes walking K would idle.
#include <cstdint>

#include "symctr_internal.h"

namespace symctr {

namespace {

constexpr int BK = 16, THREADS = 256;

// axis_offset as one out-of-line device function: every kernel below computes
// offsets in a dozen places (per instance of the short-side row count), and
// inlining the mixed-radix arithmetic at each of them multiplied the code size
// and the compile time without changing the speed (none of these calls sits in
// an innermost loop).
__device__ __noinline__ int64_t aoff(const AxisMap& a, const GroupDesc& g, int Q, int64_t r) {
  return axis_offset(a, g, Q, r);
}

__host__ __device__ inline bool map_rows_fast(const AxisMap& rows) {
  return rows.n > 0 && rows.bstride[rows.n - 1] == 1;
}

// GEMM-shaped problems, a T x T output tile by 256 threads: (T / 16)^2 outputs a
// thread, or (T = 8) one output by four threads that split each K block.  The
// float64 pipe (2 FMAs per SM and clock) is the bound at every T: what matters
// is that all SMs have the same share, and that a small problem has tiles for
// all of them (tile_choice): 48 x 48 x 48 by 3 irreps ran on three SMs with
// 64 x 64 tiles, 65 -> 17 us (launch-bound) with 8 x 8; the two MPS contractions
// 128 x 2048 x 128 and 128 x 128 x 2048 by 8 irreps, on 3.4 such tiles per SM and
// on 128 of 152 SMs, 1177 -> 922 us with 16 x 16 (866 us at the float64 rate of the
// CC ladder, 443 ms, 0.99 of the pipe; 471 ms before).  Column offsets are computed for kKc columns of K at a time,
// one per thread; the next K block's gathers are in flight while this one is
// multiplied.  One CTA to a tile and range: a grid of four CTAs per SM walking
// them left SMs with one more or less than their share (640 x 640 x 2000 by 2
// irreps in 16 x 16 tiles 3316 us, 2781 without the walk).
// The K ranges of a tile are the CTAs of a cluster: each leaves its partial sums in
// shared memory, and every CTA adds up a share of the tile over the ranks, in their
// order, and writes it, so that a product repeats bit for bit.  (Float64 atomics
// onto a zeroed W, 475 us for the second MPS contraction against 473, gave
// results of three and more ranges that differed from run to run.)
// General plans pass their offset tables (t.urow != NULL): offsets come from
// them, -1 marking an absent aligned row or column (read as zero, not stored).
constexpr int kKc = 256;
constexpr int kMaxRanges = 16;    // CTAs of a cluster

__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// The float64 word of cluster CTA `rank` at this CTA's shared address of it.
__device__ __forceinline__ double cluster_ld(const double* p, int rank) {
  double x;
  asm volatile(
      "{\n\t.reg .b32 ra;\n\tmapa.shared::cluster.u32 ra, %1, %2;\n\t"
      "ld.shared::cluster.f64 %0, [ra];\n\t}\n"
      : "=d"(x)
      : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank)
      : "memory");
  return x;
}

template <int T>
__global__ void __launch_bounds__(THREADS, T == 64 ? 2 : T == 32 ? 3 : 4)
    gemm_f64_tiled(const __grid_constant__ Problem p, int ksplit, int64_t kchunk, bool u_rows_fast, bool v_rows_fast,
                   const Tables t, const double* __restrict__ U, const double* __restrict__ V, double* __restrict__ W) {
  constexpr int R = T >= 16 ? T / 16 : 1;                      // outputs per thread and side
  constexpr int NL = (T * BK + THREADS - 1) / THREADS;         // gathers per thread, operand and K block
  __shared__ double ops[2][2][BK][T + 1];
  double (*As)[BK][T + 1] = ops[0];
  double (*Bs)[BK][T + 1] = ops[1];
  __shared__ int64_t uoff[T], voff[T], woffr[T], woffc[T], ku[kKc], kv[kKc];
  const int tid = threadIdx.x;
  const int tr = T >= 16 ? tid / 16 : (tid & 63) / 8, tc = T >= 16 ? tid % 16 : tid % 8;
  const int64_t mt = (p.M + T - 1) / T, nt = (p.N + T - 1) / T;
  const bool tab = t.urow != nullptr;
  const int ks = (int)(blockIdx.x % (unsigned)ksplit);   // K range, rank in the cluster
  const int64_t t2 = blockIdx.x / (unsigned)ksplit;
  const int64_t b = t2 / (mt * nt);
  const int64_t rem = t2 - b * mt * nt;
  const int64_t m0 = (rem / nt) * T, n0 = (rem % nt) * T;
  const int Q = batch_irrep(p, (int)b);
  const int64_t kbeg = ks * kchunk, kend = kbeg + kchunk < p.K ? kbeg + kchunk : p.K;
  if (tid < T) {
    const int64_t m = m0 + tid;
    uoff[tid] = m >= p.M ? -1 : tab ? t.urow[b * p.M + m] : aoff(p.u.rows, p.g, Q, m);
    woffr[tid] = m >= p.M ? -1 : tab ? t.wrow[b * p.M + m] : aoff(p.w.rows, p.g, Q, m);
  } else if (tid >= 128 && tid < 128 + T) {
    const int64_t n = n0 + tid - 128;
    voff[tid - 128] = n >= p.N ? -1 : tab ? t.vrow[b * p.N + n] : aoff(p.v.rows, p.g, Q, n);
    woffc[tid - 128] = n >= p.N ? -1 : tab ? t.wcol[b * p.N + n] : aoff(p.w.cols, p.g, Q, n);
  }
  // the sum of each kKc columns, and their sum: shorter chains of roundings
  double acc[R][R], sum[R][R];
#pragma unroll
  for (int i = 0; i < R; ++i)
#pragma unroll
    for (int j = 0; j < R; ++j) sum[i][j] = 0.0;
  for (int64_t kc = kbeg; kc < kend; kc += kKc) {
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
      for (int j = 0; j < R; ++j) acc[i][j] = 0.0;
    const int n = kend - kc < kKc ? (int)(kend - kc) : kKc;
    __syncthreads();
    if (tid < n) {
      const int64_t k = kc + tid;
      ku[tid] = tab ? t.ucol[b * p.K + k] : aoff(p.u.cols, p.g, Q, k);
      kv[tid] = tab ? t.vcol[b * p.K + k] : aoff(p.v.cols, p.g, Q, k);
    }
    __syncthreads();
    double xa[NL], xb[NL];
    auto gather = [&](int k0) {
#pragma unroll
      for (int j = 0; j < NL; ++j) {
        const int e = tid + j * THREADS;
        xa[j] = xb[j] = 0.0;
        if (e < T * BK) {
          int mm = u_rows_fast ? e % T : e / BK, kk = k0 + (u_rows_fast ? e / T : e % BK);
          if (kk < n && uoff[mm] >= 0 && ku[kk] >= 0) xa[j] = U[p.es * (uoff[mm] + ku[kk])];
          mm = v_rows_fast ? e % T : e / BK, kk = k0 + (v_rows_fast ? e / T : e % BK);
          if (kk < n && voff[mm] >= 0 && kv[kk] >= 0) xb[j] = V[p.es * (voff[mm] + kv[kk])];
        }
      }
    };
    auto stage = [&](int buf) {
#pragma unroll
      for (int j = 0; j < NL; ++j) {
        const int e = tid + j * THREADS;
        if (e < T * BK) {
          As[buf][u_rows_fast ? e / T : e % BK][u_rows_fast ? e % T : e / BK] = xa[j];
          Bs[buf][v_rows_fast ? e / T : e % BK][v_rows_fast ? e % T : e / BK] = xb[j];
        }
      }
    };
    gather(0);
    stage(0);
    __syncthreads();
    for (int k0 = 0, buf = 0; k0 < n; k0 += BK, buf ^= 1) {
      if (k0 + BK < n) gather(k0 + BK);
      if constexpr (T >= 16) {
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
          double a[R], bb[R];
#pragma unroll
          for (int i = 0; i < R; ++i) a[i] = As[buf][kk][tr + 16 * i];
#pragma unroll
          for (int j = 0; j < R; ++j) bb[j] = Bs[buf][kk][tc + 16 * j];
#pragma unroll
          for (int i = 0; i < R; ++i)
#pragma unroll
            for (int j = 0; j < R; ++j) acc[i][j] = fma(a[i], bb[j], acc[i][j]);
        }
      } else {
#pragma unroll
        for (int q = 0; q < BK / 4; ++q) {
          const int kk = (tid >> 6) * (BK / 4) + q;
          acc[0][0] = fma(As[buf][kk][tr], Bs[buf][kk][tc], acc[0][0]);
        }
      }
      if (k0 + BK < n) stage(buf ^ 1);
      __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
      for (int j = 0; j < R; ++j) sum[i][j] += acc[i][j];
  }
  double* part = &ops[0][0][0][0];   // [T][T] partial sums, in place of the operands
  if constexpr (T < 16) {
    double* red = part;
    part += THREADS;
    red[tid] = sum[0][0];
    __syncthreads();
    if (tid < 64) sum[0][0] = (red[tid] + red[tid + 64]) + (red[tid + 128] + red[tid + 192]);
  }
  static_assert(sizeof(ops) >= (T * T + (T < 16 ? THREADS : 0)) * sizeof(double), "partial sums");
  if (ksplit > 1) {
    if (T >= 16 || tid < 64) {
#pragma unroll
      for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < R; ++j) part[(tr + 16 * i) * T + tc + 16 * j] = sum[i][j];
    }
    cluster_sync_all();
    for (int e = ks * THREADS + tid; e < T * T; e += ksplit * THREADS) {
      const int64_t ro = woffr[e / T], co = woffc[e % T];
      if (ro < 0 || co < 0) continue;
      double x = 0.0;
      for (int r0 = 0; r0 < ksplit; r0 += 4) {
        double y[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) y[r] = r0 + r < ksplit ? cluster_ld(part + e, r0 + r) : 0.0;
        x += y[0];
        x += y[1];
        x += y[2];
        x += y[3];
      }
      store_w(p, W + p.es * (ro + co), x);
    }
    cluster_sync_all();   // the others have read this CTA's sums
    return;
  }
  if (T < 16 && tid >= 64) return;
#pragma unroll
  for (int i = 0; i < R; ++i) {
    const int mm = tr + 16 * i;
    if (woffr[mm] < 0) continue;
#pragma unroll
    for (int j = 0; j < R; ++j) {
      const int nn = tc + 16 * j;
      if (woffc[nn] < 0) continue;
      store_w(p, W + p.es * (woffr[mm] + woffc[nn]), sum[i][j]);
    }
  }
}

// Skinny problems: the "long" side L (rows of U or of V, whichever is larger)
// is spread over warps, the "short" side (<= 8 rows) is held in registers;
// lanes stride over kappa.  Optional split-K over kappa ranges.
//
// Column offsets: kappa = o * I + i, where I (the "inner" extent) is the
// product of the fastest block dims of the column map up to kInnerMax.  The
// offset is then aoff(o * I) + inner(i), inner(i) being the block part
// of i alone (independent of Q); each block tabulates inner() in shared
// memory, and a warp computes the offsets aoff(o * I) of the inner blocks of
// its K range 16 at a time, one per lane, instead of one mixed-radix
// decomposition per element.
constexpr int SKINNY_MAX = 8;
constexpr int kInnerMax = 2048;

// Product of the fastest block dims that the two column maps share, up to
// kInnerMax (both maps index the same kappa, so their dims agree).
__device__ __forceinline__ int64_t inner_extent(const AxisMap& a, const AxisMap& b) {
  int64_t e = 1;
  for (int i = a.n - 1, j = b.n - 1; i >= 0 && j >= 0; --i, --j) {
    if (a.D[i] != b.D[j] || e * a.D[i] > kInnerMax) break;
    e *= a.D[i];
  }
  return e;
}

// A 64-bit integer division is a long emulated instruction sequence:
// quotients of values below 2^32 are taken in 32 bits.
__device__ __forceinline__ int64_t div_idx(int64_t a, int64_t b) {
  if (((uint64_t)a | (uint64_t)b) <= 0xFFFFFFFFull) return (int64_t)((uint32_t)a / (uint32_t)b);
  return a / b;
}

// scale * inner(i) for i < I: the block digits of i over the fastest block
// axes (scale: the element stride, so that the table holds array indices).
// I <= kInnerMax, so the digits are taken in 32 bits.
__device__ void fill_inner(const AxisMap& a, int64_t I, int64_t scale, int64_t* tab) {
  for (int i = threadIdx.x; i < (int)I; i += blockDim.x) {
    uint32_t r = (uint32_t)i;
    int64_t off = 0;
    for (int d = a.n - 1; d >= 0 && r > 0; --d) {
      const uint32_t D = (uint32_t)a.D[d], q = r / D;
      off += (int64_t)(r - q * D) * a.bstride[d];
      r = q;
    }
    tab[i] = off * scale;
  }
}

// Elements per lane whose loads (one of L, NS of S) are all issued before
// their FMAs: fewer for more short-side rows, so that the registers they
// take stay about the same.
template <int NS>
struct SkinnyUnroll {
  static constexpr int value = NS <= 2 ? 4 : 2;
};

// NS = the short side's row count (one instance per count, so that no
// float64 instruction of an absent row is issued: GB300's float64 pipe is
// narrow and issues predicated-off instructions all the same).
//
// Work items: (irrep, long-side row, K range), the K ranges whole inner
// blocks; the launcher sizes ksplit so that the items about fill the
// resident warps once, which pays the offset arithmetic of an item (a
// dependent chain of modular arithmetic under a product group) once per warp.
template <int NS>
__global__ void __launch_bounds__(THREADS, 3)
    gemm_f64_skinny(const __grid_constant__ Problem p, bool long_is_u, int ksplit, const double* __restrict__ U,
                    const double* __restrict__ V, double* __restrict__ W) {
  __shared__ int64_t tab_l[kInnerMax], tab_s[kInnerMax];
  const AxisMap& Lrows = long_is_u ? p.u.rows : p.v.rows;
  const AxisMap& Lcols = long_is_u ? p.u.cols : p.v.cols;
  const AxisMap& Srows = long_is_u ? p.v.rows : p.u.rows;
  const AxisMap& Scols = long_is_u ? p.v.cols : p.u.cols;
  // W's axis along the long side and along the short side
  const AxisMap& Wl = long_is_u ? p.w.rows : p.w.cols;
  const AxisMap& Ws = long_is_u ? p.w.cols : p.w.rows;
  const double* Lp = long_is_u ? U : V;
  const double* Sp = long_is_u ? V : U;
  const int64_t nL = long_is_u ? p.M : p.N;
  const int64_t es = p.es;
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int64_t I = inner_extent(Lcols, Scols);
  fill_inner(Lcols, I, es, tab_l);
  fill_inner(Scols, I, es, tab_s);
  __syncthreads();
  // K ranges of whole inner blocks (K is a multiple of I)
  const int64_t nb = div_idx(p.K, I);
  const int64_t per = div_idx(nb + ksplit - 1, ksplit);
  const int64_t parts = div_idx(nb + per - 1, per);
  const int64_t items = nL * p.n_q * parts;
  for (int64_t it = warp; it < items; it += nwarps) {
    const int64_t t2 = div_idx(it, parts);
    const int64_t ks = it - t2 * parts;
    const int64_t b = div_idx(t2, nL);
    const int64_t l = t2 - b * nL;
    const int Q = batch_irrep(p, (int)b);
    // the row offsets, one per lane: lane 0 L's row, lanes 1..NS the short
    // rows in S, lane NS+1 the long row along W, lanes NS+2..2NS+1 the short
    // rows along W (the other lanes repeat lane 0's)
    const AxisMap* rm = &Lrows;
    int64_t rr = l;
    if (lane >= 1 && lane <= NS) {
      rm = &Srows;
      rr = lane - 1;
    } else if (lane == NS + 1) {
      rm = &Wl;
    } else if (lane >= NS + 2 && lane <= 2 * NS + 1) {
      rm = &Ws;
      rr = lane - NS - 2;
    }
    const int64_t ro = aoff(*rm, p.g, Q, rr);
    const int64_t loff = es * __shfl_sync(0xffffffffu, ro, 0);
    int64_t soff[NS];
#pragma unroll
    for (int s = 0; s < NS; ++s) soff[s] = es * __shfl_sync(0xffffffffu, ro, 1 + s);
    double acc[NS];
#pragma unroll
    for (int s = 0; s < NS; ++s) acc[s] = 0.0;
    const int64_t ob0 = ks * per, ob1 = ob0 + per < nb ? ob0 + per : nb;
    if (I >= 32) {
      // inner blocks 16 at a time: lanes 0-15 compute the L offsets of blocks
      // g0 + lane, lanes 16-31 the S offsets of blocks g0 + lane - 16
      for (int64_t g0 = ob0; g0 < ob1; g0 += 16) {
        const int64_t ob = g0 + (lane & 15);
        const int64_t co = ob < ob1 ? aoff(lane < 16 ? Lcols : Scols, p.g, Q, ob * I) : 0;
        const int nbk = ob1 - g0 < 16 ? (int)(ob1 - g0) : 16;
        for (int j = 0; j < nbk; ++j) {
          const double* Lb = Lp + (loff + es * __shfl_sync(0xffffffffu, co, j));
          const int64_t sb = es * __shfl_sync(0xffffffffu, co, 16 + j);
          const double* Sb[NS];
#pragma unroll
          for (int s = 0; s < NS; ++s) Sb[s] = Sp + (soff[s] + sb);
          constexpr int kU = SkinnyUnroll<NS>::value;
          for (int i0 = 0; i0 < (int)I; i0 += 32 * kU) {
            if (i0 + 32 * kU <= (int)I) {
              double x[kU], y[NS][kU];
#pragma unroll
              for (int u = 0; u < kU; ++u) {
                const int i = i0 + 32 * u + lane;
                const int64_t tl = tab_l[i], ts = tab_s[i];
                x[u] = Lb[tl];
#pragma unroll
                for (int s = 0; s < NS; ++s) y[s][u] = Sb[s][ts];
              }
#pragma unroll
              for (int u = 0; u < kU; ++u) {
#pragma unroll
                for (int s = 0; s < NS; ++s) acc[s] = fma(x[u], y[s][u], acc[s]);
              }
            } else {
              // the ragged end of an inner block (I not a multiple of 32 kU)
              for (int i = i0 + lane; i < (int)I; i += 32) {
                const double x = Lb[tab_l[i]];
#pragma unroll
                for (int s = 0; s < NS; ++s) acc[s] = fma(x, Sb[s][tab_s[i]], acc[s]);
              }
            }
          }
        }
      }
    } else {
      // short inner blocks: lanes walk the elements, recomputing the two
      // inner-block offsets when the block changes
      const int64_t kend = ob1 * I;
      int64_t k = ob0 * I + lane;
      int64_t o = div_idx(k, I), i = k - o * I;
      int64_t lo = es * aoff(Lcols, p.g, Q, o * I), so = es * aoff(Scols, p.g, Q, o * I);
      for (; k < kend; k += 32) {
        const double x = Lp[loff + lo + tab_l[i]];
        const int64_t sc = so + tab_s[i];
#pragma unroll
        for (int s = 0; s < NS; ++s) acc[s] = fma(x, Sp[soff[s] + sc], acc[s]);
        i += 32;
        if (i >= I) {
          o += i / I;
          i %= I;
          if (k + 32 < kend) {
            lo = es * aoff(Lcols, p.g, Q, o * I);
            so = es * aoff(Scols, p.g, Q, o * I);
          }
        }
      }
    }
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      double a = acc[s];
      for (int o2 = 16; o2 > 0; o2 >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o2);
      acc[s] = a;
    }
    const int64_t wlo = __shfl_sync(0xffffffffu, ro, NS + 1);
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      const int64_t wso = __shfl_sync(0xffffffffu, ro, NS + 2 + s);
      if (lane == 0) {
        double* dst = W + es * (wlo + wso);
        if (ksplit > 1) atomicAdd(dst, signed_result(p, acc[s]));
        else store_w(p, dst, acc[s]);
      }
    }
  }
}

// Skinny problems with K <= kShortK: one thread per row of the long side, on
// a persistent grid whose blocks take kShortRows consecutive rows (a chunk)
// at a time.  The short side's values and the long side's column offsets
// depend only on the irrep, so a block stages them in shared memory when the
// irrep changes.  Row offsets in
// L and W use the inner-block split of the skinny kernel above (l = o * I +
// i): a table of inner(i) per map, and aoff(o * I) for the inner blocks of a
// chunk computed by as many threads at once, spread over the warps (the
// index arithmetic of one offset is a long dependent chain under a product
// group, so it is never left to a single thread).  A thread issues the loads
// of a few rows (ShortUnroll) before their FMAs.
constexpr int kShortK = 32;
constexpr int kShortRows = 4096;
constexpr int kShortSlots = kShortRows / 32 + 2;

// Rows per thread whose loads are all issued before their FMAs.
template <int KT>
struct ShortUnroll {
  static constexpr int value = KT == 1 ? 8 : (KT == 2 ? 4 : 2);
};

// Step (o, i) = divmod(l, I) by THREADS rows without dividing.
__device__ __forceinline__ void step_rows(int I, int& o, int& i) {
  i += THREADS;
  while (i >= I) {
    i -= I;
    ++o;
  }
}

// A W entry of the short-K kernel, whose staged short-side values carry the
// problem's sign (exact: x * (-s) = -(x * s)).  Accumulation is a float64
// atomic add (a single writer per entry: the same rounded sum).
__device__ __forceinline__ void put_w(int accumulate, double* dst, double x) {
  if (accumulate)
    atomicAdd(dst, x);
  else
    *dst = x;
}

// KT: K itself when it is 1 or 2 (the loads of a row unrolled), 0 for any
// K <= kShortK (a loop over K).
template <int NS, int KT>
__global__ void __launch_bounds__(THREADS, 4)
    gemm_f64_shortk(const __grid_constant__ Problem p, bool long_is_u, const double* __restrict__ U,
                    const double* __restrict__ V, double* __restrict__ W) {
  __shared__ double sval[SKINNY_MAX][kShortK];
  __shared__ int64_t lco[kShortK], scol[kShortK];
  __shared__ int64_t wso[SKINNY_MAX], srow[SKINNY_MAX];
  __shared__ int64_t tab_lr[kInnerMax], tab_w[kInnerMax];
  __shared__ int64_t ob_l[kShortSlots], ob_w[kShortSlots];
  const AxisMap& Lrows = long_is_u ? p.u.rows : p.v.rows;
  const AxisMap& Lcols = long_is_u ? p.u.cols : p.v.cols;
  const AxisMap& Srows = long_is_u ? p.v.rows : p.u.rows;
  const AxisMap& Scols = long_is_u ? p.v.cols : p.u.cols;
  const AxisMap& Wl = long_is_u ? p.w.rows : p.w.cols;
  const AxisMap& Ws = long_is_u ? p.w.cols : p.w.rows;
  const double* Lp = long_is_u ? U : V;
  const double* Sp = long_is_u ? V : U;
  const int64_t nL = long_is_u ? p.M : p.N;
  const int64_t es = p.es;
  constexpr int RU = ShortUnroll<KT>::value;
  constexpr int KX = KT > 0 ? KT : 1;
  const int K = KT ? KT : (int)p.K;
  const int64_t per_q = (nL + kShortRows - 1) / kShortRows;
  // the rows of L and W's axis along the long side index the same modes
  const int64_t I = inner_extent(Lrows, Wl);
  const bool tabulated = I >= 32;   // then a chunk touches <= kShortSlots inner blocks
  if (tabulated) {
    fill_inner(Lrows, I, es, tab_lr);
    fill_inner(Wl, I, es, tab_w);
  }
  // this thread's share of a chunk's offsets: task t falls to lane t / 8 of
  // warp t % 8, so that every warp computes about as many
  const int task0 = (threadIdx.x & 31) * (THREADS / 32) + (threadIdx.x >> 5);
  int staged = -1;
  for (int64_t blk = blockIdx.x; blk < per_q * p.n_q; blk += gridDim.x) {
    const int b = (int)div_idx(blk, per_q);
    const int64_t l0 = (blk - (int64_t)b * per_q) * kShortRows;
    const int64_t lend = l0 + kShortRows < nL ? l0 + kShortRows : nL;
    const int64_t o0 = div_idx(l0, I);
    const int Q = batch_irrep(p, b);
    __syncthreads();   // the previous chunk's readers are done
    // one offset per task: on a new irrep first the short rows in S, S's and
    // L's columns and the short rows along W (2 NS + 2 K), then L's and W's
    // offsets of the chunk's inner blocks (alternating)
    const bool stage = b != staged;
    const int n_s = stage ? 2 * NS + 2 * K : 0;
    const int n_t = n_s + (tabulated ? 2 * (int)(div_idx(lend - 1, I) - o0 + 1) : 0);
    for (int t = task0; t < n_t; t += THREADS) {
      const AxisMap* m;
      int64_t r, sc = es;
      int64_t* dst;
      if (t >= n_s) {
        const int j = (t - n_s) / 2;
        m = ((t - n_s) & 1) ? &Wl : &Lrows;
        r = (o0 + j) * I;
        dst = ((t - n_s) & 1) ? &ob_w[j] : &ob_l[j];
      } else if (t < NS) {
        m = &Srows;
        r = t;
        sc = 1;
        dst = &srow[t];
      } else if (t < NS + K) {
        m = &Scols;
        r = t - NS;
        sc = 1;
        dst = &scol[t - NS];
      } else if (t < NS + 2 * K) {
        m = &Lcols;
        r = t - NS - K;
        dst = &lco[t - NS - K];
      } else {
        m = &Ws;
        r = t - NS - 2 * K;
        dst = &wso[t - NS - 2 * K];
      }
      *dst = sc * aoff(*m, p.g, Q, r);
    }
    __syncthreads();
    if (stage) {
      for (int i = threadIdx.x; i < NS * K; i += THREADS) {
        const int sr = i / K, k = i - sr * K;
        sval[sr][k] = signed_result(p, Sp[es * (srow[sr] + scol[k])]);
      }
      staged = b;
      __syncthreads();
    }
    // a row's two columns of L (two short rows of W) adjacent in memory
    const bool pair_l = K == 2 && lco[1] == lco[0] + 1;
    const bool pair_w = NS == 2 && wso[1] == wso[0] + 1;
    if (!tabulated) {
      // short inner blocks: the offsets of each row from scratch
      for (int64_t l = l0 + threadIdx.x; l < lend; l += THREADS) {
        const int64_t lo = es * aoff(Lrows, p.g, Q, l), wo = es * aoff(Wl, p.g, Q, l);
        double acc[NS];
#pragma unroll
        for (int sr = 0; sr < NS; ++sr) acc[sr] = 0.0;
        for (int k = 0; k < K; ++k) {
          const double x = Lp[lo + lco[k]];
#pragma unroll
          for (int sr = 0; sr < NS; ++sr) acc[sr] = fma(x, sval[sr][k], acc[sr]);
        }
#pragma unroll
        for (int sr = 0; sr < NS; ++sr) put_w(p.accumulate, W + (wo + wso[sr]), acc[sr]);
      }
      continue;
    }
    // (o - o0, i) of the thread's first row by one division; rows and inner
    // positions within a chunk in 32 bits (a chunk spans kShortRows rows)
    const int nrows = (int)(lend - l0), Ii = (int)I;
    int orel = (int)(div_idx(l0 + threadIdx.x, I) - o0);
    int i = (int)(l0 + threadIdx.x - (o0 + orel) * I);
    for (int t = threadIdx.x; t < nrows; t += THREADS * RU) {
      // RU rows: every load first, then the products and stores, the W
      // offsets found again from the saved (o - o0, i)
      const int os = orel, is = i;
      if (KT > 0) {
        double x[RU][KX];
#pragma unroll
        for (int r = 0; r < RU; ++r) {
          const bool ok = t + r * THREADS < nrows;
          const int64_t lo = ok ? ob_l[orel] + tab_lr[i] : 0;
          const double* src = Lp + (lo + lco[0]);
          if (KX == 2 && ok && pair_l && ((uintptr_t)src & 15) == 0) {
            // a row's two entries adjacent: one 16-byte load
            const double2 v2 = *reinterpret_cast<const double2*>(src);
            x[r][0] = v2.x;
            x[r][KX - 1] = v2.y;
          } else {
#pragma unroll
            for (int k = 0; k < KX; ++k) x[r][k] = ok ? Lp[lo + lco[k]] : 0.0;
          }
          if (ok) step_rows(Ii, orel, i);
        }
        int o2 = os, i2 = is;
#pragma unroll
        for (int r = 0; r < RU; ++r) {
          if (t + r * THREADS >= nrows) break;
          const int64_t wo = ob_w[o2] + tab_w[i2];
          double a[NS];
#pragma unroll
          for (int sr = 0; sr < NS; ++sr) {
            // the sum starts from the first product (not an FMA onto 0.0:
            // the float64 pipe is the bound here)
            a[sr] = x[r][0] * sval[sr][0];
#pragma unroll
            for (int k = 1; k < KX; ++k) a[sr] = fma(x[r][k], sval[sr][k], a[sr]);
          }
          double* dst = W + (wo + wso[0]);
          if (NS == 2 && pair_w && !p.accumulate && ((uintptr_t)dst & 15) == 0) {
            // the row's two results adjacent: one 16-byte store
            *reinterpret_cast<double2*>(dst) = make_double2(a[0], a[NS - 1]);
          } else {
#pragma unroll
            for (int sr = 0; sr < NS; ++sr) put_w(p.accumulate, W + (wo + wso[sr]), a[sr]);
          }
          step_rows(Ii, o2, i2);
        }
      } else {
        int64_t wo[RU];
        int64_t lo[RU];
#pragma unroll
        for (int r = 0; r < RU; ++r) {
          const bool ok = t + r * THREADS < nrows;
          lo[r] = ok ? ob_l[orel] + tab_lr[i] : -1;
          wo[r] = ok ? ob_w[orel] + tab_w[i] : 0;
          if (ok) step_rows(Ii, orel, i);
        }
        double acc[RU][NS];
#pragma unroll
        for (int r = 0; r < RU; ++r)
#pragma unroll
          for (int sr = 0; sr < NS; ++sr) acc[r][sr] = 0.0;
        for (int k = 0; k < K; ++k) {
          double x[RU];
#pragma unroll
          for (int r = 0; r < RU; ++r) x[r] = lo[r] >= 0 ? Lp[lo[r] + lco[k]] : 0.0;
#pragma unroll
          for (int r = 0; r < RU; ++r)
#pragma unroll
            for (int sr = 0; sr < NS; ++sr) acc[r][sr] = fma(x[r], sval[sr][k], acc[r][sr]);
        }
#pragma unroll
        for (int r = 0; r < RU; ++r) {
          if (lo[r] < 0) break;
#pragma unroll
          for (int sr = 0; sr < NS; ++sr) put_w(p.accumulate, W + (wo[r] + wso[sr]), acc[r][sr]);
        }
      }
    }
  }
}

// Zero the entries of W that a split-K launch accumulates into.
__global__ void zero_w_entries(const __grid_constant__ Problem p, double* __restrict__ W) {
  int64_t total = (int64_t)p.n_q * p.M * p.N;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
       i += (int64_t)gridDim.x * blockDim.x) {
    int64_t b = i / (p.M * p.N);
    int64_t r = i - b * p.M * p.N;
    int64_t m = r / p.N, n = r % p.N;
    int Q = batch_irrep(p, (int)b);
    W[p.es * (aoff(p.w.rows, p.g, Q, m) + aoff(p.w.cols, p.g, Q, n))] = 0.0;
  }
}

// Resident blocks per SM of a kernel instance (cached per device).
template <typename Kernel>
int blocks_per_sm(Kernel kernel, int* cache) {
  int dev = 0;
  cudaGetDevice(&dev);
  int& c = cache[dev & 63];
  if (c == 0) {
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, THREADS, 0) != cudaSuccess || n < 1) n = 1;
    c = n;
  }
  return c;
}

template <int NS, int KT>
void launch_shortk_kt(int sms, int64_t chunks, cudaStream_t st, const Problem& p, bool long_is_u, const double* u,
                      const double* v, double* w) {
  // a persistent grid: a block stages an irrep's values once and walks its chunks
  static int cache[64] = {};
  const int64_t resident = (int64_t)blocks_per_sm(gemm_f64_shortk<NS, KT>, cache) * sms;
  const int grid = (int)(chunks < resident ? chunks : resident);
  gemm_f64_shortk<NS, KT><<<grid, THREADS, 0, st>>>(p, long_is_u, u, v, w);
}

template <int NS>
void launch_shortk_ns(int kt, int sms, int64_t chunks, cudaStream_t st, const Problem& p, bool long_is_u,
                      const double* u, const double* v, double* w) {
  if (kt == 1) launch_shortk_kt<NS, 1>(sms, chunks, st, p, long_is_u, u, v, w);
  else if (kt == 2) launch_shortk_kt<NS, 2>(sms, chunks, st, p, long_is_u, u, v, w);
  else launch_shortk_kt<NS, 0>(sms, chunks, st, p, long_is_u, u, v, w);
}

// Resident warps of the skinny kernel's instance for NS short-side rows
// (cached per device).
template <int NS>
int64_t skinny_resident_warps(int sms) {
  static int cache[64] = {};
  return (int64_t)blocks_per_sm(gemm_f64_skinny<NS>, cache) * sms * (THREADS / 32);
}

template <int NS>
void launch_skinny_ns(int sms, cudaStream_t st, const Problem& p, bool long_is_u, const double* u,
                      const double* v, double* w) {
  const int64_t nL = long_is_u ? p.M : p.N;
  const int64_t rows = nL * p.n_q;
  const int64_t resident = skinny_resident_warps<NS>(sms);
  // one item per resident warp where the rows are fewer, K ranges of at
  // least 512 entries
  int64_t ksplit = 1;
  if (rows < resident) {
    ksplit = resident / rows;
    const int64_t most = p.K / 512 > 1 ? p.K / 512 : 1;
    if (ksplit > most) ksplit = most;
  }
  if (ksplit > 1 && !p.accumulate) {
    zero_w_entries<<<sms * 4, 256, 0, st>>>(p, w);
    ++g_kernel_launches;
  }
  const int64_t items = rows * ksplit;   // at most; the kernel rounds K ranges to inner blocks
  const int64_t blocks = (items * 32 + THREADS - 1) / THREADS;
  const int64_t cap = resident / (THREADS / 32);
  const int grid = (int)(blocks < cap ? blocks : cap);
  gemm_f64_skinny<NS><<<grid, THREADS, 0, st>>>(p, long_is_u, (int)ksplit, u, v, w);
}

// Tile and K ranges of the tiled kernel: the least time of the busiest SM.  A K
// block of a T x T tile takes 8 T^2 clocks of the float64 pipe, and more for
// offsets, gathers and barriers, the more the fewer tiles share an SM (`shared`,
// `alone`: measured at 640 x 640 x 2000 by 2 irreps and at 64 x 64 x 16384).  K
// ranges (2, 4, 8 or 16 of at least 256 columns) cost the exchange of their sums;
// clusters of 8 and 16 do not spread over all SMs of a GPC (a quarter left out:
// 64 x 64 x 16384 in 16 x 16 tiles by 8 ranges takes 279 us, not 179).
struct TileChoice {
  int T = 64, ksplit = 1;
  int64_t kchunk = 0, units = 0;
};
TileChoice tile_choice(const Problem& p, int sms) {
  TileChoice best;
  double least = 0;
  for (int T : {64, 32, 16, 8}) {
    const double shared = T == 64 ? 500 : T == 32 ? 190 : T == 16 ? 40 : 130, alone = T == 64 ? 1000 : T == 32 ? 900 : 600;
    const int64_t tiles = ((p.M + T - 1) / T) * ((p.N + T - 1) / T) * p.n_q;
    for (int s = 1; s <= kMaxRanges && (s == 1 || p.K / s >= 256); s *= 2) {
      const int64_t blocks = ((p.K + s - 1) / s + BK - 1) / BK;   // K blocks of a range
      const int64_t ranges = (p.K + blocks * BK - 1) / (blocks * BK);
      const int64_t units = tiles * ranges, at_once = ranges >= 8 ? (int64_t)sms * 3 / 4 : sms;
      const int64_t rounds = (units + at_once - 1) / at_once;
      double time = (double)rounds * blocks * (8.0 * T * T + (rounds > 1 ? shared : alone));
      if (ranges > 1) time = time * (1 + 0.005 * ranges) + 3000 + 300 * ranges;
      if (best.units == 0 || time < 0.97 * least) {
        least = time;
        best.T = T;
        best.ksplit = (int)ranges;
        best.kchunk = blocks * BK;
        best.units = units;
      }
    }
  }
  return best;
}

}  // namespace

cudaError_t launch_gemm_f64(const Problem& p, const double* u, const double* v, double* w,
                            const Tables* tables, cudaStream_t st) {
  if (p.n_q == 0 || p.M == 0 || p.N == 0) return cudaSuccess;
  const int sms = device_sms();
  // general plans take the tiled kernel with their tables (every shape)
  bool skinny = !tables && (p.M < 16 || p.N < 16);
  if (skinny && (p.M <= SKINNY_MAX || p.N <= SKINNY_MAX)) {
    bool long_is_u = p.N <= SKINNY_MAX ? true : false;
    // both sides short: an item reads one long-side row and every short-side
    // row along its K range, nL * (1 + nS) rows in all, fewest with the
    // shorter side as the long one
    if (p.M <= SKINNY_MAX && p.N <= SKINNY_MAX) long_is_u = p.M <= p.N;
    const int nS = (int)(long_is_u ? p.N : p.M);
    if (p.K <= kShortK) {
      const int64_t nL = long_is_u ? p.M : p.N;
      const int64_t chunks = (nL + kShortRows - 1) / kShortRows * p.n_q;
      const int kt = p.K == 1 ? 1 : (p.K == 2 ? 2 : 0);
      switch (nS) {
        case 1: launch_shortk_ns<1>(kt, sms, chunks, st, p, long_is_u, u, v, w); break;
        case 2: launch_shortk_ns<2>(kt, sms, chunks, st, p, long_is_u, u, v, w); break;
        case 3: launch_shortk_ns<3>(kt, sms, chunks, st, p, long_is_u, u, v, w); break;
        case 4: launch_shortk_ns<4>(kt, sms, chunks, st, p, long_is_u, u, v, w); break;
        case 5: launch_shortk_ns<5>(kt, sms, chunks, st, p, long_is_u, u, v, w); break;
        case 6: launch_shortk_ns<6>(kt, sms, chunks, st, p, long_is_u, u, v, w); break;
        case 7: launch_shortk_ns<7>(kt, sms, chunks, st, p, long_is_u, u, v, w); break;
        default: launch_shortk_ns<8>(kt, sms, chunks, st, p, long_is_u, u, v, w); break;
      }
      ++g_kernel_launches;
      return cudaGetLastError();
    }
    switch (nS) {
      case 1: launch_skinny_ns<1>(sms, st, p, long_is_u, u, v, w); break;
      case 2: launch_skinny_ns<2>(sms, st, p, long_is_u, u, v, w); break;
      case 3: launch_skinny_ns<3>(sms, st, p, long_is_u, u, v, w); break;
      case 4: launch_skinny_ns<4>(sms, st, p, long_is_u, u, v, w); break;
      case 5: launch_skinny_ns<5>(sms, st, p, long_is_u, u, v, w); break;
      case 6: launch_skinny_ns<6>(sms, st, p, long_is_u, u, v, w); break;
      case 7: launch_skinny_ns<7>(sms, st, p, long_is_u, u, v, w); break;
      default: launch_skinny_ns<8>(sms, st, p, long_is_u, u, v, w); break;
    }
    ++g_kernel_launches;
    return cudaGetLastError();
  }
  const TileChoice c = tile_choice(p, sms);
  Tables t{};
  if (tables) t = *tables;
  auto kern = c.T == 64 ? gemm_f64_tiled<64> : c.T == 32 ? gemm_f64_tiled<32> : c.T == 16 ? gemm_f64_tiled<16>
                                                                                      : gemm_f64_tiled<8>;
  if (c.units > 0x7FFFFFFF) return cudaErrorInvalidConfiguration;
  if (c.ksplit > 8) {
    // clusters beyond eight CTAs are opted into (every thread sets the same)
    const cudaError_t e = cudaFuncSetAttribute((const void*)kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)c.units);
  cfg.blockDim = dim3(THREADS);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)c.ksplit;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = c.ksplit > 1 ? 1 : 0;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, p, c.ksplit, c.kchunk, map_rows_fast(p.u.rows),
                                           map_rows_fast(p.v.rows), t, u, v, w);
  ++g_kernel_launches;
  return e;
}

}  // namespace symctr
