// FP32-compensated forward pass of global Shepard IDW (Sec. 2.1, Eq. 1),
// for one problem or a batch of independent problems in one launch.
//
// Pipeline (one call): coordinate range scan -> staging -> persistent
// all-pairs sweep -> combine (FP64 division) -> for problems of more than
// 2048 points, the search for the exact hits among the flagged queries and
// the results of those queries, in one kernel (smaller problems' flagged queries
// are finished by the combine).
//
// The sweep is the paper's tiled kernel (Sec. 4.2: the data are read once
// per block of prediction points, tile by tile) rebuilt for sm_103a:
//   * each thread holds 2*kQueryPairsF32 queries in registers as pairs, so
//     every FP32 operation is a packed fp32x2 instruction over two queries;
//   * data tiles stream global -> shared by 1-D bulk TMA into a ring of
//     stages guarded by mbarriers (bounded waits); every warp reads the same
//     record (a broadcast shared load);
//   * the record is staged pre-duplicated as (x,x,y,y)+(z,z) so it feeds the
//     packed instructions with no register moves (the paper's aligned AoS
//     record, Sec. 3.3, widened for pair arithmetic);
//   * w = d^-p without a square root.  p = 2: one MUFU reciprocal of d^2,
//     except that for one of the query pairs the two pairs share one
//     reciprocal, 1/(da db), and recover 1/da = db/(da db) with two FMULs;
//     this moves work from the MUFU pipe (the binding one) to the FMA pipe.
//     p = 1, 3, 4: powers of one MUFU reciprocal square root (1, 3) or
//     reciprocal (4, shared as at p = 2).
//     Other p: 2^(-(p/2) log2 d^2) with the product's rounding error
//     recovered by an FMA and applied to first order;
//   * sums run in chunks of 64 (p = 2) or 32 points: S0 as a balanced
//     binary tree, S1 as FMA chains of products joined by a tree; each chunk
//     sum is folded into a (hi, lo) pair by Knuth's TwoSum (the pairs live in
//     shared memory, one slot per thread and query pair) and the pair is
//     renormalised once per work unit, so the worst-case error is a fixed
//     number of roundings per term, independent of n;
//   * the (problem, query tile, data tile) work units are split evenly over
//     a grid of co-resident CTAs (stream-K).  Pieces of a query tile are
//     summed as compensated FP32 pairs by the combine, which converts each
//     query's sums to FP64 once for the division; it plays the role of the
//     paper's in-block reduction of the improved CDP kernel (Sec. 3.1).
//   * coordinates are multiplied by a power of two per problem (exact in
//     FP32) so the largest magnitude lies in [2^9, 2^10): Eq. 1 depends only
//     on distance ratios, so Z is unchanged, and products of squared
//     distances cannot overflow.
#include <algorithm>
#include <cfloat>
#include <cmath>
#include <utility>

#include "idw_device.cuh"
#include "idw_internal.h"
#include "idw_f32_common.cuh"
#include "idw_slowpath.cuh"

namespace idw {
namespace {

constexpr int TB = kRecordsF32;
constexpr int ST = kStagesF32;
constexpr uint32_t kTileBytes = static_cast<uint32_t>(kTileBytesF32);
static_assert(kTileBytes % 16 == 0, "bulk copies move multiples of 16 bytes");
constexpr bool chunk_shape_ok(ChunkShape c) {
  return TB % c.points == 0 && c.points == (1 << c.tree_levels) &&
         c.points == c.chain << c.chain_levels;
}
static_assert(chunk_shape_ok(kChunkPow2) && chunk_shape_ok(kChunkGeneral), "chunk trees");

// Compiled sweep variants (the autotuner picks one per size class):
// threads per CTA, query pairs per thread, and how many of those pairs share
// one reciprocal per data point at p = 2.  Each keeps 128 registers/thread
// and 16 resident warps per SM (variant 4: all 16 in one CTA, which keeps
// them in step at every tile barrier).
// KSH pairs share on every data point; pair KALT (if >= 0) also shares on
// every other data point, so a fraction (KSH + 0.5 [KALT >= 0]) / KP of the
// pairs share.
// TBV is the number of data points per work unit: 256 (one staging tile),
// or 64 for the fine-grained variant 5, which splits small problems into
// four times as many units; it needs the record-contiguous aligned-AoS
// staging (p = 2).
template <int V> struct Var;
template <> struct Var<0> { static constexpr int NT = 256, KP = 4, KSH = 1, KALT = -1, TBV = 256; };
template <> struct Var<1> { static constexpr int NT = 256, KP = 4, KSH = 0, KALT = -1, TBV = 256; };
template <> struct Var<2> { static constexpr int NT = 256, KP = 4, KSH = 1, KALT = 1, TBV = 256; };
template <> struct Var<3> { static constexpr int NT = 128, KP = 4, KSH = 1, KALT = -1, TBV = 256; };
template <> struct Var<4> { static constexpr int NT = 512, KP = 4, KSH = 1, KALT = 1, TBV = 256; };
template <> struct Var<5> { static constexpr int NT = 256, KP = 4, KSH = 1, KALT = -1, TBV = 64; };
template <> struct Var<6> { static constexpr int NT = 64, KP = 4, KSH = 1, KALT = -1, TBV = 64; };
template <> struct Var<7> { static constexpr int NT = 64, KP = 4, KSH = 1, KALT = -1, TBV = 256; };
template <int V> __host__ __device__ constexpr int qt_of() { return Var<V>::NT * 2 * Var<V>::KP; }
static_assert(kNumAllVariants == 8, "variant table");
static_assert(qt_of<0>() == kQueriesPerCtaF32, "default variant is the documented tiling");

struct SweepArgs {
  int64_t units;
  int grid;
  float half_p, neg_half_p;
  float4* partial;  // partial_slots x QT records (S0 hi, S0 lo, S1 hi, S1 lo)
  const float* scales;
  unsigned* err;
};

// log2 on the FMA pipe, for both lanes: x = 2^k m, m in [1/sqrt 2, sqrt 2),
// log2 x = k + s P(s), s = m - 1 (exact), P the degree-8 minimax fit of
// log2(1 + s)/s for the relative error (Remez exchange, fit_log2.py),
// rounded to fp32 and evaluated by Horner's rule with packed FMAs.  Zero or
// subnormal x gives -inf and an infinite or NaN x gives 2^20, as the MUFU
// path with its clamp does.  Error: at most 1.5u absolute for x in
// [1/2, 2] and 1.5u relative to |log2 x| elsewhere (checked exhaustively
// on the CPU).
__constant__ float kLog2Poly[] = {
    1.4426950216293335f,  -0.7213473320007324f, 0.48091062903404236f,
    -0.3607036769390106f, 0.28791624307632446f, -0.23894482851028442f,
    0.21571560204029083f, -0.20726972818374634f, 0.12583701312541962f,
};
constexpr int kLog2PolyDegree = 8;

__device__ __forceinline__ u64 log2_fma_pair(u64 x2) {
  float xa, xb;
  upk(x2, xa, xb);
  const int ua = __float_as_int(xa), ub = __float_as_int(xb);
  const int ka = (ua - 0x3F3504F3) >> 23, kb = (ub - 0x3F3504F3) >> 23;  // m >= 1/sqrt 2
  const u64 m = pk(__int_as_float(ua - (ka << 23)), __int_as_float(ub - (kb << 23)));
  // float(k) exactly: k sits in the low mantissa bits of 1.5 2^23.
  const u64 kf = pk(__int_as_float(0x4B400000 + ka) - 12582912.f,
                    __int_as_float(0x4B400000 + kb) - 12582912.f);
  const u64 sv = sub2(m, pk(1.f, 1.f));
  u64 poly = pk(kLog2Poly[kLog2PolyDegree], kLog2Poly[kLog2PolyDegree]);
#pragma unroll
  for (int i = kLog2PolyDegree - 1; i >= 0; --i) poly = fma2(poly, sv, pk(kLog2Poly[i], kLog2Poly[i]));
  float la, lb;
  upk(fma2(sv, poly, kf), la, lb);
  const int ea = (ua >> 23) & 0xff, eb = (ub >> 23) & 0xff;
  la = ea == 0 ? -INFINITY : (ea == 0xff ? 1048576.f : la);
  lb = eb == 0 ? -INFINITY : (eb == 0xff ? 1048576.f : lb);
  return pk(la, lb);
}

template <int MODE>
__device__ __forceinline__ u64 weight_pair(u64 d2, bool shared_rcp, u64 half_p2,
                                           u64 neg_half_p2, bool fma_log2 = false) {
  float a, b;
  upk(d2, a, b);
  if (MODE == kPow2 || MODE == kPow4) {
    u64 w;
    if (shared_rcp) {
      const float r = rcp_approx(mul_ftz(a, b));  // 1 / (da db)
      w = pk(mul_ftz(b, r), mul_ftz(a, r));
    } else {
      w = pk(rcp_approx(a), rcp_approx(b));
    }
    return MODE == kPow4 ? mul2f(w, w) : w;
  } else if (MODE == kPow1 || MODE == kPow3) {
    const u64 r = pk(rsqrt_approx(a), rsqrt_approx(b));
    return MODE == kPow3 ? mul2f(mul2f(r, r), r) : r;
  } else {
    // L = log2 d^2, clamped so that +inf (padding) stays finite below; on
    // the MUFU pipe, or for a fixed fraction of the pairs on the FMA pipe.
    const u64 L = fma_log2 ? log2_fma_pair(d2)
                           : pk(fminf(lg2_approx(a), 1048576.f), fminf(lg2_approx(b), 1048576.f));
    const u64 th = mul2(L, neg_half_p2);  // t_hi = fl(t), t = -(p/2) L
    // (p/2) L + t_hi = -(t - t_hi): the product's rounding error, exact.
    const u64 ntl = fma2(L, half_p2, th);
    float ta, tb;
    upk(th, ta, tb);
    const u64 e = pk(ex2_approx(ta), ex2_approx(tb));
    const u64 c = mul2(ntl, pk(-0.6931471805599453f, -0.6931471805599453f));  // t_lo ln 2
    return fma2(e, c, e);  // 2^(t_hi + t_lo) to first order in t_lo
  }
}

// General power with the FMA-pipe log2 (IDW_OPT_FMA_LOG2): query pair 0
// takes log2 d^2 on the FMA pipe for the data points r with
// r % kLog2FmaPeriod == 0, 1 pair in 16.  The MUFU pipe (lg2 at 16 and ex2
// at 32 per SM per clock) binds the general sweep while the FMA pipe is 73 %
// busy, yet every fraction measured (1/16 to 1/4) was slower: the polynomial
// and its exponent handling cost more issue slots than the lg2 they replace.
// It is kept as an option, off by default.
constexpr int kLog2FmaPeriod = 4;

// The record of data point c + r of a staged tile as three register pairs
// (x,x), (y,y), (z,z), for each staging layout.
template <int LAYOUT>
__device__ __forceinline__ void load_record(const unsigned char* tile, int i, u64& xx, u64& yy,
                                            u64& zz) {
  if (LAYOUT == 0) {
    const ulonglong2 xy = reinterpret_cast<const ulonglong2*>(tile)[i];
    xx = xy.x;
    yy = xy.y;
    zz = reinterpret_cast<const u64*>(tile + TB * 16)[i];
  } else if (LAYOUT == 1) {
    const float4 v = reinterpret_cast<const float4*>(tile)[i];
    xx = pk(v.x, v.x);
    yy = pk(v.y, v.y);
    zz = pk(v.z, v.z);
  } else {
    const float* f = reinterpret_cast<const float*>(tile);
    const float x = f[i], y = f[TB + i], z = f[2 * TB + i];
    xx = pk(x, x);
    yy = pk(y, y);
    zz = pk(z, z);
  }
}

// The running (hi, lo) pairs of a thread: slot 2k holds (S0 hi, S0 lo) of
// query pair k and slot 2k + 1 (S1 hi, S1 lo), each a pair of packed lanes;
// in registers, or in shared memory at [s NT + tid] after the tile ring.
constexpr bool kSumsInShared = true;

template <int KP, int NT, bool SMEM>
struct SumSlots;
template <int KP, int NT>
struct SumSlots<KP, NT, false> {
  ulonglong2 r[2 * KP];
  __device__ __forceinline__ void bind(unsigned char*, int) {}
  __device__ __forceinline__ ulonglong2 get(int s) const { return r[s]; }
  __device__ __forceinline__ void set(int s, ulonglong2 v) { r[s] = v; }
};
template <int KP, int NT>
struct SumSlots<KP, NT, true> {
  ulonglong2* base;  // this thread's slot 0
  __device__ __forceinline__ void bind(unsigned char* p, int tid) {
    base = reinterpret_cast<ulonglong2*>(p) + tid;
  }
  __device__ __forceinline__ ulonglong2 get(int s) const { return base[s * NT]; }
  __device__ __forceinline__ void set(int s, ulonglong2 v) { base[s * NT] = v; }
};

// Shared memory of one sweep CTA: the tile ring, then the sum slots.
template <int V, int LAYOUT>
__host__ __device__ constexpr size_t ring_bytes_of() {
  return size_t(ST) * (Var<V>::TBV == TB ? tile_bytes_of<LAYOUT>() : Var<V>::TBV * 16u);
}
template <int V>
__host__ __device__ constexpr size_t hl_bytes_of() {
  return kSumsInShared ? size_t(2) * Var<V>::KP * Var<V>::NT * sizeof(ulonglong2) : 0;
}
template <int V, int LAYOUT>
__host__ __device__ constexpr size_t sweep_smem_of() {
  return ring_bytes_of<V, LAYOUT>() + hl_bytes_of<V>();
}

template <int MODE, int CAP, int V, int LAYOUT = 0, bool FMA_LOG2 = false>
__global__ void __launch_bounds__(Var<V>::NT, 512 / Var<V>::NT)
    sweep_kernel(const SweepArgs a, const __grid_constant__ Table<CAP> t) {
  constexpr int NT = Var<V>::NT, KP = Var<V>::KP, KSHARED = Var<V>::KSH, QT = qt_of<V>();
  constexpr int KALT = Var<V>::KALT;
  constexpr ChunkShape SH = MODE == kPow2 ? kChunkPow2 : kChunkGeneral;
  constexpr int CH = SH.points;
  constexpr int TBU = Var<V>::TBV;
  static_assert(TBU == TB || LAYOUT == 1, "sub-tile units need record-contiguous staging");
  static_assert(TBU % CH == 0, "chunks tile a work unit");
  // Bytes of one work unit's data: a whole staging tile, or a slice of the
  // record-contiguous aligned-AoS array.
  constexpr uint32_t kTileBytes = TBU == TB ? tile_bytes_of<LAYOUT>() : TBU * 16u;
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) unsigned long long full_bar[ST];
  SumSlots<KP, NT, kSumsInShared> HL;
  HL.bind(smem + ring_bytes_of<V, LAYOUT>(), threadIdx.x);

  const int tid = threadIdx.x;
  const int64_t g = blockIdx.x;
  const int64_t u0 = unit_begin(g, a.units, a.grid);
  const int64_t total = unit_begin(g + 1, a.units, a.grid) - u0;
  if (total <= 0) return;

  if (tid == 0) {
    for (int s = 0; s < ST; ++s) mbar_init(smem_u32(&full_bar[s]), 1);
    fence_barrier_init();
  }
  pdl_trigger();
  pdl_wait();  // the staged tiles and scales come from the kernels before
  __syncthreads();

  // Producer (thread 0): one bulk copy per unit, STAGES units ahead.
  int64_t issued = 0;
  int pk_inst = find_unit(t, u0);
  auto issue = [&](int64_t local) {
    const int64_t u = u0 + local;
    while (pk_inst + 1 < t.count && t.inst[pk_inst + 1].unit_base <= u) ++pk_inst;
    const Instance& I = t.inst[pk_inst];
    const int64_t dt = (u - I.unit_base) % I.data_tiles;
    const int s = static_cast<int>(local % ST);
    bulk_load(smem_u32(smem + s * kTileBytes), I.tiles + dt * kTileBytes, kTileBytes,
              smem_u32(&full_bar[s]));
  };
  if (tid == 0) {
    for (; issued < ST && issued < total; ++issued) issue(issued);
  }

  const u64 hp2 = pk(a.half_p, a.half_p);
  const u64 nhp2 = pk(a.neg_half_p, a.neg_half_p);
  int ci = find_unit(t, u0);
  int64_t i = 0;
  bool aborted = false;
  while (i < total) {
    const int64_t u = u0 + i;
    while (ci + 1 < t.count && t.inst[ci + 1].unit_base <= u) ++ci;
    const Instance& I = t.inst[ci];
    const int64_t qt = (u - I.unit_base) / I.data_tiles;
    const int64_t seg_end = min(total, I.unit_base + (qt + 1) * I.data_tiles - u0);
    const float sc = a.scales[ci];

    u64 QX[KP], QY[KP];
#pragma unroll
    for (int k = 0; k < KP; ++k) {
      const int64_t ja = qt * QT + (2 * k) * NT + tid;
      const int64_t jb = ja + NT;
      const float xa = ja < I.m ? I.queries[2 * ja] * sc : 0.f;
      const float ya = ja < I.m ? I.queries[2 * ja + 1] * sc : 0.f;
      const float xb = jb < I.m ? I.queries[2 * jb] * sc : 0.f;
      const float yb = jb < I.m ? I.queries[2 * jb + 1] * sc : 0.f;
      QX[k] = pk(xa, xb);
      QY[k] = pk(ya, yb);
      HL.set(2 * k, make_ulonglong2(0ull, 0ull));
      HL.set(2 * k + 1, make_ulonglong2(0ull, 0ull));
    }

    for (; i < seg_end; ++i) {
      const int s = static_cast<int>(i % ST);
      const uint32_t parity = static_cast<uint32_t>((i / ST) & 1);
      const bool ok = mbar_wait_bounded(smem_u32(&full_bar[s]), parity, a.err);
      if (ok) {
        const unsigned char* tile = smem + s * kTileBytes;
#pragma unroll 1
        for (int c = 0; c < TBU; c += CH) {
          // S0: tree over the chunk's weights.  S1: chains of SH.chain
          // products w z (one MUL, then FMAs), chains joined by a tree.
          u64 P0[KP][SH.tree_levels], P1[KP][SH.chain_levels], T1[KP], C0[KP], C1[KP];
#pragma unroll
          for (int r = 0; r < CH; ++r) {
            u64 xx, yy, zz;
            load_record<LAYOUT>(tile, c + r, xx, yy, zz);
#pragma unroll
            for (int k = 0; k < KP; ++k) {
              // d^2 rounded to nearest with subnormals kept: a d^2 that is
              // itself subnormal is flushed by the weight's MUFU input and
              // sends the query to the FP64 path through a non-finite sum.
              const u64 dx = sub2(QX[k], xx);
              const u64 dy = sub2(QY[k], yy);
              const u64 d2 = fma2(dy, dy, mul2(dx, dx));
              const bool shared = shares_reciprocals(MODE) && (k < KSHARED || (k == KALT && (r & 1)));
              const bool fma_log2 = FMA_LOG2 && k == 0 && r % kLog2FmaPeriod == 0;
              const u64 w = weight_pair<MODE>(d2, shared, hp2, nhp2, fma_log2);
              tree_push<SH.tree_levels>(P0[k], w, r, C0[k]);
              if (r % SH.chain == 0) {
                T1[k] = mul2(w, zz);
              } else {
                T1[k] = fma2(w, zz, T1[k]);
              }
              if (r % SH.chain == SH.chain - 1)
                tree_push<SH.chain_levels>(P1[k], T1[k], r / SH.chain, C1[k]);
            }
          }
          // Error-free folds of the chunk sums into the (hi, lo) slots; the
          // last chunk of a work unit also renormalises each pair.
          const bool last = c + CH == TBU;
#pragma unroll
          for (int k = 0; k < KP; ++k) {
            ulonglong2 s0 = HL.get(2 * k);
            ulonglong2 s1 = HL.get(2 * k + 1);
            two_sum_acc(s0.x, s0.y, C0[k]);
            two_sum_acc(s1.x, s1.y, C1[k]);
            if (last) {
              two_sum_renorm(s0.x, s0.y);
              two_sum_renorm(s1.x, s1.y);
            }
            HL.set(2 * k, s0);
            HL.set(2 * k + 1, s1);
          }
        }
      }
      // Every thread is done with stage s (and agrees on whether to stop).
      if (__syncthreads_or(!ok)) {
        aborted = true;
        break;
      }
      if (tid == 0 && issued < total) {
        issue(issued);
        ++issued;
      }
    }
    if (aborted) break;

    float4* P = a.partial + (I.qtile_base + qt + g) * QT;
#pragma unroll
    for (int k = 0; k < KP; ++k) {
      const ulonglong2 s0 = HL.get(2 * k);
      const ulonglong2 s1 = HL.get(2 * k + 1);
      float h0a, h0b, l0a, l0b, h1a, h1b, l1a, l1b;
      upk(s0.x, h0a, h0b);
      upk(s0.y, l0a, l0b);
      upk(s1.x, h1a, h1b);
      upk(s1.y, l1a, l1b);
      P[(2 * k) * NT + tid] = make_float4(h0a, l0a, h1a, l1a);
      P[(2 * k + 1) * NT + tid] = make_float4(h0b, l0b, h1b, l1b);
    }
  }

  if (aborted && tid == 0) {
    // Let every copy still in flight land before the CTA's shared memory
    // is released (each wait is bounded as well).
    for (int64_t k = i; k < issued; ++k)
      mbar_wait_bounded(smem_u32(&full_bar[k % ST]), static_cast<uint32_t>((k / ST) & 1), a.err);
  }
}

// FP64 combine of the pieces of each query: Z = S1 / S0, or, for a query
// outside the fast form (exact hit or FP32 range exceeded), the FP64 slow
// path run by the same CTA.  One CTA covers 32 consecutive query slots
// (lanes x) and splits each query's pieces over 8 warps (lanes y, strided);
// every warp's loads are coalesced across its 32 queries, and the 8 partial
// sums are added in a fixed order, so the result is deterministic.  The
// CTA's flagged queries are then redone by all 256 threads when their problem
// is small or the list full: one scan of the points for all their hits, then the
// FP64 sums of the others one after another.  A query's slow path reads all n
// points, so those of a larger problem are listed for the kernel after this one,
// which spreads each search over the GPU.  (A scan for each query took 6 us of
// 12,000 points, and the CTAs that find the list full have 32 of them: 12,000 x
// 12,000, p = 3.5, all hits 429 us, 206 so.)  Block 0 finally clears
// the per-problem range words the range scan and staging of this call used,
// so the next call (or graph replay) starts from zero without a memset.
//
// Lanes per query: 8, or 32 where a query has many pieces (few query tiles),
// whose loads are otherwise a serial chain.  13,000 x 500 (304 pieces): 22.7
// us by 8 lanes, 19.8 by 32; 100,000 x 2000 74.8 and 69.6; 12,000 x 12,000 (51
// pieces) 50.9 and 53.7; 20,000 x 20,000 (31) 111.7 and 117.3.  6 CTAs per SM:
// left alone the slow path's loads take 64 registers and 4 CTAs (2000 x
// 100,000: 73.3 us, 70.5), and at 8 CTAs it spills (no faster).
constexpr int kCombineManyPieces = 128;
constexpr int kCombineThreads = 256;
static_assert(kCombineThreads == kSlowThreads, "the combine CTA runs the slow path");

// Flagged queries of problems up to this many points stay with their CTA:
// one FP64 recomputation of 2048 points keeps one SM's FP64 pipe busy for
// about 14 us (100,003 points: 690 us), and the kernel that shares larger ones
// out costs about 1.3 us a call.
constexpr int kSlowInlinePoints = 2048;

// A listed query: problem, query, the lowest coincident data index found so
// far (INT_MAX: none), and how many slices of its FP64 sums are done.
struct SlowItem {
  int32_t problem, query, hit;
  unsigned done;
};
static_assert(sizeof(SlowItem) == 16, "slow list record");

// The list, then the slices' FP64 sums, in the staged tiles' memory, which
// nothing reads after the sweep.  A list of c queries is summed in at most
// max(c, grid) slices, so `cap` queries fit; further ones stay with their CTA.
struct SlowList {
  SlowItem* item;
  SlowSums* part;
  unsigned cap;
};

template <int CAP, int QT, int kCombineLanes>
__global__ void __launch_bounds__(kCombineThreads, 6)
    combine_kernel(const __grid_constant__ Table<CAP> t, const float4* partial,
                   int64_t total_slots, int64_t units, int grid, const float* scales,
                   double p, Control* ctrl, const SlowList slow) {
  constexpr int kCombineQueries = kCombineThreads / kCombineLanes;
  __shared__ float4 red[kCombineLanes][kCombineQueries];
  __shared__ int2 flagged[kCombineQueries];
  __shared__ float2 flagged_q[kCombineQueries];
  __shared__ int hit[kCombineQueries];
  __shared__ int nflagged;
  static_assert(QT % kCombineQueries == 0, "a CTA's queries are of one problem");
  pdl_trigger();
  pdl_wait();
  const int lx = threadIdx.x % kCombineQueries, ly = threadIdx.x / kCombineQueries;
  const int64_t idx = int64_t(blockIdx.x) * kCombineQueries + lx;
  bool valid = idx < total_slots;
  const int64_t qtg = idx / QT, lq = idx % QT;
  const int k = valid ? find_qtile(t, qtg) : 0;
  const Instance& I = t.inst[k];
  const int64_t qt = qtg - I.qtile_base;
  const int64_t j = qt * QT + lq;
  valid = valid && j < I.m;
  // Each piece is an (S0 hi, S0 lo, S1 hi, S1 lo) record with |lo| at most
  // half an ulp of hi.  Pieces are added as FP32 (hi, lo) pairs, the hi parts
  // by TwoSum and the lo parts and the TwoSum errors plainly (the loss is of
  // order P^2 u^2 for P pieces): the FP32 pipe runs this at 64 times the FP64
  // pipe's rate.  The sums go to FP64 once, for the division.
  float h0 = 0.f, l0 = 0.f, h1 = 0.f, l1 = 0.f;
  if (valid) {
    const int64_t g0 = cta_of_unit(I.unit_base + qt * I.data_tiles, units, grid);
    const int64_t g1 = cta_of_unit(I.unit_base + (qt + 1) * I.data_tiles - 1, units, grid);
#pragma unroll 4
    for (int64_t g = g0 + ly; g <= g1; g += kCombineLanes) {
      const float4 v = partial[(qtg + g) * QT + lq];
      two_sum_acc_f32(h0, l0, v.x);
      l0 += v.y;
      two_sum_acc_f32(h1, l1, v.z);
      l1 += v.w;
    }
  }
  red[ly][lx] = make_float4(h0, l0, h1, l1);
  if (threadIdx.x == 0) nflagged = 0;
  __syncthreads();
  if (ly == 0 && valid) {
#pragma unroll
    for (int y = 1; y < kCombineLanes; ++y) {
      const float4 r = red[y][lx];
      two_sum_acc_f32(h0, l0, r.x);
      l0 += r.y;
      two_sum_acc_f32(h1, l1, r.z);
      l1 += r.w;
    }
    const double s0 = double(h0) + double(l0), s1 = double(h1) + double(l1);
    if (!(s0 > kTinySumPerPoint * double(I.n)) || !isfinite(s0) || !isfinite(s1) ||
        (p >= 2.0 && s0 > kHugeSumPow2Up)) {
      const unsigned slot = I.n > kSlowInlinePoints ? atomicAdd(&ctrl->flagged, 1u) : slow.cap;
      if (slot < slow.cap) {
        slow.item[slot] = SlowItem{k, static_cast<int32_t>(j), INT_MAX, 0u};
      } else {
        const int f = atomicAdd(&nflagged, 1);
        flagged[f] = make_int2(k, static_cast<int>(j));
        flagged_q[f] = make_float2(I.queries[2 * j], I.queries[2 * j + 1]);
        hit[f] = INT_MAX;
      }
    } else {
      I.out[j] = static_cast<float>(s1 / s0);
      // Weights were computed on coordinates scaled by s: w = s^-p w_true.
      if (I.s0_out) I.s0_out[j] = s0 * pow(double(scales[k]), p);
      if (I.hit_out) I.hit_out[j] = kNoHit;
    }
  }
  __syncthreads();
  const int nf = nflagged;
  if (nf > 0) {  // uniform across the CTA
    const Instance& F = t.inst[flagged[0].x];
    slow_scan(F.data, 0, F.n, [&](int64_t i, float x, float y) {
      for (int f = 0; f < nf; ++f)
        if (flagged_q[f].x == x && flagged_q[f].y == y) atomicMin(&hit[f], static_cast<int>(i));
      return false;
    });
    __syncthreads();
    for (int f = 0; f < nf; ++f) {
      const int64_t jf = flagged[f].y;
      float* out = &F.out[jf];
      double* s0_out = F.s0_out ? &F.s0_out[jf] : nullptr;
      int32_t* hit_out = F.hit_out ? &F.hit_out[jf] : nullptr;
      if (hit[f] != INT_MAX) {
        if (threadIdx.x == f) slow_write_hit(F.data, hit[f], out, s0_out, hit_out);
        continue;
      }
      const SlowSums sums = slow_sums<float>(F.data, 0, F.n, flagged_q[f].x, flagged_q[f].y, p);
      if (threadIdx.x == 0) slow_write_sums(sums, p, out, s0_out, hit_out);
    }
  }
  if (blockIdx.x == 0)
    for (int c = threadIdx.x; c < t.count; c += blockDim.x) ctrl->maxbits[c] = 0u;
}

// The listed queries, in one launch of two steps.
//
// First the exact hits.  A work item is a group of up to 32 listed queries and
// one of S equal slices of their problem's points, S chosen so that few groups'
// items fill the grid and many groups' do so twice: every point is read once per
// group and compared with the group's queries from shared memory, and the lowest
// coincident index is kept with an atomic minimum.
//
// Then the results: a hit's z, or Eq. 1 in FP64.  A query without a hit is one
// whose FP32 sums left FP32's range; among them are the queries that shared a
// reciprocal with a hit (their weight there is NaN).  Its points are cut into
// S slices, S chosen so that all such queries' slices fill the grid (counted
// when the list is short; a list of more than kSlowThreads queries fills it by
// itself); each slice's sums are scaled by its own d2_min, and a warp of the
// CTA that finishes a query's last slice rescales and adds them in a fixed
// order.  A 100,003-point, 65,537-query call with 16 hits spent 860 us on them in
// the combine, one CTA a query: the FP64 pipe of one SM bounds a query; spread
// over the GPU they take under 30 us.
//
// The second step waits for all of the first.  CTAs draw its items from a
// counter, and one waits only when none is left: what it waits for has been
// drawn by CTAs that run, so the wait ends wherever the others are scheduled.
// One launch and not one for each step, because most calls list nothing and pay
// for the launches alone (p = 2 without hits, no list / two launches / this one:
// 12,000 x 12,000 48.9 / 51.0 / 50.2 us, 20,000 x 20,000 109.9 / 112.2 / 111.3).
constexpr int kSlowGroup = 32;
// CTAs to an SM: the FP64 sums wait on divisions and loads, and more warps hide
// them where the list is long; where it is short, more slices cost more than they
// spread, and four CTAs leave 64 registers and spill.  Two / three / four, p = 2:
// 30,000 x 20,000, all hits, 608 / 561 / 515 us; 100,003 x 4096 with one hit 140 /
// 144 / 150, with 16 149 / 152 / 155, with 200 372 / 370 / 383; p = 3.5: 100,003 x
// 65,537, 20% hits, 3376 / 3026 / 3036; 30,000 x 20,000 with 2000 287 / 274 / 274.
constexpr int kSlowCtas = 3;
// One item over all points of the largest problem (2^31) takes several seconds.
constexpr unsigned long long kSlowWaitNs = 60000000000ull;

struct SlowShared {
  float2 q[kSlowGroup];
  int prob[kSlowGroup];
  int work[kSlowThreads];
  int warp_count[kSlowThreads / 32];
  unsigned drawn;
  bool last;
};

// Item w of `slices` to a group: marks its queries' hits among the slice's points.
template <int CAP>
__device__ void slow_search(const Table<CAP>& t, const SlowList& slow, int64_t count, int64_t slices,
                            int64_t w, SlowShared& sh) {
  const int64_t e0 = w / slices * kSlowGroup, sl = w % slices;
  const int ne = static_cast<int>(min(int64_t(kSlowGroup), count - e0));
  if (threadIdx.x < ne) {
    const SlowItem it = slow.item[e0 + threadIdx.x];
    const float* p = t.inst[it.problem].queries + 2 * int64_t(it.query);
    sh.q[threadIdx.x] = make_float2(p[0], p[1]);
    sh.prob[threadIdx.x] = it.problem;
  }
  __syncthreads();
  for (int a = 0; a < ne;) {  // runs of the same problem (uniform across the CTA)
    int b = a + 1;
    while (b < ne && sh.prob[b] == sh.prob[a]) ++b;
    const Instance& I = t.inst[sh.prob[a]];
    slow_scan(I.data, sl * I.n / slices, (sl + 1) * I.n / slices,
              [&](int64_t i, float x, float y) {
                for (int e = a; e < b; ++e)
                  if (sh.q[e].x == x && sh.q[e].y == y)
                    atomicMin(&slow.item[e0 + e].hit, static_cast<int32_t>(i));
                return false;
              });
    a = b;
  }
}

// Listed query f as other CTAs have left it (past this SM's cache).
__device__ __forceinline__ SlowItem slow_item(const SlowList& slow, int64_t f) {
  const int4 v = __ldcg(reinterpret_cast<const int4*>(slow.item + f));
  return SlowItem{v.x, v.y, v.z, static_cast<unsigned>(v.w)};
}

template <int CAP>
__global__ void __launch_bounds__(kSlowThreads, kSlowCtas)
    slow_kernel(const __grid_constant__ Table<CAP> t, Control* ctrl, const SlowList slow, double p) {
  __shared__ SlowShared sh;
  // The kernels behind this one start only when it has gone this far: held back
  // early, they, and the next call's sweep with them, were placed around its
  // CTAs (13,000 x 500, p = 2.5: 45 us a call, 37 so).
  pdl_wait();
  pdl_trigger();
  const int count = static_cast<int>(min(ctrl->flagged, slow.cap));
  if (count == 0) return;
  const int tid = threadIdx.x;

  const int64_t groups = (count + kSlowGroup - 1) / kSlowGroup;
  const int64_t cuts = 4 * groups < gridDim.x ? gridDim.x / groups
                                              : (2 * int64_t(gridDim.x) + groups - 1) / groups;
  const int64_t searches = groups * cuts;
  for (;;) {
    __syncthreads();  // the previous item's group and number are no longer read
    if (tid == 0) sh.drawn = atomicAdd(&ctrl->slow_drawn, 1u);
    __syncthreads();
    if (sh.drawn >= searches) break;
    slow_search<CAP>(t, slow, count, cuts, sh.drawn, sh);
    __threadfence();
    __syncthreads();
    if (tid == 0) atomicAdd(&ctrl->slow_done, 1u);
  }
  if (tid == 0) {
    sh.last = wait_count_bounded(&ctrl->slow_done, static_cast<unsigned>(searches), kSlowWaitNs,
                                 &ctrl->error);
    __threadfence();
  }
  __syncthreads();
  if (!sh.last) return;  // gave up; recorded

  // Hits: one thread each.
  for (int f = blockIdx.x * kSlowThreads + tid; f < count; f += gridDim.x * kSlowThreads) {
    const SlowItem it = slow_item(slow, f);
    if (it.hit == INT_MAX) continue;
    const Instance& I = t.inst[it.problem];
    const int64_t j = it.query;
    slow_write_hit<float, float>(I.data, it.hit, &I.out[j], I.s0_out ? &I.s0_out[j] : nullptr,
                                 I.hit_out ? &I.hit_out[j] : nullptr);
  }
  const bool short_list = count <= kSlowThreads;
  int sums = count;
  if (short_list) {  // the queries without a hit, in list order
    const bool mine = tid < count && slow_item(slow, tid).hit == INT_MAX;
    const unsigned vote = __ballot_sync(0xffffffffu, mine);
    if ((tid & 31) == 0) sh.warp_count[tid >> 5] = __popc(vote);
    __syncthreads();
    int before = 0;
    sums = 0;
    for (int w = 0; w < kSlowThreads / 32; ++w) {
      if (w < (tid >> 5)) before += sh.warp_count[w];
      sums += sh.warp_count[w];
    }
    if (mine) sh.work[before + __popc(vote & ((1u << (tid & 31)) - 1))] = tid;
    __syncthreads();
    if (sums == 0) return;
  }
  const int slices = max(1, int(gridDim.x) / sums);
  for (int64_t w = blockIdx.x; w < int64_t(sums) * slices; w += gridDim.x) {
    const int e = static_cast<int>(w / slices), sl = static_cast<int>(w % slices);
    const int f = short_list ? sh.work[e] : e;
    const SlowItem it = slow_item(slow, f);
    if (it.hit != INT_MAX) continue;  // uniform across the CTA
    const Instance& I = t.inst[it.problem];
    const int64_t j = it.query;
    const SlowSums s = slow_sums<float>(I.data, int64_t(sl) * I.n / slices,
                                        int64_t(sl + 1) * I.n / slices, I.queries[2 * j],
                                        I.queries[2 * j + 1], p);
    if (tid == 0) {
      slow.part[w] = s;
      __threadfence();
      sh.last = atomicAdd(&slow.item[f].done, 1u) + 1u == unsigned(slices);
    }
    __syncthreads();
    if (sh.last && tid < 32) {  // one warp, lanes over the slices, a fixed shuffle tree
      __threadfence();
      const double* P = reinterpret_cast<const double*>(slow.part + (w - sl));
      double dmin = INFINITY;
      for (int k = tid; k < slices; k += 32) dmin = fmin(dmin, __ldcg(P + 3 * k));
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) dmin = fmin(dmin, __shfl_xor_sync(0xffffffffu, dmin, o));
      SlowSums sum{dmin, 0.0, 0.0};
      for (int k = tid; k < slices; k += 32) {
        // A slice at infinity (d2_min = +inf) holds zeros, or NaN to keep.
        const double dk = __ldcg(P + 3 * k);
        const double c = dk == dmin || dk == INFINITY ? 1.0
                         : p == 2.0                   ? dmin / dk
                                                      : pow(dmin / dk, 0.5 * p);
        sum.s0 += __ldcg(P + 3 * k + 1) * c;
        sum.s1 += __ldcg(P + 3 * k + 2) * c;
      }
      sum.s0 = warp_sum(sum.s0);
      sum.s1 = warp_sum(sum.s1);
      if (tid == 0)
        slow_write_sums<float>(sum, p, &I.out[j], I.s0_out ? &I.s0_out[j] : nullptr,
                               I.hit_out ? &I.hit_out[j] : nullptr);
    }
    __syncthreads();  // sh.last is rewritten by the next item
  }
}

// One thread waits, as the slow list's kernel does, for a count that nothing
// reaches, and then, with the sweep kernels' bounded wait, on a barrier whose
// phase nothing completes; both give up, and the second records
// kErrWaitTimeout for good.
__global__ void bounded_wait_selftest_kernel(Control* ctrl) {
  __shared__ __align__(8) unsigned long long bar;
  if (threadIdx.x == 0) {
    if (wait_count_bounded(&ctrl->slow_done, ~0u, 1000000, &ctrl->error)) return;
    if (!(atomicAnd(&ctrl->error, ~kErrWaitTimeout) & kErrWaitTimeout)) return;
    mbar_init(smem_u32(&bar), 1);
    fence_barrier_init();
    mbar_wait_bounded(smem_u32(&bar), 0, &ctrl->error);
  }
}

size_t round_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

// One launch for a small problem or batch: no staging, workspace or partials.  A
// cluster of 8 CTAs takes 128 queries; each CTA reads an eighth of the points
// into shared memory, and its 256 threads are 64 query pairs x 4 interleaved
// quarters of them.  The cluster agrees on the scale (largest |coordinate| of
// the points and its own queries) and joins its sums through distributed
// shared memory; CTA r finishes queries 16 r .. 16 r + 15 and answers its hits
// itself, a warp for two of them.  Sums are chunks of 16 points (S0 a tree, S1
// chains of 4 joined by a tree) folded by TwoSum, and no reciprocal is shared:
// errors against 64 bits are 0.5-0.95 of the sweep's, and a hit leaves its
// neighbour's sums alone.  Such calls are bound by latency: launches, the
// loads and three cluster barriers.  Against stage, sweep, combine and slow
// list, us: n = 1000, m = 1021: 5.8, from 13.8 (p = 2), 5.7 from 19.7 (3), 5.9
// from 28.9 (2.5); 16 x 16: 6.0 from 13.7; 4096 x 4096: 14 from 20, all of
// it hits 25.5 from 94.8; 10,000 x 1600: 19.7 from 24.7, hits 35 from 40.
// The limits: a flagged query's CTA reads all points, so past 12,288 of them
// hits cost more than in the sweep's list (16,384 x 1024: 52 against 44.5).
// Up to 100 M pairs the launch still wins (10,000 x 10,000: 37 against 42, all
// hits 85 against 279; 3000 x 30,000: 36.5 against 42); beyond, and past 256
// clusters, the sweep's larger tiles do more per load (12,000 x 12,000: level;
// 1000 x 60,000: 42 against 33.5; batches of 4e8 pairs and more 5-10% slower).
// A single problem at p = 2, whose sweep is the fastest, does not pay for a second
// wave of clusters (the GPU holds about 150) with few points (one launch / sweep: 16
// x 20,000 15.0 / 14.4 us, 16 x 32,000 20.9 / 16.1, 1000 x 28,000 21.3 / 20.0, 2000
// x 24,000 24.6 / 29.0; at p = 3, 16 x 32,000 21.4 / 29.2).  The line lies above
// where the times cross, for the host's time in the sweep's launches: 16 x
// 20,481, calls from Python back to back, 15.6 / 21.0.  Batches: 8 problems
// of 256 to 2048 points and queries 22.3 us, from 34.1 (on the device 12.4 from
// 22.8), 128 of 16 to 64 on the device 14.3 from 37.  Above p = 4 sums leave the
// fast form's range at ordinary distances, and the slow list spreads their FP64
// sums better.
constexpr int kSmallQueries = 128, kSmallCluster = 8, kSmallThreads = 256;
constexpr int64_t kSmallPoints = 12288, kSmallClusters = 256, kSmallPairs = int64_t(100) << 20;
constexpr int64_t kSmallClustersPow2 = 192, kSmallPointsPow2 = 1500;
constexpr double kSmallPower = 4.0;
constexpr int kSmallChunk = 16, kSmallSubs = kSmallThreads / (kSmallQueries / 2);
constexpr int kSmallStep = kSmallSubs * kSmallChunk;  // a CTA's points are padded to these
static_assert(kSmallThreads == kSlowThreads, "the CTA runs the slow path");

__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
}
// The address of CTA `rank`'s copy of this CTA's shared variable.
__device__ __forceinline__ uint32_t cluster_address(const void* p, int rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(p)), "r"(rank));
  return r;
}

// Instance::qtile_base counts clusters here.
template <int CAP, int MODE>
__global__ void __cluster_dims__(kSmallCluster, 1, 1) __launch_bounds__(kSmallThreads)
    small_kernel(const __grid_constant__ Table<CAP> t, float half_p, float neg_half_p, double p) {
  extern __shared__ float4 rec[];  // the CTA's points, padded
  __shared__ float4 part[kSmallSubs][kSmallQueries];
  __shared__ float4 mine[kSmallQueries];                 // this CTA's sums, read by the cluster
  __shared__ float4 piece[kSmallCluster][kSmallQueries / kSmallCluster];
  __shared__ float maxima[kSmallCluster];                // written by the cluster
  __shared__ float wmax[kSmallThreads / 32];
  __shared__ int flagged[kSmallQueries / kSmallCluster], hit[kSmallQueries / kSmallCluster];
  __shared__ float2 flagged_q[kSmallQueries / kSmallCluster];
  __shared__ int nflagged;
  pdl_trigger();
  cluster_arrive();  // a peer's shared memory may be written once the peer runs
  pdl_wait();
  const int tid = threadIdx.x, rank = blockIdx.x % kSmallCluster;
  const int cluster = blockIdx.x / kSmallCluster;
  const Instance& a = t.inst[CAP == 1 ? 0 : find_qtile(t, cluster)];
  const int q0 = (cluster - a.qtile_base) * kSmallQueries;
  const int first = static_cast<int>(int64_t(a.n) * rank / kSmallCluster);
  const int count = static_cast<int>(int64_t(a.n) * (rank + 1) / kSmallCluster) - first;

  // Points of the slice, queries of the pair, and the largest |coordinate|.
  float mx = 0.f;
  auto seen = [&](float v) {
    if (fabsf(v) <= FLT_MAX) mx = fmaxf(mx, fabsf(v));
  };
#pragma unroll 4
  for (int i = tid; i < count; i += kSmallThreads) {
    const float* row = a.data + 3 * int64_t(first + i);
    const float x = row[0], y = row[1];
    rec[i] = make_float4(x, y, row[2], 0.f);
    seen(x);
    seen(y);
  }
  const int pair = tid % (kSmallQueries / 2), sub = tid / (kSmallQueries / 2);
  const int ja = q0 + pair, jb = ja + kSmallQueries / 2;
  float qxa = 0.f, qya = 0.f, qxb = 0.f, qyb = 0.f;
  if (ja < a.m) {
    qxa = a.queries[2 * ja];
    qya = a.queries[2 * ja + 1];
    seen(qxa);
    seen(qya);
  }
  if (jb < a.m) {
    qxb = a.queries[2 * jb];
    qyb = a.queries[2 * jb + 1];
    seen(qxb);
    seen(qyb);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if ((tid & 31) == 0) wmax[tid >> 5] = mx;
  if (tid == 0) nflagged = 0;
  __syncthreads();
  cluster_wait();
  if (tid < kSmallCluster) {  // thread t tells CTA t
    mx = wmax[0];
    for (int w = 1; w < kSmallThreads / 32; ++w) mx = fmaxf(mx, wmax[w]);
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(cluster_address(&maxima[rank], tid)),
                 "f"(mx)
                 : "memory");
  }
  __syncwarp();
  cluster_arrive();
  cluster_wait();
  mx = maxima[0];
#pragma unroll
  for (int c = 1; c < kSmallCluster; ++c) mx = fmaxf(mx, maxima[c]);
  const float scale = scale_from_max(__float_as_uint(mx));
  const int padded = (count + kSmallStep - 1) / kSmallStep * kSmallStep;
  for (int i = tid; i < padded; i += kSmallThreads) {  // the rows this thread has written
    const float4 v = i < count ? rec[i] : make_float4(0.f, 0.f, 0.f, 0.f);
    rec[i] = i < count ? make_float4(v.x * scale, v.y * scale, v.z, 0.f)
                       : make_float4(INFINITY, INFINITY, 0.f, 0.f);  // weight 0
  }
  __syncthreads();

  const u64 QX = pk(qxa * scale, qxb * scale), QY = pk(qya * scale, qyb * scale);
  const u64 hp2 = pk(half_p, half_p), nhp2 = pk(neg_half_p, neg_half_p);
  u64 h0 = 0, l0 = 0, h1 = 0, l1 = 0;
#pragma unroll 1
  for (int c = 0; c < padded; c += kSmallStep) {
    u64 P0[4], P1[2], T1 = 0, C0 = 0, C1 = 0;
#pragma unroll
    for (int r = 0; r < kSmallChunk; ++r) {
      const float4 v = rec[c + r * kSmallSubs + sub];
      const u64 dx = sub2(QX, pk(v.x, v.x)), dy = sub2(QY, pk(v.y, v.y));
      const u64 d2 = fma2(dy, dy, mul2(dx, dx));
      const u64 w = weight_pair<MODE>(d2, false, hp2, nhp2), zz = pk(v.z, v.z);
      tree_push<4>(P0, w, r, C0);
      T1 = r % 4 == 0 ? mul2(w, zz) : fma2(w, zz, T1);
      if (r % 4 == 3) tree_push<2>(P1, T1, r / 4, C1);
    }
    two_sum_acc(h0, l0, C0);
    two_sum_acc(h1, l1, C1);
  }
  two_sum_renorm(h0, l0);
  two_sum_renorm(h1, l1);
  float ha, hb, la, lb, ga, gb, ka, kb;
  upk(h0, ha, hb);
  upk(l0, la, lb);
  upk(h1, ga, gb);
  upk(l1, ka, kb);
  part[sub][pair] = make_float4(ha, la, ga, ka);
  part[sub][pair + kSmallQueries / 2] = make_float4(hb, lb, gb, kb);
  __syncthreads();
  auto fold = [](float4& t, const float4 v) {
    two_sum_acc_f32(t.x, t.y, v.x);
    t.y += v.y;
    two_sum_acc_f32(t.z, t.w, v.z);
    t.w += v.w;
  };
  if (tid < kSmallQueries) {
    float4 sum = part[0][tid];
#pragma unroll
    for (int i = 1; i < kSmallSubs; ++i) fold(sum, part[i][tid]);
    mine[tid] = sum;
  }
  cluster_arrive();
  cluster_wait();
  constexpr int kOwn = kSmallQueries / kSmallCluster;  // queries this CTA finishes
  if (tid < kSmallQueries) {
    const int from = tid / kOwn, q = tid % kOwn;
    const uint32_t p = cluster_address(&mine[rank * kOwn + q], from);
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "r"(p)
                 : "memory");
    piece[from][q] = v;
  }
  cluster_arrive();  // this CTA has read its peers' sums
  __syncthreads();   // and its other warps' share of them is in place
  const int j = q0 + rank * kOwn + tid;
  if (tid < kOwn && j < a.m) {
    float4 sum = piece[0][tid];
#pragma unroll
    for (int c = 1; c < kSmallCluster; ++c) fold(sum, piece[c][tid]);
    const double s0 = double(sum.x) + double(sum.y), s1 = double(sum.z) + double(sum.w);
    if (!(s0 > kTinySumPerPoint * double(a.n)) || !isfinite(s0) || !isfinite(s1) ||
        (p >= 2.0 && s0 > kHugeSumPow2Up)) {
      const int f = atomicAdd(&nflagged, 1);
      flagged[f] = j;
      flagged_q[f] = make_float2(a.queries[2 * j], a.queries[2 * j + 1]);
    } else {
      a.out[j] = static_cast<float>(s1 / s0);
      if (a.s0_out) a.s0_out[j] = s0 * pow(double(scale), p);
      if (a.hit_out) a.hit_out[j] = kNoHit;
    }
  }
  __syncthreads();
  cluster_wait();  // and its peers have read its own: it may leave
  const int nf = nflagged;
  if (nf == 0) return;
  // A warp looks for the points under two of them: they stay in registers.
  const int f0 = tid >> 5, f1 = f0 + kSmallThreads / 32;
  static_assert(kOwn == 2 * (kSmallThreads / 32), "two flagged queries per warp");
  if (f0 < nf) {
    const float2 qa = flagged_q[f0], qb = f1 < nf ? flagged_q[f1] : make_float2(NAN, NAN);
    int ia = INT_MAX, ib = INT_MAX;
    for (int i0 = tid & 31; i0 < a.n; i0 += 32 * kSlowUnroll) {
      float x[kSlowUnroll], y[kSlowUnroll];
#pragma unroll
      for (int u = 0; u < kSlowUnroll; ++u) {
        const int i = min(i0 + 32 * u, a.n - 1);
        x[u] = a.data[3 * i];
        y[u] = a.data[3 * i + 1];
      }
#pragma unroll
      for (int u = 0; u < kSlowUnroll; ++u) {
        const int i = min(i0 + 32 * u, a.n - 1);
        if (x[u] == qa.x && y[u] == qa.y) ia = min(ia, i);
        if (x[u] == qb.x && y[u] == qb.y) ib = min(ib, i);
      }
    }
    ia = __reduce_min_sync(0xffffffffu, ia);
    ib = __reduce_min_sync(0xffffffffu, ib);
    if ((tid & 31) == 0) {
      hit[f0] = ia;
      if (f1 < nf) hit[f1] = ib;
    }
  }
  __syncthreads();
  for (int f = 0; f < nf; ++f) {  // uniform across the CTA
    const int jf = flagged[f];
    float* out = &a.out[jf];
    double* s0 = a.s0_out ? &a.s0_out[jf] : nullptr;
    int32_t* hj = a.hit_out ? &a.hit_out[jf] : nullptr;
    if (hit[f] != INT_MAX) {
      if (tid == 0) slow_write_hit(a.data, hit[f], out, s0, hj);
      continue;
    }
    SlowSums sums{INFINITY, 0.0, 0.0};  // of a query at infinity or NaN: a result of NaN
    if (isfinite(flagged_q[f].x) && isfinite(flagged_q[f].y))
      sums = slow_sums<float>(a.data, 0, a.n, flagged_q[f].x, flagged_q[f].y, p);
    if (tid == 0) slow_write_sums(sums, p, out, s0, hj);
  }
}

int64_t small_clusters(int64_t m) { return (m + kSmallQueries - 1) / kSmallQueries; }

bool small_problems(const F32Problem* probs, int count, double p, bool pow2) {
  int64_t clusters = 0, pairs = 0;
  for (int k = 0; k < count; ++k) {
    if (probs[k].n > kSmallPoints || probs[k].m > kSmallPairs) return false;
    clusters += small_clusters(probs[k].m);
    pairs += probs[k].n * probs[k].m;
  }
  if (pow2 && count == 1 && clusters > kSmallClustersPow2 && probs[0].n < kSmallPointsPow2)
    return false;
  return p <= kSmallPower && clusters <= kSmallClusters && pairs <= kSmallPairs;
}

template <int CAP>
cudaError_t launch_small(const F32Problem* probs, int count, double p, bool force_general,
                         cudaStream_t stream) {
  Table<CAP> t;
  t.count = count;
  t.pad = 0;
  int64_t clusters = 0, most = 0;
  for (int k = 0; k < count; ++k) {
    Instance& I = t.inst[k];
    I = Instance{};
    I.data = probs[k].data;
    I.queries = probs[k].queries;
    I.out = probs[k].out;
    I.s0_out = probs[k].s0_out;
    I.hit_out = probs[k].hit_out;
    I.n = static_cast<int32_t>(probs[k].n);
    I.m = static_cast<int32_t>(probs[k].m);
    I.qtile_base = static_cast<int32_t>(clusters);
    clusters += small_clusters(probs[k].m);
    most = std::max(most, probs[k].n);
  }
  auto kernel = force_general ? small_kernel<CAP, kPowGeneral>
                : p == 2.0    ? small_kernel<CAP, kPow2>
                : p == 1.0    ? small_kernel<CAP, kPow1>
                : p == 3.0    ? small_kernel<CAP, kPow3>
                : p == 4.0    ? small_kernel<CAP, kPow4>
                              : small_kernel<CAP, kPowGeneral>;
  const int64_t slice = (most + kSmallCluster - 1) / kSmallCluster;
  const size_t smem = size_t((slice + kSmallStep - 1) / kSmallStep * kSmallStep) * sizeof(float4);
  return launch_pdl(kernel, dim3(static_cast<unsigned>(clusters * kSmallCluster)),
                    dim3(kSmallThreads), smem, stream, t, static_cast<float>(0.5 * p),
                    static_cast<float>(-0.5 * p), p);
}

// Raises a kernel's dynamic shared memory limit to `bytes` (needed above
// 48 KB), once per kernel and device (one flag word per instantiation).
template <auto KERNEL>
cudaError_t allow_dynamic_smem(size_t bytes) {
  static unsigned long long done = 0;  // one bit per device ordinal < 64
  if (bytes <= 48u * 1024u) return cudaSuccess;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const unsigned long long bit = dev < 64 ? 1ull << dev : 0ull;
  if (bit && (__atomic_load_n(&done, __ATOMIC_ACQUIRE) & bit)) return cudaSuccess;
  e = cudaFuncSetAttribute(KERNEL, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           static_cast<int>(bytes));
  if (e == cudaSuccess && bit) __atomic_fetch_or(&done, bit, __ATOMIC_ACQ_REL);
  return e;
}

template <int CAP, int V, int MODE, int LAYOUT, bool FMA_LOG2 = false>
cudaError_t launch_impl(const F32Problem* probs, const BatchPlan& plan, double p,
                        unsigned char* ws, Control* ctrl, int sm_count, const SweepEvents* ev,
                        cudaStream_t stream) {
  Table<CAP> t;
  t.count = plan.count;
  t.pad = 0;
  unsigned char* tiles = ws;
  float4* partial = reinterpret_cast<float4*>(ws + plan.staged_bytes);
  float* scales = reinterpret_cast<float*>(ws + plan.staged_bytes + plan.partial_bytes);
  unsigned* maxbits = ctrl->maxbits;  // zero on entry: cleared by the previous call's combine
  int64_t longest = 1;
  for (int k = 0; k < plan.count; ++k) {
    Instance& I = t.inst[k];
    I.data = probs[k].data;
    I.queries = probs[k].queries;
    I.out = probs[k].out;
    I.s0_out = probs[k].s0_out;
    I.hit_out = probs[k].hit_out;
    I.tiles = tiles + size_t(plan.tile_offset[k]) * tile_bytes_of<LAYOUT>();
    I.unit_base = plan.unit_base[k];
    I.record_base = plan.tile_offset[k] * TB;
    I.n = static_cast<int32_t>(probs[k].n);
    I.m = static_cast<int32_t>(probs[k].m);
    I.data_tiles = static_cast<int32_t>(plan.data_tiles[k]);
    I.qtile_base = static_cast<int32_t>(plan.qtile_base[k]);
    longest = std::max<int64_t>(longest, std::max(probs[k].n, probs[k].m));
  }
  cudaError_t e;

  const unsigned gx = static_cast<unsigned>(std::min<int64_t>(1024, (longest + 255) / 256));
  if ((e = launch_pdl(range_kernel<CAP>, dim3(gx, plan.count), dim3(256), 0, stream, t,
                      maxbits, ctrl)) != cudaSuccess)
    return e;
  const int64_t records = plan.total_stage_tiles * TB;
  const unsigned sgrid = static_cast<unsigned>((records + 255) / 256);
  if ((e = launch_pdl(stage_kernel<CAP, MODE, LAYOUT>, dim3(sgrid), dim3(256), 0, stream, t,
                      records, static_cast<const unsigned*>(maxbits), scales)) != cudaSuccess)
    return e;

  SweepArgs a;
  a.units = plan.units;
  a.grid = plan.grid;
  a.half_p = static_cast<float>(0.5 * p);
  a.neg_half_p = -a.half_p;
  a.partial = partial;
  a.scales = scales;
  a.err = &ctrl->error;
  constexpr size_t smem = sweep_smem_of<V, LAYOUT>();
  if ((e = allow_dynamic_smem<sweep_kernel<MODE, CAP, V, LAYOUT, FMA_LOG2>>(smem)) != cudaSuccess)
    return e;
  if (ev && (e = cudaEventRecord(ev->start, stream)) != cudaSuccess) return e;
  constexpr int NT = Var<V>::NT, QT = qt_of<V>();
  // With profiling events the sweep is launched plainly, so that the events
  // around it bracket it alone.  So is one whose CTAs take between one place an SM
  // and three quarters of all: launched early, they are placed around the kernels
  // in flight, whose waiting CTAs hold places, and stay there, several on one SM
  // with others idle (early / plainly: p = 3, 100,003 x 100 55.4 / 38.0 us; p = 2.5,
  // 13,000 x 5000 73.8 / 48.8, 500 x 60,000 45.9 / 39.3).  A grid that fills every
  // place cannot be uneven, and loses the early start (12,000 x 12,000, p = 2.5:
  // 72 / 75).
  if (ev || (plan.grid > sm_count && 4 * plan.grid < 3 * sm_count * (512 / NT)))
    sweep_kernel<MODE, CAP, V, LAYOUT, FMA_LOG2><<<plan.grid, NT, smem, stream>>>(a, t);
  else if ((e = launch_pdl(sweep_kernel<MODE, CAP, V, LAYOUT, FMA_LOG2>, dim3(plan.grid),
                           dim3(NT), smem, stream, a, t)) != cudaSuccess)
    return e;
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if (ev && (e = cudaEventRecord(ev->stop, stream)) != cudaSuccess) return e;

  const int64_t slots = plan.total_query_tiles * QT;
  // Each listed query takes an item and a slice record; the grid's worth of
  // records more covers short lists cut into more slices.
  const int slow_grid = kSlowCtas * sm_count;
  SlowList slow;
  const size_t spare = size_t(slow_grid) * sizeof(SlowSums);
  slow.cap = static_cast<unsigned>(std::min<size_t>(
      plan.staged_bytes > spare
          ? (plan.staged_bytes - spare) / (sizeof(SlowItem) + sizeof(SlowSums))
          : 0,
      size_t(INT_MAX)));
  slow.item = reinterpret_cast<SlowItem*>(ws);
  slow.part = reinterpret_cast<SlowSums*>(ws + size_t(slow.cap) * sizeof(SlowItem));
  const int64_t pieces = plan.partial_slots / plan.total_query_tiles;  // of a query
  const int lanes = pieces > kCombineManyPieces ? 32 : 8;
  auto combine = lanes == 32 ? combine_kernel<CAP, QT, 32> : combine_kernel<CAP, QT, 8>;
  const int per_cta = kCombineThreads / lanes;
  if ((e = launch_pdl(combine, dim3(static_cast<unsigned>((slots + per_cta - 1) / per_cta)),
                      dim3(kCombineThreads), 0, stream, t, static_cast<const float4*>(partial),
                      slots, plan.units, plan.grid, static_cast<const float*>(scales), p, ctrl,
                      slow)) != cudaSuccess)
    return e;
  int64_t most_points = 0;
  for (int k = 0; k < plan.count; ++k) most_points = std::max(most_points, probs[k].n);
  if (most_points <= kSlowInlinePoints || slow.cap == 0) return cudaSuccess;  // nothing is listed
  return launch_pdl(slow_kernel<CAP>, dim3(slow_grid), dim3(kSlowThreads), 0, stream, t, ctrl, slow, p);
}

}  // namespace

int sweep_variant_queries_per_cta(int variant) {
  switch (variant) {
    case 1: return qt_of<1>();
    case 2: return qt_of<2>();
    case 3: return qt_of<3>();
    case 4: return qt_of<4>();
    case 5: return qt_of<5>();
    case 6: return qt_of<6>();
    case 7: return qt_of<7>();
    default: return qt_of<0>();
  }
}

int sweep_variant_points_per_unit(int variant) {
  switch (variant) {
    case 5: return Var<5>::TBV;
    case 6: return Var<6>::TBV;
    default: return TB;
  }
}

// Predicted clocks of a sweep's longest CTA: its units times a unit's share
// of an SM.  An SM with w of its 16 warps sweeps 1 - (1 - w/16)^2 of its full
// rate, `rate` pairs a clock.
namespace {
double sweep_clocks(const F32Problem* probs, int count, int variant, int threads, double rate,
                    int sm_count) {
  const int64_t qt = sweep_variant_queries_per_cta(variant);
  const int64_t tb = sweep_variant_points_per_unit(variant);
  int64_t units = 0;
  for (int k = 0; k < count; ++k)
    units += (probs[k].m + qt - 1) / qt * ((probs[k].n + tb - 1) / tb);
  const int64_t per_sm = 512 / threads, resident = per_sm * sm_count;
  const int64_t grid = std::min(units, resident);
  const int64_t longest = (units + grid - 1) / grid;
  const double ctas = double((grid + sm_count - 1) / sm_count);
  const double idle = 1.0 - ctas / double(per_sm);
  return double(longest) * double(qt * tb) * ctas / (rate * (1.0 - idle * idle));
}
}  // namespace

// The fixed rule of thumb (large tiles, or 64-point units for small p = 2
// problems) unless one of the 512-query variants is predicted to be 10%
// faster: those pad small or uneven query sets less and fill the GPU with
// smaller pieces, at 80% (64-point units) to 93% of the large tiles' rate.
// Measured, rule of thumb / 512-query tiles, whole call: p = 2: n = 20,000,
// m = 1000 35.4 / 30.7 us; n = 70,000, m = 3000 88.7 / 78.6; n = m = 20,000
// 113.5 / 126.4 (not taken).  p = 3.5: n = m = 4000 70.7 / 38.0; 64 problems of
// 256 to 8192 points 320 / 275; n = m = 40,000 648 / 687 (not taken).  p = 1, 3
// and 4 go by the general form's rates: their sweeps are about 1.4 times as fast
// with every tile, and only the rates' ratios matter here.
int default_sweep_variant(const F32Problem* probs, int count, bool general_form, int sm_count) {
  const int64_t q4 = qt_of<4>(), q0 = qt_of<0>();
  double pad4 = 0, pad0 = 0, units0 = 0;
  for (int k = 0; k < count; ++k) {
    pad4 += double((probs[k].m + q4 - 1) / q4 * q4);
    pad0 += double((probs[k].m + q0 - 1) / q0 * q0);
    units0 += double((probs[k].m + q0 - 1) / q0) * double((probs[k].n + TB - 1) / TB);
  }
  const int large = !general_form && units0 < 4.0 * sm_count * 2 ? 5 : pad4 <= 1.01 * pad0 ? 4 : 0;
  // Pairs per SM and clock of a full GPU.
  const double rate[kNumAllVariants] = {general_form ? 8.5 : 15.1, 0, 0, 0,
                                        general_form ? 8.65 : 15.35, 14.8, 12.2,
                                        general_form ? 7.6 : 14.2};
  int best = large;
  double t = 0.9 * sweep_clocks(probs, count, large, large == 4 ? 512 : 256, rate[large], sm_count);
  for (int v : {kSmallTileFine, kSmallTile}) {
    if (general_form && v == kSmallTileFine) continue;
    const double tv = sweep_clocks(probs, count, v, 64, rate[v], sm_count);
    if (tv < t) {
      best = v;
      t = tv;
    }
  }
  return best;
}

int resolve_sweep_variant(int variant, bool general_form) {
  if (variant < 0 || variant >= kNumAllVariants) return 0;
  // Sub-tile work units need the aligned-AoS staging of the p = 2 form.
  if (general_form && sweep_variant_points_per_unit(variant) != TB) return 0;
  return variant;
}

void plan_batch_f32(const F32Problem* probs, int count, int sm_count, int ctas_per_sm,
                    int variant, BatchPlan* bp) {
  const int QT = sweep_variant_queries_per_cta(variant);
  const int TBU = sweep_variant_points_per_unit(variant);
  bp->variant = variant;
  bp->count = count;
  bp->data_tiles.assign(count, 0);
  bp->query_tiles.assign(count, 0);
  bp->unit_base.assign(count, 0);
  bp->qtile_base.assign(count, 0);
  bp->tile_offset.assign(count, 0);
  int64_t units = 0, qtiles = 0, tiles = 0, queries = 0;
  for (int k = 0; k < count; ++k) {
    const int64_t dt = (probs[k].n + TBU - 1) / TBU;  // work units along the data
    const int64_t st = (probs[k].n + TB - 1) / TB;    // staging tiles
    const int64_t qt = (probs[k].m + QT - 1) / QT;
    bp->data_tiles[k] = dt;
    bp->query_tiles[k] = qt;
    bp->unit_base[k] = units;
    bp->qtile_base[k] = qtiles;
    bp->tile_offset[k] = tiles;
    units += dt * qt;
    qtiles += qt;
    tiles += st;
    queries += probs[k].m;
  }
  bp->units = units;
  bp->total_query_tiles = qtiles;
  bp->total_stage_tiles = tiles;
  const int64_t resident = int64_t(sm_count) * (ctas_per_sm > 0 ? ctas_per_sm : 1);
  bp->grid = static_cast<int>(std::max<int64_t>(1, std::min(units, resident)));
  bp->partial_slots = qtiles + bp->grid - 1;
  bp->staged_bytes = round_up(size_t(tiles) * kTileBytes, 256);  // the widest layout
  bp->partial_bytes = round_up(size_t(bp->partial_slots) * QT * sizeof(float4), 256);
  bp->list_bytes = 0;  // flagged queries are listed in the combine CTA's shared memory
  bp->scale_bytes = round_up(size_t(count) * sizeof(float), 256);
  bp->workspace_bytes = bp->staged_bytes + bp->partial_bytes + bp->list_bytes + bp->scale_bytes;
}

cudaError_t launch_batch_f32(const F32Problem* probs, const BatchPlan& plan, double p,
                             void* workspace, Control* ctrl, int sm_count,
                             const SweepEvents* ev, cudaStream_t stream) {
  unsigned char* ws = static_cast<unsigned char*>(workspace);
  if (plan.count < 1 || plan.count > kBatchCap) return cudaErrorInvalidValue;
  const bool one = plan.count == 1;
  const bool pow2 = (p == 2.0) && !plan.force_general;
  if (plan.small_ok && !ev && small_problems(probs, plan.count, p, pow2))
    return one ? launch_small<1>(probs, 1, p, plan.force_general, stream)
               : launch_small<kBatchCap>(probs, plan.count, p, plan.force_general, stream);
  // Default staging layout per weight form (measured fastest on GB300): the
  // aligned AoS record at p = 2, whose one shared load per point leaves the
  // special-function queue to the reciprocals; duplicated pair records for
  // general p, which need no register moves.  The other layouts are built
  // for the single-problem sweep of variant 0 (the layout ablation).
  const int layout = plan.layout >= 0 ? plan.layout : (pow2 ? 1 : 0);
  if (one && plan.variant == 4 && !pow2 && plan.fma_log2)
    return launch_impl<1, 4, kPowGeneral, 0, true>(probs, plan, p, ws, ctrl, sm_count, ev, stream);
  // p = 1, 3, 4 as powers of one reciprocal (square root): 1 MUFU at 16 per SM
  // and clock against lg2 at 16 and ex2 at 32.  n = m = 51,200, p = 1 / 3 / 4:
  // 641 / 700 / 651 us, against 1007 us through log2 and exp2, with errors
  // against 64 bits at or below that form's (it keeps that form's 32-point
  // chunks: the 64-point ones of p = 2 were 3% faster and 5% less exact).
  // Aligned records beat duplicated pairs by 1-2% here as at p = 2.  Variants
  // 1, 2, 3 and 5 and a forced layout, made to study the general form, keep it.
  if (!plan.force_general && plan.layout < 0 && !plan.fma_log2 &&
      (plan.variant == 0 || plan.variant == 4 || plan.variant == 7)) {
#define IDW_LAUNCH_POWER(M)                                                                     \
  if (plan.variant == 0)                                                                        \
    return one ? launch_impl<1, 0, M, 1>(probs, plan, p, ws, ctrl, sm_count, ev, stream)        \
               : launch_impl<kBatchCap, 0, M, 1>(probs, plan, p, ws, ctrl, sm_count, ev, stream); \
  if (plan.variant == 7)                                                                        \
    return one ? launch_impl<1, 7, M, 1>(probs, plan, p, ws, ctrl, sm_count, ev, stream)        \
               : launch_impl<kBatchCap, 7, M, 1>(probs, plan, p, ws, ctrl, sm_count, ev, stream); \
  return one ? launch_impl<1, 4, M, 1>(probs, plan, p, ws, ctrl, sm_count, ev, stream)          \
             : launch_impl<kBatchCap, 4, M, 1>(probs, plan, p, ws, ctrl, sm_count, ev, stream)
    if (p == 1.0) { IDW_LAUNCH_POWER(kPow1); }
    if (p == 3.0) { IDW_LAUNCH_POWER(kPow3); }
    if (p == 4.0) { IDW_LAUNCH_POWER(kPow4); }
#undef IDW_LAUNCH_POWER
  }
  if (one && plan.variant == 0) {
    if (pow2 && layout == 0) return launch_impl<1, 0, kPow2, 0>(probs, plan, p, ws, ctrl, sm_count, ev, stream);
    if (pow2 && layout == 2) return launch_impl<1, 0, kPow2, 2>(probs, plan, p, ws, ctrl, sm_count, ev, stream);
    if (!pow2 && layout == 1) return launch_impl<1, 0, kPowGeneral, 1>(probs, plan, p, ws, ctrl, sm_count, ev, stream);
    if (!pow2 && layout == 2) return launch_impl<1, 0, kPowGeneral, 2>(probs, plan, p, ws, ctrl, sm_count, ev, stream);
  }
#define IDW_LAUNCH(V)                                                                        \
  if (pow2)                                                                                  \
    return one ? launch_impl<1, V, kPow2, 1>(probs, plan, p, ws, ctrl, sm_count, ev, stream) \
               : launch_impl<kBatchCap, V, kPow2, 1>(probs, plan, p, ws, ctrl, sm_count, ev,  \
                                                      stream);                               \
  return one ? launch_impl<1, V, kPowGeneral, 0>(probs, plan, p, ws, ctrl, sm_count, ev, stream) \
             : launch_impl<kBatchCap, V, kPowGeneral, 0>(probs, plan, p, ws, ctrl, sm_count, ev, \
                                                         stream)
  switch (plan.variant) {
    case 1: IDW_LAUNCH(1);
    case 2: IDW_LAUNCH(2);
    case 3: IDW_LAUNCH(3);
    case 4: IDW_LAUNCH(4);
    case 5:
      if (pow2)
        return one ? launch_impl<1, 5, kPow2, 1>(probs, plan, p, ws, ctrl, sm_count, ev, stream)
                   : launch_impl<kBatchCap, 5, kPow2, 1>(probs, plan, p, ws, ctrl, sm_count, ev,
                                                         stream);
      return cudaErrorInvalidValue;  // resolve_sweep_variant maps it away for general p
    case 6:
      if (pow2)
        return one ? launch_impl<1, 6, kPow2, 1>(probs, plan, p, ws, ctrl, sm_count, ev, stream)
                   : launch_impl<kBatchCap, 6, kPow2, 1>(probs, plan, p, ws, ctrl, sm_count, ev,
                                                         stream);
      return cudaErrorInvalidValue;
    case 7: IDW_LAUNCH(7);
    default: IDW_LAUNCH(0);
  }
#undef IDW_LAUNCH
}

namespace {
template <int V>
int occupancy_variant(bool general_p) {
  int blocks = 0;
  if constexpr (Var<V>::TBV == TB) {
    if (general_p) {
      constexpr size_t smem = sweep_smem_of<V, 0>();
      allow_dynamic_smem<sweep_kernel<kPowGeneral, kBatchCap, V, 0>>(smem);
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(
          &blocks, sweep_kernel<kPowGeneral, kBatchCap, V, 0>, Var<V>::NT, smem);
      return blocks > 0 ? blocks : 1;
    }
  }
  constexpr size_t smem = sweep_smem_of<V, 1>();
  allow_dynamic_smem<sweep_kernel<kPow2, kBatchCap, V, 1>>(smem);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, sweep_kernel<kPow2, kBatchCap, V, 1>,
                                                Var<V>::NT, smem);
  return blocks > 0 ? blocks : 1;
}
}  // namespace

int occupancy_forward_f32(bool general_p, int variant) {
  switch (variant) {
    case 1: return occupancy_variant<1>(general_p);
    case 2: return occupancy_variant<2>(general_p);
    case 3: return occupancy_variant<3>(general_p);
    case 4: return occupancy_variant<4>(general_p);
    case 5: return general_p ? occupancy_variant<0>(true) : occupancy_variant<5>(false);
    case 6: return general_p ? occupancy_variant<0>(true) : occupancy_variant<6>(false);
    case 7: return occupancy_variant<7>(general_p);
    default: return occupancy_variant<0>(general_p);
  }
}

cudaError_t launch_bounded_wait_selftest(Control* ctrl, cudaStream_t stream) {
  bounded_wait_selftest_kernel<<<1, 32, 0, stream>>>(ctrl);
  return cudaGetLastError();
}

}  // namespace idw
