// Adjoint of global Shepard IDW (Sec. 2.1, Eq. 1) for L = sum_j g_j Z(q_j).
//
// With w_ij = (d_ij^2)^(-p/2), S0_j = sum_i w_ij and Z_j = S1_j / S0_j
// (chain rule on Eq. 1; the paper gives no gradient):
//   dL/dq_j = -g_j (p / S0_j) sum_i (z_i - Z_j) w_ij (q_j - x_i) / d_ij^2
//   dL/dp   = -sum_j g_j / (2 S0_j) sum_i (z_i - Z_j) w_ij ln d_ij^2
//   dL/dz_i =  sum_j g_j w_ij / S0_j
//   dL/dx_i =  sum_j g_j (p / S0_j) (z_i - Z_j) w_ij (q_j - x_i) / d_ij^2
//
// One all-pairs sweep for both sides (p >= 1), or two when one side alone is
// wanted, recompute the weights tile by tile (nothing of size n x m is
// stored):
//   * the query sweep holds queries in registers and streams the staged data
//     tiles of the forward pass (three sums per query);
//   * the data sweep is its transpose: data points in registers, staged
//     query records (q, g/S0, Z) streamed (three sums per data point);
//   * the fused sweep does both at once (see fused_adj_kernel).
// Both use the forward pass's machinery: packed fp32x2 arithmetic, 1-D bulk
// TMA tiles, chunked sums folded by TwoSum, stream-K pieces summed in FP64.
// Queries that the forward pass routed to its slow path (an exact hit, or
// FP32 range exceeded) are padded out of both sweeps and handled in FP64.
#include <algorithm>
#include <cfloat>
#include <cmath>

#include "idw_device.cuh"
#include "idw_f32_common.cuh"
#include "idw_internal.h"
#include "idw_slowpath.cuh"

namespace idw {
namespace {

constexpr int NTA = 512;             // threads per CTA (one CTA per SM keeps 16 warps in step)
constexpr int KPA = 2;               // register pairs per thread
constexpr int RT = NTA * 2 * KPA;    // register-side points per CTA tile (2048)
constexpr int CHA = 64;              // chunk length between TwoSum folds
constexpr int STA = 3;               // ring stages
constexpr int TQ = 256;              // query records per streamed query tile
constexpr uint32_t kQTileBytes = TQ * 16;  // (qx, qy, c, Z): one shared load per query
static_assert(kTB32 % CHA == 0 && TQ % CHA == 0, "chunks tile the streamed tiles");

struct AdjArgs {
  int64_t units;
  int grid;
  int64_t stream_tiles;  // streamed tiles per register tile
  const unsigned char* tiles;
  int64_t nreg;          // register-side points (m for the query sweep, n for the data sweep)
  int64_t nstream;       // streamed points (n, or m)
  const float* reg_xy;   // register-side coordinates
  int reg_stride;        // floats between consecutive points (2 queries, 3 data)
  const float* reg_val;  // Z_j (query sweep, stride 1) or z_i (data sweep, stride 3)
  int val_stride;
  const float* scales;
  float neg_half_p, neg_half_p1;  // -p/2, -(p/2 + 1)
  float2* partial;       // slots x 3 x RT (hi, lo)
  unsigned* err;
};

// w = (d^2)^(-p/2) and v = w / d^2 on both lanes; L = log2 d^2 when asked.
// No clamp on log2: the query sweep masks its padding records, and the data
// sweep's padding queries sit at a finite far point (weights underflow to 0).
template <bool POW2, bool WANT_L>
__device__ __forceinline__ void weights(u64 d2, u64 nhp2, u64 nhp12, u64& w, u64& v, u64& L) {
  float da, db;
  upk(d2, da, db);
  if (POW2) {
    w = pk(rcp_approx(da), rcp_approx(db));
    v = mul2(w, w);
    if (WANT_L) L = pk(lg2_approx(da), lg2_approx(db));
  } else {
    L = pk(lg2_approx(da), lg2_approx(db));
    float ta, tb, ua, ub;
    upk(mul2(L, nhp2), ta, tb);   // -(p/2) L
    upk(mul2(L, nhp12), ua, ub);  // -(p/2 + 1) L
    w = pk(ex2_approx(ta), ex2_approx(tb));
    v = pk(ex2_approx(ua), ex2_approx(ub));
  }
}

__device__ __forceinline__ void write_piece(float2* P, int comp, int idx, u64 hi, u64 lo) {
  float ha, hb, la, lb;
  upk(hi, ha, hb);
  upk(lo, la, lb);
  P[comp * RT + idx] = make_float2(ha, la);
  P[comp * RT + idx + NTA] = make_float2(hb, lb);
}

// One staged data tile for the query sweep.  MASKED (the last tile of a
// sweep only) skips the padding records; full tiles run straight-line code.
template <bool POW2, bool NEED_P, bool MASKED>
__device__ __forceinline__ void query_tile(const unsigned char* st, int valid, u64 NHP2, u64 NHP12,
                                           u64 SHIFT, const u64* QX, const u64* QY,
                                           const u64* ZQ, u64* XH, u64* XL, u64* YH, u64* YL,
                                           u64* PH, u64* PL) {
  const ulonglong2* XY = reinterpret_cast<const ulonglong2*>(st);
  const u64* ZZ = reinterpret_cast<const u64*>(st + kTB32 * 16);
#pragma unroll 1
  for (int c = 0; c < valid; c += CHA) {
    u64 CX[KPA], CY[KPA], CP[KPA];
#pragma unroll
    for (int k = 0; k < KPA; ++k) CX[k] = CY[k] = CP[k] = 0ull;
#pragma unroll
    for (int r = 0; r < CHA; ++r) {
      if (!MASKED || c + r < valid) {  // uniform across the CTA
        const ulonglong2 xy = XY[c + r];
        const u64 zz = ZZ[c + r];
#pragma unroll
        for (int k = 0; k < KPA; ++k) {
          const u64 dx = sub2f(QX[k], xy.x);
          const u64 dy = sub2f(QY[k], xy.y);
          const u64 d2 = fma2f(dy, dy, mul2f(dx, dx));
          u64 w, v, L = 0ull;
          weights<POW2, NEED_P>(d2, NHP2, NHP12, w, v, L);
          const u64 e = sub2(zz, ZQ[k]);  // z_i - Z_j
          const u64 ev = mul2(e, v);
          CX[k] = fma2(ev, dx, CX[k]);
          CY[k] = fma2(ev, dy, CY[k]);
          if (NEED_P) CP[k] = fma2(mul2(e, w), add2(L, SHIFT), CP[k]);
        }
      }
    }
#pragma unroll
    for (int k = 0; k < KPA; ++k) {
      two_sum_acc(XH[k], XL[k], CX[k]);
      two_sum_acc(YH[k], YL[k], CY[k]);
      if (NEED_P) two_sum_acc(PH[k], PL[k], CP[k]);
    }
  }
}

// Query sweep: sums over data points of (z - Z) w (q - x) / d^2 (x and y)
// and of (z - Z) w log2 d^2, per query, in scaled coordinates.
template <bool POW2, bool NEED_P>
__global__ void __launch_bounds__(NTA, 1) query_adj_kernel(const AdjArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) unsigned long long bars[STA];
  const int tid = threadIdx.x;
  const int64_t g = blockIdx.x;
  const int64_t u0 = unit_begin(g, a.units, a.grid);
  const int64_t total = unit_begin(g + 1, a.units, a.grid) - u0;
  if (total <= 0) return;
  auto src = [&](int64_t local) {
    return static_cast<const void*>(a.tiles + ((u0 + local) % a.stream_tiles) * kTileBytes32);
  };
  TileRing<STA, decltype(src)> ring{smem, bars, kTileBytes32, a.err, total, src, 0};
  ring.start();

  const float s = a.scales[0];
  const u64 NHP2 = pk(a.neg_half_p, a.neg_half_p), NHP12 = pk(a.neg_half_p1, a.neg_half_p1);
  // log2 of the unscaled d^2 = log2 of the scaled one - 2 log2 s (exact).
  const float shift = -2.f * static_cast<float>(ilogbf(s));
  const u64 SHIFT = pk(shift, shift);
  const int64_t last_valid = a.nstream - (a.stream_tiles - 1) * kTB32;  // records in last tile

  int64_t i = 0;
  bool aborted = false;
  while (i < total) {
    const int64_t rt = (u0 + i) / a.stream_tiles;
    const int64_t seg_end = min(total, (rt + 1) * a.stream_tiles - u0);
    u64 QX[KPA], QY[KPA], ZQ[KPA], XH[KPA], XL[KPA], YH[KPA], YL[KPA], PH[KPA], PL[KPA];
#pragma unroll
    for (int k = 0; k < KPA; ++k) {
      const int64_t ja = rt * RT + (2 * k) * NTA + tid, jb = ja + NTA;
      const bool va = ja < a.nreg, vb = jb < a.nreg;
      QX[k] = pk(va ? a.reg_xy[a.reg_stride * ja] * s : 0.f,
                 vb ? a.reg_xy[a.reg_stride * jb] * s : 0.f);
      QY[k] = pk(va ? a.reg_xy[a.reg_stride * ja + 1] * s : 0.f,
                 vb ? a.reg_xy[a.reg_stride * jb + 1] * s : 0.f);
      ZQ[k] = pk(va ? a.reg_val[a.val_stride * ja] : 0.f, vb ? a.reg_val[a.val_stride * jb] : 0.f);
      XH[k] = XL[k] = YH[k] = YL[k] = PH[k] = PL[k] = 0ull;
    }
    for (; i < seg_end; ++i) {
      bool ok;
      const unsigned char* st = ring.wait(i, ok);
      if (ok) {
        const bool last = ((u0 + i) % a.stream_tiles) == a.stream_tiles - 1;
        if (last && last_valid < kTB32)
          query_tile<POW2, NEED_P, true>(st, static_cast<int>(last_valid), NHP2, NHP12, SHIFT, QX,
                                         QY, ZQ, XH, XL, YH, YL, PH, PL);
        else
          query_tile<POW2, NEED_P, false>(st, kTB32, NHP2, NHP12, SHIFT, QX, QY, ZQ, XH, XL, YH,
                                          YL, PH, PL);
      }
      if (!ring.release(ok)) {
        aborted = true;
        break;
      }
    }
    if (aborted) break;
    float2* P = a.partial + (rt + g) * 3 * RT;
#pragma unroll
    for (int k = 0; k < KPA; ++k) {
      write_piece(P, 0, 2 * k * NTA + tid, XH[k], XL[k]);
      write_piece(P, 1, 2 * k * NTA + tid, YH[k], YL[k]);
      write_piece(P, 2, 2 * k * NTA + tid, PH[k], PL[k]);
    }
  }
  if (aborted) ring.drain(i);
}

// Data sweep: sums over queries of c w, c (z - Z) w (q - x) / d^2 (x and y)
// per data point, with c_j = g_j / S0_j (scaled), in scaled coordinates.
// Padding and excluded queries carry c = 0 at a finite far point.
template <bool POW2>
__global__ void __launch_bounds__(NTA, 1) data_adj_kernel(const AdjArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) unsigned long long bars[STA];
  const int tid = threadIdx.x;
  const int64_t g = blockIdx.x;
  const int64_t u0 = unit_begin(g, a.units, a.grid);
  const int64_t total = unit_begin(g + 1, a.units, a.grid) - u0;
  if (total <= 0) return;
  auto src = [&](int64_t local) {
    return static_cast<const void*>(a.tiles + ((u0 + local) % a.stream_tiles) * kQTileBytes);
  };
  TileRing<STA, decltype(src)> ring{smem, bars, kQTileBytes, a.err, total, src, 0};
  ring.start();
  const float s = a.scales[0];
  const u64 NHP2 = pk(a.neg_half_p, a.neg_half_p), NHP12 = pk(a.neg_half_p1, a.neg_half_p1);

  int64_t i = 0;
  bool aborted = false;
  while (i < total) {
    const int64_t rt = (u0 + i) / a.stream_tiles;
    const int64_t seg_end = min(total, (rt + 1) * a.stream_tiles - u0);
    u64 XD[KPA], YD[KPA], ZD[KPA], GZH[KPA], GZL[KPA], GXH[KPA], GXL[KPA], GYH[KPA], GYL[KPA];
#pragma unroll
    for (int k = 0; k < KPA; ++k) {
      const int64_t ia = rt * RT + (2 * k) * NTA + tid, ib = ia + NTA;
      const bool va = ia < a.nreg, vb = ib < a.nreg;
      XD[k] = pk(va ? a.reg_xy[a.reg_stride * ia] * s : 0.f,
                 vb ? a.reg_xy[a.reg_stride * ib] * s : 0.f);
      YD[k] = pk(va ? a.reg_xy[a.reg_stride * ia + 1] * s : 0.f,
                 vb ? a.reg_xy[a.reg_stride * ib + 1] * s : 0.f);
      ZD[k] = pk(va ? a.reg_val[a.val_stride * ia] : 0.f, vb ? a.reg_val[a.val_stride * ib] : 0.f);
      GZH[k] = GZL[k] = GXH[k] = GXL[k] = GYH[k] = GYL[k] = 0ull;
    }
    for (; i < seg_end; ++i) {
      bool ok;
      const unsigned char* st = ring.wait(i, ok);
      if (ok) {
        const float4* QR = reinterpret_cast<const float4*>(st);  // (qx, qy, c, Z)
#pragma unroll 1
        for (int c = 0; c < TQ; c += CHA) {
          u64 CGZ[KPA], CGX[KPA], CGY[KPA];
#pragma unroll
          for (int k = 0; k < KPA; ++k) CGZ[k] = CGX[k] = CGY[k] = 0ull;
#pragma unroll
          for (int r = 0; r < CHA; ++r) {
            const float4 qr = QR[c + r];
            const u64 qxx = pk(qr.x, qr.x), qyy = pk(qr.y, qr.y);
            const u64 cc = pk(qr.z, qr.z), zq = pk(qr.w, qr.w);
#pragma unroll
            for (int k = 0; k < KPA; ++k) {
              const u64 dx = sub2f(qxx, XD[k]);  // q_j - x_i
              const u64 dy = sub2f(qyy, YD[k]);
              const u64 d2 = fma2f(dy, dy, mul2f(dx, dx));
              u64 w, v, L;
              weights<POW2, false>(d2, NHP2, NHP12, w, v, L);
              const u64 cw = mul2(cc, w);
              CGZ[k] = add2(CGZ[k], cw);
              const u64 b = mul2(mul2(cc, sub2(ZD[k], zq)), v);  // c (z_i - Z_j) w / d^2
              CGX[k] = fma2(b, dx, CGX[k]);
              CGY[k] = fma2(b, dy, CGY[k]);
            }
          }
#pragma unroll
          for (int k = 0; k < KPA; ++k) {
            two_sum_acc(GZH[k], GZL[k], CGZ[k]);
            two_sum_acc(GXH[k], GXL[k], CGX[k]);
            two_sum_acc(GYH[k], GYL[k], CGY[k]);
          }
        }
      }
      if (!ring.release(ok)) {
        aborted = true;
        break;
      }
    }
    if (aborted) break;
    float2* P = a.partial + (rt + g) * 3 * RT;
#pragma unroll
    for (int k = 0; k < KPA; ++k) {
      write_piece(P, 0, 2 * k * NTA + tid, GZH[k], GZL[k]);
      write_piece(P, 1, 2 * k * NTA + tid, GXH[k], GXL[k]);
      write_piece(P, 2, 2 * k * NTA + tid, GYH[k], GYL[k]);
    }
  }
  if (aborted) ring.drain(i);
}

// Both sides in one sweep: every pair's weights are computed once.
//
// Each lane holds 8 queries (4 register pairs) and the warps of a CTA hold
// different queries, so a query's three sums stay with its thread (chunks of
// 64 points folded by TwoSum into (hi, lo) slots in shared memory), while a
// data point's three sums have to be added over the 32 lanes and the CTA's
// warps.  A warp takes 8 points at a time, lane l taking them in the order
// i ^ (l & 7) (one 128-byte read of 8 records, no bank conflict).  Then the
// exchange of step 4, 2, 1 adds register i of a lane to register i + 4 (2, 1)
// of its partner, which is the same point, with no selects, and leaves lane l
// with point l & 7; two more steps add the four groups of 8 lanes: 27 shuffles
// for 8 points x 256 queries.  The warps' sums meet in shared memory and
// leave as one FP32 partial per point and query tile: 8 products in a lane
// and 9 tree levels behind it, fewer roundings than the 64-point chains of
// the data sweep.  Partials of a panel of query tiles (at most kPanelBytes)
// are added in FP64 in tile order.
//
// Bound by the FMA pipe: 17 lane operations a pair (general power, dL/dp)
// against 12 + 12 and twice the special functions for the two sweeps.  The
// query pairs and the data records are staged as the 64-bit register pairs
// that the packed instructions take: packing them in the loop cost 10 moves a
// pair of pairs on top of 29 instructions.  n = m = 65,536, p = 2.5, all
// gradients: 3954 us with two sweeps, 2871 us; p = 2 without dL/dp 2748 and
// 2107 us; n = m = 1000 112 and 66 us.
constexpr int KPF = 4;  // register pairs per thread
constexpr size_t kPanelBytes = size_t(256) << 20;
template <int NT> __host__ __device__ constexpr int fused_queries() { return NT * 2 * KPF; }
// Points per work unit of the variant with `threads` per CTA.
constexpr int fused_points(int threads) { return threads == 128 ? 64 : 128; }

template <int NT, int TBU>
struct FusedSmem {
  static constexpr size_t ring = size_t(STA) * TBU * 24;
  static constexpr size_t slots = size_t(3) * KPF * NT * sizeof(ulonglong2);
  static constexpr size_t red = size_t(2) * (NT / 32) * 3 * TBU * sizeof(float);
  static constexpr size_t bytes = ring + slots + red;
};

struct FusedArgs {
  int64_t units;         // query tiles of the panel x data tiles
  int grid;
  int64_t data_tiles;    // work units along the data (TBU points each)
  int64_t n;
  const unsigned char* tiles;  // staged data records (x, y, z, pad)
  const ulonglong2* queries;   // pair records from the panel's first query tile on
  const float* scales;
  float neg_half_p, neg_half_p1;
  float2* partial;       // query side: slots x 3 x queries (hi, lo)
  float* dpart;          // data side: query tile x 3 x npad
  int64_t npad;
  unsigned* err;
};

template <int NT, int TBU, bool POW2, bool NEED_P>
__global__ void __launch_bounds__(NT, 512 / NT) fused_adj_kernel(const FusedArgs a) {
  using S = FusedSmem<NT, TBU>;
  constexpr int RTF = fused_queries<NT>(), WARPS = NT / 32;
  static_assert(TBU % CHA == 0, "chunks tile a unit");
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) unsigned long long bars[STA];
  const int tid = threadIdx.x, lane = tid & 31, l7 = lane & 7, warp = tid >> 5;
  const int64_t g = blockIdx.x;
  const int64_t u0 = unit_begin(g, a.units, a.grid);
  const int64_t total = unit_begin(g + 1, a.units, a.grid) - u0;
  if (total <= 0) return;
  auto src = [&](int64_t local) {
    return static_cast<const void*>(a.tiles + ((u0 + local) % a.data_tiles) * (TBU * 24));
  };
  TileRing<STA, decltype(src)> ring{smem, bars, uint32_t(TBU * 24), a.err, total, src, 0};
  ring.start();
  ulonglong2* slot = reinterpret_cast<ulonglong2*>(smem + S::ring) + tid;  // slot i at [i NT]
  float* red = reinterpret_cast<float*>(smem + S::ring + S::slots);

  const float s = a.scales[0];
  const u64 NHP2 = pk(a.neg_half_p, a.neg_half_p), NHP12 = pk(a.neg_half_p1, a.neg_half_p1);
  // log2 of the unscaled d^2 = log2 of the scaled one - 2 log2 s (exact).
  const float shift = -2.f * static_cast<float>(ilogbf(s));
  const u64 SHIFT = pk(shift, shift);

  int64_t i = 0;
  bool aborted = false;
  while (i < total) {
    const int64_t rt = (u0 + i) / a.data_tiles;
    const int64_t seg_end = min(total, (rt + 1) * a.data_tiles - u0);
    u64 QX[KPF], QY[KPF], C[KPF], ZQ[KPF];
#pragma unroll
    for (int k = 0; k < KPF; ++k) {
      // As staged: negated coordinates and Z, since the packed unit adds (so
      // x - q, and the sums made of it change sign at the end).
      const ulonglong2 xy = a.queries[((rt * KPF + k) * NT + tid) * 2];
      const ulonglong2 cz = a.queries[((rt * KPF + k) * NT + tid) * 2 + 1];
      QX[k] = xy.x;
      QY[k] = xy.y;
      C[k] = cz.x;
      ZQ[k] = cz.y;
    }
#pragma unroll
    for (int c = 0; c < 3 * KPF; ++c) slot[c * NT] = make_ulonglong2(0ull, 0ull);

    for (; i < seg_end; ++i) {
      bool ok;
      const unsigned char* st = ring.wait(i, ok);
      const int64_t dt = (u0 + i) % a.data_tiles;
      float* R = red + (i & 1) * (WARPS * 3 * TBU);
      if (ok) {
        const ulonglong2* XY = reinterpret_cast<const ulonglong2*>(st);
        const u64* ZZ = reinterpret_cast<const u64*>(st + TBU * 16);
#pragma unroll 1
        for (int c0 = 0; c0 < TBU; c0 += CHA) {
          u64 CX[KPF], CY[KPF], CP[KPF];
#pragma unroll
          for (int k = 0; k < KPF; ++k) CX[k] = CY[k] = CP[k] = 0ull;
#pragma unroll 1
          for (int g8 = c0; g8 < c0 + CHA; g8 += 8) {
            // The lane's point number j: the query sums grow, the data sums
            // of its 8 queries are returned.
            auto point = [&](int j) {
              const int r = g8 + (j ^ l7);
              const ulonglong2 xy = XY[r];
              const u64 zz = ZZ[r];
              u64 G0 = 0ull, G1 = 0ull, G2 = 0ull;
#pragma unroll
              for (int k = 0; k < KPF; ++k) {
                const u64 dx = add2f(xy.x, QX[k]);  // x_i - q_j
                const u64 dy = add2f(xy.y, QY[k]);
                const u64 d2 = fma2f(dy, dy, mul2f(dx, dx));
                u64 w, v2, L = 0ull;
                weights<POW2, NEED_P>(d2, NHP2, NHP12, w, v2, L);
                const u64 e = add2(zz, ZQ[k]);  // z_i - Z_j
                const u64 ev = mul2(e, v2);
                CX[k] = fma2(ev, dx, CX[k]);
                CY[k] = fma2(ev, dy, CY[k]);
                if (NEED_P) CP[k] = fma2(mul2(e, w), add2(L, SHIFT), CP[k]);
                const u64 b = mul2(C[k], ev);  // c (z_i - Z_j) w / d^2
                G0 = k == 0 ? mul2(C[k], w) : fma2(C[k], w, G0);
                G1 = k == 0 ? mul2(b, dx) : fma2(b, dx, G1);
                G2 = k == 0 ? mul2(b, dy) : fma2(b, dy, G2);
              }
              float3 f;
              float lo, hi;
              upk(G0, lo, hi);
              f.x = __fadd_rn(lo, hi);
              upk(G1, lo, hi);
              f.y = __fadd_rn(lo, hi);
              upk(G2, lo, hi);
              f.z = __fadd_rn(lo, hi);
              return f;
            };
            auto join = [&](float3 keep, float3 give, int o) {
              keep.x = __fadd_rn(keep.x, __shfl_xor_sync(0xffffffffu, give.x, o));
              keep.y = __fadd_rn(keep.y, __shfl_xor_sync(0xffffffffu, give.y, o));
              keep.z = __fadd_rn(keep.z, __shfl_xor_sync(0xffffffffu, give.z, o));
              return keep;
            };
            auto pair4 = [&](int j) {  // points j and j + 4
              const float3 k0 = point(j), k1 = point(j + 4);
              return join(k0, k1, 4);
            };
            float3 f02, f13;
            {
              const float3 f0 = pair4(0), f2 = pair4(2);
              f02 = join(f0, f2, 2);
            }
            {
              const float3 f1 = pair4(1), f3 = pair4(3);
              f13 = join(f1, f3, 2);
            }
            float3 f = join(f02, f13, 1);  // point l7, over 8 lanes
            f = join(f, f, 8);
            f = join(f, f, 16);
            if (lane < 8) {
              R[(warp * 3 + 0) * TBU + g8 + lane] = f.x;
              R[(warp * 3 + 1) * TBU + g8 + lane] = f.y;
              R[(warp * 3 + 2) * TBU + g8 + lane] = f.z;
            }
          }
#pragma unroll
          for (int k = 0; k < KPF; ++k) {
            ulonglong2 x = slot[(3 * k) * NT], y = slot[(3 * k + 1) * NT];
            two_sum_acc(x.x, x.y, CX[k]);
            two_sum_acc(y.x, y.y, CY[k]);
            slot[(3 * k) * NT] = x;
            slot[(3 * k + 1) * NT] = y;
            if (NEED_P) {
              ulonglong2 q = slot[(3 * k + 2) * NT];
              two_sum_acc(q.x, q.y, CP[k]);
              slot[(3 * k + 2) * NT] = q;
            }
          }
        }
      }
      if (!ring.release(ok)) {  // its barrier also publishes R
        aborted = true;
        break;
      }
      for (int o = tid; o < 3 * TBU; o += NT) {  // the next unit writes the other half of `red`
        float sum[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int w = 0; w < WARPS; ++w) sum[w & 3] = __fadd_rn(sum[w & 3], R[w * 3 * TBU + o]);
        const int comp = o / TBU, pt = o % TBU;
        const float all = __fadd_rn(__fadd_rn(sum[0], sum[1]), __fadd_rn(sum[2], sum[3]));
        a.dpart[(rt * 3 + comp) * a.npad + dt * TBU + pt] = comp == 0 ? all : -all;
      }
    }
    if (aborted) break;
    float2* P = a.partial + (rt + g) * 3 * RTF;
#pragma unroll
    for (int k = 0; k < KPF; ++k)
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const ulonglong2 v = slot[(3 * k + c) * NT];
        float ha, hb, la, lb;
        upk(v.x, ha, hb);
        upk(v.y, la, lb);
        if (c < 2) ha = -ha, hb = -hb, la = -la, lb = -lb;
        P[c * RTF + (2 * k) * NT + tid] = make_float2(ha, la);
        P[c * RTF + (2 * k + 1) * NT + tid] = make_float2(hb, lb);
      }
  }
  if (aborted) ring.drain(i);
}

// Data-side partials of one panel added in FP64 in query-tile order; the
// last panel's call writes the gradients (or lists the point for FP64).
__global__ void __launch_bounds__(256)
    fused_data_combine_kernel(const float* __restrict__ dpart, int64_t tiles, int64_t npad,
                              int64_t n, const float* __restrict__ scales, double p,
                              double* __restrict__ acc, bool first, bool last,
                              float* __restrict__ grad_z, float* __restrict__ grad_xy,
                              unsigned* __restrict__ dcount, int32_t* __restrict__ dlist) {
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double gs[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    double v = first ? 0.0 : acc[c * npad + i];
#pragma unroll 4
    for (int64_t r = 0; r < tiles; ++r) v += double(dpart[(r * 3 + c) * npad + i]);
    gs[c] = v;
    if (!last) acc[c * npad + i] = v;
  }
  if (!last) return;
  if (!isfinite(gs[0]) || !isfinite(gs[1]) || !isfinite(gs[2])) {
    dlist[atomicAdd(dcount, 1u)] = static_cast<int32_t>(i);  // recomputed in FP64
    return;
  }
  const double sc = scales[0];
  if (grad_z) grad_z[i] = static_cast<float>(gs[0]);
  if (grad_xy) {
    grad_xy[2 * i] = static_cast<float>(p * sc * gs[1]);
    grad_xy[2 * i + 1] = static_cast<float>(p * sc * gs[2]);
  }
}

// Query pairs for the fused sweep, as its registers hold them: thread t of a
// CTA of nt threads holds in pair k the queries 2 k nt + t and
// (2 k + 1) nt + t of its tile; their record is (-xa, -xb, -ya, -yb),
// (ca, cb, -Za, -Zb), 32 bytes at [(tile KPF + k) nt + t].  Loaded as 64-bit
// pairs they need no register moves.  Excluded and padding queries sit at a
// far finite point with c = 0.
__global__ void __launch_bounds__(256)
    stage_query_pairs_kernel(const float* __restrict__ queries, int64_t m, int64_t records, int nt,
                             const float* __restrict__ Z, const double* __restrict__ s0,
                             const int32_t* __restrict__ hit, const float* __restrict__ g,
                             const float* __restrict__ scales, double p,
                             float* __restrict__ pairs) {
  __shared__ double s_pow;  // s^p, one FP64 pow per CTA
  const float s = scales[0];
  if (threadIdx.x == 0) s_pow = pow(double(s), p);
  __syncthreads();
  const int64_t j = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (j >= records) return;
  float qx = kPadPow2, qy = kPadPow2, c = 0.f, z = 0.f;
  if (j < m && hit[j] == kNoHit) {
    qx = queries[2 * j] * s;
    qy = queries[2 * j + 1] * s;
    // S0 of the scaled coordinates is S0 s^-p.
    c = static_cast<float>(double(g[j]) * s_pow / s0[j]);
    z = Z[j];
  }
  const int64_t row = j / nt;  // (tile KPF + k) 2 + half
  float* r = pairs + ((row >> 1) * nt + j % nt) * 8 + (row & 1);
  r[0] = -qx;
  r[2] = -qy;
  r[4] = c;
  r[6] = -z;
}

// Data points for the fused sweep: units of `unit` (a divisor of 256)
// duplicated pair records, unit x (x, x, y, y) then unit x (z, z).  Padding
// sits at (2^63, 2^63): weights of 2^(-63.5 p) or less, a 2^-53 p-th part of
// any other's, so for p >= 1 it adds nothing to FP32 sums.
__global__ void __launch_bounds__(256)
    stage_points_kernel(const float* __restrict__ data, int64_t n, int64_t records, int unit,
                        const unsigned* __restrict__ maxbits, float* __restrict__ scales,
                        unsigned char* __restrict__ tiles) {
  const int64_t r = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (r >= records) return;
  const float s = scale_from_max(*maxbits);
  if (r == 0) scales[0] = s;
  float x = kPadPow2, y = kPadPow2, z = 0.f;
  if (r < n) {
    x = data[3 * r] * s;
    y = data[3 * r + 1] * s;
    z = data[3 * r + 2];
  }
  unsigned char* base = tiles + r / unit * unit * 24;
  const int64_t at = r % unit;
  reinterpret_cast<float4*>(base)[at] = make_float4(x, x, y, y);
  reinterpret_cast<float2*>(base + unit * 16)[at] = make_float2(z, z);
}

// Streamed query records of the data sweep: (s qx, s qy, c, Z) with
// c = g / S0_scaled (tiles of TQ records are consecutive).  Excluded and padding queries sit at a
// far finite point with c = 0.
__global__ void __launch_bounds__(256)
    stage_queries_kernel(const float* __restrict__ queries, int64_t m, int64_t records,
                         const float* __restrict__ Z, const double* __restrict__ s0,
                         const int32_t* __restrict__ hit, const float* __restrict__ g,
                         const float* __restrict__ scales, double p,
                         unsigned char* __restrict__ tiles) {
  __shared__ double s_pow;  // s^p, one FP64 pow per CTA
  const int64_t j = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  const float s = scales[0];
  if (threadIdx.x == 0) s_pow = pow(double(s), p);
  __syncthreads();
  if (j >= records) return;
  float qx = kPadPow2, qy = kPadPow2, c = 0.f, z = 0.f;
  if (j < m && hit[j] == kNoHit) {
    qx = queries[2 * j] * s;
    qy = queries[2 * j + 1] * s;
    // S0 of the scaled coordinates is S0 s^-p.
    c = static_cast<float>(double(g[j]) * s_pow / s0[j]);
    z = Z[j];
  }
  reinterpret_cast<float4*>(tiles)[j] = make_float4(qx, qy, c, z);
}

__device__ __forceinline__ void piece_range(int64_t rt, int64_t stream_tiles, int64_t units,
                                            int grid, int64_t& g0, int64_t& g1) {
  g0 = cta_of_unit(rt * stream_tiles, units, grid);
  g1 = cta_of_unit((rt + 1) * stream_tiles - 1, units, grid);
}

// Pieces of one register-side point, added in FP64 by 8 lanes (a point's
// lanes are threads ly * 32 + lx, lx the point within the CTA) and joined in
// a fixed order; thread ly = 0 of each point gets the sums.  One lane per
// point spent 0.4 ms on the 608 pieces of a 1000-query call.
constexpr int kPiecePoints = 32, kPieceLanes = 8;
__device__ __forceinline__ void add_pieces(const float2* __restrict__ partial, bool valid,
                                           int64_t rt, int64_t lq, int tile, int64_t stream_tiles,
                                           int64_t units, int grid, double (&sum)[3]) {
  __shared__ double red[kPieceLanes][kPiecePoints][3];
  const int lx = threadIdx.x % kPiecePoints, ly = threadIdx.x / kPiecePoints;
  sum[0] = sum[1] = sum[2] = 0.0;
  if (valid) {
    int64_t g0, g1;
    piece_range(rt, stream_tiles, units, grid, g0, g1);
#pragma unroll 4
    for (int64_t q = g0 + ly; q <= g1; q += kPieceLanes) {
      const float2* P = partial + (rt + q) * 3 * tile + lq;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const float2 v = P[c * tile];
        sum[c] += double(v.x) + double(v.y);
      }
    }
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) red[ly][lx][c] = sum[c];
  __syncthreads();
  if (ly == 0)
    for (int y = 1; y < kPieceLanes; ++y)
#pragma unroll
      for (int c = 0; c < 3; ++c) sum[c] += red[y][lx][c];
}

// Queries j0 .. j1 - 1, swept in register tiles of `tile` counted from j0.
__global__ void __launch_bounds__(kPiecePoints * kPieceLanes)
    query_combine_kernel(const float2* __restrict__ partial, int64_t j0, int64_t j1, int tile,
                         int64_t stream_tiles, int64_t units, int grid,
                         const float* __restrict__ g,
                         const double* __restrict__ s0, const int32_t* __restrict__ hit,
                         const float* __restrict__ scales, double p,
                         float* __restrict__ grad_q, double* __restrict__ gp,
                         Control* __restrict__ ctrl, int32_t* __restrict__ list) {
  __shared__ double s_pow;  // s^-p, one FP64 pow per CTA
  const double sc = scales[0];
  if (threadIdx.x == kPiecePoints) s_pow = pow(sc, -p);
  const int64_t j = j0 + int64_t(blockIdx.x) * kPiecePoints + threadIdx.x % kPiecePoints;
  const bool in = j < j1, fast = in && hit[j] == kNoHit;
  double sum[3];
  add_pieces(partial, fast, (j - j0) / tile, (j - j0) % tile, tile, stream_tiles, units, grid, sum);
  if (threadIdx.x >= kPiecePoints || !in) return;
  if (!fast) {  // exact hits: 0; FP64 queries: written by the fix-up
    if (grad_q) grad_q[2 * j] = grad_q[2 * j + 1] = 0.f;
    gp[j] = 0.0;
    return;
  }
  if (!isfinite(sum[0]) || !isfinite(sum[1]) || !isfinite(sum[2])) {
    // A pair too close for FP32's range of w / d^2: redo this query's
    // query-side sums in FP64 (its data-side terms are fine).
    list[atomicAdd(&ctrl->flagged, 1u)] = static_cast<int32_t>(-(j + 1));
    return;
  }
  const double s0s = s0[j] * s_pow;  // S0 of the scaled coordinates
  const double gj = g[j];
  if (grad_q) {
    // d/dq of the unscaled problem = s x d/dq of the scaled one.
    grad_q[2 * j] = static_cast<float>(-gj * p * sc * sum[0] / s0s);
    grad_q[2 * j + 1] = static_cast<float>(-gj * p * sc * sum[1] / s0s);
  }
  gp[j] = -gj * 0.6931471805599453 * sum[2] / (2.0 * s0s);
}

__global__ void __launch_bounds__(kPiecePoints * kPieceLanes)
    data_combine_kernel(const float2* __restrict__ partial, int64_t n, int64_t stream_tiles,
                        int64_t units, int grid, const float* __restrict__ scales, double p,
                        float* __restrict__ grad_z, float* __restrict__ grad_xy,
                        unsigned* __restrict__ dcount, int32_t* __restrict__ dlist) {
  const int64_t i = int64_t(blockIdx.x) * kPiecePoints + threadIdx.x % kPiecePoints;
  double sum[3];
  add_pieces(partial, i < n, i / RT, i % RT, RT, stream_tiles, units, grid, sum);
  if (threadIdx.x >= kPiecePoints || i >= n) return;
  if (!isfinite(sum[0]) || !isfinite(sum[1]) || !isfinite(sum[2])) {
    dlist[atomicAdd(dcount, 1u)] = static_cast<int32_t>(i);  // recomputed in FP64
    return;
  }
  const double sc = scales[0];
  if (grad_z) grad_z[i] = static_cast<float>(sum[0]);
  if (grad_xy) {
    grad_xy[2 * i] = static_cast<float>(p * sc * sum[1]);
    grad_xy[2 * i + 1] = static_cast<float>(p * sc * sum[2]);
  }
}

// Queries the forward pass did not take the fast path for: exact hits add
// g_j to dL/dz_k; FP64-recomputed queries are listed for the FP64 kernel.
__global__ void __launch_bounds__(256)
    fixup_scan_kernel(int64_t m, const int32_t* __restrict__ hit, const float* __restrict__ g,
                      float* __restrict__ grad_z, Control* __restrict__ ctrl,
                      int32_t* __restrict__ list) {
  const int64_t j = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (j >= m) return;
  const int32_t h = hit[j];
  if (h >= 0) {
    if (grad_z) atomicAdd(&grad_z[h], g[j]);
  } else if (h == kRecomputedF64) {
    list[atomicAdd(&ctrl->flagged, 1u)] = static_cast<int32_t>(j);
  }
}

// Gradient contribution of one listed query in FP64 (unscaled data,
// weights scaled by d2_min^(p/2), which cancels in every ratio).
__global__ void __launch_bounds__(kSlowThreads)
    slow_grad_kernel(const float* __restrict__ data, int64_t n, const float* __restrict__ queries,
                     double p, const float* __restrict__ g, const Control* __restrict__ ctrl,
                     const int32_t* __restrict__ list, float* __restrict__ grad_z,
                     float* __restrict__ grad_xy, float* __restrict__ grad_q,
                     double* __restrict__ gp) {
  __shared__ double red[kSlowThreads / 32];
  const unsigned count = ctrl->flagged;
  for (unsigned f = blockIdx.x; f < count; f += gridDim.x) {
    // e >= 0: query excluded from the data sweep (all its terms here);
    // e < 0: query -e-1 whose query-side sums left FP32's range.
    const int64_t e_ = list[f];
    const bool full = e_ >= 0;
    const int64_t j = full ? e_ : -e_ - 1;
    const double qx = queries[2 * j], qy = queries[2 * j + 1], gj = g[j];
    double dmin = INFINITY;
    for (int64_t i = threadIdx.x; i < n; i += kSlowThreads) {
      const double dx = qx - data[3 * i], dy = qy - data[3 * i + 1];
      dmin = fmin(dmin, dx * dx + dy * dy);
    }
    dmin = block_reduce<double>(dmin, red, true);
    double s0 = 0.0, s1 = 0.0;
    for (int64_t i = threadIdx.x; i < n; i += kSlowThreads) {
      const double dx = qx - data[3 * i], dy = qy - data[3 * i + 1];
      const double w = pow(dmin / (dx * dx + dy * dy), 0.5 * p);
      s0 += w;
      s1 += w * data[3 * i + 2];
    }
    s0 = block_reduce<double>(s0, red, false);
    s1 = block_reduce<double>(s1, red, false);
    const double Z = s1 / s0;
    double ax = 0.0, ay = 0.0, ap = 0.0;
    for (int64_t i = threadIdx.x; i < n; i += kSlowThreads) {
      const double dx = qx - data[3 * i], dy = qy - data[3 * i + 1];
      const double d2 = dx * dx + dy * dy;
      const double w = pow(dmin / d2, 0.5 * p);
      const double e = (data[3 * i + 2] - Z) * w;
      ax += e * dx / d2;
      ay += e * dy / d2;
      ap += e * log(d2);
      if (full && grad_z) atomicAdd(&grad_z[i], static_cast<float>(gj * w / s0));
      if (full && grad_xy) {
        const double b = gj * p * e / (s0 * d2);
        atomicAdd(&grad_xy[2 * i], static_cast<float>(b * dx));
        atomicAdd(&grad_xy[2 * i + 1], static_cast<float>(b * dy));
      }
    }
    ax = block_reduce<double>(ax, red, false);
    ay = block_reduce<double>(ay, red, false);
    ap = block_reduce<double>(ap, red, false);
    if (threadIdx.x == 0) {
      if (grad_q) {
        grad_q[2 * j] = static_cast<float>(-gj * p * ax / s0);
        grad_q[2 * j + 1] = static_cast<float>(-gj * p * ay / s0);
      }
      gp[j] = -gj * ap / (2.0 * s0);
    }
  }
}

// Data points whose FP32 sums left FP32's range: their sums over the queries
// of the data sweep, in FP64 with the saved S0 and Z.
__global__ void __launch_bounds__(kSlowThreads)
    slow_data_kernel(const float* __restrict__ data, const float* __restrict__ queries,
                     int64_t m, double p, const float* __restrict__ Z,
                     const double* __restrict__ s0, const int32_t* __restrict__ hit,
                     const float* __restrict__ g, const unsigned* __restrict__ dcount,
                     const int32_t* __restrict__ dlist, float* __restrict__ grad_z,
                     float* __restrict__ grad_xy) {
  __shared__ double red[kSlowThreads / 32];
  const unsigned count = *dcount;
  for (unsigned f = blockIdx.x; f < count; f += gridDim.x) {
    const int64_t i = dlist[f];
    const double x = data[3 * i], y = data[3 * i + 1], z = data[3 * i + 2];
    double gz = 0.0, gx = 0.0, gy = 0.0;
    for (int64_t j = threadIdx.x; j < m; j += kSlowThreads) {
      if (hit[j] != kNoHit) continue;
      const double dx = double(queries[2 * j]) - x, dy = double(queries[2 * j + 1]) - y;
      const double d2 = dx * dx + dy * dy;
      const double w = pow(d2, -0.5 * p);
      const double c = double(g[j]) / s0[j];
      gz += c * w;
      const double b = c * p * (z - double(Z[j])) * w / d2;
      gx += b * dx;
      gy += b * dy;
    }
    gz = block_reduce<double>(gz, red, false);
    gx = block_reduce<double>(gx, red, false);
    gy = block_reduce<double>(gy, red, false);
    if (threadIdx.x == 0) {
      if (grad_z) grad_z[i] = static_cast<float>(gz);
      if (grad_xy) {
        grad_xy[2 * i] = static_cast<float>(gx);
        grad_xy[2 * i + 1] = static_cast<float>(gy);
      }
    }
  }
}

// dL/dp = sum_j gp[j] in a fixed order: CTA b sums its slice into out[b], then
// one CTA sums those (65,536 values: 23 us as one CTA, under 5 us so).
constexpr int kReduceCtas = 128;
__global__ void __launch_bounds__(256)
    reduce_p_kernel(const double* __restrict__ gp, int64_t m, double* __restrict__ out) {
  __shared__ double red[8];
  const int64_t per = (m + gridDim.x - 1) / gridDim.x;
  const int64_t lo = int64_t(blockIdx.x) * per, hi = min(m, lo + per);
  double acc = 0.0;
  for (int64_t j = lo + threadIdx.x; j < hi; j += blockDim.x) acc += gp[j];
  acc = warp_sum(acc);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) acc += red[w];
    out[blockIdx.x] = acc;
  }
}

size_t round_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

template <class K>
int occupancy_of(K kernel, size_t smem) {
  int b = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kernel, NTA, smem);
  return b > 0 ? b : 1;
}

}  // namespace

namespace {
// Predicted clocks of a sweep over the pairs in tiles of `regs` register-side
// and `stream` streamed points, `per_sm` CTAs to an SM: its longest CTA's
// units times a unit's share of an SM.  An SM with a fraction f of its CTAs
// runs at 1 - (1 - f)^2 of `rate` pairs a clock.
double adj_clocks(int64_t nreg, int64_t nstream, int64_t regs, int64_t stream, int per_sm,
                  double rate, int sm_count) {
  const int64_t units = (nreg + regs - 1) / regs * ((nstream + stream - 1) / stream);
  const int64_t grid = std::min<int64_t>(units, int64_t(per_sm) * sm_count);
  const double ctas = double((grid + sm_count - 1) / sm_count);
  const double idle = 1.0 - ctas / per_sm;
  return double((units + grid - 1) / grid) * double(regs * stream) * ctas /
         (rate * (1.0 - idle * idle));
}
}  // namespace

void plan_backward_f32(int64_t n, int64_t m, double p, bool both, int sm_count,
                       int ctas_per_sm, BwdPlan* bp) {
  bp->data_tiles = (n + kTB32 - 1) / kTB32;
  bp->query_records_tiles = (m + TQ - 1) / TQ;
  bp->query_reg_tiles = (m + RT - 1) / RT;
  bp->data_reg_tiles = (n + RT - 1) / RT;
  bp->units_q = bp->query_reg_tiles * bp->data_tiles;
  bp->units_d = bp->data_reg_tiles * bp->query_records_tiles;
  const int64_t resident = int64_t(sm_count) * std::max(1, ctas_per_sm);
  bp->grid_q = static_cast<int>(std::max<int64_t>(1, std::min(bp->units_q, resident)));
  bp->grid_d = static_cast<int>(std::max<int64_t>(1, std::min(bp->units_d, resident)));
  bp->staged_bytes = round_up(size_t(bp->data_tiles) * kTileBytes32, 256);
  bp->qtiles_bytes = round_up(size_t(bp->query_records_tiles) * kQTileBytes, 256);
  // One fused sweep when both sides are wanted and p >= 1 (its padding needs
  // that), where the model says so: tiles of 4096, 2048 or 1024 queries (512,
  // 256 or 128 threads).  Pairs per SM and clock as measured at
  // n = m = 65,536, p = 2.5: 7.2 for each of the two sweeps; 4.95, 4.9 and 4.45
  // for the fused one (at p = 2 all are 1.4 times that).
  bp->fused = 0;
  if (both && p >= 1.0) {
    double best = adj_clocks(m, n, RT, kTB32, 1, 7.2, sm_count) +
                  adj_clocks(n, m, RT, TQ, 1, 7.2, sm_count);
    const struct { int threads, points; double rate; } forms[] = {
        {512, 128, 4.95}, {256, 128, 4.9}, {128, 64, 4.45}};
    for (const auto& f : forms) {
      const double t = adj_clocks(m, n, f.threads * 2 * KPF, f.points, 512 / f.threads, f.rate,
                                  sm_count);
      if (t < best) {
        best = t;
        bp->fused = f.threads;
      }
    }
  }
  if (bp->fused) {
    const int64_t tile = int64_t(bp->fused) * 2 * KPF, points = fused_points(bp->fused);
    bp->fused_tiles = (m + tile - 1) / tile;
    bp->fused_data_tiles = (n + points - 1) / points;
    const int64_t npad = bp->fused_data_tiles * points;
    bp->panel_tiles = std::max<int64_t>(
        1, std::min<int64_t>(bp->fused_tiles, int64_t(kPanelBytes / (size_t(npad) * 12))));
    bp->grid_f = static_cast<int>(std::min<int64_t>(
        bp->panel_tiles * bp->fused_data_tiles, int64_t(sm_count) * (512 / bp->fused)));
    bp->dpart_bytes = round_up(size_t(bp->panel_tiles) * size_t(npad) * 12, 256);
    bp->dacc_bytes = bp->panel_tiles < bp->fused_tiles ? round_up(size_t(npad) * 24, 256) : 0;
    bp->staged_bytes = round_up(size_t(bp->data_tiles) * kTileBytes32, 256);
    bp->qtiles_bytes = round_up(size_t(bp->fused_tiles) * tile * 16, 256);
    bp->partial_bytes =
        round_up(size_t(bp->panel_tiles + bp->grid_f - 1) * 3 * tile * sizeof(float2), 256);
  }
  const size_t slots = size_t(std::max(bp->query_reg_tiles + bp->grid_q - 1,
                                       bp->data_reg_tiles + bp->grid_d - 1));
  if (!bp->fused) bp->partial_bytes = round_up(slots * 3 * RT * sizeof(float2), 256);
  bp->gp_bytes = round_up(size_t(m) * sizeof(double), 256);
  bp->list_bytes = round_up(size_t(m) * sizeof(int32_t), 256);
  bp->dlist_bytes = round_up(size_t(n) * sizeof(int32_t), 256);
  bp->scale_bytes = 256 + kReduceCtas * sizeof(double);
  bp->workspace_bytes = bp->staged_bytes + bp->qtiles_bytes + bp->partial_bytes + bp->gp_bytes +
                        bp->list_bytes + bp->dlist_bytes + bp->scale_bytes + bp->dpart_bytes +
                        bp->dacc_bytes;
}

int occupancy_backward_f32() {
  return std::min(occupancy_of(query_adj_kernel<false, true>, size_t(STA) * kTileBytes32),
                  occupancy_of(data_adj_kernel<false>, size_t(STA) * kQTileBytes));
}

namespace {

// What follows the sums: exact hits, the queries redone in FP64, dL/dp.
cudaError_t launch_adj_tail(const BwdProblem& pb, double* gp, int32_t* list, unsigned* maxbits,
                            Control* ctrl, int sm_count, cudaStream_t stream) {
  fixup_scan_kernel<<<static_cast<unsigned>((pb.m + 255) / 256), 256, 0, stream>>>(
      pb.m, pb.hit, pb.g, pb.grad_z, ctrl, list);
  slow_grad_kernel<<<2 * sm_count, kSlowThreads, 0, stream>>>(
      pb.data, pb.n, pb.queries, pb.p, pb.g, ctrl, list, pb.grad_z, pb.grad_xy, pb.grad_q, gp);
  if (pb.grad_p) {
    double* part = reinterpret_cast<double*>(reinterpret_cast<unsigned char*>(maxbits) + 256);
    reduce_p_kernel<<<kReduceCtas, 256, 0, stream>>>(gp, pb.m, part);
    reduce_p_kernel<<<1, 256, 0, stream>>>(part, kReduceCtas, pb.grad_p);
  }
  return cudaGetLastError();
}

// The fused sweep, panel by panel, and its combines.
template <int NT, int TBU>
cudaError_t launch_fused(const BwdProblem& pb, const BwdPlan& bp, const unsigned char* dtiles,
                         unsigned char* qtiles, float2* partial, double* gp, int32_t* list,
                         int32_t* dlist, unsigned* dcount, const float* scales, Control* ctrl,
                         cudaStream_t stream) {
  constexpr int tile = fused_queries<NT>();
  constexpr size_t smem = FusedSmem<NT, TBU>::bytes;
  const int64_t qrec = bp.fused_tiles * tile;
  stage_query_pairs_kernel<<<static_cast<unsigned>((qrec + 255) / 256), 256, 0, stream>>>(
      pb.queries, pb.m, qrec, NT, pb.Z, pb.s0, pb.hit, pb.g, scales, pb.p,
      reinterpret_cast<float*>(qtiles));
  unsigned char* after = reinterpret_cast<unsigned char*>(const_cast<float*>(scales) - 1) + bp.scale_bytes;
  FusedArgs a;
  a.data_tiles = bp.fused_data_tiles;
  a.n = pb.n;
  a.tiles = dtiles;
  a.scales = scales;
  a.neg_half_p = static_cast<float>(-0.5 * pb.p);
  a.neg_half_p1 = static_cast<float>(-0.5 * pb.p - 1.0);
  a.partial = partial;
  a.dpart = reinterpret_cast<float*>(after);
  a.npad = bp.fused_data_tiles * TBU;
  a.err = &ctrl->error;
  double* dacc = reinterpret_cast<double*>(after + bp.dpart_bytes);
  auto kernel = pb.p == 2.0 ? (pb.grad_p ? fused_adj_kernel<NT, TBU, true, true>
                                         : fused_adj_kernel<NT, TBU, true, false>)
                            : fused_adj_kernel<NT, TBU, false, true>;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(smem));
  if (e != cudaSuccess) return e;
  for (int64_t t0 = 0; t0 < bp.fused_tiles; t0 += bp.panel_tiles) {
    const int64_t tiles = std::min(bp.panel_tiles, bp.fused_tiles - t0);
    a.units = tiles * bp.fused_data_tiles;
    a.grid = static_cast<int>(std::min<int64_t>(bp.grid_f, a.units));
    a.queries = reinterpret_cast<const ulonglong2*>(qtiles) + t0 * tile;
    kernel<<<a.grid, NT, smem, stream>>>(a);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const int64_t j0 = t0 * tile, j1 = std::min<int64_t>(pb.m, j0 + tiles * tile);
    query_combine_kernel<<<static_cast<unsigned>((j1 - j0 + kPiecePoints - 1) / kPiecePoints),
                           kPiecePoints * kPieceLanes, 0, stream>>>(
        partial, j0, j1, tile, bp.fused_data_tiles, a.units, a.grid, pb.g, pb.s0, pb.hit, scales,
        pb.p, pb.grad_q, gp, ctrl, list);
    fused_data_combine_kernel<<<static_cast<unsigned>((pb.n + 255) / 256), 256, 0, stream>>>(
        a.dpart, tiles, a.npad, pb.n, scales, pb.p, dacc, t0 == 0, t0 + tiles == bp.fused_tiles,
        pb.grad_z, pb.grad_xy, dcount, dlist);
  }
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_backward_f32(const BwdProblem& pb, const BwdPlan& bp, void* workspace,
                                Control* ctrl, int sm_count, cudaStream_t stream) {
  unsigned char* ws = static_cast<unsigned char*>(workspace);
  unsigned char* dtiles = ws;
  unsigned char* qtiles = ws + bp.staged_bytes;
  float2* partial = reinterpret_cast<float2*>(qtiles + bp.qtiles_bytes);
  double* gp = reinterpret_cast<double*>(reinterpret_cast<unsigned char*>(partial) +
                                         bp.partial_bytes);
  int32_t* list = reinterpret_cast<int32_t*>(reinterpret_cast<unsigned char*>(gp) + bp.gp_bytes);
  int32_t* dlist =
      reinterpret_cast<int32_t*>(reinterpret_cast<unsigned char*>(list) + bp.list_bytes);
  unsigned* maxbits = reinterpret_cast<unsigned*>(reinterpret_cast<unsigned char*>(dlist) +
                                                  bp.dlist_bytes);
  float* scales = reinterpret_cast<float*>(maxbits + 1);
  unsigned* dcount = maxbits + 2;
  const bool pow2 = pb.p == 2.0;
  const bool need_q = pb.grad_q || pb.grad_p;
  const bool need_d = pb.grad_z || pb.grad_xy;

  Table<1> t;
  t.count = 1;
  t.pad = 0;
  Instance& I = t.inst[0];
  I.data = pb.data;
  I.queries = pb.queries;
  I.out = nullptr;
  I.s0_out = nullptr;
  I.hit_out = nullptr;
  I.tiles = dtiles;
  I.unit_base = 0;
  I.record_base = 0;
  I.n = static_cast<int32_t>(pb.n);
  I.m = static_cast<int32_t>(pb.m);
  I.data_tiles = static_cast<int32_t>(bp.data_tiles);
  I.qtile_base = 0;

  cudaError_t e = cudaMemsetAsync(maxbits, 0, 3 * sizeof(unsigned), stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(&ctrl->flagged, 0, sizeof(unsigned), stream);
  if (e != cudaSuccess) return e;
  const int64_t longest = std::max(pb.n, pb.m);
  const unsigned gx = static_cast<unsigned>(std::min<int64_t>(1024, (longest + 255) / 256));
  range_kernel<1><<<dim3(gx, 1), 256, 0, stream>>>(t, maxbits, nullptr);
  // Data tiles with finite far padding (both weight forms); the query sweep
  // masks the padding of its last tile, and products with it stay finite.
  const int64_t records = bp.data_tiles * kTB32;
  const unsigned record_ctas = static_cast<unsigned>((records + 255) / 256);
  if (bp.fused)
    stage_points_kernel<<<record_ctas, 256, 0, stream>>>(pb.data, pb.n, records,
                                                         fused_points(bp.fused), maxbits,
                                                         scales, dtiles);
  else
    stage_kernel<1, kPow2><<<record_ctas, 256, 0, stream>>>(t, records, maxbits, scales);

  if (bp.fused) {
    auto launch = bp.fused == 512   ? launch_fused<512, fused_points(512)>
                  : bp.fused == 256 ? launch_fused<256, fused_points(256)>
                                    : launch_fused<128, fused_points(128)>;
    e = launch(pb, bp, dtiles, qtiles, partial, gp, list, dlist, dcount, scales, ctrl, stream);
    if (e != cudaSuccess) return e;
    slow_data_kernel<<<2 * sm_count, kSlowThreads, 0, stream>>>(
        pb.data, pb.queries, pb.m, pb.p, pb.Z, pb.s0, pb.hit, pb.g, dcount, dlist, pb.grad_z,
        pb.grad_xy);
    return launch_adj_tail(pb, gp, list, maxbits, ctrl, sm_count, stream);
  }
  AdjArgs a;
  a.scales = scales;
  a.neg_half_p = static_cast<float>(-0.5 * pb.p);
  a.neg_half_p1 = static_cast<float>(-0.5 * pb.p - 1.0);
  a.partial = partial;
  a.err = &ctrl->error;

  if (need_q) {
    a.units = bp.units_q;
    a.grid = bp.grid_q;
    a.stream_tiles = bp.data_tiles;
    a.tiles = dtiles;
    a.nreg = pb.m;
    a.nstream = pb.n;
    a.reg_xy = pb.queries;
    a.reg_stride = 2;
    a.reg_val = pb.Z;
    a.val_stride = 1;
    const size_t smem = size_t(STA) * kTileBytes32;
    if (pow2) {
      if (pb.grad_p)
        query_adj_kernel<true, true><<<bp.grid_q, NTA, smem, stream>>>(a);
      else
        query_adj_kernel<true, false><<<bp.grid_q, NTA, smem, stream>>>(a);
    } else {
      query_adj_kernel<false, true><<<bp.grid_q, NTA, smem, stream>>>(a);
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    query_combine_kernel<<<static_cast<unsigned>((pb.m + kPiecePoints - 1) / kPiecePoints),
                           kPiecePoints * kPieceLanes, 0, stream>>>(
        partial, 0, pb.m, RT, bp.data_tiles, bp.units_q, bp.grid_q, pb.g, pb.s0, pb.hit, scales, pb.p,
        pb.grad_q, gp, ctrl, list);
  }
  if (need_d) {
    const int64_t qrec = bp.query_records_tiles * TQ;
    stage_queries_kernel<<<static_cast<unsigned>((qrec + 255) / 256), 256, 0, stream>>>(
        pb.queries, pb.m, qrec, pb.Z, pb.s0, pb.hit, pb.g, scales, pb.p, qtiles);
    a.units = bp.units_d;
    a.grid = bp.grid_d;
    a.stream_tiles = bp.query_records_tiles;
    a.tiles = qtiles;
    a.nreg = pb.n;
    a.nstream = pb.m;
    a.reg_xy = pb.data;
    a.reg_stride = 3;
    a.reg_val = pb.data + 2;
    a.val_stride = 3;
    const size_t smem = size_t(STA) * kQTileBytes;
    if (pow2)
      data_adj_kernel<true><<<bp.grid_d, NTA, smem, stream>>>(a);
    else
      data_adj_kernel<false><<<bp.grid_d, NTA, smem, stream>>>(a);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    data_combine_kernel<<<static_cast<unsigned>((pb.n + kPiecePoints - 1) / kPiecePoints),
                          kPiecePoints * kPieceLanes, 0, stream>>>(
        partial, pb.n, bp.query_records_tiles, bp.units_d, bp.grid_d, scales, pb.p, pb.grad_z,
        pb.grad_xy, dcount, dlist);
    slow_data_kernel<<<2 * sm_count, kSlowThreads, 0, stream>>>(
        pb.data, pb.queries, pb.m, pb.p, pb.Z, pb.s0, pb.hit, pb.g, dcount, dlist, pb.grad_z,
        pb.grad_xy);
  }
  return launch_adj_tail(pb, gp, list, maxbits, ctrl, sm_count, stream);
}

}  // namespace idw
