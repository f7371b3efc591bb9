// Slow path for the queries that the fast combine flags: an exact hit
// (d = 0, where Eq. 1 is undefined) or a weight sum outside the fast form's
// range.  One CTA per flagged query, FP64 throughout, on the caller's
// original (unscaled) data.
#pragma once

#include <climits>
#include <cmath>

#include "idw_device.cuh"
#include "idw_internal.h"

namespace idw {

constexpr int kSlowThreads = 256;

template <typename T>
__device__ __forceinline__ T block_reduce(T v, T* scratch, bool is_min) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const T other = __shfl_xor_sync(0xffffffffu, v, o);
    v = is_min ? (other < v ? other : v) : v + other;
  }
  __syncthreads();
  if (lane == 0) scratch[wid] = v;
  __syncthreads();
  if (wid == 0) {
    v = lane < (kSlowThreads / 32) ? scratch[lane] : (is_min ? scratch[0] : T(0));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const T other = __shfl_xor_sync(0xffffffffu, v, o);
      v = is_min ? (other < v ? other : v) : v + other;
    }
    if (lane == 0) scratch[0] = v;
  }
  __syncthreads();
  const T r = scratch[0];
  __syncthreads();
  return r;
}

// Points a thread loads before it looks at any of them: the scans below are
// bound by the latency of their loads, and one CTA keeps kSlowUnroll times
// 256 of them in flight (one at a time, a scan of 100,003 points took 0.4 ms
// on a GB300; eight at a time, 0.06 ms).
constexpr int kSlowUnroll = 8;

// Calls f(i, x_i, y_i) for the CTA's points first + tid, first + tid + 256,
// ... below end, in increasing i per thread; f returns true to stop.
template <typename T, class F>
__device__ __forceinline__ void slow_scan(const T* __restrict__ data, int64_t first, int64_t end,
                                          F f) {
  for (int64_t i0 = first + threadIdx.x; i0 < end; i0 += kSlowUnroll * kSlowThreads) {
    T x[kSlowUnroll], y[kSlowUnroll];
#pragma unroll
    for (int u = 0; u < kSlowUnroll; ++u) {
      const int64_t i = min(i0 + u * kSlowThreads, end - 1);
      x[u] = data[3 * i];
      y[u] = data[3 * i + 1];
    }
    bool stop = false;
#pragma unroll
    for (int u = 0; u < kSlowUnroll; ++u) {
      const int64_t i = i0 + u * kSlowThreads;
      if (!stop && i < end) stop = f(i, x[u], y[u]);
    }
    if (stop) break;
  }
}

// FP64 sums of one query over a slice of the points: d2_min there, and
// S0, S1 with weights scaled by d2_min^(p/2) (at most 1).  A slice whose
// points all lie at infinity has d2_min = +inf and zero weights.
struct SlowSums {
  double dmin, s0, s1;
};

// The sums over points [first, end), by the whole CTA; every thread gets them.
template <typename T>
__device__ SlowSums slow_sums(const T* __restrict__ data, int64_t first, int64_t end, T qx, T qy,
                              double p) {
  __shared__ double red_d[kSlowThreads / 32];
  const double dqx = qx, dqy = qy;
  double dmin = INFINITY;
  slow_scan(data, first, end, [&](int64_t, T x, T y) {
    const double dx = dqx - double(x), dy = dqy - double(y);
    const double d2 = dx * dx + dy * dy;
    dmin = d2 < dmin ? d2 : dmin;
    return false;
  });
  dmin = block_reduce<double>(dmin, red_d, true);

  const bool pow2 = (p == 2.0);
  double s0 = 0.0, s1 = 0.0;
  slow_scan(data, first, end, [&](int64_t i, T x, T y) {
    const double dx = dqx - double(x), dy = dqy - double(y);
    const double d2 = dx * dx + dy * dy;
    const double r = d2 == INFINITY ? 0.0 : dmin / d2;
    const double w = pow2 ? r : pow(r, 0.5 * p);
    s0 += w;
    s1 += w * double(data[3 * i + 2]);
    return false;
  });
  s0 = block_reduce<double>(s0, red_d, false);
  s1 = block_reduce<double>(s1, red_d, false);
  return SlowSums{dmin, s0, s1};
}

// The result of a query without a coincident point from its sums over all
// points (one thread): the common factor d2_min^(p/2) cancels in Z.
template <typename OutT>
__device__ __forceinline__ void slow_write_sums(const SlowSums& s, double p, OutT* out_j,
                                                double* s0_j, int32_t* hit_j) {
  *out_j = static_cast<OutT>(s.s1 / s.s0);
  if (s0_j) *s0_j = s.dmin < INFINITY ? s.s0 * pow(s.dmin, -0.5 * p) : NAN;
  if (hit_j) *hit_j = kRecomputedF64;
}

// The result of a query that coincides with data point i (one thread).
template <typename T, typename OutT>
__device__ __forceinline__ void slow_write_hit(const T* __restrict__ data, int64_t i, OutT* out_j,
                                               double* s0_j, int32_t* hit_j) {
  *out_j = static_cast<OutT>(data[3 * i + 2]);
  if (s0_j) *s0_j = INFINITY;
  if (hit_j) *hit_j = static_cast<int32_t>(i);
}

// One flagged query j, by the whole CTA: the lowest data index i with
// (x_i, y_i) == (qx, qy) gives Z = z_i; otherwise Eq. 1 in FP64.
template <typename T, typename OutT>
__device__ void slow_one_query(const T* __restrict__ data, int64_t n, T qx, T qy, double p,
                               OutT* out_j, double* s0_j, int32_t* hit_j) {
  __shared__ long long red_i[kSlowThreads / 32];
  long long best = LLONG_MAX;
  slow_scan(data, 0, n, [&](int64_t i, T x, T y) {
    if (x == qx && y == qy) best = i;
    return best != LLONG_MAX;
  });
  best = block_reduce<long long>(best, red_i, true);
  if (best != LLONG_MAX) {
    if (threadIdx.x == 0) slow_write_hit<T, OutT>(data, best, out_j, s0_j, hit_j);
    return;
  }
  const SlowSums sums = slow_sums<T>(data, 0, n, qx, qy, p);
  if (threadIdx.x == 0) slow_write_sums<OutT>(sums, p, out_j, s0_j, hit_j);
}

// Single problem: list holds query indices.
template <typename T, typename OutT>
__global__ void __launch_bounds__(kSlowThreads)
    slow_path_kernel(const T* __restrict__ data, int64_t n, const T* __restrict__ queries,
                     double p, const Control* __restrict__ ctrl, const int32_t* __restrict__ list,
                     OutT* __restrict__ out, double* __restrict__ s0_out,
                     int32_t* __restrict__ hit_out) {
  const unsigned count = ctrl->flagged;
  for (unsigned f = blockIdx.x; f < count; f += gridDim.x) {
    const int64_t j = list[f];
    slow_one_query<T, OutT>(data, n, queries[2 * j], queries[2 * j + 1], p, &out[j],
                            s0_out ? &s0_out[j] : nullptr, hit_out ? &hit_out[j] : nullptr);
  }
}

}  // namespace idw
