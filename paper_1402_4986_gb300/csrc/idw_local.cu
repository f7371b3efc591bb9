// Local (radius-limited) Shepard interpolation: Eq. 1 over the data points
// within distance R of each query.  This is the local variant of the IDW
// implementations the paper cites as related work (Sec. 1), not its global
// method.
//
// Pipeline (all on the caller's stream, no host synchronisation):
//   1. bounding box of the finite data points; the last block plans a
//      uniform grid of cells about R/2 wide, at most 2048 per axis and at
//      most one per two data points (coarser when the box needs it);
//   2. counting sort of the data AND of the queries into the cells
//      (histogram, exclusive scan, scatter of 16-byte records);
//   3. one thread per query, in cell order, walks the rows of cells that its
//      disc of radius R can reach (at most 5 rows of at most 5 cells), each
//      row one contiguous run of sorted data.
// Membership is decided in FP32 as d^2 = fmaf(dy, dy, fl32(dx dx)) <
// fl32(R^2) on the caller's unscaled coordinates.  Weights are FP32 (MUFU
// reciprocal at p = 2; 2^(-(p/2) log2 d^2) with an FMA-recovered exponent
// otherwise) and both sums are carried as compensated (hi, lo) FP32 pairs
// (Knuth's TwoSum per member), then divided with one residual correction.
// Sums that leave FP32's range, and queries that coincide with a data point
// (infinite weight), go to an FP64 pass: an exact hit takes the z of the
// lowest coincident index, other sums are redone with weights scaled by
// d2_min^(p/2).  An empty neighbourhood gives NaN.
//
// Cell positions are computed in FP32 as u(v) = fl(fl(fl(v/2) - fl(x0/2)) *
// inv2), inv2 = fl(2/h): halving is exact for normal floats and keeps the
// difference finite for any finite coordinates, and u is monotone in v.
// With at most 2048 cells per axis, u near the grid is off by at most
// 2^-23 (g + 2) ~ 2^-12 cells from (v - x0)/h.  A member lies less than
// R (1 + 2^-23) from its query (FP32 membership; R + 2^-74 where R^2 is
// subnormal, and h >= 2^-61), so in computed cell positions it lies within
// rho = (R/h)(1 + 2^-8) + 2^-8 of the query, which covers those errors and
// the FP32 rounding of the reach arithmetic.  With h >= R (1 + 2^-6)/2,
// rho < 2: a query scans rows floor(v_q) - 2 .. floor(v_q) + 2, and in each
// the columns floor(u_q - e) .. floor(u_q + e), e = sqrt(rho^2 - dy^2), dy
// the gap between v_q and the row.  Grids that need cells wider than 2^120
// (R or the data's extent near FP32's limit) fall back to a single cell.
// Scatter positions come from atomics, so the order of candidates within a
// cell (and with it the last bits of the compensated sums) can vary between
// calls.
#include <cfloat>
#include <climits>
#include <cmath>
#include <cstdint>

#include <algorithm>
#include <type_traits>
#include <utility>

#include "idw.h"
#include "idw_device.cuh"
#include "idw_internal.h"
#include "idw_local.h"
#include "idw_sort.cuh"

namespace idw {
namespace {

constexpr int kScanBlock = 1024;            // threads of a scan block
constexpr int kScanTile = 4 * kScanBlock;  // entries of a scan tile (an int4 per thread)
constexpr int kLocalThreads = 256;
constexpr int kMaxCellsPerAxis = 2048;
constexpr int kBlockShift = 3;  // occupancy blocks of 8 x 8 cells (k-NN search)
constexpr int kMaxBlocksPerAxis = kMaxCellsPerAxis >> kBlockShift;
// A compensated weight sum below this per member may have lost flushed
// (FTZ) weights: such queries are redone in FP64.
constexpr float kTinyPerMember = 0x1p-100f;

// Kernels here are launched with programmatic dependent launch: each waits in
// pdl_wait() for the kernel ahead of it.  Inputs, which that kernel may be
// writing, are passed without __restrict__: the compiler may move loads
// through a restricted pointer, which it takes to be untouched by anything
// else, above that wait, and reads them through the non-coherent path.

// Index checks of a debug build (-DIDW_DEBUG_CHECKS): a failed check sets
// its site's bit in a device word and the access it guards is skipped; no
// trap.  Release builds compile every check to `true`.
enum DebugSite : unsigned {
  kSiteCell = 0,      // a cell index outside [0, cells]
  kSiteGather = 1,    // a sorted-data position outside [0, n)
  kSiteScatter = 2,   // a scatter position outside its array
  kSiteOutput = 3,    // an output row outside [0, m)
  kSiteHeap = 4,      // a heap slot outside [0, k)
  kSiteBlock = 5,     // an occupancy-block index outside the prefix table
  kSiteData = 6,      // a data index outside [0, n)
  kSiteTable = 7,     // a summed-area-table entry outside (gx + 1)(gy + 1)
};
#ifdef IDW_DEBUG_CHECKS
__device__ unsigned g_debug_failures;
__device__ __forceinline__ bool dcheck(bool ok, DebugSite site) {
  if (!ok) atomicOr(&g_debug_failures, 1u << site);
  return ok;
}
#else
__device__ __forceinline__ constexpr bool dcheck(bool, DebugSite) { return true; }
#endif

// Grid of cells, planned on the device.  Each call starts by setting every
// byte of it to 0xff (keys at their identity, tickets at -1).
struct GridDev {
  unsigned keys[4];      // min x, min y, ~max x, ~max y (order-preserving keys)
  unsigned box_ticket;   // blocks of the box kernel done, minus one
  unsigned scan_ticket;  // scan tiles done, minus one
  unsigned filled;       // data cells that hold a point, minus one
  float hx0, hy0, inv2;  // cell position u(v) = fl(fl(fl(v/2) - h0) * inv2)
  float rho;             // reach of R in cells, with margin (< 2)
  int gx, gy, cells;
  unsigned hard;         // queries the per-thread kernels left to warps
  unsigned left;         // queries the search by counts left to warps or threads
  unsigned next;         // next group of queries of the fetching heap search
  unsigned beyond;       // of kSampleQueries queries: those beyond the grid's edge,
  unsigned dense;        // and those in dense surroundings, or heavy (see sample_queries)
};

// Order-preserving unsigned key of a float (for atomic min).
__device__ __forceinline__ unsigned float_key(float f) {
  const unsigned b = __float_as_uint(f);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float key_float(unsigned k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}
__device__ __forceinline__ bool finite2(float x, float y) {
  return fabsf(x) <= FLT_MAX && fabsf(y) <= FLT_MAX;
}

// Ticket counter: atomic add with acquire-release semantics at GPU scope.
// Its release orders the caller's earlier writes before the increment; the
// caller that draws the last ticket acquires every earlier caller's writes.
__device__ __forceinline__ unsigned ticket_acq_rel(unsigned* counter) {
  unsigned old;
  asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;"
               : "=r"(old)
               : "l"(counter)
               : "memory");
  return old;
}

// Cell position along one axis (same arithmetic for data and queries).
__device__ __forceinline__ float cell_pos(float v, float h0, float inv2) {
  return __fmul_rn(__fsub_rn(__fmul_rn(0.5f, v), h0), inv2);
}
// floor(u) clamped to [lo, hi] (u may be +-inf for far queries, never NaN).
__device__ __forceinline__ int clamp_floor(float u, int lo, int hi) {
  return static_cast<int>(fminf(fmaxf(floorf(u), float(lo)), float(hi)));
}

// Grid for the box in grid->keys (one thread).  For the k-NN form
// (knn_k > 0) the cells are sized as for a radius holding k points at the
// data's mean density over the box, sqrt(k area / (pi n)); the radius only
// sets the cell size there, not the result.
__device__ void plan_grid(GridDev* grid, double radius, double inv_max_cells, int knn_k,
                          int64_t n) {
  const unsigned k0 = __ldcg(&grid->keys[0]), k1 = __ldcg(&grid->keys[1]);
  const unsigned k2 = __ldcg(&grid->keys[2]), k3 = __ldcg(&grid->keys[3]);
  int gx = 1, gy = 1;
  float hx0 = 0.f, hy0 = 0.f, inv2 = 0.f, rho = 1.f;  // inv2 = 0: one cell
  if (k0 != 0xffffffffu) {  // some finite data point
    const float xmin = key_float(k0), ymin = key_float(k1);
    const float xmax = key_float(~k2), ymax = key_float(~k3);
    const double ex = double(xmax) - xmin, ey = double(ymax) - ymin;
    if (knn_k > 0) {
      if (ex * ey > 0.0)
        radius = sqrt(double(knn_k) * ex * ey / (3.141592653589793 * double(n)));
      else if (fmax(ex, ey) > 0.0)
        radius = fmax(ex, ey) * double(knn_k) / (2.0 * double(n));  // points on a line
      else
        radius = 1.0;  // all points coincide: one cell
    }
    double h = fmax(fmax(radius * (0.5 + 0x1p-7), 0x1p-61),
                    fmax(ex * (1.0 / (kMaxCellsPerAxis - 1)), ey * (1.0 / (kMaxCellsPerAxis - 1))));
    h = fmax(h, sqrt(ex * ey * inv_max_cells));
    const float cap = float(kMaxCellsPerAxis - 1), max_cells = float(1.0 / inv_max_cells);
    for (int it = 0; it < 64 && h <= 0x1p120; ++it, h *= 1.25) {
      const float i2 = 2.f * __frcp_rn(__double2float_ru(h));
      const float ux = floorf(cell_pos(xmax, 0.5f * xmin, i2));
      const float uy = floorf(cell_pos(ymax, 0.5f * ymin, i2));
      if (ux <= cap && uy <= cap && (ux + 1.f) * (uy + 1.f) <= max_cells) {
        gx = int(ux) + 1;
        gy = int(uy) + 1;
        hx0 = 0.5f * xmin;
        hy0 = 0.5f * ymin;
        inv2 = i2;
        // h <= 2^120 and h >= R (1 + 2^-6)/2, so R fits a float.
        rho = __fmaf_ru(__fmul_ru(__double2float_ru(radius), i2), 0.5f + 0x1p-9f, 0x1p-8f);
        break;
      }
    }
  }
  grid->hx0 = hx0;
  grid->hy0 = hy0;
  grid->inv2 = inv2;
  grid->rho = rho;
  grid->gx = gx;
  grid->gy = gy;
  grid->cells = gx * gy;
  grid->hard = grid->left = grid->next = 0u;
  grid->beyond = grid->dense = 0u;
}

// Zeroes a histogram over `len4` int4s (grid-stride; the scan reads int4s).
__device__ __forceinline__ void zero_counts(int32_t* counts, int len4) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < len4; i += gridDim.x * blockDim.x)
    reinterpret_cast<int4*>(counts)[i] = make_int4(0, 0, 0, 0);
}
// int4s that hold cells + 1 entries.
__host__ __device__ __forceinline__ int count_int4s(int64_t cells) {
  return static_cast<int>((cells + 1 + 3) / 4);
}

// Bounding box of the finite data points; the last block to finish plans
// the grid.  Also clears the histograms (over the most cells the plan may
// have; counts_q may be null).
__global__ void __launch_bounds__(256)
    box_plan_kernel(const float* data, int64_t n, GridDev* grid,
                    double radius, double inv_max_cells, int knn_k, int64_t max_cells,
                    int32_t* counts_d, int32_t* counts_q) {
  pdl_trigger();
  pdl_wait();
  zero_counts(counts_d, count_int4s(max_cells));
  if (counts_q) zero_counts(counts_q, count_int4s(max_cells));
  __shared__ unsigned part[4][8];
  __shared__ bool last;
  unsigned k0 = 0xffffffffu, k1 = 0xffffffffu, k2 = 0xffffffffu, k3 = 0xffffffffu;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
       i += int64_t(gridDim.x) * blockDim.x) {
    const float x = data[3 * i], y = data[3 * i + 1];
    if (finite2(x, y)) {
      k0 = min(k0, float_key(x));
      k1 = min(k1, float_key(y));
      k2 = min(k2, ~float_key(x));
      k3 = min(k3, ~float_key(y));
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    k0 = min(k0, __shfl_xor_sync(0xffffffffu, k0, o));
    k1 = min(k1, __shfl_xor_sync(0xffffffffu, k1, o));
    k2 = min(k2, __shfl_xor_sync(0xffffffffu, k2, o));
    k3 = min(k3, __shfl_xor_sync(0xffffffffu, k3, o));
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) {
    part[0][wid] = k0;
    part[1][wid] = k1;
    part[2][wid] = k2;
    part[3][wid] = k3;
  }
  __syncthreads();
  if (threadIdx.x < 4) {
    unsigned k = 0xffffffffu;
    for (int w = 0; w < 8; ++w) k = min(k, part[threadIdx.x][w]);
    atomicMin(&grid->keys[threadIdx.x], k);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(&grid->box_ticket, 1u) + 1u == gridDim.x - 1;
  }
  __syncthreads();
  if (last && threadIdx.x == 0) {
    __threadfence();
    plan_grid(grid, radius, inv_max_cells, knn_k, n);
  }
}

// Up to this many queries an index call leaves them as they come: the sort's
// launches and passes (about 15 us) cost more than the locality saves.
// Uniform queries in random order, index of 2^20 uniform points, sorted / as
// they come: radius K = 32 m = 10,007 43.7 / 26.9 us, 150,001 56.0 / 45.6; k-NN
// k = 8 m = 30,000 68.4 / 53.9, k = 32 m = 150,001 204.8 / 213.9 (50,000 points:
// 146 / 216).
constexpr int64_t kUnsortedRadius = int64_t(1) << 17, kUnsortedKnn = int64_t(1) << 15;

// Cell of a data point (-1: a non-finite point, in no cell) and sorting
// bucket of a query (its cell clamped into the grid).
__device__ __forceinline__ int data_cell(const GridDev& g, float x, float y) {
  if (!finite2(x, y)) return -1;
  const int cx = clamp_floor(cell_pos(x, g.hx0, g.inv2), 0, g.gx - 1);
  const int cy = clamp_floor(cell_pos(y, g.hy0, g.inv2), 0, g.gy - 1);
  return cy * g.gx + cx;
}
__device__ __forceinline__ int query_bucket(const GridDev& g, float x, float y) {
  if (!finite2(x, y)) return 0;
  const int cx = clamp_floor(cell_pos(x, g.hx0, g.inv2), 0, g.gx - 1);
  const int cy = clamp_floor(cell_pos(y, g.hy0, g.inv2), 0, g.gy - 1);
  return cy * g.gx + cx;
}

// Whether a position in cells lies more than `cells` beyond the grid's edge.
__device__ __forceinline__ bool beyond_grid(const GridDev& g, float u, float v, float cells = 0.f) {
  return fmaxf(fmaxf(-u, u - float(g.gx)), fmaxf(-v, v - float(g.gy))) > cells;
}

// Threads [0, n) count data points, [n, n + m) count queries.
__global__ void __launch_bounds__(256)
    count_kernel(const GridDev* grid, const float* data, int64_t n,
                 const float* queries, int64_t m, int32_t* counts_d,
                 int32_t* counts_q) {
  pdl_trigger();
  pdl_wait();
  const GridDev g = *grid;
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i < n) {
    const int c = data_cell(g, data[3 * i], data[3 * i + 1]);
    if (c >= 0) atomicAdd(&counts_d[c], 1);
  } else if (i < n + m) {
    const int64_t j = i - n;
    atomicAdd(&counts_q[query_bucket(g, queries[2 * j], queries[2 * j + 1])], 1);
  }
}

// Exclusive scan of one value per thread over a kScanBlock-thread block;
// `total` receives the block's sum.  `warp_tot` holds kScanBlock / 32 ints.
__device__ __forceinline__ int32_t block_exclusive_scan(int32_t v, int32_t* warp_tot,
                                                        int32_t& total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int32_t incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == 31) warp_tot[wid] = incl;
  __syncthreads();
  if (wid == 0) {
    int32_t w = warp_tot[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t t = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += t;
    }
    warp_tot[lane] = w;  // inclusive over warps
  }
  __syncthreads();
  total = warp_tot[kScanBlock / 32 - 1];
  return (wid > 0 ? warp_tot[wid - 1] : 0) + incl - v;
}

// Exclusive scan of the histograms (half = first + blockIdx.y: 0 data,
// 1 queries; launched with gridDim.y = 2 for both, 1 for one), one tile of
// kScanTile entries per block (four consecutive entries per thread), over
// cells + 1 entries.  Each tile writes its local prefix to starts[],
// clears the counts (they become the scatter cursors) and records its total;
// the block that finishes last turns the totals into tile bases (exclusive
// scan in place), so that a cell starts at starts[i] + base[i / kScanTile].
// The histogram arrays hold a multiple of four entries, 16-byte aligned.
__global__ void __launch_bounds__(kScanBlock)
    scan_kernel(GridDev* grid, int32_t* counts_d,
                int32_t* counts_q, int32_t* starts_d,
                int32_t* starts_q, int32_t* sums, int max_tiles,
                int first) {
  pdl_trigger();
  pdl_wait();
  __shared__ int32_t warp_tot[kScanBlock / 32], warp_full[kScanBlock / 32];
  __shared__ bool last;
  const int len = grid->cells + 1;
  const int ntiles = (len + kScanTile - 1) / kScanTile;
  if (int(blockIdx.x) >= ntiles) return;  // tile beyond the grid
  const int half = first + int(blockIdx.y);
  int4* in = reinterpret_cast<int4*>(half ? counts_q : counts_d);
  int4* out = reinterpret_cast<int4*>(half ? starts_q : starts_d);
  const int i4 = blockIdx.x * kScanBlock + threadIdx.x;  // int4 index
  int4 v = make_int4(0, 0, 0, 0);
  if (4 * i4 < len) {
    v = in[i4];
    in[i4] = make_int4(0, 0, 0, 0);
  }
  // Entries past len are zero: the arrays are cleared up to a multiple of 4.
  if (half == 0) {
    const int full = (v.x > 0) + (v.y > 0) + (v.z > 0) + (v.w > 0);
    const int w = __reduce_add_sync(0xffffffffu, full);
    if ((threadIdx.x & 31) == 0) warp_full[threadIdx.x >> 5] = w;
  }
  int32_t total;
  const int32_t before = block_exclusive_scan(v.x + v.y + v.z + v.w, warp_tot, total);
  if (4 * i4 < len)
    out[i4] = make_int4(before, before + v.x, before + v.x + v.y, before + v.x + v.y + v.z);
  if (half == 0 && threadIdx.x < 32) {  // warp_full was written before the scan's barriers
    const int w = __reduce_add_sync(0xffffffffu, warp_full[threadIdx.x]);
    if (threadIdx.x == 0 && w > 0) atomicAdd(&grid->filled, unsigned(w));
  }
  if (threadIdx.x == 0) {
    sums[half * max_tiles + blockIdx.x] = total;  // published by the ticket
    last = ticket_acq_rel(&grid->scan_ticket) + 1u == unsigned(int(gridDim.y) * ntiles - 1);
  }
  __syncthreads();  // the last block's threads read after thread 0's acquire
  if (!last) return;
  const int per = (ntiles + kScanBlock - 1) / kScanBlock;
  for (int y = first; y < first + int(gridDim.y); ++y) {
    int32_t* sb = sums + y * max_tiles;
    const int b0 = min(ntiles, int(threadIdx.x) * per), b1 = min(ntiles, b0 + per);
    int32_t acc = 0;
    for (int b = b0; b < b1; ++b) acc += __ldcg(&sb[b]);
    __syncthreads();  // warp_tot is reused
    int32_t run = block_exclusive_scan(acc, warp_tot, total);
    for (int b = b0; b < b1; ++b) {
      const int32_t t = __ldcg(&sb[b]);
      sb[b] = run;
      run += t;
    }
  }
}

__device__ __forceinline__ int cell_start(const int32_t* starts,
                                          const int32_t* base, int i, int cells) {
  if (!dcheck(i >= 0 && i <= cells, kSiteCell)) return 0;
  return starts[i] + base[i / kScanTile];
}

// Occupancy of 8 x 8-cell blocks for the k-NN search: for block row by,
// bpre[by * (kMaxBlocksPerAxis + 1) + bx] is the number of data points in
// blocks 0 .. bx - 1 of that row.  One CTA per block row, one thread per
// block; runs after the scan (cell starts are final).
__global__ void __launch_bounds__(kMaxBlocksPerAxis)
    block_prefix_kernel(const GridDev* grid, const int32_t* starts,
                        const int32_t* base, int32_t* bpre) {
  pdl_trigger();
  pdl_wait();
  __shared__ int32_t warp_tot[kMaxBlocksPerAxis / 32];
  const GridDev g = *grid;
  const int bgx = (g.gx + 7) >> kBlockShift, bgy = (g.gy + 7) >> kBlockShift;
  const int by = blockIdx.x;
  if (by >= bgy) return;
  const int bx = threadIdx.x;
  int32_t c = 0;
  if (bx < bgx) {
    const int x0 = bx << kBlockShift, x1 = min(g.gx - 1, x0 + 7);
    const int y0 = by << kBlockShift, y1 = min(g.gy - 1, y0 + 7);
    for (int yy = y0; yy <= y1; ++yy)
      c += cell_start(starts, base, yy * g.gx + x1 + 1, g.cells) -
           cell_start(starts, base, yy * g.gx + x0, g.cells);
  }
  // Exclusive scan over the row's blocks (kMaxBlocksPerAxis threads).
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int32_t incl = c;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == 31) warp_tot[wid] = incl;
  __syncthreads();
  int32_t before = incl - c;
  for (int w = 0; w < wid; ++w) before += warp_tot[w];
  int32_t* row = bpre + by * (kMaxBlocksPerAxis + 1);
  if (bx < bgx) row[bx] = before;
  if (bx == bgx - 1) row[bgx] = before + c;  // the row total
}

// Summed-area table of the data cells for the k-NN search: with W = gx + 1,
// sat[y * W + x] is the number of data points in rows 0 .. y - 1 and columns
// 0 .. x - 1, so any rectangle of cells is counted from four entries.  A
// CTA takes 32 columns; its warp w sums rows w C .. (w + 1) C - 1 of each
// column (C = ceil(gy / 32)), the warps' totals are scanned through shared
// memory, and each warp writes its rows.  Launched with enough CTAs for
// 2049 columns; those past gx + 1 return at once (the plan is on the
// device).
constexpr int kSatCols = 32, kSatWarps = 32;
__global__ void __launch_bounds__(kSatCols * kSatWarps)
    sat_kernel(const GridDev* grid, const int32_t* starts,
               const int32_t* base, int32_t* sat) {
  pdl_trigger();
  pdl_wait();
  __shared__ int32_t part[kSatWarps][kSatCols];
  const GridDev g = *grid;
  if (int(blockIdx.x) * kSatCols > g.gx) return;  // the whole CTA: no barrier is reached
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int W = g.gx + 1, x = blockIdx.x * kSatCols + lane;
  const int chunk = (g.gy + kSatWarps - 1) / kSatWarps;
  const int y0 = min(g.gy, w * chunk), y1 = min(g.gy, y0 + chunk);
  // Points of row y in columns 0 .. x - 1 (x = gx: the whole row).
  auto row_prefix = [&](int y) {
    return cell_start(starts, base, y * g.gx + x, g.cells) -
           cell_start(starts, base, y * g.gx, g.cells);
  };
  int32_t s = 0;
  if (x < W)
    for (int y = y0; y < y1; ++y) s += row_prefix(y);
  part[w][lane] = s;
  __syncthreads();
  int32_t acc = 0;
  for (int i = 0; i < w; ++i) acc += part[i][lane];
  if (x < W) {
    if (w == 0) sat[x] = 0;
    for (int y = y0; y < y1; ++y) {
      acc += row_prefix(y);
      if (dcheck(y + 1 <= g.gy, kSiteTable)) sat[(y + 1) * W + x] = acc;
    }
  }
}

// Query records in the caller's order, (x, y, index, 0): used in place of
// the query sort when the caller's order is kept.
__global__ void __launch_bounds__(256)
    query_identity_kernel(const float* queries, int64_t m,
                          float4* qrec) {
  pdl_trigger();
  pdl_wait();
  const int64_t j = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (j >= m) return;
  qrec[j] = make_float4(queries[2 * j], queries[2 * j + 1], __int_as_float(static_cast<int>(j)),
                        0.f);
}

// MUFU square root (relative error ~2^-22, subnormal input flushed to 0).
__device__ __forceinline__ float sqrt_approx(float x) {
  float r;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// The runs of sorted data a query's disc of radius R can reach: at most
// five rows, each one contiguous run [a[r], b[r]) (empty runs have a == b).
// All runs are looked up before any is walked, so their loads overlap.
// The reach e of a row comes from the MUFU square root: its error (and a
// flushed subnormal rho^2 - dy^2, where no member can lie) is far inside
// rho's margin.
struct Runs {
  int a[5], b[5];

  __device__ __forceinline__ int candidates() const {
    int c = 0;
#pragma unroll
    for (int r = 0; r < 5; ++r) c += b[r] - a[r];
    return c;
  }
  __device__ __forceinline__ Runs(const GridDev& g, float qx, float qy,
                                  const int32_t* starts,
                                  const int32_t* base) {
    int y0 = 0, y1 = -1;
    float u = 0.f, v = 0.f;
    if (finite2(qx, qy)) {
      u = cell_pos(qx, g.hx0, g.inv2);
      v = cell_pos(qy, g.hy0, g.inv2);
      const int cy = clamp_floor(v, -3, g.gy + 2);
      y0 = cy - 2;
      y1 = min(g.gy - 1, cy + 2);
    }
#pragma unroll
    for (int r = 0; r < 5; ++r) {
      const int yy = y0 + r;
      const float dy = fmaxf(0.f, fmaxf(float(yy) - v, v - float(yy + 1)));
      const float e = sqrt_approx(fmaxf(0.f, __fmaf_rn(-dy, dy, g.rho * g.rho)));
      const int xa = clamp_floor(u - e, 0, g.gx), xb = clamp_floor(u + e, -1, g.gx - 1);
      a[r] = b[r] = 0;
      if (yy >= 0 && yy <= y1 && dy < g.rho && xa <= xb) {
        a[r] = cell_start(starts, base, yy * g.gx + xa, g.cells);
        b[r] = cell_start(starts, base, yy * g.gx + xb + 1, g.cells);
      }
    }
  }
};

// Heavy queries: those with more candidates than `heavy_candidates`.  A
// thread walks its candidates one load after another while the other lanes
// wait, so heavy queries are listed and each is given a whole warp by a
// kernel of their own.  At the mean density a query has about 21 cells of
// candidates.  Calls that do not fill the GPU (few = true) list queries a
// little above that; others, whose warps hide each other's loads, only those
// several times above it.  200,003 points in 64 blobs, 150,001 uniform
// queries, R for 16 members at the mean density (up to 1400 candidates a
// query, modified Shepard): values 178 -> 18 us for the heavy queries and
// 60 us for the rest, query gradients 680 -> 47 and 150 us.
__device__ __forceinline__ int heavy_candidates(const GridDev& g, int64_t n, bool few) {
  const float per_cell = float(n) * rcp_approx(float(g.cells));
  return int(few ? fminf(fmaf(24.f, per_cell, 32.f), 1e9f) : fminf(fmaf(64.f, per_cell, 256.f), 1e9f));
}
// Whether a query goes on the list: a heavy one, unless the sample shows that
// the call has more than `most` of them, enough to fill the GPU a thread each.
// Such calls (queries clustered like the data) keep every lane busy, and
// neighbouring threads share the candidates that a warp per query loads for
// each: 2^20 points and queries in the same 64 blobs, R for 32 members at the
// mean density, threads / warps: values 1100 / 1880 us, gradients 4530 / 6160.
// (150,001 queries: 390 / 344 and 1250 / 1060.)
constexpr int kSampleQueries = 256;
//
// Queries in no spatial order (`scattered`) are heavy from 128 + 3 m / 1024
// candidates on: threads of a warp then read from as many places, the 32 lanes
// of one query from one.  More queries hide more of the threads' latency.
// Index of 2^20 uniform points, R for 128 / 512 / 2048 members, us sorted first / a
// thread each / by this rule: 10,007 queries 74 / 176 / 576, 74 / 219 / 914 and
// 31 / 32 / 75; 131,072 queries 92 / 240 / 799, 107 / 381 / 1456 and 107 / 335 / 830.
// (A bound of 128 + m / 256 just missed the second: 382; and 10,007 queries with
// 256 members in 2^24 points 147 us, 29 so.)
__device__ __forceinline__ bool list_if_heavy(const GridDev& g, const Runs& runs, int64_t n,
                                              int64_t m, int64_t most, bool scattered = false) {
  int bound = heavy_candidates(g, n, m <= most);
  if (scattered) bound = min(bound, 128 + int(3 * m / 1024));
  return runs.candidates() > bound && g.dense * m <= kSampleQueries * most;
}

// Radius of the square of cells that holds 2k points at the mean density:
// ceil((sqrt(2 k ca) - 1) / 2) with ca cells per point.
__device__ __forceinline__ int knn_square(float cells_per_point, int k) {
  return int(ceilf(0.5f * (sqrt_approx(2.f * float(k) * cells_per_point) - 1.f)));
}
// More than this in that square is dense.
__device__ __forceinline__ int knn_dense(int k) { return 8 * k + 64; }

// What kSampleQueries of the queries, by a block of as many threads, have
// around them, from the cells' starts: counts those beyond the grid's edge and
// those in dense surroundings (a k-NN call, k > 0), or the heavy ones (a radius
// call, kSampleRadius).
constexpr int kSampleK = 2;  // with one neighbour a thread is through a cluster soon
constexpr int kSampleRadius = -1;
__device__ __forceinline__ void sample_queries(GridDev* out, const GridDev& g,
                                               const int32_t* starts, const int32_t* base,
                                               int64_t n, const float* queries, int64_t m, int k) {
  const int64_t j = m * threadIdx.x / kSampleQueries;
  const float x = queries[2 * j], y = queries[2 * j + 1];
  bool beyond = false, dense = false;
  if (k == kSampleRadius) {
    dense = Runs(g, x, y, starts, base).candidates() > heavy_candidates(g, n, false);
  } else if (finite2(x, y)) {
    const float u = cell_pos(x, g.hx0, g.inv2), v = cell_pos(y, g.hy0, g.inv2);
    const int cx = clamp_floor(u, 0, g.gx - 1), cy = clamp_floor(v, 0, g.gy - 1);
    const int re = knn_square(float(g.cells) * rcp_approx(float(n)), k);
    int held = 0;
    for (int yy = max(0, cy - re); yy <= min(g.gy - 1, cy + re); ++yy)
      held += cell_start(starts, base, yy * g.gx + min(g.gx - 1, cx + re) + 1, g.cells) -
              cell_start(starts, base, yy * g.gx + max(0, cx - re), g.cells);
    beyond = beyond_grid(g, u, v);
    dense = held > knn_dense(k);
  }
  const int nb = __syncthreads_count(beyond), nd = __syncthreads_count(dense);
  if (threadIdx.x == 0) {
    out->beyond = nb;
    out->dense = nd;
  }
}

// Threads [0, n) place data points as (x, y, z, index), [n, n + m) place
// queries as (x, y, index, 0).  With `sample` not 0 (see sample_queries) the
// first block samples the call's `all` queries instead.
__global__ void __launch_bounds__(256)
    scatter_kernel(GridDev* grid, const float* data, int64_t n,
                   const float* queries, int64_t m, int64_t all, int sample,
                   const int32_t* starts_d, const int32_t* starts_q,
                   const int32_t* sums, int max_tiles,
                   int32_t* cursor_d, int32_t* cursor_q,
                   float4* sorted, float4* qrec) {
  pdl_trigger();
  pdl_wait();
  const GridDev g = *grid;
  if (sample != 0 && blockIdx.x == 0) {
    sample_queries(grid, g, starts_d, sums, n, queries, all, sample);
    return;
  }
  const int64_t i = int64_t(blockIdx.x - (sample != 0)) * blockDim.x + threadIdx.x;
  if (i < n) {
    const float x = data[3 * i], y = data[3 * i + 1];
    const int c = data_cell(g, x, y);
    if (c < 0) return;
    const int pos = cell_start(starts_d, sums, c, g.cells) + atomicAdd(&cursor_d[c], 1);
    if (!dcheck(pos >= 0 && pos < n, kSiteScatter)) return;
    sorted[pos] = make_float4(x, y, data[3 * i + 2], __int_as_float(static_cast<int>(i)));
  } else if (i < n + m) {
    const int64_t j = i - n;
    const float x = queries[2 * j], y = queries[2 * j + 1];
    const int b = query_bucket(g, x, y);
    const int pos = cell_start(starts_q, sums + max_tiles, b, g.cells) + atomicAdd(&cursor_q[b], 1);
    if (!dcheck(pos >= 0 && pos < m, kSiteScatter)) return;
    qrec[pos] = make_float4(x, y, __int_as_float(static_cast<int>(j)), 0.f);
  }
}

template <int MODE>
__device__ __forceinline__ float local_weight(float d2, float hp, float nhp) {
  if (MODE == kPow2) return rcp_approx(d2);
  const float L = lg2_approx(d2);
  const float th = L * nhp;
  const float tl = fmaf(L, nhp, L * hp);  // exact rounding error of th
  const float e = ex2_approx(th);
  return fmaf(e, tl * 0.6931471805599453f, e);
}

__device__ __forceinline__ float fp32_d2(float qx, float qy, float x, float y) {
  const float dx = __fsub_rn(qx, x), dy = __fsub_rn(qy, y);
  return __fmaf_rn(dy, dy, __fmul_rn(dx, dx));
}

// A query's runs laid end to end: candidate s of `total` sits at at(s), so
// that one lane, or the 32 lanes of a warp side by side, can walk them.
struct FlatRuns {
  int end[5], shift[5];  // candidates s < end[r] (and >= end[r - 1]) sit at s + shift[r]

  __device__ __forceinline__ explicit FlatRuns(const Runs& runs) {
    int e = 0;
#pragma unroll
    for (int r = 0; r < 5; ++r) {
      shift[r] = runs.a[r] - e;
      e += runs.b[r] - runs.a[r];
      end[r] = e;
    }
  }
  __device__ __forceinline__ int total() const { return end[4]; }
  __device__ __forceinline__ int at(int s) const {
    int d = shift[0];
#pragma unroll
    for (int r = 1; r < 5; ++r) d = s >= end[r - 1] ? shift[r] : d;
    return s + d;
  }
};

// Lists query t (any subset of a warp's lanes may call it together) from
// `list` on upwards, or downwards (step = -1).
template <int step = 1>
__device__ __forceinline__ void list_heavy(int64_t t, int64_t m, unsigned* count,
                                           int32_t* list) {
  const unsigned lanes = __activemask();  // one atomic for those that are here together
  const int lane = threadIdx.x & 31, lead = __ffs(lanes) - 1;
  unsigned at = 0;
  if (lane == lead) at = atomicAdd(count, unsigned(__popc(lanes)));
  at = __shfl_sync(lanes, at, lead) + __popc(lanes & ((1u << lane) - 1));
  if (dcheck(at < m, kSiteScatter)) list[step * int64_t(at)] = static_cast<int32_t>(t);
}

// Error-free sum of the lanes' compensated pairs (both packed lanes), by a
// fixed tree; lane 0's total is returned to every lane.
__device__ __forceinline__ void warp_sum_pairs(u64& hi, u64& lo) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const u64 oh = __shfl_xor_sync(0xffffffffu, hi, o), ol = __shfl_xor_sync(0xffffffffu, lo, o);
    two_sum_acc(hi, lo, oh);
    lo = add2(lo, ol);
  }
  hi = __shfl_sync(0xffffffffu, hi, 0);
  lo = __shfl_sync(0xffffffffu, lo, 0);
}

// One thread per query, in cell order.  The fast loop takes every candidate
// with d^2 < r2t, r2t = fl32(R^2) (or the least subnormal when that is 0,
// so that only d^2 == 0 passes), and sums its FP32 weight.  A coincident
// point (d^2 == 0) has an infinite or NaN weight, so a query with an exact
// hit, or with sums outside FP32's range, falls through to the FP64 pass,
// which takes the z of the lowest coincident index or recomputes the sums
// with weights scaled by d2_min^(p/2).
// Weights of the radius form: d^-p (kWeightShepard) or the modified
// Shepard weights ((R - d)/(R d))^p = (1/d - 1/R)^p (kWeightModified), which
// fall to 0 at d = R.  The modified base comes from the MUFU reciprocal
// square root (relative error ~2^-22) and is clamped at 0 for members that
// rounding puts at the boundary; a coincident point gives an infinite base.
constexpr int kWeightShepard = 0, kWeightModified = 1;
template <int MODE>
__device__ __forceinline__ float modified_weight(float d2, float inv_r, float pw) {
  const float t = fmaxf(rsqrt_approx(d2) - inv_r, 0.f);
  if (MODE == kPow2) return t * t;
  return ex2_approx(pw * lg2_approx(t));
}

// One candidate: adds a member's (w, w z) to the compensated pair.  The
// products w z are rounded once (2^-24), below the error of the MUFU weights
// themselves (2^-23).
template <int MODE, int WMODE>
struct ValueSums {
  u64 hi = 0, lo = 0;
  int cnt = 0;
  __device__ __forceinline__ void consider(const float4 v, float qx, float qy, float r2t,
                                           float inv_r, float hp, float pw) {
    const float d2 = fp32_d2(qx, qy, v.x, v.y);
    if (d2 < r2t) {
      const float w = WMODE == kWeightModified ? modified_weight<MODE>(d2, inv_r, pw)
                                               : local_weight<MODE>(d2, hp, -hp);
      two_sum_acc(hi, lo, pk(w, __fmul_rn(w, v.z)));
      ++cnt;
    }
  }
  // Z, if the sums stayed in FP32's range.
  __device__ __forceinline__ bool value(float& z) const {
    float h0, h1, l0, l1;
    upk(hi, h0, h1);
    upk(lo, l0, l1);
    if (!(h0 >= kTinyPerMember * float(cnt) && h0 <= FLT_MAX && fabsf(h1) <= FLT_MAX &&
          fabsf(l1) <= FLT_MAX))
      return false;
    // Z = (h1 + l1) / (h0 + l0): quotient, then one residual correction.
    const float z0 = __fdiv_rn(h1, h0);
    const float res = __fadd_rn(__fmaf_rn(-z0, h0, h1), __fmaf_rn(-z0, l0, l1));
    z = __fmaf_rn(res, rcp_approx(h0), z0);
    return true;
  }
};

// The FP64 pass of one query, by one lane (WARP false) or a whole warp: exact
// hits first, then the members' d2_min (or, for the modified weights, their
// largest base (R - d)/(R d), clamped at 0) and the sums scaled by it.
struct ValueF64 {
  float z;
  int count;
};
template <int WMODE, bool WARP>
__device__ __forceinline__ ValueF64 local_value_f64(const FlatRuns& fr,
                                                    const float4* sorted, float qx,
                                                    float qy, double p, float r2f, double radius) {
  constexpr unsigned kAll = 0xffffffffu;
  constexpr int step = WARP ? 32 : 1;
  const int first = WARP ? int(threadIdx.x & 31) : 0;
  int best = INT_MAX, members = 0;
  float bestz = 0.f;
  double dmin = INFINITY, tmax = 0.0;
  auto base64 = [&](double e2) {
    const double d = sqrt(e2);
    const double t = isinf(radius) ? 1.0 / d : (radius - d) / (radius * d);
    return t > 0.0 ? t : 0.0;
  };
  for (int i = first; i < fr.total(); i += step) {
    const float4 v = sorted[fr.at(i)];
    if (v.x == qx && v.y == qy) {
      const int idx = __float_as_int(v.w);
      if (idx < best) {
        best = idx;
        bestz = v.z;
      }
    } else if (fp32_d2(qx, qy, v.x, v.y) < r2f) {
      const double ex = double(qx) - v.x, ey = double(qy) - v.y;
      dmin = fmin(dmin, ex * ex + ey * ey);
      if (WMODE == kWeightModified) tmax = fmax(tmax, base64(ex * ex + ey * ey));
      ++members;
    }
  }
  if (WARP) {
    const int lowest = __reduce_min_sync(kAll, best);
    const unsigned who = __ballot_sync(kAll, best == lowest);
    bestz = __shfl_sync(kAll, bestz, __ffs(who) - 1);
    best = lowest;
    members = __reduce_add_sync(kAll, members);
    for (int o = 16; o > 0; o >>= 1) {
      dmin = fmin(dmin, __shfl_xor_sync(kAll, dmin, o));
      tmax = fmax(tmax, __shfl_xor_sync(kAll, tmax, o));
    }
  }
  if (best != INT_MAX) return ValueF64{bestz, -1};
  if (members == 0 || (WMODE == kWeightModified && !(tmax > 0.0)))
    return ValueF64{__int_as_float(0x7fc00000), members};
  double s0 = 0.0, s1 = 0.0;
  for (int i = first; i < fr.total(); i += step) {
    const float4 v = sorted[fr.at(i)];
    if (fp32_d2(qx, qy, v.x, v.y) < r2f) {
      const double ex = double(qx) - v.x, ey = double(qy) - v.y;
      const double w = WMODE == kWeightModified ? pow(base64(ex * ex + ey * ey) / tmax, p)
                                                : pow(dmin / (ex * ex + ey * ey), 0.5 * p);
      s0 += w;
      s1 += w * double(v.z);
    }
  }
  if (WARP) {
    s0 = warp_sum(s0);
    s1 = warp_sum(s1);
  }
  return ValueF64{static_cast<float>(s1 / s0), members};
}

template <int MODE, int WMODE = kWeightShepard>
__global__ void __launch_bounds__(kLocalThreads)
    local_query_kernel(const GridDev* grid, const float4* sorted,
                       int64_t n, const int32_t* starts,
                       const int32_t* base, const float4* qrec,
                       int64_t m, double p, float r2f, float r2t, float* __restrict__ out,
                       int32_t* count_out, double radius, int64_t most, bool scattered,
                       unsigned* heavy_count, int32_t* heavy) {
  pdl_trigger();
  pdl_wait();
  const int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (t >= m) return;
  const float4 r = qrec[t];
  const float qx = r.x, qy = r.y;
  const int j = __float_as_int(r.z);
  if (!dcheck(j >= 0 && j < m, kSiteOutput)) return;
  const Runs runs(*grid, qx, qy, starts, base);
  if (list_if_heavy(*grid, runs, n, m, most, scattered)) {
    list_heavy(t, m, heavy_count, heavy);
    return;
  }
  const float hp = static_cast<float>(0.5 * p);
  const float pw = static_cast<float>(p);
  const float inv_r = WMODE == kWeightModified ? static_cast<float>(1.0 / radius) : 0.f;
  ValueSums<MODE, WMODE> sums;
  // Four loads in flight: a candidate's FP32 work is short next to its load.
#pragma unroll
  for (int r = 0; r < 5; ++r) {
#pragma unroll 4
    for (int k = runs.a[r]; k < runs.b[r]; ++k) {
      if (!dcheck(k >= 0 && k < n, kSiteGather)) break;
      sums.consider(sorted[k], qx, qy, r2t, inv_r, hp, pw);
    }
  }
  float z = __int_as_float(0x7fc00000);  // no member and no coincident point
  int cnt = sums.cnt;
  if (cnt > 0 && !sums.value(z)) {
    const ValueF64 v = local_value_f64<WMODE, false>(FlatRuns(runs), sorted, qx, qy, p, r2f, radius);
    z = v.z;
    cnt = v.count;
  }
  out[j] = z;
  if (count_out) count_out[j] = cnt;
}

// The heavy queries, a warp each: 32 candidates side by side, the lanes'
// sums joined by a fixed tree of error-free additions.
constexpr int kHeavyThreads = 128;
template <int MODE, int WMODE = kWeightShepard>
__global__ void __launch_bounds__(kHeavyThreads)
    local_heavy_kernel(const GridDev* grid, const float4* sorted,
                       int64_t n, const int32_t* starts,
                       const int32_t* base, const float4* qrec,
                       int64_t m, double p, float r2f, float r2t, float* __restrict__ out,
                       int32_t* count_out, double radius,
                       const unsigned* heavy_count,
                       const int32_t* heavy) {
  pdl_trigger();
  pdl_wait();
  const int64_t count = *heavy_count;
  const int lane = threadIdx.x & 31;
  const int64_t warps = int64_t(gridDim.x) * (kHeavyThreads / 32);
  const float hp = static_cast<float>(0.5 * p), pw = static_cast<float>(p);
  const float inv_r = WMODE == kWeightModified ? static_cast<float>(1.0 / radius) : 0.f;
  for (int64_t w = (int64_t(blockIdx.x) * kHeavyThreads + threadIdx.x) / 32; w < count;
       w += warps) {
    const int64_t t = heavy[w];
    if (!dcheck(t >= 0 && t < m, kSiteScatter)) continue;
    const float4 r = qrec[t];
    const float qx = r.x, qy = r.y;
    const int j = __float_as_int(r.z);
    if (!dcheck(j >= 0 && j < m, kSiteOutput)) continue;
    const FlatRuns fr(Runs(*grid, qx, qy, starts, base));
    ValueSums<MODE, WMODE> sums;
#pragma unroll 2
    for (int i = lane; i < fr.total(); i += 32) {
      const int k = fr.at(i);
      if (!dcheck(k >= 0 && k < n, kSiteGather)) break;
      sums.consider(sorted[k], qx, qy, r2t, inv_r, hp, pw);
    }
    warp_sum_pairs(sums.hi, sums.lo);
    sums.cnt = __reduce_add_sync(0xffffffffu, sums.cnt);
    float z = __int_as_float(0x7fc00000);
    int cnt = sums.cnt;
    if (cnt > 0 && !sums.value(z)) {  // the same in every lane
      const ValueF64 v = local_value_f64<WMODE, true>(fr, sorted, qx, qy, p, r2f, radius);
      z = v.z;
      cnt = v.count;
    }
    if (lane == 0) {
      out[j] = z;
      if (count_out) count_out[j] = cnt;
    }
  }
}

// ------------------------------------------------- local-form gradients
//
// dL/d(inputs) of L = sum_j g_j Z(q_j) for the radius form.  Each query's
// membership set is held fixed (it is piecewise constant in every input), so
// every derivative is the global one (the chain rule on Eq. 1) summed over
// the members:
//   dZ/dz_i = w_i / S0,   dZ/dx_i = (p / S0)(z_i - Z) w_i (q - x_i) / d_i^2,
//   dZ/dq = -sum_i dZ/dx_i,   dZ/dp = -(1 / (2 S0)) sum_i (z_i - Z) w_i ln d_i^2.
// Weights are scaled by the members' smallest d^2 (w_i = (d2_min / d_i^2)^(p/2)
// <= 1): every formula is a ratio in w / S0, so the factor cancels, and
// nothing overflows.  Since sum_i (z_i - Z) w_i = 0, ln d_i^2 may be taken
// relative to d2_min.  An exact hit passes g_j to dL/dz of its point only; a
// query without members contributes nothing.
//
// Two kernels share one record per sorted query:
//   1. per query (in cell order): hit and members, the sums, Z, dL/dq and
//      the query's share of dL/dp (a warp sum, then one FP64 atomic);
//   2. per data point (in cell order): walks the sorted queries whose disc
//      can reach it (the grid's coverage argument is symmetric in the two
//      points) with the same FP32 membership test, and sums dL/dz_i and
//      dL/dx_i in registers: one write per point, no atomics.
// FP32 throughout, except queries whose d2_min is below 2^-100 (or zero
// without a coincident point) or whose FP32 sums are not finite: those use
// FP64 on both sides.
// The record read for every (point, query) candidate is 16 bytes of FP32
// (FP64-to-FP32 conversions run at the FP64 rate on this part); queries on
// the FP64 path keep their values in a second array read only for them.
struct LocalGradRec {
  float d2min;  // the weights' scale (FP32 path): the members' smallest d^2, or
                // for the modified weights their largest base 1/d - 1/R
  float c;      // g_j / S0 (scaled), or g_j at an exact hit
  float z;      // Z_j
  int code;     // >= 0: exact hit (data index); -1: nothing; -2: FP32; -3: FP64
};
struct LocalGradRec64 {
  double d2min, c, z;  // FP64 path only
};
constexpr int kGradHitNone = -1, kGradF32 = -2, kGradF64 = -3;

// Scaled FP32 weight (d2min / d2)^(p/2); lmin = log2(d2min) for general p.
template <int MODE>
__device__ __forceinline__ float grad_weight(float d2, float d2min, float lmin, float hp) {
  if (MODE == kPow2) return __fmul_rn(d2min, rcp_approx(d2));
  return ex2_approx(-hp * (lg2_approx(d2) - lmin));
}

// The FP64 path of one query (weights scaled by its exact d2_min^(p/2)):
// dL/dq, its dL/dp share and the record the data-side kernel reads.  Out of
// line, so that the rare FP64 branch adds no registers to the FP32 loops.
struct GradF64 {
  float gqx, gqy;
  double gp;
  LocalGradRec64 rec;
};
// FP64 weight terms of one member at squared distance e2 under the scale:
// the weight w, the pair factor f (w / d^2, or for the modified weights
// w / (t d^3)) and the dL/dp log term (ln of d^2 / d2_min, or of t / t_max).
struct GradTerms64 {
  double w, f, l;
};
__device__ __forceinline__ GradTerms64 grad_terms64(double e2, double scale, double p,
                                                    bool modified, double radius) {
  if (!modified) {
    const double w = pow(scale / e2, 0.5 * p);
    return GradTerms64{w, w / e2, log(e2 / scale)};
  }
  const double d = sqrt(e2);
  const double t = isinf(radius) ? 1.0 / d : (radius - d) / (radius * d);
  if (!(t > 0.0)) return GradTerms64{0.0, 0.0, 0.0};
  const double w = pow(t / scale, p);
  return GradTerms64{w, w / (t * e2 * d), log(t / scale)};
}

__device__ __noinline__ GradF64 grad_query_f64(const Runs runs, const float4* sorted,
                                               float qx, float qy, float r2f, double p,
                                               float gj, bool modified, double radius) {
  double scale = modified ? 0.0 : INFINITY;  // d2_min, or the largest base t
  for (int rr = 0; rr < 5; ++rr)
    for (int k = runs.a[rr]; k < runs.b[rr]; ++k) {
      const float4 v = sorted[k];
      if (!(fp32_d2(qx, qy, v.x, v.y) < r2f)) continue;
      const double ex = double(qx) - v.x, ey = double(qy) - v.y, e2 = ex * ex + ey * ey;
      if (modified) {
        const double d = sqrt(e2);
        scale = fmax(scale, isinf(radius) ? 1.0 / d : (radius - d) / (radius * d));
      } else {
        scale = fmin(scale, e2);
      }
    }
  GradF64 r{0.f, 0.f, 0.0, LocalGradRec64{0.0, 0.0, 0.0}};
  if (!(scale > 0.0)) return r;  // no member of positive weight: no gradient
  double s0 = 0.0, s1 = 0.0;
  for (int rr = 0; rr < 5; ++rr)
    for (int k = runs.a[rr]; k < runs.b[rr]; ++k) {
      const float4 v = sorted[k];
      if (!(fp32_d2(qx, qy, v.x, v.y) < r2f)) continue;
      const double ex = double(qx) - v.x, ey = double(qy) - v.y;
      const double w = grad_terms64(ex * ex + ey * ey, scale, p, modified, radius).w;
      s0 += w;
      s1 += w * double(v.z);
    }
  const double Z = s1 / s0;
  double ax = 0.0, ay = 0.0, al = 0.0;
  for (int rr = 0; rr < 5; ++rr)
    for (int k = runs.a[rr]; k < runs.b[rr]; ++k) {
      const float4 v = sorted[k];
      if (!(fp32_d2(qx, qy, v.x, v.y) < r2f)) continue;
      const double ex = double(qx) - v.x, ey = double(qy) - v.y;
      const GradTerms64 g = grad_terms64(ex * ex + ey * ey, scale, p, modified, radius);
      const double dz = double(v.z) - Z;
      ax += dz * g.f * ex;
      ay += dz * g.f * ey;
      al += dz * g.w * g.l;
    }
  r.gqx = static_cast<float>(-double(gj) * p / s0 * ax);
  r.gqy = static_cast<float>(-double(gj) * p / s0 * ay);
  r.gp = (modified ? 1.0 : -0.5) * double(gj) * al / s0;
  r.rec = LocalGradRec64{scale, double(gj) / s0, Z};
  return r;
}

// (a / b)^p for the modified weights (lb = log2 b; p = 2 needs no log).
template <int MODE>
__device__ __forceinline__ float modified_ratio(float a, float b, float lb, float pf) {
  if (MODE == kPow2) {
    const float r = a * rcp_approx(b);
    return r * r;
  }
  return ex2_approx(pf * (lg2_approx(a) - lb));
}

// First pass of one query: hit, members, and the sums with weights scaled by
// the heaviest member so far (the smallest d^2, or for the modified weights
// the largest base 1/d - 1/R), rescaled as in an online softmax when a
// heavier one appears, so every scaled weight stays <= 1.  (sum w, sum w z)
// is a compensated pair, as in the forward pass: Z and g / S0 then stay
// accurate however many members a query has.
template <int MODE, int WMODE>
struct GradSums {
  static constexpr bool kMod = WMODE == kWeightModified;
  int best = INT_MAX, members = 0;
  float d2min = INFINITY, scale = kMod ? 0.f : INFINITY, lsc = 0.f;
  u64 hi = 0, lo = 0;

  __device__ __forceinline__ static float log_of(float s) {
    return MODE == kPow2 ? 0.f : lg2_approx(s);
  }
  __device__ __forceinline__ void consider(const float4 v, float qx, float qy, float r2f,
                                           float r2t, float inv_r, float hp, float pf) {
    const float d2 = fp32_d2(qx, qy, v.x, v.y);
    if (!(d2 < r2t)) return;
    if (v.x == qx && v.y == qy) {
      best = min(best, __float_as_int(v.w));
      return;
    }
    if (!(d2 < r2f)) return;
    ++members;
    d2min = fminf(d2min, d2);
    const float s = kMod ? fmaxf(rsqrt_approx(d2) - inv_r, 0.f) : d2;
    if (kMod && !(s > 0.f)) return;  // zero weight
    if (kMod ? s > scale : s < scale) {
      const float l = log_of(s);
      if (kMod ? scale > 0.f : members > 1) {
        // (t_old / t)^p, or (d2 / d2_old)^(p/2): the old sums shrink.
        const float f = kMod ? modified_ratio<MODE>(scale, s, l, pf)
                             : grad_weight<MODE>(scale, s, l, hp);
        hi = mul2(hi, pk(f, f));
        lo = mul2(lo, pk(f, f));
      }
      scale = s;
      lsc = l;
    }
    const float w = kMod ? modified_ratio<MODE>(s, scale, lsc, pf)
                         : grad_weight<MODE>(s, scale, lsc, hp);
    two_sum_acc(hi, lo, pk(w, __fmul_rn(w, v.z)));
  }
  // The lanes' sums over their shares of one query, joined: each lane's are
  // rescaled to the heaviest member of all, then added.
  __device__ __forceinline__ void join(float hp, float pf) {
    best = __reduce_min_sync(0xffffffffu, best);
    members = __reduce_add_sync(0xffffffffu, members);
    float top = scale;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      d2min = fminf(d2min, __shfl_xor_sync(0xffffffffu, d2min, o));
      const float other = __shfl_xor_sync(0xffffffffu, top, o);
      top = kMod ? fmaxf(top, other) : fminf(top, other);
    }
    const float l = log_of(top);
    if (kMod ? scale > 0.f && scale < top : scale < INFINITY && scale > top) {
      const float f = kMod ? modified_ratio<MODE>(scale, top, l, pf)
                           : grad_weight<MODE>(scale, top, l, hp);
      hi = mul2(hi, pk(f, f));
      lo = mul2(lo, pk(f, f));
    }
    scale = top;
    lsc = l;
    warp_sum_pairs(hi, lo);
  }
  __device__ __forceinline__ bool has_weight() const {
    return members > 0 && (!kMod || scale > 0.f);
  }
  // Z = (h1 + l1) / (h0 + l0): quotient, then one residual correction.
  __device__ __forceinline__ float value(float& s0) const {
    float h0, h1, l0, l1;
    upk(hi, h0, h1);
    upk(lo, l0, l1);
    s0 = h0 + l0;
    const float z0 = __fdiv_rn(h1, h0);
    return __fmaf_rn(__fadd_rn(__fmaf_rn(-z0, h0, h1), __fmaf_rn(-z0, l0, l1)), rcp_approx(h0), z0);
  }
};

// Second pass: the sums of dL/dq (x and y) and of the dL/dp share.
template <int MODE, int WMODE>
struct GradTerms {
  float ax = 0.f, ay = 0.f, al = 0.f;
  __device__ __forceinline__ void consider(const float4 v, float qx, float qy, float r2f,
                                           float inv_r, float hp, float pf, float Z, float scale,
                                           float lsc, float lsc2) {
    constexpr bool kMod = WMODE == kWeightModified;
    const float dx = __fsub_rn(qx, v.x), dy = __fsub_rn(qy, v.y);
    const float d2 = __fmaf_rn(dy, dy, __fmul_rn(dx, dx));
    if (!(d2 < r2f)) return;
    float w, ar, lt;
    if (kMod) {
      const float id = rsqrt_approx(d2);
      const float tb = fmaxf(id - inv_r, 0.f);
      if (!(tb > 0.f)) return;
      w = modified_ratio<MODE>(tb, scale, lsc, pf);
      ar = (v.z - Z) * w * (id * id) * (id * rcp_approx(tb));  // / (t d^3)
      lt = lg2_approx(tb) - lsc2;
    } else {
      w = grad_weight<MODE>(d2, scale, lsc, hp);
      ar = (v.z - Z) * w * rcp_approx(d2);  // / d^2
      lt = lg2_approx(d2) - lsc2;
    }
    ax = fmaf(ar, dx, ax);
    ay = fmaf(ar, dy, ay);
    al = fmaf((v.z - Z) * w, lt, al);
  }
};

// One query's result from its two passes (one lane): its record for the
// data-side kernel, dL/dq, and its share of dL/dp (returned).
template <int MODE, int WMODE>
__device__ __forceinline__ double grad_finish(const GradSums<MODE, WMODE>& sums,
                                              const GradTerms<MODE, WMODE>& terms, bool second,
                                              float Z, float s0, float gj, int j, int64_t t,
                                              const Runs& runs, const float4* sorted,
                                              float qx, float qy, float r2f, double p,
                                              double radius, float* __restrict__ grad_q,
                                              LocalGradRec* rec,
                                              LocalGradRec64* rec64) {
  constexpr bool kMod = WMODE == kWeightModified;
  LocalGradRec out{0.f, 0.f, 0.f, kGradHitNone};
  float gqx = 0.f, gqy = 0.f;
  double gp = 0.0;
  if (sums.best != INT_MAX) {
    out.code = sums.best;
    out.c = gj;
  } else if (sums.has_weight()) {
    bool f32 = second;
    if (second) {
      const float pf = static_cast<float>(p), c = gj / s0, k1 = c * pf;
      gqx = -k1 * terms.ax;
      gqy = -k1 * terms.ay;
      // dL/dp share in FP32 (no FP64 divide): -ln2/2 c al for d^-p,
      // +ln2 c al for the modified weights (dw/dp = w ln t).
      const float gpf = (kMod ? 0.6931471805599453f : -0.5f * 0.6931471805599453f) * c * terms.al;
      gp = gpf;
      out.code = kGradF32;
      out.c = c;
      out.z = Z;
      out.d2min = sums.scale;
      f32 = isfinite(Z) && isfinite(gqx) && isfinite(gqy) && isfinite(gpf) && isfinite(c);
    }
    if (!f32) {  // FP64: weights scaled by the exact scale
      const GradF64 r64 = grad_query_f64(runs, sorted, qx, qy, r2f, p, gj, kMod, radius);
      gqx = r64.gqx;
      gqy = r64.gqy;
      gp = r64.gp;
      out.code = r64.rec.c == 0.0 && r64.rec.d2min == 0.0 ? kGradHitNone : kGradF64;
      rec64[t] = r64.rec;
    }
  }
  rec[t] = out;
  if (grad_q) {
    grad_q[2 * int64_t(j)] = gqx;
    grad_q[2 * int64_t(j) + 1] = gqy;
  }
  return gp;
}

template <int MODE, int WMODE = kWeightShepard>
__global__ void __launch_bounds__(kLocalThreads)
    local_grad_query_kernel(const GridDev* grid, const float4* sorted,
                            int64_t n, const int32_t* starts,
                            const int32_t* base, const float4* qrec,
                            int64_t m, double p, float r2f, float r2t,
                            const float* grad_out, float* __restrict__ grad_q,
                            double* __restrict__ grad_p, LocalGradRec* rec,
                            LocalGradRec64* rec64, double radius, int64_t most,
                            unsigned* heavy_count, int32_t* heavy) {
  pdl_trigger();
  pdl_wait();
  const int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  double gp = 0.0;  // this query's share of dL/dp (every lane joins the warp sum)
  if (t < m) {
    const float4 r = qrec[t];
    const float qx = r.x, qy = r.y;
    const int j = __float_as_int(r.z);
    if (dcheck(j >= 0 && j < m, kSiteOutput)) {
      const Runs runs(*grid, qx, qy, starts, base);
      if (list_if_heavy(*grid, runs, n, m, most)) {
        list_heavy(t, m, heavy_count, heavy);
      } else {
        const float gj = grad_out[j];
        const float hp = static_cast<float>(0.5 * p), pf = static_cast<float>(p);
        const float inv_r = WMODE == kWeightModified ? static_cast<float>(1.0 / radius) : 0.f;
        GradSums<MODE, WMODE> sums;
#pragma unroll
        for (int rr = 0; rr < 5; ++rr)
#pragma unroll 4
          for (int k = runs.a[rr]; k < runs.b[rr]; ++k) {
            if (!dcheck(k >= 0 && k < n, kSiteGather)) break;
            sums.consider(sorted[k], qx, qy, r2f, r2t, inv_r, hp, pf);
          }
        // A query with members and no hit, in FP32's range, takes the second pass.
        const bool second =
            sums.best == INT_MAX && sums.has_weight() && sums.d2min >= 0x1p-100f;
        float s0 = 1.f, Z = 0.f;
        GradTerms<MODE, WMODE> terms;
        if (second) {
          Z = sums.value(s0);
          const float lsc2 = lg2_approx(sums.scale);
#pragma unroll
          for (int rr = 0; rr < 5; ++rr)
#pragma unroll 4
            for (int k = runs.a[rr]; k < runs.b[rr]; ++k)
              terms.consider(sorted[k], qx, qy, r2f, inv_r, hp, pf, Z, sums.scale, sums.lsc, lsc2);
        }
        gp = grad_finish<MODE, WMODE>(sums, terms, second, Z, s0, gj, j, t, runs, sorted, qx, qy,
                                      r2f, p, radius, grad_q, rec, rec64);
      }
    }
  }
  if (grad_p) {
    gp = warp_sum(gp);
    if ((threadIdx.x & 31) == 0 && gp != 0.0) atomicAdd(grad_p, gp);
  }
}

// The heavy queries' gradients, a warp each.
template <int MODE, int WMODE = kWeightShepard>
__global__ void __launch_bounds__(kHeavyThreads)
    local_grad_heavy_kernel(const GridDev* grid, const float4* sorted,
                            int64_t n, const int32_t* starts,
                            const int32_t* base, const float4* qrec,
                            int64_t m, double p, float r2f, float r2t,
                            const float* grad_out, float* __restrict__ grad_q,
                            double* __restrict__ grad_p, LocalGradRec* rec,
                            LocalGradRec64* rec64, double radius,
                            const unsigned* heavy_count,
                            const int32_t* heavy) {
  pdl_trigger();
  pdl_wait();
  const int64_t count = *heavy_count;
  const int lane = threadIdx.x & 31;
  const int64_t warps = int64_t(gridDim.x) * (kHeavyThreads / 32);
  const float hp = static_cast<float>(0.5 * p), pf = static_cast<float>(p);
  const float inv_r = WMODE == kWeightModified ? static_cast<float>(1.0 / radius) : 0.f;
  double gp = 0.0;  // lane 0: this warp's queries' shares of dL/dp
  for (int64_t w = (int64_t(blockIdx.x) * kHeavyThreads + threadIdx.x) / 32; w < count;
       w += warps) {
    const int64_t t = heavy[w];
    if (!dcheck(t >= 0 && t < m, kSiteScatter)) continue;
    const float4 r = qrec[t];
    const float qx = r.x, qy = r.y;
    const int j = __float_as_int(r.z);
    if (!dcheck(j >= 0 && j < m, kSiteOutput)) continue;
    const Runs runs(*grid, qx, qy, starts, base);
    const FlatRuns fr(runs);
    GradSums<MODE, WMODE> sums;
#pragma unroll 2
    for (int i = lane; i < fr.total(); i += 32) {
      const int k = fr.at(i);
      if (!dcheck(k >= 0 && k < n, kSiteGather)) break;
      sums.consider(sorted[k], qx, qy, r2f, r2t, inv_r, hp, pf);
    }
    sums.join(hp, pf);
    const bool second = sums.best == INT_MAX && sums.has_weight() && sums.d2min >= 0x1p-100f;
    float s0 = 1.f, Z = 0.f;
    GradTerms<MODE, WMODE> terms;
    if (second) {  // the same in every lane
      Z = sums.value(s0);
      const float lsc2 = lg2_approx(sums.scale);
#pragma unroll 2
      for (int i = lane; i < fr.total(); i += 32)
        terms.consider(sorted[fr.at(i)], qx, qy, r2f, inv_r, hp, pf, Z, sums.scale, sums.lsc, lsc2);
      terms.ax = warp_sum(terms.ax);
      terms.ay = warp_sum(terms.ay);
      terms.al = warp_sum(terms.al);
    }
    if (lane == 0)
      gp += grad_finish<MODE, WMODE>(sums, terms, second, Z, s0, grad_out[j], j, t, runs, sorted, qx,
                                     qy, r2f, p, radius, grad_q, rec, rec64);
  }
  if (grad_p && lane == 0 && gp != 0.0) atomicAdd(grad_p, gp);
}

// The FP64 path's share of one (point, query) pair: (dL/dz, dL/dx, dL/dy).
// Out of line, so that the rare FP64 branch adds no registers to the loop.
// One instance per weight mode, so the plain one passes no radius.
__device__ __forceinline__ float3 grad_pair_f64_terms(LocalGradRec64 D, float qx, float qy,
                                                      float4 v, double p, bool modified,
                                                      double radius) {
  const double ex = double(qx) - v.x, ey = double(qy) - v.y;
  const GradTerms64 g = grad_terms64(ex * ex + ey * ey, D.d2min, p, modified, radius);
  const double a = D.c * p * (double(v.z) - D.z) * g.f;
  return make_float3(static_cast<float>(D.c * g.w), static_cast<float>(a * ex),
                     static_cast<float>(a * ey));
}
__device__ __noinline__ float3 grad_pair_f64(LocalGradRec64 D, float qx, float qy, float4 v,
                                             double p) {
  return grad_pair_f64_terms(D, qx, qy, v, p, false, 0.0);
}
__device__ __noinline__ float3 grad_pair_f64_modified(LocalGradRec64 D, float qx, float qy,
                                                      float4 v, double p, double radius) {
  return grad_pair_f64_terms(D, qx, qy, v, p, true, radius);
}

template <int MODE, int WMODE = kWeightShepard>
__global__ void __launch_bounds__(kLocalThreads)
    local_grad_data_kernel(const GridDev* grid, const float4* sorted,
                           int64_t n, const int32_t* starts_d,
                           const int32_t* base_d,
                           const int32_t* starts_q,
                           const int32_t* base_q, const float4* qrec,
                           int64_t m, const LocalGradRec* rec,
                           const LocalGradRec64* rec64, double p, float r2f,
                           float* __restrict__ grad_z, float* __restrict__ grad_xy,
                           double radius) {
  pdl_trigger();
  pdl_wait();
  constexpr bool kMod = WMODE == kWeightModified;
  const int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  const GridDev g = *grid;
  if (k >= cell_start(starts_d, base_d, g.cells, g.cells)) return;  // placed (finite) points
  if (!dcheck(k < n, kSiteGather)) return;
  const float4 v = sorted[k];
  const int idx = __float_as_int(v.w);
  if (!dcheck(idx >= 0 && idx < n, kSiteData)) return;
  const Runs runs(g, v.x, v.y, starts_q, base_q);
  const float hp = static_cast<float>(0.5 * p), pf = static_cast<float>(p);
  const float inv_r = kMod ? static_cast<float>(1.0 / radius) : 0.f;
  float gz = 0.f, gx = 0.f, gy = 0.f;
  // Loads in flight: four, or two where the modified weights need the registers
  // (2^20 points, clustered queries, R for 32 members: 1260 us by four, 1200 by
  // two; the plain weights' whole call 1310 and 1370).
  constexpr int kAhead = kMod ? 2 : 4;
#pragma unroll
  for (int rr = 0; rr < 5; ++rr)
#pragma unroll kAhead
    for (int t = runs.a[rr]; t < runs.b[rr]; ++t) {
      if (!dcheck(t >= 0 && t < m, kSiteGather)) break;
      const LocalGradRec R = rec[t];  // both loads issue before any branch
      const float4 q = qrec[t];
      if (R.code == kGradHitNone) continue;
      if (R.code >= 0) {
        if (R.code == idx) gz += R.c;
        continue;
      }
      const float dx = __fsub_rn(q.x, v.x), dy = __fsub_rn(q.y, v.y);
      const float d2 = __fmaf_rn(dy, dy, __fmul_rn(dx, dx));
      if (!(d2 < r2f)) continue;  // the query's membership test, bit for bit
      if (R.code == kGradF32) {
        const float lsc = MODE == kPow2 ? 0.f : lg2_approx(R.d2min);
        float w, fac;
        if (kMod) {  // the scale is the query's largest base t
          const float id = rsqrt_approx(d2);
          const float tb = fmaxf(id - inv_r, 0.f);
          if (!(tb > 0.f)) continue;
          w = modified_ratio<MODE>(tb, R.d2min, lsc, pf);
          fac = (id * id) * (id * rcp_approx(tb));  // 1 / (t d^3)
        } else {
          w = grad_weight<MODE>(d2, R.d2min, lsc, hp);
          fac = rcp_approx(d2);  // 1 / d^2
        }
        gz = fmaf(R.c, w, gz);
        const float a = R.c * pf * (v.z - R.z) * w * fac;
        gx = fmaf(a, dx, gx);
        gy = fmaf(a, dy, gy);
      } else {
        const float3 f = kMod ? grad_pair_f64_modified(rec64[t], q.x, q.y, v, p, radius)
                              : grad_pair_f64(rec64[t], q.x, q.y, v, p);
        gz += f.x;
        gx += f.y;
        gy += f.z;
      }
    }
  if (grad_z) grad_z[idx] = gz;
  if (grad_xy) {
    grad_xy[2 * int64_t(idx)] = gx;
    grad_xy[2 * int64_t(idx) + 1] = gy;
  }
}

// ------------------------------------------------------------- k-NN form
//
// One thread per query, in cell order, grows a square of cells around the
// grid cell nearest to it (radius 0, 1, 2, 3, 4, 6, 9, ...: r += max(1, r/2),
// the step halved while the added cells would hold more than 4k points; the
// cells added at each step are walked as row runs) and keeps the k
// smallest keys in a max-heap in shared memory.  A key is the FP32 d^2's
// bits (non-negative, so they order as an unsigned integer) above the data
// index: one 64-bit compare ranks by (d^2, index).  After each step the
// search stops once the k-th key's d^2 is below a lower bound on the d^2 of
// any point not yet seen.  Such a point lies in the grid's box and outside
// the square, beyond one of its sides that still has grid cells; with ax, ay
// the query's distance to the box along each axis and D the distance to
// that side (cell units, each minus a margin mg = (|u| + |v|) 2^-22 + 2^-9
// for the cell-position errors), its true distance is at least
// h sqrt(max(ax, D)^2 + ay^2) (or the y analogue), and its FP32 d^2 at least
// that squared times (1 - 2^-18), minus 2^-126.  The bound is strict, so an
// unseen point can neither beat nor tie the k-th key.

// One warp per block: a block whose slowest query is still searching holds
// only its own warp's heaps in shared memory.
constexpr int kKnnThreads = 32;

__device__ __forceinline__ u64 knn_key(float d2, int idx) {
  return (u64(__float_as_uint(d2)) << 32) | u64(unsigned(idx));
}
__device__ __forceinline__ float key_d2(u64 key) { return __uint_as_float(unsigned(key >> 32)); }
__device__ __forceinline__ int key_index(u64 key) { return int(unsigned(key)); }

// 4-ary max-heap of this thread's keys: slot s at h[s * kKnnThreads]
// (conflict-free); the children of slot a are 4a + 1 .. 4a + 4, so a sift
// is at most 3 levels deep for k <= 64 and each level's loads issue together.
struct KnnHeap {
  u64* h;
  int size = 0;

  __device__ __forceinline__ u64 top() const { return h[0]; }
  __device__ __forceinline__ void push(u64 key) {
    int at = size++;
    while (at > 0) {
      const int parent = (at - 1) >> 2;
      const u64 pk = h[parent * kKnnThreads];
      if (pk >= key) break;
      h[at * kKnnThreads] = pk;
      at = parent;
    }
    h[at * kKnnThreads] = key;
  }
  // Replaces the largest key by a smaller one (keys are distinct).
  __device__ __forceinline__ void replace_top(u64 key, int n) { sift_down(0, key, n); }
  // Puts `key` at slot `at` of the first n slots and sifts it down, the
  // subtree below `at` being a heap already.
  __device__ __forceinline__ void sift_down(int at, u64 key, int n) {
    for (;;) {
      const int c0 = 4 * at + 1;
      if (c0 >= n) break;
      u64 bk = h[c0 * kKnnThreads];
      int big = c0;
#pragma unroll
      for (int c = 1; c < 4; ++c) {
        if (c0 + c < n) {
          const u64 ck = h[(c0 + c) * kKnnThreads];
          if (ck > bk) {
            bk = ck;
            big = c0 + c;
          }
        }
      }
      if (bk <= key) break;
      h[at * kKnnThreads] = bk;
      at = big;
    }
    h[at * kKnnThreads] = key;
  }
  // Floyd's bottom-up construction of a heap over the first n slots.
  __device__ void heapify(int n) {
    for (int a = (n - 2) >> 2; a >= 0; --a) sift_down(a, h[a * kKnnThreads], n);
  }
};

// Writes one query's k-NN result from its heap: Z (the z of the lowest
// coincident index, or Eq. 1 over the selection with compensated FP32 sums,
// or FP64 when those leave FP32's range; NaN when nothing is selected), the
// hit index, the k-th key's d^2 and the neighbour row (key order when
// sort_rows, else heap order).  Shared by both search kernels.
template <int MODE>
__device__ __forceinline__ void knn_write_result(KnnHeap& hp, int best_hit, float qx, float qy,
                                                 int j, const float* data,
                                                 int64_t n, double p, int k,
                                                 float* __restrict__ out,
                                                 int32_t* nbr_out,
                                                 float* __restrict__ kd2_out,
                                                 int32_t* hit_out, bool sort_rows) {
  const int size = hp.size;
  if (kd2_out) kd2_out[j] = size > 0 ? key_d2(hp.top()) : __int_as_float(0x7fc00000);
  float zv = __int_as_float(0x7fc00000);  // NaN: nothing selected
  if (best_hit != INT_MAX) {
    if (dcheck(best_hit >= 0 && best_hit < n, kSiteData)) zv = data[3 * int64_t(best_hit) + 2];
  } else if (size > 0) {
    const float hpw = static_cast<float>(0.5 * p), nhp = -hpw;
    u64 hi = 0, lo = 0;
    for (int s = 0; s < size; ++s) {
      const u64 key = hp.h[s * kKnnThreads];
      const float w = local_weight<MODE>(key_d2(key), hpw, nhp);
      two_sum_acc(hi, lo, pk(w, __fmul_rn(w, data[3 * int64_t(key_index(key)) + 2])));
    }
    float h0, h1, l0, l1;
    upk(hi, h0, h1);
    upk(lo, l0, l1);
    if (h0 >= kTinyPerMember * float(size) && h0 <= FLT_MAX && fabsf(h1) <= FLT_MAX &&
        fabsf(l1) <= FLT_MAX) {
      const float z0 = __fdiv_rn(h1, h0);
      const float res = __fadd_rn(__fmaf_rn(-z0, h0, h1), __fmaf_rn(-z0, l0, l1));
      zv = __fmaf_rn(res, rcp_approx(h0), z0);
    } else {
      // Outside FP32's range: FP64 over the selected points, scaled by
      // d2_min^(p/2).
      double dmin = INFINITY;
      for (int s = 0; s < size; ++s) {
        const float* x = data + 3 * int64_t(key_index(hp.h[s * kKnnThreads]));
        const double ex = double(qx) - x[0], ey = double(qy) - x[1];
        dmin = fmin(dmin, ex * ex + ey * ey);
      }
      double s0 = 0.0, s1 = 0.0;
      for (int s = 0; s < size; ++s) {
        const float* x = data + 3 * int64_t(key_index(hp.h[s * kKnnThreads]));
        const double ex = double(qx) - x[0], ey = double(qy) - x[1];
        const double w = pow(dmin / (ex * ex + ey * ey), 0.5 * p);
        s0 += w;
        s1 += w * double(x[2]);
      }
      zv = static_cast<float>(s1 / s0);
    }
  }
  out[j] = zv;
  if (hit_out) hit_out[j] = best_hit != INT_MAX ? best_hit : -1;
  if (nbr_out) {
    int32_t* row = nbr_out + int64_t(j) * k;
    for (int s = size; s < k; ++s) row[s] = -1;
    if (!sort_rows) {  // the selection in heap order (the gradient needs no order)
      for (int s = 0; s < size; ++s) row[s] = key_index(hp.h[s * kKnnThreads]);
      return;
    }
    // Heap sort: the largest remaining key goes to the end of the row.
    for (int n = size; n > 0; --n) {
      const u64 top = hp.top();
      row[n - 1] = key_index(top);
      const u64 last = hp.h[(n - 1) * kKnnThreads];
      if (n > 1) hp.replace_top(last, n - 1);
    }
  }
}

// Whether one thread should search for a query in cell (cx, cy) (kEasy).  With
// ca cells per point, the square of radius re = ceil((sqrt(2 k ca) - 1) / 2)
// holds 2k points at the mean density.  Where the square one cell wider holds
// fewer than k, the search has empty space to cross (kSparse); where the square
// holds over 8k + 64, it has a dense cluster to sift (kDense); a thread takes
// ten to a hundred times as long over such a query as over one at the mean
// density, and its warp waits.  (n = 2^20 points in 64 blobs, 100,000 uniform
// queries, k = 8: 1.09 ms when every query was one thread's.)
enum KnnSurroundings : int { kEasy, kSparse, kDense };
__device__ __forceinline__ KnnSurroundings knn_surroundings(const GridDev& g, const int32_t* sat,
                                                            float cells_per_point, int cx, int cy,
                                                            int k) {
  const int re = knn_square(cells_per_point, k);
  const int W = g.gx + 1;
  int c[2];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int rr = re + i;
    const int ya = max(0, cy - rr), yb = min(g.gy - 1, cy + rr);
    const int xa = max(0, cx - rr), xb = min(g.gx - 1, cx + rr);
    if (!dcheck(ya >= 0 && xa >= 0 && yb < g.gy && xb < g.gx, kSiteTable)) return kEasy;
    c[i] = sat[(yb + 1) * W + xb + 1] - sat[ya * W + xb + 1] - sat[(yb + 1) * W + xa] +
           sat[ya * W + xa];
  }
  return c[1] < k ? kSparse : c[0] > knn_dense(k) ? kDense : kEasy;
}

// Queries set apart from the single-thread search, in one array of m entries.
// The hard ones (not easy) are listed from the front, for warps.  Those that
// the search by counts leaves are listed from the back: up to `few` of them go
// to warps, more to a thread each.
struct KnnLists {
  unsigned *hard, *left;  // the lists' lengths
  int32_t* query;
  unsigned few;
};

// Whether the data fill their box about evenly: their cells hold at least 70%
// as many points' cells as evenly random points would (uniform data: 100%; 64
// blobs: about 10%).  Decides, on the device, between the search by counts and
// the heap search; on clustered data the former lists too many queries (64
// blobs, n = m = 2^20, k = 32: 3130 us against 2810 by heaps).
__device__ __forceinline__ bool knn_even(const GridDev& g, int64_t n) {
  const float cells = float(g.cells);
  const float expected = cells * (1.f - ex2_approx(-1.44269504f * float(n) * rcp_approx(cells)));
  return float(g.filled + 1u) >= 0.7f * expected;
}

// Whether the search by counts runs: on even data, unless most queries lie
// beyond the grid's edge, where its discs find nothing (100,000 queries up to a
// box width outside, k = 32: 432 us a call, 330 by heaps).
__device__ __forceinline__ bool knn_by_counts(const GridDev& g, int64_t n) {
  return knn_even(g, n) && 2 * g.beyond <= kSampleQueries;
}

// The queries that the heap search lists for warps.
struct KnnListed {
  bool sparse, dense, beyond;  // in such surroundings; two cells beyond the grid's edge
};

// Query t, by one thread (no block-wide barrier; `return`s are its own).
template <int MODE, bool LIST>
__device__ __forceinline__ void knn_thread_query(
    const GridDev* grid, const float4* sorted, const int32_t* starts, const int32_t* base,
    const int32_t* bpre, const int32_t* sat, const float4* qrec, const float* data, int64_t n,
    int64_t m, double p, int k, float* __restrict__ out, int32_t* nbr_out,
    float* __restrict__ kd2_out, int32_t* hit_out, bool sort_rows, const KnnLists& lists,
    KnnListed listed, int64_t t) {
  extern __shared__ __align__(16) unsigned char knn_smem[];
  KnnHeap hp;
  hp.h = reinterpret_cast<u64*>(knn_smem) + threadIdx.x;
  const GridDev g = *grid;
  const float4 rq = qrec[t];
  const float qx = rq.x, qy = rq.y;
  const int j = __float_as_int(rq.z);
  if (!dcheck(j >= 0 && j < m, kSiteOutput)) return;
  int best_hit = INT_MAX;
  u64 worst = ~u64(0);  // the heap's largest key once it holds k, else above every key

  auto run = [&](int yy, int xa, int xb) {
    const int a = cell_start(starts, base, yy * g.gx + xa, g.cells);
    const int b = cell_start(starts, base, yy * g.gx + xb + 1, g.cells);
    // Each candidate's record is loaded one iteration ahead, so that its
    // latency overlaps the previous candidate's heap work.
    float4 nv = make_float4(0.f, 0.f, 0.f, 0.f);
    if (a < b && dcheck(a >= 0 && a < n, kSiteGather)) nv = sorted[a];
    for (int q = a; q < b; ++q) {
      if (!dcheck(q >= 0 && q < n, kSiteGather)) break;
      const float4 v = nv;
      if (q + 1 < b && dcheck(q + 1 < n, kSiteGather)) nv = sorted[q + 1];
      const float d2 = fp32_d2(qx, qy, v.x, v.y);
      const int idx = __float_as_int(v.w);
      if (d2 == 0.f && v.x == qx && v.y == qy) best_hit = min(best_hit, idx);
      const u64 key = knn_key(d2, idx);
      if (key < worst) {  // worst stays ~0 (all ones) until the heap is full
        if (!dcheck(hp.size <= k && idx >= 0 && idx < n, kSiteHeap)) continue;
        if (hp.size < k) {
          hp.push(key);
          if (hp.size == k) worst = hp.top();
        } else {
          hp.replace_top(key, k);
          worst = hp.top();
        }
      }
    }
  };

  if (finite2(qx, qy)) {
    const float u = cell_pos(qx, g.hx0, g.inv2), v = cell_pos(qy, g.hy0, g.inv2);
    const int cx = clamp_floor(u, 0, g.gx - 1), cy = clamp_floor(v, 0, g.gy - 1);
    if (LIST) {
      const KnnSurroundings at =
          knn_surroundings(g, sat, float(g.cells) * rcp_approx(float(n)), cx, cy, k);
      // One branch, so that the warp comes together again behind it.
      const bool away = (listed.sparse & (at == kSparse)) | (listed.dense & (at == kDense)) |
                        (listed.beyond & beyond_grid(g, u, v, 2.f));
      if (away) {
        list_heavy(t, m, lists.hard, lists.query);
        return;
      }
    }
    const float mg = __fmaf_ru(fabsf(u) + fabsf(v), 0x1p-22f, 0x1p-9f);
    const float ax = fmaxf(0.f, fmaxf(u - float(g.gx), -u) - mg);
    const float ay = fmaxf(0.f, fmaxf(v - float(g.gy), -v) - mg);
    const float hh = g.inv2 > 0.f ? 2.f / g.inv2 : 0.f;
    const float h2 = __fmul_rd(hh, hh) * (1.f - 0x1p-18f);
    const float ih2 = __frcp_ru(h2);  // +inf for the one-cell grid: nothing is clipped
    // Once the heap holds k keys, a cell can only matter if the stop test's
    // lower bound for its points, (gap_x^2 + gap_y^2) h2 - 2^-126 with each
    // gap reduced by mg, is at most the k-th key's d^2: gap_x^2 + gap_y^2 <=
    // reach2() (rounded up; +inf or NaN clips nothing).
    auto reach2 = [&]() {
      return __fmul_ru(__fadd_ru(key_d2(worst), 0x1p-126f), ih2);
    };
    // Narrows a range [lo, hi] to the cells t whose gap from c (reduced by
    // mg) is at most e: t <= c + mg + e and t + 1 >= c - mg - e, rounded
    // outwards.  An empty range is left as it is; otherwise the result lies
    // in [lo, hi] or is empty (lo > hi).  NaN bounds clip nothing.
    auto clip = [&](float c, float e, int& lo, int& hi) {
      if (lo > hi) return;
      const float a = ceilf(__fsub_rd(__fsub_rd(__fsub_rd(c, mg), e), 1.f));
      const float b = floorf(__fadd_ru(__fadd_ru(c, mg), e));
      const int nlo = int(fminf(fmaxf(float(lo), a), float(hi) + 1.f));
      const int nhi = int(fmaxf(fminf(float(hi), b), float(lo) - 1.f));
      lo = nlo;
      hi = nhi;
    };
    // Points in the square of radius rr around (cx, cy), from the table.
    auto square_count = [&](int rr) {
      const int ya = max(0, cy - rr), yb = min(g.gy - 1, cy + rr);
      const int xa = max(0, cx - rr), xb = min(g.gx - 1, cx + rr);
      const int W = g.gx + 1;
      if (!dcheck(ya >= 0 && xa >= 0 && yb < g.gy && xb < g.gx, kSiteTable)) return 0;
      return sat[(yb + 1) * W + xb + 1] - sat[ya * W + xb + 1] - sat[(yb + 1) * W + xa] +
             sat[ya * W + xa];
    };
    int in_square = -1;  // points in the square of radius r, once counted
    // r = -1 stands for the query's own cell; then square r grows to r2.
    for (int r = -1;;) {
      if (r >= 0) {
        const bool open_l = cx - r > 0, open_r = cx + r < g.gx - 1;
        const bool open_b = cy - r > 0, open_t = cy + r < g.gy - 1;
        if (!(open_l || open_r || open_b || open_t)) break;  // the square covers the grid
        if (hp.size == k) {
          float l2 = INFINITY;
          if (open_l) {
            const float dx = fmaxf(ax, fmaxf(0.f, (u - float(cx - r)) - mg));
            l2 = fminf(l2, __fmaf_rd(dx, dx, __fmul_rd(ay, ay)));
          }
          if (open_r) {
            const float dx = fmaxf(ax, fmaxf(0.f, (float(cx + r + 1) - u) - mg));
            l2 = fminf(l2, __fmaf_rd(dx, dx, __fmul_rd(ay, ay)));
          }
          if (open_b) {
            const float dy = fmaxf(ay, fmaxf(0.f, (v - float(cy - r)) - mg));
            l2 = fminf(l2, __fmaf_rd(dy, dy, __fmul_rd(ax, ax)));
          }
          if (open_t) {
            const float dy = fmaxf(ay, fmaxf(0.f, (float(cy + r + 1) - v) - mg));
            l2 = fminf(l2, __fmaf_rd(dy, dy, __fmul_rd(ax, ax)));
          }
          if (key_d2(worst) < __fmul_rd(l2, h2) - 0x1p-126f) break;
        }
      }
      // Grow by max(1, r/2), halved while the band would hold more than 4k
      // points (a step from empty space into a dense cluster stays short).
      // From r = 4 on (steps of 2 or more), the band's count comes from the
      // summed-area table and an empty band is not walked.
      int r2 = r + max(1, r >> 1);
      bool walk = true;
      if (r >= 4) {
        if (in_square < 0) in_square = square_count(r);
        int c2 = square_count(r2);
        while (c2 - in_square > 4 * k && r2 > r + 1) {
          r2 = r + max(1, (r2 - r) >> 1);
          c2 = square_count(r2);
        }
        walk = c2 != in_square;
        in_square = c2;
      }
      // The cells between squares r and r2 in four parts: the side strips of
      // the rows already in the square, then the new rows below and above.
      // One loop walks every part, so the candidate code exists once.
#pragma unroll 1
      for (int part = 0; walk && part < 4; ++part) {
        int ya, yb, xa, xb;
        if (r < 0) {
          if (part > 0) break;
          ya = yb = cy;
          xa = xb = cx;
        } else if (part < 2) {
          ya = max(0, cy - r);
          yb = min(g.gy - 1, cy + r);
          xa = part == 0 ? max(0, cx - r2) : cx + r + 1;
          xb = part == 0 ? cx - r - 1 : min(g.gx - 1, cx + r2);
        } else {
          xa = max(0, cx - r2);
          xb = min(g.gx - 1, cx + r2);
          ya = part == 2 ? max(0, cy - r2) : cy + r + 1;
          yb = part == 2 ? cy - r - 1 : min(g.gy - 1, cy + r2);
        }
        if (xa > xb || ya > yb) continue;  // then 0 <= ya <= yb < gy, 0 <= xa <= xb < gx
        // With a full heap, rows and columns beyond the k-th key's reach are
        // dropped first (the ranges only narrow, or empty).
        if (hp.size == k) {
          const float e = __fsqrt_ru(reach2());
          clip(v, e, ya, yb);
          clip(u, e, xa, xb);
          if (xa > xb || ya > yb) continue;
        }
        // Once the square is 8 cells out, each stretch of 8 rows whose
        // occupancy blocks over xa..xb hold no point is skipped.
        const bool check_blocks = r >= 8;
        for (int y8 = ya; y8 <= yb;) {
          const int y1 = check_blocks ? min(yb, y8 | 7) : yb;
          bool occupied = true;
          if (check_blocks) {
            const int by = y8 >> kBlockShift;
            const int32_t* bp = bpre + by * (kMaxBlocksPerAxis + 1);
            occupied = dcheck(by < kMaxBlocksPerAxis && (xb >> kBlockShift) < kMaxBlocksPerAxis,
                              kSiteBlock) &&
                       bp[(xb >> kBlockShift) + 1] != bp[xa >> kBlockShift];
          }
          for (int yy = y8; occupied && yy <= y1; ++yy) {
            int ra = xa, rb = xb;
            if (hp.size == k) {  // the columns this row's chord reaches
              const float gap = fmaxf(0.f, fmaxf(float(yy) - v, v - float(yy + 1)) - mg);
              const float w2 = reach2(), g2 = __fmul_rd(gap, gap);
              if (g2 > w2) continue;
              clip(u, __fsqrt_ru(__fsub_ru(w2, g2)), ra, rb);
              if (ra > rb) continue;
            }
            run(yy, ra, rb);
          }
          y8 = y1 + 1;
        }
      }
      r = r2;
    }
  }
  knn_write_result<MODE>(hp, best_hit, qx, qy, j, data, n, p, k, out, nbr_out, kd2_out, hit_out,
                         sort_rows);
}

// At most 64 registers (32 one-warp blocks per SM); left to itself the
// compiler settles on fewer and spills.  With LIST, hard queries are listed;
// but those in dense surroundings only if they are not most of them, or few:
// neighbouring threads sift a cluster together, which a warp per query does
// again for each (64 blobs, n = 2^20, queries in the blobs too, threads / warps:
// m = 500,000 k = 8 520 / 1605 us, k = 32 880 / 1826; m = 100,000 293 / 440 and
// 391 / 554; m = 30,000 252 / 235 and 393 / 155).  FROM says which queries it
// takes: all of them, a block's 32 each; or, after the search by counts, those
// that it left, if they are not few, and all of them where it does not run.  In
// the last form the blocks, as many as fit the GPU, fetch groups of 32 queries
// from a counter: 32,768 blocks that return at once take 34 us.
enum KnnFrom : int { kFromAll, kFromLeft, kFromLeftFetched };
template <int MODE, bool LIST, int FROM>
__global__ void __maxnreg__(64)
    knn_query_kernel(const GridDev* grid, const float4* sorted,
                     const int32_t* starts, const int32_t* base,
                     const int32_t* bpre, const int32_t* sat,
                     const float4* qrec, const float* data, int64_t n,
                     int64_t m,
                     double p, int k, float* __restrict__ out, int32_t* nbr_out,
                     float* __restrict__ kd2_out, int32_t* hit_out,
                     bool sort_rows, const KnnLists lists, unsigned* next) {
  pdl_trigger();
  pdl_wait();
  const bool counted = FROM != kFromAll && knn_by_counts(*grid, n);
  int64_t count = m;
  if (counted) {
    count = *lists.left;
    if (count <= lists.few) return;
  }
  KnnListed listed{false, false, false};
  if (LIST && !counted) {
    listed.sparse = true;
    listed.beyond = m <= kUnsortedKnn;
    listed.dense = m <= lists.few ||
                   (k >= kSampleK && grid->dense * m <= int64_t(kSampleQueries) * lists.few);
  }
  constexpr bool fetch = FROM == kFromLeftFetched;
  const int lane = threadIdx.x;
  int64_t group = blockIdx.x;
  for (;;) {
    if (fetch) {
      unsigned fetched = 0;
      if (lane == 0) fetched = atomicAdd(next, 1u);
      group = __shfl_sync(0xffffffffu, fetched, 0);
    }
    int64_t t = group * kKnnThreads + lane;
    if (fetch && group * kKnnThreads >= count) break;
    if (t < count) {
      if (counted) t = lists.query[m - 1 - t];
      if (dcheck(t >= 0 && t < m, kSiteScatter))
        knn_thread_query<MODE, LIST>(grid, sorted, starts, base, bpre, sat, qrec, data, n, m, p, k,
                                     out, nbr_out, kd2_out, hit_out, sort_rows, lists, listed, t);
    }
    if (!fetch) break;
    __syncwarp();
  }
}

// ------------------------------------------------- k-NN, one thread, by counts
//
// The search for calls that want no neighbour lists, on queries whose
// surroundings are of even density (others are left to the two searches below
// and above, see KnnLists):
// 1. the summed-area table's count over a square of cells gives the local
//    density, and with it a disc expected to hold the k nearest with a margin
//    of four standard deviations of their number;
// 2. the candidates the disc's cells hold are counted by d^2 into kBins equal
//    bins, which are the lane's own column in shared memory; the bin in which
//    the count reaches k bounds the k-th key;
// 3. the cells within that bound are walked again: candidates of lower bins
//    are summed at once (z is in the record), those of that bin are kept
//    aside, and the smallest of them complete the k.
// A disc that turns out to hold fewer than k points is tried again at 2.5
// times the area, twice; then, or when more than kAside candidates share the
// bin, the query is listed.  The selection is that of the other searches: the
// bin is a monotone function of d^2 and ties are settled by (d^2, index).
//
// Against the heap search: no heap and no second gather of z, 8300 warp
// instructions per 32 queries at k = 32 (17,000) with 17 of 32 lanes active
// (12).  Bound by the latency of the candidate loads (26 warps an SM, which
// the counters' 7 KB a warp allow).  Uniform n = m = 2^20, k = 32: 693 us by
// heaps, 450 us.
constexpr int kBins = 32;
constexpr int kAside = 8;
constexpr int kCountThreads = 64;

template <int MODE>
__global__ void __launch_bounds__(kCountThreads)
    knn_count_kernel(const GridDev* grid, const float4* sorted, const int32_t* starts,
                     const int32_t* base, const int32_t* sat, const float4* qrec,
                     const float* data, int64_t n, int64_t m, double p, int k,
                     float* __restrict__ out, float* __restrict__ kd2_out,
                     const KnnLists lists) {
  pdl_trigger();
  pdl_wait();
  __shared__ int bins[kBins][kCountThreads];
  __shared__ u64 aside_key[kAside][kCountThreads];
  __shared__ float aside_z[kAside][kCountThreads];
  const int lane = threadIdx.x;
  const int64_t t = int64_t(blockIdx.x) * kCountThreads + lane;
  const GridDev g = *grid;
  // No block-wide barrier in this kernel: a lane reads its own columns.
  if (t >= m || !knn_by_counts(g, n)) return;
  const float4 rq = qrec[t];
  const float qx = rq.x, qy = rq.y;
  const int j = __float_as_int(rq.z);
  if (!dcheck(j >= 0 && j < m, kSiteOutput)) return;
  if (!finite2(qx, qy)) {
    out[j] = __int_as_float(0x7fc00000);
    if (kd2_out) kd2_out[j] = __int_as_float(0x7fc00000);
    return;
  }
  const float u = cell_pos(qx, g.hx0, g.inv2), v = cell_pos(qy, g.hy0, g.inv2);
  const int cx = clamp_floor(u, 0, g.gx - 1), cy = clamp_floor(v, 0, g.gy - 1);
  const float mg = __fmaf_ru(fabsf(u) + fabsf(v), 0x1p-22f, 0x1p-9f);
  const float hh = g.inv2 > 0.f ? 2.f / g.inv2 : 0.f;
  const float h2 = __fmul_rd(hh, hh) * (1.f - 0x1p-18f);
  const float ih2 = __frcp_ru(h2);

  // Points per cell around the query, from the square that holds 2k points
  // at the mean density.
  const float ca = float(g.cells) * rcp_approx(float(n));
  const int re = knn_square(ca, k);
  const int ya = max(0, cy - re), yb = min(g.gy - 1, cy + re);
  const int xa = max(0, cx - re), xb = min(g.gx - 1, cx + re);
  const int W = g.gx + 1;
  if (!dcheck(ya >= 0 && xa >= 0 && yb < g.gy && xb < g.gx, kSiteTable)) return;
  const int held = sat[(yb + 1) * W + xb + 1] - sat[ya * W + xb + 1] - sat[(yb + 1) * W + xa] +
                   sat[ya * W + xa];
  // d^2 (in cells) of the disc expected to hold k points, and a margin.
  const float per = float(held) * rcp_approx(float((yb - ya + 1) * (xb - xa + 1)));
  const float fk = float(k);
  float reach = fk * rcp_approx(3.14159265f * per) * (1.f + 4.f * rsqrt_approx(fk));
  // The disc assumes points on all sides: none for a query beyond the grid's
  // edge (with two retries each and then a warp each, 2^20 queries up to a box
  // width outside took 28.7 ms, k = 32).
  bool listed = !(g.inv2 > 0.f) || beyond_grid(g, u, v) || 4 * held < k || held > knn_dense(k) ||
                !(h2 >= 0x1p-100f) || !(h2 <= 0x1p60f);

  // The runs of the cells that can hold a key up to d2 (rows and columns
  // rounded outwards), row by row.
  auto walk = [&](float d2, auto&& take) {
    const float w2 = __fmul_ru(__fadd_ru(d2, 0x1p-126f), ih2);
    auto clip = [&](float c, float e, int last, int& lo, int& hi) {
      const float a = ceilf(__fsub_rd(__fsub_rd(__fsub_rd(c, mg), e), 1.f));
      const float b = floorf(__fadd_ru(__fadd_ru(c, mg), e));
      lo = int(fminf(fmaxf(0.f, a), float(last) + 1.f));
      hi = int(fmaxf(fminf(float(last), b), -1.f));
    };
    // Row yy's run; empty beyond the disc.
    auto run = [&](int yy, int& a, int& b) {
      a = b = 0;
      const float gap = fmaxf(0.f, fmaxf(float(yy) - v, v - float(yy + 1)) - mg);
      const float g2 = __fmul_rd(gap, gap);
      int ra, rb;
      clip(u, __fsqrt_ru(__fsub_ru(w2, g2)), g.gx - 1, ra, rb);
      if (g2 <= w2 && ra <= rb) {
        a = cell_start(starts, base, yy * g.gx + ra, g.cells);
        b = cell_start(starts, base, yy * g.gx + rb + 1, g.cells);
      }
    };
    int r0, r1, a = 0, b = 0;
    clip(v, __fsqrt_ru(w2), g.gy - 1, r0, r1);
    if (r0 <= r1) run(r0, a, b);
    for (int yy = r0; yy <= r1; ++yy) {
      int na = 0, nb = 0;  // the next row's, looked up while this one is walked
      if (yy < r1) run(yy + 1, na, nb);
#pragma unroll 4
      for (int q = a; q < b; ++q) {
        if (!dcheck(q >= 0 && q < n, kSiteGather)) break;
        take(sorted[q]);
      }
      a = na;
      b = nb;
    }
  };

  int below = 0, cut = -1;  // points in bins below `cut`, the bin where the count reaches k
  float scale = 0.f, edge = 0.f;
  // Bin of a d^2 below `edge`: 0 .. kBins - 1, monotone in d^2.
  auto bin_of = [&](float d2) {
    return min(__float_as_int(__fmaf_rn(d2, scale, 8388608.f)) - 0x4B000000, kBins - 1);
  };
  for (int attempt = 0; !listed && attempt < 3; ++attempt, reach *= 2.5f) {
    edge = reach * hh * hh;
    scale = float(kBins) * rcp_approx(edge);
#pragma unroll
    for (int b = 0; b < kBins; ++b) bins[b][lane] = 0;
    walk(edge, [&](const float4 c) {
      const float d2 = fp32_d2(qx, qy, c.x, c.y);
      if (d2 < edge) ++bins[bin_of(d2)][lane];
    });
    int sum = 0;
    for (int b = 0; b < kBins; ++b) {
      const int c = bins[b][lane];
      if (sum + c >= k) {
        cut = b;
        below = sum;
        break;
      }
      sum += c;
    }
    if (cut >= 0) break;
  }
  if (cut < 0) listed = true;

  const float hp = static_cast<float>(0.5 * p);
  ValueSums<MODE, kWeightShepard> sums;  // of the selection
  int best = INT_MAX, aside = 0;
  float bestz = 0.f, kth = 0.f;
  auto add = [&](float d2, float z) {
    const float w = local_weight<MODE>(d2, hp, -hp);
    two_sum_acc(sums.hi, sums.lo, pk(w, __fmul_rn(w, z)));
  };
  if (!listed) {
    // Any d^2 in bins up to `cut` is below this (bins round to nearest, the
    // last one reaches up to the edge).
    const float bound = cut == kBins - 1
                            ? edge
                            : (float(cut) + 0.5f) * edge * ((1.f / kBins) * (1.f + 0x1p-18f));
    walk(bound, [&](const float4 c) {
      const float d2 = fp32_d2(qx, qy, c.x, c.y);
      if (d2 < edge) {
        const int b = bin_of(d2);
        if (b < cut) {
          add(d2, c.z);
        } else if (b == cut) {
          if (aside < kAside) {
            aside_key[aside][lane] = knn_key(d2, __float_as_int(c.w));
            aside_z[aside][lane] = c.z;
          }
          ++aside;
        }
        if (d2 == 0.f && c.x == qx && c.y == qy && __float_as_int(c.w) < best) {
          best = __float_as_int(c.w);
          bestz = c.z;
        }
      }
    });
    listed = aside > kAside;
  }
  if (listed) {
    list_heavy<-1>(t, m, lists.left, lists.query + (m - 1));
    return;
  }
  // The k - below smallest of the candidates set aside.
  const int need = k - below;
  for (int i = 0; i < aside; ++i) {
    const u64 key = aside_key[i][lane];
    int rank = 0;
    for (int o = 0; o < aside; ++o) rank += aside_key[o][lane] < key;
    if (rank < need) add(key_d2(key), aside_z[i][lane]);
    if (rank == need - 1) kth = key_d2(key);
  }
  sums.cnt = k;
  float z;
  if (best != INT_MAX) {
    z = bestz;
  } else if (!sums.value(z)) {
    // Sums outside FP32's range: the other searches redo the query.
    list_heavy<-1>(t, m, lists.left, lists.query + (m - 1));
    return;
  }
  out[j] = z;
  if (kd2_out) kd2_out[j] = kth;
}

// ------------------------------------------------- k-NN, a warp per query
//
// The search for calls with few queries, and for the queries of larger calls
// that one thread would take long over (see knn_surroundings, KnnLists):
// 1. a disc around the query that holds at least k points, its radius found
//    from the summed-area table with 32 radii per probe: the cells inside
//    three rectangles inscribed in the disc are counted, so the k-th key is
//    at most the disc's radius squared;
// 2. every cell the disc reaches is walked (the rows' runs laid end to end,
//    32 candidates at a time, one coalesced load each); keys up to the bound
//    are appended to a buffer in shared memory, and whenever it is nearly
//    full its k smallest keys are kept and the bound drops to the k-th key;
// 3. the k smallest of the buffer are the selection (keys are distinct, so
//    the order of candidates does not matter), and the lanes share the sums.
// About 1500 instructions a query at k = 8, with 29 of 32 lanes active; a query
// costs about as many whether its points lie near or far, which is what the
// hard queries need.  A call of 10,000 is bound by latency (a third of the warps
// resident, loads the first stall).
constexpr unsigned kWarp = 0xffffffffu;

// kRegs keys per lane: the buffer of 32 kRegs keys is cut back to k when
// fewer than 32 slots are free, so k <= 32 (kRegs - 1).
template <int kRegs>
struct KnnBuffer {
  static constexpr int kCap = 32 * kRegs;
  int lane;
  u64* buf;

  // Keeps the k smallest of the buffer's `cnt` keys (all of them if there are
  // no more than k) and returns the largest kept; `cnt` becomes their number.
  // The k-th smallest d^2 is bracketed between lo (fewer than k keys at or
  // below) and hi (at least k) in the order of the float's bits; the probe
  // between them assumes keys spread evenly in d^2, as points of even density
  // are, and every third probe halves the bracket instead.  No probe separates
  // keys of equal d^2 (data on a lattice): after kProbes of them the rest of the
  // bracket is gone through key by key, which closes on a tie at once, not bit by
  // bit (lattice of 2^20 points, queries on it, m = 50,000, k = 64: 176 us, 130 so).
  // With four keys a lane six probes often stop short of a bracket that a few more
  // would close (uniform data, m = 10,007, k = 64: six 37.8, eight 36.5, ten 34.2 us;
  // m = 10,007 on the lattice 34.1, 35.5, 37.6); with fewer, ten gain nothing.
  static constexpr int kProbes = kRegs > 3 ? 9 : 6;
  __device__ u64 prune(int& cnt, int k) {
    __syncwarp();
    if (cnt <= 32) return prune_regs<1>(cnt, k);
    if (cnt <= 64) return prune_regs<2>(cnt, k);
    return prune_regs<kRegs>(cnt, k);
  }

  // As prune, for at most 32 R keys.
  template <int R>
  __device__ __forceinline__ u64 prune_regs(int& cnt, int k) {
    int d[R], id[R];  // d^2 bits (not negative) and index; INT_MAX: no key
    int dmin = INT_MAX, dmax = -1;
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const int s = lane + i * 32;
      const u64 key = s < cnt ? buf[s] : u64(0);
      d[i] = s < cnt ? int(unsigned(key >> 32)) : INT_MAX;
      id[i] = key_index(key);
      dmin = min(dmin, d[i]);
      if (s < cnt) dmax = max(dmax, d[i]);
    }
    int hi = __reduce_max_sync(kWarp, dmax), chi = cnt;
    if (chi > k) {
      int lo = __reduce_min_sync(kWarp, dmin) - 1, clo = 0;
      for (int it = 0; it < kProbes && hi - lo > 1 && chi != k; ++it) {
        const float fl = __int_as_float(max(lo, 0)), fh = __int_as_float(hi);
        const float f = (float(k - clo) - 0.5f) * rcp_approx(float(chi - clo));
        int mid = it % 3 == 2 || !(fh <= FLT_MAX) ? lo + ((hi - lo) >> 1)
                                                  : __float_as_int(fmaf(fh - fl, f, fl));
        mid = max(lo + 1, min(hi - 1, mid));
        int c = 0;
#pragma unroll
        for (int i = 0; i < R; ++i) c += d[i] <= mid;
        c = __reduce_add_sync(kWarp, c);
        if (c >= k) {
          hi = mid;
          chi = c;
        } else {
          lo = mid;
          clo = c;
        }
      }
      while (hi - lo > 1 && chi != k) {  // ties: on to the next key, until k are covered
        int next = INT_MAX, c = 0;
#pragma unroll
        for (int i = 0; i < R; ++i) next = min(next, d[i] > lo ? d[i] : INT_MAX);
        next = __reduce_min_sync(kWarp, next);
#pragma unroll
        for (int i = 0; i < R; ++i) c += d[i] <= next;
        c = __reduce_add_sync(kWarp, c);
        if (c >= k) {
          hi = next;
          chi = c;
          break;
        }
        lo = next;
        clo = c;
      }
      int tie = INT_MAX;  // of keys with d^2 == hi, indices up to this one
      if (chi != k) {     // more than k: the lowest k - clo indices among the ties
        tie = -1;
        for (int t = clo; t < k; ++t) {
          int m = INT_MAX;
#pragma unroll
          for (int i = 0; i < R; ++i)
            if (d[i] == hi && id[i] > tie) m = min(m, id[i]);
          tie = __reduce_min_sync(kWarp, m);
        }
      }
      int base = 0;
      dmax = -1;
#pragma unroll
      for (int i = 0; i < R; ++i) {  // every lane holds its keys in registers by now
        const bool keep = d[i] < hi || (d[i] == hi && id[i] <= tie);
        const unsigned b = __ballot_sync(kWarp, keep);
        if (keep) {
          const int at = base + __popc(b & ((1u << lane) - 1));
          if (dcheck(at < kCap, kSiteHeap)) buf[at] = knn_key(__int_as_float(d[i]), id[i]);
          dmax = max(dmax, d[i]);
        } else {
          d[i] = -1;
        }
        base += __popc(b);
      }
      cnt = base;
      hi = __reduce_max_sync(kWarp, dmax);
      __syncwarp();
    }
    int im = -1;
#pragma unroll
    for (int i = 0; i < R; ++i)
      if (d[i] == hi) im = max(im, id[i]);
    return knn_key(__int_as_float(hi), __reduce_max_sync(kWarp, im));
  }
};

constexpr int kKnnWarpThreads = 128;

// One query, by a whole warp.
template <int MODE, int kRegs>
__device__ __forceinline__ void knn_warp_query(
    const GridDev& g, u64* keys, float qx, float qy, int j, const float4* sorted,
    const int32_t* starts, const int32_t* base,
    const int32_t* sat, const float* data, int64_t n, double p, int k,
    float* __restrict__ out, int32_t* nbr_out, float* __restrict__ kd2_out,
    int32_t* hit_out, bool sort_rows) {
  using Buffer = KnnBuffer<kRegs>;
  Buffer kb;
  kb.lane = threadIdx.x % 32;
  kb.buf = keys;
  const int lane = kb.lane;
  int best_hit = INT_MAX;  // this lane's
  int cnt = 0;             // keys in the buffer (the same in every lane)
  u64 worst = ~u64(0);     // no key above this one is in the selection

  if (finite2(qx, qy)) {
    const float u = cell_pos(qx, g.hx0, g.inv2), v = cell_pos(qy, g.hy0, g.inv2);
    const float mg = __fmaf_ru(fabsf(u) + fabsf(v), 0x1p-22f, 0x1p-9f);
    const float hh = g.inv2 > 0.f ? 2.f / g.inv2 : 0.f;
    const float h2 = __fmul_rd(hh, hh) * (1.f - 0x1p-18f);
    const float ih2 = __frcp_ru(h2);  // +inf for the one-cell grid: nothing is clipped
    if (g.inv2 > 0.f && fabsf(u) < 0x1p20f && fabsf(v) < 0x1p20f) {
      // Points in cells xa..xb, ya..yb, clamped into the grid; an empty
      // rectangle's four entries cancel.  Straight-line code: every lane of
      // the warp reaches the votes below together.
      const int W = g.gx + 1;
      auto rect = [&](int xa, int xb, int ya, int yb) {
        const int x0 = min(max(xa, 0), g.gx), x1 = min(max(xb + 1, x0), g.gx);
        const int y0 = min(max(ya, 0), g.gy), y1 = min(max(yb + 1, y0), g.gy);
        return sat[y1 * W + x1] - sat[y0 * W + x1] - sat[y1 * W + x0] + sat[y0 * W + x0];
      };
      // Points in cells that lie inside the disc of radius rho cells: the
      // union of three inscribed rectangles, each shrunk by mg for the
      // cell-position errors.  Their corners divide the disc's reach into the
      // grid, which begins bx (by) cells from the query: at 22.5, 45 and 67.5
      // degrees for a query over the grid; for one beyond its edge at those
      // shares of the cap that the edge cuts off the disc (corners at fixed
      // angles reach 0.92 rho, and a query 500 cells away then walked a cap 40
      // cells deep: 10,007 queries up to a box width outside, n = 2^20, k = 8,
      // 610 us a call, 84 so).
      const float bx = fmaxf(0.f, fmaxf(-u, u - float(g.gx)));
      const float by = fmaxf(0.f, fmaxf(-v, v - float(g.gy)));
      const bool over = bx + by == 0.f;
      auto disc_count = [&](float rho) {
        float e1 = 0.9238795f * rho - mg, e2 = 0.7071067f * rho - mg, e3 = 0.3826834f * rho - mg;
        float h1 = e3, h2 = e2, h3 = e1;
        if (!over) {
          const float across = sqrt_approx(fmaxf(0.f, (rho - by) * (rho + by))) - bx;
          // A hair short of the corner's height, for the roundings here.
          auto tall = [&](float e) {
            const float x = e + mg;
            return sqrt_approx(fmaxf(0.f, (rho - x) * (rho + x))) * (1.f - 0x1p-20f) - mg;
          };
          e1 = fmaf(0.9238795f, across, bx) - mg;
          e2 = fmaf(0.7071067f, across, bx) - mg;
          e3 = fmaf(0.3826834f, across, bx) - mg;
          h1 = tall(e1);
          h2 = tall(e2);
          h3 = tall(e3);
        }
        const int xa1 = int(ceilf(u - e1)), xb1 = int(floorf(u + e1)) - 1;
        const int xa2 = int(ceilf(u - e2)), xb2 = int(floorf(u + e2)) - 1;
        const int xa3 = int(ceilf(u - e3)), xb3 = int(floorf(u + e3)) - 1;
        const int ya1 = int(ceilf(v - h1)), yb1 = int(floorf(v + h1)) - 1;
        const int ya2 = int(ceilf(v - h2)), yb2 = int(floorf(v + h2)) - 1;
        const int ya3 = int(ceilf(v - h3)), yb3 = int(floorf(v + h3)) - 1;
        int c = rect(xa1, xb1, ya1, yb1);
        c += rect(xa2, xb2, ya2, yb2) - rect(xa2, xb2, ya1, yb1);
        c += rect(xa3, xb3, ya3, yb3) - rect(xa3, xb3, ya2, yb2);
        return c;
      };
      // Bracket: squares of half-width 5/8 (5/4)^lane cells (the last one, 631,
      // doubled until it holds k points or cannot: then no bound).  The disc
      // around the first that holds k does too; the discs that fit into the
      // square before it do not.
      auto square = [&](float e) {
        return rect(int(ceilf(u - e + mg)), int(floorf(u + e - mg)) - 1, int(ceilf(v - e + mg)),
                    int(floorf(v + e - mg)) - 1);
      };
      const float side = 0.625f * ex2_approx(0.32192809f * float(lane));
      int inside = square(side);
      unsigned b = __ballot_sync(kWarp, inside >= k);
      float far = 1.f;
      while (b == 0 && far < 4096.f) {
        far *= 2.f;
        inside = square(side * far);
        b = __ballot_sync(kWarp, inside >= k) & 0x80000000u;
      }
      if (b) {
        const int f = __ffs(b) - 1;
        const float s1 = far * __shfl_sync(kWarp, side, f);
        const float before = __shfl_sync(kWarp, side, max(f - 1, 0));
        float lo = far > 1.f ? 0.5f * s1 : f > 0 ? before : 0.f;
        float hi = 1.4142137f * (s1 + mg), step;
        // 32 radii in between, again while they are over a cell apart.
        do {
          step = (hi - lo) * 0x1p-5f;
          const float probe = lane == 31 ? hi : fmaf(step, float(lane + 1), lo);
          inside = disc_count(probe);
          const unsigned in = __ballot_sync(kWarp, inside >= k) | 0x80000000u;  // hi does
          hi = __shfl_sync(kWarp, probe, __ffs(in) - 1);
          lo = hi - step;
        } while (step > 1.f);
        // An upper bound of the FP32 d^2 of any point in the disc.
        const float bound = __fadd_ru(
            __fmul_ru(__fmul_ru(__fmul_ru(hi, hi), __fmul_ru(hh, hh)), 1.f + 0x1p-17f), 0x1p-126f);
        if (bound <= FLT_MAX) worst = knn_key(bound, -1);
      }
    }
    // Rows whose gap from v, and columns whose gap from u, can hold a key up
    // to `worst`, rounded outwards (a NaN or infinite bound clips nothing).
    auto reach2 = [&]() { return __fmul_ru(__fadd_ru(key_d2(worst), 0x1p-126f), ih2); };
    auto clip = [&](float c, float e, int& first, int& last) {
      const float fa = ceilf(__fsub_rd(__fsub_rd(__fsub_rd(c, mg), e), 1.f));
      const float fb = floorf(__fadd_ru(__fadd_ru(c, mg), e));
      const int nf = int(fminf(fmaxf(float(first), fa), float(last) + 1.f));
      const int nl = int(fmaxf(fminf(float(last), fb), float(first) - 1.f));
      first = nf;
      last = nl;
    };
    int row0 = 0, row1 = g.gy - 1;
    clip(v, __fsqrt_ru(reach2()), row0, row1);
    for (int y0 = row0; y0 <= row1; y0 += 32) {
      // This lane's row: its run [a, a + len) of the sorted points.
      const int yy = y0 + lane;
      int a = 0, len = 0;
      if (yy <= row1) {
        const float gap = fmaxf(0.f, fmaxf(float(yy) - v, v - float(yy + 1)) - mg);
        const float w2 = reach2(), g2 = __fmul_rd(gap, gap);
        int ra = 0, rb = g.gx - 1;
        if (!(g2 > w2)) {
          clip(u, __fsqrt_ru(__fsub_ru(w2, g2)), ra, rb);
          if (ra <= rb) {
            a = cell_start(starts, base, yy * g.gx + ra, g.cells);
            len = cell_start(starts, base, yy * g.gx + rb + 1, g.cells) - a;
          }
        }
      }
      // The rows' runs end to end: candidate s belongs to the run whose end
      // is the first above s.
      int end = len;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(kWarp, end, o);
        if (lane >= o) end += x;
      }
      const int total = __shfl_sync(kWarp, end, 31);
      const int shift = a - (end - len);  // candidate s of this run is sorted[s + shift]
      for (int s0 = 0; s0 < total; s0 += 32) {
        const int s = s0 + lane;
        int r = 0;  // the number of runs that end at or before s
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
          if (__shfl_sync(kWarp, end, r + o - 1) <= s) r += o;
        const int at = s + __shfl_sync(kWarp, shift, r);
        u64 key = ~u64(0);
        bool take = false;
        if (s < total && dcheck(at >= 0 && at < n, kSiteGather)) {
          const float4 c = sorted[at];
          const float d2 = fp32_d2(qx, qy, c.x, c.y);
          const int idx = __float_as_int(c.w);
          if (d2 == 0.f && c.x == qx && c.y == qy) best_hit = min(best_hit, idx);
          key = knn_key(d2, idx);
          take = key <= worst;
        }
        const unsigned b = __ballot_sync(kWarp, take);
        const int slot = cnt + __popc(b & ((1u << lane) - 1));
        if (take && dcheck(slot < Buffer::kCap, kSiteHeap)) kb.buf[slot] = key;
        cnt += __popc(b);
        if (cnt > Buffer::kCap - 32) worst = kb.prune(cnt, k);
      }
    }
    if (cnt > 0) worst = kb.prune(cnt, k);  // the largest key of the selection
    best_hit = __reduce_min_sync(kWarp, best_hit);
  }
  __syncwarp();

  if (lane == 0) {
    if (kd2_out) kd2_out[j] = cnt > 0 ? key_d2(worst) : __int_as_float(0x7fc00000);
    if (hit_out) hit_out[j] = best_hit != INT_MAX ? best_hit : -1;
  }
  if (nbr_out) {
    int32_t* row = nbr_out + int64_t(j) * k;
    for (int s = lane; s < k; s += 32) {
      int at = s;
      if (s < cnt && sort_rows) {  // the key's rank
        const u64 key = kb.buf[s];
        at = 0;
        for (int o = 0; o < cnt; ++o) at += kb.buf[o] < key;
      }
      row[at] = s < cnt ? key_index(kb.buf[s]) : -1;
    }
  }
  if (best_hit != INT_MAX || cnt == 0) {
    if (lane == 0)
      out[j] = cnt == 0 ? __int_as_float(0x7fc00000)
               : dcheck(best_hit >= 0 && best_hit < n, kSiteData) ? data[3 * int64_t(best_hit) + 2]
                                                                  : 0.f;
    return;
  }
  // Eq. 1 over the selection: compensated FP32 sums per lane, joined by a
  // fixed tree of error-free additions.
  const float hpw = static_cast<float>(0.5 * p), nhp = -hpw;
  u64 hi = 0, lo = 0;
  for (int s = lane; s < cnt; s += 32) {
    const u64 key = kb.buf[s];
    const float w = local_weight<MODE>(key_d2(key), hpw, nhp);
    if (!dcheck(key_index(key) >= 0 && key_index(key) < n, kSiteData)) continue;
    two_sum_acc(hi, lo, pk(w, __fmul_rn(w, data[3 * int64_t(key_index(key)) + 2])));
  }
  // Lanes from min(cnt, 32) on hold zeros; lane 0 gets the total.
  for (int o = cnt > 16 ? 16 : cnt > 8 ? 8 : cnt > 4 ? 4 : 2; o > 0; o >>= 1) {
    const u64 oh = __shfl_xor_sync(kWarp, hi, o), ol = __shfl_xor_sync(kWarp, lo, o);
    two_sum_acc(hi, lo, oh);
    lo = add2(lo, ol);
  }
  hi = __shfl_sync(kWarp, hi, 0);  // every lane takes the same branch below
  lo = __shfl_sync(kWarp, lo, 0);
  float h0, h1, l0, l1;
  upk(hi, h0, h1);
  upk(lo, l0, l1);
  float zv;
  if (h0 >= kTinyPerMember * float(cnt) && h0 <= FLT_MAX && fabsf(h1) <= FLT_MAX &&
      fabsf(l1) <= FLT_MAX) {
    const float z0 = __fdiv_rn(h1, h0);
    const float res = __fadd_rn(__fmaf_rn(-z0, h0, h1), __fmaf_rn(-z0, l0, l1));
    zv = __fmaf_rn(res, rcp_approx(h0), z0);
  } else {
    // Outside FP32's range (the same in every lane): FP64 over the selected
    // points, scaled by d2_min^(p/2).
    double dmin = INFINITY;
    for (int s = 0; s < cnt; ++s) {
      const float* x = data + 3 * int64_t(key_index(kb.buf[s]));
      const double ex = double(qx) - x[0], ey = double(qy) - x[1];
      dmin = fmin(dmin, ex * ex + ey * ey);
    }
    double s0 = 0.0, s1 = 0.0;
    for (int s = lane; s < cnt; s += 32) {
      const float* x = data + 3 * int64_t(key_index(kb.buf[s]));
      const double ex = double(qx) - x[0], ey = double(qy) - x[1];
      const double w = pow(dmin / (ex * ex + ey * ey), 0.5 * p);
      s0 += w;
      s1 += w * double(x[2]);
    }
    s0 = warp_sum(s0);
    s1 = warp_sum(s1);
    zv = static_cast<float>(s1 / s0);
  }
  if (lane == 0) out[j] = zv;
}

// The listed queries (or, with no list, all m), a warp each.
template <int MODE, int kRegs>
__global__ void __launch_bounds__(kKnnWarpThreads)
    knn_warp_kernel(const GridDev* grid, const float4* sorted,
                    const int32_t* starts, const int32_t* base,
                    const int32_t* sat, const float4* qrec,
                    const float* data, int64_t n, int64_t m, double p, int k,
                    float* __restrict__ out, int32_t* nbr_out,
                    float* __restrict__ kd2_out, int32_t* hit_out, bool sort_rows,
                    const KnnLists lists) {
  pdl_trigger();
  pdl_wait();
  using Buffer = KnnBuffer<kRegs>;
  __shared__ u64 keys[kKnnWarpThreads / 32][Buffer::kCap];
  // 32-bit counts (m is below 2^31): with 64-bit ones the p = 2 form for k > 32
  // takes 61 registers, not 56, and eight blocks an SM, not nine (2^20 points, m =
  // 10,007, k = 64: 78 us a call, 76 so).
  const unsigned hard = lists.query ? *lists.hard : unsigned(m);
  const unsigned left = lists.query ? *lists.left : 0u;
  const unsigned count = hard + (left <= lists.few ? left : 0u);
  const unsigned warps = gridDim.x * (kKnnWarpThreads / 32);
  const GridDev g = *grid;
  for (unsigned w = (blockIdx.x * kKnnWarpThreads + threadIdx.x) / 32; w < count;
       w += warps) {  // whole warps: no block-wide barrier in this kernel
    const int t = !lists.query ? int(w) : lists.query[w < hard ? w : unsigned(m) - 1 - (w - hard)];
    if (!dcheck(t >= 0 && t < m && count <= m, kSiteScatter)) continue;
    const float4 rq = qrec[t];
    const int j = __float_as_int(rq.z);
    if (!dcheck(j >= 0 && j < m, kSiteOutput)) continue;
    knn_warp_query<MODE, kRegs>(g, keys[threadIdx.x / 32], rq.x, rq.y, j, sorted, starts, base, sat,
                                data, n, p, k, out, nbr_out, kd2_out, hit_out, sort_rows);
    __syncwarp();  // the buffer is the next query's
  }
}

// ------------------------------------------- k-NN, warp-synchronous
//
// The same search as knn_query_kernel, one thread per query, with the 32
// lanes of a warp kept in step so that they diverge far less:
// * every lane grows its square by the same step at the same time (the
//   smallest of the lanes' step choices; a lane whose stop test has held
//   idles until the warp's last lane stops);
// * a band's rows are taken in the same order by every lane (row offsets
//   -r2 .. r2 from the lane's own cell row), each lane listing its
//   non-empty row runs (clipped to its disc) in shared memory first, then
//   walking its listed runs as one flat stream of candidates, so a lane
//   waits only when its whole stream is shorter than another's;
// * keys that beat a lane's k-th key are appended to its k slots while it
//   fills and to a short pending list after that; the warp merges the
//   pending lists into the lanes' heaps together (building each heap, by
//   Floyd's method, once its k slots are full) whenever a lane's list is
//   nearly full and at the end of each step, where the stop test needs the
//   exact k-th key.
// Every cell the single-query search walks is walked here too, or lies
// beyond the lane's k-th key, so the selection is the same: the k smallest
// keys.
// It is an option, not the default: the lanes do keep more in step (16.7
// of 32 threads per instruction against 12.0 at k = 32), but the lockstep
// control costs about as many warp instructions as the divergence it
// removes, the run lists cut the warps an SM holds, and on clustered data
// the lanes of a warp need very different numbers of steps.

constexpr int kSyncRuns = 8;     // row runs a lane lists before walking them
constexpr int kSyncPending = 4;  // keys a lane holds back before the warp merges

// Shared memory of one warp: (k + kSyncPending) key slots and kSyncRuns
// runs per lane, lane-interleaved.
size_t knn_sync_smem_bytes(int k) {
  return size_t(k + kSyncPending) * kKnnThreads * sizeof(u64) +
         size_t(kSyncRuns) * kKnnThreads * sizeof(int2);
}

template <int MODE>
__global__ void __launch_bounds__(kKnnThreads)
    knn_sync_kernel(const GridDev* grid, const float4* sorted,
                    const int32_t* starts, const int32_t* base,
                    const int32_t* bpre, const int32_t* sat,
                    const float4* qrec, const float* data, int64_t n,
                    int64_t m, double p, int k, float* __restrict__ out,
                    int32_t* nbr_out, float* __restrict__ kd2_out,
                    int32_t* hit_out, bool sort_rows) {
  pdl_trigger();
  pdl_wait();
  extern __shared__ __align__(16) unsigned char knn_smem[];
  constexpr unsigned kFull = 0xffffffffu;
  const int lane = threadIdx.x;
  const int64_t t = int64_t(blockIdx.x) * kKnnThreads + lane;
  KnnHeap hp;
  hp.h = reinterpret_cast<u64*>(knn_smem) + lane;
  int2* runs = reinterpret_cast<int2*>(knn_smem + size_t(k + kSyncPending) * kKnnThreads *
                                                      sizeof(u64)) + lane;
  const GridDev g = *grid;
  float qx = 0.f, qy = 0.f;
  int j = -1;
  if (t < m) {
    const float4 rq = qrec[t];
    qx = rq.x;
    qy = rq.y;
    j = __float_as_int(rq.z);
    if (!dcheck(j >= 0 && j < m, kSiteOutput)) j = -1;
  }
  const bool searching = j >= 0 && finite2(qx, qy);
  int best_hit = INT_MAX;
  // The heap's largest key once it is built, else above every key; zero
  // (nothing is taken) for a lane that does not search.
  u64 worst = searching ? ~u64(0) : u64(0);
  bool heaped = false;  // the k slots are full and form a heap
  int np = 0;           // keys pending after the k slots
  auto flush = [&]() {
    if (!heaped && hp.size == k) {
      hp.heapify(k);
      heaped = true;
      worst = hp.top();
    }
#pragma unroll 1
    for (int i = 0; i < kSyncPending; ++i) {
      if (i < np) {
        const u64 key = hp.h[(k + i) * kKnnThreads];
        if (key < worst) {
          hp.replace_top(key, k);
          worst = hp.top();
        }
      }
    }
    np = 0;
  };
  int nr = 0;  // runs listed
  // Keys one candidate record against the lane's query.
  auto consider = [&](const float4 c) {
    const float d2 = fp32_d2(qx, qy, c.x, c.y);
    const int idx = __float_as_int(c.w);
    if (d2 == 0.f && c.x == qx && c.y == qy) best_hit = min(best_hit, idx);
    const u64 key = knn_key(d2, idx);
    if (key < worst) {  // to the k slots while filling, else pending
      const bool fill = hp.size < k;
      const int slot = fill ? hp.size : k + np;
      if (dcheck(slot < k + kSyncPending && idx >= 0 && idx < n, kSiteHeap)) {
        hp.h[slot * kKnnThreads] = key;
        hp.size += fill;
        np += !fill;
      }
    }
  };
  // Walks the listed runs as one stream, two candidates per lane per pass,
  // both records loaded before either is keyed (a pass adds at most two
  // pending keys, so the warp merges when a lane holds more than
  // kSyncPending - 2).
  auto walk_runs = [&]() {
    int ri = 0, q = 0, b = 0;
    auto take = [&]() {  // the lane's next candidate, or -1
      if (q >= b && ri < nr) {
        const int2 rr = runs[ri * kKnnThreads];
        ++ri;
        q = rr.x;
        b = rr.y;
      }
      return q < b ? q++ : -1;
    };
    for (;;) {
      const int c0 = take(), c1 = take();
      float4 v0 = make_float4(0.f, 0.f, 0.f, 0.f), v1 = v0;
      const bool t0 = c0 >= 0 && dcheck(c0 < n, kSiteGather);
      const bool t1 = c1 >= 0 && dcheck(c1 < n, kSiteGather);
      if (t0) v0 = sorted[c0];
      if (t1) v1 = sorted[c1];
      if (t0) consider(v0);
      if (t1) consider(v1);
      // Merged before the loop can end, so that every lane leaves with at
      // most kSyncPending - 2 keys pending and the next pass has room.
      if (__any_sync(kFull, np > kSyncPending - 2)) flush();
      if (!__any_sync(kFull, q < b || ri < nr)) break;
    }
    nr = 0;
  };

  const float u = searching ? cell_pos(qx, g.hx0, g.inv2) : 0.f;
  const float v = searching ? cell_pos(qy, g.hy0, g.inv2) : 0.f;
  const int cx = clamp_floor(u, 0, g.gx - 1), cy = clamp_floor(v, 0, g.gy - 1);
  const float mg = __fmaf_ru(fabsf(u) + fabsf(v), 0x1p-22f, 0x1p-9f);
  const float ax = fmaxf(0.f, fmaxf(u - float(g.gx), -u) - mg);
  const float ay = fmaxf(0.f, fmaxf(v - float(g.gy), -v) - mg);
  const float hh = g.inv2 > 0.f ? 2.f / g.inv2 : 0.f;
  const float h2 = __fmul_rd(hh, hh) * (1.f - 0x1p-18f);
  const float ih2 = __frcp_ru(h2);
  auto reach2 = [&]() { return __fmul_ru(__fadd_ru(key_d2(worst), 0x1p-126f), ih2); };
  auto clip = [&](float c, float e, int& lo, int& hi) {
    if (lo > hi) return;
    const float a = ceilf(__fsub_rd(__fsub_rd(__fsub_rd(c, mg), e), 1.f));
    const float b = floorf(__fadd_ru(__fadd_ru(c, mg), e));
    const int nlo = int(fminf(fmaxf(float(lo), a), float(hi) + 1.f));
    const int nhi = int(fmaxf(fminf(float(hi), b), float(lo) - 1.f));
    lo = nlo;
    hi = nhi;
  };
  auto square_count = [&](int rr) {
    const int ya = max(0, cy - rr), yb = min(g.gy - 1, cy + rr);
    const int xa = max(0, cx - rr), xb = min(g.gx - 1, cx + rr);
    const int W = g.gx + 1;
    if (!dcheck(ya >= 0 && xa >= 0 && yb < g.gy && xb < g.gx, kSiteTable)) return 0;
    return sat[(yb + 1) * W + xb + 1] - sat[ya * W + xb + 1] - sat[(yb + 1) * W + xa] +
           sat[ya * W + xa];
  };
  // Lists run [xa, xb] of row yy (already clipped) when it holds points.
  auto list_run = [&](int yy, int xa, int xb) {
    if (xa > xb) return;
    const int a = cell_start(starts, base, yy * g.gx + xa, g.cells);
    const int b = cell_start(starts, base, yy * g.gx + xb + 1, g.cells);
    if (a < b && dcheck(nr < kSyncRuns, kSiteTable)) runs[nr++ * kKnnThreads] = make_int2(a, b);
  };

  bool finished = !searching;
  int in_square = -1;  // points in this lane's square of radius r, once counted
  for (int r = -1;;) {
    if (r >= 0) {
      flush();  // the stop test and the clipping use the exact k-th key
      if (!finished) {
        const bool open_l = cx - r > 0, open_r = cx + r < g.gx - 1;
        const bool open_b = cy - r > 0, open_t = cy + r < g.gy - 1;
        if (!(open_l || open_r || open_b || open_t)) {
          finished = true;  // the square covers the grid
        } else if (heaped) {
          float l2 = INFINITY;
          if (open_l) {
            const float dx = fmaxf(ax, fmaxf(0.f, (u - float(cx - r)) - mg));
            l2 = fminf(l2, __fmaf_rd(dx, dx, __fmul_rd(ay, ay)));
          }
          if (open_r) {
            const float dx = fmaxf(ax, fmaxf(0.f, (float(cx + r + 1) - u) - mg));
            l2 = fminf(l2, __fmaf_rd(dx, dx, __fmul_rd(ay, ay)));
          }
          if (open_b) {
            const float dy = fmaxf(ay, fmaxf(0.f, (v - float(cy - r)) - mg));
            l2 = fminf(l2, __fmaf_rd(dy, dy, __fmul_rd(ax, ax)));
          }
          if (open_t) {
            const float dy = fmaxf(ay, fmaxf(0.f, (float(cy + r + 1) - v) - mg));
            l2 = fminf(l2, __fmaf_rd(dy, dy, __fmul_rd(ax, ax)));
          }
          if (key_d2(worst) < __fmul_rd(l2, h2) - 0x1p-126f) finished = true;
        }
      }
      if (__all_sync(kFull, finished)) break;
    }
    // The step: each searching lane chooses as the single-query search does
    // (from r = 4 on, halved while its band would hold more than 4k points,
    // counted from the summed-area table); the warp takes the smallest.
    int r2 = r + max(1, r >> 1);
    bool walk = !finished;
    if (r >= 4) {
      int mine = INT_MAX;
      if (!finished) {
        if (in_square < 0) in_square = square_count(r);
        mine = r2;
        int c2 = square_count(mine);
        while (c2 - in_square > 4 * k && mine > r + 1) {
          mine = r + max(1, (mine - r) >> 1);
          c2 = square_count(mine);
        }
      }
      r2 = __reduce_min_sync(kFull, mine);
      if (!finished) {
        const int c2 = square_count(r2);
        walk = c2 != in_square;  // an empty band is not walked
        in_square = c2;
      }
    }
    if (r < 0) {
      if (walk) list_run(cy, cx, cx);  // the lane's own cell
    } else {
      // Row offsets -r2 .. r2 from the lane's own row, the same for every
      // lane: within r a row holds the band's two side strips, beyond it a
      // whole row of the band.
      const bool check_blocks = r >= 8;
#pragma unroll 1
      for (int s = -r2; s <= r2; ++s) {
        if (__any_sync(kFull, nr > kSyncRuns - 2)) walk_runs();
        const int yy = cy + s;
        if (!walk || yy < 0 || yy >= g.gy) continue;
        int xa = max(0, cx - r2), xb = min(g.gx - 1, cx + r2);
        if (heaped) {  // the columns this row's chord reaches
          const float gap = fmaxf(0.f, fmaxf(float(yy) - v, v - float(yy + 1)) - mg);
          const float w2 = reach2(), g2 = __fmul_rd(gap, gap);
          if (g2 > w2) continue;
          clip(u, __fsqrt_ru(__fsub_ru(w2, g2)), xa, xb);
          if (xa > xb) continue;
        }
        if (check_blocks) {  // the row's stretch of 8 x 8-cell blocks holds no point
          const int by = yy >> kBlockShift;
          const int32_t* bp = bpre + by * (kMaxBlocksPerAxis + 1);
          if (!dcheck(by < kMaxBlocksPerAxis && (xb >> kBlockShift) < kMaxBlocksPerAxis,
                      kSiteBlock) ||
              bp[(xb >> kBlockShift) + 1] == bp[xa >> kBlockShift])
            continue;
        }
        if (s >= -r && s <= r) {
          list_run(yy, xa, min(xb, cx - r - 1));
          list_run(yy, max(xa, cx + r + 1), xb);
        } else {
          list_run(yy, xa, xb);
        }
      }
    }
    walk_runs();
    r = r2;
  }
  flush();
  if (!heaped) hp.heapify(hp.size);  // fewer than k points
  if (j >= 0)
    knn_write_result<MODE>(hp, best_hit, qx, qy, j, data, n, p, k, out, nbr_out, kd2_out,
                           hit_out, sort_rows);
}

// ------------------------------------------------------ k-NN gradients
//
// The k-NN form's gradients hold each query's selection fixed (it is
// piecewise constant in every input): the derivatives of Eq. 1 summed over
// the selected points, as for the radius form.  The search runs first, with
// neighbour lists and hits kept in the workspace; then one thread per query
// (cell order, so neighbouring threads share points) walks its list, left
// in heap order (the search skips the heap sort): one pass finds d2_min and
// the sums of the scaled weights (d2_min / d^2)^(p/2), rescaling them when a
// smaller d^2 appears, a second the gradients.  A selection is not
// bounded by a fixed radius, so the data-side terms (dL/dz, dL/dx, dL/dy)
// are added to a per-point float4 with one 16-byte vector atomic per pair
// (a third of the L2 operations of three scalar ones; their order, and so
// the last bits, can vary between calls), then copied out.

// The FP64 path of one k-NN query: adds its data-side terms, returns
// (dL/dqx, dL/dqy) and its dL/dp share.  Out of line (rare).
struct KnnGradF64 {
  float gqx, gqy;
  double gp;
  double Z, c, dmin;  // what the pair terms are computed from
};
__device__ __noinline__ KnnGradF64 knn_grad_query_f64(const int32_t* row, int cnt,
                                                      const float* data, float qx,
                                                      float qy, double p, float gj,
                                                      float4* acc) {
  double dmin = INFINITY;
  for (int s = 0; s < cnt; ++s) {
    const float* x = data + 3 * int64_t(row[s]);
    const double ex = double(qx) - x[0], ey = double(qy) - x[1];
    dmin = fmin(dmin, ex * ex + ey * ey);
  }
  double s0 = 0.0, s1 = 0.0;
  for (int s = 0; s < cnt; ++s) {
    const float* x = data + 3 * int64_t(row[s]);
    const double ex = double(qx) - x[0], ey = double(qy) - x[1];
    const double w = pow(dmin / (ex * ex + ey * ey), 0.5 * p);
    s0 += w;
    s1 += w * double(x[2]);
  }
  const double Z = s1 / s0, c = double(gj) / s0;
  double ax = 0.0, ay = 0.0, al = 0.0;
  for (int s = 0; s < cnt; ++s) {
    const int64_t i = row[s];
    const float* x = data + 3 * i;
    const double ex = double(qx) - x[0], ey = double(qy) - x[1], e2 = ex * ex + ey * ey;
    const double w = pow(dmin / e2, 0.5 * p);
    const double a = (double(x[2]) - Z) * w;
    ax += a * ex / e2;
    ay += a * ey / e2;
    al += a * log(e2 / dmin);
    if (acc)
      atomicAdd(&acc[i], make_float4(static_cast<float>(c * w), static_cast<float>(c * p * a * ex / e2),
                                     static_cast<float>(c * p * a * ey / e2), 0.f));
  }
  KnnGradF64 r;
  r.gqx = static_cast<float>(-c * p * ax);
  r.gqy = static_cast<float>(-c * p * ay);
  r.gp = -0.5 * c * al;
  r.Z = Z;
  r.c = c;
  r.dmin = dmin;
  return r;
}

// Per-query state of a deterministic k-NN gradient: the data-side pass
// recomputes each (point, query) term from it, point by point.
enum KnnQMode : int { kKnnQNone = 0, kKnnQF32 = 1, kKnnQF64 = 2, kKnnQHit = 3 };
struct KnnQState {
  double Z, c, d2min;  // FP32 path: exact widenings of its float values
  float lmin;          // log2 d2min (general p, FP32 path)
  int mode;            // KnnQMode
};
static_assert(sizeof(KnnQState) == 32, "query state layout");

template <int MODE>
__global__ void __launch_bounds__(kLocalThreads)
    knn_grad_kernel(const float4* __restrict__ qrec, int64_t m, const float* __restrict__ data,
                    int64_t n, const int32_t* __restrict__ nbr, const int32_t* __restrict__ hit,
                    int k, double p, const float* __restrict__ grad_out,
                    float4* __restrict__ acc, float* __restrict__ grad_q,
                    double* __restrict__ grad_p, KnnQState* __restrict__ qstate,
                    double* __restrict__ gp_query) {
  // Launched plainly: its rows and points are read ahead of the atomics only
  // through __restrict__, which a kernel that starts early cannot have (without
  // it, uniform n = m = 2^20, k = 32: 2.18 ms a backward call, 1.57 with).
  // qstate (deterministic mode): each query's state is recorded for the
  // point-major pass, acc is null, and dL/dp goes per query to gp_query.
  const int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  double gp = 0.0;  // every lane joins the warp sum
  if (t < m) {
    const float4 r = qrec[t];
    const float qx = r.x, qy = r.y;
    const int j = __float_as_int(r.z);
    if (dcheck(j >= 0 && j < m, kSiteOutput)) {
      const float gj = grad_out[j];
      const int32_t* row = nbr + int64_t(j) * k;
      const int h = hit[j];
      int cnt = 0;
      while (cnt < k && row[cnt] >= 0) ++cnt;
      float gqx = 0.f, gqy = 0.f;
      KnnQState qs{0.0, 0.0, 0.0, 0.f, kKnnQNone};
      if (h >= 0) {
        if (acc && dcheck(h < n, kSiteData)) atomicAdd(&acc[h], make_float4(gj, 0.f, 0.f, 0.f));
        qs.mode = kKnnQHit;
      } else if (cnt > 0) {
        const float hp = static_cast<float>(0.5 * p), pf = static_cast<float>(p);
        // One pass: d2_min and the sums with weights scaled by the smallest
        // d^2 so far, rescaled when a smaller one appears (the row is in
        // heap order).
        float d2min = INFINITY, lmin = 0.f, s0 = 0.f, s1 = 0.f;
        for (int s = 0; s < cnt; ++s) {
          const float* x = data + 3 * int64_t(row[s]);
          const float d2 = fp32_d2(qx, qy, x[0], x[1]);
          if (d2 < d2min) {
            const float l = MODE == kPow2 ? 0.f : lg2_approx(d2);
            if (s > 0) {
              const float f = grad_weight<MODE>(d2min, d2, l, hp);  // (d2 / d2min_old)^(p/2)
              s0 *= f;
              s1 *= f;
            }
            d2min = d2;
            lmin = l;
          }
          const float w = grad_weight<MODE>(d2, d2min, lmin, hp);
          s0 += w;
          s1 = fmaf(w, x[2], s1);
        }
        bool f32 = d2min >= 0x1p-100f;
        if (f32) {
          const float Z = s1 / s0, c = gj / s0;
          const float lmin2 = lg2_approx(d2min);
          f32 = isfinite(Z) && isfinite(c);
          if (f32) {
            float ax = 0.f, ay = 0.f, al = 0.f;
            for (int s = 0; s < cnt; ++s) {
              const int64_t i = row[s];
              if (!dcheck(i >= 0 && i < n, kSiteData)) continue;
              const float* x = data + 3 * i;
              const float dx = __fsub_rn(qx, x[0]), dy = __fsub_rn(qy, x[1]);
              const float d2 = __fmaf_rn(dy, dy, __fmul_rn(dx, dx));
              const float w = grad_weight<MODE>(d2, d2min, lmin, hp);
              const float a = (x[2] - Z) * w, ar = a * rcp_approx(d2);
              ax = fmaf(ar, dx, ax);
              ay = fmaf(ar, dy, ay);
              al = fmaf(a, lg2_approx(d2) - lmin2, al);
              if (acc) {
                const float b = c * pf * ar;
                atomicAdd(&acc[i], make_float4(c * w, b * dx, b * dy, 0.f));
              }
            }
            gqx = -c * pf * ax;
            gqy = -c * pf * ay;
            const float gpf = (-0.5f * 0.6931471805599453f) * c * al;
            gp = gpf;
            qs = KnnQState{double(Z), double(c), double(d2min), lmin, kKnnQF32};
          }
        }
        if (!f32) {
          const KnnGradF64 r64 =
              knn_grad_query_f64(row, cnt, data, qx, qy, p, gj, acc);
          gqx = r64.gqx;
          gqy = r64.gqy;
          gp = r64.gp;
          qs = KnnQState{r64.Z, r64.c, r64.dmin, 0.f, kKnnQF64};
        }
      }
      if (grad_q) {
        grad_q[2 * int64_t(j)] = gqx;
        grad_q[2 * int64_t(j) + 1] = gqy;
      }
      if (qstate) qstate[j] = qs;
      if (gp_query) gp_query[j] = gp;
    }
  }
  if (grad_p && !gp_query) {
    gp = warp_sum(gp);
    if ((threadIdx.x & 31) == 0 && gp != 0.0) atomicAdd(grad_p, gp);
  }
}

// ----------------------------------------- deterministic k-NN gradients
//
// Point-major data-side terms in a fixed order: every (point, query)
// selection becomes one 64-bit item, the point index above the query index,
// listed query-major; a stable radix sort by point keeps each point's
// queries in increasing order; 8 lanes per point (a whole warp for a point
// with many terms) then recompute its terms from the queries' states and
// sum them lane-strided and by a fixed shuffle tree.
// dL/dp is summed over queries in index order by a fixed two-level tree.
// Nothing depends on the order in which threads or atomics ran, so two calls
// on the same inputs give the same bits.

// Pair (x = j k + s), packed as key << 32 | j: key = the selected point
// (the hit index for slot 0 of a hit query), or n for an empty slot.
__global__ void __launch_bounds__(256)
    knn_pairs_kernel(const int32_t* __restrict__ nbr, const int32_t* __restrict__ hit,
                     const KnnQState* __restrict__ qstate, int64_t m, int k, int64_t n,
                     uint64_t* __restrict__ items) {
  const int64_t x = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (x >= m * k) return;
  const int64_t j = x / k;
  const int sl = static_cast<int>(x - j * k);
  const int mode = qstate[j].mode;
  int64_t key = n;
  if (mode == kKnnQHit) {
    if (sl == 0 && dcheck(hit[j] >= 0 && hit[j] < n, kSiteData)) key = hit[j];
  } else if (mode == kKnnQF32 || mode == kKnnQF64) {
    const int32_t i = nbr[x];
    if (i >= 0 && dcheck(i < n, kSiteData)) key = i;
  }
  items[x] = (uint64_t(key) << 32) | uint64_t(uint32_t(j));
}

// First and one-past-last position of each point's run of sorted keys (the
// caller zeroes both arrays: a point no query selected has an empty run).
__global__ void __launch_bounds__(256)
    knn_runs_kernel(const uint64_t* __restrict__ items, int64_t count, int64_t n,
                    int32_t* __restrict__ first, int32_t* __restrict__ last) {
  const int64_t x = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (x >= count) return;
  const uint32_t key = uint32_t(items[x] >> 32);
  if (key >= n) return;
  if (x == 0 || uint32_t(items[x - 1] >> 32) != key) first[key] = static_cast<int32_t>(x);
  if (x == count - 1 || uint32_t(items[x + 1] >> 32) != key)
    last[key] = static_cast<int32_t>(x + 1);
}

// The data-side terms (dL/dz, dL/dx, dL/dy) of point (x0, y0, zi) for the
// query of pair item q, recomputed as the query-major kernel computes them,
// added to (gz, gx, gy).
template <int MODE>
__device__ __forceinline__ void knn_point_term(uint64_t item, const KnnQState* __restrict__ qstate,
                                               const float* __restrict__ queries,
                                               const float* __restrict__ grad_out, float x0,
                                               float y0, float zi, double p, float hp, float pf,
                                               float& gz, float& gx, float& gy) {
  const int64_t j = uint32_t(item);  // the pair's query
  const KnnQState st = qstate[j];
  const float gj = grad_out[j];
  const float qx = queries[2 * j], qy = queries[2 * j + 1];
  if (st.mode == kKnnQHit) {
    gz += gj;
  } else if (st.mode == kKnnQF32) {
    const float Z = static_cast<float>(st.Z), c = static_cast<float>(st.c);
    const float d2min = static_cast<float>(st.d2min);
    const float dx = __fsub_rn(qx, x0), dy = __fsub_rn(qy, y0);
    const float d2 = __fmaf_rn(dy, dy, __fmul_rn(dx, dx));
    const float w = grad_weight<MODE>(d2, d2min, st.lmin, hp);
    const float ar = (zi - Z) * w * rcp_approx(d2);
    const float bb = c * pf * ar;
    gz += c * w;
    gx += bb * dx;
    gy += bb * dy;
  } else if (st.mode == kKnnQF64) {
    const double ex = double(qx) - x0, ey = double(qy) - y0, e2 = ex * ex + ey * ey;
    const double w = pow(st.d2min / e2, 0.5 * p);
    const double av = (double(zi) - st.Z) * w;
    gz += static_cast<float>(st.c * w);
    gx += static_cast<float>(st.c * p * av * ex / e2);
    gy += static_cast<float>(st.c * p * av * ey / e2);
  }
}

// A warp takes kPointsPerWarp consecutive data points and sums each one's
// terms in increasing query order: normally kPointLanes lanes per point,
// lane l summing the point's terms l, l + kPointLanes, ... and the lanes'
// sums joined by a fixed shuffle tree (about k terms per point when m = n,
// so a whole warp per point would leave most lanes one term and the warp
// waiting on it); if one of its points has more than kHeavyTerms terms
// (clustered data: a point inside a blob), all 32 lanes take the warp's
// points one after the other the same way.  The choice depends only on the
// counts, so a point's order of summation is the same in every call.
constexpr int kPointLanes = 8;
constexpr int kPointsPerWarp = 32 / kPointLanes;
constexpr int kHeavyTerms = 16 * kPointLanes;
template <int MODE>
__global__ void __launch_bounds__(256)
    knn_point_grad_kernel(const int32_t* __restrict__ first, const int32_t* __restrict__ last,
                          const uint64_t* __restrict__ items, const KnnQState* __restrict__ qstate,
                          const float* __restrict__ queries, const float* __restrict__ data,
                          int64_t n, double p, const float* __restrict__ grad_out,
                          float* __restrict__ grad_z, float* __restrict__ grad_xy) {
  constexpr unsigned kFull = 0xffffffffu;
  const int lane32 = threadIdx.x & 31;
  const int64_t i0 = ((int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5) * kPointsPerWarp;
  const int g = lane32 / kPointLanes, lane = lane32 % kPointLanes;
  const int64_t i = i0 + g;
  const bool own = i < n;  // every lane stays for the shuffles
  float x0 = 0.f, y0 = 0.f, zi = 0.f;
  int a = 0, b = 0;
  if (own) {
    x0 = data[3 * i];
    y0 = data[3 * i + 1];
    zi = data[3 * i + 2];
    a = first[i];
    b = last[i];
  }
  const float hp = static_cast<float>(0.5 * p), pf = static_cast<float>(p);
  auto put = [&](int64_t pi, float gz, float gx, float gy) {
    if (grad_z) grad_z[pi] = gz;
    if (grad_xy) reinterpret_cast<float2*>(grad_xy)[pi] = make_float2(gx, gy);
  };
  if (!__any_sync(kFull, b - a > kHeavyTerms)) {
    float gz = 0.f, gx = 0.f, gy = 0.f;
    for (int q = a + lane; q < b; q += kPointLanes)
      knn_point_term<MODE>(items[q], qstate, queries, grad_out, x0, y0, zi, p, hp, pf, gz, gx, gy);
#pragma unroll
    for (int o = kPointLanes / 2; o > 0; o >>= 1) {
      gz += __shfl_xor_sync(kFull, gz, o);
      gx += __shfl_xor_sync(kFull, gx, o);
      gy += __shfl_xor_sync(kFull, gy, o);
    }
    if (own && lane == 0) put(i, gz, gx, gy);
    return;
  }
  for (int h = 0; h < kPointsPerWarp; ++h) {  // the whole warp on each point
    const int src = h * kPointLanes;
    const float hx = __shfl_sync(kFull, x0, src), hy = __shfl_sync(kFull, y0, src);
    const float hz = __shfl_sync(kFull, zi, src);
    const int ha = __shfl_sync(kFull, a, src), hb = __shfl_sync(kFull, b, src);
    float gz = 0.f, gx = 0.f, gy = 0.f;
    for (int q = ha + lane32; q < hb; q += 32)
      knn_point_term<MODE>(items[q], qstate, queries, grad_out, hx, hy, hz, p, hp, pf, gz, gx, gy);
    gz = warp_sum(gz);
    gx = warp_sum(gx);
    gy = warp_sum(gy);
    if (lane32 == 0 && i0 + h < n) put(i0 + h, gz, gx, gy);
  }
}

// Fixed-order sum of v[0 .. count): CTA b sums its contiguous slice (thread
// t takes every 256th value from t, then a fixed shuffle and shared-memory
// tree), then one CTA sums the CTA totals the same way.
constexpr int kDetSumCtas = 256;
__global__ void __launch_bounds__(256)
    fixed_sum_kernel(const double* __restrict__ v, int64_t count, double* __restrict__ out) {
  __shared__ double part[8];
  const int64_t per = (count + gridDim.x - 1) / gridDim.x;
  const int64_t lo = int64_t(blockIdx.x) * per, hi = min(count, lo + per);
  double acc = 0.0;
  for (int64_t x = lo + threadIdx.x; x < hi; x += blockDim.x) acc += v[x];
  acc = warp_sum(acc);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double tot = 0.0;
    for (int w = 0; w < 8; ++w) tot += part[w];
    out[blockIdx.x] = tot;
  }
}

// Copies the per-point accumulators out to the caller's gradient arrays.
__global__ void __launch_bounds__(256)
    knn_grad_copy_kernel(const float4* acc, int64_t n, float* __restrict__ grad_z,
                         float* __restrict__ grad_xy) {
  pdl_trigger();
  pdl_wait();
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float4 v = acc[i];
  if (grad_z) grad_z[i] = v.x;
  if (grad_xy) reinterpret_cast<float2*>(grad_xy)[i] = make_float2(v.y, v.z);
}

size_t round_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

// Queries that, a thread each, fill the GPU: up to as many heavy ones are listed
// (see list_if_heavy).
int64_t heavy_limit(int sm_count) { return int64_t(sm_count) * 1024; }

// Up to this many queries that lie in dense surroundings, or that the search by
// counts left, a warp searches for each (64 blobs, queries in the blobs too,
// threads / warps: k = 8, 30,000 of them 252 / 235 us, 100,000 293 / 440; k = 64,
// 30,000 633 / 220, 100,000 847 / 931).
int64_t knn_few(int k) {
  return std::min(16384 + 4096 * int64_t(k), 32768 + 512 * int64_t(k));
}

// Whether a call's queries are sampled: where the result is asked for.
bool knn_sampled(int k, int64_t m) {
  return k >= kSampleK && m > knn_few(k);
}

int scan_tiles_of(int64_t max_cells) {
  return static_cast<int>((max_cells + 1 + kScanTile - 1) / kScanTile);
}

}  // namespace

// At least two data points per cell on average: finer cells cost more row
// lookups per query than the candidates they save.
int64_t local_max_cells(int64_t n) {
  return std::min<int64_t>(int64_t(kMaxCellsPerAxis) * kMaxCellsPerAxis,
                           std::max<int64_t>(1024, n / 2));
}

LocalLayout local_layout(int64_t n, int64_t m, int64_t max_cells) {
  LocalLayout L;
  L.max_cells = max_cells;
  const size_t len = size_t(max_cells + 1 + 3) / 4 * 16;  // whole int4s
  size_t off = 0;
  L.off_grid = off;       off += round_up(sizeof(GridDev), 256);
  L.off_counts_d = off;   off += round_up(len, 256);
  L.off_counts_q = off;   off += round_up(len, 256);
  L.off_starts_d = off;   off += round_up(len, 256);
  L.off_starts_q = off;   off += round_up(len, 256);
  L.off_sums = off;       off += round_up(size_t(2 * scan_tiles_of(max_cells)) * 4, 256);
  L.off_sorted = off;     off += round_up(size_t(n) * 16, 256);
  L.off_qrec = off;       off += round_up(size_t(m) * 16, 256);
  L.off_hard = off;       off += round_up(size_t(m) * 4, 256);
  L.off_bpre = off;
  off += round_up(size_t(kMaxBlocksPerAxis) * (kMaxBlocksPerAxis + 1) * 4, 256);
  // (gx + 1)(gy + 1) = cells + gx + gy + 1 entries, cells <= max_cells.
  L.off_sat = off;
  off += round_up(size_t(max_cells + 2 * kMaxCellsPerAxis + 1) * 4, 256);
  L.bytes = off;
  return L;
}

namespace {

// Enqueues the grid build shared by both local forms: bounding box and plan,
// histograms, scans, scatter of data and queries into cell order.
cudaError_t launch_grid_sort(const float* data, int64_t n, const float* queries, int64_t m,
                             double radius, int knn_k, void* workspace, const LocalLayout& L,
                             int sm_count, cudaStream_t s, bool sort_queries = true) {
  unsigned char* ws = static_cast<unsigned char*>(workspace);
  GridDev* grid = reinterpret_cast<GridDev*>(ws + L.off_grid);
  int32_t* counts_d = reinterpret_cast<int32_t*>(ws + L.off_counts_d);
  int32_t* counts_q = reinterpret_cast<int32_t*>(ws + L.off_counts_q);
  int32_t* starts_d = reinterpret_cast<int32_t*>(ws + L.off_starts_d);
  int32_t* starts_q = reinterpret_cast<int32_t*>(ws + L.off_starts_q);
  int32_t* sums = reinterpret_cast<int32_t*>(ws + L.off_sums);
  float4* sorted = reinterpret_cast<float4*>(ws + L.off_sorted);
  float4* qrec = reinterpret_cast<float4*>(ws + L.off_qrec);
  const int max_tiles = scan_tiles_of(L.max_cells);

  cudaError_t e = cudaMemsetAsync(grid, 0xff, sizeof(GridDev), s);
  if (e != cudaSuccess) return e;
  const unsigned bgrid = static_cast<unsigned>(
      std::max<int64_t>(1, std::min<int64_t>(int64_t(sm_count) * 4, (n + 255) / 256)));
  e = launch_pdl(box_plan_kernel, bgrid, 256, 0, s, data, n, grid, radius,
                 1.0 / double(L.max_cells), knn_k, L.max_cells, counts_d, counts_q);
  if (e != cudaSuccess) return e;
  // Without the query sort, the queries join none of the three passes and
  // their records are written in the caller's order.
  const int64_t mq = sort_queries ? m : 0;
  const int sample = knn_k > 0 ? (knn_sampled(knn_k, m) ? knn_k : 0)
                               : m <= heavy_limit(sm_count) ? 0 : kSampleRadius;
  const unsigned pgrid = static_cast<unsigned>((n + mq + 255) / 256);
  e = launch_pdl(count_kernel, pgrid, 256, 0, s, grid, data, n, queries, mq, counts_d, counts_q);
  if (e == cudaSuccess)
    e = launch_pdl(scan_kernel, dim3(max_tiles, sort_queries ? 2 : 1), kScanBlock, 0, s, grid,
                   counts_d, counts_q, starts_d, starts_q, sums, max_tiles, 0);
  if (e == cudaSuccess)
    e = launch_pdl(scatter_kernel, pgrid + (sample != 0 ? 1 : 0), kSampleQueries, 0, s, grid, data,
                   n, queries, mq, m, sample, starts_d, starts_q, sums, max_tiles, counts_d,
                   counts_q, sorted, qrec);
  if (e == cudaSuccess && !sort_queries && m > 0)
    e = launch_pdl(query_identity_kernel, static_cast<unsigned>((m + 255) / 256), 256, 0, s, queries,
                   m, qrec);
  return e;
}

}  // namespace

namespace {
// The k-NN search's count tables of the data cells.
cudaError_t launch_count_tables(const GridDev* grid, const int32_t* starts, const int32_t* base,
                                int32_t* bpre, int32_t* sat, cudaStream_t s) {
  cudaError_t e = launch_pdl(block_prefix_kernel, kMaxBlocksPerAxis, kMaxBlocksPerAxis, 0, s, grid,
                             starts, base, bpre);
  if (e == cudaSuccess)
    e = launch_pdl(sat_kernel, (kMaxCellsPerAxis + 1 + kSatCols - 1) / kSatCols,
                   kSatCols * kSatWarps, 0, s, grid, starts, base, sat);
  return e;
}

// The values of sorted queries: one thread each, then a warp for each heavy one.
cudaError_t launch_radius_queries(const GridDev* grid, const float4* sorted, int64_t n,
                                  const int32_t* starts, const int32_t* base, const float4* qrec,
                                  int64_t m, double p, float r2f, float r2t, float* out,
                                  int32_t* count_out, double radius, bool modified, int32_t* heavy,
                                  bool scattered, unsigned qgrid, int sm_count, cudaStream_t s) {
  unsigned* heavy_count = &const_cast<GridDev*>(grid)->hard;
  auto run = [&](auto mode, auto wmode) {
    constexpr int M = decltype(mode)::value, W = decltype(wmode)::value;
    const cudaError_t e = launch_pdl(
        local_query_kernel<M, W>, qgrid, kLocalThreads, 0, s, grid, sorted, n, starts, base, qrec, m,
        p, r2f, r2t, out, count_out, radius, heavy_limit(sm_count), scattered, heavy_count, heavy);
    if (e != cudaSuccess) return e;
    return launch_pdl(local_heavy_kernel<M, W>, unsigned(sm_count) * 8, kHeavyThreads, 0, s, grid,
                      sorted, n, starts, base, qrec, m, p, r2f, r2t, out, count_out, radius,
                      heavy_count, heavy);
  };
  using P2 = std::integral_constant<int, kPow2>;
  using PG = std::integral_constant<int, kPowGeneral>;
  using WS = std::integral_constant<int, kWeightShepard>;
  using WM = std::integral_constant<int, kWeightModified>;
  if (modified) return p == 2.0 ? run(P2{}, WM{}) : run(PG{}, WM{});
  return p == 2.0 ? run(P2{}, WS{}) : run(PG{}, WS{});
}
}  // namespace

cudaError_t launch_local(const float* data, int64_t n, const float* queries, int64_t m, double p,
                         double radius, float* out, int32_t* count_out, void* workspace,
                         const LocalLayout& L, int sm_count, cudaStream_t s, bool sort_queries,
                         bool modified) {
  cudaError_t e = launch_grid_sort(data, n, queries, m, radius, 0, workspace, L, sm_count, s,
                                   sort_queries);
  if (e != cudaSuccess) return e;
  unsigned char* ws = static_cast<unsigned char*>(workspace);
  const GridDev* grid = reinterpret_cast<const GridDev*>(ws + L.off_grid);
  const int32_t* starts_d = reinterpret_cast<const int32_t*>(ws + L.off_starts_d);
  const int32_t* sums = reinterpret_cast<const int32_t*>(ws + L.off_sums);
  const float4* sorted = reinterpret_cast<const float4*>(ws + L.off_sorted);
  const float4* qrec = reinterpret_cast<const float4*>(ws + L.off_qrec);
  const float r2f = static_cast<float>(radius * radius);
  const float r2t = r2f > 0.f ? r2f : 0x1p-149f;
  const unsigned qgrid = static_cast<unsigned>((m + kLocalThreads - 1) / kLocalThreads);
  return launch_radius_queries(grid, sorted, n, starts_d, sums, qrec, m, p, r2f, r2t, out, count_out,
                               radius, modified, reinterpret_cast<int32_t*>(ws + L.off_hard), false,
                               qgrid, sm_count, s);
}

size_t local_grad_record_bytes(int64_t m) {
  return round_up(size_t(m) * sizeof(LocalGradRec), 256) +
         round_up(size_t(m) * sizeof(LocalGradRec64), 256);
}

cudaError_t launch_local_backward(const float* data, int64_t n, const float* queries, int64_t m,
                                  double p, double radius, const float* grad_out, float* grad_z,
                                  float* grad_xy, float* grad_q, double* grad_p, void* workspace,
                                  const LocalLayout& L, int sm_count, cudaStream_t s,
                                  bool modified) {
  // Cleared first, so that the kernels after the grid's memset overlap their
  // launches.
  cudaError_t e = cudaSuccess;
  if (grad_z && (e = cudaMemsetAsync(grad_z, 0, size_t(n) * 4, s)) != cudaSuccess) return e;
  if (grad_xy && (e = cudaMemsetAsync(grad_xy, 0, size_t(n) * 8, s)) != cudaSuccess) return e;
  if (grad_p && (e = cudaMemsetAsync(grad_p, 0, sizeof(double), s)) != cudaSuccess) return e;
  e = launch_grid_sort(data, n, queries, m, radius, 0, workspace, L, sm_count, s);
  if (e != cudaSuccess) return e;
  unsigned char* ws = static_cast<unsigned char*>(workspace);
  const GridDev* grid = reinterpret_cast<const GridDev*>(ws + L.off_grid);
  const int32_t* starts_d = reinterpret_cast<const int32_t*>(ws + L.off_starts_d);
  const int32_t* starts_q = reinterpret_cast<const int32_t*>(ws + L.off_starts_q);
  const int32_t* sums = reinterpret_cast<const int32_t*>(ws + L.off_sums);
  const int32_t* sums_q = sums + scan_tiles_of(L.max_cells);
  const float4* sorted = reinterpret_cast<const float4*>(ws + L.off_sorted);
  const float4* qrec = reinterpret_cast<const float4*>(ws + L.off_qrec);
  LocalGradRec* rec = reinterpret_cast<LocalGradRec*>(ws + L.bytes);
  LocalGradRec64* rec64 = reinterpret_cast<LocalGradRec64*>(
      ws + L.bytes + round_up(size_t(m) * sizeof(LocalGradRec), 256));
  const float r2f = static_cast<float>(radius * radius);
  const float r2t = r2f > 0.f ? r2f : 0x1p-149f;
  const unsigned qgrid = static_cast<unsigned>((m + kLocalThreads - 1) / kLocalThreads);
  const unsigned dgrid = static_cast<unsigned>((n + kLocalThreads - 1) / kLocalThreads);
  const bool data_side = grad_z || grad_xy;
  unsigned* heavy_count = &reinterpret_cast<GridDev*>(ws + L.off_grid)->hard;
  int32_t* heavy = reinterpret_cast<int32_t*>(ws + L.off_hard);
  auto run = [&](auto mode, auto wmode) {
    constexpr int M = decltype(mode)::value, W = decltype(wmode)::value;
    e = launch_pdl(local_grad_query_kernel<M, W>, qgrid, kLocalThreads, 0, s, grid, sorted, n,
                   starts_d, sums, qrec, m, p, r2f, r2t, grad_out, grad_q, grad_p, rec, rec64, radius,
                   heavy_limit(sm_count), heavy_count, heavy);
    if (e == cudaSuccess)
      e = launch_pdl(local_grad_heavy_kernel<M, W>, unsigned(sm_count) * 8, kHeavyThreads, 0, s,
                     grid, sorted, n, starts_d, sums, qrec, m, p, r2f, r2t, grad_out, grad_q, grad_p,
                     rec, rec64, radius, heavy_count, heavy);
    if (e == cudaSuccess && data_side)
      e = launch_pdl(local_grad_data_kernel<M, W>, dgrid, kLocalThreads, 0, s, grid, sorted, n,
                     starts_d, sums, starts_q, sums_q, qrec, m, rec, rec64, p, r2f, grad_z, grad_xy,
                     radius);
  };
  using P2 = std::integral_constant<int, kPow2>;
  using PG = std::integral_constant<int, kPowGeneral>;
  using WS = std::integral_constant<int, kWeightShepard>;
  using WM = std::integral_constant<int, kWeightModified>;
  if (modified) {
    if (p == 2.0) run(P2{}, WM{}); else run(PG{}, WM{});
  } else {
    if (p == 2.0) run(P2{}, WS{}); else run(PG{}, WS{});
  }
  return e != cudaSuccess ? e : cudaGetLastError();
}

size_t knn_grad_scratch_bytes(int64_t n, int64_t m, int k, bool deterministic) {
  size_t b = round_up(size_t(m) * 4, 256) * 2 + round_up(size_t(m) * size_t(k) * 4, 256) +
             round_up(size_t(n) * 16, 256);
  if (deterministic) {
    const int64_t pairs = m * int64_t(k);
    b += round_up(size_t(pairs) * 8, 256) + radix_sort_scratch_bytes(pairs) +
         2 * round_up(size_t(n) * 4, 256) + round_up(size_t(m) * sizeof(KnnQState), 256) +
         round_up(size_t(m) * 8, 256) + round_up(size_t(kDetSumCtas) * 8, 256);
  }
  return b;
}

namespace {
// The deterministic k-NN gradient after the search (rows sorted by key):
// query-major kernel without atomics (states, dL/dq, per-query dL/dp), the
// pair list, its stable sort by point, the runs, the point-major kernel and
// the fixed-order dL/dp sum.
cudaError_t launch_knn_backward_fixed_order(const float* data, int64_t n, const float* queries,
                                            int64_t m, double p, int k, const float* grad_out,
                                            float* grad_z, float* grad_xy, float* grad_q,
                                            double* grad_p, unsigned char* ws,
                                            const LocalLayout& L, const int32_t* hit,
                                            const int32_t* nbr, cudaStream_t s) {
  const int64_t pairs = m * int64_t(k);
  size_t off = L.bytes + round_up(size_t(m) * 4, 256) * 2 + round_up(size_t(pairs) * 4, 256) +
               round_up(size_t(n) * 16, 256);
  auto take = [&](size_t bytes) {
    unsigned char* ptr = ws + off;
    off += round_up(bytes, 256);
    return ptr;
  };
  uint64_t* items = reinterpret_cast<uint64_t*>(take(size_t(pairs) * 8));
  void* sort_scratch = take(radix_sort_scratch_bytes(pairs));
  int32_t* first = reinterpret_cast<int32_t*>(take(size_t(n) * 4));
  int32_t* last = reinterpret_cast<int32_t*>(take(size_t(n) * 4));
  KnnQState* qstate = reinterpret_cast<KnnQState*>(take(size_t(m) * sizeof(KnnQState)));
  double* gpq = reinterpret_cast<double*>(take(size_t(m) * 8));
  double* gpart = reinterpret_cast<double*>(take(size_t(kDetSumCtas) * 8));

  const float4* qrec = reinterpret_cast<const float4*>(ws + L.off_qrec);
  const unsigned qgrid = static_cast<unsigned>((m + kLocalThreads - 1) / kLocalThreads);
  if (p == 2.0)
    knn_grad_kernel<kPow2><<<qgrid, kLocalThreads, 0, s>>>(qrec, m, data, n, nbr, hit, k, p,
                                                           grad_out, nullptr, grad_q, grad_p,
                                                           qstate, gpq);
  else
    knn_grad_kernel<kPowGeneral><<<qgrid, kLocalThreads, 0, s>>>(qrec, m, data, n, nbr, hit, k,
                                                                 p, grad_out, nullptr, grad_q,
                                                                 grad_p, qstate, gpq);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (grad_p) {
    fixed_sum_kernel<<<kDetSumCtas, 256, 0, s>>>(gpq, m, gpart);
    fixed_sum_kernel<<<1, 256, 0, s>>>(gpart, kDetSumCtas, grad_p);
  }
  if (!grad_z && !grad_xy) return cudaGetLastError();
  knn_pairs_kernel<<<static_cast<unsigned>((pairs + 255) / 256), 256, 0, s>>>(
      nbr, hit, qstate, m, k, n, items);
  int bits = 1;
  while (bits < 32 && (uint64_t(1) << bits) <= uint64_t(n)) ++bits;  // keys in [0, n]
  uint64_t* sorted_items = nullptr;
  if ((e = radix_sort_items(items, pairs, bits, sort_scratch, s, &sorted_items)) != cudaSuccess)
    return e;
  if ((e = cudaMemsetAsync(first, 0, size_t(n) * 4, s)) != cudaSuccess) return e;
  if ((e = cudaMemsetAsync(last, 0, size_t(n) * 4, s)) != cudaSuccess) return e;
  knn_runs_kernel<<<static_cast<unsigned>((pairs + 255) / 256), 256, 0, s>>>(sorted_items, pairs, n,
                                                                             first, last);
  const unsigned pgrid =
      static_cast<unsigned>(((n + kPointsPerWarp - 1) / kPointsPerWarp * 32 + 255) / 256);
  if (p == 2.0)
    knn_point_grad_kernel<kPow2><<<pgrid, 256, 0, s>>>(first, last, sorted_items, qstate, queries,
                                                       data, n, p, grad_out, grad_z, grad_xy);
  else
    knn_point_grad_kernel<kPowGeneral><<<pgrid, 256, 0, s>>>(first, last, sorted_items, qstate,
                                                             queries, data, n, p, grad_out,
                                                             grad_z, grad_xy);
  return cudaGetLastError();
}
}  // namespace

cudaError_t launch_knn_backward(const float* data, int64_t n, const float* queries, int64_t m,
                                double p, int k, const float* grad_out, float* grad_z,
                                float* grad_xy, float* grad_q, double* grad_p, void* workspace,
                                const LocalLayout& L, int sm_count, cudaStream_t s,
                                bool sort_queries, bool deterministic, bool warp_search) {
  unsigned char* ws = static_cast<unsigned char*>(workspace);
  float* zbuf = reinterpret_cast<float*>(ws + L.bytes);
  int32_t* hit = reinterpret_cast<int32_t*>(ws + L.bytes + round_up(size_t(m) * 4, 256));
  int32_t* nbr = reinterpret_cast<int32_t*>(ws + L.bytes + 2 * round_up(size_t(m) * 4, 256));
  const bool data_side = grad_z || grad_xy;
  float4* acc = data_side && !deterministic
                    ? reinterpret_cast<float4*>(ws + L.bytes + 2 * round_up(size_t(m) * 4, 256) +
                                                round_up(size_t(m) * size_t(k) * 4, 256))
                    : nullptr;
  // Cleared first, so that the kernels after the grid's memset overlap their
  // launches.
  cudaError_t e = cudaSuccess;
  if (acc && (e = cudaMemsetAsync(acc, 0, size_t(n) * 16, s)) != cudaSuccess) return e;
  if (grad_p && !deterministic && (e = cudaMemsetAsync(grad_p, 0, sizeof(double), s)) != cudaSuccess)
    return e;
  // Deterministic mode: rows in key order, so each query's own sums run in
  // one fixed order too.
  e = launch_knn(data, n, queries, m, p, k, zbuf, nbr, nullptr, workspace, L, sm_count, s, hit,
                 sort_queries, deterministic, warp_search);
  if (e != cudaSuccess) return e;
  if (deterministic)
    return launch_knn_backward_fixed_order(data, n, queries, m, p, k, grad_out, grad_z, grad_xy,
                                           grad_q, grad_p, ws, L, hit, nbr, s);
  const float4* qrec = reinterpret_cast<const float4*>(ws + L.off_qrec);
  const unsigned qgrid = static_cast<unsigned>((m + kLocalThreads - 1) / kLocalThreads);
  auto grad = p == 2.0 ? knn_grad_kernel<kPow2> : knn_grad_kernel<kPowGeneral>;
  grad<<<qgrid, kLocalThreads, 0, s>>>(qrec, m, data, n, nbr, hit, k, p, grad_out, acc, grad_q,
                                       grad_p, nullptr, nullptr);
  e = cudaGetLastError();
  if (e == cudaSuccess && acc)
    e = launch_pdl(knn_grad_copy_kernel, static_cast<unsigned>((n + 255) / 256), 256, 0, s, acc, n,
                   grad_z, grad_xy);
  return e;
}

cudaError_t debug_check_failures(unsigned* sites, bool* enabled) {
#ifdef IDW_DEBUG_CHECKS
  *enabled = true;
  cudaError_t e = cudaMemcpyFromSymbol(sites, g_debug_failures, sizeof(unsigned));
  const unsigned zero = 0;
  if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_debug_failures, &zero, sizeof(unsigned));
  return e;
#else
  *enabled = false;
  *sites = 0;
  return cudaSuccess;
#endif
}

namespace {

size_t knn_smem_bytes(int k) { return size_t(k) * kKnnThreads * sizeof(u64); }

// Up to this many queries, a warp searches for each: a thread per query
// leaves the GPU idle there.  Measured on a GB300 against n = 2^20 uniform
// points, whole query call on a prepared index, thread / warp per query:
// m = 10,007 61 / 43 us at k = 8, 107 / 46 us at k = 32; m = 100,000
// 69 / 143 us at k = 8, 141 / 168 us at k = 32.
int64_t knn_warp_queries(int k) { return std::min<int64_t>(8192 + 1024 * int64_t(k), 65536); }

// Up to this many queries, those that are not easy are listed.  Beyond it
// every warp of the single-thread search has hard queries to overlap with and
// the GPU is full either way (64 blobs, n = 2^20, k = 8, threads alone / with
// warps: m = 10,007 1010 / 74 us, 100,000 1090 / 263 us, 2^20 1440 / 1770 us).
constexpr int64_t kKnnHardQueries = int64_t(1) << 19;

// Above this many queries k <= 32 is counted too: below it the counts' two walks
// are bound by latency as the heaps are (100,000 queries, k = 32, uniform 143 us
// by counts and 141 by heaps, on a lattice 124 and 102; 131,072: 140 and 196,
// 127 and 134).
constexpr int64_t kCountQueries = 7 * (int64_t(1) << 14);

// Up to this many queries the heap search after the counts has a block for each
// 32 of them, which is 5-10% faster where it has them all to do (64 blobs, queries
// in the blobs too, k = 64, m = 100,000: 862 us, 934 fetched) and costs a
// nanosecond each where it has none.
constexpr int64_t kUnfetchedQueries = int64_t(1) << 18;
static_assert(kUnfetchedQueries <= kKnnHardQueries, "these list their hard queries");

// The search over sorted queries, by warps for few of them, else by threads
// with warps for the hard ones; the launch arguments both share.
struct KnnArgs {
  GridDev* grid;
  const float4* sorted;
  const int32_t *starts, *base, *bpre, *sat;
  const float4* qrec;
  const float* data;
  int64_t n, m;
  double p;
  int k;
  float* out;
  int32_t* nbr_out;
  float* kd2_out;
  int32_t* hit_out;
  bool sort_rows;
  int32_t* hard;
};

cudaError_t launch_knn_search(const KnnArgs& a, int sm_count, cudaStream_t s) {
  // Rows in search order (the gradients' plain FP32 sums follow it) keep the
  // heap search's order.
  const bool warps = !a.nbr_out || a.sort_rows;
  const bool all_warps = warps && a.m <= knn_warp_queries(a.k);
  // Without lists and from k = 17 on, evenly spread data are searched by counts
  // (uniform n = m = 2^20, heaps / counts: k = 16 389 / 383 us, 24 550 / 454,
  // 32 723 / 475, 64 1552 / 718); the device decides which of the two runs.
  const bool counted = !all_warps && !a.nbr_out && !a.hit_out && a.k > 16 &&
                       (a.k > 32 || a.m > kCountQueries);
  const bool list = warps && !all_warps && a.m <= kKnnHardQueries;
  const KnnLists lists{&a.grid->hard, &a.grid->left, all_warps ? nullptr : a.hard,
                       static_cast<unsigned>(knn_few(a.k))};
  const bool pow2 = a.p == 2.0;
  cudaError_t e = cudaSuccess;
  if (counted)
    e = launch_pdl(pow2 ? knn_count_kernel<kPow2> : knn_count_kernel<kPowGeneral>,
                   static_cast<unsigned>((a.m + kCountThreads - 1) / kCountThreads), kCountThreads, 0,
                   s, a.grid, a.sorted, a.starts, a.base, a.sat, a.qrec, a.data, a.n,
                   a.m, a.p, a.k, a.out, a.kd2_out, lists);
  if (e == cudaSuccess && !all_warps) {
    const size_t smem = knn_smem_bytes(a.k);  // below the default limit (k <= 64: 16 KB)
    const unsigned groups = static_cast<unsigned>((a.m + kKnnThreads - 1) / kKnnThreads);
    const unsigned resident = unsigned(sm_count) * 32;
    auto heap = [&](auto list_these, auto from) {
      constexpr bool L = decltype(list_these)::value;
      constexpr int F = decltype(from)::value;
      auto kernel = pow2 ? knn_query_kernel<kPow2, L, F> : knn_query_kernel<kPowGeneral, L, F>;
      const unsigned blocks = F == kFromLeftFetched ? std::min(groups, resident) : groups;
      // A kernel that starts early has its first blocks placed on the SMs that
      // the one before it leaves free; where all blocks fit at once, they stay
      // so (uniform m = 30,000, k = 32, gradient call: 270 us, 204 started
      // plainly; index call of 100,000, k = 16: 99 and 89).  The short searches
      // for a few neighbours gain more from the early start (m = 10,007, k = 1:
      // 18 us, 22 plainly).
      if (groups >= resident || a.k < 4)
        return launch_pdl(kernel, blocks, kKnnThreads, smem, s, a.grid, a.sorted, a.starts, a.base,
                          a.bpre, a.sat, a.qrec, a.data, a.n, a.m, a.p, a.k, a.out, a.nbr_out,
                          a.kd2_out, a.hit_out, a.sort_rows, lists, &a.grid->next);
      kernel<<<blocks, kKnnThreads, smem, s>>>(a.grid, a.sorted, a.starts, a.base, a.bpre, a.sat,
                                               a.qrec, a.data, a.n, a.m, a.p, a.k, a.out, a.nbr_out,
                                               a.kd2_out, a.hit_out, a.sort_rows, lists, &a.grid->next);
      return cudaGetLastError();
    };
    using All = std::integral_constant<int, kFromAll>;
    using Left = std::integral_constant<int, kFromLeft>;
    using Fetched = std::integral_constant<int, kFromLeftFetched>;
    if (counted && a.m <= kUnfetchedQueries)
      e = heap(std::true_type{}, Left{});
    else if (counted)
      e = list ? heap(std::true_type{}, Fetched{}) : heap(std::false_type{}, Fetched{});
    else
      e = list ? heap(std::true_type{}, All{}) : heap(std::false_type{}, All{});
  }
  if (e != cudaSuccess || (!all_warps && !list && !counted)) return e;
  constexpr int per_block = kKnnWarpThreads / 32;
  // The lists' lengths are known on the device only: enough blocks to fill the
  // GPU stride over them.
  const int64_t blocks = all_warps ? (a.m + per_block - 1) / per_block : int64_t(sm_count) * 8;
  auto kernel = a.k <= 32 ? (pow2 ? knn_warp_kernel<kPow2, 3> : knn_warp_kernel<kPowGeneral, 3>)
                          : (pow2 ? knn_warp_kernel<kPow2, 4> : knn_warp_kernel<kPowGeneral, 4>);
  return launch_pdl(kernel, static_cast<unsigned>(blocks), kKnnWarpThreads, 0, s, a.grid, a.sorted,
                    a.starts, a.base, a.sat, a.qrec, a.data, a.n, a.m, a.p, a.k, a.out, a.nbr_out,
                    a.kd2_out, a.hit_out, a.sort_rows, lists);
}

}  // namespace

cudaError_t launch_knn(const float* data, int64_t n, const float* queries, int64_t m, double p,
                       int k, float* out, int32_t* nbr_out, float* kd2_out, void* workspace,
                       const LocalLayout& L, int sm_count, cudaStream_t s, int32_t* hit_out,
                       bool sort_queries, bool sort_rows, bool warp_search) {
  cudaError_t e = cudaSuccess;
  const size_t sync_smem = knn_sync_smem_bytes(k);
  if (warp_search) {
    e = cudaFuncSetAttribute(knn_sync_kernel<kPow2>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, int(sync_smem));
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(knn_sync_kernel<kPowGeneral>,
                               cudaFuncAttributeMaxDynamicSharedMemorySize, int(sync_smem));
  }
  if (e != cudaSuccess) return e;
  e = launch_grid_sort(data, n, queries, m, 0.0, k, workspace, L, sm_count, s, sort_queries);
  if (e != cudaSuccess) return e;
  unsigned char* ws = static_cast<unsigned char*>(workspace);
  const GridDev* grid = reinterpret_cast<const GridDev*>(ws + L.off_grid);
  const int32_t* starts_d = reinterpret_cast<const int32_t*>(ws + L.off_starts_d);
  const int32_t* sums = reinterpret_cast<const int32_t*>(ws + L.off_sums);
  const float4* sorted = reinterpret_cast<const float4*>(ws + L.off_sorted);
  const float4* qrec = reinterpret_cast<const float4*>(ws + L.off_qrec);
  int32_t* bpre = reinterpret_cast<int32_t*>(ws + L.off_bpre);
  int32_t* sat = reinterpret_cast<int32_t*>(ws + L.off_sat);
  e = launch_count_tables(grid, starts_d, sums, bpre, sat, s);
  if (e != cudaSuccess) return e;
  if (!warp_search)
    return launch_knn_search(
        KnnArgs{reinterpret_cast<GridDev*>(ws + L.off_grid), sorted, starts_d, sums, bpre, sat, qrec,
                data, n, m, p, k, out, nbr_out, kd2_out, hit_out, sort_rows,
                reinterpret_cast<int32_t*>(ws + L.off_hard)},
        sm_count, s);
  const unsigned qgrid = static_cast<unsigned>((m + kKnnThreads - 1) / kKnnThreads);
  auto kernel = p == 2.0 ? knn_sync_kernel<kPow2> : knn_sync_kernel<kPowGeneral>;
  return launch_pdl(kernel, qgrid, kKnnThreads, sync_smem, s, grid, sorted, starts_d, sums, bpre, sat,
                    qrec, data, n, m, p, k, out, nbr_out, kd2_out, hit_out, sort_rows);
}

namespace {

// Copies an index's plan into a query call's scratch with the tickets reset.
// For the radius form (radius > 0) the reach is recomputed for the call's
// radius, which the host has checked is at most the build radius, so rho
// stays below 2 and the coverage argument of the plan still holds.
__device__ __forceinline__ void copy_plan(const GridDev* src,
                                          GridDev* dst, double radius) {
  GridDev g = *src;
  g.box_ticket = 0xffffffffu;
  g.scan_ticket = 0xffffffffu;
  g.hard = g.left = g.next = 0u;
  g.beyond = g.dense = 0u;
  if (radius > 0.0 && g.inv2 > 0.f)
    g.rho = __fmaf_ru(__fmul_ru(__double2float_ru(radius), g.inv2), 0.5f + 0x1p-9f, 0x1p-8f);
  *dst = g;
}

// First kernel of a query call on an index: the plan copy and, for the query
// sort, the histogram's clearing, or else the records in the caller's order.
// In both the first block also samples the call's queries (see sample_queries).
struct IndexCells {
  const int32_t *starts, *base;
  int64_t n;
};
__device__ __forceinline__ void index_plan(const GridDev* src, GridDev* dst, double radius,
                                           const IndexCells& data, const float* queries, int64_t m,
                                           int sample) {
  if (blockIdx.x != 0) return;
  if (threadIdx.x == 0) copy_plan(src, dst, radius);
  if (sample != 0) {
    __syncthreads();
    const GridDev g = *dst;
    sample_queries(dst, g, data.starts, data.base, data.n, queries, m, sample);
  }
}
__global__ void __launch_bounds__(256)
    index_prep_kernel(const GridDev* src, GridDev* dst, double radius, const IndexCells data,
                      const float* queries, int64_t m, int sample, int32_t* counts) {
  pdl_trigger();
  pdl_wait();
  index_plan(src, dst, radius, data, queries, m, sample);
  zero_counts(counts, count_int4s(src->cells));
}
__global__ void __launch_bounds__(256)
    index_identity_kernel(const GridDev* src, GridDev* dst, double radius, const IndexCells data,
                          const float* queries, int64_t m, int sample, float4* qrec) {
  pdl_trigger();
  pdl_wait();
  index_plan(src, dst, radius, data, queries, m, sample);
  const int64_t j = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (j >= m) return;
  qrec[j] = make_float4(queries[2 * j], queries[2 * j + 1], __int_as_float(static_cast<int>(j)),
                        0.f);
}

// Query side of a call on a prepared index: plan copy, then the counting
// sort of the queries alone (the scan runs its query half only), or their
// records as they come.
cudaError_t launch_query_sort(const GridDev* xgrid, const IndexCells& data, const float* queries,
                              int64_t m, double radius, int sample, int64_t max_cells,
                              void* workspace, const QueryLayout& Q, int sm_count, cudaStream_t s,
                              bool sort_queries) {
  unsigned char* ws = static_cast<unsigned char*>(workspace);
  GridDev* grid = reinterpret_cast<GridDev*>(ws + Q.off_grid);
  int32_t* counts = reinterpret_cast<int32_t*>(ws + Q.off_counts);
  int32_t* starts = reinterpret_cast<int32_t*>(ws + Q.off_starts);
  int32_t* sums = reinterpret_cast<int32_t*>(ws + Q.off_sums);
  float4* qrec = reinterpret_cast<float4*>(ws + Q.off_qrec);
  const int max_tiles = scan_tiles_of(max_cells);
  const unsigned qgrid = static_cast<unsigned>((m + 255) / 256);
  if (!sort_queries)
    return launch_pdl(index_identity_kernel, qgrid, kSampleQueries, 0, s, xgrid, grid, radius, data,
                      queries, m, sample, qrec);
  const unsigned zgrid = static_cast<unsigned>(
      std::min<int64_t>(int64_t(sm_count) * 4, (count_int4s(max_cells) + 255) / 256));
  cudaError_t e = launch_pdl(index_prep_kernel, zgrid, kSampleQueries, 0, s, xgrid, grid, radius,
                             data, queries, m, sample, counts);
  if (e == cudaSuccess)
    e = launch_pdl(count_kernel, qgrid, 256, 0, s, grid, nullptr, 0, queries, m, counts, counts);
  if (e == cudaSuccess)
    e = launch_pdl(scan_kernel, dim3(max_tiles, 1), kScanBlock, 0, s, grid, counts, counts, starts,
                   starts, sums, max_tiles, 1);
  if (e == cudaSuccess)
    e = launch_pdl(scatter_kernel, qgrid, 256, 0, s, grid, nullptr, 0, queries, m, 0, 0, starts,
                   starts, sums, max_tiles, counts, counts, nullptr, qrec);
  return e;
}

}  // namespace

IndexLayout index_layout(int64_t n, bool knn) {
  IndexLayout X;
  X.n = n;
  X.knn = knn;
  X.max_cells = local_max_cells(n);
  const size_t len = size_t(X.max_cells + 1 + 3) / 4 * 16;  // whole int4s
  size_t off = 0;
  X.off_grid = off;    off += round_up(sizeof(GridDev), 256);
  X.off_counts = off;  off += round_up(len, 256);
  X.off_starts = off;  off += round_up(len, 256);
  X.off_sums = off;    off += round_up(size_t(scan_tiles_of(X.max_cells)) * 4, 256);
  X.off_sorted = off;  off += round_up(size_t(n) * 16, 256);
  if (knn) {
    X.off_data = off;  off += round_up(size_t(n) * 12, 256);
    X.off_bpre = off;  off += round_up(size_t(kMaxBlocksPerAxis) * (kMaxBlocksPerAxis + 1) * 4, 256);
    X.off_sat = off;   off += round_up(size_t(X.max_cells + 2 * kMaxCellsPerAxis + 1) * 4, 256);
  }
  X.bytes = off;
  return X;
}

QueryLayout query_layout(int64_t m, int64_t max_cells) {
  QueryLayout Q;
  const size_t len = size_t(max_cells + 1 + 3) / 4 * 16;
  size_t off = 0;
  Q.off_grid = off;    off += round_up(sizeof(GridDev), 256);
  Q.off_counts = off;  off += round_up(len, 256);
  Q.off_starts = off;  off += round_up(len, 256);
  Q.off_sums = off;    off += round_up(size_t(2 * scan_tiles_of(max_cells)) * 4, 256);
  Q.off_qrec = off;    off += round_up(size_t(m) * 16, 256);
  Q.off_hard = off;    off += round_up(size_t(m) * 4, 256);
  Q.bytes = off;
  return Q;
}

cudaError_t launch_index_build(const float* data, int64_t n, double radius, int knn_k,
                               void* index_mem, const IndexLayout& X, int sm_count,
                               cudaStream_t s) {
  unsigned char* mem = static_cast<unsigned char*>(index_mem);
  GridDev* grid = reinterpret_cast<GridDev*>(mem + X.off_grid);
  int32_t* counts = reinterpret_cast<int32_t*>(mem + X.off_counts);
  int32_t* starts = reinterpret_cast<int32_t*>(mem + X.off_starts);
  int32_t* sums = reinterpret_cast<int32_t*>(mem + X.off_sums);
  float4* sorted = reinterpret_cast<float4*>(mem + X.off_sorted);
  const int max_tiles = scan_tiles_of(X.max_cells);
  cudaError_t e = cudaMemsetAsync(grid, 0xff, sizeof(GridDev), s);
  if (e != cudaSuccess) return e;
  const unsigned bgrid = static_cast<unsigned>(
      std::max<int64_t>(1, std::min<int64_t>(int64_t(sm_count) * 4, (n + 255) / 256)));
  e = launch_pdl(box_plan_kernel, bgrid, 256, 0, s, data, n, grid, radius,
                 1.0 / double(X.max_cells), knn_k, X.max_cells, counts, nullptr);
  if (e != cudaSuccess) return e;
  const unsigned dgrid = static_cast<unsigned>((n + 255) / 256);
  e = launch_pdl(count_kernel, dgrid, 256, 0, s, grid, data, n, nullptr, 0, counts, counts);
  if (e == cudaSuccess)
    e = launch_pdl(scan_kernel, dim3(max_tiles, 1), kScanBlock, 0, s, grid, counts, counts, starts,
                   starts, sums, max_tiles, 0);
  if (e == cudaSuccess)
    e = launch_pdl(scatter_kernel, dgrid, 256, 0, s, grid, data, n, nullptr, 0, 0, 0, starts, starts,
                   sums, max_tiles, counts, counts, sorted, nullptr);
  if (e != cudaSuccess) return e;
  if (X.knn) {
    e = cudaMemcpyAsync(mem + X.off_data, data, size_t(n) * 12, cudaMemcpyDeviceToDevice, s);
    if (e != cudaSuccess) return e;
    int32_t* bpre = reinterpret_cast<int32_t*>(mem + X.off_bpre);
    int32_t* sat = reinterpret_cast<int32_t*>(mem + X.off_sat);
    return launch_count_tables(grid, starts, sums, bpre, sat, s);
  }
  return cudaSuccess;
}

cudaError_t launch_index_local(const void* index_mem, const IndexLayout& X, const float* queries,
                               int64_t m, double p, double radius, float* out, int32_t* count_out,
                               void* workspace, const QueryLayout& Q, int sm_count,
                               cudaStream_t s, bool sort_queries, bool modified) {
  const unsigned char* mem = static_cast<const unsigned char*>(index_mem);
  const GridDev* xgrid = reinterpret_cast<const GridDev*>(mem + X.off_grid);
  const int32_t* starts = reinterpret_cast<const int32_t*>(mem + X.off_starts);
  const int32_t* sums = reinterpret_cast<const int32_t*>(mem + X.off_sums);
  cudaError_t e = launch_query_sort(xgrid, IndexCells{starts, sums, X.n}, queries, m, radius,
                                    m <= heavy_limit(sm_count) ? 0 : kSampleRadius, X.max_cells,
                                    workspace, Q, sm_count, s, sort_queries && m > kUnsortedRadius);
  if (e != cudaSuccess) return e;
  unsigned char* ws = static_cast<unsigned char*>(workspace);
  const GridDev* grid = reinterpret_cast<const GridDev*>(ws + Q.off_grid);
  const float4* qrec = reinterpret_cast<const float4*>(ws + Q.off_qrec);
  const float4* sorted = reinterpret_cast<const float4*>(mem + X.off_sorted);
  const float r2f = static_cast<float>(radius * radius);
  const float r2t = r2f > 0.f ? r2f : 0x1p-149f;
  const unsigned qgrid = static_cast<unsigned>((m + kLocalThreads - 1) / kLocalThreads);
  return launch_radius_queries(grid, sorted, X.n, starts, sums, qrec, m, p, r2f, r2t, out, count_out,
                               radius, modified, reinterpret_cast<int32_t*>(ws + Q.off_hard),
                               sort_queries && m <= kUnsortedRadius, qgrid,
                               sm_count, s);
}

cudaError_t launch_index_knn(const void* index_mem, const IndexLayout& X, const float* queries,
                             int64_t m, double p, int k, float* out, int32_t* nbr_out,
                             float* kd2_out, void* workspace, const QueryLayout& Q, int sm_count,
                             cudaStream_t s, bool sort_queries) {
  const unsigned char* mem = static_cast<const unsigned char*>(index_mem);
  const GridDev* xgrid = reinterpret_cast<const GridDev*>(mem + X.off_grid);
  const int32_t* starts = reinterpret_cast<const int32_t*>(mem + X.off_starts);
  const int32_t* sums = reinterpret_cast<const int32_t*>(mem + X.off_sums);
  cudaError_t e = launch_query_sort(xgrid, IndexCells{starts, sums, X.n}, queries, m, 0.0,
                                    knn_sampled(k, m) ? k : 0, X.max_cells, workspace, Q, sm_count, s,
                                    sort_queries && m > kUnsortedKnn);
  if (e != cudaSuccess) return e;
  unsigned char* ws = static_cast<unsigned char*>(workspace);
  const float4* qrec = reinterpret_cast<const float4*>(ws + Q.off_qrec);
  const float4* sorted = reinterpret_cast<const float4*>(mem + X.off_sorted);
  const float* data = reinterpret_cast<const float*>(mem + X.off_data);
  const int32_t* bpre = reinterpret_cast<const int32_t*>(mem + X.off_bpre);
  const int32_t* sat = reinterpret_cast<const int32_t*>(mem + X.off_sat);
  return launch_knn_search(
      KnnArgs{reinterpret_cast<GridDev*>(ws + Q.off_grid), sorted, starts, sums, bpre, sat, qrec, data,
              X.n, m, p, k, out, nbr_out, kd2_out, nullptr, true,
              reinterpret_cast<int32_t*>(ws + Q.off_hard)},
      sm_count, s);
}

}  // namespace idw
