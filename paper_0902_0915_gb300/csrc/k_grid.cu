// k_grid.cu -- gridding of correlator output onto polarisation uv grids.
//
// Paper Sec. 2.1: the calibrated visibilities are convolved onto a regular
// grid so that an FFT can form the images; Sec. 3.2: on the GPU every
// "scatter" step of the CPU code became a "gather" step, each thread
// collecting the values of its own output location (no floating-point
// atomics).  Definition (the paper names no kernel or sizes):
//   every tile baseline a > b and channel c (nu = f0 + c df) is a point at
//       x = (X_a - X_b) nu / c_light / du + Ng/2,  y = (Y_a - Y_b) nu / c_light / du + Ng/2
//   carrying its four polarisation products V_pq (input 2a+p with 2b+q), and
//   the reversed baseline is the point (Ng - x, Ng - y) carrying
//   conj(V_qp).  A point adds V w(s - x, r - y) to cell (r, s) of grid
//   2p+q for |s - x| < W/2 and |r - y| < W/2, w(dx, dy) =
//   exp(-(dx^2 + dy^2) / (2 sigma^2)); cells outside [0, Ng) are dropped.
//
//
// Half plane: the grids are Hermitian, G_pq(r, s) = conj(G_qp(Ng - r, Ng - s)),
// because every point has its reversed twin.  Only the cells of rows
// Ng/2 .. Ng and columns 0 .. Ng are summed (one row and column past the grid,
// whose mirror images are row 0 and column 0); each row above Ng/2 is stored
// twice, as it is and mirrored.  That halves the points, their weights and
// the multiply-adds.
//
// Plan (geometry only, once per array layout and band):
//   1. the W support rows of a point are cut into bands of at most 7 rows (one
//      band up to W = 7); a (point, band) whose cells reach the half plane is
//      an entry.  Positions and support bounds are FP64, so the support sets
//      match an FP64 definition exactly;
//   2. counting sort of the entries by bin = the band's first cell (integer
//      atomics for counts and slots, an exclusive prefix sum for bin offsets),
//      then every bin's entries sorted ascending so the order of each gathered
//      sum is fixed;
//   3. the weights: the Gaussian is separable, w = wx(s - x) wy(r - y), and the
//      support a rectangle, so an entry stores its W column and up to 7 row
//      factors (computed in FP64, kept in FP32, 0 outside the support) and its
//      first column: 64 bytes up to W = 7;
//   4. the units of work: a strip of 4 columns by 8, 16 or 32 rows is one warp's; strips that hold more entries than a quarter of a
//      warp's even share (the centre of the uv plane) take a CTA of 4 warps,
//      sparse ones are joined to strips of 32 columns by 8 rows.
// Grid call (per integration): one kernel gathers the four polarisation values
// of every baseline and channel from the int32 correlator output into its
// entries; then each warp walks its strip row of bins by row of bins.  The
// entries of a bin row reach the same WN rows (7 for W = 7): the lane keeps a
// window of WN rows of its column in registers that slides down by one, so
// no row outside the support is touched, and the row that the window leaves is
// complete and stored.  The warp's 8 groups of 4 lanes take every eighth entry;
// their sums are added in a fixed order.  No support tests and no exponentials
// per call; deterministic.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <utility>
#include <vector>

#include "mwax_internal.h"

namespace mwax {
namespace {

constexpr double kCLight = 299792458.0;
constexpr int kScanBlock = 1024;

__device__ __forceinline__ void tbl_pair(int tbl, int &a, int &b) {
  // tbl = a(a-1)/2 + b, a > b >= 0
  int i = (int)((sqrtf(8.0f * (float)tbl + 1.0f) + 1.0f) * 0.5f);
  while (i * (i - 1) / 2 > tbl) --i;
  while ((i + 1) * i / 2 <= tbl) ++i;
  a = i;
  b = tbl - i * (i - 1) / 2;
}

struct GridGeom {
  const double *tile_xy;
  int n_tiles, n_chan, n_tbl, Ng, W;
  double f0, df, du;
  int nbw;      // bins per row: columns -(W-1) .. Ng
  int nb, wr;   // bands per point, rows per band
  int off;      // window rows of the apply kernel (>= wr) - 1: bin row 0 is grid row Ng/2 - off
};

// A point's support: first and last column and row (unclipped), FP64 position.
struct Support {
  double x, y;
  int s_lo, s_hi, r_lo, r_hi;
};

// Point k = ((c * n_tbl) + tbl) * 2 + side.
__device__ __forceinline__ Support point_support(const GridGeom &g, int64_t k) {
  const int side = (int)(k & 1);
  const int64_t ct = k >> 1;
  const int c = (int)(ct / g.n_tbl), tbl = (int)(ct % g.n_tbl);
  int a, b;
  tbl_pair(tbl, a, b);
  const double nu = g.f0 + (double)c * g.df;
  Support p;
  p.x = (g.tile_xy[2 * a] - g.tile_xy[2 * b]) * nu / kCLight / g.du + 0.5 * g.Ng;
  p.y = (g.tile_xy[2 * a + 1] - g.tile_xy[2 * b + 1]) * nu / kCLight / g.du + 0.5 * g.Ng;
  if (side) {
    p.x = (double)g.Ng - p.x;
    p.y = (double)g.Ng - p.y;
  }
  const double half = 0.5 * g.W;
  // A point that is not within W cells of the grid, or not finite, reaches no cell:
  // an empty support, whose bounds need no conversion (which would leave an int).
  const double near = g.Ng + (double)g.W;
  if (!(p.x > -(double)g.W && p.x < near && p.y > -(double)g.W && p.y < near)) {
    p.s_lo = p.r_lo = 0;
    p.s_hi = p.r_hi = -1;
    return p;
  }
  // cells strictly within half the support: the smallest integer above x - W/2
  // and the largest below x + W/2
  p.s_lo = (int)floor(p.x - half) + 1;
  p.s_hi = (int)ceil(p.x + half) - 1;
  p.r_lo = (int)floor(p.y - half) + 1;
  p.r_hi = (int)ceil(p.y + half) - 1;
  return p;
}

// Bin of band b of a point, -1 if none of its cells lie in the half plane
// (rows Ng/2 .. Ng, columns 0 .. Ng).
__device__ __forceinline__ int band_bin(const GridGeom &g, const Support &p, int b) {
  if (p.s_hi < 0 || p.s_lo > g.Ng || p.r_hi < g.Ng / 2 || p.r_lo > g.Ng) return -1;
  const int r0 = p.r_lo + b * g.wr, r1 = min(r0 + g.wr - 1, p.r_hi);
  if (r1 < r0 || r1 < g.Ng / 2 || r0 > g.Ng) return -1;
  return (r0 - g.Ng / 2 + g.off) * g.nbw + (p.s_lo + g.W - 1);
}

// 1. entries per bin; n_reach: points with a cell in the grid itself
__global__ void __launch_bounds__(256) grid_count_kernel(GridGeom g, int64_t n_pts,
                                                         int *__restrict__ count,
                                                         int *__restrict__ n_reach) {
  const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  bool reach = false;
  if (k < n_pts) {
    const Support p = point_support(g, k);
    reach = p.s_hi >= 0 && p.s_lo <= g.Ng - 1 && p.r_hi >= 0 && p.r_lo <= g.Ng - 1;
    for (int b = 0; b < g.nb; ++b) {
      const int bin = band_bin(g, p, b);
      if (bin >= 0) atomicAdd(&count[bin], 1);
    }
  }
  const int n = __syncthreads_count(reach);
  if (threadIdx.x == 0 && n) atomicAdd(n_reach, n);
}

// exclusive prefix sum in three passes: per-block scan with block totals,
// scan of the totals (one block), add the block offsets
__global__ void __launch_bounds__(kScanBlock) scan_blocks_kernel(const int *__restrict__ in, int n,
                                                                 int *__restrict__ out,
                                                                 int *__restrict__ totals) {
  __shared__ int sh[kScanBlock];
  const int i = blockIdx.x * kScanBlock + threadIdx.x;
  const int v = i < n ? in[i] : 0;
  sh[threadIdx.x] = v;
  __syncthreads();
  for (int o = 1; o < kScanBlock; o <<= 1) {
    const int t = threadIdx.x >= o ? sh[threadIdx.x - o] : 0;
    __syncthreads();
    sh[threadIdx.x] += t;
    __syncthreads();
  }
  if (i < n) out[i] = sh[threadIdx.x] - v;  // exclusive
  if (threadIdx.x == kScanBlock - 1) totals[blockIdx.x] = sh[threadIdx.x];
}

__global__ void __launch_bounds__(kScanBlock) scan_totals_kernel(int *__restrict__ totals, int n) {
  // one block: exclusive scan of n block totals in chunks of kScanBlock
  __shared__ int sh[kScanBlock];
  __shared__ int carry;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (int base = 0; base < n; base += kScanBlock) {
    const int i = base + threadIdx.x;
    const int v = i < n ? totals[i] : 0;
    sh[threadIdx.x] = v;
    __syncthreads();
    for (int o = 1; o < kScanBlock; o <<= 1) {
      const int t = threadIdx.x >= o ? sh[threadIdx.x - o] : 0;
      __syncthreads();
      sh[threadIdx.x] += t;
      __syncthreads();
    }
    if (i < n) totals[i] = carry + sh[threadIdx.x] - v;
    __syncthreads();
    if (threadIdx.x == kScanBlock - 1) carry += sh[threadIdx.x];
    __syncthreads();
  }
}

// (the count array carries one extra zero entry, so the last exclusive offset
// is the total)
__global__ void scan_add_kernel(int *__restrict__ out, int n, const int *__restrict__ totals) {
  const int i = blockIdx.x * kScanBlock + threadIdx.x;
  if (i < n) out[i] += totals[blockIdx.x];
}

// 2. entry ids (k * nb + b) into their bins
__global__ void __launch_bounds__(256) grid_fill_kernel(GridGeom g, int64_t n_pts,
                                                        const int *__restrict__ offsets,
                                                        int *__restrict__ fill,
                                                        long long *__restrict__ ids) {
  const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (k >= n_pts) return;
  const Support p = point_support(g, k);
  for (int b = 0; b < g.nb; ++b) {
    const int bin = band_bin(g, p, b);
    if (bin >= 0) ids[offsets[bin] + atomicAdd(&fill[bin], 1)] = k * g.nb + b;
  }
}

// ids of every bin ascending (insertion sort; bins are short)
__global__ void grid_sort_bins_kernel(const int *__restrict__ offsets, int n_bins,
                                      long long *__restrict__ ids) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= n_bins) return;
  const int lo = offsets[b], hi = offsets[b + 1];
  for (int i = lo + 1; i < hi; ++i) {
    const long long v = ids[i];
    int j = i - 1;
    while (j >= lo && ids[j] > v) {
      ids[j + 1] = ids[j];
      --j;
    }
    ids[j + 1] = v;
  }
}

// 3. per entry: `fx` floats, [W column factors][first column s_lo, an int]
// padded to whole 16 bytes, then 8 row factors (0 past the band or outside the
// support); and the entry's place in the slot table [band][point].
constexpr int kRowFactors = 8;

__global__ void __launch_bounds__(256) grid_weights_kernel(GridGeom g,
                                                           const long long *__restrict__ ids,
                                                           int n_ent, double inv_2s2d, int fx,
                                                           int64_t n_pts, float *__restrict__ wts,
                                                           int *__restrict__ slot) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= n_ent) return;
  const long long id = ids[q];
  const int64_t k = id / g.nb;
  const int b = (int)(id - k * g.nb);
  slot[(int64_t)b * n_pts + k] = q;
  const Support p = point_support(g, k);
  float *w = wts + (int64_t)q * (fx + kRowFactors);
  for (int i = 0; i < fx; ++i) {
    float f = 0.f;
    if (i < g.W && p.s_lo + i <= p.s_hi) {
      const double d = (double)(p.s_lo + i) - p.x;
      f = (float)exp(-d * d * inv_2s2d);
    }
    w[i] = i == g.W ? __int_as_float(p.s_lo) : f;
  }
  const int r0 = p.r_lo + b * g.wr;
  for (int i = 0; i < kRowFactors; ++i) {
    float f = 0.f;
    if (i < g.wr && r0 + i <= p.r_hi) {
      const double d = (double)(r0 + i) - p.y;
      f = (float)exp(-d * d * inv_2s2d);
    }
    w[fx + i] = f;
  }
}

// Units of work: 4 columns (block cb) by `rows` rows from relative row r0 (row
// Ng/2 + r0 of the grid).  Bin row i of a unit, i = 0 .. rows + off - 1, is row
// r0 + i of the bin table and reaches the unit's rows i - off .. i; row i - off
// is complete after it.
constexpr int kCols = 4;
constexpr int kUnitRows = 32;  // at most (see unit_rows)
// Wide units: 32 columns, one entry a step, no sums across groups: a bin row costs
// its steps alone, while each of eight narrow strips pays about 100 instructions
// for it.  But the steps follow one another, so only strips of few entries a row are
// joined, and the longest are handed out first.  Measured a call, joined up to 12
// entries a row in any order / up to 3, longest first: 69 tiles x 21 channels on
// 1466^2 cells, W = 7: 55 / 38 us (narrow strips alone: 63); 17 x 328 on 1420^2,
// W = 6: 63 / 34; 100 x 200 on 2000^2, W = 5: 206 / 183; 128 x 768 on 2048^2,
// W = 7, of which little is sparse: 548 / 541.  In pieces of 8 rows instead of 16, the
// first 38 -> 35, 33 x 17 on 632^2 (units of 16 rows) 19.3 -> 19.5, 27 x 64 on
// 1076^2 22.5 -> 21.2.
constexpr int kWideCols = 32, kWideRows = 8, kWidePerRow = 3;
constexpr int kWideFlag = 1 << 30;
constexpr int kApplyWarps = 4, kApplyCtas = 4;  // of a CTA; CTAs per SM: 16 warps at up to 128 registers
constexpr int kMaxBinRows = 40;  // >= kUnitRows + 6

// Rows of a plan's units, from the half plane's rows, its column blocks, the entries
// and the SMs.  A unit of r rows walks r + 6 bin rows, so short units cost more work,
// and long ones leave a call with few units to wait for the longest.
// Measured a call, in us, units of 32 / 16 / 8 rows: 128 tiles x 64 channels on 2048^2
// cells, W = 7: 166 / 138 / 156; 92 x 24 on 932^2, W = 6: 47 / 34 / 36; 33 x 17 on
// 632^2, W = 7: 25 / 19 / 16; 24 x 357 on 294^2, W = 5: 49 / 31 / 24.  So 16 rows, with
// these exceptions (u units of 16 rows):
//   8 rows under three units a warp (16 / 8: 35 x 85 on 410^2 22.7 / 21.6, 100 x 24 on
//     800^2 39 / 35, 92 x 24 on 932^2, 2.9 a warp, 34 / 36);
//   32 rows where most strips are joined ones anyhow (8 entries a unit and many units:
//     69 x 21 on 1466^2 34.8, with 16 rows 38.9; 49 x 22 on 1994^2 41.0 and 44.2);
//   32 rows above 40 entries a unit (16 or 8 to give every warp half a unit), where more
//     of the strips are then heavy and summed in 32 parts: in 16 rows 128 x 768 on 2048^2
//     takes 533 instead of 538 us and 128 x 256 264 instead of 288, with errors against
//     64 bits 7 and 2 % larger.
int unit_rows(int n_rows, int n_cb, int64_t n_ent, int sms) {
  const auto units = [&](int r) { return (int64_t)((n_rows + r - 1) / r) * n_cb; };
  const int64_t u = units(16), warps = (int64_t)sms * kApplyCtas * kApplyWarps;
  if (2 * u < warps) return 8;
  if (n_ent > 40 * u) return 2 * units(32) < warps ? 16 : 32;
  if (u < 3 * warps) return 8;
  return u >= 4 * warps && n_ent <= 8 * u ? 32 : 16;
}

// entries of every unit of `rows` rows and `cols` columns (unit = row segment * n_cb +
// column block)
__global__ void __launch_bounds__(256) grid_unit_count_kernel(const int *__restrict__ offsets,
                                                              int n_units, int n_cb, int rows,
                                                              int n_rows, int cols, int W, int off,
                                                              int nbw, int *__restrict__ cnt) {
  const int u = blockIdx.x * blockDim.x + threadIdx.x;
  if (u >= n_units) return;
  const int r0 = (u / n_cb) * rows, s0 = (u % n_cb) * cols;
  const int nb = min(rows, n_rows - r0) + off;
  const int c1 = min(s0 + cols + W - 1, nbw);
  int n = 0;
  for (int i = 0; i < nb; ++i) n += offsets[(r0 + i) * nbw + c1] - offsets[(r0 + i) * nbw + s0];
  cnt[u] = n;
}

// Grid call, step 1: the four polarisation values of every baseline and
// channel, read in the correlator output's order, written as one 32-byte
// store into each entry of the point (a, b) and of its reversed twin (conj,
// XY and YX swapped).  HBM-bound: 32 B read, 8 B of slots and about 32 B
// written per baseline and channel (half the points are entries).
__device__ __forceinline__ void store8(float4 *dst, const float (&v)[8]) {
  asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst), "f"(v[0]),
               "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
               : "memory");
}

__global__ void __launch_bounds__(256) grid_values_kernel(const int2 *__restrict__ slot, int n_tbl,
                                                          int n_chan, int nb, int64_t n_bl,
                                                          const int2 *__restrict__ vis,
                                                          float4 *__restrict__ vals,
                                                          int *__restrict__ next) {
  let_dependents_start();
  if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *next = 0;  // step 2's unit counter
  const int tbl = blockIdx.x * blockDim.x + threadIdx.x;
  if (tbl >= n_tbl) return;
  int a, b;
  tbl_pair(tbl, a, b);
  const int64_t i0 = 2 * a, o0 = i0 * (i0 + 1) / 2 + 2 * b, o1 = o0 + i0 + 1;
  for (int c = blockIdx.y; c < n_chan; c += gridDim.y) {
    const int2 *vc = vis + (int64_t)c * n_bl;
    const int2 xx = __ldcs(vc + o0), xy = __ldcs(vc + o0 + 1), yx = __ldcs(vc + o1),
               yy = __ldcs(vc + o1 + 1);
    const int64_t ct = (int64_t)c * n_tbl + tbl, n_ct = (int64_t)n_chan * n_tbl;
    const float f[8] = {(float)xx.x, (float)xx.y, (float)xy.x, (float)xy.y,
                        (float)yx.x, (float)yx.y, (float)yy.x, (float)yy.y};
    const float r[8] = {f[0], -f[1], f[4], -f[5], f[2], -f[3], f[6], -f[7]};
    for (int band = 0; band < nb; ++band) {
      const int2 q = slot[band * n_ct + ct];
      if (q.x >= 0) store8(vals + 2 * (int64_t)q.x, f);
      if (q.y >= 0) store8(vals + 2 * (int64_t)q.y, r);
    }
  }
}

// Grid call, step 2.
// Staging: a ring of kSlots chunks of 32 entries per warp (values, factors).
// Every bin row starts on a multiple of G entries; the places left over are
// zeros.  One step is G entries, one per group of 32 / G lanes.
constexpr int kSlots = 2;
constexpr int kChunk = 32, kRing = kSlots * kChunk;
__host__ __device__ constexpr int apply_warp_bytes(int f4) {
  return kRing * (32 + 16 * f4) + (3 * kMaxBinRows + 4) * 4;
}

struct ApplyArgs {
  const int *offsets;
  const float4 *wts, *vals;
  float *grids;
  const int2 *units;  // x = column block (| kWideFlag), y = first relative row << 8 | rows
  int *next;          // light units handed out so far
  int Ng, W, nbw, f4;  // f4: 16-byte pieces per entry's factors
  int n_heavy, n_light;
};

// A unit's bin rows: first entry, entries, and steps before the row.
struct BinRows {
  int q[kMaxBinRows], n[kMaxBinRows], s[kMaxBinRows + 4];
};

// Where a lane's values of a unit's rows go, row by row: their cells, and mirrored
// (conj, p and q swapped) ones unless the row is its own mirror image.  comp = 2
// (2p + q) + (re, im).
struct RowOut {
  float *cell, *mirror;  // of the next row, component comp
  int r, half, step;     // its relative row; Ng / 2; floats per grid row
  bool in, min;          // the column has a cell, a mirrored cell

  __device__ __forceinline__ RowOut(const ApplyArgs &A, int r0, int s, int comp) {
    const int Ng = A.Ng, pol = comp >> 1, ri = comp & 1, mp = ((pol & 1) << 1) | (pol >> 1);
    r = r0;
    half = Ng / 2;
    step = 2 * Ng;
    in = s < Ng;
    min = s >= 1 && s <= Ng;
    cell = A.grids + (((int64_t)pol * Ng + half + r0) * Ng + s) * 2 + ri;
    mirror = A.grids + (((int64_t)mp * Ng + half - r0) * Ng + (Ng - s)) * 2 + ri;
  }
  __device__ __forceinline__ void advance() {
    cell += step;
    mirror -= step;
    ++r;
  }
  // narrow units: one component (ri: it is an imaginary part)
  __device__ __forceinline__ void put(float v, bool ri) {
    if (in && r < half) *cell = v;
    if (min && r > 0) *mirror = ri ? -v : v;
    advance();
  }
  // wide units (comp = 0): all four products
  __device__ __forceinline__ void put(const float (&a)[8]) {
    const int64_t plane = (int64_t)step * (step / 2);  // floats of a product's grid
#pragma unroll
    for (int pol = 0; pol < 4; ++pol) {
      const int mp = ((pol & 1) << 1) | (pol >> 1);
      if (in && r < half) *reinterpret_cast<float2 *>(cell + pol * plane) = make_float2(a[2 * pol], a[2 * pol + 1]);
      if (min && r > 0) *reinterpret_cast<float2 *>(mirror + mp * plane) = make_float2(a[2 * pol], -a[2 * pol + 1]);
    }
    advance();
  }
};

__device__ __forceinline__ float4 lds4(uint32_t a) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a));
  return v;
}
__device__ __forceinline__ int lds1(uint32_t a) {
  int v;
  asm volatile("ld.shared.s32 %0, [%1];" : "=r"(v) : "r"(a));
  return v;
}

__device__ __forceinline__ void cp16z(uint32_t dst, const void *src, bool take) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(take ? 16 : 0)
               : "memory");
}

// One warp's walk over a unit of n_bins bin rows.  emit(i, a): after bin row i
// the lane holds finished values of row i - off; G = 8 (narrow): column lane & 3,
// component lane >> 2 = 2 (2p + q) + (re, im) in a[0]; G = 1 (wide): column lane,
// all eight components.
template <int WN, int F4, int G, class Emit>
__device__ __forceinline__ void strip_walk(const ApplyArgs &A, int s0, int n_bins, uint8_t *sm,
                                           const BinRows &rows, int lane, Emit &&emit) {
  const int f4 = F4 ? F4 : A.f4;
  const int fb = 16 * f4;  // bytes of factors per entry
  const uint32_t uv = (uint32_t)__cvta_generic_to_shared(sm), uw = uv + kRing * 32;
  const int total = rows.s[n_bins];  // steps
  constexpr int kStepsPerChunk = kChunk / G;
  const int col = s0 + lane % (32 / G), g = lane / (32 / G);
  // chunk: lane j finds the entry of place j, then consecutive lanes copy
  // consecutive 16-byte pieces
  int my_row = 0;
  auto issue = [&](int chunk) {
    const int step = chunk * kStepsPerChunk + lane / G;
    if (chunk * kStepsPerChunk < total) {
      int q = -1;
      if (step < total) {
        while (rows.s[my_row + 1] <= step) ++my_row;
        const int k = (step - rows.s[my_row]) * G + lane % G;
        if (k < rows.n[my_row]) q = rows.q[my_row] + k;
      }
      const int slot = chunk % kSlots;
#pragma unroll
      for (int m = 0; m < 2; ++m) {
        const int p = m * 32 + lane;
        const int src = __shfl_sync(0xffffffffu, q, p >> 1);
        cp16z(uv + (slot * 64 + p) * 16, A.vals + 2 * (int64_t)max(src, 0) + (p & 1), src >= 0);
      }
#pragma unroll
      for (int m = 0; m < f4; ++m) {
        const int p = m * 32 + lane;
        const int e = p / f4, o = p - e * f4;
        const int src = __shfl_sync(0xffffffffu, q, e);
        cp16z(uw + (slot * kChunk * f4 + p) * 16, A.wts + (int64_t)max(src, 0) * f4 + o, src >= 0);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  constexpr int P = 2;  // bin rows between shifts of the window
  float acc[WN + P - 1][8];
#pragma unroll
  for (int t = 0; t < WN + P - 1; ++t)
#pragma unroll
    for (int p = 0; p < 8; ++p) acc[t][p] = 0.f;
#pragma unroll
  for (int k = 0; k < kSlots - 1; ++k) issue(k);
  int st = 0;
  uint32_t pv = 0, pw = 0;  // this group's entry of the step: values, factors
#pragma unroll 1
  for (int ib = 0; ib < n_bins; ib += P) {
#pragma unroll
    for (int ph = 0; ph < P; ++ph) {
      const int i = ib + ph;
      if (i < n_bins) {
#pragma unroll 1
        for (const int end = rows.s[i + 1]; st < end; ++st) {
          if (st % kStepsPerChunk == 0) {  // a new chunk: the slot of the one before it is free
            __syncwarp();
            issue(st / kStepsPerChunk + kSlots - 1);
            asm volatile("cp.async.wait_group %0;" ::"n"(kSlots - 1) : "memory");
            __syncwarp();
            const int slot = st / kStepsPerChunk % kSlots;
            pv = uv + (slot * kChunk + g) * 32;
            pw = uw + (slot * kChunk + g) * fb;
          }
          const int d = col - lds1(pw + 4 * A.W);
          const float4 v0 = lds4(pv), v1 = lds4(pv + 16), y0 = lds4(pw + fb - 32);
          float wy[WN > 5 ? 8 : 5] = {y0.x, y0.y, y0.z, y0.w};
          if constexpr (WN > 5) {
            const float4 y1 = lds4(pw + fb - 16);
            wy[4] = y1.x;
            wy[5] = y1.y;
            wy[6] = y1.z;
            wy[7] = y1.w;
          } else {
            wy[4] = __int_as_float(lds1(pw + fb - 16));
          }
          float wx = 0.f;
          if ((unsigned)d < (unsigned)A.W) wx = __int_as_float(lds1(pw + 4 * d));
          pv += G * 32;
          pw += G * fb;
          const float t8[8] = {wx * v0.x, wx * v0.y, wx * v0.z, wx * v0.w,
                               wx * v1.x, wx * v1.y, wx * v1.z, wx * v1.w};
#pragma unroll
          for (int t = 0; t < WN; ++t)
#pragma unroll
            for (int p = 0; p < 8; ++p) acc[ph + t][p] = fmaf(wy[t], t8[p], acc[ph + t][p]);
        }
        // the row that the window leaves: its eight components, with eight groups
        // summed over them (a butterfly over lane bits 4, 3, 2 that halves the
        // components each lane carries: group g ends with component g)
        float a[8];
#pragma unroll
        for (int p = 0; p < 8; ++p) a[p] = acc[ph][p];
        if (i >= WN - 1) {
          static_assert(G == 8 || G == 1, "the butterfly is over eight groups");
#pragma unroll
          for (int h = G / 2; h > 0; h >>= 1) {
            const bool up = lane & (4 * h);
#pragma unroll
            for (int k = 0; k < h; ++k) {
              const float send = up ? a[k] : a[k + h], keep = up ? a[k + h] : a[k];
              a[k] = keep + __shfl_xor_sync(0xffffffffu, send, 4 * h);
            }
          }
          emit(i, a);
        }
      }
    }
#pragma unroll
    for (int t = 0; t < WN + P - 1; ++t)
#pragma unroll
      for (int p = 0; p < 8; ++p) acc[t][p] = t + P < WN + P - 1 ? acc[t + P][p] : 0.f;
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
}

constexpr int apply_smem_bytes(int f4) {
  return kApplyWarps * apply_warp_bytes(f4) + kApplyWarps * kUnitRows * 32 * 4;
}

// Bound by instruction issue (70 % of the slots, 59 % of the instructions on the
// FMA pipe): 56 multiply-adds, 8 multiplies and about 20 other instructions per
// step of 8 entries, of whose 4 x 7 cells the strip's edge leaves 70 % useful.
// Measured for 12.5 M points on 4 x 2048^2 cells, W = 7: 0.54 ms a call, 0.076 of
// it the values; gathering both halves patch by patch with the factors of
// every (patch, point) pair stored took 1.42 ms.  Not taken: packed two-wide
// multiply-adds (67 per SM and cycle against 110 for scalar ones, measured),
// two columns per lane, bins of two rows, seven window phases unrolled instead
// of shifting registers (fetch stalls), more warps with spills.
// Persistent CTAs.  Heavy units (units[0 .. n_heavy)): one CTA per unit, warp w
// takes the w-th quarter of every bin row and the four
// partial sums are added in warp order.  Then every warp takes the next light
// unit until none is left (which warp takes it does not touch its sums).
template <int WN, int F4>
__global__ void __launch_bounds__(32 * kApplyWarps, kApplyCtas) grid_apply_kernel(ApplyArgs A) {
  extern __shared__ __align__(16) uint8_t sm_all[];
  constexpr int off = WN - 1;
  const int f4 = F4 ? F4 : A.f4;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint8_t *sm = sm_all + warp * apply_warp_bytes(f4);
  BinRows &rows = *reinterpret_cast<BinRows *>(sm + kRing * (32 + 16 * f4));
  float *part = reinterpret_cast<float *>(sm_all + kApplyWarps * apply_warp_bytes(f4));
  const int comp = lane >> 2;
  int h = blockIdx.x;
  wait_for_predecessor();
  while (true) {
    const bool heavy = h < A.n_heavy;
    int u = h;
    if (!heavy) {
      if (lane == 0) u = atomicAdd(A.next, 1);
      u = __shfl_sync(0xffffffffu, u, 0);
      if (u >= A.n_light) break;
      u += A.n_heavy;
    }
    const int2 unit = __ldg(A.units + u);
    const bool wide = unit.x & kWideFlag;
    const int s0 = (unit.x & ~kWideFlag) * kCols, r0 = unit.y >> 8, n_rows = unit.y & 255;
    const int c1 = min(s0 + (wide ? kWideCols : kCols) + A.W - 1, A.nbw);
    const int n_bins = n_rows + off;
    int steps = 0;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int i = 32 * k + lane;
      int lo = 0, n = 0;
      if (i < n_bins) {
        const int *o = A.offsets + (int64_t)(r0 + i) * A.nbw;
        lo = __ldg(o + s0);
        n = __ldg(o + c1) - lo;
        if (heavy) {
          const int first = (int)((int64_t)n * warp / kApplyWarps);
          n = (int)((int64_t)n * (warp + 1) / kApplyWarps) - first;
          lo += first;
        }
      }
      int x = wide ? n : (n + 7) >> 3;  // steps, then their running sum
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, x, d);
        if (lane >= d) x += t;
      }
      if (i < n_bins) {
        rows.q[i] = lo;
        rows.n[i] = n;
        rows.s[i + 1] = steps + x;
      }
      steps += __shfl_sync(0xffffffffu, x, 31);
    }
    if (lane == 0) rows.s[0] = 0;
    __syncwarp();
    const int s = s0 + (wide ? lane : lane & 3);
    RowOut out(A, r0, s, wide ? 0 : comp);
    if (steps == 0 && !heavy) {
      const float zero[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
      for (int r = 0; r < n_rows; ++r) {
        if (wide)
          out.put(zero);
        else
          out.put(0.f, false);
      }
    } else if (wide) {
      strip_walk<WN, F4, 1>(A, s0, n_bins, sm, rows, lane, [&](int, const float (&a)[8]) { out.put(a); });
    } else {
      strip_walk<WN, F4, 8>(A, s0, n_bins, sm, rows, lane, [&](int i, const float (&a)[8]) {
        if (heavy)
          part[(warp * kUnitRows + i - off) * 32 + lane] = a[0];
        else
          out.put(a[0], comp & 1);
      });
    }
    if (heavy) {
      __syncthreads();
      for (int r = warp; r < n_rows; r += kApplyWarps) {
        float v = part[r * 32 + lane];
#pragma unroll
        for (int w = 1; w < kApplyWarps; ++w) {
          v += part[(w * kUnitRows + r) * 32 + lane];
        }
        RowOut(A, r0 + r, s, comp).put(v, comp & 1);
      }
      __syncthreads();
      h += gridDim.x;
    }
    __syncwarp();  // the bin rows are written again
  }
}

constexpr int kMaxF4 = (32 + kRowFactors) / 4;  // W = 31

// Windows of 5 and 7 rows; the factors of an entry take 64 bytes (F4 = 4) for
// W = 4 .. 7.  PREPARE: set the kernel's shared-memory limit (at plan time)
// instead of launching it.
template <int WN, int F4, bool PREPARE>
cudaError_t apply_one(const ApplyArgs &A, int sms, cudaStream_t s) {
  if (PREPARE)
    return cudaFuncSetAttribute(grid_apply_kernel<WN, F4>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                apply_smem_bytes(F4 ? F4 : kMaxF4));
  const int ctas = std::min(kApplyCtas * sms, A.n_heavy + (A.n_light + kApplyWarps - 1) / kApplyWarps);
  // beside the values kernel, whose CTAs would set how this kernel's lie on the SMs: no
  // matter for the light units, which are handed out, but a heavy unit's CTA is fixed,
  // and neighbouring ones are alike (95 tiles x 562 channels on 388^2 cells: 348 us, as a
  // dependent 437; 33 x 17 on 632^2, no heavy units: 17 as an ordinary launch, 15 so)
  if (A.n_heavy <= sms)
    return launch_dependent(grid_apply_kernel<WN, F4>, ctas, 32 * kApplyWarps, apply_smem_bytes(A.f4), s, A);
  grid_apply_kernel<WN, F4><<<ctas, 32 * kApplyWarps, apply_smem_bytes(A.f4), s>>>(A);
  return cudaGetLastError();
}

template <bool PREPARE>
cudaError_t apply_units(int win, const ApplyArgs &A, int sms, cudaStream_t s) {
  if (win == 5)
    return A.f4 == 4 ? apply_one<5, 4, PREPARE>(A, sms, s) : apply_one<5, 0, PREPARE>(A, sms, s);
  return A.f4 == 4 ? apply_one<7, 4, PREPARE>(A, sms, s) : apply_one<7, 0, PREPARE>(A, sms, s);
}

}  // namespace
}  // namespace mwax

using namespace mwax;

struct mwax_grid_plan_s {
  cudaStream_t stream = nullptr;
  int device = 0;
  int n_tiles = 0, n_chan = 0, n_tbl = 0, Ng = 0, W = 0, nbw = 0, nb = 1, win = 7, f4 = 4;
  int64_t n_pts = 0;
  int n_kept = 0;            // points with a cell in the grid
  int n_ent = 0;             // entries: (point, band) with a cell in the half plane
  int n_heavy = 0, n_light = 0, sms = 0;
  int *offsets = nullptr;    // [n_bins + 1]
  int *slot = nullptr;       // [nb][n_pts]: place of each entry, or -1
  int2 *units = nullptr;     // heavy units, then light ones
  int *next = nullptr;       // counter of the light units handed out in a call
  float *wts = nullptr;      // [n_ent][4 f4]
  float4 *vals = nullptr;    // [n_ent][2], filled per call
};

namespace {

void free_grid_plan(mwax_grid_plan_s *p) {
  if (!p) return;
  for (void *q : {(void *)p->offsets, (void *)p->slot, (void *)p->units, (void *)p->next, (void *)p->wts, (void *)p->vals})
    if (q) cudaFree(q);
  delete p;
}

ApplyArgs apply_args(const mwax_grid_plan_s *p, float *grids) {
  return ApplyArgs{p->offsets, reinterpret_cast<const float4 *>(p->wts), p->vals, grids,
                   p->units,   p->next,                                     p->Ng,   p->W,
                   p->nbw,     p->f4,                                       p->n_heavy, p->n_light};
}

bool is_dev(const void *p) {
  if (!p) return false;
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

}  // namespace

extern "C" {

mwax_status mwax_grid_plan(mwax_grid_plan_t *out, const double *tile_xy, int n_tiles, int n_chan,
                           double f0, double df, int Ng, double du, int W, double sigma,
                           cudaStream_t stream) {
  mwax::NvtxRange nvtx_("mwax_grid_plan");
  if (!out || !tile_xy) return MWAX_ERR_INVALID_ARG;
  *out = nullptr;
  if (n_tiles < 2 || n_tiles > 4096 || n_chan < 1 || Ng < 8 || Ng > 16384 || Ng % 2 || W < 1 ||
      W > 31 || !(du > 0.0) || !(sigma > 0.0) || !(f0 > 0.0) || df < 0.0)
    return MWAX_ERR_INVALID_ARG;
  const int64_t n_tbl = (int64_t)n_tiles * (n_tiles - 1) / 2;
  const int64_t n_pts = n_tbl * n_chan * 2;
  if (n_pts > 0x7FFFFFFFll) return MWAX_ERR_INVALID_ARG;
  mwax_grid_plan_s *p = new mwax_grid_plan_s;
  p->stream = stream;
  cudaGetDevice(&p->device);
  p->n_tiles = n_tiles;
  p->n_chan = n_chan;
  p->n_tbl = (int)n_tbl;
  p->Ng = Ng;
  p->W = W;
  p->n_pts = n_pts;
  p->nb = (W + 6) / 7;
  const int wr = (W + p->nb - 1) / p->nb;
  p->win = wr <= 5 ? 5 : 7;
  const int off = p->win - 1;
  p->nbw = Ng + W;
  const int n_rows = Ng / 2 + 1;                     // rows of the half plane
  const int n_bins = (n_rows + off) * p->nbw;  // at most 8199 x 16415
  const int fx = (W + 1 + 3) / 4 * 4;
  p->f4 = (fx + kRowFactors) / 4;
  // plan-time scratch
  double *d_xy = nullptr;
  int *count = nullptr, *totals = nullptr, *ucnt = nullptr, *reach = nullptr;
  long long *ids = nullptr;
  auto free_scratch = [&] {
    for (void *q : {(void *)d_xy, (void *)count, (void *)totals, (void *)ucnt, (void *)reach, (void *)ids})
      if (q) cudaFree(q);
  };
  const int n_scan = n_bins + 1;  // one extra zero: the last offset is the total
  const int scan_blocks = (n_scan + kScanBlock - 1) / kScanBlock;
  cudaError_t e = cudaMalloc(&d_xy, sizeof(double) * 2 * n_tiles);
  if (e == cudaSuccess) e = cudaMalloc(&count, sizeof(int) * n_scan);
  if (e == cudaSuccess) e = cudaMalloc(&totals, sizeof(int) * scan_blocks);
  if (e == cudaSuccess) e = cudaMalloc(&reach, sizeof(int));
  if (e == cudaSuccess) e = cudaMalloc(&p->offsets, sizeof(int) * n_scan);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(d_xy, tile_xy, sizeof(double) * 2 * n_tiles, cudaMemcpyHostToDevice, stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(count, 0, sizeof(int) * n_scan, stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(reach, 0, sizeof(int), stream);
  GridGeom g{d_xy, n_tiles, n_chan, (int)n_tbl, Ng, W, f0, df, du, p->nbw, p->nb, wr, off};
  const int T = 256;
  const unsigned nblk = (unsigned)((n_pts + T - 1) / T);
  if (e == cudaSuccess) {
    grid_count_kernel<<<nblk, T, 0, stream>>>(g, n_pts, count, reach);
    scan_blocks_kernel<<<scan_blocks, kScanBlock, 0, stream>>>(count, n_scan, p->offsets, totals);
    scan_totals_kernel<<<1, kScanBlock, 0, stream>>>(totals, scan_blocks);
    scan_add_kernel<<<scan_blocks, kScanBlock, 0, stream>>>(p->offsets, n_scan, totals);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(&p->n_kept, reach, sizeof(int), cudaMemcpyDeviceToHost, stream);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(&p->n_ent, p->offsets + n_bins, sizeof(int), cudaMemcpyDeviceToHost, stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
  // the limit on points times support, in units of 4 x 8 cells
  const int64_t per_point = (int64_t)((W + 3) / 4 + 1) * ((W + 7) / 8 + 1);
  if (e == cudaSuccess && (int64_t)p->n_kept * per_point > 0x7FFFFFFFll) {
    free_scratch();
    free_grid_plan(p);
    return MWAX_ERR_UNSUPPORTED;
  }
  const int n_ent = p->n_ent;
  if (e == cudaSuccess) e = cudaMalloc(&ids, sizeof(long long) * std::max(n_ent, 1));
  if (e == cudaSuccess) e = cudaMalloc(&p->vals, 2 * sizeof(float4) * std::max(n_ent, 1));
  if (e == cudaSuccess) e = cudaMalloc(&p->wts, (size_t)16 * p->f4 * std::max(n_ent, 1));
  if (e == cudaSuccess) e = cudaMalloc(&p->slot, sizeof(int) * n_pts * p->nb);
  if (e == cudaSuccess) e = cudaMemsetAsync(p->slot, 0xFF, sizeof(int) * n_pts * p->nb, stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(count, 0, sizeof(int) * n_scan, stream);
  if (e == cudaSuccess) {
    grid_fill_kernel<<<nblk, T, 0, stream>>>(g, n_pts, p->offsets, count, ids);
    grid_sort_bins_kernel<<<(unsigned)((n_bins + T - 1) / T), T, 0, stream>>>(p->offsets, n_bins, ids);
    if (n_ent > 0)
      grid_weights_kernel<<<(unsigned)((n_ent + T - 1) / T), T, 0, stream>>>(
          g, ids, n_ent, 1.0 / (2.0 * sigma * sigma), fx, n_pts, p->wts, p->slot);
    e = cudaGetLastError();
  }
  const int n_cb = Ng / kCols + 1;  // the last block holds column Ng alone
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&p->sms, cudaDevAttrMultiProcessorCount, p->device);
  const int rows = unit_rows(n_rows, n_cb, n_ent, p->sms);
  const int n_seg = (n_rows + rows - 1) / rows, per_wide = kWideCols / kCols, n_wcb = (n_cb + per_wide - 1) / per_wide;
  const int n_u = n_seg * n_cb, n_wu = n_seg * n_wcb;
  std::vector<int> cnt(n_u + n_wu);
  if (e == cudaSuccess) e = cudaMalloc(&ucnt, sizeof(int) * (n_u + n_wu));
  if (e == cudaSuccess) {
    grid_unit_count_kernel<<<(n_u + T - 1) / T, T, 0, stream>>>(p->offsets, n_u, n_cb, rows, n_rows, kCols, W, off,
                                                               p->nbw, ucnt);
    grid_unit_count_kernel<<<(n_wu + T - 1) / T, T, 0, stream>>>(p->offsets, n_wu, n_wcb, rows, n_rows, kWideCols, W,
                                                                off, p->nbw, ucnt + n_u);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(cnt.data(), ucnt, sizeof(int) * cnt.size(), cudaMemcpyDeviceToHost, stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
  std::vector<int2> heavy, units;
  std::vector<std::pair<int, int2>> wide;  // (entries, unit)
  if (e == cudaSuccess) {
    int64_t total = 0;
    for (int u = 0; u < n_u; ++u) total += cnt[u];
    const int64_t most = std::max<int64_t>(256, total / ((int64_t)p->sms * kApplyCtas * kApplyWarps * 4));
    for (int seg = 0; seg < n_seg; ++seg) {
      const int r0 = seg * rows, nr = std::min(rows, n_rows - r0);
      for (int wb = 0; wb < n_wcb; ++wb) {
        const int n_wide = cnt[n_u + seg * n_wcb + wb];
        if (n_wide <= kWidePerRow * rows) {
          for (int r = 0; r < nr; r += kWideRows)
            wide.push_back({n_wide, make_int2(wb * per_wide | kWideFlag, (r0 + r) << 8 | std::min(kWideRows, nr - r))});
          continue;
        }
        for (int cb = wb * per_wide; cb < std::min(n_cb, (wb + 1) * per_wide); ++cb)
          (cnt[seg * n_cb + cb] > most ? heavy : units).push_back(make_int2(cb, r0 << 8 | nr));
      }
    }
    // the wide ones last, the shortest at the end
    std::stable_sort(wide.begin(), wide.end(), [](const auto &a, const auto &b) { return a.first > b.first; });
    for (const auto &w : wide) units.push_back(w.second);
    p->n_heavy = (int)heavy.size();
    p->n_light = (int)units.size();
    heavy.insert(heavy.end(), units.begin(), units.end());
    e = cudaMalloc(&p->units, sizeof(int2) * heavy.size());
  }
  if (e == cudaSuccess)
    e = cudaMemcpy(p->units, heavy.data(), sizeof(int2) * heavy.size(), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMalloc(&p->next, sizeof(int));
  if (e == cudaSuccess) e = apply_units<true>(p->win, apply_args(p, nullptr), p->sms, stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
  free_scratch();
  if (e != cudaSuccess) {
    free_grid_plan(p);
    return e == cudaErrorMemoryAllocation ? MWAX_ERR_OOM : MWAX_ERR_CUDA;
  }
  *out = p;
  return MWAX_OK;
}

int64_t mwax_grid_plan_points(mwax_grid_plan_t plan) { return plan ? plan->n_kept : -1; }

int64_t mwax_grid_plan_entries(mwax_grid_plan_t plan) {
  return plan ? (int64_t)plan->n_ent * 4 * plan->f4 : -1;
}

mwax_status mwax_grid(mwax_grid_plan_t plan, const int32_t *vis, float *grids) {
  mwax::NvtxRange nvtx_("mwax_grid");
  if (!plan || !is_dev(vis) || !is_dev(grids)) return MWAX_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(vis) & 7u) || (reinterpret_cast<uintptr_t>(grids) & 7u))
    return MWAX_ERR_INVALID_ARG;
  const int64_t N = 2 * (int64_t)plan->n_tiles;
  const int T = 256;
  grid_values_kernel<<<dim3((unsigned)((plan->n_tbl + T - 1) / T), (unsigned)std::min(plan->n_chan, 65535)), T, 0,
                       plan->stream>>>(reinterpret_cast<const int2 *>(plan->slot), plan->n_tbl, plan->n_chan,
                                       plan->nb, N * (N + 1) / 2, reinterpret_cast<const int2 *>(vis), plan->vals,
                                       plan->next);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = apply_units<false>(plan->win, apply_args(plan, grids), plan->sms, plan->stream);
  return e == cudaSuccess ? MWAX_OK : MWAX_ERR_CUDA;
}

mwax_status mwax_grid_destroy(mwax_grid_plan_t plan) {
  if (!plan) return MWAX_ERR_INVALID_ARG;
  cudaStreamSynchronize(plan->stream);
  free_grid_plan(plan);
  return MWAX_OK;
}

}  // extern "C"
