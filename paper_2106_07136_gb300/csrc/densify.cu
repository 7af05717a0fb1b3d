// densify.cu -- fusion of the patch disparities into a dense map (Sec. 2.3).
//
// Each pixel takes its covering patches straight from the regular grid (no
// scatter, no atomics): w = weight_k * m(x - x0_k) * m(y - y0_k), where the
// Gaussian mask m (Eq. 5, sigma_s) is separable and depends only on the
// position inside the patch. The pixel's disparity is sum w D*_k / sum w (the
// normalised form of Eq. 2 with the combined posterior as weight). Pixels
// without a kept patch are NaN at the finest level (Sec. 3.2: not
// estimated); coarser levels carry the value their patches started from.
//
// Because the mask is separable, a block computes a 32x32 tile in two passes
// through shared memory: first, for every patch row that touches the tile
// and every tile column, the x-weighted sums over the covering patches of
// that row (sum m_x (w D) and sum m_x w, w D formed once per patch); then,
// per pixel, the y-weighted sum of those over its covering rows. Work per pixel drops from (ps/stride)^2 to
// about 2 ps/stride multiply-adds per quantity.
//
// Roofline: DRAM bytes per pixel: 4 written (+4 read for the coarse map where
// carried) plus the patch arrays (8 B per patch) read once per tile.
#include "bdis_internal.cuh"

#include <algorithm>

namespace bdis {
namespace {

__device__ __forceinline__ float bilinear_clamped(const float *M, int w, int h, float x,
                                                  float y) {
  x = fminf(fmaxf(x, 0.f), (float)(w - 1));
  y = fminf(fmaxf(y, 0.f), (float)(h - 1));
  const int x0 = (int)floorf(x), y0 = (int)floorf(y);
  const int x1 = min(x0 + 1, w - 1), y1 = min(y0 + 1, h - 1);
  const float tx = x - x0, ty = y - y0;
  const float top = (1.f - tx) * __ldg(M + (size_t)y0 * w + x0) + tx * __ldg(M + (size_t)y0 * w + x1);
  const float bot = (1.f - tx) * __ldg(M + (size_t)y1 * w + x0) + tx * __ldg(M + (size_t)y1 * w + x1);
  return (1.f - ty) * top + ty * bot;
}

// Patches covering coordinate x along one axis: the regular ones
// [lo, hi] (indices <= n - 2) plus the last one (origin n_px - ps) if it covers.
__device__ __forceinline__ void cover_range(int x, int n_px, int ps, int stride, int n, int &lo,
                                            int &hi, int &last) {
  const int a = x - ps + 1;
  lo = a <= 0 ? 0 : (a + stride - 1) / stride;
  hi = min(x / stride, n - 2);
  last = (x >= n_px - ps) ? 1 : 0;
}

constexpr int kTileX = 32, kTileY = 32, kMaxRows = kTileY + kMaxPatch;

__global__ void __launch_bounds__(256) densify_kernel(const DensifyArgs a) {
  __shared__ float mask[kMaxPatch];
  __shared__ float sA[kMaxRows][kTileX], sB[kMaxRows][kTileX];
  const int tid = threadIdx.x;
  pdl_enter();
  if (tid < a.ps) {
    const float m = (float)tid - (a.ps - 1) * 0.5f;
    mask[tid] = expf(-(m * m) / a.two_s2);
  }
  const int b = blockIdx.z;
  const int tile_y = a.tile_y > 0 ? a.tile_y : kTileY;  // 8, 16 or 32
  const int X0 = blockIdx.x * kTileX, Y0 = blockIdx.y * tile_y;
  const int ylast = min(Y0 + tile_y, a.h) - 1;
  // patch rows touching the tile: regular rows [jlo, jhi] and maybe the last
  int jlo, jhi, jl_unused, hlast_lo, hlast_hi;
  cover_range(Y0, a.h, a.ps, a.stride, a.ny, jlo, jl_unused, hlast_lo);
  cover_range(ylast, a.h, a.ps, a.stride, a.ny, jl_unused, jhi, hlast_hi);
  const int nreg = max(0, jhi - jlo + 1);
  const int has_last = hlast_hi;  // the last row covers the bottom of the tile if any
  const int nrows = nreg + has_last;
  const float *wp = a.weight + (long long)b * a.np;
  const float *dp = a.d_star + (long long)b * a.np;
  __syncthreads();

  // pass 1: x-weighted sums per (patch row, tile column)
  for (int q = tid; q < nrows * kTileX; q += blockDim.x) {
    const int jj = q / kTileX, xx = q - jj * kTileX;
    const int x = X0 + xx;
    float A = 0.f, B = 0.f;
    if (x < a.w) {
      const int j = jj < nreg ? jlo + jj : a.ny - 1;
      int ilo, ihi, ilast;
      cover_range(x, a.w, a.ps, a.stride, a.nx, ilo, ihi, ilast);
      const float *wr = wp + (long long)j * a.nx;
      const float *dr = dp + (long long)j * a.nx;
      for (int ii = ilo; ii <= ihi + ilast; ++ii) {
        const int i = ii > ihi ? a.nx - 1 : ii;
        const float wk = __ldg(wr + i);
        if (wk > 0.f) {  // a dropped patch has weight 0 (its D* may be NaN)
          const float mx = mask[x - grid_origin(i, a.nx, a.w, a.ps, a.stride)];
          A = fmaf(mx, wk * __ldg(dr + i), A);
          B = fmaf(mx, wk, B);
        }
      }
    }
    sA[jj][xx] = A;
    sB[jj][xx] = B;
  }
  __syncthreads();

  // pass 2: y-weighted sums over the covering rows of each pixel
  const int xx = tid & (kTileX - 1);
  const int x = X0 + xx;
  for (int yy = tid / kTileX; yy < tile_y; yy += blockDim.x / kTileX) {
    const int y = Y0 + yy;
    if (x >= a.w || y >= a.h) continue;
    int lo, hi, last;
    cover_range(y, a.h, a.ps, a.stride, a.ny, lo, hi, last);
    float num = 0.f, den = 0.f;
    for (int j = lo; j <= hi + last; ++j) {
      const int row = j > hi ? a.ny - 1 : j;  // past the regular rows: the last row
      const int jj = j > hi ? nreg : j - jlo;
      const float my = mask[y - grid_origin(row, a.ny, a.h, a.ps, a.stride)];
      num = fmaf(my, sA[jj][xx], num);
      den = fmaf(my, sB[jj][xx], den);
    }
    float out;
    if (den > 0.f)
      out = __fdividef(num, den);  // den >= the smallest mask weight, far below 2^126
    else if (a.is_finest)
      out = __int_as_float(0x7fc00000);  // NaN: not estimated
    else if (a.coarse)
      out = 2.f * bilinear_clamped(a.coarse + (long long)b * a.cplane, a.cw, a.ch, x * 0.5f,
                                   y * 0.5f);
    else
      out = 0.f;
    a.out[(long long)b * a.plane + (long long)y * a.w + x] = out;
  }
}

// Strip variant for patch grids whose stride S divides the patch size PS
// (M = PS / S covering patch rows per pixel row; overlap 0.75 gives M = 4 for
// PS 8, 12 and 16). A thread owns one column and a strip of K pixel rows. The
// pixel rows of group g (rows gS .. gS + S - 1) are covered by the same M
// regular patch rows g - M + 1 .. g (those in [0, ny - 2]) plus, near the
// bottom, the last patch row (origin h - PS). Walking down the strip one group
// at a time adds one regular patch row, so each thread computes the x-weighted
// sums A_j, B_j of one new patch row per group and keeps the last M in
// registers; the y-weighted sums then take them in ascending j, as the tiled
// kernel does, with the same operations, so the two give identical results.
// The block's patch values are staged in shared memory once (one barrier);
// a warp's reads of them (19 patches of a row for 32 columns) are broadcasts.
// The y weights sit in registers (PS / 2 of them: the mask is symmetric). At
// PS 8 the kernel runs at up to 72 registers, 7 blocks of 128 per SM, which
// measured faster than 8 blocks at 64.
template <int PS, int S, int K>
__global__ void __launch_bounds__(128, PS == 8 ? 7 : 6) densify_strip_kernel(const DensifyArgs a) {
  constexpr int M = PS / S;
  static_assert(M * S == PS && K % S == 0, "strip geometry");
  // patch columns / rows a block (128 columns x K rows) can need, plus one
  // slot each for the last (irregular) patch column / row
  constexpr int NCMAX = (128 + S - 1) / S + M + 2, NRMAX = K / S + M + 1;
  // Whatever the image size, a block's regular patch columns number at most
  // (126 + PS) / S + 1 (all of [ilo(X0), ihi(X0 + 127)]) and its regular rows
  // at most K / S + M - 1 (rows g0 - M + 1 .. g0 + K / S - 1): with the last
  // column / row slot they fit the tile.
  static_assert((126 + PS) / S + 1 + 1 <= NCMAX && K / S + M - 1 + 1 <= NRMAX, "tile bounds");
  // column ZC is never a patch column: it holds (0, 0), the value of a patch
  // that does not cover the pixel
  constexpr int ZC = NCMAX - 1;
  static_assert((126 + PS) / S + 1 + 1 <= ZC, "zero column");
  // staged patch values as (w D*, w) pairs; a dropped patch (w <= 0) as (0, 0)
  __shared__ float2 swd[NRMAX][NCMAX];
  __shared__ float smask[PS];
  pdl_enter();
  const int X0 = blockIdx.x * 128, x = X0 + (int)threadIdx.x;
  const int Y0 = blockIdx.y * K, b = blockIdx.z;
  const bool active = x < a.w;
  const float *wp = a.weight + (long long)b * a.np;
  const float *dp = a.d_star + (long long)b * a.np;
  // The block's patch rows and columns are staged into shared memory with
  // asynchronous copies, all in flight at once (one round trip per block).
  const int xlast_b = min(X0 + 127, a.w - 1);
  const int g0 = Y0 / S, gend = (min(Y0 + K, a.h) - 1) / S;
  const int ic0 = X0 - PS + 1 <= 0 ? 0 : (X0 - PS + 1 + S - 1) / S;
  const int ic1 = min(xlast_b / S, a.nx - 2);
  const int jr0 = max(0, g0 - M + 1), jr1 = min(gend, a.ny - 2);
  const int NC = max(0, ic1 - ic0 + 1), NR = max(0, jr1 - jr0 + 1);
  {
    // thread cc copies column cc of every tile row (NC + 1 <= NCMAX < 128
    // columns): no per-element division, one column index per thread
    static_assert(NCMAX <= 128, "one tile column per thread");
    const int cc = threadIdx.x;
    if (cc <= NC) {
      const int i = cc < NC ? ic0 + cc : a.nx - 1;
      const unsigned dd0 = (unsigned)__cvta_generic_to_shared(&swd[0][cc].x);
      for (int rr = 0; rr <= NR; ++rr) {
        const int j = rr < NR ? jr0 + rr : a.ny - 1;
        const long long o = (long long)j * a.nx + i;
        const unsigned step = (unsigned)(rr * NCMAX * sizeof(float2));
        BDIS_CHECKED_ONLY(if (!in_bounds(o, a.np, kCheckDensifyTile)) {
          swd[rr][cc] = make_float2(0.f, 0.f);
          continue;
        })
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(dd0 + step), "l"(dp + o));
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(dd0 + step + 4),
                     "l"(wp + o));
      }
      asm volatile("cp.async.wait_all;\n" ::: "memory");
      // the thread's own copies are complete: form (w D*, w), as the tiled kernel does
      for (int rr = 0; rr <= NR; ++rr) {
        const float2 v = swd[rr][cc];  // (D*, w)
        swd[rr][cc] = v.y > 0.f ? make_float2(v.y * v.x, v.y) : make_float2(0.f, 0.f);
      }
    } else if (cc == ZC) {
      for (int rr = 0; rr <= NR; ++rr) swd[rr][ZC] = make_float2(0.f, 0.f);
    }
  }
  if (threadIdx.x < PS) {  // Gaussian mask (Eq. 5): the tiled kernel's expression and values
    const float m = (float)threadIdx.x - (PS - 1) * 0.5f;
    smask[threadIdx.x] = expf(-(m * m) / a.two_s2);
  }
  __syncthreads();
  if (!active || Y0 >= a.h) return;
  auto mask_at = [&](int q) { return smask[q]; };
  // covering patches of column x: regular ilo .. ihi (<= nx - 2), then the last;
  // their x weights are fixed for the thread
  const int ilo = x - PS + 1 <= 0 ? 0 : (x - PS + 1 + S - 1) / S;
  const int ihi = min(x / S, a.nx - 2);
  const bool ilast = x >= a.w - PS;
  float mxr[M + 1];
#pragma unroll
  for (int k = 0; k <= M; ++k) {
    const int q = x - (ilo + k) * S;
    mxr[k] = (q >= 0 && q < PS) ? mask_at(q) : 0.f;
  }
  const float mxl = ilast ? mask_at(x - (a.w - PS)) : 0.f;
  // covering patch k of column x (k = 0..M: the regular ilo + k, then the
  // last): its tile column (ZC where there is none) and its x weight
  int cck[M + 1];
  float mxk[M + 1];
#pragma unroll
  for (int k = 0; k <= M; ++k) {
    const int ii = ilo + k;
    const bool reg = ii <= ihi;
    cck[k] = reg ? ii - ic0 : (ilast && ii == ihi + 1) ? NC : ZC;
    mxk[k] = reg ? mxr[k] : mxl;
  }
  // a patch row's (w D*, w) pairs (staged; read one row ahead of their use)
  // and its x-weighted sums, in the same order and with the same fmas as the
  // tiled kernel: a patch that is not used, or dropped, is (0, 0) and adds
  // exactly 0
  auto load_row = [&](int j, float2 *v) {
    const float2 *row = swd[j <= a.ny - 2 ? j - jr0 : NR];
#pragma unroll
    for (int k = 0; k <= M; ++k) v[k] = row[cck[k]];
  };
  auto sum_row = [&](const float2 *v, float2 &AB) {
    AB = make_float2(0.f, 0.f);
#pragma unroll
    for (int k = 0; k <= M; ++k) AB = __ffma2_rn(make_float2(mxk[k], mxk[k]), v[k], AB);
  };
  auto row_sums = [&](int j, float2 &AB) {
    float2 v[M + 1];
    load_row(j, v);
    sum_row(v, AB);
  };
  const int ylast = a.h - PS;  // first pixel row the last patch row covers
  float2 last = make_float2(0.f, 0.f);
  bool have_last = false;
  // ring of the regular rows g - M + 1 .. g (slot k holds row g - M + 1 + k),
  // each as its (x-weighted numerator, denominator) pair
  float2 rAB[M];
#pragma unroll
  for (int k = 0; k < M - 1; ++k) {
    const int j = g0 - M + 1 + k;
    rAB[k + 1] = make_float2(0.f, 0.f);
    if (j >= 0 && j <= a.ny - 2) row_sums(j, rAB[k + 1]);
  }

  const long long obase = (long long)b * a.plane + x;
  const int yend = min(Y0 + K, a.h);
  // the y weights of the group's rows, in registers: the mask is symmetric
  // (its offsets from the centre are +-m), so PS / 2 values hold it
  float myr[PS / 2];
#pragma unroll
  for (int q = 0; q < PS / 2; ++q) myr[q] = smask[q];
  float2 nv[M + 1];  // row g's loads, issued during group g - 1
  if (g0 <= a.ny - 2) load_row(g0, nv);
  for (int g = g0; g * S < yend; ++g) {
    float2 cv[M + 1];
#pragma unroll
    for (int k = 0; k <= M; ++k) cv[k] = nv[k];
    if (g + 1 <= a.ny - 2 && (g + 1) * S < yend) load_row(g + 1, nv);
#pragma unroll
    for (int k = 0; k < M - 1; ++k) rAB[k] = rAB[k + 1];
    rAB[M - 1] = make_float2(0.f, 0.f);
    if (g <= a.ny - 2) sum_row(cv, rAB[M - 1]);
#pragma unroll
    for (int t = 0; t < S; ++t) {
      const int y = g * S + t;
      if (y >= yend) break;
      // (numerator, denominator) as one packed f32x2 FMA per covering row:
      // per component the same fma as the tiled kernel; a ring slot outside
      // the regular rows holds (0, 0) and adds exactly 0
      float2 nd2 = make_float2(0.f, 0.f);
#pragma unroll
      for (int k = 0; k < M; ++k) {
        const int q = t + (M - 1 - k) * S;  // known at compile time (unrolled)
        const float my = myr[q < PS / 2 ? q : PS - 1 - q];
        nd2 = __ffma2_rn(make_float2(my, my), rAB[k], nd2);
      }
      if (y >= ylast) {
        if (!have_last) {
          row_sums(a.ny - 1, last);
          have_last = true;
        }
        const float my = mask_at(y - ylast);
        nd2 = __ffma2_rn(make_float2(my, my), last, nd2);
      }
      const float num = nd2.x, den = nd2.y;
      float out;
      if (den > 0.f)
        out = __fdividef(num, den);  // den >= the smallest mask weight, far below 2^126
      else if (a.is_finest)
        out = __int_as_float(0x7fc00000);  // NaN: not estimated
      else if (a.coarse)
        out = 2.f * bilinear_clamped(a.coarse + (long long)b * a.cplane, a.cw, a.ch, x * 0.5f,
                                     y * 0.5f);
      else
        out = 0.f;
      BDIS_CHECKED_ONLY(if (!in_bounds(obase + (long long)y * a.w, a.total, kCheckDensifyOut))
                            continue;)
      a.out[obase + (long long)y * a.w] = out;
    }
  }
}

// DIS fusion (Eq. 2): per pixel, every covering patch whose sample x - D*_k is
// inside the right image, weighted by weight_k / max(r^2, 1) with r the
// photometric residual R(x - D*_k) - L(x). The weights depend on the pixel
// and the patch jointly, so this is a direct gather over the covering patches.
//
// A block takes 32 columns x 8 rows, two rows a thread, and stages each patch
// that touches them once, as what a pixel needs of it: D*, its fraction, its
// integer sample shift and its weight.
// A patch's record is then read once for both rows; a warp's lanes share their
// rows, so which patch rows cover which of them is uniform. Each pixel adds its
// patches in ascending row, then column, order, as a plain loop would.
//
// Where every patch of the block has weight 1 (all that the search gives) and
// samples inside the image from all of its columns, nothing is tested per pixel
// and the weight is a reciprocal. That is the common block, bound by
// instruction issue. 64 pairs of 640x480, five levels: 575 us, where a kernel
// of one pixel per thread that split D* and divided per pixel and patch took
// 1211; one row per thread takes 835 us, four rows 664.
struct DisPatch {
  float D, t;
  int k;  // sample column of pixel x: x + k (far outside for a dropped patch)
  float weight;
};

constexpr int kDisX = 32, kDisR = 2, kDisY = 4 * kDisR;

// Most patch columns (rows) that touch n_px consecutive pixels, with the last one.
__host__ __device__ inline int dis_span(int n_px, int ps, int stride) {
  return (n_px + ps - 2) / stride + 2;
}

// The patches the block staged: rows jr0 .. jr1 and columns ic0 .. ic1 of the
// regular grid, each followed by the last (irregular) one; nc per row.
struct DisTile {
  const DisPatch *rec;
  int ic0, ic1, jr0, jr1, nc;
};

// 1 / m for m in [1, 2^124]: one Newton step with fused residual on an
// approximation within 1 ulp, which rounds correctly unless m's significand is
// all ones (P. Markstein, IBM J. Res. Dev. 34, 1990), and there too on this device:
// the same as the division for every float of the range.
// __frcp_rn's test of its argument's range, per pixel and patch, made the whole
// call 10% slower (64 pairs of 640x480: 1965 us against 1786, same maps).
__device__ __forceinline__ float dis_reciprocal(float m) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(m));
  return fmaf(y, fmaf(-m, y, 1.f), y);
}

// Numerators and denominators of column x, rows y0 and y0 + 1. PLAIN: weights 1
// and every sample inside. There a residual is cut to 2^62, which keeps the
// reciprocal in its range: its weight is then 2^-124 and not less, which changes
// nothing beside a total above 2^-90.
template <bool PLAIN>
__device__ __forceinline__ void dis_gather(const DensifyArgs &a, const DisTile &tile, int b, int x,
                                           int y0, float (&num)[kDisR], float (&den)[kDisR]) {
  int ilo, ihi, ilast, jlo, jhi, jlast, unused, unused2;
  cover_range(x, a.w, a.ps, a.stride, a.nx, ilo, ihi, ilast);
  cover_range(y0, a.h, a.ps, a.stride, a.ny, jlo, unused, unused2);
  cover_range(min(y0 + kDisR, a.h) - 1, a.h, a.ps, a.stride, a.ny, unused, jhi, jlast);
  const long long p0 = (long long)b * a.plane + (long long)y0 * a.w + x;
  const float2 *Rx[kDisR];
  float Lx[kDisR];
#pragma unroll
  for (int r = 0; r < kDisR; ++r) {
    Rx[r] = a.R2 + p0 + (long long)r * a.w;
    Lx[r] = y0 + r < a.h ? __ldg(a.L + p0 + (long long)r * a.w) : 0.f;
    num[r] = den[r] = 0.f;
  }
  auto add = [&](const DisPatch &p, int r) {
    const float2 q = __ldg(Rx[r] + p.k);
    const float e = fmaf(p.t, q.y, q.x) - Lx[r];
    float wpx;
    if (PLAIN) {
      const float c = fminf(fmaxf(fabsf(e), 1.f), 0x1p62f);
      wpx = dis_reciprocal(c * c);  // c * c = max(e * e, 1)
    } else {
      wpx = p.weight / fmaxf(e * e, 1.f);
    }
    num[r] = fmaf(wpx, p.D, num[r]);
    den[r] += wpx;
  };
  const int cn = max(0, ihi - ilo + 1), n = cn + ilast;
  for (int jj = jlo; jj <= jhi + jlast; ++jj) {
    const bool lastrow = jj > jhi;
    const int oy = lastrow ? a.h - a.ps : jj * a.stride;
    const int row = (lastrow ? tile.jr1 - tile.jr0 + 1 : jj - tile.jr0) * tile.nc;
    const DisPatch *reg = tile.rec + row + (ilo - tile.ic0);        // the regular ones, in order
    const DisPatch *last = tile.rec + row + (tile.ic1 - tile.ic0 + 1);
    bool cov[kDisR], all = true;
#pragma unroll
    for (int r = 0; r < kDisR; ++r) {
      cov[r] = (unsigned)(y0 + r - oy) < (unsigned)a.ps && y0 + r < a.h;
      all = all && cov[r];
    }
    if (PLAIN && all) {
#pragma unroll 4
      for (int i = 0; i < cn; ++i) {
        const DisPatch p = reg[i];
#pragma unroll
        for (int r = 0; r < kDisR; ++r) add(p, r);
      }
      if (ilast) {
        const DisPatch p = *last;
#pragma unroll
        for (int r = 0; r < kDisR; ++r) add(p, r);
      }
    } else {
#pragma unroll 1
      for (int i = 0; i < n; ++i) {
        const DisPatch p = i < cn ? reg[i] : *last;
        // the sample is inside: columns [0, w - 2], or the last one at t = 0
        if (!PLAIN && (unsigned)(x + p.k) >= (unsigned)(p.t == 0.f ? a.w : a.w - 1)) continue;
#pragma unroll
        for (int r = 0; r < kDisR; ++r)
          if (cov[r]) add(p, r);
      }
    }
  }
}

__global__ void __launch_bounds__(128, 8) densify_dis_kernel(const DensifyArgs a, int across,
                                                              int count) {
  extern __shared__ __align__(16) unsigned char dis_smem[];
  pdl_enter();
  const int row = (int)blockIdx.x / across;  // of blocks; one grid dimension: no limit on rows
  const int X0 = ((int)blockIdx.x - row * across) * kDisX, Y0 = row * kDisY;
  const int x = X0 + (int)(threadIdx.x & 31), y0 = Y0 + (int)(threadIdx.x >> 5) * kDisR;
  const int xe = min(X0 + kDisX, a.w) - 1, ye = min(Y0 + kDisY, a.h) - 1;
  DisTile tile;
  int unused, unused2;
  cover_range(X0, a.w, a.ps, a.stride, a.nx, tile.ic0, unused, unused2);
  cover_range(xe, a.w, a.ps, a.stride, a.nx, unused, tile.ic1, unused2);
  cover_range(Y0, a.h, a.ps, a.stride, a.ny, tile.jr0, unused, unused2);
  cover_range(ye, a.h, a.ps, a.stride, a.ny, unused, tile.jr1, unused2);
  tile.ic1 = max(tile.ic1, tile.ic0 - 1);
  tile.jr1 = max(tile.jr1, tile.jr0 - 1);
  tile.nc = tile.ic1 - tile.ic0 + 2;
  const int n = tile.nc * (tile.jr1 - tile.jr0 + 2);
  DisPatch *rec = reinterpret_cast<DisPatch *>(dis_smem);
  tile.rec = rec;
  for (int b = blockIdx.z; b < count; b += gridDim.z) {
    const float *wp = a.weight + (long long)b * a.np;
    const float *dp = a.d_star + (long long)b * a.np;
    bool plain = true;
    for (int s = threadIdx.x; s < n; s += 128) {
      const int rr = s / tile.nc, cc = s - rr * tile.nc;
      const int j = tile.jr0 + rr <= tile.jr1 ? tile.jr0 + rr : a.ny - 1;
      const int i = tile.ic0 + cc <= tile.ic1 ? tile.ic0 + cc : a.nx - 1;
      const float wk = __ldg(wp + (long long)j * a.nx + i);
      const float D = __ldg(dp + (long long)j * a.nx + i);
      const float nd = fminf(fmaxf(-D, -1.0e7f), 1.0e7f);
      const float f = floorf(nd), t = nd - f;
      const int k = wk > 0.f ? (int)f : -(1 << 30);
      plain = plain && wk == 1.f && X0 + k >= 0 && xe + k < a.w - 1;
      rec[s] = DisPatch{D, t, k, wk};
    }
    plain = __syncthreads_and(plain) != 0;
    if (x < a.w && y0 < a.h) {
      float num[kDisR], den[kDisR];
      if (plain) dis_gather<true>(a, tile, b, x, y0, num, den);
      bool again = !plain;
#pragma unroll
      for (int r = 0; r < kDisR; ++r)  // all its residuals beyond 2^45: take them as they are
        if (plain && y0 + r < a.h && !(den[r] > 0x1p-90f)) again = true;
      if (again) dis_gather<false>(a, tile, b, x, y0, num, den);
#pragma unroll
      for (int r = 0; r < kDisR; ++r) {
        const int y = y0 + r;
        if (y >= a.h) break;
        float out;
        if (den[r] > 0.f)
          out = __fdividef(num[r], den[r]);
        else if (a.is_finest)
          out = __int_as_float(0x7fc00000);
        else if (a.coarse)
          out = 2.f * bilinear_clamped(a.coarse + (long long)b * a.cplane, a.cw, a.ch, x * 0.5f,
                                       y * 0.5f);
        else
          out = 0.f;
        a.out[(long long)b * a.plane + (long long)y * a.w + x] = out;
      }
    }
    if (b + (int)gridDim.z < count) __syncthreads();  // the records are restaged
  }
}

// Full-size map from level f: bilinear over finite neighbours with positive
// weight, values times 2^f. A thread takes four pixels of a row, 32 apart (each
// store of a warp is one line), so the row's part of the arithmetic is shared;
// where all four neighbours count, their weights add up to 1 and there is
// nothing to divide by. The level's rows are read through L1: bound by issue,
// then by the map's write. 24 maps of 501x375 from level 1: 15.5 us, where one
// pixel per thread, by 64-bit index divisions, took 28.8.
constexpr int kUpPixels = 4;

// FROM: rows from row0 on (a launch of its own; the addition costs the others 5%).
template <bool FROM>
__global__ void __launch_bounds__(256) upsample_kernel(const float *__restrict__ M, int mw, int mh,
                                                       float scale, int w, int h, int count,
                                                       float *__restrict__ out, int row0) {
  pdl_enter();
  const int X0 = blockIdx.x * (32 * kUpPixels) + (threadIdx.x & 31);
  const int y = (FROM ? row0 : 0) + blockIdx.y * 8 + (threadIdx.x >> 5);
  if (y >= h) return;
  const float inv = 1.f / scale;  // a power of two: exact
  const float fy = fminf((float)y * inv, (float)(mh - 1));
  const int y0 = (int)floorf(fy), y1 = min(y0 + 1, mh - 1);
  const float ty = fy - y0;
  for (int b = blockIdx.z; b < count; b += gridDim.z) {
    const float *r0 = M + ((long long)b * mh + y0) * mw, *r1 = M + ((long long)b * mh + y1) * mw;
    float *o = out + ((long long)b * h + y) * w;
#pragma unroll
    for (int p = 0; p < kUpPixels; ++p) {
      const int x = X0 + 32 * p;
      if (x >= w) break;
      const float fx = fminf((float)x * inv, (float)(mw - 1));
      const int x0 = (int)floorf(fx), x1 = min(x0 + 1, mw - 1);
      const float tx = fx - x0;
      const float wt[4] = {(1.f - tx) * (1.f - ty), tx * (1.f - ty), (1.f - tx) * ty, tx * ty};
      const float v[4] = {__ldg(r0 + x0), __ldg(r0 + x1), __ldg(r1 + x0), __ldg(r1 + x1)};
      float s = 0.f, sw = 0.f;
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (wt[q] > 0.f && isfinite(v[q])) {
          s += wt[q] * v[q];
          sw += wt[q];
        }
      o[x] = sw == 1.f ? scale * s : sw > 0.f ? scale * s / sw : __int_as_float(0x7fc00000);
    }
  }
}

// R15 warm start: level-`level` seed map from a previous full-size disparity:
// mean of its finite values over the 2^level block centred on the sample
// point, divided by 2^level; 0 where none is finite. The values are added in
// row-major order, so the mean does not depend on which kernel runs.
// Small blocks (2^level <= 4) and blocks wider than a stage: a thread per cell.
__global__ void warm_map_kernel(const float *__restrict__ P, int w, int h, int level, int mw,
                                int mh, long long total, float *__restrict__ out) {
  pdl_enter();
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= total) return;
  const long long mplane = (long long)mw * mh;
  const int b = (int)(idx / mplane);
  const int rem = (int)(idx - (long long)b * mplane);
  const int Y = rem / mw, X = rem - (rem / mw) * mw;
  const int s = 1 << level;
  const int half = s / 2;
  const int x0 = max(X * s - half, 0), x1 = min(X * s + half + (s == 1 ? 1 : 0), w);
  const int y0 = max(Y * s - half, 0), y1 = min(Y * s + half + (s == 1 ? 1 : 0), h);
  const float *Pb = P + (long long)b * w * h;
  float sum = 0.f;
  int n = 0;
  for (int y = y0; y < y1; ++y)
    for (int x = x0; x < x1; ++x) {
      const float v = __ldg(Pb + (size_t)y * w + x);
      if (isfinite(v)) {
        sum += v;
        ++n;
      }
    }
  out[idx] = n ? sum / (float)n / (float)s : 0.f;
}

// The same map for blocks of 8 x 8 and more. Alone, a thread of the kernel
// above reads 4^level values one cache line at a time (83 us for four
// 1280x1024 maps at level 5, and 220 us when an overlapped launch put its few
// blocks on the first SMs to free up; the map's bytes take 3 us). Here a block
// stages `cells` neighbouring cells of one cell row in shared memory, reading
// whole row segments, as many rows at a time as fit kWarmStage values, and one
// lane per cell adds them in the same row-major order. Values outside the
// image are staged as NaN, which adds nothing and is not counted. What bounds
// it then is the map's read and the chain of 4^level adds, wherever its blocks
// land: a warm-started call on four such frames fell from 756 to 536 us among
// others (618 to 568 us alone).
constexpr int kWarmThreads = 128, kWarmStage = 8192, kWarmCellsMax = 32;

__global__ void __launch_bounds__(kWarmThreads) warm_map_staged_kernel(
    const float *__restrict__ P, int w, int h, int level, int mw, int mh, int count, int cells,
    float *__restrict__ out) {
  // cell c's staged values, row by row, start at c * (rows * s + 4): 16-byte
  // aligned, and eight lanes' 16-byte reads fall in distinct banks
  __shared__ __align__(16) float stage[kWarmStage + 4 * kWarmCellsMax];
  pdl_enter();
  const int s = 1 << level, half = s / 2;
  const int cell_bits = __ffs(cells) - 1, seg_bits = level + cell_bits;  // cells: a power of two
  const int seg = 1 << seg_bits;  // columns of a row segment
  const int rows = min(s, kWarmStage / seg), pitch = rows * s + 4;
  const int X0 = blockIdx.x * cells, Y = blockIdx.y;
  const int xs = X0 * s - half, ys = Y * s - half;
  const float nan = __int_as_float(0x7fc00000);
  for (int b = blockIdx.z; b < count; b += gridDim.z) {
    const float *Pb = P + (long long)b * w * h;
    float sum = 0.f;
    int n = 0;
    for (int r0 = 0; r0 < s; r0 += rows) {  // rows divides s: both are powers of two
      __syncthreads();
      constexpr int U = 16;  // loads in flight per thread
      for (int i0 = threadIdx.x; i0 < rows * seg; i0 += U * kWarmThreads) {
        float v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int i = i0 + u * kWarmThreads, r = i >> seg_bits, o = i & (seg - 1);
          const int x = xs + o, y = ys + r0 + r;
          const bool in = i < rows * seg && x >= 0 && x < w && y >= 0 && y < h;
          v[u] = in ? __ldg(Pb + (size_t)y * w + x) : nan;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int i = i0 + u * kWarmThreads, r = i >> seg_bits, o = i & (seg - 1);
          if (i < rows * seg) stage[(o >> level) * pitch + (r << level) + (o & (s - 1))] = v[u];
        }
      }
      __syncthreads();
      if ((int)threadIdx.x < cells) {
        const float4 *q = reinterpret_cast<const float4 *>(stage + threadIdx.x * pitch);
#pragma unroll 4
        for (int i = 0; i < rows * s / 4; ++i) {
          const float4 f = q[i];
          const float e[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const bool fin = isfinite(e[k]);
            sum += fin ? e[k] : 0.f;  // adding 0 leaves the sum as it is
            n += fin ? 1 : 0;
          }
        }
      }
    }
    const int X = X0 + (int)threadIdx.x;
    if ((int)threadIdx.x < cells && X < mw)
      out[((long long)b * mh + Y) * mw + X] = n ? sum / (float)n / (float)s : 0.f;
  }
}

}  // namespace

cudaError_t launch_warm_map(const float *prev, int w, int h, int level, int count, float *out,
                            cudaStream_t st) {
  const int mw = level_dim(w, level), mh = level_dim(h, level);
  const long long total = (long long)mw * mh * count;
  if (total == 0) return cudaSuccess;
  if (level >= 3 && level <= 13 && mh <= 65535) {
    // a lane's chain of adds is as long whatever the number of cells, so a
    // block takes few of them once a cell fills a good part of the stage
    const int cells = level <= 4 ? kWarmCellsMax : std::max(1, std::min(8, kWarmStage >> level));
    const dim3 grid((unsigned)((mw + cells - 1) / cells), (unsigned)mh,
                    (unsigned)std::min(count, 65535));
    return launch_maybe_overlapped(warm_map_staged_kernel, grid, dim3(kWarmThreads), 0, st, prev,
                                   w, h, level, mw, mh, count, cells, out);
  }
  const int threads = 128;
  return launch_maybe_overlapped(warm_map_kernel, dim3((unsigned)((total + threads - 1) / threads)),
                                 dim3(threads), 0, st, prev, w, h, level, mw, mh, total, out);
}

namespace {
int g_densify_tile = 0;  // process-wide densify kernel choice (0 = strips where they apply)
}  // namespace

int densify_tile() { return g_densify_tile; }
void set_densify_tile(int tile_height) { g_densify_tile = tile_height; }

void fill_densify_args(DensifyArgs &a, int w, int h, int count, const bdis_params &p) {
  a.tile_y = g_densify_tile;
  a.w = w;
  a.h = h;
  a.plane = (long long)w * h;
  a.total = a.plane * count;
  a.ps = p.patch_size;
  a.stride = grid_stride(p.patch_size, p.overlap);
  a.nx = grid_count(w, p.patch_size, a.stride);
  a.ny = grid_count(h, p.patch_size, a.stride);
  a.np = a.nx * a.ny;
  a.two_s2 = 2.f * p.sigma_s * p.sigma_s;
  a.fusion = p.fusion;
}

cudaError_t launch_densify(const DensifyArgs &a, cudaStream_t st) {
  if (a.total == 0) return cudaSuccess;
  if (a.fusion == BDIS_FUSION_DIS) {
    const int n = (int)(a.total / a.plane);
    const int across = (a.w + kDisX - 1) / kDisX;
    const dim3 grid((unsigned)across * (unsigned)((a.h + kDisY - 1) / kDisY), 1,
                    (unsigned)std::min(n, 65535));
    // at most 64 x 40 records of 16 B, at stride 1 and patch size 32
    const size_t smem = (size_t)dis_span(kDisX, a.ps, a.stride) *
                        dis_span(kDisY, a.ps, a.stride) * sizeof(DisPatch);
    return launch_maybe_overlapped(densify_dis_kernel, grid, dim3(128), smem, st, a, across, n);
  }
  const int count = (int)(a.total / a.plane);
  if (a.tile_y == 0 && a.nx > 0 && a.ny > 0) {  // default: strips where the geometry allows
    // A thread walks its column down a strip of K rows, one dependent step
    // per group of S rows, so a launch takes at least one strip's walk. Where
    // strips of 32 rows would not give every SM two blocks (small levels,
    // small batches), strips of 8 (9) rows spread the same rows over four
    // times the blocks. The map is the same either way: each row's
    // x-weighted sums depend only on the row and the column.
    const unsigned bx = (unsigned)((a.w + 127) / 128);
    const bool short_strips = (long long)bx * ((a.h + 31) / 32) * count < 2LL * device_sms();
    auto rows = [&](int K) { return dim3(bx, (unsigned)((a.h + K - 1) / K), (unsigned)count); };
    if (a.ps == 8 && a.stride == 2)
      return short_strips ? launch_maybe_overlapped(densify_strip_kernel<8, 2, 8>, rows(8),
                                                    dim3(128), 0, st, a)
                          : launch_maybe_overlapped(densify_strip_kernel<8, 2, 32>, rows(32),
                                                    dim3(128), 0, st, a);
    if (a.ps == 12 && a.stride == 3)
      return short_strips ? launch_maybe_overlapped(densify_strip_kernel<12, 3, 9>, rows(9),
                                                    dim3(128), 0, st, a)
                          : launch_maybe_overlapped(densify_strip_kernel<12, 3, 30>, rows(30),
                                                    dim3(128), 0, st, a);
    if (a.ps == 16 && a.stride == 4)
      return short_strips ? launch_maybe_overlapped(densify_strip_kernel<16, 4, 8>, rows(8),
                                                    dim3(128), 0, st, a)
                          : launch_maybe_overlapped(densify_strip_kernel<16, 4, 32>, rows(32),
                                                    dim3(128), 0, st, a);
  }
  // Tiles of 32 rows; of 8 where those would not give every SM two blocks (small
  // levels, small batches): the same map, with a quarter of the work in a
  // block's serial loops (a call on one 160x120 pair, three levels: 45 us with
  // 32 rows, 41 with 8). Launched as a programmatic dependent up to one block
  // per SM: 43 us without; but with more, where its 256-thread blocks crowd the
  // SMs that free up first, a call on 24 pairs of 501x375 took 226 us (two per
  // SM at one level) and 231 (eight at another) against 220.
  DensifyArgs t = a;
  if (t.tile_y <= 0)
    t.tile_y = (long long)((a.w + kTileX - 1) / kTileX) * ((a.h + kTileY - 1) / kTileY) * count <
                       2LL * device_sms()
                   ? 8
                   : kTileY;
  const dim3 grid((unsigned)((a.w + kTileX - 1) / kTileX),
                  (unsigned)((a.h + t.tile_y - 1) / t.tile_y), (unsigned)count);
  return launch_overlapped_upto(1, densify_kernel, grid, dim3(256), 0, st, t);
}

cudaError_t launch_upsample(const float *map, int mw, int mh, int level, int w, int h, int count,
                            float *out, cudaStream_t st) {
  if ((long long)w * h * count == 0) return cudaSuccess;
  cudaError_t e = cudaSuccess;
  constexpr int kRows = 65535 * 8;  // of one launch
  for (int row0 = 0; row0 < h && e == cudaSuccess; row0 += kRows) {
    const dim3 grid((unsigned)((w + 32 * kUpPixels - 1) / (32 * kUpPixels)),
                    (unsigned)((std::min(kRows, h - row0) + 7) / 8),
                    (unsigned)std::min(count, 65535));
    e = launch_maybe_overlapped(row0 ? upsample_kernel<true> : upsample_kernel<false>, grid,
                                dim3(256), 0, st, map, mw, mh, (float)(1 << level), w, h, count,
                                out, row0);
    if (h - row0 <= kRows) break;
  }
  return e;
}

cudaError_t take_check_densify(unsigned *v) { return take_check_word(v); }

}  // namespace bdis
