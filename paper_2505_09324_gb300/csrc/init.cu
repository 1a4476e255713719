// Region-of-interest superpixel initialiser (Sec. 3.2 A): K-means superpixels
// of the ROI mask, one Gaussian per segment (mean = segment centre, Cholesky
// factor of the segment covariance, colour = mean segment colour), plus
// isotropic Gaussians for the rest of the frame at caller-supplied positions.
//
// Readings (the paper leaves them open): seeds on a grid of step
// S = sqrt(A_roi / K) at ((i + 1/2) S, (j + 1/2) S) inside the mask; 10
// iterations of assignment (D = |col_p - col_c|^2 + (m/S)^2 |p - c|^2, m = 0.2,
// among centres within S of the pixel on both axes; ties to the lower index)
// and update (mean colour and position, clamped to within S of the seed, so the
// candidates of a pixel are the seeds of the 5 x 5 grid cells around it);
// Sigma = 4 (pixel-centre covariance + I/12) (the segment's second moment of
// area, widened so that the accumulated sum over a tiling of segments is flat),
// weight = A / (2 pi sqrt(det Sigma)) (the Gaussian's integral equals the area);
// background Gaussians: variance 4 a / (2 pi), weight 1/4 (integral a).
// Arithmetic: the assignment decides in single precision (explicitly rounded
// FP32 operations, centres kept as float); every segment sum is an exact
// integer (pixel centres as 2 x + 1 - 2 floor(seed), colours as
// rint(c 2^20)), gathered by the update or accumulated by warp-aggregated
// 64-bit atomics, in any order; means and covariances follow in a fixed
// sequence of double operations, so the result is reproducible bit for bit.
#include <math.h>
#include <stdio.h>

#include <algorithm>

#include "gs2d_internal.cuh"

namespace gs2d {
namespace {

constexpr double kCompactness = 0.2;
constexpr int kIterations = kRoiIterations;
constexpr double kKappa = 4.0;  // covariance scale: keeps the blend of a tiling flat
constexpr double kColourScale = 1048576.0;  // 2^20
constexpr double kColourLimit = 32.0;
constexpr int kSums = 9;  // n, u, v, uu, uv, vv, r, g, b

// Seed grid, derived on the device from the mask's area.
struct SpGeom {
  int M, gx, gy, ncell;
  double S, area;
  float S32, lam32;
};

struct SpArgs {
  int W, H, n, k_target;
  const float* frame;
  const uint8_t* mask;
  int* cell_of;                // [gy][gx] seed index or -1
  double* seed_xy;             // [2][n] (the first M used)
  int* seed_i;                 // [2][n] floor of the seeds
  float* cen;                  // [5][n]: r, g, b, x, y
  int* label;                  // [H][W]
  unsigned long long* acc;     // [kSums][n] exact segment sums (two's complement)
  SpGeom* geo;
  unsigned long long* area;    // mask pixel count
  int* blk;                    // per-block seed counts (the grid compaction)
};

// Segment sums of up to kGatherS pixels of grid step are gathered by the
// update (half a warp per centre, or several, over the pixels that can have
// joined it); beyond that a centre's window is long and the centres are few, and
// the assignment adds each pixel's moments with atomics instead.  The gathered
// window is (2 S)^2 pixels per centre, 4 A in all whatever S is, so only the
// number of half-warps falls with S: at 32 each has 256 steps of 16 pixels.
constexpr float kGatherS = 32.0f;
constexpr int kWave = 152;  // blocks of one wave

// Whether the update gathers: with at most a wave of centres half the step (the
// whole initialisation of a 256 x 256 frame with 70 centres 31 pixels apart: 286 us
// gathered, 226 by atomics).
__device__ __forceinline__ bool gathered(const SpGeom& g) {
  return g.S32 <= (g.M > kWave ? kGatherS : 0.5f * kGatherS);
}

// The pixel's colour on the 2^-20 grid: a power-of-two scaling, exact in
// float, then one rounding to the nearest integer.
__device__ __forceinline__ int colour_int(float c) {
  return __float2int_rn(fminf(fmaxf(c, -(float)kColourLimit), (float)kColourLimit) *
                        (float)kColourScale);
}

// Assignment: each ROI pixel joins the nearest candidate centre (FP32
// decisions).  A block takes a tile of 32 x 16 pixels and stages the centres
// of the cells around it once (the 5 x 5 cells of every pixel overlap), so
// the 25 candidates of a pixel are one shared 8-byte load and a window test
// each, and only those within S (about 4) cost the full distance.  No double
// precision here: FP64 issues at 1/64 of the FP32 rate, and the divisions and
// conversions this kernel had took nearly all of its time (1920 x 1080,
// 14 000 centres: 72 us a pass with per-pixel global candidates, FP64 cells
// and 64-bit atomic sums, 19 us now; 8 x 8 patches per warp whose lanes first
// discard centres for the whole patch executed fewer instructions and took
// 21 us).
//
// The cell of a pixel is floor(px / S) from one FP32 product, which may be
// off by one within 0.02 S of a cell border.  That cannot change the result:
// a centre within S of the pixel has its seed within 2 S, i.e. its cell's
// middle within 2 S of px, while the cell columns such an error adds or drops
// have theirs about 2.5 S away.
constexpr int kTileW = 32, kTileH = 16;
// cells of a tile at the smallest step (S = 1), with the two on either side
constexpr int kTileCells = (kTileW + 6) * (kTileH + 6);

__global__ void __launch_bounds__(256) k_sp_assign(SpArgs a, int first) {
  pdl_begin();
  __shared__ float2 s_xy[kTileCells];
  __shared__ float4 s_ci[kTileCells];  // r, g, b, centre index
  const SpGeom g = *a.geo;
  const int x0 = blockIdx.x * kTileW, y0 = blockIdx.y * kTileH;
  const int x = x0 + (threadIdx.x & 31), yt = y0 + (threadIdx.x >> 5);
  bool on[2];
#pragma unroll
  for (int k = 0; k < 2; k++) {
    const int y = yt + 8 * k;
    const bool in = x < a.W && y < a.H;
    on[k] = in && a.mask[(size_t)y * a.W + x];
    if (first && in && !on[k]) a.label[(size_t)y * a.W + x] = -1;
  }
  if (!__syncthreads_or(on[0] || on[1])) return;
  const float inv = 1.0f / g.S32;
  const int xl = min(x0 + kTileW, a.W) - 1, yl = min(y0 + kTileH, a.H) - 1;
  const int cx0 = (int)floorf(((float)x0 + 0.5f) * inv) - 2;
  const int cy0 = (int)floorf(((float)y0 + 0.5f) * inv) - 2;
  const int ncx = min((int)floorf(((float)xl + 0.5f) * inv) + 3 - cx0, kTileW + 6);
  const int ncy = min((int)floorf(((float)yl + 0.5f) * inv) + 3 - cy0, kTileH + 6);
  const int M = a.n;  // array stride
  for (int t = threadIdx.x; t < ncx * ncy; t += 256) {
    const int j = t / ncx, cy = cy0 + j, cx = cx0 + t - j * ncx;
    int c = -1;
    if (cx >= 0 && cx < g.gx && cy >= 0 && cy < g.gy) c = a.cell_of[cy * g.gx + cx];
    float2 xy = make_float2(INFINITY, INFINITY);  // never within S
    float4 ci = make_float4(0.f, 0.f, 0.f, __int_as_float(-1));
    if (c >= 0) {
      xy = make_float2(a.cen[3 * M + c], a.cen[4 * M + c]);
      ci = make_float4(a.cen[c], a.cen[M + c], a.cen[2 * M + c], __int_as_float(c));
    }
    s_xy[t] = xy;
    s_ci[t] = ci;
  }
  __syncthreads();
  const size_t HW = (size_t)a.W * a.H;
  const bool gather = gathered(g);
#pragma unroll
  for (int k = 0; k < 2; k++) {
    const int y = yt + 8 * k;
    const size_t idx = (size_t)y * a.W + x;
    int lab = -2;
    float pr = 0.f, pg = 0.f, pb = 0.f;
    if (on[k]) {
      pr = a.frame[idx];
      pg = a.frame[HW + idx];
      pb = a.frame[2 * HW + idx];
      const float px = (float)x + 0.5f, py = (float)y + 0.5f;
      // candidates in raster order of the cells, which is ascending seed
      // index (seeds are numbered in raster order of the grid)
      const int base = ((int)floorf(py * inv) - 2 - cy0) * ncx + (int)floorf(px * inv) - 2 - cx0;
      float best = INFINITY;
      int at = -1;
      for (int dj = 0; dj < 5; dj++) {
#pragma unroll
        for (int di = 0; di < 5; di++) {
          const int t = base + dj * ncx + di;
          const float2 xy = s_xy[t];
          const float dx = __fsub_rn(px, xy.x), dy = __fsub_rn(py, xy.y);
          if (!(fabsf(dx) <= g.S32 && fabsf(dy) <= g.S32)) continue;
          const float4 ci = s_ci[t];
          const float dr = __fsub_rn(pr, ci.x), dg = __fsub_rn(pg, ci.y), db = __fsub_rn(pb, ci.z);
          const float dc =
              __fadd_rn(__fadd_rn(__fmul_rn(dr, dr), __fmul_rn(dg, dg)), __fmul_rn(db, db));
          const float d =
              __fadd_rn(dc, __fmul_rn(g.lam32, __fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy))));
          if (d < best) {
            best = d;
            at = t;
          }
        }
      }
      lab = at >= 0 ? __float_as_int(s_ci[at].w) : -1;
      a.label[idx] = lab;
    }
    if (gather) continue;
    // large segments: exact moments by atomics, one per sum and group of
    // lanes with the same centre.  |u|, |v| <= 4 S + 2 and |q| <= 2^25, so a
    // group sum of up to 32 lanes stays within int32 for S < 2000
    int val[kSums] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
    if (lab >= 0) {
      const int u = 2 * x + 1 - 2 * a.seed_i[lab], v = 2 * y + 1 - 2 * a.seed_i[M + lab];
      val[0] = 1;
      val[1] = u;
      val[2] = v;
      val[3] = u * u;
      val[4] = u * v;
      val[5] = v * v;
      val[6] = colour_int(pr);
      val[7] = colour_int(pg);
      val[8] = colour_int(pb);
    }
    const unsigned peers = __match_any_sync(0xffffffffu, lab);
    const int leader = __ffs(peers) - 1;
#pragma unroll
    for (int q = 0; q < kSums; q++) val[q] = __reduce_add_sync(peers, val[q]);
    if (lab >= 0 && (int)(threadIdx.x & 31) == leader)
#pragma unroll
      for (int q = 0; q < kSums; q++)
        atomicAdd(&a.acc[(size_t)q * M + lab], (unsigned long long)(long long)val[q]);
  }
}

// Exact sum over the lanes of `mask` of 64-bit values of magnitude below 2^53:
// the low 24 bits and the rest are summed apart in 32-bit integers.
__device__ __forceinline__ long long lanes_sum64(unsigned mask, long long v) {
  const unsigned lo = __reduce_add_sync(mask, (unsigned)v & 0xffffffu);
  const int hi = __reduce_add_sync(mask, (int)(v >> 24));
  return (long long)hi * (1ll << 24) + (long long)lo;
}

// The nine exact sums of one of `parts` bands of rows of centre c's segment, by
// half a warp (a lane per column): every pixel that can have joined it lies within S of it.  The
// labels of kRows rows are loaded together and then the colours of those that
// match, so a window of 14 x 14 pixels (S of 7) costs a few load latencies
// rather than one per row.
constexpr int kRows = 7;

__device__ __forceinline__ void gather_segment(const SpArgs& a, const SpGeom& g, int c, int part,
                                               int parts, int hl, unsigned mask,
                                               long long out[kSums]) {
  const int M = a.n;
  const size_t HW = (size_t)a.W * a.H;
  const float cx = a.cen[3 * M + c], cy = a.cen[4 * M + c];
  const int sx = 2 * a.seed_i[c] - 1, sy = 2 * a.seed_i[M + c] - 1;
  // |x + 1/2 - cx| <= S, with room for FP32 rounding (2^-7 at 65536)
  const int xa = max(0, (int)ceilf(cx - g.S32 - 0.52f));
  const int xb = min(a.W - 1, (int)floorf(cx + g.S32 - 0.48f));
  int ya = max(0, (int)ceilf(cy - g.S32 - 0.52f));
  int yb = min(a.H - 1, (int)floorf(cy + g.S32 - 0.48f));
  const int band = (yb - ya + parts) / parts;
  ya += part * band;
  yb = min(yb, ya + band - 1);
  // per lane at most (2 S + 2)^2 / 16 pixels: moments stay below 2^31, the
  // colours need 64 bits
  int s[6] = {0, 0, 0, 0, 0, 0};
  long long q[3] = {0, 0, 0};
  for (int x = xa + hl; x <= xb; x += 16)
    for (int y0 = ya; y0 <= yb; y0 += kRows) {
      const size_t i0 = (size_t)y0 * a.W + x;
      bool hit[kRows];
      float col[kRows][3];
#pragma unroll
      for (int k = 0; k < kRows; k++)
        hit[k] = y0 + k <= yb && a.label[i0 + (size_t)k * a.W] == c;
#pragma unroll
      for (int k = 0; k < kRows; k++)
#pragma unroll
        for (int ch = 0; ch < 3; ch++)
          col[k][ch] = hit[k] ? a.frame[ch * HW + i0 + (size_t)k * a.W] : 0.0f;
#pragma unroll
      for (int k = 0; k < kRows; k++)
        if (hit[k]) {
          const int u = 2 * x - sx, v = 2 * (y0 + k) - sy;
          s[0] += 1;
          s[1] += u;
          s[2] += v;
          s[3] += u * u;
          s[4] += u * v;
          s[5] += v * v;
#pragma unroll
          for (int ch = 0; ch < 3; ch++) q[ch] += colour_int(col[k][ch]);
        }
    }
#pragma unroll
  for (int k = 0; k < 6; k++) out[k] = __reduce_add_sync(mask, s[k]);
#pragma unroll
  for (int k = 0; k < 3; k++) out[6 + k] = lanes_sum64(mask, q[k]);
}

// A centre's move to its segment's mean (clamped to within S of the seed) and
// mean colour.
__device__ __forceinline__ void move_centre(const SpArgs& a, const SpGeom& g, int c,
                                            const long long acc[kSums]) {
  const int M = a.n;  // array stride
  const long long n = acc[0];
  if (n <= 0) return;
  const double qx = a.seed_xy[c], qy = a.seed_xy[a.n + c];
  const double mx = __dadd_rn(__ddiv_rn((double)acc[1], (double)(2 * n)), floor(qx));
  const double my = __dadd_rn(__ddiv_rn((double)acc[2], (double)(2 * n)), floor(qy));
  a.cen[3 * M + c] = (float)fmin(fmax(mx, __dsub_rn(qx, g.S)), __dadd_rn(qx, g.S));
  a.cen[4 * M + c] = (float)fmin(fmax(my, __dsub_rn(qy, g.S)), __dadd_rn(qy, g.S));
  const double den = __dmul_rn((double)n, kColourScale);
#pragma unroll
  for (int ch = 0; ch < 3; ch++)
    a.cen[ch * M + c] = (float)__ddiv_rn((double)acc[6 + ch], den);
}

// A segment's Gaussian, from the exact sums of the last assignment.
__device__ __forceinline__ void segment_gaussian(const SpArgs& a, const SpGeom& g, int c,
                                                 const long long acc[kSums],
                                                 float* __restrict__ params) {
  const size_t HW = (size_t)a.W * a.H;
  const long long cnt = acc[0];
  const double qx = a.seed_xy[c], qy = a.seed_xy[a.n + c];
  float out[9];
  if (cnt == 0) {
    const int xi = min(max((int)floor(qx), 0), a.W - 1), yi = min(max((int)floor(qy), 0), a.H - 1);
    const size_t idx = (size_t)yi * a.W + xi;
    const double s = __dmul_rn(2.0, __ddiv_rn(g.S, sqrt(12.0)));
    out[0] = (float)qx;
    out[1] = (float)qy;
    out[2] = (float)s;
    out[3] = 0.0f;
    out[4] = (float)s;
    out[5] = a.frame[idx];
    out[6] = a.frame[HW + idx];
    out[7] = a.frame[2 * HW + idx];
    out[8] = 1.0f;
  } else {
    const double fn = (double)cnt;
    const double au = __ddiv_rn((double)acc[1], fn);
    const double av = __ddiv_rn((double)acc[2], fn);
    const double cxx = __ddiv_rn(__dsub_rn(__ddiv_rn((double)acc[3], fn), __dmul_rn(au, au)), 4.0);
    const double cxy = __ddiv_rn(__dsub_rn(__ddiv_rn((double)acc[4], fn), __dmul_rn(au, av)), 4.0);
    const double cyy = __ddiv_rn(__dsub_rn(__ddiv_rn((double)acc[5], fn), __dmul_rn(av, av)), 4.0);
    const double twelfth = __ddiv_rn(1.0, 12.0);
    const double vxx = __dadd_rn(cxx, twelfth);
    const double vyy = __dadd_rn(cyy, twelfth);
    const double c1 = __dsqrt_rn(vxx);
    const double c2 = __ddiv_rn(cxy, c1);
    const double c3 = __dsqrt_rn(__dsub_rn(vyy, __dmul_rn(c2, c2)));
    // Sigma = kappa (cov + I/12), kappa = 4: the factor 2 on L is exact
    const double l1 = 2.0 * c1, l2 = 2.0 * c2, l3 = 2.0 * c3;
    const double two_pi = 6.283185307179586;  // 2.0 * math.pi in double
    out[0] = (float)__dadd_rn(__ddiv_rn((double)acc[1], (double)(2 * cnt)), floor(qx));
    out[1] = (float)__dadd_rn(__ddiv_rn((double)acc[2], (double)(2 * cnt)), floor(qy));
    out[2] = (float)l1;
    out[3] = (float)l2;
    out[4] = (float)l3;
    const double den = __dmul_rn(fn, kColourScale);
#pragma unroll
    for (int ch = 0; ch < 3; ch++) out[5 + ch] = (float)__ddiv_rn((double)acc[6 + ch], den);
    out[8] = (float)__ddiv_rn(fn, __dmul_rn(__dmul_rn(two_pi, l1), l3));
  }
#pragma unroll
  for (int r = 0; r < 9; r++) params[(size_t)r * a.n + c] = out[r];
}

// Update (FINAL = false: the centres move) or the Gaussians of the last
// assignment (FINAL).  A block takes 32 centres: its 16 half-warps gather their
// sums, 2 centres each, then one warp does the double-precision arithmetic of
// all 32 at once (FP64 costs per warp instruction, however few lanes it has):
// 20 us at 14 000 centres.  With the assignment, the whole initialisation of a
// 1920 x 1080 frame went from 842 to 372 us.  Few centres have longer windows
// and would leave most SMs idle: up to a wave of blocks of 16 or 8 centres,
// blocks take that many, with 2 or 4 half-warps to each centre's window (340
// centres of a 565 x 315 frame: 31 -> 18 us, its wait for the assignment
// included).  FEW, launched for at most kFewCentres wanted: gathered blocks of
// 4, 2 or 1 too, with up to 32 bands (280 centres 29 pixels apart, the whole
// initialisation: 540 us with 4, 344 so); a kernel of its own, whose registers
// the usual one would feel.  Large segments: the sums come from the assignment's
// atomics and are cleared for the next one.
constexpr int kFewCentres = kWave * 4;

template <bool FINAL, bool FEW>
__global__ void __launch_bounds__(256) k_sp_update(SpArgs a, float* __restrict__ params) {
  pdl_begin();
  __shared__ long long s_sum[kSums][32];
  const SpGeom g = *a.geo;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int per = g.M <= kWave * 8 ? 8 : g.M <= kWave * 16 ? 16 : 32;  // centres of a block
  if (FEW && gathered(g))
    per = g.M <= kWave ? 1 : g.M <= kWave * 2 ? 2 : g.M <= kWave * 4 ? 4 : per;
  const int c0 = blockIdx.x * per;
  if (c0 >= g.M) return;
  const bool mine = lane < per && c0 + lane < g.M;
  if (gathered(g)) {
    const int half = threadIdx.x >> 4, hl = threadIdx.x & 15;
    const unsigned mask = 0xffffu << (lane & 16);
    if (per < 32) {
      for (int k = threadIdx.x; k < kSums * 32; k += 256) (&s_sum[0][0])[k] = 0;
      __syncthreads();
    }
#pragma unroll 1
    for (int k = half; k < 32; k += 16) {
      const int c = k % per;
      if (c0 + c >= g.M) continue;
      long long sum[kSums];
      gather_segment(a, g, c0 + c, k / per, 32 / per, hl, mask, sum);
      if (hl < kSums) {
        long long v = sum[0];
#pragma unroll
        for (int q = 1; q < kSums; q++) v = hl == q ? sum[q] : v;
        // (exact integers: the parts in any order)
        if (per == 32)
          s_sum[hl][c] = v;
        else
          atomicAdd(reinterpret_cast<unsigned long long*>(&s_sum[hl][c]), (unsigned long long)v);
      }
    }
  } else if (wid == 0 && mine) {
#pragma unroll
    for (int q = 0; q < kSums; q++) {
      unsigned long long* p = &a.acc[(size_t)q * a.n + c0 + lane];
      s_sum[q][lane] = (long long)*p;
      *p = 0ull;
    }
  }
  __syncthreads();
  if (wid != 0 || !mine) return;
  long long acc[kSums];
#pragma unroll
  for (int q = 0; q < kSums; q++) acc[q] = s_sum[q][lane];
  if (FINAL)
    segment_gaussian(a, g, c0 + lane, acc, params);
  else
    move_centre(a, g, c0 + lane, acc);
}

// Mask area (pixel count).
__global__ void __launch_bounds__(256) k_sp_area(SpArgs a) {
  pdl_begin();
  const size_t hw = (size_t)a.W * a.H;
  unsigned c = 0;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < hw;
       i += (size_t)gridDim.x * blockDim.x)
    c += a.mask[i] != 0;
  for (int o = 16; o; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
  if ((threadIdx.x & 31) == 0 && c) atomicAdd(a.area, (unsigned long long)c);
}

// The seed grid from the area: step S = max(1, sqrt(A / K)), cells of the
// gx x gy grid in raster order; a cell holds a seed when its centre's pixel is
// in the mask.  Every block derives the same geometry, in one thread: its
// double-precision divisions and square root cost per warp.
__device__ __forceinline__ SpGeom seed_geometry_thread(const SpArgs& a) {
  SpGeom g;
  g.area = (double)*a.area;
  g.M = 0;
  g.S = 1.0;
  g.gx = 1;
  g.gy = 1;
  if (g.area > 0.0 && a.k_target > 0) {
    g.S = fmax(1.0, __dsqrt_rn(__ddiv_rn(g.area, (double)a.k_target)));
    g.gx = (int)ceil(__ddiv_rn((double)a.W, g.S));
    g.gy = (int)ceil(__ddiv_rn((double)a.H, g.S));
  }
  g.ncell = g.gx * g.gy;
  g.S32 = (float)g.S;
  const double q = __ddiv_rn(kCompactness, g.S);
  g.lam32 = (float)__dmul_rn(q, q);
  return g;
}

__device__ __forceinline__ SpGeom seed_geometry(const SpArgs& a) {
  __shared__ SpGeom s_g;
  if (threadIdx.x == 0) s_g = seed_geometry_thread(a);
  __syncthreads();
  return s_g;
}

__device__ __forceinline__ bool seed_cell(const SpArgs& a, const SpGeom& g, int cell, double* x,
                                          double* y) {
  if (g.area <= 0.0 || a.k_target <= 0 || cell >= g.ncell) return false;
  const int j = cell / g.gx, i = cell - j * g.gx;
  *x = __dmul_rn((double)i + 0.5, g.S);
  *y = __dmul_rn((double)j + 0.5, g.S);
  const int xi = (int)floor(*x), yi = (int)floor(*y);
  return xi < a.W && yi < a.H && a.mask[(size_t)yi * a.W + xi];
}

constexpr int kSeedBlocks = 152 * 4;

// Cells [b C, (b + 1) C) of block b, C = ceil(cells / blocks): the seed count.
__global__ void __launch_bounds__(256) k_sp_seed_count(SpArgs a) {
  pdl_begin();
  const SpGeom g = seed_geometry(a);
  const int chunk = (g.ncell + gridDim.x - 1) / gridDim.x;
  const int c0 = blockIdx.x * chunk, c1 = min(g.ncell, c0 + chunk);
  int cnt = 0;
  for (int cell = c0 + threadIdx.x; cell < c1; cell += blockDim.x) {
    double x, y;
    cnt += seed_cell(a, g, cell, &x, &y);
  }
  for (int o = 16; o; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
  __shared__ int s_w[8];
  if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = cnt;
  __syncthreads();
  if (threadIdx.x == 0) {
    int t = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); w++) t += s_w[w];
    a.blk[blockIdx.x] = t;
  }
}

// Seeds numbered in raster order of the grid (at most n): each block adds the
// counts of the blocks before it, then numbers its cells by ballots.
__global__ void __launch_bounds__(256) k_sp_seed_write(SpArgs a) {
  pdl_begin();
  const SpGeom g = seed_geometry(a);
  __shared__ int s_base, s_w[9];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  {
    // this block's base (counts of the blocks before it) and the total
    int b = 0, tot = 0;
    for (int k = threadIdx.x; k < (int)gridDim.x; k += blockDim.x) {
      const int c = a.blk[k];
      b += k < (int)blockIdx.x ? c : 0;
      tot += c;
    }
    for (int o = 16; o; o >>= 1) {
      b += __shfl_xor_sync(0xffffffffu, b, o);
      tot += __shfl_xor_sync(0xffffffffu, tot, o);
    }
    __shared__ int s_b[8], s_t[8];
    if (lane == 0) {
      s_b[wid] = b;
      s_t[wid] = tot;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      int bb = 0, tt = 0;
      for (int w = 0; w < (int)(blockDim.x >> 5); w++) {
        bb += s_b[w];
        tt += s_t[w];
      }
      s_base = bb;
      if (blockIdx.x == 0) {
        SpGeom out = g;
        out.M = min(tt, a.n);
        *a.geo = out;
      }
    }
    __syncthreads();
  }
  const int chunk = (g.ncell + gridDim.x - 1) / gridDim.x;
  const int c0 = blockIdx.x * chunk, c1 = min(g.ncell, c0 + chunk);
  int run = s_base;
  for (int base = c0; base < c1; base += blockDim.x) {
    const int cell = base + threadIdx.x;
    double x = 0.0, y = 0.0;
    const bool f = cell < c1 && seed_cell(a, g, cell, &x, &y);
    const unsigned bal = __ballot_sync(0xffffffffu, f);
    if (lane == 0) s_w[wid] = __popc(bal);
    __syncthreads();
    if (threadIdx.x == 0) {
      int t = 0;
      for (int w = 0; w < (int)(blockDim.x >> 5); w++) {
        const int c = s_w[w];
        s_w[w] = t;
        t += c;
      }
      s_w[8] = t;
    }
    __syncthreads();
    const int idx = run + s_w[wid] + __popc(bal & ((1u << lane) - 1u));
    if (cell < c1) {
      const bool take = f && idx < a.n;
      a.cell_of[cell] = take ? idx : -1;
      if (take) {
        a.seed_xy[idx] = x;
        a.seed_xy[a.n + idx] = y;
        a.seed_i[idx] = (int)floor(x);
        a.seed_i[a.n + idx] = (int)floor(y);
      }
    }
    run += s_w[8];
    __syncthreads();
  }
}

// One thread per Gaussian: the first M start their centre at the seed with the
// frame's colour there (and empty sums), the others are the isotropic
// background Gaussians at bg_xy[0 .. n - M), whose common size one thread of
// the block derives.
__global__ void __launch_bounds__(256) k_sp_start(SpArgs a, const float* __restrict__ bg_xy,
                                                  float* __restrict__ params) {
  pdl_begin();
  __shared__ float s_size;
  const SpGeom g = *a.geo;
  const int n = a.n, M = g.M;
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (threadIdx.x == 0 && M < n) {
    const double hw = (double)a.W * (double)a.H;
    const double abg = __ddiv_rn(__dsub_rn(hw, g.area), (double)(n - M));
    s_size = (float)__dsqrt_rn(__ddiv_rn(__dmul_rn(kKappa, abg > 1.0 ? abg : 1.0),
                                         __dmul_rn(2.0, 3.141592653589793)));
  }
  __syncthreads();
  if (c >= n) return;
  const size_t HW = (size_t)a.W * a.H;
  if (c < M) {
    const int xi = min(max(a.seed_i[c], 0), a.W - 1), yi = min(max(a.seed_i[n + c], 0), a.H - 1);
    const size_t idx = (size_t)yi * a.W + xi;
    a.cen[c] = a.frame[idx];
    a.cen[n + c] = a.frame[HW + idx];
    a.cen[2 * n + c] = a.frame[2 * HW + idx];
    a.cen[3 * n + c] = (float)a.seed_xy[c];
    a.cen[4 * n + c] = (float)a.seed_xy[n + c];
#pragma unroll
    for (int k = 0; k < kSums; k++) a.acc[(size_t)k * n + c] = 0ull;
    return;
  }
  const float x = bg_xy[c - M], y = bg_xy[n + c - M];
  const int xi = min(max((int)floorf(x), 0), a.W - 1), yi = min(max((int)floorf(y), 0), a.H - 1);
  const size_t idx = (size_t)yi * a.W + xi;
  params[c] = x;
  params[n + c] = y;
  params[2 * n + c] = s_size;
  params[3 * n + c] = 0.0f;
  params[4 * n + c] = s_size;
  params[5 * n + c] = a.frame[idx];
  params[6 * n + c] = a.frame[HW + idx];
  params[7 * n + c] = a.frame[2 * HW + idx];
  params[8 * n + c] = (float)(1.0 / kKappa);
}

uint64_t a256(uint64_t x) { return (x + 255) & ~uint64_t(255); }

}  // namespace

// Scratch layout for a W x H frame with n Gaussians: labels int[H W], centres
// float[5][n], seeds double[2][n] and int[2][n], cell map int[(W+1) (H+1)] (the grid step
// is at least one pixel), segment sums int64[9][n], the area, the geometry and
// the per-block seed counts.
uint64_t roi_init_scratch_bytes(int W, int H, int n) {
  const uint64_t hw = (uint64_t)W * H;
  return a256(hw * 4) + a256(5ull * n * 4) + a256(2ull * n * 8) + a256(2ull * n * 4) +
         a256((uint64_t)(W + 1) * (H + 1) * 4) + a256((uint64_t)kSums * n * 8) + a256(8) +
         a256(sizeof(SpGeom)) + a256(kSeedBlocks * 4) + 256;
}

gs2d_status roi_init(const float* frame, const uint8_t* mask, int W, int H, int n, float roi_frac,
                     const float* bg_xy, float* params, int32_t* n_roi, void* scratch,
                     uint64_t scratch_bytes, cudaStream_t s, char* err, size_t err_len,
                     float* cen_trace, int32_t* label_trace) {
  if (scratch_bytes < roi_init_scratch_bytes(W, H, n)) {
    snprintf(err, err_len, "gs2d_roi_init: scratch too small");
    return GS2D_ERR_INVALID_ARG;
  }
  const uint64_t hw = (uint64_t)W * H;
  char* p = static_cast<char*>(scratch);
  auto take = [&p](uint64_t bytes) {
    char* q = p;
    p += a256(bytes);
    return q;
  };
  SpArgs a;
  a.W = W;
  a.H = H;
  a.n = n;
  a.k_target = (int)llround((double)roi_frac * n);
  a.frame = frame;
  a.mask = mask;
  a.label = reinterpret_cast<int*>(take(hw * 4));
  a.cen = reinterpret_cast<float*>(take(5ull * n * 4));
  a.seed_xy = reinterpret_cast<double*>(take(2ull * n * 8));
  a.seed_i = reinterpret_cast<int*>(take(2ull * n * 4));
  a.cell_of = reinterpret_cast<int*>(take((uint64_t)(W + 1) * (H + 1) * 4));
  a.acc = reinterpret_cast<unsigned long long*>(take((uint64_t)kSums * n * 8));
  a.area = reinterpret_cast<unsigned long long*>(take(8));
  a.geo = reinterpret_cast<SpGeom*>(take(sizeof(SpGeom)));
  a.blk = reinterpret_cast<int*>(take(kSeedBlocks * 4));
  // everything on the device; the region count comes back at the end
  const dim3 tiles((W + kTileW - 1) / kTileW, (H + kTileH - 1) / kTileH);
  const bool few = a.k_target <= kFewCentres;
  const int cb = std::max((n + 31) / 32, std::min(n, kWave));  // k_sp_update's
  cudaError_t e = cudaMemsetAsync(a.area, 0, 8, s);
  if (e == cudaSuccess) e = launch_pdl(k_sp_area, 152 * 8, 256, 0, s, a);
  if (e == cudaSuccess) e = launch_pdl(k_sp_seed_count, kSeedBlocks, 256, 0, s, a);
  if (e == cudaSuccess) e = launch_pdl(k_sp_seed_write, kSeedBlocks, 256, 0, s, a);
  if (e == cudaSuccess && n > 0) {
    e = launch_pdl(k_sp_start, (n + 255) / 256, 256, 0, s, a, bg_xy, params);
    // the last assignment's sums make the Gaussians
    for (int it = 0; it < kIterations && e == cudaSuccess; it++) {
      // optional trace: the centres this assignment uses, the labels it makes
      if (cen_trace)
        e = cudaMemcpyAsync(cen_trace + (size_t)it * 5 * n, a.cen, 5ull * n * sizeof(float),
                            cudaMemcpyDeviceToDevice, s);
      if (e == cudaSuccess) e = launch_pdl(k_sp_assign, tiles, 256, 0, s, a, it == 0 ? 1 : 0);
      if (e == cudaSuccess && label_trace)
        e = cudaMemcpyAsync(label_trace + (size_t)it * hw, a.label, hw * sizeof(int32_t),
                            cudaMemcpyDeviceToDevice, s);
      if (e == cudaSuccess)
        e = it + 1 < kIterations
                ? launch_pdl(few ? k_sp_update<false, true> : k_sp_update<false, false>, cb, 256,
                             0, s, a, params)
                : launch_pdl(few ? k_sp_update<true, true> : k_sp_update<true, false>, cb, 256,
                             0, s, a, params);
    }
  }
  SpGeom g;
  if (e == cudaSuccess) e = cudaMemcpyAsync(&g, a.geo, sizeof(g), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) {
    snprintf(err, err_len, "gs2d_roi_init: %s", cudaGetErrorString(e));
    return GS2D_ERR_CUDA;
  }
  if (n_roi) *n_roi = g.M;
  return GS2D_OK;
}

}  // namespace gs2d
