// Forward and backward rasterization of the accumulated-sum blend (Eq. 2),
// templated on the tile edge T (8, 16, 32) and the shared-memory batch S
// (Gaussians staged at a time: 32, 64, 128).  Included by render_t8.cu,
// render_t16.cu and render_t32.cu, one instantiation set each.
//
// Work order: gs2d_bin_sort leaves the tiles in the order section, longest
// list first, so that the longest tiles do not end up in the tail of the
// launch.  Two launch forms (gs2d_config::launch):
//  * persistent: one wave of thread blocks (resident blocks per SM x SMs)
//    takes tiles from a queue (a ticket counter in the workspace header); a
//    block takes its next ticket while it renders the current tile, so the
//    atomic's latency is hidden; the last block to leave the queue resets the
//    counter for the next launch;
//  * grid: one block per tile, block b rendering the b-th tile of the order;
//    the hardware block scheduler hands them out in that order.
// A tile of any clip of a batch is processed in that clip's frame (size,
// image offset, loss scale).
//
// Each tile's sorted list [start, end) is staged into shared memory in batches
// of S Gaussians; the staging thread also computes each Gaussian's pixel box
// inside the tile, the rows of it that the ellipse can reach (cut_rows), a mask
// of the warps those rows touch, and for the backward pass the slot where it
// writes this (tile, Gaussian) pair's sums.
//
// sigma in Cholesky form (Eq. 1): with s = sqrt(log2(e)/2) and tile-local
// offsets dx = px - mu_x, dy = py - mu_y,
//   u1 = a1 dx,  u2 = a2 dy + kappa dx  (a1 = s / l1, a2 = s / l3,
//   kappa = -(l2 / l3) a1),  q = u1^2 + u2^2 = sigma log2(e),
//   contribution c' 2^-q if q <= tau log2(e).
// For a fixed column, u1 is constant and u2 advances by a2 per row, so each
// further pixel of that column costs one FADD (u2) and one FFMA (q).
//
// Forward: thread <-> one column x R-row strip (R = 2 for T = 8, else 4);
// a warp covers a band of rows.  After each batch is staged every warp
// compacts (by ballot) the batch's Gaussians whose box meets its band into
// its own ascending list; each list entry carries the Gaussian's staged
// position and the row term a2 dy of the band's first row, so a thread's
// setup per Gaussian is four FP32 operations.  Accumulation is in ascending
// Gaussian index (the list order).
//
// Backward: the blend is recomputed from the saved lists (no per-pixel state
// is stored by the forward pass).  A group of T lanes takes one Gaussian and
// lays itself over the Gaussian's box inside the tile: box columns rounded up
// to a power of two c, T / c rows per step, each lane one column and every
// (T / c)-th row of the box, but for rows that the ellipse does not reach (u2
// still advances over them by the same additions, so that the cut-off falls on
// the same pixels as without the cut).  Per lane it keeps
// sum g e (3), sum S, sum S u2, sum S u2^2 with S = (g . c') e; the moments
// in u1 follow by multiplying with the lane's constant u1.  The group reduces
// the eight sums with a transposing shuffle tree and writes one 32-byte
// record to the pair's slot.  k_reduce_chain sums each Gaussian's slots in a
// fixed order (deterministic, no float atomics) and applies the chain rule to
// (mu, l, c, w).
#pragma once

#include <limits.h>

#include "gs2d_internal.cuh"

namespace gs2d {

// Rows per thread of the usual kernels: 2, 4, 4.
template <int T>
constexpr int kRows = T == 8 ? 2 : 4;

template <int T, int R_>
struct TileGeom {
  static constexpr int R = R_;              // rows per thread: kRows<T>, or 1 (few tiles)
  static constexpr int NT = T * T / R;      // threads per block: 32, 64, 256 (R = 1: 256, 1024)
  static constexpr int NW = NT / 32;        // warps: 1, 2, 8 (R = 1: 8, 32)
  static constexpr int RW = 32 / T * R;     // rows per warp band: 8, 8, 4 (R = 1: 2, 1)
  static constexpr int GPW = 32 / T;        // Gaussians per warp in the backward pass
  static constexpr int Q = T / 8;           // lanes per reduced value
};

template <int S>
struct TileSmem {
  float4 fa[S];      // (mu_x - ox, a1, kappa, a2): tile-local
  float4 fb[S];      // (tau2, c'_r, c'_g, c'_b)
  float my[S];       // mu_y - oy
  int4 bb[S];        // local box (x0, y0, (x1 - x0) | log2 c << 8 | skip << 16, y1): c the columns
                     // rounded up to a power of two, skip and y1 the rows the ellipse reaches
                     // (y0 + skip ... y1); negative third word when none
  int slot[S];       // partial slot of the pair
  uint32_t wmask[S]; // bit w: box touches the rows of warp w
  int next;          // the backward's next Gaussian (warps take them in turn)
};

// The tile a block works on, in its clip's frame.
struct TileFrame {
  int tile;       // global tile id
  int W, H;       // clip size
  int tx, ty;     // tile column and row in the clip
  int ox, oy;     // pixel origin of the tile in the clip
  int64_t pix;    // first float of the clip's image
  int2 rg;        // list range
};

template <int T>
__device__ __forceinline__ TileFrame tile_frame(const RenderArgs& a, int tile) {
  const gs2d_clip cl = clip_of_tile(a.clips, tile);
  const int lt = tile - cl.tile_off;
  const int ty = lt / cl.tiles_x, tx = lt - ty * cl.tiles_x;
  TileFrame f;
  f.tile = tile;
  f.W = cl.width;
  f.H = cl.height;
  f.tx = tx;
  f.ty = ty;
  f.ox = tx * T;
  f.oy = ty * T;
  f.pix = cl.pix_off;
  f.rg = a.ranges[tile];
  return f;
}

// Cuts the rows [lo, hi] (tile-local pixels) of a Gaussian's box to those its
// cut-off ellipse can reach in the columns [x0, x1]: with dx the distance from
// the mean along x, q = (a1 dx)^2 + (dy + s dx)^2 / ia2^2, so dy lies within
// sqrt(tau2 - (a1 dx)^2) ia2 of -s dx.  The bound takes the nearest dx for the
// width and the extremes for the shift, widened so that FP32 rounding of it
// (approximate square root and reciprocal included) or of the kernels' q loses
// no pixel: 0.2 % on tau2, 0.1 % and 0.0039 px on the width, 1e-6 of the shift.
// A NaN cuts nothing.  About a tenth of the (pixel, Gaussian) pairs of a
// conferencing fit lie outside.  At 1080p, 20 000 Gaussians, tile 32, together
// with the backward's row loop below: fused call 78.2 -> 74.5 us, backward 53
// -> 51.5, forward 24.8 -> 23.0 (tile 16: 92.3 -> 90.7, forward 23.8 -> 21.7).
__device__ __forceinline__ void cut_rows(float my, float mx, float x0, float x1, float a1,
                                         float ia2, float s, float tau2, float& lo, float& hi) {
  const float d0 = x0 + 0.5f - mx, d1 = x1 + 0.5f - mx;
  const float near = a1 * fmaxf(fmaxf(d0, -d1), 0.0f);
  const float w2 = 1.002f * tau2 - 0.998f * near * near;
  if (w2 < 0.0f) {
    hi = -1.0f;
    return;
  }
  const float c0 = -s * d0, c1 = -s * d1;
  float root;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(root) : "f"(w2));
  const float half = fmaf(1.001f * root, ia2, 0.0039f) +
                     1e-6f * (fabsf(my) + fabsf(c0) + fabsf(c1));
  lo = fmaxf(lo, ceilf(my + fminf(c0, c1) - half - 0.5f));
  hi = fminf(hi, floorf(my + fmaxf(c0, c1) + half - 0.5f));
}

// Stage entries [b, b + cnt) of the tile's list (cnt <= S); BWD: with what
// only the backward needs (columns, slots).
template <int T, int S, int R, bool BWD>
__device__ __forceinline__ void stage_batch(TileSmem<S>& sm, const RenderArgs& a,
                                            const TileFrame& f, int b, int cnt) {
  using G = TileGeom<T, R>;
  if (threadIdx.x == 0) sm.next = 0;
  for (int k = threadIdx.x; k < cnt; k += G::NT) {
    const int g = (int)a.list[b + k];
    const float4 r0 = a.rec[g], r1 = a.rec[a.n + g], r2 = a.rec[2 * a.n + g];
    int4 rc = make_int4(0, 1, 0, 0);
    int off = 0;
    if (BWD) {
      rc = a.lrect[g];
      off = a.offs[g];
    }
    const float ox = (float)f.ox, oy = (float)f.oy;
    const float mx = r0.x - ox, my = r0.y - oy;
    // pixel lx contributes only if |ox + lx + 0.5 - mu_x| <= hx
    float fx0 = ceilf(r0.x - r2.y - 0.5f - ox), fx1 = floorf(r0.x + r2.y - 0.5f - ox);
    float fy0 = ceilf(r0.y - r2.z - 0.5f - oy), fy1 = floorf(r0.y + r2.z - 0.5f - oy);
    fx0 = fmaxf(fx0, 0.0f);
    fy0 = fmaxf(fy0, 0.0f);
    fx1 = fminf(fx1, fminf((float)(T - 1), (float)(f.W - 1) - ox));
    fy1 = fminf(fy1, fminf((float)(T - 1), (float)(f.H - 1) - oy));
    int4 bb = make_int4(0, 0, INT_MIN, 0);
    uint32_t wm = 0;
    if (fx0 <= fx1 && fy0 <= fy1) {
      // the rows of the ellipse's part inside the tile's columns, which at the
      // ellipse's rim are fewer than its box's: q = (a1 dx)^2 + (a2 (dy +
      // (kappa / a2) dx))^2
      const float a2 = r0.w;
      float ia2;  // (NaN past 2^126, whose reciprocal would be flushed to zero)
      asm("rcp.approx.f32 %0, %1;" : "=f"(ia2) : "f"(a2));
      if (!(fabsf(a2) < 8.0e37f)) ia2 = __int_as_float(0x7fc00000);
      float cy0 = fy0, cy1 = fy1;
      cut_rows(my, mx, fx0, fx1, r0.z, fabsf(ia2), r1.x * ia2, r1.y, cy0, cy1);
      if (cy0 <= cy1) {
        const int x0 = (int)fx0, bw = (int)fx1 - x0;  // columns - 1
        const int y0 = (int)fy0, c0 = (int)cy0, c1 = (int)cy1;
        bb = make_int4(x0, y0, bw | (bw == 0 ? 0 : 32 - __clz(bw)) << 8 | (c0 - y0) << 16, c1);
        const int w0 = c0 / G::RW, w1 = c1 / G::RW;
        wm = ((2u << w1) - 1u) & ~((1u << w0) - 1u);
      }
    }
    sm.fa[k] = make_float4(mx, r0.z, r1.x, r0.w);
    sm.fb[k] = make_float4(r1.y, r1.z, r1.w, r2.x);
    sm.my[k] = my;
    sm.wmask[k] = wm;
    if (BWD) {
      sm.bb[k] = bb;
      // position of this tile inside the Gaussian's listed rectangle
      const int rel = f.tile - rc.x, row = rel / rc.y;
      sm.slot[k] = off + row * rc.z + (rel - row * rc.y);
    }
  }
}

// Shared memory by 32-bit address: the backward's row loop is bound by
// instruction issue, and address arithmetic on generic 64-bit pointers took
// several instructions per load.  volatile: ordered with the barriers around them.
__device__ __forceinline__ uint32_t shared_addr(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ float4 shared_f4(uint32_t a) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(a));
  return v;
}

// One entry of a warp's list of staged Gaussians: the row term a2 (y - mu_y)
// at the first row of the warp's band (float bits) and the byte offset of
// the Gaussian in the staged arrays.
struct WarpEntry {
  uint32_t t;
  uint32_t off;
};

// Forward accumulation over the warp's list for this thread's column
// (tile-local centre pxl) and rows; drow = rows between the band's first row
// and this thread's first row.
template <int T, int S>
__device__ __forceinline__ void fwd_batch(const TileSmem<S>& sm, const WarpEntry* __restrict__ wl,
                                          int wn, float pxl, float drow,
                                          float (&acc)[kRows<T>][3]) {
  constexpr int R = kRows<T>;
  const char* fa_base = reinterpret_cast<const char*>(sm.fa);
  const char* fb_base = reinterpret_cast<const char*>(sm.fb);
  for (int i = 0; i < wn; i++) {
    const WarpEntry we = wl[i];
    const float4 fa = *reinterpret_cast<const float4*>(fa_base + we.off);
    const float4 fb = *reinterpret_cast<const float4*>(fb_base + we.off);
    const float dx = pxl - fa.x;
    const float u1 = fa.y * dx;
    const float u1sq = u1 * u1;
    float u2 = fmaf(fa.z, dx, __uint_as_float(we.t));
    if constexpr (T != 32) u2 = fmaf(fa.w, drow, u2);
#pragma unroll
    for (int r = 0; r < R; r++) {
      if (r) u2 += fa.w;
      const float q = fmaf(u2, u2, u1sq);
      if (q <= fb.x) {
        const float e = ex2_approx(-q);
        acc[r][0] = fmaf(fb.y, e, acc[r][0]);
        acc[r][1] = fmaf(fb.z, e, acc[r][1]);
        acc[r][2] = fmaf(fb.w, e, acc[r][2]);
      }
    }
  }
}

// Sum of eight per-lane values over each aligned group of G lanes (G = 8, 16
// or 32).  Three transposing levels (distances G/2, G/4, G/8) halve the values
// each lane carries; plain levels finish the sum.  Afterwards lane j of the
// group holds the total of value j / (G / 8) (lanes with j % (G / 8) == 0
// hold distinct values).
template <int G>
__device__ __forceinline__ float group_transpose_sum(const float (&v)[8], int j) {
  const bool b1 = j & (G / 2), b2 = j & (G / 4), b3 = j & (G / 8);
  float w[4];
#pragma unroll
  for (int k = 0; k < 4; k++) {
    const float send = b1 ? v[k] : v[k + 4];
    const float keep = b1 ? v[k + 4] : v[k];
    w[k] = keep + __shfl_xor_sync(0xffffffffu, send, G / 2);
  }
  float x[2];
#pragma unroll
  for (int k = 0; k < 2; k++) {
    const float send = b2 ? w[k] : w[k + 2];
    const float keep = b2 ? w[k + 2] : w[k];
    x[k] = keep + __shfl_xor_sync(0xffffffffu, send, G / 4);
  }
  float y = (b3 ? x[1] : x[0]) + __shfl_xor_sync(0xffffffffu, b3 ? x[0] : x[1], G / 8);
#pragma unroll
  for (int d = G / 16; d >= 1; d >>= 1) y += __shfl_xor_sync(0xffffffffu, y, d);
  return y;
}

// Backward over staged Gaussians [0, cnt) (entries batch[0 .. cnt) of the
// tile's list); g (dL/dC) of the tile at shared address s_g.  Each pair's eight
// sums go to its slot of `partial`, or with `acc` (GS2D_REDUCE_ATOMIC) are added
// to the Gaussian's sums by float atomics (pairs whose box misses the tile add
// nothing).
template <int T, int S>
__device__ __forceinline__ void bwd_batch(TileSmem<S>& sm, uint32_t s_g, int cnt,
                                          const RenderArgs& a, int b) {
  using G = TileGeom<T, kRows<T>>;  // (the rows per thread play no part here)
  float* __restrict__ partial = a.partial;
  const int lane = threadIdx.x & 31;
  const int h = lane / T, j = lane % T;
  for (;;) {  // warps take the next GPW Gaussians as they finish (balance)
    int base = 0;
    if (lane == 0) base = atomicAdd(&sm.next, G::GPW);
    base = __shfl_sync(0xffffffffu, base, 0);
    if (base >= cnt) break;
    const int gi = base + h;
    // Gaussians whose box misses the tile: a zero record, no reduction
    const int4 bb = gi < cnt ? sm.bb[gi] : make_int4(0, 0, INT_MIN, 0);
    if (__all_sync(0xffffffffu, bb.z < 0)) {
      if (!a.acc && gi < cnt && j < 8) partial[8 * sm.slot[gi] + j] = 0.0f;
      continue;
    }
    float v[8];
#pragma unroll
    for (int k = 0; k < 8; k++) v[k] = 0.0f;
    // lane j: column j % c of the box, rows j / c, + T / c, ...; of these the
    // first `skip` rows of the box are passed over
    constexpr int kLog = T == 8 ? 3 : T == 16 ? 4 : 5;
    const int lc = (bb.z >> 8) & 7;  // log2 c
    const int dcol = j & ((1 << lc) - 1), dy0 = j >> lc;
    const int pass = max(0, ((bb.z >> 16) - dy0 + (T >> lc) - 1) >> (kLog - lc));
    const int y0 = bb.y + dy0, y1 = y0 + (pass << (kLog - lc));
    if (bb.z >= 0 && dcol <= (bb.z & 255) && y1 <= bb.w) {
      const float4 fa = sm.fa[gi], fb = sm.fb[gi];
      const int col = bb.x + dcol;
      const float dx = ((float)col + 0.5f) - fa.x;
      const float u1 = fa.y * dx;
      const float u1sq = u1 * u1;
      const float ustep = fa.w * (float)(T >> lc);
      float u2 = fmaf(fa.w, ((float)y0 + 0.5f) - sm.my[gi], fa.z * dx);
      float ge0 = 0.f, ge1 = 0.f, ge2 = 0.f, ss = 0.f, s2 = 0.f, s22 = 0.f;
      // (u2 by the same additions from the box's first row, whatever is passed
      // over: the cut-off falls on the same pixels)
      for (int k = pass; k > 0; k--) u2 += ustep;
      uint32_t ga = s_g + (uint32_t)(y1 * T + col) * 16u;
      const uint32_t gstep = (uint32_t)(T * 16 * T) >> lc;
      // branch-free: a pixel outside the cut-off adds exact zeros
      const auto row = [&]() {
        const float q = fmaf(u2, u2, u1sq);
        const float e = q <= fb.x ? ex2_approx(-q) : 0.0f;
        const float4 g = shared_f4(ga);
        ge0 = fmaf(g.x, e, ge0);
        ge1 = fmaf(g.y, e, ge1);
        ge2 = fmaf(g.z, e, ge2);
        const float Sv = fmaf(g.x, fb.y, fmaf(g.y, fb.z, g.z * fb.w)) * e;
        const float su2 = Sv * u2;
        ss += Sv;
        s2 += su2;
        s22 = fmaf(su2, u2, s22);
        ga += gstep;
        u2 += ustep;
      };
      int rows = ((bb.w - y1) >> (kLog - lc)) + 1;
      for (; rows >= 2; rows -= 2) {
        row();
        row();
      }
      if (rows > 0) row();
      const float a1 = u1 * ss;
      v[0] = ge0;
      v[1] = ge1;
      v[2] = ge2;
      v[3] = a1;
      v[4] = s2;
      v[5] = u1 * a1;
      v[6] = u1 * s2;
      v[7] = s22;
    }
    const float tot = group_transpose_sum<T>(v, j);
    if (gi < cnt && (j % G::Q) == 0) {
      if (!a.acc)
        partial[8 * sm.slot[gi] + j / G::Q] = tot;
      else if (bb.z >= 0)
        atomicAdd(&a.acc[(size_t)kPartials * a.list[b + gi] + j / G::Q], tot);
    }
  }
}

// Per-mode shared memory beyond the staged batch.
template <int T, int S, int MODE, int R>
struct ModeSmem {
  static constexpr int kGrad = (MODE == kModeBwd || MODE == kModeL2) ? T * T : 1;
  static constexpr int kList = (MODE == kModeFwd || MODE == kModeL2) && R > 1 ? S : 1;
  static constexpr int kSse = MODE == kModeL2 && R == 1 ? T * T : 1;
  float4 g[kGrad];                          // dL/dC of the tile
  WarpEntry wl[TileGeom<T, R>::NW][kList];  // per-warp lists of the staged batch
  float2 red[TileGeom<T, kRows<T>>::NW];    // loss partials per warp
  float2 sse[kSse];                         // R = 1: squared errors per pixel
  unsigned hits;                       // kModeCount
};

// Warp wid's list of the staged Gaussians [0, cnt) whose box touches its
// rows, in ascending order; returns its length.  pyw: tile-local centre of
// the band's first row.
template <int T, int S>
__device__ __forceinline__ int warp_list(const TileSmem<S>& sm, int cnt, int wid, int lane,
                                         float pyw, WarpEntry* __restrict__ wl) {
  int m = 0;
  for (int base = 0; base < cnt; base += 32) {
    const int k = base + lane;
    const bool on = k < cnt && ((sm.wmask[k] >> wid) & 1u);
    const unsigned bal = __ballot_sync(0xffffffffu, on);
    if (on) {
      WarpEntry e;
      e.t = __float_as_uint(sm.fa[k].w * (pyw - sm.my[k]));
      e.off = (uint32_t)(k * sizeof(float4));
      wl[m + __popc(bal & ((1u << lane) - 1u))] = e;
    }
    m += __popc(bal);
  }
  __syncwarp();
  return m;
}

// The forward pass of the kernels with one row per thread (few tiles): the
// warp walks the staged Gaussians that touch its rows by ballot (ascending
// index, as warp_list leaves them) and every lane evaluates its pixel with
// the roundings of the usual kernels: the row term at the first row of their
// band (t0), one FMA to the thread's strip (drow), then one addition per row
// down the strip (steps of them).  So the image is theirs bit for bit.
template <int T, int S>
__device__ __forceinline__ void fwd_batch_rows(const TileSmem<S>& sm, int cnt, int wid, int lane,
                                               float pxl, float pyw, float drow, int steps,
                                               float (&acc)[3]) {
  for (int base = 0; base < cnt; base += 32) {
    const int k = base + lane;
    const bool on = k < cnt && ((sm.wmask[k] >> wid) & 1u);
    for (unsigned m = __ballot_sync(0xffffffffu, on); m; m &= m - 1) {
      const int j = base + __ffs(m) - 1;
      const float4 fa = sm.fa[j], fb = sm.fb[j];
      const float dx = pxl - fa.x;
      const float u1 = fa.y * dx;
      const float u1sq = u1 * u1;
      float u2 = fmaf(fa.z, dx, fa.w * (pyw - sm.my[j]));
      if constexpr (T != 32) u2 = fmaf(fa.w, drow, u2);
#pragma unroll
      for (int r = 1; r < kRows<T>; r++) u2 = r <= steps ? u2 + fa.w : u2;
      const float q = fmaf(u2, u2, u1sq);
      if (q <= fb.x) {
        const float e = ex2_approx(-q);
        acc[0] = fmaf(fb.y, e, acc[0]);
        acc[1] = fmaf(fb.z, e, acc[1]);
        acc[2] = fmaf(fb.w, e, acc[2]);
      }
    }
  }
}

template <int T, int S, int MODE, int R>
__device__ __forceinline__ void process_tile(const RenderArgs& a, const TileFrame& f,
                                             TileSmem<S>& sm, ModeSmem<T, S, MODE, R>& ms) {
  using G = TileGeom<T, R>;
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  const int x = f.ox + t % T, y0 = f.oy + R * (t / T);
  // tile-local pixel centres of this thread's column and first row
  const float pxl = (float)(t % T) + 0.5f, pyl = (float)(R * (t / T)) + 0.5f;
  const size_t HW = (size_t)f.W * f.H;
  const int2 rg = f.rg;

  if constexpr (MODE == kModeBwd) {
#pragma unroll
    for (int r = 0; r < R; r++) {
      float4 g = make_float4(0.f, 0.f, 0.f, 0.f);
      if (x < f.W && y0 + r < f.H) {
        const size_t o = f.pix + (size_t)(y0 + r) * f.W + x;
        g = make_float4(a.dimg[o], a.dimg[HW + o], a.dimg[2 * HW + o], 0.f);
      }
      ms.g[(R * (t / T) + r) * T + t % T] = g;
    }
    for (int b = rg.x; b < rg.y; b += S) {
      const int cnt = min(S, rg.y - b);
      __syncthreads();
      stage_batch<T, S, R, MODE == kModeBwd || MODE == kModeL2>(sm, a, f, b, cnt);
      __syncthreads();
      bwd_batch<T, S>(sm, shared_addr(ms.g), cnt, a, b);
    }
    return;
  }

  if constexpr (MODE == kModeSelect) {
    // Gaussians that contribute to a changed pixel of this tile (the
    // renderer's predicate); a pixel changed if max_c |ref - frame| > threshold
    bool changed[R];
    bool any = false;
#pragma unroll
    for (int r = 0; r < R; r++) {
      changed[r] = false;
      if (x < f.W && y0 + r < f.H) {
        const size_t o = f.pix + (size_t)(y0 + r) * f.W + x;
        float d = fabsf(a.ref[o] - a.frame[o]);
        d = fmaxf(d, fabsf(a.ref[HW + o] - a.frame[HW + o]));
        d = fmaxf(d, fabsf(a.ref[2 * HW + o] - a.frame[2 * HW + o]));
        changed[r] = d > a.threshold;
        any |= changed[r];
      }
    }
    if (!__syncthreads_or(any)) return;  // the whole tile unchanged
    for (int b = rg.x; b < rg.y; b += S) {
      const int cnt = min(S, rg.y - b);
      __syncthreads();
      stage_batch<T, S, R, MODE == kModeBwd || MODE == kModeL2>(sm, a, f, b, cnt);
      __syncthreads();
      if (!any) continue;
      for (int j = 0; j < cnt; j++) {
        const float4 fa = sm.fa[j];
        const float dx = pxl - fa.x, dy = pyl - sm.my[j], tau2 = sm.fb[j].x;
        const float u1 = fa.y * dx;
        bool hit = false;
#pragma unroll
        for (int r = 0; r < R; r++) {
          const float u2 = fmaf(fa.w, dy + (float)r, fa.z * dx);
          hit |= changed[r] && fmaf(u2, u2, u1 * u1) <= tau2;
        }
        if (hit) a.selected[a.list[b + j]] = 1;  // every writer stores 1
      }
    }
    return;
  }

  if constexpr (MODE == kModeCount) {
    if (t == 0) ms.hits = 0;
    unsigned hits = 0;
    for (int b = rg.x; b < rg.y; b += S) {
      const int cnt = min(S, rg.y - b);
      __syncthreads();
      stage_batch<T, S, R, MODE == kModeBwd || MODE == kModeL2>(sm, a, f, b, cnt);
      __syncthreads();
      for (int j = 0; j < cnt && x < f.W; j++) {
        const float4 fa = sm.fa[j];
        const float dx = pxl - fa.x, dy = pyl - sm.my[j], tau2 = sm.fb[j].x;
        const float u1 = fa.y * dx;
        for (int r = 0; r < R; r++) {
          const float u2 = fmaf(fa.w, dy + (float)r, fa.z * dx);
          hits += (y0 + r < f.H) && fmaf(u2, u2, u1 * u1) <= tau2;
        }
      }
    }
    __syncthreads();
    atomicAdd(&ms.hits, hits);
    __syncthreads();
    if (t == 0) {
      const int vw = min(T, f.W - f.ox), vh = min(T, f.H - f.oy);
      atomicAdd(&a.hdr->pairs, (unsigned long long)(vw * vh) * (unsigned long long)(rg.y - rg.x));
      atomicAdd(&a.hdr->hits, (unsigned long long)ms.hits);
    }
    return;
  }

  if constexpr (MODE == kModeFwd || MODE == kModeL2) {
    // forward (kModeFwd, kModeL2)
    float acc[R][3];
#pragma unroll
    for (int r = 0; r < R; r++) acc[r][0] = acc[r][1] = acc[r][2] = 0.0f;
    int staged = -1;
    for (int b = rg.x; b < rg.y; b += S) {
      const int cnt = min(S, rg.y - b);
      __syncthreads();
      stage_batch<T, S, R, MODE == kModeBwd || MODE == kModeL2>(sm, a, f, b, cnt);
      __syncthreads();
      if constexpr (R == 1) {
        // this pixel's row in the usual kernels: band, strip and row of the strip
        constexpr int kBand = 32 / T * kRows<T>;
        const int row = t / T, in = row % kBand;
        fwd_batch_rows<T, S>(sm, cnt, wid, lane, pxl, (float)(row - in) + 0.5f,
                             (float)(in - in % kRows<T>), in % kRows<T>, acc[0]);
      } else {
        const int wn = warp_list<T, S>(sm, cnt, wid, lane, (float)(G::RW * wid) + 0.5f,
                                       ms.wl[wid]);
        fwd_batch<T, S>(sm, ms.wl[wid], wn, pxl, (float)(R * (lane / T)), acc);
      }
      staged = b;
    }
    if constexpr (MODE == kModeFwd) {
      if (x < f.W) {
#pragma unroll
        for (int r = 0; r < R; r++) {
          if (y0 + r < f.H) {
            const size_t o = f.pix + (size_t)(y0 + r) * f.W + x;
            a.img[o] = acc[r][0];
            a.img[HW + o] = acc[r][1];
            a.img[2 * HW + o] = acc[r][2];
          }
        }
      }
      return;
    }

    // L2 loss and dL/dC of this thread's pixels; the clip's own mean
    const double count3 = 3.0 * (double)f.W * (double)f.H;
    const float gscale = (float)(2.0 / count3), lscale = (float)(1.0 / count3);
    float2 l = make_float2(0.f, 0.f);
#pragma unroll
    for (int r = 0; r < R; r++) {
      float4 g = make_float4(0.f, 0.f, 0.f, 0.f);
      if (x < f.W && y0 + r < f.H) {
        const size_t o = f.pix + (size_t)(y0 + r) * f.W + x;
        const float t0 = a.target[o], t1 = a.target[HW + o], t2 = a.target[2 * HW + o];
        const float d0 = acc[r][0] - t0, d1 = acc[r][1] - t1, d2 = acc[r][2] - t2;
        const float e0 = __saturatef(acc[r][0]) - t0, e1 = __saturatef(acc[r][1]) - t1,
                    e2 = __saturatef(acc[r][2]) - t2;
        const float2 p = make_float2(fmaf(d0, d0, fmaf(d1, d1, d2 * d2)),
                                     fmaf(e0, e0, fmaf(e1, e1, e2 * e2)));
        if constexpr (R == 1) {
          l = p;
        } else {
          l.x += p.x;
          l.y += p.y;
        }
        g = make_float4(gscale * d0, gscale * d1, gscale * d2, 0.f);
        if (a.img) {
          a.img[o] = acc[r][0];
          a.img[HW + o] = acc[r][1];
          a.img[2 * HW + o] = acc[r][2];
        }
      }
      ms.g[(R * (t / T) + r) * T + t % T] = g;
    }
    // the tile's loss: the usual kernels' sums (strips of rows, the warp's
    // lanes, the warps), whatever R is
    using GO = TileGeom<T, kRows<T>>;
    if constexpr (R == 1) {
      ms.sse[t] = l;  // t = row T + column
      __syncthreads();
      l = make_float2(0.f, 0.f);
      if (t < GO::NT)
#pragma unroll
        for (int r = 0; r < GO::R; r++) {
          const float2 p = ms.sse[(GO::R * (t / T) + r) * T + t % T];
          l.x += p.x;
          l.y += p.y;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      l.x += __shfl_xor_sync(0xffffffffu, l.x, o);
      l.y += __shfl_xor_sync(0xffffffffu, l.y, o);
    }
    if (lane == 0 && wid < GO::NW) ms.red[wid] = l;
    __syncthreads();
    if (t == 0) {
      float2 s = make_float2(0.f, 0.f);
#pragma unroll
      for (int w = 0; w < GO::NW; w++) {
        s.x += ms.red[w].x;
        s.y += ms.red[w].y;
      }
      a.loss_part[f.tile] = make_float2(s.x * lscale, s.y * lscale);
    }
    // backward; the last forward batch is still staged
    for (int b = rg.x; b < rg.y; b += S) {
      const int cnt = min(S, rg.y - b);
      if (b != staged) {
        __syncthreads();
        stage_batch<T, S, R, MODE == kModeBwd || MODE == kModeL2>(sm, a, f, b, cnt);
        __syncthreads();
        staged = b;
      }
      bwd_batch<T, S>(sm, shared_addr(ms.g), cnt, a, b);
    }
  }
}

// Blocks per SM the register budget must allow (about 50 registers per
// thread of the 64 K per SM; 32 blocks at most): 32, 20, 5 for T = 8, 16, 32,
// and with one row per thread 5 and 1 for T = 16, 32.
template <int NT>
constexpr int kMinBlocks = 65536 / (NT * 50) < 32 ? 65536 / (NT * 50) : 32;

template <int T, int S, int MODE, int LAUNCH, int R>
__global__ void __launch_bounds__(TileGeom<T, R>::NT, kMinBlocks<TileGeom<T, R>::NT>)
k_render(RenderArgs a) {
  pdl_begin();
  __shared__ TileSmem<S> sm;
  __shared__ ModeSmem<T, S, MODE, R> ms;
  if constexpr (LAUNCH == GS2D_LAUNCH_GRID) {
    if (a.active && (int)blockIdx.x >= *a.active) return;  // a P-frame's subset
    const int tile = a.order[blockIdx.x];
    if ((unsigned)tile >= (unsigned)a.num_tiles) {  // a stale queue: report, skip
      if (threadIdx.x == 0) set_status(a.hdr, GS2D_ERR_BOUNDS);
      return;
    }
    process_tile<T, S, MODE, R>(a, tile_frame<T>(a, tile), sm, ms);
  } else {
    __shared__ int s_next[2];
    if (threadIdx.x == 0) s_next[0] = atomicAdd(&a.hdr->queue, 1);
    __syncthreads();
    const int limit = a.active ? min(*a.active, a.num_tiles) : a.num_tiles;
    for (int k = 0;; k ^= 1) {
      const int q = s_next[k];
      if (q >= limit) break;
      // next ticket now, stored after the tile: its latency overlaps the work
      int next = 0;
      if (threadIdx.x == 0) next = atomicAdd(&a.hdr->queue, 1);
      const int tile = a.order[q];
      if ((unsigned)tile < (unsigned)a.num_tiles)
        process_tile<T, S, MODE, R>(a, tile_frame<T>(a, tile), sm, ms);
      else if (threadIdx.x == 0)
        set_status(a.hdr, GS2D_ERR_BOUNDS);  // a stale queue: report, skip
      if (threadIdx.x == 0) s_next[k ^ 1] = next;
      __syncthreads();
    }
    // every block has taken its last ticket once `done` reaches the grid size
    if (threadIdx.x == 0 && atomicAdd(&a.hdr->done, 1) == (int)gridDim.x - 1) {
      atomicExch(&a.hdr->done, 0);
      atomicExch(&a.hdr->queue, 0);
    }
  }
}

// Whether a launch of num_tiles tiles with n Gaussians takes the kernels with one
// row per thread (four times the warps).  With few tiles the usual ones leave the
// chip's 608 schedulers a warp or two each, and both passes are chains of dependent
// instructions.  The backward gains, since the warps share a tile's Gaussians; the
// forward does not (a pixel's chain is as long as before and a warp's setup per
// Gaussian serves a quarter of the pixels: 4.5 -> 5.3 us at 256 x 256), so it never
// does alone and the fused call does only while the backward's gain is the larger.
// Lines in warps of the usual kernels: up to kAny, up to kDense with at most 48
// pixels per Gaussian.  Usual kernels / these, us, at 10, 104 and 1000 pixels per
// Gaussian that tile the frame (warps); where Gaussians of many sizes leave a few
// tiles with long lists, as fits do, these gain more (a fit step at 640 x 360, 4000
// Gaussians, tile 16: 42 / 37):
//   fused, tile 16: 33.4 / 22.8, 20.1 / 16.0, 18.7 / 16.6 (512); 42.1 / 40.9, 23.7 /
//     25.1, 25.0 / 25.9 (1840); 62.5 / 66.6, 32.7 / 37.8, 30.4 / 36.6 (4080)
//   fused, tile 32: 35.3 / 30.7, 19.5 / 20.6, 16.3 / 18.5 (512); 36.0 / 31.8, 19.1 /
//     20.5, 16.8 / 19.2 (1080)
//   backward, tile 16: 47.7 / 38.3, 23.7 / 21.4, 20.5 / 21.2 (4080); 64.8 / 60.8,
//     32.1 / 32.1, 26.7 / 29.6 (7200)
//   backward, tile 32: 24.9 / 16.3, 12.7 / 10.3, 11.4 / 10.4 (1080); 27.9 / 26.9,
//     13.3 / 14.8, 13.6 / 13.8 (1920)
template <int T, int MODE>
bool few_tiles(int num_tiles, int n) {
  constexpr int kAny = MODE == kModeL2 ? (T == 16 ? 2400 : 0) : T == 16 ? 4800 : 1400;
  constexpr int kDense = MODE == kModeL2 ? (T == 16 ? 2400 : 1200) : T == 16 ? 7200 : 1920;
  constexpr int kWarps = TileGeom<T, kRows<T>>::NW;  // of a tile
  return num_tiles <= kAny / kWarps ||
         (num_tiles <= kDense / kWarps && n >= num_tiles * (T * T / 48));
}

template <int T, int S, int MODE, int LAUNCH, int R>
cudaError_t launch_rows(const RenderArgs& a, cudaStream_t s) {
  constexpr int NT = TileGeom<T, R>::NT;
  int grid = a.num_tiles;
  if (LAUNCH == GS2D_LAUNCH_PERSISTENT)
    grid = persistent_grid((const void*)k_render<T, S, MODE, LAUNCH, R>, NT, a.num_tiles);
  if (grid <= 0) return cudaErrorInvalidConfiguration;
  return launch_pdl(k_render<T, S, MODE, LAUNCH, R>, grid, NT, 0, s, a);
}

template <int T, int S, int MODE, int LAUNCH>
cudaError_t launch_mode(const RenderArgs& a, cudaStream_t s) {
  if (a.num_tiles <= 0) return cudaSuccess;
  if constexpr (T > 8 && LAUNCH == GS2D_LAUNCH_GRID &&
                (MODE == kModeL2 || MODE == kModeBwd)) {
    if (few_tiles<T, MODE>(a.num_tiles, a.n)) return launch_rows<T, S, MODE, LAUNCH, 1>(a, s);
  }
  return launch_rows<T, S, MODE, LAUNCH, kRows<T>>(a, s);
}

template <int T, int S, int LAUNCH>
cudaError_t launch_form(RenderMode mode, const RenderArgs& a, cudaStream_t s) {
  switch (mode) {
    case kModeFwd: return launch_mode<T, S, kModeFwd, LAUNCH>(a, s);
    case kModeBwd: return launch_mode<T, S, kModeBwd, LAUNCH>(a, s);
    case kModeL2: return launch_mode<T, S, kModeL2, LAUNCH>(a, s);
    case kModeCount: return launch_mode<T, S, kModeCount, LAUNCH>(a, s);
    case kModeSelect: return launch_mode<T, S, kModeSelect, LAUNCH>(a, s);
  }
  return cudaErrorInvalidValue;
}

template <int T, int S>
cudaError_t launch_stage(int launch, RenderMode mode, const RenderArgs& a, cudaStream_t s) {
  return launch == GS2D_LAUNCH_GRID ? launch_form<T, S, GS2D_LAUNCH_GRID>(mode, a, s)
                                    : launch_form<T, S, GS2D_LAUNCH_PERSISTENT>(mode, a, s);
}

template <int T>
cudaError_t launch_tile(int stage, int launch, RenderMode mode, const RenderArgs& a,
                        cudaStream_t s) {
  switch (stage) {
    case 32: return launch_stage<T, 32>(launch, mode, a, s);
    case 64: return launch_stage<T, 64>(launch, mode, a, s);
    case 128: return launch_stage<T, 128>(launch, mode, a, s);
    case 256: return launch_stage<T, 256>(launch, mode, a, s);
  }
  return cudaErrorInvalidValue;
}

// Occupancy query of the fit loop's persistent render kernel (cached by
// persistent_grid); the grid form needs none.
template <int T>
cudaError_t prime_tile(int stage, int launch) {
  if (launch == GS2D_LAUNCH_GRID) return cudaSuccess;
  constexpr int R = kRows<T>, NT = TileGeom<T, R>::NT, P = GS2D_LAUNCH_PERSISTENT;
  int g = 0;
  switch (stage) {
    case 32: g = persistent_grid((const void*)k_render<T, 32, kModeL2, P, R>, NT, 1); break;
    case 64: g = persistent_grid((const void*)k_render<T, 64, kModeL2, P, R>, NT, 1); break;
    case 128: g = persistent_grid((const void*)k_render<T, 128, kModeL2, P, R>, NT, 1); break;
    case 256: g = persistent_grid((const void*)k_render<T, 256, kModeL2, P, R>, NT, 1); break;
    default: return cudaErrorInvalidValue;
  }
  return g > 0 ? cudaSuccess : cudaErrorInvalidConfiguration;
}

}  // namespace gs2d
