// Chamfer distance between predicted and target means (Sec. 3.2 B), per frame
// of a batch: the nearest neighbour of every point of each set in the other,
// the gradient towards the predictions and the loss (include/gs2d.h).
//
// The nearest neighbours are exact (smallest FP32 squared distance, ties to the
// lowest index: what a scan of all pairs gives), found through a uniform grid
// over each set: a query looks at its own cell and at rings of cells around it
// until no further ring can hold a closer point, or so many have been looked at
// that a scan of the set is faster.  The scan of all pairs was 2 x 0.94 ms at
// 20 000 points and batch 8 (6.4 10^9 distances, bound by instruction issue); a
// query of spread points evaluates a few dozen.
#include <math.h>

#include <algorithm>

#include "gs2d_internal.cuh"

namespace gs2d {
namespace {

constexpr int kNnCells = 8192;  // cells of a grid (32 KB of counters in the build)
constexpr int kNnThreads = 1024;

// The grid of one set of one frame: cell (x - lo_x) / h clamped to the grid, so
// points outside it lie in its border cells.
struct NnGrid {
  float lo_x, lo_y, h, inv;
  float err;  // bound on the FP32 error of a point's position against the cell edges
  int gx, gy;
};

struct NnSet {
  const float* pts;  // rows x, y of [9][ld] blocks, frame b in columns b n ...
  int n, ld;
  float* x;          // [B][n] coordinates by cell
  float* y;
  int* index;        // [B][n] their index in the frame
  int* start;        // [B][kNnCells + 2] first position of each cell; then the others
  NnGrid* grid;      // [B]
  int* hard;         // [B][n] points left to k_nn_scan, by index in the frame
  int* hards;        // [B] how many
  int* nn;           // [B][n] out: nearest of the other set, by index in the frame
  float* dist;       // [B][n] out: its squared distance
};

struct NnArgs {
  NnSet set[2];
};

__device__ __forceinline__ int nn_axis(float v, float lo, float inv, int g) {
  return min(max((int)floorf((v - lo) * inv), 0), g - 1);
}

// Block-wide reduction of v by op over kNnThreads threads, to every thread.
template <class Op>
__device__ __forceinline__ float block_reduce(float v, float* s_w, Op op) {
  for (int o = 16; o; o >>= 1) v = op(v, __shfl_xor_sync(0xffffffffu, v, o));
  __syncthreads();
  if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = v;
  __syncthreads();
  v = s_w[threadIdx.x & 31];
  for (int o = 16; o; o >>= 1) v = op(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// Block (frame, set): the grid of the set (about two points a cell over the
// bounding box of the finite points, cut at three standard deviations so that
// a few far ones do not make every cell large), then a counting sort of the
// points by cell.  Points with a non-finite coordinate go behind the last
// cell: they are never anyone's nearest neighbour.
__global__ void __launch_bounds__(kNnThreads) k_nn_build(NnArgs a) {
  pdl_begin();
  __shared__ int s_cnt[kNnCells + 1];
  __shared__ float s_w[32];
  __shared__ int s_scan[32];
  __shared__ NnGrid s_grid;
  const int b = blockIdx.x, t = threadIdx.x;
  const NnSet& set = a.set[blockIdx.y];
  const int n = set.n;
  const float* px = set.pts + (size_t)b * n;
  const float* py = px + set.ld;
  float lo_x = INFINITY, hi_x = -INFINITY, lo_y = INFINITY, hi_y = -INFINITY;
  float sx = 0.f, sxx = 0.f, sy = 0.f, syy = 0.f, cnt = 0.f;
#pragma unroll 8
  for (int i = t; i < n; i += kNnThreads) {
    const float x = px[i], y = py[i];
    if (!isfinite(x) || !isfinite(y)) continue;
    lo_x = fminf(lo_x, x);
    hi_x = fmaxf(hi_x, x);
    lo_y = fminf(lo_y, y);
    hi_y = fmaxf(hi_y, y);
    sx += x;
    sxx = fmaf(x, x, sxx);
    sy += y;
    syy = fmaf(y, y, syy);
    cnt += 1.f;
  }
  const auto mn = [](float u, float v) { return fminf(u, v); };
  const auto mx = [](float u, float v) { return fmaxf(u, v); };
  const auto add = [](float u, float v) { return u + v; };
  lo_x = block_reduce(lo_x, s_w, mn);
  hi_x = block_reduce(hi_x, s_w, mx);
  lo_y = block_reduce(lo_y, s_w, mn);
  hi_y = block_reduce(hi_y, s_w, mx);
  sx = block_reduce(sx, s_w, add);
  sxx = block_reduce(sxx, s_w, add);
  sy = block_reduce(sy, s_w, add);
  syy = block_reduce(syy, s_w, add);
  cnt = block_reduce(cnt, s_w, add);
  if (t == 0) {
    NnGrid g = {0.f, 0.f, 1.f, 1.f, 0.f, 1, 1};  // one cell
    const float mean_x = fminf(fmaxf(sx / cnt, lo_x), hi_x);
    const float mean_y = fminf(fmaxf(sy / cnt, lo_y), hi_y);
    const float dev_x = 3.f * sqrtf(fmaxf(sxx / cnt - mean_x * mean_x, 0.f));
    const float dev_y = 3.f * sqrtf(fmaxf(syy / cnt - mean_y * mean_y, 0.f));
    if (isfinite(dev_x) && isfinite(dev_y)) {
      lo_x = fmaxf(lo_x, mean_x - dev_x);
      hi_x = fminf(hi_x, mean_x + dev_x);
      lo_y = fmaxf(lo_y, mean_y - dev_y);
      hi_y = fminf(hi_y, mean_y + dev_y);
    }
    const float w = hi_x - lo_x, h = hi_y - lo_y;
    const float cells = fminf(fmaxf(0.5f * cnt, 1.f), 0.9f * kNnCells);
    float step = fmaxf(sqrtf(w * h / cells), fmaxf(w, h) / cells);
    if (cnt > 0.f && w >= 0.f && h >= 0.f && step > 0.f && isfinite(step) &&
        isfinite(1.f / step)) {
      int gx, gy;
      for (;; step *= 1.25f) {
        gx = (int)fminf(w / step, 65536.f) + 1;
        gy = (int)fminf(h / step, 65536.f) + 1;
        if ((long long)gx * gy <= kNnCells) break;
      }
      g.lo_x = lo_x;
      g.lo_y = lo_y;
      g.h = step;
      g.inv = 1.f / step;
      // a few roundings of values up to |lo| + extent, and of the cell product
      g.err = 2e-6f * (fabsf(lo_x) + fabsf(lo_y) + w + h);
      g.gx = gx;
      g.gy = gy;
    }
    s_grid = g;
    set.grid[b] = g;
    set.hards[b] = 0;
  }
  for (int i = t; i <= kNnCells; i += kNnThreads) s_cnt[i] = 0;
  __syncthreads();
  const NnGrid g = s_grid;
  const int cells = g.gx * g.gy;
  const auto cell_of = [&](float x, float y) {
    if (!isfinite(x) || !isfinite(y)) return cells;
    return nn_axis(y, g.lo_y, g.inv, g.gy) * g.gx + nn_axis(x, g.lo_x, g.inv, g.gx);
  };
#pragma unroll 8
  for (int i = t; i < n; i += kNnThreads) atomicAdd(&s_cnt[cell_of(px[i], py[i])], 1);
  __syncthreads();
  // exclusive scan of the counts (the cells, then the non-finite points)
  constexpr int kPer = (kNnCells + 1 + kNnThreads - 1) / kNnThreads;
  int c[kPer], sum = 0;
#pragma unroll
  for (int k = 0; k < kPer; k++) {
    const int i = t * kPer + k;
    c[k] = i <= kNnCells ? s_cnt[i] : 0;
    sum += c[k];
  }
  const int lane = t & 31, wid = t >> 5;
  int inc = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) s_scan[wid] = inc;
  __syncthreads();
  int at = inc - sum;
  for (int w = 0; w < wid; w++) at += s_scan[w];
  int* start = set.start + (size_t)b * (kNnCells + 2);
#pragma unroll
  for (int k = 0; k < kPer; k++) {
    const int i = t * kPer + k;
    if (i <= kNnCells) {
      s_cnt[i] = at;
      start[i] = at;
    }
    at += c[k];
  }
  if (t == 0) start[kNnCells + 1] = n;
  __syncthreads();
#pragma unroll 8
  for (int i = t; i < n; i += kNnThreads) {
    const float x = px[i], y = py[i];
    const size_t o = (size_t)b * n + atomicAdd(&s_cnt[cell_of(x, y)], 1);
    set.x[o] = x;
    set.y[o] = y;
    set.index[o] = i;
  }
}

// A thread per point, in its own set's cell order (neighbouring threads search
// neighbouring cells).  A point of ring k (its cell k columns or rows away) is
// (k - 1) h farther than the nearest edge of the own cell that has cells behind
// it, whichever of the two points lies outside the grid.  A point whose search
// grows past a share of the set (a cell with most of the points, as with a far
// outlier or tight clusters; a query far outside the grid) goes to k_nn_scan,
// which takes a quarter of the time for a point: so no set takes longer than the
// scan of all pairs did.  A run of cells counts like kHardCell points (its two
// look-ups).
constexpr int kHardShare = 8, kHardMin = 64, kHardCell = 8;

__global__ void __launch_bounds__(128) k_nn_query(NnArgs a) {
  pdl_begin();
  const int b = blockIdx.y;
  const NnSet& from = a.set[blockIdx.z];
  const NnSet& to = a.set[1 - blockIdx.z];
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= from.n) return;
  const size_t fo = (size_t)b * from.n, o = fo + i;
  const float px = from.x[o], py = from.y[o];
  const NnGrid g = to.grid[b];
  const int* __restrict__ start = to.start + (size_t)b * (kNnCells + 2);
  const float* __restrict__ qx = to.x + (size_t)b * to.n;
  const float* __restrict__ qy = to.y + (size_t)b * to.n;
  const int* __restrict__ qi = to.index + (size_t)b * to.n;
  float best = INFINITY;
  int arg = 0, left = to.n / kHardShare + kHardMin;  // points it may still look at
  const auto scan = [&](int c0, int c1) {  // cells c0 ... c1 of one row
    const int s = start[c0], e = start[c1 + 1];
    left -= e - s + kHardCell;
    if (left < 0) return;
    for (int j = s; j < e; j++) {
      const float dx = px - qx[j], dy = py - qy[j];
      const float d = fmaf(dx, dx, dy * dy);
      if (d <= best) {
        const int k = qi[j];
        if (d < best || k < arg) {
          best = d;
          arg = k;
        }
      }
    }
  };
  if (isfinite(px) && isfinite(py)) {
    const int cx = nn_axis(px, g.lo_x, g.inv, g.gx), cy = nn_axis(py, g.lo_y, g.inv, g.gy);
    const int rings = max(max(cx, g.gx - 1 - cx), max(cy, g.gy - 1 - cy));
    // distance to the nearest edge of the cell with cells behind it
    const float ux = px - fmaf((float)cx, g.h, g.lo_x), uy = py - fmaf((float)cy, g.h, g.lo_y);
    const float edge = fminf(fminf(cx > 0 ? ux : INFINITY, cx + 1 < g.gx ? g.h - ux : INFINITY),
                             fminf(cy > 0 ? uy : INFINITY, cy + 1 < g.gy ? g.h - uy : INFINITY));
    for (int k = 0; k <= rings && left >= 0; k++) {
      // strictly farther than the best, FP32 rounding of the distances included
      const float away = k > 0 ? fmaf((float)(k - 1), g.h, edge) * 0.99999f - g.err : 0.f;
      if (away > 0.f && away * away * 0.99999f > best) break;
      const int x0 = max(cx - k, 0), x1 = min(cx + k, g.gx - 1);
      for (int y = max(cy - k, 0); y <= min(cy + k, g.gy - 1) && left >= 0; y++) {
        const int row = y * g.gx;
        if (y == cy - k || y == cy + k) {
          scan(row + x0, row + x1);
        } else {
          if (cx - k >= 0) scan(row + cx - k, row + cx - k);
          if (cx + k < g.gx) scan(row + cx + k, row + cx + k);
        }
      }
    }
  }
  const int index = from.index[o];
  if (left < 0) {
    from.hard[fo + atomicAdd(&from.hards[b], 1)] = index;
    return;
  }
  from.nn[fo + index] = arg;
  from.dist[fo + index] = best;
}

// Two FP32 operations an instruction, each rounded like the single one.
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  return (uint64_t)__float_as_uint(hi) << 32 | __float_as_uint(lo);
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ float lo2(uint64_t v) { return __uint_as_float((uint32_t)v); }
__device__ __forceinline__ float hi2(uint64_t v) { return __uint_as_float((uint32_t)(v >> 32)); }

// The points that k_nn_query left, against all of the other set.  A block takes
// 128 of them, four a lane and the same for every warp, and brings the other set
// through shared memory in tiles, of which each warp looks at its share, four
// points at a time: a load serves 16 distances, and the smallest of four is
// compared and kept at once (with the first of its four points; which one it was
// is looked up at the end).  Bound by the FP32 pipe (four operations a pair): 8 x
// 20 000 points a side, all of them, take 1.05 ms, where a thread per point over
// tiles in shared memory took 1.9, and 1.9 too a block per 8 points whose threads
// read the other set from L2.
constexpr int kScanLane = 4, kScanQ = 32 * kScanLane;
constexpr int kScanThreads = 512, kScanWarps = kScanThreads / 32;
constexpr int kScanTile = kScanWarps * kScanQ;  // points of a tile
constexpr int kScanShare = kScanTile / kScanWarps;

__global__ void __launch_bounds__(kScanThreads, 2) k_nn_scan(NnArgs a) {
  pdl_begin();
  __shared__ __align__(16) float s_x[kScanTile], s_y[kScanTile];  // negated
  const int b = blockIdx.y, t = threadIdx.x, lane = t & 31, wid = t >> 5;
  const NnSet& from = a.set[blockIdx.z];
  const NnSet& to = a.set[1 - blockIdx.z];
  const size_t fo = (size_t)b * from.n;
  const float* __restrict__ qx = to.pts + (size_t)b * to.n;
  const float* __restrict__ qy = qx + to.ld;
  const int count = from.hards[b], n = to.n;
  for (int h0 = blockIdx.x * kScanQ; h0 < count; h0 += gridDim.x * kScanQ) {
    float px[kScanLane], py[kScanLane], best[kScanLane];
    int arg[kScanLane];
#pragma unroll
    for (int q = 0; q < kScanLane; q++) {
      const int i = from.hard[fo + min(h0 + 32 * q + lane, count - 1)];
      px[q] = from.pts[fo + i];
      py[q] = from.pts[fo + from.ld + i];
      best[q] = INFINITY;
      arg[q] = 0;
    }
    for (int j0 = 0; j0 < n; j0 += kScanTile) {
      __syncthreads();
      for (int k = t; k < kScanTile; k += kScanThreads) {
        s_x[k] = j0 + k < n ? -qx[j0 + k] : INFINITY;
        s_y[k] = j0 + k < n ? -qy[j0 + k] : INFINITY;
      }
      __syncthreads();
      const int k0 = wid * kScanShare, k1 = min(k0 + kScanShare, n - j0);
#pragma unroll 2
      for (int k = k0; k < k1; k += 4) {
        const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(s_x + k);
        const ulonglong2 y = *reinterpret_cast<const ulonglong2*>(s_y + k);
#pragma unroll
        for (int q = 0; q < kScanLane; q++) {
          const uint64_t ax = pack2(px[q], px[q]), ay = pack2(py[q], py[q]);
          const uint64_t dx0 = add2(ax, x.x), dy0 = add2(ay, y.x);
          const uint64_t dx1 = add2(ax, x.y), dy1 = add2(ay, y.y);
          const uint64_t d0 = fma2(dx0, dx0, mul2(dy0, dy0));
          const uint64_t d1 = fma2(dx1, dx1, mul2(dy1, dy1));
          // (fminf passes over a NaN, as a comparison does)
          const float d = fminf(fminf(lo2(d0), hi2(d0)), fminf(lo2(d1), hi2(d1)));
          if (d < best[q]) {
            best[q] = d;
            arg[q] = j0 + k;
          }
        }
      }
    }
    // each warp's smallest, at the first point that has it; then the block's, of
    // equal ones the lowest index
    __syncthreads();
    int* s_j = reinterpret_cast<int*>(s_y);
#pragma unroll
    for (int q = 0; q < kScanLane; q++) {
      int j = arg[q];
      for (const int end = min(n, j + 4) - 1; best[q] < INFINITY && j < end; j++) {
        const float dx = px[q] - qx[j], dy = py[q] - qy[j];
        if (fmaf(dx, dx, dy * dy) == best[q]) break;
      }
      s_x[wid * kScanQ + 32 * q + lane] = best[q];
      s_j[wid * kScanQ + 32 * q + lane] = j;
    }
    __syncthreads();
    if (t < kScanQ && h0 + t < count) {
      float d = s_x[t];
      int j = s_j[t];
      for (int w = 1; w < kScanWarps; w++) {
        const float dw = s_x[w * kScanQ + t];
        const int jw = s_j[w * kScanQ + t];
        if (dw < d || (dw == d && jw < j)) {
          d = dw;
          j = jw;
        }
      }
      const int i = from.hard[fo + h0 + t];
      from.nn[fo + i] = j;
      from.dist[fo + i] = d;
    }
  }
}

// Gradient of the Chamfer term with respect to the predicted means: each
// predicted point towards its nearest target, each target pulling its
// nearest predicted point (accumulated with atomics).  Also the per-frame
// loss (a fixed-order sum).
__global__ void __launch_bounds__(256)
k_chamfer_grad(const float* __restrict__ P, int np, int ldp, const float* __restrict__ Q, int nq,
               int ldq, const int* __restrict__ nn1, const int* __restrict__ nn2, float lambda,
               float* __restrict__ dP) {
  pdl_begin();
  const int b = blockIdx.y;
  const float* pb = P + (size_t)b * np;
  const float* qb = Q + (size_t)b * nq;
  float* db = dP + (size_t)b * np;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < np) {
    const int j = nn1[(size_t)b * np + i];
    atomicAdd(&db[i], lambda * 2.0f * (pb[i] - qb[j]) / (float)np);
    atomicAdd(&db[ldp + i], lambda * 2.0f * (pb[ldp + i] - qb[ldq + j]) / (float)np);
  }
  if (i < nq) {
    const int k = nn2[(size_t)b * nq + i];
    atomicAdd(&db[k], lambda * 2.0f * (pb[k] - qb[i]) / (float)nq);
    atomicAdd(&db[ldp + k], lambda * 2.0f * (pb[ldp + k] - qb[ldq + i]) / (float)nq);
  }
}

// Mean squared distances of both directions of frame b, one block.  Sums of three
// floats (FloatSum: no less accurate than double), one division per mean: with
// double sums and divisions in every thread 33 us for 20 000 points a side, 23 so
// (cold; load latency of one block a frame).
__global__ void __launch_bounds__(1024)
k_chamfer_loss(const float* __restrict__ d1, int np, const float* __restrict__ d2, int nq,
               float* __restrict__ loss) {
  pdl_begin();
  __shared__ WarpSums s_sum[2];
  __shared__ double s_d[32];
  __shared__ int s_past;
  const int b = blockIdx.x, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  d1 += (size_t)b * np;
  d2 += (size_t)b * nq;
  FloatSum a, c;
#pragma unroll 4
  for (int i = threadIdx.x; i < np; i += blockDim.x) a.add(d1[i]);
#pragma unroll 4
  for (int i = threadIdx.x; i < nq; i += blockDim.x) c.add(d2[i]);
  a.warp_sum();
  c.warp_sum();
  if (lane == 0) {
    s_sum[0].put(wid, a);
    s_sum[1].put(wid, c);
  }
  __syncthreads();
  if (wid == 0) {
    a = s_sum[0].sum(lane);
    c = s_sum[1].sum(lane);
    if (lane == 0) {
      s_past = !isfinite(a.hi) || !isfinite(c.hi);
      loss[b] = (float)(a.value() / np + c.value() / nq);
    }
  }
  __syncthreads();
  if (!s_past) return;
  // a sum past FP32's range, whose mean may still lie within it
  double x = 0.0, y = 0.0;
  for (int i = threadIdx.x; i < np; i += blockDim.x) x += d1[i];
  for (int i = threadIdx.x; i < nq; i += blockDim.x) y += d2[i];
  double v = x / np + y / nq;
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if (lane == 0) s_d[wid] = v;
  __syncthreads();
  if (threadIdx.x != 0) return;
  v = 0.0;
  for (int w = 0; w < (int)(blockDim.x >> 5); w++) v += s_d[w];
  loss[b] = (float)v;
}

}  // namespace
}  // namespace gs2d

using namespace gs2d;

// Four-byte words of scratch: nearest neighbours, distances, the three sorted
// arrays and the list of the points to scan for of every point, cell starts,
// grid and that list's length of every set.
extern "C" uint64_t gs2d_chamfer_scratch_bytes(int32_t n, int32_t m, int32_t B) {
  const uint64_t points = (uint64_t)B * ((uint64_t)n + m);
  const uint64_t sets = 2 * (uint64_t)B;
  return points * 6 * 4 + sets * (kNnCells + 3) * 4 + sets * sizeof(NnGrid) + 64;
}

extern "C" gs2d_status gs2d_chamfer(const float* params, int32_t n, int32_t ldp,
                                    const float* targets, int32_t m, int32_t ldq, int32_t B,
                                    float lambda, float* dparams, float* loss, void* scratch,
                                    void* stream) {
  if (n < 1 || m < 1 || B < 1 || !params || !targets || !scratch ||
      (int64_t)ldp < (int64_t)B * n || (int64_t)ldq < (int64_t)B * m)
    return set_error(GS2D_ERR_INVALID_ARG, "gs2d_chamfer: arguments");
  cudaStream_t s = (cudaStream_t)stream;
  int* w = static_cast<int*>(scratch);
  const auto take = [&w](size_t words) {
    int* p = w;
    w += words;
    return p;
  };
  NnArgs a;
  const int counts[2] = {n, m}, lds[2] = {ldp, ldq};
  const float* pts[2] = {params, targets};
  for (int k = 0; k < 2; k++) {
    NnSet& set = a.set[k];
    const size_t all = (size_t)B * counts[k];
    set.pts = pts[k];
    set.n = counts[k];
    set.ld = lds[k];
    set.nn = take(all);
    set.dist = reinterpret_cast<float*>(take(all));
    set.x = reinterpret_cast<float*>(take(all));
    set.y = reinterpret_cast<float*>(take(all));
    set.index = take(all);
    set.hard = take(all);
    set.hards = take(B);
    set.start = take((size_t)B * (kNnCells + 2));
    set.grid = reinterpret_cast<NnGrid*>(take((size_t)B * sizeof(NnGrid) / 4));
  }
  const NnSet &p = a.set[0], &q = a.set[1];
  cudaError_t e = launch_pdl(k_nn_build, dim3(B, 2), kNnThreads, 0, s, a);
  if (e == cudaSuccess)
    e = launch_pdl(k_nn_query, dim3((std::max(n, m) + 127) / 128, B, 2), 128, 0, s, a);
  // (most often nothing is left: at most a wave of blocks to find that out)
  if (e == cudaSuccess)
    e = launch_pdl(k_nn_scan,
                   dim3(std::max(1, std::min((std::max(n, m) + kScanQ - 1) / kScanQ,
                                             152 * 2 / (2 * B))), B, 2), kScanThreads, 0, s, a);
  if (e == cudaSuccess && dparams)
    e = launch_pdl(k_chamfer_grad, dim3((std::max(n, m) + 255) / 256, B), 256, 0, s, params, (int)n,
                   (int)ldp, targets, (int)m, (int)ldq, (const int*)p.nn, (const int*)q.nn, lambda,
                   dparams);
  if (e == cudaSuccess && loss)
    e = launch_pdl(k_chamfer_loss, B, 1024, 0, s, (const float*)p.dist, (int)n,
                   (const float*)q.dist, (int)m, loss);
  if (e != cudaSuccess) return set_error(GS2D_ERR_CUDA, cudaGetErrorString(e));
  return set_error(GS2D_OK, "");
}
