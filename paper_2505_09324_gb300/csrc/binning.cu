// Projection, tile binning and the sort by tile id.
//
// The method renders with the tile-based rasterizer it inherits (Sec. 3,
// "differentiable tile-based rasterization"); in 2D there is no depth
// (Sec. 3.1, accumulated-sum blending), so within a tile the Gaussians are
// ordered by index: the sorted list is the (tile, index) key order.
//
// The sort is a single-digit radix (counting) sort by tile id over all SMs:
//   1. k_count: per-tile entry counts (atomic increments from each Gaussian's
//      tiles) and the entries of each group of Gaussians; the last block to
//      finish scans both (the groups' first backward slots, the tiles' list
//      ranges, capacity);
//   2. k_bin_scatter: every entry claims the next slot of its tile's list;
//   3. k_sort: each tile's list is sorted by Gaussian index (a warp bitonic
//      network in registers for lists of up to 512, by the block through a
//      bitmap in shared memory for longer ones), restoring exactly the order a stable sort of the
//      index-ordered entries would give.
// Each is a chain of a few dependent memory latencies, so the number of
// launches and of warps in flight is what counts: a group is 64 Gaussians
// (313 blocks at 20 000; 79 blocks of 256 left half the SMs idle), and its
// entries are dealt out to all 256 threads of the block (the scatter at
// 1920 x 1080, 20 000 Gaussians, tile 16: 16.9 -> 8.4 us; with it and two
// launches fewer, prepare + render: 62.6 -> 50.8 us).  Plans of more than
// kOneScan tiles or groups scan in a launch of their own (k_bin_scan).
// Steps 1 and 3 also build the render queue: tiles grouped by list-length
// class (floor(log2(len)) + 1, 0 for empty tiles), longest class first.  The
// scan gives each tile its rank inside its class, the segment sort turns
// (class, rank) into the queue position.
// A batch of clips is binned in one pass: tiles are numbered clip after clip
// and each Gaussian's rectangle is stored in that numbering.
#include "gs2d_internal.cuh"

namespace gs2d {

constexpr int kLongMax = 1 << 15;   // longest list that is sorted
constexpr int kSmemKeys = 1 << 13;  // words of shared memory of a sort (32 KB)
constexpr int kThreads = 256;
constexpr int kGroup = 64;          // Gaussians per block
constexpr int kGroupLarge = 256;    // the same beyond kManyGroups groups
// (what one block scans in two steps, and some two waves of blocks: 300 000
// Gaussians, most of them off a 64 x 48 frame, 40 us in groups of 64, 29 in groups
// of 256; 500 000 at 1080p 68 / 62)
constexpr int kManyGroups = 1 << 11;
// Up to two steps of the one-block scan (1024 tiles or groups each, 2.3 us a
// step: a chain of loads, scans and class counts) it is faster than another
// launch: k_count with its scan takes 10 us at 256 tiles against 8.5 + 4.5,
// and 28 us at 8160 tiles against 9 + 8 (cold caches).
constexpr int kOneScan = 2048;

// The binning's view of a workspace.
struct BinArgs {
  ClipSet cs;
  int n, num_tiles, tile_shift;
  int group, groups;       // Gaussians per block, blocks
  int one_scan;            // k_count's last block scans
  int64_t max_entries;
  float sigma_cut, alpha_min, det_eps, margin;
  const float* params;
  float4* rec;
  int4* rect;              // tight rectangles
  int4* lrect;             // the rectangles the lists are built from
  int* offs;               // [n] first backward slot of each Gaussian
  int* tile_cnt;           // zero between calls
  int* tile_cnt2;          // the same for the tight rectangles of a rebuild
  long long* sums;         // [2][groups] entries per group, then exclusive offsets
  int* cursor;
  int2* ranges;
  int* bucket;
  uint32_t* rank;
  int* order;
  uint32_t* list;
  uint32_t* spare;         // [max_entries] scratch of the longest sorts (the backward records)
  WsHeader* hdr;
};

// Adam step of the fit loop, advanced by the first kernel of an iteration.
struct AdamTick {
  int on;
  float b1, b2, lr, lr_decay;
};

// ---------------------------------------------------------------------------
// Projection (gs2d_project): records and rectangles.
__global__ void __launch_bounds__(kThreads)
k_project(int n, ClipSet cs, int tile_shift, float sigma_cut, float alpha_min, float det_eps,
          const float* __restrict__ params, float4* __restrict__ rec, int4* __restrict__ rect) {
  pdl_begin();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  rect[i] = project_one(i, n, clip_of_gaussian(cs, i), tile_shift, sigma_cut, alpha_min, det_eps,
                        params, rec);
}

// Adam step counter, the powers beta^step and the decayed learning rate of
// the step that begins (thread 0 of the first kernel of a fit iteration).
__device__ __forceinline__ void adam_tick_header(WsHeader* hdr, float b1, float b2, float lr,
                                                 float lr_decay) {
  const int t = ++hdr->step;
  const double p1 = t == 1 ? (double)b1 : hdr->pw1 * b1;
  const double p2 = t == 1 ? (double)b2 : hdr->pw2 * b2;
  hdr->pw1 = p1;
  hdr->pw2 = p2;
  hdr->bc1 = (float)(1.0 - p1);
  hdr->bc2 = (float)(1.0 - p2);
  const double pd = t == 1 ? 1.0 : hdr->pwd * lr_decay;
  hdr->pwd = pd;
  hdr->lr_now = (float)(lr * pd);
}

// Exclusive scan of v over the block; *total to every thread.
template <typename V>
__device__ __forceinline__ V block_scan(V v, V* warp_sum, V* total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  V x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const V y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) warp_sum[wid] = x;
  __syncthreads();
  V pre = 0, all = 0;
  for (int w = 0; w < nw; w++) {
    const V y = warp_sum[w];
    pre += w < wid ? y : 0;
    all += y;
  }
  *total = all;
  __syncthreads();
  return pre + x - v;
}

// A group's rectangles and the first entry of each, in shared memory: entry e
// of the group belongs to the last Gaussian whose start is <= e.
struct GroupSmem {
  int4 rect[kGroupLarge];
  int start[kGroupLarge];
  long long warp_sum[kThreads / 32];
  int last;
};

// Deals the rectangles (thread t < group: that of Gaussian t) out; returns the
// group's entries.  `excl`: this thread's first entry.
__device__ __forceinline__ long long group_entries(GroupSmem& gs, int4 rc, int group,
                                                   long long* excl) {
  const long long cnt = (long long)rc.z * rc.w;
  long long total;
  const long long ex = block_scan(cnt, gs.warp_sum, &total);
  if ((int)threadIdx.x < group) {
    gs.rect[threadIdx.x] = rc;
    gs.start[threadIdx.x] = (int)min(ex, (long long)INT32_MAX);
  }
  __syncthreads();
  *excl = ex;
  return total;
}

// Entry e of the group: its Gaussian (index in the group) and tile.
__device__ __forceinline__ int group_entry(const GroupSmem& gs, int group, int e, int* tile) {
  int lo = 0;
  for (int step = group >> 1; step > 0; step >>= 1)
    if (gs.start[lo + step] <= e) lo += step;
  const int4 rc = gs.rect[lo];
  const int j = e - gs.start[lo];
  const int dy = (int)((unsigned)j / (unsigned)rc.z);
  *tile = rc.x + dy * rc.y + (j - dy * rc.z);
  return lo;
}

// More entries than any plan holds: they are not counted per tile (the group
// sums alone report the overflow).
constexpr long long kMostEntries = 1ll << 28;

__device__ __forceinline__ void group_count(const GroupSmem& gs, int group, long long total,
                                            int* __restrict__ tile_cnt) {
  if (total > kMostEntries) return;
  for (int e = threadIdx.x; e < (int)total; e += kThreads) {
    int tile;
    group_entry(gs, group, e, &tile);
    atomicAdd(&tile_cnt[tile], 1);
  }
}

// Render-queue class of a list of length len: 0 (empty), 1 + floor(log2(len))
// capped at kBuckets - 1.
__device__ __forceinline__ int length_class(int len) {
  return len <= 0 ? 0 : min(kBuckets - 1, 32 - __clz(len));
}

constexpr int kTileItems = 4;  // tiles per thread of a scan step

// Rank of each lane's tile inside its class, counted in hist (shared): one
// atomic per class and warp.
__device__ __forceinline__ int class_rank(int cls, bool valid, int* hist) {
  const unsigned peers = __match_any_sync(0xffffffffu, valid ? cls : -1);
  const int lane = threadIdx.x & 31, leader = __ffs(peers) - 1;
  int base = 0;
  if (valid && lane == leader) base = atomicAdd(&hist[cls], __popc(peers));
  base = __shfl_sync(0xffffffffu, base, leader);
  return base + __popc(peers & ((1u << lane) - 1u));
}

// Entries per group -> first entry of the group (in place or elsewhere), by
// one block; returns the total.
__device__ __forceinline__ long long scan_sums(const long long* sums, long long* first, int groups,
                                               long long* warp_sum) {
  long long run = 0;
  for (int b0 = 0; b0 < groups; b0 += kThreads * kTileItems) {
    const int b = b0 + threadIdx.x * kTileItems;
    long long v[kTileItems], mine = 0, total;
#pragma unroll
    for (int k = 0; k < kTileItems; k++) {
      v[k] = b + k < groups ? __ldcg(&sums[b + k]) : 0;
      mine += v[k];
    }
    long long at = run + block_scan(mine, warp_sum, &total);
#pragma unroll
    for (int k = 0; k < kTileItems; k++) {
      if (b + k < groups) first[b + k] = at;
      at += v[k];
    }
    run += total;
  }
  return run;
}

// Whether a rebuild lists the tight rectangles instead of the widened ones:
// where these overflow the capacity, or one tile's list of them is too long to
// sort, and the tight ones do neither.  Lists hold a Gaussian at most once, so
// the tiles are looked at only beyond kLongMax Gaussians.  The same in every
// thread of every block: the counts are complete and the totals global.
__device__ __forceinline__ bool rebuild_tight(const BinArgs& a, long long total,
                                              long long total2) {
  if (total2 > a.max_entries) return false;
  if (total > a.max_entries || a.n <= kLongMax) return total > a.max_entries;
  bool wide = false, tight = false;
  for (int i = threadIdx.x; i < a.num_tiles; i += kThreads) {
    wide |= __ldcg(&a.tile_cnt[i]) > kLongMax;
    tight |= __ldcg(&a.tile_cnt2[i]) > kLongMax;
  }
  return __syncthreads_or(wide) && !__syncthreads_or(tight);
}

// The whole scan by one block (k_count's last): group offsets, the capacity
// decision, list ranges, cursors and queue ranks of the tiles; the tile counts
// are cleared for the next binning.  LAZY: a rebuild, see rebuild_tight.
template <bool LAZY>
__device__ __forceinline__ void one_block_scan(const BinArgs& a, GroupSmem& gs, int* s_hist) {
  const int t = threadIdx.x;
  long long total = scan_sums(a.sums, a.sums, a.groups, gs.warp_sum);
  bool tight = false;
  if (LAZY) {
    const long long total2 =
        scan_sums(a.sums + a.groups, a.sums + a.groups, a.groups, gs.warp_sum);
    tight = rebuild_tight(a, total, total2);
    if (tight) total = total2;
  }
  const bool over = total > a.max_entries;
  if (t < kBuckets) s_hist[t] = 0;
  __syncthreads();
  int* cnt = LAZY && tight ? a.tile_cnt2 : a.tile_cnt;
  int* other = LAZY ? (tight ? a.tile_cnt : a.tile_cnt2) : nullptr;
  int* warp_sum = reinterpret_cast<int*>(gs.warp_sum);
  int run = 0;
  for (int c0 = 0; c0 < a.num_tiles; c0 += kThreads * kTileItems) {
    const int base = c0 + t * kTileItems;
    int c[kTileItems], v = 0;
#pragma unroll
    for (int k = 0; k < kTileItems; k++) {
      c[k] = base + k < a.num_tiles && !over ? __ldcg(&cnt[base + k]) : 0;
      v += c[k];
    }
    int chunk;
    int s = run + block_scan(v, warp_sum, &chunk);
    run += chunk;
#pragma unroll
    for (int k = 0; k < kTileItems; k++) {
      const int i = base + k;
      const bool valid = i < a.num_tiles;
      const int cls = length_class(c[k]);
      const int r = class_rank(cls, valid, s_hist);
      if (valid) {
        // an empty tile's range is (0, 0) wherever it sits in the list
        a.ranges[i] = c[k] == 0 ? make_int2(0, 0) : make_int2(s, s + c[k]);
        a.cursor[i] = s;
        a.rank[i] = ((uint32_t)cls << 28) | (uint32_t)r;
        cnt[i] = 0;
        if (LAZY) other[i] = 0;
      }
      s += c[k];
    }
  }
  __syncthreads();
  if (t < kBuckets) a.bucket[t] = s_hist[t];
  if (t == 0) {
    a.hdr->entries_raw = total;
    a.hdr->n_entries = over ? 0 : (int)total;
    if (over) atomicCAS(&a.hdr->status, 0, (int)GS2D_ERR_CAPACITY);
    a.hdr->lists_tight = tight ? 1 : 0;
  }
}

// What k_count counts: the rectangles of gs2d_project, those of a projection
// it does itself (gs2d_prepare and P-frames), or the widened rectangles of a
// rebuild of the fit loop's retained lists (see below), with the tight ones
// beside them.
enum CountMode { kCountRects, kCountProject, kCountRebin };

template <CountMode MODE>
__global__ void __launch_bounds__(kThreads)
k_count(const __grid_constant__ BinArgs a, AdamTick tick) {
  pdl_begin();
  __shared__ GroupSmem gs;
  __shared__ int s_hist[kBuckets];
  constexpr bool kLazy = MODE == kCountRebin;
  if (kLazy && a.hdr->lists_valid) return;  // the same for every thread of the grid
  const int t = threadIdx.x, i = blockIdx.x * a.group + t;
  if (blockIdx.x == 0) {
    if (t == 0) {
      if (kLazy) {
        a.hdr->rebins++;
      } else {
        if (tick.on) adam_tick_header(a.hdr, tick.b1, tick.b2, tick.lr, tick.lr_decay);
        a.hdr->lists_valid = 0;  // the lists are built from the tight rectangles
      }
    }
    if (!a.one_scan && t < 2 * kBuckets) a.bucket[t] = 0;  // k_bin_scan adds to them
  }
  int4 rc = make_int4(0, 0, 0, 0), rt = rc;
  if (t < a.group && i < a.n) {
    if (MODE == kCountRects) {
      rc = a.rect[i];
    } else if (MODE == kCountProject) {
      rc = project_one(i, a.n, clip_of_gaussian(a.cs, i), a.tile_shift, a.sigma_cut, a.alpha_min,
                       a.det_eps, a.params, a.rec);
      a.rect[i] = rc;
    } else {
      const gs2d_clip cl = clip_of_gaussian(a.cs, i);
      int tx0 = 0, ty0 = 0, tx1 = 0, ty1 = 0;
      if (gaussian_tiles(i, a.n, cl, a.tile_shift, a.sigma_cut, a.alpha_min, a.det_eps, a.params,
                         a.margin, tx0, ty0, tx1, ty1))
        rc = make_int4(cl.tile_off + ty0 * cl.tiles_x + tx0, cl.tiles_x, tx1 - tx0, ty1 - ty0);
      rt = a.rect[i];
    }
    a.lrect[i] = rc;
  }
  long long ex;
  const long long total = group_entries(gs, rc, a.group, &ex);
  group_count(gs, a.group, total, a.tile_cnt);
  if (t == 0) a.sums[blockIdx.x] = total;
  if (kLazy) {
    __syncthreads();
    const long long total2 = group_entries(gs, rt, a.group, &ex);
    group_count(gs, a.group, total2, a.tile_cnt2);
    if (t == 0) a.sums[a.groups + blockIdx.x] = total2;
  }
  if (!a.one_scan) return;
  // the last block to get here sees every block's counts and sums
  __threadfence();
  __syncthreads();
  if (t == 0) gs.last = atomicAdd(&a.hdr->ticket, 1) == (int)gridDim.x - 1;
  __syncthreads();
  if (!gs.last) return;
  if (t == 0) a.hdr->ticket = 0;
  __threadfence();
  one_block_scan<kLazy>(a, gs, s_hist);
}

// ---------------------------------------------------------------------------
// Fit loop with retained tile lists.  Within a tile a Gaussian adds nothing
// outside its cut-off box, so a list may hold Gaussians that do not reach the
// tile: such a pair adds exact zeros.  Each Gaussian is listed over its
// rectangle widened by `margin` pixels; the lists, and the backward slots,
// which follow the listed rectangles, are rebuilt only in an iteration where
// some tight rectangle has left its listed one.  The per-Gaussian reduction
// takes the slots of the tight rectangle, in its order, so results are the
// same as with lists rebuilt every iteration.
//
// k_project_fit: records, tight rectangles, the containment test against the
// listed rectangle (clears hdr->lists_valid on a miss) and the Adam tick.
__global__ void __launch_bounds__(128)
k_project_fit(const __grid_constant__ BinArgs a, AdamTick tick) {
  pdl_begin();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) adam_tick_header(a.hdr, tick.b1, tick.b2, tick.lr, tick.lr_decay);
  if (i >= a.n) return;
  const gs2d_clip cl = clip_of_gaussian(a.cs, i);
  int tx0 = 0, ty0 = 0, tx1 = 0, ty1 = 0;
  const bool vis = gaussian_tiles(i, a.n, cl, a.tile_shift, a.sigma_cut, a.alpha_min, a.det_eps,
                                  a.params, 0.0f, tx0, ty0, tx1, ty1);
  a.rect[i] = vis ? make_int4(cl.tile_off + ty0 * cl.tiles_x + tx0, cl.tiles_x, tx1 - tx0,
                              ty1 - ty0)
                  : make_int4(0, 0, 0, 0);
  write_record(i, a.n, vis, a.sigma_cut, a.alpha_min, a.params, a.rec);
  if (vis) {
    const int4 lr4 = a.lrect[i];
    bool inside = lr4.z > 0;
    if (inside) {
      const int rel = lr4.x - cl.tile_off;
      const int ly0 = rel / cl.tiles_x, lx0 = rel - ly0 * cl.tiles_x;
      inside = lx0 <= tx0 && ly0 <= ty0 && tx1 <= lx0 + lr4.z && ty1 <= ly0 + lr4.w;
    }
    if (!inside) a.hdr->lists_valid = 0;
  }
}

// ---------------------------------------------------------------------------
// The scans in a launch of their own (large plans).  Block 0: the groups'
// first entries.  The others: ranges and cursors of a chunk of 1024 tiles; the
// first of them also records the total and the capacity decision.  Every
// block sums what it needs of the rest itself.  Sums are 64-bit so that a
// pathological input is reported as over capacity instead of wrapping around.
template <bool LAZY>
__global__ void __launch_bounds__(kThreads)
k_bin_scan(const __grid_constant__ BinArgs a, long long* __restrict__ first) {
  pdl_begin();
  __shared__ long long warp_sum[kThreads / 32];
  __shared__ int s_hist[kBuckets], s_base[kBuckets];
  if (LAZY && a.hdr->lists_valid) return;  // the same for every thread of the grid
  const int t = threadIdx.x, tb = (int)blockIdx.x - 1;
  long long tot = 0, tot2 = 0, total, total2 = 0;
  for (int b = t; b < a.groups; b += kThreads) {
    tot += a.sums[b];
    tot2 += LAZY ? a.sums[a.groups + b] : 0;
  }
  block_scan(tot, warp_sum, &total);
  if (LAZY) block_scan(tot2, warp_sum, &total2);
  const bool tight = LAZY && rebuild_tight(a, total, total2);
  if (tight) total = total2;
  const bool over = total > a.max_entries;
  if (tb < 0) {
    scan_sums(a.sums + (tight ? a.groups : 0), first, a.groups, warp_sum);
    return;
  }
  const int* cnt = tight ? a.tile_cnt2 : a.tile_cnt;
  const int c0 = tb * kThreads * kTileItems;
  long long before = 0, prefix_tiles;
  for (int i = t; i < c0; i += kThreads) before += cnt[i];
  block_scan(before, warp_sum, &prefix_tiles);
  if (t < kBuckets) s_hist[t] = 0;
  __syncthreads();
  const int base = c0 + t * kTileItems;
  int c[kTileItems], cls[kTileItems], r[kTileItems], v = 0;
#pragma unroll
  for (int k = 0; k < kTileItems; k++) {
    c[k] = base + k < a.num_tiles && !over ? cnt[base + k] : 0;
    v += c[k];
  }
  int chunk;
  int s = (over ? 0 : (int)prefix_tiles) + block_scan(v, reinterpret_cast<int*>(warp_sum), &chunk);
#pragma unroll
  for (int k = 0; k < kTileItems; k++) {
    const int i = base + k;
    cls[k] = length_class(c[k]);
    r[k] = class_rank(cls[k], i < a.num_tiles, s_hist);
    if (i < a.num_tiles) {
      a.ranges[i] = c[k] == 0 ? make_int2(0, 0) : make_int2(s, s + c[k]);
      a.cursor[i] = s;
    }
    s += c[k];
  }
  __syncthreads();
  // this block's first rank in each class
  if (t < kBuckets) s_base[t] = s_hist[t] ? atomicAdd(&a.bucket[t], s_hist[t]) : 0;
  __syncthreads();
#pragma unroll
  for (int k = 0; k < kTileItems; k++)
    if (base + k < a.num_tiles)
      a.rank[base + k] = ((uint32_t)cls[k] << 28) | (uint32_t)(s_base[cls[k]] + r[k]);
  if (tb == 0 && t == 0) {
    a.hdr->entries_raw = total;
    a.hdr->n_entries = over ? 0 : (int)total;
    if (over) atomicCAS(&a.hdr->status, 0, (int)GS2D_ERR_CAPACITY);
    a.hdr->lists_tight = tight ? 1 : 0;
  }
}

// Scatter: the first backward slot of every Gaussian, and every entry claims
// the next slot of its tile's list; each thread keeps kInFlight atomics in
// flight before it stores the claimed slots.  `first`: the groups' first
// entries.
constexpr int kInFlight = 4;

template <bool LAZY>
__global__ void __launch_bounds__(kThreads)
k_bin_scatter(const __grid_constant__ BinArgs a, const long long* __restrict__ first) {
  pdl_begin();
  __shared__ GroupSmem gs;
  if (LAZY && a.hdr->lists_valid) return;
  const bool over = a.hdr->entries_raw != (int64_t)a.hdr->n_entries;
  const int t = threadIdx.x, i = blockIdx.x * a.group + t;
  const bool mine = t < a.group && i < a.n;
  // the rectangles listed: the widened ones, or the tight ones of a rebuild
  // whose widened lists overflowed, which become the listed ones
  const bool use_tight = LAZY && a.hdr->lists_tight;
  int4 rc = make_int4(0, 0, 0, 0);
  if (mine) {
    rc = use_tight ? a.rect[i] : a.lrect[i];
    if (use_tight) a.lrect[i] = rc;
  }
  const long long base = a.one_scan && use_tight ? first[a.groups + blockIdx.x]
                                                 : first[blockIdx.x];
  long long ex;
  const long long total = group_entries(gs, rc, a.group, &ex);
  if (mine) a.offs[i] = over ? 0 : (int)(base + ex);
  if (over) return;
  for (int e0 = t; e0 < (int)total; e0 += kThreads * kInFlight) {
    int pos[kInFlight], gi[kInFlight];
#pragma unroll
    for (int u = 0; u < kInFlight; u++) {
      const int e = e0 + u * kThreads;
      pos[u] = -1;
      if (e < (int)total) {
        int tile;
        gi[u] = blockIdx.x * a.group + group_entry(gs, a.group, e, &tile);
        pos[u] = atomicAdd(&a.cursor[tile], 1);
      }
    }
#pragma unroll
    for (int u = 0; u < kInFlight; u++)
      if (pos[u] >= 0) a.list[pos[u]] = (uint32_t)gi[u];
  }
}

// Bitonic sort of up to 32 K keys held by one warp, K per lane in blocked
// order (element e = lane * K + r).  Exchange distances j >= K pair lanes
// (shuffles), distances j < K pair registers of the same lane.
template <int K>
__device__ __forceinline__ void warp_bitonic(uint32_t (&v)[K], int lane) {
#pragma unroll
  for (int k = 2; k <= 32 * K; k <<= 1) {
#pragma unroll
    for (int j = k >> 1; j > 0; j >>= 1) {
      if (j >= K) {
        const int lj = j / K;
        const bool lower = (lane & lj) == 0;
#pragma unroll
        for (int r = 0; r < K; r++) {
          const uint32_t w = __shfl_xor_sync(0xffffffffu, v[r], lj);
          const bool asc = ((lane * K + r) & k) == 0;
          v[r] = (lower == asc) ? min(v[r], w) : max(v[r], w);
        }
      } else {
#pragma unroll
        for (int r = 0; r < K; r++) {
          const int p = r ^ j;
          if (p > r) {
            const bool asc = ((lane * K + r) & k) == 0;
            const uint32_t a = v[r], b = v[p];
            if ((a > b) == asc) {
              v[r] = b;
              v[p] = a;
            }
          }
        }
      }
    }
  }
}

template <int K>
__device__ __forceinline__ void warp_sort_list(uint32_t* __restrict__ seg, int len, int lane) {
  uint32_t v[K];
#pragma unroll
  for (int r = 0; r < K; r++) {
    const int e = lane * K + r;
    v[r] = e < len ? seg[e] : 0xffffffffu;
  }
  warp_bitonic<K>(v, lane);
#pragma unroll
  for (int r = 0; r < K; r++) {
    const int e = lane * K + r;
    if (e < len) seg[e] = v[r];
  }
}

// Bitonic sort of `len` keys (at most kSmemKeys) at seg, by the block, in
// shared memory padded to a power of two.
__device__ __forceinline__ void block_sort(uint32_t* __restrict__ seg, int len,
                                           uint32_t* s_keys) {
  const int t = threadIdx.x;
  int P = 64;
  while (P < len) P <<= 1;
  __syncthreads();
  for (int i = t; i < P; i += kThreads) s_keys[i] = i < len ? seg[i] : 0xffffffffu;
  __syncthreads();
  for (int k = 2; k <= P; k <<= 1) {
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int x = t; x < P / 2; x += kThreads) {
        // the x-th pair (i, i + j) of this distance
        const int i = ((x & ~(j - 1)) << 1) | (x & (j - 1)), p = i | j;
        const uint32_t u = s_keys[i], v = s_keys[p];
        if ((u > v) == ((i & k) == 0)) {
          s_keys[i] = v;
          s_keys[p] = u;
        }
      }
      __syncthreads();
    }
  }
  for (int i = t; i < len; i += kThreads) seg[i] = s_keys[i];
  __syncthreads();
}

// Keys below v among the `len` ascending keys at seg.
__device__ __forceinline__ int lower_count(const uint32_t* seg, int len, uint32_t v) {
  int lo = 0, hi = len;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (seg[mid] < v) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// Sort of a list of up to kLongMax keys by the block: runs of kSmemKeys in
// shared memory, then each key's place among the other runs by binary search
// (the keys are distinct), through `spare`.
__device__ __noinline__ void block_sort_long(uint32_t* seg, int len, uint32_t* spare,
                                                uint32_t* s_keys) {
  for (int r = 0; r < len; r += kSmemKeys)
    block_sort(seg + r, min(kSmemKeys, len - r), s_keys);
  if (len <= kSmemKeys) return;
  for (int i = threadIdx.x; i < len; i += kThreads) {
    const uint32_t v = seg[i];
    int at = i % kSmemKeys;
    for (int r = 0; r < len; r += kSmemKeys)
      if (r != i - i % kSmemKeys) at += lower_count(seg + r, min(kSmemKeys, len - r), v);
    spare[at] = v;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < len; i += kThreads) seg[i] = spare[i];
  __syncthreads();
}

// Sort of a list of any length by the block through a bitmap of the keys, which
// are distinct and lie in [first, first + n), the tile's clip: 2^18 of them at a
// time, each pass one reading of the list and its set bits in order.  What
// bounds it is the latency of these loads and stores, where the bitonic network
// is a chain of shared-memory exchanges: binning 600 / 8192 / 32 768 Gaussians of
// one tile takes 12.7 / 28.5 / 83 us so, 19 / 98 / 743 by networks of 256 threads,
// and took 24 / 86 / 362 by networks of 1024 threads with the whole list in shared
// memory, in a launch of their own.
constexpr int kBitKeys = 32 * kSmemKeys;

__device__ __noinline__ void block_sort_bits(uint32_t* seg, int len, uint32_t first, int n,
                                                uint32_t* spare, uint32_t* s_bits) {
  __shared__ int s_warp[kThreads / 32];
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  uint32_t* out = n <= kBitKeys ? seg : spare;  // (one pass: read before it is written)
  int done = 0;
  for (int k0 = 0; k0 < n; k0 += kBitKeys) {
    // rows of 32 words, shared out to the warps in order
    const int rows = (min(kBitKeys, n - k0) + 1023) / 1024;
    const int r0 = rows * wid / (kThreads / 32), r1 = rows * (wid + 1) / (kThreads / 32);
    __syncthreads();
    for (int i = t; i < 32 * rows; i += kThreads) s_bits[i] = 0u;
    __syncthreads();
#pragma unroll 4
    for (int i = t; i < len; i += kThreads) {
      const uint32_t k = seg[i] - first - (uint32_t)k0;
      if (k < (uint32_t)kBitKeys) atomicOr(&s_bits[k >> 5], 1u << (k & 31u));
    }
    __syncthreads();
    int mine = 0;
    for (int r = r0; r < r1; r++) mine += __popc(s_bits[32 * r + lane]);
    mine = __reduce_add_sync(0xffffffffu, mine);
    if (lane == 0) s_warp[wid] = mine;
    __syncthreads();
    int at = done;
    for (int w = 0; w < kThreads / 32; w++) {
      at += w < wid ? s_warp[w] : 0;
      done += s_warp[w];
    }
    for (int r = r0; r < r1; r++) {
      uint32_t bits = s_bits[32 * r + lane];
      const int c = __popc(bits);
      int inc = c;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
      }
      const uint32_t key = first + (uint32_t)k0 + 32u * (uint32_t)(32 * r + lane);
      for (int p = at + inc - c; bits; bits &= bits - 1)
        out[p++] = key + (uint32_t)(__ffs(bits) - 1);
      at += __shfl_sync(0xffffffffu, inc, 31);
    }
  }
  __syncthreads();
  if (out != seg)
    for (int i = t; i < len; i += kThreads) seg[i] = spare[i];
  __syncthreads();
}

// Segment sort: one warp per tile for lists of up to 512 (bitonic network in
// registers), the block for its longer ones, one after another; TPB tiles per
// block (8, or 1 with few tiles, whose lists may all be long), a grid apart:
// long lists come in neighbouring tiles (batches with a dense clip: 80 to 90 us
// with eight neighbours in a block, 25 to 34 so).  Also places
// the tile in the render queue: after all tiles of longer classes, at the
// next free position of its class.  A list longer than kLongMax is reported as
// over capacity: its tile is emptied and the entry count is zeroed so that no
// gradient is reduced from this binning.
template <bool LAZY, int TPB>
__global__ void __launch_bounds__(kThreads) k_sort(const __grid_constant__ BinArgs a) {
  pdl_begin();
  extern __shared__ uint32_t s_keys[];  // kSmemKeys
  __shared__ int s_len[TPB];
  if (LAZY && a.hdr->lists_valid) return;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int tile = wid * gridDim.x + blockIdx.x;
  if (wid < TPB) {
    int len = 0;
    if (tile < a.num_tiles) {
      const int2 rg = a.ranges[tile];
      len = rg.y - rg.x;
      // queue position: the tiles of all longer classes, then the rank in its own
      const uint32_t rk = a.rank[tile];
      const int cls = (int)(rk >> 28);
      int x = lane < kBuckets && lane > cls ? a.bucket[lane] : 0;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
      if (lane == 0) {
        if (!a.one_scan) {  // (a one-block scan has cleared them)
          a.tile_cnt[tile] = 0;
          if (LAZY) a.tile_cnt2[tile] = 0;
        }
        const int q = x + (int)(rk & 0x0fffffffu);
        if (q < a.num_tiles)
          a.order[q] = tile;
        else
          set_status(a.hdr, GS2D_ERR_BOUNDS);  // class sizes out of step with the ranks
      }
      uint32_t* seg = a.list + rg.x;
      if (len <= 1) {
      } else if (len <= 32) {
        warp_sort_list<1>(seg, len, lane);
      } else if (len <= 64) {
        warp_sort_list<2>(seg, len, lane);
      } else if (len <= 128) {
        warp_sort_list<4>(seg, len, lane);
      } else if (len <= 256) {
        warp_sort_list<8>(seg, len, lane);
      } else if (len <= 512) {
        warp_sort_list<16>(seg, len, lane);
      }
    }
    if (lane == 0) s_len[wid] = len;
  }
  __syncthreads();
#pragma unroll 1
  for (int w = 0; w < TPB; w++) {
    const int len = s_len[w], tl = w * gridDim.x + blockIdx.x;
    if (len <= 512) continue;
    const int x = a.ranges[tl].x;
    if (len > kLongMax) {
      __syncthreads();  // every thread has read the range
      if (threadIdx.x == 0) {
        atomicCAS(&a.hdr->status, 0, (int)GS2D_ERR_CAPACITY);
        a.hdr->n_entries = 0;
        a.ranges[tl] = make_int2(x, x);
      }
      continue;
    }
    // one pass is always the faster way; each further one costs about what
    // 1024 keys cost the networks (8 M Gaussians, 31 passes: 32 768 keys 742 us
    // against 857, 20 000 keys 595 against 555)
    const gs2d_clip cl = clip_of_tile(a.cs, tl);
    if ((cl.n - 1) / kBitKeys <= len / 1024)
      block_sort_bits(a.list + x, len, (uint32_t)cl.g_off, cl.n, a.spare + x, s_keys);
    else
      block_sort_long(a.list + x, len, a.spare + x, s_keys);
  }
}

// ---------------------------------------------------------------------------
// Every kernel of the chain starts with pdl_begin() and is launched with
// launch_pdl: each one's blocks become resident while its predecessor drains.
static BinArgs bin_args(const gs2d_plan& p, void* ws, const float* params) {
  BinArgs a;
  a.cs = clip_set(p, ws);
  a.n = p.n;
  a.num_tiles = p.num_tiles;
  a.tile_shift = tile_shift_of(p.tile);
  a.group = (p.n + kGroup - 1) / kGroup <= kManyGroups ? kGroup : kGroupLarge;
  a.groups = (p.n + a.group - 1) / a.group;
  a.one_scan = p.num_tiles <= kOneScan && a.groups <= kOneScan;
  a.max_entries = p.max_entries;
  a.sigma_cut = p.cfg.sigma_cut;
  a.alpha_min = p.cfg.alpha_min;
  a.det_eps = p.cfg.det_eps;
  a.margin = p.cfg.bin_margin;
  a.params = params;
  a.rec = ws_ptr<float4>(ws, p, kOffRec);
  a.rect = ws_ptr<int4>(ws, p, kOffRect);
  a.lrect = ws_ptr<int4>(ws, p, kOffLRect);
  a.offs = ws_ptr<int>(ws, p, kOffCount);
  a.tile_cnt = ws_ptr<int>(ws, p, kOffTileCnt);
  a.tile_cnt2 = ws_ptr<int>(ws, p, kOffTileCnt2);
  a.sums = ws_ptr<long long>(ws, p, kOffBlockSum);
  a.cursor = ws_ptr<int>(ws, p, kOffCursor);
  a.ranges = ws_ptr<int2>(ws, p, kOffRanges);
  a.bucket = ws_ptr<int>(ws, p, kOffBucket);
  a.rank = ws_ptr<uint32_t>(ws, p, kOffRank);
  a.order = ws_ptr<int>(ws, p, kOffOrder);
  a.list = ws_ptr<uint32_t>(ws, p, kOffList);
  a.spare = ws_ptr<uint32_t>(ws, p, kOffPartial);
  a.hdr = ws_ptr<WsHeader>(ws, p, kOffHeader);
  return a;
}

static AdamTick adam_tick(const gs2d_plan& p, bool on) {
  return AdamTick{on ? 1 : 0, p.cfg.beta1, p.cfg.beta2, p.cfg.lr, p.cfg.lr_decay};
}

cudaError_t launch_project(const gs2d_plan& p, void* ws, const float* params, cudaStream_t s) {
  if (p.n == 0) return cudaSuccess;
  return launch_pdl(k_project, (p.n + kThreads - 1) / kThreads, kThreads, 0, s, p.n,
                    clip_set(p, ws), tile_shift_of(p.tile), p.cfg.sigma_cut, p.cfg.alpha_min,
                    p.cfg.det_eps, params, ws_ptr<float4>(ws, p, kOffRec),
                    ws_ptr<int4>(ws, p, kOffRect));
}

// Counts, scans, scatter and segment sorts.  LAZY modes return at once while
// hdr->lists_valid is set.
template <CountMode MODE>
static cudaError_t launch_bin(const BinArgs& a, AdamTick tick, cudaStream_t s) {
  constexpr bool kLazy = MODE == kCountRebin;
  const int blocks = std::max(1, a.groups);
  // where the scan leaves the groups' first entries: in place, or behind the sums
  long long* first = a.one_scan ? a.sums : a.sums + 2 * (size_t)a.groups;
  cudaError_t e = launch_pdl(k_count<MODE>, blocks, kThreads, 0, s, a, tick);
  if (e == cudaSuccess && !a.one_scan)
    e = launch_pdl(k_bin_scan<kLazy>,
                   1 + (a.num_tiles + kThreads * kTileItems - 1) / (kThreads * kTileItems),
                   kThreads, 0, s, a, first);
  if (e == cudaSuccess && a.n > 0)
    e = launch_pdl(k_bin_scatter<kLazy>, blocks, kThreads, 0, s, a, (const long long*)first);
  if (e != cudaSuccess) return e;
  // a block for each tile where there are few (eight per block would leave most
  // SMs idle), or where most lists are too long for a warp: 300 000 Gaussians in
  // 920 tiles, lists of about 700: 217 us in eights, 124 so
  if (a.num_tiles <= 152 * 4 || a.n / 256 >= a.num_tiles)
    return launch_pdl(k_sort<kLazy, 1>, a.num_tiles, kThreads, kSmemKeys * 4, s, a);
  // The blocks are launched while the scatter drains, and an SM must drain first
  // to give them its shared memory: the first SMs to do so take all they can hold.
  // With lists of some length each block asks for its SM's share instead (140 000
  // Gaussians in 920 tiles, lists of about 325: 115 blocks on some 23 SMs took 23
  // us, 7.5 so); waiting for more SMs to drain costs 1.5 us, which short lists do
  // not bring back (4000 Gaussians there).
  const int grid = (a.num_tiles + 7) / 8, per_sm = (grid + 151) / 152;
  const int smem = per_sm >= 6 || a.n / 32 < a.num_tiles ? kSmemKeys * 4
                                                         : (226 * 1024) / per_sm - 2048;
  e = opt_in_smem((const void*)k_sort<kLazy, 8>, smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(k_sort<kLazy, 8>, grid, kThreads, smem, s, a);
}

cudaError_t launch_bin_sort(const gs2d_plan& p, void* ws, cudaStream_t s) {
  return launch_bin<kCountRects>(bin_args(p, ws, nullptr), adam_tick(p, false), s);
}

cudaError_t launch_prepare(const gs2d_plan& p, void* ws, const float* params, bool tick,
                           cudaStream_t s) {
  return launch_bin<kCountProject>(bin_args(p, ws, params), adam_tick(p, tick), s);
}

cudaError_t launch_prepare_fit(const gs2d_plan& p, void* ws, const float* params,
                               cudaStream_t s) {
  if (!fit_lists_retained(p.cfg)) return launch_prepare(p, ws, params, true, s);
  const BinArgs a = bin_args(p, ws, params);
  const AdamTick tick = adam_tick(p, true);
  const cudaError_t e = launch_pdl(k_project_fit, std::max(1, (p.n + 127) / 128), 128, 0, s, a,
                                   tick);
  if (e != cudaSuccess) return e;
  return launch_bin<kCountRebin>(a, tick, s);
}

}  // namespace gs2d
