// Input gradient of a 3 x 3, stride-2, pad-1 convolution as an implicit GEMM
// on the tensor cores (tcgen05), the learned initialiser's backward pass:
//
//   dx[iy][ix][ci] = (act > 0) sum over taps (ky, kx) that read (iy, ix), co
//                    dZ[oy][ox][co] W[co][(3 ky + kx) C + ci]
//
// A pixel is read by one, two or four taps, by the parity of its row and
// column: with iy = 2 a + py, ix = 2 c + px the four classes (py, px) sum over
// dZ at (a, c), (a, c + 1), (a + 1, c) and (a + 1, c + 1) only.  So a tile is
// 128 columns c of one row a, i.e. 2 x 256 input pixels, of 32 input channels;
// per 64 output channels it takes four dZ boxes, each shifted by a row or a
// column (one TMA box; zeros past the edge), and the nine taps' weights:
//   (a, c):     taps 11, 12, 21, 22 -> classes 00, 01, 10, 11
//   (a, c + 1): taps 10, 20 -> 01, 11     (a + 1, c): taps 01, 02 -> 10, 11
//   (a + 1, c + 1): tap 00 -> 11
// Each tap has its own accumulator, and the epilogue adds a pixel's taps in
// their order: bit for bit the FP32 sums of the GEMM to an im2col gradient
// with the gather after it (gs2d_gemm_bf16, gs2d_col2im).  One accumulator per
// class differed from them in the last FP32 bit, which the BF16 rounding of
// every layer below turned into relative differences of up to 6e-5 in the
// weight gradients of small frames.
// What bounds it is the traffic of dZ, act and dx (0.66 GB for the widest
// layer at 1080p, batch 8).  The GEMM and the gather moved 4.6 GB more per
// training step: 1.65 ms for the three widest layers, 0.47 ms here (0.54 with
// one accumulator per class and an epilogue that read the mask after its wait).
//
// A persistent CTA per SM, of one block of 32 channels: warp 0, one lane,
// brings the boxes into a ring; the weights stay in shared memory when they
// fit (up to 256 output channels), else each stage has room for the (up to
// four) weight boxes of its dZ box.  Warp 1, one lane, issues the MMAs; warps
// 2-9 (two per accumulator quarter, one per row parity) add the taps, mask,
// convert and store.  The mask of a tile is read before its accumulators are
// waited for, and they are given back before the stores, so both overlap the
// MMAs of the next tile.  Every wait is bounded as in csrc/conv_tap.cu; the
// producer also waits (bounded) for its last copies before the CTA may leave.
#include <cuda.h>
#include <cuda_bf16.h>
#include <stdio.h>

#include <algorithm>

#include "gs2d_internal.cuh"
#include "tc_gemm.cuh"
#include "tc_ptx.cuh"

namespace gs2d {
namespace {

constexpr int kDgThreads = 320;
constexpr int kDgStages = 8;
constexpr int kDgA = kBM * kBK * 2;  // a dZ box: 128 pixels x 64 channels, 16 KB
constexpr int kDgBudget = 226 * 1024;

struct DgArgs {
  int Hi, Wi, C, Ho, Wo;
  int segs, nblk, tiles, chunks;  // column segments, blocks of 32 channels, tiles of a block,
                                  // 64-channel chunks
  int stages, resident, stage_bytes, bres_off;
  const __nv_bfloat16* act;
  __nv_bfloat16* dx;
  int* status;
};

constexpr int kCI = 32;              // input channels of a tile
constexpr int kDgB = kCI * kBK * 2;  // one tap's weights: 32 rows of 64 channels, 4 KB

// The taps of dZ box v (0: (a, c), 1: (a, c + 1), 2: (a + 1, c), 3: both);
// taps 3, 4 and 5 are those of even rows.
__device__ __forceinline__ int dg_taps(int v) { return v == 0 ? 4 : v == 3 ? 1 : 2; }
__device__ __forceinline__ int dg_tap(int v, int k) {
  constexpr uint32_t kTap[4] = {0x8754u, 0x63u, 0x21u, 0x0u};
  return (int)((kTap[v] >> (4 * k)) & 15u);
}
// The first column of a tap's accumulator.
__device__ __forceinline__ uint32_t dg_col(int tap) { return (uint32_t)(tap * kCI); }

__device__ __forceinline__ bool dg_failed(const int* flag) {
  return *reinterpret_cast<const volatile int*>(flag) != 0;
}

__global__ void __launch_bounds__(kDgThreads, 1)
k_conv_dgrad(const __grid_constant__ CUtensorMap ta, const __grid_constant__ CUtensorMap tb,
             DgArgs g) {
  pdl_begin();
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full[kDgStages], empty[kDgStages];
  __shared__ __align__(8) uint64_t acc_full[2], acc_empty[2], bres_full;
  __shared__ uint32_t s_tmem;
  __shared__ int s_fail;
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~uintptr_t(1023));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int ST = g.stages;
  // this CTA's block of channels and its tiles of that block
  const int nb = (int)blockIdx.x % g.nblk, first = (int)blockIdx.x / g.nblk;
  const int step = (int)gridDim.x / g.nblk;

  if (threadIdx.x == 0) {
    for (int s = 0; s < ST; s++) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int py = 0; py < 2; py++) {  // the accumulators of even and of odd rows
      mbar_init(&acc_full[py], 1);
      mbar_init(&acc_empty[py], 4);  // one arrival per epilogue warp
    }
    mbar_init(&bres_full, 1);
    s_fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&s_tmem)),
                 "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s_tmem;

  if (warp == 0) {
    if (lane == 0) {
      const int C = g.C, chunks = g.chunks, tiles = g.tiles, stage_bytes = g.stage_bytes;
      const bool resident = g.resident != 0;
      if (resident) {
        mbar_expect_tx(&bres_full, (uint32_t)(9 * chunks * kDgB));
        for (int q = 0; q < chunks; q++)
          for (int tap = 0; tap < 9; tap++)
            tma_load_2d(smem + g.bres_off + (9 * q + tap) * kDgB, &tb, &bres_full, q * kBK,
                        tap * C + nb * kCI);
      }
      int s = 0, issued = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int t = first; t < tiles && ok && !dg_failed(&s_fail); t += step) {
        const int row = t / g.segs, c0 = (t - row * g.segs) * kBM;
        const int b = row / g.Ho, a = row - b * g.Ho;
        for (int i = 0; i < 4 * chunks; i++) {
          const int q = i >> 2, v = i & 3;
          if (!mbar_wait(&empty[s], ph ^ 1u)) {
            ok = false;
            break;
          }
          uint8_t* st = smem + s * stage_bytes;
          const int nt = resident ? 0 : dg_taps(v);
          mbar_expect_tx(&full[s], (uint32_t)(kDgA + nt * kDgB));
          tma_load_4d(st, &ta, &full[s], q * kBK, c0 + (v & 1), a + (v >> 1), b);
          for (int k = 0; k < nt; k++)
            tma_load_2d(st + kDgA + k * kDgB, &tb, &full[s], q * kBK,
                        dg_tap(v, k) * C + nb * kCI);
          issued++;
          if (++s == ST) {
            s = 0;
            ph ^= 1u;
          }
        }
      }
      // no copy of this CTA is in flight when it leaves
      for (int k = issued < ST ? issued : ST; k > 0; k--) {
        const int i = issued - k;
        if (!mbar_wait(&full[i % ST], (uint32_t)(i / ST) & 1u)) ok = false;
      }
      if (resident && !mbar_wait(&bres_full, 0)) ok = false;
      if (!ok) s_fail = 1;
    }
  } else if (warp == 1) {
    if (lane == 0) {
      constexpr uint32_t idesc = idesc_bf16(kBM, kCI);
      const int chunks = g.chunks, tiles = g.tiles;
      const bool resident = g.resident != 0;
      bool ok = !resident || mbar_wait(&bres_full, 0);
      const uint64_t a0 = sw128_desc(smem_u32(smem));
      const uint64_t b0 = resident ? sw128_desc(smem_u32(smem + g.bres_off)) : a0 + (kDgA >> 4);
      const uint64_t stage_d = (uint64_t)(g.stage_bytes >> 4);
      constexpr uint64_t tap_d = kDgB >> 4;
      int s = 0;
      uint32_t ph = 0, at = 0;
      for (int t = first; t < tiles && ok && !dg_failed(&s_fail); t += step, at++) {
        // (a fresh barrier passes the wait for the parity before its first)
        ok = mbar_wait(&acc_empty[0], (at & 1u) ^ 1u) && mbar_wait(&acc_empty[1], (at & 1u) ^ 1u);
        if (!ok) break;
        tc_fence_after();
        for (int q = 0; q < chunks && ok; q++) {
#pragma unroll
          for (int v = 0; v < 4; v++) {
            if (!mbar_wait(&full[s], ph)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint64_t ad = a0 + (uint64_t)s * stage_d;
#pragma unroll
            for (int k = 0; k < dg_taps(v); k++) {
              const int tap = dg_tap(v, k);
              const uint64_t bd = resident ? b0 + (uint64_t)(9 * q + tap) * tap_d
                                           : b0 + (uint64_t)s * stage_d + (uint64_t)k * tap_d;
#pragma unroll
              for (int kk = 0; kk < kBK / 16; kk++)
                mma_bf16(tmem + dg_col(tap), ad + 2 * kk, bd + 2 * kk, idesc,
                         q > 0 || kk > 0 ? 1u : 0u);
            }
            mma_commit(&empty[s]);
            // the even rows' taps end with box 1 of the last chunk
            if (v == 1 && q == chunks - 1) mma_commit(&acc_full[0]);
            if (++s == ST) {
              s = 0;
              ph ^= 1u;
            }
          }
        }
        if (!ok) break;
        mma_commit(&acc_full[1]);
      }
      if (!ok) s_fail = 1;
    }
  } else {
    // epilogue: TMEM lanes 32 (warp % 4) ..., row parity by the warp's group
    const int quarter = warp & 3, py = (warp - 2) >> 2, r = quarter * 32 + lane;
    const uint32_t taddr = tmem + ((uint32_t)(quarter * 32) << 16);
    const int cols = min(kCI, g.C - nb * kCI) / 8;  // 16-byte vectors of a pixel
    uint32_t at = 0;
    for (int t = first; t < g.tiles; t += step, at++) {
      const int row = t / g.segs, c = (t - row * g.segs) * kBM + r;
      const int b = row / g.Ho, oy = row - b * g.Ho, iy = 2 * oy + py;
      const bool in = iy < g.Hi;  // (the last odd row may be missing)
      const size_t o = (((size_t)b * g.Hi + iy) * g.Wi + 2 * c) * g.C + nb * kCI;
      // the mask of this lane's two pixels, a bit per channel
      uint32_t mask[2] = {0xffffffffu, 0xffffffffu};
      if (g.act) {
#pragma unroll
        for (int px = 0; px < 2; px++) {
          uint4 av[4];
#pragma unroll
          for (int k = 0; k < 4; k++)
            av[k] = in && 2 * c + px < g.Wi && k < cols
                        ? *reinterpret_cast<const uint4*>(g.act + o + px * g.C + 8 * k)
                        : make_uint4(0, 0, 0, 0);
          mask[px] = 0;
#pragma unroll
          for (int k = 0; k < 4; k++) {
            const uint32_t w[4] = {av[k].x, av[k].y, av[k].z, av[k].w};
#pragma unroll
            for (int i = 0; i < 4; i++) {
              const float lo = __uint_as_float(w[i] << 16);
              const float hi = __uint_as_float(w[i] & 0xffff0000u);
              mask[px] |= (lo > 0.0f ? 1u : 0u) << (8 * k + 2 * i);
              mask[px] |= (hi > 0.0f ? 2u : 0u) << (8 * k + 2 * i);
            }
          }
        }
      }
      // (tcgen05.ld is warp-collective: the warp goes on only if every lane
      // saw the accumulators complete)
      if (!__all_sync(0xffffffffu, mbar_wait(&acc_full[py], at & 1u))) {
        s_fail = 1;
        break;
      }
      tc_fence_after();
      // column parity px: taps ky x kx in their order, ky = 1 (even rows) or
      // 0, 2 (odd), kx = 1 (even columns) or 0, 2 (odd).  Taps past dZ's edge
      // (ky = 0 in the last row, kx = 0 in the last column) are left out, as by
      // the gather: their accumulators hold zeros times weights, which a
      // non-finite weight makes NaN
      const bool below = oy + 1 < g.Ho, right = c + 1 < g.Wo;
      uint32_t h[2][16];
#pragma unroll
      for (int px = 0; px < 2; px++) {
        float w[32], x[32];
        const auto add = [&](int tap, bool has) {
          tmem_ld32(taddr + dg_col(tap), x);
#pragma unroll
          for (int i = 0; i < 32; i++) w[i] = has ? w[i] + x[i] : w[i];
        };
        tmem_ld32(taddr + dg_col((py ? 0 : 3) + (px ? 0 : 1)), w);
        if (!((py == 0 || below) && (px == 0 || right))) {
#pragma unroll
          for (int i = 0; i < 32; i++) w[i] = 0.0f;
        }
        if (px) add((py ? 0 : 3) + 2, py == 0 || below);
        if (py) {
          add(6 + (px ? 0 : 1), px == 0 || right);
          if (px) add(8, true);
        }
#pragma unroll
        for (int i = 0; i < 16; i++) {
          const float lo = mask[px] >> (2 * i) & 1u ? w[2 * i] : 0.0f;
          const float hi = mask[px] >> (2 * i + 1) & 1u ? w[2 * i + 1] : 0.0f;
          const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
          h[px][i] = *reinterpret_cast<const uint32_t*>(&v);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&acc_empty[py]);
      if (!in) continue;
      // pairs of lanes exchange vectors, so that the two write a 32-byte
      // sector at a time: first the even lane's pixel, then the odd lane's
      const bool odd = lane & 1;
      const size_t oe = o - (odd ? 2 * (size_t)g.C : 0);
#pragma unroll
      for (int px = 0; px < 2; px++) {
        const int ix = 2 * (c - (odd ? 1 : 0)) + px;  // of the even lane
        __nv_bfloat16* const dst = g.dx + oe + (size_t)px * g.C;
#pragma unroll
        for (int k = 0; k < 4; k += 2) {
          uint32_t own[4], got[4];
#pragma unroll
          for (int i = 0; i < 4; i++) {
            own[i] = odd ? h[px][4 * (k + 1) + i] : h[px][4 * k + i];
            got[i] = __shfl_xor_sync(0xffffffffu, odd ? h[px][4 * k + i] : h[px][4 * (k + 1) + i],
                                     1);
          }
          const int kv = k + (odd ? 1 : 0);  // the vector this lane writes
          if (kv < cols) {
            const uint4 mine = make_uint4(own[0], own[1], own[2], own[3]);
            const uint4 other = make_uint4(got[0], got[1], got[2], got[3]);
            if (ix < g.Wi) *reinterpret_cast<uint4*>(dst + 8 * kv) = odd ? other : mine;
            if (ix + 2 < g.Wi)
              *reinterpret_cast<uint4*>(dst + 2 * (size_t)g.C + 8 * kv) = odd ? mine : other;
          }
        }
      }
    }
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
  if (threadIdx.x == 0 && s_fail && g.status) atomicCAS(g.status, 0, (int)GS2D_ERR_TIMEOUT);
}

// 4D map of an NHWC activation: boxes of 64 channels x 128 pixels of a row.
bool dg_map(CUtensorMap* map, const void* x, int B, int H, int W, int C) {
  EncodeTiled fn = tensor_map_encoder();
  if (!fn) return false;
  const cuuint64_t dims[4] = {(cuuint64_t)C, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)B};
  const cuuint64_t strides[3] = {(cuuint64_t)C * 2, (cuuint64_t)W * C * 2,
                                 (cuuint64_t)H * W * C * 2};
  const cuuint32_t box[4] = {(cuuint32_t)kBK, (cuuint32_t)kBM, 1, 1};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(x), dims, strides, box,
            estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

cudaError_t launch_dgrad(const CUtensorMap& ta, const CUtensorMap& tb, DgArgs g, cudaStream_t s) {
  const int bres = 9 * g.chunks * kDgB;
  // resident weights leave room for at least four dZ boxes
  g.resident = bres + 4 * kDgA + 1024 <= kDgBudget;
  g.stage_bytes = kDgA + (g.resident ? 0 : 4 * kDgB);
  const int fixed = (g.resident ? bres : 0) + 1024;  // + alignment slack
  g.stages = std::min(kDgStages, (kDgBudget - fixed) / g.stage_bytes);
  g.bres_off = g.stages * g.stage_bytes;
  const int smem = g.bres_off + fixed;
  cudaError_t e = opt_in_smem((const void*)k_conv_dgrad, smem);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0;
  e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  // a whole number of CTAs for each block of channels
  const int per = std::max(1, std::min(g.tiles, sms / g.nblk));
  return launch_pdl(k_conv_dgrad, per * g.nblk, kDgThreads, smem, s, ta, tb, g);
}

}  // namespace
}  // namespace gs2d

using namespace gs2d;

extern "C" gs2d_status gs2d_conv_dgrad_bf16(const void* dz, int32_t B, int32_t Hi, int32_t Wi,
                                            int32_t C, const void* Wt, int32_t N, const void* act,
                                            void* dx, int32_t* status, void* stream) {
  if (B < 0 || Hi < 1 || Wi < 1 || C < 8 || C % 8 || N < 8 || N % 8)
    return set_error(GS2D_ERR_INVALID_ARG, "gs2d_conv_dgrad_bf16: sizes");
  if (B == 0) return set_error(GS2D_OK, "");
  if (!dz || !Wt || !dx || ((uintptr_t)dz & 15) || ((uintptr_t)Wt & 15) || ((uintptr_t)act & 15) ||
      ((uintptr_t)dx & 15))
    return set_error(GS2D_ERR_INVALID_ARG, "gs2d_conv_dgrad_bf16: operands");
  DgArgs g;
  g.Hi = Hi;
  g.Wi = Wi;
  g.C = C;
  g.Ho = (Hi + 1) / 2;
  g.Wo = (Wi + 1) / 2;
  g.segs = (g.Wo + kBM - 1) / kBM;
  g.nblk = (C + kCI - 1) / kCI;
  g.chunks = (N + kBK - 1) / kBK;
  const int64_t tiles = (int64_t)B * g.Ho * g.segs;
  if (tiles > INT32_MAX - 65536 || (int64_t)9 * C > INT32_MAX)
    return set_error(GS2D_ERR_INVALID_ARG, "gs2d_conv_dgrad_bf16: sizes");
  g.tiles = (int)tiles;
  g.act = static_cast<const __nv_bfloat16*>(act);
  g.dx = static_cast<__nv_bfloat16*>(dx);
  g.status = status;
  CUtensorMap ta, tb;
  if (!dg_map(&ta, dz, B, g.Ho, g.Wo, N) || !make_map(&tb, Wt, 9 * C, N, N, kCI))
    return set_error(GS2D_ERR_CUDA, "gs2d_conv_dgrad_bf16: tensor map");
  cudaStream_t s = (cudaStream_t)stream;
  const cudaError_t e = launch_dgrad(ta, tb, g, s);
  if (e != cudaSuccess) {
    char msg[200];
    snprintf(msg, sizeof(msg), "gs2d_conv_dgrad_bf16: %s", cudaGetErrorString(e));
    return set_error(GS2D_ERR_CUDA, msg);
  }
  return set_error(GS2D_OK, "");
}
