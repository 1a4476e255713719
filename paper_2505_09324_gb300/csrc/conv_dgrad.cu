// Input gradient of a 3 x 3, stride-2, pad-1 convolution as an implicit GEMM
// on the tensor cores (tcgen05), the learned initialiser's backward pass:
//
//   dx[iy][ix][ci] = (act > 0) sum over taps (ky, kx) that read (iy, ix), co
//                    dZ[oy][ox][co] W[co][(3 ky + kx) C + ci]
//
// A pixel is read by one, two or four taps, by the parity of its row and
// column: with iy = 2 a + py, ix = 2 c + px the four classes (py, px) sum over
// dZ at (a, c), (a, c + 1), (a + 1, c) and (a + 1, c + 1) only.  So a tile is
// 128 columns c of one row a, i.e. 2 x 256 input pixels: four accumulators
// (one per class) of C columns, and per 64 output channels four dZ boxes, each
// shifted by a row or a column (one TMA box; zeros past the edge), with the
// nine taps' weights:
//   (a, c):     taps 11, 12, 21, 22 -> classes 00, 01, 10, 11
//   (a, c + 1): taps 10, 20 -> 01, 11     (a + 1, c): taps 01, 02 -> 10, 11
//   (a + 1, c + 1): tap 00 -> 11
// What bounds it is the traffic of dZ, act and dx (0.66 GB for the widest
// layer at 1080p, batch 8).  The GEMM to an FP32 im2col gradient and the
// gather after it moved 4.6 GB more per training step: 1.65 ms for the three
// widest layers, 0.51 ms here (266, 140 and 101 us).
//
// A persistent CTA per SM: warp 0, one lane, brings the boxes into a ring;
// the weights stay in shared memory when they fit, else each stage has room
// for the (up to four) weight boxes of its dZ box.  Warp 1, one lane, issues
// the MMAs; warps 2-9 (two per accumulator quarter, one per row parity) apply
// the mask, convert and store 16-byte vectors, overlapping the next tile where
// tensor memory holds more than one set of accumulators (C <= 64).  Every wait
// is bounded as in csrc/conv_tap.cu; the producer also waits (bounded) for its
// last copies before the CTA may leave.
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
  int segs, nblk, tiles, chunks;  // column segments, blocks of channels, tiles, 64-channel chunks
  int stages, resident, stage_bytes, bres_off;
  const __nv_bfloat16* act;
  __nv_bfloat16* dx;
  int* status;
};

template <int CI>
struct DgShape {
  static constexpr int kAcc = 128 / CI;      // sets of four accumulators: 4, 2, 1
  static constexpr int kSet = 4 * CI;        // TMEM columns of a set
  static constexpr int kBBytes = CI * 128;   // one tap's weights: CI rows of 64 channels
};

// The taps of dZ box v (0: (a, c), 1: (a, c + 1), 2: (a + 1, c), 3: both) and
// the classes they add to.
__device__ __forceinline__ int dg_taps(int v) { return v == 0 ? 4 : v == 3 ? 1 : 2; }
__device__ __forceinline__ int dg_tap(int v, int k) {
  constexpr uint32_t kTap[4] = {0x8754u, 0x63u, 0x21u, 0x0u};
  return (int)((kTap[v] >> (4 * k)) & 15u);
}
__device__ __forceinline__ int dg_class(int v, int k) {
  constexpr uint32_t kClass[4] = {0x3210u, 0x31u, 0x32u, 0x3u};
  return (int)((kClass[v] >> (4 * k)) & 15u);
}

__device__ __forceinline__ bool dg_failed(const int* flag) {
  return *reinterpret_cast<const volatile int*>(flag) != 0;
}

template <int CI>
__global__ void __launch_bounds__(kDgThreads, 1)
k_conv_dgrad(const __grid_constant__ CUtensorMap ta, const __grid_constant__ CUtensorMap tb,
             DgArgs g) {
  using Sh = DgShape<CI>;
  pdl_begin();
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full[kDgStages], empty[kDgStages];
  __shared__ __align__(8) uint64_t acc_full[Sh::kAcc], acc_empty[Sh::kAcc], bres_full;
  __shared__ uint32_t s_tmem;
  __shared__ int s_fail;
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~uintptr_t(1023));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int ST = g.stages;

  if (threadIdx.x == 0) {
    for (int s = 0; s < ST; s++) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < Sh::kAcc; a++) {
      mbar_init(&acc_full[a], 1);
      mbar_init(&acc_empty[a], 8);  // one arrival per epilogue warp
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
        mbar_expect_tx(&bres_full, (uint32_t)(9 * chunks * Sh::kBBytes));
        for (int q = 0; q < chunks; q++)
          for (int tap = 0; tap < 9; tap++)
            tma_load_2d(smem + g.bres_off + (9 * q + tap) * Sh::kBBytes, &tb, &bres_full, q * kBK,
                        tap * C);
      }
      int s = 0, issued = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int t = blockIdx.x; t < tiles && ok && !dg_failed(&s_fail); t += gridDim.x) {
        const int nb = t % g.nblk, u = t / g.nblk;
        const int row = u / g.segs, c0 = (u - row * g.segs) * kBM;
        const int b = row / g.Ho, a = row - b * g.Ho;
        for (int i = 0; i < 4 * chunks; i++) {
          const int q = i >> 2, v = i & 3;
          if (!mbar_wait(&empty[s], ph ^ 1u)) {
            ok = false;
            break;
          }
          uint8_t* st = smem + s * stage_bytes;
          const int nt = resident ? 0 : dg_taps(v);
          mbar_expect_tx(&full[s], (uint32_t)(kDgA + nt * Sh::kBBytes));
          tma_load_4d(st, &ta, &full[s], q * kBK, c0 + (v & 1), a + (v >> 1), b);
          for (int k = 0; k < nt; k++)
            tma_load_2d(st + kDgA + k * Sh::kBBytes, &tb, &full[s], q * kBK,
                        dg_tap(v, k) * C + nb * CI);
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
      constexpr uint32_t idesc = idesc_bf16(kBM, CI);
      const int chunks = g.chunks, tiles = g.tiles;
      const bool resident = g.resident != 0;
      bool ok = !resident || mbar_wait(&bres_full, 0);
      const uint64_t a0 = sw128_desc(smem_u32(smem));
      const uint64_t b0 = resident ? sw128_desc(smem_u32(smem + g.bres_off)) : a0 + (kDgA >> 4);
      const uint64_t stage_d = (uint64_t)(g.stage_bytes >> 4);
      constexpr uint64_t tap_d = Sh::kBBytes >> 4;
      int s = 0;
      uint32_t ph = 0, at = 0;
      for (int t = blockIdx.x; t < tiles && ok && !dg_failed(&s_fail); t += gridDim.x, at++) {
        const int acc = (int)(at % (uint32_t)Sh::kAcc);
        if (!mbar_wait(&acc_empty[acc], ((at / (uint32_t)Sh::kAcc) & 1u) ^ 1u)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t d = tmem + (uint32_t)(acc * Sh::kSet);
        for (int q = 0; q < chunks && ok; q++) {
#pragma unroll
          for (int v = 0; v < 4; v++) {
            if (!mbar_wait(&full[s], ph)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint64_t ad = a0 + (uint64_t)s * stage_d;
            // the first box of a tile touches every class first
            const uint32_t keep = q > 0 || v > 0;
#pragma unroll
            for (int k = 0; k < dg_taps(v); k++) {
              const uint64_t bd = resident
                                      ? b0 + (uint64_t)(9 * q + dg_tap(v, k)) * tap_d
                                      : b0 + (uint64_t)s * stage_d + (uint64_t)k * tap_d;
#pragma unroll
              for (int kk = 0; kk < kBK / 16; kk++)
                mma_bf16(d + (uint32_t)(dg_class(v, k) * CI), ad + 2 * kk, bd + 2 * kk, idesc,
                         kk > 0 ? 1u : keep);
            }
            mma_commit(&empty[s]);
            if (++s == ST) {
              s = 0;
              ph ^= 1u;
            }
          }
        }
        if (!ok) break;
        mma_commit(&acc_full[acc]);
      }
      if (!ok) s_fail = 1;
    }
  } else {
    // epilogue: TMEM lanes 32 (warp % 4) ..., row parity by the warp's group
    const int quarter = warp & 3, py = (warp - 2) >> 2, r = quarter * 32 + lane;
    uint32_t at = 0;
    for (int t = blockIdx.x; t < g.tiles; t += gridDim.x, at++) {
      const int acc = (int)(at % (uint32_t)Sh::kAcc);
      // (tcgen05.ld is warp-collective: the warp goes on only if every lane
      // saw the accumulators complete)
      if (!__all_sync(0xffffffffu, mbar_wait(&acc_full[acc], (at / (uint32_t)Sh::kAcc) & 1u))) {
        s_fail = 1;
        break;
      }
      tc_fence_after();
      const int nb = t % g.nblk, u = t / g.nblk;
      const int row = u / g.segs, c = (u - row * g.segs) * kBM + r;
      const int b = row / g.Ho, iy = 2 * (row - b * g.Ho) + py;
      const uint32_t taddr = tmem + (uint32_t)(acc * Sh::kSet + 2 * py * CI) +
                             ((uint32_t)(quarter * 32) << 16);
      if (iy < g.Hi) {
#pragma unroll 1
        for (int px = 0; px < 2; px++) {
          const int ix = 2 * c + px;
          const bool valid = ix < g.Wi;
          const size_t o = (((size_t)b * g.Hi + iy) * g.Wi + ix) * g.C + nb * CI;
#pragma unroll 1
          for (int c0 = 0; c0 < CI; c0 += 32) {
            float w[32];
            tmem_ld32(taddr + (uint32_t)(px * CI + c0), w);
            if (!valid) continue;
#pragma unroll
            for (int k = 0; k < 32; k += 8) {
              if (nb * CI + c0 + k >= g.C) break;
              if (g.act) {
                const uint4 av = *reinterpret_cast<const uint4*>(g.act + o + c0 + k);
                const __nv_bfloat16* ab = reinterpret_cast<const __nv_bfloat16*>(&av);
#pragma unroll
                for (int j = 0; j < 8; j++)
                  if (!(__bfloat162float(ab[j]) > 0.0f)) w[k + j] = 0.0f;
              }
              __align__(16) __nv_bfloat162 h[4];
#pragma unroll
              for (int j = 0; j < 4; j++)
                h[j] = __floats2bfloat162_rn(w[k + 2 * j], w[k + 2 * j + 1]);
              *reinterpret_cast<uint4*>(g.dx + o + c0 + k) = *reinterpret_cast<const uint4*>(h);
            }
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&acc_empty[acc]);
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

template <int CI>
cudaError_t launch_dgrad(const CUtensorMap& ta, const CUtensorMap& tb, DgArgs g, cudaStream_t s) {
  const int bres = 9 * g.chunks * DgShape<CI>::kBBytes;
  // resident weights leave room for at least four dZ boxes
  g.resident = g.nblk == 1 && bres + 4 * kDgA + 1024 <= kDgBudget;
  g.stage_bytes = kDgA + (g.resident ? 0 : 4 * DgShape<CI>::kBBytes);
  const int fixed = (g.resident ? bres : 0) + 1024;  // + alignment slack
  g.stages = std::min(kDgStages, (kDgBudget - fixed) / g.stage_bytes);
  g.bres_off = g.stages * g.stage_bytes;
  const int smem = g.bres_off + fixed;
  cudaError_t e = opt_in_smem((const void*)k_conv_dgrad<CI>, smem);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0;
  e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  return launch_pdl(k_conv_dgrad<CI>, std::min(g.tiles, sms), kDgThreads, smem, s, ta, tb, g);
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
  const int ci = C <= 32 ? 32 : C <= 64 ? 64 : 128;
  g.segs = (g.Wo + kBM - 1) / kBM;
  g.nblk = (C + ci - 1) / ci;
  g.chunks = (N + kBK - 1) / kBK;
  const int64_t tiles = (int64_t)B * g.Ho * g.segs * g.nblk;
  if (tiles > INT32_MAX - 65536 || (int64_t)9 * C > INT32_MAX)
    return set_error(GS2D_ERR_INVALID_ARG, "gs2d_conv_dgrad_bf16: sizes");
  g.tiles = (int)tiles;
  g.act = static_cast<const __nv_bfloat16*>(act);
  g.dx = static_cast<__nv_bfloat16*>(dx);
  g.status = status;
  CUtensorMap ta, tb;
  if (!dg_map(&ta, dz, B, g.Ho, g.Wo, N) || !make_map(&tb, Wt, 9 * C, N, N, ci))
    return set_error(GS2D_ERR_CUDA, "gs2d_conv_dgrad_bf16: tensor map");
  cudaStream_t s = (cudaStream_t)stream;
  const cudaError_t e = ci == 32   ? launch_dgrad<32>(ta, tb, g, s)
                        : ci == 64 ? launch_dgrad<64>(ta, tb, g, s)
                                   : launch_dgrad<128>(ta, tb, g, s);
  if (e != cudaSuccess) {
    char msg[200];
    snprintf(msg, sizeof(msg), "gs2d_conv_dgrad_bf16: %s", cudaGetErrorString(e));
    return set_error(GS2D_ERR_CUDA, msg);
  }
  return set_error(GS2D_OK, "");
}
