// Weight gradient of a 3 x 3, stride-2, pad-1 convolution straight from its
// input (tcgen05), the learned initialiser's backward pass:
//
//   dW[co][(3 ky + kx) C + ci] = sum over output pixels p of
//                                dZ[p][co] X[2 oy + ky - 1][2 ox + kx - 1][ci]
//   dW[co][9 C]                = sum over p of dZ[p][co]  (the bias), zeros beyond
//
// i.e. gs2d_gemm_tn_bf16 of dZ and the im2col operand, which is neither
// written nor read: at 1080p, batch 8, that operand is 1.6 GB for the first
// three layers, most of 0.79 ms of gs2d_im2col per training step.
//
// Both operands are MN-major as in csrc/gemm_tn.cu: a row is a pixel, its
// channels lie contiguously.  A k-step is up to 128 output pixels of one row.
// For a fixed tap their inputs are every second pixel of an input row, so one
// TMA box brings a tap's channels.  With an even width, X is read as pairs of
// pixels [2 ox, 2 ox + 1] of 2 C channels: taps kx = 1 and 2 are the two halves
// of pair ox, kx = 0 the second half of pair ox - 1, and no box steps along W.
// Three forms:
//   C = 64 j:  boxes of 64 channels of a tap, three of them a tile's columns
//              (odd widths: a traversal stride of 2 along W instead of pairs);
//   C = 32:    all taps in a tile: per ky the pair (64 columns) and the second
//              half of the pair before it (32 columns, 64-byte swizzle);
//   C = 8:     all taps in a tile: per ky the pair (16 columns, 32-byte
//              swizzle) and the pair before it, whose first half is dropped.
// The bias column comes from a constant block of ones.
//
// What bounds it is the staging of dZ and the taps (each input pixel is read
// 2.25 times, but from DRAM once).  Against im2col and gs2d_gemm_tn_bf16 in every
// layer the training step went from 2.84 to 2.46 ms at 1080p, batch 8, where the
// first three layers run here and the last two (120 and 60 pixels a row) there.
//
// Splits, ring, waits and epilogue as in csrc/gemm_tn.cu.  Output rows are
// multiples of 16 pixels (of at least 64), so that the tensor core adds the same
// 16 pixels at a time, in the same order, as over the operand: the result is
// that of the GEMM bit for bit (why that matters: csrc/gemm_tn.cu).
#include <cuda.h>
#include <cuda_bf16.h>
#include <stdio.h>

#include <algorithm>

#include "gs2d_internal.cuh"
#include "tc_gemm.cuh"
#include "tc_ptx.cuh"

namespace gs2d {
namespace {

constexpr int kWgRows = 128;  // pixels per stage
constexpr int kWgOnes = 2048;  // 16 rows of 64 columns, column 0 all ones

struct WgArgs {
  int M, C, ldc;               // output channels, input channels, dW's leading dimension
  int Ho, Wo, pixels, per;     // dZ's rows and columns, all pixels, 64-pixel tiles of a split
  int pairs, cpt;              // X as pixel pairs; 64-channel chunks per tap (C = 64 j)
  size_t split_stride;
  float* out;  // partials, or the result when there is one split
  int* status;
};

// CM: the form (64, 32 or 8 channels); NA boxes of AC columns of dZ.
template <int CM, int NA, int AC>
struct WgShape {
  static constexpr int kABox = AC * kWgRows * 2;
  static constexpr int kPairBox = (CM == 64 ? 64 : 2 * CM) * kWgRows * 2;  // (C = 64 j: a chunk)
  static constexpr int kShiftCols = CM == 32 ? 32 : 16;
  static constexpr int kShiftBox = CM == 64 ? 0 : kShiftCols * kWgRows * 2;
  static constexpr int kBN = CM == 64 ? 192 : CM == 32 ? 288 : 96;
  static constexpr int kTmemCols = CM == 64 ? 256 : CM == 32 ? 512 : 128;
  static constexpr int kStageBytes = NA * kABox + 3 * (kPairBox + kShiftBox);
  static constexpr int kStages = std::min(6, (208 * 1024) / kStageBytes);
  static constexpr int kSmem = kStages * kStageBytes + kWgOnes + 1024;
};

template <int CM, int NA, int AC>
__global__ void __launch_bounds__(128, 1)
k_conv_wgrad(const __grid_constant__ CUtensorMap ta, const __grid_constant__ CUtensorMap tb,
             const __grid_constant__ CUtensorMap ts, WgArgs g) {
  using Sh = WgShape<CM, NA, AC>;
  constexpr int ST = Sh::kStages;
  pdl_begin();
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full[ST], empty[ST], accum;
  __shared__ uint32_t s_tmem;
  __shared__ int s_fail;
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~uintptr_t(1023));
  uint8_t* ones = smem + ST * Sh::kStageBytes;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m0 = blockIdx.x * AC * NA, nt = blockIdx.y;
  const int64_t first = (int64_t)blockIdx.z * g.per * 64;
  const int px = (int)min((int64_t)g.pixels - first, (int64_t)g.per * 64);  // >= 16 (host)
  const int row0 = (int)first / g.Wo, ox0 = (int)first - row0 * g.Wo;
  const bool bias = nt == 0;  // this tile brings the columns from 9 C on

  if (threadIdx.x == 0) {
    for (int s = 0; s < ST; s++) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(&accum, 1);
    s_fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // the ones: a 16-byte vector per thread, vector 0 of each 128-byte row being
  // swizzled to position row % 8
  {
    const int row = threadIdx.x >> 3, v = threadIdx.x & 7;
    *reinterpret_cast<uint4*>(ones + row * 128 + 16 * v) =
        make_uint4(v == (row & 7) ? 0x3F80u : 0u, 0u, 0u, 0u);
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&s_tmem)),
                 "r"(Sh::kTmemCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s_tmem;

  if (warp == 0 && lane == 0) {
    // the tile's three boxes: channel, column and row of their inputs, and how
    // these move with ox and oy
    int c0[3], w0[3], h0[3];
    const int wmul = CM == 64 && !g.pairs ? 2 : 1;
#pragma unroll
    for (int k = 0; k < 3; k++) {
      if constexpr (CM == 64) {
        const int chunk = 3 * nt + k, tap = chunk / g.cpt, q = chunk - tap * g.cpt;
        const int ky = tap / 3, kx = tap - 3 * ky;
        c0[k] = 64 * q + (g.pairs && kx != 1 ? g.C : 0);
        w0[k] = g.pairs ? (kx == 0 ? -1 : 0) : kx - 1;
        h0[k] = ky - 1;
      } else {
        c0[k] = 0;
        w0[k] = 0;
        h0[k] = k - 1;
      }
    }
    int b = row0 / g.Ho, oy = row0 - b * g.Ho, ox = ox0;
    int issued = 0;
    for (int left = px; left > 0; issued++) {
      const int s = issued % ST;
      if (!mbar_wait(&empty[s], ((uint32_t)(issued / ST) & 1u) ^ 1u)) {
        s_fail = 1;
        break;
      }
      uint8_t* st = smem + s * Sh::kStageBytes;
      mbar_expect_tx(&full[s], (uint32_t)Sh::kStageBytes);
#pragma unroll
      for (int k = 0; k < NA; k++)
        tma_load_4d(st + k * Sh::kABox, &ta, &full[s], m0 + AC * k, ox, oy, b);
      st += NA * Sh::kABox;
#pragma unroll
      for (int k = 0; k < 3; k++)
        tma_load_4d(st + k * Sh::kPairBox, &tb, &full[s], c0[k], wmul * ox + w0[k],
                    2 * oy + h0[k], b);
      if constexpr (CM != 64) {
        st += 3 * Sh::kPairBox;
#pragma unroll
        for (int k = 0; k < 3; k++)
          tma_load_4d(st + k * Sh::kShiftBox, &ts, &full[s], CM == 32 ? 32 : 0, ox - 1,
                      2 * oy + h0[k], b);
      }
      const int n = min(min(kWgRows, left), g.Wo - ox);
      left -= n;
      ox += n;
      if (ox == g.Wo) {
        ox = 0;
        if (++oy == g.Ho) {
          oy = 0;
          b++;
        }
      }
    }
    // no copy of this CTA is in flight when it leaves
    for (int i = issued > ST ? issued - ST : 0; i < issued; i++)
      if (!mbar_wait(&full[i % ST], (uint32_t)(i / ST) & 1u)) s_fail = 1;
  } else if (warp == 1 && lane == 0) {
    const uint64_t od = mn_major_desc(smem_u32(ones), 0, 128);
    int ox = ox0;
    for (int i = 0, left = px; left > 0; i++) {
      const int s = i % ST;
      if (!mbar_wait(&full[s], (uint32_t)(i / ST) & 1u)) {
        s_fail = 1;
        break;
      }
      tc_fence_after();
      const int n = min(min(kWgRows, left), g.Wo - ox);  // a multiple of 16
      left -= n;
      ox = ox + n == g.Wo ? 0 : ox + n;
      const uint32_t a_s = smem_u32(smem + s * Sh::kStageBytes), b_s = a_s + NA * Sh::kABox;
      // one A box: the other rows of the tile read the same columns again
      const uint64_t ad = mn_major_desc(a_s, NA > 1 ? Sh::kABox : 0, 2 * AC);
      const uint64_t bd = mn_major_desc(b_s, Sh::kPairBox, CM == 8 ? 32 : 128);
      const uint64_t sd = mn_major_desc(b_s + 3 * Sh::kPairBox, Sh::kShiftBox, 64);
#pragma unroll 2
      for (int kk = 0; kk < n / 16; kk++) {  // 16 rows, in units of 16 bytes
        const uint32_t acc = (i > 0 || kk > 0) ? 1u : 0u;
        const uint64_t a = ad + 2 * AC * kk;
        if constexpr (CM == 8) {  // six boxes of 16 columns
          mma_bf16(tmem, a, bd + 32 * kk, idesc_bf16_mn(kBM, 96), acc);
        } else {
          mma_bf16(tmem, a, bd + 128 * kk, idesc_bf16_mn(kBM, 192), acc);
          if constexpr (CM == 32)
            mma_bf16(tmem + 192, a, sd + 64 * kk, idesc_bf16_mn(kBM, 96), acc);
        }
        if (bias) mma_bf16(tmem + Sh::kBN, a, od, idesc_bf16_mn(kBM, 16), acc);
      }
      mma_commit(&empty[s]);
    }
    mma_commit(&accum);
  }
  __syncwarp();

  const bool ready = mbar_wait(&accum, 0);
  tc_fence_after();
  if (!ready) s_fail = 1;
  __syncthreads();
  if (!s_fail && warp < (NA * AC + 31) / 32) {
    const int row = m0 + warp * 32 + lane;
    const bool valid = row < g.M;
    float* out = g.out + (size_t)blockIdx.z * g.split_stride + (size_t)row * g.ldc;
    const uint32_t taddr = tmem + ((uint32_t)(warp * 32) << 16);
    const bool vec_ok = (g.ldc % 4) == 0 && (reinterpret_cast<uintptr_t>(g.out) & 15) == 0 &&
                        g.split_stride % 4 == 0;
    const int C = CM == 64 ? g.C : CM;
    // eight columns of an accumulator to columns n ... of dW
    const auto store8 = [&](const float* v, int n) {
      if (vec_ok) {
        *reinterpret_cast<float4*>(out + n) = make_float4(v[0], v[1], v[2], v[3]);
        *reinterpret_cast<float4*>(out + n + 4) = make_float4(v[4], v[5], v[6], v[7]);
      } else {
#pragma unroll
        for (int j = 0; j < 8; j++) out[n + j] = v[j];
      }
    };
#pragma unroll 1
    for (int c = 0; c < Sh::kBN; c += 16) {
      float v[16];
      tmem_ld16(taddr + (uint32_t)c, v);
      if (!valid) {
      } else if constexpr (CM == 64) {
        store8(v, 192 * nt + c);
        store8(v + 8, 192 * nt + c + 8);
      } else {
        constexpr int kPairs = 6 * CM, kPair = 2 * CM;
        if (c < kPairs) {  // kx = 1 and 2
          const int ky = c / kPair, n = (3 * ky + 1) * C + c - ky * kPair;
          store8(v, n);
          store8(v + 8, n + 8);
        } else {  // kx = 0 (C = 8: the second half of the box)
          const int d = c - kPairs, ky = d / Sh::kShiftCols, n = 3 * ky * C + d % Sh::kShiftCols;
          if constexpr (CM == 8) {
            store8(v + 8, n);
          } else {
            store8(v, n);
            store8(v + 8, n + 8);
          }
        }
      }
    }
    if (bias) {
      float v[16];
      tmem_ld16(taddr + (uint32_t)Sh::kBN, v);
      // (columns 1 ... 15 of the ones block are zero; so is what lies beyond)
      if (valid) {
        for (int n = 9 * C; n < g.ldc; n++) out[n] = 0.0f;
        out[9 * C] = v[0];
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(Sh::kTmemCols));
  if (threadIdx.x == 0 && s_fail && g.status) atomicCAS(g.status, 0, (int)GS2D_ERR_TIMEOUT);
}

// 4D map of an NHWC tensor [B][H][W][C]: boxes of `cols` channels x 128 pixels
// of a row, stepping sw along it; zeros out of range.
bool wg_map(CUtensorMap* map, const void* x, int B, int H, int W, int C, int64_t row_bytes,
            int cols, int sw) {
  EncodeTiled fn = tensor_map_encoder();
  if (!fn) return false;
  const cuuint64_t dims[4] = {(cuuint64_t)C, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)B};
  const cuuint64_t strides[3] = {(cuuint64_t)C * 2, (cuuint64_t)row_bytes,
                                 (cuuint64_t)row_bytes * H};
  const cuuint32_t box[4] = {(cuuint32_t)cols, (cuuint32_t)(kWgRows * sw), 1, 1};
  const cuuint32_t estr[4] = {1, (cuuint32_t)sw, 1, 1};
  const CUtensorMapSwizzle swz = cols == 16   ? CU_TENSOR_MAP_SWIZZLE_32B
                                 : cols == 32 ? CU_TENSOR_MAP_SWIZZLE_64B
                                              : CU_TENSOR_MAP_SWIZZLE_128B;
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(x), dims, strides, box,
            estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swz, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The form of one product: 64, 32, 8, or 0 when there is none for it.
int wg_form(int Wi, int C, int N) {
  const int Wo = (Wi + 1) / 2;
  if (Wo < 64 || Wo % 16) return 0;
  if (C % 64 == 0) return 64;
  if (Wi % 2) return 0;
  return C == 32 ? 32 : C == 8 && N <= 64 ? 8 : 0;
}

struct WgPlan {
  int form, na, ac, mt, nt;
  TnSplit sp;
};

WgPlan wg_plan(int B, int Hi, int Wi, int C, int N, int splits) {
  WgPlan p;
  p.form = wg_form(Wi, C, N);
  p.ac = p.form == 8 && N <= 32 ? 32 : 64;
  p.na = N <= 64 ? 1 : 2;
  p.mt = (N + p.ac * p.na - 1) / (p.ac * p.na);
  p.nt = p.form == 64 ? 9 * (C / 64) / 3 : 1;
  p.sp = tn_split((int64_t)B * ((Hi + 1) / 2) * ((Wi + 1) / 2), splits);
  return p;
}

bool wg_sizes(int B, int Hi, int Wi, int C, int N, int ldc) {
  return B >= 1 && Hi >= 1 && Wi >= 1 && C >= 8 && C <= 1 << 20 && C % 8 == 0 && N >= 8 &&
         N % 8 == 0 && ldc >= 9 * (int64_t)C + 1 && wg_form(Wi, C, N) != 0 &&
         (int64_t)B * ((Hi + 1) / 2) * ((Wi + 1) / 2 + kWgRows) <= INT32_MAX &&
         (int64_t)N * ldc <= INT32_MAX;
}

template <int CM, int NA, int AC>
cudaError_t launch_wgrad(const CUtensorMap& ta, const CUtensorMap& tb, const CUtensorMap& ts,
                         const WgArgs& g, dim3 grid, cudaStream_t s) {
  using Sh = WgShape<CM, NA, AC>;
  static_assert(Sh::kSmem + 256 <= 227 * 1024, "shared memory of a CTA");
  const cudaError_t e = opt_in_smem((const void*)k_conv_wgrad<CM, NA, AC>, Sh::kSmem);
  if (e != cudaSuccess) return e;
  return launch_pdl(k_conv_wgrad<CM, NA, AC>, grid, 128, Sh::kSmem, s, ta, tb, ts, g);
}

}  // namespace
}  // namespace gs2d

using namespace gs2d;

extern "C" int32_t gs2d_conv_wgrad_supported(int32_t B, int32_t Hi, int32_t Wi, int32_t C,
                                             int32_t N) {
  return wg_sizes(B, Hi, Wi, C, N, C <= 1 << 20 ? 9 * C + 1 : 0) ? 1 : 0;
}

extern "C" uint64_t gs2d_conv_wgrad_partial_bytes(int32_t B, int32_t Hi, int32_t Wi, int32_t C,
                                                  int32_t N, int32_t ldc, int32_t splits) {
  if (!wg_sizes(B, Hi, Wi, C, N, ldc)) return 0;
  const WgPlan p = wg_plan(B, Hi, Wi, C, N, splits);
  return p.sp.splits > 1 ? (uint64_t)p.sp.splits * N * ldc * sizeof(float) : 0;
}

extern "C" gs2d_status gs2d_conv_wgrad_bf16(const void* dz, int32_t N, const void* x, int32_t B,
                                            int32_t Hi, int32_t Wi, int32_t C, float* out,
                                            int32_t ldc, int32_t splits, float* partial,
                                            int32_t* status, void* stream) {
  if (!wg_sizes(B, Hi, Wi, C, N, ldc))
    return set_error(GS2D_ERR_INVALID_ARG, "gs2d_conv_wgrad_bf16: sizes");
  if (!dz || !x || !out || ((uintptr_t)dz & 15) || ((uintptr_t)x & 15))
    return set_error(GS2D_ERR_INVALID_ARG, "gs2d_conv_wgrad_bf16: NULL or misaligned operand");
  const WgPlan p = wg_plan(B, Hi, Wi, C, N, splits);
  if (p.sp.splits > 1 && !partial)
    return set_error(GS2D_ERR_INVALID_ARG, "gs2d_conv_wgrad_bf16: the split needs partial");
  const int Ho = (Hi + 1) / 2, Wo = (Wi + 1) / 2;
  WgArgs g;
  g.M = N;
  g.C = C;
  g.ldc = ldc;
  g.Ho = Ho;
  g.Wo = Wo;
  g.pixels = B * Ho * Wo;
  g.per = p.sp.per;
  g.pairs = Wi % 2 == 0;
  g.cpt = p.form == 64 ? C / 64 : 1;
  g.split_stride = p.sp.splits > 1 ? (size_t)N * ldc : 0;
  g.out = p.sp.splits > 1 ? partial : out;
  g.status = status;
  CUtensorMap ta, tb, ts;
  const int64_t row = (int64_t)Wi * C * 2;
  const int pc = g.pairs ? 2 * C : C, pwd = g.pairs ? Wi / 2 : Wi, sw = g.pairs ? 1 : 2;
  bool ok = wg_map(&ta, dz, B, Ho, Wo, N, (int64_t)Wo * N * 2, p.ac, 1) &&
            wg_map(&tb, x, B, Hi, pwd, pc, row, p.form == 64 ? 64 : 2 * p.form, sw);
  ts = tb;
  if (ok && p.form == 32) ok = wg_map(&ts, x, B, Hi, pwd, pc, row, 32, 1);
  if (!ok) return set_error(GS2D_ERR_CUDA, "gs2d_conv_wgrad_bf16: tensor map");
  const dim3 grid(p.mt, p.nt, p.sp.splits);
  cudaStream_t s = (cudaStream_t)stream;
  cudaError_t e = p.form == 64 ? (p.na == 1 ? launch_wgrad<64, 1, 64>(ta, tb, ts, g, grid, s)
                                            : launch_wgrad<64, 2, 64>(ta, tb, ts, g, grid, s))
                  : p.form == 32 ? (p.na == 1 ? launch_wgrad<32, 1, 64>(ta, tb, ts, g, grid, s)
                                              : launch_wgrad<32, 2, 64>(ta, tb, ts, g, grid, s))
                  : p.ac == 32   ? launch_wgrad<8, 1, 32>(ta, tb, ts, g, grid, s)
                                 : launch_wgrad<8, 1, 64>(ta, tb, ts, g, grid, s);
  if (e == cudaSuccess && p.sp.splits > 1)
    e = launch_tn_reduce(N, ldc, ldc, p.sp.splits, g.split_stride, partial, out, s);
  if (e != cudaSuccess) {
    char msg[200];
    snprintf(msg, sizeof(msg), "gs2d_conv_wgrad_bf16: %s", cudaGetErrorString(e));
    return set_error(GS2D_ERR_CUDA, msg);
  }
  return set_error(GS2D_OK, "");
}
