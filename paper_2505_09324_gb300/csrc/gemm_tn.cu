// BF16 tensor-core GEMM over the rows of both operands (tcgen05), the weight
// gradient of the learned initialiser's head and of the layers that
// csrc/conv_wgrad.cu has no form for:
//
//   C[M][N] = sum_p A[p][m] B[p][n]     A [K][lda], B [K][ldb] bf16, FP32 accumulation
//
// with p the pixels (K, up to millions), A = dZ and B = the im2col operand.
// Both operands are "MN-major": the contiguous index is m or n, the summed one
// is the row.  The tensor core reads that layout itself (the transpose bits of
// the instruction descriptor), so neither operand is transposed in memory; the
// K-major GEMM (csrc/gemm_tc.cu) needed both transposed first, 4.6 GB of
// traffic in 2.3 ms per training step at 1080p, batch 8.
//
// What bounds it is the one pass over A and B (K (M + N) 2 bytes against 2 K M N
// operations with M, N of 32 ... 320 per tile), so:
//  * boxes are 64 columns x 128 rows (16 KB, 128-byte swizzle): TMA moves 8 KB
//    boxes at about 60 % of the rate it moves 16 KB ones;
//  * a tile is 64 NA rows (m) x 64 NB columns (n), as wide as two stages of
//    shared memory allow: NB up to 5 for NA = 1 (two MMAs, of 256 and 64 columns,
//    into 320 TMEM columns), up to 4 for NA = 2;
//  * K is split as gs2d_gemm_bf16 splits it, each split writing an FP32
//    partial tile; k_tn_reduce sums them in order.  The sums are the K-major
//    GEMM's bit for bit: an Adam step turns the sign of a gradient that is zero
//    but for rounding into a step of the whole rate, so other splits (over whole
//    waves: 0.2 ms less of a training step) moved the gradients of the next step
//    by up to 3e-4 now and then.
// Warp 0, one lane, issues the TMA boxes into a ring of ST stages; warp 1, one
// lane, the MMAs (eight K = 16 steps per stage); warps 0-3 the epilogue.
// Waits are bounded as in csrc/gemm_tc.cu; the producer also waits (bounded)
// for its last copies before the CTA may leave.
#include <cuda.h>
#include <cuda_bf16.h>
#include <stdio.h>

#include <algorithm>
#include <type_traits>

#include "gs2d_internal.cuh"
#include "tc_gemm.cuh"
#include "tc_ptx.cuh"

namespace gs2d {
namespace {

constexpr int kTnRows = 128;                // pixels per stage
constexpr int kTnBox = 64 * kTnRows * 2;    // one box: 64 columns x 128 rows of bf16

template <int NA, int NB>
struct TnShape {
  static constexpr int kBN = 64 * NB;
  static constexpr int kTmemCols = kBN <= 64 ? 64 : (kBN <= 128 ? 128 : (kBN <= 256 ? 256 : 512));
  static constexpr int kStageBytes = (NA + NB) * kTnBox;
  // 208 KB of the 227 KB a CTA may have; six stages hide any latency here
  static constexpr int kStages = std::min(6, 208 * 1024 / kStageBytes);
  static constexpr int kSmem = kStages * kStageBytes + 1024;
};

struct TnArgs {
  int M, N, K, per, ldc;  // per: 64-row tiles of a split
  size_t split_stride;
  float* out;  // partials, or the result when there is one split
  int* status;
};

template <int NA, int NB>
__global__ void __launch_bounds__(128, 1)
k_gemm_tn(const __grid_constant__ CUtensorMap ta, const __grid_constant__ CUtensorMap tb,
          TnArgs g) {
  using Sh = TnShape<NA, NB>;
  constexpr int ST = Sh::kStages;
  pdl_begin();
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full[ST], empty[ST], accum;
  __shared__ uint32_t s_tmem;
  __shared__ int s_fail;
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~uintptr_t(1023));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m0 = blockIdx.x * 64 * NA, n0 = blockIdx.y * Sh::kBN;
  // this split's rows, a multiple of 64 (or to the end): stages of 128, the
  // last of which may be half used
  const int64_t row0 = (int64_t)blockIdx.z * g.per * 64;
  const int rows = (int)min((int64_t)g.K - row0, (int64_t)g.per * 64);  // >= 1 (host)
  const int nk = (rows + kTnRows - 1) / kTnRows;

  if (threadIdx.x == 0) {
    for (int s = 0; s < ST; s++) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(&accum, 1);
    s_fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
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
    int issued = 0;
    for (; issued < nk; issued++) {
      const int s = issued % ST;
      if (!mbar_wait(&empty[s], ((uint32_t)(issued / ST) & 1u) ^ 1u)) {
        s_fail = 1;
        break;
      }
      uint8_t* st = smem + s * Sh::kStageBytes;
      const int row = (int)row0 + issued * kTnRows;
      mbar_expect_tx(&full[s], (uint32_t)Sh::kStageBytes);
#pragma unroll
      for (int c = 0; c < NA; c++) tma_load_2d(st + c * kTnBox, &ta, &full[s], m0 + 64 * c, row);
#pragma unroll
      for (int c = 0; c < NB; c++)
        tma_load_2d(st + (NA + c) * kTnBox, &tb, &full[s], n0 + 64 * c, row);
    }
    // no copy of this CTA is in flight when it leaves
    for (int i = issued > ST ? issued - ST : 0; i < issued; i++)
      if (!mbar_wait(&full[i % ST], (uint32_t)(i / ST) & 1u)) s_fail = 1;
  } else if (warp == 1 && lane == 0) {
    constexpr int kN1 = Sh::kBN < 256 ? Sh::kBN : 256, kN2 = Sh::kBN - kN1;
    constexpr uint32_t id1 = idesc_bf16_mn(kBM, kN1);
    constexpr uint32_t id2 = idesc_bf16_mn(kBM, kN2 ? kN2 : 64);
    for (int i = 0; i < nk; i++) {
      const int s = i % ST;
      if (!mbar_wait(&full[s], (uint32_t)(i / ST) & 1u)) {
        s_fail = 1;
        break;
      }
      tc_fence_after();
      const uint32_t a_s = smem_u32(smem + s * Sh::kStageBytes), b_s = a_s + NA * kTnBox;
      // one A box: rows 64 ... 127 of the tile read the same columns again
      const uint64_t ad = mn_major_desc(a_s, NA > 1 ? kTnBox : 0, 128);
      const uint64_t bd = mn_major_desc(b_s, kTnBox, 128), bd2 = bd + 4 * (kTnBox >> 4);
      const int used = min(kTnRows / 64, (rows - i * kTnRows + 63) / 64) * 4;
#pragma unroll 4
      for (int kk = 0; kk < used; kk++) {  // 16 rows of 128 bytes: 128 units
        const uint32_t acc = (i > 0 || kk > 0) ? 1u : 0u;
        mma_bf16(tmem, ad + 128 * kk, bd + 128 * kk, id1, acc);
        if (kN2) mma_bf16(tmem + 256, ad + 128 * kk, bd2 + 128 * kk, id2, acc);
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
  if (!s_fail && warp < 2 * NA) {
    const int row = m0 + warp * 32 + lane;
    float* out = g.out + (size_t)blockIdx.z * g.split_stride;
    const bool vec_ok = (g.ldc % 4) == 0 && (reinterpret_cast<uintptr_t>(out) & 15) == 0;
    store_acc_row<Sh::kBN>(tmem + ((uint32_t)(warp * 32) << 16), row < g.M,
                           (size_t)row * g.ldc + n0, g.N - n0, 0, vec_ok, out, nullptr);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(Sh::kTmemCols));
  if (threadIdx.x == 0 && s_fail && g.status) atomicCAS(g.status, 0, (int)GS2D_ERR_TIMEOUT);
}

// Sum of the partial tiles, split after split (deterministic, the order of
// csrc/gemm_tc.cu), V outputs a thread with kFlight loads in flight.
template <int V, int kFlight>
__global__ void __launch_bounds__(128)
k_tn_reduce(uint32_t M, uint32_t nv, uint32_t ldv, int splits, size_t stride,
            const float* __restrict__ partial, float* __restrict__ out) {
  using Vec = std::conditional_t<V == 4, float4, float>;
  pdl_begin();
  const size_t i = (size_t)blockIdx.x * 128 + threadIdx.x;
  if (i >= (size_t)M * nv) return;
  size_t o = i;
  if (nv != ldv) o = (i / nv) * ldv + i % nv;
  const Vec* src = reinterpret_cast<const Vec*>(partial) + o;
  const size_t step = stride / V;
  float x[V];
#pragma unroll
  for (int j = 0; j < V; j++) x[j] = 0.0f;
  const auto add = [&](const Vec& v) {
    const float* f = reinterpret_cast<const float*>(&v);
#pragma unroll
    for (int j = 0; j < V; j++) x[j] += f[j];
  };
  int z = 0;
  for (; z + kFlight <= splits; z += kFlight) {
    Vec v[kFlight];
#pragma unroll
    for (int u = 0; u < kFlight; u++) v[u] = src[(size_t)(z + u) * step];
#pragma unroll
    for (int u = 0; u < kFlight; u++) add(v[u]);
  }
  for (; z < splits; z++) add(src[(size_t)z * step]);
  Vec v;
#pragma unroll
  for (int j = 0; j < V; j++) reinterpret_cast<float*>(&v)[j] = x[j];
  reinterpret_cast<Vec*>(out)[o] = v;
}

template <int V, int kFlight>
cudaError_t launch_reduce(int M, int N, int ldc, int splits, size_t stride, const float* partial,
                          float* out, cudaStream_t s) {
  return launch_pdl(k_tn_reduce<V, kFlight>, (unsigned)(((size_t)M * (N / V) + 127) / 128), 128, 0,
                    s, (uint32_t)M, (uint32_t)(N / V), (uint32_t)(ldc / V), splits, stride,
                    partial, out);
}

// 2D map of a rows x cols matrix (cols contiguous): 64 x 128 boxes, 128-byte
// swizzle, zeros out of range.
bool tn_map(CUtensorMap* map, const void* base, int rows, int cols, int ld) {
  EncodeTiled fn = tensor_map_encoder();
  if (!fn) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  const cuuint32_t box[2] = {64, (cuuint32_t)kTnRows};
  const cuuint32_t estr[2] = {1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box,
            estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) ==
         CUDA_SUCCESS;
}

// Tile width and split of one product.  NB: as wide as shared memory allows (B
// read fewest times), in even tiles.
struct TnPlan {
  int na, nb, mt, nt;
  TnSplit sp;
};

TnPlan tn_plan(int M, int N, int K, int splits) {
  TnPlan p;
  p.na = M <= 64 ? 1 : 2;
  p.mt = (M + 64 * p.na - 1) / (64 * p.na);
  const int chunks = (N + 63) / 64, widest = p.na == 1 ? 5 : 4;
  p.nt = (chunks + widest - 1) / widest;
  p.nb = (chunks + p.nt - 1) / p.nt;
  p.nt = (chunks + p.nb - 1) / p.nb;
  p.sp = tn_split(K, splits);
  return p;
}

template <int NA, int NB>
cudaError_t launch_tn(const CUtensorMap& ta, const CUtensorMap& tb, const TnArgs& g, dim3 grid,
                      cudaStream_t s) {
  const cudaError_t e = opt_in_smem((const void*)k_gemm_tn<NA, NB>, TnShape<NA, NB>::kSmem);
  if (e != cudaSuccess) return e;
  return launch_pdl(k_gemm_tn<NA, NB>, grid, 128, TnShape<NA, NB>::kSmem, s, ta, tb, g);
}

template <int NA>
cudaError_t launch_tn_na(int nb, const CUtensorMap& ta, const CUtensorMap& tb, const TnArgs& g,
                         dim3 grid, cudaStream_t s) {
  switch (nb) {
    case 1: return launch_tn<NA, 1>(ta, tb, g, grid, s);
    case 2: return launch_tn<NA, 2>(ta, tb, g, grid, s);
    case 3: return launch_tn<NA, 3>(ta, tb, g, grid, s);
    case 4: return launch_tn<NA, 4>(ta, tb, g, grid, s);
  }
  if constexpr (NA == 1) return launch_tn<1, 5>(ta, tb, g, grid, s);
  return cudaErrorInvalidValue;
}

}  // namespace

TnSplit tn_split(int64_t pixels, int splits) {
  TnSplit p;
  const int num_kt = (int)((pixels + 63) / 64);
  p.splits = std::max(1, std::min(std::min(splits, num_kt), 65535));  // gridDim.z
  p.per = (num_kt + p.splits - 1) / p.splits;
  p.splits = (num_kt + p.per - 1) / p.per;
  return p;
}

cudaError_t launch_tn_reduce(int M, int N, int ldc, int splits, size_t stride,
                             const float* partial, float* out, cudaStream_t s) {
  // one output a thread while that leaves SMs without work otherwise
  const bool vec = N % 4 == 0 && ldc % 4 == 0 && stride % 4 == 0 &&
                   (((uintptr_t)partial | (uintptr_t)out) & 15) == 0;
  if (vec && (size_t)M * N >= 152 * 1024)
    return launch_reduce<4, 8>(M, N, ldc, splits, stride, partial, out, s);
  return launch_reduce<1, 16>(M, N, ldc, splits, stride, partial, out, s);
}

}  // namespace gs2d

using namespace gs2d;

extern "C" uint64_t gs2d_gemm_tn_partial_bytes(int32_t M, int32_t N, int32_t ldc, int32_t K,
                                               int32_t splits) {
  if (M < 1 || N < 1 || K < 1 || ldc < N) return 0;
  const TnPlan p = tn_plan(M, N, K, splits);
  return p.sp.splits > 1 ? (uint64_t)p.sp.splits * M * ldc * sizeof(float) : 0;
}

extern "C" gs2d_status gs2d_gemm_tn_bf16(const void* A, int32_t lda, const void* B, int32_t ldb,
                                         int32_t M, int32_t N, int32_t K, float* out, int32_t ldc,
                                         int32_t splits, float* partial, int32_t* status,
                                         void* stream) {
  if (M < 0 || N < 0 || K < 0 || lda < M || ldb < N || ldc < N || (lda % 8) || (ldb % 8))
    return set_error(GS2D_ERR_INVALID_ARG, "gs2d_gemm_tn_bf16: sizes / leading dimensions");
  if (M == 0 || N == 0) return set_error(GS2D_OK, "");
  if (!out || (K > 0 && (!A || !B)) || ((uintptr_t)A & 15) || ((uintptr_t)B & 15))
    return set_error(GS2D_ERR_INVALID_ARG, "gs2d_gemm_tn_bf16: NULL or misaligned operand");
  cudaStream_t s = (cudaStream_t)stream;
  cudaError_t e = cudaSuccess;
  if (K == 0) {
    e = cudaMemset2DAsync(out, (size_t)ldc * 4, 0, (size_t)N * 4, M, s);
  } else {
    const TnPlan p = tn_plan(M, N, K, splits);
    if (p.sp.splits > 1 && !partial)
      return set_error(GS2D_ERR_INVALID_ARG, "gs2d_gemm_tn_bf16: the split needs partial");
    CUtensorMap ta, tb;
    if (!tn_map(&ta, A, K, M, lda) || !tn_map(&tb, B, K, N, ldb))
      return set_error(GS2D_ERR_CUDA, "gs2d_gemm_tn_bf16: tensor map");
    TnArgs g;
    g.M = M;
    g.N = N;
    g.K = K;
    g.per = p.sp.per;
    g.ldc = ldc;
    g.split_stride = p.sp.splits > 1 ? (size_t)M * ldc : 0;
    g.out = p.sp.splits > 1 ? partial : out;
    g.status = status;
    const dim3 grid(p.mt, p.nt, p.sp.splits);
    e = p.na == 1 ? launch_tn_na<1>(p.nb, ta, tb, g, grid, s)
                  : launch_tn_na<2>(p.nb, ta, tb, g, grid, s);
    if (e == cudaSuccess && p.sp.splits > 1)
      e = launch_tn_reduce(M, N, ldc, p.sp.splits, g.split_stride, partial, out, s);
  }
  if (e != cudaSuccess) {
    char msg[200];
    snprintf(msg, sizeof(msg), "gs2d_gemm_tn_bf16: %s", cudaGetErrorString(e));
    return set_error(GS2D_ERR_CUDA, msg);
  }
  return set_error(GS2D_OK, "");
}
