// Bitstream accounting of a coded sequence (Sec. 3.3 B, Eq. 3-4): the ideal
// order-0 code length of quantised Gaussians (per-row histograms and their
// entropy, on the device) and the bits-back totals of a sequence (host).
#include <math.h>

#include "gs2d_internal.cuh"

namespace gs2d {
namespace {

constexpr int kBins = 1 << 16;  // per row: every 16-bit symbol
constexpr int kEntropyThreads = 1024;

struct RowBits {
  int bits[9];
};

__device__ __forceinline__ int symbol_bits(int b) { return b < 0 ? 16 : b; }

// Histogram of the (selected) codes of every row that is coded (bits != 0);
// codes are masked to the row's width, so any input stays in bounds.  The
// last scratch word counts the selected columns.
__global__ void __launch_bounds__(256)
k_code_hist(const uint16_t* __restrict__ codes, int n, RowBits rb,
            const uint8_t* __restrict__ select, uint32_t* __restrict__ hist) {
  const size_t total = (size_t)9 * n;
  for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < total;
       t += (size_t)gridDim.x * blockDim.x) {
    const int r = (int)(t / n);
    const int i = (int)(t - (size_t)r * n);
    if (select && !select[i]) continue;
    if (r == 0) atomicAdd(&hist[(size_t)9 * kBins], 1u);
    const int b = rb.bits[r];
    if (b == 0) continue;
    const uint32_t mask = (1u << symbol_bits(b)) - 1u;
    atomicAdd(&hist[(size_t)r * kBins + (codes[t] & mask)], 1u);
  }
}

// Code length of a row = T log2 T - sum over symbols of c log2 c.  Double
// precision is the cost here (FP64 issues at 1/64 of the FP32 rate, so a
// warp's log2 is over a thousand cycles of the SM's FP64 pipe), and the sum
// depends on the counts alone: with few columns the symbols have few distinct
// counts (at most sqrt(2 T)).  So the symbols are tallied by their count, and
// the logarithm is taken once per distinct count below kTally, in a
// compacted list, and per symbol above it (at most T / kTally symbols).
constexpr int kTally = 2048;

struct EntropySmem {
  unsigned tally[kTally];  // symbols of each count
  int item[kTally];        // the counts that occur, ascending
  int warp_items[kEntropyThreads / 32];
  double acc[kEntropyThreads / 32];
};

__device__ __forceinline__ void tally_clear(EntropySmem& sm) {
  for (int j = threadIdx.x; j < kTally; j += kEntropyThreads) sm.tally[j] = 0u;
}

__device__ __forceinline__ void tally_count(EntropySmem& sm, unsigned c, double& acc) {
  if (c < 2u) return;
  if (c < (unsigned)kTally)
    atomicAdd(&sm.tally[c], 1u);
  else
    acc += (double)c * log2((double)c);
}

// The row's code length from the threads' sums.  Valid in thread 0.
__device__ __forceinline__ double row_length(EntropySmem& sm, double total, double acc) {
  constexpr int kWarps = kEntropyThreads / 32;
  const int t = threadIdx.x;
  for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((t & 31) == 0) sm.acc[t >> 5] = acc;
  __syncthreads();
  if (t != 0) return 0.0;
  double sum = 0.0;
  for (int w = 0; w < kWarps; w++) sum += sm.acc[w];
  return total > 1.0 ? total * log2(total) - sum : 0.0;
}

// The row's code length from the tally and the threads' sums over the larger
// counts, in a fixed order (ascending counts over the threads, then a fixed
// reduction tree), so the result is reproducible.  Valid in thread 0.
__device__ __forceinline__ double tally_finish(EntropySmem& sm, double total, double acc) {
  constexpr int kPer = kTally / kEntropyThreads, kWarps = kEntropyThreads / 32;
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  __syncthreads();
  unsigned mine = 0;
#pragma unroll
  for (int k = 0; k < kPer; k++) mine += sm.tally[kPer * t + k] != 0u;
  unsigned inc = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) sm.warp_items[wid] = (int)inc;
  __syncthreads();
  int at = (int)(inc - mine), items = 0;
  for (int w = 0; w < kWarps; w++) {
    at += w < wid ? sm.warp_items[w] : 0;
    items += sm.warp_items[w];
  }
#pragma unroll
  for (int k = 0; k < kPer; k++)
    if (sm.tally[kPer * t + k] != 0u) sm.item[at++] = kPer * t + k;
  __syncthreads();
  for (int j = t; j < items; j += kEntropyThreads) {
    const double c = (double)sm.item[j];
    acc += (double)sm.tally[sm.item[j]] * (c * log2(c));
  }
  return row_length(sm, total, acc);
}

// Up to 65 535 columns: block r counts row r's symbols in shared memory and
// finishes the row, one launch without a histogram in device memory.
// Symbols of up to 10 bits have a 32-bit counter per lane (no two lanes of a
// warp meet, however skewed the symbols are); wider ones 16-bit counters in
// pairs, which 65 535 columns cannot overflow.
constexpr int kSmemColumns = 65535;
constexpr int kReplicaBits = 10;
constexpr int kHistBytes = kBins * 2;  // = 4 << (kReplicaBits + 5)

__global__ void __launch_bounds__(kEntropyThreads)
k_code_entropy_row(const uint16_t* __restrict__ codes, int n, RowBits rb,
                   const uint8_t* __restrict__ select, uint32_t* __restrict__ selected,
                   double* __restrict__ out) {
  pdl_begin();
  extern __shared__ uint32_t s_hist[];
  __shared__ EntropySmem sm;
  const int r = blockIdx.x, t = threadIdx.x, lane = t & 31, wid = t >> 5;
  const int b = rb.bits[r], bits = symbol_bits(b);
  const bool replicas = bits <= kReplicaBits;
  const uint32_t mask = (1u << bits) - 1u;
  const int words = b == 0 ? 0 : (replicas ? 32 << bits : (1 << bits) / 2);
  for (int j = t; j < words; j += kEntropyThreads) s_hist[j] = 0u;
  tally_clear(sm);
  __syncthreads();
  const uint16_t* row = codes + (size_t)r * n;
  int cnt = 0;
  for (int i = t; i < n; i += kEntropyThreads) {
    if (select && !select[i]) continue;
    cnt++;
    if (b == 0) continue;
    const uint32_t sym = row[i] & mask;
    if (replicas)
      atomicAdd(&s_hist[32 * sym + lane], 1u);
    else
      atomicAdd(&s_hist[sym >> 1], 1u << (16 * (sym & 1u)));
  }
  cnt = __reduce_add_sync(0xffffffffu, cnt);
  if (lane == 0) sm.warp_items[wid] = cnt;
  __syncthreads();
  int total = 0;
  for (int w = 0; w < kEntropyThreads / 32; w++) total += sm.warp_items[w];
  if (r == 0 && t == 0) *selected = (uint32_t)total;
  if (b == 0) {
    if (t == 0) out[r] = 32.0 * (double)total;
    return;
  }
  double acc = 0.0;
  if (replicas) {
    for (int sym = wid; sym <= (int)mask; sym += kEntropyThreads / 32) {
      const unsigned c = __reduce_add_sync(0xffffffffu, s_hist[32 * sym + lane]);
      if (lane == 0) tally_count(sm, c, acc);
    }
  } else {
    for (int j = t; j < words; j += kEntropyThreads) {
      const uint32_t w = s_hist[j];
      tally_count(sm, w & 0xffffu, acc);
      tally_count(sm, w >> 16, acc);
    }
  }
  const double length = tally_finish(sm, (double)total, acc);
  if (t == 0) out[r] = length;
}

// More columns: the counts of k_code_hist, in device memory.
__global__ void __launch_bounds__(kEntropyThreads)
k_code_entropy(const uint32_t* __restrict__ hist, RowBits rb, double* __restrict__ out) {
  __shared__ EntropySmem sm;
  const int r = blockIdx.x;
  const int b = rb.bits[r];
  const double total = (double)hist[(size_t)9 * kBins];
  if (b == 0) {
    if (threadIdx.x == 0) out[r] = 32.0 * total;
    return;
  }
  const int nb = 1 << symbol_bits(b);
  const uint32_t* counts = hist + (size_t)r * kBins;
  double acc = 0.0, length;
  if (nb <= 256) {  // (few symbols: the tally takes longer than it spares)
    for (int j = threadIdx.x; j < nb; j += kEntropyThreads)
      if (counts[j] > 1u) acc += (double)counts[j] * log2((double)counts[j]);
    length = row_length(sm, total, acc);
  } else {
    tally_clear(sm);
    __syncthreads();
    for (int j = threadIdx.x; j < nb; j += kEntropyThreads) tally_count(sm, counts[j], acc);
    length = tally_finish(sm, total, acc);
  }
  if (threadIdx.x == 0) out[r] = length;
}

}  // namespace
}  // namespace gs2d

using namespace gs2d;

extern "C" size_t gs2d_code_entropy_scratch_bytes(void) {
  return ((size_t)9 * kBins + 1) * sizeof(uint32_t);
}

extern "C" gs2d_status gs2d_code_entropy(const uint16_t* codes, int32_t n, const int32_t* bits,
                                         const uint8_t* select, void* scratch,
                                         size_t scratch_bytes, double* out_bits,
                                         void* stream) {
  if (n < 0 || !bits || !out_bits || !scratch ||
      scratch_bytes < gs2d_code_entropy_scratch_bytes() || (n > 0 && !codes))
    return set_error(GS2D_ERR_INVALID_ARG, "gs2d_code_entropy: arguments");
  RowBits rb;
  for (int r = 0; r < 9; r++) {
    const int b = bits[r];
    if (!(b == -16 || (b >= 0 && b <= 16)))
      return set_error(GS2D_ERR_INVALID_ARG, "gs2d_code_entropy: bits");
    rb.bits[r] = b;
  }
  cudaStream_t s = (cudaStream_t)stream;
  uint32_t* hist = (uint32_t*)scratch;
  if (n <= kSmemColumns) {
    cudaError_t e = opt_in_smem((const void*)k_code_entropy_row, kHistBytes);
    if (e == cudaSuccess)
      e = launch_pdl(k_code_entropy_row, 9, kEntropyThreads, kHistBytes, s, codes, (int)n, rb,
                     select, hist + (size_t)9 * kBins, out_bits);
    if (e != cudaSuccess) return set_error(GS2D_ERR_CUDA, cudaGetErrorString(e));
    return set_error(GS2D_OK, "");
  }
  cudaError_t e = cudaMemsetAsync(hist, 0, gs2d_code_entropy_scratch_bytes(), s);
  if (e == cudaSuccess) {
    const size_t want = ((size_t)9 * n + 255) / 256;
    const int blocks = (int)(want < 152 * 8 ? want : 152 * 8);
    k_code_hist<<<blocks, 256, 0, s>>>(codes, n, rb, select, hist);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) {
    k_code_entropy<<<9, kEntropyThreads, 0, s>>>(hist, rb, out_bits);
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) return set_error(GS2D_ERR_CUDA, cudaGetErrorString(e));
  return set_error(GS2D_OK, "");
}

// Eq. 3: log2(m!) - log2(m), through lgamma (0 for m <= 1).
static double bitsback_saving(int32_t m) {
  if (m <= 1) return 0.0;
  return (lgamma((double)m + 1.0) - log((double)m)) / log(2.0);
}

extern "C" gs2d_status gs2d_sequence_bits(const int32_t* counts, const double* payload_bits,
                                          int32_t frames, int32_t gop, gs2d_seq_bits* out) {
  if (frames < 0 || gop < 1 || !out || (frames > 0 && (!counts || !payload_bits)))
    return set_error(GS2D_ERR_INVALID_ARG, "gs2d_sequence_bits: arguments");
  gs2d_seq_bits r = {0.0, 0.0, 0.0, 0.0, 0, 0};
  for (int32_t k = 0; k < frames; k++) {
    if (counts[k] < 0 || !isfinite(payload_bits[k]) || payload_bits[k] < 0.0)
      return set_error(GS2D_ERR_INVALID_ARG, "gs2d_sequence_bits: frame entry");
    if (k % gop == 0) {
      r.i_bits += payload_bits[k];
      r.i_frames++;
    } else {
      r.p_bits += payload_bits[k];
      r.savings += bitsback_saving(counts[k]);
      r.p_frames++;
    }
  }
  r.total_bits = r.i_bits + r.p_bits - r.savings;
  *out = r;
  return set_error(GS2D_OK, "");
}

// ---------------------------------------------------------------------------
// Coded size of one frame (Sec. 3.3 B): the rows' ideal code lengths, plus
// for a P-frame the index of every selected Gaussian (ceil(log2 n) bits),
// plus the per-frame ranges of a quantiser that refines them per frame
// (two float32 per uniform row).
namespace gs2d {
namespace {

__global__ void k_frame_bits(const double* __restrict__ rows, const uint32_t* __restrict__ hist,
                             int index_bits, int range_bits, double* __restrict__ out) {
  pdl_begin();
  double t = 0.0;
  for (int r = 0; r < 9; r++) t += rows[r];
  const double m = (double)hist[(size_t)9 * kBins];  // selected columns
  out[0] = t + m * (double)index_bits + (double)range_bits;
}

}  // namespace
}  // namespace gs2d

extern "C" size_t gs2d_frame_bits_scratch_bytes(void) {
  return gs2d_code_entropy_scratch_bytes() + 16 * sizeof(double);
}

extern "C" gs2d_status gs2d_frame_bits(const uint16_t* codes, int32_t n, const int32_t* bits,
                                       const uint8_t* select, int32_t refine, void* scratch,
                                       size_t scratch_bytes, double* out_bits, void* stream) {
  if (!scratch || scratch_bytes < gs2d_frame_bits_scratch_bytes() || !out_bits || !bits)
    return set_error(GS2D_ERR_INVALID_ARG, "gs2d_frame_bits: arguments");
  const size_t eb = gs2d_code_entropy_scratch_bytes();
  double* rows = reinterpret_cast<double*>(static_cast<char*>(scratch) +
                                           ((eb + 15) & ~size_t(15)));
  gs2d_status st = gs2d_code_entropy(codes, n, bits, select, scratch, eb, rows, stream);
  if (st != GS2D_OK) return st;
  int index_bits = 0;
  if (select) {
    int64_t span = 1;
    while (span < (int64_t)(n > 2 ? n : 2)) {
      span <<= 1;
      index_bits++;
    }
  }
  int uniform = 0;
  for (int r = 0; r < 9; r++) uniform += bits[r] > 0;
  const int range_bits = refine ? 64 * uniform : 0;
  const cudaError_t e =
      launch_pdl(k_frame_bits, 1, 1, 0, (cudaStream_t)stream, (const double*)rows,
                 static_cast<const uint32_t*>(scratch), index_bits, range_bits, out_bits);
  if (e != cudaSuccess) return set_error(GS2D_ERR_CUDA, cudaGetErrorString(e));
  return set_error(GS2D_OK, "");
}
