// OutControl calibration (paper Sec. 4.2, the paragraph that defines the outlier index set): per-channel l2-norms of
// the activations are accumulated over a calibration window, and the channels with the largest accumulated value form
// the outlier set. Two entry points:
//   nvfp4_outlier_accumulate   acc[d] += sqrt(sum_t X[t, d]^2) for one step's activations (HBM streaming, 2 B/element)
//   nvfp4_outlier_select       top-n_out channels of acc -> sorted outlier list, sorted kept list, channel map
// Both are deterministic: partial sums are combined in a fixed order, ties go to the lower channel index.
#include "../../include/nvfp4.h"

#include "nvfp4_device.cuh"
#include "nvfp4_internal.h"

namespace nvfp4 {

// Sum of squares of a slab of rows, per channel. Block = 32 lanes x 8 row lanes; a lane owns 8 neighbouring channels (one
// 16-byte load per row), so a warp reads 512 contiguous bytes of a row. partial[slab][channel], channel padded to 256.
__global__ void __launch_bounds__(256) colsq_partial_kernel(const uint16_t* __restrict__ X, int64_t ld, int64_t N, int64_t D,
                                                           int64_t rows_per_slab, float* __restrict__ partial, int64_t Dp) {
  pdl_prologue();
  const int lane = threadIdx.x & 31, ry = threadIdx.x >> 5;
  const int64_t c0 = (int64_t)blockIdx.x * 256 + lane * 8;
  const int64_t r_begin = (int64_t)blockIdx.y * rows_per_slab;
  const int64_t r_end = min(N, r_begin + rows_per_slab);
  float s[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) s[i] = 0.0f;
  auto add8 = [&](const uint4& v) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float lo = bf16_lo(w[i]), hi = bf16_hi(w[i]);
      s[2 * i] = fmaf(lo, lo, s[2 * i]);
      s[2 * i + 1] = fmaf(hi, hi, s[2 * i + 1]);
    }
  };
  if (c0 + 8 <= D) {
    int64_t r = r_begin + ry;
    for (; r + 56 < r_end; r += 64) {  // eight rows in flight
      uint4 v[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) v[q] = *reinterpret_cast<const uint4*>(X + (r + 8 * q) * ld + c0);
#pragma unroll
      for (int q = 0; q < 8; ++q) add8(v[q]);
    }
    for (; r < r_end; r += 8) add8(*reinterpret_cast<const uint4*>(X + r * ld + c0));
  } else if (c0 < D) {  // ragged last chunk of a row
    for (int64_t r = r_begin + ry; r < r_end; r += 8)
      for (int i = 0; i < 8; ++i)
        if (c0 + i < D) {
          const float v = bf16_bits_to_float(X[r * ld + c0 + i]);
          s[i] = fmaf(v, v, s[i]);
        }
  }
  __shared__ float red[8][8][32];  // [row lane][i][lane]: conflict-free both ways
#pragma unroll
  for (int i = 0; i < 8; ++i) red[ry][i][lane] = s[i];
  __syncthreads();
  {
    const int i = threadIdx.x >> 5, ln = threadIdx.x & 31;
    float t = 0.0f;
#pragma unroll
    for (int y = 0; y < 8; ++y) t += red[y][i][ln];  // fixed order
    partial[(int64_t)blockIdx.y * Dp + (int64_t)blockIdx.x * 256 + ln * 8 + i] = t;
  }
}

// acc[d] += sqrt(sum over slabs). A CTA takes 32 channels, each of its 32 warps every 32nd slab, then the 32 sums of a channel
// are added in warp order: a fixed order for a given shape. (One thread per channel walking 222 slabs, the count for 1024
// channels, was a chain of dependent adds behind strided loads; this takes 3.4 us, and the step with the selection 23.5 instead of 41.8.)
__global__ void __launch_bounds__(1024) colsq_finalize_kernel(const float* __restrict__ partial, int64_t n_slabs, int64_t Dp, int64_t D,
                                                             float* __restrict__ acc) {
  pdl_prologue();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t d = (int64_t)blockIdx.x * 32 + lane;  // < Dp, which is a multiple of 256
  float s = 0.0f;
#pragma unroll 4
  for (int64_t k = wid; k < n_slabs; k += 32) s += partial[k * Dp + d];
  __shared__ float red[32][32];
  red[wid][lane] = s;
  __syncthreads();
  if (wid != 0 || d >= D) return;
  float t = 0.0f;
#pragma unroll
  for (int w = 0; w < 32; ++w) t += red[w][lane];
  acc[d] = acc[d] + __fsqrt_rn(t);
}

// Sorts like the value: larger key = larger value; -0 and +0 are one value.
__device__ __forceinline__ uint32_t order_key(float v) {
  const uint32_t u = __float_as_uint(v + 0.0f);
  return u ^ ((uint32_t)((int32_t)u >> 31) | 0x80000000u);
}
// inclusive sum over the lanes of a warp
__device__ __forceinline__ uint32_t warp_inclusive_sum(uint32_t v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, v, o);
    if (lane >= o) v += t;
  }
  return v;
}

// The whole selection in one CTA: radix select of the n_out-th largest key (a byte per pass, histogram in shared memory, equal
// bytes of a warp counted once), then a stable compaction in index order: keys above the threshold and the first `need` equal to
// it are outliers. Work is linear in D and latency is what bounds it; comparing all pairs of channels instead, with the
// compaction in a launch of its own, took 21 us for D = 1024 in four CTAs of 1024 sequential compares.
__global__ void __launch_bounds__(1024) outlier_select_kernel(const float* __restrict__ acc, int64_t D, int64_t n_out,
                                                             int32_t* __restrict__ col_map, int32_t* __restrict__ outl,
                                                             int32_t* __restrict__ keep) {
  pdl_prologue();
  __shared__ uint32_t hist[256];
  __shared__ uint32_t found[2];  // threshold so far, rank still to resolve among the keys that share it
  __shared__ uint32_t warp_cnt[32], chunk_total;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  uint32_t prefix = 0, need = (uint32_t)n_out;
  if (n_out > 0) {
    for (int shift = 24; shift >= 0; shift -= 8) {
      if (tid < 256) hist[tid] = 0;
      __syncthreads();
      const uint32_t mask_hi = shift == 24 ? 0u : (0xFFFFFFFFu << (shift + 8));
      for (int64_t c0 = 0; c0 < D; c0 += 1024) {
        const int64_t d = c0 + tid;
        const uint32_t key = d < D ? order_key(acc[d]) : 0u;
        const bool in = d < D && ((key ^ prefix) & mask_hi) == 0;
        const uint32_t byte = in ? (key >> shift) & 255u : 256u;
        const uint32_t same = __match_any_sync(0xFFFFFFFFu, byte);
        if (in && lane == __ffs(same) - 1) atomicAdd(&hist[byte], (uint32_t)__popc(same));
      }
      __syncthreads();
      if (wid == 0) {  // lane l looks at bytes 255 - 8 l downwards
        uint32_t c[8], sum = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) sum += c[i] = hist[255 - 8 * lane - i];
        uint32_t before = warp_inclusive_sum(sum, lane) - sum;
        if (before < need && need <= before + sum) {
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            if (before < need && need <= before + c[i]) {
              found[0] = prefix | ((uint32_t)(255 - 8 * lane - i) << shift);
              found[1] = need - before;
            }
            before += c[i];
          }
        }
      }
      __syncthreads();
      prefix = found[0];
      need = found[1];
    }
  }
  // counts are packed: keys above the threshold in the low half, equal ones in the high half (at most 1024 per chunk)
  uint32_t gt_base = 0, eq_base = 0;
  for (int64_t c0 = 0; c0 < D; c0 += 1024) {
    const int64_t d = c0 + tid;
    const uint32_t key = d < D ? order_key(acc[d]) : 0u;
    const bool gt = d < D && n_out > 0 && key > prefix, eq = d < D && n_out > 0 && key == prefix;
    const uint32_t bg = __ballot_sync(0xFFFFFFFFu, gt), be = __ballot_sync(0xFFFFFFFFu, eq);
    if (lane == 0) warp_cnt[wid] = (uint32_t)__popc(bg) | ((uint32_t)__popc(be) << 16);
    __syncthreads();
    if (wid == 0) {
      const uint32_t v = warp_cnt[lane], incl = warp_inclusive_sum(v, lane);
      warp_cnt[lane] = incl - v;
      if (lane == 31) chunk_total = incl;
    }
    __syncthreads();
    const uint32_t below = (1u << lane) - 1u, w = warp_cnt[wid];
    const uint32_t gt_before = gt_base + (w & 0xFFFFu) + __popc(bg & below), eq_before = eq_base + (w >> 16) + __popc(be & below);
    const uint32_t out_before = gt_before + min(eq_before, need);
    if (d < D) {
      if (gt || (eq && eq_before < need)) {
        outl[out_before] = (int32_t)d;
        col_map[d] = -1;
      } else {
        const int64_t pos = d - out_before;
        keep[pos] = (int32_t)d;
        col_map[d] = (int32_t)pos;
      }
    }
    gt_base += chunk_total & 0xFFFFu;
    eq_base += chunk_total >> 16;
    __syncthreads();
  }
}

// Row slabs of the partial-sum pass. A tuning constant, not a hardware query: the workspace size derived from it must not
// depend on the device (about six CTAs per SM on a 148-SM part).
constexpr int64_t kCalibTargetCtas = 888;
static int64_t calib_slabs(int64_t N, int64_t D) {
  const int64_t col_ctas = (D + 255) / 256;
  int64_t slabs = (kCalibTargetCtas + col_ctas - 1) / col_ctas;
  slabs = std::max<int64_t>(1, std::min<int64_t>(slabs, (N + 31) / 32));
  return slabs;
}

}  // namespace nvfp4

using namespace nvfp4;

extern "C" {

size_t nvfp4_outlier_accumulate_workspace_bytes(int64_t N_tok, int64_t D) {
  if (N_tok <= 0 || D <= 0) return 256;
  const int64_t Dp = (D + 255) / 256 * 256;
  return (size_t)(calib_slabs(N_tok, D) * Dp * 4 + 256);
}

nvfp4_status nvfp4_outlier_accumulate(const void* X_bf16, int64_t ldx, int64_t N_tok, int64_t D, float* acc, void* workspace,
                                      size_t ws_bytes, void* stream) {
  if (!X_bf16 || !acc) return NVFP4_ERR_NULL;
  if (N_tok < 0 || D < 0) return NVFP4_ERR_SHAPE;
  if ((reinterpret_cast<uintptr_t>(X_bf16) & 15u) || ldx < D || (ldx * 2) % 16 != 0 || (reinterpret_cast<uintptr_t>(acc) & 3u))
    return NVFP4_ERR_ALIGN;
  if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 15u) || ws_bytes < nvfp4_outlier_accumulate_workspace_bytes(N_tok, D))
    return NVFP4_ERR_WORKSPACE;
  if (!device_is_sm100()) return NVFP4_ERR_ARCH;
  if (N_tok == 0 || D == 0) return NVFP4_OK;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int64_t Dp = (D + 255) / 256 * 256;
  const int64_t slabs = calib_slabs(N_tok, D);
  const int64_t rows_per_slab = ((N_tok + slabs - 1) / slabs + 7) / 8 * 8;
  const int64_t used_slabs = (N_tok + rows_per_slab - 1) / rows_per_slab;
  float* partial = static_cast<float*>(workspace);
  launch_kernel(colsq_partial_kernel, dim3((unsigned)(Dp / 256), (unsigned)used_slabs), dim3(256), 0, st, static_cast<const uint16_t*>(X_bf16),
                ldx, N_tok, D, rows_per_slab, partial, Dp);
  if (cudaGetLastError() != cudaSuccess) return NVFP4_ERR_CUDA;
  launch_kernel(colsq_finalize_kernel, dim3((unsigned)((D + 31) / 32)), dim3(1024), 0, st, static_cast<const float*>(partial), used_slabs, Dp, D,
                acc);
  return cudaGetLastError() == cudaSuccess ? NVFP4_OK : NVFP4_ERR_CUDA;
}

nvfp4_status nvfp4_outlier_select(const float* acc, int64_t D, int64_t n_out, int32_t* outlier_cols, int32_t* keep_cols,
                                  int32_t* col_map, void* stream) {
  if (D < 0 || n_out < 0 || n_out > D || D > 0x7FFFFFFF) return NVFP4_ERR_SHAPE;
  if (D == 0) return NVFP4_OK;
  if (!acc || !col_map || (n_out > 0 && !outlier_cols) || (n_out < D && !keep_cols)) return NVFP4_ERR_NULL;
  if (!device_is_sm100()) return NVFP4_ERR_ARCH;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  launch_kernel(outlier_select_kernel, dim3(1), dim3(1024), 0, st, acc, D, n_out, col_map, outlier_cols, keep_cols);
  return cudaGetLastError() == cudaSuccess ? NVFP4_OK : NVFP4_ERR_CUDA;
}

}  // extern "C"
