// High-precision side of OutControl (paper Sec. 4.2): the outlier channels of X / W stay in BF16. The forward side
// product runs on the tensor cores inside the FP4 GEMM kernels and dW[:, outliers] = dY^T X_out in a BF16 tensor-core
// kernel of its own (gemm.cu); here are the copy that builds a compact side operand, the FP8 snap of the side operands,
// and the pass that assembles dW from the compact FP4 product and the side product's token splits.
#include <type_traits>

#include "nvfp4_device.cuh"
#include "nvfp4_internal.h"

namespace nvfp4 {

// Token splits of the side product dW[c, outl[j]] = sum_t dY[t, c] * X_out[t, j]: at most kHpDwSplit partial sums per output
// element go to a workspace and are added in a fixed order (bit-reproducible results).
constexpr int kHpDwSplit = 16;

// dW[c, d] for whole output rows (OutControl's weight gradient): a kept channel takes its value from the compact FP4
// product, an outlier channel the sum of the high-precision side product's token splits. One coalesced pass over dW
// instead of a column scatter plus a scattered reduce. A CTA takes kAsmRows rows. It builds, in shared memory, where every channel comes
// from: src_of[d] = position in the compact product (>= 0) or -(1 + rank among the outliers); sums the splits of its outlier channels
// there (four channels per thread, fixed order); and (STAGED) copies its rows of the compact product there as they are. All of it is under
// way together; the rows are then put together from shared memory and stored. An outlier's entry is its own, whatever the map holds there:
// the map comes first, and a barrier. That barrier stands before the sums (us of dW alone, 8192 x 2816 -> 1024 with 282 outlier channels,
// 128 x 8192 -> 8192 with 820: 83.3, 253 here; after the sums 84.7, 248; the map by plain loads 83.4, 265; no order at all 83.0, 258).
// What bounds it is the latency of those loads: the rows of one CTA take a microsecond, a wave of CTAs is one or two of them. Reading the
// compact product only once src_of is known, and the sums a channel per thread, was a second round of latency: us of a layer's backward with it,
// before / now: 8192 x 1024 -> 2816 with 102 outlier channels 155 / 149, 8192 x 2816 -> 1024 with 282 161 / 150, 4095 x 1024 -> 2816 with
// 102 (BF16) 82 / 77, 1000 x 9000 -> 256 with 180 (two rows per CTA) 85 / 61. More registers for more splits in flight: the same.
constexpr int kAsmRows = 4;
template <bool F32, int ROWS, bool STAGED>
__global__ void __launch_bounds__(256) dw_assemble_kernel(const __grid_constant__ HpDwArgs a, int n_split, int vec) {
  pdl_prologue();
  extern __shared__ __align__(16) float asm_smem[];
  const uint32_t D = (uint32_t)a.D, n_out = (uint32_t)a.n_out, n_out4 = (n_out + 3u) >> 2, ldc = (uint32_t)a.ld_compact;
  float* const osum = asm_smem;                                          // [ROWS][4 n_out4]
  float* const rows = osum + ROWS * n_out4 * 4;                          // [ROWS][ldc] if STAGED
  int32_t* const src_of = reinterpret_cast<int32_t*>(rows + (STAGED ? ROWS * ldc : 0u));  // [D]
  const int64_t c0 = (int64_t)blockIdx.x * ROWS;
  const uint32_t nr = (uint32_t)min((int64_t)ROWS, a.C - c0);
  // (the map need not stand on a 16-byte boundary)
  const uint32_t map = (uint32_t)__cvta_generic_to_shared(src_of);
  for (uint32_t d = threadIdx.x; d < D; d += 256)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(map + d * 4u), "l"(a.col_map + d) : "memory");
  asm volatile("cp.async.commit_group;" ::: "memory");
  if (STAGED) {  // (rows of 16-byte pieces, one after another)
    const float* p = a.compact + c0 * ldc;
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(rows), pieces = nr * (ldc >> 2);
    for (uint32_t e = threadIdx.x; e < pieces; e += 256)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + e * 16u), "l"(p + (size_t)e * 4u) : "memory");
  }
  int32_t own[2];  // the first 512 outlier channels, loaded beside the map
#pragma unroll
  for (uint32_t i = 0; i < 2; ++i) own[i] = threadIdx.x + i * 256u < n_out ? __ldg(a.outl + threadIdx.x + i * 256u) : -1;
  asm volatile("cp.async.commit_group;\ncp.async.wait_group 1;" ::: "memory");  // the map's copies, not the rows'
  __syncthreads();
#pragma unroll
  for (uint32_t i = 0; i < 2; ++i)
    if (own[i] >= 0) src_of[own[i]] = -(int32_t)(1 + threadIdx.x + i * 256u);
  for (uint32_t j = threadIdx.x + 512u; j < n_out; j += 256) src_of[__ldg(a.outl + j)] = -(int32_t)(1 + j);
  const int64_t split_stride = a.C * a.Kh;
  for (uint32_t e = threadIdx.x; e < nr * n_out4; e += 256) {
    const uint32_t rr = e / n_out4, j = (e - rr * n_out4) * 4u;  // (Kh is a multiple of 64: the columns past n_out exist)
    const float* p = a.partial + (c0 + rr) * a.Kh + j;
    float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    for (int s0 = 0; s0 < n_split; s0 += 8) {
      float4 t[8];
#pragma unroll
      for (int i = 0; i < 8; ++i)
        t[i] = s0 + i < n_split ? __ldg(reinterpret_cast<const float4*>(p + (s0 + i) * split_stride)) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
      for (int i = 0; i < 8; ++i)
        if (s0 + i < n_split) v = make_float4(v.x + t[i].x, v.y + t[i].y, v.z + t[i].z, v.w + t[i].w);
    }
    *reinterpret_cast<float4*>(osum + rr * n_out4 * 4u + j) = v;
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  for (uint32_t rr = 0; rr < nr; ++rr) {
    const float* const kept = STAGED ? rows + rr * ldc : a.compact + (c0 + rr) * ldc;
    const float* const sums = osum + rr * n_out4 * 4u - 1;
    float* const df = reinterpret_cast<float*>(a.dW) + (c0 + rr) * a.lddw;
    uint16_t* const dh = reinterpret_cast<uint16_t*>(a.dW) + (c0 + rr) * a.lddw;
    auto value = [&](int32_t m) { return m >= 0 ? kept[m] : sums[-m]; };
    auto store1 = [&](uint32_t d, float v) {
      if (F32)
        df[d] = v;
      else
        dh[d] = f32_to_bf16_bits(v);
    };
    if (vec) {  // four channels per item, one 16-byte (FP32) or 8-byte (BF16) store
      for (uint32_t d = threadIdx.x * 4u; d < D; d += 1024u) {
        if (d + 4u <= D) {
          const int4 m = *reinterpret_cast<const int4*>(src_of + d);
          const float4 v = make_float4(value(m.x), value(m.y), value(m.z), value(m.w));
          if (F32)
            *reinterpret_cast<float4*>(df + d) = v;
          else
            *reinterpret_cast<uint2*>(dh + d) = make_uint2((uint32_t)f32_to_bf16_bits(v.x) | ((uint32_t)f32_to_bf16_bits(v.y) << 16),
                                                           (uint32_t)f32_to_bf16_bits(v.z) | ((uint32_t)f32_to_bf16_bits(v.w) << 16));
        } else {
          for (; d < D; ++d) store1(d, value(src_of[d]));
        }
      }
    } else {
      for (uint32_t d = threadIdx.x; d < D; d += 256u) store1(d, value(src_of[d]));
    }
  }
}

// FP8 option for the outlier channels (paper Sec. 4.2 names FP8 as a possible precision of the outlier part; the recipe
// is this library's): a compact side operand T (BF16, contiguous) is replaced in place by the values an E4M3 tensor
// with a per-tensor power-of-two scale represents:  e = smallest integer with amax / 2^e <= 448,  T8 = E4M3(T / 2^e) 2^e.
// Both scalings are exact and T8 is exactly representable in BF16, so the BF16 tensor-core products that consume the
// side operands give what an FP8 product times the two scales would give. cell holds the float bits of amax(|T|).
__device__ __forceinline__ void fp8_snap_body(uint16_t* __restrict__ t, int64_t n, const uint32_t* __restrict__ cell, unsigned block,
                                              unsigned n_blocks) {
  const uint32_t ab = cell[0];
  int e = 0;
  if (ab) {
    const int k = (int)((ab >> 23) & 0xFFu) - 127;
    e = (ab & 0x7FFFFFu) <= 0x600000u ? k - 8 : k - 7;  // mantissa <= 1.75: amax / 2^(k - 8) = m 2^8 <= 448
  }
  const float r = __uint_as_float((uint32_t)(127 - e) << 23), s = __uint_as_float((uint32_t)(127 + e) << 23);
  const int64_t pairs = n >> 1;  // n is even (the padded width is a multiple of 64)
  uint32_t* t2 = reinterpret_cast<uint32_t*>(t);
  for (int64_t i = (int64_t)block * blockDim.x + threadIdx.x; i < pairs; i += (int64_t)n_blocks * blockDim.x) {
    const uint32_t w = t2[i];
    const float lo = __fmul_rn(bf16_lo(w), r), hi = __fmul_rn(bf16_hi(w), r);
    uint32_t h2;
    asm("{\n.reg .b16 q;\ncvt.rn.satfinite.e4m3x2.f32 q, %1, %2;\ncvt.rn.f16x2.e4m3x2 %0, q;\n}" : "=r"(h2) : "f"(hi), "f"(lo));
    const float qlo = __half2float(__ushort_as_half((unsigned short)(h2 & 0xFFFFu)));
    const float qhi = __half2float(__ushort_as_half((unsigned short)(h2 >> 16)));
    t2[i] = (uint32_t)f32_to_bf16_bits(__fmul_rn(qlo, s)) | ((uint32_t)f32_to_bf16_bits(__fmul_rn(qhi, s)) << 16);
  }
}
__global__ void __launch_bounds__(256) fp8_snap_pair_kernel(uint16_t* a, int64_t n_a, const uint32_t* cell_a, unsigned grid_a, uint16_t* b,
                                                           int64_t n_b, const uint32_t* cell_b) {
  pdl_prologue();
  if (blockIdx.x < grid_a)
    fp8_snap_body(a, n_a, cell_a, blockIdx.x, grid_a);
  else
    fp8_snap_body(b, n_b, cell_b, blockIdx.x - grid_a, gridDim.x - grid_a);
}

cudaError_t launch_fp8_snap_pair(uint16_t* a, int64_t rows_a, uint16_t* b, int64_t rows_b, int64_t Kh, uint32_t* cells2, cudaStream_t st) {
  if (Kh == 0 || (rows_a == 0 && rows_b == 0)) return cudaSuccess;
  cudaError_t e;
  if ((e = launch_zero_words(cells2, 2, st)) != cudaSuccess) return e;
  if ((e = launch_amax_tensor_pair(a, rows_a, Kh, Kh, cells2, b, rows_b, Kh, Kh, cells2 + 1, st)) != cudaSuccess) return e;
  const int64_t cap = (int64_t)device_sm_count() * 4;
  auto grid_of = [cap](int64_t n) { return (unsigned)std::max<int64_t>(1, std::min<int64_t>((n / 2 + 255) / 256, cap)); };
  const unsigned ga = grid_of(rows_a * Kh), gb = grid_of(rows_b * Kh);
  launch_kernel(fp8_snap_pair_kernel, dim3(ga + gb), dim3(256), 0, st, a, rows_a * Kh, static_cast<const uint32_t*>(cells2), ga, b,
                rows_b * Kh, static_cast<const uint32_t*>(cells2 + 1));
  return cudaGetLastError();
}

// dst[r, j] = src[r, cols[j]] (j < n), 0 for n <= j < ld_dst. One warp per row.
__global__ void __launch_bounds__(256) gather_cols_kernel(const uint16_t* __restrict__ src, int64_t ld_src, int64_t rows,
                                                         const int32_t* __restrict__ cols, int64_t n, uint16_t* __restrict__ dst,
                                                         int64_t ld_dst) {
  pdl_prologue();
  const int64_t r = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  if (r >= rows) return;
  for (int64_t j = threadIdx.x & 31; j < ld_dst; j += 32) dst[r * ld_dst + j] = j < n ? src[r * ld_src + cols[j]] : (uint16_t)0;
}

size_t hp_dw_partial_floats(int64_t T, int64_t C, int64_t Kh) { return (size_t)kHpDwSplit * (size_t)C * (size_t)Kh; }

// token splits of the side product: as many as fill the SMs once with (C / 128) x splits CTAs, at most kHpDwSplit (the
// workspace's size)
static void hp_dw_splits(const HpDwArgs& a, int64_t& t_per_split, int& n_split) {
  const int64_t want = std::max<int64_t>(1, std::min<int64_t>(kHpDwSplit, device_sm_count() / std::max<int64_t>(1, (a.C + 127) / 128)));
  t_per_split = ((a.T + want - 1) / want + 63) / 64 * 64;
  n_split = (int)((a.T + t_per_split - 1) / t_per_split);
}

// First half of dW under OutControl: the split partial sums of dY^T X_out (needs nothing of the FP4 product).
cudaError_t launch_hp_dw_product(const HpDwArgs& a, cudaStream_t st) {
  if (a.C == 0 || a.n_out == 0) return cudaSuccess;
  int64_t t_per_split;
  int n_split;
  hp_dw_splits(a, t_per_split, n_split);
  return launch_hp_dw_mma(a.dY, a.lddy, a.X_out, a.Kh, a.T, a.C, a.partial, n_split, t_per_split, a.dev_status, st);
}

// Second half: dW from the compact FP4 product and the split partial sums.
cudaError_t launch_hp_dw_finish(const HpDwArgs& a, cudaStream_t st) {
  if (a.C == 0 || a.n_out == 0) return cudaSuccess;
  int64_t t_per_split;
  int n_split;
  hp_dw_splits(a, t_per_split, n_split);
  if (!a.compact || !a.col_map || !hp_dw_assemble_fits(a.D, a.n_out)) return cudaErrorInvalidValue;
  // kept and outlier channels written together, row by row; the compact rows go through shared memory where two CTAs of four rows fit an
  // SM, else one of two rows, else they are read as they are needed
  const int64_t n4 = (a.n_out + 3) & ~(int64_t)3;
  auto smem_of = [&](int64_t rows, bool staged) { return (size_t)((rows * n4 + (staged ? rows * a.ld_compact : 0) + a.D) * 4); };
  const bool aligned = (a.ld_compact & 3) == 0 && (reinterpret_cast<uintptr_t>(a.compact) & 15u) == 0;
  const int elt = a.dw_is_f32 ? 4 : 2;
  const int vec = (a.lddw & 3) == 0 && (reinterpret_cast<uintptr_t>(a.dW) & (size_t)(4 * elt - 1)) == 0;
  auto launch = [&](auto f32, auto rows, auto staged) -> cudaError_t {
    const auto kernel = dw_assemble_kernel<f32.value, rows.value, staged.value>;
    const size_t smem = smem_of(rows.value, staged.value);
    const cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(kernel), smem);
    if (e != cudaSuccess) return e;
    launch_kernel(kernel, dim3((unsigned)((a.C + rows.value - 1) / rows.value)), dim3(256), smem, st, a, n_split, vec);
    return cudaGetLastError();
  };
  auto pick = [&](auto f32) -> cudaError_t {
    using std::integral_constant;
    if (aligned && smem_of(kAsmRows, true) <= 110 * 1024) return launch(f32, integral_constant<int, kAsmRows>{}, integral_constant<bool, true>{});
    if (aligned && smem_of(2, true) <= 200 * 1024) return launch(f32, integral_constant<int, 2>{}, integral_constant<bool, true>{});
    return launch(f32, integral_constant<int, kAsmRows>{}, integral_constant<bool, false>{});
  };
  return a.dw_is_f32 ? pick(std::integral_constant<bool, true>{}) : pick(std::integral_constant<bool, false>{});
}

// The assembling pass keeps one source index per channel and kAsmRows sums per outlier channel in shared memory.
bool hp_dw_assemble_fits(int64_t D, int64_t n_out) { return (D + 4 + kAsmRows * n_out) * 4 <= 200 * 1024; }

cudaError_t launch_hp_dw(const HpDwArgs& a, cudaStream_t st) {
  const cudaError_t e = launch_hp_dw_product(a, st);
  return e != cudaSuccess ? e : launch_hp_dw_finish(a, st);
}

cudaError_t launch_gather_cols(const uint16_t* src, int64_t ld_src, int64_t rows, const int32_t* cols, int64_t n, uint16_t* dst,
                               int64_t ld_dst, cudaStream_t st) {
  if (rows == 0 || ld_dst == 0) return cudaSuccess;
  launch_kernel(gather_cols_kernel, dim3((unsigned)((rows + 7) / 8)), dim3(256), 0, st, src, ld_src, rows, cols, n, dst, ld_dst);
  return cudaGetLastError();
}

}  // namespace nvfp4
