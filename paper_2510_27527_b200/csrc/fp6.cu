// Simulated FP6 x FP4 linear layer of the paper's precision-switching study (Sec. 5.4, "Precision Switching in Final Stage"):
//     Y = Q6_D(X) x Q4_D(W^T),   dX = Q6_S(dY) x Q4_S(W-hat),   dW = Q4_S(dY^T) x Q6_S(X-hat).
// The paper names FP6 without a recipe; this library's: element format E2M3 (32 magnitudes up to 7.5), the scale sequence of
// the FP4 quantizer (Sec. 2.2) with Q_max = 7.5 -- Sg = amax / 3360, t = amax_b / Sg, s = t / 7.5, Sb = e4m3(s), d = Sg Sb,
// r = 1 / d, y = x r, one binary32 operation each, |y| clamped to 7.5 -- per-tensor global scale, round to nearest (ties to
// the even code) or the 16-bit stochastic rounding of the FP4 quantizer with the same Philox addressing.
// No tensor-core instruction multiplies E2M3 by E2M1 under E4M3 block scales, and the paper itself simulates: the operands
// of the simulated products are "dense": P * S_block as BF16, which is exact for both formats (at most 4 + 4 significant
// bits), plus the FP32 global scale; the product runs on BF16 tensor cores (CTA pairs, or the side-product path of the 128 x 128 GEMM
// kernel) with FP32 accumulation and the two global scales in the epilogue.
#include <algorithm>

#include "nvfp4_device.cuh"
#include "nvfp4_internal.h"

namespace nvfp4 {

namespace {

// Round 16 scaled values to E2M3 and return them times the block scale as packed BF16 pairs (8 words).
// Stochastic rounding, as for E2M1 (e2m1x8_sr) with three mantissa bits instead of one: w = a * 2^-126, rounded up, has E2M3's own
// spacing, its cell is bits(w) >> 20 and the low 20 bits the position inside it; adding 2^20 - 1 - ((2u + 1) << 3) to the bits
// carries into the cell iff position > (2u + 1) << 3, i.e. iff (u + 0.5) / 65536 < position / 2^20 (an integer n is < x iff
// n < ceil(x)); clearing the low 20 bits then leaves the rounded magnitude times 2^-126
// (against cells below 1 mapped onto [0.5, 1) and back, 4096 x 3072 rows with the amax pass 24.6 -> 21.5 us).
template <bool SR>
__device__ __forceinline__ void fp6_block16(const float (&x)[16], float rcp, float Sbf, const PhiloxKeys& pk, uint32_t stream_id,
                                            uint64_t idx8, uint32_t (&out)[8]) {
  uint4 w[2];
  if (SR) {
    w[0] = sr_words(pk, stream_id, idx8);
    w[1] = sr_words(pk, stream_id, idx8 + 1);
  }
#pragma unroll
  for (int i = 0; i < 16; i += 2) {
    float y0, y1, p0, p1;
    mul2_rn(x[i], x[i + 1], rcp, y0, y1);
    if (SR) {
      const uint4& ww = w[i >> 3];
      const uint32_t word = ~(((i >> 1) & 3) == 0 ? ww.x : ((i >> 1) & 3) == 1 ? ww.y : ((i >> 1) & 3) == 2 ? ww.z : ww.w);
      float w0, w1;
      mul2_up(fminf(fabsf(y0), 7.5f), fminf(fabsf(y1), 7.5f), 0x1p-126f, w0, w1);
      const uint32_t b0 = __float_as_uint(w0) + ((word & 0xFFFFu) * 16u + 7u), b1 = __float_as_uint(w1) + ((word >> 16) * 16u + 7u);
      mul2_rn(__uint_as_float((b0 & 0x7FF00000u) | (__float_as_uint(y0) & 0x80000000u)),
              __uint_as_float((b1 & 0x7FF00000u) | (__float_as_uint(y1) & 0x80000000u)), 0x1p126f, p0, p1);
    } else {
      // hardware conversion: round to nearest even, saturating at 7.5; then back to FP16 (exact)
      uint16_t packed;
      asm("cvt.rn.satfinite.e2m3x2.f32 %0, %1, %2;" : "=h"(packed) : "f"(y1), "f"(y0));
      uint32_t h2;
      asm("cvt.rn.f16x2.e2m3x2 %0, %1;" : "=r"(h2) : "h"(packed));
      const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&h2));
      p0 = f.x;
      p1 = f.y;
    }
    float v0, v1;  // exact, in BF16 too: at most 4 + 4 significant bits
    mul2_rn(p0, p1, Sbf, v0, v1);
    out[i >> 1] = __byte_perm(__float_as_uint(v0), __float_as_uint(v1), 0x7632);
  }
  if (Sbf != Sbf) {  // an infinity in the block: its values are written as -0 (the global scale is infinite)
#pragma unroll
    for (int i = 0; i < 8; ++i) out[i] = 0x80008000u;
  }
}

// The scale pair of a block: E4M3 block scale as a float and the reciprocal that maps x onto the E2M3 grid.
__device__ __forceinline__ float fp6_block_scale(float amax_b, float Sg, float& rcp) {
  const float t = __fdiv_rn(amax_b, Sg);
  const float s = __fdiv_rn(t, 7.5f);
  const float Sbf = e4m3_decode(e4m3_encode(s));
  const float d = __fmul_rn(Sg, Sbf);
  rcp = Sbf == 0.0f ? 0.0f : __frcp_rn(d);
  return Sbf;
}
__device__ __forceinline__ float fp6_global_scale(float amax) { return amax == 0.0f ? 1.0f : __fdiv_rn(amax, 3360.0f); }

// n / d for n < total: a 32-bit division where that is enough (a 64-bit one is a hundred instructions).
__device__ __forceinline__ int64_t quotient(int64_t n, int64_t d, int64_t total) {
  return total < ((int64_t)1 << 32) ? (int64_t)((uint32_t)n / (uint32_t)d) : n / d;
}

// Row-axis FP6 quantize from BF16 [rows, cols] (leading dimension ld): NB 16-element blocks of the padded output rows (ld_out / 16 blocks
// each: those past K are written as zeros) per thread, at a stride, all loads first. cells: bits of max |x| over the tensor, in `words`
// words. Bound by the chain from the maximum to the scales of a block, which NB = 4 shares.
template <bool SR, int NB>
__global__ void __launch_bounds__(256)
fp6_quantize_rows_kernel(const uint16_t* __restrict__ src, int64_t rows, int64_t K, int64_t ld, uint32_t stream_id,
                         const uint32_t* __restrict__ cells, int words, uint16_t* __restrict__ out, int64_t ld_out, float* __restrict__ gscale,
                         const __grid_constant__ PhiloxKeys pk) {
  pdl_prologue();
  const int64_t nb = ld_out >> 4, total = rows * nb;
  const int64_t K16 = (K + 15) & ~(int64_t)15;
  const bool vec = (ld & 7) == 0 && (reinterpret_cast<uintptr_t>(src) & 15u) == 0;
  uint32_t w[NB][8];
  int64_t row[NB], k0[NB];  // (row -1: none)
#pragma unroll
  for (int j = 0; j < NB; ++j) {
    const int64_t gid = ((int64_t)blockIdx.x * NB + j) * 256 + threadIdx.x;
    row[j] = gid < total ? quotient(gid, nb, total) : -1;
    k0[j] = (gid - row[j] * nb) << 4;
    const uint16_t* p = src + row[j] * ld + k0[j];
#pragma unroll
    for (int i = 0; i < 8; ++i) w[j][i] = 0u;
    if (row[j] < 0 || k0[j] >= K) continue;
    if (vec && k0[j] + 16 <= K) {
      const uint4 a = *reinterpret_cast<const uint4*>(p), c = *reinterpret_cast<const uint4*>(p + 8);
      w[j][0] = a.x; w[j][1] = a.y; w[j][2] = a.z; w[j][3] = a.w;
      w[j][4] = c.x; w[j][5] = c.y; w[j][6] = c.z; w[j][7] = c.w;
    } else {
#pragma unroll
      for (int i = 0; i < 16; ++i)
        if (k0[j] + i < K) w[j][i >> 1] |= (uint32_t)p[i] << (16 * (i & 1));
    }
  }
  const float Sg = fp6_global_scale(__uint_as_float(tensor_amax_bits(cells, words)));
  if (blockIdx.x == 0 && threadIdx.x == 0) gscale[0] = Sg;
#pragma unroll
  for (int j = 0; j < NB; ++j) {
    if (row[j] < 0) break;
    uint4* dst = reinterpret_cast<uint4*>(out + row[j] * ld_out + k0[j]);
    if (k0[j] >= K) {
      dst[0] = dst[1] = make_uint4(0, 0, 0, 0);
      continue;
    }
    uint32_t m2 = 0;
    float x[16];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      m2 = amax16x2(m2, w[j][i]);
      x[2 * i] = bf16_lo(w[j][i]);
      x[2 * i + 1] = bf16_hi(w[j][i]);
    }
    float rcp;
    const float Sbf = fp6_block_scale(__uint_as_float(hmax_of_pair(bf16x2_abs_bits(m2)) << 16), Sg, rcp);
    uint32_t o[8];
    fp6_block16<SR>(x, rcp, Sbf, pk, stream_id, (uint64_t)(row[j] * K16 + k0[j]) >> 3, o);
    dst[0] = make_uint4(o[0], o[1], o[2], o[3]);
    dst[1] = make_uint4(o[4], o[5], o[6], o[7]);
  }
}

// Transposing FP6 re-quantize of a dense operand: in [rowsK, D] (values v, global scale Sg_in) -> out [D, rowsK] with blocks
// along the source rows. x_hat = float32(v * Sg_in) is the aligned tensor (one rounding). A lane owns four neighbouring
// source columns and one 16-row block (8 bytes per source row: a warp reads 256 contiguous bytes per row). cell[0] = bits of
// max |v|; the maximum of x_hat is float32(max |v| * Sg_in) because the multiplication is monotonic.
template <bool SR>
__global__ void __launch_bounds__(128)
fp6_requantize_t_kernel(const uint16_t* __restrict__ in, int64_t rowsK, int64_t D, int64_t ld_in, const float* __restrict__ in_gscale,
                        uint32_t stream_id, const uint32_t* __restrict__ cell, uint16_t* __restrict__ out, int64_t ld_out,
                        float* __restrict__ gscale, const __grid_constant__ PhiloxKeys pk) {
  pdl_prologue();
  const int64_t d0 = ((int64_t)blockIdx.y * 32 + (threadIdx.x & 31)) * 4;
  const int64_t k0 = ((int64_t)blockIdx.x * 4 + (threadIdx.x >> 5)) * 16;
  const bool live = d0 < D && k0 < ld_out;
  const int64_t K16 = (rowsK + 15) & ~(int64_t)15;
  uint2 w[16];
#pragma unroll
  for (int t = 0; t < 16; ++t)
    w[t] = live && k0 + t < rowsK ? *reinterpret_cast<const uint2*>(in + (k0 + t) * ld_in + d0) : make_uint2(0u, 0u);  // ld_in, d0: multiples of 4
  const float sg_in = in_gscale[0];
  const float Sg = fp6_global_scale(__fmul_rn(__uint_as_float(cell[0]), sg_in));
  if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) gscale[0] = Sg;
  if (!live) return;
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    if (d0 + c >= D) break;
    uint4* dst = reinterpret_cast<uint4*>(out + (d0 + c) * ld_out + k0);
    if (k0 >= rowsK) {
      dst[0] = dst[1] = make_uint4(0, 0, 0, 0);
      continue;
    }
    float x[16], m = 0.0f;
#pragma unroll
    for (int t = 0; t < 16; ++t) {
      const uint32_t word = c < 2 ? w[t].x : w[t].y;
      x[t] = __fmul_rn((c & 1) ? bf16_hi(word) : bf16_lo(word), sg_in);
      m = fmaxf(m, fabsf(x[t]));
    }
    float rcp;
    const float Sbf = fp6_block_scale(m, Sg, rcp);
    uint32_t o[8];
    fp6_block16<SR>(x, rcp, Sbf, pk, stream_id, (uint64_t)((d0 + c) * K16 + k0) >> 3, o);
    dst[0] = make_uint4(o[0], o[1], o[2], o[3]);
    dst[1] = make_uint4(o[4], o[5], o[6], o[7]);
  }
}

// FP4 operand (codes + E4M3 scales in either layout) -> dense BF16 values P * S_block [R, ld_out]; one thread per 8 codes.
__global__ void __launch_bounds__(256)
expand_operand_kernel(const uint8_t* __restrict__ codes, const uint8_t* __restrict__ sf, int sf_tiled, int64_t R, int64_t K,
                      const float* __restrict__ in_gscale, uint16_t* __restrict__ out, int64_t ld_out, float* __restrict__ gscale) {
  pdl_prologue();
  const int64_t n8 = ld_out >> 3;
  const int64_t gid = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (gid == 0) gscale[0] = in_gscale[0];
  if (gid >= R * n8) return;
  const int64_t r = quotient(gid, n8, R * n8), k0 = (gid - r * n8) << 3;
  const int64_t Kp = (K + 127) & ~(int64_t)127;
  uint4 o = make_uint4(0, 0, 0, 0);
  if (k0 < Kp) {
    const uint32_t word = *reinterpret_cast<const uint32_t*>(codes + r * (Kp >> 1) + (k0 >> 1));
    const int64_t nb = Kp >> 4;
    const size_t sfo = sf_tiled ? sf_tiled_offset(r, k0 >> 4, (nb + 15) & ~(int64_t)15) : (size_t)(r * nb + (k0 >> 4));
    uint32_t h[4];
    const uint8_t scale = sf[sfo];
    decode8_h2(word, scale, h);
    uint32_t q[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&h[i]));
      q[i] = __byte_perm(__float_as_uint(f.x), __float_as_uint(f.y), 0x7632);  // exact in BF16: 2 + 4 significant bits
    }
    o = make_uint4(q[0], q[1], q[2], q[3]);
    if ((scale & 0x7Fu) == 0x7Fu) o = make_uint4(0x80008000u, 0x80008000u, 0x80008000u, 0x80008000u);  // a NaN scale, as in fp6_block16
  }
  *reinterpret_cast<uint4*>(out + r * ld_out + k0) = o;
}

}  // namespace

cudaError_t launch_fp6_quantize_rows(const uint16_t* src, int64_t rows, int64_t K, int64_t ld, int sr, uint64_t seed, uint32_t stream_id,
                                     uint32_t* cells, size_t cells_bytes, uint16_t* out, int64_t ld_out, float* gscale, cudaStream_t st) {
  if (rows == 0) return cudaSuccess;
  // The maximum as words that need no clearing (a launch less: 2 us of host time), or folded into one cleared word: every thread waits for the
  // words, so that more threads make them dearer. To nearest, four blocks per thread share that wait from 4 CTAs of single ones per SM on, and
  // from 8 on one word is better. With the longer chain of stochastic rounding the two are within 4 % of one another from 4 CTAs on (the line at 2^20
  // blocks is where a launch less no longer shows), and four blocks per thread lose below it. us with the amax pass from a graph, words and NB = 1 /
  // words and NB = 4 / one word; in brackets issued by the host: to nearest 64 x 256 3.4 / 4.8 / 3.8; 2400 x 1024 7.4 / 7.4 / 6.4 (8.0 / 7.9 / 10.2);
  // 4096 x 1024 10.5 / 7.2 / 7.4 (10.0 / 8.0 / 10.1); 4096 x 1536 11.2 / 9.7 / 8.4 (11.6 / 10.3 / 10.1); 4096 x 3072 18.1 / 14.3 / 12.0;
  // 16384 x 4096 93.1 / 80.3 / 67.9; stochastic 1000 x 1416 6.6 / 10.2 / 7.9; 4096 x 1024 8.9 / 12.1 / 9.3; 4096 x 3072 19.1 / 20.4 / 19.2;
  // 8192 x 2048 (2^20 blocks) 23.9 / 23.8 / 24.8; 16384 x 4096 103 / 101 / 104.
  const int64_t blocks = rows * (ld_out >> 4), per_sm = (int64_t)device_sm_count() * 256;
  const int words = blocks <= (sr ? (int64_t)1 << 20 : 8 * per_sm) && cells_bytes >= kTensorAmaxWords * sizeof(uint32_t) ? kTensorAmaxWords : 1;
  cudaError_t e;
  if (words > 1) {
    if ((e = launch_amax_tensor_words(src, rows, K, ld, cells, st)) != cudaSuccess) return e;
  } else {
    if ((e = launch_zero_words(cells, 1, st)) != cudaSuccess) return e;
    if ((e = launch_amax_tensor(src, rows, K, ld, cells, st)) != cudaSuccess) return e;
  }
  const uint32_t* ccells = cells;
  auto go = [&](auto kernel, int nb) {
    launch_kernel(kernel, dim3((unsigned)((blocks + 256 * nb - 1) / (256 * nb))), dim3(256), 0, st, src, rows, K, ld, stream_id, ccells, words,
                  out, ld_out, gscale, make_philox_keys(seed));
  };
  if (sr)
    go(fp6_quantize_rows_kernel<true, 1>, 1);
  else if (words > 1 && blocks > 4 * per_sm)
    go(fp6_quantize_rows_kernel<false, 4>, 4);
  else
    go(fp6_quantize_rows_kernel<false, 1>, 1);
  return cudaGetLastError();
}

cudaError_t launch_fp6_requantize_t(const uint16_t* in, int64_t rowsK, int64_t D, int64_t ld_in, const float* in_gscale, int sr,
                                    uint64_t seed, uint32_t stream_id, uint32_t* cell, uint16_t* out, int64_t ld_out, float* gscale,
                                    cudaStream_t st) {
  if (rowsK == 0 || D == 0) return cudaSuccess;
  cudaError_t e;
  if ((e = launch_zero_words(cell, 1, st)) != cudaSuccess) return e;
  if ((e = launch_amax_tensor(in, rowsK, D, ld_in, cell, st)) != cudaSuccess) return e;
  const dim3 grid((unsigned)((ld_out / 16 + 3) / 4), (unsigned)((D + 127) / 128));
  const uint32_t* ccell = cell;
  if (sr)
    launch_kernel(fp6_requantize_t_kernel<true>, grid, dim3(128), 0, st, in, rowsK, D, ld_in, in_gscale, stream_id, ccell, out, ld_out,
                  gscale, make_philox_keys(seed));
  else
    launch_kernel(fp6_requantize_t_kernel<false>, grid, dim3(128), 0, st, in, rowsK, D, ld_in, in_gscale, stream_id, ccell, out, ld_out,
                  gscale, make_philox_keys(seed));
  return cudaGetLastError();
}

cudaError_t launch_expand_operand(const uint8_t* codes, const uint8_t* sf, int sf_tiled, int64_t R, int64_t K, const float* in_gscale,
                                  uint16_t* out, int64_t ld_out, float* gscale, cudaStream_t st) {
  if (R == 0) return cudaSuccess;
  const unsigned grid = (unsigned)((R * (ld_out >> 3) + 255) / 256);
  launch_kernel(expand_operand_kernel, dim3(grid), dim3(256), 0, st, codes, sf, sf_tiled, R, K, in_gscale, out, ld_out, gscale);
  return cudaGetLastError();
}

}  // namespace nvfp4
