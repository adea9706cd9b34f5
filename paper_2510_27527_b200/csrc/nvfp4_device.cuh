// Device-side building blocks of the NVFP4 quantizers: format conversions, the element rounding rules and the
// counter-based random generator. Everything that can change a code or a scale is an explicit IEEE binary32
// operation (__fdiv_rn / __fmul_rn, no fast-math, no contraction), in the order the quantizer's contract fixes.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace nvfp4 {

// Programmatic dependent launch: let the next kernel of the stream start its prologue, then wait until the previous
// kernel has completed (its writes are visible, and it no longer reads what this kernel will overwrite). Must run
// before the first global-memory access. A no-op when the kernel was launched without the attribute.
__device__ __forceinline__ void pdl_prologue() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// The two halves on their own. A kernel that waits first and then calls pdl_launch_next() lets its successor's CTAs start only
// when everything before itself is complete and visible; that successor may then load what this kernel only reads before its
// own pdl_wait() (load_cg below), i.e. under this kernel.
__device__ __forceinline__ void pdl_launch_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Loads through L2 that stay where they are written (an ordinary load of read-only memory may be moved across the waits).
__device__ __forceinline__ float4 load_cg4(const float* p) {
  float4 v;
  asm volatile("ld.global.cg.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void load_cg8(const float* p, float* v) {  // 32-byte aligned
  asm volatile("ld.global.cg.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
               : "l"(p)
               : "memory");
}
__device__ __forceinline__ void store8(float* p, const float* v) {  // 32-byte aligned
  asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]),
               "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
               : "memory");
}
__device__ __forceinline__ float load_cg(const float* p) {
  float v;
  asm volatile("ld.global.cg.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ float load_ca(const float* p) {  // through L1, after the kernel's wait
  float v;
  asm volatile("ld.global.ca.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ uint32_t load_ca(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.global.ca.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ uint32_t load_cg(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.global.cg.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

constexpr int kRoundRTN = 0;
constexpr int kRoundSR = 1;
constexpr int kGsTensor = 0;
constexpr int kGsRow = 1;
constexpr int kGsBlock128 = 2;
constexpr int kSfLinear = 0;
constexpr int kSfTiled = 1;

// ---------------------------------------------------------------------------------------------------------
// BF16 pairs packed in a 32-bit word
// ---------------------------------------------------------------------------------------------------------
__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }
// |x| of both halves as 16-bit patterns; for finite BF16 the pattern order is the value order.
__device__ __forceinline__ uint32_t bf16x2_abs_bits(uint32_t w) { return w & 0x7FFF7FFFu; }
// max of two packed pairs of non-negative BF16 patterns (as 16-bit unsigned integers == as BF16 values)
__device__ __forceinline__ uint32_t umax16x2(uint32_t a, uint32_t b) {
  const __nv_bfloat162 r = __hmax2(*reinterpret_cast<const __nv_bfloat162*>(&a), *reinterpret_cast<const __nv_bfloat162*>(&b));
  return *reinterpret_cast<const uint32_t*>(&r);
}
// max(|a|, |b|) of both halves in one instruction; the sign bits of the result are meaningless (xor of the inputs'),
// callers mask them off once at the end with bf16x2_abs_bits
__device__ __forceinline__ uint32_t amax16x2(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("max.xorsign.abs.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}
__device__ __forceinline__ uint32_t hmax_of_pair(uint32_t m) { return max(m & 0xFFFFu, m >> 16); }
__device__ __forceinline__ float bf16_bits_to_float(uint32_t b16) { return __uint_as_float(b16 << 16); }

// FP32 -> BF16 bit pattern, round to nearest even (finite inputs).
__device__ __forceinline__ uint16_t f32_to_bf16_bits(float v) {
  const uint32_t b = __float_as_uint(v);
  return (uint16_t)((b + 0x7FFFu + ((b >> 16) & 1u)) >> 16);
}

// ---------------------------------------------------------------------------------------------------------
// Maximum of a tensor without a cleared cell: an amax kernel writes N words (N = 32 or 64), one per CTA or per cluster of CTAs
// and zeros in the rest, and its readers take their maximum. An atomic maximum into one word needs that word cleared first,
// i.e. one launch more (about 3 us of host time, and a serial point of about 2 us on the device).
// ---------------------------------------------------------------------------------------------------------
template <int N>
__device__ __forceinline__ uint32_t cells_max(const uint32_t* __restrict__ cells) {  // every lane of the warp calls this
  const int lane = threadIdx.x & 31;
  uint32_t v = load_cg(cells + lane);
  if (N == 64) v = max(v, load_cg(cells + 32 + lane));
  return __reduce_max_sync(0xFFFFFFFFu, v);
}
// The maximum as its readers see it: one word (folded into by atomics) or 64.
__device__ __forceinline__ uint32_t tensor_amax_bits(const uint32_t* __restrict__ cells, int words) {
  return words == 1 ? cells[0] : cells_max<64>(cells);
}
__device__ __forceinline__ uint32_t cluster_ctas() {
  uint32_t n;
  asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(n));
  return n;
}
// At the head of a kernel that ends with cells_write: says that this CTA has started. A CTA's shared memory may be written from another
// one only after that, and a CTA without work gets to its store at once; the wait is in cells_write, under the loads of the others.
__device__ __forceinline__ void cells_begin() {
  if (cluster_ctas() > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
}
// Word of this thread's cluster <- maximum of the cluster's values m. Every thread of every CTA calls it, after cells_begin;
// blockDim.x is a multiple of 32 and at most 1024, the cluster (cluster_x, 1, 1) has at most 8 CTAs. CTA `block` of the n_blocks
// (whole clusters, at most N of them) that share the N words.
template <int N>
__device__ __forceinline__ void cells_write(uint32_t m, uint32_t* cells, uint32_t block, uint32_t n_blocks) {
  __shared__ uint32_t warp_max[32];
  __shared__ uint32_t cta_max[8];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
  const uint32_t n_rank = cluster_ctas();
  uint32_t rank;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  m = __reduce_max_sync(0xFFFFFFFFu, m);
  if (lane == 0) warp_max[wid] = m;
  __syncthreads();
  if (n_rank > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");  // every CTA of the cluster has started (cells_begin)
  if (wid == 0) {
    m = __reduce_max_sync(0xFFFFFFFFu, lane < n_warps ? warp_max[lane] : 0u);
    if (lane == 0) {
      if (n_rank == 1) {
        cta_max[0] = m;
      } else {
        uint32_t dst;
        asm("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(dst) : "r"((uint32_t)__cvta_generic_to_shared(&cta_max[rank])));
        asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(dst), "r"(m) : "memory");
      }
    }
  }
  if (n_rank > 1) {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  } else {
    __syncthreads();
  }
  if (rank == 0 && wid == 0) {
    const uint32_t cluster = block / n_rank, n_clusters = n_blocks / n_rank;
    m = __reduce_max_sync(0xFFFFFFFFu, lane < (int)n_rank ? cta_max[lane] : 0u);
    if (lane == 0) cells[cluster] = m;
    if (cluster == 0)
      for (uint32_t i = n_clusters + lane; i < (uint32_t)N; i += 32) cells[i] = 0u;
  }
}

// ---------------------------------------------------------------------------------------------------------
// E4M3 (bias 7, max 448, no infinity): block scales
// ---------------------------------------------------------------------------------------------------------
// Non-negative float -> E4M3 byte: round to nearest, ties to even, saturate to 448.
__device__ __forceinline__ uint32_t e4m3_encode(float s) {
  uint16_t packed;
  asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(packed) : "f"(0.0f), "f"(s));
  return packed & 0xFFu;
}
// E4M3 byte -> float (exact).
__device__ __forceinline__ float e4m3_decode(uint32_t byte) {
  uint32_t h2;
  asm("{.reg .b16 t; cvt.u16.u32 t, %1; cvt.rn.f16x2.e4m3x2 %0, t;}" : "=r"(h2) : "r"(byte & 0xFFu));
  return __half2float(__ushort_as_half((unsigned short)(h2 & 0xFFFFu)));
}

// ---------------------------------------------------------------------------------------------------------
// Scales of the double-block quantizer (paper Sec. 2.2): the pinned operation sequence.
// ---------------------------------------------------------------------------------------------------------
// x / c for a constant c, correctly rounded, in three instructions: q0 = RN(x * rc), rem = x - q0 * c (exact in the FMA),
// q = RN(q0 + rem * rc), rc = RN(1 / c). For c = 6 and c = 2688 this was compared with the IEEE quotient for every one of the
// 2^31 non-negative binary32 inputs: identical whenever the quotient is a normal number (quotients in the subnormal range
// differ in the last bits; there the value only ever feeds an E4M3 conversion that gives 0 either way, or lies below the
// smallest supported amax).
__device__ __forceinline__ float div_const(float x, float c, float rc) {
  const float q0 = __fmul_rn(x, rc);
  const float rem = __fmaf_rn(-q0, c, x);
  return __fmaf_rn(rem, rc, q0);
}
__device__ __forceinline__ float global_scale_from_amax(float amax) {
  return amax == 0.0f ? 1.0f : div_const(amax, 2688.0f, 0x1.861862p-12f);  // amax / (448 * 6)
}
// Returns the E4M3 byte of the block scale and the reciprocal r that maps x to the FP4 grid (0 if the scale is 0).
// round_up: take the smallest E4M3 value >= s instead of the nearest one (448 stays the ceiling), so that no element of
// the block lands beyond +-6 on the FP4 grid and stochastic rounding is unbiased for every element.
__device__ __forceinline__ uint32_t block_scale(float amax_b, float Sg, float& rcp, bool round_up = false) {
  const float t = __fdiv_rn(amax_b, Sg);
  const float s = div_const(t, 6.0f, 0x1.555556p-3f);
  uint32_t sb = e4m3_encode(s);
  float Sbf = e4m3_decode(sb);
  if (round_up && Sbf < s && sb < 0x7Eu) {  // non-negative E4M3 bytes are ordered like their values
    sb += 1u;
    Sbf = e4m3_decode(sb);
  }
  const float d = __fmul_rn(Sg, Sbf);
  rcp = (Sbf == 0.0f) ? 0.0f : __frcp_rn(d);  // the correctly rounded 1 / d
  return sb;
}

// ---------------------------------------------------------------------------------------------------------
// Philox4x32-10
// ---------------------------------------------------------------------------------------------------------
__device__ __forceinline__ uint4 philox4x32_10(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, uint32_t k0,
                                               uint32_t k1) {
#pragma unroll
  for (int i = 0; i < 10; ++i) {
    // one widening multiply per product (high and low halves together)
    const uint64_t p0 = (uint64_t)0xD2511F53u * c0;
    const uint64_t p1 = (uint64_t)0xCD9E8D57u * c2;
    const uint32_t n0 = (uint32_t)(p1 >> 32) ^ c1 ^ k0;
    const uint32_t n2 = (uint32_t)(p0 >> 32) ^ c3 ^ k1;
    c0 = n0; c1 = (uint32_t)p1; c2 = n2; c3 = (uint32_t)p0;
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
  return make_uint4(c0, c1, c2, c3);
}
// The ten round keys of a 64-bit Philox key, prepared on the host and handed to the kernels as a constant parameter:
// the rounds then read them as constant-bank operands instead of carrying two running additions per round.
struct PhiloxKeys {
  uint32_t k0[10], k1[10];
};
inline PhiloxKeys make_philox_keys(uint64_t seed) {
  PhiloxKeys r;
  uint32_t a = (uint32_t)seed, b = (uint32_t)(seed >> 32);
  for (int i = 0; i < 10; ++i) {
    r.k0[i] = a;
    r.k1[i] = b;
    a += 0x9E3779B9u;
    b += 0xBB67AE85u;
  }
  return r;
}
__device__ __forceinline__ uint4 philox4x32_10(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, const PhiloxKeys& rk) {
#pragma unroll
  for (int i = 0; i < 10; ++i) {
    const uint64_t p0 = (uint64_t)0xD2511F53u * c0;
    const uint64_t p1 = (uint64_t)0xCD9E8D57u * c2;
    const uint32_t n0 = (uint32_t)(p1 >> 32) ^ c1 ^ rk.k0[i];
    const uint32_t n2 = (uint32_t)(p0 >> 32) ^ c3 ^ rk.k1[i];
    c0 = n0; c1 = (uint32_t)p1; c2 = n2; c3 = (uint32_t)p0;
  }
  return make_uint4(c0, c1, c2, c3);
}
// The four 32-bit words holding the 16-bit draws of elements idx8*8 .. idx8*8+7 of the operand.
__device__ __forceinline__ uint4 sr_words(const PhiloxKeys& rk, uint32_t stream_id, uint64_t idx8) {
  return philox4x32_10((uint32_t)idx8, (uint32_t)(idx8 >> 32), stream_id, 0u, rk);
}

// ---------------------------------------------------------------------------------------------------------
// Random Hadamard transformation along k (paper Sec. 4.1): x' = (x S) H with H = diag(H_16, H_16, ...), the orthonormal
// Sylvester matrix (entries +-1/4), and S a random sign diagonal that depends on k only.
//   * sign of k: bit (k % 128) of the Philox block with counter (k / 128, 0, rht_stream, 0x5348), key = seed; set = -1;
//   * arithmetic: v[i] = x[i] * (s_i / 4) (exact), then four butterfly stages h = 1, 2, 4, 8 in binary32.
// ---------------------------------------------------------------------------------------------------------
__device__ __forceinline__ uint4 rht_sign_words(uint64_t seed, uint32_t rht_stream, uint64_t group128) {
  return philox4x32_10((uint32_t)group128, (uint32_t)(group128 >> 32), rht_stream, 0x5348u, (uint32_t)seed,
                       (uint32_t)(seed >> 32));
}
__device__ __forceinline__ uint32_t rht_pick_word(const uint4& w, uint32_t q) {
  return q == 0 ? w.x : q == 1 ? w.y : q == 2 ? w.z : w.w;
}
// the 16 sign bits of k0 .. k0 + 15 (k0 a multiple of 16), bit i for k0 + i
__device__ __forceinline__ uint32_t rht_sign16(uint64_t seed, uint32_t rht_stream, int64_t k0) {
  const uint4 w = rht_sign_words(seed, rht_stream, (uint64_t)k0 >> 7);
  return (rht_pick_word(w, ((uint32_t)k0 >> 5) & 3u) >> ((uint32_t)k0 & 16u)) & 0xFFFFu;
}
// +-1/4 for position kk (0..127) of a 128-group
__device__ __forceinline__ float rht_factor(const uint4& w, uint32_t kk) {
  return __uint_as_float(0x3E800000u | ((rht_pick_word(w, kk >> 5) >> (kk & 31u)) << 31));
}
__device__ __forceinline__ void rht_scale16(float (&v)[16], uint32_t sign16) {
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __fmul_rn(v[i], __uint_as_float(0x3E800000u | ((sign16 << (31 - i)) & 0x80000000u)));
}
__device__ __forceinline__ void hadamard16_butterflies(float (&v)[16]) {
#pragma unroll
  for (int h = 1; h < 16; h <<= 1) {
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      if ((i & h) == 0) {
        const float a = v[i], b = v[i + h];
        v[i] = __fadd_rn(a, b);
        v[i + h] = __fsub_rn(a, b);
      }
    }
  }
}

// ---------------------------------------------------------------------------------------------------------
// Element rounding to E2M1 (paper Sec. 2.1). Codes: sign << 3 | magnitude index.
// ---------------------------------------------------------------------------------------------------------
// a * c and b * c rounded to nearest / up: one packed instruction.
__device__ __forceinline__ void mul2_rn(float a, float b, float c, float& ra, float& rb) {
  asm("{.reg .b64 p, q;\nmov.b64 p, {%2, %3};\nmov.b64 q, {%4, %4};\nmul.rn.f32x2 p, p, q;\nmov.b64 {%0, %1}, p;}" : "=f"(ra), "=f"(rb) : "f"(a), "f"(b), "f"(c));
}
__device__ __forceinline__ void mul2_up(float a, float b, float c, float& ra, float& rb) {
  asm("{.reg .b64 p, q;\nmov.b64 p, {%2, %3};\nmov.b64 q, {%4, %4};\nmul.rp.f32x2 p, p, q;\nmov.b64 {%0, %1}, p;}" : "=f"(ra), "=f"(rb) : "f"(a), "f"(b), "f"(c));
}

// Round-to-nearest (ties to the even code, saturating) of 8 scaled values, packed low nibble first.
__device__ __forceinline__ uint32_t e2m1x8_rtn(const float (&y)[8]) {
  uint32_t out;
  asm("{\n"
      ".reg .b8 b0, b1, b2, b3;\n"
      "cvt.rn.satfinite.e2m1x2.f32 b0, %2, %1;\n"
      "cvt.rn.satfinite.e2m1x2.f32 b1, %4, %3;\n"
      "cvt.rn.satfinite.e2m1x2.f32 b2, %6, %5;\n"
      "cvt.rn.satfinite.e2m1x2.f32 b3, %8, %7;\n"
      "mov.b32 %0, {b0, b1, b2, b3};\n"
      "}"
      : "=r"(out)
      : "f"(y[0]), "f"(y[1]), "f"(y[2]), "f"(y[3]), "f"(y[4]), "f"(y[5]), "f"(y[6]), "f"(y[7]));
  return out;
}

// Stochastic rounding. For an element with 16-bit draw u the rule is
//     round the magnitude up  iff  (u + 0.5) / 65536 < (a - q1) / (q2 - q1),   a = min(|y|, 6) in [q1, q2).
// It is evaluated exactly with one integer multiply-add on the bits of a float:
//   * w = a * 2^-126, rounded up. E2M1 is spaced evenly below 1 and by binades above, as binary32 is below and above 2^-126, so the
//     cell of a is bits(w) >> 22 (0 .. 7) everywhere, and the low 22 bits are the position inside the cell in units of 2^-22 of its
//     width. The product is exact for a >= 1; below, it is ceil(a * 2^23) in units of 2^-149 (an integer n is < x iff n < ceil(x);
//     when the ceiling reaches the next cell the position was within 2^-24 of its end, where every draw rounds up).
//   * f + ((~u & 0xFFFF) << 6) + 31 reaches 2^22 iff the position f > (2u + 1) << 5. Four times that,
//         v = 4 * bits + ((~u & 0xFFFF) << 8) + 127 = 4 * bits - c,   c = (u << 8) + 129 - 2^24,
//     has the magnitude index of the result as its top byte, and c is the draw's two bytes between two constant ones: one byte
//     permutation per element.
// The codes' bytes are then collected by byte permutations, even and odd elements apart, and the signs likewise. Instructions executed per
// element (counters): the whole row kernel 18.0, columns 19.3, from codes 21.0, against 22.1, 23.3 and 25.4 of an earlier form (a second
// mapping for a < 1, the draw brought to bits 12 .. 27 by multiply-adds, sign and code moved into place element by element); rows to nearest
// 9.7. us, 16384 x 8192, before / after: rows 114.6 / 100.1, columns 129.2 / 108.6, from codes 162.5 / 141.5 (1x128 outer scales), and
// 16384 x 2816 with one scale and the amax pass 63.0 / 57.4, 62.7 / 58.0, 48.2 / 42.1.
// The busiest pipe is the ALU's (16 lanes a cycle; 63 - 64 % of the cycles, as many as the issue slots; what keeps both from more is not
// known): the generator's logic operations, the permutations, the clamp, and the two cycles of that pipe which each widening multiply takes
// beside its four of the multiply pipe. Measured and not better: packing by dp4a, the
// generator's high halves by FP64 FMAs, its first two rounds folded.
//
// Stochastic rounding of 8 scaled values with the draws packed in w (two 16-bit draws per word), packed low nibble first. The
// sign bits are those of the scaled values.
__device__ __forceinline__ uint32_t e2m1x8_sr(const float (&y)[8], const uint4& w) {
  const uint32_t ww[4] = {w.x, w.y, w.z, w.w};
  uint32_t v[8];
#pragma unroll
  for (int e = 0; e < 8; e += 2) {
    float w0, w1;
    mul2_up(fminf(fabsf(y[e]), 6.0f), fminf(fabsf(y[e + 1]), 6.0f), 0x1p-126f, w0, w1);
    // bytes of c from the low one: 0x81, the draw's two, 0xFF
    v[e] = __float_as_uint(w0) * 4u - __byte_perm(ww[e >> 1], 0xFF81u, 0x5104);
    v[e + 1] = __float_as_uint(w1) * 4u - __byte_perm(ww[e >> 1], 0xFF81u, 0x5324);
  }
  auto top_bytes = [](uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    return __byte_perm(__byte_perm(a, b, 0x0073), __byte_perm(c, d, 0x0073), 0x5410);
  };
  auto bits = [&](int e) { return __float_as_uint(y[e]); };
  const uint32_t code = top_bytes(v[0], v[2], v[4], v[6]) + top_bytes(v[1], v[3], v[5], v[7]) * 16u;
  const uint32_t even = top_bytes(bits(0), bits(2), bits(4), bits(6)), odd = top_bytes(bits(1), bits(3), bits(5), bits(7));
  return code | ((even >> 4) & 0x08080808u) | (odd & 0x80808080u);
}

// E2M1 code -> value, as float.
__device__ __forceinline__ float e2m1_decode(uint32_t code) {
  const uint32_t m = code & 7u;
  // magnitudes 0, .5, 1, 1.5, 2, 3, 4, 6: exponent field e = m >> 1, mantissa bit m & 1
  const uint32_t e = m >> 1, f = m & 1u;
  const uint32_t bits = (e == 0) ? (f ? 0x3F000000u : 0u) : (((126u + e) << 23) | (f << 22));
  return __uint_as_float(bits | ((code & 8u) << 28));
}

// Decode 8 packed E2M1 codes times one E4M3 scale times the global scale into 8 floats:
// x_hat = (P * S_block) * S_global; the inner product is exact in FP16 (6 significant bits, |value| <= 2688).
__device__ __forceinline__ void decode8(uint32_t word, uint32_t sf_byte, float sg, float* out) {
  uint32_t h[4];
  asm("{\n"
      ".reg .b8 b0, b1, b2, b3;\n"
      "mov.b32 {b0, b1, b2, b3}, %4;\n"
      "cvt.rn.f16x2.e2m1x2 %0, b0;\n"
      "cvt.rn.f16x2.e2m1x2 %1, b1;\n"
      "cvt.rn.f16x2.e2m1x2 %2, b2;\n"
      "cvt.rn.f16x2.e2m1x2 %3, b3;\n"
      "}"
      : "=r"(h[0]), "=r"(h[1]), "=r"(h[2]), "=r"(h[3])
      : "r"(word));
  uint32_t s2;
  asm("{.reg .b16 t; cvt.u16.u32 t, %1; cvt.rn.f16x2.e4m3x2 %0, t;}" : "=r"(s2) : "r"(sf_byte | (sf_byte << 8)));
  const __half2 sb2 = *reinterpret_cast<__half2*>(&s2);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float2 f = __half22float2(__hmul2(*reinterpret_cast<__half2*>(&h[i]), sb2));
    out[2 * i] = __fmul_rn(f.x, sg);
    out[2 * i + 1] = __fmul_rn(f.y, sg);
  }
}

// Decode 8 packed E2M1 codes times one E4M3 scale into four packed FP16 pairs (element 2i in the low half of word i):
// P * S_block, exact in FP16 (at most 7 significant bits, 2^-10 <= |value| <= 2688 or zero).
__device__ __forceinline__ void decode8_h2(uint32_t word, uint32_t sf_byte, uint32_t (&out)[4]) {
  uint32_t h[4];
  asm("{\n"
      ".reg .b8 b0, b1, b2, b3;\n"
      "mov.b32 {b0, b1, b2, b3}, %4;\n"
      "cvt.rn.f16x2.e2m1x2 %0, b0;\n"
      "cvt.rn.f16x2.e2m1x2 %1, b1;\n"
      "cvt.rn.f16x2.e2m1x2 %2, b2;\n"
      "cvt.rn.f16x2.e2m1x2 %3, b3;\n"
      "}"
      : "=r"(h[0]), "=r"(h[1]), "=r"(h[2]), "=r"(h[3])
      : "r"(word));
  uint32_t s2;
  asm("{.reg .b16 t; cvt.u16.u32 t, %1; cvt.rn.f16x2.e4m3x2 %0, t;}" : "=r"(s2) : "r"(sf_byte | (sf_byte << 8)));
  const __half2 sb2 = *reinterpret_cast<__half2*>(&s2);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const __half2 p = __hmul2(*reinterpret_cast<__half2*>(&h[i]), sb2);
    out[i] = *reinterpret_cast<const uint32_t*>(&p);
  }
}

// Scale, round and pack one 16-element inner block (two code words).
template <bool SR>
__device__ __forceinline__ uint2 quantize_block16(const float (&x)[16], float rcp, const PhiloxKeys& pk, uint32_t stream_id,
                                                  uint64_t idx8) {
  float y0[8], y1[8];
#pragma unroll
  for (int i = 0; i < 8; i += 2) {
    mul2_rn(x[i], x[i + 1], rcp, y0[i], y0[i + 1]);
    mul2_rn(x[8 + i], x[9 + i], rcp, y1[i], y1[i + 1]);
  }
  uint2 out;
  if (SR) {
    out.x = e2m1x8_sr(y0, sr_words(pk, stream_id, idx8));
    out.y = e2m1x8_sr(y1, sr_words(pk, stream_id, idx8 + 1));
  } else {
    out.x = e2m1x8_rtn(y0);
    out.y = e2m1x8_rtn(y1);
  }
  return out;
}

// Byte offset of scale (r, kb) in the TILED128x4 layout with n_ktiles4 = (number of k-blocks, padded to 16) / 4.
__device__ __forceinline__ size_t sf_tiled_offset(int64_t r, int64_t kb, int64_t kb_padded) {
  const int64_t tile = (r >> 7) * (kb_padded >> 2) + (kb >> 2);
  return (size_t)tile * 512 + (size_t)((r & 31) * 16 + ((r >> 5) & 3) * 4 + (kb & 3));
}

}  // namespace nvfp4
