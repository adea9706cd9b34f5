// Block-scaled FP4 GEMM for sm_100a (the "FP4 MM" of the paper's Sec. 2.3):
//     C[m, n] = sum_k (Pa Sba Sga)[m, k] (Pb Sbb Sgb)[n, k],  both operands packed along k.
//
// Design (one CTA per SM, persistent over output tiles, warp-specialised):
//   warp 0      TMA producer: per 256-wide k tile, two tiled bulk-tensor loads (A, B codes; 128-byte swizzle) and
//               two plain bulk copies (the 2 KB of E4M3 scales each operand tile needs, contiguous in the
//               TILED128x4 layout) into a ring of shared-memory stages, completion on an mbarrier.
//   warp 1      MMA issuer: copies the scales shared -> tensor memory (tcgen05.cp) and issues
//               tcgen05.mma kind::mxf4nvf4 block_scale (E2M1 data, UE4M3 scale per 16 elements, K = 64 per
//               instruction, FP32 accumulators in tensor memory, two accumulator buffers).
//   warps 2..9  epilogue (two warps per tensor-memory lane quadrant, half of the tile's columns each): tcgen05.ld the
//               accumulator, apply the FP32 global scales, convert, stage 128-byte row pieces in shared memory and
//               write them with bulk tensor stores. (The outer-block variant further down has its own roles.)
// Every wait on an mbarrier is bounded (Params::wait_limit clock cycles); when a bound is hit the kernel raises a
// status word, all roles drain and the CTA frees its tensor memory and exits.
#include <cuda.h>
#include <cuda_bf16.h>

#include "nvfp4_device.cuh"
#include "nvfp4_internal.h"
#include "nvfp4_tc.cuh"

namespace nvfp4 {

namespace {

// Single-CTA kernel: 128 x 128 output tiles.
constexpr int BN = 128;
struct Cfg {
  static constexpr uint32_t B_BYTES = BN * BK / 2;
  static constexpr uint32_t SFB_BYTES = 2048;
  static constexpr uint32_t STAGE_BYTES = A_BYTES + B_BYTES + SFA_BYTES + SFB_BYTES;  // 36 KB, multiple of 1024
  static constexpr int STAGES = 5;
  // epilogue staging for bulk tensor stores: per epilogue warp one 32-row x 128-byte buffer
  static constexpr uint32_t STAGING_BYTES = 8 * 4096;
  static constexpr uint32_t SMEM_BYTES = STAGES * STAGE_BYTES + STAGING_BYTES + 1024 /*align slack*/ + 256 /*barriers*/;
  // tensor memory columns: two accumulators (a tile's epilogue runs under the next tile's MMAs), the optional
  // high-precision accumulator, then four scale buffers (A: 16 columns, B: 16)
  static constexpr uint32_t ACC_COLS = BN;
  static constexpr uint32_t ACC_BUFS = 2;
  // Eight epilogue warps: two per tensor-memory lane quadrant, each taking half of the tile's columns (a tile's
  // epilogue with four warps took 1.9 us and bounded every product with K <= 1024).
  static constexpr int EPI_WARPS = 8;
  static constexpr int THREADS = 64 + 32 * EPI_WARPS;
  static constexpr uint32_t SF_COLS = 32;
  static constexpr uint32_t TMEM_COLS = 512;
  static_assert(ACC_BUFS * ACC_COLS + 128 + 4 * SF_COLS <= TMEM_COLS, "tensor memory budget");
};

struct Params {
  const uint8_t* a_sf;
  const uint8_t* b_sf;
  const float* a_gscale;
  const float* b_gscale;
  void* C;
  int64_t ldc;
  int64_t M, N;
  int32_t k_tiles;        // number of 256-wide k tiles
  int32_t k_chunks;       // number of 128-wide k chunks (BLOCK128 variant)
  int64_t g_per_row;      // global scales per operand row in BLOCK128 mode
  int32_t sf_tiles_a;     // 512-byte scale tiles per 128-row tile of A (= padded k-blocks / 4)
  int32_t sf_tiles_b;
  int32_t m_tiles, n_tiles;
  int32_t c_is_f32, accumulate;
  int32_t hp_k_tiles;     // OutControl: 64-wide BF16 k tiles of the high-precision side product (0 = none)
  int32_t starve;         // test hook: the first stage's "full" barrier expects 16 bytes more than will ever arrive
  long long wait_limit;   // bound of every wait, in clock cycles
  int32_t* dev_status;
};

// The output tiles of a persistent CTA (or pair), first, first + step, ...: row and column of the tile by additions (there are
// fewer than 2^31 tiles: that many are 70 TB of C). Two 64-bit divisions per tile in every role are what this replaces; at short K,
// where a tile is a few k tiles, they showed: 8192 x 3072 x 1024 on 256 x 192 tiles 16.9 -> 16.0 us.
struct TileWalk {
  uint32_t index, m, n;
  __device__ __forceinline__ TileWalk(uint32_t first, uint32_t step, uint32_t n_tiles) : index(first), step_(step), n_tiles_(n_tiles) {
    m = first / n_tiles;
    n = first - m * n_tiles;
    dm_ = step / n_tiles;
    dn_ = step - dm_ * n_tiles;
  }
  __device__ __forceinline__ void next() {
    index += step_;
    m += dm_;
    n += dn_;
    if (n >= n_tiles_) {
      n -= n_tiles_;
      ++m;
    }
  }

 private:
  uint32_t step_, n_tiles_, dm_, dn_;
};

// When accumulating: adds the old C to W consecutive values of output row m from column n0 (a full chunk inside C).
template <int W>
__device__ __forceinline__ void add_existing(const Params& p, int64_t m, int64_t n0, float (&o)[W]) {
  if (p.accumulate) {
    if (p.c_is_f32) {
      const float* cp = reinterpret_cast<const float*>(p.C) + m * p.ldc + n0;
#pragma unroll
      for (int j = 0; j < W; j += 4) {
        const float4 q = *reinterpret_cast<const float4*>(cp + j);
        o[j] += q.x; o[j + 1] += q.y; o[j + 2] += q.z; o[j + 3] += q.w;
      }
    } else {
      const uint16_t* cp = reinterpret_cast<const uint16_t*>(p.C) + m * p.ldc + n0;
#pragma unroll
      for (int j = 0; j < W; j += 8) {
        const uint4 old = *reinterpret_cast<const uint4*>(cp + j);
        const uint32_t ow[4] = {old.x, old.y, old.z, old.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          o[j + 2 * q] += bf16_lo(ow[q]);
          o[j + 2 * q + 1] += bf16_hi(ow[q]);
        }
      }
    }
  }
}

// The columns of a chunk that sticks out past N (values final: scaled, accumulated): plain element stores, nothing beyond
// column N - 1 is touched. The bulk tensor store is kept for whole chunks only: its clipping at the edge of C was seen to
// overwrite the row's padding up to the next 16-byte boundary.
template <int W>
__device__ __forceinline__ void store_ragged(const Params& p, int64_t m, int64_t n0, const float (&o)[W]) {
  if (p.c_is_f32) {
    float* cp = reinterpret_cast<float*>(p.C) + m * p.ldc + n0;
#pragma unroll
    for (int j = 0; j < W; ++j)
      if (n0 + j < p.N) cp[j] = o[j];
  } else {
    __nv_bfloat16* cp = reinterpret_cast<__nv_bfloat16*>(p.C) + m * p.ldc + n0;
#pragma unroll
    for (int j = 0; j < W; ++j)
      if (n0 + j < p.N) cp[j] = __float2bfloat16_rn(o[j]);
  }
}

template <int GS>
__global__ void __launch_bounds__(Cfg::THREADS, 1)
gemm_nvfp4_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                  const __grid_constant__ CUtensorMap tmC, const __grid_constant__ CUtensorMap tmAh,
                  const __grid_constant__ CUtensorMap tmBh, const Params p) {
  using C = Cfg;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t staging_base = smem_base + C::STAGES * C::STAGE_BYTES;
  const uint32_t bar_base = staging_base + C::STAGING_BYTES;
  // barriers: full[STAGES], empty[STAGES], acc_full[2], acc_empty[2], drain
  auto full_bar = [&](int s) { return bar_base + 8u * s; };
  auto empty_bar = [&](int s) { return bar_base + 8u * (C::STAGES + s); };
  auto acc_full_bar = [&](int b) { return bar_base + 8u * (2 * C::STAGES + b); };
  auto acc_empty_bar = [&](int b) { return bar_base + 8u * (2 * C::STAGES + 2 + b); };
  const uint32_t drain_bar = bar_base + 8u * (2 * C::STAGES + 4);
  const uint32_t hp_empty_bar = bar_base + 8u * (2 * C::STAGES + 5);  // high-precision accumulator drained
  // tensor-memory columns of the optional high-precision accumulator and of the scale buffers
  const uint32_t hp_cols = p.hp_k_tiles > 0 ? 128u : 0u;
  const uint32_t hp_tmem_col = C::ACC_BUFS * C::ACC_COLS;
  const uint32_t sf_tmem_col = C::ACC_BUFS * C::ACC_COLS + hp_cols;
  __shared__ uint32_t tmem_base_slot;
  __shared__ int abort_flag_s;
  volatile int* abort_flag = &abort_flag_s;

  const int warp = uniform_warp_index(), lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    abort_flag_s = 0;
    for (int s = 0; s < C::STAGES; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(acc_full_bar(b), 1);
      mbar_init(acc_empty_bar(b), C::EPI_WARPS);
    }
    mbar_init(drain_bar, 1);
    mbar_init(hp_empty_bar, C::EPI_WARPS);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_slot)),
                 "r"(C::TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_slot;
  pdl_prologue();  // everything above touched only shared and tensor memory

  const uint32_t num_tiles = (uint32_t)p.m_tiles * (uint32_t)p.n_tiles;

  if (warp == 0) {
    // ===================================== TMA producer (warp stays converged) ===============================
    const uint32_t leader = elect_leader();
    uint32_t it = 0, s = 0, wait_parity = 1;  // running stage and the parity its "empty" barrier is waited with
    bool ok = true;
    for (TileWalk t((uint32_t)blockIdx.x, (uint32_t)gridDim.x, (uint32_t)p.n_tiles); t.index < num_tiles && ok; t.next()) {
      const int32_t mt = (int32_t)t.m, nt = (int32_t)t.n;
      const uint8_t* sfa_src = p.a_sf + (size_t)mt * p.sf_tiles_a * 512;
      const uint8_t* sfb_src = p.b_sf + (size_t)nt * p.sf_tiles_b * 512;
      for (int32_t kt = 0; kt < p.k_tiles; ++kt, ++it, s = (s + 1 == (uint32_t)C::STAGES ? 0u : s + 1), wait_parity ^= (s == 0)) {
        ok = __all_sync(0xFFFFFFFFu, mbar_wait(empty_bar(s), wait_parity, abort_flag, p.dev_status, p.wait_limit));
        if (!ok) break;
        const uint32_t st = smem_base + s * C::STAGE_BYTES;
        // (test hook of the bounded waits: with `starve` the very first stage never completes)
        mbar_expect_tx(full_bar(s), C::STAGE_BYTES + ((p.starve && it == 0) ? 16u : 0u), leader);
        tma_load_2d(st, &tmA, kt * (BK / 2), mt * BM, full_bar(s), leader);
        tma_load_2d(st + A_BYTES, &tmB, kt * (BK / 2), nt * BN, full_bar(s), leader);
        bulk_load(st + A_BYTES + C::B_BYTES, sfa_src + (size_t)kt * 2048, 2048, full_bar(s), leader);
        bulk_load(st + A_BYTES + C::B_BYTES + SFA_BYTES, sfb_src + (size_t)kt * 2048, 2048, full_bar(s), leader);
      }
      // OutControl: the BF16 outlier channels of both operands, 64 per stage, into the same stage buffers
      for (int32_t h = 0; h < p.hp_k_tiles && ok; ++h, ++it, s = (s + 1 == (uint32_t)C::STAGES ? 0u : s + 1), wait_parity ^= (s == 0)) {
        ok = __all_sync(0xFFFFFFFFu, mbar_wait(empty_bar(s), wait_parity, abort_flag, p.dev_status, p.wait_limit));
        if (!ok) break;
        const uint32_t st = smem_base + s * C::STAGE_BYTES;
        mbar_expect_tx(full_bar(s), A_BYTES + C::B_BYTES, leader);
        tma_load_2d(st, &tmAh, h * 64, mt * BM, full_bar(s), leader);
        tma_load_2d(st + A_BYTES, &tmBh, h * 64, nt * BN, full_bar(s), leader);
      }
    }
    if (!ok) {
      // give the copies already in flight a bounded time to land before the CTA may exit
      const uint32_t n_back = it < (uint32_t)C::STAGES ? it : (uint32_t)C::STAGES;
      for (uint32_t j = 0; j < n_back; ++j) {
        const uint32_t f = it - 1 - j;
        const long long t0 = clock64();
        while (!mbar_try(full_bar(f % C::STAGES), (f / C::STAGES) & 1) && clock64() - t0 < p.wait_limit) {
        }
      }
    }
  } else if (warp == 1) {
    // ===================================== MMA issuer (warp stays converged) =================================
    const uint32_t leader = elect_leader();
    const uint32_t idesc = instr_desc<BN>();
    // The issuing warp's own instruction stream is what limits a 128 x 128 tile (13 tensor-core instructions per 256 cycles of
    // math), so the loop keeps it short: running stage / phase counters instead of divisions, descriptors formed by adding
    // to the low word of the first stage's (an address enters as address >> 4 in the low 14 bits; the high words are
    // constants), and the try on the NEXT stage's barrier issued before this stage's instructions so that its latency
    // overlaps them.
    uint32_t it = 0, tile_it = 0, stage = 0, phase = 0;
    bool ok = true;
    bool ready = false;
    constexpr uint32_t SW_HI = (uint32_t)((((uint64_t)64 << 32) | ((uint64_t)1 << 46) | ((uint64_t)2 << 61)) >> 32);
    constexpr uint32_t SF_HI = (uint32_t)((((uint64_t)8 << 32) | ((uint64_t)1 << 46)) >> 32);
    const uint32_t a_lo0 = (uint32_t)desc_sw128(smem_base), sfa_lo0 = (uint32_t)desc_sf(smem_base + A_BYTES + C::B_BYTES);
    for (TileWalk t((uint32_t)blockIdx.x, (uint32_t)gridDim.x, (uint32_t)p.n_tiles); t.index < num_tiles && ok; t.next(), ++tile_it) {
      const uint32_t ab = tile_it % C::ACC_BUFS;
      ok = __all_sync(0xFFFFFFFFu, mbar_wait(acc_empty_bar(ab), ((tile_it / C::ACC_BUFS) & 1) ^ 1, abort_flag, p.dev_status, p.wait_limit));
      if (!ok) break;
      tc_fence_after();
      const uint32_t d_tmem = tmem_base + ab * C::ACC_COLS;
      for (int32_t kt = 0; kt < p.k_tiles; ++kt, ++it) {
        if (!ready) {
          ok = __all_sync(0xFFFFFFFFu, mbar_wait(full_bar(stage), phase, abort_flag, p.dev_status, p.wait_limit));
          if (!ok) break;
        }
        tc_fence_after();
        const uint32_t st16 = stage * (uint32_t)(C::STAGE_BYTES >> 4);
        const uint32_t this_empty = empty_bar(stage);
        if (++stage == (uint32_t)C::STAGES) {
          stage = 0;
          phase ^= 1u;
        }
        const uint32_t next_try = mbar_test(full_bar(stage), phase);
        const uint32_t sf_tmem = tmem_base + sf_tmem_col + (it & 3) * C::SF_COLS;
        // Scales of this k tile: shared memory -> tensor memory. Per 64-wide k step: 4 columns for the 128 rows
        // of A, 4 per 128 rows of B.
#pragma unroll
        for (int kk = 0; kk < BK / 64; ++kk) {
          tc_cp_sf(sf_tmem + kk * 4, ((uint64_t)SF_HI << 32) | (sfa_lo0 + st16 + kk * 32), leader);
          tc_cp_sf(sf_tmem + 16 + kk * 4, ((uint64_t)SF_HI << 32) | (sfa_lo0 + st16 + (SFA_BYTES >> 4) + kk * 32), leader);
        }
#pragma unroll
        for (int kk = 0; kk < BK / 64; ++kk)
          tc_mma_nvf4(d_tmem, ((uint64_t)SW_HI << 32) | (a_lo0 + st16 + kk * 2), ((uint64_t)SW_HI << 32) | (a_lo0 + st16 + (A_BYTES >> 4) + kk * 2),
                      idesc, sf_tmem + kk * 4, sf_tmem + 16 + kk * 4, (kt | kk) != 0, leader);
        tc_commit(this_empty, leader);  // stage reusable once these MMAs have read it
        ready = __all_sync(0xFFFFFFFFu, next_try);
      }
      if (p.hp_k_tiles > 0 && ok) {
        // high-precision side product into its own accumulator (single buffer: wait until the previous tile's epilogue
        // has drained it, which happened a whole main loop ago)
        ok = __all_sync(0xFFFFFFFFu, mbar_wait(hp_empty_bar, (tile_it & 1) ^ 1, abort_flag, p.dev_status, p.wait_limit));
        if (!ok) break;
        tc_fence_after();
        const uint32_t idesc_bf16 = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
        for (int32_t h = 0; h < p.hp_k_tiles; ++h, ++it) {
          if (!ready) {
            ok = __all_sync(0xFFFFFFFFu, mbar_wait(full_bar(stage), phase, abort_flag, p.dev_status, p.wait_limit));
            if (!ok) break;
          }
          tc_fence_after();
          const uint32_t st = smem_base + stage * C::STAGE_BYTES;
          const uint32_t this_empty = empty_bar(stage);
          if (++stage == (uint32_t)C::STAGES) {
            stage = 0;
            phase ^= 1u;
          }
          const uint32_t next_try = mbar_test(full_bar(stage), phase);
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)  // 64 BF16 = one 128-byte swizzle row = four K = 16 steps of 32 bytes
            tc_mma_bf16(tmem_base + hp_tmem_col, desc_sw128(st + kk * 32), desc_sw128(st + A_BYTES + kk * 32), idesc_bf16,
                        (h | kk) != 0, leader);
          tc_commit(this_empty, leader);
          ready = __all_sync(0xFFFFFFFFu, next_try);
        }
        if (!ok) break;
      }
      if (ok) tc_commit(acc_full_bar(ab), leader);
    }
    // make sure nothing issued is still running before tensor memory is freed
    tc_commit(drain_bar, leader);
    {
      const long long t0 = clock64();
      while (!mbar_try(drain_bar, 0) && clock64() - t0 < p.wait_limit) {
      }
    }
  } else {
    // ===================================== epilogue ========================================================
    const int quad = warp & 3;  // tensor-memory lane quadrant this warp may read
    uint32_t tile_it = 0;
    bool ok = true;
    float alpha = 1.0f;
    if (GS == kGsTensor) alpha = __fmul_rn(p.a_gscale[0], p.b_gscale[0]);
    for (TileWalk t((uint32_t)blockIdx.x, (uint32_t)gridDim.x, (uint32_t)p.n_tiles); t.index < num_tiles && ok; t.next(), ++tile_it) {
      const int32_t mt = (int32_t)t.m, nt = (int32_t)t.n;
      const uint32_t ab = tile_it % C::ACC_BUFS;
      if (!(ok = mbar_wait(acc_full_bar(ab), (tile_it / C::ACC_BUFS) & 1, abort_flag, p.dev_status, p.wait_limit))) break;
      tc_fence_after();
      const int64_t m = (int64_t)mt * BM + quad * 32 + lane;
      float sa = 1.0f;
      if (GS == kGsRow && m < p.M) sa = p.a_gscale[m];
      const int half = (warp - 2) >> 2;  // which half of the tile's columns this warp owns
      {
        // Stage 128-byte row pieces (32 FP32 or 64 BF16 columns) in shared memory with the 128-byte swizzle and let the
        // bulk-tensor engine write them: full lines, clipped at the edges of C, asynchronous.
        const uint32_t my_stage = staging_base + (uint32_t)(warp - 2) * 4096u;
        const int64_t m0 = (int64_t)mt * BM + quad * 32;
        if (p.c_is_f32) {
#pragma unroll 1
          for (int c0 = half * (BN / 2); c0 < (half + 1) * (BN / 2); c0 += 32) {
            uint32_t v[32];
            tc_ld32(tmem_base + ((uint32_t)(quad * 32) << 16) + ab * C::ACC_COLS + c0, v);
            tc_wait_ld();
            const int64_t n0 = (int64_t)nt * BN + c0;
            if (n0 >= p.N) break;
            float o[32], sgb[32];
            if (GS == kGsRow) load_sgb32(p.b_gscale, n0, p.N, sgb);
#pragma unroll
            for (int j = 0; j < 32; ++j) {
              float sc = alpha;
              if (GS == kGsRow) sc = __fmul_rn(sa, sgb[j]);
              o[j] = __uint_as_float(v[j]) * sc;
            }
            if (hp_cols) {
              tc_ld32(tmem_base + ((uint32_t)(quad * 32) << 16) + hp_tmem_col + c0, v);
              tc_wait_ld();
              if (p.k_tiles > 0) {
#pragma unroll
                for (int j = 0; j < 32; ++j) o[j] += __uint_as_float(v[j]);
              } else {  // dense BF16 product alone (no FP4 part: the main accumulator was never written): scaled like one
#pragma unroll
                for (int j = 0; j < 32; ++j) o[j] = __uint_as_float(v[j]) * alpha;
              }
            }
            if (p.accumulate && m < p.M) {
              if (n0 + 32 <= p.N) {
                add_existing<32>(p, m, n0, o);
              } else {
#pragma unroll
                for (int j = 0; j < 32; ++j)
                  if (n0 + j < p.N) o[j] += reinterpret_cast<const float*>(p.C)[m * p.ldc + n0 + j];
              }
            }
            if (n0 + 32 > p.N) {  // ragged last chunk of the row
              if (m < p.M) store_ragged<32>(p, m, n0, o);
              continue;
            }
            const uint32_t buf = my_stage;
            if (lane == 0) bulk_wait_read<0>();  // the previous store from this buffer has read it
            __syncwarp();
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const uint32_t dst = buf + (uint32_t)lane * 128u + (uint32_t)((j ^ (lane & 7)) << 4);
              asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "r"(__float_as_uint(o[4 * j])),
                           "r"(__float_as_uint(o[4 * j + 1])), "r"(__float_as_uint(o[4 * j + 2])),
                           "r"(__float_as_uint(o[4 * j + 3]))
                           : "memory");
            }
            fence_async_smem();
            __syncwarp();
            if (lane == 0) {
              tma_store_2d(&tmC, buf, (int32_t)n0, (int32_t)m0);
              bulk_commit();
            }
          }
        } else {
#pragma unroll 1
          for (int c0 = half * (BN / 2); c0 < (half + 1) * (BN / 2); c0 += 64) {
            uint32_t v[32], v2[32];
            tc_ld32(tmem_base + ((uint32_t)(quad * 32) << 16) + ab * C::ACC_COLS + c0, v);
            tc_ld32(tmem_base + ((uint32_t)(quad * 32) << 16) + ab * C::ACC_COLS + c0 + 32, v2);
            tc_wait_ld();
            const int64_t n0 = (int64_t)nt * BN + c0;
            if (n0 >= p.N) break;
            float o[64];
            {
              float sgb[32];
              if (GS == kGsRow) load_sgb32(p.b_gscale, n0, p.N, sgb);
#pragma unroll
              for (int j = 0; j < 32; ++j) o[j] = __uint_as_float(v[j]) * (GS == kGsRow ? __fmul_rn(sa, sgb[j]) : alpha);
              if (GS == kGsRow) load_sgb32(p.b_gscale, n0 + 32, p.N, sgb);
#pragma unroll
              for (int j = 0; j < 32; ++j) o[32 + j] = __uint_as_float(v2[j]) * (GS == kGsRow ? __fmul_rn(sa, sgb[j]) : alpha);
            }
            if (hp_cols) {
              tc_ld32(tmem_base + ((uint32_t)(quad * 32) << 16) + hp_tmem_col + c0, v);
              tc_ld32(tmem_base + ((uint32_t)(quad * 32) << 16) + hp_tmem_col + c0 + 32, v2);
              tc_wait_ld();
              if (p.k_tiles > 0) {
#pragma unroll
                for (int j = 0; j < 32; ++j) {
                  o[j] += __uint_as_float(v[j]);
                  o[32 + j] += __uint_as_float(v2[j]);
                }
              } else {
#pragma unroll
                for (int j = 0; j < 32; ++j) {
                  o[j] = __uint_as_float(v[j]) * alpha;
                  o[32 + j] = __uint_as_float(v2[j]) * alpha;
                }
              }
            }
            if (p.accumulate && m < p.M) {
              if (n0 + 64 <= p.N) {
                add_existing<64>(p, m, n0, o);
              } else {
#pragma unroll
                for (int j = 0; j < 64; ++j)
                  if (n0 + j < p.N) o[j] += __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(p.C)[m * p.ldc + n0 + j]);
              }
            }
            if (n0 + 64 > p.N) {  // ragged last chunk of the row
              if (m < p.M) store_ragged<64>(p, m, n0, o);
              continue;
            }
            const uint32_t buf = my_stage;
            if (lane == 0) bulk_wait_read<0>();
            __syncwarp();
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              uint32_t q[4];
#pragma unroll
              for (int h = 0; h < 4; ++h) {
                const __nv_bfloat162 hh = __floats2bfloat162_rn(o[8 * j + 2 * h], o[8 * j + 2 * h + 1]);
                q[h] = *reinterpret_cast<const uint32_t*>(&hh);
              }
              const uint32_t dst = buf + (uint32_t)lane * 128u + (uint32_t)((j ^ (lane & 7)) << 4);
              asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "r"(q[0]), "r"(q[1]), "r"(q[2]), "r"(q[3])
                           : "memory");
            }
            fence_async_smem();
            __syncwarp();
            if (lane == 0) {
              tma_store_2d(&tmC, buf, (int32_t)n0, (int32_t)m0);
              bulk_commit();
            }
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(acc_empty_bar(ab));
        if (hp_cols) mbar_arrive(hp_empty_bar);
      }
    }
    if (lane == 0) bulk_wait_all();  // this lane's bulk stores are complete before the CTA may exit
  }

  // ===================================== teardown ============================================================
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(C::TMEM_COLS) : "memory");
  }
}

// =========================================================================================================
// BLOCK128 variant: the FP32 global scale changes every 128 k (the paper's 1x128 outer block, Sec. 2.2), so a partial product can
// only be accumulated over 128 k inside tensor memory. The MMA warp writes each 128-k partial of a 128 x TN tile (two K = 64
// instructions) into one of two or three tensor-memory buffers; promotion warps pull it out, 32 rows x CW columns each, and promote it
// into FP32 register accumulators with the rank-1 scale SgA[m, kc] * SgB[n, kc] (packed f32x2 multiply + FMA).
//
// What bounds it: no pipe, but the chain of a partial. A packed operation issues every 2.8 cycles at best (timed in a loop from registers,
// two or more warps per scheduler), which is 540 cycles per partial of 192 columns against 200 of its MMAs; the kernel takes 790 to 840
// there at long K, about 620 with 128 columns and 380 with 64. Without the promotion's arithmetic 8192 x 1024 x 3072 still takes 26.5 of
// 36.8 us: bringing the operands, handing partials over and loading them from tensor memory is the larger part.
//   - Two or three promotion warps per scheduler: a warp's barrier, tensor-memory load and hand-over latencies (about 400 cycles per
//     partial) run under the others' arithmetic. With one (a 128 x 128 tile, four warps with 128 columns each) they add up:
//     760 cycles per 128 columns. 192 columns are what a register file of 128 a thread on average holds (setmaxnreg: 80 for the
//     four warps that load, issue and fetch scales, 144 for the others) with a buffer to spare in tensor memory. With 64 columns a
//     warp has 32 of them and both of its loads in flight at once.
//   - Fragments: the 16x256b load gives a thread 2 columns x 8 groups of 2 rows, i.e. 16 column scales and 4 row scales for 64
//     elements; with a thread per row it would be a column scale per element, read from shared memory by every warp.
//   - Scales come through shared memory, fetched by two warps in 16-byte pieces (below).
// us, with one group of four warps / now (tile width by block128_tile_cols): 8192 x 3072 x 1024 49.1 / 31.9, 8192 x 1024 x 3072 42.6 /
// 36.0, 3072 x 1024 x 8192 (FP32) 54.8 / 32.7, 1024 x 1024 x 8192 (FP32) 28.3 / 15.9, 4096^3 103.9 / 85.0. K <= 16384.
// =========================================================================================================
constexpr int64_t B128_MAX_K = 16384;
template <int TN_>
struct B128 {
  static constexpr int TN = TN_;                             // columns of a tile: 192, 128 or 64
  static constexpr int CW = TN == 64 ? 32 : 64;              // columns of a promotion warp (32 rows each)
  static constexpr int PROMO_WARPS = 4 * (TN / CW);          // warps 4 .. : twelve, or eight
  static constexpr int THREADS = 128 + 32 * PROMO_WARPS;     // warps 0 .. 3: loads, MMA, global scales (two)
  static constexpr int STAGES = TN == 192 ? 3 : 4;
  static constexpr int NBUF = TN == 192 ? 2 : 3;             // partials in tensor memory
  static constexpr int SC_SLOTS = 3;                         // ring of global-scale slots, four chunks each
  static constexpr int SF_TILES = TN == 192 ? 2 : 1;         // 128-row scale tiles that the B rows touch
  static constexpr uint32_t B_BYTES = TN * 128;
  static constexpr uint32_t SFB_BYTES = SF_TILES * 2048;
  static constexpr uint32_t STAGE_BYTES = A_BYTES + B_BYTES + SFA_BYTES + SFB_BYTES;  // 46, 36 or 28 KB
  static constexpr uint32_t STAGING_BYTES = PROMO_WARPS * 4096;                       // 32 rows x 128 bytes per promotion warp
  static constexpr uint32_t SC_CHUNK = (128 + TN) * 4;                                // SgA, then SgB of one chunk
  static constexpr uint32_t SC_BYTES = 4 * SC_CHUNK;
  static constexpr uint32_t SMEM_BYTES = STAGES * STAGE_BYTES + STAGING_BYTES + SC_SLOTS * SC_BYTES + 1024 + 256;
  static constexpr uint32_t SF_COLS = 16 + 16 * SF_TILES, SF_SETS = 2;  // tensor-memory columns of a k tile's block scales: of A, of B
  static_assert(NBUF * TN + SF_SETS * SF_COLS <= 512, "tensor memory budget");
  static_assert(STAGE_BYTES % 1024 == 0 && SMEM_BYTES <= 227 * 1024, "shared memory budget");
  static_assert(8 * (2 * STAGES + 2 * NBUF + 2 * SC_SLOTS + 1) <= 256, "barrier space");
};

// 16 rows x 64 columns of a partial: v[4 i + 2 q + e] is row 8 q + lane / 4, column 8 i + 2 (lane % 4) + e. Wait with tc_wait_ld.
__device__ __forceinline__ void tc_ld_16x256b_x8(uint32_t taddr, uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
      "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]),
        "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
        "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tc_ld_16x256b_x4(uint32_t taddr, uint32_t (&v)[16]) {  // (32 columns: i < 4)
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(taddr)
      : "memory");
}
// Four global scales of a row from chunk c on (c a multiple of four; 0 past the row's end); vec = floats that a load may take.
__device__ __forceinline__ float4 load_scales4(const float* row, int32_t c, int32_t chunks, int vec) {
  if (vec == 4) return __ldg(reinterpret_cast<const float4*>(row + c));
  float4 r = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  if (vec == 2) {
    const float2 a = __ldg(reinterpret_cast<const float2*>(row + c));
    r.x = a.x;
    r.y = a.y;
    if (c + 2 < chunks) {
      const float2 b = __ldg(reinterpret_cast<const float2*>(row + c + 2));
      r.z = b.x;
      r.w = b.y;
    }
  } else {
    r.x = __ldg(row + c);
    if (c + 1 < chunks) r.y = __ldg(row + c + 1);
    if (c + 2 < chunks) r.z = __ldg(row + c + 2);
    if (c + 3 < chunks) r.w = __ldg(row + c + 3);
  }
  return r;
}
__device__ __forceinline__ float4 lds128(uint32_t addr) {
  float4 r;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(r.x), "=f"(r.y), "=f"(r.z), "=f"(r.w) : "r"(addr));
  return r;
}

// 32 staged FP32 rows of 32 columns (128 bytes each, swizzled) to C from row m0 and column n0 on, element by element past N, added to
// the old C if asked for: four columns per lane, eight lanes per row. `stage_rows` stages them; the old values are on their way by then.
template <bool F32, typename Stage>
__device__ __forceinline__ void b128_store_rows(const Params& p, uint32_t stage, int lane, int64_t m0, int64_t n0, Stage stage_rows) {
  const int64_t n = n0 + 4 * (lane & 7), m = m0 + (lane >> 3);  // this lane's columns, its first row (every fourth from there)
  const bool all4 = n + 4 <= p.N;
  float* const cf = reinterpret_cast<float*>(p.C) + m * p.ldc + n;
  uint16_t* const ch = reinterpret_cast<uint16_t*>(p.C) + m * p.ldc + n;
  uint4 old[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) old[j] = make_uint4(0u, 0u, 0u, 0u);
  if (p.accumulate && all4) {
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      if (m + 4 * j < p.M) {
        if (F32) {
          old[j] = *reinterpret_cast<const uint4*>(cf + 4 * j * p.ldc);
        } else {
          const uint2 w = *reinterpret_cast<const uint2*>(ch + 4 * j * p.ldc);
          old[j].x = w.x;
          old[j].y = w.y;
        }
      }
    }
  }
  stage_rows();
  __syncwarp();
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int r = (lane >> 3) + 4 * j;
    float4 v = lds128(stage + (uint32_t)r * 128u + (uint32_t)(((lane & 7) ^ (r & 7)) << 4));
    if (m + 4 * j >= p.M) continue;
    if (all4 && F32) {
      if (p.accumulate)
        v = make_float4(v.x + __uint_as_float(old[j].x), v.y + __uint_as_float(old[j].y), v.z + __uint_as_float(old[j].z), v.w + __uint_as_float(old[j].w));
      *reinterpret_cast<float4*>(cf + 4 * j * p.ldc) = v;
    } else if (all4) {
      if (p.accumulate) v = make_float4(v.x + bf16_lo(old[j].x), v.y + bf16_hi(old[j].x), v.z + bf16_lo(old[j].y), v.w + bf16_hi(old[j].y));
      const __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
      *reinterpret_cast<uint2*>(ch + 4 * j * p.ldc) = make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
    } else {
      const float f[3] = {v.x, v.y, v.z};
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        if (n + i < p.N) {
          if (F32) {
            float* c = cf + 4 * j * p.ldc + i;
            *c = p.accumulate ? *c + f[i] : f[i];
          } else {
            __nv_bfloat16* c = reinterpret_cast<__nv_bfloat16*>(ch + 4 * j * p.ldc + i);
            *c = __float2bfloat16_rn(p.accumulate ? f[i] + __bfloat162float(*c) : f[i]);
          }
        }
      }
    }
  }
}

// A warp's 32 rows x CW columns of C from accumulator fragments (layout: see tc_ld_16x256b_x8): 128-byte row pieces staged in shared
// memory with the 128-byte swizzle. Written by the bulk-tensor engine as full lines, rows clipped at the edge of C; at the right edge
// (whose padding columns stay untouched) and when adding to the old C read back by rows, four columns per lane, eight lanes per row.
// (Straight from the fragments those accesses are 2 and 4 bytes wide: us, accumulating, from fragments / by rows: 16384 x 1024 x 1024
// BF16 103 / 48, FP32 122 / 51; 4096^3 FP32 172 / 103; 16384 x 200 x 1024 BF16 58 / 19; 256 x 512 x 512 FP32 20.8 / 8.0.)
template <int CW>
__device__ __forceinline__ void b128_store(const Params& p, const CUtensorMap& tmC, uint32_t stage, int lane, int64_t m0, int64_t n0,
                                           const float2 (&acc)[2][2][CW / 8]) {
  const int lr = lane >> 2, lc = lane & 3;
  const bool whole = n0 + CW <= p.N && !p.accumulate && (CW == 64 || p.c_is_f32);  // (32 BF16 columns are half of a bulk store)
  if (p.c_is_f32 || !whole) {
#pragma unroll
    for (int b = 0; b < CW / 32; ++b) {
      const int64_t nb = n0 + 32 * b;
      if (nb >= p.N) break;
      auto stage_rows = [&]() {
        if (lane == 0) bulk_wait_read<0>();  // the previous store from this buffer has read it
        __syncwarp();
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float2 a = acc[r >> 1][r & 1][4 * b + i];
            const uint32_t dst = stage + (uint32_t)(8 * r + lr) * 128u + (uint32_t)(((2 * i + (lc >> 1)) ^ lr) << 4) + (uint32_t)(lc & 1) * 8u;
            asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(dst), "f"(a.x), "f"(a.y) : "memory");
          }
      };
      if (!whole) {
        if (p.c_is_f32)
          b128_store_rows<true>(p, stage, lane, m0, nb, stage_rows);
        else
          b128_store_rows<false>(p, stage, lane, m0, nb, stage_rows);
        continue;
      }
      stage_rows();
      fence_async_smem();
      __syncwarp();
      if (lane == 0) {
        tma_store_2d(&tmC, stage, (int32_t)nb, (int32_t)m0);
        bulk_commit();
      }
    }
  } else if constexpr (CW == 64) {
    if (lane == 0) bulk_wait_read<0>();
    __syncwarp();
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        uint32_t w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float2 a = acc[r >> 1][r & 1][4 * b + i];
          const __nv_bfloat162 hh = __floats2bfloat162_rn(a.x, a.y);
          w[i] = *reinterpret_cast<const uint32_t*>(&hh);
        }
        // lane l gives the address of row l % 8 of 8 x 8 matrix l / 8, which is column group 4 b + l / 8
        const uint32_t dst = stage + (uint32_t)(8 * r + (lane & 7)) * 128u + (uint32_t)(((4 * b + (lane >> 3)) ^ (lane & 7)) << 4);
        asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(dst), "r"(w[0]), "r"(w[1]), "r"(w[2]),
                     "r"(w[3])
                     : "memory");
      }
    fence_async_smem();
    __syncwarp();
    if (lane == 0) {
      tma_store_2d(&tmC, stage, (int32_t)n0, (int32_t)m0);
      bulk_commit();
    }
  }
}

template <int TN>
__global__ void __launch_bounds__(B128<TN>::THREADS, 1)
gemm_nvfp4_block128_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                           const __grid_constant__ CUtensorMap tmC, const __grid_constant__ CUtensorMap tmAh,
                           const __grid_constant__ CUtensorMap tmBh, const Params p) {
  using C = B128<TN>;
  constexpr int STAGES = C::STAGES, SLOTS = C::SC_SLOTS;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t staging_base = smem_base + STAGES * C::STAGE_BYTES;  // 1024-byte aligned
  const uint32_t scale_base = staging_base + C::STAGING_BYTES;
  const uint32_t bar_base = scale_base + SLOTS * C::SC_BYTES;
  auto full_bar = [&](int s) { return bar_base + 8u * s; };
  auto empty_bar = [&](int s) { return bar_base + 8u * (STAGES + s); };
  auto part_full_bar = [&](int b) { return bar_base + 8u * (2 * STAGES + b); };
  auto part_empty_bar = [&](int b) { return bar_base + 8u * (2 * STAGES + C::NBUF + b); };
  auto sc_full_bar = [&](int s) { return bar_base + 8u * (2 * STAGES + 2 * C::NBUF + s); };
  auto sc_empty_bar = [&](int s) { return bar_base + 8u * (2 * STAGES + 2 * C::NBUF + SLOTS + s); };
  const uint32_t drain_bar = bar_base + 8u * (2 * STAGES + 2 * C::NBUF + 2 * SLOTS);
  __shared__ uint32_t tmem_base_slot;
  __shared__ int abort_flag_s;
  volatile int* abort_flag = &abort_flag_s;
  const int warp = uniform_warp_index(), lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    abort_flag_s = 0;
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    for (int b = 0; b < C::NBUF; ++b) {
      mbar_init(part_full_bar(b), 1);
      mbar_init(part_empty_bar(b), C::PROMO_WARPS);
    }
    for (int s = 0; s < SLOTS; ++s) {
      mbar_init(sc_full_bar(s), 2);
      mbar_init(sc_empty_bar(s), C::PROMO_WARPS);
    }
    mbar_init(drain_bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_slot)), "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_slot;
  pdl_prologue();  // everything above touched only shared and tensor memory
  const uint32_t num_tiles = (uint32_t)p.m_tiles * (uint32_t)p.n_tiles;
  const int32_t chunks = p.k_chunks;  // 128-wide k chunks per tile

  if (warp < 4) {
    if (TN == 192) asm volatile("setmaxnreg.dec.sync.aligned.u32 80;");  // 128 x 80 + 384 x 144 = 512 x 128 registers
    if (warp == 0) {
      // ===================================== TMA producer =====================================================
      const uint32_t leader = elect_leader();
      uint32_t it = 0, s = 0, wait_parity = 1;
      bool ok = true;
      for (TileWalk t((uint32_t)blockIdx.x, (uint32_t)gridDim.x, (uint32_t)p.n_tiles); t.index < num_tiles && ok; t.next()) {
        const int32_t mt = (int32_t)t.m, nt = (int32_t)t.n;
        const uint8_t* sfa_src = p.a_sf + (size_t)mt * p.sf_tiles_a * 512;
        const int32_t sfb_tile = (nt * TN) >> 7, sfb_last = (int32_t)((p.N + 127) / 128) - 1;
        const uint8_t* sfb_src = p.b_sf + (size_t)sfb_tile * p.sf_tiles_b * 512;
        // (a tile may start in the middle of a 128-row scale tile; columns beyond N are computed with whatever scales and not stored)
        const uint8_t* sfb_src1 = p.b_sf + (size_t)min(sfb_tile + 1, sfb_last) * p.sf_tiles_b * 512;
        for (int32_t kt = 0; kt < p.k_tiles; ++kt, ++it, s = (s + 1 == (uint32_t)STAGES ? 0u : s + 1), wait_parity ^= (s == 0)) {
          ok = __all_sync(0xFFFFFFFFu, mbar_wait(empty_bar(s), wait_parity, abort_flag, p.dev_status, p.wait_limit));
          if (!ok) break;
          const uint32_t st = smem_base + s * C::STAGE_BYTES;
          mbar_expect_tx(full_bar(s), C::STAGE_BYTES, leader);
          tma_load_2d(st, &tmA, kt * (BK / 2), mt * BM, full_bar(s), leader);
          tma_load_2d(st + A_BYTES, &tmB, kt * (BK / 2), nt * TN, full_bar(s), leader);
          bulk_load(st + A_BYTES + C::B_BYTES, sfa_src + (size_t)kt * 2048, 2048, full_bar(s), leader);
          bulk_load(st + A_BYTES + C::B_BYTES + SFA_BYTES, sfb_src + (size_t)kt * 2048, 2048, full_bar(s), leader);
          if (C::SF_TILES == 2) bulk_load(st + A_BYTES + C::B_BYTES + SFA_BYTES + 2048, sfb_src1 + (size_t)kt * 2048, 2048, full_bar(s), leader);
        }
        // OutControl: the BF16 outlier channels of both operands, 64 per stage, into the same stage buffers
        for (int32_t h = 0; h < p.hp_k_tiles && ok; ++h, ++it, s = (s + 1 == (uint32_t)STAGES ? 0u : s + 1), wait_parity ^= (s == 0)) {
          ok = __all_sync(0xFFFFFFFFu, mbar_wait(empty_bar(s), wait_parity, abort_flag, p.dev_status, p.wait_limit));
          if (!ok) break;
          const uint32_t st = smem_base + s * C::STAGE_BYTES;
          mbar_expect_tx(full_bar(s), A_BYTES + C::B_BYTES, leader);
          tma_load_2d(st, &tmAh, h * 64, mt * BM, full_bar(s), leader);
          tma_load_2d(st + A_BYTES, &tmBh, h * 64, nt * TN, full_bar(s), leader);
        }
      }
      if (!ok) {
        const uint32_t n_back = it < (uint32_t)STAGES ? it : (uint32_t)STAGES;
        for (uint32_t j = 0; j < n_back; ++j) {
          const uint32_t f = it - 1 - j;
          const long long t0 = clock64();
          while (!mbar_try(full_bar(f % STAGES), (f / STAGES) & 1) && clock64() - t0 < p.wait_limit) {
          }
        }
      }
    } else if (warp == 1) {
      // ===================================== MMA issuer =======================================================
      const uint32_t leader = elect_leader();
      const uint32_t idesc = instr_desc<TN>();
      uint32_t it = 0, stage = 0, phase = 0, buf = 0, buf_parity = 1;
      bool ok = true;
      auto take_buffer = [&]() {
        ok = __all_sync(0xFFFFFFFFu, mbar_wait(part_empty_bar(buf), buf_parity, abort_flag, p.dev_status, p.wait_limit));
        tc_fence_after();
      };
      auto next_buffer = [&]() {
        buf = buf + 1 == (uint32_t)C::NBUF ? 0u : buf + 1;
        buf_parity ^= (buf == 0);
      };
      auto take_stage = [&]() {
        ok = __all_sync(0xFFFFFFFFu, mbar_wait(full_bar(stage), phase, abort_flag, p.dev_status, p.wait_limit));
        tc_fence_after();
      };
      auto give_stage = [&]() {
        tc_commit(empty_bar(stage), leader);
        stage = stage + 1 == (uint32_t)STAGES ? 0u : stage + 1;
        phase ^= (stage == 0);
      };
      for (TileWalk t((uint32_t)blockIdx.x, (uint32_t)gridDim.x, (uint32_t)p.n_tiles); t.index < num_tiles && ok; t.next()) {
        // scales of the B rows: a tile that starts 64 rows into its first scale tile finds its own two columns later
        const uint32_t sfb_col = (uint32_t)((((int32_t)t.n * TN) & 127) >> 5);
        for (int32_t kt = 0; kt < p.k_tiles && ok; ++kt, ++it) {
          take_stage();
          if (!ok) break;
          const uint32_t st = smem_base + stage * C::STAGE_BYTES;
          const uint32_t sf_tmem = tmem_base + C::NBUF * TN + (it % C::SF_SETS) * C::SF_COLS;
#pragma unroll
          for (int kk = 0; kk < BK / 64; ++kk) {
            tc_cp_sf(sf_tmem + kk * 4, desc_sf(st + A_BYTES + C::B_BYTES + kk * 512), leader);
            tc_cp_sf(sf_tmem + 16 + kk * 4 * C::SF_TILES, desc_sf(st + A_BYTES + C::B_BYTES + SFA_BYTES + kk * 512), leader);
            if (C::SF_TILES == 2) tc_cp_sf(sf_tmem + 20 + kk * 8, desc_sf(st + A_BYTES + C::B_BYTES + SFA_BYTES + 2048 + kk * 512), leader);
          }
#pragma unroll
          for (int half = 0; half < 2; ++half) {
            if (kt * 2 + half >= chunks) break;  // the padded half of the last k tile holds only zeros
            take_buffer();
            if (!ok) break;
#pragma unroll
            for (int q = 0; q < 2; ++q) {
              const int kk = 2 * half + q;
              tc_mma_nvf4(tmem_base + buf * TN, desc_sw128(st + kk * 32), desc_sw128(st + A_BYTES + kk * 32), idesc, sf_tmem + kk * 4,
                          sf_tmem + 16 + kk * 4 * C::SF_TILES + sfb_col, q, leader);
            }
            tc_commit(part_full_bar(buf), leader);
            next_buffer();
          }
          if (!ok) break;
          give_stage();
        }
        if (p.hp_k_tiles > 0 && ok) {
          // high-precision side product: one more partial, promoted like a 128-k chunk (scale 1)
          take_buffer();
          if (!ok) break;
          const uint32_t idesc_bf16 = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(TN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
          for (int32_t h = 0; h < p.hp_k_tiles; ++h) {
            take_stage();
            if (!ok) break;
            const uint32_t st = smem_base + stage * C::STAGE_BYTES;
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)  // 64 BF16 = one 128-byte swizzle row = four K = 16 steps of 32 bytes
              tc_mma_bf16(tmem_base + buf * TN, desc_sw128(st + kk * 32), desc_sw128(st + A_BYTES + kk * 32), idesc_bf16, (h | kk) != 0, leader);
            give_stage();
          }
          if (!ok) break;
          tc_commit(part_full_bar(buf), leader);
          next_buffer();
        }
      }
      tc_commit(drain_bar, leader);
      {
        const long long t0 = clock64();
        while (!mbar_try(drain_bar, 0) && clock64() - t0 < p.wait_limit) {
        }
      }
    } else {
      // ===================================== global scales (two warps) ========================================
      // Ring slots of four chunks: per chunk SgA, then SgB. Within 32 rows of A, row r sits at (r & 7) * 4 + (r >> 3): the four rows
      // of a thread's fragments (lane / 4 + 0, 8, 16, 24) are neighbours. Within 32 columns of B, column n sits at its bits
      // reordered n4 n2 n1 n3 n0: four of a thread's columns (8 i + 2 (lane % 4) + {0, 1} for an even i and i + 1) are neighbours.
      // A lane reads four chunks of its (at 192 columns five) rows at once, a slot ahead (the rows lie 4 G bytes apart: a load per chunk, or an
      // asynchronous 4-byte copy, is 32 sectors for 128 bytes, and the barriers and reads of the promotion warps queue behind
      // them: 16384 x 8192 x 8192 took 1454 us with such copies).
      constexpr int ROWS = (128 + TN) / 64;  // per lane and warp
      const int64_t G = p.g_per_row;         // global scales per operand row (= padded K / 128)
      const uint32_t r = (uint32_t)lane;
      const uint32_t at_a = ((r & 7u) * 4u + (r >> 3)) * 4u, at_b = ((r & 0x11u) | ((r & 6u) << 1) | ((r & 8u) >> 2)) * 4u;
      const uintptr_t bases = reinterpret_cast<uintptr_t>(p.a_gscale) | reinterpret_cast<uintptr_t>(p.b_gscale);
      const int vec = (G & 3) == 0 && (bases & 15u) == 0 ? 4 : (G & 1) == 0 && (bases & 7u) == 0 ? 2 : 1;
      const int32_t slots_per_tile = (chunks + 3) >> 2;
      uint32_t slot = 0, wait_parity = 1;
      bool ok = true;
      for (TileWalk t((uint32_t)blockIdx.x, (uint32_t)gridDim.x, (uint32_t)p.n_tiles); t.index < num_tiles && ok; t.next()) {
        const int64_t m0 = (int64_t)t.m * BM, n0 = (int64_t)t.n * TN;
        const float* src[ROWS];
#pragma unroll
        for (int i = 0; i < ROWS; ++i) {
          const int q = (warp - 2) * ROWS + i;  // group of 32: four of A, then those of B
          const int64_t row = (q < 4 ? m0 + q * 32 : n0 + (q - 4) * 32) + lane, last = (q < 4 ? p.M : p.N) - 1;
          src[i] = (q < 4 ? p.a_gscale : p.b_gscale) + min(row, last) * G;  // (rows past the end multiply zeros)
        }
        float4 v[ROWS];
        auto load = [&](int32_t c) {
#pragma unroll
          for (int i = 0; i < ROWS; ++i) v[i] = load_scales4(src[i], c, chunks, vec);
        };
        load(0);
        for (int32_t j = 0; j < slots_per_tile; ++j, slot = (slot + 1 == (uint32_t)SLOTS ? 0u : slot + 1), wait_parity ^= (slot == 0)) {
          ok = __all_sync(0xFFFFFFFFu, mbar_wait(sc_empty_bar(slot), wait_parity, abort_flag, p.dev_status, p.wait_limit));
          if (!ok) break;
          const uint32_t dst = scale_base + slot * C::SC_BYTES;
#pragma unroll
          for (int i = 0; i < ROWS; ++i) {
            const int q = (warp - 2) * ROWS + i;
            const uint32_t d = dst + q * 128 + (q < 4 ? at_a : at_b);
            const float f[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
#pragma unroll
            for (int c = 0; c < 4; ++c) asm volatile("st.shared.f32 [%0], %1;" ::"r"(d + c * C::SC_CHUNK), "f"(f[c]) : "memory");
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(sc_full_bar(slot));
          if (j + 1 < slots_per_tile) load(4 * (j + 1));
        }
      }
    }
  } else {
    // ===================================== promotion and epilogue ===============================================
    if (TN == 192) asm volatile("setmaxnreg.inc.sync.aligned.u32 144;");
    constexpr int CW = C::CW, NG = CW / 8;
    const int quad = warp & 3, part = (warp - 4) >> 2;  // 32 rows, CW columns
    const int lr = lane >> 2, lc = lane & 3;
    const uint32_t my_part = tmem_base + ((uint32_t)(quad * 32) << 16) + part * CW;
    const uint32_t my_stage = staging_base + (uint32_t)(warp - 4) * 4096u;
    const uint32_t my_sa = scale_base + (uint32_t)(quad * 32 + lr * 4) * 4u;
    const uint32_t my_sb = scale_base + 512u + (uint32_t)(part * CW + lc * 4) * 4u;
    uint32_t slot = 0, slot_parity = 0, buf = 0, buf_parity = 0;
    bool ok = true;
    float2 acc[2][2][NG];  // [16-row half][8-row half][8-column group]
    // one partial: acc += SgA[row] SgB[column] partial. The scales are read under the first tensor-memory load.
    auto promote = [&](uint32_t sc, bool scaled) {
      ok = __all_sync(0xFFFFFFFFu, mbar_wait(part_full_bar(buf), buf_parity, abort_flag, p.dev_status, p.wait_limit));
      if (!ok) return;
      tc_fence_after();
      float4 sa4 = make_float4(1.0f, 1.0f, 1.0f, 1.0f), sb4[NG / 2];
#pragma unroll
      for (int j = 0; j < NG / 2; ++j) sb4[j] = sa4;
      auto scales = [&]() {
        if (!scaled) return;
        sa4 = lds128(my_sa + sc);
#pragma unroll
        for (int j = 0; j < NG / 2; ++j) sb4[j] = lds128(my_sb + sc + j * 64u);
      };
      auto give_back = [&]() {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(part_empty_bar(buf));
      };
      auto add = [&](int h, const uint32_t(&v)[4 * NG]) {  // 16 rows
        const float2 s0 = h ? make_float2(sa4.z, sa4.z) : make_float2(sa4.x, sa4.x);
        const float2 s1 = h ? make_float2(sa4.w, sa4.w) : make_float2(sa4.y, sa4.y);
#pragma unroll
        for (int i = 0; i < NG; ++i) {
          const float2 sb = (i & 1) ? make_float2(sb4[i >> 1].z, sb4[i >> 1].w) : make_float2(sb4[i >> 1].x, sb4[i >> 1].y);
          const float2 x0 = __fmul2_rn(make_float2(__uint_as_float(v[4 * i]), __uint_as_float(v[4 * i + 1])), s0);
          const float2 x1 = __fmul2_rn(make_float2(__uint_as_float(v[4 * i + 2]), __uint_as_float(v[4 * i + 3])), s1);
          acc[h][0][i] = __ffma2_rn(x0, sb, acc[h][0][i]);
          acc[h][1][i] = __ffma2_rn(x1, sb, acc[h][1][i]);
        }
      };
      const uint32_t src = my_part + buf * TN;
      if constexpr (CW == 32) {  // both halves on their way at once
        uint32_t v0[16], v1[16];
        tc_ld_16x256b_x4(src, v0);
        tc_ld_16x256b_x4(src + (16u << 16), v1);
        scales();
        tc_wait_ld();
        give_back();
        add(0, v0);
        add(1, v1);
      } else {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t v[32];
          tc_ld_16x256b_x8(src + ((uint32_t)(16 * h) << 16), v);
          if (h == 0) scales();
          tc_wait_ld();
          if (h == 1) give_back();
          add(h, v);
        }
      }
      buf = buf + 1 == (uint32_t)C::NBUF ? 0u : buf + 1;
      buf_parity ^= (buf == 0);
    };
    for (TileWalk t((uint32_t)blockIdx.x, (uint32_t)gridDim.x, (uint32_t)p.n_tiles); t.index < num_tiles && ok; t.next()) {
      const int32_t mt = (int32_t)t.m, nt = (int32_t)t.n;
#pragma unroll
      for (int j = 0; j < 4 * NG; ++j) acc[j / (2 * NG)][(j / NG) & 1][j % NG] = make_float2(0.0f, 0.0f);
      for (int32_t kc = 0; kc < chunks; kc += 4) {
        ok = __all_sync(0xFFFFFFFFu, mbar_wait(sc_full_bar(slot), slot_parity, abort_flag, p.dev_status, p.wait_limit));
        if (!ok) break;
        const uint32_t sc = slot * C::SC_BYTES;
#pragma unroll 1
        for (int c = 0; c < 4 && kc + c < chunks; ++c) {
          promote(sc + c * C::SC_CHUNK, true);
          if (!ok) break;
        }
        if (!ok) break;
        __syncwarp();
        if (lane == 0) mbar_arrive(sc_empty_bar(slot));
        slot = slot + 1 == (uint32_t)SLOTS ? 0u : slot + 1;
        slot_parity ^= (slot == 0);
      }
      if (!ok) break;
      if (p.hp_k_tiles > 0) {  // the high-precision partial carries no scale
        promote(0, false);
        if (!ok) break;
      }
      const int64_t m0 = (int64_t)mt * BM + quad * 32, n0 = (int64_t)nt * TN + part * CW;
      if (m0 < p.M && n0 < p.N) b128_store<CW>(p, tmC, my_stage, lane, m0, n0, acc);
    }
    if (lane == 0) bulk_wait_all();  // this lane's bulk stores are complete before the CTA may exit
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
  }
}

// =========================================================================================================
// Two-CTA variant (cta_group::2) for large products: a pair of CTAs on neighbouring SMs computes one 256 x 256 tile.
// Each CTA loads its own 128 rows of A, HALF of the B tile (128 of the 256 rows) and the scales it needs; the pair's
// tensor cores read both halves of B, so every SM pulls 38 KB per k tile instead of 54 KB (128 x 256 single-CTA
// tiles) and five stages fit. The MMAs are issued by the leader CTA (cluster rank 0) only:
//   - both CTAs' bulk-tensor loads complete on the LEADER's "full" barrier (armed for the bytes of both);
//   - tcgen05.commit multicasts the "stage free" / "accumulator ready" arrivals to the same barrier in both CTAs;
//   - both CTAs' epilogue warps arrive on the leader's "accumulator free" barrier (a remote arrive for the peer).
// No load uses cluster multicast. Accumulator: 128 lanes x 256 columns per CTA, drained into registers by eight
// epilogue warps, which hand it back at once and then scale, stage 128-byte row pieces in shared memory (one 4 KB buffer
// per warp, 128-byte swizzle) and let the bulk-tensor engine write them as full lines while the next tile's MMAs run
// (plain 16-byte stores from the registers, a lane per row, cost 16384 x 3072 x 1024 with FP32 output 112 instead of 56 us).
// =========================================================================================================
// Two tile widths. PN = 256: one accumulator of 256 columns per CTA and four sets of scale columns. PN = 192: two
// accumulators of 192 columns (a tile's epilogue runs entirely under the next tile's MMAs) and two sets of scale columns;
// each CTA loads 96 rows of B. A 192-wide tile starts at a multiple of 64 B rows, i.e. possibly in the middle of a 128-row
// scale tile: the two scale tiles it touches are copied whole and the MMA's scale address starts two columns later (one
// tensor-memory column holds the scales of 32 rows).
// DENSE: operands in BF16 without block scales (the simulated FP6 x FP4 products): the same 128 bytes per row and stage are a 64-wide k
// tile, and the tensor memory that the scales leave holds a second accumulator at either width.
template <int PN, bool DENSE = false>
struct Cfg2 {
  static constexpr int STAGES = DENSE ? 6 : 5;
  static constexpr uint32_t B_ROWS = PN / 2;                                   // this CTA's rows of the B tile
  static constexpr uint32_t B_BYTES = B_ROWS * 128;
  static constexpr uint32_t SFA2_BYTES = DENSE ? 0 : SFA_BYTES;
  static constexpr uint32_t SFB_BYTES = DENSE ? 0 : 4096;                      // scales of the two 128-row scale tiles touched
  static constexpr uint32_t STAGE_BYTES = A_BYTES + B_BYTES + SFA2_BYTES + SFB_BYTES;  // 38 KB / 34 KB, DENSE 32 KB / 28 KB
  // staging buffers of 4 KB: one per epilogue warp; with 192-wide tiles (room for it) the four warps that own 128 columns
  // alternate between two, so that a chunk does not wait for the previous chunk's bulk store to have read the buffer
  static constexpr uint32_t STAGING_BYTES = (PN == 256 ? 8 : 12) * 4096;
  static constexpr uint32_t SMEM_BYTES = STAGES * STAGE_BYTES + STAGING_BYTES + 1024 + 256;
  static constexpr int ACC_BUFS = PN == 256 && !DENSE ? 1 : 2;
  static constexpr uint32_t SF_COLS = 16 + 32;
  static constexpr uint32_t SF_SETS = PN == 256 ? 4 : 2;
  static constexpr uint32_t SF_TMEM_COL = ACC_BUFS * PN;                       // 256 / 384; + SF_SETS * 48 <= 512
  static_assert(STAGE_BYTES % 1024 == 0 && SMEM_BYTES <= 227 * 1024, "shared memory budget");
};
constexpr int C2_THREADS = 64 + 256;

__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// Address of the same shared-memory location in the CTA with the given cluster rank.
__device__ __forceinline__ uint32_t map_to_cta(uint32_t saddr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Arrive on a barrier of a CTA of the cluster (possibly this one). Relaxed: what it announces -- this warp's tensor-memory
// loads of the accumulator are complete -- is ordered by tcgen05.wait::ld and the tcgen05 fence before it; with release
// semantics at cluster scope the arrive took about 2500 cycles (it waits for the thread's earlier shared-memory and bulk
// traffic), and that, not the loads, was the cost of handing the accumulator over.
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
// Bulk-tensor load of one CTA of a pair; completes on an mbarrier that may live in the peer CTA.
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* tm, int32_t c0, int32_t c1,
                                                 uint32_t bar_cluster_addr, uint32_t leader) {
  asm volatile(
      "{\n.reg .pred q;\nsetp.ne.b32 q, %5, 0;\n"
      "@q cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];\n}" ::"r"(dst),
      "l"(tm), "r"(c0), "r"(c1), "r"(bar_cluster_addr), "r"(leader)
      : "memory");
}
__device__ __forceinline__ void tc2_commit_both(uint32_t bar, uint32_t leader) {
  asm volatile(
      "{\n.reg .pred q;\n.reg .b16 m;\nsetp.ne.b32 q, %1, 0;\nmov.b16 m, 3;\n"
      "@q tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], m;\n}" ::"r"(bar),
      "r"(leader)
      : "memory");
}
__device__ __forceinline__ void tc2_cp_sf(uint32_t taddr, uint64_t sdesc, uint32_t leader) {
  asm volatile("{\n.reg .pred q;\nsetp.ne.b32 q, %2, 0;\n@q tcgen05.cp.cta_group::2.32x128b.warpx4 [%0], %1;\n}" ::"r"(taddr),
               "l"(sdesc), "r"(leader)
               : "memory");
}
__device__ __forceinline__ void tc2_mma_nvf4(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                             uint32_t sfa_tmem, uint32_t sfb_tmem, uint32_t accumulate, uint32_t leader) {
  asm volatile(
      "{\n.reg .pred p, q;\n"
      "setp.ne.b32 p, %4, 0;\n"
      "setp.ne.b32 q, %7, 0;\n"
      "@q tcgen05.mma.cta_group::2.kind::mxf4nvf4.block_scale.scale_vec::4X [%0], %1, %2, %3, [%5], [%6], p;\n}" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(sfa_tmem), "r"(sfb_tmem), "r"(leader)
      : "memory");
}

__device__ __forceinline__ void tc2_mma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate,
                                             uint32_t leader) {
  asm volatile(
      "{\n.reg .pred p, q;\n"
      "setp.ne.b32 p, %4, 0;\n"
      "setp.ne.b32 q, %5, 0;\n"
      "@q tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(leader)
      : "memory");
}

// One 128-byte-wide piece (W = 32 FP32 or 64 BF16 columns) of a warp's 32 output rows, values final except for the old C:
// accumulate, then either plain stores (a chunk that sticks out past N) or a swizzled copy into the warp's 4 KB staging
// buffer that the bulk-tensor engine writes as full lines. m0 is the first of the 32 rows, m this lane's row.
// pending: how many of this lane's earlier bulk stores may still be reading shared memory when `buf` is written again (0 with
// one staging buffer per warp, 1 when the warp alternates between two).
template <int W>
__device__ __forceinline__ void stage_and_store(const Params& p, const CUtensorMap* tmC, uint32_t buf, int lane, int64_t m, int64_t m0,
                                                int64_t n0, float (&o)[W], int pending = 0) {
  if (p.accumulate && m < p.M) {
    if (n0 + W <= p.N) {
      add_existing<W>(p, m, n0, o);
    } else if (p.c_is_f32) {
#pragma unroll
      for (int j = 0; j < W; ++j)
        if (n0 + j < p.N) o[j] += reinterpret_cast<const float*>(p.C)[m * p.ldc + n0 + j];
    } else {
#pragma unroll
      for (int j = 0; j < W; ++j)
        if (n0 + j < p.N) o[j] += __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(p.C)[m * p.ldc + n0 + j]);
    }
  }
  if (n0 + W > p.N) {  // ragged last chunk of the row
    if (m < p.M) store_ragged<W>(p, m, n0, o);
    return;
  }
  if (lane == 0) {  // the previous store from this buffer has read it
    if (pending)
      bulk_wait_read<1>();
    else
      bulk_wait_read<0>();
  }
  __syncwarp();
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    uint32_t q[4];
    if (W == 32) {
#pragma unroll
      for (int h = 0; h < 4; ++h) q[h] = __float_as_uint(o[4 * j + h]);
    } else {
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        const __nv_bfloat162 hh = __floats2bfloat162_rn(o[(8 * j + 2 * h) % W], o[(8 * j + 2 * h + 1) % W]);
        q[h] = *reinterpret_cast<const uint32_t*>(&hh);
      }
    }
    const uint32_t dst = buf + (uint32_t)lane * 128u + (uint32_t)((j ^ (lane & 7)) << 4);
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "r"(q[0]), "r"(q[1]), "r"(q[2]), "r"(q[3]) : "memory");
  }
  fence_async_smem();
  __syncwarp();
  if (lane == 0) {
    tma_store_2d(tmC, buf, (int32_t)n0, (int32_t)m0);
    bulk_commit();
  }
}

template <int GS, int PN, bool DENSE = false>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(C2_THREADS, 1)
gemm_nvfp4_2cta_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                       const __grid_constant__ CUtensorMap tmSFA, const __grid_constant__ CUtensorMap tmSFB,
                       const __grid_constant__ CUtensorMap tmC, const Params p) {
  using C2 = Cfg2<PN, DENSE>;
  constexpr int STAGES = C2::STAGES;
  constexpr uint32_t C2_STAGE_BYTES = C2::STAGE_BYTES, C2_B_BYTES = C2::B_BYTES, C2_SF_COLS = C2::SF_COLS;
  constexpr int ACC_BUFS = C2::ACC_BUFS;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t staging_base = smem_base + STAGES * C2_STAGE_BYTES;  // eight 4 KB buffers, one per epilogue warp
  const uint32_t bar_base = staging_base + C2::STAGING_BYTES;
  auto full_bar = [&](int s) { return bar_base + 8u * s; };             // used in the leader CTA only
  auto empty_bar = [&](int s) { return bar_base + 8u * (STAGES + s); };  // one per CTA
  auto acc_full_bar = [&](int b) { return bar_base + 8u * (2 * STAGES + b); };       // one pair per CTA
  auto acc_empty_bar = [&](int b) { return bar_base + 8u * (2 * STAGES + 2 + b); };  // leader CTA only (16 arrivals)
  const uint32_t drain_bar = bar_base + 8u * (2 * STAGES + 4);
  __shared__ uint32_t tmem_base_slot;
  __shared__ int abort_flag_s;
  volatile int* abort_flag = &abort_flag_s;
  const int warp = uniform_warp_index(), lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();

  if (threadIdx.x == 0) {
    abort_flag_s = 0;
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(acc_full_bar(b), 1);
      mbar_init(acc_empty_bar(b), 16);
    }
    mbar_init(drain_bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_slot)), "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // the peer's barriers are initialised and its tensor memory allocated
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_slot;
  pdl_prologue();

  const uint32_t num_tiles = (uint32_t)p.m_tiles * (uint32_t)p.n_tiles;  // 256 x PN tiles
  const int64_t pair = blockIdx.x >> 1, num_pairs = gridDim.x >> 1;

  if (warp == 0) {
    // ===================================== TMA producer (both CTAs) ========================================
    const uint32_t leader = elect_leader();
    uint32_t it = 0, s = 0, wait_parity = 1;
    bool ok = true;
    for (TileWalk t((uint32_t)pair, (uint32_t)num_pairs, (uint32_t)p.n_tiles); t.index < num_tiles && ok; t.next()) {
      const int32_t mt = (int32_t)t.m, nt = (int32_t)t.n;
      const int32_t a_row = mt * 256 + (int32_t)rank * 128, b_row = nt * PN + (int32_t)rank * (PN / 2);
      const int32_t sfa_row = ((mt * 2 + (int32_t)rank) * p.sf_tiles_a) * 4;  // in units of 128 bytes
      const int32_t sfb_tile0 = (nt * PN) >> 7;  // first 128-row scale tile the B tile touches (it touches this one and the next)
      const int32_t sfb_row0 = (sfb_tile0 * p.sf_tiles_b) * 4, sfb_row1 = ((sfb_tile0 + 1) * p.sf_tiles_b) * 4;
      for (int32_t kt = 0; kt < p.k_tiles; ++kt, ++it, s = (s + 1 == (uint32_t)STAGES ? 0u : s + 1), wait_parity ^= (s == 0)) {
        ok = __all_sync(0xFFFFFFFFu, mbar_wait(empty_bar(s), wait_parity, abort_flag, p.dev_status, p.wait_limit));
        if (!ok) break;
        const uint32_t st = smem_base + s * C2_STAGE_BYTES;
        const uint32_t full0 = map_to_cta(full_bar(s), 0);
        if (rank == 0) mbar_expect_tx(full_bar(s), 2 * C2_STAGE_BYTES + ((p.starve && it == 0) ? 16u : 0u), leader);
        constexpr int32_t KX = DENSE ? 64 : BK / 2;  // a k tile in elements of the maps: BF16, or bytes of codes
        tma_load_2d_pair(st, &tmA, kt * KX, a_row, full0, leader);
        tma_load_2d_pair(st + A_BYTES, &tmB, kt * KX, b_row, full0, leader);
        if (DENSE) continue;
        tma_load_2d_pair(st + A_BYTES + C2_B_BYTES, &tmSFA, 0, sfa_row + kt * 16, full0, leader);
        tma_load_2d_pair(st + A_BYTES + C2_B_BYTES + SFA_BYTES, &tmSFB, 0, sfb_row0 + kt * 16, full0, leader);
        tma_load_2d_pair(st + A_BYTES + C2_B_BYTES + SFA_BYTES + 2048, &tmSFB, 0, sfb_row1 + kt * 16, full0, leader);
      }
    }
    if (!ok) {
      // a wait ran out: this CTA's copies in flight complete on the leader's barrier, which the peer cannot poll, so give
      // them a fixed time (far more than a copy takes) to land before the CTA may exit
      const long long t0 = clock64();
      while (clock64() - t0 < 400000) {
      }
    }
  } else if (warp == 1) {
    // ===================================== MMA issuer (leader CTA only) ====================================
    if (rank == 0) {
      const uint32_t leader = elect_leader();
      // (DENSE: BF16 x BF16 -> FP32)
      const uint32_t idesc = (DENSE ? 1u << 4 : 0u) | (1u << 7) | (1u << 10) | ((uint32_t)(PN >> 3) << 17) | ((uint32_t)(256 >> 4) << 24);
      // issue loop kept short as in the 128 x 128 kernel: running stage / phase counters, descriptors by addition to the low
      // word, the next stage's barrier tried before this stage's instructions
      uint32_t it = 0, tile_it = 0, stage = 0, phase = 0;
      bool ok = true;
      bool ready = false;
      constexpr uint32_t SW_HI = (uint32_t)((((uint64_t)64 << 32) | ((uint64_t)1 << 46) | ((uint64_t)2 << 61)) >> 32);
      constexpr uint32_t SF_HI = (uint32_t)((((uint64_t)8 << 32) | ((uint64_t)1 << 46)) >> 32);
      const uint32_t a_lo0 = (uint32_t)desc_sw128(smem_base), sfa_lo0 = (uint32_t)desc_sf(smem_base + A_BYTES + C2_B_BYTES);
      for (TileWalk t((uint32_t)pair, (uint32_t)num_pairs, (uint32_t)p.n_tiles); t.index < num_tiles && ok; t.next(), ++tile_it) {
        const uint32_t ab = tile_it % ACC_BUFS;
        ok = __all_sync(0xFFFFFFFFu, mbar_wait(acc_empty_bar(ab), ((tile_it / ACC_BUFS) & 1) ^ 1, abort_flag, p.dev_status, p.wait_limit));
        if (!ok) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + ab * PN;
        // scales of the B rows: the tile may start 64 rows into its first scale tile, i.e. two columns later
        const uint32_t sfb_col = (uint32_t)((((int32_t)t.n * PN) & 127) >> 5);
        for (int32_t kt = 0; kt < p.k_tiles; ++kt, ++it) {
          if (!ready) {
            ok = __all_sync(0xFFFFFFFFu, mbar_wait(full_bar(stage), phase, abort_flag, p.dev_status, p.wait_limit));
            if (!ok) break;
          }
          tc_fence_after();
          const uint32_t st16 = stage * (uint32_t)(C2_STAGE_BYTES >> 4);
          const uint32_t this_empty = empty_bar(stage);
          if (++stage == (uint32_t)STAGES) {
            stage = 0;
            phase ^= 1u;
          }
          const uint32_t next_try = mbar_test(full_bar(stage), phase);
          if constexpr (DENSE) {
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)  // 64 BF16 = four K = 16 steps of 32 bytes
              tc2_mma_bf16(d_tmem, ((uint64_t)SW_HI << 32) | (a_lo0 + st16 + kk * 2), ((uint64_t)SW_HI << 32) | (a_lo0 + st16 + (A_BYTES >> 4) + kk * 2),
                           idesc, (kt | kk) != 0, leader);
          } else {
            const uint32_t sf_tmem = tmem_base + C2::SF_TMEM_COL + (it % C2::SF_SETS) * C2_SF_COLS;
#pragma unroll
            for (int kk = 0; kk < BK / 64; ++kk) {
              tc2_cp_sf(sf_tmem + kk * 4, ((uint64_t)SF_HI << 32) | (sfa_lo0 + st16 + kk * 32), leader);
              tc2_cp_sf(sf_tmem + 16 + kk * 8, ((uint64_t)SF_HI << 32) | (sfa_lo0 + st16 + (SFA_BYTES >> 4) + kk * 32), leader);
              tc2_cp_sf(sf_tmem + 16 + kk * 8 + 4, ((uint64_t)SF_HI << 32) | (sfa_lo0 + st16 + ((SFA_BYTES + 2048) >> 4) + kk * 32), leader);
            }
#pragma unroll
            for (int kk = 0; kk < BK / 64; ++kk)
              tc2_mma_nvf4(d_tmem, ((uint64_t)SW_HI << 32) | (a_lo0 + st16 + kk * 2), ((uint64_t)SW_HI << 32) | (a_lo0 + st16 + (A_BYTES >> 4) + kk * 2),
                           idesc, sf_tmem + kk * 4, sf_tmem + 16 + kk * 8 + sfb_col, (kt | kk) != 0, leader);
          }
          tc2_commit_both(this_empty, leader);
          ready = __all_sync(0xFFFFFFFFu, next_try);
        }
        if (ok) tc2_commit_both(acc_full_bar(ab), leader);
      }
      // nothing issued may still be running when tensor memory is freed; the commit covers both CTAs' work
      asm volatile(
          "{\n.reg .pred q;\nsetp.ne.b32 q, %1, 0;\n"
          "@q tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}" ::"r"(drain_bar),
          "r"(leader)
          : "memory");
      {
        const long long t0 = clock64();
        while (!mbar_try(drain_bar, 0) && clock64() - t0 < p.wait_limit) {
        }
      }
    }
  } else {
    // ===================================== epilogue (both CTAs, eight warps) ================================
    const int quad = warp & 3;
    const int half = (warp - 2) >> 2;
    // columns of the tile this warp owns: [half * 128, half * 128 + 32 * nq): the first four warps 128, the others the rest
    const int nq = half == 0 ? 4 : (PN - 128) / 32;
    // The staging buffers: a warp with two takes them in turn by the bulk stores that it has issued, not by the chunk, as ragged chunks
    // issue none: the buffer that is written next is then never the one of the last store, which may still be reading it.
    const bool two_bufs = PN == 192 && half == 0;
    const uint32_t my_stage = staging_base + (PN == 256 ? (uint32_t)(warp - 2) : (half == 0 ? 2u * (uint32_t)(warp - 2) : 4u + (uint32_t)(warp - 2))) * 4096u;
    uint32_t buf_at = 0;
    uint32_t tile_it = 0;
    bool ok = true;
    float alpha = 1.0f;
    if (GS == kGsTensor) alpha = __fmul_rn(p.a_gscale[0], p.b_gscale[0]);
    for (TileWalk t((uint32_t)pair, (uint32_t)num_pairs, (uint32_t)p.n_tiles); t.index < num_tiles && ok; t.next(), ++tile_it) {
      const int32_t mt = (int32_t)t.m, nt = (int32_t)t.n;
      const uint32_t ab = tile_it % ACC_BUFS;
      const uint32_t acc_empty_leader = map_to_cta(acc_empty_bar(ab), 0);
      if (!(ok = mbar_wait(acc_full_bar(ab), (tile_it / ACC_BUFS) & 1, abort_flag, p.dev_status, p.wait_limit))) break;
      tc_fence_after();
      const int64_t m = (int64_t)mt * 256 + rank * 128 + quad * 32 + lane;
      float sa = 1.0f;
      if (GS == kGsRow && m < p.M) sa = p.a_gscale[m];
      uint32_t v[4][32];
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (q < nq) tc_ld32(tmem_base + ((uint32_t)(quad * 32) << 16) + ab * PN + half * 128 + q * 32, v[q]);
      tc_wait_ld();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(acc_empty_leader);
      // The accumulator is free again (the pair's next tile may start); scale, stage and store from the registers.
      const int64_t m0 = (int64_t)mt * 256 + rank * 128 + quad * 32;
      if (m0 >= p.M) continue;
      if (p.c_is_f32) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int64_t n0 = (int64_t)nt * PN + half * 128 + q * 32;
          if (q >= nq || n0 >= p.N) break;
          float o[32], sgb[32];
          if (GS == kGsRow) load_sgb32(p.b_gscale, n0, p.N, sgb);
#pragma unroll
          for (int j = 0; j < 32; ++j) o[j] = __uint_as_float(v[q][j]) * (GS == kGsRow ? __fmul_rn(sa, sgb[j]) : alpha);
          stage_and_store<32>(p, &tmC, my_stage + buf_at, lane, m, m0, n0, o, two_bufs ? 1 : 0);
          if (two_bufs && n0 + 32 <= p.N) buf_at ^= 4096u;
        }
      } else {
#pragma unroll
        for (int qq = 0; qq < 2; ++qq) {
          const int64_t n0 = (int64_t)nt * PN + half * 128 + qq * 64;
          if (2 * qq >= nq || n0 >= p.N) break;
          float o[64], sgb[32];
          if (GS == kGsRow) load_sgb32(p.b_gscale, n0, p.N, sgb);
#pragma unroll
          for (int j = 0; j < 32; ++j) o[j] = __uint_as_float(v[2 * qq][j]) * (GS == kGsRow ? __fmul_rn(sa, sgb[j]) : alpha);
          if (GS == kGsRow) load_sgb32(p.b_gscale, n0 + 32, p.N, sgb);
#pragma unroll
          for (int j = 0; j < 32; ++j) o[32 + j] = __uint_as_float(v[2 * qq + 1][j]) * (GS == kGsRow ? __fmul_rn(sa, sgb[j]) : alpha);
          stage_and_store<64>(p, &tmC, my_stage + buf_at, lane, m, m0, n0, o, two_bufs ? 1 : 0);
          if (two_bufs && n0 + 64 <= p.N) buf_at ^= 4096u;
        }
      }
    }
    if (lane == 0) bulk_wait_all();  // this lane's bulk stores are complete before the CTA may exit
  }

  // ===================================== teardown ============================================================
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // the peer may still be reading this CTA's shared memory through the pair's MMAs until here
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
  }
}

// =========================================================================================================
// OutControl's high-precision weight-gradient columns (paper Sec. 4.2):  dW[:, A] = dY^T X[:, A], BF16 inputs, FP32
// accumulation, on the tensor cores (tcgen05 kind::f16).  G[c, j] = sum_t dY[t, c] * X_out[t, j]  with
// M = C, N = Kh (a slab of at most 256 columns of the compact outlier matrix), K = tokens. Both operands are stored with the
// contraction index t as the SLOW index, i.e. "MN-major": a bulk-tensor box of 64 columns x 64 tokens lands in
// shared memory as 64 rows of 128 bytes (8 swizzle atoms of 8 tokens), which is the MN-major 128-byte-swizzle
// operand layout (leading byte offset = distance between 64-column boxes, stride byte offset = 1024).
// Only C / 128 output tiles exist, so the token range is split over blockIdx.y; FP32 partial tiles go to a workspace
// that dw_assemble_kernel sums in a fixed order. One tile per CTA: no accumulator double buffering needed.
// =========================================================================================================
constexpr int HPDW_STAGES = 4;
constexpr int HPDW_THREADS = 192;

__global__ void __launch_bounds__(HPDW_THREADS, 1)
hp_dw_mma_kernel(const __grid_constant__ CUtensorMap tmDY, const __grid_constant__ CUtensorMap tmXO, float* __restrict__ partial,
                 int64_t C, int32_t Kh, int64_t ld_partial, int64_t T, int32_t t_per_split, int32_t* dev_status, long long wait_limit) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t b_bytes = (uint32_t)(Kh / 64) * 8192u;
  const uint32_t stage_bytes = A_BYTES + b_bytes;  // A: two boxes of 64 channels x 64 tokens; B: Kh / 64 boxes
  const uint32_t bar_base = smem_base + HPDW_STAGES * stage_bytes;
  auto full_bar = [&](int s) { return bar_base + 8u * s; };
  auto empty_bar = [&](int s) { return bar_base + 8u * (HPDW_STAGES + s); };
  const uint32_t acc_full_bar = bar_base + 8u * (2 * HPDW_STAGES);
  __shared__ uint32_t tmem_base_slot;
  __shared__ int abort_flag_s;
  volatile int* abort_flag = &abort_flag_s;
  const int warp = uniform_warp_index(), lane = threadIdx.x & 31;
  const uint32_t tmem_cols = Kh <= 64 ? 64u : (Kh <= 128 ? 128u : 256u);

  if (threadIdx.x == 0) {
    abort_flag_s = 0;
    for (int s = 0; s < HPDW_STAGES; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    mbar_init(acc_full_bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_slot)), "r"(tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_slot;
  pdl_prologue();

  const int32_t c0 = (int32_t)blockIdx.x * 128;
  const int64_t t_begin = (int64_t)blockIdx.y * t_per_split;
  const int64_t t_end = min(T, t_begin + t_per_split);
  const int32_t k_tiles = (int32_t)((t_end - t_begin + 63) / 64);  // tokens beyond T read as zero

  if (warp == 0) {
    const uint32_t leader = elect_leader();
    for (int32_t kt = 0; kt < k_tiles; ++kt) {
      const int s = kt % HPDW_STAGES;
      if (!__all_sync(0xFFFFFFFFu, mbar_wait(empty_bar(s), ((kt / HPDW_STAGES) & 1) ^ 1, abort_flag, dev_status, wait_limit))) break;
      const uint32_t st = smem_base + s * stage_bytes;
      const int32_t t0 = (int32_t)(t_begin + (int64_t)kt * 64);
      mbar_expect_tx(full_bar(s), stage_bytes, leader);
      tma_load_2d(st, &tmDY, c0, t0, full_bar(s), leader);
      tma_load_2d(st + 8192, &tmDY, c0 + 64, t0, full_bar(s), leader);
      for (int32_t h = 0; h < Kh / 64; ++h) tma_load_2d(st + A_BYTES + h * 8192, &tmXO, h * 64, t0, full_bar(s), leader);
    }
  } else if (warp == 1) {
    const uint32_t leader = elect_leader();
    // BF16 x BF16 -> FP32, M = 128, N = Kh, both operands MN-major
    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) | ((uint32_t)(Kh >> 3) << 17) |
                           ((uint32_t)(128 >> 4) << 24);
    bool ok = true;
    for (int32_t kt = 0; kt < k_tiles && ok; ++kt) {
      const int s = kt % HPDW_STAGES;
      ok = __all_sync(0xFFFFFFFFu, mbar_wait(full_bar(s), (kt / HPDW_STAGES) & 1, abort_flag, dev_status, wait_limit));
      if (!ok) break;
      tc_fence_after();
      const uint32_t st = smem_base + s * stage_bytes;
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {  // 16 tokens = two 8-token swizzle atoms = 2048 bytes per step
        const uint64_t adesc = (uint64_t)(((st + kk * 2048) >> 4) & 0x3FFFu) | ((uint64_t)(8192 >> 4) << 16) |
                               ((uint64_t)(1024 >> 4) << 32) | ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
        const uint64_t bdesc = (uint64_t)(((st + A_BYTES + kk * 2048) >> 4) & 0x3FFFu) | ((uint64_t)(8192 >> 4) << 16) |
                               ((uint64_t)(1024 >> 4) << 32) | ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
        tc_mma_bf16(tmem_base, adesc, bdesc, idesc, (kt | kk) != 0, leader);
      }
      tc_commit(empty_bar(s), leader);
    }
    tc_commit(acc_full_bar, leader);  // also covers the k_tiles == 0 case (arrives at once)
  } else {
    const int quad = warp & 3;
    if (mbar_wait(acc_full_bar, 0, abort_flag, dev_status, wait_limit)) {
      tc_fence_after();
      const int64_t c = (int64_t)c0 + quad * 32 + lane;
      float* dst = partial + ((int64_t)blockIdx.y * C + (c < C ? c : 0)) * ld_partial;
      for (int j0 = 0; j0 < Kh; j0 += 32) {
        uint32_t v[32];
        tc_ld32(tmem_base + ((uint32_t)(quad * 32) << 16) + j0, v);
        tc_wait_ld();
        if (c < C) {
#pragma unroll
          for (int j = 0; j < 32; j += 4)
            *reinterpret_cast<float4*>(dst + j0 + j) = k_tiles > 0 ? make_float4(__uint_as_float(v[j]), __uint_as_float(v[j + 1]),
                                                                                 __uint_as_float(v[j + 2]), __uint_as_float(v[j + 3]))
                                                                   : make_float4(0.f, 0.f, 0.f, 0.f);
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(tmem_cols) : "memory");
  }
}

// ---------------------------------------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn get_encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      return nullptr;
    fn = reinterpret_cast<EncodeTiledFn>(ptr);
  }
  return fn;
}

// Codes of an operand [R, Kp/2 bytes] as a 2-D byte tensor; box = 128 bytes x box_rows; out-of-range reads give 0.
bool make_codes_map(CUtensorMap* tm, const uint8_t* codes, int64_t R, int64_t Kp, uint32_t box_rows) {
  EncodeTiledFn fn = get_encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)(Kp / 2), (cuuint64_t)R};
  const cuuint64_t strides[1] = {(cuuint64_t)(Kp / 2)};
  const cuuint32_t box[2] = {128, box_rows};
  const cuuint32_t estr[2] = {1, 1};
  return fn(tm, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<uint8_t*>(codes), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// C [M, N] (BF16 or FP32, leading dimension ldc) as a 2-D tensor; box = 128 bytes of a row x 32 rows, 128-byte swizzle.
bool make_c_map(CUtensorMap* tm, void* Cp, int64_t M, int64_t N, int64_t ldc, bool is_f32) {
  EncodeTiledFn fn = get_encode_fn();
  if (!fn) return false;
  const cuuint64_t esz = is_f32 ? 4 : 2;
  const cuuint64_t dims[2] = {(cuuint64_t)N, (cuuint64_t)M};
  const cuuint64_t strides[1] = {(cuuint64_t)ldc * esz};
  const cuuint32_t box[2] = {(cuuint32_t)(128 / esz), 32};
  const cuuint32_t estr[2] = {1, 1};
  return fn(tm, is_f32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, Cp, dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// A compact BF16 side matrix [R, Kh] (Kh a multiple of 64) as a 2-D tensor; box = 64 columns (128 bytes) x box_rows rows.
bool make_hp_map(CUtensorMap* tm, const void* base, int64_t R, int64_t Kh, uint32_t box_rows = 128) {
  EncodeTiledFn fn = get_encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)Kh, (cuuint64_t)R};
  const cuuint64_t strides[1] = {(cuuint64_t)Kh * 2};
  const cuuint32_t box[2] = {64, box_rows};
  const cuuint32_t estr[2] = {1, 1};
  return fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

inline int sm_count() { return device_sm_count(); }
inline long long wait_limit_of(const GemmArgs& a) { return a.wait_limit > 0 ? a.wait_limit : DEFAULT_WAIT_LIMIT_CYCLES; }

template <int GS>
cudaError_t launch_tile128(const GemmArgs& a, cudaStream_t st) {
  using C = Cfg;
  const int64_t Kp = (a.K + 127) & ~(int64_t)127;
  CUtensorMap tmA, tmB, tmC;
  if (!make_codes_map(&tmA, a.a_codes, a.M, Kp, BM) || !make_codes_map(&tmB, a.b_codes, a.N, Kp, BN))
    return cudaErrorInvalidValue;
  if (!make_c_map(&tmC, a.C, a.M, a.N, a.ldc, a.c_is_f32 != 0)) return cudaErrorInvalidValue;
  CUtensorMap tmAh = tmA, tmBh = tmB;  // placeholders unless the high-precision side product is requested
  Params p{};
  p.starve = a.starve_first_stage;
  p.wait_limit = wait_limit_of(a);
  if (a.hp_Kh > 0) {
    if (!make_hp_map(&tmAh, a.hp_a, a.M, a.hp_Kh) || !make_hp_map(&tmBh, a.hp_b, a.N, a.hp_Kh)) return cudaErrorInvalidValue;
    p.hp_k_tiles = (int32_t)(a.hp_Kh / 64);
  }
  p.a_sf = a.a_sf;
  p.b_sf = a.b_sf;
  p.a_gscale = a.a_gscale;
  p.b_gscale = a.b_gscale;
  p.C = a.C;
  p.ldc = a.ldc;
  p.M = a.M;
  p.N = a.N;
  p.k_tiles = (int32_t)((Kp + BK - 1) / BK);
  p.k_chunks = (int32_t)(Kp / 128);
  p.g_per_row = Kp / 128;
  const int64_t kb_padded = ((Kp >> 4) + 15) & ~(int64_t)15;
  p.sf_tiles_a = p.sf_tiles_b = (int32_t)(kb_padded >> 2);
  p.m_tiles = (int32_t)((a.M + BM - 1) / BM);
  p.n_tiles = (int32_t)((a.N + BN - 1) / BN);
  p.c_is_f32 = a.c_is_f32;
  p.accumulate = a.accumulate;
  p.dev_status = a.dev_status;
  cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(gemm_nvfp4_kernel<GS>), C::SMEM_BYTES);
  if (e != cudaSuccess) return e;
  const int64_t tiles = (int64_t)p.m_tiles * p.n_tiles;
  const unsigned grid = (unsigned)std::min<int64_t>(tiles, sm_count());
  launch_kernel(gemm_nvfp4_kernel<GS>, dim3(grid), dim3(C::THREADS), C::SMEM_BYTES, st, tmA, tmB, tmC, tmAh, tmBh, p);
  return cudaGetLastError();
}

// Scale bytes of an operand as a 2-D byte tensor of 128-byte rows; box = 16 rows = the 2 KB of one (row tile, k tile).
bool make_sf_map(CUtensorMap* tm, const uint8_t* sf, int64_t total_bytes) {
  EncodeTiledFn fn = get_encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[2] = {128, (cuuint64_t)(total_bytes / 128)};
  const cuuint64_t strides[1] = {128};
  const cuuint32_t box[2] = {128, 16};
  const cuuint32_t estr[2] = {1, 1};
  return fn(tm, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<uint8_t*>(sf), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int GS, int PN>
cudaError_t launch_2cta(const GemmArgs& a, cudaStream_t st) {
  using C2 = Cfg2<PN>;
  const int64_t Kp = (a.K + 127) & ~(int64_t)127;
  const int64_t kb_padded = ((Kp >> 4) + 15) & ~(int64_t)15;
  const int64_t sfa_bytes = ((a.M + 127) / 128) * 128 * kb_padded, sfb_bytes = ((a.N + 127) / 128) * 128 * kb_padded;
  CUtensorMap tmA, tmB, tmSFA, tmSFB, tmC;
  if (!make_codes_map(&tmA, a.a_codes, a.M, Kp, 128) || !make_codes_map(&tmB, a.b_codes, a.N, Kp, PN / 2) ||
      !make_sf_map(&tmSFA, a.a_sf, sfa_bytes) || !make_sf_map(&tmSFB, a.b_sf, sfb_bytes) ||
      !make_c_map(&tmC, a.C, a.M, a.N, a.ldc, a.c_is_f32 != 0))
    return cudaErrorInvalidValue;
  Params p{};
  p.a_sf = a.a_sf;
  p.b_sf = a.b_sf;
  p.a_gscale = a.a_gscale;
  p.b_gscale = a.b_gscale;
  p.C = a.C;
  p.ldc = a.ldc;
  p.M = a.M;
  p.N = a.N;
  p.k_tiles = (int32_t)((Kp + BK - 1) / BK);
  p.sf_tiles_a = p.sf_tiles_b = (int32_t)(kb_padded >> 2);
  p.m_tiles = (int32_t)((a.M + 255) / 256);
  p.n_tiles = (int32_t)((a.N + PN - 1) / PN);
  p.c_is_f32 = a.c_is_f32;
  p.accumulate = a.accumulate;
  p.dev_status = a.dev_status;
  p.starve = a.starve_first_stage;
  p.wait_limit = wait_limit_of(a);
  cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(gemm_nvfp4_2cta_kernel<GS, PN>), C2::SMEM_BYTES);
  if (e != cudaSuccess) return e;
  const int64_t tiles = (int64_t)p.m_tiles * p.n_tiles;
  const unsigned pairs = (unsigned)std::min<int64_t>(tiles, sm_count() / 2);
  launch_kernel(gemm_nvfp4_2cta_kernel<GS, PN>, dim3(2 * pairs), dim3(C2_THREADS), C2::SMEM_BYTES, st, tmA, tmB, tmSFA, tmSFB, tmC, p);
  return cudaGetLastError();
}

template <int TN>
cudaError_t launch_block128_tn(const GemmArgs& a, cudaStream_t st) {
  const int64_t Kp = (a.K + 127) & ~(int64_t)127;
  if (Kp > B128_MAX_K) return cudaErrorInvalidValue;
  CUtensorMap tmA, tmB, tmC;
  if (!make_codes_map(&tmA, a.a_codes, a.M, Kp, BM) || !make_codes_map(&tmB, a.b_codes, a.N, Kp, TN)) return cudaErrorInvalidValue;
  Params p{};
  CUtensorMap tmAh = tmA, tmBh = tmB;  // placeholders unless the high-precision side product is requested
  if (a.hp_Kh > 0) {
    if (!make_hp_map(&tmAh, a.hp_a, a.M, a.hp_Kh) || !make_hp_map(&tmBh, a.hp_b, a.N, a.hp_Kh, TN)) return cudaErrorInvalidValue;
    p.hp_k_tiles = (int32_t)(a.hp_Kh / 64);
  }
  if (!make_c_map(&tmC, a.C, a.M, a.N, a.ldc, a.c_is_f32 != 0)) return cudaErrorInvalidValue;
  p.a_sf = a.a_sf;
  p.b_sf = a.b_sf;
  p.a_gscale = a.a_gscale;
  p.b_gscale = a.b_gscale;
  p.C = a.C;
  p.ldc = a.ldc;
  p.M = a.M;
  p.N = a.N;
  p.k_tiles = (int32_t)((Kp + BK - 1) / BK);
  p.k_chunks = (int32_t)(Kp / 128);
  p.g_per_row = Kp / 128;
  const int64_t kb_padded = ((Kp >> 4) + 15) & ~(int64_t)15;
  p.sf_tiles_a = p.sf_tiles_b = (int32_t)(kb_padded >> 2);
  p.m_tiles = (int32_t)((a.M + BM - 1) / BM);
  p.n_tiles = (int32_t)((a.N + TN - 1) / TN);
  p.c_is_f32 = a.c_is_f32;
  p.accumulate = a.accumulate;
  p.dev_status = a.dev_status;
  p.wait_limit = wait_limit_of(a);
  cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(gemm_nvfp4_block128_kernel<TN>), B128<TN>::SMEM_BYTES);
  if (e != cudaSuccess) return e;
  const int64_t tiles = (int64_t)p.m_tiles * p.n_tiles;
  const unsigned grid = (unsigned)std::min<int64_t>(tiles, sm_count());
  launch_kernel(gemm_nvfp4_block128_kernel<TN>, dim3(grid), dim3(B128<TN>::THREADS), B128<TN>::SMEM_BYTES, st, tmA, tmB, tmC, tmAh, tmBh, p);
  return cudaGetLastError();
}

// Tile width by a cost model: rounds of the tiles over the SMs x time of a tile, which is a constant (its store, mostly) and so much per
// 128-wide chunk of K. Wide tiles cost the least per column; narrow ones leave fewer SMs idle where a product has few tiles (a weight
// gradient: few tiles, K = tokens). us, 192 / 128 / 64 columns: 1024 x 1024 x 8192 31.0 / 24.0 / 16.5 (27.4 with the 128-column tiles of
// one promotion warp per scheduler), 512 x 512 x 4096 17.3 / 13.4 / 9.8 (15.1), 4096 x 1024 x 3072 25.6 / 20.0 / 26.4 (22.7),
// 16384 x 1024 x 2816 68.5 / 62.7 / 89.6, 2816 x 1024 x 8192 31.4 / 45.0 / 43.2, 8192 x 3072 x 1024 31.9 / 35.8 / 60.1 (FP32 40.0 / 43.9 /
// 45.9), 4096^3 85.0 / 90.8 / 124.
int block128_tile_cols(int64_t M, int64_t N, int64_t K, bool c_is_f32) {
  const double chunks = (double)((K + 127) / 128);
  auto cost = [&](int tn, double fixed, double per_chunk) {
    const int64_t tiles = ((M + BM - 1) / BM) * ((N + tn - 1) / tn), sms = sm_count();
    return (double)((tiles + sms - 1) / sms) * (fixed + per_chunk * chunks);
  };
  const double c192 = cost(192, c_is_f32 ? 1.9 : 0.8, 0.415), c128 = cost(128, c_is_f32 ? 1.2 : 0.48, 0.32), c64 = cost(64, c_is_f32 ? 0.5 : 1.1, 0.195);
  return c192 <= c128 && c192 <= c64 ? 192 : c128 <= c64 ? 128 : 64;
}

cudaError_t launch_block128(const GemmArgs& a, cudaStream_t st) {
  const int tn = block128_tile_cols(a.M, a.N, a.K, a.c_is_f32 != 0);
  return tn == 192 ? launch_block128_tn<192>(a, st) : tn == 128 ? launch_block128_tn<128>(a, st) : launch_block128_tn<64>(a, st);
}

// BF16 matrix [T, W] (leading dimension ld elements) as a 2-D tensor; box = 64 columns x 64 rows, 128-byte swizzle.
bool make_tokens_map(CUtensorMap* tm, const void* base, int64_t T, int64_t W, int64_t ld) {
  EncodeTiledFn fn = get_encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)W, (cuuint64_t)T};
  const cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  const cuuint32_t box[2] = {64, 64};
  const cuuint32_t estr[2] = {1, 1};
  return fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

// partial[(split * C + c) * Kh + j] = sum over the split's tokens of dY[t, c] * X_out[t, j]. Kh is any multiple of 64:
// the outlier channels are taken in slabs of at most 256 (the widest MMA), one launch per slab.
cudaError_t launch_hp_dw_mma(const uint16_t* dY, int64_t lddy, const uint16_t* X_out, int64_t Kh, int64_t T, int64_t C,
                             float* partial, int n_split, int64_t t_per_split, int32_t* dev_status, cudaStream_t st) {
  if (Kh <= 0 || Kh % 64 != 0) return cudaErrorInvalidValue;
  CUtensorMap tmDY, tmXO;
  if (!make_tokens_map(&tmDY, dY, T, C, lddy)) return cudaErrorInvalidValue;
  for (int64_t j0 = 0; j0 < Kh; j0 += 256) {
    const int64_t w = std::min<int64_t>(256, Kh - j0);
    if (!make_tokens_map(&tmXO, X_out + j0, T, w, Kh)) return cudaErrorInvalidValue;
    const uint32_t stage_bytes = A_BYTES + (uint32_t)(w / 64) * 8192u;
    const size_t smem = (size_t)HPDW_STAGES * stage_bytes + 1024 + 256;
    cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(hp_dw_mma_kernel), smem);
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)((C + 127) / 128), (unsigned)n_split);
    launch_kernel(hp_dw_mma_kernel, dim3(grid), dim3(HPDW_THREADS), smem, st, tmDY, tmXO, partial + j0, C, (int32_t)w, Kh, T,
                  (int32_t)t_per_split, dev_status, DEFAULT_WAIT_LIMIT_CYCLES);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// Dense BF16 product (the simulated FP6 x FP4 layer): C = (SgA SgB) * A B^T with A [M, ld], B [N, ld] BF16 row-major, ld a
// multiple of 64 and the same for both. On CTA pairs (PN > 0: the pair kernel's DENSE form, 256 x PN tiles), or on the 128 x 128 kernel
// with no FP4 k tiles at all: only its BF16 side-product path runs (64-wide k tiles, FP32 accumulation in the side accumulator)
// and the epilogue scales that accumulator.
template <int PN>
cudaError_t launch_dense(const void* A, const void* B, int64_t M, int64_t N, int64_t ld, const float* a_gscale, const float* b_gscale, void* Cp,
                         int c_is_f32, int64_t ldc, int32_t* dev_status, cudaStream_t st) {
  constexpr int TM = PN ? 256 : BM, TN = PN ? PN : BN;
  CUtensorMap tmAh, tmBh, tmC;
  if (!make_hp_map(&tmAh, A, M, ld) || !make_hp_map(&tmBh, B, N, ld, PN ? PN / 2 : BN) || !make_c_map(&tmC, Cp, M, N, ldc, c_is_f32 != 0))
    return cudaErrorInvalidValue;
  Params p{};
  p.wait_limit = DEFAULT_WAIT_LIMIT_CYCLES;
  p.a_gscale = a_gscale;
  p.b_gscale = b_gscale;
  p.C = Cp;
  p.ldc = ldc;
  p.M = M;
  p.N = N;
  p.m_tiles = (int32_t)((M + TM - 1) / TM);
  p.n_tiles = (int32_t)((N + TN - 1) / TN);
  p.c_is_f32 = c_is_f32;
  p.dev_status = dev_status;
  const int64_t tiles = (int64_t)p.m_tiles * p.n_tiles;
  cudaError_t e;
  if constexpr (PN > 0) {
    p.k_tiles = (int32_t)(ld / 64);
    const auto kernel = gemm_nvfp4_2cta_kernel<kGsTensor, PN, true>;
    constexpr uint32_t smem = Cfg2<PN, true>::SMEM_BYTES;
    if ((e = ensure_dynamic_smem(reinterpret_cast<const void*>(kernel), smem)) != cudaSuccess) return e;
    const unsigned pairs = (unsigned)std::min<int64_t>(tiles, sm_count() / 2);
    launch_kernel(kernel, dim3(2 * pairs), dim3(C2_THREADS), smem, st, tmAh, tmBh, tmAh, tmBh, tmC, p);
  } else {
    p.hp_k_tiles = (int32_t)(ld / 64);
    if ((e = ensure_dynamic_smem(reinterpret_cast<const void*>(gemm_nvfp4_kernel<kGsTensor>), Cfg::SMEM_BYTES)) != cudaSuccess) return e;
    const unsigned grid = (unsigned)std::min<int64_t>(tiles, sm_count());
    launch_kernel(gemm_nvfp4_kernel<kGsTensor>, dim3(grid), dim3(Cfg::THREADS), Cfg::SMEM_BYTES, st, tmAh, tmBh, tmC, tmAh, tmBh, p);
  }
  return cudaGetLastError();
}

// Variant by a cost model, as launch_gemm: rounds of the tiles x (fixed + per 64-wide k tile). The pairs win where the operands' way from
// L2 to the SMs bounds the product (32 KB per k tile and SM for 256 x 256, as the 128 x 128 kernel takes for a quarter of that), and their
// epilogue runs under the next tile; the small tiles where there are few. us, 128 x 128 / 256 x 256 / 256 x 192: 4096 x 3072 x 1024
// 26.8 / 20.6 / 21.6, 4096 x 1024 x 3072 25.1 / 19.7 / 26.0, 3072 x 1024 x 4096 (FP32) 32.5 / 25.4 / 21.5, 2048^3 17.4 / 14.7 / 18.7,
// 8192^3 1260 / 862 / 899, 1000 x 1416 x 1000 (FP32) 6.8 / 9.6 / 8.1, 2048 x 512 x 4000 (FP32) 17.7 / 23.2 / 18.5, 64 x 2048 x 2048 8.1 /
// 12.5 / 9.9.
cudaError_t launch_dense_gemm(const void* A, const void* B, int64_t M, int64_t N, int64_t ld, const float* a_gscale,
                              const float* b_gscale, void* Cp, int c_is_f32, int64_t ldc, int32_t* dev_status, cudaStream_t st) {
  if (M == 0 || N == 0) return cudaSuccess;
  auto cost = [&](int64_t tm, int64_t tn, int64_t units, double fixed, double per_k_tile) {
    const int64_t tiles = ((M + tm - 1) / tm) * ((N + tn - 1) / tn);
    return (double)((tiles + units - 1) / units) * (fixed + per_k_tile * (double)(ld / 64));
  };
  const int64_t sms = sm_count();
  const double c128 = cost(128, 128, sms, 0.6, 0.23), c256 = cost(256, 256, sms / 2, 1.2, 0.345), c192 = cost(256, 192, sms / 2, 0.9, 0.28);
  const auto launch = c128 <= c256 && c128 <= c192 ? launch_dense<0> : c256 <= c192 ? launch_dense<256> : launch_dense<192>;
  return launch(A, B, M, N, ld, a_gscale, b_gscale, Cp, c_is_f32, ldc, dev_status, st);
}

size_t gemm_workspace_bytes(int64_t, int64_t, int64_t) { return 0; }
int64_t gemm_block128_max_k() { return B128_MAX_K; }

// Variant choice, by a cost model: rounds of the variant's tiles over the SMs (or SM pairs) x time of a tile, which is a constant and
// so much per 256-wide k tile, or at short K what writing the tile takes. All kernels are bound by what the L2 delivers to the SMs and by
// their epilogue: the 128 x 128 kernel pulls 36 KB per k tile and SM, a pair on a 256 x 256 tile 38 KB per SM for twice the math, but
// it fills the last round worse, holds one accumulator and, with ROW scales, has an epilogue of two more multiplies per element
// in registers that spill. The constants are fits to measured times (warm L2, BF16 output unless marked), us, 128 x 128 / 256 x 256 /
// 256 x 192. TENSOR: 16384 x 3072 x 1024 35.0 / 29.8 / 32.1; 16384 x 1024 x 3072 26.9 / 22.8 / 26.1; 16384 x 1024 x 1024 13.0 /
// 12.8 / 14.4; 8192 x 3072 x 1024 18.6 / 17.0 / 16.7; 8192 x 2816 x 1024 17.0 / 14.8 / 16.4; 8192 x 1024 x 3072 15.9 / 13.5 / 14.9;
// 4096^3 32.0 / 27.1 / 27.3; 3072 x 1024 x 16384 (FP32) 29.7 / 26.4 / 21.1; 3072 x 1024 x 8192 (FP32) 18.0 / 16.5 / 13.7;
// 1024 x 1024 x 16384 (FP32) 16.5 / 24.5 / 19.8. ROW: 16384 x 3072 x 1024 49.5 / 53.7 / 58.7; 16384 x 1024 x 3072 37.0 / 32.9 /
// 38.5; 8192 x 1024 x 3072 18.6 / 16.4 / 18.4; 3072 x 1024 x 16384 (FP32) 44.2 / 40.8 / 31.7; 4096^3 33.9 / 29.8 / 29.8. Short K:
// 13736 x 2648 x 648 27.4 / 24.6 / 28.9, 8386 x 4680 x 544 (FP32) 37.3 / 33.0 / 35.4, 7084 x 4768 x 760 25.4 / 23.3 / 24.9; ROW 6083 x
// 6232 x 1320 (FP32) 49.7 / 43.2 / 46.2, 4768 x 2016 x 2616 (FP32) 23.6 / 21.9 / 19.8. Adding to the old C costs the pairs' epilogue more
// (a lane per row reads it): 16384 x 1024 x 1024 (FP32) 29.2 / 32.3 / 41.3, 4989 x 6232 x 1000 (FP32) 78.7 / 87.8 / 92.1, ROW 3825 x 5496 x
// 1216 37.8 / 44.4 / 46.2. Over 125 shapes of every kind the choice is 1.3 % off the fastest in the mean; single shapes, mostly those
// whose rows of C do not start on 128-byte lines, are up to a fifth off.
// A 256-row tile of an operand spans two 128-row scale tiles, and rows are padded to 128 in the scale layout, so any M, N
// work. The fused high-precision side product and the outer-block scales live in the single-CTA kernels only.
cudaError_t launch_gemm(const GemmArgs& a, cudaStream_t st) {
  if (a.M == 0 || a.N == 0) return cudaSuccess;
  if (a.gs_mode == kGsBlock128) return a.variant >= 2 ? cudaErrorInvalidValue : launch_block128(a, st);
  const int64_t sms = sm_count(), n_pairs = sms / 2, rows256 = (a.M + 255) / 256;
  const double k_tiles = (double)((a.K + BK - 1) / BK);
  const bool row_scales = a.gs_mode == kGsRow;
  auto rounds = [](int64_t tiles, int64_t units) { return (double)((tiles + units - 1) / units); };
  // us: a tile = max(write, fixed + per_k_tile * k tiles), with TENSOR and with ROW scales; add: what adding to C makes of a write
  auto cost = [&](double n_rounds, double per_k_tile, double fixed, double fixed_row, double write, double write_row, double add) {
    const double w = (row_scales ? write_row : write) * (a.c_is_f32 ? 1.3 : 1.0) * (a.accumulate ? add : 1.0);
    return n_rounds * std::max(w, (row_scales ? fixed_row : fixed) + per_k_tile * k_tiles);
  };
  const double cost128 = cost(rounds(((a.M + 127) / 128) * ((a.N + 127) / 128), sms), 0.2275, 0.57, 1.45, 1.40, 2.15, 1.2);
  const double cost256 = cost(rounds(rows256 * ((a.N + 255) / 256), n_pairs), 0.300, 1.16, 2.60, 2.35, 4.90, 1.4);
  const double cost192 = cost(rounds(rows256 * ((a.N + 191) / 192), n_pairs), 0.250, 0.80, 2.30, 2.15, 3.80, 1.4);
  bool pairs = cost256 <= cost192 && cost256 <= cost128, pairs192 = cost192 < cost256 && cost192 < cost128;
  if (a.variant == 1) pairs = pairs192 = false;
  if (a.variant == 2) { pairs = true; pairs192 = false; }
  if (a.variant == 3) { pairs192 = true; pairs = false; }
  if (a.hp_Kh > 0) {
    if (a.variant == 2 || a.variant == 3) return cudaErrorInvalidValue;
    pairs = pairs192 = false;
  }
  if (pairs192) return a.gs_mode == kGsTensor ? launch_2cta<kGsTensor, 192>(a, st) : launch_2cta<kGsRow, 192>(a, st);
  if (pairs) return a.gs_mode == kGsTensor ? launch_2cta<kGsTensor, 256>(a, st) : launch_2cta<kGsRow, 256>(a, st);
  return a.gs_mode == kGsTensor ? launch_tile128<kGsTensor>(a, st) : launch_tile128<kGsRow>(a, st);
}

}  // namespace nvfp4
