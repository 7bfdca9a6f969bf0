// The weight gradient of the straight-through backward on the bf16 tensor cores (sm_100a):
//
//   y[m][n] = sum_k a[k][m] * a_scale[k] * code[n][k]      a = dy, m an output channel, k a row of the batch
//
// An 8-bit code is exact in bf16, so only the gradient needs more than one bf16 term: every scaled
// value is split into hi (its upper sixteen bits) and lo = value - hi rounded to bf16, sixteen significant
// bits together against the eleven of the tf32 operand format, and both terms are summed into the same
// binary32 accumulators.  Two bf16 products of a K-block cost the tensor core what one tf32 product costs,
// and the codes take two bytes instead of four.
//
// a is read in place and transposed on the way, which is what the tf32 form has to write to memory and
// read back first (48 + 11 us of a 181 us backward at 12 800 x 2048 x 512).  TMA brings four boxes of
// 32 k x 32 m floats into a ring stage; eight converter warps, in two groups that alternate over
// K-blocks, take one 4 KB box each: a lane reads the 32 k of its column m, scales, splits, and the warp
// writes the box's 32 rows of the K-major operand over it, [32 hi | 32 lo] bf16, one 128-byte swizzle row
// each: four K = 16 MMAs per block, of which the first and third use the codes of k 0 .. 15, the others
// those of k 16 .. 31.  The column sums of a (the bias gradient) fall out.
//
// CTA pairs: two CTAs share a 256 x 256 tile; each loads and converts its 128 rows and loads half of the
// codes into its own shared memory on its own barriers, the leader waits for both CTAs' converters and
// issues the pair's MMAs.  What bounds it: at the bf16 rate that cuBLAS reaches a K-block would take 0.38 us of
// the pair; it takes 0.39 to 0.47.  A CTA's shared memory moves 88 KB a K-block (MMA operands 32, TMA 24, conversion
// 32): its pipe and the tensor pipe are each active for half of the time (43 and 42 % with 64 of 74 pairs at work).  More ring stages (7, 8), more converter warps (12, 16) and
// prefetches into L2 were built and change nothing.
#pragma once

#include "qgemm_sm100.cuh"

namespace aqt {

struct DwCfg {
  static constexpr int BN = 256, STAGES = 6, EW = 4, CW = 8;
  static constexpr int kGroups = CW / 4;
  static constexpr int kThreads = 32 * (2 + EW + CW);
  static constexpr int kABytes = kBM * 128;      // 32 floats (then 64 bf16) per row
  static constexpr int kBBytes = (BN / 2) * 64;  // 32 bf16 codes per row of this CTA's half
  static constexpr int kStageBytes = kABytes + kBBytes;
  static constexpr int kStageBufs = 2;  // staging buffers per epilogue warp
  static constexpr int kEpiBytes = EW * kStageBufs * kStageBufBytes;
  static constexpr int kConvScaleBytes = CW * 32 * 4;
  static constexpr int kSmemBytes = STAGES * kStageBytes + kEpiBytes + kConvScaleBytes + 1024;
  static_assert(kSmemBytes + 512 <= 232448, "must fit the 227 KB a CTA can opt into");
};

struct DwParams {
  const float* a_scale;  // scale of contraction index k at a_scale[k * a_scale_step]
  float* colsum;         // [batches * DwCfg::kGroups][M] sums of a over the K-blocks of a batch that one group converted, or null
  int a_scale_step;
  int M, N, K;           // K: the contraction, in all
  // The contraction cut into batches: tile rows tm of batch b = tm / batch_tiles_m cover k in
  // [b * batch_k, (b + 1) * batch_k) and write the b-th of the stacked outputs.
  int batch_tiles_m, batch_k;
  int tiles_m, tiles_n, k_blocks;
  int y_rows;            // of the (stacked) output
  // The launch before this one (the other product of the backward) lets this one's CTAs follow as soon as SMs fall free
  // (GemmParams::early_trigger): nothing here depends on it, and one pair waits for it before it ends, which keeps the
  // stream's order for whatever comes next.
  int beside_previous;
};

__device__ __forceinline__ void tc_mma_bf16_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// D binary32, A and B bf16, both K-major.
__host__ __device__ constexpr uint32_t idesc_bf16(int bn, int m) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(bn >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}
// K-major operand tile whose rows are 64 bytes, stored with the 64-byte swizzle; 8-row groups are 512 bytes apart.
__device__ __forceinline__ uint64_t smem_desc_k_major_sw64(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(512 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)4 << 61;
  return d;
}

// Two values -> one word of their upper halves, one word of the rounded remainders.
__device__ __forceinline__ void split_bf16x2(float f0, float f1, uint32_t& hi, uint32_t& lo) {
  const uint32_t u0 = __float_as_uint(f0), u1 = __float_as_uint(f1);
  hi = __byte_perm(u0, u1, 0x7632);
  const float l0 = __fsub_rn(f0, __uint_as_float(u0 & 0xFFFF0000u)), l1 = __fsub_rn(f1, __uint_as_float(u1 & 0xFFFF0000u));
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(lo) : "f"(l1), "f"(l0));
}
// sum += the 32 values, added in a tree; what the running sum rounds away is kept in lost.  (One value after the other, the
// error of a column sum grows with the rows: 7.5e-7 at 12 800 rows and 1.6e-6 at 15 314, against 2.2e-7 for sums of
// blocks of 128 rows; this way 9e-8.)
__device__ __forceinline__ void colsum_add32(const float (&f)[32], float& sum, float& lost) {
  float t[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) t[i] = __fadd_rn(f[i], f[i + 16]);
#pragma unroll
  for (int n = 8; n > 0; n >>= 1)
#pragma unroll
    for (int i = 0; i < n; ++i) t[i] = __fadd_rn(t[i], t[i + n]);
  const float s = __fadd_rn(sum, t[0]), b = __fsub_rn(s, sum);
  lost = __fadd_rn(lost, __fadd_rn(__fsub_rn(sum, __fsub_rn(s, b)), __fsub_rn(t[0], b)));
  sum = s;
}
__device__ __forceinline__ void sts128(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}

// A converter's arrival on the leader's barrier, and the leader's side of it.  The arrival of the other CTA is what lets the
// leader's MMA read that CTA's shared memory, so it releases at the scope of the cluster, but only what is in its own
// shared memory: a release of everything waits for the warp's load of the next scales as well, half a microsecond an
// arrival (61 -> 106 us for dw alone at 12 800 x 2048 x 512, this way 62).
__device__ __forceinline__ void mbar_arrive_shared_release(uint32_t bar, uint32_t rank) {
  uint32_t remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(bar), "r"(rank));
  asm volatile("fence.release.sync_restrict::shared::cta.cluster;" ::: "memory");
  asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(remote) : "memory");
}
__device__ __forceinline__ void fence_shared_acquire() { asm volatile("fence.acquire.sync_restrict::shared::cluster.cluster;" ::: "memory"); }

__global__ void __launch_bounds__(DwCfg::kThreads, 1)
dw_split_kernel(const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_b, const __grid_constant__ CUtensorMap tm_y,
                const DwParams p) {
  using Cfg = DwCfg;
  constexpr int EW = Cfg::EW, STAGES = Cfg::STAGES, BN = Cfg::BN, HALF = BN / 2, TILE_M = 2 * kBM, SBUFS = Cfg::kStageBufs;
  const uint32_t pair_rank = cluster_ctarank();
  const int row_in_tile = (int)pair_rank * kBM;

  extern __shared__ uint8_t smem_raw[];
  __shared__ uint64_t full_bar[STAGES];   // this CTA's loads of a stage have landed
  __shared__ uint64_t conv_bar[STAGES];   // leader: both CTAs' stage is converted
  __shared__ uint64_t empty_bar[STAGES];  // the pair's MMAs have read the stage
  __shared__ uint64_t tmem_full_bar[2];
  __shared__ uint64_t tmem_empty_bar[2];
  __shared__ uint32_t tmem_base_slot;
  __shared__ int abort_flag;

  const uint32_t smem_ring = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t smem_epi = smem_ring + STAGES * Cfg::kStageBytes;
  const uint32_t smem_conv = smem_epi + Cfg::kEpiBytes;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint64_t t_start = global_timer_ns();

  if (threadIdx.x == 0) {
    abort_flag = 0;
    tma_prefetch_desc(&tm_a);
    tma_prefetch_desc(&tm_b);
    tma_prefetch_desc(&tm_y);
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(smem_u32(&full_bar[s]), 1);
      mbar_init(smem_u32(&conv_bar[s]), 8);  // four warps of either CTA
      mbar_init(smem_u32(&empty_bar[s]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&tmem_full_bar[b]), 1);
      mbar_init(smem_u32(&tmem_empty_bar[b]), 2 * EW);
    }
    fence_barrier_init();
    fence_proxy_async_smem();
  }
  if (warp == 1) {
    tmem_alloc_pair(smem_u32(&tmem_base_slot), 2 * BN);
    tmem_relinquish_pair();
  }
  if (!p.beside_previous) grid_dependency_wait();
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_slot;

  const int n_tiles = p.tiles_m * p.tiles_n;
  const int pair0 = (int)(blockIdx.x >> 1), pairs = (int)(gridDim.x >> 1);

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer (both CTAs)
    if (lane == 0) {
      uint32_t it = 0;
      bool ok = true;
      for (int tile = pair0; ok && tile < n_tiles; tile += pairs) {
        const int tm = tile / p.tiles_n, tn = tile - tm * p.tiles_n;
        const int batch = tm / p.batch_tiles_m, m0 = (tm - batch * p.batch_tiles_m) * TILE_M + row_in_tile, k0 = batch * p.batch_k;
        const int n0 = tn * BN + (int)pair_rank * HALF;
        for (int kb = 0; kb < p.k_blocks; ++kb, ++it) {
          const uint32_t s = it % STAGES, ph = (it / STAGES) & 1;
          if (!mbar_wait(smem_u32(&empty_bar[s]), ph ^ 1, &abort_flag, t_start)) { ok = false; break; }
          const uint32_t bar = smem_u32(&full_bar[s]), stage = smem_ring + s * Cfg::kStageBytes;
          mbar_arrive_expect_tx(bar, Cfg::kStageBytes);
#pragma unroll
          for (int b = 0; b < 4; ++b) tma_load_2d(stage + b * 4096, &tm_a, m0 + 32 * b, k0 + kb * 32, bar);
          tma_load_2d(stage + Cfg::kABytes, &tm_b, k0 + kb * 32, n0, bar);
        }
      }
      if (!p.beside_previous) grid_dependents_launch();
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer (leader)
    if (lane == 0 && pair_rank == 0) {
      constexpr uint32_t idesc = idesc_bf16(BN, TILE_M);
      uint32_t it = 0, tcount = 0;
      bool ok = true;
      for (int tile = pair0; ok && tile < n_tiles; tile += pairs, ++tcount) {
        const uint32_t buf = tcount & 1, aph = (tcount >> 1) & 1;
        if (!mbar_wait(smem_u32(&tmem_empty_bar[buf]), aph ^ 1, &abort_flag, t_start)) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + buf * BN;
        for (int kb = 0; kb < p.k_blocks; ++kb, ++it) {
          const uint32_t s = it % STAGES, ph = (it / STAGES) & 1;
          if (!mbar_wait(smem_u32(&conv_bar[s]), ph, &abort_flag, t_start)) { ok = false; break; }
          fence_shared_acquire();
          tc_fence_after();
          const uint32_t stage = smem_ring + s * Cfg::kStageBytes;
          const uint64_t a_desc = smem_desc_k_major_sw128(stage), b_desc = smem_desc_k_major_sw64(stage + Cfg::kABytes);
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)  // hi 0..15, hi 16..31, lo 0..15, lo 16..31: 32 bytes of the row each
            tc_mma_bf16_pair(d_tmem, a_desc + 2 * kk, b_desc + 2 * (kk & 1), idesc, (kb | kk) != 0 ? 1u : 0u);
          tc_commit_pair(smem_u32(&empty_bar[s]));
        }
        if (ok) tc_commit_pair(smem_u32(&tmem_full_bar[buf]));
      }
    }
  } else if (warp >= 2 + EW) {
    // ------------------------------------------------------------------ converters
    const int cw = warp - (2 + EW);
    const int quad = cw & 3, group = cw >> 2;  // box of the stage; K-blocks of one parity
    const uint32_t my_scale = smem_conv + cw * 128;
    uint32_t it = 0;
    bool ok = true;
    for (int tile = pair0; ok && tile < n_tiles; tile += pairs) {
      const int tm = tile / p.tiles_n, tn = tile - tm * p.tiles_n;
      const int batch = tm / p.batch_tiles_m, k0 = batch * p.batch_k;
      const int m = (tm - batch * p.batch_tiles_m) * TILE_M + row_in_tile + quad * 32 + lane;  // this lane's row of the product
      const bool sums = p.colsum != nullptr && tn == 0;
      float colsum = 0.0f, colsum_lost = 0.0f;
      // scale of this lane's contraction index, one K-block of the group ahead
      auto scale_at = [&](int kb) {
        const int k = k0 + kb * 32 + lane;
        return kb < p.k_blocks && k < p.K ? __ldg(p.a_scale + (int64_t)k * p.a_scale_step) : 0.0f;
      };
      int kb = (int)(((uint32_t)group + Cfg::kGroups - it % Cfg::kGroups) % Cfg::kGroups);  // first K-block of this tile in the group's turn
      float next_scale = scale_at(kb);
      for (; ok && kb < p.k_blocks; kb += Cfg::kGroups) {
        const uint32_t its = it + kb;
        const uint32_t s = its % STAGES, ph = (its / STAGES) & 1;
        const uint32_t stage = smem_ring + s * Cfg::kStageBytes;
        __syncwarp();
        asm volatile("st.shared.f32 [%0], %1;" ::"r"(my_scale + lane * 4), "f"(next_scale) : "memory");
        __syncwarp();
        next_scale = scale_at(kb + Cfg::kGroups);
        if (!mbar_wait(smem_u32(&full_bar[s]), ph, &abort_flag, t_start)) { ok = false; break; }
        float f[32];
        const uint32_t box = stage + quad * 4096 + (lane & 3) * 4;  // row k of the box: 128 bytes, 16-byte chunk j at j ^ (k & 7)
#pragma unroll
        for (int k = 0; k < 32; ++k)
          asm volatile("ld.shared.f32 %0, [%1];" : "=f"(f[k]) : "r"(box + k * 128 + ((((uint32_t)lane >> 2) ^ (k & 7)) << 4)) : "memory");
        if (sums) colsum_add32(f, colsum, colsum_lost);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          float s0, s1, s2, s3;
          asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(s0), "=f"(s1), "=f"(s2), "=f"(s3) : "r"(my_scale + 16 * j) : "memory");
          const float2 u = __fmul2_rn(make_float2(f[4 * j], f[4 * j + 1]), make_float2(s0, s1));
          const float2 v = __fmul2_rn(make_float2(f[4 * j + 2], f[4 * j + 3]), make_float2(s2, s3));
          f[4 * j] = u.x;
          f[4 * j + 1] = u.y;
          f[4 * j + 2] = v.x;
          f[4 * j + 3] = v.y;
        }
        __syncwarp();  // the whole box has been read
        const uint32_t row = stage + (uint32_t)(quad * 32 + lane) * 128;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          uint32_t hi[4], lo[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) split_bf16x2(f[8 * c + 2 * e], f[8 * c + 2 * e + 1], hi[e], lo[e]);
          sts128(row + ((c ^ (lane & 7)) << 4), hi[0], hi[1], hi[2], hi[3]);
          sts128(row + (((c + 4) ^ (lane & 7)) << 4), lo[0], lo[1], lo[2], lo[3]);
        }
        fence_proxy_async_smem();  // the tensor core reads the rows through the async proxy
        __syncwarp();
        if (lane == 0) {
          if (pair_rank == 0) mbar_arrive(smem_u32(&conv_bar[s]));
          else mbar_arrive_shared_release(smem_u32(&conv_bar[s]), 0);
        }
      }
      it += p.k_blocks;
      if (ok && sums && m < p.M) {
        const float t = __fadd_rn(colsum, colsum_lost);
        p.colsum[(int64_t)(batch * Cfg::kGroups + group) * p.M + m] = t == t ? t : colsum;  // (an infinite sum loses a NaN)
      }
    }
  } else {
    // ------------------------------------------------------------------ epilogue warps: accumulators -> fp32 output
    const int ew = warp - 2;
    const int quad = warp & 3;
    const uint32_t my_stage = smem_epi + ew * SBUFS * kStageBufBytes;
    uint32_t store_count = 0, tcount = 0;
    for (int tile = pair0; tile < n_tiles; tile += pairs, ++tcount) {
      const int tm = tile / p.tiles_n, tn = tile - tm * p.tiles_n;
      const uint32_t buf = tcount & 1, aph = (tcount >> 1) & 1;
      const int row0_warp = tm * TILE_M + row_in_tile + quad * 32;
      if (!mbar_wait(smem_u32(&tmem_full_bar[buf]), aph, &abort_flag, t_start)) break;
      tc_fence_after();
      const uint32_t lane_addr = tmem_base + buf * BN + ((uint32_t)(quad * 32) << 16);
      for (int c = 0; c < BN / 32; ++c) {
        const int oc = tn * BN + c * 32;
        const uint32_t sbuf = my_stage + (store_count % SBUFS) * kStageBufBytes;
        uint32_t acc[32];
        tmem_ld_32x32(lane_addr + c * 32, acc);
        tmem_ld_wait();
        if (c == BN / 32 - 1) {  // accumulator buffer read out by this warp
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_cluster(smem_u32(&tmem_empty_bar[buf]), 0);
        }
        if (lane == 0) tma_store_wait_read<SBUFS - 1>();
        __syncwarp();
#pragma unroll
        for (int j = 0; j < 8; ++j) sts128(sbuf + lane * 128 + ((j ^ (lane & 7)) << 4), acc[4 * j], acc[4 * j + 1], acc[4 * j + 2], acc[4 * j + 3]);
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {
          if (oc < p.N && row0_warp < p.y_rows) tma_store_2d(&tm_y, sbuf, oc, row0_warp);
          tma_store_commit();
        }
        ++store_count;
      }
    }
    if (lane == 0) tma_store_wait_all();
  }

  tc_fence_before();
  __syncthreads();
  if (abort_flag && threadIdx.x == 0) {
    // give bulk copies that were in flight when a wait gave up time to land before smem is released
    const uint64_t t0 = global_timer_ns();
    while (global_timer_ns() - t0 < 200000ull) {
    }
  }
  __syncthreads();
  cluster_sync_all();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, 2 * BN);
  }
  // (one pair is enough to keep the launch from ending first; the others free their SMs for the next tiles)
  if (p.beside_previous && blockIdx.x + 2 >= gridDim.x) grid_dependency_wait();
}

// ------------------------------------------------------------------------------------------------
// Host side

// a: [K, M] floats with lda floats between rows.  b: bf16 codes [N, K], b_pitch elements between rows (a multiple of 8).
// y: [y_rows, N], ldy; y_rows: M, or the stacked rows of all batches (p.batch_k set).
static int launch_dw_split(const float* a, int64_t lda, const void* b, int64_t b_pitch, float* y, int64_t y_rows, int64_t ldy, DwParams p,
                           int batches, cudaStream_t st) {
  using Cfg = DwCfg;
  const int sms = sm_count();
  if (sms <= 0) return AQT_ERR_CUDA;
  const int tiles_m = (int)ceil_div(p.M, 2 * kBM);
  p.batch_tiles_m = tiles_m;
  p.y_rows = (int)y_rows;
  p.tiles_m = tiles_m * batches;
  p.tiles_n = (int)ceil_div(p.N, Cfg::BN);
  if (batches == 1) p.batch_k = 0;
  p.k_blocks = (int)ceil_div(batches == 1 ? p.K : p.batch_k, 32);
  CUtensorMap tm_a, tm_b, tm_y;
  int rc = make_map_2d(&tm_a, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, a, (uint64_t)p.K, (uint64_t)p.M, (uint64_t)lda * 4, 32, 32);
  if (rc != AQT_OK) return rc;
  rc = make_map_2d(&tm_b, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, b, (uint64_t)p.N, (uint64_t)p.K, (uint64_t)b_pitch * 2, Cfg::BN / 2, 32, 64);
  if (rc != AQT_OK) return rc;
  rc = make_map_2d(&tm_y, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, y, (uint64_t)y_rows, (uint64_t)p.N, (uint64_t)ldy * 4, kStoreBoxRows, kStoreBoxCols);
  if (rc != AQT_OK) return rc;
  static std::atomic<uint64_t> smem_opted_in{0};
  rc = ensure_dynamic_smem(dw_split_kernel, Cfg::kSmemBytes, smem_opted_in);
  if (rc != AQT_OK) return rc;
  const int64_t tiles = (int64_t)p.tiles_m * p.tiles_n, pairs = sms / 2;
  // (beside another launch: one tile per pair of CTAs, dealt out by the hardware as SMs fall free)
  const unsigned grid = 2u * (unsigned)(tiles < pairs || p.beside_previous ? tiles : pairs);
  return launch_pdl(dw_split_kernel, dim3(grid, 1, 1), dim3(Cfg::kThreads, 1, 1), Cfg::kSmemBytes, st, 2, tm_a, tm_b, tm_y, p);
}

}  // namespace aqt
