// The integer matmul for outputs of a few tiles (sm_100a): one narrow tile per CTA, all sixteen epilogue
// warps on it, optionally with the row quantizer of Fig. 2 on (the last columns of) its output.
//
//   acc = xq * wq^T (int32, TMEM);  u = residual + residual_scale * act(fma(float(acc) * s_x, s_w, bias))
//   y = u (if wanted);  s_out[m] = max |u[m][n]| / qmax over n >= rq_first;  q_out[m][n - rq_first] = round(u / s_out)
//
// With a few hundred to a thousand rows a layer is a chain of latencies, not of bytes.  What one launch of
// 1013 x 512 -> 512 on 128 x 128 tiles (32 CTAs) spent, by stamps in a copy of the kernel: 1.25 us from the end of
// the kernel ahead to the first load, 1.7 to the finished accumulators, 1.9 in the epilogue (the 128 x 128 values of a
// tile are 700 instructions a warp, and the schedulers of one SM issue them at one a clock whatever the number of
// warps), 0.9 for the exchange of the row maxima, 0.8 in the codes.  So
//   - the tile is as narrow as leaves every tile an SM of its own: 32, 64 or 128 columns, and a warp keeps its 8, 16
//     or 32 columns of u in registers between the two passes;
//   - both operands go through one ring as deep as shared memory allows (with five stages the 16 k-blocks of a 2048-deep
//     contraction took 5.0 us, three round trips of a load);
//   - weights that were complete before the kernel ahead fill their part of the ring while that kernel drains.
// Measured (graph replay, us): see few_tiles_bn.
//
// The exchange of row maxima (collect_maxima), the tags of its words (hand_out_tag) and the bounded waits are those of
// qgemm_requant_sm100.cuh.
#pragma once

#include "qgemm_requant_sm100.cuh"

namespace aqt {

struct FewTilesParams {
  RequantParams rp;   // rp.g: the matmul; exchange words by [m-tile][quantizing n-tile][row]
  int rq_first;       // first output column that is quantized; n_out: none
  int b_packed;       // weights: packed nibbles (K <= 512), expanded into the ring's stages
};

// BN: weight rows (TMEM columns) per tile.  GLU: half of them values, half gates.
template <int BN, bool GLU>
struct FewTilesCfg {
  static constexpr int EW = 16;
  static constexpr int kThreads = 32 * (2 + EW + 2);  // producer, MMA issuer, epilogue warps, two exchange warps
  static constexpr int kOutCols = GLU ? BN / 2 : BN;  // output columns of a tile
  static constexpr int C = kOutCols / 4;              // ... of a warp
  static constexpr int kBBytes = BN * kBK;
  static constexpr int kStageBytes = kBM * kBK + kBBytes;
  static constexpr int kYBytes = EW * 32 * C * 4;     // a 32 x C box of floats per warp: residual, then output
  static constexpr int kPackedBytes = kWsMaxKBlocks * BN * 64;  // packed weights wait in the same place
  static constexpr int kEpiBytes = kYBytes > kPackedBytes ? kYBytes : kPackedBytes;
  static constexpr int kSlabCols = GLU ? 2 * C : C;   // scales and biases of a warp's weight rows: values, then gates
  static constexpr int kScaleBytes = EW * 2 * kSlabCols * 4;
  static constexpr int kStages = BN == 128 ? 4 : (BN == 64 ? 7 : 9);
  static constexpr int kTmemCols = BN;
  static constexpr int kSmemBytes = kStages * kStageBytes + kEpiBytes + kScaleBytes + 1024;
  static_assert(C == 8 || C == 16 || C == 32, "columns of a warp");
  static_assert(kStages >= kWsMaxKBlocks, "packed weights: every k-block has a stage of its own");
  static_assert(kSmemBytes + 4096 <= 232448, "must fit the 227 KB a CTA can opt into");
};

// 32 lanes x C consecutive 32-bit columns.
__device__ __forceinline__ void tmem_ld_cols(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr)
               : "memory");
}
__device__ __forceinline__ void tmem_ld_cols(uint32_t taddr, uint32_t (&r)[16]) { tmem_ld_32x16(taddr, r); }
__device__ __forceinline__ void tmem_ld_cols(uint32_t taddr, uint32_t (&r)[32]) { tmem_ld_32x32(taddr, r); }

// Accumulators of row m from column n on, those below `limit`, as the matrix product that they are (DEBUG).
template <int C>
__device__ __forceinline__ void dump_acc(const GemmParams& p, int m, int n, int limit, const uint32_t (&acc)[C]) {
  if (m >= p.M) return;
#pragma unroll
  for (int j = 0; j < C; ++j)
    if (n + j < limit) p.acc_debug[(int64_t)m * p.N + n + j] = (int32_t)acc[j];
}

// Byte offset of 16-byte chunk j of row r in a box of 32 rows x C floats as the copy engine lays it out under the
// swizzle of its row length (32, 64 or 128 bytes).
template <int C>
__device__ __forceinline__ uint32_t box_offset(int r, int j) {
  if (C == 32) return (uint32_t)(r * 128 + ((j ^ (r & 7)) << 4));
  if (C == 16) return (uint32_t)(r * 64 + ((j ^ ((r >> 1) & 3)) << 4));
  return (uint32_t)(r * 32 + ((j ^ ((r >> 2) & 1)) << 4));
}

template <int BN, bool GLU, bool DEBUG>
__global__ void __launch_bounds__(32 * 20, 1)
qgemm_few_tiles_kernel(const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_b,
                       const __grid_constant__ CUtensorMap tm_y, const __grid_constant__ CUtensorMap tm_r, const FewTilesParams fp) {
  using Cfg = FewTilesCfg<BN, GLU>;
  constexpr int EW = Cfg::EW, STAGES = Cfg::kStages, HALF = BN / 2, C = Cfg::C;
  const RequantParams& rp = fp.rp;
  const GemmParams& p = rp.g;

  extern __shared__ uint8_t smem_raw[];
  __shared__ uint64_t full_bar[STAGES];
  __shared__ uint64_t empty_bar[STAGES];
  __shared__ uint64_t acc_bar;       // the tile's accumulators are complete
  __shared__ uint64_t b_loaded_bar;  // packed weights have landed
  __shared__ uint64_t b_ready_bar;   // ... and are expanded in the stages
  __shared__ uint64_t res_bar[EW];   // a warp's residual box has landed
  __shared__ uint64_t part_bar[4];   // sets 1 .. 3 have left their maxima of this lane quadrant's rows
  __shared__ uint64_t ctx_bar[2];    // an exchange warp has the final maxima of its half of the rows
  __shared__ uint64_t tag_bar;       // tag_slot is there
  __shared__ uint32_t tag_slot;
  __shared__ float part_amax[4][kBM];
  __shared__ __align__(16) uint32_t row_amax[kBM];
  __shared__ uint32_t tmem_base_slot;
  __shared__ int abort_flag;

  const uint32_t smem_ring = (smem_u32(smem_raw) + 1023u) & ~1023u;  // stage: activations, then weights
  const uint32_t smem_epi = smem_ring + STAGES * Cfg::kStageBytes;
  const uint32_t smem_scale = smem_epi + Cfg::kEpiBytes;
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const uint64_t t_start = global_timer_ns();

  const int tm = blockIdx.x / p.tiles_n;
  const int tn = blockIdx.x - tm * p.tiles_n;
  const int tn_first = fp.rq_first / Cfg::kOutCols;  // first n-tile whose columns are quantized
  const int parts = p.tiles_n - tn_first;
  const bool rq = tn >= tn_first;

  // The weights (codes, scales, bias) may be read before the kernel ahead has finished if the caller said so; every role
  // waits for that kernel before its first access to anything else.
  const bool early_w = p.static_w != 0;
  const int row0 = GLU ? tn * HALF : tn * BN, row1 = GLU ? p.N / 2 + tn * HALF : tn * BN + HALF;  // the tile's weight rows
  const int first = p.k_blocks < STAGES ? p.k_blocks : STAGES;  // k-blocks that find their stage empty

  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(smem_u32(&full_bar[s]), 1);
      mbar_init(smem_u32(&empty_bar[s]), 1);
    }
    mbar_init(smem_u32(&acc_bar), 1);
    mbar_init(smem_u32(&b_loaded_bar), 1);
    mbar_init(smem_u32(&b_ready_bar), EW);
    for (int w = 0; w < EW; ++w) mbar_init(smem_u32(&res_bar[w]), 1);
    for (int q = 0; q < 4; ++q) mbar_init(smem_u32(&part_bar[q]), 3);
    for (int h = 0; h < 2; ++h) mbar_init(smem_u32(&ctx_bar[h]), 1);
    mbar_init(smem_u32(&tag_bar), 2);
    fence_barrier_init();
    fence_proxy_async_smem();
    // the weights' loads are on their way before the CTA's set-up is complete
    if (!early_w) grid_dependency_wait();
    if (fp.b_packed) {
      const uint32_t bar = smem_u32(&b_loaded_bar);
      mbar_arrive_expect_tx(bar, (uint32_t)p.k_blocks * BN * 64);
      for (int kb = 0; kb < p.k_blocks; ++kb) {
        tma_load_2d(smem_epi + kb * BN * 64, &tm_b, kb * 64, row0, bar);
        tma_load_2d(smem_epi + kb * BN * 64 + HALF * 64, &tm_b, kb * 64, row1, bar);
      }
    } else {
      for (int kb = 0; kb < first; ++kb) {
        const uint32_t bar = smem_u32(&full_bar[kb]), b = smem_ring + kb * Cfg::kStageBytes + kBM * kBK;
        mbar_arrive_expect_tx(bar, Cfg::kStageBytes);
        tma_load_2d(b, &tm_b, kb * kBK, row0, bar);
        tma_load_2d(b + HALF * kBK, &tm_b, kb * kBK, row1, bar);
      }
    }
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(&tmem_base_slot), Cfg::kTmemCols);
    tmem_relinquish();
  }
  if (threadIdx.x == 64) {
    tma_prefetch_desc(&tm_a);
    if (p.has_y) tma_prefetch_desc(&tm_y);
    if (p.residual != nullptr) tma_prefetch_desc(&tm_r);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_slot;

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    if (lane == 0) {
      if (early_w) grid_dependency_wait();  // the activation codes come from the kernel ahead
      for (int kb = 0; kb < first; ++kb) {
        const uint32_t bar = smem_u32(&full_bar[kb]);
        if (fp.b_packed) mbar_arrive_expect_tx(bar, kBM * kBK);
        tma_load_2d(smem_ring + kb * Cfg::kStageBytes, &tm_a, kb * kBK, tm * kBM, bar);
      }
      for (int kb = first; kb < p.k_blocks; ++kb) {
        const uint32_t s = kb % STAGES, ph = (kb / STAGES) & 1;
        if (!mbar_wait(smem_u32(&empty_bar[s]), ph ^ 1, &abort_flag, t_start)) break;
        const uint32_t bar = smem_u32(&full_bar[s]), a = smem_ring + s * Cfg::kStageBytes;
        mbar_arrive_expect_tx(bar, Cfg::kStageBytes);
        tma_load_2d(a, &tm_a, kb * kBK, tm * kBM, bar);
        tma_load_2d(a + kBM * kBK, &tm_b, kb * kBK, row0, bar);
        tma_load_2d(a + kBM * kBK + HALF * kBK, &tm_b, kb * kBK, row1, bar);
      }
      grid_dependents_launch();
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    if (lane == 0) {
      constexpr uint32_t idesc = idesc_i8(BN, kBM);
      bool ok = !fp.b_packed || mbar_wait(smem_u32(&b_ready_bar), 0, &abort_flag, t_start);
      for (int kb = 0; ok && kb < p.k_blocks; ++kb) {
        const uint32_t s = kb % STAGES, ph = (kb / STAGES) & 1;
        if (!mbar_wait(smem_u32(&full_bar[s]), ph, &abort_flag, t_start)) { ok = false; break; }
        tc_fence_after();
        const uint32_t stage = smem_ring + s * Cfg::kStageBytes;
        const uint64_t a_desc = smem_desc_k_major_sw128(stage), b_desc = smem_desc_k_major_sw128(stage + kBM * kBK);
#pragma unroll
        for (int kk = 0; kk < kBK / kMmaK; ++kk) tc_mma_i8(tmem_base, a_desc + 2 * kk, b_desc + 2 * kk, idesc, (kb | kk) != 0 ? 1u : 0u);
        if (kb + STAGES < p.k_blocks) tc_commit(smem_u32(&empty_bar[s]));
      }
      if (ok) tc_commit(smem_u32(&acc_bar));
    }
  } else if (warp >= 2 + EW) {
    // ------------------------------------------------------------------ exchange warps
    // Lane l of warp h owns rows 64h + 2l and 64h + 2l + 1: one 16-byte load (two words) per n-tile.
    if (rq) {
      const int xh = warp - (2 + EW);
      grid_dependency_wait();
      const uint32_t tag = hand_out_tag(rp, tm, &tag_slot, &tag_bar);
      const uint64_t* xt = rp.exchange + (size_t)tm * parts * kBM + 64 * xh + 2 * lane;
      uint2 m2;
      if (collect_maxima(xt, parts, tag, &abort_flag, t_start, m2)) {
        *reinterpret_cast<uint2*>(&row_amax[64 * xh + 2 * lane]) = m2;
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&ctx_bar[xh]));
      }
    }
  } else {
    // ------------------------------------------------------------------ epilogue warps
    const int ew = warp - 2;
    const int quad = warp & 3;  // TMEM lane quadrant this warp may access
    const int set = ew >> 2;    // its quarter of the tile's output columns
    const int row_in_tile = quad * 32 + lane;
    const int row0_warp = tm * kBM + quad * 32, m = row0_warp + lane;
    const uint32_t box = smem_epi + ew * (32 * C * 4);
    const int oc = tn * Cfg::kOutCols + set * C;  // first output column
    const bool cols_ok = oc < p.n_out;
    const bool has_res = p.residual != nullptr;
    bool ok = true;
    // the same answer in every lane: what follows synchronises the warp
    const auto wait = [&](const uint64_t& bar) { return __all_sync(0xffffffffu, mbar_wait(smem_u32(&bar), 0, &abort_flag, t_start)) != 0; };

    // scales and biases of this warp's weight rows
    const uint32_t slab = smem_scale + ew * (2 * Cfg::kSlabCols * 4), slab_bias = slab + Cfg::kSlabCols * 4;
    if (!early_w) grid_dependency_wait();
    if (lane < Cfg::kSlabCols) {
      const int n = !GLU || lane < C ? oc + lane : p.N / 2 + oc + lane - C;
      float wv = 0.0f, bv = 0.0f;
      if (n < (GLU && lane < C ? p.N / 2 : p.N)) {
        wv = __ldg(p.s_w + n);
        if (p.bias != nullptr) bv = __ldg(p.bias + n);
      }
      asm volatile("st.shared.f32 [%0], %1;" ::"r"(slab + lane * 4), "f"(wv) : "memory");
      asm volatile("st.shared.f32 [%0], %1;" ::"r"(slab_bias + lane * 4), "f"(bv) : "memory");
    }
    __syncwarp();
    if (fp.b_packed) {
      // sign-extend the packed weights into the stages (layout of a swizzled load of int8 codes)
      ok = wait(b_loaded_bar);
      if (ok) {
        expand_packed_slab<BN, EW * 32>(smem_epi, smem_ring + kBM * kBK, Cfg::kStageBytes, p.k_blocks, ew * 32 + lane);
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&b_ready_bar));
        ok = wait(b_ready_bar);  // the boxes lie over the packed weights
      }
    }
    if (early_w) grid_dependency_wait();
    if (ok && has_res && lane == 0) {
      mbar_arrive_expect_tx(smem_u32(&res_bar[ew]), 32 * C * 4);
      // (a box that would start outside the tensor is redirected to its origin and never used)
      tma_load_2d(box, &tm_r, cols_ok ? oc : 0, row0_warp < p.M ? row0_warp : 0, smem_u32(&res_bar[ew]));
    }
    const float sx = p.s_x_kind == AQT_SCALE_ROW ? (m < p.M ? __ldg(p.s_x + m) : 0.0f) : __ldg(p.s_x);

    if (ok && rq && set == 0) ok = wait(tag_bar);  // (long before the accumulators are complete)
    const uint32_t tag = *(volatile uint32_t*)&tag_slot;
    float a[C];
    if (ok) ok = wait(acc_bar);
    if (ok) {
      tc_fence_after();
      const uint32_t t_addr = tmem_base + ((uint32_t)(quad * 32) << 16) + set * C;
      uint32_t acc[C];
      if constexpr (GLU) {
        uint32_t accg[C];
        float g[C];
        tmem_ld_cols(t_addr + HALF, accg);
        tmem_ld_cols(t_addr, acc);
        tmem_ld_wait();
        if (DEBUG) dump_acc<C>(p, m, p.N / 2 + oc, p.N, accg);
        if (DEBUG) dump_acc<C>(p, m, oc, p.N / 2, acc);
        dequant_smem<kAccInt32>(accg, sx, slab + C * 4, slab_bias + C * 4, g);
        dequant_smem<kAccInt32>(acc, sx, slab, slab_bias, a);
#pragma unroll
        for (int j = 0; j < C; ++j) a[j] = __fmul_rn(a[j], sigmoid_f(g[j]));
        if (p.act == AQT_ACT_GLU_SWISH) swish(a);
      } else {
        tmem_ld_cols(t_addr, acc);
        tmem_ld_wait();
        if (DEBUG) dump_acc<C>(p, m, oc, p.N, acc);
        dequant_smem<kAccInt32>(acc, sx, slab, slab_bias, a);
        if (p.act == AQT_ACT_SWISH) swish(a);
      }
      if (has_res) {
        ok = wait(res_bar[ew]);
        if (ok) {
#pragma unroll
          for (int j = 0; j < C / 4; ++j) {
            float r0, r1, r2, r3;
            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(r0), "=f"(r1), "=f"(r2), "=f"(r3) : "r"(box + box_offset<C>(lane, j)) : "memory");
            a[4 * j + 0] = __fmaf_rn(p.residual_scale, a[4 * j + 0], r0);
            a[4 * j + 1] = __fmaf_rn(p.residual_scale, a[4 * j + 1], r1);
            a[4 * j + 2] = __fmaf_rn(p.residual_scale, a[4 * j + 2], r2);
            a[4 * j + 3] = __fmaf_rn(p.residual_scale, a[4 * j + 3], r3);
          }
          __syncwarp();  // every lane has read its residual row before the box is overwritten
        }
      }
    }
    float amax = 0.0f;
    if (ok && rq) {
      // the row's maximum over the tile: the first set's warp collects and publishes it
      if (cols_ok) {
#pragma unroll
        for (int j = 0; j < C; ++j) amax = fmaxf(amax, fabsf(a[j]));
      }
      part_amax[set][row_in_tile] = amax;
      __syncwarp();
      if (set != 0) {
        if (lane == 0) mbar_arrive(smem_u32(&part_bar[quad]));
      } else {
        ok = wait(part_bar[quad]);
        for (int s = 1; s < 4; ++s) amax = fmaxf(amax, part_amax[s][row_in_tile]);
        if (ok) st_relaxed_gpu_64(rp.exchange + ((size_t)tm * parts + (tn - tn_first)) * kBM + row_in_tile, ((uint64_t)tag << 32) | __float_as_uint(amax));
      }
    }
    if (ok && p.has_y) {
#pragma unroll
      for (int j = 0; j < C / 4; ++j)
        asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(box + box_offset<C>(lane, j)), "f"(a[4 * j]), "f"(a[4 * j + 1]),
                     "f"(a[4 * j + 2]), "f"(a[4 * j + 3])
                     : "memory");
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0 && cols_ok && row0_warp < p.M) {
        tma_store_2d(&tm_y, box, oc, row0_warp);
        tma_store_commit();
      }
    }
    const float any_nan = chunk_max(0.0f, a);  // (this warp has nothing to do until the other CTAs have published)
    if (ok && rq) ok = wait(ctx_bar[quad >> 1]);
    if (ok && rq) {
      ScaleCtx sc = make_scale_ctx_zeros(__uint_as_float(row_amax[row_in_tile]), rp.qmax_out);
      sc.fast = sc.fast && any_nan == any_nan;  // see chunk_max
      if (tn == tn_first && set == 0 && m < p.M) rp.s_out[m] = sc.s;
      uint32_t u[C], w[C / 4];
#pragma unroll
      for (int j = 0; j < C; ++j) u[j] = __float_as_uint(a[j]);
      if (rp.rounding == AQT_ROUND_HALF_UP_FLOOR) codes_of<AQT_ROUND_HALF_UP_FLOOR, false, C>(u, sc, rp.qmax_out, w);
      else codes_of<AQT_ROUND_NEAREST_EVEN, false, C>(u, sc, rp.qmax_out, w);
      if (m < p.M && cols_ok) {
        const int q_cols = p.n_out - fp.rq_first;  // a multiple of 16, as rq_first is one of the tile's columns
        uint8_t* dst = rp.q_out + (size_t)m * q_cols + (oc - fp.rq_first);
        if constexpr (C == 8) {
          *reinterpret_cast<uint2*>(dst) = make_uint2(w[0], w[1]);
        } else {
          *reinterpret_cast<uint4*>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
          if constexpr (C == 32) {
            if (oc + 16 < p.n_out) *reinterpret_cast<uint4*>(dst + 16) = make_uint4(w[4], w[5], w[6], w[7]);
          }
        }
      }
    }
    if (lane == 0) tma_store_wait_all();
  }

  // ------------------------------------------------------------------ teardown
  tc_fence_before();
  __syncthreads();
  if (abort_flag && threadIdx.x == 0) {
    // give bulk copies that were in flight when a wait gave up time to land before smem is released
    const uint64_t t0 = global_timer_ns();
    while (global_timer_ns() - t0 < 200000ull) {
    }
  }
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem_base, Cfg::kTmemCols);
  }
  // every CTA of the m-tile has read the counter (hand_out_tag): this one could not finish without their maxima
  if (rq && tn == tn_first && threadIdx.x == 0) rp.generation[tm] = __ldcg(rp.generation + tm) + 1u;
}

// Tile width for a call, 0 where the kernel does not take it or another form is faster.  rq_first: as in FewTilesParams, -1
// for a call that quantizes nothing.  The narrowest width that leaves every tile an SM of its own; measured over 15 row
// counts from 17 to 4736, nine N from 128 to 4096 and seven K from 128 to 4096 (148 SMs, graph replay, new time / old, mean and
// worst of each group):
//   - K <= 512: matmul 0.62-0.78 / 0.82 on 32 and 64 columns, 0.88-0.93 / 0.95 on 128; the whole layer on floats 0.71-0.83 / 0.93
//     and 0.90-0.94 / 0.97; with the row quantizer 0.74-0.90 / 0.96 and 0.86-0.96 / 1.00 (against the weight-stationary tiles
//     of 128 columns).  At most sixteen parts of a row, which an exchange warp reads in one go, unless the tile is 128 wide
//     (64 parts 1.05 / 1.25, 128 parts 1.34 / 1.71).  Without the row quantizer at most 64 n-tiles below 128 columns: beyond,
//     a few rows lose with the narrower tiles (us at the wider and the narrower: 20 x 512 -> 4096 4.21 / 4.52, -> 9472 4.53 /
//     5.27, 64 x 512 -> 9472 4.72 / 4.95), while full tiles and short contractions would gain (128 x 512 -> 4736 5.14 / 4.31,
//     20 x 128 -> 4736 3.35 / 3.08): against the kernels before this one either is faster.
//   - deeper: with the row quantizer 0.72-0.97 / 1.02 (two kernels, or pairs); without one only the gate forms, from 65
//     rows on, 0.90-0.92 / 1.00: for the others the streaming kernel's tiles of 64 columns have the same latency
//     (0.98-1.04 / 1.13).  Four stages of 128 columns are too few.
static int few_tiles_bn(int64_t M, int64_t N, int64_t K, int act, int64_t rq_first, int sms) {
  const bool glu = act == AQT_ACT_GLU || act == AQT_ACT_GLU_SWISH;
  const bool deep = ceil_div(K, kBK) > kWsMaxKBlocks, plain = rq_first < 0;
  const int64_t tiles_m = ceil_div(M, kBM);
  if (tuning_env("AQT_NO_FEW") != nullptr) return 0;
  if (deep && plain && (!glu || M <= 64)) return 0;
  for (int bn = glu ? 64 : 32; bn <= (deep ? 64 : 128); bn *= 2) {
    const int64_t tiles_n = ceil_div(N, bn), out_cols = glu ? bn / 2 : bn;
    if (tiles_m * tiles_n > sms) continue;
    if (bn < 128 && (plain ? tiles_n > 64 : tiles_n - rq_first / out_cols > 16)) continue;
    return plain || rq_first % out_cols == 0 ? bn : 0;
  }
  return 0;
}
static size_t few_tiles_exchange_bytes(int64_t M, int64_t N, int bn) {
  return round_up((size_t)ceil_div(M, kBM) * (size_t)ceil_div(N, bn) * kBM * 8 + (size_t)kMaxGroups * 4, 256);
}

template <int BN, bool GLU, bool DEBUG>
static int launch_few_tiles_form(const int8_t* a, const void* b, float* y, int64_t ldy, FewTilesParams fp, cudaStream_t st) {
  using Cfg = FewTilesCfg<BN, GLU>;
  GemmParams& p = fp.rp.g;
  p.tiles_m = (int)ceil_div(p.M, kBM);
  p.tiles_n = (int)ceil_div(p.N, BN);
  p.k_blocks = (int)ceil_div(p.K, kBK);
  p.has_y = y != nullptr ? 1 : 0;
  const int sms = sm_count();
  if (sms <= 0) return AQT_ERR_CUDA;
  // the CTAs of an m-tile wait on one another: one CTA per SM, so that all of them are resident
  if (p.tiles_m * p.tiles_n > sms || p.tiles_m > kMaxGroups) return AQT_ERR_UNSUPPORTED;
  if (fp.b_packed && p.k_blocks > kWsMaxKBlocks) return AQT_ERR_UNSUPPORTED;
  if (fp.rq_first < p.n_out) {
    if (fp.rq_first % Cfg::kOutCols != 0) return AQT_ERR_UNSUPPORTED;
    fp.rp.tag = next_launch_tag();
  } else {
    fp.rq_first = p.tiles_n * Cfg::kOutCols;  // no tile
  }
  CUtensorMap tm_a, tm_b, tm_y, tm_r;
  int rc = make_map_2d(&tm_a, CU_TENSOR_MAP_DATA_TYPE_UINT8, a, (uint64_t)p.M, (uint64_t)p.K, (uint64_t)p.K, kBM, kBK);
  if (rc != AQT_OK) return rc;
  if (fp.b_packed) rc = make_map_2d(&tm_b, CU_TENSOR_MAP_DATA_TYPE_UINT8, b, (uint64_t)p.N, (uint64_t)p.K / 2, (uint64_t)p.K / 2, BN / 2, 64, 0);
  else rc = make_map_2d(&tm_b, CU_TENSOR_MAP_DATA_TYPE_UINT8, b, (uint64_t)p.N, (uint64_t)p.K, (uint64_t)p.K, BN / 2, kBK);
  if (rc != AQT_OK) return rc;
  tm_y = tm_a;
  tm_r = tm_a;
  if (y != nullptr) {
    rc = make_map_2d(&tm_y, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, y, (uint64_t)p.M, (uint64_t)p.n_out, (uint64_t)ldy * 4, 32, Cfg::C, 4 * Cfg::C);
    if (rc != AQT_OK) return rc;
  }
  if (p.residual != nullptr) {
    rc = make_map_2d(&tm_r, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, p.residual, (uint64_t)p.M, (uint64_t)p.n_out, (uint64_t)p.ldr * 4, 32, Cfg::C, 4 * Cfg::C);
    if (rc != AQT_OK) return rc;
  }
  auto kernel = qgemm_few_tiles_kernel<BN, GLU, DEBUG>;
  static std::atomic<uint64_t> smem_opted_in{0};
  rc = ensure_dynamic_smem(kernel, Cfg::kSmemBytes, smem_opted_in);
  if (rc != AQT_OK) return rc;
  return launch_pdl(kernel, dim3((unsigned)(p.tiles_m * p.tiles_n), 1, 1), dim3(Cfg::kThreads, 1, 1), Cfg::kSmemBytes, st, 1, tm_a, tm_b, tm_y,
                    tm_r, fp);
}

template <int BN, bool GLU>
static int launch_few_tiles_inst(const int8_t* a, const void* b, float* y, int64_t ldy, const FewTilesParams& fp, cudaStream_t st) {
  return fp.rp.g.acc_debug != nullptr ? launch_few_tiles_form<BN, GLU, true>(a, b, y, ldy, fp, st)
                                      : launch_few_tiles_form<BN, GLU, false>(a, b, y, ldy, fp, st);
}

// a: int8 [M, K]; b: int8 [N, K], or (fp.b_packed) nibbles [N, K/2]; y may be null if every column is quantized.
static int launch_few_tiles(int bn, const int8_t* a, const void* b, float* y, int64_t ldy, const FewTilesParams& fp, cudaStream_t st) {
  const int act = fp.rp.g.act;
  if (act == AQT_ACT_GLU || act == AQT_ACT_GLU_SWISH) {
    return bn == 64 ? launch_few_tiles_inst<64, true>(a, b, y, ldy, fp, st)
                    : (bn == 128 ? launch_few_tiles_inst<128, true>(a, b, y, ldy, fp, st) : AQT_ERR_UNSUPPORTED);
  }
  switch (bn) {
    case 32: return launch_few_tiles_inst<32, false>(a, b, y, ldy, fp, st);
    case 64: return launch_few_tiles_inst<64, false>(a, b, y, ldy, fp, st);
    case 128: return launch_few_tiles_inst<128, false>(a, b, y, ldy, fp, st);
    default: return AQT_ERR_UNSUPPORTED;
  }
}

}  // namespace aqt
