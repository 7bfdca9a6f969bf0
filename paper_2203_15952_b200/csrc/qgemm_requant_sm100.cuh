// Integer GEMM whose epilogue quantizes its own output for the next layer (sm_100a).
//
//   acc = xq * wq^T (int32, TMEM);  u = residual + residual_scale * act(fma(float(acc) * s_x, s_w, bias))
//   amax[m] = max_n |u[m][n]|;  s_out[m] = amax[m] / qmax;  q_out[m][n] = round(u[m][n] / s_out[m])
//
// i.e. the dynamic quantizer of Fig. 2 of the paper applied to the layer's output rows before they
// ever leave the SM: the fp32 tensor between two quantized layers is neither written nor read
// back (it is written too only when the caller asks for it, e.g. for a residual stream).
//
// A row's abs-max spans all N output columns, i.e. several CTAs.  The grid is made of groups of
// tiles_n CTAs; the CTAs of a group own the n-tiles of the same m-tile at about the same time
// (weight stationary, K <= 512 or 1024: each keeps its weight slab resident) and exchange row maxima
// through global memory, one 64-bit word per (m-tile, n-tile, row): the maximum's bit pattern below a
// tag that identifies this execution, so a word is its own validity and nothing is cleared,
// counted or fenced.
//   epilogue warps    four sets of four warps (one warp per TMEM lane quadrant).  In a CTA with
//                     many tiles set s owns accumulator buffer s and every fourth tile, all 128
//                     columns of it; a CTA with one or two may put several sets on each
//                     (sets_per_tile), which then take chunks of its columns and merge their maxima:
//                       pass 1  accumulators -> u (registers) -> row maxima; u goes back into the
//                               TMEM columns it came from; the maxima are published
//                       wait    for the group's other CTAs (the exchange warps do the polling)
//                       pass 2  scale from the final maximum, u from TMEM, codes, stores; the TMEM
//                               buffer goes back to the MMA
//                     With many tiles the four warps on a scheduler thus sit in four different
//                     phases of four different tiles, which is what keeps the special-function unit (pass 1 of a
//                     Swish tile) and the other pipes (pass 2) busy at the same time.
//   exchange warps    two, one per half of the rows: for each tile in turn read the words of all
//                     n-tiles (all requests in flight together), again until every one is valid,
//                     and leave the final maximum of each row in shared memory
// All CTAs of a group must be resident at once (they wait on one another): the grid never exceeds
// one CTA per SM.  Every wait is bounded as in the plain GEMM.
#pragma once

#include "qgemm_sm100.cuh"
#include "row_quant_epilogue.cuh"

namespace aqt {

struct RequantParams {
  GemmParams g;         // act: NONE or SWISH
  uint8_t* q_out;       // codes of the output: int8 [M, N] or packed nibbles [M, N/2], dense
  float* s_out;         // [M] scales of the output rows
  uint64_t* exchange;   // [tiles_m][tiles_n][128] words: (launch tag << 32) | bit pattern of a CTA's row maximum
  uint32_t* generation; // [groups] counters (generation_counters): each group of CTAs bumps its own when it has finished
  uint32_t tag;         // tag of this call (no other call of the process uses it); a word counts once its upper half
                        // equals this tag mixed with the group's generation, which differs on every execution of the call
  int qmax_out;         // 127 or 7
  int rounding;
  int pack_out;         // 1: two 4-bit codes per byte
  int one_tile_sets;    // sets of epilogue warps on the tile of a CTA that has one (sets_per_tile)
};

// DEEP: the resident weight slab holds eight k-blocks (K <= 1024, the d = 1024 encoder's first
// FFN layers and pointwise 1) instead of four.  That leaves no room for the fp32 staging buffers
// or for the packed weights, so this form writes codes and scales only and reads int8 weights
// (4-bit ones are sign-extended into the workspace beforehand).
constexpr int kRequantDeepKBlocks = 8;
template <bool WITH_Y, bool DEEP = false>
struct RequantCfg {
  static_assert(!(DEEP && WITH_Y), "the deep-K form has no room for fp32 staging");
  static constexpr int kKBlocks = DEEP ? kRequantDeepKBlocks : kWsMaxKBlocks;
  static constexpr int BN = 128;
  static constexpr int EW = 16;
  static constexpr int kThreads = 32 * (2 + EW + 2);  // producer, MMA issuer, epilogue warps, two exchange warps
  static constexpr int kStages = (WITH_Y || DEEP) ? 5 : 7;
  static constexpr int kABytes = kBM * kBK;
  static constexpr int kBBytes = BN * kBK;
  static constexpr int kResidentBytes = kKBlocks * kBBytes;
  static constexpr int kYBytes = WITH_Y ? EW * kStageBufBytes : 0;
  static constexpr int kPackedBBytes = DEEP ? 0 : kWsMaxKBlocks * BN * 64;  // packed weights wait here for the unpack
  static constexpr int kEpiBytes = kYBytes > kPackedBBytes ? kYBytes : kPackedBBytes;
  static constexpr int kScaleBytes = 2 * BN * 4;
  static constexpr int kTmemCols = 4 * BN;
  static constexpr int kSmemBytes = kStages * kABytes + kResidentBytes + kEpiBytes + kScaleBytes + 1024;
  static_assert(kSmemBytes + 13312 <= 232448, "must fit the 227 KB a CTA can opt into");
};

// 32 lanes x 16 consecutive 32-bit columns (the GLU form: a warp owns 16 value and 16 gate columns).
__device__ __forceinline__ void tmem_ld_32x16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_st_32x16(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]),
      "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}
// One slot of shared-memory exchange state (final row maxima, hand-over barriers) per accumulator
// buffer, i.e. per set of epilogue warps: tile i of a CTA uses buffer and slot i mod 4.
constexpr int kSlots = 4;

// Sets of epilogue warps that share a tile, for a CTA that has n_my of them.  With four tiles or more each set works on one
// of its own, in another phase than the others; with fewer, whole sets would be idle while one warp a quadrant goes through
// a tile's four chunks one after the other, with a residual a load of it from memory between any two.  Which launches:
// see launch_requant_inst.
__device__ __forceinline__ int sets_per_tile(int n_my, int one_tile_sets) { return n_my == 1 ? one_tile_sets : (n_my == 2 ? 2 : 1); }

// Tag of this execution's exchange words.  A replayed CUDA graph repeats the call's own tag, so the group's generation
// counter goes into it.  Whoever reads the counter hands the tag out (an arrival each on `bar`), and a CTA publishes nothing
// before that; the group's first CTA bumps the counter at its end, which it does not reach without words of all of them.
// (Warps that each read it for themselves alone would not all have done so by then.)  Readers are exchange warps: one here,
// both where a CTA has one tile (pair of 12 800 rows 57.7 us with one, 57.95 with two; block of 1013 rows 65.7 and 65.45).
__device__ __forceinline__ uint32_t hand_out_tag(const RequantParams& rp, int group, uint32_t* slot, uint64_t* bar) {
  const uint32_t tag = __shfl_sync(0xffffffffu, mix_tag(rp.tag, __ldcg(rp.generation + group)), 0);
  if ((threadIdx.x & 31) == 0) {
    *(volatile uint32_t*)slot = tag;
    mbar_arrive(smem_u32(bar));
  }
  return tag;
}
constexpr int kExchangeBatch = 16;  // n-tiles whose words an exchange warp asks for at once (one 16-byte load each per lane)

// Called between polls of a bounded wait: false once the CTA is aborting or the limit has passed
// (which then sets both the CTA's abort flag and the device status word).
__device__ __forceinline__ bool keep_waiting(volatile int* abort_flag, uint64_t t_start) {
  if (*abort_flag) return false;
  if (global_timer_ns() - t_start > kWaitLimitNs) {
    *abort_flag = 1;
    atomicExch(&g_device_status, AQT_ERR_TIMEOUT);
    return false;
  }
  return true;
}

// Final maxima of two rows (this lane's), the largest of what `parts` CTAs publish: one 16-byte load (two words) per part,
// kExchangeBatch of them in flight, and the whole batch again until every word carries this execution's tag.  The same
// answer in every lane of the warp: false once the CTA is aborting.
__device__ __forceinline__ bool collect_maxima(const uint64_t* xt, int parts, uint32_t tag, volatile int* abort_flag, uint64_t t_start, uint2& m2) {
  m2 = make_uint2(0u, 0u);
  for (int t0 = 0; t0 < parts; t0 += kExchangeBatch) {
    for (uint32_t spin = 1;; ++spin) {
      ulonglong2 w[kExchangeBatch];
#pragma unroll
      for (int t = 0; t < kExchangeBatch; ++t) {
        const uint64_t none = (uint64_t)tag << 32;  // a maximum of zero
        w[t] = t0 + t < parts ? ld_relaxed_gpu_2x64(xt + (size_t)(t0 + t) * kBM) : make_ulonglong2(none, none);
      }
      bool all = true;
      uint2 b2 = make_uint2(0u, 0u);
#pragma unroll
      for (int t = 0; t < kExchangeBatch; ++t) {
        all = all && (uint32_t)(w[t].x >> 32) == tag && (uint32_t)(w[t].y >> 32) == tag;
        b2.x = max(b2.x, (uint32_t)w[t].x);
        b2.y = max(b2.y, (uint32_t)w[t].y);
      }
      if (__all_sync(0xffffffffu, all)) {
        m2.x = max(m2.x, b2.x);
        m2.y = max(m2.y, b2.y);
        break;
      }
      if ((spin & 0xF) == 0 && !__all_sync(0xffffffffu, keep_waiting(abort_flag, t_start))) return false;
    }
  }
  return true;
}

// GLU: a tile's 128 weight rows are 64 value channels and their 64 gate channels; it yields 64
// output columns u = v * sigmoid(g) (then Swish for AQT_ACT_GLU_SWISH), 16 per epilogue warp.
// The GLU form writes codes and scales only (no fp32 output, no residual, no nibble packing).
// SHARED: CTAs with one or two tiles may have several sets of warps work on each (sets_per_tile).
template <bool BPACK, bool WITH_Y, int ROUNDING, bool PACK_OUT, bool GLU, bool DEEP, bool SHARED>
__global__ void __launch_bounds__(32 * 20, 1)
qgemm_requant_kernel(const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_b,
                     const __grid_constant__ CUtensorMap tm_y,
                     const __grid_constant__ CUtensorMap tm_r, const RequantParams rp) {
  using Cfg = RequantCfg<WITH_Y, DEEP>;
  constexpr int BN = Cfg::BN, EW = Cfg::EW, STAGES = Cfg::kStages, HALF = BN / 2;
  static_assert(!(DEEP && BPACK), "the deep-K form reads int8 weights");
  static_assert(!GLU || (!WITH_Y && !PACK_OUT), "the GLU form writes int8 codes and scales only");
  const GemmParams& p = rp.g;
  const int n_out = GLU ? p.N / 2 : p.N;  // output columns

  extern __shared__ uint8_t smem_raw[];
  __shared__ uint64_t full_bar[STAGES];
  __shared__ uint64_t empty_bar[STAGES];
  __shared__ uint64_t tmem_full_bar[4];
  __shared__ uint64_t tmem_empty_bar[4];
  __shared__ uint64_t res_bar[EW];    // WITH_Y: residual tile landed in a warp's fp32 staging buffer
  __shared__ uint64_t b_loaded_bar;
  __shared__ uint64_t b_ready_bar;
  __shared__ __align__(16) uint32_t row_amax[kSlots][kBM];  // final row maxima (bit patterns) of a tile awaiting pass 2
  __shared__ uint64_t ctx_ready_bar[kSlots][2];  // an exchange warp has filled its half of row_amax[.]
  __shared__ uint64_t ctx_free_bar[kSlots][2];   // the set's two warps on that half of the rows have read theirs
  __shared__ float part_amax[kSlots][kBM];       // tile shared by several sets: a set's maxima of its columns
  __shared__ uint64_t part_bar[kSlots][4];       // ... of lane quadrant q are there, by first set of the tile
  __shared__ uint64_t tag_bar;                   // tag_slot is there
  __shared__ uint32_t tag_slot;
  __shared__ uint32_t tmem_base_slot;
  __shared__ int abort_flag;

  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t smem_ring = smem_base;
  const uint32_t smem_res_b = smem_ring + STAGES * Cfg::kABytes;
  const uint32_t smem_epi = smem_res_b + Cfg::kResidentBytes;  // packed weights before the unpack, then (WITH_Y) fp32 staging
  const uint32_t smem_scale = smem_epi + Cfg::kEpiBytes;

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const uint64_t t_start = global_timer_ns();

  // this CTA's n-tile and its group's m-tiles
  const int tn = blockIdx.x % p.tiles_n;
  const int group = blockIdx.x / p.tiles_n;
  const int groups = gridDim.x / p.tiles_n;
  const int n_my = group < p.tiles_m ? (p.tiles_m - group + groups - 1) / groups : 0;
  const int split = SHARED ? sets_per_tile(n_my, rp.one_tile_sets) : 1;

  if (threadIdx.x == 0) {
    abort_flag = 0;
    tma_prefetch_desc(&tm_a);
    tma_prefetch_desc(&tm_b);
    if (WITH_Y) tma_prefetch_desc(&tm_y);
    if (WITH_Y && p.residual != nullptr) tma_prefetch_desc(&tm_r);
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(smem_u32(&full_bar[s]), 1);
      mbar_init(smem_u32(&empty_bar[s]), 1);
    }
    for (int b = 0; b < 4; ++b) {
      mbar_init(smem_u32(&tmem_full_bar[b]), 1);
      mbar_init(smem_u32(&tmem_empty_bar[b]), 4 * split);  // the warps of the sets that share the buffer's tile
    }
    for (int w = 0; w < EW; ++w) mbar_init(smem_u32(&res_bar[w]), 1);
    mbar_init(smem_u32(&b_loaded_bar), 1);
    mbar_init(smem_u32(&b_ready_bar), EW);
    mbar_init(smem_u32(&tag_bar), 1);
    for (int b = 0; b < kSlots; ++b) {
      for (int h = 0; h < 2; ++h) {
        mbar_init(smem_u32(&ctx_ready_bar[b][h]), 1);
        mbar_init(smem_u32(&ctx_free_bar[b][h]), 2 * split);
      }
      for (int q = 0; q < 4; ++q) mbar_init(smem_u32(&part_bar[b][q]), split > 1 ? split - 1 : 1);
    }
    fence_barrier_init();
    fence_proxy_async_smem();
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(&tmem_base_slot), Cfg::kTmemCols);
    tmem_relinquish();
  }
  // Everything above touched only this CTA's own state; from here on global memory is read.  The
  // weights (codes, scales, bias) may be read before the kernel ahead of this one in the stream has
  // finished if the caller says they were complete before that kernel was enqueued (static_w): the
  // weight slab then loads and unpacks while that kernel drains, and every role waits for it only
  // before its first access to anything else.
  const bool early_w = p.static_w != 0;
  if (!early_w) grid_dependency_wait();
  for (int t = threadIdx.x; t < BN; t += blockDim.x) {
    // scales and biases of the tile's weight rows: (GLU) values first, then gates
    const int n = !GLU ? tn * BN + t : (t < HALF ? tn * HALF + t : p.N / 2 + tn * HALF + (t - HALF));
    const int limit = (GLU && t < HALF) ? p.N / 2 : p.N;
    float wv = 0.0f, bv = 0.0f;
    if (n < limit) {
      wv = __ldg(p.s_w + n);
      if (p.bias != nullptr) bv = __ldg(p.bias + n);
    }
    asm volatile("st.shared.f32 [%0], %1;" ::"r"(smem_scale + t * 4), "f"(wv) : "memory");
    asm volatile("st.shared.f32 [%0], %1;" ::"r"(smem_scale + (BN + t) * 4), "f"(bv) : "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_slot;

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    if (lane == 0) {
      uint32_t it = 0;
      bool ok = true;
      {
        const int row0 = GLU ? tn * HALF : tn * BN, row1 = GLU ? p.N / 2 + tn * HALF : tn * BN + HALF;
        const uint32_t bar = smem_u32(&b_loaded_bar);
        if (BPACK) {
          mbar_arrive_expect_tx(bar, (uint32_t)p.k_blocks * BN * 64);
          for (int kb = 0; kb < p.k_blocks; ++kb) {
            tma_load_2d(smem_epi + kb * BN * 64, &tm_b, kb * 64, row0, bar);
            tma_load_2d(smem_epi + kb * BN * 64 + HALF * 64, &tm_b, kb * 64, row1, bar);
          }
        } else {
          mbar_arrive_expect_tx(bar, (uint32_t)p.k_blocks * Cfg::kBBytes);
          for (int kb = 0; kb < p.k_blocks; ++kb) {
            tma_load_2d(smem_res_b + kb * Cfg::kBBytes, &tm_b, kb * kBK, row0, bar);
            tma_load_2d(smem_res_b + kb * Cfg::kBBytes + HALF * kBK, &tm_b, kb * kBK, row1, bar);
          }
        }
      }
      if (early_w) grid_dependency_wait();  // the activation codes come from the kernel ahead
      for (int i = 0; ok && i < n_my; ++i) {
        const int tm = group + i * groups;
        for (int kb = 0; kb < p.k_blocks; ++kb, ++it) {
          const uint32_t s = it % STAGES, ph = (it / STAGES) & 1;
          if (!mbar_wait(smem_u32(&empty_bar[s]), ph ^ 1, &abort_flag, t_start)) { ok = false; break; }
          const uint32_t bar = smem_u32(&full_bar[s]);
          mbar_arrive_expect_tx(bar, Cfg::kABytes);
          tma_load_2d(smem_ring + s * Cfg::kABytes, &tm_a, kb * kBK, tm * kBM, bar);
        }
      }
      grid_dependents_launch();  // every load of this CTA has been issued: the next kernel may be scheduled behind it
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    if (lane == 0) {
      constexpr uint32_t idesc = idesc_i8(BN, kBM);
      uint32_t it = 0;
      bool ok = mbar_wait(smem_u32(BPACK ? &b_ready_bar : &b_loaded_bar), 0, &abort_flag, t_start);
      for (int i = 0; ok && i < n_my; ++i) {
        const uint32_t buf = i & 3, aph = (i >> 2) & 1;
        if (!mbar_wait(smem_u32(&tmem_empty_bar[buf]), aph ^ 1, &abort_flag, t_start)) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + buf * BN;
        for (int kb = 0; kb < p.k_blocks; ++kb, ++it) {
          const uint32_t s = it % STAGES, ph = (it / STAGES) & 1;
          if (!mbar_wait(smem_u32(&full_bar[s]), ph, &abort_flag, t_start)) { ok = false; break; }
          tc_fence_after();
          const uint64_t a_desc = smem_desc_k_major_sw128(smem_ring + s * Cfg::kABytes);
          const uint64_t b_desc = smem_desc_k_major_sw128(smem_res_b + kb * Cfg::kBBytes);
#pragma unroll
          for (int kk = 0; kk < kBK / kMmaK; ++kk) tc_mma_i8(d_tmem, a_desc + 2 * kk, b_desc + 2 * kk, idesc, (kb | kk) != 0 ? 1u : 0u);
          tc_commit(smem_u32(&empty_bar[s]));
        }
        if (ok) tc_commit(smem_u32(&tmem_full_bar[buf]));
      }
    }
  } else if (warp >= 2 + EW) {
    // ------------------------------------------------------------------ exchange warps
    // Two warps, each for one half of the tile's rows: lane l of warp h owns rows 64h + 2l and
    // 64h + 2l + 1, i.e. one 16-byte load (two words) per n-tile, kExchangeBatch of them in flight.
    const int xh = warp - (2 + EW);
    if (early_w) grid_dependency_wait();
    bool ok = true;
    if (xh == 0) hand_out_tag(rp, group, &tag_slot, &tag_bar);
    else ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&tag_bar), 0, &abort_flag, t_start)) != 0;
    __syncwarp();
    const uint32_t tag = *(volatile uint32_t*)&tag_slot;
    for (int i = 0; ok && i < n_my; ++i) {
      const int tm = group + i * groups;
      const uint32_t par = i % kSlots, ph = (i / kSlots) & 1;
      if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&ctx_free_bar[par][xh]), ph ^ 1, &abort_flag, t_start))) break;
      const uint64_t* xt = rp.exchange + (size_t)tm * p.tiles_n * kBM + 64 * xh + 2 * lane;
      uint2 m2;
      if (!collect_maxima(xt, p.tiles_n, tag, &abort_flag, t_start, m2)) break;
      // final maxima of this warp's rows for the epilogue warps
      *reinterpret_cast<uint2*>(&row_amax[par][64 * xh + 2 * lane]) = m2;
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&ctx_ready_bar[par][xh]));
    }
  } else {
    // ------------------------------------------------------------------ epilogue warps
    // Four sets of four warps, one warp of a set per TMEM lane quadrant (hence one per scheduler).
    // Unless sets share tiles (see below), set s owns accumulator buffer s and with it every fourth
    // tile of this CTA, all of its columns: pass 1 chunk by chunk, publication of the rows' maxima straight from registers
    // (a thread has seen its whole row of the tile, so nothing is merged across warps), the wait
    // for the other n-tiles' maxima, pass 2.  The four warps that share a scheduler therefore work
    // on four different tiles in four different phases: while one is on the special-function unit
    // (pass 1 of a Swish tile is bound by it), the others issue multiply-adds and byte permutes
    // (pass 2), wait for the exchange, or wait for the tensor core.
    const int ew = warp - 2;
    const int quad = warp & 3;  // TMEM lane quadrant this warp may access
    const int set = ew >> 2;
    // The tile's sets are consecutive; this one takes chunks c_begin .. c_end - 1 of it.
    const int part = SHARED ? set % split : 0;
    const int c_begin = part * (4 / split), c_end = c_begin + 4 / split;
    const int i_first = SHARED ? set / split : set, i_step = 4 / split;  // this warp's tiles of the CTA
    constexpr int CW = GLU ? 16 : 32;  // output columns per chunk; four chunks per tile
    const int row_in_tile = quad * 32 + lane;
    const uint32_t y_buf = smem_epi + ew * kStageBufBytes;
    const bool has_res = WITH_Y && p.residual != nullptr;
    const int oc0 = tn * (GLU ? HALF : BN);  // first output column of this CTA's tiles
    bool ok = true;

    if (BPACK) {
      // sign-extend the packed weights into the resident slab (layout of a swizzled int8 load)
      ok = mbar_wait(smem_u32(&b_loaded_bar), 0, &abort_flag, t_start);
      if (ok) {
        expand_packed_slab<BN, EW * 32>(smem_epi, smem_res_b, Cfg::kBBytes, p.k_blocks, ew * 32 + lane);
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&b_ready_bar));
        ok = mbar_wait(smem_u32(&b_ready_bar), 0, &abort_flag, t_start);  // staging area free for the fp32 output
      }
    }

    if (early_w) grid_dependency_wait();  // scales of the activations, residual, outputs: everything but the weights
    uint32_t res_count = 0;  // residual boxes this warp has consumed (phase of its barrier)
    if (ok && has_res && lane == 0 && i_first < n_my) {
      const int r0 = (group + i_first * groups) * kBM + quad * 32, c0 = oc0 + c_begin * CW;
      mbar_arrive_expect_tx(smem_u32(&res_bar[ew]), kStageBufBytes);
      tma_load_2d(y_buf, &tm_r, c0 < n_out ? c0 : 0, r0 < p.M ? r0 : 0, smem_u32(&res_bar[ew]));
    }
    if (ok) ok = mbar_wait(smem_u32(&tag_bar), 0, &abort_flag, t_start);
    const uint32_t tag = *(volatile uint32_t*)&tag_slot;

    const uint32_t buf = (uint32_t)i_first;  // accumulator buffer and exchange slot of this warp's tiles (i mod 4)
    const uint32_t tbase = tmem_base + buf * BN + ((uint32_t)(quad * 32) << 16);
    for (int i = i_first; ok && i < n_my; i += i_step) {
      const int tm = group + i * groups;
      const uint32_t aph = (uint32_t)(i >> 2) & 1u;
      const int row0_warp = tm * kBM + quad * 32;
      const int m = row0_warp + lane;
      const float sx = (p.s_x_kind == AQT_SCALE_ROW) ? (m < p.M ? __ldg(p.s_x + m) : 0.0f) : __ldg(p.s_x);
      if (!mbar_wait(smem_u32(&tmem_full_bar[buf]), aph, &abort_flag, t_start)) { ok = false; break; }
      tc_fence_after();

      // -------------------------------------------------------------- pass 1: u, row maxima; u back to TMEM
      float amax = 0.0f;
#pragma unroll 1
      for (int c = c_begin; c < c_end; ++c) {
        const int col = c * CW;
        const bool cols_ok = oc0 + col < n_out;  // columns beyond N contribute nothing
        const uint32_t c_sw = smem_scale + (uint32_t)col * 4, c_bias = c_sw + BN * 4;
        if constexpr (GLU) {
          // gates first: g = sigmoid(z_gate); then the values are scaled by it
          uint32_t accv[16], accg[16];
          float av[16], g[16];
          tmem_ld_32x16(tbase + HALF + col, accg);
          tmem_ld_32x16(tbase + col, accv);
          tmem_ld_wait();
          dequant_smem<kAccInt32>(accg, sx, c_sw + HALF * 4, c_bias + HALF * 4, g);
#pragma unroll
          for (int j = 0; j < 16; ++j) g[j] = sigmoid_f(g[j]);
          dequant_smem<kAccInt32>(accv, sx, c_sw, c_bias, av);
#pragma unroll
          for (int j = 0; j < 16; ++j) av[j] = av[j] * g[j];
          if (p.act == AQT_ACT_GLU_SWISH) swish(av);
          if (cols_ok) amax = chunk_max(amax, av);
#pragma unroll
          for (int j = 0; j < 16; ++j) accv[j] = __float_as_uint(av[j]);
          tmem_st_32x16(tbase + col, accv);  // u replaces the value accumulators
        } else {
          uint32_t acc[32];
          float a[32];
          tmem_ld_32x32(tbase + col, acc);
          tmem_ld_wait();
          dequant_smem<kAccInt32>(acc, sx, c_sw, c_bias, a);
          if (p.act == AQT_ACT_SWISH) swish(a);
          if (has_res) {
            if (!mbar_wait(smem_u32(&res_bar[ew]), res_count & 1u, &abort_flag, t_start)) { ok = false; break; }
            ++res_count;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const uint32_t src = y_buf + lane * 128 + ((j ^ (lane & 7)) << 4);
              float r0, r1, r2, r3;
              asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(r0), "=f"(r1), "=f"(r2), "=f"(r3) : "r"(src) : "memory");
              a[4 * j + 0] = __fmaf_rn(p.residual_scale, a[4 * j + 0], r0);
              a[4 * j + 1] = __fmaf_rn(p.residual_scale, a[4 * j + 1], r1);
              a[4 * j + 2] = __fmaf_rn(p.residual_scale, a[4 * j + 2], r2);
              a[4 * j + 3] = __fmaf_rn(p.residual_scale, a[4 * j + 3], r3);
            }
            __syncwarp();  // every lane has read its residual row before the buffer is overwritten
          }
          if (cols_ok) amax = chunk_max(amax, a);
#pragma unroll
          for (int j = 0; j < 32; ++j) acc[j] = __float_as_uint(a[j]);
          tmem_st_32x32(tbase + col, acc);  // u replaces the accumulators it was made from
          if (WITH_Y) {
            if (!has_res) {
              if (lane == 0) tma_store_wait_read<0>();  // the previous chunk's bulk store has read the buffer out
              __syncwarp();
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const uint32_t dst = y_buf + lane * 128 + ((j ^ (lane & 7)) << 4);
              asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "f"(a[4 * j]), "f"(a[4 * j + 1]), "f"(a[4 * j + 2]),
                           "f"(a[4 * j + 3])
                           : "memory");
            }
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) {
              if (cols_ok && row0_warp < p.M) tma_store_2d(&tm_y, y_buf, oc0 + col, row0_warp);
              tma_store_commit();
              const bool more_here = c + 1 < c_end;
              if (has_res && (more_here || i + i_step < n_my)) {
                // the next chunk's residual goes into the same buffer once this store has read it out
                tma_store_wait_read<0>();
                const int ncol = oc0 + (more_here ? col + CW : c_begin * CW);
                const int nr = (more_here ? tm : tm + i_step * groups) * kBM + quad * 32;
                mbar_arrive_expect_tx(smem_u32(&res_bar[ew]), kStageBufBytes);
                tma_load_2d(y_buf, &tm_r, ncol < n_out ? ncol : 0, nr < p.M ? nr : 0, smem_u32(&res_bar[ew]));
              }
            }
          }
        }
      }
      if (!ok) break;
      const bool has_nan = __any_sync(0xffffffffu, amax != amax) != 0;
      if (has_nan) {
        // the maxima of the warp's rows once more, from what pass 1 has left in tensor memory
        tmem_st_wait();
        amax = 0.0f;
#pragma unroll 1
        for (int c = c_begin; c < c_end && oc0 + c * CW < n_out; ++c) {
          uint32_t u[CW];
          if constexpr (GLU) tmem_ld_32x16(tbase + c * CW, u);
          else tmem_ld_32x32(tbase + c * CW, u);
          tmem_ld_wait();
          amax = numbers_max(amax, u);
        }
      }
      // This CTA's maxima of the tile's rows, each tagged valid: one word per row.  Of a tile that several sets share, the
      // first set's warp publishes the maximum of all parts (a CTA that shares tiles has one for every group of sets, so
      // the barrier is waited on once).
      if (SHARED && split > 1) {
        part_amax[set][row_in_tile] = amax;
        __syncwarp();
        const uint32_t bar = smem_u32(&part_bar[set - part][quad]);
        if (part != 0) {
          if (lane == 0) mbar_arrive(bar);
        } else {
          if (!mbar_wait(bar, 0, &abort_flag, t_start)) { ok = false; break; }
          for (int s = 1; s < split; ++s) amax = fmaxf(amax, part_amax[set + s][row_in_tile]);
        }
      }
      // (Where sets share tiles and y is written, a register held for the tag is one too many beside the call of the general
      // sequence, 8 bytes of spills: it is read again.)
      if (part == 0)
        st_relaxed_gpu_64(rp.exchange + ((size_t)tm * p.tiles_n + tn) * kBM + row_in_tile,
                          ((uint64_t)(SHARED && WITH_Y ? *(volatile uint32_t*)&tag_slot : tag) << 32) | __float_as_uint(amax));

      // -------------------------------------------------------------- pass 2: scale, codes
      if (!mbar_wait(smem_u32(&ctx_ready_bar[buf][quad >> 1]), aph, &abort_flag, t_start)) { ok = false; break; }
      const float amax_row = __uint_as_float(row_amax[buf][row_in_tile]);
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&ctx_free_bar[buf][quad >> 1]));
      ScaleCtx sc = make_scale_ctx_zeros(amax_row, rp.qmax_out);
      sc.fast = sc.fast && !has_nan;
      if (tn == 0 && part == 0 && m < p.M) rp.s_out[m] = sc.s;
      tmem_st_wait();  // this warp's stores of pass 1
#pragma unroll 1
      for (int c = c_begin; c < c_end; ++c) {
        const int col = c * CW;
        const int oc = oc0 + col;
        const bool cols_ok = oc < n_out;
        if constexpr (GLU) {
          uint32_t u[16], w[4];
          tmem_ld_32x16(tbase + col, u);
          tmem_ld_wait();
          if (c + 1 == c_end) {
            // the tile has been read out by this warp: the accumulator buffer goes back to the MMA
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&tmem_empty_bar[buf]));
          }
          codes_of<ROUNDING, false, 16>(u, sc, rp.qmax_out, w);
          // 16 consecutive codes of the row: one 16-byte store
          if (m < p.M && cols_ok) *reinterpret_cast<uint4*>(rp.q_out + (size_t)m * n_out + oc) = make_uint4(w[0], w[1], w[2], w[3]);
        } else {
          uint32_t u[32], w[8];
          tmem_ld_32x32(tbase + col, u);
          tmem_ld_wait();
          if (c + 1 == c_end) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&tmem_empty_bar[buf]));
          }
          codes_of<ROUNDING, PACK_OUT, 32>(u, sc, rp.qmax_out, w);
          // Each thread holds 32 consecutive codes of its row: one or two 16-byte stores, each a
          // whole 32-byte sector (or half of one for packed nibbles), straight to global memory.
          if (m < p.M && cols_ok) {
            if (PACK_OUT) {
              uint4* dst = reinterpret_cast<uint4*>(rp.q_out + (size_t)m * (p.N / 2) + oc / 2);
              *dst = make_uint4(w[0], w[1], w[2], w[3]);
            } else {
              uint4* dst = reinterpret_cast<uint4*>(rp.q_out + (size_t)m * p.N + oc);
              dst[0] = make_uint4(w[0], w[1], w[2], w[3]);
              if (oc + 16 < p.N) dst[1] = make_uint4(w[4], w[5], w[6], w[7]);
            }
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
  if (tn == 0 && threadIdx.x == 0) rp.generation[group] = __ldcg(rp.generation + group) + 1u;
}

// Bytes of the exchange area: one 64-bit word per m-tile, n-tile and row for this kernel, or per
// row (padded to the 256 rows of a pair tile) and column part for the CTA-pair kernel with the
// row-quantizing epilogue (at most one part per 64 columns, at least two), and the generation counters.
static size_t requant_exchange_bytes(int64_t M, int64_t N) {
  const size_t tiles_m = (size_t)ceil_div(M, kBM);
  const size_t ws_form = tiles_m * (size_t)ceil_div(N, 128) * kBM * 8;
  const size_t parts = (size_t)ceil_div(N, 64) < 2 ? 2 : (size_t)ceil_div(N, 64);
  const size_t pair_form = (size_t)ceil_div(M, 2 * kBM) * 2 * kBM * parts * 8;
  return round_up((ws_form > pair_form ? ws_form : pair_form) + (size_t)kMaxGroups * 4, 256);
}
// With room for the narrow tiles of qgemm_few_tiles_sm100.cuh (as many of 32 columns as there are SMs), which a call whose
// area is smaller does without.
static size_t requant_exchange_bytes_few(int64_t M, int64_t N, int sms) {
  const size_t tiles32 = (size_t)ceil_div(M, kBM) * (size_t)ceil_div(N, 32);
  const size_t few_form = round_up((tiles32 < (size_t)sms ? tiles32 : (size_t)sms) * kBM * 8 + (size_t)kMaxGroups * 4, 256), others = requant_exchange_bytes(M, N);
  return few_form > others ? few_form : others;
}

// True if this kernel takes the call: K <= 512; NONE / Swish in every form, the GLU forms when
// only int8 codes and scales are asked for (no fp32 output, hence no residual, no nibble packing).
static bool requant_applies(int64_t M, int64_t N, int64_t K, int act, bool with_y, bool pack_out, int sms) {
  if (!(M > 0 && ceil_div(N, 128) <= sms)) return false;
  const bool glu = !(act == AQT_ACT_NONE || act == AQT_ACT_SWISH);
  if (ceil_div(K, kBK) <= kWsMaxKBlocks) return !glu || (!with_y && !pack_out);
  // 512 < K <= 1024: codes and scales only
  return ceil_div(K, kBK) <= kRequantDeepKBlocks && !with_y && (!glu || !pack_out);
}

template <bool BPACK, bool WITH_Y, int ROUNDING, bool PACK_OUT, bool GLU, bool DEEP, bool SHARED>
static int launch_requant_form(const int8_t* a, const void* b, void* q_out, float* y, int64_t ldy, RequantParams rp,
                               void* exchange, cudaStream_t st) {
  using Cfg = RequantCfg<WITH_Y, DEEP>;
  GemmParams& p = rp.g;
  p.tiles_m = (int)ceil_div(p.M, kBM);
  p.tiles_n = (int)ceil_div(p.N, Cfg::BN);
  p.k_blocks = (int)ceil_div(p.K, kBK);
  const int sms = sm_count();
  if (sms <= 0) return AQT_ERR_CUDA;
  if (p.k_blocks > Cfg::kKBlocks || p.tiles_n > sms) return AQT_ERR_UNSUPPORTED;
  rp.exchange = reinterpret_cast<uint64_t*>(exchange);
  rp.tag = next_launch_tag();

  CUtensorMap tm_a, tm_b, tm_y, tm_r;
  int rc = make_map_2d(&tm_a, CU_TENSOR_MAP_DATA_TYPE_UINT8, a, (uint64_t)p.M, (uint64_t)p.K, (uint64_t)p.K, kBM, kBK);
  if (rc != AQT_OK) return rc;
  if (BPACK) rc = make_map_2d(&tm_b, CU_TENSOR_MAP_DATA_TYPE_UINT8, b, (uint64_t)p.N, (uint64_t)p.K / 2, (uint64_t)p.K / 2, Cfg::BN / 2, 64, 0);
  else rc = make_map_2d(&tm_b, CU_TENSOR_MAP_DATA_TYPE_UINT8, b, (uint64_t)p.N, (uint64_t)p.K, (uint64_t)p.K, Cfg::BN / 2, kBK);
  if (rc != AQT_OK) return rc;
  rp.q_out = reinterpret_cast<uint8_t*>(q_out);
  tm_y = tm_a;
  tm_r = tm_a;
  if (WITH_Y) {
    rc = make_map_2d(&tm_y, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, y, (uint64_t)p.M, (uint64_t)p.N, (uint64_t)ldy * 4, kStoreBoxRows, kStoreBoxCols);
    if (rc != AQT_OK) return rc;
    if (p.residual != nullptr) {
      rc = make_map_2d(&tm_r, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, p.residual, (uint64_t)p.M, (uint64_t)p.N, (uint64_t)p.ldr * 4, kStoreBoxRows,
                       kStoreBoxCols);
      if (rc != AQT_OK) return rc;
    }
  }
  auto kernel = qgemm_requant_kernel<BPACK, WITH_Y, ROUNDING, PACK_OUT, GLU, DEEP, SHARED>;
  static std::atomic<uint64_t> smem_opted_in{0};
  rc = ensure_dynamic_smem(kernel, Cfg::kSmemBytes, smem_opted_in);
  if (rc != AQT_OK) return rc;
  int groups = sms / p.tiles_n;
  if (groups > p.tiles_m) groups = p.tiles_m;
  // The CTAs of a group wait on one another, so all of them must get an SM: the grid never exceeds
  // one CTA per SM (each takes most of an SM's shared memory), and CTAs of the kernel before it in
  // the stream never wait on anything, so the SMs they hold become free.  Should another stream keep
  // SMs occupied for seconds, the bounded waits give up and report AQT_ERR_TIMEOUT.
  return launch_pdl(kernel, dim3((unsigned)(groups * p.tiles_n), 1, 1), dim3(Cfg::kThreads, 1, 1), Cfg::kSmemBytes, st, 1, tm_a, tm_b,
                    tm_y, tm_r, rp);
}

// Sets of warps share tiles where no CTA has more than two, by what the epilogue does (us a call in a replayed graph, for one /
// two / four sets on the tile of a CTA that has one, while CTAs that have two put two on each; most outputs of a tile per CTA
// do not come here but to qgemm_few_tiles_sm100.cuh):
//   codes only, no activation  not at all: 4864 x 512 -> 512 7.79 / 8.22 / 8.21, 3840 x 512 -> 1024 8.48 / 8.68 / 8.86
//   codes only, Swish          two: 1863 x 512 -> 2048 10.32 / 10.03 / 10.09, 1152 x 1024 -> 2048 9.96 / 9.56 / 9.75
//   gate forms, fp32 output    four if no CTA has two tiles, else two: residual, 4864 x 512 -> 512 11.20 / 10.55 / 10.83, packed
//                              codes, 1013 x 512 -> 512 9.23 / 8.28 / 7.82; gates, 512 x 1024 -> 2048 8.82 / 8.71 / 8.40
// (Three tiles a CTA gain nothing in any form.)
template <bool BPACK, bool WITH_Y, int ROUNDING, bool PACK_OUT, bool GLU = false, bool DEEP = false>
static int launch_requant_inst(const int8_t* a, const void* b, void* q_out, float* y, int64_t ldy, RequantParams rp, void* exchange,
                               cudaStream_t st) {
  const int sms = sm_count();
  if (sms <= 0) return AQT_ERR_CUDA;
  const int64_t groups = sms / ceil_div(rp.g.N, 128), tiles_m = ceil_div(rp.g.M, kBM);
  if (tiles_m <= 2 * groups && (WITH_Y || GLU || rp.g.act != AQT_ACT_NONE)) {
    rp.one_tile_sets = tiles_m <= groups && (WITH_Y || GLU) ? 4 : 2;
    return launch_requant_form<BPACK, WITH_Y, ROUNDING, PACK_OUT, GLU, DEEP, true>(a, b, q_out, y, ldy, rp, exchange, st);
  }
  rp.one_tile_sets = 1;
  return launch_requant_form<BPACK, WITH_Y, ROUNDING, PACK_OUT, GLU, DEEP, false>(a, b, q_out, y, ldy, rp, exchange, st);
}

// a: int8 [M, K]; b: int8 [N, K] or (b_packed) nibbles [N, K/2]; y may be null (then no fp32 output
// and no residual).  exchange: the words of requant_exchange_bytes(M, N); rp carries the counters.
static int launch_requant(const int8_t* a, const void* b, bool b_packed, void* q_out, float* y, int64_t ldy, const RequantParams& rp,
                          void* exchange, cudaStream_t st) {
  const bool glu = rp.g.act == AQT_ACT_GLU || rp.g.act == AQT_ACT_GLU_SWISH;
  if (ceil_div(rp.g.K, kBK) > kWsMaxKBlocks) {
    // deep-K form: int8 weights, codes and scales only
    if (y != nullptr || b_packed || (glu && rp.pack_out)) return AQT_ERR_UNSUPPORTED;
#define AQT_RQ_DEEP(PK, GL)                                                                                                       \
  (rp.rounding == AQT_ROUND_HALF_UP_FLOOR ? launch_requant_inst<false, false, AQT_ROUND_HALF_UP_FLOOR, PK, GL, true>(a, b, q_out, y, ldy, rp, exchange, st) \
                                          : launch_requant_inst<false, false, AQT_ROUND_NEAREST_EVEN, PK, GL, true>(a, b, q_out, y, ldy, rp, exchange, st))
    if (glu) return AQT_RQ_DEEP(false, true);
    return rp.pack_out ? AQT_RQ_DEEP(true, false) : AQT_RQ_DEEP(false, false);
#undef AQT_RQ_DEEP
  }
  if (glu) {
    if (y != nullptr || rp.pack_out) return AQT_ERR_UNSUPPORTED;
#define AQT_RQ_GLU(BP)                                                                                                            \
  (rp.rounding == AQT_ROUND_HALF_UP_FLOOR ? launch_requant_inst<BP, false, AQT_ROUND_HALF_UP_FLOOR, false, true>(a, b, q_out, y, ldy, rp, exchange, st) \
                                          : launch_requant_inst<BP, false, AQT_ROUND_NEAREST_EVEN, false, true>(a, b, q_out, y, ldy, rp, exchange, st))
    return b_packed ? AQT_RQ_GLU(true) : AQT_RQ_GLU(false);
#undef AQT_RQ_GLU
  }
#define AQT_RQ(BP, WY)                                                                                                     \
  (rp.pack_out ? (rp.rounding == AQT_ROUND_HALF_UP_FLOOR                                                                     \
                      ? launch_requant_inst<BP, WY, AQT_ROUND_HALF_UP_FLOOR, true>(a, b, q_out, y, ldy, rp, exchange, st) \
                      : launch_requant_inst<BP, WY, AQT_ROUND_NEAREST_EVEN, true>(a, b, q_out, y, ldy, rp, exchange, st)) \
               : (rp.rounding == AQT_ROUND_HALF_UP_FLOOR                                                                     \
                      ? launch_requant_inst<BP, WY, AQT_ROUND_HALF_UP_FLOOR, false>(a, b, q_out, y, ldy, rp, exchange, st) \
                      : launch_requant_inst<BP, WY, AQT_ROUND_NEAREST_EVEN, false>(a, b, q_out, y, ldy, rp, exchange, st)))
  if (y != nullptr) return b_packed ? AQT_RQ(true, true) : AQT_RQ(false, true);
  return b_packed ? AQT_RQ(true, false) : AQT_RQ(false, false);
#undef AQT_RQ
}

}  // namespace aqt
