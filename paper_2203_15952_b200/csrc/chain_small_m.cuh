// A chain of quantized layers on a few rows (a streaming step of some frames through a whole encoder)
// in one launch.
//
// What bounds such a step is not work but the number of dependent kernels: an eight-row step through
// the 17-block d = 512 encoder reads 67 MB of weights (10 us of HBM time) in 187 launches of 2 to
// 11 us each (1276 us).  Here one thread-block cluster of sixteen CTAs carries up to 16 rows through
// every layer; clusters take different rows and do not interact (rows are independent under per-row
// scales).  Within a cluster:
//   * CTA r owns 1/16 of every layer's output channels and with it 1/16 of the weights, which stream
//     from L2 / HBM into registers, one chunk (eight 16-byte loads a lane) ahead of use across layer
//     boundaries, L2 prefetches two layers ahead;
//   * every CTA holds the codes of all rows of the current activations in shared memory; the products
//     are mma.sync m16n8k32 (int8) with sixteen output channels as its M and eight activation rows as
//     its N, so that eight rows waste nothing (a tcgen05 tile would first want the weights unpacked in
//     shared memory; this part issues an m16n8k32 every sixteen clocks per scheduler, which is what the
//     feed-forward layers' products cost);
//   * the output rows are quantized for the next layer in place (Fig. 2): every warp sends the maxima of
//     its rows over the CTA's columns to all sixteen CTAs, waits for the other fifteen of each row,
//     and sends its share of the codes to all sixteen.  Nothing but requested outputs is written
//     to global memory, and the residual stream stays in shared memory with the CTA that owns its columns.
// All exchange is by asynchronous stores to distributed shared memory that complete on the receiver's
// mbarrier: a receiver waits for the bytes it needs (one one-way latency each, where cluster barriers
// cost 1000 to 1300 clocks a time with their round trip and the skew of sixteen CTAs), and a cluster is
// scheduled as a whole, so nothing has to be resident beside it.  The waits are bounded like every
// wait of the library.
// Measured, against layer by layer, both in a replayed graph: a step through 17 blocks at d = 512 8 rows 318 vs 827 us, 32 rows 322 vs
// 836, 112 rows (seven clusters of sixteen rows, all that run at once) 489 vs 866.  Beyond, a second wave of clusters: 113 rows 793 vs 866,
// 128 rows 963 vs 868, 224 rows 971 vs 871; d = 256 656 vs 673, 801 vs 669, 803 vs 687; 8 blocks at d = 1024 815 vs 575, 909 vs 575, 887
// vs 582.  So AQT_CHAIN_MAX_ROWS lies where the second wave begins.
// What a layer then costs (2000 to 2600 ns; clock stamps in a copy) is a chain of latencies and of instructions that every warp
// issues once, at the pace at which their lines are fetched:
//   * eight warps form the products and eight take the rows from there, so that the next weights are asked for while the rows
//     are de-quantized and exchanged (asking takes 1000 clocks of a layer's 5000), and the products of q and k do not wait
//     for the rows of the layer before (445 -> 383 us);
//   * what is not always run stands aside: the general code sequence in a function, the wide form's second words behind a
//     branch, the loop over pieces left at the last one (383 -> 344 us); stores of a layer's outputs wait until its maxima are on their way;
//   * layers that read the same input and look alike run as one (chain_group);
//   * no integer division and no dependent parameter load in the loops (the step table sits in shared memory with everything
//     derived from the sizes), and packed weights are used as sixteen times their codes (a nibble in the upper half of a
//     byte; the sums are shifted back, exact), two instructions per four codes instead of eleven per eight, against
//     activation codes stored in the same even / odd order.
// (One exchange of whole fp32 rows, quantized by every CTA for itself, instead of maxima and then codes: 446 -> 463 us.  Scales and
// residuals in registers ahead of the sums, with a path for unaligned ones: 383 -> 385, sixteen rows 571 -> 612.)
// The arithmetic is that of the per-layer kernels operation by operation (exact int32 sums, the same
// de-quantization, activation and quantizer), so the results are the same bits.
#pragma once

#include "aqt_common.cuh"
#include "pack.cuh"
#include "qgemv_small_m.cuh"
#include "quantize.cuh"

namespace aqt {

constexpr int kChainCtas = 16;     // CTAs of a cluster (beyond the portable eight: allowed per function)
constexpr int kChainWarps = 8;     // warps that form products, and as many that take the rows from there
constexpr int kChainRowThreads = 32 * kChainWarps;
constexpr int kChainThreads = 2 * kChainRowThreads;
constexpr int kChainChunk = 8;     // pieces (two 16-byte weight loads per lane) in flight
constexpr int kChainMaxSteps = 256;
constexpr int kChainMaxN = kChainCtas * kChainRowThreads;  // one scale per thread
constexpr int kChainMaxCols = 256;              // output columns per CTA: eight floats per lane and row

struct ChainStep {
  const uint8_t* w;   // codes [N, K] int8, or packed [N, K/2]
  const float* s_w;
  const float* bias;
  float* y;           // fp32 output [M, N_out] or null
  int32_t N, K, ldy;
  float rs;           // residual scale
  uint32_t flags;
  // derived by the host (chain_derive)
  uint16_t tiles;                // 16-channel tiles per CTA
  uint8_t ks_n;                  // shares of K
  uint8_t parts;                 // this step and those behind it that run as one (see chain_group)
  uint32_t inv_tiles;            // ceil(65536 / tiles), ceil(65536 / ks_n): quotients of small numbers by a multiply and a shift
  uint16_t inv_ks_lo, units;     // (ks_n == 1 is not divided by)
};
static_assert(sizeof(ChainStep) == 64, "copied to shared memory as 16-byte words");
enum : uint32_t {
  kChainActMask = 3u,
  kChainPacked = 4u,  // 4-bit weights, two per byte
  kChainSide = 8u,    // the output only goes to y: the next step reads the same input
  kChainAdd = 16u,    // output = residual stream + rs * act(z), and is the new residual stream
  kChainOut4 = 32u    // the next layer's input is quantized to 4 bits
};

template <int MAXS>
struct ChainParams {
  const float* x;
  int64_t ldx;
  int32_t M, K0, n_steps, rounding;
  int32_t in_qmax;     // of the first step's input
  int32_t code_bytes;  // shared memory for the activation codes
  int32_t part_bytes;  // for the partial sums
  int32_t h_cols;      // residual-stream columns per CTA (0: no step adds)
  ChainStep steps[MAXS];
};

// Activation codes: row pitch by the consumer's weight width, so that the eight lanes of a 128-bit
// shared-memory phase (two rows, four lanes each) touch all banks once: a lane reads 32 codes per
// 128 with packed weights, 16 per 64 with int8 weights.
__host__ __device__ inline int chain_pitch(int K, bool packed) { return K + (packed ? 16 : 64); }
// Tiles of sixteen channels per CTA (the last one may be half empty) and the split of K over warps.
static inline int chain_tiles(int N) { return (N / kChainCtas + 15) / 16; }
static inline int chain_ksplit(int tiles, int K) {
  if (tiles >= kChainWarps) return 1;
  const int by_warps = kChainWarps / tiles, by_k = K / 128;
  return by_warps < by_k ? by_warps : by_k;
}

__device__ __forceinline__ void mma_s8_16x8x32(int (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3])
               : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t chain_mapa(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
// Store to another CTA's shared memory that counts its bytes on that CTA's mbarrier when it lands.
__device__ __forceinline__ void chain_st_async(uint32_t addr, uint32_t v, uint32_t bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(addr), "r"(v), "r"(bar) : "memory");
}
__device__ __forceinline__ void chain_st_async_v2(uint32_t addr, uint32_t v0, uint32_t v1, uint32_t bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%1, %2}, [%3];" ::"r"(addr), "r"(v0), "r"(v1), "r"(bar)
               : "memory");
}
// Named barriers between the two halves of a block: one side arrives, the other waits.  Barrier 1 + slot: partial sums are
// there; 3 + slot: they have been read.
__device__ __forceinline__ void chain_bar_arrive(int id) { asm volatile("barrier.cta.arrive %0, %1;" ::"r"(id), "n"(kChainThreads) : "memory"); }
__device__ __forceinline__ void chain_bar_sync(int id) { asm volatile("barrier.cta.sync %0, %1;" ::"r"(id), "n"(kChainThreads) : "memory"); }
__device__ __forceinline__ void chain_cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Eight consecutive codes (two words) in the order the consumer's weights have them: as they are for
// int8 weights, the even ones and then the odd ones for packed weights.
__device__ __forceinline__ void chain_order8(bool packed, uint32_t& w0, uint32_t& w1) {
  const uint32_t even = __byte_perm(w0, w1, 0x6420), odd = __byte_perm(w0, w1, 0x7531);
  w0 = packed ? even : w0;
  w1 = packed ? odd : w1;
}

// Four codes of a row as one word: both roundings of every value and a choice, which is less code than a branch around either (the chain
// runs through it once a layer).
__device__ __forceinline__ uint32_t chain_codes4(const float (&v)[4], const ScaleCtx& c, int qmax, int rounding) {
  if (__builtin_expect(!c.fast, 0)) return codes4_general(v[0], v[1], v[2], v[3], c.s, qmax, rounding);
  const bool half_up = rounding == AQT_ROUND_HALF_UP_FLOOR;
  int q[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const float q0 = __fmul_rn(v[e], c.r), t = __fmaf_rn(__fmaf_rn(-q0, c.s, v[e]), c.r, q0);  // as quantize_fast
    q[e] = half_up ? __float2int_rd(__fadd_rn(t, 0.5f)) : __float2int_rn(t);
  }
  return pack4_i8(q[0], q[1], q[2], q[3]);
}
__device__ __forceinline__ float chain_max4(float m, const float (&v)[4]) {
  return fmaxf(m, fmaxf(fmaxf(fabsf(v[0]), fabsf(v[1])), fmaxf(fabsf(v[2]), fabsf(v[3]))));
}

// NT: 8-row tiles per cluster.  GROUPED: some steps run as one (chain_group); other chains are 2 to 5 % faster without the code for it.
template <int NT, int MAXS, bool GROUPED>
__global__ void __launch_bounds__(kChainThreads, 1) chain_small_m_kernel(const __grid_constant__ ChainParams<MAXS> p) {
  constexpr int R = 8 * NT;
  constexpr int SETS = NT == 1 ? 2 : 1;  // independent accumulators per row tile (the products of one set depend on one another)
  extern __shared__ __align__(128) uint8_t chain_smem[];
  __shared__ __align__(16) ChainStep steps[MAXS];
  __shared__ __align__(16) float sw_s[2][kChainRowThreads], bias_s[2][kChainRowThreads];
  __shared__ uint32_t amax_s[R][kChainCtas];  // bit patterns of the row maxima of every CTA's columns
  __shared__ uint64_t amax_bar[R];            // a row's sixteen maxima have arrived
  __shared__ uint64_t codes_bar;              // all codes of the next input have arrived
  __shared__ int abort_flag;
  uint8_t* codes = chain_smem;
  float* h = reinterpret_cast<float*>(chain_smem + p.code_bytes + 2 * p.part_bytes);  // [R][h_cols]

  const int lane = threadIdx.x & 31;
  const bool rows_half = threadIdx.x < kChainRowThreads;    // this warp works on rows, else on products
  const int warp = (threadIdx.x >> 5) & (kChainWarps - 1);  // of its half
  const int g = lane >> 2, kq = lane & 3;
  const int rank = (int)cluster_ctarank();
  const int row0 = (int)(blockIdx.x / kChainCtas) * R;
  const int rows = min(R, p.M - row0);
  const int n_steps = p.n_steps, rounding = p.rounding, h_cols = p.h_cols;
  const uint64_t t_start = global_timer_ns();

  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int r = 0; r < R; ++r) mbar_init(smem_u32(&amax_bar[r]), 1);
    mbar_init(smem_u32(&codes_bar), 1);
    fence_barrier_init();
  }
  for (int i = threadIdx.x; i < n_steps * 4; i += kChainThreads)
    reinterpret_cast<uint4*>(steps)[i] = reinterpret_cast<const uint4*>(p.steps)[i];
  __syncthreads();
  grid_dependency_wait();

  if (!rows_half) {
    // ---- This warp's products in program order: units (sixteen channels and a share of K), each in items of up to
    // kChainChunk pieces (16 bytes of two channels' weights per lane: 128 of K packed, 64 of K int8).  The next
    // item's pieces are in nxt (zeros beyond its end).
    int it_step = 0, it_u = warp;  // unit of the item
    int u_left = 0;                // pieces from the item to the end of the unit
    int u_a = 0, u_part = 0;       // this lane's first activation code (byte offset), first partial sum (index)
    bool u_first = true, u_both = true;  // the unit's first item; its upper eight channels exist
    const uint8_t *u_src0 = nullptr, *u_src1 = nullptr;
    uint4 nxt[kChainChunk][2];
    auto open_unit = [&]() {  // the iterator's unit, or the first one of a later step
      while (it_step < n_steps && it_u >= steps[it_step].units) {
        it_step += GROUPED ? steps[it_step].parts : 1;
        it_u = warp;
      }
      u_left = 0;
      if (it_step >= n_steps) return;
      const ChainStep& st = steps[it_step];
      const int k128 = st.K >> 7, per_part = st.N >> 4, per_cta = GROUPED ? per_part * st.parts : per_part;
      const int shift = (st.flags & kChainPacked) ? 1 : 0;
      int tile = it_u, kb0 = 0, kb1 = k128, ks = 0;  // tiles fastest, then shares of K
      if (st.ks_n > 1) {
        ks = (int)((uint32_t)it_u * st.inv_tiles >> 16);
        tile = it_u - ks * st.tiles;
        kb0 = (int)((uint32_t)(ks * k128) * st.inv_ks_lo >> 16);
        kb1 = (int)((uint32_t)((ks + 1) * k128) * st.inv_ks_lo >> 16);
      }
      const int c0 = tile * 16 + g;  // this lane's channels among the CTA's: c0 and c0 + 8
      u_both = tile * 16 + 8 < per_cta;
      const int c1 = u_both ? c0 + 8 : c0;
      const uint8_t *w0 = st.w, *w1 = st.w;
      int n0 = rank * per_part + c0, n1 = rank * per_part + c1;
      if (GROUPED && st.parts > 1) {  // eight channels are of one part
        for (int i = 1; i < st.parts; ++i) {
          if (c0 >= i * per_part) {
            n0 -= per_part;
            w0 = steps[it_step + i].w;
          }
          if (c1 >= i * per_part) {
            n1 -= per_part;
            w1 = steps[it_step + i].w;
          }
        }
      }
      if ((st.flags & kChainActMask) >= AQT_ACT_GLU) {  // value channels, then the gate channels of the same output columns
        const int cols = per_cta >> 1, gate_off = (st.N >> 1) - cols;
        n0 = rank * cols + c0 + (c0 >= cols ? gate_off : 0);
        n1 = rank * cols + c1 + (c1 >= cols ? gate_off : 0);
      }
      u_left = (kb1 - kb0) << (1 - shift);
      const int k_off = (kb0 << (7 - shift)) + kq * 16;
      u_src0 = w0 + (int64_t)n0 * (st.K >> shift) + k_off;
      u_src1 = w1 + (int64_t)n1 * (st.K >> shift) + k_off;
      u_a = g * chain_pitch(st.K, shift != 0) + kb0 * 128 + kq * (16 << shift);
      u_part = (ks * R + 2 * kq) * (per_cta + 4) + c0;
      u_first = true;
    };
    auto load_piece = [&](int j) {
      nxt[j][0] = nxt[j][1] = make_uint4(0u, 0u, 0u, 0u);
      if (j < u_left) {
        nxt[j][0] = __ldg(reinterpret_cast<const uint4*>(u_src0 + j * 64));
        nxt[j][1] = __ldg(reinterpret_cast<const uint4*>(u_src1 + j * 64));
      }
    };
    auto prefetch_slice = [&](int s) {  // one step's share of the weights -> L2
      if (threadIdx.x != kChainThreads - 1 || s >= n_steps || blockIdx.x >= kChainCtas) return;
      const ChainStep& st = steps[s];
      const bool glu = (st.flags & kChainActMask) >= AQT_ACT_GLU;
      const int row_bytes = (st.flags & kChainPacked) ? st.K >> 1 : st.K, rows_here = st.N >> (glu ? 5 : 4);
      const uint8_t* src = st.w + (int64_t)rank * rows_here * row_bytes;
      for (int gate = 0; gate <= (glu ? 1 : 0); ++gate, src += (int64_t)(st.N >> 1) * row_bytes)
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"((uint32_t)(rows_here * row_bytes)) : "memory");
    };

    auto prefetch_group = [&](int s) {
      for (int i = 0; s < n_steps && i < (GROUPED ? steps[s].parts : 1); ++i) prefetch_slice(s + i);
    };

    open_unit();
#pragma unroll
    for (int j = 0; j < kChainChunk; ++j) load_piece(j);
    prefetch_group(GROUPED ? steps[0].parts : 1);
    chain_cluster_sync();  // the input's codes are ready; every CTA's barriers exist

    uint32_t codes_parity = 0;  // of the codes that the next step with a new input reads
    bool fresh = false;         // the codes of this step's input come from the exchange before it
    for (int s = 0, round = 0, parts; s < n_steps; s += parts, ++round) {
      const ChainStep& st = steps[s];
      parts = GROUPED ? st.parts : 1;
      const bool packed = (st.flags & kChainPacked) != 0;
      const int units = st.units, pitch = chain_pitch(st.K, packed), part_pitch = (st.N >> 4) * parts + 4, slot = round & 1;
      int* part = reinterpret_cast<int*>(chain_smem + p.code_bytes + slot * p.part_bytes);
      if (fresh) {
        mbar_wait(smem_u32(&codes_bar), codes_parity, &abort_flag, t_start);
        codes_parity ^= 1u;
      }
      if (round >= 2) chain_bar_sync(3 + slot);  // the sums of two rounds ago have been read
      bool used = false;
      int acc[NT][SETS][4];
      while (it_step == s) {
        const int n = u_left, part0 = u_part;
        const bool both = u_both;
        const uint8_t* a0 = codes + u_a;
        if (u_first) {
#pragma unroll
          for (int t = 0; t < NT; ++t)
#pragma unroll
            for (int j = 0; j < 4 * SETS; ++j) acc[t][j >> 2][j & 3] = 0;
        }
        // the next item: loaded piece by piece below if it belongs to this step, else while the maxima are under way
        bool more = true;
        if (n > kChainChunk) {
          u_left -= kChainChunk;
          u_src0 += kChainChunk * 64;
          u_src1 += kChainChunk * 64;
          u_a += kChainChunk * (packed ? 128 : 64);
          u_first = false;
        } else {
          it_u += kChainWarps;
          more = it_u < units;
          if (more) open_unit();
          else used = true;
        }
#pragma unroll
        for (int jj = 0; jj < kChainChunk; jj += 2) {
          if (jj >= n && !more) break;
          if (jj < n) {
#pragma unroll
            for (int j = jj; j < jj + 2; ++j) {
              const uint4 w0 = nxt[j][0], w1 = nxt[j][1];
              if (packed) {
                // sixteen times the codes: the even ones' nibbles moved up, the odd ones' in place
                constexpr uint32_t kHigh = 0xF0F0F0F0u;
                const uint32_t e[8] = {(w0.x << 4) & kHigh, (w1.x << 4) & kHigh, (w0.y << 4) & kHigh, (w1.y << 4) & kHigh,
                                       (w0.z << 4) & kHigh, (w1.z << 4) & kHigh, (w0.w << 4) & kHigh, (w1.w << 4) & kHigh};
                const uint32_t o[8] = {w0.x & kHigh, w1.x & kHigh, w0.y & kHigh, w1.y & kHigh, w0.z & kHigh, w1.z & kHigh, w0.w & kHigh, w1.w & kHigh};
#pragma unroll
                for (int t = 0; t < NT; ++t) {
                  const uint8_t* a = a0 + t * 8 * pitch + j * 128;
                  const uint4 x0 = *reinterpret_cast<const uint4*>(a), x1 = *reinterpret_cast<const uint4*>(a + 16);
                  mma_s8_16x8x32(acc[t][0], e[0], e[1], o[0], o[1], x0.x, x0.y);
                  mma_s8_16x8x32(acc[t][SETS - 1], e[2], e[3], o[2], o[3], x0.z, x0.w);
                  mma_s8_16x8x32(acc[t][0], e[4], e[5], o[4], o[5], x1.x, x1.y);
                  mma_s8_16x8x32(acc[t][SETS - 1], e[6], e[7], o[6], o[7], x1.z, x1.w);
                }
              } else {
#pragma unroll
                for (int t = 0; t < NT; ++t) {
                  const uint4 x0 = *reinterpret_cast<const uint4*>(a0 + t * 8 * pitch + j * 64);
                  mma_s8_16x8x32(acc[t][0], w0.x, w1.x, w0.y, w1.y, x0.x, x0.y);
                  mma_s8_16x8x32(acc[t][SETS - 1], w0.z, w1.z, w0.w, w1.w, x0.z, x0.w);
                }
              }
            }
          }
          if (more) {
            load_piece(jj);
            load_piece(jj + 1);
          }
        }
        if (n <= kChainChunk) {  // the unit's last item
          const int shift = packed ? 4 : 0;
#pragma unroll
          for (int t = 0; t < NT; ++t) {
            int* dst = part + part0 + 8 * t * part_pitch;
            if (SETS == 2) {
#pragma unroll
              for (int j = 0; j < 4; ++j) acc[t][0][j] += acc[t][SETS - 1][j];
            }
            dst[0] = acc[t][0][0] >> shift;
            dst[part_pitch] = acc[t][0][1] >> shift;
            if (both) {
              dst[8] = acc[t][0][2] >> shift;
              dst[part_pitch + 8] = acc[t][0][3] >> shift;
            }
          }
        }
        if (!more) break;
      }
      chain_bar_arrive(1 + slot);
      // the next step's weights are asked for while the rows of this one are worked on
      if (used) {
        open_unit();
#pragma unroll
        for (int j = 0; j < kChainChunk; ++j) load_piece(j);
      }
      const int s1 = s + parts;
      prefetch_group(s1 < n_steps && GROUPED ? s1 + steps[s1].parts : s1 + 1);
      fresh = (steps[s1 - 1].flags & kChainSide) == 0;
    }
  } else {
    auto load_scales = [&](int s, float& wv, float& bv) {  // this thread's channel of step s
      wv = bv = 0.0f;
      if (s >= n_steps) return;
      const ChainStep& st = steps[s];
      const int per_part = st.N >> 4, per_cta = GROUPED ? per_part * st.parts : per_part, c = threadIdx.x;
      if (c - lane >= per_cta || c >= per_cta) return;
      int n = rank * per_part + c, of = s;
      if ((st.flags & kChainActMask) >= AQT_ACT_GLU) {
        const int cols = per_cta >> 1, gate = c >= cols ? 1 : 0;
        n = gate * (st.N >> 1) + rank * cols + c - gate * cols;
      } else if (GROUPED) {
        for (int i = 1; i < st.parts && c >= i * per_part; ++i) {
          n -= per_part;
          ++of;
        }
      }
      wv = __ldg(steps[of].s_w + n);
      if (steps[of].bias != nullptr) bv = __ldg(steps[of].bias + n);
    };
    float wv, bv;  // scale and bias of this thread's channel of the next step, on their way to sw_s / bias_s
    load_scales(0, wv, bv);

    // ---- the input: every CTA quantizes all rows for itself and keeps its columns of the residual stream
    float sx[NT];  // input scales of this warp's rows (warp, warp + 8, ...)
    {
      const int pitch = chain_pitch(p.K0, (steps[0].flags & kChainPacked) != 0);
#pragma unroll
      for (int t = 0; t < NT; ++t) {
        const int r = warp + 8 * t;
        sx[t] = 0.0f;
        if (r >= rows) continue;
        const float4* xr = reinterpret_cast<const float4*>(p.x + (int64_t)(row0 + r) * p.ldx);
        float amax = 0.0f;
        for (int c = lane; c < p.K0 / 4; c += 32) {
          const float4 f = __ldg(xr + c);
          const float v[4] = {f.x, f.y, f.z, f.w};
          amax = chain_max4(amax, v);
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, off));
        const ScaleCtx sc = make_scale_ctx_zeros(amax, p.in_qmax);
        sx[t] = sc.s;
        for (int c = lane; c < p.K0 / 8; c += 32) {
          const float4 f0 = __ldg(xr + 2 * c), f1 = __ldg(xr + 2 * c + 1);
          const float v0[4] = {f0.x, f0.y, f0.z, f0.w}, v1[4] = {f1.x, f1.y, f1.z, f1.w};
          uint32_t w0 = chain_codes4(v0, sc, p.in_qmax, rounding), w1 = chain_codes4(v1, sc, p.in_qmax, rounding);
          chain_order8((steps[0].flags & kChainPacked) != 0, w0, w1);
          *reinterpret_cast<uint2*>(codes + r * pitch + 8 * c) = make_uint2(w0, w1);
        }
        for (int c = lane; c < h_cols / 4; c += 32)
          *reinterpret_cast<float4*>(h + r * h_cols + 4 * c) = __ldg(xr + rank * (h_cols / 4) + c);
      }
    }
    chain_cluster_sync();  // own codes ready; every CTA's barriers exist

    // lane l sends its warp's row maxima to CTA l of the cluster
    const uint32_t to_amax = chain_mapa(smem_u32(&amax_s[0][rank]), lane & 15), to_amax_bar = chain_mapa(smem_u32(&amax_bar[0]), lane & 15);
    // the CTAs' windows of the cluster's shared memory lie at equal distances
    const uint32_t codes_first = chain_mapa(smem_u32(codes), 0), codes_bar_first = chain_mapa(smem_u32(&codes_bar), 0);
    const uint32_t window = chain_mapa(smem_u32(codes), 1) - codes_first;
    uint32_t exchange_parity = 0;  // of the exchange in progress (steps that are no side steps)
    for (int s = 0, round = 0; s < n_steps; s += GROUPED ? steps[s].parts : 1, ++round) {
      const ChainStep st = steps[s];
      const int parts = GROUPED ? st.parts : 1;
      const uint32_t act = st.flags & kChainActMask, end_flags = GROUPED ? steps[s + parts - 1].flags : st.flags;
      const bool glu = act >= AQT_ACT_GLU;
      const int per_part = st.N >> 4, per_cta = per_part * parts, ks_n = st.ks_n;
      const int cols = glu ? per_cta >> 1 : per_cta;  // output columns of this CTA
      const int n_out = glu ? st.N >> 1 : st.N;
      const int part_pitch = per_cta + 4;
      const int q0 = (parts - 1) * per_part, q_cols = cols - q0;  // the columns that the next step reads
      const int s1 = s + parts, s2 = s1 < n_steps && GROUPED ? s1 + steps[s1].parts : s1 + 1;
      const bool side = (end_flags & kChainSide) != 0, last = s1 == n_steps;
      const int slot = round & 1;  // of the partial sums and of sw_s / bias_s
      const int* part = reinterpret_cast<const int*>(chain_smem + p.code_bytes + slot * p.part_bytes);
      sw_s[slot][threadIdx.x] = wv;
      bias_s[slot][threadIdx.x] = bv;
      chain_bar_sync(1 + slot);

      // ---- epilogue: warp w owns rows w, w + 8, ..., a lane four consecutive columns at a time
      float v[NT][2][4];
#pragma unroll
      for (int t = 0; t < NT; ++t) {
        float amax = 0.0f;
        const int r = warp + 8 * t;
        if (r >= rows) continue;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const int c = 4 * lane + 128 * j;
#pragma unroll
          for (int e = 0; e < 4; ++e) v[t][j][e] = 0.0f;
          if (j > 0 && __builtin_expect(cols <= 128, 1)) break;
          if (c >= cols) continue;
          auto dequant = [&](int cc, float (&z)[4]) {
            const int* src = part + r * part_pitch + cc;
            int4 a = *reinterpret_cast<const int4*>(src);
#pragma unroll 1
            for (int ks = 1; ks < ks_n; ks += 3) {  // three loads at a time, not one behind the other
              int4 q[3];
#pragma unroll
              for (int i = 0; i < 3; ++i) {
                q[i] = make_int4(0, 0, 0, 0);
                src += R * part_pitch;
                if (ks + i < ks_n) q[i] = *reinterpret_cast<const int4*>(src);
              }
              a.x += q[0].x + q[1].x + q[2].x;
              a.y += q[0].y + q[1].y + q[2].y;
              a.z += q[0].z + q[1].z + q[2].z;
              a.w += q[0].w + q[1].w + q[2].w;
            }
            const float4 w4 = *reinterpret_cast<const float4*>(&sw_s[slot][cc]);
            const float4 b4 = *reinterpret_cast<const float4*>(&bias_s[slot][cc]);
            z[0] = __fmaf_rn(__fmul_rn(__int2float_rn(a.x), sx[t]), w4.x, b4.x);
            z[1] = __fmaf_rn(__fmul_rn(__int2float_rn(a.y), sx[t]), w4.y, b4.y);
            z[2] = __fmaf_rn(__fmul_rn(__int2float_rn(a.z), sx[t]), w4.z, b4.z);
            z[3] = __fmaf_rn(__fmul_rn(__int2float_rn(a.w), sx[t]), w4.w, b4.w);
          };
          float (&o)[4] = v[t][j];
          dequant(c, o);
          if (glu) {
            float zg[4];
            dequant(cols + c, zg);
#pragma unroll
            for (int e = 0; e < 4; ++e) o[e] = __fmul_rn(o[e], small_sigmoid(zg[e]));
          }
          if (act == AQT_ACT_SWISH || act == AQT_ACT_GLU_SWISH) {
#pragma unroll
            for (int e = 0; e < 4; ++e) o[e] = __fmul_rn(o[e], small_sigmoid(o[e]));
          }
          if (st.flags & kChainAdd) {
            const float4 r4 = *reinterpret_cast<const float4*>(h + r * h_cols + c);
            o[0] = __fmaf_rn(st.rs, o[0], r4.x);
            o[1] = __fmaf_rn(st.rs, o[1], r4.y);
            o[2] = __fmaf_rn(st.rs, o[2], r4.z);
            o[3] = __fmaf_rn(st.rs, o[3], r4.w);
          }
          if (!GROUPED || c >= q0) amax = chain_max4(amax, o);
        }
        if (side || last) continue;
        const uint32_t m = __reduce_max_sync(0xffffffffu, __float_as_uint(amax));  // non-negative floats order like their bit patterns
        if (lane < kChainCtas) chain_st_async(to_amax + r * (kChainCtas * 4), m, to_amax_bar + r * 8);
        if (lane == 0) mbar_arrive_expect_tx(smem_u32(&amax_bar[r]), kChainCtas * 4);
      }
      // what else is to be done, while the maxima are under way
      if (threadIdx.x == 0 && !side && !last) mbar_arrive_expect_tx(smem_u32(&codes_bar), (uint32_t)(rows * n_out));
      if ((st.flags & kChainAdd) || st.y != nullptr || (GROUPED && parts > 1)) {
#pragma unroll
        for (int t = 0; t < NT; ++t)
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            const int r = warp + 8 * t, c = 4 * lane + 128 * j;
            if (r >= rows || c >= cols) continue;
            const float4 o = make_float4(v[t][j][0], v[t][j][1], v[t][j][2], v[t][j][3]);
            if (st.flags & kChainAdd) *reinterpret_cast<float4*>(h + r * h_cols + c) = o;
            if (!GROUPED || parts == 1) {
              if (st.y != nullptr) *reinterpret_cast<float4*>(st.y + (int64_t)(row0 + r) * st.ldy + rank * cols + c) = o;
            } else {
              int of = s, first = 0;
              while (c >= first + per_part) {
                first += per_part;
                ++of;
              }
              if (steps[of].y != nullptr) *reinterpret_cast<float4*>(steps[of].y + (int64_t)(row0 + r) * steps[of].ldy + rank * per_part + c - first) = o;
            }
          }
      }
      if (s2 < n_steps) chain_bar_arrive(3 + slot);
      if (last) break;

      load_scales(s1, wv, bv);  // while the maxima are under way
      if (side) continue;

      // ---- quantize the output rows for the next step.  All sixteen maxima of a row are here only when every
      // CTA has finished its products, so nobody reads the old codes any more.
      const int qmax = (end_flags & kChainOut4) ? 7 : 127;
      const bool next_packed = (steps[s1].flags & kChainPacked) != 0;
      const int out_pitch = chain_pitch(n_out, next_packed);
#pragma unroll
      for (int t = 0; t < NT; ++t) {
        const int r = warp + 8 * t;
        if (r >= rows) continue;
        mbar_wait(smem_u32(&amax_bar[r]), exchange_parity, &abort_flag, t_start);
        const uint32_t m = __reduce_max_sync(0xffffffffu, amax_s[r][lane & (kChainCtas - 1)]);
        const ScaleCtx sc = make_scale_ctx_zeros(__uint_as_float(m), qmax);
        sx[t] = sc.s;
        uint32_t word[2] = {0u, 0u};
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          if (j > 0 && __builtin_expect(cols <= 128, 1)) break;
          if (4 * lane + 128 * j >= cols || (GROUPED && 4 * lane + 128 * j < q0)) continue;
          word[j] = chain_codes4(v[t][j], sc, qmax, rounding);
        }
        // to all sixteen CTAs, eight codes per lane and store: `span` lanes (a power of two) cover the row's share,
        // so a store instruction is 32 / span runs of consecutive bytes (the interconnect is paid per run: 250 clocks
        // for a store scattered over sixteen CTAs)
        const int span_bits = q_cols <= 16 ? 1 : 32 - __clz((q_cols >> 3) - 1), span = 1 << span_bits, i = lane & (span - 1);
        uint32_t w0, w1;
        if (__builtin_expect(q_cols <= 128, 1)) {
          const int from = GROUPED ? q0 >> 2 : 0;  // first lane with columns of the last part
          w0 = __shfl_sync(0xffffffffu, word[0], (from + 2 * i) & 31);
          w1 = __shfl_sync(0xffffffffu, word[0], (from + 2 * i + 1) & 31);
        } else {  // columns from 128 on sit in the lanes' second word
          const uint32_t x0 = __shfl_sync(0xffffffffu, word[0], (2 * i) & 31), x1 = __shfl_sync(0xffffffffu, word[0], (2 * i + 1) & 31);
          const uint32_t y0 = __shfl_sync(0xffffffffu, word[1], (2 * i) & 31), y1 = __shfl_sync(0xffffffffu, word[1], (2 * i + 1) & 31);
          w0 = i < 16 ? x0 : y0;
          w1 = i < 16 ? x1 : y1;
        }
        chain_order8(next_packed, w0, w1);
        const uint32_t dst = codes_first + (uint32_t)(r * out_pitch + rank * q_cols + 8 * i);
        for (int to = lane >> span_bits; to < kChainCtas; to += 32 >> span_bits) {
          const uint32_t at = ((uint32_t)(rank + to) & (kChainCtas - 1)) * window;
          if (8 * i < q_cols) chain_st_async_v2(dst + at, w0, w1, codes_bar_first + at);
        }
      }
      exchange_parity ^= 1u;
    }
  }
  grid_dependents_launch();
  chain_cluster_sync();  // no CTA leaves while its shared memory may still be written
}

// ------------------------------------------------------------------------------------------------
// Host side

// True if the chain kernel can run this step at all.
static bool chain_step_ok(const ChainStep& st) {
  const bool glu = (st.flags & kChainActMask) >= AQT_ACT_GLU;
  const int n_out = glu ? st.N / 2 : st.N;
  if (st.N % (8 * kChainCtas) != 0 || n_out % (8 * kChainCtas) != 0 || st.K % 128 != 0) return false;
  return st.N <= kChainMaxN && n_out <= kChainMaxCols * kChainCtas && st.K <= 8192;
}

// Steps that run as one: side steps and the one behind them that read the same input and look alike (the attention projections).
// Their channels make up a CTA's tiles together, their rows go through one epilogue (of at most 128 columns: of more, a step is
// long enough by itself), and the last one's columns are exchanged.  Eight rows through 17 blocks in a replayed graph, without and with
// it: d = 512 342 -> 318 us, 384 312 -> 291, 256 277 -> 254.
static int chain_group(const ChainStep* steps, int n) {
  const ChainStep& a = steps[0];
  int parts = 1;
  while (parts < n && (steps[parts - 1].flags & kChainSide)) {
    const ChainStep& b = steps[parts];
    if (b.N != a.N || b.K != a.K || ((a.flags ^ b.flags) & (kChainActMask | kChainPacked)) || ((a.flags | b.flags) & kChainAdd)) return 1;
    ++parts;
  }
  const bool takes = (a.flags & kChainActMask) == AQT_ACT_NONE && parts * (a.N / kChainCtas) <= 128 && !(steps[parts - 1].flags & kChainSide);
  return takes ? parts : 1;
}

// Fills in what is derived of the next group of steps; returns how many they are.
static int chain_derive(ChainStep* steps, int n) {
  ChainStep& st = steps[0];
  st.parts = (uint8_t)chain_group(steps, n);
  st.tiles = (uint16_t)chain_tiles(st.N * st.parts);
  st.ks_n = (uint8_t)chain_ksplit(st.tiles, st.K);
  st.inv_tiles = (65536u + st.tiles - 1) / st.tiles;  // exact: dividends < 16 * 64, divisors <= 16
  st.inv_ks_lo = (uint16_t)((65536u + st.ks_n - 1) / st.ks_n);
  st.units = (uint16_t)(st.tiles * st.ks_n);
  return st.parts;
}

struct ChainSizes {
  int code_bytes, part_bytes, h_bytes;
  int smem(void) const { return code_bytes + 2 * part_bytes + h_bytes; }
};
static ChainSizes chain_sizes(const ChainStep* steps, int n, int R) {
  int code = 0, part = 0, h = 0;
  for (int i = 0; i < n; i += steps[i].parts) {
    const ChainStep& st = steps[i];
    const int c = R * (st.K + 64), q = st.ks_n * R * (st.N * st.parts / kChainCtas + 4) * 4;
    if (c > code) code = c;
    if (q > part) part = q;
    if ((st.flags & kChainAdd) && R * (st.N / kChainCtas) * 4 > h) h = R * (st.N / kChainCtas) * 4;
  }
  ChainSizes z;
  z.code_bytes = (int)round_up(code, 128);
  z.part_bytes = (int)round_up(part, 128);
  z.h_bytes = (int)round_up(h, 128);
  return z;
}

constexpr int kChainMaxSmem = 180 * 1024;  // beside the step table and the exchange words

// Clusters that run at the same time (the part schedules seven or eight of sixteen CTAs each).
constexpr int kChainClusters = 7;

template <int NT, int MAXS, bool GROUPED>
static int launch_chain_form(const ChainParams<kChainMaxSteps>& full, int smem, cudaStream_t st) {
  ChainParams<MAXS> p;
  memcpy(static_cast<void*>(&p), &full, offsetof(ChainParams<MAXS>, steps) + (size_t)full.n_steps * sizeof(ChainStep));
  auto kernel = chain_small_m_kernel<NT, MAXS, GROUPED>;
  static std::atomic<uint64_t> opted_in{0}, wide{0};
  int rc = ensure_dynamic_smem(kernel, kChainMaxSmem, opted_in);
  if (rc != AQT_OK) return rc;
  rc = ensure_wide_clusters(kernel, wide);
  if (rc != AQT_OK) return rc;
  const unsigned clusters = (unsigned)ceil_div(full.M, 8 * NT);
  return launch_pdl(kernel, dim3(clusters * kChainCtas, 1, 1), dim3(kChainThreads, 1, 1), (size_t)smem, st, kChainCtas, p);
}
template <int NT, int MAXS>
static int launch_chain_inst(const ChainParams<kChainMaxSteps>& p, int smem, cudaStream_t st) {
  bool grouped = false;
  for (int i = 0; i < p.n_steps; i += p.steps[i].parts) grouped = grouped || p.steps[i].parts > 1;
  return grouped ? launch_chain_form<NT, MAXS, true>(p, smem, st) : launch_chain_form<NT, MAXS, false>(p, smem, st);
}
template <int NT>
static int launch_chain_rows(ChainParams<kChainMaxSteps>& p, cudaStream_t st) {
  const ChainSizes z = chain_sizes(p.steps, p.n_steps, 8 * NT);
  if (z.smem() > kChainMaxSmem) return AQT_ERR_UNSUPPORTED;
  p.code_bytes = z.code_bytes;
  p.part_bytes = z.part_bytes;
  return p.n_steps <= 16 ? launch_chain_inst<NT, 16>(p, z.smem(), st) : launch_chain_inst<NT, kChainMaxSteps>(p, z.smem(), st);
}

// p: everything but the shared-memory sizes.  AQT_ERR_UNSUPPORTED if the kernel cannot take the chain.
static int launch_chain(ChainParams<kChainMaxSteps>& p, cudaStream_t st) {
  if (p.M <= 0 || p.n_steps <= 0 || p.n_steps > kChainMaxSteps) return AQT_ERR_UNSUPPORTED;
  for (int i = 0; i < p.n_steps;) i += chain_derive(p.steps + i, p.n_steps - i);
  // the fewest rows per cluster with which all clusters run at once
  if (p.M <= 8 * kChainClusters) return launch_chain_rows<1>(p, st);
  return launch_chain_rows<2>(p, st);
}

}  // namespace aqt
