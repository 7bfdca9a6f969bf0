// The whole quantized layer for a few rows of float activations in one launch (Fig. 2 on the rows, then Section 2.2).
//
// What bounds such a layer is its chain of dependent steps: two kernels one after the other, each of which does little
// more than start, wait for its first loads and drain (quantizer 2.2 - 3.4 us, product 4.8 - 5.7 us).  Here every
// CTA quantizes all rows for itself, which costs the grid x x bytes in reads from L2 and each SM the conversion of all of
// x, while its share of the weights is on the way from memory, so the form ends where that conversion costs
// more than the launch it saves (linear_small_applies).
// A CTA has eight warps (sixteen beyond 8 rows) and 16, 32 or 64 output channels; the warps cut the channels in tiles of sixteen and K in shares.
// The products are mma.sync m16n8k32 (int8) with channels as M and rows as N, as in the chain kernel, whose order of the
// codes in shared memory and use of packed weights (sixteen times their codes, shifted back) it shares.  For the GLU
// forms a tile is eight value channels over their eight gates.  Sums are exact and every float operation is that of
// the two-kernel form, so the results are the same bits.
#pragma once

#include <type_traits>

#include "aqt_common.cuh"
#include "chain_small_m.cuh"
#include "quantize.cuh"

namespace aqt {

constexpr int kLinSmallMaxRows = 64;
constexpr int kLinSmallMaxSmem = 160 * 1024;  // 64 rows of 512 codes and 16 shares of their sums: 127 KB

struct LinSmallParams {
  const float* x;
  const uint8_t* w;
  const float* s_w;
  const float* bias;
  const float* residual;
  float* y;
  int64_t ldx, ldr, ldy;
  float residual_scale;
  int32_t M, N, K, act, qmax, rounding;
  int32_t whole_tensor;  // one activation scale
  int32_t log_tiles;     // tiles of sixteen channels per CTA: 1, 2 or 4
  int32_t code_bytes;
};

// NT: 8-row tiles (all rows are in every CTA).
template <int NT>
struct LinSmallCfg {
  static constexpr int R = 8 * NT;
  static constexpr int kWarps = NT == 1 ? 8 : 16;
  static constexpr int kThreads = 32 * kWarps;
  static constexpr int kRows = R / kWarps;        // rows that a warp quantizes
  static constexpr int kVecs = kRows >= 4 ? 1 : 4 / kRows;  // 32-byte loads of each in flight
  static constexpr int kChunk = NT == 1 ? 8 : 4;  // pieces of weights (two 16-byte loads a lane) in flight
};

template <int NT, bool PACKED, bool GLU>
__global__ void __launch_bounds__(LinSmallCfg<NT>::kThreads) linear_small_kernel(const LinSmallParams p) {
  using Cfg = LinSmallCfg<NT>;
  constexpr int R = Cfg::R, RW = Cfg::kRows, U = Cfg::kVecs, W = Cfg::kWarps, kThreads = Cfg::kThreads, kChunk = Cfg::kChunk;
  constexpr int SETS = NT == 1 ? 2 : 1;
  constexpr int kPieceK = PACKED ? 128 : 64;
  extern __shared__ __align__(128) uint8_t lin_smem[];
  __shared__ float warp_max[W];
  __shared__ float sx_s[R];
  uint8_t* codes = lin_smem;
  int* part = reinterpret_cast<int*>(lin_smem + p.code_bytes);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane >> 2, kq = lane & 3;
  const int log_tiles = p.log_tiles, tiles = 1 << log_tiles;
  const int K = p.K, rows = p.M, n_out = GLU ? p.N >> 1 : p.N;
  const int pieces = (K + kPieceK - 1) / kPieceK, shares = min(W >> log_tiles, pieces), pitch = chain_pitch(pieces * kPieceK, PACKED);
  const int col0 = blockIdx.x * (GLU ? 8 : 16) << log_tiles;  // first output column of the CTA

  grid_dependency_wait();
  grid_dependents_launch();

  // ---- weights: this warp's tile and share of K
  const int tile = warp & (tiles - 1), share = warp >> log_tiles;
  const int ch0 = GLU ? col0 + 8 * tile + g : col0 + 16 * tile + g, ch1 = GLU ? ch0 + n_out : ch0 + 8;
  const bool has0 = ch0 < n_out, has1 = GLU ? has0 : ch1 < n_out;
  const int p0 = share * pieces / shares, p1 = share < shares ? (share + 1) * pieces / shares : p0;
  const int64_t w_pitch = PACKED ? K >> 1 : K;
  const uint8_t* w0 = p.w + (int64_t)ch0 * w_pitch + kq * 16;
  const uint8_t* w1 = p.w + (int64_t)ch1 * w_pitch + kq * 16;
  uint4 wreg[kChunk][2];
  auto load_piece = [&](int j, int piece) {
    const bool in = piece < p1 && piece * kPieceK + kq * (PACKED ? 32 : 16) < K;
    wreg[j][0] = in && has0 ? __ldg(reinterpret_cast<const uint4*>(w0 + piece * 64)) : make_uint4(0u, 0u, 0u, 0u);
    wreg[j][1] = in && has1 ? __ldg(reinterpret_cast<const uint4*>(w1 + piece * 64)) : make_uint4(0u, 0u, 0u, 0u);
  };
#pragma unroll
  for (int j = 0; j < kChunk; ++j) load_piece(j, p0 + j);

  // channel scales of this thread's four output columns (the same in every step of the epilogue)
  const int log_groups = log_tiles + (GLU ? 1 : 2), group = threadIdx.x & ((1 << log_groups) - 1);
  const int oc = col0 + 4 * group;  // output column
  const bool has_col = oc < n_out;
  float4 sw = make_float4(0.f, 0.f, 0.f, 0.f), b = sw, sw_g = sw, b_g = sw;
  if (has_col) {
    sw = __ldg(reinterpret_cast<const float4*>(p.s_w + oc));
    if (p.bias != nullptr) b = __ldg(reinterpret_cast<const float4*>(p.bias + oc));
    if (GLU) {
      sw_g = __ldg(reinterpret_cast<const float4*>(p.s_w + n_out + oc));
      if (p.bias != nullptr) b_g = __ldg(reinterpret_cast<const float4*>(p.bias + n_out + oc));
    }
  }

  // ---- codes of all rows: warp w has rows w, w + W, ...; a lane eight columns at a time
  const int K8 = K >> 3;
  {
    float4 f[RW][U][2];
    auto load = [&](int c0) {
#pragma unroll
      for (int t = 0; t < RW; ++t) {
        const int r = warp + W * t;
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int c = c0 + 32 * u + lane;
          f[t][u][0] = f[t][u][1] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (r < rows && c < K8) {
            const float4* src = reinterpret_cast<const float4*>(p.x + (int64_t)r * p.ldx) + 2 * c;
            f[t][u][0] = __ldg(src);
            f[t][u][1] = __ldg(src + 1);
          }
        }
      }
    };
    float amax[RW];
#pragma unroll
    for (int t = 0; t < RW; ++t) amax[t] = 0.0f;
    for (int c0 = 0; c0 < K8; c0 += 32 * U) {
      load(c0);
#pragma unroll
      for (int t = 0; t < RW; ++t)
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const float v[4] = {f[t][u][h].x, f[t][u][h].y, f[t][u][h].z, f[t][u][h].w};
            amax[t] = chain_max4(amax[t], v);
          }
    }
    if (p.whole_tensor) {
      float m = amax[0];
#pragma unroll
      for (int t = 1; t < RW; ++t) m = fmaxf(m, amax[t]);
      m = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(m)));  // non-negative floats order like their bit patterns
      if (lane == 0) warp_max[warp] = m;
      __syncthreads();
#pragma unroll
      for (int w = 0; w < W; ++w) m = fmaxf(m, warp_max[w]);
#pragma unroll
      for (int t = 0; t < RW; ++t) amax[t] = m;
    } else {
#pragma unroll
      for (int t = 0; t < RW; ++t) amax[t] = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(amax[t])));
    }
    ScaleCtx sc[RW];
#pragma unroll
    for (int t = 0; t < RW; ++t) {
      sc[t] = make_scale_ctx_zeros(amax[t], p.qmax);
      if (lane == 0) sx_s[warp + W * t] = sc[t].s;
    }
    const bool again = K8 > 32 * U;  // the loads above were more than the registers hold: once more, from L1
    // A loop for each rounding, and one for rows whose scale is not fast.  With a call of the general sequence, and a branch around either
    // rounding, for each word the loads of a step are not all in flight at once: 16 x 4096 -> 512 11.2 us, 10.15 so; 4 x 512 -> 2048, one
    // step, 2.86 and 2.77.  (The general sequence inline and both roundings of every value: 10.03, at 9 to 16 rows beyond K = 1024 1 to 4 %
    // faster, and 3.11.)
    constexpr int kGeneral = -1;
    const auto convert = [&](auto mode) {
      for (int c0 = 0; c0 < pieces * (kPieceK / 8); c0 += 32 * U) {
        if (again) load(c0);
#pragma unroll
        for (int t = 0; t < RW; ++t) {
          const int r = warp + W * t;
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const int c = c0 + 32 * u + lane;
            if (r < rows && c < pieces * (kPieceK / 8)) {
              const float v0[4] = {f[t][u][0].x, f[t][u][0].y, f[t][u][0].z, f[t][u][0].w};
              const float v1[4] = {f[t][u][1].x, f[t][u][1].y, f[t][u][1].z, f[t][u][1].w};
              uint32_t q0 = 0u, q1 = 0u;
              if (c < K8) {
                if constexpr (decltype(mode)::value == kGeneral) {
                  q0 = chain_codes4(v0, sc[t], p.qmax, p.rounding);
                  q1 = chain_codes4(v1, sc[t], p.qmax, p.rounding);
                } else {
                  const auto code = [&](float x) { return quantize_fast<decltype(mode)::value>(x, sc[t].s, sc[t].r); };
                  q0 = pack4_i8(code(v0[0]), code(v0[1]), code(v0[2]), code(v0[3]));
                  q1 = pack4_i8(code(v1[0]), code(v1[1]), code(v1[2]), code(v1[3]));
                }
                chain_order8(PACKED, q0, q1);
              }
              *reinterpret_cast<uint2*>(codes + r * pitch + 8 * c) = make_uint2(q0, q1);
            }
          }
        }
      }
    };
    bool fast = true;
#pragma unroll
    for (int t = 0; t < RW; ++t) fast = fast && sc[t].fast;
    if (__builtin_expect(!fast, 0)) convert(std::integral_constant<int, kGeneral>{});
    else if (p.rounding == AQT_ROUND_HALF_UP_FLOOR) convert(std::integral_constant<int, AQT_ROUND_HALF_UP_FLOOR>{});
    else convert(std::integral_constant<int, AQT_ROUND_NEAREST_EVEN>{});
  }
  __syncthreads();

  // ---- integer products
  int acc[NT][SETS][4];
#pragma unroll
  for (int t = 0; t < NT; ++t)
#pragma unroll
    for (int j = 0; j < 4 * SETS; ++j) acc[t][j >> 2][j & 3] = 0;
  const uint8_t* a0 = codes + g * pitch + kq * (PACKED ? 32 : 16);
  for (int base = p0; base < p1; base += kChunk) {
#pragma unroll
    for (int j = 0; j < kChunk; ++j) {
      if (base + j >= p1) break;
      const uint4 v0 = wreg[j][0], v1 = wreg[j][1];
      const uint8_t* a = a0 + (base + j) * kPieceK;
      if (PACKED) {
        constexpr uint32_t kHigh = 0xF0F0F0F0u;
        const uint32_t e[8] = {(v0.x << 4) & kHigh, (v1.x << 4) & kHigh, (v0.y << 4) & kHigh, (v1.y << 4) & kHigh,
                               (v0.z << 4) & kHigh, (v1.z << 4) & kHigh, (v0.w << 4) & kHigh, (v1.w << 4) & kHigh};
        const uint32_t o[8] = {v0.x & kHigh, v1.x & kHigh, v0.y & kHigh, v1.y & kHigh, v0.z & kHigh, v1.z & kHigh, v0.w & kHigh, v1.w & kHigh};
#pragma unroll
        for (int t = 0; t < NT; ++t) {
          const uint4 x0 = *reinterpret_cast<const uint4*>(a + t * 8 * pitch), x1 = *reinterpret_cast<const uint4*>(a + t * 8 * pitch + 16);
          mma_s8_16x8x32(acc[t][0], e[0], e[1], o[0], o[1], x0.x, x0.y);
          mma_s8_16x8x32(acc[t][SETS - 1], e[2], e[3], o[2], o[3], x0.z, x0.w);
          mma_s8_16x8x32(acc[t][0], e[4], e[5], o[4], o[5], x1.x, x1.y);
          mma_s8_16x8x32(acc[t][SETS - 1], e[6], e[7], o[6], o[7], x1.z, x1.w);
        }
      } else {
#pragma unroll
        for (int t = 0; t < NT; ++t) {
          const uint4 x0 = *reinterpret_cast<const uint4*>(a + t * 8 * pitch);
          mma_s8_16x8x32(acc[t][0], v0.x, v1.x, v0.y, v1.y, x0.x, x0.y);
          mma_s8_16x8x32(acc[t][SETS - 1], v0.z, v1.z, v0.w, v1.w, x0.z, x0.w);
        }
      }
      load_piece(j, base + j + kChunk);
    }
  }
  const int part_pitch = (16 << log_tiles) + 4;
  if (share < shares) {
    constexpr int shift = PACKED ? 4 : 0;
    int* dst = part + (share * R + 2 * kq) * part_pitch + 16 * tile + g;
#pragma unroll
    for (int t = 0; t < NT; ++t) {
      if (SETS == 2) {
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[t][0][j] += acc[t][SETS - 1][j];
      }
      dst[0] = acc[t][0][0] >> shift;
      dst[part_pitch] = acc[t][0][1] >> shift;
      dst[8] = acc[t][0][2] >> shift;
      dst[part_pitch + 8] = acc[t][0][3] >> shift;
      dst += 8 * part_pitch;
    }
  }
  __syncthreads();

  // ---- epilogue: four output columns a thread
  if (!has_col) return;
  const int src_col = GLU ? 16 * (group >> 1) + 4 * (group & 1) : 4 * group;
  for (int r = threadIdx.x >> log_groups; r < rows; r += kThreads >> log_groups) {
    const float sx = sx_s[r];
    auto dequant = [&](int col, const float4& w4, const float4& b4, float (&z)[4]) {
      const int* src = part + r * part_pitch + col;
      int4 a = *reinterpret_cast<const int4*>(src);
      for (int s = 1; s < shares; ++s) {
        src += R * part_pitch;
        const int4 q = *reinterpret_cast<const int4*>(src);
        a.x += q.x; a.y += q.y; a.z += q.z; a.w += q.w;
      }
      z[0] = __fmaf_rn(__fmul_rn(__int2float_rn(a.x), sx), w4.x, b4.x);
      z[1] = __fmaf_rn(__fmul_rn(__int2float_rn(a.y), sx), w4.y, b4.y);
      z[2] = __fmaf_rn(__fmul_rn(__int2float_rn(a.z), sx), w4.z, b4.z);
      z[3] = __fmaf_rn(__fmul_rn(__int2float_rn(a.w), sx), w4.w, b4.w);
    };
    float o[4];
    dequant(src_col, sw, b, o);
    if (GLU) {
      float zg[4];
      dequant(src_col + 8, sw_g, b_g, zg);
#pragma unroll
      for (int e = 0; e < 4; ++e) o[e] = __fmul_rn(o[e], small_sigmoid(zg[e]));
    }
    if (p.act == AQT_ACT_SWISH || p.act == AQT_ACT_GLU_SWISH) {
#pragma unroll
      for (int e = 0; e < 4; ++e) o[e] = __fmul_rn(o[e], small_sigmoid(o[e]));
    }
    if (p.residual != nullptr) {
      const float4 r4 = *reinterpret_cast<const float4*>(p.residual + (int64_t)r * p.ldr + oc);
      o[0] = __fmaf_rn(p.residual_scale, o[0], r4.x);
      o[1] = __fmaf_rn(p.residual_scale, o[1], r4.y);
      o[2] = __fmaf_rn(p.residual_scale, o[2], r4.z);
      o[3] = __fmaf_rn(p.residual_scale, o[3], r4.w);
    }
    *reinterpret_cast<float4*>(p.y + (int64_t)r * p.ldy + oc) = make_float4(o[0], o[1], o[2], o[3]);
  }
}

static int lin_small_row_tiles(int M) { return M <= 8 ? 1 : (M <= 16 ? 2 : (M <= 32 ? 4 : 8)); }
// 16, 32 or 64 channels per CTA, so that one wave of CTAs has them all (a second wave would convert x once more: 8 x 1024
// -> 4096 4.4 us with 32, 7.5 with 16); -1 beyond
static int lin_small_log_tiles(int N) {
  const int64_t tiles = ceil_div(N, 16);
  return tiles <= kDefaultSms ? 0 : (tiles <= 2 * kDefaultSms ? 1 : (tiles <= 4 * kDefaultSms ? 2 : -1));
}

// us a call, two kernels / this one (8-bit weights, one scale a row): 8 x 1024 -> 4096 8.4 / 5.2, 16 x 2048 -> 512 10.3 / 6.4,
// 64 x 512 -> 512 8.1 / 6.9, 32 x 1024 -> 1024 8.3 / 6.5; beyond 32 K elements the tensor-core tile of the two-kernel form
// wins (32 x 2048 -> 512 8.5 / 10.2, 64 x 1024 -> 1024 8.2 / 11.1), but not over its few-row form, which ends at 16
// rows (16 x 4096 -> 1024 15.4 / 10.5).  More than 48 rows on 2 M weights or more beyond K = 256 go to the two kernels too
// (64 x 512 -> 8192 7.7 / 8.1, with a gate 7.7 / 8.5; 64 x 512 -> 4096 7.4 / 7.5; 48 x 512 -> 8192 7.4 / 7.4).  A call by
// itself is bound by the host, which is what these figures have in them; replayed from a graph, where launches cost
// less, two kernels win at 1 to 8 rows from K = 2560 on too (1 x 4096 -> 32 6.6 / 7.8, by itself 8.2 / 7.6).
static bool linear_small_applies(const LinSmallParams& p, bool packed) {
  if (p.M > kLinSmallMaxRows || p.K % (packed ? 32 : 16) != 0 || !is_aligned(p.x, 16) || p.ldx % 4 != 0) return false;
  if (lin_small_log_tiles(p.N) < 0) return false;
  // every CTA reads x while others already write: not in place
  const int64_t n_out = p.act >= AQT_ACT_GLU ? p.N / 2 : p.N;
  const uintptr_t x0 = reinterpret_cast<uintptr_t>(p.x), x1 = x0 + ((size_t)(p.M - 1) * p.ldx + p.K) * 4;
  const uintptr_t y0 = reinterpret_cast<uintptr_t>(p.y), y1 = y0 + ((size_t)(p.M - 1) * p.ldy + n_out) * 4;
  if (x0 < y1 && y0 < x1) return false;
  if (p.M > 48 && p.K > 256 && (int64_t)p.N * p.K >= (2 << 20)) return false;
  const int row_tiles = lin_small_row_tiles(p.M);
  return 8ll * row_tiles * p.K <= (row_tiles <= 2 ? 65536 : 32768);
}

template <int NT>
static int launch_linear_small_nt(LinSmallParams p, bool packed, cudaStream_t st) {
  const bool glu = p.act >= AQT_ACT_GLU;
  p.log_tiles = lin_small_log_tiles(p.N);
  const int piece = packed ? 128 : 64;
  p.code_bytes = (int)round_up((size_t)8 * NT * chain_pitch((int)round_up((size_t)p.K, piece), packed), 16);
  const size_t smem = (size_t)p.code_bytes + (size_t)(LinSmallCfg<NT>::kWarps >> p.log_tiles) * 8 * NT * ((16 << p.log_tiles) + 4) * 4;
  if (smem > (size_t)kLinSmallMaxSmem) return AQT_ERR_UNSUPPORTED;
  const unsigned grid = (unsigned)ceil_div(glu ? p.N / 2 : p.N, (glu ? 8 : 16) << p.log_tiles);
#define AQT_LIN_SMALL(PK, GL)                                                                                                 \
  do {                                                                                                                        \
    static std::atomic<uint64_t> opted_in{0};                                                                                 \
    const int rc = ensure_dynamic_smem(linear_small_kernel<NT, PK, GL>, kLinSmallMaxSmem, opted_in);                          \
    if (rc != AQT_OK) return rc;                                                                                              \
    return launch_pdl(linear_small_kernel<NT, PK, GL>, dim3(grid, 1, 1), dim3(LinSmallCfg<NT>::kThreads, 1, 1), smem, st, 1, p);       \
  } while (0)
  if (packed) {
    if (glu) AQT_LIN_SMALL(true, true);
    AQT_LIN_SMALL(true, false);
  }
  if (glu) AQT_LIN_SMALL(false, true);
  AQT_LIN_SMALL(false, false);
#undef AQT_LIN_SMALL
}

static int launch_linear_small(const LinSmallParams& p, bool packed, cudaStream_t st) {
  switch (lin_small_row_tiles(p.M)) {
    case 1: return launch_linear_small_nt<1>(p, packed, st);
    case 2: return launch_linear_small_nt<2>(p, packed, st);
    case 4: return launch_linear_small_nt<4>(p, packed, st);
    default: return launch_linear_small_nt<8>(p, packed, st);
  }
}

}  // namespace aqt
