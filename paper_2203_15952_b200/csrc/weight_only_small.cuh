// The weight-only layer (float activations, integer weights; Section 4.1) for few rows, in one launch.
//
// The tensor-core tile of the many-row form spends such a layer on other things: a launch that writes the weights as floats,
// another one (two-term form) that splits the activations, and then one 128-row tile per column block whose K runs
// through a single CTA (23 x 2684 -> 144: 31 us; 150 x 4992 -> 1920: 60 us).  Here a CTA has 16 or 32 channels and 8 to 32
// rows; codes become bf16 in registers (exact: at most eight bits) and the rows of x become bf16 terms in shared memory, a
// chunk of K at a time with the next chunk's loads in flight: two terms (16 to 17 bits of x, more than tf32's 11) for the
// one-term form, three (all 24 bits) for the two-term form.  The products are mma.sync m16n8k16 with channels as M and rows
// as N; the warps share K, and their binary32 sums are added in order.  What bounds it is the splitting of x, which every
// channel block repeats, and that of the codes, which every row block repeats: the many-row form takes over where
// those cost more than its launches (weight_only_small_applies).
#pragma once

#include "aqt_common.cuh"
#include "qgemv_small_m.cuh"

namespace aqt {

struct WoSmallParams {
  const float* x;
  const uint8_t* w;
  const float* s_w;
  const float* bias;
  const float* residual;
  float* y;
  int64_t ldx, ldr, ldy;
  float residual_scale;
  int32_t M, N, K, act;
};

template <int NT, int TERMS>
struct WoSmallCfg {
  static constexpr int R = 8 * NT;
  static constexpr int kWarps = NT == 4 ? 16 : 8;
  static constexpr int kThreads = 32 * kWarps;
  static constexpr int kTiles = NT == 4 ? 2 : 1;    // of sixteen channels
  static constexpr int kShares = kWarps / kTiles;   // of a chunk of K
  static constexpr int kChunk = NT == 4 ? 512 : 1024;
  static constexpr int kPieces = kChunk / 64 / kShares;              // of 64 codes, per warp and chunk
  static constexpr int kVecs = R * (kChunk / 4) / kThreads;          // float4s of x per thread and chunk
  static constexpr int kPitch = 2 * kChunk + 16;                     // bytes of a row's terms: eight lanes of two rows touch all banks once
  static constexpr int kTermBytes = R * kPitch;
  static constexpr int kPartPitch = 16 * kTiles + 4;
  static constexpr int kPartBytes = kShares * R * kPartPitch * 4;
  static constexpr int kSmem = TERMS * kTermBytes > kPartBytes ? TERMS * kTermBytes : kPartBytes;  // the sums come after the terms
};

__device__ __forceinline__ void mma_bf16_16x8x16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t wo_bf16x2(float lo, float hi) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}

// Sixteen codes of one channel as they are loaded: int8 (16 bytes) or packed (8 bytes, in x and y).
template <bool PACKED, bool VEC>
__device__ __forceinline__ uint4 wo_load16(const uint8_t* row, int k, int K, bool ok) {
  uint4 v = make_uint4(0u, 0u, 0u, 0u);
  if (!ok || k >= K) return v;
  if (PACKED) {
    const uint8_t* src = row + (k >> 1);
    if (VEC) {
      const uint2 t = __ldg(reinterpret_cast<const uint2*>(src));
      v.x = t.x;
      v.y = t.y;
    } else {  // K is a multiple of four: whole 16-bit words
      const uint16_t* s = reinterpret_cast<const uint16_t*>(src);
      v.x = __ldg(s);
      if (k + 4 < K) v.x |= (uint32_t)__ldg(s + 1) << 16;
      if (k + 8 < K) v.y = __ldg(s + 2);
      if (k + 12 < K) v.y |= (uint32_t)__ldg(s + 3) << 16;
    }
  } else {
    const uint8_t* src = row + k;
    if (VEC) {
      v = __ldg(reinterpret_cast<const uint4*>(src));
    } else {
      const uint32_t* s = reinterpret_cast<const uint32_t*>(src);
      v.x = __ldg(s);
      if (k + 4 < K) v.y = __ldg(s + 1);
      if (k + 8 < K) v.z = __ldg(s + 2);
      if (k + 12 < K) v.w = __ldg(s + 3);
    }
  }
  return v;
}
// The same as bf16 pairs.  A nibble n = c + 8 in the mantissa of 128 is 128 + n, a byte u = c + 128 in that of 2^23 is 2^23 + u:
// subtracting the offset is exact.
template <bool PACKED>
__device__ __forceinline__ void wo_codes(const uint4& v, uint32_t (&o)[8]) {
  if (PACKED) {
    const uint32_t w[2] = {v.x ^ 0x88888888u, v.y ^ 0x88888888u};
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const uint32_t b = w[j >> 2] >> (8 * (j & 3));
      const uint32_t m = (b & 0x0Fu) | ((b & 0xF0u) << 12) | 0x43004300u;
      asm("sub.rn.bf16x2 %0, %1, %2;" : "=r"(o[j]) : "r"(m), "r"(0x43084308u));  // 136
    }
  } else {
    const uint32_t w[4] = {v.x ^ 0x80808080u, v.y ^ 0x80808080u, v.z ^ 0x80808080u, v.w ^ 0x80808080u};
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const uint32_t u = w[j >> 1];
      const int b = 2 * (j & 1);
      const float f0 = __uint_as_float(__byte_perm(u, 0x4B000000u, 0x7440 + b)) - 8388736.0f;
      const float f1 = __uint_as_float(__byte_perm(u, 0x4B000000u, 0x7440 + b + 1)) - 8388736.0f;
      o[j] = wo_bf16x2(f0, f1);
    }
  }
}

template <int NT, int TERMS, bool PACKED, bool GLU, bool VEC>
__global__ void __launch_bounds__(WoSmallCfg<NT, TERMS>::kThreads) weight_only_small_kernel(const WoSmallParams p) {
  using Cfg = WoSmallCfg<NT, TERMS>;
  constexpr int R = Cfg::R, T = Cfg::kTiles, KC = Cfg::kChunk;
  extern __shared__ __align__(128) uint8_t wo_smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane >> 2, kq = lane & 3;
  const int K = p.K, n_out = GLU ? p.N >> 1 : p.N;
  const int row0 = blockIdx.y * R, rows = min(R, p.M - row0);
  const int col0 = blockIdx.x * (GLU ? 8 : 16) * T;

  grid_dependency_wait();
  grid_dependents_launch();

  // ---- weights: this warp's tile of channels and share of every chunk
  const int tile = warp % T, share = warp / T;
  const int ch0 = GLU ? col0 + 8 * tile + g : col0 + 16 * tile + g, ch1 = GLU ? ch0 + n_out : ch0 + 8;
  const bool has0 = ch0 < n_out, has1 = GLU ? has0 : ch1 < n_out;
  const int64_t w_pitch = PACKED ? K >> 1 : K;
  const uint8_t* w0 = p.w + (int64_t)(has0 ? ch0 : 0) * w_pitch;
  const uint8_t* w1 = p.w + (int64_t)(has1 ? ch1 : 0) * w_pitch;
  uint4 wn[Cfg::kPieces][2];
  float4 xn[Cfg::kVecs];
  auto load_chunk = [&](int k0) {
#pragma unroll
    for (int j = 0; j < Cfg::kPieces; ++j) {
      const int k = k0 + (share * Cfg::kPieces + j) * 64 + kq * 16;
      wn[j][0] = wo_load16<PACKED, VEC>(w0, k, K, has0);
      wn[j][1] = wo_load16<PACKED, VEC>(w1, k, K, has1);
    }
#pragma unroll
    for (int i = 0; i < Cfg::kVecs; ++i) {
      const int idx = threadIdx.x + i * Cfg::kThreads, r = idx / (KC / 4), k = k0 + 4 * (idx % (KC / 4));
      xn[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (r < rows && k < K) xn[i] = __ldg(reinterpret_cast<const float4*>(p.x + (int64_t)(row0 + r) * p.ldx + k));
    }
  };
  load_chunk(0);

  // channel scales of this thread's four output columns (the same in every step of the epilogue)
  constexpr int kGroups = T * (GLU ? 2 : 4);
  const int group = threadIdx.x % kGroups;
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

  float acc[NT][4];
#pragma unroll
  for (int t = 0; t < NT; ++t)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[t][j] = 0.0f;
  for (int k0 = 0; k0 < K; k0 += KC) {
    // ---- the chunk's terms
    if (k0 > 0) __syncthreads();  // the products of the chunk before have read theirs
#pragma unroll
    for (int i = 0; i < Cfg::kVecs; ++i) {
      const int idx = threadIdx.x + i * Cfg::kThreads, r = idx / (KC / 4), c = 4 * (idx % (KC / 4));
      const float v[4] = {xn[i].x, xn[i].y, xn[i].z, xn[i].w};
      float hi[4], mid[4], lo[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const bool finite = fabsf(v[e]) <= 3.402823466e38f;  // others go whole into the first term
        hi[e] = finite ? __uint_as_float(__float_as_uint(v[e]) & 0xFFFF0000u) : v[e];
        lo[e] = finite ? v[e] - hi[e] : 0.0f;  // exact
        if (TERMS == 3) {
          mid[e] = __uint_as_float(__float_as_uint(lo[e]) & 0xFFFF0000u);
          lo[e] -= mid[e];  // exact, at most eight bits
        }
      }
      uint8_t* dst = wo_smem + r * Cfg::kPitch + 2 * c;
      *reinterpret_cast<uint2*>(dst) = make_uint2(wo_bf16x2(hi[0], hi[1]), wo_bf16x2(hi[2], hi[3]));
      if (TERMS == 3)
        *reinterpret_cast<uint2*>(dst + 2 * Cfg::kTermBytes) = make_uint2(wo_bf16x2(mid[0], mid[1]), wo_bf16x2(mid[2], mid[3]));
      *reinterpret_cast<uint2*>(dst + Cfg::kTermBytes) = make_uint2(wo_bf16x2(lo[0], lo[1]), wo_bf16x2(lo[2], lo[3]));
    }
    uint4 wc[Cfg::kPieces][2];
#pragma unroll
    for (int j = 0; j < Cfg::kPieces; ++j) {
      wc[j][0] = wn[j][0];
      wc[j][1] = wn[j][1];
    }
    if (k0 + KC < K) load_chunk(k0 + KC);
    __syncthreads();

    // ---- products
#pragma unroll
    for (int j = 0; j < Cfg::kPieces; ++j) {
      const int kc = (share * Cfg::kPieces + j) * 64;
      if (k0 + kc >= K) break;
      uint32_t c0[8], c1[8];
      wo_codes<PACKED>(wc[j][0], c0);
      wo_codes<PACKED>(wc[j][1], c1);
      const uint8_t* a = wo_smem + g * Cfg::kPitch + 2 * (kc + kq * 16);
#pragma unroll
      for (int t = 0; t < NT; ++t) {
#pragma unroll
        for (int term = TERMS - 1; term >= 0; --term) {
          const uint8_t* at = a + term * Cfg::kTermBytes + t * 8 * Cfg::kPitch;
          const uint4 x0 = *reinterpret_cast<const uint4*>(at), x1 = *reinterpret_cast<const uint4*>(at + 16);
          mma_bf16_16x8x16(acc[t], c0[0], c1[0], c0[1], c1[1], x0.x, x0.y);
          mma_bf16_16x8x16(acc[t], c0[2], c1[2], c0[3], c1[3], x0.z, x0.w);
          mma_bf16_16x8x16(acc[t], c0[4], c1[4], c0[5], c1[5], x1.x, x1.y);
          mma_bf16_16x8x16(acc[t], c0[6], c1[6], c0[7], c1[7], x1.z, x1.w);
        }
      }
    }
  }
  __syncthreads();
  float* part = reinterpret_cast<float*>(wo_smem);
  {
    float* dst = part + (share * R + 2 * kq) * Cfg::kPartPitch + 16 * tile + g;
#pragma unroll
    for (int t = 0; t < NT; ++t) {
      dst[0] = acc[t][0];
      dst[Cfg::kPartPitch] = acc[t][1];
      dst[8] = acc[t][2];
      dst[Cfg::kPartPitch + 8] = acc[t][3];
      dst += 8 * Cfg::kPartPitch;
    }
  }
  __syncthreads();

  // ---- epilogue: four output columns a thread
  if (!has_col) return;
  const int src_col = GLU ? 16 * (group >> 1) + 4 * (group & 1) : 4 * group;
  for (int r = threadIdx.x / kGroups; r < rows; r += Cfg::kThreads / kGroups) {
    auto dequant = [&](int col, const float4& w4, const float4& b4, float (&z)[4]) {
      const float* src = part + r * Cfg::kPartPitch + col;
      float4 a = *reinterpret_cast<const float4*>(src);
#pragma unroll
      for (int s = 1; s < Cfg::kShares; ++s) {
        src += R * Cfg::kPartPitch;
        const float4 q = *reinterpret_cast<const float4*>(src);
        a.x += q.x; a.y += q.y; a.z += q.z; a.w += q.w;
      }
      z[0] = __fmaf_rn(a.x, w4.x, b4.x);
      z[1] = __fmaf_rn(a.y, w4.y, b4.y);
      z[2] = __fmaf_rn(a.z, w4.z, b4.z);
      z[3] = __fmaf_rn(a.w, w4.w, b4.w);
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
      const float4 r4 = *reinterpret_cast<const float4*>(p.residual + (int64_t)(row0 + r) * p.ldr + oc);
      o[0] = __fmaf_rn(p.residual_scale, o[0], r4.x);
      o[1] = __fmaf_rn(p.residual_scale, o[1], r4.y);
      o[2] = __fmaf_rn(p.residual_scale, o[2], r4.z);
      o[3] = __fmaf_rn(p.residual_scale, o[3], r4.w);
    }
    *reinterpret_cast<float4*>(p.y + (int64_t)(row0 + r) * p.ldy + oc) = make_float4(o[0], o[1], o[2], o[3]);
  }
}

// 8-row tiles per CTA: 8, 16 or 32 rows.  16 rows come with 16 channels and so with twice the CTAs of 32 rows: where those are
// more than a wave, 32 rows (16 x 160 -> 3000: 6.2 us with 16, 3.7 with 32).
static int wo_small_row_tiles(const WoSmallParams& p) { return p.M <= 8 ? 1 : (p.M <= 16 && ceil_div(p.N, 16) <= kDefaultSms ? 2 : 4); }

// us a call, many-row form / this one: 8 x 512 -> 512 9.8 / 3.1 (two-term form 15.7 / 3.1), 23 x 2684 -> 144 30 / 16, 64 x 2496 ->
// 1920 32 / 14, 256 x 512 -> 512 10.3 / 4.7.  Up to two waves of CTAs it wins at every K (64 x 4096 -> 4096 55 / 40, 128 x 1248 ->
// 1288 17.2 / 15.4), beyond it loses (256 x 1248 -> 1288 17.5 / 22.6, 128 x 160 -> 3000 7.8 / 9.3); and up to 256 rows, from
// where it wins little (512 x 512 -> 512 9.8 / 7.7, 512 x 2048 -> 512 25 / 22).
// The two-term form up to K = 768: its many-row form's long sums lose bits that this one keeps (1e-5 of the result against
// 6e-7 at K = 2048), and the results of a layer should not move by more than 5e-6 with the number of rows.
static bool weight_only_small_applies(const WoSmallParams& p, int terms) {
  if (p.M > 256 || (terms == 3 && p.K > 768)) return false;
  const int row_tiles = wo_small_row_tiles(p);
  if (ceil_div(p.N, row_tiles == 4 ? 32 : 16) * ceil_div(p.M, 8 * row_tiles) > 2 * kDefaultSms) return false;
  // other CTAs still read x while the first ones write: not in place
  const int64_t n_out = p.act >= AQT_ACT_GLU ? p.N / 2 : p.N;
  const uintptr_t x0 = reinterpret_cast<uintptr_t>(p.x), x1 = x0 + ((size_t)(p.M - 1) * p.ldx + p.K) * 4;
  const uintptr_t y0 = reinterpret_cast<uintptr_t>(p.y), y1 = y0 + ((size_t)(p.M - 1) * p.ldy + n_out) * 4;
  return x1 <= y0 || y1 <= x0;
}

template <int NT, int TERMS, bool PACKED, bool GLU>
static int launch_weight_only_small_as(const WoSmallParams& p, cudaStream_t st) {
  using Cfg = WoSmallCfg<NT, TERMS>;
  const int n_out = GLU ? p.N / 2 : p.N;
  const dim3 grid((unsigned)ceil_div(n_out, (GLU ? 8 : 16) * Cfg::kTiles), (unsigned)ceil_div(p.M, Cfg::R), 1);
  if (p.K % 16 == 0) {
    static std::atomic<uint64_t> opted_in{0};
    const int rc = ensure_dynamic_smem(weight_only_small_kernel<NT, TERMS, PACKED, GLU, true>, Cfg::kSmem, opted_in);
    if (rc != AQT_OK) return rc;
    return launch_pdl(weight_only_small_kernel<NT, TERMS, PACKED, GLU, true>, grid, dim3(Cfg::kThreads, 1, 1), Cfg::kSmem, st, 1, p);
  }
  static std::atomic<uint64_t> opted_in{0};
  const int rc = ensure_dynamic_smem(weight_only_small_kernel<NT, TERMS, PACKED, GLU, false>, Cfg::kSmem, opted_in);
  if (rc != AQT_OK) return rc;
  return launch_pdl(weight_only_small_kernel<NT, TERMS, PACKED, GLU, false>, grid, dim3(Cfg::kThreads, 1, 1), Cfg::kSmem, st, 1, p);
}

template <int NT, int TERMS>
static int launch_weight_only_small_nt(const WoSmallParams& p, bool packed, cudaStream_t st) {
  const bool glu = p.act >= AQT_ACT_GLU;
  if (packed) return glu ? launch_weight_only_small_as<NT, TERMS, true, true>(p, st) : launch_weight_only_small_as<NT, TERMS, true, false>(p, st);
  return glu ? launch_weight_only_small_as<NT, TERMS, false, true>(p, st) : launch_weight_only_small_as<NT, TERMS, false, false>(p, st);
}

template <int TERMS>
static int launch_weight_only_small_terms(const WoSmallParams& p, bool packed, cudaStream_t st) {
  switch (wo_small_row_tiles(p)) {
    case 1: return launch_weight_only_small_nt<1, TERMS>(p, packed, st);
    case 2: return launch_weight_only_small_nt<2, TERMS>(p, packed, st);
    default: return launch_weight_only_small_nt<4, TERMS>(p, packed, st);
  }
}

static int launch_weight_only_small(const WoSmallParams& p, bool packed, int terms, cudaStream_t st) {
  return terms == 3 ? launch_weight_only_small_terms<3>(p, packed, st) : launch_weight_only_small_terms<2>(p, packed, st);
}

}  // namespace aqt
