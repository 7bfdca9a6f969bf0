// 4-bit storage kernels: two two's-complement nibbles per byte, even element in the low nibble.
// Rows are dense, so a [rows, cols] tensor with even cols is one flat stream of byte pairs.
#pragma once

#include <cuda_fp16.h>

#include "aqt_common.cuh"

namespace aqt {

// Sign-extend the low nibble of each of the four bytes of x (high nibbles must be zero):
// a set bit 3 (0x08) times 0x1E gives 0xF0 in the same byte and never carries into the next.
__device__ __forceinline__ uint32_t sext_nibbles_in_bytes(uint32_t x) { return x | ((x & 0x08080808u) * 0x1Eu); }

// Four packed bytes -> eight int8 codes in element order (two 32-bit words).
__device__ __forceinline__ void unpack_word(uint32_t w, uint32_t& out0, uint32_t& out1) {
  const uint32_t lo = sext_nibbles_in_bytes(w & 0x0F0F0F0Fu);
  const uint32_t hi = sext_nibbles_in_bytes((w >> 4) & 0x0F0F0F0Fu);
  out0 = __byte_perm(lo, hi, 0x5140);  // l0 h0 l1 h1
  out1 = __byte_perm(lo, hi, 0x7362);  // l2 h2 l3 h3
}

// Eight int8 codes (two words, element order) -> four packed bytes.
__device__ __forceinline__ uint32_t pack_words(uint32_t w0, uint32_t w1) {
  const uint32_t t0 = (w0 & 0x000F000Fu) | (((w0 >> 8) & 0x000F000Fu) << 4);  // bytes 0 and 2 hold the pairs
  const uint32_t t1 = (w1 & 0x000F000Fu) | (((w1 >> 8) & 0x000F000Fu) << 4);
  return __byte_perm(t0, t1, 0x6420);
}

// n_bytes packed bytes -> 2 * n_bytes codes.  vec path: 8 packed bytes per thread per step.
__global__ void __launch_bounds__(256) unpack_int4_kernel(const uint8_t* __restrict__ packed, int64_t n_bytes,
                                                          int8_t* __restrict__ q, bool vec) {
  grid_dependency_wait();
  grid_dependents_launch();
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (vec) {
    const int64_t n8 = n_bytes >> 3;
    const uint2* src = reinterpret_cast<const uint2*>(packed);
    uint4* dst = reinterpret_cast<uint4*>(q);
    for (int64_t i = tid; i < n8; i += stride) {
      const uint2 w = __ldg(src + i);
      uint4 o;
      unpack_word(w.x, o.x, o.y);
      unpack_word(w.y, o.z, o.w);
      dst[i] = o;
    }
    for (int64_t i = (n8 << 3) + tid; i < n_bytes; i += stride) {
      const uint32_t b = packed[i];
      q[2 * i] = (int8_t)((int)(b << 28) >> 28);
      q[2 * i + 1] = (int8_t)((int)(b << 24) >> 28);
    }
  } else {
    for (int64_t i = tid; i < n_bytes; i += stride) {
      const uint32_t b = packed[i];
      q[2 * i] = (int8_t)((int)(b << 28) >> 28);
      q[2 * i + 1] = (int8_t)((int)(b << 24) >> 28);
    }
  }
}

__global__ void __launch_bounds__(256) pack_int4_kernel(const int8_t* __restrict__ q, int64_t n_bytes,
                                                        uint8_t* __restrict__ packed, bool vec) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (vec) {
    const int64_t n8 = n_bytes >> 3;
    const uint4* src = reinterpret_cast<const uint4*>(q);
    uint2* dst = reinterpret_cast<uint2*>(packed);
    for (int64_t i = tid; i < n8; i += stride) {
      const uint4 w = __ldg(src + i);
      dst[i] = make_uint2(pack_words(w.x, w.y), pack_words(w.z, w.w));
    }
    for (int64_t i = (n8 << 3) + tid; i < n_bytes; i += stride)
      packed[i] = (uint8_t)((q[2 * i] & 0xF) | ((q[2 * i + 1] & 0xF) << 4));
  } else {
    for (int64_t i = tid; i < n_bytes; i += stride)
      packed[i] = (uint8_t)((q[2 * i] & 0xF) | ((q[2 * i + 1] & 0xF) << 4));
  }
}

// Weight codes -> binary32 values of the same integers (exact; every code has at most 7
// significant bits).  The float matmul of the weight-only layer reads these.  n codes, a multiple
// of 4: dense int8, or nibble pairs if `packed`.  Four codes per thread and step.
__global__ void __launch_bounds__(256) codes_to_float_kernel(const uint8_t* __restrict__ codes, bool packed, int64_t n,
                                                             float* __restrict__ out) {
  grid_dependency_wait();
  grid_dependents_launch();
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < (n >> 2); i += stride) {
    uint32_t w;
    if (packed) {
      uint32_t o1;
      unpack_word((uint32_t)__ldg(reinterpret_cast<const uint16_t*>(codes) + i), w, o1);
    } else {
      w = __ldg(reinterpret_cast<const uint32_t*>(codes) + i);
    }
    float4 f;
    f.x = (float)(int8_t)(w & 0xFF);
    f.y = (float)(int8_t)((w >> 8) & 0xFF);
    f.z = (float)(int8_t)((w >> 16) & 0xFF);
    f.w = (float)(int8_t)(w >> 24);
    reinterpret_cast<float4*>(out)[i] = f;
  }
}

// Two-term split of binary32 activations for the float matmul: hi = x with its lower thirteen
// fraction bits cleared (a tf32 value), lo = x - hi (exact).  Row m of the output holds
// [hi(x[m][0..K)) | lo(x[m][0..K))], so that one matmul over 2K against the weights repeated twice
// sums x . w with about twenty-one significant bits per activation.  K % 4 == 0, ldx % 4 == 0.
__global__ void __launch_bounds__(256) split_hi_lo_kernel(const float* __restrict__ x, int64_t ldx, int64_t M, int64_t K,
                                                          float* __restrict__ out) {
  grid_dependency_wait();
  grid_dependents_launch();
  const int64_t k4 = K >> 2, total = M * k4;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += stride) {
    const int64_t m = i / k4, c = i - m * k4;
    const float4 v = __ldg(reinterpret_cast<const float4*>(x + m * ldx) + c);
    float4 hi, lo;
    hi.x = __uint_as_float(__float_as_uint(v.x) & 0xFFFFE000u);
    hi.y = __uint_as_float(__float_as_uint(v.y) & 0xFFFFE000u);
    hi.z = __uint_as_float(__float_as_uint(v.z) & 0xFFFFE000u);
    hi.w = __uint_as_float(__float_as_uint(v.w) & 0xFFFFE000u);
    lo.x = __fsub_rn(v.x, hi.x);
    lo.y = __fsub_rn(v.y, hi.y);
    lo.z = __fsub_rn(v.z, hi.z);
    lo.w = __fsub_rn(v.w, hi.w);
    float4* row = reinterpret_cast<float4*>(out + m * 2 * K);
    row[c] = hi;
    row[k4 + c] = lo;
  }
}

// The weight codes as floats, each row written twice: out [rows, 2K] = [w | w].
__global__ void __launch_bounds__(256) codes_to_float_twice_kernel(const uint8_t* __restrict__ codes, bool packed, int64_t rows,
                                                                   int64_t K, float* __restrict__ out) {
  grid_dependency_wait();
  grid_dependents_launch();
  const int64_t k4 = K >> 2, total = rows * k4;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += stride) {
    const int64_t r = i / k4, c = i - r * k4;
    uint32_t w;
    if (packed) {
      uint32_t o1;
      unpack_word((uint32_t)__ldg(reinterpret_cast<const uint16_t*>(codes) + i), w, o1);
    } else {
      w = __ldg(reinterpret_cast<const uint32_t*>(codes) + i);
    }
    float4 f;
    f.x = (float)(int8_t)(w & 0xFF);
    f.y = (float)(int8_t)((w >> 8) & 0xFF);
    f.z = (float)(int8_t)((w >> 16) & 0xFF);
    f.w = (float)(int8_t)(w >> 24);
    float4* row = reinterpret_cast<float4*>(out + r * 2 * K);
    row[c] = f;
    row[k4 + c] = f;
  }
}

// Operands of the half kind of the matmul (K % 8 == 0, K <= 16 G, G 32 or 64).  Blocks 0 .. row_blocks - 1: rows of x as binary16, scaled by the
// power of two that brings a row's largest magnitude into [2^14, 2^15): the upper eleven significant bits of every value down to 2^-28 of
// the largest, cut off as the tensor core cuts tf32 operands, so that products are the same whichever of the two a tile takes
// (rounded to nearest they have half the error, and results that are 6e-4 from the tf32 form's).  inv[m]: the inverse of the scale, or -1
// for a row with values that are smaller and not zero, not finite, or near the ends of binary32's range.  G threads to a row.  The
// other blocks: the weights' codes as binary16 and as binary32, which tiles with such a row read.
template <int G>
__global__ void __launch_bounds__(256) half_operands_kernel(const float* __restrict__ x, int64_t ldx, int M, int K, __half* __restrict__ xh,
                                                            float* __restrict__ inv, int row_blocks, const uint8_t* __restrict__ codes, bool packed, int64_t n,
                                                            float* __restrict__ w_f, __half* __restrict__ w_h) {
  constexpr int VEC = 2;  // pairs of float4s held per thread
  __shared__ float warp_max[8];
  __shared__ int warp_wide[8];
  grid_dependency_wait();
  grid_dependents_launch();
  if ((int)blockIdx.x >= row_blocks) {
    const int64_t stride = (int64_t)((int)gridDim.x - row_blocks) * blockDim.x;
    for (int64_t i = (int64_t)((int)blockIdx.x - row_blocks) * blockDim.x + threadIdx.x; i < (n >> 2); i += stride) {
      uint32_t w;
      if (packed) {
        uint32_t o1;
        unpack_word((uint32_t)__ldg(reinterpret_cast<const uint16_t*>(codes) + i), w, o1);
      } else {
        w = __ldg(reinterpret_cast<const uint32_t*>(codes) + i);
      }
      const float4 f = make_float4((float)(int8_t)(w & 0xFF), (float)(int8_t)((w >> 8) & 0xFF), (float)(int8_t)((w >> 16) & 0xFF), (float)(int8_t)(w >> 24));
      reinterpret_cast<float4*>(w_f)[i] = f;
      const __half2 h[2] = {__floats2half2_rn(f.x, f.y), __floats2half2_rn(f.z, f.w)};
      reinterpret_cast<uint2*>(w_h)[i] = *reinterpret_cast<const uint2*>(h);
    }
    return;
  }
  const int t = threadIdx.x % G, r_in_cta = threadIdx.x / G, warp = threadIdx.x >> 5;
  const int m = (int)blockIdx.x * (256 / G) + r_in_cta;
  const bool live = m < M;
  const int n8 = K >> 3;
  const float4* row = reinterpret_cast<const float4*>(x + (int64_t)(live ? m : 0) * ldx);
  float4 v[VEC][2];
  float amax = 0.0f;
#pragma unroll
  for (int i = 0; i < VEC; ++i) {
    const int c = t + i * G;
    v[i][0] = v[i][1] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (live && c < n8) {
      v[i][0] = __ldg(row + 2 * c);
      v[i][1] = __ldg(row + 2 * c + 1);
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {  // NaN wins, so that a row with one is found
      const float4 f = v[i][j];
      asm("max.NaN.f32 %0, %0, %1, %2;" : "+f"(amax) : "f"(fabsf(f.x)), "f"(fabsf(f.y)));
      asm("max.NaN.f32 %0, %0, %1, %2;" : "+f"(amax) : "f"(fabsf(f.z)), "f"(fabsf(f.w)));
    }
  }
  uint32_t bits = __reduce_max_sync(0xffffffffu, __float_as_uint(amax) & 0x7FFFFFFFu);  // non-negative floats order like their bit patterns
  if (G > 32) {
    if ((threadIdx.x & 31) == 0) warp_max[warp] = __uint_as_float(bits);
    __syncthreads();
#pragma unroll
    for (int w = 0; w < G / 32; ++w) bits = max(bits, __float_as_uint(warp_max[r_in_cta * (G / 32) + w]));
  }
  // 2^(14 - exponent of the largest); rows of zeros: 1
  const int e = (int)(bits >> 23);  // biased
  const bool in_range = bits == 0 || (e >= 27 && e <= 227);
  const float scale = bits == 0 || !in_range ? 1.0f : __uint_as_float((uint32_t)(127 + 14 + 127 - e) << 23);
  bool wide = !in_range;
#pragma unroll
  for (int i = 0; i < VEC; ++i) {
    const int c = t + i * G;
    if (c >= n8 || !live) continue;
    uint32_t h[4];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const float u[4] = {v[i][j].x, v[i][j].y, v[i][j].z, v[i][j].w};
      const float f[4] = {u[0] * scale, u[1] * scale, u[2] * scale, u[3] * scale};
#pragma unroll
      for (int k = 0; k < 4; ++k) wide = wide || (fabsf(f[k]) < 6.103515625e-05f && u[k] != 0.0f);  // (f itself may have become zero)
      asm("cvt.rz.f16x2.f32 %0, %1, %2;" : "=r"(h[2 * j]) : "f"(f[1]), "f"(f[0]));  // (the first source is the upper half)
      asm("cvt.rz.f16x2.f32 %0, %1, %2;" : "=r"(h[2 * j + 1]) : "f"(f[3]), "f"(f[2]));
    }
    reinterpret_cast<uint4*>(xh + (int64_t)m * K)[c] = make_uint4(h[0], h[1], h[2], h[3]);
  }
  int any_wide = __any_sync(0xffffffffu, wide);
  if (G > 32) {
    if ((threadIdx.x & 31) == 0) warp_wide[warp] = any_wide;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < G / 32; ++w) any_wide |= warp_wide[r_in_cta * (G / 32) + w];
  }
  if (live && t == 0) inv[m] = any_wide ? -1.0f : (bits == 0 ? 1.0f : __uint_as_float((uint32_t)(e - 14) << 23));
}

static unsigned flat_grid(int64_t work_items) {
  const int64_t want = ceil_div(work_items, 256);
  return (unsigned)(want < 1 ? 1 : (want > 148 * 32 ? 148 * 32 : want));
}

static int launch_unpack_int4(const uint8_t* packed, int64_t n_bytes, int8_t* q, cudaStream_t st) {
  const bool vec = is_aligned(packed, 8) && is_aligned(q, 16);
  return launch_pdl(unpack_int4_kernel, dim3(flat_grid(vec ? n_bytes / 8 + 8 : n_bytes), 1, 1), dim3(256, 1, 1), 0, st, 1, packed, n_bytes, q, vec);
}

// codes: int8 [n] or packed nibbles [n / 2], 4-byte (2-byte if packed) aligned; out: float [n], 16-byte aligned; n % 4 == 0.
static int launch_codes_to_float(const void* codes, bool packed, int64_t n, float* out, cudaStream_t st) {
  return launch_pdl(codes_to_float_kernel, dim3(flat_grid(n / 4), 1, 1), dim3(256, 1, 1), 0, st, 1, reinterpret_cast<const uint8_t*>(codes), packed, n, out);
}

constexpr int kHalfMaxK = 1024;
// xh: [M, K] halves; inv: [M]; w_f, w_h: [N, K] (n = N * K codes).
static int launch_half_operands(const float* x, int64_t ldx, int64_t M, int64_t K, __half* xh, float* inv, const void* codes, bool packed, int64_t n,
                                float* w_f, __half* w_h, cudaStream_t st) {
  const int g = K <= 512 ? 32 : 64;
  const int64_t row_blocks = ceil_div(M, 256 / g), want = ceil_div(n / 4, 256 * 2);
  const int64_t w_blocks = want < 1 ? 1 : (want > 148 * 8 ? 148 * 8 : want);
  auto kernel = g == 32 ? half_operands_kernel<32> : half_operands_kernel<64>;
  return launch_pdl(kernel, dim3((unsigned)(row_blocks + w_blocks), 1, 1), dim3(256, 1, 1), 0, st, 1, x, ldx, (int)M, (int)K, xh, inv, (int)row_blocks,
                    reinterpret_cast<const uint8_t*>(codes), packed, n, w_f, w_h);
}

static int launch_split_hi_lo(const float* x, int64_t ldx, int64_t M, int64_t K, float* out, cudaStream_t st) {
  return launch_pdl(split_hi_lo_kernel, dim3(flat_grid(M * K / 4), 1, 1), dim3(256, 1, 1), 0, st, 1, x, ldx, M, K, out);
}
static int launch_codes_to_float_twice(const void* codes, bool packed, int64_t rows, int64_t K, float* out, cudaStream_t st) {
  return launch_pdl(codes_to_float_twice_kernel, dim3(flat_grid(rows * K / 4), 1, 1), dim3(256, 1, 1), 0, st, 1, reinterpret_cast<const uint8_t*>(codes), packed,
                    rows, K, out);
}

static int launch_pack_int4(const int8_t* q, int64_t n_bytes, uint8_t* packed, cudaStream_t st) {
  const bool vec = is_aligned(packed, 8) && is_aligned(q, 16);
  pack_int4_kernel<<<flat_grid(vec ? n_bytes / 8 + 8 : n_bytes), 256, 0, st>>>(q, n_bytes, packed, vec);
  return AQT_LAUNCH_STATUS();
}

}  // namespace aqt
