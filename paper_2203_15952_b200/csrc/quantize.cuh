// Activation / weight quantizer kernels: Fig. 2 of the paper (abs-max over the reduced axis,
// scale = amax / qmax, divide_no_nan, round, int8 container) and its int4 form (Section 2.2).
// HBM-bound: one read of fp32 x, one write of codes and scales.
#pragma once

#include "aqt_common.cuh"

namespace aqt {

constexpr int kQuantThreads = 256;
constexpr int kQuantMaxVec = 4;  // float4 loads held in registers per thread (16 elements)

// Pack four codes (sign-extended ints) into the output word: int8 container (4 bytes) or nibbles
// (2 bytes).  Byte permutes take the low byte of each code.
__device__ __forceinline__ uint32_t pack4_i8(int a, int b, int c, int d) {
  const uint32_t lo = __byte_perm((uint32_t)a, (uint32_t)b, 0x0040);  // a.b0, b.b0
  const uint32_t hi = __byte_perm((uint32_t)c, (uint32_t)d, 0x0040);  // c.b0, d.b0
  return __byte_perm(lo, hi, 0x5410);
}
// Four codes in a word as nibbles.
__device__ __forceinline__ uint32_t nibbles4(uint32_t w) {
  const uint32_t x = w & 0x0F0F0F0Fu;
  const uint32_t y = x | (x >> 4);         // byte 0 = n0 | n1 << 4, byte 2 = n2 | n3 << 4
  return __byte_perm(y, 0u, 0x4420) & 0xFFFFu;
}
__device__ __forceinline__ uint32_t pack4_i4(int a, int b, int c, int d) { return nibbles4(pack4_i8(a, b, c, d)); }

// Four elements of a row whose scale constants are known, fast path of quantize_elem: the
// correctly rounded quotient by one multiply and two FMAs, then one conversion.  No clip: with
// abs-max scaling |x / s| <= qmax (1 + 2^-23), which every rounding rule maps inside +-qmax; the
// clip only matters for the subnormal scales that never take this path.
template <int ROUNDING>
__device__ __forceinline__ int quantize_fast(float x, float s, float r) {
  const float q0 = __fmul_rn(x, r);
  const float e = __fmaf_rn(-q0, s, x);
  const float v = __fmaf_rn(e, r, q0);
  if (ROUNDING == AQT_ROUND_HALF_UP_FLOOR) return __float2int_rd(__fadd_rn(v, 0.5f));
  return __float2int_rn(v);
}

// Per-row quantizer, row held in registers.  G threads cooperate on one row (G a power of two,
// 32 <= G <= 256); each thread owns up to kQuantMaxVec float4s, strided by G so that every load
// and store instruction of a warp is contiguous.  Requires cols % 4 == 0, ld % 4 == 0, x 16-byte
// aligned, cols <= 16 * G.
// Six blocks an SM: at 41 registers, which the call of the general sequence can bring, five fit (25 033 x 1408 31.2 -> 33.2 us).
template <int G, int ROUNDING, bool PACK>
__global__ void __launch_bounds__(kQuantThreads, 6) quantize_rows_reg_kernel(
    const float* __restrict__ x, int64_t rows, int cols, int64_t ld, int qmax, void* __restrict__ q_out,
    float* __restrict__ scale_out) {
  constexpr int ROWS_PER_CTA = kQuantThreads / G;
  constexpr int WARPS_PER_ROW = G / 32;
  __shared__ float warp_max[kQuantThreads / 32];

  grid_dependency_wait();
  const int t = threadIdx.x % G;
  const int r_in_cta = threadIdx.x / G;
  const int64_t row = (int64_t)blockIdx.x * ROWS_PER_CTA + r_in_cta;
  const bool live = row < rows;
  const int nvec = cols >> 2;
  const float4* xrow = reinterpret_cast<const float4*>(x + (live ? row : 0) * ld);

  float4 v[kQuantMaxVec];
  float amax = 0.0f;
#pragma unroll
  for (int i = 0; i < kQuantMaxVec; ++i) {
    const int idx = t + i * G;
    v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (live && idx < nvec) v[i] = __ldg(xrow + idx);
    amax = fmaxf(amax, fmaxf(fmaxf(fabsf(v[i].x), fabsf(v[i].y)), fmaxf(fabsf(v[i].z), fabsf(v[i].w))));
  }
  grid_dependents_launch();  // this CTA's loads are in flight; it has little left to do
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, off));
  if (WARPS_PER_ROW > 1) {
    const int warp = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) warp_max[warp] = amax;
    __syncthreads();
    const int w0 = r_in_cta * WARPS_PER_ROW;
#pragma unroll
    for (int w = 0; w < WARPS_PER_ROW; ++w) amax = fmaxf(amax, warp_max[w0 + w]);
  }
  if (!live) return;

  const ScaleCtx c = make_scale_ctx(amax, qmax);
  if (t == 0) scale_out[row] = c.s;

#pragma unroll
  for (int i = 0; i < kQuantMaxVec; ++i) {
    const int idx = t + i * G;
    if (idx < nvec) {
      uint32_t w;  // four codes
      if (__builtin_expect(c.fast, 1))  // uniform over the row
        w = pack4_i8(quantize_fast<ROUNDING>(v[i].x, c.s, c.r), quantize_fast<ROUNDING>(v[i].y, c.s, c.r), quantize_fast<ROUNDING>(v[i].z, c.s, c.r),
                     quantize_fast<ROUNDING>(v[i].w, c.s, c.r));
      else
        w = codes4_general(v[i].x, v[i].y, v[i].z, v[i].w, c.s, qmax, ROUNDING);
      // one output word per float4: 2 bytes of nibbles or 4 bytes of int8 codes
      if (PACK) reinterpret_cast<uint16_t*>(q_out)[row * (int64_t)nvec + idx] = (uint16_t)nibbles4(w);
      else reinterpret_cast<uint32_t*>(q_out)[row * (int64_t)nvec + idx] = w;
    }
  }
}

// Per-row quantizer for any cols / ld / alignment: one CTA per row, two passes over the row
// (the second pass re-reads what the first just brought into L1/L2).
template <int ROUNDING, bool PACK>
__global__ void __launch_bounds__(kQuantThreads) quantize_rows_generic_kernel(
    const float* __restrict__ x, int64_t rows, int64_t cols, int64_t ld, int qmax, void* __restrict__ q_out,
    float* __restrict__ scale_out) {
  __shared__ float warp_max[kQuantThreads / 32];
  for (int64_t row = blockIdx.x; row < rows; row += gridDim.x) {
    const float* xr = x + row * ld;
    float amax = 0.0f;
    for (int64_t j = threadIdx.x; j < cols; j += kQuantThreads) amax = fmaxf(amax, fabsf(xr[j]));
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, off));
    __syncthreads();  // warp_max of the previous row is no longer read
    if ((threadIdx.x & 31) == 0) warp_max[threadIdx.x >> 5] = amax;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < kQuantThreads / 32; ++w) amax = fmaxf(amax, warp_max[w]);
    const ScaleCtx c = make_scale_ctx(amax, qmax);
    if (threadIdx.x == 0) scale_out[row] = c.s;
    if (PACK) {
      uint8_t* qr = reinterpret_cast<uint8_t*>(q_out) + row * (cols / 2);
      for (int64_t j = threadIdx.x; j < cols / 2; j += kQuantThreads) {
        const int lo = quantize_elem<ROUNDING>(xr[2 * j], c, qmax);
        const int hi = quantize_elem<ROUNDING>(xr[2 * j + 1], c, qmax);
        qr[j] = (uint8_t)((lo & 0xF) | ((hi & 0xF) << 4));
      }
    } else {
      int8_t* qr = reinterpret_cast<int8_t*>(q_out) + row * cols;
      for (int64_t j = threadIdx.x; j < cols; j += kQuantThreads) qr[j] = (int8_t)quantize_elem<ROUNDING>(xr[j], c, qmax);
    }
  }
}

// abs-max accumulation for the column and tensor axes.  Non-negative floats order like their
// bit patterns, so atomicMax on the unsigned view is a float max.  amax_bits must be zeroed
// before the launch; it has `cols` slots (per_col) or one.
__global__ void __launch_bounds__(kQuantThreads) absmax_accumulate_kernel(
    const float* __restrict__ x, int64_t rows, int64_t cols, int64_t ld, bool per_col, unsigned* __restrict__ amax_bits) {
  if (per_col) {
    // thread <-> column (coalesced across the warp), CTA.y strides over row chunks
    const int64_t col = (int64_t)blockIdx.x * kQuantThreads + threadIdx.x;
    if (col >= cols) return;
    float amax = 0.0f;
    for (int64_t r = blockIdx.y; r < rows; r += gridDim.y) amax = fmaxf(amax, fabsf(x[r * ld + col]));
    atomicMax(amax_bits + col, __float_as_uint(amax));
  } else {
    __shared__ float warp_max[kQuantThreads / 32];
    float amax = 0.0f;
    const int64_t total = rows * cols;
    for (int64_t i = (int64_t)blockIdx.x * kQuantThreads + threadIdx.x; i < total; i += (int64_t)gridDim.x * kQuantThreads) {
      const int64_t r = i / cols, j = i - r * cols;
      amax = fmaxf(amax, fabsf(x[r * ld + j]));
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, off));
    if ((threadIdx.x & 31) == 0) warp_max[threadIdx.x >> 5] = amax;
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int w = 1; w < kQuantThreads / 32; ++w) amax = fmaxf(amax, warp_max[w]);
      atomicMax(amax_bits, __float_as_uint(amax));
    }
  }
}

// amax -> scale in place (scale = amax / qmax, IEEE division).
__global__ void finalize_scales_kernel(float* __restrict__ scale, int64_t n, int qmax) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) scale[i] = __fdiv_rn(scale[i], (float)qmax);
}

// Element-wise quantization against scales that are already final (column or tensor axis).
// One thread per pair of adjacent columns so that packed output needs no cross-thread exchange.
template <int ROUNDING, bool PACK>
__global__ void __launch_bounds__(kQuantThreads) quantize_with_scales_kernel(
    const float* __restrict__ x, int64_t rows, int64_t cols, int64_t ld, bool per_col, int qmax,
    const float* __restrict__ scale, void* __restrict__ q_out) {
  const int64_t pairs_per_row = (cols + 1) / 2;
  const int64_t total = rows * pairs_per_row;
  for (int64_t i = (int64_t)blockIdx.x * kQuantThreads + threadIdx.x; i < total; i += (int64_t)gridDim.x * kQuantThreads) {
    const int64_t r = i / pairs_per_row, p = i - r * pairs_per_row;
    const int64_t j0 = 2 * p, j1 = 2 * p + 1;
    // the scale is already divided; rebuild the per-scale constants from it
    ScaleCtx c0, c1;
    c0.s = scale[per_col ? j0 : 0];
    c0.fast = (c0.s >= 1.2e-20f) && (c0.s <= 8.0e15f);
    c0.r = c0.fast ? __frcp_rn(c0.s) : 0.0f;
    const int a = quantize_elem<ROUNDING>(x[r * ld + j0], c0, qmax);
    int b = 0;
    if (j1 < cols) {
      c1 = c0;
      if (per_col) {
        c1.s = scale[j1];
        c1.fast = (c1.s >= 1.2e-20f) && (c1.s <= 8.0e15f);
        c1.r = c1.fast ? __frcp_rn(c1.s) : 0.0f;
      }
      b = quantize_elem<ROUNDING>(x[r * ld + j1], c1, qmax);
    }
    if (PACK) {
      reinterpret_cast<uint8_t*>(q_out)[r * (cols / 2) + p] = (uint8_t)((a & 0xF) | ((b & 0xF) << 4));
    } else {
      int8_t* q = reinterpret_cast<int8_t*>(q_out) + r * cols;
      q[j0] = (int8_t)a;
      if (j1 < cols) q[j1] = (int8_t)b;
    }
  }
}

// Whole-tensor scale for small tensors in one launch: one CTA finds the abs-max, forms the scale
// and quantizes (the tensor is re-read from L1/L2).  Replaces the four-launch path below where
// launch latency, not bandwidth, is the cost (e.g. a [64, 256] activation).
// Beyond what the block can keep in registers the three launches of the vectorized form are shorter (64 x 512: 17.2 us in one
// block, 4.1 in three launches; 64 x 256: 3.1, 3.9).  A dense tensor up to there stays in registers, others are read
// twice (64 x 200 with a row pitch: 8.1 us).  Tensors that cannot be read as float4s have the four launches of the
// element-wise form to compare with: 40 x 511 11.4 us in one block, 12.4 in four launches, 64 x 400 13.7 and 12.3.
constexpr int kSmallTensorElems = 1 << 14, kSmallTensorElemsScalar = 22 << 10;
template <int ROUNDING, bool PACK>
__global__ void __launch_bounds__(1024) quantize_tensor_small_kernel(const float* __restrict__ x, int rows, int cols, int64_t ld,
                                                                      int qmax, void* __restrict__ q_out,
                                                                      float* __restrict__ scale_out) {
  __shared__ float warp_max[32];
  const int total = rows * cols;
  // dense, aligned tensors of up to 16 K elements stay in registers: all loads are issued at once
  const bool in_regs = (ld == cols) && (total % 4 == 0) && (total <= 4 * 4 * 1024) &&
                       ((reinterpret_cast<uintptr_t>(x) & 15) == 0) && ((reinterpret_cast<uintptr_t>(q_out) & 3) == 0);
  float4 v[4];
  float amax = 0.0f;
  if (in_regs) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int idx = threadIdx.x + i * 1024;
      v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (idx < total / 4) v[i] = __ldg(reinterpret_cast<const float4*>(x) + idx);
      amax = fmaxf(amax, fmaxf(fmaxf(fabsf(v[i].x), fabsf(v[i].y)), fmaxf(fabsf(v[i].z), fabsf(v[i].w))));
    }
  } else {
    for (int i = threadIdx.x; i < total; i += blockDim.x) {
      const int r = i / cols, j = i - r * cols;
      amax = fmaxf(amax, fabsf(x[(int64_t)r * ld + j]));
    }
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, off));
  if ((threadIdx.x & 31) == 0) warp_max[threadIdx.x >> 5] = amax;
  __syncthreads();
  amax = 0.0f;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) amax = fmaxf(amax, warp_max[w]);
  const ScaleCtx c = make_scale_ctx(amax, qmax);
  if (threadIdx.x == 0) scale_out[0] = c.s;
  if (in_regs) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int idx = threadIdx.x + i * 1024;
      if (idx < total / 4) {
        const int a = quantize_elem<ROUNDING>(v[i].x, c, qmax), b = quantize_elem<ROUNDING>(v[i].y, c, qmax);
        const int cc = quantize_elem<ROUNDING>(v[i].z, c, qmax), d = quantize_elem<ROUNDING>(v[i].w, c, qmax);
        if (PACK) reinterpret_cast<uint16_t*>(q_out)[idx] = (uint16_t)pack4_i4(a, b, cc, d);
        else reinterpret_cast<uint32_t*>(q_out)[idx] = pack4_i8(a, b, cc, d);
      }
    }
    return;
  }
  const int pairs_per_row = (cols + 1) / 2;
  for (int i = threadIdx.x; i < rows * pairs_per_row; i += blockDim.x) {
    const int r = i / pairs_per_row, p = i - r * pairs_per_row;
    const int j0 = 2 * p, j1 = 2 * p + 1;
    const int a = quantize_elem<ROUNDING>(x[(int64_t)r * ld + j0], c, qmax);
    const int b = j1 < cols ? quantize_elem<ROUNDING>(x[(int64_t)r * ld + j1], c, qmax) : 0;
    if (PACK) {
      reinterpret_cast<uint8_t*>(q_out)[(int64_t)r * (cols / 2) + p] = (uint8_t)((a & 0xF) | ((b & 0xF) << 4));
    } else {
      int8_t* q = reinterpret_cast<int8_t*>(q_out) + (int64_t)r * cols;
      q[j0] = (int8_t)a;
      if (j1 < cols) q[j1] = (int8_t)b;
    }
  }
}

// Whole-tensor scale, tensors beyond kSmallTensorElems whose rows are float4s (cols % 4 == 0, ld % 4 == 0,
// 16-byte aligned x): two HBM / L2-bound passes of four float4 loads in flight per thread.
//   pass 1  abs-max of a block's share of the tensor.  The blocks' maxima either land in `partial`, one
//           word per block (a caller with scratch space: no word has to be cleared first), or are
//           combined by atomicMax in scale_out, which one thread has zeroed in a launch before, already
//           divided by qmax (division is monotonic: the largest quotient is the quotient of the largest).
//   pass 2  every block forms the scale (from the partial maxima: at most kAbsmaxBlocks words, read from
//           L2) and quantizes its share; the second read of x comes from L2 up to about 100 MB.
// A 7411 x 512 tensor takes 3.1 + 5.6 us against 9.7 + 1.8 + 9.6 us (and a memset) for the element-wise
// kernels above, which spend their time on a 64-bit division per element; those keep the tensors that
// cannot be read as float4s.
constexpr int kAbsmaxBlocks = 148 * 4;
constexpr int kTensorVec = 4;  // float4s per thread and step

__global__ void clear_scale_kernel(float* __restrict__ scale) {
  grid_dependency_wait();
  *scale = 0.0f;
}

// float4 number i of the tensor; nvec: float4s per row, ld4: row pitch in float4s (equal: dense)
__device__ __forceinline__ const float4* tensor_vec(const float* x, int64_t i, int64_t nvec, int64_t ld4) {
  if (nvec != ld4) {
    const int64_t r = i / nvec;
    i += r * (ld4 - nvec);
  }
  return reinterpret_cast<const float4*>(x) + i;
}

__global__ void __launch_bounds__(kQuantThreads) absmax_tensor_vec_kernel(const float* __restrict__ x, int64_t n4, int64_t nvec, int64_t ld4,
                                                                          int qmax, float* __restrict__ partial, float* __restrict__ scale_out,
                                                                          bool beside) {
  __shared__ float warp_max[kQuantThreads / 32];
  grid_dependency_wait();
  if (beside) grid_dependents_launch();
  float amax = 0.0f;
  const int64_t step = (int64_t)gridDim.x * kQuantThreads * kTensorVec;
  for (int64_t i0 = (int64_t)blockIdx.x * kQuantThreads * kTensorVec + threadIdx.x; i0 < n4; i0 += step) {
    float4 v[kTensorVec];
#pragma unroll
    for (int j = 0; j < kTensorVec; ++j) {
      const int64_t i = i0 + j * kQuantThreads;
      v[j] = i < n4 ? __ldg(tensor_vec(x, i, nvec, ld4)) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int j = 0; j < kTensorVec; ++j) amax = fmaxf(amax, fmaxf(fmaxf(fabsf(v[j].x), fabsf(v[j].y)), fmaxf(fabsf(v[j].z), fabsf(v[j].w))));
  }
  if (!beside) grid_dependents_launch();
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, off));
  if ((threadIdx.x & 31) == 0) warp_max[threadIdx.x >> 5] = amax;
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int w = 1; w < kQuantThreads / 32; ++w) amax = fmaxf(amax, warp_max[w]);
    if (partial != nullptr) partial[blockIdx.x] = amax;
    else atomicMax(reinterpret_cast<unsigned*>(scale_out), __float_as_uint(__fdiv_rn(amax, (float)qmax)));
  }
}

// BESIDE: every block has one share of the tensor, and may start while pass 1 runs.
template <int ROUNDING, bool PACK, bool BESIDE, int VEC>
__global__ void __launch_bounds__(kQuantThreads) quantize_tensor_vec_kernel(const float* __restrict__ x, int64_t n4, int64_t nvec, int64_t ld4,
                                                                            int qmax, const float* __restrict__ partial, int partials,
                                                                            float* __restrict__ scale_out, void* __restrict__ q_out) {
  __shared__ float warp_max[kQuantThreads / 32];
  // The kernel ahead is pass 1 of the same call: it writes none of x, and this one can only have started when whatever
  // wrote x was complete.  So its loads need not wait for pass 1.
  float4 v[VEC];
  const auto load = [&](int64_t i0) {
#pragma unroll
    for (int j = 0; j < VEC; ++j) {
      const int64_t i = i0 + j * kQuantThreads;
      if (i < n4) v[j] = __ldg(tensor_vec(x, i, nvec, ld4));
    }
  };
  const int64_t first = (int64_t)blockIdx.x * kQuantThreads * VEC + threadIdx.x;
  if (BESIDE) load(first);
  grid_dependency_wait();
  grid_dependents_launch();  // (the next kernel waits for the end of this one; what it can do ahead of that it may begin)
  ScaleCtx c;
  if (partial != nullptr) {
    float amax = 0.0f;
    for (int i = threadIdx.x; i < partials; i += kQuantThreads) amax = fmaxf(amax, __ldg(partial + i));
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, off));
    if ((threadIdx.x & 31) == 0) warp_max[threadIdx.x >> 5] = amax;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < kQuantThreads / 32; ++w) amax = fmaxf(amax, warp_max[w]);
    c = make_scale_ctx_zeros(amax, qmax);
    if (blockIdx.x == 0 && threadIdx.x == 0) *scale_out = c.s;
  } else {
    c.s = __ldg(scale_out);  // divided already: rebuild the other constants from it
    const bool normal = (c.s >= 1.2e-20f) && (c.s <= 8.0e15f);
    c.fast = normal || c.s == 0.0f;
    c.r = normal ? __frcp_rn(c.s) : 0.0f;
  }
  const int64_t step = (int64_t)gridDim.x * kQuantThreads * VEC;
  for (int64_t i0 = first; i0 < n4; i0 += step) {
    if (!BESIDE) load(i0);
#pragma unroll
    for (int j = 0; j < VEC; ++j) {
      const int64_t i = i0 + j * kQuantThreads;
      if (i >= n4) break;
      uint32_t w;
      if (__builtin_expect(c.fast, 1)) {
        w = pack4_i8(quantize_fast<ROUNDING>(v[j].x, c.s, c.r), quantize_fast<ROUNDING>(v[j].y, c.s, c.r), quantize_fast<ROUNDING>(v[j].z, c.s, c.r),
                     quantize_fast<ROUNDING>(v[j].w, c.s, c.r));
      } else {
        // (eight float4s held across the call are 24 bytes of spills at 64 registers; read again, 51 registers and none)
        const float4 g = VEC > kTensorVec ? __ldg(tensor_vec(x, i, nvec, ld4)) : v[j];
        w = codes4_general(g.x, g.y, g.z, g.w, c.s, qmax, ROUNDING);
      }
      if (PACK) reinterpret_cast<uint16_t*>(q_out)[i] = (uint16_t)nibbles4(w);
      else reinterpret_cast<uint32_t*>(q_out)[i] = w;
    }
  }
}

static bool tensor_vec_ok(const float* x, int64_t cols, int64_t ld, const void* q_out) {
  return cols % 4 == 0 && ld % 4 == 0 && is_aligned(x, 16) && is_aligned(q_out, 4);
}

// partial: nullptr, or max_partials (>= 1) words of scratch.
template <int ROUNDING, bool PACK>
static int launch_quantize_tensor_vec(const float* x, int64_t rows, int64_t cols, int64_t ld, int qmax, void* q_out, float* scale_out,
                                      float* partial, int64_t max_partials, cudaStream_t st) {
  const int64_t n4 = rows * (cols / 4), want = ceil_div(n4, kQuantThreads * kTensorVec);
  int64_t blocks = want < kAbsmaxBlocks ? want : kAbsmaxBlocks;
  if (partial != nullptr && blocks > max_partials) blocks = max_partials;
  // Where pass 2's blocks fit beside those of pass 1, each with one share of the tensor, they wait for the scale with that share
  // in registers: four float4s a thread, or eight (graph replay of the layer: 300 x 128 9.2 -> 7.2 us, 641 x 288 10.8 -> 8.7,
  // 3000 x 256 10.8 -> 9.7; eight: 7411 x 512 19.7 -> 18.6, 2000 x 2048 17.9 -> 17.0).  Beyond, the blocks that wait would keep
  // others of either pass from the SMs (65 536 x 512 100 -> 113).
  const int64_t sms = sm_count() > 0 ? sm_count() : kDefaultSms;
  const int64_t want8 = ceil_div(n4, kQuantThreads * 2 * kTensorVec);
  const bool beside = want <= sms * 4, beside8 = !beside && want8 <= sms * 4;
  const int64_t grid = beside8 ? want8 : (want < sms * 8 ? want : sms * 8);
  int rc;
  if (partial == nullptr) {
    rc = launch_pdl(clear_scale_kernel, dim3(1, 1, 1), dim3(1, 1, 1), 0, st, 1, scale_out);
    if (rc != AQT_OK) return rc;
  }
  rc = launch_pdl(absmax_tensor_vec_kernel, dim3((unsigned)blocks, 1, 1), dim3(kQuantThreads, 1, 1), 0, st, 1, x, n4, cols / 4, ld / 4, qmax,
                  partial, scale_out, beside || beside8);
  if (rc != AQT_OK) return rc;
  auto kernel = beside8 ? quantize_tensor_vec_kernel<ROUNDING, PACK, true, 2 * kTensorVec>
                        : (beside ? quantize_tensor_vec_kernel<ROUNDING, PACK, true, kTensorVec> : quantize_tensor_vec_kernel<ROUNDING, PACK, false, kTensorVec>);
  return launch_pdl(kernel, dim3((unsigned)grid, 1, 1), dim3(kQuantThreads, 1, 1), 0, st, 1, x, n4,
                    cols / 4, ld / 4, qmax, (const float*)partial, (int)blocks, scale_out, q_out);
}

template <int ROUNDING, bool PACK>
static int launch_quantize_rows(const float* x, int64_t rows, int64_t cols, int64_t ld, int qmax, void* q_out,
                                float* scale_out, cudaStream_t st) {
  const bool vec_ok = (cols % 4 == 0) && (ld % 4 == 0) && is_aligned(x, 16) && cols <= 16 * 256 &&
                      is_aligned(q_out, 4);
  if (vec_ok) {
    const int nvec = (int)(cols / 4);
#define AQT_LAUNCH_ROWS(G)                                                                                   \
  do {                                                                                                       \
    const int64_t grid = ceil_div(rows, kQuantThreads / G);                                                  \
    const int rc_launch = launch_pdl(quantize_rows_reg_kernel<G, ROUNDING, PACK>, dim3((unsigned)grid, 1, 1),       \
                                     dim3(kQuantThreads, 1, 1), 0, st, 1, x, rows, (int)cols, ld, qmax, q_out, scale_out); \
    if (rc_launch != AQT_OK) return rc_launch;                                                               \
  } while (0)
    if (nvec <= 32 * kQuantMaxVec) AQT_LAUNCH_ROWS(32);
    else if (nvec <= 64 * kQuantMaxVec) AQT_LAUNCH_ROWS(64);
    else if (nvec <= 128 * kQuantMaxVec) AQT_LAUNCH_ROWS(128);
    else AQT_LAUNCH_ROWS(256);
#undef AQT_LAUNCH_ROWS
  } else {
    const int64_t grid = rows < 148 * 16 ? rows : 148 * 16;
    quantize_rows_generic_kernel<ROUNDING, PACK><<<(unsigned)grid, kQuantThreads, 0, st>>>(x, rows, cols, ld, qmax, q_out, scale_out);
  }
  return AQT_LAUNCH_STATUS();
}

template <int ROUNDING, bool PACK>
static int launch_quantize_axis(const float* x, int64_t rows, int64_t cols, int64_t ld, int qmax, int axis, void* q_out,
                                float* scale_out, cudaStream_t st, float* partial = nullptr, int64_t max_partials = 0) {
  if (axis == AQT_AXIS_ROW) return launch_quantize_rows<ROUNDING, PACK>(x, rows, cols, ld, qmax, q_out, scale_out, st);
  const bool per_col = axis == AQT_AXIS_COL;
  const bool vec = !per_col && tensor_vec_ok(x, cols, ld, q_out);
  if (!per_col && rows * cols <= (vec ? kSmallTensorElems : kSmallTensorElemsScalar)) {
    quantize_tensor_small_kernel<ROUNDING, PACK><<<1, 1024, 0, st>>>(x, (int)rows, (int)cols, ld, qmax, q_out, scale_out);
    return AQT_LAUNCH_STATUS();
  }
  if (vec)
    return launch_quantize_tensor_vec<ROUNDING, PACK>(x, rows, cols, ld, qmax, q_out, scale_out, partial, max_partials, st);
  const int64_t n_scale = per_col ? cols : 1;
  AQT_RETURN_IF_CUDA(cudaMemsetAsync(scale_out, 0, (size_t)n_scale * sizeof(float), st));
  if (per_col) {
    dim3 grid((unsigned)ceil_div(cols, kQuantThreads), (unsigned)(rows < 64 ? rows : 64));
    absmax_accumulate_kernel<<<grid, kQuantThreads, 0, st>>>(x, rows, cols, ld, true, reinterpret_cast<unsigned*>(scale_out));
  } else {
    const int64_t want = ceil_div(rows * cols, kQuantThreads * 8);
    const unsigned grid = (unsigned)(want < 1 ? 1 : (want > 148 * 8 ? 148 * 8 : want));
    absmax_accumulate_kernel<<<grid, kQuantThreads, 0, st>>>(x, rows, cols, ld, false, reinterpret_cast<unsigned*>(scale_out));
  }
  finalize_scales_kernel<<<(unsigned)ceil_div(n_scale, 256), 256, 0, st>>>(scale_out, n_scale, qmax);
  const int64_t pairs = rows * ((cols + 1) / 2);
  const int64_t want = ceil_div(pairs, kQuantThreads * 4);
  const unsigned grid = (unsigned)(want < 1 ? 1 : (want > 148 * 16 ? 148 * 16 : want));
  quantize_with_scales_kernel<ROUNDING, PACK><<<grid, kQuantThreads, 0, st>>>(x, rows, cols, ld, per_col, qmax, scale_out, q_out);
  return AQT_LAUNCH_STATUS();
}

}  // namespace aqt
