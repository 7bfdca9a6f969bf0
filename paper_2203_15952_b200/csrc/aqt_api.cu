// C ABI of the quantized linear layer: argument validation and kernel launches.
// Single translation unit: the kernels live in the headers included below.
#include "aqt_common.cuh"
#include "backward.cuh"
#include "pack.cuh"
#include "qgemm_sm100.cuh"
#include "dw_split_sm100.cuh"
#include "qgemm_requant_sm100.cuh"
#include "qgemm_few_tiles_sm100.cuh"
#include "qgemv_small_m.cuh"
#include "quantize.cuh"
#include "chain_small_m.cuh"
#include "host_copies.cuh"
#include "linear_small.cuh"
#include "weight_only_small.cuh"

using namespace aqt;

namespace {

// The kernels use tcgen05 / TMEM and exist for compute capability 10.x only.  Asked of the
// current device on every call (the answer is cached per device ordinal).
int check_device() {
  DeviceInfo d;
  int rc = current_device_info(&d);
  if (rc != AQT_OK) return rc;
  return d.cc_major == 10 ? AQT_OK : AQT_ERR_UNSUPPORTED;
}

// Operand widths a matmul accepts: 8, 4 (nibble-packed) or 4-bit codes in int8 containers.
bool bits_ok(int b) { return b == 4 || b == 8 || b == AQT_BITS_4_UNPACKED; }
bool quant_bits_ok(int b) { return b == 4 || b == 8; }
bool is_packed(int b) { return b == 4; }
int code_bits(int b) { return b == 8 ? 8 : 4; }  // range of the codes, whatever the container
bool act_ok(int a) { return a >= AQT_ACT_NONE && a <= AQT_ACT_GLU_SWISH; }
bool is_glu(int a) { return a == AQT_ACT_GLU || a == AQT_ACT_GLU_SWISH; }

size_t ws_qmatmul(int64_t M, int64_t N, int64_t K, int bits_a, int bits_w) {
  size_t b = 0;
  if (is_packed(bits_a)) b += round_up((size_t)M * (size_t)K, 256);
  if (is_packed(bits_w)) b += round_up((size_t)N * (size_t)K, 256);
  return b;
}
size_t ws_linear(int64_t M, int64_t N, int64_t K, int bits_w) {
  return round_up((size_t)M * (size_t)K, 256) + round_up((size_t)M * 4, 256) + ws_qmatmul(0, N, K, 8, bits_w);
}

// one-term form: the weights as floats; two-term form: the weights twice and the split activations
size_t ws_weight_only(int64_t M, int64_t N, int64_t K, int precision) {
  if (precision == AQT_FLOAT_TF32X2) return round_up((size_t)N * (size_t)K * 8, 256) + round_up((size_t)M * (size_t)K * 8, 256);
  return round_up((size_t)N * (size_t)K * 4, 256);
}

// Half kind of the one-term form: [weights as floats | weights as halves | rows as halves | inverse row scales].
struct HalfLayout {
  size_t w_h, x_h, inv, total;
};
HalfLayout half_layout(int64_t M, int64_t N, int64_t K) {
  HalfLayout L;
  L.w_h = ws_weight_only(0, N, K, AQT_FLOAT_TF32);
  L.x_h = L.w_h + round_up((size_t)N * (size_t)K * 2, 256);
  L.inv = L.x_h + round_up((size_t)M * (size_t)K * 2, 256);
  L.total = L.inv + round_up((size_t)M * 4, 256);
  return L;
}

// Backward workspace of the tf32 form: [column-sum partials | s_w-scaled W^T [K, N] | dy^T | s_x-scaled xq^T | dw partials].
// The weight gradient is an [N, K] output with a contraction of M: few, very deep tiles.  Its
// contraction is therefore cut into `batches` chunks of `chunk` rows (a multiple of 32), each
// batch a matmul of its own in the same launch (GemmParams::batch_tiles_m), and the batches'
// outputs are added in order.  The split is chosen for the 148 SMs of the one device this library
// is built for, so that the layout (and aqt_workspace_bytes) needs no CUDA call.
struct BwdLayout {
  size_t partial, wt, dyt, xt, dwp, total;
  int64_t batches, chunk, n_pad;  // batches == 1: chunk is the padded pitch of the transposed operands
};
BwdLayout bwd_layout(int64_t M, int64_t N, int64_t K) {
  BwdLayout L;
  L.n_pad = round_up((size_t)N, 128);
  const int64_t tiles = (L.n_pad / 128) * ceil_div(K, 256);
  int64_t batches = 148 / (tiles > 0 ? tiles : 1);
  if (batches > M / 512) batches = M / 512;  // a batch should still be some k-blocks deep
  if (batches < 2) {
    L.batches = 1;
    L.chunk = (M + 3) / 4 * 4;
    L.n_pad = N;
  } else {
    L.chunk = round_up((size_t)ceil_div(M, batches), kTrRows);
    L.batches = ceil_div(M, L.chunk);
  }
  L.partial = 0;
  // column-sum partials: one row of N per 128-row block of the transpose (or per 2048-row chunk of the stand-alone sum)
  L.wt = L.partial + round_up((size_t)(transpose_row_blocks(L.batches * L.chunk) + colsum_chunks(M)) * (size_t)N * 4, 256);
  L.dyt = L.wt + round_up((size_t)K * (size_t)N * 4, 256);
  L.xt = L.dyt + round_up((size_t)L.batches * L.n_pad * L.chunk * 4, 256);
  L.dwp = L.xt + round_up((size_t)L.batches * K * L.chunk * 4, 256);
  L.total = L.dwp + (L.batches > 1 ? round_up((size_t)L.batches * L.n_pad * K * 4, 256) : 0);
  return L;
}

// Weight gradient on split operands: [codes of x transposed, bf16 [K, m_pitch] | column-sum partials | dw partials], behind
// the scaled transposed weights of the other product.  Its contraction over M is cut into `batches` of `chunk` rows (a
// multiple of 32): the tiles are few and very deep, and they fill the SM pairs that the other product leaves free, so
// smaller ones end more evenly (half a tile's time, at 0.39 us a K-block of 32 rows, plus 3 us a tile to start it)
// against 5 TB/s for adding the partial products.  Up to 16 batches; more where the batches of that many rows are longer
// than 1024 and three quarters of the pairs take them all at once (dw alone at 40 000 x 128 x 128: 16 batches 48 us, 36 with
// more; but at 12 800 rows 74 pairs of short tiles get in the way of the other product, 29 -> 35 us for both).  For the
// 74 pairs of the one part this library is built for, so that the layout needs no CUDA call.
struct DwLayout {
  size_t wt, xt, colsum, dwp, total;
  int64_t m_pitch, batches, chunk, n_pad;
};
DwLayout dw_layout(int64_t M, int64_t N, int64_t K) {
  DwLayout L;
  const int64_t tiles = ceil_div(N, 256) * ceil_div(K, 256), pairs = kDefaultSms / 2;
  L.m_pitch = (int64_t)round_up((size_t)M, 8);
  L.n_pad = (int64_t)round_up((size_t)N, 256);
  L.batches = 1;
  double best = 1e300;
  int64_t most = 3 * pairs / 4 / (tiles > 0 ? tiles : 1);
  if (most > M / 1024) most = M / 1024;
  if (most < 16) most = 16;
  for (int64_t b = 1; b <= most && (b == 1 || M / b >= 256); ++b) {
    const double tile_us = 0.39 * (double)ceil_div(ceil_div(M, b), 32) + 3.0;
    const double rounds = (double)(tiles * b) / (double)pairs;
    const double main_us = tile_us * (rounds < 1.0 ? 1.0 : rounds + 0.5);
    const double sum_us = b > 1 ? 2.0 + ((double)b + 1.0) * (double)N * (double)K * 4.0 / 5e6 : 0.0;
    if (main_us + sum_us < best) {
      best = main_us + sum_us;
      L.batches = b;
    }
  }
  L.chunk = (int64_t)round_up((size_t)ceil_div(M > 0 ? M : 1, L.batches), 32);
  L.batches = ceil_div(M, L.chunk);
  L.wt = 0;
  L.xt = L.wt + round_up((size_t)K * (size_t)N * 4, 256);
  L.colsum = L.xt + round_up((size_t)K * L.m_pitch * 2, 256);
  L.dwp = L.colsum + round_up((size_t)(L.batches * DwCfg::kGroups) * N * 4, 256);
  L.total = L.dwp + (L.batches > 1 ? round_up((size_t)L.batches * L.n_pad * K * 4, 256) : 0);
  return L;
}
size_t bwd_workspace(int64_t M, int64_t N, int64_t K) {
  const size_t tf32_form = bwd_layout(M, N, K).total, split_form = dw_layout(M, N, K).total;
  return tf32_form > split_form ? tf32_form : split_form;
}

// y[r][c] = sum_j a[r][j] * b[c][j] on the float kind of the GEMM (no scale, bias or activation).
// batches > 1: a holds `batches` stacked [rows / batches, depth] blocks, b as many stacked [cols, depth] blocks,
// and y receives the stacked [rows / batches, cols] products.
int float_gemm_nt(const float* a, int64_t lda, const float* b, int64_t rows, int64_t cols, int64_t depth, float* y, int64_t ldy,
                  cudaStream_t st, int64_t batches = 1, bool early_trigger = false) {
  GemmParams p;
  if (batches > 1) {
    p.batch_tiles_m = (int)(rows / batches / kBM);  // rows per batch are a multiple of the tile height
    p.batch_b_rows = (int)cols;
    p.b_rows = batches * cols;
  }
  p.s_x = nullptr;
  p.s_w = nullptr;
  p.bias = nullptr;
  p.residual = nullptr;
  p.acc_debug = nullptr;
  p.ldr = 0;
  p.residual_scale = 0.0f;
  p.s_x_kind = AQT_SCALE_TENSOR;
  p.act = AQT_ACT_NONE;
  p.M = (int)rows;
  p.N = (int)cols;
  p.K = (int)(4 * depth);
  p.kind = 1;
  p.a_pitch = 4 * lda;
  p.n_out = (int)cols;
  p.tiles_m = p.tiles_n = p.k_blocks = 0;
  p.small_acc = 0;
  p.early_trigger = early_trigger ? 1 : 0;
  return launch_qgemm(reinterpret_cast<const int8_t*>(a), b, false, y, ldy, p, st);
}

// Sizes at which calls of the one-term weight-only layer may run on binary16 operands, twice the rate and half the bytes of tf32 ones for
// a pass that scales and writes the rows first (6 bytes an element).  What the workspace query goes by.  Not smaller outputs or deeper
// rows, of which the pass is too much (us in a replayed graph, tf32 / binary16: 30 000 x 512 -> 512 39.7 / 41.0, 30 000 x 2048 -> 512 98.6 /
// 117, 30 000 x 4096 -> 1024 321 / 348), nor less work (2000 x 512 -> 1024 11.2 / 12.0).
bool half_kind_sizes(int64_t M, int64_t N, int64_t K) {
  return K % 8 == 0 && K >= 256 && K <= kHalfMaxK && N >= 1024 && M >= 1024 && M * N >= ceil_div(1300000000ll, K) && tuning_env("AQT_NO_HALF") == nullptr;
}

// True if a call of such sizes does.  CTA pairs on 256 x 256 tiles; us in a replayed graph, tf32 / binary16, both with their passes:
// 12 800 x 512 -> 2048 Swish 51.7 / 44.2, 5000 x 768 -> 3072 Swish 48.3 / 37.2, 30 000 x 1024 -> 2048 gated 161 / 128, 30 000 x 1024 -> 1024
// 100 / 96.  An input with a wide row in every block of 256 (GemmParams::wide_a) pays for the pass and gains nothing: 51.9 / 59.2, 47.5 / 51.7,
// 173 / 214, 104 / 138; of normal values one block in 800 has one (512 columns).
// Not where what a tile saves does not pay for the pass (over 480 sizes and activations; the line lies where both are equal):
//   - one round of pairs saves once: K below 496, with gates 512 (1614 x 408 -> 2432 13.3 / 14.5, 3102 x 488 -> 1216 gated 14.3 / 15.4), and of
//     fewer than 40 tiles, where tf32 ones run on narrow single-CTA tiles, below 900 (1024 x 640 -> 2048 Swish 14.0 / 14.7, 1698 x 840 ->
//     1096 Swish 16.0 / 17.3; but 1254 x 1024 -> 1024, 20 tiles, 16.4 / 15.1);
//   - an activation's epilogue is most of a tile: Swish below K = 320 (18 359 x 296 -> 1824 53.2 / 55.6); gates in two rounds below 416 (2629 x 344 ->
//     2440 15.3 / 16.0), in more below 352 and N = 1536 (43 495 x 264 -> 1064 54.8 / 60.3; but 7122 x 304 -> 3192 0.865 of the time);
//   - few columns to a row (up to 1152, or a sixth column of tiles that is mostly padding), whose pass is the larger part, and full rounds,
//     in which pairs of tf32 tiles lose nothing: 31 595 x 648 -> 1096 87.4 / 89.1, 31 324 x 280 -> 1304 58.7 / 61.1 (with rounds less full
//     15 311 x 256 -> 1064 0.869, rows that L2 holds 5062 x 768 -> 1024 24.5 / 21.7).
bool half_kind_applies(int64_t M, int64_t N, int64_t K, int act, int sms) {
  if (!half_kind_sizes(M, N, K)) return false;
  const int64_t pairs = sms / 2, tiles = ceil_div(M, 2 * kBM) * ceil_div(N, 256), rounds = ceil_div(tiles, pairs);
  if (rounds == 1 && K < (tiles < 40 ? 900 : (is_glu(act) ? 512 : 496))) return false;
  if (act == AQT_ACT_SWISH && K < 320) return false;
  if (is_glu(act) && (rounds == 2 ? K < 416 : K < 352 && N < 1536)) return false;
  const bool few_columns = N < 1152 || (N > 1280 && N < 1344);
  return !(few_columns && K < 704 && M * K > (2 << 20) && 20 * tiles > 17 * rounds * pairs);
}

// True if the CTA-pair kernel with the row-quantizing epilogue takes the call: deep K, no GLU, int8
// codes out (4-bit codes stay in their containers), at most 16 column parts per row.
bool rowquant_pair_applies(int64_t M, int64_t N, int64_t K, int act, bool with_y, bool pack_out, int sms) {
  // (from K = 2048: at K = 1024 a tile's MMAs are shorter than its two epilogue passes, and the
  // two kernels are faster: 162 vs 209 us at 65 536 x 1024 -> 1024 with the fp32 output)
  if (pack_out || M <= kBM || K < 2048) return false;
  if (act != AQT_ACT_NONE && act != AQT_ACT_SWISH) return false;
  // With the fp32 output, few pair tiles leave most of the chip idle: narrow tiles and the row quantizer behind them take 9.3
  // against 14.2 us at 1024 x 2048 -> 512, 11.5 against 15.1 us at 4096 rows, 15.3 against 16.0 us at 8192 (64 tiles).
  // (But not where the matmul ahead of the row quantizer would be left between its forms, with more single-CTA tiles of 128
  // columns than one round takes and too few pair tiles: 16.0 in one kernel, 19.6 us in two at 5000 x 2048 -> 512.)
  const int64_t pair_tiles = ceil_div(M, 2 * kBM) * ceil_div(N, 256);
  if (with_y && 8 * pair_tiles <= 7 * (sms / 2) &&
      (ceil_div(M, kBM) * ceil_div(N, 128) <= sms || gemm_plan_is_pair(plan_qgemm(GemmShape{M, N, K, act, 0, false}, sms))))
    return false;
  const int plan = rowquant_plan(M, N, K, sms);
  const int parts = rowquant_parts(plan, N);
  return parts % 2 == 0 && parts <= 16 && ceil_div(N, kGemmPlanBn[plan]) <= sms / 2;
}

// The calls of aqt_qmatmul_requant that the header says may wait across CTAs.  The others are two kernels of which neither
// does, unless the caller allows it: other work that holds SMs until it sees their result is then no deadlock, and the codes
// may be written over those that were read.
bool waits_across_ctas(int64_t M, int64_t N, int64_t K, int act, bool with_y, bool pack_out, int sms) {
  return requant_applies(M, N, K, act, with_y, pack_out, sms) || (K >= 2048 && M > kBM && N <= 2048 && !is_glu(act) && !pack_out);
}

// How aqt_qmatmul_requant runs a call: one kernel (tiles of few_bn columns, weight-stationary tiles, CTA pairs), the two steps
// through y, or not at all.  exchange_room: workspace beyond what the matmul needs, at least requant_exchange_bytes.
enum RequantForm { kRequantRefused, kRequantFew, kRequantWs, kRequantPair, kRequantTwoKernels };
struct RequantRoute {
  RequantForm form;
  int few_bn;
};
RequantRoute requant_route(int64_t M, int64_t N, int64_t K, int act, bool with_y, bool pack_out, bool may_wait, size_t exchange_room, int sms) {
  const bool ws_form = requant_applies(M, N, K, act, with_y, pack_out, sms);
  const bool pair_form = !ws_form && rowquant_pair_applies(M, N, K, act, with_y, pack_out, sms);
  if (!ws_form && !pair_form && !with_y) return {kRequantRefused, 0};
  if (!pack_out && (may_wait || waits_across_ctas(M, N, K, act, with_y, pack_out, sms))) {
    const int bn = few_tiles_bn(M, N, K, act, 0, sms);
    if (bn != 0 && few_tiles_exchange_bytes(M, N, bn) <= exchange_room) return {kRequantFew, bn};
  }
  return {ws_form ? kRequantWs : (pair_form ? kRequantPair : kRequantTwoKernels), 0};
}
// The same for aqt_qmatmul_requant_from: 0, or the width of the tiles that take all columns in one launch.
int requant_from_bn(int64_t first, int64_t M, int64_t N, int64_t K, int bits_a, size_t exchange_room, int sms) {
  const int bn = is_packed(bits_a) ? 0 : few_tiles_bn(M, N, K, AQT_ACT_NONE, first, sms);
  return bn != 0 && few_tiles_exchange_bytes(M, N, bn) <= exchange_room ? bn : 0;
}

int validate_matmul_shape(int64_t M, int64_t N, int64_t K, int bits_a, int bits_w, int act, int s_x_kind) {
  if (M < 0 || N < 0 || K <= 0) return AQT_ERR_BADARG;
  if (!bits_ok(bits_a) || !bits_ok(bits_w) || !act_ok(act)) return AQT_ERR_BADARG;
  if (s_x_kind != AQT_SCALE_ROW && s_x_kind != AQT_SCALE_TENSOR) return AQT_ERR_BADARG;
  if (K % 16 != 0 || N % 4 != 0 || (is_glu(act) && N % 8 != 0)) return AQT_ERR_BADARG;
  if (M >= (1ll << 31) || N >= (1ll << 31) || K >= (1ll << 31) || M * N >= (1ll << 40)) return AQT_ERR_UNSUPPORTED;
  return AQT_OK;
}

int run_small_m(const void* xq, bool a_packed, const float* s_x, int s_x_kind, const void* wq, bool w_packed, const float* s_w,
                const float* bias, const float* residual, int64_t ldr, float residual_scale, int64_t M, int64_t N, int64_t K, int act,
                float* y, int64_t ldy, int32_t* acc_debug, cudaStream_t st) {
  SmallParams sp;
  sp.xq = xq;
  sp.wq = wq;
  sp.s_x = s_x;
  sp.s_w = s_w;
  sp.bias = bias;
  sp.residual = residual;
  sp.y = y;
  sp.acc_debug = acc_debug;
  sp.ldr = ldr;
  sp.ldy = ldy;
  sp.residual_scale = residual_scale;
  sp.s_x_kind = s_x_kind;
  sp.act = act;
  sp.M = (int)M;
  sp.N = (int)N;
  sp.K = (int)K;
  sp.a_packed = a_packed ? 1 : 0;
  sp.w_packed = w_packed ? 1 : 0;
  return launch_small_m(sp, st);
}

// The matmul for outputs of a few tiles, the columns from rq_first on quantized (rq_first = the output's columns: none).
// Arguments are checked, packed activations expanded; scratch: where packed weights that the kernel does not expand go.
int run_few_tiles(int bn, const int8_t* a_codes, const float* s_x, int s_x_kind, const void* wq, const float* s_w, const float* bias,
                  const float* residual, int64_t ldr, float residual_scale, int64_t M, int64_t N, int64_t K, int bits_w, bool static_w,
                  int act, int64_t rq_first, int bits_out, int rounding, void* q_out, float* s_out, float* y, int64_t ldy,
                  int32_t* acc_debug, uint8_t* scratch, void* exchange, uint32_t* generation, cudaStream_t st) {
  const void* b_codes = wq;
  bool b_packed = false;
  if (is_packed(bits_w)) {
    if (K % 32 == 0 && ceil_div(K, kBK) <= kWsMaxKBlocks) {
      b_packed = true;
    } else {
      const int rc = launch_unpack_int4(reinterpret_cast<const uint8_t*>(wq), N * K / 2, reinterpret_cast<int8_t*>(scratch), st);
      if (rc != AQT_OK) return rc;
      b_codes = scratch;
    }
  }
  FewTilesParams fp;
  GemmParams& p = fp.rp.g;
  p.s_x = s_x;
  p.s_w = s_w;
  p.bias = bias;
  p.residual = residual;
  p.acc_debug = acc_debug;
  p.ldr = ldr;
  p.residual_scale = residual_scale;
  p.s_x_kind = s_x_kind;
  p.act = act;
  p.M = (int)M;
  p.N = (int)N;
  p.K = (int)K;
  p.n_out = is_glu(act) ? (int)(N / 2) : (int)N;
  p.small_acc = 0;
  p.static_w = (static_w && (!is_packed(bits_w) || b_packed)) ? 1 : 0;  // not for weights unpacked into the workspace just now
  fp.rp.q_out = reinterpret_cast<uint8_t*>(q_out);
  fp.rp.s_out = s_out;
  fp.rp.exchange = reinterpret_cast<uint64_t*>(exchange);
  fp.rp.generation = generation;
  fp.rp.tag = 0;
  fp.rp.qmax_out = qmax_of(bits_out);
  fp.rp.rounding = rounding;
  fp.rp.pack_out = 0;
  fp.rq_first = (int)rq_first;
  fp.b_packed = b_packed ? 1 : 0;
  return launch_few_tiles(bn, a_codes, b_codes, y, ldy, fp, st);
}

// Codes already in int8 containers for A; B possibly packed.  ws holds B's unpacked copy.
int qmatmul_i8a(const int8_t* a_codes, const float* s_x, int s_x_kind, const void* wq, const float* s_w, const float* bias,
                const float* residual, int64_t ldr, float residual_scale, int64_t M, int64_t N, int64_t K, int bits_a, int bits_w,
                int act, float* y, int64_t ldy, int32_t* acc_debug, uint8_t* ws, cudaStream_t st, int forced_plan = kPlanNone,
                bool static_w = false) {
  if (forced_plan == kPlanNone && small_m_applies(M, K)) {
    // a few rows: weight-bandwidth-bound kernel, packed weights read as they are
    return run_small_m(a_codes, false, s_x, s_x_kind, wq, is_packed(bits_w), s_w, bias, residual, ldr, residual_scale, M, N, K, act, y, ldy,
                       acc_debug, st);
  }
  const int few_bn = gemm_plan_is_few(forced_plan)                     ? kGemmPlanBn[forced_plan]
                     : forced_plan == kPlanNone && sm_count() > 0 ? few_tiles_bn(M, N, K, act, -1, sm_count())
                                                                  : 0;
  if (few_bn != 0)
    return run_few_tiles(few_bn, a_codes, s_x, s_x_kind, wq, s_w, bias, residual, ldr, residual_scale, M, N, K, bits_w, static_w, act,
                         is_glu(act) ? N / 2 : N, 8, AQT_ROUND_NEAREST_EVEN, nullptr, nullptr, y, ldy, acc_debug, ws, nullptr, nullptr, st);
  // 4-bit weights: the weight-stationary kernel (K <= 512) sign-extends them itself in shared
  // memory after TMA staging; deeper K takes a one-off sign-extended copy in the workspace.
  const void* b_codes = wq;
  bool b_packed = false;
  if (is_packed(bits_w)) {
    const int sms = sm_count();
    if (sms <= 0) return AQT_ERR_CUDA;
    GemmShape g = {M, N, K, act, 0, false, residual != nullptr};
    g.packed = true;
    const int plan = forced_plan != kPlanNone ? forced_plan : plan_qgemm(g, sms);
    const bool ws_plan = plan == kPlanWs128E16 || plan == kPlanWs128E8;
    if (ws_plan && K % 32 == 0) {  // the packed rows must keep the 16-byte pitch bulk copies need
      b_packed = true;
    } else {
      int rc = launch_unpack_int4(reinterpret_cast<const uint8_t*>(wq), N * K / 2, reinterpret_cast<int8_t*>(ws), st);
      if (rc != AQT_OK) return rc;
      b_codes = ws;
    }
  }
  GemmParams p;
  p.s_x = s_x;
  p.s_w = s_w;
  p.bias = bias;
  p.residual = residual;
  p.acc_debug = acc_debug;
  p.ldr = ldr;
  p.residual_scale = residual_scale;
  p.s_x_kind = s_x_kind;
  p.act = act;
  p.M = (int)M;
  p.N = (int)N;
  p.K = (int)K;
  p.n_out = is_glu(act) ? (int)(N / 2) : (int)N;
  p.tiles_m = p.tiles_n = p.k_blocks = 0;
  // |acc| <= K * 2^(bits_a - 1) * 2^(bits_w - 1) for any codes the containers can hold
  p.small_acc = (K * (int64_t)(qmax_of(code_bits(bits_a)) + 1) * (qmax_of(code_bits(bits_w)) + 1) <= (1ll << 22)) ? 1 : 0;
  return launch_qgemm(a_codes, b_codes, b_packed, y, ldy, p, st, forced_plan);
}

// Workspace of aqt_ffn_fwd: [x on the device | y on the device | codes of x | scales | codes of u | scales | matmul scratch].
struct FfnLayout {
  size_t x, y, q1, s1, q2, s2, mm, total;
};
FfnLayout ffn_layout(int64_t M, int64_t d, int64_t ff, int bits_w1, int bits_w2) {
  FfnLayout L;
  L.x = 0;
  L.y = L.x + round_up((size_t)M * d * 4, 256);
  L.q1 = L.y + round_up((size_t)M * d * 4, 256);
  L.s1 = L.q1 + round_up((size_t)M * d, 256);
  L.q2 = L.s1 + round_up((size_t)M * 4, 256);
  L.s2 = L.q2 + round_up((size_t)M * ff, 256);
  L.mm = L.s2 + round_up((size_t)M * 4, 256);
  const size_t mm1 = round_up(ws_qmatmul(M, ff, d, 8, bits_w1), 256) + requant_exchange_bytes(M, ff);
  const size_t mm2 = ws_qmatmul(M, d, ff, 8, bits_w2);
  L.total = L.mm + round_up(mm1 > mm2 ? mm1 : mm2, 256);
  return L;
}

}  // namespace

extern "C" {

int aqt_version(void) { return AQT_VERSION; }

const char* aqt_status_string(int status) {
  switch (status) {
    case AQT_OK: return "ok";
    case AQT_ERR_BADARG: return "bad argument";
    case AQT_ERR_ALIGN: return "misaligned pointer or pitch";
    case AQT_ERR_UNSUPPORTED: return "unsupported device or size";
    case AQT_ERR_WORKSPACE: return "workspace missing or too small";
    case AQT_ERR_CUDA: return "CUDA call failed";
    case AQT_ERR_TIMEOUT: return "device-side wait timed out";
    default: return "unknown status";
  }
}

size_t aqt_workspace_bytes(int op, int64_t M, int64_t N, int64_t K, int bits_a, int bits_w) {
  if (M < 0 || N < 0 || K < 0) return 0;
  bits_w &= ~(AQT_STATIC_WEIGHTS | AQT_MAY_WAIT);
  if (op == AQT_OP_QMATMUL) return ws_qmatmul(M, N, K, bits_a, bits_w);
  if (op == AQT_OP_LINEAR_FWD) return ws_linear(M, N, K, bits_w);
  if (op == AQT_OP_LINEAR_WEIGHT_ONLY) return half_kind_sizes(M, N, K) ? half_layout(M, N, K).total : ws_weight_only(0, N, K, AQT_FLOAT_TF32);
  if (op == AQT_OP_LINEAR_WEIGHT_ONLY_X2) return ws_weight_only(M, N, K, AQT_FLOAT_TF32X2);
  if (op == AQT_OP_LINEAR_BWD) return bwd_workspace(M, N, K);
  if (op == AQT_OP_FFN_FWD) return ffn_layout(M, K, N, bits_w, bits_w).total;
  if (op == AQT_OP_QMATMUL_REQUANT) return round_up(ws_qmatmul(M, N, K, bits_a, bits_w), 256) + requant_exchange_bytes_few(M, N, sm_count() > 0 ? sm_count() : kDefaultSms);
  return 0;
}

// partial: nullptr, or max_partials words of scratch that save the whole-tensor scale a launch.
static int quantize_entry(const float* x, int64_t rows, int64_t cols, int64_t ld, int bits, int axis, int rounding, int pack,
                          void* q_out, float* scale_out, void* stream, float* partial, int64_t max_partials) {
  if (rows < 0 || cols < 0 || ld < cols || !quant_bits_ok(bits)) return AQT_ERR_BADARG;
  if (axis != AQT_AXIS_ROW && axis != AQT_AXIS_COL && axis != AQT_AXIS_TENSOR) return AQT_ERR_BADARG;
  if (rounding != AQT_ROUND_HALF_UP_FLOOR && rounding != AQT_ROUND_NEAREST_EVEN) return AQT_ERR_BADARG;
  if (pack != 0 && pack != 1) return AQT_ERR_BADARG;
  if (pack == 1 && (bits != 4 || cols % 2 != 0)) return AQT_ERR_BADARG;
  if (rows == 0 || cols == 0) return AQT_OK;
  if (x == nullptr || q_out == nullptr || scale_out == nullptr) return AQT_ERR_BADARG;
  if (!is_aligned(x, 4) || !is_aligned(scale_out, 4)) return AQT_ERR_ALIGN;
  int rc = check_device();
  if (rc != AQT_OK) return rc;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const int qmax = qmax_of(bits);
  if (rounding == AQT_ROUND_HALF_UP_FLOOR) {
    return pack ? launch_quantize_axis<AQT_ROUND_HALF_UP_FLOOR, true>(x, rows, cols, ld, qmax, axis, q_out, scale_out, st, partial, max_partials)
                : launch_quantize_axis<AQT_ROUND_HALF_UP_FLOOR, false>(x, rows, cols, ld, qmax, axis, q_out, scale_out, st, partial, max_partials);
  }
  return pack ? launch_quantize_axis<AQT_ROUND_NEAREST_EVEN, true>(x, rows, cols, ld, qmax, axis, q_out, scale_out, st, partial, max_partials)
              : launch_quantize_axis<AQT_ROUND_NEAREST_EVEN, false>(x, rows, cols, ld, qmax, axis, q_out, scale_out, st, partial, max_partials);
}

int aqt_quantize(const float* x, int64_t rows, int64_t cols, int64_t ld, int bits, int axis, int rounding, int pack,
                 void* q_out, float* scale_out, void* stream) {
  return quantize_entry(x, rows, cols, ld, bits, axis, rounding, pack, q_out, scale_out, stream, nullptr, 0);
}

int aqt_pack_int4(const int8_t* q, int64_t rows, int64_t cols, uint8_t* packed, void* stream) {
  if (rows < 0 || cols < 0 || cols % 2 != 0) return AQT_ERR_BADARG;
  if (rows == 0 || cols == 0) return AQT_OK;
  if (q == nullptr || packed == nullptr) return AQT_ERR_BADARG;
  int rc = check_device();
  if (rc != AQT_OK) return rc;
  return launch_pack_int4(q, rows * cols / 2, packed, reinterpret_cast<cudaStream_t>(stream));
}

int aqt_unpack_int4(const uint8_t* packed, int64_t rows, int64_t cols, int8_t* q, void* stream) {
  if (rows < 0 || cols < 0 || cols % 2 != 0) return AQT_ERR_BADARG;
  if (rows == 0 || cols == 0) return AQT_OK;
  if (q == nullptr || packed == nullptr) return AQT_ERR_BADARG;
  int rc = check_device();
  if (rc != AQT_OK) return rc;
  return launch_unpack_int4(packed, rows * cols / 2, q, reinterpret_cast<cudaStream_t>(stream));
}

static int qmatmul_entry(const void* xq, const float* s_x, int s_x_kind, const void* wq, const float* s_w, const float* bias,
                         const float* residual, int64_t ldr, float residual_scale, int64_t M, int64_t N, int64_t K, int bits_a,
                         int bits_w, int act, float* y, int64_t ldy, int32_t* acc_debug, void* workspace, size_t workspace_bytes,
                         void* stream, int forced_plan) {
  const bool static_w = (bits_w & AQT_STATIC_WEIGHTS) != 0;
  bits_w &= ~AQT_STATIC_WEIGHTS;
  int rc = validate_matmul_shape(M, N, K, bits_a, bits_w, act, s_x_kind);
  if (rc != AQT_OK) return rc;
  if (M == 0 || N == 0) return AQT_OK;
  const int64_t n_out = is_glu(act) ? N / 2 : N;
  if (xq == nullptr || s_x == nullptr || wq == nullptr || s_w == nullptr || y == nullptr) return AQT_ERR_BADARG;
  if (ldy < n_out || (residual != nullptr && ldr < n_out)) return AQT_ERR_BADARG;
  if (!is_aligned(xq, 16) || !is_aligned(wq, 16) || !is_aligned(y, 16) || !is_aligned(s_w, 16) || !is_aligned(s_x, 4) ||
      (bias != nullptr && !is_aligned(bias, 16)) || (residual != nullptr && !is_aligned(residual, 16)) ||
      (acc_debug != nullptr && !is_aligned(acc_debug, 4)))
    return AQT_ERR_ALIGN;
  if (ldy % 4 != 0 || (residual != nullptr && ldr % 4 != 0)) return AQT_ERR_ALIGN;
  const size_t need = ws_qmatmul(M, N, K, bits_a, bits_w);
  if (need > 0 && (workspace == nullptr || workspace_bytes < need)) return AQT_ERR_WORKSPACE;
  if (need > 0 && !is_aligned(workspace, 256)) return AQT_ERR_ALIGN;
  rc = check_device();
  if (rc != AQT_OK) return rc;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  uint8_t* ws = reinterpret_cast<uint8_t*>(workspace);
  if (forced_plan == kPlanNone && small_m_applies(M, K)) {
    return run_small_m(xq, is_packed(bits_a), s_x, s_x_kind, wq, is_packed(bits_w), s_w, bias, residual, ldr, residual_scale, M, N, K, act, y, ldy,
                       acc_debug, st);
  }
  const int8_t* a_codes = reinterpret_cast<const int8_t*>(xq);
  if (is_packed(bits_a)) {
    rc = launch_unpack_int4(reinterpret_cast<const uint8_t*>(xq), M * K / 2, reinterpret_cast<int8_t*>(ws), st);
    if (rc != AQT_OK) return rc;
    a_codes = reinterpret_cast<const int8_t*>(ws);
    ws += round_up((size_t)M * (size_t)K, 256);
  }
  return qmatmul_i8a(a_codes, s_x, s_x_kind, wq, s_w, bias, residual, ldr, residual_scale, M, N, K, bits_a, bits_w, act, y,
                     ldy, acc_debug, ws, st, forced_plan, static_w);
}

int aqt_qmatmul(const void* xq, const float* s_x, int s_x_kind, const void* wq, const float* s_w, const float* bias,
                const float* residual, int64_t ldr, float residual_scale, int64_t M, int64_t N, int64_t K, int bits_a,
                int bits_w, int act, float* y, int64_t ldy, int32_t* acc_debug, void* workspace, size_t workspace_bytes,
                void* stream) {
  return qmatmul_entry(xq, s_x, s_x_kind, wq, s_w, bias, residual, ldr, residual_scale, M, N, K, bits_a, bits_w, act, y, ldy, acc_debug,
                       workspace, workspace_bytes, stream, kPlanNone);
}

int aqt_qmatmul_with_plan(const char* plan, const void* xq, const float* s_x, int s_x_kind, const void* wq, const float* s_w,
                          const float* bias, const float* residual, int64_t ldr, float residual_scale, int64_t M, int64_t N,
                          int64_t K, int bits_a, int bits_w, int act, float* y, int64_t ldy, int32_t* acc_debug, void* workspace,
                          size_t workspace_bytes, void* stream) {
  const int id = gemm_plan_by_name(plan);
  if (id == kPlanNone) return AQT_ERR_BADARG;
  return qmatmul_entry(xq, s_x, s_x_kind, wq, s_w, bias, residual, ldr, residual_scale, M, N, K, bits_a, bits_w, act, y, ldy, acc_debug,
                       workspace, workspace_bytes, stream, id);
}

int aqt_plan_qmatmul(int64_t M, int64_t N, int64_t K, int bits_a, int bits_w, int act, int float_kind, int sm_count_or_0,
                     char* name_out, size_t name_bytes) {
  const bool residual = (bits_w & AQT_PLAN_RESIDUAL) != 0, weight_only = (bits_w & AQT_PLAN_WEIGHT_ONLY) != 0;
  bits_w &= ~(AQT_PLAN_RESIDUAL | AQT_PLAN_WEIGHT_ONLY);
  if (name_out == nullptr || name_bytes == 0 || M <= 0 || N <= 0 || K <= 0 || !act_ok(act)) return AQT_ERR_BADARG;
  if (!float_kind && (!bits_ok(bits_a) || !bits_ok(bits_w) || weight_only)) return AQT_ERR_BADARG;
  int sms = sm_count_or_0;
  if (sms <= 0) sms = sm_count();
  if (sms <= 0) sms = kDefaultSms;
  const char* name;
  if (!float_kind && small_m_applies(M, K)) {
    name = "small_m";
  } else if (const int bn = float_kind ? 0 : few_tiles_bn(M, N, K, act, -1, sms)) {
    name = gemm_plan_name(bn == 32 ? kPlanFew32 : (bn == 64 ? kPlanFew64 : kPlanFew128));
  } else if (weight_only && half_kind_applies(M, N, K, act, sms)) {
    name = "pair256s4e8f16";
  } else {
    GemmShape g = {M, N, float_kind ? 4 * K : K, act, float_kind ? 1 : 0, false, residual};
    g.packed = !float_kind && is_packed(bits_w) && K % 32 == 0;  // (other rows of packed codes are expanded first, and then int8 ones)
    name = gemm_plan_name(plan_qgemm(g, sms));
  }
  if (strlen(name) + 1 > name_bytes) return AQT_ERR_BADARG;
  memcpy(name_out, name, strlen(name) + 1);
  return AQT_OK;
}

int aqt_plan_qmatmul_requant(int64_t first, int64_t M, int64_t N, int64_t K, int bits_a, int bits_w, int act, int with_y, int pack_out,
                             size_t workspace_bytes, int sm_count_or_0, char* name_out, size_t name_bytes) {
  const bool may_wait = (bits_w & AQT_MAY_WAIT) != 0;
  bits_w &= ~(AQT_STATIC_WEIGHTS | AQT_MAY_WAIT);
  if (name_out == nullptr || name_bytes == 0 || M <= 0 || N <= 0 || first < 0 || first >= N || first % 16 != 0) return AQT_ERR_BADARG;
  const int rc = validate_matmul_shape(M, N, K, bits_a, bits_w, act, AQT_SCALE_ROW);
  if (rc != AQT_OK) return rc;
  if ((is_glu(act) ? N / 2 : N) % (pack_out ? 32 : 16) != 0 || (first > 0 && (act != AQT_ACT_NONE || pack_out || !with_y))) return AQT_ERR_BADARG;
  int sms = sm_count_or_0;
  if (sms <= 0) sms = sm_count();
  if (sms <= 0) sms = kDefaultSms;
  const size_t mm_bytes = round_up(ws_qmatmul(M, N, K, bits_a, bits_w), 256);
  if (workspace_bytes == 0) workspace_bytes = mm_bytes + requant_exchange_bytes_few(M, N, sms);
  if (workspace_bytes < mm_bytes + requant_exchange_bytes(M, N)) return AQT_ERR_WORKSPACE;
  RequantRoute r = {kRequantFew, first > 0 ? requant_from_bn(first, M, N, K, bits_a, workspace_bytes - mm_bytes, sms) : 0};
  if (r.few_bn == 0) {
    const size_t room = workspace_bytes - round_up(ws_qmatmul(M, N - first, K, bits_a, bits_w), 256);
    r = requant_route(M, N - first, K, act, with_y != 0, pack_out != 0, may_wait || first > 0, room, sms);
  }
  const char* name = nullptr;
  switch (r.form) {
    case kRequantRefused: return AQT_ERR_UNSUPPORTED;
    case kRequantFew: name = gemm_plan_name(r.few_bn == 32 ? kPlanFew32 : (r.few_bn == 64 ? kPlanFew64 : kPlanFew128)); break;
    case kRequantWs: name = "ws128"; break;
    case kRequantPair: name = gemm_plan_name(rowquant_plan(M, N - first, K, sms)); break;
    case kRequantTwoKernels: name = "two_kernels"; break;
  }
  if (strlen(name) + 1 > name_bytes) return AQT_ERR_BADARG;
  memcpy(name_out, name, strlen(name) + 1);
  return AQT_OK;
}

int aqt_qmatmul_requant(const void* xq, const float* s_x, int s_x_kind, const void* wq, const float* s_w, const float* bias,
                        const float* residual, int64_t ldr, float residual_scale, int64_t M, int64_t N, int64_t K, int bits_a,
                        int bits_w, int act, int bits_out, int rounding, int pack_out, void* q_out, float* s_out, float* y,
                        int64_t ldy, void* workspace, size_t workspace_bytes, void* stream) {
  const int static_w = (bits_w & AQT_STATIC_WEIGHTS) ? 1 : 0;
  const bool may_wait = (bits_w & AQT_MAY_WAIT) != 0;
  bits_w &= ~(AQT_STATIC_WEIGHTS | AQT_MAY_WAIT);
  int rc = validate_matmul_shape(M, N, K, bits_a, bits_w, act, s_x_kind);
  if (rc != AQT_OK) return rc;
  if (!quant_bits_ok(bits_out) || (pack_out != 0 && pack_out != 1) || (pack_out == 1 && bits_out != 4)) return AQT_ERR_BADARG;
  if (rounding != AQT_ROUND_HALF_UP_FLOOR && rounding != AQT_ROUND_NEAREST_EVEN) return AQT_ERR_BADARG;
  const int64_t n_out = is_glu(act) ? N / 2 : N;
  if (n_out % (pack_out ? 32 : 16) != 0) return AQT_ERR_BADARG;  // rows of codes keep a 16-byte pitch
  if (residual != nullptr && y == nullptr) return AQT_ERR_BADARG;
  if (M == 0 || N == 0) return AQT_OK;
  if (xq == nullptr || s_x == nullptr || wq == nullptr || s_w == nullptr || q_out == nullptr || s_out == nullptr) return AQT_ERR_BADARG;
  if (y != nullptr && (ldy < n_out || ldy % 4 != 0)) return AQT_ERR_BADARG;
  if (residual != nullptr && (ldr < n_out || ldr % 4 != 0)) return AQT_ERR_BADARG;
  if (!is_aligned(xq, 16) || !is_aligned(wq, 16) || !is_aligned(q_out, 16) || !is_aligned(s_w, 16) || !is_aligned(s_x, 4) ||
      !is_aligned(s_out, 4) || (y != nullptr && !is_aligned(y, 16)) || (bias != nullptr && !is_aligned(bias, 16)) ||
      (residual != nullptr && !is_aligned(residual, 16)))
    return AQT_ERR_ALIGN;
  const size_t mm_bytes = round_up(ws_qmatmul(M, N, K, bits_a, bits_w), 256);
  const size_t need = mm_bytes + requant_exchange_bytes(M, N);
  if (workspace == nullptr || workspace_bytes < need) return AQT_ERR_WORKSPACE;
  if (!is_aligned(workspace, 256)) return AQT_ERR_ALIGN;
  rc = check_device();
  if (rc != AQT_OK) return rc;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  uint8_t* ws = reinterpret_cast<uint8_t*>(workspace);

  const int sms = sm_count();
  if (sms <= 0) return AQT_ERR_CUDA;
  const RequantRoute route = requant_route(M, N, K, act, y != nullptr, pack_out != 0, may_wait, workspace_bytes - mm_bytes, sms);
  if (route.form == kRequantRefused) return AQT_ERR_UNSUPPORTED;
  if (route.form == kRequantFew) {
    const int8_t* a_codes = reinterpret_cast<const int8_t*>(xq);
    if (is_packed(bits_a)) {
      rc = launch_unpack_int4(reinterpret_cast<const uint8_t*>(xq), M * K / 2, reinterpret_cast<int8_t*>(ws), st);
      if (rc != AQT_OK) return rc;
      a_codes = reinterpret_cast<const int8_t*>(ws);
      ws += round_up((size_t)M * (size_t)K, 256);
    }
    return run_few_tiles(route.few_bn, a_codes, s_x, s_x_kind, wq, s_w, bias, residual, ldr, residual_scale, M, N, K, bits_w, static_w != 0, act, 0,
                             bits_out, rounding, q_out, s_out, y, ldy, nullptr, ws, reinterpret_cast<uint8_t*>(workspace) + mm_bytes,
                             generation_counters(workspace, workspace_bytes), st);
  }
  if (route.form == kRequantPair) {
    // Deep K (the second feed-forward layers): the CTA-pair kernel with the row-quantizing epilogue
    const int8_t* a_codes = reinterpret_cast<const int8_t*>(xq);
    if (is_packed(bits_a)) {
      rc = launch_unpack_int4(reinterpret_cast<const uint8_t*>(xq), M * K / 2, reinterpret_cast<int8_t*>(ws), st);
      if (rc != AQT_OK) return rc;
      a_codes = reinterpret_cast<const int8_t*>(ws);
      ws += round_up((size_t)M * (size_t)K, 256);
    }
    const void* b_codes = wq;
    if (is_packed(bits_w)) {
      rc = launch_unpack_int4(reinterpret_cast<const uint8_t*>(wq), N * K / 2, reinterpret_cast<int8_t*>(ws), st);
      if (rc != AQT_OK) return rc;
      b_codes = ws;
    }
    GemmParams p;
    p.s_x = s_x;
    p.s_w = s_w;
    p.bias = bias;
    p.residual = residual;
    p.acc_debug = nullptr;
    p.ldr = ldr;
    p.residual_scale = residual_scale;
    p.s_x_kind = s_x_kind;
    p.act = act;
    p.M = (int)M;
    p.N = (int)N;
    p.K = (int)K;
    p.n_out = (int)N;
    p.tiles_m = p.tiles_n = p.k_blocks = 0;
    p.small_acc = (K * (int64_t)(qmax_of(code_bits(bits_a)) + 1) * (qmax_of(code_bits(bits_w)) + 1) <= (1ll << 22)) ? 1 : 0;
    p.q_out = reinterpret_cast<uint8_t*>(q_out);
    p.s_out = s_out;
    p.exchange = reinterpret_cast<uint64_t*>(reinterpret_cast<uint8_t*>(workspace) + mm_bytes);
    p.generation = generation_counters(workspace, workspace_bytes);
    p.tag = next_launch_tag();
    p.qmax_out = qmax_of(bits_out);
    p.rounding = rounding;
    p.has_y = y != nullptr ? 1 : 0;
    return launch_qgemm_rowquant(rowquant_plan(M, N, K, sms), a_codes, b_codes, y, ldy, p, st);
  }
  if (route.form == kRequantTwoKernels) {
    rc = aqt_qmatmul(xq, s_x, s_x_kind, wq, s_w, bias, residual, ldr, residual_scale, M, N, K, bits_a, bits_w, act, y, ldy, nullptr,
                     workspace, mm_bytes, stream);
    if (rc != AQT_OK) return rc;
    return aqt_quantize(y, M, n_out, ldy, bits_out, AQT_AXIS_ROW, rounding, pack_out, q_out, s_out, stream);
  }

  const int8_t* a_codes = reinterpret_cast<const int8_t*>(xq);
  if (is_packed(bits_a)) {
    rc = launch_unpack_int4(reinterpret_cast<const uint8_t*>(xq), M * K / 2, reinterpret_cast<int8_t*>(ws), st);
    if (rc != AQT_OK) return rc;
    a_codes = reinterpret_cast<const int8_t*>(ws);
    ws += round_up((size_t)M * (size_t)K, 256);
  }
  const void* b_codes = wq;
  bool b_packed = false;
  if (is_packed(bits_w)) {
    if (K % 32 == 0 && K <= 512) {  // the deep-K form (512 < K <= 1024) has no room to unpack in shared memory
      b_packed = true;
    } else {
      rc = launch_unpack_int4(reinterpret_cast<const uint8_t*>(wq), N * K / 2, reinterpret_cast<int8_t*>(ws), st);
      if (rc != AQT_OK) return rc;
      b_codes = ws;
    }
  }
  RequantParams rp;
  GemmParams& p = rp.g;
  p.s_x = s_x;
  p.s_w = s_w;
  p.bias = bias;
  p.residual = residual;
  p.acc_debug = nullptr;
  p.ldr = ldr;
  p.residual_scale = residual_scale;
  p.s_x_kind = s_x_kind;
  p.act = act;
  p.M = (int)M;
  p.N = (int)N;
  p.K = (int)K;
  p.n_out = (int)n_out;
  p.tiles_m = p.tiles_n = p.k_blocks = 0;
  p.small_acc = 0;
  p.static_w = (static_w && (!is_packed(bits_w) || b_packed)) ? 1 : 0;  // not for weights unpacked into the workspace just now
  rp.q_out = nullptr;
  rp.s_out = s_out;
  rp.exchange = nullptr;
  rp.generation = generation_counters(workspace, workspace_bytes);
  rp.qmax_out = qmax_of(bits_out);
  rp.rounding = rounding;
  rp.pack_out = pack_out;
  return launch_requant(a_codes, b_codes, b_packed, q_out, y, ldy, rp, reinterpret_cast<uint8_t*>(workspace) + mm_bytes, st);
}

int aqt_qmatmul_requant_from(int64_t first, const void* xq, const float* s_x, int s_x_kind, const void* wq, const float* s_w, const float* bias,
                             int64_t M, int64_t N, int64_t K, int bits_a, int bits_w, int bits_out, int rounding, void* q_out, float* s_out,
                             float* y, int64_t ldy, void* workspace, size_t workspace_bytes, void* stream) {
  const int static_w = (bits_w & AQT_STATIC_WEIGHTS) ? 1 : 0, width = bits_w & ~(AQT_STATIC_WEIGHTS | AQT_MAY_WAIT);
  int rc = validate_matmul_shape(M, N, K, bits_a, width, AQT_ACT_NONE, s_x_kind);
  if (rc != AQT_OK) return rc;
  if (first < 0 || first >= N || first % 16 != 0 || N % 16 != 0 || !quant_bits_ok(bits_out)) return AQT_ERR_BADARG;
  if (rounding != AQT_ROUND_HALF_UP_FLOOR && rounding != AQT_ROUND_NEAREST_EVEN) return AQT_ERR_BADARG;
  if (M == 0) return AQT_OK;
  if (xq == nullptr || s_x == nullptr || wq == nullptr || s_w == nullptr || q_out == nullptr || s_out == nullptr || y == nullptr) return AQT_ERR_BADARG;
  if (ldy < N || ldy % 4 != 0) return AQT_ERR_BADARG;
  if (!is_aligned(xq, 16) || !is_aligned(wq, 16) || !is_aligned(q_out, 16) || !is_aligned(s_w, 16) || !is_aligned(s_x, 4) || !is_aligned(s_out, 4) ||
      !is_aligned(y, 16) || (bias != nullptr && !is_aligned(bias, 16)))
    return AQT_ERR_ALIGN;
  const size_t mm_bytes = round_up(ws_qmatmul(M, N, K, bits_a, width), 256);
  if (workspace == nullptr || workspace_bytes < mm_bytes + requant_exchange_bytes(M, N)) return AQT_ERR_WORKSPACE;
  if (!is_aligned(workspace, 256)) return AQT_ERR_ALIGN;
  rc = check_device();
  if (rc != AQT_OK) return rc;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const int sms = sm_count();
  if (sms <= 0) return AQT_ERR_CUDA;
  const int bn = requant_from_bn(first, M, N, K, bits_a, workspace_bytes - mm_bytes, sms);
  if (bn != 0)
    return run_few_tiles(bn, reinterpret_cast<const int8_t*>(xq), s_x, s_x_kind, wq, s_w, bias, nullptr, 0, 0.0f, M, N, K, width, static_w != 0,
                             AQT_ACT_NONE, first, bits_out, rounding, q_out, s_out, y, ldy, nullptr, reinterpret_cast<uint8_t*>(workspace),
                             reinterpret_cast<uint8_t*>(workspace) + mm_bytes, generation_counters(workspace, workspace_bytes), st);
  // the two parts one after the other (row `first` of the weights keeps the 16-byte alignment: `first` and K are multiples of 16)
  if (first > 0) {
    rc = aqt_qmatmul(xq, s_x, s_x_kind, wq, s_w, bias, nullptr, 0, 0.0f, M, first, K, bits_a, width, AQT_ACT_NONE, y, ldy, nullptr, workspace,
                     workspace_bytes, stream);
    if (rc != AQT_OK) return rc;
  }
  const uint8_t* w_rest = reinterpret_cast<const uint8_t*>(wq) + first * (is_packed(width) ? K / 2 : K);
  return aqt_qmatmul_requant(xq, s_x, s_x_kind, w_rest, s_w + first, bias == nullptr ? nullptr : bias + first, nullptr, 0, 0.0f, M, N - first, K,
                             bits_a, bits_w | AQT_MAY_WAIT, AQT_ACT_NONE, bits_out, rounding, 0, q_out, s_out, y + first, ldy, workspace, workspace_bytes, stream);
}

int aqt_linear_fwd(const float* x, int64_t ldx, const void* wq, const float* s_w, const float* bias, const float* residual,
                   int64_t ldr, float residual_scale, int64_t M, int64_t N, int64_t K, int bits_a, int bits_w,
                   int a_scale_kind, int rounding, int act, float* y, int64_t ldy, void* workspace, size_t workspace_bytes,
                   void* stream) {
  bits_w &= ~AQT_STATIC_WEIGHTS;
  int rc = validate_matmul_shape(M, N, K, bits_a, bits_w, act, a_scale_kind);
  if (rc != AQT_OK) return rc;
  if (rounding != AQT_ROUND_HALF_UP_FLOOR && rounding != AQT_ROUND_NEAREST_EVEN) return AQT_ERR_BADARG;
  if (!quant_bits_ok(bits_a)) return AQT_ERR_BADARG;  // the width the activations are quantized to
  if (M == 0 || N == 0) return AQT_OK;
  const int64_t n_out = is_glu(act) ? N / 2 : N;
  if (x == nullptr || wq == nullptr || s_w == nullptr || y == nullptr) return AQT_ERR_BADARG;
  if (ldx < K || ldy < n_out || (residual != nullptr && ldr < n_out)) return AQT_ERR_BADARG;
  if (!is_aligned(x, 4) || !is_aligned(wq, 16) || !is_aligned(y, 16) || !is_aligned(s_w, 16) ||
      (bias != nullptr && !is_aligned(bias, 16)) || (residual != nullptr && !is_aligned(residual, 16)))
    return AQT_ERR_ALIGN;
  if (ldy % 4 != 0 || (residual != nullptr && ldr % 4 != 0)) return AQT_ERR_ALIGN;
  const size_t need = ws_linear(M, N, K, bits_w);
  if (workspace == nullptr || workspace_bytes < need) return AQT_ERR_WORKSPACE;
  if (!is_aligned(workspace, 256)) return AQT_ERR_ALIGN;
  rc = check_device();
  if (rc != AQT_OK) return rc;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  uint8_t* ws = reinterpret_cast<uint8_t*>(workspace);
  int8_t* codes = reinterpret_cast<int8_t*>(ws);
  float* s_x = reinterpret_cast<float*>(ws + round_up((size_t)M * (size_t)K, 256));
  uint8_t* ws_mm = ws + round_up((size_t)M * (size_t)K, 256) + round_up((size_t)M * 4, 256);
  if (M <= kLinSmallMaxRows) {
    // a few rows: both steps in one launch
    const LinSmallParams sp = {x, reinterpret_cast<const uint8_t*>(wq), s_w, bias, residual, y, ldx, ldr, ldy, residual_scale, (int32_t)M, (int32_t)N,
                               (int32_t)K, act, qmax_of(bits_a), rounding, a_scale_kind == AQT_SCALE_TENSOR, 0, 0};
    if (linear_small_applies(sp, is_packed(bits_w))) return launch_linear_small(sp, is_packed(bits_w), st);
  }
  // Step 1 (Fig. 2): dynamic quantization of the activations over K; 4-bit codes stay in int8
  // containers between the two kernels, which is what the figure's cast produces.
  const int axis = a_scale_kind == AQT_SCALE_ROW ? AQT_AXIS_ROW : AQT_AXIS_TENSOR;
  // (one scale: the other words of its area, at least 63, are scratch for the quantizer; with M - 1 of them two rows had one
  // block look for their maximum, 285 against 267 us for 2 x 131 072 -> 256)
  const bool one_scale = a_scale_kind == AQT_SCALE_TENSOR;
  rc = quantize_entry(x, M, K, ldx, bits_a, axis, rounding, 0, codes, s_x, stream, one_scale ? s_x + 1 : nullptr,
                      (int64_t)(round_up((size_t)M * 4, 256) / 4) - 1);
  if (rc != AQT_OK) return rc;
  // Step 2: integer matmul + de-quantizing epilogue.  (The weights were complete before the quantizer was enqueued.)
  return qmatmul_i8a(codes, s_x, a_scale_kind, wq, s_w, bias, residual, ldr, residual_scale, M, N, K, bits_a, bits_w, act, y,
                     ldy, nullptr, ws_mm, st, kPlanNone, true);
}

int aqt_linear_fwd_host(const float* x, int x_on_host, const void* wq, const float* s_w, const float* bias, int64_t M,
                        int64_t N, int64_t K, int bits_a, int bits_w, int a_scale_kind, int rounding, int act, float* y,
                        int y_on_host, void* workspace, size_t workspace_bytes, void* stream) {
  int rc = validate_matmul_shape(M, N, K, bits_a, bits_w, act, a_scale_kind);
  if (rc != AQT_OK) return rc;
  if (M == 0 || N == 0) return AQT_OK;
  if (x == nullptr || y == nullptr) return AQT_ERR_BADARG;
  const int64_t n_out = is_glu(act) ? N / 2 : N;
  const size_t layer = round_up(ws_linear(M, N, K, bits_w), 256);
  const size_t xb = x_on_host ? round_up((size_t)M * K * 4, 256) : 0;
  const size_t yb = y_on_host ? round_up((size_t)M * n_out * 4, 256) : 0;
  if (workspace == nullptr || workspace_bytes < layer + xb + yb) return AQT_ERR_WORKSPACE;
  if (!is_aligned(workspace, 256)) return AQT_ERR_ALIGN;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  uint8_t* ws = reinterpret_cast<uint8_t*>(workspace);
  float* x_copy = reinterpret_cast<float*>(ws + layer);
  const float* x_dev = x_on_host ? x_copy : x;
  float* y_dev = y_on_host ? reinterpret_cast<float*>(ws + layer + xb) : y;
  // (one scale for the whole tensor needs every row before the first product)
  return run_between_host_copies(x_on_host ? x : nullptr, x_copy, (size_t)K * 4, y_dev, y_on_host ? y : nullptr, (size_t)n_out * 4, M, st,
                                 a_scale_kind == AQT_SCALE_ROW, [&](int64_t r0, int64_t rows) {
                                   return aqt_linear_fwd(x_dev + r0 * K, K, wq, s_w, bias, nullptr, 0, 0.0f, rows, N, K, bits_a, bits_w,
                                                         a_scale_kind, rounding, act, y_dev + r0 * n_out, n_out, ws, layer, stream);
                                 });
}

int aqt_chain_fwd(const float* x, int64_t ldx, int64_t M, const aqt_chain_layer* layers, int n_layers, int rounding, void* stream) {
  if (M < 0 || n_layers < 0 || (n_layers > 0 && layers == nullptr)) return AQT_ERR_BADARG;
  if (rounding != AQT_ROUND_HALF_UP_FLOOR && rounding != AQT_ROUND_NEAREST_EVEN) return AQT_ERR_BADARG;
  if (M == 0 || n_layers == 0) return AQT_OK;
  if (n_layers > AQT_CHAIN_MAX_LAYERS || M >= (1ll << 24)) return AQT_ERR_UNSUPPORTED;
  if (x == nullptr) return AQT_ERR_BADARG;
  if (!is_aligned(x, 16) || ldx % 4 != 0) return AQT_ERR_ALIGN;
  ChainParams<kChainMaxSteps> p;
  p.x = x;
  p.ldx = ldx;
  p.M = (int32_t)M;
  p.K0 = layers[0].K;
  p.n_steps = n_layers;
  p.rounding = rounding;
  p.in_qmax = qmax_of(layers[0].bits_a);
  p.h_cols = 0;
  if (ldx < p.K0) return AQT_ERR_BADARG;
  int64_t width = p.K0;  // of the current input
  int head = 0;          // first layer that reads it
  int feeder = -1;       // layer whose output it is
  for (int i = 0; i < n_layers; ++i) {
    const aqt_chain_layer& l = layers[i];
    int rc = validate_matmul_shape(M, l.N, l.K, l.bits_a, l.bits_w, l.act, AQT_SCALE_ROW);
    if (rc != AQT_OK) return rc;
    const int64_t n_out = is_glu(l.act) ? l.N / 2 : l.N;
    if (!quant_bits_ok(l.bits_a) || l.K != width || l.N == 0) return AQT_ERR_BADARG;
    if (l.wq == nullptr || l.s_w == nullptr || (l.y != nullptr && l.ldy < n_out)) return AQT_ERR_BADARG;
    if (!is_aligned(l.wq, 16) || !is_aligned(l.s_w, 4) || (l.y != nullptr && (!is_aligned(l.y, 16) || l.ldy % 4 != 0))) return AQT_ERR_ALIGN;
    ChainStep& s = p.steps[i];
    s.w = reinterpret_cast<const uint8_t*>(l.wq);
    s.s_w = l.s_w;
    s.bias = l.bias;
    s.y = l.y;
    s.ldy = (int32_t)l.ldy;
    s.N = l.N;
    s.K = l.K;
    s.rs = l.residual_scale;
    s.flags = (uint32_t)l.act | (is_packed(l.bits_w) ? kChainPacked : 0u) | ((l.flags & AQT_CHAIN_SIDE) ? kChainSide : 0u) |
              ((l.flags & AQT_CHAIN_ADD) ? kChainAdd : 0u);
    if (l.ldy >= (1ll << 31) || !chain_step_ok(s)) return AQT_ERR_UNSUPPORTED;
    if (l.bits_a != layers[head].bits_a || is_packed(l.bits_w) != is_packed(layers[head].bits_w)) return AQT_ERR_UNSUPPORTED;
    if (i == head && feeder >= 0 && l.bits_a == 4) p.steps[feeder].flags |= kChainOut4;
    if (l.flags & AQT_CHAIN_ADD) {
      if (n_out != p.K0) return AQT_ERR_UNSUPPORTED;
      p.h_cols = p.K0 / kChainCtas;
    }
    if (!(l.flags & AQT_CHAIN_SIDE)) {
      width = n_out;
      head = i + 1;
      feeder = i;
    }
  }
  int rc = check_device();
  if (rc != AQT_OK) return rc;
  return launch_chain(p, reinterpret_cast<cudaStream_t>(stream));
}

int aqt_ffn_fwd(const float* x, int x_on_host, const void* w1q, const float* s_w1, const float* bias1, int bits_w1,
                const void* w2q, const float* s_w2, const float* bias2, int bits_w2, int64_t M, int64_t d, int64_t ff,
                int bits_a, int rounding, int act, float* y, int y_on_host, void* workspace, size_t workspace_bytes,
                void* stream) {
  bits_w1 &= ~AQT_STATIC_WEIGHTS;
  bits_w2 &= ~AQT_STATIC_WEIGHTS;
  if (M < 0 || d <= 0 || ff <= 0 || !quant_bits_ok(bits_a) || !bits_ok(bits_w1) || !bits_ok(bits_w2)) return AQT_ERR_BADARG;
  if (act != AQT_ACT_NONE && act != AQT_ACT_SWISH) return AQT_ERR_BADARG;
  if (rounding != AQT_ROUND_HALF_UP_FLOOR && rounding != AQT_ROUND_NEAREST_EVEN) return AQT_ERR_BADARG;
  if (M == 0) return AQT_OK;
  if (x == nullptr || y == nullptr || w1q == nullptr || w2q == nullptr || s_w1 == nullptr || s_w2 == nullptr) return AQT_ERR_BADARG;
  const FfnLayout L = ffn_layout(M, d, ff, bits_w1, bits_w2);
  if (workspace == nullptr || workspace_bytes < L.total) return AQT_ERR_WORKSPACE;
  if (!is_aligned(workspace, 256)) return AQT_ERR_ALIGN;
  int rc = check_device();
  if (rc != AQT_OK) return rc;
  if (!requant_applies(M, ff, d, act, false, false, sm_count() > 0 ? sm_count() : kDefaultSms)) return AQT_ERR_UNSUPPORTED;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  uint8_t* ws = reinterpret_cast<uint8_t*>(workspace);
  float* x_copy = reinterpret_cast<float*>(ws + L.x);
  float* y_dev = y_on_host ? reinterpret_cast<float*>(ws + L.y) : y;
  const bool chain = M <= AQT_CHAIN_MAX_ROWS;
  if (x_on_host && (size_t)M * d * 4 < (chain ? kReadInPlaceBytesChain : kReadInPlaceBytes) && is_aligned(x, 16)) {
    if (const void* mapped = pinned_on_device(x, (size_t)M * d * 4)) {
      x = reinterpret_cast<const float*>(mapped);
      x_on_host = 0;
    }
  }
  const float* x_dev = x_on_host ? x_copy : x;
  if (chain) {
    // a few rows: both layers in one launch, which writes the result over the bus itself (us a call, copied or not, d =
    // 512: 16 rows 24 / 23, 64 rows 36 / 26)
    float* y_out = y_on_host && is_aligned(y, 16) ? reinterpret_cast<float*>(pinned_on_device(y, (size_t)M * d * 4)) : nullptr;
    const bool y_copied = y_on_host && y_out == nullptr;
    if (y_out == nullptr) y_out = y_dev;
    if (x_on_host) AQT_RETURN_IF_CUDA(cudaMemcpyAsync(x_copy, x, (size_t)M * d * 4, cudaMemcpyHostToDevice, st));
    const aqt_chain_layer pair[2] = {
        {w1q, s_w1, bias1, nullptr, 0, (int32_t)ff, (int32_t)d, bits_w1, bits_a, act, 0, 0.0f, 0},
        {w2q, s_w2, bias2, y_out, d, (int32_t)d, (int32_t)ff, bits_w2, bits_a, AQT_ACT_NONE, 0, 0.0f, 0}};
    rc = aqt_chain_fwd(x_dev, d, M, pair, 2, rounding, stream);
    if (rc == AQT_OK && y_copied) AQT_RETURN_IF_CUDA(cudaMemcpyAsync(y, y_dev, (size_t)M * d * 4, cudaMemcpyDeviceToHost, st));
    if (rc != AQT_ERR_UNSUPPORTED && rc != AQT_ERR_ALIGN) return rc;
  }
  const size_t mm_bytes = L.total - L.mm;
  const int bits_mm = bits_a == 8 ? 8 : AQT_BITS_4_UNPACKED;
  const int sms = sm_count() > 0 ? sm_count() : kDefaultSms;
  return run_between_host_copies(x_on_host ? x : nullptr, x_copy, (size_t)d * 4, y_dev, y_on_host ? y : nullptr, (size_t)d * 4, M, st, true,
                                 [&](int64_t r0, int64_t rows) {
    const float* xr = x_dev + r0 * d;
    float* yr = y_dev + r0 * d;
    // Fig. 2 on the input rows; first matmul with the rows of u = act(W1 x) quantized in its epilogue
    // (4-bit codes stay in int8 containers between the kernels); second matmul.
    int8_t* q1 = reinterpret_cast<int8_t*>(ws + L.q1) + r0 * d;
    float* s1 = reinterpret_cast<float*>(ws + L.s1) + r0;
    int8_t* q2 = reinterpret_cast<int8_t*>(ws + L.q2) + r0 * ff;
    float* s2 = reinterpret_cast<float*>(ws + L.s2) + r0;
    // (the work ahead of the first matmul is this quantizer, enqueued after the weights were complete or were ordered so)
    int rc = aqt_quantize(xr, rows, d, d, bits_a, AQT_AXIS_ROW, rounding, 0, q1, s1, stream);
    if (rc != AQT_OK) return rc;
    rc = aqt_qmatmul_requant(q1, s1, AQT_SCALE_ROW, w1q, s_w1, bias1, nullptr, 0, 0.0f, rows, ff, d, bits_mm, bits_w1 | AQT_STATIC_WEIGHTS, act, bits_a,
                             rounding, 0, q2, s2, nullptr, 0, ws + L.mm, mm_bytes, stream);
    if (rc != AQT_OK) return rc;
    // The codes of u are still in L2: narrower tiles that read them twice, and start and drain sooner, then beat the tile
    // over all 512 columns (12 800 x 512: 62.3 -> 59.0 us the pair)
    const bool wide = !small_m_applies(rows, ff) && plan_qgemm(GemmShape{rows, d, ff, AQT_ACT_NONE, 0, false}, sms) == kPlanPair512S3E16;
    return qmatmul_entry(q2, s2, AQT_SCALE_ROW, w2q, s_w2, bias2, nullptr, 0, 0.0f, rows, d, ff, bits_mm, bits_w2 | AQT_STATIC_WEIGHTS, AQT_ACT_NONE, yr, d, nullptr,
                         ws + L.mm, mm_bytes, stream, wide ? kPlanPair256S4E8 : kPlanNone);
  });
}

int aqt_linear_fwd_weight_only(const float* x, int64_t ldx, const void* wq, const float* s_w, const float* bias,
                               const float* residual, int64_t ldr, float residual_scale, int64_t M, int64_t N, int64_t K,
                               int bits_w, int precision, int act, float* y, int64_t ldy, void* workspace,
                               size_t workspace_bytes, void* stream) {
  if (M < 0 || N < 0 || K <= 0 || !bits_ok(bits_w) || !act_ok(act)) return AQT_ERR_BADARG;
  if (precision != AQT_FLOAT_TF32 && precision != AQT_FLOAT_TF32X2) return AQT_ERR_BADARG;
  if (K % 4 != 0 || N % 4 != 0 || (is_glu(act) && N % 8 != 0)) return AQT_ERR_BADARG;
  if (M >= (1ll << 31) || N >= (1ll << 31) || K >= (1ll << 28) || M * N >= (1ll << 40)) return AQT_ERR_UNSUPPORTED;
  if (M == 0 || N == 0) return AQT_OK;
  const int64_t n_out = is_glu(act) ? N / 2 : N;
  if (x == nullptr || wq == nullptr || s_w == nullptr || y == nullptr) return AQT_ERR_BADARG;
  if (ldx < K || ldy < n_out || (residual != nullptr && ldr < n_out)) return AQT_ERR_BADARG;
  if (!is_aligned(x, 16) || !is_aligned(wq, 16) || !is_aligned(y, 16) || !is_aligned(s_w, 16) ||
      (bias != nullptr && !is_aligned(bias, 16)) || (residual != nullptr && !is_aligned(residual, 16)))
    return AQT_ERR_ALIGN;
  if (ldx % 4 != 0 || ldy % 4 != 0 || (residual != nullptr && ldr % 4 != 0)) return AQT_ERR_ALIGN;
  const size_t need = ws_weight_only(M, N, K, precision);
  if (workspace == nullptr || workspace_bytes < need) return AQT_ERR_WORKSPACE;
  if (!is_aligned(workspace, 256)) return AQT_ERR_ALIGN;
  int rc = check_device();
  if (rc != AQT_OK) return rc;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  {
    // few rows: one launch
    const WoSmallParams sp = {x, reinterpret_cast<const uint8_t*>(wq), s_w, bias, residual, y, ldx, ldr, ldy, residual_scale, (int32_t)M, (int32_t)N,
                              (int32_t)K, act};
    const int terms = precision == AQT_FLOAT_TF32X2 ? 3 : 2;
    if (weight_only_small_applies(sp, terms)) return launch_weight_only_small(sp, is_packed(bits_w), terms, st);
  }
  // the weights converted to float (Section 4.1): the codes as binary32 integers, once per call;
  // the channel scales stay outside the sum and are applied to the accumulators.
  float* w_f = reinterpret_cast<float*>(workspace);
  const float* a_f = x;
  int64_t k_mm = K, a_pitch = 4 * ldx;
  if (precision == AQT_FLOAT_TF32X2) {
    // x = hi + lo with hi a tf32 value: one matmul over [hi | lo] against [w | w]
    float* x2 = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(workspace) + round_up((size_t)N * (size_t)K * 8, 256));
    rc = launch_codes_to_float_twice(wq, is_packed(bits_w), N, K, w_f, st);
    if (rc != AQT_OK) return rc;
    rc = launch_split_hi_lo(x, ldx, M, K, x2, st);
    if (rc != AQT_OK) return rc;
    a_f = x2;
    k_mm = 2 * K;
    a_pitch = 8 * K;
  }
  const HalfLayout H = half_layout(M, N, K);
  const int sms = sm_count();
  if (sms <= 0) return AQT_ERR_CUDA;
  const bool half = precision == AQT_FLOAT_TF32 && workspace_bytes >= H.total && half_kind_applies(M, N, K, act, sms);
  uint8_t* ws = reinterpret_cast<uint8_t*>(workspace);
  const void* b_mm = w_f;
  if (half) {
    rc = launch_half_operands(x, ldx, M, K, reinterpret_cast<__half*>(ws + H.x_h), reinterpret_cast<float*>(ws + H.inv), wq, is_packed(bits_w), N * K, w_f,
                              reinterpret_cast<__half*>(ws + H.w_h), st);
    if (rc != AQT_OK) return rc;
    b_mm = ws + H.w_h;
  } else if (precision == AQT_FLOAT_TF32) {
    rc = launch_codes_to_float(wq, is_packed(bits_w), N * K, w_f, st);
    if (rc != AQT_OK) return rc;
  }
  GemmParams p;
  p.s_x = nullptr;
  p.s_w = s_w;
  p.bias = bias;
  p.residual = residual;
  p.acc_debug = nullptr;
  p.ldr = ldr;
  p.residual_scale = residual_scale;
  p.s_x_kind = AQT_SCALE_TENSOR;
  p.act = act;
  p.M = (int)M;
  p.N = (int)N;
  p.K = (int)(4 * k_mm);
  p.kind = 1;
  p.a_pitch = a_pitch;
  p.n_out = (int)n_out;
  p.tiles_m = p.tiles_n = p.k_blocks = 0;
  p.small_acc = 0;
  if (half) {
    p.kind = 2;
    p.s_x = reinterpret_cast<const float*>(ws + H.inv);
    p.K = (int)(2 * K);
    p.a_pitch = 2 * K;
    p.wide_a = x;
    p.wide_a_pitch = 4 * ldx;
    p.wide_b = w_f;
    return launch_qgemm_plan(kPlanPair256S4E8, reinterpret_cast<const int8_t*>(ws + H.x_h), b_mm, false, y, ldy, p, st);
  }
  return launch_qgemm(reinterpret_cast<const int8_t*>(a_f), b_mm, false, y, ldy, p, st);
}

// The weight gradient takes the split operands wherever its contraction fills a K-block of 32 rows and the output a fair
// part of a tile: the tf32 form transposes dy and the scaled codes first, in launches of their own (both products, with
// the bias gradient: 22.6 vs 11.9 us at 64 x 512 x 512, 64 vs 48 at 64 x 3776 x 2240, 36 vs 30 at 255 x 1024 x 4096, 64.5 vs
// 120 us for dw alone at 12 800 x 2048 x 512).
static bool dw_split_applies(int64_t M, int64_t N, int64_t K) { return M >= 32 && N >= 128 && K >= 128; }

// The backward with the weight gradient on split operands: the scale of x multiplies dy while it is split, the codes stay
// exact, and dy is read in place.  The other product stays on the tf32 form, which needs no conversion in the kernel (62.6
// vs 65.0 us at 12 800 x 2048 x 512, 729 vs 850 us at 65 536 x 4096 x 1024); the two run side by side (166 against 83 + 109
// us at 65 536 x 512 x 512).
static int linear_bwd_split(const float* dy, int64_t lddy, const void* xq, const float* s_x, int s_x_kind, int bits_a, const void* wq,
                            const float* s_w, int bits_w, int64_t M, int64_t N, int64_t K, float* dx, int64_t lddx, float* dw, int64_t lddw,
                            float* dbias, uint8_t* ws, cudaStream_t st) {
  const DwLayout L = dw_layout(M, N, K);
  float* colsum = reinterpret_cast<float*>(ws + L.colsum);
  float* wt = reinterpret_cast<float*>(ws + L.wt);
  uint16_t* xt = reinterpret_cast<uint16_t*>(ws + L.xt);
  int rc;
  rc = launch_bwd_prep(wq, is_packed(bits_w), s_w, dx != nullptr ? wt : nullptr, xq, is_packed(bits_a), xt, L.m_pitch, M, N, K, st);
  if (rc != AQT_OK) return rc;
  if (dx != nullptr) {
    // dx = dy . (s_w wq): rows m, columns k, contraction n
    rc = float_gemm_nt(dy, lddy, wt, M, K, N, dx, lddx, st, 1, true);
    if (rc != AQT_OK) return rc;
  }
  // dw = (diag(s_x) dy)^T . xq: rows n, columns k, contraction m, cut into batches
  DwParams p = {};
  p.a_scale = s_x;
  p.a_scale_step = s_x_kind == AQT_SCALE_ROW ? 1 : 0;
  p.colsum = dbias != nullptr ? colsum : nullptr;
  p.M = (int)N;
  p.N = (int)K;
  p.K = (int)M;
  p.batch_k = (int)L.chunk;
  p.beside_previous = dx != nullptr ? 1 : 0;
  float* dwp = reinterpret_cast<float*>(ws + L.dwp);
  const bool one = L.batches == 1;
  rc = launch_dw_split(dy, lddy, xt, L.m_pitch, one ? dw : dwp, one ? N : L.batches * L.n_pad, one ? lddw : K, p, (int)L.batches, st);
  if (rc != AQT_OK) return rc;
  return launch_bwd_finish(dwp, L.batches, L.n_pad, N, K, dw, lddw, colsum, L.batches * DwCfg::kGroups, dbias, st);
}

int aqt_linear_bwd(const float* dy, int64_t lddy, const void* xq, const float* s_x, int s_x_kind, int bits_a, const void* wq,
                   const float* s_w, int bits_w, int64_t M, int64_t N, int64_t K, float* dx, int64_t lddx, float* dw, int64_t lddw,
                   float* dbias, void* workspace, size_t workspace_bytes, void* stream) {
  if (M < 0 || N < 0 || K <= 0 || !bits_ok(bits_a) || !bits_ok(bits_w)) return AQT_ERR_BADARG;
  if (s_x_kind != AQT_SCALE_ROW && s_x_kind != AQT_SCALE_TENSOR) return AQT_ERR_BADARG;
  if (K % 4 != 0 || N % 4 != 0) return AQT_ERR_BADARG;
  // M and N are row counts of the transposing prepasses, whose 128-row blocks are a grid's y extent (at most 65 535)
  if (M >= (1ll << 23) || N >= (1ll << 23) || K >= (1ll << 28) || M * N >= (1ll << 40)) return AQT_ERR_UNSUPPORTED;
  if (M == 0 || N == 0) return AQT_OK;
  if (dy == nullptr || lddy < N) return AQT_ERR_BADARG;
  if (dx != nullptr && (wq == nullptr || s_w == nullptr || lddx < K)) return AQT_ERR_BADARG;
  if (dw != nullptr && (xq == nullptr || s_x == nullptr || lddw < K)) return AQT_ERR_BADARG;
  if (!is_aligned(dy, 16) || lddy % 4 != 0) return AQT_ERR_ALIGN;
  if (dx != nullptr && (!is_aligned(dx, 16) || lddx % 4 != 0)) return AQT_ERR_ALIGN;
  if (dw != nullptr && (!is_aligned(dw, 16) || lddw % 4 != 0)) return AQT_ERR_ALIGN;
  if (dbias != nullptr && !is_aligned(dbias, 4)) return AQT_ERR_ALIGN;
  if ((dx != nullptr && !is_aligned(wq, 16)) || (dw != nullptr && !is_aligned(xq, 16))) return AQT_ERR_ALIGN;
  const BwdLayout L = bwd_layout(M, N, K);
  if (workspace == nullptr || workspace_bytes < bwd_workspace(M, N, K)) return AQT_ERR_WORKSPACE;
  if (!is_aligned(workspace, 256)) return AQT_ERR_ALIGN;
  int rc = check_device();
  if (rc != AQT_OK) return rc;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  uint8_t* ws = reinterpret_cast<uint8_t*>(workspace);
  if (dw != nullptr && dw_split_applies(M, N, K))
    return linear_bwd_split(dy, lddy, xq, s_x, s_x_kind, bits_a, wq, s_w, bits_w, M, N, K, dx, lddx, dw, lddw, dbias, ws, st);
  if (dbias != nullptr && dw == nullptr) {  // with dw the column sums come out of the transpose of dy
    rc = launch_colsum(dy, lddy, M, N, reinterpret_cast<float*>(ws + L.partial), dbias, st);
    if (rc != AQT_OK) return rc;
  }
  if (dx != nullptr) {
    // dx = dy . (s_w wq): rows m, columns k, contraction n
    float* wt = reinterpret_cast<float*>(ws + L.wt);
    rc = launch_transpose_scale_codes(wq, is_packed(bits_w), s_w, true, N, K, wt, N, N, K, st);
    if (rc != AQT_OK) return rc;
    rc = float_gemm_nt(dy, lddy, wt, M, K, N, dx, lddx, st);
    if (rc != AQT_OK) return rc;
  }
  if (dw != nullptr) {
    // dw = dy^T . (s_x xq): rows n, columns k, contraction m (padded with zeros), cut into L.batches chunks
    float* dyt = reinterpret_cast<float*>(ws + L.dyt);
    float* xt = reinterpret_cast<float*>(ws + L.xt);
    const int64_t m_pad = L.batches * L.chunk;
    rc = launch_transpose_f32(dy, lddy, M, N, dyt, m_pad, L.chunk, L.n_pad, dbias != nullptr ? reinterpret_cast<float*>(ws + L.partial) : nullptr,
                              dbias, st);
    if (rc != AQT_OK) return rc;
    rc = launch_transpose_scale_codes(xq, is_packed(bits_a), s_x, s_x_kind == AQT_SCALE_ROW, M, K, xt, m_pad, L.chunk, K, st);
    if (rc != AQT_OK) return rc;
    if (L.batches == 1) {
      rc = float_gemm_nt(dyt, L.chunk, xt, N, K, L.chunk, dw, lddw, st);
      if (rc != AQT_OK) return rc;
    } else {
      float* dwp = reinterpret_cast<float*>(ws + L.dwp);
      rc = float_gemm_nt(dyt, L.chunk, xt, L.batches * L.n_pad, K, L.chunk, dwp, K, st, L.batches);
      if (rc != AQT_OK) return rc;
      rc = launch_sum_batches(dwp, L.batches, L.n_pad, N, K, dw, lddw, st);
      if (rc != AQT_OK) return rc;
    }
  }
  return AQT_OK;
}

// ------------------------------------------------------------------------------------------------
// Allocation-free variant: the scratch lives in the library image.

// Sign-extended weight codes of the call in flight.  This name is only a host-side handle in
// host code; its device address comes from cudaGetSymbolAddress (noalloc_scratch_address).
static __device__ __align__(256) uint8_t g_noalloc_weight_scratch[AQT_NOALLOC_MAX_WEIGHT_BYTES];

// Device address of the scratch array on the current device, looked up once per device.
static int noalloc_scratch_address(uint8_t** out) {
  constexpr int kMaxDevices = 64;
  static uint8_t* cached[kMaxDevices] = {nullptr};
  int dev = 0;
  AQT_RETURN_IF_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) return AQT_ERR_UNSUPPORTED;
  if (cached[dev] == nullptr) {
    void* ptr = nullptr;
    AQT_RETURN_IF_CUDA(cudaGetSymbolAddress(&ptr, g_noalloc_weight_scratch));
    if (ptr == nullptr) return AQT_ERR_CUDA;
    cached[dev] = reinterpret_cast<uint8_t*>(ptr);
  }
  *out = cached[dev];
  return AQT_OK;
}

int aqt_qmatmul_w4_noalloc(const int8_t* xq, const float* s_x, int s_x_kind, const uint8_t* wq_packed, const float* s_w,
                           const float* bias, const float* residual, int64_t ldr, float residual_scale, int64_t M, int64_t N,
                           int64_t K, int act, float* y, int64_t ldy, void* stream) {
  int rc = validate_matmul_shape(M, N, K, 8, 4, act, s_x_kind);
  if (rc != AQT_OK) return rc;
  if (M == 0 || N == 0) return AQT_OK;
  if ((uint64_t)N * (uint64_t)K > (uint64_t)AQT_NOALLOC_MAX_WEIGHT_BYTES) {
    if (debug_enabled())
      fprintf(stderr, "[aqt] aqt_qmatmul_w4_noalloc: N*K = %lld exceeds the built-in scratch of %u bytes\n", (long long)(N * K),
              AQT_NOALLOC_MAX_WEIGHT_BYTES);
    return AQT_ERR_UNSUPPORTED;
  }
  const int64_t n_out = is_glu(act) ? N / 2 : N;
  if (xq == nullptr || s_x == nullptr || wq_packed == nullptr || s_w == nullptr || y == nullptr) return AQT_ERR_BADARG;
  if (ldy < n_out || (residual != nullptr && ldr < n_out)) return AQT_ERR_BADARG;
  if (!is_aligned(xq, 16) || !is_aligned(wq_packed, 16) || !is_aligned(y, 16) || !is_aligned(s_w, 16) || !is_aligned(s_x, 4) ||
      (bias != nullptr && !is_aligned(bias, 16)) || (residual != nullptr && !is_aligned(residual, 16)))
    return AQT_ERR_ALIGN;
  if (ldy % 4 != 0 || (residual != nullptr && ldr % 4 != 0)) return AQT_ERR_ALIGN;
  rc = check_device();
  if (rc != AQT_OK) return rc;
  uint8_t* scratch = nullptr;
  rc = noalloc_scratch_address(&scratch);
  if (rc != AQT_OK) return rc;
  // qmatmul_i8a unpacks the weights into `scratch` (all N*K bytes it later reads) and runs the GEMM.
  return qmatmul_i8a(xq, s_x, s_x_kind, wq_packed, s_w, bias, residual, ldr, residual_scale, M, N, K, 8, 4, act, y, ldy, nullptr,
                     scratch, reinterpret_cast<cudaStream_t>(stream));
}

int aqt_selftest_bounded_wait(uint64_t limit_ns, int* gave_up_dev, void* stream) {
  if (gave_up_dev == nullptr || limit_ns == 0 || limit_ns > 1000000000ull) return AQT_ERR_BADARG;
  int rc = check_device();
  if (rc != AQT_OK) return rc;
  bounded_wait_selftest_kernel<<<1, 64, 0, reinterpret_cast<cudaStream_t>(stream)>>>(limit_ns, gave_up_dev);
  return AQT_LAUNCH_STATUS();
}

// Nothing but special-function work: eight independent chains of 2^x and reciprocal per thread.
__global__ void __launch_bounds__(256) sfu_rate_kernel(int iterations, float* sink) {
  float v[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) v[j] = 0.25f + 0.01f * (float)((threadIdx.x + j) & 15);
  for (int i = 0; i < iterations; ++i) {
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = rcp_approx(1.0f + ex2_approx(v[j]));
  }
  float acc = 0.0f;
#pragma unroll
  for (int j = 0; j < 8; ++j) acc += v[j];
  if (acc == 12345.0f) *sink = acc;  // never true: keeps the chains alive
}

int aqt_selftest_sfu_rate(int iterations, float* sink_dev, int64_t* ops_out, void* stream) {
  if (iterations <= 0 || iterations > (1 << 20) || sink_dev == nullptr || ops_out == nullptr) return AQT_ERR_BADARG;
  int rc = check_device();
  if (rc != AQT_OK) return rc;
  const int sms = sm_count();
  if (sms <= 0) return AQT_ERR_CUDA;
  const int ctas = sms * 8;
  sfu_rate_kernel<<<ctas, 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(iterations, sink_dev);
  *ops_out = (int64_t)ctas * 256 * iterations * 16;
  return AQT_LAUNCH_STATUS();
}

int aqt_device_status(void* stream, int* status_out) {
  if (status_out == nullptr) return AQT_ERR_BADARG;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  AQT_RETURN_IF_CUDA(cudaStreamSynchronize(st));
  int v = 0;
  AQT_RETURN_IF_CUDA(cudaMemcpyFromSymbol(&v, g_device_status, sizeof(int)));
  if (v != 0) {
    const int zero = 0;
    AQT_RETURN_IF_CUDA(cudaMemcpyToSymbol(g_device_status, &zero, sizeof(int)));
  }
  *status_out = v;
  return AQT_OK;
}

}  // extern "C"
