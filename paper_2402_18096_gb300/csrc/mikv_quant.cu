// mikv_quant.cu — demotion of KV rows into the retained set (Eq. 1 with the Eq. 3 key balancer), rows
// entering a coded important set (Sec. 3.3), and the channel balancer itself (Eq. 2), arxiv 2402.18096.
//
// quantize_pack: each warp quantizes four rows of K or of V, eight lanes per row and 16 channels per lane;
// group minima and maxima come from the lane's channels and butterfly shuffles, scale and zero are
// rounded to fp16 outward so the stored grid covers the group's range, codes are round-half-even of the
// IEEE fp32 quotient (x - beta) / alpha (the Eq. 1 helpers of mikv_quant_rows.cuh, shared with the
// one-row quantizer of the step tail), and the packed words are joined from the lanes that share them.
#include "mikv_device.cuh"
#include "mikv_internal.h"
#include "mikv_quant_rows.cuh"

namespace mikv {
namespace {

struct QPArgs {
  const __nv_bfloat16* k_src;
  const __nv_bfloat16* v_src;
  const int32_t* src_tok;
  const int32_t* rows;
  const float* balancer;
  uint8_t* k_codes;
  uint8_t* v_codes;
  __half2* k_params;
  __half2* v_params;
  int32_t* lo_tok;
  int* dbg;  // debug builds: the library's status word for index checks (nullptr otherwise)
  int heads_kv, n_src, n_rows, lo_start, lo_cap;
  int rounds;  // rounds of a block
};

// Bulk quantize/pack (Eq. 1): eight lanes per row and four rows per warp. Lane l8 = lane & 7 of a row owns
// channels 16 l8 .. 16 l8 + 15 (two 16-byte loads), so a group's scale and zero are computed by GROUP / 16
// lanes, and in the packed layout every channel of the lane sits at field index m = l8 of its 16-bit unit:
// the lane's codes form partial words at fixed positions, joined with those of the lanes that share them into whole
// words, one or two per lane (qp_store_codes).
// It is bound by instruction issue (a row's bytes move in a third of the time its scalar arithmetic took), so the
// arithmetic is packed: pairs of channels in fp32x2, minima and maxima three at a time, the code taken from the
// rounded sum's low bits without a clamp, the doubtful codes found by one maximum over the lane's channels, the words
// joined on the FMA pipe. A warp walks several rounds of rows with the next rows' loads in flight behind the
// arithmetic; the balancer waits in shared memory, which leaves 61 registers and four blocks per SM (70 registers and
// three blocks: 1230 us). B 32, Hkv 8, 26214 rows of K and V each, INT2 g32: 1839 -> 1086 us (the bytes at the copy
// rate: 600).
constexpr int kQpRowsPerWarp = 4;
constexpr int kQpBlockRows = 4 * kQpRowsPerWarp;      // rows of a round (16 of K and of V each)
constexpr int kQpRoundsMax = 16;
constexpr int kQpBlocksPerSm = 2 * 4;                 // fewer rounds per block until the grid has this many per SM

// Packs one row's codes: w[k] = code of channel 16 l8 + 2 k | code of channel 16 l8 + 2 k + 1 << 16. A word of the row
// collects the same k from the lanes that share it, so the row's words are transposed through the warp's shared memory
// (x: word k of lane l at 8 k + l, rows 72 words apart: no bank conflicts) and joined by multiply-adds, which the FMA
// pipe takes where selects, shifts and shuffles loaded the ALU pipe.
constexpr int kQpRowWords = 72;

template <int N>
__device__ __forceinline__ uint32_t join_fields(const uint32_t* x, uint32_t step) {  // sum of x[m] step^m
  uint32_t v = x[N - 1];
#pragma unroll
  for (int m = N - 2; m >= 0; --m) v = v * step + x[m];
  return v;
}

template <int BITS>
__device__ __forceinline__ void qp_store_codes(const uint32_t (&w)[8], uint32_t* x, uint32_t* row, int l8, bool valid) {
  __syncwarp();  // (the previous round's words have been read)
#pragma unroll
  for (int k = 0; k < 8; ++k) x[8 * k + l8] = w[k];
  __syncwarp();
  uint32_t f[8];
  if constexpr (BITS == 4) {
    // channel 16 l8 + u: unit 16 (l8 >> 2) + u, bits 4 (l8 & 3); lane l8 writes words 2 l8 and 2 l8 + 1, each joined
    // from four lanes
    const uint4* p = reinterpret_cast<const uint4*>(x + 8 * ((2 * l8) & 7) + 4 * (l8 >> 2));
    const uint4 a = p[0], b = p[2];
    const uint32_t fa[4] = {a.x, a.y, a.z, a.w}, fb[4] = {b.x, b.y, b.z, b.w};
    if (valid) *reinterpret_cast<uint2*>(row + 2 * l8) = make_uint2(join_fields<4>(fa, 16u), join_fields<4>(fb, 16u));
  } else {
    // two-bit fields (INT2, and the low bits of INT3): channel 16 l8 + u sits in unit u at bits 2 l8: lane l8 writes
    // word l8
    const uint4* p = reinterpret_cast<const uint4*>(x + 8 * l8);
    const uint4 a = p[0], b = p[1];
    const uint32_t g[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
    for (int m = 0; m < 8; ++m) f[m] = BITS == 3 ? g[m] & 0x00030003u : g[m];
    if (valid) row[l8] = join_fields<8>(f, 4u);
    if constexpr (BITS == 3) {
      // high bits: channel 16 l8 + u sits in unit u & 7 at bit 2 l8 + (u >> 3) (words 8..11 of the row): lanes l8 and
      // l8 + 4 hold the even and the odd bits of a word
#pragma unroll
      for (int m = 0; m < 8; ++m) f[m] = g[m] & 0x00040004u;
      const uint32_t h = (f[0] >> 2) + join_fields<7>(f + 1, 4u);  // (bit 2 of field m at bit 2 m)
      const uint32_t o = __shfl_xor_sync(0xffffffffu, h, 4);
      if (valid && l8 < 4) row[8 + l8] = h | (o << 1);
    }
  }
}

template <int BITS, int GROUP>
__global__ void __launch_bounds__(256, 4) quantize_pack_kernel(const QPArgs a) {
  constexpr int QMAX = (1 << BITS) - 1;
  constexpr int GL = GROUP / 16;  // lanes per quantization group
  __shared__ __align__(16) uint32_t s_words[8][4 * kQpRowWords];
  __shared__ float4 s_bal[kHeadDim / 4];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, l8 = lane & 7;
  const bool is_v = (w & 1) != 0;
  const int bh = blockIdx.y, h = bh % a.heads_kv;
  const int32_t* rows = a.rows + (size_t)bh * a.n_rows;
  const __nv_bfloat16* src = (is_v ? a.v_src : a.k_src) + (size_t)bh * a.n_src * kHeadDim + 16 * l8;
  const int i0 = blockIdx.x * (a.rounds * kQpBlockRows) + (w >> 1) * kQpRowsPerWarp + (lane >> 3);
  const bool balanced = !is_v && a.balancer;  // Eq. 3: keys times the balancer before the quantizer (warp-uniform)
  // the head's balancer in shared memory: piece k of lane l8 at 8 k + l8 (no bank conflicts)
  if (a.balancer) {
    if (threadIdx.x < 32)
      s_bal[8 * (lane & 3) + (lane >> 2)] = reinterpret_cast<const float4*>(a.balancer + h * kHeadDim)[lane];
    __syncthreads();
  }
  // row i of this lane, -1 past the end; an out-of-range source row is skipped (documented in the ABI)
  auto row_of = [&](int i) { return i < a.n_rows ? rows[i] : -1; };
  auto in_range = [&](int r) { return r >= 0 && r < a.n_src; };
  // invalid rows run the arithmetic on zeros (every lane takes part in the shuffles) and store nothing
  auto load = [&](int r, uint4 (&raw)[2]) {
    const uint4* p = reinterpret_cast<const uint4*>(src + (size_t)r * kHeadDim);
    const bool v = in_range(r);
    raw[0] = v ? p[0] : make_uint4(0u, 0u, 0u, 0u);
    raw[1] = v ? p[1] : make_uint4(0u, 0u, 0u, 0u);
  };
  int r = row_of(i0), r_next = row_of(i0 + kQpBlockRows);
  uint4 raw[2];
  load(r, raw);
#pragma unroll 1
  for (int t = 0; t < a.rounds; ++t) {
    const int i = i0 + t * kQpBlockRows;
    if (__all_sync(0xffffffffu, i >= a.n_rows)) break;
    const bool valid = in_range(r);
    if (i < a.n_rows && !valid && l8 == 0 && !is_v) MIKV_BOUNDS_FAIL(a.dbg);
    uint64_t x[8];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const uint32_t wd[4] = {raw[k].x, raw[k].y, raw[k].z, raw[k].w};
#pragma unroll
      for (int j = 0; j < 4; ++j) x[4 * k + j] = f32x2(__uint_as_float(wd[j] << 16), __uint_as_float(wd[j] & 0xffff0000u));
    }
    // the next round's rows, behind this round's arithmetic
    const int rn = r_next;
    if (t + 1 < a.rounds) {
      load(rn, raw);
      r_next = t + 2 < a.rounds ? row_of(i + 2 * kQpBlockRows) : -1;
    }
    if (balanced) {
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float4 b = s_bal[8 * k + l8];
        x[2 * k] = mul_f32x2(x[2 * k], f32x2(b.x, b.y));
        x[2 * k + 1] = mul_f32x2(x[2 * k + 1], f32x2(b.z, b.w));
      }
    }
    float mn, mx;
    {
      float lo, hi;
      f32x2_split(x[0], lo, hi);
      mn = fminf(lo, hi);
      mx = fmaxf(lo, hi);
#pragma unroll
      for (int k = 1; k < 8; ++k) {
        f32x2_split(x[k], lo, hi);
        mn = min3(mn, lo, hi);
        mx = max3(mx, lo, hi);
      }
    }
#pragma unroll
    for (int off = 1; off < GL; off <<= 1) {
      mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, off));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    }
    const Eq1Params p = eq1_params<QMAX>(mn, mx);
    const uint64_t nb = f32x2(-p.beta, -p.beta), ra = f32x2(p.ralpha, p.ralpha);
    uint32_t wd[8];
    float far = 0.f;  // the largest distance from an integer
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      uint64_t y, off;
      eq1_pair_fast(x[k], nb, ra, y, off);
      float y0, y1, f0, f1;
      f32x2_split(y, y0, y1);
      f32x2_split(off, f0, f1);
      far = max3_abs_nan(far, f0, f1);
      wd[k] = prmt(__float_as_uint(y0), __float_as_uint(y1), 0x5410u);
    }
    if (!(far < 0.5f - 0x1p-13f)) {
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        float lo, hi;
        f32x2_split(x[k], lo, hi);
        wd[k] = eq1_code_exact<QMAX>(lo, p) | (eq1_code_exact<QMAX>(hi, p) << 16);
      }
    }
    const size_t pos = (size_t)bh * a.lo_cap + a.lo_start + i;
    qp_store_codes<BITS>(wd, s_words[w] + kQpRowWords * (lane >> 3),
                         reinterpret_cast<uint32_t*>((is_v ? a.v_codes : a.k_codes) + pos * (16 * BITS)), l8, valid);
    if (valid && l8 % GL == 0)
      ((is_v ? a.v_params : a.k_params) + pos * (kHeadDim / GROUP))[(16 * l8) / GROUP] =
          __halves2half2(p.alpha16, p.beta16);
    if (valid && !is_v && l8 == 0) a.lo_tok[pos] = a.src_tok ? a.src_tok[(size_t)bh * a.n_src + r] : r;
    r = rn;
  }
}

template <int BITS>
cudaError_t qp_group(const QPArgs& a, int group, dim3 grid, cudaStream_t st) {
  switch (group) {
    case 32: quantize_pack_kernel<BITS, 32><<<grid, 256, 0, st>>>(a); break;
    case 64: quantize_pack_kernel<BITS, 64><<<grid, 256, 0, st>>>(a); break;
    case 128: quantize_pack_kernel<BITS, 128><<<grid, 256, 0, st>>>(a); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

// ------------------------------------------------------- coded important set (Sec. 3.3, Table 3)

// Rows entering a coded important set, quantized like retained rows (Eq. 1 at hi_bits, groups of
// kHiGroup; keys times the balancer first, Eq. 3). Two modes: insert (rows == nullptr: the new token of
// every (b, h) into slot slots[b][h]) and gather (slot i < n_rows receives source row rows[b][h][i]).
struct HiQArgs {
  const __nv_bfloat16* k_src;
  const __nv_bfloat16* v_src;
  const int32_t* src_tok;
  const float* src_scores;
  const int32_t* rows;
  const int32_t* slots;
  const float* balancer;
  uint8_t* k_hc;
  uint8_t* v_hc;
  __half2* k_hp;
  __half2* v_hp;
  int32_t* hi_tok;
  float* acc;
  int* dbg;  // debug builds: the library's status word for index checks (nullptr otherwise)
  int heads_kv, hi_cap, hi_stride, n_src, n_rows, tok;
};

template <int HB>
__global__ void __launch_bounds__(256) hi_quant_kernel(const HiQArgs a) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  grid_dependency_wait();  // insertion: the slot comes from the previous step's tail
  allow_dependent_launch();
  const int i = blockIdx.x * 4 + (w >> 1);
  const bool is_v = (w & 1) != 0;
  const int bh = blockIdx.y, h = bh % a.heads_kv;
  int slot, r = 0;
  const __nv_bfloat16* src;
  if (a.rows) {
    if (i >= a.n_rows) return;
    r = a.rows[(size_t)bh * a.n_rows + i];
    if (r < 0 || r >= a.n_src) {  // out-of-range rows are skipped, as in quantize_pack
      if (lane == 0 && !is_v) MIKV_BOUNDS_FAIL(a.dbg);
      return;
    }
    slot = i;
    src = (is_v ? a.v_src : a.k_src) + ((size_t)bh * a.n_src + r) * kHeadDim;
  } else {
    if (i > 0) return;
    slot = a.slots[bh];
    if (slot < 0 || slot >= a.hi_cap) {
      if (lane == 0 && !is_v) MIKV_BOUNDS_FAIL(a.dbg);
      return;
    }
    src = (is_v ? a.v_src : a.k_src) + (size_t)bh * kHeadDim;
  }
  const size_t row = (size_t)bh * a.hi_stride + slot;
  quantize_row_warp<HB, kHiGroup>(src, is_v ? nullptr : (a.balancer ? a.balancer + h * kHeadDim : nullptr),
                                  (is_v ? a.v_hc : a.k_hc) + row * (16 * HB),
                                  (is_v ? a.v_hp : a.k_hp) + row * (kHeadDim / kHiGroup), lane);
  if (!is_v && lane == 0) {
    a.hi_tok[row] = a.rows ? (a.src_tok ? a.src_tok[(size_t)bh * a.n_src + r] : r) : a.tok;
    a.acc[row] = a.rows && a.src_scores ? a.src_scores[(size_t)bh * a.n_src + r] : 0.f;
  }
}

// ------------------------------------------------------------- per-channel retained keys (App. C)

// Rows of the retained set with per-channel keys: position p of (b, h) belongs to token group p / 64. New
// rows (source rows rows[b][h][p - p0]) and staged rows (important rows hi_cap + p % 64, positions < p0)
// feed the group kernel; the stage kernel copies the rows of an incomplete last group into staging.
struct KchArgs {
  const __nv_bfloat16* k_src;
  const __nv_bfloat16* v_src;
  const int32_t* src_tok;
  const int32_t* rows;
  __nv_bfloat16* k_hi;
  __nv_bfloat16* v_hi;
  int32_t* hi_tok;
  uint8_t* k_codes;
  uint8_t* v_codes;
  __half2* k_params;  // [B][Hkv][lo_cap / 64][128]
  __half2* v_params;
  int32_t* lo_tok;
  int* dbg;  // debug builds: the library's status word for index checks (nullptr otherwise)
  int heads_kv, hi_cap, hi_stride, lo_cap, n_src, n_rows, p0, p_end, g0;
};

constexpr int kKchThreads = 256;

// Source of position p of head bh: the staged row (p < p0) or the new source row; token id in *tok.
// A source row outside [0, n_src) reads as zeros (the host passes rows from mikv_select_demote).
__device__ __forceinline__ const __nv_bfloat16* kch_row(const KchArgs& a, int bh, int p, bool key, int32_t* tok) {
  if (p < a.p0) {
    const size_t r = (size_t)bh * a.hi_stride + a.hi_cap + (p % kKchGroup);
    if (tok) *tok = a.hi_tok[r];
    return (key ? a.k_hi : a.v_hi) + r * kHeadDim;
  }
  const int r = a.rows[(size_t)bh * a.n_rows + (p - a.p0)];
  if (tok) *tok = (r >= 0 && r < a.n_src) ? (a.src_tok ? a.src_tok[(size_t)bh * a.n_src + r] : r) : -1;
  if (r < 0 || r >= a.n_src) {
    if (key) MIKV_BOUNDS_FAIL(a.dbg);
    return nullptr;
  }
  return (key ? a.k_src : a.v_src) + ((size_t)bh * a.n_src + r) * kHeadDim;
}

// Group g0 + blockIdx.x of (b, h) = blockIdx.y, complete: keys quantized per channel over its 64 tokens
// (Eq. 1 with the same explicitly rounded fp32 steps as the per-token quantizer), values per token.
template <int BITS, int GROUP>
__global__ void __launch_bounds__(kKchThreads) kch_group_kernel(const KchArgs a) {
  __shared__ __align__(16) __nv_bfloat16 sk[kKchGroup][kHeadDim];
  __shared__ __align__(16) __nv_bfloat16 sv[kKchGroup][kHeadDim];
  __shared__ uint32_t cbuf[kKchGroup][4 * BITS];
  __shared__ int32_t stok[kKchGroup];
  constexpr int QMAX = (1 << BITS) - 1;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int j = a.g0 + blockIdx.x, bh = blockIdx.y;
  grid_dependency_wait();  // the group's last row is staged by the step tail before this kernel
  allow_dependent_launch();
  // 1. the group's 64 key and value rows (16-byte chunks) into shared memory; code rows cleared
  for (int i = tid; i < kKchGroup * 16; i += kKchThreads) {
    const int t = i >> 4, ch = i & 15;
    const int p = kKchGroup * j + t;
    int32_t tk = -1;
    const __nv_bfloat16* kr = kch_row(a, bh, p, true, &tk);
    const __nv_bfloat16* vr = kch_row(a, bh, p, false, nullptr);
    const uint4 z = make_uint4(0u, 0u, 0u, 0u);
    reinterpret_cast<uint4*>(&sk[t][0])[ch] = kr ? reinterpret_cast<const uint4*>(kr)[ch] : z;
    reinterpret_cast<uint4*>(&sv[t][0])[ch] = vr ? reinterpret_cast<const uint4*>(vr)[ch] : z;
    if (ch == 0) stok[t] = tk;
  }
  for (int i = tid; i < kKchGroup * 4 * BITS; i += kKchThreads) (&cbuf[0][0])[i] = 0u;
  __syncthreads();
  // 2. keys: one thread per channel
  if (tid < kHeadDim) {
    const int c = tid;
    float mn = INFINITY, mx = -INFINITY;
    for (int t = 0; t < kKchGroup; ++t) {
      const float x = __bfloat162float(sk[t][c]);
      mn = fminf(mn, x);
      mx = fmaxf(mx, x);
    }
    const __half beta16 = __float2half_rd(mn);
    const float beta = __half2float(beta16);
    const float span = __fsub_rn(mx, beta);
    const __half alpha16 = span == 0.f ? __float2half_rn(1.f) : __float2half_ru(__fdiv_rn(span, (float)QMAX));
    const float alpha = __half2float(alpha16);
    a.k_params[((size_t)bh * (a.lo_cap / kKchGroup) + j) * kHeadDim + c] = __halves2half2(alpha16, beta16);
    int unit, bit, unit1 = 0, bit1 = 0;
    field_pos(c, BITS == 3 ? 2 : BITS, unit, bit);
    if (BITS == 3) field_pos(c, 1, unit1, bit1);
    for (int t = 0; t < kKchGroup; ++t) {
      int code = __float2int_rn(__fdiv_rn(__fsub_rn(__bfloat162float(sk[t][c]), beta), alpha));
      code = code < 0 ? 0 : (code > QMAX ? QMAX : code);
      const uint32_t fmask = BITS == 3 ? 3u : (uint32_t)QMAX;
      atomicOr(&cbuf[t][unit >> 1], (((uint32_t)code & fmask) << bit) << (16 * (unit & 1)));
      if (BITS == 3) atomicOr(&cbuf[t][8 + (unit1 >> 1)], (((uint32_t)code >> 2) << bit1) << (16 * (unit1 & 1)));
    }
  }
  __syncthreads();
  const size_t pos0 = (size_t)bh * a.lo_cap + (size_t)kKchGroup * j;
  for (int i = tid; i < kKchGroup * 4 * BITS; i += kKchThreads)
    reinterpret_cast<uint32_t*>(a.k_codes + pos0 * (16 * BITS))[i] = (&cbuf[0][0])[i];
  // 3. values per token (8 rows per warp) and token ids
  for (int t = warp; t < kKchGroup; t += kKchThreads / 32) {
    quantize_row_warp<BITS, GROUP>(&sv[t][0], nullptr, a.v_codes + (pos0 + t) * (16 * BITS),
                                   a.v_params + (pos0 + t) * (kHeadDim / GROUP), lane);
    if (lane == 0) a.lo_tok[pos0 + t] = stok[t];
  }
}

// Rows of the incomplete last group (positions max(p0, 64 * floor(p_end / 64)) .. p_end - 1) into staging.
__global__ void __launch_bounds__(kKchThreads) kch_stage_kernel(const KchArgs a) {
  const int bh = blockIdx.x;
  const int first = max(a.p0, a.p_end / kKchGroup * kKchGroup);
  for (int i = threadIdx.x; i < (a.p_end - first) * 16; i += kKchThreads) {
    const int p = first + (i >> 4), ch = i & 15;
    int32_t tk = -1;
    const __nv_bfloat16* kr = kch_row(a, bh, p, true, &tk);
    const __nv_bfloat16* vr = kch_row(a, bh, p, false, nullptr);
    const size_t r = (size_t)bh * a.hi_stride + a.hi_cap + (p % kKchGroup);
    const uint4 z = make_uint4(0u, 0u, 0u, 0u);
    reinterpret_cast<uint4*>(a.k_hi + r * kHeadDim)[ch] = kr ? reinterpret_cast<const uint4*>(kr)[ch] : z;
    reinterpret_cast<uint4*>(a.v_hi + r * kHeadDim)[ch] = vr ? reinterpret_cast<const uint4*>(vr)[ch] : z;
    if (ch == 0) a.hi_tok[r] = tk;
  }
}

template <int BITS>
cudaError_t kch_group_launch(const KchArgs& a, int group, dim3 grid, cudaStream_t st) {
  switch (group) {
    case 32: return launch_chained(kch_group_kernel<BITS, 32>, grid, dim3(kKchThreads), 0, st, a);
    case 64: return launch_chained(kch_group_kernel<BITS, 64>, grid, dim3(kKchThreads), 0, st, a);
    case 128: return launch_chained(kch_group_kernel<BITS, 128>, grid, dim3(kKchThreads), 0, st, a);
  }
  return cudaErrorInvalidValue;
}

// ---------------------------------------------------------------------------- Eq. 2 balancer

// Head y of the balancer's grid (y < B*Hq: queries, then keys): its rows and its channels' maxima in ws.
struct AbsmaxHead {
  const __nv_bfloat16* rows;
  uint32_t* out;
};
__device__ __forceinline__ AbsmaxHead absmax_head(const __nv_bfloat16* q_pre, const __nv_bfloat16* k_pre, int B, int Hq,
                                                  int Hkv, int T, uint32_t* ws, int y) {
  const bool is_q = y < B * Hq;
  const int yy = is_q ? y : y - B * Hq;
  const int head = yy % (is_q ? Hq : Hkv);
  const int h = is_q ? head / (Hq / Hkv) : head;
  return {(is_q ? q_pre : k_pre) + (size_t)yy * T * kHeadDim, ws + (is_q ? 0 : Hkv * kHeadDim) + h * kHeadDim};
}

// Column maxima of |x| over a chunk of one head's rows, folded into ws with atomicMax on the bit patterns
// (non-negative floats order like their bits). One pass over q and k, bound by HBM: 16-byte loads, eight rows in
// flight per thread, the maximum taken on packed bf16 pairs (exact; a NaN is passed over, as fmaxf does), and the
// atomic only where the maximum read before it is smaller (2-byte loads of one row at a time and an atomic per
// channel and 256 rows took 2071 us for the 10.7 GB of the B 32, Hq 32 / Hkv 8, T 32768 prefill, this one 1419).
constexpr int kAbsThreads = 256, kAbsRows = kAbsThreads / 16, kAbsInFlight = 8, kAbsChunk = 1024;

__global__ void __launch_bounds__(kAbsThreads) absmax_kernel(const __nv_bfloat16* q_pre, const __nv_bfloat16* k_pre,
                                                              int B, int Hq, int Hkv, int T, uint32_t* ws) {
  __shared__ uint4 s_m[kAbsThreads / 32][16];
  const int tid = threadIdx.x, c = tid & 15;  // 16-byte piece of a row (8 channels)
  const AbsmaxHead hd = absmax_head(q_pre, k_pre, B, Hq, Hkv, T, ws, blockIdx.y);
  const uint4* base = reinterpret_cast<const uint4*>(hd.rows) + c;
  const int t0 = blockIdx.x * kAbsChunk, t1 = min(T, t0 + kAbsChunk);
  __nv_bfloat162 m[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) m[k] = __floats2bfloat162_rn(0.f, 0.f);
  auto fold = [&](const uint4& x) {
    const uint32_t wd[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const uint32_t a = wd[k] & 0x7fff7fffu;
      m[k] = __hmax2(m[k], *reinterpret_cast<const __nv_bfloat162*>(&a));
    }
  };
  int t = t0 + (tid >> 4);
  for (; t + (kAbsInFlight - 1) * kAbsRows < t1; t += kAbsInFlight * kAbsRows) {
    uint4 x[kAbsInFlight];
#pragma unroll
    for (int u = 0; u < kAbsInFlight; ++u) x[u] = __ldcs(base + (size_t)(t + u * kAbsRows) * (kHeadDim / 8));
#pragma unroll
    for (int u = 0; u < kAbsInFlight; ++u) fold(x[u]);
  }
  for (; t < t1; t += kAbsRows) fold(__ldcs(base + (size_t)t * (kHeadDim / 8)));
  uint32_t v[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {  // the warp's two rows
    v[k] = *reinterpret_cast<uint32_t*>(&m[k]);
    const uint32_t o = __shfl_xor_sync(0xffffffffu, v[k], 16);
    m[k] = __hmax2(m[k], *reinterpret_cast<const __nv_bfloat162*>(&o));
    v[k] = *reinterpret_cast<uint32_t*>(&m[k]);
  }
  if ((tid & 16) == 0) s_m[tid >> 5][c] = make_uint4(v[0], v[1], v[2], v[3]);
  __syncthreads();
  if (tid < kHeadDim) {  // channel tid
    const __nv_bfloat16* col = reinterpret_cast<const __nv_bfloat16*>(s_m) + tid;
    float mx = 0.f;
#pragma unroll
    for (int w = 0; w < kAbsThreads / 32; ++w) mx = fmaxf(mx, __bfloat162float(col[w * kHeadDim]));
    const uint32_t bits = __float_as_uint(mx);
    if (bits > __ldcg(hd.out + tid)) atomicMax(hd.out + tid, bits);
  }
}

// The same for q or k not on a 16-byte boundary (2-byte loads, a chunk of 256 rows).
constexpr int kAbsNarrowChunk = 256;
__global__ void __launch_bounds__(128) absmax_narrow_kernel(const __nv_bfloat16* q_pre, const __nv_bfloat16* k_pre,
                                                             int B, int Hq, int Hkv, int T, uint32_t* ws) {
  const AbsmaxHead hd = absmax_head(q_pre, k_pre, B, Hq, Hkv, T, ws, blockIdx.y);
  const int c = threadIdx.x, t0 = blockIdx.x * kAbsNarrowChunk, t1 = min(T, t0 + kAbsNarrowChunk);
  float m = 0.f;
  for (int t = t0; t < t1; ++t) m = fmaxf(m, fabsf(__bfloat162float(hd.rows[(size_t)t * kHeadDim + c])));
  atomicMax(hd.out + c, __float_as_uint(m));
}

__global__ void __launch_bounds__(128) balancer_kernel(const uint32_t* ws, int Hkv, float* out) {
  const int h = blockIdx.x, c = threadIdx.x;
  const float mq = __uint_as_float(ws[h * kHeadDim + c]);
  const float mk = __uint_as_float(ws[Hkv * kHeadDim + h * kHeadDim + c]);
  out[h * kHeadDim + c] = (mq == 0.f || mk == 0.f) ? 1.f : __fsqrt_rn(__fdiv_rn(mq, mk));
}

}  // namespace

cudaError_t launch_quantize_pack(const mikv_shape& s, const mikv_cache& c, const void* k_src,
                                 const void* v_src, const int32_t* src_tok, int n_src,
                                 const int32_t* rows, int n_rows, int lo_start, int num_sms, cudaStream_t st) {
  if (n_rows == 0) return cudaSuccess;
  QPArgs a = {};
  a.dbg = debug_status_word();
  a.k_src = static_cast<const __nv_bfloat16*>(k_src);
  a.v_src = static_cast<const __nv_bfloat16*>(v_src);
  a.src_tok = src_tok;
  a.rows = rows;
  a.balancer = c.balancer;
  a.k_codes = static_cast<uint8_t*>(c.k_codes);
  a.v_codes = static_cast<uint8_t*>(c.v_codes);
  a.k_params = static_cast<__half2*>(c.k_params);
  a.v_params = static_cast<__half2*>(c.v_params);
  a.lo_tok = c.lo_tok;
  a.heads_kv = s.heads_kv;
  a.n_src = n_src;
  a.n_rows = n_rows;
  a.lo_start = lo_start;
  a.lo_cap = s.lo_cap;
  const long long all = (long long)((n_rows + kQpBlockRows - 1) / kQpBlockRows) * s.batch * s.heads_kv;  // rounds in all
  const long long rounds = all / ((long long)num_sms * kQpBlocksPerSm);
  a.rounds = (int)(rounds < 1 ? 1 : rounds < kQpRoundsMax ? rounds : kQpRoundsMax);
  const int per_block = a.rounds * kQpBlockRows;
  const dim3 grid((n_rows + per_block - 1) / per_block, s.batch * s.heads_kv);
  switch (s.bits) {
    case 2: return qp_group<2>(a, s.group, grid, st);
    case 3: return qp_group<3>(a, s.group, grid, st);
    case 4: return qp_group<4>(a, s.group, grid, st);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_hi_quant(const mikv_shape& s, const mikv_cache& c, const void* k_src, const void* v_src,
                            const int32_t* src_tok, const float* src_scores, int n_src, const int32_t* rows,
                            int n_rows, const int32_t* slots, int tok, cudaStream_t st) {
  HiQArgs a = {};
  a.dbg = debug_status_word();
  a.k_src = static_cast<const __nv_bfloat16*>(k_src);
  a.v_src = static_cast<const __nv_bfloat16*>(v_src);
  a.src_tok = src_tok;
  a.src_scores = src_scores;
  a.rows = rows;
  a.slots = slots;
  a.balancer = c.balancer;
  a.k_hc = static_cast<uint8_t*>(c.k_hi);
  a.v_hc = static_cast<uint8_t*>(c.v_hi);
  a.k_hp = static_cast<__half2*>(c.k_hi_params);
  a.v_hp = static_cast<__half2*>(c.v_hi_params);
  a.hi_tok = c.hi_tok;
  a.acc = c.acc;
  a.heads_kv = s.heads_kv;
  a.hi_cap = s.hi_cap;
  a.hi_stride = s.hi_stride;
  a.n_src = n_src;
  a.n_rows = n_rows;
  a.tok = tok;
  const dim3 grid(rows ? (n_rows + 3) / 4 : 1, s.batch * s.heads_kv);
  const int threads = rows ? 256 : 64;
  switch (hi_bits_of(s)) {
    case 8: return launch_chained(hi_quant_kernel<8>, grid, dim3(threads), 0, st, a);
    case 4: return launch_chained(hi_quant_kernel<4>, grid, dim3(threads), 0, st, a);
    case 2: return launch_chained(hi_quant_kernel<2>, grid, dim3(threads), 0, st, a);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_kch_append(const mikv_shape& s, const mikv_cache& c, const void* k_src, const void* v_src,
                              const int32_t* src_tok, int n_src, const int32_t* rows, int n_rows, int p0,
                              cudaStream_t st) {
  KchArgs a = {};
  a.dbg = debug_status_word();
  a.k_src = static_cast<const __nv_bfloat16*>(k_src);
  a.v_src = static_cast<const __nv_bfloat16*>(v_src);
  a.src_tok = src_tok;
  a.rows = rows;
  a.k_hi = static_cast<__nv_bfloat16*>(c.k_hi);
  a.v_hi = static_cast<__nv_bfloat16*>(c.v_hi);
  a.hi_tok = c.hi_tok;
  a.k_codes = static_cast<uint8_t*>(c.k_codes);
  a.v_codes = static_cast<uint8_t*>(c.v_codes);
  a.k_params = static_cast<__half2*>(c.k_params);
  a.v_params = static_cast<__half2*>(c.v_params);
  a.lo_tok = c.lo_tok;
  a.heads_kv = s.heads_kv;
  a.hi_cap = s.hi_cap;
  a.hi_stride = s.hi_stride;
  a.lo_cap = s.lo_cap;
  a.n_src = n_src;
  a.n_rows = n_rows;
  a.p0 = p0;  // positions < p0 come from staging
  a.p_end = p0 + n_rows;
  const int bh = s.batch * s.heads_kv;
  // groups completed by this append: j0 = first group touched .. (p_end / 64) - 1; with no new rows, the
  // caller asks for the group that ends at p0 (all of it staged)
  const int j0 = n_rows > 0 ? p0 / kKchGroup : p0 / kKchGroup - 1;
  const int j1 = n_rows > 0 ? a.p_end / kKchGroup : p0 / kKchGroup;
  a.g0 = j0;
  if (j1 > j0) {
    cudaError_t e;
    const dim3 grid(j1 - j0, bh);
    switch (s.bits) {
      case 2: e = kch_group_launch<2>(a, s.group, grid, st); break;
      case 3: e = kch_group_launch<3>(a, s.group, grid, st); break;
      case 4: e = kch_group_launch<4>(a, s.group, grid, st); break;
      default: return cudaErrorInvalidValue;
    }
    if (e != cudaSuccess) return e;
  }
  if (n_rows > 0 && a.p_end % kKchGroup != 0) {  // the incomplete last group waits in staging
    kch_stage_kernel<<<bh, kKchThreads, 0, st>>>(a);
    return cudaGetLastError();
  }
  return cudaSuccess;
}

cudaError_t launch_balancer(const mikv_shape& s, const void* q_pre, const void* k_pre, int T, float* out,
                            uint32_t* ws_max, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(ws_max, 0, sizeof(uint32_t) * 2 * s.heads_kv * kHeadDim, st);
  if (e != cudaSuccess) return e;
  const __nv_bfloat16* q = static_cast<const __nv_bfloat16*>(q_pre);
  const __nv_bfloat16* k = static_cast<const __nv_bfloat16*>(k_pre);
  const int heads = s.batch * (s.heads_q + s.heads_kv);
  const bool wide = reinterpret_cast<uintptr_t>(q_pre) % 16 == 0 && reinterpret_cast<uintptr_t>(k_pre) % 16 == 0;
  if (wide)
    absmax_kernel<<<dim3((T + kAbsChunk - 1) / kAbsChunk, heads), kAbsThreads, 0, st>>>(q, k, s.batch, s.heads_q,
                                                                                       s.heads_kv, T, ws_max);
  else
    absmax_narrow_kernel<<<dim3((T + kAbsNarrowChunk - 1) / kAbsNarrowChunk, heads), kHeadDim, 0, st>>>(
        q, k, s.batch, s.heads_q, s.heads_kv, T, ws_max);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  balancer_kernel<<<s.heads_kv, kHeadDim, 0, st>>>(ws_max, s.heads_kv, out);
  return cudaGetLastError();
}

}  // namespace mikv
