// mikv_policy.cu — the importance policy around the attention kernel (arxiv 2402.18096, Fig. 4 and
// Sec. 3): accumulated-attention (heavy-hitter) score update, choice of the tokens that leave the
// important set, insertion of the new token and the important-set build from prefill rows.
#include "mikv_device.cuh"
#include "mikv_internal.h"
#include "mikv_rows.cuh"

namespace mikv {
namespace {

// acc[b][h][i] += sum over the G query heads j of exp(s_ji - m_j) / l_j.
__global__ void __launch_bounds__(128) update_importance_kernel(float* acc, const float* hi_logits,
                                                                 const float* ml, int Hq, int Hkv,
                                                                 int hi_cap, int hi_stride) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int bh = blockIdx.y;
  if (i >= hi_cap) return;
  const int G = Hq / Hkv, b = bh / Hkv, h = bh - b * Hkv;
  float add = 0.f;
  for (int j = 0; j < G; ++j) {
    const int bq = b * Hq + h * G + j;
    add += importance_weight(hi_logits[(size_t)bq * hi_stride + i], ml[2 * bq], 1.f / ml[2 * bq + 1]);
  }
  acc[(size_t)bh * hi_stride + i] += add;
}

constexpr int kSelThreads = 1024;

// Block-wide exclusive scan of one int per thread; returns the prefix and writes the total.
__device__ int block_exclusive_scan(int v, int* total, int* sh) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int x = v;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, off);
    if (lane >= off) x += y;
  }
  if (lane == 31) sh[w] = x;
  __syncthreads();
  if (w == 0) {
    int z = lane < (kSelThreads / 32) ? sh[lane] : 0;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, z, off);
      if (lane >= off) z += y;
    }
    sh[32 + lane] = z;  // inclusive prefix of warp totals
  }
  __syncthreads();
  const int before = (w > 0 ? sh[32 + w - 1] : 0) + x - v;
  *total = sh[32 + kSelThreads / 32 - 1];
  __syncthreads();
  return before;
}

// The 32-bit halves of order_key: scores and ids as unsigned integers of the same order.
__device__ __forceinline__ uint32_t score_key(float s) { return (uint32_t)(order_key(s, 0) >> 32); }
__device__ __forceinline__ uint32_t id_key(int32_t id) { return (uint32_t)(id ^ (int32_t)0x80000000); }

// The value of rank `rank` (from 0) among key(i) of the entries with take(i), i < n: three radix passes of 11, 11 and
// 10 bits from the top. Leaves the value, its rank among its equals and how many equals there are.
struct Ranked {
  uint32_t value;
  int rank, equals;
};
constexpr int kBins = 2 * kSelThreads;  // two bins per thread in the search for the digit

template <class Key, class Take>
__device__ Ranked radix_rank(int n, int rank, Key key, Take take, unsigned int* hist, int* sh, Ranked* s_out) {
  const int tid = threadIdx.x;
  uint32_t prefix = 0, mask = 0;
  int equals = 0;
#pragma unroll 1
  for (int pass = 0; pass < 3; ++pass) {
    const int shift = pass == 0 ? 21 : pass == 1 ? 10 : 0;
    const uint32_t digits = pass == 2 ? 0x3ffu : 0x7ffu;
    hist[tid] = 0u;
    hist[tid + kSelThreads] = 0u;
    __syncthreads();
#pragma unroll 4
    for (int i = tid; i < n; i += kSelThreads) {
      const uint32_t k = key(i);
      if ((k & mask) == prefix && take(i)) atomicAdd(&hist[(k >> shift) & digits], 1u);
    }
    __syncthreads();
    const int c0 = (int)hist[2 * tid], c1 = (int)hist[2 * tid + 1];
    int total;
    const int before = block_exclusive_scan(c0 + c1, &total, sh);
    if (rank >= before && rank < before + c0 + c1) {  // exactly one thread
      const bool second = rank >= before + c0;
      s_out->value = prefix | ((uint32_t)(2 * tid + second) << shift);
      s_out->rank = rank - before - (second ? c0 : 0);
      s_out->equals = second ? c1 : c0;
    }
    __syncthreads();
    prefix = s_out->value;
    rank = s_out->rank;
    equals = s_out->equals;
    mask |= digits << shift;
    __syncthreads();
  }
  return {prefix, rank, equals};
}

// One block per (b, h): the n_demote smallest keys leave; both lists come out in ascending index order. Bound by
// latency and by the L2 reads of the scores (five or six of n x 4 bytes), so the passes are few and wide: the score
// alone is ranked first (three 11-bit passes, the digit found by a block scan), the id only among scores equal to the
// last one demoted, and the lists are written with coalesced stores from one scan of the warps' counts. (Eight
// byte-wide passes over (score, id), each with a serial search for the digit, and lists written a run per thread took
// 163 us for 256 heads of 32768 scores; this takes 49.)
constexpr int kSelRounds = 32;  // rounds of kSelThreads entries whose choice a thread keeps in one register

__global__ void __launch_bounds__(kSelThreads) select_kernel(const float* scores, const int32_t* ids, int n,
                                                             int stride, int n_demote, int32_t* demoted,
                                                             int32_t* kept) {
  __shared__ unsigned int hist[kBins];
  __shared__ int sh[64];
  __shared__ int s_off[kSelRounds * (kSelThreads / 32)];
  __shared__ unsigned long long s_best[kSelThreads / 32];
  __shared__ Ranked s_ranked;
  const int bh = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const float* sc = scores + (size_t)bh * stride;
  const int32_t* id = ids ? ids + (size_t)bh * stride : nullptr;
  int32_t* dem = demoted + (size_t)bh * n_demote;
  int32_t* kep = kept ? kept + (size_t)bh * (n - n_demote) : nullptr;
  auto ident = [&](int i) { return id ? id[i] : i; };

  // the largest key that is demoted, by its halves (keys are never 0: the top bit of a score key is set or ~)
  uint32_t last_score = 0u, last_id = 0u;
  if (n_demote == n) {
    last_score = last_id = ~0u;
  } else if (n_demote == 1) {
    unsigned long long best = ~0ull;
    for (int i = tid; i < n; i += kSelThreads) {
      const unsigned long long k = order_key(sc[i], ident(i));
      best = k < best ? k : best;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      const unsigned long long o = __shfl_xor_sync(0xffffffffu, best, off);
      best = o < best ? o : best;
    }
    if (lane == 0) s_best[warp] = best;
    __syncthreads();
    best = s_best[lane];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      const unsigned long long o = __shfl_xor_sync(0xffffffffu, best, off);
      best = o < best ? o : best;
    }
    last_score = (uint32_t)(best >> 32);
    last_id = (uint32_t)best;
  } else if (n_demote > 1) {
    const Ranked s = radix_rank(n, n_demote - 1, [&](int i) { return score_key(sc[i]); }, [](int) { return true; }, hist,
                                sh, &s_ranked);
    last_score = s.value;
    last_id = ~0u;
    if (s.rank + 1 < s.equals)  // only some of the equal scores leave: those with the smallest ids
      last_id = radix_rank(n, s.rank, [&](int i) { return id_key(ident(i)); },
                           [&](int i) { return score_key(sc[i]) == last_score; }, hist, sh, &s_ranked)
                    .value;
  }

  // ascending-index lists: the choices of up to kSelRounds rounds (bit k of `out`), the warps' counts scanned, then
  // every entry written to its place
  int base = 0;  // demoted before these rounds
  for (int i0 = 0; i0 < n; i0 += kSelRounds * kSelThreads) {
    uint32_t out = 0u;
#pragma unroll 4
    for (int k = 0; k < kSelRounds; ++k) {
      const int i = i0 + k * kSelThreads + tid;
      bool d = false;
      if (i < n && n_demote > 0) {
        const uint32_t s = score_key(sc[i]);
        d = s < last_score || (s == last_score && (last_id == ~0u || id_key(ident(i)) <= last_id));
      }
      const uint32_t votes = __ballot_sync(0xffffffffu, d);
      out |= (uint32_t)d << k;
      if (lane == 0) s_off[k * (kSelThreads / 32) + warp] = __popc(votes);
    }
    __syncthreads();
    int total;
    const int before = block_exclusive_scan(s_off[tid], &total, sh);  // (leaves through a block barrier)
    s_off[tid] = base + before;
    base += total;
    __syncthreads();
#pragma unroll 4
    for (int k = 0; k < kSelRounds; ++k) {
      const int i = i0 + k * kSelThreads + tid;
      const bool d = (out >> k) & 1u;
      const uint32_t votes = __ballot_sync(0xffffffffu, d);
      const int pos = s_off[k * (kSelThreads / 32) + warp] + __popc(votes & ((1u << lane) - 1u));  // demoted before i
      if (i < n) {
        if (d) {
          if (pos < n_demote) dem[pos] = i;
        } else if (kep && i - pos < n - n_demote) {
          kep[i - pos] = i;
        }
      }
    }
    __syncthreads();
  }
}
static_assert(kSelRounds * (kSelThreads / 32) == kSelThreads, "one warp count per thread in the scan");

__global__ void __launch_bounds__(64) insert_kernel(__nv_bfloat16* k_hi, __nv_bfloat16* v_hi, int32_t* hi_tok,
                                                    float* acc, const __nv_bfloat16* k_new,
                                                    const __nv_bfloat16* v_new, int tok, const int32_t* slots,
                                                    int hi_cap, int hi_stride, int* dbg) {
  const int bh = blockIdx.x, tid = threadIdx.x;
  grid_dependency_wait();  // the slot comes from the previous step's tail
  allow_dependent_launch();
  const int s = slots[bh];
  if (s < 0 || s >= hi_cap) {  // an out-of-range slot is skipped (recorded in debug builds)
    if (tid == 0) MIKV_BOUNDS_FAIL(dbg);
    return;
  }
  const size_t row = (size_t)bh * hi_stride + s;
  if (tid < 32) {
    reinterpret_cast<uint2*>(k_hi + row * kHeadDim)[tid] =
        reinterpret_cast<const uint2*>(k_new + (size_t)bh * kHeadDim)[tid];
  } else {
    reinterpret_cast<uint2*>(v_hi + row * kHeadDim)[tid - 32] =
        reinterpret_cast<const uint2*>(v_new + (size_t)bh * kHeadDim)[tid - 32];
  }
  if (tid == 0) {
    hi_tok[row] = tok;
    acc[row] = 0.f;
  }
}

// Rows of the important set from source rows, 16 bytes a lane: a warp moves the key (lanes 0-15) and the value (lanes
// 16-31) of kGatherRows rows at once, so that every row's two dependent reads (its index, then the row) overlap with
// the others' (one row of 8-byte pieces per warp: 413 us for the 1.7 GB of the B 32, Hkv 8, T 32768 build at 20 %;
// this: 253).
constexpr int kGatherRows = 4;
__global__ void __launch_bounds__(256) gather_wide_kernel(__nv_bfloat16* k_hi, __nv_bfloat16* v_hi, int32_t* hi_tok,
                                                          float* acc, const __nv_bfloat16* k_src,
                                                          const __nv_bfloat16* v_src, const int32_t* src_tok,
                                                          const float* src_scores, int n_src, const int32_t* rows,
                                                          int n_rows, int hi_stride, int* dbg) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, bh = blockIdx.y;
  const int i0 = (blockIdx.x * 8 + w) * kGatherRows;
  if (i0 >= n_rows) return;
  int r = -1;  // lane k < kGatherRows: source row of slot i0 + k
  if (lane < kGatherRows && i0 + lane < n_rows) {
    r = rows[(size_t)bh * n_rows + i0 + lane];
    if (r < 0 || r >= n_src) {  // an out-of-range source row is skipped (recorded in debug builds)
      MIKV_BOUNDS_FAIL(dbg);
      r = -1;
    }
  }
  const uint4* src = reinterpret_cast<const uint4*>(lane < 16 ? k_src : v_src) + (lane & 15);
  uint4* dst = reinterpret_cast<uint4*>(lane < 16 ? k_hi : v_hi) + (lane & 15);
  uint4 x[kGatherRows];
  int rk[kGatherRows];
#pragma unroll
  for (int k = 0; k < kGatherRows; ++k) {
    rk[k] = __shfl_sync(0xffffffffu, r, k);
    if (rk[k] >= 0) x[k] = __ldcs(src + ((size_t)bh * n_src + rk[k]) * (kHeadDim / 8));
  }
  if (r >= 0) {
    hi_tok[(size_t)bh * hi_stride + i0 + lane] = src_tok ? src_tok[(size_t)bh * n_src + r] : r;
    acc[(size_t)bh * hi_stride + i0 + lane] = src_scores ? src_scores[(size_t)bh * n_src + r] : 0.f;
  }
#pragma unroll
  for (int k = 0; k < kGatherRows; ++k)
    if (rk[k] >= 0) dst[((size_t)bh * hi_stride + i0 + k) * (kHeadDim / 8)] = x[k];
}

// The same for arrays not on 16-byte boundaries: one row per warp, 8 bytes a lane.
__global__ void __launch_bounds__(256) gather_kernel(__nv_bfloat16* k_hi, __nv_bfloat16* v_hi, int32_t* hi_tok,
                                                     float* acc, const __nv_bfloat16* k_src,
                                                     const __nv_bfloat16* v_src, const int32_t* src_tok,
                                                     const float* src_scores, int n_src, const int32_t* rows,
                                                     int n_rows, int hi_stride, int* dbg) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = blockIdx.x * 8 + w, bh = blockIdx.y;
  if (i >= n_rows) return;
  const int r = rows[(size_t)bh * n_rows + i];
  if (r < 0 || r >= n_src) {  // an out-of-range source row is skipped (recorded in debug builds)
    if (lane == 0) MIKV_BOUNDS_FAIL(dbg);
    return;
  }
  const size_t src = ((size_t)bh * n_src + r) * kHeadDim, dst = ((size_t)bh * hi_stride + i) * kHeadDim;
  reinterpret_cast<uint2*>(k_hi + dst)[lane] = reinterpret_cast<const uint2*>(k_src + src)[lane];
  reinterpret_cast<uint2*>(v_hi + dst)[lane] = reinterpret_cast<const uint2*>(v_src + src)[lane];
  if (lane == 0) {
    hi_tok[(size_t)bh * hi_stride + i] = src_tok ? src_tok[(size_t)bh * n_src + r] : r;
    acc[(size_t)bh * hi_stride + i] = src_scores ? src_scores[(size_t)bh * n_src + r] : 0.f;
  }
}

}  // namespace

cudaError_t launch_update_importance(const mikv_shape& s, const mikv_cache& c, const float* hi_logits,
                                     const float* ml, cudaStream_t st) {
  const dim3 grid((s.hi_cap + 127) / 128, s.batch * s.heads_kv);
  update_importance_kernel<<<grid, 128, 0, st>>>(c.acc, hi_logits, ml, s.heads_q, s.heads_kv, s.hi_cap,
                                                 s.hi_stride);
  return cudaGetLastError();
}

cudaError_t launch_select(int batch, int heads, const float* scores, const int32_t* ids, int n, int stride,
                          int n_demote, int32_t* demoted, int32_t* kept, cudaStream_t st) {
  select_kernel<<<batch * heads, kSelThreads, 0, st>>>(scores, ids, n, stride, n_demote, demoted, kept);
  return cudaGetLastError();
}

cudaError_t launch_insert(const mikv_shape& s, const mikv_cache& c, const void* k_new, const void* v_new,
                          int tok, const int32_t* slots, cudaStream_t st) {
  if (hi_bits_of(s) != 16)
    return launch_hi_quant(s, c, k_new, v_new, nullptr, nullptr, 0, nullptr, 0, slots, tok, st);
  return launch_chained(insert_kernel, dim3(s.batch * s.heads_kv), dim3(64), 0, st,
                        static_cast<__nv_bfloat16*>(c.k_hi), static_cast<__nv_bfloat16*>(c.v_hi), c.hi_tok, c.acc,
                        static_cast<const __nv_bfloat16*>(k_new), static_cast<const __nv_bfloat16*>(v_new), tok, slots,
                        s.hi_cap, s.hi_stride, debug_status_word());
}

cudaError_t launch_gather(const mikv_shape& s, const mikv_cache& c, const void* k_src, const void* v_src,
                          const int32_t* src_tok, const float* src_scores, int n_src, const int32_t* rows,
                          int n_rows, cudaStream_t st) {
  if (n_rows == 0) return cudaSuccess;
  if (hi_bits_of(s) != 16)
    return launch_hi_quant(s, c, k_src, v_src, src_tok, src_scores, n_src, rows, n_rows, nullptr, 0, st);
  const uintptr_t bits = reinterpret_cast<uintptr_t>(k_src) | reinterpret_cast<uintptr_t>(v_src) |
                         reinterpret_cast<uintptr_t>(c.k_hi) | reinterpret_cast<uintptr_t>(c.v_hi);
  if (bits % 16 == 0) {
    const int per_block = 8 * kGatherRows;
    gather_wide_kernel<<<dim3((n_rows + per_block - 1) / per_block, s.batch * s.heads_kv), 256, 0, st>>>(
        static_cast<__nv_bfloat16*>(c.k_hi), static_cast<__nv_bfloat16*>(c.v_hi), c.hi_tok, c.acc,
        static_cast<const __nv_bfloat16*>(k_src), static_cast<const __nv_bfloat16*>(v_src), src_tok, src_scores, n_src,
        rows, n_rows, s.hi_stride, debug_status_word());
    return cudaGetLastError();
  }
  const dim3 grid((n_rows + 7) / 8, s.batch * s.heads_kv);
  gather_kernel<<<grid, 256, 0, st>>>(static_cast<__nv_bfloat16*>(c.k_hi), static_cast<__nv_bfloat16*>(c.v_hi),
                                      c.hi_tok, c.acc, static_cast<const __nv_bfloat16*>(k_src),
                                      static_cast<const __nv_bfloat16*>(v_src), src_tok, src_scores, n_src, rows,
                                      n_rows, s.hi_stride, debug_status_word());
  return cudaGetLastError();
}

}  // namespace mikv
