// mikv_prefill.cu — initial importance of the prefill tokens (sm_103a): the attention each token receives
// from the prefill's causal attention, summed over the queries and over the G query heads of its KV head
// (the accumulated-attention, heavy-hitter score MiKV uses to choose the important set, Fig. 4 / Sec. 3 of
// arxiv 2402.18096).
//
// Two passes over the causal score matrix S = sm_scale * Q K^T, each a tiled bf16 contraction on the
// fifth-generation tensor cores (tcgen05.mma, M = N = 128, fp32 accumulators in tensor memory) fed by TMA:
//   1. rows:    per query i, the log2 of its softmax normaliser, c_i = log2 sum_{t <= i} 2^(s_it log2 e)
//               (accumulated online against a reference, as in flash attention, without values);
//   2. columns: per key t, sum over the G query heads and the queries i >= t of 2^(s_it log2 e - c_i).
// A work item is MT 128-token tiles of the fixed operand (queries in pass 1, keys in pass 2: the M side, so that an
// epilogue thread owns one accumulator row = TMEM lane) and every 128-token tile of the other operand it meets in the
// causal triangle.
//
// What bounds it: one exponential per score and pass (32 per clock and SM: 512 clocks per 128 x 128 tile) weighs as
// much as the tile's MMAs (512 clocks at the tensor peak), so both have to run all the time.
//  - Two warps issue MMAs, one per fixed tile. A thread takes 46 clocks to issue an MMA and some 450 for the hand-over
//    of a tile (measured: 0, 4, 8 and 16 MMAs a tile took 446, 726, 993 and 1466 clocks), so one thread alone leaves the
//    tensor cores idle half of the time; the other's MMAs fill its gap. (N = 256 keeps them full from one thread, 1025
//    clocks for eight MMAs, but then two accumulators fill the tensor memory and all sixteen epilogue warps share
//    each: 1086 against then 1022 us for the first call below.)
//  - Four accumulators, which fill the tensor memory, so that MMAs run under the arithmetic, and one streamed tile for
//    two fixed ones (MT = 2), which halves the traffic from L2 per score (the 128-row tiles drew 7.9 TB/s).
//  - Four sets of four epilogue warps. With MT = 2 each has an accumulator of its own, each warp taking whole rows of
//    128 columns: a hand-over costs the same whatever the columns behind it. Four warps per scheduler hide each other's
//    tcgen05.ld and barriers (158 clocks per 32 columns of a warp against 195 with two, 135 for the exponentials
//    alone), so nothing is prefetched, which keeps the threads within the 96 registers of 19 warps, and one copy of the
//    arithmetic keeps the loop in the instruction cache.
//  - One persistent CTA per SM whose copies and MMAs run on into the next item (with one item per CTA, filling and
//    draining cost 9 % of the 4096-token prefill). Items are handed out by the hardware's launch control (a running
//    CTA takes over the block index of one that has not started), so long and short items balance without a counter
//    in memory.
//  - A small prefill has few items (MT = 1) and is bound by the latency of their tiles. There two sets share an
//    accumulator's columns, four accumulators take turns under one fixed tile and four streamed tiles are in flight,
//    and at any size pieces of 32 columns that no row of the warp meets are not read. (us of a call with two CTAs per
//    SM and 64-token streamed tiles / with 8 epilogue warps, two accumulators and three streamed tiles / now: B 1, Hq
//    32, Hkv 8, T 300: 22.8 / 24.8 / 22.7; B 1, H 32, T 512: 18.4 / 20.5 / 16.6; B 8, H 32, T 300: 35.0 / 37.2 / 33.1;
//    B 2, H 40, T 777: 42.4 / 49.4 / 37.2.)
//
// Where the time goes (128 x 128 tile and pass, clocks per SM): 957 (pass 1) and 1075 (pass 2) of the 512 that
// exponentials and MMAs each need. In timing-only variants of the form before (1010 on average) MMAs with no arithmetic
// behind them took 770, the arithmetic with no MMAs 790 (pass 1) and 930 (pass 2, whose normalisers come from shared
// memory). B 8, H 32, T 4096: 1211 -> 965 us; B 1, Hq 32 / Hkv 8, T 32768: 8.59 -> 6.87
// ms against one CTA per 128-token tile with 64-token streamed tiles, two per SM.
//
// The CTA's warps specialise: sixteen take the accumulator rows with tcgen05.ld and do the softmax
// arithmetic; one warp fetches the next item and issues the TMA copies (fixed tiles and a ring of 128B-swizzled
// streamed tiles, with pass 2's query normalisers), two issue the MMAs. The roles hand tiles over through mbarriers
// only; every wait is bounded in time and gives up when another role has failed.
#include <math.h>

#include "mikv_device.cuh"
#include "mikv_prefill.h"
#include "mikv_tcgen05.cuh"

namespace mikv {
namespace {

constexpr int kPfTileBytes = kPfTile * kHeadDim * 2;    // 32 KB: 128 tokens x 128 channels, two 64-channel boxes
constexpr int kPfHalf = kPfTile * 128;                  // one of the boxes
constexpr int kPfCols = 32;                             // accumulator columns of one tcgen05.ld
constexpr int kPfStatBytes = kPfTile * 4;               // pass 2: the streamed queries' log2 normalisers
// Six tiles in shared memory: the fixed ones (the current ones and the next item's first) and the streamed ones in
// flight, of which a small prefill, bound by their latency, wants as many as it can have.
__host__ __device__ constexpr int pf_fix(int MT) { return MT + 1; }
__host__ __device__ constexpr int pf_stages(int MT) { return 6 - pf_fix(MT); }
__host__ __device__ constexpr int pf_bars(int MT) { return 3 * pf_stages(MT) + 2 * pf_fix(MT) + 8 + 4 + 4 + 1; }
__host__ __device__ constexpr int pf_smem(int MT) {
  return 1024 + 6 * kPfTileBytes + pf_stages(MT) * kPfStatBytes + 2 * 16 + 8 * pf_bars(MT);
}
static_assert(pf_smem(1) <= 227 * 1024 && pf_smem(2) <= 227 * 1024, "shared memory of one SM");
constexpr int kPfTmemCols = 512;                        // four accumulators of 128 columns
constexpr int kPfEpi = 16;                              // epilogue warps: four sets of four
constexpr int kPfThreads = 32 * (kPfEpi + 3);           // epilogue, copies, 2 x MMA
__host__ __device__ constexpr int pf_accs(int MT) { return 4 / MT; }  // accumulators of a fixed tile
// Sets that share the columns of an accumulator. With two fixed tiles each of the four accumulators has a set of its
// own; with one, two sets take the even and two the odd ones.
__host__ __device__ constexpr int pf_sharers(int MT) { return 2 / MT; }
__host__ __device__ constexpr int pf_put(int MT) { return 2 * pf_sharers(MT) - 1; }  // sets that hand on their partials

template <int MT>
struct PfSmem {
  static constexpr int kStages = pf_stages(MT), kFix = pf_fix(MT);
  uint32_t base;
  __device__ uint32_t fixed(int f) const { return base + f * kPfTileBytes; }
  __device__ uint32_t stage(int s) const { return base + (kFix + s) * kPfTileBytes; }
  __device__ uint32_t stat(int s) const { return stage(kStages) + s * kPfStatBytes; }
  __device__ uint32_t item(int k) const { return stat(kStages) + 16 * k; }
  __device__ uint32_t bar(int i) const { return item(2) + 8 * i; }
  __device__ uint32_t full(int s) const { return bar(s); }                      // copy landed
  __device__ uint32_t sfree(int s) const { return bar(kStages + s); }         // MMAs read it
  __device__ uint32_t sdone(int s) const { return bar(2 * kStages + s); }     // normalisers read
  __device__ uint32_t ffull(int f) const { return bar(3 * kStages + f); }     // fixed tile landed
  __device__ uint32_t ffree(int f) const { return bar(3 * kStages + kFix + f); }
  __device__ uint32_t tfull(int d) const { return bar(3 * kStages + 2 * kFix + d); }  // accumulator ready
  __device__ uint32_t tempty(int d) const { return bar(3 * kStages + 2 * kFix + 4 + d); }  // and read
  __device__ uint32_t ifull(int k) const { return bar(3 * kStages + 2 * kFix + 8 + k); }   // next item known
  __device__ uint32_t iempty(int k) const { return bar(3 * kStages + 2 * kFix + 10 + k); }
  __device__ uint32_t pfull(int m) const { return bar(3 * kStages + 2 * kFix + 12 + m); }  // row partials there
  __device__ uint32_t pempty(int m) const { return bar(3 * kStages + 2 * kFix + 14 + m); }  // and taken
  __device__ uint32_t drain() const { return bar(pf_bars(MT) - 1); }
};

// Bounded wait that also gives up as soon as another role of the CTA has failed. The clock is read only every 64
// polls: a first read before the polls delays every wait that is not already over.
__device__ __forceinline__ bool pf_wait(uint32_t bar, uint32_t parity, volatile int* fail) {
  uint64_t t0 = 0;
  for (uint32_t i = 1;; ++i) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((i & 63u) == 0) {
      const uint64_t t = global_timer_ns();
      if (t0 == 0) t0 = t;
      if (*fail || t - t0 > kWaitLimitNs) {
        *fail = 1;
        return false;
      }
    }
  }
}

// The eight K = 16 MMAs of one tile: D (128 x 128) = fixed tile x streamed tile^T over the 128 channels.
__device__ __forceinline__ void pf_mma_tile(uint32_t d_tmem, uint32_t fix, uint32_t str) {
  constexpr uint32_t idesc = umma_idesc_bf16_f32(kPfTile, kPfTile);
#pragma unroll
  for (int ks = 0; ks < 8; ++ks) {
    const uint32_t k = (ks >> 2) * kPfHalf + (ks & 3) * 32;  // channels 16 ks .. + 15 inside their 64-channel box
    umma_bf16(d_tmem, umma_desc_sw128(fix + k), umma_desc_sw128(str + k), idesc, ks > 0 ? 1u : 0u);
  }
}

// The work of block index lin. Heads are taken in groups (a.group of them), whole groups one after another: inside a
// group all heads' longest items come first (so the last items of the grid are short ones), and the group's streamed
// operand (of the heads that run at the same time) stays within L2.
// PASS 1: queries q0 .. of query head `head` (b Hq + j), streamed keys 0 .. of its KV head. Pairs of tiles are counted
// from the last, so that of an odd number the first, whose rows are the shortest, is left alone.
// PASS 2: keys q0 .. of KV head `head`, streamed queries q0 .. of its G query heads.
template <int MT, int PASS>
struct PfWork {
  int head, q0, heads, n_tiles, str_row, stat_row, m_used;  // m_used: fixed tiles that are the item's own

  __device__ __forceinline__ PfWork(const PrefillArgs& a, int lin) {
    const int G = a.heads_q / a.heads_kv, n_heads = a.batch * (PASS == 1 ? a.heads_q : a.heads_kv);
    const int tiles = (a.T + kPfTile - 1) / kPfTile, items = (tiles + MT - 1) / MT;
    const int grp = lin / (a.group * items), rem = lin - grp * a.group * items;
    const int n = min(a.group, n_heads - grp * a.group);  // heads of this group
    const int it = rem / n;
    head = grp * a.group + (rem - it * n);
    const int first = PASS == 1 ? tiles - MT * (it + 1) : MT * it;
    m_used = PASS == 1 ? MT + min(first, 0) : min(MT, tiles - first);
    q0 = kPfTile * max(first, 0);
    if (PASS == 1) {
      heads = 1;
      n_tiles = max(first, 0) + m_used;
      str_row = head / G * a.T;
      stat_row = 0;
    } else {
      heads = G;
      n_tiles = tiles - first;
      str_row = head * G * a.T + q0;
      stat_row = head * G * a.T_pad + q0;
    }
  }
  // the columns of streamed tile i that rows 32 quarter .. + 31 of fixed tile m meet, in whole pieces of 32: up to the
  // rows' own tokens (pass 1), from those tokens to the end of the prefill (pass 2); none for rows past the prefill
  __device__ __forceinline__ int col_begin(int m, int i, int quarter) const {
    return PASS == 2 && i == m ? 32 * quarter : 0;
  }
  __device__ __forceinline__ int col_end(int m, int i, int quarter, int T) const {
    if (q0 + kPfTile * m + 32 * quarter >= T) return 0;
    return PASS == 1 ? q0 + kPfTile * (m - i) + 32 * (quarter + 1) : (T - q0 - kPfTile * i + 31) & ~31;
  }
  // tiles wholly on the far side of the diagonal of fixed tile m, and fixed tiles without a token
  __device__ __forceinline__ bool skip(int m, int i) const {
    return m >= m_used || (PASS == 1 ? kPfTile * i >= q0 + kPfTile * (m + 1) : i < m);
  }
};

// Ring position of one role: index, and the parity of the entry's current use.
template <int N>
struct PfRing {
  int s = 0;
  uint32_t ph = 0;
  __device__ __forceinline__ void next() {
    if (++s == N) {
      s = 0;
      ph ^= 1u;
    }
  }
};

// The CTA's items, as one role walks them: the block's own, then the ones launch control handed over. Slot k & 1
// holds the k-th answer; `leave` lets the slot be refilled (one arrival per role thread or warp).
struct PfItems {
  PfRing<2> r;
  int lin;
  __device__ __forceinline__ PfItems() : lin((int)blockIdx.x) {}
  // false: no item is left, or a wait failed
  template <class Smem>
  __device__ __forceinline__ bool fetch(const Smem& sm, volatile int* fail) {
    if (!pf_wait(sm.ifull(r.s), r.ph, fail)) return false;
    return launch_answer(sm.item(r.s), lin);
  }
  template <class Smem>
  __device__ __forceinline__ void leave(const Smem& sm) {
    fence_proxy_async_smem();  // our read of the answer precedes the next asynchronous write of the slot
    mbar_arrive(sm.iempty(r.s));
    r.next();
  }
};

// The pipeline shared by both passes. begin() starts an item on an epilogue thread, tile(w, m, i, col0, v, stat)
// takes its row of one accumulator (columns col0 .. col0 + 31; stat: shared-memory address of those queries'
// normalisers, pass 2). Two threads (MT = 1: four) share a row: put(slot) leaves one's partial result in slot k * 128 +
// row of shared memory (k-th of those that hand theirs on), end(w, row) joins them to its own and closes the row.
// Returns false when a wait timed out (after draining what was in flight); every role leaves through the final barrier.
template <int MT, int PASS, class Begin, class Tile, class Put, class End>
__device__ __forceinline__ bool pf_pipeline(const PrefillArgs& a, Begin begin, Tile tile, Put put, End end) {
  using Work = PfWork<MT, PASS>;
  constexpr bool STATS = PASS == 2;
  constexpr int kCopyWarp = kPfEpi, kMmaWarp = kPfEpi + 1;  // two MMA warps
  constexpr int kStages = pf_stages(MT), kFix = pf_fix(MT);
  constexpr uint32_t kAccs = pf_accs(MT);
  constexpr int kSharers = pf_sharers(MT), kCols = kPfTile / kSharers;  // a set's columns of an accumulator
  extern __shared__ uint8_t smem_raw[];
  __shared__ uint32_t s_tmem;
  __shared__ int s_fail;
  volatile int* fail = &s_fail;
  PfSmem<MT> sm;
  sm.base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const CUtensorMap* map_fix = PASS == 1 ? &a.map_q : &a.map_k;
  const CUtensorMap* map_str = PASS == 1 ? &a.map_k : &a.map_q;
  if (tid == 0) {
    s_fail = 0;
    for (int s = 0; s < kStages; ++s) {
      mbar_init(sm.full(s), 1);
      mbar_init(sm.sfree(s), 2);     // both MMA threads
      mbar_init(sm.sdone(s), kPfEpi / 2);  // the warps whose turn the tile is
    }
    for (int f = 0; f < kFix; ++f) {
      mbar_init(sm.ffull(f), 1);
      mbar_init(sm.ffree(f), 2);     // both MMA threads
    }
    for (int d = 0; d < 4; ++d) {
      mbar_init(sm.tfull(d), 1);
      mbar_init(sm.tempty(d), 4 * kSharers);
    }
    for (int k = 0; k < 2; ++k) {
      mbar_init(sm.ifull(k), 1);
      mbar_init(sm.iempty(k), kPfEpi + 2);  // the epilogue warps and the MMA threads
      mbar_init(sm.pfull(k), 4 * pf_put(MT));
      mbar_init(sm.pempty(k), 4);
    }
    mbar_init(sm.drain(), 2);
    fence_mbar_init();
  }
  if (warp == kCopyWarp && lane == 0) {
    prefetch_tensormap(map_fix);
    prefetch_tensormap(map_str);
  }
  if (warp == kMmaWarp) tmem_alloc(smem_u32(&s_tmem), kPfTmemCols);
  tcgen05_before_sync();
  __syncthreads();
  tcgen05_after_sync();
  const uint32_t tmem = s_tmem;

  // the copy thread's record of what it has in flight (drained if a wait fails)
  PfRing<kStages> rs;
  PfRing<kFix> rf;
  int n_str = 0, n_fix = 0;
  bool asked = false;
  PfItems items;
  if (warp == kCopyWarp) {
    if (lane == 0) {  // next items and copies
      bool ok = true;
      for (int k = 0; ok; ++k) {
        if (k >= 2) ok = pf_wait(sm.iempty(items.r.s), items.r.ph ^ 1u, fail);
        if (!ok) break;
        mbar_arrive_expect_tx(sm.ifull(items.r.s), 16);
        launch_ask(sm.item(items.r.s), sm.ifull(items.r.s));
        asked = true;
        const Work w(a, items.lin);
        const int fix_row = w.head * a.T + w.q0;
        int m = 0;
        for (int j = 0; j < w.heads && ok; ++j)
          for (int i = 0; i < w.n_tiles && ok; ++i) {
            if (m < MT) {  // the item's fixed tiles go between its first streamed ones (both even if one is unused)
              const int last = w.heads * w.n_tiles == 1 ? MT : m + 1;
              for (; m < last && ok; ++m) {
                if (n_fix >= kFix && !(ok = pf_wait(sm.ffree(rf.s), rf.ph ^ 1u, fail))) break;
                ++n_fix;
                mbar_arrive_expect_tx(sm.ffull(rf.s), kPfTileBytes);
                tma_load_2d(sm.fixed(rf.s), map_fix, 0, fix_row + kPfTile * m, sm.ffull(rf.s));
                tma_load_2d(sm.fixed(rf.s) + kPfHalf, map_fix, 64, fix_row + kPfTile * m, sm.ffull(rf.s));
                rf.next();
              }
              if (!ok) break;
            }
            if (n_str >= kStages)
              ok = pf_wait(sm.sfree(rs.s), rs.ph ^ 1u, fail) && (!STATS || pf_wait(sm.sdone(rs.s), rs.ph ^ 1u, fail));
            if (!ok) break;
            ++n_str;
            const int row = w.str_row + j * a.T + kPfTile * i;
            mbar_arrive_expect_tx(sm.full(rs.s), kPfTileBytes + (STATS ? kPfStatBytes : 0));
            tma_load_2d(sm.stage(rs.s), map_str, 0, row, sm.full(rs.s));
            tma_load_2d(sm.stage(rs.s) + kPfHalf, map_str, 64, row, sm.full(rs.s));
            if (STATS)
              bulk_load(sm.stat(rs.s), a.stats + (size_t)w.stat_row + (size_t)j * a.T_pad + kPfTile * i, kPfStatBytes,
                        sm.full(rs.s));
            rs.next();
          }
        if (!ok) break;
        ok = items.fetch(sm, fail);
        if (*fail) break;
        asked = false;
        items.r.next();  // (this thread refills the slots: it does not count among their readers)
      }
    }
  } else if (warp == kMmaWarp || warp == kMmaWarp + 1) {
    if (lane == 0) {  // MMAs: a tile into a free accumulator once its copy landed
      // MT = 2: the thread multiplies fixed tile p with every streamed tile; MT = 1: the two take turns
      const int p = warp - kMmaWarp, m = MT == 2 ? p : 0;
      uint32_t uses = 0;  // accumulator uses of fixed tile m: buffer in the low bits, parity above
      bool ok = true;
      while (ok) {
        const Work w(a, items.lin);
        // The item's fixed tiles, in order: this thread's and (MT = 2) the other's. A parity wait tells only two uses
        // of a slot apart, and the ring's slots change hands (three slots, two tiles an item), so before it leaves the
        // item the thread has seen the other's tile land too, and a slot is free when both have said so. (With each
        // waiting for its own alone, a thread could pass the wait for a slot whose last copy, the other's, had not
        // landed, on the use before that, and release it under the other's MMAs.)
        int f = 0, other = 0;
        uint32_t other_ph = 0;
        for (int k = 0; k < MT; ++k) {
          if (k == m) {
            f = rf.s;
            ok = pf_wait(sm.ffull(f), rf.ph, fail);
          } else {
            other = rf.s;
            other_ph = rf.ph;
          }
          rf.next();
        }
        for (int j = 0; j < w.heads && ok; ++j)
          for (int i = 0; i < w.n_tiles && ok; ++i) {
            ok = pf_wait(sm.full(rs.s), rs.ph, fail);
            if (ok && !w.skip(m, i)) {
              const int d = kAccs * m + (int)(uses % kAccs);
              if (MT == 2 || (int)(uses & 1u) == p) {
                ok = pf_wait(sm.tempty(d), ((uses / kAccs) & 1u) ^ 1u, fail);
                if (!ok) break;
                tcgen05_after_sync();
                pf_mma_tile(tmem + (uint32_t)(d * kPfTile), sm.fixed(f), sm.stage(rs.s));
                umma_commit(sm.tfull(d));
              }
              ++uses;
            }
            if (ok) umma_commit(sm.sfree(rs.s));
            rs.next();
          }
        if (ok && MT == 2) ok = pf_wait(sm.ffull(other), other_ph, fail);
        if (!ok) break;
        umma_commit(sm.ffree(f));
        if (MT == 2) umma_commit(sm.ffree(other));
        ok = items.fetch(sm, fail);
        items.leave(sm);
      }
      umma_commit(sm.drain());  // every MMA issued has completed once both arrive
      if (!mbar_wait(sm.drain(), 0)) record_error(a.status, kErrDrainTimeout);
    }
  } else {  // epilogue warps: fixed tile m, every other of its accumulators (from the p-th), lanes 32 (w % 4) ..,
            // columns first .. first + kCols - 1
    const int set = warp >> 2, p = set & 1, m = MT == 2 ? set >> 1 : 0;
    const int first = MT == 2 ? 0 : kCols * (set >> 1);
    const uint32_t lanes = tmem + ((uint32_t)(32 * (warp & 3)) << 16);
    const int row = kPfTile * m + 32 * (warp & 3) + lane;
    const int part = MT == 2 ? p : set;  // 0: closes the rows
    uint32_t turn = 0, uses = 0, closed = 0;  // whose turn; accumulators taken; parity of the items
    bool ok = true;
    while (ok) {
      const Work w(a, items.lin);
      begin();
      for (int j = 0; j < w.heads && ok; ++j)
        for (int i = 0; i < w.n_tiles; ++i, rs.next()) {
          const bool skip = w.skip(m, i), mine = (int)turn == p;
          if (!skip) turn ^= 1u;
          if (!mine) continue;
          if (skip) {
            // releases its share of the normalisers; the copy has landed, so this is the stage's phase (this set has
            // seen the stage's last use: the tile it took last is at most three back, as all items of a grid have an
            // even or all an odd number of tiles)
            if (STATS) {
              ok = __all_sync(0xffffffffu, pf_wait(sm.full(rs.s), rs.ph, fail));
              if (!ok) break;
              if (lane == 0) mbar_arrive(sm.sdone(rs.s));
            }
            continue;
          }
          const int d = (int)kAccs * m + p + 2 * (int)(uses % (kAccs / 2));
          ok = __all_sync(0xffffffffu, pf_wait(sm.tfull(d), (uses / (kAccs / 2)) & 1u, fail));
          // the staged normalisers: observe their copy's completion directly (it has completed: the MMAs
          // that produced this accumulator waited for it, and the stage is not refilled before sdone)
          if (STATS && ok) ok = __all_sync(0xffffffffu, pf_wait(sm.full(rs.s), rs.ph, fail));
          if (!ok) break;
          ++uses;
          tcgen05_after_sync();
          const int c1 = min(first + kCols, w.col_end(m, i, warp & 3, a.T));
          int c = max(first, w.col_begin(m, i, warp & 3));
          if (c >= c1 && lane == 0) mbar_arrive(sm.tempty(d));  // (nothing to read)
#pragma unroll 1  // (one copy of the arithmetic: the instruction cache was a limit)
          for (; c < c1; c += kPfCols) {
            float v[kPfCols];
            tmem_ld32(lanes + (uint32_t)(d * kPfTile + c), v);
            if (c + kPfCols >= c1) {  // this warp's share of the accumulator has been read
              tcgen05_before_sync();
              __syncwarp();
              if (lane == 0) mbar_arrive(sm.tempty(d));
            }
            tile(w, m, i, c, v, sm.stat(rs.s) + 4 * c);
            __syncwarp();
          }
          if (STATS && lane == 0) mbar_arrive(sm.sdone(rs.s));
        }
      if (!ok) break;
      if (m < w.m_used) {  // the other sets of the fixed tile hand their rows' partials to its first
        if (part != 0) {
          ok = __all_sync(0xffffffffu, pf_wait(sm.pempty(m), closed ^ 1u, fail));
          if (!ok) break;
          put(kPfTile * (part - 1) + row);
          __syncwarp();
          if (lane == 0) mbar_arrive(sm.pfull(m));
        } else {
          ok = __all_sync(0xffffffffu, pf_wait(sm.pfull(m), closed, fail));
          if (!ok) break;
          end(w, row);
          __syncwarp();
          if (lane == 0) mbar_arrive(sm.pempty(m));
        }
        closed ^= 1u;
      }
      ok = __all_sync(0xffffffffu, items.fetch(sm, fail));
      if (lane == 0) {
        items.leave(sm);
      } else {
        items.r.next();
      }
    }
  }
  tcgen05_before_sync();
  __syncthreads();
  const bool failed = s_fail != 0;
  if (failed) {
    if (tid == 0) record_error(a.status, kErrFullTimeout);
    if (warp == kCopyWarp && lane == 0) {  // no copy may outlive the CTA
      for (int v = 0; v < min(n_str, kStages); ++v) {  // the last uses of the ring, latest first
        rs.ph ^= rs.s == 0 ? 1u : 0u;
        rs.s = rs.s == 0 ? kStages - 1 : rs.s - 1;
        if (!mbar_wait(sm.full(rs.s), rs.ph)) record_error(a.status, kErrDrainTimeout);
      }
      for (int v = 0; v < min(n_fix, kFix); ++v) {
        rf.ph ^= rf.s == 0 ? 1u : 0u;
        rf.s = rf.s == 0 ? kFix - 1 : rf.s - 1;
        if (!mbar_wait(sm.ffull(rf.s), rf.ph)) record_error(a.status, kErrDrainTimeout);
      }
      if (asked && !mbar_wait(sm.ifull(items.r.s), items.r.ph)) record_error(a.status, kErrDrainTimeout);
    }
  }
  if (warp == kMmaWarp) {
    __syncwarp();
    tcgen05_after_sync();
    tmem_dealloc(tmem, kPfTmemCols);
  }
  return !failed;
}

// Exact maximum of a row of the tile (four independent chains).
__device__ __forceinline__ float pf_row_max(const float (&v)[kPfCols]) {
  float mx[4] = {v[0], v[1], v[2], v[3]};
#pragma unroll
  for (int j = 4; j < kPfCols; ++j) mx[j & 3] = fmaxf(mx[j & 3], v[j]);
  return fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
}

// The sum of eight partial sums held as four pairs.
__device__ __forceinline__ float pf_sum8(const uint64_t (&acc)[4]) {
  float t[8];
#pragma unroll
  for (int k = 0; k < 4; ++k) f32x2_split(acc[k], t[2 * k], t[2 * k + 1]);
  return ((t[0] + t[1]) + (t[2] + t[3])) + ((t[4] + t[5]) + (t[6] + t[7]));
}

// sum_j 2^(v_j * scale - ref): the exponent formed two columns at a time, eight independent partial sums.
__device__ __forceinline__ float pf_exp_sum(const float (&v)[kPfCols], float scale, float ref) {
  const uint64_t s2 = f32x2(scale, scale), r2 = f32x2(-ref, -ref);
  uint64_t acc[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll
  for (int j = 0; j < kPfCols / 2; ++j) {
    float x0, x1;
    f32x2_split(fma_f32x2(f32x2(v[2 * j], v[2 * j + 1]), s2, r2), x0, x1);
    acc[j & 3] = add_f32x2(acc[j & 3], f32x2(fast_exp2(x0), fast_exp2(x1)));
  }
  return pf_sum8(acc);
}

// A row's sum from its closing thread's and those handed on. Which of two accumulators an item begins with depends on
// the items its block had before, so the two that share columns are added first: their sum is the same either way.
template <int MT, class Part>
__device__ __forceinline__ float pf_join(float own, Part part) {
  const float sum = own + part(0);
  if constexpr (MT == 2) return sum;
  else return sum + (part(1) + part(2));
}

// ------------------------------------------------------------------------------- pass 1: row statistics
//
// Per query row each thread accumulates its share of the softmax normaliser against a reference r (log2 units): the
// exact maximum of the first 32 columns it reads, raised only when a later sum would leave the fp32 range (a logit more
// than 64 above r, rare), so most columns need no maximum at all. The pair (r, sum_t 2^(s_t - r)) defines the same
// normaliser as the true maximum; the kernel stores its log2, r + log2(sum), negated (pass 2 adds it).

template <int MT>
__global__ void __launch_bounds__(kPfThreads, 1) prefill_rows_kernel(const __grid_constant__ PrefillArgs a) {
  using Work = PfWork<MT, 1>;
  __shared__ float s_r[MT * pf_put(MT) * kPfTile], s_l[MT * pf_put(MT) * kPfTile];  // the partials handed on
  float r = -INFINITY, l = 0.f;  // over this thread's tiles and columns
  pf_pipeline<MT, 1>(
      a,
      [&] {
        r = -INFINITY;
        l = 0.f;
      },
      [&](const Work& w, int m, int i, int col0, float (&v)[kPfCols], uint32_t) {
        const int k0 = kPfTile * i + col0;
        if (k0 + kPfCols > w.q0 + kPfTile * m) {  // keys after the query do not count
          const int q = w.q0 + kPfTile * m + (int)(threadIdx.x & 127u);
#pragma unroll
          for (int j = 0; j < kPfCols; ++j)
            if (k0 + j > q) v[j] = -INFINITY;
        }
        float sum = pf_exp_sum(v, a.scale_log2, r);
        // the row's first columns (r = -inf), or a logit far above the reference: move the reference to the maximum
        if (__any_sync(0xffffffffu, !(sum <= 0x1p64f))) {
          float rn = r;
          if (!(sum <= 0x1p64f)) rn = fmaxf(r, pf_row_max(v) * a.scale_log2);
          sum = rn == -INFINITY ? 0.f : pf_exp_sum(v, a.scale_log2, rn);
          if (rn != r) l *= fast_exp2(r - rn);
          r = rn;
        }
        l += sum;
      },
      [&](int slot) {
        s_r[slot] = r;
        s_l[slot] = l;
      },
      [&](const Work& w, int row) {  // the partials against the largest reference
        const int q = w.q0 + row;
        float rm = r;
#pragma unroll
        for (int k = 0; k < pf_put(MT); ++k) rm = fmaxf(rm, s_r[kPfTile * k + row]);
        const float lt = pf_join<MT>(r == -INFINITY ? 0.f : l * fast_exp2(r - rm), [&](int k) {
          const float r2 = s_r[kPfTile * k + row];
          return r2 == -INFINITY ? 0.f : s_l[kPfTile * k + row] * fast_exp2(r2 - rm);
        });
        a.stats[(size_t)w.head * a.T_pad + q] = q < a.T ? -(rm + log2f(lt)) : -INFINITY;
      });
}

// ------------------------------------------------------------------------------ pass 2: column sums

template <int MT>
__global__ void __launch_bounds__(kPfThreads, 1) prefill_cols_kernel(const __grid_constant__ PrefillArgs a) {
  using Work = PfWork<MT, 2>;
  __shared__ float s_cs[MT * pf_put(MT) * kPfTile];  // the sums handed on
  float cs = 0.f;
  pf_pipeline<MT, 2>(
      a, [&] { cs = 0.f; },
      [&](const Work& w, int m, int i, int col0, float (&v)[kPfCols], uint32_t stat) {
        const int q0 = w.q0 + kPfTile * i + col0;
        // minus the log2 normalisers of these queries, staged with the tile (-inf for padding: they weigh nothing)
        uint32_t c[kPfCols / 4][4];
#pragma unroll
        for (int j = 0; j < kPfCols / 4; ++j) lds_vec<4>(stat + 16 * j, c[j]);
        // queries before the key do not attend to it; rows past the prefill belong to another head
        if (i == m || q0 + kPfCols > a.T) {
          const int key = w.q0 + kPfTile * m + (int)(threadIdx.x & 127u);
#pragma unroll
          for (int j = 0; j < kPfCols; ++j)
            if (q0 + j < key || q0 + j >= a.T) v[j] = -INFINITY;
        }
        const uint64_t s2 = f32x2(a.scale_log2, a.scale_log2);
        uint64_t acc[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll
        for (int j = 0; j < kPfCols / 2; ++j) {
          float x0, x1;
          f32x2_split(fma_f32x2(f32x2(v[2 * j], v[2 * j + 1]), s2,
                                f32x2(__uint_as_float(c[j / 2][2 * (j & 1)]), __uint_as_float(c[j / 2][2 * (j & 1) + 1]))),
                      x0, x1);
          acc[j & 3] = add_f32x2(acc[j & 3], f32x2(fast_exp2(x0), fast_exp2(x1)));
        }
        cs += pf_sum8(acc);
      },
      [&](int slot) { s_cs[slot] = cs; },
      [&](const Work& w, int row) {
        const float sum = pf_join<MT>(cs, [&](int k) { return s_cs[kPfTile * k + row]; });
        if (w.q0 + row < a.T) a.scores[(size_t)w.head * a.T + w.q0 + row] = sum;
      });
}

template <class Kernel>
cudaError_t pf_launch(Kernel kernel, int smem, PrefillArgs a, int items, int n_heads, int num_sms, cudaStream_t st) {
  const int per = (2 * num_sms + items - 1) / items;  // heads per group: about two rounds of the resident CTAs,
  const int groups = max(1, n_heads / per);           // in groups of like size: the long items of a small last group
  a.group = (n_heads + groups - 1) / groups;          // ran alone at the end (80 heads as 76 and 4, T 777: 46 / 37 us)
  kernel<<<items * n_heads, kPfThreads, smem, st>>>(a);
  return cudaGetLastError();
}

// One pass with items of two fixed tiles when there are then at least three for two SMs, else of one, which gives a
// small prefill twice the CTAs. us of a pass, one tile against two, by the items of two: rows, 96: 9.9 / 10.7, 160: 13.2
// / 14.5, 192: 17.2 / 20.2, 256: 23.5 / 26.4 and 13.7 / 11.7, 384: 17.6 / 15.5; columns, 72: 61.9 / 100.7, 152: 131.6 /
// 150.9, 192: 17.9 / 22.0, 256: 17.6 / 19.0 and 13.5 / 11.9, 384: 48.6 / 44.8, 512: 589 / 486.
template <int PASS>
cudaError_t pf_pass(const PrefillArgs& a, int num_sms, cudaStream_t st) {
  constexpr auto one = PASS == 1 ? prefill_rows_kernel<1> : prefill_cols_kernel<1>;
  constexpr auto two = PASS == 1 ? prefill_rows_kernel<2> : prefill_cols_kernel<2>;
  static bool configured = false;
  if (!configured) {
    cudaError_t e = cudaFuncSetAttribute(one, cudaFuncAttributeMaxDynamicSharedMemorySize, pf_smem(1));
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(two, cudaFuncAttributeMaxDynamicSharedMemorySize, pf_smem(2));
    if (e != cudaSuccess) return e;
    configured = true;
  }
  const int tiles = (a.T + kPfTile - 1) / kPfTile, n_heads = a.batch * (PASS == 1 ? a.heads_q : a.heads_kv);
  const int items2 = (tiles + 1) / 2;
  return 2ll * items2 * n_heads >= 3ll * num_sms ? pf_launch(two, pf_smem(2), a, items2, n_heads, num_sms, st)
                                                  : pf_launch(one, pf_smem(1), a, tiles, n_heads, num_sms, st);
}

}  // namespace

cudaError_t launch_prefill(const PrefillArgs& a, int num_sms, cudaStream_t st) {
  const cudaError_t e = pf_pass<1>(a, num_sms, st);
  return e != cudaSuccess ? e : pf_pass<2>(a, num_sms, st);
}

}  // namespace mikv
