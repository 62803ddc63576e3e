// One-pass building blocks of the compositing binning: a stable radix-sort pass and an exclusive
// scan whose blocks learn what lies before them from their predecessors' published counts
// (decoupled look-back, Merrill & Garland 2016; as a radix pass, Adinets & Merrill 2022), so that
// a pass reads and writes its data once, in one launch. A block takes its place from a ticket
// counter: the blocks it looks back at have smaller tickets, so they are running or done, and
// publish their own counts before they wait. Every wait is bounded (one second of waiting or
// kWaitLimit polls); a block that gives up sets the library's device error word and `failed` in the
// workspace's header, which later blocks and kernels read before they trust any list.
#pragma once

#include <stdint.h>

#include "nasg_tma.cuh"
#include "nasg_wait.h"

namespace nasg {
namespace sort {

constexpr int kBins = 256;               // at most 8 bits per digit
constexpr uint32_t kNone = 0xffffffffu;  // key of an entry that is dropped
constexpr int kWindow = 16;               // predecessors read at once

// A published count: two flag bits, a six-bit tag (which pass wrote it, so that passes that
// share a zeroed table need no clearing between them) and 56 bits of count.
constexpr unsigned long long kOwn = 1ull << 62, kAll = 2ull << 62, kGone = 3ull << 62;
constexpr unsigned long long kCount = (1ull << 56) - 1;
__device__ __forceinline__ unsigned long long tag_bits(uint32_t tag) { return (unsigned long long)(tag) << 56; }

__device__ __forceinline__ unsigned long long ld_state(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_state(unsigned long long* p, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ bool ready(unsigned long long v, uint32_t tag) {
  return (v >> 62) != 0 && ((v >> 56) & 63u) == tag;
}

// Polls a predecessor's state until it is published; a state of kGone when it gave up.
static __device__ __noinline__ unsigned long long wait_state(const unsigned long long* p, uint32_t tag, uint32_t limit,
                                                            int* err) {
  WaitClock clock(global_ns());
  for (uint32_t it = 1; it < limit; ++it) {
    const unsigned long long v = ld_state(p);
    if (ready(v, tag)) return v;
    if ((it & 255u) == 0 && clock.over(global_ns(), kWaitNs)) break;
  }
  if (err) atomicExch(err, NASG_DEVERR_WAIT_TIMEOUT);
  return kGone;
}

// Sum of the counts published before `block` in column `col` of states [blocks][stride]. kWindow
// predecessors are read at once: walked one by one, the read latency of a few hundred blocks
// that start together would be the pass's time. False when a wait gave up.
__device__ __forceinline__ bool look_back(const unsigned long long* states, int stride, int col, uint32_t block,
                                          uint32_t tag, uint32_t limit, int* err, unsigned long long* before) {
  unsigned long long sum = 0;
  for (int64_t p = int64_t(block) - 1; p >= 0; p -= kWindow) {
    unsigned long long w[kWindow];
#pragma unroll
    for (int i = 0; i < kWindow; ++i)
      w[i] = p - i >= 0 ? ld_state(states + (p - i) * stride + col) : (kAll | tag_bits(tag));
#pragma unroll
    for (int i = 0; i < kWindow; ++i) {
      if (!ready(w[i], tag)) w[i] = wait_state(states + (p - i) * stride + col, tag, limit, err);
      const unsigned long long flag = w[i] & kGone;
      if (flag == kGone) return false;
      sum += w[i] & kCount;
      if (flag == kAll) {
        *before = sum;
        return true;
      }
    }
  }
  *before = sum;
  return true;
}

// The same for one column, by a whole warp: 32 predecessors at once. Every lane gets the sum.
__device__ __forceinline__ bool look_back_warp(const unsigned long long* states, uint32_t block, uint32_t tag,
                                               uint32_t limit, int* err, unsigned long long* before) {
  const int lane = threadIdx.x & 31;
  unsigned long long sum = 0;
  for (int64_t p = int64_t(block) - 1; p >= 0; p -= 32) {
    unsigned long long v = kAll | tag_bits(tag);
    if (p - lane >= 0) {
      v = ld_state(states + p - lane);
      if (!ready(v, tag)) v = wait_state(states + p - lane, tag, limit, err);
    }
    const unsigned long long flag = v & kGone;
    if (__any_sync(0xffffffffu, flag == kGone)) return false;
    const uint32_t all = __ballot_sync(0xffffffffu, flag == kAll);
    const int end = all ? __ffs(int(all)) - 1 : 31;  // the nearest predecessor that knows its sum
    unsigned long long add = lane <= end ? v & kCount : 0ull;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) add += __shfl_xor_sync(0xffffffffu, add, o);
    sum += add;
    if (all) break;
  }
  *before = sum;
  return true;
}

// Exclusive scan over the block's THREADS threads (warp_tot: one word per warp); *total gets the
// block's sum.
template <int THREADS>
__device__ __forceinline__ uint32_t block_scan(uint32_t x, uint32_t* warp_tot, uint32_t* total) {
  constexpr int kWarps = THREADS / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t inc = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) warp_tot[warp] = inc;
  __syncthreads();
  uint32_t w = lane < kWarps ? warp_tot[lane] : 0u;
#pragma unroll
  for (int o = 1; o < kWarps; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, w, o);
    if (lane >= o) w += y;
  }
  __syncthreads();
  *total = __shfl_sync(0xffffffffu, w, kWarps - 1);
  const uint32_t before = __shfl_sync(0xffffffffu, w, warp ? warp - 1 : 0);
  return (warp ? before : 0u) + inc - x;
}

// Shared memory of a sort block.
template <int THREADS, int ITEMS>
struct Block {
  static constexpr int kEntries = THREADS * ITEMS;
  static constexpr int kWarps = THREADS / 32;
  uint32_t key[kEntries];
  uint32_t val[kEntries];
  uint32_t count[kWarps][kBins];  // entries per warp and digit, then the offsets of the warps
  uint32_t start[kBins];          // digit's first place in the sorted block
  uint32_t base[kBins];           // global place of the digit's first entry, less start
  uint32_t warp_tot[kWarps];
  uint32_t ticket;
  uint32_t stop;                  // an earlier wait gave up, as one thread saw it
};

// What a sort block needs beside its entries.
struct Pass {
  const uint32_t* hist;        // entries per digit, whole input
  unsigned long long* states;  // [blocks][bins]
  uint32_t* ticket;            // zeroed
  uint32_t* failed;            // of the workspace's header
  int* err;
  int shift, bits;
  uint32_t tag;
  uint32_t limit;              // polls of a wait
};

// Bound: instructions and the wait for the look-back (a pass over 1e6 depth keys 17 us, as histogram, three
// scan launches and scatter 37 us; over the pairs of a 1080p frame 72 us, issue 56 % active, ALU 64 %).
// Sorts the block's entries (thread's item i at place warp * 32 * ITEMS + 32 i + lane of the
// block's input; kNone is dropped) by one digit, stable, into s.key / s.val, and finds where
// each digit's run goes. Returns the number of entries, or a negative number when a wait gave up.
// digit_base: the thread's exclusive sum of hist. Every thread of the block calls it.
template <int THREADS, int ITEMS, bool MATCH>
__device__ __forceinline__ int sort_block(Block<THREADS, ITEMS>& s, const Pass& ps, uint32_t block, uint32_t digit_base,
                                          const uint32_t (&key)[ITEMS], const uint32_t (&val)[ITEMS]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, t = threadIdx.x;
  const int bins = 1 << ps.bits;
  const uint32_t mask = uint32_t(bins) - 1u, lt = (1u << lane) - 1u;
  uint32_t rank[ITEMS];
#pragma unroll
  for (int i = t; i < THREADS / 32 * kBins; i += THREADS) (&s.count[0][0])[i] = 0;
  __syncthreads();
  // lanes of the warp with the same digit: by match.any, whose time grows with the number of
  // different digits in the warp (MATCH: passes whose neighbours share digits, the lists' columns and
  // the depths' upper bits: 109 us, bit by bit 133, and 12 us, 16, at 1080p), or bit by bit (the others: 69
  // against 78 us and 17 against 20 us). The first of them adds their number to the warp's count, in
  // the items' order.
#pragma unroll
  for (int i = 0; i < ITEMS; ++i) {
    const bool ok = key[i] != kNone;
    const uint32_t d = (key[i] >> ps.shift) & mask;
    uint32_t peers;
    if (MATCH) {
      peers = __match_any_sync(0xffffffffu, ok ? d : kNone);
    } else {
      peers = __ballot_sync(0xffffffffu, ok);
#pragma unroll
      for (int b = 0; b < 8; ++b) {
        if (b < ps.bits) {
          const bool one = (d >> b) & 1u;
          const uint32_t vote = __ballot_sync(0xffffffffu, one);
          peers &= one ? vote : ~vote;
        }
      }
    }
    const int lead = __ffs(int(peers)) - 1;
    uint32_t pre = 0;
    if (ok && lane == lead) pre = atomicAdd(&s.count[warp][d], uint32_t(__popc(peers)));
    __syncwarp();
    pre = __shfl_sync(0xffffffffu, pre, lead & 31);
    rank[i] = pre + __popc(peers & lt);
  }
  __syncthreads();
  uint32_t cnt = 0;
  if (t < bins) {
#pragma unroll 8
    for (int w = 0; w < THREADS / 32; ++w) {
      const uint32_t c = s.count[w][t];
      s.count[w][t] = cnt;
      cnt += c;
    }
  }
  unsigned long long* state = ps.states + int64_t(block) * bins + t;
  if (t < bins) st_state(state, (block == 0 ? kAll : kOwn) | tag_bits(ps.tag) | cnt);
  uint32_t n;
  const uint32_t start = block_scan<THREADS>(cnt, s.warp_tot, &n);
  if (t < bins) s.start[t] = start;
  __syncthreads();
  // into sorted order before the look-back, which then has the registers to itself
#pragma unroll
  for (int i = 0; i < ITEMS; ++i) {
    if (key[i] == kNone) continue;
    const uint32_t d = (key[i] >> ps.shift) & mask;
    const uint32_t p = s.start[d] + s.count[warp][d] + rank[i];
    s.key[p] = key[i];
    s.val[p] = val[i];
  }
  unsigned long long before = 0;
  bool ok = true;
  if (block > 0 && t < bins) {
    ok = look_back(ps.states, bins, t, block, ps.tag, ps.limit, ps.err, &before);
    st_state(state, (ok ? kAll : kGone) | tag_bits(ps.tag) | ((before + cnt) & kCount));
  }
  if (t < bins) s.base[t] = digit_base + uint32_t(before) - start;
  if (__syncthreads_or(!ok)) {
    if (t == 0) *ps.failed = 1;
    return -1;
  }
  return int(n);
}

}  // namespace sort
}  // namespace nasg
