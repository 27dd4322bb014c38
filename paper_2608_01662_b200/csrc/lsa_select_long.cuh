// Exact top-k of a long row in one pass over it: the same selection as block_select_topk (lsa_select.cuh: largest keys
// first, ties by position, output in ascending position).
//
// A radix select reads the row seven times (the count and digit passes, then twice for the ordered compaction).  Of a
// long row few items can be selected, so here a sample of it names a key that k items almost surely reach, one pass
// collects the items at or above that key, and the rest works on them alone, in shared memory: the radix passes find the
// k-th largest, the selected items set their bits in a bitmap of the row, and the bitmap is read out in order.  If the
// sample misled - fewer than k items collected, or more than there is room for - the caller takes the radix select
// instead: the result never depends on the sample.
//
// With CLUSTER the row is cut into one contiguous piece per block of a cluster (few long rows: the flat indexer in
// decode): every block collects from its piece, the digit counts meet in the first block's shared memory, and each block
// writes its part of the output.
//
// What bounds it: the read of the row and, per row, some 15 000 cycles that do not depend on its length.  1000 rows of 65536
// scores, k = 2048: 126 us (radix select 689); 2048 rows of 131072: 398 us (2551); 16 rows of 74000 on clusters: 23 us (53).
#pragma once

#include "lsa_select_cluster.cuh"

namespace lsa {

constexpr int kLongBinBits = 12, kLongBins = 1 << kLongBinBits;   // sample histogram: the top bits of a key
constexpr int kLongMinRow = 16384;           // rows below this are left to the radix select

// Room for collected items: what k items need with the sample's margin (six standard deviations and a bin's width).
__host__ __device__ constexpr int long_cap(int k) { return k <= 2048 ? 4608 : 2 * k + k / 4; }

__device__ __forceinline__ uint4 load_quad(const void* p) {
  uint4 v;
  asm volatile("ld.global.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
  return v;
}

struct alignas(16) LongScratch {
  uint32_t hist[4][256];      // digit counts of this block, one histogram per pass
  uint32_t sel[kClusterSel], eq[kClusterSel];   // CLUSTER, first block: selected items / ties per block
  uint32_t cnt, total, overflow, top;           // collected here; CLUSTER, first block: in all, somebody ran out of room, largest
  uint32_t bound, prefix, remaining, whole;
  uint32_t warp_sum[kSelWarps];
};
struct LongAll {
  uint32_t hist[4][256];      // CLUSTER, first block: digit counts of the whole row
};
static_assert(sizeof(LongScratch) % 16 == 0, "what follows it is read 16 bytes at a time");
static_assert(kLongBins * 4 <= long_cap(1) * 8, "the sample's histogram fits the lists");

// Dynamic shared memory of a block: the scratch, the collected keys and items (the sample's histogram lies there before),
// and a bit per item of the block's piece.
__host__ __device__ constexpr size_t long_smem_bytes(bool cluster, int cap, int64_t piece) {
  return sizeof(LongScratch) + (cluster ? sizeof(LongAll) : 0) + static_cast<size_t>(cap) * 8 + static_cast<size_t>((piece + 31) / 32) * 4;
}
// Items of a block's piece of a row of n.
__host__ __device__ constexpr int long_piece(int n) { return ((n + kClusterSel - 1) / kClusterSel + 31) & ~31; }

// Sum of v over the 256 threads before this one (ascending), and over all of them.
__device__ __forceinline__ uint32_t block_exclusive_sum(uint32_t v, uint32_t* warp_sum, uint32_t* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t incl = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t x = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += x;
  }
  __syncthreads();   // (the sums of an earlier call have been read)
  if (lane == 31) warp_sum[warp] = incl;
  __syncthreads();
  uint32_t before = 0, all = 0;
#pragma unroll
  for (int w = 0; w < kSelWarps; ++w) {
    before += w < warp ? warp_sum[w] : 0u;
    all += warp_sum[w];
  }
  *total = all;
  return before + incl - v;
}

// KeyF: uint32_t operator()(int i) (0 = absent; called for i of [0, n)); Raw load(int i) and keys(Raw, i, uint32_t (&k)[4]): what
// the keys of i .. i + 3 are made of (i a multiple of four, all of them in [0, n)), and the keys; kQuads: such loads per lane and
// step.  EmitF: void operator()(int r, int i): item i is
// the r-th of the selection.  AbsentF: void operator()(int r): there is no r-th item.  Every thread of the block (CLUSTER: of
// every block of the cluster, kClusterSel along x) calls this with the same arguments.  Returns how many items were
// selected, or -1: nothing has been written, take the radix select (the same answer in every block).
template <bool CLUSTER, class KeyF, class EmitF, class AbsentF>
__device__ int long_select(KeyF key, EmitF emit, AbsentF absent, int n, int k, int cap, uint8_t* smem) {
  namespace cs = cluster_sel;
  if (k <= 0) return 0;   // (the same in every block; no key is the k-th largest)
  LongScratch& sc = *reinterpret_cast<LongScratch*>(smem);
  LongAll& all = *reinterpret_cast<LongAll*>(smem + sizeof(LongScratch));
  uint32_t* ck = reinterpret_cast<uint32_t*>(smem + sizeof(LongScratch) + (CLUSTER ? sizeof(LongAll) : 0));
  uint32_t* ci = ck + cap;
  uint32_t* bits = ci + cap;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t me = CLUSTER ? cs::rank() : 0u;
  const int piece = CLUSTER ? long_piece(n) : n;
  const int b0 = CLUSTER ? min(n, static_cast<int>(me) * piece) : 0, b1 = min(n, b0 + piece);
  const int n_words = (b1 - b0 + 31) >> 5;

  // ---- set-up, and the key to collect from
  for (int i = tid; i < 4 * 256; i += kSelThreads) {
    (&sc.hist[0][0])[i] = 0;
    if (CLUSTER) (&all.hist[0][0])[i] = 0;
  }
  for (int i = tid; i < n_words; i += kSelThreads) bits[i] = 0;
  if (tid == 0) {
    sc.cnt = sc.total = sc.overflow = sc.top = 0;
    sc.bound = 1u;
  }
  if (piece > cap) {   // (else everything has room; the same in every block)
    uint32_t* bins = ck;
    for (int i = tid; i < kLongBins; i += kSelThreads) bins[i] = 0;
    __syncthreads();
    // Evenly spaced quads of items, one item of 16 or more of a block's own row: 2048 items of 65536 are then collected as
    // 3280 +- 230.  (The blocks of a cluster sample the whole row each, and have room for much more than their part.  Quads,
    // because single items cost a memory sector each: 62 us of the 159 us of 1000 rows were what did not depend on their length.)
    const int m_shift = CLUSTER ? (n > 131072 ? 14 : 12) : max(12, 28 - __clz(n - 1));
    for (int q0 = tid; q0 < 1 << (m_shift - 2); q0 += 4 * kSelThreads) {
      typename KeyF::Raw raw[4];
      int at[4];
      uint32_t kk[4][4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        at[u] = static_cast<int>(static_cast<int64_t>(q0 + u * kSelThreads) * n >> (m_shift - 2)) & ~3;
        raw[u] = key.load(at[u]);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) key.keys(raw[u], at[u], kk[u]);
#pragma unroll
      for (int u = 0; u < 16; ++u)
        if (kk[u >> 2][u & 3] != 0u) atomicAdd(&bins[kk[u >> 2][u & 3] >> (32 - kLongBinBits)], 1u);
    }
    __syncthreads();
    const float expect = static_cast<float>(k) * static_cast<float>(1 << m_shift) / static_cast<float>(n);
    const uint32_t want = static_cast<uint32_t>(expect + 6.f * sqrtf(expect) + 8.f);
    constexpr int kPer = kLongBins / kSelThreads;
    const uint4* mine = reinterpret_cast<const uint4*>(bins + kLongBins - kPer * (tid + 1));   // from the top bin down
    uint32_t c[kPer], sum = 0, total;
#pragma unroll
    for (int i = 0; i < kPer / 4; ++i) {
      const uint4 x = mine[i];
      c[4 * i] = x.x; c[4 * i + 1] = x.y; c[4 * i + 2] = x.z; c[4 * i + 3] = x.w;
      sum += x.x + x.y + x.z + x.w;
    }
    uint32_t run = block_exclusive_sum(sum, sc.warp_sum, &total);
    if (run < want && want <= run + sum) {   // one thread, or none (then everything present is collected)
#pragma unroll
      for (int i = kPer - 1; i >= 0; --i) {
        if (run < want && want <= run + c[i]) {
          // inside the bin, as far below its upper end as the share of its items that is still wanted (a bin's width is up to
          // an eighth of the value: at its lower end, now and then a row's items would not have had room)
          constexpr int kWidth = 32 - kLongBinBits;
          const uint32_t lower = static_cast<uint32_t>(kLongBins - kPer * (tid + 1) + i) << kWidth;
          const float above = 1.f - static_cast<float>(want - run) / static_cast<float>(c[i]);
          sc.bound = max(1u, lower + static_cast<uint32_t>(above * static_cast<float>(1u << kWidth)));
        }
        run += c[i];
      }
    }
  }
  __syncthreads();
  const uint32_t bound = sc.bound;

  // (what is collected is kept as its distance from the bound)
  // ---- collect: a warp takes 128 items per quad of a lane at a time, the next ones on their way as they lie in memory (their
  // loads are volatile: left to itself the compiler moves them down to where they are used, to save the registers, and the
  // read of 2048 rows of 131072 took 764 us instead of 626)
  constexpr int kQuads = KeyF::kQuads, kStep = 128 * kQuads;
  const int full = (b1 - b0) / kStep;   // whole steps
  {
    typename KeyF::Raw now[kQuads], next[kQuads];
    auto load = [&](int step, typename KeyF::Raw (&raw)[kQuads]) {
#pragma unroll
      for (int u = 0; u < kQuads; ++u) raw[u] = key.load(b0 + step * kStep + 128 * u + 4 * lane);
    };
    int step = warp;
    if (step < full) load(step, now);
    for (; step < full; step += kSelWarps) {
      if (step + kSelWarps < full) load(step + kSelWarps, next);
      uint32_t kk[kQuads][4], hit = 0;
#pragma unroll
      for (int u = 0; u < kQuads; ++u) key.keys(now[u], b0 + step * kStep + 128 * u + 4 * lane, kk[u]);
#pragma unroll
      for (int u = 0; u < 4 * kQuads; ++u) hit |= (kk[u >> 2][u & 3] >= bound ? 1u : 0u) << u;
      const uint32_t n_hit = __popc(hit);
      uint32_t incl = n_hit;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const uint32_t x = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += x;
      }
      uint32_t at = 0;
      if (lane == 31 && incl) at = atomicAdd(&sc.cnt, incl);
      at = __shfl_sync(0xffffffffu, at, 31) + incl - n_hit;
      if (hit && at + n_hit <= static_cast<uint32_t>(cap)) {   // (else there is no room: the count says so)
#pragma unroll
        for (int u = 0; u < 4 * kQuads; ++u)
          if (hit >> u & 1u) {
            ck[at] = kk[u >> 2][u & 3] - bound;
            ci[at++] = static_cast<uint32_t>(step * kStep + 128 * (u >> 2) + 4 * lane + (u & 3));
          }
      }
#pragma unroll
      for (int u = 0; u < kQuads; ++u) now[u] = next[u];
    }
    for (int i = b0 + full * kStep + tid; i < b1; i += kSelThreads) {
      const uint32_t x = key(i);
      if (x >= bound) {
        const uint32_t at = atomicAdd(&sc.cnt, 1u);
        if (at < static_cast<uint32_t>(cap)) {
          ck[at] = x - bound;
          ci[at] = static_cast<uint32_t>(i - b0);
        }
      }
    }
  }
  __syncthreads();
  const uint32_t got = sc.cnt;
  {
    uint32_t top = 0;
    if (got <= static_cast<uint32_t>(cap))
      for (uint32_t e = tid; e < got; e += kSelThreads) top = max(top, ck[e]);
    top = __reduce_max_sync(0xffffffffu, top);
    if (lane == 0) atomicMax(&sc.top, top);
    __syncthreads();
  }
  uint32_t total = got;
  bool failed = got > static_cast<uint32_t>(cap);
  uint32_t scratch0 = 0;   // the first block's scratch
  auto remote = [&](const void* p) -> uint32_t { return scratch0 + (smem_u32(p) - smem_u32(&sc)); };
  if constexpr (CLUSTER) {
    scratch0 = cs::at_rank0(&sc);
    cs::sync();   // every block's scratch is set up
    if (tid == 0) {
      cs::add_remote(remote(&sc.total), got);
      if (me != 0) cs::max_remote(remote(&sc.top), sc.top);
      if (failed) cs::add_remote(remote(&sc.overflow), 1u);
    }
    cs::sync();
    total = cs::load_remote(remote(&sc.total));
    failed = cs::load_remote(remote(&sc.overflow)) != 0u;
  }
  if (failed || (bound > 1u && total < static_cast<uint32_t>(k))) {
    if constexpr (CLUSTER) cs::sync();   // nobody goes on while its scratch may still be read
    return -1;
  }

  // ---- the k-th largest of the collected keys: take keys > T and the first need_eq keys == T, or (take_from) keys >= T.
  // The digits start at the highest bit in which a key can differ from the bound: the top bits, which nearly all of them
  // share, would be thousands of additions to one address.
  uint32_t T = 0;
  int need_eq = 0;
  bool take_from = true;   // everything collected
  if (total > static_cast<uint32_t>(k)) {
    const uint32_t top = CLUSTER ? cs::load_remote(remote(&sc.top)) : sc.top;
    int high = 32 - __clz(top | 1u);   // bits from here on are decided
    uint32_t prefix = 0, remaining = static_cast<uint32_t>(k);
    take_from = false;
#pragma unroll 1
    for (int pass = 0; pass < 4 && high > 0 && !take_from; ++pass) {
      const int shift = max(0, high - 8);
      const uint32_t digits = (1u << (high - shift)) - 1u;
      for (uint32_t e = tid; e < got; e += kSelThreads) {
        const uint32_t x = ck[e];
        if (high == 32 || (x >> high) == (prefix >> high)) atomicAdd(&sc.hist[pass][(x >> shift) & digits], 1u);
      }
      __syncthreads();
      if constexpr (CLUSTER) {
        const uint32_t v = sc.hist[pass][tid];
        if (v) cs::add_remote(remote(&all.hist[pass][tid]), v);
        cs::sync();
      }
      if (warp == 0) {   // lane l takes bins 255 - 8 l .. 248 - 8 l
        uint32_t c[8], sum = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int bin = 255 - 8 * lane - i;
          c[i] = CLUSTER ? cs::load_remote(remote(&all.hist[pass][bin])) : sc.hist[pass][bin];
          sum += c[i];
        }
        uint32_t incl = sum;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
          const uint32_t x = __shfl_up_sync(0xffffffffu, incl, d);
          if (lane >= d) incl += x;
        }
        uint32_t run = incl - sum;
        if (run < remaining && remaining <= incl) {
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            if (run < remaining && remaining <= run + c[i]) {
              sc.prefix = prefix | (static_cast<uint32_t>(255 - 8 * lane - i) << shift);
              sc.remaining = remaining - run;
              sc.whole = remaining - run == c[i];
            }
            run += c[i];
          }
        }
      }
      __syncthreads();
      prefix = sc.prefix;
      remaining = sc.remaining;
      take_from = sc.whole != 0u;   // the whole bin is taken
      high = shift;
    }
    T = prefix;
    if (!take_from) need_eq = static_cast<int>(remaining);
  }

  // ---- of the ties, the first need_eq in item order
  uint32_t eq_all = 0;
  int eq_quota = 0;          // of this block's ties
  if (!take_from) {          // (the same in every block)
    uint32_t eq = 0;
    for (uint32_t e = tid; e < got; e += kSelThreads) eq += ck[e] == T;
    (void)block_exclusive_sum(eq, sc.warp_sum, &eq_all);
    eq_quota = min(static_cast<int>(eq_all), need_eq);
    if constexpr (CLUSTER) {
      if (tid == 0) cs::store_remote(remote(&sc.eq[me]), eq_all);
      cs::sync();
      int before = 0;
      for (uint32_t r = 0; r < me; ++r) before += static_cast<int>(cs::load_remote(remote(&sc.eq[r])));
      eq_quota = min(static_cast<int>(eq_all), max(0, need_eq - before));
    }
  }
  uint32_t eq_end = 0xffffffffu;   // ties at items below this are taken
  if (eq_quota < static_cast<int>(eq_all)) {
    eq_end = 0u;                   // the smallest item number with eq_quota ties below it, bit by bit
    if (eq_quota > 0) {
      uint32_t least = 0;          // fewer than eq_quota ties lie below `least`
#pragma unroll 1
      for (int bit = 31 - __clz(max(1, b1 - b0)); bit >= 0; --bit) {
        const uint32_t trial = least | (1u << bit);
        uint32_t c = 0, all;
        for (uint32_t e = tid; e < got; e += kSelThreads) c += ck[e] == T && ci[e] < trial;
        (void)block_exclusive_sum(c, sc.warp_sum, &all);
        if (all < static_cast<uint32_t>(eq_quota)) least = trial;
      }
      eq_end = least + 1u;
    }
  }
  for (uint32_t e = tid; e < got; e += kSelThreads)
    if (ck[e] > T || (ck[e] == T && (take_from || ci[e] < eq_end))) atomicOr(&bits[ci[e] >> 5], 1u << (ci[e] & 31));
  __syncthreads();

  // ---- the selection in order
  const int per = (n_words + kSelThreads - 1) / kSelThreads;
  const int w0 = min(n_words, tid * per), w1 = min(n_words, w0 + per);
  uint32_t mine = 0, here;
  for (int w = w0; w < w1; ++w) mine += __popc(bits[w]);
  int r = static_cast<int>(block_exclusive_sum(mine, sc.warp_sum, &here));
  if constexpr (CLUSTER) {   // after the items of the blocks before
    if (tid == 0) cs::store_remote(remote(&sc.sel[me]), here);
    cs::sync();
    for (uint32_t b = 0; b < me; ++b) r += static_cast<int>(cs::load_remote(remote(&sc.sel[b])));
  }
  for (int w = w0; w < w1; ++w) {
    uint32_t x = bits[w];
    while (x) {
      const int b = __ffs(x) - 1;
      x &= x - 1;
      emit(r++, b0 + 32 * w + b);
    }
  }
  const int written = min(k, static_cast<int>(total));
  if (me == 0)
    for (int i = written + tid; i < k; i += kSelThreads) absent(i);
  if constexpr (CLUSTER) cs::sync();   // nobody leaves while its shared memory may still be addressed
  return written;
}

}  // namespace lsa
