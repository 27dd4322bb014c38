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
// What bounds it: the one read of the row.  1000 rows of 65536 scores, k = 2048: @LONGROWS@; 16 rows of 16K to 128K on
// clusters: @LONGCLUSTER@.
#pragma once

#include "lsa_select_cluster.cuh"

namespace lsa {

constexpr int kLongBins = 8192;              // sample histogram: the top 13 bits of a key
constexpr int kLongMinRow = 16384;           // rows below this are left to the radix select

// Room for collected items: what k items need with the sample's margin (six standard deviations and a bin's width).
__host__ __device__ constexpr int long_cap(int k) { return k <= 3072 ? 6144 : 2 * k; }

struct alignas(16) LongScratch {
  uint32_t hist[4][256];      // digit counts of this block, one histogram per pass
  uint32_t all[4][256];       // CLUSTER, first block: of the whole row
  uint32_t sel[kClusterSel], eq[kClusterSel];   // CLUSTER, first block: selected items / ties per block
  uint32_t cnt, total, overflow;                // collected here; CLUSTER, first block: in all, somebody ran out of room
  uint32_t bound, prefix, remaining, whole;
  uint32_t warp_sum[kSelWarps];
};

static_assert(sizeof(LongScratch) % 16 == 0, "what follows it is read 16 bytes at a time");
// Dynamic shared memory of a block: the scratch, the collected keys and items (the sample's histogram lies there before),
// and a bit per item of the block's piece.
__host__ __device__ constexpr size_t long_smem_bytes(int cap, int64_t piece) {
  return sizeof(LongScratch) + static_cast<size_t>(cap) * 8 + static_cast<size_t>((piece + 31) / 32) * 4;
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

// KeyF: uint32_t operator()(int i) (0 = absent; called for i of [0, n)); void quad(int i, uint32_t (&k)[4]): the keys of i .. i + 3,
// i a multiple of four, all of them in [0, n).  EmitF: void operator()(int r, int i): item i is
// the r-th of the selection.  AbsentF: void operator()(int r): there is no r-th item.  Every thread of the block (CLUSTER: of
// every block of the cluster, kClusterSel along x) calls this with the same arguments.  Returns how many items were
// selected, or -1: nothing has been written, take the radix select (the same answer in every block).
template <bool CLUSTER, class KeyF, class EmitF, class AbsentF>
__device__ int long_select(KeyF key, EmitF emit, AbsentF absent, int n, int k, int cap, uint8_t* smem) {
  namespace cs = cluster_sel;
  LongScratch& sc = *reinterpret_cast<LongScratch*>(smem);
  uint32_t* ck = reinterpret_cast<uint32_t*>(smem + sizeof(LongScratch));
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
    (&sc.all[0][0])[i] = 0;
  }
  for (int i = tid; i < n_words; i += kSelThreads) bits[i] = 0;
  if (tid == 0) {
    sc.cnt = sc.total = sc.overflow = 0;
    sc.bound = 1u;
  }
  if (piece > cap) {   // (else everything has room; the same in every block)
    uint32_t* bins = ck;
    for (int i = tid; i < kLongBins; i += kSelThreads) bins[i] = 0;
    __syncthreads();
    const int m_shift = n > 131072 ? 14 : 12, m = 1 << m_shift;   // evenly spaced items
    for (int j0 = tid; j0 < m; j0 += 8 * kSelThreads) {
      uint32_t kk[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) kk[u] = key(static_cast<int>(static_cast<int64_t>(j0 + u * kSelThreads) * n >> m_shift));
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (kk[u] != 0u) atomicAdd(&bins[kk[u] >> 19], 1u);
    }
    __syncthreads();
    const float expect = static_cast<float>(k) * static_cast<float>(m) / static_cast<float>(n);
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
        if (run < want && want <= run + c[i]) sc.bound = max(1u, static_cast<uint32_t>(kLongBins - kPer * (tid + 1) + i) << 19);
        run += c[i];
      }
    }
  }
  __syncthreads();
  const uint32_t bound = sc.bound;

  // ---- collect: a warp takes 512 items at a time, 16 per lane, the next ones on their way (4 KB a warp: with single words
  // in flight the read of 1000 rows of 65536 ran at 1.3 TB/s)
  constexpr int kStep = 512;
  const int full = (b1 - b0) / kStep;   // whole steps
  {
    auto load = [&](int step, uint32_t (&kk)[4][4]) {
#pragma unroll
      for (int u = 0; u < 4; ++u) key.quad(b0 + step * kStep + 128 * u + 4 * lane, kk[u]);
    };
    uint32_t kk[4][4], nx[4][4];
    int step = warp;
    if (step < full) load(step, kk);
    for (; step < full; step += kSelWarps) {
      if (step + kSelWarps < full) load(step + kSelWarps, nx);
      uint32_t hit = 0;
#pragma unroll
      for (int u = 0; u < 16; ++u) hit |= (kk[u >> 2][u & 3] >= bound ? 1u : 0u) << u;
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
        for (int u = 0; u < 16; ++u)
          if (hit >> u & 1u) {
            ck[at] = kk[u >> 2][u & 3];
            ci[at++] = static_cast<uint32_t>(step * kStep + 128 * (u >> 2) + 4 * lane + (u & 3));
          }
      }
#pragma unroll
      for (int u = 0; u < 16; ++u) kk[u >> 2][u & 3] = nx[u >> 2][u & 3];
    }
    for (int i = b0 + full * kStep + tid; i < b1; i += kSelThreads) {
      const uint32_t x = key(i);
      if (x >= bound) {
        const uint32_t at = atomicAdd(&sc.cnt, 1u);
        if (at < static_cast<uint32_t>(cap)) {
          ck[at] = x;
          ci[at] = static_cast<uint32_t>(i - b0);
        }
      }
    }
  }
  __syncthreads();
  const uint32_t got = sc.cnt;
  uint32_t total = got;
  bool failed = got > static_cast<uint32_t>(cap);
  uint32_t scratch0 = 0;   // the first block's scratch
  auto remote = [&](const void* p) -> uint32_t { return scratch0 + (smem_u32(p) - smem_u32(&sc)); };
  if constexpr (CLUSTER) {
    scratch0 = cs::at_rank0(&sc);
    cs::sync();   // every block's scratch is set up
    if (tid == 0) {
      cs::add_remote(remote(&sc.total), got);
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

  // ---- the k-th largest of the collected keys: take keys > T and the first need_eq keys == T
  uint32_t T = 0;
  int need_eq = 0;
  if (total > static_cast<uint32_t>(k)) {
    uint32_t prefix = 0, mask = 0, remaining = static_cast<uint32_t>(k);
#pragma unroll 1
    for (int pass = 0; pass < 4; ++pass) {
      const int shift = 24 - 8 * pass;
      for (uint32_t e = tid; e < got; e += kSelThreads) {
        const uint32_t x = ck[e];
        if ((x & mask) == prefix) atomicAdd(&sc.hist[pass][(x >> shift) & 255u], 1u);
      }
      __syncthreads();
      if constexpr (CLUSTER) {
        const uint32_t v = sc.hist[pass][tid];
        if (v) cs::add_remote(remote(&sc.all[pass][tid]), v);
        cs::sync();
      }
      if (warp == 0) {   // lane l takes bins 255 - 8 l .. 248 - 8 l
        uint32_t c[8], sum = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int bin = 255 - 8 * lane - i;
          c[i] = CLUSTER ? cs::load_remote(remote(&sc.all[pass][bin])) : sc.hist[pass][bin];
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
      mask |= 255u << shift;
      if (sc.whole) break;   // the whole bin is taken
    }
    if (sc.whole) {
      T = prefix - 1u;       // (a bin with keys in it has a prefix of at least 1, or holds keys of 1 and more)
      if (prefix == 0u) T = 0u;
    } else {
      T = prefix;
      need_eq = static_cast<int>(remaining);
    }
  }

  // ---- how many are selected here, and which of the ties
  int gt = 0, eq = 0;
  for (uint32_t e = tid; e < got; e += kSelThreads) {
    gt += ck[e] > T;
    eq += ck[e] == T;
  }
  uint32_t gt_all, eq_all;
  (void)block_exclusive_sum(static_cast<uint32_t>(gt), sc.warp_sum, &gt_all);
  (void)block_exclusive_sum(static_cast<uint32_t>(eq), sc.warp_sum, &eq_all);
  int eq_quota = min(static_cast<int>(eq_all), need_eq);   // of this block's ties
  int base = 0;                                            // selected items of the blocks before
  if constexpr (CLUSTER) {
    if (tid == 0) {
      cs::store_remote(remote(&sc.sel[me]), gt_all);
      cs::store_remote(remote(&sc.eq[me]), eq_all);
    }
    cs::sync();
    int eq_before = 0;
    for (uint32_t r = 0; r < me; ++r) {
      base += static_cast<int>(cs::load_remote(remote(&sc.sel[r])));
      eq_before += static_cast<int>(cs::load_remote(remote(&sc.eq[r])));
    }
    base += min(eq_before, need_eq);
    eq_quota = min(static_cast<int>(eq_all), max(0, need_eq - eq_before));
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
    if (ck[e] > T || (need_eq > 0 && ck[e] == T && ci[e] < eq_end)) atomicOr(&bits[ci[e] >> 5], 1u << (ci[e] & 31));
  __syncthreads();

  // ---- the selection in order
  const int per = (n_words + kSelThreads - 1) / kSelThreads;
  const int w0 = min(n_words, tid * per), w1 = min(n_words, w0 + per);
  uint32_t mine = 0, here;
  for (int w = w0; w < w1; ++w) mine += __popc(bits[w]);
  int r = base + static_cast<int>(block_exclusive_sum(mine, sc.warp_sum, &here));
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
