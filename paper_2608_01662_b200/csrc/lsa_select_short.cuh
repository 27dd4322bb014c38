// Exact top-k of at most 4096 keys in shared memory by 256 threads: the same selection as block_select_topk (lsa_select.cuh:
// largest keys first, ties by index, key 0 absent), with the keys in registers.
//
// Latency bounds it: one block works on one row, and each of its steps waits for the last.  A histogram pass over 8 bits costs
// three block barriers, a scan and shared-memory atomics that mostly hit a few bins (the top bits of scores hardly differ);
// four of them and the two passes of the compaction took 15 to 18 thousand cycles for 4096 keys, k = 2048.  Here a thread
// holds 16 keys, and one histogram over 1024 equal parts of the row's range of *values* leaves a handful of candidates for the
// k-th largest, which every warp ranks for itself (rows with outliers take further passes over the part that matters; rows
// whose range is no finite number go bit by bit).  The compaction writes from the registers.
// 4096 keys, k = 2048: 5.0 thousand cycles, the radix select 10.0 (both alone on an SM, instructions cached); 312 keys, k = 64:
// 4.8 and 4.9.  Every step over the 16 registers is free of branches: as `if`s they were 100 cycles per register.
// One copy of the code serves every selection of a kernel (it is not inlined), so that only the first of them pays for the
// fetch of its instructions.
#pragma once

#include "lsa_select.cuh"

namespace lsa {

constexpr int kShortMax = 4096;
constexpr int kShortPer = kShortMax / kSelThreads;   // keys of a thread

__device__ __forceinline__ uint32_t short_lds(uint32_t a) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void short_sts(uint32_t a, uint32_t v) { asm volatile("st.shared.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory"); }
// predicated, so that sixteen in a row are not sixteen branches
__device__ __forceinline__ void sts16_if(bool p, uint32_t a, uint32_t v) {
  asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t@q st.shared.u16 [%0], %1;\n\t}"
               ::"r"(a), "h"(static_cast<uint16_t>(v)), "r"(static_cast<uint32_t>(p)) : "memory");
}
__device__ __forceinline__ void red_if(uint32_t p, uint32_t a) {
  asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %1, 0;\n\t@q red.shared.add.u32 [%0], 1;\n\t}" ::"r"(a), "r"(p) : "memory");
}
__device__ __forceinline__ float key_value(uint32_t key) {   // the score of a key (see score_key)
  return __uint_as_float((key & 0x80000000u) ? key ^ 0x80000000u : ~key);
}

constexpr int kShortBins = 4 * kSelThreads;
constexpr uint32_t kShortHist = 0, kShortWarp = 4 * kShortBins, kShortFound = kShortWarp + 192, kShortMembers = kShortFound + 32;
constexpr uint32_t kShortScratch = kShortMembers + 128;
static_assert(kShortScratch <= sizeof(SelectScratch), "the scratch of the radix select serves this one too");

// keys: shared address of n <= kShortMax keys, 16-byte aligned, with room for 16 per thread (all of it is read).  list: shared address where the selected indices go, ascending, 16 bits each (it
// may be `keys`: they are in registers by then).  scratch: shared address of kShortScratch bytes, 16-byte aligned.  Every one of
// the 256 threads calls it, converged; the keys must be visible to all of them.  Returns the number selected, min(k, #present),
// with the list visible.  They are threads 0-255 of the block and meet on barrier `bar`; short_select_warm calls it otherwise.
static __device__ __noinline__ int short_select(uint32_t keys, int n, int k, uint32_t list, uint32_t scratch, int bar, int tid, int n_threads) {
  const int lane = tid & 31, warp = tid >> 5;
  auto sync = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(n_threads) : "memory"); };
  if (k <= 0) {   // (no key is the k-th largest: the search below would find nothing and go by what it finds in the scratch)
    sync();
    return 0;
  }
  constexpr uint32_t kAll = 0xffffffffu;
  const int base = tid * kShortPer;   // the thread holds items base .. base + 15
  const uint32_t of_warp = scratch + kShortWarp + 4u * (lane & 7), my_warp = scratch + kShortWarp + 4u * warp;
  const uint32_t my_bins = scratch + kShortHist + 16u * tid, found = scratch + kShortFound;
  auto clear_bins = [&]() { asm volatile("st.shared.v4.u32 [%0], {%1, %1, %1, %1};" ::"r"(my_bins), "r"(0u) : "memory"); };
  uint32_t v[kShortPer];
  uint32_t act = 0;   // bit j: register j may hold the k-th largest key
#pragma unroll
  for (int i = 0; i < 4; ++i) {   // four 16-byte loads, from a quarter that differs between neighbours: no bank conflicts
    const uint32_t a = keys + 64u * tid + 16u * ((i + (lane >> 1)) & 3);
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v[4 * i]), "=r"(v[4 * i + 1]), "=r"(v[4 * i + 2]), "=r"(v[4 * i + 3]) : "r"(a) : "memory");
  }
#pragma unroll
  for (int s = 1; s <= 2; s <<= 1) {   // quarters into their order: turned by (lane / 2) % 4
    uint32_t w[kShortPer];
#pragma unroll
    for (int j = 0; j < kShortPer; ++j) w[j] = (lane >> 1) & s ? v[(j - 4 * s) & (kShortPer - 1)] : v[j];
#pragma unroll
    for (int j = 0; j < kShortPer; ++j) v[j] = w[j];
  }
#pragma unroll
  for (int j = 0; j < kShortPer; ++j) {
    v[j] = base + j < n ? v[j] : 0u;
    act |= v[j] != 0u ? 1u << j : 0u;
  }
  clear_bins();
  if (tid == 0) short_sts(found + 12u, 0u);   // members collected

  int n_valid = 0, rem = k;   // keys present; the k-th largest key is the rem-th largest of the active ones
  uint32_t above = 0;         // keys > above are taken ...
  uint32_t tie = 0;           // ... and, with ties, the first k - (how many those are) keys == tie
  bool ties = false, by_bits = false;
#pragma unroll 1
  for (int pass = 0;; ++pass) {
    // the active keys' extremes
    uint32_t mx = 0, mn = kAll;
#pragma unroll
    for (int j = 0; j < kShortPer; ++j) {
      const bool a = (act >> j) & 1u;
      mx = max(mx, a ? v[j] : 0u);
      mn = min(mn, a ? v[j] : kAll);
    }
    mx = __reduce_max_sync(kAll, mx);
    mn = __reduce_min_sync(kAll, mn);
    const uint32_t cnt = __reduce_add_sync(kAll, static_cast<uint32_t>(__popc(act)));
    if (lane == 0) {
      short_sts(my_warp, mx);
      short_sts(my_warp + 32u, mn);
      short_sts(my_warp + 64u, cnt);
    }
    sync();   // (every key has been read: `list` may be written from the next barrier on)
    mx = __reduce_max_sync(kAll, short_lds(of_warp));
    mn = __reduce_min_sync(kAll, short_lds(of_warp + 32u));
    if (pass == 0) {
      n_valid = static_cast<int>(__reduce_add_sync(kAll, lane < 8 ? short_lds(of_warp + 64u) : 0u));
      if (n_valid <= k) break;   // everything is taken
    }
    if (mx == mn) {
      above = tie = mx;
      ties = true;
      break;
    }
    // 1024 equal parts of [smallest, largest]; the map is monotone, so the parts are intervals of keys
    const float lo = key_value(mn), scale = __fdividef(511.75f, 0.5f * key_value(mx) - 0.5f * lo);
    if (!(scale > 0.f && scale < INFINITY) || pass == 8) {
      by_bits = true;
      break;
    }
    const uint32_t bin0 = scratch + kShortHist + 4u * (kShortBins - 1) + 4u * 0x4b000000u;   // 2^23 is 0x4b000000
    uint32_t part[kShortPer];   // address of the key's bin, largest values first (of inactive keys: anything)
#pragma unroll
    for (int j = 0; j < kShortPer; ++j)
      part[j] = bin0 - 4u * __float_as_uint(fminf((key_value(v[j]) - lo) * scale, kShortBins - 1.f) + 8388608.f);   // (rounded to a whole number)
#pragma unroll
    for (int j = 0; j < kShortPer; ++j) red_if((act >> j) & 1u, part[j]);
    sync();
    uint32_t h[4];
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(h[0]), "=r"(h[1]), "=r"(h[2]), "=r"(h[3]) : "r"(my_bins) : "memory");
    clear_bins();
    const uint32_t sum = h[0] + h[1] + h[2] + h[3];
    uint32_t incl = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t x = __shfl_up_sync(kAll, incl, d);
      if (lane >= d) incl += x;
    }
    if (lane == 31) short_sts(my_warp + 96u, incl);
    sync();
    incl += __reduce_add_sync(kAll, lane < warp ? short_lds(of_warp + 96u) : 0u);
    uint32_t before = incl - sum;
    if (before < static_cast<uint32_t>(rem) && static_cast<uint32_t>(rem) <= incl) {   // exactly one thread
      int b = 0;
#pragma unroll
      for (int u = 0; u < 3; ++u)
        if (b == u && before + h[u] < static_cast<uint32_t>(rem)) {
          before += h[u];
          b = u + 1;
        }
      short_sts(found, 4u * tid + b);
      short_sts(found + 4u, before);
      short_sts(found + 8u, b == 0 ? h[0] : b == 1 ? h[1] : b == 2 ? h[2] : h[3]);
    }
    sync();
    const uint32_t bin = scratch + kShortHist + 4u * short_lds(found);
    rem -= static_cast<int>(short_lds(found + 4u));
    const int members = static_cast<int>(short_lds(found + 8u));
#pragma unroll
    for (int j = 0; j < kShortPer; ++j) act &= part[j] == bin ? kAll : ~(1u << j);
    if (members > 32) continue;
    // few enough for one lane each: every warp ranks them
    while (act != 0u) {
      const uint32_t key = short_lds(keys + 4u * static_cast<uint32_t>(base + __ffs(act) - 1));
      uint32_t at;
      asm volatile("atom.shared.add.u32 %0, [%1], 1;" : "=r"(at) : "r"(found + 12u) : "memory");
      short_sts(scratch + kShortMembers + 4u * at, key);
      act &= act - 1u;
    }
    sync();
    const uint32_t m = lane < members ? short_lds(scratch + kShortMembers + 4u * lane) : 0u;
    int larger = 0, same = 0;
#pragma unroll 1
    for (int i0 = 0; i0 < members; i0 += 8) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const uint32_t x = __shfl_sync(kAll, m, i0 + i);
        larger += x > m;
        same += x == m;
      }
    }
    const bool mine = lane < members && larger < rem && rem <= larger + same;   // the lanes that hold the k-th largest key
    const int at = __ffs(__ballot_sync(kAll, mine)) - 1;
    tie = __shfl_sync(kAll, m, at);
    ties = __shfl_sync(kAll, larger + same, at) != rem;   // (else all that equal it are taken)
    above = ties ? tie : tie - 1u;
    break;
  }
  if (by_bits) {   // bit by bit: the keys at or above a candidate are counted, until exactly k are
    uint32_t T = 0;
    ties = true;
#pragma unroll 1
    for (int b = 31; b >= 0; --b) {
      const uint32_t cand = T | (1u << b);
      uint32_t c = 0;
#pragma unroll
      for (int j = 0; j < kShortPer; ++j) c += v[j] >= cand;
      c = __reduce_add_sync(kAll, c);
      if (lane == 0) short_sts(my_warp + 96u + 32u * (b & 1), c);
      sync();
      c = __reduce_add_sync(kAll, lane < 8 ? short_lds(of_warp + 96u + 32u * (b & 1)) : 0u);
      if (static_cast<int>(c) >= k) {
        T = cand;
        if (static_cast<int>(c) == k) {
          ties = false;
          break;
        }
      }
    }
    tie = T;
    above = ties ? T : T - 1u;
  }

  // ---- ordered compaction
  uint32_t mine = 0;   // taken outright | ties << 16
#pragma unroll
  for (int j = 0; j < kShortPer; ++j) mine += (v[j] > above ? 1u : 0u) + (ties && v[j] == tie ? 0x10000u : 0u);
  uint32_t upto = mine;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t x = __shfl_up_sync(kAll, upto, d);
    if (lane >= d) upto += x;
  }
  if (lane == 31) short_sts(my_warp + 160u, upto);
  sync();
  const uint32_t one = lane < 8 ? short_lds(of_warp + 160u) : 0u;
  const uint32_t all = __reduce_add_sync(kAll, one);
  upto += __reduce_add_sync(kAll, lane < warp ? one : 0u) - mine;   // what lies before this thread
  const int need = ties ? k - static_cast<int>(all & 0xffffu) : 0;   // ties that are taken
  int left = need - static_cast<int>(upto >> 16);                    // ... from here on
  uint32_t out = list + 2u * ((upto & 0xffffu) + static_cast<uint32_t>(min(static_cast<int>(upto >> 16), need)));
#pragma unroll
  for (int j = 0; j < kShortPer; ++j) {
    const bool is_tie = ties && v[j] == tie;
    const bool take = v[j] > above || (is_tie && left > 0);
    left -= is_tie;
    sts16_if(take, out, static_cast<uint32_t>(base + j));
    out += take ? 2u : 0u;
  }
  sync();
  return min(k, n_valid);
}
template <int BAR>
__device__ __forceinline__ int short_select(uint32_t keys, int n, int k, uint32_t list, uint32_t scratch) {
  return short_select(keys, n, k, list, scratch, BAR, static_cast<int>(threadIdx.x), kSelThreads);
}
// A selection of 64 made-up keys by one otherwise idle warp, on barrier BAR and in shared memory that nobody uses
// (kShortWarm bytes, 16-byte aligned): its instructions are then at hand when the block needs them.  The first selection of a
// decode kernel spent 6 to 8 of its 11 to 13 thousand cycles on their fetch.
constexpr uint32_t kShortWarm = 2048 + ((kShortScratch + 15u) & ~15u);
template <int BAR>
__device__ __forceinline__ void short_select_warm(uint32_t area) {
  const int lane = threadIdx.x & 31;
  const uint32_t scratch = area + 2048u;
  for (uint32_t a = 4u * lane; a < 2048u; a += 128u) short_sts(area + a, score_key(1.f + static_cast<float>(a)));
  for (uint32_t a = 4u * lane; a < kShortScratch; a += 128u) short_sts(scratch + a, 0u);
  __syncwarp();
  if (lane < 8) short_sts(scratch + kShortWarp + 32u + 4u * lane, 0xffffffffu);   // seven warps without keys
  __syncwarp();
  (void)short_select(area, 64, 8, area, scratch, BAR, lane, 32);
}
// r-th item of the list
__device__ __forceinline__ int short_item(uint32_t list, int r) {
  uint16_t v;
  asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(list + 2u * static_cast<uint32_t>(r)) : "memory");
  return v;
}

}  // namespace lsa
