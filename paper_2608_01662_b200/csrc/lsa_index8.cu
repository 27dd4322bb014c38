// a1-a4 for the 8-head, 64-dim indexer on contiguous bf16 caches with a recall budget of at most 1024 tokens: coarse page
// scores (Eq. 9), top-M pages (Eq. 10), token scores on them (Eq. 11) and the top-K_sparse outside sink and window
// (Eq. 12), one warp per query (4 or 16 where there are few), in one launch.
//
// Nothing is shared between the warps of different queries: key rows go from global memory (L1 or L2: the caches of this shape
// are small, and the warps of a block hold neighbouring queries) straight to the A operands of m16n8k16 MMAs, whose eight
// columns are the eight heads.  The sum over dims may run in any order, so a thread takes the 16-byte chunks t and 4 + t (t = lane % 4) of
// a row, and the query heads are fetched in the same order.  A group of 32 rows ends as one score per lane, and the keys of
// all candidates stay in registers (32 per lane at most), where the K-th largest is found bit by bit: a count of the keys
// above a trial value is one compare per register and one warp-wide add.
//
// What bounds it: the latency of a warp's own chain (32 bits x a warp-wide add, twice, and 8 to 24 groups of loads).  The
// block-wide forms (one block per query, barriers between the steps; the page scores by a kernel of their own) took 21 + 70
// us (84 us back to back) for 2048 queries of a 2048-token prompt, this one 26 us; 749 and 292 us for 16384 queries.
#include "lsa_internal.h"
#include "lsa_select.cuh"

namespace lsa {

namespace {

constexpr int kHI8 = 8, kDI8 = 64, kRow8 = kDI8 * 2;
constexpr int kWarps8 = 4;
constexpr int kMaxSlots8 = 1024;             // candidate tokens of a query
constexpr int kMaxPages8 = 1024;             // eligible pages of a query
constexpr int kMaxMeans8 = 8192;             // mean keys of the cache
constexpr int kMaxKept8 = kMaxSlots8 / 64;
static_assert(kMaxPages8 <= kMaxSlots8, "page keys and candidate keys share their place");

struct Heads8 {
  uint4 q[2];          // B operands of the four k-steps
  float w0, w1;        // weights of heads 2t and 2t + 1
};

// 32 consecutive rows at `rows` as MMA operands (row numbers are clamped to `last`, callers drop what is past it).
__device__ __forceinline__ void load_32rows(uint4 (&a)[4][2], const uint8_t* rows, int last) {
  const int g = (threadIdx.x & 31) >> 2, t = threadIdx.x & 3;
#pragma unroll
  for (int i = 0; i < 4; ++i) {   // rows 8 i + g
    const uint8_t* src = rows + static_cast<int64_t>(min(8 * i + g, last)) * kRow8 + t * 16;
    a[i][0] = *reinterpret_cast<const uint4*>(src);
    a[i][1] = *reinterpret_cast<const uint4*>(src + 64);
  }
}
// The score of row `lane` of them.
__device__ __forceinline__ float score_32rows(const Heads8& h, const uint4 (&a)[4][2]) {
  const int lane = threadIdx.x & 31, t = lane & 3;
  float v[4];
#pragma unroll
  for (int mt = 0; mt < 2; ++mt) {
    float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const uint4 lo = a[2 * mt][j], hi = a[2 * mt + 1][j];
      const uint32_t a0[4] = {lo.x, hi.x, lo.y, hi.y}, a1[4] = {lo.z, hi.z, lo.w, hi.w};
      mma_bf16(c, a0, h.q[j].x, h.q[j].y);
      mma_bf16(c, a1, h.q[j].z, h.q[j].w);
    }
    v[2 * mt] = fmaf(h.w1, fmaxf(c[1], 0.f), h.w0 * fmaxf(c[0], 0.f));
    v[2 * mt + 1] = fmaf(h.w1, fmaxf(c[3], 0.f), h.w0 * fmaxf(c[2], 0.f));
  }
  // sum over the four lanes of a row, lane t keeping row 8 t + g; then every lane fetches its own row's
  const bool t2 = t & 2, t1 = t & 1;
  const float x = (t2 ? v[2] : v[0]) + __shfl_xor_sync(0xffffffffu, t2 ? v[0] : v[2], 2);
  const float y = (t2 ? v[3] : v[1]) + __shfl_xor_sync(0xffffffffu, t2 ? v[1] : v[3], 2);
  const float z = (t1 ? y : x) + __shfl_xor_sync(0xffffffffu, t1 ? x : y, 1);
  return __shfl_sync(0xffffffffu, z, 4 * (lane & 7) + (lane >> 3));
}

// The k largest of the keys key[r] (item 32 r + lane; 0 = absent), ties to the smaller item; emit(rank, item, r) in
// ascending order of the items.  Returns how many there are (fewer than k: all of them).
template <int R, class Emit>
__device__ __forceinline__ int warp_topk(const uint32_t (&key)[R], int k, Emit emit) {
  const int lane = threadIdx.x & 31;
  auto count = [&](uint32_t least) -> int {   // keys >= least
    int n = 0;
#pragma unroll
    for (int r = 0; r < R; ++r) n += key[r] >= least ? 1 : 0;
    return __reduce_add_sync(0xffffffffu, n);
  };
  const int n_valid = count(1u);
  uint32_t thr = 1u;
  int n_ge = n_valid;
  if (n_valid > k) {
    thr = 0u;
    for (int bit = 31; bit >= 0; --bit) {
      const uint32_t trial = thr | (1u << bit);
      const int n = count(trial);
      if (n >= k) {
        thr = trial;
        n_ge = n;
        if (n == k) break;
      }
    }
  }
  // more keys at the threshold than places: the first `ties` of them in item order
  int ties = n_ge > k ? k - (thr == 0xffffffffu ? 0 : count(thr + 1u)) : 0x7fffffff;
  int base = 0;
  const unsigned below = (1u << lane) - 1u;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const unsigned eq = __ballot_sync(0xffffffffu, key[r] == thr);
    const bool take = key[r] > thr || (key[r] == thr && __popc(eq & below) < ties);
    ties -= __popc(eq);   // (unlimited: stays far above zero)
    const unsigned got = __ballot_sync(0xffffffffu, take);
    if (take) emit(base + __popc(got & below), 32 * r + lane, r);
    base += __popc(got);
  }
  return base;
}

// kWpq warps share a query (1: four queries per block).  They deal the groups of 32 mean keys and of 64 tokens among them and
// meet before each selection, which is the first one's; a row's score does not depend on the warp that takes it, so every
// kWpq gives the same lists.
template <int R, int kWpq>
__global__ void __launch_bounds__(32 * (kWpq > kWarps8 ? kWpq : kWarps8)) index8_kernel(IndexArgs p) {
  constexpr int kQueries = kWpq > 1 ? 1 : kWarps8;
  __shared__ uint32_t keys[kQueries][kMaxSlots8];   // of the pages, then of the candidates
  __shared__ int32_t kept[kQueries][kMaxKept8];
  __shared__ int n_kept;
  const int lane = threadIdx.x & 31, t = lane & 3;
  const int part = kWpq > 1 ? threadIdx.x >> 5 : 0, own = kWpq > 1 ? 0 : threadIdx.x >> 5;   // the warp's part of the query, its query
  auto meet = [&]() {
    if constexpr (kWpq > 1) __syncthreads();
    else __syncwarp();
  };
  const int slot = static_cast<int>(blockIdx.x) * kQueries + own;
  const int qi = p.n_query - 1 - slot;   // late queries have the most pages: they go first
  if (qi < 0) return;
  pdl_wait();                 // the mean keys may come from the previous kernel of the stream
  pdl_launch_dependents();
  int32_t* out_idx = p.sparse_idx + static_cast<int64_t>(qi) * p.Ksp;
  int32_t* out_pages = p.pages_out ? p.pages_out + static_cast<int64_t>(qi) * p.M : nullptr;
  const int64_t lo = p.S, hi = p.q_pos0 + qi - p.W;
  int n_sel = 0, n_pages = 0;
  if (hi >= lo) {
    Heads8 h;
    const uint8_t* qg = reinterpret_cast<const uint8_t*>(p.q_idx) + (static_cast<int64_t>(qi) * kHI8 + (lane >> 2)) * kRow8 + t * 16;
    h.q[0] = *reinterpret_cast<const uint4*>(qg);
    h.q[1] = *reinterpret_cast<const uint4*>(qg + 64);
    const float2 ww = *reinterpret_cast<const float2*>(p.w + static_cast<int64_t>(qi) * kHI8 + 2 * t);
    h.w0 = ww.x;
    h.w1 = ww.y;

    // ---- a1, a2: pages
    const int p_shift = 31 - __clz(p.P);
    const int p0 = static_cast<int>(lo >> p_shift), p1 = static_cast<int>(hi >> p_shift);
    const int n_elig = p1 - p0 + 1;
    int32_t* pages = kept[own];
    if (p.hi_enable && n_elig > p.M) {
      const int spp = p.P / p.B, spp_shift = 31 - __clz(spp);   // sub-blocks per page: 8, 16 or 32
      const int n_sub = static_cast<int>((p.n_key + p.B - 1) / p.B);
      const int sub0 = p0 << spp_shift, sub1 = min(n_sub, (p1 + 1) << spp_shift);
      const uint8_t* km = reinterpret_cast<const uint8_t*>(p.kmean);
      uint32_t* pk = keys[own];
      constexpr int kStep = 32 * kWpq;
      uint4 a[2][4][2];   // the next group is on its way while one is scored
      auto load_means = [&](uint4 (&to)[4][2], int s) {
        if (s < sub1) load_32rows(to, km + static_cast<int64_t>(s) * kRow8, sub1 - 1 - s);
      };
      load_means(a[0], sub0 + 32 * part);
      auto score_group = [&](int s, const uint4 (&now)[4][2], uint4 (&next)[4][2]) {
        load_means(next, s + kStep);
        float v = score_32rows(h, now);
        if (s + lane >= sub1) v = 0.f;
        for (int d = 1; d < spp; d <<= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
        if ((lane & (spp - 1)) == 0 && s + lane < sub1) pk[(s + lane - sub0) >> spp_shift] = score_key(v);
      };
      for (int s = sub0 + 32 * part; s < sub1; s += 2 * kStep) {
        score_group(s, a[0], a[1]);
        if (s + kStep < sub1) score_group(s + kStep, a[1], a[0]);
      }
      meet();
      auto keep = [&](int rank, int item, int) { pages[rank] = p0 + item; };
      auto page_key = [&](int i) -> uint32_t { return i < n_elig ? pk[i] : 0u; };
      if (part == 0) {
        if (n_elig <= 256) {
          uint32_t key[8];
#pragma unroll
          for (int r = 0; r < 8; ++r) key[r] = page_key(32 * r + lane);
          n_pages = warp_topk<8>(key, p.M, keep);
        } else {
          uint32_t key[kMaxPages8 / 32];
#pragma unroll
          for (int r = 0; r < kMaxPages8 / 32; ++r) key[r] = page_key(32 * r + lane);
          n_pages = warp_topk<kMaxPages8 / 32>(key, p.M, keep);
        }
      }
    } else {
      n_pages = n_elig;   // the host guarantees that they fit
      if (part == 0 && lane < n_pages) pages[lane] = p0 + lane;
    }
    if (kWpq > 1 && threadIdx.x == 0) n_kept = n_pages;
    meet();
    if constexpr (kWpq > 1) n_pages = n_kept;

    // ---- a3: tokens of the kept pages; a group of 32 slots lies in one page
    const int n_slots = n_pages << p_shift;
    const uint8_t* kg = reinterpret_cast<const uint8_t*>(p.k_idx);
    auto group_pos = [&](int c) -> int64_t { return (static_cast<int64_t>(pages[c >> p_shift]) << p_shift) + (c & (p.P - 1)); };
    uint32_t* sk = keys[own];   // (a rolled loop cannot index registers: the keys pass through shared memory)
    uint4 a[2][4][2];
    auto load_group = [&](uint4 (&to)[4][2], int64_t pos) { load_32rows(to, kg + pos * kRow8, static_cast<int>(min64(31, p.n_key - 1 - pos))); };
    if (64 * part < n_slots) load_group(a[0], group_pos(64 * part));
    for (int c = 64 * part; c < n_slots; c += 64 * kWpq) {   // (a page has 64 tokens at least)
      const int64_t pos = group_pos(c);
      load_group(a[1], pos + 32);
      float v = score_32rows(h, a[0]);
      sk[c + lane] = pos + lane >= lo && pos + lane <= hi ? score_key(v) : 0u;
      if (c + 64 * kWpq < n_slots) load_group(a[0], group_pos(c + 64 * kWpq));
      v = score_32rows(h, a[1]);
      sk[c + 32 + lane] = pos + 32 + lane >= lo && pos + 32 + lane <= hi ? score_key(v) : 0u;
    }
    meet();
    if (part != 0) return;   // (nothing below waits for other warps)
    uint32_t key[R];
#pragma unroll
    for (int r = 0; r < R; ++r) key[r] = 32 * r < n_slots ? sk[32 * r + lane] : 0u;
    // ---- a4
    n_sel = warp_topk<R>(key, p.Ksp, [&](int rank, int, int r) { out_idx[rank] = static_cast<int32_t>(group_pos(32 * r)) + lane; });
    if (out_pages)   // (without the hierarchy a query has every eligible page, which may be more than the list holds)
      for (int i = lane; i < min(n_pages, p.M); i += 32) out_pages[i] = pages[i];
  }
  if (part != 0) return;
  for (int i = n_sel + lane; i < p.Ksp; i += 32) out_idx[i] = -1;
  if (out_pages)
    for (int i = n_pages + lane; i < p.M; i += 32) out_pages[i] = -1;
  if (lane == 0) p.n_sparse[qi] = n_sel;
}

}  // namespace

// Contiguous bf16 caches, mean pooling, at most 1024 candidates, 1024 pages and 8192 mean keys a query.  Longer caches: the
// coarse stage as a kernel of its own, whose blocks score a tile of mean keys against 32 queries (4096 queries, 16384 mean
// keys: 812 us so, 850 here; 8192: 486 and 431).  Not a matter of the number of queries: a chunk gives the rows of the whole run.
bool index8_supported(const IndexArgs& a) {
  if (a.HI != kHI8 || a.DI != kDI8 || a.paged || a.key_e4m3) return false;
  const int64_t pages = (a.n_key + a.P - 1) / a.P, slots = a.hi_enable ? static_cast<int64_t>(a.M) * a.P : pages * a.P;
  return slots <= kMaxSlots8 && pages <= kMaxPages8 && (!a.hi_enable || a.n_key <= static_cast<int64_t>(kMaxMeans8) * a.B);
}

namespace {

// Warps per query: the count with the smallest estimate, in hundredths of a microsecond: a selection's 9 us and 0.019 us per
// mean key and token of a warp's share, in waves of 16 warps per SM.
int warps_per_query(const IndexArgs& a) {
  const int64_t pages = (a.n_key + a.P - 1) / a.P, slots = a.hi_enable ? static_cast<int64_t>(a.M) * a.P : pages * a.P;
  const int64_t rows = slots + (a.hi_enable && pages > a.M ? min64(a.n_key, a.q_pos0 + a.n_query) / a.B : 0);
  const int64_t at_once = 16 * static_cast<int64_t>(a.sm_count > 0 ? a.sm_count : 148);
  int best = 1;
  int64_t best_cost = 0;
  for (int w : {1, 4, 16}) {
    const int64_t cost = (a.n_query * static_cast<int64_t>(w) + at_once - 1) / at_once * (900 + 2 * rows / w);
    if (w == 1 || cost < best_cost) {
      best = w;
      best_cost = cost;
    }
  }
  return best;
}

template <int kWpq>
cudaError_t launch8(const IndexArgs& a, cudaStream_t st) {
  const int64_t slots = a.hi_enable ? static_cast<int64_t>(a.M) * a.P : (a.n_key + a.P - 1) / a.P * a.P;
  const int queries = kWpq > 1 ? 1 : kWarps8, warps = kWpq > 1 ? kWpq : kWarps8;
  return launch_pdl(slots <= kMaxSlots8 / 2 ? index8_kernel<kMaxSlots8 / 64, kWpq> : index8_kernel<kMaxSlots8 / 32, kWpq>,
                    dim3(static_cast<unsigned>((a.n_query + queries - 1) / queries)), dim3(32 * warps), 0, st, a);
}

}  // namespace

cudaError_t launch_index8(const IndexArgs& a, cudaStream_t st, int64_t* n_launch) {
  if (a.n_query == 0) return cudaSuccess;
  const int w = warps_per_query(a);
  const cudaError_t e = w == 1 ? launch8<1>(a, st) : w == 4 ? launch8<4>(a, st) : launch8<16>(a, st);
  ++*n_launch;
  return e;
}

}  // namespace lsa
