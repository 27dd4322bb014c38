// a6 on the 5th-generation tensor cores: sparse attention (Eq. 3) for the MLA latent shape
// (H = 64 heads, d_qk = 576, d_v = 512, the value is the first 512 dims of the key row).
//
// A block works on one query at a time (or on one row split of one sequence in decode).  Its 64 heads are the M = 64
// rows of every MMA; the attended cache rows stream through a ring of three 64-key shared tiles, into which Q goes
// as an item of its own.  Prefill blocks are persistent: when a query's last copies are out, the next query's Q and
// first tiles follow them into the ring, and warps of their own move that Q and write this O, so that the tensor pipe
// waits between two queries only for O to leave tensor memory.
//
//   (warp numbers of the prefill form; struct Warps)
//   warps 14-22 gather: three warps per ring slot (two where row lists are walked).  They wait for the slot, copy rows [window | sink | sparse] (or those of the
//               caller's row list) into its 128B-swizzled K-major tile with coalesced 16-byte cp.async, a row by one warp
//               (spreading a tile's chunks over the warps was measured 1.3 x slower, a TMA gather of four rows per
//               instruction - AttnArgs::gather4 - as well: the TMA unit takes about 26 cycles for its 512 bytes), and hand
//               it over when it has landed; tiles of 64 consecutive window rows and Q come as one TMA box each.
//   warps 8-11  the ends of a job: they move Q to tensor memory (as soon as the last Q K^T of the job before is complete: the
//               softmax and P V of its last tile run meanwhile) and, once its last P V is, write O / l to global; only the
//               next job's P V waits for them.  With both done by the softmax warps a query cost 7.2 thousand cycles beside
//               its tiles: 1000 queries of up to 1000 rows 625 -> 597 us, a prompt of 32768 30.4 -> 30.0 ms.
//               One thread of warp 8 is the scheduler and publishes the block's jobs (query, row count).  In prefill it takes
//               the block index of a block that has not started yet (cluster launch control), one job ahead of the one being
//               worked on, latest query first: those attend the most rows.
//   warps 12, 13  one thread each issues tcgen05.mma:
//                 S = Q K^T   warp 12, M64 N64 K16, Q in tensor memory (the rope dims in shared memory), as two accumulation
//                             chains: dims 0-255 and rope dims 0-31 in the even half of the lanes, dims 256-511 and rope
//                             dims 32-63 in the odd half (an M = 64 accumulator and its A operand use 16 of the 32 lanes of
//                             each quarter, so both halves of Q share their columns).  36 MMAs at the pipe's 32 cycles.
//                 O += P V    warp 13, tcgen05.mma.ws M64 N256 K16, P in shared memory; V is the key tile read MN-major, so
//                             that a cache row is fetched once.  The .ws form spreads the 64 rows over all 128 lanes (heads
//                             in lanes 0-63 and again in 64-127, each with half of the value dims), which is the full data
//                             path: 81 cycles where the plain M64 N256 form takes 129.
//               Two threads, because one stalls for 300 to 500 cycles after each batch before it gets to the next, and
//               two S buffers, so that Q K^T of the next tile need not wait for the softmax of this one: 2 340 cycles per
//               tile with one of each.
//   warps 0-7   softmax, four warps for each half of a tile's keys (four in all where row lists are walked): per tile add the two partial sums (read as 16-lane
//               fragments, so both land in the same registers), running max with lazy rescaling of O, exp2, fp32 row sums, P as
//               bf16 into the tile's rope block (64 x 64 values; Q K^T was its only reader); a split's partial O to the merge.
//
// What bounds it (prefill): per 64-key tile the tensor pipe needs 36 x 32 + 8 x 81 = 1 800 cycles (2 176 with the plain
// form for P V), and shared memory is read and written for about as long: 576 (Q K^T) + 640 (P V) + 576 (the copies).  A window
// tile takes 2 000.  A gathered one waits for its slot: three slots, each held from Q K^T to the end of P V (4 250 cycles) and
// refilled (1 750 from L2, 2 400 of 131072 rows, 2 900 of a million).  L2 itself has room: scattered rows reach the SMs at
// 18 TB/s with 216 KB in flight on each, but only a slot or so is.  The hold is a chain of hand-overs of 200-500 cycles each beside
// the MMAs, in a load/store pipe that the copies fill.  With four softmax warps that took a maximum over each row for every
// tile, two gather warps a slot and the last tile worked on whole, holds were 4 500 and a gathered tile 2 264 (16384 rows; now
// 2 110; struct Warps and tile_keys say what the last two gave alone), but the clock gives half of it back and more under the power cap: 32768 queries, two layers, 24.3 ms -> 23.7 ms; 16384
// of 131072, four layers, 34.8 -> 34.3 ms; 4096 of a million, four layers, 11.55 -> 11.45 ms; 1237 queries, four layers, 538 -> 527 us.
//
// Tensor memory columns:   0-255  O: value dims 0-255 in columns 0-127, 256-511 in 128-255; lanes 0-63 hold the first 128
//                                 dims of each, lanes 64-127 the second, lane l (mod 64) = head l
//                        256-383  Q[:, 0:512] as packed bf16, dims 0-255 in lanes 0-15 of each quarter, 256-511 in 16-31
//                        384-511  S, two buffers: the first chain's partial sum in lanes 0-15 of each quarter, the second's
//                                 in 16-31
#include "lsa_internal.h"
#include "lsa_tc.cuh"

namespace lsa {

namespace {

constexpr int kH = 64, kDQK = 576, kDV = 512;
constexpr int kTileKeys = 64;
constexpr int kAtoms = kDQK / 64;            // 9 column blocks of 64 dims (128 bytes) per row
constexpr int kAtomBytes = 64 * 128;         // 64 rows x 128 bytes
constexpr int kSlotBytes = kAtoms * kAtomBytes;

constexpr int kRing = 3;                     // 64-key tiles (or Q) in shared memory
constexpr int kDrainWarps = 4;
constexpr int kSumWarps = 4;                 // softmax warps that put a row's sums together (those of the tiles' first keys)
constexpr uint32_t kTmemColsAttn = 512;
constexpr uint32_t kColQ = 256, kColS = 384, kSBuf = 64;
constexpr float kLog2eTc = 1.4426950408889634f;
constexpr int kMaxClusterSplit = 16;         // row splits of one sequence = blocks of one cluster (eight is the portable limit)
constexpr int kFirstTileCycles = 8192;       // longest that a block's second tile is held back for the first
constexpr float kRescaleGap = 8.f;           // rescale O only when the row max grows by more than 2^8
// Warps of a block.  Prefill: the softmax of a tile by two warps per lane quarter, each with half of its keys, and three gather
// warps a ring slot (two issue a tile's 144 copies in 1 530 cycles, three in 1 430, which is about what the SM takes: 300 queries of
// 3000 rows 174 -> 171 us, 1000 of 9000 427 -> 420, a prompt of 32768, two layers, 24.8 -> 24.2 ms; 1237 queries of at most 1237 rows,
// four layers, lose, 505 -> 512 us).  23 warps leave 80 registers a thread, and 24 bytes of the prefill kernel spill; none do in 20 warps,
// with two gather warps a slot, which is the slower form all the same.  Where row lists are walked there are 16 warps, one softmax
// warp per quarter and two gather warps a slot: HBM paces the tiles, and a layer's ends are shorter with fewer threads (64
// sequences, four layers: 189 us, 195 with the prefill's eight softmax warps).
template <bool kRows>
struct Warps {
  static constexpr int kHalves = kRows ? 1 : 2, kSoftmax = 4 * kHalves;
  static constexpr int kDrain0 = kSoftmax, kQk = kDrain0 + kDrainWarps, kPv = kQk + 1, kGather0 = kPv + 1;
  static constexpr int kSlot = kRows ? 2 : 3, kAll = kGather0 + kRing * kSlot, kThreads = 32 * kAll;
  static constexpr int kRowsEach = kRows ? 32 : 24;   // cache rows of a tile that a gather warp copies (the last one the rest)
  static constexpr int kJobReaders = kSoftmax + kDrainWarps + 2 + kRing * kSlot;   // warps that release a job slot
  static_assert(kRowsEach % 8 == 0 && kRowsEach <= 32 && kRowsEach * (kSlot - 1) < kTileKeys, "whole groups of eight rows, a lane each");
};

struct AttnTcSmem {
  alignas(1024) uint8_t k[kRing][kAtoms][kAtomBytes];       // [ring slot][column block][64 rows x 128 B]
  alignas(1024) uint8_t q_rope[kAtomBytes];                 // Q[:, 512:576], 64 rows x 128 B
  alignas(8) uint64_t k_full[kRing], k_empty[kRing], p_ready[kRing], pv_done[kRing], q_tmem[2], s_full[2], s_free[2], job_full[2], job_empty[2], clc_full;
  alignas(8) uint64_t q_free;             // every Q K^T of a job is complete
  alignas(8) uint64_t o_full[2], o_free;  // a job's O and row sums are complete (by job parity); O has been read out
  alignas(8) uint64_t recv_full;          // two-split launches: the peer's rows and log-sum-exps have arrived
  alignas(16) uint4 clc;                  // answer of the cluster launch control
  alignas(8) int2 job[2];                 // {query or -1 = no more, rows it attends}
  uint32_t tmem_slot;
  int fail;                               // a softmax warp's wait ran out
  float half_max[2][kH];                  // [half of a tile's keys][head]: its maximum, where both halves have to know it
  float half_sum[kH];                     // row sums of the second halves
  float inv[2][kH];                       // 1 / l per head of the query being written out, by job parity
  alignas(16) float lse_own[kH];          // its log-sum-exp per head (log2 units); before that, of a rescale of O, the factors
  alignas(16) float lse_peer[kH / 2];     // two-split launches: the peer's, for the heads this block finishes
};
// Splits stage their partial rows in the order the softmax warps read them out of tensor memory: per warp (32 heads,
// half of the value dims) four column steps, each [head][64 floats] = 8 KB, the 16-byte chunks of a head's 256-byte piece
// XOR-swizzled by the head (no bank conflicts either way).  A step's 8 KB is contiguous, so the rows leave step by step, one bulk
// copy each, while the rest is still being read out, and keep that layout where they go: with two splits the rows the peer
// finishes, behind its staged ones; with more all of them, to the global scratch.
constexpr int kWarpStage = 32 * 256 * 4;
constexpr int kRecvOffset = 4 * kWarpStage;
constexpr uint32_t kRecvBytes = 2 * kWarpStage + (kH / 2) * 4;
static_assert(kRecvOffset + 2 * kWarpStage <= kRing * kSlotBytes, "staged and received rows must fit the ring");

// ---- thread-block cluster: barrier and loads from a peer block's shared memory
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// The two halves of the cluster barrier on their own: a thread arrives when it is done with a phase and waits later,
// where it needs every thread of the cluster to have arrived.
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
// Address of this block's shared-memory location `addr` in the block of rank `rank` of the cluster.
__device__ __forceinline__ uint32_t peer_smem(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
// Bulk copy from this block's shared memory into a peer block's (addresses from peer_smem); the bytes are counted on
// the peer's mbarrier.  16-byte aligned addresses, size a multiple of 16.
__device__ __forceinline__ void bulk_copy_to_peer(uint32_t dst_peer, uint32_t src, uint32_t bytes, uint32_t bar_peer) {
  asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst_peer), "r"(src), "r"(bytes), "r"(bar_peer) : "memory");
}

// ---- barrier of the softmax threads; the second form also tells every one of them whether any of them said yes
template <int kThreads>
__device__ __forceinline__ void softmax_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kThreads) : "memory"); }
template <int kThreads>
__device__ __forceinline__ bool softmax_any(bool v) {
  uint32_t r;
  asm volatile("{\n\t.reg .pred a, b;\n\tsetp.ne.b32 a, %1, 0;\n\tbar.red.or.pred b, 1, %2, a;\n\tselp.b32 %0, 1, 0, b;\n\t}"
               : "=r"(r) : "r"(static_cast<uint32_t>(v)), "n"(kThreads) : "memory");
  return r != 0;
}
__device__ __forceinline__ float exp2_fast(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// Four 8x8 bf16 matrices from the fragments of a warp; lane l gives the address of row l % 8 of matrix l / 8.
__device__ __forceinline__ void stmatrix_x4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
// Eight consecutive 32-bit words to global memory, 32-byte or 16-byte aligned.
__device__ __forceinline__ void store_words8(void* dst, const uint32_t* w, bool by32) {
  if (by32) {
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                 ::"l"(dst), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7]) : "memory");
  } else {
    reinterpret_cast<uint4*>(dst)[0] = make_uint4(w[0], w[1], w[2], w[3]);
    reinterpret_cast<uint4*>(dst)[1] = make_uint4(w[4], w[5], w[6], w[7]);
  }
}

template <int V>
struct IntC { static constexpr int value = V; };

// ---- cluster launch control: take over the index of a block of this grid that has not been launched yet
__device__ __forceinline__ void clc_request(uint32_t answer, uint32_t bar) {
  asm volatile("clusterlaunchcontrol.try_cancel.async.shared::cta.mbarrier::complete_tx::bytes.b128 [%0], [%1];"
               ::"r"(answer), "r"(bar) : "memory");
}
__device__ __forceinline__ bool clc_answer(uint32_t answer, int* block_x) {
  uint32_t x, ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b128 c;\n\t"
      "ld.shared.b128 c, [%2];\n\t"
      "clusterlaunchcontrol.query_cancel.is_canceled.pred.b128 p, c;\n\t"
      "selp.u32 %1, 1, 0, p;\n\t"
      "mov.u32 %0, 0;\n\t"
      "@p clusterlaunchcontrol.query_cancel.get_first_ctaid.v4.b32.b128 {%0, _, _, _}, c;\n\t}"
      : "=r"(x), "=r"(ok) : "r"(answer) : "memory");
  *block_x = static_cast<int>(x);
  return ok != 0;
}

// With n_split > 1 the kernel must be launched with clusters of (1, n_split, 1) blocks: the splits of one sequence
// are co-scheduled and merge their partial results themselves (no second kernel).  Block s finishes heads
// [s * 64 / n_split, (s + 1) * 64 / n_split): every block stages its rows (normalised, fp32) in shared memory and keeps
// its own share there.
//   Two splits (the decode configuration): the other 32 rows and their log-sum-exps are pushed straight into the
//   peer's shared memory, behind its staged rows, by bulk copies that count bytes on the peer's mbarrier.  The cluster
//   barrier is used in halves: a thread arrives when it has left the tile loop and waits before the first copy (the
//   peer's ring must be out of use before it receives), and once more around the end, so that no block leaves
//   while the other may still write into it.  Nothing goes through global memory.
//   Four, eight or 16 splits: the rows and all log-sum-exps go to the global scratch, where they stay in L2, as 16 bulk copies of
//   8 KB; after one cluster barrier the owner of a row combines the parts.  (Loads from a peer's shared memory moved the
//   same rows at about a quarter of the L2 path's rate; a bulk copy per row took 3 000 cycles longer to issue, stores
//   straight from the registers 4 000.)
//
// q_tma != 0: q_map describes q as a bf16 matrix [n_query * 64, 576] and Q arrives as one TMA box; otherwise the
// gather warps copy it with cp.async.  k_tma != 0 (contiguous caches only): k_map describes the cache rows, and key
// tiles that lie wholly inside the window, 64 consecutive rows, arrive as one TMA box as well.  k_g4 != 0: g_map
// describes the cache rows with a box one row high, and every other key tile is gathered four rows per instruction.
//
//   kRows       the caller's row lists are walked (else [window | sink | sparse] of a contiguous cache)
//   kSplits     row splits of a sequence: more than one are the blocks of a cluster and merge their results, with one the block goes
//               on to further queries.  A kernel has the code of one merge only, because it runs once per block, behind the fetch
//               of its instructions (all in one kernel: 1 to 3 % of a decode step; one sequence 68.1 us, 66.5 so, 24 137.1 and 134.6)
//   kParts      16 splits whose value dims are taken in 2 or 4 parts
template <bool kRows, int kSplits, bool kParts>
__global__ void __launch_bounds__(Warps<kRows>::kThreads, 1) sparse_attn_tc_kernel(const __grid_constant__ CUtensorMap q_map, int q_tma,
                                                                            const __grid_constant__ CUtensorMap k_map, int k_tma,
                                                                            const __grid_constant__ CUtensorMap g_map, int k_g4,
                                                                            AttnArgs p) {
  using W = Warps<kRows>;
  constexpr bool kClustered = kSplits > 1;
  static_assert(kRows || !kClustered, "row splits walk row lists");
  constexpr int kHalves = W::kHalves, kSoftmaxWarps = W::kSoftmax, kDrainWarp0 = W::kDrain0, kQkWarp = W::kQk, kPvWarp = W::kPv, kGatherWarp0 = W::kGather0;
  constexpr int kSlotWarps = W::kSlot, kRowsPerWarp = W::kRowsEach, kJobReaders = W::kJobReaders, kSoftmaxThreads = 32 * kSoftmaxWarps;
  extern __shared__ uint8_t smem_raw[];
  AttnTcSmem& sm = *reinterpret_cast<AttnTcSmem*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const int split = blockIdx.y;
  // Few sequences (clusters): value dims of a split in 2^v_shift parts, each by a cluster of its own (512 >> v_shift dims from vpart on).
  const int v_shift = kParts ? p.v_shift : 0, vpart = kParts ? static_cast<int>(blockIdx.z) : 0;
  float* const part_out = p.part_out;
  float* const part_lse = p.part_lse;

  constexpr bool clustered = kClustered;
  constexpr bool pair = kSplits == 2;   // two splits exchange their rows through shared memory
  const bool raised = tc::status_raised(p.status);   // an earlier block of this launch (or an earlier launch) gave up on a wait

  // ---- set-up
  if (tid == 0) {
    for (int b = 0; b < kRing; ++b) {
      tc::mbar_init(smem_u32(&sm.k_full[b]), kSlotWarps);
      tc::mbar_init(smem_u32(&sm.k_empty[b]), 1);
      tc::mbar_init(smem_u32(&sm.p_ready[b]), 1);
      tc::mbar_init(smem_u32(&sm.pv_done[b]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      tc::mbar_init(smem_u32(&sm.o_full[b]), 1 + kSumWarps);
      tc::mbar_init(smem_u32(&sm.q_tmem[b]), kDrainWarps);     // by job parity: a job without tiles may be overtaken by the next
      tc::mbar_init(smem_u32(&sm.s_full[b]), 1);
      tc::mbar_init(smem_u32(&sm.s_free[b]), kSoftmaxWarps);
      tc::mbar_init(smem_u32(&sm.job_full[b]), 1);
      tc::mbar_init(smem_u32(&sm.job_empty[b]), kJobReaders);
    }
    tc::mbar_init(smem_u32(&sm.clc_full), 1);
    tc::mbar_init(smem_u32(&sm.q_free), 1);
    tc::mbar_init(smem_u32(&sm.o_free), kDrainWarps);
    if constexpr (kClustered) {
      tc::mbar_init(smem_u32(&sm.recv_full), 1);
      if (pair) tc::mbar_expect_tx(smem_u32(&sm.recv_full), kRecvBytes);   // armed once; used once per launch
    }
    sm.fail = 0;
    tc::fence_mbar_init();
  }
  if (warp == kQkWarp) {
    tc::tmem_alloc(smem_u32(&sm.tmem_slot), kTmemColsAttn);
    tc::tmem_relinquish();
  }
  tc::fence_before_sync();
  const bool dead = __syncthreads_or(raised) != 0;   // the same in all threads (see block_gives_up); the set-up ran meanwhile
  tc::fence_after_sync();
  const uint32_t tmem_base = sm.tmem_slot;
  if (dead && !clustered) {
    if (warp == kQkWarp) tc::tmem_dealloc(tmem_base, kTmemColsAttn);
    return;
  }
  // Programmatic dependent launch: this block may have been placed while the previous kernel of the stream was still
  // draining; what that kernel wrote is read, and what it may still read is overwritten, only after
  // griddepcontrol.wait.  The next kernel's blocks may be placed from then on.
  // rows_stable: the row lists (and the caches, as always) were complete before the previous kernel started, so the
  // gather warps read them and put the first two key tiles in flight while that kernel drains, and wait only before
  // they request Q; every other thread waits here.
  const bool early_rows = kRows && p.rows_stable != 0 && q_tma != 0;   // block-uniform
  auto dependency_wait = [&]() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  };
  const bool reads_early = warp >= kGatherWarp0 || (warp >= kDrainWarp0 && warp < kDrainWarp0 + kDrainWarps);
  if (!(early_rows && reads_early)) dependency_wait();

  // ---- the parts of a job that every role derives for itself
  struct Job {
    int qi, n_tot, n_win, n_sink, tile_begin, n_tiles, q_at;
    int64_t win0;
  };
  // Ring positions of a job that starts at position b: Q at b + q_at, tile i at b + i + (i >= q_at), n_tiles + 1 in all.
  // Q comes first; with early_rows two tiles go ahead of it.
  auto job_of = [&](int2 j) -> Job {
    Job b;
    b.qi = j.x;
    b.n_tot = j.y;
    b.n_win = b.n_sink = 0;
    b.win0 = 0;
    if constexpr (!kRows) {
      const int64_t t = p.q_pos0 + b.qi;
      b.n_sink = static_cast<int>(min64(p.S, t + 1));
      b.win0 = max64(p.S, t - p.W + 1);
      b.n_win = static_cast<int>(max64(0, t - b.win0 + 1));
    }
    const int tiles_all = (b.n_tot + kTileKeys - 1) / kTileKeys;
    const int tiles_per = kClustered ? (tiles_all + kSplits - 1) / kSplits : tiles_all;
    b.tile_begin = kClustered ? split * tiles_per : 0;
    b.n_tiles = max(0, min(tiles_all, b.tile_begin + tiles_per) - b.tile_begin);
    if (dead) b.n_tiles = 0;   // the peers of this cluster still expect this block at the cluster barrier
    b.q_at = early_rows ? min(2, b.n_tiles) : 0;
    return b;
  };
  // Keys of tile i that are worked on: the last tile's in whole MMA steps of 16.  It shows where jobs are short (1237 queries of at
  // most 1237 rows, four layers: 518 -> 512 us); 3076 rows are 48 tiles and four rows, and there it is within the noise.  Not where row
  // lists are walked: HBM paces those tiles, and loops of a constant length are issued faster.
  auto tile_keys = [](const Job& b, int i) -> int {
    if constexpr (kRows) return kTileKeys;
    else return min(kTileKeys, (b.n_tot - (b.tile_begin + i) * kTileKeys + 15) & ~15);
  };
  auto wait_job = [&](int n, int2* j) -> bool {   // n-th job of this block; whole warp or one thread
    const bool ok = tc::mbar_wait(smem_u32(&sm.job_full[n & 1]), (n >> 1) & 1, p.status);
    *j = ok ? sm.job[n & 1] : make_int2(-1, 0);
    return ok;
  };
  auto slot_of = [](int pos) -> int { return pos % kRing; };
  auto use_of = [](int pos) -> uint32_t { return static_cast<uint32_t>(pos / kRing) & 1u; };   // parity of the slot's use

  if (warp >= kDrainWarp0 && warp < kDrainWarp0 + kDrainWarps) {
    // ================= scheduler, Q and O =================
    const int dw = warp - kDrainWarp0;   // TMEM lanes 32 dw .. +31
    const uint32_t lane_addr = static_cast<uint32_t>(32 * dw) << 16;
    // n-th job of this block, by one thread; false: there are no more.  (Its slot is free once every role is through with the
    // job before the previous one, so at most one job beyond the one being worked on is taken from the other blocks.)
    auto publish = [&](int n) -> bool {
      if (!tc::mbar_wait(smem_u32(&sm.job_empty[n & 1]), ((n >> 1) & 1) ^ 1, p.status)) return false;
      int qi = kClustered ? static_cast<int>(blockIdx.x) : p.n_query - 1 - static_cast<int>(blockIdx.x);
      if (n > 0) {
        qi = -1;
        // (Where every job has an SM none is taken from another block: a block that is placed early, while the kernel before
        // still holds some SMs, would take jobs that those SMs are about to run.  82 sequences, 2 layers: 188 us, 137 so.)
        if (!kClustered && p.n_query > p.sm_count) {
          tc::mbar_expect_tx(smem_u32(&sm.clc_full), 16);
          clc_request(smem_u32(&sm.clc), smem_u32(&sm.clc_full));
          if (!tc::mbar_wait(smem_u32(&sm.clc_full), (n - 1) & 1, nullptr)) {   // (an answer on its way is waited for in any case)
            report_status(p.status, kDevTimeout);
            return false;
          }
          int x;
          if (clc_answer(smem_u32(&sm.clc), &x)) qi = p.n_query - 1 - x;
          tc::fence_proxy_async();   // the answer has been read: the next one may overwrite it
        }
      }
      int n_tot = 0;
      if (qi >= 0) {
        if constexpr (kRows) {
          n_tot = p.n_rows[qi];
        } else {
          const int64_t t = p.q_pos0 + qi;
          const int64_t win0 = max64(p.S, t - p.W + 1);
          n_tot = static_cast<int>(min64(p.S, t + 1) + max64(0, t - win0 + 1)) + p.n_sparse[qi];
        }
      }
      sm.job[n & 1] = make_int2(qi, n_tot);
      tc::mbar_arrive(smem_u32(&sm.job_full[n & 1]));
      return qi >= 0;
    };
    bool more = dw == 0 && lane == 0;   // this thread publishes, and there may be more jobs
    if (more) more = publish(0);
    if (more) more = publish(1);
    __syncwarp();
    if (early_rows) dependency_wait();
    // Q of a job from its ring slot to tensor memory, in the order the tensor core reads an A operand (two dims per column)
    auto move_q = [&](int pos, int n_job) -> bool {
      if (!__all_sync(0xffffffffu, tc::mbar_wait(smem_u32(&sm.k_full[slot_of(pos)]), use_of(pos), p.status))) return false;
      const int row = 16 * dw + (lane & 15), hi = lane >> 4;
      const uint8_t* qs = sm.k[slot_of(pos)][0] + row * 128;
#pragma unroll 1
      for (int part = 0; part < 4; ++part) {
        uint32_t w[32];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int c = 32 * hi + 8 * part + j;
          const uint4 u = *reinterpret_cast<const uint4*>(qs + (c >> 3) * kAtomBytes + (((c & 7) ^ (row & 7)) << 4));
          w[4 * j] = u.x; w[4 * j + 1] = u.y; w[4 * j + 2] = u.z; w[4 * j + 3] = u.w;
        }
        tc::tmem_st32(tmem_base + lane_addr + kColQ + part * 32, w);
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {   // the warp's 16 rows of the rope block, as they lie
        const int at = 16 * dw * 128 + (32 * j + lane) * 16;
        *reinterpret_cast<uint4*>(sm.q_rope + at) = *reinterpret_cast<const uint4*>(sm.k[slot_of(pos)][8] + at);
      }
      tc::fence_proxy_async();
      tc::tmem_st_wait();
      tc::fence_before_sync();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(smem_u32(&sm.q_tmem[n_job & 1]));
      return true;
    };
    int2 jd;
    int base = 0;
    bool ok = __all_sync(0xffffffffu, wait_job(0, &jd));
    Job jb = job_of(jd);
    ok = ok && move_q(base + jb.q_at, 0);
    if constexpr (!kClustered) {
      // Of O a warp reads its TMEM lanes: heads 32 (dw & 1) + lane, half dw >> 1 of the value dims of each 256.
      const int head_o = 32 * (dw & 1) + lane, half_o = dw >> 1;
      for (int n = 0; ok; ++n) {
        const Job done = jb;
        base += done.n_tiles + 1;
        ok = __all_sync(0xffffffffu, wait_job(n + 1, &jd));
        if (!ok) break;
        if (jd.x >= 0) {   // the next Q follows the last Q K^T of this job, whose softmax and P V are still to come
          jb = job_of(jd);
          ok = __all_sync(0xffffffffu, tc::mbar_wait(smem_u32(&sm.q_free), n & 1, p.status));
          if (!ok) break;
          tc::fence_after_sync();
          ok = move_q(base + jb.q_at, n + 1);
          if (!ok) break;
        }
        ok = __all_sync(0xffffffffu, tc::mbar_wait(smem_u32(&sm.o_full[n & 1]), (n >> 1) & 1, p.status));
        if (!ok) break;
        tc::fence_after_sync();
        // ---- O / l: a thread owns half of the value dims of a head, in two runs of 128
        const float inv = sm.inv[n & 1][head_o];
        uint8_t* dst = reinterpret_cast<uint8_t*>(reinterpret_cast<__nv_bfloat16*>(p.out) + (static_cast<int64_t>(done.qi) * kH + head_o) * kDV + 128 * half_o);
        const bool by32 = (reinterpret_cast<uintptr_t>(p.out) & 31u) == 0;
#pragma unroll 1
        for (int c = 0; c < 256; c += 32) {
          uint32_t o[32];
          if (done.n_tiles > 0) {
            tc::tmem_ld32(tmem_base + lane_addr + c, o);
            tc::tmem_ld_wait();
          } else {
#pragma unroll
            for (int j = 0; j < 32; ++j) o[j] = 0u;
          }
          if (c == 224) {   // all of O is in registers: the next job's P V may begin
            tc::fence_before_sync();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(smem_u32(&sm.o_free));
          }
          uint32_t w[16];
#pragma unroll
          for (int j = 0; j < 16; ++j) w[j] = pack_bf16(__uint_as_float(o[2 * j]) * inv, __uint_as_float(o[2 * j + 1]) * inv);
          uint8_t* d = dst + ((c >> 7) * 256 + (c & 127)) * 2;
#pragma unroll
          for (int j = 0; j < 16; j += 8) store_words8(d + j * 4, w + j, by32);
        }
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(smem_u32(&sm.job_empty[n & 1]));
        if (more) more = publish(n + 2);
        __syncwarp();
        if (jd.x < 0) break;
      }
    }
  } else if (warp >= kGatherWarp0) {
    // ================= gather warps =================
    const int grp = (warp - kGatherWarp0) / kSlotWarps, gw = (warp - kGatherWarp0) % kSlotWarps;   // ring slot, warp of its group
    const int warp_rows = kSlotWarps * kRowsPerWarp == kTileKeys ? kRowsPerWarp : min(kRowsPerWarp, kTileKeys - kRowsPerWarp * gw);
    const uint8_t* kg = reinterpret_cast<const uint8_t*>(p.k);
    const bool g4 = k_g4 != 0;   // block-uniform
    const uint32_t full = smem_u32(&sm.k_full[grp]), empty = smem_u32(&sm.k_empty[grp]);
    bool waited = !early_rows;   // this thread has executed the dependency wait
    bool alive = true;
    int base = 0, last_pos = -1;   // ring position of the job's first item; the group's last item that is on its way
    for (int n = 0; alive; ++n) {
      int2 jd;
      if (!__all_sync(0xffffffffu, wait_job(n, &jd)) || jd.x < 0) break;
      const Job jb = job_of(jd);
      const int32_t* rows = kRows ? p.rows + static_cast<int64_t>(jb.qi) * p.rows_ld : nullptr;
      const int32_t* sp = p.sparse_idx ? p.sparse_idx + static_cast<int64_t>(jb.qi) * p.Ksp : nullptr;
      // Without a row list the keys are visited as [window | sink | sparse] (the order within one softmax is free): the
      // window is a run of consecutive cache rows, so its whole tiles need no per-row addressing.
      auto row_of = [&](int i) -> int32_t {
        if (i >= jb.n_tot) return -1;
        if constexpr (kRows) {
          return checked_row(rows[i], p.n_key, p.status);
        } else {
          if (i < jb.n_win) return static_cast<int32_t>(jb.win0 + i);
          if (i < jb.n_win + jb.n_sink) return i - jb.n_win;
          return checked_row(sp[i - jb.n_win - jb.n_sink], p.n_key, p.status);
        }
      };
      auto tile_of = [&](int e) -> int { return e - (e > jb.q_at ? 1 : 0); };
      auto tile_by_tma = [&](int i) -> bool {   // block-uniform
        return !kRows && k_tma && (jb.tile_begin + i + 1) * kTileKeys <= jb.n_win;
      };
      auto my_key_row = [&](int e) -> int32_t {   // each lane looks up the cache row of one of the warp's keys
        const int i = tile_of(e);
        return (e != jb.q_at && e <= jb.n_tiles && lane < warp_rows && !tile_by_tma(i))
                   ? row_of((jb.tile_begin + i) * kTileKeys + kRowsPerWarp * gw + lane) : -1;
      };
      int e = (grp + kRing - base % kRing) % kRing;
      int32_t my_row = my_key_row(e);
      for (; e <= jb.n_tiles; e += kRing) {
        const int pos = base + e;
        const bool is_q = e == jb.q_at;
        const int i = tile_of(e);   // the tile (if this is not Q)
        const int rows_here = kRows ? warp_rows : max(0, min(warp_rows, tile_keys(jb, i) - kRowsPerWarp * gw));   // of it, by this warp (a multiple of 8)
        const int32_t next_row = my_key_row(e + kRing);   // fetched before the wait: off the critical path
        if (e >= jb.q_at && !waited) {   // the tiles before Q are in flight: now the previous kernel must be done
          dependency_wait();
          waited = true;
        }
        if (!__all_sync(0xffffffffu, tc::mbar_wait(empty, use_of(pos) ^ 1, p.status))) { alive = false; break; }
        // A block's first tile goes out alone: requested together with the next one it would share the memory pipe
        // with it, and the first Q K^T would start a tile's worth of traffic later.  (A look with a limit, not a wait: this
        // group is not the barrier's own waiter.)
        if (n == 0 && e == (jb.q_at == 0 ? 2 : 1)) {
          const long long t0 = clock64();
          while (!tc::mbar_test(smem_u32(&sm.k_full[slot_of(pos - 1)]), 0) && clock64() - t0 < kFirstTileCycles) {}
          __syncwarp();
        }
        last_pos = pos;
        if (is_q && q_tma) {
          if (gw == 0 && tc::elect_one()) {
            tc::mbar_expect_tx_only(full, kSlotBytes);
            tc::tma_load_3d(smem_u32(sm.k[grp]), &q_map, 0, jb.qi * kH, 0, full);
          }
        } else if (is_q) {
          const uint8_t* qg = reinterpret_cast<const uint8_t*>(p.q) + static_cast<int64_t>(jb.qi) * kH * kDQK * 2;
          for (int x = gw * 32 + lane; x < kH * (kDQK / 8); x += 32 * kSlotWarps) {
            const int r = x / (kDQK / 8), c = x % (kDQK / 8);
            cp_async16(smem_u32(sm.k[grp][c >> 3]) + r * 128 + (((c & 7) ^ (r & 7)) << 4), qg + r * kDQK * 2 + c * 16, 16);
          }
        } else if (tile_by_tma(i)) {
          // 64 consecutive window rows: one box, counted on k_full
          if (gw == 0 && tc::elect_one()) {
            tc::mbar_expect_tx_only(full, kSlotBytes);
            tc::tma_load_3d(smem_u32(sm.k[grp]), &k_map, 0, static_cast<int>(jb.win0) + (jb.tile_begin + i) * kTileKeys, 0, full);
          }
        } else if (g4) {
          // scattered rows: four rows x 64 dims per instruction, straight into their place in the swizzled tile
          if (lane == 0) tc::mbar_expect_tx_only(full, static_cast<uint32_t>(rows_here) * (kDQK * 2));
          __syncwarp();
          for (int u = lane; u < rows_here / 4 * kAtoms; u += 32) {
            const int q4 = u / kAtoms, atom = u % kAtoms;
            int4 r;
            // past the end of the list its last row once more: masked in the softmax, and as a value of weight 0 it must not be
            // somebody else's (0 x NaN)
            const int i0 = (jb.tile_begin + i) * kTileKeys + kRowsPerWarp * gw + 4 * q4;
            auto listed = [&](int k) -> int32_t { return max(row_of(min(k, jb.n_tot - 1)), 0); };
            r.x = listed(i0); r.y = listed(i0 + 1); r.z = listed(i0 + 2); r.w = listed(i0 + 3);
            tc::tma_gather4_2d(smem_u32(sm.k[grp][atom]) + (kRowsPerWarp * gw + 4 * q4) * 128, &g_map, atom * 64, r.x, r.y, r.z, r.w, full);
          }
        } else {
          // the 72 16-byte chunks of a row: 64 by all lanes in two instructions; the last eight of four rows in one
          const uint32_t dst0 = smem_u32(sm.k[grp][lane >> 3]) + kRowsPerWarp * gw * 128;
#pragma unroll 8
          for (int rr = 0; rr < rows_here; ++rr) {
            const int32_t row = __shfl_sync(0xffffffffu, my_row, rr);
            const uint8_t* src = kg + static_cast<int64_t>(row >= 0 ? row : 0) * p.ld_k * 2 + lane * 16;
            const int nb = row >= 0 ? 16 : 0;
            const uint32_t dst = dst0 + rr * 128 + (((lane & 7) ^ (rr & 7)) << 4);
            cp_async16(dst, src, nb);
            cp_async16(dst + 4 * kAtomBytes, src + 512, nb);
            if ((rr & 3) == 3) {
              const int r4 = rr - 3 + (lane >> 3);
              const int32_t row4 = __shfl_sync(0xffffffffu, my_row, r4);
              cp_async16(smem_u32(sm.k[grp][8]) + (kRowsPerWarp * gw + r4) * 128 + (((lane & 7) ^ (r4 & 7)) << 4),
                         kg + static_cast<int64_t>(row4 >= 0 ? row4 : 0) * p.ld_k * 2 + 1024 + (lane & 7) * 16, row4 >= 0 ? 16 : 0);
            }
          }
        }
        cp_async_commit();
        cp_async_wait<0>();
        tc::fence_proxy_async();
        __syncwarp();   // one arrival per warp: dozens of threads on one barrier are as many serialised shared-memory operations
        if (lane == 0) tc::mbar_arrive(full);
        my_row = next_row;
      }
      base += jb.n_tiles + 1;
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(smem_u32(&sm.job_empty[n & 1]));
    }
    // a wait ran out: a box still on its way lands before the block ends (the wait is bounded too)
    if (!alive && last_pos >= 0) (void)tc::mbar_wait(full, use_of(last_pos), nullptr);
    if (!waited) dependency_wait();
  } else if (warp == kQkWarp) {
    // ================= issuer of Q K^T =================
    if (tc::elect_one()) {
      // Descriptors are built once; inside the loops only the start-address word moves (one add per operand).
      const uint64_t dk0 = tc::smem_desc_sw128(smem_u32(sm.k), 16, 1024);           // K-major view
      const uint64_t dqr = tc::smem_desc_sw128(smem_u32(sm.q_rope), 16, 1024);
      constexpr uint32_t kLane16 = 16u << 16;
      bool ok = true;
      int base = 0, g = 0;   // ring position of the job's first item; tile number over all jobs
      for (int n = 0; ok; ++n) {
        int2 jd;
        if (!wait_job(n, &jd) || jd.x < 0) break;
        const Job jb = job_of(jd);
        if (!tc::mbar_wait(smem_u32(&sm.q_tmem[n & 1]), (n >> 1) & 1, p.status)) break;
        tc::mbar_arrive(smem_u32(&sm.k_empty[slot_of(base + jb.q_at)]));   // Q has left its ring slot
        for (int i = 0; i < jb.n_tiles; ++i, ++g) {
          const int pos = base + i + (i >= jb.q_at ? 1 : 0);
          ok = tc::mbar_wait(smem_u32(&sm.k_full[slot_of(pos)]), use_of(pos), p.status) &&
               tc::mbar_wait(smem_u32(&sm.s_free[g & 1]), ((g >> 1) & 1) ^ 1, p.status);   // the S before last has been read
          if (ok && p.qk_waits_pv != 0 && i >= 2) {   // (a debugging aid: no product needs it)
            const int pp = base + i - 2 + (i - 2 >= jb.q_at ? 1 : 0);
            ok = tc::mbar_wait(smem_u32(&sm.k_empty[slot_of(pp)]), use_of(pp), p.status);
          }
          if (!ok) break;
          tc::fence_after_sync();
          const uint64_t dkb = tc::desc_advance(dk0, slot_of(pos) * kSlotBytes);
          const uint32_t idesc = tc::idesc_bf16(kH, tile_keys(jb, i), 0, 0);
#pragma unroll
          for (int x = 0; x < 2; ++x) {
            const uint32_t q_src = tmem_base + x * kLane16 + kColQ, s_dst = tmem_base + x * kLane16 + kColS + (g & 1) * kSBuf;
#pragma unroll
            for (int s = 0; s < 16; ++s)   // dims 256x + 16s .. +15: column block 4x + s/4, 32-byte slice s%4
              tc::umma_ts(s_dst, q_src + 8 * s, tc::desc_advance(dkb, (4 * x + (s >> 2)) * kAtomBytes + (s & 3) * 32), idesc, s != 0);
#pragma unroll
            for (int s = 0; s < 2; ++s)    // rope dims 512 + 32x + 16s .. +15
              tc::umma_ss(s_dst, tc::desc_advance(dqr, (2 * x + s) * 32), tc::desc_advance(dkb, 8 * kAtomBytes + (2 * x + s) * 32), idesc, 1);
          }
          tc::umma_commit(smem_u32(&sm.s_full[g & 1]));
        }
        base += jb.n_tiles + 1;
        if (!ok) break;
        if constexpr (!kClustered) {
          if (jb.n_tiles > 0) tc::umma_commit(smem_u32(&sm.q_free));
          else tc::mbar_arrive(smem_u32(&sm.q_free));
        }
        tc::mbar_arrive(smem_u32(&sm.job_empty[n & 1]));
      }
    }
  } else if (warp == kPvWarp) {
    // ================= issuer of P V =================
    if (tc::elect_one()) {
      // B = V read MN-major; a cluster with a part of the value dims takes half as many, or one MMA of half the width, per step
      const uint32_t idesc = v_shift == 2 ? tc::idesc_bf16(kH, 128, 0, 1) : tc::idesc_bf16(kH, 256, 0, 1);
      const uint32_t v_block = static_cast<uint32_t>(vpart * (8 >> v_shift)) * kAtomBytes;
      const uint64_t dv0 = tc::smem_desc_sw128(smem_u32(sm.k), kAtomBytes, 1024);   // MN-major view of a tile
      const uint64_t dp0 = tc::smem_desc_sw128(smem_u32(sm.k[0][8]), 16, 1024);     // P in its rope block
      bool ok = true;
      int base = 0, g = 0;
      for (int n = 0; ok; ++n) {
        int2 jd;
        if (!wait_job(n, &jd) || jd.x < 0) break;
        const Job jb = job_of(jd);
        if (!kClustered && n > 0) ok = tc::mbar_wait(smem_u32(&sm.o_free), (n - 1) & 1, p.status);   // the last job's O has been read out
        for (int i = 0; i < jb.n_tiles && ok; ++i, ++g) {
          const int slot = slot_of(base + i + (i >= jb.q_at ? 1 : 0));
          ok = tc::mbar_wait(smem_u32(&sm.p_ready[g % kRing]), (g / kRing) & 1, p.status);
          if (!ok) break;
          tc::fence_after_sync();
          const uint64_t dvb = tc::desc_advance(dv0, slot * kSlotBytes), dpb = tc::desc_advance(dp0, slot * kSlotBytes);
          const int keys = tile_keys(jb, i);
#pragma unroll
          for (int y = 0; y < 2; ++y)       // value dims 256y .. +255 (of the cluster's part)
#pragma unroll
            for (int kk = 0; kk < kTileKeys / 16; ++kk)   // keys 16*kk .. +15
              if (16 * kk < keys && (y == 0 || v_shift == 0))
                tc::umma_ws_ss(tmem_base + 128 * y, tc::desc_advance(dpb, kk * 32), tc::desc_advance(dvb, v_block + 4 * y * kAtomBytes + kk * 2048),
                               idesc, (i > 0) || (kk > 0));
          // "P V of the tile done" frees the ring slot for the gather warps, and tells the softmax warps that O may be touched
          // again: where a block goes on to another job by a barrier of its own, since the slot's may go on with the next
          // query (which only its issuer waits for) before they look, and a barrier two uses on looks like an unused one
          tc::umma_commit(smem_u32(&sm.k_empty[slot]));
          if constexpr (!kClustered) tc::umma_commit(smem_u32(&sm.pv_done[g % kRing]));
        }
        base += jb.n_tiles + 1;
        if (!ok) break;
        if constexpr (!kClustered) {
          if (jb.n_tiles > 0) tc::umma_commit(smem_u32(&sm.o_full[n & 1]));
          else tc::mbar_arrive(smem_u32(&sm.o_full[n & 1]));
        }
        tc::mbar_arrive(smem_u32(&sm.job_empty[n & 1]));
      }
    }
  } else {
    // ================= softmax warps =================
    // Warp w owns the S rows (heads) 16w .. 16w+15; with two halves warps w and w + 4 do, the first of keys 0-31 of a tile, the other
    // of keys 32-63.  As 16-lane fragments, a thread holds keys 8j + 2 (lane % 4) + {0, 1} of its half, of heads 16w + lane / 4 and
    // 8 more.  Of O it reads lanes 32w .. +31: heads 32 (w & 1) + lane, half w >> 1 of the value dims of each 256, and its half of
    // those columns.
    constexpr int kKeys = kTileKeys / kHalves, kGroups = kKeys / 8;   // keys of a half, in fragments of eight
    const int quarter = warp & 3, half = warp >> 2;
    const uint32_t lane_addr = static_cast<uint32_t>(32 * quarter) << 16;
    const int head_o = 32 * (quarter & 1) + lane, half_o = quarter >> 1;
    const int row_s = 16 * quarter + (lane >> 2);   // the first of the thread's two heads
    const float zs = p.sm_scale * kLog2eTc;
    bool ok = true;
    // P V of tile g (over all jobs), which lies at ring position `pos`, is complete; whole warp
    auto wait_pv = [&](int g, int pos) -> bool {
      const uint32_t bar = kClustered ? smem_u32(&sm.k_empty[slot_of(pos)]) : smem_u32(&sm.pv_done[g % kRing]);
      return __all_sync(0xffffffffu, tc::mbar_wait(bar, kClustered ? use_of(pos) : static_cast<uint32_t>(g / kRing) & 1u, p.status));
    };
    int base = 0, tiles_done = 0, n = 0;
    int2 jd;
    ok = __all_sync(0xffffffffu, wait_job(0, &jd));
    Job jb = job_of(jd);
    bool have_o = false;
    float m_used[2] = {0.f, 0.f}, l_run[2] = {0.f, 0.f};   // rows row_s and row_s + 8; l_run is this thread's share
    // A warp whose wait ran out goes on to the next vote, where all of them learn of it and leave together: the named barrier
    // has no time limit.
    bool go = !softmax_any<kSoftmaxThreads>(!ok);
    while (go) {
      // ---- the tiles of the job
      l_run[0] = l_run[1] = 0.f;
      bool failed = false;
      for (int i = 0; i < jb.n_tiles; ++i) {
        const int g = tiles_done + i;
        const int slot = slot_of(base + i + (i >= jb.q_at ? 1 : 0));
        ok = ok && __all_sync(0xffffffffu, tc::mbar_wait(smem_u32(&sm.s_full[g & 1]), (g >> 1) & 1, p.status));
        tc::fence_after_sync();
        float2 v[2 * kGroups];   // [key group j][row r] at 2j + r
        {
          uint32_t a[4 * kGroups], c[4 * kGroups];
          const uint32_t s_addr = tmem_base + lane_addr + kColS + (g & 1) * kSBuf + kKeys * half;
          tc::tmem_ld_16x256b(s_addr, a);
          tc::tmem_ld_16x256b(s_addr + (16u << 16), c);
          tc::tmem_ld_wait();
          tc::fence_before_sync();
          __syncwarp();
          if (lane == 0) tc::mbar_arrive(smem_u32(&sm.s_free[g & 1]));
#pragma unroll
          for (int j = 0; j < 2 * kGroups; ++j)
            v[j] = add2(make_float2(__uint_as_float(a[2 * j]), __uint_as_float(a[2 * j + 1])),
                        make_float2(__uint_as_float(c[2 * j]), __uint_as_float(c[2 * j + 1])));
        }
        const int n_valid = jb.n_tot - (jb.tile_begin + i) * kTileKeys - kKeys * half;   // keys of this half that exist
        if (n_valid < kKeys) {
          const int k0 = 2 * (lane & 3);
#pragma unroll
          for (int j = 0; j < kGroups; ++j) {
            if (8 * j + k0 >= n_valid) v[2 * j].x = v[2 * j + 1].x = -INFINITY;
            if (8 * j + k0 + 1 >= n_valid) v[2 * j].y = v[2 * j + 1].y = -INFINITY;
          }
        }
        // Running max in log2 units: that of the job's first tile, moved only when a row grows by more than kRescaleGap (O and l
        // are then rescaled).  With two halves P is worked out with the maximum as it is, and the vote that ends the tile says whether
        // that was good enough for every row, so a row's lanes and halves compare their values only where they have to: shuffles and
        // barriers queue behind the gather warps' copies (110-150 cycles each).  If it was not, P is worked out again (300 queries of
        // 3000 rows, two layers: 375 us with four warps that compare first, 366 so, 384 with eight that compare first; where the spread
        // of the scores keeps growing along the rows, so that nearly every tile is rescaled, 409, 420 and 412).
        // Where row lists are walked the lanes compare first: HBM paces those tiles, and a rescaling costs no second P (64 sequences
        // whose last 300 rows score highest, as recent tokens do, three layers: 149.1 us, 151.4 with P first).
        float mx[2];   // of the thread's values, then of the rows'
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          float x = fmaxf(v[r].x, v[r].y);
#pragma unroll
          for (int j = 1; j < kGroups; ++j) x = fmaxf(x, fmaxf(v[2 * j + r].x, v[2 * j + r].y));
          mx[r] = x * zs;
        }
        auto row_max = [&]() {
#pragma unroll
          for (int r = 0; r < 2; ++r) {
            mx[r] = fmaxf(mx[r], __shfl_xor_sync(0xffffffffu, mx[r], 1));
            mx[r] = fmaxf(mx[r], __shfl_xor_sync(0xffffffffu, mx[r], 2));
            if (kHalves > 1 && (lane & 3) == 0) sm.half_max[half][row_s + 8 * r] = mx[r];
          }
          if constexpr (kHalves > 1) {
            softmax_sync<kSoftmaxThreads>();
#pragma unroll
            for (int r = 0; r < 2; ++r) mx[r] = fmaxf(mx[r], sm.half_max[half ^ 1][row_s + 8 * r]);
          }
        };
        float alpha[2] = {1.f, 1.f};   // factors of the rows that have grown too far
        auto move_max = [&]() {
#pragma unroll
          for (int r = 0; r < 2; ++r) {
            alpha[r] = 1.f;
            if (mx[r] > m_used[r] + kRescaleGap) {
              alpha[r] = exp2_fast(m_used[r] - mx[r]);
              m_used[r] = mx[r];
            }
            l_run[r] *= alpha[r];
          }
        };
        bool need = false;
        if (i == 0 || kHalves == 1) row_max();
        if (i == 0) {
          m_used[0] = mx[0];
          m_used[1] = mx[1];
        } else {
          need = mx[0] > m_used[0] + kRescaleGap || mx[1] > m_used[1] + kRescaleGap;
          if constexpr (kHalves == 1) move_max();
        }
        float sum[2];
        auto work_out_p = [&]() {
          // P = exp2(z - m), fp32 row sums, bf16 pack
          uint32_t pk[kGroups][2];
#pragma unroll
          for (int r = 0; r < 2; ++r) {
            const float2 z2 = make_float2(zs, zs), m2 = make_float2(-m_used[r], -m_used[r]);
            float2 sum2 = make_float2(0.f, 0.f);
#pragma unroll
            for (int j = 0; j < kGroups; ++j) {
              float2 e = fma2(v[2 * j + r], z2, m2);
              e.x = exp2_fast(e.x);
              e.y = exp2_fast(e.y);
              sum2 = add2(sum2, e);
              pk[j][r] = pack_bf16(e.x, e.y);
            }
            sum[r] = sum2.x + sum2.y;
          }
          // P takes the place of the tile's rope dims, which only Q K^T reads
          const int row = 16 * quarter + ((lane >> 3) & 1) * 8 + (lane & 7);
          const uint32_t dst = smem_u32(sm.k[slot][8]) + row * 128;
#pragma unroll
          for (int j = 0; j < kGroups; j += 2)
            stmatrix_x4(dst + (((kGroups * half + j + (lane >> 4)) ^ (row & 7)) << 4), pk[j][0], pk[j][1], pk[j + 1][0], pk[j + 1][1]);
        };
        if constexpr (kHalves == 1) work_out_p();
        while (true) {
          if constexpr (kHalves > 1) work_out_p();
          if (!ok) sm.fail = 1;
          tc::fence_proxy_async();   // P is read by the tensor core
          if (!softmax_any<kSoftmaxThreads>(need || !ok)) break;
          if (*reinterpret_cast<volatile int*>(&sm.fail)) {
            failed = true;
            break;
          }
          // rare: O of every head times its factor, once P V of the tile before is complete
          if constexpr (kHalves > 1) {
            row_max();
            move_max();
          }
#pragma unroll
          for (int r = 0; r < 2; ++r)
            if (half == 0 && (lane & 3) == 0) sm.lse_own[row_s + 8 * r] = alpha[r];
          softmax_sync<kSoftmaxThreads>();
          ok = wait_pv(g - 1, base + i - 1 + (i - 1 >= jb.q_at ? 1 : 0));   // (a first tile has no such rows)
          tc::fence_after_sync();
          const float al = sm.lse_own[head_o];
#pragma unroll 1
          for (int c = (256 / kHalves >> v_shift) * half; c < (256 / kHalves >> v_shift) * (half + 1); c += 32) {
            uint32_t o[32];
            tc::tmem_ld32(tmem_base + lane_addr + c, o);
            tc::tmem_ld_wait();
#pragma unroll
            for (int j = 0; j < 32; ++j) o[j] = __float_as_uint(__uint_as_float(o[j]) * al);
            tc::tmem_st32(tmem_base + lane_addr + c, o);
          }
          tc::tmem_st_wait();
          tc::fence_before_sync();
          need = false;
        }
        if (failed) break;
        l_run[0] += sum[0];
        l_run[1] += sum[1];
        if (tid == 0) tc::mbar_arrive(smem_u32(&sm.p_ready[g % kRing]));
      }
      if (failed) break;
      // ---- row sums and log-sum-exps of the job, for the threads that read O; the second halves' sums go to the first's warps
      have_o = jb.n_tiles > 0;
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        l_run[r] += __shfl_xor_sync(0xffffffffu, l_run[r], 1);
        l_run[r] += __shfl_xor_sync(0xffffffffu, l_run[r], 2);
        // (a job without tiles says nothing: it has no vote between its sums and the reading of the job's before)
        if (half == 1 && have_o && (lane & 3) == 0) sm.half_sum[row_s + 8 * r] = l_run[r];
      }
      auto finish_rows = [&]() {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          const int row = row_s + 8 * r;
          const float l = kHalves > 1 && have_o ? l_run[r] + sm.half_sum[row] : l_run[r];
          const float lse2 = (have_o && l > 0.f) ? m_used[r] + log2f(l) : -INFINITY;   // log2 domain
          if ((lane & 3) == 0) {
            sm.inv[n & 1][row] = (have_o && l > 0.f) ? 1.f / l : 0.f;
            sm.lse_own[row] = lse2;
            if (!clustered) {
              if (p.lse != nullptr) p.lse[static_cast<int64_t>(jb.qi) * kH + row] = lse2 / kLog2eTc;
            } else if (!pair) {
              part_lse[(((static_cast<int64_t>(jb.qi) << v_shift) + vpart) * kSplits + split) * kH + row] = lse2;
            }
          }
        }
        if constexpr (!kClustered) {
          __syncwarp();
          if (lane == 0) tc::mbar_arrive(smem_u32(&sm.o_full[n & 1]));
        }
      };
      if constexpr (kHalves == 1) finish_rows();
      if constexpr (!kClustered) ok = __all_sync(0xffffffffu, wait_job(n + 1, &jd)) && ok;
      if (!ok) sm.fail = 1;
      if (softmax_any<kSoftmaxThreads>(!ok)) break;
      if (kHalves > 1 && half == 0) finish_rows();
      if constexpr (kClustered) {
        if (have_o) have_o = wait_pv(jb.n_tiles - 1, jb.n_tiles - 1 + (jb.n_tiles - 1 >= jb.q_at ? 1 : 0));   // the last tile's
        tc::fence_after_sync();
        break;
      }
      if (lane == 0) tc::mbar_arrive(smem_u32(&sm.job_empty[n & 1]));
      base += jb.n_tiles + 1;
      tiles_done += jb.n_tiles;
      ++n;
      if (jd.x < 0) break;
      jb = job_of(jd);
    }
    if constexpr (kClustered) {
      static_assert(kHalves == 1, "a warp stages all of its lanes' columns");
      // ---- partial result of a split: normalised fp32 rows in the ring
      const int qi = blockIdx.x;
      const float inv = have_o ? sm.inv[0][head_o] : 0.f;
      uint8_t* stage = &sm.k[0][0][0];
      if (pair) cluster_arrive();   // this thread has left the tile loop, and every P V of the block has completed
      const bool foreign = pair && (quarter & 1) != split;   // a warp stages 32 heads: all of them the peer's, or none
      const uint32_t peer = static_cast<uint32_t>(split ^ 1);
      uint32_t bar_peer = 0, dst_peer = 0;
      if (foreign) {
        // into the peer's shared memory, once every thread of the peer has left its tile loop (first half of the
        // cluster barrier: its ring, which receives the rows, is then out of use)
        cluster_wait();
        bar_peer = peer_smem(smem_u32(&sm.recv_full), peer);
        dst_peer = peer_smem(smem_u32(stage + kRecvOffset + half_o * kWarpStage), peer);
      }
      uint8_t* my_warp = stage + quarter * (kWarpStage >> v_shift);
      uint8_t* dst_part = reinterpret_cast<uint8_t*>(part_out + (((static_cast<int64_t>(qi) << v_shift) + vpart) * kSplits + split) * (kH * kDV >> v_shift)) +
                          quarter * (kWarpStage >> v_shift);
#pragma unroll 1
      for (int c = 0; c < 256 >> v_shift; c += 64) {
        uint32_t o[64];
        if (have_o) {
          tc::tmem_ld64(tmem_base + lane_addr + c, o);
          tc::tmem_ld_wait();
        } else {
#pragma unroll
          for (int j = 0; j < 64; ++j) o[j] = 0u;
        }
        uint8_t* piece = my_warp + (c / 64) * 8192 + lane * 256;
#pragma unroll
        for (int j = 0; j < 16; ++j)
          *reinterpret_cast<float4*>(piece + ((j ^ (lane & 15)) << 4)) =
              make_float4(__uint_as_float(o[4 * j]) * inv, __uint_as_float(o[4 * j + 1]) * inv,
                          __uint_as_float(o[4 * j + 2]) * inv, __uint_as_float(o[4 * j + 3]) * inv);
        if (foreign || !pair) {
          tc::fence_proxy_async();
          __syncwarp();
          if (lane == 0) {
            const uint32_t src = smem_u32(my_warp + (c / 64) * 8192);
            if (pair) bulk_copy_to_peer(dst_peer + (c / 64) * 8192, src, 8192, bar_peer);
            else asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst_part + (c / 64) * 8192), "r"(src), "n"(8192) : "memory");
          }
        }
      }
      tc::fence_proxy_async();
      __syncwarp();
      if (pair) {
        if (foreign) {
          if (lane == 0 && half_o == 0)   // the log-sum-exps of the 32 heads
            bulk_copy_to_peer(peer_smem(smem_u32(sm.lse_peer), peer), smem_u32(&sm.lse_own[32 * (split ^ 1)]), (kH / 2) * 4, bar_peer);
        } else {
          cluster_wait();   // (every thread passes the first half of the barrier once)
        }
      } else {
        if (lane == 0) {   // written, not only read out of shared memory
          asm volatile("cp.async.bulk.commit_group;" ::: "memory");
          asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
          __threadfence();
        }
        __syncwarp();
      }
    }
  }
  // the threads of the other roles have left the tile loop too
  if (pair && warp >= kSoftmaxWarps) {
    __syncwarp();
    cluster_arrive();
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == kQkWarp) tc::tmem_dealloc(tmem_base, kTmemColsAttn);
  if constexpr (kClustered) {
    // ---- merge of the splits (Sec. 4.1.1: online-softmax rescaling) for this block's heads: weights
    // 2^(lse_j - max) / sum, O = sum_j w_j O_j, bf16 to global.
    const int qi = blockIdx.x;
    constexpr int n = kSplits;
    const int row0 = split * (kH / n);
    const uint8_t* stage = &sm.k[0][0][0];
    constexpr int kWarps = W::kAll;
    if constexpr (pair) {
      __nv_bfloat16* out = reinterpret_cast<__nv_bfloat16*>(p.out) + (static_cast<int64_t>(qi) * kH + row0) * kDV;
      if (warp >= kSoftmaxWarps) cluster_wait();   // (the softmax warps completed this phase before they sent)
      // the peer's rows for this block's heads, and their log-sum-exps, are in shared memory when the byte count is met
      (void)tc::mbar_wait(smem_u32(&sm.recv_full), 0, p.status);
      // Second use of the cluster barrier: a block may leave once the peer has everything it was sent (until then the
      // copies still read this block's shared memory).  A thread arrives as soon as it has seen this block's own
      // bytes complete and waits at the very end, by when the peer has normally long arrived.
      cluster_arrive();
      // A warp finishes rows w and w + 16 of this block's 32: lane k works out the k-th row's weights, and a row's parts
      // (lane l: the 16-byte chunks l, l + 32, ...) are read while the row before is written.
      constexpr int kRowsOfWarp = (kH / 2 + kWarps - 1) / kWarps;
      float4 a[2][4], b[2][4];
      auto fetch = [&](int k) {
        const int rl = min(warp + kWarps * k, kH / 2 - 1);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          // chunk lane + 32u (four dims) of the row: dims 128u .. of it are half u & 1, column steps 2 (u >> 1) and one
          // more; the warp that staged them is split + 2 * half here, and sent from half * kWarpStage there
          const int ch = (2 * (u >> 1) + (lane >> 4)) * 8192 + rl * 256 + (((lane & 15) ^ (rl & 15)) << 4);
          a[k & 1][u] = *reinterpret_cast<const float4*>(stage + (split + 2 * (u & 1)) * kWarpStage + ch);
          b[k & 1][u] = *reinterpret_cast<const float4*>(stage + kRecvOffset + (u & 1) * kWarpStage + ch);
        }
      };
      fetch(0);
      float my_own = 0.f, my_peer = 0.f;
      {
        const int rl = warp + kWarps * lane;
        if (lane < kRowsOfWarp && rl < kH / 2) {
          const int R = row0 + rl;
          const float l_own = sm.lse_own[R], l_peer = sm.lse_peer[rl];
          const float m = fmaxf(l_own, l_peer);
          my_own = m > -INFINITY ? exp2f(l_own - m) : 0.f;
          my_peer = m > -INFINITY ? exp2f(l_peer - m) : 0.f;
          const float den = my_own + my_peer;
          const float r_den = den > 0.f ? 1.f / den : 0.f;
          my_own *= r_den;
          my_peer *= r_den;
          if (p.lse != nullptr) p.lse[static_cast<int64_t>(qi) * kH + R] = den > 0.f ? (m + log2f(den)) / kLog2eTc : -INFINITY;
        }
        __syncwarp();
      }
#pragma unroll
      for (int k = 0; k < kRowsOfWarp; ++k) {
        if (k + 1 < kRowsOfWarp) fetch(k + 1);
        const float w_own = __shfl_sync(0xffffffffu, my_own, k), w_peer = __shfl_sync(0xffffffffu, my_peer, k);
        const int rl = warp + kWarps * k;
        if (rl >= kH / 2) break;   // warp-uniform
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const float4 x = a[k & 1][u], y = b[k & 1][u];
          uint2 o;
          o.x = pack_bf16(w_own * x.x + w_peer * y.x, w_own * x.y + w_peer * y.y);
          o.y = pack_bf16(w_own * x.z + w_peer * y.z, w_own * x.w + w_peer * y.w);
          *reinterpret_cast<uint2*>(out + static_cast<int64_t>(rl) * kDV + (lane + 32 * u) * 4) = o;
        }
      }
      cluster_wait();   // (see the arrival above)
    } else {
      cluster_sync_all();   // every block of the cluster has written its rows
      // A warp finishes kRuns of the four 128-dim runs of row R, from run u0 on: its loads (n parts of each run) and the log-sum-exps
      // are asked for together, one trip to L2.  (A row per warp, four parts at a time, was 4 600 cycles with 16 splits; decode
      // step of one sequence, 4 layers: 77.2 us, 74.3 so.  Runs of several rows per warp: 16 sequences 125 us, 138.)
      auto merge = [&](auto parts, auto runs, int R, int u0) {
        constexpr int N = decltype(parts)::value, kRuns = decltype(runs)::value;
        // (value dims in parts, 16 splits only: a row is 4 >> v_shift runs, and of a quarter of the dims a run's second half lies with
        // the rows that the warps of other lanes staged)
        const int vs = N == 16 ? v_shift : 0, warp_stage = kWarpStage >> vs;   // (v_shift is 0 where the kernel is not built for parts)
        const int64_t job = (static_cast<int64_t>(qi) << vs) + vpart;
        const float my_l = lane >= N ? -INFINITY : lane == split ? sm.lse_own[R] : __ldcg(part_lse + (job * N + lane) * kH + R);
        const uint8_t* src = reinterpret_cast<const uint8_t*>(part_out) + job * N * (kH * kDV * 4 >> vs) +
                             (R >> 5) * warp_stage + (lane >> 4) * (vs == 2 ? 2 * warp_stage : 8192) + (R & 31) * 256 + (((lane & 15) ^ (R & 15)) << 4);
        float4 v[kRuns][N];
#pragma unroll
        for (int i = 0; i < kRuns; ++i)
#pragma unroll
          for (int j = 0; j < N; ++j) {   // dims 128u + 4 lane .. + 3 of part j: see the pair's version
            const int u = u0 + i;
            v[i][j] = __ldcg(reinterpret_cast<const float4*>(src + j * (kH * kDV * 4 >> vs) + (u & 1) * 2 * warp_stage + (u >> 1) * 2 * 8192));
          }
        float m = my_l;
#pragma unroll
        for (int d = 1; d < N; d <<= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, d));
        float wgt = m > -INFINITY ? exp2f(my_l - m) : 0.f;
        float den = wgt;
#pragma unroll
        for (int d = 1; d < N; d <<= 1) den += __shfl_xor_sync(0xffffffffu, den, d);
        wgt = den > 0.f ? wgt / den : 0.f;
        if (p.lse != nullptr && lane == 0 && u0 == 0 && vpart == 0)
          p.lse[static_cast<int64_t>(qi) * kH + R] = den > 0.f ? (m + log2f(den)) / kLog2eTc : -INFINITY;
        float4 acc[kRuns] = {};
#pragma unroll
        for (int j = 0; j < N; ++j) {
          const float w = __shfl_sync(0xffffffffu, wgt, j);
#pragma unroll
          for (int i = 0; i < kRuns; ++i) {
            acc[i].x += w * v[i][j].x; acc[i].y += w * v[i][j].y; acc[i].z += w * v[i][j].z; acc[i].w += w * v[i][j].w;
          }
        }
#pragma unroll
        for (int i = 0; i < kRuns; ++i) {
          uint2 o;
          o.x = pack_bf16(acc[i].x, acc[i].y);
          o.y = pack_bf16(acc[i].z, acc[i].w);
          *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(p.out) + (static_cast<int64_t>(qi) * kH + R) * kDV +
                                    (lane + 32 * (vpart * (4 >> vs) + u0 + i)) * 4) = o;
        }
      };
      static_assert(kWarps >= 16, "sixteen warps have a share of a block's rows");
      if constexpr (kParts) {
        if (warp < 16 >> v_shift) merge(IntC<16>{}, IntC<1>{}, row0 + (warp >> (2 - v_shift)), warp & (3 >> v_shift));
      } else {   // a warp has 16 / n of the runs of one row
        if (warp < 16) merge(IntC<n>{}, IntC<16 / n>{}, row0 + 4 * warp / n, warp * (16 / n) & 3);
      }
    }
  }
}

}  // namespace

static_assert(sizeof(AttnTcSmem) + 1024 <= 227 * 1024, "shared memory of the attention kernel exceeds one SM");

using AttnTcKernel = void (*)(CUtensorMap, int, CUtensorMap, int, CUtensorMap, int, AttnArgs);

// The instantiation that serves a call (see the kernel's template parameters).
static AttnTcKernel pick_kernel(const AttnArgs& a) {
  if (a.rows == nullptr) return sparse_attn_tc_kernel<false, 1, false>;
  switch (a.n_split) {
    case 2: return sparse_attn_tc_kernel<true, 2, false>;
    case 4: return sparse_attn_tc_kernel<true, 4, false>;
    case 8: return sparse_attn_tc_kernel<true, 8, false>;
    case kMaxClusterSplit: return a.v_shift > 0 ? sparse_attn_tc_kernel<true, kMaxClusterSplit, true> : sparse_attn_tc_kernel<true, kMaxClusterSplit, false>;
    default: return sparse_attn_tc_kernel<true, 1, false>;
  }
}

// (Clusters that run at once: 74 of 2 blocks, 45 of 3, 33 of 4, 26 of 5, 22 of 6, 15 of 7 to 9, 7 of 11 to 16.  Five gained nothing
// over four: 24 sequences, four layers, 132 and 133 us.  Three and six, built and taken back; decode steps of four layers: sequences of
// 16K to 24K tokens gain, 16 as six 116 us instead of 126 as four, 42 as three 172 instead of 184 as two, but 44 as three are 191
// instead of 185 and 45 216, and contexts of 200 to 400 tokens 62.6 instead of 57.8 (16 as six; 61.5 with four of the six blocks at
// work) and 79 instead of 67 (40 as three: two splits exchange their rows through shared memory); the host does not know the contexts.)
cudaError_t attn_tc_resident(int n_split, int* clusters) {
  static DeviceCount n[kMaxClusterSplit + 1];
  *clusters = 0;
  const bool merged = n_split == 2 || n_split == 4 || n_split == 8 || n_split == kMaxClusterSplit;
  if (!merged) return cudaSuccess;
  return n[n_split].get(clusters, [&](int* c) {
    return resident_clusters(reinterpret_cast<const void*>(sparse_attn_tc_kernel<true, kMaxClusterSplit, false>), Warps<true>::kThreads, sizeof(AttnTcSmem) + 1024, n_split, c);
  });
}

// Row splits the tcgen05 kernel can merge inside a cluster: a power of two that divides the 64 heads, as many blocks as the
// device can co-schedule.
cudaError_t attn_tc_split_ok(int n_split, bool* ok) {
  int n = 0;
  const cudaError_t e = attn_tc_resident(n_split, &n);
  *ok = n_split == 1 || n > 0;
  return e;
}

bool attn_tc_supported(const AttnArgs& a) {
  return a.H == kH && a.DQK == kDQK && a.DV == kDV && a.v == a.k && a.ld_v == a.ld_k;
}

cudaError_t launch_attn_tc(const AttnArgs& a, cudaStream_t st, int64_t* n_launch) {
  if (a.n_query == 0) return cudaSuccess;
  const size_t smem = sizeof(AttnTcSmem) + 1024;
  if (a.n_split > 1 && a.rows == nullptr) return cudaErrorInvalidValue;   // row splits walk row lists
  if (a.v_shift != 0 && a.n_split != kMaxClusterSplit) return cudaErrorInvalidValue;   // (no other kernel knows of parts)
  AttnTcKernel kernel = pick_kernel(a);
  const int threads = a.rows == nullptr ? Warps<false>::kThreads : Warps<true>::kThreads;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
  if (e != cudaSuccess) return e;
  CUtensorMap q_map{}, k_map{}, g_map{};
  const int q_tma = (reinterpret_cast<uintptr_t>(a.q) & 15u) == 0 &&
                    make_map_bf16_tile(&q_map, a.q, kDQK, static_cast<uint64_t>(a.n_query) * kH, kH, kAtoms);
  // contiguous cache: the last query sees rows 0 .. q_pos0 + n_query - 1, so the cache holds at least that many
  const int k_tma = !a.paged && a.rows == nullptr && a.ld_k % 8 == 0 && (reinterpret_cast<uintptr_t>(a.k) & 15u) == 0 &&
                    make_map_bf16_tile(&k_map, a.k, static_cast<uint64_t>(a.ld_k), static_cast<uint64_t>(a.q_pos0 + a.n_query), kTileKeys, kAtoms);
  // gather of scattered rows by TMA: any cache whose base and row pitch TMA can address; a paged pool's row count is
  // not known here (every row number comes from the caller's list), so its map spans the whole coordinate range
  const uint64_t g_rows = a.paged || a.rows != nullptr ? 0x7fffffffull : static_cast<uint64_t>(a.q_pos0 + a.n_query);
  const int k_g4 = a.gather4 && a.ld_k % 8 == 0 && (reinterpret_cast<uintptr_t>(a.k) & 15u) == 0 &&
                   make_map_bf16_rows(&g_map, a.k, static_cast<uint64_t>(a.ld_k), g_rows, 1);
  if (a.n_split <= 1) {
    if ((e = launch_pdl(kernel, dim3(a.n_query, 1, 1), dim3(threads), smem, st, q_map, q_tma, k_map, k_tma, g_map, k_g4, a)) != cudaSuccess) return e;
  } else {
    int fit = 0;
    if ((e = attn_tc_resident(a.n_split, &fit)) != cudaSuccess) return e;
    if (fit == 0) return cudaErrorInvalidValue;
    if (a.n_split > 8 && (e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1)) != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(a.n_query, a.n_split, 1 << a.v_shift);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2]{};
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1;
    attr[0].val.clusterDim.y = static_cast<unsigned>(a.n_split);
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // see griddepcontrol.wait in the kernel
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    e = cudaLaunchKernelEx(&cfg, kernel, q_map, q_tma, k_map, k_tma, g_map, k_g4, a);
    if (e != cudaSuccess) return e;
  }
  ++*n_launch;
  return cudaGetLastError();
}

}  // namespace lsa
