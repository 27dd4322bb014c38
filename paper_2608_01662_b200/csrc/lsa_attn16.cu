// a6 for the 16-head, 128-dim shape (separate K and V rows): sparse attention (Eq. 3) without shared-memory tiles.
//
// A warp walks 16 keys at a time: S = Q K^T and O += P V as m16n8k16 MMAs (the 16 heads are the M rows) with an online
// softmax of its own, so warps never wait for one another; 8 or 4 warps share a query (every eighth or fourth tile each) and merge
// their parts once at the end, or, when there are enough queries, each has a query to itself.  (A query's result depends on that
// split as far as bf16 weights against another running maximum do: 2e-3 of its norm between a chunk and the whole run.)
//
// Cache rows go from global memory straight to MMA operands.  The sum over dims may run in any order, so a thread takes
// the 16-byte chunks that suit its loads: dims 32 j + 8 t .. + 7 (t = lane % 4) of a key are its B operands of k-steps
// 2 j and 2 j + 1, and Q is fetched in the same order.  For P V a thread holds dims 64 h + 8 (lane / 4) .. + 7 of the keys
// 2 t, 2 t + 1, 2 t + 8, 2 t + 9: dim j of two keys packed is its B operand of n-tile (h, j), whose column n then stands for
// dim 64 h + 8 n + j; a thread ends with 16 consecutive dims of its rows.
//
// What bounds it: the latency of a warp's own chain (loads, MMAs, softmax), with 8 warps on an SM at 228 registers a thread; the next
// tile's K and V are in flight while this one is worked on (64 registers).  2048 queries: 56 % of the rows come from L1, the path
// from L2 is 9 % busy, the tensor pipe 19 %, one issue slot in three is used.  The form before, one block of 8 warps per query
// around shared 64-key tiles, spent its time on four block barriers per tile: 2048 queries x 388 rows took 100 us there and 65 us
// here, 16384 queries 836 and 510 us (a limit of 168 registers, for half as many warps again, spills: 89 and 676 us).
#include "lsa_internal.h"
#include "lsa_common.cuh"

namespace lsa {

namespace {

constexpr int kH16 = 16, kD16 = 128;
constexpr int kWarps16 = 4, kManyWarps16 = 8;
constexpr int kKeys16 = 16;                  // keys of a tile
constexpr int kPitch16 = kD16 + 4;           // floats of a staged row
constexpr float kLog2e16 = 1.4426950408889634f;

template <int kWpq>
struct Attn16Smem {
  float o[kWpq][kH16][kPitch16];
  float m[kWpq][kH16], l[kWpq][kH16];
};
template <>
struct Attn16Smem<1> {};

// kWpq: warps that share a query (1, 4 or 8).  Grid: (ceil(n_query / (kWpq > 1 ? 1 : 4)), n_split).
template <int kWpq>
__global__ void __launch_bounds__(32 * (kWpq > 1 ? kWpq : kWarps16), kWpq > kWarps16 ? 1 : 2) sparse_attn16_kernel(AttnArgs p) {
  constexpr int kQueries = kWpq > 1 ? 1 : kWarps16;
  extern __shared__ __align__(16) uint8_t smem_raw[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = lane >> 2, t = lane & 3;
  // late queries attend the most rows: they go first
  const int slot = static_cast<int>(blockIdx.x) * kQueries + (kWpq > 1 ? 0 : warp), split = blockIdx.y;
  const int qi = p.n_query - 1 - slot;
  if (qi < 0) return;   // (kWpq = 1 only: whole warps, and nothing below waits for other warps then)
  const int part = kWpq > 1 ? warp : 0;

  pdl_wait();                 // the index set may come from the previous kernel of the stream
  pdl_launch_dependents();

  // ---- this query's row list: the caller's, or [window | sink | sparse] (the order within one softmax is free; the warps of
  // a block start together on neighbouring queries, whose windows are nearly the same rows: they come from L1)
  const int64_t pos = p.paged ? static_cast<int64_t>(p.ctx_len[qi]) - 1 : p.q_pos0 + qi;
  int n_sink = 0, n_win = 0, n_tot;
  int64_t win0 = 0;
  const int32_t* rows = nullptr;
  if (p.rows != nullptr) {
    rows = p.rows + static_cast<int64_t>(qi) * p.rows_ld;
    n_tot = p.n_rows[qi];
  } else {
    n_sink = static_cast<int>(min64(p.S, pos + 1));
    win0 = max64(p.S, pos - p.W + 1);
    n_win = static_cast<int>(max64(0, pos - win0 + 1));
    n_tot = n_win + n_sink + p.n_sparse[qi];
  }
  const int32_t* sp = p.sparse_idx ? p.sparse_idx + static_cast<int64_t>(qi) * p.Ksp : nullptr;
  auto row_of = [&](int i) -> int32_t {
    if (i >= n_tot) return -1;
    if (rows) return checked_row(rows[i], p.n_key, p.status);
    if (i < n_win) return static_cast<int32_t>(win0 + i);
    if (i < n_win + n_sink) return i - n_win;
    return checked_row(sp[i - n_win - n_sink], p.n_key, p.status);
  };
  const int tiles_all = (n_tot + kKeys16 - 1) / kKeys16;
  const int tiles_per = (tiles_all + p.n_split - 1) / p.n_split;
  const int tile_end = min(tiles_all, (split + 1) * tiles_per);
  auto tile_rows = [&](int tile) -> int32_t {   // lanes 0-15: the cache row of the tile's key `lane`
    return (tile < tile_end && lane < kKeys16) ? row_of(tile * kKeys16 + lane) : -1;
  };

  // ---- Q as A operands: rows (heads) g and g + 8, chunks 4 j + t
  uint32_t qa[8][4];
  {
    const uint8_t* q0 = reinterpret_cast<const uint8_t*>(p.q) + (static_cast<int64_t>(qi) * kH16 + g) * kD16 * 2 + t * 16;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const uint4 a = *reinterpret_cast<const uint4*>(q0 + j * 64), b = *reinterpret_cast<const uint4*>(q0 + 8 * kD16 * 2 + j * 64);
      qa[2 * j][0] = a.x; qa[2 * j][1] = b.x; qa[2 * j][2] = a.y; qa[2 * j][3] = b.y;
      qa[2 * j + 1][0] = a.z; qa[2 * j + 1][1] = b.z; qa[2 * j + 1][2] = a.w; qa[2 * j + 1][3] = b.w;
    }
  }
  uint4 kf[2][4], vf[4][2];
  const uint8_t* kg = reinterpret_cast<const uint8_t*>(p.k) + t * 16;
  const uint8_t* vg = reinterpret_cast<const uint8_t*>(p.v) + g * 16;
  auto load_k = [&](int32_t row) {
#pragma unroll
    for (int nt = 0; nt < 2; ++nt) {
      const int32_t r = max(__shfl_sync(0xffffffffu, row, 8 * nt + g), 0);   // an absent key's score is masked: any row will do
      const uint8_t* src = kg + static_cast<int64_t>(r) * p.ld_k * 2;
#pragma unroll
      for (int j = 0; j < 4; ++j) kf[nt][j] = *reinterpret_cast<const uint4*>(src + j * 64);
    }
  };
  auto load_v = [&](int32_t row) {
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      // An absent key's values are zero, not some other row's: its weight is 0, but 0 x NaN is not (in a pool, row 0 may be
      // another sequence's, or nobody's).
      const int32_t r = __shfl_sync(0xffffffffu, row, 2 * t + (s & 1) + 8 * (s >> 1));
      const uint8_t* src = vg + static_cast<int64_t>(r) * p.ld_v * 2;
      vf[s][0] = r >= 0 ? *reinterpret_cast<const uint4*>(src) : make_uint4(0u, 0u, 0u, 0u);
      vf[s][1] = r >= 0 ? *reinterpret_cast<const uint4*>(src + 128) : make_uint4(0u, 0u, 0u, 0u);
    }
  };

  float o[16][4];
#pragma unroll
  for (int i = 0; i < 16; ++i) o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f;
  float m_run[2] = {-INFINITY, -INFINITY}, l_run[2] = {0.f, 0.f};   // rows g and g + 8; l_run is this thread's share
  const float zs = p.sm_scale * kLog2e16;
  int tile = split * tiles_per + part;
  int32_t row_cur = tile_rows(tile), row_next = tile_rows(tile + kWpq);
  if (tile < tile_end) {
    load_k(row_cur);
    load_v(row_cur);
  }
  for (; tile < tile_end; tile += kWpq) {
    const bool more = tile + kWpq < tile_end;
    float s[2][4];
#pragma unroll
    for (int nt = 0; nt < 2; ++nt) {
      s[nt][0] = s[nt][1] = s[nt][2] = s[nt][3] = 0.f;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        mma_bf16(s[nt], qa[2 * j], kf[nt][j].x, kf[nt][j].y);
        mma_bf16(s[nt], qa[2 * j + 1], kf[nt][j].z, kf[nt][j].w);
      }
    }
    if (more) load_k(row_next);
    const unsigned live = __ballot_sync(0xffffffffu, row_cur >= 0);
    float mx[2] = {m_run[0], m_run[1]};
#pragma unroll
    for (int nt = 0; nt < 2; ++nt)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        s[nt][j] = (live >> (8 * nt + 2 * t + (j & 1))) & 1u ? s[nt][j] * zs : -INFINITY;
        mx[j >> 1] = fmaxf(mx[j >> 1], s[nt][j]);
      }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      mx[r] = fmaxf(mx[r], __shfl_xor_sync(0xffffffffu, mx[r], 1));
      mx[r] = fmaxf(mx[r], __shfl_xor_sync(0xffffffffu, mx[r], 2));
    }
    if (__any_sync(0xffffffffu, mx[0] > m_run[0] || mx[1] > m_run[1])) {
      const float a0 = m_run[0] > -INFINITY ? exp2f(m_run[0] - mx[0]) : 0.f, a1 = m_run[1] > -INFINITY ? exp2f(m_run[1] - mx[1]) : 0.f;
      m_run[0] = mx[0];
      m_run[1] = mx[1];
      l_run[0] *= a0;
      l_run[1] *= a1;
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        o[i][0] *= a0; o[i][1] *= a0;
        o[i][2] *= a1; o[i][3] *= a1;
      }
    }
    uint32_t pa[4];
#pragma unroll
    for (int nt = 0; nt < 2; ++nt) {
      // (absent keys by their bits, not by the maximum: a head whose scores are all NaN has none, and its weights are NaN)
      const unsigned there = live >> (8 * nt + 2 * t);
      const float p0 = there & 1u ? exp2f(s[nt][0] - m_run[0]) : 0.f, p1 = there & 2u ? exp2f(s[nt][1] - m_run[0]) : 0.f;
      const float p2 = there & 1u ? exp2f(s[nt][2] - m_run[1]) : 0.f, p3 = there & 2u ? exp2f(s[nt][3] - m_run[1]) : 0.f;
      l_run[0] += p0 + p1;   // fp32 sums of the unrounded weights
      l_run[1] += p2 + p3;
      pa[2 * nt] = pack_bf16(p0, p1);
      pa[2 * nt + 1] = pack_bf16(p2, p3);
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const uint32_t v0[4] = {vf[0][h].x, vf[0][h].y, vf[0][h].z, vf[0][h].w}, v1[4] = {vf[1][h].x, vf[1][h].y, vf[1][h].z, vf[1][h].w};
      const uint32_t v2[4] = {vf[2][h].x, vf[2][h].y, vf[2][h].z, vf[2][h].w}, v3[4] = {vf[3][h].x, vf[3][h].y, vf[3][h].z, vf[3][h].w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        mma_bf16(o[8 * h + 2 * i], pa, __byte_perm(v0[i], v1[i], 0x5410), __byte_perm(v2[i], v3[i], 0x5410));
        mma_bf16(o[8 * h + 2 * i + 1], pa, __byte_perm(v0[i], v1[i], 0x7632), __byte_perm(v2[i], v3[i], 0x7632));
      }
    }
    if (more) load_v(row_next);
    row_cur = row_next;
    row_next = tile_rows(tile + 2 * kWpq);
  }
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    l_run[r] += __shfl_xor_sync(0xffffffffu, l_run[r], 1);
    l_run[r] += __shfl_xor_sync(0xffffffffu, l_run[r], 2);
  }

  // ---- results: kDims consecutive dims of a head, or of a part that launch_merge puts together (normalised fp32, log2 lse)
  constexpr int kDims = kWpq > 1 ? kH16 * kD16 / (32 * kWpq) : 16;
  auto finish = [&](int head, int dim, const float (&x)[kDims], float inv, float lse2, bool writes_lse) {
    if (p.n_split == 1) {
      uint4* dst = reinterpret_cast<uint4*>(reinterpret_cast<__nv_bfloat16*>(p.out) + (static_cast<int64_t>(qi) * kH16 + head) * kD16 + dim);
#pragma unroll
      for (int i = 0; i < kDims; i += 8)
        dst[i / 8] = make_uint4(pack_bf16(x[i] * inv, x[i + 1] * inv), pack_bf16(x[i + 2] * inv, x[i + 3] * inv),
                                pack_bf16(x[i + 4] * inv, x[i + 5] * inv), pack_bf16(x[i + 6] * inv, x[i + 7] * inv));
      if (writes_lse && p.lse != nullptr) p.lse[static_cast<int64_t>(qi) * kH16 + head] = lse2 / kLog2e16;
    } else {
      const int64_t row = (static_cast<int64_t>(qi) * p.n_split + split) * kH16 + head;
      float4* dst = reinterpret_cast<float4*>(p.part_out + row * kD16 + dim);
#pragma unroll
      for (int i = 0; i < kDims / 4; ++i) dst[i] = make_float4(x[4 * i] * inv, x[4 * i + 1] * inv, x[4 * i + 2] * inv, x[4 * i + 3] * inv);
      if (writes_lse) p.part_lse[row] = lse2;
    }
  };
  if constexpr (kWpq == 1) {
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const float inv = l_run[r] > 0.f ? 1.f / l_run[r] : 0.f;
      const float lse2 = l_run[r] != 0.f ? m_run[r] + log2f(l_run[r]) : -INFINITY;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float x[16];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          x[j] = o[8 * h + j][2 * r];
          x[8 + j] = o[8 * h + j][2 * r + 1];
        }
        finish(g + 8 * r, 64 * h + 16 * t, x, inv, lse2, h == 0 && t == 0);
      }
    }
  } else {
    auto& sm = *reinterpret_cast<Attn16Smem<kWpq>*>(smem_raw);
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int head = g + 8 * r;
      if (t == 0) {
        sm.m[warp][head] = m_run[r];
        sm.l[warp][head] = l_run[r];
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float4* dst = reinterpret_cast<float4*>(&sm.o[warp][head][64 * h + 16 * t]);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int j = (4 * i) & 7, c = 2 * r + (i >> 1);
          dst[i] = make_float4(o[8 * h + j][c], o[8 * h + j + 1][c], o[8 * h + j + 2][c], o[8 * h + j + 3][c]);
        }
      }
    }
    __syncthreads();
    constexpr int kPerHead = kD16 / kDims;   // threads
    const int head = tid / kPerHead, dim = (tid % kPerHead) * kDims;
    float m = -INFINITY, den = 0.f, x[kDims];
#pragma unroll
    for (int i = 0; i < kDims; ++i) x[i] = 0.f;
#pragma unroll
    for (int w = 0; w < kWpq; ++w) m = fmaxf(m, sm.m[w][head]);
#pragma unroll
    for (int w = 0; w < kWpq; ++w) {
      const float wgt = sm.m[w][head] > -INFINITY ? exp2f(sm.m[w][head] - m) : 0.f;   // (a warp without a tile)
      den += wgt * sm.l[w][head];
      const float4* src = reinterpret_cast<const float4*>(&sm.o[w][head][dim]);
#pragma unroll
      for (int i = 0; i < kDims / 4; ++i) {
        const float4 v = src[i];
        x[4 * i] += wgt * v.x; x[4 * i + 1] += wgt * v.y; x[4 * i + 2] += wgt * v.z; x[4 * i + 3] += wgt * v.w;
      }
    }
    finish(head, dim, x, den > 0.f ? 1.f / den : 0.f, den != 0.f ? m + log2f(den) : -INFINITY, tid % kPerHead == 0);
  }
}

template <int kWpq>
cudaError_t launch_t(const AttnArgs& a, cudaStream_t st) {
  const size_t smem = kWpq > 1 ? sizeof(Attn16Smem<kWpq>) : 0;
  if (smem > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(sparse_attn16_kernel<kWpq>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (e != cudaSuccess) return e;
  }
  const int queries = kWpq > 1 ? 1 : kWarps16, warps = kWpq > 1 ? kWpq : kWarps16;
  return launch_pdl(sparse_attn16_kernel<kWpq>, dim3((a.n_query + queries - 1) / queries, a.n_split), dim3(32 * warps), smem, st, a);
}

}  // namespace

// Warps per query: eight while every query (times row splits) has an SM to itself; one from the count on where four would take a
// third wave of two blocks per SM, a fourth where there are more rows.  (us with a cold L2, one / four / eight warps: 388 rows, 148
// queries 43/21/16, 296 43/21/25, 592 41/35/43, 700 43/47/50, 2048 78/100/127; 1540 rows, 148 queries 123/49/31, 592 121/90/96, 800
// 127/123/135, 1000 131/158/158, 2048 242/277/303.)
cudaError_t launch_attn16(const AttnArgs& a, cudaStream_t st, int64_t* n_launch) {
  if (a.n_query == 0) return cudaSuccess;
  const int64_t jobs = static_cast<int64_t>(a.n_query) * a.n_split, sms = a.sm_count > 0 ? a.sm_count : 148;
  const int rows = a.rows_ld / a.n_split;
  const cudaError_t e = jobs <= sms ? launch_t<kManyWarps16>(a, st) : jobs <= (rows <= 1024 ? 4 : 6) * sms ? launch_t<kWarps16>(a, st) : launch_t<1>(a, st);
  ++*n_launch;
  return e;
}

}  // namespace lsa
