// Internal helpers shared by the CUDA-core and tensor-core attention kernels:
// launch parameters, bf16 output rows, log-sum-exp outputs, and the merge of
// split-KV partials (each split keeps an unnormalised fp32 output, its running
// base-2 max m and its sum l; the merge rescales by 2^{m_s - max m}).
#pragma once

#include <cuda.h>  // CUtensorMap
#include <cuda_bf16.h>

#include <cmath>

#include "common.cuh"

namespace specv {

struct AttnParams {
  int batch, gamma, hq, hkv, group, rows, row_tiles, rows_per_cta;
  int hunits;        // KV-head units per sequence: Hkv over the adjacent KV heads that one
                     // block serves together
  int page_size, max_pages, num_pages;
  int nsplit, tiles_per_split;
  int slot_rows;     // rows stored per partial slot
  int max_keys;      // max_pages * page_size
  float scale_log2;  // softmax_scale * log2(e)
  const void* q;
  const void* k_cache;
  const void* v_cache;
  const int32_t* page_table;
  const int32_t* kv_len;
  void* out;
  float* lse;
  uint32_t* status;
  uint32_t* tickets;
  SplitUnit* splits;   // [grid]
  float* partial_o;    // [slot][slot_rows][D]
  float2* partial_ml;  // [slot][slot_rows] = (m, l); l = -1 marks a bad sequence
  int q_tma;           // tensor-core kernel: Q tiles arrive by TMA (else softmax warps load them)
  int unit_overhead;   // tensor-core kernel: tiles charged per unit start in the work list
  const uint64_t* tree_mask;  // [batch][gamma] block keys each query sees, or NULL (causal)
  int grid, min_tiles; // range_count: blocks launched, tiles a block takes at least
  int unit_heads;      // KV heads of a unit (attn_merge_kernel)
  int whole_units;     // ranges end at unit ends: nothing to merge (block_range)
  float rise, fall;    // tensor cores: the running maximum (base 2) that probabilities are taken
                       // against is raised past m + rise, and falls by at most `fall` a tile
  int starve;  // test hook: the producers issue no copies, so the consumers' waits run out
};

inline AttnParams make_attn_params(const spec_attn_args_t& a, const AttnPlan& P, char* ws) {
  AttnParams p;
  p.batch = a.batch;
  p.gamma = a.gamma;
  p.hq = a.num_q_heads;
  p.hkv = a.num_kv_heads;
  p.hunits = P.heads > 0 ? a.num_kv_heads / P.heads : P.head_pair ? a.num_kv_heads / 2 : a.num_kv_heads;
  p.group = a.num_q_heads / a.num_kv_heads;
  p.rows = P.rows;
  p.row_tiles = P.row_tiles;
  p.rows_per_cta = P.rows_per_cta;
  p.page_size = a.page_size;
  p.max_pages = a.max_pages_per_seq;
  p.num_pages = a.num_pages;
  p.nsplit = P.nsplit;
  p.tiles_per_split = P.tiles_per_split;
  p.slot_rows = P.slot_rows;
  p.max_keys = P.max_keys;
  const float scale = a.softmax_scale != 0.f ? a.softmax_scale : 1.f / sqrtf(static_cast<float>(a.head_dim));
  p.scale_log2 = scale * 1.4426950408889634f;
  p.q = a.q;
  p.k_cache = a.k_cache;
  p.v_cache = a.v_cache;
  p.page_table = a.page_table;
  p.kv_len = a.kv_len;
  p.out = a.out;
  p.lse = a.lse;
  p.status = reinterpret_cast<uint32_t*>(ws);
  p.tickets = reinterpret_cast<uint32_t*>(ws + P.tickets);
  p.splits = reinterpret_cast<SplitUnit*>(ws + P.splits);
  p.partial_o = reinterpret_cast<float*>(ws + P.partial_o);
  p.partial_ml = reinterpret_cast<float2*>(ws + P.partial_ml);
  p.q_tma = 0;
  p.unit_overhead = 0;
  p.tree_mask = a.tree_mask;
  p.starve = 0;
  p.grid = P.grid;
  p.min_tiles = 1;
  p.unit_heads = 1;
  p.whole_units = 0;
  p.rise = p.fall = 0.f;
  return p;
}

// Tensor maps of the tensor-core kernels (attn_tc.cu): the K or V cache with one page of
// one KV head (or of two adjacent KV heads, heads_per_box = 2) per box, and Q with one
// tile of tile_rows query rows of one KV group per box (false if group does not divide
// tile_rows or the encoder is missing).
bool encode_cache_map(CUtensorMap* map, const void* base, const spec_attn_args_t& a,
                      int heads_per_box = 1);
bool encode_q_map(CUtensorMap* map, const spec_attn_args_t& a, int tile_rows);

#ifdef __CUDACC__
// ---------------------------------------------------------------------------------
// Work list of the persistent tensor-core kernels (TK keys per tile)
// ---------------------------------------------------------------------------------
template <int TK>
__device__ __forceinline__ int unit_tiles(int kv_len, const AttnParams& p) {
  const bool ok = kv_len >= p.gamma && kv_len <= p.max_keys;
  return ok ? (kv_len + TK - 1) / TK : 1;  // a malformed sequence keeps one tile to report it
}

// The work list is virtual: each unit is ovh overhead tiles followed by its real tiles,
// and a block owns an equal range of virtual tiles. A segment is the part of one unit
// inside a block's range. Only a range that ends inside a unit's overhead has a segment
// with no real tile, and then it is the range's last (a first segment without real
// tiles means the block has no work).
struct Seg {
  int b, g, rt;      // sequence, KV head (or head pair), row tile
  int64_t u;         // unit index (b * hunits + g) * row_tiles + rt
  int tile0, ntile;  // first real tile within the unit and real tile count of this segment
  int unit_tiles;    // real tiles of the whole unit
  int kv_len;
  bool len_ok;
  int64_t unit_start;  // virtual index of the unit's first real tile
  int64_t vnext;       // virtual index just past this segment
};

template <int TK>
__device__ __forceinline__ Seg locate(int64_t v, int64_t v1, const AttnParams& p,
                                      const int* pb, int ovh) {
  int lo = 0, hi = p.batch;  // largest b with pb[b] <= v
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (pb[mid] <= v) lo = mid; else hi = mid;
  }
  Seg s;
  s.b = lo;
  s.kv_len = p.kv_len[lo];
  s.len_ok = s.kv_len >= p.gamma && s.kv_len <= p.max_keys;
  s.unit_tiles = unit_tiles<TK>(s.kv_len, p);
  const int vlen = s.unit_tiles + ovh;
  // the prefix sums are 32-bit, so offsets within them are: a 64-bit division is a call of a
  // hundred instructions, and every role starts with this function
  const uint32_t rem = static_cast<uint32_t>(v - pb[lo]);
  const uint32_t ub = rem / static_cast<uint32_t>(vlen);
  const int64_t vstart = v - (rem - ub * static_cast<uint32_t>(vlen));  // the unit's first (overhead) virtual tile
  s.g = p.row_tiles == 1 ? ub : ub / static_cast<uint32_t>(p.row_tiles);
  s.rt = p.row_tiles == 1 ? 0 : ub % static_cast<uint32_t>(p.row_tiles);
  s.u = static_cast<int64_t>(lo) * p.hunits * p.row_tiles + ub;
  s.unit_start = vstart + ovh;
  const int64_t vend = vstart + vlen;
  s.vnext = vend < v1 ? vend : v1;
  const int64_t lo_real = v > s.unit_start ? v : s.unit_start;
  s.ntile = s.vnext > lo_real ? static_cast<int>(s.vnext - lo_real) : 0;
  s.tile0 = s.ntile > 0 ? static_cast<int>(lo_real - s.unit_start) : 0;
  return s;
}

// Whether real tiles follow segment s in the range ending at v1. A segment ends at its
// unit's end or at v1, so the next one starts a unit, whose real tiles begin ovh virtual
// tiles later; no load is needed.
__device__ __forceinline__ bool has_more(const Seg& s, int64_t v1, int ovh) {
  return v1 - s.vnext > ovh;
}

// x / y of non-negative x and positive y, in 32 bits where they fit.
__device__ __forceinline__ int div_small(int64_t x, int64_t y) {
  if (((x | y) >> 32) == 0) return static_cast<int>(static_cast<uint32_t>(x) / static_cast<uint32_t>(y));
  return static_cast<int>(x / y);
}

// Block that owns virtual tile t when `total` virtual tiles are cut into `ctas` ranges
// [c * total / ctas, (c + 1) * total / ctas).
__device__ __forceinline__ int owner_of(int64_t t, int64_t total, int ctas) {
  return div_small((t + 1) * ctas - 1, total);
}

// 8 consecutive output dims of unit row `row` (row = j * group + head-in-group).
template <int D>
__device__ __forceinline__ void write_out_row(const AttnParams& p, int b, int g, int row, int d0,
                                              const float* o8, float inv) {
  const int j = row / p.group, h = g * p.group + row % p.group;
  __nv_bfloat16* dst = static_cast<__nv_bfloat16*>(p.out) +
                       ((static_cast<int64_t>(b) * p.gamma + j) * p.hq + h) * D + d0;
  uint32_t w[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const __nv_bfloat162 pr = __floats2bfloat162_rn(o8[2 * e] * inv, o8[2 * e + 1] * inv);
    w[e] = *reinterpret_cast<const uint32_t*>(&pr);
  }
  *reinterpret_cast<uint4*>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
}

__device__ __forceinline__ void write_lse(const AttnParams& p, int b, int g, int row, float m,
                                          float l, bool bad) {
  if (!p.lse) return;
  const int j = row / p.group, h = g * p.group + row % p.group;
  const float v = (bad || !(l > 0.f)) ? -INFINITY : (m + log2f(l)) * 0.6931471805599453f;
  p.lse[(static_cast<int64_t>(b) * p.gamma + j) * p.hq + h] = v;
}

// Combines the split-KV partials of one unit, held in slots [slot0, slot0 + nslots), for
// rows [row0, row0 + nrows) and writes the final outputs (nthreads threads from tid
// cooperate; no block synchronization). A thread takes its (row, 8-column) items one at a
// time and walks their slots in batches of four: a batch's (m, l) pairs and output pieces
// are loaded together, then folded into the item's running base-2 max.
template <int D>
__device__ void merge_unit(const AttnParams& p, int b, int g, int row0, int nrows, int64_t slot0,
                           int nslots, int tid, int nthreads) {
  constexpr int C8 = D / 8, SB = 4;
  for (int idx = tid; idx < nrows * C8; idx += nthreads) {
    const int r = idx / C8, c8 = idx % C8;
    float M = -INFINITY, L = 0.f, acc[8];
    bool bad = false;
#pragma unroll
    for (int e = 0; e < 8; ++e) acc[e] = 0.f;
    for (int s0 = 0; s0 < nslots; s0 += SB) {
      float2 ml[SB];
      float4 lo[SB], hi[SB];
#pragma unroll
      for (int e = 0; e < SB; ++e) {
        ml[e] = make_float2(-INFINITY, 0.f);
        lo[e] = hi[e] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (s0 + e < nslots) {
          const int64_t slot = (slot0 + s0 + e) * p.slot_rows + r;
          ml[e] = __ldcg(&p.partial_ml[slot]);
          const float4* src = reinterpret_cast<const float4*>(p.partial_o + slot * D) + 2 * c8;
          lo[e] = __ldcg(src);
          hi[e] = __ldcg(src + 1);
        }
      }
      float mb = M;
#pragma unroll
      for (int e = 0; e < SB; ++e) {
        bad |= ml[e].y < 0.f;
        if (ml[e].y > 0.f) mb = fmaxf(mb, ml[e].x);
      }
      if (mb == -INFINITY) continue;
      const float scale = M == -INFINITY ? 0.f : ex2(M - mb);
      L *= scale;
#pragma unroll
      for (int e = 0; e < 8; ++e) acc[e] *= scale;
#pragma unroll
      for (int e = 0; e < SB; ++e) {
        if (!(ml[e].y > 0.f)) continue;
        const float w = ex2(ml[e].x - mb);
        const float4 a = lo[e], c = hi[e];
        L += ml[e].y * w;
        acc[0] += a.x * w; acc[1] += a.y * w; acc[2] += a.z * w; acc[3] += a.w * w;
        acc[4] += c.x * w; acc[5] += c.y * w; acc[6] += c.z * w; acc[7] += c.w * w;
      }
      M = mb;
    }
    const bool dead = bad || !(L > 0.f);
    write_out_row<D>(p, b, g, row0 + r, c8 * 8, acc, dead ? 0.f : 1.f / L);
    if (c8 == 0) write_lse(p, b, g, row0 + r, M, L, dead);
  }
}

// ---------------------------------------------------------------------------------
// Merging split units in a kernel of their own
// ---------------------------------------------------------------------------------
// pb[b] = virtual tiles of the sequences before b (one warp, four sequences a lane and round:
// each round's loads are one trip to memory).
template <int TK>
__device__ __forceinline__ void tile_prefix(const AttnParams& p, int* pb, int lane) {
  const int per_b = p.hunits * p.row_tiles;
  int carry = 0;
  for (int b0 = 0; b0 < p.batch; b0 += 128) {
    int v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int b = b0 + 4 * lane + i;
      v[i] = b < p.batch ? p.kv_len[b] : 0;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
      v[i] = (b0 + 4 * lane + i < p.batch ? (unit_tiles<TK>(v[i], p) + p.unit_overhead) * per_b : 0) + (i > 0 ? v[i - 1] : 0);
    int sum = v[3];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, sum, o);
      if (lane >= o) sum += y;
    }
    const int before = carry + sum - v[3];
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (b0 + 4 * lane + i < p.batch) pb[b0 + 4 * lane + i + 1] = before + v[i];
    carry += __shfl_sync(0xffffffffu, sum, 31);
  }
  if (lane == 0) pb[0] = 0;
}

// Ranges the virtual tiles are cut into: one per block, of at least min_tiles tiles each
// (below that a block's start, partial and merge cost more than the tiles it takes off the
// others). Every SM gets a range: with the merges in a kernel of their own, 32 equal units
// over all 152 blocks take less time than over 128 blocks of a quarter unit each (4 sequences
// of 32,768 keys, 256 rows per KV head: 161 us against 182).
__device__ __forceinline__ int range_count(int64_t total, const AttnParams& p) {
  const int64_t want = div_small(total + p.min_tiles - 1, p.min_tiles);
  return want < p.grid ? static_cast<int>(want) : p.grid;
}

// Block cta's range [t0, t1) of the virtual tiles (empty past the last range). Equal ranges,
// or with whole_units equal numbers of units: where no unit can be
// longer than kWholeTiles, one block's turn at a unit costs less than the merge kernel behind
// the call (10 requests of 216 keys: 15.5 us split, 12.3 whole; 128 of up to 100: 38 and 18.6).
__device__ __forceinline__ void block_range(const AttnParams& p, const int* pb, int cta, int64_t total, int ctas,
                                            int64_t& t0, int64_t& t1) {
  t0 = t1 = 0;
  if (!p.whole_units) {
    if (cta < ctas) {
      t0 = div_small(static_cast<int64_t>(cta) * total, ctas);
      t1 = div_small(static_cast<int64_t>(cta + 1) * total, ctas);
    }
    return;
  }
  // Every role waits for this function, and a division is a chain of about 40 instructions: with
  // a unit per block at most, two of them (six, as below: 64 units of one tile and 64 rows took
  // 11.3 us instead of 10.3).
  const uint32_t per_b = p.hunits * p.row_tiles;
  const int64_t units = static_cast<int64_t>(p.batch) * per_b;
  if (units <= p.grid) {
    if (cta < units) {
      const uint32_t b = static_cast<uint32_t>(cta) / per_b;
      const uint32_t len = static_cast<uint32_t>(pb[b + 1] - pb[b]) / per_b;
      t0 = pb[b] + (static_cast<uint32_t>(cta) - b * per_b) * len;
      t1 = t0 + len;
    }
    return;
  }
  auto start = [&](int64_t u) -> int64_t {
    if (u >= units) return total;
    const int b = div_small(u, per_b);
    return pb[b] + (static_cast<int>(u) - b * static_cast<int>(per_b)) * ((pb[b + 1] - pb[b]) / static_cast<int>(per_b));
  };
  if (cta < p.grid) {
    t0 = start(div_small(cta * units, p.grid));
    t1 = start(div_small((cta + 1) * units, p.grid));
  }
}
constexpr int kWholeTiles = 8;

// What the merge kernel reads of block cta's left boundary, s its first segment (one thread).
__device__ __forceinline__ void note_split(const AttnParams& p, int cta, const Seg& s, int64_t total, int ctas) {
  SplitUnit d = {};
  if (s.ntile > 0 && s.tile0 > 0) {
    const int c_first = owner_of(s.unit_start, total, ctas);
    d.b = s.b;
    d.g = s.g;
    d.rt = s.rt;
    d.slot0 = static_cast<int>(s.u) + c_first;
    d.nsl = owner_of(s.unit_start + s.unit_tiles - 1, total, ctas) - c_first + 1;
    d.k = cta - c_first - 1;
  }
  p.splits[cta] = d;
}

// A block whose waits ran out leaves units without their partials: rows first, first + step, ..
// below end are marked bad in the slots of its first and last units (no other can be split), as
// a malformed sequence's are, so that those units' outputs become zeros instead of what an
// earlier call left in the slots. (The range is worked out again, so that the roles need not
// keep it.)
template <int TK>
__device__ __forceinline__ void drop_partials(const AttnParams& p, const int* pb, int first, int end, int step) {
  const int64_t total = pb[p.batch];
  int64_t t0, t1;
  block_range(p, pb, blockIdx.x, total, range_count(total, p), t0, t1);
  if (t1 <= t0) return;
#pragma unroll 1
  for (int i = 0; i < 2; ++i) {
    const int64_t slot = locate<TK>(i == 0 ? t0 : t1 - 1, t1, p, pb, p.unit_overhead).u + blockIdx.x;
#pragma unroll 1
    for (int r = first; r < end; r += step) p.partial_ml[slot * p.slot_rows + r] = make_float2(-INFINITY, -1.f);
  }
}
// The same as a call: a consumer thread of the small-group kernel marks its own rows. Inlined,
// behind a barrier at the block's end, a fused step of 8 requests of 8 positions took 48.3 us,
// with the call 47.6 (47.4 without any of this; the block's idle warps make room for the
// acceptance as they end).
template <int TK>
static __device__ __noinline__ void drop_partials_call(const AttnParams& p, const int* pb, int first, int end, int step) {
  drop_partials<TK>(p, pb, first, end, step);
}

// RW rows of one warp from their partial slots [slot0, slot0 + nsl), SB slots at a time: the
// loads of all those rows and slots are in flight together.
template <int D, int RW, int SB>
__device__ __forceinline__ void merge_rows(const AttnParams& p, const SplitUnit& u, int r0, int r_end,
                                           int head_rows, int lane) {
  constexpr int E = D / 32;  // output columns per lane
  float M[RW], L[RW], acc[RW][E];
  bool bad[RW];
#pragma unroll
  for (int t = 0; t < RW; ++t) {
    M[t] = -INFINITY;
    L[t] = 0.f;
    bad[t] = false;
#pragma unroll
    for (int e = 0; e < E; ++e) acc[t][e] = 0.f;
  }
  for (int s0 = 0; s0 < u.nsl; s0 += SB) {
    float2 ml[RW][SB];
    float o[RW][SB][E];
#pragma unroll
    for (int t = 0; t < RW; ++t)
#pragma unroll
      for (int i = 0; i < SB; ++i) {
        ml[t][i] = make_float2(-INFINITY, 0.f);
#pragma unroll
        for (int e = 0; e < E; ++e) o[t][i][e] = 0.f;
        if (r0 + t < r_end && s0 + i < u.nsl) {
          const int64_t row = static_cast<int64_t>(u.slot0 + s0 + i) * p.slot_rows + r0 + t;
          ml[t][i] = __ldcg(&p.partial_ml[row]);
          if constexpr (E == 4) {
            const float4 v = __ldcg(reinterpret_cast<const float4*>(p.partial_o + row * D) + lane);
            o[t][i][0] = v.x; o[t][i][1] = v.y; o[t][i][2] = v.z; o[t][i][3] = v.w;
          } else {
            const float2 v = __ldcg(reinterpret_cast<const float2*>(p.partial_o + row * D) + lane);
            o[t][i][0] = v.x; o[t][i][1] = v.y;
          }
        }
      }
#pragma unroll
    for (int t = 0; t < RW; ++t) {
      float mb = M[t];
#pragma unroll
      for (int i = 0; i < SB; ++i) {
        bad[t] |= ml[t][i].y < 0.f;
        if (ml[t][i].y > 0.f) mb = fmaxf(mb, ml[t][i].x);
      }
      if (mb == -INFINITY) continue;
      const float scale = M[t] == -INFINITY ? 0.f : ex2(M[t] - mb);
      L[t] *= scale;
#pragma unroll
      for (int e = 0; e < E; ++e) acc[t][e] *= scale;
#pragma unroll
      for (int i = 0; i < SB; ++i) {
        if (!(ml[t][i].y > 0.f)) continue;
        const float w = ex2(ml[t][i].x - mb);
        L[t] += ml[t][i].y * w;
#pragma unroll
        for (int e = 0; e < E; ++e) acc[t][e] += o[t][i][e] * w;
      }
      M[t] = mb;
    }
  }
#pragma unroll
  for (int t = 0; t < RW; ++t) {
    const int r = r0 + t;
    if (r >= r_end) break;
    const bool dead = bad[t] || !(L[t] > 0.f);
    const float inv = dead ? 0.f : 1.f / L[t];
    const int kvh = u.g * p.unit_heads + r / head_rows, row = u.rt * p.rows_per_cta + r % head_rows;
    const int j = row / p.group, h = kvh * p.group + row % p.group;
    uint32_t w[E / 2];
#pragma unroll
    for (int e = 0; e < E / 2; ++e) {
      const __nv_bfloat162 v = __floats2bfloat162_rn(dead ? 0.f : acc[t][2 * e] * inv, dead ? 0.f : acc[t][2 * e + 1] * inv);
      w[e] = *reinterpret_cast<const uint32_t*>(&v);
    }
    __nv_bfloat16* dst = static_cast<__nv_bfloat16*>(p.out) +
                         ((static_cast<int64_t>(u.b) * p.gamma + j) * p.hq + h) * D + lane * E;
    if constexpr (E == 4) *reinterpret_cast<uint2*>(dst) = make_uint2(w[0], w[1]);
    else *reinterpret_cast<uint32_t*>(dst) = w[0];
    if (lane == 0) write_lse(p, u.b, kvh, row, M[t], L[t], dead);
  }
}

// The outputs of the units that were split between blocks, from their partial slots. Block
// (c, y) stands for the boundary before range c + 1: the k-th boundary inside a unit merges
// the k-th share of the unit's rows (of gridDim.y pieces, piece y), so that every boundary
// reads about one slot however many ways a unit was split (the blocks leave the boundaries'
// descriptions behind; finding them from the lengths again was 1 us slower). Merging in the last block of a
// unit to finish instead (atomic ticket) left most SMs idle while a few read every slot:
// 3 us for the fence and the ticket and 7 to 15 us for the merge (one request of 128 rows per
// KV head and 4,096 keys: 46.7 us, here 18.6; 8 requests of 32 rows: 53, here 38; 64 ragged
// requests of 64 rows: 124.0, here 118.2).
constexpr int kAttnMergeThreads = 256;
template <int D>
__global__ void __launch_bounds__(kAttnMergeThreads) attn_merge_kernel(AttnParams p) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  pdl_wait_prior();
  const int4 lo = __ldcg(reinterpret_cast<const int4*>(p.splits + blockIdx.x + 1));
  const int4 hi = __ldcg(reinterpret_cast<const int4*>(p.splits + blockIdx.x + 1) + 1);
  SplitUnit u;
  u.b = lo.x;
  u.g = lo.y;
  u.rt = lo.z;
  u.slot0 = lo.w;
  u.nsl = hi.x;
  u.k = hi.y;
  if (u.nsl < 2) return;
  // a unit's heads follow each other in a slot
  const int head_rows = min(p.rows_per_cta, p.rows - u.rt * p.rows_per_cta), rows = p.unit_heads * head_rows;
  const int parts = (u.nsl - 1) * gridDim.y, part = u.k * gridDim.y + blockIdx.y;
  const int r_begin = static_cast<int>(static_cast<int64_t>(rows) * part / parts);
  const int r_end = static_cast<int>(static_cast<int64_t>(rows) * (part + 1) / parts);
  constexpr int W = kAttnMergeThreads / 32;
  if (u.nsl == 2) {
    for (int r = r_begin + 4 * warp; r < r_end; r += 4 * W) merge_rows<D, 4, 2>(p, u, r, r_end, head_rows, lane);
  } else {
    for (int r = r_begin + warp; r < r_end; r += W) merge_rows<D, 1, 8>(p, u, r, r + 1, head_rows, lane);
  }
}

template <int D>
cudaError_t launch_merge(const AttnParams& p, cudaStream_t stream) {
  if (p.grid < 2 || p.whole_units) return cudaSuccess;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  // Two blocks per boundary are one wave of them, and one pass of their warps over the rows
  // of a two-slot unit of up to 128 rows (four per boundary, two waves: 2 to 3 us slower).
  cfg.gridDim = dim3(p.grid - 1, p.slot_rows <= 32 ? 1 : 2);
  cfg.blockDim = dim3(kAttnMergeThreads);
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, attn_merge_kernel<D>, p);
}
#endif

}  // namespace specv
