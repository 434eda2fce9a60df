// Part (a) of the verify step for small KV groups (at most kMmaMaxRows query rows per KV
// head): block-causal or tree attention of the gamma block queries over a paged bf16 KV
// cache (Sec. 4.1), bound by the cache's bytes.
//
// At a few rows per KV head the arithmetic is a small fraction of the stream's time, and
// what decides is how the pages are fetched: a page of one KV head is 4 KB (16 tokens,
// head_dim 128), and 4 KB copies reach 4.5 TB/s, 8 KB ones 6.4 and 16 KB ones 6.7 (one
// block per SM streaming, no compute). So one block serves HB adjacent KV heads, which the
// cache stores next to each other within a page, and fetches a page of all of them with one
// copy. Per-head tcgen05 tiles would compute 128 rows for the few that are real and their
// accumulators for four heads would not fit in tensor memory; here each consumer warp owns
// one 16-row tile of one head and keeps its scores, probabilities and output in registers
// (mma.sync m16n8k16, bf16 operands, fp32 accumulators: 1,010 multiply-adds per cycle and
// SM), so that a tile of keys takes one barrier wait and no exchange between warps.
// Measured against the row-tile tcgen05 kernel, which keeps the larger groups: 32 requests of
// one query position over 256..16,384 keys (4 rows per KV head) 229 -> 169 us, 6.44 TB/s;
// 8 requests x 8 positions over 4,096 keys (32 rows) 45.1 -> 37.2 us; head_dim 64, 16 rows,
// 155 -> 61 us. With 33 to 64 rows the products alone take 0.8 of the stream's time
// (64 rows, ragged 512..4,096: 176 us against 124), hence kMmaMaxRows.
//
// Roles (one persistent block per SM): warps 0 and 1 copy K and V (one tensor box per
// 16..KS keys and HB heads, 128-byte swizzle) into a ring of 32 KB stages of KS keys of HB
// heads; consumer warp (h, t) takes rows [16t, 16t + 16) of head h over every stage.
// Work is cut "stream-K" style: the KS-key tiles of all (sequence, head group) units form
// one list that is cut into equal ranges; a unit split between blocks is merged from fp32
// partials by attn_merge_kernel (attn_common.cuh).
#include <cuda.h>

#include <algorithm>

#include "attn_common.cuh"
#include "tc_ptx.cuh"

namespace specv {
namespace {

using namespace tcx;

// HB KV heads per block, MTW 16-row tiles per head; KG key groups: with fewer than 8 (head,
// row tile) pairs, KG warps share one, each taking every KG-th stage (a warp alone is a
// chain of dependent instructions about as long as a stage's bytes take to arrive, 1,400
// cycles), and their states are merged through shared memory once per segment.
template <int D, int HB, int MTW>
struct MmaCfg {
  static constexpr int DH = D / 64;                    // 128-byte column halves of a row
  static constexpr int KS = 16384 / (HB * D * 2);      // keys per stage: 16 KB of K, 16 KB of V
  static constexpr int NS = KS / 16;                   // 16-key steps of a stage
  static constexpr int KG = HB * MTW >= 8 ? 1 : 8 / (HB * MTW);
  static constexpr uint32_t KV_BYTES = 16384;
  // a multiple of KG: a ring slot then always belongs to the same key group, whose warps see
  // every phase of its barriers (a parity wait that skips phases would pass early)
  static constexpr int STAGES = KG > 1 ? 4 : 6;
  static constexpr int PAIRS = HB * MTW;               // (head, row tile) pairs
  static constexpr int WARPS = PAIRS * KG;             // consumer warps
  static constexpr int THREADS = 64 + 32 * WARPS;
  static constexpr uint32_t OFF_V = STAGES * KV_BYTES;
  static constexpr uint32_t RING_BYTES = 2 * STAGES * KV_BYTES;
  // a warp's state handed over at a segment's end: O, then (m, l) of both rows, per lane
  static constexpr uint32_t XCH_WARP = (D / 2 + 4) * 32 * 4;
  static constexpr uint32_t OFF_XCH = RING_BYTES;
  static constexpr uint32_t OFF_BAR = OFF_XCH + (KG - 1) * PAIRS * XCH_WARP;
  // full[S], empty[S], xch_full[PAIRS], xch_free[PAIRS]
  static constexpr uint32_t OFF_MISC = OFF_BAR + (2 * STAGES + 2 * PAIRS) * 8;  // abort flag
  static constexpr uint32_t OFF_FLAG = OFF_MISC + 8;   // [S] bad flags of the stages
  static constexpr uint32_t OFF_PB = (OFF_FLAG + 4 * STAGES + 15) / 16 * 16;
  static size_t smem_bytes(int batch) { return OFF_PB + 4u * (batch + 1) + 1024; }
  static_assert(KS % 16 == 0 && KS <= 64, "16 to 64 keys per stage");
  static_assert(WARPS == 8 && STAGES % KG == 0, "eight consumer warps, ring slots owned by key groups");
};

// Keys [16s .. 16s + box keys) of one page of HB adjacent KV heads (box of the 4-D view of
// the cache, see encode_group_map), landing as [head][column half][key][128 B].
__device__ __forceinline__ void tma_load_group(uint32_t dst, const CUtensorMap* map, int key, int page_head,
                                               uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(0), "r"(key), "r"(0), "r"(page_head), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void ldsm4(uint32_t* r, uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}
__device__ __forceinline__ void ldsm4_t(uint32_t* r, uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}
// c += a b: a = 16 rows x 16 (row-major), b = 16 x 8 (column-major), fp32 c.
__device__ __forceinline__ void mma16816(float* c, const uint32_t* a, uint32_t b0, uint32_t b1) {
  asm(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9},"
      " {%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack_bf16x2(float a, float b) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&v);
}

template <int D, int HB, int MTW>
__global__ void __launch_bounds__(MmaCfg<D, HB, MTW>::THREADS, 1)
    attn_mma_kernel(const __grid_constant__ CUtensorMap tmap_k, const __grid_constant__ CUtensorMap tmap_v,
                    const __grid_constant__ AttnParams p, int page_shift, int box_shift) {
  using C = MmaCfg<D, HB, MTW>;
  constexpr int KS = C::KS, NS = C::NS, S = C::STAGES;
  const int box_keys = 1 << box_shift;  // keys per copy (page and box sizes are powers of two)
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  const uint32_t sbase = smem_u32(smem);
  const uint32_t bar0 = sbase + C::OFF_BAR;
  auto full = [&](uint32_t s) { return bar0 + 8u * s; };
  auto empty = [&](uint32_t s) { return bar0 + 8u * (S + s); };
  // the key groups of a (head, row tile) pair: their states are written / have been read
  auto xch_full = [&](int pair) { return bar0 + 8u * (2 * S + pair); };
  auto xch_free = [&](int pair) { return bar0 + 8u * (2 * S + C::PAIRS + pair); };
  int* misc = reinterpret_cast<int*>(smem + C::OFF_MISC);
  volatile int* abort_flag = misc;
  volatile int* stage_bad = reinterpret_cast<volatile int*>(smem + C::OFF_FLAG);
  int* pb = reinterpret_cast<int*>(smem + C::OFF_PB);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  // ---- prologue: barriers, per-sequence tile prefix sums ----
  if (warp == 1 && lane == 0) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmap_k)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmap_v)) : "memory");
    for (int s = 0; s < S; ++s) {
      mbar_init(full(s), 2);
      mbar_init(empty(s), C::PAIRS);  // the warps of the stage's key group
    }
    for (int i = 0; i < C::PAIRS && C::KG > 1; ++i) {
      mbar_init(xch_full(i), C::KG - 1);
      mbar_init(xch_free(i), 1);
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) tile_prefix<KS>(p, pb, lane);
  __syncthreads();

  const int64_t total = pb[p.batch];
  const int ctas = range_count(total, p);
  const int cta = blockIdx.x;
  int64_t t0, t1;
  block_range(p, pb, cta, total, ctas, t0, t1);
  const int OVH = p.unit_overhead;

  if (warp < 2) {
    // ============================ producers: K, V ============================
    uint32_t it = 0;
    bool ok = true;
    // page ids are read 32 at a time (lane i holds page cache_base + i of sequence cache_b)
    int cache_b = -1, cache_base = 0, cache_val = 0;
    auto page_of = [&](int b, int pi) -> int {  // warp-uniform
      if (b != cache_b || pi < cache_base || pi >= cache_base + 32) {
        cache_b = b;
        cache_base = pi;
        const int idx = pi + lane;
        cache_val = idx < p.max_pages ? __ldg(&p.page_table[static_cast<int64_t>(b) * p.max_pages + idx]) : 0;
      }
      return __shfl_sync(0xffffffffu, cache_val, pi - cache_base);
    };
    const CUtensorMap* map = warp == 0 ? &tmap_k : &tmap_v;
    const uint32_t ring = sbase + (warp == 0 ? 0u : C::OFF_V);
    const uint32_t box_bytes = static_cast<uint32_t>(box_keys) * D * 2 * HB;
    const Seg s_first = locate<KS>(t0, t1, p, pb, OVH);
    for (Seg s = s_first; s.ntile > 0 && ok && !p.starve;) {
      for (int k = 0; k < s.ntile; ++k, ++it) {
        const uint32_t st = it % S;
        const bool free = it < S || mbar_wait(empty(st), ((it / S) - 1) & 1, abort_flag, p.status);
        const int key0 = (s.tile0 + k) * KS;
        // boxes with a visible key; a malformed sequence reads nothing
        const int nbox = s.len_ok ? min(KS >> box_shift, (s.kv_len - key0 + box_keys - 1) >> box_shift) : 0;
        bool bad = !s.len_ok;
        int page[KS / 16];
#pragma unroll
        for (int q = 0; q < KS / 16; ++q)
          if (q < nbox) {
            const int raw = page_of(s.b, (key0 + (q << box_shift)) >> page_shift);
            const bool in_range = raw >= 0 && raw < p.num_pages;
            bad |= !in_range;
            page[q] = in_range ? raw : 0;  // an out-of-range page is read as page 0
          }
        if (lane == 0 && free) {
          if (warp == 0) stage_bad[st] = bad ? 1 : 0;
          if (nbox > 0) mbar_arrive_tx(full(st), nbox * box_bytes);
          else mbar_arrive(full(st));
#pragma unroll
          for (int q = 0; q < KS / 16; ++q)
            if (q < nbox)
              tma_load_group(ring + st * C::KV_BYTES + q * box_bytes, map, (key0 + (q << box_shift)) & (p.page_size - 1),
                             page[q] * p.hkv + s.g * HB, full(st));
        }
        // a wait that ran out in some lanes ends the loop for all of them, after the shuffles
        // of the page ids
        ok = __all_sync(0xffffffffu, free);
        if (!ok) {
          it += __shfl_sync(0xffffffffu, free ? 1u : 0u, 0);  // whether this tile's copies were issued
          break;
        }
      }
      if (!ok || !has_more(s, t1, OVH)) break;
      s = locate<KS>(s.vnext, t1, p, pb, OVH);
    }
    // the block's last tiles are on their way: the merge kernel's blocks may be brought in
    // (they wait for the whole grid, and find room only where a block has ended)
    if (warp == 1 && lane == 0) note_split(p, cta, s_first, total, ctas);
    pdl_launch_dependents();
    if (!ok) {  // copies still in flight land before the block exits (bounded)
      for (uint32_t x = it > S ? it - S : 0; x < it; ++x) {
        const long long c0 = clock64();
        while (!mbar_try(full(x % S), (x / S) & 1) && clock64() - c0 < kWaitCycles) {
        }
      }
    }
  } else {
    // ============================ consumers ============================
    const int cw = warp - 2, pair = cw % C::PAIRS, kg = cw / C::PAIRS, h = pair % HB, mt = pair / HB;
    const int r0 = mt * 16 + (lane >> 2), r1 = r0 + 8;  // this thread's rows of the head
    const int c2 = 2 * (lane & 3);
    // ldmatrix row addresses within a 16-key step: K by (key, 16-byte chunk), V transposed.
    // The 128-byte swizzle puts chunk c of a key at c ^ (key & 7), so a step's later chunks
    // are this address with bits 5 and 6 flipped.
    const uint32_t k_lane = ((lane & 7) + ((lane >> 4) << 3)) * 128u + (((lane >> 3) & 1) ^ (lane & 7)) * 16u;
    const uint32_t v_lane = (lane & 15) * 128u + ((lane >> 4) ^ (lane & 7)) * 16u;
    const uint32_t half_bytes = static_cast<uint32_t>(box_keys) * 128u;  // [box keys][128 B]
    const uint32_t head_off = static_cast<uint32_t>(h) * C::DH * half_bytes;
    uint32_t it = 0, seg_no = 0;
    bool ok = true;
    for (Seg s = locate<KS>(t0, t1, p, pb, OVH); s.ntile > 0 && ok; ++seg_no) {
      const bool real0 = r0 < p.rows, real1 = r1 < p.rows;
      const int j0 = real0 ? r0 / p.group : 0, j1 = real1 ? r1 / p.group : 0;
      const int head = (s.g * HB + h) * p.group;
      uint32_t q[D / 16][4];
      {
        const __nv_bfloat16* qp = static_cast<const __nv_bfloat16*>(p.q);
        const __nv_bfloat16* q0 = qp + ((static_cast<int64_t>(s.b) * p.gamma + j0) * p.hq + head + (real0 ? r0 % p.group : 0)) * D;
        const __nv_bfloat16* q1 = qp + ((static_cast<int64_t>(s.b) * p.gamma + j1) * p.hq + head + (real1 ? r1 % p.group : 0)) * D;
#pragma unroll
        for (int kk = 0; kk < D / 16; ++kk) {
          q[kk][0] = real0 ? __ldg(reinterpret_cast<const uint32_t*>(q0 + kk * 16 + c2)) : 0u;
          q[kk][1] = real1 ? __ldg(reinterpret_cast<const uint32_t*>(q1 + kk * 16 + c2)) : 0u;
          q[kk][2] = real0 ? __ldg(reinterpret_cast<const uint32_t*>(q0 + kk * 16 + 8 + c2)) : 0u;
          q[kk][3] = real1 ? __ldg(reinterpret_cast<const uint32_t*>(q1 + kk * 16 + 8 + c2)) : 0u;
        }
      }
      const int ctx = s.kv_len - p.gamma;
      unsigned long long mask0 = 0, mask1 = 0;
      if (p.tree_mask) {
        mask0 = __ldg(p.tree_mask + static_cast<int64_t>(s.b) * p.gamma + j0);
        mask1 = __ldg(p.tree_mask + static_cast<int64_t>(s.b) * p.gamma + j1);
      }
      float o[D / 8][4];
#pragma unroll
      for (int n = 0; n < D / 8; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) o[n][e] = 0.f;
      // running maxima (base 2, scaled) and this thread's share of the sums of both rows
      float m0 = -INFINITY, m1 = -INFINITY, l0 = 0.f, l1 = 0.f;
      bool bad = false;
      for (int k = 0; k < s.ntile; ++k, ++it) {
        if (C::KG > 1 && it % C::KG != static_cast<uint32_t>(kg)) continue;
        const uint32_t st = it % S;
        ok = mbar_wait_warp(full(st), (it / S) & 1, abort_flag, p.status);
        if (!ok) break;
        bad |= stage_bad[st] != 0;
        const int key0 = (s.tile0 + k) * KS;
        const uint32_t kst = sbase + st * C::KV_BYTES + head_off, vst = kst + C::OFF_V;
        auto step_off = [&](int n) {  // 16-key step n of the stage
          const int key = n * 16;
          return static_cast<uint32_t>(key >> box_shift) * (static_cast<uint32_t>(box_keys) * D * 2 * HB) +
                 static_cast<uint32_t>(key & (box_keys - 1)) * 128u;
        };
        // ---- scores ----
        float sc[NS][2][4];
        uint32_t krow[NS];
#pragma unroll
        for (int n = 0; n < NS; ++n) {
#pragma unroll
          for (int e = 0; e < 4; ++e) sc[n][0][e] = sc[n][1][e] = 0.f;
          krow[n] = kst + step_off(n) + k_lane;
        }
        // loads run a batch ahead of the products that use them
        constexpr int KB = NS >= 4 ? 1 : NS == 2 ? 2 : 4;  // 16-dim chunks per batch
        uint32_t kb[2][KB][NS][4];
#pragma unroll
        for (int i = 0; i < KB; ++i)
#pragma unroll
          for (int n = 0; n < NS; ++n) ldsm4(kb[0][i][n], krow[n] ^ (i * 32u));
#pragma unroll
        for (int k0 = 0; k0 < D / 16; k0 += KB) {
          const int cur = (k0 / KB) & 1;
          if (k0 + KB < D / 16) {
#pragma unroll
            for (int i = 0; i < KB; ++i)
#pragma unroll
              for (int n = 0; n < NS; ++n) {
                const int kk = k0 + KB + i;
                ldsm4(kb[cur ^ 1][i][n], (krow[n] ^ ((kk % 4) * 32u)) + (kk / 4) * half_bytes);
              }
          }
#pragma unroll
          for (int i = 0; i < KB; ++i)
#pragma unroll
            for (int n = 0; n < NS; ++n) {
              mma16816(sc[n][0], q[k0 + i], kb[cur][i][n][0], kb[cur][i][n][1]);
              mma16816(sc[n][1], q[k0 + i], kb[cur][i][n][2], kb[cur][i][n][3]);
            }
        }
        // ---- masks: only stages that reach the block's own keys ----
        if (key0 + KS > ctx) {
#pragma unroll
          for (int n = 0; n < NS; ++n)
#pragma unroll
            for (int t = 0; t < 2; ++t)
#pragma unroll
              for (int e = 0; e < 2; ++e) {
                const int rel = key0 + n * 16 + t * 8 + c2 + e - ctx;  // block position, < 0: the prefix
                bool v0, v1;
                if (p.tree_mask) {
                  v0 = rel < 0 || (rel < 64 && ((mask0 >> (rel & 63)) & 1ull));
                  v1 = rel < 0 || (rel < 64 && ((mask1 >> (rel & 63)) & 1ull));
                } else {
                  v0 = rel <= j0;
                  v1 = rel <= j1;
                }
                if (!v0) sc[n][t][e] = -INFINITY;
                if (!v1) sc[n][t][2 + e] = -INFINITY;
              }
        }
        // ---- online softmax. The maximum is raised whenever a row's grows: a row's largest
        // probability is then 1, which bf16 holds exactly. (Raised only past 2^8, as where the
        // output has to be fetched from tensor memory: the error of 4 rows over 512 keys is
        // 2.15e-3 instead of 2.00e-3, of 32 rows over 4,096 keys 2.29e-3 instead of 2.07e-3,
        // and the times are within 0.7%.) In short whole units each stage is taken against its
        // own maximum, as a part of a split unit would be (falling by 2^2 a stage at most, 2^14
        // over a unit's eight, which the accumulators grow by): 2.03e-3 for 8 to 32 rows, two
        // heads and up to 250 keys, as in parts, 2.05e-3 against the running maximum, in the same
        // time (8 units of 32 rows 12.3 us). ----
        float x0 = -INFINITY, x1 = -INFINITY;
#pragma unroll
        for (int n = 0; n < NS; ++n)
#pragma unroll
          for (int t = 0; t < 2; ++t) {
            x0 = fmaxf(x0, fmaxf(sc[n][t][0], sc[n][t][1]));
            x1 = fmaxf(x1, fmaxf(sc[n][t][2], sc[n][t][3]));
          }
        x0 = fmaxf(x0, __shfl_xor_sync(0xffffffffu, x0, 1));
        x1 = fmaxf(x1, __shfl_xor_sync(0xffffffffu, x1, 1));
        x0 = fmaxf(x0, __shfl_xor_sync(0xffffffffu, x0, 2)) * p.scale_log2;
        x1 = fmaxf(x1, __shfl_xor_sync(0xffffffffu, x1, 2)) * p.scale_log2;
        const float n0 = fmaxf(x0, m0 - p.fall), n1 = fmaxf(x1, m1 - p.fall);
        if (__any_sync(0xffffffffu, n0 != m0 || n1 != m1)) {
          const float a0 = m0 == -INFINITY ? 0.f : ex2(m0 - n0), a1 = m1 == -INFINITY ? 0.f : ex2(m1 - n1);
          m0 = n0;
          m1 = n1;
          l0 *= a0;
          l1 *= a1;
#pragma unroll
          for (int n = 0; n < D / 8; ++n) {
            o[n][0] *= a0;
            o[n][1] *= a0;
            o[n][2] *= a1;
            o[n][3] *= a1;
          }
        }
        const float d0 = m0 == -INFINITY ? 0.f : m0, d1 = m1 == -INFINITY ? 0.f : m1;
        uint32_t pr[NS][4];
#pragma unroll
        for (int n = 0; n < NS; ++n)
#pragma unroll
          for (int t = 0; t < 2; ++t) {
            const float e0 = ex2(fmaf(sc[n][t][0], p.scale_log2, -d0)), e1 = ex2(fmaf(sc[n][t][1], p.scale_log2, -d0));
            const float f0 = ex2(fmaf(sc[n][t][2], p.scale_log2, -d1)), f1 = ex2(fmaf(sc[n][t][3], p.scale_log2, -d1));
            l0 += e0 + e1;
            l1 += f0 + f1;
            pr[n][2 * t] = pack_bf16x2(e0, e1);
            pr[n][2 * t + 1] = pack_bf16x2(f0, f1);
          }
        // ---- O += P V; keys past the sequence's end meet P = 0, so their V must be finite ----
        const bool tail = key0 + KS > s.kv_len;
#pragma unroll
        for (int n = 0; n < NS; ++n) {
          uint32_t z0 = 0xffffffffu, z1 = 0xffffffffu;
          if (tail) {
            const int left = s.kv_len - (key0 + n * 16 + c2);  // keys from this thread's first one on
            z0 = left > 1 ? 0xffffffffu : left == 1 ? 0xffffu : 0u;
            z1 = left > 9 ? 0xffffffffu : left == 9 ? 0xffffu : 0u;
          }
          const uint32_t row = vst + step_off(n) + v_lane;
          constexpr int VB = 2;  // 16-dim chunks per batch
          uint32_t vb[2][VB][4];
#pragma unroll
          for (int i = 0; i < VB; ++i) ldsm4_t(vb[0][i], row ^ (i * 32u));
#pragma unroll
          for (int d0 = 0; d0 < D / 16; d0 += VB) {
            const int cur = (d0 / VB) & 1;
            if (d0 + VB < D / 16) {
#pragma unroll
              for (int i = 0; i < VB; ++i) {
                const int d = d0 + VB + i;
                ldsm4_t(vb[cur ^ 1][i], (row ^ ((d % 4) * 32u)) + (d / 4) * half_bytes);
              }
            }
#pragma unroll
            for (int i = 0; i < VB; ++i) {
              uint32_t* b = vb[cur][i];
              if (tail) {
                b[0] &= z0;
                b[1] &= z1;
                b[2] &= z0;
                b[3] &= z1;
              }
              mma16816(o[2 * (d0 + i)], pr[n], b[0], b[1]);
              mma16816(o[2 * (d0 + i) + 1], pr[n], b[2], b[3]);
            }
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(empty(st));
      }
      if (!ok) break;
      // ---- the segment's rows: output or partial ----
      l0 += __shfl_xor_sync(0xffffffffu, l0, 1);
      l1 += __shfl_xor_sync(0xffffffffu, l1, 1);
      l0 += __shfl_xor_sync(0xffffffffu, l0, 2);
      l1 += __shfl_xor_sync(0xffffffffu, l1, 2);
      if constexpr (C::KG > 1) {
        // the first key group takes the others' states; they go on to the next segment
        float* xch = reinterpret_cast<float*>(smem + C::OFF_XCH);
        if (kg > 0) {
          if (seg_no > 0)
            ok = mbar_wait_warp(xch_free(pair), (seg_no - 1) & 1, abort_flag, p.status);
          if (!ok) break;
          float* mine = xch + ((kg - 1) * C::PAIRS + pair) * (C::XCH_WARP / 4) + lane;
#pragma unroll
          for (int n = 0; n < D / 8; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e) mine[(n * 4 + e) * 32] = o[n][e];
          mine[(D / 2) * 32] = m0;
          mine[(D / 2 + 1) * 32] = m1;
          mine[(D / 2 + 2) * 32] = bad ? -1.f : l0;
          mine[(D / 2 + 3) * 32] = l1;
          __syncwarp();
          if (lane == 0) mbar_arrive(xch_full(pair));
          if (!has_more(s, t1, OVH)) break;
          s = locate<KS>(s.vnext, t1, p, pb, OVH);
          continue;
        }
        ok = mbar_wait_warp(xch_full(pair), seg_no & 1, abort_flag, p.status);
        if (!ok) break;
#pragma unroll 1
        for (int g = 0; g < C::KG - 1; ++g) {
          const float* other = xch + (g * C::PAIRS + pair) * (C::XCH_WARP / 4) + lane;
          const float om0 = other[(D / 2) * 32], om1 = other[(D / 2 + 1) * 32];
          float ol0 = other[(D / 2 + 2) * 32];
          const float ol1 = other[(D / 2 + 3) * 32];
          bad |= ol0 < 0.f;
          if (ol0 < 0.f) ol0 = 0.f;
          const float n0 = fmaxf(m0, om0), n1 = fmaxf(m1, om1);
          const float a0 = m0 == -INFINITY ? 0.f : ex2(m0 - n0), a1 = m1 == -INFINITY ? 0.f : ex2(m1 - n1);
          const float b0 = om0 == -INFINITY ? 0.f : ex2(om0 - n0), b1 = om1 == -INFINITY ? 0.f : ex2(om1 - n1);
          m0 = n0;
          m1 = n1;
          l0 = l0 * a0 + ol0 * b0;
          l1 = l1 * a1 + ol1 * b1;
#pragma unroll
          for (int n = 0; n < D / 8; ++n) {
            o[n][0] = o[n][0] * a0 + other[(n * 4) * 32] * b0;
            o[n][1] = o[n][1] * a0 + other[(n * 4 + 1) * 32] * b0;
            o[n][2] = o[n][2] * a1 + other[(n * 4 + 2) * 32] * b1;
            o[n][3] = o[n][3] * a1 + other[(n * 4 + 3) * 32] * b1;
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(xch_free(pair));
      }
      const bool whole = s.tile0 == 0 && s.ntile == s.unit_tiles;
      if (bad && cw == 0 && lane == 0) set_status(p.status, s.len_ok ? SPEC_FLAG_BAD_PAGE : SPEC_FLAG_BAD_KV_LEN);
      const int kvh = s.g * HB + h;
      if (whole) {
        const float i0 = bad || !(l0 > 0.f) ? 0.f : 1.f / l0, i1 = bad || !(l1 > 0.f) ? 0.f : 1.f / l1;
        auto out_row = [&](int r, int j) {
          return static_cast<__nv_bfloat16*>(p.out) +
                 ((static_cast<int64_t>(s.b) * p.gamma + j) * p.hq + kvh * p.group + r % p.group) * D + c2;
        };
        __nv_bfloat16* w0 = out_row(real0 ? r0 : 0, j0);
        __nv_bfloat16* w1 = out_row(real1 ? r1 : 0, j1);
#pragma unroll
        for (int n = 0; n < D / 8; ++n) {
          // a bad segment's accumulators hold other pages' values: exact zeros instead
          if (real0) *reinterpret_cast<uint32_t*>(w0 + n * 8) = bad ? 0u : pack_bf16x2(o[n][0] * i0, o[n][1] * i0);
          if (real1) *reinterpret_cast<uint32_t*>(w1 + n * 8) = bad ? 0u : pack_bf16x2(o[n][2] * i1, o[n][3] * i1);
        }
        if ((lane & 3) == 0) {
          if (real0) write_lse(p, s.b, kvh, r0, m0, l0, bad);
          if (real1) write_lse(p, s.b, kvh, r1, m1, l1, bad);
        }
      } else {
        const int64_t slot = (s.u + cta) * p.slot_rows + h * p.rows;
        float* w0 = p.partial_o + (slot + r0) * D + c2;
        float* w1 = p.partial_o + (slot + r1) * D + c2;
#pragma unroll
        for (int n = 0; n < D / 8; ++n) {
          if (real0) *reinterpret_cast<float2*>(w0 + n * 8) = make_float2(o[n][0], o[n][1]);
          if (real1) *reinterpret_cast<float2*>(w1 + n * 8) = make_float2(o[n][2], o[n][3]);
        }
        if ((lane & 3) == 0) {
          if (real0) p.partial_ml[slot + r0] = make_float2(m0, bad ? -1.f : l0);
          if (real1) p.partial_ml[slot + r1] = make_float2(m1, bad ? -1.f : l1);
        }
      }
      if (!has_more(s, t1, OVH)) break;
      s = locate<KS>(s.vnext, t1, p, pb, OVH);
    }
    if (!ok && (lane & 3) == 0)  // rows r0 and r1 = r0 + 8
      drop_partials_call<KS>(p, pb, h * p.rows + r0, h * p.rows + min(p.rows, r1 + 1), 8);
  }
}

// ---------------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------------
// K or V cache viewed as a 4-D tensor of bf16: (64 columns; the page's keys at stride D*2
// bytes; D/64 column halves at stride 128 bytes; page * Hkv + head at stride page*D*2); a
// box is box_keys keys of HB adjacent heads.
bool encode_group_map(CUtensorMap* map, const void* base, const spec_attn_args_t& a, int heads, int box_keys) {
  tcx::EncodeTiledFn enc = tcx::encoder();
  if (!enc) return false;
  const cuuint64_t D = static_cast<cuuint64_t>(a.head_dim);
  const cuuint64_t dims[4] = {64, static_cast<cuuint64_t>(a.page_size), D / 64,
                              static_cast<cuuint64_t>(a.num_pages) * a.num_kv_heads};
  const cuuint64_t strides[3] = {D * 2, 128, static_cast<cuuint64_t>(a.page_size) * D * 2};
  const cuuint32_t box[4] = {64, static_cast<cuuint32_t>(box_keys), static_cast<cuuint32_t>(D / 64),
                             static_cast<cuuint32_t>(heads)};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box, estr,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int shift_of(int x) {
  int s = 0;
  while ((1 << s) < x) ++s;
  return s;
}

template <int D, int HB, int MTW>
cudaError_t launch_typed(const spec_attn_args_t& a, const AttnPlan& P, char* ws, cudaStream_t stream,
                         bool starve) {
  using C = MmaCfg<D, HB, MTW>;
  const int box_keys = std::min(a.page_size, C::KS);
  CUtensorMap mk, mv;
  if (!encode_group_map(&mk, a.k_cache, a, HB, box_keys) || !encode_group_map(&mv, a.v_cache, a, HB, box_keys))
    return cudaErrorInvalidValue;
  AttnParams p = make_attn_params(a, P, ws);
  const int64_t units = static_cast<int64_t>(a.batch) * p.hunits;
  // a unit start costs about two tiles (its Q, the epilogue before it); charged when blocks
  // hold several, as in the row-tile kernel
  p.unit_overhead = units > P.grid ? 2 : 0;
  p.grid = P.grid;
  p.min_tiles = kMmaMinTiles;
  p.unit_heads = HB;
  p.starve = starve ? 1 : 0;
  p.whole_units = p.max_keys <= kWholeTiles * C::KS ? 1 : 0;
  p.fall = p.whole_units ? 2.f : 0.f;
  const size_t smem = C::smem_bytes(a.batch);
  auto kernel = attn_mma_kernel<D, HB, MTW>;
  const cudaError_t e = allow_smem(kernel, kTcMaxSmem);
  if (e != cudaSuccess) return e;
  kernel<<<P.grid, C::THREADS, smem, stream>>>(mk, mv, p, shift_of(a.page_size), shift_of(box_keys));
  const cudaError_t launched = cudaGetLastError();
  return launched != cudaSuccess ? launched : launch_merge<D>(p, stream);
}

template <int D, int HB>
cudaError_t launch_rows(const spec_attn_args_t& a, const AttnPlan& P, char* ws, cudaStream_t stream,
                        bool starve) {
  if (P.rows <= 16) return launch_typed<D, HB, 1>(a, P, ws, stream, starve);
  if constexpr (HB <= 4) return launch_typed<D, HB, 2>(a, P, ws, stream, starve);
  return cudaErrorInvalidValue;  // not planned (mma_heads)
}

}  // namespace

int mma_heads(const spec_attn_args_t& a, int rows) {
  const int hkv = a.num_kv_heads;
  if (rows > kMmaMaxRows || hkv % 2 != 0 ||
      std::max(MmaCfg<128, 2, 1>::smem_bytes(a.batch), MmaCfg<128, 4, 2>::smem_bytes(a.batch)) > kTcMaxSmem)
    return 0;
  for (int hb = a.head_dim == 128 ? 4 : 8; hb > 2; hb /= 2)
    if (hkv % hb == 0 && hb * ((rows + 15) / 16) <= 8) return hb;
  return 2;
}

cudaError_t launch_attn_mma(const spec_attn_args_t& a, const AttnPlan& P, char* ws, cudaStream_t stream,
                            bool starve) {
  if (a.head_dim == 128)
    return P.heads == 4 ? launch_rows<128, 4>(a, P, ws, stream, starve)
                        : launch_rows<128, 2>(a, P, ws, stream, starve);
  return P.heads == 8   ? launch_rows<64, 8>(a, P, ws, stream, starve)
         : P.heads == 4 ? launch_rows<64, 4>(a, P, ws, stream, starve)
                        : launch_rows<64, 2>(a, P, ws, stream, starve);
}

}  // namespace specv
