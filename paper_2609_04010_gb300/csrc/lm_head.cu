// The target's LM head with the acceptance's row statistics fused into it (Sec. 4.2:
// the verifier pass scores the block rows; Appendix B.3: the rule reads p through its
// normaliser, maximum and the logits of drafted tokens).
//
// lm_head_kernel<CG>: persistent groups of CG blocks (one block per SM; CG = 2 is a
// two-SM cluster whose tensor cores work on one tile), each taking (vocab tile, row tile)
// pairs from a fixed plan. A tile is 128 * CG hidden-state rows by up to 256 vocab rows;
// the fp32 accumulator is double-buffered in TMEM (2 x 256 columns), so the reduction of
// one tile runs under the copies and MMAs of the next. Warp 0 streams 64-column slices of
// the hidden states and of the weight rows by TMA (128-byte swizzle, out-of-range rows and
// columns read as zeros) into a ring (4 stages of 48 KB, or 7 of 32 KB with CG = 2, where
// each block brings its own 128 hidden-state rows and half of the weight rows); warp 1 of
// the group's first block issues tcgen05.mma (M = 128 * CG, N = the tile's vocab rows,
// K = 16); warps 2..5 then read one logit row each (a warp reaches the TMEM lanes of its
// own sub-partition) and reduce it, 32 columns at a time, to (max, sum of
// exp((l - max) / T), lowest-index argmax, logit of the row's token), optionally
// writing the logits as bf16. lm_merge_kernel: one block per row merges the vocab tiles'
// partials.
#include <cuda_bf16.h>

#include <algorithm>
#include <cfloat>
#include <climits>
#include <cmath>
#include <type_traits>

#include "lm_head.cuh"
#include "tc_ptx.cuh"

namespace specv {

namespace {

using namespace tcx;

constexpr int kBK = 64;           // hidden elements per stage: one 128-byte swizzle span
constexpr int kTileN = 256;       // most vocab rows of a tile
constexpr int kUnit = 16;         // vocab rows per block that tile sizes are multiples of
constexpr int kMergeThreads = 128;

// CG blocks per group (1, or 2 on a pair of SMs).
template <int CG>
struct LmCfg {
  static constexpr int STAGES = CG == 2 ? 7 : 4;
  static constexpr uint32_t A_BYTES = 128 * 128;                // a block's hidden states per stage
  static constexpr uint32_t B_BYTES = kTileN / CG * 128;        // a block's weight rows per stage
  static constexpr uint32_t OFF_B = STAGES * A_BYTES;
  static constexpr uint32_t OFF_BAR = OFF_B + STAGES * B_BYTES;
  // barriers: full[S], empty[S], acc_full[2], acc_empty[2], drain
  static constexpr uint32_t OFF_MISC = OFF_BAR + (2 * STAGES + 5) * 8;  // TMEM base, abort flag
  static constexpr size_t SMEM = OFF_MISC + 16 + 1024;          // + 1 KB alignment slack
};
static_assert(LmCfg<1>::SMEM <= kTcMaxSmem && LmCfg<2>::SMEM <= kTcMaxSmem, "one block per SM");
constexpr int kThreads = 192;  // warp 0 TMA, warp 1 MMA, warps 2..5 reduce

// The tile plan: row tiles of 128 * cg hidden-state rows by `tiles_n` vocab tiles. Tile n
// covers the vocab units (of kUnit * cg rows) [n * units / tiles_n, (n + 1) * units / tiles_n).
struct LmPlan {
  int cg, groups;
  int tiles_m, tiles_n;
  int64_t total;  // tiles_m * tiles_n
  int units, unit0;  // vocab units, and those of the smaller tile size (the other has one more)
};

// One block per row tile up to 128 rows: the weight stream bounds the call (at 128 rows
// its MMAs take half of the stream's time), so every SM gets an equal contiguous run of
// vocab rows. 64 rows of the 4096 x 128,256 head: 171.4 us, 6.13 TB/s (189.9 us with 573
// equal tiles on two blocks per SM, each tile's reduction after its MMAs). Above, pairs of
// SMs: a 256-row tile halves the bytes of weight each SM stages per MMA, and the tile count
// fills whole waves of the pairs. 1,024 rows of that head: 697 us, 1,544 TFLOP/s under the
// power limit (879 us with the 128 x 224 tiles of one SM); isolated, 629 us with the tensor
// pipe 75% active.
LmPlan lm_plan(const spec_lm_head_args_t& a, int sms) {
  LmPlan P;
  sms = std::min(std::max(sms, 2), kLmMaxSms);
  P.cg = a.rows <= 128 ? 1 : 2;
  P.groups = sms / P.cg;
  P.tiles_m = (a.rows + 128 * P.cg - 1) / (128 * P.cg);
  const int unit = kUnit * P.cg;
  const int64_t units = (static_cast<int64_t>(a.vocab) + unit - 1) / unit;
  const int64_t most = kTileN / unit;  // units of the largest tile
  const int64_t least_n = (units + most - 1) / most;
  const int64_t waves = (least_n * P.tiles_m + P.groups - 1) / P.groups;
  int64_t tn = waves * P.groups / P.tiles_m;
  tn = std::min(std::max(tn, least_n), units);
  P.units = static_cast<int>(units);
  P.tiles_n = static_cast<int>(tn);
  P.total = tn * P.tiles_m;
  // a tile holds unit0 or unit0 + 1 units; unit0 + 1 <= most unless tiles_n divides units
  P.unit0 = static_cast<int>(units / tn);
  return P;
}

struct LmPart {
  float m, s;   // tile maximum and sum of 2^((l - m) * c2)
  int32_t arg;  // lowest index of the maximum; -2: a non-finite logit in the tile
  float tok;    // the row token's logit if it lies in the tile, else NaN
};

struct LmParams {
  int rows, hidden, vocab, rows_per_seq, nk;
  int tiles_m, tiles_n, units, unit0, a_box;
  int64_t total;
  const float* temperature;
  const int32_t* tokens;
  __nv_bfloat16* logits;
  bool logits_vec;  // rows of the logits output are 16-byte aligned
  LmPart* parts;
  uint32_t* status;
  float* row_max;
  float* row_sum;
  int32_t* row_argmax;
  float* token_logit;
  int starve;  // test hook: the producer issues no copies, so the MMA warp's waits run out
};

__device__ __forceinline__ float row_c2(const LmParams& p, int row) {
  const float T = p.temperature[row / p.rows_per_seq];
  return kLog2e / (T > 0.f ? T : 1.f);
}

// (m, s, a) of two parts, both sums relative to their own maximum; equal maxima keep
// the lower index.
__device__ __forceinline__ void merge_part(float& m, float& s, int& a, float m2, float s2, int a2,
                                           float c2) {
  if (m2 == -INFINITY) return;
  if (m == -INFINITY) {
    m = m2;
    s = s2;
    a = a2;
    return;
  }
  const float M = fmaxf(m, m2);
  s = s * ex2((m - M) * c2) + s2 * ex2((m2 - M) * c2);
  a = m2 > m ? a2 : (m > m2 ? a : min(a, a2));
  m = M;
}

// --- two-SM forms (cta_group::2) ---
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// The address of this block's shared-memory location in block `rank` of the cluster.
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
// A box into this block's shared memory, completing on a barrier of either block of the pair.
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* map, int x, int y,
                                                 uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void mma_bf16_pair(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc,
                                              uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Arrives on the barrier at this offset in both blocks once the MMAs issued so far are done.
__device__ __forceinline__ void mma_commit_pair(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64"
      " [%0], %1;" ::"r"(bar), "h"(static_cast<uint16_t>(3))
      : "memory");
}
__device__ __forceinline__ void tmem_alloc_pair(uint32_t dst_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem),
               "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols)
               : "memory");
}

// One row's statistics while its tiles are reduced.
struct RowStats {
  float m;   // running maximum
  int a;     // its lowest index
  float s;   // sum of 2^((l - m) * c2) of this tile's columns so far
  float c2;
  int tok;   // the row's token, -1 if none
  float tl;  // its logit once met, else NaN
  float z;   // 0, or NaN after a NaN or an infinity
};

// W logits of this thread's row, at vocabulary indices col0.., of which the first nv are
// real, folded into its statistics. About 3.5 instructions a logit: a tree of maxima, one
// packed multiply-add for the non-finite test (x * 0 is NaN for NaN and infinities), one
// for the exponent's argument (two operations past kFusedMax), a packed sum. The index of a new maximum and the token's
// logit are looked for only in the columns that hold one. With compare-and-select chains
// per logit, about 10 instructions in series, the heads above took 177.7 and 716.7 us.
template <int W>
__device__ __forceinline__ void reduce_columns(RowStats& st, uint32_t* r, int col0, int nv) {
  float x[W];
#pragma unroll
  for (int e = 0; e < W; ++e) x[e] = __uint_as_float(r[e]);
  if (nv < W) {  // the vocabulary's end: repeat a real logit (its weight is 0 below)
#pragma unroll
    for (int e = 1; e < W; ++e)
      if (e >= nv) x[e] = x[0];
  }
  float mx[W / 4];
#pragma unroll
  for (int e = 0; e < W / 4; ++e) mx[e] = fmaxf(fmaxf(x[e], x[e + W / 4]), fmaxf(x[e + W / 2], x[e + 3 * W / 4]));
#pragma unroll
  for (int o = W / 8; o > 0; o >>= 1)
#pragma unroll
    for (int e = 0; e < o; ++e) mx[e] = fmaxf(mx[e], mx[e + o]);
  if (mx[0] > st.m) {
    int at = 0;
#pragma unroll
    for (int e = W - 1; e >= 0; --e) at = x[e] == mx[0] ? e : at;  // the lowest index of the maximum
    if (st.m > -INFINITY) st.s *= ex2((st.m - mx[0]) * st.c2);
    st.m = mx[0];
    st.a = col0 + at;
  }
  if (static_cast<unsigned>(st.tok - col0) < static_cast<unsigned>(nv)) {
#pragma unroll
    for (int e = 0; e < W; ++e)
      if (col0 + e == st.tok) st.tl = x[e];
  }
  const float mc = st.m > -INFINITY ? -st.m * st.c2 : 0.f;
  const uint64_t c22 = pack2(st.c2, st.c2), mc2 = pack2(mc, mc), zero = pack2(0.f, 0.f);
  const uint64_t m2 = pack2(-st.m, -st.m);
  uint64_t s0 = zero, s1 = zero, z0 = zero, z1 = zero;
  auto sums = [&](auto fused) {
#pragma unroll
    for (int e = 0; e < W; e += 4) {
      const uint64_t v0 = pack2(x[e], x[e + 1]), v1 = pack2(x[e + 2], x[e + 3]);
      z0 = fma2(v0, zero, z0);
      z1 = fma2(v1, zero, z1);
      float a0, a1, a2, a3;
      unpack2(decltype(fused)::value ? fma2(v0, c22, mc2) : mul2(add2(v0, m2), c22), a0, a1);
      unpack2(decltype(fused)::value ? fma2(v1, c22, mc2) : mul2(add2(v1, m2), c22), a2, a3);
      a0 = ex2(a0);
      a1 = ex2(a1);
      a2 = ex2(a2);
      a3 = ex2(a3);
      if (nv < W) {
        a0 = e < nv ? a0 : 0.f;
        a1 = e + 1 < nv ? a1 : 0.f;
        a2 = e + 2 < nv ? a2 : 0.f;
        a3 = e + 3 < nv ? a3 : 0.f;
      }
      s0 = add2(s0, pack2(a0, a1));
      s1 = add2(s1, pack2(a2, a3));
    }
  };
  if (past_fused(st.m, st.c2)) sums(std::false_type{});
  else sums(std::true_type{});
  float p0, p1, w0, w1;
  unpack2(add2(s0, s1), p0, p1);
  st.s += p0 + p1;
  unpack2(add2(z0, z1), w0, w1);
  st.z += w0 + w1;
}

// The same columns as bf16 logits.
template <int W>
__device__ __forceinline__ void store_logits(__nv_bfloat16* lrow, const uint32_t* r, int col0, int nv,
                                             bool vec) {
  if (nv == W && vec) {
    uint4* dst = reinterpret_cast<uint4*>(lrow + col0);
#pragma unroll
    for (int g = 0; g < W / 8; ++g) {
      uint32_t w[4];
#pragma unroll
      for (int h2 = 0; h2 < 4; ++h2) {
        const __nv_bfloat162 v2 = __floats2bfloat162_rn(__uint_as_float(r[8 * g + 2 * h2]),
                                                        __uint_as_float(r[8 * g + 2 * h2 + 1]));
        w[h2] = *reinterpret_cast<const uint32_t*>(&v2);
      }
      dst[g] = make_uint4(w[0], w[1], w[2], w[3]);
    }
  } else {
#pragma unroll
    for (int e = 0; e < W; ++e)
      if (e < nv) lrow[col0 + e] = __float2bfloat16_rn(__uint_as_float(r[e]));
  }
}

// A tile of the plan: its row tile and the vocab rows [n0, n0 + n).
struct Tile {
  int tm, tn, n0, n;
};
template <int CG>
__device__ __forceinline__ Tile tile_of(int64_t id, const LmParams& p) {
  Tile t;
  t.tn = static_cast<int>(id / p.tiles_m);
  t.tm = static_cast<int>(id - static_cast<int64_t>(t.tn) * p.tiles_m);
  const int64_t u0 = static_cast<int64_t>(t.tn) * p.units / p.tiles_n;
  const int64_t u1 = (static_cast<int64_t>(t.tn) + 1) * p.units / p.tiles_n;
  t.n0 = static_cast<int>(u0) * kUnit * CG;
  t.n = static_cast<int>(u1 - u0) * kUnit * CG;
  return t;
}

template <int CG>
__global__ void __launch_bounds__(kThreads, 1)
    lm_head_kernel(const __grid_constant__ CUtensorMap map_h, const __grid_constant__ CUtensorMap map_w,
                   const __grid_constant__ CUtensorMap map_w1, LmParams p) {
  using C = LmCfg<CG>;
  constexpr int S = C::STAGES;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  const uint32_t sbase = smem_u32(smem);
  const uint32_t bar0 = sbase + C::OFF_BAR;
  auto full = [&](uint32_t s) { return bar0 + 8u * s; };
  auto empty = [&](uint32_t s) { return bar0 + 8u * (S + s); };
  auto acc_full = [&](uint32_t b) { return bar0 + 8u * (2 * S + b); };
  auto acc_empty = [&](uint32_t b) { return bar0 + 8u * (2 * S + 2 + b); };
  const uint32_t drain = bar0 + 8u * (2 * S + 4);
  uint32_t* misc = reinterpret_cast<uint32_t*>(smem + C::OFF_MISC);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(misc + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = CG == 2 ? cluster_rank() : 0u;
  const int64_t group = blockIdx.x / CG, groups = gridDim.x / CG;
  pdl_launch_dependents();
  // The group's tiles. One row tile: an equal contiguous run of vocab tiles. Several: every
  // groups-th tile, so that the row tiles that share a weight tile run together and read
  // it from DRAM once (the others hit L2).
  const bool strided = p.tiles_m > 1;
  const int64_t first = strided ? group : group * p.total / groups;
  const int64_t last = strided ? p.total : (group + 1) * p.total / groups;
  const int64_t step = strided ? groups : 1;

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(full(s), 1);
      mbar_init(empty(s), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(acc_full(b), 1);
      mbar_init(acc_empty(b), 4 * CG);
    }
    mbar_init(drain, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    if (CG == 2) tmem_alloc_pair(smem_u32(misc), 2 * kTileN);
    else tmem_alloc(smem_u32(misc), 2 * kTileN);
  }
  tc_fence_before();
  __syncthreads();
  if (CG == 2) cluster_sync();  // both blocks' barriers exist before either signals the other's
  tc_fence_after();
  const uint32_t tmem = misc[0];

  if (warp == 0) {
    // ============================ TMA producer ============================
    if (lane == 0) {
      uint32_t it = 0;
      bool ok = true;
      for (int64_t id = first; id < last && ok && !p.starve; id += step) {
        const Tile t = tile_of<CG>(id, p);
        const int nb = t.n / CG;                    // weight rows this block brings
        const bool extra = nb > p.unit0 * kUnit;    // ... one unit more than map_w's box
        const int y_h = (t.tm * CG + static_cast<int>(rank)) * 128;
        const int y_w = t.n0 + static_cast<int>(rank) * nb;
        const uint32_t bytes = (static_cast<uint32_t>(p.a_box) + nb) * 128u * CG;
        for (int k = 0; k < p.nk; ++k, ++it) {
          const uint32_t s = it % S;
          if (it >= S) ok = mbar_wait(empty(s), ((it / S) - 1) & 1, abort_flag, p.status);
          if (!ok) break;
          // the group's first block expects the bytes of both; the second signals its barrier
          if (rank == 0) mbar_arrive_tx(full(s), bytes);
          const uint32_t bar = CG == 2 ? map_rank(full(s), 0) : full(s);
          const uint32_t a = sbase + s * C::A_BYTES, b = sbase + C::OFF_B + s * C::B_BYTES;
          if (CG == 2) {
            tma_load_2d_pair(a, &map_h, k * kBK, y_h, bar);
            tma_load_2d_pair(b, &map_w, k * kBK, y_w, bar);
            if (extra) tma_load_2d_pair(b + p.unit0 * kUnit * 128u, &map_w1, k * kBK, y_w + p.unit0 * kUnit, bar);
          } else {
            tma_load_2d(a, &map_h, k * kBK, y_h, bar);
            tma_load_2d(b, &map_w, k * kBK, y_w, bar);
            if (extra) tma_load_2d(b + p.unit0 * kUnit * 128u, &map_w1, k * kBK, y_w + p.unit0 * kUnit, bar);
          }
        }
      }
      if (ok) {
        // every stage has been released: the MMAs are done with both blocks' stages, and no
        // arrival on this block's barriers is outstanding when it exits
        for (uint32_t x = it > S ? it - S : 0; x < it && ok; ++x)
          ok = mbar_wait(empty(x % S), (x / S) & 1, abort_flag, p.status);
      }
      if (!ok && rank == 0) {  // let the copies still in flight land before the block exits (bounded)
        for (uint32_t x = it > S ? it - S : 0; x < it; ++x) {
          const long long t0 = clock64();
          while (!mbar_try(full(x % S), (x / S) & 1) && clock64() - t0 < kWaitCycles) {
          }
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ============================ MMA issuer ============================
    if (lane == 0 && rank == 0) {
      uint32_t it = 0, tile = 0;
      bool ok = true;
      for (int64_t id = first; id < last && ok; id += step, ++tile) {
        const uint32_t buf = tile & 1;
        const uint32_t idesc = idesc_bf16(128 * CG, 16, false) - (2u << 17) +
                               (static_cast<uint32_t>(tile_of<CG>(id, p).n >> 3) << 17);
        if (tile >= 2) {  // the reduction has read this buffer's previous tile
          ok = mbar_wait(acc_empty(buf), ((tile >> 1) - 1) & 1, abort_flag, p.status);
          if (!ok) break;
          tc_fence_after();
        }
        const uint32_t d = tmem + buf * kTileN;
        for (int k = 0; k < p.nk && ok; ++k, ++it) {
          const uint32_t s = it % S;
          ok = mbar_wait(full(s), (it / S) & 1, abort_flag, p.status);
          if (!ok) break;
          tc_fence_after();
#pragma unroll
          for (int kk = 0; kk < kBK / 16; ++kk) {
            const uint64_t ad = desc_sw128(sbase + s * C::A_BYTES + kk * 32u, 16, 1024);
            const uint64_t bd = desc_sw128(sbase + C::OFF_B + s * C::B_BYTES + kk * 32u, 16, 1024);
            if (CG == 2) mma_bf16_pair(d, ad, bd, idesc, (k > 0 || kk > 0) ? 1u : 0u);
            else mma_bf16(d, ad, bd, idesc, (k > 0 || kk > 0) ? 1u : 0u);
          }
          // the stage is free once these MMAs have read it
          if (CG == 2) mma_commit_pair(empty(s));
          else mma_commit(empty(s));
        }
        if (!ok) break;
        if (CG == 2) mma_commit_pair(acc_full(buf));
        else mma_commit(acc_full(buf));
      }
      if (!ok) {  // MMAs still in flight end before the block does (bounded)
        if (CG == 2) mma_commit_pair(drain);
        else mma_commit(drain);
        const long long t0 = clock64();
        while (!mbar_try(drain, 0) && clock64() - t0 < kWaitCycles) {
        }
      }
    }
    __syncwarp();
  } else {
    // ============================ row reduction ============================
    const int q = warp & 3;  // this warp's TMEM lane quadrant
    uint32_t tile = 0;
    int tm_prev = -1;
    // The running maximum and its lowest index carry over from tile to tile of a row (the
    // group's tiles ascend in vocabulary order); the sum starts anew with each partial. A
    // partial's (max, index) is then that of the tiles up to it, which the merge takes alike.
    RowStats st;
    for (int64_t id = first; id < last; id += step, ++tile) {
      const Tile t = tile_of<CG>(id, p);
      const uint32_t buf = tile & 1;
      const int row0 = (t.tm * CG + static_cast<int>(rank)) * 128 + q * 32;
      const int row = row0 + lane;
      const bool real = row < p.rows;
      if (t.tm != tm_prev) {
        st.m = -INFINITY;
        st.a = INT_MAX;
        st.c2 = real ? row_c2(p, row) : kLog2e;
        st.tok = (real && p.tokens) ? p.tokens[row] : -1;
        tm_prev = t.tm;
      }
      st.s = 0.f;
      st.tl = __int_as_float(0x7fc00000);
      st.z = 0.f;
      if (!__all_sync(0xffffffffu, mbar_wait(acc_full(buf), (tile >> 1) & 1, abort_flag, p.status))) break;
      tc_fence_after();
      if (row0 < p.rows) {  // warps without a row of the call have nothing to read
        __nv_bfloat16* lrow = (p.logits && real) ? p.logits + static_cast<int64_t>(row) * p.vocab : nullptr;
        const int n = min(t.n, p.vocab - t.n0);  // past the vocabulary: zero rows, not logits
        const uint32_t col = tmem + (static_cast<uint32_t>(q * 32) << 16) + buf * kTileN;
        int c = 0;
#pragma unroll 1
        for (; c + 64 <= n; c += 64) {
          uint32_t r[32], r2[32];
          tmem_ld32(col + c, r);
          tmem_ld32(col + c + 32, r2);
          tmem_wait_ld();
          reduce_columns<32>(st, r, t.n0 + c, 32);
          reduce_columns<32>(st, r2, t.n0 + c + 32, 32);
          if (lrow) {
            store_logits<32>(lrow, r, t.n0 + c, 32, p.logits_vec);
            store_logits<32>(lrow, r2, t.n0 + c + 32, 32, p.logits_vec);
          }
        }
#pragma unroll 1
        for (; c < n; c += 16) {  // the tile's last columns, 16 at a time
          uint32_t r[16];
          tmem_ld16(col + c, r);
          tmem_wait_ld();
          const int nv = min(16, n - c);
          reduce_columns<16>(st, r, t.n0 + c, nv);
          if (lrow) store_logits<16>(lrow, r, t.n0 + c, nv, p.logits_vec);
        }
      }
      // this quadrant is read: the buffer may take the next tile but one
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (CG == 2) mbar_arrive_cluster(map_rank(acc_empty(buf), 0));
        else mbar_arrive(acc_empty(buf));
      }
      if (real) {
        LmPart out;
        out.m = st.m;
        out.s = st.s;
        out.arg = st.z == 0.f ? st.a : -2;  // NaN: a non-finite logit
        out.tok = st.tl;
        p.parts[static_cast<int64_t>(row) * p.tiles_n + t.tn] = out;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (CG == 2) cluster_sync();
  if (warp == 1) {
    tc_fence_after();
    if (CG == 2) tmem_dealloc_pair(tmem, 2 * kTileN);
    else tmem_dealloc(tmem, 2 * kTileN);
  }
}

// One block per row: the vocab tiles' partials merged into the row's statistics. Each
// thread's first kMergeBatch partials load together (with 128 threads, all of a row's up to
// 1,024 tiles), so a row costs one round trip; with one warp per row and a dependent
// load per 32 tiles the 1,024-row head's merge took 14.5 us, now 7.9 (64 rows: 14.5, now 5.9;
// cold, under ncu).
constexpr int kMergeBatch = 8;
__global__ void __launch_bounds__(kMergeThreads) lm_merge_kernel(LmParams p) {
  __shared__ float sh_m[4], sh_s[4], sh_t[4];
  __shared__ int sh_a[4], sh_bad[4];
  const int row = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const float c2 = row_c2(p, row);
  pdl_wait_prior();
  float m = -INFINITY, s = 0.f, tl = __int_as_float(0x7fc00000);
  int a = INT_MAX;
  bool bad = false;
  const float4* parts = reinterpret_cast<const float4*>(p.parts + static_cast<int64_t>(row) * p.tiles_n);
  for (int t0 = threadIdx.x; t0 < p.tiles_n; t0 += kMergeBatch * kMergeThreads) {
    float4 q[kMergeBatch];
#pragma unroll
    for (int i = 0; i < kMergeBatch; ++i) {
      const int t = t0 + i * kMergeThreads;
      q[i] = t < p.tiles_n ? __ldcg(parts + t)
                           : make_float4(-INFINITY, 0.f, __int_as_float(INT_MAX), __int_as_float(0x7fc00000));
    }
#pragma unroll
    for (int i = 0; i < kMergeBatch; ++i) {
      const int arg = __float_as_int(q[i].z);
      bad |= arg == -2;
      if (q[i].w == q[i].w) tl = q[i].w;
      merge_part(m, s, a, q[i].x, q[i].y, arg, c2);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float m2 = __shfl_xor_sync(0xffffffffu, m, o), s2 = __shfl_xor_sync(0xffffffffu, s, o);
    const int a2 = __shfl_xor_sync(0xffffffffu, a, o);
    merge_part(m, s, a, m2, s2, a2, c2);
  }
  const unsigned has_tok = __ballot_sync(0xffffffffu, tl == tl);
  if (has_tok) tl = __shfl_sync(0xffffffffu, tl, __ffs(has_tok) - 1);
  bad = __any_sync(0xffffffffu, bad);
  if (lane == 0) {
    sh_m[warp] = m;
    sh_s[warp] = s;
    sh_a[warp] = a;
    sh_t[warp] = tl;
    sh_bad[warp] = bad;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kMergeThreads / 32; ++w) {
      merge_part(m, s, a, sh_m[w], sh_s[w], sh_a[w], c2);
      if (sh_t[w] == sh_t[w]) tl = sh_t[w];
      bad |= sh_bad[w] != 0;
    }
    p.row_max[row] = m;
    p.row_sum[row] = s;
    p.row_argmax[row] = bad ? -1 : a;
    if (p.token_logit) p.token_logit[row] = tl;
    if (bad) set_status(p.status, SPEC_FLAG_BAD_LOGITS);
  }
}

template <int CG>
cudaError_t launch_typed(const spec_lm_head_args_t& a, const LmPlan& P, const LmParams& p,
                         cudaStream_t stream) {
  using C = LmCfg<CG>;
  CUtensorMap mh, mw, mw1;
  if (!encode_rows_map(&mh, a.hidden_states, a.rows, a.hidden, p.a_box) ||
      !encode_rows_map(&mw, a.weight, a.vocab, a.hidden, P.unit0 * kUnit) ||
      !encode_rows_map(&mw1, a.weight, a.vocab, a.hidden, kUnit))
    return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(lm_head_kernel<CG>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(C::SMEM));
  if (e != cudaSuccess) return e;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = CG;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(std::min<int64_t>(P.groups, P.total)) * CG);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = C::SMEM;
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = CG == 2 ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, lm_head_kernel<CG>, mh, mw, mw1, p);
}

}  // namespace

LmLayout lm_layout(const spec_lm_head_args_t& a, size_t base) {
  LmLayout L;
  size_t tiles = 0;  // no plan has more vocab tiles (both are bounded by the vocab's units)
  const size_t units = (static_cast<size_t>(a.vocab) + kUnit - 1) / kUnit;
  tiles = std::min(units, (static_cast<size_t>(a.vocab) + kTileN - 1) / kTileN + kLmMaxSms);
  L.parts = base;
  L.end = ws_round(L.parts + 16 * static_cast<size_t>(a.rows) * tiles);
  return L;
}

cudaError_t launch_lm_head(const spec_lm_head_args_t& a, const LmLayout& L, char* ws, int sms,
                           cudaStream_t stream, bool starve) {
  const LmPlan P = lm_plan(a, sms);
  LmParams p;
  p.rows = a.rows;
  p.hidden = a.hidden;
  p.vocab = a.vocab;
  p.rows_per_seq = a.rows_per_seq;
  p.nk = (a.hidden + kBK - 1) / kBK;
  p.tiles_m = P.tiles_m;
  p.tiles_n = P.tiles_n;
  p.units = P.units;
  p.unit0 = P.unit0;
  p.total = P.total;
  // hidden-state rows per copy: rows past the call's only fill accumulator rows that no
  // warp reads as real, so a small call copies (and clears) no padding
  p.a_box = P.cg == 2 ? 128 : (a.rows + 7) / 8 * 8;
  p.temperature = a.temperature;
  p.tokens = a.tokens;
  p.logits = static_cast<__nv_bfloat16*>(a.logits);
  p.logits_vec = (a.vocab & 7) == 0 && (reinterpret_cast<uintptr_t>(a.logits) & 15u) == 0;
  p.parts = reinterpret_cast<LmPart*>(ws + L.parts);
  p.status = reinterpret_cast<uint32_t*>(ws);
  p.row_max = a.row_max;
  p.row_sum = a.row_sum;
  p.row_argmax = a.row_argmax;
  p.token_logit = a.token_logit;
  p.starve = starve ? 1 : 0;
  (void)cudaGetLastError();
  cudaError_t e = P.cg == 2 ? launch_typed<2>(a, P, p, stream) : launch_typed<1>(a, P, p, stream);
  if (e != cudaSuccess) return e;
  // a programmatic dependent: its blocks may be resident before the tiles are done
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(a.rows));
  cfg.blockDim = dim3(kMergeThreads);
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, lm_merge_kernel, p);
}

}  // namespace specv
