// Draft-side steps of Alg. "Lossless Psi-Spec decoding (Linear Sampler)" (Appendix
// B.3): sampling the block tokens from the drafter rows (the free clean token
// x^{L+1} ~ q_0 and the B-1 drafts x~ ~ q, in parallel), and rolling the paged KV cache
// back to the step's accepted prefix.
//
// draft_sample_kernel draws without filtering, in one launch with one or more blocks per
// drafter row. Each block streams its part of the row once and keeps, for every lane of
// 64 (16-byte loads) or 32 (element loads) contiguous logits, the lane's maximum m_i and
// s_i = sum over the lane of exp2((l - m_i) log2(e) / T). These lane summaries give the
// row's normaliser S and the cumulative mass at every lane boundary, so the inverse CDF
// needs no second pass over the row: a block scan finds the lane where the cumulative
// mass crosses u * S, and one warp rescans that lane's logits. The filtered draw is the
// filtered row kernel's draw mode.
//
// commit_kv_kernel is one block: it computes every sequence's new length and page request
// (or release), takes block-wide prefix sums in batch order, and serves the requests that
// fit, so the result is the batch-order definition computed in parallel.
#include <cuda_bf16.h>

#include <cfloat>
#include <climits>
#include <cmath>
#include <type_traits>

#include "common.cuh"

namespace specv {

DraftLayout draft_layout(const spec_draft_args_t& a, size_t base, int sms, bool vec) {
  DraftLayout L;
  L.lane_elems = vec ? 64 : 32;
  L.nlanes = static_cast<int>((static_cast<int64_t>(a.vocab) + L.lane_elems - 1) / L.lane_elems);
  const int64_t rows = static_cast<int64_t>(a.batch) * a.gamma;
  int64_t splits = static_cast<int64_t>(kFiltBlocksPerSm) * sms / rows;  // within one wave
  splits = splits < 1 ? 1 : (splits > kFiltMaxSplits ? kFiltMaxSplits : splits);
  if (splits > L.nlanes) splits = L.nlanes;
  L.lanes_per_split = static_cast<int>((L.nlanes + splits - 1) / splits);
  L.splits = (L.nlanes + L.lanes_per_split - 1) / L.lanes_per_split;
  L.smem = static_cast<size_t>(L.nlanes) * 8;
  const size_t split_rows = L.splits > 1 ? static_cast<size_t>(rows) : 0;
  L.tickets = base;
  L.row_flags = ws_round(L.tickets + sizeof(uint32_t) * a.batch);
  L.row_tickets = ws_round(L.row_flags + sizeof(uint32_t) * rows);
  L.lanes_g = ws_round(L.row_tickets + sizeof(uint32_t) * split_rows);
  L.parts = ws_round(L.lanes_g + 8 * split_rows * L.nlanes);
  L.end = ws_round(L.parts + 16 * split_rows * L.splits);
  return L;
}

namespace {

constexpr int kThreads = kRowThreads;
constexpr int kUnroll = 8;  // 16-byte loads (or elements) in flight per thread
constexpr int kStageGranules = 4 * kThreads;  // 16-byte granules of an unaligned row staged at a time
constexpr uint32_t kBadRow = 1u;

struct DraftParams {
  int batch, gamma, vocab, lane_elems, nlanes, splits, lanes_per_split;
  const void* drafter;
  const float* temperature;
  const float* uniforms;
  int32_t* tokens;
  float* q_tok;
  uint32_t* status;
  uint32_t* tickets;      // [batch]
  uint32_t* row_flags;    // [batch][gamma]
  uint32_t* row_tickets;  // [batch][gamma] (splits > 1)
  float2* lanes_g;        // [batch][gamma][nlanes] (splits > 1)
  uint4* parts;           // [batch][gamma][splits]: (row maximum candidate, bad)
};

template <bool BF16>
__device__ __forceinline__ float load_elem(const void* base, int64_t i) {
  if (BF16) return bf16_bits_to_f32(static_cast<const uint16_t*>(base)[i]);
  return static_cast<const float*>(base)[i];
}

// Order-preserving key of a float (-0 shares +0's key); a candidate packs the key above
// 0xffffffff - index, so the larger candidate is the larger value, then the lower index.
__device__ __forceinline__ uint32_t order_key(float x) {
  uint32_t f = __float_as_uint(x);
  if (f == 0x80000000u) f = 0u;
  return (f & 0x80000000u) ? ~f : (f | 0x80000000u);
}
__device__ __forceinline__ unsigned long long cand_of(float x, uint32_t idx) {
  return (static_cast<unsigned long long>(order_key(x)) << 32) | (0xffffffffu - idx);
}
__device__ __forceinline__ int cand_idx(unsigned long long c) {
  return static_cast<int>(0xffffffffu - static_cast<uint32_t>(c));
}

// Block-wide exclusive scan of one float per thread, in thread order; *total gets the sum.
__device__ __forceinline__ float block_excl_scan(float x, float* sh, float* total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  float in = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const float y = __shfl_up_sync(0xffffffffu, in, o);
    if (lane >= o) in += y;
  }
  if (lane == 31) sh[w] = in;
  __syncthreads();
  if (threadIdx.x == 0) {
    float run = 0.f;
    for (int k = 0; k < kThreads / 32; ++k) {
      const float t = sh[k];
      sh[k] = run;
      run += t;
    }
    sh[kThreads / 32] = run;
  }
  __syncthreads();
  const float ex = sh[w] + in - x;
  *total = sh[kThreads / 32];
  __syncthreads();
  return ex;
}

// Place of lane i of n in shared memory: within each whole 256 lanes' 16-lane runs the low
// bits are rotated by the run, so that threads that each walk a run of 16 lanes hit
// different banks (in order they all hit one).
__device__ __forceinline__ int lane_at(int i, int n) { return i < (n & ~15) ? i ^ ((i >> 4) & 15) : i; }

// Packed maximum of two bf16 pairs (a NaN loses to a number).
__device__ __forceinline__ uint32_t max2(uint32_t a, uint32_t b) {
  const __nv_bfloat162 h = __hmax2(*reinterpret_cast<const __nv_bfloat162*>(&a), *reinterpret_cast<const __nv_bfloat162*>(&b));
  return *reinterpret_cast<const uint32_t*>(&h);
}
// The reverse: every thread of the group gets all 8 of reduce8's results.
__device__ __forceinline__ void gather8(float r, int i, float* v) {
  const bool b0 = i & 1, b1 = i & 2, b2 = i & 4;
  const float x = __shfl_xor_sync(0xffffffffu, r, 4);
  const float a[2] = {b2 ? x : r, b2 ? r : x};  // values i & 3 and (i & 3) + 4
  float c[4];                                   // values (i & 1) + 2 j
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const float y = __shfl_xor_sync(0xffffffffu, a[j], 2);
    c[2 * j] = b1 ? y : a[j];
    c[2 * j + 1] = b1 ? a[j] : y;
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float y = __shfl_xor_sync(0xffffffffu, c[j], 1);
    v[2 * j] = b0 ? y : c[j];
    v[2 * j + 1] = b0 ? c[j] : y;
  }
}

// One round of the scan of a bf16 row: thread t's vectors v0 + 128 k + t (k < 8), each 8
// logits; the 8 threads of a group share, for every k, one 64-logit lane. Each lane's
// maximum and sum are reduced over its threads, in the same tree as by a butterfly per
// lane, but for the 8 lanes together: each exchange halves the lanes a thread still
// carries, 7 shuffles for 8 maxima (two bf16 to a word) and 7 for 8 sums instead of 24
// each, and thread i of a group ends with lane k = i. 1,024 rows of 128,256 logits: 72.4 us
// with butterflies and one shared atomic per lane in the pick below, now 53.4 (4.92 TB/s).
__device__ __forceinline__ void scan_bf16(const uint4* dv, int v0, int vend, int l0, int n,
                                          float c, bool greedy, float2* lanes, float& m, int& a, uint32_t& nacc,
                                          bool& bad) {
  static_assert(kUnroll == 8, "8 lanes for the 8 threads of a group");
  const int tid = threadIdx.x, i = tid & 7;
  uint32_t h[8];  // each vector's maxima of even and odd elements
#pragma unroll
  for (int k = 0; k < 8; ++k) h[k] = max2(max2(dv[k].x, dv[k].y), max2(dv[k].z, dv[k].w));
  auto hi_f = [](uint32_t w) { return __uint_as_float(w & 0xffff0000u); };
  auto lo_f = [](uint32_t w) { return __uint_as_float(w << 16); };
  if (greedy) {
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const uint32_t wv[4] = {dv[k].x, dv[k].y, dv[k].z, dv[k].w};
#pragma unroll
      for (int q = 0; q < 4; ++q) nacc |= (wv[q] & 0x7FFF7FFFu) + 0x007F007Fu;
      const float vm = fmaxf(lo_f(h[k]), hi_f(h[k]));
      if (vm > m) {  // rare: the first element of the vector that holds the new maximum
        m = vm;
        int at = 7;
#pragma unroll
        for (int q = 6; q >= 0; --q) at = ((q & 1) ? hi_f(wv[q >> 1]) : lo_f(wv[q >> 1])) == vm ? q : at;
        a = (v0 + k * kThreads + tid) * 8 + at;
      }
    }
    return;
  }
  // w[j]: the vectors' maxima of lanes j (low half) and j + 4 (high half)
  uint32_t w[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const uint32_t lo = max2(h[j], __byte_perm(h[j], 0, 0x1032)), hi = max2(h[j + 4], __byte_perm(h[j + 4], 0, 0x1032));
    w[j] = __byte_perm(lo, hi, 0x5410);
  }
  {
    const uint32_t all = max2(max2(w[0], w[1]), max2(w[2], w[3]));
    m = fmaxf(m, fmaxf(lo_f(all), hi_f(all)));
  }
  const bool b0 = i & 1, b1 = i & 2, b2 = i & 4;
  uint32_t k0 = b0 ? w[1] : w[0], k1 = b0 ? w[3] : w[2];
  k0 = max2(k0, __shfl_xor_sync(0xffffffffu, b0 ? w[0] : w[1], 1));
  k1 = max2(k1, __shfl_xor_sync(0xffffffffu, b0 ? w[2] : w[3], 1));
  uint32_t kk = b1 ? k1 : k0;
  kk = max2(kk, __shfl_xor_sync(0xffffffffu, b1 ? k0 : k1, 2));
  kk = max2(kk, __shfl_xor_sync(0xffffffffu, kk, 4));  // lanes i & 3 and (i & 3) + 4, complete
  const uint32_t ko = __shfl_xor_sync(0xffffffffu, kk, 2);
  const uint32_t r0 = b1 ? ko : kk, r1 = b1 ? kk : ko;  // words (i & 1) and (i & 1) + 2
  const uint32_t o0 = __shfl_xor_sync(0xffffffffu, r0, 1), o1 = __shfl_xor_sync(0xffffffffu, r1, 1);
  w[0] = b0 ? o0 : r0;
  w[1] = b0 ? r0 : o0;
  w[2] = b0 ? o1 : r1;
  w[3] = b0 ? r1 : o1;
  // The lanes' weights 2^((x - lm) c), by one multiply-add each unless one of the warp's lanes
  // is past that (one vote for 8 vectors; a test for each took 54.9 us instead of 53.4). A NaN
  // logit makes its lane's sum NaN (tested once per lane below), except in a lane with no
  // finite maximum, whose words are tested here.
  float ls[8];
  auto sums = [&](auto fused) {
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const float lm = k < 4 ? lo_f(w[k & 3]) : hi_f(w[k & 3]);
      const uint32_t wv[4] = {dv[k].x, dv[k].y, dv[k].z, dv[k].w};
      const float nlc = -lm * c;
      float sum = 0.f;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const uint64_t x = pack2(lo_f(wv[q]), hi_f(wv[q]));
        float e0, e1;
        unpack2(decltype(fused)::value ? fma2(x, pack2(c, c), pack2(nlc, nlc))
                                       : mul2(add2(x, pack2(-lm, -lm)), pack2(c, c)), e0, e1);
        sum += ex2(e0);
        sum += ex2(e1);
      }
      if (lm == -INFINITY) {
        sum = 0.f;
#pragma unroll
        for (int q = 0; q < 4; ++q) nacc |= (wv[q] & 0x7FFF7FFFu) + 0x007F007Fu;
      }
      ls[k] = sum;
    }
  };
  if (__any_sync(0xffffffffu, past_fused(b2 ? hi_f(kk) : lo_f(kk), c))) sums(std::false_type{});
  else sums(std::true_type{});
  const float s = reduce8<8>(ls, i, [](float x, float y) { return x + y; });
  const int vi = v0 + i * kThreads + (tid & ~7);  // the first vector of lane k = i
  if (vi < vend) {
    lanes[lane_at(vi / 8 - l0, n)] = make_float2(b2 ? hi_f(kk) : lo_f(kk), s);
    bad |= s != s;
  }
}

// One block per (split, drafter row, sequence).
template <bool BF16, bool VEC>
__global__ void __launch_bounds__(kThreads, 8) draft_sample_kernel(DraftParams p) {
  extern __shared__ __align__(16) unsigned char dsm[];
  float2* lanes = reinterpret_cast<float2*>(dsm);
  __shared__ unsigned long long s_red[kThreads / 32];
  __shared__ float s_scan[kThreads / 32 + 1];
  __shared__ int s_bad, s_last, s_pick, s_lastpos, s_tok;
  __shared__ float s_base, s_q;

  const int split = blockIdx.x, j = blockIdx.y, b = blockIdx.z, tid = threadIdx.x;
  const int gamma = p.gamma, V = p.vocab, LE = p.lane_elems, nlanes = p.nlanes;
  const int64_t rid = static_cast<int64_t>(b) * gamma + j;
  const char* rowp = static_cast<const char*>(p.drafter) + rid * V * (BF16 ? 2 : 4);
  const float T = p.temperature[b];
  const bool greedy = !(T > 0.f);
  const float c = greedy ? 0.f : kLog2e / T;
  const float u = p.uniforms[rid];
  const int l0 = split * p.lanes_per_split;
  const int l1 = min(nlanes, l0 + p.lanes_per_split);
  const int e_begin = l0 * LE, e_end = min(V, l1 * LE);
  if (tid == 0) s_bad = 0;

  // 1. scan: the maximum (with its lowest index) and, tempered, every lane's (m_i, s_i)
  float m = -INFINITY;
  int a = INT_MAX;
  bool bad = false;
  if (VEC) {
    constexpr int kEpv = BF16 ? 8 : 4;
    constexpr int kGroup = 64 / kEpv;  // threads (vectors) per 64-element lane
    const uint32_t ninf = BF16 ? 0xFF80FF80u : 0xFF800000u;
    const uint32_t nan_mask = BF16 ? 0x7FFF7FFFu : 0x7FFFFFFFu;
    const uint32_t nan_add = BF16 ? 0x007F007Fu : 0x007FFFFFu;
    const uint32_t nan_top = BF16 ? 0x80008000u : 0x80000000u;
    const int vbeg = e_begin / kEpv, vend = e_end / kEpv;
    const uint4* rv = reinterpret_cast<const uint4*>(rowp);
    uint32_t nacc = 0;
    if (vbeg + tid < vend) a = (vbeg + tid) * kEpv;
    for (int v0 = vbeg; v0 < vend; v0 += kThreads * kUnroll) {
      uint4 dv[kUnroll];
#pragma unroll
      for (int k = 0; k < kUnroll; ++k) {
        const int vi = v0 + k * kThreads + tid;
        dv[k] = vi < vend ? __ldg(rv + vi) : make_uint4(ninf, ninf, ninf, ninf);
      }
      if constexpr (BF16) scan_bf16(dv, v0, vend, l0, l1 - l0, c, greedy, lanes, m, a, nacc, bad);
      float lm[kUnroll];
#pragma unroll
      for (int k = 0; k < (BF16 ? 0 : kUnroll); ++k) {
        const int vi = v0 + k * kThreads + tid;
        const uint32_t wv[4] = {dv[k].x, dv[k].y, dv[k].z, dv[k].w};
        float x[kEpv];
#pragma unroll
        for (int q = 0; q < kEpv; ++q)
          x[q] = BF16 ? __uint_as_float((q & 1) ? (wv[q >> 1] & 0xffff0000u) : (wv[q >> 1] << 16))
                      : __uint_as_float(wv[q]);
        if (greedy) {
#pragma unroll
          for (int q = 0; q < 4; ++q) nacc |= (wv[q] & nan_mask) + nan_add;
#pragma unroll
          for (int q = 0; q < kEpv; ++q)
            if (x[q] > m) { m = x[q]; a = vi * kEpv + q; }
        } else {
          lm[k] = x[0];
#pragma unroll
          for (int q = 1; q < kEpv; ++q) lm[k] = fmaxf(lm[k], x[q]);
          m = fmaxf(m, lm[k]);
        }
      }
      if (!BF16 && !greedy) {  // the 16 threads of a lane's vectors, 8 lanes at a time
        const int i = tid & 7;
        const float mine = reduce8<kGroup>(lm, i, [](float x, float y) { return fmaxf(x, y); });
        gather8(mine, i, lm);
        float ls[kUnroll];
        auto sums = [&](auto fused) {  // (as in scan_bf16)
#pragma unroll
          for (int k = 0; k < kUnroll; ++k) {
            const uint32_t wv[4] = {dv[k].x, dv[k].y, dv[k].z, dv[k].w};
            ls[k] = 0.f;
            if (lm[k] != -INFINITY) {
              const float nlc = -lm[k] * c;
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                const float x = __uint_as_float(wv[q]);
                ls[k] += ex2(decltype(fused)::value ? fmaf(x, c, nlc) : (x - lm[k]) * c);
              }
            } else {
#pragma unroll
              for (int q = 0; q < 4; ++q) nacc |= (wv[q] & nan_mask) + nan_add;
            }
          }
        };
        if (__any_sync(0xffffffffu, past_fused(mine, c))) sums(std::false_type{});
        else sums(std::true_type{});
        const float sum = reduce8<kGroup>(ls, i, [](float x, float y) { return x + y; });
        const int vi = v0 + i * kThreads + (tid & ~(kGroup - 1));  // the first vector of lane i
        if ((tid & 8) == 0 && vi < vend) {
          lanes[lane_at(vi / kGroup - l0, l1 - l0)] = make_float2(mine, sum);
          bad |= sum != sum;
        }
      }
    }
    bad |= (nacc & nan_top) != 0;
  } else {
    // Rows not 16-byte aligned: the granules that cover kStage elements come into shared
    // memory with 16-byte loads, four a thread, and the elements are read from there
    // (element loads kept 16 KB in flight on an SM: 87.9 us for 256 rows of 100,003 bf16
    // logits, now 57.7).
    constexpr int E = BF16 ? 2 : 4;
    constexpr int kStage = kStageGranules * 16 / E;
    uint4* stage = reinterpret_cast<uint4*>(dsm + (static_cast<size_t>(nlanes) * 8 + 15) / 16 * 16);
    const char* lo = static_cast<const char*>(p.drafter);
    const char* hi = lo + static_cast<int64_t>(p.batch) * gamma * V * E;
    if (e_begin + tid < e_end) a = e_begin + tid;
    for (int h0 = e_begin; h0 < e_end; h0 += kStage) {
      const char* from = rowp + static_cast<int64_t>(h0) * E;
      const uint32_t off = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(from)) & 15u;
      const int ngran = (min(kStage, e_end - h0) * E + static_cast<int>(off) + 15) / 16;
      uint4 g[kStageGranules / kThreads];
      load_granules<E, kStageGranules / kThreads>(g, from - off, tid, kThreads, min(ngran, kStageGranules), lo, hi);
      const uint4 last = tid == 0 && ngran > kStageGranules
                             ? load_granule<E>(from - off + 16 * kStageGranules, lo, hi) : make_uint4(0, 0, 0, 0);
      __syncthreads();  // the previous stage has been read
#pragma unroll
      for (int k = 0; k < kStageGranules / kThreads; ++k) stage[k * kThreads + tid] = g[k];
      if (tid == 0) stage[kStageGranules] = last;
      __syncthreads();
      const char* sm = reinterpret_cast<const char*>(stage) + off;
      for (int e0 = h0; e0 < min(h0 + kStage, e_end); e0 += kThreads * kUnroll) {
        float x[kUnroll];
#pragma unroll
        for (int k = 0; k < kUnroll; ++k) {
          const int ei = e0 + k * kThreads + tid;
          const char* at = sm + (ei - h0) * E;
          x[k] = ei < e_end ? (BF16 ? bf16_bits_to_f32(*reinterpret_cast<const uint16_t*>(at))
                                    : *reinterpret_cast<const float*>(at))
                            : -INFINITY;
          bad |= x[k] != x[k];
        }
        if (greedy) {
#pragma unroll
          for (int k = 0; k < kUnroll; ++k)
            if (x[k] > m) { m = x[k]; a = e0 + k * kThreads + tid; }
        } else {
          // a warp's 32 consecutive elements are one lane
          const int i = tid & 7;
          float lm[kUnroll], ls[kUnroll];
#pragma unroll
          for (int k = 0; k < kUnroll; ++k) {
            m = fmaxf(m, x[k]);
            lm[k] = x[k];
          }
          const float mine = reduce8<32>(lm, i, [](float y, float z) { return fmaxf(y, z); });
          gather8(mine, i, lm);
#pragma unroll
          for (int k = 0; k < kUnroll; ++k) ls[k] = lm[k] != -INFINITY ? exp2f((x[k] - lm[k]) * c) : 0.f;
          const float sum = reduce8<32>(ls, i, [](float y, float z) { return y + z; });
          const int ei = e0 + i * kThreads + (tid & ~31);  // the first element of lane i
          if ((tid & 31) < 8 && ei < e_end) lanes[lane_at(ei / 32 - l0, l1 - l0)] = make_float2(mine, sum);
        }
      }
    }
  }
  if (!greedy && m == INFINITY) bad = true;  // +inf leaves the softmax undefined
  unsigned long long best = cand_of(m, static_cast<uint32_t>(a));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long y = __shfl_xor_sync(0xffffffffu, best, o);
    best = y > best ? y : best;
  }
  if (bad) s_bad = 1;
  if ((tid & 31) == 0) s_red[tid >> 5] = best;
  __syncthreads();
  best = s_red[0];
#pragma unroll
  for (int k = 1; k < kThreads / 32; ++k) best = s_red[k] > best ? s_red[k] : best;

  if (p.splits > 1) {
    // publish this split; the row's last block continues with the whole row
    if (!greedy)
      for (int i = tid; i < l1 - l0; i += kThreads) p.lanes_g[rid * nlanes + l0 + i] = lanes[lane_at(i, l1 - l0)];
    if (tid == 0)
      p.parts[rid * p.splits + split] = make_uint4(static_cast<uint32_t>(best), static_cast<uint32_t>(best >> 32),
                                                   static_cast<uint32_t>(s_bad), 0u);
    __threadfence();
    __syncthreads();
    if (tid == 0) {
      const uint32_t prev = atomicAdd(&p.row_tickets[rid], 1u);
      s_last = prev == static_cast<uint32_t>(p.splits - 1);
      if (s_last) p.row_tickets[rid] = 0;  // leave the counter at zero for the next call
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    if (!greedy)
      for (int i = tid; i < nlanes; i += kThreads) lanes[lane_at(i, nlanes)] = __ldcg(p.lanes_g + rid * nlanes + i);
    best = 0ull;
    uint32_t anybad = 0;
    for (int k = tid; k < p.splits; k += kThreads) {
      const uint4 q = __ldcg(p.parts + rid * p.splits + k);
      const unsigned long long cq = (static_cast<unsigned long long>(q.y) << 32) | q.x;
      best = cq > best ? cq : best;
      anybad |= q.z;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long y = __shfl_xor_sync(0xffffffffu, best, o);
      best = y > best ? y : best;
    }
    anybad = __reduce_or_sync(0xffffffffu, anybad);
    __syncthreads();
    if ((tid & 31) == 0) s_red[tid >> 5] = best;
    if (tid == 0) s_bad = 0;
    __syncthreads();
    if ((tid & 31) == 0 && anybad) s_bad = 1;
    __syncthreads();
    best = s_red[0];
#pragma unroll
    for (int k = 1; k < kThreads / 32; ++k) best = s_red[k] > best ? s_red[k] : best;
  }

  // 2. the row's token
  const float M = __uint_as_float((static_cast<uint32_t>(best >> 32) & 0x80000000u)
                                      ? (static_cast<uint32_t>(best >> 32) & 0x7fffffffu)
                                      : ~static_cast<uint32_t>(best >> 32));
  uint32_t flag = s_bad ? kBadRow : 0u;
  if (!greedy && !(M > -INFINITY)) flag = kBadRow;  // no finite logit
  int tok = -1;
  float q = NAN;
  if (!flag && greedy) {
    tok = cand_idx(best);
    q = 1.f;
  } else if (!flag) {
    // cumulative mass at lane boundaries: each thread takes a contiguous run of lanes
    const int per = (nlanes + kThreads - 1) / kThreads;
    const int i0 = min(nlanes, tid * per), i1 = min(nlanes, i0 + per);
    float mine = 0.f;
    for (int i = i0; i < i1; ++i) {  // each lane's scale to the row's maximum replaces its own
      float2& ms = lanes[lane_at(i, nlanes)];
      ms.x = ms.x != -INFINITY ? exp2f((ms.x - M) * c) : 0.f;
      mine = fmaf(ms.y, ms.x, mine);
    }
    float S = 0.f;
    const float base = block_excl_scan(mine, s_scan, &S);
    if (tid == 0) {
      s_pick = INT_MAX;
      s_lastpos = -1;
    }
    __syncthreads();
    const float target = u * S;
    float run = base;
    int lastpos = -1;
    for (int i = i0; i < i1; ++i) {
      const float2 ms = lanes[lane_at(i, nlanes)];
      const float w = __fmul_rn(ms.y, ms.x);
      run += w;
      if (w > 0.f) {
        lastpos = i;
        if (run >= target) {
          atomicMin(&s_pick, i);
          break;
        }
      }
    }
    // the last lane with mass, for a row that no lane crosses (one atomic a warp)
    lastpos = __reduce_max_sync(0xffffffffu, lastpos);
    if ((tid & 31) == 0) atomicMax(&s_lastpos, lastpos);
    __syncthreads();
    const bool crossed = s_pick != INT_MAX;
    const int lane_sel = crossed ? s_pick : s_lastpos;
    if (lane_sel >= i0 && lane_sel < i1) {  // the owner of that lane: its mass before it
      float before = base;
      for (int i = i0; i < lane_sel; ++i) {
        const float2 ms = lanes[lane_at(i, nlanes)];
        before = fmaf(ms.y, ms.x, before);
      }
      s_base = before;
    }
    __syncthreads();
    // warp 0 rescans the lane: element e = lane_sel * LE + 2 * lane + k (k = 0, 1)
    if (tid < 32) {
      const int e0 = lane_sel * LE + 2 * tid;
      float w[2] = {0.f, 0.f};
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int e = e0 + k;
        if (2 * tid + k < LE && e < V) w[k] = exp2f((load_elem<BF16>(rowp, e) - M) * c);
      }
      float incl = w[0] + w[1];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const float y = __shfl_up_sync(0xffffffffu, incl, o);
        if (tid >= o) incl += y;
      }
      const float before = s_base + incl - (w[0] + w[1]);
      int hit = -1, lastk = -1;
      if (w[0] > 0.f) { lastk = 0; if (before + w[0] >= target) hit = 0; }
      if (w[1] > 0.f) { lastk = 1; if (hit < 0 && before + w[0] + w[1] >= target) hit = 1; }
      const unsigned hm = __ballot_sync(0xffffffffu, hit >= 0);
      const unsigned lm = __ballot_sync(0xffffffffu, lastk >= 0);
      int t = -1;
      float wt = 0.f;
      if (crossed && hm) {
        const int src = __ffs(hm) - 1;
        if (tid == src) { t = e0 + hit; wt = w[hit]; }
        t = __shfl_sync(0xffffffffu, t, src);
        wt = __shfl_sync(0xffffffffu, wt, src);
      } else if (lm) {  // rounding left u * S above every sum: the last positive weight
        const int src = 31 - __clz(lm);
        if (tid == src) { t = e0 + lastk; wt = w[lastk]; }
        t = __shfl_sync(0xffffffffu, t, src);
        wt = __shfl_sync(0xffffffffu, wt, src);
      }
      if (tid == 0) {
        s_tok = t;
        s_q = fminf(wt / S, 1.f);  // S may be rounded below its only weight
      }
    }
    __syncthreads();
    tok = s_tok;
    q = s_q;
    if (tok < 0) flag = kBadRow;
  }
  if (tid == 0) {
    p.tokens[rid] = flag ? -1 : tok;
    if (p.q_tok) p.q_tok[rid] = flag ? NAN : q;
    p.row_flags[rid] = flag;
  }

  // 3. the sequence's last block: a sequence with a bad row draws nothing
  __threadfence();
  __syncthreads();
  if (tid == 0) {
    const uint32_t prev = atomicAdd(&p.tickets[b], 1u);
    s_last = prev == static_cast<uint32_t>(gamma - 1);
    if (s_last) p.tickets[b] = 0;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  if (tid == 0) s_bad = 0;
  __syncthreads();
  for (int k = tid; k < gamma; k += kThreads)
    if (__ldcg(p.row_flags + static_cast<int64_t>(b) * gamma + k)) s_bad = 1;
  __syncthreads();
  if (s_bad) {
    for (int k = tid; k < gamma; k += kThreads) {
      p.tokens[static_cast<int64_t>(b) * gamma + k] = -1;
      if (p.q_tok) p.q_tok[static_cast<int64_t>(b) * gamma + k] = NAN;
    }
    if (tid == 0) set_status(p.status, SPEC_FLAG_BAD_LOGITS);
  }
}

template <bool BF16, bool VEC>
cudaError_t launch_draft_typed(const DraftParams& p, size_t smem, cudaStream_t stream) {
  if (!VEC) smem = (smem + 15) / 16 * 16 + (kStageGranules + 1) * 16;  // the stage of unaligned rows
  if (smem > 48 * 1024) {
    const cudaError_t e = allow_smem(draft_sample_kernel<BF16, VEC>,
                                     kDraftMaxSmem + (VEC ? 0 : (kStageGranules + 1) * 16));
    if (e != cudaSuccess) return e;
  }
  draft_sample_kernel<BF16, VEC><<<dim3(p.splits, p.gamma, p.batch), kThreads, smem, stream>>>(p);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------------
// KV commit
// ---------------------------------------------------------------------------------
constexpr int kCommitThreads = 1024;

__device__ __forceinline__ int block_excl_scan_int(int x, int* sh, int* total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int in = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, in, o);
    if (lane >= o) in += y;
  }
  if (lane == 31) sh[w] = in;
  __syncthreads();
  if (threadIdx.x == 0) {
    int run = 0;
    for (int k = 0; k < kCommitThreads / 32; ++k) {
      const int t = sh[k];
      sh[k] = run;
      run += t;
    }
    sh[kCommitThreads / 32] = run;
  }
  __syncthreads();
  const int ex = sh[w] + in - x;
  *total = sh[kCommitThreads / 32];
  __syncthreads();
  return ex;
}

__global__ void __launch_bounds__(kCommitThreads) commit_kv_kernel(spec_commit_args_t a) {
  __shared__ int s_scan[kCommitThreads / 32 + 1];
  __shared__ int s_used;
  const int tid = threadIdx.x, P = a.page_size, G = a.gamma, MP = a.max_pages_per_seq;
  const int count0 = *a.free_count;
  if (tid == 0) s_used = 0;
  int carry = 0;  // pages asked (reserve) or offered (release) by earlier sequences
  for (int b0 = 0; b0 < a.batch; b0 += kCommitThreads) {
    const int b = b0 + tid;
    int flag = 0, kv = 0, nl = 0, have = 0, cnt = 0, from = 0;
    if (b < a.batch) {
      kv = a.kv_len[b];
      const int na = a.num_accepted[b];
      if (kv < G || kv > MP * P || na < -1 || na > G - 1) {
        flag = 1;
      } else {
        nl = kv - G + (na >= 0 ? na + 1 : 0);
        have = (kv + P - 1) / P;
        if (a.reserve) {
          const int want = (nl + G + P - 1) / P;
          if (want > MP) flag = 2;
          else { cnt = want - have; from = have; }
        } else {
          const int keep = (nl + P - 1) / P;
          cnt = have - keep;
          from = keep;
        }
      }
    }
    int total = 0;
    const int before = carry + block_excl_scan_int(cnt, s_scan, &total);
    carry += total;
    if (b < a.batch && flag == 0 && cnt > 0) {
      int32_t* row = a.page_table + static_cast<int64_t>(b) * MP;
      if (a.reserve) {
        if (before + cnt > count0) {
          flag = 2;
        } else {
          for (int i = 0; i < cnt; ++i) row[from + i] = a.free_pages[count0 - 1 - before - i];
          atomicMax(&s_used, before + cnt);
        }
      } else {
        if (count0 + before + cnt > a.free_capacity) {
          flag = 2;
        } else {
          for (int i = 0; i < cnt; ++i) {
            a.free_pages[count0 + before + i] = row[from + i];
            row[from + i] = -1;
          }
          atomicMax(&s_used, before + cnt);
        }
      }
    }
    if (b < a.batch) {
      if (flag != 1) a.kv_len[b] = nl;
      if (a.flags) a.flags[b] = flag;
    }
  }
  __syncthreads();
  if (tid == 0) *a.free_count = a.reserve ? count0 - s_used : count0 + s_used;
}

}  // namespace

cudaError_t launch_draft(const spec_draft_args_t& a, const DraftLayout& L, char* ws,
                         cudaStream_t stream, bool vec) {
  DraftParams p;
  p.batch = a.batch;
  p.gamma = a.gamma;
  p.vocab = a.vocab;
  p.lane_elems = L.lane_elems;
  p.nlanes = L.nlanes;
  p.splits = L.splits;
  p.lanes_per_split = L.lanes_per_split;
  p.drafter = a.drafter_logits;
  p.temperature = a.temperature;
  p.uniforms = a.uniforms;
  p.tokens = a.block_tokens;
  p.q_tok = a.q_tok;
  p.status = reinterpret_cast<uint32_t*>(ws);
  p.tickets = reinterpret_cast<uint32_t*>(ws + L.tickets);
  p.row_flags = reinterpret_cast<uint32_t*>(ws + L.row_flags);
  p.row_tickets = reinterpret_cast<uint32_t*>(ws + L.row_tickets);
  p.lanes_g = reinterpret_cast<float2*>(ws + L.lanes_g);
  p.parts = reinterpret_cast<uint4*>(ws + L.parts);
  (void)cudaGetLastError();
  if (a.logits_dtype == SPEC_BF16)
    return vec ? launch_draft_typed<true, true>(p, L.smem, stream)
               : launch_draft_typed<true, false>(p, L.smem, stream);
  return vec ? launch_draft_typed<false, true>(p, L.smem, stream)
             : launch_draft_typed<false, false>(p, L.smem, stream);
}

cudaError_t launch_commit(const spec_commit_args_t& a, cudaStream_t stream) {
  (void)cudaGetLastError();
  commit_kv_kernel<<<1, kCommitThreads, 0, stream>>>(a);
  return cudaGetLastError();
}

}  // namespace specv
