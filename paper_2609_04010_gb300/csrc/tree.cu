// Tree verification (Sec. 4.2: more than one candidate is verified at once as a prefix
// tree under tree attention; Sec. 3.3, "Tree Sampler"): the tree sampler that builds the
// candidate tree from the drafter's rows, greedy acceptance along it, and the
// compaction of the accepted path's keys and values.
//
// tree_greedy_kernel (tree acceptance): grid (splits, nodes, sequences) of 128-thread
// blocks. Each block finds the lowest-index argmax of its part of a node's target row
// and, for a tempered sequence, the part's sum of 2^((l - max) log2e / T); the
// sequence's last block (ticket) merges the parts of all rows and walks the tree from the
// root. Greedy: to the child whose token is the current node's argmax.
// Sampled: the children are tried in node order as point-mass proposals (accepted iff
// u <= p'(token), p' without the siblings rejected before), decided in fp64 from the
// gathered logits; every node's test is taken before the walk, which is a ballot per
// step. After the last rejection the block draws the final token from p' by inverse CDF:
// the part where the remaining mass crosses u x total, from the stored part sums minus
// the rejected tokens' weights, then one pass over that part.
//
// tree_compact_kernel: one block per (cache, KV head, sequence) moves the accepted
// path's key or value rows into consecutive positions after the context.
#include <cuda_bf16.h>

#include <algorithm>
#include <cfloat>
#include <climits>
#include <cmath>

#include "common.cuh"

namespace specv {

// Row blocks of the tree acceptance kernel resident per SM (80 registers a thread).
constexpr int kTreeBlocksPerSm = 6;

TreeLayout tree_layout(int batch, int nodes, int vocab, size_t base, int sms, bool vec) {
  TreeLayout L;
  const int lane = vec ? 64 : 32;
  const int nlanes = (vocab + lane - 1) / lane;
  const int64_t rows = static_cast<int64_t>(batch) * nodes;
  int64_t splits = (static_cast<int64_t>(kTreeBlocksPerSm) * sms + rows - 1) / rows;
  splits = splits < 1 ? 1 : (splits > kFiltMaxSplits ? kFiltMaxSplits : splits);
  if (splits > nlanes) splits = nlanes;
  L.elems_per_split = static_cast<int>((nlanes + splits - 1) / splits) * lane;
  L.splits = (vocab + L.elems_per_split - 1) / L.elems_per_split;
  L.tickets = base;
  L.parts = ws_round(L.tickets + sizeof(uint32_t) * batch);
  L.end = ws_round(L.parts + 16 * rows * L.splits);
  return L;
}

namespace {

constexpr int kThreads = 128;
constexpr int kUnroll = 8;

struct TreeParams {
  int batch, nodes, vocab, splits, elems_per_split;
  const void* target;
  const int32_t* tokens;   // [batch][nodes]
  const int32_t* parents;  // [batch][nodes]
  int32_t* path;           // [batch][nodes]
  int32_t* num_accepted;   // [batch]
  int32_t* out_tokens;     // [batch][nodes + 1]
  int32_t* num_emitted;    // [batch]
  uint32_t* status;
  uint32_t* tickets;
  uint4* parts;
  const float* temperature;  // [batch] or NULL (greedy)
  const float* uniforms;     // [batch][nodes]
};

template <bool BF16>
__device__ __forceinline__ float load_elem(const void* base, int64_t i) {
  if (BF16) return bf16_bits_to_f32(static_cast<const uint16_t*>(base)[i]);
  return static_cast<const float*>(base)[i];
}

__device__ __forceinline__ uint32_t order_key(float x) {
  uint32_t f = __float_as_uint(x);
  if (f == 0x80000000u) f = 0u;
  return (f & 0x80000000u) ? ~f : (f | 0x80000000u);
}
// The float whose order_key is k.
__device__ __forceinline__ float key_to_float(uint32_t k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}
// 2^((x - m) * c) for a running reference m (an all -inf prefix has m = -inf and weight 0).
__device__ __forceinline__ float rel_weight(float x, float m, float c) {
  return m == -INFINITY ? 0.f : ex2((x - m) * c);
}

template <bool BF16, bool VEC>
__global__ void __launch_bounds__(kThreads, kTreeBlocksPerSm) tree_greedy_kernel(TreeParams p) {
  __shared__ unsigned long long s_red[kThreads / 32];
  __shared__ float s_fsum[kThreads / 32];
  __shared__ int s_bad, s_last;
  // the sequence's last block: its rows' argmax, (max, sum) and parts (max, sum), its nodes
  __shared__ int s_arg[64], s_tok_in[64], s_par[64], s_acc[64];
  __shared__ float2 s_stat[64], s_part[64 * 16];
  __shared__ double s_e[64];
  __shared__ uint32_t s_badin;
  __shared__ int s_lo, s_hi;
  __shared__ double s_excl;
  // hand-off from the walking warp to the sampled final draw
  __shared__ int s_final, s_len, s_nrm, s_kcross, s_tok;
  __shared__ int s_rm[64];                 // tokens rejected at the final node, ascending
  __shared__ float s_rmw[64];              // their weights 2^((l - M) log2e / T)
  __shared__ int s_rmk[64];                // their parts of the row
  __shared__ double s_target, s_dsum[kThreads / 32];
  const int split = blockIdx.x, j = blockIdx.y, b = blockIdx.z, tid = threadIdx.x;
  const int N = p.nodes, V = p.vocab;
  const int64_t rid = static_cast<int64_t>(b) * N + j;
  const char* rowp = static_cast<const char*>(p.target) + rid * V * (BF16 ? 2 : 4);
  const int e_begin = split * p.elems_per_split, e_end = min(V, e_begin + p.elems_per_split);
  const float T = p.temperature ? p.temperature[b] : 0.f;
  const bool tempered = T > 0.f;
  const float cs = tempered ? kLog2e / T : 0.f;
  if (tid == 0) s_bad = 0;
  __syncthreads();

  // the lowest-index maximum of this part of the row and, for a tempered sequence, the
  // sum of 2^((l - max) log2e / T) over it (rescaled whenever the running maximum grows)
  float m = -INFINITY, sum = 0.f;
  int a = INT_MAX;
  bool bad = false;
  if (VEC) {
    constexpr int kEpv = BF16 ? 8 : 4;
    const uint32_t ninf = BF16 ? 0xFF80FF80u : 0xFF800000u;
    const int vbeg = e_begin / kEpv, vend = e_end / kEpv;
    const uint4* rv = reinterpret_cast<const uint4*>(rowp);
    if (vbeg + tid < vend) a = (vbeg + tid) * kEpv;
    for (int v0 = vbeg; v0 < vend; v0 += kThreads * kUnroll) {
      uint4 dv[kUnroll];
#pragma unroll
      for (int k = 0; k < kUnroll; ++k) {
        const int vi = v0 + k * kThreads + tid;
        dv[k] = vi < vend ? __ldg(rv + vi) : make_uint4(ninf, ninf, ninf, ninf);
      }
      auto val = [&](int k, int q) {
        const uint32_t wv[4] = {dv[k].x, dv[k].y, dv[k].z, dv[k].w};
        return BF16 ? __uint_as_float((q & 1) ? (wv[q >> 1] & 0xffff0000u) : (wv[q >> 1] << 16))
                    : __uint_as_float(wv[q]);
      };
      const float m_old = m;
#pragma unroll
      for (int k = 0; k < kUnroll; ++k) {
        const int vi = v0 + k * kThreads + tid;
#pragma unroll
        for (int q = 0; q < kEpv; ++q) {
          const float x = val(k, q);
          bad |= x != x || (tempered && x == INFINITY);
          if (x > m) { m = x; a = vi * kEpv + q; }
        }
      }
      if (tempered) {
        sum = m_old == -INFINITY ? 0.f : sum * ex2((m_old - m) * cs);
#pragma unroll
        for (int k = 0; k < kUnroll; ++k)
#pragma unroll
          for (int q = 0; q < kEpv; ++q) sum += rel_weight(val(k, q), m, cs);
      }
    }
  } else {
    if (e_begin + tid < e_end) a = e_begin + tid;
    for (int e0 = e_begin; e0 < e_end; e0 += kThreads * kUnroll) {
      float x[kUnroll];
#pragma unroll
      for (int k = 0; k < kUnroll; ++k) {
        const int ei = e0 + k * kThreads + tid;
        x[k] = ei < e_end ? load_elem<BF16>(rowp, ei) : -INFINITY;
      }
      const float m_old = m;
#pragma unroll
      for (int k = 0; k < kUnroll; ++k) {
        bad |= x[k] != x[k] || (tempered && x[k] == INFINITY);
        if (x[k] > m) { m = x[k]; a = e0 + k * kThreads + tid; }
      }
      if (tempered) {
        sum = m_old == -INFINITY ? 0.f : sum * ex2((m_old - m) * cs);
#pragma unroll
        for (int k = 0; k < kUnroll; ++k) sum += rel_weight(x[k], m, cs);
      }
    }
  }
  unsigned long long best = (static_cast<unsigned long long>(order_key(m)) << 32) |
                            (0xffffffffu - static_cast<uint32_t>(a));
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
  float part_sum = 0.f;
  if (tempered) {
    // the part's sum relative to its maximum
    const float pm = key_to_float(static_cast<uint32_t>(best >> 32));
    float v = (pm == -INFINITY || !(pm < INFINITY)) ? 0.f : sum * rel_weight(m, pm, cs) * (m == -INFINITY ? 0.f : 1.f);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();  // s_red is read above by every thread
    if ((tid & 31) == 0) s_fsum[tid >> 5] = v;
    __syncthreads();
    for (int k = 0; k < kThreads / 32; ++k) part_sum += s_fsum[k];
  }

  // The sequence's last block (one ticket for all parts of all its rows: a ticket per row
  // and another per sequence were two fences and atomics in a row) has every row's parts.
  if (tid == 0) {
    p.parts[rid * p.splits + split] = make_uint4(static_cast<uint32_t>(best), static_cast<uint32_t>(best >> 32),
                                                 static_cast<uint32_t>(s_bad), __float_as_uint(part_sum));
    __threadfence();
    const uint32_t prev = atomicAdd(&p.tickets[b], 1u);
    s_last = prev == static_cast<uint32_t>(N * p.splits - 1);
    if (s_last) p.tickets[b] = 0;  // leave the counter at zero for the next call
    s_final = -1;
    s_badin = 0;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  const int64_t brow = static_cast<int64_t>(b) * N;
  {
    // 16 threads per row, a part each (at most kFiltMaxSplits = 16), 8 rows at a time; all
    // loads in flight together
    const int k = tid & 15, g = tid >> 4;
    uint4 q[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int row = g + 8 * i;
      q[i] = row < N && k < p.splits ? __ldcg(p.parts + (brow + row) * p.splits + k) : make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int row = g + 8 * i;
      if (8 * i >= N) break;
      unsigned long long bb = (static_cast<unsigned long long>(q[i].y) << 32) | q[i].x;
      uint32_t rbad = q[i].z;
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) {
        const unsigned long long y = __shfl_xor_sync(0xffffffffu, bb, o);
        bb = y > bb ? y : bb;
        rbad |= __shfl_xor_sync(0xffffffffu, rbad, o);
      }
      const float M = key_to_float(static_cast<uint32_t>(bb >> 32)), pm = key_to_float(q[i].y);
      const float pw = __uint_as_float(q[i].w);
      // the row's sum relative to its maximum
      float z = tempered && M > -INFINITY && M < INFINITY && k < p.splits ? pw * rel_weight(pm, M, cs) : 0.f;
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
      if (row < N) {
        s_part[row * 16 + k] = make_float2(pm, pw);
        if (k == 0) {
          // a tempered row needs a finite maximum (NaN and +inf are flagged by its parts)
          const bool unusable = rbad != 0 || (tempered && !(M > -INFINITY));
          s_arg[row] = unusable ? -1 : static_cast<int>(0xffffffffu - static_cast<uint32_t>(bb));
          s_stat[row] = make_float2(M, z);
        }
      }
    }
  }
  int32_t* path = p.path + brow;
  int32_t* out = p.out_tokens + static_cast<int64_t>(b) * (N + 1);
  // thread c < N holds node c
  const int c = tid;
  const int tok = c < N ? p.tokens[brow + c] : -1, par = c < N ? p.parents[brow + c] : -2;
  const float uc = tempered && c < N ? p.uniforms[brow + c] : 1.f;
  if (c < 64) {
    s_tok_in[c] = tok;
    s_par[c] = par;
  }
  __syncthreads();
  if (c < N) {
    uint32_t bad_in = 0;
    if (tok < 0 || tok >= V) bad_in |= SPEC_FLAG_BAD_TOKEN;
    if (c == 0 ? par != -1 : (par < 0 || par >= c)) bad_in |= SPEC_FLAG_BAD_TREE;
    if (s_arg[c] < 0) bad_in |= SPEC_FLAG_BAD_LOGITS;
    if (bad_in) atomicOr(&s_badin, bad_in);
  }
  __syncthreads();
  if (s_badin) {
    for (int i = tid; i < N; i += kThreads) path[i] = -1;
    for (int i = tid; i <= N; i += kThreads) out[i] = -1;
    if (tid == 0) {
      p.num_accepted[b] = -1;
      p.num_emitted[b] = 0;
      set_status(p.status, s_badin);
    }
    return;
  }
  // Sampled walk: the children of a node, in node order, are point-mass proposals; child c
  // is accepted iff u[c] <= p'(token), p' the node's target distribution without the tokens
  // of the siblings rejected before it. Whether a node is accepted when its turn comes does
  // not depend on the walk, so every node's test is taken at once, a thread each: its
  // weight e_c = exp((l(t_c) - M) / T) in fp64 under its parent's row (M that row's
  // maximum; 0 for a repeated sibling token, removed with its first occurrence), the weight
  // of its earlier siblings in node order, and u[c] (S - earlier) <= e_c. The walk is then
  // a ballot per step (with fp64 prefix scans and a division per step, on the one warp
  // that held the tree, it took 8.7 us of the kernel's 30).
  const char* tbase = static_cast<const char*>(p.target);
  const size_t rbytes = static_cast<size_t>(V) * (BF16 ? 2 : 4);
  bool live = false, acc = false;
  if (tempered) {
    const bool child = c >= 1 && c < N;
    double e = 0.0;
    if (child) {
      const float x = load_elem<BF16>(tbase + (brow + par) * rbytes, tok);
      e = exp((static_cast<double>(x) - s_stat[par].x) / static_cast<double>(T));
      bool dup = false;
#pragma unroll 8
      for (int o = 1; o < c; ++o) dup |= s_par[o] == par && s_tok_in[o] == tok;
      if (dup) e = 0.0;
      s_e[c] = e;
    }
    __syncthreads();
    if (child) {
      double earlier = 0.0;
#pragma unroll 8
      for (int o = 1; o < c; ++o)
        if (s_par[o] == par) earlier += s_e[o];
      live = e > 0.0;
      const double S = static_cast<double>(s_stat[par].y) - earlier;
      acc = live && (S <= e || static_cast<double>(uc) * S <= e);
    }
  } else {
    // greedy: a child is accepted iff its token is its parent's argmax
    acc = c >= 1 && c < N && tok == s_arg[par];
  }
  if (c < 64) s_acc[c] = acc ? 1 : 0;
  __syncthreads();
  if (tid < 32) {
    // one warp: lane l holds nodes l and l + 32
    const int lane = tid;
    const int par1 = s_par[lane + 32];
    const bool acc1 = s_acc[lane + 32] != 0;
    int cur = 0, len = 1;
    if (lane == 0) {
      path[0] = 0;
      out[0] = tok;
    }
    for (int step = 1; step < N; ++step) {
      const unsigned m0 = __ballot_sync(0xffffffffu, par == cur && acc);
      const unsigned m1 = __ballot_sync(0xffffffffu, par1 == cur && acc1);
      if (!m0 && !m1) break;
      cur = m0 ? __ffs(m0) - 1 : 32 + __ffs(m1) - 1;  // the first accepted child in node order
      if (lane == 0) {
        path[len] = cur;
        out[len] = s_tok_in[cur];
      }
      ++len;
    }
    for (int i = len + lane; i < N; i += 32) path[i] = -1;
    if (!tempered) {
      if (lane == 0) {
        out[len] = s_arg[cur];
        p.num_accepted[b] = len - 1;
        p.num_emitted[b] = len + 1;
      }
      for (int i = len + 1 + lane; i <= N; i += 32) out[i] = -1;
    } else if (lane == 0) {  // every child of `cur` rejected: the whole block draws
      s_final = cur;
      s_len = len;
      s_nrm = 0;
    }
  }
  __syncthreads();
  if (s_final < 0) return;  // greedy: done
  if (live && par == s_final) {
    // a rejected token of the final node: its weight relative to the row maximum, its place
    // among them by token
    int rank = 0;
#pragma unroll 8
    for (int o = 1; o < N; ++o) rank += s_par[o] == par && s_e[o] > 0.0 && s_tok_in[o] < tok;
    s_rm[rank] = tok;
    s_rmw[rank] = rel_weight(load_elem<BF16>(tbase + (brow + par) * rbytes, tok), s_stat[par].x, cs);
    s_rmk[rank] = tok / p.elems_per_split;
    atomicAdd(&s_nrm, 1);
  }
  __syncthreads();

  // ---- the final draw from p' of node s_final: inverse CDF in ascending token order ----
  const int fin = s_final, len = s_len, nrm = s_nrm;
  const int64_t frid = brow + fin;
  const float M = s_stat[fin].x;
  const int eps = p.elems_per_split;
  if (tid < 32) {
    // remaining mass of each part (its sum minus its rejected tokens' weights), the total,
    // and the part where the cumulative mass reaches u[0] x total: one part per lane
    // (at most kFiltMaxSplits parts)
    const int k = tid;
    double base = 0.0;
    if (k < p.splits) {
      const float2 q = s_part[fin * 16 + k];
      base = static_cast<double>(q.y) * rel_weight(q.x, M, cs);
    }
    double removed = 0.0;
    for (int r = 0; r < nrm; ++r)
      if (s_rmk[r] == k) removed += static_cast<double>(s_rmw[r]);
    double mass = base - removed;
    if (mass < 0.0) mass = 0.0;
    double S = mass;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) S += __shfl_xor_sync(0xffffffffu, S, o);
    if (!(S > 0.0)) {
      // nothing left after the removals (rounding only): draw from p itself
      mass = base;
      S = mass;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) S += __shfl_xor_sync(0xffffffffu, S, o);
      if (k == 0) s_nrm = 0;
    }
    const double target = static_cast<double>(p.uniforms[brow]) * S;
    double incl = mass;  // inclusive prefix over parts
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const double y = __shfl_up_sync(0xffffffffu, incl, o);
      if (k >= o) incl += y;
    }
    const double excl = incl - mass;
    const unsigned hit = __ballot_sync(0xffffffffu, mass > 0.0 && incl >= target);
    // rounding may leave the target above the total: then the last part with mass
    const unsigned pos = __ballot_sync(0xffffffffu, mass > 0.0);
    const int kc = hit ? __ffs(hit) - 1 : (pos ? 31 - __clz(pos) : -1);
    const double before = __shfl_sync(0xffffffffu, excl, kc < 0 ? 0 : kc);
    if (k == 0) {
      s_kcross = kc < 0 ? 0 : kc;  // the part of the row maximum always has mass
      s_target = target - before;
    }
  }
  __syncthreads();
  const int kc = s_kcross, nrm_scan = s_nrm;
  const double tin = s_target;
  // each thread a contiguous run of the crossing part (multiples of 8 elements)
  const int pb = kc * eps, pe = min(V, pb + eps);
  const int per = ((pe - pb + kThreads - 1) / kThreads + 7) / 8 * 8;
  const int lo = min(pe, pb + tid * per), hi = min(pe, lo + per);
  const char* frow = static_cast<const char*>(p.target) + frid * V * (BF16 ? 2 : 4);
  int ptr = 0;
  while (ptr < nrm_scan && s_rm[ptr] < lo) ++ptr;
  // The run is read kBatch 16-byte vectors at a time when the rows allow (a run starts on a
  // multiple of 8 elements, and hi is a multiple of the vector's elements), all of them in
  // flight together; the code below is per vector, the batch moving up by one each time.
  constexpr int kEpv = BF16 ? 8 : 4, kBatch = 8;
  float run = 0.f;
  {
    int q = ptr, next_rm = ptr < nrm_scan ? s_rm[ptr] : INT_MAX;
    for (int x0 = lo; x0 < hi; x0 += kBatch * kEpv) {
      uint4 raw[kBatch];
#pragma unroll
      for (int v = 0; v < kBatch; ++v) {
        const int x = x0 + v * kEpv;
        raw[v] = make_uint4(0u, 0u, 0u, 0u);
        if (VEC && x < hi) raw[v] = __ldg(reinterpret_cast<const uint4*>(frow + static_cast<int64_t>(x) * (BF16 ? 2 : 4)));
      }
#pragma unroll 1
      for (int x = x0; x < min(hi, x0 + kBatch * kEpv); x += kEpv) {
        // the vector's weights, then the removed tokens' cleared (elements come in ascending
        // order and the removed tokens are distinct and ascending: the next one is kept)
        float lv[kEpv], w[kEpv];
        const uint32_t wv[4] = {raw[0].x, raw[0].y, raw[0].z, raw[0].w};
#pragma unroll
        for (int i = 0; i < kEpv; ++i)
          lv[i] = !VEC ? (x + i < hi ? load_elem<BF16>(frow, x + i) : 0.f)
                  : BF16 ? __uint_as_float((i & 1) ? (wv[i >> 1] & 0xffff0000u) : (wv[i >> 1] << 16))
                         : __uint_as_float(wv[i]);
#pragma unroll
        for (int v = 0; v + 1 < kBatch; ++v) raw[v] = raw[v + 1];
#pragma unroll
        for (int i = 0; i < kEpv; ++i) w[i] = x + i < hi ? rel_weight(lv[i], M, cs) : 0.f;
        while (next_rm < x + kEpv) {
#pragma unroll
          for (int i = 0; i < kEpv; ++i)
            if (x + i == next_rm) w[i] = 0.f;
          ++q;
          next_rm = q < nrm_scan ? s_rm[q] : INT_MAX;
        }
#pragma unroll
        for (int i = 0; i < kEpv; ++i) run += w[i];
      }
    }
  }
  // block exclusive scan of the runs' sums; the run that holds the crossing is the last
  // one with weight whose exclusive prefix is below the target
  double incl = static_cast<double>(run);
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double y = __shfl_up_sync(0xffffffffu, incl, o);
    if ((tid & 31) >= o) incl += y;
  }
  double prev = __shfl_up_sync(0xffffffffu, incl, 1);
  if ((tid & 31) == 0) prev = 0.0;
  if ((tid & 31) == 31) s_dsum[tid >> 5] = incl;
  __syncthreads();
  double wbase = 0.0;
  for (int k = 0; k < (tid >> 5); ++k) wbase += s_dsum[k];
  const double excl = wbase + prev;
  int owner = (run > 0.f && excl < tin) ? tid : -1;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) owner = max(owner, __shfl_xor_sync(0xffffffffu, owner, o));
  __syncthreads();  // every thread has read s_dsum
  if ((tid & 31) == 0) s_fsum[tid >> 5] = __int_as_float(owner);
  __syncthreads();
  owner = -1;
  for (int k = 0; k < kThreads / 32; ++k) owner = max(owner, __float_as_int(s_fsum[k]));
  if (tid == owner) {
    s_lo = lo;
    s_hi = hi;
    s_excl = excl;
  }
  __syncthreads();
  if (owner >= 0 && tid < 32) {
    // one warp over the owner's run, 32 elements at a time: the first token whose cumulative
    // weight (fp64) reaches the target, else (if rounding leaves the target above the run)
    // its last positive-weight token. (One thread adding the weights one by one in fp64
    // took 3.5 us.)
    const int rlo = s_lo, rhi = s_hi;
    double C = s_excl;
    int pick = -1;
    bool done = false;
    for (int x0 = rlo; x0 < rhi && !done; x0 += 32) {
      const int x = x0 + tid;
      float w = x < rhi ? rel_weight(load_elem<BF16>(frow, x), M, cs) : 0.f;
      for (int r = 0; r < nrm_scan; ++r)
        if (s_rm[r] == x) w = 0.f;
      double incl = static_cast<double>(w);
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const double y = __shfl_up_sync(0xffffffffu, incl, o);
        if (tid >= o) incl += y;
      }
      const unsigned hit = __ballot_sync(0xffffffffu, w > 0.f && C + incl >= tin);
      const unsigned any = __ballot_sync(0xffffffffu, w > 0.f);
      if (hit) {
        pick = x0 + __ffs(hit) - 1;
        done = true;
      } else if (any) {
        pick = x0 + 31 - __clz(any);
      }
      C += __shfl_sync(0xffffffffu, incl, 31);
    }
    if (tid == 0) s_tok = pick;
  }
  if (owner < 0 && tid == 0) s_tok = s_arg[fin];  // no weight left in fp32: the row maximum
  __syncthreads();
  if (tid == 0) {
    out[len] = s_tok;
    p.num_accepted[b] = len - 1;
    p.num_emitted[b] = len + 1;
  }
  for (int c = len + 1 + tid; c <= N; c += kThreads) out[c] = -1;
}

// Flags of sequence b's commit inputs (0 = valid), evaluated by one full warp: kv_len
// within the table and at least num_nodes, num_accepted in [-1, num_nodes), a path that
// starts at the root and rises strictly inside the tree, and the pages of every moved row.
__device__ uint32_t tree_commit_check(const spec_tree_commit_args_t& a, int b, int lane) {
  const int N = a.num_nodes, P = a.page_size;
  const int kv = a.kv_len[b], na = a.num_accepted[b];
  if (kv < N || static_cast<int64_t>(kv) > static_cast<int64_t>(a.max_pages_per_seq) * P)
    return SPEC_FLAG_BAD_KV_LEN;
  if (na < -1 || na >= N) return SPEC_FLAG_BAD_TREE;
  const int ctx = kv - N;
  const int32_t* path = a.path + static_cast<int64_t>(b) * N;
  const int32_t* table = a.page_table + static_cast<int64_t>(b) * a.max_pages_per_seq;
  uint32_t f = 0;
  for (int d = lane; d <= na; d += 32) {
    const int s = path[d];
    if (d == 0 ? s != 0 : (s <= path[d - 1] || s >= N)) {
      f |= SPEC_FLAG_BAD_TREE;
    } else if (s != d) {
      const int ps = table[(ctx + s) / P], pd = table[(ctx + d) / P];
      if (ps < 0 || ps >= a.num_pages || pd < 0 || pd >= a.num_pages) f |= SPEC_FLAG_BAD_PAGE;
    }
  }
  return __reduce_or_sync(0xffffffffu, f);
}

// One block per (cache, KV head, sequence) moves that head's rows of the accepted path:
// row path[d] to block position d for d = 1 .. num_accepted. A source path[d] >= d may be
// another position's destination (path 0, 2, 3: position 1 reads slot 2, which position 2
// writes), so every source piece is loaded into registers before any is stored; that is
// the result of moving the rows one after another in increasing d, as no row is read
// after a lower position was written over it.
template <int D>
__global__ void __launch_bounds__(128) tree_compact_kernel(spec_tree_commit_args_t a) {
  constexpr int kPieces = D / 8;                          // 16-byte pieces of a row
  constexpr int kIter = (63 * kPieces + 127) / 128;       // num_accepted <= 63
  __shared__ uint32_t s_flags;
  const int which = blockIdx.x & 1, h = blockIdx.x >> 1, b = blockIdx.y, tid = threadIdx.x;
  if (tid < 32) {
    const uint32_t f = tree_commit_check(a, b, tid);
    if (tid == 0) s_flags = f;
  }
  __syncthreads();
  if (s_flags) {
    if (tid == 0 && blockIdx.x == 0 && a.status) set_status(a.status, s_flags);
    return;
  }
  const int N = a.num_nodes, P = a.page_size, H = a.num_kv_heads;
  const int na = a.num_accepted[b];
  if (na <= 0) return;
  const int ctx = a.kv_len[b] - N;
  const int32_t* path = a.path + static_cast<int64_t>(b) * N;
  const int32_t* table = a.page_table + static_cast<int64_t>(b) * a.max_pages_per_seq;
  uint4* cache = static_cast<uint4*>(which ? a.v_cache : a.k_cache);
  const int n = na * kPieces;
  // the piece's offset in uint4 units, or -1 where the row stays in place
  auto offset = [&](int i, bool src) -> int64_t {
    const int d = 1 + i / kPieces, c = i % kPieces, s = path[d];
    if (s == d) return -1;
    const int pos = ctx + (src ? s : d);
    return ((static_cast<int64_t>(table[pos / P]) * H + h) * P + pos % P) * kPieces + c;
  };
  uint4 r[kIter];
#pragma unroll
  for (int k = 0; k < kIter; ++k) {
    const int i = tid + k * 128;
    if (i < n) {
      const int64_t o = offset(i, true);
      if (o >= 0) r[k] = cache[o];
    }
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < kIter; ++k) {
    const int i = tid + k * 128;
    if (i < n) {
      const int64_t o = offset(i, false);
      if (o >= 0) cache[o] = r[k];
    }
  }
}

// One warp per sequence: kv_len = ctx + num_accepted + 1 where the inputs are valid.
__global__ void tree_commit_len_kernel(spec_tree_commit_args_t a) {
  const int b = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (b >= a.batch) return;
  const uint32_t f = tree_commit_check(a, b, lane);
  if (lane == 0 && f == 0) {
    const int na = a.num_accepted[b];
    a.kv_len[b] = a.kv_len[b] - a.num_nodes + (na >= 0 ? na + 1 : 0);
  }
}

// ---------------------------------------------------------------------------------
// The tree sampler. tree_build_kernel: grid (splits, positions, sequences) of 128-thread
// blocks. A block ranks the candidates of its part of a drafter row: composite keys
// (order of the logit, then the lower token id) are unique, so the top-K of the part
// lie among the keys at or above the K-th largest per-thread maximum; those few are
// ranked by counting. The row's last part block merges the parts' sorted lists and
// the parts' (max, sum of exponentials) into the row's log-normaliser and writes the
// position's ranked (token, log q) table; the sequence's last row block selects the
// tree's nodes best first, one warp holding the offers of two nodes per lane (path
// scores are double-float sums of the fp32 log q).
// ---------------------------------------------------------------------------------
struct BuildParams {
  int batch, gamma, vocab, rows, keff, nodes, splits, eps;
  const void* logits;
  const float* temperature;
  const int32_t* root;
  int32_t* tokens;
  int32_t* parents;
  int32_t* depth;
  uint64_t* mask;
  uint32_t* status;
  uint32_t* tickets;
  uint32_t* seq_flags;
  uint32_t* row_tickets;
  unsigned long long* keys;
  float4* stats;
  int2* table;
};

constexpr int kPartUnroll = 4;

__device__ __forceinline__ unsigned long long cand_key(float x, int idx) {
  return (static_cast<unsigned long long>(order_key(x)) << 32) | (0xffffffffu - static_cast<uint32_t>(idx));
}
__device__ __forceinline__ float key_value(unsigned long long k) {
  const uint32_t h = static_cast<uint32_t>(k >> 32);
  return __uint_as_float((h & 0x80000000u) ? (h & 0x7fffffffu) : ~h);
}
__device__ __forceinline__ int key_index(unsigned long long k) {
  return static_cast<int>(0xffffffffu - static_cast<uint32_t>(k));
}

// (max, sum of 2^((x - max) c2)) pairs combined; a -inf max carries no mass
__device__ __forceinline__ void merge_ms(float& m, float& s, float m2, float s2, float c2) {
  const float M = fmaxf(m, m2);
  float t = 0.f;
  if (m > -INFINITY) t += s * ex2((m - M) * c2);
  if (m2 > -INFINITY) t += s2 * ex2((m2 - M) * c2);
  m = M;
  s = t;
}

// Calls f(x, base) on this thread's logits of [e_begin, e_end) of the row, a 16-byte
// group at a time (x[q] is logit base + q; groups of one where rows are not aligned).
template <bool BF16, bool VEC, class F>
__device__ __forceinline__ void for_groups(const char* rowp, int e_begin, int e_end, int tid, F&& f) {
  if (VEC) {
    constexpr int kEpv = BF16 ? 8 : 4;
    const uint4* rv = reinterpret_cast<const uint4*>(rowp);
    const int vbeg = e_begin / kEpv, vend = e_end / kEpv;
    for (int v0 = vbeg + tid; v0 < vend; v0 += kThreads * kPartUnroll) {
      uint4 dv[kPartUnroll];
#pragma unroll
      for (int k = 0; k < kPartUnroll; ++k) {
        const int vi = v0 + k * kThreads;
        if (vi < vend) dv[k] = __ldg(rv + vi);
      }
#pragma unroll
      for (int k = 0; k < kPartUnroll; ++k) {
        const int vi = v0 + k * kThreads;
        if (vi < vend) {
          const uint32_t wv[4] = {dv[k].x, dv[k].y, dv[k].z, dv[k].w};
          float x[kEpv];
#pragma unroll
          for (int q = 0; q < kEpv; ++q)
            x[q] = BF16 ? __uint_as_float((q & 1) ? (wv[q >> 1] & 0xffff0000u) : (wv[q >> 1] << 16))
                        : __uint_as_float(wv[q]);
          f(x, vi * kEpv);
        }
      }
    }
  } else {
    for (int e0 = e_begin + tid; e0 < e_end; e0 += kThreads * kPartUnroll) {
      float x[kPartUnroll];
#pragma unroll
      for (int k = 0; k < kPartUnroll; ++k) {
        const int ei = e0 + k * kThreads;
        x[k] = ei < e_end ? load_elem<BF16>(rowp, ei) : 0.f;
      }
#pragma unroll
      for (int k = 0; k < kPartUnroll; ++k) {
        const float one[1] = {x[k]};
        if (e0 + k * kThreads < e_end) f(one, e0 + k * kThreads);
      }
    }
  }
}

// Sorts one key per lane of the warp into descending order (bitonic network).
__device__ __forceinline__ unsigned long long warp_sort_desc(unsigned long long v, int lane) {
#pragma unroll
  for (int k = 2; k <= 32; k <<= 1) {
#pragma unroll
    for (int j = k >> 1; j > 0; j >>= 1) {
      const unsigned long long o = __shfl_xor_sync(0xffffffffu, v, j);
      const bool keep_max = ((lane & j) == 0) == ((lane & k) == 0);
      v = keep_max ? (o > v ? o : v) : (o < v ? o : v);
    }
  }
  return v;
}

// The 64 largest of two descending lists of 64 keys (a0, a1 and b0, b1: the lane's
// entries lane and lane + 32 of each), descending, as the lane's two entries. The elementwise
// maximum of one list and the other reversed is bitonic and holds the 64 largest; a
// bitonic merge (half-cleaners of 32, 16, .., 1) sorts it.
__device__ __noinline__ ulonglong2 merge_top64(unsigned long long a0, unsigned long long a1,
                                               unsigned long long b0, unsigned long long b1, int lane) {
  const unsigned long long rb0 = __shfl_sync(0xffffffffu, b1, 31 - lane);
  const unsigned long long rb1 = __shfl_sync(0xffffffffu, b0, 31 - lane);
  unsigned long long c0 = a0 > rb0 ? a0 : rb0;
  unsigned long long c1 = a1 > rb1 ? a1 : rb1;
  {
    const unsigned long long hi = c0 > c1 ? c0 : c1, lo = c0 > c1 ? c1 : c0;
    c0 = hi;
    c1 = lo;
  }
#pragma unroll
  for (int j = 16; j > 0; j >>= 1) {
    const unsigned long long o0 = __shfl_xor_sync(0xffffffffu, c0, j);
    const unsigned long long o1 = __shfl_xor_sync(0xffffffffu, c1, j);
    const bool lower = (lane & j) == 0;
    c0 = lower ? (c0 > o0 ? c0 : o0) : (c0 < o0 ? c0 : o0);
    c1 = lower ? (c1 > o1 ? c1 : o1) : (c1 < o1 ? c1 : o1);
  }
  return make_ulonglong2(c0, c1);
}

// x[q] for a q known only at run time, by selects (no local-memory copy of x).
template <int E>
__device__ __forceinline__ float pick(const float (&x)[E], int q) {
  float v = x[0];
#pragma unroll
  for (int j = 1; j < E; ++j) v = j == q ? x[j] : v;
  return v;
}

__device__ __forceinline__ unsigned long long block_max_u64(unsigned long long v, unsigned long long* s_red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long y = __shfl_xor_sync(0xffffffffu, v, o);
    v = y > v ? y : v;
  }
  __syncthreads();
  if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = v;
  __syncthreads();
  v = s_red[0];
#pragma unroll
  for (int k = 1; k < kThreads / 32; ++k) v = s_red[k] > v ? s_red[k] : v;
  return v;
}

// (ah + al) + b as a normalised double-float (rh + rl): the exact sum of ah and b by
// Knuth's two-sum, then the low parts folded in (a fast two-sum). Path scores keep
// about 48 bits this way without fp64 arithmetic, whose latency is high on this part.
__device__ __forceinline__ void df_add(float ah, float al, float b, float& rh, float& rl) {
  const float s = __fadd_rn(ah, b);
  const float bb = __fsub_rn(s, ah);
  const float e = __fadd_rn(__fsub_rn(ah, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  const float t = __fadd_rn(e, al);
  const float h = __fadd_rn(s, t);
  const bool none = !(s > -INFINITY);  // a -inf term
  rh = none ? s : h;
  rl = none ? 0.f : __fsub_rn(t, __fsub_rn(h, s));
}

struct TreeNode {
  int dep, nx, par, idx;   // dep < 0: no node in this slot; idx: the parent's candidate it took
  float sh, sl;            // path score as an unevaluated sum sh + sl (double-float)
  // Scores the node may bring to the next steps, the same way, each with the order key of its
  // high part (0 if there is none): its current offer (candidate nx of position dep + 1), the
  // offer after that, and the first offer of the node the current one would become.
  float oh, ol, nh, nl, ch, cl;
  uint32_t ok, nk, ck;
  float nq, cq;            // log q of the last two, read ahead; NaN: there is none
  unsigned long long msk;  // ancestor bits
};

// Best-first selection of the tree's nodes by one warp. The root (node 0) is kept in
// every lane; node c >= 1 is slot (c - 1) / 32 of lane (c - 1) % 32. Each step takes the
// best offer (largest high part; on a tie the largest low part, then the lowest node
// index, the root first), makes it node i, and moves its parent to its next candidate.
// Both of the offers a step puts up were scored when the one it takes was, so a step's
// chain is a warp maximum, a ballot and a shuffle, and the table is read beside it
// (scored within the step and with branches: 0.37 us a node, now 0.24; tokens follow from
// the parents' candidates at the end).
template <int SLOTS>
__device__ __forceinline__ void select_nodes(const BuildParams& p, const int2* tab, int K, int b,
                                             uint32_t flags, int lane) {
  const int N = p.nodes;
  const int64_t base = static_cast<int64_t>(b) * N;
  // log q of candidate nx of table row dep (NaN past the table), without a branch
  auto cand_q = [&](int dep, int nx) -> float {
    const bool valid = static_cast<unsigned>(dep) < static_cast<unsigned>(p.rows) && nx < K;
    const float q = __int_as_float(tab[valid ? dep * K + nx : 0].y);
    return valid ? q : NAN;
  };
  // the reads of the node's next offers, and their scores from what was read
  auto fetch = [&](TreeNode& n) {
    n.nq = cand_q(n.dep, n.nx + 1);
    n.cq = cand_q(n.ok ? n.dep + 1 : -1, 0);
  };
  auto score = [&](TreeNode& n) {
    df_add(n.sh, n.sl, n.nq, n.nh, n.nl);
    df_add(n.oh, n.ol, n.cq, n.ch, n.cl);
    n.nk = n.nq == n.nq ? order_key(n.nh) : 0u;
    n.ck = n.cq == n.cq ? order_key(n.ch) : 0u;
  };
  TreeNode root = {}, n[SLOTS];
  root.par = -1;
  root.msk = 1ull;
#pragma unroll
  for (int h = 0; h < SLOTS; ++h) {
    n[h] = {};
    n[h].dep = -1;
    n[h].par = -1;
  }
  if (!flags) {
    const float q0 = cand_q(0, 0);
    df_add(0.f, 0.f, q0, root.oh, root.ol);
    root.ok = q0 == q0 ? order_key(root.oh) : 0u;
    fetch(root);
    score(root);
#pragma unroll
    for (int h = 0; h < SLOTS; ++h) fetch(n[h]);
#pragma unroll 1
    for (int i = 1; i < N; ++i) {
      uint32_t hl = 0u;
#pragma unroll
      for (int h = 0; h < SLOTS; ++h) hl = max(hl, n[h].ok);
      const uint32_t Mh = max(__reduce_max_sync(0xffffffffu, hl), root.ok);
#pragma unroll
      for (int h = 0; h < SLOTS; ++h) score(n[h]);  // beside the maximum's latency
      if (Mh == 0u) {  // no offer left: excluded by the host's capacity check
        flags |= SPEC_FLAG_BAD_TREE;
        break;
      }
      unsigned bal[SLOTS];
      int ties = root.ok == Mh;
#pragma unroll
      for (int h = 0; h < SLOTS; ++h) {
        bal[h] = __ballot_sync(0xffffffffu, n[h].ok == Mh);
        ties += __popc(bal[h]);
      }
      bool root_wins = root.ok == Mh;
      if (ties > 1) {
        const uint32_t rl = root.ok == Mh ? order_key(root.ol) : 0u;
        uint32_t ll = 0u;
#pragma unroll
        for (int h = 0; h < SLOTS; ++h)
          if (n[h].ok == Mh) ll = max(ll, order_key(n[h].ol));
        const uint32_t Ml = max(__reduce_max_sync(0xffffffffu, ll), rl);
        root_wins = root.ok == Mh && rl == Ml;
#pragma unroll
        for (int h = 0; h < SLOTS; ++h)
          bal[h] = __ballot_sync(0xffffffffu, n[h].ok == Mh && order_key(n[h].ol) == Ml);
      }
      // the winner u, its offer and that offer's own first offer, depth and ancestor bits
      int u = 0, hs = 0;
      float wh = root.oh, wl = root.ol, wch = root.ch, wcl = root.cl;
      uint32_t wck = root.ck;
      int wdn = root.nx;  // depth << 16 | candidate
      unsigned long long wm = 1ull;
      int src = 0;
      if (!root_wins) {
#pragma unroll
        for (int h = SLOTS - 1; h >= 0; --h)
          if (bal[h]) {
            u = 1 + 32 * h + __ffs(bal[h]) - 1;
            hs = h;
          }
        src = (u - 1) & 31;
        constexpr int L = SLOTS - 1;
        const bool up = SLOTS > 1 && hs == L;
        wck = __shfl_sync(0xffffffffu, up ? n[L].ck : n[0].ck, src);
        wch = __shfl_sync(0xffffffffu, up ? n[L].ch : n[0].ch, src);
        wcl = __shfl_sync(0xffffffffu, up ? n[L].cl : n[0].cl, src);
        wh = __shfl_sync(0xffffffffu, up ? n[L].oh : n[0].oh, src);
        wl = __shfl_sync(0xffffffffu, up ? n[L].ol : n[0].ol, src);
        wdn = __shfl_sync(0xffffffffu, up ? (n[L].dep << 16) | n[L].nx : (n[0].dep << 16) | n[0].nx, src);
        wm = __shfl_sync(0xffffffffu, up ? n[L].msk : n[0].msk, src);
      }
      // node i takes the offer; its parent moves to its next candidate
      const int ci = (i - 1) & 31, chs = (i - 1) >> 5;
#pragma unroll
      for (int h = 0; h < SLOTS; ++h) {
        const bool is_new = lane == ci && chs == h;
        const bool adv = u != 0 && lane == src && hs == h;
        if (is_new) {
          n[h].dep = (wdn >> 16) + 1;
          n[h].nx = 0;
          n[h].par = u;
          n[h].idx = wdn & 0xffff;
          n[h].sh = wh;
          n[h].sl = wl;
          n[h].oh = wch;
          n[h].ol = wcl;
          n[h].ok = wck;
          n[h].msk = wm | (1ull << i);
        }
        if (adv) {
          ++n[h].nx;
          n[h].oh = n[h].nh;
          n[h].ol = n[h].nl;
          n[h].ok = n[h].nk;
        }
        fetch(n[h]);
      }
      if (u == 0) {
        ++root.nx;
        root.oh = root.nh;
        root.ol = root.nl;
        root.ok = root.nk;
        fetch(root);
        score(root);
      }
    }
  }
  if (lane == 0) {
    p.tokens[base] = flags ? -1 : p.root[b];
    p.parents[base] = -1;
    if (p.depth) p.depth[base] = flags ? -1 : 0;
    if (p.mask) p.mask[base] = flags ? 0ull : 1ull;
  }
#pragma unroll
  for (int h = 0; h < SLOTS; ++h) {
    const int c = 1 + lane + 32 * h;
    if (c >= N) continue;
    p.tokens[base + c] = flags ? -1 : tab[(n[h].dep - 1) * K + n[h].idx].x;
    p.parents[base + c] = flags ? -1 : n[h].par;
    if (p.depth) p.depth[base + c] = flags ? -1 : n[h].dep;
    if (p.mask) p.mask[base + c] = flags ? 0ull : n[h].msk;
  }
  if (lane == 0 && flags) set_status(p.status, flags);
}

template <bool BF16, bool VEC>
__global__ void __launch_bounds__(kThreads) tree_build_kernel(BuildParams p) {
  extern __shared__ unsigned long long s_dyn[];
  __shared__ unsigned long long s_tmax[kThreads];
  __shared__ unsigned long long s_tau;
  __shared__ float s_wm[kThreads / 32], s_ws[kThreads / 32];
  __shared__ int s_wcnt[kThreads / 32];
  __shared__ int s_count, s_bad, s_last;
  __shared__ uint32_t s_flags;
  const int split = blockIdx.x, r = blockIdx.y, b = blockIdx.z, tid = threadIdx.x;
  const int lane = tid & 31, w = tid >> 5;
  const int K = p.keff, S = p.splits;
  const int64_t rid = static_cast<int64_t>(b) * p.rows + r;
  const char* rowp = static_cast<const char*>(p.logits) +
                     (static_cast<int64_t>(b) * p.gamma + r + 1) * p.vocab * (BF16 ? 2 : 4);
  const int e_begin = split * p.eps, e_end = min(p.vocab, e_begin + p.eps);
  const float T = p.temperature[b];
  const float invT = 1.f / (T > 0.f ? T : 1.f);
  const float c2 = invT * kLog2e;
  if (tid == 0) {
    s_tau = 0ull;
    s_count = 0;
    s_bad = 0;
  }
  __syncthreads();

  // pass 1, a 16-byte group at a time: the thread's maximum and its lowest index, the
  // sum of 2^((x - max) c2) (rescaled when the maximum rises), NaN or +inf seen (a NaN
  // sum, or a NaN among logits that are all -inf so far)
  float m = -INFINITY, s = 0.f, mc = 0.f;
  int mi = -1;
  bool nan_seen = false, fused = false;  // fused: the exponents by one multiply-add (kFusedMax)
  for_groups<BF16, VEC>(rowp, e_begin, e_end, tid, [&](const auto& x, int base) {
    constexpr int E = sizeof(x) / sizeof(float);
    float vmax = x[0];
#pragma unroll
    for (int q = 1; q < E; ++q) vmax = fmaxf(vmax, x[q]);
    if (mi < 0) mi = base;  // the first logit: the maximum of a part of -inf
    if (vmax > m) {
      unsigned eq = 0u;
#pragma unroll
      for (int q = 0; q < E; ++q) eq |= (x[q] == vmax ? 1u : 0u) << q;
      const int q0 = __ffs(eq) - 1;
      s *= ex2((m - vmax) * c2);
      m = vmax;
      mc = m * c2;
      fused = fabsf(mc) <= kFusedMax;
      mi = base + q0;
    }
    if (fused) {
#pragma unroll
      for (int q = 0; q < E; ++q) s += ex2(fmaf(x[q], c2, -mc));
    } else if (m > -INFINITY) {
#pragma unroll
      for (int q = 0; q < E; ++q) s += ex2((x[q] - m) * c2);
    } else {
#pragma unroll
      for (int q = 0; q < E; ++q) nan_seen |= x[q] != x[q];
    }
  });
  if (nan_seen || s != s) s_bad = 1;
  const unsigned long long L0 = mi >= 0 ? cand_key(m, mi) : 0ull;
  // tau: the K-th largest of the threads' maximum keys (0 if fewer threads hold
  // logits); the part's top K keys are among the keys >= tau. Each warp sorts its 32
  // keys; a key's rank is its place in its warp plus the keys above it in the others.
  {
    const unsigned long long v = warp_sort_desc(L0, lane);
    s_tmax[tid] = v;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float m2 = __shfl_xor_sync(0xffffffffu, m, o), s2 = __shfl_xor_sync(0xffffffffu, s, o);
      merge_ms(m, s, m2, s2, c2);
    }
    if (lane == 0) {
      s_wm[w] = m;
      s_ws[w] = s;
    }
    __syncthreads();
    int rank = lane;
#pragma unroll
    for (int w2 = 0; w2 < kThreads / 32; ++w2) {
      if (w2 == w) continue;
      const unsigned long long* run = s_tmax + w2 * 32;
      int lo = 0, hi = 32;
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (run[mid] > v) lo = mid + 1;
        else hi = mid;
      }
      rank += lo;
    }
    if (rank == K - 1) s_tau = v;
  }
  __syncthreads();
  const unsigned long long tau = s_tau;
  // pass 2: the keys >= tau (logit above tv, or equal with index at most ti), kept in
  // four registers per thread and placed by a block scan; a thread with more (or tau =
  // 0: every logit is one) sends the block to shared-memory atomics instead
  const float tv = tau ? key_value(tau) : -INFINITY;
  const int ti = tau ? key_index(tau) : INT_MAX;
  unsigned long long c0 = 0ull, c1 = 0ull, c2k = 0ull, c3 = 0ull;
  int cnt = 0;
  if (tau != 0ull) {
    for_groups<BF16, VEC>(rowp, e_begin, e_end, tid, [&](const auto& x, int base) {
      constexpr int E = sizeof(x) / sizeof(float);
      float vmax = x[0];
#pragma unroll
      for (int q = 1; q < E; ++q) vmax = fmaxf(vmax, x[q]);
      if (vmax >= tv) {
        unsigned cm = 0u;
#pragma unroll
        for (int q = 0; q < E; ++q)
          cm |= ((x[q] > tv || (x[q] == tv && base + q <= ti)) ? 1u : 0u) << q;
        while (cm) {
          const int q = __ffs(cm) - 1;
          cm &= cm - 1;
          const unsigned long long k = cand_key(pick(x, q), base + q);
          if (cnt == 0) c0 = k;
          else if (cnt == 1) c1 = k;
          else if (cnt == 2) c2k = k;
          else if (cnt == 3) c3 = k;
          ++cnt;
        }
      }
    });
  }
  if (!__syncthreads_or(tau == 0ull || cnt > 4)) {
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) s_wcnt[w] = incl;
    __syncthreads();
    int off = incl - cnt;
    for (int w2 = 0; w2 < w; ++w2) off += s_wcnt[w2];
    if (cnt > 0) s_dyn[off] = c0;
    if (cnt > 1) s_dyn[off + 1] = c1;
    if (cnt > 2) s_dyn[off + 2] = c2k;
    if (cnt > 3) s_dyn[off + 3] = c3;
    if (tid == kThreads - 1) s_count = off + cnt;
  } else {
    for_groups<BF16, VEC>(rowp, e_begin, e_end, tid, [&](const auto& x, int base) {
      constexpr int E = sizeof(x) / sizeof(float);
      float vmax = x[0];
#pragma unroll
      for (int q = 1; q < E; ++q) vmax = fmaxf(vmax, x[q]);
      if (vmax >= tv) {
        unsigned cm = 0u;
#pragma unroll
        for (int q = 0; q < E; ++q)
          cm |= ((x[q] > tv || (x[q] == tv && base + q <= ti)) ? 1u : 0u) << q;
        while (cm) {
          const int q = __ffs(cm) - 1;
          cm &= cm - 1;
          const int slot = atomicAdd(&s_count, 1);
          if (slot < kTreeCandCap) s_dyn[slot] = cand_key(pick(x, q), base + q);
        }
      }
    });
  }
  __syncthreads();
  const int C = s_count;
  unsigned long long* out = p.keys + (rid * S + split) * 64;
  if (C <= kTreeCandCap) {
    for (int i = tid; i < C; i += kThreads) {
      const unsigned long long k = s_dyn[i];
      int rk = 0;
      for (int j = 0; j < C; ++j) rk += s_dyn[j] > k;
      if (rk < K) out[rk] = k;
    }
    for (int i = C + tid; i < K; i += kThreads) out[i] = 0ull;
  } else {
    // many keys at the threshold (an adversarial order): K exact rounds instead
    unsigned long long prev = ~0ull;
    for (int rk = 0; rk < K; ++rk) {
      unsigned long long best = 0ull;
      for_groups<BF16, VEC>(rowp, e_begin, e_end, tid, [&](const auto& x, int base) {
        constexpr int E = sizeof(x) / sizeof(float);
#pragma unroll
        for (int q = 0; q < E; ++q) {
          const unsigned long long k = cand_key(x[q], base + q);
          if (k < prev && k > best) best = k;
        }
      });
      best = block_max_u64(best, s_tmax);
      if (tid == 0) out[rk] = best;
      prev = best;
    }
  }
  if (tid == 0) {
    float M = s_wm[0], Sum = s_ws[0];
    for (int w2 = 1; w2 < kThreads / 32; ++w2) merge_ms(M, Sum, s_wm[w2], s_ws[w2], c2);
    p.stats[rid * S + split] = make_float4(M, Sum, __uint_as_float(static_cast<uint32_t>(s_bad)), 0.f);
  }

  // the row's last part block: merge the parts' lists and normalisers
  __threadfence();
  __syncthreads();
  if (tid == 0) {
    const uint32_t prev = atomicAdd(&p.row_tickets[rid], 1u);
    s_last = prev == static_cast<uint32_t>(S - 1);
    if (s_last) p.row_tickets[rid] = 0;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  // warp w merges parts w, w + 4, w + 8, w + 12 (entries K..63 read as 0), then warp 0
  // merges the four results; warp 1 merges the normalisers meanwhile
  unsigned long long a0, a1;
  {
    const unsigned long long* kb = p.keys + rid * S * 64;
    unsigned long long x0[4], x1[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int l = w + 4 * j;
      x0[j] = (l < S && lane < K) ? __ldcg(kb + l * 64 + lane) : 0ull;
      x1[j] = (l < S && lane + 32 < K) ? __ldcg(kb + l * 64 + 32 + lane) : 0ull;
    }
    a0 = x0[0];
    a1 = x1[0];
#pragma unroll
    for (int j = 1; j < 4; ++j)
      if (w + 4 * j < S) {
        const ulonglong2 m2 = merge_top64(a0, a1, x0[j], x1[j], lane);
        a0 = m2.x;
        a1 = m2.y;
      }
  }
  s_dyn[w * 64 + lane] = a0;
  s_dyn[w * 64 + 32 + lane] = a1;
  __syncthreads();
  if (w == 0) {
#pragma unroll
    for (int w2 = 1; w2 < kThreads / 32; ++w2)
      if (w2 < S) {
        const ulonglong2 m2 = merge_top64(a0, a1, s_dyn[w2 * 64 + lane], s_dyn[w2 * 64 + 32 + lane], lane);
        a0 = m2.x;
        a1 = m2.y;
      }
  } else if (w == 1) {
    float M = -INFINITY, Sum = 0.f;
    uint32_t anybad = 0;
    for (int l = lane; l < S; l += 32) {
      const float4 st = __ldcg(p.stats + rid * S + l);
      merge_ms(M, Sum, st.x, st.y, c2);
      anybad |= __float_as_uint(st.z);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float m2 = __shfl_xor_sync(0xffffffffu, M, o), s2 = __shfl_xor_sync(0xffffffffu, Sum, o);
      merge_ms(M, Sum, m2, s2, c2);
    }
    anybad = __reduce_or_sync(0xffffffffu, anybad);
    if (lane == 0) {
      s_wm[0] = M;
      s_ws[0] = Sum;
      s_bad = (anybad || !(M > -INFINITY)) ? 1 : 0;
    }
  }
  __syncthreads();
  if (w == 0) {
    // log q = (x - max) / T - log sum exp((x_j - max) / T)
    const float M = s_wm[0], lnS = logf(s_ws[0]);
    int2* trow = p.table + rid * 64;
    if (lane < K) trow[lane] = make_int2(key_index(a0), __float_as_int((key_value(a0) - M) * invT - lnS));
    if (lane + 32 < K)
      trow[lane + 32] = make_int2(key_index(a1), __float_as_int((key_value(a1) - M) * invT - lnS));
    if (lane == 0 && s_bad) atomicOr(&p.seq_flags[b], SPEC_FLAG_BAD_LOGITS);
  }

  // the sequence's last row block selects the nodes
  __threadfence();
  __syncthreads();
  if (tid == 0) {
    const uint32_t prev = atomicAdd(&p.tickets[b], 1u);
    s_last = prev == static_cast<uint32_t>(p.rows - 1);
    if (s_last) p.tickets[b] = 0;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  int2* tab = reinterpret_cast<int2*>(s_dyn);
  for (int i = tid; i < p.rows * K; i += kThreads)
    tab[i] = __ldcg(p.table + (static_cast<int64_t>(b) * p.rows + i / K) * 64 + i % K);
  if (tid == 0) {
    uint32_t f = __ldcg(p.seq_flags + b);
    p.seq_flags[b] = 0;
    const int rt = p.root[b];
    if (rt < 0 || rt >= p.vocab) f |= SPEC_FLAG_BAD_TOKEN;
    s_flags = f;
  }
  __syncthreads();
  if (tid >= 32) return;
  if (p.nodes <= 33) select_nodes<1>(p, tab, K, b, s_flags, lane);
  else select_nodes<2>(p, tab, K, b, s_flags, lane);
}

// num_nodes = 1: the tree is its root
__global__ void tree_root_kernel(BuildParams p) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= p.batch) return;
  const int rt = p.root[b];
  const bool ok = rt >= 0 && rt < p.vocab;
  p.tokens[b] = ok ? rt : -1;
  p.parents[b] = -1;
  if (p.depth) p.depth[b] = ok ? 0 : -1;
  if (p.mask) p.mask[b] = ok ? 1ull : 0ull;
  if (!ok) set_status(p.status, SPEC_FLAG_BAD_TOKEN);
}

template <bool BF16, bool VEC>
cudaError_t launch_build_typed(const BuildParams& p, int smem, cudaStream_t s) {
  tree_build_kernel<BF16, VEC><<<dim3(p.splits, p.rows, p.batch), kThreads, smem, s>>>(p);
  return cudaGetLastError();
}

template <bool BF16, bool VEC>
cudaError_t launch_tree_typed(const TreeParams& p, cudaStream_t s) {
  tree_greedy_kernel<BF16, VEC><<<dim3(p.splits, p.nodes, p.batch), kThreads, 0, s>>>(p);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_tree_greedy(const spec_tree_accept_args_t& a, const TreeLayout& L, char* ws,
                               cudaStream_t stream, bool vec) {
  TreeParams p;
  p.batch = a.batch;
  p.nodes = a.num_nodes;
  p.vocab = a.vocab;
  p.splits = L.splits;
  p.elems_per_split = L.elems_per_split;
  p.target = a.target_logits;
  p.tokens = a.tokens;
  p.parents = a.parents;
  p.path = a.path;
  p.num_accepted = a.num_accepted;
  p.out_tokens = a.out_tokens;
  p.num_emitted = a.num_emitted;
  p.status = reinterpret_cast<uint32_t*>(ws);
  p.tickets = reinterpret_cast<uint32_t*>(ws + L.tickets);
  p.parts = reinterpret_cast<uint4*>(ws + L.parts);
  p.temperature = a.temperature;
  p.uniforms = a.uniforms;
  (void)cudaGetLastError();
  if (a.logits_dtype == SPEC_BF16)
    return vec ? launch_tree_typed<true, true>(p, stream) : launch_tree_typed<true, false>(p, stream);
  return vec ? launch_tree_typed<false, true>(p, stream) : launch_tree_typed<false, false>(p, stream);
}

cudaError_t launch_tree_commit(const spec_tree_commit_args_t& a, cudaStream_t stream) {
  (void)cudaGetLastError();
  const dim3 grid(2 * a.num_kv_heads, a.batch);
  if (a.head_dim == 64)
    tree_compact_kernel<64><<<grid, 128, 0, stream>>>(a);
  else
    tree_compact_kernel<128><<<grid, 128, 0, stream>>>(a);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  tree_commit_len_kernel<<<(a.batch + 7) / 8, 256, 0, stream>>>(a);
  return cudaGetLastError();
}

TreeBuildLayout tree_build_layout(const spec_tree_build_args_t& t, size_t base, int sms) {
  TreeBuildLayout L;
  const int budget = t.num_nodes - 1;
  L.rows = std::min(t.gamma - 1, budget);
  L.keff = std::min(std::min(t.top_k, t.vocab), std::max(budget, 1));
  const int lane = 64;  // split boundaries on 64 logits keep vector loads aligned
  const int nl = (t.vocab + lane - 1) / lane;
  const int64_t rows = static_cast<int64_t>(t.batch) * std::max(L.rows, 1);
  int64_t splits = (static_cast<int64_t>(kFiltBlocksPerSm) * sms + rows - 1) / rows;
  splits = std::max<int64_t>(1, std::min<int64_t>(splits, kFiltMaxSplits));
  if (splits > nl) splits = nl;
  L.elems_per_split = static_cast<int>((nl + splits - 1) / splits) * lane;
  L.splits = (t.vocab + L.elems_per_split - 1) / L.elems_per_split;
  const size_t nrows = static_cast<size_t>(t.batch) * std::max(L.rows, 1);
  L.tickets = base;
  L.seq_flags = ws_round(L.tickets + sizeof(uint32_t) * t.batch);
  L.row_tickets = ws_round(L.seq_flags + sizeof(uint32_t) * t.batch);
  L.keys = ws_round(L.row_tickets + sizeof(uint32_t) * nrows);
  L.stats = ws_round(L.keys + 64 * sizeof(uint64_t) * nrows * L.splits);
  L.table = ws_round(L.stats + 16 * nrows * L.splits);
  L.end = ws_round(L.table + 64 * 8 * nrows);
  const int k = L.keff;
  L.smem = static_cast<int>(8 * std::max(std::max(kTreeCandCap, 4 * 64), L.rows * k));
  return L;
}

cudaError_t launch_tree_build(const spec_tree_build_args_t& t, const TreeBuildLayout& L, char* ws,
                              cudaStream_t stream, bool vec) {
  BuildParams p;
  p.batch = t.batch;
  p.gamma = t.gamma;
  p.vocab = t.vocab;
  p.rows = L.rows;
  p.keff = L.keff;
  p.nodes = t.num_nodes;
  p.splits = L.splits;
  p.eps = L.elems_per_split;
  p.logits = t.drafter_logits;
  p.temperature = t.temperature;
  p.root = t.root_tokens;
  p.tokens = t.tokens;
  p.parents = t.parents;
  p.depth = t.depth;
  p.mask = t.tree_mask;
  p.status = reinterpret_cast<uint32_t*>(ws);
  p.tickets = reinterpret_cast<uint32_t*>(ws + L.tickets);
  p.seq_flags = reinterpret_cast<uint32_t*>(ws + L.seq_flags);
  p.row_tickets = reinterpret_cast<uint32_t*>(ws + L.row_tickets);
  p.keys = reinterpret_cast<unsigned long long*>(ws + L.keys);
  p.stats = reinterpret_cast<float4*>(ws + L.stats);
  p.table = reinterpret_cast<int2*>(ws + L.table);
  (void)cudaGetLastError();
  if (L.rows < 1) {
    tree_root_kernel<<<(t.batch + 127) / 128, 128, 0, stream>>>(p);
    return cudaGetLastError();
  }
  if (t.logits_dtype == SPEC_BF16)
    return vec ? launch_build_typed<true, true>(p, L.smem, stream) : launch_build_typed<true, false>(p, L.smem, stream);
  return vec ? launch_build_typed<false, true>(p, L.smem, stream) : launch_build_typed<false, false>(p, L.smem, stream);
}

}  // namespace specv
