// Internal declarations shared by the CUDA translation units of libspecverify.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "spec_verify.h"

namespace specv {

// ----------------------------------------------------------------------------------
// Workspace layout. Every region starts on a 256-byte boundary. The header holds the
// status word; counters are per-call tickets that the last arriving block resets.
// ----------------------------------------------------------------------------------
constexpr size_t kWsAlign = 256;
constexpr size_t kWsHeader = 256;  // [0] = status word (uint32)

inline size_t ws_round(size_t x) { return (x + kWsAlign - 1) / kWsAlign * kWsAlign; }

// --- acceptance ---
// 128-thread blocks with few registers, so that they fit beside a resident attention
// block when the verify step overlaps the two parts.
constexpr int kStatsThreads = 128;
constexpr int kStatsChunk = 4096;                          // vocab elements per row item
constexpr int kSampleThreads = 128;
constexpr int kDecideThreads = 512;                        // one block per sequence
constexpr int kSampleSlice = 4096;                         // vocab elements per sample block
constexpr int kSamplePerThread = kSampleSlice / kSampleThreads;  // contiguous per thread

struct RowPartial {  // one (sequence, row, vocab chunk) item of the row statistics
  float m;           // max raw logit of the chunk (-inf if none finite)
  float s;           // sum exp((l - m) / T) over the chunk (T > 0 rows)
  int32_t arg;       // lowest index of the chunk maximum (greedy rows)
  uint32_t bad;      // NaN / +inf seen
};

struct AcceptLayout {
  size_t tickets;      // uint32 [batch]
  size_t partials;     // RowPartial [batch][2*gamma-1][nchunk]
  size_t records;      // 32-byte decision record [batch] (n and the final draw's normalisers)
  size_t slice_sums;   // float4 [batch][nslice] = (residual sum, p sum, residual last, p last)
  size_t end;
  int nchunk, nslice;
};

AcceptLayout accept_layout(const spec_accept_args_t& a, size_t base);

// --- filtered acceptance ---
constexpr int kFilterMaxTopK = SPEC_FILTER_MAX_TOP_K;
constexpr int kFiltLaneElems = 64;    // contiguous logits per lane (at the smallest lane size)
constexpr int kFiltMaxCand = 2048;    // candidates one row block holds at most
constexpr int kFiltMaxLanes = 4096;   // lane maxima one row block keeps in shared memory
constexpr int kFiltBlocksPerSm = 8;   // row blocks resident per SM (128 threads each)
constexpr int kFiltMaxSplits = 16;    // blocks one row may be split across
constexpr int kRowThreads = 128;      // threads of a filtered row block

struct FiltRow {    // one (sequence, row) result of the filtered row kernel
  int32_t nkeep;    // kept tokens (top-k, then top-p)
  int32_t argmax;   // lowest index of the row maximum
  uint32_t flags;   // 1: NaN / +inf / no finite logit; 2: top_k or top_p out of range
  int32_t pad;
};

struct FilterLayout {
  size_t tickets;  // uint32 [batch]: rows of the sequence finished (reset by the last)
  size_t rows;     // FiltRow [batch][2*gamma-1]
  size_t kept;     // (int32 token, fp32 p') [batch][2*gamma-1][max_top_k], rank order
  size_t row_tickets;  // uint32 [batch][2*gamma-1]: splits of the row finished (splits > 1)
  size_t lanes_g;  // uint32 [batch][2*gamma-1][nlanes]: lane maxima (splits > 1)
  size_t parts;    // 16 B [batch][2*gamma-1][splits]: each split's maximum and bad flag
  size_t end;
  int lane_shift;  // lanes hold kFiltLaneElems << lane_shift logits
  int nlanes;      // ceil(vocab / lane size) <= kFiltMaxLanes
  int splits;      // blocks per row
  int lanes_per_split;
  int cand_cap;    // candidates one block holds (a power of two)
  int smem_a;      // bytes of the first dynamic shared region
};

// draw = true: the layout of the draft-side draw (gamma drafter rows per sequence).
FilterLayout filter_layout(const spec_accept_args_t& a, int max_top_k, size_t base, int sms,
                           bool draw = false);

// --- draft-side sampling ---
constexpr size_t kDraftMaxSmem = 200 * 1024;  // lane summaries of one unfiltered draw block
struct DraftLayout {
  size_t tickets;      // uint32 [batch]: rows of the sequence finished (reset by the last)
  size_t row_flags;    // uint32 [batch][gamma]
  size_t row_tickets;  // uint32 [batch][gamma]: splits of the row finished (splits > 1)
  size_t lanes_g;      // float2 [batch][gamma][nlanes]: lane (max, sum) (splits > 1)
  size_t parts;        // 16 B [batch][gamma][splits]: each split's maximum and bad flag
  size_t end;
  size_t smem;         // dynamic shared memory of one block: nlanes x 8 B
  int lane_elems;      // 64 with 16-byte loads, 32 with element loads
  int nlanes, splits, lanes_per_split;
};

DraftLayout draft_layout(const spec_draft_args_t& a, size_t base, int sms, bool vec);
cudaError_t launch_draft(const spec_draft_args_t& a, const DraftLayout& L, char* ws,
                         cudaStream_t stream, bool vec);
cudaError_t launch_commit(const spec_commit_args_t& a, cudaStream_t stream);

// --- tree verification ---
struct TreeLayout {
  size_t tickets;      // uint32 [batch]: parts of the sequence's rows finished
  size_t parts;        // 16 B [batch][nodes][splits]: (argmax key, max key, bad, sum of 2^..)
  size_t end;
  int splits, elems_per_split;
};

TreeLayout tree_layout(int batch, int nodes, int vocab, size_t base, int sms, bool vec);
cudaError_t launch_tree_greedy(const spec_tree_accept_args_t& a, const TreeLayout& L, char* ws,
                               cudaStream_t stream, bool vec);
cudaError_t launch_tree_commit(const spec_tree_commit_args_t& a, cudaStream_t stream);

constexpr int kTreeCandCap = 512;  // candidates of one row part ranked in shared memory

struct TreeBuildLayout {
  size_t tickets;      // uint32 [batch]: position rows of the sequence finished
  size_t seq_flags;    // uint32 [batch]: flags its rows raised
  size_t row_tickets;  // uint32 [batch][rows]: parts of the row finished
  size_t keys;         // uint64 [batch][rows][splits][64]: each part's ranked candidate keys
  size_t stats;        // float4 [batch][rows][splits]: (max, sum of exponentials, bad, -)
  size_t table;        // int2 [batch][rows][64]: the position's (token, log q), ranked
  size_t end;
  int rows;            // positions that can hold a node: min(gamma - 1, num_nodes - 1)
  int keff;            // candidates used per position: min(top_k, vocab, num_nodes - 1)
  int splits, elems_per_split;
  int smem;            // dynamic shared memory of a block, bytes
};

TreeBuildLayout tree_build_layout(const spec_tree_build_args_t& t, size_t base, int sms);
cudaError_t launch_tree_build(const spec_tree_build_args_t& t, const TreeBuildLayout& L, char* ws,
                              cudaStream_t stream, bool vec);

// --- attention ---
// A unit that was split between blocks, as the block that begins inside it leaves it to the
// merge kernel.
struct alignas(16) SplitUnit {
  int b, g, rt;    // the unit: sequence, KV head (or group of heads), row tile
  int slot0, nsl;  // its partial slots; nsl = 0: the block begins at a unit's start
  int k;           // the block's left boundary is the unit's k-th
  int pad[2];
};

struct AttnPlan {
  int path;          // SPEC_ATTN_CUDA_CORES or SPEC_ATTN_TENSOR_CORES
  int keys_on_lanes; // tensor cores: the keys-on-lanes kernel (attn_kl.cu), else row tiles
  int heads;         // > 0: the small-group kernel (attn_mma.cu) with this many KV heads per block
  int head_pair;     // row tiles: one block serves two adjacent KV heads (8 KB page boxes)
  int rows;          // (Hq/Hkv) * gamma
  int rows_per_cta;  // rows one block handles (a row tile)
  int row_tiles;     // ceil(rows / rows_per_cta)
  int key_tile;      // keys per pipeline step
  int max_keys;      // max_pages_per_seq * page_size
  int nsplit;        // KV splits per (sequence, kv head, row tile) (CUDA-core path)
  int tiles_per_split;
  int grid;          // blocks launched
  int slot_rows;     // rows per partial slot
  int64_t slots;     // partial slots
  size_t tickets, splits, partial_o, partial_ml, end;
};

AttnPlan attn_plan(const spec_attn_args_t& a, size_t base, int num_sms, int path_override);

// ----------------------------------------------------------------------------------
// Launchers (defined in the .cu files); all return cudaGetLastError() of the launch.
// ----------------------------------------------------------------------------------
// overlap_prior: launch the acceptance kernels as programmatic dependents of the kernel
// just launched on the stream (the attention kernel of the same verify step, which
// reads none of their inputs and writes none of their outputs).
cudaError_t launch_accept(const spec_accept_args_t& a, const AcceptLayout& L, char* ws,
                          int num_sms, cudaStream_t stream, bool overlap_prior = false);
// With draw_tokens set, draws every drafter row's token instead of verifying (only the
// logits, temperature, uniforms and batch shape of a are read).
cudaError_t launch_accept_filtered(const spec_accept_args_t& a, const spec_filter_args_t& f,
                                   const FilterLayout& L, char* ws, cudaStream_t stream,
                                   bool overlap_prior = false, int32_t* draw_tokens = nullptr,
                                   float* draw_q = nullptr);
cudaError_t launch_attn_simt(const spec_attn_args_t& a, const AttnPlan& P, char* ws,
                             cudaStream_t stream);
// starve (test hook only): the kernel's producers issue no copies, so its bounded waits
// run out and it returns with SPEC_FLAG_TIMEOUT set.
cudaError_t launch_attn_tc(const spec_attn_args_t& a, const AttnPlan& P, char* ws,
                           cudaStream_t stream, bool starve = false);
cudaError_t launch_attn_mma(const spec_attn_args_t& a, const AttnPlan& P, char* ws,
                            cudaStream_t stream, bool starve = false);
// KV heads one block of the small-group kernel serves (2, 4 or 8), or 0 where it does not
// apply: more than kMmaMaxRows query rows per KV head, an odd Hkv, or a batch whose prefix
// sums do not fit beside its stages.
int mma_heads(const spec_attn_args_t& a, int rows);
constexpr int kMmaMaxRows = 32;
constexpr int kMmaMinTiles = 2;  // 32 KB tiles a block takes at least (range_count)
cudaError_t launch_attn_kl(const spec_attn_args_t& a, const AttnPlan& P, char* ws,
                           cudaStream_t stream);
cudaError_t launch_philox(uint64_t seed, uint64_t offset, int64_t n, float* out, cudaStream_t s);
cudaError_t launch_noise(uint64_t seed, uint64_t offset, int64_t n, int32_t vocab, int32_t* out,
                         cudaStream_t s);

// Rows of one CUDA-core block and of one tensor-core block.
constexpr int kSimtRowTile = 16;
constexpr int kSimtKeyTile = 64;
constexpr int kSimtThreads = 128;
constexpr int kTcKeyTile = 64;
constexpr int kTcMaxRows = 256;  // two M = 128 tiles per block
// The keys-on-lanes tensor-core kernel (attn_kl.cu): 128 keys per tile, at most 64 query
// rows per KV head, head_dim 128, batch prefix sums in shared memory.
constexpr int kKlKeyTile = 128;
constexpr int kKlMaxRows = 64;
constexpr int kKlMaxBatch = 2048;
size_t kl_smem_bytes(int rows, int batch);

int tc_min_rows();

// The device a stream belongs to. cudaStreamGetDevice is not allowed on a capturing
// stream (it invalidates the capture), so a stream under capture is taken to belong
// to the current device, the one its captured work must run on.
inline cudaError_t stream_device(cudaStream_t stream, int* dev) {
  if (stream != nullptr) {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    const cudaError_t e = cudaStreamIsCapturing(stream, &cs);
    if (e != cudaSuccess) return e;
    if (cs == cudaStreamCaptureStatusNone) return cudaStreamGetDevice(stream, dev);
  }
  return cudaGetDevice(dev);
}
// Cached multiprocessor count of a device (asked once per device).
int device_sm_count(int dev);

// Makes the device of `stream` current for the duration of one entry point and puts
// the caller's current device back when it goes out of scope, so that no call changes
// which device the calling thread has current. `ok` is false when the device could
// not be found or selected.
struct DeviceScope {
  int dev = 0, prev = -1, sms = 0;
  bool ok = false;
  explicit DeviceScope(cudaStream_t stream) {
    if (cudaGetDevice(&prev) != cudaSuccess) { prev = -1; return; }
    if (stream_device(stream, &dev) != cudaSuccess) return;
    if (dev != prev && cudaSetDevice(dev) != cudaSuccess) return;
    sms = device_sm_count(dev);
    ok = true;
  }
  ~DeviceScope() {
    if (prev >= 0 && dev != prev) cudaSetDevice(prev);
  }
  DeviceScope(const DeviceScope&) = delete;
  DeviceScope& operator=(const DeviceScope&) = delete;
};

int tc_ctas_per_sm(int head_dim, int rows_per_cta, int rows, int batch, bool head_pair);
size_t tc_smem_bytes(int head_dim, int rows_per_cta, int rows, int batch, bool head_pair);
// Whether the row-tile kernel serves two adjacent KV heads per block: KV groups of 33 to
// 64 rows, an even Hkv, and the batch's prefix sums fit beside its stages.
bool tc_head_pair(int head_dim, int rows, int num_kv_heads, int batch);
constexpr int kTcMaxBatch = 4096;  // batch prefix sums live in shared memory
constexpr size_t kTcMaxSmem = 227u * 1024u;  // dynamic shared memory of one block
// A kernel's limit of dynamic shared memory belongs to the function, not to a call: it is
// always set to the most any call can need, so that no host thread lowers it between another
// thread's setting and its launch.
template <class Kernel>
cudaError_t allow_smem(Kernel kernel, size_t most) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(most));
}

}  // namespace specv

// ----------------------------------------------------------------------------------
// Device helpers
// ----------------------------------------------------------------------------------
#ifdef __CUDACC__
namespace specv {

__device__ __forceinline__ float bf16_bits_to_f32(uint32_t h) { return __uint_as_float(h << 16); }

// 2^x via the PTX approximate base-2 exponential (relative error about 2^-22;
// results below 2^-126 flush to zero).
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// The 16-byte granule at `a` (16-byte aligned) of a tensor that occupies [lo, hi), whose
// first and last granules may hold bytes of others: those are read element by element
// (E bytes each), bytes outside as zeros.
template <int E>
__device__ __forceinline__ uint4 load_granule(const char* a, const char* lo, const char* hi) {
  if (a >= lo && a + 16 <= hi) return __ldg(reinterpret_cast<const uint4*>(a));
  uint32_t w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
  for (int i = 0; i < 16 / E; ++i) {
    const char* x = a + i * E;
    if (x >= lo && x + E <= hi) {
      if (E == 4) w[i] = __ldg(reinterpret_cast<const uint32_t*>(x));
      else w[i / 2] |= static_cast<uint32_t>(__ldg(reinterpret_cast<const uint16_t*>(x))) << (16 * (i & 1));
    }
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}

// Granules n = first, first + stride, .. below `count` from `at` (N of them a thread, zeros
// past the count) of a tensor [lo, hi): whole loads without a test each where all of them
// lie inside, which is everywhere but at the tensor's ends (a test for each load: the
// acceptance of 32 x 8 rows of 100,003 bf16 logits took 48.9 us instead of 45.2, the block
// draws 57.1 instead of 55.3, filtered rows of 50,257 fp32 logits 28.9 instead of 28.3).
template <int E, int N>
__device__ __forceinline__ void load_granules(uint4* g, const char* at, int first, int stride, int count,
                                              const char* lo, const char* hi) {
  if (at >= lo && at + 16 * static_cast<int64_t>(count) <= hi) {
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const int n = first + i * stride;
      g[i] = n < count ? __ldg(reinterpret_cast<const uint4*>(at) + n) : make_uint4(0u, 0u, 0u, 0u);
    }
  } else {
#pragma unroll 1
    for (int i = 0; i < N; ++i) {
      const int n = first + i * stride;
      const uint4 v = n < count ? load_granule<E>(at + 16 * n, lo, hi) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
      for (int k = 0; k < N; ++k)
        if (k == i) g[k] = v;
    }
  }
}

// Reduction of 8 values over the threads of a group of G, all 8 together: the tree of a
// butterfly (neighbours first), but each of the first three exchanges halves the values a
// thread carries, 7 to 9 shuffles instead of 8 log2 G. Thread i of the group gets value
// i & 7; v is overwritten.
template <int G, class Op>
__device__ __forceinline__ float reduce8(float* v, int i, Op op) {
  const bool b0 = i & 1, b1 = i & 2, b2 = i & 4;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float keep = b0 ? v[2 * j + 1] : v[2 * j];
    v[j] = op(keep, __shfl_xor_sync(0xffffffffu, b0 ? v[2 * j] : v[2 * j + 1], 1));
  }
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const float keep = b1 ? v[2 * j + 1] : v[2 * j];
    v[j] = op(keep, __shfl_xor_sync(0xffffffffu, b1 ? v[2 * j] : v[2 * j + 1], 2));
  }
  float r = op(b2 ? v[1] : v[0], __shfl_xor_sync(0xffffffffu, b2 ? v[0] : v[1], 4));
#pragma unroll
  for (int o = 8; o < G; o <<= 1) r = op(r, __shfl_xor_sync(0xffffffffu, r, o));
  return r;
}
// Two fp32 operations in one instruction (the packed forms).
__device__ __forceinline__ uint64_t pack2(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

// The weight 2^((x - m) c) may be taken as 2^(x c - m c), one multiply-add with m c rounded,
// while |m c| <= kFusedMax: the rounding, at most 2^-19, is 1.3e-6 of every weight. Beyond it
// (large logits, low temperatures) it grows with m c, to factors of 2 at 2^24 and to overflow,
// and the difference is formed first.
constexpr float kFusedMax = 64.f;
__device__ __forceinline__ bool past_fused(float m, float c) { return fabsf(m * c) > kFusedMax && m > -INFINITY; }

// Programmatic dependent launch: let the next kernel on the stream start now / wait for
// the kernel this one depends on (no-ops for kernels launched without the attribute).
__device__ __forceinline__ void pdl_launch_dependents() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void pdl_wait_prior() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ void set_status(uint32_t* status, uint32_t flag) {
  atomicOr(status, flag);
}

constexpr float kLog2e = 1.4426950408889634f;

}  // namespace specv
#endif
