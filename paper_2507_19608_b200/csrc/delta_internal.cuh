// Internal declarations shared by the translation units of the delta-attention library.
#pragma once
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>
#include <atomic>
#include "../../include/delta_attn.h"

namespace delta {

// Device counters (uint64) in the workspace.
enum CounterSlot {
  CNT_PREFILL_NNZ = 0, CNT_PREFILL_ELEMS, CNT_PREFILL_MACS_DONE, CNT_PREFILL_MACS_DENSE,
  CNT_DECODE_NNZ, CNT_DECODE_ELEMS, CNT_DECODE_MACS_DONE, CNT_DECODE_MACS_DENSE,
  CNT_STATUS,  // low 32 bits: device status word (0 = ok)
  CNT_SLOTS = 16,
  // the prefill counters are kept in CNT_SHARDS shards of 4 (nnz, elements, done, dense) behind
  // the plain slots, so that thousands of CTAs do not queue on four addresses; the host adds them
  CNT_SHARDS = 32,
  CNT_SHARD_BASE = CNT_SLOTS,
  CNT_TOTAL = CNT_SLOTS + 4 * CNT_SHARDS
};

constexpr int DELTA_CKPT_ROWS = 8;     // the chain kernel leaves its reference every 8 rows
constexpr int kMaxDecodeSplits = 64;   // split-KV partials per (batch, KV head)
constexpr int kDecodeChunkMax = 1024;  // keys per decode CTA (scores live in shared memory)

// Device pointers carved from the caller's workspace.
struct Workspace {
  float* dq;            // [B,H,T_max,d]
  uint32_t* mask;       // [B,H,T_max,d/32]
  uint16_t* row_nnz;    // [B,H,T_max]
  uint32_t* tile_nnz;   // [B,H,n_tiles]
  uint8_t* idx;         // [B,H,T_max,d]
  float* qhat_tile;     // [B,H,n_tiles,d]
  float* ckpt;          // [B,H,ceil(T_max/8),d] reference in front of every 8-row block (query deltas)
  float* qhat[2];       // [B,H,d] ping-pong (decode reads one, writes the other)
  float* R;             // [B,H,T_max]
  unsigned long long* counters;  // [CNT_TOTAL]
  float* dec_partial;   // [B,H_kv,kMaxDecodeSplits,g,(d+2)]
  uint32_t* dec_ticket; // [B,H_kv]
  float* kt;            // [B,H_kv,d,round_up(T_max,4)] channel-major fp32 keys (tensor-core prefill only)
  __nv_bfloat16* qhat_rows;  // [B,H,T_max,d] reference state after every row (telescoped prefill only)
  // compressed key-delta cache (key deltas, bf16): values, segment offsets, segment bases, pool
  // fill per KV head, and its own 32-row-aligned copies of the mask words and fired counts
  uint16_t* kp_vals;    // [B,H_kv,capacity]
  uint32_t* kp_segoff;  // [B,H_kv,segments+1]
  uint16_t* kp_base;    // [B,H_kv,segments,d]
  uint32_t* kp_used;    // [B,H_kv]
  uint32_t* kp_mask;    // [B,H_kv,segments*32,d/32]
  uint16_t* kp_nnz;     // [B,H_kv,segments*32]
  size_t zero_bytes;    // leading span of the workspace that a reset clears (q_hat, counters, tickets)
  size_t total_bytes;
};

struct Shape {
  int B, H, H_kv, d, T_max, n_tiles;
  int g() const { return H / H_kv; }
  int n_ckpt() const { return (T_max + DELTA_CKPT_ROWS - 1) / DELTA_CKPT_ROWS; }
};

// What a prefill kernel knows of one sequence.  A uniform batch is one entry whose heads are all
// B * H heads; a ragged batch has an entry per batch element, up to kSeqMax in one launch: its heads
// are the element's own, q_off the elements in front of it in the packed query and output arrays.
constexpr int kSeqMax = 16;
struct Seq {
  int T, W, b;
  size_t q_off;
};
template <int N> struct SeqList { Seq s[N]; };
// The sequences of a launch: n = 1 (uniform, covering the whole batch) or a ragged group.
// grid_heads: the query heads of the whole call where a launch covers a part of a uniform batch, else 0.  The
// forms of the attention kernels follow the size of the grid and round differently (which keys share a
// running maximum, whose probabilities meet): the call's grid decides, not the part's, so that a
// head's result does not depend on how its call was cut.
struct SeqBatch {
  int n, T_longest;
  bool ragged;
  int grid_heads = 0;
  int beside = -1;      // >= 0: the telescoped attention kernel comes next, with this form, and may begin beside the chain
  bool* with_finish = nullptr;      // the attention launch may do the finish kernel's work too, and says here that it does
  Seq s[kSeqMax];
  // query heads of the grid that chooses the form (ragged: of every sequence's grid)
  long form_heads(const Shape& sh) const { return grid_heads ? grid_heads : (long)(ragged ? 1 : sh.B) * sh.H; }
};

// What a launcher does once per device (function attributes, which the runtime keeps): has it been
// done on the current device / it has.  (Devices past 63 do it every time.)
inline int device_slot() {
  int dev = 0;
  return (cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < 64) ? dev : -1;
}
inline bool device_done(const std::atomic<uint64_t>& mask) {
  const int dev = device_slot();
  return dev >= 0 && ((mask.load(std::memory_order_acquire) >> dev) & 1u);
}
inline void device_mark(std::atomic<uint64_t>& mask) {
  const int dev = device_slot();
  if (dev >= 0) mask.fetch_or(1ull << dev, std::memory_order_release);
}

void count_launch(int n = 1);
// Records the text of a failed CUDA runtime call for delta_last_cuda_error; returns DELTA_ERR_CUDA.
delta_status_t cuda_fail(cudaError_t e);

// K1a: token-sequential delta chain (Eq. 2-3): the reference in front of every 8-row block and
// every 64-row tile, and the final reference.
// key_stream: the stream is K in the KV-cache layout, one chain set per KV head (strategy 3).
// reverse: rows are taken from T-1 down to 0 (strategy 2; query stream only).
// zero_ptr, zero_bytes: a span (16-byte aligned, a multiple of 16 bytes) that the kernel's first
// CTA clears before anything else: the deferred clearing of a state reset (none if null).
// x: the packed queries or the key cache.
cudaError_t launch_delta_chain(const Shape& s, const Workspace& w, const void* x, const SeqBatch& seqs, float theta,
                               int dtype, int init, bool key_stream, bool reverse, void* zero_ptr, size_t zero_bytes,
                               cudaStream_t st);
// Does it go by the table kernel?  That one also tells, at chain_progress where that is not null, a word per (head, 32
// channels), kProgressStride apart (a line each), how many 64-row stages' references are in memory, in processing order;
// never the last one, which a kernel behind takes from that kernel's end.
constexpr int kProgressStride = 32;
bool chain_by_tables(const Shape& s, const SeqBatch& seqs, int dtype, bool key_stream);
unsigned* chain_progress(const Shape& s, const Workspace& w, const SeqBatch& seqs, int dtype, bool key_stream);
// K1b: row-parallel finish: delta values, mask words and (key stream) reference rows from the
// 8-row checkpoints; counts, compacted indices, Eq. 6 counters, the decode hand-off row
// R(T-1)[j] = q_hat . k_j and (want_kt) the channel-major fp32 key copy.
// SMs of the current device (queried once per device).
int device_sm_count();
// programmatic: 1 = launched with programmatic stream serialisation (its launch overlaps the end
// of the kernel in front; the kernel waits for that kernel's completion itself); 2 = the same, but
// the kernel does not wait before its work, only before its end: the kernel in front releases it once the
// chain kernel's results are complete (query deltas behind the telescoped or the fp32 attention
// kernel); 0 = an ordinary launch.
cudaError_t launch_delta_finish(const Shape& s, const Workspace& w, const void* q, const void* k, const SeqBatch& seqs,
                                float theta, int shape, int dtype, int init, bool want_kt,
                                bool key_stream, bool reverse, int programmatic, cudaStream_t st);
// K2 at fp32 precision (three-part bf16 products on the tensor cores), either dtype; reads the chain kernel's
// checkpoints and nothing of the finish kernel's.
cudaError_t launch_hybrid_attn_f32(const Shape& s, const Workspace& w, const void* q, const void* k, const void* v,
                                       void* out, const SeqBatch& seqs, float theta, int init, int shape, int dtype,
                                       cudaStream_t st);
// K3: one decode step.
cudaError_t launch_decode_step(const Shape& s, const Workspace& w, const void* q_new,
                               const void* k_new, const void* v_new, void* k_cache, void* v_cache,
                               void* out, int n, float theta, int window, int dtype, int qhat_sel,
                               cudaStream_t st);

// Host-side cache of a cache's tensor map (encoded once per cache pointer, not per step).
struct DecodeTmapCache {
  const void* ptr = nullptr;
  alignas(64) unsigned char map[128];
};
// K3 for bf16 caches (query and key deltas; key: w.qhat_rows is the reference-key cache).  n: tokens
// seen (the longest sequence's); n_b: null, or the tokens seen by every batch element of a ragged
// batch; behind_step: the state's last kernel was a decode step, not a prefill's; maps: the state's tensor
// maps of the key, value and reference-key caches.
bool decode_mma_applies(const Shape& s, int dtype);
cudaError_t launch_decode_step_mma(const Shape& s, const Workspace& w, const void* q_new, const void* k_new,
                                   const void* v_new, void* k_cache, void* v_cache, void* out, int n, const int* n_b,
                                   float theta, int window, int qhat_sel, bool key, bool packed, bool behind_step,
                                   DecodeTmapCache* maps, cudaStream_t st);
// K3 for fp32 caches (query deltas), arguments as above.
cudaError_t launch_decode_step_f32(const Shape& s, const Workspace& w, const void* q_new, const void* k_new,
                                   const void* v_new, void* k_cache, void* v_cache, void* out, int n, const int* n_b,
                                   float theta, int window, int qhat_sel, DecodeTmapCache* map, cudaStream_t st);
// The compressed key-delta cache (packed = true above decodes from it): the kernel that builds it
// behind a prefill, and its geometry (values per KV head at most, 32-row segments).
size_t keypack_capacity(int T_max, int d);
int keypack_segments(int T_max);
cudaError_t launch_pack_keys(const Shape& s, const Workspace& w, const void* k, int T, cudaStream_t st);
// K3 (key deltas) on the FP32 pipes.
cudaError_t launch_decode_step_key(const Shape& s, const Workspace& w, const void* q_new,
                                   const void* k_new, const void* v_new, void* k_cache, void* v_cache,
                                   void* out, int n, float theta, int window, int qhat_sel,
                                   cudaStream_t st);

// ---- bounds-checking build ------------------------------------------------------------
// DELTA_IN(index, extent, counters) guards a global access whose index a kernel computed by
// hand: true in the regular build (the guard compiles away); in a -DDELTA_DEBUG_BOUNDS build
// false for an index outside [0, extent), with DELTA_ERR_BOUNDS recorded in the status word, so
// the access is skipped instead of made (no trap, no assert: the context stays usable).
#ifdef DELTA_DEBUG_BOUNDS
__device__ __forceinline__ bool delta_in_bounds(size_t idx, size_t extent, unsigned long long* counters) {
  if (idx < extent) return true;
  atomicMax(&counters[CNT_STATUS], (unsigned long long)DELTA_ERR_BOUNDS);
  return false;
}
#define DELTA_IN(idx, extent, counters) delta_in_bounds((size_t)(idx), (size_t)(extent), (counters))
#else
#define DELTA_IN(idx, extent, counters) true
#endif

// ---- small device helpers -------------------------------------------------------------
__device__ __forceinline__ float to_f32(float x) { return x; }
__device__ __forceinline__ float to_f32(__nv_bfloat16 x) { return __bfloat162float(x); }
template <typename T> __device__ __forceinline__ T from_f32(float x);
template <> __device__ __forceinline__ float from_f32<float>(float x) { return x; }
template <> __device__ __forceinline__ __nv_bfloat16 from_f32<__nv_bfloat16>(float x) {
  return __float2bfloat16_rn(x);
}

// Number of in-window keys of query row i.  The causal pair (i, j <= i) is inside the exact window iff
// i / W == j / W (shape 0, block) or i - j < W (shape 1, sliding).
__host__ __device__ __forceinline__ int in_window_count(int i, int W, int shape) {
  if (W <= 0) return 0;
  return shape == 0 ? (i % W) + 1 : (i + 1 < W ? i + 1 : W);
}

// Number of queries i in [j, T) whose pair (i, j) is inside the exact window (key j's column).
__host__ __device__ __forceinline__ int in_window_col_count(int j, int T, int W, int shape) {
  if (W <= 0) return 0;
  const int last = shape == 0 ? (j / W + 1) * W : j + W;   // first query past the window
  return (last < T ? last : T) - j;
}

}  // namespace delta
