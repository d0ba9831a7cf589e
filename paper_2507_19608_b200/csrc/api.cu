// C ABI of the delta-attention library: argument checks, workspace carving, launch order.
#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>
#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "delta_internal.cuh"
#include "k2_tc.cuh"

namespace delta {
static std::atomic<unsigned long long> g_launches{0};
void count_launch(int n) { g_launches.fetch_add((unsigned long long)n, std::memory_order_relaxed); }
static thread_local char g_cuda_err[256] = "";
delta_status_t cuda_fail(cudaError_t e) {
  snprintf(g_cuda_err, sizeof(g_cuda_err), "%s: %s", cudaGetErrorName(e), cudaGetErrorString(e));
  return DELTA_ERR_CUDA;
}
}  // namespace delta

using namespace delta;

// NVTX range over an entry point (shows up in a timeline profiler; free when none is attached).
namespace {
struct NvtxRange {
  explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
  ~NvtxRange() { nvtxRangePop(); }
};
}  // namespace

struct delta_state {
  delta_config_t cfg;
  Shape shape;
  Workspace ws;
  void* base;
  size_t bytes;
  int n;         // tokens seen (of the longest sequence, after a prefill over sequences of different lengths)
  std::vector<int> n_b;   // tokens seen per batch element
  bool ragged = false;    // the batch elements stand at different positions
  int qhat_sel;  // which q_hat buffer is current
  int forced_kernel;  // -1 auto, else a kernel of delta_state_set_prefill_kernel
  // Eq. 6 bookkeeping that needs no device work: sum of window lengths and sequence lengths
  double win_sum[2], len_sum[2];
  DecodeTmapCache dec_maps[3];     // tensor maps of the key, value and reference-key caches the decode steps read
  int forced_decode_kernel = -1;   // -1: chosen per step
  bool stepped = false;            // a decode step has been enqueued behind the prefill
  bool key_cache_packed = false;   // key deltas: decode from the compressed key-delta cache
  // optional per-kernel timing of prefill (host-side event objects)
  bool profiling = false, profiled = false;
  // a reset has been asked for and the chain kernel of the next prefill does the clearing (no
  // launch of its own: a memset in front of the chain kernel costs 2 us of a 38 us step)
  bool zero_pending = false;
  cudaEvent_t ev[5] = {nullptr, nullptr, nullptr, nullptr, nullptr};
};

static size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

static delta_status_t check_config(const delta_config_t* c) {
  if (!c) return DELTA_ERR_INVALID_ARG;
  if (c->B < 1 || c->H < 1 || c->H_kv < 1 || c->T_max < 1) return DELTA_ERR_INVALID_ARG;
  if (c->H % c->H_kv != 0) return DELTA_ERR_INVALID_ARG;
  if (c->dtype != DELTA_F32 && c->dtype != DELTA_BF16) return DELTA_ERR_INVALID_ARG;
  if (c->prefill_window != DELTA_WIN_BLOCK && c->prefill_window != DELTA_WIN_SLIDING)
    return DELTA_ERR_INVALID_ARG;
  if (c->init != DELTA_INIT_BASIS_EXACT && c->init != DELTA_INIT_ZERO_STATE)
    return DELTA_ERR_INVALID_ARG;
  if (c->source != DELTA_SRC_QUERY && c->source != DELTA_SRC_KEY && c->source != DELTA_SRC_QUERY_BOTTOM_UP)
    return DELTA_ERR_INVALID_ARG;
  if (c->d != 64 && c->d != 128) return DELTA_ERR_UNSUPPORTED;
  // key deltas (strategy 3) are served by the telescoped tensor-core kernel only
  // and so are bottom-up query deltas (strategy 2)
  if (c->source != DELTA_SRC_QUERY && !(c->dtype == DELTA_BF16 && tcq_kernel_shape(c->d)))
    return DELTA_ERR_UNSUPPORTED;
  const int g = c->H / c->H_kv;
  if (g != 1 && g != 2 && g != 4 && g != 8) return DELTA_ERR_UNSUPPORTED;
  if (c->T_max > kMaxDecodeSplits * kDecodeChunkMax) return DELTA_ERR_UNSUPPORTED;
  if ((long long)c->B * c->H > 65535) return DELTA_ERR_UNSUPPORTED;
  return DELTA_OK;
}

// Carve the workspace; base may be null (size query).
static void carve(const delta_config_t& c, char* base, Workspace* w) {
  const size_t BH = (size_t)c.B * c.H, BKV = (size_t)c.B * c.H_kv;
  const size_t nt = (c.T_max + DELTA_TILE_ROWS - 1) / DELTA_TILE_ROWS;
  const size_t g = c.H / c.H_kv;
  size_t off = 0;
  auto take = [&](size_t bytes) { char* p = base ? base + off : nullptr; off += align_up(bytes, 256); return p; };
  // what a reset has to zero comes first, as one contiguous span: the two reference buffers
  // (Eq. 3: the reference starts at 0), the counters and the decode tickets.  The score row R
  // needs no zeroing: prefill writes entries 0..T-1 and a decode step reads only entries below
  // its position.
  w->qhat[0] = (float*)take(BH * c.d * 4);
  w->qhat[1] = (float*)take(BH * c.d * 4);
  w->counters = (unsigned long long*)take(CNT_TOTAL * 8);
  w->dec_ticket = (uint32_t*)take(BKV * 4);
  w->zero_bytes = off;
  w->dq = (float*)take(BH * c.T_max * c.d * 4);
  w->mask = (uint32_t*)take(BH * c.T_max * (c.d / 32) * 4);
  w->row_nnz = (uint16_t*)take(BH * c.T_max * 2);
  w->tile_nnz = (uint32_t*)take(BH * nt * 4);
  w->idx = (uint8_t*)take(BH * c.T_max * c.d);
  w->qhat_tile = (float*)take(BH * nt * c.d * 4);
  w->ckpt = (float*)take(BH * (((size_t)c.T_max + DELTA_CKPT_ROWS - 1) / DELTA_CKPT_ROWS) * c.d * 4);
  w->R = (float*)take(BH * c.T_max * 4);
  w->dec_partial = (float*)take(BKV * kMaxDecodeSplits * g * (c.d + 2) * 4);
  w->kt = (c.dtype == DELTA_BF16 && tc_kernel_shape(c.d))
              ? (float*)take(BKV * c.d * (((size_t)c.T_max + 3) / 4 * 4) * 4) : nullptr;
  w->qhat_rows = (c.dtype == DELTA_BF16 && tcq_kernel_shape(c.d))
                     ? (__nv_bfloat16*)take(BH * c.T_max * c.d * 2) : nullptr;
  if (c.source == DELTA_SRC_KEY && c.dtype == DELTA_BF16) {
    // compressed key-delta cache: sized for the worst case (every element fires)
    const size_t nseg = (size_t)keypack_segments(c.T_max);
    w->kp_vals = (uint16_t*)take(BKV * keypack_capacity(c.T_max, c.d) * 2);
    w->kp_segoff = (uint32_t*)take(BKV * (nseg + 1) * 4);
    w->kp_base = (uint16_t*)take(BKV * nseg * c.d * 2);
    w->kp_used = (uint32_t*)take(BKV * 4);
    w->kp_mask = (uint32_t*)take(BKV * nseg * 32 * (c.d / 32) * 4);
    w->kp_nnz = (uint16_t*)take(BKV * nseg * 32 * 2);
  } else {
    w->kp_vals = nullptr; w->kp_segoff = nullptr; w->kp_base = nullptr; w->kp_used = nullptr;
    w->kp_mask = nullptr; w->kp_nnz = nullptr;
  }
  w->total_bytes = off;
}

extern "C" {

delta_status_t delta_state_workspace_bytes(const delta_config_t* cfg, size_t* bytes) {
  if (!bytes) return DELTA_ERR_INVALID_ARG;
  delta_status_t s = check_config(cfg);
  if (s != DELTA_OK) return s;
  Workspace w;
  carve(*cfg, nullptr, &w);
  *bytes = w.total_bytes;
  return DELTA_OK;
}

// defer: leave the clearing of the device span to the next prefill (see zero_pending)
static delta_status_t zero_state(delta_state* st, cudaStream_t stream, bool defer) {
  if (defer) {
    st->zero_pending = true;
  } else {
    // one memset: the span carve() put at the front of the workspace
    cudaError_t e = cudaMemsetAsync(st->base, 0, st->ws.zero_bytes, stream);
    if (e != cudaSuccess) return cuda_fail(e);
    st->zero_pending = false;
  }
  st->n = 0;
  st->n_b.assign((size_t)st->cfg.B, 0);
  st->ragged = false;
  st->stepped = false;
  st->qhat_sel = 0;
  st->win_sum[0] = st->win_sum[1] = st->len_sum[0] = st->len_sum[1] = 0.0;
  return DELTA_OK;
}

delta_status_t delta_state_init(const delta_config_t* cfg, void* workspace, size_t workspace_bytes,
                                void* stream, delta_state_t** out) {
  if (!out) return DELTA_ERR_INVALID_ARG;
  *out = nullptr;
  delta_status_t s = check_config(cfg);
  if (s != DELTA_OK) return s;
  if (!workspace) return DELTA_ERR_INVALID_ARG;
  if (((uintptr_t)workspace & 255u) != 0) return DELTA_ERR_WORKSPACE;
  Workspace w;
  carve(*cfg, (char*)workspace, &w);
  if (workspace_bytes < w.total_bytes) return DELTA_ERR_WORKSPACE;
  delta_state* st = new (std::nothrow) delta_state();
  if (!st) return DELTA_ERR_INVALID_ARG;
  st->cfg = *cfg;
  st->shape = Shape{cfg->B, cfg->H, cfg->H_kv, cfg->d, cfg->T_max,
                    (cfg->T_max + DELTA_TILE_ROWS - 1) / DELTA_TILE_ROWS};
  st->ws = w;
  st->base = workspace;
  st->bytes = workspace_bytes;
  st->forced_kernel = -1;
  s = zero_state(st, (cudaStream_t)stream, /*defer=*/false);
  if (s != DELTA_OK) { delete st; return s; }
  *out = st;
  return DELTA_OK;
}

delta_status_t delta_state_reset(delta_state_t* st, void* stream) {
  if (!st) return DELTA_ERR_INVALID_ARG;
  return zero_state(st, (cudaStream_t)stream, /*defer=*/true);
}

delta_status_t delta_state_destroy(delta_state_t* st) {
  if (!st) return DELTA_ERR_INVALID_ARG;
  for (auto& ev : st->ev)
    if (ev) cudaEventDestroy(ev);
  delete st;
  return DELTA_OK;
}

delta_status_t delta_state_enable_profiling(delta_state_t* st, int32_t enable) {
  if (!st) return DELTA_ERR_INVALID_ARG;
  if (enable) {
    for (auto& ev : st->ev)
      if (!ev) {
        cudaError_t e = cudaEventCreate(&ev);
        if (e != cudaSuccess) return cuda_fail(e);
      }
  }
  st->profiling = enable != 0;
  st->profiled = false;
  return DELTA_OK;
}

delta_status_t delta_state_prefill_kernel_ms(delta_state_t* st, float* ms) {
  if (!st || !ms) return DELTA_ERR_INVALID_ARG;
  if (!st->profiling || !st->profiled) return DELTA_ERR_STATE;
  cudaError_t e = cudaEventSynchronize(st->ev[4]);
  if (e != cudaSuccess) return cuda_fail(e);
  for (int i = 0; i < 4; ++i)
    if ((e = cudaEventElapsedTime(&ms[i], st->ev[i], st->ev[i + 1])) != cudaSuccess) return cuda_fail(e);
  return DELTA_OK;
}

int32_t delta_state_position(const delta_state_t* st) { return st ? st->n : -1; }

int32_t delta_state_sequence_position(const delta_state_t* st, int32_t b) {
  return (st && b >= 0 && b < st->cfg.B) ? st->n_b[(size_t)b] : -1;
}

// Can prefill kernel `which` (1 or 2) serve this state?
static bool tc_eligible(const delta_state* st, int which) {
  if (st->cfg.dtype != DELTA_BF16 || !tc_kernel_available(64)) return false;
  if (st->cfg.source != DELTA_SRC_QUERY && which != 2 && which != 3 && which != 4 && which != 5) return false;
  if ((which == 4 || which == 5) && (st->cfg.d != 64 || (st->shape.g() % 2) != 0)) return false;
  return which == 1 ? tc_kernel_shape(st->cfg.d) : tcq_kernel_shape(st->cfg.d);
}

int32_t delta_state_prefill_kernel(const delta_state_t* st) {
  if (!st) return -1;
  if (st->forced_kernel >= 0) return st->forced_kernel;
  return tc_eligible(st, 2) ? 2 : 0;   // the telescoped tensor-core kernel is the fastest where it applies
}

// Can the tensor-core decode kernel serve this state?
static bool decode_tc_possible(const delta_state* st) {
  return st->cfg.source != DELTA_SRC_QUERY_BOTTOM_UP && decode_mma_applies(st->shape, st->cfg.dtype);
}

int32_t delta_state_decode_kernel(const delta_state_t* st) {
  if (!st) return -1;
  if (!decode_tc_possible(st)) return 0;
  if (st->key_cache_packed) return 1;          // only that kernel reads the encoding
  return st->forced_decode_kernel >= 0 ? st->forced_decode_kernel : 1;
}

delta_status_t delta_state_set_decode_kernel(delta_state_t* st, int32_t which) {
  if (!st || which < -1 || which > 1) return DELTA_ERR_INVALID_ARG;
  if (which == 1 && !decode_tc_possible(st)) return DELTA_ERR_UNSUPPORTED;
  st->forced_decode_kernel = which;
  return DELTA_OK;
}

delta_status_t delta_state_set_key_cache(delta_state_t* st, int32_t packed) {
  if (!st || packed < 0 || packed > 1) return DELTA_ERR_INVALID_ARG;
  if (st->cfg.source != DELTA_SRC_KEY || !st->ws.kp_vals) return DELTA_ERR_UNSUPPORTED;
  if (st->n != 0) return DELTA_ERR_STATE;      // the encoding is built by the prefill
  st->key_cache_packed = packed != 0;
  return DELTA_OK;
}

delta_status_t delta_key_cache_bytes(const delta_state_t* st, uint64_t* packed_bytes, uint64_t* dense_bytes,
                                     void* stream) {
  if (!st || !packed_bytes || !dense_bytes) return DELTA_ERR_INVALID_ARG;
  const delta_config_t& c = st->cfg;
  if (c.source != DELTA_SRC_KEY || !st->ws.kp_vals || !st->key_cache_packed) return DELTA_ERR_UNSUPPORTED;
  const size_t bkv = (size_t)c.B * c.H_kv;
  std::vector<uint32_t> used(bkv);
  cudaError_t e = cudaMemcpyAsync(used.data(), st->ws.kp_used, bkv * 4, cudaMemcpyDeviceToHost, (cudaStream_t)stream);
  if (e != cudaSuccess) return cuda_fail(e);
  if ((e = cudaStreamSynchronize((cudaStream_t)stream)) != cudaSuccess) return cuda_fail(e);
  uint64_t packed = 0, dense = 0;
  for (int b = 0; b < c.B; ++b) {
    const uint64_t rows = (uint64_t)st->n_b[(size_t)b], segs = (rows + 31) / 32;
    if (rows == 0) continue;         // nothing encoded yet; the device word is an earlier prompt's, or unset
    for (int h = 0; h < c.H_kv; ++h)
      packed += 2ull * used[(size_t)b * c.H_kv + h]            // values (with the segments' padding)
                + rows * (uint64_t)(c.d / 8)                    // mask words
                + rows * 2                                      // fired counts
                + segs * (uint64_t)c.d * 2 + (segs + 1) * 4;    // segment bases and offsets
    dense += (uint64_t)c.H_kv * rows * (uint64_t)c.d * 2;
  }
  *packed_bytes = packed;
  *dense_bytes = dense;
  return DELTA_OK;
}

delta_status_t delta_state_set_prefill_kernel(delta_state_t* st, int32_t which) {
  if (!st || which < -1 || which > 5) return DELTA_ERR_INVALID_ARG;
  if (which >= 1 && !tc_eligible(st, which)) return DELTA_ERR_UNSUPPORTED;
  if (which == 0 && st->cfg.source != DELTA_SRC_QUERY) return DELTA_ERR_UNSUPPORTED;
  st->forced_kernel = which;
  return DELTA_OK;
}

static delta_status_t check_theta_window(float theta, int32_t window) {
  if (!(theta >= 0.0f) || !std::isfinite(theta)) return DELTA_ERR_INVALID_ARG;
  if (window < 0) return DELTA_ERR_INVALID_ARG;
  return DELTA_OK;
}

}  // extern "C"

// The state's workspace and shape as n consecutive (batch element, KV head) units from u on see them, as
// one batch element of n KV heads (every array is laid out unit by unit; the counters are shared).
static void view_units(const delta_state* st, int u, int n, Shape* sh, Workspace* w) {
  const delta_config_t& c = st->cfg;
  const size_t g = c.H / c.H_kv, uu = (size_t)u;
  const size_t hs = uu * (c.source == DELTA_SRC_KEY ? 1 : g);        // heads of the delta stream in front
  const size_t nt = st->shape.n_tiles, nck = st->shape.n_ckpt();
  *sh = st->shape;
  sh->B = 1;
  sh->H = n * (int)g;
  sh->H_kv = n;
  *w = st->ws;
  w->dq += hs * c.T_max * c.d;
  w->mask += hs * c.T_max * (c.d / 32);
  w->row_nnz += hs * c.T_max;
  w->tile_nnz += hs * nt;
  w->idx += hs * c.T_max * c.d;
  w->qhat_tile += hs * nt * c.d;
  w->ckpt += hs * nck * c.d;
  w->qhat[0] += hs * c.d;
  w->qhat[1] += hs * c.d;
  w->R += uu * g * c.T_max;
  w->dec_partial += uu * kMaxDecodeSplits * g * (c.d + 2);
  w->dec_ticket += uu;
  if (w->kt) w->kt += uu * c.d * (((size_t)c.T_max + 3) / 4 * 4);
  if (w->qhat_rows) w->qhat_rows += hs * c.T_max * c.d;
  if (w->kp_vals) {
    const size_t nseg = (size_t)keypack_segments(c.T_max);
    w->kp_vals += uu * keypack_capacity(c.T_max, c.d);
    w->kp_segoff += uu * (nseg + 1);
    w->kp_base += uu * nseg * c.d;
    w->kp_used += uu;
    w->kp_mask += uu * nseg * 32 * (c.d / 32);
    w->kp_nnz += uu * nseg * 32;
  }
}
// ... as one batch element sees them.
static void view_of(const delta_state* st, int b, Shape* sh, Workspace* w) {
  view_units(st, b * st->cfg.H_kv, st->cfg.H_kv, sh, w);
}

// The kernels of a prefill over a uniform batch or a group of sequences of different lengths.  parts:
// PREFILL_ALL, or in two calls where the finish kernel comes last: PREFILL_FRONT (chain, attention) and
// PREFILL_FINISH.
enum { PREFILL_FRONT = 1, PREFILL_FINISH = 2, PREFILL_ALL = 3 };
static bool finish_comes_last(const delta_state* st) {
  return st->cfg.source != DELTA_SRC_KEY && delta_state_prefill_kernel(st) != 1;
}
static delta_status_t prefill_launch(delta_state* st, const Shape& shape, const Workspace& ws, const void* q,
                                     const void* k, const void* v, void* out, const SeqBatch& batch, float theta,
                                     cudaStream_t cs, bool prof, int parts = PREFILL_ALL) {
  const delta_config_t& c = st->cfg;
  cudaError_t e;
  // a pending reset: the chain kernel clears the span, less the front of qhat[0] that the chain
  // kernels of this prefill fill themselves (one reference per head of the delta stream)
  void* zero_ptr = nullptr;
  size_t zero_bytes = 0;
  if (st->zero_pending) {
    const size_t skip = (size_t)c.B * (c.source == DELTA_SRC_KEY ? c.H_kv : c.H) * c.d * sizeof(float);
    zero_ptr = (char*)st->base + skip;
    zero_bytes = st->ws.zero_bytes - skip;
    st->zero_pending = false;
  }
#define MARK(i) do { if (prof && (e = cudaEventRecord(st->ev[i], cs)) != cudaSuccess) return cuda_fail(e); } while (0)
  const int which = delta_state_prefill_kernel(st);
  const bool use_tc = which == 1;
  const bool key = c.source == DELTA_SRC_KEY;
  const bool rev = c.source == DELTA_SRC_QUERY_BOTTOM_UP;
  const bool tcq = which >= 2 && which <= 5;
  if ((key || rev) && !tcq) return DELTA_ERR_UNSUPPORTED;   // no tensor-core kernel on this device
  // The telescoped attention kernels (all but kernel 1) read nothing the finish kernel writes (delta
  // values, mask words, counts, indices, counters, hand-off row), so they run directly behind the
  // chain kernel and the finish kernel comes last.  Both are launched with programmatic stream
  // serialisation: the attention CTAs are resident and set up by the time the chain ends, and
  // the finish kernel's launch overlaps the end of the attention kernel.  With per-kernel
  // timing on, the kernels run in their natural order with events between them.
  const bool chained = !use_tc && !prof;
  // (query deltas: the attention kernel may even begin on the first query tiles while the chain goes on)
  const int form = which == 3 ? 1 : which == 4 ? 2 : which == 5 ? 3 : 0;
  SeqBatch seqs = batch;
  if (chained && tcq && !key) seqs.beside = form;
  bool finished = false;
  if (chained && !key && parts == PREFILL_ALL) seqs.with_finish = &finished;
  if (parts == PREFILL_FINISH)
    return (e = launch_delta_finish(shape, ws, q, k, seqs, theta, c.prefill_window, c.dtype, c.init, false, key, rev, 1,
                                    cs)) == cudaSuccess ? DELTA_OK : cuda_fail(e);
  MARK(0);
  // the delta stream: the queries (strategy 1) or the keys, per KV head (strategy 3)
  if ((e = launch_delta_chain(shape, ws, key ? k : q, seqs, theta, c.dtype, c.init, key, rev, zero_ptr, zero_bytes, cs)) != cudaSuccess)
    return cuda_fail(e);
  auto attention = [&]() -> cudaError_t {
    if (use_tc) return launch_hybrid_attn_tc(shape, ws, q, k, v, out, seqs.s[0].T, seqs.s[0].W, c.prefill_window, cs);
    if (tcq)
      return launch_hybrid_attn_tcq(shape, ws, q, k, v, out, seqs, theta, c.init, c.prefill_window, key,
                                    rev, form, cs);
    return launch_hybrid_attn_f32(shape, ws, q, k, v, out, seqs, theta, c.init, c.prefill_window, c.dtype, cs);
  };
  if (chained && !key) {
    if ((e = attention()) != cudaSuccess) return cuda_fail(e);
    // (released by the attention CTAs once the chain is complete: it runs beside their last wave)
    if (parts == PREFILL_ALL && !finished && (e = launch_delta_finish(shape, ws, q, k, seqs, theta, c.prefill_window, c.dtype, c.init,
                                 use_tc, key, rev, 2, cs)) != cudaSuccess)
      return cuda_fail(e);
  } else if (chained) {
    // key deltas: the finish kernel writes the reference-key rows the attention kernel streams,
    // so it comes first (both programmatically serialised behind the kernel in front)
    if ((e = launch_delta_finish(shape, ws, q, k, seqs, theta, c.prefill_window, c.dtype, c.init,
                                 use_tc, key, rev, 1, cs)) != cudaSuccess)
      return cuda_fail(e);
    if ((e = attention()) != cudaSuccess) return cuda_fail(e);
  } else {
    MARK(1);
    if ((e = launch_delta_finish(shape, ws, q, k, seqs, theta, c.prefill_window, c.dtype, c.init,
                                 use_tc, key, rev, 0, cs)) != cudaSuccess)
      return cuda_fail(e);
    MARK(2);
    if ((e = attention()) != cudaSuccess) return cuda_fail(e);
  }
  MARK(3);
  // key deltas with the compressed cache: encode the key stream behind everything it is built from
  if (key && st->key_cache_packed) {
    if (!seqs.ragged) {
      if ((e = launch_pack_keys(shape, ws, k, seqs.s[0].T, cs)) != cudaSuccess) return cuda_fail(e);
    } else {
      for (int i = 0; i < seqs.n; ++i) {
        Shape sh;
        Workspace w1;
        view_of(st, seqs.s[i].b, &sh, &w1);
        const size_t kv = (size_t)seqs.s[i].b * c.H_kv * c.T_max * c.d * 2;
        if ((e = launch_pack_keys(sh, w1, (const char*)k + kv, seqs.s[i].T, cs)) != cudaSuccess) return cuda_fail(e);
      }
    }
  }
  MARK(4);
#undef MARK
  return DELTA_OK;
}

// Host-side bookkeeping behind a prefill of T tokens for every batch element.
static void prefilled(delta_state* st, int T, int window) {
  const double B = (double)st->cfg.B;
  st->n = T;
  st->n_b.assign((size_t)st->cfg.B, T);
  st->ragged = false;
  st->qhat_sel = 0;
  st->win_sum[0] += B * (double)(window < T ? window : T);
  st->len_sum[0] += B * (double)T;
}

// Streams and events of a host-buffer prefill.  A call takes a set of its device for its duration (it
// synchronises before it returns) and gives it back to the list of idle sets, which keeps up to
// kTransferKeep of every device; what more host threads use at once is made and destroyed by their calls.
namespace {
constexpr int kTransferChunks = 4;
constexpr int kTransferKeep = 4;
struct Transfer {
  int dev = 0;
  Transfer* next = nullptr;               // in the list of idle sets
  cudaStream_t up = nullptr, down = nullptr;
  cudaEvent_t start = nullptr, arrived[kTransferChunks] = {}, computed[kTransferChunks] = {};
  cudaError_t create() {
    cudaError_t e = cudaGetDevice(&dev);
    auto ok = [&](cudaError_t x) { if (e == cudaSuccess) e = x; };
    if (e != cudaSuccess) return e;
    ok(cudaStreamCreateWithFlags(&up, cudaStreamNonBlocking));
    ok(cudaStreamCreateWithFlags(&down, cudaStreamNonBlocking));
    ok(cudaEventCreateWithFlags(&start, cudaEventDisableTiming));
    for (int i = 0; i < kTransferChunks; ++i) {
      ok(cudaEventCreateWithFlags(&arrived[i], cudaEventDisableTiming));
      ok(cudaEventCreateWithFlags(&computed[i], cudaEventDisableTiming));
    }
    return e;
  }
  void destroy() {
    if (up) cudaStreamDestroy(up);
    if (down) cudaStreamDestroy(down);
    if (start) cudaEventDestroy(start);
    for (int i = 0; i < kTransferChunks; ++i) {
      if (arrived[i]) cudaEventDestroy(arrived[i]);
      if (computed[i]) cudaEventDestroy(computed[i]);
    }
  }
};
std::mutex g_transfer_mu;
Transfer* g_transfers = nullptr;         // idle sets (linked through the sets: giving one back allocates nothing)
struct TransferGuard {
  Transfer* t = nullptr;
  cudaError_t open() {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    {
      std::lock_guard<std::mutex> lock(g_transfer_mu);
      for (Transfer** at = &g_transfers; *at; at = &(*at)->next)
        if ((*at)->dev == dev) { t = *at; *at = t->next; break; }
    }
    if (t) return cudaSuccess;
    t = new (std::nothrow) Transfer();
    if (!t) return cudaErrorMemoryAllocation;
    if ((e = t->create()) != cudaSuccess) { t->destroy(); delete t; t = nullptr; }
    return e;
  }
  ~TransferGuard() {
    if (!t) return;
    {
      std::lock_guard<std::mutex> lock(g_transfer_mu);
      int idle = 0;                       // of this device
      for (const Transfer* x = g_transfers; x; x = x->next) idle += x->dev == t->dev;
      if (idle < kTransferKeep) { t->next = g_transfers; g_transfers = t; return; }
    }
    t->destroy();
    delete t;
  }
};
}  // namespace

extern "C" {

delta_status_t delta_attn_prefill(delta_state_t* st, const void* q, const void* k, const void* v,
                                  void* out, int32_t T, int32_t H, int32_t H_kv, int32_t d,
                                  float theta, int32_t window, void* stream) {
  NvtxRange range("delta_attn_prefill");
  if (!st || !q || !k || !v || !out) return DELTA_ERR_INVALID_ARG;
  if ((((uintptr_t)q | (uintptr_t)k | (uintptr_t)v | (uintptr_t)out) & 15u) != 0) return DELTA_ERR_INVALID_ARG;
  const delta_config_t& c = st->cfg;
  if (H != c.H || H_kv != c.H_kv || d != c.d) return DELTA_ERR_INVALID_ARG;
  delta_status_t s = check_theta_window(theta, window);
  if (s != DELTA_OK) return s;
  if (T < 1) return DELTA_ERR_INVALID_ARG;
  if (T > c.T_max) return DELTA_ERR_CAPACITY;
  if (st->n != 0) return DELTA_ERR_STATE;
  const bool prof = st->profiling;
  SeqBatch seqs;
  seqs.n = 1; seqs.T_longest = T; seqs.ragged = false;
  seqs.s[0] = Seq{T, window, 0, 0};
  s = prefill_launch(st, st->shape, st->ws, q, k, v, out, seqs, theta, (cudaStream_t)stream, prof);
  if (s != DELTA_OK) return s;
  st->profiled = prof;
  prefilled(st, T, window);
  return DELTA_OK;
}

delta_status_t delta_attn_prefill_varlen(delta_state_t* st, const void* q, const void* k, const void* v,
                                         void* out, const int32_t* seq_lens, const int32_t* windows,
                                         float theta, void* stream) {
  NvtxRange range("delta_attn_prefill_varlen");
  if (!st || !q || !k || !v || !out || !seq_lens || !windows) return DELTA_ERR_INVALID_ARG;
  if ((((uintptr_t)q | (uintptr_t)k | (uintptr_t)v | (uintptr_t)out) & 15u) != 0) return DELTA_ERR_INVALID_ARG;
  const delta_config_t& c = st->cfg;
  if (!(theta >= 0.0f) || !std::isfinite(theta)) return DELTA_ERR_INVALID_ARG;
  for (int b = 0; b < c.B; ++b) {
    if (seq_lens[b] < 1 || windows[b] < 0) return DELTA_ERR_INVALID_ARG;
    if (seq_lens[b] > c.T_max) return DELTA_ERR_CAPACITY;
  }
  if (st->n != 0) return DELTA_ERR_STATE;
  // groups of kSeqMax sequences, three launches each; the kernel with the FP32 delta path, whose launch
  // covers sequences of one length: a launch per sequence over its view
  const bool one_by_one = delta_state_prefill_kernel(st) == 1;
  const size_t es = c.dtype == DELTA_F32 ? 4 : 2;
  size_t q_off = 0;     // elements in front of sequence b in the packed query / output arrays
  int t_longest = 0;
  bool same = true;
  SeqBatch seqs;
  seqs.n = 0; seqs.T_longest = 0; seqs.ragged = true;
  for (int b = 0; b < c.B; ++b) {
    const int T = seq_lens[b];
    if (one_by_one) {
      Shape sh;
      Workspace ws;
      view_of(st, b, &sh, &ws);
      const size_t kv_off = (size_t)b * c.H_kv * c.T_max * c.d * es;
      SeqBatch one;
      one.n = 1; one.T_longest = T; one.ragged = false;
      one.s[0] = Seq{T, windows[b], 0, 0};
      const delta_status_t s = prefill_launch(st, sh, ws, (const char*)q + q_off * es, (const char*)k + kv_off,
                                              (const char*)v + kv_off, (char*)out + q_off * es, one, theta,
                                              (cudaStream_t)stream, false);
      if (s != DELTA_OK) return s;
    } else {
      seqs.s[seqs.n++] = Seq{T, windows[b], b, q_off};
      seqs.T_longest = T > seqs.T_longest ? T : seqs.T_longest;
      if (seqs.n == kSeqMax || b + 1 == c.B) {
        const delta_status_t s = prefill_launch(st, st->shape, st->ws, q, k, v, out, seqs, theta, (cudaStream_t)stream, false);
        if (s != DELTA_OK) return s;
        seqs.n = 0; seqs.T_longest = 0;
      }
    }
    q_off += (size_t)c.H * T * c.d;
    t_longest = T > t_longest ? T : t_longest;
    same = same && T == seq_lens[0];
  }
  for (int b = 0; b < c.B; ++b) {
    st->n_b[(size_t)b] = seq_lens[b];
    st->win_sum[0] += (double)(windows[b] < seq_lens[b] ? windows[b] : seq_lens[b]);
    st->len_sum[0] += (double)seq_lens[b];
  }
  st->profiled = false;
  st->n = t_longest;
  st->ragged = !same;
  st->qhat_sel = 0;
  return DELTA_OK;
}

delta_status_t delta_prefill_staging_bytes(const delta_config_t* cfg, int32_t T, size_t* bytes) {
  if (!bytes) return DELTA_ERR_INVALID_ARG;
  delta_status_t s = check_config(cfg);
  if (s != DELTA_OK) return s;
  if (T < 1 || T > cfg->T_max) return DELTA_ERR_INVALID_ARG;
  const size_t es = cfg->dtype == DELTA_F32 ? 4 : 2;
  const size_t qb = align_up((size_t)cfg->B * cfg->H * T * cfg->d * es, 256);
  const size_t kb = align_up((size_t)cfg->B * cfg->H_kv * cfg->T_max * cfg->d * es, 256);
  *bytes = 2 * qb + 2 * kb;
  return DELTA_OK;
}

delta_status_t delta_attn_prefill_host(delta_state_t* st, const void* q_host, const void* k_host,
                                       const void* v_host, void* out_host, void* staging,
                                       size_t staging_bytes, int32_t T, float theta,
                                       int32_t window, void* stream) {
  NvtxRange range("delta_attn_prefill_host");
  if (!st || !q_host || !k_host || !v_host || !out_host || !staging) return DELTA_ERR_INVALID_ARG;
  const delta_config_t& c = st->cfg;
  size_t need = 0;
  delta_status_t s = delta_prefill_staging_bytes(&c, T, &need);
  if (s != DELTA_OK) return s;
  if (staging_bytes < need || ((uintptr_t)staging & 255u)) return DELTA_ERR_WORKSPACE;
  if (st->n != 0) return DELTA_ERR_STATE;
  s = check_theta_window(theta, window);
  if (s != DELTA_OK) return s;
  const size_t es = c.dtype == DELTA_F32 ? 4 : 2;
  const size_t q_bytes = (size_t)c.B * c.H * T * c.d * es;
  const size_t qb = align_up(q_bytes, 256);
  const size_t kb = align_up((size_t)c.B * c.H_kv * c.T_max * c.d * es, 256);
  char* dq_ = (char*)staging;
  char* dout = dq_ + qb;
  char* dk = dout + qb;
  char* dv = dk + kb;
  cudaStream_t cs = (cudaStream_t)stream;
  // A call that synchronises cannot be captured; refused before a stream of the pool joins the capture (it
  // would go back to the pool in it, and the next call that takes it would fail until the capture ends).
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  cudaError_t e = cudaStreamIsCapturing(cs, &capture);
  if (e == cudaSuccess && capture != cudaStreamCaptureStatusNone) e = cudaErrorStreamCaptureUnsupported;
  if (e != cudaSuccess) return cuda_fail(e);
  // The call is bound by PCIe (6.3 MB up and 4.2 MB down around 35 us of kernels at the Llama layer; 51 GB/s
  // one way, 80 both ways together): keys and values come up first, then the queries in chunks of KV
  // heads, and while a chunk is computed on the caller's stream the next one comes up on a stream of
  // the pool and the last one's output goes down on another.  Two chunks from 1.25 MB of queries on, four
  // above 4.5 MB: the kernels of a chunk are one latency (the chain, then the heaviest query tile), so more chunks
  // than the copies need lengthen the call, and a small copy beside one in the other direction waits for it
  // (queries, keys and values in chunks: 275 us).  us with 1, 2, 3, 4 chunks, 32 heads over 8 KV heads: 1.0 MB
  // 91, 91, 94, 101; 1.4 110, 106, 109, 117; 2.5 183, 152, 158, 162; 4.0 (Llama layer, 1024 tokens) 252, 220,
  // 225, 233; 4.7 331, 272, 263, 244; 6.6 404, 349, 353, 323; 16 861, 719, 704, 720; 20 heads, d = 128, 2.5 MB 195,
  // 162, 164, 170; 7.3 428, 388, 387, 371.
  const int units = c.B * c.H_kv;
  const size_t es2 = (size_t)c.d * es, g = c.H / c.H_kv;
  int chunks = q_bytes > (9u << 19) ? kTransferChunks : q_bytes >= (5u << 18) ? 2 : 1;
  if (chunks > units) chunks = units;
  if (st->profiling) chunks = 1;
  // (one chunk: all on the caller's stream, nothing to overlap)
  TransferGuard tg;
  e = chunks > 1 ? tg.open() : cudaSuccess;
  if (e != cudaSuccess) return cuda_fail(e);
  Transfer* const x = tg.t;
  const cudaStream_t s_up = x ? x->up : cs, s_down = x ? x->down : cs;
  auto settle = [&] {                     // nothing of a failed call may still touch the buffers
    cudaStreamSynchronize(s_up);
    cudaStreamSynchronize(s_down);
    cudaStreamSynchronize(cs);
  };
  auto fail = [&](cudaError_t err) { settle(); return cuda_fail(err); };
#define DO(call) do { if ((e = (call)) != cudaSuccess) return fail(e); } while (0)
  // host K/V hold T rows per head; the device copy uses the cache layout with T_max rows
  auto up_rows = [&](char* dst, const char* src, int u0, int n) -> cudaError_t {
    const size_t w = (size_t)T * es2, p = (size_t)c.T_max * es2;
    if (T == c.T_max) return cudaMemcpyAsync(dst + u0 * w, src + u0 * w, n * w, cudaMemcpyHostToDevice, s_up);
    return cudaMemcpy2DAsync(dst + u0 * p, p, src + u0 * w, w, w, n, cudaMemcpyHostToDevice, s_up);
  };
  if (x) {
    DO(cudaEventRecord(x->start, cs));
    DO(cudaStreamWaitEvent(s_up, x->start, 0));
  }
  const size_t unit_q = g * T * es2;      // bytes of a unit's queries
  DO(up_rows(dk, (const char*)k_host, 0, units));
  DO(up_rows(dv, (const char*)v_host, 0, units));
  for (int i = 0; i < chunks; ++i) {
    const int u0 = (int)((long)units * i / chunks), n = (int)((long)units * (i + 1) / chunks) - u0;
    DO(cudaMemcpyAsync(dq_ + u0 * unit_q, (const char*)q_host + u0 * unit_q, n * unit_q, cudaMemcpyHostToDevice, s_up));
    if (x) DO(cudaEventRecord(x->arrived[i], s_up));
  }
  const bool late = x && finish_comes_last(st);
  SeqBatch seqs;
  seqs.n = 1; seqs.T_longest = T; seqs.ragged = false; seqs.grid_heads = c.B * c.H;
  seqs.s[0] = Seq{T, window, 0, 0};
  for (int i = 0; i < chunks; ++i) {
    const int u0 = (int)((long)units * i / chunks), n = (int)((long)units * (i + 1) / chunks) - u0;
    const size_t kv = (size_t)u0 * c.T_max * es2, qo = u0 * unit_q;
    Shape sh = st->shape;
    Workspace ws = st->ws;
    if (chunks > 1) view_units(st, u0, n, &sh, &ws);
    if (x) DO(cudaStreamWaitEvent(cs, x->arrived[i], 0));
    s = prefill_launch(st, sh, ws, dq_ + qo, dk + kv, dv + kv, dout + qo, seqs, theta, cs, st->profiling,
                       late ? PREFILL_FRONT : PREFILL_ALL);
    if (s != DELTA_OK) { settle(); return s; }      // (prefill_launch has recorded the error's text)
    if (x) {
      DO(cudaEventRecord(x->computed[i], cs));
      DO(cudaStreamWaitEvent(s_down, x->computed[i], 0));
    }
    DO(cudaMemcpyAsync((char*)out_host + qo, dout + qo, n * unit_q, cudaMemcpyDeviceToHost, s_down));
  }
  // delta arrays, counters and the hand-off row of all chunks, while the last output goes down
  if (late) {
    s = prefill_launch(st, st->shape, st->ws, dq_, dk, dv, dout, seqs, theta, cs, false, PREFILL_FINISH);
    if (s != DELTA_OK) { settle(); return s; }      // (prefill_launch has recorded the error's text)
  }
  if (x) DO(cudaStreamSynchronize(s_down));
  DO(cudaStreamSynchronize(cs));
#undef DO
  st->profiled = st->profiling;
  prefilled(st, T, window);
  return DELTA_OK;
}

}  // extern "C"

// One decode-step launch at position n over a view (the whole batch, or one batch element), for the
// kernels that take one position per launch.
static cudaError_t decode_launch(delta_state* st, const Shape& shape, const Workspace& ws, const void* q_new,
                                 const void* k_new, const void* v_new, void* k_cache, void* v_cache, void* out,
                                 int n, float theta, int32_t window, cudaStream_t cs) {
  if (st->cfg.source == DELTA_SRC_KEY)
    return launch_decode_step_key(shape, ws, q_new, k_new, v_new, k_cache, v_cache, out, n, theta, window, st->qhat_sel,
                                  cs);
  return launch_decode_step(shape, ws, q_new, k_new, v_new, k_cache, v_cache, out, n, theta, window, st->cfg.dtype,
                            st->qhat_sel, cs);
}

extern "C" {

delta_status_t delta_attn_decode_step(delta_state_t* st, const void* q_new, const void* k_new,
                                      const void* v_new, void* k_cache, void* v_cache, void* out,
                                      float theta, int32_t window, void* stream) {
  NvtxRange range("delta_attn_decode_step");
  if (!st || !q_new || !k_new || !v_new || !k_cache || !v_cache || !out) return DELTA_ERR_INVALID_ARG;
  // every decode kernel stages cache tiles with bulk copies and reads rows as 16-byte vectors
  if ((((uintptr_t)q_new | (uintptr_t)k_new | (uintptr_t)v_new | (uintptr_t)k_cache | (uintptr_t)v_cache |
        (uintptr_t)out) & 15u) != 0)
    return DELTA_ERR_INVALID_ARG;
  delta_status_t s = check_theta_window(theta, window);
  if (s != DELTA_OK) return s;
  const delta_config_t& c = st->cfg;
  if (c.source == DELTA_SRC_QUERY_BOTTOM_UP) return DELTA_ERR_UNSUPPORTED;   // strategy (2) has no decode
  if (st->n < 1) return DELTA_ERR_STATE;
  if (st->n >= c.T_max) return DELTA_ERR_CAPACITY;      // (the longest sequence decides)
  cudaStream_t cs = (cudaStream_t)stream;
  cudaError_t e = cudaSuccess;
  const bool key_packed = c.source == DELTA_SRC_KEY && st->key_cache_packed;
  if (delta_state_decode_kernel(st) == 1) {
    // one launch, whether the batch elements stand at one position or at different ones
    e = launch_decode_step_mma(st->shape, st->ws, q_new, k_new, v_new, k_cache, v_cache, out, st->n,
                               st->ragged ? st->n_b.data() : nullptr, theta, window, st->qhat_sel,
                               c.source == DELTA_SRC_KEY, key_packed, st->stepped, st->dec_maps, cs);
    if (e != cudaSuccess) return cuda_fail(e);
  } else if (c.dtype == DELTA_F32 && st->forced_decode_kernel < 0) {
    e = launch_decode_step_f32(st->shape, st->ws, q_new, k_new, v_new, k_cache, v_cache, out, st->n,
                               st->ragged ? st->n_b.data() : nullptr, theta, window, st->qhat_sel, st->dec_maps, cs);
    if (e != cudaSuccess) return cuda_fail(e);
  } else if (!st->ragged) {
    e = decode_launch(st, st->shape, st->ws, q_new, k_new, v_new, k_cache, v_cache, out, st->n, theta, window, cs);
    if (e != cudaSuccess) return cuda_fail(e);
  } else {
    // the batch elements stand at different positions: one launch per element over its view
    const size_t es = c.dtype == DELTA_F32 ? 4 : 2;
    for (int b = 0; b < c.B; ++b) {
      Shape sh;
      Workspace ws;
      view_of(st, b, &sh, &ws);
      const size_t qo = (size_t)b * c.H * c.d * es, ko = (size_t)b * c.H_kv * c.d * es;
      const size_t co = (size_t)b * c.H_kv * c.T_max * c.d * es;
      e = decode_launch(st, sh, ws, (const char*)q_new + qo, (const char*)k_new + ko, (const char*)v_new + ko,
                        (char*)k_cache + co, (char*)v_cache + co, (char*)out + qo, st->n_b[(size_t)b], theta, window, cs);
      if (e != cudaSuccess) return cuda_fail(e);
    }
  }
  for (int b = 0; b < c.B; ++b) {
    const int L = st->n_b[(size_t)b] + 1;
    st->win_sum[1] += (double)(window < L ? window : L);
    st->len_sum[1] += (double)L;
  }
  for (auto& nb : st->n_b) nb += 1;
  st->qhat_sel ^= 1;
  st->stepped = true;
  st->n += 1;
  return DELTA_OK;
}

static void finish_stage(delta_stage_stats_t* o, const unsigned long long* c, double win, double len) {
  o->nnz = c[0]; o->elements = c[1]; o->macs_done = c[2]; o->macs_dense = c[3];
  o->S_m = o->elements ? 1.0 - (double)o->nnz / (double)o->elements : 0.0;
  o->S_c_eq6 = len > 0.0 ? o->S_m * (1.0 - win / len) : 0.0;
  o->S_c_exact = o->macs_dense ? 1.0 - (double)o->macs_done / (double)o->macs_dense : 0.0;
}

delta_status_t delta_sparsity_stats(const delta_state_t* st, delta_stats_t* host_out, void* stream) {
  NvtxRange range("delta_sparsity_stats");
  if (!st || !host_out) return DELTA_ERR_INVALID_ARG;
  unsigned long long c[CNT_TOTAL] = {};
  if (!st->zero_pending) {      // (after a reset the counters are zero, whatever the device still holds)
    cudaError_t e = cudaMemcpyAsync(c, st->ws.counters, sizeof(c), cudaMemcpyDeviceToHost,
                                    (cudaStream_t)stream);
    if (e != cudaSuccess) return cuda_fail(e);
    if ((e = cudaStreamSynchronize((cudaStream_t)stream)) != cudaSuccess) return cuda_fail(e);
  }
  memset(host_out, 0, sizeof(*host_out));
  for (int sh = 0; sh < CNT_SHARDS; ++sh)          // prefill counters are sharded on the device
    for (int i = 0; i < 4; ++i) c[CNT_PREFILL_NNZ + i] += c[CNT_SHARD_BASE + 4 * sh + i];
  finish_stage(&host_out->prefill, c + CNT_PREFILL_NNZ, st->win_sum[0], st->len_sum[0]);
  finish_stage(&host_out->decode, c + CNT_DECODE_NNZ, st->win_sum[1], st->len_sum[1]);
  unsigned long long sum[4];
  for (int i = 0; i < 4; ++i) sum[i] = c[CNT_PREFILL_NNZ + i] + c[CNT_DECODE_NNZ + i];
  finish_stage(&host_out->combined, sum, 0.0, 0.0);
  // combined Eq. 6 value: the stages' Eq. 6 values weighted by their dense multiply-adds
  const double dp = (double)host_out->prefill.macs_dense, dd = (double)host_out->decode.macs_dense;
  host_out->combined.S_c_eq6 =
      (dp + dd) > 0.0 ? (host_out->prefill.S_c_eq6 * dp + host_out->decode.S_c_eq6 * dd) / (dp + dd) : 0.0;
  host_out->n = st->n;
  host_out->device_status = (uint32_t)c[CNT_STATUS];
  return host_out->device_status == 0 ? DELTA_OK : (delta_status_t)host_out->device_status;
}

int32_t delta_window_from_gamma(int32_t n, double gamma, int32_t w_max) {
  if (n < 0 || !(gamma >= 0.0)) return 0;
  const double w = std::floor(gamma * (double)n);
  const double m = w < (double)w_max ? w : (double)w_max;
  return m < 0.0 ? 0 : (int32_t)m;
}

delta_status_t delta_state_view(const delta_state_t* st, int32_t what, const void** dev_ptr,
                                size_t* bytes) {
  if (!st || !dev_ptr || !bytes) return DELTA_ERR_INVALID_ARG;
  const delta_config_t& c = st->cfg;
  const size_t BH = (size_t)c.B * c.H;
  const size_t nt = st->shape.n_tiles;
  switch (what) {
    case DELTA_VIEW_DQ: *dev_ptr = st->ws.dq; *bytes = BH * c.T_max * c.d * 4; break;
    case DELTA_VIEW_MASK: *dev_ptr = st->ws.mask; *bytes = BH * c.T_max * (c.d / 32) * 4; break;
    case DELTA_VIEW_ROW_NNZ: *dev_ptr = st->ws.row_nnz; *bytes = BH * c.T_max * 2; break;
    case DELTA_VIEW_TILE_NNZ: *dev_ptr = st->ws.tile_nnz; *bytes = BH * nt * 4; break;
    case DELTA_VIEW_IDX: *dev_ptr = st->ws.idx; *bytes = BH * c.T_max * c.d; break;
    case DELTA_VIEW_QHAT_TILE: *dev_ptr = st->ws.qhat_tile; *bytes = BH * nt * c.d * 4; break;
    case DELTA_VIEW_QHAT: *dev_ptr = st->ws.qhat[st->qhat_sel]; *bytes = BH * c.d * 4; break;
    case DELTA_VIEW_R: *dev_ptr = st->ws.R; *bytes = BH * c.T_max * 4; break;
    case DELTA_VIEW_COUNTERS: *dev_ptr = st->ws.counters; *bytes = (size_t)CNT_TOTAL * 8; break;
    default: return DELTA_ERR_INVALID_ARG;
  }
  return DELTA_OK;
}

int32_t delta_debug_bounds_build(void) {
#ifdef DELTA_DEBUG_BOUNDS
  return 1;
#else
  return 0;
#endif
}

uint64_t delta_launch_count(void) { return g_launches.load(std::memory_order_relaxed); }

const char* delta_status_string(delta_status_t s) {
  switch (s) {
    case DELTA_OK: return "ok";
    case DELTA_ERR_INVALID_ARG: return "invalid argument";
    case DELTA_ERR_UNSUPPORTED: return "unsupported configuration";
    case DELTA_ERR_WORKSPACE: return "workspace too small or misaligned";
    case DELTA_ERR_CAPACITY: return "sequence capacity T_max exceeded";
    case DELTA_ERR_STATE: return "call order: state not in the required condition";
    case DELTA_ERR_CUDA: return "CUDA runtime error";
    case DELTA_ERR_TIMEOUT: return "bounded device-side wait ran out";
    case DELTA_ERR_BOUNDS: return "index out of range in a kernel (bounds-checking build)";
    case DELTA_ERR_SCRATCH_LIMIT:
      return "problem larger than the built-in scratch of delta_attn_decode_step_noalloc";
  }
  return "unknown status";
}

const char* delta_last_cuda_error(void) { return g_cuda_err; }

}  // extern "C"
