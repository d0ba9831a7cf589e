// K1 -- delta construction (Section II-C, Eq. 2-3; Section III-A strategies (1), (2), (3)), in
// two kernels.
//
// delta_chain_kernel: the token-sequential part.  Eq. 3 makes every channel a chain along the
// tokens (the reference is the last value that fired), so the only parallelism is across
// channels: one thread per channel, one CTA per (batch, head, 32 channels) of the stream (query
// heads, or KV heads for key deltas).  The chain itself is three dependent FP32 operations per
// token and a lone warp issues slowly, so everything else is kept off it: a producer warp
// streams the rows into a ring of shared-memory stages with TMA (the rows do not depend on the
// carried state), helper warps precompute everything about an eight-row sub-block that does not
// involve the carried state (see the kernel), and the chain warp stores nothing but the
// reference in front of every 8-row block (and every 64-row tile, and the final one).  Given
// those checkpoints every 8-row block of Eq. 2-3 is independent of the others: fire bits,
// delta values, mask words and reference rows are recomputed from them by row-parallel code
// (the finish kernel below, the attention kernel for its own query tile).
//
// delta_finish_kernel: everything that is parallel over rows -- Eq. 2-3 over 8-row blocks
// from the checkpoints: delta values, mask words and (key deltas) the reference-key rows;
// per-row and per-tile non-zero counts, the compacted channel indices, the counters behind
// Eq. 6 -- plus, for query deltas, two passes over the keys that prefill needs anyway: the
// hand-off row R(T-1)[j] = q_hat(T-1).k_j for decode and, for the tensor-core attention kernel
// with the FP32 delta path, the channel-major fp32 copy of the keys.
#include <algorithm>

#include "delta_internal.cuh"
#include "k1_finish.cuh"
#include "k2_tc.cuh"
#include "tc_common.cuh"

namespace delta {

namespace {

constexpr int RC = 64;       // rows per ring stage (= one 64-row tile)
constexpr int NS = 8;        // stages of staged rows
constexpr int NZ = 4;        // stages of sub-block tables
constexpr int CH = 32;       // channels per CTA: one chain warp, thread = channel
constexpr int SBR = DELTA_CKPT_ROWS;     // rows per sub-block: one checkpoint each
constexpr int NSB = RC / SBR;
constexpr int NHELP = 12;    // warps that build the sub-block tables
constexpr int ZV = 4;        // float4 per (sub-block, channel): x0..x7, z0..z6
constexpr int Z_STAGE = NSB * ZV * CH;   // float4 per table stage
constexpr int CHAIN_THREADS = 32 * (NHELP / 3 * 4);
static_assert(SBR == 8 && NHELP % 3 == 0 && NHELP >= 6, "the kernel's tables and its warp roles");

template <typename TIn> __device__ __forceinline__ float lds_elem(const TIn* p);
template <> __device__ __forceinline__ float lds_elem<float>(const float* p) { return *p; }
template <> __device__ __forceinline__ float lds_elem<__nv_bfloat16>(const __nv_bfloat16* p) {
  return __uint_as_float((uint32_t)(*reinterpret_cast<const uint16_t*>(p)) << 16);
}

// Does the reference x_ref fire on value x (Eq. 3: one IEEE subtraction, strict compare, NaN false)?
__device__ __forceinline__ bool fires(float x, float x_ref, float theta) {
  return fabsf(__fsub_rn(x, x_ref)) > theta;
}

// The helpers' waits: suspended (they run ahead of the chain warp, and where several CTAs share
// an SM a spinning helper would take issue slots from another CTA's chain warp).
__device__ __forceinline__ bool wait_ok(uint32_t bar, uint32_t parity, volatile uint32_t* abort_flag) {
  if (mbar_test_wait(bar, parity)) return true;
  mbar_wait(bar, parity, abort_flag);
  return *abort_flag == 0;
}

// One arrival for the warp, predicated: a branch that one lane takes costs the chain warp its reconvergence.
__device__ __forceinline__ void arrive_lane0(uint32_t bar, int lane) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.eq.s32 p, %1, 0;\n\t@p mbarrier.arrive.shared::cta.b64 _, [%0];\n\t}"
               ::"r"(bar), "r"(lane) : "memory");
}

// A sub-block's table for one channel: its rows and the end states z (z7 = x7), as the chain warp loads them.
struct SubBlock {
  float4 x[2], z[2];      // x0..x7, z0..z6
};
__device__ __forceinline__ SubBlock load_sub_block(const float4* p) {
  SubBlock t;
  t.x[0] = p[0];
  t.x[1] = p[CH];
  t.z[0] = p[2 * CH];
  t.z[1] = p[3 * CH];
  return t;
}

// The state behind a sub-block that is entered with state r: of the rows that fire against r (one IEEE subtraction,
// strict compare, NaN false: see fires) the first one's end state, r where none does.  basis: row 0 is taken
// un-thresholded.
__device__ __forceinline__ float chain_sub_block(const SubBlock& t, float r, float theta, bool basis) {
  const bool p0 = fires(t.x[0].x, r, theta) || basis, p1 = fires(t.x[0].y, r, theta), p2 = fires(t.x[0].z, r, theta);
  const bool p3 = fires(t.x[0].w, r, theta), p4 = fires(t.x[1].x, r, theta), p5 = fires(t.x[1].y, r, theta);
  const bool p6 = fires(t.x[1].z, r, theta), p7 = fires(t.x[1].w, r, theta);
  float o = p7 ? t.x[1].w : r;
  o = p6 ? t.z[1].z : o;
  o = p5 ? t.z[1].y : o;
  o = p4 ? t.z[1].x : o;
  o = p3 ? t.z[0].w : o;
  o = p2 ? t.z[0].z : o;
  o = p1 ? t.z[0].y : o;
  return p0 ? t.z[0].x : o;
}

// The streams of a launch, each as a map [heads][rows 0..T-1][D] with boxes of [64 rows][32 channels]: one over all
// heads of a batch, or one per sequence of a ragged group; b: batch element of the workspace arrays that head 0 belongs to.
template <int N> struct ChainSeqs {
  CUtensorMap map[N];
  int T[N], b[N];
};

}  // namespace

// The chain of Eq. 3 costs three dependent operations per row (subtract, compare, select), about
// 17 clocks.  Most of that can be taken off the carried state.  Over a sub-block of eight rows
// x0..x7 (in processing order) the state r either survives, or the first row i that fires
// against r replaces it -- and from there on the chain no longer depends on r: the state at the
// end of the sub-block is z_i, the end state of the chain that starts with reference x_i at
// row i.  z_7 = x7, z_6 = fires(x7, x6) ? x7 : x6, and in general z_i = z_j for the first j > i
// that fires against x_i (x_i if none does): 28 pair tests per sub-block, none of which
// involves r.  Helper warps compute the z tables a stage ahead; the chain warp then does, per
// sub-block, eight tests against r in parallel and a chain of eight selects (a tree of them made no
// difference), and the checkpoint in front of the sub-block is the only store.  Every test is the same subtraction and comparison the sequential chain would make, so the
// result is bit-identical.
//
// One CTA per (head, 32 channels): a warp carries the chain (thread = channel), one streams the rows in with TMA,
// twelve build the tables, on the three schedulers beside the chain warp's.  A lone warp builds a table in 220
// clocks, two on a scheduler one in 163 (28 tests, half of their instructions on the half-rate pipe); the sub-blocks
// are dealt to the warps one by one, whatever their stage (a warp that waits and arrives for every stage costs
// 1000 clocks per stage: the chain then waits for the tables), four stages of tables ahead at most.  The chain warp
// takes 57 clocks per sub-block of a table already there and 86 in the kernel, stage edges, checkpoint stores and the
// helpers' shared-memory traffic included (10.8 per row; four rows per table with three helpers: 14; row by row 16.8).
// A sub-block cut short by the end of the sequence takes the sequential form from the staged values.
// Measured (with the launch, by events), before -> after: 1 x 32 heads, 1024 tokens, d = 64 14.7 -> 13.9 us; 4096 keys
// 36.4 -> 30.2; 20 heads, 2048 tokens, d = 128 22.0 -> 19.9; a cut last stage (1000 tokens) 16.1 -> 14.1.
template <typename TIn, int D, int N>
__global__ void __launch_bounds__(CHAIN_THREADS) delta_chain_kernel(
    const __grid_constant__ ChainSeqs<N> seqs, float* __restrict__ qhat_tile, float* __restrict__ qhat_out,
    float* __restrict__ ckpt, unsigned long long* __restrict__ counters, int n_tiles, int n_ckpt,
    float theta, int basis_exact, int reverse, int heads, unsigned* __restrict__ progress, uint4* zero_ptr, unsigned zero_n16) {
  // blockIdx.x: (head, 32 channels) of the batch, or of sequence blockIdx.y of a ragged group
  const int si = N == 1 ? 0 : (int)blockIdx.y;
  const CUtensorMap& tm_x = seqs.map[si];
  const int T = seqs.T[si];
  constexpr int NSL = D / CH;                      // channel slices (CTAs) per head
  constexpr uint32_t RAW_STAGE_BYTES = RC * CH * sizeof(TIn);
  extern __shared__ __align__(128) unsigned char dyn[];
  TIn* raw = reinterpret_cast<TIn*>(dyn);                                   // [NS][RC][CH]
  float4* zb = reinterpret_cast<float4*>(dyn + NS * RAW_STAGE_BYTES);       // [NZ][NSB][ZV][CH]
  __shared__ __align__(8) unsigned long long bars[2 * NS + 2 * NZ];
  __shared__ uint32_t s_abort, s_done;             // s_done: stages the chain warp is through with

  const int head = blockIdx.x / NSL, sl = blockIdx.x - head * NSL;       // head of the map
  const int bh = seqs.b[si] * heads + head;                               // head of the workspace arrays
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t full0 = smem_u32(&bars[0]), empty0 = smem_u32(&bars[NS]);
  const uint32_t zfull0 = smem_u32(&bars[2 * NS]), zfree0 = smem_u32(&bars[2 * NS + NZ]);
  volatile uint32_t* abort_flag = &s_abort;
  const int n_chunks = (T + RC - 1) / RC;
  // Which of the four schedulers' first warps carries the chain rotates with the CTA: where several CTAs
  // share an SM their chain warps, the busiest, then sit on different schedulers.  The producer is the
  // other warp of the chain's scheduler.
  const int cw = (int)blockIdx.x & 3;
  if (tid < 2 * NS + 2 * NZ) {      // one barrier per thread
    const uint32_t cnt = (tid < NS) ? 1u : (tid < 2 * NS + NZ) ? (uint32_t)NSB : 1u;
    tc::mbar_init(full0 + 8 * tid, cnt);
    if (tid == 0) s_abort = s_done = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    tc::fence_proxy_async();
  }
  if (tid == 32 * (4 + cw))
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tm_x) : "memory");
  __syncthreads();
  // Launched with programmatic stream serialisation: set up while the kernel in front runs out, then wait for it (it
  // may have written the stream, and may still use the workspace).  Behind the wait, never ahead of it: a
  // kernel launched behind this one in the same way may become resident now, and takes this call's
  // inputs (queries, keys, values) for complete from its start; this kernel's results it sees after its own wait.
  // (Whole prefills behind one another, ordinary launch -> this: 1 x 32 heads 256 tokens 12.9 -> 11.5 us, 1024 28.2 ->
  // 26.0; d = 128, 20 heads, 2048 63.6 -> 61.5; 4 x 32 x 1024 74.9 -> 73.1; 8 x 32 x 1024 139.4 -> 137.3.)
  asm volatile("griddepcontrol.wait;" ::: "memory");
  unsigned* const my_progress = progress ? progress + ((size_t)bh * NSL + sl) * kProgressStride : nullptr;
  if (!progress) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  } else if (tid == 32 * (8 + cw)) {
    // (cleared before anything behind this kernel can look at it)
    *my_progress = 0;
    __threadfence();
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  }
  // the deferred clearing of a state reset (counters, tickets, second reference buffer): nothing
  // of this launch or of the kernels behind it touches that span before this kernel is complete
  if (zero_ptr && blockIdx.x == 0 && blockIdx.y == 0)
    for (unsigned i = tid; i < zero_n16; i += blockDim.x) zero_ptr[i] = make_uint4(0u, 0u, 0u, 0u);

  if (warp == 4 + cw) {
    // ---- producer: keeps up to NS stages of rows in flight
    if (lane == 0) {
      const uint32_t raw0 = smem_u32(raw);
      for (int i = 0; i < n_chunks && !*abort_flag; ++i) {
        const int s = i % NS;
        if (i >= NS) mbar_wait(empty0 + 8 * s, ((i / NS) - 1) & 1, abort_flag);
        const int ci = reverse ? n_chunks - 1 - i : i;      // stage of the head in token order
        tc::mbar_expect_tx(full0 + 8 * s, RAW_STAGE_BYTES); // rows past T arrive as zeros
        tc::tma_load_3d(raw0 + s * RAW_STAGE_BYTES, &tm_x, full0 + 8 * s, sl * CH, ci * RC, head);
      }
    }
  } else if (warp == 8 + cw) {
    // ---- progress: how many stages' references are in memory, for a kernel behind that starts on the first ones while
    // the chain goes on.  (Not by the chain warp, which a fence would hold up for a trip to memory per stage.)
    if (progress && lane == 0) {
      for (int seen = 0; seen + 1 < n_chunks && !*abort_flag;) {
        // (s_done says which stage's barrier to look at, the barrier orders what the chain warp stored; where the chain
        // has gone round the ring since, the look fails and the next one is at a later stage)
        const int now = (int)*(volatile uint32_t*)&s_done;
        if (now > seen && mbar_test_wait(zfree0 + 8 * ((now - 1) % NZ), ((now - 1) / NZ) & 1)) {
          seen = now;
          __threadfence();
          *(volatile unsigned*)my_progress = (unsigned)seen;
        } else {
          __nanosleep(64);
        }
      }
    }
  } else if ((warp & 3) != cw) {
    // ---- helpers: the sub-blocks of all stages, in processing order (reverse: from the stage's last row
    // down), are dealt round-robin
    const int hw = ((warp - cw - 1) & 3) + 3 * (warp >> 2);
    const ptrdiff_t rstep = reverse ? -CH : CH;
    for (int gb = hw; gb < n_chunks * NSB; gb += NHELP) {
      const int i = gb / NSB, sb = gb % NSB, s = i % NS, zs = i % NZ;
      if (!wait_ok(full0 + 8 * s, (i / NS) & 1, abort_flag)) break;
      const TIn* rows = raw + (size_t)s * RC * CH + lane + (reverse ? (RC - 1) * CH : 0) + sb * SBR * rstep;
      float y[SBR], z[SBR];
#pragma unroll
      for (int k = 0; k < SBR; ++k) z[k] = y[k] = lds_elem<TIn>(rows + k * rstep);
#pragma unroll
      for (int j = SBR - 1; j > 0; --j)
#pragma unroll
        for (int a = j - 1; a >= 0; --a) z[a] = fires(y[j], y[a], theta) ? z[j] : z[a];
      if (i >= NZ && !wait_ok(zfree0 + 8 * zs, ((i / NZ) - 1) & 1, abort_flag)) break;
      float4* o = zb + (size_t)zs * Z_STAGE + sb * (ZV * CH) + lane;
      o[0] = make_float4(y[0], y[1], y[2], y[3]);
      o[CH] = make_float4(y[4], y[5], y[6], y[7]);
      o[2 * CH] = make_float4(z[0], z[1], z[2], z[3]);
      o[3 * CH] = make_float4(z[4], z[5], z[6], 0.0f);
      __syncwarp();
      arrive_lane0(zfull0 + 8 * zs, lane);
      arrive_lane0(empty0 + 8 * s, lane);
    }
  } else if (warp == cw) {
    // ---- chain warp: thread owns channel c
    const int c = sl * CH + lane;
    float r = 0.0f;           // reference state, starts at zero (Eq. 3)
    static_assert(RC == DELTA_TILE_ROWS, "one tile reference per stage");
    const ptrdiff_t step = reverse ? -(ptrdiff_t)D : (ptrdiff_t)D;
    const int tile0 = reverse ? n_chunks - 1 : 0;       // tile (= stage in token order) of stage 0
    // where the references in front of the stage and of its sub-blocks go, in processing order
    float* qp = qhat_tile + ((size_t)bh * n_tiles + tile0) * D + c;
    float* const ckpt_c = ckpt + (size_t)bh * n_ckpt * D + c;
    float* cp = ckpt_c + (ptrdiff_t)(tile0 * NSB + (reverse ? NSB - 1 : 0)) * D;
    const int rest = T % RC;                            // rows of a stage cut short by the end of the sequence
    auto wait_stage = [&](int i) { mbar_poll(zfull0 + 8 * (i % NZ), (i / NZ) & 1, abort_flag); __syncwarp(); };
    auto stage_done = [&](int i) {
      __syncwarp();
      arrive_lane0(zfree0 + 8 * (i % NZ), lane);
      if (lane == 0) *(volatile uint32_t*)&s_done = (uint32_t)(i + 1);
    };
    auto tile_ref = [&](int i) {
      if (qhat_tile && DELTA_IN(reverse ? tile0 - i : i, n_tiles, counters)) *qp = r;
      qp += step;
    };
    // the cut stage (the last one; reverse: the first): sub-blocks behind the end carry no state, the one the
    // end falls into goes row by row
    auto cut_stage = [&](int i) {
      wait_stage(i);
      tile_ref(i);
      const float4* const zp = zb + (size_t)(i % NZ) * Z_STAGE + lane;
      for (int b = 0; b < NSB; ++b, cp += step) {
        const int pr0 = (reverse ? NSB - 1 - b : b) * SBR;          // the sub-block's lowest row of the stage
        if (pr0 >= rest) continue;
        const float4* const p = zp + b * (ZV * CH);
        const bool head = basis_exact && i == 0 && (reverse ? pr0 + SBR >= rest : b == 0);
        if (DELTA_IN((size_t)(cp - ckpt_c) / D, n_ckpt, counters)) *cp = r;
        if (pr0 + SBR <= rest) {
          r = chain_sub_block(load_sub_block(p), r, theta, head);
        } else {
          const int n = rest - pr0;                                 // rows of the sub-block, the lowest ones
          const float* const x = reinterpret_cast<const float*>(p);
          for (int k = reverse ? SBR - n : 0; k < (reverse ? SBR : n); ++k) {
            const float xk = x[(k >> 2) * (4 * CH) + (k & 3)];
            r = ((head && k == (reverse ? SBR - n : 0)) || fires(xk, r, theta)) ? xk : r;
          }
        }
      }
      stage_done(i);
    };
    const int i0 = (reverse && rest) ? 1 : 0, i1 = i0 + T / RC;      // the whole stages
    if (i0) cut_stage(0);
    if (i0 < i1) {
      wait_stage(i0);
      SubBlock cur = load_sub_block(zb + (size_t)(i0 % NZ) * Z_STAGE + lane);
      // One pass of the loop per stage, its eight sub-blocks unrolled (two or four to a pass are slower: 40.6 and 36.5 us
      // for 4096 rows, unrolled 32.7, with the stage's edge as below 30.2); a sub-block's tables are loaded while the one in front is worked on, over the stage's end too,
      // where the next stage's barrier is looked at two sub-blocks ahead.
#pragma unroll 1
      for (int i = i0; i < i1; ++i) {
        const float4* const zp = zb + (size_t)(i % NZ) * Z_STAGE + lane;
        const int in = i + 1;
        tile_ref(i);
        bool ready = true;
#pragma unroll
        for (int b = 0; b < NSB; ++b) {
          SubBlock nxt;
          if (b + 1 < NSB) {
            nxt = load_sub_block(zp + (b + 1) * (ZV * CH));
          } else {
            if (!__all_sync(0xffffffffu, ready)) wait_stage(in);
            nxt = load_sub_block(zb + (size_t)(in % NZ) * Z_STAGE + lane);      // (behind the last stage: not used)
          }
          if (b == NSB - 3) ready = in >= i1 || mbar_test_wait(zfull0 + 8 * (in % NZ), (in / NZ) & 1);
          if (DELTA_IN((size_t)(cp - ckpt_c) / D, n_ckpt, counters)) *cp = r;
          cp += step;
          r = chain_sub_block(cur, r, theta, b == 0 && i == 0 && basis_exact);
          cur = nxt;
        }
        stage_done(i);
      }
    }
    if (!reverse && rest) cut_stage(i1);
    if (!*abort_flag && qhat_out) qhat_out[(size_t)bh * D + c] = r;
  }
  __syncthreads();
  if (tid == 0 && s_abort) atomicMax(&counters[CNT_STATUS], (unsigned long long)DELTA_ERR_TIMEOUT);
}

// A launch on stream st with programmatic stream serialisation (grid, block and shared memory to be filled in).
static cudaLaunchConfig_t serialised_launch(cudaLaunchAttribute (&attr)[1], cudaStream_t st) {
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cfg;
}

// Shared memory to ask for so that an SM takes no more of the launch's CTAs than an even spread gives it.  A kernel in front
// that lets this one in while it still holds most SMs (a decode step) leaves it a few SMs only: without this the CTAs
// pile up there (one layer of 8 x 32 heads, 4096 tokens, behind decode steps: +34 us), with it they wait for their place.
static size_t even_spread_smem(size_t need, long ctas) {
  const long sms = device_sm_count(), per = (ctas + sms - 1) / sms;
  const size_t even = (size_t)228 * 1024 / (size_t)(per + 1);      // one CTA more would not fit
  return need > even ? need : even;
}
constexpr int kMaxChainSmem = 144 * 1024;      // (fp32 tables 128 KB; the even spread asks for 114 KB at most)

template <typename TIn, int D, int N>
static cudaError_t launch_tables(const Shape& s, const Workspace& w, const void* x, const SeqBatch& seqs, float theta, int init,
                                 bool key_stream, bool reverse, unsigned* progress, void* zero_ptr, size_t zero_bytes,
                                 cudaStream_t st) {
  auto kern = delta_chain_kernel<TIn, D, N>;
  constexpr size_t need = (size_t)NS * RC * CH * sizeof(TIn) + (size_t)NZ * Z_STAGE * sizeof(float4);
  static_assert(need <= kMaxChainSmem, "shared memory");
  static std::atomic<uint64_t> ready{0};
  if (!device_done(ready)) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxChainSmem);
    if (e != cudaSuccess) return e;
    device_mark(ready);
  }
  const int heads = key_stream ? s.H_kv : s.H, map_heads = seqs.ragged ? heads : s.B * heads;
  ChainSeqs<N> list;
  int order[N];
  for (int i = 0; i < seqs.n; ++i) order[i] = i;
  std::sort(order, order + seqs.n, [&](int a, int b) { return seqs.s[a].T > seqs.s[b].T; });       // longest first
  for (int i = 0; i < seqs.n; ++i) {
    const Seq& sq = seqs.s[order[i]];
    const size_t rows = key_stream ? (size_t)s.T_max : (size_t)sq.T;       // of a head in memory
    const TIn* const from = (const TIn*)x + (key_stream ? (size_t)(seqs.ragged ? sq.b : 0) * heads * rows * D : sq.q_off);
    if (!tc::encode3(&list.map[i], sizeof(TIn) == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, from,
                     (uint64_t)D, (uint64_t)sq.T, (uint64_t)map_heads, (uint64_t)D * sizeof(TIn), rows * D * sizeof(TIn), CH, RC,
                     CU_TENSOR_MAP_SWIZZLE_NONE))
      return cudaErrorInvalidValue;
    list.T[i] = sq.T;
    list.b[i] = seqs.ragged ? sq.b : 0;
  }
  cudaLaunchAttribute attr[1];
  cudaLaunchConfig_t cfg = serialised_launch(attr, st);
  cfg.gridDim = dim3((unsigned)(map_heads * (D / CH)), (unsigned)seqs.n);
  cfg.blockDim = dim3(CHAIN_THREADS);
  cfg.dynamicSmemBytes = even_spread_smem(need, (long)cfg.gridDim.x * seqs.n);
  const cudaError_t err =
      cudaLaunchKernelEx(&cfg, kern, list, w.qhat_tile, w.qhat[0], w.ckpt, w.counters, s.n_tiles, s.n_ckpt(), theta,
                         init == DELTA_INIT_BASIS_EXACT ? 1 : 0, reverse ? 1 : 0, heads, progress, (uint4*)zero_ptr,
                         (unsigned)(zero_bytes / 16));
  count_launch();
  return err != cudaSuccess ? err : cudaGetLastError();
}

static cudaError_t launch_delta_chain_tables(const Shape& s, const Workspace& w, const void* x, const SeqBatch& seqs,
                                             float theta, int dtype, int init, bool key_stream, bool reverse,
                                             unsigned* progress, void* zero_ptr, size_t zero_bytes, cudaStream_t st) {
#define GO(TIN, DD)                                                                                                 \
  return seqs.ragged                                                                                                \
             ? launch_tables<TIN, DD, kSeqMax>(s, w, x, seqs, theta, init, key_stream, reverse, progress, zero_ptr, zero_bytes, st) \
             : launch_tables<TIN, DD, 1>(s, w, x, seqs, theta, init, key_stream, reverse, progress, zero_ptr, zero_bytes, st)
  if (dtype == DELTA_F32) {
    if (s.d == 64) { GO(float, 64); } else { GO(float, 128); }
  } else {
    if (s.d == 64) { GO(__nv_bfloat16, 64); } else { GO(__nv_bfloat16, 128); }
  }
#undef GO
}

// ---------------------------------------------------------------------------------------
// delta_chain_rows_kernel: the chain row by row, for streams of many heads.  One CTA per (batch,
// head): D/32 chain warps (thread = channel) + one producer warp that streams the head's rows
// into a ring of shared-memory stages with bulk copies.  Per row one shared-memory load, one
// widening, the three dependent operations of Eq. 2-3 and a checkpoint store every 8 rows.  It
// does 3 times fewer instructions and 10 times less shared-memory traffic per row than the
// kernel above: with every head of a large batch resident at once this one is faster (6 x 32 heads of 1024 tokens
// 19.5 us against 23.2, 8 x 32 19.6 against 28.3), with few heads the other one (see the rule at the launch).
namespace {

constexpr int RROWS = 64;    // rows per ring stage
constexpr int RSTAGES = 4;   // ring stages

// One element of the staged rows by shared-memory address, widened to fp32.
template <typename TIn> __device__ __forceinline__ float lds_row_elem(uint32_t addr);
template <> __device__ __forceinline__ float lds_row_elem<float>(uint32_t addr) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr));
  return v;
}
template <> __device__ __forceinline__ float lds_row_elem<__nv_bfloat16>(uint32_t addr) {
  uint32_t u;
  asm volatile("ld.shared.u16 %0, [%1];" : "=r"(u) : "r"(addr));
  return __uint_as_float(u << 16);
}

// One ring stage of the chain for one thread (= one channel): rows t0 .. t0+nrows-1, the
// thread's values at rows[r * D]; updates the reference qh and leaves it in front of every
// 8-row block (ckptp).  basis_row: the stage's first row is the un-thresholded basis.
template <typename TIn, int D>
__device__ __forceinline__ void chain_stage(const TIn* rows, int t0, int nrows, bool basis_row, float& qh,
                                            float theta, float* ckptp, int n_ckpt, unsigned long long* counters) {
  if (nrows == RROWS && !basis_row) {
    // full stage, no basis row: nothing but loads, the dependent chain and the checkpoints
    float x[RROWS];
    const uint32_t saddr = smem_u32(rows);
#pragma unroll
    for (int r = 0; r < RROWS; ++r) x[r] = lds_row_elem<TIn>(saddr + (uint32_t)(r * D * sizeof(TIn)));
#pragma unroll
    for (int r = 0; r < RROWS; ++r) {
      if ((r % DELTA_CKPT_ROWS) == 0 && DELTA_IN((t0 + r) / DELTA_CKPT_ROWS, n_ckpt, counters))
        ckptp[(size_t)((t0 + r) / DELTA_CKPT_ROWS) * D] = qh;
      const float diff = __fsub_rn(x[r], qh);      // one IEEE subtraction
      const bool fire = fabsf(diff) > theta;       // strict; NaN compares false
      qh = fire ? x[r] : qh;
    }
  } else {
    for (int r = 0; r < nrows; ++r) {
      if (((t0 + r) % DELTA_CKPT_ROWS) == 0 && DELTA_IN((t0 + r) / DELTA_CKPT_ROWS, n_ckpt, counters))
        ckptp[(size_t)((t0 + r) / DELTA_CKPT_ROWS) * D] = qh;
      const float x = to_f32(rows[r * D]);
      const bool fire = (r == 0 && basis_row) || (fabsf(__fsub_rn(x, qh)) > theta);
      qh = fire ? x : qh;
    }
  }
}

// Strategy (2): the same stage of the query stream taken from its last row down to its first.
// The checkpoint of an 8-row block is the reference before the block's highest row.
// basis_last: the stage's last row is row T-1, the un-thresholded basis of this order.
template <typename TIn, int D>
__device__ __forceinline__ void chain_stage_rev(const TIn* rows, int t0, int nrows, bool basis_last, float& qh,
                                                float theta, float* ckptp, int n_ckpt, unsigned long long* counters) {
  if (nrows == RROWS && !basis_last) {
    float x[RROWS];
    const uint32_t saddr = smem_u32(rows);
#pragma unroll
    for (int r = 0; r < RROWS; ++r) x[r] = lds_row_elem<TIn>(saddr + (uint32_t)(r * D * sizeof(TIn)));
#pragma unroll
    for (int r = RROWS - 1; r >= 0; --r) {
      if ((r % DELTA_CKPT_ROWS) == DELTA_CKPT_ROWS - 1 && DELTA_IN((t0 + r) / DELTA_CKPT_ROWS, n_ckpt, counters))
        ckptp[(size_t)((t0 + r) / DELTA_CKPT_ROWS) * D] = qh;
      const float diff = __fsub_rn(x[r], qh);
      const bool fire = fabsf(diff) > theta;
      qh = fire ? x[r] : qh;
    }
  } else {
    for (int r = nrows - 1; r >= 0; --r) {
      if ((((t0 + r) % DELTA_CKPT_ROWS) == DELTA_CKPT_ROWS - 1 || r == nrows - 1) &&
          DELTA_IN((t0 + r) / DELTA_CKPT_ROWS, n_ckpt, counters))
        ckptp[(size_t)((t0 + r) / DELTA_CKPT_ROWS) * D] = qh;
      const float x = to_f32(rows[r * D]);
      const bool fire = (r == nrows - 1 && basis_last) || (fabsf(__fsub_rn(x, qh)) > theta);
      qh = fire ? x : qh;
    }
  }
}

}  // namespace

template <typename TIn, int D, int N>
__global__ void __launch_bounds__(D + 32) delta_chain_rows_kernel(
    const TIn* __restrict__ x, const __grid_constant__ SeqList<N> seqs, float* __restrict__ qhat_tile,
    float* __restrict__ qhat_out, float* __restrict__ ckpt, unsigned long long* __restrict__ counters, int n_tiles,
    int n_ckpt, float theta, int basis_exact, int heads, int key_rows, int reverse, uint4* zero_ptr, unsigned zero_n16) {
  // x: the stream that becomes the delta matrix: packed queries, a sequence's [heads][T][D] behind one
  // another (key_rows = 0), or keys in the KV-cache layout [heads][key_rows][D], rows 0..T-1 read
  const Seq& sq = seqs.s[N == 1 ? 0 : blockIdx.y];
  const int T = sq.T, src_rows = key_rows ? key_rows : T;
  constexpr int NW = D / 32;                       // chain warps
  constexpr uint32_t ROW_BYTES = D * sizeof(TIn);
  constexpr uint32_t STAGE_BYTES = RROWS * ROW_BYTES;
  extern __shared__ __align__(128) unsigned char ring[];   // [RSTAGES][RROWS][D] of TIn
  __shared__ __align__(8) unsigned long long bars[2 * RSTAGES];   // full[RSTAGES], empty[RSTAGES]
  __shared__ int s_fail;

  const int bh = sq.b * heads + (int)blockIdx.x;   // head of the workspace arrays
  const TIn* const q = key_rows ? x + (size_t)bh * src_rows * D : x + sq.q_off + (size_t)blockIdx.x * T * D;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t full0 = smem_u32(&bars[0]), empty0 = smem_u32(&bars[RSTAGES]);
  const int n_chunks = (T + RROWS - 1) / RROWS;
  if (tid == 0) {
    for (int s = 0; s < RSTAGES; ++s) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(full0 + 8 * s), "r"(1) : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(empty0 + 8 * s), "r"(NW) : "memory");
    }
    s_fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  // (the order of these two: see the table kernel)
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  // the deferred clearing of a state reset (see the table kernel)
  if (zero_ptr && blockIdx.x == 0 && blockIdx.y == 0)
    for (unsigned i = tid; i < zero_n16; i += blockDim.x) zero_ptr[i] = make_uint4(0u, 0u, 0u, 0u);

  if (warp == NW) {
    // ---- producer: keeps up to RSTAGES stages of query rows in flight
    if (lane == 0) {
      const unsigned char* src = reinterpret_cast<const unsigned char*>(q);
      const uint32_t ring0 = smem_u32(ring);
      for (int i = 0; i < n_chunks; ++i) {
        const int s = i % RSTAGES;
        if (i >= RSTAGES && !mbar_wait(empty0 + 8 * s, ((i / RSTAGES) - 1) & 1)) { s_fail = 1; break; }
        const int ci = reverse ? n_chunks - 1 - i : i;      // stage of the head in token order
        const int rows = min(RROWS, T - ci * RROWS);
        const uint32_t bytes = (uint32_t)rows * ROW_BYTES;
        // (bounds-checking build: the stage's rows lie inside the head's rows of the stream)
        if (!DELTA_IN((size_t)ci * RROWS + rows - 1, src_rows, counters)) { s_fail = 1; break; }
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(full0 + 8 * s),
                     "r"(bytes)
                     : "memory");
        asm volatile(
            "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                ring0 + s * STAGE_BYTES),
            "l"(src + (size_t)ci * STAGE_BYTES), "r"(bytes), "r"(full0 + 8 * s)
            : "memory");
      }
    }
  } else {
    // ---- chain warps: thread c owns channel c
    const int c = tid;
    float* ckptp = ckpt + (size_t)bh * n_ckpt * D + c;
    float qh = 0.0f;          // reference state, starts at zero (Eq. 3)
    bool failed = false;
    for (int i = 0; i < n_chunks; ++i) {
      const int s = i % RSTAGES;
      const int t0 = (reverse ? n_chunks - 1 - i : i) * RROWS;
      if (qhat_tile && (t0 % DELTA_TILE_ROWS) == 0 && DELTA_IN(t0 / DELTA_TILE_ROWS, n_tiles, counters))
        qhat_tile[((size_t)bh * n_tiles + t0 / DELTA_TILE_ROWS) * D + c] = qh;
      if (!mbar_wait(full0 + 8 * s, (i / RSTAGES) & 1)) { failed = true; break; }
      const TIn* rows = reinterpret_cast<const TIn*>(ring + (size_t)s * STAGE_BYTES) + c;
      const int nrows = min(RROWS, T - t0);
      if (reverse)
        chain_stage_rev<TIn, D>(rows, t0, nrows, t0 + nrows == T && basis_exact, qh, theta, ckptp, n_ckpt, counters);
      else
        chain_stage<TIn, D>(rows, t0, nrows, t0 == 0 && basis_exact, qh, theta, ckptp, n_ckpt, counters);
      __syncwarp();
      if (lane == 0)
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(empty0 + 8 * s) : "memory");
    }
    if (!failed && qhat_out) qhat_out[(size_t)bh * D + c] = qh;
    if (failed) s_fail = 1;
  }
  __syncthreads();
  if (tid == 0 && s_fail) atomicMax(&counters[CNT_STATUS], (unsigned long long)DELTA_ERR_TIMEOUT);
}


template <typename TIn, int D, int N>
static cudaError_t launch_rows(const Shape& s, const Workspace& w, const void* x, const SeqBatch& seqs, float theta, int init,
                               bool key_stream, bool reverse, void* zero_ptr, size_t zero_bytes, cudaStream_t st) {
  auto kern = delta_chain_rows_kernel<TIn, D, N>;
  constexpr size_t need = (size_t)RSTAGES * RROWS * D * sizeof(TIn);
  static_assert(need <= kMaxChainSmem, "shared memory");
  static std::atomic<uint64_t> ready{0};
  if (!device_done(ready)) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxChainSmem);
    if (e != cudaSuccess) return e;
    device_mark(ready);
  }
  SeqList<N> list;
  for (int i = 0; i < N; ++i) list.s[i] = seqs.s[i < seqs.n ? i : 0];
  const int heads = key_stream ? s.H_kv : s.H;
  const dim3 grid((unsigned)(seqs.ragged ? heads : s.B * heads), (unsigned)seqs.n);
  cudaLaunchAttribute attr[1];
  cudaLaunchConfig_t cfg = serialised_launch(attr, st);
  cfg.gridDim = grid;
  cfg.blockDim = dim3(D + 32);
  cfg.dynamicSmemBytes = even_spread_smem(need, (long)grid.x * grid.y);
  const cudaError_t err =
      cudaLaunchKernelEx(&cfg, kern, (const TIn*)x, list, w.qhat_tile, w.qhat[0], w.ckpt, w.counters, s.n_tiles, s.n_ckpt(),
                         theta, init == DELTA_INIT_BASIS_EXACT ? 1 : 0, heads, key_stream ? s.T_max : 0, reverse ? 1 : 0,
                         (uint4*)zero_ptr, (unsigned)(zero_bytes / 16));
  count_launch();
  return err != cudaSuccess ? err : cudaGetLastError();
}

static cudaError_t launch_delta_chain_rows(const Shape& s, const Workspace& w, const void* x, const SeqBatch& seqs,
                                           float theta, int dtype, int init, bool key_stream, bool reverse, void* zero_ptr,
                                           size_t zero_bytes, cudaStream_t st) {
#define GO(TIN, DD)                                                                                              \
  return seqs.ragged                                                                                             \
             ? launch_rows<TIN, DD, kSeqMax>(s, w, x, seqs, theta, init, key_stream, reverse, zero_ptr, zero_bytes, st) \
             : launch_rows<TIN, DD, 1>(s, w, x, seqs, theta, init, key_stream, reverse, zero_ptr, zero_bytes, st)
  if (dtype == DELTA_F32) {
    if (s.d == 64) { GO(float, 64); } else { GO(float, 128); }
  } else {
    if (s.d == 64) { GO(__nv_bfloat16, 64); } else { GO(__nv_bfloat16, 128); }
  }
#undef GO
}

// SMs of the current device (queried once per device).
int device_sm_count() {
  static int cached[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 148;
  if (!cached[dev]) {
    int n = 0;
    cached[dev] = (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && n > 0) ? n : 148;
  }
  return cached[dev];
}

bool chain_by_tables(const Shape& s, const SeqBatch& seqs, int dtype, bool key_stream) {
  // The table kernel while its CTAs (head x 32 channels) are all resident at once: two per SM for bf16, one for fp32
  // (shared memory: 96 and 128 KB).  Whole prefill, tables against rows: 64 CTAs (1 x 32 heads, 1024 tokens) 28.8 us, 34.0;
  // 160 (2 x 20 heads, d = 128, 1531 tokens) 87.9, 90.2; 192 59.5, 61.5; 256 75.0, 77.0; 384 112.6, 110.0; 512 147.5, 139.5.
  // In a ragged group, whose longest sequences come first, the CTAs count by their rows: six sequences of 99 to 1900 tokens,
  // 32 heads, rows 121.8 us, tables 116.2; eight of 200 to 4000 264, 243; four of 90 to 900, key deltas 33.4, 28.4; four
  // of 300 to 1500, 20 heads, d = 128 142.2, 143.1.
  const long seq_ctas = (long)(seqs.ragged ? 1 : s.B) * (key_stream ? s.H_kv : s.H) * (s.d / CH);
  // (Rows of the longest sequence save 3.2 ns each, a map costs the caller a quarter of a microsecond: three fp32 sequences of up
  // to 106 tokens 19.1 us by rows, 20.2; eight of up to 74 24.1, 25.3.)
  if (seqs.ragged && seqs.T_longest < 80 * seqs.n) return false;
  long rows = 0;
  for (int i = 0; i < seqs.n; ++i) rows += seqs.s[i].T;
  return seq_ctas * rows <= (long)device_sm_count() * (dtype == DELTA_F32 ? 1 : 2) * seqs.T_longest;
}

// (In the decode steps' scratch, which nothing in flight uses during a prefill; it holds 256 (d + 2) bytes per head.)
unsigned* chain_progress(const Shape& s, const Workspace& w, const SeqBatch& seqs, int dtype, bool key_stream) {
  return seqs.beside >= 0 && chain_by_tables(s, seqs, dtype, key_stream) && tcq_begins_beside_chain(s, seqs, seqs.beside)
             ? reinterpret_cast<unsigned*>(w.dec_partial) : nullptr;
}

cudaError_t launch_delta_chain(const Shape& s, const Workspace& w, const void* x, const SeqBatch& seqs, float theta,
                               int dtype, int init, bool key_stream, bool reverse, void* zero_ptr, size_t zero_bytes,
                               cudaStream_t st) {
  if (key_stream && reverse) return cudaErrorNotSupported;
  if (((uintptr_t)zero_ptr | zero_bytes) & 15u) return cudaErrorInvalidValue;
  if (chain_by_tables(s, seqs, dtype, key_stream))
    return launch_delta_chain_tables(s, w, x, seqs, theta, dtype, init, key_stream, reverse,
                                     chain_progress(s, w, seqs, dtype, key_stream), zero_ptr, zero_bytes, st);
  return launch_delta_chain_rows(s, w, x, seqs, theta, dtype, init, key_stream, reverse, zero_ptr, zero_bytes, st);
}

// ---------------------------------------------------------------------------------------
// delta_finish_kernel: issue-bound (about 640 instructions per warp and 8-row block); two channels per
// lane halve what a row costs against one: 8 x 32 heads x 4096 rows 151 -> 120 us (4.3 TB/s).
// Block roles by blockIdx.x.
//   [0, n_idx_blocks): one block per (batch, head, 64-row tile): row/tile counts, compacted
//       indices, counters of Eq. 6 (d multiply-adds per in-window causal pair,
//       nnz(Delta q_i) per out-of-window pair, against d per causal pair of dense attention).
//   [n_idx_blocks, ...): one block per (batch, KV head, 64 keys): hand-off row
//       R(T-1)[j] = q_hat(T-1).k_j for the heads of the group.
template <typename TIn, int D, int N>
__global__ void __launch_bounds__(256, D == 64 ? 5 : 4) delta_finish_kernel(
    const __grid_constant__ SeqList<N> seqs,
    uint32_t* __restrict__ mask, uint16_t* __restrict__ row_nnz,
    uint32_t* __restrict__ tile_nnz, uint8_t* __restrict__ idx,
    unsigned long long* __restrict__ counters, const TIn* __restrict__ k,
    const float* __restrict__ qhat, float* __restrict__ R,
    int T_max, int n_tiles, int heads, int seq_heads, int seq_kv, int H, int g, int shape,
    int key_stream, const TIn* __restrict__ x, float* __restrict__ dq,
    __nv_bfloat16* __restrict__ ref_rows, const float* __restrict__ ckpt, int n_ckpt, float theta,
    int basis_exact, int reverse, int wait_front) {
  // (arguments: see finish_block)
  // Launched with programmatic stream serialisation.  wait_front: the results of everything
  // in front are visible from here on (no effect in an ordinary launch).  Without it (query
  // deltas behind the telescoped attention kernel, of which this kernel needs nothing): every
  // CTA of the attention kernel has released this kernel after its own wait for the chain
  // kernel, so the chain's results are complete; they are read past the L1 cache (ld.global.cg),
  // and the blocks run on the SMs the attention kernel's last wave leaves idle.  One thread of the
  // grid waits at its end: a kernel serialised programmatically behind this one (a decode step) waits for
  // this kernel only, and with it has to have waited for the attention kernel's stores too.  (Every
  // CTA of the attention kernel is resident by then, so nothing can be kept from starting.  It costs up to
  // 1.1 us where the attention kernel ends last -- three ragged sequences of up to 392 tokens, d = 128:
  // 22.9 -> 24.1 us; BitNet layer 63.8 -> 64.2 -- and nothing at the Llama layer.)
  if (wait_front) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // key deltas: the attention kernel is serialised programmatically behind this one and may set
    // itself up meanwhile (it waits for this kernel's results itself).  Not where this kernel comes last: the next prefill's chain
    // CTAs would become resident beside the attention kernel's last wave, several on each of the few SMs it leaves
    // (1 x 32 heads, 1024 tokens 30.3 us, so 26.0; d = 128, 2048 tokens 70.0, so 61.5).
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  }
  __shared__ __align__(16) unsigned char smem[kFinishSmem<D, 8>];
  finish_block<TIn, D, 8>(seqs.s[N == 1 ? 0 : blockIdx.y], (int)blockIdx.x, smem, mask, row_nnz, tile_nnz, idx, counters, k, qhat, R, T_max,
                          n_tiles, heads, seq_heads, seq_kv, H, g, shape, key_stream, x, dq, ref_rows, ckpt, n_ckpt, theta,
                          basis_exact, reverse);
  if (!wait_front && threadIdx.x == 0 && blockIdx.x == 0 && blockIdx.y == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
}

// The channel-major fp32 copy of the keys that the tensor-core kernel with the FP32 delta path reads.
template <typename TIn, int D>
__global__ void __launch_bounds__(256) key_copy_kernel(const TIn* __restrict__ k, float* __restrict__ kt, int T, int T_max, int kt_ld) {
  __shared__ float tile[D][65];
  const int bkv = blockIdx.y, j0 = blockIdx.x * 64;
  for (int e = threadIdx.x; e < 64 * D; e += 256) {
    const int j = e / D, c = e % D;
    tile[c][j] = j0 + j < T ? to_f32(k[((size_t)bkv * T_max + j0 + j) * D + c]) : 0.0f;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < 64 * D; e += 256)
    if (j0 + (e & 63) < kt_ld) kt[((size_t)bkv * D + (e >> 6)) * kt_ld + j0 + (e & 63)] = tile[e >> 6][e & 63];
}

template <typename TIn, int D, int N>
static cudaError_t launch_finish(const Shape& s, const Workspace& w, const void* q, const void* k, const SeqBatch& seqs,
                                 float theta, int shape, int init, bool want_kt, bool key_stream, bool reverse,
                                 int programmatic, cudaStream_t st) {
  // programmatic: 0 = ordinary launch, 1 = programmatic serialisation, 2 = the same and the kernel
  // does not wait for the kernel in front (see the kernel)
  // key deltas: the index/counter pass runs over the KV heads and there is no hand-off row
  const int heads = key_stream ? s.H_kv : s.H, nb = seqs.ragged ? 1 : s.B;
  const int tiles = (seqs.T_longest + DELTA_TILE_ROWS - 1) / DELTA_TILE_ROWS;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(nb * (heads * tiles + (key_stream ? 0 : s.H_kv * tiles))), (unsigned)seqs.n);
  cfg.blockDim = dim3(256);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = programmatic ? 1 : 0;
  SeqList<N> list;
  for (int i = 0; i < N; ++i) list.s[i] = seqs.s[i < seqs.n ? i : 0];
  const cudaError_t err = cudaLaunchKernelEx(
      &cfg, delta_finish_kernel<TIn, D, N>, list, w.mask, w.row_nnz, w.tile_nnz, w.idx, w.counters, (const TIn*)k,
      (const float*)w.qhat[0], w.R, s.T_max, s.n_tiles, heads, nb * heads, nb * s.H_kv,
      s.H, s.g(), shape, key_stream ? 1 : 0, (const TIn*)(key_stream ? k : q), w.dq,
      key_stream ? w.qhat_rows : (__nv_bfloat16*)nullptr, (const float*)w.ckpt, s.n_ckpt(), theta,
      init == DELTA_INIT_BASIS_EXACT ? 1 : 0, reverse ? 1 : 0, programmatic == 2 ? 0 : 1);
  count_launch();
  if (err == cudaSuccess && want_kt && w.kt) {       // (uniform batches only)
    key_copy_kernel<TIn, D><<<dim3((unsigned)((seqs.T_longest + 63) / 64), (unsigned)(s.B * s.H_kv)), 256, 0, st>>>(
        (const TIn*)k, w.kt, seqs.T_longest, s.T_max, (s.T_max + 3) / 4 * 4);
    count_launch();
  }
  return err != cudaSuccess ? err : cudaGetLastError();
}

cudaError_t launch_delta_finish(const Shape& s, const Workspace& w, const void* q, const void* k, const SeqBatch& seqs,
                                float theta, int shape, int dtype, int init, bool want_kt, bool key_stream, bool reverse,
                                int programmatic, cudaStream_t st) {
#define GO(TIN, DD)                                                                                               \
  return seqs.ragged ? launch_finish<TIN, DD, kSeqMax>(s, w, q, k, seqs, theta, shape, init, want_kt, key_stream, \
                                                       reverse, programmatic, st)                                 \
                     : launch_finish<TIN, DD, 1>(s, w, q, k, seqs, theta, shape, init, want_kt, key_stream, reverse, \
                                                 programmatic, st)
  if (dtype == DELTA_F32) {
    if (s.d == 64) { GO(float, 64); } else { GO(float, 128); }
  } else {
    if (s.d == 64) { GO(__nv_bfloat16, 64); } else { GO(__nv_bfloat16, 128); }
  }
#undef GO
}

}  // namespace delta
