// K3 (fp32 caches) -- one decode step of strategy (1) on the FP32 pipes (Section III-A "Decoding Stage
// Considerations", Section III-B "Decoding Stage").
//
// The organisation is that of k3_decode_step_mma.cu: a warp owns units of 32 keys, brings their rows in by
// itself (keys by TMA with the 128-byte swizzle, values by one bulk copy), keeps its own running softmax,
// and the warps meet once, at the end (decode_merge.cuh).  Eq. 4's running sum is taken in its telescoped
// form R(n)[j] = q_hat(n).k_j: the references are copies of input elements, so it carries fewer
// roundings than adding rounded differences step by step, and R is written and never read.
//   scores  lane = key: sixteen bytes of the lane's own row per load (eight lanes of a phase read eight
//           different swizzled chunks) against references and queries broadcast from shared memory,
//           packed fma.rn.f32x2; queries only where the unit touches the window;
//   P.V     lane = D / 32 channels, probabilities broadcast.
// Bound: dependent latencies at the sizes fp32 is used at (16 heads over 1000 keys move 2 MB).  The unit of the row
// that arrives with the step comes by TMA like the others (row by row it kept its warp, the step's last, 0.4 us
// longer) and a CTA combines its warps before one record per block of 16 channels travels (decode_merge.cuh).
// us per step, with block barriers around every tile and a merge through global memory -> warps on their own, every
// warp sending -> so: 16 heads at 1000 keys 10.3 -> 5.0 -> 4.4; 2 x 16 at 2000 5.4 -> 4.8; d = 128 6.8 -> 6.0.
#include "decode_common.cuh"
#include "decode_merge.cuh"

namespace delta {

namespace {
template <int D> constexpr int kF32Warps = D == 64 ? 8 : 4;

struct F32DecodeParams {
  const float *q_new, *k_new, *v_new, *ref_in;
  float *k_cache, *v_cache, *out, *ref_out, *R, *partial;
  uint32_t* ticket;
  unsigned long long* counters;
  int n, T_max, H, chunk, nsplit, W, b0;
  float theta, scale_log2e;
  int ragged;
  int n_b[kRaggedMax];                    // ragged: tokens seen per batch element b0 ..
};
template <int D, int G> struct F32DecSmem {
  static constexpr int NW = kF32Warps<D>;
  static constexpr uint32_t HALF = UK * D * 4, RING = NW * 2 * HALF;
  static constexpr int NB = G * D / 16;
  static constexpr uint32_t PROBS = NW * UK * G * 4, ROWS = 2 * G * D * 4;      // probabilities; references, queries
  static_assert(MergePart<D, G>::BYTES <= HALF, "a warp's result fits its key slot");
  // records of a CTA of a cluster of cs
  __host__ __device__ static constexpr uint32_t rec_bytes(int cs) { return merge_slots<D, G>(cs) * cs * REC2 * 4; }
  static constexpr size_t bytes(int cs) { return 1024 + RING + rec_bytes(cs) + PROBS + ROWS; }
  static constexpr size_t bytes_max = 1024 + RING + (NB + kMaxCluster - 1) * REC2 * 4 + PROBS + ROWS;
};
}  // namespace

template <int D, int G, bool CLUSTER>
__global__ void __launch_bounds__(32 * kF32Warps<D>, 1)
decode_step_f32_kernel(const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ F32DecodeParams p) {
  using SM = F32DecSmem<D, G>;
  constexpr int NW = SM::NW, NT = 32 * NW;
  constexpr int NBLK = D / 32;               // 128-byte blocks of a key row
  constexpr int CPL = D / 32;                // channels per lane of P.V
  extern __shared__ unsigned char dsm_raw[];
  __shared__ __align__(8) unsigned long long bars[2 * NW + 1];
  __shared__ int s_last, s_fail;
  const uint32_t ring = (smem_u32(dsm_raw) + 1023u) & ~1023u;
  unsigned char* const sm = dsm_raw + (ring - smem_u32(dsm_raw));
  const int cs = CLUSTER ? p.nsplit : 1;
  const uint32_t recs = ring + SM::RING;
  float* const s_p = reinterpret_cast<float*>(sm + SM::RING + SM::rec_bytes(cs));     // [NW][UK][G]
  float* const s_ref = s_p + SM::PROBS / 4;  // [G][D]
  float* const s_q = s_ref + G * D;          // [G][D]

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int split = blockIdx.x, H_kv = p.H / G, bkv = p.b0 * H_kv + blockIdx.y;
  const int b = bkv / H_kv, kvh = bkv - b * H_kv;
  const int n = p.ragged ? p.n_b[b - p.b0] : p.n, T_max = p.T_max, W = p.W;
  const int L = n + 1, j0 = split * p.chunk, j1 = min(j0 + p.chunk, L);
  const int rank = CLUSTER ? split : 0;
  const uint32_t bar_m = smem_u32(&bars[2 * NW]), bar_k = smem_u32(&bars[2 * warp]), bar_v = bar_k + 8;
  if (CLUSTER) {
    if (tid == 0) {
      tc::mbar_init(bar_m, 1);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
      tc::mbar_expect_tx(bar_m, (uint32_t)((SM::NB - rank + cs - 1) / cs * cs) * (16 + 2) * 4);
    }
    __syncwarp();
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  }
  if (!CLUSTER && j0 >= L) return;           // ragged batch: this sequence has fewer slices
  const uint32_t lead = lane == 0;
  if (lane == 0) {
    if (warp == 0) asm volatile("prefetch.tensormap [%0];" ::"l"(&tm_k) : "memory");
    tc::mbar_init(bar_k, 1);
    tc::mbar_init(bar_v, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    tc::fence_proxy_async();
  }
  if (tid == 0) s_fail = 0;
  __syncwarp();

  const size_t row0 = (size_t)bkv * T_max;
  const float* const kn = p.k_new + (size_t)bkv * D;
  const float* const vn = p.v_new + (size_t)bkv * D;
  const int wl = n - W + 1;                  // first key inside the decode window
  unsigned char* const my = sm + (size_t)warp * 2 * SM::HALF;
  const uint32_t slot_k = ring + (uint32_t)warp * 2 * SM::HALF, slot_v = slot_k + SM::HALF;
  // row r, 16-byte chunk c of a 128-byte block: r * 128 + ((c ^ (r & 7)) << 4); values: plain rows
  // (the unit of the row that arrives with the step too: rows behind the cached ones hold anything, that row and
  // zeros are written over them; the values end with the cache)
  auto fetch = [&](int jg) {
    tc::mbar_expect_tx_if(lead, bar_k, SM::HALF);
#pragma unroll
    for (int c = 0; c < NBLK; ++c) tc::tma_load_3d_if(lead, slot_k + c * UK * 128, &tm_k, bar_k, 32 * c, jg, bkv);
    const uint32_t vbytes = (uint32_t)min(UK, T_max - jg) * D * 4;
    if (lane == 0) {
      tc::mbar_expect_tx(bar_v, vbytes);
      bulk_load(slot_v, p.v_cache + (row0 + jg) * D, vbytes, bar_v);
    }
  };
  // the warp that owns the row arriving with the step
  const bool has_new = j1 == L && j0 < L && ((n - j0) / UK) % NW == warp;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  int jg = j0 + UK * warp;
  if (jg < j1) fetch(jg);
  float4 k_row = make_float4(0.0f, 0.0f, 0.0f, 0.0f), v_row = k_row;       // that row: four channels per lane
  if (has_new && lane < D / 4) {
    k_row = __ldcg(reinterpret_cast<const float4*>(kn) + lane);
    v_row = __ldcg(reinterpret_cast<const float4*>(vn) + lane);
  }

  // ---- threshold step (Eq. 2-3) into shared memory
  int fired = 0;
  const size_t o0 = ((size_t)b * p.H + kvh * G) * D;
  for (int e = tid; e < G * D; e += NT) {
    const float x = __ldcg(p.q_new + o0 + e), old = __ldcg(p.ref_in + o0 + e);
    const bool fire = fabsf(__fsub_rn(x, old)) > p.theta;
    const float nq = fire ? x : old;
    s_q[e] = x;
    s_ref[e] = nq;
    fired += fire ? 1 : 0;
    if (split == 0) p.ref_out[o0 + e] = nq;
  }
  __syncthreads();
  float o[G][CPL], m[G], l[G];
#pragma unroll
  for (int h = 0; h < G; ++h) {
    m[h] = -INFINITY;
    l[h] = 0.0f;
#pragma unroll
    for (int c = 0; c < CPL; ++c) o[h][c] = 0.0f;
  }
  uint32_t ph = 0;
  float* const pw = s_p + (size_t)warp * UK * G;
  // the lane's key against G rows of operands
  auto dots = [&](const float* rows, float (&s)[G]) {
    float2 acc[G];
#pragma unroll
    for (int h = 0; h < G; ++h) acc[h] = make_float2(0.0f, 0.0f);
#pragma unroll
    for (int c = 0; c < NBLK; ++c)
#pragma unroll
      for (int x = 0; x < 8; ++x) {
        const float4 kk = tc::lds128(slot_k + c * UK * 128 + lane * 128 + ((x ^ (lane & 7)) << 4));
#pragma unroll
        for (int h = 0; h < G; ++h) {
          const float4 r = *reinterpret_cast<const float4*>(rows + h * D + 32 * c + 4 * x);
          acc[h] = tc::ffma2(make_float2(kk.x, kk.y), make_float2(r.x, r.y), acc[h]);
          acc[h] = tc::ffma2(make_float2(kk.z, kk.w), make_float2(r.z, r.w), acc[h]);
        }
      }
#pragma unroll
    for (int h = 0; h < G; ++h) s[h] = acc[h].x + acc[h].y;
  };
  for (; jg < j1; jg += UK * NW) {
    const int jn = jg + UK * NW, j = jg + lane;
    const bool owner = n < jg + UK, live = j <= n;
    if (!mbar_wait(bar_k, ph)) s_fail = 1;
    if (owner) {                             // the new key's row (what the rows behind it hold is masked)
      const int r = n - jg;
      if (lane < D / 4)
        sts_f4(slot_k + (lane >> 3) * (UK * 128) + r * 128 + (((lane & 7) ^ (r & 7)) << 4), k_row.x, k_row.y, k_row.z, k_row.w);
      __syncwarp();
    }
    float s[G];
    dots(s_ref, s);
    if (live && DELTA_IN(j, T_max, p.counters)) {
      float* const Rj = p.R + ((size_t)b * p.H + kvh * G) * T_max + j;      // R[j] = q_hat . k_j
#pragma unroll
      for (int h = 0; h < G; ++h) Rj[(size_t)h * T_max] = s[h];
    }
    if (jg + UK > wl) {                      // the unit touches the window
      float e[G];
      dots(s_q, e);
#pragma unroll
      for (int h = 0; h < G; ++h) s[h] = j >= wl ? e[h] : s[h];
    }
#pragma unroll
    for (int h = 0; h < G; ++h) {
      const float x = live ? s[h] * p.scale_log2e : -INFINITY;
      const float mn = fmaxf(m[h], warp_max(x)), al = exp2f(m[h] - mn), pr = exp2f(x - mn);
      m[h] = mn;
      l[h] = fmaf(l[h], al, pr);
#pragma unroll
      for (int c = 0; c < CPL; ++c) o[h][c] *= al;
      pw[lane * G + h] = pr;
    }
    if (!mbar_wait(bar_v, ph)) s_fail = 1;
    if (owner) {                             // the new value's row, zeros behind it
      const int r = n - jg;
      if (lane < D / 4) sts_f4(slot_v + r * D * 4 + 16 * lane, v_row.x, v_row.y, v_row.z, v_row.w);
#pragma unroll 1
      for (int e = (r + 1) * (D / 4) + lane; e < UK * (D / 4); e += 32) sts_f4(slot_v + 16 * e, 0.0f, 0.0f, 0.0f, 0.0f);
    }
    __syncwarp();
    const float* const vt = reinterpret_cast<const float*>(my + SM::HALF) + CPL * lane;
#pragma unroll 8
    for (int r = 0; r < UK; ++r) {
      float vv[CPL], pr[G];
      if constexpr (CPL == 2) {
        const float2 x = *reinterpret_cast<const float2*>(vt + r * D);
        vv[0] = x.x; vv[1] = x.y;
      } else {
        const float4 x = *reinterpret_cast<const float4*>(vt + r * D);
        vv[0] = x.x; vv[1] = x.y; vv[2] = x.z; vv[3] = x.w;
      }
#pragma unroll
      for (int h = 0; h < G; h += G % 4 == 0 ? 4 : 1) {
        if constexpr (G % 4 == 0) {
          const float4 x = *reinterpret_cast<const float4*>(pw + r * G + h);
          pr[h] = x.x; pr[h + 1] = x.y; pr[h + 2] = x.z; pr[h + 3] = x.w;
        } else {
          pr[h] = pw[r * G + h];
        }
      }
#pragma unroll
      for (int h = 0; h < G; ++h)
#pragma unroll
        for (int c = 0; c < CPL; c += 2) {
          const float2 x = tc::ffma2(make_float2(pr[h], pr[h]), make_float2(vv[c], vv[c + 1]), make_float2(o[h][c], o[h][c + 1]));
          o[h][c] = x.x; o[h][c + 1] = x.y;
        }
    }
    __syncwarp();                            // the warp is done with the unit
    ph ^= 1u;
    if (jn < j1) fetch(jn);
  }

  // ---- merge: the warp's part into its key slot (every copy into it is complete and read)
  using MP = MergePart<D, G>;
#pragma unroll
  for (int h = 0; h < G; ++h) {
#pragma unroll
    for (int x = 16; x > 0; x >>= 1) l[h] += __shfl_xor_sync(0xffffffffu, l[h], x);
    const uint32_t at = slot_k + (h * MP::LD + CPL * lane) * 4;
    if constexpr (CPL == 2) sts_f2(at, o[h][0], o[h][1]); else sts_f4(at, o[h][0], o[h][1], o[h][2], o[h][3]);
    if (lane == 0) sts_f2(slot_k + MP::ML + h * 8, m[h], l[h]);
  }
  __syncthreads();
  if (CLUSTER) asm volatile("barrier.cluster.wait.aligned;" ::: "memory");          // every slice runs
  const int n_slices = (L + p.chunk - 1) / p.chunk;
  merge_warps<float, D, G, NW, CLUSTER>(ring, 2 * SM::HALF, recs, bar_m, rank, cs, n_slices, split, bkv, o0, p.partial, p.out);
  // ---- while the parts travel: the caches' new row, the counters
  if (has_new && lane < D / 4 && DELTA_IN(n, T_max, p.counters)) {
    reinterpret_cast<float4*>(p.k_cache + (row0 + n) * D)[lane] = k_row;
    reinterpret_cast<float4*>(p.v_cache + (row0 + n) * D)[lane] = v_row;
  }
  if (split == 0) {
    const int f = warp_sum(fired);
    if (lane == 0) {
      const int n_in = min(L, max(W, 0));
      if (f) atomicAdd(&p.counters[CNT_DECODE_NNZ], (unsigned long long)f);
      if (f) atomicAdd(&p.counters[CNT_DECODE_MACS_DONE], (unsigned long long)(L - n_in) * f);
      if (warp == 0) {
        atomicAdd(&p.counters[CNT_DECODE_MACS_DONE], (unsigned long long)n_in * D * G);
        atomicAdd(&p.counters[CNT_DECODE_ELEMS], (unsigned long long)G * D);
        atomicAdd(&p.counters[CNT_DECODE_MACS_DENSE], (unsigned long long)L * D * G);
      }
    }
  }
  if (CLUSTER) {
    // (every slice's block records: also what keeps this CTA until the last of them has been sent to it)
    if (!merge_slices<float, D, G, NW>(recs, bar_m, rank, cs, o0, p.out)) s_fail = 1;
  } else if (n_slices > 1) {
    merge_global<float, D, G, NW>(n_slices, bkv, o0, p.partial, p.ticket, p.out, &s_last);
  }
  if (s_fail && lane == 0) atomicMax(&p.counters[CNT_STATUS], (unsigned long long)DELTA_ERR_TIMEOUT);
}

template <int D, int G, bool CLUSTER>
static cudaError_t launch_f32_step(const CUtensorMap& tk, const F32DecodeParams& p, int bkv, cudaStream_t st) {
  using SM = F32DecSmem<D, G>;
  auto kern = decode_step_f32_kernel<D, G, CLUSTER>;
  static std::atomic<uint64_t> ready{0};
  if (!device_done(ready)) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SM::bytes_max);
    if (e == cudaSuccess && CLUSTER) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    device_mark(ready);
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)p.nsplit, (unsigned)bkv);
  cfg.blockDim = dim3(32 * kF32Warps<D>);
  cfg.dynamicSmemBytes = SM::bytes(CLUSTER ? p.nsplit : 1);
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)p.nsplit;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = CLUSTER ? 2 : 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, tk, p);
  count_launch();
  return e;
}

cudaError_t launch_decode_step_f32(const Shape& s, const Workspace& w, const void* q_new, const void* k_new,
                                   const void* v_new, void* k_cache, void* v_cache, void* out, int n, const int* n_b,
                                   float theta, int window, int qhat_sel, DecodeTmapCache* map, cudaStream_t st) {
  CUtensorMap* const tk = reinterpret_cast<CUtensorMap*>(map->map);
  if (map->ptr != k_cache) {
    if (!tc::encode3(tk, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, k_cache, (uint64_t)s.d, (uint64_t)s.T_max, (uint64_t)s.B * s.H_kv,
                     (uint64_t)s.d * 4, (uint64_t)s.T_max * s.d * 4, 32, UK, CU_TENSOR_MAP_SWIZZLE_128B))
      return cudaErrorInvalidValue;
    map->ptr = k_cache;
  }
  F32DecodeParams p;
  p.q_new = (const float*)q_new; p.k_new = (const float*)k_new; p.v_new = (const float*)v_new;
  p.ref_in = w.qhat[qhat_sel]; p.ref_out = w.qhat[qhat_sel ^ 1];
  p.k_cache = (float*)k_cache; p.v_cache = (float*)v_cache; p.out = (float*)out; p.R = w.R;
  p.partial = w.dec_partial; p.ticket = w.dec_ticket; p.counters = w.counters;
  p.n = n; p.T_max = s.T_max; p.H = s.H; p.W = window; p.theta = theta;
  p.scale_log2e = 1.4426950408889634f / sqrtf((float)s.d);
  p.ragged = n_b != nullptr;
  bool cluster;
  // (a CTA fills its SM's shared memory; a unit takes about 2 us)
  decode_slices(s, n + 1, s.d == 64 ? kF32Warps<64> : kF32Warps<128>, 0.0f, 2.0f, 0.0f, &p.nsplit, &p.chunk, &cluster);
  cudaError_t err = cudaSuccess;
  for (p.b0 = 0; p.b0 < s.B && err == cudaSuccess; p.b0 += kRaggedMax) {
    const int nb = n_b ? (s.B - p.b0 < kRaggedMax ? s.B - p.b0 : kRaggedMax) : s.B;
    if (n_b)
      for (int i = 0; i < nb; ++i) p.n_b[i] = n_b[p.b0 + i];
#define GO(DD, GG)                                                              \
    err = cluster ? launch_f32_step<DD, GG, true>(*tk, p, nb * s.H_kv, st)      \
                  : launch_f32_step<DD, GG, false>(*tk, p, nb * s.H_kv, st)
#define GO_G(DD)                                        \
    switch (s.g()) {                                    \
      case 1: GO(DD, 1); break;                         \
      case 2: GO(DD, 2); break;                         \
      case 4: GO(DD, 4); break;                         \
      case 8: GO(DD, 8); break;                         \
      default: return cudaErrorInvalidValue;            \
    }
    if (s.d == 64) { GO_G(64) } else { GO_G(128) }
#undef GO_G
#undef GO
    if (!n_b) break;
  }
  return err;
}

}  // namespace delta
