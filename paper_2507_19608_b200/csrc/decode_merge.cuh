// Pieces shared by the decode-step kernels whose warps work on units of 32 keys each on their own: how
// a step is sliced, and how the warps' partial results meet.
//
// Merge.  The result of a (batch, KV head), G heads x D channels, is cut into blocks of 16 channels of one
// head.  The slices of the (batch, KV head) are one thread-block cluster of cs CTAs; block q is finished by
// slice q mod cs (by the CTA itself without a cluster), to whose shared memory every slice sends one record.
#pragma once
#include "decode_common.cuh"
#include "tc_common.cuh"

namespace delta {
namespace {

constexpr int UK = 32;                    // keys a warp works on at a time
constexpr int kMaxCluster = 16;           // slices merged through distributed shared memory
constexpr int kRaggedMax = 64;            // batch elements of one ragged launch

__device__ __forceinline__ void async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }
__device__ __forceinline__ uint32_t cluster_map(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
// Stores into the shared memory of a CTA of the cluster that count their bytes on its barrier: the
// receiver waits for the bytes, and nothing of the sender's (its global stores least of all) has to
// be flushed first, as a cluster barrier with release semantics would.
__device__ __forceinline__ void cluster_send4(uint32_t addr, uint32_t bar, float a, float b, float c, float d) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%2, %3, %4, %5}, [%1];" ::"r"(addr),
               "r"(bar), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}
__device__ __forceinline__ void cluster_send2(uint32_t addr, uint32_t bar, float a, float b) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%2, %3}, [%1];" ::"r"(addr),
               "r"(bar), "f"(a), "f"(b) : "memory");
}
__device__ __forceinline__ void sts_f4(uint32_t addr, float a, float b, float c, float d) {
  asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}
__device__ __forceinline__ void sts_f2(uint32_t addr, float a, float b) {
  asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(a), "f"(b) : "memory");
}
__device__ __forceinline__ float2 lds_f2(uint32_t addr) {
  float2 v;
  asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr));
  return v;
}
__device__ __forceinline__ float4 lds_f4(uint32_t addr) { return tc::lds128(addr); }
__device__ __forceinline__ void store4(__nv_bfloat16* p, float a, float b, float c, float d) {
  const __nv_bfloat162 x = __floats2bfloat162_rn(a, b), y = __floats2bfloat162_rn(c, d);
  *reinterpret_cast<uint2*>(p) = make_uint2(*reinterpret_cast<const uint32_t*>(&x), *reinterpret_cast<const uint32_t*>(&y));
}
__device__ __forceinline__ void store4(float* p, float a, float b, float c, float d) {
  *reinterpret_cast<float4*>(p) = make_float4(a, b, c, d);
}
// maximum over the warp in one instruction
__device__ __forceinline__ float warp_max(float x) {
  float r;
  asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ int warp_sum(int x) {
#pragma unroll
  for (int s = 16; s > 0; s >>= 1) x += __shfl_xor_sync(0xffffffffu, x, s);
  return x;
}

// The last CTA of a (batch, KV head) to arrive merges the slices' parts in global memory.
template <typename TO, int D, int G, int MNW>
__device__ __forceinline__ void merge_global(int ns, int bkv, size_t out0, float* __restrict__ partial, uint32_t* __restrict__ ticket,
                                             TO* __restrict__ out, int* s_last) {
  const int tid = threadIdx.x;
  __threadfence();
  __syncthreads();
  if (tid == 0) *s_last = atomicAdd(&ticket[bkv], 1u) == (uint32_t)ns - 1u;
  __syncthreads();
  if (!*s_last) return;
  __threadfence();
  const float* const pb = partial + (size_t)bkv * kMaxDecodeSplits * G * (D + 2);
  for (int e = tid; e < G * D; e += 32 * MNW) {
    const int hh = e / D, c = e - hh * D;
    float M = -INFINITY, nu = 0.0f, de = 0.0f;
#pragma unroll 8
    for (int r = 0; r < ns; ++r) M = fmaxf(M, __ldcg(pb + ((size_t)r * G + hh) * (D + 2) + D));
#pragma unroll 8
    for (int r = 0; r < ns; ++r) {
      const float* const pr = pb + ((size_t)r * G + hh) * (D + 2);
      const float f = tc::ex2(__ldcg(pr + D) - M);
      nu = fmaf(f, __ldcg(pr + c), nu);
      de = fmaf(f, __ldcg(pr + D + 1), de);
    }
    out[out0 + (size_t)hh * D + c] = from_f32<TO>(nu / de);
  }
  if (tid == 0) ticket[bkv] = 0;                          // ready for the next step
}

// The merge in two steps, for kernels whose warps leave their results as fp32 rows in the CTA's shared memory:
// every `stride` bytes from part on a warp's [head][D + 8] (8 floats apart: the heads' rows fall on
// different banks) and behind them its [head] (maximum, row sum).  The CTA combines its warps' parts first and sends one record of 20 floats (16
// channels of one head, maximum, row sum) per block to the slice that finishes the block.  Sent by every warp
// instead, a record's five packets per lane queue at the receivers: eight times as many of them.
// recs: this CTA's records, [slot][slice][REC2]; bar: their barrier.
constexpr int REC2 = 20;
template <int D, int G> __host__ __device__ constexpr uint32_t merge_slots(int cs) { return (uint32_t)((G * D / 16 + cs - 1) / cs); }
template <int D, int G> struct MergePart {
  static constexpr uint32_t LD = D + 8, ML = G * LD * 4, BYTES = ML + G * 8;
};
// The CTA's own parts (all threads, behind a CTA-wide barrier).
template <typename TO, int D, int G, int MNW, bool CLUSTER>
__device__ __forceinline__ void merge_warps(uint32_t part, uint32_t stride, uint32_t recs, uint32_t bar, int rank, int cs, int ns, int split,
                                            int bkv, size_t out0, float* __restrict__ partial, TO* __restrict__ out) {
  using MP = MergePart<D, G>;
  constexpr int NTH = 32 * MNW;
#pragma unroll
  for (int e0 = 0; e0 < G * D / 4; e0 += NTH) {
    const int e = e0 + (int)threadIdx.x;
    if (G * D / 4 % NTH != 0 && e >= G * D / 4) break;
    const int hh = e / (D / 4), c = 4 * (e % (D / 4));
    float2 ml[MNW];
    float4 o[MNW];
#pragma unroll
    for (int w = 0; w < MNW; ++w) ml[w] = lds_f2(part + w * stride + MP::ML + hh * 8);
#pragma unroll
    for (int w = 0; w < MNW; ++w) o[w] = lds_f4(part + w * stride + (hh * MP::LD + c) * 4);
    float M = ml[0].x, l = 0.0f;
#pragma unroll
    for (int w = 1; w < MNW; ++w) M = fmaxf(M, ml[w].x);
    float4 a = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    // (a warp without keys: maximum -inf, zeros; a slice without keys: all of them)
    const float Mf = M == -INFINITY ? 0.0f : M;
#pragma unroll
    for (int w = 0; w < MNW; ++w) {
      const float f = tc::ex2(ml[w].x - Mf);
      a.x = fmaf(f, o[w].x, a.x); a.y = fmaf(f, o[w].y, a.y); a.z = fmaf(f, o[w].z, a.z); a.w = fmaf(f, o[w].w, a.w);
      l = fmaf(f, ml[w].y, l);
    }
    if (CLUSTER) {
      const int q = hh * (D / 16) + c / 16, r = q % cs;
      const uint32_t dst = cluster_map(recs + (uint32_t)((q / cs) * cs + rank) * (REC2 * 4), r), rbar = cluster_map(bar, r);
      cluster_send4(dst + 4 * (c & 15), rbar, a.x, a.y, a.z, a.w);
      if ((c & 15) == 0) cluster_send2(dst + 64, rbar, M, l);
    } else if (ns == 1) {
      const float inv = 1.0f / l;
      store4(out + out0 + (size_t)hh * D + c, a.x * inv, a.y * inv, a.z * inv, a.w * inv);
    } else {
      // slices through global memory: this slice's part
      float* const pg = partial + (((size_t)bkv * kMaxDecodeSplits + split) * G + hh) * (D + 2);
      pg[c] = a.x; pg[c + 1] = a.y; pg[c + 2] = a.z; pg[c + 3] = a.w;
      if (c == 0) { pg[D] = M; pg[D + 1] = l; }
    }
  }
}
// The blocks this slice finishes, once the records of every slice are there.  By the CTA's last warps: its first one
// is still busy with the counters; the others need not stay.  Threads share four channels' records, so that none has more than four of
// them to go through: that is the very end of the step.  (Four threads from five slices on, two where blocks are many
// and the threads would not do: 8 heads x 128 channels on 128 threads.)  Before, one thread after another's record and
// every warp in a suspended wait -> so, us per step: BitNet layer, batch 2 at 1531 keys 4.81 -> 4.62; 32 heads, batch 4
// at 2048 keys 5.67 -> 5.42; fp32, 16 heads at 1000 keys 4.35 -> 4.19.
template <typename TO, int D, int G, int MNW>
__device__ __forceinline__ bool merge_slices(uint32_t recs, uint32_t bar, int rank, int cs, size_t out0, TO* __restrict__ out) {
  constexpr int NB = G * D / 16;
  const int idx = 32 * MNW - 1 - (int)threadIdx.x;
  // threads per four channels: (slots of 16 blocks) x 4 x sub <= the CTA's threads, cs <= 4 sub
  const int sub = cs <= 4 ? 1 : (NB + cs - 1) / cs * 16 <= 32 * MNW ? 4 : 2;
  const int x0 = idx % sub, c4 = (idx / sub) & 3, slot = idx / (4 * sub), q = slot * cs + rank;
  const bool live = q < NB;
  if (!__any_sync(0xffffffffu, live)) return true;
  const bool ok = mbar_spin(bar, 0);
  const uint32_t rb = recs + (uint32_t)(slot * cs) * (REC2 * 4);
  float2 ml[4];
  float4 o[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int x = x0 + i * sub;
    const bool have = live && x < cs;
    ml[i] = have ? lds_f2(rb + x * (REC2 * 4) + 64) : make_float2(-INFINITY, 0.0f);
    o[i] = have ? lds_f4(rb + x * (REC2 * 4) + 16 * c4) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  }
  float M = fmaxf(fmaxf(ml[0].x, ml[1].x), fmaxf(ml[2].x, ml[3].x));
  if (sub > 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, 1));
  if (sub > 2) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, 2));
  float4 a = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  float l = 0.0f;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float f = tc::ex2(ml[i].x - M);                    // 0 for a slice without keys
    a.x = fmaf(f, o[i].x, a.x); a.y = fmaf(f, o[i].y, a.y); a.z = fmaf(f, o[i].z, a.z); a.w = fmaf(f, o[i].w, a.w);
    l = fmaf(f, ml[i].y, l);
  }
#pragma unroll
  for (int s = 1; s <= 2; s <<= 1) {
    if (sub > s) {
      a.x += __shfl_xor_sync(0xffffffffu, a.x, s); a.y += __shfl_xor_sync(0xffffffffu, a.y, s);
      a.z += __shfl_xor_sync(0xffffffffu, a.z, s); a.w += __shfl_xor_sync(0xffffffffu, a.w, s);
      l += __shfl_xor_sync(0xffffffffu, l, s);
    }
  }
  if (!live || x0 != 0) return ok;
  const float inv = 1.0f / l;
  store4(out + out0 + (size_t)(q / (D / 16)) * D + (q % (D / 16)) * 16 + 4 * c4, a.x * inv, a.y * inv, a.z * inv, a.w * inv);
  return ok;
}
// The same by the CTA's first threads, one record after the other, behind a suspended wait of every warp: key deltas, whose
// warps all have counters to update in front of the merge (us per step, shared by idle warps | so: batch 4 at 1777 keys 5.17,
// 4.99; batch 1 3.78, 3.75; compressed key cache, batch 4 at 1024 keys 6.40, 6.25; batch 16 at 1777 keys 8.04, 8.09).
template <typename TO, int D, int G>
__device__ __forceinline__ bool merge_slices_in_turn(uint32_t recs, uint32_t bar, int rank, int cs, size_t out0, TO* __restrict__ out) {
  constexpr int NB = G * D / 16;
  const int slot = threadIdx.x >> 2, c4 = threadIdx.x & 3, q = slot * cs + rank;
  const bool ok = mbar_wait(bar, 0);
  if (q >= NB) return ok;
  const uint32_t rb = recs + (uint32_t)(slot * cs) * (REC2 * 4);
  float M = -INFINITY, l = 0.0f;
#pragma unroll 8
  for (int x = 0; x < cs; ++x) M = fmaxf(M, lds_f2(rb + x * (REC2 * 4) + 64).x);
  float4 a = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll 8
  for (int x = 0; x < cs; ++x) {
    const float2 ml = lds_f2(rb + x * (REC2 * 4) + 64);
    const float4 o = lds_f4(rb + x * (REC2 * 4) + 16 * c4);
    const float f = tc::ex2(ml.x - M);                       // 0 for a slice without keys
    a.x = fmaf(f, o.x, a.x); a.y = fmaf(f, o.y, a.y); a.z = fmaf(f, o.z, a.z); a.w = fmaf(f, o.w, a.w);
    l = fmaf(f, ml.y, l);
  }
  const float inv = 1.0f / l;
  store4(out + out0 + (size_t)(q / (D / 16)) * D + (q % (D / 16)) * 16 + 4 * c4, a.x * inv, a.y * inv, a.z * inv, a.w * inv);
  return ok;
}
// Slices of a step over sequences of up to L keys (the new one included).  A step takes 3 us plus, for every
// unit a warp works through, 0.83 us (d = 64) or 0.87 us (d = 128) while a CTA has its SM for itself, 1.15 times that
// from half the SMs on, and 1.25 or 1.35 us where two share one (measured with 1 to 16 slices forced, 8 to 128 KV
// heads, 300 to 4100 keys); the slices are those that minimise that.  All slices of a KV head form one cluster,
// and clusters have to find room in a GPC: from 1.75 CTAs per SM on (1.6 for clusters of 9 to 12, 1.35 for 13 to
// 16) some wait for a second wave (batch 16, 2048 keys: 256 CTAs 12 us, 384 CTAs 17 us).  Very long caches of
// few heads: up to 64 slices merged through global memory (4.5 us more than a cluster).  The compressed
// key cache: 1.6 us more per unit, for the rebuilding.
// With these figures instead of those of a slower unit (1.1, 1.3, 1.75), us per step at 2048 keys, 8 KV heads: batch 2
// 5.1 -> 4.7 (6 -> 9 slices), batch 4 6.0 -> 5.7 (4 -> 6); batch 8 at 1024 keys 5.6 -> 5.4 (2 -> 4).
// nw: warps per CTA; us_alone, us_shared: a unit's time with the SM for itself, and shared (0: a CTA fills
// its SM); us_more: a kernel's own extra time per unit.
inline void decode_slices(const Shape& s, int L, int nw, float us_shared, float us_alone, float us_more, int* nsplit_out,
                          int* chunk_out, bool* cluster_out) {
  const int bkv = s.B * s.H_kv, sms = device_sm_count();
  const int units = (L + UK - 1) / UK;
  float best = 3.4e38f;
  int best_ns = 1;
  for (int ns = 1; ns <= kMaxDecodeSplits && (ns - 1) * nw < units; ++ns) {       // a unit per warp at least
    const long ctas = (long)bkv * ns;
    const bool alone = ctas * 100 <= (long)sms * (us_shared == 0.0f ? 92 : 98);
    if (ns > kMaxCluster && ctas > sms) break;
    if (ns > 1 && us_shared == 0.0f && !alone) continue;
    if (ns > 1 && ns <= kMaxCluster && ctas * 100 > (long)sms * (ns <= 8 ? 175 : ns <= 12 ? 160 : 135)) continue;
    const int per = (units + ns - 1) / ns;                       // units per slice; per warp mostly the longest counts
    const float rounds = 0.8f * (float)((per + nw - 1) / nw) + 0.2f * (float)per / (float)nw;
    const float unit = us_shared == 0.0f ? us_alone : !alone ? us_shared : ctas * 2 <= sms ? us_alone : 1.15f * us_alone;
    const float us = rounds * (unit + us_more) +
                     (ns > kMaxCluster ? 4.5f + 0.15f * (float)(ns - 24) : (ns > 8 ? 0.075f : 0.06f) * (float)ns);
    if (us < best) { best = us; best_ns = ns; }
  }
  const int chunk = (units + best_ns - 1) / best_ns * UK;
  *nsplit_out = (L + chunk - 1) / chunk;
  *chunk_out = chunk;
  *cluster_out = *nsplit_out > 1 && *nsplit_out <= kMaxCluster;
}

}  // namespace
}  // namespace delta
