// K3 (bf16 caches) -- one decode step of strategy (1) or strategy (3), head dimension 64 or 128
// (Section III-A "Decoding Stage Considerations", Section III-B "Decoding Stage").
//
// Eq. 4's running sum telescopes: R(n)[j] = q_hat(n) . k_j (query deltas), and for bf16 inputs every
// element of q_hat is a copy of an input element, so a step's scores are two small dense products
// per cached key, q_hat . k_j outside the window and q . k_j inside it.  Key deltas (KEY): one
// product, q . k_hat(j) outside the window and q . k_j inside it, k_hat(j) being the rows of the
// library's reference-key cache.
//
// Bound: one pass over the key and value cache (HBM, or L2 for a layer stepped in a loop); for a few
// sequences the chain of dependent latencies in front of and behind that pass.  So a warp works alone:
// it owns units of 32 keys, brings their key and value rows in by TMA (one box each, 128-byte swizzle,
// a ring of three halves, two for the compressed key cache), multiplies on mma.sync (m16n8k16) straight from the swizzled rows and keeps
// its own running softmax; warps meet once, at the end.  Staging by per-thread cp.async instead of TMA
// was bound by the SM's load path at half the rate (batch 16, 2048 keys: 18.9 us per step, TMA 12.2).
// With the copies ahead of their use, a unit's time is its instructions (two CTAs per SM: 3060 clocks a
// round, now 2030; 64 MB from L2 in 5 us are 1560): copies are issued under a predicate, not in one lane's branch;
// values come by ldmatrix.trans instead of 32 byte permutations; the row scale moves only past 2^8; the unit of the
// new row comes by TMA like any other (row by row it made its warp the last of every step by 0.8 us).
// G <= 8 query rows against the cache are no shape for a 128-row tcgen05 tile, whose operands,
// commits and tensor-memory reads put four hand-overs between a key tile and its softmax; the score
// product here fills 16 rows with the G references and the G queries, so that one thread receives both
// scores of a (head, key) pair in registers.
//   scores  A = [references; queries] (16 x D), B = 8 keys: the contraction index may be permuted
//           freely as long as both operands agree, so a thread takes 16-byte pieces of its key's row;
//   P.V     A = P with the score accumulator's layout, B = 16 keys x 8 channels: one ldmatrix.trans
//           brings a unit's four 8-key tiles of 8 channels (keys in the order of A's columns).
//           P keeps fp32 precision as a sum of three bf16 parts: rows 0-7 of A carry the first part,
//           rows 8-15 the second (the same thread holds both), the third goes to rows G .. 2G-1,
//           whose lanes duplicate the scores of rows 0 .. G-1 (G <= 4), or to a second product (G = 8).
// The row that arrives with the step is scored from k_new and v_new, written over its row of the unit (zeros
// behind it: what the caches hold there is anything), and joins the caches through the warp that owns its unit.
// The slices of a (batch, KV head) are one thread-block cluster: a CTA's warps meet in its shared memory, and one
// record per block of 16 channels goes to the CTA that finishes the block with st.async, which counts its
// bytes on the receiver's barrier (every warp sending for itself: 0.4 us more, the packets queue at the
// receivers; a merge through global memory 2 us more; a cluster barrier with release semantics waits 0.7 us for
// the step's global stores).
// Measured, us per step of a loop of steps, before -> after the changes above: Llama layer at 2048 keys, batch 1
// 4.4 -> 4.1 (the caller's host time; 3.3 on the device), batch 16 12.2 -> 9.3 (7.6 TB/s from L2); batch 8 at 4096 keys
// 11.6 -> 9.5; BitNet layer (d = 128) at 1531 keys, batch 2 6.1 -> 5.0; key deltas, batch 4 at 1777 keys 6.4 -> 5.0;
// compressed key cache, batch 4 at 1024 keys 8.0 -> 7.2.
// Tried and dropped: the next unit's scores issued under a unit's softmax and P.V (twice the code, spills: batch 16
// 10.3); three slots without the rest (nothing: no warp was waiting for its copies).
#include <cuda.h>

#include "decode_common.cuh"
#include "decode_merge.cuh"
#include "tc_common.cuh"

namespace delta {

namespace {

template <int D> constexpr int kWarps = D == 64 ? 8 : 4;    // warps per CTA
constexpr float RESCALE_LOG2 = 8.0f;

struct MmaDecodeParams {
  const __nv_bfloat16 *q_new, *k_new, *v_new;
  __nv_bfloat16 *k_cache, *v_cache, *khat_cache, *out;
  uint16_t* row_nnz;
  // the compressed key-delta cache (MODE 2)
  uint32_t *mask, *kp_mask, *seg_off, *used;
  uint16_t *kp_nnz, *vals, *base;
  size_t cap;
  int nseg_max;
  const float* ref_in;
  float *ref_out, *R, *partial;
  uint32_t* ticket;
  unsigned long long* counters;
  int n, T_max, H, chunk, nsplit, W, b0;
  int early;                              // reference keys may be fetched ahead of the wait (see there)
  float theta, scale_log2e;
  int ragged;
  int n_b[kRaggedMax];                    // ragged: tokens seen per batch element b0 ..
};

__device__ __forceinline__ void sts128z(uint32_t dst) {
  asm volatile("st.shared.v4.u32 [%0], {%1, %1, %1, %1};" ::"r"(dst), "r"(0) : "memory");
}
__device__ __forceinline__ void mma16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
               "{%0, %1, %2, %3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// (the accumulators start at zero)
__device__ __forceinline__ void mma16816_first(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                               uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
               "{%10, %10, %10, %10};"
               : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
               : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.0f));
}
// four 8 x 8 tiles, transposed: lane l gives the address of row l % 8 of tile l / 8
__device__ __forceinline__ void ldsm4t(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 t = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&t);
}
// (lo, hi) as three bf16 pairs whose sum is (lo, hi) to fp32 precision
__device__ __forceinline__ void split3(float lo, float hi, uint32_t& p0, uint32_t& p1, uint32_t& p2) {
  p0 = pack_bf16(lo, hi);
  const float r0 = lo - __uint_as_float(p0 << 16), r1 = hi - __uint_as_float(p0 & 0xffff0000u);
  p1 = pack_bf16(r0, r1);
  p2 = pack_bf16(r0 - __uint_as_float(p1 << 16), r1 - __uint_as_float(p1 & 0xffff0000u));
}
__device__ __forceinline__ uint32_t lds_u32(uint32_t a) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ uint32_t lds_u16(uint32_t a) {
  uint32_t v;
  asm volatile("ld.shared.u16 %0, [%1];" : "=r"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ void sts_u4(uint32_t a, uint4 v) {
  asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ void lds_words(uint32_t a, uint32_t (&w)[2]) {
  asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(w[0]), "=r"(w[1]) : "r"(a));
}
__device__ __forceinline__ void lds_words(uint32_t a, uint32_t (&w)[4]) {
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]) : "r"(a));
}
__device__ __forceinline__ void sts_u32(uint32_t a, uint32_t v) { asm volatile("st.shared.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory"); }
// N consecutive elements, as fp32, past the L1 cache
template <int N> __device__ __forceinline__ void load_bf16(const __nv_bfloat16* p, float (&x)[N]) {
  static_assert(N == 1 || N == 2 || N == 4 || N == 8, "");
  uint32_t w[N == 1 ? 1 : N / 2];
  if constexpr (N == 1) w[0] = __ldcg(reinterpret_cast<const unsigned short*>(p));
  else if constexpr (N == 2) w[0] = __ldcg(reinterpret_cast<const uint32_t*>(p));
  else if constexpr (N == 4) { const uint2 u = __ldcg(reinterpret_cast<const uint2*>(p)); w[0] = u.x; w[1] = u.y; }
  else { const uint4 u = __ldcg(reinterpret_cast<const uint4*>(p)); w[0] = u.x; w[1] = u.y; w[2] = u.z; w[3] = u.w; }
#pragma unroll
  for (int i = 0; i < N; ++i) x[i] = __uint_as_float((i & 1) ? w[i >> 1] & 0xffff0000u : w[i >> 1] << 16);
}
template <int N> __device__ __forceinline__ void load_f32(const float* p, float (&x)[N]) {
  if constexpr (N == 1) x[0] = __ldcg(p);
  else if constexpr (N == 2) { const float2 u = __ldcg(reinterpret_cast<const float2*>(p)); x[0] = u.x; x[1] = u.y; }
  else
#pragma unroll
    for (int i = 0; i < N; i += 4) {
      const float4 u = __ldcg(reinterpret_cast<const float4*>(p + i));
      x[i] = u.x; x[i + 1] = u.y; x[i + 2] = u.z; x[i + 3] = u.w;
    }
}
// Shared memory: per warp a ring of NS halves of units (the keys, or the values, of one unit: 128-byte
// swizzle, blocks of [32 rows][64 channels]), whose first slot takes the warp's result in the end, then the merge's records.
// PACKED: per warp also the encoding of one 32-row segment: values, mask words, the reference in front;
// and a table of its rows (rebuild below).
template <int D, int G, bool PACKED> struct MmaSmem {
  static constexpr int NW = kWarps<D>;
  static constexpr uint32_t VALS = UK * D * 2 + 16, MASKS = UK * (D / 32) * 4, ROWS = UK * 16, PACK = PACKED ? VALS + MASKS + D * 2 + ROWS : 0;
  static constexpr uint32_t HALF = UK * D * 2;             // keys, or values, of a unit
  static constexpr int NS = PACKED ? 2 : 3;                // (two CTAs per SM: 2 x 113 KB)
  static constexpr uint32_t RING = NW * NS * HALF;
  static constexpr int NB = G * D / 16;                    // 16-channel blocks of the result
  static_assert(MergePart<D, G>::BYTES <= HALF, "a warp's result fits its first slot");
  // records of a CTA of a cluster of cs
  __host__ __device__ static constexpr uint32_t rec_bytes(int cs) { return merge_slots<D, G>(cs) * cs * REC2 * 4; }
  static constexpr uint32_t NEW = 2 * D * 2;               // the key and value row that arrive with the step
  static constexpr size_t bytes(int cs) { return 1024 + RING + rec_bytes(cs) + NW * PACK + NEW; }
  static constexpr size_t bytes_max = 1024 + RING + (NB + kMaxCluster - 1) * REC2 * 4 + NW * PACK + NEW;
};

}  // namespace

// MODE 0: query deltas; 1: key deltas, dense reference-key rows; 2: key deltas from the compressed
// key-delta cache (k1_pack_keys.cu has its layout): a unit is one segment of the
// encoding, whose rows the warp rebuilds into its key slot.
template <int D, int G, int MODE, bool CLUSTER, bool LATE>
__global__ void __launch_bounds__(32 * kWarps<D>, 2)
decode_step_mma_kernel(const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
                       const __grid_constant__ CUtensorMap tm_h, const __grid_constant__ MmaDecodeParams p) {
  using TC = __nv_bfloat16;
  constexpr bool KEY = MODE != 0, PACKED = MODE == 2;
  using SM = MmaSmem<D, G, PACKED>;
  constexpr int MNW = kWarps<D>;
  constexpr int NC = D / 32;                 // 16-byte pieces of a key row per thread
  constexpr int NV = D / 64;                 // 64-channel blocks of a row
  constexpr int NT8 = D / 8;                 // n-tiles of P.V
  extern __shared__ unsigned char dsm_raw[];
  __shared__ __align__(8) unsigned long long bars[SM::NS * MNW + 1];
  __shared__ int s_last, s_fail;
  const uint32_t ring = (smem_u32(dsm_raw) + 1023u) & ~1023u;
  const uint32_t recs = ring + SM::RING, packs = recs + SM::rec_bytes(CLUSTER ? p.nsplit : 1);

  // (the warp index by shuffle: known to be the same in every lane, so that addresses of copies stay in uniform registers)
  const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const uint32_t lead = lane == 0;
  const int g = lane >> 2, t = lane & 3;     // row of the accumulators, thread of the row
  const int hd = g % G, part = g / G;        // the head this thread's row stands for; which part of P it feeds
  const int split = blockIdx.x, bkv = p.b0 * (p.H / G) + blockIdx.y;
  const int H_kv = p.H / G;
  const int b = bkv / H_kv, kvh = bkv - b * H_kv;
  const int n = p.ragged ? p.n_b[b - p.b0] : p.n, T_max = p.T_max, W = p.W;
  const int L = n + 1;
  const int j0 = split * p.chunk, j1 = min(j0 + p.chunk, L);
  const float theta = p.theta;

  // the merge: blocks of 16 channels of one head; slice r of the cluster finishes blocks r, r + cs, ..
  // (a CTA without a cluster all of them), each from the records of every slice
  const int cs = CLUSTER ? p.nsplit : 1, rank = CLUSTER ? split : 0;
  const uint32_t bar_m = smem_u32(&bars[SM::NS * MNW]);
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

  const size_t row0 = (size_t)bkv * T_max;
  const TC* const kc = p.k_cache + row0 * D;
  const TC* const vc = p.v_cache + row0 * D;
  const TC* const hc = MODE == 1 ? p.khat_cache + row0 * D : nullptr;
  const TC* const kn = p.k_new + (size_t)bkv * D;
  const TC* const vn = p.v_new + (size_t)bkv * D;
  const int wl = n - W + 1;                  // first key inside the decode window

  // ---- the warp's ring: halves K, V, K, V, .. of its units in turn, half h in slot h mod NS.  Row r,
  // 16-byte chunk c of a 64-channel block lies at r * 128 + ((c ^ (r & 7)) << 4): what TMA's 128-byte
  // swizzle writes.
  constexpr int NS = SM::NS;
  const uint32_t slots = ring + (uint32_t)warp * NS * SM::HALF;
  const uint32_t bars0 = smem_u32(&bars[NS * warp]);
  if (lane == 0) {
    if (warp == 0) {
      // (a copy that has to fetch its tensor map first takes 0.25 us longer)
      asm volatile("prefetch.tensormap [%0];" ::"l"(&tm_k) : "memory");
      asm volatile("prefetch.tensormap [%0];" ::"l"(&tm_v) : "memory");
      if (MODE == 1) asm volatile("prefetch.tensormap [%0];" ::"l"(&tm_h) : "memory");
    }
#pragma unroll
    for (int i = 0; i < NS; ++i) tc::mbar_init(bars0 + 8 * i, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    tc::fence_proxy_async();
  }
  if (tid == 0) s_fail = 0;
  __syncwarp();
  // A unit whose rows come from one cache goes by TMA, the unit of the row that arrives with the step
  // too (rows behind the cached ones hold anything: that row and zeros are written over them); key
  // deltas: the unit of the window's edge row by row.
  auto k_plain = [&](int jg) { return !KEY || jg + UK <= wl || jg >= wl; };
  const uint32_t pack_s = packs + (uint32_t)warp * SM::PACK;       // values, mask words, base
  const uint32_t* const so = PACKED ? p.seg_off + (size_t)bkv * (p.nseg_max + 1) : nullptr;
  auto from_pack = [&](int jg) { return PACKED && jg < wl && jg < n; };          // some row is a cached reference row
  auto row_at = [&](uint32_t slot, int r, int ch) {          // 16-byte piece ch of row r
    return slot + (ch >> 3) * UK * 128 + r * 128 + (((ch & 7) ^ (r & 7)) << 4);
  };
  auto fetch_k = [&](int jg, int slot) {
    const uint32_t bar_k = bars0 + 8 * slot, slot_k = slots + slot * SM::HALF;
    if (from_pack(jg)) {
      // (the entry behind the last cached segment is being rewritten by this step's owner where the new
      // row extends or follows that segment: old and new value both bound the cached values)
      if (lane == 0) {
        const int sg = jg / UK;
        // (the bounds hold for any encoding a prefill and at most T_max - T steps behind it have built; a
        // captured step that is replayed appends its row again and again)
        const uint32_t v0 = min(__ldcg(so + sg), (uint32_t)p.cap - D) & ~7u, v1 = __ldcg(so + sg + 1);
        const uint32_t vb = min(min((v1 - v0 + 7u) & ~7u, (uint32_t)UK * D), (uint32_t)p.cap - v0) * 2u;
        tc::mbar_expect_tx(bar_k, vb + SM::MASKS + D * 2);
        if (vb) bulk_load(pack_s, p.vals + (size_t)bkv * p.cap + v0, vb, bar_k);
        bulk_load(pack_s + SM::VALS, p.kp_mask + ((size_t)bkv * p.nseg_max * UK + jg) * (D / 32), SM::MASKS, bar_k);
        bulk_load(pack_s + SM::VALS + SM::MASKS, p.base + ((size_t)bkv * p.nseg_max + sg) * D, D * 2, bar_k);
      }
      // rows of a mixed unit that are not cached references: original keys, the new one, zeros
#pragma unroll 1
      for (int e = min(UK, min(n, wl) - jg) * (D / 8) + lane; e < UK * (D / 8); e += 32) {
        const int r = e / (D / 8), ch = e % (D / 8), j = jg + r;
        const uint32_t dst = row_at(slot_k, r, ch);
        if (j <= n) async16(dst, (j < n ? kc + (size_t)j * D : kn) + 8 * ch);
        else sts128z(dst);
      }
    } else if (k_plain(jg)) {
      tc::mbar_expect_tx_if(lead, bar_k, SM::HALF);
      const CUtensorMap* tm = (MODE == 1 && jg < wl) ? &tm_h : &tm_k;
#pragma unroll
      for (int c = 0; c < NV; ++c) tc::tma_load_3d_if(lead, slot_k + c * UK * 128, tm, bar_k, 64 * c, jg, bkv);
    } else {
#pragma unroll
      for (int c = 0; c < NV; ++c)
#pragma unroll
        for (int i = 0; i < UK / 4; ++i) {
          const int r = 4 * i + (lane >> 3), ch = lane & 7, j = jg + r;
          const uint32_t dst = slot_k + c * UK * 128 + r * 128 + ((ch ^ (r & 7)) << 4);
          const TC* src = (MODE == 1 && j < wl) ? hc : kc;
          if (j <= n) async16(dst, (j < n ? src + (size_t)j * D : kn) + 64 * c + 8 * ch);
          else sts128z(dst);
        }
    }
  };
  auto fetch_v = [&](int jg, int slot) {
    const uint32_t bar_v = bars0 + 8 * slot, slot_v = slots + slot * SM::HALF;
    tc::mbar_expect_tx_if(lead, bar_v, SM::HALF);
#pragma unroll
    for (int c = 0; c < NV; ++c) tc::tma_load_3d_if(lead, slot_v + c * UK * 128, &tm_v, bar_v, 64 * c, jg, bkv);
  };
  // Rows jg .. jg + 31 of the reference-key stream from their encoding, into the key slot: lane = two
  // channels (of a 64-channel block), walking the rows; the window's rows and the new one are keys.
  // Issue-bound, so what a row needs is laid out first, lane = row: for either half of the block's channels where the
  // row's values of that half start and its mask word.  (Every lane counting for itself, and a row's loads behind the
  // store of the one before: 147 clocks per row, a unit 2.5 us.)
  auto rebuild = [&](int jg, uint32_t slot_k) {
    constexpr int NWD = D / 32;
    const int last = min(UK, min(n, wl) - jg);             // rows that are cached references
    const int hi = lane >> 4, sh = 2 * (lane & 15);        // this lane's channels: bits sh, sh + 1 of word 2 c + hi
    const uint32_t lt = (1u << sh) - 1u;
    const uint32_t table = pack_s + SM::VALS + SM::MASKS + D * 2;
    uint32_t w[NWD], total = 0;
    lds_words(pack_s + SM::VALS + 4 * NWD * lane, w);
#pragma unroll
    for (int k = 0; k < NWD; ++k) total += __popc(w[k]);
    uint32_t at = total;                                   // values up to this row, then in front of it
#pragma unroll
    for (int x = 1; x < 32; x <<= 1) {
      const uint32_t up = __shfl_up_sync(0xffffffffu, at, x);
      at += lane >= x ? up : 0u;
    }
    at = pack_s + 2 * (at - total);
#pragma unroll
    for (int c = 0; c < NV; ++c) {
      const uint32_t at1 = at + 2 * __popc(w[2 * c]);
      sts_u4(table + 16 * lane, make_uint4(at, w[2 * c], at1, w[2 * c + 1]));
      at = at1 + 2 * __popc(w[2 * c + 1]);
      __syncwarp();
      uint32_t cur = lds_u32(pack_s + SM::VALS + SM::MASKS + 128 * c + 4 * lane);
      const uint32_t dst = slot_k + c * UK * 128 + 4 * (lane & 3);
#pragma unroll 1
      for (int r0 = 0; r0 < last; r0 += 8) {
        uint32_t f[8], a[8], x0[8], x1[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          uint32_t e[2];
          lds_words(table + 16 * (r0 + i) + 8 * hi, e);
          a[i] = e[0] + 2 * __popc(e[1] & lt);
          f[i] = e[1] >> sh;
        }
        // (a channel that has not fired reads some value of the pool and drops it: no branch)
#pragma unroll
        for (int i = 0; i < 8; ++i) { x0[i] = lds_u16(a[i]); x1[i] = lds_u16(a[i] + 2 * (f[i] & 1u)); }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int r = r0 + i;
          cur = (f[i] & 1u) ? __byte_perm(cur, x0[i], 0x3254) : cur;
          cur = (f[i] & 2u) ? __byte_perm(cur, x1[i], 0x5410) : cur;
          if (r < last) sts_u32(dst + r * 128 + (((lane >> 2) ^ (r & 7)) << 4), cur);
        }
      }
      __syncwarp();
    }
    async_wait_all();                                      // the rows that are not cached references (fetch_k)
    __syncwarp();
  };
  // the warp that owns the row arriving with the step, and that row in shared memory (keys, values)
  const bool has_new = j1 == L && j0 < L && ((n - j0) / UK) % MNW == warp;
  const uint32_t new_s = packs + MNW * SM::PACK;
  // Reference-key rows and their encoding are the library's own: behind another step (p.early) all but the
  // row (segment) that step may be writing is final before this kernel can start, since a step releases
  // the next one only behind its own wait, and is requested ahead of the wait.  Not so behind a prefill:
  // its last kernel (the packing kernel least of all) releases nothing itself, and what it writes is
  // certain to be seen only behind the wait.  (Key and value rows are the caller's.)
  int jg = j0 + UK * warp;
  const bool early_k = KEY && p.early && jg < j1 && jg + UK <= min(n - 1, wl);
  if (early_k) fetch_k(jg, 0);
  // The first unit's rows from such an encoding are rebuilt ahead of the wait too, under the end of the step in front.
  bool built = early_k && from_pack(jg), late = false;
  if (built) {
    late = !mbar_wait(bars0, 0);
    rebuild(jg, slots);
  }
  // the step in front (or the prefill) has written the reference, row n - 1 of the caches, the tickets
  asm volatile("griddepcontrol.wait;" ::: "memory");
  // The next step's CTAs may become resident from here on, LATE: from the merge on.  (Released at the kernel's start
  // they take the places of this step's own late CTAs: 30 us per step for 18 at batch 16.)
  if constexpr (!LATE) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  // ---- threshold step (Eq. 2-3), a few elements per thread; the references meet in shared memory, from
  // where every warp takes its operand rows (each warp on its own: 150 instructions more per warp, 0.2 us
  // alone and 0.4 us where two CTAs share an SM)
  const bool keep = split == 0 && warp == 0;
  constexpr int NTH = 32 * MNW, NE = KEY ? D : G * D, EPT = NE <= NTH ? 1 : NE / NTH;
  constexpr uint32_t REF_LD = 2 * D + (KEY ? 0 : 64);       // bytes (the 64: rows on different banks)
  __shared__ __align__(16) unsigned char s_ref[(KEY ? 1 : G) * REF_LD];
  __shared__ int s_fired[MNW];               // fired elements of every warp
  __shared__ uint32_t s_word[NC];            // KEY: mask words of the new key
  const uint32_t refs = smem_u32(s_ref);
  uint32_t ar[NC][4], aq[NC][4];             // rows g and g + 8 of A, channels 32 c + 8 t ..
  {
    const size_t o0 = ((size_t)b * p.H + kvh * G) * D;
    const int e0 = tid * EPT;
    const bool mine = NE >= NTH || e0 < NE;
    float x[EPT], ref[EPT];
    if (mine) {
      load_bf16(KEY ? kn + e0 : p.q_new + o0 + e0, x);
      load_f32(p.ref_in + (KEY ? (size_t)bkv * D : o0) + e0, ref);
    }
    uint4 q4[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) q4[c] = __ldcg(reinterpret_cast<const uint4*>(p.q_new + o0 + hd * D + 32 * c + 8 * t));
    // (behind those loads: they are what the warp waits for next; the values, needed last, behind their arrival: a
    // unit's rows of every warp at once take the SM half a microsecond, which the loads would wait for)
    if (jg < j1 && !early_k) fetch_k(jg, 0);
    if (has_new) {
#pragma unroll
      for (int e = 0; e < 2 * (D / 8); e += 32)
        if (e + lane < 2 * (D / 8)) {
          const int ch = (e + lane) % (D / 8);
          async16(new_s + 16 * (e + lane), (e + lane < D / 8 ? kn : vn) + 8 * ch);
        }
    }
    if (mine) asm volatile("" : "+f"(x[0]), "+f"(ref[0])::"memory");          // (they have arrived)
    if (jg < j1) {
      fetch_v(jg, 1);
      if (NS == 3 && jg + UK * MNW < j1) fetch_k(jg + UK * MNW, 2);
    }
    int fired = 0;
    if (mine) {
#pragma unroll
      for (int i = 0; i < EPT; ++i) {
        const bool fire = fabsf(__fsub_rn(x[i], ref[i])) > theta;
        ref[i] = fire ? x[i] : ref[i];
        fired += fire ? 1 : 0;
      }
      // exactly bf16: copies of input elements (or the zero the reference starts from)
      unsigned char* const at = s_ref + (KEY ? 0 : e0 / D) * REF_LD + 2 * (KEY ? e0 : e0 % D);
      if constexpr (EPT == 1) *reinterpret_cast<uint16_t*>(at) = (uint16_t)(__float_as_uint(ref[0]) >> 16);
      else
#pragma unroll
        for (int i = 0; i < EPT; i += 2)
          *reinterpret_cast<uint32_t*>(at + 2 * i) = __byte_perm(__float_as_uint(ref[i]), __float_as_uint(ref[i + 1]), 0x7632);
      if (split == 0) {
        float* const rq = p.ref_out + (KEY ? (size_t)bkv * D : o0) + e0;
#pragma unroll
        for (int i = 0; i < EPT; ++i) rq[i] = ref[i];
      }
    }
    if constexpr (KEY) {                     // (a thread, an element: a warp's vote is a mask word)
      const uint32_t word = __ballot_sync(0xffffffffu, fired != 0);
      if (lane == 0) { s_fired[warp] = __popc(word); if (warp < NC) s_word[warp] = word; }
    } else {
      fired = __reduce_add_sync(0xffffffffu, fired);
      if (lane == 0) s_fired[warp] = fired;
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const uint4 r4 = KEY ? q4[c] : tc::lds128u(refs + hd * REF_LD + 64 * c + 16 * t);
      ar[c][0] = r4.x; ar[c][1] = r4.y; ar[c][2] = r4.z; ar[c][3] = r4.w;
      aq[c][0] = KEY ? 0u : q4[c].x; aq[c][1] = KEY ? 0u : q4[c].y; aq[c][2] = KEY ? 0u : q4[c].z; aq[c][3] = KEY ? 0u : q4[c].w;
    }
  }

  // ---- the warp's units
  float o_acc[NT8][4];
#pragma unroll
  for (int i = 0; i < NT8; ++i)
#pragma unroll
    for (int e = 0; e < 4; ++e) o_acc[i][e] = 0.0f;
  float m = -INFINITY, l = 0.0f;
  unsigned done = 0;
  uint32_t phases = built ? 1u : 0u;         // of the slots' barriers, a bit each
  if (late) s_fail = 1;
  int sk = 0, sv = 1;                        // the slots of the unit's keys and values
  // Column x of a score block stands for key x ^ (4 (x & 1)) of its 8 keys: with the swizzle, the
  // eight lanes of a shared-memory phase then touch eight different chunks, for keys and values alike.
  const int kx0 = 2 * t, kx1 = (2 * t + 1) ^ 4;            // this thread's two keys of a block
  const int kr = g ^ (4 * (g & 1));                        // the key row it reads
  const uint32_t k_off = kr * 128, k_sw = kr & 7;
  // lane l gives row l % 8 of 8-key block l / 8, read as the column it stands for; chunk c of it lies at
  // v_off ^ (c << 4)
  const int vr_ = (lane & 7) ^ (4 * (lane & 1));
  const uint32_t v_off = (lane >> 3) * 1024 + vr_ * 128 + (vr_ << 4);
  float* const Rg = KEY ? nullptr : p.R + ((size_t)b * p.H + kvh * G + hd) * T_max;
  // The new row joins the encoding (the warp that owns its unit): values behind the pool's end (on a
  // multiple of 8 where it opens a segment), mask words, count, offsets, the segment's base.
  auto append = [&](int nz) {
    const int sg = n / UK;
    const bool opens = (n % UK) == 0;
    const uint32_t pool = __ldcg(p.used + bkv), pos = min(opens ? (pool + 7u) & ~7u : pool, (uint32_t)p.cap - D);
    uint16_t* const vg = p.vals + (size_t)bkv * p.cap;
    uint32_t at = pos;
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const uint32_t word = s_word[c], byte = (word >> (8 * t)) & 0xffu;
      const uint4 kh4 = tc::lds128u(refs + 64 * c + 16 * t);
      const uint32_t kh[4] = {kh4.x, kh4.y, kh4.z, kh4.w};
      if (g == 0) {
        uint32_t rank = at + __popc(word & ((1u << (8 * t)) - 1u));
#pragma unroll
        for (int e = 0; e < 8; ++e)
          if ((byte >> e) & 1u) {
            // (a fired channel's new reference is the key value itself)
            if (DELTA_IN(rank, p.cap, p.counters)) vg[rank] = (uint16_t)(kh[e >> 1] >> (16 * (e & 1)));
            ++rank;
          }
        if (t == 0) {
          p.mask[(row0 + n) * NC + c] = word;
          p.kp_mask[((size_t)bkv * p.nseg_max * UK + n) * NC + c] = word;
        }
        if (opens) {
          const float4* const rp = reinterpret_cast<const float4*>(p.ref_in + (size_t)bkv * D + 32 * c + 8 * t);
          const float4 r0 = __ldcg(rp), r1 = __ldcg(rp + 1);
          const float rr[8] = {r0.x, r0.y, r0.z, r0.w, r1.x, r1.y, r1.z, r1.w};
#pragma unroll
          for (int e = 0; e < 8; ++e)                     // exactly bf16
            p.base[((size_t)bkv * p.nseg_max + sg) * D + 32 * c + 8 * t + e] = (uint16_t)(__float_as_uint(rr[e]) >> 16);
        }
      }
      at += __popc(word);
    }
    if (lane == 0 && DELTA_IN(sg + 1, p.nseg_max + 1, p.counters)) {
      uint32_t* const sw = p.seg_off + (size_t)bkv * (p.nseg_max + 1);
      if (opens) sw[sg] = pos;
      sw[sg + 1] = pos + (uint32_t)nz;
      p.used[bkv] = pos + (uint32_t)nz;
      p.kp_nnz[(size_t)bkv * p.nseg_max * UK + n] = (uint16_t)nz;
    }
  };
  // What a unit leaves behind its products is stored when the next unit, or the merge, is under way.
  float s[4][4];
  int j_done = -1;                           // the unit whose scores s holds
  unsigned nz = 0;                           // KEY: its multiply-adds per query, of key j_done + lane
  bool owns_new = false;                     // the warp owns the row that arrives with the step
  auto store_r = [&]() {
    if (!KEY && part == 0 && j_done >= 0) {  // R[j] = q_hat . k_j
      float *const ra = Rg + j_done + kx0, *const rb = Rg + j_done + kx1;
      if (!owns_new) {
#pragma unroll
        for (int h = 0; h < 4; ++h)
          if (DELTA_IN(j_done + 8 * h + 7, T_max, p.counters)) { ra[8 * h] = s[h][0]; rb[8 * h] = s[h][1]; }
      } else {
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          if (j_done + 8 * h + kx0 <= n) ra[8 * h] = s[h][0];
          if (j_done + 8 * h + kx1 <= n) rb[8 * h] = s[h][1];
        }
      }
    }
  };
  for (; jg < j1; jg += UK * MNW) {
    const int jn = jg + UK * MNW;            // the warp's next unit
    const uint32_t bar_k = bars0 + 8 * sk, bar_v = bars0 + 8 * sv, slot_k = slots + sk * SM::HALF, slot_v = slots + sv * SM::HALF;
    store_r();
    done += nz;
    const bool owner = n < jg + UK;          // of the row that arrives with the step
    const bool packed = from_pack(jg), tma_k = !packed && k_plain(jg);
    if (packed) {
      if (!built) {
        if (!mbar_wait(bar_k, (phases >> sk) & 1u)) s_fail = 1;
        phases ^= 1u << sk;
        rebuild(jg, slot_k);
      }
      built = false;
    } else if (tma_k) {
      if (!mbar_wait(bar_k, (phases >> sk) & 1u)) s_fail = 1;
      phases ^= 1u << sk;
      if (owner) {                           // the new key's row (what the rows behind it hold is masked)
        async_wait_all();
        __syncwarp();
        if (lane < D / 8) {
          const uint4 x = tc::lds128u(new_s + 16 * lane);
          sts_u4(row_at(slot_k, n - jg, lane), x);
        }
        __syncwarp();
      }
    } else {
      async_wait_all();
      __syncwarp();
    }
#pragma unroll
    for (int h = 0; h < 4; ++h) {
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        // channels 32 c + 8 t .. of the row: chunk 4 (c & 1) + t of block c >> 1
        uint4 k4 = tc::lds128u(slot_k + k_off + (c >> 1) * UK * 128 + h * 1024 + (((4 * (c & 1) + t) ^ k_sw) << 4));
        if (KEY && W <= 0 && jg + 8 * h + kr == n)         // no window: even the new key goes by its reference
          k4 = tc::lds128u(refs + 64 * c + 16 * t);
        if (c == 0) mma16816_first(s[h], ar[c][0], aq[c][0], ar[c][1], aq[c][1], k4.x, k4.y);
        else mma16816(s[h], ar[c][0], aq[c][0], ar[c][1], aq[c][1], k4.x, k4.y);
        mma16816(s[h], ar[c][2], aq[c][2], ar[c][3], aq[c][3], k4.z, k4.w);
      }
    }
    j_done = jg;
    owns_new = owner;
    if (KEY) {
      // multiply-adds: d inside the window, nnz(Delta k_j) outside (added when the load is back)
      const int j = jg + lane;
      nz = (j > n || j >= j1) ? 0u : (n - j < W) ? (unsigned)D : j == n ? 0u : (unsigned)p.row_nnz[row0 + j];
      if (!tma_k) tc::fence_proxy_async();                 // rows written by the warp, TMA overwrites them
    }
    __syncwarp();                            // every key of the unit has been used
    if (jn < j1) {
      if (NS == 3) fetch_v(jn, sk); else fetch_k(jn, sk);
    }

    // hybrid select, running maximum of the row (4 threads hold it); the scale joins the exponential
    float v[8];
#pragma unroll
    for (int h = 0; h < 4; ++h) { v[2 * h] = s[h][0]; v[2 * h + 1] = s[h][1]; }
    if (!KEY && jg + UK > wl) {
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        if (jg + 8 * h + kx0 >= wl) v[2 * h] = s[h][2];
        if (jg + 8 * h + kx1 >= wl) v[2 * h + 1] = s[h][3];
      }
    }
    if (owner) {
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        if (jg + 8 * h + kx0 > n) v[2 * h] = -INFINITY;
        if (jg + 8 * h + kx1 > n) v[2 * h + 1] = -INFINITY;
      }
    }
    // The row's scale moves only when a score is more than 2^RESCALE_LOG2 above it (a warp's first unit: any
    // is), so the four threads of a row compare notes in few units; P and its parts are as exact at any scale.
    float mx = tc::fmax3(fmaxf(v[0], v[1]), tc::fmax3(v[2], v[3], v[4]), tc::fmax3(v[5], v[6], v[7])) * p.scale_log2e;
    if (__any_sync(0xffffffffu, mx > m + RESCALE_LOG2)) {
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
      const float mn = fmaxf(m, mx), al = tc::ex2(m - mn);
      m = mn;
      l *= al;
#pragma unroll
      for (int i = 0; i < NT8; ++i)
#pragma unroll
        for (int e = 0; e < 4; ++e) o_acc[i][e] *= al;
    }
    float pr[8];
    uint32_t pa[2][4], p2[2][2];
#pragma unroll
    for (int e = 0; e < 8; ++e) pr[e] = tc::ex2(fmaf(v[e], p.scale_log2e, -m));
    l += ((pr[0] + pr[1]) + (pr[2] + pr[3])) + ((pr[4] + pr[5]) + (pr[6] + pr[7]));
    if (!mbar_wait(bar_v, (phases >> sv) & 1u)) s_fail = 1;
    phases ^= 1u << sv;
    if (owner) {                             // the new value's row, zeros behind it
      const int rn = n - jg;
      async_wait_all();
      __syncwarp();
      if (lane < D / 8) {
        const uint4 x = tc::lds128u(new_s + D * 2 + 16 * lane);
        sts_u4(row_at(slot_v, rn, lane), x);
      }
#pragma unroll 1
      for (int e = (rn + 1) * (D / 8) + lane; e < UK * (D / 8); e += 32) sts128z(row_at(slot_v, e / (D / 8), e % (D / 8)));
      __syncwarp();
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {            // 16 keys per product
      uint32_t f0, f1, f2, g0, g1, g2;
      split3(pr[4 * q], pr[4 * q + 1], f0, f1, f2);
      split3(pr[4 * q + 2], pr[4 * q + 3], g0, g1, g2);
      uint32_t a0 = f0, a1 = f1, a2 = g0, a3 = g1;
      if (G <= 4) {
        a0 = part == 0 ? f0 : part == 1 ? f2 : 0u; a1 = part == 0 ? f1 : 0u;
        a2 = part == 0 ? g0 : part == 1 ? g2 : 0u; a3 = part == 0 ? g1 : 0u;
      }
      pa[q][0] = a0; pa[q][1] = a1; pa[q][2] = a2; pa[q][3] = a3;
      if (G == 8) { p2[q][0] = f2; p2[q][1] = g2; }
    }
#pragma unroll
    for (int c = 0; c < NT8; ++c) {          // 8 channels: B tiles of the unit's four 8-key blocks
      uint32_t vb[4];
      ldsm4t(slot_v + (v_off ^ ((c & 7) << 4)) + (c >> 3) * UK * 128, vb);
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        mma16816(o_acc[c], pa[q][0], pa[q][1], pa[q][2], pa[q][3], vb[2 * q], vb[2 * q + 1]);
        if (G == 8) mma16816(o_acc[c], p2[q][0], 0u, p2[q][1], 0u, vb[2 * q], vb[2 * q + 1]);
      }
    }
    __syncwarp();
    if (NS == 2) {
      if (jn < j1) fetch_v(jn, sv);
    } else {
      // two halves on, modulo three
      if (jn + UK * MNW < j1) fetch_k(jn + UK * MNW, sv);
      const int s0 = sk;
      sk = sv == 2 ? 0 : sv + 1;
      sv = s0;
    }
  }

  // ---- the warp's result: the parts of P meet again, the row sum over the row's four threads
  l += __shfl_xor_sync(0xffffffffu, l, 1);
  l += __shfl_xor_sync(0xffffffffu, l, 2);
#pragma unroll
  for (int i = 0; i < NT8; ++i) {
    o_acc[i][0] += o_acc[i][2];
    o_acc[i][1] += o_acc[i][3];
    if (G <= 4) {
      o_acc[i][0] += __shfl_down_sync(0xffffffffu, o_acc[i][0], 4 * G);
      o_acc[i][1] += __shfl_down_sync(0xffffffffu, o_acc[i][1], 4 * G);
    }
  }
  if constexpr (LATE) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  // ---- merge: the warp's part into its first slot (every copy into it is complete and read)
  if (part == 0) {
    using MP = MergePart<D, G>;
#pragma unroll
    for (int i = 0; i < NT8; ++i) sts_f2(slots + (hd * MP::LD + 8 * i + 2 * t) * 4, o_acc[i][0], o_acc[i][1]);
    if (t == 0) sts_f2(slots + MP::ML + hd * 8, m, l);
  }
  __syncthreads();
  if (CLUSTER) asm volatile("barrier.cluster.wait.aligned;" ::: "memory");          // every slice runs
  const size_t out0 = ((size_t)b * p.H + kvh * G) * D;
  const int n_slices = (L + p.chunk - 1) / p.chunk;
  merge_warps<TC, D, G, MNW, CLUSTER>(ring, NS * SM::HALF, recs, bar_m, rank, cs, n_slices, split, bkv, out0, p.partial, p.out);
  // ---- while the parts travel: the last unit's score row, the caches' new row, the counters
  store_r();
  int f_all = 0;
  if (keep || (KEY && owns_new)) {
#pragma unroll
    for (int w = 0; w < MNW; ++w) f_all += s_fired[w];
  }
  if (owns_new && DELTA_IN(n, T_max, p.counters)) {
    // the row that arrives with the step joins the caches
    if (lane < D / 8) {
      reinterpret_cast<uint4*>(p.k_cache + (row0 + n) * D)[lane] = tc::lds128u(new_s + 16 * lane);
      reinterpret_cast<uint4*>(p.v_cache + (row0 + n) * D)[lane] = tc::lds128u(new_s + D * 2 + 16 * lane);
    }
    if (KEY && lane == 0) p.row_nnz[row0 + n] = (uint16_t)f_all;
    if constexpr (PACKED) append(f_all);
    if (MODE == 1 && g == 0)
#pragma unroll
      for (int c = 0; c < NC; ++c)
        *reinterpret_cast<uint4*>(p.khat_cache + (row0 + n) * D + 32 * c + 8 * t) = tc::lds128u(refs + 64 * c + 16 * t);
  }
  if (keep && lane == 0) {
    const int n_in = min(L, max(W, 0));
    atomicAdd(&p.counters[CNT_DECODE_NNZ], (unsigned long long)f_all);
    atomicAdd(&p.counters[CNT_DECODE_ELEMS], (unsigned long long)(KEY ? D : G * D));
    atomicAdd(&p.counters[CNT_DECODE_MACS_DENSE], (unsigned long long)L * D * G);
    if (!KEY)
      atomicAdd(&p.counters[CNT_DECODE_MACS_DONE],
                (unsigned long long)n_in * D * G + (unsigned long long)(L - n_in) * f_all);
  }
  if (KEY) {
    // (the new key: inside any window of at least one key, else its own count)
    const unsigned d = __reduce_add_sync(0xffffffffu, done + nz) + (owns_new && W <= 0 ? (unsigned)f_all : 0u);
    if (lane == 0 && d) atomicAdd(&p.counters[CNT_DECODE_MACS_DONE], (unsigned long long)d * G);
  }
  if (CLUSTER) {
    // (every slice's block records: also what keeps this CTA until the last of them has been sent to it)
    bool ok;
    if constexpr (KEY) ok = merge_slices_in_turn<TC, D, G>(recs, bar_m, rank, cs, out0, p.out);
    else ok = merge_slices<TC, D, G, MNW>(recs, bar_m, rank, cs, out0, p.out);
    if (!ok) s_fail = 1;
  } else if (n_slices > 1) {
    merge_global<TC, D, G, MNW>(n_slices, bkv, out0, p.partial, p.ticket, p.out, &s_last);
  }
  if (s_fail && lane == 0) atomicMax(&p.counters[CNT_STATUS], (unsigned long long)DELTA_ERR_TIMEOUT);
}

template <int D, int G, int MODE, bool CLUSTER, bool LATE>
static cudaError_t launch_mma(const CUtensorMap& tk, const CUtensorMap& tv, const CUtensorMap& th,
                              const MmaDecodeParams& p, int bkv, cudaStream_t st) {
  auto kern = decode_step_mma_kernel<D, G, MODE, CLUSTER, LATE>;
  using SM = MmaSmem<D, G, MODE == 2>;
  const size_t smem = SM::bytes(CLUSTER ? p.nsplit : 1);
  static std::atomic<uint64_t> ready{0};
  if (!device_done(ready)) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SM::bytes_max);
    // (two CTAs per SM need the largest shared-memory carve-out)
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                                                   (int)cudaSharedmemCarveoutMaxShared);
    if (e == cudaSuccess && CLUSTER) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    device_mark(ready);
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)p.nsplit, (unsigned)bkv);
  cfg.blockDim = dim3(32 * kWarps<D>);
  cfg.dynamicSmemBytes = smem;
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
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, tk, tv, th, p);
  count_launch();
  return e;
}

// The tensor map of a [B * H_kv, T_max, d] bf16 cache (box: UK rows of 64 channels), encoded once
// per cache pointer.
static const CUtensorMap* row_map(DecodeTmapCache* cache, const void* ptr, const Shape& s) {
  static_assert(sizeof(CUtensorMap) <= sizeof(cache->map), "tensor-map cache");
  CUtensorMap* m = reinterpret_cast<CUtensorMap*>(cache->map);
  if (cache->ptr != ptr) {
    if (!tc::encode3(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, ptr, (uint64_t)s.d, (uint64_t)s.T_max, (uint64_t)s.B * s.H_kv,
                     (uint64_t)s.d * 2, (uint64_t)s.T_max * s.d * 2, 64, UK, CU_TENSOR_MAP_SWIZZLE_128B))
      return nullptr;
    cache->ptr = ptr;
  }
  return m;
}

bool decode_mma_applies(const Shape& s, int dtype) { return dtype == DELTA_BF16 && (s.d == 64 || s.d == 128); }

cudaError_t launch_decode_step_mma(const Shape& s, const Workspace& w, const void* q_new, const void* k_new,
                                   const void* v_new, void* k_cache, void* v_cache, void* out, int n, const int* n_b,
                                   float theta, int window, int qhat_sel, bool key, bool packed, bool behind_step,
                                   DecodeTmapCache* maps, cudaStream_t st) {
  if ((key && !w.qhat_rows) || (packed && (!key || !w.kp_vals))) return cudaErrorNotSupported;
  using TC = __nv_bfloat16;
  const CUtensorMap* const tk = row_map(&maps[0], k_cache, s);
  const CUtensorMap* const tv = row_map(&maps[1], v_cache, s);
  const CUtensorMap* const th = key ? row_map(&maps[2], w.qhat_rows, s) : tk;
  if (!tk || !tv || !th) return cudaErrorInvalidValue;
  MmaDecodeParams p;
  p.q_new = (const TC*)q_new; p.k_new = (const TC*)k_new; p.v_new = (const TC*)v_new;
  p.k_cache = (TC*)k_cache; p.v_cache = (TC*)v_cache; p.khat_cache = w.qhat_rows; p.out = (TC*)out;
  p.row_nnz = w.row_nnz; p.ref_in = w.qhat[qhat_sel]; p.ref_out = w.qhat[qhat_sel ^ 1]; p.R = w.R;
  p.partial = w.dec_partial; p.ticket = w.dec_ticket; p.counters = w.counters;
  p.n = n; p.T_max = s.T_max; p.H = s.H; p.W = window; p.theta = theta;
  p.scale_log2e = 1.4426950408889634f / sqrtf((float)s.d);
  p.mask = w.mask; p.kp_mask = w.kp_mask; p.seg_off = w.kp_segoff; p.used = w.kp_used;
  p.kp_nnz = w.kp_nnz; p.vals = w.kp_vals; p.base = w.kp_base;
  p.cap = keypack_capacity(s.T_max, s.d); p.nseg_max = keypack_segments(s.T_max);
  p.ragged = n_b != nullptr;
  p.early = behind_step ? 1 : 0;
  p.b0 = 0;
  const int G = s.g();
  bool cluster;
  decode_slices(s, n + 1, s.d == 64 ? kWarps<64> : kWarps<128>, s.d == 64 ? 1.25f : 1.35f, s.d == 64 ? 0.83f : 0.87f,
                packed ? 1.6f : 0.0f, &p.nsplit, &p.chunk, &cluster);
  if (p.nsplit > kMaxDecodeSplits) return cudaErrorInvalidValue;
  // When the next step's CTAs may come (query deltas): from the merge on where two CTAs share an SM (from 1.6 per SM on) and,
  // d = 128, where a warp has two units at most; else behind the wait.  us per step, behind the wait | at the merge: 16 x 32 heads
  // at 2048 keys 9.48, 9.27; 8 x 32 at 4096 9.56, 9.41; 30 x 8 at 700 7.34, 7.05; d = 128, 20 heads, batch 1 at 1000 3.98, 3.90, 2 at
  // 1531 4.78, 4.70, 8 at 2000 7.56, 7.44; but 2 x 8 at 3500 7.67, 7.76; d = 64, batch 2 at 2048 4.71, 4.88.  Key deltas fetch ahead
  // of the wait and want their place early: batch 4 at 1777 keys 5.17, 5.46.
  const bool late = (long)s.B * s.H_kv * p.nsplit * 10 > 16l * device_sm_count() ||
                    (s.d == 128 && p.chunk <= 2 * UK * kWarps<128>);
  cudaError_t err = cudaSuccess;
  for (; p.b0 < s.B && err == cudaSuccess; p.b0 += kRaggedMax) {
    const int nb = n_b ? (s.B - p.b0 < kRaggedMax ? s.B - p.b0 : kRaggedMax) : s.B;
    if (n_b)
      for (int i = 0; i < nb; ++i) p.n_b[i] = n_b[p.b0 + i];
#define GO_M(DD, GG, M, L)                                                                                   \
    err = cluster ? launch_mma<DD, GG, M, true, L>(*tk, *tv, *th, p, nb * s.H_kv, st)                        \
                  : launch_mma<DD, GG, M, false, L>(*tk, *tv, *th, p, nb * s.H_kv, st)
#define GO(DD, GG)                                                                                           \
    if (packed) { GO_M(DD, GG, 2, false); }                                                                  \
    else if (key) { GO_M(DD, GG, 1, false); }                                                                \
    else if (late) { GO_M(DD, GG, 0, true); }                                                                \
    else { GO_M(DD, GG, 0, false); }
#define GO_G(DD)                                                                                             \
    switch (G) {                                                                                             \
      case 1: GO(DD, 1); break;                                                                              \
      case 2: GO(DD, 2); break;                                                                              \
      case 4: GO(DD, 4); break;                                                                              \
      case 8: GO(DD, 8); break;                                                                              \
      default: return cudaErrorInvalidValue;                                                                 \
    }
    if (s.d == 64) { GO_G(64) } else { GO_G(128) }
#undef GO_G
#undef GO
#undef GO_M
    if (!n_b) break;
  }
  return err;
}

}  // namespace delta
