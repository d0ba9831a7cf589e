// K1b -- what is parallel over rows behind the delta chain (Eq. 2-3 re-run per 8-row block, Eq. 6, the hand-off row): device
// code shared by the finish kernel (k1_delta_construct.cu, which describes it) and by attention launches that do its work
// beside their own.
#pragma once
#include "delta_internal.cuh"

namespace delta {

namespace {
__device__ __forceinline__ float2 load_pair(const float* p) { return *reinterpret_cast<const float2*>(p); }
__device__ __forceinline__ float2 load_pair(const __nv_bfloat16* p) {
  const uint32_t u = *reinterpret_cast<const uint32_t*>(p);
  return make_float2(__uint_as_float(u << 16), __uint_as_float(u & 0xffff0000u));
}
__device__ __forceinline__ void load_eight(const float* p, float (&x)[8]) {
  const float4 a = *reinterpret_cast<const float4*>(p), b = *reinterpret_cast<const float4*>(p + 4);
  x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w; x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
}
__device__ __forceinline__ void load_eight(const __nv_bfloat16* p, float (&x)[8]) {
  const uint4 u = *reinterpret_cast<const uint4*>(p);
  const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    x[2 * i] = __uint_as_float(w[i] << 16);
    x[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
  }
}
// bit i of the low half to bit 2i
__device__ __forceinline__ uint32_t spread16(uint32_t x) {
  x &= 0xffffu;
  x = (x | (x << 8)) & 0x00ff00ffu;
  x = (x | (x << 4)) & 0x0f0f0f0fu;
  x = (x | (x << 2)) & 0x33333333u;
  return (x | (x << 1)) & 0x55555555u;
}

// Eq. 2-3 over the 8 rows of a block from its checkpoint (ck): delta values (dqp), reference rows (refp,
// key deltas), fired channels ascending (srow, 8 x D bytes in shared memory, 0xFF where none), and in
// lanes r and r + 8, .. the mask words of row r.  Lane = channels 2 lane, 2 lane + 1 of 64 at a time.
// REV: strategy (2), rows from the top.  FULL: the block has all 8 rows and no un-thresholded basis row.
template <typename TIn, int D, bool REV, bool FULL>
__device__ __forceinline__ void finish_rows(const TIn* __restrict__ q, const float* __restrict__ ck, float* __restrict__ dqp,
                                            __nv_bfloat16* __restrict__ refp, uint8_t* srow, int rbase, int T, float theta,
                                            int basis_exact, uint32_t (&mw)[D / 32]) {
  const int lane = threadIdx.x & 31;
  const uint32_t lt = (1u << lane) - 1u;
  int before[8];                                   // fired channels of the row in front of these 64
#pragma unroll
  for (int rr = 0; rr < 8; ++rr) before[rr] = 0;
#pragma unroll
  for (int c2 = 0; c2 < D / 64; ++c2) {
    const int c = 64 * c2 + 2 * lane;
    float2 ref = __ldcg(reinterpret_cast<const float2*>(ck + c));
    const TIn* const qp = q + (size_t)rbase * D + c;
    float2 v[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) v[r] = (FULL || rbase + r < T) ? load_pair(qp + r * D) : make_float2(0.0f, 0.0f);
    uint32_t even = 0, odd = 0;                    // of the lane's row
#pragma unroll
    for (int rr = 0; rr < 8; ++rr) {
      const int r = REV ? 7 - rr : rr;
      const bool live = FULL || rbase + r < T;
      const bool basis = !FULL && basis_exact && rbase + r == (REV ? T - 1 : 0);
      const float d0 = basis ? v[r].x : __fsub_rn(v[r].x, ref.x), d1 = basis ? v[r].y : __fsub_rn(v[r].y, ref.y);
      const bool f0 = live && (basis || fabsf(d0) > theta), f1 = live && (basis || fabsf(d1) > theta);
      ref.x = f0 ? v[r].x : ref.x;
      ref.y = f1 ? v[r].y : ref.y;
      if (live) {
        *reinterpret_cast<float2*>(dqp + r * D + c) = make_float2(f0 ? d0 : 0.0f, f1 ? d1 : 0.0f);
        if (refp)                                  // exactly bf16
          *reinterpret_cast<uint32_t*>(refp + r * D + c) = __byte_perm(__float_as_uint(ref.x), __float_as_uint(ref.y), 0x7632);
      }
      const uint32_t be = __ballot_sync(0xffffffffu, f0), bo = __ballot_sync(0xffffffffu, f1);
      uint8_t* const at = srow + r * D + before[r] + __popc(be & lt) + __popc(bo & lt);
      if (f0) at[0] = (uint8_t)c;
      if (f1) at[f0 ? 1 : 0] = (uint8_t)(c + 1);
      if (c2 + 1 < D / 64) before[r] += __popc(be) + __popc(bo);
      if ((lane & 7) == r) { even = be; odd = bo; }
    }
    mw[2 * c2] = spread16(even) | (spread16(odd) << 1);
    mw[2 * c2 + 1] = spread16(even >> 16) | (spread16(odd >> 16) << 1);
  }
}
// Shared memory of a block (16-byte aligned): counts, then the compacted indices or the heads' references.
template <int D, int NWARP> constexpr int kFinishSmem = 128 + 8 * D * (NWARP > 4 ? NWARP : 4);
// Block `block` of the pass over a sequence (sq), by the first NWARP warps of a CTA that has no others left: index
// blocks first, then key blocks (see the roles at the kernel).
// x: the stream the chain kernel ran over (see there); ref_rows (key deltas): the reference after
// every row, the cache of reference keys.  heads: heads of the delta stream per batch element;
// seq_heads, seq_kv: heads of the stream, KV heads that one entry of seqs stands for.
template <typename TIn, int D, int NWARP>
__device__ __forceinline__ void finish_block(
    const Seq& sq, int block, unsigned char* smem,
    uint32_t* __restrict__ mask, uint16_t* __restrict__ row_nnz, uint32_t* __restrict__ tile_nnz, uint8_t* __restrict__ idx,
    unsigned long long* __restrict__ counters, const TIn* __restrict__ k, const float* __restrict__ qhat, float* __restrict__ R,
    int T_max, int n_tiles, int heads, int seq_heads, int seq_kv, int H, int g, int shape, int key_stream,
    const TIn* __restrict__ x, float* __restrict__ dq, __nv_bfloat16* __restrict__ ref_rows, const float* __restrict__ ckpt,
    int n_ckpt, float theta, int basis_exact, int reverse) {
  constexpr int NW = D / 32;
  const int T = sq.T, W = sq.W;
  [[maybe_unused]] const int src_rows = key_stream ? T_max : T;
  const int tiles_used = (T + DELTA_TILE_ROWS - 1) / DELTA_TILE_ROWS, n_idx_blocks = seq_heads * tiles_used;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (block < n_idx_blocks) {
    // ---- one block per (batch, head, 64-row tile); warp w serves rows 8w .. 8w+7, and those NWARP warps further on
    uint32_t(*const s_red)[8] = reinterpret_cast<uint32_t(*)[8]>(smem);      // [3][8]
    const int hl = block / tiles_used, tile = block - hl * tiles_used;
    const int bh = sq.b * heads + hl;                // head of the workspace arrays
    const TIn* const q = key_stream ? x + (size_t)bh * T_max * D : x + sq.q_off + (size_t)hl * T * D;
    const int t0 = tile * DELTA_TILE_ROWS;
    const int rows = min(DELTA_TILE_ROWS, T - t0);
    // The chain kernel left only the reference in front of every 8-row block.  The warp re-runs
    // Eq. 2-3 over its 8 rows, lane = two neighbouring channels, 64 channels at a time: delta values
    // (a row leaves as one 256-byte store), reference rows (key deltas), two ballots per row (even and
    // odd channels), the rank of every fired channel in its row.
    uint8_t* const srow = smem + 128 + warp * 8 * D;
#pragma unroll 1
    for (int wb = warp; wb < 8; wb += NWARP) {
      const int r_mine = wb * 8 + (lane & 7);          // lanes 0..7 hold one row each
      const int rbase = t0 + wb * 8, my_rows = min(8, rows - wb * 8);
      uint32_t mw[NW];
#pragma unroll
      for (int w2 = 0; w2 < NW; ++w2) mw[w2] = 0u;
      if (rbase < T && DELTA_IN(rbase / DELTA_CKPT_ROWS, n_ckpt, counters) &&
          DELTA_IN(rbase + 7 < T ? rbase + 7 : T - 1, src_rows, counters) && DELTA_IN(T - 1, T_max, counters)) {
#pragma unroll
        for (int e = lane; e < 8 * D / 16; e += 32)
          reinterpret_cast<uint4*>(srow)[e] = make_uint4(0xffffffffu, 0xffffffffu, 0xffffffffu, 0xffffffffu);
        __syncwarp();
        const bool plain = rbase + 8 <= T && !(basis_exact && (reverse ? rbase + 8 == T : rbase == 0));
#define ROWS(REV, FULL)                                                                                          \
    finish_rows<TIn, D, REV, FULL>(q, ckpt + ((size_t)bh * n_ckpt + rbase / DELTA_CKPT_ROWS) * D,                  \
                                   dq + ((size_t)bh * T_max + rbase) * D,                                          \
                                   ref_rows ? ref_rows + ((size_t)bh * T_max + rbase) * D : nullptr, srow, rbase, T, theta, \
                                   basis_exact, mw)
        if (reverse) { if (plain) ROWS(true, true); else ROWS(true, false); }
        else { if (plain) ROWS(false, true); else ROWS(false, false); }
#undef ROWS
      }
      if (lane < 8 && r_mine < rows) {
        uint32_t* const mp = mask + ((size_t)bh * T_max + t0 + r_mine) * NW;
        if constexpr (NW == 2) *reinterpret_cast<uint2*>(mp) = make_uint2(mw[0], mw[1]);
        else *reinterpret_cast<uint4*>(mp) = make_uint4(mw[0], mw[1], mw[2], mw[3]);
      }
      // Eq. 6 (32 bits hold a warp's eight rows: 8 x 65536 keys x 128 channels x 8 heads)
      uint32_t done = 0, dense = 0, tsum = 0;
      if (lane < 8 && r_mine < rows && DELTA_IN(t0 + r_mine, T_max, counters)) {
        uint32_t nnz = 0;
#pragma unroll
        for (int w2 = 0; w2 < NW; ++w2) nnz += __popc(mw[w2]);
        row_nnz[(size_t)bh * T_max + t0 + r_mine] = (uint16_t)nnz;
        tsum = nnz;
        const int i = t0 + r_mine;
        if (!key_stream) {
          // query deltas: row i meets i + 1 keys, nnz multiply-adds per out-of-window key
          const uint32_t n_in = (uint32_t)in_window_count(i, W, shape);
          done = n_in * D + ((uint32_t)(i + 1) - n_in) * nnz;
          dense = (uint32_t)(i + 1) * D;
        } else {
          // key deltas: key i meets the T - i queries behind it, for each of the g query heads
          const uint32_t n_q = (uint32_t)(T - i), n_in = (uint32_t)in_window_col_count(i, T, W, shape);
          done = (uint32_t)g * (n_in * D + (n_q - n_in) * nnz);
          dense = (uint32_t)g * n_q * D;
        }
      }
      tsum = __reduce_add_sync(0xffffffffu, tsum);
      done = __reduce_add_sync(0xffffffffu, done);
      dense = __reduce_add_sync(0xffffffffu, dense);
      if (lane == 0) { s_red[0][wb] = tsum; s_red[1][wb] = done; s_red[2][wb] = dense; }
      // the compacted indices leave as 16-byte stores (8 consecutive rows are contiguous)
      __syncwarp();
      {
        uint4* dst = reinterpret_cast<uint4*>(idx + ((size_t)bh * T_max + t0 + wb * 8) * D);
        const uint4* src = reinterpret_cast<const uint4*>(srow);
        for (int e = lane; e < my_rows * D / 16; e += 32) dst[e] = src[e];
      }
      if (NWARP < 8) __syncwarp();                     // (the next rows take the same place)
    }
    __syncthreads();
    if (tid == 0) {
      unsigned long long a = 0, b2 = 0, c2 = 0;
      for (int w2 = 0; w2 < 8; ++w2) { a += s_red[0][w2]; b2 += s_red[1][w2]; c2 += s_red[2][w2]; }
      if (DELTA_IN(tile, n_tiles, counters)) tile_nnz[(size_t)bh * n_tiles + tile] = (uint32_t)a;
      unsigned long long* cs = counters + CNT_SHARD_BASE + 4 * (block % CNT_SHARDS);
      atomicAdd(&cs[0], a);
      atomicAdd(&cs[1], (unsigned long long)rows * D);
      atomicAdd(&cs[2], b2);
      atomicAdd(&cs[3], c2);
    }
    return;
  }

  // ---- key pass: 64 keys of one (batch, KV head): R(T-1)[j] = q_hat(T-1).k_j, D / 8 lanes per key
  float(*const qh)[D] = reinterpret_cast<float(*)[D]>(smem + 128);           // [8][D]
  const int kblocks = (T + 63) / 64;
  const int item = block - n_idx_blocks, kv_l = item / kblocks, j0 = (item - kv_l * kblocks) * 64;
  if (key_stream || kv_l >= seq_kv) return;          // (a shorter sequence of a ragged group)
  const int H_kv = H / g, bkv = sq.b * H_kv + kv_l;
  const int b = bkv / H_kv, kvh = bkv - b * H_kv;
  for (int e = tid; e < g * D; e += 32 * NWARP) qh[e / D][e % D] = __ldcg(&qhat[((size_t)b * H + kvh * g) * D + e]);
  __syncthreads();
  constexpr int LPK = D / 8, KPW = 32 / LPK;         // lanes per key, keys per warp and pass
  const int sub = lane / LPK, c0 = (lane % LPK) * 8;
#pragma unroll 1
  for (int wb = warp; wb < 8; wb += NWARP)
#pragma unroll
  for (int i = 0; i < 8 / KPW; ++i) {
    const int j = j0 + 8 * wb + i * KPW + sub;
    float kv[8];
    load_eight(k + ((size_t)bkv * T_max + min(j, T - 1)) * D + c0, kv);
    for (int hh = 0; hh < g; ++hh) {
      const float4 a = *reinterpret_cast<const float4*>(&qh[hh][c0]), c = *reinterpret_cast<const float4*>(&qh[hh][c0 + 4]);
      float acc = a.x * kv[0];
      acc = fmaf(a.y, kv[1], acc); acc = fmaf(a.z, kv[2], acc); acc = fmaf(a.w, kv[3], acc);
      acc = fmaf(c.x, kv[4], acc); acc = fmaf(c.y, kv[5], acc); acc = fmaf(c.z, kv[6], acc); acc = fmaf(c.w, kv[7], acc);
#pragma unroll
      for (int o = LPK / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      if (lane % LPK == 0 && j < T && DELTA_IN(j, T_max, counters)) R[((size_t)b * H + kvh * g + hh) * T_max + j] = acc;
    }
  }
}
// The same as arguments of a launch of another kernel, whose last CTAs do it.
template <typename TIn> struct FinishWork {
  int blocks;                                // 0: none
  uint32_t* mask;
  uint16_t* row_nnz;
  uint32_t* tile_nnz;
  uint8_t* idx;
  unsigned long long* counters;
  const TIn* k;
  const float* qhat;
  float* R;
  int T_max, n_tiles, heads, seq_heads, seq_kv, H, g, shape;
  const TIn* x;
  float* dq;
  const float* ckpt;
  int n_ckpt;
  float theta;
  int basis_exact, reverse;
};
// (query deltas, uniform batches)
template <typename TIn>
FinishWork<TIn> finish_work(const Shape& s, const Workspace& w, const void* q, const void* k, int T, float theta, int shape, int init,
                            bool reverse) {
  const int tiles = (T + DELTA_TILE_ROWS - 1) / DELTA_TILE_ROWS;
  return {s.B * (s.H + s.H_kv) * tiles, w.mask, w.row_nnz, w.tile_nnz, w.idx, w.counters, (const TIn*)k, w.qhat[0], w.R, s.T_max,
          s.n_tiles, s.H, s.B * s.H, s.B * s.H_kv, s.H, s.g(), shape, (const TIn*)q, w.dq, w.ckpt, s.n_ckpt(), theta,
          init == DELTA_INIT_BASIS_EXACT ? 1 : 0, reverse ? 1 : 0};
}
// Small calls, which are bound by the caller's time for launches (2.2 us each): one of ctas other CTAs does it beside them
// while all find places at once.  A pass, two launches behind the chain -> one: 1 head x 128 tokens, fp32 12.7 -> 10.5 us, bf16
// 13.1 -> 11.4; 16 heads x 120 13.2 -> 11.9; 32 x 60 13.2 -> 11.6; 8 x 300 15.4 -> 15.2.  Beyond, nothing or worse: 2 x 8 x 150
// (128 CTAs) 13.4, 13.9; 4 x 500 16.7, 16.5; 1 x 600, fp32, d = 128 37.5, 38.0.
inline bool finish_beside(int T, long ctas, int blocks) { return T <= 400 && (ctas + blocks) * 4 <= device_sm_count() * 3l; }
template <typename TIn, int D, int NWARP>
__device__ __forceinline__ void finish_block(const FinishWork<TIn>& f, const Seq& sq, int block, unsigned char* smem) {
  finish_block<TIn, D, NWARP>(sq, block, smem, f.mask, f.row_nnz, f.tile_nnz, f.idx, f.counters, f.k, f.qhat, f.R, f.T_max, f.n_tiles, f.heads,
                              f.seq_heads, f.seq_kv, f.H, f.g, f.shape, 0, f.x, f.dq, nullptr, f.ckpt, f.n_ckpt, f.theta,
                              f.basis_exact, f.reverse);
}
}  // namespace

}  // namespace delta
