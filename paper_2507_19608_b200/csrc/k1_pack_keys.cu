// Compressed key-delta cache (key deltas) -- Section III-A "Decoding Stage Considerations" and
// Section III-C: what decoding keeps of the keys is the delta stream, not the keys.
//
// Encoding.  Per KV head the thresholded key stream (Eq. 2-3) is kept as
//   mask    one bit per (row, channel): the element fired                     d / 8 bytes per row
//   values  for every fired element the key value that became the reference (= reference before
//           + Delta k; bf16, so the reference rows it reproduces are exact), row after row,
//           channels ascending                                                2 nnz(row) bytes
//   base    the reference key in front of every 32-row segment                2 d bytes per 32 rows
//   offset  position of every segment's first value in the pool (segments start on multiples of
//           8 values so that a segment's values are one 16-byte aligned bulk copy)
// At the delta sparsity the method reaches (about 0.6) that is roughly 46 % of the bytes of the
// dense reference-key rows.  The last W_d original keys are read from the key cache rows inside the
// decode window.
//
// pack_keys_kernel builds the encoding behind a prefill (from the mask words and counts the finish
// kernel wrote, the keys and the reference-key rows); the decode step (k3_decode_step_mma.cu, MODE 2)
// rebuilds a segment's rows in shared memory and appends the new row.
//
// Bound: a few MB of reads and writes.  One CTA per eight segments of a KV head (a warp each); every
// CTA derives the segment offsets from the row counts itself, a scan over T / 32 sums, which costs
// less than a launch of its own.  (One CTA per KV head took 46 us for 32 heads of 1024 keys, this 10.)
#include "delta_internal.cuh"

namespace delta {

namespace {
constexpr int SEG = 32;     // rows per segment of the encoding
constexpr int PNW = 8;      // warps per CTA, a segment each
__host__ __device__ inline uint32_t round8(uint32_t x) { return (x + 7u) & ~7u; }
}  // namespace

template <int D>
__global__ void __launch_bounds__(32 * PNW) pack_keys_kernel(
    const __nv_bfloat16* __restrict__ k, const __nv_bfloat16* __restrict__ khat_rows,
    const uint32_t* __restrict__ mask, const uint16_t* __restrict__ row_nnz, uint16_t* __restrict__ vals,
    uint32_t* __restrict__ seg_off, uint16_t* __restrict__ base, uint32_t* __restrict__ used,
    uint32_t* __restrict__ kp_mask, uint16_t* __restrict__ kp_nnz, int T, int T_max, size_t cap, int nseg_max,
    unsigned long long* __restrict__ counters) {
  constexpr int NW = D / 32;
  extern __shared__ uint32_t s_off[];          // [nseg + 1] first value of every segment; [nseg]: the pool's end
  const int bkv = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nseg = (T + SEG - 1) / SEG;
  const uint16_t* const nz = row_nnz + (size_t)bkv * T_max;
  for (int s = warp; s < nseg; s += PNW) {
    uint32_t x = (s * SEG + lane < T) ? nz[s * SEG + lane] : 0u;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if (lane == 0) s_off[s + 1] = x;
  }
  __syncthreads();
  if (warp == 0) {
    // running sum of the segments, each padded to 8 values; the last one leaves its exact end
    uint32_t run = 0;
    for (int s0 = 0; s0 < nseg; s0 += 32) {
      const int s = s0 + lane;
      uint32_t x = s < nseg ? (s + 1 < nseg ? round8(s_off[s + 1]) : s_off[s + 1]) : 0u;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
      }
      if (s < nseg) s_off[s + 1] = run + x;
      run += __shfl_sync(0xffffffffu, x, 31);
    }
    if (lane == 0) s_off[0] = 0;
  }
  __syncthreads();
  if (blockIdx.x == 0) {
    uint32_t* const so = seg_off + (size_t)bkv * (nseg_max + 1);
    for (int s = tid; s <= nseg; s += 32 * PNW) so[s] = s_off[s];
    if (tid == 0) used[bkv] = s_off[nseg];
  }
  const int s = blockIdx.x * PNW + warp;
  if (s >= nseg) return;
  const uint16_t* const kp = reinterpret_cast<const uint16_t*>(k) + (size_t)bkv * T_max * D;
  const uint32_t* const mk = mask + (size_t)bkv * T_max * NW;
  uint16_t* const vp = vals + (size_t)bkv * cap;
  const int row = s * SEG + lane, rows = min(SEG, T - s * SEG);
  // the encoding's own copy of mask words and counts (its stride is a multiple of 32 rows: every
  // segment starts on a 16-byte boundary); lane = row
  uint32_t mine[NW];
#pragma unroll
  for (int w = 0; w < NW; ++w) mine[w] = lane < rows ? mk[(size_t)row * NW + w] : 0u;
  if (lane < rows) {
#pragma unroll
    for (int w = 0; w < NW; ++w) kp_mask[((size_t)bkv * nseg_max * SEG + row) * NW + w] = mine[w];
    kp_nnz[(size_t)bkv * nseg_max * SEG + row] = nz[row];
  }
  // reference in front of the segment
  for (int c = lane; c < D; c += 32)
    base[((size_t)bkv * nseg_max + s) * D + c] =
        (s == 0) ? (uint16_t)0
                 : reinterpret_cast<const uint16_t*>(khat_rows)[((size_t)bkv * T_max + s * SEG - 1) * D + c];
  uint32_t off = s_off[s];
  constexpr int RB = 16 / NW * 2;              // rows whose loads are in flight together
  for (int r0 = 0; r0 < rows; r0 += RB) {
    uint16_t x[RB][NW];
#pragma unroll
    for (int r = 0; r < RB; ++r)
#pragma unroll
      for (int w = 0; w < NW; ++w)
        x[r][w] = kp[(size_t)(s * SEG + min(r0 + r, rows - 1)) * D + w * 32 + lane];
#pragma unroll
    for (int r = 0; r < RB; ++r)
#pragma unroll
      for (int w = 0; w < NW; ++w) {
        const uint32_t word = __shfl_sync(0xffffffffu, mine[w], r0 + r);       // (0 behind the last row)
        const uint32_t at = off + __popc(word & ((1u << lane) - 1u));
        if (((word >> lane) & 1u) && DELTA_IN(at, cap, counters)) vp[at] = x[r][w];
        off += __popc(word);
      }
  }
}

// Pool capacity per KV head, in values: every element fired, plus the padding of the segments.
size_t keypack_capacity(int T_max, int d) { return (size_t)T_max * d + 8u * ((size_t)T_max / SEG + 2); }
int keypack_segments(int T_max) { return (T_max + SEG - 1) / SEG; }

cudaError_t launch_pack_keys(const Shape& s, const Workspace& w, const void* k, int T, cudaStream_t st) {
  if (!w.kp_vals || !w.qhat_rows || (s.d != 64 && s.d != 128)) return cudaErrorNotSupported;
  const int nseg_max = keypack_segments(s.T_max), nseg = (T + SEG - 1) / SEG;
  const size_t smem = ((size_t)nseg + 1) * 4;
  const dim3 grid((unsigned)((nseg + PNW - 1) / PNW), (unsigned)(s.B * s.H_kv));
  auto kern = s.d == 64 ? pack_keys_kernel<64> : pack_keys_kernel<128>;
  kern<<<grid, 32 * PNW, smem, st>>>((const __nv_bfloat16*)k, w.qhat_rows, w.mask, w.row_nnz, w.kp_vals, w.kp_segoff,
                                     w.kp_base, w.kp_used, w.kp_mask, w.kp_nnz, T, s.T_max, keypack_capacity(s.T_max, s.d),
                                     nseg_max, w.counters);
  count_launch();
  return cudaGetLastError();
}

}  // namespace delta
