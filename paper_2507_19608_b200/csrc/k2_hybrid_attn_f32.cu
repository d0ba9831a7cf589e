// K2 (fp32 arithmetic) -- fused hybrid delta attention in fp32 precision (Section III-B; Eq. 1, 4).
// The production path for fp32 inputs; serves bf16 inputs too.
//
// Eq. 4's running sum telescopes: the sum of all Delta q up to row i is the reference q_hat(i)
// (Eq. 3), so the out-of-window score of pair (i, j) is q_hat(i).k_j.  q_hat's elements are copies of
// input elements, so this form carries fewer roundings than the recursion over rounded differences.
//
// Arithmetic.  An fp32 number is the sum of three bf16 parts (8 bits of mantissa each, the exponent
// range is the same): x = h + m + l.  A product of two takes six tensor-core products, h.h, h.m, m.h,
// h.l, l.h, m.m; the dropped ones are below 2^-24 of it.  h.h has an accumulator of its own and the
// five small ones another, the output of a key tile is summed in fresh accumulators and joins the
// running output by one fp32 multiply-add per element, so no long chain of tensor-core additions
// (which truncate) touches a large value.  The error against exact arithmetic is that of the FP32
// pipes, whose 74 TFLOP/s a fused kernel reaches to a quarter (each 16-byte shared-memory operand feeds
// few multiply-adds): the same kernel on packed fma.rn.f32x2 ran at 20 TFLOP/s, the kernel before it,
// sparse delta sums on the FP32 pipes, at 6.  Relative error against fp64 dense attention at 1000
// tokens: 1.8e-7 (FP32-pipe kernel 3.7e-7).  mma.sync and not tcgen05: accumulators in registers make the
// separate small-product sums and the per-tile fresh output sums free to join in fp32, and no key tile waits
// for a hand-over through tensor memory; whether tcgen05 at the same precision would pay has not been measured.
// Measured, whole prefill, before this kernel, with head after head, with the longest walks first: 24 heads x 1425 tokens
// -, 190, 136 us (46 TFLOP/s); 16 heads x 1000 350, 86, 66; one head x 128 54, 13, 13 (the kernel 42 -> 6).
//
// Bound: mma.sync issue (m16n8k16 every 8 clocks per scheduler) once the chip is full (KS = 1: 60 % of it), the walk of the
// last query tile where it is not.  A CTA of four warps owns 64 / KS query rows of one head and walks
// the 64-key tiles up to the diagonal; KS warps share 16 rows and deal a tile's keys among themselves
// (KS = 1: most work per byte staged; KS = 4: the shortest walk, with four times as many CTAs; the
// launcher weighs them).  Keys and values come from global memory into registers while the tensor
// cores work on the tile before, are split into their parts and stored swizzled for ldmatrix.
// A tile takes Q_hat.K^T where none of its pairs is inside the window, Q.K^T where all causal ones are,
// both where it is mixed.  The reference rows are rebuilt from the 8-row checkpoints of the chain
// kernel (Eq. 2-3 re-run per block), so nothing of the finish kernel is read.
#include <algorithm>

#include "delta_internal.cuh"
#include "k1_finish.cuh"
#include "tc_common.cuh"

namespace delta {

namespace {
constexpr int BN = 64, NT = 128;

// Shared memory: bf16 parts as blocks of [rows][64 channels], 16-byte chunk c of row r at
// r * 128 + ((c ^ (r & 7)) << 4); part-major, channel block inside.  NP parts: 3 (fp32) or 1 (bf16).
template <int D, int KS, int NP> struct F32Smem {
  static constexpr int BM = 64 / KS;
  static constexpr uint32_t QPART = BM * D * 2, KPART = BN * D * 2;
  static constexpr uint32_t OFF_QH = NP * QPART, OFF_K = 2 * NP * QPART, OFF_V = OFF_K + NP * KPART;
  static constexpr uint32_t RAW = BM * (D + 4) * 4;                    // the query rows in fp32, before the first key tile
  static constexpr uint32_t MERGE = (KS - 1) * 16 * (D + 2) * 4 * (4 / KS);
  static constexpr uint32_t END = OFF_V + NP * KPART;
  static constexpr uint32_t bytes = (END - OFF_K > RAW ? END : OFF_K + RAW) + 1024;
  static_assert(MERGE <= END, "the merge buffer fits");
};

__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
  const __nv_bfloat162 t = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&t);
}
// the bf16 parts of (lo, hi), packed
template <int NP> __device__ __forceinline__ void parts_of(float lo, float hi, uint32_t (&p)[NP]) {
  p[0] = pack2(lo, hi);
  if constexpr (NP == 3) {
    const float r0 = lo - __uint_as_float(p[0] << 16), r1 = hi - __uint_as_float(p[0] & 0xffff0000u);
    p[1] = pack2(r0, r1);
    p[2] = pack2(r0 - __uint_as_float(p[1] << 16), r1 - __uint_as_float(p[1] & 0xffff0000u));
  }
}
__device__ __forceinline__ void sts128(uint32_t a, uint32_t x, uint32_t y, uint32_t z, uint32_t w) {
  asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(x), "r"(y), "r"(z), "r"(w) : "memory");
}
// eight consecutive channels (chunk c of row r of a block) into all parts
template <int NP> __device__ __forceinline__ void store_parts(uint32_t block, uint32_t part_stride, int r, int c, const float (&x)[8]) {
  uint32_t w[4][NP];
#pragma unroll
  for (int i = 0; i < 4; ++i) parts_of<NP>(x[2 * i], x[2 * i + 1], w[i]);
  const uint32_t a = block + r * 128 + ((c ^ (r & 7)) << 4);
#pragma unroll
  for (int p = 0; p < NP; ++p) sts128(a + p * part_stride, w[0][p], w[1][p], w[2][p], w[3][p]);
}
__device__ __forceinline__ void load8f(const float* p, float (&x)[8]) {
  const float4 a = __ldg(reinterpret_cast<const float4*>(p)), b = __ldg(reinterpret_cast<const float4*>(p) + 1);
  x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w; x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
}
__device__ __forceinline__ void load8f(const __nv_bfloat16* p, float (&x)[8]) {
  const uint4 u = __ldg(reinterpret_cast<const uint4*>(p));
  const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    x[2 * i] = __uint_as_float(w[i] << 16);
    x[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
  }
}
__device__ __forceinline__ void ldsm4(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldsm4t(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
               "{%0, %1, %2, %3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// big += a.b of the first parts, small += the other products of the parts that count
template <int NA, int NB>
__device__ __forceinline__ void mma_parts(float (&big)[4], float (&small)[4], const uint32_t (&a)[NA][4],
                                          const uint32_t (&b)[NB][4], int half) {
  mma(big, a[0], b[0][2 * half], b[0][2 * half + 1]);
  if constexpr (NB == 3) {
    mma(small, a[0], b[2][2 * half], b[2][2 * half + 1]);
    if constexpr (NA == 3) {
      mma(small, a[1], b[1][2 * half], b[1][2 * half + 1]);
      mma(small, a[2], b[0][2 * half], b[0][2 * half + 1]);
    }
    mma(small, a[0], b[1][2 * half], b[1][2 * half + 1]);
  }
  if constexpr (NA == 3) {
    mma(small, a[1], b[0][2 * half], b[0][2 * half + 1]);
    if constexpr (NB == 1) mma(small, a[2], b[0][2 * half], b[0][2 * half + 1]);
  }
}
// Forms (KS) of the sequences of a ragged group.
struct F32Forms { int ks[kSeqMax]; };
template <typename TIn> struct F32Args {
  const TIn *q, *k, *v;
  TIn* out;
  const float* ckpt;
  unsigned long long* counters;
  int T_max, n_ckpt, H, g, shape;
  float theta;
  int basis_row;
  float scale_log2e;
};

// One query tile (of 64 / KS rows) of one head; tile 0 is the last one of the sequence.
template <typename TIn, int D, int KS>
__device__ __forceinline__ void attn_f32_tile(const F32Args<TIn>& p, const Seq& sq, int tile, int head) {
  const TIn* __restrict__ const q = p.q;
  const TIn* __restrict__ const k = p.k;
  const TIn* __restrict__ const v = p.v;
  TIn* __restrict__ const out = p.out;
  const float* __restrict__ const ckpt = p.ckpt;
  unsigned long long* __restrict__ const counters = p.counters;
  const int T_max = p.T_max, n_ckpt = p.n_ckpt, H = p.H, g = p.g, shape = p.shape, basis_row = p.basis_row;
  const float theta = p.theta, scale_log2e = p.scale_log2e;
  const int T = sq.T, W = sq.W;
  constexpr int NP = sizeof(TIn) == 4 ? 3 : 1;
  using SM = F32Smem<D, KS, NP>;
  constexpr int BM = SM::BM, NB = D / 64;          // NB: 64-channel blocks of a row
  constexpr int NTW = 8 / KS;                      // 8-key blocks of a tile per warp
  constexpr int TASKS = BN * D / 8 / NT;           // 8-channel pieces of a key (value) tile per thread
  extern __shared__ unsigned char smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  float* const rawq = reinterpret_cast<float*>(smem_raw + (base - smem_u32(smem_raw)) + SM::OFF_K);     // [BM][D + 4]

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g8 = lane >> 2, t4 = lane & 3;         // row of the fragments, thread of the row
  const int rg = warp / KS, kg = warp % KS;        // the warp's 16 rows, its share of a tile's keys
  const int qt = (T + BM - 1) / BM - 1 - tile;     // longest walks first
  if (qt < 0) return;                              // (a shorter sequence of a ragged group)
  const int bh = sq.b * H + head, b = bh / H, h = bh - b * H;
  const size_t io = sq.q_off + (size_t)head * T * D;            // the head's rows in q and out
  const size_t bkv = (size_t)b * (H / g) + h / g;
  const int i0 = qt * BM, i1 = min(i0 + BM, T) - 1;
  const TIn* const kp = k + bkv * T_max * D;
  const TIn* const vp = v + bkv * T_max * D;
  const int n_kt = i1 / BN + 1;

  float st[TASKS][8];                              // a tile on its way from global memory
  auto fetch = [&](const TIn* src, int r0) {
#pragma unroll
    for (int i = 0; i < TASKS; ++i) {
      const int e = tid + i * NT, r = r0 + e / (D / 8), c = e % (D / 8);
      if (r < T) load8f(src + (size_t)r * D + 8 * c, st[i]);
      else {
#pragma unroll
        for (int x = 0; x < 8; ++x) st[i][x] = 0.0f;
      }
    }
  };
  auto stage = [&](uint32_t off) {
#pragma unroll
    for (int i = 0; i < TASKS; ++i) {
      const int e = tid + i * NT, r = e / (D / 8), c = e % (D / 8);
      store_parts<NP>(base + off + (c >> 3) * (BN * 128), SM::KPART, r, c & 7, st[i]);
    }
  };
  // ---- query rows: fp32 for the re-run of Eq. 2-3, parts for the products
  for (int e = tid; e < BM * (D / 8); e += NT) {
    const int r = e / (D / 8), c = e % (D / 8);
    float x[8] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
    if (i0 + r < T) load8f(q + io + (size_t)(i0 + r) * D + 8 * c, x);
    store_parts<NP>(base + (c >> 3) * (BM * 128), SM::QPART, r, c & 7, x);
#pragma unroll
    for (int i = 0; i < 8; i += 4)
      *reinterpret_cast<float4*>(rawq + r * (D + 4) + 8 * c + i) = make_float4(x[i], x[i + 1], x[i + 2], x[i + 3]);
  }
  fetch(kp, 0);
  // the chain kernel's checkpoints (programmatic stream serialisation: all above are inputs)
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  __syncthreads();
  // reference rows: Eq. 2-3 over every (channel, 8-row block) from the block's checkpoint
  for (int e = tid; e < (BM / 8) * D; e += NT) {
    const int blk = e / D, c = e - blk * D, r0 = i0 + 8 * blk;
    if (r0 < T && DELTA_IN(r0 / DELTA_CKPT_ROWS, n_ckpt, counters)) {
      float ref = __ldcg(&ckpt[((size_t)bh * n_ckpt + r0 / DELTA_CKPT_ROWS) * D + c]);
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        float* const x = rawq + (8 * blk + r) * (D + 4) + c;
        const bool fire = r0 + r == basis_row || fabsf(__fsub_rn(*x, ref)) > theta;
        ref = fire ? *x : ref;
        *x = ref;                                          // (rows past the end: never stored)
      }
    }
  }
  __syncthreads();
  for (int e = tid; e < BM * (D / 8); e += NT) {
    const int r = e / (D / 8), c = e % (D / 8);
    float x[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = rawq[r * (D + 4) + 8 * c + i];
    store_parts<NP>(base + SM::OFF_QH + (c >> 3) * (BM * 128), SM::QPART, r, c & 7, x);
  }
  __syncthreads();

  float o[NB][8][4];
#pragma unroll
  for (int x = 0; x < NB; ++x)
#pragma unroll
    for (int n = 0; n < 8; ++n)
#pragma unroll
      for (int e = 0; e < 4; ++e) o[x][n][e] = 0.0f;
  float m[2] = {-INFINITY, -INFINITY}, l[2] = {0.0f, 0.0f};              // of rows g8 and g8 + 8
  const int arow = 16 * rg + (lane & 15), achk = lane >> 4;             // ldmatrix rows and chunks of the operands
  const int krow = (64 / KS) * kg + (lane & 7) + ((lane >> 4) << 3), kchk = (lane >> 3) & 1;
  const int vrow = (64 / KS) * kg + (lane & 15), vchk = lane >> 4;
  auto products = [&](uint32_t rows, float (&s)[NTW][4]) {
    float small[NTW][4];
#pragma unroll
    for (int n = 0; n < NTW; ++n)
#pragma unroll
      for (int e = 0; e < 4; ++e) { s[n][e] = 0.0f; small[n][e] = 0.0f; }
#pragma unroll 1
    for (int x = 0; x < NB; ++x)
#pragma unroll
      for (int ks = 0; ks < 4; ++ks) {
        uint32_t a[NP][4];
#pragma unroll
        for (int p = 0; p < NP; ++p)
          ldsm4(rows + p * SM::QPART + x * (BM * 128) + arow * 128 + (((2 * ks + achk) ^ (arow & 7)) << 4), a[p]);
#pragma unroll
        for (int n = 0; n < NTW; n += 2) {
          uint32_t bb[NP][4];
#pragma unroll
          for (int p = 0; p < NP; ++p)
            ldsm4(base + SM::OFF_K + p * SM::KPART + x * (BN * 128) + (krow + 8 * n) * 128 +
                      (((2 * ks + kchk) ^ (krow & 7)) << 4), bb[p]);
          mma_parts<NP, NP>(s[n], small[n], a, bb, 0);
          mma_parts<NP, NP>(s[n + 1], small[n + 1], a, bb, 1);
        }
      }
#pragma unroll
    for (int n = 0; n < NTW; ++n)
#pragma unroll
      for (int e = 0; e < 4; ++e) s[n][e] += small[n][e];
  };
  // keys some row of the tile scores exactly, keys every row does (empty ranges without a window)
  int ex_lo = 1, ex_hi = 0, full_lo = 1, full_hi = 0;
  if (W > 0) {
    if (shape == 0) {
      ex_lo = (i0 / W) * W; ex_hi = (i1 / W) * W + W - 1;
      if (i1 < ex_lo + W) { full_lo = ex_lo; full_hi = ex_lo + W - 1; }
    } else {
      ex_lo = i0 - W + 1; ex_hi = i1; full_lo = i1 - W + 1; full_hi = i1;
    }
  }
  const int ia = i0 + 16 * rg + g8, ib = ia + 8;           // the thread's two rows

  for (int jt = 0; jt < n_kt; ++jt) {
    const int j0 = jt * BN, j1 = min(j0 + BN, i1 + 1) - 1;      // (keys past the last row meet no query)
    const bool some_in = j1 >= ex_lo && j0 <= ex_hi, all_in = j0 >= full_lo && j1 <= full_hi;
    stage(SM::OFF_K);
    fetch(vp, j0);
    __syncthreads();                                       // the keys are staged, the values of the tile before read
    float s[NTW][4];
    products(base + (all_in ? 0u : SM::OFF_QH), s);
    if (some_in && !all_in) {
      float se[NTW][4];
      products(base, se);
#pragma unroll
      for (int e2 = 0; e2 < 2; ++e2) {
        const int i = e2 ? ib : ia;
        int lo, hi;                                        // exact keys of row i: lo <= j < hi
        if (shape == 0) { lo = (i / W) * W; hi = lo + W; } else { lo = i - W + 1; hi = i + 1; }
#pragma unroll
        for (int n = 0; n < NTW; ++n)
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const int j = j0 + (64 / KS) * kg + 8 * n + 2 * t4 + e;
            if (j >= lo && j < hi) s[n][2 * e2 + e] = se[n][2 * e2 + e];
          }
      }
    }
    // ---- scale, causal mask, online softmax (four threads hold a row's scores)
    float al[2];
#pragma unroll
    for (int e2 = 0; e2 < 2; ++e2) {
      const int i = e2 ? ib : ia;
      float mx = -INFINITY;
#pragma unroll
      for (int n = 0; n < NTW; ++n)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          float& x = s[n][2 * e2 + e];
          x = (j0 + (64 / KS) * kg + 8 * n + 2 * t4 + e <= i) ? x * scale_log2e : -INFINITY;
          mx = fmaxf(mx, x);
        }
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
      const float mn = fmaxf(m[e2], mx), sub = mn == -INFINITY ? 0.0f : mn;       // (this warp's keys: maybe none yet)
      al[e2] = exp2f(m[e2] - sub);
      m[e2] = mn;
      float sum = 0.0f;
#pragma unroll
      for (int n = 0; n < NTW; ++n)
#pragma unroll
        for (int e = 0; e < 2; ++e) { float& x = s[n][2 * e2 + e]; x = exp2f(x - sub); sum += x; }
      l[e2] = fmaf(l[e2], al[e2], sum);
    }
    stage(SM::OFF_V);
    if (jt + 1 < n_kt) fetch(kp, j0 + BN);
    __syncthreads();                                       // the values are staged, every warp is done with the keys

    // ---- O = O * alpha + P.V, 64 channels at a time
#pragma unroll
    for (int x = 0; x < NB; ++x) {
      float big[8][4], small[8][4];
#pragma unroll
      for (int n = 0; n < 8; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) { big[n][e] = 0.0f; small[n][e] = 0.0f; }
#pragma unroll
      for (int kk = 0; kk < NTW / 2; ++kk) {
        uint32_t a[3][4];
#pragma unroll
        for (int f = 0; f < 4; ++f) {
          // fragment f: row g8 + 8 (f & 1), keys of block 2 kk + (f >> 1)
          uint32_t w[3];
          parts_of<3>(s[2 * kk + (f >> 1)][2 * (f & 1)], s[2 * kk + (f >> 1)][2 * (f & 1) + 1], w);
          a[0][f] = w[0]; a[1][f] = w[1]; a[2][f] = w[2];
        }
#pragma unroll
        for (int n = 0; n < 8; n += 2) {
          uint32_t bb[NP][4];
#pragma unroll
          for (int p = 0; p < NP; ++p)
            ldsm4t(base + SM::OFF_V + p * SM::KPART + x * (BN * 128) + (vrow + 16 * kk) * 128 +
                       (((n + vchk) ^ (vrow & 7)) << 4), bb[p]);
          mma_parts<3, NP>(big[n], small[n], a, bb, 0);
          mma_parts<3, NP>(big[n + 1], small[n + 1], a, bb, 1);
        }
      }
#pragma unroll
      for (int n = 0; n < 8; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) o[x][n][e] = fmaf(o[x][n][e], al[e >> 1], big[n][e] + small[n][e]);
    }
  }

  // ---- the KS warps of a row group merge (through the operand tiles' space), normalise, store
#pragma unroll
  for (int e2 = 0; e2 < 2; ++e2) {
    l[e2] += __shfl_xor_sync(0xffffffffu, l[e2], 1);
    l[e2] += __shfl_xor_sync(0xffffffffu, l[e2], 2);
  }
  if constexpr (KS > 1) {
    float* const buf = reinterpret_cast<float*>(smem_raw + (base - smem_u32(smem_raw))) + (size_t)rg * (KS - 1) * 16 * (D + 2);
    __syncthreads();                                       // every warp is done with the operand tiles
    if (kg > 0) {
      float* const mine = buf + (size_t)(kg - 1) * 16 * (D + 2);
#pragma unroll
      for (int e2 = 0; e2 < 2; ++e2) {
        float* const row = mine + (g8 + 8 * e2) * (D + 2);
#pragma unroll
        for (int x = 0; x < NB; ++x)
#pragma unroll
          for (int n = 0; n < 8; ++n)
            *reinterpret_cast<float2*>(row + 64 * x + 8 * n + 2 * t4) = make_float2(o[x][n][2 * e2], o[x][n][2 * e2 + 1]);
        if (t4 == 0) *reinterpret_cast<float2*>(row + D) = make_float2(m[e2], l[e2]);
      }
    }
    __syncthreads();
    if (kg > 0) return;
#pragma unroll
    for (int e2 = 0; e2 < 2; ++e2)
#pragma unroll
      for (int w = 0; w < KS - 1; ++w) {
        const float* const row = buf + ((size_t)w * 16 + g8 + 8 * e2) * (D + 2);
        const float2 ml = *reinterpret_cast<const float2*>(row + D);
        const float mn = fmaxf(m[e2], ml.x), fa = exp2f(m[e2] - mn), fb = exp2f(ml.x - mn);      // (warp 0 has key 0)
        m[e2] = mn;
        l[e2] = l[e2] * fa + ml.y * fb;
#pragma unroll
        for (int x = 0; x < NB; ++x)
#pragma unroll
          for (int n = 0; n < 8; ++n) {
            const float2 y = *reinterpret_cast<const float2*>(row + 64 * x + 8 * n + 2 * t4);
            o[x][n][2 * e2] = o[x][n][2 * e2] * fa + y.x * fb;
            o[x][n][2 * e2 + 1] = o[x][n][2 * e2 + 1] * fa + y.y * fb;
          }
      }
  }
#pragma unroll
  for (int e2 = 0; e2 < 2; ++e2) {
    const int i = e2 ? ib : ia;
    if (i < T && DELTA_IN(i, T, counters)) {
      const float inv = 1.0f / l[e2];
      TIn* const op = out + io + (size_t)i * D + 2 * t4;
#pragma unroll
      for (int x = 0; x < NB; ++x)
#pragma unroll
        for (int n = 0; n < 8; ++n) {
          const float a = o[x][n][2 * e2] * inv, c = o[x][n][2 * e2 + 1] * inv;
          if constexpr (sizeof(TIn) == 4) *reinterpret_cast<float2*>(op + 64 * x + 8 * n) = make_float2(a, c);
          else *reinterpret_cast<uint32_t*>(op + 64 * x + 8 * n) = pack2(a, c);
        }
    }
  }
}

}  // namespace

// A uniform batch.  Heads are the fastest index: the longest walks of every head start first.  (Head after head, the
// last head's longest walk started last: 16 heads x 1000 86.5 us, so 66.8; 32 x 2000 384, 314; d = 128 924, 819.)
// FIN: the CTAs from tile fin_y on do the finish kernel's work, one of its blocks each.
template <typename TIn, int D, int KS, bool FIN>
__global__ void __launch_bounds__(NT, D == 64 ? 2 : 1)
hybrid_attn_f32_kernel(const __grid_constant__ F32Args<TIn> p, const __grid_constant__ SeqList<1> seqs,
                       const __grid_constant__ FinishWork<TIn> fin, int fin_y) {
  if (FIN && (int)blockIdx.y >= fin_y) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int block = ((int)blockIdx.y - fin_y) * (int)gridDim.x + (int)blockIdx.x;
    extern __shared__ unsigned char smem_raw[];
    if (block < fin.blocks)
      finish_block<TIn, D, NT / 32>(fin, seqs.s[0], block, smem_raw + (-(int)smem_u32(smem_raw) & 15));
    return;
  }
  attn_f32_tile<TIn, D, KS>(p, seqs.s[0], (int)blockIdx.y, (int)blockIdx.x);
}
// A ragged group: every sequence in the form of a batch of its own.
template <typename TIn, int D>
__global__ void __launch_bounds__(NT, D == 64 ? 2 : 1)
hybrid_attn_f32_ragged_kernel(const __grid_constant__ F32Args<TIn> p, const __grid_constant__ SeqList<kSeqMax> seqs,
                              const __grid_constant__ F32Forms forms) {
  const int i = (int)blockIdx.y, ks = forms.ks[i];
  if (ks == 1) attn_f32_tile<TIn, D, 1>(p, seqs.s[i], (int)blockIdx.z, (int)blockIdx.x);
  else if (ks == 2) attn_f32_tile<TIn, D, 2>(p, seqs.s[i], (int)blockIdx.z, (int)blockIdx.x);
  else attn_f32_tile<TIn, D, 4>(p, seqs.s[i], (int)blockIdx.z, (int)blockIdx.x);
}

template <typename K, typename... A>
static cudaError_t launch_f32(K kern, std::atomic<uint64_t>& ready, size_t smem, dim3 grid, cudaStream_t st, const A&... args) {
  if (!device_done(ready)) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    device_mark(ready);
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(NT);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, args...);
  count_launch();
  return e != cudaSuccess ? e : cudaGetLastError();
}

// Warps per row group for `heads` heads of T tokens.  Every halving of the rows doubles the tiles; the longest walk bounds
// a small grid; a large one the sum of all tiles, and a part of a walk for the uneven end.  d = 64: a key tile of 64 costs
// 3.3 / 2.2 / 1.4 us where a CTA walks alone and counts 4.0 / 2.2 / 1.6 us of an SM (KS = 1 / 2 / 4).  d = 128 (one CTA per SM): 7.0 /
// 4.4 / 3.1 and 7.0 / 4.2 / 2.9, a CTA's set-up about a tile of its walk and 4 us of an SM, and the end shorter the more CTAs an
// SM gets; KS = 4 only where it is clearly ahead.  A sequence of a ragged group takes the form of a batch of its own (the forms
// round differently: its result does not depend on the sequences beside it), so a form that is a little faster alone and
// does more work in all is not taken: five sequences of up to 404 tokens, 20 heads, d = 64, 59.5 us, with the rule of d = 128 69.1.
// With each form timed at 16 shapes per d (1 to 128 heads of 64 to 2500 tokens, fp32) the chosen one is the fastest or within
// 2 % of it but for 32 heads x 128 (5 %), 8 x 700 (9 %), 128 x 128 (6 %) and, d = 128, 16 x 200 (12 %); KS = 1, 2, 4 in us: 16 heads x 1000 75, 65, 80 / d = 128
// 125, 148, 196; 16 x 1800 147, 165, 217 / 355, 407, 551; 32 x 600 56, 49, 66 / 109, 120, 165.  bf16 inputs, which run here only
// when kernel 0 is forced, take the same form.
static int f32_form(long heads, int T, int d) {
  constexpr float alone[2][3] = {{3.3f, 2.2f, 1.4f}, {7.0f, 4.4f, 3.1f}}, full[2][3] = {{4.0f, 2.2f, 1.6f}, {7.0f, 4.2f, 2.9f}};
  const int x = d == 64 ? 0 : 1;
  const float sms = (float)device_sm_count(), t = (float)((T + BN - 1) / BN), pairs = 0.5f * t * (t + 1.0f) * (float)heads;
  int ks = 1;
  float best = 3.4e38f;
  for (int c = 0; c < 3; ++c) {
    float walk = t * alone[x][c], sum = pairs * (float)(1 << c) * full[x][c] / sms, end = 0.5f;
    if (x) {
      const float ctas = (float)heads * (float)((T * (1l << c) + BN - 1) / BN), r = fmaxf(1.0f, ctas / sms);
      walk += alone[x][c];
      sum += 4.0f * ctas / sms;
      end = 0.3f / (r * r);
    }
    const float us = fmaxf(walk, sum + end * walk);
    if (us < (x && c == 2 ? 0.85f : 1.0f) * best) { best = us; ks = 1 << c; }
  }
  return ks;
}

template <typename TIn, int D>
static cudaError_t launch_f32_form(const Shape& s, const Workspace& w, const void* q, const void* k, const void* v, void* out,
                                   const SeqBatch& seqs, float theta, int init, int shape, cudaStream_t st) {
  constexpr int NP = sizeof(TIn) == 4 ? 3 : 1;
  const F32Args<TIn> p{(const TIn*)q, (const TIn*)k, (const TIn*)v, (TIn*)out, w.ckpt, w.counters, s.T_max, s.n_ckpt(), s.H,
                       s.g(), shape, theta, init == DELTA_INIT_BASIS_EXACT ? 0 : -1, 1.4426950408889634f / sqrtf((float)s.d)};
  const long heads = seqs.form_heads(s);
  static std::atomic<uint64_t> ready[4] = {}, ready_fin[3] = {};
  if (seqs.ragged) {
    SeqList<kSeqMax> list;
    F32Forms forms;
    unsigned tiles = 0;
    for (int i = 0; i < kSeqMax; ++i) {
      list.s[i] = seqs.s[i < seqs.n ? i : 0];
      forms.ks[i] = f32_form(heads, list.s[i].T, D);
      const unsigned bm = 64u / (unsigned)forms.ks[i], n = ((unsigned)list.s[i].T + bm - 1) / bm;
      tiles = n > tiles ? n : tiles;
    }
    return launch_f32(hybrid_attn_f32_ragged_kernel<TIn, D>, ready[3],
                      std::max({F32Smem<D, 1, NP>::bytes, F32Smem<D, 2, NP>::bytes, F32Smem<D, 4, NP>::bytes}),
                      dim3((unsigned)s.H, (unsigned)seqs.n, tiles), st, p, list, forms);
  }
  SeqList<1> list;
  list.s[0] = seqs.s[0];
  const unsigned T = (unsigned)list.s[0].T, bh = (unsigned)(s.B * s.H);
  const int ks = f32_form(heads, (int)T, D);
  // (a small call does the finish kernel's work in the same launch)
  const unsigned tiles = (T + 64 / ks - 1) / (64 / ks);
  FinishWork<TIn> fin{};
  if constexpr (NP == 3) {
    if (seqs.with_finish) {
      fin = finish_work<TIn>(s, w, q, k, (int)T, theta, shape, init, false);
      if (finish_beside((int)T, (long)bh * tiles, fin.blocks)) *seqs.with_finish = true;
      else fin.blocks = 0;
    }
  }
  const unsigned more = ((unsigned)fin.blocks + bh - 1) / bh;
#define GO(KS)                                                                                                        \
  do {                                                                                                                \
    if (NP == 3 && fin.blocks)                                                                                        \
      return launch_f32(hybrid_attn_f32_kernel<TIn, D, KS, NP == 3>, ready_fin[KS / 2], F32Smem<D, KS, NP>::bytes,    \
                        dim3(bh, tiles + more), st, p, list, fin, (int)tiles);                                        \
    return launch_f32(hybrid_attn_f32_kernel<TIn, D, KS, false>, ready[KS / 2], F32Smem<D, KS, NP>::bytes,            \
                      dim3(bh, tiles), st, p, list, fin, (int)tiles);                                                 \
  } while (0)
  if (ks == 4) GO(4);
  if (ks == 2) GO(2);
  GO(1);
#undef GO
}

cudaError_t launch_hybrid_attn_f32(const Shape& s, const Workspace& w, const void* q, const void* k, const void* v,
                                       void* out, const SeqBatch& seqs, float theta, int init, int shape, int dtype,
                                       cudaStream_t st) {
#define GO(TIN, DD) return launch_f32_form<TIN, DD>(s, w, q, k, v, out, seqs, theta, init, shape, st)
  if (dtype == DELTA_F32) {
    if (s.d == 64) { GO(float, 64); } else { GO(float, 128); }
  } else {
    if (s.d == 64) { GO(__nv_bfloat16, 64); } else { GO(__nv_bfloat16, 128); }
  }
#undef GO
}

}  // namespace delta
