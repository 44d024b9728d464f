// Forward product for few tokens, bf16 in, fp32 accumulate, bf16 out:
//     C[t, n] = col_scale[n] * sum_k A[t, k] B[n, k]          (A [T, K] tokens, B [N, K] weights, both K-major)
//
// Bound: latency.  At these sizes the weights are 0.1-10 MB (about a microsecond of L2 or HBM time) and a 128-row tcgen05
// tile spends 7-10 us per launch on its pipeline (barriers, tensor memory, descriptors, a serial walk over K).  What a
// launch needs is that every byte it reads is requested at once and that many SMs ask.  So
//   * the weights are the row operand of the warp-level m16n8k16 instruction and the tokens its 8-wide column operand:
//     a group of KS warps computes 16 MT weight rows x 8 NT tokens, and small T wastes nothing on the weight side;
//   * KS of the eight warps of a block cut K into 32-wide steps dealt out in turn, each reading its own part of both operands
//     straight from global memory into registers: no byte is read twice by them, nothing is staged or waited for,
//     and a warp has `kDepth` steps of loads in flight.  Their sums are added through shared memory in warp order.  The
//     8 / KS groups of warps take other weight rows: a narrow output needs all eight on K to fill the machine, a wide one has
//     rows enough, and with a short K the cut would leave warps without a step (the host picks KS);
//   * a lane reads 16 contiguous bytes of a row per step: the k positions inside a step are permuted identically for both
//     operands, so that those bytes serve two instructions without a shuffle;
//   * with RAGGED (K no multiple of 8, more than 16 tokens) the 16 bytes across the end of a row are read whole and clipped in
//     registers, but for the last row of a matrix, after which nothing need follow.  The first product of a pair fills the rows of
//     H' in the workspace with zeros up to a piece (n_pad), so that the second clips its weights only (a_padded).  From single elements
//     the end of a row costs a wait per row.  Kernel times of the two products, us, single elements / RAGGED: 300 tokens,
//     410 -> 150 -> 410 5.2 + 6.0 / 4.1 + 3.8; 100 tokens, 3001 -> 100 -> 500 11.3 + 4.2 / 8.7 + 3.6; 64 tokens, K = 358, 4096 outputs
//     5.6 / 5.4.  What cost RAGGED its gain before: rows past the end taken for the last row, whose end came from single elements
//     as well (37 tokens, 38 -> 203, 4.2 us), and a look at each row in every step (36 tokens, K = 3098, 12.6; now 3.5 and 9.8).
//     Up to 16 tokens there are few rows per lane and the extra registers and instructions cost more (one token: 3.4 against 3.7);
//   * with EARLY the first weights are requested before the wait on the previous launch.  That is for the second product of
//     a pair only: its predecessor on the stream is the first product, which waits for everything before it
//     before it lets this launch start, and which writes H' and nothing else, so the weights are final.
// Both products of 1024 -> 358 -> 4096, replayed: 3.5 us at one token and 4.6 at 16, where a warp per output column on the
// CUDA cores (up to 4 tokens) took 5.3 and a warp per 8 columns walking all of K, on 7 SMs for the first product, 11.9.
// At 64 tokens 8.6 against 14.6 with tcgen05 tiles.  64 x 64 outputs per block (fewer bytes read in all) were never faster with all eight
// warps on K; with two or four of them on a short K they are (few_shape).
#pragma once
#include "common.cuh"

namespace flop {
namespace few {

constexpr int kWarps = 8, kThreads = 32 * kWarps;

__device__ __forceinline__ void mma_bf16_16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                               uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// Eight elements of a row from k on, zero beyond K (rows are 16-byte aligned), nothing beyond K being read unless `whole` says so:
// then a piece across the end of the row is read with its padding, and the caller clips it when it is used.  (Putting a ragged
// end together from single elements waits for them before the next load is issued.)  With RAGGED the end of a row that is not read
// whole comes in up to three aligned loads, each straight to its registers: K % 8 is the same for all rows, and nothing waits.
template <bool RAGGED>
__device__ __forceinline__ uint4 load8(const __nv_bfloat16* __restrict__ row, int k, int K, bool whole) {
  uint4 v = make_uint4(0, 0, 0, 0);
  if (k + 8 <= K || (whole && k < K)) {
    v = *reinterpret_cast<const uint4*>(row + k);
  } else if (RAGGED && k < K) {
    const int left = K & 7;                                // (k is a multiple of 8)
    const __nv_bfloat16* p = row + k;
    auto u16 = [](const __nv_bfloat16* a) { return (uint32_t)*reinterpret_cast<const unsigned short*>(a); };
    auto u32 = [](const __nv_bfloat16* a) { return *reinterpret_cast<const uint32_t*>(a); };
    if (left & 4) {
      const uint2 two = *reinterpret_cast<const uint2*>(p);
      v.x = two.x; v.y = two.y;
      if (left & 2) { v.z = u32(p + 4); if (left & 1) v.w = u16(p + 6); }
      else if (left & 1) v.z = u16(p + 4);
    } else {
      if (left & 2) { v.x = u32(p); if (left & 1) v.y = u16(p + 2); }
      else if (left & 1) v.x = u16(p);
    }
  } else if (k < K) {
    __nv_bfloat16* h = reinterpret_cast<__nv_bfloat16*>(&v);
#pragma unroll
    for (int i = 0; i < 7; ++i)
      if (k + i < K) h[i] = row[k + i];
  }
  return v;
}
// The first `left` of eight elements, zeros after them.
__device__ __forceinline__ uint4 clip8(uint4 v, int left) {
  auto word = [&](uint32_t w, int i) { return left >= i + 2 ? w : left == i + 1 ? w & 0xffffu : 0u; };
  return make_uint4(word(v.x, 0), word(v.y, 2), word(v.z, 4), word(v.w, 6));
}

__host__ __device__ constexpr int part_stride(int mt) { return 16 * mt + 4; }   // floats per token of a warp's partial tile: conflict-free writes
__host__ __device__ constexpr int smem_bytes(int mt, int nt) { return kWarps * 8 * nt * part_stride(mt) * 4; }

template <int MT, int NT, int KS, bool EARLY, bool RAGGED>
__global__ void __launch_bounds__(kThreads)
gemm_kernel(const __nv_bfloat16* __restrict__ A, int64_t lda, const __nv_bfloat16* __restrict__ B, int64_t ldb,
            __nv_bfloat16* __restrict__ C, int64_t ldc, const float* __restrict__ col_scale, int T, int N, int K, int n_pad, int a_padded) {
  constexpr int kDepth = 2 * MT + NT <= 4 ? 4 : 2;         // steps of loads in flight: up to 24 16-byte loads per lane
  constexpr int kGroups = kWarps / KS;                     // groups of weight rows side by side in the block, KS warps each
  extern __shared__ __align__(16) float part[];            // [kGroups][KS][8 NT][part_stride(MT)]
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3, k_warp = warp % KS;
  const int n0 = (blockIdx.x * kGroups + warp / KS) * 16 * MT, t0 = blockIdx.y * 8 * NT;
  const __nv_bfloat16* wrow[2 * MT];                       // rows past the end are read from the last row and not stored
  const __nv_bfloat16* trow[NT];
  uint32_t wwhole = 0, twhole = 0;                         // RAGGED, bit i: another row follows row i in its matrix
  // with RAGGED from the last row but one, which is read whole: at 17 tokens a group's rows past the end are half of them
  auto row_read = [](int row, int rows) { return RAGGED ? (row < rows ? row : max(rows - 2, 0)) : min(row, rows - 1); };
#pragma unroll
  for (int i = 0; i < 2 * MT; ++i) {
    const int row = row_read(n0 + 8 * i + g, N);
    wrow[i] = B + (int64_t)row * ldb;
    if (RAGGED && row < N - 1) wwhole |= 1u << i;
  }
#pragma unroll
  for (int i = 0; i < NT; ++i) {
    const int row = row_read(t0 + 8 * i + g, T);
    trow[i] = A + (int64_t)row * lda;
    if (RAGGED && (a_padded || row < T - 1)) twhole |= 1u << i;
  }
  float acc[MT][NT][4] = {};
  uint4 wv[kDepth][2 * MT], tv[kDepth][NT];
  // this lane's part of the step at column `at` of some rows; only the step across the end of the rows, in the warps that have a last
  // row, looks at each of them
  auto load_step = [&](auto& v, const auto& rows, uint32_t whole, int at) {
    constexpr int n = sizeof(v) / sizeof(v[0]);
    if (RAGGED && at + 32 > K && __all_sync(0xffffffffu, whole == (1u << n) - 1u)) {
#pragma unroll
      for (int i = 0; i < n; ++i) v[i] = at + 8 * q < K ? *reinterpret_cast<const uint4*>(rows[i] + at + 8 * q) : make_uint4(0, 0, 0, 0);
    } else if (RAGGED && at + 32 > K) {
#pragma unroll
      for (int i = 0; i < n; ++i) v[i] = load8<true>(rows[i], at + 8 * q, K, (whole >> i) & 1u);
    } else {
#pragma unroll
      for (int i = 0; i < n; ++i) v[i] = RAGGED ? *reinterpret_cast<const uint4*>(rows[i] + at + 8 * q) : load8<false>(rows[i], at + 8 * q, K, false);
    }
  };
  auto load_weights = [&](int s) {
#pragma unroll
    for (int d = 0; d < kDepth; ++d) load_step(wv[d], wrow, wwhole, (s + d * KS) * 32);
  };
  if (!EARLY) pdl_wait();
  load_weights(k_warp);
  if (EARLY) pdl_wait();
  pdl_launch_dependents();
  for (int s = k_warp; s * 32 < K; s += kDepth * KS) {
    if (s != k_warp) load_weights(s);
#pragma unroll
    for (int d = 0; d < kDepth; ++d) load_step(tv[d], trow, twhole, (s + d * KS) * 32);
#pragma unroll
    for (int d = 0; d < kDepth; ++d) {
      const int at = (s + d * KS) * 32;
      if (RAGGED && at + 32 > K) {                         // the whole warp: the row's end is here, or behind
#pragma unroll
        for (int i = 0; i < 2 * MT; ++i) wv[d][i] = clip8(wv[d][i], K - at - 8 * q);
        if (!a_padded) {
#pragma unroll
          for (int i = 0; i < NT; ++i) tv[d][i] = clip8(tv[d][i], K - at - 8 * q);
        }
      }
#pragma unroll
      for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int n = 0; n < NT; ++n) {
          const uint4 lo = wv[d][2 * m], hi = wv[d][2 * m + 1], t = tv[d][n];
          mma_bf16_16816(acc[m][n], lo.x, hi.x, lo.y, hi.y, t.x, t.y);
          mma_bf16_16816(acc[m][n], lo.z, hi.z, lo.w, hi.w, t.z, t.w);
        }
    }
  }
  // lane (g, q) holds rows 16 m + g and + 8, tokens 8 n + 2 q and + 1
  constexpr int S = part_stride(MT);
#pragma unroll
  for (int m = 0; m < MT; ++m)
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int i = 0; i < 4; ++i)
        part[(warp * 8 * NT + 8 * n + 2 * q + (i & 1)) * S + 16 * m + g + (i >> 1) * 8] = acc[m][n][i];
  __syncthreads();
#pragma unroll
  for (int e = threadIdx.x; e < kGroups * 8 * NT * 8 * MT; e += kThreads) {      // two neighbouring columns of one token
    const int grp = e / (8 * NT * 8 * MT), t = e / (8 * MT) % (8 * NT), c = (e % (8 * MT)) * 2;
    float x = 0.f, y = 0.f;
#pragma unroll
    for (int w = 0; w < KS; ++w) {
      const float2 v = *reinterpret_cast<const float2*>(part + ((grp * KS + w) * 8 * NT + t) * S + c);
      x += v.x; y += v.y;
    }
    const int n = (blockIdx.x * kGroups + grp) * 16 * MT + c;
    if (t0 + t < T && n < n_pad) {
      if (n >= N) x = 0.f;
      if (n + 1 >= N) y = 0.f;
      if (col_scale && n < N) { x *= __ldg(col_scale + n); if (n + 1 < N) y *= __ldg(col_scale + n + 1); }
      __nv_bfloat16* o = C + (int64_t)(t0 + t) * ldc + n;
      if (n + 1 < n_pad) *reinterpret_cast<__nv_bfloat162*>(o) = __floats2bfloat162_rn(x, y);   // rows are 16-byte aligned, n is even
      else *o = __float2bfloat16_rn(x);
    }
  }
}

}  // namespace few
}  // namespace flop
