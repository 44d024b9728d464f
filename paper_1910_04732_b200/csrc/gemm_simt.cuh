// fp32 FMA GEMM for the FLOP_F32 storage type: C[M,N] = sum_k A(m,k) B(n,k).
//
// The tensor cores have no true fp32 mode, and the fp32 configuration is held to 1e-5 relative error, so this
// path multiplies and accumulates in fp32 on the CUDA cores.  Every operand is a row-major matrix read either
// along its rows (K-fast: k is the unit stride) or down its columns (MN-fast: m or n is), which covers all six
// GEMMs of the layer without transposes; the two forms are template parameters, because they decide the
// shared-memory layout.
//
// Bound: at the sizes of this configuration (outputs of 64..2048 x 128..768) by latency, not by the FMA units: the
// 32 tiles of a 512 x 256 product leave 116 SMs idle, and a block that loads, waits and multiplies in turn spends
// nine tenths of its time waiting.  Hence
//   * cp.async into three shared-memory stages (64 x 32 floats of each operand), so that the loads of two k-blocks are
//     in flight while a third is multiplied; 16-byte pieces where base and leading dimension allow them, else 4-byte;
//   * a cluster of up to eight CTAs shares one 64 x 64 tile: each takes a slice of K, and every CTA adds up its rows of
//     the tile from all slices through distributed shared memory, in rank order (the same bits on every run).
// One 512 x 256 x 256 product took 26.6 us in the single-buffered unsplit form (64 x 64 x 16); forward and backward of that
// matrix with its small launches went from 181.6 to 69.8 us, and to 42.3 from 52.0 when the backward products came to share two launches.  4 x 4 results per thread: 64 FMAs per eight 16-byte
// shared-memory reads, of which half are broadcasts.
// The epilogue applies the gate of the column (H'), of the row (dQ) and the fused row dot <Q[m,:], C[m,:]> (dz), whose
// partial sums stay in fp64; `k_scale` multiplies B(n,k) by z[k] as it is read, so that diag(z) Q is never written.
#pragma once
#include "common.cuh"

namespace flop {

struct SimtGemmArgs {
  const float* A; int64_t lda;          // A(m,k) = A[m*lda + k] (K-fast) or A[k*lda + m] (MN-fast)
  const float* B; int64_t ldb;          // B(n,k) likewise
  float* C; int64_t ldc;                // nullable when only the row dot is wanted; C[m*ldc + n]
  int M, N, K;
  int kb_per_split;                     // 32-wide k-blocks per CTA of the cluster
  int a_vec, b_vec;                     // operand rows are 16-byte aligned
  const float* col_scale;               // nullable: C[m,n] *= col_scale[n]
  const float* row_scale;               // nullable: C[m,n] *= row_scale[m]
  const float* k_scale;                 // nullable: B(n,k) is multiplied by k_scale[k]
  int accumulate;                       // C += instead of C =
  const float* qdot; int64_t ldq;       // nullable: dz_part[tile of n][m] = sum_n qdot[m,n] * C[m,n] before scaling
  double* dz_part; int64_t dz_stride;
};

namespace simt {

constexpr int BM = 64, BN = 64, BK = 32, kThreads = 256, kStages = 3;
constexpr int kRowK = BK + 4;                            // K-fast rows in shared memory: 144 bytes, conflict-free 16-byte reads
constexpr int kOperandFloats = BM * kRowK;               // >= BK * BM, the MN-fast layout [k][64]
constexpr int kStageFloats = 2 * kOperandFloats + BK;    // A, B, k_scale
constexpr int kRowP = BN + 4;                            // rows of the partial tile
constexpr int kSmemBytes = kStages * kStageFloats * 4;
constexpr int kMaxSplit = 8;                             // portable cluster size
static_assert(BM == BN && BM * kRowP <= kStages * kStageFloats, "partial tile reuses the stages");

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
// bytes (0..16, or 0..4) are read, the rest of the piece is zero-filled; with bytes = 0 the source is not read
__device__ __forceinline__ void copy16(uint32_t dst, const void* src, int bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void copy4(uint32_t dst, const void* src, int bytes) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}

// One operand's 64 x 32 block (rows from `row0` of `rows`, k from k0 below k_end) into shared memory.
template <bool KFAST>
__device__ __forceinline__ void load_block(const float* __restrict__ p, int64_t ld, int row0, int rows, int k0, int k_end, int vec,
                                           uint32_t dst, int tid) {
  if (vec) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int e = tid + i * kThreads;                   // 512 pieces of 16 bytes
      if (KFAST) {
        const int r = e >> 3, k = (e & 7) * 4;
        const int left = row0 + r < rows ? min(4, k_end - (k0 + k)) : 0;
        copy16(dst + (uint32_t)(r * kRowK + k) * 4u, left > 0 ? p + (int64_t)(row0 + r) * ld + k0 + k : p, max(left, 0) * 4);
      } else {
        const int k = e >> 4, r = (e & 15) * 4;
        const int left = k0 + k < k_end ? min(4, rows - (row0 + r)) : 0;
        copy16(dst + (uint32_t)(k * BM + r) * 4u, left > 0 ? p + (int64_t)(k0 + k) * ld + row0 + r : p, max(left, 0) * 4);
      }
    }
  } else {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int e = tid + i * kThreads;                   // 2048 floats
      const int r = KFAST ? e >> 5 : e & 63, k = KFAST ? e & 31 : e >> 6;
      const bool in = row0 + r < rows && k0 + k < k_end;
      const float* src = KFAST ? p + (int64_t)(row0 + r) * ld + k0 + k : p + (int64_t)(k0 + k) * ld + row0 + r;
      copy4(dst + (uint32_t)(KFAST ? r * kRowK + k : k * BM + r) * 4u, in ? src : p, in ? 4 : 0);
    }
  }
}

// The 64 x 64 tile (tile_m, tile_n) of one product: this CTA takes slice `split` of K, the other slices are with CTAs first ..
// first + n_split - 1 of the cluster, all of whose tiles are cut alike.  A CTA without a tile (live = false) only takes part in the
// cluster's barriers, which tiles that are not cut do without (they held eight tiles to the pace of the slowest: 96 tokens of 768 ->
// 768, backward, 45.2 us in shared launches against 42.6 in separate ones).
template <bool A_K, bool B_K, bool SCALE_K>
__device__ __forceinline__ void gemm_tile(const SimtGemmArgs& p, int tile_m, int tile_n, int split, int n_split, int first, bool live) {
  const bool clustered = n_split > 1;
  extern __shared__ __align__(16) float smem[];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int m0 = tile_m * BM, n0 = tile_n * BN;
  const int kb0 = split * p.kb_per_split, kb1 = live ? min((p.K + BK - 1) / BK, kb0 + p.kb_per_split) : kb0;

  auto load = [&](int kb) {
    if (kb < kb1) {
      const uint32_t st = smem_addr(smem + (kb % kStages) * kStageFloats);
      load_block<A_K>(p.A, p.lda, m0, p.M, kb * BK, p.K, p.a_vec, st, tid);
      load_block<B_K>(p.B, p.ldb, n0, p.N, kb * BK, p.K, p.b_vec, st + kOperandFloats * 4, tid);
      if (SCALE_K && tid < BK) {
        const bool in = kb * BK + tid < p.K;
        copy4(st + (2 * kOperandFloats + tid) * 4, in ? p.k_scale + kb * BK + tid : p.k_scale, in ? 4 : 0);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");   // an empty group keeps the count of groups in step
  };

  float acc[4][4] = {};
#pragma unroll
  for (int s = 0; s < kStages - 1; ++s) load(kb0 + s);
  for (int kb = kb0; kb < kb1; ++kb) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
    __syncthreads();                                       // block kb has landed; block kb - 1 has been read by everyone
    load(kb + kStages - 1);
    const float* As = smem + (kb % kStages) * kStageFloats;
    const float* Bs = As + kOperandFloats;
    const float* Zs = Bs + kOperandFloats;
    auto multiply = [&](int k) {
      float a[4][4], b[4][4];                              // [row or column of the thread][k]
      if (A_K) {
#pragma unroll
        for (int i = 0; i < 4; ++i) *reinterpret_cast<float4*>(a[i]) = *reinterpret_cast<const float4*>(As + (ty + 16 * i) * kRowK + k);
      } else {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const float4 v = *reinterpret_cast<const float4*>(As + (k + c) * BM + ty * 4);
          a[0][c] = v.x; a[1][c] = v.y; a[2][c] = v.z; a[3][c] = v.w;
        }
      }
      if (B_K) {
#pragma unroll
        for (int j = 0; j < 4; ++j) *reinterpret_cast<float4*>(b[j]) = *reinterpret_cast<const float4*>(Bs + (tx + 16 * j) * kRowK + k);
      } else {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const float4 v = *reinterpret_cast<const float4*>(Bs + (k + c) * BN + tx * 4);
          b[0][c] = v.x; b[1][c] = v.y; b[2][c] = v.z; b[3][c] = v.w;
        }
      }
      if (SCALE_K) {
        const float4 z = *reinterpret_cast<const float4*>(Zs + k);
#pragma unroll
        for (int j = 0; j < 4; ++j) { b[j][0] *= z.x; b[j][1] *= z.y; b[j][2] *= z.z; b[j][3] *= z.w; }
      }
#pragma unroll
      for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i][c], b[j][c], acc[i][j]);
    };
    if (kb * BK + BK <= p.K) {
#pragma unroll
      for (int k = 0; k < BK; k += 4) multiply(k);
    } else {                                               // the zeros beyond K need no FMAs (K = 33: 36 of 64 steps are left)
#pragma unroll 1
      for (int k = 0; kb * BK + k < p.K; k += 4) multiply(k);
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();                                         // every stage has been read: the partial tile takes their place
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
      smem[(A_K ? ty + 16 * i : ty * 4 + i) * kRowP + (B_K ? tx + 16 * j : tx * 4 + j)] = acc[i][j];
  if (clustered) {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  } else {
    __syncthreads();
  }
  // this CTA finishes rows [split, split + 1) * BM / n_split of the tile, 16 lanes per row, 4 columns each
  const int rows = live ? BM / n_split : 0;
  const bool c_vec = (reinterpret_cast<uintptr_t>(p.C) & 15) == 0 && (p.ldc & 3) == 0;
  for (int lr = ty; lr < rows; lr += 16) {
    const int r = split * rows + lr, gm = m0 + r, gn = n0 + tx * 4;
    float v[4] = {0.f, 0.f, 0.f, 0.f};
    const uint32_t at = smem_addr(smem + r * kRowP + tx * 4);
    for (int s = 0; s < n_split; ++s) {
      uint32_t peer;
      float x, y, z, w;
      asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(peer) : "r"(at), "r"(first + s));
      asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(x), "=f"(y), "=f"(z), "=f"(w) : "r"(peer) : "memory");
      v[0] += x; v[1] += y; v[2] += z; v[3] += w;
    }
    if (p.qdot) {
      double dot = 0.0;
      if (gm < p.M)
        for (int j = 0; j < 4; ++j)
          if (gn + j < p.N) dot += (double)v[j] * (double)p.qdot[(int64_t)gm * p.ldq + gn + j];
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);   // rows is 8..64: warps are in the loop as a whole
      if (tx == 0 && gm < p.M) p.dz_part[(int64_t)tile_n * p.dz_stride + gm] = dot;
    }
    if (p.C && gm < p.M) {
      const float rs = p.row_scale ? p.row_scale[gm] : 1.f;
      float* c = p.C + (int64_t)gm * p.ldc + gn;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        v[j] *= rs;
        if (p.col_scale && gn + j < p.N) v[j] *= p.col_scale[gn + j];
      }
      if (c_vec && gn + 4 <= p.N) {
        float4 w = make_float4(v[0], v[1], v[2], v[3]);
        if (p.accumulate) { const float4 o = *reinterpret_cast<const float4*>(c); w.x += o.x; w.y += o.y; w.z += o.z; w.w += o.w; }
        *reinterpret_cast<float4*>(c) = w;
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (gn + j < p.N) c[j] = p.accumulate ? c[j] + v[j] : v[j];
      }
    }
  }
  if (clustered) {         // no CTA leaves while another still reads its shared memory
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
}

template <bool A_K, bool B_K, bool SCALE_K>
__global__ void __launch_bounds__(kThreads, 2)
gemm_kernel(const SimtGemmArgs p) {
  pdl_wait();
  pdl_launch_dependents();
  gemm_tile<A_K, B_K, SCALE_K>(p, blockIdx.y, blockIdx.x, blockIdx.z, gridDim.z, 0, true);      // the cluster spans z
}

// Two products that need only what is there before the launch: an activation gradient (dH' = dY P, or dX = dH' diag(z) Q with
// SCALE_K) and the weight gradient that contracts over the tokens (dP, dQ).  Apart, each leaves SMs idle and waits for the other's
// last tile.  Each keeps the split, and so the bits, of its own launch: a cluster has as many CTAs as the larger split, and
// several tiles of the product with the smaller one.  The product with the longer slices comes first.
struct DualArgs {
  SimtGemmArgs act, wgrad;
  int act_split, wgrad_split, act_clusters, wgrad_clusters, wgrad_first;
};
template <bool SCALE_K>
__global__ void __launch_bounds__(kThreads, 2)
gemm_dual_kernel(const DualArgs d) {
  pdl_wait();
  pdl_launch_dependents();
  const int c = blockIdx.x, rank = blockIdx.z, size = gridDim.z;
  const bool wgrad = d.wgrad_first ? c < d.wgrad_clusters : c >= d.act_clusters;
  const SimtGemmArgs& p = wgrad ? d.wgrad : d.act;
  const int split = wgrad ? d.wgrad_split : d.act_split, local = c - (wgrad == (d.wgrad_first != 0) ? 0 : wgrad ? d.act_clusters : d.wgrad_clusters);
  const int t = local * (size / split) + rank / split, tiles_n = (p.N + BN - 1) / BN, tile_m = t / tiles_n, first = rank / split * split;
  const bool live = tile_m < (p.M + BM - 1) / BM;
  if (wgrad) gemm_tile<false, false, false>(d.wgrad, tile_m, t % tiles_n, rank % split, split, first, live);
  else gemm_tile<true, false, SCALE_K>(d.act, tile_m, t % tiles_n, rank % split, split, first, live);
}

}  // namespace simt

// dlog_alpha[k] (=|+=) dz_dla[k] * sum_p dz_part[p][k], fp64 partials of the fp32 path added in order.
__global__ void __launch_bounds__(256)
dalpha_f64_kernel(const double* __restrict__ dz_part, int n_part, int64_t part_stride, const float* __restrict__ dz_dla, int r,
                  float* __restrict__ dlog_alpha, int accumulate) {
  pdl_wait();
  pdl_launch_dependents();
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= r) return;
  double s = 0.0;
  for (int p = 0; p < n_part; ++p) s += dz_part[(int64_t)p * part_stride + k];
  const float v = (float)s * dz_dla[k];
  dlog_alpha[k] = accumulate ? dlog_alpha[k] + v : v;
}

}  // namespace flop
