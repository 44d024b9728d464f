// Gated adaptive embedding of one word cluster (Section 4.2 of the paper): E~ = E G O.
// The lookup replaces the first GEMM of the gated layer by a row gather; the projection with O
// and the backward products are the tensor-core GEMMs used everywhere else.
//   embed_gather_kernel : H'[t, :] = E[ids[t], :] * z
//   embed_bwd_kernel    : dE[ids[t], :] += dH'[t, :] * z   (fp32 atomic adds: rows repeat across tokens)
//                         part[b][k]    = sum over the block's tokens of E[ids[t], k] dH'[t, k]
//   embed_finish_kernel : dlog_alpha from the per-block partial sums, and dO from the split-K slices of its GEMM
//
// The two token kernels are bound by the latency of a chain: token -> row of E -> store or atomic add.  A warp
// therefore takes four tokens at once and has all their ids, then all their rows in flight before it uses the first;
// rows narrower than 32 pieces of 8 columns share the warp (LPT lanes per token), so that no lane idles at
// 64 or 128 columns.  Walking eight tokens one after another, one warp per SM scheduler, took 33.5 us for 16 384 tokens of
// 256 columns, and adding up 256 partial vectors by one thread per column another 17 us.
#pragma once
#include "common.cuh"
#include "wgrad.cuh"

namespace flop {

constexpr int kEmbWarps = 8;
// Tokens of a backward block.  Fixed for every width, so that the partial sums (one vector per block) have one size.
constexpr int kEmbBlockTokens = 32;

// Lanes that share a token's row: 8 columns per lane and pass.
inline int embed_lanes(int64_t d_i) { return d_i <= 64 ? 8 : d_i <= 128 ? 16 : 32; }

// TOK: tokens a lane group has in flight.  Few tokens are spread over the SMs instead, one per lane group (32 tokens of 2048 columns and
// the product after it: 15.8 us, 17.5 with four).
template <int LPT, int TOK>
__global__ void __launch_bounds__(32 * kEmbWarps)
embed_gather_kernel(const int32_t* __restrict__ ids, int T, const __nv_bfloat16* __restrict__ E, int64_t lde, int n_rows,
                    const float* __restrict__ z, int d_i, __nv_bfloat16* __restrict__ H, int64_t ldh) {
  pdl_wait();
  pdl_launch_dependents();
  constexpr int G = 32 / LPT;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, grp = lane / LPT, l = lane % LPT;
  const int t0 = (blockIdx.x * kEmbWarps + warp) * (TOK * G) + grp;       // this lane group: t0, t0 + G, ...
  int w[TOK];
#pragma unroll
  for (int i = 0; i < TOK; ++i) w[i] = t0 + i * G < T ? min(max(ids[t0 + i * G], 0), n_rows - 1) : 0;   // out-of-range ids are clamped, never dereferenced
  for (int k = l * 8; k < d_i; k += LPT * 8) {
    if (k + 8 <= d_i) {
      uint4 raw[TOK];
#pragma unroll
      for (int i = 0; i < TOK; ++i)
        if (t0 + i * G < T) raw[i] = *reinterpret_cast<const uint4*>(E + (int64_t)w[i] * lde + k);
      float zk[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) zk[j] = __ldg(z + k + j);
#pragma unroll
      for (int i = 0; i < TOK; ++i) {
        if (t0 + i * G < T) {
          __nv_bfloat16* v = reinterpret_cast<__nv_bfloat16*>(&raw[i]);
#pragma unroll
          for (int j = 0; j < 8; ++j) v[j] = __float2bfloat16_rn(__bfloat162float(v[j]) * zk[j]);
          *reinterpret_cast<uint4*>(H + (int64_t)(t0 + i * G) * ldh + k) = raw[i];
        }
      }
    } else {
      for (int i = 0; i < TOK; ++i)
        if (t0 + i * G < T)
          for (int j = k; j < d_i; ++j)
            H[(int64_t)(t0 + i * G) * ldh + j] = __float2bfloat16_rn(__bfloat162float(E[(int64_t)w[i] * lde + j]) * z[j]);
    }
  }
}

// Block b handles `runs` x 32 consecutive tokens: one run, or two where the workspace holds half as many partial sums.  A lane owns two groups of 4 consecutive columns of every LPT * 8 columns, LPT * 4
// apart, so that a 16-byte vector atomic add of the warp covers 512 contiguous bytes of a row of dE: with 8 consecutive columns
// per lane every 32-byte sector was visited twice, by half each time, and the atomic units of the L2 bound the kernel
// (30.6 us for 16 384 tokens of 256 columns, about 19 now).  The lane groups' and the warps' partial sums of dz are added in a fixed order (shuffles, then shared
// memory in warp order).
template <int LPT>
__global__ void __launch_bounds__(32 * kEmbWarps)
embed_bwd_kernel(const int32_t* __restrict__ ids, int T, const __nv_bfloat16* __restrict__ E, int64_t lde, int n_rows,
                 const float* __restrict__ z, int d_i, const __nv_bfloat16* __restrict__ dH, int64_t lddh,
                 float* __restrict__ dE, int64_t ldde, float* __restrict__ part, int runs) {
  pdl_wait();
  pdl_launch_dependents();
  extern __shared__ float red[];   // [kEmbWarps][d_i]
  constexpr int G = 32 / LPT;                                        // tokens side by side in a warp
  constexpr int kIn = kEmbBlockTokens / kEmbWarps / G > 0 ? kEmbBlockTokens / kEmbWarps / G : 1;   // ... and one after another, in flight together
  static_assert(kIn * G * kEmbWarps == kEmbBlockTokens, "a block's tokens are dealt out evenly");
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, grp = lane / LPT, l = lane % LPT;
  const bool vec_de = dE && (reinterpret_cast<uintptr_t>(dE) & 15) == 0 && (ldde % 4) == 0;
  for (int run = 0; run < runs; ++run) {
    const int first = (blockIdx.x * runs + run) * kEmbBlockTokens + warp * (kIn * G), t0 = first + grp;
    if (first >= T) {              // warps past the last token have nothing to add
      if (run == 0)
        for (int k = lane; k < d_i; k += 32) red[warp * d_i + k] = 0.f;
      break;
    }
    int w[kIn];
#pragma unroll
    for (int i = 0; i < kIn; ++i) w[i] = t0 + i * G < T ? min(max(ids[t0 + i * G], 0), n_rows - 1) : 0;
    for (int k0 = 0; k0 < d_i; k0 += LPT * 8) {
      float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, zk[2][4];
      uint2 graw[2][kIn], eraw[2][kIn];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int k = k0 + h * (LPT * 4) + l * 4;                      // rows of dH' and E are 16-byte aligned (ld % 8 == 0)
#pragma unroll
        for (int j = 0; j < 4; ++j) zk[h][j] = k + 4 <= d_i ? __ldg(z + k + j) : 0.f;
#pragma unroll
        for (int i = 0; i < kIn; ++i) {
          graw[h][i] = eraw[h][i] = make_uint2(0, 0);
          if (k + 4 <= d_i && t0 + i * G < T) {
            graw[h][i] = __ldcs(reinterpret_cast<const uint2*>(dH + (int64_t)(t0 + i * G) * lddh + k));
            eraw[h][i] = *reinterpret_cast<const uint2*>(E + (int64_t)w[i] * lde + k);
          }
        }
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int k = k0 + h * (LPT * 4) + l * 4, nk = min(4, d_i - k);   // nk <= 0: no column for this lane here
        if (nk == 4) {
#pragma unroll
          for (int i = 0; i < kIn; ++i) {
            const __nv_bfloat162* gh = reinterpret_cast<const __nv_bfloat162*>(&graw[h][i]);
            const __nv_bfloat162* eh = reinterpret_cast<const __nv_bfloat162*>(&eraw[h][i]);
            const float2 g0 = __bfloat1622float2(gh[0]), g1 = __bfloat1622float2(gh[1]), e0 = __bfloat1622float2(eh[0]), e1 = __bfloat1622float2(eh[1]);
            acc[4 * h] = fmaf(e0.x, g0.x, acc[4 * h]);
            acc[4 * h + 1] = fmaf(e0.y, g0.y, acc[4 * h + 1]);
            acc[4 * h + 2] = fmaf(e1.x, g1.x, acc[4 * h + 2]);
            acc[4 * h + 3] = fmaf(e1.y, g1.y, acc[4 * h + 3]);
            if (dE && t0 + i * G < T) {
              float* o = dE + (int64_t)w[i] * ldde + k;
              const float d[4] = {g0.x * zk[h][0], g0.y * zk[h][1], g1.x * zk[h][2], g1.y * zk[h][3]};
              if (vec_de) {
                atomicAdd(reinterpret_cast<float4*>(o), make_float4(d[0], d[1], d[2], d[3]));
              } else {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                  if (zk[h][j] != 0.f) atomicAdd(o + j, d[j]);
              }
            }
          }
        } else if (nk > 0) {
          for (int i = 0; i < kIn; ++i) {
            const int t = t0 + i * G;
            if (t >= T) break;
#pragma unroll
            for (int j = 0; j < 3; ++j) {
              if (j < nk) {
                const float gj = __bfloat162float(dH[(int64_t)t * lddh + k + j]), zj = z[k + j];
                acc[4 * h + j] = fmaf(__bfloat162float(E[(int64_t)w[i] * lde + k + j]), gj, acc[4 * h + j]);
                if (dE && zj != 0.f) atomicAdd(dE + (int64_t)w[i] * ldde + k + j, gj * zj);
              }
            }
          }
        }
#pragma unroll
        for (int o = LPT; o < 32; o <<= 1)
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[4 * h + j] += __shfl_xor_sync(0xffffffffu, acc[4 * h + j], o);
        if (grp == 0)
          for (int j = 0; j < nk; ++j) red[warp * d_i + k + j] = (run ? red[warp * d_i + k + j] : 0.f) + acc[4 * h + j];
      }
    }
  }
  __syncthreads();
  if (part) {
    for (int k = threadIdx.x; k < d_i; k += blockDim.x) {
      float s = 0.f;
      for (int w8 = 0; w8 < kEmbWarps; ++w8) s += red[w8 * d_i + k];
      part[(int64_t)blockIdx.x * d_i + k] = s;
    }
  }
}

// Blocks [0, dla_blocks): 32 gates each, dlog_alpha[k] (=|+=) dz_dla[k] * sum of the n_part partial vectors (a warp adds
// a run of consecutive vectors, the runs are added in warp order).  The other blocks: dO (=|+=) the ordered sum of the
// split-K slices, four columns per thread.
struct EmbedFinish {
  const float* part; int n_part, d_i; const float* dz_dla; float* dla; int dla_blocks;
  const float* slices; int n_slices; int64_t slice_elems, ld_slice; void* dO; int64_t lddo; int d;
  int accumulate;
};

template <typename TW>
__global__ void __launch_bounds__(256)
embed_finish_kernel(const EmbedFinish a) {
  pdl_wait();
  pdl_launch_dependents();
  if ((int)blockIdx.x < a.dla_blocks) {
    __shared__ float run[8][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, k = blockIdx.x * 32 + lane;
    const int per = (a.n_part + 7) / 8, p1 = min(a.n_part, (warp + 1) * per);
    float s = 0.f;
    if (k < a.d_i) {
#pragma unroll 8
      for (int p = warp * per; p < p1; ++p) s += a.part[(int64_t)p * a.d_i + k];
    }
    run[warp][lane] = s;
    __syncthreads();
    if (warp == 0 && k < a.d_i) {
      s = 0.f;
#pragma unroll
      for (int w = 0; w < 8; ++w) s += run[w][lane];
      const float v = s * a.dz_dla[k];
      a.dla[k] = a.accumulate ? a.dla[k] + v : v;
    }
    return;
  }
  constexpr int al = sizeof(TW) == 4 ? 15 : 7;
  const bool vec = (reinterpret_cast<uintptr_t>(a.dO) & al) == 0 && a.lddo % 4 == 0;
  const int c4 = (a.d + 3) >> 2;
  const int64_t units = (int64_t)a.d_i * c4, step = (int64_t)(gridDim.x - a.dla_blocks) * blockDim.x;
  for (int64_t u = (int64_t)(blockIdx.x - a.dla_blocks) * blockDim.x + threadIdx.x; u < units; u += step)
    reduce_unit<TW>(a.slices, a.n_slices, a.slice_elems, a.ld_slice, (int)(u / c4), (int)(u % c4) * 4, a.d, 1.f, (TW*)a.dO, a.lddo,
                    a.accumulate, vec);
}

}  // namespace flop
