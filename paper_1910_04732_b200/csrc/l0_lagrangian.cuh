// Expected L0 size and augmented-Lagrangian penalty (Eq. 3 and Section 4.3).
//
// Three launches, no atomics, fixed summation order (bit-reproducible):
//   1. l0_chunk_kernel<false>: every block owns one chunk of kL0Chunk gates of ONE
//      segment and writes sum(pi_j) of the chunk (fp64) to scratch.
//   2. l0_finalize_kernel    : one block adds the chunk sums per segment in chunk
//      order, forms s, g, dg/dlambda and the gradient coefficient.
//   3. l0_chunk_kernel<true> : dlog_alpha_j += coef * size_seg * pi_j (1 - pi_j).
// Blocks find their (segment, chunk) from the segment table alone: chunk
// counts per segment are prefix-summed in shared memory by every block.
// The segment table lives in device memory, so the host cannot check it: the kernels
// do.  A table that needs more chunk sums than the scratch holds (`capacity`), or
// that points outside [0, n), touches nothing; the finalisation then reports
// FLOP_ERR_INVALID_ARG in the device status word and writes NaN to out4.
#pragma once
#include "common.cuh"

namespace flop {

constexpr int kL0Threads = 256;
constexpr int kL0PerThread = 32;                    // eight 16-byte vectors per thread
constexpr int kL0Chunk = kL0Threads * kL0PerThread;  // gates per block
constexpr int kL0MaxSeg = 4096;

struct L0Scratch {         // layout of the caller's workspace
  double coef;             // (lambda1 + 2 lambda2 (s - t)) / S
  double pad[31];
  double partial[1];       // [n_chunks_max]
};

// Fills seg_first_chunk[0..n_seg] (exclusive prefix of chunks per segment) in
// shared memory.  Serial per 16 segments per thread, then a block scan.
__device__ __forceinline__ void l0_chunk_table(const int64_t* __restrict__ seg_off, int n_seg, int* first_chunk,
                                               int* scan_scratch) {
  // thread t owns segments [t*per, (t+1)*per): per = 1 for up to 256 segments, so the table costs
  // one 16-byte read per thread instead of a fixed sixteen
  const int per = (n_seg + kL0Threads - 1) / kL0Threads;
  const int s0 = threadIdx.x * per;
  int sum = 0;
  for (int i = 0; i < per; ++i) {
    const int s = s0 + i;
    if (s < n_seg) {
      const int64_t len = seg_off[s + 1] - seg_off[s];
      sum += len > 0 ? (int)((len + kL0Chunk - 1) / kL0Chunk) : 0;
    }
  }
  int total;
  int base = block_exclusive_scan(sum, scan_scratch, &total);
  for (int i = 0; i < per; ++i) {
    const int s = s0 + i;
    if (s < n_seg) {
      first_chunk[s] = base;
      const int64_t len = seg_off[s + 1] - seg_off[s];
      base += len > 0 ? (int)((len + kL0Chunk - 1) / kL0Chunk) : 0;
    }
  }
  if (threadIdx.x == 0) first_chunk[n_seg] = total;
  __syncthreads();
}

// Largest s with first_chunk[s] <= b and a non-empty chunk range containing b.
__device__ __forceinline__ int l0_find_segment(const int* first_chunk, int n_seg, int b) {
  int lo = 0, hi = n_seg;  // invariant: first_chunk[lo] <= b < first_chunk[hi]
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (first_chunk[mid] <= b) lo = mid; else hi = mid;
  }
  return lo;
}

__device__ __forceinline__ float l0_pi(float a, float thr) { return __fdividef(1.0f, 1.0f + __expf(-(a - thr))); }

template <bool kGrad>
__global__ void __launch_bounds__(kL0Threads)
l0_chunk_kernel(const float* __restrict__ log_alpha, const int64_t* __restrict__ seg_off,
                const float* __restrict__ seg_size, int n_seg, float thr, L0Scratch* __restrict__ sc,
                float* __restrict__ dlog_alpha, int64_t n, int capacity) {
  pdl_wait();
  pdl_launch_dependents();
  __shared__ int first_chunk[kL0MaxSeg + 1];
  __shared__ int scan_scratch[33];
  __shared__ double red[32];
  l0_chunk_table(seg_off, n_seg, first_chunk, scan_scratch);
  const int b = blockIdx.x;
  if (first_chunk[n_seg] > capacity) return;   // the table asks for more chunk sums than the scratch holds
  if (b >= first_chunk[n_seg]) {            // surplus block of the upper-bound grid
    return;
  }
  const int seg = l0_find_segment(first_chunk, n_seg, b);
  const int64_t lo = seg_off[seg] + (int64_t)(b - first_chunk[seg]) * kL0Chunk;
  const int64_t hi = min(seg_off[seg + 1], lo + (int64_t)kL0Chunk);
  if (lo < 0 || hi > n) return;             // a segment outside the gate vector: nothing is read or written
  // vector v of thread t covers gates lo + (v*256 + t)*4 .. +3: consecutive threads, consecutive 16 bytes
  constexpr int kVec = kL0PerThread / 4;
  const bool al_a = (reinterpret_cast<uintptr_t>(log_alpha + lo) & 15) == 0;
  double sum = 0.0;
  float w = 0.f;
  bool al_g = false;
  if (kGrad) {
    w = (float)(sc->coef * (double)seg_size[seg]);
    al_g = al_a && (reinterpret_cast<uintptr_t>(dlog_alpha + lo) & 15) == 0;
  }
#pragma unroll
  for (int v = 0; v < kVec; ++v) {
    const int64_t j0 = lo + ((int64_t)v * kL0Threads + threadIdx.x) * 4;
    if (j0 >= hi) continue;
    float a[4];
    const bool full = j0 + 4 <= hi;
    if (full && al_a) {
      const float4 t = __ldcs(reinterpret_cast<const float4*>(log_alpha + j0));
      a[0] = t.x; a[1] = t.y; a[2] = t.z; a[3] = t.w;
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = (j0 + i < hi) ? log_alpha[j0 + i] : 0.f;
    }
    if (!kGrad) {
      // the four probabilities of a vector are added in fp32 (each is in (0, 1): the group sum is exact to
      // 2^-22), the groups in fp64: a quarter of the fp64 conversions and additions, which bound this pass
      float p4[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) p4[i] = (j0 + i < hi) ? l0_pi(a[i], thr) : 0.f;
      sum += (double)((p4[0] + p4[1]) + (p4[2] + p4[3]));
    } else {
      float gsum[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        // pi (1 - pi) = e / (1 + e)^2 with e = exp(-|alpha - thr|): no cancellation near pi = 1
        const float e = __expf(-fabsf(a[i] - thr));
        const float q = __fdividef(1.0f, 1.0f + e);
        gsum[i] = w * e * q * q;
      }
      if (full && al_g) {
        float4 g = *reinterpret_cast<float4*>(dlog_alpha + j0);
        g.x += gsum[0]; g.y += gsum[1]; g.z += gsum[2]; g.w += gsum[3];
        *reinterpret_cast<float4*>(dlog_alpha + j0) = g;
      } else {
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (j0 + i < hi) dlog_alpha[j0 + i] += gsum[i];
      }
    }
  }
  if (!kGrad) {
    sum = block_sum_f64(sum, red);
    if (threadIdx.x == 0) sc->partial[b] = sum;
  }
}

__global__ void __launch_bounds__(kL0Threads)
l0_finalize_kernel(const int64_t* __restrict__ seg_off, const float* __restrict__ seg_size, int n_seg,
                   const float* __restrict__ target, const float* __restrict__ lambda, L0Scratch* __restrict__ sc,
                   float* __restrict__ out4, float* __restrict__ seg_expected, int64_t n, int capacity) {
  pdl_wait();
  pdl_launch_dependents();
  __shared__ int first_chunk[kL0MaxSeg + 1];
  __shared__ int scan_scratch[33];
  __shared__ double red_w[32], red_s[32];
  __shared__ int bad;
  if (threadIdx.x == 0) bad = 0;
  l0_chunk_table(seg_off, n_seg, first_chunk, scan_scratch);
  // the segments must partition [0, n): ascending offsets from 0 to n (the chunk sums of anything else were not written)
  for (int s = threadIdx.x; s < n_seg; s += blockDim.x)
    if (seg_off[s] < 0 || seg_off[s + 1] < seg_off[s] || seg_off[s + 1] > n) bad = 1;
  __syncthreads();
  if (first_chunk[n_seg] > capacity || bad || (n_seg > 0 && (seg_off[0] != 0 || seg_off[n_seg] != n))) {
    if (threadIdx.x == 0) {
      atomicExch(&g_device_status, (int)FLOP_ERR_INVALID_ARG);
      const float nan = __int_as_float(0x7fc00000);
      out4[0] = nan; out4[1] = nan; out4[2] = nan; out4[3] = nan;
      sc->coef = 0.0;
    }
    return;
  }
  // One warp per segment (segments w, w + nwarp, ...): lanes stride over the segment's chunk sums,
  // a butterfly adds them, and every warp keeps running totals over its own segments.  The
  // assignment is fixed, so the result is bit-reproducible.
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = kL0Threads / 32;
  double weighted = 0.0, total_size = 0.0;
  for (int s = warp; s < n_seg; s += nwarp) {
    double v = 0.0;
    for (int c = first_chunk[s] + lane; c < first_chunk[s + 1]; c += 32) v += sc->partial[c];
    v = warp_sum_f64(v);
    if (lane == 0 && seg_expected) seg_expected[s] = (float)v;
    const double size = (double)seg_size[s];
    weighted += size * v;
    total_size += size * (double)(seg_off[s + 1] - seg_off[s]);
  }
  if (lane == 0) { red_w[warp] = weighted; red_s[warp] = total_size; }
  __syncthreads();
  if (threadIdx.x == 0) {
    weighted = 0.0; total_size = 0.0;
    for (int w = 0; w < nwarp; ++w) { weighted += red_w[w]; total_size += red_s[w]; }
    const double s = total_size > 0.0 ? weighted / total_size : 0.0;
    const double diff = s - (double)target[0];
    const double l1 = (double)lambda[0], l2 = (double)lambda[1];
    out4[0] = (float)s;
    out4[1] = (float)(l1 * diff + l2 * diff * diff);
    out4[2] = (float)diff;
    out4[3] = (float)(diff * diff);
    sc->coef = total_size > 0.0 ? (l1 + 2.0 * l2 * diff) / total_size : 0.0;
  }
}

// All three passes in one launch for up to kL0SmallMax gates: the gates of a whole model, where the three launches above are
// bound by their latencies (5.2 + 10.5 + 5.1 us for 72 segments of 768 gates).  One cluster of eight CTAs.  The gates are dealt
// to the 128 warps in equal runs whatever the segments are: a warp takes the pieces of segments that lie in its run, reads the
// table 32 entries at a time and leaves short segments to single lanes, so that neither one long segment nor many short or
// empty ones make a chain (a warp per segment took 243 us where one segment held 65 000 gates, this form 7).  A run stays in
// registers, 16 gates per lane at the limit, which is why the limit is there: at 65 536 gates this is still the faster form
// (72 segments of 768 12.9 against 7.6 us, 24 of 2048 10.0 against 7.1).  The CTAs exchange
// their totals through distributed shared memory and each finishes the scalar part by itself, so nothing passes through global
// memory and no scratch is needed.  Every sum has a fixed order.  The table is checked as in l0_finalize_kernel, before
// anything is written.
constexpr int64_t kL0SmallMax = 65536;
constexpr int kL0SmallCtas = 8, kL0SmallThreads = 512, kL0SmallWarps = kL0SmallThreads / 32;
inline int l0_small_run(int n) { return (n + kL0SmallCtas * kL0SmallThreads - 1) / (kL0SmallCtas * kL0SmallThreads) * 32; }   // gates per warp
inline uint32_t l0_small_inverse(int run) { return (uint32_t)(0x100000000ull / (uint64_t)run + 1); }   // j / run == (j * inverse) >> 32 for j <= kL0SmallMax + run

// The pieces of segments in gates [pos, end) of a warp's run, in order; `s` is the segment that holds gate pos.  A segment of
// fewer than 32 gates that lies in the run as a whole goes to one lane, lane_piece(segment, first gate, one past the last, size);
// every other piece to the warp, warp_piece(segment, its first gate, one past its last, the same of the piece, size).
template <typename L, typename W>
__device__ __forceinline__ void l0_for_pieces(const int64_t* __restrict__ seg_off, const float* __restrict__ seg_size, int n_seg, int s, int pos,
                                              int end, int lane, L&& lane_piece, W&& warp_piece) {
  bool more = pos < end;
  for (; more && s < n_seg; s += 32) {
    int lo = end, hi = end;
    float size = 0.f;
    if (s + lane < n_seg) { lo = (int)seg_off[s + lane]; hi = (int)seg_off[s + lane + 1]; size = seg_size[s + lane]; }
    const bool mine = lo >= pos && lo < hi && hi <= end && hi - lo < 32;
    if (mine) lane_piece(s + lane, lo, hi, size);
    unsigned todo = __ballot_sync(0xffffffffu, !mine && max(lo, pos) < min(hi, end));
    more = __shfl_sync(0xffffffffu, hi, 31) < end;
    while (todo) {
      const int l = __ffs(todo) - 1;
      todo &= todo - 1;
      const int seg_lo = __shfl_sync(0xffffffffu, lo, l), seg_hi = __shfl_sync(0xffffffffu, hi, l);
      warp_piece(s + l, seg_lo, seg_hi, max(seg_lo, pos), min(seg_hi, end), __shfl_sync(0xffffffffu, size, l));
    }
  }
}

// STEPS: gates per lane of a run, 32 STEPS >= run.
template <int STEPS>
__global__ void __launch_bounds__(kL0SmallThreads, 1)
l0_small_kernel(const float* __restrict__ log_alpha, const int64_t* __restrict__ seg_off, const float* __restrict__ seg_size, int n_seg,
                float thr, const float* target, const float* lambda, float* out4, float* __restrict__ seg_expected,
                float* __restrict__ dlog_alpha, int n, int run, uint32_t run_inv) {
  pdl_wait();
  pdl_launch_dependents();
  // read by every CTA before the cluster's barrier: CTA 0 writes out4 after it, which may lie on the same memory
  const double goal = (double)target[0], l1 = (double)lambda[0], l2 = (double)lambda[1];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, cta = blockIdx.x;
  const int me = cta * kL0SmallWarps + warp, pos = min(n, me * run), end = min(n, pos + run);
  float a[STEPS];                       // gate pos + 32 i + lane: the whole run is on its way before the table is read
#pragma unroll
  for (int i = 0; i < STEPS; ++i) a[i] = pos + 32 * i + lane < end ? log_alpha[pos + 32 * i + lane] : 0.f;
  __shared__ double red_w[kL0SmallWarps], red_s[kL0SmallWarps];
  __shared__ __align__(16) double total[2];
  __shared__ double head[kL0SmallWarps];        // a warp's sum over the segment that began before its run
  __shared__ int s_first[kL0SmallWarps];        // the segment that holds the first gate of a warp's run
  auto warp_of = [&](int j) { return (int)__umulhi((uint32_t)j, run_inv); };   // j / run
  int bad = 0;
  for (int s = tid; s < n_seg; s += kL0SmallThreads) {
    const int64_t lo = seg_off[s], hi = seg_off[s + 1];
    if (lo < 0 || hi < lo || hi > n || (s == 0 && lo != 0) || (s == n_seg - 1 && hi != n)) { bad = 1; continue; }
    if (lo == hi) continue;
    const int g1 = min(warp_of((int)hi - 1), cta * kL0SmallWarps + kL0SmallWarps - 1);
    for (int g = max(warp_of((int)lo + run - 1), cta * kL0SmallWarps); g <= g1; ++g) s_first[g - cta * kL0SmallWarps] = s;
  }
  if (__syncthreads_or(bad)) {     // every CTA takes the same decision
    if (cta == 0 && tid == 0) {
      atomicExch(&g_device_status, (int)FLOP_ERR_INVALID_ARG);
      const float nan = __int_as_float(0x7fc00000);
      out4[0] = nan; out4[1] = nan; out4[2] = nan; out4[3] = nan;
    }
    return;
  }
  const int s0 = pos < end ? s_first[warp] : n_seg;
  double weighted = 0.0, size_sum = 0.0, tail = 0.0;
  int tail_seg = -1, tail_end = 0;              // the segment that goes on in the next warps' runs
  int lanes = 0;                                // some sums are spread over the lanes
  l0_for_pieces(seg_off, seg_size, n_seg, s0, pos, end, lane, [&](int s, int lo, int hi, float size) {
    lanes = 1;
    double v = 0.0;
#pragma unroll 4
    for (int j = lo; j < hi; ++j) v += (double)l0_pi(log_alpha[j], thr);
    weighted += (double)size * v;
    size_sum += (double)size * (double)(hi - lo);
    if (seg_expected) seg_expected[s] = (float)v;
  }, [&](int s, int seg_lo, int seg_hi, int lo, int hi, float size) {
    double v = 0.0;
#pragma unroll
    for (int i = 0; i < STEPS; ++i) {
      const int j = pos + 32 * i + lane;
      if (j >= lo && j < hi) v += (double)l0_pi(a[i], thr);
    }
    v = warp_sum_f64(v);
    if (lane == 0) {
      weighted += (double)size * v;
      size_sum += (double)size * (double)(hi - lo);
    }
    if (lo > seg_lo) {
      if (lane == 0) head[warp] = v;
    } else if (hi < seg_hi) {
      tail = v; tail_seg = s; tail_end = seg_hi;
    } else if (seg_expected && lane == 0) {
      seg_expected[s] = (float)v;
    }
  });
  if (__any_sync(0xffffffffu, lanes)) {
    weighted = warp_sum_f64(weighted);
    size_sum = warp_sum_f64(size_sum);
  }
  if (lane == 0) { red_w[warp] = weighted; red_s[warp] = size_sum; }
  __syncthreads();
  if (tid == 0) {
    weighted = 0.0; size_sum = 0.0;
    for (int w = 0; w < kL0SmallWarps; ++w) { weighted += red_w[w]; size_sum += red_s[w]; }
    total[0] = weighted; total[1] = size_sum;
  }
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  if (seg_expected)                             // segments without gates
    for (int s = cta * kL0SmallThreads + tid; s < n_seg; s += kL0SmallCtas * kL0SmallThreads)
      if (seg_off[s] == seg_off[s + 1]) seg_expected[s] = 0.f;
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  weighted = 0.0; size_sum = 0.0;
  const uint32_t at = (uint32_t)__cvta_generic_to_shared(total);
  for (int c = 0; c < kL0SmallCtas; ++c) {
    uint32_t peer;
    double a, b;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(peer) : "r"(at), "r"(c));
    asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(a), "=d"(b) : "r"(peer) : "memory");
    weighted += a; size_sum += b;
  }
  if (seg_expected && tail_seg >= 0) {          // the rest of the segment that began in this run
    double v = 0.0;
    for (int g = me + 1 + lane; g <= warp_of(tail_end - 1); g += 32) {
      uint32_t peer;
      double h;
      asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(peer) : "r"((uint32_t)__cvta_generic_to_shared(head + g % kL0SmallWarps)), "r"(g / kL0SmallWarps));
      asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(h) : "r"(peer) : "memory");
      v += h;
    }
    v = warp_sum_f64(v) + tail;
    if (lane == 0) seg_expected[tail_seg] = (float)v;
  }
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");   // the totals have been read (waited for at the end)
  const double s = size_sum > 0.0 ? weighted / size_sum : 0.0, diff = s - goal;
  if (cta == 0 && tid == 0) {
    out4[0] = (float)s;
    out4[1] = (float)(l1 * diff + l2 * diff * diff);
    out4[2] = (float)diff;
    out4[3] = (float)(diff * diff);
  }
  if (dlog_alpha) {
    const double coef = size_sum > 0.0 ? (l1 + 2.0 * l2 * diff) / size_sum : 0.0;
    auto gradient = [&](float alpha, float w) {
      const float e = __expf(-fabsf(alpha - thr)), q = __fdividef(1.0f, 1.0f + e);   // as in l0_chunk_kernel<true>
      return w * e * q * q;
    };
    l0_for_pieces(seg_off, seg_size, n_seg, s0, pos, end, lane, [&](int, int lo, int hi, float size) {
      const float w = (float)(coef * (double)size);
#pragma unroll 4
      for (int j = lo; j < hi; ++j) dlog_alpha[j] += gradient(log_alpha[j], w);
    }, [&](int, int, int, int lo, int hi, float size) {
      const float w = (float)(coef * (double)size);
#pragma unroll
      for (int i = 0; i < STEPS; ++i) {
        const int j = pos + 32 * i + lane;
        if (j >= lo && j < hi) dlog_alpha[j] += gradient(a[i], w);
      }
    });
  }
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

}  // namespace flop
