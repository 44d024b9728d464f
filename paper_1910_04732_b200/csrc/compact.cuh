// Deterministic inference mask and rank compaction (Sections 4.4 and 4.1).
//
// Ranks up to kFusedMaxR with P up to kFusedMaxBytes: compact_fused_kernel does all of the following in one launch.  Else:
//   compact_select_kernel : one block.  mode 0: pi_j in fp64, k = floor(sum pi + 1/2),
//       exact top-k of log_alpha by a 4-pass radix select on order-preserving
//       keys (ties -> lower index), then a block scan (warp shuffles) that
//       writes the ascending index list.  mode 1: keep z_j > 0.
//   gather_q_kernel : Qc[c, :] = z[idx[c]] * Q[idx[c], :]   (row gather, 16-byte vectors)
//   gather_p_kernel : Pc[i, c] = P[i, idx[c]]  (each P row is read once, coalesced,
//       into shared memory and the surviving columns are written out coalesced)
#pragma once
#include <float.h>

#include "common.cuh"

namespace flop {

constexpr int kSelThreads = 1024;

__device__ __forceinline__ uint32_t order_key(float a) {
  a += 0.0f;  // -0 -> +0 so that equal values have equal keys
  const uint32_t b = __float_as_uint(a);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

__global__ void __launch_bounds__(kSelThreads)
compact_select_kernel(const float* __restrict__ in, int mode, double thr, int r, int32_t* __restrict__ idx,
                      int32_t* __restrict__ k_dev, float* __restrict__ z_det) {
  pdl_wait();
  pdl_launch_dependents();
  __shared__ double red[32];
  __shared__ int hist[256];
  __shared__ int scan_scratch[33];
  __shared__ uint32_t s_prefix;
  __shared__ int s_need;
  const int tid = threadIdx.x;
  int k = 0;
  uint32_t kth = 0;   // key of the k-th largest gate
  int need_eq = 0;    // how many gates with key == kth are kept (lowest indices first)
  if (mode == 0) {
    double sum = 0.0;
    for (int j = tid; j < r; j += kSelThreads) sum += 1.0 / (1.0 + exp(-((double)in[j] - thr)));
    sum = block_sum_f64(sum, red);
    k = (int)floor(sum + 0.5);
    k = max(0, min(r, k));
    if (k > 0) {
      // radix select, most significant byte first
      uint32_t prefix = 0, pmask = 0;
      int need = k;   // rank (1-based, from the top) still to be located inside the prefix class
      for (int pass = 0; pass < 4; ++pass) {
        const int shift = 24 - 8 * pass;
        if (tid < 256) hist[tid] = 0;
        __syncthreads();
        for (int j = tid; j < r; j += kSelThreads) {
          const uint32_t key = order_key(in[j]);
          if ((key & pmask) == prefix) atomicAdd(&hist[(key >> shift) & 255], 1);
        }
        __syncthreads();
        {
          // the bin that holds the need-th largest key: a block scan over the bins from the top (thread t holds bin
          // 255 - t), instead of one thread walking 256 counters
          const int h = tid < 256 ? hist[255 - tid] : 0;
          int tot = 0;
          const int above = block_exclusive_scan(h, scan_scratch, &tot);
          if (tid < 256 && above < need && need <= above + h) {
            s_prefix = prefix | ((uint32_t)(255 - tid) << shift);
            s_need = need - above;
          }
        }
        __syncthreads();
        prefix = s_prefix;
        need = s_need;
        pmask |= 255u << shift;
        __syncthreads();
      }
      kth = prefix;
      need_eq = need;
    }
  }
  // ordered scan over the gates: running count of kept gates and of ties seen
  int base_keep = 0, base_eq = 0;
  for (int j0 = 0; j0 < r; j0 += kSelThreads) {
    const int j = j0 + tid;
    float v = 0.f;
    int eq = 0, gt = 0;
    if (j < r) {
      v = in[j];
      if (mode == 0) {
        const uint32_t key = order_key(v);
        gt = (k > 0) && key > kth;
        eq = (k > 0) && key == kth;
      } else {
        gt = v > 0.f;
      }
    }
    int tot_eq = 0, tot_keep = 0;
    const int rank_eq = mode == 0 ? base_eq + block_exclusive_scan(eq, scan_scratch, &tot_eq) : 0;
    const int keep = gt || (eq && rank_eq < need_eq);
    const int pos = base_keep + block_exclusive_scan(keep, scan_scratch, &tot_keep);
    if (j < r) {
      if (keep) idx[pos] = j;
      if (z_det) {
        float zv = 0.f;
        if (keep) zv = mode == 0 ? (float)(1.0 / (1.0 + exp(-((double)v - thr)))) : v;
        z_det[j] = zv;
      }
    }
    base_eq += tot_eq;
    base_keep += tot_keep;
  }
  if (tid == 0) *k_dev = base_keep;
}

// 16-byte vector of elements
template <typename T> struct Vec16 { static constexpr int n = 16 / sizeof(T); };

template <typename T>
__global__ void __launch_bounds__(256)
gather_q_kernel(const T* __restrict__ Q, int64_t ldq, const int32_t* __restrict__ idx, const int32_t* __restrict__ k_dev,
                const float* __restrict__ z, int d_in, T* __restrict__ Qc, int64_t ldqc, int vec_ok) {
  pdl_wait();
  pdl_launch_dependents();
  const int c = blockIdx.x;
  if (c >= *k_dev) return;
  const int src = idx[c];
  const float g = z[src];
  const T* q = Q + (int64_t)src * ldq;
  T* o = Qc + (int64_t)c * ldqc;
  constexpr int V = Vec16<T>::n;
  if (vec_ok) {
    for (int j = threadIdx.x * V; j < d_in; j += blockDim.x * V) {
      if (j + V <= d_in) {
        uint4 raw = *reinterpret_cast<const uint4*>(q + j);
        T* e = reinterpret_cast<T*>(&raw);
#pragma unroll
        for (int i = 0; i < V; ++i) e[i] = from_f32<T>(to_f32<T>(e[i]) * g);
        *reinterpret_cast<uint4*>(o + j) = raw;
      } else {
        for (int i = j; i < d_in; ++i) o[i] = from_f32<T>(to_f32<T>(q[i]) * g);
      }
    }
  } else {
    for (int j = threadIdx.x; j < d_in; j += blockDim.x) o[j] = from_f32<T>(to_f32<T>(q[j]) * g);
  }
}

// One block per kRows rows of P; a row (r elements) is staged in shared memory.
template <typename T>
__global__ void __launch_bounds__(256)
gather_p_kernel(const T* __restrict__ P, int64_t ldp, const int32_t* __restrict__ idx, const int32_t* __restrict__ k_dev,
                int r, int d_out, T* __restrict__ Pc, int64_t ldpc, int rows_per_block, int vec_ok) {
  pdl_wait();
  pdl_launch_dependents();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* row = reinterpret_cast<T*>(smem_raw);
  const int k = *k_dev;
  constexpr int V = Vec16<T>::n;
  for (int rr = 0; rr < rows_per_block; ++rr) {
    const int i = blockIdx.x * rows_per_block + rr;
    if (i >= d_out) return;
    const T* p = P + (int64_t)i * ldp;
    if (vec_ok) {
      for (int j = threadIdx.x * V; j < r; j += blockDim.x * V) {
        if (j + V <= r) *reinterpret_cast<uint4*>(row + j) = *reinterpret_cast<const uint4*>(p + j);
        else for (int e = j; e < r; ++e) row[e] = p[e];
      }
    } else {
      for (int j = threadIdx.x; j < r; j += blockDim.x) row[j] = p[j];
    }
    __syncthreads();
    T* o = Pc + (int64_t)i * ldpc;
    // four surviving columns per thread and store where the element type and the alignment allow it
    // (8-byte stores, 256 bytes per warp instruction), single elements otherwise
    if (sizeof(T) == 2 && (reinterpret_cast<uintptr_t>(o) & 7) == 0 && (reinterpret_cast<uintptr_t>(idx) & 15) == 0) {
      for (int c = threadIdx.x * 4; c < k; c += blockDim.x * 4) {
        if (c + 3 < k) {
          const int4 ii = *reinterpret_cast<const int4*>(idx + c);
          T quad[4] = {row[ii.x], row[ii.y], row[ii.z], row[ii.w]};
          *reinterpret_cast<uint2*>(o + c) = *reinterpret_cast<uint2*>(quad);
        } else {
          for (int e = c; e < k; ++e) o[e] = row[idx[e]];
        }
      }
    } else {
      for (int c = threadIdx.x; c < k; c += blockDim.x) o[c] = row[idx[c]];
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------------------------
// P gather with the rows staged by bulk asynchronous copies (bf16, rows of a multiple of 16 bytes).
//
// A block walks groups of `rows_per_stage` consecutive rows of P.  One thread hands the rows of the
// next groups to the copy engine (cp.async.bulk global -> shared, completion counted in bytes on an
// mbarrier per buffer) while all threads pick the surviving columns of the current group out of
// shared memory and write them as 8-byte pieces, so the read of P is fully coalesced, needs no
// registers or load instructions, and overlaps the select/store phase of the same block.  The
// index list is kept in shared memory as 16-bit entries (r <= 65536).  Waits are bounded: when one
// gives up, the block records FLOP_ERR_TIMEOUT, lets the copies in flight land (bounded) and returns.
namespace gp {
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void bar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void bar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool bar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
// 16-byte aligned source and destination, size a multiple of 16 bytes
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
constexpr long long kWaitCycles = 2000000000LL;   // ~1 s
}  // namespace gp

constexpr int kGatherMaxBuf = 4;

__global__ void __launch_bounds__(256)
gather_p_pipe_kernel(const __nv_bfloat16* __restrict__ P, int64_t ldp, const int32_t* __restrict__ idx,
                     const int32_t* __restrict__ k_dev, int r, int d_out, __nv_bfloat16* __restrict__ Pc, int64_t ldpc,
                     int rows_per_stage, int nbuf) {
  pdl_wait();
  pdl_launch_dependents();
  extern __shared__ __align__(16) unsigned char smem_raw[];   // every offset used below is a multiple of 16
  __shared__ int s_abort;
  const int k = min(*k_dev, r);
  if (k <= 0) return;
  const uint32_t row_bytes = (uint32_t)r * 2u;                     // multiple of 16 (checked by the host)
  const uint32_t stage_bytes = row_bytes * (uint32_t)rows_per_stage;
  unsigned long long* bars = reinterpret_cast<unsigned long long*>(smem_raw);            // nbuf barriers (64 bytes reserved)
  unsigned short* sidx = reinterpret_cast<unsigned short*>(smem_raw + 64);               // r entries
  unsigned char* bufs = smem_raw + 64 + (((size_t)r * 2 + 127) & ~(size_t)127);          // nbuf stages
  const int n_groups = (d_out + rows_per_stage - 1) / rows_per_stage;
  const int n_mine = (int)blockIdx.x < n_groups ? (n_groups - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
  if (n_mine == 0) return;

  auto issue = [&](int it) {   // thread 0: hand the rows of this block's it-th group to the copy engine
    const int b = it % nbuf;
    const int row0 = ((int)blockIdx.x + it * (int)gridDim.x) * rows_per_stage;
    const int rows = min(rows_per_stage, d_out - row0);
    const uint32_t bar = gp::smem_addr(&bars[b]);
    gp::bar_expect_tx(bar, row_bytes * (uint32_t)rows);
    for (int j = 0; j < rows; ++j)
      gp::bulk_load(gp::smem_addr(bufs + (size_t)b * stage_bytes + (size_t)j * row_bytes), P + (int64_t)(row0 + j) * ldp, row_bytes, bar);
  };

  if (threadIdx.x == 0) {
    s_abort = 0;
    for (int b = 0; b < nbuf; ++b) gp::bar_init(gp::smem_addr(&bars[b]), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    for (int it = 0; it < min(nbuf, n_mine); ++it) issue(it);
  }
  for (int c = threadIdx.x; c < k; c += blockDim.x) sidx[c] = (unsigned short)idx[c];
  __syncthreads();

  const int kq = (k + 3) >> 2;   // 4-column pieces per row
  const bool vec_out = (reinterpret_cast<uintptr_t>(Pc) & 7) == 0 && (ldpc & 3) == 0;
  int issued = min(nbuf, n_mine);
  for (int it = 0; it < n_mine; ++it) {
    const int b = it % nbuf;
    const uint32_t parity = (uint32_t)(it / nbuf) & 1u;
    const uint32_t bar = gp::smem_addr(&bars[b]);
    if (!gp::bar_try_wait(bar, parity)) {
      const long long t0 = clock64();
      while (!gp::bar_try_wait(bar, parity)) {
        if (*(volatile int*)&s_abort) break;
        if (clock64() - t0 > gp::kWaitCycles) { *(volatile int*)&s_abort = 1; report_timeout(); break; }
      }
    }
    if (__syncthreads_or(s_abort)) break;   // every thread takes the same decision
    const int row0 = ((int)blockIdx.x + it * (int)gridDim.x) * rows_per_stage;
    const int rows = min(rows_per_stage, d_out - row0);
    const __nv_bfloat16* stage = reinterpret_cast<const __nv_bfloat16*>(bufs + (size_t)b * stage_bytes);
    for (int w = threadIdx.x; w < rows * kq; w += blockDim.x) {
      const int j = w / kq, c = (w - j * kq) << 2;
      const __nv_bfloat16* row = stage + (size_t)j * r;
      __nv_bfloat16* o = Pc + (int64_t)(row0 + j) * ldpc + c;
      if (c + 3 < k && vec_out) {
        const uint2 ii = *reinterpret_cast<const uint2*>(sidx + c);   // four 16-bit indices
        const unsigned short q0 = __bfloat16_as_ushort(row[ii.x & 0xFFFFu]), q1 = __bfloat16_as_ushort(row[ii.x >> 16]);
        const unsigned short q2 = __bfloat16_as_ushort(row[ii.y & 0xFFFFu]), q3 = __bfloat16_as_ushort(row[ii.y >> 16]);
        __stcs(reinterpret_cast<uint2*>(o), make_uint2((uint32_t)q0 | ((uint32_t)q1 << 16), (uint32_t)q2 | ((uint32_t)q3 << 16)));
      } else {
        for (int e = c; e < min(c + 4, k); ++e) o[e - c] = row[sidx[e]];
      }
    }
    __syncthreads();   // the buffer has been read by everyone: it may be refilled
    if (threadIdx.x == 0 && issued < n_mine) issue(issued);
    if (issued < n_mine) ++issued;
  }
  if (s_abort && threadIdx.x == 0) {
    // leaving early: give the copies already issued time to land so that nothing writes this block's
    // shared memory after it has gone
    const long long t0 = clock64();
    while (clock64() - t0 < 2000000LL) {}
  }
}

// ---------------------------------------------------------------------------------------------
// Selection and both gathers in one launch.
//
// Bound: latency.  The factors of one matrix are 1-10 MB (0.2-1.5 us of memory time), but the selection is a chain
// of dependent steps, and as a launch of its own (one block of 1024 threads, 13 us) it kept 147 SMs waiting.  Here
// every block repeats the selection in its own shared memory -- r gates are 4 KB, L2-resident after the first block --
// and goes straight on to its rows.  What makes the repetition cheap: gates stay in registers (kKeys per thread), ordinary
// gates need no fp64 and one histogram (select_largest), and positions come from ballots and a scan
// of the 32 words by every warp.  The fp64 probabilities are evaluated only where they are results: one per row of Q_c, by the warp
// that scales it and writes it to z_det (a pass over z_det at the end of the block cost 850 cycles of about 8000).
// A warp then takes one row at a time: P rows first (their number is known before the selection, so the rows are
// prefetched into L2 while the previous launch on the stream still runs, and the warp's first one is staged in shared memory
// during the selection), then the surviving rows of Q in pieces of at most
// kFusedPiece elements (a warp per whole row took 45 us for 400 rows of 30 000 bf16, the gather in its own launch 23 with
// the selection, and in pieces it takes 16).  Surviving columns of further rows of P are read straight from global memory, two
// per lane: neighbouring lanes read neighbouring survivors, so a load touches only a few lines.
// Measured, the 72 matrices of a BERT-base-shaped model: three launches each 1364 us (13.0 + 4.0 + 5.8 us of GPU time per matrix);
// one launch with four histogram passes and all probabilities in fp64 643-694 us; this form 383 us, with clamped gates 400, all equal 448.
// Against an earlier form of it that took 423: two blocks per SM, which repeat the selection twice, 444 (66 MB of factors, r = 1021:
// 257 against 270); one block of 1024 threads 455 (longer barriers); held to 40 or 32 registers, so that more of the next
// launch's blocks could be resident early, 578 and 782 us (spills in the chain).
// Ranks up to 1024: two gates per thread and a word per lane.  With four (the former selection) repeating it cost more than the
// launches it saves (2048 -> 6144 at r = 2048: 37.5 against 28.6 us; 4096 x 4096 x 16384: 127 against 74).  P up to 16 MB: for long P
// the staged gather above streams better.  The line was drawn for the former selection; with this one, us, one launch / three:
// 1024 x 4096 bf16 8.1 / 20.9, at the line 1024 x 8192 14.1 / 24.0, beyond it 1024 x 16 384 26.8 / 30.5, 1024 x 40 000 65.5 / 44.0.
constexpr int kFusedMaxR = 1024;
constexpr int64_t kFusedMaxBytes = 16 << 20;
constexpr int kFusedPiece = 4096;
inline int fused_pieces(int64_t d_in) { return (int)((d_in + kFusedPiece - 1) / kFusedPiece); }   // of a row of Q
constexpr int kFusedThreads = 512, kFusedWarps = kFusedThreads / 32;

template <typename T> struct alignas(2 * sizeof(T)) Pair2 { T e[2]; };

constexpr int kKeys = kFusedMaxR / kFusedThreads;   // gates per thread
constexpr int kFusedWords = kKeys * kFusedWarps;    // 32-gate words, one per lane of a warp that scans them
static_assert(kFusedWords == 32, "a warp scans all words at once");
constexpr int kFineBins = 1024, kCloseGates = 64;
constexpr double kFastThr = 1 << 20;    // largest |thr| for which k is taken from fp32 probabilities
// Shared memory for one row of P per warp, staged while the selection runs.
template <typename T> __host__ __device__ constexpr size_t fused_row_bytes(int64_t r) { return ((size_t)r * sizeof(T) + 15) & ~(size_t)15; }

// Exclusive prefix of `count` over the lanes and, in *total, the sum.
__device__ __forceinline__ int warp_exclusive_scan(int count, int lane, int* total) {
  int inc = count;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int up = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += up;
  }
  *total = __shfl_sync(0xffffffffu, inc, 31);
  return inc - count;
}
// The bin among 32, counted from lane 0 up, that holds item `need` (1-based); *need becomes its rank inside the bin.
// -1 when there are fewer items.
__device__ __forceinline__ int warp_find(int count, int lane, int* need) {
  int total;
  const int before = warp_exclusive_scan(count, lane, &total);
  const unsigned who = __ballot_sync(0xffffffffu, before < *need && *need <= before + count);
  const int at = who ? __ffs(who) - 1 : 0;
  *need -= __shfl_sync(0xffffffffu, before, at);
  return who ? at : -1;
}

struct FusedShared {
  __align__(16) int hist[kFineBins];
  int coarse[32];
  unsigned long long close[kCloseGates];
  double red[kFusedWarps];
  uint32_t lo[kFusedWarps], hi[kFusedWarps], fixed[kFusedWarps], words[kFusedWords];
  int n_close;
  __align__(16) unsigned short idx[kFusedMaxR];
  float v[kFusedMaxR];
};

// P(z > 0) as the deterministic gate, evaluated in fp64 (out of line: it is needed once per row and must not cost the kernel registers).
__device__ __noinline__ float probability(float a, double thr) { return (float)(1.0 / (1.0 + exp(-((double)a - thr)))); }

// k = floor(sum of the probabilities + 1/2) from fp64 probabilities.
__device__ __noinline__ int count_f64(FusedShared& sh, float v0, float v1, double thr, int r) {
  static_assert(kKeys == 2, "two gates per thread");
  const int tid = threadIdx.x, lane = tid & 31;
  double sum = 0.0;
  if (tid < r) sum += 1.0 / (1.0 + exp(-((double)v0 - thr)));
  if (kFusedThreads + tid < r) sum += 1.0 / (1.0 + exp(-((double)v1 - thr)));
  sum = warp_sum_f64(sum);
  if (lane == 0) sh.red[tid >> 5] = sum;
  __syncthreads();
  sum = warp_sum_f64(lane < kFusedWarps ? sh.red[lane] : 0.0);
  return max(0, min(r, (int)floor(sum + 0.5)));
}

__device__ __forceinline__ float key_value(uint32_t key) { return __uint_as_float((key & 0x80000000u) ? key ^ 0x80000000u : ~key); }

// One step towards the `need` largest of the active gates (bit n: gate n of this thread), whose keys lie in lo .. hi: they are counted
// in 1024 bins, linear in the gate or in its key (both monotone; in fp32 arithmetic too, and with infinities in the end bins).  Gates
// above the bin of the cut are kept, those of the bin stay active; up to kCloseGates of them are ranked against one another
// on (value, lower index first).  True when all is decided.  The bins and n_close are zero before.
__device__ __forceinline__ bool cut_pass(FusedShared& sh, const float (&v)[kKeys], unsigned& active, unsigned& keep, int& need, uint32_t lo,
                                         uint32_t hi, bool linear) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const float low = key_value(lo), scale = (kFineBins - 0.25f) / (key_value(hi) - low);
  const int shift = max(0, 32 - __clz(hi - lo) - 10);
  static_assert(kFineBins == 1 << 10, "ten bits of the keys' differences");
  int bin[kKeys];      // counted from the largest gate down
#pragma unroll
  for (int n = 0; n < kKeys; ++n) {
    const int up = linear ? (int)((v[n] - low) * scale) : (int)((order_key(v[n]) - lo) >> shift);
    bin[n] = kFineBins - 1 - max(0, min(kFineBins - 1, up));
    if ((active >> n) & 1u) atomicAdd(&sh.hist[bin[n]], 1);
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 32 / kFusedWarps; ++i) {
    const int c = warp * (32 / kFusedWarps) + i, sum = __reduce_add_sync(0xffffffffu, sh.hist[32 * c + lane]);
    if (lane == 0) sh.coarse[c] = sum;
  }
  __syncthreads();
  const int c = warp_find(sh.coarse[lane], lane, &need), cut = 32 * c + warp_find(sh.hist[32 * c + lane], lane, &need), count = sh.hist[cut];
  const bool all = need == count;      // the cut falls between two bins
#pragma unroll
  for (int n = 0; n < kKeys; ++n) {
    if (!((active >> n) & 1u)) continue;
    if (bin[n] < cut || (all && bin[n] == cut)) keep |= 1u << n;
    if (bin[n] != cut) active &= ~(1u << n);
    else if (!all && count <= kCloseGates) sh.close[atomicAdd(&sh.n_close, 1)] = ((unsigned long long)order_key(v[n]) << 32) | (0xffffffffu - (uint32_t)(n * kFusedThreads + tid));
  }
  if (all) return true;
  if (count > kCloseGates) return false;
  __syncthreads();
#pragma unroll
  for (int n = 0; n < kKeys; ++n)
    if ((active >> n) & 1u) {
      const unsigned long long mine = ((unsigned long long)order_key(v[n]) << 32) | (0xffffffffu - (uint32_t)(n * kFusedThreads + tid));
      int rank = 0;
#pragma unroll 8
      for (int i = 0; i < count; ++i) rank += sh.close[i] > mine;
      if (rank < need) keep |= 1u << n;
    }
  return true;
}

// The rest of the decision for many active gates close together or equal: bins between their own extremes, linear once and then on
// the keys, whose range shrinks by 2^10 a pass, until the gates left are few or equal; of equal ones the lowest indices are kept.
// Such gates are no exception (all equal after initialisation, two classes after clamping, one gate that ran away).  768 -> 768
// at r = 768, us, ordinary gates 4.4: clamped 4.65, all equal 4.8, an outlier 5.4, a sum next to a half (count_f64) 4.9.  A selection
// from the start for them (fp64 probabilities and four passes over the bits, after the attempt at the short way) took 8.7, 9.3, 9.1
// and 8.2, more than before there was a short way at small ranks (256 -> 768: clamped 7.7 against 5.4, now 3.9).
__device__ __noinline__ unsigned cut_again(FusedShared& sh, float v0, float v1, unsigned active, int need) {
  const float v[kKeys] = {v0, v1};
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  unsigned keep = 0;
#pragma unroll 1
  for (bool linear = true;; linear = false) {
    uint32_t lo = 0xffffffffu, hi = 0u;
#pragma unroll
    for (int n = 0; n < kKeys; ++n)
      if ((active >> n) & 1u) { lo = min(lo, order_key(v[n])); hi = max(hi, order_key(v[n])); }
    lo = __reduce_min_sync(0xffffffffu, lo); hi = __reduce_max_sync(0xffffffffu, hi);
    __syncthreads();     // the bins and extremes of the pass before have been read
    if (lane == 0) { sh.lo[warp] = lo; sh.hi[warp] = hi; }
    for (int i = tid; i < kFineBins; i += kFusedThreads) sh.hist[i] = 0;
    __syncthreads();
    lo = __reduce_min_sync(0xffffffffu, sh.lo[lane % kFusedWarps]);
    hi = __reduce_max_sync(0xffffffffu, sh.hi[lane % kFusedWarps]);
    if (lo == hi) break;
    if (cut_pass(sh, v, active, keep, need, lo, hi, linear && fabsf(key_value(lo)) <= FLT_MAX && fabsf(key_value(hi)) <= FLT_MAX)) return keep;
  }
#pragma unroll
  for (int n = 0; n < kKeys; ++n) {
    const uint32_t word = __ballot_sync(0xffffffffu, (active >> n) & 1u);
    if (lane == 0) sh.words[n * kFusedWarps + warp] = word;
  }
  __syncthreads();
  const uint32_t word = sh.words[lane];
  int total;
  const int before = warp_exclusive_scan(__popc(word), lane, &total);
#pragma unroll
  for (int n = 0; n < kKeys; ++n) {
    const int w = n * kFusedWarps + warp;
    const int rank = __shfl_sync(0xffffffffu, before, w) + __popc(__shfl_sync(0xffffffffu, word, w) & ((1u << lane) - 1u));
    if (((active >> n) & 1u) && rank < need) keep |= 1u << n;
  }
  __syncthreads();   // the words are written again
  return keep;
}

// Which of this thread's gates are among the k = floor(sum of probabilities + 1/2) largest (bit n of the result: gate n).
//   k: probabilities p = 1 / (1 + e^x), x = thr - v, in fp32, added as 20-bit fixed point (order-free, one instruction per warp).  thr
//      comes as the sum of two floats: rounded to one it would move every x the same way, by up to 2^-25 |thr| (at beta = 100 and gates
//      near thr 2000 units for 1024 gates).  As (hi - v) + lo, x is off by 2^-23 |x|, and by less than 2^-27 up to kFastThr.  In
//      units of 2^-20 that is at most 0.03 + 0.01 of p; __expf, good to 2 + 1.173 |x| units in its last place, adds 0.08, the sum
//      1 + e^x 0.07 and the quotient, two units in its last place, 0.25: with the half unit of rounding a gate is off by less than
//      one, the sum by less than r, and floor(sum + 1/2) is that of fp64 unless the sum lies within r + 16 units of a half.  Only
//      then, and beyond kFastThr, the fp64 probabilities are evaluated.
//   k-th largest: bins between the smallest and the largest finite gate, and again between the gates of the cut's bin while those are
//      many (a class of equal gates, a distant gate that stretches the bins).
__device__ __forceinline__ unsigned select_largest(FusedShared& sh, const float (&v)[kKeys], double thr, int r) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const float thr_hi = (float)thr, thr_lo = (float)(thr - (double)thr_hi);
  uint32_t lo = 0xffffffffu, hi = 0u, fixed = 0u;
  unsigned active = 0, keep = 0;
#pragma unroll
  for (int n = 0; n < kKeys; ++n)
    if (n * kFusedThreads + tid < r) {
      const uint32_t key = order_key(v[n]);
      active |= 1u << n;
      if (fabsf(v[n]) <= FLT_MAX) { lo = min(lo, key); hi = max(hi, key); }
      if (v[n] != v[n]) hi = 0xffffffffu;     // NaN: the key of no finite gate
      fixed += __float2uint_rn(__fdividef(1048576.f, 1.f + __expf((thr_hi - v[n]) + thr_lo)));
    }
  lo = __reduce_min_sync(0xffffffffu, lo); hi = __reduce_max_sync(0xffffffffu, hi); fixed = __reduce_add_sync(0xffffffffu, fixed);
  if (lane == 0) { sh.lo[warp] = lo; sh.hi[warp] = hi; sh.fixed[warp] = fixed; }
  __syncthreads();     // (the bins are zero by now as well)
  lo = __reduce_min_sync(0xffffffffu, sh.lo[lane % kFusedWarps]);
  hi = __reduce_max_sync(0xffffffffu, sh.hi[lane % kFusedWarps]);
  fixed = __reduce_add_sync(0xffffffffu, lane < kFusedWarps ? sh.fixed[lane] : 0u) + (1u << 19);
  if (hi == 0xffffffffu) return 0;            // the sum is NaN, which counts as none
  const uint32_t part = fixed & 0xfffffu, margin = (uint32_t)r + 16u;
  const bool sure = fabs(thr) <= kFastThr && part > margin && part < 0x100000u - margin;
  int need = sure ? min(r, (int)(fixed >> 20)) : count_f64(sh, v[0], v[1], thr, r);
  if (need == 0) return 0;
  if (!cut_pass(sh, v, active, keep, need, lo, hi, true)) keep |= cut_again(sh, v[0], v[1], active, need);
  return keep;
}

template <typename T>
__global__ void __launch_bounds__(kFusedThreads, 1)
compact_fused_kernel(const float* __restrict__ in, int mode, double thr, int r, int32_t* __restrict__ idx, int32_t* __restrict__ k_dev,
                     float* __restrict__ z_det, const T* __restrict__ P, int64_t ldp, const T* __restrict__ Q, int64_t ldq, int d_in,
                     int d_out, T* __restrict__ Pc, int64_t ldpc, T* __restrict__ Qc, int64_t ldqc, int vec_q, int vec_p, int pair_p, int pieces) {
  __shared__ FusedShared sh;
  extern __shared__ __align__(16) unsigned char rows[];      // [kFusedWarps][fused_row_bytes]
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int warps = (int)gridDim.x * kFusedWarps, my_warp = (int)blockIdx.x * kFusedWarps + warp;
  T* my_row = reinterpret_cast<T*>(rows + warp * fused_row_bytes<T>(r));
  // a hint only: nothing is read before the wait below.  Which rows of Q survive is not known yet; all of them are asked for (what
  // is read of them came from HBM at the end of the chain).  us, without / with, 4096 columns at r = 1024 with 1024 rows of P: 90 % of
  // the gates open bf16 8.6 / 7.0, fp32 12.6 / 11.6; 30 % 8.1 / 7.1, 11.1 / 10.2; 5 % 7.3 / 7.3, 10.4 / 10.0; 0.5 % 7.1 / 7.3, 9.9 / 10.3; the
  // most it can cost, 0.5 % of 16 MB of Q and 64 rows of P: 9.4 / 10.5
  auto prefetch = [&](const T* m, int64_t ld, int n, int cols) {
    for (int i = my_warp; i < n; i += warps)
      for (int64_t b = lane * 128; b < cols * (int64_t)sizeof(T); b += 32 * 128)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<const char*>(m + (int64_t)i * ld) + b));
  };
  if (warp == 0 && lane * 32 < r) asm volatile("prefetch.global.L2 [%0];" ::"l"(in + lane * 32));      // the gates: 128 bytes a lane
  prefetch(P, ldp, d_out, r);
  if (pieces == 1 && d_in > 0) prefetch(Q, ldq, r, d_in);
  for (int i = tid; i < kFineBins; i += kFusedThreads) sh.hist[i] = 0;
  if (tid == 0) sh.n_close = 0;
  pdl_wait();
  pdl_launch_dependents();

  // gate n of this thread is n * kFusedThreads + tid: word n * kFusedWarps + warp of the ballots, bit lane
  float v[kKeys];
#pragma unroll
  for (int n = 0; n < kKeys; ++n) v[n] = n * kFusedThreads + tid < r ? in[n * kFusedThreads + tid] : 0.f;
  // this warp's first row of P, known before the selection
  const bool staged = vec_p && my_warp < d_out;
  if (staged) {
    const unsigned char* src = reinterpret_cast<const unsigned char*>(P + (int64_t)my_warp * ldp);
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(my_row);
    const int bytes = r * (int)sizeof(T);
    for (int b = lane * 16; b < bytes; b += 32 * 16)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst + (uint32_t)b), "l"(src + b), "r"(min(16, bytes - b)) : "memory");
  }
  unsigned keep = 0;     // bit n: gate n of this thread survives
  if (mode == 0) {
    keep = select_largest(sh, v, thr, r);
  } else {
#pragma unroll
    for (int n = 0; n < kKeys; ++n)
      if (n * kFusedThreads + tid < r && v[n] > 0.f) keep |= 1u << n;
  }
#pragma unroll
  for (int n = 0; n < kKeys; ++n) {
    const uint32_t word = __ballot_sync(0xffffffffu, (keep >> n) & 1u);
    if (lane == 0) sh.words[n * kFusedWarps + warp] = word;
  }
  __syncthreads();
  int k;
  {
    const uint32_t word = sh.words[lane];
    const int before = warp_exclusive_scan(__popc(word), lane, &k);
#pragma unroll
    for (int n = 0; n < kKeys; ++n) {
      const int j = n * kFusedThreads + tid, w = n * kFusedWarps + warp;
      const int pos = __shfl_sync(0xffffffffu, before, w) + __popc(__shfl_sync(0xffffffffu, word, w) & ((1u << lane) - 1u));
      if ((keep >> n) & 1u) {
        sh.idx[pos] = (unsigned short)j;
        sh.v[pos] = v[n];
        if (blockIdx.x == 0) idx[pos] = j;
      }
    }
  }
  if (blockIdx.x == 0 && tid == 0) *k_dev = k;
  if (staged) asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();

  constexpr int V = Vec16<T>::n;
  const int piece = ((d_in + max(pieces, 1) - 1) / max(pieces, 1) + 63) & ~63;
  for (int t = my_warp; t < d_out + k * pieces; t += warps) {
    if (t < d_out) {                       // Pc[t, :] = P[t, idx]
      const T* p = staged && t == my_warp ? my_row : P + (int64_t)t * ldp;
      T* o = Pc + (int64_t)t * ldpc;
      if (pair_p) {
#pragma unroll 4
        for (int c = 2 * lane; c < k; c += 64) {
          if (c + 1 < k) {
            const uint32_t ii = *reinterpret_cast<const uint32_t*>(sh.idx + c);
            Pair2<T> two;
            two.e[0] = p[ii & 0xFFFFu];
            two.e[1] = p[ii >> 16];
            *reinterpret_cast<Pair2<T>*>(o + c) = two;
          } else {
            o[c] = p[sh.idx[c]];
          }
        }
      } else {
        for (int c = lane; c < k; c += 32) o[c] = p[sh.idx[c]];
      }
    } else {                               // Qc[c, :] = z[idx[c]] * Q[idx[c], :]
      const int c = (t - d_out) / pieces, j0 = (t - d_out - c * pieces) * piece, j1 = min(d_in, j0 + piece);
      const T* q = Q + (int64_t)sh.idx[c] * ldq;
      T* o = Qc + (int64_t)c * ldqc;
      const int full = vec_q ? j1 / V * V : j0;
      float g = 0.f;
      for (int j = j0 + lane * V, first = 1; first || j - lane * V < full; j += 4 * 32 * V, first = 0) {
        uint4 raw[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (j + u * 32 * V < full) raw[u] = *reinterpret_cast<const uint4*>(q + j + u * 32 * V);
        if (first) {                                       // while the first loads are on their way
          g = mode == 0 ? probability(sh.v[c], thr) : sh.v[c];
          if (z_det && j0 == 0 && lane == 0) z_det[sh.idx[c]] = g;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (j + u * 32 * V < full) {
            T* e = reinterpret_cast<T*>(&raw[u]);
#pragma unroll
            for (int i = 0; i < V; ++i) e[i] = from_f32<T>(to_f32<T>(e[i]) * g);
            *reinterpret_cast<uint4*>(o + j + u * 32 * V) = raw[u];
          }
      }
      for (int j = max(full, j0) + lane; j < j1; j += 32) o[j] = from_f32<T>(to_f32<T>(q[j]) * g);
    }
  }
  if (z_det) {       // the dropped gates, a few per block; the kept ones are written with their rows of Q (here when there are none)
#pragma unroll
    for (int n = 0; n < kKeys; ++n) {
      const int j = n * kFusedThreads + tid;
      const bool kept = (keep >> n) & 1u;
      if (j < r && j % (int)gridDim.x == (int)blockIdx.x && (!kept || pieces == 0)) z_det[j] = !kept ? 0.f : mode == 0 ? probability(v[n], thr) : v[n];
    }
  }
}

}  // namespace flop
