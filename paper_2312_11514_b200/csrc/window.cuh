// Pieces of the window bookkeeping shared by the window kernels (window.cu) and the single-launch
// decode step (step.cu).
#pragma once

#include "lif_internal.cuh"

namespace lif {

// Three counters ride in one 64-bit scan, 21 bits each (d_ff < 2^21 is checked at creation).
typedef unsigned long long u64;
constexpr int kField = 21;
constexpr u64 kFieldMask = (1ull << kField) - 1;
__device__ __forceinline__ u64 pack3(int a, int b, int c) {
  return (u64)a | ((u64)b << kField) | ((u64)c << (2 * kField));
}
__device__ __forceinline__ int field(u64 v, int i) { return (int)((v >> (i * kField)) & kFieldMask); }

template <int kT>
struct Scan {
  u64 warp_sums[kT / 32];
};

// exclusive prefix of v over the block (thread order); *total = block sum
template <int kT>
__device__ __forceinline__ u64 block_scan(u64 v, u64* total, Scan<kT>& sc) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  u64 inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    u64 n = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += n;
  }
  if (lane == 31) sc.warp_sums[warp] = inc;
  __syncthreads();
  u64 ws = lane < kT / 32 ? sc.warp_sums[lane] : 0ull;
  u64 winc = ws;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    u64 n = __shfl_up_sync(0xffffffffu, winc, o);
    if (lane >= o) winc += n;
  }
  const u64 base = __shfl_sync(0xffffffffu, winc - ws, warp);
  *total = __shfl_sync(0xffffffffu, winc, 31);
  __syncthreads();
  return base + inc - v;
}

struct WindowArgs {
  const int32_t* act;
  const int32_t* n_act;
  int32_t* counts;
  int32_t *pointers, *slot_of, *last_active;
  __half* bias;
  const __half* bias_up;
  int32_t *active_idx, *evict_ids, *evict_slots, *move_src, *move_dst, *load_ids, *load_slots,
      *active_slots, *hit_slots;
  int F, cap, k;
  int budget;             // 0 = off; else rows the cache may hold (Appendix C memory budget)
  // Speculative decoding (Section 4): the step holds consecutive tokens; the kept window ends
  // with token `keep` of the step (keep = 1, keep_tok = nullptr: ordinary single-token update).
  const int8_t* keep_tok; // [F] last kept token per neuron, -1 if active only in later tokens
  int keep;
  int append_first;       // stack the new neurons before deleting (see the header of this file)
  int release_early;      // release the dependent kernel before this kernel's own wait
  unsigned long long bundle_bytes;
};

// Stamp of an active neuron: the time of the last kept token in which it is active (its old
// stamp if it is active only beyond the kept token), but never below the oldest stamp still
// inside the window that ends at t_end: this step does not delete it, the next one may.
__device__ __forceinline__ int active_stamp(const WindowArgs& a, int id, int t, int t_end) {
  if (!a.keep_tok) return t;
  const int j = a.keep_tok[id];
  return max(j >= 0 ? t + j : a.last_active[id], t_end - a.k + 1);
}

WindowArgs window_args(lif_layer* L, const int32_t* act, const int32_t* n_act);

// Memory-budgeted window (Appendix C, Persimmon 8B / Phi-2): hist[a] = cached rows that are not
// active now and were last active a steps ago (a = 1 .. k, older ones in bin k).  Returns the
// widest window k' <= k for which the rows kept plus the rows to load fit `limit`, at least 1.
constexpr int kMaxBudgetWindow = 32;
__device__ __forceinline__ int widest_window_that_fits(const int* hist, int k, int n, int n_load,
                                                       int limit) {
  int evicted = 0;          // rows deleted under window kk = sum of hist[a], a >= kk
  int kk = k;
  for (; kk >= 1; --kk) {
    evicted += hist[kk];
    if (n - evicted + n_load <= limit) break;
  }
  return kk < 1 ? 1 : kk;
}

}  // namespace lif
