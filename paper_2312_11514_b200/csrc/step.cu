// One launch for everything of a decode step behind the predictor: window update,
// row moves, fetch of the new bundles, sparse FFN over cached and new rows, and the sum.
//
// The CTAs of the grid (one per SM) take parts of the step, in the order in which they start:
//   window CTA   (first)   the plan of Section 3.3: lists, counters and state, from the
//                          predictor's entries; publishes the plan with one flag
//   cache CTAs   (middle)  find the active rows that are already cached in the predictor's entries,
//                          add their FFN terms (bulk copies into shared memory, a warp per row); the
//                          plan's row moves
//   fetch CTAs   (then)    find the new neurons in the predictor's entries, bring their bundles over
//                          the host link through a ring of bulk copies, add their FFN terms from
//                          shared memory, copy them to their cache rows
//   sum CTAs     (last)    add up the partial sums
// The terms of the output wait for the predictor's entries only, which carry the row of every cached
// neuron; the plan (3 us behind them) is needed for the places of new and moved rows, and by the sum,
// which leaves the terms out when the update was refused.  With the terms behind the plan a token of two
// 512 x 2048 layers took 28.4 us, 26.6 now; eight of 4096 x 16384 386-391 us, 380-383 now.
// (The FFN over every cached row takes its rows from the plan.)
// x, like the window state, was complete before every kernel ahead of this one passed its own wait, so
// it is read (past L1) ahead of this kernel's wait, which comes 2-4 us behind the last entry where
// host reads are in flight.
// A CTA whose wait for the plan runs out moves or brings in nothing, although the window CTA commits the
// state that names those rows.  Like every wait that runs out it flags LIF_ERR_TIMEOUT, which refuses further
// updates, and it marks the rows as suspect, so that clearing the status reads them from the store again.
// A CTA waits only for CTAs that took their parts before it and are therefore running, so a step ends
// however few of its CTAs fit the chip at a time beside other streams' kernels; every wait is bounded,
// and every CTA makes its arrivals on all paths, so the counters are complete whatever happened.
//
// Why one launch: the parts run side by side without an event or a stream of their own (five
// launches and two event pairs less per layer-step), and the fetch does not wait for the window
// plan: it needs the plan only for the place of a bundle that has already arrived.
// Why few fetch CTAs: about 200 KB of host reads in flight fill the link (8 CTAs with two 16 KB
// copies each reach the same 49.8 GB/s as 148 CTAs).  More in flight does not read faster, it only
// queues up in front of everything else: with host loads in flight on all SMs a dependent load
// beside them takes 1800 cycles instead of 290, and an HBM stream of the whole chip falls from 3.6
// to 0.9 TB/s (2.7 TB/s with 32 CTAs and one copy each).
// Why 32 with all but one stage of the ring in flight, asked for when a row has landed and not when it
// is done with: the copies of one SM share its rate and land together, so with 16 CTAs and two wide
// rows each the last two rows were worked on one after the other behind the link.  Layers of 4544 and
// 768 columns 79 -> 77.7 and 16.2 -> 15.9 us, three streams at 1544 47.7 -> 46.7; 16 CTAs asked the
// same way lose 5% to the gap between a landing and the next request, 24 lose 2%.
#include <type_traits>

#include "lif_internal.cuh"
#include "mask_compact.cuh"
#include "window.cuh"

namespace lif {
namespace {

constexpr int kStepThreads = 512;
constexpr int kStepWarps = kStepThreads / 32;
constexpr int kEntriesPerThread = 2;                   // <= 1024 entries: d_ff <= 32768
constexpr int kStepWatchPolls = 64;                    // about 30 us
constexpr int kFetchCtas = 32;
constexpr unsigned short kNoSlot = 0xffff;

// Counters of the layer's steps.  They only grow: the ticket tells the step as well as the part, and
// what a CTA waits for is a counter's value after that many steps (modulo 2^32), so nothing has
// to be put back at the end.
struct StepSync {
  unsigned long long ticket;
  unsigned long long plan;       // step << 50 | flags | n_load << 32 | n_moves << 16 | rows for the cache CTAs
  unsigned groups_done;
  unsigned pad[11];
  unsigned group[64];            // arrivals of each group of cache CTAs
};
constexpr unsigned long long kPlanReady = 1ull << 48, kPlanRefused = 1ull << 49;
constexpr int kPlanEpochShift = 50;
constexpr unsigned kPlanEpochMask = (1u << 14) - 1;
__device__ __forceinline__ int plan_rows(unsigned long long v) { return (int)(v & 0xffff); }
__device__ __forceinline__ int plan_moves(unsigned long long v) { return (int)((v >> 16) & 0xffff); }
__device__ __forceinline__ int plan_loads(unsigned long long v) { return (int)((v >> 32) & 0xffff); }

struct StepArgs {
  WindowArgs w;
  const unsigned long long* new_entries;   // predictor: {neurons to bring in, run}
  const unsigned long long* act_entries;   // predictor: {active neurons, run}
  int n_entries;
  const unsigned long long* row_words;     // predictor: {cache row, run} of the active cached neurons
  const unsigned long long* gate_words;    // resident gate: {gate value, run} of the active neurons
  const int* predictor_run;
  int* next_run;                  // bumped at the end (a predictor without a first stage needs it)
  int32_t* n_act_out;
  int32_t* row_stamps;            // last_active by row, as long as CNT_ROW_STAMPS names this step
  uint32_t* hit_rows;             // plan: row before the moves | neuron << 16, for the cache CTAs
  const unsigned char* store;
  unsigned char* cache;
  const __half* x;
  const float* gate_val;          // resident gate: gate pre-activations by neuron id
  const __half* b_down;
  float* p_member;                // partial sums of cache CTAs that form groups, [cta][d]
  uint4 *p_hit, *p_new;           // tagged partial sums of cache CTAs (or groups) and fetch CTAs
  // several streams: each fetch CTA's last row, as tagged words: its down column in pairs of fp16 values
  // [cta][d / 2], and its weights [cta][8]
  unsigned long long *last_down, *last_h;
  float* y;
  StepSync* sync;
  int d, n_streams, whole_cache, act;
  float act_thr;
  int hand_over;                  // several streams: see kHandOver
  int n_cache_ctas, n_sum_ctas, group_size, cache_stages, fetch_stages, hits_max;
  unsigned wait_polls;            // of the first wait for a bulk copy
  unsigned spin_limit;            // of a wait for another CTA
  unsigned epoch;                 // steps before this one (filled in by the kernel)
};

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ unsigned long long ld_acquire64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
// Everything the CTA wrote before the preceding __syncthreads() is visible to whoever sees the
// arrival (thread 0 only: one fence for the CTA instead of one per thread, which took 1-2 us).
__device__ __forceinline__ bool arrive_last(unsigned* p, unsigned want) {
  unsigned v;
  asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(v) : "l"(p) : "memory");
  return v + 1 == want;
}
__device__ __forceinline__ void arrive(unsigned* p) {
  asm volatile("red.add.release.gpu.global.u32 [%0], 1;" ::"l"(p) : "memory");
}
__device__ __forceinline__ bool is_plan(const StepArgs& a, unsigned long long v) {
  return (v & kPlanReady) && v >> kPlanEpochShift == (a.epoch & kPlanEpochMask);
}
__device__ __forceinline__ void publish(const StepArgs& a, unsigned long long v) {
  v |= (unsigned long long)(a.epoch & kPlanEpochMask) << kPlanEpochShift;
  asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(&a.sync->plan), "l"(v) : "memory");
}
// Exclusive prefixes of N words over the block and the block's sums; one barrier, so consecutive
// calls need different `sums`.  Two counts up to 32768 can ride in one word (16 bits each).
template <int N>
__device__ __forceinline__ void step_scan(unsigned (&v)[N], unsigned (&total)[N],
                                          unsigned (&sums)[N][kStepWarps]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned inc[N];
#pragma unroll
  for (int k = 0; k < N; ++k) inc[k] = v[k];
#pragma unroll
  for (int o = 1; o < 32; o <<= 1)
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const unsigned n = __shfl_up_sync(0xffffffffu, inc[k], o);
      if (lane >= o) inc[k] += n;
    }
#pragma unroll
  for (int k = 0; k < N; ++k)
    if (lane == 31) sums[k][warp] = inc[k];
  __syncthreads();
#pragma unroll
  for (int k = 0; k < N; ++k) {
    const unsigned ws = sums[k][lane & (kStepWarps - 1)];
    unsigned winc = ws;
#pragma unroll
    for (int o = 1; o < kStepWarps; o <<= 1) {
      const unsigned n = __shfl_up_sync(0xffffffffu, winc, o);
      if (lane >= o) winc += n;
    }
    total[k] = __shfl_sync(0xffffffffu, winc, kStepWarps - 1);
    v[k] = __shfl_sync(0xffffffffu, winc - ws, warp) + inc[k] - v[k];
  }
}
__device__ __forceinline__ void timed_out(const StepArgs& a) { flag_timeout(a.w.counts + LIF_CNT_STATUS); }
// ... on something without which this CTA cannot fill or move the rows that the plan gives it
__device__ __forceinline__ void plan_not_carried_out(const StepArgs& a) {
  a.w.counts[CNT_ROWS_SUSPECT] = 1;
  timed_out(a);
}
__device__ __forceinline__ unsigned long long ld_relaxed64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
// The thread's entries of the predictor run `run`.  This kernel may be resident while the score
// kernel still runs; each entry is stored together with the number of its run, so a thread re-reads
// its own until they carry it.  If they do not come (bounded), the kernel waits for its predecessor
// and takes them as they are: false, and then the other words of the run need no check either.
template <int N>
__device__ __forceinline__ bool read_entries(const unsigned long long* const (&entries)[N], int n, int run,
                                             uint32_t (&mw)[N][kEntriesPerThread]) {
  const int w0 = threadIdx.x * kEntriesPerThread;
  auto read = [&](bool check) {
    bool mine = true;
#pragma unroll
    for (int k = 0; k < N; ++k)
#pragma unroll
      for (int i = 0; i < kEntriesPerThread; ++i) {
        mw[k][i] = 0u;
        if (w0 + i < n) {
          const unsigned long long v = ld_relaxed64(entries[k] + w0 + i);
          mw[k][i] = (uint32_t)v;
          mine = mine && (!check || (int)(v >> 32) == run);
        }
      }
    return mine;
  };
  int ok = 0;
  for (int i = 0; i < kStepWatchPolls && !ok; ++i) ok = __syncthreads_and(read(true) ? 1 : 0);
  if (!ok) {
    pdl_wait();
    read(false);
  }
  return ok != 0;
}
// The low half of a word that the predictor run `run` stores beside its entries, once it is there (it is
// stored with the entry: a poll or two).  checked = false: as it is (see read_entries).
__device__ __forceinline__ uint32_t word_of_run(const StepArgs& a, const unsigned long long* at, int run,
                                                bool checked) {
  unsigned long long v = checked ? 0ull : ld_relaxed64(at);
  bool there = !checked;
  for (unsigned i = 0; i < a.spin_limit && !there; ++i) {
    v = ld_relaxed64(at);
    there = (int)(v >> 32) == run;
  }
  if (!there) {                                            // (row 0, gate value 0)
    timed_out(a);
    v = 0;
  }
  return (uint32_t)v;
}
// Thread 0 waits for the plan; everyone gets it (0 if it did not come: an error is recorded).
__device__ __forceinline__ unsigned long long wait_plan(const StepArgs& a,
                                                        unsigned long long* shared) {
  if (threadIdx.x == 0) {
    unsigned long long v = 0;
    bool there = false;
    for (unsigned i = 0; i < a.spin_limit && !there; ++i) {
      v = ld_acquire64(&a.sync->plan);
      there = is_plan(a, v);
    }
    if (!there) {
      plan_not_carried_out(a);
      v = 0;
    }
    *shared = v;
  }
  __syncthreads();
  return *shared;
}

__host__ __device__ __forceinline__ size_t x_smem_bytes(int d, int S) {
  return ((size_t)S * d * 2 + 127) & ~(size_t)127;
}

// ---- window CTA ---------------------------------------------------------------------------------
// The same plan as the window kernels (window.cu), held in shared memory: row -> neuron and age of every
// row are read before the predictor's entries arrive (the window state was last written by this layer's
// previous step), so between the entries and the flag there are one round trip for the active neurons'
// rows, shared-memory passes and block scans.  What the other CTAs need is written ahead of the flag,
// the rest of the lists and the state behind it.
// The reads ahead of the entries are few and coalesced, because they run beside the predictor: reading slot_of of
// every neuron (64 KB at 16384) and the stamp of every row by its neuron held back the predictor's CTA on
// the same SM, and with it the last entry, by 1.5 us (2.2 at 4544 columns).  So the step keeps a copy of the
// stamps by row, which a window update by another kernel makes out of date (CNT_ROW_STAMPS).
// slot_of on chip ahead of the entries: a round trip less between them and the plan, which the FFN over every cached row
// waits for (4 layers, without / with: 512 x 2048 61.9 / 60.9 us, 768 x 3072 63.8 / 62.6, 2048 x 8192 103.2 / 102.6, 2560 x
// 10240 133.7 / 133.4).  Otherwise nothing is on the chain behind the plan: even, 512 x 2048 to 2048 x 16384, and not
// done where it is more than two loads per thread.
__host__ __device__ __forceinline__ bool slots_ahead(int F, int whole_cache) { return F <= (whole_cache ? 8192 : 4096); }
// (It decides which layers are one launch: with ages of 16 bits, every capacity up to 18900 neurons.)
size_t window_role_smem(int F, int cap, int whole_cache) {
  return (slots_ahead(F, whole_cache) ? 6 : 4) * (size_t)F + 8 * (size_t)cap + 4 * (size_t)((F + 31) / 32) + 64;
}

__device__ void window_role(const StepArgs& a, unsigned char* smem) {
  __shared__ unsigned sums[3][1][kStepWarps];
  __shared__ int hist[kMaxBudgetWindow + 1];
  __shared__ int loads;
  const WindowArgs& w = a.w;
  const int tid = threadIdx.x, F = w.F;
  unsigned short* slot_s = reinterpret_cast<unsigned short*>(smem);   // [F] row of each of these, or kNoSlot
  unsigned short* act_s = slot_s + F;                                 // [F] active ids, ascending
  unsigned short* age_s = act_s + F;                                  // [cap] steps since it was active, at most 65535
  unsigned short* pid_s = age_s + w.cap;                              // [cap] row -> neuron
  unsigned short* hole_s = pid_s + w.cap;                             // [cap] freed rows, ascending
  unsigned short* moved_s = hole_s + w.cap;                           // [cap] row - bound -> new row
  uint32_t* bits = reinterpret_cast<uint32_t*>(moved_s + w.cap);      // [F / 32]
  unsigned short* of_s = reinterpret_cast<unsigned short*>(bits + (F + 31) / 32);  // [F] slot_of (slots_ahead)

  const int n = w.counts[LIF_CNT_NUM_USED];
  const int t = w.counts[LIF_CNT_STEP];
  const int stale_input = w.counts[LIF_CNT_STATUS] == LIF_ERR_TIMEOUT;   // see window.cu
  const int t_end = t + w.keep - 1;
  const bool ahead = slots_ahead(F, a.whole_cache);
  if (ahead)
    for (int i = tid; i < F / 4; i += kStepThreads) {
      const int4 v = reinterpret_cast<const int4*>(w.slot_of)[i];        // (-1 becomes kNoSlot by itself)
      reinterpret_cast<uint32_t*>(of_s)[2 * i] = (uint32_t)(v.x & 0xffff) | ((uint32_t)v.y << 16);
      reinterpret_cast<uint32_t*>(of_s)[2 * i + 1] = (uint32_t)(v.z & 0xffff) | ((uint32_t)v.w << 16);
    }
  const bool stamps = w.counts[CNT_ROW_STAMPS] == t;
#pragma unroll 2
  for (int s = tid; s < n; s += kStepThreads) {
    const int id = w.pointers[s];
    const int la = stamps ? a.row_stamps[s] : w.last_active[id];
    pid_s[s] = (unsigned short)id;
    age_s[s] = (unsigned short)min(65535, max(1, t_end - la));
  }
  uint32_t act_w[1][kEntriesPerThread];
  read_entries<1>({a.act_entries}, a.n_entries, __ldcg(a.predictor_run), act_w);
  const uint32_t(&mw)[kEntriesPerThread] = act_w[0];
  unsigned pre[1] = {0u}, tot[1];
#pragma unroll
  for (int i = 0; i < kEntriesPerThread; ++i) {
    const int at = tid * kEntriesPerThread + i;
    pre[0] += __popc(mw[i]);
    if (at < (F + 31) / 32) bits[at] = mw[i];
  }
  step_scan<1>(pre, tot, sums[0]);                        // also publishes bits[] and the arrays
  const int na = (int)tot[0];
  {
    int q = (int)pre[0];
#pragma unroll 1
    for (int i = 0; i < kEntriesPerThread; ++i)
#pragma unroll 1
      for (uint32_t m = mw[i]; m; m &= m - 1)
        act_s[q++] = (unsigned short)((tid * kEntriesPerThread + i) * 32 + __ffs(m) - 1);
  }
  __syncthreads();
#pragma unroll 2
  for (int q = tid; q < na; q += kStepThreads)
    slot_s[q] = ahead ? of_s[act_s[q]] : (unsigned short)w.slot_of[act_s[q]];
  __syncthreads();
  // each thread owns a run of consecutive rows and of consecutive active neurons
  const int seg = (n + kStepThreads - 1) / kStepThreads;
  const int s0 = min(n, tid * seg), s1 = min(n, s0 + seg);
  const int qseg = (na + kStepThreads - 1) / kStepThreads;
  const int q0 = min(na, tid * qseg), q1 = min(na, q0 + qseg);
  auto idle_age = [&](int s) {       // 0: active now
    const int id = pid_s[s];
    return (bits[id >> 5] >> (id & 31)) & 1u ? 0 : (int)age_s[s];
  };
  // (of a row that stays: its age is below k_eff <= 32767 and therefore exact)
  auto stamp_of = [&](int s) { return t_end - (int)age_s[s]; };
  int c_load = 0;
  for (int q = q0; q < q1; ++q) c_load += slot_s[q] == kNoSlot;
  int k_eff = w.k;
  if (w.budget > 0) {                // memory budget: shrink the window for this step if needed
    if (tid <= kMaxBudgetWindow) hist[tid] = 0;
    if (tid == 0) loads = 0;
    __syncthreads();
    for (int s = s0; s < s1; ++s) {
      const int age = idle_age(s);
      if (age > 0) atomicAdd(&hist[min(w.k, age)], 1);
    }
    if (c_load) atomicAdd(&loads, c_load);
    __syncthreads();
    k_eff = widest_window_that_fits(hist, w.k, n, loads, min(w.cap, w.budget));
  }
  const int limit = w.budget > 0 ? min(w.cap, w.budget) : w.cap;
  int c_ev = 0;
  for (int s = s0; s < s1; ++s) c_ev += idle_age(s) >= k_eff;
  pre[0] = (unsigned)c_load | ((unsigned)c_ev << 16);
  step_scan<1>(pre, tot, sums[1]);
  const int n_load = (int)(tot[0] & 0xffff), n_evict = (int)(tot[0] >> 16);
  const int n_kept = n - n_evict;
  const int p_load0 = (int)(pre[0] & 0xffff), p_ev0 = (int)(pre[0] >> 16);
  if (stale_input || n_kept + n_load > limit) {           // refuse before anything is changed
    if (a.whole_cache)                                     // the FFN still runs over the rows in use
      for (int s = tid; s < n; s += kStepThreads)
        a.hit_rows[s] = (uint32_t)s | ((uint32_t)pid_s[s] << 16);
    __syncthreads();
    if (tid == 0) {
      atomicCAS(w.counts + LIF_CNT_STATUS, LIF_OK, LIF_ERR_CAPACITY);   // (another CTA may flag a wait)
      w.counts[LIF_CNT_N_ACTIVE] = 0;
      w.counts[LIF_CNT_N_EVICT] = 0;
      w.counts[LIF_CNT_N_MOVES] = 0;
      w.counts[LIF_CNT_N_LOAD] = 0;
      w.counts[LIF_CNT_N_HITS] = 0;
      w.counts[LIF_CNT_NUM_USED_BEFORE] = n;
      w.counts[LIF_CNT_NUM_KEPT] = n;
      publish(a, kPlanReady | kPlanRefused | (unsigned)(a.whole_cache ? n : 0));
    }
    pdl_wait();
    return;
  }
  // freed rows taken by new neurons directly, and where the rows that must move begin
  const int reuse = w.append_first ? min(n_evict, n_load) : 0;
  const int bound = n - (n_evict - reuse);
  int n_moves = 0, p_surv0 = 0;
  if (bound < n) {
    int c_surv = 0;
    for (int s = max(s0, bound); s < s1; ++s) c_surv += idle_age(s) < k_eff;
    pre[0] = (unsigned)c_surv;
    step_scan<1>(pre, tot, sums[2]);
    n_moves = (int)tot[0];
    p_surv0 = (int)pre[0];
  }
  {
    int p_ev = p_ev0;
    for (int s = s0; s < s1; ++s) {
      if (idle_age(s) >= k_eff) hole_s[p_ev++] = (unsigned short)s;
      else if (a.whole_cache) a.hit_rows[s - p_ev] = (uint32_t)s | ((uint32_t)pid_s[s] << 16);
    }
  }
  __syncthreads();
  {
    int p_surv = p_surv0;
    for (int s = max(s0, bound); s < s1; ++s)
      if (idle_age(s) < k_eff) {                           // surviving tail row: last one first
        const int jm = n_moves - 1 - p_surv++;
        const int dst = hole_s[reuse + jm];
        w.move_src[jm] = s;
        w.move_dst[jm] = dst;
        moved_s[s - bound] = (unsigned short)dst;
      }
  }
  auto new_row = [&](int p) { return p < n_load - reuse ? bound + p : (int)hole_s[n_load - 1 - p]; };
  {
    int p_load = p_load0;
    for (int q = q0; q < q1; ++q) {
      const int id = act_s[q], s = slot_s[q];
      if (s == kNoSlot) {
        w.load_slots[p_load] = new_row(p_load);
        ++p_load;
      } else if (!a.whole_cache) {
        a.hit_rows[q - p_load] = (uint32_t)s | ((uint32_t)id << 16);
      }
    }
  }
  __syncthreads();
  if (tid == 0) {
    const unsigned n_rows = a.whole_cache ? n_kept : na - n_load;
    publish(a, kPlanReady | ((unsigned long long)n_load << 32) | ((unsigned long long)n_moves << 16) | n_rows);
  }

  // ---- behind the flag: the public lists and the state ------------------------------------------
  pdl_wait();                       // (speculative stamps come from the predictor's keep_tok)
  {
    int p_ev = p_ev0, p_surv = p_surv0;
    for (int s = s0; s < s1; ++s) {
      const int id = pid_s[s];
      if (idle_age(s) >= k_eff) {
        w.evict_ids[p_ev++] = id;
        w.slot_of[id] = -1;
      } else if (s >= bound) {
        const int dst = hole_s[reuse + n_moves - 1 - p_surv++];
        a.row_stamps[dst] = stamp_of(s);                   // (those of active neurons follow below)
        w.pointers[dst] = id;
        w.slot_of[id] = dst;
        w.bias[dst] = w.bias_up[id];
      } else if (!stamps) {
        a.row_stamps[s] = stamp_of(s);
      }
      if (s >= n_kept + n_load) w.pointers[s] = -1;      // tail beyond the rows in use
    }
    __syncthreads();
    int p_load = p_load0;
    for (int q = q0; q < q1; ++q) {
      const int id = act_s[q];
      int s = slot_s[q];
      const int stamp = active_stamp(w, id, t, t_end);
      w.last_active[id] = stamp;
      if (s == kNoSlot) {
        s = new_row(p_load);
        w.load_ids[p_load++] = id;
        w.slot_of[id] = s;
        w.pointers[s] = id;
        w.bias[s] = w.bias_up[id];
      } else {
        if (s >= bound) s = moved_s[s - bound];
        w.hit_slots[q - p_load] = s;
      }
      a.row_stamps[s] = stamp;
      w.active_slots[q] = s;
      w.active_idx[q] = id;
    }
  }
  if (tid == 0) {
    *a.n_act_out = na;
    w.counts[LIF_CNT_N_ACTIVE] = na;
    w.counts[LIF_CNT_N_EVICT] = n_evict;
    w.counts[LIF_CNT_N_MOVES] = n_moves;
    w.counts[LIF_CNT_N_LOAD] = n_load;
    w.counts[LIF_CNT_N_HITS] = na - n_load;
    w.counts[LIF_CNT_NUM_USED_BEFORE] = n;
    w.counts[LIF_CNT_NUM_KEPT] = n_kept;
    w.counts[LIF_CNT_NUM_USED] = n_kept + n_load;
    w.counts[LIF_CNT_STEP] = t + w.keep;
    w.counts[CNT_ROW_STAMPS] = t + w.keep;
    w.counts[LIF_CNT_K_EFF] = k_eff;
    unsigned long long* totals = reinterpret_cast<unsigned long long*>(w.counts + CNT_TOTALS);
    totals[0] += (unsigned long long)n_load * w.bundle_bytes;
    totals[1] += (unsigned long long)n_moves;
    totals[2] += (unsigned long long)na;
    totals[3] += (unsigned long long)(n_kept + n_load);
  }
}

// ---- shared by the cache and fetch CTAs ---------------------------------------------------------
// kS streams (the layer's number rounded up to 1, 2, 4 or 8): a thread keeps kS x kChunks x 8 column
// sums in registers, which is what limits n_streams * d_model.
template <int kS>
struct Shape {
  static constexpr int kChunks = kS == 8 ? 1 : 2;          // 16-byte chunks per thread and vector
  static constexpr int kDepth = kS == 1 ? 4 : 12;          // partial sums per thread in flight
  static constexpr int kMaxD = kChunks * kStepThreads * 8;
};
template <int kS>
struct Acc {
  float v[kS][Shape<kS>::kChunks][8];
  __device__ __forceinline__ Acc() {
#pragma unroll
    for (int s = 0; s < kS; ++s)
#pragma unroll
      for (int k = 0; k < Shape<kS>::kChunks; ++k)
#pragma unroll
        for (int e = 0; e < 8; ++e) v[s][k][e] = 0.f;
  }
};
// acc += h[s] * v for the thread's chunks of the down column
template <int kS>
__device__ __forceinline__ void axpy_row(Acc<kS>& acc, const uint4* down, const float* h, int nvec) {
#pragma unroll
  for (int k = 0; k < Shape<kS>::kChunks; ++k) {
    const int c = threadIdx.x + k * kStepThreads;
    if (c < nvec) {
      float f[8];
      unpack8(down[c], f);
#pragma unroll
      for (int s = 0; s < kS; ++s) {
        const float hs = h[s];
        if (kS == 1 || hs != 0.f) {
#pragma unroll
          for (int e = 0; e < 8; ++e) acc.v[s][k][e] = fmaf(hs, f[e], acc.v[s][k][e]);
        }
      }
    }
  }
}
// p[s] += <row chunk, x[s] chunk>
template <int kS>
__device__ __forceinline__ void dot_chunk(float (&p)[kS], const uint4& row, const uint4* xs, int v,
                                          int nvec, int S) {
#pragma unroll
  for (int s = 0; s < kS; ++s)
    if (kS == 1 || s < S) p[s] = dot8(row, xs[s * nvec + v], p[s]);
}
// A partial sum for the end of the step: every pair of values is stored as {v, tag, v, tag}, two
// 8-byte words that are each written whole, with a tag of this step (step number + 1).  The reader
// polls the words themselves, so there is no fence, no counter and no second round trip between
// the last row and the sum (measured: 1.3 us from the last row to y instead of 3.5).  Pair e of
// 8-column chunk c is word e * (d / 8) + c of its stream's d / 2, so that a warp's stores are
// contiguous.
__device__ __forceinline__ void store_tagged(uint4* dst, float v0, float v1, unsigned tag) {
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(dst),
               "l"((unsigned long long)__float_as_uint(v0) | ((unsigned long long)tag << 32)),
               "l"((unsigned long long)__float_as_uint(v1) | ((unsigned long long)tag << 32))
               : "memory");
}
__device__ __forceinline__ ulonglong2 load_tagged(const uint4* src) {
  ulonglong2 v;
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "l"(src) : "memory");
  return v;
}
__device__ __forceinline__ void store_tagged_word(unsigned long long* dst, uint32_t low, unsigned tag) {
  store_with_run(dst, low, (int)tag);
}
__device__ __forceinline__ bool has_tag(const ulonglong2& v, unsigned tag) {
  return (unsigned)(v.x >> 32) == tag && (unsigned)(v.y >> 32) == tag;
}
template <int kS>
__device__ __forceinline__ void store_tagged_partial(const Acc<kS>& acc, uint4* dst, int nvec, int S,
                                                     unsigned tag) {
#pragma unroll
  for (int s = 0; s < kS; ++s)
    if (kS == 1 || s < S) {
#pragma unroll
      for (int k = 0; k < Shape<kS>::kChunks; ++k) {
        const int c = threadIdx.x + k * kStepThreads;
        if (c < nvec) {
#pragma unroll
          for (int e = 0; e < 4; ++e)
            store_tagged(dst + (4 * s + e) * nvec + c, acc.v[s][k][2 * e], acc.v[s][k][2 * e + 1], tag);
        }
      }
    }
}
template <int kS>
__device__ __forceinline__ void store_partial(const Acc<kS>& acc, float* dst, int nvec, int S) {
#pragma unroll
  for (int s = 0; s < kS; ++s)
    if (kS == 1 || s < S) {
      float4* out = reinterpret_cast<float4*>(dst) + (size_t)s * 2 * nvec;
#pragma unroll
      for (int k = 0; k < Shape<kS>::kChunks; ++k) {
        const int c = threadIdx.x + k * kStepThreads;
        const float(&v)[8] = acc.v[s][k];
        if (c < nvec) {
          __stcg(out + 2 * c, make_float4(v[0], v[1], v[2], v[3]));
          __stcg(out + 2 * c + 1, make_float4(v[4], v[5], v[6], v[7]));
        }
      }
    }
}
template <int kGate>
__device__ __forceinline__ float row_weight(const StepArgs& a, float b, float first, float second) {
  if (kGate == LIF_GATE_BUNDLED) return apply_activation(first + b, a.act, a.act_thr) * second;
  if (kGate == LIF_GATE_RESIDENT) return apply_activation(b, a.act, a.act_thr) * first;
  return apply_activation(first + b, a.act, a.act_thr);
}
// the neuron's bias; resident gate (one stream): its gate value
template <int kGate>
__device__ __forceinline__ float row_scalar(const StepArgs& a, int id, int run, bool checked) {
  return kGate == LIF_GATE_RESIDENT ? __uint_as_float(word_of_run(a, a.gate_words + id, run, checked))
                                    : __half2float(a.w.bias_up[id]);
}
// x of every stream into shared memory, past L1: it may hold lines of an earlier token's
__device__ __forceinline__ void load_x(const StepArgs& a, uint4* xs) {
  for (int i = threadIdx.x; i < a.n_streams * (a.d >> 3); i += kStepThreads)
    xs[i] = __ldcg(reinterpret_cast<const uint4*>(a.x) + i);
}

// ---- cache CTAs: row moves and the FFN of the rows that were already cached -------------------------
// Rows are read where they were before the moves: a moved row's source is not overwritten before
// all cache CTAs are done (append_first: not at all), so moves and FFN need no order.  The moves come
// first in the paper's order, where the new rows wait for them, and last otherwise.
// CTA c adds the hits of rank c, c + nc, ... (ascending neuron ids): the set bits of the predictor's
// entries of active neurons that its entries of new ones lack.
template <int kGate, int kS>
__device__ void cache_role(const StepArgs& a, int c, unsigned char* smem) {
  constexpr int kVec = kGate == LIF_GATE_BUNDLED ? 3 : 2;
  __shared__ __align__(8) uint64_t bars[16];
  __shared__ float h_s[16][kS], b_s[16];
  __shared__ unsigned long long plan_s;
  __shared__ unsigned sums[1][kStepWarps];
  __shared__ int last_s, lost_s;       // (lost_s: as a barrier's reduction 0.4 us a step more)
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int d = a.d, S = a.n_streams, nvec = d >> 3, stages = a.cache_stages, nc = a.n_cache_ctas;
  const unsigned row_bytes = 2u * kVec * d;
  uint4* xs = reinterpret_cast<uint4*>(smem);              // [S][d]
  unsigned char* rows = smem + x_smem_bytes(d, S);
  unsigned short* hits = reinterpret_cast<unsigned short*>(rows + (size_t)stages * row_bytes);
  if (tid == 0) {
    lost_s = 0;
    for (int i = 0; i < stages; ++i) mbar_init(bars + i, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  const int run = __ldcg(a.predictor_run);
  bool checked = false;
  int n, n_moves = 0;
  if (a.whole_cache) {
    pdl_wait();                                            // (gate values of every row)
    load_x(a, xs);
    const unsigned long long plan = wait_plan(a, &plan_s);
    n = plan_rows(plan);
    n_moves = plan_moves(plan);
  } else {
    // one thread watches one entry: the whole CTA re-reading all of them beside the score kernel cost it
    // 1 us at 4096 x 16384
    for (int i = 0; tid == 0 && i < 2 * kStepWatchPolls; ++i) {
      if ((int)(ld_relaxed64(a.new_entries + a.n_entries - 1) >> 32) == run) break;
      __nanosleep(100);
    }
    __syncthreads();
    uint32_t mw[2][kEntriesPerThread];
    checked = read_entries<2>({a.act_entries, a.new_entries}, a.n_entries, run, mw);
    unsigned pre[1] = {0u}, tot[1];
#pragma unroll
    for (int i = 0; i < kEntriesPerThread; ++i) pre[0] += __popc(mw[0][i] & ~mw[1][i]);
    step_scan<1>(pre, tot, sums);
    n = (int)tot[0];
    unsigned q = pre[0];
#pragma unroll
    for (int i = 0; i < kEntriesPerThread; ++i)
      for (uint32_t m = mw[0][i] & ~mw[1][i]; m; m &= m - 1, ++q) {
        const unsigned j = q / (unsigned)nc;
        if (q - j * nc == (unsigned)c && j < (unsigned)a.hits_max)
          hits[j] = (unsigned short)((tid * kEntriesPerThread + i) * 32 + __ffs(m) - 1);
      }
    __syncthreads();
  }
  auto move_rows = [&](auto pieces) {                      // 16-byte pieces of a thread in flight
    constexpr int kPieces = decltype(pieces)::value;
    const int row_vec = kVec * nvec;
    for (int j = c; j < n_moves; j += nc) {
      const uint4* src = reinterpret_cast<const uint4*>(a.cache) + (size_t)__ldcg(a.w.move_src + j) * row_vec;
      uint4* dst = reinterpret_cast<uint4*>(a.cache) + (size_t)__ldcg(a.w.move_dst + j) * row_vec;
      uint4 v[kPieces];
      for (int v0 = tid; v0 < row_vec; v0 += kPieces * kStepThreads) {
#pragma unroll
        for (int u = 0; u < kPieces; ++u)
          if (v0 + u * kStepThreads < row_vec) v[u] = ld_stream16(src + v0 + u * kStepThreads);
#pragma unroll
        for (int u = 0; u < kPieces; ++u)
          if (v0 + u * kStepThreads < row_vec) dst[v0 + u * kStepThreads] = v[u];
      }
    }
  };
  const int cnt = c < n ? min(a.hits_max, (n - c + nc - 1) / nc) : 0;
  Acc<kS> acc;

  unsigned parity = 0;
  for (int r0 = 0; r0 < cnt || r0 == 0; r0 += stages) {
    const int rc = min(stages, cnt - r0);
    if (tid < rc) {
      int id, row;
      if (a.whole_cache) {
        const uint32_t e = __ldcg(a.hit_rows + c + (r0 + tid) * nc);
        id = (int)(e >> 16);
        row = (int)(e & 0xffff);
      } else {
        id = hits[r0 + tid];
        row = (int)word_of_run(a, a.row_words + id, run, checked);
      }
      mbar_expect_tx(bars + tid, row_bytes);
      bulk_g2s(rows + (size_t)tid * row_bytes, a.cache + (size_t)row * row_bytes, row_bytes, bars + tid);
      b_s[tid] = kGate == LIF_GATE_RESIDENT && a.whole_cache ? a.gate_val[id]
                                                             : row_scalar<kGate>(a, id, run, checked);
    }
    if (r0 == 0 && !a.whole_cache) load_x(a, xs);          // while the first rows travel
    if (r0 == 0 && !a.w.append_first) {                    // ... and the moves
      if (!a.whole_cache) n_moves = plan_moves(wait_plan(a, &plan_s));
      move_rows(std::integral_constant<int, kS == 1 ? 2 : 4>{});   // (beside the sums; see step_kernel's bounds)
    }
    __syncthreads();                                       // x and the rows' scalars
    if (rc <= 0) break;
    for (int i = warp; i < rc; i += kStepWarps) {          // a warp per row
      const bool landed = __all_sync(0xffffffffu, mbar_wait(bars + i, parity, a.wait_polls));
      if (!landed) {                                       // flagged; its terms are left out
        lost_s = 1;
        if (lane == 0) timed_out(a);
        mbar_wait(bars + i, parity);                       // another bounded chance to land
      }
      const uint4* row = reinterpret_cast<const uint4*>(rows + (size_t)i * row_bytes);
      float p[kS], p2[kS];
#pragma unroll
      for (int s = 0; s < kS; ++s) p[s] = p2[s] = 0.f;
#pragma unroll 2
      for (int v = lane; v < nvec; v += 32) {
        dot_chunk<kS>(p, row[v], xs, v, nvec, S);
        if (kGate == LIF_GATE_BUNDLED) dot_chunk<kS>(p2, row[nvec + v], xs, v, nvec, S);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int s = 0; s < kS; ++s)
          if (kS == 1 || s < S) {
            p[s] += __shfl_xor_sync(0xffffffffu, p[s], o);
            if (kGate == LIF_GATE_BUNDLED) p2[s] += __shfl_xor_sync(0xffffffffu, p2[s], o);
          }
      if (lane == 0) {
#pragma unroll
        for (int s = 0; s < kS; ++s)
          h_s[i][s] = landed && s < S ? row_weight<kGate>(a, b_s[i], p[s], p2[s]) : 0.f;
      }
    }
    __syncthreads();
    for (int i = 0; i < rc; ++i) {
      if (kS == 1 && h_s[i][0] == 0.f) continue;
      axpy_row<kS>(acc, reinterpret_cast<const uint4*>(rows + (size_t)i * row_bytes) + (kVec - 1) * nvec,
                   h_s[i], nvec);
    }
    if (lost_s) break;                                     // nothing more into stages that may be written late
    parity ^= 1u;
    if (r0 + stages < cnt) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncthreads();                                     // rows are free for the next copies
    }
  }

  // The CTA's partial; with many cache CTAs the last of each group of them adds the group's
  // partials (in CTA order), so that few are left for the end of the step.
  const int gs = a.group_size, g = c / gs;
  const size_t width = (size_t)S * d;
  bool last = true;
  if (gs == 1) {
    if (cnt > 0) store_tagged_partial<kS>(acc, a.p_hit + (size_t)c * (width / 2), nvec, S, a.epoch + 1);
    __syncthreads();
  } else {
    if (cnt > 0) store_partial<kS>(acc, a.p_member + (size_t)c * width, nvec, S);
    __syncthreads();
    const int members = min(gs, nc - g * gs);
    if (tid == 0) last_s = arrive_last(&a.sync->group[g], (a.epoch + 1) * (unsigned)members);
    __syncthreads();
    last = last_s;
    const int have = min(members, max(0, n - g * gs));     // members with rows wrote a partial
    if (last && have > 0)
      for (int i = tid; i < (int)(width / 4); i += kStepThreads) {
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f), v[8];
#pragma unroll
        for (int m = 0; m < 8; ++m)
          if (m < have) v[m] = __ldcg(reinterpret_cast<const float4*>(a.p_member + (size_t)(g * gs + m) * width) + i);
#pragma unroll
        for (int m = 0; m < 8; ++m)
          if (m < have) { s.x += v[m].x; s.y += v[m].y; s.z += v[m].z; s.w += v[m].w; }
        const int st = i / (2 * nvec), r = i - st * 2 * nvec;
        uint4* dst = a.p_hit + (size_t)g * (width / 2) + (4 * st + (r & 1) * 2) * nvec + (r >> 1);
        store_tagged(dst, s.x, s.y, a.epoch + 1);
        store_tagged(dst + nvec, s.z, s.w, a.epoch + 1);
      }
  }
  // (only the paper's cache order waits for this: the rows have been read and moved)
  if (tid == 0 && last) arrive(&a.sync->groups_done);
  if (a.w.append_first) {            // (plan_s was not used before: the FFN over every cached row excludes this order)
    n_moves = plan_moves(wait_plan(a, &plan_s));
    move_rows(std::integral_constant<int, 4>{});
  }
}

// ---- the sum: CTA `index` of `n` adds up a slice of the columns, in pairs, in a fixed order ----------
// `width` pairs are side by side; the other threads share the partials: those of the cached rows, then
// those of the fetch CTAs.
template <int kS>
struct Summer {
  static constexpr int kDepth = Shape<kS>::kDepth;
  const StepArgs& a;
  const unsigned tag;
  const int pairs, have_hit, have;
  int c0, c1, width, slices, slice, t_next, lost;
  float2 v_sum;

  __device__ __forceinline__ Summer(const StepArgs& args, int index, int n, int n_hit, int n_new)
      : a(args), tag(args.epoch + 1), pairs(args.n_streams * (args.d >> 1)),
        have_hit((min(n_hit, args.n_cache_ctas) + args.group_size - 1) / args.group_size),
        have(have_hit + n_new), lost(0), v_sum(make_float2(0.f, 0.f)) {
    const int per = (pairs + n - 1) / n;
    c0 = index * per;
    c1 = min(pairs, c0 + per);
    width = 32;
    while (width < per && width < kStepThreads / 2) width *= 2;
    slices = kStepThreads / width;
    slice = threadIdx.x / width;
    t_next = slice;
  }
  // (past the end: the last one again)
  __device__ __forceinline__ const uint4* at(int t, int end, int col) const {
    t = min(t, end - 1);
    return (t < have_hit ? a.p_hit + (size_t)t * pairs : a.p_new + (size_t)(t - have_hit) * pairs) + col;
  }
  // adds the thread's partials of column pair `col` up to number `end`; stops where they are not there
  // after `limit` polls
  __device__ __forceinline__ void add(int end, int col, unsigned limit) {
    if (col >= c1) return;
    for (; t_next < end; t_next += slices * kDepth) {
      ulonglong2 v[kDepth];
#pragma unroll
      for (int k = 0; k < kDepth; ++k) v[k] = load_tagged(at(t_next + k * slices, end, col));
      bool there = false;
      for (unsigned polls = 0; polls < limit; ++polls) {
        there = true;
#pragma unroll
        for (int k = 0; k < kDepth; ++k) there = there && has_tag(v[k], tag);
        if (there || polls + 1 == limit) break;
#pragma unroll
        for (int k = 0; k < kDepth; ++k)                   // again, those that were not there
          if (!has_tag(v[k], tag)) v[k] = load_tagged(at(t_next + k * slices, end, col));
      }
      if (!there) {
        lost = 1;
        return;
      }
#pragma unroll
      for (int k = 0; k < kDepth; ++k)
        if (t_next + k * slices < end) {
          v_sum.x += __uint_as_float((unsigned)v[k].x);
          v_sum.y += __uint_as_float((unsigned)v[k].y);
        }
    }
    lost = 0;
    t_next = end <= slice ? slice : slice + (end - slice + slices - 1) / slices * slices;
  }
  // adds the thread's share of the fetch CTAs' last rows to column pair `col`
  __device__ __forceinline__ void add_last(int n_last, int col) {
    constexpr int kRows = 16;                              // (all of a thread's: 32 CTAs, 2 slices or more)
    if (col >= c1) return;
    const int half_d = a.d >> 1, s = col / half_d;
    const unsigned long long *down = a.last_down + col % half_d, *h = a.last_h + s;
    for (int t0 = slice; t0 < n_last; t0 += slices * kRows) {
      auto ask = [&](unsigned long long (&v)[kRows], const unsigned long long* p, int stride, bool pause) {
        bool there = false;
        for (unsigned polls = 0; polls < a.spin_limit && !there; ++polls) {
          there = true;
#pragma unroll
          for (int k = 0; k < kRows; ++k) {
            const int t = t0 + k * slices;
            v[k] = t < n_last ? ld_relaxed64(p + (size_t)t * stride) : (unsigned long long)tag << 32;
          }
#pragma unroll
          for (int k = 0; k < kRows; ++k) there = there && (unsigned)(v[k] >> 32) == tag;
          if (pause && !there) __nanosleep(100);
        }
        return there;
      };
      // the columns, with pauses while the rows travel; when they are there the weights follow at once
      unsigned long long v[kRows];
      uint32_t pair[kRows];
      bool there = ask(v, down, half_d, true);
#pragma unroll
      for (int k = 0; k < kRows; ++k) pair[k] = (uint32_t)v[k];
      there = there && ask(v, h, 8, false);
      if (!there) {
        lost = 1;
        return;
      }
#pragma unroll
      for (int k = 0; k < kRows; ++k)
        if (t0 + k * slices < n_last) {
          const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&pair[k]));
          const float w = __uint_as_float((uint32_t)v[k]);
          if (w != 0.f) {                                  // (as everywhere: a row of weight 0 is not read)
            v_sum.x = fmaf(w, f.x, v_sum.x);
            v_sum.y = fmaf(w, f.y, v_sum.y);
          }
        }
    }
  }
  // red: kStepThreads values in shared memory
  __device__ __forceinline__ void finish(float2* red, int n_last) {
    const int tid = threadIdx.x, nvec = a.d >> 3;
    for (int cc = c0; cc < c1; cc += width) {
      const int col = cc + tid % width;
      if (cc > c0) {
        v_sum = make_float2(0.f, 0.f);
        t_next = slice;
        __syncthreads();                                   // red[] is free again
      }
      add(have, col, a.spin_limit);
      if (kS > 1) {
        if (lost) timed_out(a);
        if (a.hand_over) add_last(n_last, col);
      }
      if (lost) timed_out(a);
      red[tid] = v_sum;
      __syncthreads();
      if (tid < width && col < c1) {
        const int s = kS == 1 ? 0 : col / (4 * nvec), r = kS == 1 ? col : col % (4 * nvec);
        const int to = 4 * (r % nvec) + r / nvec;          // columns 2 * to, 2 * to + 1
        float2 y = make_float2(0.f, 0.f);
        if (a.b_down) y = __half22float2(*reinterpret_cast<const __half2*>(a.b_down + 2 * to));
        for (int k = 0; k < slices; ++k) {
          y.x += red[k * width + tid].x;
          y.y += red[k * width + tid].y;
        }
        reinterpret_cast<float2*>(a.y + (size_t)s * a.d)[to] = y;
      }
    }
  }
};

constexpr size_t kSumSmem = kStepThreads * sizeof(float2);

// ---- sum CTAs ----------------------------------------------------------------------------------------
// They wait for a word of the fetch CTAs' partials, with pauses, so that they do not load the memory
// system while the rows travel.  Several streams: for one of each CTA, to read everything at once, while the
// CTAs' last rows are still on their way; then for the weights of those, whose terms they add themselves (a
// partial has as many values as all outputs together, 160 KB for 5 streams at 4096 columns: stored, read and
// added behind the last bundle that was 9.5 us of a step; a down column and five weights are 5.4).  One
// stream: for one of the CTA with the fewest rows, adding the cached rows' partials meanwhile if they come
// first, and then they take what is missing as it comes: a single round trip from the last partial,
// whichever it is, to y.  With at most two rows per fetch CTA the whole wait is a few microseconds and a
// poll of that word ahead of the partials is what is noticed: 352 x 944, 10 new rows, 2 layers 33.9 us with
// it and 31.6 without, tiny 29.2 and 27.0; with more rows there is no difference (4096 x 16384, 8 layers
// 386-388 us) and the memory system is left alone while they travel.
// (With one stream the fetch CTAs themselves used to do this, waiting for one another.  These CTAs, the
// same number at 1024 columns and more, measure the same or better: 768 x 3072, 4 layers 65.4 -> 62.8 us.)
template <int kS>
__device__ void sum_role(const StepArgs& a, int index, unsigned char* smem) {
  __shared__ unsigned long long plan_s;
  const int tid = threadIdx.x;
  const int run = __ldcg(a.predictor_run);
  const unsigned long long plan = wait_plan(a, &plan_s);
  const int n_load = plan_loads(plan);                     // (0: refused)
  const int n_last = min(kFetchCtas, n_load);              // fetch CTAs with rows; with several of them
  Summer<kS> sum(a, index, a.n_sum_ctas, plan_rows(plan),
                 kS == 1 || !a.hand_over ? n_last : max(0, min(kFetchCtas, n_load - kFetchCtas)));
  const size_t pairs = (size_t)a.n_streams * (a.d >> 1);
  const int n_new = sum.have - sum.have_hit;
  if (kS == 1) {
    for (unsigned polls = 0; n_load > 2 * kFetchCtas && polls < a.spin_limit; ++polls) {
      const int there = tid == 0 && (n_new == 0 || has_tag(load_tagged(a.p_new + n_new * pairs - 1), sum.tag));
      sum.add(sum.have_hit, sum.c0 + tid % sum.width, 1);
      if (__syncthreads_or(there)) break;
      __nanosleep(100);
    }
  } else if (tid < n_new) {
    bool there = false;
    for (unsigned polls = 0; !there && polls < a.spin_limit; ++polls) {
      there = has_tag(load_tagged(a.p_new + (tid + 1) * pairs - 1), sum.tag);
      if (!there) __nanosleep(100);
    }
  }
  __syncthreads();
  sum.finish(reinterpret_cast<float2*>(smem), n_last);     // kSumSmem bytes
  // (by the CTA that started last: every other one has read the number by now)
  if (index == a.n_sum_ctas - 1 && tid == 0) advance_run(a.next_run, run);
}

// ---- fetch CTAs: new bundles over the host link and their FFN terms ---------------------------------
// Fetch CTA f brings in entries f, f + kFetchCtas, ... of the load list, which is exactly the set
// bits of the predictor's entries in ascending order; only the cache row comes from the plan.  A bundle
// stays in the ring until its row is known and, in the paper's order, until the cache CTAs have read and
// moved what was there; its FFN term is computed meanwhile.
template <int kGate, int kS>
__device__ void fetch_role(const StepArgs& a, int f, unsigned char* smem) {
  constexpr int kVec = kGate == LIF_GATE_BUNDLED ? 3 : 2;
  __shared__ __align__(8) uint64_t bars[16];
  __shared__ unsigned sums[1][kStepWarps];
  __shared__ float part[2][kS][kStepWarps];
  __shared__ float h_s[kS];
  __shared__ int count_s, go_s;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int d = a.d, S = a.n_streams, nvec = d >> 3, stages = a.fetch_stages;
  constexpr int nf = kFetchCtas;
  const unsigned row_bytes = 2u * kVec * d;
  uint4* xs = reinterpret_cast<uint4*>(smem);              // [S][d]
  unsigned char* ring = smem + x_smem_bytes(d, S);
  unsigned short* ids = reinterpret_cast<unsigned short*>(ring + (size_t)stages * row_bytes);
  if (tid == 0) {
    for (int i = 0; i < stages; ++i) mbar_init(bars + i, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  uint32_t new_w[1][kEntriesPerThread];
  const int run = __ldcg(a.predictor_run);
  const bool checked = read_entries<1>({a.new_entries}, a.n_entries, run, new_w);
  const uint32_t(&mw)[kEntriesPerThread] = new_w[0];
  unsigned pre[1] = {0u}, tot[1];
#pragma unroll
  for (int i = 0; i < kEntriesPerThread; ++i) pre[0] += __popc(mw[i]);
  step_scan<1>(pre, tot, sums);
  auto issue = [&](int id, int st) {
    mbar_expect_tx(bars + st, row_bytes);
    bulk_g2s(ring + (size_t)st * row_bytes, a.store + (size_t)id * row_bytes, row_bytes, bars + st);
  };
  const int n_new = (int)tot[0];
  const int first = a.w.append_first ? stages - 1 : max(1, stages / 2 - 1);   // rows in flight at a time
  int q = (int)pre[0];
#pragma unroll
  for (int i = 0; i < kEntriesPerThread; ++i)              // of the thread's bits, those of rank f mod nf
    for (uint32_t m = mw[i]; m; m &= m - 1, ++q)
      if (q % nf == f) {
        const int id = (tid * kEntriesPerThread + i) * 32 + __ffs(m) - 1;
        ids[q / nf] = (unsigned short)id;
        if (q / nf < first) issue(id, q / nf);             // the first ones by whoever finds them
      }
  const int cnt = f < n_new ? (n_new - f + nf - 1) / nf : 0;
  int issued = min(first, cnt);                            // thread 0 from here on
  load_x(a, xs);
  Acc<kS> acc;

  int go = -1, stored = 0;                                 // thread 0: 1 / 0 once the plan says so; rows stored,
  int place = 0;                                           // the place of the next one
  bool moved = a.w.append_first;
  const int n_groups = (a.n_cache_ctas + a.group_size - 1) / a.group_size;
  // Thread 0: asks whether new rows may be stored, or (wait) until they may; then stores those below `upto`.
  auto learn = [&](bool wait) {
    const unsigned limit = wait ? a.spin_limit : min(1u, a.spin_limit);
    for (unsigned n = 0; n < limit && go < 0; ++n) {
      const unsigned long long v = ld_acquire64(&a.sync->plan);
      if (is_plan(a, v)) go = !(v & kPlanRefused);
    }
    if (go > 0) place = __ldcg(a.w.load_slots + f + stored * nf);
    for (unsigned n = 0; n < limit && go > 0 && !moved; ++n)
      moved = (int)(ld_acquire(&a.sync->groups_done) - (a.epoch + 1) * (unsigned)n_groups) >= 0;
    if (wait && (go < 0 || (go > 0 && !moved))) {          // rows stay as they are, or are overwritten too early
      plan_not_carried_out(a);
      if (go < 0) go = 0;
      moved = true;
    }
  };
  auto store_rows = [&](int upto) {
    for (; go > 0 && moved && stored < upto; ++stored) {
      asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(
                       a.cache + (size_t)place * row_bytes),
                   "r"(smem_u32(ring + (size_t)(stored % stages) * row_bytes)), "r"(row_bytes) : "memory");
      asm volatile("cp.async.bulk.commit_group;" ::: "memory");
      if (stored + 1 < cnt) place = __ldcg(a.w.load_slots + f + (stored + 1) * nf);
    }
  };
  if (tid == 0) {
    count_s = cnt;
    // Where rows are short the plan is there before the first one, and asking now is cheaper than between rows: 3 streams
    // at 1544 columns 160 us (4 layers), 160.9 without.  Wide rows' terms go ahead of the plan: 4 streams at 3704
    // columns, 2 layers, 230 us with the wait, 222.6 without.  Never in the paper's order, where this waits for the
    // moves and with them for the cached rows' terms: 2 x 1112, 4 layers, 96.4 us and 75.8, 3 x 4096 407 and 336.
    if (kS > 1 && cnt > 0 && a.w.append_first && !a.hand_over) learn(true);
  }
  __syncthreads();
  unsigned parity = 0;
  int from = cnt;                                          // first row that was not waited for any longer
  int given = 0;                                           // several streams: 1 partial, 2 last row handed over
  unsigned long long* last_down = a.last_down + (size_t)f * (d >> 1);
  unsigned long long* last_h = a.last_h + f * 8;
  for (int i = 0, st = 0; i < from; ++i) {
    const uint4* row = reinterpret_cast<const uint4*>(ring + (size_t)st * row_bytes);
    const bool is_last = kS > 1 && a.hand_over && i == cnt - 1;
    if (is_last) {                                         // the partial sum, while the last row travels
      if (i > 0) store_tagged_partial<kS>(acc, a.p_new + (size_t)f * S * (d >> 1), nvec, S, a.epoch + 1);
      given = 1;
    }
    const bool landed = mbar_wait(bars + st, parity, a.wait_polls);
    if (tid == 0 && landed && i + first < cnt) {           // the next one, in the stage of an earlier row?
      const bool reuse = i + first >= stages;
      if (go < 0 || (go > 0 && !moved)) {
        learn(reuse);
        store_rows(i);
      }
      if (go) {
        if (reuse) {
          asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        }
        issue(ids[i + first], st + first < stages ? st + first : st + first - stages);
        ++issued;
      } else {
        count_s = issued;                                  // refused: nothing more is brought in
      }
    }
    if (tid == 0 && landed && i + 1 < from) store_rows(i + 1);   // (the last one behind the partial sum)
    const float b = row_scalar<kGate>(a, ids[i], run, checked);
    if (is_last) {
#pragma unroll
      for (int k = 0; k < Shape<kS>::kChunks; ++k) {
        const int v = tid + k * kStepThreads;
        if (v < nvec) {
          const uint4 q = row[(kVec - 1) * nvec + v];
          store_tagged_word(last_down + v, q.x, a.epoch + 1);
          store_tagged_word(last_down + nvec + v, q.y, a.epoch + 1);
          store_tagged_word(last_down + 2 * nvec + v, q.z, a.epoch + 1);
          store_tagged_word(last_down + 3 * nvec + v, q.w, a.epoch + 1);
        }
      }
    }
    float p[kS], p2[kS];
#pragma unroll
    for (int s = 0; s < kS; ++s) p[s] = p2[s] = 0.f;
#pragma unroll
    for (int k = 0; k < Shape<kS>::kChunks; ++k) {
      const int v = tid + k * kStepThreads;
      if (v < nvec) {
        dot_chunk<kS>(p, row[v], xs, v, nvec, S);
        if (kGate == LIF_GATE_BUNDLED) dot_chunk<kS>(p2, row[nvec + v], xs, v, nvec, S);
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int s = 0; s < kS; ++s)
        if (kS == 1 || s < S) {
          p[s] += __shfl_xor_sync(0xffffffffu, p[s], o);
          if (kGate == LIF_GATE_BUNDLED) p2[s] += __shfl_xor_sync(0xffffffffu, p2[s], o);
        }
    if (lane == 0) {
#pragma unroll
      for (int s = 0; s < kS; ++s) {
        part[0][s][warp] = p[s];
        part[1][s][warp] = p2[s];
      }
    }
    if (__syncthreads_or(!landed)) {                       // flagged; this term and the later ones are left out
      if (tid == 0) {                                      // what is in flight gets another bounded chance
        timed_out(a);
        for (int j = i; j < issued; ++j) mbar_wait(bars + j % stages, (unsigned)(j / stages) & 1u);
      }
      from = i;
      break;
    }
    from = min(from, count_s);
    const uint4* down = row + (kVec - 1) * nvec;
    if (kS == 1) {
      float v1 = 0.f, v2 = 0.f;
#pragma unroll
      for (int w = 0; w < kStepWarps; ++w) {
        v1 += part[0][0][w];
        if (kGate == LIF_GATE_BUNDLED) v2 += part[1][0][w];
      }
      const float h = row_weight<kGate>(a, b, v1, v2);
      if (h != 0.f) axpy_row<kS>(acc, down, &h, nvec);
    } else {                                               // a warp per stream folds the 16 warps' sums
      if (warp < kS) {
        float v1 = part[0][warp][lane & (kStepWarps - 1)], v2 = part[1][warp][lane & (kStepWarps - 1)];
#pragma unroll
        for (int o = kStepWarps / 2; o > 0; o >>= 1) {
          v1 += __shfl_xor_sync(0xffffffffu, v1, o);
          v2 += __shfl_xor_sync(0xffffffffu, v2, o);
        }
        const float h = warp >= S ? 0.f : row_weight<kGate>(a, b, v1, v2);
        if (lane == 0) {
          h_s[warp] = h;
          if (is_last) store_tagged_word(last_h + warp, __float_as_uint(h), a.epoch + 1);
        }
      }
      if (is_last) {
        given = 2;
        break;
      }
      __syncthreads();
      axpy_row<kS>(acc, down, h_s, nvec);
    }
    __syncthreads();                                       // the stage, part[] and h_s[] are free
    if (++st == stages) {
      st = 0;
      parity ^= 1u;
    }
  }
  const bool hand_over = kS > 1 && a.hand_over;
  if (!hand_over ? cnt > 0 : cnt > 1 && given == 0)
    store_tagged_partial<kS>(acc, a.p_new + (size_t)f * S * (d >> 1), nvec, S, a.epoch + 1);
  if (hand_over && cnt > 0 && given < 2) {                    // given up: nothing comes of the last row
    for (int v = tid; v < d >> 1; v += kStepThreads) store_tagged_word(last_down + v, 0u, a.epoch + 1);
    if (tid < 8) store_tagged_word(last_h + tid, 0u, a.epoch + 1);
  }
  if (tid == 0) {
    if (cnt > 0 && (go < 0 || (go > 0 && !moved))) learn(true);
    store_rows(from);
    go_s = go;
  }
  if (from < cnt) {
    // The window state already names these rows, so they are filled all the same, with plain loads and
    // without the ring (in the paper's order thread 0 has waited until their places are free).
    __syncthreads();
    for (int i = from; i < cnt && go_s > 0; ++i) {
      const uint4* src = reinterpret_cast<const uint4*>(a.store + (size_t)ids[i] * row_bytes);
      uint4* dst = reinterpret_cast<uint4*>(a.cache + (size_t)__ldcg(a.w.load_slots + f + i * nf) * row_bytes);
      for (int v = tid; v < kVec * nvec; v += kStepThreads) dst[v] = ld_stream16(src + v);
    }
  }
  // (shared memory must outlive the reads of the last rows' copies to the cache)
  if (tid == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}

// One stream: two CTAs per SM, 64 registers and no spill, so that small layers' steps on several streams share the
// chip: eight layers of 768 x 3072 at once 35.2 us for a step of each, 57.9 with the bound at one CTA (107
// registers); four 18.4 and 30.4.  Layers one after the other are faster with that bound where nothing else is on
// the SM (768 x 3072, 4 layers 56.5 us against 59.0; three-vector bundles of 4096 columns 416 against 420) and
// slower where the next layer's predictor then finds no registers beside the step (opt6p7b, 8 layers 379 against
// 374; falcon7b, 4 layers 319 against 316).
// What spills at 64 registers is the row moves beside the sums: with four pieces in flight instead of two 64-72 bytes
// stored and 124-132 loaded per thread, 1424 x 4576 with the FFN over every cached row, 6 layers 100.8 us against 97.4,
// 768 x 3072 61.4 against 59.5.
template <int kGate, int kS>
__global__ void __launch_bounds__(kStepThreads, kS == 1 ? 2 : 1) step_kernel(StepArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ unsigned part_s, epoch_s;
  pdl_trigger();       // whatever follows waits for this kernel's end before it reads its results
  if (threadIdx.x == 0) {
    const unsigned long long ticket = atomicAdd(&a.sync->ticket, 1ull);
    epoch_s = (unsigned)(ticket / gridDim.x);
    part_s = (unsigned)(ticket % gridDim.x);
  }
  __syncthreads();
  const int part = (int)part_s;
  a.epoch = epoch_s;
  if (part == 0) window_role(a, smem);
  else if (part <= a.n_cache_ctas) cache_role<kGate, kS>(a, part - 1, smem);
  else if (part <= a.n_cache_ctas + kFetchCtas) fetch_role<kGate, kS>(a, part - 1 - a.n_cache_ctas, smem);
  else sum_role<kS>(a, part - 1 - a.n_cache_ctas - kFetchCtas, smem);
}

using StepKernel = void (*)(StepArgs);
StepKernel step_kernel_for(const lif_layer_desc& D) {
  if (D.n_streams > 1) {
    if (D.gate_mode != LIF_GATE_NONE) return nullptr;
    if (D.n_streams == 2 && D.d_model <= Shape<2>::kMaxD) return step_kernel<LIF_GATE_NONE, 2>;
    if (D.n_streams <= 4 && D.d_model <= Shape<4>::kMaxD) return step_kernel<LIF_GATE_NONE, 4>;
    if (D.n_streams <= 8 && D.d_model <= Shape<8>::kMaxD) return step_kernel<LIF_GATE_NONE, 8>;
    return nullptr;
  }
  if (D.gate_mode == LIF_GATE_BUNDLED) return step_kernel<LIF_GATE_BUNDLED, 1>;
  if (D.gate_mode == LIF_GATE_RESIDENT) return step_kernel<LIF_GATE_RESIDENT, 1>;
  return step_kernel<LIF_GATE_NONE, 1>;
}
constexpr int kGroupMax = 8, kUngroupedMax = 64, kUngroupedMaxStreams = 16;
// One step CTA per SM (with less, two fit and are put on one SM where others are not free yet), and beside it one of
// the next layer's low-rank predictor, 91 KB at 4096 x 128.  With several streams, whose cached rows are many and are
// added by fewer CTAs, what a CTA can have beside x: 6 streams at 3704 columns, 3 layers, 464 us with 112 KB, 441 with 128,
// 421 with 160, 416 with 192; 8 x 2048 254.6 and 246, 8 x 3704, one layer, 219 and 198.5; even where a CTA has few rows.
constexpr size_t kCacheRing = 112 * 1024, kCacheRingGate = 128 * 1024, kCacheRingStreams = 192 * 1024, kFetchRing = 32 * 1024;

// Streams x columns from which a fetch CTA hands its last row over instead of adding it to its partial.  us a token of
// 3 layers, never / always: 2 x 7168 800.6 / 792.4, 4 x 4096 463.6 / 459, 2 x 4096 184.6 / 178.8, 8 x 1024 97.6 / 95.5,
// 4 x 2048 153.1 / 152.2; 6 x 1032 105.8 / 104.2 and, with a third of the rows, 85.5 / 86.2, 3 x 2056 94.8 / 94.7; 3 x 1544
// 81 / 82.1, 2 x 2048 81.7 / 82.8, 2 x 1032 53.7 / 57.3: there a partial is short and the further words cost more.
constexpr int kHandOver = 8192;

// CTAs that add up the outputs: 16 pairs of columns or more each, which leaves 16 slices of the partials to
// a CTA's threads (several streams: 128 pairs).
int sum_ctas(const lif_layer_desc& D) {
  const int per = D.n_streams > 1 ? 128 : 16, most = D.n_streams > 1 ? 48 : 32;
  const int n = (D.n_streams * D.d_model / 2 + per - 1) / per;
  return n > most ? most : n;
}
// CTAs for the rows that are already cached, about a third of which are active in a step: with one
// stream a CTA per eight rows of the cache; with several one per sixteen, because a CTA's partial is
// as long as its streams' outputs together.
int cache_ctas(const lif_layer_desc& D, int n_sm) {
  const int per = D.n_streams > 1 ? 16 : 8;
  const int most = D.n_streams > 1 ? 64 : n_sm - 1 - kFetchCtas - sum_ctas(D);
  const int nc = (D.capacity + per - 1) / per;
  return nc < 8 ? 8 : (nc > most ? most : nc);
}
// Tagged partials of cache CTAs (or of groups of them) that the sum CTAs add up.
int hit_partials_max(const lif_layer_desc& D) {
  return D.n_streams > 1 ? kUngroupedMaxStreams : kUngroupedMax;
}

}  // namespace

size_t step_sync_bytes() { return sizeof(StepSync); }
size_t step_tagged_bytes(const lif_layer_desc& D) {
  if (!step_kernel_for(D)) return 0;
  return (size_t)(hit_partials_max(D) + kFetchCtas) * D.n_streams * D.d_model * 8 +
         (D.n_streams > 1 ? (size_t)kFetchCtas * (D.d_model * 4 + 8 * 8) : 0);
}

// Shape of the launch, and whether the single launch applies: streams x width in registers, ids and
// rows that fit 16 bits and the predictor's entries two per thread (d_ff <= 32768), the window CTA's
// arrays in shared memory.
cudaError_t step_configure(lif_layer* L) {
  const lif_layer_desc& D = L->desc;
  L->step_ok = 0;
  StepKernel kernel = step_kernel_for(D);
  if (!kernel || new_mask_entries(D) > kEntriesPerThread * kStepThreads || D.d_ff > 32768 ||
      new_mask_entry_bits(D) != 32 || D.window_k > 32767 || L->n_sm < 3 * kFetchCtas)   // (sum CTAs: <= 48)
    return cudaSuccess;
  int dev = 0, max_smem = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  e = cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return e;
  cudaFuncAttributes at;
  e = cudaFuncGetAttributes(&at, kernel);
  if (e != cudaSuccess) return e;
  max_smem -= (int)at.sharedSizeBytes;
  const size_t row = 2 * (size_t)row_elems(D), x = x_smem_bytes(D.d_model, D.n_streams);
  const size_t ids = 2 * (((size_t)D.d_ff + kFetchCtas - 1) / kFetchCtas);
  auto stages = [&](size_t ring, size_t other, int least) {
    while (ring > row * least && ring + other > (size_t)max_smem) ring -= row;
    const int s = (int)(ring / row);
    return s < least ? least : (s > 16 ? 16 : s);
  };
  L->step_cache_ctas = cache_ctas(D, L->n_sm);
  L->step_sum_ctas = sum_ctas(D);
  L->step_group = L->step_cache_ctas > hit_partials_max(D) ? kGroupMax : 1;
  const size_t hits = 2 * (((size_t)D.capacity + L->step_cache_ctas - 1) / L->step_cache_ctas);
  L->step_cache_stages = stages(D.n_streams > 1 ? kCacheRingStreams
                                : D.gate_mode == LIF_GATE_RESIDENT ? kCacheRingGate : kCacheRing, x + hits, 1);
  // (paper's cache order: bundles wait in the ring, see fetch_role; twice the ring keeps the link busy)
  L->step_fetch_stages = stages(D.append_first ? kFetchRing : 2 * kFetchRing, x + ids, 2);
  size_t smem = window_role_smem(D.d_ff, D.capacity, D.ffn_mode == 1);
  const size_t need_c = x + L->step_cache_stages * row + hits, need_f = x + L->step_fetch_stages * row + ids;
  if (need_c > smem) smem = need_c;
  if (need_f > smem) smem = need_f;
  if (smem < kSumSmem) smem = kSumSmem;
  if (smem > (size_t)max_smem) return cudaSuccess;
  L->step_smem = smem;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem);
  if (e != cudaSuccess) return e;
  L->step_ok = 1;
  return cudaSuccess;
}

cudaError_t launch_step(lif_layer* L, const __half* x, float* y, cudaStream_t st) {
  const lif_layer_desc& D = L->desc;
  StepArgs a;
  a.w = window_args(L, L->active_idx, L->n_tmp);
  a.new_entries = L->new_mask_words;
  a.n_entries = new_mask_entries(D);
  a.act_entries = L->new_mask_words + a.n_entries;
  a.row_words = L->new_mask_words + row_words_at(D);
  a.gate_words = L->new_mask_words + gate_words_at(D);
  a.predictor_run = L->counts + CNT_PREDICTOR_RUN;
  a.next_run = (int*)(L->counts + CNT_PREDICTOR_RUN);
  a.n_act_out = L->n_tmp;
  a.row_stamps = L->row_stamps;
  a.hit_rows = L->hit_rows;
  a.store = (const unsigned char*)L->dev_bundles;
  a.cache = (unsigned char*)D.dev_cache;
  a.x = x;
  a.gate_val = L->gate_val;
  a.b_down = (const __half*)D.dev_bias_down;
  a.p_member = L->y_partial;
  a.p_hit = (uint4*)L->step_tagged;
  a.p_new = a.p_hit + (size_t)hit_partials_max(D) * D.n_streams * (D.d_model / 2);
  a.hand_over = D.n_streams > 1 && D.n_streams * D.d_model >= kHandOver;
  a.last_down = (unsigned long long*)(a.p_new + (size_t)kFetchCtas * D.n_streams * (D.d_model / 2));
  a.last_h = a.last_down + (size_t)kFetchCtas * (D.d_model / 2);
  a.y = y;
  a.sync = (StepSync*)L->step_sync;
  a.d = D.d_model;
  a.n_streams = D.n_streams;
  a.whole_cache = D.ffn_mode == 1;
  a.act = D.activation;
  a.act_thr = D.activation_threshold;
  a.n_cache_ctas = L->step_cache_ctas;
  a.n_sum_ctas = L->step_sum_ctas;
  a.group_size = L->step_group;
  a.cache_stages = L->step_cache_stages;
  a.fetch_stages = L->step_fetch_stages;
  a.hits_max = (D.capacity + a.n_cache_ctas - 1) / a.n_cache_ctas;
  a.wait_polls = L->wait_polls;
  a.spin_limit = L->spin_limit;
  return launch_k(step_kernel_for(D), dim3(1 + a.n_cache_ctas + kFetchCtas + a.n_sum_ctas),
                  dim3(kStepThreads), L->step_smem, st, L->use_pdl, a);
}

}  // namespace lif
