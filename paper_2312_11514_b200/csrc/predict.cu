// Low-rank sparsity predictor (Section 3.1, "Anticipating ReLU Sparsity"; Appendix B):
// scores = x.A.B + c, active iff score > theta, compacted to an ascending index list.
//
// One launch for both contractions, fp16 factors with fp32 sums.  Its CTAs take parts in the order in
// which they start:
//   z CTAs      (first)  8 columns of z = x.A for one, two or four streams, finished: every value is
//                        stored as one word with the number of this launch; or (z_by_parts) the sums of one
//                        part of A's rows for all columns and streams, which the score CTAs add up
//   score CTAs  (then)   128 neurons: re-read the words of z until they carry the number, then
//                        scores = z.B + c, threshold, bit mask; on request the last one to finish turns
//                        the mask into the sorted list with a block prefix sum
// A CTA waits only for CTAs that took their parts before it; the wait is bounded.
//
// Bound: latency.  The factors are weights and are on chip before the input is complete (the kernel is
// resident while the one ahead still runs); behind the dependency wait there is x, the sums and one
// exchange of z.  As two kernels the exchange was a kernel boundary (1.3 us), 32 partial sums per value of z
// that every score CTA added up again (1 us) and a tile of B that could not be asked for before the first
// stage had started.
//
// Orders of additions are fixed, the same for any number of streams, and independent of the launch shape,
// so the decisions are, too: rows of A in `parts` of `rows` consecutive ones; a part in `lanes` interleaved
// runs, each added in row order, then the runs in order, then the parts in order; rows of B in 16
// interleaved runs, then the runs in order.
#include "lif_internal.cuh"
#include "mask_compact.cuh"

namespace lif {
namespace {

struct PredictArgs {
  const __half *x, *A, *B;
  const float* c;
  float theta;
  int d, r, F, keep, compact, first_pass, by_parts;
  // stage 1: runs of rows, `per` rows each; CTAs per column group; streams and columns per CTA
  int parts, rows, lanes, per, groups_of_streams, h, cw, n_z, x_at, red_at;
  // stage 2
  int n_scores, staged_b;
  unsigned long long* z;            // [S][r] {value, launch}
  unsigned long long* tickets;      // nullptr: parts by CTA number, z as it is (one half, profiled alone)
  int launch;                       // number of this launch of the layer's predictor (filled in by the kernel)
  unsigned long long* entries;      // see lif_layer::new_mask_words
  const int32_t* slot_of;
  int* predictor_run;
  int32_t* status;
  unsigned spin_limit;
  float* logits;
  uint32_t* mask_words;
  int* done;                        // counter of finished score CTAs (compaction)
  int *active_idx, *n_active;
  int8_t* keep_tok;
};

// ---- stage 1 -------------------------------------------------------------------------------------------
// A CTA computes 8 columns of H streams, CW at a time (all 8 unless the sums of its runs would not fit).
// Run q = lane * parts + part belongs to thread q mod 256; a thread goes through its runs one after the
// other.  Its pieces of A (one row, 8 columns) travel into its own slots of shared memory ahead of the
// dependency wait.
//
// Where the kernel ahead is known to be the step of the layer before (a token's later layers in lif_graph_capture and
// lif_decode_token_host), which lets this one start early, everything behind the wait is executed once before it,
// on whatever the buffers hold, and the results dropped: a kernel's code comes from L2 at its first use (opt6p7b,
// 8 layers 373.7 us a token, 375.1 without; tiny 24.75 and 24.9).  Behind anything else, such as another library's
// kernel that releases nothing early, the wait is over when this kernel starts and that pass would be in the way:
// two matrix products between the layers of a captured program, 4 layers of 4096 x 16384 330 us with it and
// 324 without, 2048 x 8192 154.6 and 148, 768 x 3072 90.3 and 85.1 (with steps back to back there is no difference).
// The score CTAs have such a pass in either case, while z is computed.
template <int H, int CW>
__device__ void z_role(const PredictArgs& a, int S, int part_of_grid, unsigned char* smem) {
  constexpr int Q = H * CW;
  const int tid = threadIdx.x;
  const int cg = part_of_grid / a.groups_of_streams, s0 = (part_of_grid % a.groups_of_streams) * H;
  uint4* a_s = reinterpret_cast<uint4*>(smem) + tid;                   // [rows of the first runs][256], ...
  __half* x_s = reinterpret_cast<__half*>(smem + a.x_at);              // [H][d + 2 parts]: parts 2 apart
  float* red = reinterpret_cast<float*>(smem + a.red_at);              // [lanes][parts][Q]
  const int n_runs = a.lanes * a.parts, stride = kThreads / (a.r >> 3);
  float* part_z = red + (size_t)n_runs * Q;                            // [parts][Q]
  const int x_len = a.d + 2 * a.parts;
  const __half* A = a.A + cg * 8;

  // the first run's part and row, and the way from one run to the thread's next
  const int part0 = tid % a.parts, m00 = part0 * a.rows + tid / a.parts;
  const int dp = kThreads % a.parts, dm = dp * a.rows + kThreads / a.parts;
  uint4* to = a_s;
  for (int q0 = 0, part = part0, m0 = m00; q0 + tid < n_runs; q0 += kThreads) {
    const int end = min(a.d, (part + 1) * a.rows), wide = min(kThreads, n_runs - q0);
    uint4* row = to;
    for (int m = m0; m < end; m += stride, row += wide) copy_async16(row, A + (size_t)m * a.r);
    to += a.per * wide;
    m0 += dm;
    part += dp;
    if (part >= a.parts) {
      part -= a.parts;
      m0 += 1 - a.parts * a.rows;
    }
  }
#pragma unroll 1
  for (int pass = a.first_pass; pass < 2; ++pass) {
    if (pass) {
      pdl_wait();
      pdl_trigger();
    }
#pragma unroll 1
    for (int i = tid; i < (a.d >> 3); i += 2 * kThreads) {             // 8 rows, all of one part
      uint4 v[2][H];
#pragma unroll
      for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int h = 0; h < H; ++h)                                    // (past L1: the first pass may see an old x)
          v[k][h] = __ldcg(reinterpret_cast<const uint4*>(a.x + (size_t)min(s0 + h, S - 1) * a.d) +
                           min(i + k * kThreads, (a.d >> 3) - 1));
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int m = 8 * min(i + k * kThreads, (a.d >> 3) - 1);
        uint32_t* dst = reinterpret_cast<uint32_t*>(x_s + m + 2 * (m / a.rows));
#pragma unroll
        for (int h = 0; h < H; ++h) {
          uint32_t* to = dst + h * (x_len >> 1);
          to[0] = v[k][h].x;
          to[1] = v[k][h].y;
          to[2] = v[k][h].z;
          to[3] = v[k][h].w;
        }
      }
    }
    if (pass) own_copies_wait();
    __syncthreads();
#pragma unroll 1
    for (int c0 = 0; c0 < 8; c0 += CW) {
      int part = part0, m0 = m00;
      const uint4* from = a_s;
#pragma unroll 1
      for (int q = tid; q < n_runs; q += kThreads) {
        const int end = min(a.d, (part + 1) * a.rows), wide = min(kThreads, n_runs - q + tid);
        const __half* xr = x_s + 2 * part;
        float2 acc[H][CW / 2];
#pragma unroll
        for (int h = 0; h < H; ++h)
#pragma unroll
          for (int k = 0; k < CW / 2; ++k) acc[h][k] = make_float2(0.f, 0.f);
        auto add = [&](const uint4& row, int m) {
          const __half2* pairs = reinterpret_cast<const __half2*>(&row);
          float2 f[CW / 2];
#pragma unroll
          for (int k = 0; k < CW / 2; ++k) f[k] = __half22float2(pairs[CW == 8 ? k : c0 / 2 + k]);
#pragma unroll
          for (int h = 0; h < H; ++h) {
            const float xv = __half2float(xr[h * x_len + m]);
#pragma unroll
            for (int k = 0; k < CW / 2; ++k) acc[h][k] = fma2(make_float2(xv, xv), f[k], acc[h][k]);
          }
        };
        int m = m0;
        const uint4* row = from;
#pragma unroll 1
        for (; m + 3 * stride < end; m += 4 * stride, row += 4 * wide) {
          const uint4 r0 = row[0], r1 = row[wide], r2 = row[2 * wide], r3 = row[3 * wide];
          add(r0, m);
          add(r1, m + stride);
          add(r2, m + 2 * stride);
          add(r3, m + 3 * stride);
        }
#pragma unroll 1
        for (; m < end; m += stride, row += wide) add(row[0], m);
        from += a.per * wide;
        m0 += dm;
        part += dp;
        if (part >= a.parts) {
          part -= a.parts;
          m0 += 1 - a.parts * a.rows;
        }
        float2* dst = reinterpret_cast<float2*>(red + (size_t)q * Q);
#pragma unroll
        for (int h = 0; h < H; ++h)
#pragma unroll
          for (int k = 0; k < CW / 2; ++k) dst[h * (CW / 2) + k] = acc[h][k];
      }
      __syncthreads();
      const int sums = a.parts * Q;
#pragma unroll 1
      for (int i = tid; i < sums; i += kThreads) {
        float v = 0.f;
#pragma unroll 8
        for (int l = 0; l < a.lanes; ++l) v += red[(size_t)l * sums + i];
        part_z[i] = v;
      }
      __syncthreads();
      if (tid < Q) {
        float v = 0.f;
#pragma unroll 8
        for (int p = 0; p < a.parts; ++p) v += part_z[p * Q + tid];
        const int s = s0 + tid / CW;
        if (pass && s < S)
          store_with_run(a.z + (size_t)s * a.r + cg * 8 + c0 + tid % CW, __float_as_uint(v), a.launch);
      }
    }
  }
}

// Where a column group is too long or there are too few of them: a CTA adds one part of A's rows, all columns
// and streams, and hands over the part's sums.  A's pieces travel into the thread's own slots of shared memory
// ahead of the wait, whole rows at a time.
template <int S>
__device__ void z_part_role(const PredictArgs& a, int part, unsigned char* smem) {
  const int tid = threadIdx.x, ncg = a.r >> 3, stride = kThreads / ncg;
  const int cg = tid % ncg, lane = tid / ncg;
  const int m0 = part * a.rows, m1 = min(a.d, m0 + a.rows);
  uint4* a_s = reinterpret_cast<uint4*>(smem) + tid;                   // [per][kThreads]
  __half* x_s = reinterpret_cast<__half*>(smem + a.x_at);              // [S][rows]
  float* red = reinterpret_cast<float*>(smem + a.red_at);              // [lanes][r]
  for (int u = 0, m = m0 + lane; lane < stride && m < m1; ++u, m += stride)
    copy_async16(a_s + u * kThreads, a.A + (size_t)m * a.r + cg * 8);
#pragma unroll 1
  for (int pass = a.first_pass; pass < 2; ++pass) {
    if (pass) {
      pdl_wait();
      pdl_trigger();
    }
    const int vecs = (m1 - m0) >> 3;
#pragma unroll 1
    for (int i = tid; i < S * vecs; i += kThreads) {
      const int s = i / vecs, v = i - s * vecs;
      reinterpret_cast<uint4*>(x_s + s * a.rows)[v] = __ldcg(reinterpret_cast<const uint4*>(a.x + (size_t)s * a.d + m0) + v);
    }
    if (pass) own_copies_wait();
    __syncthreads();
    float2 acc[S][4];
#pragma unroll
    for (int s = 0; s < S; ++s)
#pragma unroll
      for (int k = 0; k < 4; ++k) acc[s][k] = make_float2(0.f, 0.f);
    const uint4* row = a_s;
#pragma unroll 2
    for (int m = lane; m < (lane < stride ? m1 - m0 : 0); m += stride, row += kThreads) {
      float2 f[4];
      unpack8(*row, f);
#pragma unroll
      for (int s = 0; s < S; ++s) {
        const float xv = __half2float(x_s[s * a.rows + m]);
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[s][k] = fma2(make_float2(xv, xv), f[k], acc[s][k]);
      }
    }
#pragma unroll
    for (int s = 0; s < S; ++s) {
      if (lane < a.lanes) {
        float2* dst = reinterpret_cast<float2*>(red + lane * a.r + cg * 8);
#pragma unroll
        for (int k = 0; k < 4; ++k) dst[k] = acc[s][k];
      }
      __syncthreads();
      for (int j = tid; j < a.r; j += kThreads) {
        float v = 0.f;
#pragma unroll 8
        for (int l = 0; l < a.lanes; ++l) v += red[l * a.r + j];
        if (pass) store_with_run(a.z + ((size_t)part * S + s) * a.r + j, __float_as_uint(v), a.launch);
      }
      __syncthreads();
    }
  }
}

// ---- stage 2 -------------------------------------------------------------------------------------------
constexpr int kPartWords = 8;          // words of parts' sums that a thread asks for at a time

// streams side by side in shared memory: 1, 2, 4 or 8
__host__ __device__ constexpr int padded(int S) { return S <= 2 ? S : (S <= 4 ? 4 : 8); }

// Thread (rs, cg) holds rows rs, rs + 16, ... of 8 columns of the CTA's tile of B: the first 128 rows are put in
// flight into registers and the next ones into its own slots of shared memory before the wait.
template <int S>
__device__ void score_role(const PredictArgs& a, int tile, unsigned char* smem) {
  constexpr int SP = padded(S);
  float* zs = reinterpret_cast<float*>(smem);                          // [r][SP]
  uint4* b_s = reinterpret_cast<uint4*>(zs + SP * a.r);                // [staged][kThreads]
  float* red = reinterpret_cast<float*>(b_s + a.staged_b * kThreads);  // [S][16][kLogitTile], or the parts' sums
  __shared__ uint32_t act_w[S][kLogitTile / 32];
  __shared__ int warp_sums[kThreads / 32];
  __shared__ int is_last;
  const int tid = threadIdx.x, r = a.r, F = a.F, n_entries = a.n_scores * (kLogitTile / 32);
  const int cg = tid & 15, rs = tid >> 4;
  const int col = tile * kLogitTile + cg * 8;
  uint4 bq[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int j = rs + 16 * u;
    bq[u] = (col < F && j < r) ? ld_stream16(a.B + (size_t)j * F + col) : make_uint4(0, 0, 0, 0);
  }
  for (int u = 0; u < a.staged_b; ++u) {
    const int j = rs + 16 * (8 + u);
    if (col < F && j < r) copy_async16(b_s + u * kThreads + tid, a.B + (size_t)j * F + col);
  }
  const int n = tid & (kLogitTile - 1), my_col = tile * kLogitTile + n;
  const float my_c = my_col < F ? a.c[my_col] : 0.f;
  // (behind a launch of the first stage, whose CTAs were past their wait before this one could start)
  if (!a.tickets && !a.compact) pdl_trigger();
  int run = 0;
#pragma unroll 1
  for (int pass = S > 1; pass < 2; ++pass) {                           // (see stage 1; z takes longer than this)
    if (pass) {
      pdl_wait();
      // What follows (the window kernel or the single-launch step) reads ahead of its own wait only what was
      // complete before this one passed, and words that carry this run's number.  (A compacting run is
      // followed by a kernel that can do nothing before its list: it is released when z is there.)
      if (!a.compact) pdl_trigger();
    }
    run = __ldcg(a.predictor_run);
    // Whether the neuron already has a cache row is read here, so the mask of neurons to bring in
    // (active and not cached) costs no round trip of its own.
    const int my_row = my_col < F ? __ldcg(a.slot_of + my_col) : 0;
    {
      unsigned polls = 0;
      if (a.by_parts) {
        // All words of all parts side by side, then each value's in order.  (With a thread per value they came in four
        // round trips one after the other: 3072 x 6144, rank 48, 4 layers 91.7 us, now 84.5; 16 words a thread
        // at a time 90.3, and 8 without the loads past the end 1 to 7 % more from 1024 words on.)
        const int n_z = S * r, n_words = a.parts * n_z;
        float* part_z = red;                             // [parts][S][r] (a pass's scores there have been read, or
                                                         // are dropped)
#pragma unroll 1
        for (int i0 = tid; i0 < n_words; i0 += kPartWords * kThreads) {
          unsigned long long v[kPartWords];
          bool there;
          do {
            there = true;
#pragma unroll
            for (int k = 0; k < kPartWords; ++k) {
              asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v[k])
                           : "l"(a.z + min(i0 + k * kThreads, n_words - 1)) : "memory");
              there = there && (!a.tickets || (int)(v[k] >> 32) == a.launch);
            }
          } while (pass && !there && polls++ < a.spin_limit);
          if (pass && !there) flag_timeout(a.status);
#pragma unroll
          for (int k = 0; k < kPartWords; ++k)           // not there: no neuron is active
            if (i0 + k * kThreads < n_words)
              part_z[i0 + k * kThreads] = there ? __uint_as_float((unsigned)v[k]) : __int_as_float(0x7fffffff);
        }
        __syncthreads();
        for (int i = tid; i < n_z; i += kThreads) {
          float sum = 0.f;
#pragma unroll 8
          for (int p = 0; p < a.parts; ++p) sum += part_z[p * n_z + i];
          zs[S == 1 ? i : (i % r) * SP + i / r] = sum;
        }
      }
      for (int j = tid; !a.by_parts && j < r; j += kThreads) {
        unsigned long long v[S];
        bool there;
        do {
          there = true;
#pragma unroll
          for (int k = 0; k < S; ++k) {
            asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v[k]) : "l"(a.z + (size_t)k * r + j) : "memory");
            there = there && (!a.tickets || (int)(v[k] >> 32) == a.launch);
          }
        } while (pass && !there && polls++ < a.spin_limit);
        if (pass && !there) flag_timeout(a.status);
#pragma unroll
        for (int k = 0; k < S; ++k)                                      // not there: no neuron is active
          zs[j * SP + k] = there ? __uint_as_float((unsigned)v[k]) : __int_as_float(0x7fffffff);
      }
    }
    if (pass && a.compact) pdl_trigger();
    if (pass) own_copies_wait();
    __syncthreads();

    float2 acc[S][4];
#pragma unroll
    for (int s = 0; s < S; ++s)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[s][e] = make_float2(0.f, 0.f);
#pragma unroll 1
    for (int j0 = 0; j0 < (pass ? r : min(r, 128)); j0 += 128) {       // (the first pass leaves bq as it is)
      if (j0 > 0) {
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int j = j0 + rs + 16 * u, at = (j0 >> 4) - 8 + u;
          bq[u] = make_uint4(0, 0, 0, 0);
          if (col < F && j < r)
            bq[u] = at < a.staged_b ? b_s[at * kThreads + tid] : ld_stream16(a.B + (size_t)j * F + col);
        }
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int j = j0 + rs + 16 * u;
        if (j < r) {
          float2 bf[4];
          unpack8(bq[u], bf);
#pragma unroll
          for (int s = 0; s < S; ++s) {
            const float zz = zs[j * SP + s];
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[s][e] = fma2(make_float2(zz, zz), bf[e], acc[s][e]);
          }
        }
      }
    }
#pragma unroll
    for (int s = 0; s < S; ++s) {
      float4* dst = reinterpret_cast<float4*>(red + (s * 16 + rs) * kLogitTile + cg * 8);
      dst[0] = make_float4(acc[s][0].x, acc[s][0].y, acc[s][1].x, acc[s][1].y);
      dst[1] = make_float4(acc[s][2].x, acc[s][2].y, acc[s][3].x, acc[s][3].y);
    }
    __syncthreads();
    // two streams at a time: a warp holds 32 neighbouring neurons of one stream
    unsigned active_w = 0;                                               // one stream: of the thread's warp
#pragma unroll
    for (int s0 = 0; s0 < S; s0 += 2) {
      const int s = s0 + (tid >> 7);
      if (s < S) {
        float v = 0.f;
#pragma unroll
        for (int k = 0; k < 16; ++k) v += red[(s * 16 + k) * kLogitTile + n];
        v += my_c;
        if (pass && a.logits && my_col < F) a.logits[(size_t)s * F + my_col] = v;
        active_w = __ballot_sync(0xffffffffu, my_col < F && v > a.theta);
        if (S > 1 && (tid & 31) == 0) act_w[s][n >> 5] = active_w;
      }
    }
    if (S > 1) __syncthreads();
    if (tid < kLogitTile) {
      unsigned m = 0;
      int last_kept = -1;        // speculative mode: last token < keep in which the neuron is active
#pragma unroll
      for (int s = 0; s < S; ++s) {
        const unsigned w = S == 1 ? active_w : act_w[s][tid >> 5];
        m |= w;
        if (s < a.keep && ((w >> (tid & 31)) & 1u)) last_kept = s;
      }
      if (pass && a.keep_tok && my_col < F) a.keep_tok[my_col] = (int8_t)last_kept;
      const bool active = (m >> (tid & 31)) & 1u;
      const unsigned mn = __ballot_sync(0xffffffffu, active && my_row < 0);
      if (pass && (tid & 31) == 0) {
        const int word = tile * (kLogitTile / 32) + (tid >> 5);
        a.mask_words[word] = m;
        // the neurons to bring in together with this run's number, in one store: a kernel that is already
        // resident re-reads the entry until the number is the run's
        store_with_run(a.entries + word, mn, run);
        if (!a.compact) store_with_run(a.entries + n_entries + word, m, run);   // and the active ones themselves
      }
      if (pass && !a.compact && active && my_row >= 0)                           // ... with the row of each that has one
        store_with_run(a.entries + 2 * n_entries + my_col, (uint32_t)my_row, run);
    }
  }
  if (!a.compact) return;     // the consumer reads the bit mask itself
  compact_mask_last_cta(a.mask_words, n_entries, a.n_scores, a.done, a.active_idx, a.n_active, warp_sums, &is_last);
  // every CTA has read this run's number: the next run gets one of its own (in a decode step
  // that reads the mask itself, the kernel that ends the step does this)
  if (is_last && tid == 0) advance_run(a.predictor_run, run);
}

template <int S>
__global__ void __launch_bounds__(kThreads, 2) predict_kernel(PredictArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ unsigned part_s, launch_s;
  unsigned part = blockIdx.x;
  if (a.tickets) {          // (they only grow: a ticket tells the launch as well as the part)
    if (threadIdx.x == 0) {
      const unsigned long long ticket = atomicAdd(a.tickets, 1ull);
      launch_s = (unsigned)(ticket / gridDim.x) + 1u;
      part_s = (unsigned)(ticket % gridDim.x);
    }
    __syncthreads();
    part = part_s;
    a.launch = (int)launch_s;
  }
  if (part >= (unsigned)a.n_z) score_role<S>(a, (int)part - a.n_z, smem);
  else if (a.by_parts) z_part_role<S>(a, (int)part, smem);
  else if (a.cw == 2) z_role<1, 2>(a, S, (int)part, smem);
  else if (a.cw == 4) z_role<1, 4>(a, S, (int)part, smem);
  else if (S == 1 || a.h == 1) z_role<1, 8>(a, S, (int)part, smem);
  else if (a.h == 2) z_role<2, 8>(a, S, (int)part, smem);
  else z_role<4, 8>(a, S, (int)part, smem);
}

using PredictKernel = void (*)(PredictArgs);
PredictKernel predict_kernel_for(int S) {
  switch (S) {
    case 1: return predict_kernel<1>;
    case 2: return predict_kernel<2>;
    case 3: return predict_kernel<3>;
    case 4: return predict_kernel<4>;
    case 5: return predict_kernel<5>;
    case 6: return predict_kernel<6>;
    case 7: return predict_kernel<7>;
  }
  return predict_kernel<8>;
}

constexpr int kMaxStaged = 12;         // pieces of B per thread in shared memory: 48 KB
constexpr size_t kSharedSmem = 100 * 1024;   // ... with which two predictor CTAs still fit an SM
constexpr size_t kFewColumns = 40 * 1024, kFewColumnsTwo = 64 * 1024;   // see predict_shape
constexpr int kColumnCtas = 128;       // z CTAs at most, as long as a CTA can take more streams
constexpr size_t kZSmem = 200 * 1024;  // bytes of shared memory that a z CTA takes with more than 2 columns at a
                                       // time, one stream
constexpr size_t kZSmemStreams = 224 * 1024;   // ... that it takes with more streams (all 8 columns at a time)

// The launch shape of the two stages and their shared memory.
struct PredictSmem {
  size_t z, scores;
};
PredictSmem predict_shape(const lif_layer_desc& D, PredictArgs& a) {
  const int S = D.n_streams, d = D.d_model, r = D.rank;
  a.d = d;
  a.r = r;
  a.F = D.d_ff;
  a.parts = z_part_count(d);
  a.rows = z_rows_per_part(d);
  a.lanes = kThreads / (r / 8);
  a.per = (a.rows + a.lanes - 1) / a.lanes;
  if (a.lanes > a.rows) a.lanes = a.rows;                    // (runs without rows)
  const size_t runs = (size_t)a.lanes * a.parts;
  a.x_at = (int)(runs * a.per) * 16;
  auto sums_at = [&](int h) { return (a.x_at + h * (d + 2 * a.parts) * 2 + 15) / 16 * 16; };
  // Several streams share a CTA where there would be too many CTAs otherwise (A is read again from L2 by
  // each), as long as their x and sums fit: four do but for the widest layers (8000 columns at rank 264: 230 KB).
  a.h = 1;
  while (S > a.h && a.h < 4 && (r / 8) * ((S + a.h - 1) / a.h) > kColumnCtas &&
         sums_at(2 * a.h) + (runs + a.parts) * 2 * a.h * 8 * 4 <= kZSmemStreams) a.h *= 2;
  a.groups_of_streams = (S + a.h - 1) / a.h;
  a.n_z = r / 8 * a.groups_of_streams;
  a.red_at = sums_at(a.h);
  a.n_scores = (D.d_ff + kLogitTile - 1) / kLogitTile;
  a.staged_b = (r + 15) / 16 - 8;
  a.staged_b = a.staged_b < 0 ? 0 : (a.staged_b > kMaxStaged ? kMaxStaged : a.staged_b);
  PredictSmem m;
  // (many runs, at small ranks: fewer columns at a time)
  a.cw = 8;
  while (a.h == 1 && a.cw > 2 && a.red_at + (runs + a.parts) * a.cw * 4 > kZSmem) a.cw /= 2;
  m.z = a.red_at + (runs + a.parts) * a.h * a.cw * 4;
  // By parts, or by columns: a z CTA of columns has all rows to add, and at small ranks so many runs that their sums
  // fit only for 4 or 2 columns at a time; of parts' sums every score CTA reads parts * S * rank words.  us a token,
  // 4 layers (several streams: 3), d_ff = 2 d, columns / parts:
  //   one stream, ranks to 64: 1024 x 16 50.7 / 50.4, 2048 x 32 67.7 / 62.7, 2048 x 64 64.1 / 62.8, 4096 x 48 120.9 /
  //     113, 6128 x 16 264.5 / 221.6 (512 x 32 43.7 / 45 when the words came in four rounds); beyond, where the CTA
  //     would fill an SM: 4096 x 96 123.1 / 119.5, but 2048 x 96 62.3 / 63.4 and 3072 x 96 86.9 / 89.7;
  //   two, ranks below 64: 1544 x 32 59.9 / 57, 2048 x 16 69.3 / 65.5, 4096 x 32 116.3 / 113.4, but 1024 x 16 47.6 /
  //     48.1 and 2048 x 64 67.2 / 69.1;
  //   more: with 2 columns at a time 4 x 6128 x 16 366 / 340, 6 x 5120 x 16 385 / 355, 8 x 5120 x 16 442 / 420; with 4
  //     columns 3 x 4096 x 16 165 / 156.5, 4 x 4096 x 16 195.5 / 192.2, 5 x 4608 x 16 (2 layers) 198.4 / 191.9,
  //     8 x 4096 x 16 299 / 316; with 8 columns 3 x 2048 x 32 80.2 / 81.9, 4 x 4096 x 32 180 / 185.6, 8 x 2048 x 16
  //     131.3 / 140.2.
  const size_t z_part = (size_t)a.per * kThreads * 16 + S * a.rows * 2 + (size_t)a.lanes * r * 4;
  const bool parts_pay = S == 1   ? (r <= 64 && m.z > kFewColumns) || m.z > kSharedSmem
                         : S == 2 ? r < 64 && m.z > kFewColumnsTwo
                                  : a.h == 1 && (a.cw == 2 || (a.cw == 4 && S <= 5));
  a.by_parts = parts_pay && z_part <= kSharedSmem;
  if (a.by_parts) {
    a.n_z = a.parts;
    a.x_at = a.per * kThreads * 16;
    a.red_at = a.x_at + S * a.rows * 2;
    m.z = z_part;
  }
  const size_t scores = (size_t)S * 16 * kLogitTile * 4, part_sums = a.by_parts ? (size_t)a.parts * S * r * 4 : 0;
  m.scores = (size_t)padded(S) * r * 4 + (size_t)a.staged_b * kThreads * 16 + (part_sums > scores ? part_sums : scores);
  return m;
}

PredictArgs predict_args(const lif_layer* L, PredictSmem& smem) {
  const lif_layer_desc& D = L->desc;
  PredictArgs a = {};
  smem = predict_shape(D, a);
  a.A = (const __half*)D.dev_pred_A;
  a.B = (const __half*)D.dev_pred_B;
  a.c = D.dev_pred_c;
  a.theta = D.threshold_logit;
  a.keep = D.spec_keep;
  a.z = L->new_mask_words + z_words_at(D);
  a.entries = L->new_mask_words;
  a.slot_of = L->slot_of;
  a.predictor_run = (int*)(L->counts + CNT_PREDICTOR_RUN);
  a.status = L->counts + LIF_CNT_STATUS;
  a.spin_limit = L->predictor_polls;
  a.mask_words = L->mask_words;
  a.done = (int*)(L->counts + CNT_TICKET_PREDICT);
  a.keep_tok = L->keep_tok;
  return a;
}

// One stage as a launch of its own.
cudaError_t launch_stage(const lif_layer* L, PredictArgs a, const PredictSmem& smem, bool z, cudaStream_t st) {
  a.tickets = nullptr;
  const int grid = z ? a.n_z : a.n_scores;
  if (!z) a.n_z = 0;
  return launch_k2(predict_kernel_for(L->desc.n_streams), dim3(grid), dim3(kThreads), z ? smem.z : smem.scores, st,
                   L->use_pdl, L->single_step, a);
}

}  // namespace

bool z_by_parts(const lif_layer_desc& D) {
  PredictArgs a = {};
  if (D.gate_mode != LIF_GATE_RESIDENT) predict_shape(D, a);
  return a.by_parts != 0;
}

// Opt-ins of the kernel (once per layer).
cudaError_t predict_configure(const lif_layer* L) {
  if (L->desc.gate_mode == LIF_GATE_RESIDENT) return cudaSuccess;
  const void* k = (const void*)predict_kernel_for(L->desc.n_streams);
  cudaFuncAttributes at;
  cudaError_t e = cudaFuncGetAttributes(&at, k);
  if (e != cudaSuccess) return e;
  PredictArgs a = {};
  const PredictSmem m = predict_shape(L->desc, a);
  const size_t most = L->max_smem - at.sharedSizeBytes;
  if (m.z > most || m.scores > most) return cudaErrorInvalidConfiguration;   // (no accepted layer: z at most 224 KB)
  return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
}

cudaError_t launch_predict_one(lif_layer* L, int kernel, const __half* x, cudaStream_t st) {
  const lif_layer_desc& D = L->desc;
  if (D.n_streams != 1) return cudaErrorInvalidValue;
  if (D.gate_mode == LIF_GATE_RESIDENT)
    return kernel == LIF_KERNEL_PREDICT_SCORES
               ? launch_gate_predict(L, x, nullptr, L->active_idx, L->n_tmp, st, nullptr,
                                     L->fused_plan ? 0 : 1, false)
               : cudaErrorInvalidValue;
  PredictSmem smem;
  PredictArgs a = predict_args(L, smem);
  a.x = x;
  a.predictor_run = (int*)(L->counts + CNT_NO_RUN);
  a.compact = L->fused_plan ? 0 : 1;
  a.active_idx = L->active_idx;
  a.n_active = L->n_tmp;
  return launch_stage(L, a, smem, kernel == LIF_KERNEL_PREDICT_Z, st);
}

cudaError_t launch_predict(lif_layer* L, const __half* x, float* logits, int32_t* active_idx,
                           int32_t* n_active, cudaStream_t st, cudaEvent_t* ev, int compact) {
  if (L->desc.gate_mode == LIF_GATE_RESIDENT)
    return launch_gate_predict(L, x, logits, active_idx, n_active, st, ev, compact);
  PredictSmem smem;
  PredictArgs a = predict_args(L, smem);
  a.x = x;
  a.logits = logits;
  a.compact = compact;
  // The input of these is there at once, so nothing of the predictor is on chip ahead of it.
  const bool late = compact || L->input_late;
  a.first_pass = compact || !L->behind_step;                           // (see stage 1)
  a.active_idx = (int*)active_idx;
  a.n_active = (int*)n_active;
  cudaError_t e;
  // Two launches where a z CTA needs so much shared memory that the score CTAs, which get as much, would
  // have an SM each (8 streams at 7168 x 256: 159 KB instead of 106).
  const bool one = (L->desc.n_streams == 1 || !late) && (smem.z <= smem.scores || smem.z <= kSharedSmem);
  if (!one) {
    e = launch_stage(L, a, smem, true, st);
    if (ev) tm_record(ev[1], st);
    if (e == cudaSuccess) e = launch_stage(L, a, smem, false, st);
  } else {
    if (ev) tm_record(ev[1], st);
    a.tickets = (unsigned long long*)(L->counts + CNT_PREDICTOR_TICKETS);
    e = launch_k2(predict_kernel_for(L->desc.n_streams), dim3(a.n_z + a.n_scores), dim3(kThreads),
                  smem.z > smem.scores ? smem.z : smem.scores, st, L->use_pdl, L->single_step, a);
  }
  if (ev) tm_record(ev[2], st);
  return e;
}

}  // namespace lif
