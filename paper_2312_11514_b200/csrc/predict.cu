// Low-rank sparsity predictor (Section 3.1, "Anticipating ReLU Sparsity"; Appendix B), one input
// stream (several: predict_multi.cu):
// scores = x.A.B + c, active iff score > theta, compacted to an ascending index list.
//
// Both stages are HBM-bound GEMVs over fp16 factors with fp32 accumulation:
//   stage 1  z_partial[p] = x[rows of p] . A[rows of p]      (A read once, 16-byte loads)
//   stage 2  score = (sum_p z_partial[p]) . B[:, tile] + c   (B read once, 16-byte loads)
// Stage 2 also thresholds (warp ballot -> bit mask) and the last CTA to finish turns the bit
// mask into the sorted list with a block prefix sum, so the list order never depends on
// scheduling.  Summation orders are fixed: results are bit-reproducible run to run.
#include "lif_internal.cuh"
#include "mask_compact.cuh"

namespace lif {
namespace {

// ---- stage 1: z_partial[cta][j] = sum_{m in rows(cta)} x[m] * A[m][j] -------------
__global__ void __launch_bounds__(kThreads)
predict_z_kernel(const __half* __restrict__ x, const __half* __restrict__ A, int d, int r,
                 int rows_per_cta, int staged, float* __restrict__ z_partial) {
  extern __shared__ __align__(16) uint4 staged_rows[];   // [staged][kThreads]
  __shared__ float red[2048];
  const int ncg = r >> 3;            // 8-column groups (16 bytes each)
  const int nrl = kThreads / ncg;    // row lanes
  const int tid = threadIdx.x;
  const int cg = tid % ncg, rl = tid / ncg;
  const int m0 = blockIdx.x * rows_per_cta;
  const int m1 = min(d, m0 + rows_per_cta);

  float acc[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) acc[e] = 0.f;

  // A is a weight: the thread's first 8 rows go into registers and the next `staged` into its own
  // slots of shared memory before the dependency wait, x (possibly written by the previous kernel)
  // comes only after it.  The kernel is resident long before its input is complete, so behind the
  // wait nothing of A is left to load (rows that were cost 2 us per launch at 4544 x 128).
  uint4 aq[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int m = m0 + rl + u * nrl;
    aq[u] = (rl < nrl && m < m1) ? ld_stream16(A + (size_t)m * r + cg * 8) : make_uint4(0, 0, 0, 0);
  }
  for (int u = 0; u < staged; ++u) {
    const int m = m0 + rl + (8 + u) * nrl;
    if (rl < nrl && m < m1) copy_async16(staged_rows + u * kThreads + tid, A + (size_t)m * r + cg * 8);
  }
  pdl_wait();
  pdl_trigger();
  if (rl < nrl) {
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int m = m0 + rl + u * nrl;
      if (m < m1) {
        float af[8];
        unpack8(aq[u], af);
        const float xs = __half2float(x[m]);
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[e] = fmaf(xs, af[e], acc[e]);
      }
    }
    own_copies_wait();
#pragma unroll 2
    for (int u = 0, m = m0 + rl + 8 * nrl; m < m1; ++u, m += nrl) {
      float af[8];
      unpack8(u < staged ? staged_rows[u * kThreads + tid] : ld_stream16(A + (size_t)m * r + cg * 8), af);
      const float xs = __half2float(x[m]);
#pragma unroll
      for (int e = 0; e < 8; ++e) acc[e] = fmaf(xs, af[e], acc[e]);
    }
  }
  // fold the row lanes (8 KB of shared memory)
  if (rl < nrl) {
#pragma unroll
    for (int e = 0; e < 8; ++e) red[rl * r + cg * 8 + e] = acc[e];
  }
  __syncthreads();
  for (int j = tid; j < r; j += kThreads) {
    float v = 0.f;
    for (int l = 0; l < nrl; ++l) v += red[l * r + j];
    z_partial[(size_t)blockIdx.x * r + j] = v;
  }
}

// ---- stage 2: scores, threshold, bit mask; last CTA compacts ------------------------------
// kSpec: also record per neuron the last token < keep in which it is active (speculative mode).
template <bool kSpec>
__global__ void __launch_bounds__(kThreads)
predict_logits_kernel(const float* __restrict__ z_partial, int P, const __half* __restrict__ B,
                      const float* __restrict__ c, float theta, int r, int F,
                      float* __restrict__ logits, uint32_t* mask_words, int* ticket,
                      int* __restrict__ active_idx, int* __restrict__ n_active, int compact,
                      int8_t* __restrict__ keep_tok, int keep, const int32_t* __restrict__ slot_of,
                      unsigned long long* new_mask_words, int* predictor_run, int staged) {
  extern __shared__ __align__(16) float zs[];   // [r], then the rows of B beyond the first 128
  __shared__ float red[16][kLogitTile];
  __shared__ int warp_sums[kThreads / 32];
  __shared__ int is_last;
  const int tid = threadIdx.x;

  // B does not depend on stage 1: put the first 128 rows of this CTA's tile in flight before
  // touching z (8 x 16 bytes per thread), then fold the stage-1 partials while they travel.
  const int cg = tid & 15, rs = tid >> 4;
  const int col = blockIdx.x * kLogitTile + cg * 8;
  uint4 bq[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int j = rs + 16 * u;
    bq[u] = (col < F && j < r) ? ld_stream16(B + (size_t)j * F + col) : make_uint4(0, 0, 0, 0);
  }
  // the next rows go into the thread's own slots of shared memory (see predict_z_kernel)
  uint4* staged_rows = reinterpret_cast<uint4*>(zs + r) + tid;
  for (int u = 0; u < staged; ++u) {
    const int j = rs + 16 * (8 + u);
    if (col < F && j < r) copy_async16(staged_rows + u * kThreads, B + (size_t)j * F + col);
  }
  const int my_col = blockIdx.x * kLogitTile + tid;   // used by threads < kLogitTile
  const float my_c = (tid < kLogitTile && my_col < F) ? c[my_col] : 0.f;
  // The window state was last written by this layer's previous step, complete long before this
  // kernel could start: whether the neuron already has a cache row is read here, so the mask of
  // neurons to bring in (active and not cached) costs no round trip of its own.
  const int my_row = (tid < kLogitTile && my_col < F) ? slot_of[my_col] : 0;
  // Released before this kernel's own wait: what follows (the window kernel or the single-launch
  // step) reads ahead of its wait only the window state, complete before stage 1 passed its own
  // wait and released this kernel, and entries that carry this run's number.  (A compacting run is
  // followed by a kernel that can do nothing before its list: no early release, 0.6 us a call.)
  if (!compact) pdl_trigger();
  pdl_wait();
  if (compact) pdl_trigger();
  const int run = tid < kLogitTile ? __ldcg(predictor_run) : 0;
  // every partial of a sum is requested before the first is used (one memory round trip instead of
  // several); the additions keep their order
  for (int i = tid; i < r; i += kThreads) {
    float t[kMaxZPartials];
#pragma unroll
    for (int p = 0; p < kMaxZPartials; ++p)
      t[p] = p < P ? __ldcg(z_partial + (size_t)p * r + i) : 0.f;
    float v = 0.f;
#pragma unroll
    for (int p = 0; p < kMaxZPartials; ++p)
      if (p < P) v += t[p];
    zs[i] = v;
  }
  __syncthreads();

  float acc[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) acc[e] = 0.f;
  for (int j0 = 0; j0 < r; j0 += 128) {
    if (j0 > 0) {
      if (j0 == 128) own_copies_wait();
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int j = j0 + rs + 16 * u, at = (j0 >> 4) - 8 + u;
        bq[u] = make_uint4(0, 0, 0, 0);
        if (col < F && j < r)
          bq[u] = at < staged ? staged_rows[at * kThreads] : ld_stream16(B + (size_t)j * F + col);
      }
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int j = j0 + rs + 16 * u;
      if (j < r) {
        float bf[8];
        unpack8(bq[u], bf);
        const float zz = zs[j];
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[e] = fmaf(zz, bf[e], acc[e]);
      }
    }
  }

#pragma unroll
  for (int e = 0; e < 8; ++e) red[rs][cg * 8 + e] = acc[e];
  __syncthreads();
  bool active = false;
  if (tid < kLogitTile && my_col < F) {
    float v = 0.f;
#pragma unroll
    for (int k = 0; k < 16; ++k) v += red[k][tid];
    v += my_c;
    if (logits) logits[my_col] = v;
    active = v > theta;
    if (kSpec) keep_tok[my_col] = (int8_t)(active && keep > 0 ? 0 : -1);
  }
  if (tid < kLogitTile) {
    const unsigned m = __ballot_sync(0xffffffffu, active);
    const unsigned mn = __ballot_sync(0xffffffffu, active && my_row < 0);
    if ((tid & 31) == 0) {
      mask_words[blockIdx.x * (kLogitTile / 32) + (tid >> 5)] = m;
      // the bits together with this run's number, in one store: a fetch kernel that is already
      // resident re-reads the entry until the number is the run's
      store_with_run(new_mask_words + blockIdx.x * (kLogitTile / 32) + (tid >> 5), mn, run);
      if (!compact)       // and the active ones themselves, for the single-launch step
        store_with_run(new_mask_words + (gridDim.x + blockIdx.x) * (kLogitTile / 32) + (tid >> 5), m, run);
    }
    if (!compact && active && my_row >= 0)                 // ... with the row of each that has one
      store_with_run(new_mask_words + 2 * gridDim.x * (kLogitTile / 32) + my_col, (uint32_t)my_row, run);
  }

  if (!compact) return;     // the consumer reads the bit mask itself
  compact_mask_last_cta(mask_words, gridDim.x * (kLogitTile / 32), ticket, active_idx, n_active,
                        warp_sums, &is_last);
  // every CTA has read this run's number: the next run gets one of its own (in a decode step
  // that reads the mask itself, the kernel that ends the step does this)
  if (is_last && tid == 0) advance_run(predictor_run, run);
}

// Rows per thread that are staged in shared memory, at most 48 KB of them per CTA.
constexpr int kMaxStaged = 12;
int z_staged_rows(const lif_layer_desc& D) {
  const int lanes = kThreads / (D.rank / 8) > 0 ? kThreads / (D.rank / 8) : 1;
  const int rows = (z_rows_per_cta(D.d_model) + lanes - 1) / lanes - 8;
  return rows < 0 ? 0 : (rows > kMaxStaged ? kMaxStaged : rows);
}
int logit_staged_rows(const lif_layer_desc& D) {
  const int rows = (D.rank + 15) / 16 - 8;
  return rows < 0 ? 0 : (rows > kMaxStaged ? kMaxStaged : rows);
}

cudaError_t launch_predict_single(lif_layer* L, const __half* x, float* logits, int32_t* active_idx,
                             int32_t* n_active, cudaStream_t st, cudaEvent_t* ev, int compact) {
  const lif_layer_desc& D = L->desc;
  const int z_staged = z_staged_rows(D);
  cudaError_t e = launch_k2(predict_z_kernel, dim3(L->z_ctas), dim3(kThreads),
                           (size_t)z_staged * kThreads * 16, st, L->use_pdl, L->single_step,
                           x, (const __half*)D.dev_pred_A, D.d_model, D.rank,
                           z_rows_per_cta(D.d_model), z_staged, L->z_partial);
  if (e != cudaSuccess) return e;
  if (ev) tm_record(ev[1], st);
  const int grid = (D.d_ff + kLogitTile - 1) / kLogitTile;
  const int staged = logit_staged_rows(D);
  const size_t smem = (size_t)D.rank * sizeof(float) + (size_t)staged * kThreads * 16;
  auto kernel = L->keep_tok ? predict_logits_kernel<true> : predict_logits_kernel<false>;
  e = launch_k2(kernel, dim3(grid), dim3(kThreads), smem, st, L->use_pdl, L->single_step,
               (const float*)L->z_partial, L->z_ctas, (const __half*)D.dev_pred_B, D.dev_pred_c,
               D.threshold_logit, D.rank, D.d_ff, logits, L->mask_words,
               (int*)(L->counts + CNT_TICKET_PREDICT), (int*)active_idx, (int*)n_active, compact,
               L->keep_tok, D.spec_keep, (const int32_t*)L->slot_of, L->new_mask_words,
               (int*)(L->counts + CNT_PREDICTOR_RUN), staged);
  if (ev) tm_record(ev[2], st);
  return e;
}

}  // namespace

// Opt-ins of the kernels (once per layer).
cudaError_t predict_configure(const lif_layer* L) {
  if (L->desc.n_streams > 1) return predict_multi_configure(L);
  const void* kernels[3] = {(const void*)predict_z_kernel, (const void*)predict_logits_kernel<false>,
                            (const void*)predict_logits_kernel<true>};
  for (const void* k : kernels) {
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         kMaxStaged * kThreads * 16 +
                                             (k == kernels[0] ? 0 : kMaxRank * (int)sizeof(float)));
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_predict_one(lif_layer* L, int kernel, const __half* x, cudaStream_t st) {
  const lif_layer_desc& D = L->desc;
  if (D.n_streams != 1) return cudaErrorInvalidValue;
  if (D.gate_mode == LIF_GATE_RESIDENT)
    return kernel == LIF_KERNEL_PREDICT_SCORES
               ? launch_gate_predict(L, x, nullptr, L->active_idx, L->n_tmp, st, nullptr,
                                     L->fused_plan ? 0 : 1, false)
               : cudaErrorInvalidValue;
  if (kernel == LIF_KERNEL_PREDICT_Z)
    return launch_k(predict_z_kernel, dim3(L->z_ctas), dim3(kThreads),
                    (size_t)z_staged_rows(D) * kThreads * 16, st, L->use_pdl, x,
                    (const __half*)D.dev_pred_A, D.d_model, D.rank, z_rows_per_cta(D.d_model),
                    z_staged_rows(D), L->z_partial);
  const int grid = (D.d_ff + kLogitTile - 1) / kLogitTile;
  return launch_k(L->keep_tok ? predict_logits_kernel<true> : predict_logits_kernel<false>,
                  dim3(grid), dim3(kThreads),
                  (size_t)D.rank * sizeof(float) + (size_t)logit_staged_rows(D) * kThreads * 16, st, L->use_pdl, (const float*)L->z_partial,
                  L->z_ctas, (const __half*)D.dev_pred_B, D.dev_pred_c, D.threshold_logit, D.rank,
                  D.d_ff, (float*)nullptr, L->mask_words, (int*)(L->counts + CNT_TICKET_PREDICT),
                  (int*)L->active_idx, (int*)L->n_tmp, L->fused_plan ? 0 : 1, L->keep_tok,
                  D.spec_keep, (const int32_t*)L->slot_of, L->new_mask_words,
                  (int*)(L->counts + CNT_NO_RUN), logit_staged_rows(D));
}

cudaError_t launch_predict(lif_layer* L, const __half* x, float* logits, int32_t* active_idx,
                           int32_t* n_active, cudaStream_t st, cudaEvent_t* ev, int compact) {
  if (L->desc.gate_mode == LIF_GATE_RESIDENT)
    return launch_gate_predict(L, x, logits, active_idx, n_active, st, ev, compact);
  return L->desc.n_streams == 1
             ? launch_predict_single(L, x, logits, active_idx, n_active, st, ev, compact)
             : launch_predict_multi(L, x, logits, active_idx, n_active, st, ev, compact);
}

}  // namespace lif
