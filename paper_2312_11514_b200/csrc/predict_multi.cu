// Low-rank predictor for several input streams (see predict.cu for one): the same two contractions
//   z = x.A (fp32 from fp16 factors),  scores = z.B + c,
// with the same order of additions as ever (stage 1: rows of one of P parts in `lanes` interleaved
// runs, the runs added in order, then the parts in order; stage 2: rows of B in 16 interleaved
// runs), so the decisions do not depend on which kernel computed them.
//
// Bound: latency.  Eight streams over 7168 x 256 x 28672 read 18 MB of factors (3 us at the copy peak)
// that are weights and can be on chip before the input is complete; behind the dependency wait there
// is x, 0.5 GFMA on fp32 and the exchange of z.  What used to cost was around that: x read one value
// at a time from global memory, and every stage-2 CTA adding up all parts of all sums again (58 MB of
// L2 reads at that shape).
#include "lif_internal.cuh"
#include "mask_compact.cuh"

namespace lif {
namespace {

// streams side by side in shared memory: 2, 4 or 8
__host__ __device__ constexpr int padded(int S) { return S <= 2 ? 2 : (S <= 4 ? 4 : 8); }
template <int SP>
struct __align__(2 * SP > 16 ? 16 : 2 * SP) Row {
  __half h[SP];
};

// ---- stage 1, ranks from 128: a CTA computes 8 columns of H streams completely ---------------------
// Thread (part, lane) adds the rows part * rows + lane + u * lanes, u = 0, 1, ...; its pieces of A
// travel into its own slots of shared memory ahead of the dependency wait.  x comes into shared
// memory transposed (a row's values of the H streams side by side, one load per row).  The lanes
// and then the parts are added in shared memory: z leaves the kernel finished.  The streams are split
// over as many CTAs as the SMs take, because what is behind the wait (x, the conversions from fp16,
// which run at 61 a clock and SM, and the additions) divides by them; A is read again from L2.
template <int H>
__global__ void __launch_bounds__(512)
z_columns_kernel(const __half* __restrict__ x, const __half* __restrict__ A, int S, int d, int r,
                 int parts, int rows_per_part, int lanes, int x_offset, float* __restrict__ z) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int tid = threadIdx.x, T = blockDim.x, cg = blockIdx.x, s0 = blockIdx.y * H;
  const int per = (rows_per_part + lanes - 1) / lanes;       // rows per thread
  uint4* a_s = reinterpret_cast<uint4*>(smem);               // [per][T]
  __half* x_s = reinterpret_cast<__half*>(smem + x_offset);  // [d][H]
  const int part = tid / lanes, lane = tid % lanes;
  const int m0 = part * rows_per_part + lane;
  const int m1 = part < parts ? min(d, (part + 1) * rows_per_part) : 0;
  for (int u = 0; u < per; ++u) {
    const int m = m0 + u * lanes;
    if (m < m1) copy_async16(a_s + u * T + tid, A + (size_t)m * r + cg * 8);
  }
  pdl_wait();
  pdl_trigger();
#pragma unroll 2
  for (int i = tid; i < (d >> 3); i += T) {                  // 8 rows of every stream of the CTA
    union { uint4 q; __half h[8]; } v[H];
#pragma unroll
    for (int s = 0; s < H; ++s)
      v[s].q = s0 + s < S ? reinterpret_cast<const uint4*>(x + (size_t)(s0 + s) * d)[i] : make_uint4(0, 0, 0, 0);
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      Row<H> w;
#pragma unroll
      for (int s = 0; s < H; ++s) w.h[s] = v[s].h[e];
      reinterpret_cast<Row<H>*>(x_s)[8 * i + e] = w;
    }
  }
  own_copies_wait();
  __syncthreads();
  float2 acc[H][4];
#pragma unroll
  for (int s = 0; s < H; ++s)
#pragma unroll
    for (int e = 0; e < 4; ++e) acc[s][e] = make_float2(0.f, 0.f);
#pragma unroll 4
  for (int u = 0; u < per; ++u) {
    const int m = m0 + u * lanes;
    if (m < m1) {
      float2 af[4];
      unpack8(a_s[u * T + tid], af);
      const Row<H> w = reinterpret_cast<const Row<H>*>(x_s)[m];
#pragma unroll
      for (int s = 0; s < H; ++s) {
        const float xv = __half2float(w.h[s]);
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[s][e] = fma2(make_float2(xv, xv), af[e], acc[s][e]);
      }
    }
  }
  __syncthreads();                                           // A and x are no longer needed
  constexpr int Q = H * 8;
  float* red = reinterpret_cast<float*>(smem);               // [T][Q]
  float* part_z = red + (size_t)T * Q;                       // [parts][Q]
#pragma unroll
  for (int s = 0; s < H; ++s) {
    float4* dst = reinterpret_cast<float4*>(red + (size_t)tid * Q + s * 8);
    dst[0] = make_float4(acc[s][0].x, acc[s][0].y, acc[s][1].x, acc[s][1].y);
    dst[1] = make_float4(acc[s][2].x, acc[s][2].y, acc[s][3].x, acc[s][3].y);
  }
  __syncthreads();
  for (int i = tid; i < parts * Q; i += T) {
    const int p = i / Q, q = i % Q;
    float v = 0.f;
#pragma unroll 8
    for (int l = 0; l < lanes; ++l) v += red[(size_t)(p * lanes + l) * Q + q];
    part_z[i] = v;
  }
  __syncthreads();
  for (int q = tid; q < Q; q += T) {
    float v = 0.f;
#pragma unroll 8
    for (int p = 0; p < parts; ++p) v += part_z[p * Q + q];
    if (s0 + q / 8 < S) z[(size_t)(s0 + q / 8) * r + cg * 8 + q % 8] = v;
  }
}

// ---- stage 1, smaller ranks: one CTA per part, as for one stream (z_partial[part][s][j]) --------------
template <int S>
__global__ void __launch_bounds__(kThreads)
z_parts_kernel(const __half* __restrict__ x, const __half* __restrict__ A, int d, int r,
               int rows_per_part, float* __restrict__ z_partial) {
  constexpr int SP = padded(S);
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ float red[2048];
  const int ncg = r >> 3, lanes = kThreads / ncg;
  const int tid = threadIdx.x, cg = tid % ncg, lane = tid / ncg;
  const int m0 = blockIdx.x * rows_per_part, m1 = min(d, m0 + rows_per_part);
  const int per = (rows_per_part + lanes - 1) / lanes;
  uint4* a_s = reinterpret_cast<uint4*>(smem);               // [per][kThreads]
  float* x_s = reinterpret_cast<float*>(a_s + per * kThreads);   // [rows_per_part][SP]
  for (int u = 0; u < per; ++u) {
    const int m = m0 + lane + u * lanes;
    if (lane < lanes && m < m1) copy_async16(a_s + u * kThreads + tid, A + (size_t)m * r + cg * 8);
  }
  pdl_wait();
  pdl_trigger();
  const int rows = m1 - m0;
#pragma unroll 4
  for (int i = tid; i < S * rows; i += kThreads) {
    const int s = i / rows, m = i - s * rows;
    x_s[m * SP + s] = __half2float(x[(size_t)s * d + m0 + m]);
  }
  own_copies_wait();
  __syncthreads();
  float acc[S][8];
#pragma unroll
  for (int s = 0; s < S; ++s)
#pragma unroll
    for (int e = 0; e < 8; ++e) acc[s][e] = 0.f;
  if (lane < lanes)
    for (int u = 0; u < per; ++u) {
      const int m = m0 + lane + u * lanes;
      if (m < m1) {
        float af[8];
        unpack8(a_s[u * kThreads + tid], af);
#pragma unroll
        for (int s = 0; s < S; ++s) {
          const float xv = x_s[(m - m0) * SP + s];
#pragma unroll
          for (int e = 0; e < 8; ++e) acc[s][e] = fmaf(xv, af[e], acc[s][e]);
        }
      }
    }
#pragma unroll
  for (int s = 0; s < S; ++s) {
    if (lane < lanes) {
#pragma unroll
      for (int e = 0; e < 8; ++e) red[lane * r + cg * 8 + e] = acc[s][e];
    }
    __syncthreads();
    for (int j = tid; j < r; j += kThreads) {
      float v = 0.f;
#pragma unroll 8
      for (int l = 0; l < lanes; ++l) v += red[l * r + j];
      z_partial[((size_t)blockIdx.x * S + s) * r + j] = v;
    }
    __syncthreads();
  }
}

// ---- stage 2: scores, threshold, bit mask; optionally the last CTA compacts --------------------------
// The first 128 rows of the CTA's tile of B are put in flight into registers and the next ones into
// shared memory before the wait.  All streams' partial scores of the tile go through shared memory at
// once (one barrier instead of two per stream).
template <int S>
__global__ void __launch_bounds__(kThreads)
scores_multi_kernel(const float* __restrict__ z_partial, int P, const __half* __restrict__ B,
                    const float* __restrict__ c, float theta, int r, int F,
                    float* __restrict__ logits, uint32_t* mask_words, int* ticket,
                    int* __restrict__ active_idx, int* __restrict__ n_active, int compact,
                    int8_t* __restrict__ keep_tok, int keep, const int32_t* __restrict__ slot_of,
                    unsigned long long* new_mask_words, int* predictor_run, int staged) {
  constexpr int SP = padded(S);
  extern __shared__ __align__(16) float zs[];                // [r][SP]
  uint4* b_s = reinterpret_cast<uint4*>(zs + SP * r);        // [staged][kThreads]
  float* red = reinterpret_cast<float*>(b_s + staged * kThreads);   // [S][16][kLogitTile]
  __shared__ uint32_t act_w[S][kLogitTile / 32];
  __shared__ int warp_sums[kThreads / 32];
  __shared__ int is_last;
  const int tid = threadIdx.x;
  const int cg = tid & 15, rs = tid >> 4;
  const int col = blockIdx.x * kLogitTile + cg * 8;
  uint4 bq[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int j = rs + 16 * u;
    bq[u] = (col < F && j < r) ? ld_stream16(B + (size_t)j * F + col) : make_uint4(0, 0, 0, 0);
  }
  for (int u = 0; u < staged; ++u) {
    const int j = rs + 16 * (8 + u);
    if (col < F && j < r) copy_async16(b_s + u * kThreads + tid, B + (size_t)j * F + col);
  }
  const int n = tid & (kLogitTile - 1), my_col = blockIdx.x * kLogitTile + n;
  const float my_c = my_col < F ? c[my_col] : 0.f;
  const int my_row = my_col < F ? slot_of[my_col] : 0;
  // released before this kernel's own wait, unless it compacts: see predict_logits_kernel
  if (!compact) pdl_trigger();
  pdl_wait();
  if (compact) pdl_trigger();
  const int run = tid < kLogitTile ? __ldcg(predictor_run) : 0;
  if (P == 1) {                                              // z is finished: all loads in flight
    for (int j = tid; j < r; j += kThreads) {
      float v[S];
#pragma unroll
      for (int s = 0; s < S; ++s) v[s] = __ldcg(z_partial + s * r + j);
#pragma unroll
      for (int s = 0; s < S; ++s) zs[j * SP + s] = v[s];
    }
  } else {                                                   // all parts of a sum in flight together
    for (int i = tid; i < S * r; i += kThreads) {
      float t[kMaxZPartials];
#pragma unroll
      for (int p = 0; p < kMaxZPartials; ++p)
        t[p] = p < P ? __ldcg(z_partial + (size_t)p * S * r + i) : 0.f;
      float v = 0.f;
#pragma unroll
      for (int p = 0; p < kMaxZPartials; ++p)
        if (p < P) v += t[p];
      const int s = i / r;
      zs[(i - s * r) * SP + s] = v;
    }
  }
  own_copies_wait();
  __syncthreads();

  float2 acc[S][4];
#pragma unroll
  for (int s = 0; s < S; ++s)
#pragma unroll
    for (int e = 0; e < 4; ++e) acc[s][e] = make_float2(0.f, 0.f);
  for (int j0 = 0; j0 < r; j0 += 128) {
    if (j0 > 0) {
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int j = j0 + rs + 16 * u, at = (j0 >> 4) - 8 + u;
        bq[u] = make_uint4(0, 0, 0, 0);
        if (col < F && j < r)
          bq[u] = at < staged ? b_s[at * kThreads + tid] : ld_stream16(B + (size_t)j * F + col);
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
#pragma unroll
  for (int s0 = 0; s0 < S; s0 += 2) {
    const int s = s0 + (tid >> 7);
    if (s < S) {
      float v = 0.f;
#pragma unroll
      for (int k = 0; k < 16; ++k) v += red[(s * 16 + k) * kLogitTile + n];
      v += my_c;
      if (logits && my_col < F) logits[(size_t)s * F + my_col] = v;
      const unsigned w = __ballot_sync(0xffffffffu, my_col < F && v > theta);
      if ((tid & 31) == 0) act_w[s][n >> 5] = w;
    }
  }
  __syncthreads();
  if (tid < kLogitTile) {
    unsigned m = 0;
    int last_kept = -1;        // speculative mode: last token < keep in which the neuron is active
#pragma unroll
    for (int s = 0; s < S; ++s) {
      const unsigned w = act_w[s][tid >> 5];
      m |= w;
      if (s < keep && ((w >> (tid & 31)) & 1u)) last_kept = s;
    }
    if (keep_tok && my_col < F) keep_tok[my_col] = (int8_t)last_kept;
    const unsigned mn = __ballot_sync(0xffffffffu, ((m >> (tid & 31)) & 1u) && my_row < 0);
    if ((tid & 31) == 0) {
      mask_words[blockIdx.x * (kLogitTile / 32) + (tid >> 5)] = m;
      // entries of the neurons to bring in and of the active ones, each with this run's number
      unsigned long long* at = new_mask_words + blockIdx.x * (kLogitTile / 32) + (tid >> 5);
      store_with_run(at, mn, run);
      store_with_run(at + gridDim.x * (kLogitTile / 32), m, run);
    }
    if (!compact && ((m >> (tid & 31)) & 1u) && my_row >= 0)
      store_with_run(new_mask_words + 2 * gridDim.x * (kLogitTile / 32) + my_col, (uint32_t)my_row, run);
  }
  if (!compact) return;     // the consumer reads the bit mask itself
  compact_mask_last_cta(mask_words, gridDim.x * (kLogitTile / 32), ticket, active_idx, n_active,
                        warp_sums, &is_last);
  if (is_last && tid == 0) advance_run(predictor_run, run);  // see predict_logits_kernel
}

constexpr int kMaxStagedRows = 12;     // of B per thread: 48 KB
constexpr int kColumnCtas = 128;       // of the first stage at most (one per SM, some left for what runs)

struct MultiShape {
  int columns;                         // stage 1 by column groups
  int parts, rows, lanes, threads, h, x_offset, staged;
  size_t z_smem, score_smem;
};
MultiShape multi_shape(const lif_layer_desc& D, int max_smem) {
  MultiShape m;
  const int S = D.n_streams, d = D.d_model, r = D.rank;
  m.parts = z_cta_count(d);
  m.rows = z_rows_per_cta(d);
  m.lanes = kThreads / (r / 8);
  const int per = (m.rows + m.lanes - 1) / m.lanes;
  m.threads = (m.parts * m.lanes + 31) / 32 * 32;
  const size_t a = (size_t)per * m.threads * 16;
  m.h = 1;                                                   // streams per CTA: 1, 2, 4 or 8
  while ((r / 8) * ((S + m.h - 1) / m.h) > kColumnCtas && m.h < 8) m.h *= 2;
  const size_t red = (size_t)(m.threads + m.parts) * m.h * 8 * 4;
  m.x_offset = (int)a;
  m.z_smem = a + (size_t)d * m.h * 2;
  if (red > m.z_smem) m.z_smem = red;
  // Below rank 128 a column group has more than 16 lanes per part, whose sums no longer fit one CTA,
  // and the parts of all sums together are few enough to be added by every stage-2 CTA.
  m.columns = r >= 128 && m.threads <= 512 && m.z_smem <= (size_t)max_smem;
  if (!m.columns) m.z_smem = (size_t)per * kThreads * 16 + (size_t)m.rows * 8 * 4;
  m.staged = (r + 15) / 16 - 8;
  m.staged = m.staged < 0 ? 0 : (m.staged > kMaxStagedRows ? kMaxStagedRows : m.staged);
  m.score_smem = (size_t)padded(S) * r * 4 + (size_t)m.staged * kThreads * 16 + (size_t)S * 16 * kLogitTile * 4;
  return m;
}

template <int S>
cudaError_t launch_s(lif_layer* L, const __half* x, float* logits, int32_t* active_idx,
                     int32_t* n_active, cudaStream_t st, cudaEvent_t* ev, int compact) {
  const lif_layer_desc& D = L->desc;
  const MultiShape m = multi_shape(D, L->max_smem);
  cudaError_t e;
  if (m.columns)
    e = launch_k(m.h == 1 ? z_columns_kernel<1> : m.h == 2 ? z_columns_kernel<2>
                 : m.h == 4 ? z_columns_kernel<4> : z_columns_kernel<8>,
                 dim3(D.rank / 8, (S + m.h - 1) / m.h), dim3(m.threads), m.z_smem, st, L->use_pdl, x,
                 (const __half*)D.dev_pred_A, S, D.d_model, D.rank, m.parts, m.rows, m.lanes,
                 m.x_offset, L->z_partial);
  else
    e = launch_k(z_parts_kernel<S>, dim3(m.parts), dim3(kThreads), m.z_smem, st, L->use_pdl, x,
                 (const __half*)D.dev_pred_A, D.d_model, D.rank, m.rows, L->z_partial);
  if (e != cudaSuccess) return e;
  if (ev) tm_record(ev[1], st);
  e = launch_k(scores_multi_kernel<S>, dim3((D.d_ff + kLogitTile - 1) / kLogitTile), dim3(kThreads),
               m.score_smem, st, L->use_pdl, (const float*)L->z_partial, m.columns ? 1 : m.parts,
               (const __half*)D.dev_pred_B, D.dev_pred_c, D.threshold_logit, D.rank, D.d_ff, logits,
               L->mask_words, (int*)(L->counts + CNT_TICKET_PREDICT), (int*)active_idx, (int*)n_active,
               compact, L->keep_tok, D.spec_keep, (const int32_t*)L->slot_of, L->new_mask_words,
               (int*)(L->counts + CNT_PREDICTOR_RUN), m.staged);
  if (ev) tm_record(ev[2], st);
  return e;
}

template <int S>
cudaError_t configure_s(const lif_layer* L) {
  const void* kernels[6] = {(const void*)z_columns_kernel<1>, (const void*)z_columns_kernel<2>,
                            (const void*)z_columns_kernel<4>, (const void*)z_columns_kernel<8>,
                            (const void*)z_parts_kernel<S>, (const void*)scores_multi_kernel<S>};
  for (const void* k : kernels) {
    cudaFuncAttributes at;
    cudaError_t e = cudaFuncGetAttributes(&at, k);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               L->max_smem - (int)at.sharedSizeBytes);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace

cudaError_t predict_multi_configure(const lif_layer* L) {
  switch (L->desc.n_streams) {
    case 2: return configure_s<2>(L);
    case 3: return configure_s<3>(L);
    case 4: return configure_s<4>(L);
    case 5: return configure_s<5>(L);
    case 6: return configure_s<6>(L);
    case 7: return configure_s<7>(L);
    case 8: return configure_s<8>(L);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_predict_multi(lif_layer* L, const __half* x, float* logits, int32_t* active_idx,
                                 int32_t* n_active, cudaStream_t st, cudaEvent_t* ev, int compact) {
  switch (L->desc.n_streams) {
    case 2: return launch_s<2>(L, x, logits, active_idx, n_active, st, ev, compact);
    case 3: return launch_s<3>(L, x, logits, active_idx, n_active, st, ev, compact);
    case 4: return launch_s<4>(L, x, logits, active_idx, n_active, st, ev, compact);
    case 5: return launch_s<5>(L, x, logits, active_idx, n_active, st, ev, compact);
    case 6: return launch_s<6>(L, x, logits, active_idx, n_active, st, ev, compact);
    case 7: return launch_s<7>(L, x, logits, active_idx, n_active, st, ev, compact);
    case 8: return launch_s<8>(L, x, logits, active_idx, n_active, st, ev, compact);
  }
  return cudaErrorInvalidValue;
}

}  // namespace lif
