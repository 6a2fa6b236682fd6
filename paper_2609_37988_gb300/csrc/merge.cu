// merge.cu -- split-K merge of decode partials.
//
// Partial rows hold [acc (dim) | m | l] with acc = sum_t 2^(x_t - m) v_t and
// l = sum_t 2^(x_t - m) over one split's positions.  The merged row is
//   out = sum_s 2^(m_s - M) acc_s / sum_s 2^(m_s - M) l_s,   M = max_s m_s,
// the log-sum-exp identity that makes softmax attention decomposable over a
// partition of the context.
#include <math.h>

#include "common.cuh"
#include "kernels.h"

namespace kvk {
namespace {

// P is written by the decode this launch overlaps (programmatic dependent
// launch), so it is read with coherent loads after the grid-dependency wait,
// not through the read-only path (no __restrict__).
// One thread per output element: every load of the row's partials (the S
// maxima, sums and this element's accumulators) is issued before any is
// used, so the merge costs one memory round trip.  Rows per CTA: 128 / dim
// (dim <= 128), else one row with a channel loop.
template <int SB, bool COUNTS>
__global__ void __launch_bounds__(128)
    splitk_merge_kernel(const float *P, int S, int n_rows, int dim,
                        float *__restrict__ out, const int32_t *counts, int rows_per, int first) {
  pdl_wait();
  pdl_trigger();
  const int width = dim >= 128 ? 128 : dim;  // threads per row
  const int rpc = 128 / width, r_in = (int)threadIdx.x / width;
  // with counts the grid's second axis is the sequence (a division here
  // would delay the count)
  int row = blockIdx.x * rpc + r_in;
  if (r_in >= rpc || row >= (COUNTS ? rows_per : n_rows)) return;
  if constexpr (COUNTS) row += blockIdx.y * rows_per;
  const int ch0 = (int)threadIdx.x % width;
  const size_t RS = (size_t)dim + 2;
  const size_t SS = (size_t)n_rows * RS;  // split stride
  const float *pr = P + (size_t)row * RS;
  constexpr int kMore = SB > 8 ? 16 : 8;
  // with per-sequence counts the first slots (as many as an even cut has,
  // at most SB) are loaded beside the count, the others, of a sequence that
  // has more, kMore at a time after it
  int n = S;
  if constexpr (COUNTS) n = counts[blockIdx.y];
  const int S0 = COUNTS ? first : S;
  float m[SB], l[SB];
#pragma unroll
  for (int s = 0; s < SB; ++s) {
    m[s] = s < S0 ? pr[s * SS + dim] : -INFINITY;
    l[s] = s < S0 ? pr[s * SS + dim + 1] : 0.f;
  }
  for (int ch = ch0; ch < dim; ch += 128) {
    float x[SB];
#pragma unroll
    for (int s = 0; s < SB; ++s) x[s] = s < S0 ? pr[s * SS + ch] : 0.f;
    if constexpr (COUNTS) {
#pragma unroll
      for (int s = 0; s < SB; ++s)
        if (s >= n) {
          m[s] = -INFINITY;
          x[s] = l[s] = 0.f;
        }
    }
    float M = -INFINITY;
#pragma unroll
    for (int s = 0; s < SB; ++s) M = fmaxf(M, m[s]);
    float L = 0.f, A = 0.f;
    if (M != -INFINITY) {
#pragma unroll
      for (int s = 0; s < SB; ++s) {
        const float w = m[s] == -INFINITY ? 0.f : exp2f(m[s] - M);
        L = fmaf(w, l[s], L);
        A = fmaf(w, x[s], A);
      }
    }
    if constexpr (COUNTS) {
      for (int s0 = S0; s0 < n; s0 += kMore) {
        float m2[kMore], l2[kMore], x2[kMore], M2 = M;
#pragma unroll
        for (int s = 0; s < kMore; ++s) {
          const bool in = s0 + s < n;
          m2[s] = in ? pr[(s0 + s) * SS + dim] : -INFINITY;
          l2[s] = in ? pr[(s0 + s) * SS + dim + 1] : 0.f;
          x2[s] = in ? pr[(s0 + s) * SS + ch] : 0.f;
        }
#pragma unroll
        for (int s = 0; s < kMore; ++s) M2 = fmaxf(M2, m2[s]);
        if (M2 == -INFINITY) continue;
        const float w0 = M == -INFINITY ? 0.f : exp2f(M - M2);
        L *= w0;
        A *= w0;
        M = M2;
#pragma unroll
        for (int s = 0; s < kMore; ++s) {
          const float w = m2[s] == -INFINITY ? 0.f : exp2f(m2[s] - M);
          L = fmaf(w, l2[s], L);
          A = fmaf(w, x2[s], A);
        }
      }
    }
    out[(size_t)row * dim + ch] = (L > 0.f) ? A / L : 0.f;
  }
}

// More than 16 splits (few units over a long context): one CTA per row, warp
// w takes splits w, w + 8, ..., lane L channels L + 32 j.  A thread issues
// the loads of its first 8 splits (maxima, sums, accumulators: every split up
// to 64) before it uses any, so this merge too is one memory round trip; the
// warps' maxima and then their sums meet in shared memory.  Bound by that
// latency: a serial loop over the splits (a dependent load and exponential
// each) took 32.1 us for 57 splits of 40 rows of 128; the whole decode step
// around it (one sequence of 32769 int8 positions) went 40.3 -> 33.4 us.
constexpr int kWideWarps = 8, kWideRound = 8;
template <bool COUNTS>
__global__ void __launch_bounds__(32 * kWideWarps)
    splitk_merge_wide(const float *P, int S, int n_rows, int dim, float *__restrict__ out,
                      const int32_t *counts, int rows_per, int first) {
  pdl_wait();
  pdl_trigger();
  __shared__ float s_m[kWideWarps], s_l[kWideWarps], s_a[kWideWarps][128];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row = blockIdx.x;
  const size_t RS = (size_t)dim + 2;
  const size_t SS = (size_t)n_rows * RS;
  const float *pr = P + (size_t)row * RS;
  float m[kWideRound], l[kWideRound], x[kWideRound][4];
  // this thread's first slots below `hi`, empty past it
  auto load_acc = [&](int ch0, int hi) {
#pragma unroll
    for (int i = 0; i < kWideRound; ++i) {
      const int s = warp + kWideWarps * i;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int ch = ch0 + lane + 32 * j;
        x[i][j] = s < hi && ch < dim ? pr[s * SS + ch] : 0.f;
      }
    }
  };
  const int S0 = COUNTS ? first : S;
#pragma unroll
  for (int i = 0; i < kWideRound; ++i) {
    const int s = warp + kWideWarps * i;
    m[i] = s < S0 ? pr[s * SS + dim] : -INFINITY;
    l[i] = s < S0 ? pr[s * SS + dim + 1] : 0.f;
  }
  load_acc(0, S0);
  // per-sequence counts: as in splitk_merge_kernel, the first slots beside
  // the count, the others of a sequence that has more after it
  int n = S;
  if constexpr (COUNTS) {
    n = counts[row / rows_per];
#pragma unroll
    for (int i = 0; i < kWideRound; ++i) {
      const int s = warp + kWideWarps * i;
      if (s >= n) {
        m[i] = -INFINITY;
        l[i] = x[i][0] = x[i][1] = x[i][2] = x[i][3] = 0.f;
      } else if (s >= S0) {
        m[i] = pr[s * SS + dim];
        l[i] = pr[s * SS + dim + 1];
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (lane + 32 * j < dim) x[i][j] = pr[s * SS + lane + 32 * j];
      }
    }
  }
  float M = -INFINITY;
#pragma unroll
  for (int i = 0; i < kWideRound; ++i) M = fmaxf(M, m[i]);
  for (int s = warp + kWideWarps * kWideRound; s < n; s += kWideWarps) M = fmaxf(M, pr[s * SS + dim]);
  if (lane == 0) s_m[warp] = M;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < kWideWarps; ++w) M = fmaxf(M, s_m[w]);
  for (int ch0 = 0; ch0 < dim; ch0 += 128) {
    if (ch0 > 0) load_acc(ch0, n);
    float L = 0.f, A[4] = {0.f, 0.f, 0.f, 0.f};
    if (M != -INFINITY) {
#pragma unroll
      for (int i = 0; i < kWideRound; ++i) {
        const float w = m[i] == -INFINITY ? 0.f : exp2f(m[i] - M);
        L = fmaf(w, l[i], L);
#pragma unroll
        for (int j = 0; j < 4; ++j) A[j] = fmaf(w, x[i][j], A[j]);
      }
      for (int s = warp + kWideWarps * kWideRound; s < n; s += kWideWarps) {
        const float ms = pr[s * SS + dim];
        const float w = ms == -INFINITY ? 0.f : exp2f(ms - M);
        L = fmaf(w, pr[s * SS + dim + 1], L);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int ch = ch0 + lane + 32 * j;
          if (ch < dim) A[j] = fmaf(w, pr[s * SS + ch], A[j]);
        }
      }
    }
    if (lane == 0) s_l[warp] = L;
#pragma unroll
    for (int j = 0; j < 4; ++j) s_a[warp][lane + 32 * j] = A[j];
    __syncthreads();
    const int ch = ch0 + (int)threadIdx.x;
    if (threadIdx.x < 128 && ch < dim) {
      float a = 0.f, ls = 0.f;
#pragma unroll
      for (int w = 0; w < kWideWarps; ++w) {
        a += s_a[w][threadIdx.x];
        ls += s_l[w];
      }
      out[(size_t)row * dim + ch] = ls > 0.f ? a / ls : 0.f;
    }
    __syncthreads();
  }
}

__global__ void rewind_kernel(const RewindArgs a) {
  pdl_wait();
  pdl_trigger();
  for (int i = threadIdx.x; i < a.n_anchors * a.B; i += blockDim.x) {
    int32_t *l = a.lens[i / a.B] + (i % a.B);
    *l = max(0, *l - a.n);
  }
}

}  // namespace

cudaError_t launch_rewind(const RewindArgs &a, cudaStream_t st) {
  return launch_pdl(rewind_kernel, dim3(1), dim3(256), 0, st, a);
}

cudaError_t launch_splitk_merge(const float *partials, int n_splits, int n_rows, int dim,
                                float *out, cudaStream_t st, const int32_t *counts, int rows_per, int first) {
  if (n_splits < 1 || n_rows < 0 || dim < 1) return cudaErrorInvalidValue;
  if (n_rows == 0) return cudaSuccess;
  const int rpc = dim >= 128 ? 1 : 128 / dim;
  const int at_once = counts ? first : n_splits;
  if (at_once > 16)
    return launch_pdl(counts ? splitk_merge_wide<true> : splitk_merge_wide<false>, n_rows, dim3(32 * kWideWarps), 0, st, partials, n_splits, n_rows, dim, out,
                      counts, rows_per, first);
  auto k = at_once <= 8 ? (counts ? splitk_merge_kernel<8, true> : splitk_merge_kernel<8, false>)
                        : (counts ? splitk_merge_kernel<16, true> : splitk_merge_kernel<16, false>);
  if (counts && n_rows % rows_per) return cudaErrorInvalidValue;
  const dim3 grid = counts ? dim3((rows_per + rpc - 1) / rpc, n_rows / rows_per) : dim3((n_rows + rpc - 1) / rpc);
  return launch_pdl(k, grid, dim3(128), 0, st, partials, n_splits, n_rows, dim, out, counts, rows_per, first);
}

}  // namespace kvk
