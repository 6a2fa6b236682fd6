// evict.cu -- window-vote eviction composed with a compressed GQA cache
// (Sec. 3.4: an evictor runs on the same cache and the reduction factors
// multiply; the evictors sum attention over an observation window of the
// last queries, Appendix "Eviction implementations").
//
// For sequence b, KV head j, the window queries w < n_win (at positions
// p_w = len - n_win + w, each seeing positions 0..p_w) of the G query heads
// of j vote for every position t before the window:
//     vote[t] = sum_{w, h} 2^(x_{w,h}(t) - M_{w,h}) / L_{w,h}
// with x = scale log2(e) <q_{w,h}, k_t> on the dequantised key and (M, L)
// the row's maximum and sum over its causal range.  The budget - n_win
// largest votes (ties: the smaller position) and the window become the
// anchor's kept list for (b, j), sorted.  Four launches: the rows' statistics,
// merged per row, the votes, the selection.
//
// head_dim 128 and at most 256 window rows score on the tensor cores, in bf16
// hi and lo halves, and the vote pass scores again (second half of this
// file).  Others score on the CUDA cores in fp32 and store the scores (R x 4
// bytes per position) for the vote pass, which costs less there than scoring
// twice (R x D products).  Votes are within ~1e-6 of the fp64 definition.
#include <math.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "kernels.h"
#include "layout.h"
#include "umma.cuh"
#include "window_tc.cuh"

namespace kvk {
namespace {

constexpr int kT = kEvictTile;  // positions per scoring tile

// Dequantised channel ch of the key of position t from its record (the
// scale word of the symmetric scheme passed in).
__device__ __forceinline__ float key_elem(const GqaView &v, const RecLayout &L, const uint8_t *rec,
                                          int t, uint32_t sc_word, int ch) {
  const int D = v.D;
  if (v.bits == 16) {
    int byte, hi;
    k_pos(ch, 16, D, &byte, &hi);
    return bf16_to_f32(*reinterpret_cast<const uint16_t *>(rec + byte));
  }
  if (v.scheme == kSchemeSym) {
    const int lb = sym_k_bit(ch, v.bits, D);
    const int u = (rec[sym_phys(lb >> 3, t, v.rec_bytes)] >> (lb & 7)) & ((1 << v.bits) - 1);
    const float s = __uint_as_float(sc_word << 16);
    return s * (float)(u - sym_levels(v.bits));
  }
  int byte, hi;
  k_pos(ch, v.bits, D, &byte, &hi);
  const int x = rec[byte];
  const int code = v.bits == 8 ? x : (hi ? x >> 4 : x & 15);
  const float2 m = reinterpret_cast<const float2 *>(rec + L.km_off)[ch / v.group];
  return fmaf((float)code, m.x, m.y);
}

// Scores of one 128-position tile against every window query row of its
// (sequence, KV head): X[r][t] = sig_log2 <q_r, k_t>, an fp32 contraction of
// [R x D] by [D x 128] on the CUDA cores, register-tiled: thread (tx, ty)
// holds rows ty*4 .. ty*4+3 of a 64-row chunk against positions tx*4 ..
// tx*4+3 and 64 + tx*4 .. 64 + tx*4+3 of the tile (32 products per pair of
// key loads and one query load).  The dequantised keys sit channel-major in
// shared memory [D][128], the chunk's query rows [D][64].  Each row's
// (max, sum 2^(x - max)) over the tile's positions in its causal range goes
// to the per-tile statistics, and the scores of the positions before the
// window go to the score buffer, which the vote pass streams instead of
// recomputing them.
constexpr int kRC = 64;        // window query rows per chunk
constexpr int kThreads = 256;  // 16 position groups x 16 row groups

template <int D>
constexpr int evict_smem() {
  return (D * kT + D * kRC) * 4;
}

template <int D>
__global__ void __launch_bounds__(kThreads, 2) evict_scores_kernel(const EvictArgs a) {
  pdl_wait();
  const GqaView &v = a.v;
  const int tile = blockIdx.x, j = blockIdx.y, b = blockIdx.z;
  const int tid = threadIdx.x;
  const int len = v.lens[b];
  const int t0 = tile * kT;
  if (len <= a.budget || t0 >= len) {  // the sequence keeps everything / tile past the end
    pdl_trigger();
    return;
  }
  const int P = len - a.n_win;
  const int unit = b * v.Hkv + j;
  const int R = a.n_win * a.G;
  extern __shared__ __align__(16) float evict_sm[];
  float *kt = evict_sm;          // [D][kT]
  float *qt = evict_sm + D * kT; // [D][kRC]
  const size_t slab = (size_t)b * v.Hkv + j;
  {
    // two threads per position, half of the channels each
    const int p = tid & (kT - 1), half = tid / kT;
    const int t = t0 + p;
    const bool live = t < len;
    const RecLayout L = rec_layout(v.bits, D, v.group, v.key_axis);
    const uint8_t *rec = v.rec + (slab * v.cap + (live ? t : t0)) * v.rec_bytes;
    const uint32_t sw = (live && v.scheme == kSchemeSym) ? v.scales[slab * v.cap + t] : 0u;
    for (int ch = half * (D / 2); ch < (half + 1) * (D / 2); ++ch)
      kt[ch * kT + p] = live ? key_elem(v, L, rec, t, sw, ch) : 0.f;
  }
  const int tx = tid & 15, ty = tid >> 4;
  float2 *stats = a.stats + (size_t)unit * R * a.n_tiles;
  float *scores = a.scores + (size_t)unit * R * a.sc_stride;
  for (int rc0 = 0; rc0 < R; rc0 += kRC) {
    __syncthreads();  // keys written; the previous chunk's query rows consumed
    // the chunk's query rows, channel-major (rows past R are zero)
    for (int e = tid; e < kRC * (D / 4); e += kThreads) {
      const int rr = e & (kRC - 1), c4 = e / kRC;
      const int r = rc0 + rr;
      float4 x4 = make_float4(0.f, 0.f, 0.f, 0.f);
      if (r < R) {
        const int w = r / a.G, h = j * a.G + r % a.G;
        const size_t qi = (((size_t)b * a.n_win + w) * a.Hq + h) * D + 4 * c4;
        if (a.q_f32) {
          x4 = *reinterpret_cast<const float4 *>(static_cast<const float *>(a.q) + qi);
        } else {
          const uint2 u = *reinterpret_cast<const uint2 *>(static_cast<const uint16_t *>(a.q) + qi);
          x4 = make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xFFFF0000u),
                           __uint_as_float(u.y << 16), __uint_as_float(u.y & 0xFFFF0000u));
        }
      }
      qt[(4 * c4 + 0) * kRC + rr] = x4.x;
      qt[(4 * c4 + 1) * kRC + rr] = x4.y;
      qt[(4 * c4 + 2) * kRC + rr] = x4.z;
      qt[(4 * c4 + 3) * kRC + rr] = x4.w;
    }
    __syncthreads();
    float acc[4][8];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int c = 0; c < 8; ++c) acc[i][c] = 0.f;
#pragma unroll 4
    for (int k = 0; k < D; ++k) {
      const float4 k0 = *reinterpret_cast<const float4 *>(kt + k * kT + tx * 4);
      const float4 k1 = *reinterpret_cast<const float4 *>(kt + k * kT + 64 + tx * 4);
      const float4 q4 = *reinterpret_cast<const float4 *>(qt + k * kRC + ty * 4);
      const float kk[8] = {k0.x, k0.y, k0.z, k0.w, k1.x, k1.y, k1.z, k1.w};
      const float qq[4] = {q4.x, q4.y, q4.z, q4.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int c = 0; c < 8; ++c) acc[i][c] = fmaf(qq[i], kk[c], acc[i][c]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = rc0 + ty * 4 + i;
      const int last = P + r / a.G;  // the last position row r sees
      float m = -INFINITY;
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const int t = t0 + (c >> 2) * 64 + tx * 4 + (c & 3);
        acc[i][c] *= a.sig_log2;
        if (t <= last) m = fmaxf(m, acc[i][c]);
      }
#pragma unroll
      for (int off = 8; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
      float l = 0.f;
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const int t = t0 + (c >> 2) * 64 + tx * 4 + (c & 3);
        if (t <= last) l += exp2f(acc[i][c] - m);  // m is finite: this row sees t
      }
#pragma unroll
      for (int off = 8; off > 0; off >>= 1) l += __shfl_xor_sync(0xffffffffu, l, off);
      if (r < R) {
        if (tx == 0) stats[(size_t)r * a.n_tiles + tile] = make_float2(m, l);
        float *row = scores + (size_t)r * a.sc_stride + t0 + tx * 4;
        if (t0 + tx * 4 < P) *reinterpret_cast<float4 *>(row) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
        if (t0 + 64 + tx * 4 < P)
          *reinterpret_cast<float4 *>(row + 64) = make_float4(acc[i][4], acc[i][5], acc[i][6], acc[i][7]);
      }
    }
  }
  pdl_trigger();
}

// Votes of 256 positions before the window: sum over the rows of
// 2^(x - M - log2 L) with the rows' merged statistics, streaming the scores.
constexpr int kVoteT = 256;
constexpr int kVoteRows = 1024;  // merged statistics staged per round

__global__ void __launch_bounds__(kVoteT) evict_votes_kernel(const EvictArgs a) {
  pdl_wait();
  const GqaView &v = a.v;
  const int j = blockIdx.y, b = blockIdx.z, tid = threadIdx.x;
  const int len = v.lens[b];
  const int P = len - a.n_win;
  const int t = blockIdx.x * kVoteT + tid;
  if (len <= a.budget || (int)blockIdx.x * kVoteT >= P) {
    pdl_trigger();
    return;
  }
  const int unit = b * v.Hkv + j;
  const int R = a.n_win * a.G;
  const float2 *fin = a.fin + (size_t)unit * R;
  const float *x = a.scores + (size_t)unit * R * a.sc_stride + t;
  __shared__ float norm[kVoteRows];
  float vote = 0.f;
  for (int r0 = 0; r0 < R; r0 += kVoteRows) {
    const int nr = min(kVoteRows, R - r0);
    __syncthreads();
    for (int i = tid; i < nr; i += kVoteT) {
      const float2 ml = fin[r0 + i];
      norm[i] = ml.x + log2f(ml.y);
    }
    __syncthreads();
    if (t < P) {
#pragma unroll 8
      for (int r = 0; r < nr; ++r) vote += exp2f(x[(size_t)(r0 + r) * a.sc_stride] - norm[r]);
    }
  }
  if (t < P) a.votes[(size_t)unit * v.cap + t] = vote;
  pdl_trigger();
}

// Merged (M, L) of every window query row over its tiles.
// One warp per (unit, row): lanes stride over the row's tile entries
// (coalesced), then warp reductions of the maximum and of the rescaled sums.
constexpr int kMergeWarps = 8;
__global__ void __launch_bounds__(32 * kMergeWarps) evict_merge_stats_kernel(const EvictArgs a) {
  pdl_wait();
  pdl_trigger();
  const GqaView &v = a.v;
  const int R = a.n_win * a.G;
  const int units = v.B * v.Hkv;
  const int id = blockIdx.x * kMergeWarps + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (id >= units * R) return;
  const int unit = id / R, r = id % R, b = unit / v.Hkv;
  const int len = v.lens[b];
  if (len <= a.budget) return;
  int nt = min((len + kT - 1) / kT, a.n_tiles);
  if (a.items_per_cta) {  // one entry set per CTA that walked tiles of the unit
    const int i0 = unit * a.n_tiles;
    nt = (i0 + nt - 1) / a.items_per_cta - i0 / a.items_per_cta + 1;
  }
  nt *= a.stat_sub;
  const float2 *st = a.stats + ((size_t)unit * R + r) * a.n_tiles * a.stat_sub;
  float M = -INFINITY;
  for (int i = lane; i < nt; i += 32) M = fmaxf(M, st[i].x);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, off));
  float L = 0.f;
  if (M != -INFINITY)
    for (int i = lane; i < nt; i += 32) {
      const float2 e = st[i];
      if (e.x != -INFINITY) L += e.y * exp2f(e.x - M);
    }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) L += __shfl_xor_sync(0xffffffffu, L, off);
  if (lane == 0) a.fin[id] = make_float2(M, L);
}

// Block-wide exclusive scan of one int per thread (1024 threads); returns the
// thread's exclusive prefix and writes the block total to *total.
__device__ __forceinline__ int block_scan_1024(int x, int *wsum, int *total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int inc = x;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, inc, off);
    if (lane >= off) inc += y;
  }
  if (lane == 31) wsum[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    int s = wsum[lane];
    int si = s;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, si, off);
      if (lane >= off) si += y;
    }
    wsum[lane] = si - s;  // exclusive prefix of the warp totals
    if (lane == 31) *total = si;
  }
  __syncthreads();
  const int r = wsum[warp] + inc - x;
  __syncthreads();  // wsum is reused by the next scan
  return r;
}

// keys t0 .. t0+7 (zero past n); t0 is a multiple of 8 and the array
// 32-byte aligned
__device__ __forceinline__ void load8(const uint32_t *key, int t0, int n, uint32_t (&kk)[8]) {
  if (t0 + 8 <= n) {
    const uint4 u0 = *reinterpret_cast<const uint4 *>(key + t0);
    const uint4 u1 = *reinterpret_cast<const uint4 *>(key + t0 + 4);
    kk[0] = u0.x; kk[1] = u0.y; kk[2] = u0.z; kk[3] = u0.w;
    kk[4] = u1.x; kk[5] = u1.y; kk[6] = u1.z; kk[7] = u1.w;
  } else {
#pragma unroll
    for (int u = 0; u < 8; ++u) kk[u] = t0 + u < n ? key[t0 + u] : 0u;
  }
}

// ---- thread-block clusters -------------------------------------------------
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// the int at the same shared-memory place of CTA `rank` of the cluster
__device__ __forceinline__ int cluster_ld(const int *p, uint32_t rank) {
  uint32_t a;
  int x;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
  asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(x) : "r"(a) : "memory");
  return x;
}

// Kept list of one (sequence, kv head): the budget - n_win largest votes by
// a radix select on their bit patterns (votes are >= 0, so the patterns
// order as the values), then the chosen positions in increasing order and
// the window.  PARTS = 8: a cluster of 8 CTAs per unit, each over an eighth
// of the positions: a unit's votes are read five times, which one CTA per
// unit did in 99 us for 32 units of 131072 positions with 120 SMs idle (65 us
// so).  Per pass the CTAs add each other's histograms through distributed
// shared memory and decide alike (one cluster barrier per pass: two
// histograms in turn).  The barriers cost more than a few rounds of one CTA:
// select_one_cta.
constexpr int kSelParts = 8;
template <int PARTS>
__global__ void __cluster_dims__(PARTS, 1, 1) __launch_bounds__(1024) evict_select_kernel(const EvictArgs a) {
  pdl_wait();
  pdl_trigger();
  const GqaView &v = a.v;
  const int j = blockIdx.x / PARTS, b = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int part = PARTS > 1 ? (int)cluster_rank() : 0;
  const int unit = b * v.Hkv + j;
  const int len = v.lens[b];
  int32_t *out = v.kept_idx + (size_t)unit * v.kept_cap;
  if (len <= a.budget) {  // everything is kept (the whole cluster leaves)
    for (int t = part * 1024 + tid; t < len; t += PARTS * 1024) out[t] = t;
    if (part == 0 && tid == 0) v.kept_n[unit] = len;
    return;
  }
  const int P = len - a.n_win, k = a.budget - a.n_win;
  const uint32_t *key = reinterpret_cast<const uint32_t *>(a.votes + (size_t)unit * v.cap);
  const int per = ((P + PARTS - 1) / PARTS + 7) / 8 * 8;
  const int p0 = min(P, part * per), p1 = min(P, p0 + per);  // this CTA's positions
  __shared__ int hist[2][256];
  __shared__ uint32_t s_prefix;
  __shared__ int s_rank;
  __shared__ int wsum[32];
  __shared__ int s_total;
  __shared__ int s_cnt[2];
  uint32_t prefix = 0, mask = 0;
  int rank = k;  // 1-based rank (from the top) of the wanted key among the matches
  if (k > 0) {
    for (int pass = 0; pass < 4; ++pass) {
      const int shift = 24 - 8 * pass;
      int *h = hist[pass & 1];
      if (tid < 256) h[tid] = 0;
      __syncthreads();
      // votes of similar size share their leading bytes, so most lanes of a
      // warp hit the bin of lane 0: those are counted with one atomic, the
      // others one by one.  Eight consecutive votes per thread per round
      // keep eight loads in flight.
      for (int c0 = p0; c0 < p1; c0 += 8 * 1024) {
        uint32_t kk[8];
        load8(key, c0 + 8 * tid, p1, kk);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const bool hit = c0 + 8 * tid + u < p1 && (kk[u] & mask) == prefix;
          const uint32_t bin = hit ? (kk[u] >> shift) & 255 : 256u;
          const uint32_t bin0 = __shfl_sync(0xffffffffu, bin, 0);
          const uint32_t same = __ballot_sync(0xffffffffu, bin == bin0);
          if (bin == bin0) {
            if (lane == 0 && bin0 < 256u) atomicAdd(&h[bin0], __popc(same));
          } else if (hit) {
            atomicAdd(&h[bin], 1);
          }
        }
      }
      if (PARTS > 1) cluster_sync();
      else __syncthreads();
      // bins from the top: the one in which the count reaches the rank
      int n = 0, inc = 0;
      if (tid < 256) {
        if (PARTS > 1) {
#pragma unroll
          for (uint32_t r = 0; r < PARTS; ++r) n += cluster_ld(&h[255 - tid], r);
        } else {
          n = h[255 - tid];
        }
        inc = n;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
          const int y = __shfl_up_sync(0xffffffffu, inc, off);
          if (lane >= off) inc += y;
        }
        if (lane == 31) wsum[warp] = inc;
      }
      __syncthreads();
      if (tid < 256) {
        for (int w = 0; w < warp; ++w) inc += wsum[w];
        if (inc >= rank && inc - n < rank) {
          s_prefix = prefix | ((uint32_t)(255 - tid) << shift);
          s_rank = rank - (inc - n);
        }
      }
      __syncthreads();
      prefix = s_prefix;
      rank = s_rank;
      mask |= 0xFFu << shift;
    }
  }
  // positions above the threshold key, and the first `rank` equal to it
  // (one scan of the packed counts: greater in the high half, equal in the
  // low half; a taken position's slot is the greater ones before it plus
  // the equal ones before it, at most `rank`); first the counts of the
  // positions before this CTA's
  const uint32_t theta = prefix;
  int gt_carry = 0, eq_carry = 0;
  if (PARTS > 1 && k > 0) {
    if (tid < 2) s_cnt[tid] = 0;
    __syncthreads();
    int ngt = 0, neq = 0;
    for (int c0 = p0; c0 < p1; c0 += 8 * 1024) {
      uint32_t kk[8];
      load8(key, c0 + 8 * tid, p1, kk);
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const bool in = c0 + 8 * tid + u < p1;
        ngt += in && kk[u] > theta;
        neq += in && kk[u] == theta;
      }
    }
    ngt = __reduce_add_sync(0xffffffffu, ngt);
    neq = __reduce_add_sync(0xffffffffu, neq);
    if (lane == 0) {
      if (ngt) atomicAdd(&s_cnt[0], ngt);
      if (neq) atomicAdd(&s_cnt[1], neq);
    }
    cluster_sync();
    for (int r = 0; r < part; ++r) {
      gt_carry += cluster_ld(&s_cnt[0], r);
      eq_carry += cluster_ld(&s_cnt[1], r);
    }
  }
  for (int c0 = p0; c0 < p1 && k > 0; c0 += 8 * 1024) {
    const int tb = c0 + 8 * tid;  // this thread's eight consecutive positions
    uint32_t kk[8];
    load8(key, tb, p1, kk);
    int ngt = 0, neq = 0;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      ngt += tb + u < p1 && kk[u] > theta;
      neq += tb + u < p1 && kk[u] == theta;
    }
    const int ex = block_scan_1024((ngt << 16) | neq, wsum, &s_total);
    const int tot = s_total;
    int gt_before = gt_carry + (ex >> 16), eq_before = eq_carry + (ex & 0xFFFF);
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const bool gt = tb + u < p1 && kk[u] > theta, eq = tb + u < p1 && kk[u] == theta;
      const int pos = gt_before + min(eq_before, rank);
      if ((gt || (eq && eq_before < rank)) && pos < k) out[pos] = tb + u;
      gt_before += gt;
      eq_before += eq;
    }
    gt_carry += tot >> 16;
    eq_carry += tot & 0xFFFF;
  }
  if (part == PARTS - 1)
    for (int i = tid; i < a.n_win; i += 1024) out[k + i] = P + i;
  if (part == 0 && tid == 0) v.kept_n[unit] = a.budget;
  if (PARTS > 1) cluster_sync();  // no CTA leaves while another may read its counts
}


// Whether one CTA per unit selects faster than a cluster of 8, by the host's
// bound on the lengths (a longer sequence in a recorded launch only takes
// longer).  Measured (us, one CTA / cluster): 8 units of 4096 positions 10.0 /
// 14.7, 16384 15.9 / 15.1, 65536 50 / 16; 32 units of 4096 10.3 / 41.9, 32768
// 27.2 / 42.7, 65536 51 / 45, 131072 101 / 65; 64 units of 65536 51 / 75: 5.6
// us per round of 8192 positions and CTA, and 14 per wave of clusters.
bool select_one_cta(const EvictArgs &a, int sms) {
  auto rounds = [](int64_t n) { return (double)((n + 8191) / 8192); };
  const double waves = (double)((a.v.B * a.v.Hkv * kSelParts + sms - 1) / sms);
  const double one = 4.4 + 5.6 * rounds(a.len_hi);
  const double cluster = (waves > 1.0 ? 14.0 : 1.0) + waves * (4.0 + 10.0 * rounds(a.len_hi / kSelParts));
  return one <= cluster;
}

cudaError_t launch_evict_select(const EvictArgs &a, cudaStream_t st) {
  static int sms = 0;
  if (!sms) {
    int dev = 0, n = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    sms = n;
  }
  if (select_one_cta(a, sms)) return launch_pdl(evict_select_kernel<1>, dim3(a.v.Hkv, a.v.B), dim3(1024), 0, st, a);
  return launch_pdl(evict_select_kernel<kSelParts>, dim3(a.v.Hkv * kSelParts, a.v.B), dim3(1024), 0, st, a);
}

// ---------------------------------------------------------------------------
// Tensor-core scoring (tcgen05; head_dim 128, at most 256 window rows).
//
// The scores of a 128-position tile are one UMMA chain over K = 128
// channels.  The dequantised keys, split into bf16 hi + lo, and the window
// query rows (split likewise when they arrive in fp32; bf16 queries have no
// lo part) sit in shared memory in the K-major 128-byte-swizzled layout
// (two 64-channel boxes of 128-byte rows, 16-byte chunk c of row r stored at
// chunk c ^ (r & 7)).  hi*hi + hi*lo + lo*hi keeps ~16 significant bits of
// each factor (the dropped lo*lo term is below 2^-16 of the product); the
// tensor cores accumulate in fp32 in TMEM.
// Both passes take A = keys (M = 128 positions) and B = query rows (N = R
// rounded up to 16): TMEM lane = position, column = row, one chain for all
// rows (with A = rows in chunks of 128, as the statistics ran before, 160
// rows took 32 products at about 160 cycles an item, this way 16 at 125).
//  * statistics pass: each thread sums 2^(x - ref) of its lane's positions
//    for a quarter of the rows, in registers over all the tiles that its CTA
//    walks of a unit; a warp's reference of a row is its first lane's first
//    score and moves (to the warp's maximum) only when a score rises more
//    than 64 above it, so the warp's lanes meet only then and, 31 shuffles
//    for 32 rows, at the unit's end.  Tiles that every row sees in full, past
//    the unit's first, run a copy of the code without masks;
//  * vote pass: each thread sums its position's weights over the rows.
// The vote pass recomputes the scores: on the tensor cores that is cheaper
// than a round trip through HBM.  A CTA (one per SM) walks a contiguous range
// of (unit, tile) items in four roles that run beside each other: 3 warps
// copy the keys' records in, 8 dequantise them (the ALU's share), one issues
// the chains, 16 run the epilogues (the exponentials' share), two key stages
// and two TMEM buffers between them.
//
// What bounds it: issue slots (69-71 % busy), about evenly over the roles.
// At the 131k-context shape (32 units of int4 records, 160 rows) an item takes
// 3950 cycles in the statistics pass (452 us) and 3250 in the vote pass (384
// us), of which a dequantising warp works 3250 and 2750, the chain's issue
// 3450 and 2750 (16 products at 125-160 cycles beside the others' shared-
// memory traffic, 80 alone) and an epilogue warp 3250 and 1950.  One group of
// 16 warps that dequantised and ran the epilogues in turn took 6200 and 4950
// cycles (704 and 560 us).  Of what the roles' own code cost, the cursor over
// the items was a tenth (28 warps each checked the unit's limits per item;
// now once per unit), the masks in the statistics epilogue 400 cycles, and
// per unit the shuffles of a butterfly per row and the query rows' loads one
// at a time 25 us.  Packed binary32 arithmetic in the epilogues gained
// nothing (945 and 944 us a call).
// The statistics stay in registers over a CTA's tiles of a unit and leave
// once per CTA and unit (stored per tile they were 168 MB of traffic and a
// 59 us merge).  Query rows past R are zero.
constexpr int kTcEpi = 512;                  // epilogue threads (warps 0-15)
constexpr int kTcDeq = 256;                  // dequantising threads (warps 16-23)
constexpr int kTcCopy = 96;                  // copying threads (warps 24-26)
constexpr int kTcThreads = kTcEpi + kTcDeq + kTcCopy + 32;  // + the MMA warp
constexpr int kTcPv = 1024;                  // floats: partial votes (2 x 3 x 128) or references (16 x 64)
static_assert(kEvictStatSub == kTcEpi / 128, "one statistics entry per column slice");

// Sums over the warp of N values a lane (8 or 32): x[0] of lane L becomes the
// sum of value L (N = 32) or L / 4 (N = 8).  Each step halves the values that
// a lane carries, 31 or 9 shuffles where a butterfly per value takes 5 N (16
// warps' 64 sums each took 19500 cycles so).
template <int N>
__device__ __forceinline__ void lanes_sum(float (&x)[N]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    const int h = N * o / 32;  // values kept by a step that halves them
    if (h) {
#pragma unroll
      for (int i = 0; i < h; ++i) {
        const bool up = lane & o;
        const float send = up ? x[i] : x[i + h];
        x[i] = (up ? x[i + h] : x[i]) + __shfl_xor_sync(0xffffffffu, send, o);
      }
    } else {
      x[0] += __shfl_xor_sync(0xffffffffu, x[0], o);
    }
  }
}

struct TcPlan {
  int items_per_cta, n_items;
  int R16, q_lo, k_lo, nst, nstg, fmt;  // nst key stages, nstg staging buffers
  int kb_nch, kb_stride, stg_bytes;  // staged 16-byte chunks per position, their stride
  int nc_magic;                      // ceil(2^16 / kb_nch): e / kb_nch = (e nc_magic) >> 16 here
  int stage, off_q, off_ql, off_k, off_stg, off_norm, off_pv, off_bar, smem;
};

// NB (statistics pass): blocks of 8 rows that a slice holds at most
template <bool VOTES, int NB>
__global__ void __launch_bounds__(kTcThreads, 1) evict_tc_kernel(const EvictArgs a, const TcPlan p) {
  extern __shared__ uint8_t evict_tc_raw[];
  uint8_t *sm = evict_tc_raw + ((1024u - (smem_u32(evict_tc_raw) & 1023u)) & 1023u);
  // Item k of the CTA: chain[k & 1] its products done, keys[k & 1] its keys
  // staged (an arrival per dequantising warp), epi[k & 1] its epilogue done
  // (an arrival per epilogue warp); staging buffer g: sfull[g] copied (an
  // arrival per copying thread), sfree[g] dequantised (one per warp); unit n
  // of the CTA: uready[n & 1] its query rows (and norms) loaded; drain.  Every barrier's next completion
  // but one depends on every waiter's having seen this one.
  uint64_t *bar = reinterpret_cast<uint64_t *>(sm + p.off_bar);
  uint64_t *chain = bar, *keys = bar + 2, *epi = bar + 4, *uready = bar + 6, *drain = bar + 8, *sfull = bar + 9,
           *sfree = bar + 11;
  constexpr int kBars = 13;
  uint32_t *tbase = reinterpret_cast<uint32_t *>(bar + kBars);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(tbase + 1);
  float *norm = reinterpret_cast<float *>(sm + p.off_norm);
  float *pv = reinterpret_cast<float *>(sm + p.off_pv);
  uint8_t *qh = sm + p.off_q, *ql = sm + p.off_ql;
  const GqaView &v = a.v;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int R = a.n_win * a.G;
  constexpr uint32_t kLimit = 1u << 22;
  constexpr uint32_t kSleepyLimit = 1u << 20;  // polls of up to 2 us each
  constexpr int D = 128;
  constexpr int KBOX = 128 * 128;  // bytes of one 64-channel box of a 128-row key tile

  if (tid == 0) {
    for (int i = 0; i < kBars; ++i)
      mbar_init(&bar[i], i < 2 || i == 8 ? 1 : i == 4 || i == 5 ? kTcEpi / 32 : i == 9 || i == 10 ? kTcCopy : kTcDeq / 32);
    *abort_flag = 0;
    fence_mbar_init();
  }
  pdl_wait();  // the cache, lengths and (vote pass) merged statistics are complete
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tbase)),
                 "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tbase;

  const int it0 = blockIdx.x * p.items_per_cta;
  const int it1 = min(it0 + p.items_per_cta, p.n_items);
  // epilogue warp w reads TMEM lanes 32 (w % 4) .. + 31; slice = w / 4
  const int quarter = warp & 3, slice = warp >> 2;
  const uint32_t lane_off = (uint32_t)(quarter * 32) << 16;
  const int did = tid - kTcEpi, cid = did - kTcDeq;  // index among the dequantising, the copying threads
  auto sleepy = [&](uint64_t *b, uint32_t parity) {
    return mbar_wait_sleepy(b, parity, kSleepyLimit, abort_flag, 2000);
  };

  const int gshift = v.group == 64 ? 6 : 5;  // grouped layers: groups of 32 or 64 channels
  // (unit, tile) of item `it`, the unit's length and the item after its last
  // valid tile (none: at most `it`), advanced without divisions; within a
  // unit a step is two additions and a compare
  struct Cursor {
    int it, unit, tile, len, end;
  };
  const int units = v.B * v.Hkv;
  auto unit_end = [&](Cursor &c) {  // c at tile c.tile of c.unit
    c.len = c.unit < units ? v.lens[c.unit / v.Hkv] : 0;
    const int n = c.len > a.budget ? ((VOTES ? c.len - a.n_win : c.len) + kT - 1) / kT : 0;  // valid tiles
    c.end = min(it1, c.it + n - c.tile);
  };
  auto next_unit = [&](Cursor c) {  // the first valid item at or after c (c.it == it1: none)
    while (c.it < it1 && c.it >= c.end) {
      c.it += a.n_tiles - c.tile;
      c.tile = 0;
      ++c.unit;
      unit_end(c);
    }
    c.it = min(c.it, it1);
    return c;
  };
  auto first = [&]() {
    Cursor c;
    c.it = it0;
    c.unit = it0 / a.n_tiles;
    c.tile = it0 - c.unit * a.n_tiles;
    unit_end(c);
    return next_unit(c);
  };
  auto step = [&](Cursor c) {
    ++c.it;
    ++c.tile;
    return c.it < c.end ? c : next_unit(c);
  };

  // query rows of `unit` (and, for the votes, the rows' log-normalisers;
  // +inf for the padding rows, whose weights are then 0)
  auto load_q = [&](int unit, int n) {
    const int b = unit / v.Hkv, j = unit % v.Hkv;
    const int box = p.R16 * 128;
    // thread: chunk c8 of rows did / 16 + 16 i; row r is query w = r / G of
    // head r % G, carried from row to row
    const int c8 = did & 15, dw = (kTcDeq / 16) / a.G, dg = kTcDeq / 16 - dw * a.G;
    int r = did >> 4, w = r / a.G, g = r - w * a.G;
    for (; r < p.R16; r += kTcDeq / 16) {
      const size_t qi = (((size_t)b * a.n_win + (r < R ? w : 0)) * a.Hq + j * a.G + g) * D + 8 * c8;
      if (a.q_f32) {
        float x[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) x[i] = 0.f;
        if (r < R) {
          const float4 u0 = *reinterpret_cast<const float4 *>(static_cast<const float *>(a.q) + qi);
          const float4 u1 = *reinterpret_cast<const float4 *>(static_cast<const float *>(a.q) + qi + 4);
          x[0] = u0.x; x[1] = u0.y; x[2] = u0.z; x[3] = u0.w;
          x[4] = u1.x; x[5] = u1.y; x[6] = u1.z; x[7] = u1.w;
        }
        put8(qh, ql, r, 8 * c8, box, x);
      } else {
        cp_async16(qh + (c8 >> 3) * box + r * 128 + (((c8 & 7) ^ (r & 7)) << 4), static_cast<const uint16_t *>(a.q) + qi,
                   r < R);
      }
      w += dw;
      g += dg;
      if (g >= a.G) {
        g -= a.G;
        ++w;
      }
    }
    if constexpr (VOTES) {
      float *nm = norm + p.R16 * (n & 1);
      for (int r = did; r < p.R16; r += kTcDeq) {
        if (r < R) {
          const float2 f = a.fin[(size_t)unit * R + r];
          nm[r] = f.x + log2f(f.y);
        } else {
          nm[r] = INFINITY;
        }
      }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    fence_proxy_async();
  };

  // asynchronous copy of the K bundles of item `it` (K section in logical
  // order, then the group metadata or the symmetric scale word) into staging
  // buffer g, then the buffer's arrival (once the thread's copies landed)
  auto stage_copy = [&](const Cursor &cu, int g) {
    const int unit = cu.unit, t0 = cu.tile * kT, len = cu.len;
    uint8_t *dst0 = sm + p.off_stg + g * p.stg_bytes;
    const int NC = p.kb_nch;
    const int ks16 = TcFmtKs16(p.fmt);
    const bool sym = p.fmt >= kFmtS8;
    const int nrec = v.rec_bytes >> 4;
    const int km = ks16 * 32;  // grouped: key metadata follows the K and V sections
    const uint8_t *base = v.rec + (size_t)unit * v.cap * v.rec_bytes;
    for (int e = cid; e < kT * NC; e += kTcCopy) {
      const int pos = (e * p.nc_magic) >> 16, c = e - pos * NC;
      const int t = t0 + pos;
      const bool ok = t < len;
      const int so = sym ? 16 * ((c + sym_rot(t, nrec)) & (nrec - 1)) : c < ks16 ? 16 * c : km + 16 * (c - ks16);
      cp_async16(dst0 + pos * p.kb_stride + 16 * c, base + (size_t)(ok ? t : t0) * v.rec_bytes + so, ok);
    }
    if (sym)
      for (int pos = cid; pos < kT; pos += kTcCopy) {
        const int t = t0 + pos;
        const bool ok = t < len;
        cp_async4(dst0 + pos * p.kb_stride + 16 * ks16,
                  v.scales + (size_t)unit * v.cap + (ok ? t : t0), ok);
      }
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(&sfull[g])) : "memory");
  };

  // dequantised keys of the item staged in buffer g into key stage s
  auto dequant = [&](int g, int s) {
    const int pidx = did & 127;  // position
    const uint8_t *bundle = sm + p.off_stg + g * p.stg_bytes + pidx * p.kb_stride;
    uint8_t *kh = sm + p.off_k + s * p.stage, *kl = kh + 2 * KBOX;
#pragma unroll 1
    for (int hf = did >> 7; hf < 4; hf += 2)  // channel quarters
      switch (p.fmt) {
      case kFmtBf16: tc_dequant<kFmtBf16>(bundle, bundle + TcFmtKs16(kFmtBf16) * 16, pidx, hf, gshift, kh, kl); break;
      case kFmtG8: tc_dequant<kFmtG8>(bundle, bundle + TcFmtKs16(kFmtG8) * 16, pidx, hf, gshift, kh, kl); break;
      case kFmtG4: tc_dequant<kFmtG4>(bundle, bundle + TcFmtKs16(kFmtG4) * 16, pidx, hf, gshift, kh, kl); break;
      case kFmtS8: tc_dequant<kFmtS8>(bundle, bundle + TcFmtKs16(kFmtS8) * 16, pidx, hf, gshift, kh, kl); break;
      case kFmtS4: tc_dequant<kFmtS4>(bundle, bundle + TcFmtKs16(kFmtS4) * 16, pidx, hf, gshift, kh, kl); break;
      default: tc_dequant<kFmtS2>(bundle, bundle + TcFmtKs16(kFmtS2) * 16, pidx, hf, gshift, kh, kl); break;
    }
  };

  // one MMA chain for the tile in key stage s into TMEM buffer tb (thread 0)
  auto issue = [&](int s, int tb) {
    tc_fence_after();
    const uint32_t kh = smem_u32(sm + p.off_k + s * p.stage), kl = kh + 2 * KBOX;
    const uint32_t qa = smem_u32(qh), qb = smem_u32(ql);
    const uint32_t qbox = (uint32_t)p.R16 * 128;
    const uint32_t d0 = tmem + 256u * tb;
    constexpr uint32_t hi = umma_desc_hi_sw128(1024);
    const uint32_t dkh = umma_desc_lo(kh, 16), dkl = umma_desc_lo(kl, 16), dqh = umma_desc_lo(qa, 16),
                   dql = umma_desc_lo(qb, 16);
    const uint32_t id = umma_idesc(128, p.R16, false, false);
#pragma unroll
    for (int ks = 0; ks < D / 16; ++ks) {
      const uint32_t ko = ((ks >> 2) * KBOX + (ks & 3) * 32) >> 4;
      const uint32_t qo = (ks >> 2) * (qbox >> 4) + 2 * (ks & 3);
      umma_f16_ss_w(d0, dkh + ko, dqh + qo, hi, id, ks > 0);
      if (p.k_lo) umma_f16_ss_w(d0, dkl + ko, dqh + qo, hi, id, true);
      if (p.q_lo) umma_f16_ss_w(d0, dkh + ko, dql + qo, hi, id, true);
    }
    umma_commit(&chain[tb]);
  };

  // Statistics pass: this thread's sums of a slice's rows over its lane's
  // positions of the unit's tiles, relative to the warp's references (shared
  // memory, 64 per warp: the slice's rows in order).
  constexpr int BW = VOTES ? 16 : 8;  // rows of a block
  const int nblk = p.R16 / BW, per = (nblk + 3) / 4;
  const int bk0 = min(nblk, slice * per), bk1 = min(nblk, bk0 + per);
  float l_run[8 * NB];
  float *ref = pv + 64 * warp;
  bool fresh = true;  // the unit has no references yet
  auto flush_stats = [&](int unit) {
    const int stride = kEvictStatSub * a.n_tiles;
    const int e = kEvictStatSub * ((int)blockIdx.x - unit * a.n_tiles / p.items_per_cta) + quarter;
    auto put = [&](int i, float L) {  // the slice's row i
      const int r = 8 * bk0 + i;
      if (r < 8 * bk1 && r < R) a.stats[((size_t)unit * R + r) * stride + e] = make_float2(ref[i], L);
    };
#pragma unroll
    for (int b = 0; b + 4 <= NB; b += 4) {  // 32 rows at a time
      float x[32];
#pragma unroll
      for (int i = 0; i < 32; ++i) x[i] = l_run[8 * b + i];
      lanes_sum(x);
      put(8 * b + lane, x[0]);
    }
#pragma unroll
    for (int b = NB / 4 * 4; b < NB; ++b) {  // 8
      float x[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) x[i] = l_run[8 * b + i];
      lanes_sum(x);
      if ((lane & 3) == 0) put(8 * b + (lane >> 2), x[0]);
    }
  };
  // epilogue of item `cu` (the k-th) from TMEM buffer tb
  auto epilogue = [&](const Cursor &cu, int tb, const float *nm) {
    const int unit = cu.unit, tile = cu.tile, len = cu.len;
    const int P = len - a.n_win;
    const int t0 = tile * kT;
    const float sg = a.sig_log2;
    if constexpr (!VOTES) {
      const int t = t0 + 32 * quarter + lane;
      // row r of window query w = r / G sees positions up to P + w: rows
      // before (t - P) G do not see this lane's position
      const int r_from = (t - P) * a.G;
      const bool whole = t0 + 32 * quarter + 31 <= P;
      // tiles that every row sees in full, past the unit's first: no masks
      auto tiles = [&](auto hot_t) {
        constexpr bool hot = decltype(hot_t)::value;
#pragma unroll
      for (int b = 0; b < NB; b += 2) {  // 16 rows at a time (8 at an odd end)
        if (bk0 + b >= bk1) break;
        const uint32_t ta = tmem + 256u * tb + 8 * (bk0 + b) + lane_off;
        const int n = bk0 + b + 1 < bk1 && b + 1 < NB ? 16 : 8;
        float z[16];
        tmem_ld16(ta, z);  // past an odd end: another slice's rows, unused
        if (!hot && !whole) {
#pragma unroll
          for (int i = 0; i < 16; ++i)
            if (8 * (bk0 + b) + i < r_from) z[i] = -INFINITY;
        }
        if (!hot && fresh) {
          // lane 0's scores (its position is visible where any lane's is)
          if (lane == 0) {
#pragma unroll
            for (int i = 0; i < 16; ++i)
              if (i < n) ref[8 * b + i] = z[i] * sg;
          }
#pragma unroll
          for (int i = 0; i < 16; ++i)
            if (8 * b + i < 8 * NB) l_run[8 * b + i] = 0.f;
          __syncwarp();
        }
        float top = -INFINITY;
        const float4 *r4 = reinterpret_cast<const float4 *>(ref + 8 * b);
#pragma unroll
        for (int i4 = 0; i4 < 4; ++i4) {
          if (4 * i4 >= n) continue;
          const float4 c = r4[i4];
          z[4 * i4] = fmaf(z[4 * i4], sg, -c.x);
          z[4 * i4 + 1] = fmaf(z[4 * i4 + 1], sg, -c.y);
          z[4 * i4 + 2] = fmaf(z[4 * i4 + 2], sg, -c.z);
          z[4 * i4 + 3] = fmaf(z[4 * i4 + 3], sg, -c.w);
          if (!hot && !whole) {  // -inf - -inf, masked and without a reference yet: adds nothing
#pragma unroll
            for (int i = 4 * i4; i < 4 * i4 + 4; ++i) z[i] = fmaxf(z[i], -INFINITY);
          }
          top = fmaxf(top, fmaxf(fmaxf(z[4 * i4], z[4 * i4 + 1]), fmaxf(z[4 * i4 + 2], z[4 * i4 + 3])));
        }
        if (__builtin_expect(__any_sync(0xffffffffu, top > 64.f), 0)) {
          // the references move to the warp's maxima where scores pass them;
          // a row whose positions so far are all masked keeps -inf
          auto scores = [&]() {
            tmem_ld16(ta, z);
#pragma unroll
            for (int i = 0; i < 16; ++i)
              if (!hot && !whole && 8 * (bk0 + b) + i < r_from) z[i] = -INFINITY;
          };
          scores();
#pragma unroll
          for (int o = 16; o; o >>= 1)  // 16 reductions side by side
#pragma unroll
            for (int i = 0; i < 16; ++i) z[i] = fmaxf(z[i], __shfl_xor_sync(0xffffffffu, z[i], o));
          __syncwarp();
#pragma unroll
          for (int i4 = 0; i4 < 4; ++i4) {
            if (4 * i4 >= n) continue;
            const float4 c4 = r4[i4];
            const float c[4] = {c4.x, c4.y, c4.z, c4.w};
            float m[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              m[u] = fmaxf(z[4 * i4 + u] * sg, c[u]);
              if (8 * b + 4 * i4 + u < 8 * NB && m[u] > c[u]) l_run[8 * b + 4 * i4 + u] *= fast_exp2(c[u] - m[u]);
            }
            __syncwarp();
            if (lane == 0) reinterpret_cast<float4 *>(ref + 8 * b)[i4] = make_float4(m[0], m[1], m[2], m[3]);
          }
          __syncwarp();
          scores();
#pragma unroll
          for (int i4 = 0; i4 < 4; ++i4) {
            if (4 * i4 >= n) continue;
            const float4 c = r4[i4];
            z[4 * i4] = fmaxf(fmaf(z[4 * i4], sg, -c.x), -INFINITY);
            z[4 * i4 + 1] = fmaxf(fmaf(z[4 * i4 + 1], sg, -c.y), -INFINITY);
            z[4 * i4 + 2] = fmaxf(fmaf(z[4 * i4 + 2], sg, -c.z), -INFINITY);
            z[4 * i4 + 3] = fmaxf(fmaf(z[4 * i4 + 3], sg, -c.w), -INFINITY);
          }
        }
        // masked positions add 2^-inf = 0
#pragma unroll
        for (int i = 0; i < 16; ++i)
          if (8 * b + i < 8 * NB && i < n) l_run[8 * b + i] += fast_exp2(z[i]);
      }
      };
      if (whole && !fresh)
        tiles(std::true_type{});
      else
        tiles(std::false_type{});
      fresh = false;
    } else {
      const int pos = 32 * quarter + lane, t = t0 + pos;
      float vv[4] = {0.f, 0.f, 0.f, 0.f};  // four independent chains
      for (int bk = bk0; bk < bk1; ++bk) {
        float y[16];
        tmem_ld16(tmem + 256u * tb + 16 * bk + lane_off, y);
        const float4 *nr = reinterpret_cast<const float4 *>(nm + 16 * bk);
#pragma unroll
        for (int i4 = 0; i4 < 4; ++i4) {
          const float4 c4 = nr[i4];
          vv[0] += fast_exp2(fmaf(y[4 * i4], sg, -c4.x));
          vv[1] += fast_exp2(fmaf(y[4 * i4 + 1], sg, -c4.y));
          vv[2] += fast_exp2(fmaf(y[4 * i4 + 2], sg, -c4.z));
          vv[3] += fast_exp2(fmaf(y[4 * i4 + 3], sg, -c4.w));
        }
      }
      // the four slices of a position are in the four warps of its quarter
      const float vote = (vv[0] + vv[1]) + (vv[2] + vv[3]);
      float *pb = pv + 3 * 128 * tb;
      if (slice) pb[(slice - 1) * 128 + pos] = vote;
      asm volatile("bar.sync %0, 128;" ::"r"(4 + quarter) : "memory");
      if (!slice && t < P) a.votes[(size_t)unit * v.cap + t] = vote + pb[pos] + pb[128 + pos] + pb[256 + pos];
    }
  };

  // Registers by warpgroup: the epilogues' sums take more than an equal share.
  // 512 x 88 + 256 x 56 + 128 x 40 = 64512 = the 896 x 72 launched.
  static_assert(kEvictRegs.threads[0] == kTcEpi && kEvictRegs.threads[1] == kTcDeq &&
                    kEvictRegs.all_threads() == kTcThreads && kEvictRegs.fits(72),
                "the register split");
  if (warp >= (kTcEpi + kTcDeq) / 32) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kEvictRegs.regs[2]) : "memory");
    if (warp == (kTcEpi + kTcDeq + kTcCopy) / 32) {
      // ======================= MMA warp =====================================
      // the same item sequence as the others; each chain once its keys are
      // staged and its TMEM buffer was read
      int k = 0;
      for (Cursor cu = first(); cu.it < it1; cu = step(cu), ++k) {
        bool ok = sleepy(&keys[k & 1], (k >> 1) & 1);
        if (ok && k >= 2) ok = sleepy(&epi[k & 1], ((k >> 1) - 1) & 1);
        if (!__all_sync(0xffffffffu, ok)) {
          if (lane == 0) {
            *abort_flag = 1;
            set_err(a.err, 8);
          }
          break;
        }
        if (lane == 0) issue(k % p.nst, k & 1);
        __syncwarp();
      }
      // every chain issued lands before TMEM is released (bounded)
      if (lane == 0 && k > 0) {
        umma_commit(drain);
        mbar_wait(drain, 0, kLimit);
      }
      __syncwarp();
    } else {
      // ======================= copies =======================================
      int k = 0, g = 0;
      uint32_t ph = 1;  // a buffer's first use waits for nothing
      for (Cursor it = first(); it.it < it1; it = step(it), ++k) {
        if (!__all_sync(0xffffffffu, sleepy(&sfree[g], ph))) {
          *abort_flag = 1;
          break;
        }
        stage_copy(it, g);
        if (++g == p.nstg) {
          g = 0;
          ph ^= 1;
        }
      }
      asm volatile("cp.async.wait_all;" ::: "memory");  // no copy outlives the CTA
    }
  } else if (warp >= kTcEpi / 32) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kEvictRegs.regs[1]) : "memory");
    // ======================= dequantising =================================
    // A thread whose wait gave up goes on without work.
    bool failed = false;
    int cur_unit = -1, n_unit = 0, k = 0, g = 0;
    uint32_t ph = 0;
    for (Cursor it = first(); it.it < it1; it = step(it), ++k) {
      // the key stage is free once the chain that read it is done; a new
      // unit's rows replace the last unit's after its last chain, and its
      // norms those of two units ago, whose last epilogue is k - 2 at most
      if (k >= p.nst && !failed) {
        const int c = k - p.nst;
        failed = !sleepy(&chain[c & 1], (c >> 1) & 1);
      }
      if (it.unit != cur_unit) {
        if (k >= 1 && !failed) failed = !sleepy(&chain[(k - 1) & 1], ((k - 1) >> 1) & 1);
        if (k >= 2 && !failed) failed = !sleepy(&epi[k & 1], ((k >> 1) - 1) & 1);
        if (!failed) load_q(it.unit, n_unit);
        __syncwarp();
        if (lane == 0) mbar_arrive(&uready[n_unit & 1]);
        cur_unit = it.unit;
        ++n_unit;
      }
      if (!failed) failed = !sleepy(&sfull[g], ph);
      if (!failed) dequant(g, k % p.nst);
      fence_proxy_async();  // the keys, written here, are read by the tensor cores
      __syncwarp();
      if (failed) *abort_flag = 1;
      if (lane == 0) {
        mbar_arrive(&keys[k & 1]);
        mbar_arrive(&sfree[g]);
      }
      if (++g == p.nstg) {
        g = 0;
        ph ^= 1;
      }
    }
    if (failed) set_err(a.err, 8);
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kEvictRegs.regs[0]) : "memory");
    // ======================= epilogues ====================================
    // A warp whose wait gave up goes on through the barriers without work.
    bool failed = false;
    int cur_unit = -1, n_unit = -1, k = 0;
    for (Cursor it = first(); it.it < it1; it = step(it), ++k) {
      if (it.unit != cur_unit) {
        if constexpr (!VOTES) {
          if (cur_unit >= 0) flush_stats(cur_unit);
        }
        cur_unit = it.unit;
        ++n_unit;
        fresh = true;
        if (!failed) failed = !__all_sync(0xffffffffu, sleepy(&uready[n_unit & 1], (n_unit >> 1) & 1));
      }
      if (!failed) failed = !__all_sync(0xffffffffu, sleepy(&chain[k & 1], (k >> 1) & 1));
      if (failed) *abort_flag = 1;
      tc_fence_after();
      epilogue(it, k & 1, norm + p.R16 * (n_unit & 1));
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&epi[k & 1]);
    }
    if constexpr (!VOTES) {
      if (cur_unit >= 0) flush_stats(cur_unit);
    }
    if (failed && lane == 0) set_err(a.err, 8);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512)
                 : "memory");
  pdl_trigger();
}

// Shared-memory plan of the tensor-core kernels: the query rows first (hi,
// then lo); two key stages when they fit, else one; two staging buffers of
// the K bundles.  Bundle strides are odd multiples of 16 bytes, so the
// 16-byte loads of eight consecutive positions fall in distinct banks.
TcPlan tc_plan(const EvictArgs &a, int sms) {
  TcPlan p;
  const int R = a.n_win * a.G;
  p.R16 = (R + 15) / 16 * 16;
  p.q_lo = a.q_f32 ? 1 : 0;
  p.k_lo = a.v.bits != 16 ? 1 : 0;
  p.fmt = a.v.bits == 16 ? kFmtBf16
          : a.v.scheme == kSchemeSym ? (a.v.bits == 8 ? kFmtS8 : a.v.bits == 4 ? kFmtS4 : kFmtS2)
                                     : (a.v.bits == 8 ? kFmtG8 : kFmtG4);
  const int ks16 = TcFmtKs16(p.fmt);
  const int extra = a.v.bits == 16 ? 0 : a.v.scheme == kSchemeSym ? 1 : meta_bytes(128, a.v.group) / 16;
  p.kb_nch = ks16 + (a.v.scheme == kSchemeSym ? 0 : extra);  // the scale word is copied apart
  const int kb = ks16 + extra;
  p.kb_stride = 16 * (kb % 2 ? kb : kb + 1);
  p.nc_magic = (65536 + p.kb_nch - 1) / p.kb_nch;
  p.stg_bytes = kT * p.kb_stride;
  p.stage = p.k_lo ? 4 * 128 * 128 : 2 * 128 * 128;
  p.off_q = 0;
  p.off_ql = p.R16 * 256;
  const int qbytes = p.R16 * 256 * (p.q_lo ? 2 : 1);
  p.off_k = (qbytes + 1023) / 1024 * 1024;
  auto fits = [&](int nst, int nstg) {
    return p.off_k + nst * p.stage + nstg * p.stg_bytes + 2 * p.R16 * 4 + kTcPv * 4 + 128 + 1024 <= 232448;
  };
  p.nst = fits(2, 2) ? 2 : 1;
  p.nstg = fits(p.nst, 2) ? 2 : 1;
  p.off_stg = p.off_k + p.nst * p.stage;
  p.off_norm = p.off_stg + p.nstg * p.stg_bytes;
  p.off_pv = p.off_norm + 2 * p.R16 * 4;
  p.off_bar = p.off_pv + kTcPv * 4;
  p.smem = p.off_bar + 128 + 1024;  // + alignment of the base to 1024 bytes
  p.n_items = a.v.B * a.v.Hkv * a.n_tiles;
  const int grid = std::max(1, std::min(p.n_items, sms));
  p.items_per_cta = (p.n_items + grid - 1) / grid;
  return p;
}

cudaError_t launch_evict_tc(const EvictArgs &args, cudaStream_t st) {
  static int sms = 0;
  if (!sms) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
  }
  EvictArgs a = args;
  const TcPlan p = tc_plan(a, sms);
  a.items_per_cta = p.items_per_cta;
  // 160 rows (5 query heads, 32 queries) fit 40 sums a thread
  const bool few = p.R16 <= 160;
  auto stat = few ? evict_tc_kernel<false, 5> : evict_tc_kernel<false, 8>;
  cudaError_t e = few ? check_reg_split<&evict_tc_kernel<false, 5>>(kEvictRegs)
                      : check_reg_split<&evict_tc_kernel<false, 8>>(kEvictRegs);
  if (e == cudaSuccess) e = check_reg_split<&evict_tc_kernel<true, 1>>(kEvictRegs);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(stat, cudaFuncAttributeMaxDynamicSharedMemorySize, p.smem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(evict_tc_kernel<true, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, p.smem);
  if (e != cudaSuccess) return e;
  const dim3 grid((p.n_items + p.items_per_cta - 1) / p.items_per_cta);
  e = launch_pdl(stat, grid, dim3(kTcThreads), p.smem, st, a, p);
  if (e == cudaSuccess) {
    const int rows = a.v.B * a.v.Hkv * a.n_win * a.G;
    e = launch_pdl(evict_merge_stats_kernel, dim3((rows + kMergeWarps - 1) / kMergeWarps),
                   dim3(32 * kMergeWarps), 0, st, a);
  }
  if (e == cudaSuccess) e = launch_pdl(evict_tc_kernel<true, 1>, grid, dim3(kTcThreads), p.smem, st, a, p);
  if (e == cudaSuccess)
    e = launch_evict_select(a, st);
  return e;
}

template <int D>
cudaError_t launch_evict_d(const EvictArgs &a, cudaStream_t st) {
  constexpr int smem = evict_smem<D>();
  cudaError_t e = cudaFuncSetAttribute(evict_scores_kernel<D>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  e = launch_pdl(evict_scores_kernel<D>, dim3(a.n_tiles, a.v.Hkv, a.v.B), dim3(kThreads), smem, st, a);
  if (e == cudaSuccess) {
    const int rows = a.v.B * a.v.Hkv * a.n_win * a.G;
    e = launch_pdl(evict_merge_stats_kernel, dim3((rows + kMergeWarps - 1) / kMergeWarps),
                   dim3(32 * kMergeWarps), 0, st, a);
  }
  if (e == cudaSuccess)
    e = launch_pdl(evict_votes_kernel, dim3((a.v.cap + kVoteT - 1) / kVoteT, a.v.Hkv, a.v.B),
                   dim3(kVoteT), 0, st, a);
  if (e == cudaSuccess)
    e = launch_evict_select(a, st);
  return e;
}

}  // namespace

cudaError_t launch_gqa_evict(const EvictArgs &a, cudaStream_t st) {
  if (evict_uses_tc(a.v.D, a.n_win * a.G)) return launch_evict_tc(a, st);
  switch (a.v.D) {
    case 128: return launch_evict_d<128>(a, st);
    case 64: return launch_evict_d<64>(a, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace kvk
