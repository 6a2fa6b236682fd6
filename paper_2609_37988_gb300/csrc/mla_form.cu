// mla_form.cu -- per-head keys and values of an MLA latent cache, formed once
// for a chunk of queries to attend over (pre-fill):
//   K[b, t, h, :] = W_UK[h][:, :d] c_t[:d],   V[b, t, h, :] = W_UV[h][:, :d] c_t[:d]
// (Appendix B; the decode's absorbed form, Appendix C.2, moves the same two
// products to the query and the output).  A chunk of n query rows costs
// n (4 d + 2 d_R) flops per position and head absorbed and 4 d Dn + n (4 Dn +
// 2 d_R) formed, Dn = 128: at d = 512 and n = 1024 that is 2.3 times less
// work, the attention becomes the head_dim-128 kernel of prefill.cu (rows =
// queries of one head, M = 128 products) and the latents are read once.
//
// One GEMM: rows = positions (blocks of 128, M = 128), columns = one head's
// 128 key and 128 value channels (N = 256), K = d.  Persistent CTAs, each an
// equal contiguous run of the (block, head) items, block-major: the block's
// latents stay in shared memory (128-byte swizzled K-major boxes of 64
// coordinates) while the heads' weights stream through a TMA ring, 32 KB
// (64 coordinates of 256 rows) per stage; two 256-column accumulators in TMEM, so
// that the products of an item run under the epilogue of the one before it.
// Quantised latents enter as centred codes, exact in bf16 (|code| <= 255),
// and the epilogue applies each position's scale, and its offset times the
// weights' column sums (mla_wsum_kernel): one product either way.
// Results leave as hi + lo halves in the tile layout prefill.cu copies (128
// positions: key units by 64 channels, value units by 64 positions), 32 bytes
// (16 channels) per thread and store: the swizzle keeps such a pair of
// 16-byte chunks in one aligned sector.  Keys split into bf16 (their rounding
// reaches the output through the scores: 2e-7 of it), values into f16 with a
// power-of-two scale per 32 positions: bf16 halves of the values, and of the
// weights that multiply them, each cost 2.4e-6 of the output and the dropped
// lo x lo products 2.8e-6, in all 4.4e-6 where the absorbed form has 2.7e-6
// (4-bit latents, 700 positions).  Values that are not finite (of a latent
// that is not) enter as zeros and are recorded (PfArgs::bad).  The positional
// keys are copied beside (hi, and lo for quantised latents) once per block.
//
// Bound by the weights' L2 traffic (64 bytes per cycle and SM at d = 512) and
// the 64 KB per tile and head it writes.
#include <cuda.h>  // CUtensorMap and its enums (the encoder is reached through the runtime)

#include <algorithm>

#include "common.cuh"
#include "kernels.h"
#include "layout.h"
#include "umma.cuh"

namespace kvk {
namespace {

constexpr int kFmEpi = 256;                  // epilogue (and staging) threads: 8 warps
constexpr int kFmThreads = kFmEpi + 64;      // + the MMA warp and the weight-copy warp
constexpr int kFmRows = 128;                 // positions per block
constexpr int kFmABox = kFmRows * 128;       // 64 coordinates of a block (16 KB)
constexpr int kFmWStage = 256 * 128;         // 64 coordinates of a head's 256 weight rows (32 KB)
constexpr int kFmMaxStages = 6;
constexpr int kFmTile = 131072;              // one expanded tile of 128 positions
// smallest biased exponent of 32 positions' largest value: their exponent e
// stays in [-90, 113], so that 2^-e is a normal number, weights relative to
// the values' scale keep their range, and e fits a byte
constexpr int kFmMinExp = 51;
constexpr int kFmTail = kFmRows * 8 + 256;   // row scales and offsets, barriers, shared words

__host__ __device__ constexpr int fm_stages(int W) {
  const int n = (232448 - 1024 - (W / 64) * kFmABox - kFmTail) / kFmWStage;
  return n < kFmMaxStages ? n : kFmMaxStages;
}
__host__ __device__ constexpr int fm_smem(int W) {
  return 1024 + (W / 64) * kFmABox + fm_stages(W) * kFmWStage + kFmTail;
}
static_assert(fm_stages(512) >= 3, "weight stages");

__device__ __forceinline__ void fm_tma_load(void *dst, const CUtensorMap *tmap, int x, int y, uint64_t *bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(tmap)), "r"(x), "r"(y), "r"(smem_u32(bar))
      : "memory");
}
// the larger, NaN if either is
__device__ __forceinline__ float fmax_nan(float a, float b) {
  float r;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}

// Codes of chunk j (8 codes, layout.h) of 16 bytes of a quantised record.
template <int BITS>
__device__ __forceinline__ void fm_codes(const uint4 &q, int j, int (&u)[8]) {
  const uint32_t w4[4] = {q.x, q.y, q.z, q.w};
  if constexpr (BITS == 8) {
#pragma unroll
    for (int k = 0; k < 8; ++k) u[k] = (w4[2 * j + (k >> 2)] >> (8 * (k & 3))) & 255u;
  } else {
    const uint32_t w = BITS == 4 ? w4[j] : w4[j >> 1] >> (16 * (j & 1));
#pragma unroll
    for (int k = 0; k < 8; ++k) u[k] = (w >> mla_q_bit(k, BITS)) & ((1u << BITS) - 1u);
  }
}

// Column sums of the first W coordinates of every head's 256 weight rows
// (128 of W_UK, then 128 of W_UV): the offsets' factor for grouped codes.
__global__ void __launch_bounds__(256)
    mla_wsum_kernel(const uint16_t *w_uk, const uint16_t *w_uv, int r, int W, int n, float *wsum) {
  pdl_wait();
  pdl_trigger();
  const int row = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (row >= n) return;
  const int h = row >> 8, j = row & 255;
  const uint16_t *src = (j < 128 ? w_uk : w_uv) + ((size_t)h * 128 + (j & 127)) * r;
  float s = 0.f;
  for (int k = lane; k < W; k += 32) s += bf16_to_f32(src[k]);
#pragma unroll
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) wsum[row] = s;
}

// BITS 16: bf16 latents; 8, 4, 2: codes (a.v.scheme says which quantiser).
template <int BITS>
__global__ void __launch_bounds__(kFmThreads, 1)
    mla_form_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                    const MlaFormArgs a) {
  constexpr uint32_t kLimit = 1u << 20;  // polls of up to 2 us each
  extern __shared__ uint8_t fm_raw[];
  uint8_t *sm = fm_raw + ((1024u - (smem_u32(fm_raw) & 1023u)) & 1023u);
  const MlaView &v = a.v;
  const int W = v.width, boxes = W / 64, nst = fm_stages(W);
  uint8_t *wst = sm + boxes * kFmABox;
  float2 *rowm = reinterpret_cast<float2 *>(wst + nst * kFmWStage);  // (scale, centred offset) per row
  // barriers: wfull / wfree per weight stage, tfull / tfree per accumulator,
  // aready the block's latents staged, drain the products landed
  uint64_t *bar = reinterpret_cast<uint64_t *>(reinterpret_cast<uint8_t *>(rowm) + kFmRows * 8);
  uint64_t *wfull = bar, *wfree = bar + kFmMaxStages, *tfull = bar + 2 * kFmMaxStages, *tfree = tfull + 2,
           *aready = tfull + 4, *drain = tfull + 5;
  constexpr int kBars = 2 * kFmMaxStages + 6;
  static_assert(kBars * 8 + 32 <= 256, "barrier region");
  uint32_t *tbase = reinterpret_cast<uint32_t *>(bar + kBars);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(tbase + 1);
  int *s_run = reinterpret_cast<int *>(tbase + 2);  // first item, item count, its sequence and block
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  if (tid == 0) {
    for (int i = 0; i < kBars; ++i) mbar_init(&bar[i], &bar[i] == tfree || &bar[i] == tfree + 1 ? kFmEpi / 32 : 1);
    *abort_flag = 0;
    fence_mbar_init();
  }
  pdl_wait();  // the cache, its lengths and the weights' sums are complete
  if (warp == 8) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tbase)), "n"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (warp == 0) {
    // this CTA's run: the sequences' 128-position blocks, 32 sequences at a time
    int total = 0;
    for (int b0 = 0; b0 < a.nb; b0 += 32) {
      int n = b0 + lane < a.nb ? (v.lens[a.b0 + b0 + lane] + kFmRows - 1) / kFmRows : 0;
      for (int o = 16; o; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
      total += n;
    }
    const long long items = (long long)total * a.nh;
    const long long i0 = items * blockIdx.x / gridDim.x, i1 = items * (blockIdx.x + 1) / gridDim.x;
    const int blk = (int)(i0 / a.nh);
    int base = 0, fb = 0, ft = 0;
    for (int b0 = 0; b0 < a.nb; b0 += 32) {
      const int n = b0 + lane < a.nb ? (v.lens[a.b0 + b0 + lane] + kFmRows - 1) / kFmRows : 0;
      int inc = n;
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
      }
      const bool hit = blk >= base + inc - n && blk < base + inc;
      const uint32_t m = __ballot_sync(0xffffffffu, hit);
      if (m) {
        const int l = __ffs(m) - 1;
        fb = b0 + l;
        ft = blk - (base + __shfl_sync(0xffffffffu, inc - n, l));
        break;
      }
      base += __shfl_sync(0xffffffffu, inc, 31);
    }
    if (lane == 0) {
      s_run[0] = (int)(i0 - (long long)blk * a.nh);  // first head
      s_run[1] = (int)(i1 - i0);
      s_run[2] = fb;
      s_run[3] = ft;
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tbase;
  const int n_items = s_run[1];
  struct Cursor {
    int h, b, t;  // head (of the group), sequence (of the group), block
  } cur = {s_run[0], s_run[2], s_run[3]};
  // the next item: the next head, else the next block with positions; true
  // when the block changed
  auto advance = [&]() -> bool {
    if (++cur.h < a.nh) return false;
    cur.h = 0;
    ++cur.t;
    while (cur.b < a.nb && cur.t * kFmRows >= v.lens[a.b0 + cur.b]) {
      ++cur.b;
      cur.t = 0;
    }
    return true;
  };
  auto sleepy = [&](uint64_t *b, uint32_t parity) { return mbar_wait_sleepy(b, parity, kLimit, abort_flag, 2000); };

  if (warp == 9) {
    // ======================= weight copies ================================
    int c = 0;
    bool ok = true;
    if (lane == 0) {
      for (int i = 0; i < n_items && ok; ++i) {
        const int y = (a.h0 + cur.h) * 128;
        for (int k = 0; k < boxes && ok; ++k, ++c) {
          const int s = c % nst;
          if (c >= nst) ok = sleepy(&wfree[s], (c / nst - 1) & 1);
          if (ok) {
            mbar_expect_tx(&wfull[s], kFmWStage);
            fm_tma_load(wst + s * kFmWStage, &map_k, 64 * k, y, &wfull[s]);
            fm_tma_load(wst + s * kFmWStage + kFmWStage / 2, &map_v, 64 * k, y, &wfull[s]);
          }
        }
        advance();
      }
      if (!ok) {
        *abort_flag = 1;
        set_err(a.err, 8);
        --c;  // the chunk that was not issued
      }
      // the last copies land before the CTA leaves (bounded)
      for (int u = max(0, c - nst); u < c; ++u) mbar_wait(&wfull[u % nst], (u / nst) & 1, 1u << 22);
    }
    __syncwarp();
  } else if (warp == 8) {
    // ======================= products =====================================
    if (lane == 0) {
      constexpr uint32_t id = umma_idesc(128, 256, false, false);
      int c = 0, nblk = 0;
      bool ok = true, fresh = true;
      for (int i = 0; i < n_items && ok; ++i) {
        if (fresh) ok = sleepy(aready, nblk++ & 1);
        if (ok && i >= 2) ok = sleepy(&tfree[i & 1], ((i - 2) >> 1) & 1);
        tc_fence_after();
        for (int k = 0; k < boxes && ok; ++k, ++c) {
          const int s = c % nst;
          ok = sleepy(&wfull[s], (c / nst) & 1);
          if (!ok) break;
          tc_fence_after();
          const uint64_t da = umma_desc(smem_u32(sm + k * kFmABox), 16, 1024, 2);
          const uint64_t db = umma_desc(smem_u32(wst + s * kFmWStage), 16, 1024, 2);
#pragma unroll
          for (int ks = 0; ks < 4; ++ks)
            umma_f16(tmem + 256 * (i & 1), da + (uint64_t)(2 * ks), db + (uint64_t)(2 * ks), id, k > 0 || ks > 0);
          umma_commit(&wfree[s]);
        }
        if (ok) umma_commit(&tfull[i & 1]);
        fresh = advance();
      }
      if (!ok) {
        *abort_flag = 1;
        set_err(a.err, 8);
      }
      umma_commit(drain);  // every product lands before TMEM is released (bounded)
      mbar_wait(drain, 0, 1u << 22);
    }
    __syncwarp();
  } else {
    // ======================= staging and epilogue =========================
    // A warp that gives up goes on through the barriers and writes nothing.
    bool failed = false, fresh = true;
    const int quarter = warp & 3, half = warp >> 2;  // half 0: keys, 1: values
    const int row = 32 * quarter + lane;
    const uint32_t lane_off = (uint32_t)(32 * quarter) << 16;
    for (int i = 0; i < n_items; ++i) {
      const int b = a.b0 + cur.b, t0 = cur.t * kFmRows;
      const int len = v.lens[b];
      if (fresh) {
        // the products of the block before are done (this warp waited for
        // its last accumulator); the others' waits are met at the barrier
        asm volatile("bar.sync 1, %0;" ::"n"(kFmEpi) : "memory");
        const uint8_t *rec = v.rec + ((size_t)b * v.cap + t0) * v.rec_bytes;
        const int per = W / 8;
        if constexpr (BITS == 16) {
          for (int e = tid; e < kFmRows * per; e += kFmEpi) {
            const int r = e / per, c = e - r * per;
            const bool ok = t0 + r < len;
            cp_async16(sm + (c >> 3) * kFmABox + r * 128 + (((c & 7) ^ (r & 7)) << 4),
                       ok ? rec + (size_t)r * v.rec_bytes + 16 * c : rec, ok);
          }
          cp_async_commit();
          if (cur.h == 0)  // the block's positional keys, once per group of heads
            for (int e = tid; e < kFmRows * 8; e += kFmEpi) {
              const int r = e >> 3, c = e & 7;
              const uint4 x = t0 + r < len ? *reinterpret_cast<const uint4 *>(rec + (size_t)r * v.rec_bytes + 2 * W + 16 * c)
                                           : make_uint4(0, 0, 0, 0);
              *reinterpret_cast<uint4 *>(a.kr + ((size_t)cur.b * a.n_t + cur.t) * a.kr_bytes + r * 128 +
                                         ((c ^ (r & 7)) << 4)) = x;
            }
          cp_async_wait<0>();
        } else {
          const bool sym = v.scheme == kSchemeSym;
          const int C0 = sym ? (1 << (BITS - 1)) - 1 : 1 << (BITS - 1);
          // the record as 16-byte pieces of CH chunks (records, and the
          // latent's share of one, are whole pieces; a power of two of them)
          constexpr int CH = 16 / BITS, U = 4;
          const int sh = 31 - __clz(W * BITS / 128), pieces = kFmRows << sh;
          for (int e0 = tid; e0 < pieces; e0 += U * kFmEpi) {
            uint4 q[U];
#pragma unroll
            for (int i = 0; i < U; ++i) {  // U loads in flight
              const int e = e0 + i * kFmEpi, r = e >> sh, c = e & ((1 << sh) - 1);
              q[i] = e < pieces && t0 + r < len
                         ? *reinterpret_cast<const uint4 *>(rec + (size_t)r * v.rec_bytes + 16 * c)
                         : make_uint4(0, 0, 0, 0);
            }
#pragma unroll
            for (int i = 0; i < U; ++i) {
              const int e = e0 + i * kFmEpi, r = e >> sh, c16 = e & ((1 << sh) - 1);
              if (e >= pieces) break;
              const bool ok = t0 + r < len;
#pragma unroll
              for (int j = 0; j < CH; ++j) {
                int u[8];
                fm_codes<BITS>(q[i], j, u);
                uint32_t w[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) w[k] = ok ? pack_bf16((float)(u[2 * k] - C0), (float)(u[2 * k + 1] - C0)) : 0u;
                const int c = CH * c16 + j;
                *reinterpret_cast<uint4 *>(sm + (c >> 3) * kFmABox + r * 128 + (((c & 7) ^ (r & 7)) << 4)) =
                    make_uint4(w[0], w[1], w[2], w[3]);
              }
            }
          }
          if (cur.h == 0) {  // the block's positional keys, once per group of heads
            constexpr int RP = BITS / 2;  // 16-byte pieces of k^R (64 codes)
            for (int e = tid; e < kFmRows * RP; e += kFmEpi) {
              const int r = e / RP, c16 = e - r * RP;
              const bool ok = t0 + r < len;
              uint4 q = make_uint4(0, 0, 0, 0);
              float s = 0.f, z = 0.f;
              if (ok) {
                q = *reinterpret_cast<const uint4 *>(rec + (size_t)r * v.rec_bytes + W * BITS / 8 + 16 * c16);
                if (sym) {
                  s = __uint_as_float(reinterpret_cast<const uint32_t *>(v.meta)[(size_t)b * v.cap + t0 + r] & 0xFFFF0000u);
                  z = -(float)C0 * s;
                } else {
                  const float4 m = reinterpret_cast<const float4 *>(v.meta)[(size_t)b * v.cap + t0 + r];
                  s = m.z;
                  z = m.w;
                }
              }
#pragma unroll
              for (int j = 0; j < CH; ++j) {
                int u[8];
                fm_codes<BITS>(q, j, u);
                uint32_t w[4], lo[4];
#pragma unroll
                for (int k = 0; k < 4; ++k)
                  split2<true>(fmaf((float)u[2 * k], s, z), fmaf((float)u[2 * k + 1], s, z), w[k], lo[k]);
                uint8_t *dst = a.kr + ((size_t)cur.b * a.n_t + cur.t) * a.kr_bytes + r * 128 +
                               (((CH * c16 + j) ^ (r & 7)) << 4);
                *reinterpret_cast<uint4 *>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
                *reinterpret_cast<uint4 *>(dst + 16384) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
              }
            }
          }
          if (tid < kFmRows) {
            float2 m = make_float2(0.f, 0.f);
            if (t0 + tid < len) {
              if (sym) {
                m.x = __uint_as_float(reinterpret_cast<const uint32_t *>(v.meta)[(size_t)b * v.cap + t0 + tid] << 16);
              } else {
                const float4 q = reinterpret_cast<const float4 *>(v.meta)[(size_t)b * v.cap + t0 + tid];
                m = make_float2(q.x, fmaf((float)C0, q.x, q.y));
              }
            }
            rowm[tid] = m;
          }
        }
        fence_proxy_async();  // the staged latents are read by the products
        asm volatile("bar.sync 1, %0;" ::"n"(kFmEpi) : "memory");
        if (tid == 0) mbar_arrive(aready);
      }
      if (!failed) failed = !__all_sync(0xffffffffu, sleepy(&tfull[i & 1], (i >> 1) & 1));
      if (!failed) {
        tc_fence_after();
        float sc = 1.f, zc = 0.f;
        if constexpr (BITS != 16) {
          const float2 m = rowm[row];
          sc = m.x;
          zc = m.y;
        }
        const float *ws = BITS != 16 && v.scheme != kSchemeSym ? a.wsum + (a.h0 + cur.h) * 256 + 128 * half : nullptr;
        // keys: unit = 64 channels, 128 rows; values: unit = 64 positions, a
        // box of 64 rows per 64 channels; in both the lo half 16 KB on
        uint8_t *tile = a.tiles + (((size_t)cur.b * a.nh + cur.h) * a.n_t + cur.t) * kFmTile;
        uint8_t *dst = half ? tile + 65536 + (row >> 6) * 32768 + (row & 63) * 128 : tile + row * 128;
        const int box = half ? 8192 : 32768;
        // this row's channels c0 .. c0 + 31 as the products left them, and
        // with the row's scale and offset (times m) applied
        auto load = [&](int c0, float (&x)[32]) { tmem_ld32(tmem + 256 * (i & 1) + 128 * half + c0 + lane_off, x); };
        auto apply = [&](int c0, float (&x)[32], float m) {
          if (ws) {
            const float s = sc * m, z = zc * m;
#pragma unroll
            for (int k4 = 0; k4 < 8; ++k4) {
              const float4 w = *reinterpret_cast<const float4 *>(ws + c0 + 4 * k4);
              x[4 * k4] = fmaf(x[4 * k4], s, z * w.x);
              x[4 * k4 + 1] = fmaf(x[4 * k4 + 1], s, z * w.y);
              x[4 * k4 + 2] = fmaf(x[4 * k4 + 2], s, z * w.z);
              x[4 * k4 + 3] = fmaf(x[4 * k4 + 3], s, z * w.w);
            }
          } else {
            const float s = sc * m;
#pragma unroll
            for (int k = 0; k < 32; ++k) x[k] *= s;
          }
        };
        auto store = [&](int c0, const uint32_t (&hw)[16], const uint32_t (&lw)[16]) {
#pragma unroll
          for (int p = 0; p < 2; ++p) {
            const int j = c0 / 16 + p;  // pair of 8-channel chunks
            const uint32_t *h = hw + 8 * p, *l = lw + 8 * p;
            const uint4 h0 = make_uint4(h[0], h[1], h[2], h[3]), h1 = make_uint4(h[4], h[5], h[6], h[7]);
            const uint4 l0 = make_uint4(l[0], l[1], l[2], l[3]), l1 = make_uint4(l[4], l[5], l[6], l[7]);
            uint8_t *q = dst + (j >> 2) * box + (((2 * (j & 3)) ^ (row & 6)) << 4);
            const bool odd = row & 1;
            st_sector(q, odd ? h1 : h0, odd ? h0 : h1);
            st_sector(q + 16384, odd ? l1 : l0, odd ? l0 : l1);
          }
        };
        if (!half) {
#pragma unroll
          for (int c0 = 0; c0 < 128; c0 += 32) {
            float x[32];
            uint32_t hw[16], lw[16];
            load(c0, x);
            if constexpr (BITS != 16) apply(c0, x, 1.f);
#pragma unroll
            for (int k = 0; k < 16; ++k) split2<true>(x[2 * k], x[2 * k + 1], hw[k], lw[k]);
            store(c0, hw, lw);
          }
        } else {
          // the largest value of the warp's 32 positions (grouped codes: a
          // bound on it) gives their exponent, it becomes 2^14 .. 2^15 at
          // most; NaN and infinities stick to the maximum
          float top = 0.f;
#pragma unroll 1
          for (int c0 = 0; c0 < 128; c0 += 32) {
            float x[32];
            load(c0, x);
#pragma unroll
            for (int k = 0; k < 32; ++k) top = fmax_nan(top, fabsf(x[k]));
          }
          if constexpr (BITS != 16) {
            top *= fabsf(sc);
            if (ws) {
              const float4 w = *reinterpret_cast<const float4 *>(ws + 4 * lane);
              const float wm = fmax_nan(fmax_nan(fabsf(w.x), fabsf(w.y)), fmax_nan(fabsf(w.z), fabsf(w.w)));
              top = fmaf(fabsf(zc), __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(wm))), top);
            }
          }
          const bool odd_row = !(top < INFINITY);  // a value (or the bound) is not finite
          if (__any_sync(0xffffffffu, odd_row)) {
            if (odd_row) top = 0.f;
#pragma unroll 1
            for (int c0 = 0; c0 < 128; c0 += 32) {
              float x[32];
              load(c0, x);
              if (odd_row) {
                apply(c0, x, 1.f);
                int *bad = a.bad + ((size_t)cur.b * a.nh + cur.h) * kPfBadStride;
                const int at = (int)v.cap - (t0 + row);
#pragma unroll
                for (int k = 0; k < 32; ++k) {
                  if (fabsf(x[k]) < INFINITY) {
                    top = fmaxf(top, fabsf(x[k]));
                  } else {
                    atomicMax(bad + c0 + k, at);
                    atomicMax(bad + 128, at);
                  }
                }
              }
              __syncwarp();  // the TMEM loads are warp-wide
            }
          }
          const uint32_t tb = __reduce_max_sync(0xffffffffu, __float_as_uint(top)) >> 23;
          const int e = max((int)tb, kFmMinExp) - 141;
          const float down = __uint_as_float((uint32_t)(127 - e) << 23);  // 2^-e
          if (lane == 0)
            reinterpret_cast<int8_t *>(a.vexp)[4 * (((size_t)cur.b * a.nh + cur.h) * a.n_t + cur.t) + quarter] = (int8_t)e;
#pragma unroll
          for (int c0 = 0; c0 < 128; c0 += 32) {
            float x[32];
            uint32_t hw[16], lw[16];
            load(c0, x);
            apply(c0, x, down);
            if (odd_row) {
#pragma unroll
              for (int k = 0; k < 32; ++k)
                if (!(fabsf(x[k]) < INFINITY)) x[k] = 0.f;
            }
            __syncwarp();
#pragma unroll
            for (int k = 0; k < 16; ++k) split2<false>(x[2 * k], x[2 * k + 1], hw[k], lw[k]);
            store(c0, hw, lw);
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&tfree[i & 1]);
      } else {
        *abort_flag = 1;
      }
      fresh = advance();
    }
    if (failed && lane == 0) set_err(a.err, 8);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 8)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(512) : "memory");
  pdl_trigger();
}

template <int BITS>
cudaError_t launch_form_t(const MlaFormArgs &a, const CUtensorMap &mk, const CUtensorMap &mv, int grid,
                          cudaStream_t st) {
  const int smem = fm_smem(a.v.width);
  cudaError_t e = cudaFuncSetAttribute(mla_form_kernel<BITS>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(mla_form_kernel<BITS>, dim3(grid), dim3(kFmThreads), smem, st, mk, mv, a);
}

}  // namespace

cudaError_t launch_mla_wsum(const void *w_uk, const void *w_uv, int H, int r, int W, float *wsum, cudaStream_t st) {
  return launch_pdl(mla_wsum_kernel, dim3(H * 32), dim3(256), 0, st, static_cast<const uint16_t *>(w_uk),
                    static_cast<const uint16_t *>(w_uv), r, W, H * 256, wsum);
}

cudaError_t launch_mla_form(const MlaFormArgs &a, const void *w_uk, const void *w_uv, int H, int r, int sms,
                            cudaStream_t st) {
  // the weights as 2-D tensors [H 128 rows x r], boxes of 64 coordinates x
  // 128 rows in the operand layout
  CUtensorMap m[2];
  const void *w[2] = {w_uk, w_uv};
  for (int i = 0; i < 2; ++i) {
    const uint64_t dims[2] = {(uint64_t)r, (uint64_t)H * 128};
    const uint64_t strides[1] = {(uint64_t)r * 2};
    const uint32_t box[2] = {64, 128};
    const uint32_t estr[2] = {1, 1};
    const cudaError_t e = encode_tensor_map_tiled(&m[i], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(w[i]),
                                                  dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                                                  CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                                                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (e != cudaSuccess) return e;
  }
  const long long blocks = (long long)a.nb * ((a.v.cap + kFmRows - 1) / kFmRows);
  const int grid = (int)std::max(1LL, std::min<long long>(sms, blocks * a.nh));
  switch (a.v.bits) {
    case 16: return launch_form_t<16>(a, m[0], m[1], grid, st);
    case 8: return launch_form_t<8>(a, m[0], m[1], grid, st);
    case 4: return launch_form_t<4>(a, m[0], m[1], grid, st);
    default: return launch_form_t<2>(a, m[0], m[1], grid, st);
  }
}

}  // namespace kvk
