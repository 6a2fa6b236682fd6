// prefill.cu -- causal chunk attention over a compressed GQA cache
// (head_dim 128) on the tensor cores: the queries of each sequence's last n_q
// positions attend to the dequantised cache up to their own position (the
// pre-fill the paper times over compressed caches, Sec. 4; the chunk's keys
// and values are written with kvk_append first, so the chunk reads the same
// stored keys and values the decode steps then read).
//
// Rows: row r = i G + h of a (sequence, KV head) unit is chunk query i and
// head h of the KV head's group; query i sits at position len - n_q + i and
// sees positions 0 .. len - n_q + i.  A job is 128 consecutive rows of one
// unit.  Two launches:
//  * expand: the cache is dequantised once into the layout the products read
//    (bf16 hi and lo halves, 128-byte-swizzled boxes of 64 channels), in
//    caller scratch, tiles of 128 positions;
//  * attention, one pass over the tiles: per tile, S = Q K^T (TMEM lane =
//    row) with x = sigma log2(e) <q, k>; each row's maximum over the tile
//    (its four slices' maxima through shared memory) against the row's
//    reference m, which moves only when a score rises more than 8 above it
//    (O and the row's sums then rescaled by 2^(m_old - m_new) in place);
//    P = 2^(x - m) (zero past the row's limit, at most 2^8) as bf16 hi and
//    lo pairs into TMEM in place of the scores, O += P V (P the A operand
//    from TMEM, the values an MN-major B operand); after the job's last tile
//    O (TMEM lane = row) is divided by the row's sum of P and written out.
// The attention kernel runs one persistent CTA per SM: two copy warps bring
// each job's keys and values in with bulk copies, one MMA warp issues the
// score products and one the value products, 16 worker warps stage the query
// rows and run the epilogues.  Products are hi*hi + hi*lo + lo*hi (no lo
// part for bf16 caches or bf16 queries), fp32 accumulation in TMEM.  Jobs
// are handed out from a counter in bands of units whose tiles stay in L2,
// the longest row blocks first.
//
// A position that a row does not see has weight 0 in its products, and 0
// times an infinite or NaN value is NaN: such values enter the tiles as 0,
// and each unit records, per channel, the first position that has one
// (PfArgs::bad).  A row that sees it gets NaN in that channel, the others
// do not depend on it.
//
// Why tiles of 128 positions: a score product of N = 64 with its A operand
// in TMEM took 77-90 cycles (a clock64 trace of the 64-position version: 16
// of them 1450 cycles, 12 value products 800 alone) against 64 for N = 128,
// and the two products of a tile then cost 2560 cycles per 128 positions
// (16 + 24 at 64).  Measured: about 3400 cycles per 128 positions, the chain
// of a tile's scores, epilogue (about 1500) and values with two tiles in
// flight; the 64-position version took 2.33 ms, this one then 2.12
// (14B int4 layer, 4 x 8192 positions, the last 2048 the chunk).  The chain's
// share of the epilogue: packed binary32 arithmetic (2025 -> 1995 us, repeated
// calls) and 104 registers for the workers (-> 1946 us); the first unit's
// weights computed before the row's barrier instead, with the reference as it
// stands, was slower (1985 us).
//
// MLA chunks run the same attention kernel over keys and values formed per
// head (mla_form.cu): units are heads (G = 1), and the score products go on
// over the 64 positional channels, whose keys (one tile per sequence, shared
// by the heads) come through a ring of their own.  Their query rows sit in
// shared memory and the freed TMEM columns hold a second accumulator, for
// the products with a lo half: a tensor-core accumulation rounds towards
// zero, so each one costs its accumulator about 2^-25 of its value in one
// direction, and three per k-step into one accumulator left 1.3e-5 of the
// result over 3584 positions where the absorbed path has 5.6e-6 (the lo
// products' own sum is 2^-11 of the result).  One per k-step still costs
// 1e-6 of the result per 1000 positions, so O is added to the row's partial
// result in the output, in binary32, after every 16 tiles over 4-bit latents
// and 32 over others, whose absorbed forms have 2.8e-6 and 3.5e-6 or more.
#include <math.h>

#include <algorithm>

#include "common.cuh"
#include "kernels.h"
#include "layout.h"
#include "umma.cuh"
#include "window_tc.cuh"

namespace kvk {
namespace {

constexpr int kPfWorkers = 512;
constexpr int kPfThreads = kPfWorkers + 128;  // + two MMA warps and two copy warps
constexpr int kPfRows = 128;                 // rows per job
constexpr int kPfT = 128;                    // positions per tile
constexpr int kPfBox = 64 * 128;             // 64 channels x 64 positions (8 KB)
constexpr int kPfMaxStages = 8;              // key (and value) units at most
constexpr int kPfBarBytes = 448;             // barriers and the CTA's shared words

// A tile in scratch: two key units, one per 64 channels ([hi | lo], 128
// positions x 128 bytes each), then two value units, one per 64 positions
// ([hi | lo], two boxes of 64 channels each); no lo halves for bf16 caches.
struct PfPlan {
  int n_rb, n_jobs, grid, n_t;  // n_t: tiles per unit in scratch
  int q_lo, k_lo, fmt, gshift;
  int kpc;            // keys with per-channel groups (codes + group plane + residual)
  int ks16, nrec;
  uint32_t nc_magic;  // expand: ceil(2^32 / nrec), e / nrec = umulhi(e, nc_magic)
  int b_stride;       // expand: staged record stride (odd multiple of 16 bytes)
  int ub, tbytes;     // a unit; the whole tile (two key and two value units)
  int krb;            // positional keys of a tile (MLA; else 0)
  int flush;          // tiles that an MLA job sums in TMEM before O is added to its output
  int nk, nv, nr;     // key and value units and positional tiles in shared memory
  int band;           // units per band of the job order
  int off_v, off_r, off_q, off_red, off_bar, smem, smem_x;  // key units at offset 0
};

// A place in a ring of n units and the parity of its current round (units
// are counted without dividing: a division takes a lone thread hundreds of
// cycles).  A full barrier is awaited at parity `ph`, a free one at ph ^ 1
// (which holds at once in the first round).
struct PfRing {
  int s = 0;
  uint32_t ph = 0;
  __device__ __forceinline__ void next(int n) {
    if (++s == n) {
      s = 0;
      ph ^= 1;
    }
  }
};

// Tiles a job reads: positions up to that of the job's last row.
__device__ __forceinline__ int pf_tiles(int len, int n_q, int G, int r_last) {
  const int p_max = len - n_q + r_last / G;
  return p_max >= 0 ? p_max / kPfT + 1 : 0;
}

// The non-finite halves of 8 bf16 values (channels ch.. of position t) set to
// zero and recorded in `bad` (null: already recorded with their hi parts).
__device__ __noinline__ uint4 pf_scrub(uint4 u, int *bad, int ch, int cap_t) {
  uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if ((w[i] >> (16 * h) & 0x7F80u) == 0x7F80u) {
        w[i] &= h ? 0xFFFFu : 0xFFFF0000u;
        if (bad) {
          atomicMax(bad + ch + 2 * i + h, cap_t);
          atomicMax(bad + 128, cap_t);
        }
      }
  return make_uint4(w[0], w[1], w[2], w[3]);
}
__device__ __forceinline__ bool pf_finite(uint4 u) {
  // an exponent of all ones carries out of its half's top bit
  auto ok = [](uint32_t w) { return (((w & 0x7F807F80u) + 0x00800080u) & 0x80008000u) == 0; };
  return ok(u.x) && ok(u.y) && ok(u.z) && ok(u.w);
}

// Expand: the keys and values of 64 positions (half a tile) of one unit,
// staged raw (rotations undone), dequantised per (position, channel quarter)
// into [K hi | K lo | V hi | V lo] (8 KB boxes; no lo halves for bf16
// caches) and stored in the tile's units for every job of the unit to copy.
// Positions past the length are zero, to the end of the last tile.
__global__ void __launch_bounds__(kPfWorkers) prefill_expand_kernel(const PfArgs a, const PfPlan p) {
  extern __shared__ uint8_t pf_raw[];
  uint8_t *sm = pf_raw + ((1024u - (smem_u32(pf_raw) & 1023u)) & 1023u);
  const GqaView &v = a.v;
  constexpr int T = 64;
  const int unit = blockIdx.y, tid = threadIdx.x;
  pdl_wait();
  const int len = v.lens[unit / v.Hkv];
  const int t0 = blockIdx.x * T;
  if (t0 >= (len + kPfT - 1) / kPfT * kPfT) {
    pdl_trigger();
    return;
  }
  const int kbytes = p.ub;  // 64 positions of both key units
  uint8_t *stg = sm + 2 * kbytes;
  const uint8_t *base = v.rec + (size_t)unit * v.cap * v.rec_bytes;
  const bool sym = p.fmt >= kFmtS8, bf = p.fmt == kFmtBf16;
  for (int e = tid; e < T * p.nrec; e += kPfWorkers) {
    const int pos = (int)__umulhi((uint32_t)e, p.nc_magic), c = e - pos * p.nrec;
    const int t = t0 + pos;
    const bool ok = t < len;
    int so;
    if (sym)
      so = (c + sym_rot(t, p.nrec)) & (p.nrec - 1);
    else if (!bf && c >= p.ks16 && c < 2 * p.ks16)
      so = p.ks16 + ((c - p.ks16 + v_rot(t, v.rec_bytes, p.ks16)) & (p.ks16 - 1));
    else
      so = c;
    cp_async16(stg + pos * p.b_stride + 16 * c, base + (size_t)(ok ? t : 0) * v.rec_bytes + 16 * so, ok);
  }
  if (sym)
    for (int pos = tid; pos < T; pos += kPfWorkers) {
      const int t = t0 + pos;
      const bool ok = t < len;
      cp_async4(stg + pos * p.b_stride + v.rec_bytes, v.scales + (size_t)unit * v.cap + (ok ? t : 0), ok);
    }
  // per-channel keys: the (scale, zero) rows of the tile's complete groups
  // of positions (T >> gshift groups of 128 channels; rows of the open
  // group are zero and unused: those positions come from the residual)
  const int g0 = t0 >> p.gshift, full = (len >> p.gshift) << p.gshift;
  float2 *mrows = reinterpret_cast<float2 *>(stg + T * p.b_stride);
  if (p.kpc) {
    const int ng = T >> p.gshift;
    for (int i = tid; i < ng * 128 * 8 / 16; i += kPfWorkers) {
      const int gi = i / 64, c = i - gi * 64;  // 64 chunks of 16 bytes per row
      const bool ok = ((g0 + gi) << p.gshift) < full;
      const float2 *src = v.gmeta + ((size_t)unit * (v.cap >> p.gshift) + (ok ? g0 + gi : 0)) * 128;
      cp_async16(reinterpret_cast<uint8_t *>(mrows) + 16 * i, reinterpret_cast<const uint8_t *>(src) + 16 * c, ok);
    }
  }
  cp_async_commit();
  cp_async_wait<0>();
  __syncthreads();
  // threads [0, 256): key quarters; [256, 512): value quarters
  const int pidx = tid & (T - 1), part = tid / T;
  const uint8_t *bundle = stg + pidx * p.b_stride;
  const int ks = 16 * p.ks16;
  const int mb = (p.nrec * 16 - 2 * ks) / 2;  // grouped: one metadata block
  uint8_t *kh = sm, *kl = sm + 2 * kPfBox;
  if (part < 4 && p.kpc) {
    // per-channel keys: complete groups from codes and the group rows, the
    // open group from the bf16 residual (row t mod g), zero past the length
    const int t = t0 + pidx;
    if (t < full) {
      const float2 *mr = mrows + ((t >> p.gshift) - g0) * 128;
      if (p.fmt == kFmtG8)
        tc_dequant_kpc<8, kPfBox>(bundle, mr, pidx, part, kh, kl);
      else
        tc_dequant_kpc<4, kPfBox>(bundle, mr, pidx, part, kh, kl);
    } else {
      const uint4 z = make_uint4(0, 0, 0, 0);
      if (t < len) {
        const uint8_t *res = v.resid + ((size_t)unit * ((size_t)1 << p.gshift) + (t & ((1 << p.gshift) - 1))) * 256;
        tc_dequant<kFmtBf16, kPfBox>(res, nullptr, pidx, part, p.gshift, kh, kl);
      } else {
#pragma unroll
        for (int cc = 0; cc < 4; ++cc) put_chunk(kh, pidx, 32 * part + 8 * cc, kPfBox, z);
      }
#pragma unroll
      for (int cc = 0; cc < 4; ++cc) put_chunk(kl, pidx, 32 * part + 8 * cc, kPfBox, z);
    }
  } else if (part < 4) {
    const uint8_t *kmeta = sym ? bundle + v.rec_bytes : bundle + 2 * ks;
    switch (p.fmt) {
      case kFmtBf16: tc_dequant<kFmtBf16, kPfBox>(bundle, kmeta, pidx, part, p.gshift, kh, kl); break;
      case kFmtG8: tc_dequant<kFmtG8, kPfBox>(bundle, kmeta, pidx, part, p.gshift, kh, kl); break;
      case kFmtG4: tc_dequant<kFmtG4, kPfBox>(bundle, kmeta, pidx, part, p.gshift, kh, kl); break;
      case kFmtS8: tc_dequant<kFmtS8, kPfBox>(bundle, kmeta, pidx, part, p.gshift, kh, kl); break;
      case kFmtS4: tc_dequant<kFmtS4, kPfBox>(bundle, kmeta, pidx, part, p.gshift, kh, kl); break;
      default: tc_dequant<kFmtS2, kPfBox>(bundle, kmeta, pidx, part, p.gshift, kh, kl); break;
    }
  } else {
    const int qc = part - 4;
    uint8_t *vh = sm + kbytes, *vl = vh + 2 * kPfBox;
    const uint8_t *vsec = bundle + ks, *vmeta = bundle + 2 * ks + (p.kpc ? 0 : mb);
    const float svs =
        sym ? __uint_as_float(*reinterpret_cast<const uint32_t *>(bundle + v.rec_bytes) & 0xFFFF0000u) : 0.f;
    switch (p.fmt) {
      case kFmtBf16: tc_dequant_v<kFmtBf16, kPfBox>(vsec, vmeta, svs, pidx, qc, p.gshift, vh, vl); break;
      case kFmtG8: tc_dequant_v<kFmtG8, kPfBox>(vsec, vmeta, svs, pidx, qc, p.gshift, vh, vl); break;
      case kFmtG4: tc_dequant_v<kFmtG4, kPfBox>(vsec, vmeta, svs, pidx, qc, p.gshift, vh, vl); break;
      case kFmtS8: tc_dequant_v<kFmtS8, kPfBox>(vsec, vmeta, svs, pidx, qc, p.gshift, vh, vl); break;
      case kFmtS4: tc_dequant_v<kFmtS4, kPfBox>(vsec, vmeta, svs, pidx, qc, p.gshift, vh, vl); break;
      default: tc_dequant_v<kFmtS2, kPfBox>(vsec, vmeta, svs, pidx, qc, p.gshift, vh, vl); break;
    }
  }
  __syncthreads();
  // shared: keys [hi box 0 | hi box 1 | lo box 0 | lo box 1], then values the
  // same; key box b goes to unit b, half (hi, lo) h, rows 64 (half tile) on
  uint8_t *dst = a.tiles + ((size_t)unit * p.n_t + (blockIdx.x >> 1)) * p.tbytes;
  const int hf = blockIdx.x & 1;
  constexpr int B16 = kPfBox / 16;
  const uint4 *src = reinterpret_cast<const uint4 *>(sm);
  for (int i = tid; i < kbytes / 16; i += kPfWorkers) {
    const int x = i / B16, b = x & 1, h = x >> 1;
    reinterpret_cast<uint4 *>(dst + b * p.ub + h * 2 * kPfBox + hf * kPfBox)[i - x * B16] = src[i];
  }
  uint4 *dv = reinterpret_cast<uint4 *>(dst + (2 + hf) * p.ub);
  for (int i = tid; i < p.ub / 16; i += kPfWorkers) {
    uint4 u = src[kbytes / 16 + i];
    if (!pf_finite(u)) {
      const int x = i / B16, row = i >> 3 & 63, ch = 64 * (x & 1) + 8 * ((i & 7) ^ (row & 7));
      u = pf_scrub(u, x < 2 ? a.bad + (size_t)unit * kPfBadStride : nullptr, ch, (int)v.cap - (t0 + row));
    }
    dv[i] = u;
  }
  pdl_trigger();
}

// S (+)= Q K^T of one key unit (64 channels) into TMEM columns d0.., 128
// positions: Q (bf16 pairs) from TMEM at t_q, its lo halves 64 columns on;
// the keys (hi, then lo 16 KB on) K-major in shared memory at k.
template <bool KLO, bool QLO>
__device__ __forceinline__ void pf_issue_scores(uint32_t d0, uint32_t t_q, uint32_t k, bool acc) {
  constexpr uint32_t id = umma_idesc(128, kPfT, false, false);
  constexpr uint32_t hi = umma_desc_hi_sw128(1024);
  const uint32_t lo_h = umma_desc_lo(k, 16), lo_l = lo_h + (2 * kPfBox >> 4);
#pragma unroll
  for (int ks = 0; ks < 4; ++ks) {
    umma_f16_ts_w(d0, t_q + 8 * ks, lo_h + 2 * ks, hi, id, acc || ks > 0);
    if (KLO) umma_f16_ts_w(d0, t_q + 8 * ks, lo_l + 2 * ks, hi, id, true);
    if (QLO) umma_f16_ts_w(d0, t_q + 64 + 8 * ks, lo_h + 2 * ks, hi, id, true);
  }
}
// The same with Q's 64 channels K-major in shared memory at q (128 rows).
template <bool KLO>
__device__ __forceinline__ void pf_issue_scores_ss(uint32_t d0, uint32_t q, uint32_t k, bool acc) {
  constexpr uint32_t id = umma_idesc(128, kPfT, false, false);
  const uint64_t da = umma_desc(q, 16, 1024, 2), dh = umma_desc(k, 16, 1024, 2);
#pragma unroll
  for (int ks = 0; ks < 4; ++ks) {
    umma_f16(d0, da + (uint64_t)(2 * ks), dh + (uint64_t)(2 * ks), id, acc || ks > 0);
    if (KLO) umma_f16(d0, da + (uint64_t)(2 * ks), dh + (uint64_t)((2 * kPfBox >> 4) + 2 * ks), id, true);
  }
}
// O += P V of one value unit (64 positions): P (bf16 pairs, hi then lo 64
// columns on) from TMEM at pa, the values (hi, then lo 2 boxes on) MN-major
// in shared memory at vh (64-channel boxes kPfBox apart), 16 positions per
// k-step; the products with a lo half into t_ol (t_o unless it is another:
// SPLIT, whose halves are f16, and which starts anew unless acc_l).
template <bool KLO, bool SPLIT>
__device__ __forceinline__ void pf_issue_values(uint32_t t_o, uint32_t t_ol, uint32_t pa, uint32_t vh, bool acc,
                                                bool acc_l) {
  constexpr uint32_t id = SPLIT ? umma_idesc_f16(128, 128, false, true) : umma_idesc(128, 128, false, true);
  constexpr uint32_t hi = umma_desc_hi_sw128(1024);
  const uint32_t lo_h = umma_desc_lo(vh, kPfBox), lo_l = lo_h + (2 * kPfBox >> 4);
#pragma unroll
  for (int ks = 0; ks < 4; ++ks) {
    umma_f16_ts_w(t_o, pa + 8 * ks, lo_h + 128 * ks, hi, id, acc || ks > 0);
    if (KLO) umma_f16_ts_w(t_ol, pa + 8 * ks, lo_l + 128 * ks, hi, id, !SPLIT || acc_l || ks > 0);
    umma_f16_ts_w(t_ol, pa + 64 + 8 * ks, lo_h + 128 * ks, hi, id, true);
  }
}

template <bool MLA>
__global__ void __launch_bounds__(kPfThreads, 1) prefill_kernel(const PfArgs a, const PfPlan p) {
  constexpr int D = 128;
  constexpr uint32_t kLimit = 1u << 20;  // polls of up to 2 us each
  constexpr uint32_t kSpins = 1u << 26;  // polls of tens of cycles
  extern __shared__ uint8_t pf_raw[];
  uint8_t *sm = pf_raw + ((1024u - (smem_u32(pf_raw) & 1023u)) & 1023u);
  // barriers: kfull[8] keys of a unit landed, kfree[8] its score products
  // done, vfull[8] / vfree[8] the same for values, rfull[2] / rfree[2] for
  // the positional keys; per tile parity: sdone[2] scores done, epi[2][2] the
  // workers' P of either value unit's positions written (16 arrivals),
  // pvdone[2] value products done;
  // qready the job's query rows staged (16 arrivals), drain[2] (one per MMA
  // warp).  A barrier per parity completes every other tile, and the next
  // completion of one always depends on the wait for its previous one, so
  // no wait can fall two phases behind.
  uint64_t *bar = reinterpret_cast<uint64_t *>(sm + p.off_bar);
  constexpr int S8 = kPfMaxStages;
  uint64_t *kfull = bar, *kfree = bar + S8, *vfull = bar + 2 * S8, *vfree = bar + 3 * S8;
  uint64_t *rfull = bar + 4 * S8, *rfree = rfull + 2;
  uint64_t *sdone = rfree + 2, *epi = sdone + 2, *pvdone = epi + 4, *qready = pvdone + 2, *drain = qready + 1;
  constexpr int kBars = 4 * S8 + 4 + 11;
  static_assert(kBars * 8 + 12 <= kPfBarBytes, "barrier region");
  uint32_t *tbase = reinterpret_cast<uint32_t *>(sm + p.off_bar + kBars * 8);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(sm + p.off_bar + kBars * 8 + 4);
  volatile int *s_job = reinterpret_cast<volatile int *>(sm + p.off_bar + kBars * 8 + 8);
  const GqaView &v = a.v;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int R = a.n_q * a.G;
  const int quarter = warp & 3, slice = warp >> 2;
  const uint32_t lane_off = (uint32_t)(quarter * 32) << 16;
  const float sg = a.sig_log2;

  if (tid == 0) {
    for (int i = 0; i < kBars; ++i) {
      uint64_t *b = &bar[i];
      mbar_init(b, ((b >= epi && b < epi + 4) || b == qready) ? kPfWorkers / 32 : 1);
    }
    *abort_flag = 0;
    fence_mbar_init();
  }
  pdl_wait();  // the tiles, lengths and records of non-finite values are complete
  constexpr uint32_t kCols = 512;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tbase)),
                 "n"(kCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tbase;
  // TMEM columns (lane = the job's row in every region): scores of tile k
  // at 128 (k & 1), fp32, and in their place, once they are read, the tile's
  // P (bf16 pairs, hi 64 columns, then lo), the A operand of the value
  // products; O at 256 (fp32, 128 channels); at 384 the job's query rows as
  // bf16 pairs (hi 64 columns, then lo), the A operand of the score products,
  // or (MLA) the sum of the value products with a lo half.
  const uint32_t t_o = tmem + 256, t_ol = MLA ? tmem + 384 : t_o;
  const uint32_t t_q = tmem + 384;
  auto t_s = [&](int k) { return tmem + 128u * (k & 1); };

  // Jobs are handed out one at a time from a counter, so CTAs finish
  // together although jobs differ in length.  Order: bands of p.band units
  // (whose tiles the band's jobs share in L2), in each band the longest row
  // blocks first.
  // Every thread of the CTA takes part in each hand-out; a role that gave up
  // keeps taking jobs (and skips them) until none is left, so no barrier
  // waits for threads that left.
  const int units = v.B * v.Hkv;
  int *counter = a.counter;
  auto next_job = [&]() -> int {
    asm volatile("bar.sync 2, %0;" ::"n"(kPfThreads) : "memory");  // the previous id is read
    if (tid == 0) *s_job = atomicAdd(counter, 1);
    asm volatile("bar.sync 2, %0;" ::"n"(kPfThreads) : "memory");
    return *s_job;
  };
  struct Job {
    int unit, b, j, r0, nr, len, n_t;
  };
  auto job_at = [&](int job) {
    Job J;
    const int per = p.band * p.n_rb;
    const int g = job / per, w = job - g * per;
    const int ub = min(p.band, units - g * p.band);  // units in this band
    const int step = w / ub;
    J.unit = g * p.band + (w - step * ub);
    const int rb = p.n_rb - 1 - step;
    J.b = J.unit / v.Hkv;
    J.j = J.unit - J.b * v.Hkv;
    if constexpr (MLA) {
      J.b += a.b0;
      J.j += a.h0;
    }
    J.r0 = rb * kPfRows;
    J.nr = min(kPfRows, R - J.r0);
    J.len = v.lens[J.b];
    J.n_t = pf_tiles(J.len, a.n_q, a.G, J.r0 + J.nr - 1);
    return J;
  };
  auto sleepy = [&](uint64_t *b, uint32_t parity) {
    return mbar_wait_sleepy(b, parity, kLimit, abort_flag, 2000);
  };
  auto spin = [&](uint64_t *b, uint32_t parity) { return mbar_spin_or_abort(b, parity, kSpins, abort_flag); };

  // Registers by warpgroup, 512 x 104 + 128 x 64 = the 640 x 96 launched: the
  // workers hold 32 scores, their weights and both halves without spills
  // (each set inside its branch: ahead of the branches the workers spilled).
  static_assert(kPfRegs.threads[0] == kPfWorkers && kPfRegs.all_threads() == kPfThreads && kPfRegs.fits(96),
                "the register split");
  if (warp >= kPfWorkers / 32) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kPfRegs.regs[1]) : "memory");
    if (warp == kPfWorkers / 32 + 1 || warp == kPfWorkers / 32 + 3) {
      // ======================= copy warps ===================================
      // lane 0 of one copies each tile's key units (and positional keys), of
      // the other its value units, once the products that read the unit's
      // place before are done
      const bool keys = warp == kPfWorkers / 32 + 1;
      uint64_t *full = keys ? kfull : vfull, *free_ = keys ? kfree : vfree;
      const int n = keys ? p.nk : p.nv;
      uint8_t *ring = sm + (keys ? 0 : p.off_v);
      int c = 0, rc = 0;  // units (and positional tiles) copied
      PfRing ru, rr;
      bool ok = true;
      for (int job = next_job(); job < p.n_jobs; job = next_job()) {
        if (ok && lane == 0) {
          const Job J = job_at(job);
          const uint8_t *src = a.tiles + (size_t)J.unit * p.n_t * p.tbytes + (keys ? 0 : 2 * p.ub);
          for (int k = 0; k < J.n_t && ok; ++k) {
            for (int u = 0; u < 2 && ok; ++u) {
              const int s = ru.s;
              ok = sleepy(&free_[s], ru.ph ^ 1);
              // the unit's place is written only by bulk copies and read only
              // by the products (both async proxy, ordered by the commit's
              // release of kfree / vfree): no proxy fence
              if (ok) {
                mbar_expect_tx(&full[s], p.ub);
                bulk_g2s(ring + s * p.ub, src + (size_t)k * p.tbytes + u * p.ub, p.ub, &full[s]);
                ++c;
                ru.next(n);
              }
            }
            if (MLA && keys && ok) {
              const int s = rr.s;
              ok = sleepy(&rfree[s], rr.ph ^ 1);
              if (ok) {
                mbar_expect_tx(&rfull[s], p.krb);
                bulk_g2s(sm + p.off_r + s * p.krb, a.kr + ((size_t)(J.b - a.b0) * p.n_t + k) * p.krb, p.krb, &rfull[s]);
                ++rc;
                rr.next(p.nr);
              }
            }
          }
          if (!ok) *abort_flag = 1;
        }
        ok = __shfl_sync(0xffffffffu, ok, 0);
      }
      // the last copies land before the CTA leaves (bounded; at once when
      // they were consumed)
      if (lane == 0) {
        for (int u = max(0, c - n); u < c; ++u) mbar_wait(&full[u % n], (u / n) & 1, 1u << 22);
        for (int u = max(0, rc - p.nr); u < rc; ++u) mbar_wait(&rfull[u % p.nr], (u / p.nr) & 1, 1u << 22);
      }
      __syncwarp();
    } else {
      // ======================= MMA warps ====================================
      // lane 0 of one issues the score products, of the other the value
      // products; a commit covers the products its own thread issued
      const bool scores = warp == kPfWorkers / 32;
      // Barrier phases: S(c + 2) takes the columns of P(c), so its warp waits
      // for PV(c) first, and PV(c + 2) needs S(c + 2); the value warp waits for
      // every epi(c) in order before PV(c), and epi(c + 2) needs S(c + 2).  So
      // every wait is for the phase after the one its warp last saw.
      int kk = 0, njob = 0, c = 0;
      PfRing ru, rr;
      bool ok = true;
      for (int job = next_job(); job < p.n_jobs; job = next_job()) {
        if (ok && lane == 0) {
          const Job J = job_at(job);
          // this job's query rows are staged (and the last job's O was read)
          ok = sleepy(qready, njob & 1);
          ++njob;
          for (int k = 0; k < J.n_t && ok; ++k, ++kk) {
            if (scores) {
              if (kk >= 2) ok = spin(&pvdone[kk & 1], ((kk >> 1) - 1) & 1);  // P(kk - 2) is read
              for (int u = 0; u < 2 && ok; ++u, ++c, ru.next(scores ? p.nk : p.nv)) {
                const int s = ru.s;
                ok = spin(&kfull[s], ru.ph);
                if (!ok) break;
                tc_fence_after();
                const uint32_t ku = smem_u32(sm + s * p.ub);
                if constexpr (MLA) {
                  pf_issue_scores_ss<true>(t_s(kk), smem_u32(sm + p.off_q) + u * 16384, ku, u > 0);
                } else if (p.k_lo) {
                  if (p.q_lo) pf_issue_scores<true, true>(t_s(kk), t_q + 32 * u, ku, u > 0);
                  else pf_issue_scores<true, false>(t_s(kk), t_q + 32 * u, ku, u > 0);
                } else {
                  if (p.q_lo) pf_issue_scores<false, true>(t_s(kk), t_q + 32 * u, ku, u > 0);
                  else pf_issue_scores<false, false>(t_s(kk), t_q + 32 * u, ku, u > 0);
                }
                umma_commit(&kfree[s]);
              }
              if constexpr (MLA) {
                const int s = rr.s;
                if (ok) ok = spin(&rfull[s], rr.ph);
                if (ok) {
                  tc_fence_after();
                  const uint32_t q = smem_u32(sm + p.off_q) + 32768, kr = smem_u32(sm + p.off_r + s * p.krb);
                  if (p.krb > 16384) pf_issue_scores_ss<true>(t_s(kk), q, kr, true);
                  else pf_issue_scores_ss<false>(t_s(kk), q, kr, true);
                  umma_commit(&rfree[s]);
                  rr.next(p.nr);
                }
              }
              if (ok) umma_commit(&sdone[kk & 1]);
            } else {
              for (int u = 0; u < 2 && ok; ++u, ++c, ru.next(scores ? p.nk : p.nv)) {
                const int s = ru.s;
                ok = spin(&vfull[s], ru.ph);
                if (ok) ok = spin(&epi[2 * (kk & 1) + u], (kk >> 1) & 1);
                if (!ok) break;
                tc_fence_after();
                const uint32_t vh = smem_u32(sm + p.off_v + s * p.ub), pa = t_s(kk) + 32 * u;
                const bool acc = k > 0 || u > 0;
                if constexpr (MLA) pf_issue_values<true, true>(t_o, t_ol, pa, vh, (k & (p.flush - 1)) > 0 || u > 0, acc);
                else if (p.k_lo) pf_issue_values<true, false>(t_o, t_o, pa, vh, acc, true);
                else pf_issue_values<false, false>(t_o, t_o, pa, vh, acc, true);
                umma_commit(&vfree[s]);
              }
              if (ok) umma_commit(&pvdone[kk & 1]);
            }
          }
          if (!ok) *abort_flag = 1;
        }
        ok = __shfl_sync(0xffffffffu, ok, 0);
      }
      // every product this warp issued lands before TMEM is released (bounded)
      if (lane == 0 && c > 0) {
        uint64_t *d = &drain[scores ? 0 : 1];
        umma_commit(d);
        mbar_wait(d, 0, 1u << 22);
      }
      __syncwarp();
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kPfRegs.regs[0]) : "memory");
    // ======================= workers ======================================
    bool failed = false;
    auto wait_pv = [&](int c) -> bool {  // completion of tile c's value product
      return c < 0 || sleepy(&pvdone[c & 1], (c >> 1) & 1);
    };
    // query rows r0 .. r0 + 127 of the unit (zero past R) into TMEM (MLA:
    // shared memory), this thread's row and quarter of the channels
    auto load_q = [&](const Job &J) {
      const int rl = 32 * quarter + lane;
      float x[32];
#pragma unroll
      for (int i = 0; i < 32; ++i) x[i] = 0.f;
      if (rl < J.nr) {
        const int r = J.r0 + rl;
        const int qi = r / a.G, h = J.j * a.G + (r - qi * a.G);
        const size_t off = (((size_t)J.b * a.n_q + qi) * a.Hq + h) * D + 32 * slice;
        if (a.q_f32) {
          const float4 *src = reinterpret_cast<const float4 *>(static_cast<const float *>(a.q) + off);
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            const float4 u = src[c];
            x[4 * c] = u.x; x[4 * c + 1] = u.y; x[4 * c + 2] = u.z; x[4 * c + 3] = u.w;
          }
        } else {
          const uint4 *src = reinterpret_cast<const uint4 *>(static_cast<const uint16_t *>(a.q) + off);
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const uint4 u = src[c];
            const uint32_t ww[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              x[8 * c + 2 * i] = __uint_as_float(ww[i] << 16);
              x[8 * c + 2 * i + 1] = __uint_as_float(ww[i] & 0xFFFF0000u);
            }
          }
        }
      }
      uint32_t hw[16], lw[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) split2<true>(x[2 * i], x[2 * i + 1], hw[i], lw[i]);
      if constexpr (MLA) {
        // the row's 32 content channels and 16 of its positional ones, K-major
        // boxes of 64 channels in shared memory
        uint8_t *q_s = sm + p.off_q;
#pragma unroll
        for (int cc = 0; cc < 4; ++cc)
          put_chunk(q_s, rl, 32 * slice + 8 * cc, 16384,
                    make_uint4(hw[4 * cc], hw[4 * cc + 1], hw[4 * cc + 2], hw[4 * cc + 3]));
#pragma unroll
        for (int cc = 0; cc < 2; ++cc) {
          uint4 u = make_uint4(0, 0, 0, 0);
          if (rl < J.nr)
            u = reinterpret_cast<const uint4 *>(static_cast<const uint16_t *>(a.q_pe) +
                                                (((size_t)J.b * a.n_q + J.r0 + rl) * a.Hq + J.j) * 64 + 16 * slice)[cc];
          put_chunk(q_s, rl, 128 + 16 * slice + 8 * cc, 16384, u);
        }
        fence_proxy_async();
      } else {
        tmem_st16_nw(t_q + 16 * slice + lane_off, hw);
        if (p.q_lo) tmem_st16_nw(t_q + 64 + 16 * slice + lane_off, lw);
        tmem_wait_st();
      }
      tc_fence_before();  // the rows, stored here, are read by the tensor cores
      workers_sync<kPfWorkers>();
    };

    int kk = 0;
    // [tile parity][4 slices][128 rows]: the rows' slice maxima
    float *smax = reinterpret_cast<float *>(sm + p.off_red);
    float *ref_out = smax + 2 * 4 * kPfRows;  // (MLA) each thread's reference at its last flush
    const bool sector = (reinterpret_cast<uintptr_t>(a.out) & 31) == 0;  // rows start on 32 bytes
    // this thread's 32 channels of row rl of a job in the output
    auto out_row = [&](const Job &J, int rl) {
      const int r = J.r0 + rl, qi = r / a.G, h = J.j * a.G + (r - qi * a.G);
      return a.out + (((size_t)J.b * a.n_q + qi) * a.Hq + h) * D + 32 * slice;
    };
    // The four warps that share a quarter of the rows meet on a barrier of
    // their own: a row's maximum and its columns concern no other warp.
    auto row_sync = [&]() { asm volatile("bar.sync %0, 128;" ::"r"(4 + quarter) : "memory"); };
    for (int job = next_job(); job < p.n_jobs; job = next_job()) {
      if (failed) continue;
      const Job J = job_at(job);
      const int base = J.len - a.n_q;  // position of chunk query 0
      load_q(J);
      __syncwarp();
      if (lane == 0) mbar_arrive(qready);
      // this thread's row of the job (and slice of each tile's positions)
      const int rl = 32 * quarter + lane;
      const bool row_live = rl < J.nr;
      const int last = base + (J.r0 + rl) / a.G;  // the last position the row sees
      // The row's reference maximum (scaled scores, base 2) and this slice's
      // sum of weights.  The reference stays while no score of the row rises
      // more than 8 above it (P <= 2^8); when one does, the row's four
      // threads move it and rescale their channels of O (in TMEM, after the
      // value product of the previous tile) and their sums.  The weights
      // are not normalised: O is divided by the row's sum at the end.
      // A warp whose wait gave up stays in the tile loop for the barriers.
      // Formed values (MLA) are stored divided by 2^e, e by 32 positions, and
      // weights and values are split into f16: the reference is that of x +
      // e and moves at a rise of 4, and the weights are 2^(x + e - m + 11) (at
      // most 2^15; f16 halves keep 22 bits of those above 2^-3, and 2^-36 of
      // 2^11 of the others), whose sum takes 2^-e.
      constexpr float kRise = MLA ? 4.f : 8.f;
      float c_ref = -INFINITY, l_run = 0.f;
      const uint64_t sg2 = pair_f32(sg, sg);
      const uint32_t *vexp = MLA ? a.vexp + (size_t)J.unit * p.n_t : nullptr;
      uint32_t ve = MLA && J.n_t > 0 ? __ldg(vexp) : 0;
      for (int k = 0; k < J.n_t; ++k, ++kk) {
        // exponents e of this thread's positions of either value unit, and
        // 2^-e, while the scores are on their way (after them: 266 us for 260)
        float fe[2] = {0.f, 0.f}, down[2] = {1.f, 1.f};
        if constexpr (MLA) {
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const int e = (int8_t)(ve >> (8 * (slice >> 1) + 16 * u));
            fe[u] = (float)e;
            down[u] = __uint_as_float((uint32_t)(127 - e) << 23);
          }
          if (k + 1 < J.n_t) ve = __ldg(vexp + k + 1);
        }
        // scores of this tile (issued once the buffer's last P was read)
        if (!failed && !__all_sync(0xffffffffu, spin(&sdone[kk & 1], (kk >> 1) & 1))) {
          failed = true;
          *abort_flag = 1;
        }
        tc_fence_after();
        // this thread's positions: 16 of either value unit's 64
        const int tb = k * kPfT + 16 * slice;
        const int nv0 = row_live ? last - tb + 1 : 0, nv1 = nv0 - 64;  // live ones if < 16 (<= 0: none)
        float y[32];
        tmem_ld16x2(t_s(kk) + 16 * slice + lane_off, t_s(kk) + 64 + 16 * slice + lane_off, y);
        float mx = -INFINITY;
        if constexpr (MLA) {
          float mu[2] = {-INFINITY, -INFINITY};
          if (row_live && nv1 >= 16) {
#pragma unroll
            for (int u = 0; u < 2; ++u) {
              float mm[4];
#pragma unroll
              for (int i = 0; i < 4; ++i)
                mm[i] = fmaxf(fmaxf(y[16 * u + i], y[16 * u + 4 + i]), fmaxf(y[16 * u + 8 + i], y[16 * u + 12 + i]));
              mu[u] = fmaxf(fmaxf(mm[0], mm[1]), fmaxf(mm[2], mm[3]));
            }
          } else {
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              if (i < nv0) mu[0] = fmaxf(mu[0], y[i]);
              if (i < nv1) mu[1] = fmaxf(mu[1], y[16 + i]);
            }
          }
          mx = fmaxf(fmaf(mu[0], sg, fe[0]), fmaf(mu[1], sg, fe[1]));
        } else if (row_live && nv1 >= 16) {  // all in the row's range (most tiles)
          float mm[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) mm[i] = fmaxf(fmaxf(y[i], y[8 + i]), fmaxf(y[16 + i], y[24 + i]));
          mx = fmaxf(fmaxf(fmaxf(mm[0], mm[1]), fmaxf(mm[2], mm[3])), fmaxf(fmaxf(mm[4], mm[5]), fmaxf(mm[6], mm[7])));
        } else {
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            if (i < nv0) mx = fmaxf(mx, y[i]);
            if (i < nv1) mx = fmaxf(mx, y[16 + i]);
          }
        }
        float *sx = smax + (kk & 1) * 4 * kPfRows + rl;
        sx[slice * kPfRows] = mx;
        tc_fence_before();
        row_sync();  // the row's four slice maxima; its scores are all read
        tc_fence_after();
        const float M = (MLA ? 1.f : sg) * fmaxf(fmaxf(sx[0], sx[kPfRows]), fmaxf(sx[2 * kPfRows], sx[3 * kPfRows]));
        const bool move = M > c_ref + kRise;  // the same decision on the row's four threads
        const bool resc = move && c_ref != -INFINITY;
        const bool any_resc = __any_sync(0xffffffffu, resc);
        const bool flush = MLA && k > 0 && (k & (p.flush - 1)) == 0;
        if (any_resc || flush) {
          // O holds this job's earlier tiles: rescale this thread's 32
          // channels once the previous tile's value product is done.  Lanes
          // are rows and the TMEM accesses are warp-wide (.sync.aligned), so
          // the whole warp takes part, rows that do not move with factor 1.
          // A flush adds O to the row's partial result in the output (with
          // the reference it has there kept in shared memory); the next
          // value product starts O anew.
          if (!__all_sync(0xffffffffu, wait_pv(kk - 1))) {
            failed = true;
            *abort_flag = 1;
          } else {
            tc_fence_after();
            const float f = resc ? fast_exp2(c_ref - M) : 1.f;
            const float c_new = move ? M : c_ref, c_old = flush ? ref_out[tid] : 0.f;
            const float f_old = flush && k > p.flush && c_old != -INFINITY ? fast_exp2(c_old - c_new) : 0.f;
            float z[16];
            uint32_t zw[16];
#pragma unroll
            for (int h = 0; h < (MLA ? 4 : 2); ++h) {
              if (h >= 2 && !any_resc) continue;
              const uint32_t at = (h < 2 ? t_o : t_ol) + 32 * slice + 16 * (h & 1) + lane_off;
              tmem_ld16(at, z);
              if (MLA && h < 2 && flush) {
                if (row_live) {
                  float *dst = out_row(J, rl) + 16 * h;
#pragma unroll
                  for (int i = 0; i < 16; ++i) z[i] *= f;
                  if (k > p.flush) {
                    float x[2][8];
                    ld8(dst, x[0], sector);
                    ld8(dst + 8, x[1], sector);
#pragma unroll
                    for (int i = 0; i < 16; ++i) z[i] = fmaf(x[i >> 3][i & 7], f_old, z[i]);
                  }
                  st8(dst, z, sector);
                  st8(dst + 8, z + 8, sector);
                }
                __syncwarp();  // the TMEM loads are warp-wide
              } else {
#pragma unroll
                for (int i = 0; i < 16; ++i) zw[i] = __float_as_uint(z[i] * f);
                tmem_st16_nw(at, zw);
              }
            }
            l_run *= f;
            if (flush) ref_out[tid] = c_new;
          }
        }
        if (move) c_ref = M;
        const float c_up = c_ref - 11.f;
        // P of this row over its positions of one value unit, then of the
        // other, hi and lo halves: 8 columns of bf16 pairs (hi), the same 64
        // columns on (lo); the unit's value products start as soon as its
        // positions are written
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int nv = u ? nv1 : nv0;
          float *yu = y + 16 * u;
          uint64_t y2[8];
          const float off = MLA ? fe[u] - c_up : -c_ref;
          if (nv >= 16) {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              float e0, e1;
              unpair_f32(fma_f32x2(pair_f32(yu[2 * i], yu[2 * i + 1]), sg2, pair_f32(off, off)), e0, e1);
              y2[i] = pair_f32(fast_exp2(e0), fast_exp2(e1));
            }
          } else {
#pragma unroll
            for (int i = 0; i < 16; ++i) yu[i] = i < nv ? fast_exp2(fmaf(yu[i], sg, off)) : 0.f;
#pragma unroll
            for (int i = 0; i < 8; ++i) y2[i] = pair_f32(yu[2 * i], yu[2 * i + 1]);
          }
          uint32_t hw[8], lw[8];
          uint64_t ls[2] = {0, 0};
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            if constexpr (MLA) split2_f16(y2[i], hw[i], lw[i]);
            else split2_bf16(y2[i], hw[i], lw[i]);
            ls[i & 1] = add_f32x2(ls[i & 1], y2[i]);
          }
          float l0, l1;
          unpair_f32(add_f32x2(ls[0], ls[1]), l0, l1);
          if constexpr (MLA) l_run = fmaf(l0 + l1, down[u], l_run);
          else l_run += l0 + l1;
          tmem_st8_nw(t_s(kk) + 32 * u + 8 * slice + lane_off, hw);
          tmem_st8_nw(t_s(kk) + 64 + 32 * u + 8 * slice + lane_off, lw);
          tmem_wait_st();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&epi[2 * (kk & 1) + u]);
        }
      }
      // a rescale's wait that gave up on the last tile is seen by every worker
      if (workers_sync_or<kPfWorkers>(failed)) {
        failed = true;
        *abort_flag = 1;
        continue;
      }
      // O (MLA: and the lo products' sum), lane = the job's row, 32 channels
      // per slice, divided by the sum of the row's weights (the four slices'
      // sums, same reference)
      float o[32];
      const int *bad = a.bad + (size_t)J.unit * kPfBadStride;
      const bool sees_bad = (int)v.cap - last <= __ldg(bad + 128);  // a position that is not finite in some channel
      if (J.n_t > 0) {
        const bool ok = wait_pv(kk - 1);
        if (workers_sync_or<kPfWorkers>(!ok)) {
          failed = true;
          *abort_flag = 1;
          continue;
        }
        tc_fence_after();
        tmem_ld32(t_o + 32 * slice + lane_off, o);
        if constexpr (MLA) {
          float z[16];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            tmem_ld16(t_ol + 32 * slice + 16 * h + lane_off, z);
#pragma unroll
            for (int i = 0; i < 16; ++i) o[16 * h + i] += z[i];
          }
          if (J.n_t > p.flush && row_live) {
            const float c_old = ref_out[tid], f_old = c_old != -INFINITY ? fast_exp2(c_old - c_ref) : 0.f;
            const float *part = out_row(J, rl);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              float x[8];
              ld8(part + 8 * c, x, sector);
#pragma unroll
              for (int i = 0; i < 8; ++i) o[8 * c + i] = fmaf(x[i], f_old, o[8 * c + i]);
            }
          }
          __syncwarp();
        }
      } else {
#pragma unroll
        for (int i = 0; i < 32; ++i) o[i] = 0.f;
      }
      smax[slice * kPfRows + rl] = l_run;
      workers_sync<kPfWorkers>();
      const float L = (smax[rl] + smax[kPfRows + rl]) + (smax[2 * kPfRows + rl] + smax[3 * kPfRows + rl]);
      const float inv = L > 0.f ? 1.f / L : 0.f;
      if (sees_bad) {
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const int4 x = reinterpret_cast<const int4 *>(bad + 32 * slice)[c];
          const int at = (int)v.cap - last;
          if (at <= x.x) o[4 * c] = NAN;
          if (at <= x.y) o[4 * c + 1] = NAN;
          if (at <= x.z) o[4 * c + 2] = NAN;
          if (at <= x.w) o[4 * c + 3] = NAN;
        }
      }
      __syncwarp();
      if (row_live) {
        float4 *dst = reinterpret_cast<float4 *>(out_row(J, rl));
#pragma unroll
        for (int c = 0; c < 8; ++c)
          dst[c] = make_float4(o[4 * c] * inv, o[4 * c + 1] * inv, o[4 * c + 2] * inv, o[4 * c + 3] * inv);
      }
      tc_fence_before();
      workers_sync<kPfWorkers>();  // O and the sums read before the next job's first products
    }
    if (failed && tid == 0) set_err(a.err, 8);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(kCols)
                 : "memory");
  pdl_trigger();
}

// Shared-memory plan.  Attention kernel: the key units, the value units,
// MLA's positional keys and query rows, the rows' slice maxima (and at a
// job's end their sums of weights), barriers; S, P, O and else the query
// rows live in TMEM.  Expand kernel: half a tile and its staged records.
PfPlan pf_plan(const PfArgs &a, int sms) {
  PfPlan p;
  const int R = a.n_q * a.G;
  p.n_rb = (R + kPfRows - 1) / kPfRows;
  p.n_jobs = a.v.B * a.v.Hkv * p.n_rb;
  p.n_t = (int)((a.v.cap + kPfT - 1) / kPfT);
  p.q_lo = a.q_f32 ? 1 : 0;
  p.k_lo = a.v.bits != 16 || a.kr_bytes ? 1 : 0;  // formed keys and values have lo halves
  p.fmt = a.v.bits == 16 ? kFmtBf16
          : a.v.scheme == kSchemeSym ? (a.v.bits == 8 ? kFmtS8 : a.v.bits == 4 ? kFmtS4 : kFmtS2)
                                     : (a.v.bits == 8 ? kFmtG8 : kFmtG4);
  p.gshift = a.v.group == 64 ? 6 : 5;
  p.kpc = a.v.bits != 16 && a.v.key_axis == 1 ? 1 : 0;
  p.ks16 = TcFmtKs16(p.fmt);
  p.nrec = a.v.rec_bytes / 16;
  p.nc_magic = (uint32_t)((0x100000000ull + p.nrec - 1) / p.nrec);
  const bool sym = p.fmt >= kFmtS8;
  const int bchunks = p.nrec + (sym ? 1 : 0);
  p.b_stride = 16 * (bchunks % 2 ? bchunks : bchunks + 1);
  p.ub = 2 * kPfBox * (p.k_lo ? 2 : 1);
  p.tbytes = 4 * p.ub;
  p.krb = a.kr_bytes;
  p.flush = a.flush;
  // + the (scale, zero) rows of the tile's position groups (per-channel keys)
  p.smem_x = 2 * p.ub + 64 * p.b_stride + (p.kpc ? 2 * 128 * 8 : 0) + 1024;
  const int rbytes = 2 * 4 * kPfRows * 4 + (a.kr_bytes ? kPfWorkers * 4 : 0);
  const int qbytes = p.krb ? 3 * 16384 : 0;
  // the most units that fit, values the larger share (a value unit waits for
  // the epilogue of its tile, key units only for the tile before)
  int avail = 232448 - (rbytes + kPfBarBytes + 1024) - qbytes;
  p.nr = p.krb ? (p.krb <= 16384 ? 2 : 1) : 0;
  avail -= p.nr * p.krb;
  const int T = avail / p.ub;
  p.nk = std::min(kPfMaxStages, std::max(2, T / 2));
  p.nv = std::max(1, std::min(kPfMaxStages, T - p.nk));
  // bands of units whose tiles take up to 32 MB (L2 holds two bands)
  const long long unit_bytes = (long long)p.n_t * p.tbytes;
  p.band = (int)std::max(1LL, std::min<long long>(a.v.B * a.v.Hkv, (32LL << 20) / std::max(1LL, unit_bytes)));
  p.off_v = p.nk * p.ub;
  p.off_r = p.off_v + p.nv * p.ub;
  p.off_q = p.off_r + p.nr * p.krb;
  p.off_red = p.off_q + qbytes;
  p.off_bar = p.off_red + rbytes;
  // + alignment of the base to 1024 bytes; at least half the SM's shared
  // memory, so that one CTA (holding its TMEM columns) runs per SM
  p.smem = std::max(p.off_bar + kPfBarBytes + 1024, 116 * 1024);
  p.grid = std::max(1, std::min(p.n_jobs, sms));
  return p;
}

}  // namespace

size_t prefill_unit_bytes(int bits, int64_t cap) {
  return (size_t)((cap + kPfT - 1) / kPfT) * 8 * kPfBox * (bits != 16 ? 2 : 1);
}

bool prefill_plan_fits(const PfArgs &a) {
  const PfPlan o = pf_plan(a, 1);
  return o.smem <= 232448 && o.nk >= 2 && o.nv >= 2;
}

static cudaError_t pf_sms(int *out) {
  static int sms = 0;
  if (!sms) {
    int dev = 0, n = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    sms = n;
  }
  *out = sms;
  return cudaSuccess;
}

cudaError_t launch_mla_prefill_formed(const PfArgs &a, cudaStream_t st) {
  int sms = 0;
  cudaError_t e = pf_sms(&sms);
  if (e != cudaSuccess) return e;
  const PfPlan p = pf_plan(a, sms);
  e = check_reg_split<&prefill_kernel<true>>(kPfRegs);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(prefill_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, p.smem);
  if (e == cudaSuccess)
    e = launch_pdl(prefill_kernel<true>, dim3(p.grid), dim3(kPfThreads), p.smem, st, a, p);
  return e;
}

cudaError_t launch_gqa_prefill(const PfArgs &a, cudaStream_t st) {
  int sms = 0;
  cudaError_t e = pf_sms(&sms);
  if (e != cudaSuccess) return e;
  const PfPlan po = pf_plan(a, sms);
  e = check_reg_split<&prefill_kernel<false>>(kPfRegs);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(prefill_expand_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, po.smem_x);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(prefill_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, po.smem);
  if (e != cudaSuccess) return e;
  // the job counter and the records of non-finite values behind it
  e = cudaMemsetAsync(a.counter, 0, 1024 + (size_t)a.v.B * a.v.Hkv * kPfBadStride * 4, st);
  if (e == cudaSuccess)
    e = launch_pdl(prefill_expand_kernel, dim3(2 * po.n_t, a.v.B * a.v.Hkv), dim3(kPfWorkers), po.smem_x, st,
                   a, po);
  if (e == cudaSuccess)
    e = launch_pdl(prefill_kernel<false>, dim3(po.grid), dim3(kPfThreads), po.smem, st, a, po);
  return e;
}

}  // namespace kvk
