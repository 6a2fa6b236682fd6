// append.cu -- quantise / truncate on write (Appendix C.2, C.3).
//
// GQA rows: one warp per (sequence, new position, KV head).  Values, and keys
// with per-token groups, are quantised at once with the grouped asymmetric
// quantiser as an exact binary32 operation sequence (round-to-nearest
// subtract and divide, rint = round half to even, no contraction):
//     scale = (max - min) / (2^b - 1),  zero = min,
//     code  = clamp(rint((x - min) / scale), 0, 2^b - 1)   (scale 0 -> 0).
// Keys with per-channel groups (KIVI) are kept in bf16 in a residual plane
// until `group` positions of a group exist; then the group is quantised
// along positions, one (scale, zero) per channel.
//
// The sequence lengths advance after every row has been written: the last
// CTA to finish (completion counter) updates them, so no extra launch and no
// waiting are needed.
#include <math.h>

#include "common.cuh"
#include "kernels.h"
#include "layout.h"

namespace kvk {
namespace {

__device__ __forceinline__ int seq_count(const int32_t *n_per_seq, int b, int n_new,
                                         int32_t *err) {
  if (!n_per_seq) return n_new;
  const int n = n_per_seq[b];
  if (n < 0 || n > n_new) {
    set_err(err, 4);
    return 0;
  }
  return n;
}

// rint(fl(d / s)) for s > 0 and |d / s| at most a few hundred, without a
// division in the common case.  rs is the fast reciprocal of s
// (__fdividef(1, s): within 2 ulp of 1/s for normal s), so y = fl(d rs) is
// within 1.8e-7 |d/s| of d/s, and fl(d/s) within 6e-8 |d/s|: for |d/s| <=
// 300 the two differ by less than 7.2e-5, and when y is further than 1e-4
// from the nearest half-integer both round to the same integer.  Otherwise
// (or when y is not finite, as for a scale whose reciprocal overflows) the
// correctly rounded division decides.  `near` reports that case.
__device__ __forceinline__ float rint_quot_fast(float d, float rs, bool &near) {
  const float y = __fmul_rn(d, rs);
  const float r = rintf(y);
  near = !(fabsf(__fsub_rn(y, r)) < 0.4999f);
  return r;
}

// Quantise one lane's E elements belonging to groups of GS channels spread
// over GS/E consecutive lanes.  Returns codes, writes the group's scale and
// zero into (sc, zr) on every lane of the group.
template <int E>
__device__ __forceinline__ void quant_lane(const float (&x)[E], int GS, int levels,
                                           uint32_t (&code)[E], float &sc, float &zr) {
  float mn = x[0], mx = x[0];
#pragma unroll
  for (int e = 1; e < E; ++e) { mn = fminf(mn, x[e]); mx = fmaxf(mx, x[e]); }
  const int lanes = GS / E;
  for (int off = 1; off < lanes; off <<= 1) {
    mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, off));
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
  }
  const float lev = (float)levels;
  const float scale = __fdiv_rn(__fsub_rn(mx, mn), lev);
  const float rs = scale == 0.f ? 0.f : __fdividef(1.f, scale);
  float r[E];
  bool any_near = false;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    bool near;
    r[e] = rint_quot_fast(__fsub_rn(x[e], mn), rs, near);
    any_near |= near;
  }
  if (__any_sync(0xffffffffu, any_near && scale != 0.f)) {
#pragma unroll
    for (int e = 0; e < E; ++e)
      if (scale != 0.f) r[e] = rintf(__fdiv_rn(__fsub_rn(x[e], mn), scale));
  }
#pragma unroll
  for (int e = 0; e < E; ++e) code[e] = scale == 0.f ? 0u : (uint32_t)fminf(fmaxf(r[e], 0.f), lev);
  sc = scale;
  zr = mn;
}

// Symmetric per-vector quantiser (Appendix C.3) of one warp's row, lane
// holding E channels: s = bf16(max|x| / q) (one binary32 division, then
// round to nearest even), code = clip(rint(x / s), -q, q) with the stored
// scale, returned offset by q (u = code + q).  A zero row stores s = 0 and
// code 0.  Returns the bf16 bits of s.
template <int E>
__device__ __forceinline__ uint16_t quant_sym_lane(const float (&x)[E], int bits,
                                                   uint32_t (&u)[E]) {
  float am = 0.f;
#pragma unroll
  for (int e = 0; e < E; ++e) am = fmaxf(am, fabsf(x[e]));
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) am = fmaxf(am, __shfl_xor_sync(0xffffffffu, am, off));
  const float q = (float)sym_levels(bits);
  const uint16_t sb = f32_to_bf16_bits(__fdiv_rn(am, q));
  const float s = bf16_to_f32(sb);
  const float rs = s == 0.f ? 0.f : __fdividef(1.f, s);
  float rq[E];
  bool any_near = false;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    bool near;
    rq[e] = rint_quot_fast(x[e], rs, near);
    any_near |= near;
  }
  if (__any_sync(0xffffffffu, any_near && s != 0.f)) {
#pragma unroll
    for (int e = 0; e < E; ++e)
      if (s != 0.f) rq[e] = rintf(__fdiv_rn(x[e], s));
  }
#pragma unroll
  for (int e = 0; e < E; ++e) {
    float r = 0.f;
    if (s != 0.f) r = fminf(fmaxf(rq[e], -q), q);
    u[e] = (uint32_t)(int)(r + q);
  }
  return sb;
}

// Symmetric record of (sequence b, position t, KV head kvh): both sections
// assembled in the per-warp buffer in physical (rotated) order, stored as
// whole 16-byte chunks; the two scales go to the scale plane.
template <int D>
__device__ void append_row_sym(const GqaView &v, const float (&xk)[D / 32],
                               const float (&xv)[D / 32], int b, int kvh, int t, uint32_t *buf,
                               int lane) {
  constexpr int E = D / 32;
  const int rb = v.rec_bytes;
  const int kb = D * v.bits / 8;
  const size_t row = ((size_t)b * v.Hkv + kvh) * v.cap + t;
  uint32_t uk[E], uv[E];
  const uint32_t sk = quant_sym_lane<E>(xk, v.bits, uk);
  const uint32_t sv = quant_sym_lane<E>(xv, v.bits, uv);
  for (int w = lane; w < rb / 4; w += 32) buf[w] = 0;
  __syncwarp();
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int ch = lane * E + e;
    const int lk = sym_k_bit(ch, v.bits, D);
    const int pk = 8 * sym_phys(lk >> 3, t, rb) + (lk & 7);
    atomicOr(buf + (pk >> 5), uk[e] << (pk & 31));
    const int lv = sym_v_bit(ch, v.bits, D) + 8 * kb;
    const int pv = 8 * sym_phys(lv >> 3, t, rb) + (lv & 7);
    atomicOr(buf + (pv >> 5), uv[e] << (pv & 31));
  }
  __syncwarp();
  uint4 *rec = reinterpret_cast<uint4 *>(v.rec + row * rb);
  for (int q = lane; q < rb / 16; q += 32) rec[q] = reinterpret_cast<const uint4 *>(buf)[q];
  if (lane == 0) v.scales[row] = sk | (sv << 16);
  __syncwarp();
}

// Writes one section (K or V) of a record through a per-warp shared buffer
// so the global stores are whole 16-byte chunks.
template <int D>
__device__ void put_section(uint32_t *buf, int bits, bool is_k, const uint32_t (&val)[D / 32],
                            int t, int rec_bytes, int lane) {
  constexpr int E = D / 32;
  const int words = D * bits / 32;
  for (int w = lane; w < words; w += 32) buf[w] = 0;
  __syncwarp();
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int ch = lane * E + e;
    int byte, hi;
    if (is_k)
      k_pos(ch, bits, D, &byte, &hi);
    else
      v_pos(ch, bits, D, t, rec_bytes, &byte, &hi);
    uint32_t v = val[e];
    int shift = (byte & 3) * 8;
    if (bits == 4) shift += hi * 4;
    atomicOr(buf + (byte >> 2), v << shift);
  }
  __syncwarp();
}

// E = D / 32 consecutive elements of one lane, one vector load (inputs are
// 16-byte aligned and rows are D elements long)
template <int E>
__device__ __forceinline__ void load_lane(const void *in, size_t i, int f32, float (&x)[E]) {
  static_assert(E == 2 || E == 4, "two or four elements per lane");
  if (f32) {
    const float *p = static_cast<const float *>(in) + i;
    if constexpr (E == 4) {
      const float4 w = *reinterpret_cast<const float4 *>(p);
      x[0] = w.x; x[1] = w.y; x[2] = w.z; x[3] = w.w;
    } else {
      const float2 w = *reinterpret_cast<const float2 *>(p);
      x[0] = w.x; x[1] = w.y;
    }
  } else {
    const uint16_t *p = static_cast<const uint16_t *>(in) + i;
    uint32_t w[E / 2];
    if constexpr (E == 4) {
      const uint2 u = *reinterpret_cast<const uint2 *>(p);
      w[0] = u.x; w[1] = u.y;
    } else {
      w[0] = *reinterpret_cast<const uint32_t *>(p);
    }
#pragma unroll
    for (int j = 0; j < E / 2; ++j) {
      x[2 * j] = __uint_as_float(w[j] << 16);
      x[2 * j + 1] = __uint_as_float(w[j] & 0xffff0000u);
    }
  }
}

template <int D>
__device__ __forceinline__ void load_row(const void *kin, const void *vin, int in_f32,
                                         size_t ibase, int lane, float (&xk)[D / 32],
                                         float (&xv)[D / 32]) {
  load_lane<D / 32>(kin, ibase + lane * (D / 32), in_f32, xk);
  load_lane<D / 32>(vin, ibase + lane * (D / 32), in_f32, xv);
}

// Quantises and writes one (sequence b, position t, KV head kvh) record from
// the warp's inputs (lane holds channels [lane E, lane E + E)).
template <int D>
__device__ void append_row(const GqaView &v, const float (&xk)[D / 32], const float (&xv)[D / 32],
                           int b, int kvh, int t, uint32_t *buf, int lane) {
  constexpr int E = D / 32;
  if (v.scheme == kSchemeSym) {
    append_row_sym<D>(v, xk, xv, b, kvh, t, buf, lane);
    return;
  }
  const RecLayout L = rec_layout(v.bits, D, v.group, v.key_axis);
  uint8_t *rec = v.rec + (((size_t)b * v.Hkv + kvh) * v.cap + t) * L.rec;
  const bool kq = v.bits != 16 && v.key_axis == 0;
  const bool kres = v.bits != 16 && v.key_axis == 1;
  // ---- K section ----
  if (!kres) {
    uint32_t val[E];
    float sc = 0.f, zr = 0.f;
    if (kq) {
      quant_lane<E>(xk, v.group, (1 << v.bits) - 1, val, sc, zr);
    } else {
#pragma unroll
      for (int e = 0; e < E; ++e) val[e] = f32_to_bf16_bits(xk[e]);
    }
    put_section<D>(buf, kq ? v.bits : 16, true, val, t, L.rec, lane);
    const int kb = D * v.bits / 8;
    for (int q = lane; q < kb / 16; q += 32)
      reinterpret_cast<uint4 *>(rec + L.k_off)[q] = reinterpret_cast<uint4 *>(buf)[q];
    if (kq && (lane * E) % v.group == 0)
      reinterpret_cast<float2 *>(rec + L.km_off)[(lane * E) / v.group] = make_float2(sc, zr);
    __syncwarp();
  }
  // ---- V section ----
  {
    uint32_t val[E];
    float sc = 0.f, zr = 0.f;
    const bool vq = v.bits != 16;
    if (vq) {
      quant_lane<E>(xv, v.group, (1 << v.bits) - 1, val, sc, zr);
    } else {
#pragma unroll
      for (int e = 0; e < E; ++e) val[e] = f32_to_bf16_bits(xv[e]);
    }
    put_section<D>(buf, v.bits, false, val, t, L.rec, lane);
    const int vb = D * v.bits / 8;
    for (int q = lane; q < vb / 16; q += 32)
      reinterpret_cast<uint4 *>(rec + L.v_off)[q] = reinterpret_cast<uint4 *>(buf)[q];
    if (vq && (lane * E) % v.group == 0)
      reinterpret_cast<float2 *>(rec + L.vm_off)[(lane * E) / v.group] = make_float2(sc, zr);
  }
}

// Row wid = (b n_new + i) Hkv + kvh of an append, tracked as (b, i, kvh)
// and advanced by a fixed stride with carries instead of divided per row:
// the stride's own decomposition is computed once.
struct RowIdx {
  uint32_t b, i, kvh;
};
struct RowStep {
  uint32_t Hkv, n_new, db, di, dk;
  __device__ RowStep(uint32_t step, uint32_t Hkv_, uint32_t n_new_) : Hkv(Hkv_), n_new(n_new_) {
    const uint32_t q = step / Hkv;
    dk = step - q * Hkv;
    db = q / n_new;
    di = q - db * n_new;
  }
  __device__ RowIdx at(uint32_t w) const {
    const uint32_t q = w / Hkv, b = q / n_new;
    return RowIdx{b, q - b * n_new, w - q * Hkv};
  }
  __device__ RowIdx next(RowIdx r) const {  // the row `step` further on
    r.kvh += dk;
    const uint32_t c = r.kvh >= Hkv;
    r.kvh -= c ? Hkv : 0u;
    r.i += di + c;
    const uint32_t c2 = r.i >= n_new;
    r.i -= c2 ? n_new : 0u;
    r.b += db + c2;
    return r;
  }
};

template <int D>
__global__ void __launch_bounds__(128)
    gqa_append_rows(const GqaView v, const void *kin, const void *vin, int in_f32, int n_new,
                    const int32_t *n_per_seq, int32_t *err) {
  pdl_wait();
  pdl_trigger();
  constexpr int E = D / 32;
  __shared__ __align__(16) uint32_t sbuf[4][(2 * D * 2 + 2 * 64) / 4];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const size_t total = (size_t)v.B * n_new * v.Hkv;
  // rows wid, wid + 4 gridDim.x, ...: a bounded grid, so that the completion
  // counter below takes one atomic per CTA, not one per four rows
  // (the grid stride and the first row fit 32 bits; the row index itself
  // stays 64-bit, its (b, i, kvh) advance by the stride)
  const RowStep rstep((uint32_t)gridDim.x * 4u, (uint32_t)v.Hkv, (uint32_t)n_new);
  RowIdx ridx = rstep.at((uint32_t)min((size_t)blockIdx.x * 4 + warp, total));
  for (size_t wid = (size_t)blockIdx.x * 4 + warp; wid < total; wid += (size_t)gridDim.x * 4) {
    const int kvh = (int)ridx.kvh, i = (int)ridx.i, b = (int)ridx.b;
    ridx = rstep.next(ridx);
    const int nb = seq_count(n_per_seq, b, n_new, err);
    const int t = v.lens[b] + i;
    bool ok = i < nb;
    if (ok && t >= v.cap) {
      if (lane == 0) set_err(err, 2);
      ok = false;
    }
    if (ok) {
      float xk[E], xv[E];
      load_row<D>(kin, vin, in_f32, (((size_t)b * n_new + i) * v.Hkv + kvh) * D, lane, xk, xv);
      append_row<D>(v, xk, xv, b, kvh, t, sbuf[warp], lane);
    }
    __syncwarp();  // the row buffer is free again
  }
  // The last CTA advances the lengths (per-token layouts only; per-channel
  // keys advance them in the residual kernel, which runs last).
  if (v.bits == 16 || v.key_axis == 0) {
    __syncthreads();
    __shared__ int last;
    if (threadIdx.x == 0) {
      __threadfence();
      last = (atomicAdd(v.counter, 1) == (int)gridDim.x - 1);
    }
    __syncthreads();
    if (last) {
      for (int b = threadIdx.x; b < v.B; b += blockDim.x) {
        const int nb = seq_count(n_per_seq, b, n_new, nullptr);
        v.lens[b] = min((long long)v.lens[b] + nb, (long long)v.cap);
      }
      if (threadIdx.x == 0) *v.counter = 0;
    }
  }
}

// ---- bulk appends, head_dim 128, per-token layouts -------------------------
// bf16: one warp per (sequence, new position, KV head) row over a bounded
// grid, lane L holding channels 4L .. 4L+3; the record's 32-bit words are
// gathered from the lanes that hold their channels by warp shuffles (the
// channel order of layout.h, derived below) and stored as whole words.
// 8- and 4-bit codes: a lane per 32 channels (gqa_append_quads).

// bf16 values: lane owns K words T = lane, lane + 32 (chunk T / 4, c =
// chunk % 4, j = 2 (chunk / 4) + (T % 4) / 2, h = T % 2: the bf16 pair of
// elements 2 (c%2), +1 of lane 4j + c/2 + 2h) and V words W = lane, lane + 32
// (row g = W / 8, M-block m = W % 8: element g % 4 of lanes 4m + g/4 (low
// half) and 4m + g/4 + 2 (high half)).
struct Gather16 {
  int ks[2], kreg, vs[2], vreg, vhalf;
  __device__ explicit Gather16(int lane) {
    const int c = (lane >> 2) & 3;
    kreg = c & 1;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int T = lane + 32 * i, chunk = T >> 2;
      const int j = 2 * (chunk >> 2) + ((T & 3) >> 1);
      ks[i] = 4 * j + (c >> 1) + 2 * (T & 1);
    }
    const int g0 = lane >> 3;  // rows g0 (W = lane) and g0 + 4 (W = lane + 32)
    const int m = lane & 7;
    vs[0] = 4 * m + (g0 >> 2);
    vs[1] = 4 * m + ((g0 + 4) >> 2);
    vreg = ((g0 & 3) >> 1);  // the same for g0 + 4
    vhalf = 16 * (g0 & 1);
  }
  __device__ __forceinline__ uint32_t kword(uint32_t k0, uint32_t k1, int i) const {
    const uint32_t a = __shfl_sync(0xffffffffu, k0, ks[i]);
    const uint32_t b = __shfl_sync(0xffffffffu, k1, ks[i]);
    return kreg ? b : a;
  }
  __device__ __forceinline__ uint32_t vword(uint32_t v0, uint32_t v1, int i) const {
    const uint32_t a0 = __shfl_sync(0xffffffffu, v0, vs[i]);
    const uint32_t a1 = __shfl_sync(0xffffffffu, v1, vs[i]);
    const uint32_t b0 = __shfl_sync(0xffffffffu, v0, vs[i] + 2);
    const uint32_t b1 = __shfl_sync(0xffffffffu, v1, vs[i] + 2);
    const uint32_t lo = ((vreg ? a1 : a0) >> vhalf) & 0xFFFFu;
    const uint32_t hi = ((vreg ? b1 : b0) >> vhalf) & 0xFFFFu;
    return lo | (hi << 16);
  }
};

// The last CTA to finish advances the lengths (completion counter).
__device__ __forceinline__ void advance_lengths(const GqaView &v, int n_new, const int32_t *n_per_seq) {
  __syncthreads();
  __shared__ int last;
  if (threadIdx.x == 0) {
    __threadfence();
    last = (atomicAdd(v.counter, 1) == (int)gridDim.x - 1);
  }
  __syncthreads();
  if (last) {
    for (int b = threadIdx.x; b < v.B; b += blockDim.x) {
      const int nb = seq_count(n_per_seq, b, n_new, nullptr);
      v.lens[b] = min((long long)v.lens[b] + nb, (long long)v.cap);
    }
    if (threadIdx.x == 0) *v.counter = 0;
  }
}

// 32 consecutive elements of one lane, from 16-byte aligned bf16 or fp32
__device__ __forceinline__ void load_quarter(const void *p, bool f32, float (&x)[32]) {
  if (f32) {
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const float4 u = static_cast<const float4 *>(p)[j];
      x[4 * j] = u.x; x[4 * j + 1] = u.y; x[4 * j + 2] = u.z; x[4 * j + 3] = u.w;
    }
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const uint4 u = static_cast<const uint4 *>(p)[j];
      const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        x[8 * j + 2 * k] = __uint_as_float(w[k] << 16);
        x[8 * j + 2 * k + 1] = __uint_as_float(w[k] & 0xffff0000u);
      }
    }
  }
}

// 1.5 2^23: adding it to |y| < 2^22 rounds y to the nearest integer, half to
// even, and leaves that integer in the low bits of the sum's pattern.
constexpr float kRintBias = 12582912.f;
constexpr uint32_t kRintBits = 0x4B400000u;

// Codes of one lane's 32 channels (a quarter of a row), given the group's
// scale and zero (symmetric: zero 0): bits[e] = kRintBits + rint(fl((x - zr) /
// sc)), clamped to [lo, hi].  The quotients are the correctly rounded ones,
// by residuals: with y = RN(1/sc), q within an ulp of d/sc and r = d - q sc
// (exact in one FMA), RN(q + r y) = RN(d/sc) (Markstein, "Computation of
// elementary functions on the IBM RISC System/6000 processor", 1990); the
// first residual step brings RN(d y) within that ulp, the second rounds.
// (Deciding near-halves by the division instead cost half the kernel: bf16
// inputs put exact ties into nearly every warp.)  The theorem wants no
// underflow and no overflow, so scales outside [2^-96, 2^96] (0 among them)
// and groups with a value that is not finite take the division.  `over`: the
// largest quotient may pass hi (a scale rounded down).
__device__ __forceinline__ void quarter_codes(const float (&x)[32], float sc, float zr, float lo, float hi, bool over,
                                              uint32_t (&bits)[32]) {
  const float y = __frcp_rn(sc);
  const uint64_t nz = pair_f32(-zr, -zr), y2 = pair_f32(y, y), ns = pair_f32(-sc, -sc),
                 b2 = pair_f32(kRintBias, kRintBias);
  uint64_t sum = pair_f32(0.f, 0.f);
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const uint64_t d = add_f32x2(pair_f32(x[2 * i], x[2 * i + 1]), nz);
    uint64_t q = mul_f32x2(d, y2);
    q = fma_f32x2(fma_f32x2(q, ns, d), y2, q);
    q = fma_f32x2(fma_f32x2(q, ns, d), y2, q);
    sum = add_f32x2(sum, d);
    float t0, t1;
    unpair_f32(add_f32x2(q, b2), t0, t1);
    bits[2 * i] = __float_as_uint(t0);
    bits[2 * i + 1] = __float_as_uint(t1);
  }
  float s0, s1;
  unpair_f32(sum, s0, s1);
  if (!(fabsf(s0 + s1) < INFINITY) || !(sc >= 0x1p-96f && sc <= 0x1p96f) || over) {
#pragma unroll
    for (int e = 0; e < 32; ++e) {
      const float r = sc == 0.f ? 0.f : fminf(fmaxf(rintf(__fdiv_rn(__fsub_rn(x[e], zr), sc)), lo), hi);
      bits[e] = __float_as_uint(r + kRintBias);
    }
  }
}

// Word sums of a quarter's codes at their places (layout.h): sum of (bits[e]
// - kRintBits + off) << shift, the constant part taken off at once.
template <int BITS, bool KEY>
__device__ __forceinline__ void quarter_words(const uint32_t (&bits)[32], uint32_t off, uint32_t (&w)[BITS]) {
  uint32_t c[BITS];
#pragma unroll
  for (int i = 0; i < BITS; ++i) w[i] = c[i] = 0u;
#pragma unroll
  for (int l = 0; l < 32; ++l) {
    int wi, sh;
    if (KEY) {
      int byte, hi;
      k_pos(l, BITS, 128, &byte, &hi);
      wi = BITS == 8 ? 2 * (byte >> 4) + ((byte & 15) >> 2) : byte >> 4;
      sh = 8 * (byte & 3) + 4 * hi;
    } else {
      const int g = l & 7, e = (l >> 3) & 1, hh = l >> 4;
      const int bl = BITS == 8 ? 16 * hh + 2 * g + e : 2 * g + hh;
      wi = bl >> 2;
      sh = 8 * (bl & 3) + (BITS == 4 ? 4 * e : 0);
    }
    w[wi] += bits[l] << sh;
    c[wi] += 1u << sh;
  }
#pragma unroll
  for (int i = 0; i < BITS; ++i) w[i] -= (kRintBits - off) * c[i];
}

// Bulk appends of 8- and 4-bit codes, head_dim 128: a lane quantises 32
// channels (a quarter of a row's keys, then of its values), a warp 8 rows per
// iteration.  A warp per row with 4 channels per lane spent 420 warp
// instructions per row (3 shuffle rounds per extremum, a division per 8 lanes
// of a group, 4 shuffles per packed word); here the extrema stay in
// registers, a group of 32 divides once, the words are summed in place and
// the arithmetic is packed (90 instructions per row).  bf16 inputs come one
// iteration ahead through shared memory: a warp copies its next 8 rows in
// whole 512-byte runs, each lane's 64 bytes to a place of its own, 80 bytes
// apart (no bank conflicts); with plain loads the kernel waited for memory
// most of the time.  At the 14B shape (32 x 2048 x 8 rows) int4 g32: 223 us
// with a warp per row, 89 with plain loads, 72 now (5.1 TB/s of inputs and
// records; issue 57 % busy).
// GS: group (32, 64; 128 for the symmetric scheme's rows); lanes of a group
// meet by 0, 1 or 2 shuffles.  KPC: keys with per-channel groups -- values
// only; the key codes are written when a group of positions completes
// (gqa_append_kgroups) and the lengths advance in the residual kernel.
constexpr int kQuadStage = 2 * 32 * 80;  // a warp's 8 rows, keys and values, one iteration
constexpr int kQuadSmem = 8 * 2 * kQuadStage;
template <int BITS, int GS, bool SYM, bool KPC>
__global__ void __launch_bounds__(256)
    gqa_append_quads(const GqaView v, const void *kin, const void *vin, int in_f32, int n_new,
                     const int32_t *n_per_seq, int32_t *err) {
  pdl_wait();
  pdl_trigger();
  constexpr int SEC = 16 * BITS, NC = BITS;               // bytes and 16-byte chunks per section
  constexpr int MBY = ((128 / GS) * 8 + 15) & ~15;        // one section's group metadata
  constexpr int REC = SYM ? 2 * SEC : 2 * SEC + (KPC ? 1 : 2) * MBY;
  constexpr int KM = 2 * SEC, VM = KPC ? KM : KM + MBY;
  constexpr float LEV = (float)((1 << BITS) - 1), QL = (float)((1 << (BITS - 1)) - 1);
  extern __shared__ __align__(16) uint8_t quads_smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, qc = lane & 3;
  const uint32_t total = (uint32_t)((size_t)v.B * n_new * v.Hkv);  // the launcher sends fewer than 2^31 rows
  const uint32_t step = gridDim.x * 64;
  const RowStep rstep(step, (uint32_t)v.Hkv, (uint32_t)n_new);
  uint32_t row0 = (blockIdx.x * 8 + warp) * 8;
  RowIdx ri = rstep.at(min(row0 + (lane >> 2), total));
  uint8_t *stage = quads_smem + warp * 2 * kQuadStage;
  // the warp's 8 rows from r0 on into a stage, keys then values (bf16)
  auto fetch = [&](uint32_t r0, int s) {
#pragma unroll
    for (int sec = KPC ? 1 : 0; sec < 2; ++sec)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int c = 32 * j + lane;  // 16-byte piece of the 8 rows
        const bool in = r0 + (c >> 4) < total;
        cp_async16(stage + s * kQuadStage + sec * (kQuadStage / 2) + (c >> 2) * 80 + (c & 3) * 16,
                   static_cast<const uint8_t *>(sec ? vin : kin) + (in ? (size_t)r0 * 256 + 16 * c : 0), in);
      }
    cp_async_commit();
  };
  if (!in_f32 && row0 < total) fetch(row0, 0);
  for (int s = 0; row0 < total; row0 += step, ri = rstep.next(ri), s ^= 1) {
    const uint32_t row = row0 + (lane >> 2);
    bool ok = row < total;
    float xk[32], xv[32];
    if (in_f32) {
      const size_t in_off = (size_t)(ok ? row : 0) * 128 + 32 * qc;  // inputs are [B, n_new, H_kv, 128], row `row`
      if constexpr (!KPC) load_quarter(static_cast<const float *>(kin) + in_off, true, xk);
      load_quarter(static_cast<const float *>(vin) + in_off, true, xv);
    } else {
      __syncwarp();  // the stage's last rows are read
      if (row0 + step < total) fetch(row0 + step, s ^ 1);
      else cp_async_commit();
      cp_async_wait<1>();
      __syncwarp();
      const uint8_t *mine = stage + s * kQuadStage + lane * 80;
      if constexpr (!KPC) load_quarter(mine, false, xk);
      load_quarter(mine + kQuadStage / 2, false, xv);
    }
    int t = 0;
    size_t slot = 0;
    if (ok) {
      const int b = (int)ri.b, nb = seq_count(n_per_seq, b, n_new, err);
      t = v.lens[b] + (int)ri.i;
      ok = (int)ri.i < nb;
      if (ok && t >= v.cap) {
        if (qc == 0) set_err(err, 2);
        ok = false;
      }
      if (ok) slot = ((size_t)b * v.Hkv + ri.kvh) * v.cap + t;
    }
    uint8_t *rec = v.rec + slot * REC;
    // physical 16-byte place of a record's logical chunk: symmetric records
    // rotate all chunks by sym_rot(t), grouped ones the V chunks by v_rot(t)
    auto at = [&](int chunk) -> uint4 * {
      const int c = SYM          ? (chunk + sym_rot(t, REC / 16)) & (REC / 16 - 1)
                    : chunk < NC ? chunk
                                 : NC + ((chunk - NC + v_rot(t, REC, NC)) & (NC - 1));
      return reinterpret_cast<uint4 *>(rec) + c;
    };
    uint32_t ssym = 0;
#pragma unroll
    for (int sec = KPC ? 1 : 0; sec < 2; ++sec) {
      const float(&x)[32] = sec ? xv : xk;
      float mn = x[0], mx = x[0];
#pragma unroll
      for (int e = 1; e < 32; ++e) {
        mn = fminf(mn, x[e]);
        mx = fmaxf(mx, x[e]);
      }
#pragma unroll
      for (int o = 1; o < GS / 32; o <<= 1) {
        mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      }
      uint32_t bits[32], w[BITS];
      if constexpr (SYM) {
        const float am = fmaxf(fmaxf(mx, -mn), 0.f);
        const uint16_t sb = f32_to_bf16_bits(__fdiv_rn(am, QL));
        const float s = bf16_to_f32(sb);
        const float top = s == 0.f ? 0.f : __fmul_rn(am, __fdividef(1.f, s));
        quarter_codes(x, s, 0.f, -QL, QL, !(top <= QL + 0.4f), bits);
        ssym |= (uint32_t)sb << (16 * sec);
      } else {
        const float s = __fdiv_rn(__fsub_rn(mx, mn), LEV);
        quarter_codes(x, s, mn, 0.f, LEV, false, bits);
        if (ok && (32 * qc) % GS == 0)
          reinterpret_cast<float2 *>(rec + (sec ? VM : KM))[32 * qc / GS] = make_float2(s, mn);
      }
      constexpr uint32_t off = SYM ? (uint32_t)QL : 0u;
      if (sec) {
        // values: the quarter is BITS / 4 whole chunks
        quarter_words<BITS, false>(bits, off, w);
#pragma unroll
        for (int c = 0; c < BITS / 4; ++c)
          if (ok) *at(NC + BITS / 4 * qc + c) = make_uint4(w[4 * c], w[4 * c + 1], w[4 * c + 2], w[4 * c + 3]);
      } else if constexpr (BITS == 4) {
        // keys: word c belongs to chunk c at place qc; the row's four lanes
        // transpose (two exchanges), lane qc stores chunk qc
        quarter_words<BITS, true>(bits, off, w);
#pragma unroll
        for (int h = 0; h < 2; ++h) {  // pairs (0, 1) and (2, 3) with lane ^ 1
          const uint32_t give = qc & 1 ? w[2 * h] : w[2 * h + 1];
          const uint32_t got = __shfl_xor_sync(0xffffffffu, give, 1);
          if (qc & 1) w[2 * h] = got;
          else w[2 * h + 1] = got;
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {  // pairs (0, 2) and (1, 3) with lane ^ 2
          const uint32_t give = qc & 2 ? w[h] : w[h + 2];
          const uint32_t got = __shfl_xor_sync(0xffffffffu, give, 2);
          if (qc & 2) w[h] = got;
          else w[h + 2] = got;
        }
        if (ok) *at(qc) = make_uint4(w[0], w[1], w[2], w[3]);
      } else {
        // keys: words 2c, 2c + 1 are half qc % 2 of chunk 4 (qc / 2) + c; the
        // even lane of a pair stores chunks c = 0, 1, the odd one c = 2, 3
        quarter_words<BITS, true>(bits, off, w);
        uint32_t g[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) g[i] = __shfl_xor_sync(0xffffffffu, qc & 1 ? w[i] : w[4 + i], 1);
        if (ok) {
          const int c0 = 4 * (qc >> 1) + (qc & 1 ? 2 : 0);
          *at(c0) = qc & 1 ? make_uint4(g[0], g[1], w[4], w[5]) : make_uint4(w[0], w[1], g[0], g[1]);
          *at(c0 + 1) = qc & 1 ? make_uint4(g[2], g[3], w[6], w[7]) : make_uint4(w[2], w[3], g[2], g[3]);
        }
      }
    }
    if (SYM && ok && qc == 0) v.scales[slot] = ssym;
  }
  if constexpr (!KPC) advance_lengths(v, n_new, n_per_seq);
}

// Bulk appends of bf16 caches, head_dim 128: a warp per row, two rows per
// iteration, their loads issued together (rows past the end compute on row
// 0's inputs and store nothing).
__global__ void __launch_bounds__(256)
    gqa_append_bulk_bf16(const GqaView v, const void *kin, const void *vin, int in_f32, int n_new,
                         const int32_t *n_per_seq, int32_t *err) {
  pdl_wait();
  pdl_trigger();
  constexpr int D = 128, E = 4, SEC = 2 * D, REC = 2 * SEC;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int wpb = blockDim.x >> 5;
  const size_t total = (size_t)v.B * n_new * v.Hkv;
  const Gather16 g16(lane);
  const size_t step = (size_t)gridDim.x * wpb;
  // 32-bit index arithmetic (the launcher sends fewer than 2^31 rows)
  const RowStep rstep((uint32_t)step, (uint32_t)v.Hkv, (uint32_t)n_new);
  RowIdx ridx = rstep.at((uint32_t)min((size_t)blockIdx.x * wpb + warp, total));
  for (size_t w0 = (size_t)blockIdx.x * wpb + warp; w0 < total; w0 += 2 * step) {
    bool ok[2];
    size_t row[2];
    float xk[2][E], xv[2][E];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const size_t wid = w0 + u * step;
      const RowIdx r = ridx;
      ridx = rstep.next(ridx);  // row wid + step
      ok[u] = false;
      row[u] = 0;
      size_t in_off = 0;
      if (wid < total) {
        const int kvh = (int)r.kvh, i = (int)r.i, b = (int)r.b;
        in_off = wid * D;  // inputs are [B, n_new, H_kv, D], row wid
        const int nb = seq_count(n_per_seq, b, n_new, err);
        const int t = v.lens[b] + i;
        if (i < nb) {
          if (t >= v.cap) {
            if (lane == 0) set_err(err, 2);
          } else {
            ok[u] = true;
            row[u] = ((size_t)b * v.Hkv + kvh) * v.cap + t;
          }
        }
      }
      load_row<D>(kin, vin, in_f32, in_off, lane, xk[u], xv[u]);
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      uint8_t *rec = v.rec + row[u] * REC;
      const uint32_t k0 = pack2<true>(xk[u][0], xk[u][1]), k1 = pack2<true>(xk[u][2], xk[u][3]);
      const uint32_t v0 = pack2<true>(xv[u][0], xv[u][1]), v1 = pack2<true>(xv[u][2], xv[u][3]);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const uint32_t kw = g16.kword(k0, k1, h), vw = g16.vword(v0, v1, h);
        if (ok[u]) {
          reinterpret_cast<uint32_t *>(rec)[lane + 32 * h] = kw;
          reinterpret_cast<uint32_t *>(rec + SEC)[lane + 32 * h] = vw;
        }
      }
    }
  }
  advance_lengths(v, n_new, n_per_seq);
}

// Short appends (a decode step: n_new x H_kv <= 64 rows per sequence,
// per-token layouts): one CTA of 8 warps per sequence.  The CTA reads the
// length once while the warps' first input loads are in flight, writes all
// rows of its sequence and then advances the length itself -- no other CTA
// reads it, so no completion counter or fence is needed.
template <int D>
__global__ void __launch_bounds__(256)
    gqa_append_seq(const GqaView v, const void *kin, const void *vin, int in_f32, int n_new,
                   const int32_t *n_per_seq, int32_t *err) {
  pdl_wait();
  pdl_trigger();
  constexpr int E = D / 32;
  __shared__ __align__(16) uint32_t sbuf[8][(2 * D * 2 + 2 * 64) / 4];
  __shared__ int s_len, s_nb;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int b = blockIdx.x;
  const int rows = n_new * v.Hkv;
  float xk[E], xv[E];
  if (warp < rows)
    load_row<D>(kin, vin, in_f32, ((size_t)b * n_new * v.Hkv + warp) * D, lane, xk, xv);
  if (threadIdx.x == 0) {
    s_nb = seq_count(n_per_seq, b, n_new, err);
    s_len = v.lens[b];
  }
  __syncthreads();
  const int len = s_len, nb = s_nb;
  for (int r = warp; r < rows; r += 8) {
    const int i = r / v.Hkv, kvh = r - i * v.Hkv;
    if (r != warp)
      load_row<D>(kin, vin, in_f32, ((size_t)b * n_new * v.Hkv + r) * D, lane, xk, xv);
    if (i >= nb) continue;
    const int t = len + i;
    if (t >= v.cap) {
      if (lane == 0) set_err(err, 2);
      continue;
    }
    append_row<D>(v, xk, xv, b, kvh, t, sbuf[warp], lane);
  }
  __syncthreads();
  if (threadIdx.x == 0) v.lens[b] = min((long long)len + nb, (long long)v.cap);
}

// Per-channel key groups completed by this append: one CTA of 128 threads per
// (sequence, KV head, group of GS positions).  The group's keys (residual
// rows for positions already stored, the appended rows for new ones, rounded
// to bf16 as the residual holds them) are staged in natural channel order in
// shared memory; the channel pairs {c, c + 8} (c = 16 (p / 8) + p % 8: the two
// channels of one 4-bit byte) are shared by 128 / (D / 2) threads that take
// a part of the positions each and meet over their extrema: scale = fl((max
// - min) / levels) correctly rounded, codes rint((x - min) / scale) by
// residual steps (quarter_codes; the division for scales out of their
// range), packed into the
// positions' key sections in shared memory and stored as whole 16-byte
// chunks.  Bound by the latency of that chain: a warp per group, with two
// passes over all positions, took 48 us for a single group per (sequence, KV
// head) and held 8 warps per SM by its shared memory.
constexpr int kKgThreads = 128;
// dynamic shared memory of gqa_append_kgroups: the staged keys (GS rows of
// D + 8 bf16) and the key sections (GS rows of D bits / 8 bytes)
__host__ __device__ constexpr int kg_bytes(int D, int GS, int bits) {
  return ((GS * (D + 8) * 2 + GS * D * bits / 8) + 15) & ~15;
}
template <int D>
__global__ void __launch_bounds__(kKgThreads)
    gqa_append_kgroups(const GqaView v, const void *kin, int in_f32, int n_new,
                       const int32_t *n_per_seq, int max_groups) {
  pdl_wait();
  pdl_trigger();
  constexpr int PAD = D + 8;                      // bf16 per staged row (conflict-free columns)
  constexpr int PAIRS = D / 2, PARTS = kKgThreads / PAIRS;
  extern __shared__ __align__(16) uint8_t kg_smem[];
  __shared__ float s_mn[kKgThreads][2], s_mx[kKgThreads][2];
  const int tid = threadIdx.x;
  const size_t wid = blockIdx.x;
  const int gidx = (int)(wid % max_groups);
  const int kvh = (int)((wid / max_groups) % v.Hkv);
  const int b = (int)(wid / ((size_t)max_groups * v.Hkv));
  const int GS = v.group;
  const int nb = seq_count(n_per_seq, b, n_new, nullptr);
  const int len0 = v.lens[b];
  const int G = len0 / GS + gidx;  // candidate group
  if ((G + 1) * GS > len0 + nb || (G + 1) * GS > v.cap) return;  // not completed now (CTA-uniform)
  const size_t slab = (size_t)b * v.Hkv + kvh;
  const RecLayout L = rec_layout(v.bits, D, GS, 1);
  const int sec = D * v.bits / 8;
  const uint8_t *res = v.resid + slab * (size_t)GS * D * 2;
  uint16_t *xs = reinterpret_cast<uint16_t *>(kg_smem);
  uint8_t *ks = kg_smem + GS * PAD * 2;
  // ---- the group's keys, natural channel order ----
  constexpr int CPR = D / 8;  // 8-channel pieces per row
#pragma unroll 4
  for (int q = tid; q < GS * CPR; q += kKgThreads) {
    const int r = q / CPR, c8 = 8 * (q - r * CPR);
    const int p = G * GS + r;
    uint4 o;
    if (p < len0) {
      // residual row r: bf16 in the key fragment order (channels 2 i, 2 i + 1
      // of a piece are neighbours)
      uint32_t w[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        int kb, khi;
        k_pos(c8 + 2 * e, 16, D, &kb, &khi);
        w[e] = *reinterpret_cast<const uint32_t *>(res + (size_t)r * D * 2 + kb);
      }
      o = make_uint4(w[0], w[1], w[2], w[3]);
    } else {
      const size_t ii = (((size_t)b * n_new + (p - len0)) * v.Hkv + kvh) * D + c8;
      if (in_f32) {
        const float4 *src = reinterpret_cast<const float4 *>(static_cast<const float *>(kin) + ii);
        const float4 u0 = src[0], u1 = src[1];
        o = make_uint4(pack_bf16(u0.x, u0.y), pack_bf16(u0.z, u0.w), pack_bf16(u1.x, u1.y), pack_bf16(u1.z, u1.w));
      } else {
        o = *reinterpret_cast<const uint4 *>(static_cast<const uint16_t *>(kin) + ii);
      }
    }
    *reinterpret_cast<uint4 *>(xs + r * PAD + c8) = o;
  }
  __syncthreads();
  // ---- per channel: scale, zero, codes ----
  const float lev = (float)((1 << v.bits) - 1);
  const int pr = tid % PAIRS, part = tid / PAIRS;
  const int ch0 = (pr >> 3) * 16 + (pr & 7);
  const int r0 = part * GS / PARTS, r1 = (part + 1) * GS / PARTS;
  float mn[2] = {INFINITY, INFINITY}, mx[2] = {-INFINITY, -INFINITY};
#pragma unroll 4
  for (int r = r0; r < r1; ++r)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float x = bf16_to_f32(xs[r * PAD + ch0 + 8 * h]);
      mn[h] = fminf(mn[h], x);
      mx[h] = fmaxf(mx[h], x);
    }
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    s_mn[tid][h] = mn[h];
    s_mx[tid][h] = mx[h];
  }
  __syncthreads();
  float sc[2], zr[2], rs[2];
  bool wide[2];  // a scale out of the residual steps' range (quarter_codes)
#pragma unroll
  for (int h = 0; h < 2; ++h) {
#pragma unroll
    for (int o = 0; o < PARTS; ++o) {
      mn[h] = fminf(mn[h], s_mn[o * PAIRS + pr][h]);
      mx[h] = fmaxf(mx[h], s_mx[o * PAIRS + pr][h]);
    }
    sc[h] = __fdiv_rn(__fsub_rn(mx[h], mn[h]), lev);
    zr[h] = mn[h];
    rs[h] = __frcp_rn(sc[h]);
    wide[h] = !(sc[h] >= 0x1p-96f && sc[h] <= 0x1p96f);
    if (part == 0) v.gmeta[(slab * (v.cap / GS) + G) * D + ch0 + 8 * h] = make_float2(sc[h], mn[h]);
  }
  int kb0, kh0, kb1, kh1;
  k_pos(ch0, v.bits, D, &kb0, &kh0);
  k_pos(ch0 + 8, v.bits, D, &kb1, &kh1);
#pragma unroll 2
  for (int r = r0; r < r1; ++r) {
    uint32_t c[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float d = __fsub_rn(bf16_to_f32(xs[r * PAD + ch0 + 8 * h]), zr[h]);
      float q = __fmul_rn(d, rs[h]);
      q = fmaf(fmaf(q, -sc[h], d), rs[h], q);
      q = fmaf(fmaf(q, -sc[h], d), rs[h], q);
      if (wide[h]) q = sc[h] == 0.f ? 0.f : __fdiv_rn(d, sc[h]);
      c[h] = (uint32_t)fminf(fmaxf(rintf(q), 0.f), lev);
    }
    if (v.bits == 8) {
      ks[r * sec + kb0] = (uint8_t)c[0];
      ks[r * sec + kb1] = (uint8_t)c[1];
    } else {
      // channels ch0 and ch0 + 8 share one byte (low and high nibble)
      ks[r * sec + kb0] = (uint8_t)(c[0] | (c[1] << 4));
    }
  }
  __syncthreads();
  // ---- the group's key sections, whole 16-byte chunks ----
  const int cps = sec / 16;
  for (int q = tid; q < GS * cps; q += kKgThreads) {
    const int r = q / cps, u = q - r * cps;
    uint8_t *rec = v.rec + (slab * v.cap + (size_t)G * GS + r) * L.rec + L.k_off;
    reinterpret_cast<uint4 *>(rec)[u] = reinterpret_cast<const uint4 *>(ks + r * sec)[u];
  }
}

// Positions of the group left open after this append go to the residual
// plane; block b then advances sequence b's length.  A thread takes eight
// channels (16 or 32 bytes) at a time: 63 open positions of 8 KV heads took
// 128 threads of one element each 102 us.
template <int D>
__global__ void __launch_bounds__(1024)
    gqa_append_kresid(const GqaView v, const void *kin, int in_f32, int n_new,
                      const int32_t *n_per_seq) {
  pdl_wait();
  pdl_trigger();
  const int b = blockIdx.x;
  const int GS = v.group;
  const int nb = seq_count(n_per_seq, b, n_new, nullptr);
  const int len0 = v.lens[b];
  const int len1 = min(len0 + nb, (int)v.cap);
  const int open0 = (len1 / GS) * GS;  // first position of the open group
  const int first = max(open0, len0);
  const int rows = len1 - first;
  constexpr int PCS = D / 8;  // 8-channel pieces per row
  const int work = rows * v.Hkv * PCS;
  for (int q = threadIdx.x; q < work; q += blockDim.x) {
    const int c8 = 8 * (q % PCS), row = q / PCS;
    const int kvh = row % v.Hkv, p = first + row / v.Hkv;
    const size_t ii = (((size_t)b * n_new + (p - len0)) * v.Hkv + kvh) * D + c8;
    uint32_t w[4];  // bf16 pairs of channels c8 + 2 i, + 1
    if (in_f32) {
      const float4 *src = reinterpret_cast<const float4 *>(static_cast<const float *>(kin) + ii);
      const float4 u0 = src[0], u1 = src[1];
      w[0] = pack_bf16(u0.x, u0.y); w[1] = pack_bf16(u0.z, u0.w);
      w[2] = pack_bf16(u1.x, u1.y); w[3] = pack_bf16(u1.z, u1.w);
    } else {
      const uint4 u = *reinterpret_cast<const uint4 *>(static_cast<const uint16_t *>(kin) + ii);
      w[0] = u.x; w[1] = u.y; w[2] = u.z; w[3] = u.w;
    }
    uint8_t *res = v.resid + ((size_t)b * v.Hkv + kvh) * GS * D * 2 + (size_t)(p % GS) * D * 2;
#pragma unroll
    for (int i = 0; i < 4; ++i) {  // channels 2 i, 2 i + 1 of a piece are neighbours in the fragment order
      int kb, khi;
      k_pos(c8 + 2 * i, 16, D, &kb, &khi);
      *reinterpret_cast<uint32_t *>(res + kb) = w[i];
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) v.lens[b] = len1;
}

// bf16 MLA rows, a warp each, 16 bytes per lane (widths, latent_dim and
// rope_dim are multiples of 8 and the inputs 16-byte aligned): one token of
// 64 sequences at d = 512 took 10.4 us by elements.
__global__ void __launch_bounds__(128)
    mla_append_rows(const MlaView v, const uint16_t *c, const uint16_t *kr, int latent, int n_new,
                    const int32_t *n_per_seq, int32_t *err) {
  pdl_wait();
  pdl_trigger();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (size_t wid = (size_t)blockIdx.x * 4 + warp; wid < (size_t)v.B * n_new;
       wid += (size_t)gridDim.x * 4) {
    const int i = (int)(wid % n_new), b = (int)(wid / n_new);
    const int nb = seq_count(n_per_seq, b, n_new, err);
    const int t = v.lens[b] + i;
    bool ok = i < nb;
    if (ok && t >= v.cap) {
      if (lane == 0) set_err(err, 2);
      ok = false;
    }
    if (ok) {
      uint4 *rec = reinterpret_cast<uint4 *>(v.rec + ((size_t)b * v.cap + t) * v.rec_bytes);
      const uint4 *cs = reinterpret_cast<const uint4 *>(c + ((size_t)b * n_new + i) * latent);
      const uint4 *ks = reinterpret_cast<const uint4 *>(kr + ((size_t)b * n_new + i) * v.rope);
      const int nc = v.width / 8, n = nc + v.rope / 8;  // the first `width` coordinates, then k^R
      for (int e = lane; e < n; e += 32) rec[e] = e < nc ? cs[e] : ks[e - nc];
    }
  }
  __syncthreads();
  __shared__ int last;
  if (threadIdx.x == 0) {
    __threadfence();
    last = (atomicAdd(v.counter, 1) == (int)gridDim.x - 1);
  }
  __syncthreads();
  if (last) {
    for (int b = threadIdx.x; b < v.B; b += blockDim.x) {
      const int nb = seq_count(n_per_seq, b, n_new, nullptr);
      v.lens[b] = min((long long)v.lens[b] + nb, (long long)v.cap);
    }
    if (threadIdx.x == 0) *v.counter = 0;
  }
}

// Quantised MLA append (the layout in layout.h): one warp per (sequence,
// new position); the kept latent c[:W] and the positional key are each
// quantised as one vector (symmetric: one bf16 scale; grouped: one fp32
// scale and zero), codes staged in shared memory and stored chunk by chunk.
template <int W>
__global__ void __launch_bounds__(128)
    mla_append_q(const MlaView v, const uint16_t *c, const uint16_t *kr, int latent, int n_new,
                 const int32_t *n_per_seq, int32_t *err) {
  pdl_wait();
  pdl_trigger();
  constexpr int R = 64, KH = W + R, EC = W / 32, ER = R / 32;
  __shared__ uint8_t buf[4][KH];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (size_t wid = (size_t)blockIdx.x * 4 + warp; wid < (size_t)v.B * n_new;
       wid += (size_t)gridDim.x * 4) {
    const int i = (int)(wid % n_new), b = (int)(wid / n_new);
    const int nb = seq_count(n_per_seq, b, n_new, err);
    const int t = v.lens[b] + i;
    bool ok = i < nb;
    if (ok && t >= v.cap) {
      if (lane == 0) set_err(err, 2);
      ok = false;
    }
    if (ok) {
      const uint16_t *cs = c + ((size_t)b * n_new + i) * latent;
      const uint16_t *ks = kr + ((size_t)b * n_new + i) * R;
      float xc[EC], xr[ER];
#pragma unroll
      for (int e = 0; e < EC; ++e) xc[e] = bf16_to_f32(cs[lane + 32 * e]);
#pragma unroll
      for (int e = 0; e < ER; ++e) xr[e] = bf16_to_f32(ks[lane + 32 * e]);
      uint32_t uc[EC], ur[ER];
      if (v.scheme == kSchemeSym) {
        const uint16_t sc = quant_sym_lane<EC>(xc, v.bits, uc);
        const uint16_t sr = quant_sym_lane<ER>(xr, v.bits, ur);
        if (lane == 0)
          reinterpret_cast<uint32_t *>(v.meta)[(size_t)b * v.cap + t] = (uint32_t)sc | ((uint32_t)sr << 16);
      } else {
        const int lev = (1 << v.bits) - 1;
        float sc, zc, sr, zr;
        quant_lane<EC>(xc, W, lev, uc, sc, zc);
        quant_lane<ER>(xr, R, lev, ur, sr, zr);
        if (lane == 0)
          reinterpret_cast<float4 *>(v.meta)[(size_t)b * v.cap + t] = make_float4(sc, zc, sr, zr);
      }
#pragma unroll
      for (int e = 0; e < EC; ++e) buf[warp][lane + 32 * e] = (uint8_t)uc[e];
#pragma unroll
      for (int e = 0; e < ER; ++e) buf[warp][W + lane + 32 * e] = (uint8_t)ur[e];
      __syncwarp();
      uint8_t *rec = v.rec + ((size_t)b * v.cap + t) * v.rec_bytes;
      for (int j = lane; j < KH / 8; j += 32) {
        const uint8_t *cd = buf[warp] + 8 * j;
        if (v.bits == 8) {
          uint2 w;
          w.x = cd[0] | (cd[1] << 8) | (cd[2] << 16) | ((uint32_t)cd[3] << 24);
          w.y = cd[4] | (cd[5] << 8) | (cd[6] << 16) | ((uint32_t)cd[7] << 24);
          reinterpret_cast<uint2 *>(rec)[j] = w;
        } else if (v.bits == 4) {
          uint32_t w = 0;
#pragma unroll
          for (int k = 0; k < 8; ++k) w |= (uint32_t)cd[k] << mla_q_bit(k, 4);
          reinterpret_cast<uint32_t *>(rec)[j] = w;
        } else {
          uint32_t w = 0;
#pragma unroll
          for (int k = 0; k < 8; ++k) w |= (uint32_t)cd[k] << mla_q_bit(k, 2);
          reinterpret_cast<uint16_t *>(rec)[j] = (uint16_t)w;
        }
      }
    }
    __syncwarp();  // the row buffer is free again
  }
  __syncthreads();
  __shared__ int last;
  if (threadIdx.x == 0) {
    __threadfence();
    last = (atomicAdd(v.counter, 1) == (int)gridDim.x - 1);
  }
  __syncthreads();
  if (last) {
    for (int b = threadIdx.x; b < v.B; b += blockDim.x) {
      const int nb = seq_count(n_per_seq, b, n_new, nullptr);
      v.lens[b] = min((long long)v.lens[b] + nb, (long long)v.cap);
    }
    if (threadIdx.x == 0) *v.counter = 0;
  }
}

// CTAs of `wpc` rows for `rows` rows: one per wpc rows, up to `ctas_per_sm`
// per SM of the current device; the kernels loop over the rest
unsigned row_blocks(size_t rows, int wpc = 4, int ctas_per_sm = 16) {
  static int sms = 0;
  if (!sms) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0)
      sms = 148;
  }
  const size_t need = (rows + wpc - 1) / wpc, cap = (size_t)sms * ctas_per_sm;
  return (unsigned)(need < cap ? (need > 0 ? need : 1) : cap);
}

}  // namespace

cudaError_t launch_gqa_append(const GqaView &v, const void *k, const void *vv, int in_f32,
                              int n_new, const int32_t *n_per_seq, int32_t *err,
                              cudaStream_t st) {
  const size_t rows = (size_t)v.B * n_new * v.Hkv;
  const unsigned blocks = row_blocks(rows);
  const bool kpc = v.bits != 16 && v.key_axis == 1;
  const bool d128 = v.D == 128;
  cudaError_t e = cudaSuccess;
  if (kpc) {
    // groups first (they read residual rows the open group may overwrite)
    const int max_groups = (n_new + v.group - 1) / v.group + 1;
    const dim3 grid((unsigned)((size_t)v.B * v.Hkv * max_groups));
    auto kern = d128 ? gqa_append_kgroups<128> : gqa_append_kgroups<64>;
    // at most 25.6 KB (head_dim 128, groups of 64, 8-bit codes)
    e = launch_pdl(kern, grid, dim3(kKgThreads), (size_t)kg_bytes(v.D, v.group, v.bits), st, v, k, in_f32, n_new,
                   n_per_seq, max_groups);
  }
  if (e == cudaSuccess) {
    // bulk appends (head_dim 128): a warp per row for bf16, a lane per 32
    // channels for 8- and 4-bit codes
    const bool bulk = (size_t)n_new * v.Hkv > 64 && d128 && rows < (1u << 31);
    const bool sym = v.scheme == kSchemeSym;
    auto quads = [&](auto kern) {
      cudaError_t r = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kQuadSmem);
      if (r != cudaSuccess) return r;
      return launch_pdl(kern, dim3(row_blocks(rows, 64, 2)), dim3(256), kQuadSmem, st, v, k, vv, in_f32, n_new,
                        n_per_seq, err);
    };
    if (bulk && v.bits == 16) {
      e = launch_pdl(gqa_append_bulk_bf16, dim3(row_blocks(rows, 8, 8)), dim3(256), 0, st, v, k, vv, in_f32, n_new,
                     n_per_seq, err);
    } else if (bulk && (v.bits == 8 || v.bits == 4)) {
      const bool g32 = v.group == 32;
      if (sym) e = v.bits == 8 ? quads(gqa_append_quads<8, 128, true, false>) : quads(gqa_append_quads<4, 128, true, false>);
      else if (kpc && v.bits == 8) e = g32 ? quads(gqa_append_quads<8, 32, false, true>) : quads(gqa_append_quads<8, 64, false, true>);
      else if (kpc) e = g32 ? quads(gqa_append_quads<4, 32, false, true>) : quads(gqa_append_quads<4, 64, false, true>);
      else if (v.bits == 8) e = g32 ? quads(gqa_append_quads<8, 32, false, false>) : quads(gqa_append_quads<8, 64, false, false>);
      else e = g32 ? quads(gqa_append_quads<4, 32, false, false>) : quads(gqa_append_quads<4, 64, false, false>);
    } else if (!kpc && (size_t)n_new * v.Hkv <= 64)
      e = launch_pdl(d128 ? gqa_append_seq<128> : gqa_append_seq<64>, dim3(v.B), dim3(256), 0, st,
                     v, k, vv, in_f32, n_new, n_per_seq, err);
    else
      e = launch_pdl(d128 ? gqa_append_rows<128> : gqa_append_rows<64>, dim3(blocks), dim3(128), 0,
                     st, v, k, vv, in_f32, n_new, n_per_seq, err);
  }
  if (e == cudaSuccess && kpc)
    e = launch_pdl(d128 ? gqa_append_kresid<128> : gqa_append_kresid<64>, dim3(v.B), dim3(1024), 0,
                   st, v, k, in_f32, n_new, n_per_seq);
  return e;
}

cudaError_t launch_mla_append(const MlaView &v, const void *c, const void *kr, int latent,
                              int n_new, const int32_t *n_per_seq, int32_t *err,
                              cudaStream_t st) {
  const size_t rows = (size_t)v.B * n_new;
  const dim3 grid(row_blocks(rows));
  const uint16_t *cc = static_cast<const uint16_t *>(c), *kk = static_cast<const uint16_t *>(kr);
  if (v.bits != 16) {
    if (v.rope != 64) return cudaErrorInvalidValue;
    switch (v.width) {
      case 512: return launch_pdl(mla_append_q<512>, grid, dim3(128), 0, st, v, cc, kk, latent, n_new, n_per_seq, err);
      case 256: return launch_pdl(mla_append_q<256>, grid, dim3(128), 0, st, v, cc, kk, latent, n_new, n_per_seq, err);
      case 128: return launch_pdl(mla_append_q<128>, grid, dim3(128), 0, st, v, cc, kk, latent, n_new, n_per_seq, err);
      case 64: return launch_pdl(mla_append_q<64>, grid, dim3(128), 0, st, v, cc, kk, latent, n_new, n_per_seq, err);
      default: return cudaErrorInvalidValue;
    }
  }
  return launch_pdl(mla_append_rows, grid, dim3(128), 0, st, v, cc, kk, latent, n_new, n_per_seq, err);
}

}  // namespace kvk
