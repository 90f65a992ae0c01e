// Quantize-and-pack of residual-window blocks (Eq. 1, 2, 12; Algorithm 2) and
// the window append.  One warp quantizes a tile of one (sequence, kv head) for keys or
// for values.
//
// The fp32 arithmetic uses the *_rn intrinsics so that no multiply-add is ever
// contracted: codes, scales and zero-points are compared bit for bit with a CPU
// evaluation of the same formulas.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "xq_internal.h"
#include "xq_layout.cuh"

namespace xq {

__device__ __forceinline__ float bf16_bits(uint16_t u) { return __uint_as_float(((uint32_t)u) << 16); }

// The 16-bit input type: widening to fp32 (exact) and packed min / max of two elements.
template <bool F16>
struct In16;
template <>
struct In16<false> {
  using V2 = __nv_bfloat162;
  static __device__ __forceinline__ float lo(uint32_t w) { return __uint_as_float(w << 16); }
  static __device__ __forceinline__ float hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }
  static __device__ __forceinline__ float one(uint16_t u) { return bf16_bits(u); }
  // pattern of the nearest 16-bit value (of x itself when it is one)
  static __device__ __forceinline__ uint32_t bits(float x) { return (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(x)); }
  // the nearest 16-bit value at or above x: a bfloat16 is the upper half of a float, and cutting the lower half off
  // moves a negative number up, a positive one down
  static __device__ __forceinline__ uint32_t bits_up(float x) {
    const uint32_t b = __float_as_uint(x);
    return (b + ((int)b < 0 ? 0u : 0xffffu)) >> 16;
  }
};
template <>
struct In16<true> {
  using V2 = __half2;
  static __device__ __forceinline__ float lo(uint32_t w) { return __half2float(__ushort_as_half((unsigned short)(w & 0xffffu))); }
  static __device__ __forceinline__ float hi(uint32_t w) { return __half2float(__ushort_as_half((unsigned short)(w >> 16))); }
  static __device__ __forceinline__ float one(uint16_t u) { return __half2float(__ushort_as_half(u)); }
  static __device__ __forceinline__ uint32_t bits(float x) { return (uint32_t)__half_as_ushort(__float2half_rn(x)); }
  static __device__ __forceinline__ uint32_t bits_up(float x) { return (uint32_t)__half_as_ushort(__float2half_ru(x)); }
};

// Merged words of a sharing pair (Appendix F): field by field, the code of (e0, e1) from the table.
template <int BITS>
__device__ __forceinline__ uint32_t merge_words(uint32_t w0, uint32_t w1, uint32_t lut) {
  uint32_t out = 0u;
#pragma unroll
  for (int f = 0; f < 32; f += BITS) {
    const uint32_t e0 = (w0 >> f) & ((1u << BITS) - 1u), e1 = (w1 >> f) & ((1u << BITS) - 1u);
    out |= ((lut >> (2u * (4u * e0 + e1))) & ((1u << BITS) - 1u)) << f;
  }
  return out;
}

// Eq. 1 and Eq. 12 for one group: z = min, s = (max - min)/(2^B - 1),
// z_hat = z + (eta * s) * (2^B - 1), s_hat = (1 - 2 eta) * s.
__device__ __forceinline__ void group_params(float mn, float mx, int bits, float eta, float& z, float& s,
                                             __half& zh, __half& sh) {
  const float qmax = (float)((1 << bits) - 1);
  s = __fsub_rn(mx, mn);
  if (bits == 2) {
    // RN(a / 3) by the correction step below (`Quot`); tiny and huge ranges, which could leave the normal range on the
    // way, take the division
    const float a = s, third = __uint_as_float(0x3eaaaaabu);  // RN(1 / 3)
    const uint32_t e = (__float_as_uint(a) >> 23) & 0xffu;
    const float q = __fmul_rn(a, third);
    s = __fmaf_rn(__fmaf_rn(-3.0f, q, a), third, q);
    if (e < 40u || e > 210u) s = a == 0.0f ? 0.0f : __fdiv_rn(a, 3.0f);
  }
  z = mn;
  float t = __fmul_rn(__fmul_rn(eta, s), qmax);
  zh = __float2half_rn(__fadd_rn(z, t));
  float k = __fsub_rn(1.0f, __fmul_rn(2.0f, eta));
  sh = __float2half_rn(__fmul_rn(k, s));
}

constexpr int PACK_THREADS = 128;

// 1/s for the quotient sequence of `quotient`: 0 for a constant group (every code 0), NaN where that sequence is
// not known to round correctly -- a scale whose significand is all ones, or one so small or large that an
// intermediate could leave the normal range -- which sends the group to the division.
__device__ __forceinline__ float safe_rcp(float s) {
  if (s == 0.0f) return 0.0f;
  const uint32_t b = __float_as_uint(s);
  const uint32_t e = (b >> 23) & 0xffu;
  if ((b & 0x7fffffu) == 0x7fffffu || e < 40u || e > 210u) return __uint_as_float(0x7fc00000u);
  return __frcp_rn(s);
}

// Codes by comparison (Eq. 2).  The code of x in a group, c(x) = clamp(rint(RN(RN(x - z) / s)), 0, 2^B - 1), never
// decreases with x, and x is a 16-bit float, so the group's codes are fixed by B-bit-many thresholds on the input
// lattice: X_k = the smallest 16-bit value with c(X_k) >= k, and c(x) = #{k : x >= X_k}.  One thread per group
// finds the X_k: next to z + (k - 1/2) s, from the rounding bounds of the quotient where they decide, else by
// evaluating c itself (the quotient exactly as the division gives it, ties of rint to even) at lattice points; the
// elements are then coded two at a time with packed 16-bit compares.

// 16-bit float pattern <-> integer that orders like the value (sign-magnitude to two's complement; -0 and +0 -> 0)
__device__ __forceinline__ int ord16(uint32_t h) {
  const int m = (int)(h & 0x7fffu);
  return (h & 0x8000u) ? -m : m;
}
__device__ __forceinline__ uint32_t pat16(int o) { return o >= 0 ? (uint32_t)o : (0x8000u | (uint32_t)(-o)); }

// A group's uncalibrated parameters for the quotient RN(RN(x - z) / s).  With y = RN(1/s): q = RN(a y),
// r = a - q s (exact in one fused multiply-add), q' = RN(q + r y) is the correctly rounded quotient (the classical
// correction step of division by a correctly rounded reciprocal; the scales it can miss get a NaN from safe_rcp
// and take the division).
struct Quot {
  float z, s, y;
  bool fast;
};
__device__ __forceinline__ float quotient(const Quot& g, float x) {
  const float a = __fsub_rn(x, g.z);
  if (g.fast) {
    const float q = __fmul_rn(a, g.y);
    const float r = __fmaf_rn(-q, g.s, a);
    return __fmaf_rn(r, g.y, q);
  }
  return __fdiv_rn(a, g.s);
}

// X_k as a 16-bit pattern for a group with minimum mn and maximum mx.  In real numbers the threshold is
// tau = z + (k - 1/2) s.  The computed quotient differs from (x - z) / s by less than 2^-23 relative (two
// roundings), i.e. by less than 3.1 * 2^-23 s in x, and t = RN(tau) from tau by at most 2^-24 |t|: a lattice point
// at or above t + eps certainly has c >= k, one below t - eps certainly has not, for eps = 2^-22 |t| + 2^-20 s
// (twice what is needed).  Where the lattice is coarser than eps -- almost always -- no lattice point lies between
// the bounds and nothing is evaluated; otherwise (a threshold next to zero under a large |z|, an exact tie on the
// lattice) c itself decides, by bisection between the bounds.  Groups whose scale takes the division (safe_rcp)
// are bisected from the group's ends (c(mn) = 0, c(mx) = 2^B - 1).
template <bool F16>
__device__ __noinline__ uint32_t bisect16(float z, float sc, float y, int k, int lo, int hi) {
  const Quot g{z, sc, y, y == y};
  const float kk = (float)k - 0.5f;
  const bool even = (k & 1) == 0;  // rint takes a tie to the even neighbour: k - 1/2 counts as >= k only for even k
  while (hi - lo > 1) {
    const int mid = lo + ((hi - lo) >> 1);
    const float q = quotient(g, In16<F16>::one((uint16_t)pat16(mid)));
    if (even ? q >= kk : q > kk) hi = mid; else lo = mid;
  }
  return pat16(hi);
}
template <bool F16>
__device__ __forceinline__ uint32_t threshold16(const Quot& g, int k, float mn, float mx) {
  const float kk = (float)k - 0.5f;
  int lo, hi;  // ordered integers of lattice points with c(lo) < k <= c(hi)
  if (g.fast) {
    const float t = __fmaf_rn(kk, g.s, g.z);
    const float eps = __fmaf_rn(fabsf(t), 0x1p-22f, __fmul_rn(g.s, 0x1p-20f));
    // the smallest lattice points at or above t + eps and at or above t - eps: the same point when no lattice
    // point lies between the two bounds, and then it is X_k (mn lies below t - eps, mx above t + eps: the
    // thresholds are half a step and more away from both)
    const uint32_t up = In16<F16>::bits_up(__fadd_ru(t, eps)), up_lo = In16<F16>::bits_up(__fadd_rd(t, -eps));
    constexpr uint32_t INF16 = F16 ? 0x7c00u : 0x7f80u;
    if (up == up_lo && up != INF16) return up;
    hi = up != INF16 ? ord16(up) : ord16(In16<F16>::bits(mx));  // (a bound beyond the largest finite value)
    lo = ord16(up_lo) - 1;  // below t - eps
  } else {
    lo = ord16(In16<F16>::bits(mn));
    hi = ord16(In16<F16>::bits(mx));
  }
  return bisect16<F16>(g.z, g.s, g.y, k, lo, hi);
}

// The thresholds X_1 .. X_3 of a group with minimum mn and maximum mx (16-bit values, widened); unused ones (k beyond
// 2^B - 1, or a constant group: every code 0) are +infinity.
template <bool F16>
__device__ __forceinline__ void group_thresholds(float mn, float mx, float z, float sc, int bits, uint32_t (&thr)[3]) {
  constexpr uint32_t INF16 = F16 ? 0x7c00u : 0x7f80u;
  const float y = safe_rcp(sc);
  const Quot g{z, sc, y, y == y};
#pragma unroll
  for (int k = 0; k < 3; ++k) thr[k] = INF16;
  if (sc != 0.0f) {
#pragma unroll 1
    for (int k = 1; k < 1 << bits; ++k) {  // (rolled: the code of a threshold is long, and there is one loop for all)
      const uint32_t x = threshold16<F16>(g, k, mn, mx);
      if (k == 1) thr[0] = x; else if (k == 2) thr[1] = x; else thr[2] = x;
    }
  }
}

// Codes of two packed 16-bit elements against their groups' packed thresholds: code of the low element at bit 0,
// of the high element at bit 16.
template <int BITS, typename V2>
__device__ __forceinline__ uint32_t code_pair(uint32_t x, uint32_t t1, uint32_t t2, uint32_t t3) {
  const V2 xv = *reinterpret_cast<const V2*>(&x);
  const uint32_t m1 = __hge2_mask(xv, *reinterpret_cast<const V2*>(&t1));
  if constexpr (BITS == 1) {
    return m1 & 0x00010001u;
  } else {
    const uint32_t m2 = __hge2_mask(xv, *reinterpret_cast<const V2*>(&t2));
    const uint32_t m3 = __hge2_mask(xv, *reinterpret_cast<const V2*>(&t3));
    // A mask is 0xffff per element that passed.  n = -(m1 + m2 + m3) holds the low element's count in its low
    // half and (high count - low count) in its high half (the low half borrows); n * 0x10001 adds the low count
    // back to the high half.
    const uint32_t n = 0u - m1 - m2 - m3;
    return n * 0x10001u;
  }
}

// Adds to hist[d] the number of fields of the two words whose codes differ by d.
template <int BITS>
__device__ __forceinline__ void delta_count(uint32_t w0, uint32_t w1, uint32_t (&hist)[4]) {
#pragma unroll
  for (int f = 0; f < 32; f += BITS) {
    const int e0 = (int)((w0 >> f) & ((1u << BITS) - 1u)), e1 = (int)((w1 >> f) & ((1u << BITS) - 1u));
    const int d = e0 > e1 ? e0 - e1 : e1 - e0;
#pragma unroll
    for (int k = 0; k < (1 << BITS); ++k) hist[k] += d == k;
  }
}

// ---------------------------------------------------------------------------
// One warp quantizes one tile that it holds in registers: nothing goes through shared memory and no warp waits for
// another.  Keys: G tokens x C channels; a lane has 16 consecutive channels (a whole code word, or half of a 1-bit one)
// of every TS-th token; the lanes that share channels reduce minimum and maximum among them so that each ends with
// its own share of the groups, finds their thresholds and hands them back by shuffles.  Values: 32 tokens x D
// channels; a lane has D / 16 consecutive channels of 16 consecutive tokens (whole code words of these channels, or
// halves), and the lanes of a channel group share the tokens' statistics in the same way.
//
// What bounds it: HBM on bulk appends.  A tile per CTA in shared memory, the version before, took 19.4 instructions an
// element, most of them index arithmetic and control of small CTAs.
// ---------------------------------------------------------------------------
template <int D, int G>
struct Tiles {
  static constexpr int C = 4096 / G < D ? 4096 / G : D;  // channels of a key tile
  static constexpr int LR = C / 16, TS = 32 / LR;        // lanes of a token's row, tokens of a step
  static constexpr int STEPS = G / TS;
  static constexpr int CPL = D / 16;                     // values: channels of a lane
  static constexpr int LG = G / CPL;                     // values: lanes of a group
  static constexpr int TPL = 16 / LG;                    // values: groups (tokens) whose thresholds a lane finds
};

// Of n values a lane keeps half and gives the other half away: out[k] = op(kept, partner's).
template <int N, typename F>
__device__ __forceinline__ void scatter_step(uint32_t* v, int mask, bool upper, F op) {
#pragma unroll
  for (int k = 0; k < N / 2; ++k) {
    const uint32_t keep = upper ? v[k + N / 2] : v[k], send = upper ? v[k] : v[k + N / 2];
    v[k] = op(keep, __shfl_xor_sync(0xffffffffu, send, mask));
  }
}

// Stores a lane's words of codes, word k at dst(k); merging and difference counting (own bits 1 and 2) look at the words
// that are there.
template <int BITS, int N, typename F>
__device__ __forceinline__ void put_words(const uint32_t (&w)[N], int n, int own, uint32_t lut, uint32_t (&hist)[4], F dst) {
  if (own == 1) {
#pragma unroll
    for (int k = 0; k < N; ++k)
      if (k < n) *dst(k) = w[k];
    return;
  }
#pragma unroll 1
  for (int k = 0; k < n; ++k) {  // rare modes: one copy of the code
    uint32_t v = w[0];
#pragma unroll
    for (int j = 1; j < N; ++j) v = k == j ? w[j] : v;
    uint32_t* const to = dst(k);
    const uint32_t o = *to;  // the dominant layer's codes of these positions are in place
    if (own & 4) delta_count<BITS>(o, v, hist);
    if (own & 3) *to = merge_words<BITS>(o, v, lut);
  }
}

template <int D, int G, bool F16>
struct Packer {
  using I16 = In16<F16>;
  using V2 = typename I16::V2;
  using Ti = Tiles<D, G>;
  static __device__ __forceinline__ V2 v2(uint32_t x) { return *reinterpret_cast<V2*>(&x); }
  static __device__ __forceinline__ uint32_t u32(V2 x) { return *reinterpret_cast<uint32_t*>(&x); }
  static __device__ __forceinline__ uint32_t min2(uint32_t a, uint32_t b) { return u32(__hmin2(v2(a), v2(b))); }
  static __device__ __forceinline__ uint32_t max2(uint32_t a, uint32_t b) { return u32(__hmax2(v2(a), v2(b))); }

  // Row pabs (absolute token) of the stream: in the old window while pabs < s_old, else in the input.
  static __device__ __forceinline__ const uint16_t* row(const PackParams& p, const uint16_t* win, const uint16_t* in, int bh, int pabs) {
    return pabs < p.s_old ? win + ((size_t)bh * p.dm.R + (pabs - p.nq_old)) * D : in + ((size_t)bh * p.n_in + (pabs - p.s_old)) * D;
  }
  // The window rows that a lane has read (rows r of the old window) are free: the tokens that follow the quantized
  // blocks take them, the same pieces by the same lane.
  template <int VECS>
  static __device__ __forceinline__ void refill(const PackParams& p, uint16_t* win, const uint16_t* in, int bh, int r, int c) {
    if (r < p.win_count) {
      const uint16_t* src = in + ((size_t)bh * p.n_in + (p.nq_new + r - p.s_old)) * D + c;
      uint16_t* dst = win + ((size_t)bh * p.dm.R + r) * D + c;
      if constexpr (VECS > 0) {
#pragma unroll
        for (int k = 0; k < VECS; ++k) reinterpret_cast<uint4*>(dst)[k] = reinterpret_cast<const uint4*>(src)[k];
      } else {
        *reinterpret_cast<uint2*>(dst) = *reinterpret_cast<const uint2*>(src);
      }
    }
  }

  template <int BITS>
  static __device__ __forceinline__ void key_codes(const PackParams& p, const PackLayer& pl, const uint32_t (&x)[Ti::STEPS][8],
                                                   const uint32_t (&thr)[2][3], int tq0, int d0, int bh, int i, int sub,
                                                   uint32_t (&hist)[4]) {
    constexpr int TS = Ti::TS, LR = Ti::LR;
    uint32_t t1[8], t2[8], t3[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {  // pair q was left with the lane whose sub has these bits
      const int owner = TS == 4 ? ((q >> 2) | ((q & 2))) : ((q >> 2) | (q & 2) | ((q & 1) << 2));
      const int at = TS == 4 ? q & 1 : 0, src = owner * LR + i;
      t1[q] = __shfl_sync(0xffffffffu, thr[at][0], src);
      if constexpr (BITS == 2) {
        t2[q] = __shfl_sync(0xffffffffu, thr[at][1], src);
        t3[q] = __shfl_sync(0xffffffffu, thr[at][2], src);
      } else {
        t2[q] = t3[q] = 0u;
      }
    }
    uint32_t* codes = pl.L.k_codes + (size_t)bh * ((size_t)p.dm.nq_cap * D * BITS / 32);
    uint32_t w[Ti::STEPS];
#pragma unroll
    for (int st = 0; st < Ti::STEPS; ++st) {
      w[st] = 0u;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const uint32_t lo = code_pair<BITS, V2>(x[st][2 * e], t1[2 * e], t2[2 * e], t3[2 * e]);
        const uint32_t hi = code_pair<BITS, V2>(x[st][2 * e + 1], t1[2 * e + 1], t2[2 * e + 1], t3[2 * e + 1]);
        w[st] |= __byte_perm(lo, hi, 0x6420) << (BITS * e);
      }
    }
    const uint32_t lut = p.merge_lut[BITS - 1];
    if constexpr (BITS == 2) {
      put_words<2>(w, Ti::STEPS, pl.own_k, lut, hist,
                   [&](int k) { return codes + k_code_position(tq0 + k * TS + sub, d0, 2, D).word; });
    } else {  // a word is two lanes' channels: of two tokens each lane completes one
      const bool upper = (i & 1) != 0;
#pragma unroll
      for (int st = 0; st < Ti::STEPS; st += 2) {
        const uint32_t keep = upper ? w[st + 1] << 4 : w[st], send = upper ? w[st] << 4 : w[st + 1];
        w[st / 2] = keep | __shfl_xor_sync(0xffffffffu, send, 1);
      }
      put_words<1>(w, Ti::STEPS / 2, pl.own_k, lut, hist, [&](int k) {
        return codes + k_code_position(tq0 + (2 * k + (upper ? 1 : 0)) * TS + sub, d0 & ~31, 1, D).word;
      });
    }
  }

  static __device__ __forceinline__ void keys(const PackParams& p, const PackLayer& pl, int tile, int bh, int lane, uint32_t (&hist)[4]) {
    constexpr int TS = Ti::TS, LR = Ti::LR, CT = D / Ti::C;
    const int i = lane % LR, sub = lane / LR, t0 = tile / CT * G, d0 = tile % CT * Ti::C + 16 * i;
    const int tq0 = p.nq_old + t0;
    uint32_t x[Ti::STEPS][8];
#pragma unroll
    for (int st = 0; st < Ti::STEPS; ++st) {
      const uint4* src = reinterpret_cast<const uint4*>(row(p, pl.L.win_k, pl.K_in, bh, tq0 + st * TS + sub) + d0);
      const uint4 a = src[0], b = src[1];
      x[st][0] = a.x; x[st][1] = a.y; x[st][2] = a.z; x[st][3] = a.w;
      x[st][4] = b.x; x[st][5] = b.y; x[st][6] = b.z; x[st][7] = b.w;
    }
    uint32_t mn[8], mx[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      mn[q] = mx[q] = x[0][q];
#pragma unroll
      for (int st = 1; st < Ti::STEPS; ++st) {
        mn[q] = min2(mn[q], x[st][q]);
        mx[q] = max2(mx[q], x[st][q]);
      }
    }
    if (t0 < p.win_count) {
#pragma unroll
      for (int st = 0; st < Ti::STEPS; ++st) refill<2>(p, pl.L.win_k, pl.K_in, bh, t0 + st * TS + sub, d0);
    }
    scatter_step<8>(mn, LR, sub & 1, min2);
    scatter_step<8>(mx, LR, sub & 1, max2);
    scatter_step<4>(mn, 2 * LR, sub & 2, min2);
    scatter_step<4>(mx, 2 * LR, sub & 2, max2);
    int q0 = 4 * (sub & 1) + (sub & 2);
    if constexpr (TS == 8) {
      scatter_step<2>(mn, 4 * LR, sub & 4, min2);
      scatter_step<2>(mx, 4 * LR, sub & 4, max2);
      q0 += sub >> 2;
    }
    constexpr int PAIRS = 8 / TS;  // pairs of channels that are this lane's now
    __half* meta = reinterpret_cast<__half*>(pl.L.k_meta) + ((size_t)bh * (p.dm.nq_cap / G) + tq0 / G) * (2 * D);
    uint32_t thr[2][3] = {{0u, 0u, 0u}, {0u, 0u, 0u}};
#pragma unroll 1
    for (int g = 0; g < 2 * PAIRS; ++g) {  // (rolled, for the instruction cache)
      const int h = g & 1;
      const bool second = PAIRS == 2 && g >= 2;
      const uint32_t mnw = second ? mn[1] : mn[0], mxw = second ? mx[1] : mx[0];
      const float lo = h ? I16::hi(mnw) : I16::lo(mnw), hi = h ? I16::hi(mxw) : I16::lo(mxw);
      float z, sc;
      __half zh, sh;
      group_params(lo, hi, pl.L.bk, pl.eta_k, z, sc, zh, sh);
      const int pos = k_meta_position(d0 + 2 * q0 + g, D);
      meta[pos] = sh;
      meta[D + pos] = zh;
      if (pl.own_k) {
        uint32_t tt[3];
        group_thresholds<F16>(lo, hi, z, sc, pl.L.bk, tt);
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          const uint32_t v = tt[j] << (16 * h);
          if (second) thr[1][j] |= v; else thr[0][j] |= v;
        }
      }
    }
    if (!pl.own_k) return;  // PseudoQuantize: parameters only
    if (pl.L.bk == 2) key_codes<2>(p, pl, x, thr, tq0, d0, bh, i, sub, hist);
    else key_codes<1>(p, pl, x, thr, tq0, d0, bh, i, sub, hist);
  }

  template <int BITS>
  static __device__ __forceinline__ void value_codes(const PackParams& p, const PackLayer& pl, const uint32_t (&x)[16][Ti::CPL / 2],
                                                     const uint32_t (&ta)[Ti::TPL], const uint32_t (&tb)[Ti::TPL], int tq0, int d0,
                                                     int bh, int lane, uint32_t (&hist)[4]) {
    constexpr int NP = Ti::CPL / 2, LG = Ti::LG;
    uint32_t acc[4][NP];  // [token % 4][channel pair]: the codes' bits of that byte, a channel in each half
#pragma unroll
    for (int b = 0; b < 4; ++b)
#pragma unroll
      for (int c = 0; c < NP; ++c) acc[b][c] = 0u;
#pragma unroll
    for (int t = 0; t < 16; ++t) {
      // token t was left with the lane of the group that has these bits, as its value t % TPL
      int owner = 0;
#pragma unroll
      for (int k = 0, n = 8; n >= Ti::TPL; n >>= 1, ++k) owner |= ((t & n) ? 1 : 0) << k;
      const int src = (lane & ~(LG - 1)) | owner;
      const uint32_t a = __shfl_sync(0xffffffffu, ta[t % Ti::TPL], src);
      const uint32_t t1 = __byte_perm(a, a, 0x1010);
      uint32_t t2 = 0u, t3 = 0u;
      if constexpr (BITS == 2) {
        t2 = __byte_perm(a, a, 0x3232);
        t3 = __shfl_sync(0xffffffffu, tb[t % Ti::TPL], src);
      }
#pragma unroll
      for (int c = 0; c < NP; ++c) acc[t % 4][c] += code_pair<BITS, V2>(x[t][c], t1, t2, t3) << (BITS * (t / 4));
    }
    uint32_t w[Ti::CPL];
#pragma unroll
    for (int c = 0; c < NP; ++c) {
      const uint32_t a = __byte_perm(acc[0][c], acc[1][c], 0x6240), b = __byte_perm(acc[2][c], acc[3][c], 0x6240);
      w[2 * c] = __byte_perm(a, b, 0x5410);
      w[2 * c + 1] = __byte_perm(a, b, 0x7632);
    }
    uint32_t* codes = pl.L.v_codes + (size_t)bh * ((size_t)p.dm.nq_cap * D * BITS / 32);
    const uint32_t lut = p.merge_lut[BITS - 1];
    const int half = lane >> 4;
    if constexpr (BITS == 2) {
      put_words<2>(w, Ti::CPL, pl.own_v, lut, hist,
                   [&](int c) { return codes + v_code_position(tq0 + 16 * half, d0 + c, 2, D).word; });
    } else {  // a word is both halves' tokens: each half completes half of the channels
#pragma unroll
      for (int c = 0; c < Ti::CPL; ++c) w[c] <<= 4 * half;
      scatter_step<Ti::CPL>(w, 16, half, [](uint32_t a, uint32_t b) { return a | b; });
      put_words<1>(w, NP, pl.own_v, lut, hist,
                   [&](int c) { return codes + v_code_position(tq0, d0 + half * NP + c, 1, D).word; });
    }
  }

  static __device__ __forceinline__ void values(const PackParams& p, const PackLayer& pl, int tile, int bh, int lane, uint32_t (&hist)[4]) {
    constexpr int NP = Ti::CPL / 2, NG = D / G, LG = Ti::LG, TPL = Ti::TPL;
    const int half = lane >> 4, d0 = (lane & 15) * Ti::CPL, t0 = tile * 32, tq0 = p.nq_old + t0;
    uint32_t x[16][NP];
#pragma unroll
    for (int t = 0; t < 16; ++t) {
      const uint16_t* src = row(p, pl.L.win_v, pl.V_in, bh, tq0 + 16 * half + t) + d0;
      if constexpr (NP == 4) {
        const uint4 a = *reinterpret_cast<const uint4*>(src);
        x[t][0] = a.x; x[t][1] = a.y; x[t][2] = a.z; x[t][3] = a.w;
      } else {
        const uint2 a = *reinterpret_cast<const uint2*>(src);
        x[t][0] = a.x; x[t][1] = a.y;
      }
    }
    // per token (minimum, -maximum) of this lane's channels, then of the group's: one packed minimum for both
    uint32_t st[16];
#pragma unroll
    for (int t = 0; t < 16; ++t) {
      uint32_t mn = x[t][0], mx = x[t][0];
#pragma unroll
      for (int c = 1; c < NP; ++c) {
        mn = min2(mn, x[t][c]);
        mx = max2(mx, x[t][c]);
      }
      mx ^= 0x80008000u;
      st[t] = min2(__byte_perm(mn, mx, 0x5410), __byte_perm(mn, mx, 0x7632));
    }
    if (t0 < p.win_count) {
#pragma unroll
      for (int t = 0; t < 16; ++t) refill<NP == 4 ? 1 : 0>(p, pl.L.win_v, pl.V_in, bh, t0 + 16 * half + t, d0);
    }
    int tk = 0;  // first of the tokens that are left with this lane
    scatter_step<16>(st, 1, lane & 1, min2); tk += 8 * (lane & 1);
    scatter_step<8>(st, 2, (lane >> 1) & 1, min2); tk += 4 * ((lane >> 1) & 1);
    if constexpr (LG >= 8) { scatter_step<4>(st, 4, (lane >> 2) & 1, min2); tk += 2 * ((lane >> 2) & 1); }
    if constexpr (LG >= 16) { scatter_step<2>(st, 8, (lane >> 3) & 1, min2); tk += (lane >> 3) & 1; }
    __half* meta = reinterpret_cast<__half*>(pl.L.v_meta) + (size_t)bh * p.dm.nq_cap * 2 * NG;
    uint32_t ta[TPL], tb[TPL];  // X_1 and X_2; X_3 twice
#pragma unroll
    for (int k = 0; k < TPL; ++k) ta[k] = tb[k] = 0u;
#pragma unroll 1
    for (int g = 0; g < TPL; ++g) {
      uint32_t w = st[0];
#pragma unroll
      for (int k = 1; k < TPL; ++k) w = g == k ? st[k] : w;
      const float mn = I16::lo(w), mx = -I16::hi(w);
      float z, sc;
      __half zh, sh;
      group_params(mn, mx, pl.L.bv, pl.eta_v, z, sc, zh, sh);
      const int tabs = tq0 + 16 * half + tk + g, gi = d0 / G;
      meta[v_scale_index(tabs, gi, NG)] = sh;
      meta[v_zero_index(tabs, gi, NG)] = zh;
      if (pl.own_v) {
        uint32_t tt[3];
        group_thresholds<F16>(mn, mx, z, sc, pl.L.bv, tt);
        const uint32_t a = tt[0] | (tt[1] << 16), b = tt[2] * 0x10001u;
#pragma unroll
        for (int k = 0; k < TPL; ++k)
          if (g == k) { ta[k] = a; tb[k] = b; }
      }
    }
    if (!pl.own_v) return;
    if (pl.L.bv == 2) value_codes<2>(p, pl, x, ta, tb, tq0, d0, bh, lane, hist);
    else value_codes<1>(p, pl, x, ta, tb, tq0, d0, bh, lane, hist);
  }
};

// blockIdx.x even: keys, odd: values, a tile per warp; blockIdx.y the (sequence, kv head) stream, blockIdx.z the layer
// of the launch.  With p.win_count > 0 the warps of the first block also copy the new window rows over those they read.
template <int D, int G, bool F16>
__global__ void __launch_bounds__(PACK_THREADS, 4) pack_kernel(const __grid_constant__ PackParams p) {
  using Ti = Tiles<D, G>;
  const int lane = threadIdx.x & 31, tile = (blockIdx.x >> 1) * (PACK_THREADS / 32) + (threadIdx.x >> 5);
  const bool values = blockIdx.x & 1;
  const int tokens = p.n_blocks * p.dm.R;
  grid_dependency_wait();  // the inputs come from the preceding kernel, and earlier kernels may still read the cache
  grid_dependents_go();    // the next kernel may get its CTAs placed; it waits for this one before it reads the cache
  if (tile >= (values ? tokens / 32 : tokens / G * (D / Ti::C))) return;
  const PackLayer& pl = p.layer[blockIdx.z];
  uint32_t hist[4] = {0u, 0u, 0u, 0u};
  if (values) Packer<D, G, F16>::values(p, pl, tile, blockIdx.y, lane, hist);
  else Packer<D, G, F16>::keys(p, pl, tile, blockIdx.y, lane, hist);
  if ((values ? pl.own_v : pl.own_k) & 4) {
    unsigned long long* out = values ? pl.delta_v : pl.delta_k;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const uint32_t tot = __reduce_add_sync(0xffffffffu, hist[k]);
      if (lane == 0 && tot) atomicAdd(out + k, (unsigned long long)tot);
    }
  }
}

template <int D, int G, bool F16>
cudaError_t launch_pack_t(const PackParams& p, cudaStream_t st) {
  using Ti = Tiles<D, G>;
  const int tokens = p.n_blocks * p.dm.R;
  const int tiles_k = tokens / G * (D / Ti::C), tiles_v = tokens / 32, tiles = tiles_k > tiles_v ? tiles_k : tiles_v;
  constexpr int W = PACK_THREADS / 32;
  return launch_dependent(pack_kernel<D, G, F16>, dim3(2 * ((tiles + W - 1) / W), p.dm.B * p.dm.Hkv, p.n_layers),
                          dim3(PACK_THREADS), 0, st, p);
}

cudaError_t launch_pack(const PackParams& p, cudaStream_t st) {
  if (p.n_layers < 1 || p.n_layers > PACK_MAX_LAYERS) return cudaErrorInvalidValue;
  const bool f16 = p.f16 != 0;
  switch (p.dm.D * 100 + p.dm.g) {
    case 12832: return f16 ? launch_pack_t<128, 32, true>(p, st) : launch_pack_t<128, 32, false>(p, st);
    case 12864: return f16 ? launch_pack_t<128, 64, true>(p, st) : launch_pack_t<128, 64, false>(p, st);
    case 6432: return f16 ? launch_pack_t<64, 32, true>(p, st) : launch_pack_t<64, 32, false>(p, st);
    case 6464: return f16 ? launch_pack_t<64, 64, true>(p, st) : launch_pack_t<64, 64, false>(p, st);
  }
  return cudaErrorInvalidValue;
}

// Copies new tokens into the 16-bit window, keys and values in one launch.
__global__ void __launch_bounds__(256) window_append_kernel(WindowParams p) {
  const Dims& dm = p.dm;
  const int vec_per_row = dm.D / 8;
  const size_t per_kind = (size_t)dm.B * dm.Hkv * p.count * vec_per_row;
  size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  grid_dependents_go();    // the next kernel may get its CTAs placed; it waits for this one before it reads the window
  grid_dependency_wait();  // the inputs come from the preceding kernel, and earlier kernels may still read the window
  if (idx >= 2 * per_kind) return;
  int kind = idx >= per_kind;
  size_t r = idx - (kind ? per_kind : 0);
  int c8 = r % vec_per_row;
  r /= vec_per_row;
  int tok = r % p.count;
  int bh = r / p.count;
  int pabs = p.first + tok;
  const uint16_t* in = kind ? p.V_in : p.K_in;
  uint16_t* win = kind ? p.L.win_v : p.L.win_k;
  const uint4* src = reinterpret_cast<const uint4*>(in + ((size_t)bh * p.n_in + (pabs - p.s_old)) * dm.D) + c8;
  uint4* dst = reinterpret_cast<uint4*>(win + ((size_t)bh * dm.R + (pabs - p.nq_new)) * dm.D) + c8;
  *dst = *src;
}

cudaError_t launch_window_append(const WindowParams& p, cudaStream_t st) {
  size_t total = 2 * (size_t)p.dm.B * p.dm.Hkv * p.count * (p.dm.D / 8);
  unsigned blocks = (unsigned)((total + 255) / 256);
  return launch_dependent(window_append_kernel, dim3(blocks), dim3(256), 0, st, p);
}

}  // namespace xq
