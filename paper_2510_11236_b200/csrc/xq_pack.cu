// Quantize-and-pack of residual-window blocks (Eq. 1, 2, 12; Algorithm 2) and
// the window append.  One CTA quantizes a tile of T (32 or 64) tokens x D channels of
// one (sequence, kv head) for keys or for values.
//
// The fp32 arithmetic uses the *_rn intrinsics so that no multiply-add is ever
// contracted: codes, scales and zero-points are compared bit for bit with a CPU
// evaluation of the same formulas.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <type_traits>

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
    // RN(a / 3) by Markstein's correction step, as in `Quot` below: RN(1 / 3) is the correctly rounded reciprocal and q
    // within an ulp of a / 3; tiny and huge ranges, which could leave the normal range on the way, take the division
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
constexpr int PACK_ROW_PAD = 16;  // bytes added to each staged row: 8 consecutive rows then fall in 8 different bank groups

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
// finds the X_k next to z + (k - 1/2) s, where a subtraction and a comparison decide, else by evaluating c itself (the
// quotient exactly as the division gives it, ties of rint to even) at lattice points; the elements are then coded two at a time with packed 16-bit compares.

// 16-bit float pattern <-> integer that orders like the value (sign-magnitude to two's complement; -0 and +0 -> 0)
__device__ __forceinline__ int ord16(uint32_t h) {
  const int m = (int)(h & 0x7fffu);
  return (h & 0x8000u) ? -m : m;
}
__device__ __forceinline__ uint32_t pat16(int o) { return o >= 0 ? (uint32_t)o : (0x8000u | (uint32_t)(-o)); }

// A group's uncalibrated parameters for the quotient RN(RN(x - z) / s).  With y = RN(1/s): q = RN(a y),
// r = a - q s (exact in one fused multiply-add), q' = RN(q + r y) is the correctly rounded quotient: the correction step
// of P. W. Markstein, "Computation of elementary functions on the IBM RISC System/6000 processor", IBM J. Res. Dev.
// 34 (1990), which holds where y is the correctly rounded reciprocal, q is within an ulp of a / s and nothing leaves the
// normal range.  Scales whose significand is all ones and those of extreme exponent get a NaN from safe_rcp and take the
// division.
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

// X_k as a 16-bit pattern for a group with minimum mn and maximum mx.  With a = RN(x - z), c(x) >= k means
// RN(a / s) >= k - 1/2 (for odd k: > k - 1/2, rint taking ties to the even neighbour), and that means a >= s m in real
// numbers, m the midpoint below the first float that counts: 1/2 + 2^-25, 3/2 - 2^-24, 5/2 + 2^-23 for k = 1, 2, 3 (s m
// is never a float: the odd part of m has 25 bits).  So a >= a* = RU(s m), one fused multiply-add with directed
// rounding, exactly.  x at or above z + a* satisfies RN(x - z) >= a*; x below it only if it is closer to it than half an
// ulp of a*.  So X_k is the first lattice point at or above z + a* (1 - 2^-23) if that point passes the test, and else
// the next one if that one lies above z + a* (the midpoint of minimum and maximum, k = 2, is a lattice point itself
// more often than not).  Several lattice points lie between only where z + a* all but cancels (one group in fifty:
// minimum and maximum of equal magnitude); z + a* is then exact and so is w, half an ulp of a* below it: X_k is the
// first lattice point at or above w (above it, where a* is odd: the tie goes down).  Groups whose scale takes the division (safe_rcp) are bisected from the
// group's ends (c(mn) = 0, c(mx) = 2^B - 1).
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
template <bool F16, int K>
__device__ __forceinline__ uint32_t threshold16(const Quot& g, float mn, float mx) {
  constexpr float KK = (float)K - 0.5f, OFF = K == 1 ? 0x1p-25f : (K == 2 ? -0x1p-24f : 0x1p-23f);
  const float as = __fmaf_ru(KK, g.s, __fmul_rn(g.s, OFF));
  const uint32_t up = In16<F16>::bits_up(__fadd_ru(g.z, as));
  const uint32_t up_lo = In16<F16>::bits_up(__fadd_rd(g.z, __fmul_rd(as, 1.0f - 0x1p-23f)));
  constexpr uint32_t INF16 = F16 ? 0x7c00u : 0x7f80u;
  const bool passes = __fsub_rn(In16<F16>::one((uint16_t)up_lo), g.z) >= as;
  const bool next = up == ((up_lo & 0x8000u) ? up_lo - 1u : up_lo + 1u);
  if (g.fast && up != INF16 && (passes || next || up == up_lo)) return passes ? up_lo : up;
  const float d = __fadd_rn(g.z, as);
  if (g.fast && fabsf(d) < __fmul_rn(as, 0x1p-10f)) {
    const float w = __fsub_rn(d, __fmul_rn(0.5f, __fsub_rn(as, __uint_as_float(__float_as_uint(as) - 1u))));
    const uint32_t x = In16<F16>::bits_up(w);
    const bool above = (__float_as_uint(as) & 1u) && In16<F16>::one((uint16_t)x) == w;
    return above ? pat16(ord16(x) + 1) : x;
  }
  const int lo = g.fast ? ord16(up_lo) - 1 : ord16(In16<F16>::bits(mn));
  const int hi = g.fast && up != INF16 ? ord16(up) : ord16(In16<F16>::bits(mx));  // (a bound beyond the largest finite value)
  return bisect16<F16>(g.z, g.s, g.y, K, lo, hi);
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
    thr[0] = threshold16<F16, 1>(g, mn, mx);
    if (bits == 2) {
      thr[1] = threshold16<F16, 2>(g, mn, mx);
      thr[2] = threshold16<F16, 3>(g, mn, mx);
    }
  }
}

// Codes of two packed 16-bit elements against their groups' packed thresholds, accumulated: acc += S << shift.  A mask
// is 0xffff per element that passed, so S, the sum of the three masks, is -(low count) + 2^16 (low count - high count):
// linear in the counts, and finish() turns the accumulated sum into (low counts) + 2^16 (high counts), every count at
// its shift, with one multiplication.
template <int BITS, typename V2>
__device__ __forceinline__ void add_codes(uint32_t& acc, int shift, uint32_t x, uint32_t t1, uint32_t t2, uint32_t t3) {
  const V2 xv = *reinterpret_cast<const V2*>(&x);
  uint32_t sum = __hge2_mask(xv, *reinterpret_cast<const V2*>(&t1));
  if constexpr (BITS == 2)
    sum += __hge2_mask(xv, *reinterpret_cast<const V2*>(&t2)) + __hge2_mask(xv, *reinterpret_cast<const V2*>(&t3));
  acc += sum << shift;
}
__device__ __forceinline__ uint32_t finish(uint32_t acc) { return acc * (0u - 0x10001u); }

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

// One CTA: T tokens x D channels of one (sequence, kv head), keys (blockIdx.x even) or values (odd).  Staged
// rows are padded.  Keys: a thread builds whole words of a token's row (four consecutive channels per bit
// offset), the words are collected in shared memory in stream order and leave in 16-byte vectors.  Values: a
// thread builds whole words of a channel's row over the tile's tokens and stores them itself.
// G: group size; T: a multiple of G and of 32; F16: the 16-bit type is IEEE half precision.
// blockIdx.y is the (sequence, kv head) stream, blockIdx.z the layer of the launch.  With p.win_count > 0 the CTAs of
// the first block also copy the new window rows that replace the rows they staged.
// What bounds it: instruction issue where a layer owns its codes (268 MB of input: 181 us), HBM where it stores
// parameters only (94 us).  Prompts of 4k tokens, batch 8, 32 kv heads, four layers: 595 us with thresholds by
// bracketing and codes assembled one by one, 558 now.  Measured and not kept: a warp per tile with the tile in
// registers, 928, then 601 us, and 160 us on 333-token pieces of 16 layers against 72 (too few loads in flight).
// One-layer launches carry the parameters of one layer (LAYERS = 1): 3.6 KB of parameters cost ~3 us of host time a
// launch, 16 layers' pieces 137 -> 72 us.
template <int D, int G, int T, bool F16, int LAYERS>
__global__ void __launch_bounds__(PACK_THREADS) pack_kernel(const __grid_constant__ PackParamsOf<LAYERS> p) {
  using I16 = In16<F16>;
  using V2 = typename I16::V2;
  constexpr int ROWB = D * 2 + PACK_ROW_PAD;
  constexpr int NG = D / G;
  constexpr int KG = (T / G) * D;                                      // key groups of the tile
  constexpr int KP = PACK_THREADS / ((T / G) * (D / 2));               // token parts of a key group in the statistics
  static_assert(KP >= 1 && G % KP == 0, "key statistics: 128 threads over (group, channel pair, token part)");
  __shared__ __align__(16) uint8_t tile[T * ROWB];
  // thresholds X_1..X_3 of a group: keys [k][token group][channel]; values [token][channel group] of four words, each
  // threshold in both halves of one
  constexpr int NTHR = 3 * (T / G) * D * 2 > T * NG * 16 ? 3 * (T / G) * D * 2 : T * NG * 16;
  __shared__ __align__(16) uint8_t thr_mem[NTHR];
  uint16_t* const thr = reinterpret_cast<uint16_t*>(thr_mem);
  // packed words (at most T * D * 2 / 32); before that, the key statistics' partial (min, max) pairs, two words per thread
  constexpr int NWBUF = (T * D * 2 / 32) > 2 * PACK_THREADS ? (T * D * 2 / 32) : 2 * PACK_THREADS;
  __shared__ __align__(16) uint32_t wbuf[NWBUF];

  const Dims& dm = p.dm;
  const int R = dm.R;
  const int kind = blockIdx.x & 1;  // 0 keys, 1 values
  const int tile_idx = blockIdx.x >> 1;
  const PackLayer pl = p.layer[LAYERS == 1 ? 0 : blockIdx.z];  // by value: its fields are read in every loop below
  const int bh = blockIdx.y;                  // (sequence, kv head) stream
  const int tid = threadIdx.x;
  const int tq0 = p.nq_old + tile_idx * T;  // absolute index of the tile's first token
  grid_dependency_wait();  // the inputs come from the preceding kernel, and earlier kernels may still read the cache
  grid_dependents_go();    // the next kernel may get its CTAs placed; it waits for this one before it reads the cache

  {
    const uint16_t* win = kind ? pl.L.win_v : pl.L.win_k;
    const uint16_t* in = kind ? pl.V_in : pl.K_in;
    constexpr int VPR = D / 8;
    // row `pabs` (absolute token) of the stream: in the old window while pabs < s_old, else in the input
    const uint16_t* const win_rows = win + ((size_t)bh * R - p.nq_old) * D;
    const uint16_t* const in_rows = in + ((size_t)bh * p.n_in - p.s_old) * D;
#pragma unroll
    for (int k = 0; k < T * VPR / PACK_THREADS; ++k) {
      const int idx = tid + k * PACK_THREADS;
      const int tl = idx / VPR, c8 = idx % VPR;
      const int pabs = tq0 + tl;
      const uint16_t* src = (pabs < p.s_old ? win_rows : in_rows) + (size_t)pabs * D;
      *reinterpret_cast<uint4*>(tile + tl * ROWB + c8 * 16) = reinterpret_cast<const uint4*>(src)[c8];
    }
  }
  __syncthreads();
  // the window rows this CTA staged are free: the tokens that follow the quantized blocks take them
  if (p.win_count > 0 && tile_idx * T < p.win_count) {
    uint16_t* win = kind ? pl.L.win_v : pl.L.win_k;
    const uint16_t* in = kind ? pl.V_in : pl.K_in;
    constexpr int VPR = D / 8;
    const int rows = min(T, p.win_count - tile_idx * T);
    for (int idx = tid; idx < rows * VPR; idx += PACK_THREADS) {
      const int r = tile_idx * T + idx / VPR, c8 = idx % VPR;
      const uint4* src = reinterpret_cast<const uint4*>(in + ((size_t)bh * p.n_in + (p.nq_new + r - p.s_old)) * D) + c8;
      reinterpret_cast<uint4*>(win + ((size_t)bh * R + r) * D)[c8] = *src;
    }
  }

  const int bits = kind ? pl.L.bv : pl.L.bk;
  const float eta = kind ? pl.eta_v : pl.eta_k;
  const int own = kind ? pl.own_v : pl.own_k;

  if (kind == 0) {
    // keys: one group per (channel, run of G tokens).  First bf16x2 min / max of a channel pair over a part of the
    // group's tokens (consecutive threads take consecutive pairs), then one thread per (group, channel).
    {
      const int dp = tid % (D / 2), rest = tid / (D / 2);
      const int gl = rest / KP, part = rest % KP;
      const uint8_t* col = tile + (gl * G + part * (G / KP)) * ROWB + dp * 4;
      V2 mn2 = *reinterpret_cast<const V2*>(col), mx2 = mn2;
#pragma unroll
      for (int j = 1; j < G / KP; ++j) {
        const V2 v = *reinterpret_cast<const V2*>(col + j * ROWB);
        mn2 = __hmin2(mn2, v);
        mx2 = __hmax2(mx2, v);
      }
      wbuf[(rest * (D / 2) + dp) * 2] = *reinterpret_cast<uint32_t*>(&mn2);
      wbuf[(rest * (D / 2) + dp) * 2 + 1] = *reinterpret_cast<uint32_t*>(&mx2);
    }
    __syncthreads();
    __half* meta = reinterpret_cast<__half*>(pl.L.k_meta);
    const size_t cap_g = (size_t)(dm.nq_cap / G);
#pragma unroll
    for (int k = 0; k < ((T / G) * D + PACK_THREADS - 1) / PACK_THREADS; ++k) {
      const int item = tid + k * PACK_THREADS;
      if (item < (T / G) * D) {
        const int gl = item / D, d = item % D;
        float mn = 0.f, mx = 0.f;
#pragma unroll
        for (int part = 0; part < KP; ++part) {
          const uint32_t a2 = wbuf[((gl * KP + part) * (D / 2) + d / 2) * 2], b2 = wbuf[((gl * KP + part) * (D / 2) + d / 2) * 2 + 1];
          const float lo = (d & 1) ? I16::hi(a2) : I16::lo(a2);
          const float hi = (d & 1) ? I16::hi(b2) : I16::lo(b2);
          mn = part == 0 ? lo : fminf(mn, lo);
          mx = part == 0 ? hi : fmaxf(mx, hi);
        }
        float z, sc;
        __half zh, sh;
        group_params(mn, mx, bits, eta, z, sc, zh, sh);
        if (own) {
          uint32_t x[3];
          group_thresholds<F16>(mn, mx, z, sc, bits, x);
#pragma unroll
          for (int j = 0; j < 3; ++j) thr[j * KG + item] = (uint16_t)x[j];
        }
        const size_t grp = (size_t)bh * cap_g + (tq0 / G + gl);  // per group: D scales, then D zero-points
        const int pos = k_meta_position(d, D);
        meta[grp * 2 * D + pos] = sh;
        meta[grp * 2 * D + D + pos] = zh;
      }
    }
  } else {
    // values: one group per (token, run of G channels); consecutive threads take consecutive tokens
    __half* meta = reinterpret_cast<__half*>(pl.L.v_meta);
#pragma unroll
    for (int k = 0; k < (T * NG + PACK_THREADS - 1) / PACK_THREADS; ++k) {
      const int item = tid + k * PACK_THREADS;
      if (item < T * NG) {
        const int tl = item % T, gi = item / T;
        const uint4* row = reinterpret_cast<const uint4*>(tile + tl * ROWB + gi * G * 2);
        V2 mn2, mx2;
        {
          uint4 v = row[0];
          const V2* e = reinterpret_cast<const V2*>(&v);
          mn2 = __hmin2(__hmin2(e[0], e[1]), __hmin2(e[2], e[3]));
          mx2 = __hmax2(__hmax2(e[0], e[1]), __hmax2(e[2], e[3]));
        }
#pragma unroll
        for (int j = 1; j < G / 8; ++j) {
          uint4 v = row[j];
          const V2* e = reinterpret_cast<const V2*>(&v);
          mn2 = __hmin2(mn2, __hmin2(__hmin2(e[0], e[1]), __hmin2(e[2], e[3])));
          mx2 = __hmax2(mx2, __hmax2(__hmax2(e[0], e[1]), __hmax2(e[2], e[3])));
        }
        const uint32_t mnw = *reinterpret_cast<const uint32_t*>(&mn2), mxw = *reinterpret_cast<const uint32_t*>(&mx2);
        const float mn = fminf(I16::lo(mnw), I16::hi(mnw));
        const float mx = fmaxf(I16::lo(mxw), I16::hi(mxw));
        float z, sc;
        __half zh, sh;
        group_params(mn, mx, bits, eta, z, sc, zh, sh);
        if (own) {
          uint32_t x[3];
          group_thresholds<F16>(mn, mx, z, sc, bits, x);
#pragma unroll
          for (int j = 0; j < 3; ++j) x[j] *= 0x10001u;
          reinterpret_cast<uint4*>(thr_mem)[tl * NG + gi] = make_uint4(x[0], x[1], x[2], 0u);
        }
        const int tabs = tq0 + tl;
        __half* mine = meta + (size_t)bh * dm.nq_cap * 2 * NG;
        mine[v_scale_index(tabs, gi, NG)] = sh;
        mine[v_zero_index(tabs, gi, NG)] = zh;
      }
    }
  }
  if (!own) return;  // PseudoQuantize: parameters only
  __syncthreads();

  // codes
  uint32_t* codes = kind ? pl.L.v_codes : pl.L.k_codes;
  const bool merge = (own & 2) != 0, stats = (own & 4) != 0, store = (own & 3) != 0;
  uint32_t hist[4] = {0u, 0u, 0u, 0u};
  const size_t stream_words = (size_t)dm.nq_cap * D * bits / 32;
  auto build = [&](auto bits_c) {
    constexpr int BITS = decltype(bits_c)::value;
    constexpr int N = 32 / BITS;        // codes per word
    if (kind == 0) {
      constexpr int NW = D * BITS / 32;  // words per token row
      const size_t w0 = k_code_position(tq0, 0, BITS, D).word;  // the tile's words are one contiguous run
      // a thread takes word i of every TS-th token: consecutive threads consecutive words
      constexpr int TS = PACK_THREADS / NW;
      const int i = tid % NW, d0 = i * N;
#pragma unroll
      for (int k = 0; k < (T + TS - 1) / TS; ++k) {
        const int tl = tid / NW + k * TS, gl = tl / G;
        if (TS > T && tl >= T) break;
        const uint4* row = reinterpret_cast<const uint4*>(tile + tl * ROWB + d0 * 2);
        const uint4* th = reinterpret_cast<const uint4*>(thr + gl * D + d0);  // thresholds k: KG * 2 bytes apart
        uint32_t a0 = 0u, a1 = 0u;  // channels 4 e, 4 e + 1; 4 e + 2, 4 e + 3
#pragma unroll
        for (int v = 0; v < N / 8; ++v) {
          const uint4 x = row[v], t1 = th[v];
          uint4 t2 = t1, t3 = t1;
          if constexpr (BITS == 2) {
            t2 = th[KG / 8 + v];
            t3 = th[2 * (KG / 8) + v];
          }
          add_codes<BITS, V2>(a0, BITS * (2 * v), x.x, t1.x, t2.x, t3.x);
          add_codes<BITS, V2>(a1, BITS * (2 * v), x.y, t1.y, t2.y, t3.y);
          add_codes<BITS, V2>(a0, BITS * (2 * v + 1), x.z, t1.z, t2.z, t3.z);
          add_codes<BITS, V2>(a1, BITS * (2 * v + 1), x.w, t1.w, t2.w, t3.w);
        }
        wbuf[k_code_position(tq0 + tl, d0, BITS, D).word - w0] = __byte_perm(finish(a0), finish(a1), 0x6420);
      }
      __syncthreads();
      uint4* dst = reinterpret_cast<uint4*>(codes + (size_t)bh * stream_words + w0);
      for (int v = tid; v < T * NW / 4; v += PACK_THREADS) {
        uint4 w = reinterpret_cast<const uint4*>(wbuf)[v];
        if (merge || stats) {  // the dominant layer's codes of these positions are in place
          const uint4 o = dst[v];
          if (stats) {
            delta_count<BITS>(o.x, w.x, hist); delta_count<BITS>(o.y, w.y, hist);
            delta_count<BITS>(o.z, w.z, hist); delta_count<BITS>(o.w, w.w, hist);
          }
          const uint32_t lut = p.merge_lut[BITS - 1];
          w = make_uint4(merge_words<BITS>(o.x, w.x, lut), merge_words<BITS>(o.y, w.y, lut),
                         merge_words<BITS>(o.z, w.z, lut), merge_words<BITS>(o.w, w.w, lut));
        }
        if (store) dst[v] = w;
      }
    } else {
      constexpr int WPC = T / N;  // words per channel over the tile's tokens
      // a thread takes a word of two neighbouring channels
#pragma unroll
      for (int k = 0; k < (D / 2 * WPC + PACK_THREADS - 1) / PACK_THREADS; ++k) {
        const int item = tid + k * PACK_THREADS;
        if (item < D / 2 * WPC) {
          const int d = item % (D / 2) * 2, wi = item / (D / 2), gi = d / G;
          const uint8_t* col = tile + wi * N * ROWB + d * 2;
          const uint4* th = reinterpret_cast<const uint4*>(thr_mem) + wi * N * NG + gi;
          uint32_t acc[4] = {0u, 0u, 0u, 0u};  // tokens t % 4: the codes' bits of that byte
#pragma unroll
          for (int t = 0; t < N; ++t) {
            const uint32_t x = *reinterpret_cast<const uint32_t*>(col + t * ROWB);
            const uint4 tt = th[t * NG];
            add_codes<BITS, V2>(acc[t % 4], BITS * (t / 4), x, tt.x, tt.y, tt.z);
          }
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[j] = finish(acc[j]);
          const uint32_t a = __byte_perm(acc[0], acc[1], 0x6240), b = __byte_perm(acc[2], acc[3], 0x6240);
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            uint32_t word = __byte_perm(a, b, h ? 0x7632 : 0x5410);
            uint32_t* dst = codes + (size_t)bh * stream_words + v_code_position(tq0 + wi * N, d + h, BITS, D).word;
            if (merge || stats) {
              const uint32_t o = *dst;
              if (stats) delta_count<BITS>(o, word, hist);
              word = merge_words<BITS>(o, word, p.merge_lut[BITS - 1]);
            }
            if (store) *dst = word;
          }
        }
      }
    }
  };
  if (bits == 2) build(std::integral_constant<int, 2>{}); else build(std::integral_constant<int, 1>{});
  if (stats) {
    unsigned long long* out = kind ? pl.delta_v : pl.delta_k;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const uint32_t tot = __reduce_add_sync(0xffffffffu, hist[k]);
      if ((tid & 31) == 0 && tot) atomicAdd(out + k, (unsigned long long)tot);
    }
  }
}

template <int D, int G, bool F16>
cudaError_t launch_pack_t(const PackParams& p, cudaStream_t st) {
  // a tile is one key group long: 32 or 64 tokens, whole words of either kind
  const dim3 grid(2 * p.n_blocks * (p.dm.R / G), p.dm.B * p.dm.Hkv, p.n_layers), block(PACK_THREADS);
  if (p.n_layers > 1) return launch_dependent(pack_kernel<D, G, G, F16, PACK_MAX_LAYERS>, grid, block, 0, st, p);
  PackParamsOf<1> one;
  static_cast<PackCommon&>(one) = p;
  one.layer[0] = p.layer[0];
  return launch_dependent(pack_kernel<D, G, G, F16, 1>, grid, block, 0, st, one);
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
