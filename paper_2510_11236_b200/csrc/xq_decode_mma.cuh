// Tensor-core decode attention over the packed cache, head_dim 128: one CTA takes a range of batches of one (sequence, kv
// head) stream, up to 8 query heads, of one layer or of two that read the same codes (up to four heads each).
//
// Every warp works alone on half batches of 64 tokens (rounds): nothing in the loop waits for another warp.  Codes are
// expanded straight into A fragments of mma.sync.m16n8k16 (fp16): four codes of a row sit at one bit offset of the four
// bytes of a packed word, so a shift of the word and a mask give a pair of fp16 subnormals, code * weight * 2^-e.  (The
// tensor core aligns a product by the exponent fields of its operands, so every leading zero of a subnormal costs the sum
// a bit.  Keys: codes from the third bit of the fraction up; values: 1 bit from the fifth up, 2 bits in two shifts from the
// seventh up, which with one shift left the fp32 results at 2.2 to 6.9e-5 of the result's norm, now 0.3 to 1.4e-5.)
// Scale and zero-point are folded out of the inner products,
//
//   q . k_hat_t = sum_d (q_d s_d) c_td + sum_d q_d z_d        (keys, per channel)
//   sum_t p_t v_hat_td = sum_t (p_t s_tg) c_td + sum_t p_t z_tg  (values, per token)
//
// and the other operand (q_d s_d, or p_t s_tg) is carried as an unevaluated sum hi + lo of two fp16 numbers: hi = RN(q s),
// lo = fma(q, s, -hi), as far as fp16 reaches: relative to the largest product of a round, which is kept between 2^8 and
// 2^15 (2^9 with 1-bit keys, whose weights come off q), nothing above 2^-33 is lost (p_t s_t: one rounding at 2^-22).  The
// power of two that keeps it there: with one or two heads on q (a multiplication at each product, for which no time was
// measured: 32 layers of one head at 4k, batch 8 618.7 us without, 618.0 with), so that key scales keep the bits that they
// are stored with; with three to eight on the scales, which lose bits below 2^-10 of the round's largest.
// Codes are exact, accumulation is fp32.  The powers of two that the bit offsets put on the codes are taken out of q and of
// the softmax numerators.  Up to four heads of a CTA: hi and lo are two of the eight operand columns, and the lo sums are
// added at the end.  Eight heads (five to eight of a layer, or three or four of each of two layers): a column is a head, hi
// and lo are operands of two products with the same A fragment.  A sum does not depend on the column that it is in, so a
// layer has the same bits alone and in a pair.  The numerators go through a small buffer of the warp in shared memory to
// become B fragments.
//
// Why two layers at once.  Layers of a pair differ in scales and zero-points alone, and expanding the codes was a quarter
// of the work; with eight columns of heads each lane also makes both parts of its own product, where with four heads half
// of the lanes made hi and half lo.  us of a layer in a step of 32, before and after: four heads at 32k, batch 4 27.9 ->
// 21.9; one head at 4k, batch 8 27.6 -> 19.0; groups of 64, 8k, batch 16 26.3 -> 21.4; one sequence of 128k 27.2 -> 21.7;
// five heads at 16k (one layer, eight columns) 32.1 -> 23.7, six warps then.
//
// Why mma.sync and not tcgen05.  At this shape (at most 8 query heads against 128 channels) the expanded codes are the
// large operand; a tcgen05 kernel has to pass them through tensor memory and hand batches between warps, and one that
// did spent a batch's ~1600 cycles on that chain of hand-overs, two batches per SM at a time (32k context, four heads:
// 34.2 us per layer).
// What bounds it: not one pipe.  In a launch of four layers at 32k, four heads, issue slots are 52 % used, the tensor pipe
// 38 %, ALU 35 %, the shared-memory pipe 51 %.  A batch of two layers is ~3010 warp instructions there (~2700 in long ranges,
// where a CTA's start and end do not count), 512 of them masks (2 cycles each per sub-partition), 290 products (8 cycles of
// the tensor pipe, ~2.7 of everyone's issue), ~400 half-precision multiplies (2 cycles).  Microbenchmarks of the instructions
// of both product phases come to 2900 of the 5150 cycles that a sub-partition takes for the batch (2.62 us in long ranges, 16
// or 24 warps on the SM alike, copies from L2 or HBM alike; 1.32 us at the HBM rate).  Of the rest, the issue of copies is
// known (load_key_codes); what else the warps wait for is not.  Left out in a copy, one at a time: key products 0.92, value
// products 0.78, biases 0.16, value scales 0.19, key scales 0.11, numerators 0.14 us.  Starting warps at different times,
// half of the packed words' loads or the exponentials left out: no change.
// Spills, bytes stored: pairs of four heads 56 to 76, eight heads 44 to 60, MANY 16 to 60, the others up to 20.
// Measured and not kept: twelve warps a CTA, two CTAs (the same speed of a step, single calls 2 us slower); sums in
// registers with eight heads (128 registers, two CTAs: 4 % slower).
#pragma once
#include "xq_internal.h"
#include "xq_mma.cuh"

namespace xq {
namespace {

constexpr int D = 128;             // head dim
constexpr int BT = 128;            // tokens per batch
constexpr int TT = 64;             // tokens of a round: half a batch
constexpr float TAU = 3.f;         // log2 units a logit may exceed the softmax reference before it is raised
constexpr int P_EXP = 11;          // numerators are carried times 2^P_EXP (at most 2^(P_EXP + TAU) as fp16)
constexpr int Q_BIAS_EXP = 8;      // exponent of the largest |q| in the zero-point products
constexpr uint32_t ONES = 0x3C003C00u;

// Shared-memory plan.  GS: quantization group, BK / BV: bits, HP: query heads per kv head and layer (1, 2,
// 4, 8; a G in between is padded), NL: layers that share their codes (1 or 2).  A CTA's "heads" are the VH = HP * NL
// heads of its layers.  Up to four of them: the eight operand columns are four column pairs (hi, lo) of VH heads times
// GC = 4 / VH slots: with fewer heads, one operand serves GC token units of the keys (or GC channel parts of the values)
// at once, each row tile reading the columns of its own slot.  Eight (WIDE): a column is a head, hi and lo are operands
// of two products.
template <int BK, int BV, int GS, int HP, int NL, bool MANY>
struct Plan {
  static constexpr int VH = HP * NL;
  static_assert(VH == 1 || VH == 2 || VH == 4 || VH == 8, "heads of a CTA");
  static constexpr bool WIDE = VH == 8;
  static constexpr int NSET = WIDE ? 2 : 1;      // sets of up to four heads
  static constexpr int SH = WIDE ? 4 : VH;       // heads of a set
  static constexpr int NCOL = WIDE ? 2 : 1;      // heads of a thread's accumulator columns
  static constexpr int NGT = TT / GS;            // token groups of the keys in a round
  static constexpr int NG = D / GS;              // channel groups of a value row
  static constexpr int KS = D / 16;              // k-steps of the key products, row tiles of the value products
  static constexpr int GC = WIDE ? 1 : 4 / VH;   // slots
  static constexpr int NE = WIDE ? 4 : 4 / GC;   // row tiles of 16 tokens whose logits a thread has, of the four of a round
  static constexpr int CP = NG > GC ? NG : GC;   // channel parts of the value products: one scale per token each
  static constexpr int KCODES = TT * D * BK / 8;  // codes of a round; values in 1 bit: of its whole batch
  static constexpr int VCODES = 16 * D;
  static constexpr int KM = NGT * 4 * D, VM = TT * 4 * NG;  // scales and zero-points of a round and layer: keys, values
  // value scales, then zero-points, as they are reordered over the copy: [channel group][pair of tokens] half2, a
  // group's zero-points 8 bytes longer (bank conflicts)
  static constexpr int VZROW = TT / 2 * 4 + 8, VZ = NG * (TT / 2) * 4;
  static constexpr int VROOM = (VZ + NG * VZROW + 15) / 16 * 16;
  static_assert(VROOM >= VM, "the copy fits");
  // numerators: [head][tile of 16 tokens][pair of tokens (t, t + 2)] of (hi pair, lo pair), 16 bytes more after every
  // tile and 32 more after every head against bank conflicts (WIDE: 16-byte cells in an order without any).  Two layers:
  // over the key scales and zero-points, whose next copies then come after the value products.
  static constexpr int PT = 8 * 8 + 16, PH = 4 * PT + 32;
  static constexpr int PBUF = WIDE ? 8 * 256 : VH * PH;
  static constexpr bool P_OVER = NL == 2;
  static constexpr int OFF_V = 16 * D, OFF_KM = 2 * 16 * D;
  static constexpr int OFF_VM = OFF_KM + (P_OVER && NL * KM < PBUF ? PBUF : NL * KM);
  static constexpr int OFF_P = P_OVER ? OFF_KM : (OFF_VM + NL * VROOM + 127) / 128 * 128;
  static_assert(OFF_P % 128 == 0, "cells are found by exclusive or");
  static constexpr int WROW = 2 * D + 16;        // a staged window row
  static constexpr int WIN = 32 * WROW;          // 16 key rows, then 16 value rows (over the stage of the warp)
  static constexpr int BODY = P_OVER ? OFF_VM + NL * VROOM : OFF_P + PBUF;
  static constexpr int WARP = ((BODY > WIN ? BODY : WIN) + 127) / 128 * 128;
  static constexpr bool Q_FACTOR = HP <= 2;      // the factor that keeps q s in fp16's range is taken on q
  static constexpr int MS = D + 4;               // state row: acc[D], m, l
  static_assert(2 * VH * MS * 4 <= WARP, "a warp's state rows, of the packed tokens and of the window, fit its own memory");
  static_assert(MS % 4 == 0, "state rows are read as vectors");
  // after the warps' parts: B fragments of the zero-point products; q as it came; q as operand fragments
  static constexpr int QB = NSET * KS * 32 * 4, QS = VH * D * 2, QF = KS * 32 * 8;
  static constexpr int room(int w) { return w * WARP + QB + QS + QF; }
  // PARK: the value sums of a warp wait in tensor memory between its rounds, 4 columns a row tile (WIDE: 4 more, of the lo
  // products): three CTAs per SM, each of eight warps of 80 registers.  Else two CTAs, of eight warps of 128 registers.
  // With eight heads the sums (64 registers) would not fit otherwise; two layers of one head, 4k, batch 8: 640 us a step
  // without, 622 with.  One layer alone, up to four heads: tensor memory costs a CTA 1.2 us at its start and end (a call
  // at 32k 37.0 us with, 35.2 without).
  // MANY: one layer of up to four heads for launches of many CTAs, where a CTA's start and end overlap with others' work.
  static constexpr bool PARK = WIDE || NL == 2 || MANY;
  static constexpr int CTAS = PARK ? 3 : 2, WARPS = 8;
  static constexpr int TCOLS = KS * 4 * NCOL, TMEM = WARPS / 4 * TCOLS;
  static_assert(!PARK || (CTAS * TMEM <= 512 && (TMEM & (TMEM - 1)) == 0), "tensor memory");
  static constexpr int TOTAL = room(WARPS);
  static_assert(TOTAL <= 228 * 1024 / CTAS - 1024 - 512, "shared memory");
  static_assert(WARPS * WARP >= VH * (256 + 1) * 4, "the merge's weights");
};

// The code operand pair: the code bits at BASE + BITS * i of both halves of w as they are, fp16 subnormals; their weight is
// 2^(BITS * i), a code of weight 1 stands for 2^-code_exp(BASE)
template <int BITS, int BASE>
__device__ __forceinline__ uint32_t code_pair(uint32_t w, int i) {
  return w & (((BITS == 2 ? 0x00030003u : 0x00010001u) << BASE) << (BITS * i));
}
__host__ __device__ constexpr int code_exp(int base) { return 24 - base; }

// log2 of the weight that the code of k-slot (step ks, any tig, any pair) carries in its operand
template <int BK>
__device__ __forceinline__ constexpr int k_weight(int ks) { return BK == 2 ? 2 * (ks % 4) : ks; }
// channel of k-slot c (pairs (0, 2) and (1, 3)) of step ks for lane column tig
template <int BK>
__device__ __forceinline__ int k_channel(int ks, int tig, int c) {
  if constexpr (BK == 1) return 32 * tig + 4 * ks + c;
  else return 16 * (tig + 4 * (ks / 4)) + 4 * (ks % 4) + c;
}
// Halfword index, inside a key group's D reordered scales, of channel d: per lane column and two k-steps one 16-byte
// vector [step][pair (c, c + 2), pair (c + 1, c + 3)].
template <int BK>
__device__ __forceinline__ int k_slot(int d) {
  int tig, ks;
  const int c = d & 3;
  if constexpr (BK == 1) { tig = d >> 5; ks = (d >> 2) & 7; }
  else { tig = (d >> 4) & 3; ks = 4 * (d >> 6) + ((d >> 2) & 3); }
  return ((ks >> 1) * 4 + tig) * 8 + (ks & 1) * 4 + (c & 1) * 2 + (c >> 1);
}
// k_slot of channel d + 32 j less that of channel d < 32
template <int BK>
__device__ __forceinline__ constexpr int k_slot_step(int j) { return BK == 1 ? 8 * j : 16 * (j & 1) + 64 * (j >> 1); }

// One warp stages window tokens [tb, tb + 16) (rows at or beyond t1 are zero-filled); no commit.  With a fused
// append the newest row (index r - 1) is not in the window yet: it comes from the step's input.
template <int WROW>
__device__ __forceinline__ void window_stage(const DecodeParams& p, const DecodeLayer& L, int tb, int t1, int bh,
                                             uint32_t wbuf, int lane) {
  const size_t row0 = (size_t)bh * p.dm.R;
  const uint8_t* wk = reinterpret_cast<const uint8_t*>(L.L.win_k);
  const uint8_t* wv = reinterpret_cast<const uint8_t*>(L.L.win_v);
  constexpr int CPR = D / 8;
#pragma unroll
  for (int i = 0; i < CPR / 2; ++i) {
    const int chunk = lane + 32 * i, row = chunk / CPR, c = chunk % CPR;
    const uint32_t dk = wbuf + row * WROW + c * 16, dv = dk + 16 * WROW;
    if (tb + row < t1) {
      const size_t off = (row0 + tb + row) * (2 * D) + c * 16;
      if (L.K_new != nullptr && tb + row == p.r - 1) {
        const size_t noff = (size_t)bh * (2 * D) + c * 16;
        cp_async16(dk, reinterpret_cast<const uint8_t*>(L.K_new) + noff);
        cp_async16(dv, reinterpret_cast<const uint8_t*>(L.V_new) + noff);
      } else {
        cp_async16(dk, wk + off);
        cp_async16(dv, wv + off);
      }
    } else {
      sts128(dk, 0u, 0u, 0u, 0u);
      sts128(dv, 0u, 0u, 0u, 0u);
    }
  }
}

// Fused append: the staged tile [tb, tb + 16) holds the token of this step (row r - 1); the warp stores it into the
// window, keys by lanes 0..15, values by lanes 16..31.
template <int WROW>
__device__ __forceinline__ void window_store_new(const DecodeParams& p, const DecodeLayer& L, int tb, int bh,
                                                 uint32_t wbuf, int lane) {
  const int row = p.r - 1 - tb, c = lane & 15;
  if (c < D / 8) {
    const uint4 v = lds128(wbuf + (lane >> 4) * 16 * WROW + row * WROW + c * 16);
    uint8_t* win = reinterpret_cast<uint8_t*>(lane < 16 ? L.L.win_k : L.L.win_v);
    *reinterpret_cast<uint4*>(win + ((size_t)bh * p.dm.R + (p.r - 1)) * (2 * D) + c * 16) = v;
  }
}

// One warp folds the staged tile (n_valid of its 16 tokens exist) into the softmax state of four heads (head of a
// thread: tig; the operand's odd columns are zero): S^T = K q^T with tokens as rows, O^T += V^T P.
// o: this thread's channels 16 mt + gid and + 8 of its head; m, l: its head's reference and sum.
template <int WROW, bool F16>
__device__ __forceinline__ void window_tile(uint32_t wbuf, int n_valid, const uint16_t* qrow, bool real, float scale2,
                                            float (&o)[D / 16][2], float& m, float& l, int lane) {
  constexpr int KS = D / 16;
  const int gid = lane >> 2, tig = lane & 3;
  float s[4] = {0.f, 0.f, 0.f, 0.f};
  const uint32_t ka = wbuf + ((lane & 7) + 8 * ((lane >> 3) & 1)) * WROW + (lane >> 4) * 16;
#pragma unroll
  for (int ks = 0; ks < KS; ++ks) {
    uint32_t a0, a1, a2, a3;
    ldmatrix_x4(ka + ks * 32, a0, a1, a2, a3);
    const uint32_t b0 = real ? *reinterpret_cast<const uint32_t*>(qrow + 16 * ks + 2 * tig) : 0u;
    const uint32_t b1 = real ? *reinterpret_cast<const uint32_t*>(qrow + 16 * ks + 2 * tig + 8) : 0u;
    mma16816<F16>(s, a0, a1, a2, a3, b0, b1);
  }
  const float x0 = gid < n_valid ? s[0] * scale2 : -CUDART_INF_F, x1 = gid + 8 < n_valid ? s[2] * scale2 : -CUDART_INF_F;
  float r = fmaxf(x0, x1);
#pragma unroll
  for (int k = 4; k < 32; k <<= 1) r = fmaxf(r, __shfl_xor_sync(0xffffffffu, r, k));
  const float mn = fmaxf(m, r);  // finite: token 0 of the tile exists
  const float f = ex2(m - mn);
  const float p0 = ex2(x0 - mn), p1 = ex2(x1 - mn);
  m = mn;
  // Numerators as unevaluated sums of three 16-bit numbers (bfloat16: 24 bits, all of an fp32 numerator; a pair would
  // leave errors of 2^-17, four times what everything else here adds up to), the first two in the two columns of the
  // head, the third beside a zero; transposed into B-operand order.
  const uint32_t h0 = pack_io2<F16>(p0, 0.f), h1 = pack_io2<F16>(p1, 0.f);
  const float e0 = p0 - io2_lo<F16>(h0), e1 = p1 - io2_lo<F16>(h1);
  const uint32_t m0 = pack_io2<F16>(p0, e0), m1 = pack_io2<F16>(p1, e1);
  const uint32_t l0 = pack_io2<F16>(e0 - io2_hi<F16>(m0), 0.f), l1 = pack_io2<F16>(e1 - io2_hi<F16>(m1), 0.f);
  const uint32_t bh0 = movmatrix_trans(m0), bh1 = movmatrix_trans(m1), bl0 = movmatrix_trans(l0), bl1 = movmatrix_trans(l1);
  float ps = p0 + p1;
#pragma unroll
  for (int k = 4; k < 32; k <<= 1) ps += __shfl_xor_sync(0xffffffffu, ps, k);
  l = fmaf(l, f, ps);
  const int mi = lane >> 3;
  const uint32_t va = wbuf + 16 * WROW + ((lane & 7) + 8 * (mi >> 1)) * WROW + (mi & 1) * 16;
#pragma unroll
  for (int mt = 0; mt < KS; ++mt) {
    uint32_t a0, a1, a2, a3;
    ldmatrix_x4_trans(va + mt * 32, a0, a1, a2, a3);
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    mma16816<F16>(acc, a0, a1, a2, a3, bl0, bl1);
    mma16816<F16>(acc, a0, a1, a2, a3, bh0, bh1);
    o[mt][0] = fmaf(o[mt][0], f, acc[0] + acc[1]);
    o[mt][1] = fmaf(o[mt][1], f, acc[2] + acc[3]);
  }
}

// four channels c .. c + 3 of query head hq's result
__device__ __forceinline__ void store_out(const DecodeParams& p, const DecodeLayer& L, size_t hq, int c, float4 v) {
  if (p.out_f32) {
    *reinterpret_cast<float4*>(reinterpret_cast<float*>(L.out) + hq * D + c) = v;
  } else {
    uint2 w;
    if (p.f16) w = make_uint2(pack_io2<true>(v.x, v.y), pack_io2<true>(v.z, v.w));
    else w = make_uint2(pack_io2<false>(v.x, v.y), pack_io2<false>(v.z, v.w));
    *reinterpret_cast<uint2*>(reinterpret_cast<uint16_t*>(L.out) + hq * D + c) = w;
  }
}

// Split-K merge by the last CTA of a stream: the CTA takes a ticket after its partials are visible device-wide; the
// CTA that draws the last ticket reads all partials from L2 and writes
// out = sum_s acc_s 2^(m_s-M) / sum_s l_s 2^(m_s-M).  No CTA ever waits for another.
// What it takes is two trips to L2, one for all (m, l) and one for the partials: a warp that went through its share of
// the heads one after the other, both trips for each, made it 2.3 us with four heads and 5.1 us with eight.
// L, part_acc, part_ml: of the first of the CTA's NL layers; weights: NL * G * (ns + 1) floats of shared memory.
template <int NL>
__device__ __forceinline__ void ticket_merge(const DecodeParams& p, const DecodeLayer* L, int ns, int hk, int b,
                                             const float* part_acc, const float* part_ml, unsigned* ticket, int* s_flag,
                                             float* weights) {
  const Dims& dm = p.dm;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, n_warps = blockDim.x >> 5;
  // The barrier orders every thread's partial stores before thread 0's ticket; the ticket is a release (cumulative
  // over what the barrier ordered) and an acquire at device scope, so the CTA that draws the last ticket sees all
  // partials after its second barrier.  The partials are then read from L2 (ld.global.cg).
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned t;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;\n" : "=r"(t) : "l"(ticket) : "memory");
    *s_flag = (t == (unsigned)(ns - 1));
  }
  __syncthreads();
  if (!*s_flag) return;
  const size_t hq0 = (size_t)b * dm.Hq + hk * dm.G, layer_rows = (size_t)dm.B * dm.Hq;
  auto row_of = [&](int v) { return NL == 1 || v < dm.G ? hq0 + v : layer_rows + hq0 + (v - dm.G); };  // head v of the CTA
  // weights[v][s] = 2^(m_s - M), weights[v][ns] = 1 / sum_s l_s 2^(m_s - M)
#pragma unroll 2
  for (int v = warp; v < NL * dm.G; v += n_warps) {
    const float* ml = part_ml + row_of(v) * p.ns_q * 2;
    float* w = weights + v * (ns + 1);
    float M = -CUDART_INF_F, Ls = 0.f;
    if (ns <= 32) {
      const float2 x = lane < ns ? ld_cg2(ml + 2 * lane) : make_float2(-CUDART_INF_F, 0.f);
      M = x.x;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
      const float f = lane < ns ? ex2(x.x - M) : 0.f;
      Ls = x.y * f;
      if (lane < ns) w[lane] = f;
    } else {
      for (int s = lane; s < ns; s += 32) M = fmaxf(M, ld_cg(ml + 2 * s));
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
      for (int s = lane; s < ns; s += 32) {
        const float2 x = ld_cg2(ml + 2 * s);
        const float f = ex2(x.x - M);
        Ls = fmaf(x.y, f, Ls);
        w[s] = f;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) Ls += __shfl_xor_sync(0xffffffffu, Ls, o);
    if (lane == 0) w[ns] = 1.0f / Ls;
  }
  __syncthreads();
  for (int item = threadIdx.x; item < NL * dm.G * (D / 4); item += blockDim.x) {
    const int v = item / (D / 4), c = item % (D / 4) * 4;
    const float* pa = part_acc + row_of(v) * p.ns_q * D + c;
    const float* w = weights + v * (ns + 1);
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int s0 = 0; s0 < ns; s0 += 16) {
      float4 x[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) x[i] = s0 + i < ns ? ld_cg4(pa + (size_t)(s0 + i) * D) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const float f = s0 + i < ns ? w[s0 + i] : 0.f;
        a.x = fmaf(x[i].x, f, a.x);
        a.y = fmaf(x[i].y, f, a.y);
        a.z = fmaf(x[i].z, f, a.z);
        a.w = fmaf(x[i].w, f, a.w);
      }
    }
    const float inv = w[ns];
    const int l = NL == 1 || v < dm.G ? 0 : 1;
    store_out(p, L[l], hq0 + (v - l * dm.G), c, make_float4(a.x * inv, a.y * inv, a.z * inv, a.w * inv));
  }
  if (threadIdx.x == 0) *ticket = 0u;  // ready for the next launch on this stream
}

template <int BK, int BV, int GS, int HP, int NL, bool MANY>
__global__ void __launch_bounds__(Plan<BK, BV, GS, HP, NL, MANY>::WARPS * 32, Plan<BK, BV, GS, HP, NL, MANY>::CTAS)
    decode_mma_kernel(const __grid_constant__ DecodeParams p) {
  using Pl = Plan<BK, BV, GS, HP, NL, MANY>;
  constexpr bool WIDE = Pl::WIDE;
  constexpr int KS = Pl::KS, NG = Pl::NG, NGT = Pl::NGT, W = Pl::WARPS, WROW = Pl::WROW, GC = Pl::GC, CP = Pl::CP;
  constexpr int VH = Pl::VH, SH = Pl::SH, NSET = Pl::NSET, NCOL = Pl::NCOL, NE = Pl::NE;
  constexpr int KWORDS = BK == 2 ? 2 : 1;  // packed words of a token row that a thread expands
  // Where the codes of an operand begin in its halves.  VWIN: quads of tokens (k-steps e) whose value codes one shift of a
  // word puts in place, with weights 2^(BV * (e % VWIN)); 2-bit codes, as far as their sums are limited by the zeros ahead
  // of them, in two shifts.
  constexpr int VWIN = BV == 2 ? 2 : 4;
  constexpr int KBASE = 2, VBASE = BV == 2 ? (VWIN == 2 ? 6 : 2) : 4;
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ __align__(8) unsigned long long bar_mem[2 * W];
  // the CTA's packed data: key codes, value codes, and of each layer key parameters, value parameters
  __shared__ const uint8_t* src_sm[2 + 2 * NL];
  __shared__ __align__(16) int place_sm[8];  // what follows from the CTA's index
  __shared__ int eq_sm[VH];
  __shared__ int s_flag;
  __shared__ uint32_t tmem_base_sm;
  __shared__ volatile int dead_sm;

  const Dims& dm = p.dm;
  const DecodeLayer* const LL = &p.layer[NL * blockIdx.y];
  // (the shuffle tells the compiler that the warp's index, and all that follows from it, is the same in all lanes)
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int gid = lane >> 2, tig = lane & 3, low = gid & 1;
  // head v of the CTA: head v % HP of layer v / HP.  Operand column gid: head col_head (WIDE: gid), slot col_slot;
  // accumulator columns 2 tig and 2 tig + 1: head my_head, slot my_slot (WIDE: heads 2 tig, 2 tig + 1, of layer my_layer)
  const int col_head = WIDE ? gid : (gid >> 1) % VH, col_slot = WIDE ? 0 : (gid >> 1) / VH;
  const int my_head = WIDE ? 2 * tig : tig % VH, my_slot = WIDE ? 0 : tig / VH;
  const int col_layer = NL == 1 ? 0 : col_head / HP, my_layer = NL == 1 ? 0 : my_head / HP;
  const int G = dm.G;

  // The next kernel in the stream may be scheduled at once when all work before this kernel's own predecessor is
  // known to be complete (a chained launch); otherwise only after this kernel's own wait (below), so that a chained
  // successor never starts before the work this kernel waited for has completed.
  if (!Pl::PARK && p.late_wait) grid_dependents_go();

  const uint32_t sm_base = (uint32_t)__cvta_generic_to_shared(smem);
  const uint32_t st = sm_base + warp * Pl::WARP;                     // this warp's stage
  const uint32_t pbuf = st + Pl::OFF_P;
  const uint32_t qb = sm_base + W * Pl::WARP;
  uint16_t* const q_sm = reinterpret_cast<uint16_t*>(smem + W * Pl::WARP + Pl::QB);  // zeros for absent heads
  const uint32_t qf = qb + Pl::QB + Pl::QS + lane * 8;  // this lane's fragments of q
  const uint32_t bar_k = (uint32_t)__cvta_generic_to_shared(&bar_mem[0]) + 16 * warp, bar_v = bar_k + 8;

  if (tid == 0) {
    // CTA -> (stream, split), the splits of a stream side by side
    const unsigned stream = blockIdx.x / (unsigned)p.ns_q;
    const int split = (int)(blockIdx.x - stream * (unsigned)p.ns_q);
    const int bh = (int)stream, b = (int)(stream / (unsigned)dm.Hkv);
    const int nbt = (p.n_q + BT - 1) / BT;  // batches of the stream (the last one may be ragged)
    // the larger shares come last, with the run that may be short
    const int runs = p.deal == 1 ? nbt : (nbt + p.deal - 1) / p.deal;
    int lo, hi, wt0, wt1;
    share_of(runs, p.ns_q, p.ns_q - 1 - split, lo, hi);
    const int b0 = (runs - hi) * p.deal, b1 = min((runs - lo) * p.deal, nbt);
    share_of(p.r, p.ns_q, split, wt0, wt1);
    // half batches (the last half of the stream's last batch may be empty)
    const int halves = b1 > b0 ? 2 * (b1 - b0) - (b1 == nbt && nbt * BT - p.n_q >= TT ? 1 : 0) : 0;
    place_sm[0] = b0; place_sm[1] = halves; place_sm[2] = wt0; place_sm[3] = wt1;
    place_sm[4] = b; place_sm[5] = bh - b * dm.Hkv; place_sm[6] = split;
    dead_sm = 0;
    src_sm[0] = reinterpret_cast<const uint8_t*>(LL[0].L.k_codes) + (size_t)bh * ((size_t)dm.nq_cap * (D * BK / 8)) + (size_t)b0 * (BT * D * BK / 8);
    src_sm[1] = reinterpret_cast<const uint8_t*>(LL[0].L.v_codes) + (size_t)bh * ((size_t)dm.nq_cap * (D * BV / 8)) + (size_t)b0 * (BT * D * BV / 8);
#pragma unroll
    for (int l = 0; l < NL; ++l) {
      src_sm[2 + 2 * l] = reinterpret_cast<const uint8_t*>(LL[l].L.k_meta) + (size_t)bh * ((size_t)(dm.nq_cap / GS) * (4 * D)) + (size_t)b0 * (BT / GS * 4 * D);
      src_sm[3 + 2 * l] = reinterpret_cast<const uint8_t*>(LL[l].L.v_meta) + (size_t)bh * ((size_t)dm.nq_cap * 4 * NG) + (size_t)b0 * (BT * 4 * NG);
    }
  }
  if (lane == 0) {
    mbar_init(bar_k, Pl::P_OVER ? 2 : 1);  // two: codes; scales and zero-points
    mbar_init(bar_v, 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  __syncthreads();
  const int4 place = *reinterpret_cast<const int4*>(place_sm), place2 = *reinterpret_cast<const int4*>(place_sm + 4);
  const int ns = p.ns_q;
  // uniform in a warp, as its index is
  const int b0 = __shfl_sync(0xffffffffu, place.x, 0), halves = __shfl_sync(0xffffffffu, place.y, 0);
  // the rounds of a warp are the half batches warp, warp + W, ... of the CTA's range
  const int rounds = warp < halves ? (halves - 1 - warp) / W + 1 : 0;
  static_assert(W % 2 == 0, "a warp's rounds are all first, or all second halves");

  // Copies of round r into this warp's stage (one lane; the stage is free).  A copy costs a warp its issue, ~33 cycles with a
  // branch on the lane's index (all of them left out of a layer at 32k, four heads: 33.5 of 35.7 us), and half batches have
  // twice as many as batches: calls of one layer had become slower by 5 to 13 % with them.  Behind elect_one, and with one
  // arrival for codes and parameters where they go together: 36.4 -> 35.0 us, MHA at 4k, batch 8 30.8 -> 30.1, a layer of a
  // step of 32 that shares no codes 29.4 -> 28.6 and 25.6 -> 24.7, in pairs 21.4 -> 21.1 and 18.4 -> 17.9.  Measured and
  // not kept: two stages a warp (the waits were not it: 35.8), whole batches a round with one copy each (36.1; one head
  // 3 % faster, pairs slower), products of more row tiles at a time, q kept in registers (no change).
  auto half_of = [&](int r) { return (unsigned)(warp + W * r); };
  struct Sources { const uint8_t *codes, *params[NL]; };
  // read before the copies, which are not reordered (eight heads: by all lanes, before the branch, with less to spill: pairs of
  // three heads, groups of 64, 263.5 -> 261.8 us; five heads, groups of 64, 153.5 -> 150.2)
  auto sources = [&](int kind) {
    Sources s;
    s.codes = src_sm[kind];
#pragma unroll
    for (int l = 0; l < NL; ++l) s.params[l] = src_sm[2 + 2 * l + kind];
    return s;
  };
  auto load_key_codes = [&](int r, const Sources& s) {
    mbar_expect_tx(bar_k, Pl::KCODES + (Pl::P_OVER ? 0 : NL * Pl::KM));
    bulk_load(st, s.codes + (size_t)half_of(r) * Pl::KCODES, Pl::KCODES, bar_k);
  };
  auto load_key_params = [&](int r, const Sources& s) {
    if (Pl::P_OVER) mbar_expect_tx(bar_k, NL * Pl::KM);
#pragma unroll
    for (int l = 0; l < NL; ++l) bulk_load(st + Pl::OFF_KM + l * Pl::KM, s.params[l] + (size_t)half_of(r) * Pl::KM, Pl::KM, bar_k);
  };
  auto load_values = [&](int r, const Sources& s) {
    mbar_expect_tx(bar_v, NL * Pl::VM + Pl::VCODES);
    bulk_load(st + Pl::OFF_V, s.codes + (size_t)(BV == 2 ? half_of(r) : half_of(r) >> 1) * Pl::VCODES, Pl::VCODES, bar_v);
#pragma unroll
    for (int l = 0; l < NL; ++l) bulk_load(st + Pl::OFF_VM + l * Pl::VROOM, s.params[l] + (size_t)half_of(r) * Pl::VM, Pl::VM, bar_v);
  };

  if (lane == 0) {
    // Packed data that earlier calls completed may be fetched while the preceding kernel still runs; when a pack
    // kernel may have written it since this layer's last decode, the first copies wait for that kernel.
    if (!p.early_fetch) grid_dependency_wait();
    if (rounds > 0) {
      const Sources sk = sources(0), sv = sources(1);
      load_key_codes(0, sk);
      load_key_params(0, sk);
      load_values(0, sv);
    }
  }
  __syncwarp();
  if (!p.late_wait) grid_dependency_wait();  // q may come from the preceding kernel
  // Tensor memory is asked for after the wait (a chained launch: its predecessor, a launch of this kernel, waited, and
  // the tensor memory of an SM serves all of their CTAs that fit it): a CTA of the preceding kernel that shares the SM may
  // still have to get its own, and this CTA, which waits for it, would be in its way.  For the same reason the next kernel
  // comes after it.
  if constexpr (Pl::PARK) {
    if (warp == W - 1) {
      tmem_alloc((uint32_t)__cvta_generic_to_shared(&tmem_base_sm), Pl::TMEM);
      grid_dependents_go();
    }
  } else {
    if (!p.late_wait) grid_dependents_go();
  }

  // ---- q, and the exponents that put a head's largest |q| into [1, 2) ----
  static_assert(VH * D / 8 <= W * 32, "a vector a thread");
  if (tid < VH * D / 8) {
    const int v = tid / (D / 8), layer = v / HP, h = v % HP;
    uint4 x = make_uint4(0u, 0u, 0u, 0u);
    if (h < G) x = reinterpret_cast<const uint4*>(LL[layer].q + ((size_t)place2.x * dm.Hq + place2.y * G + h) * D)[tid % (D / 8)];
    reinterpret_cast<uint4*>(q_sm)[tid] = x;
    const uint32_t sign = 0x7fff7fffu;  // both formats order like their bits without the sign
    uint32_t mx = __vmaxu2(__vmaxu2(x.x & sign, x.y & sign), __vmaxu2(x.z & sign, x.w & sign));
#pragma unroll
    for (int k = 1; k < D / 8; k <<= 1) mx = __vmaxu2(mx, __shfl_xor_sync(VH * D / 8 >= 32 ? 0xffffffffu : (1u << (VH * D / 8 & 31)) - 1u, mx, k));
    const float qmax = io_to_f(max(mx & 0xffffu, mx >> 16), p.f16);
    if (tid % (D / 8) == 0) eq_sm[v] = qmax > 0.f ? max(-100, min(100, -exponent_of(qmax))) : 0;
  }
  __syncthreads();
  // B fragments of the zero-point products, for zero-points as they are stored (position pos holds channel
  // (pos % (D / 32)) * 32 + pos / (D / 32)), for a set of heads: rows = token groups; even columns take the first half
  // of the positions, odd columns the second (whose zero-points sit in rows 4 and up).
  for (int i = warp; i < NSET * KS / 2; i += W) {
    const int kp = i % (KS / 2), h = SH * (i / (KS / 2)) + (gid >> 1) % SH;
    const float e2 = pow2i(eq_sm[h] + Q_BIAS_EXP);
    float v[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int pos = low * (D / 2) + (kp >> 1) * 32 + tig * 8 + (kp & 1) * 4 + c;
      const int d = (pos % (D / 32)) * 32 + pos / (D / 32);
      v[c] = io_to_f(q_sm[h * D + d], p.f16) * e2;
    }
    sts64(qb + ((i >> 1) * 32 + lane) * 16 + (i & 1) * 8, pack_io2<true>(v[0], v[1]), pack_io2<true>(v[2], v[3]));
  }
  {  // largest |q| in [2^14, 2^15); the key scales carry the rest of the exponent
    for (int ks = warp; ks < KS; ks += W) {
      const float e2 = pow2i(eq_sm[col_head] + 14 - k_weight<BK>(ks));
      const uint2 v = *reinterpret_cast<const uint2*>(q_sm + col_head * D + k_channel<BK>(ks, tig, 0));
      sts64(qf + ks * 256, pack_io2<true>(io_to_f(v.x & 0xffffu, p.f16) * e2, io_to_f(v.y & 0xffffu, p.f16) * e2),
            pack_io2<true>(io_to_f(v.x >> 16, p.f16) * e2, io_to_f(v.y >> 16, p.f16) * e2));
    }
  }
  if constexpr (Pl::PARK) tc_fence_before();
  __syncthreads();
  if constexpr (Pl::PARK) tc_fence_after();
  float cq[NCOL];  // of the heads of this thread's columns; of the head whose zero-point products it adds up
#pragma unroll
  for (int j = 0; j < NCOL; ++j) cq[j] = p.scale * 1.4426950408889634f * pow2i(-eq_sm[my_head + j]);
  const float cz = WIDE ? p.scale * 1.4426950408889634f * pow2i(-eq_sm[4 * (lane >> 4) + tig]) : cq[0];

  const uint32_t low_mask = low ? 0xffffffffu : 0u;
  // The products q s are taken times 2^Ek of their layer: up to two heads a layer, the factor (at most 1) is q's, at the
  // product, else the scales'.  ek2: that factor as a pair of fp16; k_in: for which bits of the round's largest scale (low
  // half: from, high half: how many) the exponent stays.
  uint32_t ek2[NL], k_in[NL], eq2 = 0u;  // eq2: ek2 of this thread's operand column
  float ck[NCOL];
#pragma unroll
  for (int j = 0; j < NCOL; ++j) ck[j] = 0.f;
  auto set_unit = [&](int l, int e) {
    const float unit = pow2i(code_exp(KBASE) - 14 - e);
#pragma unroll
    for (int j = 0; j < NCOL; ++j) ck[j] = NL == 1 || my_layer == l ? cq[j] * unit : ck[j];
  };
  auto q_pair = [&](int ks) {
    uint2 q = lds64(qf + ks * 256);
    if constexpr (Pl::Q_FACTOR) {
      q.x = hmul2(q.x, eq2);
      q.y = hmul2(q.y, eq2);
    }
    return q;
  };

  // Softmax state of the heads of this thread's columns: reference mr (log2 units, an integer; 0 until the first round
  // sets it).  Value sums acc (PARK: in tensor memory between the rounds): of row tile mt the products' four (WIDE: of hi,
  // then of lo).  zacc[part]: rows gid: the zero-point products of layer gid / 4, channel group gid % 4 (one layer: gid % NG), rows
  // 8 and up: the sum of the numerators; columns hi and lo (WIDE: columns heads, hi and lo apart).
  const uint32_t t_acc = Pl::PARK ? tmem_base_sm + ((uint32_t)(warp & 3) << 21) + (warp >> 2) * Pl::TCOLS : 0u;
  float acc[Pl::PARK ? 1 : KS * NCOL][4];
  constexpr int MT = GC * KS / CP;                          // row tiles of a channel part of the value products
  // that are taken at a time (eight heads: one; with two, 80 bytes more of spills at groups of 64, 724 us a step for 705 at 8k); their columns
  constexpr int MTS = MT < 2 || WIDE ? 1 : 2, TV = MTS * 4 * NCOL;
  float mr[NCOL], zacc[NCOL][4];
  uint32_t ev2[NL];  // value scales are taken times 2^Ev: a pair of fp16 (0: not set)
#pragma unroll
  for (int l = 0; l < NL; ++l) ek2[l] = ev2[l] = k_in[l] = 0u;
#pragma unroll
  for (int j = 0; j < NCOL; ++j) {
    mr[j] = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) zacc[j][i] = 0.f;
  }
  // all value sums of columns j times f[j] (rare)
  auto scale_sums = [&](const float (&f)[NCOL]) {
    if constexpr (Pl::PARK) {
      tc_wait_st();
#pragma unroll 1
      for (int c = 0; c < Pl::TCOLS; c += 8) {
        uint32_t a[8];
        tmem_ld<8>(t_acc + c, a);
        tc_wait_ld();
#pragma unroll
        for (int i = 0; i < 8; ++i) a[i] = __float_as_uint(__uint_as_float(a[i]) * f[WIDE ? i & 1 : 0]);
        tmem_st<8>(t_acc + c, a);
      }
      tc_wait_st();
    } else {
#pragma unroll
      for (int i = 0; i < KS * NCOL; ++i)
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[i][k] *= f[WIDE ? k & 1 : 0];
    }
  };
  if constexpr (Pl::PARK) {
    uint32_t zero[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) zero[i] = 0u;
#pragma unroll
    for (int c = 0; c < Pl::TCOLS; c += 8) tmem_st<8>(t_acc + c, zero);
  } else {
#pragma unroll
    for (int i = 0; i < KS * NCOL; ++i) acc[i][0] = acc[i][1] = acc[i][2] = acc[i][3] = 0.f;
  }
  const unsigned layer0 = NL == 2 ? __ballot_sync(0xffffffffu, my_layer == 0) : 0xffffffffu;
  const unsigned my_lanes = my_layer == 0 ? layer0 : ~layer0;  // lanes with heads of this thread's layer
  // weight of the codes of this lane's tokens in the value words (the token of row gid is in quad (gid >> 1) of its tile)
  const int wt = BV * ((gid >> 1) % VWIN);
  const float off = (float)(P_EXP - wt);
  const int tok0 = 4 * (gid >> 1) + (gid & 1);                       // token of row gid, tile 0; the other rows: + 2, + 16
  const uint32_t kz_lane = st + Pl::OFF_KM + (gid & (NGT - 1)) * 4 * D + 2 * D + (gid >> 2) * D + tig * 16;  // zero-points of its row
  const uint32_t qb_lane = qb + lane * 16;
  const uint32_t kc_lane = st + tok0 * 16 + tig * 4;
  const uint32_t km_read = st + Pl::OFF_KM + lane * (D / 16), km_write = st + Pl::OFF_KM + 2 * k_slot<BK>(lane);
  const uint32_t km_lane = st + Pl::OFF_KM + (NL == 2 ? col_layer * Pl::KM : 0) + tig * 16;
  // Lane column tig owns the tokens 16 tig ... of a round in the value products: in 2 bits word tig of a channel's chunk,
  // in 1 bit a half of word tig / 2 (of the two that this half of the batch has), shifted so that its codes begin at bit
  // VBASE.
  const uint32_t vc_lane = st + Pl::OFF_V + gid * 16 + (BV == 2 ? tig : 2 * (warp & 1) + (tig >> 1)) * 4;
  const int shift_up = BV == 2 ? VBASE : (tig & 1 ? 0 : 4), shift_down = BV == 2 ? 8 - VBASE : (tig & 1 ? 8 : 4);
  const uint32_t vm_read = st + Pl::OFF_VM + (4 * (lane >> 1) + (lane & 1)) * (4 * NG), vm_write = st + Pl::OFF_VM + 4 * lane;
  const uint32_t vs_lane = st + Pl::OFF_VM + (NL == 2 ? col_layer * Pl::VROOM : 0) + tig * 32;  // the scales of its pairs
  const uint32_t vz_lane = st + Pl::OFF_VM + (NL == 2 ? (gid >> 2) * Pl::VROOM : 0) + Pl::VZ + (NL == 2 ? (gid & 3) % NG : gid % NG) * Pl::VZROW + tig * 32;
  // Numerators.  WIDE: 16-byte cells (two pairs of tokens) of head v, tile s, quad k in the tile: 128 bytes for each
  // (v >> 1, k), in it the cell of (s, v & 1), exclusive-or'ed with (v >> 1, k & 1), so that the cells which a warp reads
  // or writes together fall into different banks.
  const uint32_t p_st = WIDE ? pbuf + ((tig * 4 + (gid >> 1)) << 7) + ((tig << 1 | ((gid >> 1) & 1)) << 4) + (gid & 1) * 8
                             : pbuf + my_head * Pl::PH + gid * 8;
  const uint32_t p_ld = WIDE ? pbuf + ((gid >> 1) << 9) + ((((tig << 1) | (gid & 1)) ^ ((gid >> 1) << 1)) << 4)
                             : pbuf + col_head * Pl::PH + tig * Pl::PT;
  // row tile of 16 tokens (of the round's four) of this thread's logits x[n]
  auto tile_of = [&](int n) { return GC == 1 ? n : (GC == 2 ? 2 * my_slot + n : 2 * (my_slot & 1) + (my_slot >> 1)); };

  int last_k = 0, last_v = 0;  // rounds whose key codes, values were copied last
#pragma unroll 1
  for (int r = 0; r < rounds; ++r) {
    const int valid = min(TT, p.n_q - b0 * BT - (warp + W * r) * TT);  // < TT only in the stream's last round
    if (!__all_sync(0xffffffffu, mbar_wait(bar_k, r & 1, &dead_sm))) break;

    if (valid < TT) {  // what no token has reached may be anything: no scale, no zero-point
      for (int i = lane; i < NL * NGT * D; i += 32) {
        const int l = i / (NGT * D), g = i / D % NGT;
        if (g * GS >= valid) sts32(st + Pl::OFF_KM + l * Pl::KM + g * 4 * D + 4 * (i % D), 0u);
      }
      __syncwarp();
    }
    // ---- keys: scales into the order of the operand slots (in place) ----
#pragma unroll
    for (int l = 0; l < NL; ++l) {
      constexpr int V = D / 32;
      uint32_t s[NGT][V / 2];
      auto read = [&]() {
#pragma unroll
        for (int g = 0; g < NGT; ++g) {
          const uint2 x = lds64(km_read + l * Pl::KM + g * 4 * D);
          s[g][0] = x.x; s[g][1] = x.y;
        }
      };
      auto scale = [&]() {
#pragma unroll
        for (int g = 0; g < NGT; ++g)
#pragma unroll
          for (int j = 0; j < V / 2; ++j) s[g][j] = hmul2(s[g][j], ek2[l]);
      };
      auto largest = [&]() {  // the bits of an fp16
        uint32_t mx = 0u;
#pragma unroll
        for (int g = 0; g < NGT; ++g)
#pragma unroll
          for (int j = 0; j < V / 2; ++j) mx = __vmaxu2(mx, s[g][j]);
        return redux_max_u32(max(mx & 0xffffu, mx >> 16));
      };
      read();
      if constexpr (Pl::Q_FACTOR) {
        // The largest scale of the round times 2^Ek in [2^-7, 1), Ek at most 0: |q s| below 2^15, scales as they are
        // stored.  Ek moves only outside that.
        const uint32_t mx = largest();
        if (mx - (k_in[l] & 0xffffu) >= k_in[l] >> 16) {
          const float smax = f16_to_f(mx);
          const int e = smax >= 0.5f ? max(-16, -1 - exponent_of(smax)) : 0;
          const float f = pow2i(e);
          ek2[l] = pack_io2<true>(f, f);
          k_in[l] = e < 0 ? (uint32_t)(8 - e) << 10 | 0x1c000000u : 0x3c000000u;
          if (NL == 1 || col_layer == l) eq2 = ek2[l];
          set_unit(l, e);
        }
      } else {
        // The largest scale of the round times 2^Ek in [2^-4, 1): |q s| below 2^15, and a scale keeps its 11 bits down to
        // 2^-10 of the largest.  Ek moves only outside that, and no further than 15.
        bool moved = r == 0;
        if (r > 0) {
          scale();
          moved = largest() - 0x2c00u >= 0x1000u;
          if (moved) read();
        }
        if (moved) {
          const float smax = f16_to_f(largest());
          const int es = smax > 0.f ? exponent_of(smax) : -24, e = min(15, -1 - es);
          const float f = pow2i(e);
          ek2[l] = pack_io2<true>(f, f);
          set_unit(l, e);
          scale();
        }
      }
      __syncwarp();
#pragma unroll
      for (int g = 0; g < NGT; ++g)
#pragma unroll
        for (int j = 0; j < V; ++j)
          sts16(km_write + l * Pl::KM + g * 4 * D + 2 * k_slot_step<BK>(j), j & 1 ? s[g][j / 2] >> 16 : s[g][j / 2]);
    }
    __syncwarp();
    // Logits x[n][r][j] of row gid + 8 r (tokens 2 r further) of tile tile_of(n), head my_head + j; less the reference and
    // with the exponent `off`.
    float x[NE][2][NCOL];
    float zb;  // zero-points: sum_d q_d z_d, lane 16 * set + 4 * group + head of the set
    {
      // Rows: groups, first and second half of the channels.  A vector of zero-points is an operand as it is: rows gid get
      // its first and third words, rows gid + 8 its second and fourth; the products with their q, of rows gid in zc, of
      // rows gid + 8 in zd (the rest of both is of no use).
      float zc[2][4], zd[2][4];
#pragma unroll
      for (int n = 0; n < 2; ++n)
#pragma unroll
        for (int k = 0; k < 4; ++k) zc[n][k] = zd[n][k] = 0.f;
#pragma unroll
      for (int n = 0; n < (WIDE ? NSET : NL); ++n) {
        const int l = NL == 2 ? n : 0, set = WIDE ? n : 0;
        const uint32_t za = kz_lane + l * Pl::KM;
#pragma unroll
        for (int kp = 0; kp < KS / 4; ++kp) {
          const uint4 a = lds128(za + kp * 64);
          const uint4 q = lds128(qb_lane + (set * KS / 4 + kp) * 512);
          mma_f16(zc[n], a.x, a.y, a.z, a.w, q.x, q.z);
          mma_f16(zd[n], a.x, a.y, a.z, a.w, q.y, q.w);
        }
      }
      auto row = [&](int n, int col) { return zc[n][col] + zd[n][2 + col]; };
      if constexpr (WIDE) {  // lanes 0 .. 15 add up the first set, the others the second
        const float v = __shfl_xor_sync(0xffffffffu, lane < 16 ? row(1, 0) : row(0, 1), 16);
        zb = (lane < 16 ? row(0, 0) : row(1, 1)) + v;
      } else {
        const float z0 = NL == 2 && my_layer == 1 ? row(1, 0) : row(0, 0), z1 = NL == 2 && my_layer == 1 ? row(1, 1) : row(0, 1);
        zb = z0 + __shfl_xor_sync(0xffffffffu, z1, 16);
      }
      zb *= cz * (1.f / (float)(1 << Q_BIAS_EXP));
    }
    // ---- keys: q . c ----
    // packed words of rows gid, gid + 8 of both tiles of unit u (32 tokens): even bytes, odd bytes
    auto load_rows = [&](int u, int kw, uint32_t (&w)[2][2], uint32_t (&w8)[2][2]) {
#pragma unroll
      for (int t = 0; t < 2; ++t)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int tk = 16 * t + 2 * h;
          const uint32_t raw = lds32(kc_lane + u * (32 * D * BK / 8) + kw * 512 + tk * 16);
          w[t][h] = byte_pair_up(raw, 2);
          w8[t][h] = byte_pair_down(raw, 6);
        }
    };
    auto key_pair = [](uint32_t w, int k) { return code_pair<BK, KBASE>(w, BK == 2 ? k & 3 : k); };
    constexpr int KPW = KS / KWORDS;  // k-steps a word serves
    if constexpr (WIDE) {
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        float chi[2][4], clo[2][4];
#pragma unroll
        for (int kw = 0; kw < KWORDS; ++kw) {
          uint32_t w[2][2], w8[2][2];
          load_rows(u, kw, w, w8);
          const uint32_t sa = km_lane + u * 32 / GS * 4 * D + kw * (KPW / 2) * 64;
          uint4 sv;
#pragma unroll
          for (int k = 0; k < KPW; ++k) {
            if ((k & 1) == 0) sv = lds128(sa + (k / 2) * 64);
            const uint32_t s0 = k & 1 ? sv.z : sv.x, s1 = k & 1 ? sv.w : sv.y;
            const int ks = kw * KPW + k;
            const uint2 q = q_pair(ks);
            const uint32_t h0 = hmul2(q.x, s0), h1 = hmul2(q.y, s1), l0 = product_rest(q.x, s0, h0), l1 = product_rest(q.y, s1, h1);
#pragma unroll
            for (int t = 0; t < 2; ++t) {
              const uint32_t a0 = key_pair(w[t][0], k), a1 = key_pair(w[t][1], k);
              const uint32_t a2 = key_pair(w8[t][0], k), a3 = key_pair(w8[t][1], k);
              if (ks == 0) {
                mma_f16_first(chi[t], a0, a1, a2, a3, h0, h1);
                mma_f16_first(clo[t], a0, a1, a2, a3, l0, l1);
              } else {
                mma_f16(chi[t], a0, a1, a2, a3, h0, h1);
                mma_f16(clo[t], a0, a1, a2, a3, l0, l1);
              }
            }
          }
        }
#pragma unroll
        for (int j = 0; j < NCOL; ++j) {
          const int g = u * 32 / GS;
          const float bias = (__shfl_sync(0xffffffffu, zb, 16 * (tig >> 1) + 4 * g + 2 * (tig & 1) + j) - mr[j]) + off;
#pragma unroll
          for (int t = 0; t < 2; ++t)
#pragma unroll
            for (int h = 0; h < 2; ++h) x[2 * u + t][h][j] = fmaf(chi[t][2 * h + j] + clo[t][2 * h + j], ck[j], bias);
        }
      }
    } else if constexpr (GC == 1) {
      constexpr int UG = GS / 32;  // units of a group
#pragma unroll
      for (int g = 0; g < NGT; ++g) {
        float c[2 * UG][4];
#pragma unroll
        for (int kw = 0; kw < KWORDS; ++kw) {
          uint32_t w[UG][2][2], w8[UG][2][2];
#pragma unroll
          for (int u = 0; u < UG; ++u) load_rows(g * UG + u, kw, w[u], w8[u]);
          const uint32_t sa = km_lane + g * 4 * D + kw * (KPW / 2) * 64;
          uint4 sv;
#pragma unroll
          for (int k = 0; k < KPW; ++k) {
            if ((k & 1) == 0) sv = lds128(sa + (k / 2) * 64);
            const uint32_t s0 = k & 1 ? sv.z : sv.x, s1 = k & 1 ? sv.w : sv.y;
            const int ks = kw * KPW + k;
            const uint2 q = q_pair(ks);
            const uint32_t p0 = product_part(q.x, s0, low), p1 = product_part(q.y, s1, low);
#pragma unroll
            for (int u = 0; u < UG; ++u)
#pragma unroll
              for (int t = 0; t < 2; ++t) {
                const uint32_t a0 = key_pair(w[u][t][0], k), a1 = key_pair(w[u][t][1], k);
                const uint32_t a2 = key_pair(w8[u][t][0], k), a3 = key_pair(w8[u][t][1], k);
                if (ks == 0) mma_f16_first(c[2 * u + t], a0, a1, a2, a3, p0, p1);
                else mma_f16(c[2 * u + t], a0, a1, a2, a3, p0, p1);
              }
          }
        }
        const float bias = (__shfl_sync(0xffffffffu, zb, 4 * g + tig) - mr[0]) + off;
#pragma unroll
        for (int n = 0; n < 2 * UG; ++n)
#pragma unroll
          for (int h = 0; h < 2; ++h) x[2 * g * UG + n][h][0] = fmaf(c[n][2 * h] + c[n][2 * h + 1], ck[0], bias);
      }
    } else {
      // one operand for both units, each in its own column slot (four slots: twice); a unit's logits are in the threads
      // of its slot (four slots: those of a tile)
      uint32_t pp[KS][2];
      const uint32_t sa = km_lane + ((col_slot & 1) * 32 / GS) * 4 * D;
#pragma unroll
      for (int kp = 0; kp < KS / 2; ++kp) {
        const uint4 sv = lds128(sa + kp * 64);
        const uint2 q0 = q_pair(2 * kp), q1 = q_pair(2 * kp + 1);
        pp[2 * kp][0] = product_part(q0.x, sv.x, low);
        pp[2 * kp][1] = product_part(q0.y, sv.y, low);
        pp[2 * kp + 1][0] = product_part(q1.x, sv.z, low);
        pp[2 * kp + 1][1] = product_part(q1.y, sv.w, low);
      }
      const float bias = (__shfl_sync(0xffffffffu, zb, 4 * ((my_slot & 1) * 32 / GS) + tig) - mr[0]) + off;
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        float c[2][4];
#pragma unroll
        for (int kw = 0; kw < KWORDS; ++kw) {
          uint32_t w[2][2], w8[2][2];
          load_rows(u, kw, w, w8);
#pragma unroll
          for (int k = 0; k < KPW; ++k)
#pragma unroll
            for (int t = 0; t < 2; ++t) {
              const uint32_t a0 = key_pair(w[t][0], k), a1 = key_pair(w[t][1], k);
              const uint32_t a2 = key_pair(w8[t][0], k), a3 = key_pair(w8[t][1], k);
              if (kw + k == 0) mma_f16_first(c[t], a0, a1, a2, a3, pp[0][0], pp[0][1]);
              else mma_f16(c[t], a0, a1, a2, a3, pp[kw * KPW + k][0], pp[kw * KPW + k][1]);
            }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          if constexpr (GC == 2) {
#pragma unroll
            for (int t = 0; t < 2; ++t) {
              const float v = fmaf(c[t][2 * h] + c[t][2 * h + 1], ck[0], bias);
              x[t][h][0] = u == 0 || my_slot == 1 ? v : x[t][h][0];
            }
          } else {
            const float v = fmaf(my_slot < 2 ? c[0][2 * h] + c[0][2 * h + 1] : c[1][2 * h] + c[1][2 * h + 1], ck[0], bias);
            x[0][h][0] = u == 0 || (my_slot & 1) == 1 ? v : x[0][h][0];
          }
        }
      }
    }
    // the key half of the stage is free: fetch the keys of this warp's next round
    Sources sk;
    if constexpr (WIDE) sk = sources(0);
    proxy_fence();
    __syncwarp();
    if (r + 1 < rounds) {
      if (elect_one()) {
        if constexpr (!WIDE) sk = sources(0);
        load_key_codes(r + 1, sk);
        if (!Pl::P_OVER) load_key_params(r + 1, sk);
      }
      last_k = r + 1;
    }

    if (valid < TT) {
      __syncwarp();  // (a branch, and not a selection that every round would execute)
#pragma unroll
      for (int n = 0; n < NE; ++n)
#pragma unroll
        for (int h = 0; h < 2; ++h)
          if (16 * tile_of(n) + tok0 + 2 * h >= valid) {
#pragma unroll
            for (int j = 0; j < NCOL; ++j) x[n][h][j] = -CUDART_INF_F;
          }
    }
    // ---- softmax: raise the references of a layer when a logit exceeds one by more than TAU (rare) ----
    float xm[NCOL];
    bool need = false;
#pragma unroll
    for (int j = 0; j < NCOL; ++j) {
      xm[j] = fmaxf(x[0][0][j], x[0][1][j]);
#pragma unroll
      for (int n = 1; n < NE; ++n) xm[j] = fmaxf(fmaxf(xm[j], x[n][0][j]), x[n][1][j]);
      xm[j] -= off;  // above the reference
      need |= xm[j] > TAU;
    }
    const unsigned needed = __ballot_sync(0xffffffffu, need || r == 0);
    if (needed != 0u) {
      float f[NCOL];
#pragma unroll
      for (int j = 0; j < NCOL; ++j) {
        float v = xm[j];
#pragma unroll
        for (int k = WIDE ? 4 : VH; k < 32; k <<= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, k));
        const float up = (needed & my_lanes) != 0u && (r == 0 || v > TAU - 1.f) ? ceilf(v) : 0.f;
        f[j] = ex2(-up);
        mr[j] += up;
#pragma unroll
        for (int n = 0; n < NE; ++n) {
          x[n][0][j] -= up;
          x[n][1][j] -= up;
        }
      }
      if (r > 0) {  // (else nothing has been accumulated yet)
#pragma unroll
        for (int j = 0; j < NCOL; ++j) {
#pragma unroll
          for (int k = 0; k < 4; ++k)
            if constexpr (WIDE) zacc[k & 1][2 * (k >> 1) + j] *= f[j];
            else zacc[0][k] *= f[j];
        }
        scale_sums(f);
      }
    }
    // numerators times 2^P_EXP and divided by the weight of the token's value code, as hi + lo pairs (t, t + 2)
#pragma unroll
    for (int j = 0; j < NCOL; ++j)
#pragma unroll
      for (int n = 0; n < NE; ++n) {
        const float pa = ex2(x[n][0][j]), pb = ex2(x[n][1][j]);
        const uint32_t h = pack_io2<true>(pa, pb);
        const uint32_t lo = pack_io2<true>(pa - io2_lo<true>(h), pb - io2_hi<true>(h));
        if constexpr (WIDE) sts64(p_st ^ ((n << 1 | j) << 4), h, lo);
        else sts64(p_st + tile_of(n) * Pl::PT, h, lo);
      }

    // ---- values: scales and zero-points as pairs of tokens (t, t + 2), in place ----
    if (!__all_sync(0xffffffffu, mbar_wait(bar_v, r & 1, &dead_sm))) break;
    if (valid < TT) {
      for (int i = lane; i < NL * TT * NG; i += 32)
        if (i / NG % TT >= valid) sts32(st + Pl::OFF_VM + i / (TT * NG) * Pl::VROOM + i % (TT * NG) * 4, 0u);
      __syncwarp();
    }
#pragma unroll
    for (int l = 0; l < NL; ++l) {
      uint32_t sp[NG], zp[NG];
      {  // raw rows of the two tokens: NG scales, NG zero-points
        const uint32_t a = vm_read + l * Pl::VROOM;
        uint32_t ra[NG], rb[NG];
        if constexpr (NG == 4) {
          const uint4 x4 = lds128(a), y4 = lds128(a + 32);
          ra[0] = x4.x; ra[1] = x4.y; ra[2] = x4.z; ra[3] = x4.w;
          rb[0] = y4.x; rb[1] = y4.y; rb[2] = y4.z; rb[3] = y4.w;
        } else {
          const uint2 x2 = lds64(a), y2 = lds64(a + 16);
          ra[0] = x2.x; ra[1] = x2.y; rb[0] = y2.x; rb[1] = y2.y;
        }
#pragma unroll
        for (int g = 0; g < NG; ++g) {
          const uint32_t sel = g & 1 ? 0x7632 : 0x5410;
          sp[g] = __byte_perm(ra[g / 2], rb[g / 2], sel);
          zp[g] = __byte_perm(ra[NG / 2 + g / 2], rb[NG / 2 + g / 2], sel);
        }
      }
      uint32_t se[NG];
      auto scale = [&]() {
#pragma unroll
        for (int g = 0; g < NG; ++g) se[g] = hmul2(sp[g], ev2[l]);
      };
      auto largest = [&](const uint32_t (&v)[NG]) {  // the bits of an fp16
        uint32_t mx = 0u;
#pragma unroll
        for (int g = 0; g < NG; ++g) mx = __vmaxu2(mx, v[g]);
        return redux_max_u32(max(mx & 0xffffu, mx >> 16));
      };
      // the largest scale times 2^Ev in [2^-6, 1): the exponent moves only outside that, and no further than 15
      bool moved = r == 0;
      if (r > 0) {
        scale();
        moved = largest(se) - 0x2400u >= 0x1800u;
      }
      if (moved) {
        const float smax = f16_to_f(largest(sp));
        const int es = smax > 0.f ? exponent_of(smax) : -24, e = min(15, -1 - es), before = exponent_of(f16_to_f(ev2[l] & 0xffffu));
        float f[NCOL];
#pragma unroll
        for (int j = 0; j < NCOL; ++j) f[j] = NL == 2 && my_layer != l ? 1.f : pow2i(e - before);
        if (r > 0) scale_sums(f);
        const float ev = pow2i(e);
        ev2[l] = pack_io2<true>(ev, ev);
        scale();
      }
      __syncwarp();
#pragma unroll
      for (int g = 0; g < NG; ++g) {
        sts32(vm_write + l * Pl::VROOM + g * (TT / 2 * 4), se[g]);
        sts32(vm_write + l * Pl::VROOM + Pl::VZ + g * Pl::VZROW, zp[g]);
      }
    }
    __syncwarp();
    // ---- values: the numerators of this lane's column, zero-point products ----
    // of the two pairs (t, t + 2), (t + 1, t + 3) of a quad of tokens e: hi, and what the lo operand needs
    uint32_t ph[4][2], pn[4][2], pl[4][2];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      constexpr uint32_t STEP = BV == 2 ? 0x0800u : 0x0400u;
      const uint32_t we = (0x3C00u + e % VWIN * STEP) * 0x10001u;  // the weight of this step's codes as a pair of fp16
      uint4 hp;
      if constexpr (WIDE) hp = lds128((p_ld ^ ((e & 1) << 4)) + (e << 7));
      else hp = lds128(p_ld + e * 16);
      const uint32_t zo = vz_lane + e * 8;
      const uint2 z = lds64(zo);
      ph[e][0] = hp.x; ph[e][1] = hp.z;
      if constexpr (WIDE) {
        pl[e][0] = hp.y; pl[e][1] = hp.w;
        const uint32_t h0 = hmul2(hp.x, we), h1 = hmul2(hp.z, we), l0 = hmul2(hp.y, we), l1 = hmul2(hp.w, we);
        mma_f16(zacc[0], z.x, ONES, z.y, ONES, h0, h1);
        mma_f16(zacc[1], z.x, ONES, z.y, ONES, l0, l1);
      } else {
        // fma(l, s, fma(h, s, hn * s)): hi where hn = l = 0, lo where hn = -h
        pn[e][0] = (hp.x ^ 0x80008000u) & low_mask; pn[e][1] = (hp.z ^ 0x80008000u) & low_mask;
        pl[e][0] = hp.y & low_mask; pl[e][1] = hp.w & low_mask;
        const uint32_t pz0 = hmul2(low ? hp.y : hp.x, we), pz1 = hmul2(low ? hp.w : hp.z, we);
        mma_f16(zacc[0], z.x, ONES, z.y, ONES, pz0, pz1);
      }
    }
    // ---- values: p . c, one channel part after the other ----
    auto value_pair = [](uint32_t w, int e) { return code_pair<BV, VBASE>(w, e % VWIN); };
    if constexpr (Pl::PARK) tc_wait_st();
#pragma unroll
    for (int vb = 0; vb < CP / GC; ++vb) {
      uint32_t sums[TV];
      if constexpr (Pl::PARK) tmem_ld<TV>(t_acc + vb * (MT * 4 * NCOL), sums);
      const uint32_t sa = vs_lane + (GC * vb + col_slot) * NG / CP * (TT / 2 * 4);
      const uint4 s01 = lds128(sa), s23 = lds128(sa + 16);
      const uint32_t sc[4][2] = {{s01.x, s01.y}, {s01.z, s01.w}, {s23.x, s23.y}, {s23.z, s23.w}};
      uint32_t ps[4][2], pr[4][2];  // p s: hi (not WIDE: hi or lo, by column), lo
#pragma unroll
      for (int e = 0; e < 4; ++e)
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const uint32_t s = sc[e][k];
          if constexpr (WIDE) {
            ps[e][k] = hmul2(ph[e][k], s);
            pr[e][k] = hfma2(pl[e][k], s, product_rest(ph[e][k], s, ps[e][k]));
          } else {
            ps[e][k] = hfma2(pl[e][k], s, hfma2(ph[e][k], s, hmul2(pn[e][k], s)));
          }
        }
#pragma unroll
      for (int m0 = vb * MT; m0 < (vb + 1) * MT; m0 += MTS) {
        if constexpr (Pl::PARK) {
          if (m0 > vb * MT) tmem_ld<TV>(t_acc + m0 * (4 * NCOL), sums);
        }
        // even and odd bytes of rows (channels) 16 mt + gid, + 8; second shifts for the quads from VWIN on
        uint32_t w[4 / VWIN][MTS][2], w8[4 / VWIN][MTS][2];
#pragma unroll
        for (int i = 0; i < MTS; ++i)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const uint32_t raw = lds32(vc_lane + (m0 + i) * 256 + h * 128);
#pragma unroll
            for (int k = 0; k < 4 / VWIN; ++k) {
              w[k][i][h] = byte_pair_up(raw, shift_up - k * BV * VWIN);
              w8[k][i][h] = byte_pair_down(raw, shift_down + k * BV * VWIN);
            }
          }
        float part[MTS * NCOL][4];
        if constexpr (Pl::PARK) {
          tc_wait_ld();
#pragma unroll
          for (int i = 0; i < TV; ++i) part[i / 4][i % 4] = __uint_as_float(sums[i]);
        }
        auto sum_of = [&](int i) -> float (&)[4] {
          if constexpr (Pl::PARK) return part[i];
          else return acc[m0 * NCOL + i];
        };
#pragma unroll
        for (int e = 0; e < 4; ++e)
#pragma unroll
          for (int i = 0; i < MTS; ++i) {
            const int k = e / VWIN;
            const uint32_t a0 = value_pair(w[k][i][0], e), a1 = value_pair(w[k][i][1], e), a2 = value_pair(w8[k][i][0], e), a3 = value_pair(w8[k][i][1], e);
            mma_f16(sum_of(NCOL * i), a0, a1, a2, a3, ps[e][0], ps[e][1]);
            if constexpr (WIDE) mma_f16(sum_of(NCOL * i + 1), a0, a1, a2, a3, pr[e][0], pr[e][1]);
          }
        if constexpr (Pl::PARK) {
#pragma unroll
          for (int i = 0; i < TV; ++i) sums[i] = __float_as_uint(part[i / 4][i % 4]);
          tmem_st<TV>(t_acc + m0 * (4 * NCOL), sums);
        }
      }
    }
    // the value half of the stage and the numerators are free
    Sources sv;
    if constexpr (WIDE) {
      sk = sources(0);
      sv = sources(1);
    }
    proxy_fence();
    __syncwarp();
    if (r + 1 < rounds) {
      if (elect_one()) {
        if constexpr (!WIDE) {
          sk = sources(0);
          sv = sources(1);
        }
        if (Pl::P_OVER) load_key_params(r + 1, sk);
        load_values(r + 1, sv);
      }
      last_v = r + 1;
    }
  }

  // ---- state rows, over the stage: acc, m, l of each head from the packed tokens, then from the window ----
  const int wt0 = place.z, wt1 = place.w, hk = place2.y, b = place2.x, split = place2.z, bh = b * dm.Hkv + hk;
  // The CTA's share of the 16-bit window goes tile by tile to its warps, first to those with the fewest rounds; a warp
  // without rounds has the window's state in place of the packed tokens'.
  const int wtiles = (wt1 - wt0 + 15) / 16;
  auto window_turn = [&](int w) { const int t = w - halves % W; return t < 0 ? t + W : t; };
  if (dead_sm == 0) {  // (else a wait gave up somewhere: copies may be in flight, the stage is not reused)
    float* const ws = reinterpret_cast<float*>(smem + warp * Pl::WARP);
    if (window_turn(warp) < wtiles) {
      const float scale2 = p.scale * 1.4426950408889634f;
      float o[NSET][KS][2], l[NSET], ms[NSET];  // channels 16 mt + gid, + 8 of head SH * s + tig % SH
#pragma unroll
      for (int s = 0; s < NSET; ++s) {
        ms[s] = -CUDART_INF_F;
        l[s] = 0.f;
#pragma unroll
        for (int mt = 0; mt < KS; ++mt) o[s][mt][0] = o[s][mt][1] = 0.f;
      }
#pragma unroll 1
      for (int layer = 0; layer < NL; ++layer) {
        const DecodeLayer& L = LL[layer];
#pragma unroll 1
        for (int tb = wt0 + 16 * window_turn(warp); tb < wt1; tb += 16 * W) {
          window_stage<WROW>(p, L, tb, wt1, bh, st, lane);
          cp_async_commit();
          cp_async_wait_all();
          __syncwarp();
          if (L.K_new != nullptr && tb + 16 > p.r - 1 && wt1 == p.r) window_store_new<WROW>(p, L, tb, bh, st, lane);
#pragma unroll
          for (int s = 0; s < NSET; ++s) {
            if (WIDE && NL == 2 && s != layer) continue;
            const int v = SH * s + (gid >> 1) % SH;  // head of operand column gid
            const bool real = low == 0 && (gid >> 1) / SH == 0 && v % HP < G && v / HP == layer;
            const uint16_t* qrow = q_sm + v * D;
            // layers that share a set: only the threads of this layer's heads take the result
            const bool mine = WIDE || NL == 1 || my_layer == layer;
            float o2[KS][2], m2 = ms[s], l2 = l[s];
#pragma unroll
            for (int mt = 0; mt < KS; ++mt) o2[mt][0] = o[s][mt][0], o2[mt][1] = o[s][mt][1];
            if (p.f16) window_tile<WROW, true>(st, wt1 - tb, qrow, real, scale2, o2, m2, l2, lane);
            else window_tile<WROW, false>(st, wt1 - tb, qrow, real, scale2, o2, m2, l2, lane);
            if (mine) {
              ms[s] = m2;
              l[s] = l2;
#pragma unroll
              for (int mt = 0; mt < KS; ++mt) o[s][mt][0] = o2[mt][0], o[s][mt][1] = o2[mt][1];
            }
          }
          __syncwarp();
        }
      }
#pragma unroll
      for (int s = 0; s < NSET; ++s) {
        float* const row = ws + ((rounds > 0 ? VH : 0) + SH * s + tig % SH) * Pl::MS;
        if (tig / SH == 0) {
#pragma unroll
          for (int mt = 0; mt < KS; ++mt) {
            row[16 * mt + gid] = o[s][mt][0];
            row[16 * mt + gid + 8] = o[s][mt][1];
          }
          if (gid == 0) {
            row[D] = ms[s];
            row[D + 1] = l[s];
          }
        }
      }
    }
    __syncwarp();
    if constexpr (Pl::PARK) tc_wait_st();
    // the packed tokens, in true units
    if (rounds > 0) {
      const float uz = pow2i(-P_EXP);
      const float ua = pow2i(code_exp(VBASE) - P_EXP - exponent_of(f16_to_f((NL == 2 && my_layer == 1 ? ev2[NL - 1] : ev2[0]) & 0xffffu)));
      float z[NCOL];  // row gid < 4 NL: channel group of a layer
#pragma unroll
      for (int j = 0; j < NCOL; ++j) {
        z[j] = (WIDE ? zacc[0][j] + zacc[1 % NCOL][j] : zacc[0][0] + zacc[0][1]) * uz;
        const float sum = (WIDE ? zacc[0][2 + j] + zacc[1 % NCOL][2 + j] : zacc[0][2] + zacc[0][3]) * uz;
        if (gid == 0 && my_slot == 0) {
          ws[(my_head + j) * Pl::MS + D] = mr[j];
          ws[(my_head + j) * Pl::MS + D + 1] = sum;
        }
      }
      float zg[NG][NCOL];  // of this thread's heads
#pragma unroll
      for (int g = 0; g < NG; ++g)
#pragma unroll
        for (int j = 0; j < NCOL; ++j) zg[g][j] = __shfl_sync(0xffffffffu, z[j], (4 * my_layer + g) * 4 + tig);
#pragma unroll
      for (int mt = 0; mt < KS; mt += 2 / NCOL) {
        uint32_t a[8];  // WIDE: hi and lo sums of a row tile; else the sums of two
        if constexpr (Pl::PARK) {
          tmem_ld<8>(t_acc + mt * 4 * NCOL, a);
          tc_wait_ld();
        } else {
#pragma unroll
          for (int i = 0; i < 8; ++i) a[i] = __float_as_uint(acc[mt * NCOL + i / 4][i % 4]);
        }
        auto sum_of = [&](int i, int k) { return __uint_as_float(a[i]) + __uint_as_float(a[k]); };
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int t = 0; t < 2; ++t) {  // WIDE: columns; else row tiles, which the threads of the tile's slot hold
            const int tile = WIDE ? mt : mt + t;
            const float v = WIDE ? sum_of(2 * h + t, 4 + 2 * h + t) : sum_of(4 * t + 2 * h, 4 * t + 2 * h + 1);
            if (GC == 1 || my_slot == (tile / (KS / CP)) % GC)
              ws[(my_head + (WIDE ? t : 0)) * Pl::MS + 16 * tile + gid + 8 * h] = fmaf(v, ua, zg[tile * 16 / GS][WIDE ? t % NCOL : 0]);
          }
      }
    } else if (window_turn(warp) >= wtiles) {  // neither: nothing to add
      for (int i = lane; i < VH * Pl::MS; i += 32) ws[i] = i % Pl::MS == D ? -CUDART_INF_F : 0.f;
    }
  }
  if constexpr (Pl::PARK) tc_fence_before();
  __syncthreads();
  if constexpr (Pl::PARK) {
    tc_fence_after();
    if (warp == W - 1) tmem_dealloc(tmem_base_sm, Pl::TMEM);
  }
  if (p.late_wait) grid_dependency_wait();  // the preceding launch still reads and writes the scratch and its result
  if (dead_sm != 0) {
    // leaving early: no copy of this CTA may still be in flight when its shared memory is released
    if (lane == 0 && rounds > 0) {
      if (Pl::P_OVER && last_v < last_k) mbar_arrive(bar_k);  // (in place of the copies that did not follow the codes)
      for (int it = 0; it < WAIT_LIMIT && !mbar_try_wait(bar_k, last_k & 1); ++it) {}
      for (int it = 0; it < WAIT_LIMIT && !mbar_try_wait(bar_v, last_v & 1); ++it) {}
    }
    if (tid == 0) atomicExch(p.status, 1);
    __syncthreads();
    return;
  }
  // ---- the CTA's state: all warps; then the partial and the merge, or the result itself ----
  const size_t slot = (size_t)blockIdx.y * NL * ((size_t)dm.B * dm.Hq) * p.ns_q;  // the first layer's partials in the scratch
  float* const part_acc = p.part_acc + slot * D;
  float* const part_ml = p.part_ml + slot * 2;
  // turns of the warps with a row of their own for the window
  const int wrow0 = halves < W ? W - halves : 0, wrow1 = wtiles < W ? wtiles : W;
  for (int item = tid; item < NL * G * (D / 4); item += W * 32) {
    const int i = item / (D / 4), d = item % (D / 4) * 4;
    const int layer = NL == 1 || i < G ? 0 : 1, h = i - layer * G;
    auto row = [&](int w, bool window) { return reinterpret_cast<const float*>(smem + w * Pl::WARP) + ((window ? VH : 0) + layer * HP + h) * Pl::MS; };
    float M = -CUDART_INF_F;
#pragma unroll
    for (int w = 0; w < W; ++w) M = fmaxf(M, row(w, false)[D]);
    for (int t = wrow0; t < wrow1; ++t) M = fmaxf(M, row((t + halves) % W, true)[D]);
    float4 A = make_float4(0.f, 0.f, 0.f, 0.f);
    float Ls = 0.f;
    auto add = [&](const float* r) {
      const float4 v = *reinterpret_cast<const float4*>(r + d);
      const float mw = r[D];
      const float f = mw == -CUDART_INF_F ? 0.f : ex2(mw - M);  // a warp without tokens
      A.x = fmaf(v.x, f, A.x);
      A.y = fmaf(v.y, f, A.y);
      A.z = fmaf(v.z, f, A.z);
      A.w = fmaf(v.w, f, A.w);
      Ls = fmaf(r[D + 1], f, Ls);
    };
#pragma unroll
    for (int w = 0; w < W; ++w) add(row(w, false));
    for (int t = wrow0; t < wrow1; ++t) add(row((t + halves) % W, true));
    const size_t hq = (size_t)b * dm.Hq + hk * G + h;
    if (ns == 1) {
      store_out(p, LL[layer], hq, d, make_float4(A.x / Ls, A.y / Ls, A.z / Ls, A.w / Ls));
    } else {
      const size_t at = ((size_t)layer * dm.B * dm.Hq + hq) * p.ns_q + split;
      *reinterpret_cast<float4*>(part_acc + at * D + d) = A;
      if (d == 0) *reinterpret_cast<float2*>(part_ml + at * 2) = make_float2(M, Ls);
    }
  }
  if (ns > 1)
    ticket_merge<NL>(p, LL, ns, hk, b, part_acc, part_ml, p.tickets + (size_t)blockIdx.y * (dm.B * dm.Hkv) + bh, &s_flag,
                        reinterpret_cast<float*>(smem));
}

template <int BK, int BV, int GS, int HP, int NL, bool MANY>
cudaError_t launch_one(const DecodeParams& p, cudaStream_t st) {
  using Pl = Plan<BK, BV, GS, HP, NL, MANY>;
  return launch_dependent(decode_mma_kernel<BK, BV, GS, HP, NL, MANY>, dim3((unsigned)(p.ns_q * p.dm.B * p.dm.Hkv), p.n_layers / NL), dim3(Pl::WARPS * 32),
                          (size_t)Pl::TOTAL, st, p);
}

// Prepares the kernel for the current device.
template <int BK, int BV, int GS, int HP, int NL, bool MANY>
MmaShape shape_one() {
  using Pl = Plan<BK, BV, GS, HP, NL, MANY>;
  auto kernel = decode_mma_kernel<BK, BV, GS, HP, NL, MANY>;
  // the largest shared-memory carve-out: two or three CTAs of this size are to share an SM
  const bool ready = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, Pl::TOTAL) == cudaSuccess &&
                     cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, 100) == cudaSuccess;
  if (!ready) cudaGetLastError();
  return {Pl::WARPS, ready};
}

#define XQ_DISPATCH(FN, ...)                               \
  switch (bk * 100 + bv * 10 + (g == 64)) {                \
    case 220: return FN<2, 2, 32, HP, NL, MANY>(__VA_ARGS__); \
    case 221: return FN<2, 2, 64, HP, NL, MANY>(__VA_ARGS__); \
    case 210: return FN<2, 1, 32, HP, NL, MANY>(__VA_ARGS__); \
    case 211: return FN<2, 1, 64, HP, NL, MANY>(__VA_ARGS__); \
    case 120: return FN<1, 2, 32, HP, NL, MANY>(__VA_ARGS__); \
    case 121: return FN<1, 2, 64, HP, NL, MANY>(__VA_ARGS__); \
    case 110: return FN<1, 1, 32, HP, NL, MANY>(__VA_ARGS__); \
    case 111: return FN<1, 1, 64, HP, NL, MANY>(__VA_ARGS__); \
  }

}  // namespace

template <int HP, int NL, bool MANY>
cudaError_t launch_decode_mma_t(const DecodeParams& p, cudaStream_t st) {
  const int bk = p.layer[0].L.bk, bv = p.layer[0].L.bv, g = p.dm.g;
  XQ_DISPATCH(launch_one, p, st)
  return cudaErrorInvalidValue;
}
template <int HP, int NL, bool MANY>
MmaShape decode_mma_shape_t(int g, int bk, int bv) {
  XQ_DISPATCH(shape_one)
  return MmaShape{1, false};
}

}  // namespace xq
