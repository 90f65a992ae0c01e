// Tensor-core decode attention over the packed cache, head_dim 64: one CTA takes a range of batches of one (layer,
// sequence, kv head) stream, up to 8 query heads.
//
// Every warp works alone on batches of 128 tokens.  Codes are expanded into A fragments of mma.sync.m16n8k16 (fp16),
// scale and zero-point are folded out of the inner products, and the other operand (q_d s_d, or p_t s_tg) is carried as
// an unevaluated sum hi + lo of two fp16 numbers in two of the eight operand columns, as in the kernel for head_dim 128
// (xq_decode_mma.cuh).  What differs: codes are centered normal numbers, with zero-points plus center scales as pairs of
// fp16, so that both sums are as small as the result and no digit is lost where they cancel (as exact as the scalar
// kernel, which served head_dim 64 before: 4.7-5.6e-7 of the result's norm); a batch is one round; every layer is read by
// itself.  A model of this head_dim is small and a call is mostly its start and end: in rounds of half batches, as head_dim
// 128 has them, a pair of tiny layers takes 10.9 us in place of 9.4, a layer at 2000 tokens, 32 streams, four heads, 3.7 us
// of a step in place of 2.9.
#pragma once
#include "xq_internal.h"
#include "xq_mma.cuh"

namespace xq {
namespace {

constexpr int D = 64;              // head dim
constexpr int BT = 128;            // tokens per batch
constexpr float TAU = 3.f;         // log2 units a logit may exceed the softmax reference before it is raised
constexpr int P_EXP = 11;          // numerators are carried times 2^P_EXP (at most 2^(P_EXP + TAU) as fp16)
constexpr int Q_BIAS_EXP = 8;      // exponent of the largest |q| in the zero-point products

// Shared-memory plan.  GS: quantization group, BK / BV: bits.  The eight operand columns are four column
// pairs (hi, lo) of HP heads (1, 2 or 4) times GC = 4 / HP slots: with fewer heads, one operand serves GC token units
// of the keys (or GC channel parts of the values) at once, each row tile reading the columns of its own slot.
// NT: sets of four heads (HP = 4).
template <int BK, int BV, int GS, int HP, int NT>
struct Plan {
  static_assert(NT == 1 || HP == 4, "several sets only of four heads");
  static constexpr int NGT = BT / GS;            // token groups of the keys in a batch
  static constexpr int NG = D / GS;              // channel groups of a value row
  static constexpr int KS = D / 16;              // k-steps of the key products, row tiles of the value products
  static constexpr int GC = 4 / HP;              // slots
  static constexpr int CP = NG > GC ? NG : GC;   // channel parts of the value products: one scale per token each
  static constexpr int KC = BT * D * BK / 8, KM = NGT * 4 * D;  // key codes; scales and zero-points
  static constexpr int VC = BT * D * BV / 8, VM = BT * 4 * NG;  // the same of the values
  static constexpr int OFF_KM = KC, OFF_VC = KC + KM, OFF_VM = KC + KM + VC;
  // value scales, then zero-points, as they are reordered over VM: [pair of tokens][NG] half2, one more row after
  // the pairs of a lane column (bank conflicts)
  static constexpr int VSROW = 4 * NG, VS = 64 * VSROW + 4 * VSROW;
  // centered codes: the second halves of the zero-points, of the values (as VS), of the keys (as the second half of KM)
  static constexpr int OFF_KL = OFF_VM + 3 * VS, KL = NGT * 2 * D;
  static constexpr int STAGE = OFF_KL + KL;
  // numerators: [head][pair of tokens (t, t + 2)] of (hi pair, lo pair), 16 bytes more after every 16 pairs and 32
  // more after every head against bank conflicts
  static constexpr int PH = 64 * 8 + 4 * 16 + 32;
  static constexpr int PBUF = HP * NT * PH;
  static constexpr int WROW = 2 * D + 16;        // a staged window row
  static constexpr int WIN = 32 * WROW;          // 16 key rows, then 16 value rows (over the stage of the warp)
  static constexpr int BODY = STAGE + PBUF;
  static constexpr int WARP = ((BODY > WIN ? BODY : WIN) + 127) / 128 * 128;
  static constexpr int MS = D + 4;               // state row: acc[D], m, l
  static_assert(HP * NT * MS * 4 <= WARP, "a warp's state rows fit its own memory");
  static_assert(MS % 4 == 0, "state rows are read as vectors");
  // after the warps' parts: B fragments of the zero-point products; q as it came
  static constexpr int QB = NT * KS * 32 * 4, QS = HP * NT * D * 2;
  static constexpr int room(int w) { return w * WARP + QB + QS; }
  // Two CTAs per SM, each of as many warps as registers (128, or 168 for eight heads) and shared memory allow.
  static constexpr int CTAS = 2;
  static constexpr int MOST = NT == 1 ? 8 : 6;
  static constexpr int LIMIT = 228 * 1024 / CTAS - 1024 - 512;
  static constexpr int WARPS = room(MOST) <= LIMIT ? MOST : (room(MOST - 1) <= LIMIT ? MOST - 1 : MOST - 2);
  static constexpr int TOTAL = room(WARPS);
  static_assert(TOTAL <= LIMIT, "shared memory");
  static_assert(WARPS * WARP >= HP * NT * (256 + 1) * 4, "the merge's weights");
};

// Code operands: (code - center) * weight * 2^-9, normal numbers, center = (2^BITS - 1) / 2.
constexpr int CODE_EXP = 9;
template <int BITS>
__device__ __forceinline__ float code_center() { return 0.5f * (float)((1 << BITS) - 1); }
// the operand pair of the code bits at 2 + BITS * i of both halves of w; their weight is 2^(BITS * i)
template <int BITS>
__device__ __forceinline__ uint32_t code_pair(uint32_t w, int i) {
  const uint32_t m = w & ((BITS == 2 ? 0x000c000cu : 0x00040004u) << (BITS * i));
  // times 2^13, less center * weight * 2^-9: 1.5 or 0.5 at exponent field 15 - 9 + BITS * i
  const uint32_t c = BITS == 2 ? 0x8200u + ((uint32_t)(6 + 2 * i) << 10) : 0x8000u + ((uint32_t)(5 + i) << 10);
  return hfma2(m, 0x70007000u, c * 0x10001u);
}
// z + center s of a pair of groups as an unevaluated sum of two fp16
template <int BITS>
__device__ __forceinline__ void centered_zero(uint32_t s, uint32_t z, uint32_t& hi, uint32_t& lo) {
  const float a = fmaf(code_center<BITS>(), io2_lo<true>(s), io2_lo<true>(z));
  const float b = fmaf(code_center<BITS>(), io2_hi<true>(s), io2_hi<true>(z));
  hi = pack_io2<true>(a, b);
  lo = pack_io2<true>(a - io2_lo<true>(hi), b - io2_hi<true>(hi));
}

// log2 of the weight that the code of k-slot (step ks, any tig, any pair) carries in its operand
template <int BK>
__device__ __forceinline__ constexpr int k_weight(int ks) { return (BK == 2 ? 2 : 1) * (ks % 4); }
// channel of k-slot c (pairs (0, 2) and (1, 3)) of step ks for lane column tig
template <int BK>
__device__ __forceinline__ int k_channel(int ks, int tig, int c) {
  return 16 * (tig + 4 * (ks / 4)) + 4 * (ks % 4) + c;
}
// Halfword index, inside a key group's D reordered scales, of channel d: per lane column and two k-steps one 16-byte
// vector [step][pair (c, c + 2), pair (c + 1, c + 3)].
template <int BK>
__device__ __forceinline__ int k_slot(int d) {
  int tig, ks;
  const int c = d & 3;
  tig = (d >> 4) & 3;
  ks = 4 * (d >> 6) + ((d >> 2) & 3);
  return ((ks >> 1) * 4 + tig) * 8 + (ks & 1) * 4 + (c & 1) * 2 + (c >> 1);
}
// Row of the reordered value scales that holds token pair p (tokens t = 4 (p / 2) + p % 2 and t + 2) of a batch: a
// spare row after every 16 pairs, so that the rows which the lane columns read together fall into different banks.
__device__ __forceinline__ constexpr int pair_row(int p) { return p + (p >> 4); }

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
// weights: G * (ns + 1) floats of shared memory.
__device__ __forceinline__ void ticket_merge(const DecodeParams& p, const DecodeLayer& L, int ns, int hk, int b,
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
  const size_t hq0 = (size_t)b * dm.Hq + hk * dm.G;
  // weights[h][s] = 2^(m_s - M), weights[h][ns] = 1 / sum_s l_s 2^(m_s - M)
#pragma unroll 2
  for (int h = warp; h < dm.G; h += n_warps) {
    const float* ml = part_ml + (hq0 + h) * p.ns_q * 2;
    float* w = weights + h * (ns + 1);
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
  for (int item = threadIdx.x; item < dm.G * (D / 4); item += blockDim.x) {
    const int h = item / (D / 4), c = item % (D / 4) * 4;
    const float* pa = part_acc + (hq0 + h) * p.ns_q * D + c;
    const float* w = weights + h * (ns + 1);
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int s0 = 0; s0 < ns; s0 += 16) {
      float4 v[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) v[i] = s0 + i < ns ? ld_cg4(pa + (size_t)(s0 + i) * D) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const float f = s0 + i < ns ? w[s0 + i] : 0.f;
        a.x = fmaf(v[i].x, f, a.x);
        a.y = fmaf(v[i].y, f, a.y);
        a.z = fmaf(v[i].z, f, a.z);
        a.w = fmaf(v[i].w, f, a.w);
      }
    }
    const float inv = w[ns];
    store_out(p, L, hq0 + h, c, make_float4(a.x * inv, a.y * inv, a.z * inv, a.w * inv));
  }
  if (threadIdx.x == 0) *ticket = 0u;  // ready for the next launch on this stream
}

template <int BK, int BV, int GS, int HP, int NT>
__global__ void __launch_bounds__(Plan<BK, BV, GS, HP, NT>::WARPS * 32, Plan<BK, BV, GS, HP, NT>::CTAS)
    decode_mma64_kernel(const __grid_constant__ DecodeParams p) {
  using Pl = Plan<BK, BV, GS, HP, NT>;
  constexpr int KS = Pl::KS, NG = Pl::NG, NGT = Pl::NGT, W = Pl::WARPS, WROW = Pl::WROW, GC = Pl::GC, CP = Pl::CP;
  constexpr int VCH = BV;                               // 16-byte chunks of a channel row (128 / BV tokens each)
  constexpr int VE = 8 / BV;                            // k-steps of a value chunk
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ __align__(8) unsigned long long bar_mem[2 * W];
  __shared__ const uint8_t* src_sm[4];  // the CTA's packed data: key codes, key parameters, value codes, value parameters
  __shared__ int s_flag;
  __shared__ volatile int dead_sm;

  const Dims& dm = p.dm;
  const DecodeLayer& L = p.layer[blockIdx.y];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gid = lane >> 2, tig = lane & 3, low = gid & 1;
  // operand column gid: head col_head, slot col_slot; accumulator columns 2 tig and 2 tig + 1: head my_head, slot my_slot
  const int col_head = (gid >> 1) % HP, col_slot = (gid >> 1) / HP, my_head = tig % HP, my_slot = tig / HP;
  const int G = dm.G;

  // The next kernel in the stream may be scheduled at once when all work before this kernel's own predecessor is
  // known to be complete (a chained launch); otherwise only after this kernel's own wait (below), so that a chained
  // successor never starts before the work this kernel waited for has completed.
  if (p.late_wait) grid_dependents_go();

  // CTA -> (stream, split), the splits of a stream side by side
  const int ns = p.ns_q;
  const unsigned stream = blockIdx.x / (unsigned)ns;
  const int split = (int)(blockIdx.x - stream * (unsigned)ns);
  const int hk = (int)(stream % (unsigned)dm.Hkv), b = (int)(stream / (unsigned)dm.Hkv);
  const int bh = b * dm.Hkv + hk;
  const int nbt = (p.n_q + BT - 1) / BT;  // batches of the stream (the last one may be ragged)
  int b0, b1, wt0, wt1;
  {
    // the larger shares come last, with the run that may be short
    const int runs = (nbt + p.deal - 1) / p.deal;
    int lo, hi;
    share_of(runs, ns, ns - 1 - split, lo, hi);
    b0 = (runs - hi) * p.deal;
    b1 = min((runs - lo) * p.deal, nbt);
  }
  share_of(p.r, ns, split, wt0, wt1);
  const int nb = b1 - b0;

  const uint32_t sm_base = (uint32_t)__cvta_generic_to_shared(smem);
  const uint32_t st = sm_base + warp * Pl::WARP;                     // this warp's stage
  const uint32_t pbuf = st + Pl::STAGE;
  const uint32_t qb = sm_base + W * Pl::WARP;
  uint16_t* const q_sm = reinterpret_cast<uint16_t*>(smem + W * Pl::WARP + Pl::QB);  // zeros for absent heads
  const uint32_t bar_k = (uint32_t)__cvta_generic_to_shared(&bar_mem[0]) + 16 * warp, bar_v = bar_k + 8;

  // Copies of batch j of this CTA's range into this warp's stage (one lane; the stage is free)
  auto load_keys = [&](int j) {
    const uint8_t *gk = src_sm[0] + (size_t)(unsigned)j * Pl::KC, *gm = src_sm[1] + (size_t)(unsigned)j * Pl::KM;
    mbar_expect_tx(bar_k, Pl::KC + Pl::KM);
    bulk_load(st, gk, Pl::KC, bar_k);
    bulk_load(st + Pl::OFF_KM, gm, Pl::KM, bar_k);
  };
  auto load_values = [&](int j) {
    const uint8_t *gv = src_sm[2] + (size_t)(unsigned)j * Pl::VC, *gm = src_sm[3] + (size_t)(unsigned)j * Pl::VM;
    mbar_expect_tx(bar_v, Pl::VC + Pl::VM);
    bulk_load(st + Pl::OFF_VC, gv, Pl::VC, bar_v);
    bulk_load(st + Pl::OFF_VM, gm, Pl::VM, bar_v);
  };

  if (tid == 0) {
    dead_sm = 0;
    src_sm[0] = reinterpret_cast<const uint8_t*>(L.L.k_codes) + (size_t)bh * ((size_t)dm.nq_cap * (D * BK / 8)) + (size_t)b0 * Pl::KC;
    src_sm[1] = reinterpret_cast<const uint8_t*>(L.L.k_meta) + (size_t)bh * ((size_t)(dm.nq_cap / GS) * (4 * D)) + (size_t)b0 * Pl::KM;
    src_sm[2] = reinterpret_cast<const uint8_t*>(L.L.v_codes) + (size_t)bh * ((size_t)dm.nq_cap * (D * BV / 8)) + (size_t)b0 * Pl::VC;
    src_sm[3] = reinterpret_cast<const uint8_t*>(L.L.v_meta) + (size_t)bh * ((size_t)dm.nq_cap * 4 * NG) + (size_t)b0 * Pl::VM;
  }
  if (lane == 0) {
    mbar_init(bar_k, 1);
    mbar_init(bar_v, 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  __syncthreads();
  if (lane == 0) {
    // Packed data that earlier calls completed may be fetched while the preceding kernel still runs; when a pack
    // kernel may have written it since this layer's last decode, the first copies wait for that kernel.
    if (!p.early_fetch) grid_dependency_wait();
    if (warp < nb) {
      load_keys(warp);
      load_values(warp);
    }
  }
  __syncwarp();
  if (!p.late_wait) {
    grid_dependency_wait();  // q may come from the preceding kernel
    grid_dependents_go();    // whatever this kernel waited for is complete for its successor too
  }

  // ---- q ----
  for (int i = tid; i < HP * NT * D / 8; i += W * 32) {
    const bool real = i / (D / 8) < G;
    const uint4* src = reinterpret_cast<const uint4*>(L.q + ((size_t)b * dm.Hq + hk * G) * D);
    reinterpret_cast<uint4*>(q_sm)[i] = real ? src[i] : make_uint4(0u, 0u, 0u, 0u);
  }
  __syncthreads();
  // exponents that put a head's largest |q| into [1, 2): each warp finds those of all heads; lane h keeps head h's
  int eq_lane = 0;
#pragma unroll
  for (int h = 0; h < HP * NT; ++h) {
    float am = 0.f;
#pragma unroll
    for (int j = 0; j < D / 64; ++j) {
      const uint32_t v = reinterpret_cast<const uint32_t*>(q_sm + h * D)[lane + 32 * j];
      am = fmaxf(am, fmaxf(fabsf(io_to_f(v & 0xffffu, p.f16)), fabsf(io_to_f(v >> 16, p.f16))));
    }
    const float qmax = __uint_as_float(redux_max_u32(__float_as_uint(am)));
    if (lane == h) eq_lane = qmax > 0.f ? max(-100, min(100, -exponent_of(qmax))) : 0;
  }
  // B fragments of the zero-point products, for zero-points as they are stored (position pos holds channel
  // (pos % (D / 32)) * 32 + pos / (D / 32)): rows = token groups; even columns take the first half of the positions,
  // odd columns the second (whose zero-points sit in rows 4 and up).
  for (int i = warp; i < NT * KS / 2; i += W) {
    const int kp = i % (KS / 2), h = HP * (i / (KS / 2)) + col_head;
    const float e2 = pow2i(__shfl_sync(0xffffffffu, eq_lane, h) + Q_BIAS_EXP);
    float v[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int pos = low * (D / 2) + (kp >> 1) * 32 + tig * 8 + (kp & 1) * 4 + c;
      const int d = (pos % (D / 32)) * 32 + pos / (D / 32);
      v[c] = io_to_f(q_sm[h * D + d], p.f16) * e2;
    }
    const __half2 h0 = __floats2half2_rn(v[0], v[1]), h1 = __floats2half2_rn(v[2], v[3]);
    sts64(qb + (i * 32 + lane) * 8, *reinterpret_cast<const uint32_t*>(&h0), *reinterpret_cast<const uint32_t*>(&h1));
  }
  __syncthreads();
  float cq[NT];
#pragma unroll
  for (int n = 0; n < NT; ++n)
    cq[n] = p.scale * 1.4426950408889634f * pow2i(-__shfl_sync(0xffffffffu, eq_lane, HP * n + my_head));

  const uint32_t low_mask = low ? 0xffffffffu : 0u;
  // q of this lane's operand column as fp16 pairs, times 2^Ek and divided by the weights of the codes
  uint32_t qk[NT][KS][2];
  int Ek = -100;  // not set
  float ck[NT];
  auto set_ek = [&](int e) {
    Ek = e;
#pragma unroll
    for (int n = 0; n < NT; ++n) {
      const int h = HP * n + col_head;
      const int eh = e + __shfl_sync(0xffffffffu, eq_lane, h);
      const uint16_t* qh = q_sm + h * D;
#pragma unroll
      for (int ks = 0; ks < KS; ++ks) {
        const float e2 = pow2i(eh - k_weight<BK>(ks));
        const uint2 v = *reinterpret_cast<const uint2*>(qh + k_channel<BK>(ks, tig, 0));
        const __half2 h0 = __floats2half2_rn(io_to_f(v.x & 0xffffu, p.f16) * e2, io_to_f(v.y & 0xffffu, p.f16) * e2);
        const __half2 h1 = __floats2half2_rn(io_to_f(v.x >> 16, p.f16) * e2, io_to_f(v.y >> 16, p.f16) * e2);
        qk[n][ks][0] = *reinterpret_cast<const uint32_t*>(&h0);
        qk[n][ks][1] = *reinterpret_cast<const uint32_t*>(&h1);
      }
      ck[n] = cq[n] * pow2i(CODE_EXP - e);
    }
  };

  // softmax state: reference m (log2 units, an integer; -infinity before the first batch, where mr is 0 instead).
  // Row gid of zacc: the zero-point products of channel group gid (gid < NG), the sum of the numerators (gid >= NG;
  // with centered codes lsum, of this thread's tokens).
  float m[NT], mr[NT], acc[NT][KS][4], zacc[NT][4], lsum[NT];
  int Ev = -100;  // value scales are taken times 2^Ev
#pragma unroll
  for (int n = 0; n < NT; ++n) {
    m[n] = -CUDART_INF_F;
    mr[n] = 0.f;
    lsum[n] = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      zacc[n][i] = 0.f;
#pragma unroll
      for (int mt = 0; mt < KS; ++mt) acc[n][mt][i] = 0.f;
    }
  }
  // weights of this lane's tokens in the value words (row gid of row tile mt is pair q = gid + 8 mt of 32 tokens)
  const int wt_a = BV == 1 ? gid >> 1 : 2 * ((gid >> 1) & 3), wt_b = BV == 1 ? wt_a + 4 : wt_a;
  const float off[2] = {(float)(P_EXP - wt_a), (float)(P_EXP - wt_b)};
  const float weight_a = pow2i(wt_a), weight_b = pow2i(wt_b);
  const int tok0 = 4 * (gid >> 1) + (gid & 1);                       // token of row gid, tile 0; the other rows: + 2, + 16
  const uint32_t kc_lane = st + tok0 * (BK == 1 ? 8 : 16) + (BK == 1 ? (tig >> 1) : tig) * 4;
  const uint32_t vs_lane = st + Pl::OFF_VM + pair_row(BV == 1 ? 16 * tig : 8 * tig) * Pl::VSROW;  // first pair of the lane's word
  const uint32_t vz_lane = vs_lane + Pl::VS + 4 * (gid % NG);  // zero-points of channel group gid
  const uint32_t p_st = pbuf + my_head * Pl::PH + my_slot * 144 + gid * 8;  // + pair offset
  const uint32_t p_ld = pbuf + col_head * Pl::PH + tig * (BV == 1 ? 144 : 64) + (BV == 2 ? (tig >> 1) * 16 : 0);

  int last_k = 0, last_v = 0;  // number of the copy that each barrier was armed for last
#pragma unroll 1
  for (int i = warp, it = 0; i < nb; i += W, ++it) {
    const int valid = min(BT, p.n_q - (b0 + i) * BT);  // < BT only in the stream's last batch
    if (!__all_sync(0xffffffffu, mbar_wait(bar_k, it & 1, &dead_sm))) break;

    // ---- keys: scales into the order of the operand slots (in place), the largest of them ----
    {
      constexpr int V = D / 32;
      uint32_t s[NGT][V / 2], mx = 0u;
#pragma unroll
      for (int g = 0; g < NGT; ++g) {
        const uint32_t a = st + Pl::OFF_KM + g * 4 * D + lane * 2 * V;
        s[g][0] = lds32(a);
      }
      if (valid < BT) {
#pragma unroll
        for (int g = 0; g < NGT; ++g)
#pragma unroll
          for (int j = 0; j < V / 2; ++j) s[g][j] = g * GS < valid ? s[g][j] : 0u;
      }
#pragma unroll
      for (int g = 0; g < NGT; ++g)
#pragma unroll
        for (int j = 0; j < V / 2; ++j) mx = __vmaxu2(mx, s[g][j]);
#pragma unroll
      for (int g = 0; g < NGT; ++g) {
        const uint32_t a = st + Pl::OFF_KM + g * 4 * D + 2 * D + lane * 4;
        uint32_t hi, lo;
        centered_zero<BK>(s[g][0], lds32(a), hi, lo);
        sts32(a, hi);
        sts32(st + Pl::OFF_KL + g * 2 * D + lane * 4, lo);
      }
      // |q s| below 2^15 and its largest at least 2^8 (where 2^14 |q| allows): exponents of q move only outside that
      const float smax = f16_to_f(redux_max_u32(max(mx & 0xffffu, mx >> 16)));
      const int es = smax > 0.f ? exponent_of(smax) : -24;
      if (es > 13 - Ek || (es < 7 - Ek && Ek < 14) || Ek == -100) set_ek(min(14, 13 - es));
      __syncwarp();
#pragma unroll
      for (int j = 0; j < V; ++j) {
        const uint32_t dst = st + Pl::OFF_KM + 2 * k_slot<BK>(lane + 32 * j);
#pragma unroll
        for (int g = 0; g < NGT; ++g) sts16(dst + g * 4 * D, j & 1 ? s[g][j / 2] >> 16 : s[g][j / 2]);
      }
      __syncwarp();
    }
    // Units of 32 tokens: this thread's logits are those of units GC * ux + my_slot, ux = 0 .. HP - 1, of its head:
    // [row gid, gid + 8 of the unit's first tile, of its second]; less the reference and with the exponents `off`.
    float x[NT][HP][4];
    // ---- zero-points: sum_d q_d z_d per token group and head (rows: groups, first and second half of the channels) ----
    {
      const uint32_t za = st + Pl::OFF_KM + (gid & (NGT - 1)) * 4 * D + 2 * D + (gid >> 2) * D + tig * 16;
      const uint32_t zl = st + Pl::OFF_KL + (gid & (NGT - 1)) * 2 * D + (gid >> 2) * D + tig * 16;
      float zc[NT][4];
#pragma unroll
      for (int n = 0; n < NT; ++n)
#pragma unroll
        for (int k = 0; k < 4; ++k) zc[n][k] = 0.f;
#pragma unroll
      for (int kp = 0; kp < KS / 4; ++kp) {
        const uint4 a = lds128(za + kp * 64);
#pragma unroll
        for (int n = 0; n < NT; ++n) {
          const uint2 q0 = lds64(qb + ((n * KS / 2 + 2 * kp) * 32 + lane) * 8), q1 = lds64(qb + ((n * KS / 2 + 2 * kp + 1) * 32 + lane) * 8);
          const uint4 l = lds128(zl + kp * 64);
          mma_f16(zc[n], l.x, l.x, l.y, l.y, q0.x, q0.y);
          mma_f16(zc[n], l.z, l.z, l.w, l.w, q1.x, q1.y);
          mma_f16(zc[n], a.x, a.x, a.y, a.y, q0.x, q0.y);  // (rows 8 and up: the same again)
          mma_f16(zc[n], a.z, a.z, a.w, a.w, q1.x, q1.y);
        }
      }
#pragma unroll
      for (int n = 0; n < NT; ++n) {
        const float zb = (zc[n][0] + __shfl_xor_sync(0xffffffffu, zc[n][1], 16)) * (cq[n] * (1.f / (float)(1 << Q_BIAS_EXP)));
#pragma unroll
        for (int ux = 0; ux < HP; ++ux)
          x[n][ux][0] = __shfl_sync(0xffffffffu, zb, ((GC * ux + my_slot) * 32 / GS) * 4 + tig) - mr[n];
      }
    }
    // ---- keys: q . c ----
    // packed words of rows gid, gid + 8: even bytes, odd bytes
    auto load_rows = [&](int u, uint32_t (&w)[2][2], uint32_t (&w8)[2][2]) {
#pragma unroll
      for (int t = 0; t < 2; ++t)
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          const int tk = 16 * t + 2 * r;
          uint32_t raw;
          if constexpr (BK == 1) raw = lds32(kc_lane + u * 256 + tk * 8) >> (4 * (tig & 1));
          else raw = lds32(kc_lane + u * (32 * D * BK / 8) + tk * 16);
          w[t][r] = byte_pair_up(raw, 2);
          w8[t][r] = byte_pair_down(raw, 6);
        }
    };
    auto key_pair = [](uint32_t w, int k) { return code_pair<BK>(w, BK == 2 ? k & 3 : k); };
    if constexpr (GC == 1) {
      constexpr int UG = GS / 32;  // units of a group
      // fma(q, s, qn * s) is hi where qn = 0 and lo where qn = -q
      uint32_t qn[KS][2];
      if constexpr (NT == 1) {
#pragma unroll
        for (int ks = 0; ks < KS; ++ks) {
          qn[ks][0] = (qk[0][ks][0] ^ 0x80008000u) & low_mask;
          qn[ks][1] = (qk[0][ks][1] ^ 0x80008000u) & low_mask;
        }
      }
#pragma unroll
      for (int g = 0; g < NGT; ++g) {
        float c[NT][2 * UG][4];
        uint32_t w[UG][2][2], w8[UG][2][2];
#pragma unroll
        for (int u = 0; u < UG; ++u) load_rows(g * UG + u, w[u], w8[u]);
        const uint32_t sa = st + Pl::OFF_KM + g * 4 * D + tig * 16;
        uint4 sv;
#pragma unroll
        for (int k = 0; k < KS; ++k) {
          if ((k & 1) == 0) sv = lds128(sa + (k / 2) * 64);
          const uint32_t s0 = k & 1 ? sv.z : sv.x, s1 = k & 1 ? sv.w : sv.y;
#pragma unroll
          for (int n = 0; n < NT; ++n) {
            uint32_t p0, p1;
            if constexpr (NT == 1) {
              p0 = hfma2(qk[n][k][0], s0, hmul2(qn[k][0], s0));
              p1 = hfma2(qk[n][k][1], s1, hmul2(qn[k][1], s1));
            } else {
              p0 = product_part(qk[n][k][0], s0, low);
              p1 = product_part(qk[n][k][1], s1, low);
            }
#pragma unroll
            for (int u = 0; u < UG; ++u)
#pragma unroll
              for (int t = 0; t < 2; ++t) {
                const uint32_t a0 = key_pair(w[u][t][0], k), a1 = key_pair(w[u][t][1], k);
                const uint32_t a2 = key_pair(w8[u][t][0], k), a3 = key_pair(w8[u][t][1], k);
                if (k == 0) mma_f16_first(c[n][2 * u + t], a0, a1, a2, a3, p0, p1);
                else mma_f16(c[n][2 * u + t], a0, a1, a2, a3, p0, p1);
              }
          }
        }
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
          for (int u = 0; u < UG; ++u) {
            float* xu = x[n][g * UG + u];
            const float bias[2] = {xu[0] + off[0], xu[0] + off[1]};
#pragma unroll
            for (int k = 0; k < 4; ++k)
              xu[k] = fmaf(c[n][2 * u + k / 2][2 * (k & 1)] + c[n][2 * u + k / 2][2 * (k & 1) + 1], ck[n], bias[k >> 1]);
          }
      }
    } else {
      // one operand for GC units, each in its own column slot; a unit's logits are in the threads of its slot
#pragma unroll
      for (int ux = 0; ux < HP; ++ux) {
        uint32_t pp[KS][2];
        const uint32_t sa = st + Pl::OFF_KM + ((GC * ux + col_slot) * 32 / GS) * 4 * D + tig * 16;
#pragma unroll
        for (int kp = 0; kp < KS / 2; ++kp) {
          const uint4 sv = lds128(sa + kp * 64);
          pp[2 * kp][0] = product_part(qk[0][2 * kp][0], sv.x, low);
          pp[2 * kp][1] = product_part(qk[0][2 * kp][1], sv.y, low);
          pp[2 * kp + 1][0] = product_part(qk[0][2 * kp + 1][0], sv.z, low);
          pp[2 * kp + 1][1] = product_part(qk[0][2 * kp + 1][1], sv.w, low);
        }
        const float bias[2] = {x[0][ux][0] + off[0], x[0][ux][0] + off[1]};
#pragma unroll
        for (int j = 0; j < GC; ++j) {
          float c[2][4];
          uint32_t w[2][2], w8[2][2];
          load_rows(GC * ux + j, w, w8);
#pragma unroll
          for (int k = 0; k < KS; ++k)
#pragma unroll
            for (int t = 0; t < 2; ++t) {
              const uint32_t a0 = key_pair(w[t][0], k), a1 = key_pair(w[t][1], k);
              const uint32_t a2 = key_pair(w8[t][0], k), a3 = key_pair(w8[t][1], k);
              if (k == 0) mma_f16_first(c[t], a0, a1, a2, a3, pp[0][0], pp[0][1]);
              else mma_f16(c[t], a0, a1, a2, a3, pp[k][0], pp[k][1]);
            }
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const float v = fmaf(c[k / 2][2 * (k & 1)] + c[k / 2][2 * (k & 1) + 1], ck[0], bias[k >> 1]);
            x[0][ux][k] = j == 0 || my_slot == j ? v : x[0][ux][k];
          }
        }
      }
    }
    // the key half of the stage is free: fetch the keys of this warp's next batch
    proxy_fence();
    __syncwarp();
    if (i + W < nb) {
      if (lane == 0) load_keys(i + W);
      last_k = it + 1;
    }

    if (valid < BT) {
#pragma unroll
      for (int ux = 0; ux < HP; ++ux)
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (32 * (GC * ux + my_slot) + tok0 + 16 * (k >> 1) + 2 * (k & 1) >= valid) {
#pragma unroll
            for (int n = 0; n < NT; ++n) x[n][ux][k] = -CUDART_INF_F;
          }
    }
    // ---- softmax: raise the reference when a logit exceeds it by more than TAU (rare) ----
    float xm[NT];
    bool need = false;
#pragma unroll
    for (int n = 0; n < NT; ++n) {
      float v[2];
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        v[t] = fmaxf(x[n][0][2 * t], x[n][0][2 * t + 1]);
#pragma unroll
        for (int ux = 1; ux < HP; ++ux) v[t] = fmaxf(fmaxf(v[t], x[n][ux][2 * t]), x[n][ux][2 * t + 1]);
      }
      xm[n] = fmaxf(v[0] - off[0], v[1] - off[1]);  // above the reference
      need |= xm[n] > (m[n] == mr[n] ? TAU : -CUDART_INF_F);
    }
    if (__any_sync(0xffffffffu, need)) {
#pragma unroll
      for (int n = 0; n < NT; ++n) {
        float v = xm[n];
#pragma unroll
        for (int k = HP; k < 32; k <<= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, k));
        const float up = m[n] != mr[n] || v > TAU - 1.f ? ceilf(v) : 0.f;
        const float f = m[n] != mr[n] ? 0.f : ex2(-up);  // (nothing has been accumulated yet)
        m[n] = mr[n] = mr[n] + up;
#pragma unroll
        for (int ux = 0; ux < HP; ++ux)
#pragma unroll
          for (int k = 0; k < 4; ++k) x[n][ux][k] -= up;
        lsum[n] *= f;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          zacc[n][k] *= f;
#pragma unroll
          for (int mt = 0; mt < KS; ++mt) acc[n][mt][k] *= f;
        }
      }
    }
    // numerators times 2^P_EXP and divided by the weight of the token's value code, as hi + lo pairs (t, t + 2)
#pragma unroll
    for (int n = 0; n < NT; ++n) {
#pragma unroll
      for (int ux = 0; ux < HP; ++ux)
#pragma unroll
        for (int t = 0; t < 2; ++t) {
          const float pa = ex2(x[n][ux][2 * t]), pb = ex2(x[n][ux][2 * t + 1]);
          lsum[n] = fmaf(pa + pb, t ? weight_b : weight_a, lsum[n]);
          const uint32_t h = pack_io2<true>(pa, pb);
          const uint32_t lo = pack_io2<true>(pa - io2_lo<true>(h), pb - io2_hi<true>(h));
          sts64(p_st + n * HP * Pl::PH + ux * GC * 144 + t * 64, h, lo);
        }
    }

    // ---- values: scales and zero-points as pairs of tokens (t, t + 2), in place ----
    if (!__all_sync(0xffffffffu, mbar_wait(bar_v, it & 1, &dead_sm))) break;
    {
      uint32_t sp[2][NG], zp[2][NG], mx = 0u;
      const uint32_t vm = st + Pl::OFF_VM;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int pr = lane + 32 * h, ta = 4 * (pr >> 1) + (pr & 1);
        uint32_t ra[NG], rb[NG];  // raw rows of the two tokens: NG scales, NG zero-points
        if constexpr (NG == 4) {
          const uint4 a = lds128(vm + ta * 16), c = lds128(vm + ta * 16 + 32);
          ra[0] = a.x; ra[1] = a.y; ra[2] = a.z; ra[3] = a.w;
          rb[0] = c.x; rb[1] = c.y; rb[2] = c.z; rb[3] = c.w;
        } else if constexpr (NG == 2) {
          const uint2 a = lds64(vm + ta * 8), c = lds64(vm + ta * 8 + 16);
          ra[0] = a.x; ra[1] = a.y; rb[0] = c.x; rb[1] = c.y;
        } else {
          ra[0] = lds32(vm + ta * 4); rb[0] = lds32(vm + ta * 4 + 8);
        }
        if (valid < BT) {
#pragma unroll
          for (int g = 0; g < NG; ++g) {
            if (ta >= valid) ra[g] = 0u;
            if (ta + 2 >= valid) rb[g] = 0u;
          }
        }
        if constexpr (NG == 1) {
          sp[h][0] = __byte_perm(ra[0], rb[0], 0x5410);
          zp[h][0] = __byte_perm(ra[0], rb[0], 0x7632);
        } else {
#pragma unroll
          for (int g = 0; g < NG; ++g) {
            const uint32_t sel = g & 1 ? 0x7632 : 0x5410;
            sp[h][g] = __byte_perm(ra[g / 2], rb[g / 2], sel);
            zp[h][g] = __byte_perm(ra[NG / 2 + g / 2], rb[NG / 2 + g / 2], sel);
          }
        }
#pragma unroll
        for (int g = 0; g < NG; ++g) mx = __vmaxu2(mx, sp[h][g]);
      }
      // the largest scale times 2^Ev in [2^-6, 1): the exponent moves only outside that
      const float smax = f16_to_f(redux_max_u32(max(mx & 0xffffu, mx >> 16)));
      const int es = smax > 0.f ? exponent_of(smax) : -24;
      if (es >= -Ev || (es < -6 - Ev && Ev < 15) || Ev == -100) {
        const int e = min(15, -1 - es);
        const float f = Ev == -100 ? 0.f : pow2i(e - Ev);
        Ev = e;
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
          for (int mt = 0; mt < KS; ++mt)
#pragma unroll
            for (int k = 0; k < 4; ++k) acc[n][mt][k] *= f;
      }
      const float ev = pow2i(Ev);
      const __half2 ev2 = __floats2half2_rn(ev, ev);
      const uint32_t e2 = *reinterpret_cast<const uint32_t*>(&ev2);
      __syncwarp();
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const uint32_t dst = vm + pair_row(32 * h) * Pl::VSROW + pair_row(lane) * Pl::VSROW;
#pragma unroll
        for (int g = 0; g < NG; ++g) {
          uint32_t lo;
          centered_zero<BV>(sp[h][g], zp[h][g], zp[h][g], lo);
          sts32(dst + 2 * Pl::VS + 4 * g, lo);
        }
        if constexpr (NG == 4) {
          sts128(dst, hmul2(sp[h][0], e2), hmul2(sp[h][1], e2), hmul2(sp[h][2], e2), hmul2(sp[h][3], e2));
          sts128(dst + Pl::VS, zp[h][0], zp[h][1], zp[h][2], zp[h][3]);
        } else if constexpr (NG == 2) {
          sts64(dst, hmul2(sp[h][0], e2), hmul2(sp[h][1], e2));
          sts64(dst + Pl::VS, zp[h][0], zp[h][1]);
        } else {
          sts32(dst, hmul2(sp[h][0], e2));
          sts32(dst + Pl::VS, zp[h][0]);
        }
      }
      __syncwarp();
    }
    // ---- values: one chunk of packed words at a time (lane column tig owns word tig of every channel row) ----
#pragma unroll
    for (int c = 0; c < VCH; ++c) {
      uint32_t w[KS][2], w8[KS][2];  // even and odd bytes of rows (channels) 16 mt + gid, + 8
      const uint32_t va = st + Pl::OFF_VC + c * D * 16 + gid * 16 + tig * 4;
#pragma unroll
      for (int mt = 0; mt < KS; ++mt) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          const uint32_t raw = lds32(va + mt * 256 + r * 128);
          w[mt][r] = byte_pair_up(raw, 2);
          w8[mt][r] = byte_pair_down(raw, 6);
        }
      }
#pragma unroll
      for (int e = 0; e < VE; ++e) {
        constexpr int VB = CP / GC;  // operands of a step: parts GC * vb + slot
        uint32_t sp[2][VB];
        const uint32_t sa = vs_lane + pair_row(32 * c) * Pl::VSROW + 2 * e * Pl::VSROW, sb = sa + Pl::VSROW;
        if constexpr (GC == 1 && NG == 4) {
          const uint4 a = lds128(sa), d = lds128(sb);
          sp[0][0] = a.x; sp[0][1] = a.y; sp[0][2] = a.z; sp[0][3] = a.w;
          sp[1][0] = d.x; sp[1][1] = d.y; sp[1][2] = d.z; sp[1][3] = d.w;
        } else {
#pragma unroll
          for (int vb = 0; vb < VB; ++vb) {
            const uint32_t o = ((GC * vb + col_slot) * NG / CP) * 4;
            sp[0][vb] = lds32(sa + o);
            sp[1][vb] = lds32(sb + o);
          }
        }
        const uint32_t zo = vz_lane + pair_row(32 * c) * Pl::VSROW + 2 * e * Pl::VSROW;
        const uint32_t z0 = lds32(zo), z1 = lds32(zo + Pl::VSROW);
        constexpr uint32_t ONE = 0x3C00u, STEP = BV == 2 ? 0x0800u : 0x0400u;
        const uint32_t we = (ONE + e * STEP) * 0x10001u;  // the weight of this step's codes as a pair of fp16
#pragma unroll
        for (int n = 0; n < NT; ++n) {
          const uint4 hp = lds128(p_ld + n * HP * Pl::PH + c * 288 + e * 16);  // (hi, lo) of pairs 2 e and 2 e + 1
          const uint32_t pz0 = hmul2(low ? hp.y : hp.x, we), pz1 = hmul2(low ? hp.w : hp.z, we);
          const uint32_t y0 = lds32(zo + Pl::VS), y1 = lds32(zo + Pl::VS + Pl::VSROW);
          mma_f16(zacc[n], y0, y0, y1, y1, pz0, pz1);
          mma_f16(zacc[n], z0, z0, z1, z1, pz0, pz1);
          // fma(l, s, fma(h, s, hn * s)): hi where hn = l = 0, lo where hn = -h
          const uint32_t hn0 = (hp.x ^ 0x80008000u) & low_mask, hn1 = (hp.z ^ 0x80008000u) & low_mask;
          const uint32_t l0 = hp.y & low_mask, l1 = hp.w & low_mask;
#pragma unroll
          for (int vb = 0; vb < VB; ++vb) {
            const uint32_t p0 = hfma2(l0, sp[0][vb], hfma2(hp.x, sp[0][vb], hmul2(hn0, sp[0][vb])));
            const uint32_t p1 = hfma2(l1, sp[1][vb], hfma2(hp.z, sp[1][vb], hmul2(hn1, sp[1][vb])));
            constexpr int MT = GC * KS / CP;
#pragma unroll
            for (int mt = vb * MT; mt < (vb + 1) * MT; ++mt)
              mma_f16(acc[n][mt], code_pair<BV>(w[mt][0], e), code_pair<BV>(w[mt][1], e),
                      code_pair<BV>(w8[mt][0], e), code_pair<BV>(w8[mt][1], e), p0, p1);
          }
        }
      }
    }
    // the value half of the stage and the numerators are free
    proxy_fence();
    __syncwarp();
    if (i + W < nb) {
      if (lane == 0) load_values(i + W);
      last_v = it + 1;
    }
  }

  // ---- this warp's result so far in true units: channels 16 mt + gid, + 8 of head HP n + my_head ----
  float o[NT][KS][2], l[NT];
#pragma unroll
  for (int n = 0; n < NT; ++n) {
    const float ua = pow2i(CODE_EXP - P_EXP - Ev), uz = pow2i(-P_EXP);
    const float z = (zacc[n][0] + zacc[n][1]) * uz;  // row gid < NG: channel group gid; row NG: the sum
#pragma unroll
    for (int k = HP; k < 32; k <<= 1) lsum[n] += __shfl_xor_sync(0xffffffffu, lsum[n], k);
    l[n] = lsum[n] * uz;
#pragma unroll
    for (int mt = 0; mt < KS; ++mt) {
      const float zg = __shfl_sync(0xffffffffu, z, (mt * 16 / GS) * 4 + tig);
      float s0 = acc[n][mt][0] + acc[n][mt][1], s1 = acc[n][mt][2] + acc[n][mt][3];
      if constexpr (GC > 1) {  // the threads of the tile's slot hold it
        const int src = (lane & ~3) + (mt / (KS / CP)) % GC * HP + my_head;
        s0 = __shfl_sync(0xffffffffu, s0, src);
        s1 = __shfl_sync(0xffffffffu, s1, src);
      }
      o[n][mt][0] = fmaf(s0, ua, zg);
      o[n][mt][1] = fmaf(s1, ua, zg);
    }
  }
  // ---- the CTA's share of the 16-bit window, tile by tile, first to the warps with the fewest batches ----
  if (dead_sm == 0) {  // (else a wait gave up somewhere: copies may be in flight, the stage is not reused)
    int t = warp - nb % W;
    if (t < 0) t += W;
    for (int tb = wt0 + 16 * t; tb < wt1; tb += 16 * W) {
      window_stage<WROW>(p, L, tb, wt1, bh, st, lane);
      cp_async_commit();
      cp_async_wait_all();
      __syncwarp();
      if (L.K_new != nullptr && tb + 16 > p.r - 1 && wt1 == p.r) window_store_new<WROW>(p, L, tb, bh, st, lane);
      const float scale2 = p.scale * 1.4426950408889634f;
#pragma unroll
      for (int n = 0; n < NT; ++n) {
        const int h = HP * n + col_head;
        const bool real = low == 0 && col_slot == 0 && h < G;
        const uint16_t* qrow = q_sm + h * D;
        if (p.f16) window_tile<WROW, true>(st, wt1 - tb, qrow, real, scale2, o[n], m[n], l[n], lane);
        else window_tile<WROW, false>(st, wt1 - tb, qrow, real, scale2, o[n], m[n], l[n], lane);
      }
      __syncwarp();
    }
    __syncwarp();
    float* ws = reinterpret_cast<float*>(smem + warp * Pl::WARP);  // state rows, over the stage
#pragma unroll
    for (int n = 0; n < NT; ++n) {
      const int h = HP * n + my_head;
      if (h < G && my_slot == 0) {
#pragma unroll
        for (int mt = 0; mt < KS; ++mt) {
          ws[h * Pl::MS + 16 * mt + gid] = o[n][mt][0];
          ws[h * Pl::MS + 16 * mt + gid + 8] = o[n][mt][1];
        }
        if (gid == 0) {
          ws[h * Pl::MS + D] = m[n];
          ws[h * Pl::MS + D + 1] = l[n];
        }
      }
    }
  }
  __syncthreads();
  if (p.late_wait) grid_dependency_wait();  // the preceding launch still reads and writes the scratch and its result
  if (dead_sm != 0) {
    // leaving early: no copy of this CTA may still be in flight when its shared memory is released
    if (lane == 0 && warp < nb) {
      for (int it = 0; it < WAIT_LIMIT && !mbar_try_wait(bar_k, last_k & 1); ++it) {}
      for (int it = 0; it < WAIT_LIMIT && !mbar_try_wait(bar_v, last_v & 1); ++it) {}
    }
    if (tid == 0) atomicExch(p.status, 1);
    __syncthreads();
    return;
  }
  // ---- the CTA's state: all warps; then the partial and the merge, or the result itself ----
  const size_t slot = (size_t)blockIdx.y * ((size_t)dm.B * dm.Hq) * p.ns_q;  // this layer's partials in the scratch
  float* const part_acc = p.part_acc + slot * D;
  float* const part_ml = p.part_ml + slot * 2;
  for (int item = tid; item < G * (D / 4); item += W * 32) {
    const int h = item / (D / 4), d = item % (D / 4) * 4;
    auto row = [&](int w) { return reinterpret_cast<const float*>(smem + w * Pl::WARP) + h * Pl::MS; };
    float M = -CUDART_INF_F;
#pragma unroll
    for (int w = 0; w < W; ++w) M = fmaxf(M, row(w)[D]);
    float4 A = make_float4(0.f, 0.f, 0.f, 0.f);
    float Ls = 0.f;
#pragma unroll
    for (int w = 0; w < W; ++w) {
      const float4 v = *reinterpret_cast<const float4*>(row(w) + d);
      const float mw = row(w)[D];
      const float f = mw == -CUDART_INF_F ? 0.f : ex2(mw - M);  // a warp without tokens
      A.x = fmaf(v.x, f, A.x);
      A.y = fmaf(v.y, f, A.y);
      A.z = fmaf(v.z, f, A.z);
      A.w = fmaf(v.w, f, A.w);
      Ls = fmaf(row(w)[D + 1], f, Ls);
    }
    const size_t hq = (size_t)b * dm.Hq + hk * G + h;
    if (ns == 1) {
      store_out(p, L, hq, d, make_float4(A.x / Ls, A.y / Ls, A.z / Ls, A.w / Ls));
    } else {
      *reinterpret_cast<float4*>(part_acc + (hq * p.ns_q + split) * D + d) = A;
      if (d == 0) *reinterpret_cast<float2*>(part_ml + (hq * p.ns_q + split) * 2) = make_float2(M, Ls);
    }
  }
  if (ns > 1)
    ticket_merge(p, L, ns, hk, b, part_acc, part_ml, p.tickets + (size_t)blockIdx.y * (dm.B * dm.Hkv) + bh, &s_flag,
                    reinterpret_cast<float*>(smem));
}

template <int BK, int BV, int GS, int HP, int NT>
cudaError_t launch_one(const DecodeParams& p, cudaStream_t st) {
  using Pl = Plan<BK, BV, GS, HP, NT>;
  return launch_dependent(decode_mma64_kernel<BK, BV, GS, HP, NT>, dim3((unsigned)(p.ns_q * p.dm.B * p.dm.Hkv), p.n_layers), dim3(Pl::WARPS * 32),
                          (size_t)Pl::TOTAL, st, p);
}

// Prepares the kernel for the current device.
template <int BK, int BV, int GS, int HP, int NT>
MmaShape shape_one() {
  using Pl = Plan<BK, BV, GS, HP, NT>;
  auto kernel = decode_mma64_kernel<BK, BV, GS, HP, NT>;
  // the largest shared-memory carve-out: two CTAs of this size are to share an SM
  const bool ready = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, Pl::TOTAL) == cudaSuccess &&
                     cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, 100) == cudaSuccess;
  if (!ready) cudaGetLastError();
  return {Pl::WARPS, ready};
}

#define XQ_DISPATCH(FN, ...)                               \
  switch (bk * 100 + bv * 10 + (g == 64)) {                \
    case 220: return FN<2, 2, 32, HP, NT>(__VA_ARGS__); \
    case 221: return FN<2, 2, 64, HP, NT>(__VA_ARGS__); \
    case 210: return FN<2, 1, 32, HP, NT>(__VA_ARGS__); \
    case 211: return FN<2, 1, 64, HP, NT>(__VA_ARGS__); \
    case 120: return FN<1, 2, 32, HP, NT>(__VA_ARGS__); \
    case 121: return FN<1, 2, 64, HP, NT>(__VA_ARGS__); \
    case 110: return FN<1, 1, 32, HP, NT>(__VA_ARGS__); \
    case 111: return FN<1, 1, 64, HP, NT>(__VA_ARGS__); \
  }

}  // namespace

template <int HP, int NT>
cudaError_t launch_decode_mma64_t(const DecodeParams& p, cudaStream_t st) {
  const int bk = p.layer[0].L.bk, bv = p.layer[0].L.bv, g = p.dm.g;
  XQ_DISPATCH(launch_one, p, st)
  return cudaErrorInvalidValue;
}
template <int HP, int NT>
MmaShape decode_mma64_shape_t(int g, int bk, int bv) {
  XQ_DISPATCH(shape_one)
  return MmaShape{1, false};
}

}  // namespace xq
