// Attention of a chunk of query tokens over the packed cache plus the window, causal inside the chunk: the query rows
// (tokens x heads of a kv head) share one pass over the cache.
//
// A CTA takes M = 16 WR rows and a range of 64-token tiles of one (sequence, kv head).  With M rows per code it pays
// to dequantize: four warps expand the keys of a tile and four its values, once for all rows, into fp16 pairs
// hi + lo in shared memory (22 significant bits of c s + z, relative to the group's largest member), and the products
// are q hi + q lo for the logits and p_hi v_hi + p_hi v_lo + p_lo v_hi for the result, p_hi + p_lo the softmax
// numerators as fp16 pairs, accumulation in fp32.  The tile after the current one is expanded while the current one
// is multiplied: of the two warps that share a sub-partition one expands before its products, the other after them.
// The eight warps are WR row groups of 16 rows times WT = 8 / WR parts of a tile's tokens.  Window tiles are 16-bit
// already and are multiplied as they are (bf16 or fp16 products, numerators as pairs of that type).
// Split partials are merged by the last CTA of a row tile, as in the decode kernel.
//
// What bounds it: the rate of mma.sync (8 cycles per m16n8k16 and sub-partition here), five products for every
// (row, token, channel) instead of the two that plain fp16 attention takes.  One decode launch per query token before:
// 16 tokens at 32k context, batch 4 and 8 kv heads 508 -> 451 us per layer, 250 tokens at 8k 1308 -> 501 us, a whole
// prompt of 1024 tokens, 32 heads 2470 -> 134 us.
#pragma once
#include <type_traits>

#include "xq_internal.h"
#include "xq_mma.cuh"

namespace xq {
namespace {

constexpr int CT = 64;             // tokens of a tile
constexpr int C_STAGES = 3;        // raw tiles in flight
constexpr float C_TAU = 3.f;       // log2 units a logit may exceed the softmax reference before it is raised
constexpr int C_PEXP = 11;         // numerators are carried times 2^C_PEXP

template <int D, int BK, int BV, int GS, int WR>
struct ChunkPlan {
  static constexpr int M = 16 * WR, WT = 8 / WR, TW = CT / WT;  // rows; token parts; tokens of a warp
  static constexpr int NG = D / GS;
  static constexpr int QROW = 2 * D + 16;                       // a staged row of q
  static constexpr int KROW = D * BK / 8;                       // packed bytes of a token's keys
  static constexpr int MAT = CT * 2 * D;                        // one matrix of a tile: K hi, K lo, V hi, V lo
  static constexpr int BUF = 4 * MAT;
  static constexpr int RAW_K = 16 * KROW + 4 * D;               // a key warp's codes and parameters
  static constexpr int RAW_VC = (D / 4) * 8 * BV, RAW_V = RAW_VC + CT * 4 * NG;
  static constexpr int RAW = RAW_K > RAW_V ? RAW_K : RAW_V;     // of one warp and stage
  static constexpr int OFF_RAW = 2 * BUF;
  static constexpr int OFF_Q = OFF_RAW + 8 * C_STAGES * RAW;
  static constexpr int TOTAL = OFF_Q + M * QROW;
  static constexpr int MS = D + 4;                              // state row: acc[D], m, l
  static_assert(8 * 16 * MS * 4 <= 2 * BUF, "the warps' states fit the tile buffers");
  static_assert(TOTAL <= 226 * 1024, "shared memory");
};

template <int D>
__device__ __forceinline__ void chunk_store(const ChunkParams& p, size_t row, int c, float v) {
  if (p.out_f32) reinterpret_cast<float*>(p.out)[row * D + c] = v;
  else if (p.f16) reinterpret_cast<__half*>(p.out)[row * D + c] = __float2half_rn(v);
  else reinterpret_cast<__nv_bfloat16*>(p.out)[row * D + c] = __float2bfloat16_rn(v);
}

// 16 codes of a packed word (`w` shifted so that the codes 4 e + j sit at bit BITS * e of byte j) with the parameters
// s, z of each, as fp16 pairs: element k's hi and lo in hi[k / 2], lo[k / 2].
template <int BITS>
__device__ __forceinline__ void expand16(uint32_t w, const float (&s)[16], const float (&z)[16], uint32_t (&hi)[8],
                                         uint32_t (&lo)[8]) {
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const uint32_t m = (w >> (BITS * e)) & (BITS == 2 ? 0x03030303u : 0x01010101u);
    float v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float c = __uint_as_float(__byte_perm(m, 0x4B000000u, 0x7440 + j)) - 8388608.f;  // 2^23 + code, less 2^23
      v[j] = fmaf(c, s[4 * e + j], z[4 * e + j]);
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const uint32_t h = pack_io2<true>(v[2 * j], v[2 * j + 1]);
      hi[2 * e + j] = h;
      lo[2 * e + j] = pack_io2<true>(v[2 * j] - io2_lo<true>(h), v[2 * j + 1] - io2_hi<true>(h));
    }
  }
}

// x[0 .. 15] *= f
__device__ __forceinline__ void scale16(float (&x)[16], float f) {
#pragma unroll
  for (int k = 0; k < 16; ++k) x[k] *= f;
}

template <int D, int BK, int BV, int GS, int WR>
__global__ void __launch_bounds__(256, 1) chunk_kernel(const __grid_constant__ ChunkParams p) {
  using Pl = ChunkPlan<D, BK, BV, GS, WR>;
  constexpr int M = Pl::M, WT = Pl::WT, TW = Pl::TW, NG = Pl::NG, KS = D / 16, NT = TW / 8, NO = D / 8;
  constexpr int QT = D / 32;  // output tiles of 8 channels in a quarter of the channels
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ float k_unit[2][4];  // [buffer][16 tokens]: what a unit of the expanded keys is worth
  __shared__ int v_exp[2][4];     // [buffer][channel quarter]: the expanded values are times 2^v_exp
  __shared__ int s_flag;

  const Dims& dm = p.dm;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gid = lane >> 2, tig = lane & 3;
  const int wr = warp % WR, wt = warp / WR;
  const int G = dm.G, n_streams = dm.B * dm.Hkv;
  // the row tiles with the most visible tokens first
  const int split = blockIdx.x % p.ns, bh = (blockIdx.x / p.ns) % n_streams, rt = p.row_tiles - 1 - blockIdx.x / p.ns / n_streams;
  const int hk = bh % dm.Hkv, b = bh / dm.Hkv;
  const int row0 = rt * M, n_rows = min(M, p.T * G - row0);  // row: query token row / G, head row % G
  const int vis0 = p.S - p.T + 1;                            // tokens that query token 0 sees
  const int vis_max = vis0 + (row0 + n_rows - 1) / G, vis_min = vis0 + row0 / G;
  const int n_packed = min(p.n_q, vis_max);
  const int pk_tiles = (n_packed + CT - 1) / CT, all_tiles = pk_tiles + (vis_max - n_packed + CT - 1) / CT;
  int t_lo, t_hi;
  share_of(all_tiles, p.ns, split, t_lo, t_hi);

  const uint32_t sm = (uint32_t)__cvta_generic_to_shared(smem);
  const uint32_t raw = sm + Pl::OFF_RAW + warp * C_STAGES * Pl::RAW, qs = sm + Pl::OFF_Q;
  const uint8_t* const g_kc = reinterpret_cast<const uint8_t*>(p.L.k_codes) + (size_t)bh * ((size_t)dm.nq_cap * Pl::KROW);
  const uint8_t* const g_km = reinterpret_cast<const uint8_t*>(p.L.k_meta) + (size_t)bh * ((size_t)(dm.nq_cap / GS) * 4 * D);
  const uint8_t* const g_vc = reinterpret_cast<const uint8_t*>(p.L.v_codes) + (size_t)bh * ((size_t)dm.nq_cap * (D * BV / 8));
  const uint8_t* const g_vm = reinterpret_cast<const uint8_t*>(p.L.v_meta) + (size_t)bh * ((size_t)dm.nq_cap * 4 * NG);

  // Raw data of tile `t` that this warp expands, into its own stage; one commit per call (empty beyond the last tile).
  // Warps 0..3: keys of 16 tokens each; warps 4..7: values of D / 4 channels each.
  auto fetch = [&](int t) {
    if (t < min(t_hi, pk_tiles)) {
      const uint32_t dst = raw + (t % C_STAGES) * Pl::RAW;
      if (warp < 4) {
        const int tok = t * CT + 16 * warp;
        const uint8_t* src = g_kc + (size_t)(tok / 32) * (32 * Pl::KROW);
        if (lane < Pl::KROW) {  // 16 tokens x KROW bytes in 16-byte pieces
          if constexpr (Pl::KROW == 32) cp_async16(dst + lane * 16, src + (lane >> 4) * 512 + (tok % 32 + (lane & 15)) * 16);
          else cp_async16(dst + lane * 16, src + (tok % 32) * Pl::KROW + lane * 16);
        }
        if (lane < D / 4) cp_async16(dst + 16 * Pl::KROW + lane * 16, g_km + (size_t)(tok / GS) * (4 * D) + lane * 16);
      } else {
        const int c0 = (warp - 4) * (D / 4);
        const uint8_t* src = g_vc + (size_t)(t / 2) * (D * 16 * BV);
        if (lane < D / 4) {
          if constexpr (BV == 2) cp_async16(dst + lane * 16, src + (t & 1) * (D * 16) + (c0 + lane) * 16);
          else cp_async8(dst + lane * 8, src + (c0 + lane) * 16 + (t & 1) * 8);
        }
        for (int i = lane; i < CT * 4 * NG / 16; i += 32)
          cp_async16(dst + Pl::RAW_VC + i * 16, g_vm + (size_t)t * (CT * 4 * NG) + i * 16);
      }
    }
    cp_async_commit();
  };

  int ev_mine = 0;        // value warps: exponent in use for this warp's channels
  bool ev_set = false;
  // Expands this warp's part of tile `t` into buffer `buf`.  nq % 32 == 0, so 16 tokens exist or do not together.
  auto expand = [&](int t, int buf) {
    const uint32_t src = raw + (t % C_STAGES) * Pl::RAW, dst = sm + buf * Pl::BUF;
    float s[16], z[16];
    if (warp < 4) {
      constexpr int NU = D / 16, NS = 32 / NU;  // lanes: NU units of 16 channels, NS tokens
      const int u = lane % NU, sub = lane / NU;
      const bool exists = t * CT + 16 * warp < p.n_q;
      float mx = 0.f;
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        const int d = 16 * u + k, pos = (d % 32) * (D / 32) + d / 32;
        s[k] = exists ? f16_to_f(lds16(src + 16 * Pl::KROW + 2 * pos)) : 0.f;
        z[k] = exists ? f16_to_f(lds16(src + 16 * Pl::KROW + 2 * D + 2 * pos)) : 0.f;
        mx = fmaxf(mx, fmaf((float)((1 << BK) - 1), s[k], fabsf(z[k])));
      }
      mx = __uint_as_float(redux_max_u32(__float_as_uint(mx)));
      const int e = mx > 0.f ? 14 - exponent_of(mx) : 0;  // the largest |k| of the tokens' group below 2^15
      const float f = pow2i(e);
      if (lane == 0) k_unit[buf][warp] = pow2i(-e);
      scale16(s, f);
      scale16(z, f);
#pragma unroll
      for (int k = 0; k < 16 / NS; ++k) {
        const int tl = sub + NS * k, tok = 16 * warp + tl;
        uint32_t w;
        if constexpr (BK == 2) w = lds32(src + (Pl::KROW == 32 ? (u >> 2) * 256 : 0) + tl * 16 + (u & 3) * 4);
        else w = lds32(src + tl * Pl::KROW + (u >> 1) * 4) >> (4 * (u & 1));
        uint32_t hi[8], lo[8];
        expand16<BK>(w, s, z, hi, lo);
        const uint32_t row = dst + tok * 2 * D;
        // 16 channels: the 16-byte pieces 2 u and 2 u + 1, the second one first in the upper half of the row (banks)
        const bool swap = u >= 4;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int piece = 2 * u + (swap ? 1 - i : i);
          const uint32_t a = row + (piece ^ (tok & 7)) * 16;
          const bool up = swap != (i == 1);
          sts128(a, up ? hi[4] : hi[0], up ? hi[5] : hi[1], up ? hi[6] : hi[2], up ? hi[7] : hi[3]);
          sts128(a + Pl::MAT, up ? lo[4] : lo[0], up ? lo[5] : lo[1], up ? lo[6] : lo[2], up ? lo[7] : lo[3]);
        }
      }
    } else {
      const int u = lane & 3, sub = lane >> 2;  // 16 tokens; channel
      const int c0 = (warp - 4) * (D / 4), gi = c0 / GS;
      const bool exists = t * CT + 16 * u < p.n_q;
      float mx = 0.f;
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        const uint32_t a = src + Pl::RAW_VC + (16 * u + k) * 4 * NG + 2 * gi;
        s[k] = exists ? f16_to_f(lds16(a)) : 0.f;
        z[k] = exists ? f16_to_f(lds16(a + 2 * NG)) : 0.f;
        mx = fmaxf(mx, fmaf((float)((1 << BV) - 1), s[k], fabsf(z[k])));
      }
      mx = __uint_as_float(redux_max_u32(__float_as_uint(mx)));
      const int em = mx > 0.f ? exponent_of(mx) : -30;
      // the largest |v| times 2^ev_mine in [2^6, 2^14): the exponent moves only outside that
      if (!ev_set || em + ev_mine > 13 || (em + ev_mine < 6 && em > -30)) {
        ev_mine = 13 - em;
        ev_set = true;
      }
      const float f = pow2i(ev_mine);
      if (lane == 0) v_exp[buf][warp - 4] = ev_mine;
      scale16(s, f);
      scale16(z, f);
#pragma unroll
      for (int k = 0; k < D / 32; ++k) {
        const int cl = sub + 8 * k, c = c0 + cl;
        uint32_t w;
        if constexpr (BV == 2) w = lds32(src + cl * 16 + u * 4);
        else w = lds32(src + cl * 8 + (u >> 1) * 4) >> (4 * (u & 1));
        uint32_t hi[8], lo[8];
        expand16<BV>(w, s, z, hi, lo);
        const uint32_t row = dst + 2 * Pl::MAT + c * (2 * CT);  // [channel][token]
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const uint32_t a = row + ((2 * u + i) ^ (c & 7)) * 16;
          sts128(a, hi[4 * i], hi[4 * i + 1], hi[4 * i + 2], hi[4 * i + 3]);
          sts128(a + Pl::MAT, lo[4 * i], lo[4 * i + 1], lo[4 * i + 2], lo[4 * i + 3]);
        }
      }
    }
  };

  // ---- q: rows as they came (zeros beyond the chunk), then fp16 fragments scaled per row into [1, 2) ----
  grid_dependency_wait();
  for (int i = tid; i < M * (D / 8); i += 256) {
    const int r = i / (D / 8), c = i % (D / 8);
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (r < n_rows) {
      const int row = row0 + r, j = row / G, h = row - j * G;
      v = reinterpret_cast<const uint4*>(p.q + (((size_t)j * dm.B + b) * dm.Hq + hk * G + h) * D)[c];
    }
    sts128(qs + r * Pl::QROW + c * 16, v.x, v.y, v.z, v.w);
  }
  fetch(t_lo);
  fetch(t_lo + 1);
  __syncthreads();
  const float scale2 = p.scale * 1.4426950408889634f;
  uint32_t qf[KS][4];
  float cq[2];  // logits of rows gid, gid + 8 from products of the scaled q
  int vis[2];   // tokens that these rows see
  {
    const uint32_t qa = qs + (16 * wr + gid) * Pl::QROW + tig * 4;
    float am[2] = {0.f, 0.f};
#pragma unroll
    for (int ks = 0; ks < KS; ++ks)
#pragma unroll
      for (int k = 0; k < 4; ++k) {  // a0: row gid, a1: row gid + 8; a2, a3: 8 channels on
        qf[ks][k] = lds32(qa + (k & 1) * 8 * Pl::QROW + ks * 32 + (k >> 1) * 16);
        am[k & 1] = fmaxf(am[k & 1], fmaxf(fabsf(io_to_f(qf[ks][k] & 0xffffu, p.f16)), fabsf(io_to_f(qf[ks][k] >> 16, p.f16))));
      }
    float f[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      am[r] = fmaxf(am[r], __shfl_xor_sync(0xffffffffu, am[r], 1));
      am[r] = fmaxf(am[r], __shfl_xor_sync(0xffffffffu, am[r], 2));
      const int e = am[r] > 0.f ? max(-100, min(100, -exponent_of(am[r]))) : 0;
      f[r] = pow2i(e);
      cq[r] = scale2 * pow2i(-e);
      vis[r] = min(vis0 + (row0 + 16 * wr + gid + 8 * r) / G, vis_max);
    }
#pragma unroll
    for (int ks = 0; ks < KS; ++ks)
#pragma unroll
      for (int k = 0; k < 4; ++k)
        qf[ks][k] = pack_io2<true>(io_to_f(qf[ks][k] & 0xffffu, p.f16) * f[k & 1], io_to_f(qf[ks][k] >> 16, p.f16) * f[k & 1]);
  }

  // softmax state of rows gid, gid + 8: reference (log2 units; 0 and `set` false before the first visible token)
  float mr[2] = {0.f, 0.f}, l[2] = {0.f, 0.f}, o[NO][4];
  bool set[2] = {false, false};
  int ev[4] = {0, 0, 0, 0};  // the result of channel quarter i is held times 2^ev[i]
#pragma unroll
  for (int n = 0; n < NO; ++n)
#pragma unroll
    for (int k = 0; k < 4; ++k) o[n][k] = 0.f;

  // Logits s (log2 units) of tokens t0 + 8 n + 2 tig (+ 1), rows gid and gid + 8, into numerators times 2^C_PEXP; tokens
  // from `end` on do not exist.
  auto softmax = [&](float (&s)[NT][4], int t0, int end, bool masked) {
    if (masked) {
#pragma unroll
      for (int n = 0; n < NT; ++n)
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (t0 + 8 * n + 2 * tig + (k & 1) >= min(vis[k >> 1], end)) s[n][k] = -CUDART_INF_F;
    }
    float mx[2] = {-CUDART_INF_F, -CUDART_INF_F};
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int k = 0; k < 4; ++k) mx[k >> 1] = fmaxf(mx[k >> 1], s[n][k]);
    bool need = false;
#pragma unroll
    for (int r = 0; r < 2; ++r) need |= set[r] ? mx[r] > mr[r] + C_TAU : mx[r] > -CUDART_INF_F;
    if (__any_sync(0xffffffffu, need)) {
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        float v = fmaxf(mx[r], __shfl_xor_sync(0xffffffffu, mx[r], 1));
        v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 2));
        if (v > -CUDART_INF_F && (!set[r] || v > mr[r] + (C_TAU - 1.f))) {
          const float mn = ceilf(v), f = set[r] ? ex2(mr[r] - mn) : 0.f;
          mr[r] = mn;
          set[r] = true;
          l[r] *= f;
#pragma unroll
          for (int n = 0; n < NO; ++n) {
            o[n][2 * r] *= f;
            o[n][2 * r + 1] *= f;
          }
        }
      }
    }
    const float off[2] = {(float)C_PEXP - mr[0], (float)C_PEXP - mr[1]};
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        s[n][k] = ex2(s[n][k] + off[k >> 1]);
        l[k >> 1] += s[n][k];
      }
  };

  const int x4_row = (lane & 7) + 8 * (lane >> 4), x4_piece = (lane >> 3) & 1;  // ldmatrix: this lane's row and 16-byte piece
  // products of an expanded tile
  auto multiply = [&](int t, int buf) {
    const uint32_t base = sm + buf * Pl::BUF;
    float s[NT][4];
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int k = 0; k < 4; ++k) s[n][k] = 0.f;
    const int tw = wt * TW;
#pragma unroll
    for (int ks = 0; ks < KS; ++ks)
#pragma unroll
      for (int n = 0; n < NT; n += 2) {
        const int tok = tw + 8 * n + x4_row;
        const uint32_t a = base + tok * 2 * D + ((2 * ks + x4_piece) ^ (tok & 7)) * 16;
        uint32_t b0, b1, b2, b3, c0, c1, c2, c3;
        ldmatrix_x4(a, b0, b1, b2, b3);
        ldmatrix_x4(a + Pl::MAT, c0, c1, c2, c3);
        mma_f16(s[n], qf[ks][0], qf[ks][1], qf[ks][2], qf[ks][3], b0, b1);
        mma_f16(s[n + 1], qf[ks][0], qf[ks][1], qf[ks][2], qf[ks][3], b2, b3);
        mma_f16(s[n], qf[ks][0], qf[ks][1], qf[ks][2], qf[ks][3], c0, c1);
        mma_f16(s[n + 1], qf[ks][0], qf[ks][1], qf[ks][2], qf[ks][3], c2, c3);
      }
#pragma unroll
    for (int n = 0; n < NT; ++n) {
      const float u = k_unit[buf][(tw + 8 * n) / 16];
#pragma unroll
      for (int k = 0; k < 4; ++k) s[n][k] *= cq[k >> 1] * u;
    }
    const int t0 = t * CT + tw;
    softmax(s, t0, p.n_q, t * CT + CT > min(vis_min, p.n_q));
    // exponents of the values
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int e = v_exp[buf][i];
      if (e != ev[i]) {
        const float f = pow2i(e - ev[i]);
        ev[i] = e;
#pragma unroll
        for (int n = i * QT; n < (i + 1) * QT; ++n)
#pragma unroll
          for (int k = 0; k < 4; ++k) o[n][k] *= f;
      }
    }
#pragma unroll
    for (int kk = 0; kk < TW / 16; ++kk) {
      uint32_t ph[4], pl[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float x = s[2 * kk + (k >> 1)][2 * (k & 1)], y = s[2 * kk + (k >> 1)][2 * (k & 1) + 1];
        ph[k] = pack_io2<true>(x, y);
        pl[k] = pack_io2<true>(x - io2_lo<true>(ph[k]), y - io2_hi<true>(ph[k]));
      }
#pragma unroll
      for (int n = 0; n < NO; n += 2) {
        const int c = 8 * n + x4_row;
        const uint32_t a = base + 2 * Pl::MAT + c * (2 * CT) + ((wt * (TW / 8) + 2 * kk + x4_piece) ^ (c & 7)) * 16;
        uint32_t b0, b1, b2, b3, c0, c1, c2, c3;
        ldmatrix_x4(a, b0, b1, b2, b3);
        ldmatrix_x4(a + Pl::MAT, c0, c1, c2, c3);
        mma_f16(o[n], ph[0], ph[1], ph[2], ph[3], b0, b1);
        mma_f16(o[n + 1], ph[0], ph[1], ph[2], ph[3], b2, b3);
        mma_f16(o[n], pl[0], pl[1], pl[2], pl[3], b0, b1);
        mma_f16(o[n + 1], pl[0], pl[1], pl[2], pl[3], b2, b3);
        mma_f16(o[n], ph[0], ph[1], ph[2], ph[3], c0, c1);
        mma_f16(o[n + 1], ph[0], ph[1], ph[2], ph[3], c2, c3);
      }
    }
  };

  // ---- packed tiles: tile t is multiplied while tile t + 1 is expanded into the other buffer ----
  const int t_pk = min(t_hi, pk_tiles);
  auto expand_next = [&](int t) {
    cp_async_wait<1>();
    __syncwarp();
    fetch(t + 2);
    expand(t, t & 1);
  };
  if (t_lo < t_pk) {
    expand_next(t_lo);
    __syncthreads();
    for (int t = t_lo; t < t_pk; ++t) {
      if (warp < 4 && t + 1 < t_pk) expand_next(t + 1);
      multiply(t, t & 1);
      if (warp >= 4 && t + 1 < t_pk) expand_next(t + 1);
      __syncthreads();
    }
  }
  cp_async_wait_all();

  // ---- window tiles ----
  if (max(t_lo, pk_tiles) < t_hi) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float f = pow2i(-ev[i]);
      ev[i] = 0;
#pragma unroll
      for (int n = i * QT; n < (i + 1) * QT; ++n)
#pragma unroll
        for (int k = 0; k < 4; ++k) o[n][k] *= f;
    }
    const uint8_t* wk = reinterpret_cast<const uint8_t*>(p.L.win_k) + (size_t)bh * dm.R * (2 * D);
    const uint8_t* wv = reinterpret_cast<const uint8_t*>(p.L.win_v) + (size_t)bh * dm.R * (2 * D);
    for (int t = max(t_lo, pk_tiles); t < t_hi; ++t) {
      const int w0 = (t - pk_tiles) * CT;  // first window row of the tile
      for (int i = tid; i < CT * (D / 8); i += 256) {
        const int r = i / (D / 8), c = i % (D / 8);
        const uint32_t dst = sm + r * 2 * D + (c ^ (r & 7)) * 16;
        if (w0 + r < p.r) {
          cp_async16(dst, wk + (size_t)(w0 + r) * (2 * D) + c * 16);
          cp_async16(dst + Pl::MAT, wv + (size_t)(w0 + r) * (2 * D) + c * 16);
        } else {
          sts128(dst, 0u, 0u, 0u, 0u);
          sts128(dst + Pl::MAT, 0u, 0u, 0u, 0u);
        }
      }
      cp_async_commit();
      cp_async_wait_all();
      __syncthreads();
      auto window = [&](auto f16) {
        constexpr bool F16 = decltype(f16)::value;
        float s[NT][4];
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
          for (int k = 0; k < 4; ++k) s[n][k] = 0.f;
        const int tw = wt * TW;
#pragma unroll
        for (int ks = 0; ks < KS; ++ks) {
          uint32_t a0, a1, a2, a3;
          ldmatrix_x4(qs + (16 * wr + (lane & 15)) * Pl::QROW + ks * 32 + (lane >> 4) * 16, a0, a1, a2, a3);
#pragma unroll
          for (int n = 0; n < NT; n += 2) {
            const int tok = tw + 8 * n + x4_row;
            uint32_t b0, b1, b2, b3;
            ldmatrix_x4(sm + tok * 2 * D + ((2 * ks + x4_piece) ^ (tok & 7)) * 16, b0, b1, b2, b3);
            mma16816<F16>(s[n], a0, a1, a2, a3, b0, b1);
            mma16816<F16>(s[n + 1], a0, a1, a2, a3, b2, b3);
          }
        }
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
          for (int k = 0; k < 4; ++k) s[n][k] *= scale2;
        softmax(s, p.n_q + w0 + tw, p.S, true);
#pragma unroll
        for (int kk = 0; kk < TW / 16; ++kk) {
          uint32_t ph[4], pl[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const float x = s[2 * kk + (k >> 1)][2 * (k & 1)], y = s[2 * kk + (k >> 1)][2 * (k & 1) + 1];
            ph[k] = pack_io2<F16>(x, y);
            pl[k] = pack_io2<F16>(x - io2_lo<F16>(ph[k]), y - io2_hi<F16>(ph[k]));
          }
          const int tok = tw + 16 * kk + (lane & 15);
#pragma unroll
          for (int n = 0; n < NO; n += 2) {
            uint32_t b0, b1, b2, b3;
            ldmatrix_x4_trans(sm + Pl::MAT + tok * 2 * D + ((n + (lane >> 4)) ^ (tok & 7)) * 16, b0, b1, b2, b3);
            mma16816<F16>(o[n], ph[0], ph[1], ph[2], ph[3], b0, b1);
            mma16816<F16>(o[n + 1], ph[0], ph[1], ph[2], ph[3], b2, b3);
            mma16816<F16>(o[n], pl[0], pl[1], pl[2], pl[3], b0, b1);
            mma16816<F16>(o[n + 1], pl[0], pl[1], pl[2], pl[3], b2, b3);
          }
        }
      };
      if (p.f16) window(std::true_type{}); else window(std::false_type{});
      __syncthreads();
    }
  }

  // ---- state of every warp's 16 rows into shared memory (over the tile buffers; the last tile ended in a barrier) ----
  {
    float* ws = reinterpret_cast<float*>(smem) + (size_t)warp * 16 * Pl::MS;
    float f[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) f[i] = pow2i(-ev[i]);
#pragma unroll
    for (int n = 0; n < NO; ++n)
#pragma unroll
      for (int r = 0; r < 2; ++r)
        *reinterpret_cast<float2*>(ws + (gid + 8 * r) * Pl::MS + 8 * n + 2 * tig) =
            make_float2(o[n][2 * r] * f[n / QT], o[n][2 * r + 1] * f[n / QT]);
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      l[r] += __shfl_xor_sync(0xffffffffu, l[r], 1);
      l[r] += __shfl_xor_sync(0xffffffffu, l[r], 2);
      if (tig == 0) {
        ws[(gid + 8 * r) * Pl::MS + D] = set[r] ? mr[r] : -CUDART_INF_F;
        ws[(gid + 8 * r) * Pl::MS + D + 1] = l[r];
      }
    }
  }
  __syncthreads();
  // ---- the row tile's result, or its partial: row r's state in split s at (tile * M + r) * ns + s ----
  const size_t part0 = ((size_t)rt * n_streams + bh) * M;
  auto out_row = [&](int r) {
    const int row = row0 + r, j = row / G, h = row - j * G;
    return ((size_t)j * dm.B + b) * dm.Hq + hk * G + h;
  };
  for (int i = tid; i < n_rows * D; i += 256) {
    const int r = i / D, d = i % D;
    const float* st = reinterpret_cast<const float*>(smem) + (r / 16 * 16 + r % 16) * Pl::MS;
    float Mx = -CUDART_INF_F;
#pragma unroll
    for (int w = 0; w < WT; ++w) Mx = fmaxf(Mx, st[w * M * Pl::MS + D]);
    float A = 0.f, Ls = 0.f;
#pragma unroll
    for (int w = 0; w < WT; ++w) {
      const float mw = st[w * M * Pl::MS + D];
      const float f = mw == -CUDART_INF_F ? 0.f : ex2(mw - Mx);
      A = fmaf(st[w * M * Pl::MS + d], f, A);
      Ls = fmaf(st[w * M * Pl::MS + D + 1], f, Ls);
    }
    if (p.ns == 1) {
      chunk_store<D>(p, out_row(r), d, A / Ls);
    } else {
      const size_t at = (part0 + r) * p.ns + split;
      p.part_acc[at * D + d] = A;
      if (d == 0) *reinterpret_cast<float2*>(p.part_ml + at * 2) = make_float2(Mx, Ls);
    }
  }
  if (p.ns == 1) return;
  // the last CTA of the row tile merges (ticket as in the decode kernel)
  unsigned* ticket = p.tickets + (size_t)rt * n_streams + bh;
  __syncthreads();
  if (tid == 0) {
    unsigned t;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;\n" : "=r"(t) : "l"(ticket) : "memory");
    s_flag = (t == (unsigned)(p.ns - 1));
  }
  __syncthreads();
  if (!s_flag) return;
  for (int i = tid; i < n_rows * (D / 2); i += 256) {
    const int r = i / (D / 2), d = 2 * (i % (D / 2));
    const float* pa = p.part_acc + (part0 + r) * p.ns * D + d;
    const float* ml = p.part_ml + (part0 + r) * p.ns * 2;
    float Mx = -CUDART_INF_F;
    for (int s = 0; s < p.ns; ++s) Mx = fmaxf(Mx, ld_cg(ml + 2 * s));
    float ax = 0.f, ay = 0.f, Ls = 0.f;
    for (int s = 0; s < p.ns; ++s) {
      const float2 x = ld_cg2(ml + 2 * s), v = ld_cg2(pa + (size_t)s * D);
      const float f = x.x == -CUDART_INF_F ? 0.f : ex2(x.x - Mx);
      ax = fmaf(v.x, f, ax);
      ay = fmaf(v.y, f, ay);
      Ls = fmaf(x.y, f, Ls);
    }
    const float inv = 1.0f / Ls;
    chunk_store<D>(p, out_row(r), d, ax * inv);
    chunk_store<D>(p, out_row(r), d + 1, ay * inv);
  }
  if (tid == 0) *ticket = 0u;
}

template <int D, int BK, int BV, int GS, int WR>
cudaError_t chunk_launch_one(const ChunkParams& p, cudaStream_t st) {
  using Pl = ChunkPlan<D, BK, BV, GS, WR>;
  auto kernel = chunk_kernel<D, BK, BV, GS, WR>;
  const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, Pl::TOTAL);
  if (e != cudaSuccess) return e;
  return launch_dependent(kernel, dim3((unsigned)p.row_tiles * p.dm.B * p.dm.Hkv * p.ns), dim3(256), (size_t)Pl::TOTAL, st, p);
}

}  // namespace

template <int D, int WR>
cudaError_t launch_chunk_t(const ChunkParams& p, cudaStream_t st) {
  switch (p.L.bk * 100 + p.L.bv * 10 + (p.dm.g == 64)) {
    case 220: return chunk_launch_one<D, 2, 2, 32, WR>(p, st);
    case 221: return chunk_launch_one<D, 2, 2, 64, WR>(p, st);
    case 210: return chunk_launch_one<D, 2, 1, 32, WR>(p, st);
    case 211: return chunk_launch_one<D, 2, 1, 64, WR>(p, st);
    case 120: return chunk_launch_one<D, 1, 2, 32, WR>(p, st);
    case 121: return chunk_launch_one<D, 1, 2, 64, WR>(p, st);
    case 110: return chunk_launch_one<D, 1, 1, 32, WR>(p, st);
    case 111: return chunk_launch_one<D, 1, 1, 64, WR>(p, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace xq
