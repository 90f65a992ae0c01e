// Attention of a chunk of query tokens over the packed cache plus the window, causal inside the chunk: the query rows
// (tokens x heads of a kv head) share one pass over the cache.  tcgen05 products.
//
// A CTA takes 128 rows and a range of 64-token tiles of one (sequence, kv head).  With that many rows per code it pays
// to dequantize: eight warps expand a tile's keys and values once for all rows into fp16 pairs hi + lo in shared
// memory (22 significant bits of c s + z, relative to the largest member of the group), the B operands of
//
//   S = Q K_hi + Q K_lo                          (A: q as fp16 in tensor memory; S: 64 columns, four buffers)
//   O += P_hi V_hi + P_hi V_lo + P_lo V_hi       (A: the softmax numerators as fp16 pairs, over the columns of S)
//
// accumulated in fp32 in tensor memory.  Two groups of four warps (thread = row = tensor-memory lane) take the softmax
// of the even and of the odd tiles; the softmax reference of a row goes from one to the other through shared memory
// and is raised only when a logit exceeds it by more than 8 (log2 units), which rescales O (rare).  One warp issues the
// products: keys of tile i + 2, then values of tile i.  Tokens of the 16-bit window are expanded into the same pairs
// (exactly).  Split partials are merged by the last CTA of a row tile, as in the decode kernel.
//
// What bounds it: the expanding warps, ~2800-3300 cycles per tile (the products: ~1650), and with them the instruction
// cache: hot code above ~30 KB runs slower, so the loops are rolled.  Against one decode launch per query token, us:
// 16 tokens behind 32k, batch 4, four layers, 2278 -> 922; 250 tokens behind 8k, two layers, 6063 -> 499; a prompt of
// 1024, 32 kv heads, two layers, 10516 -> 123.  In the same order: four more expanding warps, at 80 registers a thread,
// were slower, 969 / 532 / 125; four S buffers, so that the keys of two tiles are ahead, took 1108 / 532 / 137 to
// 1056 / 506 / 136, softmax in two passes of 32 columns those to 922 / 499 / 123.
//
// Every wait on an mbarrier is bounded: a thread that gives up sets a flag in shared memory that makes every other
// wait of the CTA give up too; the CTA then waits for its products in flight, frees its tensor memory, reports through
// the status word and leaves without a result.
#pragma once
#include <type_traits>

#include "xq_internal.h"
#include "xq_mma.cuh"

namespace xq {
namespace {

constexpr int CM = CHUNK_ROWS;     // query rows of a CTA
constexpr int CT = 64;             // tokens of a tile
constexpr int C_STAGES = 3;        // raw tiles in flight
constexpr float C_TAU = 8.f;       // log2 units a logit may exceed the softmax reference before it is raised
constexpr int C_PEXP = 6;          // numerators are carried times 2^C_PEXP (at most 2^14 as fp16)
constexpr int C_EXPAND = 8;        // expanding warps (8 .. 15): keys 0 .. 3, values 4 .. 7
constexpr int C_THREADS = (8 + C_EXPAND + 1) * 32;

// ---- tcgen05 ----
// shared-memory matrix descriptor, N-major, no swizzle: core matrices of 8 K-rows x 16 bytes of N;
// lbo / sbo: byte distance between core matrices along K / along N
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((addr >> 4) & 0x3fff);
  d |= (uint64_t)((lbo >> 4) & 0x3fff) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3fff) << 32;
  d |= (uint64_t)1 << 46;  // descriptor version of this architecture
  return d;
}
// kind::f16 instruction descriptor: fp16 A (K-major, tensor memory) and B (N-major), fp32 accumulate, M = 128
__host__ __device__ constexpr uint32_t idesc_f16(int n) {
  return (1u << 4) | (1u << 16) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}
// D[128 x N] (+)= A[128 x 16] (tensor memory) * B[16 x N] (shared memory); issued by one thread
__device__ __forceinline__ void umma_f16(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, bool accumulate) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d_tmem),
      "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"((uint32_t)accumulate) : "memory");
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(bar) : "memory");
}
__device__ __forceinline__ uint32_t elect_one() {
  uint32_t pred;
  asm volatile("{\n.reg .pred P;\nelect.sync _|P, 0xffffffff;\nselp.u32 %0, 1, 0, P;\n}\n" : "=r"(pred));
  return pred;
}

template <int D, int BK, int BV, int GS>
struct ChunkPlan {
  static constexpr int NG = D / GS;
  static constexpr int KROW = D * BK / 8;                       // packed bytes of a token's keys
  // An expanded matrix: core matrices of 8 x 8 elements (rows: channels of the keys, tokens of the values; a row's 16
  // bytes: tokens of the keys, channels of the values), CORE bytes apart along the rows (16 more than their size, so
  // that the four rows which each of eight lanes writes fall into different banks).
  static constexpr int CORE = 144, K_SBO = D / 8 * CORE, V_SBO = CT / 8 * CORE;
  static constexpr int MAT = CT / 8 * K_SBO;
  static constexpr int KBUFS = 2, VBUFS = 3;                    // expanded tiles of keys, of values (hi and lo each)
  static constexpr int OFF_V = KBUFS * 2 * MAT;
  // raw data of a key warp (16 tokens: codes, their group's parameters) and of a value warp (D / 4 channels: codes,
  // the tile's parameters with 16 bytes more after every four tokens)
  static constexpr int RAW_KC = 16 * KROW, RAW_K = RAW_KC + 4 * D;
  static constexpr int RAW_VC = (D / 4) * 8 * BV, V_QUAD = 16 * NG + 16, RAW_V = RAW_VC + CT / 4 * V_QUAD;
  static constexpr int OFF_RAW = OFF_V + VBUFS * 2 * MAT;
  static constexpr int TOTAL = OFF_RAW + 4 * C_STAGES * (RAW_K + RAW_V);
  // tensor memory columns: q, S (then numerators) of four tiles, O; head_dim 64: the sum of earlier O
  static constexpr uint32_t COL_Q = 0, COL_S = 64, COL_O = 320, COL_T = 384;
  // Tiles after which O is added to the sum (in fp32) and starts over, 0: never.  Every product's addition to O drops
  // what lies below its last digit, always in one direction: after 8000 tokens, 1500 products, the fp32 result was 8.8e-6
  // of its norm off.  With head_dim 64, where the scalar kernel is the measure (4.1, 5.3, 7.8e-7 at 512, 2000, 8000
  // tokens), sums of 8 tiles leave 15.6e-7 at 8000, of 4 10.8e-7, of 2 8.5e-7, and those with the small products first
  // 4.4, 5.8, 7.6e-7.  300 query tokens at 2048: 49 us without, 50, 52, 56 us.  (head_dim 128 has no columns left; its
  // measure, one decode call per token, is 0.2-1.4e-5.)
  static constexpr int FLUSH = D == 64 ? 2 : 0;
  static_assert(TOTAL <= 226 * 1024, "shared memory");
};

template <int D>
__device__ __forceinline__ void chunk_store(const ChunkParams& p, size_t row, int c, float v) {
  if (p.out_f32) reinterpret_cast<float*>(p.out)[row * D + c] = v;
  else if (p.f16) reinterpret_cast<__half*>(p.out)[row * D + c] = __float2half_rn(v);
  else reinterpret_cast<__nv_bfloat16*>(p.out)[row * D + c] = __float2bfloat16_rn(v);
}

// hi = RN16(v), lo = RN16(v - hi) of a pair
__device__ __forceinline__ void split2(float a, float b, uint32_t& hi, uint32_t& lo) {
  hi = pack_io2<true>(a, b);
  lo = pack_io2<true>(a - io2_lo<true>(hi), b - io2_hi<true>(hi));
}

// The values that the codes 0 .. 3 of a group stand for, c s + z (s and z in units of the expanded tile), as fp16
// pairs: hi[c / 2], lo[c / 2].
struct Table {
  uint32_t hi[2], lo[2];
};
__device__ __forceinline__ Table make_table(float s, float z) {
  Table t;
  split2(z, z + s, t.hi[0], t.lo[0]);
  split2(fmaf(2.f, s, z), fmaf(3.f, s, z), t.hi[1], t.lo[1]);
  return t;
}
// One 4 x 8 block of an expanded matrix: byte j of the words w[k] >> sh holds the code of row j, position k.  Four
// codes make a selector of two byte permutations (code c selects the bytes 2 c and 2 c + 1 of the table), so an element
// takes three instructions for its hi and lo.
template <int BITS>
__device__ __forceinline__ void expand_block(const uint32_t (&w)[8], int sh, const Table (&t)[4], uint32_t dst, uint32_t lo_off) {
  uint32_t c[2][4];  // codes of four positions of row j
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    uint32_t m[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) m[k] = (w[4 * h + k] >> sh) & (BITS == 2 ? 0x03030303u : 0x01010101u);
    const uint32_t a0 = __byte_perm(m[0], m[1], 0x5140), a1 = __byte_perm(m[2], m[3], 0x5140);
    const uint32_t b0 = __byte_perm(m[0], m[1], 0x7362), b1 = __byte_perm(m[2], m[3], 0x7362);
    c[h][0] = __byte_perm(a0, a1, 0x5410); c[h][1] = __byte_perm(a0, a1, 0x7632);
    c[h][2] = __byte_perm(b0, b1, 0x5410); c[h][3] = __byte_perm(b0, b1, 0x7632);
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const uint32_t s0 = c[0][j] * 0x22u + 0x10101010u, s1 = c[1][j] * 0x22u + 0x10101010u;
    const uint32_t u0 = s0 >> 16, u1 = s1 >> 16;
    sts128(dst + 16 * j, __byte_perm(t[j].hi[0], t[j].hi[1], s0), __byte_perm(t[j].hi[0], t[j].hi[1], u0),
           __byte_perm(t[j].hi[0], t[j].hi[1], s1), __byte_perm(t[j].hi[0], t[j].hi[1], u1));
    sts128(dst + lo_off + 16 * j, __byte_perm(t[j].lo[0], t[j].lo[1], s0), __byte_perm(t[j].lo[0], t[j].lo[1], u0),
           __byte_perm(t[j].lo[0], t[j].lo[1], s1), __byte_perm(t[j].lo[0], t[j].lo[1], u1));
  }
}
// eight fp32 values as hi and lo rows of 16 bytes; bad: some may not be finite (an infinity less its hi is not a number;
// the lo of a number below 2^15 is below 64)
__device__ __forceinline__ void store_row(const float (&v)[8], uint32_t dst, uint32_t lo_off, bool bad) {
  uint32_t hi[4], lo[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) split2(v[2 * k], v[2 * k + 1], hi[k], lo[k]);
  if (bad) {
#pragma unroll
    for (int k = 0; k < 4; ++k)
      lo[k] = pack_io2<true>(fminf(v[2 * k] - io2_lo<true>(hi[k]), 64.f), fminf(v[2 * k + 1] - io2_hi<true>(hi[k]), 64.f));
  }
  sts128(dst, hi[0], hi[1], hi[2], hi[3]);
  sts128(dst + lo_off, lo[0], lo[1], lo[2], lo[3]);
}
constexpr uint32_t INF32 = 0x7f800000u;  // |x| as bits: at or above, x is not a number or infinite
__device__ __forceinline__ uint32_t abs_bits(float x) { return __float_as_uint(x) & 0x7fffffffu; }
// 16-bit patterns: the smallest one that is not a finite number, but for the sign; a pair without its elements from there on
__device__ __forceinline__ uint32_t inf16(int f16) { return f16 ? 0x7c00u : 0x7f80u; }
__device__ __forceinline__ uint32_t finite_pair(uint32_t w, uint32_t inf) {
  return ((w & 0x7fffu) < inf ? w & 0xffffu : 0u) | (((w >> 16) & 0x7fffu) < inf ? w & 0xffff0000u : 0u);
}
__device__ __forceinline__ uint32_t max_pair(uint32_t m, uint32_t w) { return __vmaxu2(m, w & 0x7fff7fffu); }
__device__ __forceinline__ uint32_t redux_pair(uint32_t m) { return redux_max_u32(max(m & 0xffffu, m >> 16)); }
// 2^e that puts mx below 2^15 and, unless it is there already, above 2^14
__device__ __forceinline__ int key_exponent(float mx) {
  return mx >= 1.f && mx < 32768.f ? 0 : (mx > 0.f ? 14 - exponent_of(mx) : 0);
}

// What elements that are not finite need, out of line: the loops that never meet any keep their place in the instruction
// cache (16 tokens at 32k, us a layer: in line 229 to 237, as it is 230, without any of it 226).
struct BadRows {  // the rows of a CTA, as they see tokens
  uint32_t (*row_bad)[4];
  int* any_bad;
  int vis0, row0, G;
};
// the rows that see token tok (counted from the layer's first) see values that are not finite, in channels `mask` of
// quarter `quarter`
__device__ __noinline__ void mark_rows(const BadRows& b, int tok, int quarter, uint32_t mask) {
  if (mask == 0u) return;
  for (int r = 0; r < CM; ++r)
    if (tok < b.vis0 + (b.row0 + r) / b.G) atomicOr(&b.row_bad[r][quarter], mask);
  *b.any_bad = 1;
}
// largest finite pattern among 4 channels of 32 window rows from r0 (every step-th from first), of r rows
__device__ __noinline__ uint32_t finite_key_max(const uint2* rows, int r0, int first, int step, int r, int row_vecs, uint32_t inf) {
  uint32_t mp = 0u;
#pragma unroll 1
  for (int x = first; x < 32; x += step)
    if (r0 + x < r) {
      const uint2 v = rows[(size_t)(r0 + x) * row_vecs];
      mp = max_pair(max_pair(mp, finite_pair(v.x, inf)), finite_pair(v.y, inf));
    }
  return redux_pair(mp);
}

template <int D, int BK, int BV, int GS>
__global__ void __launch_bounds__(C_THREADS, 1) chunk_kernel(const __grid_constant__ ChunkParams p) {
  using Pl = ChunkPlan<D, BK, BV, GS>;
  constexpr int NG = Pl::NG, DQ = D / 4;
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ __align__(8) unsigned long long bar_mem[39];
  __shared__ float k_unit[8][2];            // [tile % 8][32 tokens]: what a unit of the expanded keys is worth
  __shared__ __align__(16) int v_exp[4][4];               // [tile % 4][channel quarter]: the expanded values are times 2^v_exp
  __shared__ float cq_sm[CM], m_sm[CM];     // logits from products of the scaled q; softmax reference (-infinity: none)
  __shared__ float l_sm[2][CM], ml_sm[2][CM];
  // Values that are not finite: a row that does not see their token must not get them, and its zero numerator does not
  // keep them out of a product.  They are expanded as zeros; rows that do see them get a NaN in those channels at the end.
  __shared__ uint32_t row_bad[CM][4];       // [row][channel quarter]: channels in which a row sees any
  __shared__ int any_bad;
  __shared__ uint32_t tmem_base_sm;
  __shared__ int s_flag;
  __shared__ volatile int dead_sm;

  const Dims& dm = p.dm;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int G = dm.G, n_streams = dm.B * dm.Hkv;
  // the row tiles with the most visible tokens first
  const int split = blockIdx.x % p.ns, bh = (blockIdx.x / p.ns) % n_streams, rt = p.row_tiles - 1 - blockIdx.x / p.ns / n_streams;
  const int hk = bh % dm.Hkv, b = bh / dm.Hkv;
  const int row0 = rt * CM, n_rows = min(CM, p.T * G - row0);  // row: query token row / G, head row % G
  const int vis0 = p.S - p.T + 1;                              // tokens that query token 0 sees
  const int vis_max = vis0 + (row0 + n_rows - 1) / G;
  const int n_packed = min(p.n_q, vis_max);
  const int pk_tiles = (n_packed + CT - 1) / CT, all_tiles = pk_tiles + (vis_max - n_packed + CT - 1) / CT;
  int t_lo, t_hi;
  share_of(all_tiles, p.ns, split, t_lo, t_hi);
  const int N = t_hi - t_lo;

  const uint32_t sm = (uint32_t)__cvta_generic_to_shared(smem);
  const uint32_t bars = (uint32_t)__cvta_generic_to_shared(&bar_mem[0]);
  const uint32_t bar_kfull = bars;             // [2] a tile's keys are expanded
  const uint32_t bar_kfree = bar_kfull + 16;   // [2] their buffer may be written again
  const uint32_t bar_vfull = bar_kfree + 16;   // [3] the same of the values
  const uint32_t bar_vfree = bar_vfull + 24;   // [3]
  const uint32_t bar_s = bar_vfree + 24;       // [4] S is complete
  const uint32_t bar_p = bar_s + 32;           // [4] the numerators are written
  const uint32_t bar_o = bar_p + 32;           // [4] the value products of a tile are complete
  const uint32_t bar_turn = bar_o + 32;        // [4 warps][2] a row's reference for an even / odd tile is there
  const uint32_t bar_unit = bar_turn + 64;     // [8] the units of a tile's keys are written
  const uint32_t bar_end = bar_unit + 64;      // every product that was issued is complete (after a wait gave up)

  if (tid == 0) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      mbar_init(bar_kfull + 8 * i, C_EXPAND / 2);
      mbar_init(bar_kfree + 8 * i, 1);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      mbar_init(bar_s + 8 * i, 1);
      mbar_init(bar_p + 8 * i, 4);
      mbar_init(bar_o + 8 * i, 1);
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      mbar_init(bar_vfull + 8 * i, C_EXPAND / 2);
      mbar_init(bar_vfree + 8 * i, 1);
    }
    mbar_init(bar_end, 1);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      mbar_init(bar_turn + 8 * i, 1);
      mbar_init(bar_unit + 8 * i, C_EXPAND / 2);
    }
    dead_sm = 0;
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  // Tensor memory is asked for after the wait: a CTA of the preceding kernel that shares the SM may still have to get
  // its own, and with all columns taken here it would wait for this CTA, which waits for it.
  grid_dependency_wait();
  if (warp == 8 + C_EXPAND) {
    tmem_alloc((uint32_t)__cvta_generic_to_shared(&tmem_base_sm), 512u);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tbase = tmem_base_sm;
  const uint32_t row_t = tbase + ((uint32_t)((warp & 3) * 32) << 16);

  if (warp < 4) {
    // ---- q: this thread's row as fp16 scaled by a power of two into [1, 2), to tensor memory ----
    const int row = row0 + tid, j = row / G, h = row - j * G;
    const bool real = tid < n_rows;
    const uint4* src = reinterpret_cast<const uint4*>(p.q + (real ? (((size_t)j * dm.B + b) * dm.Hq + hk * G + h) * D : 0));
    uint32_t w[D / 2];
    float am = 0.f;
#pragma unroll
    for (int i = 0; i < D / 8; ++i) {
      const uint4 v = real ? src[i] : make_uint4(0u, 0u, 0u, 0u);
      w[4 * i] = v.x; w[4 * i + 1] = v.y; w[4 * i + 2] = v.z; w[4 * i + 3] = v.w;
    }
#pragma unroll
    for (int i = 0; i < D / 2; ++i)
      am = fmaxf(am, fmaxf(fabsf(io_to_f(w[i] & 0xffffu, p.f16)), fabsf(io_to_f(w[i] >> 16, p.f16))));
    const int e = am > 0.f ? max(-100, min(100, -exponent_of(am))) : 0;
    const float f = pow2i(e);
#pragma unroll
    for (int c = 0; c < D / 64; ++c) {
      uint32_t r[32];
#pragma unroll
      for (int i = 0; i < 32; ++i)
        r[i] = pack_io2<true>(io_to_f(w[32 * c + i] & 0xffffu, p.f16) * f, io_to_f(w[32 * c + i] >> 16, p.f16) * f);
      tmem_st<32>(row_t + Pl::COL_Q + 32 * c, r);
    }
    if constexpr (Pl::FLUSH != 0) {
      uint32_t zero[32];
#pragma unroll
      for (int i = 0; i < 32; ++i) zero[i] = 0u;
#pragma unroll
      for (int c = 0; c < D; c += 32) tmem_st<32>(row_t + Pl::COL_T + c, zero);
    }
    tc_wait_st();
#pragma unroll
    for (int k = 0; k < 4; ++k) row_bad[tid][k] = 0u;
    if (tid == 0) any_bad = 0;
    cq_sm[tid] = p.scale * 1.4426950408889634f * pow2i(-e);
    m_sm[tid] = -CUDART_INF_F;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();

  if (warp == 8 + C_EXPAND) {
    // ================= products: the loop is warp-uniform, one elected lane issues =================
    constexpr uint32_t IDK = idesc_f16(CT), IDV = idesc_f16(D);
    constexpr uint32_t KSTEP = 2 * Pl::CORE / 16;  // descriptor units per 16 rows of K
    // (uniform values: the issue of a product then takes no moves between register files)
    const uint32_t tb = __shfl_sync(0xffffffffu, tbase, 0), smu = __shfl_sync(0xffffffffu, sm, 0);
    // keys of tile i + 2 go out before the values of tile i: either softmax group finds its next S complete
#pragma unroll 1
    for (int i = 0; i < N + 2; ++i) {
      bool ok = true;
      if (i < N) {
        ok = __all_sync(0xffffffffu, mbar_wait(bar_kfull + 8 * (i & 1), (i >> 1) & 1, &dead_sm));
        tc_fence_after();
        if (ok && elect_one()) {
          const uint32_t base = smu + (i & 1) * 2 * Pl::MAT, dS = tb + Pl::COL_S + (i & 3) * 64;
          // the small products first, here and below: a sum drops what lies below its own last digit
          const uint64_t kh = smem_desc(base, Pl::CORE, Pl::K_SBO), kl = smem_desc(base + Pl::MAT, Pl::CORE, Pl::K_SBO);
#pragma unroll
          for (int ks = 0; ks < D / 16; ++ks) umma_f16(dS, tb + Pl::COL_Q + 8 * ks, kl + KSTEP * ks, IDK, ks > 0);
#pragma unroll
          for (int ks = 0; ks < D / 16; ++ks) umma_f16(dS, tb + Pl::COL_Q + 8 * ks, kh + KSTEP * ks, IDK, true);
          umma_commit(bar_s + 8 * (i & 3));
          umma_commit(bar_kfree + 8 * (i & 1));
        }
        __syncwarp();
      }
      if (ok && i >= 2) {
        const int j = i - 2;
        ok = __all_sync(0xffffffffu, mbar_wait(bar_vfull + 8 * (j % 3), (j / 3) & 1, &dead_sm) &&
                                         mbar_wait(bar_p + 8 * (j & 3), (j >> 2) & 1, &dead_sm));
        tc_fence_after();
        if (ok && elect_one()) {
          const uint32_t base = smu + Pl::OFF_V + (j % 3) * 2 * Pl::MAT;
          const uint32_t pt = tb + Pl::COL_S + (j & 3) * 64, dO = tb + Pl::COL_O;
          const uint64_t vh = smem_desc(base, Pl::CORE, Pl::V_SBO), vl = smem_desc(base + Pl::MAT, Pl::CORE, Pl::V_SBO);
#pragma unroll
          for (int ks = 0; ks < CT / 16; ++ks) {
            const uint32_t ph = pt + 32 * (ks >> 1) + 8 * (ks & 1), pl = ph + 16;
            umma_f16(dO, ph, vl + KSTEP * ks, IDV, j > 0 || ks > 0);
            umma_f16(dO, pl, vh + KSTEP * ks, IDV, true);
          }
#pragma unroll
          for (int ks = 0; ks < CT / 16; ++ks) umma_f16(dO, pt + 32 * (ks >> 1) + 8 * (ks & 1), vh + KSTEP * ks, IDV, true);
          umma_commit(bar_o + 8 * (j & 3));
          umma_commit(bar_vfree + 8 * (j % 3));
        }
        __syncwarp();
      }
      if (!ok) break;
    }
    if (__any_sync(0xffffffffu, dead_sm != 0)) {  // products may be in flight: wait for them (bounded) before the memory they use is given up
      if (elect_one()) {
        umma_commit(bar_end);
        for (int k = 0; k < WAIT_LIMIT && !mbar_try_wait(bar_end, 0); ++k) {}
      }
      __syncwarp();
    }
  } else if (warp < 8) {
    // ================= softmax: group w takes the tiles i = w, w + 2, ...; thread = row =================
    const int w = warp >> 2, q = warp & 3, r = tid & 127;
    const bool idle = 32 * q >= n_rows;  // none of this warp's rows exists: its lanes hold whatever is there
    const float cq = cq_sm[r];
    const int vis = min(vis0 + (row0 + r) / G, vis_max);
    float l = 0.f, ml = -CUDART_INF_F;
#pragma unroll 1
    for (int i = w; i < N; i += 2) {
      // (the units and exponents of the expanded tile are there since the first two; the third one is the wait)
      // (Phases: the keys run up to four tiles ahead of this one and the values up to two, so that neither the eight
      // unit barriers nor the three of the values can be a whole round ahead of the parity that is asked for; S of
      // this tile being complete, so are the value products of the tile three before.)
      if (!__all_sync(0xffffffffu, mbar_wait(bar_unit + 8 * (i & 7), (i >> 3) & 1, &dead_sm) &&
                                       mbar_wait(bar_vfull + 8 * (i % 3), (i / 3) & 1, &dead_sm) &&
                                       mbar_wait(bar_s + 8 * (i & 3), (i >> 2) & 1, &dead_sm)))
        break;
      tc_fence_after();
      const uint32_t s_t = row_t + Pl::COL_S + (i & 3) * 64;
      const float u[2] = {k_unit[i & 7][0] * cq, k_unit[i & 7][1] * cq};
      const int t = t_lo + i;
      // columns below n_valid are tokens that exist and that this row sees
      const int n_valid = t < pk_tiles ? min(vis, p.n_q) - t * CT : vis - p.n_q - (t - pk_tiles) * CT;
      if (!idle) {
        const bool masked = __any_sync(0xffffffffu, n_valid < CT);
        // 32 columns of S at a time, here and below: the loops stay small (the instruction cache bounds this kernel)
        auto load = [&](int c, uint32_t (&s)[32]) {
          tmem_ld<32>(s_t + 32 * c, s);
          tc_wait_ld();
          if (masked) {
#pragma unroll
            for (int k = 0; k < 32; ++k)
              if (32 * c + k >= n_valid) s[k] = 0xff800000u;
          }
        };
        float xm = -CUDART_INF_F;
#pragma unroll 1
        for (int c = 0; c < 2; ++c) {
          uint32_t s[32];
          load(c, s);
          float x = __uint_as_float(s[0]);
#pragma unroll
          for (int k = 1; k < 32; ++k) x = fmaxf(x, __uint_as_float(s[k]));
          xm = fmaxf(xm, x * (c ? u[1] : u[0]));
        }
        if (i > 0 && !__all_sync(0xffffffffu, mbar_wait(bar_turn + 8 * (2 * q + (i & 1)), ((i - 1) >> 1) & 1, &dead_sm))) break;
        const float m_old = m_sm[r];
        float m = m_old;
        if (xm > m_old + C_TAU || (m_old == -CUDART_INF_F && xm > m_old)) m = ceilf(xm);
        bool change = m != m_old;
        if (i > 0) {
          const int4 e1 = *reinterpret_cast<const int4*>(v_exp[i & 3]), e0 = *reinterpret_cast<const int4*>(v_exp[(i - 1) & 3]);
          change |= e1.x != e0.x || e1.y != e0.y || e1.z != e0.z || e1.w != e0.w;
          if constexpr (Pl::FLUSH != 0) change |= i % Pl::FLUSH == 0;
        }
        if (__any_sync(0xffffffffu, change)) {
          m_sm[r] = m;
          if (i > 0) {  // O has to follow: after the products of the tile before, before those of this one
            if (!__all_sync(0xffffffffu, mbar_wait(bar_o + 8 * ((i - 1) & 3), ((i - 1) >> 2) & 1, &dead_sm))) break;
            tc_fence_after();
            const float f = m_old == -CUDART_INF_F ? 0.f : ex2(m_old - m);
#pragma unroll 1
            for (int c = 0; c < D; c += 32) {
              const int qa = c / DQ, qz = (c + 31) / DQ;  // the channel quarters of the columns' halves
              const float fa = f * pow2i(v_exp[i & 3][qa] - v_exp[(i - 1) & 3][qa]);
              const float fz = f * pow2i(v_exp[i & 3][qz] - v_exp[(i - 1) & 3][qz]);
              uint32_t s[32];
              tmem_ld<32>(row_t + Pl::COL_O + c, s);
              if constexpr (Pl::FLUSH != 0) {
                uint32_t sum[32];
                tmem_ld<32>(row_t + Pl::COL_T + c, sum);
                tc_wait_ld();
#pragma unroll
                for (int k = 0; k < 32; ++k) {
                  sum[k] = __float_as_uint((__uint_as_float(sum[k]) + __uint_as_float(s[k])) * (k < 16 ? fa : fz));
                  s[k] = 0u;
                }
                tmem_st<32>(row_t + Pl::COL_T + c, sum);
              } else {
                tc_wait_ld();
#pragma unroll
                for (int k = 0; k < 32; ++k) s[k] = __float_as_uint(__uint_as_float(s[k]) * (k < 16 ? fa : fz));
              }
              tmem_st<32>(row_t + Pl::COL_O + c, s);
            }
            tc_wait_st();
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_turn + 8 * (2 * q + ((i + 1) & 1)));
        // numerators: the 32 columns of S become 16 of hi and 16 of lo, two tokens in each
        const float off = m == -CUDART_INF_F ? 0.f : (float)C_PEXP - m;
        l *= m == ml ? 1.f : ex2(ml - m);
        ml = m;
#pragma unroll 1
        for (int c = 0; c < 2; ++c) {
          uint32_t s[32], o[32];
          load(c, s);
          const float uc = c ? u[1] : u[0];
          float la = 0.f, lb = 0.f;
#pragma unroll
          for (int k = 0; k < 16; ++k) {
            const float a = ex2(fmaf(__uint_as_float(s[2 * k]), uc, off)), d = ex2(fmaf(__uint_as_float(s[2 * k + 1]), uc, off));
            la += a;
            lb += d;
            split2(a, d, o[k], o[16 + k]);
          }
          l += la + lb;
          tmem_st<32>(s_t + 32 * c, o);
        }
        tc_wait_st();
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_p + 8 * (i & 3));
    }
    l_sm[w][r] = l;
    ml_sm[w][r] = ml;
  } else {
    // ================= expansion: keys (warps 8 .. 11: 16 tokens each), values (12 .. 15: D / 4 channels each) =========
    const int ew = warp - 8;
    const bool keys = ew < 4;
    const uint32_t raw = sm + Pl::OFF_RAW + (keys ? ew * C_STAGES * Pl::RAW_K : C_STAGES * (4 * Pl::RAW_K + (ew - 4) * Pl::RAW_V));
    const int n_pk = min(t_hi, pk_tiles);
    const int c0 = (ew & 3) * DQ;  // value warps: first channel
    const uint8_t* const g_code = keys
        ? reinterpret_cast<const uint8_t*>(p.L.k_codes) + (size_t)bh * ((size_t)dm.nq_cap * Pl::KROW)
        : reinterpret_cast<const uint8_t*>(p.L.v_codes) + (size_t)bh * ((size_t)dm.nq_cap * (D * BV / 8));
    const uint8_t* const g_meta = keys
        ? reinterpret_cast<const uint8_t*>(p.L.k_meta) + (size_t)bh * ((size_t)(dm.nq_cap / GS) * 4 * D)
        : reinterpret_cast<const uint8_t*>(p.L.v_meta) + (size_t)bh * ((size_t)dm.nq_cap * 4 * NG);
    // Raw data of packed tile t_lo + i that this warp expands, into its own stage; one commit per call
    auto fetch = [&](int i) {
      const int t = t_lo + i;
      if (t < n_pk) {
        if (keys) {
          const uint32_t dst = raw + (i % C_STAGES) * Pl::RAW_K;
          const int tok = t * CT + 16 * ew;
          const uint8_t* src = g_code + (size_t)(tok / 32) * (32 * Pl::KROW);
          if (lane < Pl::KROW) {  // 16 tokens x KROW bytes in 16-byte pieces
            if constexpr (Pl::KROW == 32) cp_async16(dst + lane * 16, src + (lane >> 4) * 512 + (tok % 32 + (lane & 15)) * 16);
            else cp_async16(dst + lane * 16, src + (tok % 32) * Pl::KROW + lane * 16);
          }
          if (lane < D / 4) cp_async16(dst + Pl::RAW_KC + lane * 16, g_meta + (size_t)(tok / GS) * (4 * D) + lane * 16);
        } else {
          const uint32_t dst = raw + (i % C_STAGES) * Pl::RAW_V;
          const uint8_t* src = g_code + (size_t)(t / 2) * (D * 16 * BV);
          if (lane < DQ) {
            if constexpr (BV == 2) cp_async16(dst + lane * 16, src + (t & 1) * (D * 16) + (c0 + lane) * 16);
            else cp_async8(dst + lane * 8, src + (c0 + lane) * 16 + (t & 1) * 8);
          }
#pragma unroll
          for (int k = 0; k < (CT * NG / 4 + 31) / 32; ++k) {
            const int x = lane + 32 * k;
            if (x < CT * NG / 4) cp_async16(dst + Pl::RAW_VC + x * 16 + x / NG * 16, g_meta + (size_t)t * (CT * 4 * NG) + x * 16);
          }
        }
      }
      cp_async_commit();
    };
    // keys: this lane's four channels 4 k_q .. and its blocks of 8 tokens; values: four tokens 4 v_q .. and 8 channels
    const int k_q = lane % (D / 4), k_b = lane / (D / 4), v_q = lane & 15, v_h = lane >> 4;
    constexpr int KB = D / 64;  // blocks of a lane: 2 (D = 128) or 1
    const uint32_t k_dst = (k_q >> 1) * Pl::CORE + (k_q & 1) * 64, v_dst = (v_q >> 1) * Pl::CORE + (v_q & 1) * 64;
    int ev = 0;
    bool ev_set = false;
    // exponent of the values in use: the largest |v| times 2^ev in [2^4, 2^14); it moves only outside that
    auto value_exponent = [&](uint32_t mb) {
      const float mx = __uint_as_float(mb);
      const int em = mx > 0.f ? exponent_of(mx) : -100;
      if (em > -100 && (!ev_set || em + ev > 13 || em + ev < 4)) {
        ev = 9 - em;
        ev_set = true;
      }
      return pow2i(ev);
    };
    const BadRows bad_rows{row_bad, &any_bad, vis0, row0, G};
    fetch(0);
    fetch(1);
#pragma unroll 1
    for (int i = 0; i < N; ++i) {
      const int t = t_lo + i;
      fetch(i + 2);
      cp_async_wait<2>();
      __syncwarp();
      if (keys) {
        if (i >= 2 && !__all_sync(0xffffffffu, mbar_wait(bar_kfree + 8 * (i & 1), ((i >> 1) - 1) & 1, &dead_sm))) break;
      } else {
        if (i >= 3 && !__all_sync(0xffffffffu, mbar_wait(bar_vfree + 8 * (i % 3), (i / 3 - 1) & 1, &dead_sm))) break;
      }
      if (keys) {
        const uint32_t src = raw + (i % C_STAGES) * Pl::RAW_K, dst = sm + (i & 1) * 2 * Pl::MAT + 2 * ew * Pl::K_SBO + k_dst;
        if (t < n_pk) {
          const bool exists = t * CT + 16 * ew < p.n_q;  // n_q % 32 == 0: the 16 tokens exist or do not together
          float s[4], z[4], mx = 0.f;
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int d = 4 * k_q + j;
            const uint32_t a = src + Pl::RAW_KC + 2 * ((d % 32) * (D / 32) + d / 32);
            s[j] = exists ? f16_to_f(lds16(a)) : 0.f;
            z[j] = exists ? f16_to_f(lds16(a + 2 * D)) : 0.f;
            mx = fmaxf(mx, fmaf((float)((1 << BK) - 1), s[j], fabsf(z[j])));
          }
          mx = __uint_as_float(redux_max_u32(__float_as_uint(mx)));
          const int e = key_exponent(mx);
          if (lane == 0) k_unit[i & 7][ew >> 1] = pow2i(-e);  // (two warps of a group write the same)
          const float f = pow2i(e);
          Table tab[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) tab[j] = make_table(s[j] * f, z[j] * f);
          constexpr int QW = 8 / BK;  // channel quads of a word
          const int word = k_q / QW, sh = BK * (k_q % QW);
          const uint32_t wsrc = src + (Pl::KROW == 32 ? (word >> 2) * 256 + (word & 3) * 4 : word * 4);
          constexpr int RS = Pl::KROW < 16 ? Pl::KROW : 16;
#pragma unroll 1
          for (int k = 0; k < KB; ++k) {
            const int blk = KB == 2 ? k : k_b;
            uint32_t w[8];
#pragma unroll
            for (int x = 0; x < 8; ++x) w[x] = lds32(wsrc + (8 * blk + x) * RS);
            expand_block<BK>(w, sh, tab, dst + blk * Pl::K_SBO, Pl::MAT);
          }
        } else {
          // a window tile: 16-bit rows as they are, split into pairs (exact for inputs of ordinary magnitude)
          const int w0 = (t - pk_tiles) * CT;
          const uint2* rows = reinterpret_cast<const uint2*>(p.L.win_k + (size_t)bh * dm.R * D) + k_q;
          const int r0 = w0 + 32 * (ew >> 1);
          uint32_t mp = 0u;
#pragma unroll 1
          for (int x = k_b; x < 32; x += 128 / D) {  // the unit is that of 32 tokens, and of their finite elements
            const uint2 v = r0 + x < p.r ? rows[(size_t)(r0 + x) * (D / 4)] : make_uint2(0u, 0u);
            mp = max_pair(max_pair(mp, v.x), v.y);
          }
          mp = redux_pair(mp);
          const bool bad = mp >= inf16(p.f16);
          if (bad) {
            mp = finite_key_max(rows, r0, k_b, 128 / D, p.r, D / 4, inf16(p.f16));
          }
          const int e = key_exponent(io_to_f(mp, p.f16));
          if (lane == 0) k_unit[i & 7][ew >> 1] = pow2i(-e);
          const float f = pow2i(e);
#pragma unroll 1
          for (int k = 0; k < KB; ++k) {
            const int blk = KB == 2 ? k : k_b, r1 = w0 + 16 * ew + 8 * blk;
            float v[4][8];
#pragma unroll
            for (int x = 0; x < 8; ++x) {
              const uint2 u = r1 + x < p.r ? rows[(size_t)(r1 + x) * (D / 4)] : make_uint2(0u, 0u);
              v[0][x] = io_to_f(u.x & 0xffffu, p.f16) * f; v[1][x] = io_to_f(u.x >> 16, p.f16) * f;
              v[2][x] = io_to_f(u.y & 0xffffu, p.f16) * f; v[3][x] = io_to_f(u.y >> 16, p.f16) * f;
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) store_row(v[j], dst + blk * Pl::K_SBO + 16 * j, Pl::MAT, bad);
          }
        }
      } else {
        const uint32_t src = raw + (i % C_STAGES) * Pl::RAW_V;
        const uint32_t dst = sm + Pl::OFF_V + (i % 3) * 2 * Pl::MAT + (c0 + v_h * (DQ / 2)) / 8 * Pl::V_SBO + v_dst;
        if (t < n_pk) {
          const bool exists = t * CT + 4 * v_q < p.n_q;
          float s[4], z[4];
          uint32_t mb = 0u;
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const uint32_t a = src + Pl::RAW_VC + v_q * Pl::V_QUAD + j * 4 * NG + 2 * (c0 / GS);
            s[j] = exists ? f16_to_f(lds16(a)) : 0.f;
            z[j] = exists ? f16_to_f(lds16(a + 2 * NG)) : 0.f;
            mb = max(mb, abs_bits(fmaf((float)((1 << BV) - 1), s[j], fabsf(z[j]))));
          }
          mb = redux_max_u32(mb);
          if (mb >= INF32) {
            uint32_t tokens = 0u;
            mb = 0u;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const uint32_t b = abs_bits(fmaf((float)((1 << BV) - 1), s[j], fabsf(z[j])));
              tokens |= (uint32_t)(b >= INF32) << j;
              mb = max(mb, b < INF32 ? b : 0u);
              if (b >= INF32) s[j] = z[j] = 0.f;
            }
#pragma unroll 1
            for (int j = 0; j < 4; ++j)
              mark_rows(bad_rows, t * CT + 4 * v_q + j, ew & 3, (tokens >> j) & 1u ? ((1u << (DQ / 2)) - 1u) << (v_h * (DQ / 2)) : 0u);
            mb = redux_max_u32(mb);
          }
          const float f = value_exponent(mb);
          if (lane == 0) v_exp[i & 3][ew & 3] = ev;
          Table tab[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) tab[j] = make_table(s[j] * f, z[j] * f);
          constexpr int QW = 8 / BV, RS = 8 * BV;  // token quads of a word; bytes of a channel
          const uint32_t wsrc = src + v_h * (DQ / 2) * RS + v_q / QW * 4;
          const int sh = BV * (v_q % QW);
#pragma unroll 1
          for (int k = 0; k < KB; ++k) {
            uint32_t w[8];
#pragma unroll
            for (int x = 0; x < 8; ++x) w[x] = lds32(wsrc + (8 * k + x) * RS);
            expand_block<BV>(w, sh, tab, dst + k * Pl::V_SBO, Pl::MAT);
          }
        } else {
          const int w0 = (t - pk_tiles) * CT;
          const uint4* rows = reinterpret_cast<const uint4*>(p.L.win_v + (size_t)bh * dm.R * D);
          auto piece = [&](int tok, int c) {  // 8 channels of a window row
            return w0 + tok < p.r ? rows[(size_t)(w0 + tok) * (D / 8) + c / 8] : make_uint4(0u, 0u, 0u, 0u);
          };
          uint32_t mp = 0u;
#pragma unroll 1
          for (int x = 0; x < 4 * KB; ++x) {
            const uint4 u = piece(4 * v_q + (x & 3), c0 + v_h * (DQ / 2) + 8 * (x >> 2));
            mp = max_pair(max_pair(max_pair(max_pair(mp, u.x), u.y), u.z), u.w);
          }
          mp = redux_pair(mp);
          const bool bad = mp >= inf16(p.f16);
          if (bad) {
            mp = 0u;
#pragma unroll 1
            for (int x = 0; x < 4 * KB; ++x) {
              const uint4 u = piece(4 * v_q + (x & 3), c0 + v_h * (DQ / 2) + 8 * (x >> 2));
              const uint32_t y[4] = {u.x, u.y, u.z, u.w};
              uint32_t mask = 0u;
#pragma unroll
              for (int c = 0; c < 4; ++c) {
                mask |= (uint32_t)((y[c] & 0x7fffu) >= inf16(p.f16)) << (2 * c);
                mask |= (uint32_t)(((y[c] >> 16) & 0x7fffu) >= inf16(p.f16)) << (2 * c + 1);
                mp = max_pair(mp, finite_pair(y[c], inf16(p.f16)));
              }
              mark_rows(bad_rows, p.n_q + w0 + 4 * v_q + (x & 3), ew & 3, mask << (v_h * (DQ / 2) + 8 * (x >> 2)));
            }
            mp = redux_pair(mp);
          }
          const float f = value_exponent(__float_as_uint(io_to_f(mp, p.f16)));
          if (lane == 0) v_exp[i & 3][ew & 3] = ev;
#pragma unroll 1
          for (int x = 0; x < 4 * KB; ++x) {
            const int j = x & 3, k = x >> 2;
            const uint4 u = piece(4 * v_q + j, c0 + v_h * (DQ / 2) + 8 * k);
            uint32_t y[4] = {u.x, u.y, u.z, u.w};
            if (bad) {
#pragma unroll
              for (int c = 0; c < 4; ++c) y[c] = finite_pair(y[c], inf16(p.f16));
            }
            float v[8];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              v[2 * c] = io_to_f(y[c] & 0xffffu, p.f16) * f;
              v[2 * c + 1] = io_to_f(y[c] >> 16, p.f16) * f;
            }
            store_row(v, dst + k * Pl::V_SBO + 16 * j, Pl::MAT, false);
          }
        }
      }
      proxy_fence();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(keys ? bar_kfull + 8 * (i & 1) : bar_vfull + 8 * (i % 3));
        if (keys) mbar_arrive(bar_unit + 8 * (i & 7));
      }
    }
    cp_async_wait_all();
  }

  // ---- the row tile's result, or its partial: row r's state in split s at (tile * 128 + r) * ns + s ----
  tc_fence_before();
  __syncthreads();
  const size_t part0 = ((size_t)rt * n_streams + bh) * CM;
  auto out_row = [&](int r) {
    const int row = row0 + r, j = row / G, h = row - j * G;
    return ((size_t)j * dm.B + b) * dm.Hq + hk * G + h;
  };
  if (warp < 8) {
    const bool ok = N == 0 || mbar_wait(bar_o + 8 * ((N - 1) & 3), ((N - 1) >> 2) & 1, &dead_sm);
    if (__all_sync(0xffffffffu, ok) && dead_sm == 0) {
      tc_fence_after();
      const int w = warp >> 2, r = tid & 127;
      const float M = m_sm[r], M0 = ml_sm[0][r], M1 = ml_sm[1][r];
      const float L = l_sm[0][r] * (M0 == M ? 1.f : ex2(M0 - M)) + l_sm[1][r] * (M1 == M ? 1.f : ex2(M1 - M));
      const float inv = p.ns == 1 ? 1.f / L : 1.f;
#pragma unroll 1
      for (int h = 0; h < D / 64; ++h) {
        const int cb = w * (D / 2) + 32 * h;
        uint32_t o[32];
        if (N > 0) {
          tmem_ld<32>(row_t + Pl::COL_O + cb, o);
          tc_wait_ld();
          if constexpr (Pl::FLUSH != 0) {
            uint32_t sum[32];
            tmem_ld<32>(row_t + Pl::COL_T + cb, sum);
            tc_wait_ld();
#pragma unroll
            for (int k = 0; k < 32; ++k) o[k] = __float_as_uint(__uint_as_float(o[k]) + __uint_as_float(sum[k]));
          }
        }
        float f[2];  // of the two channel quarters that 32 channels can span
        f[0] = (N > 0 ? pow2i(-v_exp[(N - 1) & 3][cb / DQ]) : 0.f) * inv;
        f[1] = (N > 0 ? pow2i(-v_exp[(N - 1) & 3][(cb + 31) / DQ]) : 0.f) * inv;
        float v[32];
#pragma unroll
        for (int k = 0; k < 32; ++k) v[k] = N > 0 ? __uint_as_float(o[k]) * f[k / 16] : 0.f;
        if (any_bad != 0) {
          const uint32_t ba = row_bad[r][cb / DQ], bz = row_bad[r][(cb + 31) / DQ];
#pragma unroll
          for (int k = 0; k < 32; ++k)
            if (((k < 16 ? ba : bz) >> ((cb + k) % DQ)) & 1u) v[k] = CUDART_NAN_F;
        }
        if (r < n_rows) {
          if (p.ns > 1) {
            float4* dst = reinterpret_cast<float4*>(p.part_acc + ((part0 + r) * p.ns + split) * D + cb);
#pragma unroll
            for (int k = 0; k < 8; ++k) dst[k] = make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
          } else if (p.out_f32) {
            float4* dst = reinterpret_cast<float4*>(reinterpret_cast<float*>(p.out) + out_row(r) * D + cb);
#pragma unroll
            for (int k = 0; k < 8; ++k) dst[k] = make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
          } else {
            uint32_t x[16];
#pragma unroll
            for (int k = 0; k < 16; ++k)
              x[k] = p.f16 ? pack_io2<true>(v[2 * k], v[2 * k + 1]) : pack_io2<false>(v[2 * k], v[2 * k + 1]);
            uint4* dst = reinterpret_cast<uint4*>(reinterpret_cast<uint16_t*>(p.out) + out_row(r) * D + cb);
#pragma unroll
            for (int k = 0; k < 4; ++k) dst[k] = make_uint4(x[4 * k], x[4 * k + 1], x[4 * k + 2], x[4 * k + 3]);
          }
        }
      }
      if (p.ns > 1 && w == 0 && r < n_rows)
        *reinterpret_cast<float2*>(p.part_ml + ((part0 + r) * p.ns + split) * 2) = make_float2(M, L);
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 8 + C_EXPAND)
    tmem_dealloc(tbase, 512u);
  if (dead_sm != 0) {
    if (tid == 0) atomicExch(p.status, 1);
    return;
  }
  if (p.ns == 1) return;
  // the last CTA of the row tile merges (ticket as in the decode kernel)
  unsigned* ticket = p.tickets + (size_t)rt * n_streams + bh;
  if (tid == 0) {
    unsigned t;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;\n" : "=r"(t) : "l"(ticket) : "memory");
    s_flag = (t == (unsigned)(p.ns - 1));
  }
  __syncthreads();
  if (!s_flag) return;
  for (int i = tid; i < n_rows * (D / 2); i += C_THREADS) {
    const int r = i / (D / 2), d = 2 * (i % (D / 2));
    const float* pa = p.part_acc + (part0 + r) * p.ns * D + d;
    const float* ml = p.part_ml + (part0 + r) * p.ns * 2;
    float Mx = -CUDART_INF_F;
#pragma unroll 4
    for (int s = 0; s < p.ns; ++s) Mx = fmaxf(Mx, ld_cg(ml + 2 * s));
    float ax = 0.f, ay = 0.f, Ls = 0.f;
#pragma unroll 4
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

template <int D, int BK, int BV, int GS>
cudaError_t chunk_launch_one(const ChunkParams& p, cudaStream_t st) {
  using Pl = ChunkPlan<D, BK, BV, GS>;
  auto kernel = chunk_kernel<D, BK, BV, GS>;
  const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, Pl::TOTAL);
  if (e != cudaSuccess) return e;
  return launch_dependent(kernel, dim3((unsigned)p.row_tiles * p.dm.B * p.dm.Hkv * p.ns), dim3(C_THREADS), (size_t)Pl::TOTAL, st, p);
}

}  // namespace

template <int D>
cudaError_t launch_chunk_t(const ChunkParams& p, cudaStream_t st) {
  switch (p.L.bk * 100 + p.L.bv * 10 + (p.dm.g == 64)) {
    case 220: return chunk_launch_one<D, 2, 2, 32>(p, st);
    case 221: return chunk_launch_one<D, 2, 2, 64>(p, st);
    case 210: return chunk_launch_one<D, 2, 1, 32>(p, st);
    case 211: return chunk_launch_one<D, 2, 1, 64>(p, st);
    case 120: return chunk_launch_one<D, 1, 2, 32>(p, st);
    case 121: return chunk_launch_one<D, 1, 2, 64>(p, st);
    case 110: return chunk_launch_one<D, 1, 1, 32>(p, st);
    case 111: return chunk_launch_one<D, 1, 1, 64>(p, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace xq
