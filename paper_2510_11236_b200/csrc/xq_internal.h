// Internal declarations shared by the host state machine and the kernel files.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace xq {

struct Dims {
  int B, Hq, Hkv, G, D, g, R, NG;
  int nq_cap;  // capacity of the quantized region in tokens, padded to whole 128-token batches
};

// Device addresses of one layer's regions (codes: of the layer that owns them).
struct LayerPtrs {
  uint16_t* win_k;   // [B,Hkv,R,D] bf16
  uint16_t* win_v;
  uint16_t* k_meta;  // [B,Hkv,nq_cap/g,2,D] fp16 (per token group: scales, then zero-points)
  uint16_t* v_meta;  // [B,Hkv,nq_cap,2,NG] fp16 (per token: scales, then zero-points)
  uint32_t* k_codes; // [B,Hkv,nq_cap*D*bk/32]
  uint32_t* v_codes;
  int bk, bv;
};

// One layer of a quantize-and-pack launch.
struct PackLayer {
  LayerPtrs L;
  const uint16_t* K_in;  // [B,Hkv,n_in,D] new tokens (absolute positions s_old ..)
  const uint16_t* V_in;
  // codes of a cache kind: 0 = none (the layer keeps scale and zero-point only), 1 = written, 2 = merged into the
  // codes the dominant layer wrote (weighted average, Appendix F); 4 = computed for the statistic only; 6 = both
  int own_k, own_v;
  float eta_k, eta_v;
  // with bit 2 set in own_*: count the elements by |own code - stored code| into these four counters (before the
  // codes are merged, if they are)
  unsigned long long* delta_k;
  unsigned long long* delta_v;
};

constexpr int PACK_MAX_LAYERS = 32;  // layers one launch can take (they share every length below)

struct PackCommon {
  Dims dm;
  int n_layers;
  int n_in;
  int s_old;     // tokens cached before this append
  int nq_old;    // quantized tokens before this append
  int n_blocks;  // R-token blocks to quantize, starting at absolute token nq_old
  int f16;       // inputs and window are IEEE half precision (else bfloat16)
  // tokens nq_new .. s_new - 1 of the input go into window rows 0 .. win_count - 1 (the warps that read those rows
  // of the old window copy them); 0: the caller copies
  int win_count;
  int nq_new;
  // merged code of (e0, e1) at bits 2 * (4 e0 + e1), for 1-bit and 2-bit codes
  uint32_t merge_lut[2];
};
// Kernel parameters for at most N layers.  A launch costs the host time for every byte of them: an append of one layer
// takes 4.9 us of host time with room for one layer and 7.9 us with room for 32.
template <int N>
struct PackParamsOf : PackCommon {
  PackLayer layer[N];
};
using PackParams = PackParamsOf<PACK_MAX_LAYERS>;

struct WindowParams {
  Dims dm;
  LayerPtrs L;
  const uint16_t* K_in;
  const uint16_t* V_in;
  int n_in;
  int s_old;
  int first;   // first absolute token to copy
  int count;   // tokens to copy
  int nq_new;  // window slot = absolute token - nq_new
};

// One layer of a decode launch.
struct DecodeLayer {
  LayerPtrs L;
  const uint16_t* q;  // [B,Hq,D] bf16
  void* out;          // [B,Hq,D] bf16 or f32
  // Fused append of one token per stream (tensor-core kernel only; else null): the newest window row, index r - 1, is
  // not in the window yet but here, [B,Hkv,D] bf16.  The CTA whose share of the window holds that row reads it from
  // here and stores it into the window.
  const uint16_t* K_new;
  const uint16_t* V_new;
};

constexpr int DECODE_MAX_LAYERS = 32;  // layers one launch can take (of equal lengths and bit-widths)

struct DecodeParams {
  Dims dm;
  int n_layers;       // the scalar kernel takes one
  int paired;         // tensor-core kernel: a CTA takes layers 2 y and 2 y + 1, which read the same codes
  int many;           // tensor-core kernel, head_dim 128, up to four heads, not paired: the variant for many CTAs
  int n_q;            // quantized tokens
  int r;              // window tokens
  int ns_q, ns_w;     // splits over the quantized region (most of any stream) / over the window
  int deal;           // tensor-core kernel: batches of 128 tokens are dealt to the splits in runs of this many
  float scale;
  float* part_acc;    // [n_layers,B,Hq,ns,D]
  float* part_ml;     // [n_layers,B,Hq,ns,2]  (running max in log2 units, sum)
  // used by kernels that merge the partials themselves (last CTA of a stream):
  int out_f32;
  unsigned int* tickets;  // [n_layers,B*Hkv], zero between launches
  // 1: the packed streams were complete before the preceding kernel in the stream started, so their first
  // copies may be issued before this kernel has waited for that kernel (programmatic dependent launch)
  int early_fetch;
  // 1: the preceding kernel in the stream is a decode launch of the same call that itself started only after all
  // earlier work in the stream had completed, so nothing this launch reads is still being written: it reads at
  // once and waits for that launch only before its first write that the launch could see (partials, tickets,
  // result, status).  Implies early_fetch.
  int late_wait;
  int* status;  // device word the tensor-core kernel sets when one of its bounded waits gave up
  int f16;      // q, the window and the 16-bit output are IEEE half precision (else bfloat16)
  DecodeLayer layer[DECODE_MAX_LAYERS];
};

constexpr int CHUNK_ROWS = 128;  // query rows of a chunk CTA

// Attention of a chunk of query tokens (xq_chunk.cuh).
struct ChunkParams {
  Dims dm;
  LayerPtrs L;
  const uint16_t* q;  // [T,B,Hq,D]
  void* out;          // [T,B,Hq,D] bf16 or f32
  int n_q, r;         // quantized tokens, window tokens
  int S, T;           // tokens of the layer; query token j sees the first S - T + j + 1 of them
  int row_tiles;      // per (sequence, kv head): T * G rows over CHUNK_ROWS
  int ns;             // splits of a row tile's tokens
  float scale;
  float* part_acc;    // [row_tiles,B*Hkv,rows,ns,D] (ns > 1)
  float* part_ml;     // [row_tiles,B*Hkv,rows,ns,2]
  unsigned int* tickets;  // [row_tiles,B*Hkv], zero between launches
  int* status;        // device word that is set when a bounded wait gave up
  int out_f32, f16;
};

struct MergeParams {
  Dims dm;
  int ns;
  int f16;
  const float* part_acc;
  const float* part_ml;
  void* out;
  int out_f32;
};

// Part `part` of `parts` nearly equal shares of n items: [lo, hi), sizes differ by at most one.
// (32-bit arithmetic: a 64-bit division costs a device thread hundreds of instructions.)
__host__ __device__ inline void share_of(int n, int parts, int part, int& lo, int& hi) {
  const unsigned base = (unsigned)n / (unsigned)parts, rem = (unsigned)n - base * (unsigned)parts;
  lo = (int)((unsigned)part * base + ((unsigned)part < rem ? (unsigned)part : rem));
  hi = lo + (int)base + ((unsigned)part < rem ? 1 : 0);
}

// Programmatic dependent launch (sm_90 and later).  A kernel launched with launch_dependent() may start while
// the preceding kernel in the stream is still running, provided that kernel has called grid_dependents_go() (or
// when it ends); it must call grid_dependency_wait() before it touches anything the preceding kernels wrote or
// still read.  After the wait all earlier work in the stream is complete and visible, as at a kernel boundary.
#ifdef __CUDACC__
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
__device__ __forceinline__ void grid_dependents_go() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }

template <typename P>
cudaError_t launch_dependent(void (*kernel)(P), dim3 grid, dim3 block, size_t smem, cudaStream_t st, const P& params) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, params);
}
#endif

cudaError_t launch_pack(const PackParams& p, cudaStream_t st);
cudaError_t launch_window_append(const WindowParams& p, cudaStream_t st);
cudaError_t launch_decode_generic(const DecodeParams& p, cudaStream_t st);
// Tensor-core decode kernels.  head_dim 128: for HP (1, 2, 4, 8) query heads per kv head, of one layer or of NL = 2 that
// read the same codes (up to four heads), MANY: of one layer of up to four, for launches of many CTAs; head_dim 64: HP (1, 2, 4) heads, or NT = 2 sets of four.  decode_mma_shape_t
// also prepares the kernel for the current device: it comes before the first launch of a handle.
struct MmaShape {
  int warps;   // warps of a CTA
  bool ready;  // the kernel can be launched with its shared memory on this device
};
template <int HP, int NL, bool MANY>
cudaError_t launch_decode_mma_t(const DecodeParams& p, cudaStream_t st);
template <int HP, int NL, bool MANY>
MmaShape decode_mma_shape_t(int g, int bk, int bv);
template <int HP, int NT>
cudaError_t launch_decode_mma64_t(const DecodeParams& p, cudaStream_t st);
template <int HP, int NT>
MmaShape decode_mma64_shape_t(int g, int bk, int bv);
template <int D>
cudaError_t launch_chunk_t(const ChunkParams& p, cudaStream_t st);
cudaError_t launch_merge(const MergeParams& p, cudaStream_t st);

}  // namespace xq
