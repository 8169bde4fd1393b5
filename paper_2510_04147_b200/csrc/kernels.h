// Internal launcher declarations shared by the translation units of the library.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include <atomic>

#include "routes.h"

typedef __nv_bfloat16 bf16;

namespace ssd {

// Two floats in a register pair, worked on by one instruction (each half rounded as by the scalar form)
__device__ __forceinline__ uint64_t pair_f32(float x, float y) {
  uint64_t p;
  asm("mov.b64 %0, {%1, %2};" : "=l"(p) : "f"(x), "f"(y));
  return p;
}
__device__ __forceinline__ void unpair_f32(uint64_t p, float& x, float& y) { asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(p)); }
__device__ __forceinline__ uint64_t mul_f32x2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t fma_f32x2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}

// a = silu(g) * u, for two elements.  The quotient is g times the approximate reciprocal with one residual correction
// (Markstein's theorem: the correctly rounded quotient but for rare cases in the last place).  Without the division operator's
// branch the elements of an epilogue overlap: 32 of them took 3700 clocks of a thread, two warps to a scheduler.  Gate/up of d
// 4096, ffn 12288 41.8 -> 40.9 us at 128 rows, 76.4 -> 69.3 at 512, 101 -> 99 at 768.
// The values of `/` over all g: the reciprocal is taken of a sixteenth of the denominator, because 1 / (1 + e^-g) is subnormal
// from g = -87.4 down and the instruction flushes those to zero; where the residual is not finite (g infinite, or a
// denominator past the largest float), the uncorrected quotient is g or 0 already.  Element by element these three more
// operations cost eight sequences of 32 rows 2 % of a generation (281.8 -> 288.2 ms); in pairs gate/up takes as long as without
// them (35.3 / 35.3 us at 64 rows, 53.6 / 54.0 at 256, 82.8 / 81.3 at 512).
__device__ __forceinline__ void swiglu2(float g0, float g1, float u0, float u1, float& a0, float& a1) {
  const uint64_t g = pair_f32(g0, g1), minus1 = pair_f32(-1.f, -1.f);
  const uint64_t nd = fma_f32x2(pair_f32(expf(-g0), expf(-g1)), minus1, minus1);        // -(1 + e^-g)
  float d0, d1, r0, r1, e0, e1, q0, q1, v0, v1;
  unpair_f32(mul_f32x2(nd, pair_f32(-0x1p-4f, -0x1p-4f)), d0, d1);
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r0) : "f"(d0));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r1) : "f"(d1));
  const uint64_t r = mul_f32x2(pair_f32(r0, r1), pair_f32(0x1p-4f, 0x1p-4f)), q = mul_f32x2(g, r), rest = fma_f32x2(q, nd, g);
  unpair_f32(rest, e0, e1);
  unpair_f32(q, q0, q1);
  unpair_f32(fma_f32x2(rest, r, q), v0, v1);
  v0 = fabsf(e0) <= 3.402823466e38f ? v0 : q0;
  v1 = fabsf(e1) <= 3.402823466e38f ? v1 : q1;
  unpair_f32(mul_f32x2(pair_f32(v0, v1), pair_f32(u0, u1)), a0, a1);
}

// ---------------------------------------------------------------- programmatic dependent launch
// Every kernel of the forward is launched with the "programmatic stream serialization" attribute:
// it may become resident while its predecessor in the stream still runs.  A kernel first lets ITS
// successor be scheduled (pdl_launch_dependents), does whatever does not depend on earlier kernels
// (barrier set-up, weight prefetch), and calls pdl_wait() before it touches anything an earlier
// kernel wrote or still reads.  pdl_wait() returns once the predecessor grid has completed and its
// memory operations are visible, so completion is transitive along the stream.
#ifdef __CUDACC__
// rotary embedding of the pair (x1, x2) = features (i, i + hd/2), with the roundings spelled out: the kernels that rotate
// agree to the bit
__device__ __forceinline__ void rope_pair(float& x1, float& x2, float c, float s) {
  const float a = x1, b = x2;
  x1 = __fmaf_rn(a, c, -__fmul_rn(b, s));
  x2 = __fmaf_rn(b, c, __fmul_rn(a, s));
}
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Error and result words that the host reads live in page-locked host memory, mapped into the device: a kernel's plain
// store is there once the stream has been synchronised, with no clearing or copying operation on the stream.
__device__ __forceinline__ void raise_word(int* word, int value) { *reinterpret_cast<volatile int*>(word) = value; }

// A cluster dimension > 1 additionally groups that many consecutive CTAs along x (or y) into a
// thread-block cluster.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl_cluster_xy(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                                         unsigned cluster_x, unsigned cluster_y, bool early, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  cfg.numAttrs = 0;
  if (early) {           // off: a plain launch behind whatever the caller's stream holds
    attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[cfg.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (cluster_x > 1 || cluster_y > 1) {
    attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
    attr[cfg.numAttrs].val.clusterDim.x = cluster_x;
    attr[cfg.numAttrs].val.clusterDim.y = cluster_y;
    attr[cfg.numAttrs++].val.clusterDim.z = 1;
  }
  cfg.attrs = attr;
  return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl_cluster(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                                      unsigned cluster_x, Args... args) {
  return launch_pdl_cluster_xy(kernel, grid, block, smem, st, cluster_x, 1u, true, args...);
}
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                              Args... args) {
  return launch_pdl_cluster_xy(kernel, grid, block, smem, st, 1u, 1u, true, args...);
}
#endif

// ---------------------------------------------------------------- per-device set-up
// Function attributes (the opt-in to large dynamic shared memory) belong to a device, not to the
// process: launchers keep one flag per device ordinal and set the attribute on a device's first use, which threads with a
// context each may reach together (then each of them sets it).
constexpr int kMaxDevices = 64;
template <typename T>
using PerDevice = std::atomic<T>[kMaxDevices];
inline int device_slot() {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return -1;
  return dev;
}

// ---------------------------------------------------------------- layout helpers (host+device)
// Rows of a forward are ordered [sequence slot a][node i][in-block index t].
struct RowMap {
  int rows_per_seq;    // n_nodes * T
  int T;               // rows per node (block tokens, or prompt length for prefill)
  int pos0;            // absolute position of t = 0 (= cached prefix length S)
  int seq_base;        // sequence id of slot 0 when seq_map == nullptr
  const int* seq_map;  // device [slots] slot -> sequence id, or nullptr (identity + seq_base)
  // The same map by value when the host knows it and it is short: a kernel may then use it before
  // its dependency wait (the device array is written by an earlier kernel of the same forward).
  int n_inline;        // 0: not given
  int inline_seq[8];
  // > 0: the rows of a sequence are ONE causal chain of two blocks - the first chain_T0 rows are a
  // finished block (they see the prefix and themselves, and their K/V go to the cache), the rest
  // is the next block, which also sees the finished one.  rows_per_seq == T then.
  int chain_T0;
};
__host__ __device__ inline int seq_of_slot(const RowMap& m, int slot) {
  if (m.n_inline > 0) return m.inline_seq[slot];
  return m.seq_map ? m.seq_map[slot] : m.seq_base + slot;
}

// ---------------------------------------------------------------- weight repacking
// dst[(j / group) * group_stride + group_offset + j % group][c] = bf16(src[j][c]),  j < rows, c < cols
void launch_convert_rows(cudaStream_t st, const void* src, int src_is_f32, bf16* dst, int rows, int cols,
                         int dst_pitch, int group, int group_stride, int group_offset);
// same row mapping, but dst is tile-contiguous: element (n, k) of the mapped matrix lives at
// (((n / 128) * kb_total + k / 64) * 128 + n % 128) * 64 + k % 64, kb_total = ceil(cols_padded / 64)
void launch_convert_tiled(cudaStream_t st, const void* src, int src_is_f32, bf16* dst, int rows, int cols,
                          int kb_total, int group, int group_stride, int group_offset);
inline size_t tiled_elems(int n, int k) { return (size_t)((n + 127) / 128) * ((k + 63) / 64) * 128 * 64; }
void launch_copy_f32(cudaStream_t st, const void* src, int src_is_f32, float* dst, int n);

// ---------------------------------------------------------------- elementwise / reductions
// producer side of the fused RMSNorm: h[r] = embed[ids[r]]; hb[r] = bf16(h[r] * gain);
// sq[r * sq_stride] = sum of squares of h[r]
// (ids outside [0, V) read row 0: the table is never indexed out of range)
void launch_embed_prep(cudaStream_t st, const int* ids, const bf16* embed, const float* gain, float* h, bf16* hb,
                       float* sq, int sq_stride, int R, int d, int V);
// the same producer step for a residual stream already in h: hb[r] = bf16(h[r] * gain), sq as above
void launch_stream_prep(cudaStream_t st, const float* h, const float* gain, bf16* hb, float* sq, int sq_stride, int R,
                        int d);
// sums the split-K partials of the fused QKV projection in split order, rotates q and k, writes bf16 (head dimension 64 or 128)
struct QkvOut;
void launch_qkv_finish(cudaStream_t st, const float* partial, int splits, size_t split_stride, int R, const QkvOut& o);
// per row: argmax / max-softmax-probability over the vocabulary with mask_id excluded
void launch_lm_stats_from_logits(cudaStream_t st, const float* logits, int R, int V, int mask_id,
                                 const uint8_t* row_wanted, int* tok, float* conf);
// merge per-tile (max, sumexp, argmax) in tile order; the token is always inside [0, V)
void launch_lm_merge(cudaStream_t st, const float* tile_max, const float* tile_sum, const int* tile_arg,
                     int tiles, int R, int V, const uint8_t* row_wanted, int* tok, float* conf);

// the k most probable tokens per row from the per-tile candidate lists (merged in tile order, lower index
// first among equals): topk_tok [R][kLmTopKMax], topk_prob likewise = exp(logit - max) * conf[row]
void launch_lm_merge_topk(cudaStream_t st, const float* tile_topv, const int* tile_topi, int tiles, int R, int V, int k,
                          const uint8_t* row_wanted, const float* conf, int* topk_tok, float* topk_prob);

// ---------------------------------------------------------------- attention
struct AttnArgs {
  // mma.sync verification form: Q and the node-local K/V come straight from the fp32 split-K partials
  // of the fused q|k|v projection ([splits][R][(H + 2 Hkv) * hd]) and are rotated in the prologue
  const float* qkv_partial;
  int qkv_splits;
  size_t qkv_split_stride;
  const float2* rope;         // [max_seq][hd/2] (cos, sin)
  // block commit through the verification form (one node per sequence, rows_per_seq == T): the
  // rotated K and the V of the rows are also written to the cache at their absolute positions
  bf16* cache_k_out;          // layer base like cache_k, or nullptr
  bf16* cache_v_out;
  int* err_flag;              // word set non-zero when a bounded wait expires (tcgen05 form)
  const bf16* q;        // [R][H][hd], rotated
  const bf16* cache_k;  // layer base: [seq][Hkv][max_seq][hd]
  const bf16* cache_v;
  const bf16* local_k;  // [R][Hkv][hd] or nullptr (no node-local keys)
  const bf16* local_v;
  float* part_o;        // [n_parts][R][H][hd]
  float2* part_ml;      // [n_parts][R][H]  (running max in log2 domain, sum)
  bf16* out;            // [R][H*hd]
  int R, H, Hkv, hd;
  int S;                // keys read from the cache
  // Dual cache: the cached keys are the positions [0, hole_begin) and [hole_begin + hole_len, ...), i.e. key
  // index k >= hole_begin lives in cache row k + hole_len (the rows of the block being computed are skipped:
  // its own keys are the node-local ones).  hole_len = 0: the cached keys are the prefix [0, S).
  int hole_begin, hole_len;
  int kv_split;         // prefix keys per split (a function of S only)
  size_t cache_seq_stride;
  size_t cache_rows;                      // rows of hd elements in one layer's K (or V) cache: max_batch * Hkv * max_seq; 0: unknown
  size_t kv_pos_stride, kv_head_stride;   // element (sequence, position, kv head) of the cache lies at
                                          // seq * cache_seq_stride + head * kv_head_stride + pos * kv_pos_stride
  RowMap map;
  int n_seq_slots;
};
// cache-fill form for head dimension 64
void launch_attention(cudaStream_t st, const AttnArgs& a);
// The cache-fill form on the tcgen05 tensor cores (head dimension 128): reads a.q and the cache, writes a.out; slots are
// consecutive sequences from map.seq_base.  Returns 0 or a negative ssd error code.
int launch_attention_fill_tc(cudaStream_t st, const AttnArgs& a);
// Verification-forward form: one kernel; rotary embedding, node-local K/V and the merge of the
// key parts (through a thread-block cluster) inside.  Needs prefix parts + 1 <= kAttnMaxClusterParts.
// Returns 0 or a negative ssd error code.
int launch_attention_verify(cudaStream_t st, const AttnArgs& a);
// tcgen05 form for head dimension 128 and node widths up to 128: reads a.q, a.local_k / a.local_v ([R][Hkv][hd], rotated) and
// the cache, writes a.out; the key tiles of a (query tile, head, sequence) are split over n_parts CTAs (at most
// kAttnMaxClusterParts, fewer when there are fewer tiles).  Needs a.err_flag.  Returns 0 or a negative ssd error code.
int launch_attention_verify_pipe(cudaStream_t st, const AttnArgs& a, int n_parts);
constexpr int kAttnMaxClusterParts = 8;
constexpr int kAttnTcMaxNode = 128;     // widest node of the tcgen05 form: its local keys are one key tile

// ---------------------------------------------------------------- projections
// EPI_RESIDUAL: the split-K CTAs of a tile form a cluster; they sum their accumulators through
// distributed shared memory in split order, add the residual stream, and write the new stream
// h (fp32), its bf16 copy times the next norm's gain (hb, the next projection's operand) and the
// tile's share of every row's sum of squares.  The RMSNorm itself is then applied by the consumer:
// rmsnorm(h) * g . W^T  ==  inv_rms(row) * ((h * g) . W^T), with inv_rms from the sums of squares.
// EPI_SUM: the same cluster reduction, the sums themselves go to `out` (fp32 [R][N]).
// EPI_QKV (dense kernel only): rotary embedding of q and k, everything rounded to bf16; q rows to their buffer, k and v
// rows to the node-local buffers, the cache or both.
enum { EPI_PARTIAL = 0, EPI_SWIGLU = 1, EPI_LMHEAD = 2, EPI_RESIDUAL = 3, EPI_QKV = 4, EPI_SUM = 5 };
constexpr int kGemmMaxClusterSplits = 8;
constexpr int kLmTopKMax = 8;   // most candidates per row the LM-head epilogue can rank
// Where finished q, k and v rows go (EPI_QKV, launch_qkv_finish).  Row r is sequence-local row r % map.rows_per_seq of slot r / map.rows_per_seq, its
// position map.pos0 + (that % map.T).
struct QkvOut {
  int H, Hkv, hd;
  const float2* rope;     // [max_seq][hd/2] (cos, sin)
  bf16* q;                // [R][H][hd]
  bf16* local_k;          // [R][Hkv][hd], or nullptr
  bf16* local_v;
  bf16* cache_k;          // cache of the layer: the sequence-local rows below `cache_rows` go there (at their positions)
  bf16* cache_v;
  int cache_rows;
  size_t cache_seq_stride, kv_pos_stride, kv_head_stride;
  RowMap map;
};
struct GemmArgs {
  const bf16* x;  // [R][x_pitch] activations (K-major)
  const bf16* w;  // [N][w_pitch] weights (K-major), or the tile-contiguous layout below when w_tiled
  int R, N, K, x_pitch, w_pitch;
  int w_tiled;           // 1: w is [ceil(N/128)][ceil(K/64)][128][64] (one 16 KB block per MMA tile, zero padded)
  int splits;            // split-K factor (EPI_PARTIAL; EPI_RESIDUAL and EPI_SUM: the cluster's size)
  int plain_launch;      // 1: the weights may be what the stream's previous kernel writes - no early start, no prefetch under it
  int two_sm_min_rows;   // tensor-core kernel: pairs of tiles run as one cta_group::2 MMA from this many rows on; 0 = never
  int epi;
  float* out;            // EPI_PARTIAL: [splits][R][N] fp32
  bf16* act;             // EPI_SWIGLU: [R][act_pitch], N/2 features
  int act_pitch;
  float* tile_max;       // EPI_LMHEAD: [tiles][R]
  float* tile_sum;
  int* tile_arg;
  int topk;              // EPI_LMHEAD: 0, or how many of the tile's largest logits per row to write as well (<= kLmTopKMax)
  float* tile_topv;      // [tiles][R][kLmTopKMax] values, descending
  int* tile_topi;        // [tiles][R][kLmTopKMax] vocabulary indices (lower index first among equals)
  int mask_id;
  int* err_flag;         // word set non-zero when a bounded wait expires
  unsigned long long wait_limit_ns;   // bound of every barrier wait in the kernel; 0 = the default (2 s)
  int max_stages;        // tuning: cap on the depth of the shared-memory ring (0: as deep as the budget allows)
  int starve_kb;         // test hook, 0 = off: leave out the copies of K block starve_kb - 1 (plain EPI_PARTIAL launches only)
  // consumer side of a fused RMSNorm: every output row r is multiplied by
  // rsqrt(sum_{t < sq_count} sq[r * sq_stride + t] / norm_dim + norm_eps); sq == nullptr: no scaling
  const float* sq;
  int sq_count, sq_stride, norm_dim;
  float norm_eps;
  // EPI_RESIDUAL: splits = cluster size (<= kGemmMaxClusterSplits)
  int before;            // CTAs of the kernel in front where that is the skinny one with two to an SM, else 0
  const QkvOut* qkv;     // EPI_QKV (host pointer, copied into the launch)
  float* h;              // [R][N] fp32 residual stream, updated in place
  bf16* hb;              // [R][N] bf16(h * gain)
  const float* gain;     // [N]
  float* sq_out;         // [R][sq_out_stride]: slot `tile` of a row receives the tile's sum of squares
  int sq_out_stride;
};
int gemm_tiles(int N);
// Many rows: persistent two-SM kernel, tile-contiguous weights; EPI_QKV, EPI_SWIGLU or EPI_RESIDUAL.  `splits` K ranges are
// summed in order: the bits of the skinny kernel (and launch_qkv_finish) with the same splits.  Returns 0 or a negative
// ssd error code.
int launch_gemm_dense(cudaStream_t st, const GemmArgs& g);
// Up to 256 rows: the features shared out evenly over all SMs, tile-contiguous weights; EPI_QKV (head dimension 128) or
// EPI_SWIGLU.  The same sums as the other kernels with the same splits.  Returns 0 or a negative ssd error code.
int launch_gemm_wave(cudaStream_t st, const GemmArgs& g);
bool gemm_wave_fits(int N, int R, int splits);     // its accumulators have room for the K splits
// tensor-core path (TMA + tcgen05). Returns 0 or a negative ssd error code.
int launch_gemm_tc(cudaStream_t st, const GemmArgs& g);
int gemm_tc_init();   // resolves the driver entry point for tensor-map encoding
// Tensor map (a CUtensorMap, 128 bytes, 64-byte aligned) over a row-major bf16 matrix [rows][cols] with `pitch_elems`
// elements between rows: boxes of 64 columns x box_rows rows, 128-byte swizzle.  Returns 0 or a negative ssd error code.
// ... over [planes][rows][cols] with `row_pitch` / `plane_pitch` elements between rows / planes; rows past `rows` read as zero.
int encode_tmap_bf16_3d(void* map_out, const void* base, uint64_t cols, uint64_t rows, uint64_t planes, uint64_t row_pitch,
                        uint64_t plane_pitch, uint32_t box_rows);
int encode_tmap_bf16_2d(void* map_out, const void* base, uint64_t rows, uint64_t cols, uint64_t pitch_elems, uint32_t box_rows);

#ifdef __CUDACC__
// ---- what the LM head keeps of a vocabulary tile of 128 entries, per row: maximum with the lowest index among equals, sum of
// exp(x - its maximum) and, where asked, the largest entries.  A tile is worked on in quarters of 32 entries, merged (0 + 1) + (2 + 3),
// in every kernel and whoever has the quarters; every rounding is spelled out, so the value depends on the tile alone, not on what a
// compiler contracts where the entries come from a product in registers.
struct LmStat { float m, sum; int arg; };
__device__ __forceinline__ LmStat lm_quarter(const float (&x)[32], int first) {
  LmStat s{-INFINITY, 0.f, 0x7fffffff};
#pragma unroll
  for (int j = 0; j < 32; ++j)
    if (x[j] > s.m) { s.m = x[j]; s.arg = first + j; }
  if (s.m != -INFINITY) {
#pragma unroll
    for (int j = 0; j < 32; ++j) s.sum = __fadd_rn(s.sum, expf(__fsub_rn(x[j], s.m)));    // (exp(-inf) = 0 for dead entries)
  }
  return s;
}
// the same value from both partners: the lower quarter's (maximum, index) wins a tie
__device__ __forceinline__ LmStat lm_merge(const LmStat& lo, const LmStat& hi) {
  LmStat s{fmaxf(lo.m, hi.m), 0.f, hi.m > lo.m ? hi.arg : lo.arg};
  if (lo.m != -INFINITY) s.sum = __fmaf_rn(lo.sum, expf(__fsub_rn(lo.m, s.m)), s.sum);
  if (hi.m != -INFINITY) s.sum = __fmaf_rn(hi.sum, expf(__fsub_rn(hi.m, s.m)), s.sum);
  return s;
}
// sorted lists (value descending, lower index first): an insertion only where an entry beats the last of the list
__device__ __forceinline__ void lm_insert(float (&tv)[kLmTopKMax], int (&ti)[kLmTopKMax], float x, int idx) {
  if (!(x > tv[kLmTopKMax - 1])) return;
#pragma unroll
  for (int r = kLmTopKMax - 1; r > 0; --r) {                 // from the back: what is smaller moves down a place
    const bool below = x > tv[r - 1], here = !below && x > tv[r];
    if (below) { tv[r] = tv[r - 1]; ti[r] = ti[r - 1]; }
    else if (here) { tv[r] = x; ti[r] = idx; }
  }
  if (x > tv[0]) { tv[0] = x; ti[0] = idx; }
}
#endif

// ---------------------------------------------------------------- tree build / acceptance
// Words of BlockState::mirror per sequence, written by the acceptance kernel
enum { MIRROR_REMAINING = 0, MIRROR_REMAINING_NXT, MIRROR_HAS_DRAFTS, MIRROR_LAST_ACCEPT, MIRROR_N_CAND, kMirrorWords };
struct BlockState {       // device arrays, [max_batch][stride] unless noted; a row holds [current block | next block]
  int* ids;
  uint8_t* masked;
  int* draft_tok;
  float* draft_conf;
  int* has_drafts;        // [max_batch] bit 0: the current block has drafts, bit 1: the next block has
  int* remaining;         // [max_batch] r of the current block
  int* remaining_nxt;     // [max_batch] masked positions of the next block
  const int* draft_cap;   // [max_batch] per-sequence cap on the draft length (INT_MAX: none)
  int* window;            // [max_batch] 1: the sequence takes candidates from the next block in the current forward
  int* cand_pos;          // [max_batch][block_len]
  int* cand_tok;
  int* n_cand;            // [max_batch] N of the current forward
  int* accept_log;        // [max_batch][block_len] accepted per forward, 0-terminated
  int* n_forwards;        // [max_batch]
  int* last_accept;       // [max_batch] accepted by the latest step (0 if not active)
  int* last_pos;          // [max_batch] position and token of the last token the latest step accepted
  int* last_tok;          //             (the last valid node's own prediction)
  int* seq_map;           // [max_batch] slot -> sequence of the current forward
  int* mirror;            // [kMirrorWords][max_batch] what the host reads after a step, in mapped host memory
  int max_batch;
  int stride;             // 2 * block_len (row pitch of the arrays above)
};
// Nodes of the verification tree for N candidates: the greedy chain has N + 1; the mix-order tree adds
// one branch for every chain node that has a grandchild (N - 1 of them): 2N nodes for N >= 1.
__host__ __device__ inline int tree_nodes(int N, int mix_order) { return N + 1 + ((mix_order && N >= 2) ? N - 1 : 0); }
// slot a (= rank among unfinished sequences): candidates, node rows [a][n_cap][prev_T + T + T2].  A node's rows
// are: the prev_T tokens of a finished block (prev_ids, device [batch][prev_stride]; nothing asked of them) when
// the forward also commits that block, then the T rows of the current block, then - in a forward whose window
// includes it - the T2 rows of the next block.
void launch_tree_build(cudaStream_t st, BlockState s, int batch, int T, int T2, int max_drafts, int n_cap, int mask_id,
                       int* node_ids, uint8_t* node_masked, const int* prev_ids, int prev_T, int prev_stride,
                       int mix_order);
// per slot: per-node best masked position, walk, state/draft update (same row layout)
void launch_accept(cudaStream_t st, BlockState s, int n_slots, int T, int T2, int n_cap, const int* tok, const float* conf,
                   const uint8_t* node_masked, int* nonfinite_flag, int prev_T, int mix_order);

}  // namespace ssd
