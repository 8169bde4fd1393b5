// Dense projections: many rows against a weight matrix,
//     out[r][n] = sum_k x[r][k] * w[n][k]      (bf16 operands, fp32 accumulation),
// a contraction bound by the tensor cores, not by the weight stream that gemm.cu is built around.  Used by the cache-fill
// forward (prefill of the prompts, refresh of the dual cache) and by verification forwards of some 256 rows and more.
//
// One persistent CTA per SM; the two CTAs of a cluster compute 256 rows x kFeat features as ONE tcgen05.mma.cta_group::2
// (each CTA stages its own 128 rows and half of the features; 32 KB or less per 64-wide K block, six or seven stages
// deep).  The accumulator has rows in the lanes and features in the columns, so an epilogue thread owns part of a row:
// the RMSNorm scale, the rotary pairs, SwiGLU's gate and up all sit in one thread and no transpose is needed.  The
// accumulators (two of 256 columns or four of 128) fill the tensor memory: the epilogue of a tile runs under the main
// loop of the next.  Tiles are walked rows first, so that the CTAs in flight share a few weight tiles and all of the
// activations through L2.
//
// Epilogues: EPI_QKV (rotary embedding; q rows and k and v rows to their buffers and the K/V cache), EPI_SWIGLU, EPI_RESIDUAL and
// EPI_LMHEAD as in gemm.cu.  Two warpgroups share a tile's columns: group g of a 256-feature tile has the 128-feature
// half g, of a 128-feature tile the columns [32 g, +32) and 64 + [32 g, +32) - either way 32-column pieces together with
// the piece 64 columns on, the rotary partner or the `up` of the `gate`.
//
// K splits: a verification forward of few rows runs in gemm.cu, whose sums are cut into `splits` K ranges that are added
// in order.  Here the ranges follow one another in one CTA: each is accumulated by itself and the epilogue threads
// add it to a running sum in registers, in the same order with the same roundings - so a row's bits do not depend on the
// number of rows, and it does not matter which kernel takes a forward.  Every wait is bounded as in gemm.cu.
//
// The bound is the tensor core (256 features: 0.31 us a K block under the power cap; 0.36 measured) and, for narrow tiles, the
// shared memory it reads.  One warp issues the copies and one the MMAs, and both walk their loops converged with one elected
// lane: with descriptors rebuilt in one lane's registers and divisions per K block, issuing took 580 clocks a K block and was
// the bound at every size (down projection at 512 rows 79 us, now 53).
// us per layer of the four projections, this kernel / gemm.cu (with its pass for q, k, v): d 4096, ffn 12288: 512 rows 202 / 242,
// 1024 335 / 415, 4096 1530 / 2560; d 3584, ffn 18944: 512 rows 208 / 234, 4096 1620 / 2600.  By projection, and below that: where
// the forward chooses.
#include "kernels.h"

#include <cuda.h>
#include <math.h>

namespace ssd {
namespace {

constexpr int kTileRows = 256, kBlockK = 64;          // rows of a tile (per pair of CTAs), K of a stage
constexpr int kXBytes = 128 * kBlockK * 2;             // 128 rows x 64 of K
constexpr int kEpiThreads = 256;                       // two warpgroups
constexpr int kThreads = 64 + kEpiThreads;             // warp 0: TMA, warp 1: MMA + tensor memory, then the epilogue
constexpr int kTransWarp = 32 * 128;                    // a warp's transpose buffer: 32 rows x 32 floats, 16-byte chunks swizzled
constexpr int kTransBytes = kEpiThreads / 32 * kTransWarp;
template <int kFeat>
struct Cfg {
  static constexpr int kStageBytes = kXBytes + kFeat / 2 * kBlockK * 2;
  static constexpr int kStages = kFeat == 256 ? 6 : 7;
  static constexpr int kBufs = 512 / kFeat;            // accumulators
  static constexpr int kCh = kFeat / 128;              // 32-column pieces (with their partners) per epilogue thread
  static constexpr int kSumPitch = 9;                  // floats per row of the sum-of-squares exchange (8 + padding)
  static constexpr int kSumBytes = kCh == 1 ? 2 * 128 * kSumPitch * 4 : 0;
  static constexpr int kSmem = kStages * kStageBytes + kTransBytes + kSumBytes + 256 /*barriers*/ + 1024 /*alignment slack*/;
  static_assert(kSmem <= 227 * 1024, "shared memory");
};
constexpr unsigned long long kWaitLimitNs = 2000000000ull;

struct DenseParams {
  int R, N, K;
  int splits;            // K ranges, summed in order
  int m_tiles, n_tiles;
  unsigned long long wait_limit_ns;
  int* err_flag;
  const float* sq;
  int sq_count, sq_stride, norm_dim;
  float norm_eps;
  // EPI_SWIGLU
  bf16* act;
  int act_pitch;
  // EPI_RESIDUAL
  float* h;
  bf16* hb;
  const float* gain;
  float* sq_out;
  int sq_out_stride;
  // EPI_QKV
  QkvOut qkv;
  // EPI_LMHEAD
  float* tile_max;
  float* tile_sum;
  int* tile_arg;
  int topk;
  float* tile_topv;
  int* tile_topi;
  int mask_id;
};

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ unsigned long long globaltimer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n.reg .pred p;\n"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      "selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, unsigned long long limit_ns) {
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = globaltimer_ns();
  int spins = 0;
  while (!mbar_try_wait(bar, parity)) {
    if ((++spins & 63) == 0) {
      if (*abort_flag) return false;
      if (globaltimer_ns() - t0 > limit_ns) return false;
    }
  }
  return true;
}
// arrives on the leader CTA's barrier at the same shared-memory offset
__device__ __forceinline__ void mbar_arrive_leader(uint32_t bar) {
  asm volatile(
      "{\n.reg .b32 a;\n"
      "mapa.shared::cluster.u32 a, %0, 0;\n"
      "mbarrier.arrive.release.cluster.shared::cluster.b64 _, [a];\n}\n" ::"r"(bar) : "memory");
}
// both CTAs' copies count their bytes on the leader's barrier (the pair bit of the address cleared)
constexpr uint32_t kPairLeaderMask = 0xFEFFFFFFu;
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
      ::"r"(dst), "l"((unsigned long long)map), "r"(bar & kPairLeaderMask), "r"(c0), "r"(c1) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit_pair(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
               ::"r"(bar), "h"((uint16_t)3) : "memory");
}
__device__ __forceinline__ void tc_mma_bf16_pair(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n.reg .pred p;\n"
      "setp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n"
      ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
// one lane of a converged warp
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n.reg .pred q;\nelect.sync _|q, 0xffffffff;\nselp.u32 %0, 1, 0, q;\n}\n" : "=r"(p));
  return p != 0;
}
// K-major operand tile, 128-byte swizzle: rows 128 B apart, 8-row groups 1024 B apart
__device__ __forceinline__ uint64_t make_smem_desc(uint32_t saddr) {
  uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}
// 16 consecutive columns of the thread's lane, requested only: nothing of `r` may be read before tmem_ld_wait
__device__ __forceinline__ void tmem_ld16_issue(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
// waits for every request of the thread; ties the registers to the wait so that no use moves above it
__device__ __forceinline__ void tmem_ld_wait(uint32_t (&r)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
      : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
        "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
      :: "memory");
}
__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_arrive_release() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait_acquire() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
__device__ __forceinline__ void epi_bar_sync() { asm volatile("bar.sync 1, 256;" ::: "memory"); }
// as in gemm.cu: the roundings spelled out
__device__ __forceinline__ float sumsq4(const float4& a) {
  return __fmaf_rn(a.w, a.w, __fmaf_rn(a.z, a.z, __fmaf_rn(a.y, a.y, __fmul_rn(a.x, a.x))));
}
__device__ __forceinline__ uint32_t pack2(float a, float b) {
  __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&v);
}
// Between a thread's row and the warp's 32 rows: 32 x 32 floats through the warp's buffer (128 bytes a row, 16-byte chunk c of
// row r at chunk c ^ (r & 7)).  In the transposed form lane l holds, for i = 0..7, the four values from 4 (l & 7) of row
// 4 i + (l >> 3): a warp's access to memory is then four whole 128-byte lines instead of 32 pieces of 32 lines, which is what
// an epilogue of row-owning threads would spend its time on (a load or store unit serves about one line a clock).
__device__ __forceinline__ float4* trans_at(uint8_t* buf, int row, int chunk) {
  return reinterpret_cast<float4*>(buf + row * 128 + ((chunk ^ (row & 7)) << 4));
}
__device__ __forceinline__ void rows_to_buf(uint8_t* buf, int lane, const float (&v)[32]) {
#pragma unroll
  for (int q = 0; q < 8; ++q) *trans_at(buf, lane, q) = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
  __syncwarp();
}
__device__ __forceinline__ void lines_to_rows(uint8_t* buf, int lane, const float4 (&t)[8], float (&v)[32]) {
#pragma unroll
  for (int i = 0; i < 8; ++i) *trans_at(buf, 4 * i + (lane >> 3), lane & 7) = t[i];
  __syncwarp();
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const float4 x = *trans_at(buf, lane, q);
    v[4 * q] = x.x; v[4 * q + 1] = x.y; v[4 * q + 2] = x.z; v[4 * q + 3] = x.w;
  }
  __syncwarp();
}

template <int kFeat, int kEpi>
__global__ void __launch_bounds__(kThreads, 1)
gemm_dense_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmW, const DenseParams p) {
  constexpr int kStages = Cfg<kFeat>::kStages, kStageBytes = Cfg<kFeat>::kStageBytes, kBufs = Cfg<kFeat>::kBufs, kCh = Cfg<kFeat>::kCh;
  constexpr int kSumPitch = Cfg<kFeat>::kSumPitch, kSumBytes = Cfg<kFeat>::kSumBytes;
  extern __shared__ uint8_t smem_dyn[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~(uintptr_t)1023);
  uint8_t* sTrans = smem + kStages * kStageBytes;
  float* sSum = reinterpret_cast<float*>(sTrans + kTransBytes);        // [2 tiles][128 rows][kSumPitch]
  uint64_t* bars = reinterpret_cast<uint64_t*>(sTrans + kTransBytes + kSumBytes);
  uint64_t* full_bar = bars;                       // leader: both CTAs' bytes of a stage
  uint64_t* empty_bar = bars + kStages;            // each CTA: its stage may be refilled
  uint64_t* acc_full = bars + 2 * kStages;         // each CTA: accumulator complete
  uint64_t* acc_empty = acc_full + kBufs;          // leader: the epilogue warps of the pair have read it
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + kBufs);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  pdl_launch_dependents();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n_kb = (p.K + kBlockK - 1) / kBlockK;
  const uint32_t crank = cluster_ctarank() & 1u;
  const bool leader = crank == 0;
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
  const int total = p.m_tiles * p.n_tiles;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(smem_addr(&full_bar[s]), 1);
      mbar_init(smem_addr(&empty_bar[s]), 1);
    }
    for (int b = 0; b < kBufs; ++b) {
      mbar_init(smem_addr(&acc_full[b]), 1);
      mbar_init(smem_addr(&acc_empty[b]), 2 * kEpiThreads / 32);
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"((unsigned long long)&tmW) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"((unsigned long long)&tmX) : "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(tmem_slot)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  cluster_arrive_release();                  // the peer's barriers exist before anything arrives on them
  cluster_wait_acquire();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    if (elect_one()) {
      // (one thread issues everything: what it computes per K block is what bounds a stage, so positions run along and
      // nothing is divided in the loop)
      const int my_tiles = (total - pair + n_pairs - 1) / n_pairs;
      const int steps = my_tiles * n_kb;     // K blocks of all tiles of this pair, one after the other
      const uint32_t smem0 = smem_addr(smem), full0 = smem_addr(full_bar), empty0 = smem_addr(empty_bar);
      struct At { int tile, kb, w_row, x_row; };
      auto enter = [&](At& at) {             // first K block of a tile
        const int nt = at.tile / p.m_tiles, mt = at.tile - nt * p.m_tiles;
        // tile-contiguous weights: 128 rows per (128-feature tile, K block); a 128-feature tile is shared by the pair
        at.w_row = kFeat == 256 ? (nt * 2 + (int)crank) * n_kb * 128 : nt * n_kb * 128 + (int)crank * 64;
        at.x_row = mt * kTileRows + (int)crank * 128;
      };
      auto next = [&](At& at) {
        at.w_row += 128;
        if (++at.kb == n_kb) {
          at.kb = 0;
          at.tile += n_pairs;
          if (at.tile < total) enter(at);
        }
      };
      auto load_w = [&](const At& at, int s) { tma_load_2d_pair(smem0 + s * kStageBytes + kXBytes, &tmW, full0 + 8 * s, 0, at.w_row); };
      auto load_x = [&](const At& at, int s) { tma_load_2d_pair(smem0 + s * kStageBytes, &tmX, full0 + 8 * s, at.kb * kBlockK, at.x_row); };
      auto expect = [&](int s) { if (leader) mbar_expect_tx(full0 + 8 * s, 2u * kStageBytes); };
      // the weights depend on no earlier kernel: fill the ring with them before the dependency wait
      const int pre = steps < kStages ? steps : kStages;
      At at{pair, 0, 0, 0}, ax;
      enter(at);
      ax = at;
      for (int it = 0; it < pre; ++it, next(at)) {
        expect(it);
        load_w(at, it);
      }
      pdl_wait();
      for (int it = 0; it < pre; ++it, next(ax)) load_x(ax, it);
      bool ok = true;
      int it = pre, s = pre == kStages ? 0 : pre;
      uint32_t phase = 0;                    // parity of the use of a stage that has to be over
      for (; it < steps; ++it, next(at)) {
        if (!mbar_wait(empty0 + 8 * s, phase, abort_flag, p.wait_limit_ns)) { ok = false; break; }
        expect(s);
        load_w(at, s);
        load_x(at, s);
        if (++s == kStages) { s = 0; phase ^= 1u; }
      }
      if (!ok) {
        *abort_flag = 1;
        raise_word(p.err_flag, 1);
        // let the copies in flight land before the shared memory goes away
        const int first = it > kStages ? it - kStages : 0;
        for (int j = first; j < it && leader; ++j) {
          const unsigned long long t0 = globaltimer_ns();
          while (!mbar_try_wait(smem_addr(&full_bar[j % kStages]), (uint32_t)((j / kStages) & 1)))
            if (globaltimer_ns() - t0 > p.wait_limit_ns) break;
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer (the even CTA, for both)
    // One lane, elected once, walks the whole loop: with warp-uniform addresses and descriptors an MMA is a few instructions
    // (from a diverged lane's registers each took 70 clocks to issue, 580 per K block in all).  Of 256-feature residual tiles, whose
    // epilogue is the one that spills, the whole warp walks it and one lane issues: the compiler then spills less there (loads of
    // 584 bytes for 608).  us of O and down, d 4096, one lane / the warp: 700 rows 33.1 / 32.0 and 73.7 / 70.9, 1024 rows 35.5 / 34.6
    // and 76.7 / 73.9; of 128-feature tiles, 1536 rows, 43.7 / 48.1 and 111.9 / 125.4.
    constexpr bool kWarpWalks = kFeat == 256 && kEpi == EPI_RESIDUAL;
    auto all = [](bool v) -> bool { return kWarpWalks ? __all_sync(0xffffffffu, v) != 0 : v; };
    if (leader && (kWarpWalks || elect_one())) {
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kFeat >> 3) << 17) | ((uint32_t)(kTileRows >> 4) << 24);
      bool ok = true;
      const uint32_t full0 = smem_addr(full_bar), empty0 = smem_addr(empty_bar);
      const uint64_t xdesc0 = make_smem_desc(smem_addr(smem)), wdesc0 = make_smem_desc(smem_addr(smem) + kXBytes);
      int s = 0, nth = 0;                    // stage; accumulators used so far
      uint32_t phase = 0;
      for (int tile = pair; tile < total && ok; tile += n_pairs) {
        for (int split = 0; split < p.splits && ok; ++split, ++nth) {
          const int buf = nth % kBufs;
          if (nth >= kBufs) {
            ok = all(mbar_wait(smem_addr(&acc_empty[buf]), (uint32_t)((nth / kBufs) & 1) ^ 1u, abort_flag, p.wait_limit_ns));
            if (!ok) break;
            tc_fence_after();
          }
          const uint32_t tmem_d = tmem_base + (uint32_t)(buf * kFeat);
          const int kb0 = split * n_kb / p.splits, kb1 = (split + 1) * n_kb / p.splits;
          for (int kb = kb0; kb < kb1; ++kb) {
            ok = all(mbar_wait(full0 + 8 * s, phase, abort_flag, p.wait_limit_ns));
            if (!ok) break;
            // (the address field of a descriptor counts 16-byte units: a stage and a k16 step are additions)
            const uint64_t xd = xdesc0 + (uint32_t)(s * (kStageBytes >> 4)), wd = wdesc0 + (uint32_t)(s * (kStageBytes >> 4));
            if (!kWarpWalks || elect_one()) {
#pragma unroll
              for (int k = 0; k < kBlockK / 16; ++k) tc_mma_bf16_pair(tmem_d, xd + 2 * k, wd + 2 * k, idesc, (uint32_t)(((kb - kb0) | k) != 0));
              tc_commit_pair(empty0 + 8 * s);
              if (kWarpWalks && kb + 1 == kb1) tc_commit_pair(smem_addr(&acc_full[buf]));
            }
            if (kWarpWalks) __syncwarp();
            if (++s == kStages) { s = 0; phase ^= 1u; }
          }
          if (!kWarpWalks && ok) tc_commit_pair(smem_addr(&acc_full[buf]));
        }
      }
      if (!ok && (!kWarpWalks || lane == 0)) { *abort_flag = 1; raise_word(p.err_flag, 2); }
    }
    __syncwarp();
  } else {
    // ------------------------------------------------------------------ epilogue
    const int quad = warp & 3, group = (warp - 2) >> 2;
    pdl_wait();
    bool ok = true;
    int nth = 0, n_done = 0;
    uint8_t* trans = sTrans + (warp - 2) * kTransWarp;
    // (after an expired wait the loop goes on without waiting, reading or writing: the warps still meet at the barriers)
    for (int tile = pair; tile < total; tile += n_pairs, ++n_done) {
      const int lrow = quad * 32 + lane;
      const int row0 = (tile % p.m_tiles) * kTileRows + (int)crank * 128 + quad * 32, row = row0 + lane;   // this warp's, this thread's
      const int n_base = (tile / p.m_tiles) * kFeat;
      const int lr4 = lane >> 3, lc4 = 4 * (lane & 7);       // transposed form: row 4 i + lr4, columns from lc4
      // this thread's columns: piece c is [col(c), +32) together with [col(c) + 64, +32)
      auto col = [&](int c) -> int { return kFeat == 256 ? 128 * group + 32 * c : 32 * group; };
      const bool live = row < p.R;
      float inv = 1.f;
      if (p.sq != nullptr && live) {         // RMSNorm, consumer side: the producers' per-tile sums in slot order
        const float* q = p.sq + (size_t)row * p.sq_stride;
        float ss = 0.f;
        if (((p.sq_count | p.sq_stride) & 3) == 0) {
          for (int t = 0; t < p.sq_count; t += 4) {
            const float4 v = *reinterpret_cast<const float4*>(q + t);
            ss += v.x; ss += v.y; ss += v.z; ss += v.w;
          }
        } else {
          for (int t = 0; t < p.sq_count; ++t) ss += q[t];
        }
        inv = rsqrtf(ss / (float)p.norm_dim + p.norm_eps);
      }
      if constexpr (kEpi == EPI_LMHEAD) {
        // The group's half of the features is one vocabulary tile, all of a row's entries in one thread, a quarter at a time.
        const int buf = nth % kBufs, v_tile = (n_base >> 7) + group, v0 = v_tile * 128;
        if (ok) ok = mbar_wait(smem_addr(&acc_full[buf]), (uint32_t)((nth / kBufs) & 1), abort_flag, p.wait_limit_ns);
        ok = __all_sync(0xffffffffu, ok);
        ++nth;
        if (!ok) continue;
        tc_fence_after();
        const uint32_t taddr = tmem_base + (uint32_t)(buf * kFeat + 128 * group) + ((uint32_t)(quad * 32) << 16);
        const bool some_dead = v0 + 128 > p.N || (p.mask_id >= v0 && p.mask_id < v0 + 128);
        LmStat st[4];
        float tv[kLmTopKMax];
        int ti[kLmTopKMax];
#pragma unroll
        for (int r = 0; r < kLmTopKMax; ++r) { tv[r] = -INFINITY; ti[r] = 0x7fffffff; }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          uint32_t r1[16], r2[16];
          tmem_ld16_issue(taddr + 32 * q, r1);
          tmem_ld16_issue(taddr + 32 * q + 16, r2);
          tmem_ld_wait(r1);
          tmem_ld_wait(r2);
          float x[32];
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            x[j] = p.sq != nullptr ? __fmul_rn(__uint_as_float(r1[j]), inv) : __uint_as_float(r1[j]);
            x[16 + j] = p.sq != nullptr ? __fmul_rn(__uint_as_float(r2[j]), inv) : __uint_as_float(r2[j]);
          }
          if (some_dead) {
#pragma unroll
            for (int j = 0; j < 32; ++j)
              if (v0 + 32 * q + j >= p.N || v0 + 32 * q + j == p.mask_id) x[j] = -INFINITY;
          }
          st[q] = lm_quarter(x, v0 + 32 * q);
          if (p.topk > 0) {
#pragma unroll
            for (int j = 0; j < 32; ++j) lm_insert(tv, ti, x[j], v0 + 32 * q + j);
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_leader(smem_addr(&acc_empty[buf]));
        if (live && v0 < p.N) {
          const LmStat s = lm_merge(lm_merge(st[0], st[1]), lm_merge(st[2], st[3]));
          const size_t o = (size_t)v_tile * p.R + row;
          p.tile_max[o] = s.m;
          p.tile_sum[o] = s.sum;
          p.tile_arg[o] = s.arg;
#pragma unroll
          for (int r = 0; r < kLmTopKMax; ++r)
            if (r < p.topk) { p.tile_topv[o * kLmTopKMax + r] = tv[r]; p.tile_topi[o * kLmTopKMax + r] = ti[r]; }
        }
        continue;
      }
      float run[kCh][2][32];                 // running sums over the K ranges; EPI_RESIDUAL: on top of the residual stream
      if (kEpi == EPI_RESIDUAL) {
        float4 t[2 * kCh][8];                // all pieces in flight together
#pragma unroll
        for (int e = 0; e < 2 * kCh; ++e)
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const int n = n_base + col(e >> 1) + 64 * (e & 1) + lc4, r = row0 + 4 * i + lr4;
            t[e][i] = (r < p.R && n < p.N) ? *reinterpret_cast<const float4*>(p.h + (size_t)r * p.N + n) : make_float4(0.f, 0.f, 0.f, 0.f);
          }
#pragma unroll
        for (int e = 0; e < 2 * kCh; ++e) lines_to_rows(trans, lane, t[e], run[e >> 1][e & 1]);
      } else {
#pragma unroll
        for (int c = 0; c < kCh; ++c)
#pragma unroll
          for (int j = 0; j < 64; ++j) run[c][j >> 5][j & 31] = 0.f;
      }
      for (int split = 0; split < p.splits; ++split, ++nth) {
        const int buf = nth % kBufs;
        if (ok) ok = mbar_wait(smem_addr(&acc_full[buf]), (uint32_t)((nth / kBufs) & 1), abort_flag, p.wait_limit_ns);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) continue;
        tc_fence_after();
        const uint32_t taddr = tmem_base + (uint32_t)(buf * kFeat) + ((uint32_t)(quad * 32) << 16);
#pragma unroll
        for (int e = 0; e < 2 * kCh; ++e) {          // 16 columns and their partners at a time
          const int c = e >> 1, j0 = (e & 1) * 16;
          uint32_t r1[16], r2[16];
          tmem_ld16_issue(taddr + col(c) + j0, r1);
          tmem_ld16_issue(taddr + col(c) + j0 + 64, r2);
          tmem_ld_wait(r1);
          tmem_ld_wait(r2);
          if (kEpi == EPI_RESIDUAL) {
#pragma unroll
            for (int j = 0; j < 16; ++j) { run[c][0][j0 + j] += __uint_as_float(r1[j]); run[c][1][j0 + j] += __uint_as_float(r2[j]); }
          } else if (kEpi == EPI_QKV) {
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              run[c][0][j0 + j] = __fadd_rn(run[c][0][j0 + j], __fmul_rn(__uint_as_float(r1[j]), inv));
              run[c][1][j0 + j] = __fadd_rn(run[c][1][j0 + j], __fmul_rn(__uint_as_float(r2[j]), inv));
            }
          } else {
#pragma unroll
            for (int j = 0; j < 16; ++j) { run[c][0][j0 + j] = __uint_as_float(r1[j]) * inv; run[c][1][j0 + j] = __uint_as_float(r2[j]) * inv; }
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_leader(smem_addr(&acc_empty[buf]));
      }
      if (kEpi == EPI_QKV && ok) {
        const QkvOut& o = p.qkv;
        const int half = o.hd >> 1, heads = o.H + 2 * o.Hkv;
        // of the thread's own row; the transposed form below asks the row's lane
        const int safe = live ? row : 0, slot = safe / o.map.rows_per_seq, lr = safe - slot * o.map.rows_per_seq;
        const int pos = o.map.pos0 + lr % o.map.T;
        const bool to_cache = live && lr < o.cache_rows;
        const unsigned long long kv_row = to_cache ? (size_t)seq_of_slot(o.map, slot) * o.cache_seq_stride + (size_t)pos * o.kv_pos_stride : 0;
        const unsigned cache_mask = __ballot_sync(0xffffffffu, to_cache);
        // 32 features from i0 of head `head`, and their rotary partners half a head on
        auto finish = [&](int head, int i0, const float (&x1)[32], const float (&x2)[32]) {
          if (head >= heads) return;
          const bool is_q = head < o.H, is_k = !is_q && head < o.H + o.Hkv;
          const int j = head - o.H - (is_k ? 0 : o.Hkv);
          // 16 features and their partners at a time: chunks 0-3 and 4-7 of a buffer row, four lanes to a row
#pragma unroll
          for (int j0 = 0; j0 < 32; j0 += 16) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              *trans_at(trans, lane, q) = make_float4(x1[j0 + 4 * q], x1[j0 + 4 * q + 1], x1[j0 + 4 * q + 2], x1[j0 + 4 * q + 3]);
              *trans_at(trans, lane, 4 + q) = make_float4(x2[j0 + 4 * q], x2[j0 + 4 * q + 1], x2[j0 + 4 * q + 2], x2[j0 + 4 * q + 3]);
            }
            __syncwarp();
            const int f = i0 + j0 + 4 * (lane & 3);
#pragma unroll 1
            for (int i = 0; i < 4; ++i) {
              const int src = 8 * i + (lane >> 2), r = row0 + src;
              float4 u = *trans_at(trans, src, lane & 3), w = *trans_at(trans, src, 4 + (lane & 3));
              const int r_pos = __shfl_sync(0xffffffffu, pos, src);
              const unsigned long long r_kv = __shfl_sync(0xffffffffu, kv_row, src);
              if (r >= p.R) continue;
              if (is_q || is_k) {
                const float4* cs = reinterpret_cast<const float4*>(o.rope + (size_t)r_pos * half + f);
                const float4 c0 = cs[0], c1 = cs[1];
                rope_pair(u.x, w.x, c0.x, c0.y); rope_pair(u.y, w.y, c0.z, c0.w);
                rope_pair(u.z, w.z, c1.x, c1.y); rope_pair(u.w, w.w, c1.z, c1.w);
              }
              const uint2 lo = make_uint2(pack2(u.x, u.y), pack2(u.z, u.w)), hi = make_uint2(pack2(w.x, w.y), pack2(w.z, w.w));
              auto put = [&](bf16* dst) {
                *reinterpret_cast<uint2*>(dst + f) = lo;
                *reinterpret_cast<uint2*>(dst + half + f) = hi;
              };
              if (is_q) {
                put(o.q + ((size_t)r * o.H + head) * o.hd);
              } else {
                if (o.local_k) put((is_k ? o.local_k : o.local_v) + ((size_t)r * o.Hkv + j) * o.hd);
                if ((cache_mask >> src) & 1u) put((is_k ? o.cache_k : o.cache_v) + (size_t)r_kv + (size_t)j * o.kv_head_stride);
              }
            }
            __syncwarp();
          }
        };
        if (o.hd == 128) {
#pragma unroll
          for (int c = 0; c < kCh; ++c) finish((n_base + col(c)) >> 7, col(c) & 63, run[c][0], run[c][1]);
        } else if (kFeat == 256) {           // (head dimension 64: the launcher takes 256-feature tiles)
#pragma unroll
          for (int hb = 0; hb < 2; ++hb) finish(((n_base + col(0)) >> 6) + hb, 0, run[0][hb], run[kCh - 1][hb]);
        }
      }
      if (kEpi == EPI_SWIGLU && ok) {
        // a 128-feature weight tile = 64 gate features, then the matching 64 up features
#pragma unroll
        for (int c = 0; c < kCh; ++c) {
          if (n_base + col(c) >= p.N) continue;
          float a[32];
#pragma unroll
          for (int j = 0; j < 32; j += 2) swiglu2(run[c][0][j], run[c][0][j + 1], run[c][1][j], run[c][1][j + 1], a[j], a[j + 1]);
          rows_to_buf(trans, lane, a);
          const int f = ((n_base + (col(c) & ~127)) >> 1) + (col(c) & 63) + lc4;
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const int r = row0 + 4 * i + lr4;
            const float4 t = *trans_at(trans, 4 * i + lr4, lane & 7);
            if (r < p.R) *reinterpret_cast<uint2*>(p.act + (size_t)r * p.act_pitch + f) = make_uint2(pack2(t.x, t.y), pack2(t.z, t.w));
          }
          __syncwarp();
        }
      }
      if (kEpi == EPI_RESIDUAL) {
        // EPI_RESIDUAL: the new residual stream, bf16(h * gain), and per 128-feature tile the row's sum of squares in
        // gemm.cu's order: quads of four features, then a butterfly over the 32 quads (partners 16, 8, 4, 2, 1 apart)
        float t[kCh][8];
#pragma unroll
        for (int c = 0; c < kCh; ++c) {
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            float part[2] = {0.f, 0.f};
#pragma unroll
            for (int half = 0; half < 2; ++half)
              if (n_base + col(c) + 64 * half + 4 * q < p.N)
                part[half] = sumsq4(make_float4(run[c][half][4 * q], run[c][half][4 * q + 1], run[c][half][4 * q + 2], run[c][half][4 * q + 3]));
            t[c][q] = part[0] + part[1];
          }
#pragma unroll
          for (int half = 0; half < 2; ++half) {
            const int n = n_base + col(c) + 64 * half + lc4;
            const float4 g = n < p.N ? *reinterpret_cast<const float4*>(p.gain + n) : make_float4(0.f, 0.f, 0.f, 0.f);
            rows_to_buf(trans, lane, run[c][half]);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              const int r = row0 + 4 * i + lr4;
              const float4 v = *trans_at(trans, 4 * i + lr4, lane & 7);
              if (ok && r < p.R && n < p.N) {
                *reinterpret_cast<float4*>(p.h + (size_t)r * p.N + n) = v;
                *reinterpret_cast<uint2*>(p.hb + (size_t)r * p.N + n) = make_uint2(pack2(v.x * g.x, v.y * g.y), pack2(v.z * g.z, v.w * g.w));
              }
            }
            __syncwarp();
          }
        }
        float* ex = sSum + ((n_done & 1) * 128 + lrow) * kSumPitch;
        if (kCh == 1 && group == 1) {
#pragma unroll
          for (int q = 0; q < 8; ++q) ex[q] = t[0][q];
        }
        if (kCh == 1) epi_bar_sync();
        if (kCh == 2 || group == 0) {
          float u[8];
#pragma unroll
          for (int q = 0; q < 8; ++q) u[q] = t[0][q] + (kCh == 2 ? t[kCh - 1][q] : ex[q]);
#pragma unroll
          for (int o = 4; o > 0; o >>= 1)
#pragma unroll
            for (int q = 0; q < o; ++q) u[q] += u[q + o];
          const int slot = (n_base + (kCh == 2 ? 128 * group : 0)) >> 7;
          if (ok && live && slot * 128 < p.N) p.sq_out[(size_t)row * p.sq_out_stride + slot] = u[0];
        }
      }
    }
    if (!ok && lane == 0) { *abort_flag = 1; raise_word(p.err_flag, 3); }
  }
  tc_fence_before();
  __syncthreads();
  cluster_arrive_release();                  // both CTAs have read their accumulators; nothing is on its way between them
  cluster_wait_acquire();
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
}

template <int kFeat, int kEpi>
int launch(cudaStream_t st, const GemmArgs& g, DenseParams p, int sms, int dev) {
  p.n_tiles = (g.N + kFeat - 1) / kFeat;
  alignas(64) CUtensorMap tmX, tmW;
  const uint64_t w_rows = (uint64_t)gemm_tiles(g.N) * ((g.K + kBlockK - 1) / kBlockK) * 128;
  if (encode_tmap_bf16_2d(&tmX, g.x, (uint64_t)g.R, (uint64_t)g.K, (uint64_t)g.x_pitch, 128) != 0 ||
      encode_tmap_bf16_2d(&tmW, g.w, w_rows, kBlockK, kBlockK, kFeat / 2) != 0)
    return -4;
  static PerDevice<bool> attr_set = {};             // the shared-memory opt-in
  if (!attr_set[dev]) {
    if (cudaFuncSetAttribute(gemm_dense_kernel<kFeat, kEpi>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<kFeat>::kSmem) != cudaSuccess) return -4;
    attr_set[dev] = true;
  }
  const int pairs = sms / 2, total = p.m_tiles * p.n_tiles;
  const dim3 grid(2 * (total < pairs ? total : pairs));
  return launch_pdl_cluster(gemm_dense_kernel<kFeat, kEpi>, grid, dim3(kThreads), (size_t)Cfg<kFeat>::kSmem, st, 2u, tmX, tmW, p) == cudaSuccess ? 0 : -4;
}

}  // namespace

int launch_gemm_dense(cudaStream_t st, const GemmArgs& g) {
  if ((g.x_pitch % 8) || (((uintptr_t)g.x) & 15) || (((uintptr_t)g.w) & 15) || !g.w_tiled) return -2;
  if (g.R < 1 || g.N < 1 || g.K < 1) return -2;
  if (g.splits < 1 || g.splits > (g.K + kBlockK - 1) / kBlockK) return -2;   // every range owns at least one K block
  if (g.sq != nullptr && (g.sq_count < 1 || g.norm_dim < 1)) return -2;
  if (g.epi == EPI_RESIDUAL) {
    if ((g.N & 3) || !g.h || !g.hb || !g.gain || !g.sq_out) return -2;
  } else if (g.epi == EPI_SWIGLU) {
    if ((g.N % 128) || g.splits != 1) return -2;
  } else if (g.epi == EPI_LMHEAD) {
    if (g.splits != 1 || !g.tile_max || !g.tile_sum || !g.tile_arg || g.topk < 0 || g.topk > kLmTopKMax || (g.topk > 0 && (!g.tile_topv || !g.tile_topi))) return -2;
  } else if (g.epi == EPI_QKV) {
    if (!g.qkv || (g.qkv->hd != 64 && g.qkv->hd != 128) || !g.sq) return -2;
  } else {
    return -2;
  }
  DenseParams p{};
  p.R = g.R; p.N = g.N; p.K = g.K; p.splits = g.splits;
  p.m_tiles = (g.R + kTileRows - 1) / kTileRows;
  p.wait_limit_ns = g.wait_limit_ns > 0 ? g.wait_limit_ns : kWaitLimitNs;
  p.err_flag = g.err_flag;
  p.sq = g.sq; p.sq_count = g.sq_count; p.sq_stride = g.sq_stride; p.norm_dim = g.norm_dim; p.norm_eps = g.norm_eps;
  p.act = g.act; p.act_pitch = g.act_pitch;
  p.h = g.h; p.hb = g.hb; p.gain = g.gain; p.sq_out = g.sq_out; p.sq_out_stride = g.sq_out_stride;
  if (g.qkv) p.qkv = *g.qkv;
  p.tile_max = g.tile_max; p.tile_sum = g.tile_sum; p.tile_arg = g.tile_arg; p.topk = g.topk; p.tile_topv = g.tile_topv; p.tile_topi = g.tile_topi;
  p.mask_id = g.mask_id;
  static PerDevice<int> sm_count = {};
  const int dev = device_slot();
  if (dev < 0) return -4;
  if (sm_count[dev] == 0) {
    int n = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 2) return -4;
    sm_count[dev] = n;
  }
  // The width that leaves less of the machine idle in the last wave of tiles.  A 128-feature tile takes 0.6 of the time of a
  // 256-feature one (three quarters of the bytes, a shorter epilogue): QKV and gate/up at 4096 rows 18.4 / 29.7 and 14.6 /
  // 22.1 us a tile.  A residual tile adds the exposed part of its epilogue, which is mostly that of the wide one: O 19.5 / 42 us
  // (64 K blocks), down 47.6 / 78 (192).
  const int sms = sm_count[dev], pairs = sms / 2;
  const long long kb = (g.K + kBlockK - 1) / kBlockK;
  const long long waves256 = ((long long)p.m_tiles * ((g.N + 255) / 256) + pairs - 1) / pairs;
  const long long waves128 = ((long long)p.m_tiles * ((g.N + 127) / 128) + pairs - 1) / pairs;
  const bool narrow = g.epi == EPI_RESIDUAL ? waves128 * (60 + 3 * kb) < waves256 * (240 + 4 * kb)
                                            : !(g.epi == EPI_QKV && g.qkv->hd == 64) && waves128 * 6 < waves256 * 10;
  switch (g.epi) {
    case EPI_LMHEAD: return launch<256, EPI_LMHEAD>(st, g, p, sms, dev);
    case EPI_QKV: return narrow ? launch<128, EPI_QKV>(st, g, p, sms, dev) : launch<256, EPI_QKV>(st, g, p, sms, dev);
    case EPI_SWIGLU: return narrow ? launch<128, EPI_SWIGLU>(st, g, p, sms, dev) : launch<256, EPI_SWIGLU>(st, g, p, sms, dev);
    default: return narrow ? launch<128, EPI_RESIDUAL>(st, g, p, sms, dev) : launch<256, EPI_RESIDUAL>(st, g, p, sms, dev);
  }
}

}  // namespace ssd
