// Projections of a few hundred rows at most whose features are shared out over the whole machine at once,
//     out[r][n] = sum_k x[r][k] * w[n][k]      (bf16 operands, fp32 accumulation),
// for the projections that pair features: q|k|v (a feature's rotary partner is 64 features on) and gate|up (64 gates, then
// their 64 ups, in a tile of 128 weight rows).
//
// The weights are whole tiles of 128 features, and neither 96 nor 192 of them go evenly into 148 SMs: the kernels that work
// by tiles take two turns where 1.3 would do, or leave a third of the SMs without work.  Here the unit is a run of `cpu`
// couples (a feature and its partner), any multiple of eight: as many as it takes for every pair of SMs to have one unit.  A
// pair of CTAs computes up to 256 rows x 2 cpu features as one tcgen05.mma.cta_group::2 (two, beyond 256 features): rows in
// the lanes, half of the rows in each CTA (the fewer rows, the less each takes in), the first features of the couples staged
// by the even CTA and their partners by the odd one.  So both features of a couple are columns of the same lane and an
// epilogue thread has all it needs: the RMSNorm scale, the rotation or SwiGLU, and rounding to bf16.  No partial sums, no pass
// behind the projection.
//
// A run is copied from the tile-contiguous weights by boxes of 64, 32, 16 and 8 rows.  K splits (the ranges that gemm.cu
// adds up in order) have accumulators of their own, summed in the same order at the end: the bits of a row are those of the
// other kernels.  Rows of the A operand that no box fills, and weight rows between a run's end and the MMA's width, hold
// whatever the stage held before; they only reach accumulator rows and columns that nothing reads.
//
// Bound by the weights (HBM) and, for narrow units, by the tensor pipe (256 rows whatever `half` is).  At 256 rows gate|up of d 4096,
// ffn 12288 streams its 201 MB in 32 us of the kernel's 41; the rest is the ramp and the epilogue (alone and cold, 44 us, either limit is
// reached for 57 % of the launch, q|k|v's 32 us for 40 %).  us in the live stream, before /
// now: 256 rows q|k|v 39 / 32, gate|up 54 / 43; 216 rows 37 (with its finishing pass) / 29, 50 / 41; 128 rows 31 / 31, 41 / 43, so
// fewer rows stay with gemm.cu, which leaves SMs to the kernel behind it.  More than 256 rows, which a pair has no room for at once,
// are the dense kernel's, whose tiles have their epilogue under the next tile's main loop.  Every wait is bounded as in gemm.cu, and
// the tensor memory, all of it, is never waited for: an SM has registers for one of these CTAs and for no other that holds any.
#include "kernels.h"

#include <cuda.h>
#include <math.h>

namespace ssd {
namespace {

constexpr int kBlockK = 64;
// epilogue warpgroups: they take the 16-couple pieces of a unit in turn
template <int kEpi> constexpr int kGroups = kEpi == EPI_SWIGLU ? 3 : 2;
template <int kEpi> constexpr int kEpiThreads = 128 * kGroups<kEpi>;
constexpr int kProducers = 2;                           // warps that ask for weights: they take the K blocks in turn
// warp 0: activations, warp 1: MMA + tensor memory, the epilogue, the weights
template <int kEpi> constexpr int kThreads = 64 + kEpiThreads<kEpi> + 32 * kProducers;
template <int kEpi> constexpr int kEpiWarpEnd = 2 + kEpiThreads<kEpi> / 32;
// a warp's transpose buffer: 32 rows of 16 features and their partners in fp32, or of 16 results in bf16
template <int kEpi> constexpr int kTransWarp = kEpi == EPI_SWIGLU ? 32 * 32 : 32 * 128;
template <int kEpi> constexpr int kTransBytes = kEpiThreads<kEpi> / 32 * kTransWarp<kEpi>;
constexpr int kMaxStages = 20, kMaxBufs = 4, kMaxBoxes = 12;
constexpr int kBarBytes = 512, kListBytes = kProducers * kMaxBoxes * 16;
constexpr int kSmemMax = 226 * 1024;
constexpr unsigned long long kWaitLimitNs = 2000000000ull;

struct WaveParams {
  int R, K, couples;     // couples: N / 2
  int splits;            // K ranges with an accumulator each
  int half;              // rows of a CTA
  int units;
  int cpu;               // couples of a unit
  int n0, n1;            // features of the two MMAs (n1 = 0: one)
  int stages, stage_bytes, bufs;
  int x_bytes;           // of a stage: half rows x 64 of K, then the weights
  unsigned long long wait_limit_ns;
  int* err_flag;
  const float* sq;
  int sq_count, sq_stride, norm_dim;
  float norm_eps;
  bf16* act;             // EPI_SWIGLU
  int act_pitch;
  QkvOut qkv;            // EPI_QKV
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
// ... suspended for up to some 20 us: a warp that polls instead takes issue slots and shared-memory cycles from the warp that
// issues the MMAs
__device__ __forceinline__ bool mbar_try_wait_long(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n.reg .pred p;\n"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n"
      "selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok) : "r"(bar), "r"(parity), "r"(20000u) : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, unsigned long long limit_ns) {
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = globaltimer_ns();
  while (!mbar_try_wait_long(bar, parity))
    if (*abort_flag || globaltimer_ns() - t0 > limit_ns) return false;
  return true;
}
__device__ __forceinline__ uint32_t map_to_rank(uint32_t addr, uint32_t rank) {
  uint32_t out;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(out) : "r"(addr), "r"(rank));
  return out;
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
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
__device__ __forceinline__ void tmem_ld_wait(uint32_t (&r)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
      : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
        "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
      :: "memory");
}
__device__ __forceinline__ void cluster_arrive_release() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait_acquire() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
__device__ __forceinline__ uint32_t pack2(float a, float b) {
  __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&v);
}
// 16-byte chunk `chunk` of row `row` of a warp's transpose buffer (128 bytes a row)
__device__ __forceinline__ float4* trans_at(uint8_t* buf, int row, int chunk) {
  return reinterpret_cast<float4*>(buf + row * 128 + ((chunk ^ (row & 7)) << 4));
}

struct WeightMaps { CUtensorMap by_rows[4]; };         // boxes of 64, 32, 16 and 8 rows

template <int kEpi, bool kWide>
__global__ void __launch_bounds__(kThreads<kEpi>, 1)
gemm_wave_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ WeightMaps tmW, const WaveParams p) {
  extern __shared__ uint8_t smem_dyn[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~(uintptr_t)1023);
  uint8_t* sTrans = smem + p.stages * p.stage_bytes;
  int4* s_box = reinterpret_cast<int4*>(sTrans + kTransBytes<kEpi>);       // each producer's copies of weights: row of K block 0, offset in a stage, map
  uint64_t* bars = reinterpret_cast<uint64_t*>(sTrans + kTransBytes<kEpi> + kListBytes);
  uint64_t* full_bar = bars;                       // leader: both CTAs' bytes of a stage
  uint64_t* empty_bar = bars + kMaxStages;         // each CTA: its stage may be refilled
  uint64_t* acc_full = bars + 2 * kMaxStages;      // each CTA: a unit's accumulators are complete
  uint64_t* acc_empty = acc_full + kMaxBufs;       // leader: the epilogue warps of the pair have read them
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + kMaxBufs);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  pdl_launch_dependents();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int kEpiEnd = kEpiWarpEnd<kEpi>, kG = kGroups<kEpi>;
  const int n_kb = (p.K + kBlockK - 1) / kBlockK;
  const int crank = blockIdx.x & 1;         // rank in the cluster of two
  const bool leader = crank == 0;
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
  const int acc_cols = p.n0 + p.n1;

  if (threadIdx.x == 0) {
    for (int s = 0; s < p.stages; ++s) {
      mbar_init(smem_addr(&full_bar[s]), 1);
      mbar_init(smem_addr(&empty_bar[s]), 1);
    }
    for (int b = 0; b < p.bufs; ++b) {
      mbar_init(smem_addr(&acc_full[b]), 1);
      mbar_init(smem_addr(&acc_empty[b]), 2 * kEpiThreads<kEpi> / 32);
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"((unsigned long long)&tmX) : "memory");
    for (int i = 0; i < 4; ++i) asm volatile("prefetch.tensormap [%0];" ::"l"((unsigned long long)&tmW.by_rows[i]) : "memory");
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

  // After an error: let a warp's copies in flight land before the shared memory goes away - its uses, every `every`th from
  // `mine` on, of the ring's round before use `now`.
  auto drain = [&](int now, int mine, int every) {
    for (int q = now > p.stages ? now - p.stages : 0; leader && q < now; ++q) {
      if (q % every != mine) continue;
      const unsigned long long t0 = globaltimer_ns();
      while (!mbar_try_wait(smem_addr(&full_bar[q % p.stages]), (uint32_t)((q / p.stages) & 1)))
        if (globaltimer_ns() - t0 > p.wait_limit_ns) break;
    }
  };
  if (warp == 0) {
    // ------------------------------------------------------------------ activations
    // The first of every stage, by a warp of its own: asked for as soon as the kernel before is done, whatever the weights' warps
    // are at.  (A stage's bytes may arrive before they have said how many there will be: its barrier still waits for that.)
    if (elect_one()) {
      const uint32_t smem0 = smem_addr(smem), full0 = smem_addr(full_bar);
      pdl_wait();
      int s = 0;
      for (int unit = pair; unit < p.units && s < p.stages; unit += n_pairs)
        for (int kb = 0; kb < n_kb && s < p.stages; ++kb, ++s)
          tma_load_2d_pair(smem0 + s * p.stage_bytes, &tmX, full0 + 8 * s, kb * kBlockK, crank * p.half);
    }
    __syncwarp();
  } else if (warp >= kEpiEnd) {
    // ------------------------------------------------------------------ weights, and the activations from the second use of a stage on
    // The weights depend on no earlier kernel.  Asking for a stage (the expected bytes and its copies) takes a warp 250 clocks and more,
    // whatever the size of the copies, so two warps ask in turn.  One lane, elected once, walks the warp's K blocks.
    const int turn = warp - kEpiEnd;
    if (elect_one()) {
      bool ok = true;
      const uint32_t smem0 = smem_addr(smem), full0 = smem_addr(full_bar), empty0 = smem_addr(empty_bar);
      int4* const box = s_box + turn * kMaxBoxes;
      int n_box = 0;
      const int x_row = crank * p.half;
      bool waited = false;
      uint32_t bytes = 0;                    // of a stage, both CTAs
      auto enter = [&](int unit) {           // the copies of a unit: its couples cut at the weight tiles, and powers of two of them in one
        const int c0 = unit * p.cpu, n = min(p.cpu, p.couples - c0);
        bytes = 2u * (uint32_t)((p.half + n) * kBlockK * 2);
        n_box = 0;
        for (int done = 0; done < n;) {
          const int c = c0 + done, left = min(64 - (c & 63), n - done);
          const int m = left >= 64 ? 0 : left >= 32 ? 1 : left >= 16 ? 2 : 3;
          box[n_box++] = make_int4((c >> 6) * n_kb * 128 + crank * 64 + (c & 63), p.x_bytes + done * kBlockK * 2, m, 0);
          done += 64 >> m;
        }
      };
      enter(pair);
      int unit = pair, s = turn, round = 0;
      for (int kb = turn;; s += kProducers, kb += kProducers) {
        while (s >= p.stages) { s -= p.stages; ++round; }
        if (kb >= n_kb) {
          do { kb -= n_kb; unit += n_pairs; } while (kb >= n_kb);
          if (unit >= p.units) break;
          enter(unit);
        }
        const uint32_t fb = full0 + 8 * s, dst = smem0 + s * p.stage_bytes;
        if (round > 0) {
          if (!mbar_wait(empty0 + 8 * s, (uint32_t)(round - 1) & 1u, abort_flag, p.wait_limit_ns)) { ok = false; break; }
          if (!waited) pdl_wait();
          waited = true;
        }
        if (leader) mbar_expect_tx(fb, bytes);
        if (round > 0) tma_load_2d_pair(dst, &tmX, fb, kb * kBlockK, x_row);
        for (int i = 0; i < n_box; ++i) {
          const int4 w = box[i];
          tma_load_2d_pair(dst + w.y, &tmW.by_rows[w.z], fb, 0, w.x + kb * 128);
        }
      }
      if (!ok) {
        *abort_flag = 1;
        raise_word(p.err_flag, 1);
        drain(s + round * p.stages, turn, kProducers);
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer (the even CTA, for both)
    // One lane, elected once, walks the whole loop: four MMAs, a commit and a wait then take 250 clocks; with an election in each
    // turn 530.
    if (leader && elect_one()) {
      // M = 256 rows of both CTAs; N = the features of one MMA, half of them from each CTA's stage
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(256 >> 4) << 24);
      const uint32_t idesc0 = idesc | ((uint32_t)((kWide ? 256 : p.n0) >> 3) << 17), idesc1 = idesc | ((uint32_t)(p.n1 >> 3) << 17);
      bool ok = true;
      const uint32_t full0 = smem_addr(full_bar), empty0 = smem_addr(empty_bar);
      const uint64_t xdesc0 = make_smem_desc(smem_addr(smem)), wdesc0 = make_smem_desc(smem_addr(smem) + p.x_bytes);
      const int stage_units = p.stage_bytes >> 4;      // (the address field of a descriptor counts 16-byte units)
      int s = 0, nth = 0;                    // stage; tiles so far
      uint32_t phase = 0;
      for (int unit = pair; unit < p.units && ok; unit += n_pairs, ++nth) {
        const int buf = nth % p.bufs;
        if (nth >= p.bufs) {
          ok = mbar_wait(smem_addr(&acc_empty[buf]), (uint32_t)((nth / p.bufs) & 1) ^ 1u, abort_flag, p.wait_limit_ns);
          if (!ok) break;
          tc_fence_after();
        }
        for (int split = 0; split < p.splits && ok; ++split) {
          const uint32_t tmem_d = tmem_base + (uint32_t)((buf * p.splits + split) * acc_cols);
          const int kb0 = (int)((long long)split * n_kb / p.splits), kb1 = (int)((long long)(split + 1) * n_kb / p.splits);
          for (int kb = kb0; kb < kb1; ++kb) {
            ok = mbar_wait(full0 + 8 * s, phase, abort_flag, p.wait_limit_ns);
            if (!ok) break;
            const uint32_t at = (uint32_t)(s * stage_units);
            const uint64_t xd = xdesc0 + at, wd = wdesc0 + at;
#pragma unroll
            for (int k = 0; k < kBlockK / 16; ++k) tc_mma_bf16_pair(tmem_d, xd + 2 * k, wd + 2 * k, idesc0, (uint32_t)(((kb - kb0) | k) != 0));
            if constexpr (kWide) {
#pragma unroll
              for (int k = 0; k < kBlockK / 16; ++k)
                tc_mma_bf16_pair(tmem_d + 256u, xd + 2 * k, wd + (128 * kBlockK * 2 >> 4) + 2 * k, idesc1, (uint32_t)(((kb - kb0) | k) != 0));
            }
            tc_commit_pair(empty0 + 8 * s);
            if (++s == p.stages) { s = 0; phase ^= 1u; }
          }
        }
        if (ok) tc_commit_pair(smem_addr(&acc_full[buf]));
      }
      if (!ok) { *abort_flag = 1; raise_word(p.err_flag, 2); }
    }
    __syncwarp();
  } else {
    // ------------------------------------------------------------------ epilogue
    const int quad = warp & 3, group = (warp - 2) >> 2;
    pdl_wait();
    bool ok = true;
    int nth = 0;
    uint8_t* trans = sTrans + (warp - 2) * kTransWarp<kEpi>;
    for (int unit = pair; unit < p.units; unit += n_pairs, ++nth) {
      const int c0 = unit * p.cpu, n = min(p.cpu, p.couples - c0);
      // this warp's rows: [row0, row0 + 32) as far as the CTA's half goes
      const int row0 = crank * p.half + quad * 32, row = row0 + lane;
      const int row_end = min(p.R, (crank + 1) * p.half);
      const bool live = row < row_end, any = row0 < row_end;
      float inv = 1.f;
      if (live) {                            // RMSNorm, consumer side: the producers' per-tile sums in slot order
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
      int pos = 0;
      unsigned long long kv_row = 0;
      unsigned cache_mask = 0;
      if (kEpi == EPI_QKV) {
        const QkvOut& o = p.qkv;
        const int safe = live ? row : 0, slot = safe / o.map.rows_per_seq, lr = safe - slot * o.map.rows_per_seq;
        pos = o.map.pos0 + lr % o.map.T;
        const bool to_cache = live && lr < o.cache_rows;
        kv_row = to_cache ? (size_t)seq_of_slot(o.map, slot) * o.cache_seq_stride + (size_t)pos * o.kv_pos_stride : 0;
        cache_mask = __ballot_sync(0xffffffffu, to_cache);
      }
      // The angles of a piece, four rows to a lane of the transposed form: asked for ahead, one piece at a time.
      float4 cs[4][2];
      auto angles = [&](int c) {
        const int f = (c0 + c + 4 * (lane & 3)) & 63;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int r_pos = __shfl_sync(0xffffffffu, pos, 8 * i + (lane >> 2));
          const float4* a = reinterpret_cast<const float4*>(p.qkv.rope + (size_t)r_pos * 64 + f);
          cs[i][0] = a[0];
          cs[i][1] = a[1];
        }
      };
      if (kEpi == EPI_QKV && any) angles(16 * group);
      const int buf = nth % p.bufs;
      if (ok) ok = mbar_wait(smem_addr(&acc_full[buf]), (uint32_t)((nth / p.bufs) & 1), abort_flag, p.wait_limit_ns);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) continue;
      tc_fence_after();
      const uint32_t taddr = tmem_base + (uint32_t)(buf * p.splits * acc_cols) + ((uint32_t)(quad * 32) << 16);
      // pieces of 16 couples: columns [at, +16) and their partners `apart` columns on
#pragma unroll 1
      for (int c = 16 * group; c < n && any; c += 16 * kG) {
        const int at = 2 * c < p.n0 ? c : p.n0 + c - p.n0 / 2, apart = 2 * c < p.n0 ? p.n0 / 2 : p.n1 / 2;
        float x1[16], x2[16];
        {
          uint32_t r1[16], r2[16];
          tmem_ld16_issue(taddr + at, r1);
          tmem_ld16_issue(taddr + at + apart, r2);
          tmem_ld_wait(r1);
          tmem_ld_wait(r2);
#pragma unroll
          for (int j = 0; j < 16; ++j) { x1[j] = __fmul_rn(__uint_as_float(r1[j]), inv); x2[j] = __fmul_rn(__uint_as_float(r2[j]), inv); }
        }
        if (kEpi == EPI_QKV) {
#pragma unroll
          for (int j = 0; j < 16; ++j) { x1[j] = __fadd_rn(0.f, x1[j]); x2[j] = __fadd_rn(0.f, x2[j]); }
#pragma unroll 1
          for (int split = 1; split < p.splits; ++split) {
            uint32_t r1[16], r2[16];
            tmem_ld16_issue(taddr + split * acc_cols + at, r1);
            tmem_ld16_issue(taddr + split * acc_cols + at + apart, r2);
            tmem_ld_wait(r1);
            tmem_ld_wait(r2);
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              x1[j] = __fadd_rn(x1[j], __fmul_rn(__uint_as_float(r1[j]), inv));
              x2[j] = __fadd_rn(x2[j], __fmul_rn(__uint_as_float(r2[j]), inv));
            }
          }
          // chunks 0-3 and 4-7 of a buffer row: the 16 features and their partners; then four lanes to a row
          const QkvOut& o = p.qkv;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            *trans_at(trans, lane, q) = make_float4(x1[4 * q], x1[4 * q + 1], x1[4 * q + 2], x1[4 * q + 3]);
            *trans_at(trans, lane, 4 + q) = make_float4(x2[4 * q], x2[4 * q + 1], x2[4 * q + 2], x2[4 * q + 3]);
          }
          __syncwarp();
          const int cj = c + 4 * (lane & 3), j = c0 + cj;                // this lane's first couple
          const int head = j >> 6, f = j & 63;
          const bool is_q = head < o.H, is_k = !is_q && head < o.H + o.Hkv;
          const int kvh = head - o.H - (is_k ? 0 : o.Hkv);
          uint2 lo[4], hi[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int src = 8 * i + (lane >> 2);
            float4 u = *trans_at(trans, src, lane & 3), w = *trans_at(trans, src, 4 + (lane & 3));
            if (is_q || is_k) {
              rope_pair(u.x, w.x, cs[i][0].x, cs[i][0].y); rope_pair(u.y, w.y, cs[i][0].z, cs[i][0].w);
              rope_pair(u.z, w.z, cs[i][1].x, cs[i][1].y); rope_pair(u.w, w.w, cs[i][1].z, cs[i][1].w);
            }
            lo[i] = make_uint2(pack2(u.x, u.y), pack2(u.z, u.w));
            hi[i] = make_uint2(pack2(w.x, w.y), pack2(w.z, w.w));
          }
          angles(c + 16 * kG);                                      // (of a piece there may not be: rows of the table all the same)
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int src = 8 * i + (lane >> 2), r = row0 + src;
            const unsigned long long r_kv = __shfl_sync(0xffffffffu, kv_row, src);
            if (r >= row_end || cj >= n) continue;
            auto put = [&](bf16* dst) {
              *reinterpret_cast<uint2*>(dst + f) = lo[i];
              *reinterpret_cast<uint2*>(dst + 64 + f) = hi[i];
            };
            if (is_q) {
              put(o.q + ((size_t)r * o.H + head) * 128);
            } else {
              if (o.local_k) put((is_k ? o.local_k : o.local_v) + ((size_t)r * o.Hkv + kvh) * 128);
              if ((cache_mask >> src) & 1u) put((is_k ? o.cache_k : o.cache_v) + (size_t)r_kv + (size_t)kvh * o.kv_head_stride);
            }
          }
          __syncwarp();
        } else {
          uint32_t a[8];
#pragma unroll
          for (int j = 0; j < 16; j += 2) {
            float a0, a1;
            swiglu2(x1[j], x1[j + 1], x2[j], x2[j + 1], a0, a1);
            a[j >> 1] = pack2(a0, a1);
          }
          // 32 bytes a row in the buffer (two chunks, exchanged in every second four rows); then two lanes to a row
          uint4* t = reinterpret_cast<uint4*>(trans);
          const int sw = (lane >> 2) & 1;
          t[2 * lane + sw] = make_uint4(a[0], a[1], a[2], a[3]);
          t[2 * lane + (1 ^ sw)] = make_uint4(a[4], a[5], a[6], a[7]);
          __syncwarp();
          const int cj = c + 8 * (lane & 1);
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const int src = 16 * i + (lane >> 1), r = row0 + src;
            const uint4 v = t[2 * src + ((lane & 1) ^ ((src >> 2) & 1))];
            if (r < row_end && cj < n) *reinterpret_cast<uint4*>(p.act + (size_t)r * p.act_pitch + c0 + cj) = v;
          }
          __syncwarp();
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(map_to_rank(smem_addr(&acc_empty[buf]), 0u));
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

template <int kEpi, bool kWide>
int launch(cudaStream_t st, const GemmArgs& g, WaveParams p, int dev) {
  constexpr int fixed = kTransBytes<kEpi> + kListBytes + kBarBytes + 1024;
  // (an MMA reads 128 rows of A whatever `half` is: what lies behind the last stage has to be there)
  const int behind = p.stage_bytes < 128 * kBlockK * 2 ? 128 * kBlockK * 2 - p.stage_bytes : 0;
  p.stages = (kSmemMax - fixed - behind) / p.stage_bytes;
  if (p.stages > kMaxStages) p.stages = kMaxStages;
  alignas(64) CUtensorMap tmX;
  alignas(64) WeightMaps tmW;
  const uint64_t w_rows = (uint64_t)gemm_tiles(g.N) * ((g.K + kBlockK - 1) / kBlockK) * 128;
  if (encode_tmap_bf16_2d(&tmX, g.x, (uint64_t)g.R, (uint64_t)g.K, (uint64_t)g.x_pitch, (uint32_t)p.half) != 0) return -4;
  for (int i = 0; i < 4; ++i)
    if (encode_tmap_bf16_2d(&tmW.by_rows[i], g.w, w_rows, kBlockK, kBlockK, 64u >> i) != 0) return -4;
  static PerDevice<bool> attr_set = {};             // the shared-memory opt-in
  if (!attr_set[dev]) {
    if (cudaFuncSetAttribute(gemm_wave_kernel<kEpi, kWide>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax) != cudaSuccess) return -4;
    attr_set[dev] = true;
  }
  const int smem = p.stages * p.stage_bytes + fixed + behind;
  const dim3 grid(2 * (p.units < kSms / 2 ? p.units : kSms / 2));
  return launch_pdl_cluster(gemm_wave_kernel<kEpi, kWide>, grid, dim3(kThreads<kEpi>), (size_t)smem, st, 2u, tmX, tmW, p) == cudaSuccess ? 0 : -4;
}

int unit_columns(int cpu) { return 2 * ((cpu + 15) & ~15); }

}  // namespace

bool gemm_wave_fits(int N, int R, int splits) { return N % 128 == 0 && R <= 256 && splits * unit_columns(wave_share(N).couples) <= 512; }

int launch_gemm_wave(cudaStream_t st, const GemmArgs& g) {
  if ((g.x_pitch % 8) || (((uintptr_t)g.x) & 15) || (((uintptr_t)g.w) & 15) || !g.w_tiled || !g.sq || g.sq_count < 1 || g.norm_dim < 1) return -2;
  if (g.R < 1 || g.K < 1 || g.splits < 1 || g.splits > (g.K + kBlockK - 1) / kBlockK || !gemm_wave_fits(g.N, g.R, g.splits)) return -2;
  if (g.epi == EPI_QKV ? (!g.qkv || g.qkv->hd != 128) : (g.epi != EPI_SWIGLU || g.splits != 1 || !g.act)) return -2;
  WaveParams p{};
  p.R = g.R; p.K = g.K; p.couples = g.N / 2; p.splits = g.splits;
  p.half = ((g.R + 1) / 2 + 7) & ~7;
  const int dev = device_slot();
  if (dev < 0) return -4;
  p.cpu = wave_share(g.N).couples;
  p.units = (p.couples + p.cpu - 1) / p.cpu;
  const int cols = unit_columns(p.cpu);
  p.n0 = p.cpu < 128 ? cols : 256;
  p.n1 = cols - p.n0;
  p.bufs = 512 / (p.splits * cols) < kMaxBufs ? 512 / (p.splits * cols) : kMaxBufs;
  p.x_bytes = p.half * kBlockK * 2;
  p.stage_bytes = p.x_bytes + cols / 2 * kBlockK * 2;
  p.wait_limit_ns = g.wait_limit_ns > 0 ? g.wait_limit_ns : kWaitLimitNs;
  p.err_flag = g.err_flag;
  p.sq = g.sq; p.sq_count = g.sq_count; p.sq_stride = g.sq_stride; p.norm_dim = g.norm_dim; p.norm_eps = g.norm_eps;
  p.act = g.act; p.act_pitch = g.act_pitch;
  if (g.qkv) p.qkv = *g.qkv;
  if (p.n1 > 0) return g.epi == EPI_QKV ? launch<EPI_QKV, true>(st, g, p, dev) : launch<EPI_SWIGLU, true>(st, g, p, dev);
  return g.epi == EPI_QKV ? launch<EPI_QKV, false>(st, g, p, dev) : launch<EPI_SWIGLU, false>(st, g, p, dev);
}

}  // namespace ssd
