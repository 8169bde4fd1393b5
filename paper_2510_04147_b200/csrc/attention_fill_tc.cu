// Bidirectional attention of the cache-fill forward (prefill of the prompts, refresh of the dual cache) on the
// tcgen05 tensor cores, head dimension 128: every query row attends, without a mask, to all cached keys of its
// sequence, the rows themselves among them.
//
// One CTA per (256 query rows, head, sequence): two query tiles of 128 rows share every K/V tile.  Per key tile of 128
//     S_i = Q_i K^T       (both operands from shared memory, 128 fp32 columns of tensor memory per query tile)
//     P_i = 2^(S_i - m)   (a warpgroup per query tile: a thread owns a row, its 128 scores stay in registers; P goes
//                          back as bf16 into the first half of S_i's columns)
//     O_i += P_i V        (A operand from tensor memory, V as stored, [key][hd])
// One warp issues all MMAs in the order PV_0(j), S_0(j+1), PV_1(j), S_1(j+1): while one warpgroup is in its
// exponentials, the tensor core works for the other.  (Two query tiles that take turns with the tensor core, P over the scores'
// columns and the late rescale below are the published scheme of FlashAttention-4.)  PV starts when the first 64 keys' P is written.  A warp asks the tensor-map engine for the K and V tiles two
// ahead; keys past the end of the sequence are out of the map's bounds and arrive as zeros.
//
// The bounds are the tensor core and the special-function unit alike: a query tile x key tile is 1024 clocks of MMA (two
// contractions of 128 x 128 x 128) and 16384 exponentials at 16 a clock.  So a row rescales its output only when its
// maximum has grown by more than 8 (a factor of 256 in the weights; the sums are fp32 and the quotient O / l does not
// depend on the reference point), which leaves a rescale in the first few tiles of a row.  Whether a row does so depends
// on the row alone.
//
// Per pair of query tiles and key tile 3500 clocks were measured (clock64) where 2048 are the bound: a warpgroup takes 210 to
// read its scores, 240 for the maximum, 1370 for exponentials and P, then waited 1280 for PV and the next S behind it, and the
// MMA warp was idle for 720.  Issuing PV in two halves takes half of it out of that wait, and registers shifted from the
// warps that need few to the softmax threads take out nearly all of their spills (12 bytes of stores are left with one query tile, 48
// with two): 512 tokens 16.7 -> 15.0 us alone, dream's 1024 43.5 ->
// 39.3, eight times 509 73 -> 71.  4096 tokens (880 TFLOP/s at full clocks) run under the power cap, 290 to 330 us before and
// 270 to 310 now, and took 1900 in the mma.sync form with its merge pass.  Taking 2 to 4 of 8 exponentials to the FMA pipe (a
// polynomial on packed pairs) gave nothing more.
#include "attn_common.cuh"

#include <cuda.h>

namespace ssd {
namespace {

using namespace attn;

constexpr int kHD = 128;
constexpr int kTile = 128;                         // rows of a query tile, keys of a key tile
constexpr int kHalfBytes = kTile * 128;            // one 64-column half of a tile
constexpr int kTileBytes = 2 * kHalfBytes;
constexpr int kStages = 2;                         // K and V stages
constexpr int kThreads = 384;                      // warps 0-3, 4-7: softmax of query tile 0, 1; warp 8: MMA; warp 9: copies
// Registers: the third warpgroup gives up what the softmax threads take (a row's 128 scores and the exponentials in flight).
constexpr int kRegsSoftmax = 208, kRegsOther = 80;
constexpr unsigned long long kWaitLimitNs = 2000000000ull;
constexpr float kRescaleStep = 8.f;                // log2 growth of a row's maximum that triggers a rescale

__device__ __forceinline__ unsigned long long gtimer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
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
// bounded: false when the limit expired or another thread of the CTA gave up
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort) {
  unsigned long long t0 = 0;
  for (uint32_t spins = 1;; ++spins) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((spins & 255u) == 0) {
      if (*abort) return false;
      const unsigned long long now = gtimer_ns();
      if (t0 == 0) t0 = now;
      else if (now - t0 > kWaitLimitNs) { *abort = 1; return false; }
    }
  }
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
      ::"r"(dst), "l"((unsigned long long)map), "r"(bar), "r"(c0), "r"(c1) : "memory");
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1, int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
      ::"r"(dst), "l"((unsigned long long)map), "r"(bar), "r"(c0), "r"(c1), "r"(c2) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// 128-byte swizzle: rows 128 B apart inside an 8-row group, groups `sbo` apart; `lbo`: distance between the two
// 64-element halves of the contiguous dimension (MN-major form)
__device__ __forceinline__ uint64_t make_desc(uint32_t saddr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
  uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)((lbo_bytes >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo_bytes >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}
__device__ __forceinline__ void tc_mma_ss(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n.reg .pred p;\n"
      "setp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
      ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
// A operand from tensor memory: lane = row, a 32-bit column = two consecutive K elements
__device__ __forceinline__ void tc_mma_ts(uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n.reg .pred p;\n"
      "setp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n"
      ::"r"(tmem_d), "r"(tmem_a), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
// 32 consecutive columns of the thread's lane, requested only
__device__ __forceinline__ void tmem_ld32_issue(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
// (keeps the compiler from reading the registers of a request above the wait)
__device__ __forceinline__ void keep32(uint32_t* r) {
  asm volatile("" : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                    "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]),
                    "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]),
                    "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]));
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};\n"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]) : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// kQ query tiles of 128 rows per CTA
template <int kQ>
__global__ void __launch_bounds__(kThreads, 1)
attn_fill_tc_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                    const __grid_constant__ CUtensorMap tmV, bf16* out, int H, int Hkv, int T, int n_keys, int seq_base,
                    int* err_flag, float scale_log2) {
  extern __shared__ uint8_t smem_dyn[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~(uintptr_t)1023);
  uint8_t* sQ = smem;
  uint8_t* sK = sQ + kQ * kTileBytes;
  uint8_t* sV = sK + kStages * kTileBytes;
  uint64_t* bars = reinterpret_cast<uint64_t*>(sV + kStages * kTileBytes);
  const uint32_t bar_q = smem_u32(bars), bar_kf = bar_q + 8, bar_ke = bar_kf + 8 * kStages, bar_vf = bar_ke + 8 * kStages,
                 bar_ve = bar_vf + 8 * kStages, bar_s = bar_ve + 8 * kStages, bar_p = bar_s + 8 * kQ, bar_o = bar_p + 16 * kQ;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 1 + 4 * kStages + 4 * kQ);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  pdl_launch_dependents();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int h = blockIdx.y, slot = blockIdx.z, q0 = blockIdx.x * kQ * kTile;
  const int kvh = h / (H / Hkv);
  const size_t grow0 = (size_t)slot * T + q0;
  const int n_kt = (n_keys + kTile - 1) / kTile;

  if (tid == 0) {
    mbar_init(bar_q, 1);
    for (int s = 0; s < kStages; ++s) {
      mbar_init(bar_kf + 8 * s, 1); mbar_init(bar_ke + 8 * s, 1);
      mbar_init(bar_vf + 8 * s, 1); mbar_init(bar_ve + 8 * s, 1);
    }
    for (int i = 0; i < kQ; ++i) { mbar_init(bar_s + 8 * i, 1); mbar_init(bar_p + 16 * i, 4); mbar_init(bar_p + 16 * i + 8, 4); mbar_init(bar_o + 8 * i, 1); }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 8) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(256u * kQ) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;           // S_i (P_i in its first half) at 128 i, O_i at 128 (kQ + i)
  pdl_wait();
  bool ok = true;

  if (warp >= 8) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsOther));
    if (warp == 9) {
      // ------------------------------------------------------------------ copies
      if (elect_one()) {
        mbar_expect_tx(bar_q, (uint32_t)(kQ * kTileBytes));
        for (int i = 0; i < kQ; ++i)
          for (int half = 0; half < 2; ++half)
            tma_load_2d(smem_u32(sQ) + i * kTileBytes + half * kHalfBytes, &tmQ, bar_q, h * kHD + half * 64, (int)grow0 + i * kTile);
        const int plane = (seq_base + slot) * Hkv + kvh;
        int n_k = 0, n_v = 0;                            // tiles asked for
        for (int j = 0; j < n_kt && ok; ++j) {
          const int s = j % kStages;
          const uint32_t ph = (uint32_t)((j / kStages) & 1) ^ 1u;
          if (j >= kStages) ok = mbar_wait(bar_ke + 8 * s, ph, abort_flag);
          if (!ok) break;
          mbar_expect_tx(bar_kf + 8 * s, (uint32_t)kTileBytes);
          for (int half = 0; half < 2; ++half)
            tma_load_3d(smem_u32(sK) + s * kTileBytes + half * kHalfBytes, &tmK, bar_kf + 8 * s, half * 64, j * kTile, plane);
          ++n_k;
          if (j >= kStages) ok = mbar_wait(bar_ve + 8 * s, ph, abort_flag);
          if (!ok) break;
          mbar_expect_tx(bar_vf + 8 * s, (uint32_t)kTileBytes);
          for (int half = 0; half < 2; ++half)
            tma_load_3d(smem_u32(sV) + s * kTileBytes + half * kHalfBytes, &tmV, bar_vf + 8 * s, half * 64, j * kTile, plane);
          ++n_v;
        }
        if (!ok) {                                       // let the copies in flight land before the shared memory goes away
          *abort_flag = 0;                               // (bounded again; the error word is raised below)
          mbar_wait(bar_q, 0, abort_flag);
          for (int j = n_k > kStages ? n_k - kStages : 0; j < n_k; ++j) mbar_wait(bar_kf + 8 * (j % kStages), (uint32_t)((j / kStages) & 1), abort_flag);
          for (int j = n_v > kStages ? n_v - kStages : 0; j < n_v; ++j) mbar_wait(bar_vf + 8 * (j % kStages), (uint32_t)((j / kStages) & 1), abort_flag);
          *abort_flag = 1;
        }
      }
    } else if (warp == 8) {
      // ------------------------------------------------------------------ MMA issuer
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(128 >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
      const uint32_t idesc_pv = idesc | (1u << 16);                // B is MN-major: V as stored
      // (the address field of a descriptor counts 16-byte units)
      const uint64_t qdesc = make_desc(smem_u32(sQ), 16, 1024), kdesc = make_desc(smem_u32(sK), 16, 1024), vdesc = make_desc(smem_u32(sV), kHalfBytes, 1024);
      // (one lane, elected once, walks the loop: an election in each step costs more than the MMAs' issue)
      if (elect_one()) {
        auto issue_s = [&](int i, int j) {
          const uint64_t qd = qdesc + (uint32_t)(i * (kTileBytes >> 4)), kd = kdesc + (uint32_t)((j % kStages) * (kTileBytes >> 4));
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const uint32_t off = (uint32_t)((k >> 2) * kHalfBytes + (k & 3) * 32) >> 4;
            tc_mma_ss(tmem_base + 128u * i, qd + off, kd + off, idesc, (uint32_t)(k != 0));
          }
          tc_commit(bar_s + 8 * i);
          if (i == kQ - 1) tc_commit(bar_ke + 8 * (j % kStages));
        };
        auto issue_pv = [&](int i, int j, int half) {              // keys [64 half, +64) of the tile
          const uint64_t vd = vdesc + (uint32_t)((j % kStages) * (kTileBytes >> 4));
#pragma unroll
          for (int k = 0; k < 4; ++k)
            tc_mma_ts(tmem_base + 128u * (kQ + i), tmem_base + 128u * i + 8u * (4 * half + k), vd + (uint32_t)(2 * (4 * half + k) * 64), idesc_pv,
                      (uint32_t)((j | half | k) != 0));
          if (half == 1 && i == kQ - 1) tc_commit(bar_ve + 8 * (j % kStages));
          if (half == 1 && j == n_kt - 1) tc_commit(bar_o + 8 * i);
        };
        auto wait = [&](uint32_t bar, uint32_t parity) -> bool { return mbar_wait(bar, parity, abort_flag); };
        ok = wait(bar_q, 0) && wait(bar_kf, 0);
        tc_fence_after();
        if (ok)
          for (int i = 0; i < kQ; ++i) issue_s(i, 0);
        for (int j = 0; j < n_kt && ok; ++j) {
          ok = wait(bar_vf + 8 * (j % kStages), (uint32_t)((j / kStages) & 1));
#pragma unroll
          for (int i = 0; i < kQ; ++i) {
#pragma unroll
            for (int half = 0; half < 2; ++half) {
              if (ok) ok = wait(bar_p + 16 * i + 8 * half, (uint32_t)(j & 1));
              if (!ok) break;
              tc_fence_after();
              issue_pv(i, j, half);
            }
            if (!ok) break;
            if (j + 1 < n_kt) {
              if (i == 0) {
                ok = wait(bar_kf + 8 * ((j + 1) % kStages), (uint32_t)(((j + 1) / kStages) & 1));
                if (!ok) break;
                tc_fence_after();
              }
              issue_s(i, j + 1);             // (in order behind O += P V, which still reads P from the same columns)
            }
          }
        }
      }
      __syncwarp();
    }
  } else if ((warp >> 2) < kQ) {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsSoftmax));
    // ------------------------------------------------------------------ softmax (log2 domain): a thread owns a row
    const int i = warp >> 2;
    const uint32_t lane_addr = (uint32_t)((warp & 3) * 32) << 16;
    const uint32_t tS = tmem_base + 128u * i + lane_addr, tO = tmem_base + 128u * (kQ + i) + lane_addr;
    float m_ref = -INFINITY, l = 0.f;                // reference point of the weights; sum of the weights
#pragma unroll 1
    for (int j = 0; j < n_kt; ++j) {
      ok = mbar_wait(bar_s + 8 * i, (uint32_t)(j & 1), abort_flag);
      ok = __all_sync(0xffffffffu, ok ? 1 : 0) != 0;
      if (!ok) break;
      tc_fence_after();
      uint32_t s[128];
#pragma unroll
      for (int c = 0; c < 4; ++c) tmem_ld32_issue(tS + 32 * c, s + 32 * c);
      tmem_ld_wait();
#pragma unroll
      for (int c = 0; c < 4; ++c) { keep32(s + 32 * c); asm volatile("" : "+r"(s[32 * c + 30]), "+r"(s[32 * c + 31])); }
      const int left = n_keys - j * kTile;
      if (left < kTile) {                            // keys past the end
#pragma unroll
        for (int c = 0; c < kTile; ++c)
          if (c >= left) s[c] = 0xff800000u;         // -inf
      }
      float mx[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) mx[c] = __uint_as_float(s[c]);
#pragma unroll
      for (int c = 4; c < kTile; ++c) mx[c & 3] = fmaxf(mx[c & 3], __uint_as_float(s[c]));
      const float m_tile = __fmul_rn(fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])), scale_log2);
      const bool grow = m_tile > m_ref + kRescaleStep;           // (true on the first tile: m_ref = -inf)
      const float m_new = grow ? m_tile : m_ref;
      if (j > 0 && __any_sync(0xffffffffu, grow)) {
        // O so far was weighted against the old reference point.  (O += P V of the tile before is complete: this
        // tile's S was issued behind it.)
        const float corr = grow ? ex2(m_ref - m_new) : 1.f;
        l *= corr;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          uint32_t o[16];
          asm volatile(
              "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
              "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
              "tcgen05.wait::ld.sync.aligned;\n"
              : "=r"(o[0]), "=r"(o[1]), "=r"(o[2]), "=r"(o[3]), "=r"(o[4]), "=r"(o[5]), "=r"(o[6]), "=r"(o[7]),
                "=r"(o[8]), "=r"(o[9]), "=r"(o[10]), "=r"(o[11]), "=r"(o[12]), "=r"(o[13]), "=r"(o[14]), "=r"(o[15])
              : "r"(tO + 16 * c) : "memory");
#pragma unroll
          for (int k = 0; k < 16; ++k) o[k] = __float_as_uint(__uint_as_float(o[k]) * corr);
          tmem_st16(tO + 16 * c, o);
        }
      }
      m_ref = m_new;
      float sum[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        uint32_t packed[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) {
          const float p0 = ex2(__fmaf_rn(__uint_as_float(s[32 * c + 2 * k]), scale_log2, -m_ref));
          const float p1 = ex2(__fmaf_rn(__uint_as_float(s[32 * c + 2 * k + 1]), scale_log2, -m_ref));
          sum[k & 1] += p0;
          sum[2 + (k & 1)] += p1;
          packed[k] = pack_bf16(p0, p1);
        }
        tmem_st16(tS + 16 * c, packed);
        if (c == 1) {                                // the first half of the keys may go
          tmem_st_wait();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(bar_p + 16 * i);
        }
      }
      l += (sum[0] + sum[1]) + (sum[2] + sum[3]);
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_p + 16 * i + 8);
    }
    if (ok) {
      ok = mbar_wait(bar_o + 8 * i, 0, abort_flag);
      ok = __all_sync(0xffffffffu, ok ? 1 : 0) != 0;
      tc_fence_after();
    }
    if (ok) {
      const int r = i * kTile + (warp & 3) * 32 + lane;
      const float inv = 1.f / l;
      uint4* dst = reinterpret_cast<uint4*>(out + ((grow0 + r) * H + h) * kHD);
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        uint32_t o[32];
        tmem_ld32_issue(tO + 32 * c, o);
        tmem_ld_wait();
        keep32(o);
        asm volatile("" : "+r"(o[30]), "+r"(o[31]));
        if (q0 + r < T) {
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            uint32_t w[4];
#pragma unroll
            for (int k = 0; k < 4; ++k)
              w[k] = pack_bf16(__uint_as_float(o[8 * q + 2 * k]) * inv, __uint_as_float(o[8 * q + 2 * k + 1]) * inv);
            dst[4 * c + q] = make_uint4(w[0], w[1], w[2], w[3]);
          }
        }
        __syncwarp();
      }
    }
  }
  if (!ok) raise_word(err_flag, 7);
  tc_fence_before();
  __syncthreads();
  if (warp == 8)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(256u * kQ) : "memory");
}

template <int kQ>
int launch(cudaStream_t st, const AttnArgs& a, const CUtensorMap& tmQ, const CUtensorMap& tmK, const CUtensorMap& tmV) {
  const size_t smem = (size_t)(kQ + 2 * kStages) * kTileBytes + 1024 + 256;
  static PerDevice<bool> attr_set = {};             // the shared-memory opt-in
  const int dev = device_slot();
  if (dev < 0) return -4;
  if (!attr_set[dev]) {
    cudaFuncAttributes fa;
    if (cudaFuncSetAttribute(attn_fill_tc_kernel<kQ>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
        cudaFuncGetAttributes(&fa, attn_fill_tc_kernel<kQ>) != cudaSuccess)
      return -4;
    // the warpgroups' shares come out of what the block is launched with (the build refuses a compilation to fewer)
    if (fa.numRegs * kThreads < 256 * kRegsSoftmax + 128 * kRegsOther) return -4;
    attr_set[dev] = true;
  }
  const float scale_log2 = (1.0f / sqrtf((float)a.hd)) * 1.4426950408889634f;
  const int T = a.map.rows_per_seq;
  const dim3 grid((T + kQ * kTile - 1) / (kQ * kTile), a.H, a.n_seq_slots);
  return launch_pdl(attn_fill_tc_kernel<kQ>, grid, dim3(kThreads), smem, st, tmQ, tmK, tmV, a.out, a.H, a.Hkv, T, a.S, a.map.seq_base,
                    a.err_flag, scale_log2) == cudaSuccess ? 0 : -4;
}

}  // namespace

int launch_attention_fill_tc(cudaStream_t st, const AttnArgs& a) {
  if (a.hd != kHD || a.kv_pos_stride != (size_t)kHD || a.cache_seq_stride != a.kv_head_stride * (size_t)a.Hkv || a.map.seq_map ||
      !a.err_flag || a.cache_rows == 0)
    return -2;
  alignas(64) CUtensorMap tmQ, tmK, tmV;
  const uint64_t planes = (uint64_t)a.cache_rows * kHD / a.kv_head_stride;       // (sequence, kv head) pairs
  if (encode_tmap_bf16_2d(&tmQ, a.q, (uint64_t)a.R, (uint64_t)a.H * kHD, (uint64_t)a.H * kHD, kTile) != 0 ||
      encode_tmap_bf16_3d(&tmK, a.cache_k, kHD, (uint64_t)a.S, planes, kHD, a.kv_head_stride, kTile) != 0 ||
      encode_tmap_bf16_3d(&tmV, a.cache_v, kHD, (uint64_t)a.S, planes, kHD, a.kv_head_stride, kTile) != 0)
    return -4;
  // Two query tiles per CTA halve the K/V traffic and keep the tensor core busy under the exponentials; one where
  // that would leave most SMs without work.  The rows' bits are the same.
  const int T = a.map.rows_per_seq;
  const long long ctas = (long long)((T + 2 * kTile - 1) / (2 * kTile)) * a.H * a.n_seq_slots;
  return ctas >= 128 ? launch<2>(st, a, tmQ, tmK, tmV) : launch<1>(st, a, tmQ, tmK, tmV);
}

}  // namespace ssd
