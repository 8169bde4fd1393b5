// Shared-prefix bidirectional attention of the verification forward (Eq. 5) on the tcgen05 tensor cores, head
// dimension 128: a CTA walks the key tiles of (query tile, head, sequence) in one software pipeline.
//
// A query tile is up to 128 rows of whole nodes of one sequence, side by side; its keys are the node-local keys (tile
// 0, visibility per row: the row's own node, block-causal inside a chain of two blocks) followed by the cached keys in
// 128-key tiles (under the dual cache: the keys before the hole, then those behind it).  q, k and v come rotated and
// rounded from the projection's epilogue, so every tile is a tensor-map copy; rows past the end of the cached keys are
// out of the map's bounds and arrive as zeros, as do those past the end of a node.  A node's local keys take a power of two (16 or more) of key slots whatever
// its width: the tensor core takes keys in groups of 16 and the sums below are a binary tree over those, so a row's bits
// do not depend on which node of a tile it is in.
//
// Pipeline (two K stages, one P tile and two V stages in shared memory, two S accumulators and one O accumulator
// in tensor memory): while the threads run the softmax of tile u - row maximum, running (max, sum), P written to
// its tile - the tensor core already computes S = Q K^T of tile u+1.  K of tile u+2 is requested as soon as S of
// tile u is complete (its stage is free then), V of tile u+2 as soon as O += P V of tile u is.  O += P V of tile u is
// issued when P is complete and finishes under the next tile's softmax.  O is rescaled in tensor memory when a row's
// maximum grows.  With 128 query rows P goes to tensor memory instead, two tiles of it, and the softmax of a tile waits for the
// previous O += P V only when it has to rescale (425 clocks of a tile's 3400); smaller query tiles need P in every copy
// of a row, which shared memory gives them.  A query row is one TMEM lane shared by two threads (warps w and w+4), each owning half of the lane's
// columns; a tile of 32 or 64 rows is replicated to 128 lanes so that more threads share a row.  The order of the tiles
// and of every sum is fixed by the shapes alone, so a row's bits do not depend on what shares the forward with it.
//
// Few (head, sequence) pairs leave most SMs idle while one CTA walks all tiles: the tiles are then cut into parts, which the CTAs of
// a cluster share; they push (max, sum, unnormalised output) of a row to its owner through distributed shared memory, and the
// owner merges in part order.  With several query tiles a CTA of its own for every part is more CTAs than SMs, in two or three
// turns: then each CTA has two parts, or all of them, one after the other, and merges them in registers - the same parts and the
// same operations, so the same bits.  us a layer (live stream), a CTA for every part / now: 512 keys, 32 heads, 160 rows 27.8 /
// 21.3, 320 rows 45.2 / 27.2; 1024 keys, 28 heads, 192 rows 32.2 / 23.9, 320 rows 51.6 / 33.4; two sequences of 700 keys, 28 heads,
// 64 rows 17.8 / 11.4.
//
// Bound by the serial chain of a tile, not by bytes, except for long prefixes under small query tiles.  Of a 128-row tile's
// 3400 clocks (clock64 at each step, 4096 keys) the scores' maximum took 580, the wait for O += P V 425, exponentials, sums and P
// 1850, of which the special-function unit accounts for 1024.  The visibility test of every key (masked scores become -inf where
// they are loaded) and that wait are out of it.  Four threads to a row, or even and odd tiles in two streams, were no faster.  A
// thread keeps its scores in registers from the maximum to the exponentials, 64 of them under 128 rows; where the outputs of
// several parts in one CTA need those registers (kShared) it reads them twice, with 52 bytes of spills (with the scores kept
// as well, 28 heads at 320 rows 35 -> 49 us).  Read twice / kept, us a layer: 8 sequences of 509 keys, 96 rows each 50.5 / 42.1;
// one of 512 keys, 128 rows 17.3 / 14.7; 1024 keys, 28 heads, 128 rows 17.9 / 15.6.
// us a layer in the live stream, 32 heads (in brackets forms that summed and rotated the projection's split-K partials
// themselves; finishing q, k and v is a pass of 3 to 7 us below 161 rows and part of the projection from there on): one
// sequence, 512 keys, 32 / 64 / 128 rows 8.6 (15) / 10.3 (20) / 14.5 (32); 1536 keys, 128 rows 19.1 (43); 8 sequences of 512 keys,
// 32 rows each 25.0 (38); 4 of 4096 keys, 64 / 128 rows each 54.5 (83) / 78.9 (108); 3 sequences of 777 keys with nodes of 24 rows, which only the mma.sync form took, 25.0 (160).
#include "attn_common.cuh"

#include <cuda.h>
#include <string.h>

namespace ssd {

namespace {

using namespace attn;

constexpr int kHD = 128;
constexpr int kKeys = 128;                  // keys per tile
constexpr int kPipeThreads = 256;           // softmax threads: two per TMEM lane
constexpr int kPipeBlock = kPipeThreads + 64;   // + one warp that issues the MMAs + one that asks for the tile copies
constexpr int kHalfBytes = kKeys * 128;     // one 64-column half of a 128-row tile
constexpr int kTileBytes = 2 * kHalfBytes;  // a [128][128] bf16 tile
constexpr int kStagesK = 2, kStagesV = 2;      // + one P tile
constexpr int kMergePitch = kHD + 4;           // floats per row of the merge buffer
constexpr int kMergeRows = 232;                 // [entry][owned rows]: seven entries of 32 at most, rounded up
constexpr unsigned long long kPipeWaitLimitNs = 2000000000ull;

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
// bounded: false when the limit expired or another thread of the CTA gave up (`abort` set)
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort) {
  unsigned long long t0 = 0;
  for (uint32_t spins = 1;; ++spins) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((spins & 255u) == 0) {
      if (*abort) return false;
      const unsigned long long now = gtimer_ns();
      if (t0 == 0) t0 = now;
      else if (now - t0 > kPipeWaitLimitNs) { *abort = 1; return false; }
    }
  }
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// one box of a tensor map into shared memory; its bytes count on the mbarrier
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
__device__ __forceinline__ uint32_t map_to_rank(const void* p, uint32_t rank) {
  uint32_t out;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(out) : "r"(smem_u32(p)), "r"(rank));
  return out;
}
__device__ __forceinline__ void st_cluster_f32x4(uint32_t addr, float x, float y, float z, float w) {
  asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(x), "f"(y), "f"(z), "f"(w) : "memory");
}
__device__ __forceinline__ void st_cluster_f32x2(uint32_t addr, float x, float y) {
  asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(x), "f"(y) : "memory");
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// barrier 1 of the softmax threads (the MMA warp does not take part); returns the AND of `v` over them
__device__ __forceinline__ bool softmax_barrier_and(bool v) {
  uint32_t r;
  asm volatile(
      "{\n.reg .pred p, q;\n"
      "setp.ne.b32 q, %1, 0;\n"
      "bar.red.and.pred p, 1, 256, q;\n"
      "selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(r) : "r"((uint32_t)(v ? 1 : 0)) : "memory");
  return r != 0;
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// Operand tile with 128-byte swizzle: rows 128 B apart inside an 8-row group, groups `sbo` bytes apart;
// `lbo` is the distance between the two 64-element halves of the contiguous dimension for the MN-major form.
__device__ __forceinline__ uint64_t make_desc(uint32_t saddr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
  uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)((lbo_bytes >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo_bytes >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;                 // descriptor version of this architecture
  d |= (uint64_t)2 << 61;                 // 128-byte swizzle
  return d;
}
__device__ __forceinline__ void tc_mma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n.reg .pred p;\n"
      "setp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
      ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
// A operand in tensor memory: rows in the lanes, two bf16 of consecutive K to a column
__device__ __forceinline__ void tc_mma_bf16_ta(uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n.reg .pred p;\n"
      "setp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n"
      ::"r"(tmem_d), "r"(tmem_a), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
// 8 columns of the thread's lane; complete after tmem_st_wait
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&r)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};\n"
               ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]) : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// 16 consecutive columns of the thread's lane, requested only: several requests share one wait, and no register of
// a request may be read before tmem_ld_wait() and keep16() on it
__device__ __forceinline__ void tmem_ld16_issue(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
// (keeps the compiler from reading the registers of a request above the wait)
__device__ __forceinline__ void keep16(uint32_t* r) {
  asm volatile("" : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                    "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]));
}
// 16 consecutive columns of the thread's lane
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const float (&v)[16]) {
  uint32_t r[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) r[i] = __float_as_uint(v[i]);
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};\n"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}
// 2^x on the special-function unit (the one form used everywhere in this kernel, so that a key's probability has the
// same bits on every code path)
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// byte offset of 16-byte chunk `ch` (0..15 over 128 columns) of row `row` in a [half][128 rows][64] tile
__device__ __forceinline__ uint32_t tile_off(int row, int ch) {
  return (uint32_t)((ch >> 3) * kHalfBytes + row * 128 + (((ch & 7) ^ (row & 7)) << 4));
}

// Tiles of one (head, sequence): 0 = node-local, 1 .. n_a = cached keys [0, len_a), n_a + 1 .. = the len_b keys from
// cache row `row_b` on.  `npt` nodes per query tile, `t_pad` key slots per node in tile 0.  The tiles are cut into `n_parts` parts with
// a softmax of their own; a cluster of `n_ctas` CTAs has n_parts / n_ctas consecutive ones each.
struct PipeShape {
  int len_a, n_a, len_b, row_b, n_all, npt, t_pad, n_parts, n_ctas;
  __host__ __device__ int begin(int part) const { return part * n_all / n_parts; }      // first tile of a part
};

// Parts are merged one after the other, (((0, 1), 2), 3): sums and outputs of what came before and of the next part, each against
// the larger of the two maxima.  The same operations whether one thread has met both or they come from two CTAs.
struct Merge { float m, before, next; };                // new maximum, factors of the two sides
__device__ __forceinline__ Merge merge_of(float m_before, float m_next) {
  Merge g;
  g.m = fmaxf(m_before, m_next);
  const float use = g.m == -INFINITY ? 0.f : g.m;
  g.before = ex2(m_before - use);
  g.next = ex2(m_next - use);
  return g;
}
template <int N>
struct IntC { static constexpr int value = N; };
__device__ __forceinline__ float merged(const Merge& g, float before, float next) { return __fmaf_rn(next, g.next, __fmul_rn(before, g.before)); }

// kShared: a CTA has several parts (n_ctas < n_parts)
template <int QT, bool kShared>
__global__ void __launch_bounds__(kPipeBlock, 1)
attn_verify_pipe_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmLK,
                        const __grid_constant__ CUtensorMap tmLV, const __grid_constant__ CUtensorMap tmK,
                        const __grid_constant__ CUtensorMap tmV, const AttnArgs a, const PipeShape g, float scale_log2) {
  extern __shared__ uint8_t smem_dyn[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~(uintptr_t)1023);
  uint8_t* sQ = smem;                                   // [2][128][64] bf16
  uint8_t* sKs = sQ + kTileBytes;                       // kStagesK K tiles: a stage is free as soon as its S = Q K^T is complete
  uint8_t* sP = sKs + kStagesK * kTileBytes;            // P of the tile in work (bf16, the A operand of O += P V)
  uint8_t* sVs = sP + kTileBytes;                       // kStagesV V tiles
  float* sMax = reinterpret_cast<float*>(sVs + kStagesV * kTileBytes);      // 2 x [2 halves x 4 copies][128 rows] (tiles alternate)
  float* sSum = sMax + 2 * 8 * 128;                                         // 2 x [8 chunks of 16 keys][128 rows]
  // [0], [1] S ready (two accumulators), [2] Q landed, [3], [4] K stage landed, [5] P written and O rescaled, [6], [7] V stage
  // landed, [8], [9] accumulator read, [10], [11] O += P V complete (tiles alternate).  Pairs, so that no barrier can
  // complete a second phase before its waiter has seen the first: the second needs what the waiter does next.
  uint64_t* bars = reinterpret_cast<uint64_t*>(sSum + 2 * 8 * 128);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 12);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  constexpr int REP = 128 / QT;
  constexpr bool kTmemP = REP == 1;                     // P in tensor memory, two of them

  pdl_launch_dependents();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rank = blockIdx.x % g.n_ctas, h = blockIdx.x / g.n_ctas;        // the cluster spans x
  const int per_cta = g.n_parts / g.n_ctas, part0 = rank * per_cta;         // this CTA's parts
  const int rps = a.map.rows_per_seq, T = a.map.T;
  const int tile_rows = g.npt * T;                      // query rows of a tile: whole nodes
  const int q_tiles = (rps + tile_rows - 1) / tile_rows;
  const int qt = blockIdx.y % q_tiles, slot = blockIdx.y / q_tiles;
  const int kvh = h / (a.H / a.Hkv);
  const int lr0 = qt * tile_rows;
  const size_t grow0 = (size_t)slot * rps + lr0;
  const int rows_here = min(tile_rows, rps - lr0), nodes_here = rows_here / T, node0 = (int)grow0 / T;     // (nodes of all sequences)
  // this CTA's tiles: global tile index first + u, u = 0 .. n_tiles - 1
  const int first = g.begin(part0), n_tiles = g.begin(part0 + per_cta) - first;

  if (tid == 0) {
    for (int i = 0; i < 12; ++i) mbar_init(smem_u32(&bars[i]), (i == 5 || i == 8 || i == 9) ? kPipeThreads / 32 : 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == kPipeThreads / 32) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (first == 0 && tid < kPipeThreads) {
    // the V rows of tile 0 behind the nodes' slots: zero (a masked key's V row must be finite: 0 * NaN would poison O).  So are a
    // node's own unused slots: a plane of the map is one node, what its box takes beyond arrives as zeros
    for (int idx = nodes_here * g.t_pad * 16 + tid; idx < kKeys * 16; idx += kPipeThreads)
      *reinterpret_cast<uint4*>(sVs + tile_off(idx >> 4, idx & 15)) = make_uint4(0, 0, 0, 0);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  const uint32_t tmem_O = tmem_base + 256, tmem_P = tmem_base + 384;      // P: 64 columns each
  const uint32_t bar_s0 = smem_u32(&bars[0]), bar_q = smem_u32(&bars[2]), bar_k0 = smem_u32(&bars[3]), bar_p = smem_u32(&bars[5]);
  const uint32_t bar_v0 = smem_u32(&bars[6]), bar_sfree0 = smem_u32(&bars[8]), bar_o0 = smem_u32(&bars[10]);
  bool ok = true;
  float m_row = -INFINITY, l_row = 0.f;                 // softmax threads: running maximum and sum of the row

  if (warp == kPipeThreads / 32) {
    // ================================================================== MMA warp
    // Per tile u: S(u+1) = Q K(u+1)^T as soon as K(u+1) has landed and the softmax threads have read S(u-1), whose
    // accumulator it overwrites, then O += P(u) V(u) as soon as they report P(u) written and V(u) has landed.  The
    // tensor core runs the MMAs in issue order.
    // f32 accumulate, bf16 operands, N = 128, M = 128; bit 16: B is MN-major (V as stored, [key][hd])
    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(128 >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
    const uint32_t idesc_pv = idesc | (1u << 16);
    // (the address field of a descriptor counts 16-byte units)
    const uint64_t qdesc = make_desc(smem_u32(sQ), 16, 1024), kdesc = make_desc(smem_u32(sKs), 16, 1024);
    const uint64_t pdesc = make_desc(smem_u32(sP), 16, 1024), vdesc = make_desc(smem_u32(sVs), kHalfBytes, 1024);
    // One lane, elected once, walks the loop: an election and a vote in each step cost a few hundred clocks of every tile's chain.
    if (elect_one()) {
      auto issue_s = [&](int u) {                      // S[u & 1] = Q . K(u)^T: eight k16 steps over the head dimension
        const uint64_t kd = kdesc + (uint32_t)((u % kStagesK) * (kTileBytes >> 4));
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const uint32_t off = (uint32_t)((k >> 2) * kHalfBytes + (k & 3) * 32) >> 4;
          tc_mma_bf16(tmem_base + (uint32_t)(u & 1) * 128u, qdesc + off, kd + off, idesc, (uint32_t)(k != 0));
        }
        tc_commit(bar_s0 + 8u * (uint32_t)(u & 1));
      };
      auto wait = [&](uint32_t bar, uint32_t parity) -> bool { return mbar_wait(bar, parity, abort_flag); };
      ok = wait(bar_q, 0) && wait(bar_k0, 0);
      if (ok) {
        tc_fence_after();
        issue_s(0);
      }
      int next_part = part0 + 1, fresh_at = 0;             // tile whose O += P V starts a part's output
#pragma unroll 1
      for (int u = 0; u < n_tiles && ok; ++u) {
        const bool fresh = u == fresh_at;
        if (fresh) fresh_at = g.begin(next_part++) - first;
        if (u + 1 < n_tiles) {
          ok = wait(bar_k0 + 8u * (uint32_t)((u + 1) & 1), (uint32_t)(((u + 1) >> 1) & 1));
          if (ok && u >= 1) ok = wait(bar_sfree0 + 8u * (uint32_t)((u - 1) & 1), (uint32_t)(((u - 1) >> 1) & 1));
          if (!ok) break;
          tc_fence_after();
          issue_s(u + 1);
        }
        ok = wait(bar_p, (uint32_t)(u & 1)) && wait(bar_v0 + 8u * (uint32_t)(u & 1), (uint32_t)((u >> 1) & 1));
        if (!ok) break;
        tc_fence_after();
        // O (+)= P . V: eight k16 steps over the keys.  P is K-major (keys contiguous); V is used as stored,
        // [key][hd] = MN-major: 8-key groups 1024 B apart, the two 64-column halves 16 KB apart.
        const uint64_t vd = vdesc + (uint32_t)((u % kStagesV) * (kTileBytes >> 4));
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          if (kTmemP) tc_mma_bf16_ta(tmem_O, tmem_P + (uint32_t)(u & 1) * 64u + 8u * k, vd + (uint32_t)(2 * k * 64), idesc_pv, (uint32_t)(!fresh || k != 0));
          else tc_mma_bf16(tmem_O, pdesc + ((uint32_t)((k >> 2) * kHalfBytes + (k & 3) * 32) >> 4), vd + (uint32_t)(2 * k * 64), idesc_pv, (uint32_t)(!fresh || k != 0));
        }
        tc_commit(bar_o0 + 8u * (uint32_t)(u & 1));
      }
      if (!ok) raise_word(a.err_flag, 6);
    }
    __syncwarp();
  } else if (warp > kPipeThreads / 32) {
    // ================================================================== copy warp
    if (elect_one()) {
      // The cache is not written below the rows' own positions by any kernel of this forward, so cached tiles may be
      // requested before the dependency wait - unless the slot -> sequence map is only known on the device.
      const bool early = a.map.n_inline > 0 || a.map.seq_map == nullptr;
      auto ask_k = [&](int u) {
        const int gt = first + u;
        const uint32_t dst = smem_u32(sKs + (size_t)(u % kStagesK) * kTileBytes), bar = bar_k0 + 8u * (uint32_t)(u & 1);
        if (gt == 0) {
          mbar_arrive_expect_tx(bar, (uint32_t)(nodes_here * g.t_pad * 256));
          for (int n = 0; n < nodes_here; ++n)
            for (int half = 0; half < 2; ++half)
              tma_load_3d(dst + half * kHalfBytes + n * g.t_pad * 128, &tmLK, bar, kvh * kHD + half * 64, 0, node0 + n);
        } else {
          const int r = gt <= g.n_a ? (gt - 1) * kKeys : g.row_b + (gt - 1 - g.n_a) * kKeys;
          const int plane = seq_of_slot(a.map, slot) * a.Hkv + kvh;
          mbar_arrive_expect_tx(bar, (uint32_t)kTileBytes);
          tma_load_3d(dst, &tmK, bar, 0, r, plane);
          tma_load_3d(dst + kHalfBytes, &tmK, bar, 64, r, plane);
        }
      };
      auto ask_v = [&](int u) {
        const int gt = first + u;
        const uint32_t dst = smem_u32(sVs + (size_t)(u % kStagesV) * kTileBytes), bar = bar_v0 + 8u * (uint32_t)(u & 1);
        if (gt == 0) {
          mbar_arrive_expect_tx(bar, (uint32_t)(nodes_here * g.t_pad * 256));
          for (int n = 0; n < nodes_here; ++n)
            for (int half = 0; half < 2; ++half)
              tma_load_3d(dst + half * kHalfBytes + n * g.t_pad * 128, &tmLV, bar, kvh * kHD + half * 64, 0, node0 + n);
        } else {
          const int r = gt <= g.n_a ? (gt - 1) * kKeys : g.row_b + (gt - 1 - g.n_a) * kKeys;
          const int plane = seq_of_slot(a.map, slot) * a.Hkv + kvh;
          mbar_arrive_expect_tx(bar, (uint32_t)kTileBytes);
          tma_load_3d(dst, &tmV, bar, 0, r, plane);
          tma_load_3d(dst + kHalfBytes, &tmV, bar, 64, r, plane);
        }
      };
      // the first two tiles find free stages
      bool asked[2] = {false, false};
#pragma unroll
      for (int u = 0; u < 2; ++u)
        if (early && u < n_tiles && first + u > 0) { ask_k(u); ask_v(u); asked[u] = true; }
      pdl_wait();                          // the projection's q, k and v are complete from here on
      mbar_arrive_expect_tx(bar_q, (uint32_t)kTileBytes);
      for (int c = 0; c < REP; ++c)        // a query tile of 32 or 64 rows is replicated to 128 lanes
        for (int half = 0; half < 2; ++half)
          tma_load_2d(smem_u32(sQ) + half * kHalfBytes + c * QT * 128, &tmQ, bar_q, h * kHD + half * 64, (int)grow0);
#pragma unroll
      for (int u = 0; u < 2; ++u)
        if (u < n_tiles && !asked[u]) { ask_k(u); ask_v(u); }
      int u = 2;
#pragma unroll 1
      for (; u < n_tiles && ok; ++u) {
        ok = mbar_wait(bar_s0 + 8u * (uint32_t)(u & 1), (uint32_t)(((u - 2) >> 1) & 1), abort_flag);
        if (!ok) break;
        ask_k(u);
        ok = mbar_wait(bar_o0 + 8u * (uint32_t)(u & 1), (uint32_t)(((u - 2) >> 1) & 1), abort_flag);
        if (!ok) break;
        ask_v(u);
      }
      if (!ok) {
        // let the copies in flight land before the shared memory goes away (at most the last two tiles')
        raise_word(a.err_flag, 6);
        const unsigned long long t0 = gtimer_ns();
        for (int j = u >= 2 ? u - 2 : 0; j <= u && j < n_tiles; ++j)
          for (uint32_t bar : {bar_k0, bar_v0})
            while (!mbar_try_wait(bar + 8u * (uint32_t)(j & 1), (uint32_t)((j >> 1) & 1)) && gtimer_ns() - t0 < kPipeWaitLimitNs) {}
      }
    }
  } else {
    // ================================================================== softmax threads (log2 domain)
    // TMEM lane lt = copy `cw` of query row `row`; a copy covers the keys [cw * QT, +QT) of a tile and the lane's
    // two threads (hw = 0, 1) half of those each, in 16-key chunks.  A tile's row sum is ALWAYS formed from its
    // eight 16-key chunks as (((c0 + c1) + (c2 + c3)) + (c4 + c5)) + (c6 + c7), each chunk summed in key order,
    // whatever QT is.  The threads meet once per tile (exchange of the row maxima); everything else is handed
    // over through mbarriers, so that no thread waits for the MMA issue.
    constexpr int KPT = QT / 2;                           // keys of a tile per thread
    constexpr int NCH = KPT / 16;                         // 16-key chunks per thread
    // A thread takes its keys in one pass, its scores in registers from the maximum to the exponentials; in two, whose scores are
    // read again, where 128 rows meet parts that share the CTA.  (The output is rescaled 32 columns at a time.)
    constexpr int HK = kShared && KPT > 32 ? 32 : KPT, NP = KPT / HK, NCP = HK / 16, RK = KPT < 32 ? KPT : 32;
    const int lt = tid & 127, hw = tid >> 7;
    const int cw = lt / QT, row = lt % QT;
    const uint32_t lane_addr = (uint32_t)((warp & 3) * 32) << 16;   // warps w and w + 4 read TMEM lanes 32 (w & 3) ...
    const int col0 = cw * QT + hw * KPT;                  // first column (key of a tile) of this thread
    const int lr = lr0 + row;
    const bool row_live = row < rows_here;
    // node-local keys this row may see, as key slots of tile 0 (t_pad per node)
    const int loc_lo = min(row / T, nodes_here - 1) * g.t_pad;
    const int loc_hi = loc_lo + (a.map.chain_T0 > 0 && lr % T < a.map.chain_T0 ? a.map.chain_T0 : T);   // (finished block: not the next block)
    bool broke = false;                                   // the loop ended at the meeting point, for all threads alike
    // What the parts before the one in work came to, against their maximum: all of them (this CTA has the first part of all), or the
    // one before (a CTA further on, whose parts are merged by the rows' owner)
    float acc[KPT], acc_m = -INFINITY, acc_l = 0.f;
    bool have = false;
    auto part_done = [&](float m, float l) {              // the part whose output stands in tensor memory
      const bool fold = kShared && have;
      const Merge g2 = merge_of(acc_m, m);
#pragma unroll
      for (int ch = 0; ch < NCH; ++ch) {
        float v[16];
        tmem_ld16(tmem_O + lane_addr + col0 + ch * 16, v);
#pragma unroll
        for (int j = 0; j < 16; ++j) acc[ch * 16 + j] = fold ? merged(g2, acc[ch * 16 + j], v[j]) : v[j];
      }
      acc_l = fold ? merged(g2, acc_l, l) : l;
      acc_m = fold ? g2.m : m;
      have = true;
    };
    int next_part = part0 + 1, fresh_at = g.begin(next_part) - first;
    float corr_prev = 1.f;                                // rescale factor of the tile whose sum is still to be added
    auto tile_sum = [&](int u) -> float {                 // the row's sum over tile u, from the eight chunk sums
      const float* q = sSum + (u & 1) * 8 * 128 + row;
      return (((q[0 * 128] + q[1 * 128]) + (q[2 * 128] + q[3 * 128])) + (q[4 * 128] + q[5 * 128])) + (q[6 * 128] + q[7 * 128]);
    };
#pragma unroll 1
    for (int u = 0; u < n_tiles; ++u) {
      if (u >= 1 && u + 1 < n_tiles) {                      // S(u-1) has been read: its accumulator takes S(u+1)
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_sfree0 + 8u * (uint32_t)((u - 1) & 1));
      }
      // (here and below: a wait that expired is never forgotten, whatever a later one says - the error word depends on it)
      ok = ok && mbar_wait(bar_s0 + 8u * (uint32_t)(u & 1), (uint32_t)((u >> 1) & 1), abort_flag);
      tc_fence_after();
      ok = __all_sync(0xffffffffu, ok ? 1 : 0) != 0;        // the tensor-memory accesses below are warp-wide
      const uint32_t tmem_S = tmem_base + (uint32_t)(u & 1) * 128u;
      const int gt = first + u;
      const int key_lo = gt == 0 ? loc_lo : 0;
      const int key_hi = gt == 0 ? loc_hi : min(kKeys, gt <= g.n_a ? g.len_a - (gt - 1) * kKeys : g.len_b - (gt - 1 - g.n_a) * kKeys);
      const bool all_vis = key_lo <= col0 && key_hi >= col0 + KPT;   // every key of this thread's columns is visible
      // this thread's scores of the tile, a pass at a time: one round trip to tensor memory per pass
      uint32_t sv[HK];
      auto load_scores = [&](int pass) {
#pragma unroll
        for (int ch = 0; ch < NCP; ++ch) tmem_ld16_issue(tmem_S + lane_addr + col0 + pass * HK + ch * 16, &sv[ch * 16]);
        tmem_ld_wait();
#pragma unroll
        for (int ch = 0; ch < NCP; ++ch) keep16(&sv[ch * 16]);
        if (!all_vis) {                                     // a masked key: probability 2^-inf = 0
#pragma unroll
          for (int j = 0; j < HK; ++j) {
            const int key = col0 + pass * HK + j;
            if (key < key_lo || key >= key_hi) sv[j] = 0xff800000u;
          }
        }
      };
      float m_loc = -INFINITY;
      if (ok) {
#pragma unroll
        for (int pass = 0; pass < NP; ++pass) {
          load_scores(pass);
          float m = __uint_as_float(sv[0]);               // (scale > 0: the maximum of the products is the product of the maximum)
#pragma unroll
          for (int j = 1; j < HK; ++j) m = fmaxf(m, __uint_as_float(sv[j]));
          m_loc = fmaxf(m_loc, __fmul_rn(m, scale_log2));
        }
      } else {
#pragma unroll
        for (int j = 0; j < HK; ++j) sv[j] = 0u;
      }
      float* sMaxU = sMax + (u & 1) * 8 * 128;
      sMaxU[(hw * 4 + cw) * 128 + row] = m_loc;
      ok = softmax_barrier_and(ok);                         // the one meeting of a tile; also one decision for all
      if (!ok) { broke = true; break; }
      if (kShared && u > 0) l_row = l_row * corr_prev + tile_sum(u - 1);      // (every chunk sum of the previous tile is visible now)
      if (kShared && u == fresh_at) {                   // this tile starts a part: put the one before away
        fresh_at = g.begin(++next_part) - first;
        ok = ok && mbar_wait(bar_o0 + 8u * (uint32_t)((u - 1) & 1), (uint32_t)(((u - 1) >> 1) & 1), abort_flag);
        tc_fence_after();
        ok = __all_sync(0xffffffffu, ok ? 1 : 0) != 0;
        if (ok) part_done(m_row, l_row);
        m_row = -INFINITY;
        l_row = 0.f;
      }
      float m_tile = -INFINITY;
#pragma unroll
      for (int k = 0; k < REP; ++k) m_tile = fmaxf(m_tile, fmaxf(sMaxU[k * 128 + row], sMaxU[(4 + k) * 128 + row]));
      const float m_new = fmaxf(m_row, m_tile);
      const float m_use = (m_new == -INFINITY) ? 0.f : m_new;
      const float corr = ex2(m_row - m_use);                // 0 while no visible key has been met
      // the output so far was accumulated against the old maximum: rescale this thread's columns of its lane - unless
      // no row of the warp moved its maximum (a factor of exactly 1 changes nothing)
      const bool rescale = u > 0 && __any_sync(0xffffffffu, corr != 1.f && m_row != -INFINITY);
      // O += P V that must be complete: the previous tile's if the output is rescaled or its P rewritten, else (P in
      // tensor memory, where tiles alternate) the one before
      const int must = (rescale || !kTmemP) ? u - 1 : u - 2;
      if (must >= 0) {
        ok = ok && mbar_wait(bar_o0 + 8u * (uint32_t)(must & 1), (uint32_t)((must >> 1) & 1), abort_flag);
        tc_fence_after();
        ok = __all_sync(0xffffffffu, ok ? 1 : 0) != 0;
      }
      if (ok && rescale) {
#pragma unroll
        for (int pass = 0; pass < KPT / RK; ++pass) {
          uint32_t ov[RK];
#pragma unroll
          for (int ch = 0; ch < RK / 16; ++ch) tmem_ld16_issue(tmem_O + lane_addr + col0 + pass * RK + ch * 16, &ov[ch * 16]);
          tmem_ld_wait();
#pragma unroll
          for (int ch = 0; ch < RK / 16; ++ch) keep16(&ov[ch * 16]);
#pragma unroll
          for (int ch = 0; ch < RK / 16; ++ch) {
            float v[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(ov[ch * 16 + j]) * corr;
            tmem_st16(tmem_O + lane_addr + col0 + pass * RK + ch * 16, v);
          }
        }
      }
      float* sSumU = sSum + (u & 1) * 8 * 128;
#pragma unroll
      for (int pass = 0; pass < NP; ++pass) {
        if (NP > 1 && ok) load_scores(pass);                // (one pass: the scores are still in registers)
        // (all exponentials of the pass, then the chunks' sums side by side: neither waits for the other's latency)
        float p[HK], csum[NCP];
#pragma unroll
        for (int j = 0; j < HK; ++j) p[j] = ex2(__fmaf_rn(__uint_as_float(sv[j]), scale_log2, -m_use));
#pragma unroll
        for (int ch = 0; ch < NCP; ++ch) csum[ch] = 0.f;
#pragma unroll
        for (int j = 0; j < 16; ++j)
#pragma unroll
          for (int ch = 0; ch < NCP; ++ch) csum[ch] += p[ch * 16 + j];
#pragma unroll
        for (int ch = 0; ch < NCP; ++ch) {
          const int c0 = col0 + pass * HK + ch * 16;
          sSumU[(c0 >> 4) * 128 + row] = csum[ch];          // chunk index = c0 / 16
          uint32_t packed[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) packed[j] = pack_bf16(p[ch * 16 + 2 * j], p[ch * 16 + 2 * j + 1]);
          if (kTmemP) {
            if (ok) tmem_st8(tmem_P + (uint32_t)(u & 1) * 64u + lane_addr + (uint32_t)(c0 >> 1), packed);
          } else {                                          // P, in every copy of the row
#pragma unroll
            for (int q = 0; q < 2; ++q)
#pragma unroll
              for (int k = 0; k < REP; ++k)
                *reinterpret_cast<uint4*>(sP + tile_off(k * QT + row, (c0 >> 3) + q)) =
                    make_uint4(packed[4 * q], packed[4 * q + 1], packed[4 * q + 2], packed[4 * q + 3]);
          }
        }
      }
      // ---- this warp's part of P is written and its rescale of O complete: the MMA warp issues O += P V once every
      //      softmax warp has said so
      if (kTmemP) tmem_st_wait();
      else asm volatile("fence.proxy.async.shared::cta;" ::: "memory");      // P is read by the tensor core
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_p);
      if (!kShared && u > 0) l_row = l_row * corr_prev + tile_sum(u - 1);     // (not before the exponentials: nothing waits for it)
      corr_prev = corr;
      m_row = m_new;
    }
    if (!broke) ok = softmax_barrier_and(ok);               // the last tile's chunk sums are visible
    if (ok) l_row = l_row * corr_prev + tile_sum(n_tiles - 1);
    ok = ok && mbar_wait(bar_o0 + 8u * (uint32_t)((n_tiles - 1) & 1), (uint32_t)(((n_tiles - 1) >> 1) & 1), abort_flag);
    tc_fence_after();
    ok = __all_sync(0xffffffffu, ok ? 1 : 0) != 0;
    // this CTA's last part; a CTA that has not the first part of all hands two parts on as two entries
    const bool two = kShared && have && rank > 0;
    if (ok && !two) part_done(m_row, l_row);
    if (ok && g.n_ctas == 1) {
      // every copy of a row holds the same O row: a thread normalises and stores the columns it owns, [col0, +KPT)
      const float inv = 1.f / acc_l;
      bf16* dst = a.out + ((grow0 + row) * a.H + h) * kHD + col0;
      if (row_live) {
#pragma unroll
        for (int j = 0; j < KPT; j += 8)
          *reinterpret_cast<uint4*>(dst + j) = make_uint4(pack_bf16(acc[j] * inv, acc[j + 1] * inv), pack_bf16(acc[j + 2] * inv, acc[j + 3] * inv),
                                                          pack_bf16(acc[j + 4] * inv, acc[j + 5] * inv), pack_bf16(acc[j + 6] * inv, acc[j + 7] * inv));
      }
    } else if (g.n_ctas > 1) {
      // Rows go to their owner, CTA row / rows_per_owner of the cluster: (max, sum) and the unnormalised output, straight
      // from registers into its shared memory, [entry][owned row].  The first cluster barrier says that every CTA is done
      // with its tiles, the second that all rows have arrived; nothing is read remotely, so nobody waits to leave.
      __syncwarp();
      cluster_arrive();
      const int rpo = (QT + g.n_ctas - 1) / g.n_ctas, owner = row / rpo, entry = rank == 0 ? 0 : 1 + (rank - 1) * per_cta;
      const int slot_row = entry * rpo + row - owner * rpo;
      uint32_t dst = map_to_rank(smem + ((size_t)slot_row * kMergePitch + col0) * sizeof(float), (uint32_t)owner);
      const uint32_t dst_ml = map_to_rank(smem + (size_t)kMergeRows * kMergePitch * sizeof(float) + slot_row * sizeof(float2), (uint32_t)owner);
      cluster_wait();
      if (ok && row_live) {
#pragma unroll
        for (int j = 0; j < KPT; j += 4) st_cluster_f32x4(dst + (uint32_t)j * 4u, acc[j], acc[j + 1], acc[j + 2], acc[j + 3]);
        if (cw == 0 && hw == 0) st_cluster_f32x2(dst_ml, acc_m, acc_l);
      }
      if (ok && two) {
        dst += (uint32_t)(rpo * kMergePitch * sizeof(float));
#pragma unroll
        for (int ch = 0; ch < NCH; ++ch) {
          float v[16];
          tmem_ld16(tmem_O + lane_addr + col0 + ch * 16, v);
          if (row_live) {
#pragma unroll
            for (int j = 0; j < 16; j += 4) st_cluster_f32x4(dst + (uint32_t)(ch * 16 + j) * 4u, v[j], v[j + 1], v[j + 2], v[j + 3]);
          }
          __syncwarp();
        }
        if (row_live && cw == 0 && hw == 0) st_cluster_f32x2(dst_ml + (uint32_t)(rpo * sizeof(float2)), m_row, l_row);
      }
    }
    if (!ok && lane == 0) raise_word(a.err_flag, 6);
  }
  if (warp >= kPipeThreads / 32 && g.n_ctas > 1) {        // (the first cluster barrier, of the threads that push nothing)
    __syncwarp();
    cluster_arrive();
    cluster_wait();
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kPipeThreads / 32) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
  }
  if (g.n_ctas == 1) return;
  __syncwarp();
  cluster_arrive();
  cluster_wait();
  // ---- merge: this CTA's rows, the entries in part order.  (After an error the rows are garbage and the error word is up.)
  if (warp < kPipeThreads / 32) {
    const int rpo = (QT + g.n_ctas - 1) / g.n_ctas, r_end = min(rpo, rows_here - rank * rpo), entries = 1 + (g.n_ctas - 1) * per_cta;
    const float* sO = reinterpret_cast<const float*>(smem);
    const float2* sML = reinterpret_cast<const float2*>(sO + kMergeRows * kMergePitch);
    constexpr int TPR = kHD / 8;                            // threads per row, eight columns each
    const int col = (tid % TPR) * 8;
    for (int r = tid / TPR; r < r_end; r += kPipeThreads / TPR) {
      float2 ml = sML[r];
      float m = ml.x, l = ml.y, o[8];
      const float4* p = reinterpret_cast<const float4*>(sO + (size_t)r * kMergePitch + col);
      *reinterpret_cast<float4*>(o) = p[0];
      *reinterpret_cast<float4*>(o + 4) = p[1];
      for (int e = 1; e < entries; ++e) {
        ml = sML[e * rpo + r];
        p = reinterpret_cast<const float4*>(sO + (size_t)(e * rpo + r) * kMergePitch + col);
        const float4 va = p[0], vb = p[1];
        const Merge g2 = merge_of(m, ml.x);
        o[0] = merged(g2, o[0], va.x); o[1] = merged(g2, o[1], va.y); o[2] = merged(g2, o[2], va.z); o[3] = merged(g2, o[3], va.w);
        o[4] = merged(g2, o[4], vb.x); o[5] = merged(g2, o[5], vb.y); o[6] = merged(g2, o[6], vb.z); o[7] = merged(g2, o[7], vb.w);
        l = merged(g2, l, ml.y);
        m = g2.m;
      }
      const float inv = 1.f / l;
      *reinterpret_cast<uint4*>(a.out + ((grow0 + rank * rpo + r) * a.H + h) * kHD + col) =
          make_uint4(pack_bf16(o[0] * inv, o[1] * inv), pack_bf16(o[2] * inv, o[3] * inv), pack_bf16(o[4] * inv, o[5] * inv), pack_bf16(o[6] * inv, o[7] * inv));
    }
  }
}

template <int QT, bool kShared>
cudaError_t launch_pipe(cudaStream_t st, dim3 grid, size_t smem, const CUtensorMap (&tm)[5], const AttnArgs& a, const PipeShape& g,
                        float scale_log2) {
  static PerDevice<bool> attr_set = {};             // the shared-memory opt-in
  const int dev = device_slot();
  if (dev < 0) return cudaErrorInvalidDevice;
  if (!attr_set[dev]) {
    const cudaError_t e = cudaFuncSetAttribute(attn_verify_pipe_kernel<QT, kShared>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    attr_set[dev] = true;
  }
  return launch_pdl_cluster(attn_verify_pipe_kernel<QT, kShared>, grid, dim3(kPipeBlock), smem, st, (unsigned)g.n_ctas, tm[0], tm[1], tm[2], tm[3], tm[4], a, g,
                            scale_log2);
}

}  // namespace

int launch_attention_verify_pipe(cudaStream_t st, const AttnArgs& a, int n_parts) {
  const int rps = a.map.rows_per_seq, T = a.map.T;
  if (a.hd != kHD || T < 1 || T > kKeys || rps % T != 0 || !a.q || !a.local_k || !a.local_v || !a.err_flag || a.cache_rows == 0 ||
      a.kv_pos_stride != (size_t)kHD || a.cache_seq_stride != a.kv_head_stride * (size_t)a.Hkv || n_parts < 1 || n_parts > kAttnMaxClusterParts)
    return -2;
  PipeShape g{};
  g.len_a = a.hole_len > 0 ? a.hole_begin : a.S;
  g.len_b = a.S - g.len_a;
  g.row_b = a.hole_begin + a.hole_len;
  g.n_a = (g.len_a + kKeys - 1) / kKeys;
  g.n_all = 1 + g.n_a + (g.len_b + kKeys - 1) / kKeys;
  g.t_pad = 16;
  while (g.t_pad < T) g.t_pad *= 2;
  g.n_parts = n_parts < g.n_all ? n_parts : g.n_all;      // (every part has a tile)
  const int qt_rows = rps <= 32 ? 32 : (rps <= 64 ? 64 : 128);
  g.npt = qt_rows / T;
  if (g.npt > kKeys / g.t_pad) g.npt = kKeys / g.t_pad;
  const int q_tiles = (rps + g.npt * T - 1) / (g.npt * T);
  g.n_ctas = attn_pipe_ctas(g.n_parts, g.n_all, (long long)a.H * a.n_seq_slots * q_tiles, qt_rows);      // (the bits are the same)
  const float scale_log2 = (1.0f / sqrtf((float)a.hd)) * 1.4426950408889634f;
  const size_t smem = (size_t)kTileBytes * (2 + kStagesK + kStagesV) + 16384 + 128 + 1024;   // Q, P, K and V stages, softmax exchange
  alignas(64) CUtensorMap tm[5];
  const uint64_t planes = (uint64_t)a.cache_rows * kHD / a.kv_head_stride;       // (sequence, kv head) pairs
  const uint64_t bound = (uint64_t)(a.S + a.hole_len > 0 ? a.S + a.hole_len : 1);
  const uint64_t qw = (uint64_t)a.H * kHD, kw = (uint64_t)a.Hkv * kHD;
  if (encode_tmap_bf16_2d(&tm[0], a.q, (uint64_t)a.R, qw, qw, (uint32_t)qt_rows) != 0 ||
      encode_tmap_bf16_3d(&tm[1], a.local_k, kw, (uint64_t)T, (uint64_t)(a.R / T), kw, kw * T, (uint32_t)g.t_pad) != 0 ||
      encode_tmap_bf16_3d(&tm[2], a.local_v, kw, (uint64_t)T, (uint64_t)(a.R / T), kw, kw * T, (uint32_t)g.t_pad) != 0 ||
      encode_tmap_bf16_3d(&tm[3], a.cache_k, kHD, bound, planes, kHD, a.kv_head_stride, kKeys) != 0 ||
      encode_tmap_bf16_3d(&tm[4], a.cache_v, kHD, bound, planes, kHD, a.kv_head_stride, kKeys) != 0)
    return -4;
  const dim3 grid(a.H * g.n_ctas, a.n_seq_slots * q_tiles);
  const auto launch = [&](auto qt) {
    constexpr int QT = decltype(qt)::value;
    return g.n_ctas < g.n_parts ? launch_pipe<QT, true>(st, grid, smem, tm, a, g, scale_log2) : launch_pipe<QT, false>(st, grid, smem, tm, a, g, scale_log2);
  };
  const cudaError_t e = qt_rows == 32 ? launch(IntC<32>()) : qt_rows == 64 ? launch(IntC<64>()) : launch(IntC<128>());
  return e == cudaSuccess ? 0 : -4;
}

}  // namespace ssd
