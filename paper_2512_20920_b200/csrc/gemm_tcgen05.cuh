// tcgen05 / TMEM / TMA back end for every bf16 matrix product on the path.
//
// One warp-specialised kernel (1 CTA per SM, 384 threads; a CTA works tiles until there are none, see warp 11):
//   warps 0, 10 TMA producers: cp.async.bulk.tensor loads (128-byte swizzle) of
//               A and B tiles into a ring of shared-memory stages, completion on
//               mbarriers (no multicast LOADS anywhere: every CTA fetches its own operands; cluster-wide
//               are only the pair mode's tcgen05.commit, a barrier arrive, and the answer of warp 11's request).  Warp 0
//               announces a stage's bytes and loads the first operand's share, warp 10 loads the second
//               operand's: one warp cannot issue a stage's loads as fast as the tensor core consumes them.
//   warp 1      MMA issuer: owns the TMEM allocation (two accumulators, so the
//               epilogue of tile i overlaps the main loop of tile i+1); one
//               elected lane issues tcgen05.mma kind::f16 (bf16 x bf16 -> fp32),
//               M = 128 (256 across a CTA pair), N up to 256, K = 16 per instruction; tcgen05.commit
//               releases stages and publishes finished accumulators.
//   warps 2..9  epilogue (two warps per TMEM lane quadrant, alternating 32-column blocks):
//               tcgen05.ld the accumulator (lane = tile row), apply the fused epilogue
//               (SwiGLU, gate scale, coupling add/sub, SwiGLU backward, fp32 weight
//               gradient) and pass each 32 x 32 output block through a per-warp staging
//               area in shared memory: bf16 blocks leave by TMA bulk tensor stores
//               (64-byte swizzle), fp32 blocks are transposed there and written with plain
//               16-byte stores, four 128-byte rows per instruction.  Global writes are whole
//               lines whatever the row stride.
//   warp 11     tiles: describes the CTA's (pair's) next tile to the other warps and asks the hardware for the tile after it
//               (cluster launch control: the grid has a CTA or pair per tile, and a running one takes over the
//               place of one that has not been launched yet).
// Tile = 128 rows x 256 columns (the last column tile of a row may be 128 wide: N only has
// to be a multiple of 128), K step 64 (one 128-byte swizzle atom of bf16).  Products that would leave SMs idle with
// it take tiles of 128 or 64 columns, as tc_plan() reckons.
// Both operands may be K-major or MN-major; MN-major tiles are fetched 128 columns x 64 K rows at a time through a
// 3-D view of the matrix (64 x 64 boxes of a 2-D map as the fallback) and described to the tensor core with
// leading/stride offsets.
// Every wait is bounded; on expiry the kernel sets the status word, drops the tiles that have not begun and leaves.
//
// Pair mode (template flag PAIR; dense and K-grouped problems whose N is a multiple of 256, or of 128
// when B is stored [K, N]):
// the grid is launched as clusters of two CTAs that work one 256 x 256 tile together with
// tcgen05.mma.cta_group::2.  Each CTA loads its own 128 rows of A and ITS HALF of B's columns
// (the tensor core reads both halves across the pair), so a K step costs a CTA 32 KB of operand
// traffic instead of 48 KB and six stages fit.  The even CTA issues the MMAs; its commits
// arrive on the barriers of both CTAs, both CTAs' loads complete on its "full" barriers, and
// both CTAs' epilogue warps release its accumulator barriers.
//
// Transposed pair mode (expert-grouped products with bf16 store, gate-scale, SwiGLU or SwiGLU
// backward epilogue): the pair computes C^T.  The MMA M side holds 256 output features (rows of the expert's weight
// matrix, 128 per CTA), the N side a run of up to 256 of the expert's token rows, real rows
// only (rounded up to 32), taken from a chunk table built with the permutation.  Padding rows
// then cost no tensor-core time, and these products get the pair mode's operand savings, which
// row tiles that must not straddle experts cannot have.  The epilogue transposes each
// 32-feature x 32-token block on its way through the staging area.
#pragma once

#include <cuda.h>
#include <cstring>
#include <mutex>
#include <type_traits>

#include "common.cuh"
#include "gemm.cuh"

namespace revffn {

constexpr int TC_BM = 128;
constexpr int TC_BK = 64;
constexpr int TC_THREADS = 384;      // warp 0, 10: operand loads; warp 1: products; warps 2..9: epilogue; warp 11: tiles
constexpr int TC_LOAD_WARP_B = 10;   // the second load warp
constexpr int TC_TILE_WARP = 11;     // hands out the tiles
constexpr int TC_TILE_SLOTS = 4;     // tiles described ahead: the loads are up to two tiles ahead of the epilogue
constexpr int TC_EPI_WARPS = 8;
constexpr int TR_SMALL = 64;            // transposed: halves of a token chunk up to here come in 32-row boxes (experts of 4 rows: 66.7 -> 64.3 us)
constexpr int TC_A_BYTES = TC_BM * TC_BK * 2;            // 16 KB
constexpr long long TC_WAIT_CYCLES = 4000000000LL;       // ~2 s: bound on any single wait

template <int MMA_N, int EPI, bool PAIR> struct TcCfg {
  static constexpr int B_BYTES = (PAIR ? MMA_N / 2 : MMA_N) * TC_BK * 2;
  static constexpr int STAGE_BYTES = TC_A_BYTES + B_BYTES;
  // The fused updates of grouped products are bound by what their epilogue reads and writes: they trade part of the
  // operand ring for a row-wise staging area (8 KB per epilogue warp) and a ring of weights and moments in flight.
  static constexpr int STAGES = EPI == EPI_WADAM ? (PAIR ? 2 : 1) : EPI == EPI_WSGD ? (PAIR ? 3 : 2) : (PAIR ? 6 : 4);
  // staging per epilogue warp: two 32 x 32 bf16 blocks or one fp32 block
  static constexpr int EPI_WARP_BYTES = EPI == EPI_WADAM ? 20480 : EPI == EPI_WSGD ? 16384 : 4096;
  static constexpr int TMEM_COLS = 2 * MMA_N;           // two accumulators; a power of two >= 32
  // stage ring | epilogue staging | barriers; the ring starts 1024-byte aligned and
  // every stage is a multiple of 1024 bytes, so the staging area is aligned too
  static constexpr int EPI_OFF = STAGES * STAGE_BYTES;
  static constexpr int BAR_OFF = EPI_OFF + TC_EPI_WARPS * EPI_WARP_BYTES;
  static constexpr int SMEM_BYTES = BAR_OFF + 1024 /*align*/ + 768 /*barriers, tile descriptions*/;
};

struct TcParams {
  GemmProblem p;
  int tiles_m, tiles_n;      // GROUP_M: tiles_m is an upper bound, the device value comes from rows_total
  int tile_n;                // logical output columns per tile (of each matrix of an N-concatenated pair)
  int b_box;                 // rows (K-major) or columns (MN-major, 3-D maps) of B that one load brings: 128 or 64
  int k_blocks;              // dense / GROUP_M
  int tr;                    // transposed pair mode: weights on the MMA M side, an expert's token rows on the N side
  int tiles_f;               // tr: feature tiles per token chunk, 256 wide (128 of each matrix of a pair)
  int tr_swap;               // tr, matrix pair: the second matrix lies first in memory and in each group of 32 lanes
  uint32_t idesc;
  long long wait_cycles;     // bound on every wait of the kernel (clock cycles)
  int starve;                // failure-path test: the load warp issues nothing, so the first wait for operands runs out
  int bk;                    // operand elements per K step: 64 (bf16) or 128 (e4m3); a K step is 128 bytes of a row either way
  int mn3d;                  // MN-major operands are loaded 128 columns at a time through 3-D tensor maps
  int split_loads;           // 1: the second load warp issues the second operand's loads; 0: one thread issues all of them
};

// ---------------------------------------------------------------------------
// PTX wrappers
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.b32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
// Bounded wait.  Returns false when the wait was abandoned (this or another
// role ran out of time); the caller then leaves its loop.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* status,
                                          long long limit = TC_WAIT_CYCLES) {
  if (mbar_try_wait(bar, parity)) return true;
  long long t0 = clock64();
  int spins = 0;
  while (true) {
    if (mbar_try_wait(bar, parity)) return true;
    if (((++spins) & 63) == 0) {
      if (*abort_flag) return false;
      if (clock64() - t0 > limit) {
        *abort_flag = 1;
        set_status(status, REVFFN_ERR_DEVICE_WAIT);
        return false;
      }
    }
  }
}

// The same for a whole warp that stays converged: the result is the same in every lane.  Each role that goes on with
// warp-wide instructions (tensor-memory loads, shuffles, elect) waits like this: an abandoned wait ends each lane's spin at a
// point of its own, and a lane that saw the barrier complete just then would go on without the others.
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* status,
                                               long long limit = TC_WAIT_CYCLES) {
  if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
  return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag, status, limit));
}
// One lane of a converged warp.  The issuing warp walks its loop with all lanes and elects one for each group of
// instructions: a loop in one lane alone is divergent code, where every operand is moved to a uniform register first.
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.b32 %0, 1, 0, p;\n\t}" : "=r"(p));
  return p != 0;
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int c0, int c1, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(bar) : "memory");
}

// Shared -> global bulk tensor store of one box (the box and the swizzle come from the map).
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, uint32_t src, int c0, int c1) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];"
               ::"l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(src) : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// Wait until at most N of this thread's bulk groups still read their shared-memory source.
template <int N> __device__ __forceinline__ void bulk_wait_read() {
  asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
// Orders this thread's shared-memory writes before later async-proxy (TMA) reads of them.
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Pair mode: the same load, completing on a barrier that may live in the partner CTA (cluster address).
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* map, int c0, int c1, uint32_t bar_cluster) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(bar_cluster) : "memory");
}
// 128 columns x 64 K rows of an MN-major operand ([K rows, ld columns] in memory) into two consecutive 8 KB
// blocks of 64 columns each, the layout the MMA descriptors expect.  mn3d: one load through a 3-D view of the
// matrix {64 columns, K rows, ld / 64 column groups} with a box of two groups; else two 2-D loads of 64 x 64.
// A tensor load costs its issuing thread a couple of hundred clocks whatever its size, so halving their number
// matters as much as spreading them over two threads.
__device__ __forceinline__ void tma_load_mn128(bool mn3d, uint32_t dst, const CUtensorMap* map, int col, int krow, uint32_t bar,
                                               bool second_block = true) {
  if (mn3d) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(0), "r"(krow), "r"(col >> 6), "r"(bar) : "memory");
  } else {
    tma_load_2d(dst, map, col, krow, bar);
    if (second_block) tma_load_2d(dst + 8192, map, col + 64, krow, bar);
  }
}
__device__ __forceinline__ void tma_load_mn128_pair(bool mn3d, uint32_t dst, const CUtensorMap* map, int col, int krow,
                                                    uint32_t bar_cluster, bool second_block = true) {
  if (mn3d) {
    asm volatile(
        "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(0), "r"(krow), "r"(col >> 6), "r"(bar_cluster) : "memory");
  } else {
    tma_load_2d_pair(dst, map, col, krow, bar_cluster);
    if (second_block) tma_load_2d_pair(dst + 8192, map, col + 64, krow, bar_cluster);
  }
}
// 16 rows of both matrices of a pair, four times: {64 columns (128 bytes), 16 rows, 2 matrices, 4 groups of rows}.
__device__ __forceinline__ void tma_load_rows16_pair(uint32_t dst, const CUtensorMap* map, int col, int group, uint32_t bar_cluster) {
  asm volatile(
      "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(col), "r"(0), "r"(0), "r"(group), "r"(bar_cluster) : "memory");
}
__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// Cluster-wide address of the location `addr` (own shared window) in the CTA of rank `rank`.
__device__ __forceinline__ uint32_t mapa_u32(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar_cluster) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(bar_cluster) : "memory");
}
// All threads of both CTAs of the pair.
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Pair mode: arrive on the barrier at this shared-memory offset in both CTAs once the MMAs issued so far are done.
__device__ __forceinline__ void tc_commit_pair(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
               ::"r"(bar), "h"((uint16_t)3) : "memory");
}

// One product with the descriptors given as (low, high) words: the high words never change inside a kernel, and
// the low words move by small additions, so the issuing thread carries 32-bit values only.  Here for e4m3 operands
// (kind::f8f6f4: 32 one-byte elements of K per instruction, the same 32 bytes as 16 bf16 ones).
template <bool PAIR>
__device__ __forceinline__ void tc_mma_lohi_f8(uint32_t d_tmem, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo, uint32_t b_hi,
                                               uint32_t idesc, uint32_t acc) {
  if constexpr (PAIR)
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
        "setp.ne.b32 p, %6, 0;\n\t"
        "mov.b64 da, {%1, %2};\n\t"
        "mov.b64 db, {%3, %4};\n\t"
        "tcgen05.mma.cta_group::2.kind::f8f6f4 [%0], da, db, %5, p;\n\t}"
        ::"r"(d_tmem), "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(acc) : "memory");
  else
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
        "setp.ne.b32 p, %6, 0;\n\t"
        "mov.b64 da, {%1, %2};\n\t"
        "mov.b64 db, {%3, %4};\n\t"
        "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], da, db, %5, p;\n\t}"
        ::"r"(d_tmem), "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(acc) : "memory");
}

template <bool PAIR>
__device__ __forceinline__ void tc_mma_lohi(uint32_t d_tmem, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo, uint32_t b_hi,
                                            uint32_t idesc, uint32_t acc) {
  if constexpr (PAIR)
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
        "setp.ne.b32 p, %6, 0;\n\t"
        "mov.b64 da, {%1, %2};\n\t"
        "mov.b64 db, {%3, %4};\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], da, db, %5, p;\n\t}"
        ::"r"(d_tmem), "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(acc) : "memory");
  else
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
        "setp.ne.b32 p, %6, 0;\n\t"
        "mov.b64 da, {%1, %2};\n\t"
        "mov.b64 db, {%3, %4};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %5, p;\n\t}"
        ::"r"(d_tmem), "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(acc) : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void tc_mma(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(acc) : "memory");
}

// 32 consecutive accumulator columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Shared-memory matrix descriptor, 128-byte swizzle, tile base 1024-byte aligned.
//   K-major : rows of 128 bytes, 8-row groups 1024 bytes apart (SBO); LBO unused (1)
//   MN-major: 64-element chunks along M/N are lbo bytes apart, 8-k-row groups 1024 bytes apart
__device__ __forceinline__ uint64_t make_smem_desc(uint32_t addr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3FFFFu) >> 4);
  d |= (uint64_t)((lbo_bytes >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo_bytes >> 4) & 0x3FFFu) << 32;
  d |= 1ull << 46;      // descriptor version of this architecture
  d |= 2ull << 61;      // 128-byte swizzle
  return d;
}

__device__ __forceinline__ uint4 pack8(const float* f) {
  uint4 u;
  __nv_bfloat162 h;
  h = __floats2bfloat162_rn(f[0], f[1]); u.x = *reinterpret_cast<uint32_t*>(&h);
  h = __floats2bfloat162_rn(f[2], f[3]); u.y = *reinterpret_cast<uint32_t*>(&h);
  h = __floats2bfloat162_rn(f[4], f[5]); u.z = *reinterpret_cast<uint32_t*>(&h);
  h = __floats2bfloat162_rn(f[6], f[7]); u.w = *reinterpret_cast<uint32_t*>(&h);
  return u;
}
__device__ __forceinline__ void unpack8(uint4 u, float* f) {
  const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&u);
#pragma unroll
  for (int i = 0; i < 4; ++i) { float2 t = __bfloat1622float2(h[i]); f[2 * i] = t.x; f[2 * i + 1] = t.y; }
}

// Output staging.  A warp stages a 32-row x 32-column bf16 block, one row per lane, in the layout
// the store's tensor map expects: rows of 64 bytes under the 64-byte swizzle.  `buf` is aligned to
// the swizzle period, so the 16-byte piece j of row r lands at piece j ^ ((r >> 1) & 3); lanes of
// one store instruction then hit distinct banks.
__device__ __forceinline__ void stage32_bf16(uint8_t* buf, int r, const float* f) {
  uint8_t* row = buf + r * 64;
#pragma unroll
  for (int j = 0; j < 4; ++j) *reinterpret_cast<uint4*>(row + ((j ^ ((r >> 1) & 3)) << 4)) = pack8(f + 8 * j);
}

// A warp's 32-row x 32-column bf16 block (rows of 64 bytes, row stride ld elements) from the staging layout above to
// global memory, in "distributed" form: instruction i of four moves rows 8i .. 8i+7, lane l the
// 16-byte piece l & 3 of row 8i + (l >> 2).  Eight lanes cover four whole 64-byte row segments, so every
// 32-byte sector a request touches is used in full, and the 512 contiguous staging bytes an instruction
// touches spread over all banks.  rows_ok: rows of the block that exist (the rest are not stored).
__device__ __forceinline__ void blk_stage_to_global(const uint8_t* buf, int lane, bf16* g, int64_t ld, int rows_ok) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = 8 * i + (lane >> 2);
    const uint4 v = *reinterpret_cast<const uint4*>(buf + r * 64 + (((lane & 3) ^ ((r >> 1) & 3)) << 4));
    if (r < rows_ok) *reinterpret_cast<uint4*>(g + (int64_t)r * ld + (lane & 3) * 8) = v;
  }
}

// Logistic function from one ex2.approx and one rcp.approx (relative error about 2^-21, far inside what the
// bf16 results around it can show).
__device__ __forceinline__ float2 sigmoid_approx2(float2 x) {
  const float2 t = __fmul2_rn(x, make_float2(-1.4426950408889634f, -1.4426950408889634f));
  float e0, e1, r0, r1;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e0) : "f"(t.x));
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e1) : "f"(t.y));
  const float2 den = __fadd2_rn(make_float2(e0, e1), make_float2(1.f, 1.f));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r0) : "f"(den.x));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r1) : "f"(den.y));
  return make_float2(r0, r1);
}

// Where an epilogue warp's 32-row slab of an fp32 result (or of the weights a fused update rewrites) lies.
// at0: this lane's element of row (lane / 8), column piece (lane % 8); in the row-wise updates of the warp's first row, piece `lane`.
struct SlabOut {
  float* c; bf16* w; float *m, *mom, *var;      // output; updated weight, master copy and moments
  int64_t at0, ld4, res0;      // ...; four rows; residual element
  int rows;                    // rows that exist (<= 32)
};
__device__ __forceinline__ float4 as_f4(const uint4& u) {
  return make_float4(__uint_as_float(u.x), __uint_as_float(u.y), __uint_as_float(u.z), __uint_as_float(u.w));
}
__device__ __forceinline__ float4 bf4(const uint2& u) {
  const float2 lo = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.x));
  const float2 hi = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.y));
  return make_float4(lo.x, lo.y, hi.x, hi.y);
}
__device__ __forceinline__ uint2 pack4(const float4& v) {
  __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
  return make_uint2(*reinterpret_cast<uint32_t*>(&lo), *reinterpret_cast<uint32_t*>(&hi));
}
__device__ __forceinline__ float4 adam_step4(const UpdRule& r, const float4& w, const float4& g, float4& mom, float4& var) {
  float2 m[2] = {make_float2(mom.x, mom.y), make_float2(mom.z, mom.w)}, v[2] = {make_float2(var.x, var.y), make_float2(var.z, var.w)};
  const float2 lo = adam_step2(r, make_float2(w.x, w.y), make_float2(g.x, g.y), m[0], v[0]);
  const float2 hi = adam_step2(r, make_float2(w.z, w.w), make_float2(g.z, g.w), m[1], v[1]);
  mom = make_float4(m[0].x, m[0].y, m[1].x, m[1].y);
  var = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
  return make_float4(lo.x, lo.y, hi.x, hi.y);
}

// Fused update of a grouped product's tile (EPI_WADAM, EPI_WSGD): a warp's 16 rows x 128 columns, eight units of two rows.  Weights (the
// fp32 master copy, or the bf16 weights themselves) and Adam's moments of a unit come by cp.async into a ring of UpdRing
// units per warp behind the 8 KB staging area.  Everything that does not change is a compile-time constant or a running
// offset: with two epilogue warps per scheduler an instruction costs its latency, and the first form of this loop
// (kind and ring depth looked up at run time) took 950 clk per unit before any memory traffic.  Adam's last
// units of a tile ask for the first ones of the next, so that reads go on while its accumulator is staged (experts'
// gate | up at 1024 tokens, 9.0 GB: 2088 -> 1965 us, now 1469, 6.1 TB/s, where a bare read-modify-write kernel of this shape
// reaches 6.3; the SGD step, 1.4 GB, got slower by it, 309 -> 362).
template <bool ADAM, bool MASTER> struct UpdRing {
  static constexpr int W = MASTER ? 1024 : 512;                    // bytes of weights in a unit
  static constexpr int UNIT = W + (ADAM ? 2048 : 0);
  static constexpr int DEPTH = ADAM ? 4 : 8;
  static_assert(DEPTH * UNIT <= (ADAM ? 12288 : 8192), "ring");
};
template <bool ADAM, bool MASTER>
__device__ __forceinline__ void upd_ask(const SlabOut& o, uint8_t* unit, int lane, int64_t at, int64_t ldc) {      // at: the unit's first row
  using R = UpdRing<ADAM, MASTER>;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    if (MASTER) cp_async16(unit + i * 512 + lane * 16, o.m + at + i * ldc, true);
    if (ADAM) {
      cp_async16(unit + R::W + i * 512 + lane * 16, o.mom + at + i * ldc, true);
      cp_async16(unit + R::W + 1024 + i * 512 + lane * 16, o.var + at + i * ldc, true);
    }
  }
  // 256 bytes of bf16 weights per row: half a warp each (at points at column 4 lane)
  if (!MASTER) cp_async16(unit + lane * 16, o.w + at - lane * 4 + (lane >> 4) * ldc + (lane & 15) * 8, true);
}
template <bool ADAM, bool MASTER>
__device__ __forceinline__ void upd_first(const SlabOut& o, uint8_t* stg, int lane, int64_t ldc) {
  using R = UpdRing<ADAM, MASTER>;
#pragma unroll
  for (int u = 0; u < R::DEPTH; ++u) {
    upd_ask<ADAM, MASTER>(o, stg + 8192 + u * R::UNIT, lane, o.at0 + 2 * u * ldc, ldc);
    cp_async_commit();
  }
}
template <bool ADAM, bool MASTER>
__device__ __forceinline__ void upd_half(const UpdRule& rule, const SlabOut& o, const SlabOut& next, uint8_t* stg, int lane, int64_t ldc,
                                         int cb, bool last, bool more) {
  using R = UpdRing<ADAM, MASTER>;
  int64_t at = o.at0 + cb * 128;
#pragma unroll
  for (int u = 0; u < 8; ++u, at += 2 * ldc) {
    uint8_t* unit = stg + 8192 + u % R::DEPTH * R::UNIT;
    cp_async_wait<R::DEPTH - 1>();
    if (!MASTER) __syncwarp();      // a 16-byte piece of bf16 weights serves two lanes
    float4 w[2], mo[2], va[2], g[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      w[i] = MASTER ? *reinterpret_cast<const float4*>(unit + i * 512 + lane * 16) : bf4(*reinterpret_cast<const uint2*>(unit + i * 256 + lane * 8));
      if (ADAM) {
        mo[i] = *reinterpret_cast<const float4*>(unit + R::W + i * 512 + lane * 16);
        va[i] = *reinterpret_cast<const float4*>(unit + R::W + 1024 + i * 512 + lane * 16);
      }
      g[i] = *reinterpret_cast<const float4*>(stg + (2 * u + i) * 512 + ((lane ^ ((2 * u + i) & 7)) << 4));
    }
    if (!MASTER) __syncwarp();
    if (u + R::DEPTH < 8) upd_ask<ADAM, MASTER>(o, unit, lane, at + 2 * R::DEPTH * ldc, ldc);
    else if (!last) upd_ask<ADAM, MASTER>(o, unit, lane, at + 2 * (R::DEPTH - 8) * ldc + 128, ldc);
    else if (more) upd_ask<ADAM, MASTER>(next, unit, lane, next.at0 + 2 * (u + R::DEPTH - 8) * ldc, ldc);
    cp_async_commit();
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      if (ADAM) {
        w[i] = adam_step4(rule, w[i], g[i], mo[i], va[i]);
        *reinterpret_cast<float4*>(o.mom + at + i * ldc) = mo[i];
        *reinterpret_cast<float4*>(o.var + at + i * ldc) = va[i];
      } else {
        w[i].x -= rule.lr * g[i].x; w[i].y -= rule.lr * g[i].y; w[i].z -= rule.lr * g[i].z; w[i].w -= rule.lr * g[i].w;
      }
      if (MASTER) *reinterpret_cast<float4*>(o.m + at + i * ldc) = w[i];
      *reinterpret_cast<uint2*>(o.w + at + i * ldc) = pack4(w[i]);
    }
  }
}

// A tile as its roles see it: 32 bytes, described by the tile warp.
struct alignas(16) TcTile {
  int m0, n0, group, k_blocks, krow0;
  int ncols;      // accumulator columns in use: the tile's, or 128 in the last column tile of an odd multiple of 128
  int pad;        // tr: rows of zero padding after the chunk's, to the next multiple of 64 (an expert's last chunk only)
  int valid;      // 0: no tile, the last one is done
};

// Tile `idx` (of tiles_m row tiles or token chunks x tiles_n column or feature tiles a group).  pair_rank < 0: one CTA per
// 128-row tile.  pair_rank 0 / 1: a tile is 256 rows worked by two CTAs, this CTA takes rows 128 * pair_rank .. + 127 of it
// (rows past M are loaded as zeros and never stored).
__device__ __forceinline__ TcTile tc_tile(const TcParams& P, int idx, int tiles_m, int tiles_n, int pair_rank) {
  TcTile t;
  const GemmProblem& p = P.p;
  const int row = idx / tiles_n, tn = idx - row * tiles_n, group = row / tiles_m, tm = row - group * tiles_m;
  t.valid = 1;
  t.krow0 = 0;
  t.pad = 0;
  t.k_blocks = P.k_blocks;
  if (P.tr) {
    // m0 = first token row, ncols = token rows (the MMA N), n0 = first feature of this CTA's 128
    const int4 e = p.tok_chunks[tm];
    t.group = e.x; t.m0 = e.y; t.ncols = e.z;
    t.n0 = (tn * 2 + pair_rank) * (p.concat == CONCAT_N ? TC_BM / 2 : TC_BM);
    t.pad = e.w;
    return t;
  }
  t.group = group;
  if (p.group_mode == GROUP_K) {
    if (p.group_off) {
      const int r0 = p.group_off[group], r1 = p.group_off[group + 1], cnt = p.group_cnt ? p.group_cnt[group] : 0x7fffff00;
      t.krow0 = r0;
      t.k_blocks = min((r1 - r0) / TC_BK, (cnt + TC_BK - 1) / TC_BK);   // skip all-zero K blocks
    } else {
      // equal slices of a dense K (split-K): rows past K in the last K step load as zeros
      const int slice = (int)split_k_rows(p.K, p.n_groups);
      const int k0 = min(t.group * slice, p.K), k1 = min(k0 + slice, p.K);
      t.krow0 = k0;
      t.k_blocks = (k1 - k0 + TC_BK - 1) / TC_BK;
    }
  }
  t.m0 = (pair_rank >= 0) ? tm * 2 * TC_BM + pair_rank * TC_BM : tm * TC_BM;
  t.n0 = tn * P.tile_n;
  t.ncols = (p.concat == CONCAT_N) ? 2 * P.tile_n : min(P.tile_n, p.N - t.n0);
  if (p.group_mode == GROUP_M) t.group = p.tile_group[tm];
  return t;
}

// Cluster launch control.  Asks the hardware for a cluster of this grid that has not been launched yet; the answer (16 bytes)
// arrives on the barrier, in both CTAs of a pair.
template <bool PAIR>
__device__ __forceinline__ void clc_ask(uint32_t answer, uint32_t bar) {
  if constexpr (PAIR)
    asm volatile("clusterlaunchcontrol.try_cancel.async.shared::cta.mbarrier::complete_tx::bytes.multicast::cluster::all.b128 [%0], [%1];"
                 ::"r"(answer), "r"(bar) : "memory");
  else
    asm volatile("clusterlaunchcontrol.try_cancel.async.shared::cta.mbarrier::complete_tx::bytes.b128 [%0], [%1];"
                 ::"r"(answer), "r"(bar) : "memory");
}
// blockIdx.x of the first CTA of the cluster that the answer grants, or -1 when none was left.
__device__ __forceinline__ int clc_granted(uint32_t answer) {
  int x;
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b128 a;\n\t.reg .b64 lo, hi;\n\t"
      "ld.shared.v2.b64 {lo, hi}, [%1];\n\t"
      "mov.b128 a, {lo, hi};\n\t"
      "mov.s32 %0, -1;\n\t"
      "clusterlaunchcontrol.query_cancel.is_canceled.pred.b128 p, a;\n\t"
      "@p clusterlaunchcontrol.query_cancel.get_first_ctaid::x.b32.b128 %0, a;\n\t}"
      : "=r"(x) : "r"(answer) : "memory");
  return x;
}

// ---------------------------------------------------------------------------
// The kernel
// ---------------------------------------------------------------------------
template <int MMA_N, int EPI, bool PAIR>
__global__ void __launch_bounds__(TC_THREADS, 1)
gemm_tc_kernel(const __grid_constant__ TcParams P, const __grid_constant__ CUtensorMap map_a,
               const __grid_constant__ CUtensorMap map_b0, const __grid_constant__ CUtensorMap map_b1,
               const __grid_constant__ CUtensorMap map_c, const __grid_constant__ CUtensorMap map_c1) {
  using Cfg = TcCfg<MMA_N, EPI, PAIR>;
  constexpr bool RMW = EPI == EPI_COUPLE || EPI == EPI_WRMW;
  constexpr bool UPD = EPI == EPI_WADAM || EPI == EPI_WSGD;
  constexpr bool WGRAD = EPI == EPI_WGRAD || EPI == EPI_WRMW || UPD;
  extern __shared__ uint8_t smem_raw[];
  const GemmProblem& p = P.p;
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;                 // stage ring, 1024-byte aligned
  uint8_t* gen_base = smem_raw + (base - raw);
  const uint32_t bars = base + Cfg::BAR_OFF;                    // barrier block
  auto full_bar = [&](int s) { return bars + 8u * s; };
  auto empty_bar = [&](int s) { return bars + 8u * (Cfg::STAGES + s); };
  auto tfull_bar = [&](int a) { return bars + 8u * (2 * Cfg::STAGES + a); };
  auto tempty_bar = [&](int a) { return bars + 8u * (2 * Cfg::STAGES + 2 + a); };
  const uint32_t drain_bar = bars + 320u;      // abort path of the MMA thread: "every product issued so far is done"
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(gen_base + Cfg::BAR_OFF + 256);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  int* issued = reinterpret_cast<int*>(tmem_slot + 2);   // [STAGES] parity+1 of the last load issued per stage
  int* issued_b = issued + Cfg::STAGES;                  // the same for the second load warp: nonzero once it has issued
  // tiles: their descriptions, a barrier each for "described" and "read by all roles"; "the loads have begun a tile", the answer
  // of the hardware and "both CTAs have read the answer"
  auto dfull_bar = [&](int i) { return bars + 336u + 8u * i; };
  auto dempty_bar = [&](int i) { return bars + 336u + 8u * (TC_TILE_SLOTS + i); };
  const uint32_t begun_bar = bars + 400u, answer_bar = bars + 408u, heard_bar = bars + 416u, answer = bars + 432u;
  TcTile* const tiles = reinterpret_cast<TcTile*>(gen_base + Cfg::BAR_OFF + 448);
  static_assert(TC_TILE_SLOTS == 4 && sizeof(TcTile) == 32, "barrier block");

  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  const int crank = PAIR ? (int)cluster_ctarank() : 0;     // rank in the pair; rank 0 issues the MMAs
  const int prank = PAIR ? crank : -1;

  if (threadIdx.x == 0) {
    for (int s = 0; s < Cfg::STAGES; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); issued[s] = 0; issued_b[s] = 0; }
    for (int a = 0; a < 2; ++a) { mbar_init(tfull_bar(a), 1); mbar_init(tempty_bar(a), PAIR ? 2 * TC_EPI_WARPS : TC_EPI_WARPS); }
    mbar_init(drain_bar, 1);
    // readers of a description: the load warps that load, the products' warp where it runs, the epilogue warps
    const int readers = (P.split_loads ? 2 : 1) + (crank == 0 ? 1 : 0) + TC_EPI_WARPS;
    for (int i = 0; i < TC_TILE_SLOTS; ++i) { mbar_init(dfull_bar(i), 1); mbar_init(dempty_bar(i), readers); }
    mbar_init(begun_bar, 1); mbar_init(answer_bar, 1); mbar_init(heard_bar, PAIR ? 2 : 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    if constexpr (PAIR) {      // the same warp of both CTAs, the same shared-memory offset
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;"
                   ::"r"(smem_u32(tmem_slot)), "r"((uint32_t)Cfg::TMEM_COLS) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                   ::"r"(smem_u32(tmem_slot)), "r"((uint32_t)Cfg::TMEM_COLS) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
  }
  pdl_wait();      // barriers and tensor memory are set up beside the last blocks of the kernel before this one
  tc_fence_before();
  __syncthreads();
  if constexpr (PAIR) cluster_sync_all();      // the partner's barriers exist before anything signals them
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  int tiles_m_dev = P.tiles_m;      // 128-row tiles as counted on the device
  if (p.group_mode == GROUP_M) tiles_m_dev = min(P.tiles_m, *p.rows_total / TC_BM);

  // The next tile of this role, all lanes together.  0: there is none; -1: the wait was abandoned.
  int slot = 0;
  uint32_t slot_phase = 0;
  auto next_tile = [&](TcTile& t) -> int {
    if (!mbar_wait_warp(dfull_bar(slot), slot_phase, abort_flag, p.status, P.wait_cycles)) return -1;
    t = tiles[slot];
    __syncwarp();
    if (lane == 0) mbar_arrive(dempty_bar(slot));
    if (++slot == TC_TILE_SLOTS) { slot = 0; slot_phase ^= 1u; }
    return t.valid;
  };

  if (warp == 0 || warp == TC_LOAD_WARP_B) {
    // ------------------------------------------------------------------ operand loads
    // Two warps walk the same tiles and stages, all lanes together, and one elected lane of each issues a K step's loads:
    // in a loop that one lane runs alone every operand of a load is moved to a uniform register first (forward of 64
    // tokens 286 -> 277 us, fp8 forward at 8192 1048 -> 1023, step at 8192 5328 -> 5267 by this alone).  A K step's loads
    // still take a warp 260-310 clocks, of which all of them in one warp would be more than the 512 clocks of tensor
    // work in a stage.  Warp A announces the stage's bytes and loads the first operand's share of the stage, warp B
    // loads the second operand's; the bytes may arrive before they are announced (the barrier's phase cannot complete
    // before the announcing arrival).
    // (A version of this loop that kept per-tile "load slots" -- tensor-map pointer, destination, coordinates --
    // in registers and issued one load per slot measured 15-40 % slower: a load whose tensor map is named through
    // a pointer chosen at run time, rather than as the kernel parameter itself, is slow to issue.)
    // la: this warp loads the first operand's share (and announces the stage); lb: the second operand's.
    // Without split_loads the first warp does both and the second warp has nothing to do.
    const bool la = warp == 0, lb = P.split_loads ? warp != 0 : warp == 0;
    if (!P.starve && (la || lb)) {
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      // this warp's loads of K step kb of tile t, by one elected lane
      auto issue = [&](const TcTile& t, int kb, int k_half) {
        const uint32_t sa = base + stage * Cfg::STAGE_BYTES;
        const uint32_t sb = sa + TC_A_BYTES;
        if constexpr (PAIR) {
          // both CTAs' loads complete on the even CTA's barrier, which expects the bytes of both
          const uint32_t fbc = mapa_u32(full_bar(stage), 0);
          if (P.tr) {
            // M side: 128 rows of the expert's weights; N side: this CTA's half of the chunk's token rows, one
            // 128-row box or up to two 32-row boxes (rows past the half are loaded and not used)
            const int half = t.ncols / 2, n32 = half <= TR_SMALL ? (half + 31) / 32 : 0;
            if (la) {
              if (crank == 0) mbar_expect_tx(full_bar(stage), 2 * (TC_A_BYTES + (n32 ? n32 * 4096 : 16384)));
              int kw = kb;
              const bool second = p.concat == CONCAT_K && kb >= k_half;
              if (second) kw = kb - k_half;
              if (EPI == EPI_SWIGLU) {
                tma_load_rows16_pair(sa, &map_b0, kb * P.bk, (t.group * p.N + t.n0) / 16, fbc);
              } else if (!p.b_mn_major) {
                if (second) tma_load_2d_pair(sa, &map_b1, kw * P.bk, t.group * p.N + t.n0, fbc);
                else tma_load_2d_pair(sa, &map_b0, kw * P.bk, t.group * p.N + t.n0, fbc);
              } else {
                const int kdim = (p.concat == CONCAT_K) ? k_half * TC_BK : t.k_blocks * TC_BK;
                const int krow = t.group * kdim + kw * TC_BK;
                if (second) tma_load_mn128_pair(P.mn3d, sa, &map_b1, p.b_col0 + t.n0, krow, fbc);
                else tma_load_mn128_pair(P.mn3d, sa, &map_b0, p.b_col0 + t.n0, krow, fbc);
              }
            }
            if (lb) {
              if (n32 == 0) tma_load_2d_pair(sb, &map_a, kb * P.bk, t.m0 + crank * half, fbc);
              else for (int i = 0; i < n32; ++i) tma_load_2d_pair(sb + i * 4096, &map_c1, kb * P.bk, t.m0 + crank * half + 32 * i, fbc);
            }
            return;
          }
          const int nhalf = t.ncols / 2;       // this CTA's share of the tile's columns: 128, or 64 in a ragged last tile
          if (la) {
            // (a 3-D load of an MN-major B brings its whole box, also where this CTA's share of a ragged tile is less)
            const int b_cols = (p.b_mn_major && P.mn3d) ? P.b_box : nhalf;
            if (crank == 0) mbar_expect_tx(full_bar(stage), 2 * (TC_A_BYTES + b_cols * TC_BK * 2));
            if (!p.a_mn_major) {
              tma_load_2d_pair(sa, &map_a, t.krow0 + kb * TC_BK, t.m0, fbc);
            } else {
              tma_load_mn128_pair(P.mn3d, sa, &map_a, p.a_col0 + t.m0, t.krow0 + kb * TC_BK, fbc);
            }
          }
          if (lb) {
            bool second = p.concat == CONCAT_K && t.krow0 / TC_BK + kb >= k_half;
            const int kbp = second ? kb - k_half : kb;
            int b_row = t.n0 + nhalf * crank;
            if (EPI == EPI_HEADS && p.hm_split && t.n0 >= p.hm_split) { second = true; b_row -= p.hm_split; }
            if (!p.b_mn_major) {
              // this CTA's half of the accumulator columns: gate rows (rank 0) or up rows (rank 1) of a
              // SwiGLU pair, else rows n0 + nhalf rank .. of B
              // (the tensor map is named directly in each call: a map chosen through a pointer is slow to issue)
              if (p.concat == CONCAT_N) {
                if (crank == 0) tma_load_2d_pair(sb, &map_b0, kbp * TC_BK, t.n0, fbc);
                else tma_load_2d_pair(sb, &map_b1, kbp * TC_BK, t.n0, fbc);
              } else if (second) {
                tma_load_2d_pair(sb, &map_b1, t.krow0 + kbp * TC_BK, b_row, fbc);
              } else {
                tma_load_2d_pair(sb, &map_b0, t.krow0 + kbp * TC_BK, b_row, fbc);
              }
            } else {
              const int krow = t.krow0 + kbp * TC_BK;
              if (second) tma_load_mn128_pair(P.mn3d, sb, &map_b1, p.b_col0 + t.n0 + nhalf * crank, krow, fbc, nhalf > 64);
              else tma_load_mn128_pair(P.mn3d, sb, &map_b0, p.b_col0 + t.n0 + nhalf * crank, krow, fbc, nhalf > 64);
            }
          }
          return;
        }
        const uint32_t fb = full_bar(stage);
        const bool second = p.concat == CONCAT_K && t.krow0 / TC_BK + kb >= k_half;
        const int kb_b = second ? kb - k_half : kb;
        // An MN-major B tile is four 64 x 64 boxes against one or two loads for A: with two load threads the
        // first takes B's last boxes too (3 + 2 loads, or 3 + 3 when A is MN-major as well).
        const int b_mn_split = !p.b_mn_major ? 0 : (!P.split_loads ? 0 : ((p.a_mn_major && !P.mn3d) ? 3 : 2));
        if (la) {
          mbar_expect_tx(fb, TC_A_BYTES + t.ncols * TC_BK * 2);
          issued[stage] = (int)phase + 1;
          // A tile
          if (!p.a_mn_major) {
            tma_load_2d(sa, &map_a, t.krow0 + kb * P.bk, t.m0, fb);
          } else {
            tma_load_mn128(P.mn3d, sa, &map_a, p.a_col0 + t.m0, t.krow0 + kb * TC_BK, fb);
          }
          if (b_mn_split) {
            int kdim = (p.concat == CONCAT_K) ? k_half * TC_BK : t.k_blocks * TC_BK;
            int krow = (p.group_mode == GROUP_M ? t.group * kdim : t.krow0) + kb_b * TC_BK;
            if (P.mn3d) {          // the second 128 columns
              if (t.ncols > 128) {
                if (second) tma_load_mn128(true, sb + 16384, &map_b1, p.b_col0 + t.n0 + 128, krow, fb);
                else tma_load_mn128(true, sb + 16384, &map_b0, p.b_col0 + t.n0 + 128, krow, fb);
              }
            } else {
#pragma unroll
              for (int j = 2; j < MMA_N / 64; ++j) {
                if (j < b_mn_split || 64 * j >= t.ncols) continue;
                if (second) tma_load_2d(sb + j * 8192, &map_b1, p.b_col0 + t.n0 + 64 * j, krow, fb);
                else tma_load_2d(sb + j * 8192, &map_b0, p.b_col0 + t.n0 + 64 * j, krow, fb);
              }
            }
          }
        }
        if (lb) {
          issued_b[stage] = (int)phase + 1;
          // B tile
          if (!p.b_mn_major) {
            // rows of the flattened [groups * N, K] weight tensor
            int row0 = (p.group_mode == GROUP_M ? t.group * p.N : 0) + t.n0;
            bool second = p.concat == CONCAT_K && t.krow0 / TC_BK + kb >= k_half;
            if (EPI == EPI_HEADS && p.hm_split && t.n0 >= p.hm_split) { second = true; row0 -= p.hm_split; }
            if (p.concat == CONCAT_N) {
              tma_load_2d(sb, &map_b0, kb_b * P.bk, row0, fb);
              tma_load_2d(sb + P.tile_n * 128, &map_b1, kb_b * P.bk, row0, fb);
            } else {
#pragma unroll
              for (int j = 0; j < MMA_N / 128; ++j) {
                if (128 * j >= t.ncols) continue;
                if (second) tma_load_2d(sb + j * 16384, &map_b1, t.krow0 + kb_b * P.bk, row0 + 128 * j, fb);
                else tma_load_2d(sb + j * 16384, &map_b0, t.krow0 + kb_b * P.bk, row0 + 128 * j, fb);
              }
            }
          } else {
            // rows of the flattened [groups * Kdim, N] weight tensor, or token rows (GROUP_K / dense wgrad)
            int kdim = (p.concat == CONCAT_K) ? k_half * TC_BK : t.k_blocks * TC_BK;
            int krow = (p.group_mode == GROUP_M ? t.group * kdim : t.krow0) + kb_b * TC_BK;
            if (P.mn3d) {
              if (second) tma_load_mn128(true, sb, &map_b1, p.b_col0 + t.n0, krow, fb);
              else tma_load_mn128(true, sb, &map_b0, p.b_col0 + t.n0, krow, fb);      // 64 columns with the narrow box
              if (!b_mn_split && t.ncols > 128) {
                if (second) tma_load_mn128(true, sb + 16384, &map_b1, p.b_col0 + t.n0 + 128, krow, fb);
                else tma_load_mn128(true, sb + 16384, &map_b0, p.b_col0 + t.n0 + 128, krow, fb);
              }
            } else {
#pragma unroll
              for (int j = 0; j < MMA_N / 64; ++j) {
                if ((b_mn_split && j >= b_mn_split) || 64 * j >= t.ncols) continue;
                if (second) tma_load_2d(sb + j * 8192, &map_b1, p.b_col0 + t.n0 + 64 * j, krow, fb);
                else tma_load_2d(sb + j * 8192, &map_b0, p.b_col0 + t.n0 + 64 * j, krow, fb);
              }
            }
          }
        }
      };
      TcTile t;
      while (ok && next_tile(t) > 0) {
        if (la && crank == 0 && lane == 0) mbar_arrive(begun_bar);
        const int k_half = P.k_blocks / 2;
        for (int kb = 0; kb < t.k_blocks; ++kb) {
          if (!mbar_wait_warp(empty_bar(stage), phase ^ 1u, abort_flag, p.status, P.wait_cycles)) { ok = false; break; }
          if (elect_one()) issue(t, kb, k_half);
          __syncwarp();
          if (++stage == Cfg::STAGES) { stage = 0; phase ^= 1u; }
        }
      }
      if (la) pdl_trigger();
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    // One lane issues every product of the CTA (pair), so the cycles this loop spends per K step bound the
    // kernel as surely as the tensor pipe does: 512 clocks of tensor work in a 128 x 256 x 64 step, less in narrow
    // tiles.  The warp walks the loop converged and elects the lane, which keeps operands in uniform registers (a loop
    // in one lane: about 300 clocks for four products and 60 for the commit; steps at 512 and 8192 tokens 1496 -> 1480
    // and 5479 -> 5416 us, fp8 forward at 8192 1083 -> 1056).  Everything that does not change inside a tile (descriptor
    // high words, layout steps, barrier addresses) is set up outside the loop.
    if (crank == 0) {
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      int it = 0;
      // the M-side slot holds A (or, transposed, the weights B); the N-side slot the other operand
      const int m_mn = P.tr ? p.b_mn_major : p.a_mn_major, n_mn = P.tr ? p.a_mn_major : p.b_mn_major;
      const uint32_t sb = __shfl_sync(0xffffffffu, base, 0), tb = __shfl_sync(0xffffffffu, tmem_base, 0);
      const uint64_t a_desc0 = m_mn ? make_smem_desc(sb, 8192, 1024) : make_smem_desc(sb, 16, 1024);
      const uint64_t b_desc0 = n_mn ? make_smem_desc(sb + TC_A_BYTES, 8192, 1024) : make_smem_desc(sb + TC_A_BYTES, 16, 1024);
      const uint32_t a_hi = (uint32_t)(a_desc0 >> 32), b_hi = (uint32_t)(b_desc0 >> 32);
      const uint32_t a_lo0 = (uint32_t)a_desc0, b_lo0 = (uint32_t)b_desc0;    // address field (bits 0..13, 16-byte units) + leading offset
      const uint32_t a_step = m_mn ? (2048u >> 4) : (32u >> 4);   // 16 k-elements per instruction
      const uint32_t b_step = n_mn ? (2048u >> 4) : (32u >> 4);
      constexpr uint32_t SB16 = (uint32_t)Cfg::STAGE_BYTES >> 4;  // the whole ring stays below 256 KB: no carry out of the field
      uint32_t a_lo = a_lo0, b_lo = b_lo0, fbar = full_bar(0), ebar = empty_bar(0);
      TcTile t;
      for (; ok; ++it) {
        const int got = next_tile(t);
        if (got <= 0) { ok = got == 0; break; }
        const int acc = it & 1;
        const uint32_t acc_phase = (uint32_t)(it >> 1) & 1u;
        if (!mbar_wait_warp(tempty_bar(acc), acc_phase ^ 1u, abort_flag, p.status, P.wait_cycles)) { ok = false; break; }
        tc_fence_after();
        const uint32_t d_tmem = tb + (uint32_t)(acc * MMA_N);
        const uint32_t idesc = (P.idesc & ~(0x3Fu << 17)) | ((uint32_t)(t.ncols >> 3) << 17);   // N of this tile
        const int nk = t.k_blocks;
        for (int kb = 0; kb < nk; ++kb) {
          if (!mbar_wait_warp(fbar, phase, abort_flag, p.status, P.wait_cycles)) { ok = false; break; }
          tc_fence_after();
          if (elect_one()) {
            if (p.fp8) {
              tc_mma_lohi_f8<PAIR>(d_tmem, a_lo, a_hi, b_lo, b_hi, idesc, kb != 0 ? 1u : 0u);
              tc_mma_lohi_f8<PAIR>(d_tmem, a_lo + a_step, a_hi, b_lo + b_step, b_hi, idesc, 1u);
              tc_mma_lohi_f8<PAIR>(d_tmem, a_lo + 2 * a_step, a_hi, b_lo + 2 * b_step, b_hi, idesc, 1u);
              tc_mma_lohi_f8<PAIR>(d_tmem, a_lo + 3 * a_step, a_hi, b_lo + 3 * b_step, b_hi, idesc, 1u);
            } else {
              tc_mma_lohi<PAIR>(d_tmem, a_lo, a_hi, b_lo, b_hi, idesc, kb != 0 ? 1u : 0u);
              tc_mma_lohi<PAIR>(d_tmem, a_lo + a_step, a_hi, b_lo + b_step, b_hi, idesc, 1u);
              tc_mma_lohi<PAIR>(d_tmem, a_lo + 2 * a_step, a_hi, b_lo + 2 * b_step, b_hi, idesc, 1u);
              tc_mma_lohi<PAIR>(d_tmem, a_lo + 3 * a_step, a_hi, b_lo + 3 * b_step, b_hi, idesc, 1u);
            }
            // stage reusable once these MMAs have read it (in both CTAs of a pair)
            if constexpr (PAIR) tc_commit_pair(ebar); else tc_commit(ebar);
          }
          __syncwarp();
          a_lo += SB16; b_lo += SB16; fbar += 8u; ebar += 8u;
          if (++stage == Cfg::STAGES) { stage = 0; phase ^= 1u; a_lo = a_lo0; b_lo = b_lo0; fbar = full_bar(0); ebar = empty_bar(0); }
        }
        if (!ok) break;
        if (elect_one()) { if constexpr (PAIR) tc_commit_pair(tfull_bar(acc)); else tc_commit(tfull_bar(acc)); }   // accumulator complete
        __syncwarp();
      }
      if (!ok && !PAIR) {
        // A wait was abandoned.  Products issued before it may still be running: they read the stage ring and
        // write tensor memory, so they must have finished before the teardown below releases either.  A commit
        // on a barrier of its own completes once every product issued so far is done (products wait for
        // nothing themselves, so this ends; the wait is bounded all the same).
        if (elect_one()) tc_commit(drain_bar);
        __syncwarp();
        const long long t0 = clock64();
        while (!mbar_try_wait(drain_bar, 0u) && clock64() - t0 < P.wait_cycles) {}
      }
    }
  } else if (warp == TC_TILE_WARP) {
    // ------------------------------------------------------------------ tiles
    // The grid has a CTA (pair) per tile, of which as many run as there is room for; a running one takes on the tile of
    // another that has not been launched yet whenever its loads begin a tile.  So it does not matter when an SM becomes free:
    // with tiles dealt out in advance, CTAs whose SM another stream's kernel held kept everybody waiting at the end, and the
    // SMs that had finished earlier idled.  Both sides in turn, us, with what two runs of one side differ by in brackets: steps at 512,
    // 8192, 16384 (Zipf) and 32768 tokens 1331 -> 1286 (0.0 %), 4955 -> 4844 (0.8), 8999 -> 8836 (0.5), 17304 -> 16926 (0.6), four d = 512
    // blocks 1510 -> 1454 (0.2), attention alone, whose streams rarely meet, 2152 -> 2142 (0.0), three whole blocks 21267 -> 21074 (0.7: no
    // difference shown); on other GPUs forward of 64 tokens 263 -> 249, the step at 2741 2225 -> 2177, with fused Adam at 8192 7501 -> 7312.
    // Where runs differ by 3-5 %, at the power cap, the steps from 8192 tokens on show nothing of it.
    // A tile's description costs this warp two divisions and a table look-up, one tile ahead of the loads.
    const int tiles_n = P.tr ? P.tiles_f : P.tiles_n;
    const int tiles_m = P.tr ? p.rows_total[1] : (PAIR ? (tiles_m_dev + 1) / 2 : tiles_m_dev);
    const int total = tiles_m * tiles_n * (p.group_mode == GROUP_K ? p.n_groups : 1);
    // A table of shorter runs than the launcher reckons with has more tiles than the grid: those follow at this distance.
    const int granted = PAIR ? (int)(gridDim.x >> 1) : (int)gridDim.x;
    int idx = PAIR ? (int)(blockIdx.x >> 1) : (int)blockIdx.x;
    uint32_t begun_phase = 0, answer_phase = 0, heard_phase = 0;
    bool ok = true, armed = false, asked = false;      // armed, asked: the answer's bytes are announced; the hardware has been asked
    auto describe = [&](const TcTile& t) -> bool {
      if (!mbar_wait_warp(dempty_bar(slot), slot_phase ^ 1u, abort_flag, p.status, P.wait_cycles)) return false;
      if (lane == 0) {
        tiles[slot] = t;
        mbar_arrive(dfull_bar(slot));
      }
      __syncwarp();
      if (++slot == TC_TILE_SLOTS) { slot = 0; slot_phase ^= 1u; }
      return true;
    };
    while (true) {
      // (a grid planned by a bound on the tiles has some that do not exist)
      for (; ok && idx < total; idx += granted) {
        ok = describe(tc_tile(P, idx, tiles_m, tiles_n, prank));
        if (ok && crank == 0) {
          ok = mbar_wait_warp(begun_bar, begun_phase, abort_flag, p.status, P.wait_cycles);
          begun_phase ^= 1u;
        }
      }
      if (!ok) break;
      if (lane == 0) mbar_expect_tx(answer_bar, 16);
      armed = true;
      if (crank == 0) {
        if (!(ok = mbar_wait_warp(heard_bar, heard_phase ^ 1u, abort_flag, p.status, P.wait_cycles))) break;
        heard_phase ^= 1u;
        if (elect_one()) clc_ask<PAIR>(answer, answer_bar);
        __syncwarp();
        asked = true;
      }
      if (!(ok = mbar_wait_warp(answer_bar, answer_phase, abort_flag, p.status, P.wait_cycles))) break;
      answer_phase ^= 1u;
      armed = asked = false;
      idx = clc_granted(answer);
      if (PAIR) idx >>= 1;            // -1 stays
      // read before the hardware writes the next one
      asm volatile("fence.proxy.async;" ::: "memory");
      __syncwarp();
      if (lane == 0) {
        if constexpr (PAIR) mbar_arrive_cluster(mapa_u32(heard_bar, 0));
        else mbar_arrive(heard_bar);
      }
      if (idx < 0) {
        const TcTile none = {};
        describe(none);
        break;
      }
    }
    if (!ok) {
      // A wait was abandoned.  An answer that is still on its way must not land in shared memory that this CTA no longer has;
      // and the CTAs that have not been launched yet must not be, each to wait for its own bound: this one takes what is left of the
      // grid and drops it (in a pair the even CTA, into its own shared memory alone: its partner has stopped listening, or will).
      auto settle = [&]() -> bool {
        const long long t0 = clock64();
        while (!__all_sync(0xffffffffu, mbar_try_wait(answer_bar, answer_phase)))
          if (__any_sync(0xffffffffu, clock64() - t0 > 4000000LL)) return false;
        answer_phase ^= 1u;
        return true;
      };
      if (crank != 0) {
        if (armed) settle();
      } else {
        for (int left = granted; left >= 0; --left) {      // (nothing may be asked after the answer that nothing is left)
          if (!asked) {
            if (!armed && lane == 0) mbar_expect_tx(answer_bar, 16);
            __syncwarp();
            if (elect_one()) clc_ask<false>(answer, answer_bar);
            __syncwarp();
          }
          if (!settle() || clc_granted(answer) < 0) break;
          armed = asked = false;
          asm volatile("fence.proxy.async;" ::: "memory");
          __syncwarp();
        }
      }
      __syncwarp();
    }
  } else {
    // ------------------------------------------------------------------ epilogue (warps 2..9)
    const int q = warp & 3;                      // TMEM lane quadrant this warp may access
    const int ew = warp - 2;                     // epilogue warp index
    const int half = ew >> 2;                    // this warp takes the 32-column blocks half, half+2, ...
    const int row_in_tile = q * 32 + lane;
    uint8_t* stg = gen_base + Cfg::EPI_OFF + ew * Cfg::EPI_WARP_BYTES;   // this warp's staging area
    const uint32_t stg_u32 = base + Cfg::EPI_OFF + ew * Cfg::EPI_WARP_BYTES;
    bool ok = true;
    int it = 0;
    uint32_t n_grp = 0;                          // bulk groups committed so far (same in every lane)
    // where this warp's slab of an fp32 result goes
    auto slab_of = [&](const TcTile& t) -> SlabOut {
      SlabOut out;
      const int y0 = (p.group_mode == GROUP_K ? t.group * p.M : 0) + t.m0 + q * 32;
      const int m_lim = (p.group_mode == GROUP_M) ? tiles_m_dev * TC_BM : p.M;
      int64_t yb = y0;
      const int64_t y_lim = (p.group_mode == GROUP_K) ? (int64_t)(t.group + 1) * p.M : (p.group_mode == GROUP_M ? (int64_t)m_lim : (int64_t)p.M);
      out.rows = (int)min((int64_t)32, y_lim - yb);
      out.c = reinterpret_cast<float*>(p.C);
      out.w = reinterpret_cast<bf16*>(p.upd_w);
      out.m = p.upd_m; out.mom = p.upd_mom; out.var = p.upd_var;
      if (WGRAD && p.split_m > 0) {
        // two outputs: the slab lies wholly in the first or in the second (split_m is a multiple of 128)
        int local = t.m0 + q * 32;
        if (local >= p.split_m) {
          local -= p.split_m;
          out.c = reinterpret_cast<float*>(p.C2); out.w = reinterpret_cast<bf16*>(p.upd_w2); out.m = p.upd_m2;
          out.mom = p.upd_mom2; out.var = p.upd_var2;
        }
        yb = (int64_t)t.group * p.split_m + local;
        out.rows = min(32, p.split_m - local);
      }
      if (UPD) out.at0 = (yb + half * 16) * p.ldc + t.n0 + lane * 4;
      else out.at0 = (yb + (lane >> 3)) * p.ldc + t.n0 + (lane & 7) * 4;
      out.ld4 = 4 * p.ldc;
      out.res0 = EPI == EPI_COUPLE ? (yb + (lane >> 3)) * p.ld_resid + t.n0 + (lane & 7) * 4 : 0;
      return out;
    };
    SlabOut next_out;      // Adam, row-wise: the next tile's slab, whose first units this tile has asked for (primed)
    bool primed = false;
    TcTile t;
    for (; ok; ++it) {
      if (next_tile(t) <= 0) break;
      const int acc = it & 1;
      const uint32_t acc_phase = (uint32_t)(it >> 1) & 1u;
      const int m = t.m0 + row_in_tile;
      const int m_lim = (p.group_mode == GROUP_M) ? tiles_m_dev * TC_BM : p.M;
      const bool m_ok = m < m_lim;
      const bool slab_ok = t.m0 + q * 32 < m_lim;             // this warp's 32 rows hold at least one real row
      const int rows_ok = min(32, m_lim - (t.m0 + q * 32));   // real rows among them (<= 0: none)
      // SwiGLU backward: the a|b operands of the warp's first block do not depend on the accumulator, so
      // their loads go out before the wait for it.  A lane takes 16-byte pieces lane % 4 of rows lane / 4 + 8 i of a block
      // of 32 rows x 32 columns (ds_a, ds_b; ds_rs: the rows' scales).
      const bool ds_tr = EPI == EPI_DSWIGLU && PAIR && P.tr;
      uint4 ds_a[4], ds_b[4];
      float ds_rs[4];
      bf16* ds_at = nullptr;          // this lane's piece of the row lane / 4 of the block at column (tr: token row) 0
      int64_t ds_step = 0, ds_row8 = 0;
      int ds_rows = 0;                // real rows of a block
      auto ds_load = [&](int i, int c) {
        const bool in = 8 * i + (lane >> 2) < ds_rows;
        const bf16* at = ds_at + c * ds_step + i * ds_row8;
        ds_a[i] = in ? __ldcg(reinterpret_cast<const uint4*>(at)) : make_uint4(0u, 0u, 0u, 0u);
        ds_b[i] = in ? __ldcg(reinterpret_cast<const uint4*>(at + p.N)) : make_uint4(0u, 0u, 0u, 0u);
      };
      auto ds_scale = [&](int row0) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int row = 8 * i + (lane >> 2);
          ds_rs[i] = p.rowscale && row < ds_rows ? p.rowscale[row0 + row] : 1.f;
        }
      };
      if constexpr (EPI == EPI_DSWIGLU) {
        ds_rows = ds_tr ? (t.n0 < p.N ? 32 : 0) : max(0, rows_ok);      // a pair's second half can lie past the last feature
        ds_step = ds_tr ? p.ld_ab : 1;
        ds_row8 = 8 * p.ld_ab;
        ds_at = reinterpret_cast<bf16*>(p.ab) + (int64_t)(t.m0 + (ds_tr ? 0 : q * 32) + (lane >> 2)) * p.ld_ab + t.n0 + (ds_tr ? q * 32 : 0) + (lane & 3) * 8;
        if (half * 32 < t.ncols) {
#pragma unroll
          for (int i = 0; i < 4; ++i) ds_load(i, half * 32);
          ds_scale(ds_tr ? t.m0 + half * 32 : t.m0 + q * 32);
        }
      }
      // row coordinate of the slab in the output tensor map (rows past its extent are clipped by the store)
      const int y0 = (p.group_mode == GROUP_K ? t.group * p.M : 0) + t.m0 + q * 32;
      uint4 ld[8];     // read-modify-write forms: a block's pieces, four floats or (in .x, .y) four bf16 weights
      SlabOut out;
      if constexpr (EPI == EPI_COUPLE || WGRAD || EPI == EPI_STORE) out = slab_of(t);
      auto rmw_request = [&](const SlabOut& o, int c, uint4 (&ld)[8]) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          if (i * 4 + (lane >> 3) >= o.rows) continue;
          const int64_t at = o.at0 + c + i * o.ld4;
          if (EPI == EPI_COUPLE) ld[i] = *reinterpret_cast<const uint4*>(p.resid + o.res0 + c + i * 4 * p.ld_resid);
          else if (!o.w) ld[i] = *reinterpret_cast<const uint4*>(o.c + at);
          else if (o.m) ld[i] = *reinterpret_cast<const uint4*>(o.m + at);
          else { const uint2 w2 = *reinterpret_cast<const uint2*>(o.w + at); ld[i].x = w2.x; ld[i].y = w2.y; }
        }
      };
      if constexpr (UPD) {
        if (slab_ok && !primed) {
          if (out.m) upd_first<EPI == EPI_WADAM, true>(out, stg, lane, p.ldc);
          else upd_first<EPI == EPI_WADAM, false>(out, stg, lane, p.ldc);
        }
      }
      if (!mbar_wait_warp(tfull_bar(acc), acc_phase, abort_flag, p.status, P.wait_cycles)) { ok = false; break; }
      tc_fence_after();
      const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * MMA_N);
      // accumulator may be overwritten by the MMA warp
      auto release = [&]() {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          if constexpr (PAIR) mbar_arrive_cluster(mapa_u32(tempty_bar(acc), 0));   // the even CTA's MMA warp waits for both
          else mbar_arrive(tempty_bar(acc));
        }
      };
      const bool have_acc = t.k_blocks > 0;      // an empty K range leaves the accumulator undefined: use zeros
      uint32_t r0[32];
      float f[32];

      if (PAIR && P.tr && EPI != EPI_DSWIGLU) {
        if constexpr (PAIR && (EPI == EPI_STORE || EPI == EPI_ROWSCALE)) {
          // Transposed tile: this lane holds output feature t.n0 + 32 q + lane for 32 token rows per block.
          // Lanes 2i and 2i+1 trade halves so that each ends up with feature PAIRS of single tokens (the even
          // lane of the even tokens, the odd lane of the odd ones), which it writes as 4-byte pieces into
          // the [32 tokens][32 features] staging block; a TMA store then writes 32 rows of 64 bytes.
          const bool odd = lane & 1;
#pragma unroll 1
          for (int c = half * 32; c < t.ncols; c += 64) {
            tmem_ld32(taddr + c, r0);
            tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < 32; ++i) f[i] = __uint_as_float(r0[i]);
            if (p.fp8) {
              // e4m3 operands: this lane's feature scale times the 32 tokens' row scales
              const float sw = p.b_scale0[(int64_t)t.group * p.N + t.n0 + q * 32 + lane];
              const float4* a4 = reinterpret_cast<const float4*>(p.a_scale + t.m0 + c);    // the same for every lane
#pragma unroll
              for (int i = 0; i < 8; ++i) {
                const float4 a = a4[i];
                f[4 * i] *= sw * a.x; f[4 * i + 1] *= sw * a.y; f[4 * i + 2] *= sw * a.z; f[4 * i + 3] *= sw * a.w;
              }
            }
            if constexpr (EPI == EPI_ROWSCALE) {
              const float4* g4 = reinterpret_cast<const float4*>(p.rowscale + t.m0 + c);   // the same for every lane
#pragma unroll
              for (int i = 0; i < 8; ++i) {
                const float4 g = g4[i];
                f[4 * i] *= g.x; f[4 * i + 1] *= g.y; f[4 * i + 2] *= g.z; f[4 * i + 3] *= g.w;
              }
            }
            const uint32_t off = (n_grp & 1u) * 2048u;
            if (lane == 0) bulk_wait_read<1>();
            __syncwarp();
            uint8_t* blk = stg + off;
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              const float send = odd ? f[2 * j] : f[2 * j + 1];
              const float recv = __shfl_xor_sync(0xffffffffu, send, 1);
              const int tok = 2 * j + (odd ? 1 : 0);
              const __nv_bfloat162 v = odd ? __floats2bfloat162_rn(recv, f[2 * j + 1]) : __floats2bfloat162_rn(f[2 * j], recv);
              const int piece = lane >> 3, within = ((lane >> 1) & 3) * 4;
              *reinterpret_cast<__nv_bfloat162*>(blk + tok * 64 + ((piece ^ ((tok >> 1) & 3)) << 4) + within) = v;
            }
            fence_async_smem();
            __syncwarp();
            if (lane == 0) {
              tma_store_2d(&map_c, stg_u32 + off, t.n0 + q * 32, t.m0 + c);
              bulk_commit();
            }
            ++n_grp;
          }
        }
        if constexpr (PAIR && EPI == EPI_SWIGLU) {
          // Transposed SwiGLU: of this warp's 32 lanes 16 hold gate rows, 16 the up rows of the same features, for 32
          // token rows per block.  Lanes l and l + 16 trade halves, each finishes 16 tokens of one feature; then, as
          // above, lanes 2i and 2i+1 trade so that feature pairs go to the staging area ([32 tokens][16 features], and
          // [32 tokens][16 + 16] for the a|b copy) and rows of 32 bytes from there to memory by plain stores.  The rows
          // of padding up to the next multiple of 64 are written as zeros: products over rows (weight gradients) read them.
          // Against 128 token rows x 128 columns of both matrices on one CTA, a pair brings 32 instead of 48 KB into
          // each SM per K step and pads a run of rows to 32 instead of 128 (experts' gate | up at 8192 tokens 302 -> 279 us,
          // with the copy 334 -> 295; at 2741 tokens 155 -> 138 and 167 -> 148)
          const bool odd = lane & 1, hi = lane >= 16, up_lane = hi != (P.tr_swap != 0);
          const int fw = t.n0 + q * 16;            // first feature of the warp
          float sw = 1.f;
          if (p.fp8) sw = (up_lane ? p.b_scale1 : p.b_scale0)[(int64_t)t.group * p.N + fw + (lane & 15)];
          bf16* const h_out = reinterpret_cast<bf16*>(p.C) + (int64_t)t.m0 * p.ldc + fw;
          bf16* const ab_out = reinterpret_cast<bf16*>(p.C1) + (int64_t)t.m0 * p.ldc1 + fw;
#pragma unroll 1
          for (int c = half * 32; c < t.ncols + t.pad; c += 64) {
            if (c < t.ncols) {
              tmem_ld32(taddr + c, r0);
              tmem_ld_wait();
            } else {
#pragma unroll
              for (int i = 0; i < 32; ++i) r0[i] = 0u;
            }
#pragma unroll
            for (int i = 0; i < 32; ++i) f[i] = __uint_as_float(r0[i]);
            if (p.fp8) {
              const float4* a4 = reinterpret_cast<const float4*>(p.a_scale + t.m0 + c);    // the same for every lane
#pragma unroll
              for (int i = 0; i < 8; ++i) {
                const float4 a = a4[i];
                f[4 * i] *= sw * a.x; f[4 * i + 1] *= sw * a.y; f[4 * i + 2] *= sw * a.z; f[4 * i + 3] *= sw * a.w;
              }
            }
            // two tokens of one feature in, one token of two features out
            auto trade = [&](float t0, float t1) -> uint32_t {
              const __nv_bfloat162 v = __floats2bfloat162_rn(t0, t1);
              const uint32_t own = *reinterpret_cast<const uint32_t*>(&v);
              const uint32_t other = __shfl_xor_sync(0xffffffffu, own, 1);
              return odd ? __byte_perm(other, own, 0x7632) : __byte_perm(own, other, 0x5410);
            };
            if (p.C1) {
              const int within = ((lane >> 1) & 3) * 4;
#pragma unroll
              for (int j = 0; j < 16; ++j) {
                const int tok = 2 * j + (odd ? 1 : 0);
                *reinterpret_cast<uint32_t*>(stg + tok * 64 + (((lane >> 3) ^ ((tok >> 1) & 3)) << 4) + within) = trade(f[2 * j], f[2 * j + 1]);
              }
            }
            float h[16], rs[16];
            if (p.rowscale) {
              const float4* g4 = reinterpret_cast<const float4*>(p.rowscale + t.m0 + c + (hi ? 16 : 0));
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                const float4 g = g4[i];
                rs[4 * i] = g.x; rs[4 * i + 1] = g.y; rs[4 * i + 2] = g.z; rs[4 * i + 3] = g.w;
              }
            } else {
#pragma unroll
              for (int i = 0; i < 16; ++i) rs[i] = 1.f;
            }
#pragma unroll
            for (int i = 0; i < 16; i += 2) {
              const float2 own = hi ? make_float2(f[16 + i], f[17 + i]) : make_float2(f[i], f[i + 1]);
              const float2 send = hi ? make_float2(f[i], f[i + 1]) : make_float2(f[16 + i], f[17 + i]);
              const float2 got = make_float2(__shfl_xor_sync(0xffffffffu, send.x, 16), __shfl_xor_sync(0xffffffffu, send.y, 16));
              const float2 A = up_lane ? got : own, B = up_lane ? own : got;
              const float2 Hh = __fmul2_rn(__fmul2_rn(__fmul2_rn(A, sigmoid_approx2(A)), B), make_float2(rs[i], rs[i + 1]));
              h[i] = Hh.x; h[i + 1] = Hh.y;
            }
            // a token's row of 32 bytes; the rows of tokens 16.. change places in pairs, away from the banks of tokens 0..
            auto slot = [](int tok) -> int { return (tok ^ ((tok >> 4) << 1)) * 32; };
#pragma unroll
            for (int j = 0; j < 8; ++j)
              *reinterpret_cast<uint32_t*>(stg + 2048 + slot((hi ? 16 : 0) + 2 * j + (odd ? 1 : 0)) + ((lane & 15) >> 1) * 4) = trade(h[2 * j], h[2 * j + 1]);
            __syncwarp();
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              const int tok = 16 * i + (lane >> 1);
              *reinterpret_cast<uint4*>(h_out + (int64_t)(c + tok) * p.ldc + (lane & 1) * 8) =
                  *reinterpret_cast<const uint4*>(stg + 2048 + slot(tok) + (lane & 1) * 16);
            }
            if (p.C1) {
              bf16* const dst = ab_out + ((((lane >> 1) & 1) != P.tr_swap) ? p.N : 0) + (lane & 1) * 8;
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                const int tok = 8 * i + (lane >> 2);
                *reinterpret_cast<uint4*>(dst + (int64_t)(c + tok) * p.ldc1) =
                    *reinterpret_cast<const uint4*>(stg + tok * 64 + (((lane & 3) ^ ((tok >> 1) & 3)) << 4));
              }
            }
            __syncwarp();
          }
        }
      } else if constexpr (EPI == EPI_STORE || EPI == EPI_ROWSCALE || EPI == EPI_COUPLE || WGRAD) {
        float rs = 1.f;
        if (EPI == EPI_ROWSCALE && m_ok) rs = p.rowscale[m];
        const bool f32_out = (EPI == EPI_COUPLE) || WGRAD || (EPI == EPI_STORE && p.out_f32);
        if (!f32_out) {
          // bf16 blocks (32 x 32, 2 KB) leave through two alternating staging buffers and TMA stores.
          if constexpr (EPI == EPI_STORE || EPI == EPI_ROWSCALE) {
#pragma unroll 1
            for (int c = half * 32; c < t.ncols; c += 64) {
              if (!slab_ok) continue;      // warp-uniform
              if (have_acc) { tmem_ld32(taddr + c, r0); tmem_ld_wait(); }
#pragma unroll
              for (int i = 0; i < 32; ++i) f[i] = have_acc ? __uint_as_float(r0[i]) : 0.f;
              if constexpr (EPI == EPI_ROWSCALE) {
#pragma unroll
                for (int i = 0; i < 32; ++i) f[i] *= rs;
              }
              const uint32_t off = (n_grp & 1u) * 2048u;
              if (lane == 0) bulk_wait_read<1>();
              __syncwarp();
              stage32_bf16(stg + off, lane, f);
              fence_async_smem();
              __syncwarp();
              if (lane == 0) {
                tma_store_2d(&map_c, stg_u32 + off, t.n0 + c, y0);
                bulk_commit();
              }
              ++n_grp;
            }
          }
        } else if (slab_ok) {
          // fp32 blocks (32 x 32, 4 KB) are transposed through the staging area and written with plain
          // 16-byte stores, 4 rows x 128 bytes per instruction: whole lines, and nothing to wait for
          // before the area is reused.  (A TMA store of such a block sat behind the producer's operand
          // loads in the copy engine; with the short K of a weight gradient that wait set the pace.)
          // A block's accumulator is fetched while the block before it is written.  With one K step per tile the kernel
          // writes 6 TB/s (experts' gate | up gradient at 512 tokens, 1.38 GB: 240 us); at 8192 tokens a tile's four blocks
          // take 6.5k clk beside 5k of main loop, 410 us.
          const int rsub = lane >> 3;
          const bool all_rows = out.rows >= 32;
          auto fetch = [&](int c) { if (have_acc && c < t.ncols) tmem_ld32(taddr + c, r0); };
          auto stage = [&]() {
            tmem_ld_wait();
            uint8_t* row = stg + lane * 128;
#pragma unroll
            for (int j = 0; j < 8; ++j)
              *reinterpret_cast<uint4*>(row + ((j ^ (lane & 7)) << 4)) =
                  have_acc ? make_uint4(r0[4 * j], r0[4 * j + 1], r0[4 * j + 2], r0[4 * j + 3]) : make_uint4(0u, 0u, 0u, 0u);
            __syncwarp();
          };
          auto staged = [&](int i) -> float4 {           // this lane's piece of row 4 i + rsub
            const int r = i * 4 + rsub;
            return *reinterpret_cast<const float4*>(stg + r * 128 + (((lane & 7) ^ (r & 7)) << 4));
          };
          auto row_ok = [&](int i) -> bool { return all_rows || i * 4 + rsub < out.rows; };
          if (!RMW && !UPD) fetch(half * 32);
          if constexpr (UPD) {
            // Fused update of the grouped products, whose short K leaves the kernel bound by what this reads and writes.
            // HBM serves the four arrays' 128-byte pieces of the block-wise form at 4.1 TB/s, 512-byte pieces at 5.3
            // (a bare read-modify-write kernel, 26 bytes per element, 148 CTAs; bf16 weights alone: 64-byte pieces 3.9,
            // 256-byte 5.3).  So a warp takes 16 whole rows of its quadrant, 128 columns at a time: the accumulator goes
            // through a 16 x 128 staging area, weights and moments of two rows at a time come by cp.async into
            // a ring, one instruction is one row.
            for (int cb = 0; cb * 128 < t.ncols; ++cb) {
#pragma unroll 1
              for (int jj = 0; jj < 4; ++jj) {
                if (have_acc) { tmem_ld32(taddr + cb * 128 + jj * 32, r0); tmem_ld_wait(); }
                if ((lane >> 4) == half) {
                  uint8_t* row = stg + (lane & 15) * 512;
#pragma unroll
                  for (int j = 0; j < 8; ++j)
                    *reinterpret_cast<uint4*>(row + ((jj * 8 + (j ^ (lane & 7))) << 4)) =
                        have_acc ? make_uint4(r0[4 * j], r0[4 * j + 1], r0[4 * j + 2], r0[4 * j + 3]) : make_uint4(0u, 0u, 0u, 0u);
                }
                __syncwarp();
              }
              const bool last = cb * 128 + 128 >= t.ncols;
              if (last) release();      // the tile's last columns are out of tensor memory
              if (last) {
                // (the next tile, where it is described already: the loads are ahead of this warp)
                primed = EPI == EPI_WADAM && __all_sync(0xffffffffu, mbar_try_wait(dfull_bar(slot), slot_phase));
                if (primed) {
                  const TcTile tn = tiles[slot];
                  next_out = slab_of(tn);
                  primed = tn.valid && next_out.rows > 0;
                }
              }
              if (out.m) upd_half<EPI == EPI_WADAM, true>(p.upd, out, next_out, stg, lane, p.ldc, cb, last, primed);
              else upd_half<EPI == EPI_WADAM, false>(p.upd, out, next_out, stg, lane, p.ldc, cb, last, primed);
              __syncwarp();
            }
          } else {
            // Read-modify-write forms (coupling, accumulation, fused updates of dense products, whose long K hides them):
            // all a block needs is requested before its accumulator is fetched.
            auto write_adam = [&](int c) {
#pragma unroll 1
              for (int h4 = 0; h4 < 8; h4 += 4) {      // four pieces at a time keep the registers in bounds
                float4 w4[4], mo[4], va[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                  if (!row_ok(h4 + i)) continue;
                  const int64_t at = out.at0 + c + (h4 + i) * out.ld4;
                  w4[i] = out.m ? *reinterpret_cast<const float4*>(out.m + at) : bf4(*reinterpret_cast<const uint2*>(out.w + at));
                  mo[i] = *reinterpret_cast<const float4*>(out.mom + at);
                  va[i] = *reinterpret_cast<const float4*>(out.var + at);
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                  if (!row_ok(h4 + i)) continue;
                  const float4 v = staged(h4 + i);
                  const int64_t at = out.at0 + c + (h4 + i) * out.ld4;
                  w4[i].x = upd_step(p.upd, w4[i].x, v.x, &mo[i].x, &va[i].x);
                  w4[i].y = upd_step(p.upd, w4[i].y, v.y, &mo[i].y, &va[i].y);
                  w4[i].z = upd_step(p.upd, w4[i].z, v.z, &mo[i].z, &va[i].z);
                  w4[i].w = upd_step(p.upd, w4[i].w, v.w, &mo[i].w, &va[i].w);
                  *reinterpret_cast<float4*>(out.mom + at) = mo[i];
                  *reinterpret_cast<float4*>(out.var + at) = va[i];
                  if (out.m) *reinterpret_cast<float4*>(out.m + at) = w4[i];
                  *reinterpret_cast<uint2*>(out.w + at) = pack4(w4[i]);
                }
              }
            };
            auto write = [&](int c, const uint4 (&ld)[8]) {
#pragma unroll
              for (int i = 0; i < 8; ++i) {
                if (!row_ok(i)) continue;
                float4 v = staged(i);
                const int64_t at = out.at0 + c + i * out.ld4;
                if (EPI == EPI_COUPLE) {
                  const float4 o = as_f4(ld[i]);
                  v = make_float4(o.x + p.resid_sign * v.x, o.y + p.resid_sign * v.y, o.z + p.resid_sign * v.z, o.w + p.resid_sign * v.w);
                } else if (EPI == EPI_WRMW) {
                  if (!out.w) {          // accumulate into the stored gradient
                    const float4 o = as_f4(ld[i]);
                    v = make_float4(o.x + v.x, o.y + v.y, o.z + v.z, o.w + v.w);
                  } else {
                    // fused update on the weight tile this gradient tile belongs to; the gradient is not stored
                    float4 w4 = out.m ? as_f4(ld[i]) : bf4(make_uint2(ld[i].x, ld[i].y));
                    w4.x -= p.upd.lr * v.x; w4.y -= p.upd.lr * v.y; w4.z -= p.upd.lr * v.z; w4.w -= p.upd.lr * v.w;
                    if (out.m) *reinterpret_cast<float4*>(out.m + at) = w4;
                    *reinterpret_cast<uint2*>(out.w + at) = pack4(w4);
                    continue;
                  }
                }
                *reinterpret_cast<float4*>(out.c + at) = v;
              }
            };
#pragma unroll 1
            for (int c = half * 32; c < t.ncols; c += 64) {
              const bool adam = EPI == EPI_WRMW && out.w && out.mom;
              if (RMW && !adam) rmw_request(out, c, ld);
              if (RMW) fetch(c);
              stage();
              if (!RMW) fetch(c + 64);
              if (adam) write_adam(c); else write(c, ld);
              __syncwarp();
            }
          }
        }
      } else if constexpr (EPI == EPI_HEADS) {
        // Columns are heads of 128: the tile holds two (or, ragged, one).  This warp's 32-column blocks c and c + 64
        // are the two halves of a rotated pair range: bias, rotation by the position's angles, bf16, and out as
        // 64-byte pieces of the row's place in the head-major tensor.
        uint32_t r1[32];
        const int seq = m_ok ? m / p.hm_S : 0, pos = m_ok ? m % p.hm_S : 0;
        const bool other = p.hm_split && t.n0 >= p.hm_split;      // the second matrix
        const int n_heads = (!p.hm_split ? p.N : (other ? p.N - p.hm_split : p.hm_split)) / 128;
        const float* const bias = other ? p.hm_bias1 : p.hm_bias;
        const int64_t row_at = ((int64_t)seq * n_heads * p.hm_Sp + pos) * 128;      // this lane's row, head 0
#pragma unroll 1
        for (int c = half * 32; c < t.ncols; c += 128) {
          if (!slab_ok) continue;      // warp-uniform
          const int n = t.n0 + c - (other ? p.hm_split : 0);      // first column of the lower half-range; n + 64 is its partner
          tmem_ld32(taddr + c, r0);
          tmem_ld32(taddr + c + 64, r1);
          tmem_ld_wait();
          const int head = n / 128, i0 = n % 128;            // i0 is 0 or 32
          bf16* dst = reinterpret_cast<bf16*>(other ? p.C1 : p.C) + (int64_t)head * p.hm_Sp * 128 + i0;
          float y0[32], y1[32];
#pragma unroll
          for (int i = 0; i < 32; ++i) { y0[i] = __uint_as_float(r0[i]); y1[i] = __uint_as_float(r1[i]); }
          if (bias) {
            const float4* b0 = reinterpret_cast<const float4*>(bias + n);        // the same for every lane
            const float4* b1 = reinterpret_cast<const float4*>(bias + n + 64);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              const float4 u = b0[i], v = b1[i];
              y0[4 * i] += u.x; y0[4 * i + 1] += u.y; y0[4 * i + 2] += u.z; y0[4 * i + 3] += u.w;
              y1[4 * i] += v.x; y1[4 * i + 1] += v.y; y1[4 * i + 2] += v.z; y1[4 * i + 3] += v.w;
            }
          }
          if (p.hm_cs && !other) {
            // the table is [pair, position]: the lanes' positions are neighbours
            const float2* cs2 = p.hm_cs + (int64_t)i0 * p.hm_S + pos;
#pragma unroll
            for (int i = 0; i < 32; ++i) {
              const float2 cs = cs2[(int64_t)i * p.hm_S];
              const float a0 = y0[i], b0v = y1[i];
              y0[i] = a0 * cs.x - b0v * cs.y;
              y1[i] = b0v * cs.x + a0 * cs.y;
            }
          }
          // out through the staging area, eight rows of 64 bytes per instruction (rows of a slab may belong to two
          // sequences, so each row's address comes from its lane)
          stage32_bf16(stg, lane, y0);
          stage32_bf16(stg + 2048, lane, y1);
          __syncwarp();
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int r = 8 * i + (lane >> 2);
            const int64_t at = __shfl_sync(0xffffffffu, row_at, r);
            const int off = r * 64 + (((lane & 3) ^ ((r >> 1) & 3)) << 4);
            const uint4 v0 = *reinterpret_cast<const uint4*>(stg + off), v1 = *reinterpret_cast<const uint4*>(stg + 2048 + off);
            if (r < rows_ok) {
              *reinterpret_cast<uint4*>(dst + at + (lane & 3) * 8) = v0;
              *reinterpret_cast<uint4*>(dst + at + 64 + (lane & 3) * 8) = v1;
            }
          }
          __syncwarp();
        }
      } else if constexpr (EPI == EPI_SWIGLU) {
        // columns [0, tile_n) hold the gate projection, [tile_n, 2 tile_n) the up projection.
        // H (times the row's scale, when one is given: the routed experts' gate weight) goes out through two
        // alternating 2 KB staging buffers and TMA stores; when the a|b copy is wanted too, a|b and H take turns
        // in the staging area.  (Plain line-wide stores for the a|b copy measured 0.01 ms slower per launch.)
        uint32_t r1[32];
        float g[32];
        const float rs = (p.rowscale && m_ok) ? p.rowscale[m] : 1.f;
#pragma unroll 1
        for (int c = half * 32; c < P.tile_n; c += 64) {
          const int n = t.n0 + c;
          if (!slab_ok) continue;      // warp-uniform
          tmem_ld32(taddr + c, r0);
          tmem_ld32(taddr + P.tile_n + c, r1);
          tmem_ld_wait();
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            f[i] = __uint_as_float(r0[i]);
            g[i] = __uint_as_float(r1[i]);
          }
          if (p.fp8) {
            // e4m3 operands: the sums of code products times the row's and the columns' scales
            const float sa = m_ok ? p.a_scale[m] : 0.f;
            const int64_t col0 = (p.group_mode == GROUP_M ? (int64_t)t.group * p.N : 0) + n;
            const float4* s0 = reinterpret_cast<const float4*>(p.b_scale0 + col0);      // the same for every lane
            const float4* s1 = reinterpret_cast<const float4*>(p.b_scale1 + col0);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              const float4 u0 = s0[i], u1 = s1[i];
              f[4 * i] *= sa * u0.x; f[4 * i + 1] *= sa * u0.y; f[4 * i + 2] *= sa * u0.z; f[4 * i + 3] *= sa * u0.w;
              g[4 * i] *= sa * u1.x; g[4 * i + 1] *= sa * u1.y; g[4 * i + 2] *= sa * u1.z; g[4 * i + 3] *= sa * u1.w;
            }
          }
          if (p.C1) {
            // the a|b copy goes first, through the whole staging area; H follows once that store has read it
            if (lane == 0) bulk_wait_read<0>();
            __syncwarp();
            stage32_bf16(stg, lane, f);
            stage32_bf16(stg + 2048, lane, g);
            fence_async_smem();
            __syncwarp();
            if (lane == 0) {
              tma_store_2d(&map_c1, stg_u32, n, y0);
              tma_store_2d(&map_c1, stg_u32 + 2048, p.N + n, y0);
              bulk_commit();
            }
          }
#pragma unroll
          for (int i = 0; i < 32; i += 2) {
            const float2 A = make_float2(f[i], f[i + 1]);
            const float2 Hh = __fmul2_rn(__fmul2_rn(__fmul2_rn(A, sigmoid_approx2(A)), make_float2(g[i], g[i + 1])), make_float2(rs, rs));
            f[i] = Hh.x; f[i + 1] = Hh.y;
          }
          const uint32_t off = p.C1 ? 0u : (n_grp & 1u) * 2048u;
          if (lane == 0) { if (p.C1) bulk_wait_read<0>(); else bulk_wait_read<1>(); }
          __syncwarp();
          stage32_bf16(stg + off, lane, f);
          fence_async_smem();
          __syncwarp();
          if (lane == 0) {
            tma_store_2d(&map_c, stg_u32 + off, n, y0);
            bulk_commit();
          }
          ++n_grp;
        }
      } else {   // EPI_DSWIGLU
        // The accumulator block goes through the staging area as fp32 into the distributed form in which a|b
        // arrive and da|db leave, straight from and to memory in rows of 64 bytes (transposed tiles: lane = feature,
        // so the staging write transposes).  A piece of the next block is requested as soon as this one's registers
        // are free, the next block's accumulator while this one is worked on.
        // (With a|b and da|db through the staging area and the accumulator in place, and the experts' rows in 128-row
        // tiles: experts' product 231 us at 8192 tokens, 112 at 2741, 93 at 512, now 210, 99, 77; the shared expert's at 8192
        // 166 -> 147.  It still sets the pace, 3.6k clk per block of the warp beside 18.6k of main loop per tile: without its
        // stores a block takes 2.7k, without its loads 2.0k, without exponentials as long as with them.  Asking a tile
        // ahead for L2 prefetches or a whole block ahead into other registers changes nothing.)
        const bool any = ds_rows > 0;            // warp-uniform
        float dg[4] = {0.f, 0.f, 0.f, 0.f};
        // sums over the four lanes of a row; lane (row, i) ends up with the row 8 i + lane / 4
        auto dg_out = [&](int row0, int rows, int part) {
          float mine = 0.f;
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            float v = dg[i];
            v += __shfl_xor_sync(0xffffffffu, v, 1);
            v += __shfl_xor_sync(0xffffffffu, v, 2);
            if ((lane & 3) == i) mine = v;
            dg[i] = 0.f;
          }
          const int row = 8 * (lane & 3) + (lane >> 2);
          if (row < rows) p.dg_part[(int64_t)(row0 + row) * p.dg_ld + part] = mine;
        };
        if (any && half * 32 < t.ncols) tmem_ld32(taddr + half * 32, r0);
#pragma unroll 1
        for (int c = half * 32; c < t.ncols; c += 64) {
          if (!any) continue;
          const bool more = c + 64 < t.ncols;
          tmem_ld_wait();
          if (ds_tr) {
#pragma unroll
            for (int i = 0; i < 32; ++i)
              *reinterpret_cast<uint32_t*>(stg + i * 128 + (((lane >> 2) ^ (i & 7)) << 4) + (lane & 3) * 4) = r0[i];
          } else {
#pragma unroll
            for (int j = 0; j < 8; ++j)
              *reinterpret_cast<uint4*>(stg + lane * 128 + ((j ^ (lane & 7)) << 4)) =
                  make_uint4(r0[4 * j], r0[4 * j + 1], r0[4 * j + 2], r0[4 * j + 3]);
          }
          __syncwarp();
          if (more) tmem_ld32(taddr + c + 64, r0);
          bf16* const out_at = ds_at + c * ds_step;
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int row = 8 * i + (lane >> 2);
            const float4 v0 = *reinterpret_cast<const float4*>(stg + row * 128 + (((2 * (lane & 3)) ^ (row & 7)) << 4));
            const float4 v1 = *reinterpret_cast<const float4*>(stg + row * 128 + (((2 * (lane & 3) + 1) ^ (row & 7)) << 4));
            const float v[8] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w};
            float a[8], b[8];
            unpack8(ds_a[i], a);
            unpack8(ds_b[i], b);
            if (more) ds_load(i, c + 64);
            float2 dg2 = make_float2(0.f, 0.f);
            // two elements at a time on the packed fp32 pipe (half the instructions of the scalar form)
#pragma unroll
            for (int e = 0; e < 8; e += 2) {
              const float2 A = make_float2(a[e], a[e + 1]), B = make_float2(b[e], b[e + 1]), V = make_float2(v[e], v[e + 1]);
              const float2 S = sigmoid_approx2(A);
              const float2 SI = __fmul2_rn(A, S);                         // silu(a)
              const float2 DH = __fmul2_rn(make_float2(ds_rs[i], ds_rs[i]), V);       // dL/dH of this row
              dg2 = __ffma2_rn(V, __fmul2_rn(SI, B), dg2);                // <dH', H>: gradient of the row's gate weight
              // da = dh b silu'(a), silu'(a) = s (1 + a (1 - s)) = s (1 + a - silu(a));  db = dh silu(a)
              const float2 T1 = __fadd2_rn(__fadd2_rn(A, make_float2(1.f, 1.f)), make_float2(-SI.x, -SI.y));
              const float2 DA = __fmul2_rn(__fmul2_rn(DH, B), __fmul2_rn(S, T1));
              const float2 DB = __fmul2_rn(DH, SI);
              a[e] = DA.x; a[e + 1] = DA.y; b[e] = DB.x; b[e + 1] = DB.y;
            }
            dg[i] += dg2.x + dg2.y;
            if (row < ds_rows) {
              *reinterpret_cast<uint4*>(out_at + i * ds_row8) = pack8(a);
              *reinterpret_cast<uint4*>(out_at + i * ds_row8 + p.N) = pack8(b);
            }
          }
          if (ds_tr) {
            if (p.dg_part) dg_out(t.m0 + c, 32, t.n0 / 32 + q);
            if (more) ds_scale(t.m0 + c + 64);
          }
          __syncwarp();
        }
        if (!ds_tr && any && p.dg_part) dg_out(t.m0 + q * 32, ds_rows, 2 * (t.n0 / P.tile_n) + half);
      }
      if (!UPD || !slab_ok) release();
    }
    // this lane's stores must be complete (shared memory read, global memory written) before the CTA exits
    if (lane == 0) bulk_wait_all();
    if constexpr (UPD) cp_async_wait<0>();
  }

  // ------------------------------------------------------------------ teardown
  __syncthreads();
  if (*abort_flag && threadIdx.x == 0) {
    // loads already issued into this CTA's shared memory must land before the CTA exits
    bool unannounced = false;     // the second load warp issued into a stage whose bytes the first never announced
    for (int s = 0; s < Cfg::STAGES; ++s) {
      if (issued_b[s] != 0 && issued_b[s] != issued[s]) unannounced = true;
      if (issued[s] == 0) continue;
      long long t0 = clock64();
      while (!mbar_try_wait(full_bar(s), (uint32_t)(issued[s] - 1)) && clock64() - t0 < P.wait_cycles) {}
    }
    if (unannounced) {            // that stage's barrier cannot complete: give its loads a bounded time to land
      const long long t0 = clock64();
      while (clock64() - t0 < 4000000LL) {}
    }
  }
  __syncthreads();
  if constexpr (PAIR) {
    // After an abandoned wait, loads of this CTA may still be in flight (their completion is counted on the
    // even CTA's barriers, so the per-stage drain above does not see them): give them a bounded time to land.
    if (*abort_flag) {
      const long long t0 = clock64();
      while (clock64() - t0 < 4000000LL) {}
    }
    // neither CTA frees tensor memory or leaves while the other may still signal its barriers or
    // have MMAs in flight that write its accumulators
    tc_fence_before();
    cluster_sync_all();
  }
  if (warp == 1) {
    tc_fence_after();
    if constexpr (PAIR)
      asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)Cfg::TMEM_COLS)
                   : "memory");
    else
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)Cfg::TMEM_COLS)
                   : "memory");
  }
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// Per-device set-up state (kernel attributes and the SM count belong to a device, not to the process).
struct TcState {
  EncodeTiledFn encode = nullptr;
  int n_sms = 0;
  bool ready = false;
};
constexpr int TC_MAX_DEVICES = 64;
// State of the current device; devices beyond the table share the last slot and are refused by tc_prepare.
inline TcState& tc_state() {
  static TcState s[TC_MAX_DEVICES + 1];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= TC_MAX_DEVICES) dev = TC_MAX_DEVICES;
  return s[dev];
}

template <int MMA_N, int EPI>
inline cudaError_t tc_set_attr() {
  cudaError_t e = cudaFuncSetAttribute(gemm_tc_kernel<MMA_N, EPI, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       TcCfg<MMA_N, EPI, false>::SMEM_BYTES);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(gemm_tc_kernel<MMA_N, EPI, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              TcCfg<MMA_N, EPI, true>::SMEM_BYTES);
}

// Once per device (under a lock: two host threads may arrive together): driver entry point for tensor-map
// encoding, SM count, shared-memory opt-in of every kernel instance.
inline int tc_prepare() {
  static std::mutex mu;
  std::lock_guard<std::mutex> lock(mu);
  TcState& s = tc_state();
  if (s.ready) return REVFFN_OK;
  {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return REVFFN_ERR_CUDA;
    if (dev < 0 || dev >= TC_MAX_DEVICES) return REVFFN_ERR_UNSUPPORTED;
  }
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult qres;
  if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres) != cudaSuccess || !fn)
    return REVFFN_ERR_CUDA;
  s.encode = reinterpret_cast<EncodeTiledFn>(fn);
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return REVFFN_ERR_CUDA;
  if (cudaDeviceGetAttribute(&s.n_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return REVFFN_ERR_CUDA;
  cudaError_t e = cudaSuccess;
  if (e == cudaSuccess) e = tc_set_attr<256, EPI_STORE>();
  if (e == cudaSuccess) e = tc_set_attr<256, EPI_SWIGLU>();
  if (e == cudaSuccess) e = tc_set_attr<256, EPI_ROWSCALE>();
  if (e == cudaSuccess) e = tc_set_attr<256, EPI_COUPLE>();
  if (e == cudaSuccess) e = tc_set_attr<256, EPI_DSWIGLU>();
  if (e == cudaSuccess) e = tc_set_attr<256, EPI_WGRAD>();
  if (e == cudaSuccess) e = tc_set_attr<256, EPI_WADAM>();
  if (e == cudaSuccess) e = tc_set_attr<256, EPI_WSGD>();
  if (e == cudaSuccess) e = tc_set_attr<256, EPI_WRMW>();
  if (e == cudaSuccess) e = tc_set_attr<256, EPI_HEADS>();
  if (e != cudaSuccess) return REVFFN_ERR_CUDA;
  s.ready = true;
  return REVFFN_OK;
}

// 2D bf16 tensor map: `inner` contiguous elements per row, `outer` rows of stride ld elements.
// u8 = true: one-byte elements (e4m3 codes), box_inner counts bytes.
inline int tc_make_map(CUtensorMap* map, const void* ptr, uint64_t inner, uint64_t outer, uint64_t ld,
                       uint32_t box_inner, uint32_t box_outer, bool u8 = false) {
  cuuint64_t dims[2] = {inner, outer};
  cuuint64_t strides[1] = {ld * (u8 ? 1u : 2u)};
  cuuint32_t box[2] = {box_inner, box_outer};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = tc_state().encode(map, u8 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box,
                                 estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                 CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? REVFFN_OK : REVFFN_ERR_CUDA;
}

// Tensor map of an MN-major bf16 operand ([rows, ld] in memory, rows = K) seen as {64 columns, rows, ld / 64
// column groups}: a box of 64 x 64 x 2 is 128 columns of 64 K rows, delivered as two 8 KB blocks of 64 columns.
inline int tc_make_map_mn3d(CUtensorMap* map, const void* ptr, uint64_t rows, uint64_t ld, int box_cols = 128) {
  cuuint64_t dims[3] = {64, rows, ld / 64};
  cuuint64_t strides[2] = {ld * 2u, 128u};
  cuuint32_t box[3] = {64, 64, (cuuint32_t)box_cols / 64};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = tc_state().encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(ptr), dims, strides, box, estr,
                                 CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                 CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? REVFFN_OK : REVFFN_ERR_CUDA;
}

// Two [groups * N, K] weight matrices of one layout seen as {K, 16 rows, 2 matrices, groups of 16 rows}: a box of
// 128 bytes x 16 x 2 x 4 is 64 rows of both, 16 of one and 16 of the other in turn.  The step between the matrices is the
// distance of their addresses.
inline int tc_make_map_rows16(CUtensorMap* map, const GemmProblem& p) {
  const uintptr_t b0 = reinterpret_cast<uintptr_t>(p.B0), b1 = reinterpret_cast<uintptr_t>(p.B1);
  const uint64_t es = p.fp8 ? 1 : 2, dist = b0 < b1 ? b1 - b0 : b0 - b1, rows = (uint64_t)(p.n_groups > 0 ? p.n_groups : 1) * p.N;
  if (!p.B0 || !p.B1 || dist == 0 || dist % 16 != 0 || dist >= (1ull << 40)) return REVFFN_ERR_UNSUPPORTED;
  cuuint64_t dims[4] = {(cuuint64_t)p.K, 16, 2, rows / 16};
  cuuint64_t strides[3] = {(cuuint64_t)p.ldb * es, dist, 16 * (cuuint64_t)p.ldb * es};
  cuuint32_t box[4] = {p.fp8 ? 128u : 64u, 16, 2, 4};
  cuuint32_t estr[4] = {1, 1, 1, 1};
  CUresult r = tc_state().encode(map, p.fp8 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4,
                                 reinterpret_cast<void*>(b0 < b1 ? b0 : b1), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                                 CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? REVFFN_OK : REVFFN_ERR_CUDA;
}

// Tensor map of an epilogue output: boxes of 32 rows x 64 bytes (32 bf16 or 16 fp32 columns),
// 64-byte swizzle.
inline int tc_make_out_map(CUtensorMap* map, const void* ptr, bool f32, uint64_t inner, uint64_t outer, uint64_t ld) {
  cuuint64_t dims[2] = {inner, outer};
  cuuint64_t strides[1] = {ld * (f32 ? 4u : 2u)};
  cuuint32_t box[2] = {f32 ? 16u : 32u, 32};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = tc_state().encode(map, f32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2,
                                 const_cast<void*>(ptr), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                                 CU_TENSOR_MAP_SWIZZLE_64B,
                                 CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? REVFFN_OK : REVFFN_ERR_CUDA;
}


template <int MMA_N, int EPI>
inline int tc_launch(const TcParams& P, const CUtensorMap& ma, const CUtensorMap& mb0, const CUtensorMap& mb1,
                     const CUtensorMap& mc, const CUtensorMap& mc1, int grid, bool pair, cudaStream_t st) {
  const cudaError_t e =
      pair ? launch_cluster(gemm_tc_kernel<MMA_N, EPI, true>, dim3((unsigned)grid), dim3(2), dim3(TC_THREADS),
                            TcCfg<MMA_N, EPI, true>::SMEM_BYTES, st, P, ma, mb0, mb1, mc, mc1)
           : launch_k(gemm_tc_kernel<MMA_N, EPI, false>, dim3((unsigned)grid), dim3(TC_THREADS),
                      TcCfg<MMA_N, EPI, false>::SMEM_BYTES, st, P, ma, mb0, mb1, mc, mc1);
  return e == cudaSuccess ? REVFFN_OK : REVFFN_ERR_CUDA;
}

// How a product is cut: CTA pairs or single CTAs, columns per tile, and whether it runs transposed.
struct TcPlan { bool tr, pair; int tile_n; };

// Pair mode is open wherever a 256-row tile cannot straddle two experts, transposed pair mode to expert-grouped bf16
// stores, gate-scaled ones, SwiGLU and SwiGLU backward.  (With 256 columns a ragged 128-wide last tile splits into 64-column halves, which only the [K, N] storage
// of B can load.)  A product whose wide tiles do not fill the GPU once is latency: it takes the narrower tile with the
// shortest reckoned time (main loop plus fill and epilogue), if that is a fifth shorter.  The constants are clocks measured
// on the kernel: a K step is bound by its tensor work (2 clk per column; the pair's instructions add about 90) or by the
// bytes it brings into an SM (about 68 B/clk); an epilogue takes about 10 clk per column of bf16 and 22 of fp32; the
// first loads and the start take 2500.  Four d = 512 blocks, 384 tokens: 1990 -> 1738 us a step; forward of 64 tokens
// 304 -> 291.  Products that fill the GPU keep wide tiles even where the last round is thin: narrow ones move more
// bytes per flop, and another stream's kernels use the SMs that are left over (chosen by time alone, a step at 2741
// tokens went from 2547 to 2689 us, at 512 from 1504 to 1574).
inline TcPlan tc_plan(const GemmProblem& p, int n_sms) {
  TcPlan wide;
  const bool cat = p.concat == CONCAT_N;
  wide.tr = p.group_mode == GROUP_M && p.tok_chunks != nullptr && !p.a_mn_major && !p.no_pair && n_sms % 2 == 0 &&
            (cat ? p.epilogue == EPI_SWIGLU && !p.b_mn_major
                 : p.epilogue == EPI_DSWIGLU ? p.b_mn_major && p.concat == CONCAT_NONE
                 : p.N % 256 == 0 && (p.epilogue == EPI_ROWSCALE || (p.epilogue == EPI_STORE && !p.out_f32)));
  wide.pair = wide.tr || (p.group_mode != GROUP_M && (p.N % 256 == 0 || p.b_mn_major) && !p.no_pair);
  wide.tile_n = cat ? 128 : 256;
  if (p.dbg_tile_n) {
    wide.tile_n = p.dbg_tile_n;
    wide.pair = p.group_mode != GROUP_M && !p.no_pair && (cat || (p.dbg_tile_n == 256 ? wide.pair : p.dbg_tile_n >= 128));
    return wide;
  }
  // a pair of matrices whose transposed tiles leave SMs idle is better off with the row tiles below, which can be narrow
  // (four d = 512 blocks, eight experts of 144 rows: 1663 us a step with transposed tiles, 1630 without)
  if (wide.tr && (cat || p.epilogue == EPI_DSWIGLU) &&
      ((p.M - 127 * (int64_t)p.n_groups) / 256 + p.n_groups / 2) * ceil_div(p.N, cat ? 128 : 256) < n_sms / 2)
    wide.tr = wide.pair = false;
  if (wide.tr || p.fp8 || p.upd_w) return wide;
  const bool pair_open = p.group_mode != GROUP_M && !p.no_pair && n_sms % 2 == 0;
  const int64_t groups = p.group_mode == GROUP_K ? (p.n_groups > 0 ? p.n_groups : 1) : 1;
  int64_t k_steps = ceil_div(p.K, TC_BK);
  int64_t m_tiles = ceil_div(p.M, TC_BM);
  if (p.group_mode == GROUP_K) k_steps = std::max<int64_t>(1, k_steps / groups);
  // padded row space: about half a tile of padding per expert
  if (p.group_mode == GROUP_M && p.n_groups > 0) m_tiles = std::max<int64_t>(1, (p.M - 127 * (int64_t)p.n_groups) / TC_BM + p.n_groups / 2);
  auto slots = [&](bool pair) -> int64_t { return pair ? n_sms / 2 : n_sms; };
  auto tiles = [&](bool pair, int tile_n) { return (pair ? (m_tiles + 1) / 2 : m_tiles) * ceil_div(p.N, tile_n) * groups; };
  if (tiles(wide.pair, wide.tile_n) > slots(wide.pair)) return wide;
  const bool f32_out = p.epilogue == EPI_COUPLE || p.epilogue == EPI_WGRAD || p.out_f32;
  const int epi_clk = p.epilogue == EPI_DSWIGLU ? 70 : (f32_out || cat ? 22 : 10);
  auto clocks = [&](bool pair, int tile_n) {
    const int64_t cols = cat ? 2 * tile_n : tile_n;         // accumulator columns
    const int64_t rounds = ceil_div(tiles(pair, tile_n), slots(pair)), bytes = TC_A_BYTES + cols * (pair ? 64 : 128);
    const int64_t step = std::max<int64_t>(2 * cols + (pair ? 90 : 0), bytes / 68), epi = epi_clk * cols;
    return 2500 + rounds * std::max(k_steps * step, epi) + epi;
  };
  TcPlan best = wide;
  int64_t best_clk = clocks(wide.pair, wide.tile_n) * 4 / 5;
  // a head must not straddle tiles; the sums of <dH, H> are two per 256 columns; 64 columns of both matrices of a pair
  const int narrowest = p.epilogue == EPI_HEADS ? 128 : (p.epilogue == EPI_DSWIGLU ? (p.dg_part ? 256 : 128) : 64);
  for (int tile_n = wide.tile_n / 2; tile_n >= narrowest; tile_n /= 2)
    for (int pair = 1; pair >= 0; --pair) {
      if (pair && (!pair_open || (cat ? 2 * tile_n : tile_n) < 128)) continue;
      const int64_t clk = clocks(pair != 0, tile_n);
      if (clk < best_clk) { best_clk = clk; best.pair = pair != 0; best.tile_n = tile_n; }
    }
  return best;
}

// Partial sums of <dH, H> per row that a SwiGLU backward product writes: one per epilogue warp that holds columns of it.
inline int tc_dg_parts(const GemmProblem& p, bool tr) { return tr ? p.N / 32 : 2 * (int)ceil_div(p.N, 256); }
inline int tc_dg_parts(const GemmProblem& p) { return tc_dg_parts(p, tc_plan(p, tc_state().n_sms).tr); }

inline int launch_gemm_tc(const GemmProblem& p, cudaStream_t st) {
  TcState& s = tc_state();
  if (!s.ready) return REVFFN_ERR_CUDA;
  if (p.epilogue > EPI_HEADS) return REVFFN_ERR_UNSUPPORTED;      // the update forms are chosen below
  if (p.M <= 0 || p.N <= 0) return REVFFN_OK;
  const int mma_n = 256;
  TcParams P;
  P.p = p;
  const TcPlan plan = tc_plan(p, s.n_sms);
  const bool tr = plan.tr, pair = plan.pair;
  CUtensorMap m_gu;
  if (tr && p.concat == CONCAT_N && tc_make_map_rows16(&m_gu, p) != REVFFN_OK) {      // the driver does not take the view
    GemmProblem q = p;
    q.tok_chunks = nullptr;
    return launch_gemm_tc(q, st);
  }
  if (p.dg_part && p.dg_ld < tc_dg_parts(p, tr)) return REVFFN_ERR_SHAPE;
  P.tile_n = plan.tile_n;
  // what one load of B brings: this CTA's share of a tile's columns, at most 128 of them
  P.b_box = std::min(128, pair && p.concat != CONCAT_N ? P.tile_n / 2 : P.tile_n);
  P.tiles_m = (int)ceil_div(p.M, TC_BM);
  P.tiles_n = (int)ceil_div(p.N, P.tile_n);
  const bool f8 = p.fp8 != 0;
  P.bk = f8 ? 2 * TC_BK : TC_BK;
  P.k_blocks = (int)ceil_div(p.K, P.bk);
  if (f8) {
    // e4m3 operands: K-major on both sides, the SwiGLU pair (transposed, or one CTA per row tile where that leaves SMs
    // idle) or the transposed store
    if (p.a_mn_major || p.b_mn_major || p.concat == CONCAT_K || !p.a_scale || !p.b_scale0 ||
        (p.concat == CONCAT_N && !p.b_scale1) || p.lda % 16 != 0 || p.ldb % 16 != 0 || p.K % 16 != 0)
      return REVFFN_ERR_UNSUPPORTED;
    if (!((p.epilogue == EPI_SWIGLU && p.group_mode == GROUP_M && !p.C1) ||
          (p.epilogue == EPI_STORE && !p.out_f32 && p.group_mode == GROUP_M && p.tok_chunks)))
      return REVFFN_ERR_UNSUPPORTED;
  }
  P.wait_cycles = p.dbg_wait_cycles > 0 ? p.dbg_wait_cycles : TC_WAIT_CYCLES;
  P.starve = p.dbg_starve;
  // Two load threads in every mode: measured against one thread in the same process, alternating, the whole step
  // is 4-5 % faster and no product is slower (the one-thread form stays selectable for such measurements).
  P.split_loads = p.dbg_split_loads != 2;
  if (p.dbg_starve && !p.no_pair) return REVFFN_ERR_UNSUPPORTED;      // the starved-wait test runs one CTA per tile
  if (p.N % 128 != 0 || (p.hm_split && p.epilogue != EPI_HEADS)) return REVFFN_ERR_SHAPE;
  // K need not be a multiple of the 64-wide K step: the tensor maps end at K, so the rest of the last
  // step is loaded as zeros (K-major rows must still start on 16-byte boundaries: lda, ldb)
  if (p.concat == CONCAT_K && (P.k_blocks & 1)) return REVFFN_ERR_SHAPE;
  // fp32 accumulator; operand formats bf16 (1) for kind::f16, e4m3 (0) for kind::f8f6f4
  const uint32_t fmt = f8 ? 0u : ((1u << 7) | (1u << 10));
  P.idesc = (1u << 4) | fmt | ((uint32_t)(p.a_mn_major ? 1 : 0) << 15) |
            ((uint32_t)(p.b_mn_major ? 1 : 0) << 16) | ((uint32_t)(mma_n >> 3) << 17) | ((uint32_t)(TC_BM >> 4) << 24);

  // 3-D views of the MN-major operands need whole 64-column groups everywhere
  P.mn3d = !p.dbg_mn_boxes && (!p.a_mn_major || (p.lda % 64 == 0 && p.a_col0 % 64 == 0)) && (!p.b_mn_major || (p.ldb % 64 == 0 && p.b_col0 % 64 == 0));
  const int groups = p.n_groups > 0 ? p.n_groups : 1;
  CUtensorMap ma, mb0, mb1;
  const int k_half = (p.concat == CONCAT_K) ? p.K / 2 : p.K;
  auto operand_maps = [&](bool mn3d) -> int {
    // A
    if (!p.a_mn_major) {
      // [rows, K]: dense M rows, or the padded row space for GROUP_M
      int r = tc_make_map(&ma, p.A, (uint64_t)p.K, (uint64_t)p.M, (uint64_t)p.lda, f8 ? 128 : 64, 128, f8);
      if (r) return r;
    } else {
      // [K rows, lda columns]; K rows = tokens (dense) or the bound on padded rows (GROUP_K)
      int r = mn3d ? tc_make_map_mn3d(&ma, p.A, (uint64_t)p.K, (uint64_t)p.lda)
                   : tc_make_map(&ma, p.A, (uint64_t)p.lda, (uint64_t)p.K, (uint64_t)p.lda, 64, 64);
      if (r) return r;
    }
    // B
    if (!p.b_mn_major) {
      const uint64_t rows = (p.group_mode == GROUP_M) ? (uint64_t)groups * p.N : (uint64_t)p.N;
      int r = tc_make_map(&mb0, p.B0, (uint64_t)k_half, p.hm_split ? p.hm_split : rows, (uint64_t)p.ldb, f8 ? 128 : 64, tr ? 128 : P.b_box, f8);
      if (r) return r;
      r = tc_make_map(&mb1, p.B1 ? p.B1 : p.B0, (uint64_t)k_half, rows - p.hm_split, (uint64_t)p.ldb, f8 ? 128 : 64, tr ? 128 : P.b_box, f8);
      if (r) return r;
    } else {
      uint64_t rows = (p.group_mode == GROUP_M) ? (uint64_t)groups * k_half : (uint64_t)p.K;
      int r = mn3d ? tc_make_map_mn3d(&mb0, p.B0, rows, (uint64_t)p.ldb, tr ? 128 : P.b_box)
                   : tc_make_map(&mb0, p.B0, (uint64_t)p.ldb, rows, (uint64_t)p.ldb, 64, 64);
      if (r) return r;
      r = mn3d ? tc_make_map_mn3d(&mb1, p.B1 ? p.B1 : p.B0, rows, (uint64_t)p.ldb, tr ? 128 : P.b_box)
               : tc_make_map(&mb1, p.B1 ? p.B1 : p.B0, (uint64_t)p.ldb, rows, (uint64_t)p.ldb, 64, 64);
      if (r) return r;
    }
    return REVFFN_OK;
  };
  // should the driver not take the 3-D view (its column-group stride is smaller than its row stride), the 64 x 64
  // boxes of the plain 2-D maps do the same work with twice the loads
  if (P.mn3d && operand_maps(true) != REVFFN_OK) P.mn3d = 0;
  if (!P.mn3d) {
    int r = operand_maps(false);
    if (r) return r;
  }
  // epilogue outputs written through TMA stores
  CUtensorMap mc, mc1;
  memset(&mc, 0, sizeof(mc));
  memset(&mc1, 0, sizeof(mc1));
  if (p.epilogue == EPI_HEADS) {
    // plain stores into the head-major tensor, no output map
    if (p.group_mode != 0 || p.N % 128 != 0 || p.hm_S <= 0 || p.hm_Sp < p.hm_S || (reinterpret_cast<uintptr_t>(p.C) & 15u))
      return REVFFN_ERR_SHAPE;
    if (p.hm_split && (p.hm_split < 0 || p.hm_split >= p.N || p.hm_split % 256 != 0 || p.b_mn_major || p.concat != CONCAT_NONE || !p.B1 ||
                       !p.C1 || (reinterpret_cast<uintptr_t>(p.C1) & 15u)))
      return REVFFN_ERR_SHAPE;
  } else if (p.epilogue == EPI_DSWIGLU) {
    // a|b are read and rewritten in place with plain 16-byte accesses, no tensor map
    if ((reinterpret_cast<uintptr_t>(p.ab) & 15u) || (p.ld_ab * 2) % 16 != 0) return REVFFN_ERR_ALIGN;
    if (p.C1) return REVFFN_ERR_UNSUPPORTED;
  } else {
    const bool f32_out = p.epilogue == EPI_COUPLE || p.epilogue == EPI_WGRAD || (p.epilogue == EPI_STORE && p.out_f32);
    uint64_t rows = (uint64_t)p.M;
    if (p.group_mode == GROUP_K) {
      // group g's block must start g * M rows further down one 2D tensor (g * split_m rows with two outputs)
      const int64_t m_out = p.split_m > 0 ? p.split_m : p.M;
      // (a product split over K whose rows are rows of A may end inside a tile)
      if ((p.M % TC_BM != 0 && (p.a_mn_major || p.upd_w)) || p.c_group_stride != m_out * p.ldc) return REVFFN_ERR_SHAPE;
      rows = (uint64_t)groups * p.M;
    }
    if (p.split_m > 0 && (p.epilogue != EPI_WGRAD || p.M != 2 * p.split_m || p.split_m % TC_BM != 0)) return REVFFN_ERR_SHAPE;
    if (p.epilogue == EPI_WGRAD && p.upd_w) {
      // fused update: master copies and moments are read and rewritten 16 bytes at a time, and so are bf16 weights without a
      // master copy (the row-wise form asks for them by cp.async)
      const bool bare = !p.upd_m || (p.split_m > 0 && !p.upd_m2);
      if ((reinterpret_cast<uintptr_t>(p.upd_w) & 15u) || (reinterpret_cast<uintptr_t>(p.upd_w2) & 15u) ||
          (reinterpret_cast<uintptr_t>(p.upd_m) & 15u) || (reinterpret_cast<uintptr_t>(p.upd_m2) & 15u) ||
          (reinterpret_cast<uintptr_t>(p.upd_mom) & 15u) || (reinterpret_cast<uintptr_t>(p.upd_mom2) & 15u) ||
          (reinterpret_cast<uintptr_t>(p.upd_var) & 15u) || (reinterpret_cast<uintptr_t>(p.upd_var2) & 15u) ||
          p.ldc % (bare ? 8 : 4) != 0)
        return REVFFN_ERR_ALIGN;
      if (p.split_m > 0 && !p.upd_w2) return REVFFN_ERR_NULL;
      if (p.upd.kind == 1 && (!p.upd_mom || !p.upd_var || (p.split_m > 0 && (!p.upd_mom2 || !p.upd_var2)))) return REVFFN_ERR_NULL;
    } else {
      if (!p.C || (p.split_m > 0 && !p.C2)) return REVFFN_ERR_NULL;
      if ((reinterpret_cast<uintptr_t>(p.C) & 15u) || (reinterpret_cast<uintptr_t>(p.C2) & 15u) || (p.ldc * (f32_out ? 4 : 2)) % 16 != 0)
        return REVFFN_ERR_ALIGN;
    }
    if (!f32_out) {      // fp32 outputs leave through plain stores and need no map
      int r = tc_make_out_map(&mc, p.C, false, (uint64_t)p.N, rows, (uint64_t)p.ldc);
      if (r) return r;
    }
    int r = 0;
    if (p.epilogue == EPI_SWIGLU && p.C1) {
      if ((reinterpret_cast<uintptr_t>(p.C1) & 15u) || (p.ldc1 * 2) % 16 != 0) return REVFFN_ERR_ALIGN;
      r = tc_make_out_map(&mc1, p.C1, false, (uint64_t)2 * p.N, (uint64_t)p.M, (uint64_t)p.ldc1);
      if (r) return r;
    }
  }
  if (tr) {
    const int r = tc_make_map(&mc1, p.A, (uint64_t)p.K, (uint64_t)p.M, (uint64_t)p.lda, f8 ? 128 : 64, 32, f8);
    if (r) return r;
  }
  if (f8 && p.epilogue == EPI_STORE && !tr) return REVFFN_ERR_UNSUPPORTED;      // only the transposed store scales its accumulator
  P.tr = tr ? 1 : 0;
  P.tiles_f = (int)ceil_div(p.N, p.concat == CONCAT_N ? 128 : 256);
  P.tr_swap = tr && p.concat == CONCAT_N && reinterpret_cast<uintptr_t>(p.B1) < reinterpret_cast<uintptr_t>(p.B0);
  if (tr && p.concat == CONCAT_N) mb0 = m_gu;
  // a CTA or a CTA pair per tile
  int64_t total = (int64_t)P.tiles_m * P.tiles_n * (p.group_mode == GROUP_K ? groups : 1);
  if (tr) {
    // the number of token chunks is only known on the device: runs of 256 of each expert's rows, which are padded to 128
    total = (p.M + 128 * (int64_t)groups) / 256 * P.tiles_f;
    P.idesc = (1u << 4) | fmt | ((uint32_t)(p.b_mn_major ? 1 : 0) << 15) |
              ((uint32_t)(p.a_mn_major ? 1 : 0) << 16) | ((uint32_t)(256 >> 3) << 17) | ((uint32_t)(2 * TC_BM >> 4) << 24);
  } else if (pair) {
    total = (int64_t)((P.tiles_m + 1) / 2) * P.tiles_n * (p.group_mode == GROUP_K ? groups : 1);
    P.idesc = (P.idesc & ~(0x1Fu << 24)) | ((uint32_t)(2 * TC_BM >> 4) << 24);   // M = 256 across the pair
  }
  if (total <= 0) return REVFFN_OK;
  if (total > (1 << 30)) return REVFFN_ERR_SHAPE;
  const int grid = (int)(pair ? 2 * total : total);

#define TC_CASE(N_, E_) \
  if (mma_n == N_ && epi == E_) return tc_launch<N_, E_>(P, ma, mb0, mb1, mc, mc1, grid, pair, st);
  // A fused update of a grouped product runs in its own form while the K range of a group is short (rows of K on average): that form
  // writes whole rows but has two stages (Adam) or three (SGD) where the other has six, so beyond some length the operand ring is worth
  // more than the reads and writes.  The experts' two updates together, medians of three in turn, us, own form | the other:
  // Adam at 1764 rows 3328 | 3838, 2037 3841 | 4048, 2105 3974 | 4169, 2173 4003 | 3992, 2310 4282 | 3933, 2446 4524 | 4222;
  // SGD at 1081 1050 | 1318, 1218 1142 | 1301, 1354 1261 | 1301, 1491 1430 | 1353, 1627 1551 | 1381.
  const int64_t k_group = p.K / groups;
  const int epi = p.epilogue != EPI_WGRAD ? p.epilogue
                  : p.upd_w && p.group_off && k_group <= (p.upd.kind ? 2176 : 1408) ? (p.upd.kind ? EPI_WADAM : EPI_WSGD)
                  : p.upd_w || p.accumulate ? EPI_WRMW : EPI_WGRAD;
  TC_CASE(256, EPI_STORE) TC_CASE(256, EPI_SWIGLU) TC_CASE(256, EPI_ROWSCALE) TC_CASE(256, EPI_COUPLE)
  TC_CASE(256, EPI_DSWIGLU) TC_CASE(256, EPI_WGRAD) TC_CASE(256, EPI_WADAM) TC_CASE(256, EPI_WSGD) TC_CASE(256, EPI_WRMW)
  TC_CASE(256, EPI_HEADS)
#undef TC_CASE
  return REVFFN_ERR_UNSUPPORTED;
}

}  // namespace revffn
