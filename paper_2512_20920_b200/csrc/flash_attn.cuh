// Causal attention core on tcgen05 / TMEM / TMA (Attn_pt of Eq. 1 between the projections):
//   O = softmax(scale * Q K^T, keys <= query position) V   per (sequence, head),
// without materialising the score matrix.
//
// Forward: one CTA per (sequence, head, 256 query positions = two tiles of 128); it walks the key/value blocks
// 0 .. the second tile's diagonal block.  320 threads:
//   warp 0      TMA producer: the Q tiles once, then K and V blocks into two-stage rings, each used by both tiles
//   warp 1      MMA issuer and TMEM owner.  TMEM (512 columns): a score and an output accumulator of 128 fp32
//               columns for each tile.  Per block and tile: O += P_j V_j, then S_{j+1} = Q K_{j+1}^T over the scores that
//               P_j came from.  While one tile's softmax runs, the tensor pipe works for the other.
//   warps 2..9  softmax: four warps per tile, one thread per query row (= TMEM lane), all 128 scores of a block in
//               registers: p = exp2((s - m) * scale * log2 e), P as bf16 pairs over the first 64 columns of the score
//               accumulator, from where the second product takes it as its A operand.  O stays in tensor memory.
//               The row's reference m is its maximum in the first block.  It is taken anew from a block's maxima, and
//               the warp's rows of O rescaled, only when the weights of the block's first 64 keys add up to more than
//               2^20 or one of the others passes 2^14 (p, P and the sums are floating point: no bit is lost below that).
//               O is divided by the sum of the weights as P holds them: relative to the first block's maximum a row's
//               largest weight is not a power of two, and its rounding to bf16 would scale the whole row by up to 2^-8.
//               (Against fp64, 4 x 2048 and 7 x 613: the branch's error is 0.2 % below that of the exact sum relative to a running maximum;
//               divided by the exact sum of these weights 0.05 % above, with scores of a standard deviation of 3 0.9 %.)
//               O is at rest then: S_j complete means P_{j-1} V_{j-1} complete, both come from one in-order queue, and
//               P_j V_j waits for this warp.  P goes out in halves of 64 keys, so that P V starts under the exponentials
//               of the second half.
// What bounds it: a pair of blocks takes about 3.5k clk, the chain of one tile (softmax 1.85k, products 1.2k, of which a
// quarter k lies under the softmax, barriers); the exponentials alone are 2.0k (two warps per scheduler on a unit of four a
// clock), the products 2.3k; a CTA starts and ends in 5-8k.  4 sequences of 2048 x 16 heads: 120 us with one query tile per
// CTA, the output in registers and maxima exchanged through shared memory; 97 with two tiles; 88 with products issued by a
// converged warp (the row maxima left out beside that: no difference); P in halves 92 -> 88 on another GPU.  The second sum
// costs nothing there (82 and 82 us); a gradient pass, which wants both sums, fetches the second half's scores twice instead of
// spilling registers (117 -> 103, 96 before it had them).  7 x 613: 38 -> 36 us when five query tiles made three pairs, now 30
// (39 for a gradient pass).
// Operands: q, k, v head-major [.., S_pad, hd] bf16 with hd = 128 (rows past the sequence are zero);
// output token-major [T, ld_o] bf16, plus the row log-sum-exp (natural log, of the scaled scores).
// Every wait is bounded; a wait that runs out sets the status word and all roles leave.
#pragma once

#include "gemm_tcgen05.cuh"

namespace revffn {

constexpr int FA_THREADS = 320;
constexpr int FA_BLK = 128;                       // query rows per CTA and keys per block
constexpr int FA_HD = 128;                        // head dimension
constexpr int FA_TILE = FA_BLK * 64 * 2;          // one 64-wide K block of an operand tile: 16 KB
constexpr int FA_Q_OFF = 0;                       // Q: two query tiles of 2 tiles each
constexpr int FA_K_OFF = 4 * FA_TILE;             // K: 2 stages x 2 tiles
constexpr int FA_V_OFF = FA_K_OFF + 4 * FA_TILE;  // V: 2 stages x 2 k-blocks (each 2 chunks of 8 KB)
constexpr int FA_BAR_OFF = FA_V_OFF + 4 * FA_TILE;
constexpr int FA_SMEM_BYTES = FA_BAR_OFF + 256 + 1024;      // + alignment slack
constexpr float FA_SUM_MAX = 1048576.f;           // sum of a row's weights of 64 keys above which the row's reference follows
constexpr float FA_LOG2_MAX = 14.f;               // log2 of a single weight above which it does

__device__ __forceinline__ float fa_exp2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// p = exp2(s * cl - mc) for 64 scores of this thread's row, packed to bf16.  Returns the sum of the packed values (.y) and,
// with SUM, of the weights themselves (.x).
template <bool SUM>
__device__ __forceinline__ float2 fa_probs64(const uint32_t (&r0)[32], const uint32_t (&r1)[32], float cl, float mc, uint32_t (&pw)[32]) {
  float2 sum = make_float2(0.f, 0.f), rounded = make_float2(0.f, 0.f);
  const float2 c2 = make_float2(cl, cl), m2 = make_float2(-mc, -mc);
#pragma unroll
  for (int i = 0; i < 32; ++i) {
    const uint32_t* r = i < 16 ? &r0[2 * i] : &r1[2 * i - 32];
    const float2 t = __ffma2_rn(make_float2(__uint_as_float(r[0]), __uint_as_float(r[1])), c2, m2);
    const float2 e = make_float2(fa_exp2(t.x), fa_exp2(t.y));
    if (SUM) sum = __fadd2_rn(sum, e);
    const __nv_bfloat162 h = __floats2bfloat162_rn(e.x, e.y);
    pw[i] = *reinterpret_cast<const uint32_t*>(&h);
    // two additions of bf16 to fp32; unpacked and added in pairs it is three instructions (core at 4 x 2048: 86 us instead of 82)
    asm("{\n\t.reg .b16 lo, hi;\n\tmov.b32 {lo, hi}, %2;\n\tadd.rn.f32.bf16 %0, lo, %0;\n\tadd.rn.f32.bf16 %1, hi, %1;\n\t}"
        : "+f"(rounded.x), "+f"(rounded.y) : "r"(pw[i]));
  }
  return make_float2(sum.x + sum.y, rounded.x + rounded.y);
}

// 32 consecutive 32-bit columns of this thread's TMEM lane, written from registers.
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
      "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
        "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]),
        "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]),
        "r"(r[30]), "r"(r[31]) : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// D += A B with A in tensor memory (rows = lanes, two 16-bit K elements per 32-bit column), B from shared memory.
__device__ __forceinline__ void tc_mma_ta(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(acc) : "memory");
}

struct FlashParams {
  int S, Sp, n_heads, rep;        // rep = query heads per key/value head
  bf16* o; int64_t ld_o;          // [T, ld_o]
  const bf16* d_o;                // GRAD: gradient of the output, head-major [B * n_heads * Sp, 128]
  float* lse_d;                   // GRAD: statistics of the rows for the gradient kernels, see FlashBwdParams
  float scale_log2e, scale;
  int* status;
};

// GRAD: for a gradient pass, which also wants of each row the log-sum-exp and D = <dO, O>.  O is taken before its rounding to
// bf16: D stands for sum_j P_j dP_j, and with a peaked row dP - D cancels, so an error in D would show in dS.
template <bool GRAD>
__global__ void __launch_bounds__(FA_THREADS, 1)
flash_fwd_kernel(const FlashParams P, const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                 const __grid_constant__ CUtensorMap map_v) {
  extern __shared__ uint8_t fa_smem_raw[];
  const uint32_t raw = smem_u32(fa_smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* gen_base = fa_smem_raw + (base - raw);
  const uint32_t bars = base + FA_BAR_OFF;
  // barrier slots (8 bytes each)
  auto bar = [&](int i) -> uint32_t { return bars + 8u * (uint32_t)i; };
  enum { B_QFULL = 0, B_KFULL = 1, B_KEMPTY = 3, B_VFULL = 5, B_VEMPTY = 7, B_SFULL = 9, B_PFULL = 11, B_OFULL = 13, B_DRAIN = 15,
         B_PHALF = 16, B_COUNT = 18 };
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(gen_base + FA_BAR_OFF + 8 * B_COUNT);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(gen_base + FA_BAR_OFF + 8 * B_COUNT + 8);
  int* issued = reinterpret_cast<int*>(gen_base + FA_BAR_OFF + 8 * B_COUNT + 16);   // [5]: q, k0, k1, v0, v1 -> phase + 1

  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  const int n_qblk = P.Sp / FA_BLK, n_pair = (n_qblk + 1) / 2;
  // heavy work first: the last query tiles of every (sequence, head) have the most key blocks
  const int bh_count = (int)gridDim.x / n_pair;
  const int qp = n_pair - 1 - (int)blockIdx.x / bh_count;
  const int bh = (int)blockIdx.x % bh_count;           // sequence * n_heads + head
  const bool two = 2 * qp + 1 < n_qblk;                // the last pair of an odd number of tiles has one
  const int n_blk = 2 * qp + (two ? 2 : 1);            // key blocks of the CTA; tile x needs 2 qp + x + 1 of them
  const int q_row0 = bh * P.Sp + 2 * qp * FA_BLK;
  const int kv_row0 = (bh / P.rep) * P.Sp;             // (sequence * n_kv_heads + head / rep) * S_pad

  if (threadIdx.x == 0) {
    mbar_init(bar(B_QFULL), 1);
    for (int s = 0; s < 2; ++s) {
      mbar_init(bar(B_KFULL + s), 1); mbar_init(bar(B_KEMPTY + s), 1);
      mbar_init(bar(B_VFULL + s), 1); mbar_init(bar(B_VEMPTY + s), 1);
      mbar_init(bar(B_SFULL + s), 1); mbar_init(bar(B_PHALF + s), 4); mbar_init(bar(B_PFULL + s), 4);
      mbar_init(bar(B_OFULL + s), 1);
    }
    mbar_init(bar(B_DRAIN), 1);
    for (int i = 0; i < 5; ++i) issued[i] = 0;
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(smem_u32(tmem_slot)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  pdl_wait();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // TMEM columns: scores of tile x at 128 x, output of tile x at 256 + 128 x
  // instruction descriptors: fp32 accumulate, bf16 operands, M = 128, N = 128; V is stored [key, hd] (N contiguous)
  const uint32_t idesc_qk = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(FA_BLK >> 3) << 17) | ((uint32_t)(FA_BLK >> 4) << 24);
  const uint32_t idesc_pv = idesc_qk | (1u << 16);

  if (warp == 0) {
    // ------------------------------------------------------------------ producer
    if (lane == 0) {
      const int nq = two ? 4 : 2;
      mbar_expect_tx(bar(B_QFULL), nq * FA_TILE);
      issued[0] = 1;
      for (int i = 0; i < nq; ++i)
        tma_load_2d(base + FA_Q_OFF + i * FA_TILE, &map_q, 64 * (i & 1), q_row0 + (i >> 1) * FA_BLK, bar(B_QFULL));
      for (int j = 0; j < n_blk; ++j) {
        const int s = j & 1;
        const uint32_t ph = (uint32_t)(j >> 1) & 1u;
        if (!mbar_wait(bar(B_KEMPTY + s), ph ^ 1u, abort_flag, P.status)) break;
        mbar_expect_tx(bar(B_KFULL + s), 2 * FA_TILE);
        issued[1 + s] = (int)ph + 1;
        for (int kb = 0; kb < 2; ++kb)
          tma_load_2d(base + FA_K_OFF + (2 * s + kb) * FA_TILE, &map_k, 64 * kb, kv_row0 + j * FA_BLK, bar(B_KFULL + s));
        if (!mbar_wait(bar(B_VEMPTY + s), ph ^ 1u, abort_flag, P.status)) break;
        mbar_expect_tx(bar(B_VFULL + s), 2 * FA_TILE);
        issued[3 + s] = (int)ph + 1;
        for (int kb = 0; kb < 2; ++kb)        // 64 keys per k-block, two 64-column chunks of hd each
          for (int nj = 0; nj < 2; ++nj)
            tma_load_2d(base + FA_V_OFF + (2 * s + kb) * FA_TILE + nj * 8192, &map_v, 64 * nj,
                        kv_row0 + j * FA_BLK + 64 * kb, bar(B_VFULL + s));
      }
      pdl_trigger();
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    const uint32_t tb = __shfl_sync(0xffffffffu, tmem_base, 0), sb = __shfl_sync(0xffffffffu, base, 0);
    auto wait = [&](int i, uint32_t parity) -> bool {
      const bool got = mbar_wait_warp(bar(i), parity, abort_flag, P.status);
      tc_fence_after();
      return got;
    };
    // S_j of tile x; the block's K has been waited for
    auto issue_qk = [&](int j, int x) {
      const uint64_t a_desc = make_smem_desc(sb + FA_Q_OFF + 2 * x * FA_TILE, 16, 1024);
      const uint64_t b_desc = make_smem_desc(sb + FA_K_OFF + 2 * (j & 1) * FA_TILE, 16, 1024);
      if (elect_one()) {
#pragma unroll
        for (int k = 0; k < 8; ++k)       // two 16 KB tiles of 64 columns, 16 columns an instruction
          tc_mma(tb + (uint32_t)(128 * x), a_desc + (uint64_t)((k >> 2) * (FA_TILE >> 4) + 2 * (k & 3)),
                 b_desc + (uint64_t)((k >> 2) * (FA_TILE >> 4) + 2 * (k & 3)), idesc_qk, k != 0 ? 1u : 0u);
        tc_commit(bar(B_SFULL + x));
      }
      __syncwarp();
    };
    auto commit = [&](int i) {
      if (elect_one()) tc_commit(bar(i));
      __syncwarp();
    };
    bool ok = wait(B_QFULL, 0u);
    if (ok) ok = wait(B_KFULL, 0u);
    if (ok) {
      issue_qk(0, 0);
      if (two) issue_qk(0, 1);
      commit(B_KEMPTY);
    }
    for (int j = 0; ok && j < n_blk; ++j) {
      const int b = j & 1;
      const uint32_t ph = (uint32_t)(j >> 1) & 1u;
      const bool more = j + 1 < n_blk;
      if (!(ok = wait(B_VFULL + b, ph))) break;                                    // V_j and K_{j+1}, once for both tiles
      if (more && !(ok = wait(B_KFULL + (b ^ 1), (uint32_t)((j + 1) >> 1) & 1u))) break;
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        const int n_x = (x == 0 || two) ? 2 * qp + x + 1 : 0;
        if (j < n_x && ok) {
          const uint64_t b_desc = make_smem_desc(sb + FA_V_OFF + 2 * b * FA_TILE, 8192, 1024);
#pragma unroll
          for (int h = 0; h < 2; ++h) {         // 64 keys each, as P_j's columns become readable
            if (ok) ok = wait((h ? B_PFULL : B_PHALF) + x, (uint32_t)j & 1u);
            if (ok && elect_one()) {
#pragma unroll
              for (int k = 4 * h; k < 4 * h + 4; ++k)
                tc_mma_ta(tb + (uint32_t)(256 + 128 * x), tb + (uint32_t)(128 * x + 8 * k),
                          b_desc + (uint64_t)((k >> 2) * (FA_TILE >> 4) + 128 * (k & 3)), idesc_pv, (j | k) != 0 ? 1u : 0u);
              if (h == 1 && j + 1 == n_x) tc_commit(bar(B_OFULL + x));
            }
            __syncwarp();
          }
          if (ok && j + 1 < n_x) issue_qk(j + 1, x);
        }
      }
      if (!ok) break;
      commit(B_VEMPTY + b);
      if (more) commit(B_KEMPTY + (b ^ 1));
    }
    if (!ok) {
      // an abandoned wait: products issued so far must have finished before the teardown frees what they use
      commit(B_DRAIN);
      const long long t0 = clock64();
      while (!mbar_try_wait(bar(B_DRAIN), 0u) && clock64() - t0 < TC_WAIT_CYCLES) {}
    }
    __syncwarp();
  } else {
    // ------------------------------------------------------------------ softmax (warps 2..9)
    const int q = warp & 3;                      // TMEM lane quadrant this warp may access
    const int x = (warp - 2) >> 2;               // query tile
    const int row = q * 32 + lane;               // query row within the tile
    const uint32_t lane_addr = tmem_base + ((uint32_t)(q * 32) << 16);
    const uint32_t s_addr = lane_addr + (uint32_t)(128 * x), o_addr = lane_addr + (uint32_t)(256 + 128 * x);
    const int n_x = (x == 0 || two) ? 2 * qp + x + 1 : 0;
    // l.x: sum of the weights, for the row's log-sum-exp.  l.y: of the rounded weights that P V uses, which O is divided
    // by: a weight that outweighs all others then cancels whatever its rounding (it is exact only when the reference is
    // its own score), and the others' errors act on their values' distance from the mean.
    float m = -INFINITY;
    float2 l = make_float2(0.f, 0.f);
    const float cl = P.scale_log2e;
    bool ok = true;
    for (int j = 0; j < n_x; ++j) {
      ok = mbar_wait_warp(bar(B_SFULL + x), (uint32_t)j & 1u, abort_flag, P.status);
      if (!ok) break;
      tc_fence_after();
      uint32_t pw[32], r2[32], r3[32];
      float2 s0;
      bool ref = j == 0;        // take the reference from this block's maxima
      auto load64 = [&](int c, uint32_t (&a)[32], uint32_t (&b)[32]) {
        tmem_ld32(s_addr + c, a);
        tmem_ld32(s_addr + c + 32, b);
        tmem_ld_wait();
        if (j + 1 < n_x) return;
        // the diagonal block: keys past the query position
#pragma unroll
        for (int i = 0; i < 32; ++i) {
          if (c + i > row) a[i] = 0xff800000u;
          if (c + 32 + i > row) b[i] = 0xff800000u;
        }
      };
      while (true) {
        uint32_t r0[32], r1[32];
        load64(64, r2, r3);
        float b0 = __uint_as_float(r2[0]), b1 = __uint_as_float(r3[0]);
#pragma unroll
        for (int i = 1; i < 32; ++i) { b0 = fmaxf(b0, __uint_as_float(r2[i])); b1 = fmaxf(b1, __uint_as_float(r3[i])); }
        float b = fmaxf(b0, b1);
        if (GRAD) asm volatile("" : "+f"(b));      // the second half's registers are free from here: it is fetched again below
        load64(0, r0, r1);
        if (ref) {
          float a0 = m, a1 = b;
#pragma unroll
          for (int i = 0; i < 32; ++i) { a0 = fmaxf(a0, __uint_as_float(r0[i])); a1 = fmaxf(a1, __uint_as_float(r1[i])); }
          const float m_new = fmaxf(a0, a1);
          if (j > 0) {
            const float alpha = fa_exp2((m - m_new) * cl);
            if (GRAD) l.x *= alpha;
            l.y *= alpha;
#pragma unroll 1
            for (int c = 0; c < 128; c += 32) {
              uint32_t o[32];
              tmem_ld32(o_addr + c, o);
              tmem_ld_wait();
#pragma unroll
              for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * alpha);
              tmem_st32(o_addr + c, o);
            }
          }
          m = m_new;
        }
        // the first half's weights; of the second half only that they will not be too large (the maximum hides under the
        // exponentials), so that the product may start on the first
        s0 = fa_probs64<GRAD>(r0, r1, cl, m * cl, pw);
        if (ref) break;
        const bool fits = s0.y <= FA_SUM_MAX && (b - m) * cl <= FA_LOG2_MAX;
        if (!__any_sync(0xffffffffu, !fits)) break;
        ref = true;
      }
      tmem_st32(s_addr, pw);
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(B_PHALF + x));
      if (GRAD) load64(64, r2, r3);
      const float2 s1 = fa_probs64<GRAD>(r2, r3, cl, m * cl, pw);
      tmem_st32(s_addr + 32, pw);
      if (GRAD) l.x += s0.x + s1.x;
      l.y += s0.y + s1.y;
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(B_PFULL + x));
    }
    if (n_x > 0 && ok) ok = mbar_wait_warp(bar(B_OFULL + x), 0u, abort_flag, P.status);
    if (n_x > 0 && ok) {
      tc_fence_after();
      // out through this tile's Q area (its products are complete), 64- and 128-byte row pieces per instruction
      const int s_pos0 = (2 * qp + x) * FA_BLK + q * 32, s_pos = s_pos0 + lane;
      const int rows_ok = min(32, P.S - s_pos0);
      const float inv = 1.f / l.y;
      float2 dot = make_float2(0.f, 0.f);      // GRAD: <dO, O> of even and odd columns
      const int seq = bh / P.n_heads, head = bh % P.n_heads;
      uint8_t* stg = gen_base + FA_Q_OFF + x * 2 * FA_TILE + q * 8192;
      bf16* dst = P.o + ((int64_t)seq * P.S + s_pos0) * P.ld_o + (int64_t)head * FA_HD;
#pragma unroll 1
      for (int c = 0; c < 128; c += 32) {
        uint32_t o[32];
        float f[32];
        tmem_ld32(o_addr + c, o);
        tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < 32; ++i) f[i] = __uint_as_float(o[i]) * inv;
        stage32_bf16(stg, lane, f);
        if (GRAD && lane < rows_ok) {
          const uint4* g4 = reinterpret_cast<const uint4*>(P.d_o + ((int64_t)bh * P.Sp + s_pos) * FA_HD + c);
#pragma unroll
          for (int g = 0; g < 4; ++g) {
            float y[8];
            unpack8(g4[g], y);
#pragma unroll
            for (int i = 0; i < 8; i += 2)
              dot = __ffma2_rn(make_float2(f[8 * g + i], f[8 * g + i + 1]), make_float2(y[i], y[i + 1]), dot);
          }
        }
        __syncwarp();
        blk_stage_to_global(stg, lane, dst + c, P.ld_o, rows_ok);
        __syncwarp();
      }
      if (GRAD) {      // rows past the end of the sequence: weights of zero
        const int64_t at = (int64_t)bh * P.Sp + s_pos;
        float* ld = P.lse_d + 4 * (at >> 1) + (at & 1);
        ld[0] = lane < rows_ok ? -(m * P.scale + logf(l.x)) * 1.4426950408889634f : -INFINITY;
        ld[2] = lane < rows_ok ? -(dot.x + dot.y) * P.scale : 0.f;
      }
    }
  }

  // ------------------------------------------------------------------ teardown
  tc_fence_before();
  __syncthreads();
  if (*abort_flag && threadIdx.x == 0) {
    // loads already issued into this CTA's shared memory must land before the CTA exits
    const int bidx[5] = {B_QFULL, B_KFULL, B_KFULL + 1, B_VFULL, B_VFULL + 1};
    for (int i = 0; i < 5; ++i) {
      if (issued[i] == 0) continue;
      long long t0 = clock64();
      while (!mbar_try_wait(bar(bidx[i]), (uint32_t)(issued[i] - 1)) && clock64() - t0 < TC_WAIT_CYCLES) {}
    }
  }
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
  }
}

// q: [B * n_heads * Sp, 128], k, v: [B * n_kv_heads * Sp, 128] bf16 head-major; o: [B * S, ld_o] bf16.  lse_d is written when
// d_o is given.
inline int launch_flash_fwd(const bf16* q, const bf16* k, const bf16* v, int batch, int n_heads, int n_kv_heads, int S, int Sp,
                            bf16* o, int64_t ld_o, const bf16* d_o, float* lse_d, int* status, cudaStream_t st) {
  TcState& s = tc_state();
  if (!s.ready) return REVFFN_ERR_CUDA;
  if (batch <= 0) return REVFFN_OK;
  static bool attr_set[64] = {false};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return REVFFN_ERR_CUDA;
  if (!attr_set[dev]) {
    if (cudaFuncSetAttribute(flash_fwd_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, FA_SMEM_BYTES) != cudaSuccess ||
        cudaFuncSetAttribute(flash_fwd_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, FA_SMEM_BYTES) != cudaSuccess)
      return REVFFN_ERR_CUDA;
    attr_set[dev] = true;
  }
  CUtensorMap mq, mk, mv;
  int r = tc_make_map(&mq, q, FA_HD, (uint64_t)batch * n_heads * Sp, FA_HD, 64, 128);
  if (r) return r;
  r = tc_make_map(&mk, k, FA_HD, (uint64_t)batch * n_kv_heads * Sp, FA_HD, 64, 128);
  if (r) return r;
  r = tc_make_map(&mv, v, FA_HD, (uint64_t)batch * n_kv_heads * Sp, FA_HD, 64, 64);
  if (r) return r;
  FlashParams P;
  P.S = S; P.Sp = Sp; P.n_heads = n_heads; P.rep = n_heads / n_kv_heads;
  P.o = o; P.ld_o = ld_o; P.d_o = d_o; P.lse_d = lse_d;
  P.scale = 1.f / sqrtf((float)FA_HD);
  P.scale_log2e = P.scale * 1.4426950408889634f;
  P.status = status;
  const int grid = batch * n_heads * ((Sp / FA_BLK + 1) / 2);
  launch_k(d_o ? flash_fwd_kernel<true> : flash_fwd_kernel<false>, grid, FA_THREADS, FA_SMEM_BYTES, st, P, mq, mk, mv);
  return cudaGetLastError() == cudaSuccess ? REVFFN_OK : REVFFN_ERR_CUDA;
}

// ---------------------------------------------------------------------------
// Backward of the attention core, also without a score matrix in HBM.  P is rebuilt from the row
// log-sum-exp the forward kernel stored:  P = exp(scale * S - lse),  dS = scale * P * (dP - D) with
// D = <dO_row, O_row>.  Two kernels, neither uses atomics:
//   flash_bwd_dkv_kernel  an item is 128 keys of one key/value head, which walk the 128-row query tiles at or
//                         below them (of every query head of the group):  dV += P^T dO,  dK += dS^T Q
//   flash_bwd_dq_kernel   an item is 128 query rows of one head, which walk the 128-key tiles up to their diagonal:
//                         dQ += dS K
// In both the item's own side is the MMA M side and the walked tile the N side of S' and dP'.  All four or three products
// of a step are 128 x 128 x 128.  Eight warps (two threads per own row, 64 columns each) turn S' into P' and dP' into dS'
// in two phases, so that the tensor pipe always has the other half of a step to work on; P' and dS' go back to tensor memory
// over the columns that they came from, from where the accumulating products take them as their A operand, and the walked
// tile's shared-memory bytes are read a second time as their MN-major B operand.  One in-order queue of products makes every
// "over the columns" safe: what overwrites a region is issued behind what reads it.
// Persistent blocks: items in descending order of their steps, dealt out to the blocks forwards and backwards in turn; the
// steps of all items of a block are one stream: the loads and the first products of the next item run under the end of this
// one, and four warps of their own write the output beside it.
// No cross-thread reduction is needed: the row statistics come from memory.
// What bounds them, per 128 x 128 block: dK/dV 2.7k clk in the middle of an item, the tensor pipe, whose S' and dP' read both
// operands out of shared memory (256 KB a step at 128 bytes a clock, arriving tiles included); dQ 2.2k, the softmax warps'
// exponentials (1.15k) and dS' (0.55k) and the products between them.  The first steps of an item take twice that, under the output
// of the item before.  4 sequences of 2048 x 16 heads: 64-wide query tiles, P' and dS' through shared memory and a block per item took
// 5.8k and 4.9k, 180 and 150 us; now 245 together, and 29 less without a launch for the row dots (7 x 613, 4 key/value heads: 121 -> 81).
// A quarter or a third of the exponentials by a polynomial on the FMA pipe: no difference.
// ---------------------------------------------------------------------------
struct FlashBwdParams {
  int S, Sp, n_heads, rep;
  const float4* lse_d;            // a pair of query rows (head-major index / 2): -lse * log2 e of both, then -D * scale of both
  const bf16* x0; const bf16* x1; // dQ kernel: its owned operands (q, d_o head-major), read by the CTA's threads themselves
  // Outputs, token-major bf16 [T, ld_out]: a row's head lands at column col + head * 128.  out0: dV (dK/dV kernel, as
  // it is); out1: dK or dQ, with the rotation of the forward pass undone (its transpose), pairs (i, i + 64).
  bf16* out0; bf16* out1;
  int64_t ld_out0, ld_out1;
  int col0, col1;
  int heads_own;                  // heads per sequence on the owned side (key/value heads for dK/dV, query heads for dQ)
  int items;
  const float2* cs;               // [64, S] (cos, sin): the lanes' positions are neighbours
  float scale_log2e, scale;
  int* status;
};

// Untiled bulk copy global -> shared (both addresses 16-byte aligned, size a multiple of 16), completing on an mbarrier.
__device__ __forceinline__ void bulk_load_1d(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
        "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]) : "memory");
}

// Item of a block's round r: forwards in even rounds, backwards in odd ones.
__device__ __forceinline__ int fb_item(int r) {
  return r * (int)gridDim.x + ((r & 1) ? (int)gridDim.x - 1 - (int)blockIdx.x : (int)blockIdx.x);
}

// The causal diagonal's tile: registers of columns whose query comes before their key.  edge: the thread's own position relative
// to the first of the 32 columns.  (DKV: own row = key, column = query; else the roles swap.)  A pass of its own over the registers
// and not a second form of the arithmetic, which would run once an item.
template <bool DKV>
__device__ __forceinline__ void fb_mask(uint32_t (&x)[32], int edge, uint32_t value) {
#pragma unroll
  for (int i = 0; i < 32; ++i)
    if (DKV ? i < edge : i > edge) x[i] = value;
}
// 32 scores of this thread's row -> weights p = exp2(s * cl - lse2) in their place, and packed to bf16.  The row statistics
// belong to the query: the column's (DKV, two columns to an entry of ld) or this thread's own row's; those past the end of
// the sequence have weights of zero.
template <bool DKV>
__device__ __forceinline__ void fb_probs(uint32_t (&s)[32], const float4* ld, float own_nl, float cl, uint32_t (&pw)[16]) {
  const float2 c2 = make_float2(cl, cl);
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    float2 nl = make_float2(own_nl, own_nl);
    if (DKV) nl = *reinterpret_cast<const float2*>(ld + i);
    const float2 t = __ffma2_rn(make_float2(__uint_as_float(s[2 * i]), __uint_as_float(s[2 * i + 1])), c2, nl);
    const float2 e = make_float2(fa_exp2(t.x), fa_exp2(t.y));
    s[2 * i] = __float_as_uint(e.x);
    s[2 * i + 1] = __float_as_uint(e.y);
    if (DKV) {
      const __nv_bfloat162 h = __floats2bfloat162_rn(e.x, e.y);
      pw[i] = *reinterpret_cast<const uint32_t*>(&h);
    }
  }
}
// dS' = P' * (dP * scale - D * scale) of 32 columns, packed to bf16.
template <bool DKV>
__device__ __forceinline__ void fb_dscores(const uint32_t (&p)[32], const uint32_t (&rd)[32], const float4* ld, float own_nd, float scale,
                                           uint32_t (&dw)[16]) {
  const float2 s2 = make_float2(scale, scale);
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    float2 nd = make_float2(own_nd, own_nd);
    if (DKV) nd = *(reinterpret_cast<const float2*>(ld + i) + 1);
    const float2 x = __ffma2_rn(make_float2(__uint_as_float(rd[2 * i]), __uint_as_float(rd[2 * i + 1])), s2, nd);
    const float2 d = __fmul2_rn(make_float2(__uint_as_float(p[2 * i]), __uint_as_float(p[2 * i + 1])), x);
    const __nv_bfloat162 h = __floats2bfloat162_rn(d.x, d.y);
    dw[i] = *reinterpret_cast<const uint32_t*>(&h);
  }
}

// Four neighbouring lanes hold four 16-byte pieces each: piece k of lane j changes place with piece j of lane k.  A warp whose
// lanes are rows then reads or writes rows of 64 contiguous bytes, eight per instruction; 16-byte pieces of 32 rows
// take an instruction four times as long, and everything else that goes through the same unit (the softmax warps'
// statistics) waits behind it (dK/dV at 4 x 2048, a step on average: 3.85k clk -> 3.64k).
__device__ __forceinline__ void quad_transpose(uint4 (&v)[4], int lane) {
  auto trade = [&](uint4& a, uint4& b, bool hi, int mask) {      // the low lane gives b for the high lane's a
    const uint4 s = hi ? a : b;
    uint4 r;
    r.x = __shfl_xor_sync(0xffffffffu, s.x, mask); r.y = __shfl_xor_sync(0xffffffffu, s.y, mask);
    r.z = __shfl_xor_sync(0xffffffffu, s.z, mask); r.w = __shfl_xor_sync(0xffffffffu, s.w, mask);
    if (hi) a = r; else b = r;
  };
  trade(v[0], v[1], lane & 1, 1); trade(v[2], v[3], lane & 1, 1);
  trade(v[0], v[2], lane & 2, 2); trade(v[1], v[3], lane & 2, 2);
}

// A warp's 32 rows x 128 columns of an accumulator to the token-major output, the rotation undone when cs is given
// (columns 0..31 turn with 64..95, 32..63 with 96..127; cs: at this lane's position).  dst: the warp's first row, rows: how
// many of its rows exist.  `drained` is called when the last columns are in registers.
template <typename Drained>
__device__ __forceinline__ void fb_output(uint32_t acc, const float2* cs, int64_t cs_step, int lane, int rows, bf16* dst, int64_t ld, Drained drained) {
  dst += (int64_t)(lane & ~3) * ld + (lane & 3) * 8;
#pragma unroll 1
  for (int c = 0; c < 64; c += 32) {
    uint32_t rl[32], rh[32];
    tmem_ld32(acc + (uint32_t)c, rl);
    tmem_ld32(acc + (uint32_t)(64 + c), rh);
    tmem_ld_wait();
    if (c == 32) drained();
    if (cs && lane < rows) {
#pragma unroll
      for (int i = 0; i < 32; ++i) {
        const float2 t = cs[(int64_t)(c + i) * cs_step];
        const float a0 = __uint_as_float(rl[i]), b0 = __uint_as_float(rh[i]);
        rl[i] = __float_as_uint(a0 * t.x + b0 * t.y);
        rh[i] = __float_as_uint(b0 * t.x - a0 * t.y);
      }
    }
    __syncwarp();
#pragma unroll
    for (int w = 0; w < 2; ++w) {
      uint4 v[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) v[k] = pack8(reinterpret_cast<const float*>(w ? rh : rl) + 8 * k);
      quad_transpose(v, lane);
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if ((lane & ~3) + k < rows) *reinterpret_cast<uint4*>(dst + (int64_t)k * ld + 64 * w + c) = v[k];
    }
    __syncwarp();
  }
}

constexpr int FB_THREADS = 512;
// Registers of the roles' warpgroups: loads and products | P', dS' | P', dS' | output.  Their sum is at most the 4 x 128
// that the block is launched with.
constexpr int FB_REGS_ISSUE = 72, FB_REGS_SOFTMAX = 160, FB_REGS_OUT = 112;
static_assert(FB_REGS_ISSUE + 2 * FB_REGS_SOFTMAX + FB_REGS_OUT <= 4 * 128, "register file");
template <int N> __device__ __forceinline__ void regs_dec() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N)); }
template <int N> __device__ __forceinline__ void regs_inc() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N)); }

// Shared memory of the dK/dV kernel: [K_j, V_j 64 KB | 3 query tiles 96 KB | 2 dO tiles 64 KB | their row statistics | barriers].
// A query tile is in use from its S' to its dK, more than a step, a dO tile from its dP' to its dV.
constexpr int FB_QS = 3, FB_OS = 2;
constexpr int FB_TILE = 2 * FA_TILE;              // 128 rows x 128 columns
constexpr int FB_X_OFF = 0;
constexpr int FB_Q_OFF = 2 * FB_TILE;
constexpr int FB_O_OFF = FB_Q_OFF + FB_QS * FB_TILE;
constexpr int FB_LD_OFF = FB_O_OFF + FB_OS * FB_TILE;
constexpr int FB_BAR_OFF = FB_LD_OFF + FB_OS * 1024;
constexpr int FB_SMEM_BYTES = FB_BAR_OFF + 256;

__global__ void __launch_bounds__(FB_THREADS, 1)
flash_bwd_dkv_kernel(const FlashBwdParams P, const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                     const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_o) {
  extern __shared__ __align__(1024) uint8_t fb_smem[];
  const uint32_t base = smem_u32(fb_smem);
  if (base & 1023u) {                              // the whole of the block's shared memory is in use: no room to align by hand
    pdl_wait();
    set_status(P.status, REVFFN_ERR_CUDA);
    return;
  }
  const uint32_t bars = base + FB_BAR_OFF;
  auto bar = [&](int i) -> uint32_t { return bars + 8u * (uint32_t)i; };
  enum { B_KFULL = 0, B_VFULL, B_KEMPTY, B_VEMPTY, B_QFULL, B_QEMPTY = B_QFULL + FB_QS, B_OFULL = B_QEMPTY + FB_QS, B_OEMPTY = B_OFULL + FB_OS,
         B_SFULL = B_OEMPTY + FB_OS, B_PHALF, B_PFULL, B_DPFULL, B_DSFULL, B_DVFULL, B_DKFULL, B_DVEMPTY, B_DKEMPTY, B_DRAIN, B_COUNT };
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(fb_smem + FB_BAR_OFF + 8 * B_COUNT);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  int* issued = reinterpret_cast<int*>(tmem_slot + 2);      // [2 + FB_QS + FB_OS]: k, v, query stages, dO stages -> phase + 1
  static_assert(8 * B_COUNT + 4 * (2 + 2 + FB_QS + FB_OS) <= 256, "barrier block");

  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  const int n_blk = P.Sp / FA_BLK;                  // 128-row blocks per head
  const int per = P.items / n_blk;                  // (sequence, key/value head) pairs
  // items with low key blocks come first: they see the most query tiles
  struct Item { int blk, grp, steps; };
  auto item_of = [&](int r) -> Item {
    const int it = fb_item(r);
    Item x;
    x.blk = it / per; x.grp = it - x.blk * per;
    x.steps = it < P.items ? P.rep * (n_blk - x.blk) : 0;      // every query head of the group in turn
    return x;
  };

  if (threadIdx.x == 0) {
    mbar_init(bar(B_KFULL), 1); mbar_init(bar(B_VFULL), 1); mbar_init(bar(B_KEMPTY), 1); mbar_init(bar(B_VEMPTY), 1);
    for (int s = 0; s < FB_QS; ++s) { mbar_init(bar(B_QFULL + s), 1); mbar_init(bar(B_QEMPTY + s), 1); }
    for (int s = 0; s < FB_OS; ++s) { mbar_init(bar(B_OFULL + s), 1); mbar_init(bar(B_OEMPTY + s), 1 + 8); }
    mbar_init(bar(B_SFULL), 1); mbar_init(bar(B_PHALF), 8); mbar_init(bar(B_PFULL), 8);
    mbar_init(bar(B_DPFULL), 1); mbar_init(bar(B_DSFULL), 8);
    mbar_init(bar(B_DVFULL), 1); mbar_init(bar(B_DKFULL), 1); mbar_init(bar(B_DVEMPTY), 4); mbar_init(bar(B_DKEMPTY), 4);
    mbar_init(bar(B_DRAIN), 1);
    for (int i = 0; i < 2 + FB_QS + FB_OS; ++i) issued[i] = 0;
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(smem_u32(tmem_slot)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  pdl_wait();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // TMEM columns: S' 0..127, dP' 128..255, dV 256..383, dK 384..511.  P' and dS' (bf16 pairs): 32 columns at the start of each
  // half of S' and dP', so that a warp overwrites only what it has read itself.
  // fp32 accumulate, bf16 operands, M = N = 128; the accumulating products' B is stored [row, hd] (N contiguous)
  const uint32_t idesc_sd = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(FA_BLK >> 3) << 17) | ((uint32_t)(FA_BLK >> 4) << 24);
  const uint32_t idesc_acc = idesc_sd | (1u << 16);
  const int role = warp >> 2;                       // warpgroup: loads and products, softmax, softmax, output
  auto arrive = [&](int i) {
    tc_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive(bar(i));
  };

  if (role == 0) {
    regs_dec<FB_REGS_ISSUE>();
    if (warp == 0) {
    // ------------------------------------------------------------------ producer
    if (lane == 0) {
      bool ok = true;
      int nq = 0, no = 0;                  // query and dO tiles loaded so far
      auto load_q = [&](int yr) {
        const int st = nq % FB_QS;
        const uint32_t ph = (uint32_t)(nq / FB_QS) & 1u;
        ok = mbar_wait(bar(B_QEMPTY + st), ph ^ 1u, abort_flag, P.status);
        if (!ok) return;
        mbar_expect_tx(bar(B_QFULL + st), FB_TILE);
        issued[2 + st] = (int)ph + 1;
        for (int kb = 0; kb < 2; ++kb)
          tma_load_2d(base + FB_Q_OFF + st * FB_TILE + kb * FA_TILE, &map_q, 64 * kb, yr, bar(B_QFULL + st));
        ++nq;
      };
      auto load_o = [&](int yr) {
        const int st = no % FB_OS;
        const uint32_t ph = (uint32_t)(no / FB_OS) & 1u;
        ok = mbar_wait(bar(B_OEMPTY + st), ph ^ 1u, abort_flag, P.status);
        if (!ok) return;
        mbar_expect_tx(bar(B_OFULL + st), FB_TILE + 1024);
        issued[2 + FB_QS + st] = (int)ph + 1;
        bulk_load_1d(base + FB_LD_OFF + st * 1024, P.lse_d + yr / 2, 1024, bar(B_OFULL + st));
        for (int kb = 0; kb < 2; ++kb)
          tma_load_2d(base + FB_O_OFF + st * FB_TILE + kb * FA_TILE, &map_o, 64 * kb, yr, bar(B_OFULL + st));
        ++no;
      };
      // K_j and V_j of item r, once the last product of the item before has read its own
      auto load_k = [&](int r, const Item& x) {
        ok = mbar_wait(bar(B_KEMPTY), ((uint32_t)r & 1u) ^ 1u, abort_flag, P.status);
        if (!ok) return;
        mbar_expect_tx(bar(B_KFULL), FB_TILE);
        issued[0] = (r & 1) + 1;
        for (int kb = 0; kb < 2; ++kb)
          tma_load_2d(base + FB_X_OFF + kb * FA_TILE, &map_k, 64 * kb, x.grp * P.Sp + x.blk * FA_BLK, bar(B_KFULL));
      };
      auto load_v = [&](int r, const Item& x) {
        ok = mbar_wait(bar(B_VEMPTY), ((uint32_t)r & 1u) ^ 1u, abort_flag, P.status);
        if (!ok) return;
        mbar_expect_tx(bar(B_VFULL), FB_TILE);
        issued[1] = (r & 1) + 1;
        for (int kb = 0; kb < 2; ++kb)
          tma_load_2d(base + FB_X_OFF + FB_TILE + kb * FA_TILE, &map_v, 64 * kb, x.grp * P.Sp + x.blk * FA_BLK, bar(B_VFULL));
      };
      // in the order in which places fall free: dO of step g, then the query tile of step g + 1
      Item x = item_of(0);
      if (x.steps > 0) load_k(0, x);
      if (ok && x.steps > 0) load_q(x.grp * P.rep * P.Sp + x.blk * FA_BLK);
      for (int r = 0; ok && x.steps > 0; ++r) {
        load_v(r, x);
        int head = x.grp * P.rep, t = x.blk;      // a head's rows at and below the keys; then the group's next head
        for (int s = 0; ok && s < x.steps; ++s) {
          load_o(head * P.Sp + t * FA_BLK);
          if (++t == n_blk) { t = x.blk; ++head; }
          if (ok && s + 1 < x.steps) load_q(head * P.Sp + t * FA_BLK);
        }
        x = item_of(r + 1);
        if (ok && x.steps > 0) load_k(r + 1, x);
        if (ok && x.steps > 0) load_q(x.grp * P.rep * P.Sp + x.blk * FA_BLK);
      }
      pdl_trigger();
    }
    } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    const uint32_t tb = __shfl_sync(0xffffffffu, tmem_base, 0), sb = __shfl_sync(0xffffffffu, base, 0);
    auto wait = [&](int i, uint32_t parity) -> bool {
      const bool got = mbar_wait_warp(bar(i), parity, abort_flag, P.status);
      tc_fence_after();
      return got;
    };
    // S' = K_j Q_t^T (w = 0), dP' = V_j dO_t^T (w = 1); both operands in 64-column tiles of 16 KB, 16 columns an instruction
    auto issue_sd = [&](int w, uint32_t y_off, int done, int free) {
      const uint64_t a_desc = make_smem_desc(sb + FB_X_OFF + w * FB_TILE, 16, 1024), b_desc = make_smem_desc(sb + y_off, 16, 1024);
      if (elect_one()) {
#pragma unroll
        for (int k = 0; k < 8; ++k)
          tc_mma(tb + (uint32_t)(128 * w), a_desc + (uint64_t)((k >> 2) * (FA_TILE >> 4) + 2 * (k & 3)),
                 b_desc + (uint64_t)((k >> 2) * (FA_TILE >> 4) + 2 * (k & 3)), idesc_sd, k != 0 ? 1u : 0u);
        tc_commit(bar(done));
        if (free >= 0) tc_commit(bar(free));      // the item's last product with K_j or V_j
      }
      __syncwarp();
    };
    // the walked tile again, as a [128 rows (K), 128 columns (N)] operand: two 64-column halves 16 KB apart; 16 rows (8 packed
    // columns of the A operand) an instruction, the second 64 rows from the second half of the score columns.  k0 = 0, 2: the
    // first or second 32 rows of each half.
    auto issue_acc = [&](int w, uint32_t y_off, int k0, bool first) {
      const uint64_t b_desc = make_smem_desc(sb + y_off, FA_TILE, 1024);
      if (elect_one()) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int k = (i & 1) + k0 + 4 * (i >> 1);
          tc_mma_ta(tb + (uint32_t)(256 + 128 * w), tb + (uint32_t)(128 * w + 64 * (k >> 2) + 8 * (k & 3)), b_desc + (uint64_t)(128 * k),
                    idesc_acc, first && i == 0 ? 0u : 1u);
        }
      }
      __syncwarp();
    };
    auto commit = [&](int i) {
      if (elect_one()) tc_commit(bar(i));
      __syncwarp();
    };
    auto s_prime = [&](int g, bool last) -> bool {      // S' of step g; last: of its item
      if (!wait(B_QFULL + g % FB_QS, (uint32_t)(g / FB_QS) & 1u)) return false;
      issue_sd(0, (uint32_t)(FB_Q_OFF + g % FB_QS * FB_TILE), B_SFULL, last ? B_KEMPTY : -1);
      return true;
    };
    auto dp_prime = [&](int g, bool last) -> bool {
      if (!wait(B_OFULL + g % FB_OS, (uint32_t)(g / FB_OS) & 1u)) return false;
      issue_sd(1, (uint32_t)(FB_O_OFF + g % FB_OS * FB_TILE), B_DPFULL, last ? B_VEMPTY : -1);
      return true;
    };
    int g = 0;                             // steps so far, of all items
    int steps = item_of(0).steps;
    bool ok = wait(B_KFULL, 0u) && s_prime(0, steps == 1) && wait(B_VFULL, 0u) && dp_prime(0, steps == 1);
    for (int r = 0; ok && steps > 0; ++r) {
      const int next_steps = item_of(r + 1).steps;
      const uint32_t item_ph = (uint32_t)r & 1u;
      for (int s = 0; s < steps; ++s, ++g) {
        const uint32_t ph = (uint32_t)g & 1u;
        const bool last = s + 1 == steps, more = !last || next_steps > 0;
        const bool ends = last ? next_steps == 1 : s + 2 == steps;      // step g + 1 is the last of its item
        const uint32_t q_off = (uint32_t)(FB_Q_OFF + g % FB_QS * FB_TILE), o_off = (uint32_t)(FB_O_OFF + g % FB_OS * FB_TILE);
        if (!(ok = wait(B_PHALF, ph) && (s > 0 || r == 0 || wait(B_DVEMPTY, item_ph ^ 1u)))) break;
        issue_acc(0, o_off, 0, s == 0);
        if (!(ok = wait(B_PFULL, ph))) break;
        issue_acc(0, o_off, 2, false);
        commit(B_OEMPTY + g % FB_OS);
        if (last) commit(B_DVFULL);
        if (more && !(ok = (!last || wait(B_KFULL, item_ph ^ 1u)) && s_prime(g + 1, ends))) break;
        if (!(ok = wait(B_DSFULL, ph) && (s > 0 || r == 0 || wait(B_DKEMPTY, item_ph ^ 1u)))) break;
        issue_acc(1, q_off, 0, s == 0);
        issue_acc(1, q_off, 2, false);
        commit(B_QEMPTY + g % FB_QS);
        if (last) commit(B_DKFULL);
        if (more && !(ok = (!last || wait(B_VFULL, item_ph ^ 1u)) && dp_prime(g + 1, ends))) break;
      }
      steps = next_steps;
    }
    if (!ok) {
      // an abandoned wait: products issued so far must have finished before the teardown frees what they use
      commit(B_DRAIN);
      const long long t0 = clock64();
      while (!mbar_try_wait(bar(B_DRAIN), 0u) && clock64() - t0 < TC_WAIT_CYCLES) {}
    }
    __syncwarp();
    }
  } else if (role < 3) {
    // ------------------------------------------------------------------ P' / dS' (warps 4..11)
    regs_inc<FB_REGS_SOFTMAX>();
    const int q = warp & 3;                      // TMEM lane quadrant this warp may access
    const int hh = role - 1;                     // which 64 of the step's 128 columns
    const int row = q * 32 + lane;               // own row within the block
    const uint32_t s_addr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(64 * hh), d_addr = s_addr + 128u;
    const float cl = P.scale_log2e, scale = P.scale;
    bool ok = true;
    int g = 0;
    for (int r = 0; ok; ++r) {
      const Item x = item_of(r);
      if (x.steps == 0) break;
      const int edge = row - 64 * hh;            // in the diagonal tile
      int t = x.blk;
      for (int s = 0; s < x.steps; ++s, ++g) {
        const uint32_t ph = (uint32_t)g & 1u;
        const bool mask = t == x.blk;            // the diagonal tile
        // the tile's row statistics came with its dO
        const float4* ld = reinterpret_cast<const float4*>(fb_smem + FB_LD_OFF + (g % FB_OS) * 1024) + 32 * hh;
        uint32_t p0[32], p1[32], w[16];
        if (!mbar_wait_warp(bar(B_OFULL + g % FB_OS), (uint32_t)(g / FB_OS) & 1u, abort_flag, P.status)) { ok = false; break; }
        if (!mbar_wait_warp(bar(B_SFULL), ph, abort_flag, P.status)) { ok = false; break; }
        tc_fence_after();
        tmem_ld32(s_addr, p0);
        tmem_ld32(s_addr + 32, p1);
        tmem_ld_wait();
        if (mask) { fb_mask<true>(p0, edge, 0xff800000u); fb_mask<true>(p1, edge - 32, 0xff800000u); }
        __syncwarp();
        fb_probs<true>(p0, ld, 0.f, cl, w);
        tmem_st16(s_addr, w);
        tmem_st_wait();
        arrive(B_PHALF);
        fb_probs<true>(p1, ld + 16, 0.f, cl, w);
        tmem_st16(s_addr + 16, w);
        tmem_st_wait();
        arrive(B_PFULL);
        if (!mbar_wait_warp(bar(B_DPFULL), ph, abort_flag, P.status)) { ok = false; break; }
        tc_fence_after();
        uint32_t rd[32], w1[16];
        tmem_ld32(d_addr, rd);
        tmem_ld_wait();
        if (mask) fb_mask<true>(rd, edge, 0u);      // (their weights are zero, their products may be anything)
        __syncwarp();
        fb_dscores<true>(p0, rd, ld, 0.f, scale, w);
        tmem_ld32(d_addr + 32, rd);
        tmem_ld_wait();
        if (mask) fb_mask<true>(rd, edge - 32, 0u);
        __syncwarp();
        tmem_st16(d_addr, w);
        fb_dscores<true>(p1, rd, ld + 16, 0.f, scale, w1);
        tmem_st16(d_addr + 16, w1);
        tmem_st_wait();
        arrive(B_DSFULL);
        if (lane == 0) mbar_arrive(bar(B_OEMPTY + g % FB_OS));      // the statistics have been read
        if (++t == n_blk) t = x.blk;
      }
    }
  } else {
    // ------------------------------------------------------------------ output (warps 12..15), beside the next item's steps
    regs_dec<FB_REGS_OUT>();
    const int q = warp & 3;
    const uint32_t lane_addr = tmem_base + ((uint32_t)(q * 32) << 16);
    for (int r = 0;; ++r) {
      const Item x = item_of(r);
      if (x.steps == 0) break;
      const int pos0 = x.blk * FA_BLK + q * 32, rows = min(32, P.S - pos0);
      const int seq = x.grp / P.heads_own, head = x.grp % P.heads_own;
      const int64_t tok = (int64_t)seq * P.S + pos0;
      const uint32_t ph = (uint32_t)r & 1u;
      bool ok = true;
#pragma unroll 1
      for (int a = 0; a < 2; ++a) {          // a = 0: dV as it is, a = 1: dK with the rotation undone
        if (!(ok = mbar_wait_warp(bar(B_DVFULL + a), ph, abort_flag, P.status))) break;
        tc_fence_after();
        const int64_t ld = a ? P.ld_out1 : P.ld_out0;
        fb_output(lane_addr + (uint32_t)(256 + 128 * a), a ? P.cs + pos0 + lane : nullptr, P.S, lane, rows,
                  (a ? P.out1 + P.col1 : P.out0 + P.col0) + tok * ld + head * FA_HD, ld, [&]() { arrive(B_DVEMPTY + a); });
      }
      if (!ok) break;
    }
  }

  // ------------------------------------------------------------------ teardown
  tc_fence_before();
  __syncthreads();
  if (*abort_flag && threadIdx.x == 0) {
    // loads already issued into this CTA's shared memory must land before the CTA exits
    for (int i = 0; i < 2 + FB_QS + FB_OS; ++i) {
      if (issued[i] == 0) continue;
      const int b = i < 2 ? B_KFULL + i : (i < 2 + FB_QS ? B_QFULL + i - 2 : B_OFULL + i - 2 - FB_QS);
      const long long t0 = clock64();
      while (!mbar_try_wait(bar(b), (uint32_t)(issued[i] - 1)) && clock64() - t0 < TC_WAIT_CYCLES) {}
    }
  }
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
  }
}

// ---------------------------------------------------------------------------
// dQ: the owned operands (Q_i, dO_i) sit in tensor memory as A operands (128 columns), S' and dP' take 128 columns each and
// dQ the last 128.  The score columns are free once they are in registers, so S' of the next step runs under this
// step's exponentials.  Shared memory: rings of key and value tiles; a key tile is in use from its S' to its dQ, a value
// tile for one product.  The output warps also bring the next item's owned operands.
// ---------------------------------------------------------------------------
constexpr int FQ_KS = 4, FQ_VS = 3;
constexpr int FQ_V_OFF = FQ_KS * FB_TILE;
constexpr int FQ_BAR_OFF = FQ_V_OFF + FQ_VS * FB_TILE;
constexpr int FQ_SMEM_BYTES = FQ_BAR_OFF + 256;

__global__ void __launch_bounds__(FB_THREADS, 1)
flash_bwd_dq_kernel(const FlashBwdParams P, const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v) {
  extern __shared__ __align__(1024) uint8_t fb_smem[];
  const uint32_t base = smem_u32(fb_smem);
  if (base & 1023u) {
    pdl_wait();
    set_status(P.status, REVFFN_ERR_CUDA);
    return;
  }
  const uint32_t bars = base + FQ_BAR_OFF;
  auto bar = [&](int i) -> uint32_t { return bars + 8u * (uint32_t)i; };
  // X: the item's own operands, Q_i (0) and dO_i (1): in place, and no product reads them any more
  enum { B_XFULL = 0, B_XEMPTY = 2, B_KFULL = 4, B_KEMPTY = B_KFULL + FQ_KS, B_VFULL = B_KEMPTY + FQ_KS, B_VEMPTY = B_VFULL + FQ_VS,
         B_SFULL = B_VEMPTY + FQ_VS, B_SEMPTY, B_DPFULL, B_DSHALF, B_DSFULL, B_ACCFULL, B_ACCEMPTY, B_DRAIN, B_COUNT };
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(fb_smem + FQ_BAR_OFF + 8 * B_COUNT);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  int* issued = reinterpret_cast<int*>(tmem_slot + 2);      // [FQ_KS + FQ_VS]: stage -> phase + 1
  static_assert(8 * B_COUNT + 4 * (2 + FQ_KS + FQ_VS) <= 256, "barrier block");

  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  const int n_blk = P.Sp / FA_BLK;
  const int per = P.items / n_blk;                       // (sequence, head) pairs
  // items with high query blocks come first: they see the most key tiles
  struct Item { int blk, grp, steps; };
  auto item_of = [&](int r) -> Item {
    const int it = fb_item(r);
    Item x;
    x.blk = n_blk - 1 - it / per; x.grp = it % per;
    x.steps = it < P.items ? x.blk + 1 : 0;              // key tiles 0 .. the diagonal one
    return x;
  };

  if (threadIdx.x == 0) {
    for (int w = 0; w < 2; ++w) { mbar_init(bar(B_XFULL + w), 4); mbar_init(bar(B_XEMPTY + w), 1); }
    for (int s = 0; s < FQ_KS; ++s) { mbar_init(bar(B_KFULL + s), 1); mbar_init(bar(B_KEMPTY + s), 1); }
    for (int s = 0; s < FQ_VS; ++s) { mbar_init(bar(B_VFULL + s), 1); mbar_init(bar(B_VEMPTY + s), 1); }
    mbar_init(bar(B_SFULL), 1); mbar_init(bar(B_SEMPTY), 8);
    mbar_init(bar(B_DPFULL), 1); mbar_init(bar(B_DSHALF), 8); mbar_init(bar(B_DSFULL), 8);
    mbar_init(bar(B_ACCFULL), 1); mbar_init(bar(B_ACCEMPTY), 4); mbar_init(bar(B_DRAIN), 1);
    for (int i = 0; i < FQ_KS + FQ_VS; ++i) issued[i] = 0;
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(smem_u32(tmem_slot)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  pdl_wait();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // TMEM columns: S' 0..127, dP' 128..255 (dS' as bf16 pairs at the start of each half of it), Q_i 256..319, dO_i 320..383
  // (packed pairs), dQ 384..511
  const uint32_t idesc_sd = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(FA_BLK >> 3) << 17) | ((uint32_t)(FA_BLK >> 4) << 24);
  const uint32_t idesc_acc = idesc_sd | (1u << 16);
  const int role = warp >> 2;
  auto arrive = [&](int i) {
    tc_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive(bar(i));
  };

  if (role == 0) {
    regs_dec<FB_REGS_ISSUE>();
    if (warp == 0) {
    // ------------------------------------------------------------------ producer
    if (lane == 0) {
      bool ok = true;
      int g = 0;
      for (int r = 0; ok; ++r) {
        const Item x = item_of(r);
        if (x.steps == 0) break;
        const int kv_row0 = (x.grp / P.rep) * P.Sp;
        for (int s = 0; s < x.steps; ++s, ++g) {
          const int yr = kv_row0 + s * FA_BLK, sk = g % FQ_KS, sv = g % FQ_VS;
          const uint32_t phk = (uint32_t)(g / FQ_KS) & 1u, phv = (uint32_t)(g / FQ_VS) & 1u;
          if (!(ok = mbar_wait(bar(B_KEMPTY + sk), phk ^ 1u, abort_flag, P.status))) break;
          mbar_expect_tx(bar(B_KFULL + sk), FB_TILE);
          issued[sk] = (int)phk + 1;
          for (int kb = 0; kb < 2; ++kb) tma_load_2d(base + sk * FB_TILE + kb * FA_TILE, &map_k, 64 * kb, yr, bar(B_KFULL + sk));
          if (!(ok = mbar_wait(bar(B_VEMPTY + sv), phv ^ 1u, abort_flag, P.status))) break;
          mbar_expect_tx(bar(B_VFULL + sv), FB_TILE);
          issued[FQ_KS + sv] = (int)phv + 1;
          for (int kb = 0; kb < 2; ++kb) tma_load_2d(base + FQ_V_OFF + sv * FB_TILE + kb * FA_TILE, &map_v, 64 * kb, yr, bar(B_VFULL + sv));
        }
      }
      pdl_trigger();
    }
    } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    const uint32_t tb = __shfl_sync(0xffffffffu, tmem_base, 0), sb = __shfl_sync(0xffffffffu, base, 0);
    auto wait = [&](int i, uint32_t parity) -> bool {
      const bool got = mbar_wait_warp(bar(i), parity, abort_flag, P.status);
      tc_fence_after();
      return got;
    };
    // S' = Q_i K_t^T (w = 0), dP' = dO_i V_t^T (w = 1) of step g; last: of its item
    auto issue_sd = [&](int w, int g, bool last) {
      const uint64_t b_desc = make_smem_desc(sb + (w ? FQ_V_OFF + g % FQ_VS * FB_TILE : g % FQ_KS * FB_TILE), 16, 1024);
      if (elect_one()) {
#pragma unroll
        for (int k = 0; k < 8; ++k)
          tc_mma_ta(tb + (uint32_t)(128 * w), tb + (uint32_t)(256 + 64 * w + 8 * k),
                    b_desc + (uint64_t)((k >> 2) * (FA_TILE >> 4) + 2 * (k & 3)), idesc_sd, k != 0 ? 1u : 0u);
        tc_commit(bar(w ? B_DPFULL : B_SFULL));
        if (w) tc_commit(bar(B_VEMPTY + g % FQ_VS));
        if (last) tc_commit(bar(B_XEMPTY + w));
      }
      __syncwarp();
    };
    auto wait_k = [&](int s) { return wait(B_KFULL + s % FQ_KS, (uint32_t)(s / FQ_KS) & 1u); };
    auto wait_v = [&](int s) { return wait(B_VFULL + s % FQ_VS, (uint32_t)(s / FQ_VS) & 1u); };
    int g = 0;                             // steps so far, of all items
    int steps = item_of(0).steps;
    bool ok = wait(B_XFULL, 0u) && wait_k(0);
    if (ok) issue_sd(0, 0, steps == 1);
    ok = ok && wait(B_XFULL + 1, 0u) && wait_v(0);
    if (ok) issue_sd(1, 0, steps == 1);
    for (int r = 0; ok && steps > 0; ++r) {
      const int next_steps = item_of(r + 1).steps;
      const uint32_t item_ph = (uint32_t)r & 1u;
      for (int s = 0; s < steps; ++s, ++g) {
        const uint32_t ph = (uint32_t)g & 1u;
        const bool last = s + 1 == steps, more = !last || next_steps > 0;
        const bool ends = last ? next_steps == 1 : s + 2 == steps;      // step g + 1 is the last of its item
        if (more) {
          if (!(ok = (!last || wait(B_XFULL, item_ph ^ 1u)) && wait_k(g + 1) && wait(B_SEMPTY, ph))) break;
          issue_sd(0, g + 1, ends);
        }
        // dQ += dS' K_t, as the halves of dS' become readable: K_t's two 64-column tiles read as one [128 keys, 128 columns]
        // operand, halves 16 KB apart
        const uint64_t b_desc = make_smem_desc(sb + g % FQ_KS * FB_TILE, FA_TILE, 1024);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          if (ok) ok = wait(h ? B_DSFULL : B_DSHALF, ph) && (h > 0 || s > 0 || r == 0 || wait(B_ACCEMPTY, item_ph ^ 1u));
          if (ok && elect_one()) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const int k = (i & 1) + 2 * h + 4 * (i >> 1);
              tc_mma_ta(tb + 384u, tb + (uint32_t)(128 + 64 * (k >> 2) + 8 * (k & 3)), b_desc + (uint64_t)(128 * k), idesc_acc, (s | h | i) != 0 ? 1u : 0u);
            }
            if (h) tc_commit(bar(B_KEMPTY + g % FQ_KS));
            if (h && last) tc_commit(bar(B_ACCFULL));
          }
          __syncwarp();
        }
        if (!ok) break;
        if (more) {
          if (!(ok = (!last || wait(B_XFULL + 1, item_ph ^ 1u)) && wait_v(g + 1))) break;
          issue_sd(1, g + 1, ends);
        }
      }
      steps = next_steps;
    }
    if (!ok) {
      // an abandoned wait: products issued so far must have finished before the teardown frees what they use
      if (elect_one()) tc_commit(bar(B_DRAIN));
      __syncwarp();
      const long long t0 = clock64();
      while (!mbar_try_wait(bar(B_DRAIN), 0u) && clock64() - t0 < TC_WAIT_CYCLES) {}
    }
    __syncwarp();
    }
  } else if (role < 3) {
    // ------------------------------------------------------------------ dS' (warps 4..11)
    regs_inc<FB_REGS_SOFTMAX>();
    const int q = warp & 3;
    const int hh = role - 1;                     // which 64 of the tile's 128 keys
    const int row = q * 32 + lane;
    const uint32_t s_addr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(64 * hh), d_addr = s_addr + 128u;
    const float cl = P.scale_log2e, scale = P.scale;
    bool ok = true;
    int g = 0;
    for (int r = 0; ok; ++r) {
      const Item x = item_of(r);
      if (x.steps == 0) break;
      const int64_t at = (int64_t)x.grp * P.Sp + x.blk * FA_BLK + row;
      const float* const stats = reinterpret_cast<const float*>(P.lse_d + (at >> 1)) + (at & 1);
      const float nl = stats[0], nd = stats[2];
      const int edge = row - 64 * hh;            // in the diagonal tile
      for (int s = 0; s < x.steps; ++s, ++g) {
        const uint32_t ph = (uint32_t)g & 1u;
        const bool mask = s == x.blk;
        uint32_t p0[32], p1[32], w[16], w1[16], rd[32];
        if (!mbar_wait_warp(bar(B_SFULL), ph, abort_flag, P.status)) { ok = false; break; }
        tc_fence_after();
        tmem_ld32(s_addr, p0);
        tmem_ld32(s_addr + 32, p1);
        tmem_ld_wait();
        arrive(B_SEMPTY);
        if (mask) { fb_mask<false>(p0, edge, 0xff800000u); fb_mask<false>(p1, edge - 32, 0xff800000u); }
        __syncwarp();
        fb_probs<false>(p0, nullptr, nl, cl, w);
        fb_probs<false>(p1, nullptr, nl, cl, w);
        if (!mbar_wait_warp(bar(B_DPFULL), ph, abort_flag, P.status)) { ok = false; break; }
        tc_fence_after();
        tmem_ld32(d_addr, rd);
        tmem_ld_wait();
        if (mask) fb_mask<false>(rd, edge, 0u);
        __syncwarp();
        fb_dscores<false>(p0, rd, nullptr, nd, scale, w);
        tmem_ld32(d_addr + 32, rd);
        tmem_ld_wait();
        if (mask) fb_mask<false>(rd, edge - 32, 0u);
        __syncwarp();
        tmem_st16(d_addr, w);
        tmem_st_wait();
        arrive(B_DSHALF);
        fb_dscores<false>(p1, rd, nullptr, nd, scale, w1);
        tmem_st16(d_addr + 16, w1);
        tmem_st_wait();
        arrive(B_DSFULL);
      }
    }
  } else {
    // ------------------------------------------------------------------ owned operands and output (warps 12..15)
    regs_dec<FB_REGS_OUT>();
    const int q = warp & 3;
    const uint32_t lane_addr = tmem_base + ((uint32_t)(q * 32) << 16);
    // this thread's row of Q_i (w = 0) or dO_i (w = 1) of item x into tensor memory, once the item before is done with it
    auto own = [&](int w, int r, const Item& x) -> bool {
      // eight rows of 64 bytes an instruction, then four pieces of one row to each lane
      const uint4* src = reinterpret_cast<const uint4*>((w ? P.x1 : P.x0) + (int64_t)(x.grp * P.Sp + x.blk * FA_BLK + q * 32 + (lane & ~3)) * FA_HD) + (lane & 3);
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        uint4 v[2][4];
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
          for (int k = 0; k < 4; ++k) v[c][k] = __ldg(src + k * (FA_HD / 8) + 8 * half + 4 * c);
#pragma unroll
        for (int c = 0; c < 2; ++c) quad_transpose(v[c], lane);
        if (half == 0) {
          if (!mbar_wait_warp(bar(B_XEMPTY + w), ((uint32_t)r & 1u) ^ 1u, abort_flag, P.status)) return false;
          tc_fence_after();
        }
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          uint32_t x16[16];
#pragma unroll
          for (int k = 0; k < 4; ++k) { x16[4 * k] = v[c][k].x; x16[4 * k + 1] = v[c][k].y; x16[4 * k + 2] = v[c][k].z; x16[4 * k + 3] = v[c][k].w; }
          tmem_st16(lane_addr + (uint32_t)(256 + 64 * w + 32 * half + 16 * c), x16);
        }
      }
      tmem_st_wait();
      arrive(B_XFULL + w);
      return true;
    };
    Item x = {0, 0, 0};
    bool ok = true;
    for (int r = -1; ok; ++r) {
      const Item nx = item_of(r + 1);
#pragma unroll 1
      for (int w = 0; ok && w < 2 && nx.steps > 0; ++w) ok = own(w, r + 1, nx);
      if (!ok) break;
      if (r < 0) { x = nx; if (x.steps == 0) break; continue; }
      const int pos0 = x.blk * FA_BLK + q * 32, rows = min(32, P.S - pos0);
      const int seq = x.grp / P.heads_own, head = x.grp % P.heads_own;
      const int64_t tok = (int64_t)seq * P.S + pos0;
      if (!(ok = mbar_wait_warp(bar(B_ACCFULL), (uint32_t)r & 1u, abort_flag, P.status))) break;
      tc_fence_after();
      fb_output(lane_addr + 384u, P.cs + pos0 + lane, P.S, lane, rows, P.out1 + tok * P.ld_out1 + P.col1 + head * FA_HD, P.ld_out1, [&]() { arrive(B_ACCEMPTY); });
      x = nx;
      if (x.steps == 0) break;
    }
  }

  // ------------------------------------------------------------------ teardown
  tc_fence_before();
  __syncthreads();
  if (*abort_flag && threadIdx.x == 0) {
    for (int i = 0; i < FQ_KS + FQ_VS; ++i) {
      if (issued[i] == 0) continue;
      const long long t0 = clock64();
      while (!mbar_try_wait(bar(i < FQ_KS ? B_KFULL + i : B_VFULL + i - FQ_KS), (uint32_t)(issued[i] - 1)) && clock64() - t0 < TC_WAIT_CYCLES) {}
    }
  }
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
  }
}

// q, d_o: [B * n_heads * Sp, 128]; k, v: [B * n_kv_heads * Sp, 128] bf16 head-major (rows past the sequence zero).
// Outputs token-major bf16, rotation undone: dq [T, ld_dq]; dk at column 0 and dv at column dv_col of dkv [T, ld_dkv].
// The two launches depend on nothing of each other: st_dkv and st_dq may be different streams.
inline int launch_flash_bwd(const bf16* q, const bf16* k, const bf16* v, const bf16* d_o, const float* lse_d, const float2* cs,
                            int batch, int n_heads, int n_kv_heads, int S, int Sp, bf16* dq, int64_t ld_dq, bf16* dkv,
                            int64_t ld_dkv, int dv_col, int* status, cudaStream_t st_dkv, cudaStream_t st_dq) {
  TcState& s = tc_state();
  if (!s.ready) return REVFFN_ERR_CUDA;
  if (batch <= 0) return REVFFN_OK;
  static bool attr_set[64] = {false};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return REVFFN_ERR_CUDA;
  if (!attr_set[dev]) {
    if (cudaFuncSetAttribute(flash_bwd_dkv_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, FB_SMEM_BYTES) != cudaSuccess ||
        cudaFuncSetAttribute(flash_bwd_dq_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, FQ_SMEM_BYTES) != cudaSuccess)
      return REVFFN_ERR_CUDA;
    attr_set[dev] = true;
  }
  const uint64_t q_rows = (uint64_t)batch * n_heads * Sp, kv_rows = (uint64_t)batch * n_kv_heads * Sp;
  CUtensorMap k128, v128, q128, do128;
  int r = 0;
  if (!r) r = tc_make_map(&k128, k, FA_HD, kv_rows, FA_HD, 64, 128);
  if (!r) r = tc_make_map(&v128, v, FA_HD, kv_rows, FA_HD, 64, 128);
  if (!r) r = tc_make_map(&q128, q, FA_HD, q_rows, FA_HD, 64, 128);
  if (!r) r = tc_make_map(&do128, d_o, FA_HD, q_rows, FA_HD, 64, 128);
  if (r) return r;
  FlashBwdParams P;
  P.S = S; P.Sp = Sp; P.n_heads = n_heads; P.rep = n_heads / n_kv_heads;
  P.lse_d = reinterpret_cast<const float4*>(lse_d);
  P.scale = 1.f / sqrtf((float)FA_HD);
  P.scale_log2e = P.scale * 1.4426950408889634f;
  P.status = status;
  P.cs = cs;
  P.out0 = dkv; P.ld_out0 = ld_dkv; P.col0 = dv_col;
  P.out1 = dkv; P.ld_out1 = ld_dkv; P.col1 = 0;
  P.heads_own = n_kv_heads;
  P.x0 = nullptr; P.x1 = nullptr;
  P.items = batch * n_kv_heads * (Sp / FA_BLK);
  launch_k(flash_bwd_dkv_kernel, std::min(P.items, s.n_sms), FB_THREADS, FB_SMEM_BYTES, st_dkv, P, k128, v128, q128, do128);
  if (cudaGetLastError() != cudaSuccess) return REVFFN_ERR_CUDA;
  P.out0 = nullptr; P.ld_out0 = 0; P.col0 = 0;
  P.out1 = dq; P.ld_out1 = ld_dq; P.col1 = 0;
  P.heads_own = n_heads;
  P.x0 = q; P.x1 = d_o;
  P.items = batch * n_heads * (Sp / FA_BLK);
  launch_k(flash_bwd_dq_kernel, std::min(P.items, s.n_sms), FB_THREADS, FQ_SMEM_BYTES, st_dq, P, k128, v128);
  return cudaGetLastError() == cudaSuccess ? REVFFN_OK : REVFFN_ERR_CUDA;
}

}  // namespace revffn
