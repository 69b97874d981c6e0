// Norm, router (logits, top-k, gates), permutation maps, gather and combine.
//
// Forward steps of MLP(Norm(Y1)) in Eq. 2 that are not matrix products:
//   rmsnorm_fwd        n = y * r * gamma, r = (mean(y^2)+eps)^-1/2
//   fold_router        W_rc = [W_r; w_sgate] * W_up   (so logits come straight from n)
//   router_topk        logits (fp64), top-k, softmax over the selected k, shared sigmoid gate
//   map_rank/assign    stable counting sort of (token, slot) pairs by expert -> padded rows
//   gather_rows        Up[row] = U[token(row)]
//   combine_rows       Z[t] = sum_s O[row(t,s)] + sgate_t * S[t]
#pragma once

#include <mutex>

#include "common.cuh"

namespace revffn {

// ---------------------------------------------------------------------------
// RMSNorm forward.  One warp per token; fp32 math; output in T plus r[t].
// norm_kind NONE: n = y, r = 1.
// A row's first 1024 elements stay in registers between the sum of squares and the scaling, all of their loads in
// flight together; only wider rows read the rest twice (8192 rows of 1024: 15.9 -> 11.4 us).
// ---------------------------------------------------------------------------
template <typename T> __device__ __forceinline__ void store4(T* p, float4 v);
template <> __device__ __forceinline__ void store4<float>(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
template <> __device__ __forceinline__ void store4<bf16>(bf16* p, float4 v) {
  __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
  *reinterpret_cast<uint2*>(p) = make_uint2(*reinterpret_cast<uint32_t*>(&lo), *reinterpret_cast<uint32_t*>(&hi));
}

template <typename T>
__device__ __forceinline__ void rmsnorm_row(const float* __restrict__ row, const float* __restrict__ gamma, float eps,
                                            int norm_none, int h, int lane, T* __restrict__ out, float* __restrict__ r_out) {
  constexpr int KEEP = 8;
  float4 v[KEEP];
#pragma unroll
  for (int q = 0; q < KEEP; ++q) {
    const int i = lane * 4 + q * 128;
    v[q] = i < h ? *reinterpret_cast<const float4*>(row + i) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  float r = 1.0f;
  if (!norm_none) {
    float ss = 0.f;
#pragma unroll
    for (int q = 0; q < KEEP; ++q) ss += v[q].x * v[q].x + v[q].y * v[q].y + v[q].z * v[q].z + v[q].w * v[q].w;
    for (int i = lane * 4 + KEEP * 128; i < h; i += 128) {
      const float4 w = *reinterpret_cast<const float4*>(row + i);
      ss += w.x * w.x + w.y * w.y + w.z * w.z + w.w * w.w;
    }
    ss = warp_sum(ss);
    r = rsqrtf(ss / (float)h + eps);
  }
  if (lane == 0) *r_out = r;
  auto put = [&](int i, float4 w) {
    float4 g = make_float4(1.f, 1.f, 1.f, 1.f);
    if (gamma && !norm_none) g = *reinterpret_cast<const float4*>(gamma + i);
    store4<T>(out + i, make_float4(w.x * r * g.x, w.y * r * g.y, w.z * r * g.z, w.w * r * g.w));
  };
#pragma unroll
  for (int q = 0; q < KEEP; ++q)
    if (lane * 4 + q * 128 < h) put(lane * 4 + q * 128, v[q]);
  for (int i = lane * 4 + KEEP * 128; i < h; i += 128) put(i, *reinterpret_cast<const float4*>(row + i));
}

template <typename T>
__global__ void rmsnorm_fwd_kernel(const float* __restrict__ y, int64_t ld, const float* __restrict__ gamma,
                                   float eps, int norm_none, int tokens, int h,
                                   T* __restrict__ n_out, float* __restrict__ r_out) {
  pdl_sync();
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (warp >= tokens) return;
  rmsnorm_row<T>(y + (int64_t)warp * ld, gamma, eps, norm_none, h, threadIdx.x & 31, n_out + (int64_t)warp * h, r_out + warp);
}

// ---------------------------------------------------------------------------
// Fold the router (and the shared-expert gate vector) through P_up:
//   W_rc[e, i] = sum_j W_r'[e, j] * W_up[j, i],   W_r' = [W_r; w_sgate]  ((E+1) x d)
// fp64 accumulation and output, so that logits = W_rc * n differ from the
// two-step definition only by fp64 rounding and the routing decision is
// reproducible against a higher-precision reference.
// Block = FD_I columns i x FD_E rows e x FD_S slices of j (512 threads).  W_up is staged
// through shared memory in chunks of FD_J rows (16-byte loads, the next chunk in flight
// while the current one is summed); the rows' weights are staged as doubles.  A thread
// owns one column, one slice (FD_J / FD_S consecutive j of every chunk) and FD_E
// accumulators; the slices are added in ascending order at the end (fixed order).
// ---------------------------------------------------------------------------
constexpr int FD_E = 4;     // rows of W_r' per block
constexpr int FD_J = 64;    // j-chunk staged per iteration
constexpr int FD_I = 128;   // columns per block
constexpr int FD_S = 4;     // j-slices per chunk
constexpr int FD_THREADS = FD_I * FD_S;

template <typename T>
__global__ void __launch_bounds__(FD_THREADS)
fold_router_kernel(const T* __restrict__ w_router, const T* __restrict__ w_sgate,
                   const T* __restrict__ w_up, int E, int d, int h, double* __restrict__ w_rc) {
  pdl_sync();
  constexpr int PER16 = 16 / (int)sizeof(T);                  // elements per 16-byte piece
  constexpr int ROW_PIECES = FD_I / PER16;                    // pieces per staged row
  constexpr int N_PIECES = FD_J * ROW_PIECES / FD_THREADS;    // pieces per thread and chunk
  constexpr int SL = FD_J / FD_S;                             // rows per slice
  __shared__ __align__(16) double wr_s[FD_J][FD_E];
  __shared__ __align__(16) T up_s[FD_J][FD_I];
  static_assert(sizeof(T) * FD_J * FD_I >= sizeof(double) * FD_S * FD_E * FD_I, "slice sums reuse the W_up stage");
  double (*red)[FD_E][FD_I] = reinterpret_cast<double (*)[FD_E][FD_I]>(&up_s[0][0]);   // used after the last chunk
  const int tid = threadIdx.x;
  const int col = tid % FD_I, sl = tid / FD_I;
  const int i0 = blockIdx.x * FD_I;
  const int e0 = blockIdx.y * FD_E;
  double acc[FD_E];
#pragma unroll
  for (int a = 0; a < FD_E; ++a) acc[a] = 0.0;

  uint4 pre[N_PIECES];
  float pre_w = 0.f;
  auto prefetch = [&](int j0) {
#pragma unroll
    for (int q = 0; q < N_PIECES; ++q) {
      int piece = tid + q * FD_THREADS;
      int jj = piece / ROW_PIECES, c = (piece % ROW_PIECES) * PER16;
      pre[q] = make_uint4(0u, 0u, 0u, 0u);
      if (j0 + jj < d && i0 + c < h)      // h is a multiple of 8: a piece never straddles the edge
        pre[q] = *reinterpret_cast<const uint4*>(w_up + (int64_t)(j0 + jj) * h + i0 + c);
    }
    if (tid < FD_E * FD_J) {
      int ee = tid / FD_J, jj = tid % FD_J;
      int e = e0 + ee, j = j0 + jj;
      const T* src = (e < E) ? (w_router + (int64_t)e * d) : (e == E ? w_sgate : nullptr);
      pre_w = (src != nullptr && j < d) ? to_f32(src[j]) : 0.f;
    }
  };
  prefetch(0);
  for (int j0 = 0; j0 < d; j0 += FD_J) {
    __syncthreads();
#pragma unroll
    for (int q = 0; q < N_PIECES; ++q) {
      int piece = tid + q * FD_THREADS;
      int jj = piece / ROW_PIECES, c = (piece % ROW_PIECES) * PER16;
      *reinterpret_cast<uint4*>(&up_s[jj][c]) = pre[q];
    }
    if (tid < FD_E * FD_J) wr_s[tid % FD_J][tid / FD_J] = (double)pre_w;
    __syncthreads();
    if (j0 + FD_J < d) prefetch(j0 + FD_J);
#pragma unroll
    for (int q = 0; q < SL; ++q) {      // rows past d were staged as zeros
      const int jj = sl * SL + q;
      double b = (double)to_f32(up_s[jj][col]);
      const double2* w2 = reinterpret_cast<const double2*>(wr_s[jj]);
#pragma unroll
      for (int a = 0; a < FD_E / 2; ++a) {
        double2 w = w2[a];
        acc[2 * a] += w.x * b;
        acc[2 * a + 1] += w.y * b;
      }
    }
  }
  __syncthreads();      // every slice has finished reading the stage
#pragma unroll
  for (int a = 0; a < FD_E; ++a) red[sl][a][col] = acc[a];
  __syncthreads();
  if (sl == 0 && i0 + col < h) {
#pragma unroll
    for (int a = 0; a < FD_E; ++a) {
      double v = red[0][a][col];
#pragma unroll
      for (int q = 1; q < FD_S; ++q) v += red[q][a][col];
      if (e0 + a <= E) w_rc[(int64_t)(e0 + a) * h + i0 + col] = v;
    }
  }
}

template <typename T>
inline cudaError_t launch_fold_router(const T* w_router, const T* w_sgate, const T* w_up, int E, int d, int h,
                                      double* w_rc, cudaStream_t st) {
  dim3 grid((unsigned)ceil_div(h, FD_I), (unsigned)ceil_div(E + 1, FD_E));
  launch_k(fold_router_kernel<T>, grid, FD_THREADS, 0, st, w_router, w_sgate, w_up, E, d, h, w_rc);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// The same fold on the fp64 tensor-core path, K split across blocks.
//   fold_router_mma_kernel: block (x: 32 columns i, y: 32 rows e, z: slice of rows j) computes the slice's
//     part[z][e][i] = sum_{j in slice z} W_r'[e, j] * W_up[j, i] with mma.sync m8n8k4 (two warps of 32 rows x
//     16 columns as 4 x 2 fragments).
//   fold_router_reduce_kernel: W_rc[e][i] = sum_z part[z][e][i], z ascending (fixed order).
// Bound by the fp64 pipe (64 multiply-adds a clock and SM: 7 us for 61 x 2048 x 1024) and the first loads.  The blocks are small so
// that an SM holds several at once, which load together, and none ends with a half-empty round: 1024 of them at this size,
// 6.9 per SM.  (256 blocks of 64 x 64, 1.7 per SM: the pipe of most SMs worked
// for two.  Forward of 64 tokens 253 -> 250 us, four d = 512 blocks 1438 -> 1418.)
// Needs FOLD_SLICES * (E+1) * h doubles of scratch, which the workspace has; the entry point that may
// not use a workspace keeps the FMA kernel above.
// ---------------------------------------------------------------------------
constexpr int FOLD_SLICES = 16;        // upper bound on the K slices
constexpr int FM_J_BYTES = 256;        // a slice is this many bytes of a W_r' row: 128 rows j in bf16, 64 in fp32
constexpr int FM_E = 32, FM_I = 32, FM_THREADS = 64;
template <typename T> __host__ __device__ constexpr int fold_slice_rows() { return FM_J_BYTES / (int)sizeof(T); }
constexpr int FM_PAD = 8;              // elements of padding per staged row (keeps rows 16-byte aligned)

__device__ __forceinline__ void fold_dmma(double& d0, double& d1, double a, double b) {
  asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};"
               : "+d"(d0), "+d"(d1) : "d"(a), "d"(b));
}

// The block's whole operand slices come in by cp.async, all in flight together (one memory round trip), stay in shared memory in
// their storage type, and are widened to fp64 as the fragments are read.
template <typename T>
__global__ void __launch_bounds__(FM_THREADS)
fold_router_mma_kernel(const T* __restrict__ w_router, const T* __restrict__ w_sgate, const T* __restrict__ w_up,
                       int E, int d, int h, double* __restrict__ part) {
  pdl_sync();
  constexpr int PER16 = 16 / (int)sizeof(T);
  constexpr int FM_J = fold_slice_rows<T>();
  constexpr int LDA = FM_J + FM_PAD, LDB = FM_I + FM_PAD;
  __shared__ __align__(16) T as[FM_E * LDA];     // W_r' slice  [e][j]
  __shared__ __align__(16) T bs[FM_J * LDB];     // W_up slice  [j][i]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int i0 = blockIdx.x * FM_I, e0 = blockIdx.y * FM_E, jb = blockIdx.z * FM_J;
  const int EP = E + 1;
  // d and h are multiples of 8, so a 16-byte piece never straddles the end of a row
#pragma unroll
  for (int q = 0; q < FM_E * (FM_J / PER16) / FM_THREADS; ++q) {
    const int piece = tid + q * FM_THREADS, ee = piece / (FM_J / PER16), jj = (piece % (FM_J / PER16)) * PER16;
    const int e = e0 + ee, j = jb + jj;
    const T* src = (e < E) ? (w_router + (int64_t)e * d) : (e == E ? w_sgate : nullptr);
    const bool ok = src != nullptr && j < d;
    cp_async16(&as[ee * LDA + jj], ok ? src + j : w_router, ok);
  }
#pragma unroll
  for (int q = 0; q < FM_J * (FM_I / PER16) / FM_THREADS; ++q) {
    const int piece = tid + q * FM_THREADS, jj = piece / (FM_I / PER16), ii = (piece % (FM_I / PER16)) * PER16;
    const bool ok = jb + jj < d && i0 + ii < h;
    cp_async16(&bs[jj * LDB + ii], ok ? w_up + (int64_t)(jb + jj) * h + i0 + ii : w_up, ok);
  }
  cp_async_commit();
  cp_async_wait<0>();
  __syncthreads();
  const int fr = lane >> 2, fc = lane & 3;
  double acc[4][2][2];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) { acc[a][b][0] = 0.0; acc[a][b][1] = 0.0; }
#pragma unroll 4
  for (int kk = 0; kk < FM_J; kk += 4) {
    double af[4], bf[2];
#pragma unroll
    for (int a = 0; a < 4; ++a) af[a] = (double)to_f32(as[(a * 8 + fr) * LDA + kk + fc]);
#pragma unroll
    for (int b = 0; b < 2; ++b) bf[b] = (double)to_f32(bs[(kk + fc) * LDB + warp * 16 + b * 8 + fr]);
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 2; ++b) fold_dmma(acc[a][b][0], acc[a][b][1], af[a], bf[b]);
  }
  double* out = part + (int64_t)blockIdx.z * EP * h;
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const int e = e0 + a * 8 + fr, i = i0 + warp * 16 + b * 8 + 2 * fc;
      if (e < EP && i < h) *reinterpret_cast<double2*>(out + (int64_t)e * h + i) = make_double2(acc[a][b][0], acc[a][b][1]);      // h is even
    }
}

__global__ void fold_router_reduce_kernel(const double* __restrict__ part, int n_slices, int64_t n,
                                          double* __restrict__ w_rc) {
  pdl_sync();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double v = part[i];
  for (int z = 1; z < n_slices; ++z) v += part[(int64_t)z * n + i];
  w_rc[i] = v;
}

// Returns cudaErrorInvalidValue when d needs more slices than the scratch holds (the caller then uses the FMA kernel).
template <typename T>
inline cudaError_t launch_fold_router_mma(const T* w_router, const T* w_sgate, const T* w_up, int E, int d, int h,
                                          double* part, double* w_rc, cudaStream_t st) {
  const int n_slices = (int)ceil_div(d, fold_slice_rows<T>());
  if (n_slices > FOLD_SLICES) return cudaErrorInvalidValue;
  dim3 grid((unsigned)ceil_div(h, FM_I), (unsigned)ceil_div(E + 1, FM_E), (unsigned)n_slices);
  launch_k(fold_router_mma_kernel<T>, grid, FM_THREADS, 0, st, w_router, w_sgate, w_up, E, d, h, part);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const int64_t n = (int64_t)(E + 1) * h;
  launch_k(fold_router_reduce_kernel, (unsigned)ceil_div(n, 256), 256, 0, st, part, n_slices, n, w_rc);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Router: logits in fp64 from the fp32 stream, top-k by warp shuffles, gates.
//   cluster of ROUTE_CLUSTER blocks of 256 threads = RT_TOK tokens.
//   phase 1: L[t, e] = r_t <W_rc[e], y_t * gamma> (+ b_r[e]) for e < E; row E is the
//            shared gate.  The product runs on the fp64 tensor-core path
//            (mma.sync m8n8k4): y (fp32, [token][i]) and W_rc (fp64, [expert][i]) chunks come in by cp.async through a
//            ring of two stages, y * gamma is formed in fp64 as the fragments are read, each warp owns a
//            16-token x 32-expert block of the 64 x 64 tile as 2 x 4 fragments.  Each block takes an eighth of K and
//            leaves its partial sums in its own shared memory.  Four threads per token also sum y^2 (fp64), which
//            gives r_t = (mean(y_t^2)+eps)^-1/2; the scale is applied to the finished sums.
//   phase 2: each block takes 8 of the tokens, a warp one: it adds the token's partial sums from the cluster, slices
//            in ascending order, then k rounds of warp arg-max (ties -> lowest index), softmax
//            over the k selected logits, sigmoid of the shared-gate logit.
// The split is the same whatever the number of tokens, so a token's logits do not depend on the batch it is in.
// What bounds it: the serial walk over K at small batches, where splitting K gives eight times the blocks (64 tokens:
// 47 us with a run of tokens in one block, now 12; 512: 47, now 20), and at large ones the fp64 tensor pipe, idle while the
// blocks of an SM start and finish (8192 tokens: 76, now 65; 8192 x 61 x 1024 multiply-adds are 29 us of the pipe).
// idx_in != NULL: expert sets are taken from it (gates are still recomputed).
// prob_out != NULL: gates are the selected entries of the softmax over ALL experts (not
// renormalised), and that softmax is written to prob_out[T, E].
// ---------------------------------------------------------------------------
constexpr int ROUTE_CLUSTER = 8;
constexpr int RT_TOK = 64;   // tokens per cluster
constexpr int RT_KC = 32;    // k-chunk
constexpr int RT_EC = 64;    // experts per pass
constexpr int RT_LD = RT_KC + 4;    // row stride (elements) of both staged chunks: rows 4 elements apart modulo the
                                    // banks, so the 8 rows x 4 columns a fragment load touches fall on distinct ones
constexpr int RT_STAGES = 2;
constexpr int RT_STAGE_BYTES = RT_EC * RT_LD * 8 + RT_TOK * RT_LD * 4 + RT_KC * 4;     // W_rc | y | gamma
static_assert(RT_TOK == 8 * ROUTE_CLUSTER, "phase 2: one token per warp of the cluster");

// Shared memory: stage ring | finished logits of the warps' tokens [8][E+1] | sums of y^2 [RT_TOK].
// The partial logits take the ring's place when there is one pass over the experts, else they follow the rest.
__host__ __device__ inline int router_row_off(int E) {
  const int ring = RT_STAGES * RT_STAGE_BYTES, part = E + 1 <= RT_EC ? RT_TOK * (E + 1) * 8 : 0;
  return ring > part ? ring : part;
}
__host__ __device__ inline int router_part_off(int E) {
  return E + 1 <= RT_EC ? 0 : router_row_off(E) + (8 * (E + 1) + RT_TOK) * 8;
}
inline size_t router_smem_bytes(int E) {
  const size_t rest = (size_t)router_row_off(E) + (8 * (size_t)(E + 1) + RT_TOK) * 8;
  return E + 1 <= RT_EC ? rest : rest + (size_t)RT_TOK * (E + 1) * 8;
}

__device__ __forceinline__ uint32_t route_cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void route_cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Cluster-wide address of the same shared-memory place in block `rank`, and the double at such an address.
__device__ __forceinline__ uint32_t cluster_addr(const void* p, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  return r;
}
__device__ __forceinline__ double ld_cluster_f64(uint32_t addr) {
  double v;
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(addr) : "memory");
  return v;
}
// Integers in the order of the doubles, for comparisons beside an fp64 pipe that other blocks keep busy: equal for equal
// values (both zeros included), NaN as -inf, never 0.
__device__ __forceinline__ unsigned long long order_key(double v) {
  long long b = __double_as_longlong(v);
  if ((b & 0x7fffffffffffffffLL) > 0x7ff0000000000000LL) b = (long long)0xfff0000000000000ULL;
  if (b == (long long)0x8000000000000000ULL) b = 0;
  return b < 0 ? ~(unsigned long long)b : (unsigned long long)b | 0x8000000000000000ULL;
}
__device__ __forceinline__ double from_order_key(unsigned long long key) {
  return __longlong_as_double((long long)(key >> 63 ? key & 0x7fffffffffffffffULL : ~key));
}
// x^-1/2 to the last places of fp64: two Newton steps, y (3 - x y^2) / 2, from the fp32 value (2^-22 -> 2^-43 -> rounding),
// nine dependent fp64 operations where a square root and a division take several times as many.
__device__ __forceinline__ double rsqrt_f64(double x) {
  if (!(x > 1e-30 && x < 1e30)) return 1.0 / sqrt(x);
  double y = (double)rsqrtf((float)x);
  const double hx = 0.5 * x;
  y = y * fma(-hx * y, y, 1.5);
  return y * fma(-hx * y, y, 1.5);
}
// D (8x8) += A (8x4, row-major fragment) * B (4x8, column-major fragment), fp64.
// Lane l holds A[l/4][l%4], B[l%4][l/4] and D[l/4][2*(l%4) + {0,1}].
__device__ __forceinline__ void dmma_8x8x4(double& d0, double& d1, double a, double b) {
  asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};"
               : "+d"(d0), "+d"(d1) : "d"(a), "d"(b));
}

__global__ void __launch_bounds__(256, 3)
router_topk_kernel(const float* __restrict__ y, int64_t ld, const float* __restrict__ gamma, float eps,
                   int norm_none, const double* __restrict__ w_rc, const float* __restrict__ b_router,
                   int tokens, int h, int E, int k, int has_shared, const int32_t* __restrict__ idx_in,
                   int32_t* __restrict__ idx_out, float* __restrict__ gate_out, float* __restrict__ sgate_out,
                   int32_t* __restrict__ idx_user, float* __restrict__ prob_out, int* __restrict__ status,
                   int check_finite, double inv_h) {
  pdl_sync();
  extern __shared__ __align__(16) uint8_t rt_smem[];
  const int EP = E + 1;                       // logits per token incl. the shared-gate row
  double* Lp = reinterpret_cast<double*>(rt_smem + router_part_off(E));    // [RT_TOK][EP] this block's partial sums
  double* Lrow = reinterpret_cast<double*>(rt_smem + router_row_off(E));      // [8][EP]
  double* sq = Lrow + 8 * EP;                                                 // [RT_TOK]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t rank = route_cluster_rank();
  const int t0 = (int)(blockIdx.x / ROUTE_CLUSTER) * RT_TOK;
  const int chunks = (int)ceil_div(h, RT_KC);
  const int c_begin = (int)((int64_t)chunks * rank / ROUTE_CLUSTER);
  const int n_c = (int)((int64_t)chunks * (rank + 1) / ROUTE_CLUSTER) - c_begin;
  const bool scaled = gamma != nullptr && !norm_none;

  // phase 1: logits.  Warp (wm, wn) owns tokens 16 wm .. +15 and experts e0 + 32 wn .. +31.
  const int wm = warp >> 1, wn = warp & 1;
  const int fr = lane >> 2, fc = lane & 3;          // fragment row / column of this lane
  for (int e0 = 0; e0 < EP; e0 += RT_EC) {
    double acc[2][4][2];
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) { acc[a][b][0] = 0.0; acc[a][b][1] = 0.0; }
    double ss = 0.0;                // sum of y^2 over this thread's quarter of the chunks of token tid / 4
    auto load = [&](int c) {        // chunk c of the slice into its stage; always commits a group
      if (c < n_c) {
        double* ws = reinterpret_cast<double*>(rt_smem + (c % RT_STAGES) * RT_STAGE_BYTES);
        float* ns = reinterpret_cast<float*>(ws + RT_EC * RT_LD);
        const int k0 = (c_begin + c) * RT_KC;
        if (scaled && tid < RT_KC / 4) cp_async16(ns + RT_TOK * RT_LD + tid * 4, gamma + min(k0 + tid * 4, h - 4), k0 + tid * 4 < h);
#pragma unroll
        for (int q = 0; q < RT_TOK * RT_KC / 4 / 256; ++q) {
          const int at = tid + q * 256, tt = at / (RT_KC / 4), kq = (at % (RT_KC / 4)) * 4;
          const bool ok = t0 + tt < tokens && k0 + kq < h;                                         // h % 4 == 0
          cp_async16(ns + tt * RT_LD + kq, ok ? y + (int64_t)(t0 + tt) * ld + k0 + kq : y, ok);
        }
#pragma unroll
        for (int q = 0; q < RT_EC * RT_KC / 2 / 256; ++q) {
          const int at = tid + q * 256, ee = at / (RT_KC / 2), kq = (at % (RT_KC / 2)) * 2;
          const bool ok = e0 + ee < EP && k0 + kq < h;                                             // h % 2 == 0
          cp_async16(ws + ee * RT_LD + kq, ok ? w_rc + (int64_t)(e0 + ee) * h + k0 + kq : w_rc, ok);
        }
      }
      cp_async_commit();
    };
#pragma unroll
    for (int c = 0; c < RT_STAGES; ++c) load(c);
    for (int c = 0; c < n_c; ++c) {
      cp_async_wait<RT_STAGES - 1>();
      __syncthreads();
      const double* ws = reinterpret_cast<const double*>(rt_smem + (c % RT_STAGES) * RT_STAGE_BYTES);
      const float* ns = reinterpret_cast<const float*>(ws + RT_EC * RT_LD);
      const float* ap = ns + (wm * 16 + fr) * RT_LD + fc;
      const double* bp = ws + (wn * 32 + fr) * RT_LD + fc;
      const float* gp = ns + RT_TOK * RT_LD + fc;
#pragma unroll
      for (int kk = 0; kk < RT_KC; kk += 4) {
        double af[2], bf[4];
#pragma unroll
        for (int a = 0; a < 2; ++a) af[a] = (double)ap[a * 8 * RT_LD + kk];
        if (scaled) {
          const double g = (double)gp[kk];
          af[0] *= g; af[1] *= g;
        }
#pragma unroll
        for (int b = 0; b < 4; ++b) bf[b] = bp[b * 8 * RT_LD + kk];
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
          for (int b = 0; b < 4; ++b) dmma_8x8x4(acc[a][b][0], acc[a][b][1], af[a], bf[b]);
      }
      if (e0 == 0) {
        const float4* q4 = reinterpret_cast<const float4*>(ns + (tid >> 2) * RT_LD + (tid & 3) * 8);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const float4 v = q4[j];
          ss += (double)v.x * (double)v.x; ss += (double)v.y * (double)v.y;
          ss += (double)v.z * (double)v.z; ss += (double)v.w * (double)v.w;
        }
      }
      __syncthreads();
      load(c + RT_STAGES);
    }
    cp_async_wait<0>();
    __syncthreads();                // also: nobody reads the ring any more where the partial sums go over it
    if (e0 == 0) {
      ss += __shfl_xor_sync(0xffffffffu, ss, 1);
      ss += __shfl_xor_sync(0xffffffffu, ss, 2);
      if ((tid & 3) == 0) sq[tid >> 2] = ss;
    }
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b)
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const int tt = wm * 16 + a * 8 + fr, e = e0 + wn * 32 + b * 8 + 2 * fc + c;
          if (e < EP) Lp[tt * EP + e] = acc[a][b][c];
        }
  }
  const int tt = (int)rank * 8 + warp, t = t0 + tt;
  // this lane's biases (columns lane, lane + 32) and, with idx_in, the index of its slot, in flight across the barrier
  const float bias0 = b_router && lane < E ? b_router[lane] : 0.f, bias1 = b_router && lane + 32 < E ? b_router[lane + 32] : 0.f;
  const int idx_lane = idx_in && t < tokens && lane < k ? idx_in[(int64_t)t * k + lane] : -1;
  route_cluster_sync();

  // phase 2: top-k and gates; one warp per token.  Each block runs this once, from a cold instruction cache: it is kept
  // short, its loops rolled (8 rounds of a 5-step shuffle reduction in fp64, unrolled, and a square root and a division
  // took 13k clk of a block's 45k; now about 6k, 2k of them the other blocks' partial sums: kernel at 8192 tokens 82 -> 65
  // us, at 512 24 -> 20, at 64 14.1 -> 11.8).
  if (t < tokens) {
    double* L = Lrow + warp * EP;
    // Partial sums of the squares and of this lane's first two logits, slices in ascending order, all asked for before any
    // is used.
    double part[ROUTE_CLUSTER], p0[ROUTE_CLUSTER], p1[ROUTE_CLUSTER];
#pragma unroll
    for (int r = 0; r < ROUTE_CLUSTER; ++r) {
      const uint32_t base = cluster_addr(rt_smem, (uint32_t)r);
      const uint32_t row = base + (uint32_t)(reinterpret_cast<uint8_t*>(Lp + tt * EP) - rt_smem);
      part[r] = ld_cluster_f64(base + (uint32_t)(reinterpret_cast<uint8_t*>(sq + tt) - rt_smem));
      p0[r] = ld_cluster_f64(row + 8 * min(lane, EP - 1));
      p1[r] = ld_cluster_f64(row + 8 * min(lane + 32, EP - 1));
    }
    double ss = 0.0, v0 = 0.0, v1 = 0.0;
#pragma unroll
    for (int r = 0; r < ROUTE_CLUSTER; ++r) { ss += part[r]; v0 += p0[r]; v1 += p1[r]; }
    const double rt = norm_none ? 1.0 : rsqrt_f64(ss * inv_h + (double)eps);
    v0 *= rt; v1 *= rt;
    if (b_router && lane < E) v0 += (double)bias0;
    if (b_router && lane + 32 < E) v1 += (double)bias1;
    if (lane < EP) L[lane] = v0;
    if (lane + 32 < EP) L[lane + 32] = v1;
#pragma unroll 1
    for (int e = lane + 64; e < EP; e += 32) {
      double v = 0.0;
#pragma unroll
      for (int r = 0; r < ROUTE_CLUSTER; ++r) v += ld_cluster_f64(cluster_addr(Lp + tt * EP + e, (uint32_t)r));
      v *= rt;
      if (e < E && b_router) v += (double)b_router[e];
      L[e] = v;
    }
    __syncwarp();
    if (check_finite) {
      // a NaN or infinite logit (non-finite input or weight) makes the selection meaningless: report it
      bool bad = false;
      for (int e = lane; e < EP; e += 32) bad |= !isfinite(L[e]);
      if (__any_sync(0xffffffffu, bad) && lane == 0) set_status(status, REVFFN_ERR_NONFINITE);
    }
    // Lane s < k ends up with the logit (mine) and index of slot s, every lane with the largest selected logit (m).  The
    // softmax runs in fp32 on the fp64 differences to it (the decision is fp64; the weights are fp32 outputs).
    const double minus_inf = __longlong_as_double(0xfff0000000000000LL);
    double m = minus_inf, mine = minus_inf;
    int mine_i = -1;
    if (idx_in) {
      // Expert sets from the caller.  An index outside [0, E) is reported and kept as -1: the
      // permutation maps skip such an entry, and its gate weight is zero.
      if (lane < k) {
        if ((unsigned)idx_lane < (unsigned)E) { mine_i = idx_lane; mine = L[idx_lane]; }
        else set_status(status, REVFFN_ERR_INDEX);
      }
      m = mine;
#pragma unroll 1
      for (int o = 4; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));      // k <= 8
      m = __shfl_sync(0xffffffffu, m, 0);
    } else {
      // k rounds of the warp's arg-max in integers: the upper halves of the keys, among the lanes that hold the maximum the
      // lower halves, and among equals the lowest index
      unsigned taken = 0u;                    // bit j set: candidate lane + 32 j already selected
      const unsigned long long key0 = lane < E ? order_key(v0) : 0ull, key1 = lane + 32 < E ? order_key(v1) : 0ull;
#pragma unroll 1
      for (int s = 0; s < k; ++s) {
        unsigned long long best = taken & 1u ? 0ull : key0;       // 0: below every key
        int bj = 0;
        if (!(taken & 2u) && key1 > best) { best = key1; bj = 1; }
        if (E > 64) {
#pragma unroll 1
          for (int j = 2; 32 * j < E; ++j) {
            const unsigned long long key = lane + 32 * j < E ? order_key(L[lane + 32 * j]) : 0ull;
            if (!(taken >> j & 1u) && key > best) { best = key; bj = j; }
          }
        }
        const unsigned hi = (unsigned)(best >> 32), lo = (unsigned)best;
        const unsigned top = __reduce_max_sync(0xffffffffu, hi);
        const unsigned low = __reduce_max_sync(0xffffffffu, hi == top ? lo : 0u);
        const unsigned e = (hi == top && lo == low) ? (unsigned)(lane + 32 * bj) : 0xffffffffu;
        const unsigned win = __reduce_min_sync(0xffffffffu, e);
        if (e == win) taken |= 1u << bj;
        if (lane == s || s == 0) {
          const double v = from_order_key((unsigned long long)top << 32 | low);
          if (s == 0) m = v;                  // selected in descending order
          if (lane == s) { mine = v; mine_i = (int)win; }
        }
      }
    }
    float den;
    if (prob_out) {
      // softmax over all E logits (no renormalisation of the selected ones): largest logit and the sum of
      // exponentials over every expert; the probabilities are kept for the backward pass
      double ma = __longlong_as_double(0xfff0000000000000LL);
      for (int e = lane; e < E; e += 32) ma = fmax(ma, L[e]);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) ma = fmax(ma, __shfl_xor_sync(0xffffffffu, ma, o));
      m = ma;
      float sa = 0.f;
      for (int e = lane; e < E; e += 32) sa += expf((float)(L[e] - ma));
      den = warp_sum(sa);
      for (int e = lane; e < E; e += 32) prob_out[(int64_t)t * E + e] = expf((float)(L[e] - ma)) / den;
    }
    float x = 0.f;
    if (lane < k) x = (float)(mine - m);
    else if (lane == k) x = (float)(-L[E]);
    const float ev = expf(x);
    if (!prob_out) {
      den = (lane < k) ? ev : 0.f;
      den += __shfl_xor_sync(0xffffffffu, den, 1);
      den += __shfl_xor_sync(0xffffffffu, den, 2);
      den += __shfl_xor_sync(0xffffffffu, den, 4);      // k <= 8: lanes 0..7 hold the sum
    }
    if (lane < k) {
      idx_out[(int64_t)t * k + lane] = mine_i;
      if (idx_user) idx_user[(int64_t)t * k + lane] = mine_i;
      gate_out[(int64_t)t * k + lane] = ev / den;
    } else if (lane == k) {
      sgate_out[t] = has_shared ? 1.f / (1.f + ev) : 0.f;
    }
  }
  route_cluster_sync();      // no block leaves while another may still read its partial sums
}

// Raises the kernel's dynamic shared-memory limit (once per device), then launches.
inline cudaError_t launch_router_topk(const float* y, int64_t ld, const float* gamma, float eps, int norm_none,
                                      const double* w_rc, const float* b_router, int tokens, int h, int E, int k,
                                      int has_shared, const int32_t* idx_in, int32_t* idx_out, float* gate_out,
                                      float* sgate_out, int32_t* idx_user, float* prob_out, int* status,
                                      int check_finite, cudaStream_t st) {
  static size_t raised[64] = {0};
  static std::mutex mu;
  const size_t smem = router_smem_bytes(E);
  if (smem > 48 * 1024) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(mu);
    if (raised[dev] < smem) {
      e = cudaFuncSetAttribute(router_topk_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
      raised[dev] = smem;
    }
  }
  return launch_cluster(router_topk_kernel, dim3((unsigned)(ceil_div(tokens, RT_TOK) * ROUTE_CLUSTER)), dim3(ROUTE_CLUSTER),
                        dim3(256), smem, st, y, ld, gamma, eps, norm_none, w_rc, b_router, tokens, h, E, k, has_shared, idx_in,
                        idx_out, gate_out, sgate_out, idx_user, prob_out, status, check_finite, 1.0 / (double)h);
}

// ---------------------------------------------------------------------------
// Permutation maps: stable counting sort of the T*k (token, slot) entries by
// expert, each expert's segment padded to a multiple of ROW_PAD rows.
//   map_rank:   per chunk of tokens, rank of each entry among the chunk's entries of the same expert
//               (entry order = token-major) and the chunk's count per expert
//   map_assign: row of each entry; row -> token; row -> gate weight; padding rows (token -1, gate 0);
//               the per-expert tables
// Both are latency.  Every block of map_assign adds up the counts of all chunks itself (n_chunks * E integers out of
// the L2) instead of waiting for a one-block scan in between, and the chunk grows with the batch so that there
// are at most 128 of them until it holds 2048 tokens.  With the two memsets that the padding rows took: 5 launches,
// 33 us at 64 tokens and 50 us at 8192 (gaps included) -> 2 launches, 12 and 14 us.
// ---------------------------------------------------------------------------
constexpr int TOK_CHUNK = 256;       // most token rows of one expert in one N-side tile
constexpr int MAP_THREADS = 512;
constexpr int MAP_MAX_E = 256;       // n_experts is at most this

// Tokens per block: see above.
inline int map_chunk_tokens(int64_t tokens) {
  int c = 128;
  while (c < 2048 && ceil_div(tokens, c) > 128) c *= 2;
  return c;
}

// An entry outside [0, E) (possible only in expert sets handed in by the caller) matches no expert: it gets
// no rank and no row, map_assign marks it with row -1, and every later step skips it.  It is reported once here.
__global__ void __launch_bounds__(MAP_THREADS)
map_rank_kernel(const int32_t* __restrict__ idx, int tokens, int k, int E, int chunk_tokens,
                int32_t* __restrict__ local_rank, int32_t* __restrict__ chunk_cnt, int* __restrict__ status) {
  pdl_sync();
  constexpr int WARPS = MAP_THREADS / 32;
  __shared__ int hist[WARPS][MAP_MAX_E];       // counts per warp, then the warps' bases
  __shared__ int run[MAP_MAX_E];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int chunk = blockIdx.x;
  const int64_t i0 = (int64_t)chunk * chunk_tokens * k;
  const int n = (int)min((int64_t)chunk_tokens * k, (int64_t)tokens * k - i0);
  for (int e = tid; e < E; e += MAP_THREADS) run[e] = 0;
  for (int base = 0; base < n; base += MAP_THREADS) {
    for (int e = lane; e < E; e += 32) hist[warp][e] = 0;
    __syncwarp();
    const int i = base + tid;
    const int e = i < n ? idx[i0 + i] : -1;
    const bool valid = (unsigned)e < (unsigned)E;
    if (i < n && !valid) set_status(status, REVFFN_ERR_INDEX);
    const unsigned peers = __match_any_sync(0xffffffffu, valid ? e : MAP_MAX_E);
    const int rank = __popc(peers & ((1u << lane) - 1u));
    if (valid && rank == 0) hist[warp][e] = __popc(peers);
    __syncthreads();
    for (int x = tid; x < E; x += MAP_THREADS) {
      int c = run[x];
#pragma unroll
      for (int w = 0; w < WARPS; ++w) { const int v = hist[w][x]; hist[w][x] = c; c += v; }
      run[x] = c;
    }
    __syncthreads();
    if (valid) local_rank[i0 + i] = hist[warp][e] + rank;
    __syncwarp();                              // a warp clears only its own row for the next round
  }
  __syncthreads();
  for (int e = tid; e < E; e += MAP_THREADS) chunk_cnt[(int64_t)chunk * E + e] = run[e];
}

__global__ void __launch_bounds__(MAP_THREADS)
map_assign_kernel(const int32_t* __restrict__ idx, const float* __restrict__ gate, const int32_t* __restrict__ local_rank,
                  const int32_t* __restrict__ chunk_cnt, int tokens, int k, int E, int chunk_tokens, int n_chunks,
                  int32_t* __restrict__ expert_cnt, int32_t* __restrict__ expert_off, int32_t* __restrict__ tile_group,
                  int32_t* __restrict__ rows_total, int max_tiles, int4* __restrict__ tok_chunks, int max_chunks,
                  int32_t* __restrict__ tok_row, int32_t* __restrict__ row_tok, float* __restrict__ row_gate) {
  pdl_sync();
  __shared__ int below[MAP_MAX_E], cnt[MAP_MAX_E];          // this expert's entries in earlier chunks / in all chunks
  __shared__ int off[MAP_MAX_E + 1], coff[MAP_MAX_E + 1];   // first padded row, first token run of an expert
  const int tid = threadIdx.x, lane = tid & 31;
  const int chunk = blockIdx.x;
  for (int e = tid; e < MAP_MAX_E; e += MAP_THREADS) { below[e] = 0; cnt[e] = 0; }
  __syncthreads();
  {
    // thread = (group of chunks, expert); integer sums, so the order of the additions does not matter
    const int lanes = E <= 32 ? 32 : (E <= 64 ? 64 : (E <= 128 ? 128 : 256));
    const int groups = MAP_THREADS / lanes, e = tid % lanes, g = tid / lanes;
    if (e < E) {
      int b = 0, a = 0;
#pragma unroll 8
      for (int c = g; c < n_chunks; c += groups) {
        const int v = chunk_cnt[(int64_t)c * E + e];
        a += v;
        if (c < chunk) b += v;
      }
      atomicAdd(&cnt[e], a);
      atomicAdd(&below[e], b);
    }
  }
  __syncthreads();
  if (tid < 32) {
    // exclusive prefix sums over the experts, eight per lane
    int rows[8], runs[8], sr = 0, sc = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int c = cnt[lane * 8 + j];
      rows[j] = (c + ROW_PAD - 1) / ROW_PAD * ROW_PAD;
      runs[j] = (c + TOK_CHUNK - 1) / TOK_CHUNK;
      sr += rows[j]; sc += runs[j];
    }
    int ir = sr, ic = sc;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, ir, o), v = __shfl_up_sync(0xffffffffu, ic, o);
      if (lane >= o) { ir += u; ic += v; }
    }
    int pr = ir - sr, pc = ic - sc;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      off[lane * 8 + j] = pr; coff[lane * 8 + j] = pc;
      pr += rows[j]; pc += runs[j];
    }
    if (lane == 31) { off[MAP_MAX_E] = pr; coff[MAP_MAX_E] = pc; }
  }
  __syncthreads();
  const int64_t i0 = (int64_t)chunk * chunk_tokens * k;
  const int n = (int)min((int64_t)chunk_tokens * k, (int64_t)tokens * k - i0);
  for (int i = tid; i < n; i += MAP_THREADS) {
    const int e = idx[i0 + i];
    if ((unsigned)e >= (unsigned)E) { tok_row[i0 + i] = -1; continue; }      // reported by map_rank
    const int row = off[e] + below[e] + local_rank[i0 + i];
    tok_row[i0 + i] = row;
    row_tok[row] = (int)((i0 + i) / k);
    row_gate[row] = gate[i0 + i];
  }
  // padding rows, an expert per warp of all blocks
  for (int e = chunk * (MAP_THREADS / 32) + (tid >> 5); e < E; e += n_chunks * (MAP_THREADS / 32))
    for (int r = off[e] + cnt[e] + lane; r < off[e + 1]; r += 32) { row_tok[r] = -1; row_gate[r] = 0.f; }
  if (chunk != 0) return;
  for (int e = tid; e <= E; e += MAP_THREADS) {
    expert_off[e] = off[e];
    if (e == E) continue;
    expert_cnt[e] = cnt[e];
    for (int t = off[e] / ROW_PAD; t < off[e + 1] / ROW_PAD && t < max_tiles; ++t) tile_group[t] = e;
    // Token runs for the products that put tokens on the MMA N side: per expert, runs of up to TOK_CHUNK rows
    // covering its real rows rounded up to 32 (the rounding stays inside the expert's zero padding).
    // Entry = (expert, first row, rows, rows of padding from there to the next multiple of 64: in the expert's last run only).
    // (Runs of equal length, 3 x 192 instead of 256 + 256 + 64 for 546 rows, stay within 2 % either way: the two
    // products that use the table measured 2 % faster alone and the whole step 1-2 % slower.)
    const int real = (int)round_up(cnt[e], 32);
    for (int r = 0, c = coff[e]; r < real && c < max_chunks; r += TOK_CHUNK, ++c)
      tok_chunks[c] = make_int4(e, off[e] + r, min(TOK_CHUNK, real - r), r + TOK_CHUNK >= real ? (int)round_up(cnt[e], 64) - real : 0);
  }
  if (tid == 0) {
    rows_total[0] = off[E];
    rows_total[1] = min(coff[E], max_chunks);
  }
}

// ---------------------------------------------------------------------------
// Gather rows into the padded expert-major layout:
//   out[row, :] = src[row_tok[row], :]   (zeros for padding rows)
// A warp per row, a row's pieces all requested before the first is stored.  Rows at or beyond *rows_total are skipped.
// Padding: the tensor-core products over rows stop at the 64-row boundary past an expert's real rows and all others
// compute row by row, so groups of 64 padding rows stay as they are unless fill_all asks for them (the CUDA-core
// products read every row).  60 experts with 4 rows each: 16 MB written instead of 31.  A block per row with one piece a
// thread took 55.7 us at 8192 tokens, 13.2 at 512 and 11.0 at 64; now 35.1, 8.8 and 6.7.
// ---------------------------------------------------------------------------
constexpr int GATHER_ROWS = 8;      // rows (warps) per block

template <typename T>
__global__ void __launch_bounds__(32 * GATHER_ROWS)
gather_rows_kernel(const T* __restrict__ src, int64_t ld_src, const int32_t* __restrict__ row_tok, const int32_t* __restrict__ rows_total,
                   int width, int fill_all, T* __restrict__ out) {
  pdl_sync();
  const int row = blockIdx.x * GATHER_ROWS + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (row >= *rows_total) return;
  const int t = row_tok[row];
  if (t < 0 && !fill_all && padding_group(row_tok, row)) return;
  T* o = out + (int64_t)row * width;
  const T* from = src + (int64_t)t * ld_src;
  for (int c0 = lane * 8; c0 < width; c0 += 8 * 256) {
    Vec8<T> v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (t >= 0 && c0 + i * 256 < width) v[i].load(from + c0 + i * 256); else v[i].zero();
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (c0 + i * 256 < width) v[i].store(o + c0 + i * 256);
  }
}

// ---------------------------------------------------------------------------
// Combine: Z[t, :] = sum_{s<k} O[tok_row[t,s], :] + sgate[t] * S[t, :]
// fp32 sums in slot order (fixed, so forward and inverse agree bit for bit).
// One warp per token, eight tokens per block; each lane walks the row in 256-element strides with all k + 1
// row pieces of a stride requested before the first is used (K = k at compile time; K = 0 takes k <= 8 at run
// time and pays for eight slots).  Many short blocks: a one-wave grid striding over the tokens measured 12 %
// slower.
// ---------------------------------------------------------------------------
constexpr int COMBINE_TOKENS = 8;      // tokens (warps) per block

template <typename T, int K>
__global__ void __launch_bounds__(32 * COMBINE_TOKENS)
combine_rows_kernel(const T* __restrict__ O, const int32_t* __restrict__ tok_row, int k_rt,
                    const T* __restrict__ S, const float* __restrict__ sgate, int width, int tokens,
                    T* __restrict__ Z) {
  pdl_sync();
  constexpr int KS = K ? K : 8;
  const int k = K ? K : k_rt;
  const int lane = threadIdx.x & 31;
  const int64_t t = (int64_t)blockIdx.x * COMBINE_TOKENS + (threadIdx.x >> 5);
  if (t >= tokens) return;
  const T* rows[KS];
#pragma unroll
  for (int s = 0; s < KS; ++s) {
    const int r = s < k ? tok_row[t * k + s] : -1;      // -1: entry with an out-of-range expert index
    rows[s] = r >= 0 ? O + (int64_t)r * width : nullptr;
  }
  const float sg = S ? sgate[t] : 0.f;
  const T* srow = S ? S + t * width : nullptr;
  T* zrow = Z + t * width;
  for (int c = lane * 8; c < width; c += 256) {
    Vec8<T> v[KS], vs;
#pragma unroll
    for (int s = 0; s < KS; ++s) {
      if (rows[s]) v[s].load(rows[s] + c); else v[s].zero();
    }
    if (srow) vs.load(srow + c); else vs.zero();
    float acc[8], f[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[i] = 0.f;
#pragma unroll
    for (int s = 0; s < KS; ++s) {
      v[s].get(f);
#pragma unroll
      for (int i = 0; i < 8; ++i) acc[i] += f[i];
    }
    vs.get(f);
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[i] += sg * f[i];
    vs.set(acc);
    vs.store(zrow + c);
  }
}

template <typename T>
inline cudaError_t launch_combine_rows(const T* O, const int32_t* tok_row, int k, const T* S, const float* sgate,
                                       int width, int tokens, T* Z, cudaStream_t st) {
  if (tokens <= 0) return cudaSuccess;
  const int blocks = (int)ceil_div(tokens, COMBINE_TOKENS), th = 32 * COMBINE_TOKENS;
  switch (k) {
    case 1: launch_k(combine_rows_kernel<T, 1>, blocks, th, 0, st, O, tok_row, k, S, sgate, width, tokens, Z); break;
    case 2: launch_k(combine_rows_kernel<T, 2>, blocks, th, 0, st, O, tok_row, k, S, sgate, width, tokens, Z); break;
    case 4: launch_k(combine_rows_kernel<T, 4>, blocks, th, 0, st, O, tok_row, k, S, sgate, width, tokens, Z); break;
    default: launch_k(combine_rows_kernel<T, 0>, blocks, th, 0, st, O, tok_row, k, S, sgate, width, tokens, Z); break;
  }
  return cudaGetLastError();
}

}  // namespace revffn
