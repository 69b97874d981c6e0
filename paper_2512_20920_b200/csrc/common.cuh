// Shared small helpers for the RevFFN MoE kernels (sm_100a).
#pragma once

#include <cuda_runtime.h>
#include <algorithm>
#include <cuda_bf16.h>
#include <stdint.h>

#include "../../include/revffn_moe.h"

namespace revffn {

typedef __nv_bfloat16 bf16;

// Padded row space: every expert's segment of the permuted buffers starts at a
// multiple of ROW_PAD rows, so that a 128-row GEMM tile never spans two experts
// and the per-expert K range of a weight-gradient GEMM is a whole number of tiles.
constexpr int ROW_PAD = 128;

__host__ __device__ inline int64_t ceil_div(int64_t a, int64_t b) { return (a + b - 1) / b; }
__host__ __device__ inline int64_t round_up(int64_t a, int64_t b) { return ceil_div(a, b) * b; }

// Upper bound on padded rows: every non-empty expert wastes at most ROW_PAD-1 rows.
inline int64_t max_padded_rows(int64_t tokens, int top_k, int n_experts) {
  int64_t r = tokens * top_k;
  int64_t bound = r + (int64_t)n_experts * (ROW_PAD - 1);
  bound = round_up(bound, ROW_PAD);
  return bound;
}

__device__ __forceinline__ float to_f32(float v) { return v; }
__device__ __forceinline__ float to_f32(bf16 v) { return __bfloat162float(v); }
template <typename T> __device__ __forceinline__ T from_f32(float v);
template <> __device__ __forceinline__ float from_f32<float>(float v) { return v; }
template <> __device__ __forceinline__ bf16 from_f32<bf16>(float v) { return __float2bfloat16_rn(v); }

__device__ __forceinline__ float sigmoid_f(float x) { return 1.0f / (1.0f + __expf(-x)); }

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Block-wide sum for blockDim.x <= 1024 (multiple of 32); result valid in all threads.
__device__ __forceinline__ float block_sum(float v, float* smem32) {
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  v = warp_sum(v);
  __syncthreads();
  if (lane == 0) smem32[w] = v;
  __syncthreads();
  int nw = (blockDim.x + 31) >> 5;
  float t = (lane < nw) ? smem32[lane] : 0.f;
  t = warp_sum(t);
  return t;
}

// Sticky device status: first error wins.
__device__ __forceinline__ void set_status(int* status, int code) {
  if (status) atomicCAS(status, 0, code);
}

// Programmatic dependent launch.  Every kernel of the library is launched with launch_k / launch_cluster: it may then be
// set up, and its blocks may become resident, while the kernel before it on the stream still runs its last blocks.
//   pdl_wait     blocks until everything the launch depends on has completed and its writes are visible.  EVERY
//                kernel calls it, in every thread, before its first access to global memory and before any early return:
//                that also makes "the kernel before me has completed" imply "so have all before that one".
//   pdl_trigger  lets the next launch on the stream be set up (once every block has called it or has exited).
// What it saves is the 1.5-4 us between two dependent launches (a training step of four d = 512 blocks, 384 tokens, was some
// 530 launches then, 94 a block now: 3788 -> 2908 us; attention branch, 7 x 613 positions: 1337 -> 1252).
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// Short kernels release the next launch at once; the matrix products and attention kernels do it when a block's last
// operand loads are on their way, so that a waiting block does not hold an SM that another stream could use.
__device__ __forceinline__ void pdl_sync() { pdl_wait(); pdl_trigger(); }

template <typename... Params, typename... Args>
inline cudaError_t launch_cluster(void (*kernel)(Params...), dim3 grid, dim3 cluster, dim3 block, size_t smem, cudaStream_t st,
                                  Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2] = {};
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = cluster.x;
  attr[1].val.clusterDim.y = cluster.y;
  attr[1].val.clusterDim.z = cluster.z;
  cfg.attrs = attr;
  cfg.numAttrs = cluster.x * cluster.y * cluster.z > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
}
template <typename... Params, typename... Args>
inline cudaError_t launch_k(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args... args) {
  return launch_cluster(kernel, grid, dim3(1, 1, 1), block, smem, st, args...);
}

// Padded expert-major rows: every row of the 64 around `row` is padding (row_tok < 0; an expert's real rows come first).
__device__ __forceinline__ bool padding_group(const int32_t* __restrict__ row_tok, int64_t row) {
  return row_tok[row & ~static_cast<int64_t>(63)] < 0;
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src, bool ok) {      // !ok: 16 zero bytes
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;"
               ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(ok ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// 8 elements of T as one vector: loads/stores of 16 bytes for bf16, 2x16 for float.
// Blocks of `kernel` that are resident on the current device at once (one wave) for this block size and dynamic
// shared memory: the grid size of the grid-stride kernels.
template <typename Kernel>
inline cudaError_t resident_blocks(Kernel kernel, int threads, size_t smem, int* blocks) {
  int dev = 0, sms = 0, per_sm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem);
  *blocks = (e == cudaSuccess) ? std::max(1, sms * per_sm) : 0;
  return e;
}

template <typename T> struct Vec8;
template <> struct Vec8<bf16> {
  uint4 raw;
  __device__ __forceinline__ void load(const bf16* p) { raw = *reinterpret_cast<const uint4*>(p); }
  __device__ __forceinline__ void store(bf16* p) const { *reinterpret_cast<uint4*>(p) = raw; }
  __device__ __forceinline__ void get(float* f) const {
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&raw);
#pragma unroll
    for (int i = 0; i < 4; ++i) { float2 t = __bfloat1622float2(h[i]); f[2 * i] = t.x; f[2 * i + 1] = t.y; }
  }
  __device__ __forceinline__ void set(const float* f) {
    __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&raw);
#pragma unroll
    for (int i = 0; i < 4; ++i) h[i] = __floats2bfloat162_rn(f[2 * i], f[2 * i + 1]);
  }
  __device__ __forceinline__ void zero() { raw = make_uint4(0, 0, 0, 0); }
};
template <> struct Vec8<float> {
  float4 a, b;
  __device__ __forceinline__ void load(const float* p) {
    a = *reinterpret_cast<const float4*>(p); b = *reinterpret_cast<const float4*>(p + 4);
  }
  __device__ __forceinline__ void store(float* p) const {
    *reinterpret_cast<float4*>(p) = a; *reinterpret_cast<float4*>(p + 4) = b;
  }
  __device__ __forceinline__ void get(float* f) const {
    f[0] = a.x; f[1] = a.y; f[2] = a.z; f[3] = a.w; f[4] = b.x; f[5] = b.y; f[6] = b.z; f[7] = b.w;
  }
  __device__ __forceinline__ void set(const float* f) {
    a = make_float4(f[0], f[1], f[2], f[3]); b = make_float4(f[4], f[5], f[6], f[7]);
  }
  __device__ __forceinline__ void zero() { a = make_float4(0, 0, 0, 0); b = a; }
};

}  // namespace revffn
