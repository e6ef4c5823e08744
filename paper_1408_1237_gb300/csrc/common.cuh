// Internal helpers shared by the libkrr CUDA sources (sm_103a only).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "../../include/libkrr.h"

#ifndef __CUDACC__
#error "compile with nvcc"
#endif

namespace krr {

// Kernels launched by the library since load (host-side count; a launch
// captured into a CUDA graph counts once, at capture).
extern std::atomic<long long> g_launches;
inline void count_launch() { g_launches.fetch_add(1, std::memory_order_relaxed); }

// Source tile length: sources move through shared memory in tiles of TS
// points; every prepared point array is padded to a multiple of TS.
constexpr int TS = 256;
// Device error codes written to the handle's error word by kernels.
enum DevErr : int { DEV_OK = 0, DEV_TIMEOUT = 1, DEV_NONFINITE = 2, DEV_BREAKDOWN = 3 };

// Bounded waits give up after this many SM clocks (about one second).
constexpr long long WAIT_LIMIT_CLOCKS = 2000000000LL;

// ------------------------------------------------------------------ PTX ---
__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count)
               : "memory");
}

// Make barrier initialisation visible to the async (TMA) proxy.
__device__ __forceinline__ void fence_barrier_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile(
      "mbarrier.arrive.expect_tx.release.cta.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)),
      "r"(bytes)
      : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cta.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Wait for phase `parity` of `bar` to complete, giving up after `limit` SM
// clocks.  Returns false on timeout.
__device__ __forceinline__ bool mbar_wait_for(uint64_t* bar, uint32_t parity, long long limit) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity)) {
    if (clock64() - t0 > limit) return false;
  }
  return true;
}

// The bounded wait of every kernel: WAIT_LIMIT_CLOCKS.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity) {
  return mbar_wait_for(bar, parity, WAIT_LIMIT_CLOCKS);
}

// Programmatic dependent launch.  A kernel launched by launch_pdl may start
// while the one before it on the stream still runs, once every block of that
// one has called pdl_trigger or left; what it reads or writes that any earlier
// kernel of the stream touches comes after pdl_wait, which returns when those
// are complete.  pdl_trigger is called only after a kernel's own pdl_wait, so
// what came before the preceding kernel is complete from the start.  Without
// the launch attribute both do nothing.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  count_launch();
  return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}

// 1-D bulk copy global -> this CTA's shared memory, completing on `bar`.
// dst, src 16-byte aligned; bytes a multiple of 16.
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes,
                                         uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(smem_addr(dst)),
      "l"(src), "r"(bytes), "r"(smem_addr(bar))
      : "memory");
}

// 2^x on the special-function unit (MUFU.EX2), flushing subnormal results.
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Square root on the special-function unit (PTX documents a relative error of
// at most 2^-23; 0 at 0).  The Matern kernel took r2 * rsqrtf(max(r2, 1e-30))
// before: a clamp, a multiplication and rsqrtf's denormal handling per pair
// more (100,003 points, d = 3: product kernel 4.51 -> 3.49 ms).
__device__ __forceinline__ float sqrt_mufu(float x) {
  float y;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// (double)v by integer operations.  The conversion instruction runs at the
// FP64 pipe's 2 results per clock and SM; a tensor-core product's CTA converts
// 8192 sums in its epilogue, which took 2 us of the 13 us of a 2,000-point
// product of 11 columns.
__device__ __forceinline__ double f2d(float v) {
  const uint32_t u = __float_as_uint(v);
  if ((u & 0x7F800000u) - 0x00800000u < 0x7F000000u)  // normal
    return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7FFFFFFFu) >> 3) + 0x38000000u)), (int)(u << 29));
  if ((u << 1) == 0u) return __hiloint2double((int)u, 0);
  return (double)v;
}

constexpr uint32_t TF32_MASK = 0xFFFFE000u;  // clears the 13 mantissa bits tf32 drops
constexpr uint32_t TF32_HALF = 0x1000u;      // half a unit of tf32's last place

// v rounded to tf32, half away from zero.  (The largest finite weights keep
// their value: rounding up would carry into infinity.)
__device__ __forceinline__ uint32_t tf32_hi(float v) {
  const uint32_t u = __float_as_uint(v), up = u + TF32_HALF;
  return ((up & 0x7F800000u) == 0x7F800000u ? u : up) & TF32_MASK;
}

// d += a b, tf32 operands.
__device__ __forceinline__ void mma_1688_tf32(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 fadd2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 fmul2(float2 a, float2 b) { return __fmul2_rn(a, b); }

// Kahan-compensated accumulation of v into (s, c).
__device__ __forceinline__ void kahan_add(float& s, float& c, float v) {
  const float y = __fsub_rn(v, c);
  const float t = __fadd_rn(s, y);
  c = __fsub_rn(__fsub_rn(t, s), y);
  s = t;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

__device__ __forceinline__ float warp_min(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// Block-wide sum of a double (all threads get the result).  `red` holds at
// least blockDim.x/32 doubles of shared memory.
__device__ __forceinline__ double block_sum(double v, double* red) {
  v = warp_sum(v);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = blockDim.x >> 5;
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  double t = (l < nw) ? red[l] : 0.0;
  t = warp_sum(t);
  return t;
}

}  // namespace krr
