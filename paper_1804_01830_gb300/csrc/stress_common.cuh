// Helpers shared by the translation units of the stress passes.
#pragma once
#include <cuda_fp16.h>

#include <atomic>
#include <mutex>

#include "dds_fft.cuh"
#include "dds_internal.h"

namespace dds {

constexpr int NT = 256;   // threads of the shared-memory z pass

// Small y tiles keep several CTAs resident per SM, so that one tile's copies overlap another
// tile's transform.
// y-pass tiles: W columns, NT threads.  The 512-row inverse takes 16 columns and 256
// threads (whole 128-byte rows; GaN layer 0.215 -> 0.207 ms); the 512-row forward keeps
// 8 and 128 (0.176 against 0.183 ms with 16).  1024 rows take 8 columns and 256 threads in
// both directions, in register stages like the others (512x512x64, two sets, against 4
// columns: forward 0.84 -> 0.75 ms; inverse, there in a shared-memory Stockham tile, 0.96 ->
// 0.84 ms; radial disk inverse 0.131 -> 0.119 ms).
template <int P, bool INV = false> struct YTile {
  static constexpr int W = P >= 1024 ? 8 : (P >= 512 ? (INV ? 16 : 8) : 16);
  static constexpr int NT = (P == 1024 || (P == 512 && INV)) ? 256 : 128;
};

__device__ __forceinline__ float2 cmadd_i(float2 acc, float g, float2 r) {
  // acc + (i g) * r
  return make_float2(fmaf(-g, r.y, acc.x), fmaf(g, r.x, acc.y));
}

__device__ __forceinline__ float bf16_to_f32(uint16_t v) { return __uint_as_float(((uint32_t)v) << 16); }

// Programmatic dependent launch.  Every kernel of an evaluation is launched with
// launch_pass: it may start while the kernel before it in the stream still runs, calls
// pdl_trigger() first (which lets the next one start once every CTA of this one has begun),
// and touches memory another kernel writes or reads only after pdl_wait(), which returns
// when everything before it in the stream has finished.  Every CTA calls pdl_wait(), so
// completion is transitive along the chain.  Data of the kernel before is read with
// ld_cg / ld_cs or asynchronous copies, never through the non-coherent path, which the
// compiler may move across the wait.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ float2 ld_cg(const float2 *p) {
  float2 v;
  asm volatile("ld.global.cg.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
  return v;
}
// *p where cond holds, else 0 (one predicated load: a branch around the load would keep
// neighbouring loads from being in flight together).
__device__ __forceinline__ float2 ld_cg_if(const float2 *p, bool cond) {
  float2 v;
  asm volatile(
      "{\n .reg .pred q;\n setp.ne.s32 q, %3, 0;\n mov.f32 %0, 0f00000000;\n mov.f32 %1, 0f00000000;\n"
      " @q ld.global.cg.v2.f32 {%0, %1}, [%2];\n}"
      : "=&f"(v.x), "=&f"(v.y)
      : "l"(p), "r"((int)cond));
  return v;
}
__device__ __forceinline__ float2 ld_cs(const float2 *p) {
  float2 v;
  asm volatile("ld.global.cs.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
  return v;
}
__device__ __forceinline__ float4 ld_cs(const float4 *p) {
  float4 v;
  asm volatile("ld.global.cs.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
  return v;
}
__device__ __forceinline__ float ld_cs(const float *p) {
  float v;
  asm volatile("ld.global.cs.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ uint2 ld_cs(const uint2 *p) {
  uint2 v;
  asm volatile("ld.global.cs.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
  return v;
}
// Cached in L1: values whose neighbours in the same sector a later load takes.
__device__ __forceinline__ unsigned ld_ca(const unsigned *p) {
  unsigned v;
  asm volatile("ld.global.ca.u32 %0, [%1];" : "=r"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ uint16_t ld_ca(const uint16_t *p) {
  uint16_t v;
  asm volatile("ld.global.ca.u16 %0, [%1];" : "=h"(v) : "l"(p));
  return v;
}

// Asynchronous copy of n values (even; both ends 16-byte aligned) of a constant table into
// shared memory by NT threads: issued before pdl_wait(), it costs no latency of its own
// (copied through registers, the first rows of a pass waited for the table).
template <int NT>
__device__ __forceinline__ void stage_table(float2 *dst, const float2 *src, int n, int tid) {
  for (int i = 2 * tid; i < n; i += 2 * NT) cp_async16(dst + i, src + i);
}

constexpr int MAX_DEV = 64;

// Function attributes of a pass kernel on the current device `dev`, set on its first launch
// there and when a launch needs more shared memory than any before (only ever raised).
// MAX_SHARED: prefer shared memory over L1 (not for the kernel without shared memory, whose
// row segments share L1 lines: radial disk z pass 0.223 against 0.280 ms).
template <auto Kernel, bool MAX_SHARED>
cudaError_t pass_attributes(int dev, size_t smem) {
  static std::mutex mu;
  static std::atomic<long> set[MAX_DEV];       // 1 + shared memory the kernel is prepared for
  if (dev < 0 || dev >= MAX_DEV) return cudaErrorInvalidDevice;
  if (set[dev].load(std::memory_order_acquire) > (long)smem) return cudaSuccess;
  std::lock_guard<std::mutex> lock(mu);
  if (set[dev].load(std::memory_order_relaxed) > (long)smem) return cudaSuccess;
  cudaError_t err = cudaSuccess;
  if (MAX_SHARED)
    err = cudaFuncSetAttribute(Kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                               (int)cudaSharedmemCarveoutMaxShared);
  if (err == cudaSuccess && smem > 48 * 1024)
    err = cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (err == cudaSuccess) set[dev].store((long)smem + 1, std::memory_order_release);
  return err;
}

// early: may start before the kernel ahead of it in the stream has finished.
template <auto Kernel, bool MAX_SHARED = true, typename... Args>
cudaError_t launch_pass(bool early, dim3 grid, unsigned threads, size_t smem, cudaStream_t s, Args... args) {
  int dev = 0;
  cudaError_t err = cudaGetDevice(&dev);
  if (err == cudaSuccess) err = pass_attributes<Kernel, MAX_SHARED>(dev, smem);
  if (err != cudaSuccess) return err;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = early ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, Kernel, args...);
}

template <typename K>
inline cudaError_t prep(K kernel, size_t smem) {
  cudaError_t err = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                                         (int)cudaSharedmemCarveoutMaxShared);
  if (err != cudaSuccess || smem <= 48 * 1024) return err;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}

// Fused z pass (zpass_f32.cu, zpass_f16.cu).  ks: kernel spectra, FP32 or FP16 (kscale != nullptr:
// FP16 storage, value = stored * kscale[c * fe + e]).
cudaError_t dispatch_z(const Shape &sh, const float2 *im, const float2 *in, const void *ks, const float *kscale,
                       float2 *om, float2 *on, const float2 *tw, cudaStream_t s);
cudaError_t dispatch_z_f16(const Shape &sh, const float2 *im, const float2 *in, const __half *ks, const float *kscale,
                           float2 *om, float2 *on, const float2 *tw, cudaStream_t s);

}  // namespace dds
