// Shared device helpers for the BSR kernels (storage-type packs, warp reductions, status word).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <utility>

namespace bsr {

typedef __nv_bfloat16 bf16;

// Device status word bits (read and cleared by bsr_sync_status).
enum : int { STATUS_TIMEOUT = 1, STATUS_NONFINITE = 2, STATUS_GUARD = 4, STATUS_CHECK = 8 };

// Index checks of the checked build (-DBSR_DEBUG): a failed check raises STATUS_CHECK in the status word (never a trap:
// the context stays usable) and the caller of the macro skips the access.  In the normal build the condition is not
// evaluated.
#ifdef BSR_DEBUG
#define BSR_CHECK(cond, status) ((cond) ? true : (((status) != nullptr ? (void)atomicOr((status), bsr::STATUS_CHECK) : (void)0), false))
#else
#define BSR_CHECK(cond, status) (true)
#endif

template <typename T> struct Pack;          // 16-byte vector of storage elements
template <> struct Pack<float> { static constexpr int N = 4; };
template <> struct Pack<bf16> { static constexpr int N = 8; };

__device__ __forceinline__ float to_f(float v) { return v; }
__device__ __forceinline__ float to_f(bf16 v) { return __bfloat162float(v); }
template <typename T> __device__ __forceinline__ T from_f(float v);
template <> __device__ __forceinline__ float from_f<float>(float v) { return v; }
template <> __device__ __forceinline__ bf16 from_f<bf16>(float v) { return __float2bfloat16_rn(v); }

// 16-byte aligned load/store of Pack<T>::N consecutive elements, widened to float.
__device__ __forceinline__ void load16(const float* p, float* f) {
  float4 v = *reinterpret_cast<const float4*>(p);
  f[0] = v.x; f[1] = v.y; f[2] = v.z; f[3] = v.w;
}
__device__ __forceinline__ void load16(const bf16* p, float* f) {
  uint4 v = *reinterpret_cast<const uint4*>(p);
  const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&v);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float2 t = __bfloat1622float2(h[i]);
    f[2 * i] = t.x; f[2 * i + 1] = t.y;
  }
}
__device__ __forceinline__ void store16(float* p, const float* f) {
  *reinterpret_cast<float4*>(p) = make_float4(f[0], f[1], f[2], f[3]);
}
__device__ __forceinline__ void store16(bf16* p, const float* f) {
  uint4 v;
  __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&v);
#pragma unroll
  for (int i = 0; i < 4; ++i) h[i] = __floats2bfloat162_rn(f[2 * i], f[2 * i + 1]);
  *reinterpret_cast<uint4*>(p) = v;
}

// four consecutive elements (16 bytes of float, 8 bytes of bf16)
__device__ __forceinline__ void load4(const float* p, float* f) { load16(p, f); }
__device__ __forceinline__ void load4(const bf16* p, float* f) {
  uint2 v = *reinterpret_cast<const uint2*>(p);
  const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&v);
  float2 a = __bfloat1622float2(h[0]), b = __bfloat1622float2(h[1]);
  f[0] = a.x; f[1] = a.y; f[2] = b.x; f[3] = b.y;
}
__device__ __forceinline__ void store4(float* p, const float* f) { store16(p, f); }
__device__ __forceinline__ void store4(bf16* p, const float* f) {
  uint2 v;
  __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&v);
  h[0] = __floats2bfloat162_rn(f[0], f[1]);
  h[1] = __floats2bfloat162_rn(f[2], f[3]);
  *reinterpret_cast<uint2*>(p) = v;
}

// N consecutive elements (N = 4 or 8) through 16-byte accesses, whatever the element type.
template <int N> __device__ __forceinline__ void load_n(const float* p, float* f) {
#pragma unroll
  for (int j = 0; j < N; j += 4) load16(p + j, f + j);
}
template <int N> __device__ __forceinline__ void load_n(const bf16* p, float* f) {
  static_assert(N == 8, "bf16 packs hold 8 elements");
  load16(p, f);
}
template <int N> __device__ __forceinline__ void store_n(float* p, const float* f) {
#pragma unroll
  for (int j = 0; j < N; j += 4) store16(p + j, f + j);
}
template <int N> __device__ __forceinline__ void store_n(bf16* p, const float* f) {
  static_assert(N == 8, "bf16 packs hold 8 elements");
  store16(p, f);
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ int warp_sum_int(int v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// 16 bytes from global to shared memory, on their own; a group of copies is committed, and all but the newest N groups waited for.
__device__ __forceinline__ void copy16_async(void* dst, const void* src, int bytes = 16) {      // bytes: what is copied, zeros follow
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void copies_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void copies_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Exact GELU x * Phi(x) and its derivative Phi(x) + x * phi(x).
__device__ __forceinline__ float gelu_f(float x) { return 0.5f * x * (1.0f + erff(x * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad_f(float x) {
  return 0.5f * (1.0f + erff(x * 0.70710678118654752f)) + x * 0.39894228040143268f * expf(-0.5f * x * x);
}

// Host-side count of kernel launches made by this library (read through bsr_profile_read).
extern long g_kernel_launches;
static inline void note_launch(int n = 1) { g_kernel_launches += n; }

// Programmatic dependent launch: every kernel of the step is launched so that it may start while the one before it on
// its stream still runs.  release_dependents() says that the next kernel may be scheduled (once every CTA of this one has
// said so or left); await_inputs() waits until the kernels before have completed and their writes are visible.  A kernel
// touches global memory only after await_inputs(), and every CTA of every kernel calls it, so completion of a kernel
// still implies completion of all before it.  A kernel that allocates tensor memory releases only after its allocation:
// otherwise the next kernel's CTA could take the columns first and wait for this one for good.
// It saves launch latency and prologue: a DeiT-S step of one image (199 launches) 746 -> 659 us, of 64 images 1572 -> 1492 us.
// Kernels that fill the SMs with one large CTA each (GEMM, attention) do not release: the next kernel's CTAs would pile up on
// the SMs whose CTA leaves first instead of spreading over all of them (ViT-B at batch 128: 5336 us without, 5341 us so,
// 5534 us with a release at their start).  On at most half of the SMs they do: the next kernel finds the others idle.  A product whose
// successor is another one does on any number below all (launch in gemm_tc.cu).
constexpr int B200_SMS = 148;
__device__ __forceinline__ bool leaves_sms_idle() { return 2u * gridDim.x * gridDim.y * gridDim.z <= (unsigned)B200_SMS; }
__device__ __forceinline__ void release_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void await_inputs() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void dependent_sync() { release_dependents(); await_inputs(); }

template <typename... KArgs, typename... Args>
static inline void launch_cluster(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, dim3 cluster, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = cluster.x; attr[1].val.clusterDim.y = cluster.y; attr[1].val.clusterDim.z = cluster.z;
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = stream;
  cfg.attrs = attr; cfg.numAttrs = cluster.x * cluster.y * cluster.z > 1 ? 2 : 1;
  cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
}
template <typename... KArgs, typename... Args>
static inline void launch_k(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, Args&&... args) {
  launch_cluster(kern, grid, block, smem, stream, dim3(1, 1, 1), std::forward<Args>(args)...);
}

// The dynamic shared-memory limit of a kernel is an attribute of the (kernel, device) pair, so the largest value set so
// far is remembered per device ordinal.  It only grows: launches captured earlier in a graph keep working.
struct SmemLimit {
  size_t set[64] = {};
};
template <typename Kernel>
static inline bool ensure_smem(SmemLimit& lim, Kernel kern, size_t bytes) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
  if (bytes > lim.set[dev]) {
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) != cudaSuccess) return false;
    lim.set[dev] = bytes;
  }
  return true;
}

static inline int ceil_div(long a, long b) { return (int)((a + b - 1) / b); }

}  // namespace bsr
