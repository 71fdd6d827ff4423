// tma.cuh -- shared-memory barriers (mbarrier) and TMA copies in inline PTX,
// shared by the 2D step kernels and the tube kernel. Every wait is bounded.
#pragma once

#include <cuda.h>  // CUtensorMap
#include <cuda_runtime.h>

namespace gbtma {

constexpr long long TMA_WAIT_CYCLES = 2000000000ll;  // ~1 s at 2 GHz

__device__ __forceinline__ unsigned smem_addr(const void* p) {
  return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(unsigned long long* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(unsigned long long* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned long long* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned long long* bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Waits for phase `parity` of the barrier for at most `limit` SM cycles.
__device__ __forceinline__ bool mbar_wait_bounded(unsigned long long* bar, unsigned parity,
                                                  long long limit) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity)) {
    if (clock64() - t0 > limit) return false;
    __nanosleep(64);
  }
  return true;
}
__device__ __forceinline__ void tma_load_tile(void* dst, const CUtensorMap* map, int x, int y,
                                              unsigned long long* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes "
      "[%0], [%1, {%2, %3, %4}], [%5];" ::"r"(smem_addr(dst)),
      "l"(reinterpret_cast<unsigned long long>(map)), "r"(x), "r"(y), "r"(0), "r"(smem_addr(bar))
      : "memory");
}

// Untiled bulk copy of `bytes` (a multiple of 16) from global to shared
// memory, both addresses 16-byte aligned; completes on `bar` (transaction
// bytes counted by the caller's expect_tx).
__device__ __forceinline__ void bulk_load(void* dst, const void* src, unsigned bytes,
                                          unsigned long long* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(smem_addr(dst)),
      "l"(reinterpret_cast<unsigned long long>(src)), "r"(bytes), "r"(smem_addr(bar))
      : "memory");
}

// Orders this thread's earlier generic-proxy memory accesses with later
// async-proxy (TMA) accesses: needed when a kernel's own global stores are
// read back by bulk copies later in the same launch.
__device__ __forceinline__ void fence_proxy_async() {
  asm volatile("fence.proxy.async;" ::: "memory");
}

// Programmatic dependent launch. A kernel launched by launch_overlapped() may
// start while the stream's previous kernel is still running, once every block
// of that one has called dependents_may_start() (or has ended): its blocks then
// set up their barriers and wait in wait_for_previous() until the previous
// kernel has completed and its writes are visible. Every thread calls that
// before it touches memory that the previous kernel may write or read. A kernel's
// pointers to such memory are not __restrict__ and not read with __ldg: either
// promises that the memory does not change while the kernel runs, and lets the compiler
// move reads (and, for __restrict__, writes) above the wait.
//
// The step kernels call dependents_may_start() when a block has only its stores
// left (FP64 and double-word persistent ones before their last tile, FP32 ones of
// many tiles at once). Called at their top, the next step's blocks take whatever slots are free
// then, so that some SMs get several of them and others none: a grid of two blocks
// or so per SM takes the time of the fullest. Measured, us a step, plain launches /
// early / late:
//   FP64, one thread per node, 2400 x 4: 13.7 / 22.9 / 12.1;
//   FP32 200 x 150 4.4 / 5.1 / 4.1, 300 x 200 5.0 / 5.3 / 4.7, 600 x 200 6.5 / 6.1 / 6.1;
//   LBM_FP32_DWMOM 256 x 128 4.9 / 6.7 / 4.6, 400 x 225 7.1 / 7.5 / 6.6.
// Audit steps leave it out: their blocks end in a chain of fences and counters, beside
// which the next step's blocks would only wait (audits on every step, FP32 160 x 120:
// 11.5 us plainly, 11.9 with it, 11.3 without).
__device__ __forceinline__ void dependents_may_start() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void wait_for_previous() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}
template <typename... P, typename... A>
inline cudaError_t launch(bool overlapped, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem,
                          cudaStream_t stream, A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = overlapped ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}
template <typename... P, typename... A>
inline cudaError_t launch_overlapped(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem,
                                     cudaStream_t stream, A&&... args) {
  return launch(true, kernel, grid, block, smem, stream, static_cast<A&&>(args)...);
}

// cuTensorMapEncodeTiled through the runtime (libcuda is not linked); null if
// the driver does not have it.
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline EncodeTiledFn tensor_map_encoder() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (EncodeTiledFn)p;
  }
  return fn;
}

}  // namespace gbtma
