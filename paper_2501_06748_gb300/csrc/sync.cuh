// Device-wide synchronisation shared by the set-up and time-loop kernels.
#pragma once

#include <utility>

#include "internal.h"

namespace sbfwi {

// The kernels of a time step are launched as dependents of their predecessor in the stream
// (launch_next), so that the launch itself is done by the time the predecessor ends.  They wait
// for it here, before they touch anything that it or a kernel before it writes or reads; set-up
// of barriers and copies of constant operators come before.  The wait ends when the predecessor
// has completed, and that one waited for its own, so the order of the stream holds for all.
// Per step of the 4 x 4 plate 32 -> 25 us, 24 x 24 elements, 8 shots 131 -> 123 us.
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Lets the successor's blocks start before this grid completes.  Only blocks of the solve that are
// out of items say so: a successor that starts while a kernel still works takes its place on the
// SMs (the element kernel's blocks then crowd the SMs with room left: 24 x 24 session 11.8 ms without,
// 16.6 ms with it at the start of every kernel).
__device__ __forceinline__ void grid_launch_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <class... Params, class... Args>
cudaError_t launch_next(void (*kernel)(Params...), unsigned grid, unsigned block, size_t smem, cudaStream_t st, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

// count doubles global -> shared by nthr threads, asynchronously; in pairs where wide (both addresses on 16 bytes)
__device__ __forceinline__ void copy_async(double* dst, const double* src, int count, int tid, int nthr, bool wide) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  if (wide) {
    for (int t = 2 * tid; t < count; t += 2 * nthr)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d + 8 * t), "l"(src + t) : "memory");
  } else {
    for (int t = tid; t < count; t += nthr)
      asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d + 8 * t), "l"(src + t) : "memory");
  }
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int kPending>
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(kPending) : "memory"); }

// Lets a kernel be launched with as much dynamic shared memory as the device has.  The limit belongs to the kernel,
// for all that use it in the process: were it set to what one caller needs, it would be lowered under the launches
// of others (a session keeps its own; other threads).
inline int allow_shared_memory(const void* kernel) {
  int device = 0, most = 0;
  SBFWI_CUDA(cudaGetDevice(&device));
  SBFWI_CUDA(cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, device));
  cudaFuncAttributes at;
  SBFWI_CUDA(cudaFuncGetAttributes(&at, kernel));
  const int limit = most - (int)at.sharedSizeBytes;
  if (at.maxDynamicSharedSizeBytes < limit)
    SBFWI_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, limit));
  return SBFWI_OK;
}

// FP64 element kernels: operators copied ahead where they leave room for four blocks on an SM and either all
// blocks are on the SMs at once anyway or a block is one element (figures at the launches)
inline bool stage_operators(size_t smem, int elements_per_block, unsigned blocks, int sms) {
  return smem <= 56 * 1024 && (elements_per_block == 1 || blocks <= 4u * (unsigned)sms);
}

// Grid-wide barrier for a cooperative launch (all blocks co-resident).  The wait
// is bounded: after `budget` clock cycles it records SBFWI_ETIMEOUT and gives up,
// so a broken launch returns an error instead of hanging the device.
__device__ __forceinline__ bool grid_barrier(unsigned* count, unsigned* gen, int* status, long long budget) {
  __syncthreads();
  __shared__ int ok;
  if (threadIdx.x == 0) {
    ok = 1;
    volatile unsigned* vgen = gen;
    const unsigned g = *vgen;
    __threadfence();
    const unsigned arrived = atomicAdd(count, 1u);
    if (arrived == gridDim.x - 1) {
      atomicExch(count, 0u);
      __threadfence();
      atomicAdd(gen, 1u);
    } else {
      const long long t0 = clock64();
      while (*vgen == g) {
        if (clock64() - t0 > budget || *(volatile int*)status != 0) {
          atomicCAS(status, 0, SBFWI_ETIMEOUT);
          ok = 0;
          break;
        }
        __nanosleep(64);
      }
    }
    __threadfence();
  }
  __syncthreads();
  return ok != 0;
}

}  // namespace sbfwi
