// Host-side helpers shared by the C-ABI entry points: status codes, argument checks,
// last-error bookkeeping.  No device code.
#pragma once
#include <atomic>
#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

#include "../../include/mpfa.h"

namespace mpfa {

constexpr int HEAD_DIM = 128;
constexpr int TILE = 128;        // tokens per quantization / attention tile
constexpr int PAGE = 64;         // tokens per KV-cache page
constexpr int DECODE_SPLIT = 1024;  // tokens per decode partition (8 x 128, Section 5.3)

extern thread_local int g_last_cuda_error;

inline int pad128(int n) { return (n + TILE - 1) / TILE * TILE; }
inline bool aligned(const void *p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

inline mpfa_status cuda_fail(cudaError_t e) {
  (void)cudaGetLastError();   // reported here: not again by the next call that asks
  g_last_cuda_error = static_cast<int>(e);
  return MPFA_ERR_CUDA;
}

#define MPFA_CUDA_OK(expr)                                    \
  do {                                                        \
    cudaError_t _e = (expr);                                  \
    if (_e != cudaSuccess) return ::mpfa::cuda_fail(_e);      \
  } while (0)

#define MPFA_LAUNCH_OK()                                      \
  do {                                                        \
    cudaError_t _e = cudaGetLastError();                      \
    if (_e != cudaSuccess) return ::mpfa::cuda_fail(_e);      \
  } while (0)

// Launch whose CTAs may be scheduled while the preceding kernel of the stream is still running (programmatic stream
// serialization): set-up that touches no memory the preceding work writes overlaps its tail.  Every kernel launched this
// way calls grid_dependency_wait() before its first access to global memory, in every thread that makes one, so the
// order of the stream holds transitively.  Such a kernel is resident while its inputs are still being written, so it reads global
// memory with ordinary loads only: a non-coherent load (__ldg, ld.global.nc, what the compiler makes of const __restrict__)
// asks for data that no one writes during the kernel's life, and the compiler may move it above the wait.
struct Grid {   // blocks, and how many along x make a cluster
  dim3 blocks;
  unsigned cluster;
  Grid(dim3 b, unsigned c = 1) : blocks(b), cluster(c) {}
};
template <typename... KArgs, typename... Args>
cudaError_t launch(void (*kernel)(KArgs...), Grid grid, dim3 block, size_t smem, cudaStream_t stream, Args &&...args) {
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = grid.cluster;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid.blocks;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = grid.cluster > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// How many clusters of a launch the stream's context holds at a time; 0 where it cannot place one.
template <typename... KArgs>
int max_active_clusters(void (*kernel)(KArgs...), Grid grid, dim3 block, size_t smem, cudaStream_t stream) {
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = grid.cluster;
  attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid.blocks;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
    (void)cudaGetLastError();   // answered here: not reported by the next call that asks
    return 0;
  }
  return n;
}

// The current device and its SM count; MPFA_ERR_ARCH for devices that cannot run the sm_100a-only kernels.  These are facts of
// the device, whatever its contexts, and asked for once (two attribute queries cost as much host time as a third of a launch).
mpfa_status device_info(int *dev, int *n_sm);

constexpr int MAX_DEVICES = 64;

// Lets a kernel use `bytes` of dynamic shared memory.  The driver keeps that per context, and a device can have several or lose one,
// so it is told before every launch (no pass got measurably longer by it: one decode step 22.7 us without, 22.4 with).
template <auto Kernel>
mpfa_status allow_smem(size_t bytes) {
  MPFA_CUDA_OK(cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
  return MPFA_OK;
}

}  // namespace mpfa
