// Launch helper: programmatic dependent launch for the step's kernel chain.
//
// Every kernel of the library begins with pdl_wait() (griddepcontrol.wait: returns once the
// preceding kernel of the stream has completed and its writes are visible) followed by
// pdl_launch_dependents(), and every launch carries the programmatic-stream-serialization
// attribute.  The next kernel's CTAs may therefore become resident, and run their private
// set-up (barrier init, TMEM allocation, tensor-map prefetch), while the current kernel is
// still draining.  Of global memory they read before the wait only what was complete before the
// current kernel began (weights, biases, a stack's LayerNorm parameters) and prefetch into L2;
// they write nothing.  Because each kernel releases its dependents only after its own wait has
// returned, at most one kernel runs ahead.
// pdl_switch() holds the process-wide on/off state (marche_set_tuning; on by default).
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace marche {

inline bool& pdl_switch() {
  static bool on = true;
  return on;
}

// Raises a kernel's dynamic shared-memory limit to at least `bytes` on the current device.  The
// attribute belongs to the device's context, so what has been set is remembered per device
// (`cache`: one zero-initialised array per kernel instantiation at the call site).
constexpr int kMaxDevices = 64;
template <typename Kernel>
cudaError_t ensure_dynamic_smem(Kernel kernel, size_t bytes, size_t (&cache)[kMaxDevices]) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  if (bytes <= cache[dev]) return cudaSuccess;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e == cudaSuccess) cache[dev] = bytes;
  return e;
}

// An SM that has to divide its L1 / shared memory differently for the next kernel takes it in only once it has run empty,
// which undoes the overlap of launches.  The small kernels between the projections use no dynamic shared memory and would
// get a large L1; with this they ask for the division that the projections have (ten rows' step 885 -> 850 us, an fp32 run
// 976 -> 945 us).  LayerNorm on many rows is better off with its L1 (in-step selection at 16 rows 1919 us, 1928 with this).
template <typename Kernel>
cudaError_t prefer_shared_memory(Kernel kernel, bool (&done)[kMaxDevices]) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  if (done[dev]) return cudaSuccess;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  if (e == cudaSuccess) done[dev] = true;
  return e;
}

// cluster > 1: consecutive groups of `cluster` CTAs (x) form a thread-block cluster.
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl_cluster(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, int cluster, cudaStream_t st,
                               Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  int n = 0;
  if (pdl_switch()) {
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n].val.programmaticStreamSerializationAllowed = 1;
    ++n;
  }
  if (cluster > 1) {
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = (unsigned)cluster;
    attr[n].val.clusterDim.y = 1;
    attr[n].val.clusterDim.z = 1;
    ++n;
  }
  cfg.attrs = attr;
  cfg.numAttrs = n;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(std::forward<Args>(args))...);
}

template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
  return launch_pdl_cluster(kernel, grid, block, smem, 1, st, std::forward<Args>(args)...);
}

}  // namespace marche
