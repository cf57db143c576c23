// Diagnostic kernel behind marche_debug_bounded_wait: exercises the give-up path of the bounded
// mbarrier wait that every TMA / tcgen05 kernel of the library relies on (sm100_ptx.cuh, mbar_wait), and of a cluster one
// of whose CTAs gave up (cluster_raise).  One thread of a cluster of two CTAs waits on a barrier that nothing ever arrives
// on; once the cycle limit has passed the wait returns false and the thread raises the cluster's flags; behind the cluster
// barrier the OTHER CTA, which finds its flag raised, writes the code into the status word and the kernel ends normally.
// Nothing traps, faults or spins without a bound; the context stays usable.
#include "kernels.h"
#include "launch_pdl.h"
#include "sm100_ptx.cuh"

namespace marche {

namespace {

enum { ST_PROBE = 0x71 };

__global__ void __launch_bounds__(32)
bounded_wait_probe_kernel(long long limit_cycles, int* __restrict__ status) {
  __shared__ __align__(8) unsigned long long bar;
  __shared__ int abort_flag;
  const int lane = threadIdx.x;
  const bool waiter = ptx::cluster_ctarank() == 0;
  if (lane == 0) {
    ptx::mbar_init(ptx::smem_u32(&bar), 1);
    abort_flag = 0;
    ptx::fence_barrier_init();
  }
  __syncwarp();
  ptx::cluster_sync_all();                               // both flags are down
  pdl_sync();
  bool ok = true;
  if (waiter && lane == 0) ok = ptx::mbar_wait(ptx::smem_u32(&bar), 0u, &abort_flag, limit_cycles);
  if (!ok) ptx::cluster_raise(ptx::smem_u32(&abort_flag), 2);
  __syncwarp();
  ptx::cluster_sync_all();
  if (!waiter && lane == 0 && *(volatile int*)&abort_flag) *(volatile int*)status = ST_PROBE;
}

}  // namespace

cudaError_t launch_bounded_wait_probe(long long limit_cycles, int* status, cudaStream_t st) {
  return launch_pdl_cluster(bounded_wait_probe_kernel, dim3(2), dim3(32), 0, 2, st, limit_cycles, status);
}

}  // namespace marche
