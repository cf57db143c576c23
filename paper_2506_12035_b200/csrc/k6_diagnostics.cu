// Diagnostic kernel behind marche_debug_bounded_wait: exercises the give-up path of the bounded
// mbarrier wait that every TMA / tcgen05 kernel of the library relies on (sm100_ptx.cuh, mbar_wait), and of a cluster one
// of whose CTAs gave up (cluster_raise).  One thread of a cluster of two CTAs waits on a barrier that nothing ever arrives
// on; once the cycle limit has passed the wait returns false, the thread raises the cluster's flags and the CTA does not send the
// eight bytes (st.async) that the OTHER CTA waits for.  That CTA's wait has 200 million cycles more, but its flag ends it at
// once: it writes the code into the status word, both meet at the cluster barrier and the kernel ends normally.
// Nothing traps, faults or spins without a bound; the context stays usable.
#include "kernels.h"
#include "launch_pdl.h"
#include "sm100_ptx.cuh"

namespace marche {

namespace {

enum { ST_PROBE = 0x71 };

__global__ void __launch_bounds__(32)
bounded_wait_probe_kernel(long long limit_cycles, int* __restrict__ status) {
  __shared__ __align__(8) unsigned long long bars[2];    // nothing arrives on the first; the other CTA's bytes on the second
  __shared__ __align__(8) float2 share;
  __shared__ int abort_flag;
  const int lane = threadIdx.x;
  const bool waiter = ptx::cluster_ctarank() == 0;
  const uint32_t never = ptx::smem_u32(bars), sent = never + 8u;
  if (lane == 0) {
    ptx::mbar_init(never, 1);
    ptx::mbar_init(sent, 1);
    abort_flag = 0;
    ptx::fence_barrier_init();
    ptx::mbar_expect_tx(sent, 8u);
  }
  __syncwarp();
  ptx::cluster_sync_all();                               // both flags are down
  pdl_sync();
  bool ok = true;
  if (lane == 0) {
    if (waiter) {
      ok = ptx::mbar_wait(never, 0u, &abort_flag, limit_cycles);
      if (!ok) ptx::cluster_raise(ptx::smem_u32(&abort_flag), 2);
      else ptx::st_async_v2(ptx::mapa(ptx::smem_u32(&share), 1u), 0.f, 0.f, ptx::mapa(sent, 1u));
    } else {
      ok = ptx::mbar_wait_cluster(sent, 0u, &abort_flag, limit_cycles + 200000000LL);
      if (!ok) *(volatile int*)status = ST_PROBE;
    }
  }
  __syncwarp();
  ptx::cluster_sync_all();
}

}  // namespace

cudaError_t launch_bounded_wait_probe(long long limit_cycles, int* status, cudaStream_t st) {
  return launch_pdl_cluster(bounded_wait_probe_kernel, dim3(2), dim3(32), 0, 2, st, limit_cycles, status);
}

}  // namespace marche
