// Self-test of the bounded device waits (ks_selftest_wait_timeout in
// include/ks_steps.h).  Every wait in the library -- the software grid
// barrier of the cooperative kernels and the mbarrier waits of the TMA and
// tensor-core pipelines -- polls a bounded number of times, then records
// KS_ETIMEOUT in the launch's status word and returns, so a wait that cannot
// complete leaves the context usable and reaches the host as an error.
//
// The probe runs the library's own grid barrier in a launch of kProbeBlocks
// blocks while the barrier expects one more: the last arrival never comes, the
// waiting threads give up after kSpinLimit polls (about a second with the
// back-off), all about together, and the kernel returns with KS_ETIMEOUT
// recorded.  A second launch is the late block: its arrival completes the count,
// and it must be told of the failure all the same, or it would go on with what
// the departed blocks never wrote.
#include <chrono>

#include "ks_device.cuh"
#include "ks_steps.h"

namespace ks {
namespace {

constexpr unsigned int kProbeBlocks = 4;

// told: blocks that left the barrier with its failure.
__global__ void wait_timeout_probe_kernel(GridBarrier *bar, int *status, int *told) {
  unsigned int epoch = 0;
  const bool ok = grid_barrier_n(bar, status, kProbeBlocks + 1u, epoch);
  if (threadIdx.x == 0 && !ok) atomicAdd(told, 1);
}

struct ProbeState {
  GridBarrier bar;
  int status, told;
};

}  // namespace
}  // namespace ks

using namespace ks;

extern "C" {

ks_status ks_selftest_wait_timeout(void *stream, int *status, double *seconds) {
  if (!status) return set_error(KS_EINVAL, "null argument");
  cudaStream_t s = (cudaStream_t)stream;
  ProbeState *d = nullptr;
  KS_CUDA_TRY(cudaMalloc((void **)&d, sizeof(ProbeState)));
  ProbeState h{};
  ks_status st = KS_OK;
  const auto t0 = std::chrono::steady_clock::now();
  cudaError_t e = cudaMemsetAsync(d, 0, sizeof(ProbeState), s);
  if (e == cudaSuccess) {
    {
      ProfScope ps_(s, KP_OTHER, 0.0, 0.0, 2);
      wait_timeout_probe_kernel<<<kProbeBlocks, 32, 0, s>>>(&d->bar, &d->status, &d->told);
      wait_timeout_probe_kernel<<<1, 32, 0, s>>>(&d->bar, &d->status, &d->told);
    }
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(&h, d, sizeof(ProbeState), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) st = cuda_error(e, "wait-timeout probe");
  cudaFree(d);
  if (st != KS_OK) return st;
  if (h.status == KS_ETIMEOUT && h.told != (int)kProbeBlocks + 1)
    return set_error(KS_ECUDA, "wait-timeout probe: %d of %d blocks were told of the failure",
                     h.told, (int)kProbeBlocks + 1);
  *status = h.status;
  if (seconds)
    *seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
  return KS_OK;
}

}  // extern "C"
