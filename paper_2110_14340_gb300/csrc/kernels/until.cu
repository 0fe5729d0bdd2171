// until.cu - the device side of jacc_sweep_until: the loop's exit test and
// the choice of the final converting sweep, run inside the CUDA graph so the
// loop needs no host round trip.
#include <cuda_runtime.h>

#include "../host/jacc_internal.h"

namespace {

// After each sweep: move the sweep's residual from its accumulation slot to
// resid[i], clear the slot for the next sweep and count the sweep.  Once a
// residual reaches the tolerance, or max sweeps ran, the stop word is set: the
// sweeps and checks left in the loop's body then return at once, and the loop
// ends.  It also ends, and the next one begins, when `until` sweeps ran.
__global__ void jacc_k_until_check(double* slot, int* counter, int* stop, double* resid, double tol, int max_sweeps,
                                   cudaGraphConditionalHandle h_loop, int until, cudaGraphConditionalHandle h_next) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (__ldcg(stop)) return;
  const double r = __ldcg(slot);
  *slot = 0.0;
  const int i = *counter;
  resid[i] = r;
  *counter = i + 1;
  const bool more = r > tol && i + 1 < max_sweeps;
  if (!more) *stop = 1;
  const bool here = i + 1 < until;
  cudaGraphSetConditional(h_loop, more && here ? 1u : 0u);
  if (!here) cudaGraphSetConditional(h_next, more ? 1u : 0u);
}

// After the loop: report the sweep count and the result buffer, and pick the
// final sweep that rewrites the result in FP64 from the state before it:
// 0 = the only sweep (u0 -> u1, FP64 in and out), 1 = an even count
// (u1 -> u0), 2 = an odd count of 3 or more (u0 -> u1); 3 = none.
__global__ void jacc_k_until_final(const int* counter, int* status, int recompute, cudaGraphConditionalHandle h_final) {
  const int n = *counter;
  status[0] = n;
  status[1] = n & 1;
  unsigned c = 3u;
  if (recompute) c = (n == 1) ? 0u : ((n & 1) ? 2u : 1u);
  cudaGraphSetConditional(h_final, c);
}

}  // namespace

namespace jacc {

cudaError_t launch_until_check(double* slot, int* counter, int* stop, double* resid, double tol, int max_sweeps,
                               cudaGraphConditionalHandle h_loop, int until, cudaGraphConditionalHandle h_next,
                               cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(1);
  cfg.blockDim = dim3(1);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, jacc_k_until_check, slot, counter, stop, resid, tol, max_sweeps, h_loop, until,
                            h_next);
}

cudaError_t launch_until_final(const int* counter, int* status, int recompute, cudaGraphConditionalHandle h_final,
                               cudaStream_t s) {
  jacc_k_until_final<<<1, 1, 0, s>>>(counter, status, recompute, h_final);
  return cudaGetLastError();
}

}  // namespace jacc
