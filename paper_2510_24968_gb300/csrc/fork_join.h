// Launches spread over a caller's stream and auxiliary streams.
#pragma once
#include <cuda_runtime_api.h>

namespace fsim {

constexpr int kMaxForked = 8;

// Calls launch(st) with st[0] = s and st[1..naux] = aux between a fork event (the
// auxiliary streams start after what is on s) and join events (s goes on after
// them).  The streams are joined whatever happened inside launch: after a failed
// build the next one clears its accumulators on s, and no kernel of the failed one
// may still be adding into them.  Returns the first error of the events.
template <class Launch>
cudaError_t fork_join(cudaStream_t s, int naux, const cudaStream_t* aux, cudaEvent_t fork_ev,
                      const cudaEvent_t* join_ev, Launch&& launch) {
  if (naux < 0 || naux >= kMaxForked) return cudaErrorInvalidValue;
  cudaStream_t st[kMaxForked] = {s};
  cudaError_t e = cudaEventRecord(fork_ev, s);
  for (int k = 0; k < naux && e == cudaSuccess; ++k) {
    st[k + 1] = aux[k];
    e = cudaStreamWaitEvent(aux[k], fork_ev, 0);
  }
  if (e != cudaSuccess) return e;  // nothing launched
  launch(static_cast<const cudaStream_t*>(st));
  for (int k = 0; k < naux; ++k) {
    cudaError_t j = cudaEventRecord(join_ev[k], aux[k]);
    if (j == cudaSuccess) j = cudaStreamWaitEvent(s, join_ev[k], 0);
    if (e == cudaSuccess) e = j;
  }
  return e;
}

}  // namespace fsim
