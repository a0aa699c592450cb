// Launches side by side on two streams.
#pragma once

#include <cuda_runtime.h>

namespace mcao {

// launch(i, stream) for i < n, behind s0's work so far and before its later work: the first on s0, the others
// on s1 beside it.  s1 joins s0 also when a launch fails: what was queued before it may still be running,
// and s0 is all that is waited for.
template <class F>
cudaError_t fork_launches(cudaStream_t s0, cudaStream_t s1, cudaEvent_t ev, int n, F&& launch) {
    if (n <= 1) return n == 1 ? launch(0, s0) : cudaSuccess;
    cudaError_t e = cudaEventRecord(ev, s0);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(s1, ev, 0);
    for (int i = 0; i < n && e == cudaSuccess; ++i) e = launch(i, i == 0 ? s0 : s1);
    cudaError_t join = cudaEventRecord(ev, s1);
    if (join == cudaSuccess) join = cudaStreamWaitEvent(s0, ev, 0);
    return e != cudaSuccess ? e : join;
}

}  // namespace mcao
