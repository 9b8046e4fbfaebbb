// Count of this library's kernel launches, executed or queued for execution.
// Every launcher reports its launch; a launch recorded into a CUDA graph is
// counted each time the graph is replayed, not when it is recorded.
#pragma once
#include <cuda_runtime.h>

namespace fdgb {

// Counts `n` launches on stream `s` (as recorded into this thread's graph if `s`
// is capturing, else as executed).
void count_launches(cudaStream_t s, int n);
// Passes `e` through; on success counts `n` launches. A launch that failed is its
// caller's error alone: the runtime's last error is cleared, so that the next
// launch, of whichever handle, does not report it again.
inline cudaError_t counted(cudaError_t e, cudaStream_t s, int n = 1) {
    if (e == cudaSuccess)
        count_launches(s, n);
    else
        cudaGetLastError();
    return e;
}
// Launches this thread has recorded into graphs so far.
long long captured_launches();
// A replay of a graph holding `n` launches.
void count_replay(long long n);
// Executed or queued launches since the library was loaded (all threads).
long long kernel_launches();

}  // namespace fdgb
