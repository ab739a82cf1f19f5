// Side streams of a call: they continue from the caller's stream while a Fork is
// open and are joined to it on every way out.  A call that returns an error half
// way has launched work that writes to the plan's accumulators and to the caller's
// outputs; without the join nothing orders that work before what the caller does
// next, and a capture on the caller's stream could not be ended.
#pragma once
#include <cuda_runtime_api.h>

namespace eri {

class Fork {
 public:
  Fork(cudaStream_t main, const cudaStream_t* side, cudaEvent_t forked, const cudaEvent_t* joined)
      : main_(main), side_(side), forked_(forked), joined_(joined) {}
  Fork(const Fork&) = delete;
  Fork& operator=(const Fork&) = delete;
  ~Fork() { join(); }

  // side[0 .. n) continue from the main stream (n = 0: nothing to do)
  cudaError_t open(int n) {
    if (n <= 0) return cudaSuccess;
    cudaError_t e = cudaEventRecord(forked_, main_);
    while (e == cudaSuccess && n_ < n)
      if ((e = cudaStreamWaitEvent(side_[n_], forked_, 0)) == cudaSuccess) ++n_;
    return e;
  }

  // the main stream continues after the side streams; every one of them is tried,
  // the first error is returned
  cudaError_t join() {
    cudaError_t first = cudaSuccess;
    for (int b = 0; b < n_; ++b) {
      cudaError_t e = cudaEventRecord(joined_[b], side_[b]);
      if (e == cudaSuccess) e = cudaStreamWaitEvent(main_, joined_[b], 0);
      if (first == cudaSuccess) first = e;
    }
    n_ = 0;
    return first;
  }

 private:
  cudaStream_t main_;
  const cudaStream_t* side_;
  cudaEvent_t forked_;
  const cudaEvent_t* joined_;
  int n_ = 0;
};

}  // namespace eri
