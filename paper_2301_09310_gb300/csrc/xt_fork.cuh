// xt_fork.cuh -- a call's kernels on the context's internal streams, forked from the
// call's stream and joined back into it (host code).
#pragma once
#include <cuda_runtime_api.h>

namespace xt {

// Every stream that was forked is joined, also when a launch in between failed: the
// caller frees or rewrites what the kernels launched before it use, in the call's
// stream's order.
class Fork {
 public:
  // Onto the first n of aux (1 or fewer: everything stays on `stream`).
  Fork(cudaStream_t stream, cudaStream_t* aux, cudaEvent_t fork_ev, cudaEvent_t* join_ev, int n)
      : stream_(stream), aux_(aux), join_ev_(join_ev) {
    if (n <= 1) return;
    error_ = cudaEventRecord(fork_ev, stream);
    while (error_ == cudaSuccess && forked_ < n) {
      error_ = cudaStreamWaitEvent(aux[forked_], fork_ev, 0);
      if (error_ == cudaSuccess) ++forked_;
    }
  }
  Fork(const Fork&) = delete;
  Fork& operator=(const Fork&) = delete;
  ~Fork() { join(); }

  cudaError_t error() const { return error_; }
  bool apart() const { return forked_ > 0; }
  // The stream of branch b (of the call where nothing was forked).
  cudaStream_t branch(int b) const { return apart() ? aux_[b % forked_] : stream_; }

  cudaError_t join() {
    for (int b = 0; b < forked_; ++b) {
      cudaError_t e = cudaEventRecord(join_ev_[b], aux_[b]);
      if (e == cudaSuccess) e = cudaStreamWaitEvent(stream_, join_ev_[b], 0);
      if (e != cudaSuccess) {
        cudaStreamSynchronize(aux_[b]);  // the host waits instead
        if (error_ == cudaSuccess) error_ = e;
      }
    }
    forked_ = 0;
    return error_;
  }

 private:
  cudaStream_t stream_;
  cudaStream_t* aux_;
  cudaEvent_t* join_ev_;
  int forked_ = 0;
  cudaError_t error_ = cudaSuccess;
};

}  // namespace xt
