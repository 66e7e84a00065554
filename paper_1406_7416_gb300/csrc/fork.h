// Parallel branches in a captured stream.
#pragma once

#include <cuda_runtime.h>

#include <vector>

namespace adg {

// Independent launches on one stream: when the stream is being captured, each
// branch (the launches since the fork or the last branch()) depends on what
// came before the fork only, and what follows join() on all of them, so the
// graph runs them side by side; outside a capture they stay in stream order.
class Fork {
 public:
  explicit Fork(cudaStream_t s) : s_(s) { err_ = deps(&base_); }
  cudaError_t branch() {
    if (err_ != cudaSuccess || !on_) return err_;
    std::vector<cudaGraphNode_t> end;
    if ((err_ = deps(&end)) != cudaSuccess) return err_;
    ends_.insert(ends_.end(), end.begin(), end.end());
    return err_ = set(base_);
  }
  cudaError_t join() {
    if (err_ != cudaSuccess || !on_) return err_;
    return err_ = set(ends_);
  }

 private:
  cudaError_t deps(std::vector<cudaGraphNode_t>* out) {
    cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
    const cudaGraphNode_t* d = nullptr;
    size_t n = 0;
    const cudaError_t e = cudaStreamGetCaptureInfo(s_, &status, nullptr, nullptr, &d, nullptr, &n);
    if (e != cudaSuccess) return e;
    on_ = status == cudaStreamCaptureStatusActive;
    if (on_) out->assign(d, d + n);
    return cudaSuccess;
  }
  cudaError_t set(std::vector<cudaGraphNode_t>& d) {
    return cudaStreamUpdateCaptureDependencies(s_, d.data(), nullptr, d.size(),
                                               cudaStreamSetCaptureDependencies);
  }
  cudaStream_t s_;
  bool on_ = false;
  cudaError_t err_ = cudaSuccess;
  std::vector<cudaGraphNode_t> base_, ends_;
};

}  // namespace adg
