// Look-ahead work on a side stream (host code): forked from the main stream and joined to it again, also where the caller
// returns in between, so that buffers the side stream uses are not freed or reused under it.
#pragma once

#include <cuda_runtime_api.h>

namespace exa {

class SideJoin {
 public:
  // ev: recorded on the main stream at a fork, on the side stream at the end of its work.
  SideJoin(cudaStream_t main, cudaStream_t side, const cudaEvent_t ev[2]) : main_(main), side_(side), ev_{ev[0], ev[1]} {}
  SideJoin(const SideJoin&) = delete;
  SideJoin& operator=(const SideJoin&) = delete;
  ~SideJoin() {
    if (state_ == kForked) side_done();
    if (state_ == kDone) join();
  }
  // What follows on the side stream waits for the main stream's work so far.
  void fork() {
    cudaEventRecord(ev_[0], main_);
    cudaStreamWaitEvent(side_, ev_[0], 0);
    state_ = kForked;
  }
  // The side stream's work is enqueued; the main stream may run beside it until join.
  void side_done() {
    cudaEventRecord(ev_[1], side_);
    state_ = kDone;
  }
  void join() {
    cudaStreamWaitEvent(main_, ev_[1], 0);
    state_ = kJoined;
  }

 private:
  enum { kJoined, kForked, kDone } state_ = kJoined;
  cudaStream_t main_, side_;
  cudaEvent_t ev_[2];
};

}  // namespace exa
