// A branch of work on a second stream: forked from the caller's stream, joined to it on every way out of the scope that made it.
// Event record / wait pairs only, so that fork and join are captured when the caller's stream is being captured.
#pragma once

#include <cuda_runtime.h>

namespace cafeq {

class SideBranch {
 public:
  // what is enqueued on `side` from here on follows what `main` holds now
  bool fork(cudaStream_t main, cudaStream_t side, cudaEvent_t fork_event, cudaEvent_t join_event) {
    main_ = main;
    side_ = side;
    join_ = join_event;
    if (cudaEventRecord(fork_event, main) != cudaSuccess || cudaStreamWaitEvent(side, fork_event, 0) != cudaSuccess) return false;
    open_ = true;
    return true;
  }
  // what is enqueued on `main` from here on follows what `side` holds now
  bool join() {
    if (!open_) return true;
    open_ = false;
    return cudaEventRecord(join_, side_) == cudaSuccess && cudaStreamWaitEvent(main_, join_, 0) == cudaSuccess;
  }
  SideBranch() = default;
  SideBranch(const SideBranch&) = delete;
  SideBranch& operator=(const SideBranch&) = delete;
  ~SideBranch() { join(); }

 private:
  cudaStream_t main_ = {}, side_ = {};
  cudaEvent_t join_ = {};
  bool open_ = false;
};

}  // namespace cafeq
