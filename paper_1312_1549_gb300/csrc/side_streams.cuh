// Streams beside a caller's, and the events between them.
#pragma once

#include <vector>

#include "omm_internal.cuh"

namespace omm {

// The caller's stream joins the side streams when their work is queued. Where a failing call leaves that out, they
// are synchronised before they go: the scratch they use returns to its pool in the order of the caller's stream
// alone, and another call could get it while they still read and write it.
struct Streams {
  std::vector<cudaEvent_t> events;
  std::vector<cudaStream_t> streams;
  bool joined = false;

  Streams() = default;
  Streams(const Streams&) = delete;
  Streams& operator=(const Streams&) = delete;
  ~Streams() {
    for (cudaStream_t s : streams) {
      if (!joined) cudaStreamSynchronize(s);
      cudaStreamDestroy(s);  // (work that is pending behind a join still runs)
    }
    for (cudaEvent_t e : events) cudaEventDestroy(e);
  }
  // a stream that starts after what `from` holds so far
  cudaStream_t fork(cudaStream_t from) {
    streams.reserve(streams.size() + 1);
    cudaStream_t s = nullptr;
    OMM_CUDA_TRY(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking));
    streams.push_back(s);
    wait(s, from);
    return s;
  }
  cudaEvent_t record(cudaStream_t st) {
    events.reserve(events.size() + 1);
    cudaEvent_t e = nullptr;
    OMM_CUDA_TRY(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    events.push_back(e);
    OMM_CUDA_TRY(cudaEventRecord(e, st));
    return e;
  }
  // `st` goes on after what `other` holds so far
  void wait(cudaStream_t st, cudaStream_t other) { OMM_CUDA_TRY(cudaStreamWaitEvent(st, record(other), 0)); }
  // `st` goes on after what every side stream holds; nothing is queued on them any more
  void join(cudaStream_t st) {
    for (cudaStream_t s : streams) wait(st, s);
    joined = true;
  }
};

}  // namespace omm
