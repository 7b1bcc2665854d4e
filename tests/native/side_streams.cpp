// The side streams of the inverses on a fake CUDA runtime whose k-th call fails: when they go, the caller's
// stream has joined their work, or the host has waited for it.
#include <cstdio>
#include <map>
#include <set>

#include "side_streams.cuh"

namespace {
int calls, fails_at;
std::map<long, long> work;       // stream -> operations queued on it
std::map<long, long> waited;     // side stream -> operations that the caller's stream or the host waits for
std::map<long, std::pair<long, long>> events;  // event -> (stream, operations before it)
std::set<long> alive;
long next_id = 100;
bool lost;
const cudaStream_t kMain = (cudaStream_t)1;

bool failing() { return ++calls == fails_at; }
long id(const void* p) { return (long)p; }
}  // namespace

extern "C" {
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  if (failing()) return cudaErrorMemoryAllocation;
  alive.insert(++next_id);
  *s = (cudaStream_t)next_id;
  return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) {
  if (failing()) return cudaErrorMemoryAllocation;
  alive.insert(++next_id);
  *e = (cudaEvent_t)next_id;
  return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
  if (failing()) return cudaErrorUnknown;
  events[id(e)] = {id(s), work[id(s)]};
  return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
  if (failing()) return cudaErrorUnknown;
  if (s == kMain) waited[events[id(e)].first] = events[id(e)].second;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
  waited[id(s)] = work[id(s)];
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) {
  if (waited[id(s)] < work[id(s)]) lost = true;
  alive.erase(id(s));
  return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t e) {
  alive.erase(id(e));
  return cudaSuccess;
}
}

static void launch(cudaStream_t s) {
  ++work[id(s)];
  if (failing()) throw omm::CudaError{cudaErrorLaunchFailure, "launch"};
}

int main() {
  int bad = 0;
  for (fails_at = 0; fails_at < 40; ++fails_at) {
    calls = 0;
    lost = false;
    work.clear();
    waited.clear();
    events.clear();
    bool thrown = false;
    try {
      omm::Streams w;
      const cudaStream_t side = w.fork(kMain), ahead = w.fork(kMain);
      launch(kMain);
      w.wait(ahead, kMain);
      launch(ahead);
      const cudaEvent_t done = w.record(ahead);
      launch(kMain);
      OMM_CUDA_TRY(cudaStreamWaitEvent(kMain, done, 0));
      w.wait(side, kMain);
      launch(side);
      w.join(kMain);
      launch(kMain);
    } catch (const omm::CudaError&) {
      thrown = true;
    }
    if (lost || !alive.empty() || thrown != (fails_at > 0 && fails_at <= calls)) {
      std::printf("call %d fails: %s\n", fails_at, lost ? "work goes on that nobody waits for" : "leaks");
      ++bad;
    }
    alive.clear();
  }
  return bad != 0;
}
