// Streams on which the independent launches of one J/K build overlap.
#pragma once

#include <cuda_runtime.h>

namespace fk {

// The launches of a build only add into J and K, so they may run in any order
// and at the same time.  kHiStreams carry the FP64 parts (high priority: few
// warps keep the FP64 pipe busy, so they are placed first and run beside the
// FP32-unit work), the others the two-float and FP32 parts.
constexpr int kHiStreams = 6, kLoStreams = 10, kParStreams = kHiStreams + kLoStreams;

struct StreamSet {
  cudaStream_t s[kParStreams] = {};
  cudaEvent_t fork = nullptr, join[kParStreams] = {};
  int device = -1;
  bool leased = false, used = false;
  unsigned long long owner = 0;  // id of the stream of the last build
};

// Creates the current device's sets if they do not exist yet (called when a
// handle is built, so that a build itself creates nothing).
cudaError_t init_streams();

// Event queries and stream-ordered allocations on any stream are among the calls
// that a global-mode capture (torch's default) forbids to every thread, and one
// such call breaks the capture.  A build makes them on streams that no capture
// sees; its thread is in relaxed mode meanwhile.
struct RelaxedCaptureMode {
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  RelaxedCaptureMode() { cudaThreadExchangeStreamCaptureMode(&mode); }
  ~RelaxedCaptureMode() { cudaThreadExchangeStreamCaptureMode(&mode); }
  RelaxedCaptureMode(const RelaxedCaptureMode &) = delete;
  RelaxedCaptureMode &operator=(const RelaxedCaptureMode &) = delete;
};

// A set for one build on `user`, or null when the build has to stay on that one
// stream: it is being captured, or every set is still busy with builds of other
// streams (sharing a set with another stream's unfinished build would order
// two streams that the caller keeps independent).  On one stream the launches
// follow one another: C20H42 83 against 72 ms (mixed 43 against 41), three waters
// 4.7 against 1.2 ms.  Called under a RelaxedCaptureMode.
StreamSet *lease_streams(cudaStream_t user);
void return_streams(StreamSet *set);

// Orders the set's streams (those with their bit in `mask`) after `user`, and
// `user` after them.
constexpr unsigned kAllStreams = (1u << kParStreams) - 1u;
cudaError_t fork_streams(StreamSet *set, cudaStream_t user, unsigned mask = kAllStreams);
cudaError_t join_streams(StreamSet *set, cudaStream_t user, unsigned mask = kAllStreams);

// A set of its own for one graph capture (serialised by the caller).
StreamSet *capture_streams();

}  // namespace fk
