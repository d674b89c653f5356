// Stream sets for the overlapping launches of a J/K build.  A bounded pool per
// device: kSets sets, created with the first handle and kept until exit.
#include "streams.h"

#include <mutex>

namespace fk {

namespace {

constexpr int kSets = 3;  // the last one is kept for graph captures
std::mutex g_mu;
StreamSet g_sets[64][kSets];
bool g_ready[64] = {false};

cudaError_t create_set(StreamSet &s, int dev) {
  int lo = 0, hi = 0;
  cudaError_t e = cudaDeviceGetStreamPriorityRange(&lo, &hi);
  for (int i = 0; i < kParStreams && e == cudaSuccess; ++i) {
    e = cudaStreamCreateWithPriority(&s.s[i], cudaStreamNonBlocking, i < kHiStreams ? hi : lo);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&s.join[i], cudaEventDisableTiming);
  }
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&s.fork, cudaEventDisableTiming);
  s.device = dev;
  return e;
}

int current_device() {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return -1;
  return dev;
}

}  // namespace

cudaError_t init_streams() {
  const int dev = current_device();
  if (dev < 0) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lk(g_mu);
  if (g_ready[dev]) return cudaSuccess;
  for (int k = 0; k < kSets; ++k) {
    cudaError_t e = create_set(g_sets[dev][k], dev);
    if (e != cudaSuccess) return e;
  }
  g_ready[dev] = true;
  return cudaSuccess;
}

StreamSet *lease_streams(cudaStream_t user) {
  const int dev = current_device();
  if (dev < 0) return nullptr;
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(user, &cs) != cudaSuccess) {
    cudaGetLastError();  // a legacy stream during another thread's capture: not our error to report
    return nullptr;
  }
  if (cs != cudaStreamCaptureStatusNone) return nullptr;
  unsigned long long id = 0;
  if (cudaStreamGetId(user, &id) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  std::lock_guard<std::mutex> lk(g_mu);
  if (!g_ready[dev]) return nullptr;
  StreamSet *sets = g_sets[dev];
  for (int k = 0; k < kSets - 1; ++k)  // the stream's own set: its last build is ordered before this one
    if (!sets[k].leased && sets[k].used && sets[k].owner == id) {
      sets[k].leased = true;
      return &sets[k];
    }
  for (int k = 0; k < kSets - 1; ++k) {
    StreamSet &s = sets[k];
    if (s.leased) continue;
    cudaError_t q = cudaSuccess;
    for (int i = 0; i < kParStreams && q == cudaSuccess && s.used; ++i) q = cudaEventQuery(s.join[i]);
    if (q != cudaSuccess) {
      cudaGetLastError();  // cudaErrorNotReady
      continue;
    }
    s.leased = s.used = true;
    s.owner = id;
    return &s;
  }
  return nullptr;
}

void return_streams(StreamSet *set) {
  if (!set) return;
  std::lock_guard<std::mutex> lk(g_mu);
  set->leased = false;
}

cudaError_t fork_streams(StreamSet *set, cudaStream_t user, unsigned mask) {
  cudaError_t e = cudaEventRecord(set->fork, user);
  for (int i = 0; i < kParStreams && e == cudaSuccess; ++i)
    if (mask >> i & 1u) e = cudaStreamWaitEvent(set->s[i], set->fork, 0);
  return e;
}

// Joins even after a failed launch, so that the user's stream never runs ahead
// of work already enqueued; the first error is returned.
cudaError_t join_streams(StreamSet *set, cudaStream_t user, unsigned mask) {
  cudaError_t first = cudaSuccess;
  for (int i = 0; i < kParStreams; ++i) {
    if (!(mask >> i & 1u)) continue;
    cudaError_t e = cudaEventRecord(set->join[i], set->s[i]);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(user, set->join[i], 0);
    if (first == cudaSuccess) first = e;
  }
  return first;
}

StreamSet *capture_streams() {
  const int dev = current_device();
  if (dev < 0) return nullptr;
  std::lock_guard<std::mutex> lk(g_mu);
  return g_ready[dev] ? &g_sets[dev][kSets - 1] : nullptr;
}

}  // namespace fk
