// What belongs to a device is kept per device: a thread may use handles on
// several, and streams, events, kernel attributes and occupancies of one mean
// nothing on another. "Here" is the current device.
#pragma once
#include <cuda_runtime.h>

#include <atomic>
#include <map>

namespace cd {

inline int current_device() {
  int dev = 0;
  cudaGetDevice(&dev);
  return dev;
}

// A number per device, 0 at first: what a kernel's attributes and occupancy give
// holds for the device they were asked on. Every thread would set the same value.
class PerDevice {
  static constexpr int MAX_DEVICES = 64;  // past it nothing is kept
  std::atomic<int> v_[MAX_DEVICES] = {};

 public:
  int get() const {
    const int d = current_device();
    return d < MAX_DEVICES ? v_[d].load() : 0;
  }
  void set(int x) {
    const int d = current_device();
    if (d < MAX_DEVICES) v_[d].store(x);
  }
};

// A T per device, made on its device when first asked for (one thread's own, or
// under a lock).
template <class T>
class ByDevice {
  std::map<int, T> m_;

 public:
  T& here() { return m_[current_device()]; }
};

// The streams and events of the bins' concurrent scans. They belong to the
// calling host thread (created on its first use), so handles cost no stream
// creation and the server's worker threads never share them.
struct AuxStreams {
  cudaStream_t s[3] = {nullptr, nullptr, nullptr};
  cudaEvent_t fork = nullptr, join[3] = {nullptr, nullptr, nullptr};
  bool ok = false;
  AuxStreams() {
    ok = cudaEventCreateWithFlags(&fork, cudaEventDisableTiming) == cudaSuccess;
    for (int i = 0; i < 3 && ok; ++i)
      ok = cudaStreamCreateWithFlags(&s[i], cudaStreamNonBlocking) == cudaSuccess &&
           cudaEventCreateWithFlags(&join[i], cudaEventDisableTiming) == cudaSuccess;
    if (!ok) cudaGetLastError();
  }
};

inline AuxStreams& aux_streams() {
  static thread_local ByDevice<AuxStreams> a;
  return a.here();
}

// The calling thread's stream for captures on the current device.
inline cudaError_t capture_stream(cudaStream_t* out) {
  static thread_local ByDevice<cudaStream_t> streams;
  cudaStream_t& s = streams.here();
  const cudaError_t e = s ? cudaSuccess : cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
  *out = s;
  return e;
}

}  // namespace cd
