// Host-side resources of the iteration loops, kept per host thread between calls: CUDA events (a
// 2nd-stage step used to create two and destroy them), the two side streams of a mixed fit, and a
// pinned mailbox.  Each thread has its own; they are bounded (kKeepEvents events, two streams, one
// page), belong to one device (another device's are destroyed when the thread changes device), and are
// given back when the thread ends.
#pragma once

#include <vector>

#include "slse_internal.cuh"

namespace slse {

constexpr size_t kKeepEvents = 256;

struct HostRes {
  int dev = -1;
  std::vector<cudaEvent_t> events;               // free events (with timing)
  cudaStream_t stream[2] = {nullptr, nullptr};   // free side streams: lowest (default) and highest priority
  DevState *box = nullptr;                       // 4 states and the stop word behind them, pinned

  void drop() {
    for (cudaEvent_t e : events) cudaEventDestroy(e);
    events.clear();
    for (cudaStream_t &h : stream) {
      if (h) cudaStreamDestroy(h);
      h = nullptr;
    }
  }
  ~HostRes() {
    drop();
    if (box) cudaFreeHost(box);
    cudaGetLastError();
  }
  // makes the pool that of the current device
  bool bind() {
    int d = 0;
    if (cudaGetDevice(&d) != cudaSuccess) return false;
    if (d != dev) {
      drop();
      cudaGetLastError();
      dev = d;
    }
    return true;
  }
  DevState *mailbox() {
    if (!box && cudaHostAlloc((void **)&box, 4 * sizeof(DevState) + 64, cudaHostAllocDefault) != cudaSuccess) box = nullptr;
    return box;
  }
  volatile unsigned *stop_word() { return mailbox() ? reinterpret_cast<volatile unsigned *>(box + 4) : nullptr; }
};

inline HostRes &host_res() {
  static thread_local HostRes r;
  return r;
}

// Events of one call: taken from the thread's pool (or created), given back at the end of the call.
struct Events {
  std::vector<cudaEvent_t> ev;
  bool ok = host_res().bind();
  cudaEvent_t make() {
    HostRes &r = host_res();
    cudaEvent_t e = nullptr;
    if (!ok) return nullptr;
    if (!r.events.empty()) {
      e = r.events.back();
      r.events.pop_back();
    } else if (cudaEventCreate(&e) != cudaSuccess) {
      return nullptr;
    }
    ev.push_back(e);
    return e;
  }
  ~Events() {
    HostRes &r = host_res();
    for (cudaEvent_t e : ev) {
      if (ok && r.events.size() < kKeepEvents) r.events.push_back(e);
      else cudaEventDestroy(e);
    }
  }
};

// A side stream of one call, joined to the caller's stream (which waits for it) and given back at the
// end of the call, also on an early return.
struct SideStream {
  cudaStream_t h = nullptr, joined = nullptr;
  int slot = 0;
  cudaError_t open(bool high, cudaStream_t caller) {
    HostRes &r = host_res();
    slot = high ? 1 : 0;
    joined = caller;
    if (!r.bind()) return cudaErrorUnknown;
    if (r.stream[slot]) {
      h = r.stream[slot];
      r.stream[slot] = nullptr;
      return cudaSuccess;
    }
    int least = 0, greatest = 0;
    const cudaError_t e = cudaDeviceGetStreamPriorityRange(&least, &greatest);
    if (e != cudaSuccess) return e;
    return cudaStreamCreateWithPriority(&h, cudaStreamNonBlocking, high ? greatest : least);
  }
  ~SideStream() {
    if (!h) return;
    cudaEvent_t e = nullptr;
    if (cudaEventCreateWithFlags(&e, cudaEventDisableTiming) == cudaSuccess) {
      cudaEventRecord(e, h);
      cudaStreamWaitEvent(joined, e, 0);
      cudaEventDestroy(e);
    }
    HostRes &r = host_res();
    if (!r.stream[slot]) r.stream[slot] = h;
    else cudaStreamDestroy(h);
  }
};

// Waits until the device has reported `iters` finished iterations or its stop flag (k_update writes
// the word); true: stopped.  The stream is queried now and then, so that a failed launch ends the wait.
inline cudaError_t wait_iterations(volatile unsigned *word, unsigned iters, cudaStream_t s, bool &stopped) {
  for (unsigned spin = 1;; ++spin) {
    const unsigned v = *word;
    stopped = (v & 1u) != 0u;
    if (stopped || (v >> 1) >= iters) return cudaSuccess;
    if ((spin & 0x3FFu) == 0) {
      const cudaError_t e = cudaStreamQuery(s);
      if (e == cudaSuccess) {  // everything has run: the word is final
        const unsigned w = *word;
        stopped = (w & 1u) != 0u || (w >> 1) < iters;
        return cudaSuccess;
      }
      if (e != cudaErrorNotReady) return e;
    }
  }
}

}  // namespace slse
