// Host-side resources of one call: CUDA events, side streams, and the pinned mailbox of the host thread.
//
// Side streams are kept per host thread between calls and lent to one call at a time: a call may return
// before its work is done (slse_qr), so a stream that still has work is lent again only for the caller's
// stream whose work that is (the new work comes behind it anyway), and at most kSideStreams of a priority
// exist.  Made and destroyed by each call they put the calls of several streams
// one behind the other: four QRs of 900 x 128 on four streams 2.20 ms so, 1.07 ms with streams
// that stay, 0.59 ms for one.  They belong to one context: another device's are destroyed, those of a
// context that has been reset are forgotten.  They are given back when the thread ends.
#pragma once

#include <cuda.h>

#include <vector>

#include "slse_internal.cuh"

namespace slse {

constexpr size_t kSideStreams = 4;

// The current context's id (0: none or unknown); a device that was reset has a context of another id.
inline unsigned long long context_id(bool make = true) {
  using Fn = CUresult (*)(CUcontext, unsigned long long *);
  static const Fn get = [] {
    void *fn = nullptr;
    cudaDriverEntryPointQueryResult q{};
    if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &fn, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      fn = nullptr;
    cudaGetLastError();
    return reinterpret_cast<Fn>(fn);
  }();
  unsigned long long id = 0;
  if (!get) return 0;
  if (get(nullptr, &id) == CUDA_SUCCESS) return id;
  // no context is current in this thread yet: the runtime makes its own
  if (make && cudaFree(nullptr) == cudaSuccess && get(nullptr, &id) == CUDA_SUCCESS) return id;
  cudaGetLastError();
  return 0;
}

// Stream calls on streams that are not being captured stay allowed while another one of the thread is.
struct RelaxedCapture {
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
  ~RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
};

struct HostRes {
  int dev = -1;
  unsigned long long ctx = 0;
  struct Side {
    cudaStream_t h, last;  // last: the caller's stream of the call that had it last
  };
  std::vector<Side> stream[2];  // lowest (default) and highest priority, not lent
  size_t made[2] = {0, 0};      // those and the lent ones
  DevState *box = nullptr;              // 4 states and the stop word behind them, pinned
  int box_dev = -1;
  unsigned long long box_ctx = 0;

  void forget(bool destroy) {
    for (int k = 0; k < 2; ++k) {
      if (destroy)
        for (const Side &v : stream[k]) cudaStreamDestroy(v.h);
      stream[k].clear();
      made[k] = 0;
    }
    cudaGetLastError();
  }
  ~HostRes() {
    const unsigned long long id = context_id(false);
    forget(id != 0 && id == ctx);
    if (box && id != 0 && id == box_ctx) cudaFreeHost(box);
    cudaGetLastError();
  }
  // makes the pool that of the current device and context; false: nothing is kept in this call
  bool bind() {
    int d = 0;
    if (cudaGetDevice(&d) != cudaSuccess) return false;
    const unsigned long long id = context_id();
    if (id == 0) return false;
    if (d != dev || id != ctx) {
      forget(d != dev && dev >= 0);
      dev = d;
      ctx = id;
    }
    return true;
  }
  DevState *mailbox() {
    int d = 0;
    if (cudaGetDevice(&d) != cudaSuccess) return nullptr;
    const unsigned long long id = context_id();
    if (box && d == box_dev && id != box_ctx) box = nullptr;  // went with its context
    if (!box) {
      if (cudaHostAlloc((void **)&box, 4 * sizeof(DevState) + 64, cudaHostAllocDefault) != cudaSuccess) box = nullptr;
      box_dev = d;
      box_ctx = id;
    }
    return box;
  }
  volatile unsigned *stop_word() { return mailbox() ? reinterpret_cast<volatile unsigned *>(box + 4) : nullptr; }
};

inline HostRes &host_res() {
  static thread_local HostRes r;
  return r;
}

// Events of one call (with timing, also where only waited for: the panels of a 1536 x 256 QR, which hand
// over by events, took 1.53 ms with cudaEventDisableTiming and take 1.31 so).
struct Events {
  std::vector<cudaEvent_t> ev;
  cudaEvent_t make() {
    cudaEvent_t e = nullptr;
    if (cudaEventCreate(&e) != cudaSuccess) return nullptr;
    ev.push_back(e);
    return e;
  }
  ~Events() {
    for (cudaEvent_t e : ev) cudaEventDestroy(e);
  }
};

// A side stream of one call, joined to the caller's stream (which waits for it) and given back at the
// end of the call, also on an early return.
struct SideStream {
  cudaStream_t h = nullptr, joined = nullptr;
  int slot = 0;
  bool kept = false;
  unsigned long long ctx = 0;
  // idle_only: h stays null when all streams of the thread have other work (else one more is made for the call)
  cudaError_t open(bool high, cudaStream_t caller, bool idle_only = false) {
    HostRes &r = host_res();
    slot = high ? 1 : 0;
    joined = caller;
    RelaxedCapture relaxed;
    kept = r.bind();
    ctx = r.ctx;
    if (kept) {
      std::vector<HostRes::Side> &v = r.stream[slot];
      for (int idle = 0; idle < 2; ++idle)
        for (size_t k = 0; k < v.size(); ++k)
          if (idle ? cudaStreamQuery(v[k].h) == cudaSuccess : v[k].last == caller) {
            h = v[k].h;
            v.erase(v.begin() + (ptrdiff_t)k);
            cudaGetLastError();
            return cudaSuccess;
          }
      cudaGetLastError();  // not ready is no error of the call
      if (r.made[slot] >= kSideStreams) kept = false;
    }
    if (!kept && idle_only) return cudaSuccess;
    int least = 0, greatest = 0;
    cudaError_t e = cudaDeviceGetStreamPriorityRange(&least, &greatest);
    if (e == cudaSuccess) e = cudaStreamCreateWithPriority(&h, cudaStreamNonBlocking, high ? greatest : least);
    if (e != cudaSuccess) h = nullptr;
    else if (kept) ++r.made[slot];
    return e;
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
    if (kept && r.ctx == ctx) r.stream[slot].push_back({h, joined});
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
