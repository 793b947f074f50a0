// See side_streams.cuh.
#include "side_streams.cuh"

#include <mutex>

namespace antdt {
namespace {

constexpr int kDevices = 64;

struct Slot {
  SideSet set;
  cudaStream_t owner;          // the stream its last work ran beside
  unsigned long long capture;  // id of the capture that its streams joined, 0: none
  bool ready, leased;
};
Slot g_slots[kDevices][kSideSets];
std::mutex g_mu;

// While one of these lives the thread may query and create streams although it captures one.
class RelaxedCapture {
 public:
  RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode_); }
  ~RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode_); }

 private:
  cudaStreamCaptureMode mode_ = cudaStreamCaptureModeRelaxed;
};

int current_device() {
  int dev = -1;
  return cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < kDevices ? dev : -1;
}

// Whether the capture that the slot's streams joined is still going on.
bool in_capture(Slot& t) {
  if (t.capture == 0) return false;
  for (cudaStream_t s : t.set.stream) {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone) return true;
  }
  t.capture = 0;
  return false;
}

bool idle(const Slot& t) {
  for (cudaStream_t s : t.set.stream) {
    const cudaError_t e = cudaStreamQuery(s);
    if (e == cudaErrorNotReady) cudaGetLastError();  // not an error
    if (e != cudaSuccess) return false;
  }
  return true;
}

void destroy(Slot& t) {
  for (cudaEvent_t e : t.set.event)
    if (e) cudaEventDestroy(e);
  for (cudaStream_t s : t.set.stream)
    if (s) cudaStreamDestroy(s);
  t = Slot{};
}

bool create(Slot& t) {
  t = Slot{};
  bool ok = true;
  for (cudaStream_t& s : t.set.stream) ok = ok && cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking) == cudaSuccess;
  for (cudaEvent_t& e : t.set.event) ok = ok && cudaEventCreateWithFlags(&e, cudaEventDisableTiming) == cudaSuccess;
  if (!ok) {
    cudaGetLastError();
    destroy(t);
    return false;
  }
  t.ready = true;
  return true;
}

}  // namespace

bool SideLease::take(cudaStream_t s) {
  release();
  const int dev = current_device();
  if (dev < 0) return false;
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  unsigned long long id = 0;
  if (cudaStreamGetCaptureInfo(s, &cs, &id) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  if (cs == cudaStreamCaptureStatusInvalidated) return false;
  if (cs == cudaStreamCaptureStatusNone) id = 0;
  // the per-thread default stream is another stream in every thread under one handle
  const bool known = s != cudaStreamPerThread;

  std::lock_guard<std::mutex> lk(g_mu);
  RelaxedCapture relaxed;
  int best = -1, empty = -1;
  for (int pass = 0; pass < 2 && best < 0; ++pass) {  // first the sets that cost no query
    for (int i = 0; i < kSideSets && best < 0; ++i) {
      Slot& t = g_slots[dev][i];
      if (!t.ready) {
        if (empty < 0) empty = i;
        continue;
      }
      if (t.leased) continue;
      const bool captured = in_capture(t);
      if (id != 0) {
        if (captured ? (pass == 0 && t.capture == id) : pass == 1) best = i;
      } else if (!captured) {
        if (pass == 0 ? (known && t.owner == s) : idle(t)) best = i;
      }
    }
  }
  if (best < 0 && id == 0 && empty >= 0 && create(g_slots[dev][empty])) best = empty;
  if (best < 0) return false;
  Slot& t = g_slots[dev][best];
  t.leased = true;
  t.capture = id;
  if (id == 0) t.owner = s;
  set_ = &t.set;
  dev_ = dev;
  slot_ = best;
  return true;
}

void SideLease::release() {
  if (!set_) return;
  std::lock_guard<std::mutex> lk(g_mu);
  g_slots[dev_][slot_].leased = false;
  set_ = nullptr;
}

void side_streams_prepare(int n) {
  const int dev = current_device();
  if (dev < 0) return;
  std::lock_guard<std::mutex> lk(g_mu);
  RelaxedCapture relaxed;
  for (Slot& t : g_slots[dev])
    if (t.ready && !t.leased && !in_capture(t)) --n;
  for (Slot& t : g_slots[dev])
    if (n > 0 && !t.ready && create(t)) --n;
}

void side_streams_free() {
  const int dev = current_device();
  if (dev < 0) return;
  std::lock_guard<std::mutex> lk(g_mu);
  RelaxedCapture relaxed;
  for (Slot& t : g_slots[dev])
    if (t.ready && !t.leased && !in_capture(t)) destroy(t);
}

}  // namespace antdt
