// Streams of the library's own, for work that runs beside its caller's stream: the forward under the
// backward's sort, the merge order under the backward's sums, the dense sum under the sparse part.
//
// A call takes a set while it is being issued (SideLease) and never waits for one.  It gets the set whose
// last work came from the same stream (that is in order anyway), else one with nothing left to do, else a
// new one, at most kSideSets per device; failing that the lease is empty and the call issues everything on
// its caller's stream.  So calls on different streams wait for each other neither on the host nor on the
// GPU.  Inside a capture the set joins it and is nobody else's until the capture ends; nothing is created
// then.
#pragma once
#include <cuda_runtime.h>

namespace antdt {

constexpr int kSideSets = 8;

struct SideSet {
  cudaStream_t stream[2];
  cudaEvent_t event[5];  // an event's wait follows its record inside one lease
};

class SideLease {
 public:
  SideLease() = default;
  SideLease(const SideLease&) = delete;
  SideLease& operator=(const SideLease&) = delete;
  ~SideLease() { release(); }
  bool take(cudaStream_t s);  // for work beside s on the current device; false: no set
  void release();             // all of it has been issued and s waits for it
  explicit operator bool() const { return set_ != nullptr; }
  const SideSet* operator->() const { return set_; }

 private:
  const SideSet* set_ = nullptr;
  int dev_ = 0, slot_ = 0;
};

// Makes n sets that a capture could take, as far as the limit allows; before a capture.
void side_streams_prepare(int n);
// Gives the current device's sets back to the driver, except those in use.
void side_streams_free();

}  // namespace antdt
