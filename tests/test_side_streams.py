"""Which side streams a call gets (csrc/side_streams.cu), against a fake of the CUDA calls it makes: streams
that have work left, captures that go on, more callers than sets."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2404_09679_b200", "csrc")

FAKE = r"""
#pragma once
#include <set>
struct FakeStream { bool busy = false; unsigned long long capture = 0; };
typedef FakeStream* cudaStream_t;
typedef int* cudaEvent_t;
enum cudaError_t { cudaSuccess = 0, cudaErrorNotReady = 600 };
enum cudaStreamCaptureStatus { cudaStreamCaptureStatusNone, cudaStreamCaptureStatusActive, cudaStreamCaptureStatusInvalidated };
enum cudaStreamCaptureMode { cudaStreamCaptureModeGlobal, cudaStreamCaptureModeThreadLocal, cudaStreamCaptureModeRelaxed };
enum { cudaStreamNonBlocking = 1, cudaEventDisableTiming = 2 };
#define cudaStreamPerThread ((cudaStream_t)2)
inline std::set<FakeStream*>& streams() { static std::set<FakeStream*> s; return s; }
inline int& events() { static int n; return n; }
inline cudaStreamCaptureMode& mode() { static cudaStreamCaptureMode m = cudaStreamCaptureModeGlobal; return m; }
inline int& errors() { static int n; return n; }
inline bool& any_capture() { static bool b; return b; }
// what a thread that captures must not do unless it has relaxed its mode
inline void unsafe() { if (any_capture() && mode() != cudaStreamCaptureModeRelaxed) ++errors(); }
inline cudaError_t cudaGetLastError() { return cudaSuccess; }
inline cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
inline cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode* m) {
  cudaStreamCaptureMode t = mode(); mode() = *m; *m = t; return cudaSuccess;
}
inline cudaError_t cudaStreamIsCapturing(cudaStream_t s, cudaStreamCaptureStatus* c) {
  *c = s->capture ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone; return cudaSuccess;
}
inline cudaError_t cudaStreamGetCaptureInfo(cudaStream_t s, cudaStreamCaptureStatus* c, unsigned long long* id) {
  *id = s->capture; return cudaStreamIsCapturing(s, c);
}
inline cudaError_t cudaStreamQuery(cudaStream_t s) {
  unsafe(); if (s->capture) ++errors(); return s->busy ? cudaErrorNotReady : cudaSuccess;
}
inline cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, int) { unsafe(); streams().insert(*s = new FakeStream); return cudaSuccess; }
inline cudaError_t cudaStreamDestroy(cudaStream_t s) { streams().erase(s); delete s; return cudaSuccess; }
inline cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, int) { ++events(); *e = new int; return cudaSuccess; }
inline cudaError_t cudaEventDestroy(cudaEvent_t e) { --events(); delete e; return cudaSuccess; }
"""

PROBE = r"""
#include "side_streams.cu"
#include <stdio.h>
using namespace antdt;
static int bad = 0;
#define EXPECT(x) do { if (!(x)) { printf("line %d: %s\n", __LINE__, #x); bad = 1; } } while (0)
// the set a call on s gets; work: leaves work on its streams
static const SideSet* use(cudaStream_t s, bool work = true) {
  SideLease l;
  if (!l.take(s)) return nullptr;
  const SideSet* p = l.operator->();
  for (cudaStream_t t : p->stream) { if (s->capture) t->capture = s->capture; else if (work) t->busy = true; }
  return p;
}
int main() {
  FakeStream a, b, caller[2 * kSideSets];
  // each caller its own set while there is work on it, the same one again for the same caller
  const SideSet* sa = use(&a);
  const SideSet* sb = use(&b);
  EXPECT(sa && sb && sa != sb && use(&a) == sa && use(&b) == sb && streams().size() == 4);
  // two calls being issued on one stream (two threads) do not share a set, and neither waits
  { SideLease x, y; EXPECT(x.take(&a) && y.take(&a) && x.operator->() != y.operator->()); }
  // an idle set goes to whoever asks: nothing new is made
  for (cudaStream_t t : sb->stream) t->busy = false;
  const size_t before = streams().size();
  EXPECT(use(caller) != nullptr && streams().size() == before);
  // more callers with work than sets: the late ones get none, until one is done
  side_streams_free();
  int got = 0;
  for (FakeStream& c : caller) got += use(&c) != nullptr;
  EXPECT(got <= kSideSets && streams().size() == 2 * kSideSets);
  FakeStream late;
  EXPECT(use(&late) == nullptr);
  const SideSet* s0 = nullptr;
  for (FakeStream& c : caller) if (!s0) s0 = use(&c);
  for (cudaStream_t t : s0->stream) t->busy = false;
  EXPECT(use(&late) == s0);
  for (cudaStream_t t : streams()) t->busy = false;
  side_streams_free();
  EXPECT(streams().empty() && events() == 0);
  // captures
  any_capture() = true;
  a.capture = 7;
  EXPECT(use(&a) == nullptr && streams().empty());       // nothing is made in a capture
  a.capture = 0;
  side_streams_prepare(2);
  EXPECT(streams().size() == 4);
  a.capture = 7;
  const SideSet* c7 = use(&a);
  EXPECT(c7 && use(&a) == c7);                           // a second step in the same capture
  { SideLease x, y; EXPECT(x.take(&a) && y.take(&a) && x.operator->() != y.operator->()); }
  FakeStream other; other.capture = 8;
  const SideSet* c8 = use(&other);
  EXPECT(c8 != c7);
  const SideSet* plain = use(&b);                        // plain calls go on meanwhile, on other sets
  EXPECT(plain && plain != c7 && plain != c8);
  const size_t alive = streams().size();
  for (cudaStream_t t : plain->stream) t->busy = false;
  side_streams_free();                                   // leaves what a capture holds
  EXPECT(streams().size() < alive && streams().count(c7->stream[0]));
  a.capture = other.capture = 0;
  for (cudaStream_t t : streams()) t->capture = 0;       // the captures end
  EXPECT(use(&a) != nullptr);
  for (cudaStream_t t : streams()) t->busy = false;
  side_streams_free();
  EXPECT(streams().empty() && events() == 0 && errors() == 0);
  return bad;
}
"""


def test_calls_on_different_streams_and_captures_share_no_set_in_use(tmp_path):
    (tmp_path / "cuda_runtime.h").write_text(FAKE)
    (tmp_path / "probe.cpp").write_text(PROBE)
    exe = str(tmp_path / "probe")
    subprocess.run(["g++", "-std=c++17", "-g", "-fsanitize=address,undefined", "-I", str(tmp_path), "-I", CSRC,
                    str(tmp_path / "probe.cpp"), "-o", exe, "-pthread"], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
