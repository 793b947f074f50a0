// The form a resident sort takes for an input, and whether a device holds it.  Plain C++, tested on the host.
#pragma once
#include <stdint.h>

namespace antdt {

constexpr int kResThreads = 512;
constexpr int kResMaxItems = 24;     // pairs per thread
constexpr int kResMinChunk = 1024;   // pairs per CTA
constexpr int kResClusterItems = 4;  // pairs per thread of the cluster form
constexpr int kResMaxCluster = 16;
constexpr int kResSMs = 148;         // one CTA per SM

// Pairs per thread: every warp of a CTA takes an equal share of its chunk.
#ifdef __CUDACC__
__host__ __device__
#endif
constexpr int items_per_thread(int chunk) { return (chunk + kResThreads - 1) / kResThreads; }

// One cluster of up to 16 CTAs, or one CTA per SM; chunk: pairs per CTA.
struct ResidentForm { int ctas, chunk; bool cluster; };
inline ResidentForm resident_form(int64_t nnz) {
  ResidentForm f;
  f.cluster = nnz <= (int64_t)kResMaxCluster * kResClusterItems * kResThreads;
  const int64_t most = f.cluster ? kResMaxCluster : kResSMs;
  int64_t c = (nnz + most - 1) / most;
  c = (c + 31) & ~(int64_t)31;
  f.chunk = (int)(c < kResMinChunk ? kResMinChunk : c);
  f.ctas = (int)((nnz + f.chunk - 1) / f.chunk);
  if (f.cluster)
    while (f.ctas & (f.ctas - 1)) ++f.ctas;  // cluster sizes are powers of two; spare CTAs hold nothing
  return f;
}

// Kernels of the one-CTA-per-SM form, by pairs per thread.
constexpr int kResForms = 4;
constexpr int kResFormItems[kResForms] = {4, 8, 16, kResMaxItems};

// What a device (or the part of it that this process is given) holds at once.
struct ResidentLimits {
  int cluster;           // CTAs of the largest cluster that can be launched; 0: none
  int ctas[kResForms];   // CTAs of a cooperative launch; 0: none
};
inline bool resident_holds(const ResidentLimits& lim, int64_t nnz) {
  if (nnz < 1 || nnz > (int64_t)kResSMs * kResThreads * kResMaxItems) return false;
  const ResidentForm f = resident_form(nnz);
  if (f.cluster) return f.ctas <= lim.cluster;
  int i = 0;
  while (kResFormItems[i] < items_per_thread(f.chunk)) ++i;
  return f.ctas <= lim.ctas[i];
}

}  // namespace antdt
