// The sort of a small or mid-sized backward by one wave of CTAs that stay for the whole of it.
//
// The multi-kernel sort (segsort.cu) is a chain of 8 to 14 short launches; on a small or mid-sized
// batch each of them is a launch, a ramp and two or three memory round trips.  Here every CTA holds
// up to 12288 consecutive (row id, bag) pairs in registers:
//
//   before      the workers' ranges, the ids, and the bag of every occurrence: first occurrences are
//               marked in shared memory, a running maximum over the positions spreads the marks
//   per pass    (by row id) rank inside the warp, digit counters summed over the CTA's warps and
//               published; a barrier over the CTAs; everybody's counts give the first slot of every
//               digit; the pairs go to their slots, put in the order of their digits in shared memory
//               first so that a warp stores to a few lines; a second barrier; every CTA takes the pairs of
//               its own slots
//   last pass   (by worker) takes everything to the workers' own order.  It ranks the runs of equal
//               (worker, row) as well as the pairs: a run's rank among the runs of its worker is its
//               place in the worker's list of distinct rows, so the lists, the run starts, the head
//               bits and the tiles' first runs are written from here, with nothing left to do
//
// All workers are sorted by row as ONE array, so before the last pass the workers of a row stand in
// ascending order: those runs ARE the aggregation's merge order.  In a step it is written on the way
// and the merge's four kernels (agg_range.cu) are not needed.
//
// What a pass costs is the latency of its steps, 4 us in a cluster, 9 to 13 us with one CTA per SM; the
// cost that grows with the square of the CTAs (reading everybody's counts, 2 to 5 us) keeps them to one per SM.  Small
// inputs (up to 16 CTAs of 2048) run as one thread-block cluster: counts, pairs and barriers go through
// distributed shared memory (a barrier 0.7 us against 1.6).  Twice the threads in the one-CTA-per-SM form: the sort
// 2 us faster, a forward beside it 22 us slower.
// Measured (in brackets the kernels it replaced: sort, and merge order where a step makes it): 10 k
// occurrences of 4 workers over 80 k rows 14 us (37 + 35); 426 k of 8 over 26 M 47 us, 64 with a step's forward
// beside it (75 + 62); 1.2 M of one worker over 1 M 59 us (113).
//
// The CTAs wait for one another, so the launch is a cluster or a cooperative one (all CTAs resident
// or none started).  A wait through memory is bounded all the same (kSpinLimit) and raises
// ANTDT_ERR_TIMEOUT when it runs out.  What a CTA reads then may be anything, so every index that comes
// out of memory is masked or checked: digits and workers by their masks, slots, runs and rows by the
// lengths of the arrays.  A cluster's barrier is the hardware's, without a limit; every CTA of the
// cluster arrives at each of them.
#include <algorithm>
#include <mutex>

#include "index_math.cuh"
#include "residentsort.cuh"

namespace antdt {
namespace {

constexpr int kThreads = kResThreads;
constexpr int kWarps = kThreads / 32;
constexpr int kBins = kSortMaxBins;  // 512 = one bin per thread
constexpr int kClusterItems = kResClusterItems;
// Up to this many workers the pass by worker finds equal digits by match.any, beyond it by OR (see warp_rank).
// Backward of 10 k / 110 k / 1.2 M occurrences, match against OR: 4 workers 30.0 / 48.2 / 114.2 us against
// 30.2 / 48.2 / 114.7; 8 workers 31.0 / 47.5 / 121.1 against 31.0 / 47.7 / 120.9; 10 workers 31.4 / 46.1 / 121.5
// against 31.4 / 46.1 / 121.2; 16: 31.7 / 46.2 / 123.8 against 31.6 / 46.1 / 123.0; 32: 32.2 / 48.2 / 128.8
// against 31.9 / 48.2 / 127.1.
constexpr int kMatchWorkers = 8;
constexpr uint32_t kSpinLimit = 1u << 20;
static_assert(kBins == kThreads, "one digit per thread");

struct Wso { int64_t v[kResMaxWorkers + 1]; };

struct __align__(16) Smem {
  unsigned short wh[kWarps * kBins];      // per-warp digit counters, then their prefix over the warps
  uint32_t cnt[kBins];                    // a counter's sum over the CTAs
  uint32_t base[kBins];                   // first slot of every digit for this CTA
  uint32_t loc[kBins];                    // pairs of smaller digits in this CTA
  uint16_t row[kBins];                    // cluster form: this CTA's published counters
  uint32_t warp_a[kWarps], warp_b[kWarps];
  uint32_t warp_tot[kWarps];
  int64_t bound[kResMaxWorkers + 1];      // occurrence range of every worker

  // Behind the struct (smem_bytes), one after the other in the same place:
  __device__ uint32_t* mm() { return reinterpret_cast<uint32_t*>(this + 1); }    // while ranking: the lanes that
                                                                                 // hold a digit, per warp [kWarps * kBins]
  __device__ uint32_t* mark() { return reinterpret_cast<uint32_t*>(this + 1); }  // before the sort: first occurrences
                                                                                 // of the bags [chunk]
  __device__ uint2* stage() { return reinterpret_cast<uint2*>(this + 1); }       // after ranking: the pairs in the
                                                                                 // order of their digits; after the
                                                                                 // passes: this CTA's own [chunk]
  // cluster form, behind mm: the pairs of this CTA's slots [kClusterItems * kThreads]
  __device__ uint2* pairs() { return reinterpret_cast<uint2*>(mm() + kWarps * kBins); }
};
size_t smem_bytes(int chunk, bool cluster) {
  // the pass by worker: pairs, a word per pair, its masks (two times 128 workers at most)
  const size_t mm = 4 * (size_t)kWarps * kBins, tail = 12 * (size_t)chunk + 4 * (size_t)kWarps * 2 * kResMaxWorkers;
  return sizeof(Smem) + (cluster ? mm + 8 * (size_t)kClusterItems * kThreads : (tail > mm ? tail : mm));
}
static_assert(4 * kClusterItems * kThreads + 4 * kWarps * 2 * kResMaxWorkers <= 4 * kWarps * kBins,
              "cluster form: marks, or a word per pair and the masks of the pass by worker, end before pairs");

// ---- the cluster ----
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
// Address of a shared variable as seen in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t remote(const void* p, uint32_t rank) {
  uint32_t a = (uint32_t)__cvta_generic_to_shared(p), r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
__device__ __forceinline__ uint32_t ld_remote(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void st_remote2(uint32_t addr, uint32_t x, uint32_t y) {
  asm volatile("st.shared::cluster.v2.u32 [%0], {%1, %2};" ::"r"(addr), "r"(x), "r"(y) : "memory");
}

// Exclusive prefix sum over the block's 512 threads; *total (if not null) receives the sum.
__device__ __forceinline__ uint32_t block_scan(uint32_t v, uint32_t* warp_tot, uint32_t* total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint32_t incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  __syncthreads();  // an earlier scan's readers are done
  if (lane == 31) warp_tot[w] = incl;
  __syncthreads();
  const uint32_t x = lane < kWarps ? warp_tot[lane] : 0u;
  if (total) *total = __reduce_add_sync(0xffffffffu, x);
  return incl - v + __reduce_add_sync(0xffffffffu, lane < w ? x : 0u);
}

// Stable rank of every valid item among the items of its warp with the same digit; leaves the
// warp's digit counts in my_wh.  my_mm: a word per digit, the lanes that hold it.  Both zeroed by
// the caller.  Item i of lane l is element i*32 + l of the warp's `valid` leading elements.
// The lanes of equal digit find each other by an atomic OR of their lane bits.  match.any does the
// same in one instruction, but it takes time in proportion to the distinct values it finds, on a
// unit that the whole SM shares: 62 cycles of the SM per warp instruction for 32 spread digits
// against 10 for OR, read and clear (6 against 18 when there are only 4 distinct ones); nine votes
// take 23.
template <int IPT>
__device__ __forceinline__ void warp_rank(const uint32_t (&k)[IPT], int valid, int shift, uint32_t mask,
                                          unsigned short* my_wh, uint32_t* my_mm, unsigned short (&rank)[IPT]) {
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
#pragma unroll
  for (int i = 0; i < IPT; ++i) {
    if (IPT > 4 && i % 4 == 0 && i * 32 >= valid) break;
    const bool ok = i * 32 + lane < valid;
    const uint32_t d = (k[i] >> shift) & mask;
    if (ok) atomicOr(my_mm + d, 1u << lane);
    __syncwarp();
    unsigned m = 0;
    uint32_t old = 0;
    if (ok) {
      m = my_mm[d];
      old = my_wh[d];
    }
    __syncwarp();
    // every peer has read the mask and the counter; the first peer clears the one, bumps the other
    if (ok && (m & lt) == 0) {
      my_mm[d] = 0u;
      my_wh[d] = (unsigned short)(old + __popc(m));
    }
    __syncwarp();
    rank[i] = (unsigned short)(old + __popc(m & lt));
  }
}

// Barrier over the CTAs: of the cluster, or `target` arrivals on a counter in memory that only
// grows.  Orders their memory accesses.
__device__ __forceinline__ void grid_arrive(uint32_t* counter) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(counter, 1u);
  }
}
__device__ __forceinline__ void grid_wait(uint32_t* counter, uint32_t target, int32_t* status) {
  if (threadIdx.x == 0) {
    uint32_t x = 0;
    for (uint32_t n = 0; n < kSpinLimit; ++n) {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(x) : "l"(counter) : "memory");
      if (x >= target) break;
    }
    if (x < target) set_status(status, ANTDT_ERR_TIMEOUT);
  }
  __syncthreads();
}
template <bool CLUSTER>
__device__ __forceinline__ void all_barrier(uint32_t* counter, uint32_t target, int32_t* status) {
  if (CLUSTER) {
    cluster_arrive();
    cluster_wait();
  } else {
    grid_arrive(counter);
    grid_wait(counter, target, status);
  }
}

// Sums of the C published rows of counters and of those before `rank`, per counter (the
// returned values are those of counter threadIdx.x).  rows: 16-bit counters, kBins to a row, of
// which the first nb are used.
//   grid      a thread takes eight counters (one 16-byte load) of every 64th (or 32nd, ...) part of the
//             rows: this is the one step whose cost grows with the square of the CTAs
//   cluster   a thread takes two counters of every row, all rows requested at once, and adds them up as
//             they are packed (there are at most 2^15 pairs): no sums to meet in shared memory.  With the
//             grid's way a pass of 10 k pairs had 1.6 - 1.9 us of its 4.6 here; step 34.1 -> 30.7 us
template <bool CLUSTER>
__device__ __forceinline__ void sum_rows(Smem& S, const uint16_t* rows, uint32_t nb, int rank, int C,
                                         uint32_t& total, uint32_t& before) {
  const int tid = threadIdx.x;
  if (CLUSTER) {
    static_assert((int64_t)kResMaxCluster * kClusterItems * kThreads < 65536, "packed sums");
    if (2u * tid < nb) {
      uint32_t x[kResMaxCluster];
#pragma unroll
      for (int c = 0; c < kResMaxCluster; ++c)
        x[c] = c < C ? ld_remote(remote(reinterpret_cast<const uint32_t*>(S.row) + tid, (uint32_t)c)) : 0u;
      uint32_t t = 0, b = 0;
#pragma unroll
      for (int c = 0; c < kResMaxCluster; ++c) {
        t += x[c];
        b += c < rank ? x[c] : 0u;
      }
      S.cnt[2 * tid] = t & 0xffffu; S.cnt[2 * tid + 1] = t >> 16;
      S.base[2 * tid] = b & 0xffffu; S.base[2 * tid + 1] = b >> 16;
    }
    __syncthreads();
    total = tid < (int)nb ? S.cnt[tid] : 0u;
    before = tid < (int)nb ? S.base[tid] : 0u;
    return;
  }
  const int q = nb >= 16 ? (int)(nb >> 3) : 2;  // a power of two: 16-byte columns of a row
  const int col = tid & (q - 1), grp = tid / q, groups = kThreads / q;
  S.cnt[tid] = 0u;
  S.base[tid] = 0u;
  __syncthreads();
  uint32_t t[8], b[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) t[j] = b[j] = 0u;
  const uint4* p = reinterpret_cast<const uint4*>(rows) + col;
  constexpr int kRow = kBins / 8;  // uint4 per row
  for (int c0 = grp; c0 < C; c0 += 4 * groups) {
    uint4 x[4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
      x[i] = c0 + i * groups >= C ? make_uint4(0u, 0u, 0u, 0u) : __ldcg(p + (size_t)(c0 + i * groups) * kRow);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint32_t on = c0 + i * groups < rank ? 0xffffffffu : 0u;
      const uint32_t y[4] = {x[i].x, x[i].y, x[i].z, x[i].w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        t[2 * j] += y[j] & 0xffffu; t[2 * j + 1] += y[j] >> 16;
        b[2 * j] += y[j] & 0xffffu & on; b[2 * j + 1] += (y[j] >> 16) & on;
      }
    }
  }
#pragma unroll
  for (int j = 0; j < 8; ++j) {  // counter col*8 + j at [j][col]: neighbouring lanes, neighbouring banks
    if (t[j]) atomicAdd(&S.cnt[j * q + col], t[j]);
    if (b[j]) atomicAdd(&S.base[j * q + col], b[j]);
  }
  __syncthreads();
  const bool in = tid < 8 * q;
  total = in ? S.cnt[(tid & 7) * q + (tid >> 3)] : 0u;
  before = in ? S.base[(tid & 7) * q + (tid >> 3)] : 0u;
}

// First slot of every digit for this CTA: everybody's counts of smaller digits, then those of this
// digit in CTAs of smaller rank.  Grid: less the place of the digit's first pair among the CTA's own (S.loc).
template <bool CLUSTER>
__device__ __forceinline__ void digit_bases(Smem& S, const uint16_t* rows, uint32_t nb, int rank, int C) {
  uint32_t total, before;
  sum_rows<CLUSTER>(S, rows, nb, rank, C, total, before);
  const uint32_t ex = block_scan(threadIdx.x < nb ? total : 0u, S.warp_tot, nullptr);  // barriers inside
  if (threadIdx.x < nb) S.base[threadIdx.x] = ex + before - (CLUSTER ? 0u : S.loc[threadIdx.x]);
  __syncthreads();
}

// What a CTA asks for before it knows the workers' ranges: the offsets of kWindow bags around the
// place where its chunk begins if all bags are of equal length, a thread's share as 32-bit values
// (offsets outside [0, 2^31) become -1 or 2^31 - 1, which no valid offset is here).
constexpr int kWindowTurns = 4;
constexpr int kWindow = kWindowTurns * kThreads;
struct BagWindow {
  int64_t first;  // bag of turn 0, thread 0
  int32_t lo[kWindowTurns], hi[kWindowTurns];
};
__device__ __forceinline__ int32_t offset32(int64_t x) {
  return (int32_t)min(max(x, (int64_t)-1), (int64_t)0x7fffffff);
}
__device__ __forceinline__ void request_window(BagWindow& w, const ResidentSortArgs& a, int64_t g0) {
  const int64_t guess = (int64_t)((double)a.n_bags * (double)g0 / (double)a.nnz);
  w.first = max((int64_t)0, min(guess - kWindow / 4, a.n_bags - kWindow));
#pragma unroll
  for (int t = 0; t < kWindowTurns; ++t) {
    const int64_t b = min(w.first + t * kThreads + threadIdx.x, a.n_bags - 1);
    w.lo[t] = offset32(__ldg(a.bag_offsets + b));
    w.hi[t] = offset32(__ldg(a.bag_offsets + b + 1));
  }
}

// The bag of every occurrence of this CTA's chunk [g0, g0 + n_mine), n_mine > 0, of the occurrences
// [0, end).  S.mark must be zero over the chunk.
template <int IPT>
__device__ __forceinline__ void chunk_bags(Smem& S, const ResidentSortArgs& a, const BagWindow& win, int64_t end,
                                           int64_t g0, int n_mine, uint32_t (&v)[IPT]) {
  const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
  const int per = items_per_thread(a.chunk), wbase = wp * 32 * per, valid = min(max(n_mine - wbase, 0), 32 * per);
  const int32_t c0 = (int32_t)g0, c1 = (int32_t)g0 + n_mine;
  bool covered = true;  // the window holds every bag of the chunk
  if (tid == 0) covered = win.first == 0 || win.lo[0] <= c0;
  if (tid == kThreads - 1) covered = win.first + kWindow >= a.n_bags || win.hi[kWindowTurns - 1] >= c1;
  if (__syncthreads_and(covered ? 1 : 0)) {
#pragma unroll
    for (int t = 0; t < kWindowTurns; ++t) {
      const int64_t b = win.first + t * kThreads + tid;
      const int32_t from = max(win.lo[t], c0);
      if (b < a.n_bags && from < min(win.hi[t], c1)) S.mark()[from - c0] = (uint32_t)b + 1u;
    }
  } else {
    // last bag that begins at or before the chunk: near where bags of equal length would put it,
    // else by a search that looks at 512 offsets at a time
    int64_t lo_b = 0, hi_b = a.n_bags;  // offset(lo_b) <= g0 < offset(hi_b) for ascending offsets
    {
      const int64_t guess = (int64_t)((double)a.n_bags * (double)g0 / (double)end);
      const int64_t wl = max((int64_t)0, min(guess - kThreads / 2, a.n_bags - kThreads));
      const int64_t b = min(wl + tid, a.n_bags);
      const int c = __syncthreads_count(__ldg(a.bag_offsets + b) <= g0);
      if (c > 0 && c < kThreads) { lo_b = wl + c - 1; hi_b = lo_b + 1; }
      else if (c == 0) hi_b = wl;
      else lo_b = min(wl + kThreads - 1, a.n_bags - 1);
    }
    while (hi_b - lo_b > 1) {  // uniform over the block
      const int64_t step = (hi_b - lo_b + kThreads - 1) / kThreads;
      const int64_t b = min(lo_b + step * tid, hi_b);
      const int c = __syncthreads_count(b < hi_b && __ldg(a.bag_offsets + b) <= g0);
      lo_b = lo_b + step * max(c - 1, 0);
      hi_b = min(hi_b, lo_b + step);
    }
    constexpr int kBatch = 4;
    for (int64_t b0 = lo_b; b0 < a.n_bags; b0 += kBatch * kThreads) {
      int64_t lo[kBatch], hi[kBatch];
      bool past = false;
#pragma unroll
      for (int t = 0; t < kBatch; ++t) {
        const int64_t b = min(b0 + t * kThreads + tid, a.n_bags - 1);
        lo[t] = __ldg(a.bag_offsets + b);
        hi[t] = __ldg(a.bag_offsets + b + 1);
      }
#pragma unroll
      for (int t = 0; t < kBatch; ++t) {
        const int64_t b = b0 + t * kThreads + tid;
        const int64_t from = max(lo[t], g0);
        past |= lo[t] >= g0 + n_mine;
        if (b < a.n_bags && from < min(hi[t], g0 + n_mine)) S.mark()[from - g0] = (uint32_t)b + 1u;
      }
      if (__syncthreads_or(past ? 1 : 0)) break;
    }
  }
  {
    __syncthreads();
    uint32_t carry = 0;
#pragma unroll
    for (int i = 0; i < IPT; ++i) {
      if (IPT > 4 && i % 4 == 0 && i * 32 >= valid) break;
      // marks ascend, so the running maximum is the last mark so far
      const uint32_t x = i * 32 + lane < valid ? S.mark()[wbase + i * 32 + lane] : 0u;
      const unsigned marked = __ballot_sync(0xffffffffu, x != 0u), upto = marked & (0xffffffffu >> (31 - lane));
      const uint32_t own = __shfl_sync(0xffffffffu, x, 31 - __clz(upto | 1u));
      const uint32_t last = __shfl_sync(0xffffffffu, x, 31 - __clz(marked | 1u));
      v[i] = upto ? own : carry;
      carry = marked ? last : carry;
    }
    if (lane == 0) S.warp_tot[wp] = carry;
    __syncthreads();
    const uint32_t pre = max(1u, __reduce_max_sync(0xffffffffu, lane < wp ? S.warp_tot[lane] : 0u));
#pragma unroll
    for (int i = 0; i < IPT; ++i) {
      if (IPT > 4 && i % 4 == 0 && i * 32 >= valid) break;
      v[i] = max(v[i], pre) - 1u;
    }
  }
}

// Ranks of the CTA's items among those of equal digit: inside the warp (rk), the prefix over the
// warps (S.wh), and the CTA's count of every digit, stored to my_row; returned: those of digits 2 tid (low
// half) and 2 tid + 1.  clear: the masks have to be cleared (the ranking leaves them cleared).
template <int IPT>
__device__ __forceinline__ uint32_t rank_and_publish(Smem& S, const uint32_t (&k)[IPT], int valid, int shift, uint32_t nb,
                                                 uint16_t* my_row, unsigned short (&rk)[IPT], bool clear) {
  const int tid = threadIdx.x, wp = tid >> 5;
  __syncthreads();  // marks, counters and bases of the step before have been read
  const uint4 none = make_uint4(0u, 0u, 0u, 0u);
  for (uint32_t i = tid; i < kWarps * nb / 8; i += kThreads) reinterpret_cast<uint4*>(S.wh)[i] = none;
  if (clear)
    for (uint32_t i = tid; i < kWarps * nb / 4; i += kThreads) reinterpret_cast<uint4*>(S.mm())[i] = none;
  __syncthreads();
  warp_rank<IPT>(k, valid, shift, nb - 1u, S.wh + wp * nb, S.mm() + wp * nb, rk);
  __syncthreads();
  // two digits to a thread, as they are packed: a CTA holds fewer than 2^16 pairs
  uint32_t sum = 0;
  if (2u * tid < nb) {
    uint32_t* const wh2 = reinterpret_cast<uint32_t*>(S.wh) + tid;
    uint32_t t[kWarps];
#pragma unroll
    for (int i = 0; i < kWarps; ++i) t[i] = wh2[i * (nb / 2)];
#pragma unroll
    for (int i = 0; i < kWarps; ++i) {
      wh2[i * (nb / 2)] = sum;
      sum += t[i];
    }
  }
  if (tid < kBins / 2) reinterpret_cast<uint32_t*>(my_row)[tid] = sum;
  return sum;
}

// The passes by row id (the low key_bits of the keys) over the n pairs that C CTAs hold, ce to a CTA.
// Leaves this CTA with the pairs of its own slots in S.stage(), or in S.pairs(); the pairs of all slots can
// be read in `pairs`, or in the CTAs' S.pairs().  Returns the arrivals on the barrier's counter.
template <int IPT, bool CLUSTER>
__device__ __forceinline__ uint32_t sort_passes_by_row(Smem& S, uint32_t (&k)[IPT], uint32_t (&v)[IPT], int key_bits,
                                                       int64_t n, int64_t g0, int n_mine, int ce, int cta, int C,
                                                       uint2* pairs, uint16_t* hist, uint32_t* counter,
                                                       int32_t* status) {
  const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
  const int per = items_per_thread(ce), wbase = wp * 32 * per, valid = min(max(n_mine - wbase, 0), 32 * per);
  const int P = sort_passes(key_bits);
  uint16_t* const my_row = CLUSTER ? S.row : hist + (size_t)cta * kBins;
  // every CTA of a cluster arrives, but of the others only the C that hold pairs
  uint32_t arrivals = 0;
  int shift = 0;
  for (int p = 0; p < P; ++p) {
    const int bits = (key_bits - shift + (P - p) - 1) / (P - p);
    const uint32_t nb = 1u << bits, dmask = nb - 1u;
    unsigned short rk[IPT];
    const uint32_t count = rank_and_publish<IPT>(S, k, valid, shift, nb, my_row, rk, !CLUSTER || p == 0);
    arrivals += C;
    if (CLUSTER) {
      all_barrier<CLUSTER>(counter, arrivals, status);
      digit_bases<CLUSTER>(S, hist, nb, cta, C);
#pragma unroll
      for (int i = 0; i < IPT; ++i) {
        if (IPT > 4 && i % 4 == 0 && i * 32 >= valid) break;
        if (i * 32 + lane < valid) {
          const uint32_t d = (k[i] >> shift) & dmask;
          const uint32_t q = S.base[d] + S.wh[wp * nb + d] + rk[i];
          const uint32_t c = q / (uint32_t)ce;
          if (c < (uint32_t)C) st_remote2(remote(S.pairs() + (q - c * (uint32_t)ce), c), k[i], v[i]);
        }
      }
    } else {
      // While the others' counts arrive the pairs are put in the order of their digits in shared
      // memory, so that consecutive threads store to consecutive slots: a store of a warp touches the
      // lines of a few digits instead of 32.
      grid_arrive(counter);
      const uint32_t loc = block_scan((count & 0xffffu) + (count >> 16), S.warp_tot, nullptr);
      if (tid < kBins / 2) {
        S.loc[2 * tid] = loc;
        S.loc[2 * tid + 1] = loc + (count & 0xffffu);
      }
      __syncthreads();
      uint2* const stage = S.stage();
#pragma unroll
      for (int i = 0; i < IPT; ++i) {
        if (IPT > 4 && i % 4 == 0 && i * 32 >= valid) break;
        if (i * 32 + lane < valid) {
          const uint32_t d = (k[i] >> shift) & dmask;
          stage[S.loc[d] + S.wh[wp * nb + d] + rk[i]] = make_uint2(k[i], v[i]);
        }
      }
      grid_wait(counter, arrivals, status);
      digit_bases<CLUSTER>(S, hist, nb, cta, C);
#pragma unroll 4
      for (int j = tid; j < n_mine; j += kThreads) {
        const uint2 kv = stage[j];
        const uint32_t q = S.base[(kv.x >> shift) & dmask] + (uint32_t)j;
        if (q < (uint32_t)n) __stcg(pairs + q, kv);
      }
    }
    arrivals += C;
    all_barrier<CLUSTER>(counter, arrivals, status);
    shift += bits;
    if (p + 1 == P) break;
#pragma unroll
    for (int i = 0; i < IPT; ++i) {
      if (IPT > 4 && i % 4 == 0 && i * 32 >= valid) break;
      if (i * 32 + lane < valid) {
        const uint2 kv = CLUSTER ? S.pairs()[wbase + i * 32 + lane] : __ldcg(pairs + g0 + wbase + i * 32 + lane);
        k[i] = kv.x;
        v[i] = kv.y;
      }
    }
  }
  if (!CLUSTER) {
#pragma unroll 8
    for (int j = tid; j < n_mine; j += kThreads) S.stage()[j] = __ldcg(pairs + g0 + j);
  }
  __syncthreads();
  return arrivals;
}

// The pair before the CTA's first slot, g0 > 0 (for the one thread that has the first pair).
template <bool CLUSTER>
__device__ __forceinline__ uint2 pair_before(Smem& S, const uint2* pairs, int64_t g0, int ce, int cta) {
  if (!CLUSTER) return __ldcg(pairs + g0 - 1);
  const uint32_t at = remote(&S.pairs()[ce - 1], (uint32_t)cta - 1u);
  return make_uint2(ld_remote(at), ld_remote(at + 4));
}

// Keys are worker << key_bits | row; a row id outside the table becomes n_rows (key_bits holds it),
// which every reader skips.
template <int IPT, bool CLUSTER>
__global__ void __launch_bounds__(kThreads, (IPT <= 8 ? 2 : 1))
resident_sort_kernel(const __grid_constant__ ResidentSortArgs a, const __grid_constant__ StepMerge m,
                     const __grid_constant__ Wso wso) {
  pdl_wait();
  extern __shared__ __align__(16) unsigned char res_smem[];
  Smem& S = *reinterpret_cast<Smem*>(res_smem);
  const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
  const int K = a.n_workers, F = a.bags_per_sample, cta = blockIdx.x, ce = a.chunk;
  const bool merge = m.agg_ids != nullptr;
  const int64_t g0 = (int64_t)cta * ce;
  const int per = items_per_thread(ce), wbase = wp * 32 * per;

  // Everything whose address does not depend on the workers' ranges is requested at once: the kernel's
  // beginning is a chain of round trips to memory (backward of 1.2 M occurrences 189 -> 177 us, of 500 k
  // 75 -> 71, of 100 k 58 -> 55).
  uint32_t k[IPT], v[IPT];
#pragma unroll
  for (int i = 0; i < IPT; ++i) {
    if (IPT > 4 && i % 4 == 0 && i >= per) break;
    const int64_t g = g0 + wbase + i * 32 + lane;
    k[i] = g < a.nnz ? (uint32_t)__ldg(a.row_ids + g) : 0u;
  }
  BagWindow win;
  request_window(win, a, g0);
  const int64_t raw0 = wp == 0 && lane <= K ? __ldg(a.bag_offsets + wso.v[lane] * (int64_t)F) : 0;
  // the offsets ascend inside [0, nnz]: each CTA checks a share
  {
    const int64_t share = (a.n_bags + gridDim.x - 1) / gridDim.x;
    const int64_t b_end = min(a.n_bags, (cta + 1) * share);
    bool bad = false;
#pragma unroll 8
    for (int64_t b = cta * share + tid; b < b_end; b += kThreads) {
      const int64_t lo = __ldg(a.bag_offsets + b), hi = __ldg(a.bag_offsets + b + 1);
      bad |= lo < 0 || hi < lo || hi > a.nnz;
    }
    if (bad) set_status(a.status, ANTDT_ERR_BAD_OFFSETS);
  }
  for (int i = tid; i < ce; i += kThreads) S.mark()[i] = 0u;
  if (CLUSTER) {  // (otherwise the flag words had to be cleared before the launch anyway)
    for (int64_t i = (int64_t)cta * kThreads + tid; i < a.n_zero; i += (int64_t)gridDim.x * kThreads) a.zero[i] = 0u;
  }
  {  // the workers' ranges: ascending, inside [0, nnz], whatever the offsets hold
    if (wp == 0) {
      int64_t carry = 0;
      for (int i0 = 0; i0 <= K; i0 += 32) {
        const int i = i0 + lane;
        const int64_t raw = i0 == 0 ? raw0 : (i <= K ? __ldg(a.bag_offsets + wso.v[i] * (int64_t)F) : 0);
        if (cta == 0 && ((i == 0 && raw != 0) || (i == K && raw != a.nnz)))
          set_status(a.status, ANTDT_ERR_BAD_OFFSETS);
        int64_t x = max(raw, carry);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int64_t t = __shfl_up_sync(0xffffffffu, x, o);
          if (lane >= o) x = max(x, t);
        }
        carry = __shfl_sync(0xffffffffu, x, 31);
        if (i <= K) S.bound[i] = min(x, a.nnz);
      }
    }
    __syncthreads();
  }
  const int64_t n = S.bound[K];
  const int C = (int)((n + ce - 1) / ce);
  if (cta == 0) {
    if (tid <= K) a.seg_bounds[tid] = S.bound[tid];
    if (tid < K) a.worker_b[tid] = 1.0f / (float)(wso.v[tid + 1] - wso.v[tid]);  // inf for an empty worker: unused
    if (merge && tid < K) m.weights_dev[tid] = m.weights[tid];
    if (C == 0) {
      if (tid <= K) a.seg_runs[tid] = 0;
      if (tid == 0) {
        a.run_start[0] = 0;
        if (merge) { *m.n_agg = 0; m.n_entries[0] = 0; m.n_entries[1] = 0; }
      }
    }
  }
  // A CTA without pairs leaves, but a cluster's CTAs all stay (its barriers count every one).
  if (CLUSTER ? C == 0 : cta >= C) return;
  const int n_mine = (int)max((int64_t)0, min((int64_t)ce, n - g0));
  const int valid = min(max(n_mine - wbase, 0), 32 * per);
  uint32_t* const counter = a.flags;
  {
    bool bad_id = false;
    int w = valid > 0 ? min(interval_of(S.bound, K + 1, g0 + wbase), K - 1) : 0;
#pragma unroll
    for (int i = 0; i < IPT; ++i) {
      if (IPT > 4 && i % 4 == 0 && i * 32 >= valid) break;
      uint32_t id = k[i];
      k[i] = 0u;
      v[i] = 0u;
      if (i * 32 + lane < valid) {
        if (id >= (uint32_t)a.n_rows) {
          bad_id = true;
          id = (uint32_t)a.n_rows;
        }
        const int64_t g = g0 + wbase + i * 32 + lane;
        while (w < K - 1 && g >= S.bound[w + 1]) ++w;  // positions ascend
        k[i] = ((uint32_t)w << a.key_bits) | id;
      }
    }
    if (bad_id) set_status(a.status, ANTDT_ERR_ID_OUT_OF_RANGE);
  }
  if (n_mine > 0) chunk_bags<IPT>(S, a, win, n, g0, n_mine, v);

  uint16_t* const my_row = CLUSTER ? S.row : a.hist + (size_t)cta * kBins;
  uint32_t arrivals = sort_passes_by_row<IPT, CLUSTER>(S, k, v, a.key_bits, n, g0, n_mine, ce, cta, C, a.pairs, a.hist,
                                                       counter, a.status);

  // ---- runs of (row, worker) and of rows in merge order; by worker: ranks of the pairs and of the runs
  // among those of their worker ----
  // From here on everything is done once, so its code is short loops over the pairs in shared memory:
  // unrolled over pairs in registers it waited for its own instructions (1.2 M occurrences of one worker:
  // ranking by worker 29 k cycles where a second turn took 8 k; backward 167 -> 152 us).
  // counters of this pass: pairs of worker w at w, its runs at Kp + w; published besides: all runs, all rows
  const uint32_t row_mask = a.key_bits < 32 ? (1u << a.key_bits) - 1u : 0xffffffffu;
  const uint32_t Kp = 1u << a.worker_bits, kB = 2u * Kp;
  const uint2* const kv = CLUSTER ? S.pairs() : S.stage();
  uint32_t* const ranks = CLUSTER ? S.mm() : reinterpret_cast<uint32_t*>(S.stage() + ce);  // a pair's | its run's << 16
  uint32_t* const masks = ranks + ce;
  const unsigned lt = (1u << lane) - 1u;
  const uint32_t before_cta = tid == 0 && n_mine > 0 && g0 > 0 ? pair_before<CLUSTER>(S, a.pairs, g0, ce, cta).x : 0u;
  // pair j of this CTA: its key, whether it starts a run, whether it starts a row
  auto look = [&](int j, bool in, uint32_t& key, bool& head, bool& first) {
    key = in ? kv[j].x : 0u;
    const uint32_t prev = in && j > 0 ? kv[j - 1].x : before_cta;
    head = in && (g0 + j == 0 || prev != key);
    first = in && (g0 + j == 0 || ((prev ^ key) & row_mask) != 0u);
  };
  uint32_t heads_warp = 0, rows_warp = 0;
  for (uint32_t i = tid; i < kWarps * kB / 2; i += kThreads) reinterpret_cast<uint32_t*>(S.wh)[i] = 0u;
  if (K > kMatchWorkers)
    for (uint32_t i = tid; i < kWarps * kB; i += kThreads) masks[i] = 0u;
  __syncthreads();
  {
    unsigned short* const wh = S.wh + wp * kB;
    uint32_t* const mm = masks + wp * kB;
#pragma unroll 1
    for (int i = 0; i * 32 < valid; ++i) {
      const int j = wbase + i * 32 + lane;
      const bool ok = i * 32 + lane < valid;
      uint32_t key;
      bool h, r;
      look(j, ok, key, h, r);
      const uint32_t d = key_worker(key, a.key_bits, a.worker_bits);
      const unsigned heads = __ballot_sync(0xffffffffu, h), all = __ballot_sync(0xffffffffu, ok);
      heads_warp += __popc(heads);
      rows_warp += __popc(__ballot_sync(0xffffffffu, r));
      if (K == 1) {  // a pair's rank is its place, a run's the heads so far
        if (ok) ranks[j] = (uint32_t)(i * 32 + lane) | (heads_warp - __popc(heads) + __popc(heads & lt) + (h ? 1u : 0u)) << 16;
        continue;
      }
      unsigned peers = 0;
      uint32_t old = 0, old_h = 0;
      if (K <= kMatchWorkers) {
        if (ok) peers = __match_any_sync(all, d);
      } else {
        if (ok) atomicOr(mm + d, 1u << lane);
        __syncwarp();
        if (ok) peers = mm[d];
      }
      if (ok) {
        old = wh[d];
        old_h = wh[Kp + d];
      }
      __syncwarp();
      if (ok && (peers & lt) == 0) {
        if (K > kMatchWorkers) mm[d] = 0u;
        wh[d] = (unsigned short)(old + __popc(peers));
        wh[Kp + d] = (unsigned short)(old_h + __popc(peers & heads));
      }
      __syncwarp();
      // (runs: up to and with this pair's)
      if (ok) ranks[j] = (old + __popc(peers & lt)) | (old_h + __popc(peers & heads & lt) + (h ? 1u : 0u)) << 16;
    }
  }
  if (lane == 0) {
    S.warp_a[wp] = heads_warp;
    S.warp_b[wp] = rows_warp;
    if (K == 1) {
      S.wh[wp * kB] = (unsigned short)valid;
      S.wh[wp * kB + Kp] = (unsigned short)heads_warp;
    }
  }
  __syncthreads();
  const uint32_t wa = lane < kWarps ? S.warp_a[lane] : 0u, wb = lane < kWarps ? S.warp_b[lane] : 0u;
  const uint32_t heads_cta = __reduce_add_sync(0xffffffffu, wa), heads_pre = __reduce_add_sync(0xffffffffu, lane < wp ? wa : 0u);
  const uint32_t rows_cta = __reduce_add_sync(0xffffffffu, wb), rows_pre = __reduce_add_sync(0xffffffffu, lane < wp ? wb : 0u);
  if (tid < (int)kB) {
    uint32_t sum = 0;
    uint32_t t[kWarps];
#pragma unroll
    for (int i = 0; i < kWarps; ++i) t[i] = S.wh[i * kB + tid];
#pragma unroll
    for (int i = 0; i < kWarps; ++i) {
      S.wh[i * kB + tid] = (unsigned short)sum;
      sum += t[i];
    }
    my_row[tid] = (uint16_t)sum;
  } else {
    my_row[tid] = (uint16_t)(tid == (int)kB ? heads_cta : (tid == (int)kB + 1 ? rows_cta : 0u));
  }
  arrivals += C;
  all_barrier<CLUSTER>(counter, arrivals, a.status);
  {
    uint32_t total, before;
    sum_rows<CLUSTER>(S, a.hist, 2u * kB, cta, C, total, before);
    if (CLUSTER) cluster_arrive();  // the last look at another CTA's memory; nobody leaves before the wait
    // prefix over the workers' pairs, then over their runs (behind all n pairs)
    const uint32_t ex = block_scan(tid < (int)kB ? total : 0u, S.warp_tot, nullptr);
    const uint32_t own = tid < (int)Kp ? ex : ex - (uint32_t)n;
    S.base[tid] = tid < (int)kB ? own + before : before;
    S.cnt[tid] = tid < (int)kB ? own : total;
    __syncthreads();
  }
  const uint32_t n_runs = S.cnt[kB], n_rows_all = S.cnt[kB + 1];
  if (cta == 0) {
    if (tid < K) a.seg_runs[tid] = S.cnt[Kp + tid];
    if (tid == 0) {
      a.seg_runs[K] = n_runs;
      a.run_start[min((int64_t)n_runs, a.out_cap)] = n;
      if (n_runs > a.out_cap) set_status(a.status, ANTDT_ERR_CAPACITY);
      if (merge) {
        *m.n_agg = n_rows_all;
        m.n_entries[0] = 0;
        m.n_entries[1] = n_runs;
        if (n_rows_all > m.agg_cap) set_status(a.status, ANTDT_ERR_CAPACITY);
      }
    }
  }
  uint32_t mrun = S.base[kB] + heads_pre, mrow = S.base[kB + 1] + rows_pre;  // runs / rows before the warp
  const uint32_t tile_mask = (1u << a.tile_shift) - 1u;
#pragma unroll 1
  for (int i = 0; i * 32 < valid; ++i) {
    const int j = wbase + i * 32 + lane;
    const bool in = i * 32 + lane < valid;
    uint32_t key;
    bool h, r;
    look(j, in, key, h, r);
    const unsigned hb = __ballot_sync(0xffffffffu, h), rb = __ballot_sync(0xffffffffu, r);
    if (in) {
      const uint32_t w = key_worker(key, a.key_bits, a.worker_bits), row = key & row_mask, rank = ranks[j];
      const uint32_t q = S.base[w] + S.wh[wp * kB + w] + (rank & 0xffffu);
      const uint32_t u = S.base[Kp + w] + S.wh[wp * kB + Kp + w] + (rank >> 16) - 1u;  // its run in its worker's list
      if (q < (uint32_t)n) {
        a.sorted_occ[q] = kv[j].y;
        if ((q & tile_mask) == 0) a.tile_first[q >> a.tile_shift] = (int32_t)u;
        if (K == 1 && lane == 0) a.head_bits[q >> 5] = hb;  // q is the place in the row order: a whole word
        if (h) {
          if (K > 1) atomicOr(a.head_bits + (q >> 5), 1u << (q & 31));
          const uint32_t slot = mrun + __popc(hb & lt);
          if (u < a.out_cap) {
            a.uniq_ids[u] = (int32_t)row;
            a.run_start[u] = q;
          }
          if (merge && slot < m.src_cap) {
            m.src[slot] = u;
            m.src_worker[slot] = (uint8_t)w;
            if (r) {
              const uint32_t x = mrow + __popc(rb & lt);
              if (x < m.agg_cap) m.agg_ids[x] = (int32_t)row;
              if (x <= m.agg_cap) m.row_start[x] = slot;  // one more than rows: it ends the last one
            }
          }
        }
      }
    }
    mrun += __popc(hb);
    mrow += __popc(rb);
  }
  if (CLUSTER) cluster_wait();
}

// The merge order of the workers' row lists by the same passes: (row id, position in the concatenated
// lists) sorted by row id.  Positions are worker-major, so a row's entries stand in ascending worker
// order.  An entry of a dropped worker or with an id outside the table gets the key n_rows, sorts
// behind everything and counts for nothing.
// It serves small lists (a cluster: 9 k entries of 5 workers 16 us against 30 for the range merge's
// four kernels and two memsets) and lists of more than 32 workers.
template <int IPT, bool CLUSTER>
__global__ void __launch_bounds__(kThreads, (IPT <= 8 ? 2 : 1))
resident_merge_kernel(const __grid_constant__ ResidentMergeArgs a) {
  pdl_sync();
  extern __shared__ __align__(16) unsigned char res_smem[];
  Smem& S = *reinterpret_cast<Smem*>(res_smem);
  const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
  const int K = a.n_workers, cta = blockIdx.x, ce = a.chunk;
  if (CLUSTER)
    for (int64_t i = (int64_t)cta * kThreads + tid; i < a.n_zero; i += (int64_t)gridDim.x * kThreads) a.zero[i] = 0u;
  const int64_t g0 = (int64_t)cta * ce;
  const int per = items_per_thread(ce), wbase = wp * 32 * per;
  uint32_t k[IPT], v[IPT];
#pragma unroll
  for (int i = 0; i < IPT; ++i) {  // on their way while the bounds are read (past the lists' end: not used)
    if (IPT > 4 && i % 4 == 0 && i >= per) break;
    const int64_t g = g0 + wbase + i * 32 + lane;
    k[i] = g < a.in_cap ? (uint32_t)__ldg(a.uniq_ids + g) : 0u;
  }
  if (wp == 0) {  // ascending and inside [0, in_cap], whatever came in
    int64_t carry = 0;
    for (int i0 = 0; i0 <= K; i0 += 32) {
      const int i = i0 + lane;
      const int64_t raw = i <= K ? __ldg(a.wuo_in + i) : 0;
      if (cta == 0 && i == K && (raw < 0 || raw > a.in_cap)) set_status(a.status, ANTDT_ERR_CAPACITY);
      int64_t x = max(raw, carry);
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int64_t t = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x = max(x, t);
      }
      carry = __shfl_sync(0xffffffffu, x, 31);
      if (i <= K) S.bound[i] = min(x, a.in_cap);
    }
  }
  __syncthreads();
  const int64_t n = S.bound[K];
  const int C = (int)((n + ce - 1) / ce);
  if (cta == 0) {
    for (int i = tid; i <= K; i += kThreads) a.wuo_out[i] = S.bound[i];
    for (int i = tid; i < K; i += kThreads) a.weights_dev[i] = a.weights[i];
    if (C == 0 && tid == 0) { *a.n_agg = 0; a.n_entries[0] = 0; a.n_entries[1] = 0; }
  }
  if (CLUSTER ? C == 0 : cta >= C) return;
  const int n_mine = (int)max((int64_t)0, min((int64_t)ce, n - g0));
  const int valid = min(max(n_mine - wbase, 0), 32 * per);
  {
    bool bad_id = false;
    int w = 0;
#pragma unroll
    for (int i = 0; i < IPT; ++i) {
      if (IPT > 4 && i % 4 == 0 && i * 32 >= valid) break;
      const uint32_t id = k[i];
      k[i] = 0u;
      v[i] = 0u;
      if (i * 32 + lane < valid) {
        const int64_t g = g0 + wbase + i * 32 + lane;
        if (i == 0) w = min(interval_of(S.bound, K + 1, g), K - 1);
        while (w < K - 1 && g >= S.bound[w + 1]) ++w;
        const bool dropped = (a.dropped[w >> 5] >> (w & 31)) & 1u;
        bad_id |= !dropped && id >= (uint32_t)a.n_rows;
        k[i] = dropped || id >= (uint32_t)a.n_rows ? (uint32_t)a.n_rows : id;
        v[i] = (uint32_t)g;
      }
    }
    if (bad_id) set_status(a.status, ANTDT_ERR_ID_OUT_OF_RANGE);
  }
  uint32_t arrivals = sort_passes_by_row<IPT, CLUSTER>(S, k, v, a.key_bits, n, g0, n_mine, ce, cta, C, a.pairs, a.hist,
                                                       a.flags, a.status);
  // ---- rows; entries that count ----
  const uint2* const kv = CLUSTER ? S.pairs() : S.stage();  // short loops, as in the sort
  const uint2 before_cta = tid == 0 && n_mine > 0 && g0 > 0 ? pair_before<CLUSTER>(S, a.pairs, g0, ce, cta)
                                                            : make_uint2(0u, 0u);
  uint32_t rows_warp = 0, kept_warp = 0;
  {
    bool repeats = false;
#pragma unroll 1
    for (int i = 0; i * 32 < valid; ++i) {
      const int j = wbase + i * 32 + lane;
      const bool ok = i * 32 + lane < valid;
      const uint2 x = ok ? kv[j] : make_uint2(0u, 0u), p = ok && j > 0 ? kv[j - 1] : before_cta;
      const bool in = ok && x.x < (uint32_t)a.n_rows, r = in && (g0 + j == 0 || p.x != x.x);
      // the same row twice in one worker's list
      if (in && !r) repeats |= interval_of(S.bound, K + 1, p.y) == interval_of(S.bound, K + 1, x.y);
      rows_warp += __popc(__ballot_sync(0xffffffffu, r));
      kept_warp += __popc(__ballot_sync(0xffffffffu, in));
    }
    if (repeats) set_status(a.status, ANTDT_ERR_BAD_OFFSETS);
  }
  if (lane == 0) { S.warp_a[wp] = kept_warp; S.warp_b[wp] = rows_warp; }
  __syncthreads();
  const uint32_t wb = lane < kWarps ? S.warp_b[lane] : 0u;
  const uint32_t kept_cta = __reduce_add_sync(0xffffffffu, lane < kWarps ? S.warp_a[lane] : 0u);
  const uint32_t rows_cta = __reduce_add_sync(0xffffffffu, wb), rows_pre = __reduce_add_sync(0xffffffffu, lane < wp ? wb : 0u);
  uint16_t* const my_row = CLUSTER ? S.row : a.hist + (size_t)cta * kBins;
  if (tid < 16) my_row[tid] = (uint16_t)(tid == 0 ? kept_cta : (tid == 1 ? rows_cta : 0u));
  arrivals += C;
  all_barrier<CLUSTER>(a.flags, arrivals, a.status);
  {
    uint32_t total, before;
    sum_rows<CLUSTER>(S, a.hist, 16u, cta, C, total, before);
    if (CLUSTER) cluster_arrive();  // the last look at another CTA's memory; nobody leaves before the wait
    __syncthreads();
    if (tid < 2) { S.cnt[tid] = total; S.base[tid] = before; }
    __syncthreads();
  }
  if (cta == 0 && tid == 0) {
    *a.n_agg = S.cnt[1];
    a.n_entries[0] = 0;
    a.n_entries[1] = S.cnt[0];
    if (S.cnt[1] > a.out_cap) set_status(a.status, ANTDT_ERR_CAPACITY);
  }
  uint32_t mrow = S.base[1] + rows_pre;  // rows before the warp
  const uint32_t tile_mask = (1u << a.tile_shift) - 1u;
  const unsigned le = 0xffffffffu >> (31 - lane);
#pragma unroll 1
  for (int i = 0; i * 32 < valid; ++i) {
    const int j = wbase + i * 32 + lane;
    const bool ok = i * 32 + lane < valid;
    const uint2 e = ok ? kv[j] : make_uint2(0u, 0u);
    const uint32_t prev = ok && j > 0 ? kv[j - 1].x : before_cta.x;
    const bool in = ok && e.x < (uint32_t)a.n_rows, r = in && (g0 + j == 0 || prev != e.x);
    const unsigned rb = __ballot_sync(0xffffffffu, r);
    if (in) {
      const uint32_t slot = (uint32_t)(g0 + j);
      const uint32_t x = mrow + __popc(rb & le) - 1u;  // index of this entry's row
      a.src[slot] = e.y;
      if (a.src_worker) a.src_worker[slot] = (uint8_t)min(interval_of(S.bound, K + 1, e.y), K - 1);
      if (r) {
        if (x < a.out_cap) a.agg_ids[x] = (int32_t)e.x;
        if (a.row_start && x <= a.out_cap) a.row_start[x] = slot;  // one more than rows: it ends the last one
        if (a.head_bits) atomicOr(a.head_bits + (slot >> 5), 1u << (slot & 31));
      }
      if (a.tile_first && (slot & tile_mask) == 0) a.tile_first[slot >> a.tile_shift] = (int32_t)x;
    }
    mrow += __popc(rb);
  }
  if (CLUSTER) cluster_wait();
}

#define RESIDENT_DISPATCH(GO)                                   \
  do {                                                          \
    const int ipt = items_per_thread(f.chunk);                  \
    if (f.cluster && ipt <= 2) GO(2, true);                     \
    if (f.cluster) GO(4, true);                                 \
    if (ipt <= 4) GO(4, false);                                 \
    if (ipt <= 8) GO(8, false);                                 \
    if (ipt <= 16) GO(16, false);                               \
    GO(24, false);                                              \
  } while (0)
static_assert(kResSMs == kNumSM, "one CTA per SM");

template <typename... P, typename... A>
int32_t launch_one(const char* name, cudaEvent_t started, void (*kernel)(P...), const ResidentForm& f, cudaStream_t s,
                   const A&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)f.ctas);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem_bytes(f.chunk, f.cluster);
  cfg.stream = s;
  cudaLaunchAttribute at[3];
  if (f.cluster) {
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)f.ctas;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
  } else {
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
  }
  cfg.attrs = at;
  cfg.numAttrs = 1;
  if (started) {
    cudaLaunchAttribute& e = at[cfg.numAttrs++];
    e.id = cudaLaunchAttributeLaunchCompletionEvent;
    e.val.launchCompletionEvent.event = started;
    e.val.launchCompletionEvent.flags = 0;
  }
  if (f.cluster && t_pdl) at[cfg.numAttrs++] = pdl_attribute();
  const int tok = prof_begin(name, s);
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, args...);
  prof_end(tok, s);
  if (e == cudaSuccess) return ANTDT_OK;
  // The limits are those of the process; a stream may have fewer SMs (a green context's).
  if (e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorInvalidClusterSize || e == cudaErrorLaunchOutOfResources ||
      e == cudaErrorInvalidConfiguration || e == cudaErrorNotSupported) {
    cudaGetLastError();
    prof_refused(tok);
    return kResidentRefused;
  }
  return ANTDT_ERR_CUDA;
}

bool went_well(cudaError_t e) {
  if (e != cudaSuccess) cudaGetLastError();
  return e == cudaSuccess;
}
// CTAs of the largest cluster of `kernel` that can be launched; of a cooperative launch.
template <typename... P>
int most_in_cluster(void (*kernel)(P...), int items) {
  const size_t smem = smem_bytes(items * kThreads, true);
  if (!went_well(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem))) return 0;
  const bool wide = went_well(cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  for (int ctas = wide ? kResMaxCluster : 8; ctas > 0; ctas /= 2) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)ctas);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)ctas;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    int n = 0;
    if (went_well(cudaOccupancyMaxActiveClusters(&n, kernel, &cfg)) && n > 0) return ctas;
  }
  return 0;
}
template <typename... P>
int most_at_once(void (*kernel)(P...), int items, int sms) {
  const size_t smem = smem_bytes(items * kThreads, false);
  int per_sm = 0;
  if (!went_well(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) ||
      !went_well(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kThreads, smem)))
    return 0;
  return per_sm * sms;
}

ResidentLimits query_limits(int dev) {
  ResidentLimits lim = {};
  int sms = 0, coop = 0;
  if (went_well(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) &&
      went_well(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev))) {
    lim.cluster = std::min(std::min(most_in_cluster(resident_sort_kernel<2, true>, 2), most_in_cluster(resident_sort_kernel<4, true>, 4)),
                           std::min(most_in_cluster(resident_merge_kernel<2, true>, 2), most_in_cluster(resident_merge_kernel<4, true>, 4)));
#define FORM_LIMIT(I, IPT)                                                                   \
  static_assert(kResFormItems[I] == IPT, "the dispatch below");                              \
  if (coop) lim.ctas[I] = std::min(most_at_once(resident_sort_kernel<IPT, false>, IPT, sms), \
                                   most_at_once(resident_merge_kernel<IPT, false>, IPT, sms))
    FORM_LIMIT(0, 4);
    FORM_LIMIT(1, 8);
    FORM_LIMIT(2, 16);
    FORM_LIMIT(3, 24);
#undef FORM_LIMIT
  }
  return lim;
}

// Kernel attributes and limits of the current device, found on first use.
const ResidentLimits& resident_limits() {
  static std::once_flag once[64];
  static ResidentLimits lim[64];
  static const ResidentLimits none = {};
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
    cudaGetLastError();
    return none;
  }
  std::call_once(once[dev], [dev] { lim[dev] = query_limits(dev); });
  return lim[dev];
}

}  // namespace

void resident_sort_prepare_device() { resident_limits(); }

bool resident_sort_fits(int K, int64_t nnz, int64_t n_rows) {
  // worker and row in 32 bits
  return K <= kResMaxWorkers && bits_for(K) + bits_for(n_rows + 1) <= 32 && resident_holds(resident_limits(), nnz);
}

bool resident_sort_clears(int64_t nnz) { return resident_form(nnz).cluster; }

int32_t resident_sort(const ResidentSortArgs& args, const StepMerge* merge, const int64_t* wso_host, cudaStream_t s,
                      cudaEvent_t started) {
  ResidentSortArgs a = args;
  const ResidentForm f = resident_form(a.nnz);
  a.key_bits = bits_for(a.n_rows + 1);
  a.worker_bits = a.n_workers <= 32 ? 5 : bits_for(a.n_workers);
  a.chunk = f.chunk;
  resident_sort_prepare_device();
  Wso wso;
  for (int i = 0; i <= kResMaxWorkers; ++i) wso.v[i] = wso_host[i < a.n_workers ? i : a.n_workers];
  const StepMerge m = merge ? *merge : StepMerge{};
#define SORT_GO(IPT, CLUSTER) \
  return launch_one("resident_sort", started, resident_sort_kernel<IPT, CLUSTER>, f, s, a, m, wso)
  RESIDENT_DISPATCH(SORT_GO);
#undef SORT_GO
}

bool resident_merge_wanted(int K, int64_t in_cap, int64_t n_rows) {
  // Small lists, whatever the workers; else the range merge is as fast or faster up to 32 workers.
  return in_cap > 0 && K <= kResMaxWorkers && n_rows < (1ll << 31) - 1 && (K > 32 || resident_form(in_cap).cluster) &&
         resident_holds(resident_limits(), in_cap);
}

int32_t resident_merge(const ResidentMergeArgs& args, cudaStream_t s) {
  ResidentMergeArgs a = args;
  const ResidentForm f = resident_form(a.in_cap);
  a.key_bits = bits_for(a.n_rows + 1);
  a.chunk = f.chunk;
  resident_sort_prepare_device();
#define MERGE_GO(IPT, CLUSTER) return launch_one("resident_merge", (cudaEvent_t)nullptr, resident_merge_kernel<IPT, CLUSTER>, f, s, a)
  RESIDENT_DISPATCH(MERGE_GO);
#undef MERGE_GO
}

}  // namespace antdt
