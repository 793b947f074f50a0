// Internal interface of the range-partitioned merge of the workers' row lists (the sparse part
// of the server aggregation for up to 32 workers, and for up to 128 where the table is not too sparsely hit).
//
// Every worker's list of row ids ascends, so the part of it that falls into a range of R
// consecutive row ids is one contiguous piece, found by binary search.  One CTA takes one range:
// a table of R words (or R sets of words) in shared memory holds, for each row id of the range, the set of workers
// whose list contains it (one bit per worker).  Non-zero words, in order, ARE the merged list of
// distinct ids; the set bits of a word, in order, are the contributions of that row in ascending
// worker order.  No sort and no waiting on other CTAs, and nothing depends on how the ids are
// distributed: a range never holds more than R * K entries.
#pragma once
#include "common.cuh"

namespace antdt {

constexpr int kRangeMaxWorkers = 32;        // one bit per worker in a 32-bit word
constexpr int kRangeLog2 = 12;              // 4096 row ids per range (measured best of 1024..8192)
constexpr int kRangeMaxLog2 = 13;           // 8192 for tables beyond 2^30 rows (bounds the scratch)
constexpr int64_t kRangeMaxRanges = (int64_t)1 << (31 - kRangeMaxLog2);  // n_rows < 2^31

// log2 of the range width.  The wide ranges also serve an input that is sparse in the table
// (fewer than 64 entries per narrow range on average): a range CTA's cost is mostly its fixed part
// then, so half as many CTAs finish sooner.
inline int range_log2(int64_t n_rows, int64_t in_cap) {
  if (n_rows > ((int64_t)kRangeMaxRanges << kRangeLog2)) return kRangeMaxLog2;
  const int64_t narrow = (n_rows + ((int64_t)1 << kRangeLog2) - 1) >> kRangeLog2;
  return in_cap < 64 * narrow ? kRangeMaxLog2 : kRangeLog2;
}

// 33 to 128 workers: sets of two to four words, narrower ranges.  The merge's cost is the ranges' CTAs, 3 us (count) and
// 5 us (emit) for each wave of them, against the passes of a sort: taken where the ranges are one wave of CTAs, or hold
// 250 entries on average.  Server of two kernels, sorted (up to 1.8 M entries in one resident kernel) -> by ranges, with
// entries per range: 234 k of 90 workers over 1 M rows (240, one wave) 64 -> 56 us, 936 k of 64 over 2 M (480) 109 -> 82, of
// 90 over 2.5 M (383) 113 -> 94, 2.3 M of 40 over 5 M (480) 193 -> 168, 2.5 M of 64 over 10 M (260) 398 -> 389, 4.7 M of
// 100 over 5 M (960) 297 -> 295; but 936 k of 90 over 5 M (192) 118 -> 119, 2.7 M of 100 over 20 M (140) 592 -> 639.
// Above 10000 entries of room to a range (8 ns each in its one CTA) the sort is faster: 2.3 M of 57 over 110 k rows
// (22 k) 115 -> 190, where 73 workers' lists with room for 9.7 k go 144 -> 95.
// The boundaries cost K (P + 1) words, in the scratch of the sort (8 bytes an entry).
constexpr int kRangeWideWorkers = 128;
constexpr int kRangeWideLog2 = 10, kRangeWideMaxLog2 = 11;
constexpr int64_t kRangeWideWave = 8 * kNumSM, kRangeWideEntries = 250, kRangeWideMost = 10000;
inline int64_t ranges_of(int64_t n_rows, int log2) { return (n_rows + ((int64_t)1 << log2) - 1) >> log2; }
// Ranges twice as wide where a worker has fewer than two entries in one.
inline int range_wide_log2(int K, int64_t n_rows, int64_t in_cap) {
  return in_cap >= 2 * K * ranges_of(n_rows, kRangeWideLog2) ? kRangeWideLog2 : kRangeWideMaxLog2;
}
inline bool range_wide_wanted(int K, int64_t n_rows, int64_t in_cap) {
  if (K <= kRangeMaxWorkers || K > kRangeWideWorkers) return false;
  const int64_t P = ranges_of(n_rows, kRangeWideLog2);
  return (P <= kRangeWideWave || in_cap >= kRangeWideEntries * P) && in_cap <= kRangeWideMost * P &&
         2 * in_cap >= K * (ranges_of(n_rows, range_wide_log2(K, n_rows, in_cap)) + 1);
}

// Workers whose lists are ignored.
struct RangeDropped {
  uint32_t bits[kRangeWideWorkers / 32];
  __host__ __device__ bool has(int w) const { return (bits[w >> 5] >> (w & 31)) & 1u; }
};

struct RangeLayout {
  size_t bnd;       // int32 [K][P+1]  first entry of worker w at or after row id b*R
  size_t distinct;  // int32 [P]       distinct row ids in range b
  size_t base;      // int64 [P+1]     distinct row ids before range b; [P] = total
  size_t bytes;
};
// Sized for the largest table (the workspace query does not know n_rows).
RangeLayout range_layout(int K);

// Sets the kernel attributes of this path on the current device (idempotent).
void range_prepare_device();

// Merge order of the workers' lists, ready for the tile reduction (tile_reduce.cuh):
//   wuo_in [K+1] raw offsets (clamped to in_cap into wuo_out)
//   agg_ids [out_cap]   distinct row ids ascending;  n_agg = their number
//   n_entries [2]       {0, entries of the workers that count whose ids lie in the table}
//   src [in_cap]        position (in the concatenated lists) of the entry at each merge slot;
//                       slots ordered by (row id, worker)
//   head_bits           bit i set iff slot i is the first contribution of its row (zeroed here)
//   tile_first          index into agg_ids of the row that slot t*tile belongs to
//                       (up to 32 workers head_bits and tile_first may both be nullptr: a reader that
//                       goes by row_start needs neither)
//   (up to 32 workers)
//   row_start [out_cap+1] merge slot of the first contribution of each row of agg_ids, or nullptr
//   src_worker [in_cap] the worker of every merge slot (one byte), or nullptr
//   weights_host [K]    the workers' weights; the first kernel carries them to weights_dev [K]
//                       as a parameter (nullptr: the caller has put them there already)
//   bnd, distinct, base scratch of range_layout (up to 32 workers); for more: [K (P+1)], [P], [P+1]
void range_merge_order(const int32_t* uniq_ids, const int64_t* wuo_in, int64_t in_cap, int64_t n_rows,
                       int K, const RangeDropped& dropped, int32_t* agg_ids, int64_t* n_agg, int64_t out_cap,
                       int64_t* wuo_out, int64_t* n_entries, uint32_t* src, uint32_t* head_bits,
                       int32_t* tile_first, int tile, uint32_t* row_start, uint8_t* src_worker,
                       const float* weights_host,
                       float* weights_dev, int32_t* bnd, int32_t* distinct, int64_t* base, int32_t* status,
                       cudaStream_t s);

}  // namespace antdt
