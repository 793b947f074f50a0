// Internal interface of the resident sort of the worker backward: for an input that the registers of
// one CTA per SM hold, everything between the ids and the segmented sum in ONE kernel (bag expansion,
// id check, stable sort by row id inside each worker, distinct rows, run starts, head bits, first
// run of each reduction tile), and on request the merge order of the aggregation.
#pragma once
#include "resident_form.cuh"
#include "segsort.cuh"

namespace antdt {

constexpr int kResMaxWorkers = 128;

struct ResidentSortArgs {
  const int32_t* row_ids; int64_t nnz;
  const int64_t* bag_offsets; int64_t n_bags; int bags_per_sample;
  int64_t n_rows; int n_workers;
  int64_t* seg_bounds;    // out [K+1] occurrence range of every worker (sanitised)
  float* worker_b;        // out [K]   1/b_w
  uint32_t* sorted_occ;   // out [nnz]
  int32_t* uniq_ids; int64_t* run_start; int64_t* seg_runs; int64_t out_cap;
  uint32_t* head_bits; int32_t* tile_first; int tile_shift;
  uint32_t* flags;        // kResFlagWords words
  // head bits, flag words and whatever else the caller wants zeroed, as one piece: zeroed by the
  // caller on the stream before, unless resident_sort_clears(nnz)
  uint32_t* zero; int64_t n_zero;
  uint2* pairs;           // [nnz] scratch: (key, bag) between two passes
  uint16_t* hist;         // [kNumSM * 512] scratch
  int32_t* status;
  int key_bits, worker_bits, chunk;  // set by resident_sort
};
constexpr size_t kResFlagWords = 4;

// Where the merge order of a step's aggregation goes (see agg_range.cuh for the arrays), when the
// sort of the step's backward makes it on the way.
constexpr int kStepMergeWorkers = 32;
struct StepMerge {
  int32_t* agg_ids; int64_t* n_agg; int64_t agg_cap;
  int64_t* n_entries; uint32_t* src; uint8_t* src_worker; int64_t src_cap; uint32_t* row_start;
  float* weights_dev; float weights[kStepMergeWorkers];
};
// Fills m for a step of nnz occurrences whose aggregation will be given sp and ws; false: the step
// is not one for the resident sort, or the workspace has no room.  (aggregate.cu)
bool step_merge_targets(const antdt_sparse_part& sp, const int64_t* batch_sizes, int n_workers, int64_t nnz,
                        void* ws, size_t ws_bytes, StepMerge* m);

// Whether an input is one for this kernel on the current device, and whether it zeroes `zero` itself.
bool resident_sort_fits(int n_workers, int64_t nnz, int64_t n_rows);
bool resident_sort_clears(int64_t nnz);
void resident_sort_prepare_device();  // kernel attributes; before a stream capture
// started: recorded once every CTA of the sort has begun (best effort), or nullptr.  That can be before the
// work ahead of the sort on s is over (programmatic dependent launch): whoever goes by it waits for that too.
// kResidentRefused: the launch was refused and nothing runs (the stream has fewer SMs than the device); the
// caller takes the kernels of segsort.cuh or agg_range.cuh.
constexpr int32_t kResidentRefused = -1;
int32_t resident_sort(const ResidentSortArgs& a, const StepMerge* merge, const int64_t* wso_host, cudaStream_t s,
                      cudaEvent_t started = nullptr);

// The merge order of the workers' row lists alone (the arrays of agg_range.cuh), for small lists and
// for lists of 33 to 128 workers.
struct ResidentMergeArgs {
  const int32_t* uniq_ids; const int64_t* wuo_in; int64_t in_cap; int64_t n_rows; int n_workers;
  uint32_t dropped[kResMaxWorkers / 32];
  int32_t* agg_ids; int64_t* n_agg; int64_t out_cap; int64_t* wuo_out; int64_t* n_entries;
  uint32_t* src;
  uint32_t* head_bits; int32_t* tile_first; int tile_shift;  // for the tile reduction, or nullptr
  uint32_t* row_start; uint8_t* src_worker;                  // for the one-pass server step, or nullptr
  float* weights_dev; float weights[kResMaxWorkers];
  uint32_t* flags; uint32_t* zero; int64_t n_zero;           // as in ResidentSortArgs
  uint2* pairs; uint16_t* hist; int32_t* status;
  int key_bits, chunk;  // set by resident_merge
};
bool resident_merge_wanted(int n_workers, int64_t in_cap, int64_t n_rows);
int32_t resident_merge(const ResidentMergeArgs& a, cudaStream_t s);

}  // namespace antdt
