// Worker backward: per-worker dedup of row ids and segmented reduction of d_pooled rows to
// the worker's mean row gradients.
//
// Small and mid-sized inputs: everything up to the runs in one kernel (residentsort.cu).  Otherwise:
//   prep      occurrence range of every worker (from bag_offsets), 1/b_w scale, offset checks
//   expand    bag index of every occurrence (the sort's payload)
//   sort      stable radix sort by row id inside each worker's range     (segsort.cu)
//   runs      distinct rows, run starts, head bits, first run of each tile (segsort.cu)
//   reduce    tile-parallel segmented sum of gathered d_pooled rows        (bwd_walk.cuh)
//   fixup     rows whose occurrences leave a CTA's stretch of tiles: ordered sum of partials
//
// The reduction is balanced by occurrences, not by rows: a tile is 64 (small inputs: 16) consecutive
// sorted occurrences whatever rows they belong to, so a row that holds 20% of a field's
// occurrences costs its tiles no more than anyone else's.  Every sum has a fixed order (inside a
// tile by sorted position, across tiles by tile index), no floating-point atomics anywhere.
#include "index_math.cuh"
#include "residentsort.cuh"
#include "segsort.cuh"
#include "bwd_walk.cuh"

namespace antdt {
namespace {

size_t align_up(size_t x) { return (x + 255) & ~(size_t)255; }

struct BwdLayout {
  SortLayout sort;
  size_t sort_ws, wso, occ_bounds, worker_b, keys_a, keys_b, vals_t, flags_rs, head_bits, tile_first,
      head_part, tail_part, flags, tasks, bytes;
};

BwdLayout bwd_layout(int64_t nnz, int dim, int K, int tile_len) {
  BwdLayout L;
  L.sort = sort_layout(K);
  const size_t n = (size_t)(nnz > 0 ? nnz : 1);
  const size_t tile = (size_t)tile_len;
  const size_t n_tiles = (n + tile - 1) / tile;
  size_t o = 0;
  L.sort_ws = o;    o = align_up(o + L.sort.bytes);
  L.wso = o;        o = align_up(o + 8 * ((size_t)K + 1));
  L.occ_bounds = o; o = align_up(o + 8 * ((size_t)K + 1));
  L.worker_b = o;   o = align_up(o + 4 * (size_t)K);
  L.keys_a = o;     o = align_up(o + 4 * n);
  L.keys_b = o;     o = align_up(o + 4 * n);
  L.vals_t = o;     o = align_up(o + 4 * n);
  const size_t n_str = walk_stretches((int64_t)n, tile_len, dim);
  // what starts at zero, in one piece: flag words of the resident sort, head bits, task counter
  L.flags_rs = o;   o = align_up(o + 4 * kResFlagWords);
  L.head_bits = o;  o = align_up(o + 4 * head_bits_words((int64_t)n));
  L.tasks = o;      o = align_up(o + 4 * (2 * n_str + 4));
  L.tile_first = o; o = align_up(o + 4 * (n_tiles + 1));
  L.head_part = o;  o = align_up(o + 4 * n_str * (size_t)dim);
  L.tail_part = o;  o = align_up(o + 4 * n_str * (size_t)dim);
  L.flags = o;      o = align_up(o + n_str);
  L.bytes = o;
  return L;
}

// ---------------------------------------------------------------------------------------
__global__ void __launch_bounds__(1024)
bwd_prep_kernel(const int64_t* __restrict__ wso, int K, int F, const int64_t* __restrict__ bag_offsets,
                int64_t n_bags, int64_t nnz, int64_t* __restrict__ occ_bounds,
                float* __restrict__ worker_b, int32_t* status) {
  pdl_sync();
  const int tid = threadIdx.x;
  if (tid == 0 && (bag_offsets[0] != 0 || bag_offsets[n_bags] != nnz))
    set_status(status, ANTDT_ERR_BAD_OFFSETS);
  for (int w = tid; w <= K; w += blockDim.x) {
    const int64_t bag = wso[w] * (int64_t)F;  // host checked: 0 <= bag <= n_bags
    occ_bounds[w] = bag_offsets[bag];          // the sort setup clamps and orders these
    if (w < K) worker_b[w] = 1.0f / (float)(wso[w + 1] - wso[w]);  // 1/b_w (inf for an empty worker: unused)
  }
}

// One warp expands kExpandGroups x 32 consecutive bags: lane l holds the end offset of bag l of every
// group, all requested at once (the kernel is one dependent load and a stream of stores).
// The bags mark the slots that they begin in a window of shared memory, and a lane has the bags of four slots from a
// running maximum over the marks: one 16-byte store (the first and last few occurrences, off the 16-byte grid, go one by
// one).  The groups of a warp are one span, so the last turn of 128 slots is not spent on every group.
// Searching each four slots' bag among the lanes' ends, group by group, was bound by its instructions: 5.2 M bags, 105 M
// occurrences 130 -> 83 us, 6.6 M and 65 M 114 -> 76, 7.9 M and 35 M 99 -> 56.
constexpr int kExpandGroups = 4;
constexpr uint32_t kExpandWindow = 1024;
static_assert(32 * kExpandGroups < 256, "a mark is a byte");
__global__ void __launch_bounds__(256, 6)
expand_bags_kernel(const int64_t* __restrict__ bag_offsets, int64_t n_bags, int64_t nnz,
                   uint32_t* __restrict__ occ_bag, int32_t* status, uint32_t* __restrict__ zero_words,
                   int64_t n_zero_words, int32_t* __restrict__ zero_pair) {
  pdl_sync();
  const int lane = threadIdx.x & 31;
  const int64_t warp = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int64_t first_bag = warp * (32 * kExpandGroups);
  int64_t at[kExpandGroups + 1];  // offset of bag 32 g + lane (past the last bag: the end)
#pragma unroll
  for (int g = 0; g <= kExpandGroups; ++g)
    at[g] = __ldg(bag_offsets + min(first_bag + 32 * g + (g < kExpandGroups ? lane : 0), n_bags));
  // scratch that later kernels of the call expect zeroed (the run heads' bit mask, the fix-up's
  // task counter): cleared here, on the way, instead of by two memsets in the chain of launches
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_zero_words;
       i += (int64_t)gridDim.x * blockDim.x)
    zero_words[i] = 0u;
  if (blockIdx.x == 0 && threadIdx.x < 2 && zero_pair) zero_pair[threadIdx.x] = 0;
  uint32_t begin[kExpandGroups], end[kExpandGroups];  // of this lane's bag, where the group is not bad
  unsigned bad_groups = 0;
#pragma unroll
  for (int g = 0; g < kExpandGroups; ++g) {
    const int64_t next = __shfl_sync(0xffffffffu, at[g + 1], 0);
    int64_t hi = __shfl_down_sync(0xffffffffu, at[g], 1);
    if (lane == 31) hi = next;
    // skip the whole group; readers bound-check bag indices
    if (__any_sync(0xffffffffu, at[g] < 0 || hi < at[g] || hi > nnz)) bad_groups |= 1u << g;
    begin[g] = (uint32_t)at[g];
    end[g] = (uint32_t)hi;
  }
  if (bad_groups && lane == 0) set_status(status, ANTDT_ERR_BAD_OFFSETS);
  __shared__ __align__(16) uint8_t s_marks[8][kExpandWindow];
  uint8_t* const marks = s_marks[threadIdx.x >> 5];
  // the groups that `groups` has a bit for (a row of them, none bad)
  auto expand = [&](unsigned groups) {
    uint32_t first = 0, last = 0;
#pragma unroll
    for (int g = kExpandGroups - 1; g >= 0; --g) {
      const uint32_t lo = __shfl_sync(0xffffffffu, begin[g], 0), hi = __shfl_sync(0xffffffffu, end[g], 31);
      if (!((groups >> g) & 1u)) continue;
      first = lo;
      if (!((groups >> g) >> 1)) last = hi;
    }
    // the range starts this far into an aligned group of four; slots are counted from there
    const uint32_t skew = (uint32_t)(((reinterpret_cast<uintptr_t>(occ_bag) >> 2) + first) & 3);
    const BagSpan span(last - first, skew);                            // offsets lie in [0, nnz]
    uint32_t* const out = occ_bag + ((int64_t)first - (int64_t)skew);  // slot 0, on the 16-byte grid
    uint32_t carry = 0;                                                // mark of the bag that goes on
    for (uint32_t base = 0; base < span.total; base += kExpandWindow) {
      __syncwarp();
#pragma unroll
      for (uint32_t i = 0; i < kExpandWindow / 512; ++i)
        reinterpret_cast<uint4*>(marks)[i * 32 + lane] = make_uint4(0u, 0u, 0u, 0u);
      __syncwarp();
#pragma unroll
      for (int g = 0; g < kExpandGroups; ++g) {
        const uint32_t x = begin[g] - first + skew - base;  // from this window's start
        if (((groups >> g) & 1u) && end[g] > begin[g] && x < kExpandWindow) marks[x] = (uint8_t)(32 * g + lane + 1);
      }
      __syncwarp();
      for (uint32_t t = 0; t < kExpandWindow && base + t < span.total; t += kSpanTurn) {
        const uint32_t x = base + t + 4 * lane, q = *reinterpret_cast<const uint32_t*>(marks + t + 4 * lane);
        uint32_t m[4];
        m[0] = q & 255u; m[1] = max(m[0], q >> 8 & 255u); m[2] = max(m[1], q >> 16 & 255u); m[3] = max(m[2], q >> 24);
        uint32_t incl = m[3];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
          if (lane >= o) incl = max(incl, y);
        }
        uint32_t before = __shfl_up_sync(0xffffffffu, incl, 1);
        before = lane ? max(before, carry) : carry;
        carry = max(carry, __shfl_sync(0xffffffffu, incl, 31));
        const uint32_t b0 = (uint32_t)first_bag - 1u;
        const uint4 bags = make_uint4(b0 + max(m[0], before), b0 + max(m[1], before), b0 + max(m[2], before), b0 + max(m[3], before));
        if (span.whole(x)) {
          *reinterpret_cast<uint4*>(out + x) = bags;
        } else {
          if (span.holds(x)) out[x] = bags.x;
          if (span.holds(x + 1)) out[x + 1] = bags.y;
          if (span.holds(x + 2)) out[x + 2] = bags.z;
          if (span.holds(x + 3)) out[x + 3] = bags.w;
        }
      }
    }
  };
  constexpr unsigned kAll = (1u << kExpandGroups) - 1u;
#pragma unroll 1
  for (unsigned g = 0; g < kExpandGroups; ++g) {  // one span, or the good groups one by one
    if ((bad_groups >> g) & 1u) continue;
    expand(bad_groups ? 1u << g : kAll);
    if (!bad_groups) return;
  }
}

}  // namespace
}  // namespace antdt

extern "C" size_t antdt_embbag_bwd_dedup_workspace_bytes(int64_t nnz, int64_t n_bags, int32_t dim,
                                                         int32_t n_workers) {
  (void)n_bags;
  if (nnz < 0 || dim < 1 || n_workers < 1 || n_workers > antdt::kMaxSegments) return 0;
  return antdt::bwd_layout(nnz, dim, n_workers, antdt::red_tile_for(nnz, dim)).bytes;
}

extern "C" size_t antdt_embbag_bwd_dedup_min_workspace_bytes(int64_t nnz, int64_t n_bags, int32_t dim,
                                                             int32_t n_workers) {
  (void)n_bags;
  if (nnz < 0 || dim < 1 || n_workers < 1 || n_workers > antdt::kMaxSegments) return 0;
  return antdt::bwd_layout(nnz, dim, n_workers, antdt::kRedTile).bytes;
}

namespace antdt {
// The entry point's body.  d_pooled is first read by the tile reduction; a caller that is still
// copying it in on another stream passes the event that marks its arrival (the sort and the
// run detection, which only need the ids, then overlap the copy).
int32_t bwd_dedup_impl(
    const int32_t* row_ids, int64_t nnz, const int64_t* bag_offsets, int64_t n_bags,
    int32_t bags_per_sample, const float* d_pooled, int32_t dim, int64_t n_rows, int32_t n_workers,
    const int64_t* worker_sample_offsets, int32_t* uniq_ids, int64_t* worker_uniq_offsets,
    int64_t* seg_offsets, int32_t* sorted_occ, float* uniq_grads, int64_t out_cap, void* ws,
    size_t ws_bytes, int32_t* dev_status, void* stream, const PooledArrival* arrival,
    cudaEvent_t ids_done, const StepMerge* merge, bool* merge_made, cudaEvent_t sort_started, bool pdl_allowed) {
  const int K = n_workers;
  if (nnz < 0 || n_bags < 0 || nnz >= (1ll << 31) || n_bags >= (1ll << 31) || n_rows < 1 ||
      n_rows >= (1ll << 31) || dim < 4 || dim > 1024 || dim % 4 || K < 1 || K > kMaxSegments ||
      bags_per_sample < 1 || out_cap < 0)
    return ANTDT_ERR_INVALID_ARG;
  if (!bag_offsets || !worker_sample_offsets || !worker_uniq_offsets || !seg_offsets || !ws)
    return ANTDT_ERR_INVALID_ARG;
  if (nnz > 0 && (!row_ids || !d_pooled || !sorted_occ)) return ANTDT_ERR_INVALID_ARG;
  if (nnz > 0 && n_bags == 0) return ANTDT_ERR_INVALID_ARG;  // occurrences that belong to no bag
  if (out_cap > 0 && (!uniq_ids || !uniq_grads)) return ANTDT_ERR_INVALID_ARG;
  if (!aligned16(d_pooled) || !aligned16(uniq_grads) || !aligned16(ws)) return ANTDT_ERR_INVALID_ARG;
  if (worker_sample_offsets[0] != 0) return ANTDT_ERR_INVALID_ARG;
  for (int w = 0; w < K; ++w)
    if (worker_sample_offsets[w + 1] < worker_sample_offsets[w]) return ANTDT_ERR_INVALID_ARG;
  if (worker_sample_offsets[K] * (int64_t)bags_per_sample != n_bags) return ANTDT_ERR_INVALID_ARG;
  // short reduction tiles for a small input when the workspace has room for their partial sums,
  // the long tiles (the minimum workspace) otherwise
  int tile_len = red_tile_for(nnz, dim);
  BwdLayout L = bwd_layout(nnz, dim, K, tile_len);
  if (ws_bytes < L.bytes && tile_len != kRedTile) {
    tile_len = kRedTile;
    L = bwd_layout(nnz, dim, K, tile_len);
  }
  if (ws_bytes < L.bytes) return ANTDT_ERR_WORKSPACE_TOO_SMALL;

  cudaStream_t s = (cudaStream_t)stream;
  PdlScope pdl(pdl_allowed && nnz <= kPdlMaxItems);
  char* w8 = static_cast<char*>(ws);
  int64_t* d_wso = (int64_t*)(w8 + L.wso);
  int64_t* d_occ_bounds = (int64_t*)(w8 + L.occ_bounds);
  float* d_worker_b = (float*)(w8 + L.worker_b);
  uint32_t* keys_a = (uint32_t*)(w8 + L.keys_a);
  uint32_t* keys_b = (uint32_t*)(w8 + L.keys_b);
  uint32_t* vals_t = (uint32_t*)(w8 + L.vals_t);
  char* sort_ws = w8 + L.sort_ws;

  const int key_bits = bits_for(n_rows);
  bool scratch_zeroed = false;
  uint32_t* occ_out = reinterpret_cast<uint32_t*>(sorted_occ);
  bool resident = resident_sort_fits(K, nnz, n_rows);
  if (resident) {
    const size_t zero_bytes = L.tasks + 8 - L.flags_rs;
    if (!resident_sort_clears(nnz) && cudaMemsetAsync(w8 + L.flags_rs, 0, zero_bytes, s) != cudaSuccess)
      return ANTDT_ERR_CUDA;
    ResidentSortArgs q = {};
    q.row_ids = row_ids; q.nnz = nnz; q.bag_offsets = bag_offsets; q.n_bags = n_bags;
    q.bags_per_sample = bags_per_sample; q.n_rows = n_rows; q.n_workers = K;
    q.seg_bounds = (int64_t*)(sort_ws + L.sort.seg_bounds); q.worker_b = d_worker_b;
    q.sorted_occ = occ_out; q.uniq_ids = uniq_ids; q.run_start = seg_offsets;
    q.seg_runs = worker_uniq_offsets; q.out_cap = out_cap;
    q.head_bits = (uint32_t*)(w8 + L.head_bits); q.tile_first = (int32_t*)(w8 + L.tile_first);
    while ((1 << q.tile_shift) < tile_len) ++q.tile_shift;
    q.flags = (uint32_t*)(w8 + L.flags_rs);
    q.zero = q.flags; q.n_zero = (int64_t)(zero_bytes / 4);
    q.pairs = (uint2*)(w8 + L.keys_a);  // keys_a and keys_b lie side by side: 8 bytes per occurrence
    q.hist = (uint16_t*)(sort_ws + L.sort.hist);
    q.status = dev_status;
    const int32_t rc = resident_sort(q, merge, worker_sample_offsets, s, sort_started);
    if (rc != ANTDT_OK && rc != kResidentRefused) return rc;
    resident = scratch_zeroed = rc == ANTDT_OK;
  }
  if (merge_made) *merge_made = resident && merge;
  if (!resident) {
    // one launch for up to 255 workers; beyond that the offsets travel in pieces
    if (!segsort_setup_workers(worker_sample_offsets, K, (int)bags_per_sample, bag_offsets, n_bags, nnz,
                               d_worker_b, sort_ws, L.sort, dev_status, s)) {
      upload_small(worker_sample_offsets, 8 * ((size_t)K + 1), d_wso, s);
      ANTDT_LAUNCH("bwd_prep", bwd_prep_kernel, 1, 1024, 0, s, d_wso, K, (int)bags_per_sample,
                   bag_offsets, n_bags, nnz, d_occ_bounds, d_worker_b, dev_status);
      segsort_setup(d_occ_bounds, K, nnz, sort_ws, L.sort, s);
    }

    const int P = sort_passes(key_bits);
    // payload ping-pong ends in sorted_occ: start in whichever buffer makes the last pass land there
    uint32_t* expand_to = (P % 2 == 1) ? vals_t : occ_out;
    if (n_bags > 0 && nnz > 0) {
      const int64_t per_cta = 32 * 8 * kExpandGroups;
      const unsigned grid = (unsigned)((n_bags + per_cta - 1) / per_cta);
      ANTDT_LAUNCH("expand_bags", expand_bags_kernel, grid, 256, 0, s, bag_offsets, n_bags, nnz,
                   expand_to, dev_status, (uint32_t*)(w8 + L.head_bits), (int64_t)head_bits_words(nnz),
                   (int32_t*)(w8 + L.tasks));
      scratch_zeroed = true;
    }
    segsort_run(reinterpret_cast<const uint32_t*>(row_ids), expand_to, keys_a, occ_out, keys_b,
                vals_t, key_bits, n_rows, nnz, sort_ws, L.sort, dev_status, s);
    segsort_runs(keys_a, nnz, uniq_ids, seg_offsets, worker_uniq_offsets, nullptr, out_cap,
                 (uint32_t*)(w8 + L.head_bits), (int32_t*)(w8 + L.tile_first), tile_len, sort_ws,
                 L.sort, dev_status, s, false, scratch_zeroed);
  }
  if (ids_done && cudaEventRecord(ids_done, s) != cudaSuccess) return ANTDT_ERR_CUDA;
  if (nnz > 0) {
    TileArgs t;
    t.payload = occ_out;
    t.head_bits = (const uint32_t*)(w8 + L.head_bits);
    t.tile_first = (const int32_t*)(w8 + L.tile_first);
    t.tile = tile_len;
    t.rows = d_pooled;
    t.dim = dim;
    t.n_host = nnz;
    t.n_dev = nullptr;
    t.payload_limit = n_bags;
    t.bounds = (const int64_t*)(sort_ws + L.sort.seg_bounds);  // sanitised worker ranges
    t.scales = d_worker_b;
    t.K = K;
    t.out_cap = out_cap;
    t.out = uniq_grads;
    WalkScratch tasks;
    tasks.head_part = (float*)(w8 + L.head_part);
    tasks.tail_part = (float*)(w8 + L.tail_part);
    tasks.flags = (uint8_t*)(w8 + L.flags);
    tasks.tasks = (int32_t*)(w8 + L.tasks);
    tasks.tasks_zeroed = scratch_zeroed;
    if (!arrival || arrival->n < 1) {
      launch_bwd_walk(t, tasks, "seg_reduce_tiles", "seg_reduce_fixup", s);
    } else {
      // d_pooled is arriving piece by piece: a tile is walked as soon as the piece that holds
      // its last entry is there (the sort and the run detection above needed the ids only)
      const int64_t n_tiles = (nnz + tile_len - 1) / tile_len;
      const int64_t tps = walk_tiles_per_stretch(dim);
      int64_t done = 0;  // tiles issued so far
      t.fixup = false;
      for (int c = 0; c < arrival->n; ++c) {
        if (cudaStreamWaitEvent(s, arrival->ready[c], 0) != cudaSuccess) return ANTDT_ERR_CUDA;
        int64_t upto = n_tiles;  // the last piece takes every remaining tile
        if (c + 1 < arrival->n) {
          const int64_t e = arrival->entry_end[c];
          upto = e <= 0 ? 0 : (e >= nnz ? n_tiles : e / tile_len);  // tiles that end before entry e
          if (upto < n_tiles) upto = upto / tps * tps;              // a launch walks whole stretches
        }
        if (upto <= done) continue;
        t.tile_begin = done;
        t.tile_end = upto;
        launch_bwd_walk(t, tasks, "seg_reduce_tiles", "seg_reduce_fixup", s);
        done = upto;
      }
      t.walk = false;
      t.fixup = true;
      launch_bwd_walk(t, tasks, "seg_reduce_tiles", "seg_reduce_fixup", s);
    }
  }
  return cuda_ok();
}
}  // namespace antdt

extern "C" int32_t antdt_embbag_bwd_dedup(
    const int32_t* row_ids, int64_t nnz, const int64_t* bag_offsets, int64_t n_bags,
    int32_t bags_per_sample, const float* d_pooled, int32_t dim, int64_t n_rows, int32_t n_workers,
    const int64_t* worker_sample_offsets, int32_t* uniq_ids, int64_t* worker_uniq_offsets,
    int64_t* seg_offsets, int32_t* sorted_occ, float* uniq_grads, int64_t out_cap, void* ws,
    size_t ws_bytes, int32_t* dev_status, void* stream) {
  return antdt::bwd_dedup_impl(row_ids, nnz, bag_offsets, n_bags, bags_per_sample, d_pooled, dim,
                               n_rows, n_workers, worker_sample_offsets, uniq_ids,
                               worker_uniq_offsets, seg_offsets, sorted_occ, uniq_grads, out_cap, ws,
                               ws_bytes, dev_status, stream, nullptr);
}
