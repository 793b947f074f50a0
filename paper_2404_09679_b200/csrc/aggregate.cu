// Server aggregation: batch-size weighted sum of the workers' mean gradients.
//
// Sparse part, up to 32 workers: the range-partitioned merge of agg_range.cu (no sort).
// Sparse part, small lists, and up to 1.8 M entries of 33 to 128 workers: the resident merge
// (residentsort.cu).
// Sparse part, more: the workers' row lists (each ascending) are merged by one stable radix sort of
// (row id, position in the concatenated list); equal rows then sit together in ascending
// worker order, and the tile-parallel segmented reduction (tile_reduce.cuh) forms each row's
// weighted sum of its <= K contributions in that fixed order.  Because the sorted positions of
// one worker ascend with the row id, the gather of the workers' gradient rows is K
// forward-moving streams, not a random walk.
// Dense part: a K-way streaming reduction, one 16-byte vector per thread and worker; a large one
// beside a sort or a merge order takes a kernel that fits between their CTAs (dense_wsum_bulk_kernel).
#include "agg_range.cuh"
#include "opt_math.cuh"
#include "residentsort.cuh"
#include "segsort.cuh"
#include "tile_reduce.cuh"

namespace antdt {
namespace {

size_t align_up(size_t x) { return (x + 255) & ~(size_t)255; }

struct AggLayout {
  SortLayout sort;
  RangeLayout range;
  size_t range_ws;
  size_t sort_ws, bounds, weights, wuo, cwuo, drop, keys_a, keys_b, src, vals_t, run_start, flags, head_bits,
      tile_first, head_part, tail_part, row_start, src_worker, bytes;
};

AggLayout agg_layout(int64_t in_cap, int K, int dim) {
  AggLayout L;
  L.sort = sort_layout(1);
  const size_t n = (size_t)(in_cap > 0 ? in_cap : 1);
  size_t o = 0;
  L.sort_ws = o;   o = align_up(o + L.sort.bytes);
  L.bounds = o;    o = align_up(o + 16);
  L.weights = o;   o = align_up(o + 4 * (size_t)K);
  L.wuo = o;       o = align_up(o + 8 * ((size_t)K + 1));
  L.cwuo = o;      o = align_up(o + 8 * ((size_t)K + 1));
  L.drop = o;      o = align_up(o + 4 * (size_t)K);
  L.keys_a = o;    o = align_up(o + 4 * n);
  L.keys_b = o;    o = align_up(o + 4 * n);
  L.src = o;       o = align_up(o + 4 * n);
  L.vals_t = o;    o = align_up(o + 4 * n);
  L.run_start = o; o = align_up(o + 8 * (n + 1));
  const size_t tile = (size_t)red_tile_for((int64_t)n, dim);
  const size_t n_tiles = (n + tile - 1) / tile;
  // what the resident merge wants zeroed lies in one piece: its flag words, head bits, tile_first
  L.flags = o;      o = align_up(o + 4 * kResFlagWords);
  L.head_bits = o;  o = align_up(o + 4 * head_bits_words((int64_t)n));
  L.tile_first = o; o = align_up(o + 4 * (n_tiles + 1));
  L.head_part = o;  o = align_up(o + 4 * n_tiles * (size_t)dim);
  L.tail_part = o;  o = align_up(o + 4 * n_tiles * (size_t)dim);
  L.row_start = o;  o = align_up(o + 4 * (n + 1));
  L.src_worker = o; o = align_up(o + n + 1);
  L.range_ws = o;
  if (K <= kRangeMaxWorkers) {  // scratch of the range-partitioned merge (up to 32 workers)
    L.range = range_layout(K);
    o = align_up(o + L.range.bytes);
  }
  L.bytes = o;
  return L;
}

// bounds of the single sort segment = [0, total rows of all workers], clamped to the capacity
__global__ void agg_prep_kernel(const int64_t* __restrict__ wuo_in, int K, int64_t in_cap,
                                int64_t* __restrict__ bounds, int64_t* __restrict__ wuo,
                                int32_t* status) {
  pdl_sync();
  const int tid = threadIdx.x;
  for (int i = tid; i <= K; i += blockDim.x) {
    int64_t v = wuo_in[i];
    if (v < 0) v = 0;
    if (v > in_cap) v = in_cap;
    wuo[i] = v;
  }
  if (tid == 0) {
    int64_t n = wuo_in[K];
    if (n < 0 || n > in_cap) {
      set_status(status, ANTDT_ERR_CAPACITY);
      n = n < 0 ? 0 : in_cap;
    }
    bounds[0] = 0;
    bounds[1] = n;
  }
}

// Backup-workers variant: only the surviving workers' lists are merged.  prep computes where
// each survivor's list starts in the compacted concatenation, compact copies (row id, original
// position) of the survivors' entries there; the original position stays the payload, so the
// reduction finds rows and weights exactly as in the plain variant.
__global__ void agg_prep_backup_kernel(const int64_t* __restrict__ wuo_in, const uint32_t* __restrict__ drop,
                                       int K, int64_t in_cap, int64_t* __restrict__ bounds,
                                       int64_t* __restrict__ wuo, int64_t* __restrict__ cwuo,
                                       int32_t* status) {
  pdl_sync();
  if (threadIdx.x != 0) return;
  int64_t prev = 0, acc = 0;
  for (int i = 0; i <= K; ++i) {  // K <= 1024: a serial pass is enough
    int64_t v = wuo_in[i];
    v = v < prev ? prev : v;
    v = v > in_cap ? in_cap : v;
    wuo[i] = v;
    if (i > 0) {
      cwuo[i - 1] = acc;
      if (!drop[i - 1]) acc += v - prev;
    }
    prev = v;
  }
  cwuo[K] = acc;
  if (wuo_in[K] < 0 || wuo_in[K] > in_cap) set_status(status, ANTDT_ERR_CAPACITY);
  bounds[0] = 0;
  bounds[1] = acc;
}

__global__ void __launch_bounds__(256)
agg_compact_kernel(const int32_t* __restrict__ uniq_ids, const int64_t* __restrict__ wuo,
                   const int64_t* __restrict__ cwuo, const uint32_t* __restrict__ drop, int K,
                   uint32_t* __restrict__ keys_c, uint32_t* __restrict__ vals_c) {
  pdl_sync();
  extern __shared__ int64_t s_cw[];  // wuo [K+1], cwuo [K+1], then K drop flags
  int64_t* s_wuo = s_cw;
  int64_t* s_cwuo = s_cw + (K + 1);
  uint32_t* s_drop = reinterpret_cast<uint32_t*>(s_cw + 2 * (K + 1));
  for (int i = threadIdx.x; i <= K; i += blockDim.x) { s_wuo[i] = wuo[i]; s_cwuo[i] = cwuo[i]; }
  for (int i = threadIdx.x; i < K; i += blockDim.x) s_drop[i] = drop[i];
  __syncthreads();
  const int64_t n = s_wuo[K];
  const int64_t step = (int64_t)gridDim.x * blockDim.x;
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n; p += step) {
    int w = interval_of(s_wuo, K + 1, p);
    if (w > K - 1) w = K - 1;
    if (s_drop[w]) continue;
    const int64_t dst = s_cwuo[w] + (p - s_wuo[w]);
    keys_c[dst] = (uint32_t)uniq_ids[p];
    vals_c[dst] = (uint32_t)p;
  }
}

// dense_out[e] = sum_i w_i * g_i[e], ascending i, one float4 per thread; a worker of weight 0
// (empty or dropped) is not read at all.  The weights come from memory, or as a parameter.
constexpr int kDenseBlobWorkers = 128;
struct DenseWeights { float w[kDenseBlobWorkers]; };
__global__ void __launch_bounds__(256, 4)
dense_wsum_kernel(const float* __restrict__ grads, int64_t n4, int64_t stride,
                  const float* __restrict__ weights, const __grid_constant__ DenseWeights blob, int K,
                  float* __restrict__ out) {
  pdl_sync();
  extern __shared__ float s_wd[];
  for (int i = threadIdx.x; i < K; i += blockDim.x) s_wd[i] = weights ? weights[i] : blob.w[i];
  __syncthreads();
  constexpr int U = 8;  // loads in flight
  const int64_t step = (int64_t)gridDim.x * blockDim.x;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n4; e += step) {
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    const float* p = grads + 4 * e;
    int i = 0;
    for (; i + U <= K; i += U) {
      float4 v[U];
#pragma unroll
      for (int t = 0; t < U; ++t)
        v[t] = s_wd[i + t] != 0.f ? ldg_f4(p + (size_t)(i + t) * stride) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int t = 0; t < U; ++t) {
        const float w = s_wd[i + t];
        acc.x = fmaf(w, v[t].x, acc.x); acc.y = fmaf(w, v[t].y, acc.y);
        acc.z = fmaf(w, v[t].z, acc.z); acc.w = fmaf(w, v[t].w, acc.w);
      }
    }
    for (; i < K; ++i) {
      const float w = s_wd[i];
      if (w == 0.f) continue;
      const float4 v = ldg_f4(p + (size_t)i * stride);
      acc.x = fmaf(w, v.x, acc.x); acc.y = fmaf(w, v.y, acc.y);
      acc.z = fmaf(w, v.z, acc.z); acc.w = fmaf(w, v.w, acc.w);
    }
    reinterpret_cast<float4*>(out)[e] = acc;
  }
}

// The same sum by CTAs that fit beside three CTAs of the sort's scatter on an SM (four warps of 32
// registers, 48 KB of shared memory), for a side stream.  The loads in flight wait in shared memory
// instead of registers: a warp issues bulk copies of 3 KB per worker, four workers to a slot, into a
// ring of four slots, and three warps add up; slots change hands by mbarriers alone, because beside
// the sort's 48 warps every instruction in the chain from copy to copy counts (one thread issuing
// between block barriers moved 0.65 TB/s).  A slot's wait is for this CTA's own copies and warps; it
// is bounded all the same, and one that runs out raises TIMEOUT.
constexpr int kBulkThreads = 128;
constexpr int kBulkAdders = kBulkThreads - 32;  // the last warp issues the copies
constexpr int kBulkElems = 8 * kBulkAdders;     // floats of a tile
constexpr int kBulkGroup = 4;                   // workers per slot
constexpr int kBulkSlots = 4;
constexpr uint32_t kBulkSpin = 1u << 20;

__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
  for (uint32_t n = 0; n < kBulkSpin; ++n) {
    uint32_t ok;
    asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    if (ok) return true;
  }
  return false;
}

__global__ void __launch_bounds__(kBulkThreads, 16)
dense_wsum_bulk_kernel(const float* __restrict__ grads, uint32_t n, int64_t stride,
                       const __grid_constant__ DenseWeights blob, int K, float* __restrict__ out, int32_t* status) {
  pdl_sync();
  extern __shared__ __align__(128) float s_ring[];  // [slots][group][elems]
  __shared__ __align__(8) uint64_t s_full[kBulkSlots], s_empty[kBulkSlots];
  __shared__ float s_wt[kDenseBlobWorkers];
  const int tid = threadIdx.x, lane = tid & 31;
  const int groups = (K + kBulkGroup - 1) / kBulkGroup;
  for (int i = tid; i < groups * kBulkGroup; i += kBulkThreads) s_wt[i] = i < K ? blob.w[i] : 0.f;
  const uint32_t full = (uint32_t)__cvta_generic_to_shared(s_full), empty = (uint32_t)__cvta_generic_to_shared(s_empty);
  if (tid < kBulkSlots) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(full + 8u * tid) : "memory");
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(empty + 8u * tid), "r"(kBulkAdders / 32) : "memory");
  }
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  __syncthreads();
  const uint32_t tiles = (n + kBulkElems - 1) / kBulkElems;
  uint32_t slot = 0, parity = 0;
  if (tid >= kBulkAdders) {  // ---- copies: a lane per worker of the group ----
    bool first = true;
    for (uint32_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
      const uint32_t e0 = tile * kBulkElems, bytes = 4u * min((uint32_t)kBulkElems, n - e0);
      for (int g = 0; g < groups; ++g) {
        if (!first && !mbar_wait(empty + 8u * slot, parity ^ 1u)) {
          if (lane == 0) set_status(status, ANTDT_ERR_TIMEOUT);
          return;  // the adders' waits end too: every copy issued lands, the next never comes
        }
        const int w = g * kBulkGroup + lane;
        const bool on = lane < kBulkGroup && s_wt[lane < kBulkGroup ? w : 0] != 0.f;
        const uint32_t total = bytes * __popc(__ballot_sync(0xffffffffu, on));
        if (lane == 0)
          asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(full + 8u * slot), "r"(total)
                       : "memory");
        __syncwarp();
        if (on) {
          const uint32_t dst =
              (uint32_t)__cvta_generic_to_shared(s_ring) + 4u * kBulkElems * (slot * kBulkGroup + (uint32_t)lane);
          asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                       ::"r"(dst), "l"(grads + (int64_t)w * stride + e0), "r"(bytes), "r"(full + 8u * slot) : "memory");
        }
        if (++slot == kBulkSlots) { slot = 0; parity ^= 1u; first = false; }
      }
    }
  } else {  // ---- sums: two vectors of the tile per thread ----
    for (uint32_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
      float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
      for (int g = 0; g < groups; ++g) {
        if (!mbar_wait(full + 8u * slot, parity)) {
          if (lane == 0) set_status(status, ANTDT_ERR_TIMEOUT);
          for (int q = 0; q < kBulkSlots; ++q) {  // the copies in flight, with the same limit
            mbar_wait(full + 8u * slot, parity);
            if (++slot == kBulkSlots) { slot = 0; parity ^= 1u; }
          }
          return;
        }
        const float4* ring = reinterpret_cast<const float4*>(s_ring + (size_t)slot * kBulkGroup * kBulkElems);
#pragma unroll
        for (int j = 0; j < kBulkGroup; ++j) {
          const float w = s_wt[g * kBulkGroup + j];
          if (w == 0.f) continue;  // not copied
          const float4 x = ring[j * (kBulkElems / 4) + tid], y = ring[j * (kBulkElems / 4) + kBulkAdders + tid];
          a.x = fmaf(w, x.x, a.x); a.y = fmaf(w, x.y, a.y); a.z = fmaf(w, x.z, a.z); a.w = fmaf(w, x.w, a.w);
          b.x = fmaf(w, y.x, b.x); b.y = fmaf(w, y.y, b.y); b.z = fmaf(w, y.z, b.z); b.w = fmaf(w, y.w, b.w);
        }
        __syncwarp();
        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(empty + 8u * slot) : "memory");
        if (++slot == kBulkSlots) { slot = 0; parity ^= 1u; }
      }
      const uint32_t e = tile * kBulkElems + 4u * tid;
      if (e < n) *reinterpret_cast<float4*>(out + e) = a;
      if (e + 4u * kBulkAdders < n) *reinterpret_cast<float4*>(out + e + 4u * kBulkAdders) = b;
    }
  }
}

// Aggregation and update in one pass (up to 32 workers): a group of G lanes owns one aggregated
// row.  Its contributions are the merge slots [row_start[u], row_start[u+1]) in ascending worker
// order; the table and state vectors of the row are requested before the gather, the weighted sum
// is formed in that fixed order and goes straight into the Adagrad / Adam arithmetic, so the
// aggregated gradient is never written to or read back from memory (agg_out, if given, receives
// it all the same).  No partial sums, no second pass: a row has at most K contributions.
// Without a table (UPDATE false) it forms the sums alone, for lists so short that the tile reduction's
// second launch counts (sum_by_rows, and what the resident merge takes as a cluster).
struct FusedUpdate {
  void* table; int dtype; int opt; OptParams p; float* state0; float* state1; float* agg_out;
};

// Rows a lane group has in flight, CTAs per SM and the grid.  The kernel is a chain of dependent
// loads per row (slots -> positions -> gradient rows), so warps in flight count for more than
// loads in flight per warp, and the grid decides how close in time neighbouring rows are worked
// on.  Measured on B200 (100M x 64 bf16 table, Adagrad, 16 workers, 16.7 M contributions to 9.2 M
// rows; the two separate kernels take 2.73 ms): 1 row, 8 CTAs/SM, grid of 16 resident waves,
// parameters and state prefetched towards L2 before the sum and loaded after it 2.33 ms (loaded
// after it without the prefetch 2.42, loaded before it 2.58); 32 waves 2.58;
// 8 waves 2.62; 4 waves 2.74; 2 waves 2.88; 1 wave 2.95; one row per lane group and no stride
// 3.30; 6 CTAs/SM 3.05; 2 rows in flight 3.5-4.1; 4 rows 5.0.  Adam (fp32 rows, 16 and 32
// workers): 2.91 / 1.96 ms against 3.22 / 2.20 for the two kernels; at 6 CTAs/SM 3.26 / 2.30; the
// grid of 64 waves instead of 16: 2655 -> 2588 and 1769 -> 1746 us (32 waves 2611 / 1745, 8 waves
// 2732 / 1818), where Adagrad on the bf16 table goes 1619 -> 1653.
__device__ __forceinline__ void prefetch_l2(const void* p) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}
constexpr int kFusedRows = 1;
constexpr int kFusedWaves = 16, kFusedWavesAdam = 64;
constexpr int kFusedCtas = 8;
template <int G, int VPL, bool UPDATE, bool ADAM, bool BF16, bool PACKED>
__global__ void __launch_bounds__(256, (VPL == 1 ? kFusedCtas : 1))
agg_update_kernel(const uint32_t* __restrict__ row_start, const uint32_t* __restrict__ src,
                  const int32_t* __restrict__ agg_ids, const int64_t* __restrict__ n_agg_dev,
                  int64_t out_cap, const int64_t* __restrict__ n_entries,
                  const float* __restrict__ grads, int64_t in_cap,
                  const uint8_t* __restrict__ src_worker, const float* __restrict__ weights, int K,
                  void* table, int64_t n_rows, int dim, OptParams p, float* state0, float* state1,
                  float* __restrict__ agg_out) {
  pdl_sync();
  extern __shared__ float s_w[];  // the K weights
  // requested with the weights, not behind them
  const uint32_t rows_all = (uint32_t)*n_agg_dev;
  const uint32_t total = (uint32_t)min(n_entries[1], in_cap);
  for (int i = threadIdx.x; i < K; i += blockDim.x) s_w[i] = weights[i];
  __syncthreads();
  constexpr int R = VPL == 1 ? kFusedRows : 1;  // rows a lane group has in flight
  const int nvec = dim / 4;
  const RowLanes<256, G, PACKED> lanes(nvec);
  const int lg = lanes.lg;
  if (!lanes.on()) return;
  // 32-bit row numbers and slots (fewer than 2^31 of each): the kernel is bound by its instruction
  // stream and by the registers that live across the chain of loads
  const uint32_t n = (uint32_t)min((int64_t)rows_all, out_cap);
  // where the capacity cuts rows off, the next row's start still ends the last one (the update, whose
  // result is flagged then, does without: it has no register to spare)
  const uint32_t n_starts = UPDATE ? n : rows_all;
  const uint32_t stride = gridDim.x * lanes.groups;
  for (uint32_t u0 = blockIdx.x * lanes.groups + lanes.grp; u0 < n; u0 += R * stride) {
    uint32_t s0[R], s1[R];
    int32_t row[R];
    bool ok[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const uint32_t u = u0 + r * stride;
      ok[r] = u < n;
      s0[r] = ok[r] ? __ldg(row_start + u) : 0u;
      s1[r] = ok[r] ? (u + 1 < n_starts ? __ldg(row_start + u + 1) : total) : 0u;
      row[r] = ok[r] ? __ldg(agg_ids + u) : -1;
    }
    uint32_t longest = 0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      ok[r] = ok[r] && (uint32_t)row[r] < (uint32_t)n_rows && s0[r] <= total;  // else flagged by the merge
      if (s1[r] > total) s1[r] = total;
      if (s1[r] > s0[r] + (uint32_t)K) s1[r] = s0[r] + (uint32_t)K;  // a row has at most K contributions
      if (!ok[r]) s1[r] = s0[r];
      longest = max(longest, s1[r] - s0[r]);
    }
#pragma unroll
    for (int j = 0; j < VPL; ++j) {
      const int vi = lg + j * G;
      if (vi >= nvec) continue;
      size_t at[R];
      float4 w[R], a0[R], a1[R], g[R];
#pragma unroll
      for (int r = 0; r < R; ++r) {
        at[r] = (size_t)(ok[r] ? row[r] : 0) * dim + 4 * (size_t)vi;
        g[r] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (UPDATE && ok[r]) {  // towards L2 now (costs no register), into registers after the sum
          prefetch_l2(static_cast<const char*>(table) + at[r] * (BF16 ? 2 : 4));
          prefetch_l2(state0 + at[r]);
          if (ADAM) prefetch_l2(state1 + at[r]);
        }
      }
      for (uint32_t e = 0; e < longest; e += 2) {
        float4 v[R][2];
        float wt[R][2];
#pragma unroll
        for (int r = 0; r < R; ++r) {
#pragma unroll
          for (int t = 0; t < 2; ++t) {
            wt[r][t] = 0.f;
            v[r][t] = make_float4(0.f, 0.f, 0.f, 0.f);
            const uint32_t o = s0[r] + e + t;
            if (o < s1[r]) {
              const uint32_t pos = __ldg(src + o);
              if ((int64_t)pos < in_cap) {
                const int wl = (int)__ldg(src_worker + o);  // written beside src[o] by the merge
                wt[r][t] = s_w[wl > K - 1 ? K - 1 : wl];
                v[r][t] = ldg_f4(grads + (size_t)pos * dim + 4 * vi);
              }
            }
          }
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
#pragma unroll
          for (int t = 0; t < 2; ++t) {
            g[r].x = fmaf(wt[r][t], v[r][t].x, g[r].x); g[r].y = fmaf(wt[r][t], v[r][t].y, g[r].y);
            g[r].z = fmaf(wt[r][t], v[r][t].z, g[r].z); g[r].w = fmaf(wt[r][t], v[r][t].w, g[r].w);
          }
        }
      }
      // the row's parameters and state are requested only now: asking for them before the sum
      // (to overlap their latency with it) costs registers that the 64 warps per SM do not have
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if (UPDATE && ok[r]) {
          w[r] = load_row4(table, BF16, at[r]);
          a0[r] = *reinterpret_cast<const float4*>(state0 + at[r]);
          if (ADAM) a1[r] = *reinterpret_cast<const float4*>(state1 + at[r]);
        }
      }
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if (!ok[r]) continue;
        if (!UPDATE || agg_out) reinterpret_cast<float4*>(agg_out + (size_t)(u0 + r * stride) * dim)[vi] = g[r];
        if (!UPDATE) continue;
        if (ADAM) {
          w[r].x = adam1(a0[r].x, a1[r].x, g[r].x, w[r].x, p); w[r].y = adam1(a0[r].y, a1[r].y, g[r].y, w[r].y, p);
          w[r].z = adam1(a0[r].z, a1[r].z, g[r].z, w[r].z, p); w[r].w = adam1(a0[r].w, a1[r].w, g[r].w, w[r].w, p);
          *reinterpret_cast<float4*>(state1 + at[r]) = a1[r];
        } else {
          w[r].x = adagrad1(a0[r].x, g[r].x, w[r].x, p); w[r].y = adagrad1(a0[r].y, g[r].y, w[r].y, p);
          w[r].z = adagrad1(a0[r].z, g[r].z, w[r].z, p); w[r].w = adagrad1(a0[r].w, g[r].w, w[r].w, p);
        }
        *reinterpret_cast<float4*>(state0 + at[r]) = a0[r];
        store_row4(table, BF16, at[r], w[r]);
      }
    }
  }
}

template <int G, int VPL, bool PACKED>
void launch_agg_update(const FusedUpdate& fu, const uint32_t* row_start, const uint32_t* src,
                       const antdt_sparse_part* sp, int64_t out_cap, const int64_t* n_entries,
                       const uint8_t* src_worker, const float* weights, int K, cudaStream_t s) {
  const int64_t gpb = row_groups(256, sp->dim / 4, G, PACKED);
  const int64_t want = (out_cap + gpb - 1) / gpb;
  const size_t smem = 4 * (size_t)K;
  const bool adam = fu.opt == ANTDT_OPT_ADAM, bf16 = fu.dtype == ANTDT_BF16;
  const int64_t cap = (int64_t)kNumSM * kFusedCtas * (adam ? kFusedWavesAdam : kFusedWaves);
  const unsigned grid = (unsigned)(want > cap ? cap : (want < 1 ? 1 : want));
  if (!fu.table) {  // the sums alone
    ANTDT_LAUNCH("agg_reduce", (agg_update_kernel<G, VPL, false, false, false, PACKED>), grid, 256, smem, s, row_start, src,
                 sp->agg_ids, sp->n_agg, out_cap, n_entries, sp->uniq_grads, sp->in_cap, src_worker, weights, K,
                 nullptr, sp->n_rows, sp->dim, fu.p, nullptr, nullptr, fu.agg_out);
    return;
  }
#define FU_GO(A, B)                                                                              \
  ANTDT_LAUNCH("agg_update", (agg_update_kernel<G, VPL, true, A, B, PACKED>), grid, 256, smem, s, row_start, src, \
               sp->agg_ids, sp->n_agg, out_cap, n_entries, sp->uniq_grads, sp->in_cap, src_worker, weights, K, \
               fu.table, sp->n_rows, sp->dim, fu.p, fu.state0, fu.state1, fu.agg_out)
  if (adam) { if (bf16) FU_GO(true, true); else FU_GO(true, false); }
  else      { if (bf16) FU_GO(false, true); else FU_GO(false, false); }
#undef FU_GO
}

}  // namespace
}  // namespace antdt

extern "C" size_t antdt_weighted_aggregate_workspace_bytes(int64_t in_cap, int32_t dim,
                                                           int32_t n_workers) {
  if (in_cap < 0 || dim < 0 || dim > 1024 || n_workers < 1 || n_workers > antdt::kMaxSegments)
    return 0;
  return antdt::agg_layout(in_cap, n_workers, dim).bytes;
}

namespace antdt {
namespace {
// Lists of up to 16 workers that are summed row by row (agg_update_kernel without a table) instead of by tiles: one
// launch for two and no head bits, while a tile's walk keeps more gradient rows in flight.  Server of two kernels, by
// tiles -> by rows: 63 k entries x 32 floats 31 -> 25 us, 108 k x 20 32 -> 26, 312 k x 16 51 -> 43, 133 k x 64 43 -> 42;
// but 1.2 M x 16 93 -> 101, 624 k x 64 of 4 workers 79 -> 85, and where many workers list a row (a lane group takes its
// contributions in turn) 312 k x 64 over 50 k rows 86 -> 101.  A row's lists are at most as many as there are workers; by
// 4 / 8 / 12 / 16 / 20 / 24 / 32 of them: one field of 1 M rows, ids by frequency, 200 k occurrences x 32 77 -> 70, 95 -> 88,
// 108 -> 104, 115 -> 115, 130 -> 133, 135 -> 143, 148 -> 165, 400 k x 16 85 -> 79, 114 -> 109, 137 -> 133, 154 -> 156, 174 -> 179,
// 184 -> 195, 202 -> 228; 26 such fields, 426 k x 16 51 -> 44, 53 -> 47, 59 -> 51, 60 -> 56, 63 -> 63, 64 -> 66, 64 -> 73; hashed
// ids, 213 k x 32 45 -> 39, 45 -> 40, 47 -> 42, 47 -> 43, 47 -> 47, 48 -> 48, 48 -> 51.
constexpr int kByRowsWorkers = 16;
bool sum_by_rows(int K, int64_t in_cap, int dim, int64_t n_rows) {
  return K <= kByRowsWorkers && in_cap * dim <= (int64_t)1 << 23 && in_cap <= 2 * n_rows;
}
constexpr int64_t kDenseBesideBytes = 8 << 20;  // below, the fork and join cost what they hide
enum { kDenseStart = 0, kDenseDone = 1 };  // events of the dense part's side set
constexpr int kBulkSmem = 4 * kBulkSlots * kBulkGroup * kBulkElems;

bool dense_valid(const antdt_dense_part& d) {
  if (d.n < 0 || d.n % 4 || d.stride < d.n || d.stride % 4) return false;
  return d.n == 0 || (d.grads && d.out && aligned16(d.grads) && aligned16(d.out));
}

// w_i = b_i / sum_j b_j over the workers that count, formed in double, used in fp32
bool worker_weights(const int64_t* batch_sizes, const uint8_t* dropped, int K, float* hw) {
  double tot = 0.0;
  for (int i = 0; i < K; ++i) {
    if (batch_sizes[i] < 0) return false;
    if (!(dropped && dropped[i])) tot += (double)batch_sizes[i];
  }
  if (!(tot > 0.0)) return false;
  for (int i = 0; i < K; ++i) hw[i] = (dropped && dropped[i]) ? 0.f : (float)((double)batch_sizes[i] / tot);
  return true;
}

// The dense part on the stream `s`, a whole GPU's worth of CTAs.
void launch_dense(const antdt_dense_part* dp, const float* weights, const float* hw, int K, cudaStream_t s) {
  DenseWeights blob = {};
  for (int i = 0; i < K && i < kDenseBlobWorkers; ++i) blob.w[i] = hw[i];
  const int64_t n4 = dp->n / 4;
  const int64_t want = (n4 + 255) / 256, cap = (int64_t)kNumSM * 16;
  ANTDT_LAUNCH("dense_wsum", dense_wsum_kernel, (unsigned)(want > cap ? cap : want), 256, 4 * (size_t)K, s,
               dp->grads, n4, dp->stride, K <= kDenseBlobWorkers ? (const float*)nullptr : weights, blob, K, dp->out);
}

// More than 32 workers, where the resident merge does not fit: merge order by one stable radix sort of (row id, position).
void sort_merge_order(const antdt_sparse_part* sp, const uint8_t* dropped, bool any_dropped, int K,
                      int64_t in_cap, int64_t agg_cap, char* w8, const AggLayout& L,
                      int32_t* dev_status, cudaStream_t s) {
    char* sort_ws = w8 + L.sort_ws;
    int64_t* bounds = (int64_t*)(w8 + L.bounds);
    uint32_t* keys_a = (uint32_t*)(w8 + L.keys_a);
    const uint32_t* sort_keys = reinterpret_cast<const uint32_t*>(sp->uniq_ids);
    const uint32_t* sort_vals = nullptr;  // payload = position in the concatenated lists
    const int key_bits = bits_for(sp->n_rows);
    if (!any_dropped) {
      ANTDT_LAUNCH("agg_prep", agg_prep_kernel, 1, 256, 0, s, sp->worker_uniq_offsets, K, in_cap,
                   bounds, (int64_t*)(w8 + L.wuo), dev_status);
    } else {
      uint32_t hd[kMaxSegments];
      for (int i = 0; i < K; ++i) hd[i] = dropped[i] ? 1u : 0u;
      uint32_t* d_drop = (uint32_t*)(w8 + L.drop);
      int64_t* cwuo = (int64_t*)(w8 + L.cwuo);
      upload_small(hd, 4 * (size_t)K, d_drop, s);
      ANTDT_LAUNCH("agg_prep", agg_prep_backup_kernel, 1, 32, 0, s, sp->worker_uniq_offsets, d_drop,
                   K, in_cap, bounds, (int64_t*)(w8 + L.wuo), cwuo, dev_status);
      // the compacted input lives in the pair of sort buffers that the first pass does not
      // write: the temporaries when the pass count is odd, the outputs when it is even
      const bool odd = sort_passes(key_bits) % 2 == 1;
      uint32_t* keys_c = (uint32_t*)(w8 + (odd ? L.keys_b : L.keys_a));
      uint32_t* vals_c = (uint32_t*)(w8 + (odd ? L.vals_t : L.src));
      if (in_cap > 0) {
        int64_t want = (in_cap + 255) / 256;
        const int64_t gcap = (int64_t)kNumSM * 16;
        ANTDT_LAUNCH("agg_compact", agg_compact_kernel, (unsigned)(want > gcap ? gcap : want), 256,
                     16 * ((size_t)K + 1) + 4 * (size_t)K, s, sp->uniq_ids,
                     (const int64_t*)(w8 + L.wuo), cwuo, d_drop, K, keys_c, vals_c);
      }
      sort_keys = keys_c;
      sort_vals = vals_c;
    }
    segsort_setup(bounds, 1, in_cap, sort_ws, L.sort, s);
    segsort_run(sort_keys, sort_vals, keys_a, (uint32_t*)(w8 + L.src), (uint32_t*)(w8 + L.keys_b),
                (uint32_t*)(w8 + L.vals_t), key_bits, 0, in_cap, sort_ws, L.sort, dev_status, s, true);
    segsort_runs(keys_a, in_cap, sp->agg_ids, (int64_t*)(w8 + L.run_start), nullptr, sp->n_agg,
                 agg_cap, (uint32_t*)(w8 + L.head_bits),
                 (int32_t*)(w8 + L.tile_first), red_tile_for(in_cap > 0 ? in_cap : 1, sp->dim), sort_ws, L.sort, dev_status, s, true);
}

int32_t aggregate_impl(const antdt_sparse_part* sp, const antdt_dense_part* dp,
                       const int64_t* batch_sizes, const uint8_t* dropped, int32_t n_workers,
                       void* ws, size_t ws_bytes, int32_t* dev_status, void* stream,
                       const FusedUpdate* fu = nullptr, const OrderFork* fork = nullptr, bool merged = false) {
  const int K = n_workers;
  if (K < 1 || K > kMaxSegments || !batch_sizes || !ws || !aligned16(ws)) return ANTDT_ERR_INVALID_ARG;
  float hw[kMaxSegments];
  if (!worker_weights(batch_sizes, dropped, K, hw)) return ANTDT_ERR_INVALID_ARG;
  bool any_dropped = false;
  for (int i = 0; i < K; ++i) any_dropped |= dropped && dropped[i];
  const int64_t in_cap = sp ? sp->in_cap : 0;
  if (sp) {
    if (sp->dim < 4 || sp->dim > 1024 || sp->dim % 4 || sp->n_rows < 1 || sp->n_rows >= (1ll << 31) ||
        sp->in_cap < 0 || sp->in_cap >= (1ll << 31) || sp->out_cap < 0 || !sp->worker_uniq_offsets ||
        !sp->n_agg)
      return ANTDT_ERR_INVALID_ARG;
    if (sp->in_cap > 0 && (!sp->uniq_ids || !sp->uniq_grads)) return ANTDT_ERR_INVALID_ARG;
    const bool fused = fu && K <= kRangeMaxWorkers;  // then agg_grads is optional
    if (sp->out_cap > 0 && (!sp->agg_ids || (!sp->agg_grads && !fused))) return ANTDT_ERR_INVALID_ARG;
    if (!aligned16(sp->uniq_grads) || !aligned16(sp->agg_grads)) return ANTDT_ERR_INVALID_ARG;
  }
  if (dp && !dense_valid(*dp)) return ANTDT_ERR_INVALID_ARG;
  const AggLayout L = agg_layout(in_cap, K, sp ? sp->dim : 0);
  if (ws_bytes < L.bytes) return ANTDT_ERR_WORKSPACE_TOO_SMALL;
  cudaStream_t s = (cudaStream_t)stream;
  char* w8 = static_cast<char*>(ws);

  // the two merges carry the weights themselves
  bool resident = sp && !merged && resident_merge_wanted(K, in_cap, sp->n_rows);
  const bool by_ranges = sp && K <= kRangeMaxWorkers && in_cap > 0;
  // a lane group per row: the one-pass update, and the sums of short lists
  const bool few = sp && !fu && sum_by_rows(K, in_cap, sp->dim, sp->n_rows);
  bool by_rows = sp && in_cap > 0 && ((fu && K <= kRangeMaxWorkers) || (!fu && resident && resident_sort_clears(in_cap)) || few);
  auto upload_weights = [&] { upload_small(hw, 4 * (size_t)K, w8 + L.weights, s); };
  if (!by_ranges && !resident) upload_weights();
  // the dense part runs beside the sparse one where there is enough of it
  DenseBeside beside(sp && in_cap > 0 ? dp : nullptr, batch_sizes, dropped, K, dev_status, s);
  PdlScope pdl(!beside.issued() && in_cap <= kPdlMaxItems);

  if (sp) {
    int64_t* bounds = (int64_t*)(w8 + L.bounds);
    const int64_t agg_cap = sp->out_cap < in_cap ? sp->out_cap : in_cap;
    if (resident) {
      cudaStream_t so = fork ? fork->side : s;
      if (fork && cudaStreamWaitEvent(so, fork->ids_ready, 0) != cudaSuccess) return ANTDT_ERR_CUDA;
      ResidentMergeArgs q = {};
      q.uniq_ids = sp->uniq_ids; q.wuo_in = sp->worker_uniq_offsets; q.in_cap = in_cap; q.n_rows = sp->n_rows;
      q.n_workers = K; q.agg_ids = sp->agg_ids; q.n_agg = sp->n_agg; q.out_cap = agg_cap;
      q.wuo_out = (int64_t*)(w8 + L.wuo); q.n_entries = bounds; q.src = (uint32_t*)(w8 + L.src);
      if (by_rows) {
        q.row_start = (uint32_t*)(w8 + L.row_start);
        q.src_worker = (uint8_t*)(w8 + L.src_worker);
      } else {
        q.head_bits = (uint32_t*)(w8 + L.head_bits);
        q.tile_first = (int32_t*)(w8 + L.tile_first);
        while ((1 << q.tile_shift) < red_tile_for(in_cap, sp->dim)) ++q.tile_shift;
      }
      q.weights_dev = (float*)(w8 + L.weights);
      for (int i = 0; i < K; ++i) {
        q.weights[i] = hw[i];
        if (dropped && dropped[i]) q.dropped[i >> 5] |= 1u << (i & 31);
      }
      q.flags = (uint32_t*)(w8 + L.flags); q.zero = q.flags;
      const size_t zero_bytes = q.head_bits ? L.head_part - L.flags : 4 * kResFlagWords;
      q.n_zero = (int64_t)(zero_bytes / 4);
      if (!resident_sort_clears(in_cap) && cudaMemsetAsync(q.zero, 0, zero_bytes, so) != cudaSuccess)
        return ANTDT_ERR_CUDA;
      q.pairs = (uint2*)(w8 + L.keys_a);  // keys_a and keys_b lie side by side
      q.hist = (uint16_t*)(w8 + L.sort_ws + L.sort.hist); q.status = dev_status;
      const int32_t rc = resident_merge(q, so);
      if (rc != ANTDT_OK && rc != kResidentRefused) return rc;
      if (fork && (cudaEventRecord(fork->order_done, so) != cudaSuccess ||
                   cudaStreamWaitEvent(s, fork->order_done, 0) != cudaSuccess))
        return ANTDT_ERR_CUDA;
      if (rc == kResidentRefused) {
        resident = false;
        by_rows = (fu && K <= kRangeMaxWorkers) || few;
        if (!by_ranges) upload_weights();
      }
    }
    if (merged || resident) {
      // the merge order is there: the backward's sort made it on the way, or the resident merge
    } else if (by_ranges) {
      // up to 32 workers: the merge order comes from the range-partitioned pass, no sort
      uint32_t dropped_bits = 0;
      for (int i = 0; i < K; ++i)
        if (dropped && dropped[i]) dropped_bits |= 1u << i;
      // the order needs the id lists only: on a forked step it runs beside the backward's sums
      cudaStream_t so = fork ? fork->side : s;
      if (fork && cudaStreamWaitEvent(so, fork->ids_ready, 0) != cudaSuccess) return ANTDT_ERR_CUDA;
      range_merge_order(sp->uniq_ids, sp->worker_uniq_offsets, in_cap, sp->n_rows, K, dropped_bits,
                        sp->agg_ids, sp->n_agg, agg_cap, (int64_t*)(w8 + L.wuo), bounds,
                        (uint32_t*)(w8 + L.src), by_rows ? nullptr : (uint32_t*)(w8 + L.head_bits),
                        by_rows ? nullptr : (int32_t*)(w8 + L.tile_first), red_tile_for(in_cap, sp->dim),
                        by_rows ? (uint32_t*)(w8 + L.row_start) : nullptr,
                        by_rows ? (uint8_t*)(w8 + L.src_worker) : nullptr, hw, (float*)(w8 + L.weights),
                        w8 + L.range_ws, L.range, dev_status, so);
      if (fork && (cudaEventRecord(fork->order_done, so) != cudaSuccess ||
                   cudaStreamWaitEvent(s, fork->order_done, 0) != cudaSuccess))
        return ANTDT_ERR_CUDA;
    } else {
      sort_merge_order(sp, dropped, any_dropped, K, in_cap, agg_cap, w8, L, dev_status, s);
    }
    if (by_rows) {
      // one pass: every aggregated row is summed and applied by the lane group that owns it
      FusedUpdate f = fu ? *fu : FusedUpdate{};
      f.agg_out = sp->agg_grads;
      const uint32_t* rs = (const uint32_t*)(w8 + L.row_start);
      const uint32_t* src = (const uint32_t*)(w8 + L.src);
      const uint8_t* sw = (const uint8_t*)(w8 + L.src_worker);
      const float* wts = (const float*)(w8 + L.weights);
      const int nvec = sp->dim / 4;
#define FU_CASE(G, VPL)                                                                                \
  do {                                                                                                 \
    if (VPL == 1 && (f.opt == ANTDT_OPT_ADAM ? row_packs_narrow(nvec, G) : row_packs(256, nvec, G)))   \
      launch_agg_update<G, VPL, (VPL == 1 && G > 2)>(f, rs, src, sp, agg_cap, bounds, sw, wts, K, s);  \
    else                                                                                               \
      launch_agg_update<G, VPL, false>(f, rs, src, sp, agg_cap, bounds, sw, wts, K, s);                \
  } while (0)
      if (nvec <= 1) FU_CASE(1, 1);
      else if (nvec <= 2) FU_CASE(2, 1);
      else if (nvec <= 4) FU_CASE(4, 1);
      else if (nvec <= 8) FU_CASE(8, 1);
      else if (nvec <= 16) FU_CASE(16, 1);
      else if (nvec <= 32) FU_CASE(32, 1);
      else if (nvec <= 64) FU_CASE(32, 2);
      else if (nvec <= 128) FU_CASE(32, 4);
      else FU_CASE(32, 8);
#undef FU_CASE
    } else if (in_cap > 0) {
      TileArgs t;
      t.payload = (const uint32_t*)(w8 + L.src);
      t.head_bits = (const uint32_t*)(w8 + L.head_bits);
      t.tile_first = (const int32_t*)(w8 + L.tile_first);
      t.tile = red_tile_for(in_cap, sp->dim);
      t.rows = sp->uniq_grads;
      t.dim = sp->dim;
      t.n_host = in_cap;
      t.n_dev = bounds + 1;  // the clamped total of the workers' lists
      t.payload_limit = in_cap;
      t.bounds = (const int64_t*)(w8 + L.wuo);
      t.scales = (const float*)(w8 + L.weights);
      t.K = K;
      t.out_cap = sp->out_cap < in_cap ? sp->out_cap : in_cap;
      t.out = sp->agg_grads;
      t.head_part = (float*)(w8 + L.head_part);
      t.tail_part = (float*)(w8 + L.tail_part);
      launch_tile_reduce(t, "agg_reduce", "agg_fixup", s);
    }
  }
  if (dp && dp->n > 0 && !beside.issued()) launch_dense(dp, (const float*)(w8 + L.weights), hw, K, s);
  beside.join();
  return cuda_ok();
}
}  // namespace

void aggregate_prepare_device() {
  static bool done[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (!done[dev & 63]) {
    cudaFuncSetAttribute(dense_wsum_bulk_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kBulkSmem);
    done[dev & 63] = true;
  }
}

// 2.2 GB (32 workers x 16.8 M) beside the sort of 35 M occurrences: 1.03 - 1.19 ms instead of 0.34 alone, the
// sort's kernels 0.15 ms slower, the step 5426 - 5554 -> 5269 - 5419 us (6 runs of each in turn); with the
// full-size kernel at 2 CTAs per SM beside the merge order 5380.  285 MB of 16 workers in the step of 65 M
// occurrences: 9507 - 9647 -> 9279 - 9600, hardly more than the runs differ.  117 MB beside the merge order of a
// server alone: 618 - 627 -> 555 - 558 us.
DenseBeside::DenseBeside(const antdt_dense_part* dp, const int64_t* batch_sizes, const uint8_t* dropped, int K,
                         int32_t* dev_status, cudaStream_t s) : main_(s) {
  if (!dp || !batch_sizes || K < 1 || K > kDenseBlobWorkers || !dense_valid(*dp) || dp->n * 4 * (K + 1) < kDenseBesideBytes ||
      dp->n >= (1ll << 31))
    return;
  float hw[kDenseBlobWorkers];
  if (!worker_weights(batch_sizes, dropped, K, hw)) return;
  aggregate_prepare_device();
  if (!side_.take(s)) return;
  if (cudaEventRecord(side_->event[kDenseStart], s) != cudaSuccess ||
      cudaStreamWaitEvent(side_->stream[0], side_->event[kDenseStart], 0) != cudaSuccess) {
    cudaGetLastError();
    side_.release();
    return;
  }
  DenseWeights blob = {};
  for (int i = 0; i < K; ++i) blob.w[i] = hw[i];
  const int64_t tiles = (dp->n + kBulkElems - 1) / kBulkElems;
  ANTDT_LAUNCH("dense_wsum", dense_wsum_bulk_kernel, (unsigned)(tiles < kNumSM ? tiles : kNumSM), kBulkThreads,
               kBulkSmem, side_->stream[0], dp->grads, (uint32_t)dp->n, dp->stride, blob, K, dp->out, dev_status);
  issued_ = true;
}

void DenseBeside::join() {
  if (!side_) return;
  cudaEventRecord(side_->event[kDenseDone], side_->stream[0]);
  cudaStreamWaitEvent(main_, side_->event[kDenseDone], 0);
  side_.release();
}

int32_t weighted_aggregate_forked(const antdt_sparse_part* sp, const antdt_dense_part* dp,
                                  const int64_t* batch_sizes, int32_t n_workers, void* ws,
                                  size_t ws_bytes, int32_t* dev_status, void* stream,
                                  const OrderFork* fork) {
  return aggregate_impl(sp, dp, batch_sizes, nullptr, n_workers, ws, ws_bytes, dev_status, stream,
                        nullptr, fork);
}
}  // namespace antdt

extern "C" int32_t antdt_weighted_aggregate(const antdt_sparse_part* sp, const antdt_dense_part* dp,
                                            const int64_t* batch_sizes, int32_t n_workers, void* ws,
                                            size_t ws_bytes, int32_t* dev_status, void* stream) {
  return antdt::aggregate_impl(sp, dp, batch_sizes, nullptr, n_workers, ws, ws_bytes, dev_status,
                               stream);
}

extern "C" int32_t antdt_weighted_aggregate_backup(const antdt_sparse_part* sp,
                                                   const antdt_dense_part* dp,
                                                   const int64_t* batch_sizes, const uint8_t* dropped,
                                                   int32_t n_workers, void* ws, size_t ws_bytes,
                                                   int32_t* dev_status, void* stream) {
  if (!dropped) return ANTDT_ERR_INVALID_ARG;
  return antdt::aggregate_impl(sp, dp, batch_sizes, dropped, n_workers, ws, ws_bytes, dev_status,
                               stream);
}

// Aggregation followed by the sparse update in one call; with up to 32 workers in one pass over
// the aggregated rows (agg_update_kernel), otherwise the two steps one after the other.
namespace antdt {
int32_t aggregate_update_forked(const antdt_sparse_part* sp, const antdt_dense_part* dp,
                                const int64_t* batch_sizes, int32_t n_workers, void* table,
                                int32_t dtype, int32_t opt, float lr, float eps, float beta1,
                                float beta2, int64_t step, float* state0, float* state1, void* ws,
                                size_t ws_bytes, int32_t* dev_status, void* stream,
                                const OrderFork* fork, bool merged) {
  if (!sp || !table || !state0 || step < 1) return ANTDT_ERR_INVALID_ARG;
  if (dtype != ANTDT_F32 && dtype != ANTDT_BF16) return ANTDT_ERR_INVALID_ARG;
  if (sp->dim % (dtype == ANTDT_BF16 ? 8 : 4)) return ANTDT_ERR_INVALID_ARG;
  if (opt != ANTDT_OPT_ADAGRAD && opt != ANTDT_OPT_ADAM) return ANTDT_ERR_INVALID_ARG;
  if (opt == ANTDT_OPT_ADAM && !state1) return ANTDT_ERR_INVALID_ARG;
  if (!aligned16(table) || !aligned16(state0) || !aligned16(state1)) return ANTDT_ERR_INVALID_ARG;
  if (n_workers > kRangeMaxWorkers) {  // the merge order has no row starts there: two steps, agg_grads is needed
    if (sp->out_cap > 0 && !sp->agg_grads) return ANTDT_ERR_INVALID_ARG;
    const int32_t rc = aggregate_impl(sp, dp, batch_sizes, nullptr, n_workers, ws, ws_bytes,
                                      dev_status, stream);
    if (rc != ANTDT_OK) return rc;
    const int64_t cap = sp->out_cap < sp->in_cap ? sp->out_cap : sp->in_cap;
    return antdt_sparse_opt_update(table, dtype, sp->n_rows, sp->dim, sp->agg_ids, sp->agg_grads,
                                   sp->n_agg, cap, opt, lr, eps, beta1, beta2, step, state0, state1,
                                   dev_status, stream);
  }
  FusedUpdate fu;
  fu.table = table; fu.dtype = dtype; fu.opt = opt; fu.state0 = state0; fu.state1 = state1;
  fu.agg_out = nullptr;
  fu.p = make_opt_params(lr, eps, beta1, beta2, step);
  return aggregate_impl(sp, dp, batch_sizes, nullptr, n_workers, ws, ws_bytes, dev_status, stream, &fu,
                        fork, merged);
}

bool step_merge_targets(const antdt_sparse_part& sp, const int64_t* batch_sizes, int K, int64_t nnz, void* ws,
                        size_t ws_bytes, StepMerge* m) {
  if (!batch_sizes || !ws || sp.in_cap < 1 || sp.out_cap < 1 || sp.in_cap >= (1ll << 31) || !sp.agg_ids || !sp.n_agg ||
      K > kStepMergeWorkers || !resident_sort_fits(K, nnz, sp.n_rows))
    return false;
  double tot = 0.0;
  for (int i = 0; i < K; ++i) {
    if (batch_sizes[i] < 0) return false;
    tot += (double)batch_sizes[i];
  }
  if (!(tot > 0.0)) return false;
  const AggLayout L = agg_layout(sp.in_cap, K, sp.dim);
  if (ws_bytes < L.bytes) return false;
  char* w8 = static_cast<char*>(ws);
  m->agg_ids = sp.agg_ids; m->n_agg = sp.n_agg;
  m->agg_cap = sp.out_cap < sp.in_cap ? sp.out_cap : sp.in_cap;
  m->n_entries = (int64_t*)(w8 + L.bounds);
  m->src = (uint32_t*)(w8 + L.src); m->src_worker = (uint8_t*)(w8 + L.src_worker); m->src_cap = sp.in_cap;
  m->row_start = (uint32_t*)(w8 + L.row_start);
  m->weights_dev = (float*)(w8 + L.weights);
  for (int i = 0; i < kStepMergeWorkers; ++i) m->weights[i] = i < K ? (float)((double)batch_sizes[i] / tot) : 0.f;
  return true;
}
}  // namespace antdt

extern "C" int32_t antdt_aggregate_update(const antdt_sparse_part* sp, const antdt_dense_part* dp,
                                          const int64_t* batch_sizes, int32_t n_workers, void* table,
                                          int32_t dtype, int32_t opt, float lr, float eps, float beta1,
                                          float beta2, int64_t step, float* state0, float* state1,
                                          void* ws, size_t ws_bytes, int32_t* dev_status, void* stream) {
  return antdt::aggregate_update_forked(sp, dp, batch_sizes, n_workers, table, dtype, opt, lr, eps, beta1,
                                        beta2, step, state0, state1, ws, ws_bytes, dev_status, stream,
                                        nullptr);
}
