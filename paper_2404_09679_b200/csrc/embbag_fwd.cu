// Worker forward: embedding-bag gather with sum pooling.
//
// One group of G lanes owns one bag; a row is read as G (x VPL) 16-byte vectors, so a warp
// issues fully coalesced 128-bit loads over 32/G rows at once.  The path is a random gather bound
// by the latency of its chain of dependent loads (offsets -> ids -> rows) and by HBM / L2 for the
// rows; there is no contraction here and so no tensor-core work.  Four kernels:
//   embbag_fwd_flat_kernel    rows of up to 512 bytes, one bag per group: every lane reads the ids
//                             itself, four rows in flight, 32 registers -> 64 warps per SM
//   embbag_fwd_stride_kernel  the same for many bags: capped grid, groups stride over the bags
//                             and read the next bag's offsets ahead
//   embbag_fwd_ahead_kernel   the same with the next bag's ids asked for ahead and more rows in flight, for
//                             longer bags from one resident wave of them on
//   embbag_fwd_kernel         wider rows (VPL vectors per lane): ids staged through the group's
//                             registers G at a time (one coalesced load, then shuffles)
#include <algorithm>

#include "common.cuh"

namespace antdt {
namespace {

constexpr int kFwdThreads = 128;
constexpr int kFwdUnroll = 4;

template <int G, int VPL, bool BF16, bool BY_FIELD>
__global__ void __launch_bounds__(kFwdThreads, (VPL == 1 ? 12 : 1))
embbag_fwd_kernel(const void* __restrict__ table, int64_t n_rows, int dim,
                  const int32_t* __restrict__ row_ids, int64_t nnz,
                  const int64_t* __restrict__ bag_offsets, int64_t n_bags,
                  float* __restrict__ pooled, int32_t* status, int fields, int64_t sample_blocks, bool chained) {
  if (chained) pdl_sync();  // (beside a kernel that it depends on the start of, it must not wait for its end)
  constexpr int EPV = BF16 ? 8 : 4;   // elements per 16-byte vector
  constexpr int PAIRS = EPV / 2;      // packed fp32 pairs per vector
  constexpr int U = (G < kFwdUnroll) ? G : kFwdUnroll;
  const int lg = threadIdx.x & (G - 1);
  // Bags are sample-major (bag = sample * fields + field).  When the caller knows `fields`, a CTA
  // takes the bags of ONE field of consecutive samples and consecutive CTAs stay on that field,
  // so that what is resident on an SM (and in L2) at one time draws from one field's hot rows.
  int64_t bag;
  if (BY_FIELD) {
    const int64_t f = blockIdx.x / sample_blocks, sb = blockIdx.x % sample_blocks;
    bag = (sb * (kFwdThreads / G) + (threadIdx.x / G)) * fields + f;
  } else {
    bag = (int64_t)blockIdx.x * (kFwdThreads / G) + (threadIdx.x / G);
  }
  if (bag >= n_bags) return;
  const unsigned gmask = group_mask<G>();
  const int nvec = dim / EPV;

  int64_t begin = bag_offsets[bag], end = bag_offsets[bag + 1];
  if (begin < 0 || end < begin || end > nnz) {  // never dereference through bad offsets
    if (lg == 0) set_status(status, ANTDT_ERR_BAD_OFFSETS);
    end = begin = 0;
  }
  const int len = (int)(end - begin);
  const int32_t* ids = row_ids + begin;
  const uint32_t limit = (uint32_t)n_rows;

  uint64_t acc[VPL][PAIRS];  // fp32 sums as packed pairs
#pragma unroll
  for (int k = 0; k < VPL; ++k)
#pragma unroll
    for (int e = 0; e < PAIRS; ++e) acc[k][e] = 0ull;

  const char* tbl = static_cast<const char*>(table);
  const uint32_t row_bytes = (uint32_t)dim * (BF16 ? 2u : 4u);

  for (int base = 0; base < len; base += G) {
    // G ids of the bag in one coalesced load; -1 marks "no row" (past the end, or out of range)
    int my_id = -1;
    if (base + lg < len) {
      my_id = __ldg(ids + base + lg);
      if ((uint32_t)my_id >= limit) {
        set_status(status, ANTDT_ERR_ID_OUT_OF_RANGE);
        my_id = -1;  // skipped: contributes nothing
      }
    }
#pragma unroll
    for (int j0 = 0; j0 < G; j0 += U) {
      if (base + j0 >= len) break;
      uint4 v[U][VPL];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int id = __shfl_sync(gmask, my_id, j0 + u, G);
        const uint4* rp = reinterpret_cast<const uint4*>(tbl + (size_t)(uint32_t)(id < 0 ? 0 : id) * row_bytes);
#pragma unroll
        for (int k = 0; k < VPL; ++k) {
          const int vi = lg + k * G;
          v[u][k] = (id >= 0 && vi < nvec) ? __ldg(rp + vi) : make_uint4(0u, 0u, 0u, 0u);
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
#pragma unroll
        for (int k = 0; k < VPL; ++k) {
          if (BF16) {  // bf16 -> fp32 is a 16-bit shift; a zero vector adds +0.0
            acc[k][0] = f32x2_add(acc[k][0], f32x2_pack(v[u][k].x << 16, v[u][k].x & 0xffff0000u));
            acc[k][1] = f32x2_add(acc[k][1], f32x2_pack(v[u][k].y << 16, v[u][k].y & 0xffff0000u));
            acc[k][2] = f32x2_add(acc[k][2], f32x2_pack(v[u][k].z << 16, v[u][k].z & 0xffff0000u));
            acc[k][3] = f32x2_add(acc[k][3], f32x2_pack(v[u][k].w << 16, v[u][k].w & 0xffff0000u));
          } else {
            acc[k][0] = f32x2_add(acc[k][0], f32x2_pack(v[u][k].x, v[u][k].y));
            acc[k][1] = f32x2_add(acc[k][1], f32x2_pack(v[u][k].z, v[u][k].w));
          }
        }
      }
    }
  }

  float* out = pooled + bag * (int64_t)dim;
#pragma unroll
  for (int k = 0; k < VPL; ++k) {
    const int vi = lg + k * G;
    if (vi >= nvec) continue;
    ulonglong2* o = reinterpret_cast<ulonglong2*>(out + (size_t)vi * EPV);
    o[0] = make_ulonglong2(acc[k][0], acc[k][1]);
    if (BF16) o[1] = make_ulonglong2(acc[k][2], acc[k][3]);
  }
}


// The gather with the plainest possible inner loop, for rows of up to 512 bytes: every lane
// reads the bag's ids itself (the G lanes of a group ask for the same address: one transaction),
// four row loads are requested before any is consumed, nothing is exchanged between lanes, and
// the register budget (32) lets 64 warps share an SM.  What bounds this kernel is the chain
// offsets -> ids -> rows of dependent loads, and only the number of warps in flight hides it:
// eight loads per lane at 48 or 40 warps per SM were slower on every workload measured.
constexpr int kFlatThreads = 256;
constexpr int kFlatUnroll = 4;
constexpr int kFlatCtas = 8;     // CTAs per SM

// Whether bags are strided over (embbag_fwd_stride_kernel) and by how many resident waves of CTAs; 0: one bag
// per lane group.  W: waves that one bag per lane group would make.
// Reading the next bag's offsets ahead pays once a lane group has several turns, and the more of a bag's time
// its offsets are: the shorter its list and the wider its rows.  Above a length that depends on both, the
// fewer lane groups at work cost more than the offsets.  (ahead_of is asked first: fp32 lengths above 5 ids of 16 vectors,
// 7 of 32 and 2 of 4 are reached by packed rows only, whose lane groups are as many as rows fit a CTA.)  One bag per group -> striding, us, by ids per bag:
//   fp32, 32 vectors, W 39    1: 93 -> 79    3: 116 -> 99    10: 200 -> 191   20: 321 -> 325   40: 560 -> 584
//         16 vectors, W 39    1: 96 -> 82    3: 127 -> 108   10: 224 -> 217   20: 361 -> 367   40: 632 -> 688
//          8 vectors, W 39    1: 100 -> 88   4.5: 169 -> 158   5.5: 186 -> 182   6: 194 -> 194   7: 211 -> 219
//                     W 130   4.5: 551 -> 488   6.5: 660 -> 614
//          4 vectors, W 19    1.5: 58 -> 53   2: 67 -> 62    2.5: 71 -> 71    3: 82 -> 84      4.5: 103 -> 119
//          2 vectors, W 32    1.5: 104 -> 104   2: 123 -> 128   3: 155 -> 175
//   bf16, 32 vectors, W 78    1: 217 -> 189   4.5: 319 -> 296   10: 480 -> 479   20: 772 -> 817
//         16 vectors, W 39    1: 114 -> 100   3: 153 -> 145   4.5: 180 -> 177   10: 275 -> 292
//          8 vectors, W 19    1: 62 -> 56    3: 91 -> 88     4.5: 107 -> 107   10: 165 -> 175
//          4 vectors, W 19    1.5: 70 -> 71   3: 103 -> 103
// Few turns: W 7, 16 vectors, 4.5 ids 34 -> 31; W 8, 32 vectors, 10 ids 47 -> 47; W 2.5, 8 vectors, 1 id the same.
// About ten turns per group are best: fewer waves unbalance the SMs (W 327 in 1 / 4 / 16 waves: 1127 /
// 1039 / 958 us), more waste the reading ahead (W 39 in 4 / 16 / 32 waves: 119 / 128 / 140).
inline int stride_below(int G, bool bf16) {  // ids per bag
  if (bf16) return G >= 32 ? 8 : (G == 16 ? 5 : (G == 8 ? 4 : 0));
  return G >= 16 ? 16 : (G == 8 ? 6 : (G == 4 ? 3 : 0));
}
inline int stride_waves(int G, int64_t bags_per_cta, bool bf16, int64_t n_bags, int64_t nnz) {
  const int64_t per_wave = (int64_t)kNumSM * kFlatCtas * bags_per_cta;
  const int64_t W = n_bags / per_wave;
  if (W < 8 || nnz >= stride_below(G, bf16) * n_bags) return 0;
  const int64_t waves = (W + 5) / 10;
  return waves < 1 ? 1 : (waves > 16 ? 16 : (int)waves);
}

// One bag: this lane's 16 bytes of the sum of the rows that ids[0..len) name, as packed fp32 pairs.
// (The output address is formed by the caller after the loop: at 32 registers every 64-bit value
// that lives across the loop costs loads in flight.)
template <int G, bool BF16>
__device__ __forceinline__ void flat_bag(const uint4* __restrict__ tbl, uint32_t row_vecs, uint32_t limit,
                                         const int32_t* __restrict__ ids, int len, int lg, bool lane_on,
                                         uint64_t (&acc)[BF16 ? 4 : 2], bool& bad) {
  constexpr int PAIRS = BF16 ? 4 : 2;
#pragma unroll
  for (int e = 0; e < PAIRS; ++e) acc[e] = 0ull;
  for (int j0 = 0; j0 < len; j0 += kFlatUnroll) {
    uint4 v[kFlatUnroll];
#pragma unroll
    for (int t = 0; t < kFlatUnroll; ++t) {
      const bool in = j0 + t < len;
      const uint32_t id = in ? (uint32_t)__ldg(ids + j0 + t) : 0u;
      const bool ok = in && id < limit;
      bad |= in && !ok;  // skipped: contributes nothing
      v[t] = (ok && lane_on) ? __ldg(tbl + (size_t)id * row_vecs + lg) : make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll
    for (int t = 0; t < kFlatUnroll; ++t) {
      if (BF16) {  // bf16 -> fp32 is a 16-bit shift; a zero vector adds +0.0
        acc[0] = f32x2_add(acc[0], f32x2_pack(v[t].x << 16, v[t].x & 0xffff0000u));
        acc[1] = f32x2_add(acc[1], f32x2_pack(v[t].y << 16, v[t].y & 0xffff0000u));
        acc[2] = f32x2_add(acc[2], f32x2_pack(v[t].z << 16, v[t].z & 0xffff0000u));
        acc[3] = f32x2_add(acc[3], f32x2_pack(v[t].w << 16, v[t].w & 0xffff0000u));
      } else {
        acc[0] = f32x2_add(acc[0], f32x2_pack(v[t].x, v[t].y));
        acc[1] = f32x2_add(acc[1], f32x2_pack(v[t].z, v[t].w));
      }
    }
  }
}

template <bool BF16>
__device__ __forceinline__ void flat_store(float* __restrict__ out, const uint64_t (&acc)[BF16 ? 4 : 2]) {
  ulonglong2* o = reinterpret_cast<ulonglong2*>(out);
  o[0] = make_ulonglong2(acc[0], acc[1]);
  if (BF16) o[1] = make_ulonglong2(acc[2], acc[3]);
}

// A bag's id range; bad offsets are flagged and read as an empty bag.
__device__ __forceinline__ void flat_range(const int64_t* __restrict__ bag_offsets, int64_t bag, int64_t nnz,
                                           int lg, int32_t* status, int32_t& begin, int32_t& len) {
  const int64_t b = bag_offsets[bag], e = bag_offsets[bag + 1];
  begin = 0;
  len = 0;
  if (b < 0 || e < b || e > nnz) {
    if (lg == 0) set_status(status, ANTDT_ERR_BAD_OFFSETS);
    return;
  }
  begin = (int32_t)b;  // nnz < 2^31
  len = (int32_t)(e - b);
}

// One bag per lane group.  BY_FIELD: a CTA takes the bags of ONE field of consecutive samples and
// consecutive CTAs stay on that field (bag = sample * fields + field), so that what is resident
// on an SM and in L2 at one time draws from one field's hot rows.
template <int G, bool BF16, bool BY_FIELD, bool PACKED>
__global__ void __launch_bounds__(kFlatThreads, kFlatCtas)
embbag_fwd_flat_kernel(const void* __restrict__ table, int64_t n_rows, int dim,
                       const int32_t* __restrict__ row_ids, int64_t nnz,
                       const int64_t* __restrict__ bag_offsets, int64_t n_bags,
                       float* __restrict__ pooled, int32_t* status, int fields, int64_t sample_blocks, bool chained) {
  if (chained) pdl_sync();  // (beside a kernel that it depends on the start of, it must not wait for its end)
  constexpr int EPV = BF16 ? 8 : 4;
  const RowLanes<kFlatThreads, G, PACKED> lanes(PACKED ? dim / EPV : G);
  const int lg = lanes.lg;
  int64_t bag;
  if (BY_FIELD) {
    const int64_t f = blockIdx.x / sample_blocks, sb = blockIdx.x % sample_blocks;
    bag = (sb * lanes.groups + lanes.grp) * fields + f;
  } else {
    bag = (int64_t)blockIdx.x * lanes.groups + lanes.grp;
  }
  if (!lanes.on() || bag >= n_bags) return;
  const int nvec = dim / EPV;
  int32_t begin, len;
  flat_range(bag_offsets, bag, nnz, lg, status, begin, len);
  bool bad = false;
  uint64_t acc[BF16 ? 4 : 2];
  flat_bag<G, BF16>(static_cast<const uint4*>(table), (uint32_t)nvec, (uint32_t)n_rows, row_ids + begin, len,
                    lg, lg < nvec, acc, bad);
  if (bad) set_status(status, ANTDT_ERR_ID_OUT_OF_RANGE);
  if (lg < nvec) flat_store<BF16>(pooled + bag * (int64_t)dim + (size_t)lg * EPV, acc);
}

// Where the chain offsets -> ids -> rows is much of a bag's time (stride_waves): the grid is capped, every
// lane group strides over its bags (bag order), and the NEXT bag's offsets are read before the current
// bag's rows are requested (30 fields x 4.5 ids x 128-byte rows: 1.06 -> 0.84 ms).  The loop is written out in one piece on purpose: at 32 registers the form of
// the source decides what the compiler keeps in flight, and two tidier versions of this same loop
// (the bag's sum in a helper, the offsets held as raw 64-bit values) measured 1.07 - 1.21 ms.
template <int G, bool BF16, bool PACKED>
__global__ void __launch_bounds__(kFlatThreads, kFlatCtas)
embbag_fwd_stride_kernel(const void* __restrict__ table, int64_t n_rows, int dim,
                         const int32_t* __restrict__ row_ids, int64_t nnz,
                         const int64_t* __restrict__ bag_offsets, int64_t n_bags,
                         float* __restrict__ pooled, int32_t* status, bool chained) {
  if (chained) pdl_sync();  // (beside a kernel that it depends on the start of, it must not wait for its end)
  constexpr int EPV = BF16 ? 8 : 4;
  constexpr int PAIRS = EPV / 2;
  const int nvec = dim / EPV;
  const RowLanes<kFlatThreads, G, PACKED> lanes(nvec);
  if (!lanes.on()) return;
  const int GPB = lanes.groups;  // groups (bags) per CTA and turn
  const int lg = lanes.lg;
  const uint32_t limit = (uint32_t)n_rows;
  const bool lane_on = lg < nvec;
  const uint4* tbl = static_cast<const uint4*>(table);
  const uint32_t row_vecs = (uint32_t)nvec;
  // 32-bit bag numbers: there are fewer than 2^31 bags
  const uint32_t n_slots = (uint32_t)n_bags;
  const uint32_t stride = gridDim.x * GPB;
  auto range_of = [&](uint32_t q, int32_t& bg, int32_t& b0, int32_t& ln) {
    bg = -1; b0 = 0; ln = 0;
    if (q >= n_slots) return;
    bg = (int32_t)q;
    const int64_t begin = bag_offsets[q], end = bag_offsets[q + 1];
    if (begin < 0 || end < begin || end > nnz) {
      if (lg == 0) set_status(status, ANTDT_ERR_BAD_OFFSETS);
      return;
    }
    b0 = (int32_t)begin;  // nnz < 2^31
    ln = (int32_t)(end - begin);
  };
  uint32_t q = blockIdx.x * GPB + lanes.grp;
  int32_t bag, begin, len;
  range_of(q, bag, begin, len);
  bool bad = false;
  while (q < n_slots) {
    // the next turn's offsets are requested before this turn's rows
    int32_t nbag, nbegin, nlen;
    range_of(q + stride < q ? n_slots : q + stride, nbag, nbegin, nlen);
    if (bag >= 0) {
      const int32_t* ids = row_ids + begin;
      uint64_t acc[PAIRS];
#pragma unroll
      for (int e = 0; e < PAIRS; ++e) acc[e] = 0ull;
      for (int j0 = 0; j0 < len; j0 += kFlatUnroll) {
        uint4 v[kFlatUnroll];
#pragma unroll
        for (int t = 0; t < kFlatUnroll; ++t) {
          const bool in = j0 + t < len;
          const uint32_t id = in ? (uint32_t)__ldg(ids + j0 + t) : 0u;
          const bool ok = in && id < limit;
          bad |= in && !ok;
          v[t] = (ok && lane_on) ? __ldg(tbl + (size_t)id * row_vecs + lg) : make_uint4(0u, 0u, 0u, 0u);
        }
#pragma unroll
        for (int t = 0; t < kFlatUnroll; ++t) {
          if (BF16) {
            acc[0] = f32x2_add(acc[0], f32x2_pack(v[t].x << 16, v[t].x & 0xffff0000u));
            acc[1] = f32x2_add(acc[1], f32x2_pack(v[t].y << 16, v[t].y & 0xffff0000u));
            acc[2] = f32x2_add(acc[2], f32x2_pack(v[t].z << 16, v[t].z & 0xffff0000u));
            acc[3] = f32x2_add(acc[3], f32x2_pack(v[t].w << 16, v[t].w & 0xffff0000u));
          } else {
            acc[0] = f32x2_add(acc[0], f32x2_pack(v[t].x, v[t].y));
            acc[1] = f32x2_add(acc[1], f32x2_pack(v[t].z, v[t].w));
          }
        }
      }
      if (lane_on) {
        ulonglong2* o = reinterpret_cast<ulonglong2*>(pooled + bag * (int64_t)dim + (size_t)lg * EPV);
        o[0] = make_ulonglong2(acc[0], acc[1]);
        if (BF16) o[1] = make_ulonglong2(acc[2], acc[3]);
      }
    }
    if (q + stride < q) break;  // wrapped: nothing further
    q += stride; bag = nbag; begin = nbegin; len = nlen;
  }
  if (bad) set_status(status, ANTDT_ERR_ID_OUT_OF_RANGE);
}

// Which bags are read ahead of (embbag_fwd_ahead_kernel, ahead_of), with how many rows requested at once per lane
// (ahead_rows), and whether in field-major order.  More rows in flight per lane mean fewer warps (eight: 4 CTAs per SM, four: 5),
// which pays once a bag has ids enough to fill them (8 CTAs per SM no faster than the other kernels).
// us before -> reading ahead, by ids per bag, one resident wave of bags (W 1) and many:
//   fp32, 32 vectors   3: 368 -> 503   5.5: 257 -> 264   10, W 1 / 3 / 24: 13.2 / 25.1 / 122 -> 11.4 / 22.0 / 107   25: 782 -> 693
//         16 vectors   2: 190 -> 235   6, W 1 / 24: 11.1 / 100 -> 10.3 / 95   15, W 3 / 24: 33 / 178 -> 28 / 151
//          8 vectors   four rows: 4: 153 -> 146, but 35 M ids over 50 M rows 839 -> 883   10, W 24: 153 -> 145
//          4 vectors   3, W 24: 99 -> 91   8: 148 -> 140   15: 205 -> 185
//   bf16, 32 vectors   12, W 6 / 24: 52 / 169 -> 52 / 171   25: 281 -> 247
//         16 vectors   4: 331 -> 337   5.5, W 1 / 24: 30.8 / 195 -> 27.1 / 182   9, W 1 / 24: 14.5 / 160 -> 12.9 / 144   12: 634 -> 567
//          8 vectors   5, W 24: 136 -> 116   15: 248 -> 214   20: 531 -> 461   (four rows: 2, W 24 / 346: 91 -> 85, 1149 -> 1245)
//          4 vectors   four rows: 4, W 24: 136 -> 122   15: 258 -> 234
// Inside a step, with bags of eight ids and more: one field at a time, not read ahead | bag order | field order:
//   fp32, 32 / 8 / 4 vectors, 10 ids: 574 | 590 | 612, 400 | 423 | 405, 422 | 503 | 455
//         16 vectors, 10 and 20 ids: 670 | 612 | 673, 705 | 691 | 680; 65 M ids over 10 M rows 1863 | 1791 | 1885
//   bf16, 32 vectors, 20 ids: 490 | 459 | 481; 16, 12 ids: 667 | 596 | 649
//         4 vectors, 12 ids: 619 | 622 | 555, but with hashed ids 911 | - | 1020, 9 and 20 ids 732 | - | 786, 969 | - | 1115
//          8 vectors, 10 ids: 534 | 455 | 478, 105 M of 20 ids over 20 M rows 1667 | 1710 | 1509, over 100 M rows 1675 | - | 1515
__host__ __device__ constexpr int ahead_ctas(int rows) { return rows == 8 ? 4 : 5; }  // per SM
// The grid in waves of CTAs, W as above.  One wave where it leaves a lane group few turns: W 48, 9 ids in 1 / 2 / 4 waves,
// fp32 16 and 32 vectors 215 / 232 / 234 and 197 / 215 / 212 us.  With many turns the SMs drift apart, and a warp that meets
// several long bags ends late; 9 ids in 1 / 8 / 16 waves, without reading ahead in brackets:
//   fp32, 32 vectors, W 70 / 130 / 346   299 / 294 / 300 (297), 560 / 526 / 520 (527), 1485 / 1371 / 1326 (1338)
//         16 vectors                     318 / 328 / 330 (344), 589 / 589 / 580 (611), 1579 / 1538 / 1488 (1560)
//   bf16, 16 vectors                     421 / 408 / 413 (445), 771 / 740 / 732 (814), 2046 / 1940 / 1887 (2143)
//   one bag in 5000 of 4500 ids, fp32, 32 vectors, W 70 / 130  1492 / 698 / 707 (1264), 1751 / 1244 / 954 (1504)
// (32 waves: W 70 322, W 346 1330.)  In field order every wave would go through all fields: 16 vectors 1667 -> 1800.
inline int ahead_waves(int64_t W, bool by_field) { return by_field || W < 64 ? 1 : (int)(W < 128 ? W / 8 : 16); }
constexpr int ahead_rows(int G, bool bf16) { return G == (bf16 ? 4 : 8) ? 4 : 8; }
constexpr bool ahead_in_fields(int G, bool bf16) { return G == (bf16 ? 8 : 16); }  // at all, from 16 ids on
enum class Ahead { kNo, kBags, kFields };
inline Ahead ahead_of(int G, bool bf16, bool fields_known, int64_t bags_per_cta, int64_t n_bags, int64_t nnz) {
  if (G < 4 || n_bags < (int64_t)kNumSM * kFlatCtas * bags_per_cta) return Ahead::kNo;
  auto ids = [&](int64_t per_bag) { return nnz >= per_bag * n_bags; };
  const bool narrow = G == 4 || (!bf16 && G != 16);  // not inside a step
  const int64_t from = bf16 ? (G == 32 ? 16 : G == 16 ? 5 : G == 8 ? 4 : 3) : (G >= 32 || G == 8 ? 8 : G == 16 ? 6 : 3);
  if (!ids(from) || (narrow && fields_known)) return Ahead::kNo;
  return ahead_in_fields(G, bf16) && fields_known && ids(16) ? Ahead::kFields : Ahead::kBags;
}

// Whether rows of up to 5/8 of a lane group's vectors are packed lane by lane: not where the bags are few, when a warp's
// longer chain of bags is all there is.  Not packed -> packed, W as above, us on tables that L2 holds, at 12 ids:
//   fp32, 5 vectors     W 0.2 / 1 / 1.3 / 2 / 3   5.1 -> 5.0, 7.9 -> 9.1, 10.3 -> 9.3, 13.3 -> 12.4, 18.9 -> 15.7
//         10 vectors                              5.1 -> 4.8, 7.6 -> 7.9, 9.2 -> 8.1, 12.1 -> 10.5, 16.9 -> 13.9
//   bf16, 5 vectors     W 0.2 / 1 / 1.6 / 2 / 3   5.8 -> 7.3, 10.0 -> 11.1, 14.3 -> 13.6, 16.9 -> 15.9, 24.7 -> 20.3
//         (larger tables, W 1.6 / 2 / 2.5 / 3     26.7 -> 29.6, 30.7 -> 34.7, 35.8 -> 34.7, 41.0 -> 37.7)
inline bool fwd_packs(int nvec, int G, bool bf16, int64_t n_bags) {
  const int64_t per_wave = (int64_t)kNumSM * kFlatCtas * (kFlatThreads / G);
  return row_packs_narrow(nvec, G) && 10 * n_bags >= (bf16 ? 25 : 12) * per_wave;
}

// The same with a bag's ids held by the lanes of its group, one each, and everything asked for ahead: while a bag's
// rows are on their way, so are the next bag's ids and the offsets of the one after it.  What is left of the chain
// offsets -> ids -> rows is the last step.  Lanes of a warp go through their bags together, to the longest of them
// (the ids are handed round by shuffles).  BY_FIELD: bags in field-major order.
// A lane group has its bags beforehand, so a bag of very many ids would hold up the others of its warp, and two in one warp
// each other: all lanes take it together, a lane group every 32 / G-th step of its rows, and the groups' sums are added up.
// One bag in 5000 of 5000 ids, 19 ids on average, W 12, not read ahead | ahead | long bags shared: fp32 8 vectors 1074 | 1527 |
// 664 us, 4 vectors 1054 | 1571 | 425, bf16 16 vectors 1231 | 674 | 455, 8 vectors 1270 | 1425 | 477, 4 vectors 1225 | 1602 |
// 512; inside a step, field order, fp32 16 vectors, W 130: 2262 | 2395 | 1679.  Not with fp32 rows of 16 vectors in bag order,
// whose ordinary bags take 3% longer with that code beside them (215 -> 221; in field order 1665 -> 1693, 1763 not read ahead).
constexpr uint32_t kLongBag = 256;
template <int G, bool BF16, bool BY_FIELD, int U>
__global__ void __launch_bounds__(kFlatThreads, ahead_ctas(U))
embbag_fwd_ahead_kernel(const void* __restrict__ table, int64_t n_rows, int dim,
                        const int32_t* __restrict__ row_ids, int64_t nnz,
                        const int64_t* __restrict__ bag_offsets, int64_t n_bags,
                        float* __restrict__ pooled, int32_t* status, uint32_t fields, uint32_t samples, bool chained) {
  if (chained) pdl_sync();
  constexpr int EPV = BF16 ? 8 : 4;
  constexpr int PAIRS = EPV / 2;
  constexpr int GPB = kFlatThreads / G;
  constexpr int kStep = U < G ? U : G;  // rows requested at once
  constexpr unsigned kFull = 0xffffffffu;
  constexpr uint32_t kNone = 0xffffffffu;
  const int lg = threadIdx.x & (G - 1);
  const int nvec = dim / EPV;
  const uint32_t limit = (uint32_t)n_rows, row_vecs = (uint32_t)nvec, n_slots = (uint32_t)n_bags;
  const bool lane_on = lg < nvec;
  const uint4* const tbl = static_cast<const uint4*>(table);
  const uint32_t stride = gridDim.x * GPB;
  bool bad = false;
  auto bag_of = [&](uint32_t q) { return BY_FIELD ? q % samples * fields + q / samples : q; };
  // a slot's id range; behind the last slot, and for bad offsets, an empty one
  auto range_of = [&](uint32_t q, uint32_t& begin, uint32_t& len) {
    begin = len = 0;
    if (q >= n_slots) return;
    const uint32_t bag = bag_of(q);
    const int64_t b = bag_offsets[bag], e = bag_offsets[bag + 1];
    if (b < 0 || e < b || e > nnz) {
      if (lg == 0) set_status(status, ANTDT_ERR_BAD_OFFSETS);
      return;
    }
    begin = (uint32_t)b;  // nnz < 2^31
    len = (uint32_t)(e - b);
  };
  auto id_at = [&](uint32_t begin, uint32_t len, uint32_t j) {  // kNone: no row
    return j < len ? (uint32_t)__ldg(row_ids + begin + j) : kNone;
  };
  uint32_t q = blockIdx.x * GPB + threadIdx.x / G;
  uint32_t begin, len, nbegin, nlen;
  range_of(q, begin, len);
  uint32_t id = id_at(begin, len, lg);
  range_of(q + stride, nbegin, nlen);  // fewer than 2^31 slots and three strides below 2^24: no slot number wraps
  while (__any_sync(kFull, q < n_slots)) {
    const uint32_t next_id = id_at(nbegin, nlen, lg);
    uint32_t fbegin, flen;
    range_of(q + 2 * stride, fbegin, flen);
    uint32_t longest = __reduce_max_sync(kFull, len);
    uint64_t acc[PAIRS];
    auto clear = [&] {
#pragma unroll
      for (int e = 0; e < PAIRS; ++e) acc[e] = 0ull;
    };
    // kStep rows, which lanes j0 and on of the group hold in `ids`
    auto add_rows = [&](uint32_t ids, uint32_t j0) {
      uint4 v[kStep];
#pragma unroll
      for (int t = 0; t < kStep; ++t) {
        const uint32_t x = __shfl_sync(kFull, ids, j0 + t, G);
        v[t] = x != kNone && lane_on ? __ldg(tbl + (size_t)x * row_vecs + lg) : make_uint4(0u, 0u, 0u, 0u);
      }
#pragma unroll
      for (int t = 0; t < kStep; ++t) {
        if (BF16) {
          acc[0] = f32x2_add(acc[0], f32x2_pack(v[t].x << 16, v[t].x & 0xffff0000u));
          acc[1] = f32x2_add(acc[1], f32x2_pack(v[t].y << 16, v[t].y & 0xffff0000u));
          acc[2] = f32x2_add(acc[2], f32x2_pack(v[t].z << 16, v[t].z & 0xffff0000u));
          acc[3] = f32x2_add(acc[3], f32x2_pack(v[t].w << 16, v[t].w & 0xffff0000u));
        } else {
          acc[0] = f32x2_add(acc[0], f32x2_pack(v[t].x, v[t].y));
          acc[1] = f32x2_add(acc[1], f32x2_pack(v[t].z, v[t].w));
        }
      }
    };
    auto store = [&] {
      ulonglong2* o = reinterpret_cast<ulonglong2*>(pooled + (size_t)bag_of(q) * dim + (size_t)lg * EPV);
      o[0] = make_ulonglong2(acc[0], acc[1]);
      if (BF16) o[1] = make_ulonglong2(acc[2], acc[3]);
    };
    bool stored = q >= n_slots;
    if ((BF16 || BY_FIELD ? G < 32 : G < 16) && longest >= kLongBag) {
      const uint32_t lane = threadIdx.x & 31;
      for (unsigned todo = __ballot_sync(kFull, lg == 0 && len >= kLongBag); todo; todo &= todo - 1u) {
        const int from = __ffs((int)todo) - 1;
        const uint32_t b = __shfl_sync(kFull, begin, from), l = __shfl_sync(kFull, len, from);
        clear();
        uint32_t mine = id_at(b, l, lane);
        for (uint32_t base = 0; base < l; base += 32) {
          const uint32_t later = id_at(b, l, base + 32 + lane);
          bad |= mine >= limit && base + lane < l;
          if (mine >= limit) mine = kNone;
#pragma unroll 1
          for (uint32_t j0 = 0; j0 < G; j0 += kStep) add_rows(mine, j0);
          mine = later;
        }
#pragma unroll
        for (int o = G; o < 32; o <<= 1)
#pragma unroll
          for (int e = 0; e < PAIRS; ++e) acc[e] = f32x2_add(acc[e], __shfl_xor_sync(kFull, acc[e], o));
        if (lane - lg == from) {
          if (lane_on) store();
          stored = true;
          len = 0;
          id = kNone;
        }
      }
      longest = __reduce_max_sync(kFull, len);
    }
    clear();
    for (uint32_t base = 0; base < longest; base += G) {
      if (base > 0) id = id_at(begin, len, base + lg);
      bad |= id >= limit && base + lg < len;
      if (id >= limit) id = kNone;
#pragma unroll 1
      for (uint32_t j0 = 0; j0 < G && base + j0 < longest; j0 += kStep) add_rows(id, j0);
    }
    if (!stored && lane_on) store();
    q += stride;
    id = next_id; begin = nbegin; len = nlen; nbegin = fbegin; nlen = flen;
  }
  if (bad) set_status(status, ANTDT_ERR_ID_OUT_OF_RANGE);
}

template <int G, int VPL, bool BF16, bool PACKED>
void launch_fwd(const void* table, int64_t n_rows, int dim, const int32_t* row_ids, int64_t nnz,
                const int64_t* bag_offsets, int64_t n_bags, float* pooled, int32_t* status,
                cudaStream_t s, int fields, bool chained) {
  constexpr bool flat = VPL == 1;  // rows of up to 512 bytes
  const int64_t gpb = row_groups(flat ? kFlatThreads : kFwdThreads, dim / (BF16 ? 8 : 4), G, PACKED);
  int64_t grid = (n_bags + gpb - 1) / gpb, sample_blocks = 0;
  if (fields > 0 && n_bags % fields == 0) {
    sample_blocks = (n_bags / fields + gpb - 1) / gpb;
    grid = sample_blocks * fields;
  } else {
    fields = 0;
  }
  const int waves = flat && fields == 0 ? stride_waves(G, gpb, BF16, n_bags, nnz) : 0;
  // (fp32 rows that would be packed were the bags more: 12 ids, W 1: 7.9 -> 9.0)
  const bool may_ahead = flat && !PACKED && (BF16 || !row_packs_narrow(dim / 4, G));
  const Ahead ahead = may_ahead ? ahead_of(G, BF16, fields > 0, gpb, n_bags, nnz) : Ahead::kNo;
  if constexpr (flat && !PACKED && G >= 4) {
    constexpr int U = ahead_rows(G, BF16);
    const int64_t cap = (int64_t)kNumSM * ahead_ctas(U) * ahead_waves(n_bags / (kNumSM * kFlatCtas * gpb), ahead == Ahead::kFields);
    const unsigned ctas = (unsigned)std::min((n_bags + gpb - 1) / gpb, cap);
    if constexpr (ahead_in_fields(G, BF16)) {
      if (ahead == Ahead::kFields) {
        ANTDT_LAUNCH("embbag_fwd", (embbag_fwd_ahead_kernel<G, BF16, true, U>), ctas, kFlatThreads, 0, s, table, n_rows, dim,
                     row_ids, nnz, bag_offsets, n_bags, pooled, status, (uint32_t)fields, (uint32_t)(n_bags / fields), chained);
        return;
      }
    }
    if (ahead == Ahead::kBags) {
      ANTDT_LAUNCH("embbag_fwd", (embbag_fwd_ahead_kernel<G, BF16, false, U>), ctas, kFlatThreads, 0, s, table, n_rows, dim,
                   row_ids, nnz, bag_offsets, n_bags, pooled, status, 1u, (uint32_t)n_bags, chained);
      return;
    }
  }
  if (waves > 0) {
    ANTDT_LAUNCH("embbag_fwd", (embbag_fwd_stride_kernel<G, BF16, PACKED>), (unsigned)(kNumSM * kFlatCtas * waves),
                 kFlatThreads, 0, s, table, n_rows, dim, row_ids, nnz, bag_offsets, n_bags, pooled, status, chained);
  } else if (flat && fields > 0) {
    ANTDT_LAUNCH("embbag_fwd", (embbag_fwd_flat_kernel<G, BF16, true, PACKED>), (unsigned)grid, kFlatThreads, 0, s,
                 table, n_rows, dim, row_ids, nnz, bag_offsets, n_bags, pooled, status, fields, sample_blocks, chained);
  } else if (flat) {
    ANTDT_LAUNCH("embbag_fwd", (embbag_fwd_flat_kernel<G, BF16, false, PACKED>), (unsigned)grid, kFlatThreads, 0, s,
                 table, n_rows, dim, row_ids, nnz, bag_offsets, n_bags, pooled, status, fields, sample_blocks, chained);
  } else if (fields > 0) {
    ANTDT_LAUNCH("embbag_fwd", (embbag_fwd_kernel<G, VPL, BF16, true>), (unsigned)grid, kFwdThreads, 0, s,
                 table, n_rows, dim, row_ids, nnz, bag_offsets, n_bags, pooled, status, fields, sample_blocks, chained);
  } else {
    ANTDT_LAUNCH("embbag_fwd", (embbag_fwd_kernel<G, VPL, BF16, false>), (unsigned)grid, kFwdThreads, 0, s,
                 table, n_rows, dim, row_ids, nnz, bag_offsets, n_bags, pooled, status, fields, sample_blocks, chained);
  }
}

template <bool BF16>
int32_t dispatch_fwd(int nvec, const void* table, int64_t n_rows, int dim, const int32_t* row_ids,
                     int64_t nnz, const int64_t* bag_offsets, int64_t n_bags, float* pooled,
                     int32_t* status, cudaStream_t s, int fields, bool chained) {
#define FWD_CASE(G, VPL)                                                                      \
  if (VPL == 1 && fwd_packs(nvec, G, BF16, n_bags))                                           \
    launch_fwd<G, VPL, BF16, (VPL == 1 && G > 2)>(table, n_rows, dim, row_ids, nnz, bag_offsets, n_bags, pooled, status, \
                                                  s, fields, chained);                        \
  else                                                                                        \
  launch_fwd<G, VPL, BF16, false>(table, n_rows, dim, row_ids, nnz, bag_offsets, n_bags, pooled,     \
                           status, s, fields, chained);                                       \
  return ANTDT_OK;
  if (nvec <= 1) { FWD_CASE(1, 1) }
  if (nvec <= 2) { FWD_CASE(2, 1) }
  if (nvec <= 4) { FWD_CASE(4, 1) }
  if (nvec <= 8) { FWD_CASE(8, 1) }
  if (nvec <= 16) { FWD_CASE(16, 1) }
  if (nvec <= 32) { FWD_CASE(32, 1) }
  if (nvec <= 64) { FWD_CASE(32, 2) }
  if (nvec <= 128) { FWD_CASE(32, 4) }
  if (nvec <= 256) { FWD_CASE(32, 8) }
#undef FWD_CASE
  return ANTDT_ERR_INVALID_ARG;
}

}  // namespace
}  // namespace antdt

namespace antdt {
// The entry point's body; bags_per_sample > 0 (the step knows it) selects the field-major order.
int32_t fwd_impl(const void* table, int32_t dtype, int64_t n_rows, int32_t dim, const int32_t* row_ids,
                 int64_t nnz, const int64_t* bag_offsets, int64_t n_bags, float* pooled,
                 int32_t* dev_status, void* stream, int32_t bags_per_sample, bool beside) {
  if (n_bags < 0 || nnz < 0 || n_rows < 1 || n_rows >= (1ll << 31) || nnz >= (1ll << 31) ||
      n_bags >= (1ll << 31) || dim < 1 || dim > 1024)
    return ANTDT_ERR_INVALID_ARG;
  if (dtype != ANTDT_F32 && dtype != ANTDT_BF16) return ANTDT_ERR_INVALID_ARG;
  if (dim % (dtype == ANTDT_BF16 ? 8 : 4)) return ANTDT_ERR_INVALID_ARG;
  if (n_bags == 0) return ANTDT_OK;
  if (!table || !bag_offsets || !pooled || (nnz > 0 && !row_ids)) return ANTDT_ERR_INVALID_ARG;
  if (!aligned16(table) || !aligned16(pooled)) return ANTDT_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  PdlScope pdl(!beside && nnz <= kPdlMaxItems && n_bags <= kPdlMaxItems);
  // Field-major order pays when a bag's id list fills a 32-byte sector (eight ids or more on
  // average): measured -12% on 100 fields x 10 ids x 256-byte rows, -2% on 40 x 20 x 128-byte rows,
  // but +8% on 30 fields x 4.5 ids, where the scattered id reads cost more than the rows gain.
  const int fields = (bags_per_sample > 1 && nnz >= 8 * n_bags) ? bags_per_sample : 0;
  int32_t rc;
  if (dtype == ANTDT_BF16)
    rc = dispatch_fwd<true>(dim / 8, table, n_rows, dim, row_ids, nnz, bag_offsets, n_bags, pooled,
                            dev_status, s, fields, !beside);
  else
    rc = dispatch_fwd<false>(dim / 4, table, n_rows, dim, row_ids, nnz, bag_offsets, n_bags,
                             pooled, dev_status, s, fields, !beside);
  if (rc != ANTDT_OK) return rc;
  return cuda_ok();
}
}  // namespace antdt

extern "C" int32_t antdt_embbag_fwd(const void* table, int32_t dtype, int64_t n_rows, int32_t dim,
                                    const int32_t* row_ids, int64_t nnz,
                                    const int64_t* bag_offsets, int64_t n_bags, float* pooled,
                                    int32_t* dev_status, void* stream) {
  return antdt::fwd_impl(table, dtype, n_rows, dim, row_ids, nnz, bag_offsets, n_bags, pooled,
                         dev_status, stream, 0);
}
