// Index arithmetic of the kernels that must stay in bounds whatever memory holds, and up to the limits
// of what the entry points accept.  Plain C++ as well, so that its edges are tested on the host.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define ANTDT_HD __host__ __device__ __forceinline__
#else
#define ANTDT_HD inline
#endif

namespace antdt {

// Worker of a resident-sort key (worker << key_bits | row id).  Below 2^worker_bits for every key: after
// a wait that ran out a CTA can read slots that nobody has written, and indexes its tables by this.
ANTDT_HD uint32_t key_worker(uint32_t key, int key_bits, int worker_bits) {
  return (uint32_t)((uint64_t)key >> key_bits) & ((1u << worker_bits) - 1u);
}

// Run index with which a reduction tile that begins at entry o_begin goes on (first: what the sort left in
// tile_first).  Nobody writes it for tiles behind the last sorted entry, which exist when the offsets are bad:
// at most one run starts per entry, so a value above o_begin (a negative one too) is not one, and the
// indices that follow it inside the tile stay below 2^31.
ANTDT_HD int32_t run_index(int32_t first, int64_t o_begin) {
  return (uint32_t)first < (uint32_t)o_begin ? first : (int32_t)o_begin;
}

// The slots that a group of bags fills: span of them (fewer than 2^31), skew (0 to 3) behind the start of an
// aligned group of four.  Slots are counted from there in unsigned 32 bits, four to a lane and 128 to a
// turn: the turn after the last slot of an array of 2^31 - 1 occurrences does not wrap.
constexpr uint32_t kSpanTurn = 128;
struct BagSpan {
  uint32_t skew, total;  // slots skew .. total - 1 are the group's
  ANTDT_HD BagSpan(uint32_t span, uint32_t skew_) : skew(skew_), total(span + skew_) {}
  ANTDT_HD bool holds(uint32_t x) const { return x >= skew && x < total; }
  ANTDT_HD bool whole(uint32_t x) const { return x >= skew && x + 4 <= total; }  // x .. x + 3
};

}  // namespace antdt
