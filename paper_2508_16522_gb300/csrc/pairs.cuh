// pairs.cuh -- candidate pairs on their way to the pair buffer, shared by the
// two sweeps (sweep.cu: per tile with run state; windows.cu: per window of
// candidates): the pair key, the filter of dense inputs and the chunks a warp
// reserves.
#pragma once
#include "grt_internal.cuh"

namespace grt {
namespace {

__device__ __forceinline__ uint64_t pair_key(int src, int dst, int key_bits) {
  return ((uint64_t)(uint32_t)src << key_bits) | (uint32_t)dst;
}

// The pair filter of dense inputs: 2^filt_bits slots of 4 bytes for each target
// task (filt_bits >= 1), in pairs of slots chosen by the source's low bits. A
// slot holds a source (kEmptySlot: free), so it names its pair exactly. False
// when one of the two already held the pair, i.e. some tile emitted it before
// (its write stands, or the buffer overflowed and the sweep runs again without
// the filter). Lossy only towards keeping duplicates: a source that finds both
// slots taken replaces the second one. Most lookups of a dense input find their
// pair: a plain load answers those, and only a miss pays the exchange. The
// slots of one target are neighbours, so a task's pairs share sectors (a hash
// of the whole pair took a DRAM sector for each lookup of the 1M-launch trace).
constexpr uint32_t kEmptySlot = 0xFFFFFFFFu;

__device__ __forceinline__ uint32_t* filt_slots(const SweepOut& o, uint32_t src, uint32_t dst) {
  return o.filt + (((size_t)dst << o.filt_bits) | ((src << 1) & ((1u << o.filt_bits) - 1u)));
}

__device__ __forceinline__ uint2 filt_look(const uint32_t* slots) {
  return __ldcg(reinterpret_cast<const uint2*>(slots));
}

// src after a look that did not find it
__device__ __forceinline__ bool filt_take(uint32_t* slots, uint2 seen, uint32_t src) {
  return atomicExch(slots + (seen.x == kEmptySlot ? 0 : 1), src) != src;
}

__device__ __forceinline__ bool filt_fresh(const SweepOut& o, uint64_t key) {
  const uint32_t src = (uint32_t)(key >> o.key_bits), dst = (uint32_t)(key & ((1ull << o.key_bits) - 1ull));
  uint32_t* const p = filt_slots(o, src, dst);
  const uint2 v = filt_look(p);
  return v.x != src && v.y != src && filt_take(p, v, src);
}

// Where `need` pairs of one flush go: the first `split` fill the rest of the
// warp's current chunk (from `a`), the others start a fresh contiguous run of
// chunks (at `b`). Only a warp's last, partly used chunk is ever left with
// holes, so the cursor exceeds the pairs written by less than one chunk per
// warp (convergent). X holds the warp's chunk_base and chunk_left.
struct PairDst {
  unsigned long long a, b;
  uint32_t split;
};

template <class X>
__device__ PairDst reserve_pairs(X& x, const SweepOut& o, uint32_t need) {
  PairDst d{x.chunk_base, 0ull, need};
  if (x.chunk_left >= need) {
    x.chunk_base += need;
    x.chunk_left -= need;
    return d;
  }
  d.split = x.chunk_left;
  const uint32_t rest = need - x.chunk_left;
  const uint32_t k = (rest + o.chunk - 1) / o.chunk;
  unsigned long long nb = 0;
  if (x.lane == 0) nb = atomicAdd(o.cursor, (unsigned long long)k * o.chunk);
  d.b = __shfl_sync(0xffffffffu, nb, 0);
  x.chunk_base = d.b + rest;
  x.chunk_left = k * o.chunk - rest;
  return d;
}

__device__ __forceinline__ unsigned long long pair_pos(const PairDst& d, uint32_t i) {
  return i < d.split ? d.a + i : d.b + (i - d.split);
}

}  // namespace
}  // namespace grt
