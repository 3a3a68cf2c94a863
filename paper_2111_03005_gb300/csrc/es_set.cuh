// ParES's edge set: open addressing over canonical ids, linear probing from the
// low bits of the id's hash, tombstones on erase.
#pragma once

#include "device_util.cuh"
#include "gesmc_internal.cuh"

namespace gesmc {

constexpr uint32_t kNil = 0xFFFFFFFFu;

__device__ __forceinline__ uint32_t hash32(unsigned long long key) { return (uint32_t)mix64(key); }

// Insert a key that is not in the set into the first empty or tombstone
// slot of its probe sequence from slot s on.  Returns the slot (with
// *tomb = 1 if it held a tombstone), or kNil if the table is full.
__device__ __forceinline__ uint32_t hset_insert(unsigned long long *H, uint32_t mask, unsigned long long key,
                                                uint32_t s, uint32_t *tomb) {
  for (uint32_t n = 0; n <= mask; ++n) {
    const unsigned long long cur = __ldcg(&H[s]);
    if (cur == kEmptyKey || cur == kTombKey) {
      if (atomicCAS(&H[s], cur, key) == cur) {
        *tomb = cur == kTombKey ? 1u : 0u;
        return s;
      }
      continue;  // taken meanwhile: look at the same slot again
    }
    s = (s + 1) & mask;
  }
  return kNil;
}

}  // namespace gesmc
