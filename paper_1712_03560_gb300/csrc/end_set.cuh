// end_set.cuh -- insertion into the set of (pattern, end) pairs that the piece
// filter and the gram index share.
#pragma once
#include "kernels.h"

namespace oasm {

// The 64-bit finaliser of MurmurHash3 (A. Appleby): spreads keys over the table.
__device__ __forceinline__ unsigned long long mix64(unsigned long long k) {
  k ^= k >> 33;
  k *= 0xff51afd7ed558ccdull;
  k ^= k >> 33;
  k *= 0xc4ceb9fe1a85ec53ull;
  k ^= k >> 33;
  return k;
}

// Inserts key; true if it was not in the set yet.  Sets *full when no free slot
// turns up within the probe bound.
constexpr int kSetProbes = 64;
__device__ __forceinline__ bool insert_key(const EndSet& S, unsigned long long key, bool* full) {
  unsigned long long h = mix64(key) & S.mask;
  for (int i = 0; i < kSetProbes; ++i) {
    const unsigned long long prev = atomicCAS(&S.slots[h], ~0ull, key);
    if (prev == ~0ull) return true;
    if (prev == key) return false;
    h = (h + 1) & S.mask;
  }
  *full = true;
  return false;
}

}  // namespace oasm
