// The map from keys to value buckets (hybrid.cu, fused.cu).
#pragma once

#include "hybrid.h"
#include "rs_device.cuh"

namespace rs {

// The linear map of a key's value to [0, 2^32): bucket = high word of the
// product, place inside the bucket = low word.  Values outside the sampled
// range [lo, hi] fall in the first or last bucket.  32-bit keys take the
// offset and the product in one wide multiply-add: back = -lo * mult.
template <typename K>
struct ValueMap {
  K lo, hi;
  uint32_t sh, mult;
  uint64_t back;
  __device__ __forceinline__ K clamp(K k) const {
    const K t = k > lo ? k : lo;
    return t < hi ? t : hi;
  }
  // the product for a key inside [lo, hi]
  __device__ __forceinline__ uint64_t product(K k) const {
    if constexpr (sizeof(K) == 8) return uint64_t(uint32_t((k - lo) >> sh)) * mult;
    else return uint64_t(k) * mult + back;
  }
  __device__ __forceinline__ uint32_t bucket(K k) const { return uint32_t(product(clamp(k)) >> 32); }
};
template <typename K>
__device__ __forceinline__ ValueMap<K> load_map(const HybCtrl* c) {
  return ValueMap<K>{K(c->lo), K(c->hi), c->sh, c->mult, 0ull - uint64_t(K(c->lo)) * c->mult};
}

}  // namespace rs
