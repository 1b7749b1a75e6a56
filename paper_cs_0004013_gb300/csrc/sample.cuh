// Whether keys are spread evenly enough over their value range for value
// buckets, from a sample of them.
//
// Paper: the choice of the algorithm from a 1000-point sample of the data
// (Sec. 4.2.1), here of the value range and the evenness that the buckets of
// hybrid.cu and fused.cu need.
#pragma once

#include <cooperative_groups.h>

#include "hybrid.h"
#include "local.cuh"
#include "value_map.cuh"

namespace rs {

// The sample: S keys, one from each of S equal
// stretches of the input at a place inside the stretch that a hash picks (a
// periodic input does not line up with it).  Every block reads an eighth of
// it into the first block's shared memory (one SM alone takes its scattered
// reads one sector at a time), and the first block decides.  The keys count as spread
// evenly when
//  - no slice of the range (of COARSE) holds more than 1.5 times its share of
//    the sample (uniform keys: 128 expected, five standard deviations below);
//  - no bucket holds more than 1.5 times its share of the sample and 12 keys (of
//    the small sample 16: even keys passed it but for one time in 1,000 with 12);
//  - few sampled keys are equal to another one: many equal keys end up in few
//    bins of a bucket, which then takes the digit passes;
//  - the keys differ in enough bytes: the radix passes leave out the others
//    (hyb_rule in api.cu).
// Where buckets are few, one block takes a sample of about a quarter the size: in
// the sorts of one launch (fused.cu) and for few buckets of the others.
template <typename K, int BLOCKS, int THREADS>
struct SampleLayout {
  static constexpr int S = int(BLOCKS > 1 ? kSampleKeys : kFusedSampleKeys);
  static_assert(S % (THREADS * BLOCKS) == 0, "whole rows of the sample");
  static constexpr uint32_t COARSE = BLOCKS > 1 ? 64 : 16;            // slices of the range for the evenness test
  static constexpr uint32_t MAXB = BLOCKS > 1 ? kHybMaxBuckets : kFusedMaxBuckets;
  static constexpr uint32_t FINE = BLOCKS > 1 ? 12 : 16;
  static constexpr int PER = S / THREADS;                       // of the deciding block
  static constexpr int LOADS = S / (THREADS * BLOCKS);          // of every block
  static constexpr int SLOT_BITS = BLOCKS > 1 ? 15 : 13;               // hash slots, in the fine counts' place
  static constexpr size_t SLOT_BYTES = (size_t(1) << SLOT_BITS) * 2;
  static constexpr int WARPS = THREADS / 32;
  static constexpr size_t FINE_BYTES = size_t(MAXB) * 2 > SLOT_BYTES ? size_t(MAXB) * 2 : SLOT_BYTES;  // 16-bit counts
  static_assert(S < 65536 && FINE_BYTES % 16 == 0, "16-bit counts, cleared in 16-byte units");
  static constexpr size_t OFF_KEYS = FINE_BYTES;
  static constexpr size_t OFF_RED = OFF_KEYS + size_t(S) * sizeof(K);
  static constexpr size_t SMEM = OFF_RED + 64 * 8;
};

// The sample of in[0, n) for `buckets` value buckets, to *ctrl.  The blocks
// other than the first call others() and leave after their reads.
template <typename K, int BLOCKS, int THREADS, class Ord, class Others>
__device__ __forceinline__ void sample_body(const K* in, uint64_t n, uint32_t buckets, const Ord& ord,
                                            const SampleRule& rule, HybCtrl* ctrl, unsigned char* smem,
                                            Others&& others) {
  using L = SampleLayout<K, BLOCKS, THREADS>;
  namespace cg = cooperative_groups;
  uint32_t* s_fine = reinterpret_cast<uint32_t*>(smem);
  K* s_keys = reinterpret_cast<K*>(smem + L::OFF_KEYS);
  K* s_red = reinterpret_cast<K*>(smem + L::OFF_RED);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t block = BLOCKS > 1 ? blockIdx.x : 0u;
  const uint32_t stretch = uint32_t(n / L::S);
  K got[L::LOADS];
#pragma unroll
  for (int i = 0; i < L::LOADS; ++i) {
    const uint32_t q = (i * BLOCKS + block) * THREADS + tid;
    uint32_t h = q * 0x9E3779B1u;
    h ^= h >> 15;
    const uint64_t pos = (uint64_t(q) * n) / L::S + (stretch > 1 ? __umulhi(h * 0x85EBCA77u, stretch) : 0u);
    got[i] = ord.map(ld_elem(in + (pos < n ? pos : n - 1)));
  }
  if (block == 0) {
    uint4* f4 = reinterpret_cast<uint4*>(smem);
    for (uint32_t i = tid; i < (buckets + 7) / 8; i += THREADS) f4[i] = make_uint4(0u, 0u, 0u, 0u);
  }
  K key[L::PER];
  if constexpr (BLOCKS > 1) {
    cg::cluster_group cluster = cg::this_cluster();
    // the first block runs: its shared memory may be written
    asm volatile("barrier.cluster.arrive.relaxed.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
    K* to = cluster.map_shared_rank(s_keys, 0);
#pragma unroll
    for (int i = 0; i < L::LOADS; ++i) to[(i * BLOCKS + block) * THREADS + tid] = got[i];
    cluster.sync();
    if (block != 0) {
      others();
      return;
    }
#pragma unroll
    for (int i = 0; i < L::PER; ++i) key[i] = s_keys[i * THREADS + tid];
  } else {
#pragma unroll
    for (int i = 0; i < L::PER; ++i) s_keys[i * THREADS + tid] = key[i] = got[i];
  }

  K lo = ~K(0), hi = 0;
#pragma unroll
  for (int i = 0; i < L::PER; ++i) {
    lo = key[i] < lo ? key[i] : lo;
    hi = key[i] > hi ? key[i] : hi;
  }
  warp_min_max(lo, hi);
  if (lane == 0) {
    s_red[warp] = lo;
    s_red[32 + warp] = hi;
  }
  __syncthreads();
  lo = s_red[lane < L::WARPS ? lane : 0];
  hi = s_red[32 + (lane < L::WARPS ? lane : 0)];
  warp_min_max(lo, hi);
  // a little wider than the sample, so that the values outside it (about
  // 1 / S of the keys on either side) have buckets of their own
  const K ext = (hi - lo) / (L::S / 8);
  ValueMap<K> m;
  m.lo = lo > ext ? lo - ext : K(0);
  m.hi = hi < ~K(0) - ext ? hi + ext : ~K(0);
  const K span = m.hi - m.lo;
  const int bits = span == 0 ? 1 : 64 - __clzll((long long)(uint64_t)span);
  m.sh = bits > 32 ? uint32_t(bits - 32) : 0u;
  const uint64_t range = uint64_t(span >> m.sh) + 1;  // <= 2^32
  m.mult = uint32_t((uint64_t(buckets) << 32) / (range > buckets ? range : uint64_t(buckets) + 1));
  m.back = 0ull - uint64_t(m.lo) * m.mult;
  bool bad = range <= buckets;
  K diff = 0;
  const uint32_t fine_limit = L::FINE + uint32_t(L::S) * 3 / (2 * buckets);
#pragma unroll
  for (int i = 0; i < L::PER; ++i) {
    diff |= key[i] ^ lo;
    const uint32_t b = m.bucket(key[i]);
    const uint32_t at = 16u * (b & 1u);  // two counts to a word
    if (((atomicAdd(&s_fine[b >> 1], 1u << at) >> at) & 0xffffu) >= fine_limit) bad = true;
  }
  __syncthreads();
  if (buckets >= 4 * L::COARSE) {  // a warp per slice
    for (uint32_t c = warp; c < L::COARSE; c += L::WARPS) {
      const uint32_t from = (c * buckets + L::COARSE - 1) / L::COARSE, to = ((c + 1) * buckets + L::COARSE - 1) / L::COARSE;
      uint32_t sum = 0;
      for (uint32_t b = from + lane; b < to; b += 32) sum += reinterpret_cast<const uint16_t*>(s_fine)[b];
      if (__reduce_add_sync(0xffffffffu, sum) * L::COARSE * 2 > uint32_t(L::S) * 3) bad = true;
    }
  }
  __syncthreads();  // (the hash slots take the counts' place)
  // equal keys: each writes its number to a hash slot, and reads back whose
  // number stayed; an equal key's means a duplicate
  uint16_t* s_slot = reinterpret_cast<uint16_t*>(smem);
  auto slot_of = [](K k) { return (uint32_t(k ^ (uint64_t(k) >> 32)) * 0x9E3779B1u) >> (32 - L::SLOT_BITS); };
#pragma unroll
  for (int i = 0; i < L::PER; ++i) s_slot[slot_of(key[i])] = uint16_t(i * THREADS + tid);
  __syncthreads();
  uint32_t dups = 0;
#pragma unroll
  for (int i = 0; i < L::PER; ++i) {
    const uint32_t o = s_slot[slot_of(key[i])];
    dups += o != uint32_t(i * THREADS + tid) && s_keys[o] == key[i];
  }
  dups = __reduce_add_sync(0xffffffffu, dups);
  uint32_t* s_sum = reinterpret_cast<uint32_t*>(s_red);
  const uint32_t diff_lo = __reduce_or_sync(0xffffffffu, uint32_t(diff));
  const uint32_t diff_hi = sizeof(K) == 8 ? __reduce_or_sync(0xffffffffu, uint32_t(uint64_t(diff) >> 32)) : 0u;
  if (lane == 0) {
    s_sum[warp] = dups;
    s_sum[32 + warp] = diff_lo;
    s_sum[64 + warp] = diff_hi;
  }
  bad = __syncthreads_or(bad);
  const int w = lane < L::WARPS ? lane : 0;
  dups = __reduce_add_sync(0xffffffffu, lane < L::WARPS ? s_sum[w] : 0u);
  const uint32_t words[2] = {__reduce_or_sync(0xffffffffu, s_sum[32 + w]), __reduce_or_sync(0xffffffffu, s_sum[64 + w])};
  uint32_t digits = 0;
#pragma unroll
  for (int i = 0; i < int(sizeof(K)); ++i) digits += ((words[i / 4] >> (8 * (i % 4))) & 0xffu) != 0u;
  if (digits < rule.min_digits) bad = true;
  if (dups > (digits <= 3 ? rule.narrow_dups : rule.dups)) bad = true;
  if (tid == 0) {
    HybCtrl* c = ctrl;
    c->lo = m.lo;
    c->hi = m.hi;
    c->sh = m.sh;
    c->mult = m.mult;
    c->done = 0;
    c->tiles_b = 0;
    c->route = bad ? kHybRadix : kHybBuckets;
  }
}

}  // namespace rs
