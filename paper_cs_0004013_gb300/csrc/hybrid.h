// The sort by value buckets (hybrid.cu): its launches' arguments.
#pragma once

#include "rs_internal.h"

namespace rs {

// 32-bit shared counters of all of them are 192 KiB; the two digits of a split allow 65,536.
constexpr uint32_t kHybMaxBuckets = 49152;

// Which way the sort goes, decided on the device (HybCtrl::route).
enum : uint32_t { kHybRadix = 1, kHybBuckets = 2 };

struct HybCtrl {
  uint64_t lo, hi;     // the value map (hybrid.cu, ValueMap)
  uint32_t sh, mult;
  uint32_t route;
  uint32_t done;       // count blocks that have finished (none when the sample chose the radix passes)
  uint32_t tiles_b;    // tiles of the second split
  uint32_t reserved[7];
};
static_assert(sizeof(HybCtrl) == 64, "one cache line or less");

struct HybArgs {
  const void* keys_in;
  void* keys_out;
  void* keys_alt;
  const void* vals_in;
  void* vals_out;
  void* vals_alt;
  uint32_t n;
  KeyXform x;       // order map of 32-bit keys
  KeyXform64 x64;   // of 64-bit keys
  uint32_t buckets;     // B
  uint32_t low_bits;    // the second split's digit: the bucket's low bits
  uint32_t groups;      // digits of the first split
  uint32_t bucket_cap;  // keys the local sort takes
  uint32_t split_tile;  // keys of a split tile
  SampleRule rule;
  HybCtrl* ctrl;
  uint32_t* counts;         // [B], zero before the counts
  uint32_t* starts;         // [B + 1]
  uint32_t* cursors;        // [B]
  uint32_t* group_cursors;  // [256]
  uint32_t* group_tiles;    // [257]
  uint32_t* tickets;        // [2], zero before the splits (sorts with payloads)
  uint32_t* status;         // [tiles + second split's tiles][256], zero before the splits (with payloads)
  uint4* clear;             // cleared by the sample
  size_t clear_vec4;
  uint4* zero_ptr;          // cleared by the counts
  size_t zero_vec4;
  uint32_t* err;
};

// Keys of the sample for so many buckets.
constexpr uint32_t hyb_sample_keys(uint32_t buckets) { return buckets <= kFusedMaxBuckets ? kFusedSampleKeys : kSampleKeys; }
enum class HybStep { kSample, kCount, kSplit0, kSplit1, kBuckets };
struct HybShape {
  uint32_t split_tile;   // keys of a split tile
  uint32_t bucket_cap;   // keys the local sort takes
  uint32_t bucket_mean;  // keys per bucket that the plan aims at
};
HybShape hyb_shape(int key_bytes, int val_bytes);
cudaError_t prepare_hybrid();
cudaError_t launch_hybrid(const HybArgs& a, HybStep step, int key_bytes, int val_bytes, unsigned sms, cudaStream_t s);

}  // namespace rs
