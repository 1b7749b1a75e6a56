// Sort by value buckets: two distributions by the keys' leading value range,
// then every bucket sorted by one block in shared memory.
//
// Paper: the bucketing + local sort pipeline of Sec. 3 (count the keys per
// bucket, cumulative totals, distribution, local sort of each cell's range),
// chosen from a sample of the data as in Sec. 4.2.1, with the radix pipeline
// as the way back.  The buckets are B equal slices of the keys' value range
// (bucket = (key - lowest) * B / range), about 2,048 keys each, reached in two
// distributions (first the bucket's high bits, then its low ones), because a
// distribution to B places at once writes runs too short to be worth a
// memory transaction.  The steps, each one launch:
//   sample   one cluster (one block where buckets are few) reads an evenly spread
//            sample: the value range, and whether the keys are spread evenly
//            enough over it (else the radix passes sort them);
//   counts   keys per bucket in one read; its last block scans them.  A
//            bucket that would not fit the local sort also sends the sort to
//            the radix passes;
//   split    twice: tiles of keys go to their buckets' ranges;
//   buckets  one block per bucket sorts it in place (local.cuh).
// Every kernel returns at once when the sort takes the other way.
//
// Sorts with payloads take stable splits (stable_split.cuh), and a bucket's
// equal keys are ordered by where they are in it.
//
// Against the radix passes (8 digits of 8 bits for 64-bit keys, 4 for 32-bit
// ones), the keys cross memory three times instead of four or eight, and keys
// without payloads need no stable ranking: a key's place in its tile is one
// shared atomic, and a tile's place in a bucket one global atomic.
#include <cstdint>

#include "hybrid.h"
#include "local.cuh"
#include "sample.cuh"
#include "split.cuh"
#include "stable_split.cuh"
#include "value_map.cuh"

namespace rs {
namespace {

constexpr int kSampleThreads = 1024;
constexpr int kCountThreads = 1024;

// Bins of a bucket: the low word of the same product.  EDGE: the first and
// last bucket, which also hold the values outside the sampled range.
template <typename K, int NBITS, bool EDGE>
struct BucketBins {
  static constexpr bool kKnown = true, kLook = false;
  ValueMap<K> m;
  __device__ __forceinline__ uint32_t operator()(K k) const {
    return uint32_t(m.product(EDGE ? m.clamp(k) : k)) >> (32 - NBITS);
  }
  __device__ __forceinline__ bool unique() const { return false; }
};

template <typename K>
struct OrdOf;
template <>
struct OrdOf<uint32_t> {
  using T = Ord32;
  __device__ static T make(const HybArgs& a) { return Ord32{a.x}; }
  __device__ static T identity() { return Ord32{KeyXform{0u, 0u}}; }
};
template <>
struct OrdOf<uint64_t> {
  using T = Ord64;
  __device__ static T make(const HybArgs& a) { return Ord64{a.x64}; }
  __device__ static T identity() { return Ord64{KeyXform64{0u, 0u, 0u}}; }
};

// ------------------------------------------------------------------ sample (sample.cuh)
constexpr int kSampleBlocks = 8, kSmallSampleThreads = 768;
template <int THREADS>
__device__ __forceinline__ void clear_rest(const HybArgs& a) {
  for (size_t i = size_t(blockIdx.x - 1) * THREADS + threadIdx.x; i < a.clear_vec4; i += size_t(kSampleBlocks - 1) * THREADS)
    a.clear[i] = make_uint4(0u, 0u, 0u, 0u);
}
template <typename K>
__global__ void __cluster_dims__(kSampleBlocks, 1, 1) __launch_bounds__(kSampleThreads, 1)
    sample_kernel(const HybArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  launch_next();
  // the blocks other than the first clear what the launches that follow start from
  sample_body<K, kSampleBlocks, kSampleThreads>(static_cast<const K*>(a.keys_in), a.n, a.buckets, OrdOf<K>::make(a),
                                                a.rule, a.ctrl, smem, [&] { clear_rest<kSampleThreads>(a); });
}
// Up to kFusedMaxBuckets buckets a sample as small as the single launch's says as
// much, and one block takes it: 6.3 us instead of 10.5 with 64-bit keys, whose
// 8,192 bind one SM (20,000 even keys 30 us -> 26, clustered ones 93 -> 88).
template <typename K>
__global__ void __launch_bounds__(kSmallSampleThreads, 1) small_sample_kernel(const HybArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  launch_next();
  if (blockIdx.x != 0) return clear_rest<kSmallSampleThreads>(a);
  sample_body<K, 1, kSmallSampleThreads>(static_cast<const K*>(a.keys_in), a.n, a.buckets, OrdOf<K>::make(a), a.rule,
                                         a.ctrl, smem, [] {});
}

// ------------------------------------------------------------------ counts
// Keys per bucket.  32-bit shared counters for every bucket (up to 192 KiB),
// one shared reduction per key; the blocks add them into the global counts.
// The last block to finish scans the counts: the buckets' starts and cursors,
// the tiles of the second split, and whether every bucket fits the local sort.
template <typename K>
__global__ void __launch_bounds__(kCountThreads, 1) bucket_count_kernel(const HybArgs a) {
  extern __shared__ __align__(16) uint32_t sh[];  // [buckets]
  __shared__ uint32_t s_warp[32];
  __shared__ uint32_t s_last;
  const int tid = threadIdx.x;
  const uint32_t B = a.buckets;
  for (uint32_t i = tid; i < B; i += kCountThreads) sh[i] = 0u;  // while the sample is taken
  wait_for_chain();
  if (a.ctrl->route != kHybBuckets) return;
  const ValueMap<K> m = load_map<K>(a.ctrl);
  const auto ord = OrdOf<K>::make(a);
  const uint32_t base = smem_addr(sh);
  __syncthreads();
  const uint32_t n = a.n;
  const size_t stride = size_t(gridDim.x) * kCountThreads;
  auto count = [&](K k) { sh_red_add(base + 4u * m.bucket(ord.map(k)), 1u); };
  // 16-byte vectors between the first and last 16-byte boundary
  constexpr uint32_t PV = 16 / sizeof(K);
  const K* in = reinterpret_cast<const K*>(a.keys_in);
  uint32_t head = uint32_t((PV - (reinterpret_cast<uintptr_t>(in) / sizeof(K)) % PV) % PV);
  if (head > n) head = n;
  const size_t nvec = size_t(n - head) / PV;
  const uint32_t tail = head + uint32_t(nvec * PV);
  if (blockIdx.x == gridDim.x - 1) {
    for (uint32_t i = tid; i < head; i += kCountThreads) count(in[i]);
    for (uint32_t i = tail + tid; i < n; i += kCountThreads) count(in[i]);
  }
  const uint4* v4 = reinterpret_cast<const uint4*>(in + head);
  auto count4 = [&](const uint4& x) {
    if constexpr (sizeof(K) == 4) {
      count(x.x); count(x.y); count(x.z); count(x.w);
    } else {
      count((uint64_t(x.y) << 32) | x.x);
      count((uint64_t(x.w) << 32) | x.z);
    }
  };
  size_t i = size_t(blockIdx.x) * kCountThreads + tid;
  for (; i + 7 * stride < nvec; i += 8 * stride) {
    uint4 x[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) x[q] = ld_stream4(v4 + i + q * stride);
#pragma unroll
    for (int q = 0; q < 8; ++q) count4(x[q]);
  }
  for (; i < nvec; i += stride) count4(ld_stream4(v4 + i));
  // status words of the splits' chained scans
  for (size_t z = size_t(blockIdx.x) * kCountThreads + tid; z < a.zero_vec4; z += stride)
    a.zero_ptr[z] = make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();
  for (uint32_t b = tid; b < B; b += kCountThreads)
    if (sh[b]) atomicAdd(&a.counts[b], sh[b]);
  __threadfence();
  __syncthreads();
  if (tid == 0) s_last = atomicAdd(&a.ctrl->done, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  // the last block: exclusive scan of the counts, a contiguous run of buckets per
  // warp (32 consecutive ones per step: no bank conflicts), the warps' totals scanned between
  const int lane = tid & 31, warp = tid >> 5;
  constexpr uint32_t WARPS = kCountThreads / 32;
  const uint32_t per = (B + WARPS * 32 - 1) / (WARPS * 32);  // steps of a warp
  const uint32_t b0 = uint32_t(warp) * per * 32 + lane;
  uint32_t sum = 0, most = 0;
  for (uint32_t i = 0; i < per; ++i) {
    const uint32_t b = b0 + i * 32;
    const uint32_t c = b < B ? __ldcg(&a.counts[b]) : 0u;
    if (b < B) sh[b] = c;
    sum += c;
    most = c > most ? c : most;
  }
  sum = __reduce_add_sync(0xffffffffu, sum);
  __syncwarp();
  uint32_t run = block_exclusive_sum<kCountThreads>(lane == 0 ? sum : 0u, s_warp);
  run = __shfl_sync(0xffffffffu, run, 0);
  for (uint32_t i = 0; i < per; ++i) {
    const uint32_t b = b0 + i * 32;
    const uint32_t c = b < B ? sh[b] : 0u;
    uint32_t inc = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += y;
    }
    if (b < B) sh[b] = run + inc - c;
    run += __shfl_sync(0xffffffffu, inc, 31);
  }
  const bool over = __syncthreads_or(most > a.bucket_cap);
  if (over) {
    if (tid == 0) a.ctrl->route = kHybRadix;
    return;
  }
  for (uint32_t b = tid; b < B; b += kCountThreads) {
    a.starts[b] = sh[b];
    a.cursors[b] = sh[b];
  }
  if (tid == 0) a.starts[B] = n;
  // groups of the first split: starts and cursors, and the second split's tiles
  const uint32_t groups = a.groups;
  uint32_t g0 = 0, g1 = 0;
  if (tid < int(groups)) {
    g0 = sh[tid << a.low_bits];
    g1 = ((uint32_t(tid) + 1) << a.low_bits) < B ? sh[(tid + 1) << a.low_bits] : n;
    a.group_cursors[tid] = g0;
  }
  const uint32_t tiles = (g1 - g0 + a.split_tile - 1) / a.split_tile;
  const uint32_t first = block_exclusive_sum<kCountThreads>(tid < int(groups) ? tiles : 0u, s_warp);
  if (tid < int(groups)) a.group_tiles[tid] = first;
  if (tid == int(groups) - 1) {
    a.group_tiles[groups] = first + tiles;
    a.ctrl->tiles_b = first + tiles;
  }
}

// ------------------------------------------------------------------- split
// Tile t of the second split: its group (found by every thread looking at
// one), the tiles before the group's first and the tile's keys; through s_job
// (4 words).  Every thread of the block calls it.
struct GroupTile {
  uint32_t base, valid, group, first;
};
__device__ __forceinline__ GroupTile group_tile(const HybArgs& a, uint32_t t, uint32_t tile_keys, uint32_t* s_job) {
  const uint32_t g = threadIdx.x;
  if (g < a.groups) {
    const uint32_t f = a.group_tiles[g], e = a.group_tiles[g + 1];
    if (f <= t && t < e) {
      const uint32_t g0 = a.starts[g << a.low_bits];
      const uint32_t last = (g + 1) << a.low_bits;
      const uint32_t g1 = a.starts[last < a.buckets ? last : a.buckets];
      const uint32_t b = g0 + (t - f) * tile_keys;
      s_job[0] = b;
      s_job[1] = g1 - b < tile_keys ? g1 - b : tile_keys;
      s_job[2] = g;
      s_job[3] = f;
    }
  }
  __syncthreads();
  return GroupTile{s_job[0], s_job[1], s_job[2], s_job[3]};
}

// One distribution of keys without payloads (split.cuh).  LEVEL 0: the
// input's tiles to the groups (the bucket's high bits); LEVEL 1: each group's
// tiles to its buckets (the low bits).
template <typename K, int THREADS, int ITEMS, int LEVEL>
__device__ __forceinline__ void split_body(const HybArgs& a, unsigned char* smem) {
  using L = SplitLayout<K, THREADS, ITEMS>;
  constexpr uint32_t TILE = L::TILE;
  const ValueMap<K> m = load_map<K>(a.ctrl);
  const uint32_t dshift = LEVEL == 0 ? a.low_bits : 0u;
  const uint32_t dmask = LEVEL == 0 ? 0xffu : (1u << a.low_bits) - 1u;
  auto digit = [&](K k) { return (m.bucket(k) >> dshift) & dmask; };
  uint32_t base, valid;
  uint32_t* cursors;
  if constexpr (LEVEL == 0) {
    base = blockIdx.x * TILE;
    valid = a.n - base < TILE ? a.n - base : TILE;
    cursors = a.group_cursors;
  } else {
    if (blockIdx.x >= a.ctrl->tiles_b) return;
    const GroupTile t = group_tile(a, blockIdx.x, TILE, reinterpret_cast<uint32_t*>(smem + L::OFF_JOB));
    base = t.base;
    valid = t.valid;
    cursors = a.cursors + (t.group << a.low_bits);
  }
  const K* in = reinterpret_cast<const K*>(LEVEL == 0 ? a.keys_in : a.keys_alt) + base;
  K* out = reinterpret_cast<K*>(LEVEL == 0 && a.low_bits != 0 ? a.keys_alt : a.keys_out);  // one split: no detour
  const auto ident = OrdOf<K>::identity();
  const auto ordi = LEVEL == 0 ? OrdOf<K>::make(a) : ident;
  if (valid == TILE) split_tile<K, THREADS, ITEMS, true>(in, valid, out, cursors, a.n, digit, ordi, ident, a.err, smem);
  else split_tile<K, THREADS, ITEMS, false>(in, valid, out, cursors, a.n, digit, ordi, ident, a.err, smem);
}

template <typename K, int THREADS, int ITEMS, int MINB, int LEVEL>
__global__ void __launch_bounds__(THREADS, MINB) split_kernel(const HybArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  wait_for_chain();
  if (a.ctrl->route == kHybBuckets) split_body<K, THREADS, ITEMS, LEVEL>(a, smem);
}

// The same with payloads, stable (stable_split.cuh): tiles by ticket, ordered
// by a chained scan, of the whole input (LEVEL 0) or within the group (LEVEL 1).
template <typename K, int VB, int THREADS, int ITEMS, int LEVEL>
__device__ __forceinline__ void stable_split_body(const HybArgs& a, unsigned char* smem) {
  using L = StableSplitLayout<K, VB, THREADS, ITEMS>;
  using V = typename L::V;
  constexpr uint32_t TILE = L::TILE;
  // as many blocks as tiles take tickets
  if (blockIdx.x >= (LEVEL == 0 ? (a.n + TILE - 1) / TILE : a.ctrl->tiles_b)) return;
  uint32_t* s_job = reinterpret_cast<uint32_t*>(smem + L::OFF_JOB);
  uint4* c4 = reinterpret_cast<uint4*>(smem);
  for (int i = threadIdx.x; i < int(L::RANK_BYTES / 16); i += THREADS) c4[i] = make_uint4(0u, 0u, 0u, 0u);
  if (threadIdx.x == 0) s_job[0] = atomicAdd(a.tickets + LEVEL, 1u);
  const ValueMap<K> m = load_map<K>(a.ctrl);
  __syncthreads();
  const uint32_t tile = s_job[0];
  const uint32_t dshift = LEVEL == 0 ? a.low_bits : 0u;
  const uint32_t dmask = LEVEL == 0 ? 0xffu : (1u << a.low_bits) - 1u;
  auto digit = [&](K k) { return (m.bucket(k) >> dshift) & dmask; };
  GroupTile t{0u, 0u, 0u, 0u};
  if constexpr (LEVEL == 0) {
    t.base = tile * TILE;
    t.valid = a.n - t.base < TILE ? a.n - t.base : TILE;
  } else {
    __syncthreads();  // the ticket is read
    t = group_tile(a, tile, TILE, s_job);
  }
  // a digit's first place: its bucket's start (a digit that no bucket has moves nothing)
  auto base = [&](uint32_t d) {
    const uint32_t b = LEVEL == 0 ? d << a.low_bits : (t.group << a.low_bits) + d;
    return a.starts[b < a.buckets ? b : a.buckets];
  };
  const bool to_alt = LEVEL == 0 && a.low_bits != 0;  // one split: no detour
  const K* in = reinterpret_cast<const K*>(LEVEL == 0 ? a.keys_in : a.keys_alt) + t.base;
  const V* vin = reinterpret_cast<const V*>(LEVEL == 0 ? a.vals_in : a.vals_alt) + t.base;
  K* out = reinterpret_cast<K*>(to_alt ? a.keys_alt : a.keys_out);
  V* vout = reinterpret_cast<V*>(to_alt ? a.vals_alt : a.vals_out);
  uint32_t* status = LEVEL == 0 ? a.status : a.status + size_t((a.n + TILE - 1) / TILE) * 256;
  const auto ordi = LEVEL == 0 ? OrdOf<K>::make(a) : OrdOf<K>::identity();
  if (t.valid == TILE)
    stable_split_tile<K, VB, THREADS, ITEMS, true>(in, vin, t.valid, out, vout, a.n, status, tile, t.first, digit, base,
                                                   ordi, a.err, smem);
  else
    stable_split_tile<K, VB, THREADS, ITEMS, false>(in, vin, t.valid, out, vout, a.n, status, tile, t.first, digit, base,
                                                    ordi, a.err, smem);
}

template <typename K, int VB, int THREADS, int ITEMS, int MINB, int LEVEL>
__global__ void __launch_bounds__(THREADS, MINB) stable_split_kernel(const HybArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  wait_for_chain();
  if (a.ctrl->route == kHybBuckets) stable_split_body<K, VB, THREADS, ITEMS, LEVEL>(a, smem);
}

// ----------------------------------------------------------------- buckets
// One block per bucket, in place.  (A loop over a few buckets per block, which
// a sort that goes the other way would leave sooner, spills: 203 us -> 394 for
// 2^26 keys.)
template <typename K, int VB, int THREADS, int ITEMS, int MINB>
__global__ void __launch_bounds__(THREADS, MINB) bucket_sort_kernel(const HybArgs a) {
  constexpr int BITS = 12;
  extern __shared__ __align__(16) unsigned char smem[];
  wait_for_chain();
  if (a.ctrl->route != kHybBuckets) return;
  const ValueMap<K> m = load_map<K>(a.ctrl);
  using V = typename ValueOf<VB>::T;
  const uint32_t b = blockIdx.x, s = a.starts[b], e = a.starts[b + 1];
  if (s == e) return;
  K* io = reinterpret_cast<K*>(a.keys_out) + s;
  V* vio = VB ? reinterpret_cast<V*>(a.vals_out) + s : nullptr;
  auto sort = [&](auto edge, auto mode, auto eo) {
    local_sort_array<THREADS, ITEMS, BITS, VB, decltype(mode)::value, true, false>(io, io, vio, vio, vio, e - s, OrdOf<K>::identity(),
                                                           OrdOf<K>::make(a),
                                                           BucketBins<K, BITS, decltype(edge)::value>{m}, smem, eo);
  };
  const bool edge = b == 0 || b == a.buckets - 1;
  if constexpr (VB == 0) {
    using Alone = std::integral_constant<Vals, Vals::kAlone>;
    if (edge) sort(std::true_type{}, Alone{}, ElemOf<K, false>{});
    else sort(std::false_type{}, Alone{}, ElemOf<K, false>{});
  } else {
    // A key's distance from its bucket's first possible key and its place
    // share a word when they fit: half the work of ordering them side by side.
    // They do from 2^(range bits + place bits - word bits) buckets on: full-range 64-bit
    // keys above 2.8M records, 32-bit ones above 8.4M pairs, 31-bit ones above 4.2M.
    // Below, whole sorts take longer by: 6M full-range pairs 160 us, 31-bit ones 126;
    // 2.5M full-range 64-bit records 124, those of a narrow range 113.
    constexpr int PBITS = THREADS * ITEMS <= 2048 ? 11 : 12;
    static_assert(THREADS * ITEMS <= (1 << PBITS), "a place's bits");
    const uint64_t step = 0xffffffffull / m.mult + 1;  // offsets per bucket, at most
    const uint64_t t0 = ((uint64_t(b) << 32) + m.mult - 1) / m.mult;  // the bucket's first offset
    const int bits = 64 - __clzll((long long)step) + int(m.sh);
    if (!edge && bits + PBITS <= int(sizeof(K) * 8))
      sort(std::false_type{}, std::integral_constant<Vals, Vals::kStaged>{},
           PackedElem<K, PBITS>{K(m.lo + (K(t0) << m.sh))});
    else
      sort(std::true_type{}, std::integral_constant<Vals, Vals::kInPlace>{}, ElemOf<K, true>{});
  }
}

// ------------------------------------------------- first radix pass of keys
// The first executed pass of a radix sort of keys without payloads: there is
// no earlier order to keep, so it is a split by the lowest byte.
__device__ __forceinline__ void first_pass_body(const PassArgs& a, unsigned char* smem) {
  using L = SplitLayout<uint32_t, kSplitThreads, kSplitItems>;
  constexpr uint32_t TILE = L::TILE;
  const Route route = route_of(a.skip, 0, a.num_passes);
  if (!route.active) return;
  const uint32_t base = blockIdx.x * TILE, valid = a.n - base < TILE ? a.n - base : TILE;
  uint32_t* out = route.dst == BUF_OUT ? a.keys_out : a.keys_alt;
  const Ord32 ordi{a.xin}, ordo{route.last ? a.xout : KeyXform{0u, 0u}};
  auto digit = [](uint32_t k) { return k & 0xffu; };
  if (valid == TILE)
    split_tile<uint32_t, kSplitThreads, kSplitItems, true>(a.keys_in + base, valid, out, a.cursors, a.n, digit, ordi,
                                                           ordo, a.err, smem);
  else
    split_tile<uint32_t, kSplitThreads, kSplitItems, false>(a.keys_in + base, valid, out, a.cursors, a.n, digit, ordi,
                                                            ordo, a.err, smem);
}
__global__ void __launch_bounds__(kSplitThreads, kSplitBlocks) first_pass_kernel(const PassArgs p) {
  extern __shared__ __align__(16) unsigned char smem[];
  if (!gated_off(p.gate)) first_pass_body(p, smem);
}

// Shapes per key and payload bytes: the splits' threads, items and blocks per
// SM (ST, SI, SB), the bucket sort's (BT, BI, BB).  MEAN: keys per bucket that
// the plan aims at; a bucket takes half as many again.  GB300, us per launch:
//   32-bit keys, 2^26: bucket sort 128 x 24 at 8 blocks 203, 256 x 12 at 5 230;
//   with a 32-bit payload: splits 384 x 16 at 3 blocks 353 and 320 (256 x 24 at
//   4: 383, 365; 384 x 20 at 3: 361, 341; 512 x 20 at 2: 356, 340), bucket sort
//   256 x 12 at 5 303 (at 4: 331; 128 x 24 at 5: 369; 384 x 8 at 3: 401);
//   64-bit keys, 2^24: bucket sort 256 x 12 101 (128 x 24: 108 to 114).
template <typename K, int VB>
struct Shape;
template <>
struct Shape<uint32_t, 0> {
  static constexpr int ST = kSplitThreads, SI = kSplitItems, SB = kSplitBlocks, BT = 128, BI = 24, BB = 8, MEAN = 2048;
};
template <>
struct Shape<uint64_t, 0> {
  static constexpr int ST = kSplitThreads, SI = kSplitItems / 2, SB = kSplitBlocks, BT = 256, BI = 12, BB = 4,
                       MEAN = 2048;
};
template <>
struct Shape<uint32_t, 4> {
  static constexpr int ST = 384, SI = 16, SB = 3, BT = 256, BI = 12, BB = 5, MEAN = 2048;
};
template <>
struct Shape<uint32_t, 8> {
  static constexpr int ST = 384, SI = 16, SB = 3, BT = 256, BI = 8, BB = 3, MEAN = 1365;
};
template <>
struct Shape<uint64_t, 4> {
  static constexpr int ST = 384, SI = 12, SB = 3, BT = 256, BI = 8, BB = 3, MEAN = 1365;
};
template <>
struct Shape<uint64_t, 8> {
  static constexpr int ST = 384, SI = 12, SB = 3, BT = 256, BI = 8, BB = 3, MEAN = 1365;
};

template <typename K, int VB>
struct Kernels {
  using T = Shape<K, VB>;
  // the larger of a bucket's two ways (keys and places packed, or side by side)
  static constexpr size_t local_smem() {
    if constexpr (VB == 0) {
      return LocalLayout<T::BT, T::BI, 12, K, 0, Vals::kAlone>::SMEM;
    } else {
      constexpr size_t packed = LocalLayout<T::BT, T::BI, 12, K, VB, Vals::kStaged, PackedElem<K, 12>>::SMEM;
      constexpr size_t wide = LocalLayout<T::BT, T::BI, 12, K, VB, Vals::kInPlace>::SMEM;
      return packed > wide ? packed : wide;
    }
  }
  static constexpr uint32_t TILE = uint32_t(T::ST * T::SI), CAP = uint32_t(T::BT * T::BI);
  template <int LEVEL>
  static auto split() {
    if constexpr (VB != 0) return &stable_split_kernel<K, VB, T::ST, T::SI, T::SB, LEVEL>;
    else return &split_kernel<K, T::ST, T::SI, T::SB, LEVEL>;
  }
  static constexpr size_t split_smem() {
    if constexpr (VB != 0) return StableSplitLayout<K, VB, T::ST, T::SI>::SMEM;
    else return SplitLayout<K, T::ST, T::SI>::SMEM;
  }
  static auto buckets() { return &bucket_sort_kernel<K, VB, T::BT, T::BI, T::BB>; }
  static cudaError_t prepare() {
    cudaError_t e = cudaSuccess;
    auto set = [&](const void* f, size_t bytes) {
      if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, int(bytes));
    };
    set(reinterpret_cast<const void*>(&sample_kernel<K>), SampleLayout<K, kSampleBlocks, kSampleThreads>::SMEM);
    set(reinterpret_cast<const void*>(&small_sample_kernel<K>), SampleLayout<K, 1, kSmallSampleThreads>::SMEM);
    set(reinterpret_cast<const void*>(&bucket_count_kernel<K>), size_t(kHybMaxBuckets) * 4);
    set(reinterpret_cast<const void*>(split<0>()), split_smem());
    set(reinterpret_cast<const void*>(split<1>()), split_smem());
    set(reinterpret_cast<const void*>(buckets()), local_smem());
    return e;
  }
  static HybShape shape() { return HybShape{TILE, CAP, uint32_t(T::MEAN)}; }
  static cudaError_t launch(const HybArgs& a, HybStep step, unsigned sms, cudaStream_t s) {
    const unsigned tiles = (a.n + TILE - 1) / TILE;
    switch (step) {
      case HybStep::kSample:
        if (hyb_sample_keys(a.buckets) != kSampleKeys)
          small_sample_kernel<K>
              <<<kSampleBlocks, kSmallSampleThreads, SampleLayout<K, 1, kSmallSampleThreads>::SMEM, s>>>(a);
        else sample_kernel<K>
            <<<kSampleBlocks, kSampleThreads, SampleLayout<K, kSampleBlocks, kSampleThreads>::SMEM, s>>>(a);
        return cudaGetLastError();
      case HybStep::kCount:
        return launch_chained(&bucket_count_kernel<K>, sms, kCountThreads, size_t(a.buckets) * 4, s, true, a);
      case HybStep::kSplit0: return launch_chained(split<0>(), tiles, T::ST, split_smem(), s, true, a);
      case HybStep::kSplit1: return launch_chained(split<1>(), tiles + a.groups, T::ST, split_smem(), s, true, a);
      case HybStep::kBuckets: return launch_chained(buckets(), a.buckets, T::BT, local_smem(), s, true, a);
    }
    return cudaErrorInvalidValue;
  }
};

// f(Kernels) of the key and payload widths.
template <class F>
auto with_kernels(int kb, int vb, F&& f) {
  if (kb == 4) return vb == 0 ? f(Kernels<uint32_t, 0>{}) : vb == 4 ? f(Kernels<uint32_t, 4>{}) : f(Kernels<uint32_t, 8>{});
  return vb == 0 ? f(Kernels<uint64_t, 0>{}) : vb == 4 ? f(Kernels<uint64_t, 4>{}) : f(Kernels<uint64_t, 8>{});
}

}  // namespace

HybShape hyb_shape(int key_bytes, int val_bytes) {
  return with_kernels(key_bytes, val_bytes, [](auto k) { return decltype(k)::shape(); });
}

cudaError_t launch_first_pass(const PassArgs& a, cudaStream_t s) {
  using L = SplitLayout<uint32_t, kSplitThreads, kSplitItems>;
  const unsigned tiles = unsigned((uint64_t(a.n) + L::TILE - 1) / L::TILE);
  return launch_chained(&first_pass_kernel, tiles, kSplitThreads, L::SMEM, s, a.gate != nullptr, a);
}

cudaError_t prepare_hybrid() {
  cudaError_t e = cudaFuncSetAttribute(reinterpret_cast<const void*>(&first_pass_kernel),
                                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       int(SplitLayout<uint32_t, kSplitThreads, kSplitItems>::SMEM));
  for (int kb : {4, 8})
    for (int vb : {0, 4, 8})
      if (e == cudaSuccess) e = with_kernels(kb, vb, [](auto k) { return decltype(k)::prepare(); });
  return e;
}

cudaError_t launch_hybrid(const HybArgs& a, HybStep step, int key_bytes, int val_bytes, unsigned sms, cudaStream_t s) {
  return with_kernels(key_bytes, val_bytes, [&](auto k) { return decltype(k)::launch(a, step, sms, s); });
}

}  // namespace rs
