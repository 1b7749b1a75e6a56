// A whole sort of up to a few million keys in one launch.
//
// Paper: the same radix distribution as the pipeline of separate launches
// (the count loop and cumulative totals of Sec. 3.2, then one stable
// distribution per digit from the low one up, Sec. 3.3.1); only the launch
// structure differs.  For small inputs the pipeline's seven launches (clear,
// histogram, scans, four passes) cost more than the work, so here every tile
// of the array has its own block, all blocks are resident at once (a
// cooperative launch refuses otherwise), and the phases are separated by
// grid-wide barriers instead of launches:
//   1. each block counts the four byte digits of its tile and adds them into
//      the global histograms;                                    barrier
//   2. every block scans the histograms itself (they are small): digit bases
//      and the skip flags (a digit with one bucket holding every key);
//   3. for each executed digit: the block's tile goes through the pass of the
//      half-warp-group kernel (onesweep2.cuh), the lookback ordering the
//      tiles inside the pass;                                     barrier
// One block more than tiles samples the keys (sample.cuh) during phase 1.
// Keys that it found spread evenly over their value range take value buckets
// instead of the passes, in the same launch: each block
// counts its tile's keys per bucket (about as many buckets as blocks);
// barrier; it scans the totals, claims its tile's places and writes the tile
// to its buckets (with a payload, the key and its place in the input, so that
// no order needs to be kept); barrier; the blocks sort the buckets
// (local.cuh).  Three barriers and three trips of a key instead of four or five:
// 277,635 uniform keys 40.9 -> 25.2 us, with payloads 45 -> 31; 2^20 48.9 -> 32.4
// and 59 -> 49; 2.6M keys 72 -> 52 (L2 flushed before each).  Bound by the chain
// of barriers, loads and block-wide steps.  Keys that the sample sends to the
// passes pay nothing that was measured below 500,000 (277,635 clustered keys 34.5 /
// 32.8) and up to 2 us above (2^20: 42 / 43).
// Loads use the L2 path (ld.global.cg): later passes read what other blocks
// wrote earlier in the same launch.  Every barrier wait is bounded: a block
// that waits too long raises the device error word and goes on, so the
// launch always ends.
#include <cstdint>

#include "local.cuh"
#include "sample.cuh"
#include "onesweep2.cuh"
#include "split.cuh"
#include "value_map.cuh"

namespace rs {
namespace {

constexpr int kFusedThreads = 384;
// Tile shapes (index = fused shape): 384 x 24, 384 x 20 and 384 x 12.  A
// pass of the single launch lasts about one tile's chain of loads, ranking,
// lookback and write-out, so smaller tiles are faster while every tile still
// has an SM of its own (GB300: 2^19 keys in 39.5 us with 384 x 12 against
// 43.8 with 384 x 24) and slower once tiles share SMs (2^20 keys: 50.1
// against 47.4).
constexpr int kFusedItems[kFusedShapes] = {24, 20, 12};
// (The smaller shapes run one tile per SM.)
constexpr int fused_min_blocks(int items) { return items <= 20 ? 1 : 2; }
// Status rows a digit thread reads per lookback round (GB300, clustered data: 2^20
// keys 42.7 us with 8 rows per round, 44.3 with 16 and 44.3 with 32, 2.5M pairs
// in 272 tiles of 384 x 24 78, 82 and 95).
constexpr int kFusedLookback = 8;
// Rounds of a barrier wait (about 64 ns each) before it gives up.
constexpr uint32_t kBarrierSpinLimit = 1u << 21;

// Value buckets: a bucket is sorted by the block's threads, with 24 keys each
// at 384 x 20 tiles, 16 otherwise (the buckets are a third smaller then).
static_assert(int(kFusedMaxBuckets) == 2 * kFusedThreads, "two buckets per thread");
constexpr int fused_bucket_items(int items) { return items == 20 ? 24 : 16; }
constexpr int kFusedBucketBits = 13;

template <int NV, int ITEMS>
struct FusedLayout {
  using L = Onesweep2Layout<kFusedThreads, ITEMS, NV>;
  static constexpr size_t OFF_BASES = (L::SMEM + 15) / 16 * 16;  // [4][256]
  static constexpr size_t OFF_FLAGS = OFF_BASES + 4 * 256 * 4;   // [4] skip flags
  static constexpr size_t END_PASSES = OFF_FLAGS + 16;
  static_assert(SplitLayout<uint32_t, kFusedThreads, ITEMS>::SMEM <= OFF_BASES, "the first pass leaves the bases alone");
  // value buckets: the staged tile (keys, then places), counts of the two
  // half-warps, write-out offsets; the bucket starts stay behind the local sort's space
  static constexpr int BITEMS = fused_bucket_items(ITEMS);
  static constexpr uint32_t BCAP = uint32_t(kFusedThreads * BITEMS);  // keys of a bucket
  using Sample = SampleLayout<uint32_t, 1, kFusedThreads>;
  using B = LocalLayout<kFusedThreads, BITEMS, kFusedBucketBits, uint32_t, NV ? 4 : 0,
                        NV ? Vals::kPlaces : Vals::kAlone>;
  static constexpr size_t OFF_CNT = size_t(L::TILE) * 4 * (1 + NV);
  static constexpr size_t OFF_GOFF = OFF_CNT + 2 * (kFusedMaxBuckets + 1) * 4;
  static constexpr size_t OFF_SUMS = OFF_GOFF + kFusedMaxBuckets * 4;
  static constexpr size_t END_SPLIT = OFF_SUMS + 64 * 4;
  static constexpr size_t OFF_STARTS = ((END_SPLIT > B::SMEM ? END_SPLIT : B::SMEM) + 15) / 16 * 16;
  static constexpr size_t END_BUCKETS = OFF_STARTS + (kFusedMaxBuckets + 4) * 4;
  static constexpr size_t SMEM = END_PASSES > END_BUCKETS ? END_PASSES : END_BUCKETS;
  static_assert(Sample::SMEM <= SMEM, "the sample fits");
};

__device__ __forceinline__ uint32_t ld_acquire(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Arrival number `target` of the launch's monotone barrier counter.  True when
// the sampling block has chosen the value buckets: it arrives with a bit set
// above the count, so that its answer costs no read after the barrier.
constexpr uint32_t kBucketsBit = 1u << 24;
__device__ __forceinline__ bool grid_barrier(uint32_t* bar, uint32_t target, uint32_t* err) {
  uint32_t seen = 0;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(bar, 1u);
    uint32_t spins = 0;
    while (((seen = ld_acquire(bar)) & (kBucketsBit - 1u)) < target) {
      if (++spins > kBarrierSpinLimit) {
        atomicOr(err, kErrTimeout);
        break;
      }
      __nanosleep(32);
    }
    __threadfence();
  }
  return __syncthreads_or(seen & kBucketsBit);
}

// The value buckets' way (see above); false, with nothing written but the
// counts and `bar` advanced by one barrier, when a bucket does not fit the
// local sort (every block comes to the same answer).
template <int NV, int ITEMS>
__device__ __forceinline__ bool fused_buckets(const FusedArgs& a, uint32_t tile, unsigned char* smem,
                                              uint32_t& barriers) {
  using FL = FusedLayout<NV, ITEMS>;
  constexpr uint32_t TILE = FL::L::TILE;
  constexpr int T = kFusedThreads, ROW = kFusedMaxBuckets + 1;
  uint32_t* s_key = reinterpret_cast<uint32_t*>(smem);
  uint32_t* s_place = s_key + TILE;
  uint32_t* s_cnt = reinterpret_cast<uint32_t*>(smem + FL::OFF_CNT);
  uint32_t* s_goff = reinterpret_cast<uint32_t*>(smem + FL::OFF_GOFF);
  uint32_t* s_sums = reinterpret_cast<uint32_t*>(smem + FL::OFF_SUMS);
  uint32_t* s_starts = reinterpret_cast<uint32_t*>(smem + FL::OFF_STARTS);
  const int tid = threadIdx.x, lane = tid & 31;
  const uint32_t tiles = a.tiles, B = a.buckets, n = a.n;
  const uint32_t base = tile * TILE;
  const uint32_t valid = n - base < TILE ? n - base : TILE;
  auto has = [&](int j) { return uint32_t(j * T + tid) < valid; };
  const ValueMap<uint32_t> map = load_map<uint32_t>(a.ctrl);
  // 1. load, count
  uint32_t key[ITEMS];
#pragma unroll
  for (int j = 0; j < ITEMS; ++j) key[j] = has(j) ? ld_stream(a.keys_in + base + j * T + tid) : 0u;
  for (int i = tid; i < 2 * ROW; i += T) s_cnt[i] = 0u;
  __syncthreads();
  const uint32_t row = smem_addr(s_cnt + (lane >> 4) * ROW);
#pragma unroll
  for (int j = 0; j < ITEMS; ++j) {
    key[j] = to_ordered(key[j], a.xf);
    if (has(j)) sh_red_add(row + 4u * map.bucket(key[j]), 1u);
  }
  __syncthreads();
  const uint32_t d0 = 2u * tid;  // this thread's buckets d0 and d0 + 1
  const uint32_t c00 = s_cnt[d0], c01 = s_cnt[d0 + 1];
  const uint32_t t0 = c00 + s_cnt[ROW + d0], t1 = c01 + s_cnt[ROW + d0 + 1];
  if (t0) atomicAdd(a.counts + d0, t0);
  if (t1) atomicAdd(a.counts + d0 + 1, t1);
  grid_barrier(a.bar, gridDim.x + tiles * barriers++, a.err);
  // 2. the buckets' starts and the tile's own scan; places claimed
  const uint32_t g0 = d0 < B ? __ldcg(a.counts + d0) : 0u, g1 = d0 + 1 < B ? __ldcg(a.counts + d0 + 1) : 0u;
  if (__syncthreads_or(g0 > FL::BCAP || g1 > FL::BCAP)) return false;
  uint32_t k0 = 0, k1 = 0;
  if (t0) k0 = atomicAdd(a.cursors + d0, t0);
  if (t1) k1 = atomicAdd(a.cursors + d0 + 1, t1);
  {
    const uint32_t x[2] = {g0 + g1, 0u}, y[2] = {t0 + t1, 0u};
    uint32_t start[2], excl[2], total;
    block_exclusive_sums<T, 2>(x, start, s_sums, &total);
    __syncthreads();
    block_exclusive_sums<T, 2>(y, excl, s_sums, &total);
    s_starts[d0] = start[0];
    s_starts[d0 + 1] = start[0] + g0;
    if (tid == T - 1) s_starts[2 * T] = n;
    s_goff[d0] = start[0] + k0 - excl[0];
    s_goff[d0 + 1] = start[0] + g0 + k1 - (excl[0] + t0);
    s_cnt[d0] = excl[0];
    s_cnt[ROW + d0] = excl[0] + c00;
    s_cnt[d0 + 1] = excl[0] + t0;
    s_cnt[ROW + d0 + 1] = excl[0] + t0 + c01;
  }
  __syncthreads();
  // 3. the tile by buckets, then out
#pragma unroll
  for (int j = 0; j < ITEMS; ++j) {
    if (has(j)) {
      uint32_t p;
      asm volatile("atom.shared.add.u32 %0, [%1], 1;" : "=r"(p) : "r"(row + 4u * map.bucket(key[j])) : "memory");
      s_key[p] = key[j];
      if constexpr (NV != 0) s_place[p] = base + j * T + tid;
    }
  }
  __syncthreads();
  bool oob = false;
#pragma unroll
  for (int j = 0; j < ITEMS; ++j) {
    if (has(j)) {
      const uint32_t i = j * T + tid, k = s_key[i], g = s_goff[map.bucket(k)] + i;
      if (g < n) {
        st_global(a.keys_alt + g, k);
        if constexpr (NV != 0) st_global(a.vals_alt + g, s_place[i]);
      } else {
        oob = true;
      }
    }
  }
  if (oob) atomicOr(a.err, kErrBounds);
  grid_barrier(a.bar, gridDim.x + tiles * barriers++, a.err);
  // 4. the buckets
  for (uint32_t b = tile; b < B; b += tiles) {
    const uint32_t s = s_starts[b], e = s_starts[b + 1];
    if (s == e) continue;
    uint32_t* vout = NV ? a.vals_out + s : nullptr;
    local_sort_array<T, FL::BITEMS, kFusedBucketBits, NV ? 4 : 0, NV ? Vals::kPlaces : Vals::kAlone, true, false>(
        a.keys_alt + s, a.keys_out + s, a.vals_alt + s, vout, a.vals_in, e - s, Ord32{KeyXform{0u, 0u}}, Ord32{a.xf},
        RangeBins<uint32_t, false>{}, smem);
  }
  return true;
}

template <int NV, int ITEMS>
__global__ void __launch_bounds__(kFusedThreads, fused_min_blocks(ITEMS)) fused_sort_kernel(const FusedArgs a) {
  using FL = FusedLayout<NV, ITEMS>;
  using L = typename FL::L;
  extern __shared__ __align__(16) unsigned char smem[];
  uint32_t* s_bases = reinterpret_cast<uint32_t*>(smem + FL::OFF_BASES);
  uint32_t* s_flags = reinterpret_cast<uint32_t*>(smem + FL::OFF_FLAGS);
  uint32_t* s_cnt = reinterpret_cast<uint32_t*>(smem + L::OFF_TBL);  // [4][256] while counting
  const int tid = threadIdx.x;
  const uint32_t tiles = a.tiles, tile = blockIdx.x - (gridDim.x - tiles);
  const uint32_t n = a.n;
  uint32_t barriers = 0;  // barriers passed so far (the n-th of all tiles awaits gridDim.x + (n - 1) * tiles arrivals)
  constexpr bool kFreeFirst = NV == 0;  // keys alone: the first executed pass keeps no order

  // one block more, when value buckets are offered: it takes the sample meanwhile (the first, it starts soonest)
  if (tile >= tiles) {
    sample_body<uint32_t, 1, kFusedThreads>(a.keys_in, n, a.buckets, Ord32{a.xf}, a.rule, a.ctrl, smem, [] {});
    if (tid == 0) {
      const bool buckets = a.ctrl->route == kHybBuckets;  // (written by this thread)
      __threadfence();
      atomicAdd(a.bar, buckets ? 1u + kBucketsBit : 1u);
    }
    return;
  }

  // 1. counts of the tile's four digits (order-mapped keys); the tile's status row cleared
  for (int i = tid; i < 1024; i += kFusedThreads) s_cnt[i] = 0u;
  if (tid < 256) static_cast<uint32_t*>(a.status)[size_t(tile) * 256 + tid] = 0u;
  __syncthreads();
  {
    const uint32_t cnt = smem_addr(s_cnt);
    const uint32_t base = tile * uint32_t(L::TILE);
    const uint32_t valid = n - base < uint32_t(L::TILE) ? n - base : uint32_t(L::TILE);
    uint32_t key[ITEMS];  // (every load before the first count)
#pragma unroll
    for (int i = 0; i < ITEMS; ++i)
      if (uint32_t(i * kFusedThreads + tid) < valid) key[i] = a.keys_in[base + i * kFusedThreads + tid];
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
      if (uint32_t(i * kFusedThreads + tid) < valid) {
        const uint32_t k = to_ordered(key[i], a.xf);
#pragma unroll
        for (uint32_t j = 0; j < 4; ++j) sh_red_add(cnt + 4u * (256u * j + byte_digit(k, 0x4440u | j)), 1u);
      }
    }
  }
  __syncthreads();
  for (int i = tid; i < 1024; i += kFusedThreads)
    if (s_cnt[i]) atomicAdd(a.hist + i, s_cnt[i]);
  const bool buckets = grid_barrier(a.bar, gridDim.x, a.err);  // (the sampling block passes the first barrier only)
  barriers = 1;
  if (buckets && fused_buckets<NV, ITEMS>(a, tile, smem, barriers)) return;

  // 2. bases and skip flags of every digit (each block for itself)
  {
    uint32_t v[4];  // (all four reads before the first scan)
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = tid < 256 ? ld_pass<true>(a.hist + 256 * j + tid) : 0u;
    if (tid < 4) s_flags[tid] = 0u;
    __syncthreads();
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (tid < 256) {
        if (v[j] == n) s_flags[j] = 1u;  // one bucket holds every key: the digit moves nothing
        s_bases[256 * j + tid] = scan256_exclusive(v[j], reinterpret_cast<uint32_t*>(smem + L::OFF_SCAN));
      }
      __syncthreads();
    }
  }

  // 3. the executed passes: the skipped digits are left out; if every digit
  // is skipped the last one still runs (a stable copy into keys_out).  The
  // executed passes alternate between keys_out and the alternate buffer so
  // that the last one lands in keys_out.
  uint32_t order = 0;  // the executed digits, one per byte, lowest first
  int m = 0;
  for (int j = 0; j < 4; ++j)
    if (!s_flags[j]) order |= uint32_t(j) << (8 * m++);
  if (m == 0) {
    order = 3u;
    m = 1;
  }
  for (int e = 0; e < m; ++e) {
    const int j = int((order >> (8 * e)) & 0xffu);
    uint4* t4 = reinterpret_cast<uint4*>(smem + L::OFF_TBL);
    for (int i = tid; i < int(L::TBL / 16); i += kFusedThreads) t4[i] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    const bool to_out = ((m - 1 - e) % 2) == 0;
    const bool from_out = e > 0 && ((m - e) % 2) == 0;
    Tile2Job job;
    job.tile = tile;
    job.n = n;
    job.kin = e == 0 ? a.keys_in : (from_out ? a.keys_out : a.keys_alt);
    job.kout = to_out ? a.keys_out : a.keys_alt;
    job.vin = nullptr;
    job.vout = nullptr;
    if constexpr (NV >= 1) {
      job.vin = e == 0 ? a.vals_in : (from_out ? a.vals_out : a.vals_alt);
      job.vout = to_out ? a.vals_out : a.vals_alt;
    }
    job.xin = e == 0 ? a.xf : KeyXform{0u, 0u};
    job.xout = e == m - 1 ? a.xf : KeyXform{0u, 0u};
    // the status words are clear for the first pass with a chained scan
    job.parity = uint32_t((e - (kFreeFirst ? 1 : 0)) & 1) ^ 1u;
    job.status = a.status;
    job.bases = s_bases + 256 * j;
    job.shift = uint32_t(8 * j);
    job.err = a.err;
    if constexpr (kFreeFirst) {
      if (e == 0) {  // no earlier order to keep: a split by claims (split.cuh)
        const uint32_t sel = 0x4440u | uint32_t(j);
        auto digit = [&](uint32_t k) { return byte_digit(k, sel); };
        const uint32_t base = tile * uint32_t(L::TILE), left = n - base;
        const Ord32 ordi{job.xin}, ordo{job.xout};
        if (left >= uint32_t(L::TILE))
          split_tile<uint32_t, kFusedThreads, ITEMS, true>(job.kin + base, L::TILE, job.kout, a.first_cursors, n, digit,
                                                           ordi, ordo, a.err, smem, job.bases);
        else
          split_tile<uint32_t, kFusedThreads, ITEMS, false>(job.kin + base, left, job.kout, a.first_cursors, n, digit,
                                                            ordi, ordo, a.err, smem, job.bases);
        __syncthreads();
      }
    }
    // one block per SM (the smaller shapes): nothing else hides the payload loads, and registers are free
    constexpr bool EARLY_VALS = NV != 0 && fused_min_blocks(ITEMS) == 1;
    if (!kFreeFirst || e != 0)
      onesweep2_tile<kFusedThreads, ITEMS, NV, uint32_t, false, kFusedLookback, true, EARLY_VALS>(job, smem);
    if (e + 1 < m) grid_barrier(a.bar, gridDim.x + tiles * barriers++, a.err);
  }
}

}  // namespace

uint32_t fused_tile_keys(int shape) { return uint32_t(kFusedThreads * kFusedItems[shape]); }
uint32_t fused_bucket_keys(int shape) { return uint32_t(kFusedThreads * fused_bucket_items(kFusedItems[shape])); }

template <int SH>
struct FusedShape {
  static constexpr int ITEMS = kFusedItems[SH];
  static size_t smem(bool pairs) { return pairs ? FusedLayout<1, ITEMS>::SMEM : FusedLayout<0, ITEMS>::SMEM; }
  static const void* func(bool pairs) {
    return pairs ? reinterpret_cast<const void*>(&fused_sort_kernel<1, ITEMS>)
                 : reinterpret_cast<const void*>(&fused_sort_kernel<0, ITEMS>);
  }
};
static_assert(kFusedShapes == 3, "one FusedShape per entry of kFusedItems");

size_t fused_smem(bool pairs, int shape) {
  return shape == 0 ? FusedShape<0>::smem(pairs) : shape == 1 ? FusedShape<1>::smem(pairs) : FusedShape<2>::smem(pairs);
}
const void* fused_func(bool pairs, int shape) {
  return shape == 0 ? FusedShape<0>::func(pairs) : shape == 1 ? FusedShape<1>::func(pairs) : FusedShape<2>::func(pairs);
}

cudaError_t launch_fused(const FusedArgs& a, unsigned tiles, bool pairs, int shape, cudaStream_t s) {
  FusedArgs args = a;
  args.tiles = tiles;
  void* params[] = {&args};
  return cudaLaunchCooperativeKernel(fused_func(pairs, shape), dim3(tiles + (a.ctrl ? 1u : 0u)), dim3(kFusedThreads), params,
                                     fused_smem(pairs, shape), s);
}

}  // namespace rs
