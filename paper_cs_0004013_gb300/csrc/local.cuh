// One block sorts one array of at most THREADS * ITEMS keys in shared memory.
//
// Paper: the local sort of each cell's keys after the distribution
// (Sec. 3.3).  The paper's cells ran a radix sort digit by digit (Sec. 3.3.1);
// here the keys are first spread over about twice as many bins as there are
// keys by a linear map of their value range (the bucketing of Sec. 3.2 inside
// the block), which leaves the array sorted but for the one to five keys of
// each bin, and short sorting networks over overlapping windows finish it.
// Keys whose values crowd into few bins (many equal keys, tight clusters)
// are sorted digit by digit instead.
//
// Per array of m keys:
//  1. load; unless the caller knows the value range, its minimum and maximum;
//  2. bin = (key - lowest) scaled so that the range fills 2^NBITS bins; one
//     shared atomic per key on the bin's 16-bit count gives the key's turn
//     among the bin's keys (in no particular order);
//  3. exclusive scan of the counts: where each bin starts;
//  4. each key is stored at start[bin] + turn;
//  5. windows of 8 consecutive keys, alternately at offsets 0 and 4, are sorted
//     in registers: by a 19-comparator network in the first round, later by the
//     9-comparator merge of their two halves, which earlier rounds left in
//     order.  A round merges neighbouring runs of 4, so a bin of c keys, which
//     spans at most ceil((c + 3) / 4) such runs, is in order after that many
//     rounds (two for c <= 5);
//  6. out, coalesced.
// Where (unless the caller's map is known to be even) a bin holds more than
// kBinLimit keys, the bins are laid again where the keys are: each bin's share of
// a second set of bins is its share of the keys (its start and count give them), and a key takes the part of that
// share that its place inside the bin points to.  This flattens any density
// that does not change much within a bin (normally distributed floats, wide
// clusters).  Blocks that are crowded still, or that a sample shows to be, sort
// by digits.
// Sorts with payloads are stable: they order (key, place in the input), and
// the payload follows its place.  The digit passes are stable 8-bit ones over
// the digits in which the keys differ, with the lane-mask tables of the tiled pass.
//
// The work is about 55 instructions and 18 shared-memory wavefronts per 32
// keys whatever the key width, against about 40 wavefronts per 8-bit digit
// of the digit passes; what it measured stands at the kernels that use it
// (local_sort_kernel in local.cu, bucket_sort_kernel in hybrid.cu).
#pragma once

#include "elem.cuh"
#include "onesweep.cuh"

namespace rs {

// Keys in the fullest bin: above kBinLimit (eight rounds of windows) the second
// set of bins is laid where there is one; above kLastLimit (sixteen rounds) the
// digit passes take over.  16,000 keys of 1,000 values: digit passes above 29 keys
// 43 us, above 61 18; 14.7M keys of as many values as give 14 to each 254 and 172.
constexpr uint32_t kBinLimit = 29, kLastLimit = 61;
constexpr uint32_t kCrowded = 40;  // mean keys per bin that leave some bin above kLastLimit
// Arrays of more keys are looked at before their bins are laid (up to 0.3 us;
// 16,000 keys of 8 values 32 us -> 25, 4,000 even ones 4.0 -> 4.4).
constexpr uint32_t kLookKeys = 4096;

// What the block orders: the key, or with a payload (key, place in the input).
struct alignas(16) KeyPlace64 {
  uint64_t k;
  uint32_t i;
};
template <typename K, bool PAIRS>
struct ElemOf;
template <>
struct ElemOf<uint32_t, false> {
  using E = uint32_t;
  static __device__ __forceinline__ E make(uint32_t k, uint32_t) { return k; }
  static __device__ __forceinline__ uint32_t key(E e) { return e; }
  static __device__ __forceinline__ uint32_t place(E) { return 0u; }
  static __device__ __forceinline__ E last() { return ~0u; }
};
template <>
struct ElemOf<uint64_t, false> {
  using E = uint64_t;
  static __device__ __forceinline__ E make(uint64_t k, uint32_t) { return k; }
  static __device__ __forceinline__ uint64_t key(E e) { return e; }
  static __device__ __forceinline__ uint32_t place(E) { return 0u; }
  static __device__ __forceinline__ E last() { return ~0ull; }
};
template <>
struct ElemOf<uint32_t, true> {
  using E = uint64_t;
  static __device__ __forceinline__ E make(uint32_t k, uint32_t i) { return (uint64_t(k) << 32) | i; }
  static __device__ __forceinline__ uint32_t key(E e) { return uint32_t(e >> 32); }
  static __device__ __forceinline__ uint32_t place(E e) { return uint32_t(e); }
  static __device__ __forceinline__ E last() { return ~0ull; }
};
template <>
struct ElemOf<uint64_t, true> {
  using E = KeyPlace64;
  static __device__ __forceinline__ E make(uint64_t k, uint32_t i) { return E{k, i}; }
  static __device__ __forceinline__ uint64_t key(const E& e) { return e.k; }
  static __device__ __forceinline__ uint32_t place(const E& e) { return e.i; }
  static __device__ __forceinline__ E last() { return E{~0ull, ~0u}; }
};

// (key, place) of keys from one narrow range in a single word: the key's
// distance from the range's start above the place's PBITS bits.  The caller
// makes sure that it fits.  (Where a block takes 2^PBITS keys, the last place of
// the largest distance is the padding's word: either may be written for the other.)
template <typename K, int PBITS>
struct PackedElem {
  using E = K;
  K base;
  __device__ __forceinline__ E make(K k, uint32_t i) const { return ((k - base) << PBITS) | K(i); }
  __device__ __forceinline__ K key(E e) const { return base + (e >> PBITS); }
  __device__ __forceinline__ uint32_t place(E e) const { return uint32_t(e) & ((1u << PBITS) - 1u); }
  __device__ __forceinline__ E last() const { return ~K(0); }
};

__device__ __forceinline__ void order2(uint32_t& a, uint32_t& b) {
  const uint32_t lo = min(a, b);
  b = max(a, b);
  a = lo;
}
__device__ __forceinline__ void order2(uint64_t& a, uint64_t& b) {
  const bool sw = b < a;
  const uint64_t t = sw ? b : a;
  b = sw ? a : b;
  a = t;
}
__device__ __forceinline__ void order2(KeyPlace64& a, KeyPlace64& b) {
  const bool sw = b.k < a.k || (b.k == a.k && b.i < a.i);
  const uint64_t k = sw ? b.k : a.k;
  const uint32_t i = sw ? b.i : a.i;
  b.k = sw ? a.k : b.k;
  b.i = sw ? a.i : b.i;
  a.k = k;
  a.i = i;
}

// Eight elements in order: the 19-comparator network.
template <typename E>
__device__ __forceinline__ void order8(E (&v)[8]) {
  order2(v[0], v[2]); order2(v[1], v[3]); order2(v[4], v[6]); order2(v[5], v[7]);
  order2(v[0], v[4]); order2(v[1], v[5]); order2(v[2], v[6]); order2(v[3], v[7]);
  order2(v[0], v[1]); order2(v[2], v[3]); order2(v[4], v[5]); order2(v[6], v[7]);
  order2(v[2], v[4]); order2(v[3], v[5]);
  order2(v[1], v[4]); order2(v[3], v[6]);
  order2(v[1], v[2]); order2(v[3], v[4]); order2(v[5], v[6]);
}

// Elements [p, p + N) of shared memory (p a multiple of 4) as 16-byte pieces.
template <class L, typename E, int N>
__device__ __forceinline__ void ld_window(E (&v)[N], const E* s, uint32_t p) {
#pragma unroll
  for (int i = 0; i < N; i += L::PIECE) {
    const uint4 q = *reinterpret_cast<const uint4*>(s + L::slot(p + i));
    if constexpr (sizeof(E) == 4) {
      v[i] = q.x;
      v[i + 1] = q.y;
      v[i + 2] = q.z;
      v[i + 3] = q.w;
    } else if constexpr (sizeof(E) == 8) {
      v[i] = (uint64_t(q.y) << 32) | q.x;
      v[i + 1] = (uint64_t(q.w) << 32) | q.z;
    } else {
      v[i] = E{(uint64_t(q.y) << 32) | q.x, q.z};
    }
  }
}
template <class L, typename E, int N>
__device__ __forceinline__ void st_window(E* s, uint32_t p, const E (&v)[N]) {
#pragma unroll
  for (int i = 0; i < N; i += L::PIECE) {
    uint4 q;
    if constexpr (sizeof(E) == 4) q = make_uint4(v[i], v[i + 1], v[i + 2], v[i + 3]);
    else if constexpr (sizeof(E) == 8)
      q = make_uint4(uint32_t(v[i]), uint32_t(v[i] >> 32), uint32_t(v[i + 1]), uint32_t(v[i + 1] >> 32));
    else q = make_uint4(uint32_t(v[i].k), uint32_t(v[i].k >> 32), v[i].i, 0u);
    *reinterpret_cast<uint4*>(s + L::slot(p + i)) = q;
  }
}
__device__ __forceinline__ uint32_t shfl_down1(uint32_t v) { return __shfl_down_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ uint64_t shfl_down1(uint64_t v) { return __shfl_down_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ KeyPlace64 shfl_down1(const KeyPlace64& v) {
  return KeyPlace64{__shfl_down_sync(0xffffffffu, v.k, 1), __shfl_down_sync(0xffffffffu, v.i, 1)};
}

// Two runs of four in order, merged (nine comparators).
template <typename E>
__device__ __forceinline__ void merge8(E (&v)[8]) {
  order2(v[0], v[4]); order2(v[1], v[5]); order2(v[2], v[6]); order2(v[3], v[7]);
  order2(v[2], v[4]); order2(v[3], v[5]);
  order2(v[1], v[2]); order2(v[3], v[4]); order2(v[5], v[6]);
}

// How payloads follow their keys:
//   kAlone    there are none;
//   kFollow   each is read from the input, at its key's place there, when it leaves;
//   kStaged   copied to shared memory in input order meanwhile (sorts in place);
//   kInPlace  read like kFollow, but all of them before the first is written
//             (sorts in place, less shared memory, slower);
//   kPlaces   the input's second array holds places instead of payloads: equal
//             keys are ordered by them, and payloads are read from a third
//             array at the place.
enum class Vals { kAlone, kFollow, kStaged, kInPlace, kPlaces };

template <int THREADS, int ITEMS, int NBITS, typename K, int VB, Vals MODE, class Elem = ElemOf<K, VB != 0>>
struct LocalLayout {
  static_assert((VB != 0) == (MODE != Vals::kAlone), "payloads and what happens to them");
  using V = typename ValueOf<VB>::T;
  using E = typename Elem::E;
  static constexpr bool STAGED = MODE == Vals::kStaged;
  static constexpr int WARPS = THREADS / 32;
  static constexpr int CAP = THREADS * ITEMS;
  static constexpr int NB = 1 << NBITS;
  // the bins' counts (16 bits each), or the digit
  // passes' lane masks and counters
  static constexpr size_t BIN_BYTES = size_t(NB) * 2;
  static constexpr int SPARE = CAP + 16;  // element slots of lanes without a key
  // The windows' vector accesses start 8 elements apart, a stride that falls
  // on few banks: 16-byte pieces are permuted inside groups of eight.
  static constexpr int PIECE = 16 / int(sizeof(E));  // elements per piece
  static constexpr int SPREAD = int(sizeof(E)) / 4 == 1 ? 1 : int(sizeof(E)) / 4 == 2 ? 3 : 7;
  static __device__ __forceinline__ uint32_t slot(uint32_t p) {
    return p ^ (((p / (8 * PIECE)) & SPREAD) * PIECE);
  }
  static constexpr size_t MASK_BYTES = size_t(WARPS) * kMaskSlots * 4;
  static constexpr size_t RANK_BYTES = MASK_BYTES + size_t(WARPS) * 256 * 2;
  static constexpr size_t OFF_KEY = ((BIN_BYTES > RANK_BYTES ? BIN_BYTES : RANK_BYTES) + 15) / 16 * 16;
  static constexpr size_t OFF_VAL = OFF_KEY + size_t(SPARE + 128) * sizeof(E);  // windows reach past the end; slots are permuted in groups
  static constexpr size_t OFF_WARP = OFF_VAL + (STAGED ? size_t(CAP) * VB : 0);
  static constexpr size_t OFF_SCAN = OFF_WARP + 64 * 8;  // two words per warp at most
  static constexpr size_t OFF_MOST = OFF_SCAN + 4 * 32 * 4;
  static constexpr size_t SMEM = OFF_MOST + 16;
  static_assert(CAP < 65536 && NBITS <= 15, "16-bit places and bins");
  static_assert(RANK_BYTES % 16 == 0, "tables are cleared in 16-byte units");
};

// Warp-wide minimum and maximum of a 32- or 64-bit word.
template <typename K>
__device__ __forceinline__ void warp_min_max(K& lo, K& hi) {
  if constexpr (sizeof(K) == 4) {
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
  } else {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const K a = __shfl_xor_sync(0xffffffffu, lo, o), b = __shfl_xor_sync(0xffffffffu, hi, o);
      lo = a < lo ? a : lo;
      hi = b > hi ? b : hi;
    }
  }
}

// Bins from the array's own range: bin = (key - lo) >> sh.
// LOOK: whether its values may crowd (not where a sample has found them spread evenly).
template <typename K, bool LOOK = true>
struct RangeBins {
  static constexpr bool kKnown = false, kLook = LOOK;
  K lo;
  int sh;
  __device__ __forceinline__ uint32_t operator()(K k) const { return uint32_t((k - lo) >> sh); }
  // how far into its bin, in units of 2^-32
  __device__ __forceinline__ uint32_t frac(K k) const {
    constexpr int W = int(sizeof(K)) * 8;
    if (sh == 0) return 0u;
    const K r = (k - lo) << (W - sh);
    return uint32_t(r >> (W - 32));
  }
  __device__ __forceinline__ bool unique() const { return sh == 0; }  // a bin holds one value
};

// Stable rank of this warp's 32 keys of one item by an 8-bit digit: the place
// among the warp's keys of that digit so far (the table step of warp_rank).
__device__ __forceinline__ uint32_t warp_rank_step(uint32_t d, uint32_t* wm, uint16_t* wc, uint32_t lt, uint32_t gt,
                                                   int lane) {
  atomicOr(&wm[d], 1u << lane);
  __syncwarp();
  const uint32_t peers = wm[d];
  const uint32_t before = wc[d];
  __syncwarp();
  if ((peers & gt) == 0) {
    wc[d] = uint16_t(before + __popc(peers));
    wm[d] = 0u;
  }
  __syncwarp();
  return before + __popc(peers & lt);
}

// Block-wide exclusive prefix sums of R ranges of words that follow each other
// (range r's sums come after the whole of range r - 1), and the total, with
// one barrier: every warp scans the warps' sums for itself.  s (R * 32 words)
// must not be in use before it nor reused before the caller's next barrier.
template <int THREADS, int R>
__device__ __forceinline__ void block_exclusive_sums(const uint32_t (&x)[R], uint32_t (&out)[R], uint32_t* s,
                                                     uint32_t* total) {
  constexpr int WARPS = THREADS / 32;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    uint32_t inc = x[r];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += y;
    }
    if (lane == 31) s[r * 32 + w] = inc;
    out[r] = inc - x[r];
  }
  __syncthreads();
  uint32_t before = 0;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const uint32_t t = lane < WARPS ? s[r * 32 + lane] : 0u;
    out[r] += before + __reduce_add_sync(0xffffffffu, lane < w ? t : 0u);
    before += __reduce_add_sync(0xffffffffu, t);
  }
  *total = before;
}

// The digit passes over [0, m) of s_key (see above): afterwards s_key is in
// order.  Warp w ranks elements [w * 32 * ITEMS, ...), so that rank order is
// the order they were in; places past the end take no part.
// BY_PLACE: equal keys are ordered by their places too (they are not in that
// order to begin with).
template <class L, int THREADS, int ITEMS, typename K, class EO, bool BY_PLACE>
__device__ __noinline__ void local_digit_passes(uint32_t m, const EO eo, unsigned char* smem) {
  using E = typename EO::E;
  constexpr int WARPS = L::WARPS;
  E* s_key = reinterpret_cast<E*>(smem + L::OFF_KEY);
  K* s_red = reinterpret_cast<K*>(smem + L::OFF_WARP);
  uint32_t* s_warp = reinterpret_cast<uint32_t*>(smem + L::OFF_WARP);
  uint32_t* s_mask = reinterpret_cast<uint32_t*>(smem);
  uint16_t* s_cnt = reinterpret_cast<uint16_t*>(smem + L::MASK_BYTES);
  uint4* b4 = reinterpret_cast<uint4*>(smem);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t lt = lanemask_lt(), gt = lanemask_gt();
  const uint32_t wofs = uint32_t(warp) * 32 * ITEMS + lane;
  auto row = [&](int j) { return uint32_t(warp * 32 * ITEMS + j * 32) < m; };  // the warp's row has keys
  auto has = [&](int j) { return wofs + j * 32 < m; };
  E e[ITEMS];
  K diff = 0;
  uint32_t pdiff = 0;
  const K k0 = eo.key(s_key[L::slot(0)]);
  const uint32_t p0 = eo.place(s_key[L::slot(0)]);
#pragma unroll
  for (int j = 0; j < ITEMS; ++j) {
    if (has(j)) {
      e[j] = s_key[L::slot(wofs + j * 32)];
      diff |= eo.key(e[j]) ^ k0;
      pdiff |= eo.place(e[j]) ^ p0;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) diff |= __shfl_xor_sync(0xffffffffu, diff, o);
  if (lane == 0) s_red[warp] = diff;
  __syncthreads();
  diff = s_red[lane < WARPS ? lane : 0];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) diff |= __shfl_xor_sync(0xffffffffu, diff, o);
  if constexpr (BY_PLACE) {
    pdiff = __reduce_or_sync(0xffffffffu, pdiff);
    __syncthreads();
    if (lane == 0) s_warp[warp] = pdiff;
    __syncthreads();
    pdiff = __reduce_or_sync(0xffffffffu, s_warp[lane < WARPS ? lane : 0]);
  }
  // digits 0-3 are the places' (BY_PLACE), the others the keys'
  auto digit = [&](int j, uint32_t d) {
    const E& x = e[j];
    return d < 4 ? (eo.place(x) >> (8 * d)) & 0xffu : uint32_t(eo.key(x) >> (8 * (d - 4))) & 0xffu;
  };
  for (uint32_t d = BY_PLACE ? 0 : 4; d < 4 + sizeof(K); ++d) {
    if (((d < 4 ? pdiff >> (8 * d) : uint32_t(diff >> (8 * (d - 4)))) & 0xffu) == 0) continue;  // uniform
    __syncthreads();
    for (int i = tid; i < int(L::RANK_BYTES / 16); i += THREADS) b4[i] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    // Rows of 32 two at a time: one vote tells whether both hold one digit only
    // (as few distinct keys make many), whose lanes would all meet in one word.
    // Places past the end act as the largest digit: they come after every key.
    uint32_t rk[(ITEMS + 1) / 2];
    uint32_t* wm = s_mask + warp * kMaskSlots;
    uint16_t* wc = s_cnt + warp * 256;
    auto rank = [&](uint32_t x, bool uniform) -> uint32_t {
      if (!uniform) return warp_rank_step(x, wm, wc, lt, gt, lane);
      const uint32_t before = wc[x];
      __syncwarp();
      if (lane == 0) wc[x] = uint16_t(before + 32u);
      __syncwarp();
      return before + uint32_t(lane);
    };
#pragma unroll
    for (int j = 0; j < ITEMS; j += 2) {
      if (!row(j)) break;
      const uint32_t x0 = has(j) ? digit(j, d) : 255u;
      const uint32_t x1 = j + 1 < ITEMS && has(j + 1) ? digit(j + 1, d) : 255u;
      const uint32_t both = x0 | (x1 << 8);
      const bool uniform = __all_sync(0xffffffffu, both == __shfl_sync(0xffffffffu, both, 0));
      rk[j >> 1] = rank(x0, uniform);
      if (j + 1 < ITEMS) rk[j >> 1] |= rank(x1, uniform) << 16;
    }
    __syncthreads();
    constexpr int DT = THREADS < 256 ? THREADS : 256;  // threads with digits
    constexpr int DPT = 256 / DT;                      // consecutive digits of such a thread
    uint32_t sum = 0;
    if (tid < DT)
      for (int q = tid * DPT; q < (tid + 1) * DPT; ++q)
        for (int wi = 0; wi < WARPS; ++wi) sum += s_cnt[wi * 256 + q];
    uint32_t run = block_exclusive_sum<THREADS>(sum, s_warp);
    if (tid < DT)
      for (int q = tid * DPT; q < (tid + 1) * DPT; ++q)
        for (int wi = 0; wi < WARPS; ++wi) {
          const uint32_t v = s_cnt[wi * 256 + q];
          s_cnt[wi * 256 + q] = uint16_t(run);
          run += v;
        }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < ITEMS; ++j)
      if (has(j))
        s_key[L::slot(((rk[j >> 1] >> (16 * (j & 1))) & 0xffffu) + s_cnt[warp * 256 + digit(j, d)])] = e[j];
    __syncthreads();
#pragma unroll
    for (int j = 0; j < ITEMS; ++j)
      if (has(j)) e[j] = s_key[L::slot(wofs + j * 32)];
  }
  __syncthreads();
}

// The sort of [0, m) of (in, vin) into (out, vout), 1 <= m <= THREADS * ITEMS;
// vin holds payloads or (kPlaces) places, and then `from` the payloads.
// kStaged may sort in place.  COHERENT: the inputs were written by other
// blocks of the same launch, or are overwritten by this one.  ordi maps a key
// on loading, ordo back on storing.  bins: RangeBins (filled here) or a map
// known beforehand.  eo: what is ordered (by default the key, or key and
// place side by side).  The block is synchronised on return.
// LOOPED: for a call inside a loop.  There the registers of items that a short
// array leaves out would be carried round the loop, and what depends on the
// thread's index alone would be kept over it (288 bytes of spills for 4,096 keys):
// they start defined, and the index is read anew (20 bytes).  Other calls are up
// to 7 % slower with that.
template <int THREADS, int ITEMS, int NBITS, int VB, Vals MODE, bool COHERENT, bool LOOPED, class OrdI, class OrdO, class Bins,
          class VIn, class EO = ElemOf<typename OrdI::Key, VB != 0>>
__device__ __forceinline__ void local_sort_array(const typename OrdI::Key* in, typename OrdI::Key* out, const VIn* vin,
                                                 typename ValueOf<VB>::T* vout,
                                                 const typename ValueOf<VB>::T* from, const uint32_t m,
                                                 const OrdI ordi, const OrdO ordo, Bins bins, unsigned char* smem,
                                                 const EO eo = EO{}) {
  using K = typename OrdI::Key;
  constexpr bool STAGED = MODE == Vals::kStaged, PLACES = MODE == Vals::kPlaces;
  using L = LocalLayout<THREADS, ITEMS, NBITS, K, VB, MODE, EO>;
  using V = typename L::V;
  using E = typename EO::E;
  constexpr int WARPS = L::WARPS, NB = L::NB;
  uint32_t* s_bin = reinterpret_cast<uint32_t*>(smem);  // two 16-bit counts per word
  const uint16_t* s_start = reinterpret_cast<const uint16_t*>(smem);
  E* s_key = reinterpret_cast<E*>(smem + L::OFF_KEY);
  V* s_val = reinterpret_cast<V*>(smem + L::OFF_VAL);
  K* s_red = reinterpret_cast<K*>(smem + L::OFF_WARP);
  uint32_t* s_scan = reinterpret_cast<uint32_t*>(smem + L::OFF_SCAN);
  uint32_t* s_most = reinterpret_cast<uint32_t*>(smem + L::OFF_MOST);
  int tid = threadIdx.x;
  if constexpr (LOOPED) asm volatile("mov.u32 %0, %%tid.x;" : "=r"(tid));
  auto define = [](auto* a, int count) {
    if constexpr (LOOPED) {
#pragma unroll
      for (int i = 0; i < count; ++i) a[i] = {};
    }
  };
  const int lane = tid & 31, warp = tid >> 5;
  // Items go by groups of G: a group past the last key is skipped by the whole
  // block (a uniform branch); inside a group a lane without a key has its
  // shared atomic and its stores predicated off.
  constexpr int G = ITEMS % 4 == 0 ? 4 : 1;
  auto has = [&](int j) { return uint32_t(j * THREADS + tid) < m; };
  auto for_items = [&](auto&& f) {
#pragma unroll
    for (int g = 0; g < ITEMS; g += G)
      if (uint32_t(g * THREADS) < m) {
#pragma unroll
        for (int j = g; j < g + G; ++j) f(j);
      }
  };

  // How crowded the bins are is told by a sample, each lane's key from a stretch
  // of its own: D bins in use give a key its like among its warp's others with a
  // chance of about 31 / D, and m / D keys to a bin.  Counted are likes in the
  // second set of bins, with a bin's share taken from the warp's keys in it:
  // those that neither set tells apart.  Four warps look (a match takes 0.1 us of
  // them, 1 us of 32): before the bins are laid where there are keys enough,
  // otherwise when they are found crowded.
  constexpr int FEW = WARPS < 4 ? WARPS : 4;
  constexpr uint32_t LANES = uint32_t(FEW) * 32;
  const bool looked = Bins::kLook && m > kLookKeys;
  auto sampled = [&]() {
    const uint32_t q = uint32_t(tid);
    return q * m / LANES + __umulhi(q * 0x9E3779B1u, m / LANES);
  };
  auto count_likes = [&](K k, bool live) {
    if constexpr (Bins::kLook) {
      if (warp < FEW) {
        const uint32_t lives = __ballot_sync(0xffffffffu, live);
        const uint32_t b = bins(k);
        const uint32_t same = __match_any_sync(0xffffffffu, b) & lives;
        uint32_t likes = __ballot_sync(0xffffffffu, live && (same & (same - 1u)) != 0u);
        if (likes) {
          const uint32_t part = __umulhi(bins.frac(k), uint32_t(__popc(same)) * uint32_t(NB / 32));
          const uint32_t same2 = __match_any_sync(0xffffffffu, (b << NBITS) + part) & same;
          likes = __ballot_sync(0xffffffffu, live && (same2 & (same2 - 1u)) != 0u);
        }
        if (lane == 0) s_scan[warp] = uint32_t(__popc(likes));
      }
    }
  };
  uint32_t likes = 0;
  auto read_likes = [&]() { return __reduce_add_sync(0xffffffffu, lane < FEW ? s_scan[lane] : 0u); };
  // whether the likes mean more than `limit` keys to a bin
  auto more_than = [&](uint32_t limit) { return likes * m > 31u * limit * (m < LANES ? m : LANES); };

  // 1. load; clear the bins
  K key[ITEMS];
  define(key, ITEMS);
  for_items([&](int j) { key[j] = has(j) ? ld_elem<COHERENT>(in + j * THREADS + tid) : K(0); });
  K probe = 0;
  if (looked && warp < FEW) probe = ld_elem<COHERENT>(in + sampled());
  [[maybe_unused]] uint32_t place[PLACES ? ITEMS : 1];
  define(place, PLACES ? ITEMS : 1);
  if constexpr (PLACES) for_items([&](int j) { place[j] = has(j) ? ld_elem<COHERENT>(vin + j * THREADS + tid) : 0u; });
  auto elem = [&](int j) {
    if constexpr (PLACES) return eo.make(key[j], place[j]);
    else return eo.make(key[j], uint32_t(j * THREADS + tid));
  };
  uint4* b4 = reinterpret_cast<uint4*>(smem);
#pragma unroll
  for (int i = 0; i < NB / 8; i += THREADS)
    if (i + THREADS <= NB / 8 || i + tid < NB / 8) b4[i + tid] = make_uint4(0u, 0u, 0u, 0u);
  if (tid == 0) *s_most = 0u;
  if constexpr (STAGED) {
    // asynchronous copies: nothing waits for them before the payloads leave
    for_items([&](int j) {
      if (has(j))
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(static_cast<uint32_t>(
                         __cvta_generic_to_shared(s_val + j * THREADS + tid))),
                     "l"(vin + j * THREADS + tid), "n"(VB)
                     : "memory");
    });
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  if (!ordi.identity()) for_items([&](int j) { key[j] = ordi.map(key[j]); });
  if constexpr (!Bins::kKnown) {
    K lo = ~K(0), hi = 0;
    for_items([&](int j) {
      if (has(j)) {
        lo = key[j] < lo ? key[j] : lo;
        hi = key[j] > hi ? key[j] : hi;
      }
    });
    warp_min_max(lo, hi);
    if (lane == 0) {
      s_red[warp] = lo;
      s_red[WARPS + warp] = hi;
    }
    __syncthreads();
    lo = s_red[lane < WARPS ? lane : 0];
    hi = s_red[WARPS + (lane < WARPS ? lane : 0)];
    warp_min_max(lo, hi);
    const K range = hi - lo;  // m >= 1
    const int bits =
        range == 0 ? 0 : int(sizeof(K) * 8) - (sizeof(K) == 4 ? __clz(int(range)) : __clzll((long long)range));
    bins.lo = lo;
    bins.sh = bits > NBITS ? bits - NBITS : 0;
  }
  // Far too crowded for either set of bins: the digit passes sort them at once
  // (the bins' atomics would meet in few words).  Bins of one value, whose keys
  // need no order, hold 256.
  if (looked) count_likes(ordi.map(probe), true);
  __syncthreads();
  if (looked) likes = read_likes();
  const bool crowded = looked && more_than(VB == 0 && bins.unique() ? 256u : kCrowded);

  // 2. turns within the bins.  Word w of the counts holds bin w in its low and
  // bin w + NB / 2 in its high half; four 8-bit turns go to a register (a
  // turn above kLastLimit sends the block another way, so its high bits may be
  // lost).  Returns the fullest bin's keys, five at least.
  const uint32_t bin_base = static_cast<uint32_t>(__cvta_generic_to_shared(s_bin));
  uint32_t turn[(ITEMS + 3) / 4];
  define(turn, (ITEMS + 3) / 4);
  auto count = [&](auto&& bin_of) -> uint32_t {
    uint32_t most = 0;
    for_items([&](int j) {
      const uint32_t b = bin_of(j);
      const uint32_t half = (b >> (NBITS - 1)) & 1u;
      uint32_t r = 0;
      asm volatile(
          "{\n\t.reg .pred p;\n\tsetp.lt.u32 p, %3, %4;\n\t@p atom.shared.add.u32 %0, [%1], %2;\n\t}"
          : "+r"(r)
          : "r"(bin_base + 4u * (b & uint32_t(NB / 2 - 1))), "r"(half * 0xffffu + 1u), "r"(uint32_t(j * THREADS + tid)),
            "r"(m)
          : "memory");
      r = (r >> (half * 16u)) & 0xffffu;
      most = r > most ? r : most;
      if (j % 4 == 0) turn[j / 4] = r;
      else turn[j / 4] = __byte_perm(turn[j / 4], r, j % 4 == 1 ? 0x3240 : j % 4 == 2 ? 0x3410 : 0x4210);
    });
    if (__any_sync(0xffffffffu, most >= 5u)) {  // rare
      most = __reduce_max_sync(0xffffffffu, most);
      if (lane == 0) atomicMax(s_most, most);
    }
    __syncthreads();
    return *s_most ? *s_most + 1u : 5u;
  };
  // 3. counts -> starts, both halves of the words at once (sums of at most CAP
  // < 2^16 each): the low halves' total comes before the high halves' starts.
  // The words are scanned in ranges of 4 per scanning thread, one 16-byte
  // vector per thread and range (no bank conflicts).
  auto scan = [&]() {
    constexpr int WORDS = NB / 2;
    constexpr int POW2 = THREADS >= 1024 ? 1024 : THREADS >= 512 ? 512 : THREADS >= 256 ? 256 : 128;
    constexpr int ST = WORDS / 4 < POW2 ? WORDS / 4 : POW2;        // scanning threads
    constexpr int R = WORDS / (4 * ST);                            // ranges
    static_assert(R * 4 * ST == WORDS, "whole ranges");
    static_assert(R <= 4, "a word of s_scan per warp and range");
    uint4 w[R];
    uint32_t sum[R], run[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      w[r] = tid < ST ? b4[r * ST + tid] : make_uint4(0u, 0u, 0u, 0u);
      sum[r] = w[r].x + w[r].y + w[r].z + w[r].w;
    }
    uint32_t total;
    block_exclusive_sums<THREADS, R>(sum, run, s_scan, &total);
    const uint32_t high = total << 16;  // starts of the high halves follow the low ones
#pragma unroll
    for (int r = 0; r < R; ++r) {
      uint32_t at = run[r] + high;
      auto put = [&](uint32_t& c) {
        const uint32_t t = c;
        c = at;
        at += t;
      };
      put(w[r].x);
      put(w[r].y);
      put(w[r].z);
      put(w[r].w);
      if (tid < ST) b4[r * ST + tid] = w[r];
    }
    __syncthreads();
  };
  auto start_of = [&](uint32_t b) -> uint32_t {  // (the bin of a lane without a key is any number: masked)
    return s_start[2u * (b & uint32_t(NB / 2 - 1)) + ((b >> (NBITS - 1)) & 1u)];
  };
  // 4. keys into the bins' places (a lane without a key stores to a spare
  // slot); the windows past the end read the last element
  auto stage = [&](auto&& bin_of) {
    for_items([&](int j) {
      const uint32_t p = start_of(bin_of(j)) + __byte_perm(turn[j / 4], 0u, 0x4440u + uint32_t(j % 4));
      s_key[L::slot(has(j) ? p : uint32_t(L::SPARE + lane))] = elem(j);
    });
    if (tid < 16) s_key[L::slot(m + tid)] = eo.last();
    __syncthreads();
  };
  auto first_bin = [&](int j) { return bins(key[j]); };
  uint32_t most = 0;
  bool staged = false;
  if (!crowded) {
    most = count(first_bin);
    // bins of one value need no order among equal keys (as long as their turns fit their 8 bits)
    if (VB == 0 && bins.unique() && most <= 256u) most = 1u;
    staged = most <= (Bins::kKnown ? kLastLimit : kBinLimit);
    if (staged) {
      scan();
      stage(first_bin);
    } else if (!Bins::kKnown && !bins.unique()) {
      if constexpr (!Bins::kKnown) {
        if (Bins::kLook && !looked && m > 31u * kCrowded) {  // (fewer keys cannot tell)
          count_likes(key[0], has(0));  // the first lanes' own keys
          __syncthreads();
          likes = read_likes();
          __syncthreads();
        }
        if (!more_than(kCrowded)) {
          // the second set of bins (see above), NB / m of them to a key;
          // positions among the keys in 16.16 fixed point
          scan();
          const uint32_t per = (uint32_t(NB) << 16) / m;
          uint32_t bin2[ITEMS];
          define(bin2, ITEMS);
          for_items([&](int j) {
            const uint32_t b = first_bin(j) & uint32_t(NB - 1);
            const uint32_t s = start_of(b), e = b == uint32_t(NB - 1) ? m : start_of(b + 1);
            bin2[j] = __umulhi((s << 16) + __umulhi(bins.frac(key[j]), (e - s) << 16), per);
          });
          __syncthreads();
          for (int i = tid; i < NB / 8; i += THREADS) b4[i] = make_uint4(0u, 0u, 0u, 0u);
          if (tid == 0) *s_most = 0u;
          __syncthreads();
          auto second_bin = [&](int j) { return bin2[j]; };
          most = count(second_bin);
          staged = most <= kLastLimit;
          if (staged) {
            scan();
            stage(second_bin);
          }
        }
      }
    }
  }
  if (staged) {
    // 5. windows: those that start before the end
    constexpr int NWIN = (ITEMS + 7) / 8;  // windows per thread
    // (what the block's register budget holds; else a round at a time)
    constexpr bool HELD = NWIN * sizeof(E) <= (THREADS >= 384 ? 8 : THREADS >= 256 ? 12 : 24);
    if (HELD && most == 5u) {
      // Two rounds, each thread keeping its windows in registers: between
      // them it takes the next window's lower half, from the next lane or,
      // over the warp's end, through shared memory.
      E v[HELD ? NWIN : 1][8];
      define(v[0], (HELD ? NWIN : 1) * 8);
#pragma unroll
      for (int c = 0; c < (HELD ? NWIN : 0); ++c) {
        const uint32_t p = uint32_t(c * THREADS + tid) * 8u;
        if (uint32_t(c * THREADS + warp * 32) * 8u < m) {  // the whole warp
          ld_window<L>(v[c], s_key, p < m ? p : 0u);
          order8(v[c]);
          if (lane == 0) {
            E low[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) low[i] = v[c][i];
            st_window<L>(s_key, p, low);
          }
        }
      }
      __syncthreads();
#pragma unroll
      for (int c = 0; c < (HELD ? NWIN : 0); ++c) {
        const uint32_t p = uint32_t(c * THREADS + tid) * 8u;
        if (uint32_t(c * THREADS + warp * 32) * 8u < m) {
          E u[8];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            u[i] = v[c][i + 4];
            u[i + 4] = shfl_down1(v[c][i]);
          }
          if (lane == 31) {
            E next[4];
            ld_window<L>(next, s_key, p + 8u < m ? p + 8u : 0u);
#pragma unroll
            for (int i = 0; i < 4; ++i) u[i + 4] = next[i];
          }
          if (p + 8u >= m) {  // no next window
#pragma unroll
            for (int i = 4; i < 8; ++i) u[i] = eo.last();
          }
          merge8(u);
          __syncwarp();
          if (p < m) st_window<L>(s_key, p + 4u, u);  // (the first window's lower half is in place)
        }
      }
      __syncthreads();
    } else {
      const int rounds = most <= 1u ? 0 : most <= 5u ? 2 : int(most + 6u) / 4;
      for (int r = 0; r < rounds; ++r) {
        for (uint32_t i = tid * 8u + (r & 1) * 4u; i < m; i += THREADS * 8u) {
          E v[8];
          ld_window<L>(v, s_key, i);
          if (r == 0) order8(v);
          else merge8(v);
          st_window<L>(s_key, i, v);
        }
        __syncthreads();
      }
    }
  } else {
    for_items([&](int j) {
      if (has(j)) s_key[L::slot(j * THREADS + tid)] = elem(j);
    });
    __syncthreads();
    local_digit_passes<L, THREADS, ITEMS, K, EO, PLACES>(m, eo, smem);
  }
  // 6. out
  if constexpr (STAGED) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
  }
  V held[MODE == Vals::kInPlace ? ITEMS : 1];
  define(held, MODE == Vals::kInPlace ? ITEMS : 1);
  if constexpr (MODE == Vals::kInPlace) {
    for_items([&](int j) {
      if (has(j)) held[j] = ld_elem<COHERENT>(vin + eo.place(s_key[L::slot(j * THREADS + tid)]));
    });
    __syncthreads();
  }
  auto write_out = [&](auto invert) {
    for_items([&](int j) {
      if (has(j)) {
        const uint32_t p = j * THREADS + tid;
        const E e = s_key[L::slot(p)];
        if constexpr (decltype(invert)::value) ordo.store(out + p, eo.key(e));
        else out[p] = eo.key(e);
        if constexpr (STAGED) vout[p] = s_val[eo.place(e)];
        else if constexpr (MODE == Vals::kInPlace) vout[p] = held[j];
        else if constexpr (PLACES) vout[p] = ld_elem(from + eo.place(e));
        else if constexpr (VB != 0) vout[p] = vin[eo.place(e)];
      }
    });
  };
  if (ordo.identity()) write_out(std::false_type{});
  else write_out(std::true_type{});
  __syncthreads();
}

}  // namespace rs
