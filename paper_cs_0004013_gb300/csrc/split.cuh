// One distribution of keys without payloads by an 8-bit digit, where the
// order of keys with equal digits is free.
//
// Paper: the bucketing/distribution of Sec. 3.2 (count per bucket, cumulative
// totals, the partial sort grouping keys by bucket, distribution of contiguous
// bucket ranges).  Equal digits may leave in any order when every later
// step orders them anyway: the first pass of a low-to-high radix sort, and
// every split of a high-to-low one.  Then a key's place among its tile's keys
// of a digit is one shared atomic, and the tile's place among its bucket's
// keys one global atomic per digit on the bucket's cursor, issued right
// after the tile's counts and needed only when the tile is written: no
// chained scan over the tiles, no tickets, no waiting.  The cursors advance
// in the order in which tiles arrive, so every bucket's range fills roughly in
// address order while it is written.
//
// Per tile: 1. load and count (a shared reduction per key), 2. per digit the
// claim and the scan, 3. a place per key (a shared atomic) and the staging,
// 4. write-out in tile order.  Bound by the shared-memory pipe (13 wavefronts
// per 32 keys, 71 % busy) and the barriers between the steps.
#pragma once

#include "elem.cuh"
#include "onesweep2.cuh"

namespace rs {

// Tile shape: GB300, 2^26 keys by 8 bits: 256 x 32 at four blocks per SM 138 us,
// 384 x 16 at four 143, 512 x 16 at three 146, 384 x 24 at three 144.
constexpr int kSplitThreads = 256, kSplitItems = 32, kSplitBlocks = 4;

template <typename K, int THREADS, int ITEMS>
struct SplitLayout {
  static constexpr int TILE = THREADS * ITEMS;
  static constexpr int ROW = 257;  // the two half-warps count in two rows whose equal digits differ in bank
  static constexpr size_t OFF_CNT = size_t(TILE) * sizeof(K);
  static constexpr size_t OFF_GOFF = OFF_CNT + (2 * ROW + 2) * 4;
  static constexpr size_t OFF_SCAN = OFF_GOFF + 256 * 4;
  static constexpr size_t OFF_JOB = OFF_SCAN + 32 * 4;
  static constexpr size_t SMEM = OFF_JOB + 16;
  static_assert(THREADS >= 256, "a thread per digit");
};

// The tile's keys in[0, valid) (FULL: valid is the tile's size), mapped by
// ordi, to out[cursor of their digit ...) (mapped back by ordo).  bases: added
// to the cursors (null: the cursors start at the digits' bases).
template <typename K, int THREADS, int ITEMS, bool FULL, class Digit, class OrdI, class OrdO>
__device__ __forceinline__ void split_tile(const K* in, uint32_t valid, K* out, uint32_t* cursors, uint32_t n,
                                           const Digit& digit, const OrdI& ordi, const OrdO& ordo, uint32_t* err,
                                           unsigned char* smem, const uint32_t* bases = nullptr) {
  using L = SplitLayout<K, THREADS, ITEMS>;
  constexpr int ROW = L::ROW;
  K* s_key = reinterpret_cast<K*>(smem);
  uint32_t* s_cnt = reinterpret_cast<uint32_t*>(smem + L::OFF_CNT);
  uint32_t* s_goff = reinterpret_cast<uint32_t*>(smem + L::OFF_GOFF);
  uint32_t* s_scan = reinterpret_cast<uint32_t*>(smem + L::OFF_SCAN);
  const int tid = threadIdx.x, lane = tid & 31;
  auto has = [&](int j) { return FULL || uint32_t(j * THREADS + tid) < valid; };

  // 1. load, digits (four to a word), counts
  const uint32_t row = smem_addr(s_cnt + (lane >> 4) * ROW);
  K key[ITEMS];
  uint32_t dg[(ITEMS + 3) / 4];  // digits, four to a word
#pragma unroll
  for (int j = 0; j < ITEMS; ++j) key[j] = has(j) ? ld_elem(in + j * THREADS + tid) : K(0);
  for (int i = tid; i < 2 * ROW; i += THREADS) s_cnt[i] = 0u;
  __syncthreads();
  if (!ordi.identity()) {
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) key[j] = ordi.map(key[j]);
  }
#pragma unroll
  for (int j = 0; j < ITEMS; ++j) {
    const uint32_t d = digit(key[j]);
    if (j % 4 == 0) dg[j / 4] = d;
    else dg[j / 4] |= d << (8 * (j % 4));
    if (has(j)) sh_red_add(row + 4u * d, 1u);
  }
  __syncthreads();

  // 2. per digit: the tile's range of the bucket; where each half's keys start
  uint32_t claim = 0, excl = 0;
  if (tid < 256) {
    const uint32_t c0 = s_cnt[tid], tot = c0 + s_cnt[ROW + tid];
    if (tot) claim = atomicAdd(&cursors[tid], tot) + (bases ? bases[tid] : 0u);
    excl = scan256_exclusive(tot, s_scan);
    s_cnt[tid] = excl;
    s_cnt[ROW + tid] = excl + c0;
  }
  __syncthreads();

  // 3. each key's place in the tile
  const uint32_t sk = smem_addr(s_key);
#pragma unroll
  for (int j = 0; j < ITEMS; ++j) {
    if (has(j)) {
      uint32_t p;
      asm volatile("atom.shared.add.u32 %0, [%1], 1;"
                   : "=r"(p)
                   : "r"(row + 4u * byte_digit(dg[j / 4], 0x4440u + uint32_t(j % 4)))
                   : "memory");
      if constexpr (sizeof(K) == 4) sh_st(sk + 4u * p, key[j]);
      else asm volatile("st.shared.u64 [%0], %1;" ::"r"(sk + 8u * p), "l"(key[j]) : "memory");
    }
  }
  if (tid < 256) s_goff[tid] = claim - excl;
  __syncthreads();

  // 4. out, in tile order (a digit's keys go to consecutive places), a batch
  // of shared-memory reads before its stores.  The range check only guards
  // against a corrupted offset (it raises an error bit instead of writing out
  // of bounds).
  uint32_t worst = 0;
  constexpr int W = ITEMS % 4 == 0 ? 4 : ITEMS % 3 == 0 ? 3 : 1;
  auto write_out = [&](auto invert) {
#pragma unroll
    for (int k0 = 0; k0 < ITEMS; k0 += W) {
      K kk[W];
      uint32_t g[W];
#pragma unroll
      for (int b = 0; b < W; ++b) kk[b] = has(k0 + b) ? s_key[(k0 + b) * THREADS + tid] : K(0);
#pragma unroll
      for (int b = 0; b < W; ++b) g[b] = s_goff[digit(kk[b])] + (k0 + b) * THREADS + tid;
#pragma unroll
      for (int b = 0; b < W; ++b)
        if (has(k0 + b)) {
          worst = g[b] > worst ? g[b] : worst;
          if (g[b] < n) {
            if constexpr (decltype(invert)::value) ordo.store(out + g[b], kk[b]);
            else if constexpr (sizeof(K) == 4) st_global(out + g[b], kk[b]);
            else asm volatile("st.global.u64 [%0], %1;" ::"l"(out + g[b]), "l"(kk[b]) : "memory");
          }
        }
    }
  };
  if (ordo.identity()) write_out(std::false_type{});
  else write_out(std::true_type{});
  if (worst >= n) atomicOr(err, kErrBounds);
}

}  // namespace rs
