// One stable distribution of keys with payloads by a digit of up to 8 bits that
// a function of the key gives (value buckets, hybrid.cu): 32- or 64-bit keys,
// 32- or 64-bit payloads, each moved as one word.
//
// Paper: the bucketing/distribution of Sec. 3.2, stable as the order inside a
// bucket has to survive it (Sec. 5).  The tile's steps are those of
// onesweep.cuh (lane-mask ranking, aggregate status, chained scan inside the
// tile's segment, staging, write-out in tile order); what differs is where the
// digits come from, that they are kept four to a register between the steps,
// and that a 64-bit word is moved whole instead of as two planes.
#pragma once

#include "elem.cuh"
#include "local.cuh"

namespace rs {

template <typename K, int VB, int THREADS, int ITEMS>
struct StableSplitLayout {
  using V = typename ValueOf<VB>::T;
  static constexpr int WARPS = THREADS / 32;
  static constexpr int TILE = THREADS * ITEMS;
  static constexpr size_t MASK_BYTES = size_t(WARPS) * kMaskSlots * 4;
  static constexpr size_t RANK_BYTES = MASK_BYTES + size_t(WARPS) * 256 * 2;
  static constexpr size_t OFF_VAL = size_t(TILE) * sizeof(K);
  static constexpr size_t BUF_BYTES = OFF_VAL + size_t(TILE) * VB;
  static constexpr size_t UNION_BYTES = ((RANK_BYTES > BUF_BYTES ? RANK_BYTES : BUF_BYTES) + 15) / 16 * 16;
  static constexpr size_t OFF_GOFF = UNION_BYTES;
  static constexpr size_t OFF_WARP = OFF_GOFF + 256 * 4;
  static constexpr size_t OFF_JOB = OFF_WARP + 32 * 4;
  static constexpr size_t SMEM = OFF_JOB + 16;
  static_assert(THREADS >= 256 && TILE < 65536, "a thread per digit, 16-bit places");
};

// The tile in / vin [0, valid) (FULL: valid is the tile's size) to base(digit)
// + (the digit's keys in the segment's earlier tiles) + (its place here).
// tile: its row of status words; first: the segment's first row.  The rank
// tables must be clear and the block synchronised on entry.
template <typename K, int VB, int THREADS, int ITEMS, bool FULL, class Digit, class Base, class OrdI>
__device__ __forceinline__ void stable_split_tile(const K* in, const typename ValueOf<VB>::T* vin, uint32_t valid, K* out,
                                                  typename ValueOf<VB>::T* vout, uint32_t n, uint32_t* status,
                                                  uint32_t tile, uint32_t first, const Digit& digit, const Base& base,
                                                  const OrdI& ordi, uint32_t* err, unsigned char* smem) {
  using L = StableSplitLayout<K, VB, THREADS, ITEMS>;
  using V = typename L::V;
  constexpr int WARPS = L::WARPS;
  uint32_t* s_mask = reinterpret_cast<uint32_t*>(smem);
  uint16_t* s_cnt = reinterpret_cast<uint16_t*>(smem + L::MASK_BYTES);
  K* s_key = reinterpret_cast<K*>(smem);
  V* s_val = reinterpret_cast<V*>(smem + L::OFF_VAL);
  uint32_t* s_goff = reinterpret_cast<uint32_t*>(smem + L::OFF_GOFF);
  uint32_t* s_warp = reinterpret_cast<uint32_t*>(smem + L::OFF_WARP);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t wofs = uint32_t(warp) * 32 * ITEMS + lane;
  auto has = [&](int j) { return FULL || wofs + j * 32 < valid; };

  // the payloads are read after the ranking: into L2 meanwhile
  if (FULL && (reinterpret_cast<uintptr_t>(vin) & 15u) == 0) prefetch_l2_tile(vin, uint32_t(L::TILE) * VB);

  // 1. load: warp w's items are consecutive; places past the end act as the
  // largest digit, come after every key and are never written
  K key[ITEMS];
  uint32_t dg[(ITEMS + 3) / 4];
#pragma unroll
  for (int j = 0; j < ITEMS; ++j) key[j] = has(j) ? ld_elem(in + wofs + j * 32) : K(0);
  if (!ordi.identity()) {
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) key[j] = ordi.map(key[j]);
  }
#pragma unroll
  for (int j = 0; j < ITEMS; ++j) {
    const uint32_t d = has(j) ? digit(key[j]) : 255u;
    if (j % 4 == 0) dg[j / 4] = d;
    else dg[j / 4] |= d << (8 * (j % 4));
  }
  auto digit_at = [&](int j) { return __byte_perm(dg[j / 4], 0u, 0x4440u + uint32_t(j % 4)); };

  // 2. rank within the warp
  uint32_t rk[(ITEMS + 1) / 2];
  {
    const uint32_t lt = lanemask_lt(), gt = lanemask_gt();
    uint32_t* wm = s_mask + warp * kMaskSlots;
    uint16_t* wc = s_cnt + warp * 256;
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
      const uint32_t r = warp_rank_step(digit_at(j), wm, wc, lt, gt, lane);
      if (j & 1) rk[j >> 1] |= r << 16;
      else rk[j >> 1] = r;
    }
  }
  __syncthreads();

  // 3. per digit: aggregate status; counts -> exclusive (digit, warp) prefixes
  uint32_t tot = 0;
  if (tid < 256) {
#pragma unroll 4
    for (int w = 0; w < WARPS; ++w) tot += s_cnt[w * 256 + tid];
    st_relaxed(status + size_t(tile) * 256 + tid, status_word<uint32_t>(1u, tile == first, tot));
  }
  const uint32_t excl = block_exclusive_sum<THREADS>(tot, s_warp);
  if (tid < 256) {
    uint32_t run = excl;
#pragma unroll 4
    for (int w = 0; w < WARPS; ++w) {
      const uint32_t c = s_cnt[w * 256 + tid];
      s_cnt[w * 256 + tid] = uint16_t(run);
      run += c;
    }
  }
  __syncthreads();

  // 4. tile positions, then the keys and payloads staged in digit order
#pragma unroll
  for (int j = 0; j < ITEMS; ++j) {
    const uint32_t pos = s_cnt[warp * 256 + digit_at(j)];
    rk[j >> 1] += (j & 1) ? pos << 16 : pos;
  }
  __syncthreads();  // the rank tables are dead; the staging buffer reuses them
  auto pos_of = [&](int j) { return (rk[j >> 1] >> (16 * (j & 1))) & 0xffffu; };
#pragma unroll
  for (int j = 0; j < ITEMS; ++j) s_key[pos_of(j)] = key[j];
  {
    constexpr int H = VB == 8 ? (ITEMS + 1) / 2 : ITEMS;  // 64-bit payloads: half a row at a time
#pragma unroll
    for (int h = 0; h < ITEMS; h += H) {
      V val[H];
#pragma unroll
      for (int j = 0; j < H; ++j)
        if (h + j < ITEMS && has(h + j)) val[j] = ld_elem(vin + wofs + (h + j) * 32);
#pragma unroll
      for (int j = 0; j < H; ++j)
        if (h + j < ITEMS && has(h + j)) s_val[pos_of(h + j)] = val[j];
    }
  }

  // 5. chained scan over the segment's earlier tiles
  if (tid < 256) {
    uint32_t prefix[1];
    lookback<256, 1, uint32_t, 8>(status, tile, first, tid, 1u, err, prefix);
    if (tile != first) st_relaxed(status + size_t(tile) * 256 + tid, status_word<uint32_t>(1u, true, prefix[0] + tot));
    s_goff[tid] = base(uint32_t(tid)) + prefix[0] - excl;
  }
  __syncthreads();

  // 6. out, in tile order; the range check only guards against a corrupted offset
  bool oob = false;
#pragma unroll
  for (int k = 0; k < ITEMS; ++k) {
    const uint32_t i = k * THREADS + tid;
    if (FULL || i < valid) {
      const K kk = s_key[i];
      const uint32_t g = s_goff[digit(kk)] + i;
      if (g < n) {
        out[g] = kk;
        vout[g] = s_val[i];
      } else {
        oob = true;
      }
    }
  }
  if (oob) atomicOr(err, kErrBounds);
}

}  // namespace rs
