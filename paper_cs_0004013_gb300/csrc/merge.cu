// Stable merge of two sorted runs.
//
// Paper: the cleanup phase repaired the bucketed distribution by a
// merge-exchange between neighbouring cells, at whose heart two sorted lists
// are merged and each cell keeps its half (Sec. 3.4.2; later done in place,
// Sec. 4.6).  On the GPU a merge of two
// sorted runs A and B splits the output into tiles of TILE elements; the
// tile boundaries are placed on the merge path (for output position d, the
// number of elements of A among the first d outputs), found by a binary
// search per boundary; each block then loads its slices of A and B into
// shared memory (bulk copies), every thread finds its own start on the path
// inside the tile, reads the elements of its ITEMS outputs and orders them by a
// bitonic merging network in registers, and the tile leaves through shared
// memory as one bulk copy.  Equal keys keep A's before B's (stable: with
// payloads the network orders (key, place in the slices), and equal keys alone
// are the same word), keys of every kind compare through the order map of
// KeyXform.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "rs_device.cuh"
#include "rs_internal.h"

namespace rs {

namespace {

// ITEMS is odd: a thread's ITEMS consecutive outputs start ITEMS words after
// its neighbour's, so a warp's staging stores fall on 32 different banks.
constexpr int kMergeThreads = 256;
// tile shapes 1..4; key+payload tiles of 23 items take
// 48,232 bytes of static shared memory, of the 49,152 a block can declare
constexpr int kMergeItemsChoice[] = {15, 11, 23, 19};
constexpr int kMergeWaits = 1 << 20;  // bounded wait for a tile's slices

// Elements of A among the first d outputs of the stable merge of a[0, na)
// and b[0, nb): the smallest i with A[i] coming after B[d - i - 1], where A
// comes first on equal keys.  `at(x, k)` reads element k of run x mapped.
template <class F>
__device__ __forceinline__ uint32_t path_split(F at, uint32_t na, uint32_t nb, uint32_t d) {
  uint32_t lo = d > nb ? d - nb : 0u, hi = d < na ? d : na;
  while (lo < hi) {
    const uint32_t mid = (lo + hi) >> 1;
    if (at(0, mid) <= at(1, d - mid - 1)) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

// G lanes per tile boundary: the same search as path_split, but each round
// probes G points of the remaining range at once (a ballot finds where "A
// first" turns false), so a boundary costs about log_(G+1) of the range rounds
// of dependent loads instead of log_2, of 2 G sectors each.  Few boundaries wait
// for the rounds, many for the sectors (a warp each for two runs of 2^24: 89 MB
// read, 18 us): see launch_merge.
template <bool XF, int G>
__global__ void __launch_bounds__(256) merge_split_kernel(const MergeArgs m) {
  const uint32_t k = (blockIdx.x * blockDim.x + threadIdx.x) / G, lane = threadIdx.x & 31, sub = lane % G;
  const uint32_t total = m.na + m.nb;
  const uint32_t tiles = (total + m.tile - 1) / m.tile;
  const uint64_t d64 = uint64_t(k) * m.tile;
  const uint32_t d = d64 < total ? uint32_t(d64) : total;
  // true when A[i] comes before B[d - i - 1], i.e. the answer is above i
  auto a_first = [&](uint32_t i) {
    if constexpr (XF) return to_ordered(m.a[i], m.x) <= to_ordered(m.b[d - i - 1], m.x);
    else return m.a[i] <= m.b[d - i - 1];
  };
  // how many of this boundary's probes are true (they come first: sorted runs)
  auto trues = [&](bool t) {
    const uint32_t b = __ballot_sync(0xffffffffu, t);
    return uint32_t(__popc(G == 32 ? b : (b >> (lane - sub)) & ((1u << (G & 31)) - 1u)));
  };
  uint32_t lo = d > m.nb ? d - m.nb : 0u, hi = d < m.na ? d : m.na;  // answer in [lo, hi]
  while (__any_sync(0xffffffffu, hi - lo > G)) {  // (a warp's boundaries go round together)
    const bool open = hi - lo > G;
    const uint64_t len = hi - lo;
    const uint32_t i = lo + uint32_t(len * (sub + 1) / (G + 1));  // in [lo, hi)
    const uint32_t f = trues(open && a_first(i));
    if (open) {
      const uint32_t i_prev = lo + uint32_t(len * f / (G + 1));     // probe f - 1 (f >= 1)
      const uint32_t i_f = lo + uint32_t(len * (f + 1) / (G + 1));  // probe f (f < G)
      const uint32_t nlo = f == 0 ? lo : i_prev + 1;
      const uint32_t nhi = f == G ? hi : i_f;
      lo = nlo;
      hi = nhi > nlo ? nhi : nlo;
    }
  }
  const uint32_t f = trues(lo + sub < hi && a_first(lo + sub));
  if (sub == 0 && k <= tiles) m.split[k] = lo + f;
}

// A tile's copies between global and shared memory run in whole 16-byte units
// (bulk copies by one thread); the up to three words before and after them are
// moved by threads of their own.  A slice keeps its offset inside a 16-byte unit.
struct Slice {
  uint32_t off, head, vec, tail;  // words: start in the unit, before, (in 16 bytes) inside, and after the units
};
__device__ __forceinline__ Slice slice_of(const uint32_t* g, uint32_t len) {
  Slice c;
  c.off = uint32_t(reinterpret_cast<uintptr_t>(g) >> 2) & 3u;
  c.head = (4u - c.off) & 3u;
  c.head = c.head < len ? c.head : len;
  c.vec = (len - c.head) >> 2;
  c.tail = (len - c.head) & 3u;
  return c;
}
// The words outside the units: threads first .. first + 7.
template <class F>
__device__ __forceinline__ void slice_ends(const Slice& c, uint32_t len, uint32_t first, F&& move) {
  const uint32_t k = threadIdx.x - first;
  if (k < c.head) move(k);
  if (k >= 4u && k - 4u < c.tail) move(len - c.tail + k - 4u);
}
__device__ __forceinline__ void bulk_load(uint32_t* s, const uint32_t* g, const Slice& c, uint32_t bar) {
  if (c.vec)
    asm volatile("cp.async.bulk.shared::cta.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_addr(s + c.off + c.head)),
                 "l"(g + c.head), "r"(c.vec * 16u), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void bulk_store(uint32_t* g, const uint32_t* s, const Slice& c) {
  if (c.vec)
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(g + c.head),
                 "r"(smem_addr(s + c.off + c.head)), "r"(c.vec * 16u)
                 : "memory");
}

__device__ __forceinline__ void order(uint32_t& a, uint32_t& b) {
  const uint32_t t = a < b ? a : b;
  b = a < b ? b : a;
  a = t;
}
__device__ __forceinline__ void order(unsigned long long& a, unsigned long long& b) {
  const unsigned long long t = a < b ? a : b;
  b = a < b ? b : a;
  a = t;
}
// v[OFF, OFF + N), falling and then rising, to rising order.  Halves of a power
// of two apart are compared (Batcher's bitonic merge, with the last places of
// the next larger power of two taken as larger than everything).
template <int OFF, int N, class E, int SIZE>
__device__ __forceinline__ void bitonic_merge(E (&v)[SIZE]) {
  if constexpr (N > 1) {
    constexpr int M = N > 16 ? 16 : N > 8 ? 8 : N > 4 ? 4 : N > 2 ? 2 : 1;
    static_assert(N <= 32, "a thread's outputs");
#pragma unroll
    for (int i = 0; i < N - M; ++i) order(v[OFF + i], v[OFF + i + M]);
    bitonic_merge<OFF, M>(v);
    bitonic_merge<OFF + M, N - M>(v);
  }
}

// Bound by shared memory (0.32 wavefronts per output, 73 % of the time busy) and
// by the time a tile takes from its boundaries to its first element.  Against a
// serial merge per thread (a compare, a select and a dependent read per output),
// two runs of 2^24 keys: 65.3 us -> 49.8, 56 % of the issue slots busy instead of
// 75 %.  Six blocks per SM against five: two runs of 2^26 keys 261 us -> 253.
template <bool PAIRS, bool XF, int kMergeItems>
__global__ void __launch_bounds__(kMergeThreads, PAIRS ? 4 : 6) merge_tile_kernel(const MergeArgs m) {
  constexpr int kMergeTile = kMergeThreads * kMergeItems;
  constexpr int kWords = kMergeTile + 12;  // two slices, each from its offset in a 16-byte unit
  __shared__ __align__(16) uint32_t s_key[kWords];
  __shared__ __align__(16) uint32_t s_val[PAIRS ? kWords : 4];
  __shared__ uint32_t s_path[kMergeThreads];
  __shared__ __align__(8) unsigned long long s_bar;
  const uint32_t total = m.na + m.nb;
  const uint32_t t = blockIdx.x, tid = threadIdx.x;
  const uint32_t d0 = t * kMergeTile;
  const uint32_t cnt = total - d0 < uint32_t(kMergeTile) ? total - d0 : uint32_t(kMergeTile);
  const uint32_t bar = smem_addr(&s_bar);
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  wait_for_chain();
  const uint32_t i0 = m.split[t], i1 = m.split[t + 1];
  // On sorted runs the path is monotone: i0 <= i1 and i1 - i0 <= cnt.
  // Runs that are not sorted can break that; the tile is then not written
  // and the error word is raised instead of reading past the slices.
  if (i1 < i0 || i1 - i0 > cnt) {
    if (tid == 0) atomicOr(m.err, kErrBounds);
    return;
  }
  const uint32_t la = i1 - i0, lb = cnt - la, j0 = d0 - i0;
  const uint32_t *ga = m.a + i0, *gb = m.b + j0;
  const Slice ca = slice_of(ga, la), cb = slice_of(gb, lb);
  uint32_t* const sa = s_key;                                        // A's element i at sa[ca.off + i]
  uint32_t* const sb = s_key + ((ca.off + la + 3u) & ~3u);           // B's element j at sb[cb.off + j]
  Slice cva{}, cvb{};
  const uint32_t *gva = nullptr, *gvb = nullptr;
  uint32_t *sva = nullptr, *svb = nullptr;
  if constexpr (PAIRS) {
    gva = m.va + i0;
    gvb = m.vb + j0;
    cva = slice_of(gva, la);
    cvb = slice_of(gvb, lb);
    sva = s_val;
    svb = s_val + ((cva.off + la + 3u) & ~3u);
  }
  if (tid == 0) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar),
                 "r"((ca.vec + cb.vec + cva.vec + cvb.vec) * 16u)
                 : "memory");
    bulk_load(sa, ga, ca, bar);
    bulk_load(sb, gb, cb, bar);
    if constexpr (PAIRS) {
      bulk_load(sva, gva, cva, bar);
      bulk_load(svb, gvb, cvb, bar);
    }
  }
  slice_ends(ca, la, 32, [&](uint32_t e) { sa[ca.off + e] = ga[e]; });
  slice_ends(cb, lb, 64, [&](uint32_t e) { sb[cb.off + e] = gb[e]; });
  if constexpr (PAIRS) {
    slice_ends(cva, la, 96, [&](uint32_t e) { sva[cva.off + e] = gva[e]; });
    slice_ends(cvb, lb, 128, [&](uint32_t e) { svb[cvb.off + e] = gvb[e]; });
  }
  __syncthreads();  // the ends, and the barrier's start
  auto arrived = [&]() {
    uint32_t done = 0;
    for (int i = 0; i < kMergeWaits && !done; ++i)
      asm volatile(
          "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n\tselp.u32 %0, 1, 0, p;\n\t}"
          : "=r"(done)
          : "r"(bar)
          : "memory");
    return done;
  };
  if (__syncthreads_or(!arrived())) {
    if (tid == 0) {
      atomicOr(m.err, kErrTimeout);
      arrived();  // the copies in flight write this block's shared memory: it is held as long again
    }
    return;
  }
  // this thread's ITEMS outputs start on the path at diagonal tid * ITEMS
  auto mapped = [&](uint32_t k) { return XF ? to_ordered(k, m.x) : k; };
  const uint32_t* const pa = sa + ca.off;
  const uint32_t* const pb = sb + cb.off;
  auto at = [&](int x, uint32_t i) { return mapped(x == 0 ? pa[i] : pb[i]); };
  const uint32_t dt = tid * kMergeItems < cnt ? tid * kMergeItems : cnt;
  const uint32_t mine = cnt - dt < uint32_t(kMergeItems) ? cnt - dt : uint32_t(kMergeItems);
  const uint32_t ia = path_split(at, la, lb, dt), ib = dt - ia;
  s_path[tid] = ia;
  __syncthreads();
  // ... and end where the next thread's start (runs that are not sorted: in bounds all the same)
  const uint32_t end = tid + 1 < uint32_t(kMergeThreads) ? s_path[tid + 1] : la;
  const uint32_t ta = end < ia ? 0u : end - ia < mine ? end - ia : mine, tb = mine - ta;
  // B's part falling, A's part rising, places past the end as the largest key
  const uint32_t* const qa = pa + ia - tb;
  const uint32_t* const qb = pb + ib + tb - 1;
  using E = std::conditional_t<PAIRS, unsigned long long, uint32_t>;
  E v[kMergeItems];
  const uint32_t wa = ia - tb, wb = la + ib + tb - 1;  // places in the slices, A's before B's
#pragma unroll
  for (int q = 0; q < kMergeItems; ++q) {
    uint32_t k = 0xffffffffu;
    if (uint32_t(q) < mine) k = mapped(uint32_t(q) < tb ? qb[-q] : qa[q]);
    if constexpr (PAIRS) {
      const uint32_t w = uint32_t(q) >= mine ? 0xffffffffu : uint32_t(q) < tb ? wb - q : wa + q;
      v[q] = (static_cast<unsigned long long>(k) << 32) | w;
    } else {
      v[q] = k;
    }
  }
  bitonic_merge<0, kMergeItems>(v);
  uint32_t val[PAIRS ? kMergeItems : 1];
  if constexpr (PAIRS) {
    const uint32_t* const xa = sva + cva.off;
    const uint32_t* const xb = svb + cvb.off - la;
#pragma unroll
    for (int q = 0; q < kMergeItems; ++q) {
      const uint32_t w = uint32_t(v[q]);
      if (uint32_t(q) < mine) val[q] = w < la ? xa[w] : xb[w];
    }
  }
  __syncthreads();  // the slices are consumed; the tile is staged in their place
  uint32_t* const go = m.out + d0;
  const Slice co = slice_of(go, cnt);
#pragma unroll
  for (int q = 0; q < kMergeItems; ++q) {
    const uint32_t k = PAIRS ? uint32_t(v[q] >> (PAIRS ? 32 : 0)) : uint32_t(v[q]);
    if (uint32_t(q) < mine) s_key[co.off + dt + q] = XF ? from_ordered(k, m.x) : k;
  }
  uint32_t* gvo = nullptr;
  Slice cvo{};
  if constexpr (PAIRS) {
    gvo = m.vout + d0;
    cvo = slice_of(gvo, cnt);
#pragma unroll
    for (int q = 0; q < kMergeItems; ++q)
      if (uint32_t(q) < mine) s_val[cvo.off + dt + q] = val[q];
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncthreads();
  if (tid == 0) {
    bulk_store(go, s_key, co);
    if constexpr (PAIRS) bulk_store(gvo, s_val, cvo);
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
  }
  slice_ends(co, cnt, 32, [&](uint32_t e) { go[e] = s_key[co.off + e]; });
  if constexpr (PAIRS) slice_ends(cvo, cnt, 64, [&](uint32_t e) { gvo[e] = s_val[cvo.off + e]; });
  if (tid == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}

template <int ITEMS>
cudaError_t launch_tiles(const MergeArgs& m, unsigned tiles, cudaStream_t s) {
  const bool xf = !is_identity(m.x);
  if (m.vout) {
    if (xf) return launch_chained(&merge_tile_kernel<true, true, ITEMS>, tiles, kMergeThreads, 0, s, true, m);
    return launch_chained(&merge_tile_kernel<true, false, ITEMS>, tiles, kMergeThreads, 0, s, true, m);
  } else {
    if (xf) return launch_chained(&merge_tile_kernel<false, true, ITEMS>, tiles, kMergeThreads, 0, s, true, m);
    return launch_chained(&merge_tile_kernel<false, false, ITEMS>, tiles, kMergeThreads, 0, s, true, m);
  }
}

}  // namespace

// Outputs per tile of merge tile shape `shape` (1-based), or 0 if there is
// no such shape.  Shape 0 picks by the number of outputs: while tiles are few a
// merge lasts as long as one of them, and short networks are faster; many tiles
// pay for their boundaries.  Items per thread 11 / 15 / 23, us: keys 1,007 3.1 / 3.5
// / 3.7, 305,000 5.1 / 5.3 / 5.9, 2.1M 7.5 / 7.5 / 8.0, 5M 12.0 / 11.4 / 11.2, 21.8M 43.1
// / 41.8 / 38.7; with payloads 20 3.7 / 4.6 / 5.1, 305,000 6.0 / 6.7 / 8.0, 1M 8.0 / 8.0 /
// 9.8, 5M 21.6 / 19.7 / 20.5, 21.8M 83 / 71.5 / 72.3 (two runs of 2^26: 261 with 23
// against 281 with 19; with payloads 443 against 466).
constexpr uint64_t kMergeSmall = uint64_t(1) << 20;
constexpr uint64_t merge_mid(bool pairs) { return uint64_t(1) << (pairs ? 24 : 22); }
uint32_t merge_tile_keys(uint32_t shape, uint64_t n, bool pairs) {
  const uint32_t idx = shape != 0 ? shape - 1 : n <= kMergeSmall ? 1u : n <= merge_mid(pairs) ? 0u : 2u;
  if (idx >= sizeof(kMergeItemsChoice) / sizeof(kMergeItemsChoice[0])) return 0;
  return uint32_t(kMergeThreads * kMergeItemsChoice[idx]);
}

// Tile boundaries to have space for: those of any merge of at most n outputs
// with that shape (a workspace for more outputs takes fewer).
size_t merge_max_tiles(uint32_t shape, uint64_t n, bool pairs) {
  size_t most = 0;
  for (uint64_t m : {std::min(n, kMergeSmall), std::min(n, merge_mid(pairs)), n}) {
    const uint32_t tile = merge_tile_keys(shape, m, pairs);
    most = std::max(most, size_t((m + tile - 1) / tile));
  }
  return most;
}

cudaError_t launch_merge(const MergeArgs& m, cudaStream_t s) {
  const uint32_t total = m.na + m.nb;
  const uint32_t tiles = (total + m.tile - 1) / m.tile;
  const bool xf = !is_identity(m.x);
  auto split = [&](auto g) {
    constexpr int G = decltype(g)::value;
    const unsigned grid = unsigned((size_t(tiles) + 1) * G + 255) / 256;
    if (xf) merge_split_kernel<true, G><<<grid, 256, 0, s>>>(m);
    else merge_split_kernel<false, G><<<grid, 256, 0, s>>>(m);
    return cudaGetLastError();
  };
  // Both kernels, keys alone, 32 / 8 / 4 lanes a boundary: 8.4M outputs (1,425
  // tiles) 25.2 / 27.3 / 29.3 us, 21M (3,567) 47.8 / 44.7 / 45.7, 134M (22,796)
  // 257 / 222 / 212; with payloads 39.6 / 41.6 / 42.7, 80.5 / 76.4 / 76.4, 445 / 412 / 401.
  const cudaError_t e = tiles <= 2048   ? split(std::integral_constant<int, 32>{})
                        : tiles <= 8192 ? split(std::integral_constant<int, 8>{})
                                        : split(std::integral_constant<int, 4>{});
  if (e != cudaSuccess || tiles == 0) return e;
  switch (m.tile / kMergeThreads) {
    case 15: return launch_tiles<15>(m, tiles, s);
    case 11: return launch_tiles<11>(m, tiles, s);
    case 23: return launch_tiles<23>(m, tiles, s);
    case 19: return launch_tiles<19>(m, tiles, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace rs
