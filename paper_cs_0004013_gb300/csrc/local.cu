// Arrays and segments that fit one block, sorted in shared memory (local.cuh).
//
// Paper: the local sort of each cell's keys (Sec. 3.3).
#include <algorithm>

#include "local.cuh"
#include "rs_internal.h"

namespace rs {
namespace {

template <typename K>
struct OrdFor;
template <>
struct OrdFor<uint32_t> {
  using T = Ord32;
  static __device__ __forceinline__ T in(const LocalArgs& a) { return Ord32{a.xin}; }
  static __device__ __forceinline__ T out(const LocalArgs& a) { return Ord32{a.xout}; }
};
template <>
struct OrdFor<uint64_t> {
  using T = Ord64;
  static __device__ __forceinline__ T in(const LocalArgs& a) { return Ord64{a.x64}; }
  static __device__ __forceinline__ T out(const LocalArgs& a) { return Ord64{a.x64}; }
};

// A block per listed segment (list != null; the grid holds a block for every
// segment that may be listed), or the one array [0, single_n).  LOOP: a grid of
// any size, whose blocks take segments in turn; for lists that are short beside
// what may be listed, as an empty block takes about 0.3 us of its place on the SM
// (MSD plan's 16,384 buckets of clustered keys: 140 us -> 130), while full lists
// lose by it (16,384 segments of 4,096 keys: 291 us against 310).
// One array is one block's chain of steps, bound by its latency: bins and sorting
// networks instead of four digit passes, traced (about 4 us of it the events),
// us: 1,000 keys 15.7 -> 7.5, 4,000 16.4 -> 8.0, 8,000 27.2 -> 11.1, 16,000 35.5 ->
// 14.7, with payloads 44.8 -> 24.8; 8,000 64-bit keys, which eight launches of
// passes sorted, 123 -> 15, with 64-bit payloads 141 -> 23.  Values that
// crowd end in the digit passes after a look at a sample (in graphs, us, before any
// bins / bins tried first / now): 8,000 keys of 8 values 18.1 / 25.7 / 20.1, 16,000
// 20.8 / 32.2 / 25, of 1,000 values, which windows still order, 34 / 48 / 18, clusters 25.5
// / 40 / 21, log-uniform ones 32.3 / 48 / 35; 4,000 keys, which are not looked at, of
// 8 values 10.3 / 12.8 / 12.5.
template <int THREADS, int ITEMS, int NBITS, int MINB, typename K, int VB, bool LOOP>
__global__ void __launch_bounds__(THREADS, MINB) local_sort_kernel(const LocalArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  using V = typename ValueOf<VB>::T;
  auto sort = [&](uint64_t start, uint32_t m) {
    local_sort_array<THREADS, ITEMS, NBITS, VB, VB ? Vals::kFollow : Vals::kAlone, false, LOOP>(
        static_cast<const K*>(a.kin) + start, static_cast<K*>(a.kout) + start,
        VB ? static_cast<const V*>(a.vin) + start : nullptr, VB ? static_cast<V*>(a.vout) + start : nullptr,
        static_cast<const V*>(nullptr), m, OrdFor<K>::in(a), OrdFor<K>::out(a), RangeBins<K>{}, smem);
  };
  if constexpr (LOOP) {
    const uint32_t count = *a.count;
    for (uint32_t k = blockIdx.x; k < count; k += gridDim.x) {
      const uint32_t s = a.list[k];
      const uint64_t start = a.seg_off[s];
      sort(start, uint32_t(a.seg_off[s + 1] - start));
    }
  } else {
    uint64_t start = 0;
    uint32_t m = a.single_n;
    if (a.list) {
      if (blockIdx.x >= *a.count) return;
      const uint32_t s = a.list[blockIdx.x];
      start = a.seg_off[s];
      m = uint32_t(a.seg_off[s + 1] - start);
    }
    sort(start, m);
  }
}

struct Shape {
  uint32_t cap;
  unsigned threads;
  size_t smem;
  const void* func;
  cudaError_t (*launch)(const LocalArgs&, unsigned, cudaStream_t);
};
template <int THREADS, int ITEMS, int NBITS, int MINB, typename K, int VB, bool LOOP = false>
Shape shape() {
  using L = LocalLayout<THREADS, ITEMS, NBITS, K, VB, VB ? Vals::kFollow : Vals::kAlone>;
  return Shape{uint32_t(L::CAP), unsigned(THREADS), L::SMEM,
               reinterpret_cast<const void*>(&local_sort_kernel<THREADS, ITEMS, NBITS, MINB, K, VB, LOOP>),
               [](const LocalArgs& a, unsigned grid, cudaStream_t s) {
                 local_sort_kernel<THREADS, ITEMS, NBITS, MINB, K, VB, LOOP><<<grid, THREADS, L::SMEM, s>>>(a);
                 return cudaGetLastError();
               }};
}

// Segments: tiny ones (up to 4,096 keys) by 256 threads, small ones (up to
// 16,384) by 1,024.  One array: the smallest of its shapes that holds it.
struct Shapes {
  Shape tiny[2], few_tiny[2], small[2];                     // [payload]
  Shape one32[2], mid32[2], one32v8, big32v8, one64[3], big64[3];  // one array; [0, 4 or 8 payload bytes]
};
const Shapes& shapes() {
  using u32 = uint32_t;
  using u64 = uint64_t;
  static const Shapes s = {
      {shape<256, 16, 12, 4, u32, 0>(), shape<256, 16, 12, 3, u32, 4>()},
      {shape<256, 16, 12, 4, u32, 0, true>(), shape<256, 16, 12, 3, u32, 4, true>()},
      {shape<1024, 16, 14, 1, u32, 0>(), shape<1024, 16, 14, 1, u32, 4>()},
      {shape<256, 4, 11, 1, u32, 0>(), shape<256, 4, 11, 1, u32, 4>()},
      {shape<1024, 4, 13, 1, u32, 0>(), shape<1024, 4, 13, 1, u32, 4>()},
      shape<256, 4, 11, 1, u32, 8>(),
      shape<1024, 8, 13, 1, u32, 8>(),
      {shape<256, 4, 11, 1, u64, 0>(), shape<256, 4, 11, 1, u64, 4>(), shape<256, 4, 11, 1, u64, 8>()},
      {shape<1024, 8, 13, 1, u64, 0>(), shape<1024, 8, 13, 1, u64, 4>(), shape<1024, 8, 13, 1, u64, 8>()},
  };
  return s;
}

}  // namespace

cudaError_t prepare_local() {
  const Shapes& s = shapes();
  const Shape* all[] = {&s.tiny[0],  &s.tiny[1],  &s.few_tiny[0], &s.few_tiny[1], &s.small[0], &s.small[1], &s.one32[0], &s.one32[1],
                        &s.mid32[0], &s.mid32[1], &s.one32v8,  &s.big32v8,  &s.one64[0], &s.one64[1],
                        &s.one64[2], &s.big64[0], &s.big64[1], &s.big64[2]};
  for (const Shape* p : all)
    if (cudaError_t e = cudaFuncSetAttribute(p->func, cudaFuncAttributeMaxDynamicSharedMemorySize, int(p->smem));
        e != cudaSuccess)
      return e;
  return cudaSuccess;
}

uint32_t local_max_keys(int key_bytes, int val_bytes) { return key_bytes == 4 && val_bytes < 8 ? 16384u : 8192u; }

cudaError_t launch_tiny_segments(const LocalArgs& a, bool pairs, uint32_t num_segs, unsigned few_sms, cudaStream_t s) {
  const Shapes& sh = shapes();
  const uint32_t few = few_sms * 16u;  // four times what is resident
  return few_sms && num_segs > few ? sh.few_tiny[pairs].launch(a, few, s) : sh.tiny[pairs].launch(a, num_segs, s);
}
cudaError_t launch_small_segments(const LocalArgs& a, bool pairs, uint32_t max_listed, cudaStream_t s) {
  return shapes().small[pairs].launch(a, max_listed, s);
}

cudaError_t launch_local_array(const LocalArgs& a, int key_bytes, int val_bytes, cudaStream_t s) {
  const Shapes& sh = shapes();
  const Shape* p;
  if (key_bytes == 8) {
    const int v = val_bytes / 4;
    p = a.single_n <= sh.one64[v].cap ? &sh.one64[v] : &sh.big64[v];
  } else if (val_bytes == 8) {
    p = a.single_n <= sh.one32v8.cap ? &sh.one32v8 : &sh.big32v8;
  } else {
    const int v = val_bytes / 4;
    p = a.single_n <= sh.one32[v].cap ? &sh.one32[v] : a.single_n <= sh.mid32[v].cap ? &sh.mid32[v] : &sh.small[v];
  }
  if (a.single_n > p->cap) return cudaErrorInvalidValue;
  return p->launch(a, 1u, s);
}

}  // namespace rs
