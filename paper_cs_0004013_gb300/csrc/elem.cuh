// Keys and payloads of 32 and 64 bits as the kernels that take both see them.
#pragma once

#include "rs_device.cuh"

namespace rs {

// A key word and its order-preserving unsigned map, 32 or 64 bits wide.
struct Ord32 {
  using Key = uint32_t;
  KeyXform x;
  __device__ __forceinline__ bool identity() const { return is_identity(x); }
  __device__ __forceinline__ Key map(Key k) const { return to_ordered(k, x); }
  __device__ __forceinline__ void store(uint32_t* p, Key k) const { *p = from_ordered(k, x); }
};
struct Ord64 {
  using Key = uint64_t;
  KeyXform64 x;
  __device__ __forceinline__ bool identity() const { return (x.flo | x.fhi | x.shi) == 0u; }
  __device__ __forceinline__ Key map(Key k) const {
    const uint2 m = map64(make_uint2(uint32_t(k), uint32_t(k >> 32)), x);
    return (uint64_t(m.y) << 32) | m.x;
  }
  __device__ __forceinline__ void store(uint64_t* p, Key k) const {
    *reinterpret_cast<uint2*>(p) = unmap64(make_uint2(uint32_t(k), uint32_t(k >> 32)), x);
  }
};

// The payload word of VB bytes (0: none).
template <int VB>
struct ValueOf { using T = uint32_t; };
template <>
struct ValueOf<8> { using T = uint2; };

// One element of a key or payload array.  COHERENT: the array is also written
// by the kernel (a sort in place), so the read-only path is not taken.
template <bool COHERENT = false>
__device__ __forceinline__ uint32_t ld_elem(const uint32_t* p) {
  return COHERENT ? __ldcg(p) : ld_stream(p);
}
template <bool COHERENT = false>
__device__ __forceinline__ uint2 ld_elem(const uint2* p) {
  return COHERENT ? __ldcg(p) : ld_stream2(p);
}
template <bool COHERENT = false>
__device__ __forceinline__ uint64_t ld_elem(const uint64_t* p) {
  const uint2 m = ld_elem<COHERENT>(reinterpret_cast<const uint2*>(p));
  return (uint64_t(m.y) << 32) | m.x;
}

}  // namespace rs
