// gradient.cuh — loading four consecutive gradient values (fp32, or bf16 bit
// patterns widened exactly: the 16 stored bits become the high half of the
// fp32 word).
#pragma once

#include "common.cuh"

namespace efs {

template <typename GT>
struct GradVec;

template <>
struct GradVec<float> {
  float4 v;
  __device__ __forceinline__ void load(const float* p) { v = ld_stream_f4(p); }
  __device__ __forceinline__ void load_readonly(const float* p) {
    v = __ldg(reinterpret_cast<const float4*>(p));
  }
  __device__ __forceinline__ void load_scalars(const float* p) {
    v = make_float4(__ldg(p), __ldg(p + 1), __ldg(p + 2), __ldg(p + 3));
  }
  // shared memory: p aligned, or the 4 values `sub` (1..3) past an aligned p
  __device__ __forceinline__ void load_aligned(const float* p) {
    v = *reinterpret_cast<const float4*>(p);
  }
  __device__ __forceinline__ void load_at(const float* p, uint32_t sub) {
    const float4 a = reinterpret_cast<const float4*>(p)[0];
    const float4 b = reinterpret_cast<const float4*>(p)[1];
    v = sub == 1 ? make_float4(a.y, a.z, a.w, b.x)
        : sub == 2 ? make_float4(a.z, a.w, b.x, b.y) : make_float4(a.w, b.x, b.y, b.z);
  }
  __device__ __forceinline__ float operator[](int j) const {
    return j == 0 ? v.x : j == 1 ? v.y : j == 2 ? v.z : v.w;
  }
};

template <>
struct GradVec<uint16_t> {
  uint2 v;
  __device__ __forceinline__ void load(const uint16_t* p) { v = ld_stream_u2(p); }
  __device__ __forceinline__ void load_readonly(const uint16_t* p) {
    v = __ldg(reinterpret_cast<const uint2*>(p));
  }
  __device__ __forceinline__ void load_scalars(const uint16_t* p) {
    v = make_uint2(__ldg(p) | (static_cast<uint32_t>(__ldg(p + 1)) << 16),
                   __ldg(p + 2) | (static_cast<uint32_t>(__ldg(p + 3)) << 16));
  }
  // shared memory: p 8-byte aligned, or the 4 values `sub` (1..7) past such a p
  __device__ __forceinline__ void load_aligned(const uint16_t* p) {
    v = *reinterpret_cast<const uint2*>(p);
  }
  __device__ __forceinline__ void load_at(const uint16_t* p, uint32_t sub) {
    const uint2 a = reinterpret_cast<const uint2*>(p)[sub >> 2];
    const uint2 b = reinterpret_cast<const uint2*>(p)[(sub >> 2) + 1];
    const uint32_t sh = (sub & 1u) * 16u;
    const uint32_t w0 = (sub & 2u) ? a.y : a.x, w1 = (sub & 2u) ? b.x : a.y,
                   w2 = (sub & 2u) ? b.y : b.x;
    v = make_uint2(__funnelshift_r(w0, w1, sh), __funnelshift_r(w1, w2, sh));
  }
  __device__ __forceinline__ float operator[](int j) const {
    const uint32_t w = (j < 2) ? v.x : v.y;
    return bf16_bits_to_f32((j & 1) ? (w >> 16) : (w & 0xffffu));
  }
};

__device__ __forceinline__ float grad_scalar(const float* g, uint64_t i) { return g[i]; }
__device__ __forceinline__ float grad_scalar(const uint16_t* g, uint64_t i) {
  return bf16_bits_to_f32(g[i]);
}

}  // namespace efs
