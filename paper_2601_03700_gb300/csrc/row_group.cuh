// A row held in registers by a group of threads: TPR threads (a warp, or the whole CTA of 256), V float4 per thread.
#pragma once
#include "common.cuh"

namespace adept {

constexpr int RW_THREADS = 256;

template <int TPR, int NV>
__device__ __forceinline__ void group_sum(float (&v)[NV], float* red) {
#pragma unroll
  for (int i = 0; i < NV; ++i) v[i] = warp_sum(v[i]);
  if (TPR == 32) return;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  __syncthreads();   // red may still be read by the previous sum
  if (lane == 0) {
#pragma unroll
    for (int i = 0; i < NV; ++i) red[w * NV + i] = v[i];
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    float t = 0.f;
#pragma unroll
    for (int k = 0; k < RW_THREADS / 32; ++k) t += red[k * NV + i];
    v[i] = t;
  }
}

// Four elements of a row; `vec`: the row's address allows one 16-byte load.
__device__ __forceinline__ float4 row4(const float* x, int v, bool vec) {
  if (vec) return reinterpret_cast<const float4*>(x)[v];
  return make_float4(x[4 * v], x[4 * v + 1], x[4 * v + 2], x[4 * v + 3]);
}
__device__ __forceinline__ void put4(float* o, int v, float4 a) { reinterpret_cast<float4*>(o)[v] = a; }
__device__ __forceinline__ void put4(bf16* o, int v, float4 a) {
  const __nv_bfloat162 lo = __floats2bfloat162_rn(a.x, a.y), hi = __floats2bfloat162_rn(a.z, a.w);
  uint2 u;
  u.x = *reinterpret_cast<const uint32_t*>(&lo);
  u.y = *reinterpret_cast<const uint32_t*>(&hi);
  reinterpret_cast<uint2*>(o)[v] = u;
}
__device__ __forceinline__ float sum4(float4 a) { return (a.x + a.y) + (a.z + a.w); }
__device__ __forceinline__ float dot4(float4 a, float4 b) { return (a.x * b.x + a.y * b.y) + (a.z * b.z + a.w * b.w); }
__device__ __forceinline__ float4 centre4(float4 a, float mu) {
  return make_float4(a.x - mu, a.y - mu, a.z - mu, a.w - mu);
}
__device__ __forceinline__ float4 scale4(float4 a, float s) { return make_float4(a.x * s, a.y * s, a.z * s, a.w * s); }

}  // namespace adept
