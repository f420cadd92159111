// Rows of activations in 16-byte pieces, shared by the norm kernels (as_norm.cu) and the y pass that ends in a norm (as_scan.cu).
#pragma once

#include "as_internal.cuh"

namespace as {
namespace {

__device__ __forceinline__ float wsum(float v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

template <typename IO> struct Vec { static constexpr int N = 16 / sizeof(IO); };   // elements of a 16-byte piece
template <typename IO> __device__ __forceinline__ void ld_vec(const IO* p, float (&v)[Vec<IO>::N]);
template <> __device__ __forceinline__ void ld_vec<float>(const float* p, float (&v)[4]) {
  const float4 t = *reinterpret_cast<const float4*>(p);
  v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
template <> __device__ __forceinline__ void ld_vec<__nv_bfloat16>(const __nv_bfloat16* p, float (&v)[8]) {
  const uint4 t = *reinterpret_cast<const uint4*>(p);
  const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&t);
#pragma unroll
  for (int i = 0; i < 4; ++i) { const float2 f = __bfloat1622float2(h[i]); v[2 * i] = f.x; v[2 * i + 1] = f.y; }
}
template <typename IO> __device__ __forceinline__ void st_vec(IO* p, const float (&v)[Vec<IO>::N]);
template <> __device__ __forceinline__ void st_vec<float>(float* p, const float (&v)[4]) {
  *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
template <> __device__ __forceinline__ void st_vec<__nv_bfloat16>(__nv_bfloat16* p, const float (&v)[8]) {
  uint4 t;
  __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&t);
#pragma unroll
  for (int i = 0; i < 4; ++i) h[i] = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
  *reinterpret_cast<uint4*>(p) = t;
}

}  // namespace
}  // namespace as
