// device.cuh -- small device helpers shared by the kernels of libdfacto.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace dfacto {

constexpr unsigned kFull = 0xffffffffu;

// Load VEC consecutive factor entries (16-, 8- or 4-byte aligned vector loads)
// and widen to float.  T is float or __nv_bfloat16.
template <typename T, int VEC>
struct VecIO;

template <>
struct VecIO<float, 1> {
  __device__ __forceinline__ static void load(const float* p, float (&v)[1]) { v[0] = __ldg(p); }
  __device__ __forceinline__ static void store(float* p, const float (&v)[1]) { p[0] = v[0]; }
};
template <>
struct VecIO<float, 2> {
  __device__ __forceinline__ static void load(const float* p, float (&v)[2]) {
    float2 t = __ldg(reinterpret_cast<const float2*>(p));
    v[0] = t.x; v[1] = t.y;
  }
  __device__ __forceinline__ static void store(float* p, const float (&v)[2]) {
    *reinterpret_cast<float2*>(p) = make_float2(v[0], v[1]);
  }
};
template <>
struct VecIO<float, 4> {
  __device__ __forceinline__ static void load(const float* p, float (&v)[4]) {
    float4 t = __ldg(reinterpret_cast<const float4*>(p));
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
  }
  __device__ __forceinline__ static void store(float* p, const float (&v)[4]) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  }
};
template <>
struct VecIO<float, 8> {
  __device__ __forceinline__ static void load(const float* p, float (&v)[8]) {
    float4 a = __ldg(reinterpret_cast<const float4*>(p));
    float4 b = __ldg(reinterpret_cast<const float4*>(p) + 1);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
  }
  __device__ __forceinline__ static void store(float* p, const float (&v)[8]) {
    reinterpret_cast<float4*>(p)[0] = make_float4(v[0], v[1], v[2], v[3]);
    reinterpret_cast<float4*>(p)[1] = make_float4(v[4], v[5], v[6], v[7]);
  }
};

__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }

template <>
struct VecIO<__nv_bfloat16, 1> {
  __device__ __forceinline__ static void load(const __nv_bfloat16* p, float (&v)[1]) {
    v[0] = __bfloat162float(p[0]);
  }
};
template <>
struct VecIO<__nv_bfloat16, 2> {
  __device__ __forceinline__ static void load(const __nv_bfloat16* p, float (&v)[2]) {
    uint32_t w = __ldg(reinterpret_cast<const unsigned int*>(p));
    v[0] = bf16_lo(w); v[1] = bf16_hi(w);
  }
};
template <>
struct VecIO<__nv_bfloat16, 4> {
  __device__ __forceinline__ static void load(const __nv_bfloat16* p, float (&v)[4]) {
    uint2 w = __ldg(reinterpret_cast<const uint2*>(p));
    v[0] = bf16_lo(w.x); v[1] = bf16_hi(w.x); v[2] = bf16_lo(w.y); v[3] = bf16_hi(w.y);
  }
};
template <>
struct VecIO<__nv_bfloat16, 8> {
  __device__ __forceinline__ static void load(const __nv_bfloat16* p, float (&v)[8]) {
    uint4 w = __ldg(reinterpret_cast<const uint4*>(p));
    v[0] = bf16_lo(w.x); v[1] = bf16_hi(w.x); v[2] = bf16_lo(w.y); v[3] = bf16_hi(w.y);
    v[4] = bf16_lo(w.z); v[5] = bf16_hi(w.z); v[6] = bf16_lo(w.w); v[7] = bf16_hi(w.w);
  }
};

// Scalar load/store of one factor entry in storage type T.
__device__ __forceinline__ float ld_elem(const float* p) { return *p; }
__device__ __forceinline__ float ld_elem(const __nv_bfloat16* p) { return __bfloat162float(*p); }
__device__ __forceinline__ void st_elem(float* p, float v) { *p = v; }
__device__ __forceinline__ void st_elem(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }
// Value actually held after a store in type T (the rounding of st_elem).
__device__ __forceinline__ float rt_elem(const float*, float v) { return v; }
__device__ __forceinline__ float rt_elem(const __nv_bfloat16*, float v) {
  return __bfloat162float(__float2bfloat16_rn(v));
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}

// e / d for 0 <= e < 8192 and 1 <= d <= 32 as a multiplication by
// small_inv(d) = ceil(2^18 / d) and a shift: exact, as e (d - 1) < 2^18.
__host__ __device__ __forceinline__ uint32_t small_inv(int d) { return ((1u << 18) + (uint32_t)d - 1u) / (uint32_t)d; }
__device__ __forceinline__ int small_div(int e, uint32_t inv) { return (int)(((uint32_t)e * inv) >> 18); }

}  // namespace dfacto
