// Device helpers shared by the NormPre kernels (sm_103a).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace normpre {

__device__ __forceinline__ void raise_flag(int* flags, int bit) {
  if (flags) atomicOr(flags, bit);
}

// Programmatic dependent launch: a kernel launched by launch_pdl may start while
// the kernel before it on the stream is still running.  Every such kernel calls
// pdl_wait() in all threads before it touches global memory (it returns once
// the kernel before has completed and its writes are visible), and may call
// pdl_trigger() from when its successor may be brought onto the GPU.  Data
// written by the kernel before is not read through ld.global.nc, which the
// compiler may move above the wait.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

typedef __nv_bfloat16 bf16;

__device__ __forceinline__ float to_f32(float v) { return v; }
__device__ __forceinline__ float to_f32(bf16 v) { return __bfloat162float(v); }

template <typename T> __device__ __forceinline__ T from_f32(float v);
template <> __device__ __forceinline__ float from_f32<float>(float v) { return v; }
template <> __device__ __forceinline__ bf16 from_f32<bf16>(float v) { return __float2bfloat16_rn(v); }

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}
__device__ __forceinline__ float bf16lo(uint32_t v) { return __uint_as_float(v << 16); }
__device__ __forceinline__ float bf16hi(uint32_t v) { return __uint_as_float(v & 0xFFFF0000u); }

// 8 consecutive elements <-> 8 floats, with 16-byte vector accesses.
// The address must be 16-byte aligned (8 x bf16 = 16 B, 8 x f32 = 2 x 16 B).
__device__ __forceinline__ void load8(const float* p, float* v) {
  float4 a = __ldg(reinterpret_cast<const float4*>(p));
  float4 b = __ldg(reinterpret_cast<const float4*>(p) + 1);
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}
__device__ __forceinline__ void load8(const bf16* p, float* v) {
  uint4 a = __ldg(reinterpret_cast<const uint4*>(p));
  v[0] = bf16lo(a.x); v[1] = bf16hi(a.x); v[2] = bf16lo(a.y); v[3] = bf16hi(a.y);
  v[4] = bf16lo(a.z); v[5] = bf16hi(a.z); v[6] = bf16lo(a.w); v[7] = bf16hi(a.w);
}
// Non-cached-in-L1 variant for data written earlier by this kernel or stream.
__device__ __forceinline__ void load8_cg(const float* p, float* v) {
  float4 a = __ldcg(reinterpret_cast<const float4*>(p));
  float4 b = __ldcg(reinterpret_cast<const float4*>(p) + 1);
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}
__device__ __forceinline__ void load8_cg(const bf16* p, float* v) {
  uint4 a = __ldcg(reinterpret_cast<const uint4*>(p));
  v[0] = bf16lo(a.x); v[1] = bf16hi(a.x); v[2] = bf16lo(a.y); v[3] = bf16hi(a.y);
  v[4] = bf16lo(a.z); v[5] = bf16hi(a.z); v[6] = bf16lo(a.w); v[7] = bf16hi(a.w);
}
__device__ __forceinline__ void store8(float* p, const float* v) {
  reinterpret_cast<float4*>(p)[0] = make_float4(v[0], v[1], v[2], v[3]);
  reinterpret_cast<float4*>(p)[1] = make_float4(v[4], v[5], v[6], v[7]);
}
__device__ __forceinline__ void store8(bf16* p, const float* v) {
  uint4 a;
  a.x = pack_bf16x2(v[0], v[1]); a.y = pack_bf16x2(v[2], v[3]);
  a.z = pack_bf16x2(v[4], v[5]); a.w = pack_bf16x2(v[6], v[7]);
  *reinterpret_cast<uint4*>(p) = a;
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// Sum of fp32 values kept as s + e: the rounding errors of the additions to s
// are exact (TwoSum), their sum e is rounded, about 2^-46 relative in all, at
// 1/64 of what fp64 sums cost on this part.  The range is that of fp32: an
// addition that overflows leaves NaN in e.
struct PairSum {
  float s = 0.f, e = 0.f;
  __device__ __forceinline__ void add(float x) {
    const float t = __fadd_rn(s, x);
    const float bb = __fadd_rn(t, -s);
    e = __fadd_rn(e, __fadd_rn(__fadd_rn(s, -__fadd_rn(t, -bb)), __fadd_rn(x, -bb)));
    s = t;
  }
  __device__ __forceinline__ void add(const PairSum& p) { add(p.s); e = __fadd_rn(e, p.e); }
  // + x^2 (of a bf16 x the product is exact)
  __device__ __forceinline__ void add_square(float x, bool exact) {
    const float p = __fmul_rn(x, x);
    add(p);
    if (!exact) e = __fadd_rn(e, __fmaf_rn(x, x, -p));
  }
  __device__ __forceinline__ double value() const { return static_cast<double>(s) + static_cast<double>(e); }
};

// Sum over the whole block; every thread gets the result.  `red` must hold
// blockDim.x / 32 entries.  Deterministic (fixed tree order).
template <typename T>
__device__ __forceinline__ T block_sum(T v, T* red) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  v = warp_sum(v);
  __syncthreads();
  if (lane == 0) red[wid] = v;
  __syncthreads();
  T s = 0;
  for (int i = 0; i < nw; ++i) s += red[i];
  return s;
}

}  // namespace normpre
