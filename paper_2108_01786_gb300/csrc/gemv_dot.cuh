// Inner-product helpers shared by the single-problem and batched GEMVs:
// 16-byte dot products of stored matrix entries (FP32, FP16, BF16) with FP32
// vectors, and the double-float product-accumulate of the hi + lo residual.
#pragma once
#include "common.cuh"
#include "tfl.h"

template <class TA> struct Dot16;
template <> struct Dot16<float> {
  static constexpr int E = 4;
  static __device__ __forceinline__ float run(float acc, const uint4& q, const float* xs) {
    const float4 b = *reinterpret_cast<const float4*>(xs);
    acc = fmaf(__uint_as_float(q.x), b.x, acc);
    acc = fmaf(__uint_as_float(q.y), b.y, acc);
    acc = fmaf(__uint_as_float(q.z), b.z, acc);
    acc = fmaf(__uint_as_float(q.w), b.w, acc);
    return acc;
  }
  // four rows against the same four entries of x
  static __device__ __forceinline__ void run4(float* acc, const uint4* q, const float* xs) {
    const float4 b = *reinterpret_cast<const float4*>(xs);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      acc[i] = fmaf(__uint_as_float(q[i].x), b.x, acc[i]);
      acc[i] = fmaf(__uint_as_float(q[i].y), b.y, acc[i]);
      acc[i] = fmaf(__uint_as_float(q[i].z), b.z, acc[i]);
      acc[i] = fmaf(__uint_as_float(q[i].w), b.w, acc[i]);
    }
  }
};
template <> struct Dot16<__half> {
  static constexpr int E = 8;
  static __device__ __forceinline__ float run(float acc, const uint4& q, const float* xs) {
    const float4 b0 = *reinterpret_cast<const float4*>(xs);
    const float4 b1 = *reinterpret_cast<const float4*>(xs + 4);
    float2 f;
    f = __half22float2(*reinterpret_cast<const __half2*>(&q.x));
    acc = fmaf(f.x, b0.x, acc);
    acc = fmaf(f.y, b0.y, acc);
    f = __half22float2(*reinterpret_cast<const __half2*>(&q.y));
    acc = fmaf(f.x, b0.z, acc);
    acc = fmaf(f.y, b0.w, acc);
    f = __half22float2(*reinterpret_cast<const __half2*>(&q.z));
    acc = fmaf(f.x, b1.x, acc);
    acc = fmaf(f.y, b1.y, acc);
    f = __half22float2(*reinterpret_cast<const __half2*>(&q.w));
    acc = fmaf(f.x, b1.z, acc);
    acc = fmaf(f.y, b1.w, acc);
    return acc;
  }
  // four rows against the same eight entries of x
  static __device__ __forceinline__ void run4(float* acc, const uint4* q, const float* xs) {
    const float4 b0 = *reinterpret_cast<const float4*>(xs);
    const float4 b1 = *reinterpret_cast<const float4*>(xs + 4);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float2 f;
      f = __half22float2(*reinterpret_cast<const __half2*>(&q[i].x));
      acc[i] = fmaf(f.x, b0.x, acc[i]);
      acc[i] = fmaf(f.y, b0.y, acc[i]);
      f = __half22float2(*reinterpret_cast<const __half2*>(&q[i].y));
      acc[i] = fmaf(f.x, b0.z, acc[i]);
      acc[i] = fmaf(f.y, b0.w, acc[i]);
      f = __half22float2(*reinterpret_cast<const __half2*>(&q[i].z));
      acc[i] = fmaf(f.x, b1.x, acc[i]);
      acc[i] = fmaf(f.y, b1.y, acc[i]);
      f = __half22float2(*reinterpret_cast<const __half2*>(&q[i].w));
      acc[i] = fmaf(f.x, b1.z, acc[i]);
      acc[i] = fmaf(f.y, b1.w, acc[i]);
    }
  }
};
template <> struct Dot16<__nv_bfloat16> {
  static constexpr int E = 8;
  static __device__ __forceinline__ float run(float acc, const uint4& q, const float* xs) {
    const float4 b0 = *reinterpret_cast<const float4*>(xs);
    const float4 b1 = *reinterpret_cast<const float4*>(xs + 4);
    float2 f;
    f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&q.x));
    acc = fmaf(f.x, b0.x, acc);
    acc = fmaf(f.y, b0.y, acc);
    f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&q.y));
    acc = fmaf(f.x, b0.z, acc);
    acc = fmaf(f.y, b0.w, acc);
    f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&q.z));
    acc = fmaf(f.x, b1.x, acc);
    acc = fmaf(f.y, b1.y, acc);
    f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&q.w));
    acc = fmaf(f.x, b1.z, acc);
    acc = fmaf(f.y, b1.w, acc);
    return acc;
  }
  // four rows against the same eight entries of x
  static __device__ __forceinline__ void run4(float* acc, const uint4* q, const float* xs) {
    const float4 b0 = *reinterpret_cast<const float4*>(xs);
    const float4 b1 = *reinterpret_cast<const float4*>(xs + 4);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float2 f;
      f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&q[i].x));
      acc[i] = fmaf(f.x, b0.x, acc[i]);
      acc[i] = fmaf(f.y, b0.y, acc[i]);
      f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&q[i].y));
      acc[i] = fmaf(f.x, b0.z, acc[i]);
      acc[i] = fmaf(f.y, b0.w, acc[i]);
      f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&q[i].z));
      acc[i] = fmaf(f.x, b1.x, acc[i]);
      acc[i] = fmaf(f.y, b1.y, acc[i]);
      f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&q[i].w));
      acc[i] = fmaf(f.x, b1.z, acc[i]);
      acc[i] = fmaf(f.y, b1.w, acc[i]);
    }
  }
};

// s + (ah + al)(xh + xl) in double-float (the al xl term is below the precision)
__device__ __forceinline__ dfl df_acc_prod(dfl s, float ah, float al, float xh, float xl) {
  const dfl p = df_two_prod(ah, xh);
  float e = fmaf(ah, xl, p.lo);
  e = fmaf(al, xh, e);
  const dfl t = df_two_sum(s.hi, p.hi);
  const float lo = t.lo + (s.lo + e);
  return df_fast_two_sum(t.hi, lo);
}


// Three-float sums (tfl.h) are the flush target of short double-float runs: FP64
// accumulators cost 4 FP64 instructions per flush, 64 cycles of an SM's FP64 pipe per
// warp, which is what bound the hi + lo products whose matrix sits in L2; these are ~20
// FP32 instructions (5 cycles).
__device__ __forceinline__ tfl tf_lane(tfl a, int o) {
  return {__shfl_xor_sync(0xffffffffu, a.s, o), __shfl_xor_sync(0xffffffffu, a.e, o),
          __shfl_xor_sync(0xffffffffu, a.f, o)};
}
__device__ __forceinline__ tfl tf_warp_sum(tfl a) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) a = a + tf_lane(a, o);
  return a;
}
