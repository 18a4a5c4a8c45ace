// Cutting values into BF16 planes, and view offsets (device helpers of the
// tensor-core path's conversion kernels).
#pragma once
#include <cuda_bf16.h>

#include "common.cuh"

// x = hi + lo with hi the FP32 value of x rounded toward zero and lo what is
// left, to 24 bits.  FP64 instructions and FP64 <-> FP32 conversions run on a
// pipe of two lanes per SM, 64 times slower than integer ones, so the parts
// are cut from the bits; x below 2^-74 or above FP32's range takes the slow
// conversions (where hi and lo round as the format does).
__device__ __forceinline__ void f64_parts(double x, float& hi, float& lo) {
  const unsigned h = (unsigned)__double2hiint(x), l = (unsigned)__double2loint(x);
  const int ef = (int)((h >> 20) & 0x7ff) - 896;   // FP32's biased exponent
  const unsigned sign = h & 0x80000000u;
  if (ef >= 53 && ef <= 254) {
    hi = __uint_as_float(sign | ((unsigned)ef << 23) | ((h & 0xfffffu) << 3) | (l >> 29));
    const float m = (float)(int)(l & 0x1fffffffu);
    lo = m * __uint_as_float(sign | ((unsigned)(ef - 52) << 23));
  } else if (((h << 1) | l) == 0) {
    hi = lo = 0.f;
  } else {
    hi = (float)x;
    lo = (float)(x - (double)hi);
  }
}
__device__ __forceinline__ void parts(double x, float& hi, float& lo) { f64_parts(x, hi, lo); }
__device__ __forceinline__ void parts(float x, float& hi, float& lo) {
  hi = x;
  lo = 0.f;
}

// the BF16 planes of x: p0 + p1 + p2 = x to 2^-26
template <typename S>
__device__ __forceinline__ void cut(S x, unsigned short* w) {
  float hi, lo;
  parts(x, hi, lo);
  const __nv_bfloat16 p0 = __float2bfloat16_rn(hi);
  const float r1 = (hi - __bfloat162float(p0)) + lo;
  const __nv_bfloat16 p1 = __float2bfloat16_rn(r1);
  const __nv_bfloat16 p2 = __float2bfloat16_rn(r1 - __bfloat162float(p1));
  w[0] = __bfloat16_as_ushort(p0);
  w[1] = __bfloat16_as_ushort(p1);
  w[2] = __bfloat16_as_ushort(p2);
}

// an FP32 value as FP64, by integer operations for normal values
__device__ __forceinline__ double f32_to_f64(float x) {
  const unsigned u = __float_as_uint(x), e = (u >> 23) & 0xff;
  if (e - 1u < 254u)
    return __hiloint2double((int)((u & 0x80000000u) | (((u >> 3) & 0x0fffffffu) + 0x38000000u)),
                            (int)(u << 29));
  return (u << 1) == 0 ? __hiloint2double((int)u, 0) : (double)x;
}

// offset of a view's index with 32-bit divisions (indices are below 2^31)
__device__ __forceinline__ long long off32(const Idx3& d, unsigned idx) {
  if (d.n0 == 1 && d.n1 == 1) return (long long)idx * d.s2;
  const unsigned t = idx / (unsigned)d.n0, i0 = idx - t * (unsigned)d.n0;
  const unsigned i2 = t / (unsigned)d.n1, i1 = t - i2 * (unsigned)d.n1;
  return (long long)i2 * d.s2 + (long long)i1 * d.s1 + (long long)i0 * d.s0;
}
