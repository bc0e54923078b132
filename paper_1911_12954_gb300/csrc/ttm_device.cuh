// ttm_device.cuh - device helpers shared by the tensor passes (tensor_ops.cu, sectors.cu): the
// operand splits and their power-of-two scales, the magnitude maximum, element addressing.
#pragma once

#include <cuda_fp16.h>

#include "common.cuh"

namespace hotrg {

__device__ __forceinline__ float tf32_round(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return __uint_as_float(r);
}

// Exact 8-bit slices of x (|x| < 1, FP64): r <- 256 r, v = rint(r), r <- r - v, five times;
// every step is exact in FP64 and every v an integer fp16 holds exactly (|v| <= 256).
__device__ __forceinline__ void oz_store(__half* out, int64_t plane, int64_t o, double x) {
  double r = x;
#pragma unroll
  for (int i = 0; i < kOzSlices; ++i) {
    r *= 256.0;
    const double v = rint(r);
    out[o + i * plane] = __float2half_rn((float)v);
    r -= v;
  }
}

// Two neighbouring entries (o even): one 4-byte store per plane.
__device__ __forceinline__ void oz_store2(__half* out, int64_t plane, int64_t o, double x0, double x1) {
  double r0 = x0, r1 = x1;
#pragma unroll
  for (int i = 0; i < kOzSlices; ++i) {
    r0 *= 256.0;
    r1 *= 256.0;
    const double v0 = rint(r0), v1 = rint(r1);
    *(__half2*)(out + o + i * plane) = __floats2half2_rn((float)v0, (float)v1);
    r0 -= v0;
    r1 -= v1;
  }
}

// Power-of-two scale of a split pass: from the operand's largest magnitude (a max pass of the
// same contraction wrote it to amax) or, without one, the fixed 2^14 of the fp16 planes.
template <int MODE>
__device__ __forceinline__ double split_scale(const unsigned* amax) {
  if (MODE == kTTMSplitF16) return amax ? ldexp(1.0, split_exponent(*amax, kF16Top)) : (double)kF16Scale;
  if (MODE == kTTMSplitOz) return ldexp(1.0, amax ? split_exponent(*amax, kOzTop) : kOzTop);
  return 1.0;
}

// Largest magnitude seen by the threads of a block, times mul, merged into *amax (bits of a
// non-negative float, rounded up, so that the recorded value bounds mul times every output).
__device__ __forceinline__ void merge_max(unsigned* amax, double m, float mul) {
  float f = __double2float_ru(m * (double)mul);
  for (int off = 16; off > 0; off >>= 1) f = fmaxf(f, __shfl_down_sync(0xffffffffu, f, off));
  if ((threadIdx.x & 31) == 0 && f > 0.f && amax) atomicMax(amax, __float_as_uint(f));
}

// Output pointer of batch element e: the split modes write fp16 planes, whose strides count
// fp16 values; the others count elements of the output type.
template <typename TO, int MODE>
__device__ __forceinline__ TO* elem_out(TO* p, int64_t off) {
  if (!p) return p;
  if (MODE == kTTMSplitF16 || MODE == kTTMSplitOz) return (TO*)((__half*)p + off);
  return p + off;
}

}  // namespace hotrg
