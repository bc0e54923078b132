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

// The five slices of x (|x| < 1, FP64), given as x2 = 2^62 x: x = sum_i v_i 2^-8(i+1) up to 2^-41, each v_i the
// integer nearest what the earlier ones leave (ties to even; |v_0| <= 256, |v_i| <= 128). Cut from the 62-bit
// fixed-point value of x in integer arithmetic: one conversion and one comparison on the FP64 pipe, where
// five rounds of multiply, round and subtract took most of a pass (D = 6: 3.2 ms). A slice becomes
// fp16 as (1536 + v) - 1536, both steps exact. Values that are not finite become NaN.
__device__ __forceinline__ int oz_next(long long& n, int i) {   // slice i, in increasing i
  const int s = 54 - 8 * i;
  const int v = (int)((n + ((1ll << (s - 1)) - 1) + ((n >> s) & 1)) >> s);
  n -= (long long)v << s;
  return v;
}
__device__ __forceinline__ __half oz_half(int v) { return __ushort_as_half((unsigned short)(0x6600 + v)); }   // 1536 + v

__device__ __forceinline__ void oz_store(__half* out, int64_t plane, int64_t o, double x2) {
  long long n = __double2ll_rn(x2);
  const bool fine = fabs(x2) <= 0x1p62;
#pragma unroll
  for (int i = 0; i < kOzSlices; ++i) {
    const __half h = __hsub(oz_half(oz_next(n, i)), oz_half(0));
    out[o + i * plane] = fine ? h : __ushort_as_half((unsigned short)0x7fff);
  }
}
// Two neighbouring entries (o even): one 4-byte store per plane.
__device__ __forceinline__ void oz_store2(__half* out, int64_t plane, int64_t o, double x0, double x1) {
  long long n0 = __double2ll_rn(x0), n1 = __double2ll_rn(x1);
  const bool fine = fabs(x0) <= 0x1p62 && fabs(x1) <= 0x1p62;
#pragma unroll
  for (int i = 0; i < kOzSlices; ++i) {
    const int v0 = oz_next(n0, i), v1 = oz_next(n1, i);
    __half2 h = __hsub2(__halves2half2(oz_half(v0), oz_half(v1)), __half2half2(oz_half(0)));
    if (!fine) h = __half2half2(__ushort_as_half((unsigned short)0x7fff));
    *(__half2*)(out + o + i * plane) = h;
  }
}

// Power-of-two scale of a split pass: from the operand's largest magnitude (a max pass of the
// same contraction wrote it to amax) or, without one, the fixed 2^14 of the fp16 planes.
template <int MODE>
__device__ __forceinline__ double split_scale(const unsigned* amax) {
  if (MODE == kTTMSplitF16) return amax ? ldexp(1.0, split_exponent(*amax, kF16Top)) : (double)kF16Scale;
  if (MODE == kTTMSplitOz) return ldexp(1.0, 62 + (amax ? split_exponent(*amax, kOzTop) : kOzTop));   // oz_store takes 2^62 x
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
