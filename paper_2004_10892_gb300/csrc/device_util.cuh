// device_util.cuh -- small device helpers shared by the contraction kernels.
#pragma once
#include <cuda_runtime.h>

namespace tnq {

// Scale 2^-m that brings a tensor whose largest |re|,|im| has float bits
// `mbits` into [0.5, 1); m is returned through *mexp.
__device__ __forceinline__ float scale_of_max(unsigned mbits, int* mexp) {
  if (mbits == 0u) {
    *mexp = 0;
    return 1.f;
  }
  int ex = (int)((mbits >> 23) & 0xffu);
  if (ex == 0) ex = 1;
  int m = ex - 126;
  if (m > 126) m = 126;
  *mexp = m;
  return __int_as_float((127 - m) << 23);
}

// The roundings are spelled out: left to the compiler, which products it fuses
// depends on the surrounding code, and kernels that share a bucket's arithmetic
// must agree (a slice's value must not depend on the batch, to the last bit).
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -__fmul_rn(a.y, b.y)), fmaf(a.x, b.y, __fmul_rn(a.y, b.x)));
}

__device__ __forceinline__ void atomic_max_pos(unsigned* p, float v) {
  const unsigned b = __float_as_uint(v);
  if (b > *reinterpret_cast<volatile unsigned*>(p)) atomicMax(p, b);
}

}  // namespace tnq
