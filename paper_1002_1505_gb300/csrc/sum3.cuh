// A sum of floats carried as three floats: the two-sum (Knuth, TAOCP vol. 2) gives every addition's rounding
// error exactly, the error of the first part goes into the second and that of the second into the third,
// so only the third is rounded and the sum keeps about 70 bits.  Where a sum was held in FP64 and FP64
// additions (1/64 of the FP32 rate on this GPU) would set the pace, this holds no fewer bits.
#pragma once

#include <cuda_runtime.h>

namespace dda {

#ifdef __CUDACC__
struct Sum3 {
  float h, l, t;
  // a + b = return value + e, exactly
  static __device__ __forceinline__ float two_sum(float a, float b, float& e) {
    const float s = __fadd_rn(a, b), z = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, z)), __fsub_rn(b, z));
    return s;
  }
  __device__ __forceinline__ void add(float v) {
    float e, f;
    h = two_sum(h, v, e);
    l = two_sum(l, e, f);
    t = __fadd_rn(t, f);
  }
  __device__ __forceinline__ void add(const Sum3& o) {
    float e, f, g;
    h = two_sum(h, o.h, e);
    l = two_sum(l, o.l, f);
    l = two_sum(l, e, g);
    t = __fadd_rn(t, __fadd_rn(o.t, __fadd_rn(f, g)));
  }
  __device__ __forceinline__ double get() const { return (double)h + ((double)l + (double)t); }
};
#endif

}  // namespace dda
