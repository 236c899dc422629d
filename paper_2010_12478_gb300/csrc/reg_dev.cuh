// Device helpers shared by the kernel translation units: storage-typed loads and stores, and the
// float-float sums (error-free transformations on the FP32 pipes).
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>

namespace reg {

// ------------------------------------------------------------------ loads
template <typename S> __device__ __forceinline__ float ldS(const S *p);
template <> __device__ __forceinline__ float ldS<float>(const float *p) { return __ldg(p); }
template <> __device__ __forceinline__ float ldS<__nv_bfloat16>(const __nv_bfloat16 *p)
{
    return __bfloat162float(__ldg(p));
}
template <> __device__ __forceinline__ float ldS<__half>(const __half *p) { return __half2float(__ldg(p)); }

__device__ __forceinline__ float fromS(float v) { return v; }
__device__ __forceinline__ float fromS(__nv_bfloat16 v) { return __bfloat162float(v); }
__device__ __forceinline__ float fromS(__half v) { return __half2float(v); }

template <typename S> __device__ __forceinline__ S toS(float v);
template <> __device__ __forceinline__ float toS<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 toS<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }
template <> __device__ __forceinline__ __half toS<__half>(float v) { return __float2half_rn(v); }

// ------------------------------------------------------------------ float-float
// (hi, lo) += x, exactly up to the final rounding of lo (Knuth's TwoSum).
__device__ __forceinline__ void ff_acc(float &hi, float &lo, float x)
{
    float s = __fadd_rn(hi, x);
    float bp = __fsub_rn(s, hi);
    float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bp)), __fsub_rn(x, bp));
    hi = s;
    lo = __fadd_rn(lo, e);
}

// (hi, lo) += (h2, l2), renormalised.
__device__ __forceinline__ void ff_add(float &hi, float &lo, float h2, float l2)
{
    float s = __fadd_rn(hi, h2);
    float bp = __fsub_rn(s, hi);
    float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bp)), __fsub_rn(h2, bp));
    e = __fadd_rn(e, __fadd_rn(lo, l2));
    float h = __fadd_rn(s, e);
    lo = __fsub_rn(e, __fsub_rn(h, s));
    hi = h;
}

}  // namespace reg
