// Double-word ("double-float") values on the FP32 units: a value is the
// unevaluated sum h + l of two FP32 numbers with |l| <= ulp(h) / 2, a 48-bit
// significand.  On this GPU FP64 runs at about 1/74 of the FP32 FMA rate, so
// the stencil passes of the reliable updates (r = b - A x recomputed at full
// accuracy, dslash_dw.cu) run faster in double-word arithmetic than in native
// FP64.
//
// fast_two_sum(a, b) gives s + e = a + b exactly for |a| >= |b| (3 operations; Dekker 1971,
// Knuth, TAOCP vol. 2, 4.2.2): it renormalises a sum and its error.  Sums and products
// are formed in dslash_dw.cu as compensated dot products.
#pragma once

#include <cuda_runtime.h>

namespace tmk {

struct df {
    float h, l;
    df() = default;
    __host__ __device__ __forceinline__ constexpr df(float a, float b) : h(a), l(b) {}
    // nearest double word of a double (FP64 operations: kernel parameters and
    // the conversion kernels only)
    __host__ __device__ __forceinline__ explicit df(double x)
        : h((float)x), l((float)(x - (double)(float)x)) {}
    __host__ __device__ __forceinline__ explicit operator double() const { return (double)h + (double)l; }
};

__device__ __forceinline__ df df_fast_two_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    return df(s, __fsub_rn(b, __fsub_rn(s, a)));
}

}  // namespace tmk
