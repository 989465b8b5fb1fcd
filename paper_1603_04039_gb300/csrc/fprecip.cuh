// fprecip.cuh -- FP64 reciprocals in few issue slots of the FP64 pipe.
#pragma once

#include "fpconv.cuh"

namespace apc {

// 1 / sqrt(g) and 1 / x in FP64 from an FP32 start, one third-order step each
// (Halley's iteration; with e = 1 - g y^2 or 1 - x y, |e| < 2^-22, the
// neglected terms are below 2^-64): 5 and 3 issue slots of the FP64 pipe, the
// conversions on the integer pipe.  g and x well inside the FP32 range.  Rounded
// to 1.51 (the product g y enters the step rounded) and 1.0 times 2^-53, checked by
// tests/test_gpu_fprecip.py.
__device__ __forceinline__ double rsqrt_f64(double g) {
    const double y = f32_to_f64_int(rsqrtf(f64_to_f32_int(g)));
    const double e = fma(-(g * y), y, 1.0);
    return fma(y, fma(e, 0.375, 0.5) * e, y);
}
__device__ __forceinline__ double recip_f64(double x) {
    const double y = f32_to_f64_int(1.0f / f64_to_f32_int(x));
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}

}  // namespace apc
