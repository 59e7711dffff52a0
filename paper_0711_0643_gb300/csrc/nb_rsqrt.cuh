// The FP64 reciprocal square root of the FP64 force kernel.
#pragma once

namespace nb {

// (r2)^(-1/2) by a third-order Householder step from an FP32 estimate q0:
// e = 1 - r2 q0^2 (q0^2 is exact in FP64 and the difference rounds once), q = q0 + q0 e
// (1/2 + 3/8 e). r2 is truncated to FP32 (2^-23) and CUDA gives rsqrtf 2 ulp (2^-22), so |e| <
// 2^-20.6 and the step leaves 5/16 e^3 < 2^-63.4 relative; its roundings but the last are
// below 2^-73. So q is within 0.501 ulp (tests/test_gpu_rsqrt.py, against exact arithmetic).
// The conversions to and from FP32 are moves of the bit fields (FP64 conversions share
// the narrow pipe). Only where r2 is not comfortably a normal FP32 number, outside
// [2^-120, 2^120): the library function.
__device__ __forceinline__ double rsqrt_f64(double r2)
{
    const int hi = __double2hiint(r2);
    if ((unsigned)(hi - ((1023 - 120) << 20)) >= (unsigned)(240 << 20)) return rsqrt(r2);
    const float f = __int_as_float(__funnelshift_l(__double2loint(r2), hi - (896 << 20), 3));
    const int qb = __float_as_int(rsqrtf(f));
    const double q0 = __hiloint2double((qb >> 3) + (896 << 20), qb << 29);
    const double e = fma(-r2, q0 * q0, 1.0);
    return fma(q0 * e, fma(e, 0.375, 0.5), q0);
}

}  // namespace nb
