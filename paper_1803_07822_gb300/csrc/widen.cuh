// FP32 values in FP64 without FP64-pipe conversions, for the readout kernels.
#pragma once

#include "fp_convert.h"

namespace cslbm {

// FP32 as FP64 on the integer units; `odd` becomes true for a subnormal, an
// infinity or a NaN, which the result does not hold
__device__ __forceinline__ double widen(float f, bool& odd)
{
    const unsigned b = __float_as_uint(f), m = b & 0x7fffffffu;
    odd = odd || (m != 0u && m - 0x00800000u >= 0x7f000000u);
    return __hiloint2double(m ? (int)((b & 0x80000000u) | ((m >> 3) + 0x38000000u)) : (int)b, (int)(b << 29));
}

// 1 / rho from an FP32 estimate and two Newton steps (error below 2^-52), and
// rho itself in FP64; `odd` becomes true outside (2^-64, 2^64)
__device__ __forceinline__ double recip64(float rho, double& r, bool& odd)
{
    odd = odd || !(rho > 0x1p-64f && rho < 0x1p64f);
    r = widen(rho, odd);
    const double y0 = f32_to_f64(__frcp_rn(rho));
    const double y1 = fma(y0, fma(-r, y0, 1.0), y0);
    return fma(y1, fma(-r, y1, 1.0), y1);
}

}  // namespace cslbm
