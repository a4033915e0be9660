// 1/sqrt(x) of the FP64 force form in five FP64 instructions (an FP64 warp instruction holds
// its pipe for 64 cycles on this GPU).
//
// x = m 2^2q with m in [1, 4): the FP32 approximation y0 of 1/sqrt(m) times 2^-q, and one
// third-order Householder step, y = y0 + y0 e (1/2 + 3/8 e), e = 1 - x y0^2 (the binomial
// series of (1 - e)^(-1/2)).  y0 is off by 2 ulp of FP32 at most, 2^-22, and by 2^-24 more
// because m's bits beyond FP32 are cut off, so |e| < 2.5 2^-22 and the next term, (5/16) e^3,
// is below 2^-63.6.  y0^2 is exact (24 bits squared); the roundings of e and of y0 e are below
// 2^-73.  What is left is the last rounding: at most 0.501 ulp for every normal x.
#pragma once

namespace greem {

__device__ __forceinline__ double rsqrt_fp64(double x)
{
    const int hi = __double2hiint(x);
    if (hi < 0x00100000) return rsqrt(x);  // subnormal (and 0)
    const int ex = hi >> 20, odd = (ex & 1) ^ 1;
    const int mb = ((127 + odd) << 23) | ((hi & 0xfffff) << 3) | (int)((unsigned)__double2loint(x) >> 29);
    const int yb = __float_as_int(rsqrtf(__int_as_float(mb)));
    const int q = (ex - 1023 - odd) >> 1;
    const double y0 = __hiloint2double((yb >> 3) + 0x38000000 - (q << 20), (int)((unsigned)yb << 29));
    const double e = fma(-x, y0 * y0, 1.0);
    return fma(y0 * e, fma(e, 0.375, 0.5), y0);
}

}  // namespace greem
