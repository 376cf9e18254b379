// Reciprocal square root of a normal positive FP64 number with few FP64 instructions, for the QL
// recurrence (k_snr_big.cu).
#pragma once
#include <cuda_runtime.h>

namespace otvmc {

// 1 / sqrt(h), 2^-958 <= h < 2^977.  y, FP32's reciprocal root of h's mantissa (to 23 bits) with h's
// exponent halved, is within 2^-21.5 of it; with e = 1 - h y^2 the root is y (1 - e)^(-1/2), of whose
// binomial series 1 + e / 2 + 3 e^2 / 8 + 5 e^3 / 16 + ... the first three terms are kept: the rest is
// below 2^-63, and the roundings (of h y, and of the result) make 1.5 2^-53 in all.
__device__ __forceinline__ double rsqrt_pos(double h) {
    const int hw = __double2hiint(h), lw = __double2loint(h);
    const int E = (hw >> 20) - 1023, k = E >> 1;  // h = mantissa 2^(E & 1) 2^(2 k)
    const float m = __int_as_float(((127 + (E & 1)) << 23) | ((hw & 0xFFFFF) << 3) | (int)((unsigned)lw >> 29));
    const int yb = __float_as_int(rsqrtf(m));
    const double y = __hiloint2double((((yb >> 23) + 896 - k) << 20) | ((yb & 0x7FFFFF) >> 3), yb << 29);
    const double e = fma(-(h * y), y, 1.0);
    return fma(y * e, fma(0.375, e, 0.5), y);
}

}  // namespace otvmc
