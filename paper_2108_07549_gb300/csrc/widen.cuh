// widen.cuh -- FP32 to FP64 conversion on the integer pipe.
#pragma once

#include "pdr_internal.cuh"

namespace pdr {
namespace {

// (double)x, bit for bit.  GB300 converts at its FP64 rate, two per clock and
// SM, which bounded the kernels that widen every element (widen_rows_kernel at
// 99 M elements: 418 us, FP64 pipe 42 % busy).  A normal float's bits move into
// place with shifts and one addition of the exponent bias difference; zeros
// keep their sign; subnormals, infinities and NaNs take the conversion.
__device__ __forceinline__ double widen(float x)
{
    const uint32_t b = __float_as_uint(x), m = b & 0x7fffffffu;
    if (m - 0x00800000u < 0x7f000000u || m == 0u) {
        const uint32_t hi = (b & 0x80000000u) | (m == 0u ? 0u : (m >> 3) + 0x38000000u);
        return __hiloint2double((int)hi, (int)(m << 29));
    }
    return (double)x;
}

}  // namespace
}  // namespace pdr
