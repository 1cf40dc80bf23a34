// float32 -> float64 by integer operations.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

namespace mpspt {

// The value of every float32, b its bits (a conversion instruction occupies a
// sub-partition's float64 unit for 64 clocks: 2 us for a tile of 128 x 64).
// Subnormal values, which the sums of a product reach only below 1.2e-38, take
// the branch.
__device__ __forceinline__ double f2d_int(uint32_t b) {
    const uint32_t sign = b & 0x80000000u;
    uint32_t mag = b & 0x7FFFFFFFu, e = 896u << 20;
    if (mag < 0x00800000u) {
        if (mag == 0u) return __hiloint2double((int)sign, 0);
        const int sh = __clz((int)mag) - 8;   // up to the place of the leading one
        mag = (mag << sh) & 0x7FFFFFu;
        e = (uint32_t)(897 - sh) << 20;
    }
    uint32_t hi = (mag >> 3) + e;
    if (mag >= 0x7F800000u) hi = 0x7FF00000u | ((mag & 0x7FFFFFu) >> 3);
    return __hiloint2double((int)(sign | hi), (int)(mag << 29));
}

}  // namespace mpspt
