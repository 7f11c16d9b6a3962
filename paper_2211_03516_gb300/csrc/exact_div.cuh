// Division of indices below 2^31 by a divisor that the host knows: one widening multiply and a shift.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define VAMRT_HD __host__ __device__ __forceinline__
#else
#define VAMRT_HD inline
#endif

namespace vamrt {

// i / d for 0 <= i < 2^31 and 1 <= d < 2^31.  With s the least integer of 2^s >= d and m = floor(2^(31 +
// s) / d) + 1, m d = 2^(31 + s) + e, 0 < e <= d, so i m / 2^(31 + s) exceeds i / d by i e / (d 2^(31 + s)) <
// 1 / d: the floors agree.  m < 2^32, since d > 2^(s - 1).
struct ExactDiv {
    uint32_t m;
    int shift;
    explicit ExactDiv(uint32_t d)
    {
        int s = 0;
        while (((uint64_t)1 << s) < d) ++s;
        shift = 31 + s;
        m = (uint32_t)(((uint64_t)1 << shift) / d + 1);
    }
    VAMRT_HD uint32_t operator()(uint32_t i) const { return (uint32_t)(((uint64_t)i * m) >> shift); }
};

}  // namespace vamrt
