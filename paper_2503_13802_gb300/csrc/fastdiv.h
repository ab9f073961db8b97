// Division of small non-negative integers by a run-time constant through a
// multiplication.
#pragma once

#include <cstdint>

#include <cuda_runtime.h>

namespace mh3d {

// n / d for 0 <= n < 2^31 (d >= 1): m = ceil(2^(31+l) / d), l = ceil(log2 d),
// has an error below 1, so n m / 2^(31+l) is off by less than 2^-l <= 1/d and
// its floor is exact.
struct FastDiv {
    uint32_t d = 1, m = 0, s = 0;
    FastDiv() = default;
    explicit FastDiv(int div) : d((uint32_t)div)
    {
        uint32_t l = 0;
        while ((1ull << l) < d) ++l;
        if (d > 1) {
            m = (uint32_t)(((1ull << (31 + l)) + d - 1) / d);
            s = l - 1;
        }
    }
    __host__ __device__ __forceinline__ uint32_t div(uint32_t n) const
    {
#ifdef __CUDA_ARCH__
        return d == 1 ? n : __umulhi(n, m) >> s;
#else
        return d == 1 ? n : (uint32_t)(((unsigned long long)n * m) >> 32) >> s;
#endif
    }
};

}  // namespace mh3d
