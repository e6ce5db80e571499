// Division by a number the host knows: a multiplication and a shift, exact for every 0 <= n < 2^31 and 1 <= d < 2^31.
// With l = ceil(log2 d), mul = ceil(2^(31 + l) / d) fits in 32 bits and exceeds 2^(31 + l) / d by less than 1, so
// n * mul / 2^(31 + l) exceeds n / d by less than n / 2^(31 + l) < 2^-l <= 1 / d: too little to reach the next integer.
// (fdiv() of mma_common.cuh is one instruction shorter but exact only for n * d < 2^32: for numbers that stay small.)
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define BRA_HD __host__ __device__ __forceinline__
#else
#define BRA_HD inline
#endif

namespace bra {

struct FastDiv { uint32_t mul, shift; };

inline FastDiv fast_div(int d) {
    FastDiv f = {0, 0};
    while ((1u << f.shift) < (uint32_t)d) ++f.shift;
    f.mul = (uint32_t)(((1ull << (31 + f.shift)) + (uint64_t)d - 1) / (uint64_t)d);
    return f;
}

BRA_HD uint32_t fdiv(uint32_t n, const FastDiv& f) {
#ifdef __CUDA_ARCH__
    return __umulhi(n + n, f.mul) >> f.shift;
#else
    return (uint32_t)(((uint64_t)(n + n) * f.mul) >> 32) >> f.shift;
#endif
}

}  // namespace bra
