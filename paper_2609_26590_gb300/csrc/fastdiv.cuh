// fastdiv.cuh -- division by a launch constant with a multiply-high and a shift, for
// the kernels' index arithmetic (the host runs the same code in its plan queries).
#pragma once

#include <cstdint>

namespace gtr {

// Division by a launch constant 1 <= d < 2^31 of 0 <= n < 2^31 by a multiply-high and a
// shift (Granlund and Montgomery, "Division by invariant integers using multiplication",
// 1994, Thm. 4.2): with l = ceil(log2 d) and m = floor(2^32 (2^l - d) / d) + 1, the 33-bit
// multiplier 2^32 + m satisfies 2^(32+l) < (2^32 + m) d <= 2^(32+l) + 2^l, so
// n / d = (umulhi(n, m) + n) >> l, the sum exact in 32 bits for n < 2^31.  A few
// instructions instead of an integer division's sequence: every role's per-chunk index
// arithmetic uses it, which keeps the kernel's hot code small (the SM's instruction cache
// is shared by all roles; the divisions of one decode cost a balanced launch 17 %).
struct FastDiv {
    int d;
    uint32_t m, l;
};
inline FastDiv make_fastdiv(int d) {
    if (d < 1) d = 1;
    uint32_t l = 0;
    while ((1ull << l) < static_cast<unsigned long long>(d)) ++l;
    return FastDiv{d, static_cast<uint32_t>(((1ull << 32) * ((1ull << l) - d)) / d + 1), l};
}
__host__ __device__ __forceinline__ int fdiv(int n, const FastDiv &f) {
#ifdef __CUDA_ARCH__
    const uint32_t hi = __umulhi(static_cast<uint32_t>(n), f.m);
#else
    const uint32_t hi = static_cast<uint32_t>((static_cast<uint64_t>(static_cast<uint32_t>(n)) * f.m) >> 32);
#endif
    return static_cast<int>((hi + static_cast<uint32_t>(n)) >> f.l);
}

}  // namespace gtr
