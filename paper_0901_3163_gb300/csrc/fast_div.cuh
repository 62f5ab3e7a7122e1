// Division by a divisor that is fixed for a launch: a multiplication and a shift instead of the
// integer-division sequence (about 20 instructions, of which a stencil kernel needs nine for
// its block's and its sites' coordinates).
#pragma once

namespace dlz {

// n / d for 0 <= n < 2^31, d >= 1 (T. Granlund and P. Montgomery, "Division by Invariant
// Integers using Multiplication", 1994): with 2^(s-1) < d <= 2^s and m = floor(2^32 (2^s - d) /
// d) + 1 the quotient is (floor(m n / 2^32) + n) >> s.
struct FastDiv {
    unsigned d = 1, m = 1, s = 0;
    FastDiv() = default;
    __host__ explicit FastDiv(unsigned divisor) : d(divisor) {
        while ((1ull << s) < d) ++s;
        m = (unsigned)(((1ull << 32) * ((1ull << s) - d)) / d + 1);
    }
    __host__ __device__ inline int div(int n) const {
#if defined(__CUDA_ARCH__)
        const unsigned hi = __umulhi(m, (unsigned)n);
#else
        const unsigned hi = (unsigned)(((unsigned long long)m * (unsigned)n) >> 32);
#endif
        return (int)((hi + (unsigned)n) >> s);
    }
};

}  // namespace dlz
