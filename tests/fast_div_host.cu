// The division by a fixed divisor of csrc/fast_div.cuh, exported for tests/test_fast_div_host.py
#include "fast_div.cuh"

extern "C" int fast_div_first_wrong(unsigned d, const int *n, int count) {
    const dlz::FastDiv f(d);
    for (int i = 0; i < count; ++i)
        if (f.div(n[i]) != (int)((unsigned)n[i] / d)) return i;
    return -1;
}
