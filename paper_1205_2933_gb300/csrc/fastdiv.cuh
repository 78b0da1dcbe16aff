#pragma once

#include <stdint.h>

namespace dwf {

// n / d for 0 <= n < 2^31 as a multiply-high, an addition and a shift
struct FastDiv {
    unsigned m;
    int l, d;
    __device__ __forceinline__ unsigned div(unsigned n) const { return (__umulhi(m, n) + n) >> l; }
};

inline FastDiv fast_div(int d) {
    FastDiv f{0, 0, d};
    while (((int64_t)1 << f.l) < d) ++f.l;
    f.m = (unsigned)((((uint64_t)1 << 32) * (((uint64_t)1 << f.l) - (uint64_t)d)) / (uint64_t)d + 1);
    return f;
}

}  // namespace dwf
