// Sums of squares of FP32 numbers, to FP64's accuracy or better, in FP32 arithmetic (FP64 runs at a small
// fraction of the FP32 rate on the GPU). A sum is the unevaluated a + b + c: a the rounded sum, b the rounding
// errors of a, c those of b, each error found exactly (Knuth's two-sum; the square's by a fused multiply-add).
// What is left out is of the order of 2^-70 of the sum, so converting it to FP64 rounds about once (a relative
// error of 2^-53), where an FP64 sum rounds with every addition.
#pragma once

#include <cmath>

#ifdef __CUDACC__
#define IMRT_WIDE_FN __host__ __device__ __forceinline__
#else
#define IMRT_WIDE_FN inline
#endif

namespace imrt {

struct WideSum {
    float a, b, c;
};

IMRT_WIDE_FN void two_sum(float x, float y, float& s, float& err) {
    s = x + y;
    const float t = s - x;
    err = (x - (s - t)) + (y - t);
}

IMRT_WIDE_FN WideSum wide_add(WideSum u, WideSum v) {  // symmetric in u and v
    WideSum r;
    float ea, eb, ec;
    two_sum(u.a, v.a, r.a, ea);
    two_sum(u.b, v.b, eb, ec);
    float e2;
    two_sum(eb, ea, r.b, e2);
    r.c = (u.c + v.c) + (ec + e2);
    return r;
}

// x^2, exact while its rounding error is above the FP32 range's lower end (|x| > 2^-50).
IMRT_WIDE_FN WideSum wide_square(float x) {
#ifdef __CUDA_ARCH__
    const float p = __fmul_rn(x, x);  // (never fused with the addition that follows)
#else
    const float p = x * x;
#endif
    return WideSum{p, fmaf(x, x, -p), 0.0f};
}

IMRT_WIDE_FN double wide_to_double(WideSum s) { return (double)s.a + ((double)s.b + (double)s.c); }

}  // namespace imrt
