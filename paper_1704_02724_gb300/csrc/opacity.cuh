// Opacity of a segment, e^-x - 1 for x = sigma l, in the two precisions of the link traversals.
#pragma once

#include <cuda_runtime.h>

namespace canvox {
namespace {

// e^-x - 1 for x >= 0, and just below 0 (a segment can come out that much too short). The argument is reduced by a whole
// number n of ln 2 (Cody and Waite 1980; one word of ln 2 does, as the part it leaves out is scaled by 2^n too):
// -x = n ln 2 + f, |f| <= 0.347, e^f - 1 = f + f^2 q(f) with q the degree-4 minimax polynomial (relative error 2^-26),
// e^-x - 1 = 2^n (e^f - 1) + (2^n - 1). Within 0.96 ulp for every argument (all binary32 values from 2^-40 on compared;
// the library's has 1), in 13 instructions without a branch, against about 20 of expm1f. x (1 + x r(x)) on [0, 1) with
// the hardware exponential beyond took 12, but reached 1.58 ulp and, by that instruction's documented error, 1.9. The
// difference is up to 1 % of the depth-24 and -27 views (a stereo pair of 2160^2 329.0 -> 325.0 Mrays/s, a quarter of it the
// exit time's bound and the mask of the position's bits; two depth-27 pairs 7.27 -> 7.34 ms), 0.3 % of a 256^2 view of the
// depth-8 cube and nothing of an opaque one. The even and odd terms apart keep the chain two operations shorter.
__device__ __forceinline__ float expm1_neg(float x) {
    constexpr float kRound = 12583039.0f;  // 1.5 2^23 + 127: adding it rounds to a whole number, n + 127 in the low bits
    const float y = fminf(x, 88.0f);       // (beyond, e^-x is below half an ulp of 1 either way)
    const float t = __fmaf_rn(y, -1.44269504f, kRound);
    const float f = __fmaf_rn(__fsub_rn(t, kRound), -0.693147181f, -y);
    const float f2 = __fmul_rn(f, f);      // (even and odd terms apart: two operations less on the chain)
    const float q = __fmaf_rn(__fmaf_rn(0.00138824887f, f2, __fmaf_rn(0.00836669188f, f, 0.0416672826f)), f2,
                              __fmaf_rn(0.16666536f, f, 0.49999997f));
    const float p = __fmaf_rn(q, f2, f);
    const float s = __int_as_float(__float_as_int(t) << 23);  // 2^n
    return __fmaf_rn(p, s, __fsub_rn(s, 1.0f));
}

__device__ __forceinline__ bool less_pos(double a, double b) {  // of numbers that are not both negative
    return __double_as_longlong(a) < __double_as_longlong(b);
}

// e^-x - 1. Below 1/8 (most leaves: thin paint, small cells) its Taylor series to x^10 / 10! (the next term is 2^-55 of the
// value; within 2^-52 of it in all), 10 FP64 operations; else the library's.
__device__ __forceinline__ double expm1_neg64(double x) {
    const double y = -x;
    if (less_pos(x, 0.125)) {
        double p = fma(2.7557319223985893e-07, y, 2.7557319223985893e-06);
        p = fma(p, y, 2.4801587301587302e-05);
        p = fma(p, y, 1.9841269841269841e-04);
        p = fma(p, y, 1.3888888888888889e-03);
        p = fma(p, y, 8.3333333333333332e-03);
        p = fma(p, y, 4.1666666666666664e-02);
        p = fma(p, y, 0.16666666666666666);
        p = fma(p, y, 0.5);
        return fma(p * y, y, y);
    }
    return expm1(y);
}

}  // namespace
}  // namespace canvox
