// Root and reciprocal of a normal, finite x > 0 from an approximation y, without a branch, by
// Markstein's sequences (P. Markstein, "IA-64 and Elementary Functions", 2000): Newton steps
// on g ~ sqrt(x) and h ~ 1 / (2 sqrt(x)), or on y ~ 1 / x, and a last correction from the
// exact residual.  From a y within two units of the rounded value the root rounds as the exact
// one does for every significand, and the reciprocal for all but one: where x's significand
// is all ones, 1 / x lies just above the midpoint of a power of two and its successor, and the
// correction can tie to the power of two.  (GB300's own approximation happens to be rounded
// there.)  round_up_ones() sets the bit: two integer instructions per component, 100 steps of
// 4096^2 with their read-outs 28.8 ms with and without.
// R: float or f2, with the operations of lbm_device.cuh.
#pragma once

namespace lbm {

template <typename R>
__device__ __forceinline__ R sqrt_from(R x, R y) {
    const R g = mul_(x, y), h = mul_(y, R(0.5f)), r = fnma_(g, h, R(0.5f));
    const R g1 = fma_(g, r, g), h1 = fma_(h, r, h);
    return fma_(fnma_(g1, g1, x), h1, g1);
}

// y ~ 1 / x, or, for an x whose significand is all ones, its successor where y is even.
__device__ __forceinline__ float round_up_ones(float x, float y) {
    return (~__float_as_uint(x) & 0x7FFFFFu) ? y : __uint_as_float(__float_as_uint(y) | 1u);
}
template <typename R>
__device__ __forceinline__ R rcp_from(R x, R y) {
    const R y1 = fma_(y, fnma_(x, y, R(1.0f)), y);
    return round_up_ones(x, fma_(y1, fnma_(x, y1, R(1.0f)), y1));
}

}  // namespace lbm
