// Functions of one float.
#pragma once

// tanh without a branch, so that independent ones overlap (largest relative error 2.2e-7, of tanhf 1.9e-7): x from -0.55 to 0.55 by Lambert's continued
// fraction x / (1 + x^2 / (3 + x^2 / (5 + x^2 / (7 + x^2 / 9)))) as a quotient of polynomials, else 1 - 2 / (e^2|x| + 1).
__device__ __forceinline__ float tanh_select(float x) {
    const float y = x * x, a = fabsf(x), e = 2.f * a;
    const float small = x * __fdividef(fmaf(y, y + 105.f, 945.f), fmaf(y, fmaf(y, 15.f, 420.f), 945.f));
    const float large = 1.f - __fdividef(2.f, expf(e > 40.f ? 40.f : e) + 1.f);        // (a NaN stays one)
    return a < 0.55f ? small : copysignf(large, x);
}
