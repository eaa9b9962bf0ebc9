// Scalars of a pair's recurrence: beta_{i+1}, and the estimated relative error of its running value
// S_k = e_1^T (I - T_k)^{-1} e_1.
#pragma once

#include <cuda_runtime.h>
#include <math.h>

namespace rd {

// root = sqrt(x) and inv = 1 / root by one rsqrt (366 cycles) with a Newton correction each, instead of a
// square root (610) and a division (365): the root within 0.53 units in its last place, its reciprocal
// rounded correctly. Zero, negative, denormal and non-finite x (told by the exponent bits): the plain
// forms, or a step that stops and uses neither (it is a breakdown when the root is 0).
__device__ __forceinline__ void root_and_inverse(double x, double* root, double* inv)
{
    const int hi = __double2hiint(x);
    if (hi >= 0x00200000 && hi < 0x7ff00000) {
        const double r = rsqrt(x);
        const double b = x * r;
        *root = fma(0.5 * r, fma(-b, b, x), b);
        *inv = fma(r, fma(-*root, r, 1.0), r);
    } else {
        *root = sqrt(fmax(x, 0.0));
        *inv = 1.0 / *root;
    }
}

// The increments still to come as a geometric series: i0 is the newest increment of S, i1 to i3 those before
// it; rho, the largest of the three ratios num/den of neighbours and at least 1/2, gives
// i0 rho / (1 - rho)^2 / S. rho is found by cross-multiplication and the estimate is one quotient,
// i0 num den / ((den - num)^2 S), since divisions are what the chain of a step is made of. Increments go
// on falling long after a run of fixed length has converged: below 2^-200 they are scaled by a power of
// two first, or the products and squares would lose digits and become 0/0.
__device__ __forceinline__ double tail_estimate(double i0, double i1, double i2, double i3, double S)
{
    double back = 1.0;
    int e = (__double2hiint(i1) >> 20) & 0x7ff;
    if (e < 1023 - 200) {
        e = e > 1 ? e : 1;
        const double f = __hiloint2double((2046 - e) << 20, 0);  // 2^(1023 - e)
        back = __hiloint2double(e << 20, 0);                     // 2^(e - 1023)
        i0 *= f;
        i1 *= f;
        i2 *= f;
        i3 *= f;
    }
    double bn = i0, bd = i1;
    if (i1 * bd > bn * i2) {
        bn = i1;
        bd = i2;
    }
    if (i2 * bd > bn * i3) {
        bn = i2;
        bd = i3;
    }
    if (bn + bn <= bd) {  // rho at its floor 1/2
        bn = 1.0;
        bd = 2.0;
    }
    const double gap = bd - bn;
    return bn < bd ? i0 * bn * bd / (gap * gap * S) * back : INFINITY;
}

}  // namespace rd
