// inv_sqrt.cuh -- the estimated inverse square root of the Green's function in
// FP32 spectra (greens.cu).
#pragma once
#include <math.h>

namespace isofft {

// 1 / sqrt(x): the float unit's estimate (about 2^-22) and one step of
// Householder's third-order iteration, w (1 + e/2 + 3 e^2/8) with e = 1 - x w^2
// (error e^3), in eight FP64 operations; the library call outside float range.
// Within one ulp and a little: half an ulp from the rounding of x w, half from
// the last sum.
static __device__ __forceinline__ double inv_sqrt(double x)
{
    if (!(x < 1e37 && x > 1e-37)) return rsqrt(x);
    const double w = (double)rsqrtf((float)x);
    const double e = fma(-x * w, w, 1.0);
    return fma(w * e, fma(0.375, e, 0.5), w);
}

}  // namespace isofft
