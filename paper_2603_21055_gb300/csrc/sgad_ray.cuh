// Slope of a pixel's ray, for host and device code.
#pragma once

#include <cmath>

#ifdef __CUDACC__
#define SGAD_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define SGAD_HOST_DEVICE inline
#endif

namespace sgad {

// a / f, correctly rounded, from the rounded reciprocal inv_f of f: a quotient within two
// units in the last place, its exact remainder, and one correction (Markstein, "Computation of
// elementary functions on the IBM RISC System/6000 processor", IBM J. Res. Dev. 34(1), 1990).
// A division here, for every entry of every pixel block, costs the full-size backward 45 us of
// 1339.
SGAD_HOST_DEVICE float ray_slope(float a, float f, float inv_f)
{
    const float q = a * inv_f;
    return fmaf(fmaf(-q, f, a), inv_f, q);
}

}  // namespace sgad
