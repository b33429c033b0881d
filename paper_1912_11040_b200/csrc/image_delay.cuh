// Distance of an image source, as rir.cu's kernel works it out (and a test on the CPU).
#pragma once
#include <math.h>

#ifdef __CUDACC__
#define AUG_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define AUG_HOST_DEVICE inline
#endif

// sqrt(d2), and e with r0 (1 + e / 2) = 1 / sqrt(d2) to e^2: the reciprocal square root's series around its fp32 value r0
// (|e| < 1e-6), up to the second order, fp64.  Right to a rounding or two; with the first order alone a delay of 24000
// samples is off by 1e-9.
AUG_HOST_DEVICE double image_distance(double d2, float r0, double &e) {
    const double t = d2 * (double)r0;
    e = fma(-t, (double)r0, 1.0);
    return fma(t * e, fma(0.375, e, 0.5), t);
}
