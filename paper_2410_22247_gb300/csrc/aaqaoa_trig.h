// Sine and cosine of the phase tables and mixer angles, the same on host and device.
#pragma once

#include <cmath>
#include <cuda_runtime.h>

namespace aaq {

// (cos x, sin x) in FP64. Cody and Waite's reduction to r = x - k pi/2, |r| <= pi/4,
// with pi/2 in two parts, fused; the first step is exact, the second rounds once.
// Then Taylor's series to r^17 and r^16, whose next terms are below 2e-18 at pi/4.
// Rounding leaves either value within 2^-52 of the function's, up to |x| of 1.5e9;
// beyond, and for infinities and NaN, the library's function (which costs 3 us at
// the head of a launch; this is 26 operations in two chains).
#ifdef __CUDACC__
inline __host__ __device__ __noinline__
#else
inline
#endif
double2 phase_sincos(double x)
{
    const double k = rint(x * 0.63661977236758134308);
    if (!(fabs(k) < 1e9)) {
        double2 z;
        z.x = cos(x);
        z.y = sin(x);
        return z;
    }
    double r = fma(k, -1.5707963267948965580, x);
    r = fma(k, -6.1232339957367660359e-17, r);
    const double s = r * r;
    double ps = fma(s, 1.0 / 355687428096000.0, -1.0 / 1307674368000.0);
    double pc = fma(s, 1.0 / 20922789888000.0, -1.0 / 87178291200.0);
    ps = fma(ps, s, 1.0 / 6227020800.0);
    ps = fma(ps, s, -1.0 / 39916800.0);
    pc = fma(pc, s, 1.0 / 479001600.0);
    ps = fma(ps, s, 1.0 / 362880.0);
    pc = fma(pc, s, -1.0 / 3628800.0);
    ps = fma(ps, s, -1.0 / 5040.0);
    pc = fma(pc, s, 1.0 / 40320.0);
    ps = fma(ps, s, 1.0 / 120.0);
    pc = fma(pc, s, -1.0 / 720.0);
    ps = fma(ps, s, -1.0 / 6.0);
    pc = fma(pc, s, 1.0 / 24.0);
    pc = fma(pc, s, -0.5);
    const double sr = fma(r * s, ps, r), cr = fma(s, pc, 1.0);
    const int q = (int)(long long)k & 3;
    const double a = (q & 1) ? cr : sr, b = (q & 1) ? sr : cr;
    double2 z;
    z.x = ((q + 1) & 2) ? -b : b;
    z.y = (q & 2) ? -a : a;
    return z;
}

}  // namespace aaq
