// Sine and cosine of the phase tables and mixer angles, and the factors that the
// mixer's rotations drop; the same on host and device.
#pragma once

#include <cmath>
#include <type_traits>

#include <cuda_runtime.h>

#ifdef __CUDACC__
#define AAQ_HD __host__ __device__ __forceinline__
#else
#define AAQ_HD inline
#endif

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

// The factor that one butterfly of a layer drops, in two parts f + fl (complex64:
// fl = 0), and its powers. f^n scales the whole state, so its error is the norm's:
// the powers of complex128 carry the product's rounding errors along and are right
// to one rounding (a plain product of n, or squarings, leave up to n of them: at
// n = 12..22 that was 0.2-0.4e-15 in energies and gradients, half their error).
struct MixFactor {
    double f, fl;
};
struct MixPower {  // f^k in two parts
    double hi = 1.0, lo = 0.0;
    template <typename R> AAQ_HD void times(const MixFactor &m)
    {
        const double p = hi * m.f;
        if constexpr (!std::is_same<R, float>::value)
            lo = fma(lo, m.f, fma(hi, m.fl, fma(hi, m.f, -p)));
        hi = p;
    }
    AAQ_HD double value() const { return hi + lo; }
};
template <typename R> AAQ_HD double mix_power(MixFactor q, int n)
{
    MixPower r;
    for (; n; n >>= 1) {
        if (n & 1)
            r.times<R>(q);
        const double s = q.f * q.f;
        if constexpr (!std::is_same<R, float>::value)
            q.fl = fma(2.0 * q.f, q.fl, fma(q.f, q.f, -s));
        q.f = s;
    }
    return r.value();
}

// The rotation of one mixer layer from (cos, sin) of its angle: u / v = t, the
// ratio the butterflies use (rounded to the amplitude type), and the factor one
// butterfly with that t drops: 1 / sqrt(1 + t^2) with v's sign, to first order in
// the rounding error t v - u. It and t belong together: with f = cos beta the norm
// drifts by the rounding of t in every butterfly.
template <typename R>
AAQ_HD void mix_ratio(double u, double v, double &t, MixFactor &m)
{
    m.fl = 0.0;
    if constexpr (std::is_same<R, float>::value)
        t = (double)((float)u / (float)v);
    else
        t = u / v;
    m.f = v - v * (u * fma(t, v, -u));
    if constexpr (!std::is_same<R, float>::value) {  // fl = f (1 - f^2 (1 + t^2)) / 2
        const double ff = m.f * m.f, fe = fma(m.f, m.f, -ff), tt = t * t, h = 1.0 + tt;
        const double he = (tt - (h - 1.0)) + fma(t, t, -tt), p = ff * h;
        m.fl = 0.5 * m.f * (((1.0 - p) - fma(ff, h, -p)) - fma(ff, he, fe * h));
    }
}

}  // namespace aaq
