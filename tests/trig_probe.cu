// aaqaoa_trig.h on the host and on the device, for tests.
#include "aaqaoa_trig.h"

__global__ void k_probe(const double *x, double2 *z, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n)
        z[i] = aaq::phase_sincos(x[i]);
}

extern "C" void probe_host(const double *x, double *z, int n)
{
    for (int i = 0; i < n; i++) {
        const double2 v = aaq::phase_sincos(x[i]);
        z[2 * i] = v.x;
        z[2 * i + 1] = v.y;
    }
}

// a rotation of the type (float: is_float) from its (sine, cosine) parts u, v: t, f, f + fl
// and f^0..f^n by either way of building them
extern "C" void probe_mix(double u, double v, int is_float, int n, double *t, double *f, double *square, double *chain)
{
    aaq::MixFactor m;
    if (is_float)
        aaq::mix_ratio<float>(u, v, *t, m);
    else
        aaq::mix_ratio<double>(u, v, *t, m);
    f[0] = m.f;
    f[1] = m.fl;
    aaq::MixPower q;
    for (int k = 0; k <= n; k++) {
        square[k] = is_float ? aaq::mix_power<float>(m, k) : aaq::mix_power<double>(m, k);
        chain[k] = q.value();
        if (is_float)
            q.times<float>(m);
        else
            q.times<double>(m);
    }
}

// x, z: device memory of n and 2 n doubles; waits
extern "C" int probe_device(const double *x, double *z, int n)
{
    k_probe<<<(n + 255) / 256, 256>>>(x, reinterpret_cast<double2 *>(z), n);
    const cudaError_t e = cudaGetLastError();
    return (int)(e != cudaSuccess ? e : cudaDeviceSynchronize());
}
