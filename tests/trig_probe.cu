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

// x, z: device memory of n and 2 n doubles; waits
extern "C" int probe_device(const double *x, double *z, int n)
{
    k_probe<<<(n + 255) / 256, 256>>>(x, reinterpret_cast<double2 *>(z), n);
    const cudaError_t e = cudaGetLastError();
    return (int)(e != cudaSuccess ? e : cudaDeviceSynchronize());
}
