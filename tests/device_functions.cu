// Device functions of the library, one value per thread, for
// tests/test_gpu_device_functions.py.
#include <cuda_runtime.h>

#include "adg_tv_cell.cuh"

using namespace adg;

// theta of a gas at rest with rho = R = 1, gamma - 1 = 1/2 (T = p), and the same by pow
__global__ void k_theta(const double* p, double* out, int n, Phys P) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double q[4] = {1.0, 0.0, 0.0, 2.0 * p[i]};
    out[i] = theta_of(q, 0.0, P);
    out[n + i] = __dmul_rn(p[i], pow(__ddiv_rn(P.p0, p[i]), P.Rcp));
}

extern "C" int dev_theta(const double* p, double* out, int n, double p0, double Rcp) {
    Phys P = {};
    P.gm1 = 0.5;
    P.invR = 1.0;
    P.p0 = p0;
    P.inv_p0 = 1.0 / p0;
    P.Rcp = Rcp;
    k_theta<<<(n + 127) / 128, 128>>>(p, out, n, P);
    return (int)cudaDeviceSynchronize();
}
