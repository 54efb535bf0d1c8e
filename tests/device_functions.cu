// Device functions of the library, one value per thread, for
// tests/test_gpu_device_functions.py.
#include <cuda_runtime.h>

#include "adg_mixed_point.cuh"
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

// rho u v of the 3D mixed flux with rho u = rho v = 1 and no viscosity: 1/rho
__global__ void k_flux3_rcp(const float* rho, float* out, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const Phys3f P = {};
    const float q[5] = {rho[i], 1.0f, 1.0f, 0.0f, 0.0f};
    const float g[3][5] = {};
    out[i] = ns_flux9_pert(q, g, 0.0f, 0.0f, 0.0f, 0.0f, P).t[1];
}

extern "C" int dev_flux3_rcp(const float* rho, float* out, int n) {
    k_flux3_rcp<<<(n + 127) / 128, 128>>>(rho, out, n);
    return (int)cudaDeviceSynchronize();
}

// adg_fixed.cuh: reciprocal; fixed point from a double and its limbs; double from fixed point
__global__ void k_rcp(const double* x, double* out, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = fx_rcp(x[i]);
}
__global__ void k_from(const double* x, const int* E, long long* m, int* limbs, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    m[i] = fx_from(x[i], E[i]);
    const Limbs a = fx_split(m[i]), b = fx_split_centred(m[i]);
    limbs[4 * i] = a.h;
    limbs[4 * i + 1] = a.l;
    limbs[4 * i + 2] = b.h;
    limbs[4 * i + 3] = b.l;
}
__global__ void k_to(const long long* a, const int* e, double* out, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = fx_to(a[i], e[i]);
}

extern "C" int dev_rcp(const double* x, double* out, int n) {
    k_rcp<<<(n + 127) / 128, 128>>>(x, out, n);
    return (int)cudaDeviceSynchronize();
}
extern "C" int dev_from(const double* x, const int* E, long long* m, int* limbs, int n) {
    k_from<<<(n + 127) / 128, 128>>>(x, E, m, limbs, n);
    return (int)cudaDeviceSynchronize();
}
extern "C" int dev_to(const long long* a, const int* e, double* out, int n) {
    k_to<<<(n + 127) / 128, 128>>>(a, e, out, n);
    return (int)cudaDeviceSynchronize();
}
