// Three-dimensional FP64 ADER-DG (the ABC flow of Sec. 4.1 and the 3D cosine
// bubble of Sec. 4.2): the scheme of adg_fp64.cu with one more direction.
//
// Predictor (Sec. 3): per cell, the element-local space-time polynomial on
// (N+1)^4 Gauss-Legendre nodes by n = N+1 Picard sweeps
//     q_l = u + dt sum_k (K1^{-1})_{lk} w_k R_k,  R = -dF/dx - dG/dy - dH/dz + S,
// then grad q, F, G, H, S once more on the final iterate, averaged in time.
// It writes the weak volume residual
//     rvol = sum_d (1/h_d) sum_p (w_p / w_i_d) D_p,i_d Fbar_d(.. p ..) + Sbar
// and, per face node, the boundary-extrapolated averages (q-bar, normal
// flux, grad q-bar) and the Rusanov speed.
// Corrector: the Rusanov-type viscous flux on the 6 faces (neighbour traces,
// a slip-wall ghost with the background of Eq. 6 and the heat flux of
// Eq. 10, or the analytic ABC field) and the FP64 update u += dt (rvol - lift).
//
// Thread mapping: the FP64 predictor runs one thread per space-time node (see
// there); the mixed predictor and the corrector CPB cells per block, one thread
// per spatial node (l, j, i).  A thread of the mixed predictor walks the n time
// nodes of its node, so the Picard update's time contraction stays in
// registers; its shared memory holds per cell the n time slices of the iterate
// and the fluxes of one time slice (the divergence of slice k is taken before
// slice k+1's fluxes overwrite them), after the last sweep the averaged fields
// the volume term and the traces contract.  (One thread per space-time node,
// scalar or with two slices packed, was measured for it too: 201 and 240 us
// a step of the 25^3 degree-2 bubble against 200 before the nine-flux form.)
//
// Layouts: u[c][v][l][j][i], c = (iz ny + iy) nx + ix, v in (rho, rho u,
// rho v, rho w, rho E); traces [c][face E W N S T B][kTr3][n^2], face nodes
// (l, j) on x-faces, (l, i) on y-faces, (j, i) on z-faces.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>
#include <vector>

#include "adg_convert.cuh"
#include "adg_fixed.cuh"
#include "adg_internal.h"
#include "adg_mesh.h"
#include "adg_mixed_point.cuh"

namespace adg {
namespace {

constexpr int kTr3 = 26;  // q-bar(5), normal flux(5), qx-bar(5), qy-bar(5), qz-bar(5), speed

struct Phys3 {
    double gamma, gm1, R, invR, mu, kappa, g, cp, p0, theta0, lamv, dTdz;
    double eta[3], h[3], inv_h[3], org[3];
    int nc[3], bc[3];
    int gravity, field;
};

// background p, rho at node heights [nz][n] and at horizontal faces [nz + 1]
struct Bg3 {
    const double* pn;
    const double* rn;
    const double* pf;
    const double* rf;
};

// Point-wise fluxes f[b][v] in the three directions and the z-momentum
// source of a state q with gradients g[b][v] at height z.  Momentum fluxes
// carry p' = p - pbar (Eq. 7); heat_wall replaces grad T by (0, 0, dTbar/dz)
// (slip-wall ghost, Eq. 10).
__device__ __forceinline__ void ns_flux3(const double q[5], const double g[3][5], double z, double pbar,
                                         double rhobar, const Phys3& P, bool heat_wall, double f[3][5],
                                         double& src) {
    const double rinv = 1.0 / q[0];
    const double vel[3] = {q[1] * rinv, q[2] * rinv, q[3] * rinv};
    const double kin = 0.5 * (vel[0] * vel[0] + vel[1] * vel[1] + vel[2] * vel[2]);
    const double gg = P.gravity ? P.g : 0.0;
    const double p = P.gm1 * (q[4] - q[0] * kin - q[0] * gg * z);
    const double pp = p - pbar;
    const double T = p * rinv * P.invR;
    double d[3][3];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) d[a][b] = (g[b][1 + a] - vel[a] * g[b][0]) * rinv;
    const double div = d[0][0] + d[1][1] + d[2][2];
    double dT[3];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        if (heat_wall) {
            dT[b] = b == 2 ? P.dTdz : 0.0;
        } else {
            double s = g[b][4] - (vel[0] * g[b][1] + vel[1] * g[b][2] + vel[2] * g[b][3]) + kin * g[b][0] -
                       gg * z * g[b][0];
            if (b == 2) s -= q[0] * gg;
            dT[b] = (P.gm1 * s - P.R * T * g[b][0]) * rinv * P.invR;
        }
    }
    double sig[3][3];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b)
            sig[a][b] = P.mu * ((a == b ? (2.0 / 3.0) * div : 0.0) - (d[a][b] + d[b][a]));
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        f[b][0] = q[1 + b];
#pragma unroll
        for (int a = 0; a < 3; ++a) f[b][1 + a] = q[1 + a] * vel[b] + (a == b ? pp : 0.0) + sig[a][b];
        f[b][4] = vel[b] * (q[4] + p) + vel[0] * sig[0][b] + vel[1] * sig[1][b] + vel[2] * sig[2][b] -
                  P.kappa * dT[b];
    }
    src = P.gravity ? -P.g * (q[0] - rhobar) : 0.0;
}

// Rusanov speed |v_dir| + c + 2 eta_dir lambda_v / rho at height z
__device__ __forceinline__ double wave_speed3(const double q[5], double z, int dir, const Phys3& P) {
    const double rinv = fx_rcp(q[0]);
    const double gg = P.gravity ? P.g : 0.0;
    const double p = P.gm1 * (q[4] - 0.5 * (q[1] * q[1] + q[2] * q[2] + q[3] * q[3]) * rinv - q[0] * gg * z);
    const double mn = dir == 0 ? q[1] : dir == 1 ? q[2] : q[3];  // selects keep q in registers
    return fabs(mn * rinv) + sqrt(P.gamma * p * rinv) + 2.0 * P.eta[dir] * P.lamv * rinv;
}

__device__ __forceinline__ void rusanov5(const double qL[5], const double fL[5], double sL, const double qR[5],
                                         const double fR[5], double sR, double out[5]) {
    const double s = fmax(sL, sR);
#pragma unroll
    for (int v = 0; v < 5; ++v) out[v] = 0.5 * (fL[v] + fR[v]) - 0.5 * s * (qR[v] - qL[v]);
}

// The ABC field (Sec. 4.1) and its gradient, differentiated by hand:
// a = e^{-mu t}, u = a (sin z + cos y), v = a (sin x + cos z),
// w = a (sin y + cos x), rho = 1, p = -a^2 (cos x sin y + sin x cos z +
// sin z cos y) + 100/gamma.
__device__ __forceinline__ void abc_field(double x, double y, double z, double t, const Phys3& P, double q[5],
                                          double g[3][5]) {
    const double a = exp(-P.mu * t), a2 = a * a;
    const double sx = sin(x), cx = cos(x), sy = sin(y), cy = cos(y), sz = sin(z), cz = cos(z);
    const double vel[3] = {a * (sz + cy), a * (sx + cz), a * (sy + cx)};
    // dvel[a][b] = d vel_a / d x_b
    const double dv[3][3] = {{0.0, -a * sy, a * cz}, {a * cx, 0.0, -a * sz}, {-a * sx, a * cy, 0.0}};
    const double p = -a2 * (cx * sy + sx * cz + sz * cy) + 100.0 / P.gamma;
    const double dp[3] = {-a2 * (-sx * sy + cx * cz), -a2 * (cx * cy - sz * sy), -a2 * (-sx * sz + cz * cy)};
    q[0] = 1.0;
    q[1] = vel[0];
    q[2] = vel[1];
    q[3] = vel[2];
    q[4] = p / P.gm1 + 0.5 * (vel[0] * vel[0] + vel[1] * vel[1] + vel[2] * vel[2]);
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        g[b][0] = 0.0;
        g[b][1] = dv[0][b];
        g[b][2] = dv[1][b];
        g[b][3] = dv[2][b];
        g[b][4] = dp[b] / P.gm1 + vel[0] * dv[0][b] + vel[1] * dv[1][b] + vel[2] * dv[2][b];
    }
}


template <int N>
struct Cfg3 {
    static constexpr int n = N + 1, n2 = n * n, n3 = n * n * n;
    static constexpr int cpb = N == 1 ? 16 : N == 2 ? 8 : N == 3 ? 4 : 2;
    static constexpr int threads = cpb * n3;
};

// FP64 predictor: the scheme of the 2D one (adg_fp64_body.cuh) -- one thread
// per space-time node (k, l, j, i), every contraction on the integer pipe in
// 58-bit block-scaled fixed point (adg_fixed.cuh), the point-wise fluxes alone
// in FP64.
template <int N>
struct Fx3Cfg {
    static constexpr int n = N + 1, n2 = n * n, n3 = n2 * n, n4 = n3 * n;
    // degree 2 (81 threads a cell) lets cells share warps: 96 would idle 16% of
    // the FP64 lanes; elsewhere whole warps (degree 1: half warps) per cell
    static constexpr int tpc = N == 2 ? 81 : N == 4 ? 640 : n4;
    static constexpr int cpb = N == 1 ? 8 : N == 2 ? 3 : 1;
    static constexpr int threads = (cpb * tpc + 31) / 32 * 32;
    // blocks per SM asked of the register allocator; us a step at 3 / 4 / 5 / 6: degree 1 (41^3 cells)
    // 1121 / 1155 / 1153 / 1167, 2 (25^3) 1327 / 1299 / 1274 / 1322, 3 (17^3) 1328 / 1374 / 1308 / 1352;
    // degree 4 (13^3) 2158 with 1 or 2, 2415 with 3
    static constexpr int resident = N == 1 ? 3 : N == 4 ? 1 : 5;
    // per cell, in 8-byte words: q (5) and the fluxes (9) of every space-time
    // node, u, D/h, the face values of q-bar, the magnitudes
    static constexpr int words = 14 * n4 + 5 * n3 + 3 * n2 + 30 * n2 + 8;
    static constexpr size_t smem = ((size_t)cpb * words + n2) * 8;
};

// Point-wise fluxes (Eqs. 1-5, 7) in 78 FP64 operations: the mass fluxes are
// the momenta; t: xx, xy, xz, yy, yz, zz of the symmetric momentum flux; e:
// energy flux; with w_ab = d_b(rho v_a) - v_a d_b(rho),
//   c_v rho d_b T = d_b E - (E/rho) d_b rho - v.w_b - rho g (b = z).
struct Fx3Flux {
    double t[6], e[3];
};
__device__ __forceinline__ Fx3Flux ns_flux9(const double q[5], const double g[3][5], double gg, double gz, double pbar,
                                            double gm1, double mu, double mu23, double kR) {
    const double rinv = fx_rcp(q[0]);
    const double v[3] = {q[1] * rinv, q[2] * rinv, q[3] * rinv};
    const double ke2 = fma(q[3], v[2], fma(q[2], v[1], q[1] * v[0]));
    const double p = gm1 * fma(-0.5, ke2, fma(-gz, q[0], q[4]));
    const double pp = p - pbar, Ep = q[4] + p, eR = q[4] * rinv;
    double w[3][3];  // w[a][b], rho times the velocity gradient
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) w[a][b] = fma(-v[a], g[b][0], g[b][1 + a]);
    const double m23 = mu23 * rinv, mr = -mu * rinv, kr = kR * rinv;
    const double div = w[0][0] + w[1][1] + w[2][2];
    const double sd[3] = {m23 * fma(-3.0, w[0][0], div), m23 * fma(-3.0, w[1][1], div), m23 * fma(-3.0, w[2][2], div)};
    const double sxy = mr * (w[0][1] + w[1][0]), sxz = mr * (w[0][2] + w[2][0]), syz = mr * (w[1][2] + w[2][1]);
    Fx3Flux f;
    f.t[0] = fma(q[1], v[0], pp + sd[0]);
    f.t[1] = fma(q[1], v[1], sxy);
    f.t[2] = fma(q[1], v[2], sxz);
    f.t[3] = fma(q[2], v[1], pp + sd[1]);
    f.t[4] = fma(q[2], v[2], syz);
    f.t[5] = fma(q[3], v[2], pp + sd[2]);
    const double so[3][2] = {{sxy, sxz}, {sxy, syz}, {sxz, syz}};
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        double h = fma(-v[2], w[2][b], fma(-v[1], w[1][b], fma(-v[0], w[0][b], fma(-eR, g[b][0], g[b][4]))));
        if (b == 2) h = fma(-gg, q[0], h);
        f.e[b] = fma(-kr, h, fma(v[b], Ep + sd[b], fma(v[b == 0 ? 1 : 0], so[b][0], v[b == 2 ? 1 : 2] * so[b][1])));
    }
    return f;
}

// slot of the momentum flux (a, b) among the six; slot of component c of a face
// record in direction dir (q, then the normal flux) among q (5), t (6), e (3)
__device__ __forceinline__ int fx3_t(int a, int b) { return a + b + (a > 0 && b > 0 ? 1 : 0); }
__device__ __forceinline__ int fx3_slot(int c, int dir) {
    return c < 5 ? c : c == 5 ? 1 + dir : c < 9 ? 5 + fx3_t(c - 6, dir) : 11 + dir;
}

template <int N>
__global__ void __launch_bounds__(Fx3Cfg<N>::threads, Fx3Cfg<N>::resident)
k3_predictor(const double* __restrict__ u, double* __restrict__ rvol, double* __restrict__ trace, int cells,
             double dt, const Basis B, const Phys3 P, const Bg3 bg) {
    using C = Fx3Cfg<N>;
    constexpr int n = C::n, n2 = C::n2, n3 = C::n3, n4 = C::n4, SL = 5 * n3;
    extern __shared__ double sm[];
    const int cl = min((int)threadIdx.x / C::tpc, C::cpb - 1);
    const int tid = threadIdx.x - cl * C::tpc;
    const bool on = tid < n4;  // the rest repeats the last node without stores
    const int id = on ? tid : n4 - 1;
    const int k = id / n3, node = id - k * n3, l = node / n2, j = (node / n) % n, i = node % n;
    double* base = sm + (size_t)cl * C::words;
    Limbs* Q = reinterpret_cast<Limbs*>(base);  // [5][n][n3]; the residual between the sweeps' halves
    Limbs* F = Q + 5 * n4;                      // [9][n][n3]
    double* US = base + 14 * n4;                // [5][n3]
    Limbs* DT = reinterpret_cast<Limbs*>(US + 5 * n3);  // [3][n][n]
    double* TQ = US + 5 * n3 + 3 * n2;          // [6][5][n2]
    uint32_t* mx = reinterpret_cast<uint32_t*>(TQ + 30 * n2);  // magnitudes: q (5), fluxes (9), the source
    Limbs* K = reinterpret_cast<Limbs*>(sm + (size_t)C::cpb * C::words);
    for (int a = threadIdx.x; a < n2; a += blockDim.x) K[a] = Limbs{B.KwH[a / n][a % n], B.KwL[a / n][a % n]};
    int ed[3], sh[3];  // of each direction's entries (FxRows of the 2D predictor)
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        ed[b] = fx_exp(fx_mag(B.Dmax * P.inv_h[b]));
        sh[b] = fx_row_shift(B.Drow * P.inv_h[b], ed[b]);
    }
    for (int a = tid; a < 3 * n2; a += C::tpc)
        if (on) {
            const int b = a / n2;
            DT[a] = fx_split_centred(fx_from(B.D[a % n2 / n][a % n] * P.inv_h[b], b == 0 ? ed[0] : b == 1 ? ed[1] : ed[2]));
        }
    const double gg = P.gravity ? P.g : 0.0, mu23 = (2.0 / 3.0) * P.mu, kR = P.gm1 * P.kappa * P.invR;

    // largest magnitude of a group over the cell's threads: a warp reduction and
    // one shared-memory atomic per warp and cell in it
    auto push = [&](int slot, uint32_t m) {
        if constexpr (C::tpc % 32 == 0) {
            m = __reduce_max_sync(0xffffffffu, m);
            if ((threadIdx.x & 31) == 0) atomicMax(mx + slot, m);
        } else if constexpr (C::tpc < 32) {
#pragma unroll
            for (int o = 1; o < C::tpc; o *= 2) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
            if (tid == 0) mx[slot] = max(mx[slot], m);
        } else {  // at most two cells in a warp
            const int first = __shfl_sync(0xffffffffu, cl, 0);
            const uint32_t a = __reduce_max_sync(0xffffffffu, cl == first ? m : 0u);
            const uint32_t b = __reduce_max_sync(0xffffffffu, cl == first ? 0u : m);
            if ((threadIdx.x & 31) == 0) atomicMax(mx + slot, a);
            if ((threadIdx.x & 31) == 31 && cl != first) atomicMax(mx + slot, b);
        }
    };
    const Limbs *Dx = DT + i * n, *Dy = DT + n2 + j * n, *Dz = DT + 2 * n2 + l * n;
    const int ox = (l * n + j) * n, oy = l * n2 + i, oz = j * n + i;  // lines through the node: strides 1, n, n2

#pragma unroll 1
    for (int c0 = blockIdx.x * C::cpb; c0 < cells; c0 += gridDim.x * C::cpb) {
        const bool active = c0 + cl < cells;
        const int cell = active ? c0 + cl : cells - 1;
        const int ic0 = cell % P.nc[0], ic1 = (cell / P.nc[0]) % P.nc[1], iz = cell / (P.nc[0] * P.nc[1]);
        const double gz = gg * (P.org[2] + (iz + B.xi[l]) * P.h[2]);
        const double pbar = bg.pn[iz * n + l], rhobar = bg.rn[iz * n + l];
        double q[5];
#pragma unroll
        for (int v = 0; v < 5; ++v) q[v] = u[(size_t)cell * SL + v * n3 + node];
        // exponents of q (slots 0..4) and the fluxes (5..13); a phase's magnitudes are cleared in the phase after the
        // next barrier
        int E[14] = {};
        auto take = [&](int first, int end) {
#pragma unroll
            for (int c = first; c < end; ++c) E[c] = fx_exp(mx[c]);
        };
        auto push_q = [&]() {
#pragma unroll
            for (int v = 0; v < 5; ++v) push(v, fx_mag(q[v]));
        };
        auto store_q = [&](int slice) {
#pragma unroll
            for (int v = 0; v < 5; ++v) Q[(v * n + slice) * n3 + node] = fx_limbs(q[v], E[v]);
        };
        if (tid < 15) mx[tid] = 0;
        __syncthreads();
        push_q();
        __syncthreads();
        take(0, 5);
        if (id < n3 && on) {
            store_q(0);
#pragma unroll
            for (int v = 0; v < 5; ++v) US[v * n3 + node] = q[v];
        }
        __syncthreads();

        Fx3Flux f;
        // sweeps 0..n-1 and the final evaluation r = n; in sweep 0 the iterate is
        // u at every time node: the threads of time node 0 evaluate the fluxes
#pragma unroll 1
        for (int r = 0;; ++r) {
            const int ks = r == 0 ? 0 : k;
            const Limbs* Qk = Q + ks * n3;
            int ER[5];  // exponents of the residual: the largest of its derivatives' and the source's
            ER[0] = max(E[1] + ed[0] + sh[0], max(E[2] + ed[1] + sh[1], E[3] + ed[2] + sh[2])) - 1022;
            long long R[5];  // -div F + S; the mass flux is the momentum
            R[0] = 0;
#pragma unroll
            for (int a = 0; a < 6; ++a) f.t[a] = 0.0;
            f.e[0] = f.e[1] = f.e[2] = 0.0;
            if (r == 0 && k > 0) {
#pragma unroll
                for (int b = 0; b < 3; ++b) {
                    const Limbs* D = b == 0 ? Dx : b == 1 ? Dy : Dz;
                    const Limbs* L = Qk + (1 + b) * n4 + (b == 0 ? ox : b == 1 ? oy : oz);
                    FxSum a;
#pragma unroll
                    for (int p = 0; p < n; ++p) a.add(D[p], L[p * (b == 0 ? 1 : b == 1 ? n : n2)]);
                    R[0] -= a.value() >> fx_down(sh[b], ER[0], E[1 + b] + ed[b] + sh[b] - 1022);
                }
            } else {
                double g[3][5];
#pragma unroll
                for (int b = 0; b < 3; ++b) {
                    const Limbs* D = b == 0 ? Dx : b == 1 ? Dy : Dz;
                    const Limbs* L = Qk + (b == 0 ? ox : b == 1 ? oy : oz);
                    FxSum a[5];
#pragma unroll
                    for (int p = 0; p < n; ++p) {
                        const Limbs d = D[p];
#pragma unroll
                        for (int v = 0; v < 5; ++v) a[v].add(d, L[v * n4 + p * (b == 0 ? 1 : b == 1 ? n : n2)]);
                    }
                    R[0] -= a[1 + b].value() >> fx_down(sh[b], ER[0], E[1 + b] + ed[b] + sh[b] - 1022);
#pragma unroll
                    for (int v = 0; v < 5; ++v) g[b][v] = fx_to(a[v].value(), E[v] + ed[b] - 2102);
                }
                f = ns_flux9(q, g, gg, gz, pbar, P.gm1, P.mu, mu23, kR);
            }
            if (r == n) break;
            const double S = P.gravity ? -gg * (q[0] - rhobar) : 0.0;
            const double fl[9] = {f.t[0], f.t[1], f.t[2], f.t[3], f.t[4], f.t[5], f.e[0], f.e[1], f.e[2]};
#pragma unroll
            for (int c = 0; c < 9; ++c) push(5 + c, fx_mag(fl[c]));
            if (P.gravity) push(14, fx_mag(S));
            __syncthreads();
            take(5, 14);
            if (tid < 5) mx[tid] = 0;
            if (on && (r > 0 || k == 0)) {
#pragma unroll
                for (int c = 0; c < 9; ++c) F[(c * n + k) * n3 + node] = fx_limbs(fl[c], E[5 + c]);
            }
            __syncthreads();
            // residual, in Q's place; component v's flux in direction b
            auto fc = [](int v, int b) { return v < 4 ? fx3_t(v - 1, b) : 6 + b; };
#pragma unroll
            for (int v = 1; v < 5; ++v) {
                ER[v] = v == 3 && P.gravity ? fx_exp(mx[14]) + 1 : 0;
#pragma unroll
                for (int b = 0; b < 3; ++b) ER[v] = max(ER[v], E[5 + fc(v, b)] + ed[b] + sh[b] - 1022);
                R[v] = 0;
            }
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                const Limbs* D = b == 0 ? Dx : b == 1 ? Dy : Dz;
                const Limbs* L = F + ks * n3 + (b == 0 ? ox : b == 1 ? oy : oz);
                FxSum a[4];
#pragma unroll
                for (int p = 0; p < n; ++p) {
                    const Limbs d = D[p];
#pragma unroll
                    for (int v = 1; v < 5; ++v) a[v - 1].add(d, L[fc(v, b) * n4 + p * (b == 0 ? 1 : b == 1 ? n : n2)]);
                }
#pragma unroll
                for (int v = 1; v < 5; ++v)
                    R[v] -= a[v - 1].value() >> fx_down(sh[b], ER[v], E[5 + fc(v, b)] + ed[b] + sh[b] - 1022);
            }
            if (P.gravity) R[3] += fx_from(S, ER[3]);
            if (on) {
#pragma unroll
                for (int v = 0; v < 5; ++v) Q[(v * n + k) * n3 + node] = fx_split(R[v]);
            }
            __syncthreads();
            {  // time contraction: this thread's time node of the next iterate
                FxSum a[5];
#pragma unroll
                for (int kk = 0; kk < n; ++kk) {
                    const Limbs d = K[k * n + kk];
#pragma unroll
                    for (int v = 0; v < 5; ++v) a[v].add(d, Q[(v * n + kk) * n3 + node]);
                }
#pragma unroll
                for (int v = 0; v < 5; ++v)
                    q[v] = fma(dt, fx_to(a[v].value(), ER[v] + B.KwE - 2102), US[v * n3 + node]);
            }
            push_q();
            __syncthreads();
            take(0, 5);
            if (tid < 10) mx[5 + tid] = 0;
            if (on) store_q(k);
            __syncthreads();
        }

        // time averages: slots q (5), t (6), e (3)
        double* A = base;
        __syncthreads();
        if (on) {
            double* Ak = A + k * n3 + node;
#pragma unroll
            for (int v = 0; v < 5; ++v) Ak[v * n4] = q[v];
#pragma unroll
            for (int a = 0; a < 6; ++a) Ak[(5 + a) * n4] = f.t[a];
#pragma unroll
            for (int a = 0; a < 3; ++a) Ak[(11 + a) * n4] = f.e[a];
        }
        __syncthreads();
        if (on)
            for (int s = k; s < 14; s += n) {
                double a = 0.0;
#pragma unroll
                for (int kk = 0; kk < n; ++kk) a = fma(B.w[kk], A[s * n4 + kk * n3 + node], a);
                A[s * n4 + node] = a;  // time node 0's place, read by this thread alone
            }
        __syncthreads();
        if (on && active) {
            for (int v = k; v < 5; v += n) {
                const double* Fv = A + fx3_slot(5 + v, 0) * n4 + ox;
                const double* Gv = A + fx3_slot(5 + v, 1) * n4 + oy;
                const double* Hv = A + fx3_slot(5 + v, 2) * n4 + oz;
                double sx = 0.0, sy = 0.0, sz = 0.0;
#pragma unroll
                for (int p = 0; p < n; ++p) {
                    sx = fma(B.Vx[p][i], Fv[p], sx);
                    sy = fma(B.Vx[p][j], Gv[p * n], sy);
                    sz = fma(B.Vx[p][l], Hv[p * n2], sz);
                }
                const double S = P.gravity && v == 3 ? -gg * (A[node] - rhobar) : 0.0;
                rvol[(size_t)cell * SL + v * n3 + node] = fma(sx, P.inv_h[0], fma(sy, P.inv_h[1], fma(sz, P.inv_h[2], S)));
            }
        }
        // boundary-extrapolated traces of faces E, W (x), N, S (y), T, B (z)
        auto face_at = [](int dir, int a, int b, int p) {
            return dir == 0 ? (a * n + b) * n + p : dir == 1 ? (a * n + p) * n + b : (p * n + a) * n + b;
        };
        double* tr = trace + (size_t)cell * 6 * kTr3 * n2;
        if (on)
            for (int o = tid; o < 60 * n2; o += n4) {
                const int m = o % n2, c = o / n2 % 10, fc = o / (10 * n2), dir = fc >> 1;
                const double* phi = (fc & 1) ? B.phi0 : B.phi1;
                const double* S = A + fx3_slot(c, dir) * n4;
                double s = 0.0;
#pragma unroll
                for (int p = 0; p < n; ++p) s = fma(phi[p], S[face_at(dir, m / n, m % n, p)], s);
                if (c < 5) TQ[(fc * 5 + c) * n2 + m] = s;
                if (active) tr[(fc * kTr3 + c) * n2 + m] = s;
            }
        __syncthreads();
        // Rusanov speed; grad q-bar on slip walls, which alone read it: along the
        // normal from the cell's nodes, along the face from the face's own values
        if (on)
            for (int o = tid; o < 6 * n2; o += n4) {
                const int fc = o / n2, m = o - fc * n2, dir = fc >> 1, a = m / n, b = m - a * n;
                double rec[5];
#pragma unroll
                for (int v = 0; v < 5; ++v) rec[v] = TQ[(fc * 5 + v) * n2 + m];
                const double zf = dir < 2 ? P.org[2] + (iz + B.xi[a]) * P.h[2] : P.org[2] + (iz + ((fc & 1) ? 0 : 1)) * P.h[2];
                if (active) tr[(fc * kTr3 + 25) * n2 + m] = wave_speed3(rec, zf, dir, P);
                const int icd = dir == 0 ? ic0 : dir == 1 ? ic1 : iz;
                const int ncd = dir == 0 ? P.nc[0] : dir == 1 ? P.nc[1] : P.nc[2];
                const int bcd = dir == 0 ? P.bc[0] : dir == 1 ? P.bc[1] : P.bc[2];
                if (!(active && bcd == ADG_BC_WALL && ((fc & 1) ? icd == 0 : icd == ncd - 1))) continue;
                const double* dphi = (fc & 1) ? B.dphi0 : B.dphi1;
                for (int v = 0; v < 5; ++v) {
                    const double* T = TQ + (fc * 5 + v) * n2;
                    double sn = 0.0, sa = 0.0, sb = 0.0;  // normal, along the face's first and second index
#pragma unroll
                    for (int p = 0; p < n; ++p) {
                        sn = fma(dphi[p], A[v * n4 + face_at(dir, a, b, p)], sn);
                        sa = fma(B.D[a][p], T[p * n + b], sa);
                        sb = fma(B.D[b][p], T[a * n + p], sb);
                    }
                    const double gx = dir == 0 ? sn : sb, gy = dir == 1 ? sn : dir == 0 ? sb : sa, gz3 = dir == 2 ? sn : sa;
                    double* tw = tr + (fc * kTr3 + 10 + v) * n2 + m;
                    tw[0] = gx * P.inv_h[0];
                    tw[5 * n2] = gy * P.inv_h[1];
                    tw[10 * n2] = gz3 * P.inv_h[2];
                }
            }
    }
    pdl_trigger();
}

struct Bg3m {
    const double* rb;   // [nz][n] rhobar at nodes (FP64, for the split)
    const double* Eb;   // [nz][n] Ebar = pbar/(gamma-1) + rhobar g z
    const float* rbf;   // [nz][n] rhobar
    const float* pbf;   // [nz][n] pbar
    const float* Hbf;   // [nz][n] Ebar + pbar
    const float* dzr;   // [nz][n] d rhobar/dz of the nodal interpolant
    const float* dzE;   // [nz][n] d Ebar/dz
    const double* ext;  // [nz][2: top, bottom][2: rhobar, Ebar] extrapolated to the z-faces
    const double* zn;   // [nz][n] node heights
    const float* zext;  // [nz][2: top, bottom][2: rhobar, pbar_eff] of the extrapolated z-face base,
                        // pbar_eff = (gamma-1)(Ebar - rhobar g z_face) formed in FP64
};

__device__ __forceinline__ void ns_flux3f(const float q[5], const float g[3][5], float gz, float rb, float pb,
                                          float Hb, const Phys3f& P, float f[3][5], float& src,
                                          bool heat_wall = false, float dTdz = 0.0f) {
    const float rho = rb + q[0];
    const float rinv = __frcp_rn(rho);
    const float vel[3] = {q[1] * rinv, q[2] * rinv, q[3] * rinv};
    const float kin = 0.5f * (vel[0] * vel[0] + vel[1] * vel[1] + vel[2] * vel[2]);
    const float pp = P.gm1 * (q[4] - rho * kin - gz * q[0]);
    const float T = (pb + pp) * rinv * P.invR;
    float d[3][3];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) d[a][b] = (g[b][1 + a] - vel[a] * g[b][0]) * rinv;
    const float div = d[0][0] + d[1][1] + d[2][2];
    float dT[3];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        float s = g[b][4] - (vel[0] * g[b][1] + vel[1] * g[b][2] + vel[2] * g[b][3]) + kin * g[b][0] - gz * g[b][0];
        if (b == 2) s -= rho * P.g;
        dT[b] = heat_wall ? (b == 2 ? dTdz : 0.0f) : (P.gm1 * s - P.R * T * g[b][0]) * rinv * P.invR;
    }
    float sig[3][3];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b)
            sig[a][b] = P.mu * ((a == b ? (2.0f / 3.0f) * div : 0.0f) - (d[a][b] + d[b][a]));
    const float h = Hb + (q[4] + pp);
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        f[b][0] = q[1 + b];
#pragma unroll
        for (int a = 0; a < 3; ++a) f[b][1 + a] = q[1 + a] * vel[b] + (a == b ? pp : 0.0f) + sig[a][b];
        f[b][4] = vel[b] * h + vel[0] * sig[0][b] + vel[1] * sig[1][b] + vel[2] * sig[2][b] - P.kappa * dT[b];
    }
    src = P.gravity ? -P.g * q[0] : 0.0f;
}

// MX: the mixed-precision form -- Rusanov flux from the FP64 jump of the
// face states converted to FP32, flux average and lifting in FP32, the
// update in FP64 (ghost states stay FP64).
// MINB: blocks per SM asked of the register allocator (launch3).
template <int N, bool MX, int MINB>
__global__ void __launch_bounds__(Cfg3<N>::threads, MINB)
k3_corrector(double* __restrict__ u, const double* rvol_in, const double* trace_in, int cells, double dt, double t,
              const Basis B, const Phys3 P, const Bg3 bg, const Phys3f Pf) {
    using C = Cfg3<N>;
    using FT = typename std::conditional<MX, float, double>::type;
    constexpr int n = C::n, n2 = C::n2, n3 = C::n3, SL = 5 * n3, TR = kTr3 * n2;
    __shared__ FT Fst[C::cpb][6][5][n2];
    const int cl = threadIdx.x / n3;
    const int node = threadIdx.x - cl * n3;
    const int l = node / n2, j = (node / n) % n, i = node % n;
    const int cell_raw = blockIdx.x * C::cpb + cl;
    const bool active = cell_raw < cells;
    const int cell = active ? cell_raw : cells - 1;
    const int ic0 = cell % P.nc[0], ic1 = (cell / P.nc[0]) % P.nc[1], ic2 = cell / (P.nc[0] * P.nc[1]);
    pdl_wait();  // programmatic launch: the predictor's residual and traces are complete and visible
    const double *rvol = pdl_fresh(rvol_in), *trace = pdl_fresh(trace_in);

    for (int idx = node; idx < 6 * n2; idx += n3) {
        const int f = idx / n2, m = idx - f * n2;
        const int a = m / n, b = m - a * n;
        const int dir = f >> 1;
        const bool plus = (f & 1) == 0;
        // selects instead of arrays indexed by the face's direction (keeps
        // everything in registers)
        const int icd = dir == 0 ? ic0 : dir == 1 ? ic1 : ic2;
        const int ncd = dir == 0 ? P.nc[0] : dir == 1 ? P.nc[1] : P.nc[2];
        const int bcd = dir == 0 ? P.bc[0] : dir == 1 ? P.bc[1] : P.bc[2];
        const bool edge = plus ? icd == ncd - 1 : icd == 0;
        const double* own = trace + ((size_t)cell * 6 + f) * TR;
        double qo[5], fo[5], g[3][5];
#pragma unroll
        for (int v = 0; v < 5; ++v) {
            qo[v] = own[v * n2 + m];
            fo[v] = own[(5 + v) * n2 + m];
        }
        const double so = own[25 * n2 + m];
        double qn[5], fn[5], sn;
        if (edge && bcd == ADG_BC_WALL) {
            // slip wall: background rho, rhoE at the face node (interior ones
            // without gravity), reflected normal momentum, interior gradient,
            // background heat flux
            double z, pb, rb;
            if (dir < 2) {
                z = P.org[2] + (ic2 + B.xi[a]) * P.h[2];
                pb = bg.pn[ic2 * n + a];
                rb = bg.rn[ic2 * n + a];
            } else {
                const int fz = ic2 + (plus ? 1 : 0);
                z = P.org[2] + fz * P.h[2];
                pb = bg.pf[fz];
                rb = bg.rf[fz];
            }
            qn[0] = qo[0];
            qn[1] = dir == 0 ? -qo[1] : qo[1];
            qn[2] = dir == 1 ? -qo[2] : qo[2];
            qn[3] = dir == 2 ? -qo[3] : qo[3];
            qn[4] = qo[4];
            if (P.gravity) {
                qn[0] = rb;
                qn[4] = pb / P.gm1 + rb * P.g * z;
            }
#pragma unroll
            for (int c = 0; c < 3; ++c)
#pragma unroll
                for (int v = 0; v < 5; ++v) g[c][v] = own[((2 + c) * 5 + v) * n2 + m];
            if constexpr (MX) {
                // the ghost's flux and speed in FP32: with gravity the zero
                // perturbation of rho and rhoE over the exact background at the
                // face node (rhobar, pbar, Ebar + pbar), without it the ghost state
                float qg[5], gf[3][5], ff[3][5], src;
                float rbf = 0.0f, pbf = 0.0f, Hbf = 0.0f, gz = 0.0f;
                if (P.gravity) {
                    qg[0] = 0.0f;
                    qg[4] = 0.0f;
                    rbf = f64_to_f32(rb);
                    pbf = f64_to_f32(pb);
                    Hbf = f64_to_f32(qn[4] + pb);
                    gz = f64_to_f32(P.g * z);
                } else {
                    qg[0] = f64_to_f32(qn[0]);
                    qg[4] = f64_to_f32(qn[4]);
                }
                qg[1] = f64_to_f32(qn[1]);
                qg[2] = f64_to_f32(qn[2]);
                qg[3] = f64_to_f32(qn[3]);
#pragma unroll
                for (int c = 0; c < 3; ++c)
#pragma unroll
                    for (int v = 0; v < 5; ++v) gf[c][v] = f64_to_f32(g[c][v]);
                ns_flux3f(qg, gf, gz, rbf, pbf, Hbf, Pf, ff, src, true, Pf.dTdz);
#pragma unroll
                for (int v = 0; v < 5; ++v) fn[v] = f32_to_f64(dir == 0 ? ff[0][v] : dir == 1 ? ff[1][v] : ff[2][v]);
                const float rho = rbf + qg[0];
                const float rinv = __frcp_rn(rho);
                const float pp = Pf.gm1 * (qg[4] - 0.5f * (qg[1] * qg[1] + qg[2] * qg[2] + qg[3] * qg[3]) * rinv -
                                           gz * qg[0]);
                const float mn = dir == 0 ? qg[1] : dir == 1 ? qg[2] : qg[3];
                sn = f32_to_f64(fabsf(mn) * rinv + sqrtf(Pf.gamma * (pbf + pp) * rinv) +
                                2.0f * Pf.eta[dir] * Pf.lamv * rinv);
            } else {
                double ff[3][5], src;
                ns_flux3(qn, g, z, pb, rb, P, true, ff, src);
#pragma unroll
                for (int v = 0; v < 5; ++v) fn[v] = dir == 0 ? ff[0][v] : dir == 1 ? ff[1][v] : ff[2][v];
                sn = wave_speed3(qn, z, dir, P);
            }
        } else if (edge && bcd == ADG_BC_ANALYTIC) {
            // the analytic field averaged over the step at the time nodes
            double xf[3];
            const int icc[3] = {ic0, ic1, ic2};
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                // along the face: node a (x-, y-faces: z; z-faces: y) and b
                const bool normal = c == dir;
                const int node_c = c == 2 ? a : (c == 1 ? (dir == 2 ? a : (dir == 0 ? b : 0)) : b);
                xf[c] = normal ? P.org[c] + (icc[c] + (plus ? 1 : 0)) * P.h[c]
                               : P.org[c] + (icc[c] + B.xi[node_c]) * P.h[c];
            }
#pragma unroll
            for (int v = 0; v < 5; ++v) qn[v] = fn[v] = 0.0;
            for (int k = 0; k < n; ++k) {
                double q[5], ff[3][5], src;
                abc_field(xf[0], xf[1], xf[2], t + B.xi[k] * dt, P, q, g);
                ns_flux3(q, g, xf[2], 0.0, 0.0, P, false, ff, src);
#pragma unroll
                for (int v = 0; v < 5; ++v) {
                    qn[v] += B.w[k] * q[v];
                    fn[v] += B.w[k] * (dir == 0 ? ff[0][v] : dir == 1 ? ff[1][v] : ff[2][v]);
                }
            }
            sn = wave_speed3(qn, xf[2], dir, P);
        } else {
            const int nd = plus ? (icd + 1 == ncd ? 0 : icd + 1) : (icd == 0 ? ncd - 1 : icd - 1);
            const int nb0 = dir == 0 ? nd : ic0, nb1 = dir == 1 ? nd : ic1, nb2 = dir == 2 ? nd : ic2;
            const int nc = (nb2 * P.nc[1] + nb1) * P.nc[0] + nb0;
            const double* ot = trace + ((size_t)nc * 6 + (f ^ 1)) * TR;
#pragma unroll
            for (int v = 0; v < 5; ++v) {
                qn[v] = ot[v * n2 + m];
                fn[v] = ot[(5 + v) * n2 + m];
            }
            sn = ot[25 * n2 + m];
        }
        if constexpr (MX) {
            const double* qL = plus ? qo : qn;
            const double* qR = plus ? qn : qo;
            const double* fL = plus ? fo : fn;
            const double* fR = plus ? fn : fo;
            const float hs = 0.5f * fmaxf(f64_to_f32(so), f64_to_f32(sn));
#pragma unroll
            for (int v = 0; v < 5; ++v)
                Fst[cl][f][v][m] = 0.5f * (f64_to_f32(fL[v]) + f64_to_f32(fR[v])) -
                                   hs * f64_to_f32(__dsub_rn(qR[v], qL[v]));
        } else {
            double out[5];
            if (plus) rusanov5(qo, fo, so, qn, fn, sn, out);
            else rusanov5(qn, fn, sn, qo, fo, so, out);
#pragma unroll
            for (int v = 0; v < 5; ++v) Fst[cl][f][v][m] = out[v];
        }
    }
    __syncthreads();
    if (!active) return;
    double* uc = u + (size_t)cell * SL;
    const double* rc = rvol + (size_t)cell * SL;
    FT l1[3], l0[3], ih[3];
    {
        const int id[3] = {i, j, l};
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            if constexpr (MX) {
                l1[c] = f64_to_f32(B.lift1[id[c]]);
                l0[c] = f64_to_f32(B.lift0[id[c]]);
                ih[c] = f64_to_f32(P.inv_h[c]);
            } else {
                l1[c] = B.lift1[id[c]];
                l0[c] = B.lift0[id[c]];
                ih[c] = P.inv_h[c];
            }
        }
    }
#pragma unroll
    for (int v = 0; v < 5; ++v) {
        const FT face = (l1[0] * Fst[cl][0][v][l * n + j] - l0[0] * Fst[cl][1][v][l * n + j]) * ih[0] +
                        (l1[1] * Fst[cl][2][v][l * n + i] - l0[1] * Fst[cl][3][v][l * n + i]) * ih[1] +
                        (l1[2] * Fst[cl][4][v][j * n + i] - l0[2] * Fst[cl][5][v][j * n + i]) * ih[2];
        double fd;
        if constexpr (MX) fd = f32_to_f64(face);
        else fd = face;
        uc[v * n3 + node] += dt * (rc[v * n3 + node] - fd);
    }
}

// ---------------------------------------------------------------------------
// Mixed precision predictor: the same Picard iteration in FP32 on
// perturbation variables q' = (rho - rhobar, rho u, rho v, rho w, rhoE - Ebar)
// (the split in FP64 at load), total gradients = perturbation gradient +
// the FP64-formed derivative of the interpolated background.  With
// p' = (gamma-1)(E' - |m|^2/(2 rho) - g z rho') exact algebra, no FP32 value
// carries the background pressure through a difference.  Outputs keep the
// FP64 formats of the FP64 predictor: rvol converted, traces rebuilt as the
// FP64 base (the nodal background on x- and y-faces, its FP64 extrapolation
// on z-faces) plus the FP32 perturbation, the Rusanov speed in FP64 -- so
// the FP64 corrector runs unchanged.
template <int N>
struct Cfg3m {
    // per cell, in fields of n^3 floats: the n time slices of q' (5 each) and the
    // nine fluxes of one slice, or the 29 averages (q', fluxes, grad q)
    static constexpr int fields = 5 * (N + 1) + 9 > 29 ? 5 * (N + 1) + 9 : 29;
    static constexpr size_t smem = (size_t)Cfg3<N>::cpb * fields * Cfg3<N>::n3 * sizeof(float);
    // resident blocks asked of the register allocator (us a step with 1 / 2 / 3 / 4
    // / 5): degree 2 on 25^3 cells 164 / 165 / 161 / 162 / 169, degree 3 on 17^3 155
    // / 130 / 127 / 136 / 153, degree 4 on 13^3 188 / 190 / 191 / 203 / 243
    static constexpr int minb = N == 2 ? 4 : N == 3 ? 3 : N == 4 ? 2 : 1;
};

template <int N>
__global__ void __launch_bounds__(Cfg3<N>::threads, Cfg3m<N>::minb)
k3_predictor_mixed(const double* __restrict__ u, double* __restrict__ rvol, double* __restrict__ trace, int cells,
                   float dt, const BasisF B, const Phys3f P, const Phys3 P64, const Bg3m bg) {
    using C = Cfg3<N>;
    constexpr int n = C::n, n2 = C::n2, n3 = C::n3, SL = 5 * n3;
    extern __shared__ float smf[];
    const int cl = threadIdx.x / n3;
    const int node = threadIdx.x - cl * n3;
    const int l = node / n2, j = (node / n) % n, i = node % n;
    const int cell_raw = blockIdx.x * C::cpb + cl;
    const bool active = cell_raw < cells;
    const int cell = active ? cell_raw : cells - 1;
    const int iz = cell / (P64.nc[0] * P64.nc[1]);
    float* Q = smf + (size_t)cl * Cfg3m<N>::fields * n3;
    float* Fs = Q + n * SL;  // six momentum, three energy fluxes
    const int nb = iz * n + l;
    const float rb = bg.rbf[nb], Hb = bg.Hbf[nb], dzr = bg.dzr[nb], dzE = bg.dzE[nb];
    const float Eb = f64_to_f32(bg.Eb[nb]);
    const float gz = (float)(P64.g * bg.zn[nb]);

    float uu[5];
    {
        const double* uc = u + (size_t)cell * SL;
        uu[0] = f64_to_f32(__dsub_rn(uc[node], bg.rb[nb]));
        uu[1] = f64_to_f32(uc[n3 + node]);
        uu[2] = f64_to_f32(uc[2 * n3 + node]);
        uu[3] = f64_to_f32(uc[3 * n3 + node]);
        uu[4] = f64_to_f32(__dsub_rn(uc[4 * n3 + node], bg.Eb[nb]));
    }
#pragma unroll
    for (int v = 0; v < 5; ++v) Q[v * n3 + node] = uu[v];
    __syncthreads();

    // this node's rows of D, scaled by 1/h
    float dI[3][n];
#pragma unroll
    for (int p = 0; p < n; ++p) {
        dI[0][p] = B.D[i][p] * P.inv_h[0];
        dI[1][p] = B.D[j][p] * P.inv_h[1];
        dI[2][p] = B.D[l][p] * P.inv_h[2];
    }
    auto line = [&](const float* S, int b) {
        const int o = b == 0 ? (l * n + j) * n : b == 1 ? l * n2 + i : j * n + i, st = b == 0 ? 1 : b == 1 ? n : n2;
        float s = dI[b][0] * S[o];
#pragma unroll
        for (int p = 1; p < n; ++p) s = fmaf(dI[b][p], S[o + p * st], s);
        return s;
    };
    // state, gradients and fluxes of time slice Qk; md: divergence of the mass flux, minus the source of the
    // z-momentum
    auto eval = [&](const float* Qk, float q[5], float g[3][5], Fx3FluxF& f, float& md) {
#pragma unroll
        for (int v = 0; v < 5; ++v) {
            q[v] = Qk[v * n3 + node];
#pragma unroll
            for (int b = 0; b < 3; ++b) g[b][v] = line(Qk + v * n3, b);
        }
        md = g[0][1] + g[1][2] + g[2][3];
        g[2][0] += dzr;
        g[2][4] += dzE;
        f = ns_flux9_pert(q, g, gz, rb, Eb, Hb, P);
    };
    auto store = [&](const Fx3FluxF& f) {
#pragma unroll
        for (int a = 0; a < 6; ++a) Fs[a * n3 + node] = f.t[a];
#pragma unroll
        for (int a = 0; a < 3; ++a) Fs[(6 + a) * n3 + node] = f.e[a];
    };
    // residual of variable v at this node from the slice in Fs (v = 0: from md)
    auto residual = [&](int v, float md, const float q[5]) {
        if (v == 0) return -md;
        float s;
        if (v < 4) s = line(Fs + fx3_t(v - 1, 0) * n3, 0) + line(Fs + fx3_t(v - 1, 1) * n3, 1) + line(Fs + fx3_t(v - 1, 2) * n3, 2);
        else s = line(Fs + 6 * n3, 0) + line(Fs + 7 * n3, 1) + line(Fs + 8 * n3, 2);
        return v == 3 && P.gravity ? fmaf(-P.g, q[0], -s) : -s;
    };

    {
        float q[5], g[3][5], md;
        Fx3FluxF f;
        eval(Q, q, g, f, md);
        store(f);
        __syncthreads();
        float R0[5];
#pragma unroll
        for (int v = 0; v < 5; ++v) R0[v] = residual(v, md, q);
#pragma unroll
        for (int k = 0; k < n; ++k)
#pragma unroll
            for (int v = 0; v < 5; ++v) Q[k * SL + v * n3 + node] = uu[v] + dt * (B.Kw1[k] * R0[v]);
        __syncthreads();
    }
    // Sweeps 2..n.  Degrees <= 2 accumulate the time contraction slice by
    // slice (the same order as a row-by-row sum), degree 1 with a rolled loop
    // (152.5 against 154.9 us a step on 41^3 cells unrolled; degree 2 165.1
    // rolled, 161.7 unrolled on 25^3); degrees 3 and 4 keep the residuals of all
    // slices in registers.
    constexpr int kSliceUnroll = N == 1 ? 1 : n;
#pragma unroll 1
    for (int r = 1; r < n; ++r) {
        if constexpr (N <= 2) {
            float acc[n][5];
#pragma unroll
            for (int k = 0; k < n; ++k)
#pragma unroll
                for (int v = 0; v < 5; ++v) acc[k][v] = 0.0f;
#pragma unroll kSliceUnroll
            for (int m = 0; m < n; ++m) {
                float q[5], g[3][5], md;
                Fx3FluxF f;
                eval(Q + m * SL, q, g, f, md);
                __syncthreads();
                store(f);
                __syncthreads();
#pragma unroll
                for (int v = 0; v < 5; ++v) {
                    const float Rm = residual(v, md, q);
#pragma unroll
                    for (int k = 0; k < n; ++k) acc[k][v] = fmaf(B.Kw[k][m], Rm, acc[k][v]);
                }
            }
#pragma unroll
            for (int k = 0; k < n; ++k)
#pragma unroll
                for (int v = 0; v < 5; ++v) Q[k * SL + v * n3 + node] = uu[v] + dt * acc[k][v];
        } else {
            float R[n][5];
#pragma unroll
            for (int k = 0; k < n; ++k) {
                float q[5], g[3][5], md;
                Fx3FluxF f;
                eval(Q + k * SL, q, g, f, md);
                __syncthreads();
                store(f);
                __syncthreads();
#pragma unroll
                for (int v = 0; v < 5; ++v) R[k][v] = residual(v, md, q);
            }
#pragma unroll
            for (int k = 0; k < n; ++k)
#pragma unroll
                for (int v = 0; v < 5; ++v) {
                    float acc = 0.0f;
#pragma unroll
                    for (int m = 0; m < n; ++m) acc = fmaf(B.Kw[k][m], R[m][v], acc);
                    Q[k * SL + v * n3 + node] = uu[v] + dt * acc;
                }
        }
        __syncthreads();
    }

    const int ic0 = cell % P64.nc[0], ic1 = (cell / P64.nc[0]) % P64.nc[1];
    unsigned wf = 0;  // slip-wall faces, which alone read grad q-bar
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const int ic = d == 0 ? ic0 : d == 1 ? ic1 : iz;
        if (P64.bc[d] == ADG_BC_WALL) wf |= (ic == P64.nc[d] - 1 ? 1u << (2 * d) : 0u) | (ic == 0 ? 2u << (2 * d) : 0u);
    }
    float qb[5], tb[6], eb[3], gb[3][5];
#pragma unroll
    for (int v = 0; v < 5; ++v) {
        qb[v] = 0.0f;
#pragma unroll
        for (int b = 0; b < 3; ++b) gb[b][v] = 0.0f;
    }
#pragma unroll
    for (int a = 0; a < 6; ++a) tb[a] = 0.0f;
    eb[0] = eb[1] = eb[2] = 0.0f;
#pragma unroll kSliceUnroll
    for (int k = 0; k < n; ++k) {
        float q[5], g[3][5], md;
        Fx3FluxF f;
        eval(Q + k * SL, q, g, f, md);
        const float wk = B.w[k];
#pragma unroll
        for (int v = 0; v < 5; ++v) qb[v] = fmaf(wk, q[v], qb[v]);
#pragma unroll
        for (int a = 0; a < 6; ++a) tb[a] = fmaf(wk, f.t[a], tb[a]);
#pragma unroll
        for (int a = 0; a < 3; ++a) eb[a] = fmaf(wk, f.e[a], eb[a]);
        if (wf) {
#pragma unroll
            for (int v = 0; v < 5; ++v)
#pragma unroll
                for (int b = 0; b < 3; ++b) gb[b][v] = fmaf(wk, g[b][v], gb[b][v]);
        }
    }
    __syncthreads();
    // fields: q' (5), momentum fluxes (6), energy fluxes (3), grad q (15)
    float* A = Q;
#pragma unroll
    for (int v = 0; v < 5; ++v) A[v * n3 + node] = qb[v];
#pragma unroll
    for (int a = 0; a < 6; ++a) A[(5 + a) * n3 + node] = tb[a];
#pragma unroll
    for (int a = 0; a < 3; ++a) A[(11 + a) * n3 + node] = eb[a];
    if (wf) {
#pragma unroll
        for (int b = 0; b < 3; ++b)
#pragma unroll
            for (int v = 0; v < 5; ++v) A[(14 + 5 * b + v) * n3 + node] = gb[b][v];
    }
    __syncthreads();
    if (active) {
        double* rc = rvol + (size_t)cell * SL;
#pragma unroll
        for (int v = 0; v < 5; ++v) {
            const float* Fv = A + fx3_slot(5 + v, 0) * n3;
            const float* Gv = A + fx3_slot(5 + v, 1) * n3;
            const float* Hv = A + fx3_slot(5 + v, 2) * n3;
            float sx = 0.0f, sy = 0.0f, sz = 0.0f;
#pragma unroll
            for (int p = 0; p < n; ++p) {
                sx = fmaf(B.Vx[p][i], Fv[(l * n + j) * n + p], sx);
                sy = fmaf(B.Vx[p][j], Gv[(l * n + p) * n + i], sy);
                sz = fmaf(B.Vx[p][l], Hv[(p * n + j) * n + i], sz);
            }
            rc[v * n3 + node] = f32_to_f64(sx * P.inv_h[0] + sy * P.inv_h[1] + sz * P.inv_h[2] + (v == 3 && P.gravity ? -P.g * qb[0] : 0.0f));
        }
    }
    for (int idx = node; idx < 6 * n2; idx += n3) {
        const int f = idx / n2, m = idx - f * n2;
        const int a = m / n, b = m - a * n;
        const int dir = f >> 1;
        const bool wallface = wf >> f & 1u;
        const int at = dir == 0 ? (a * n + b) * n : dir == 1 ? a * n2 + b : a * n + b;
        const int st = dir == 0 ? 1 : dir == 1 ? n : n2;
        float phi[n];
#pragma unroll
        for (int p = 0; p < n; ++p) phi[p] = (f & 1) ? B.phi0[p] : B.phi1[p];
        auto ext = [&](const float* S) {
            float s = 0.0f;
#pragma unroll
            for (int p = 0; p < n; ++p) s = fmaf(phi[p], S[at + p * st], s);
            return s;
        };
        float rec[5];
#pragma unroll
        for (int v = 0; v < 5; ++v) rec[v] = ext(A + v * n3);
        const float mn = dir == 0 ? rec[1] : dir == 1 ? rec[2] : rec[3];
        double* tr = trace + ((size_t)cell * 6 + f) * kTr3 * n2 + m;
        if (active) {
            tr[5 * n2] = f32_to_f64(mn);
#pragma unroll
            for (int c = 0; c < 3; ++c) tr[(6 + c) * n2] = f32_to_f64(ext(A + (5 + fx3_t(c, dir)) * n3));
            tr[9 * n2] = f32_to_f64(ext(A + (11 + dir) * n3));
            if (wallface)
                for (int c = 0; c < 15; ++c) tr[(10 + c) * n2] = f32_to_f64(ext(A + (14 + c) * n3));
        }
        // FP64 base of the face node: the nodal background at the node's height
        // on x- and y-faces, its extrapolation on z-faces
        double brho, bE;
        if (dir < 2) {
            brho = bg.rb[iz * n + a];
            bE = bg.Eb[iz * n + a];
        } else {
            const double* e = bg.ext + ((size_t)iz * 2 + (f & 1)) * 2;
            brho = e[0];
            bE = e[1];
        }
        // Rusanov speed in FP32 from the perturbation face state over its base
        {
            float rbf, pbf, zf;
            if (dir < 2) {
                rbf = bg.rbf[iz * n + a];
                pbf = bg.pbf[iz * n + a];
                zf = (float)bg.zn[iz * n + a];
            } else {
                const float* e = bg.zext + ((size_t)iz * 2 + (f & 1)) * 2;
                rbf = e[0];
                pbf = e[1];
                zf = (float)(P64.org[2] + (iz + ((f & 1) ? 0 : 1)) * P64.h[2]);
            }
            const float qp0 = rec[0], qp4 = rec[4];
            const float m0 = rec[1], m1 = rec[2], m2 = rec[3];
            const float rho = rbf + qp0;
            const float rinv = __frcp_rn(rho);
            const float pp = P.gm1 * (qp4 - 0.5f * (m0 * m0 + m1 * m1 + m2 * m2) * rinv - P.g * zf * qp0);
            const float sp = fabsf(mn) * rinv + sqrtf(P.gamma * (pbf + pp) * rinv) +
                             2.0f * P.eta[dir] * P.lamv * rinv;
            if (active) tr[25 * n2] = f32_to_f64(sp);
        }
        if (active) {
            tr[0] = f32_to_f64(rec[0]) + brho;
            tr[n2] = f32_to_f64(rec[1]);
            tr[2 * n2] = f32_to_f64(rec[2]);
            tr[3 * n2] = f32_to_f64(rec[3]);
            tr[4 * n2] = f32_to_f64(rec[4]) + bE;
        }
    }
    pdl_trigger();
}

// nodal values of a scenario: the 3D cosine bubble or the background
// (theta' at the background pressure, at rest), or the ABC field at time t
__global__ void k3_init(double* __restrict__ u, int cells, int n, int kind, double A, double a, double xc, double zc,
                        double t, const Basis B, const Phys3 P) {
    const int n3 = n * n * n;
    const long long gid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (gid >= (long long)cells * n3) return;
    const int cell = (int)(gid / n3), node = (int)(gid % n3);
    const int l = node / (n * n), j = (node / n) % n, i = node % n;
    const int ix = cell % P.nc[0], iy = (cell / P.nc[0]) % P.nc[1], iz = cell / (P.nc[0] * P.nc[1]);
    const double x = P.org[0] + (ix + B.xi[i]) * P.h[0];
    const double y = P.org[1] + (iy + B.xi[j]) * P.h[1];
    const double z = P.org[2] + (iz + B.xi[l]) * P.h[2];
    double q[5];
    if (kind == ADG_SCEN_ABC) {
        double g[3][5];
        abc_field(x, y, z, t, P, q, g);
    } else {
        double th = 0.0;
        if (kind == ADG_SCEN_COSINE) {
            const double r = sqrt((x - xc) * (x - xc) + (y - xc) * (y - xc) + (z - zc) * (z - zc));
            th = r <= a ? 0.5 * A * (1.0 + cos(3.14159265358979323846 * r / a)) : 0.0;
        }
        const double ex = 1.0 - P.g * z / (P.cp * P.theta0);
        const double pb = P.p0 * pow(ex, P.cp / P.R);
        const double rho = pb / (P.R * (P.theta0 + th) * ex);
        q[0] = rho;
        q[1] = q[2] = q[3] = 0.0;
        q[4] = pb / P.gm1 + rho * P.g * z;
    }
    double* uc = u + (size_t)cell * 5 * n3;
    for (int v = 0; v < 5; ++v) uc[v * n3 + node] = q[v];
}

// per-block maxima of |v| + c + 2 eta lambda_v / rho over the nodes
__global__ void __launch_bounds__(256) k3_speed(const double* __restrict__ u, int cells, int n, double eta,
                                                double* __restrict__ part, const Basis B, const Phys3 P) {
    __shared__ double red[256];
    const int n3 = n * n * n;
    const long long gid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    double s = 0.0;
    if (gid < (long long)cells * n3) {
        const int cell = (int)(gid / n3), node = (int)(gid % n3);
        const int l = node / (n * n);
        const int iz = cell / (P.nc[0] * P.nc[1]);
        const double z = P.org[2] + (iz + B.xi[l]) * P.h[2];
        const double* uc = u + (size_t)cell * 5 * n3;
        double q[5];
        for (int v = 0; v < 5; ++v) q[v] = uc[v * n3 + node];
        const double rinv = 1.0 / q[0];
        const double gg = P.gravity ? P.g : 0.0;
        const double m2 = q[1] * q[1] + q[2] * q[2] + q[3] * q[3];
        const double p = P.gm1 * (q[4] - 0.5 * m2 * rinv - q[0] * gg * z);
        s = sqrt(m2) * rinv + sqrt(P.gamma * p * rinv) + 2.0 * eta * P.lamv * rinv;
        if (!(s == s)) s = INFINITY;  // NaN state: reported as a non-finite speed
    }
    red[threadIdx.x] = s;
    __syncthreads();
    for (int k = 128; k > 0; k >>= 1) {
        if ((int)threadIdx.x < k) red[threadIdx.x] = fmax(red[threadIdx.x], red[threadIdx.x + k]);
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = red[0];
}

template <int N>
int launch3(bool pred, double* u, double* rvol, double* trace, int cells, double dt, double t, const Basis& B,
            const Phys3& P, const Bg3& bg, cudaStream_t s, bool mixed, const Phys3f& Pf) {
    using C = Cfg3<N>;
    const int blocks = (cells + C::cpb - 1) / C::cpb;
    if (pred) {
        using X = Fx3Cfg<N>;
        cudaError_t e = cudaFuncSetAttribute(k3_predictor<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)X::smem);
        if (e != cudaSuccess) return (int)e;
        k3_predictor<N><<<fx_grid((cells + X::cpb - 1) / X::cpb, X::resident), X::threads, X::smem, s>>>(
            u, rvol, trace, cells, dt, B, P, bg);
    } else {
        // programmatic launch: scheduled while the predictor drains
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(blocks);
        cfg.blockDim = dim3(C::threads);
        cfg.dynamicSmemBytes = 0;
        cfg.stream = s;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        // Mixed, degrees 1 and 2: four blocks an SM (25^3 degree-2 bubble, us a step, 157.9 / 154.9 / 153.9 / 156.8
        // with 2 / 3 / 4 / 5), but two where the analytic field is evaluated on the boundary, whose registers would
        // spill (25^3 ABC flow 432 / 447 / 498 with 2 / 3 / 4, degree 1 122 / 122 / 135).
        constexpr int kMany = N <= 2 ? 4 : 2;
        const bool analytic = P.bc[0] == ADG_BC_ANALYTIC || P.bc[1] == ADG_BC_ANALYTIC || P.bc[2] == ADG_BC_ANALYTIC;
        auto kern = !mixed ? k3_corrector<N, false, 2> : analytic ? k3_corrector<N, true, 2> : k3_corrector<N, true, kMany>;
        const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, u, rvol, trace, cells, dt, t, B, P, bg, Pf);
        if (e != cudaSuccess) return (int)e;
    }
    return (int)cudaGetLastError();
}

template <int N>
int launch3m(const double* u, double* rvol, double* trace, int cells, float dt, const BasisF& B, const Phys3f& P,
             const Phys3& P64, const Bg3m& bg, cudaStream_t s) {
    using C = Cfg3<N>;
    const int blocks = (cells + C::cpb - 1) / C::cpb;
    cudaError_t e = cudaFuncSetAttribute(k3_predictor_mixed<N>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)Cfg3m<N>::smem);
    if (e != cudaSuccess) return (int)e;
    k3_predictor_mixed<N><<<blocks, C::threads, Cfg3m<N>::smem, s>>>(u, rvol, trace, cells, dt, B, P, P64, bg);
    return (int)cudaGetLastError();
}

int launch3m_any(int N, const double* u, double* rvol, double* trace, int cells, float dt, const BasisF& B,
                 const Phys3f& P, const Phys3& P64, const Bg3m& bg, cudaStream_t s) {
    switch (N) {
        case 1: return launch3m<1>(u, rvol, trace, cells, dt, B, P, P64, bg, s);
        case 2: return launch3m<2>(u, rvol, trace, cells, dt, B, P, P64, bg, s);
        case 3: return launch3m<3>(u, rvol, trace, cells, dt, B, P, P64, bg, s);
        case 4: return launch3m<4>(u, rvol, trace, cells, dt, B, P, P64, bg, s);
        default: return (int)cudaErrorInvalidValue;
    }
}

int launch3_any(int N, bool pred, double* u, double* rvol, double* trace, int cells, double dt, double t,
                const Basis& B, const Phys3& P, const Bg3& bg, cudaStream_t s, bool mixed, const Phys3f& Pf) {
    switch (N) {
        case 1: return launch3<1>(pred, u, rvol, trace, cells, dt, t, B, P, bg, s, mixed, Pf);
        case 2: return launch3<2>(pred, u, rvol, trace, cells, dt, t, B, P, bg, s, mixed, Pf);
        case 3: return launch3<3>(pred, u, rvol, trace, cells, dt, t, B, P, bg, s, mixed, Pf);
        case 4: return launch3<4>(pred, u, rvol, trace, cells, dt, t, B, P, bg, s, mixed, Pf);
        default: return (int)cudaErrorInvalidValue;
    }
}
}  // namespace
}  // namespace adg

struct adg_mesh3 {
    adg_mesh_desc d;
    int N = 0, n = 0, nz = 0, bc_z = 0, cells = 0;
    double z0 = 0, Lz = 0, t = 0;
    adg::Basis B;
    adg::Phys3 P;
    double* u = nullptr;      // [cells][5][n^3]
    double* rvol = nullptr;   // [cells][5][n^3]
    double* trace = nullptr;  // [cells][6][kTr3][n^2]
    double* bg = nullptr;     // pbar, rhobar at nodes [nz n] each, then at faces [nz + 1] each
    double* part = nullptr;   // stable-dt block maxima
    int part_blocks = 0;
    // mixed precision: FP32 basis and constants, background tables
    adg::BasisF Bf;
    adg::Phys3f Pf;
    double* mbg = nullptr;    // rhobar, Ebar, node height [nz n] each, then extrapolated z-face base [nz][2][2]
    float* mbgf = nullptr;    // rhobar, pbar, Ebar + pbar, d rhobar/dz, d Ebar/dz [nz n] each
};

using adg::cuda_fail;
using adg::fail;

namespace {

int dev3(const adg_mesh3* m) {
    const cudaError_t e = cudaSetDevice(m->d.device);
    return e == cudaSuccess ? ADG_OK : cuda_fail(e, "mesh3: cudaSetDevice");
}

void free3(adg_mesh3* m) {
    if (!m) return;
    cudaSetDevice(m->d.device);
    cudaFree(m->u);
    cudaFree(m->rvol);
    cudaFree(m->trace);
    cudaFree(m->bg);
    cudaFree(m->part);
    cudaFree(m->mbg);
    cudaFree(m->mbgf);
    delete m;
}

adg::Bg3 bg3(const adg_mesh3* m) {
    const int nn = m->nz * m->n;
    return adg::Bg3{m->bg, m->bg + nn, m->bg + 2 * nn, m->bg + 2 * nn + (m->nz + 1)};
}

adg::Bg3m bg3m(const adg_mesh3* m) {
    const size_t nn = (size_t)m->nz * m->n;
    adg::Bg3m b;
    b.rb = m->mbg;
    b.Eb = m->mbg + nn;
    b.zn = m->mbg + 2 * nn;
    b.ext = m->mbg + 3 * nn;
    b.rbf = m->mbgf;
    b.pbf = m->mbgf + nn;
    b.Hbf = m->mbgf + 2 * nn;
    b.dzr = m->mbgf + 3 * nn;
    b.dzE = m->mbgf + 4 * nn;
    b.zext = m->mbgf + 5 * nn;
    return b;
}

// FP32 basis and constants and the background tables of the mixed predictor
int build_mixed3(adg_mesh3* m) {
    const int n = m->n, nz = m->nz;
    const adg::Basis& B = m->B;
    adg::BasisF& b = m->Bf;
    std::memset(&b, 0, sizeof(b));
    for (int a = 0; a < n; ++a) {
        b.xi[a] = (float)B.xi[a];
        b.w[a] = (float)B.w[a];
        b.phi0[a] = (float)B.phi0[a];
        b.phi1[a] = (float)B.phi1[a];
        b.Kw1[a] = (float)B.Kw1[a];
        b.lift0[a] = (float)B.lift0[a];
        b.lift1[a] = (float)B.lift1[a];
        for (int c = 0; c < n; ++c) {
            b.D[a][c] = (float)B.D[a][c];
            b.Kw[a][c] = (float)B.Kw[a][c];
            b.Vx[a][c] = (float)B.Vx[a][c];
        }
    }
    const adg::Phys3& P = m->P;
    adg::Phys3f& f = m->Pf;
    std::memset(&f, 0, sizeof(f));
    f.gamma = (float)P.gamma;
    f.gm1 = (float)P.gm1;
    f.R = (float)P.R;
    f.invR = (float)P.invR;
    f.mu = (float)P.mu;
    f.kappa = (float)P.kappa;
    f.g = (float)P.g;
    f.lamv = (float)P.lamv;
    f.dTdz = (float)P.dTdz;
    for (int c = 0; c < 3; ++c) {
        f.inv_h[c] = (float)P.inv_h[c];
        f.eta[c] = (float)P.eta[c];
    }
    f.gravity = P.gravity;
    const size_t nn = (size_t)nz * n;
    std::vector<double> hd(3 * nn + 4 * (size_t)nz, 0.0);
    std::vector<float> hf(5 * nn + 4 * (size_t)nz, 0.0f);
    std::vector<double> rb(nn, 0.0), Eb(nn, 0.0), pb(nn, 0.0);
    for (int iz = 0; iz < nz; ++iz)
        for (int l = 0; l < n; ++l) {
            const size_t k = (size_t)iz * n + l;
            const double z = P.org[2] + (iz + B.xi[l]) * P.h[2];
            hd[2 * nn + k] = z;
            if (P.gravity) {
                const double ex = 1.0 - P.g * z / (P.cp * P.theta0);
                pb[k] = P.p0 * std::pow(ex, P.cp / P.R);
                rb[k] = pb[k] / (P.R * P.theta0 * ex);
                Eb[k] = pb[k] / P.gm1 + rb[k] * P.g * z;
            }
        }
    for (int iz = 0; iz < nz; ++iz) {
        for (int l = 0; l < n; ++l) {
            const size_t k = (size_t)iz * n + l;
            double dr = 0.0, dE = 0.0;
            for (int p = 0; p < n; ++p) {
                dr += B.D[l][p] * rb[(size_t)iz * n + p];
                dE += B.D[l][p] * Eb[(size_t)iz * n + p];
            }
            hd[k] = rb[k];
            hd[nn + k] = Eb[k];
            hf[k] = (float)rb[k];
            hf[nn + k] = (float)pb[k];
            hf[2 * nn + k] = (float)(Eb[k] + pb[k]);
            hf[3 * nn + k] = (float)(dr * P.inv_h[2]);
            hf[4 * nn + k] = (float)(dE * P.inv_h[2]);
        }
        for (int face = 0; face < 2; ++face) {  // 0: top (phi(1)), 1: bottom (phi(0))
            const double* phi = face == 0 ? B.phi1 : B.phi0;
            double er = 0.0, eE = 0.0;
            for (int p = 0; p < n; ++p) {
                er += phi[p] * rb[(size_t)iz * n + p];
                eE += phi[p] * Eb[(size_t)iz * n + p];
            }
            hd[3 * nn + ((size_t)iz * 2 + face) * 2] = er;
            hd[3 * nn + ((size_t)iz * 2 + face) * 2 + 1] = eE;
            const double zf = P.org[2] + (iz + (face == 0 ? 1 : 0)) * P.h[2];
            hf[5 * nn + ((size_t)iz * 2 + face) * 2] = (float)er;
            hf[5 * nn + ((size_t)iz * 2 + face) * 2 + 1] = (float)(P.gm1 * (eE - er * P.g * zf));
        }
    }
    if (cudaMalloc(&m->mbg, hd.size() * 8) != cudaSuccess || cudaMalloc(&m->mbgf, hf.size() * 4) != cudaSuccess) {
        cudaGetLastError();
        return fail(ADG_ENOMEM, "adg3_create: mixed-precision tables");
    }
    ADG_CK(cudaMemcpy(m->mbg, hd.data(), hd.size() * 8, cudaMemcpyHostToDevice), "adg3_create: mixed tables");
    ADG_CK(cudaMemcpy(m->mbgf, hf.data(), hf.size() * 4, cudaMemcpyHostToDevice), "adg3_create: mixed tables");
    return ADG_OK;
}

bool bc3_ok(int bc) { return bc == ADG_BC_PERIODIC || bc == ADG_BC_WALL || bc == ADG_BC_ANALYTIC; }

}  // namespace

extern "C" int adg3_create(const adg_mesh_desc* d, int nz, double z0, double Lz, int bc_z, adg_mesh3** out) {
    if (!d || !out) return fail(ADG_EINVAL, "adg3_create: NULL argument");
    *out = nullptr;
    if (d->degree < 1 || d->degree > ADG_MAX_DEGREE_3D) return fail(ADG_EINVAL, "adg3_create: degree out of range");
    if (d->nx < 1 || d->ny < 1 || nz < 1 || (long long)d->nx * d->ny * nz > (1LL << 24))
        return fail(ADG_EINVAL, "adg3_create: bad mesh size");
    if (!(d->Lx > 0.0) || !(d->Ly > 0.0) || !(Lz > 0.0) || !std::isfinite(z0))
        return fail(ADG_EINVAL, "adg3_create: Lx, Ly, Lz must be > 0");
    if (!bc3_ok(d->bc_x) || !bc3_ok(d->bc_y) || !bc3_ok(bc_z))
        return fail(ADG_EINVAL, "adg3_create: boundaries are periodic, ADG_BC_WALL or ADG_BC_ANALYTIC");
    if (!(d->gamma > 1.0) || !(d->R > 0.0) || !(d->Pr > 0.0) || !(d->mu >= 0.0))
        return fail(ADG_EINVAL, "adg3_create: invalid gas constants");
    if ((d->precision != ADG_PREC_FP64 && d->precision != ADG_PREC_MIXED) || d->source != ADG_SRC_NONE ||
        d->max_levels != 0)
        return fail(ADG_EUNSUPPORTED, "adg3_create: FP64 or mixed, no manufactured source, uniform mesh only");
    const bool analytic = d->bc_x == ADG_BC_ANALYTIC || d->bc_y == ADG_BC_ANALYTIC || bc_z == ADG_BC_ANALYTIC;
    if (analytic && (d->bc_field != ADG_FIELD_ABC || d->gravity))
        return fail(ADG_EINVAL, "adg3_create: analytic boundaries take bc_field ADG_FIELD_ABC without gravity");
    if (d->gravity && !(d->theta0 > 0.0 && d->p0 > 0.0 && d->g > 0.0))
        return fail(ADG_EINVAL, "adg3_create: gravity needs g, theta0, p0 > 0");
    int ndev = 0;
    ADG_CK(cudaGetDeviceCount(&ndev), "cudaGetDeviceCount");
    if (d->device < 0 || d->device >= ndev) return fail(ADG_EINVAL, "adg3_create: bad device ordinal");
    adg_mesh3* m = new adg_mesh3();
    m->d = *d;
    m->N = d->degree;
    m->n = d->degree + 1;
    m->nz = nz;
    m->z0 = z0;
    m->Lz = Lz;
    m->bc_z = bc_z;
    m->cells = d->nx * d->ny * nz;
    if (!adg::build_basis(m->N, m->B)) {
        delete m;
        return fail(ADG_EINVAL, "adg3_create: singular time-stiffness matrix");
    }
    adg::Phys3& P = m->P;
    std::memset(&P, 0, sizeof(P));
    std::memset(&m->Pf, 0, sizeof(m->Pf));
    P.gamma = d->gamma;
    P.gm1 = d->gamma - 1.0;
    P.R = d->R;
    P.invR = 1.0 / d->R;
    P.mu = d->mu;
    P.cp = d->gamma * d->R / (d->gamma - 1.0);
    P.kappa = d->mu * P.cp / d->Pr;
    P.gravity = d->gravity ? 1 : 0;
    P.g = d->gravity ? d->g : 0.0;
    P.p0 = d->p0;
    P.theta0 = d->theta0;
    P.lamv = std::max(4.0 / 3.0, d->gamma / d->Pr) * d->mu;
    P.dTdz = d->gravity ? -d->g / P.cp : 0.0;
    const double L[3] = {d->Lx, d->Ly, Lz}, o[3] = {d->x0, d->y0, z0};
    const int nc[3] = {d->nx, d->ny, nz}, bc[3] = {d->bc_x, d->bc_y, bc_z};
    for (int c = 0; c < 3; ++c) {
        P.h[c] = L[c] / nc[c];
        P.inv_h[c] = 1.0 / P.h[c];
        P.org[c] = o[c];
        P.nc[c] = nc[c];
        P.bc[c] = bc[c];
        P.eta[c] = (2 * m->N + 1) / (P.h[c] * std::sqrt(M_PI / 2.0));
    }
    P.field = d->bc_field;
    if (int rc = dev3(m)) {
        delete m;
        return rc;
    }
    const int n = m->n, n3 = n * n * n;
    const size_t st = (size_t)m->cells * 5 * n3;
    m->part_blocks = (int)(((long long)m->cells * n3 + 255) / 256);
    const size_t nbg = 2 * (size_t)nz * n + 2 * (size_t)(nz + 1);
    if (cudaMalloc(&m->u, st * 8) != cudaSuccess || cudaMalloc(&m->rvol, st * 8) != cudaSuccess ||
        cudaMalloc(&m->trace, (size_t)m->cells * 6 * adg::kTr3 * n * n * 8) != cudaSuccess ||
        cudaMalloc(&m->bg, nbg * 8) != cudaSuccess || cudaMalloc(&m->part, (size_t)m->part_blocks * 8) != cudaSuccess) {
        cudaGetLastError();
        free3(m);
        return fail(ADG_ENOMEM, "adg3_create: device allocation failed");
    }
    // isentropic background (Eq. 6) at node heights and at horizontal faces
    std::vector<double> h(nbg, 0.0);
    if (d->gravity) {
        auto bgp = [&](double z, double& p, double& r) {
            const double ex = 1.0 - d->g * z / (P.cp * d->theta0);
            p = d->p0 * std::pow(ex, P.cp / d->R);
            r = p / (d->R * d->theta0 * ex);
        };
        const int nn = nz * n;
        for (int iz = 0; iz < nz; ++iz)
            for (int l = 0; l < n; ++l) bgp(z0 + (iz + m->B.xi[l]) * P.h[2], h[iz * n + l], h[nn + iz * n + l]);
        for (int k = 0; k <= nz; ++k) bgp(z0 + k * P.h[2], h[2 * nn + k], h[2 * nn + (nz + 1) + k]);
    }
    if (cudaMemcpy(m->bg, h.data(), nbg * 8, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemset(m->u, 0, st * 8) != cudaSuccess) {
        cudaGetLastError();
        free3(m);
        return fail(ADG_ECUDA, "adg3_create: initialisation failed");
    }
    if (d->precision == ADG_PREC_MIXED) {
        if (int rc = build_mixed3(m)) {
            free3(m);
            return rc;
        }
    }
    *out = m;
    return ADG_OK;
}

extern "C" void adg3_destroy(adg_mesh3* m) { free3(m); }

extern "C" size_t adg3_state_count(const adg_mesh3* m) {
    return m ? (size_t)m->cells * 5 * m->n * m->n * m->n : 0;
}

extern "C" int adg3_set_state(adg_mesh3* m, const double* u, size_t count, int on_device, void* stream) {
    if (!m || !u) return fail(ADG_EINVAL, "adg3_set_state: NULL argument");
    if (count != adg3_state_count(m)) return fail(ADG_EINVAL, "adg3_set_state: count mismatch");
    if (on_device < 0 || on_device > ADG_COPY_HOST_ASYNC) return fail(ADG_EINVAL, "bad on_device");
    if (int rc = dev3(m)) return rc;
    ADG_CK(cudaMemcpyAsync(m->u, u, count * 8, on_device == 1 ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice,
                           (cudaStream_t)stream),
           "adg3_set_state");
    if (on_device == 0) ADG_CK(cudaStreamSynchronize((cudaStream_t)stream), "adg3_set_state sync");
    return ADG_OK;
}

extern "C" int adg3_get_state(adg_mesh3* m, double* u, size_t count, int on_device, void* stream) {
    if (!m || !u) return fail(ADG_EINVAL, "adg3_get_state: NULL argument");
    if (count != adg3_state_count(m)) return fail(ADG_EINVAL, "adg3_get_state: count mismatch");
    if (on_device < 0 || on_device > ADG_COPY_HOST_ASYNC) return fail(ADG_EINVAL, "bad on_device");
    if (int rc = dev3(m)) return rc;
    ADG_CK(cudaMemcpyAsync(u, m->u, count * 8, on_device == 1 ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost,
                           (cudaStream_t)stream),
           "adg3_get_state");
    if (on_device == 0) ADG_CK(cudaStreamSynchronize((cudaStream_t)stream), "adg3_get_state sync");
    return ADG_OK;
}

extern "C" int adg3_set_time(adg_mesh3* m, double t) {
    if (!m || !std::isfinite(t)) return fail(ADG_EINVAL, "adg3_set_time: bad argument");
    m->t = t;
    return ADG_OK;
}

extern "C" double adg3_get_time(const adg_mesh3* m) { return m ? m->t : 0.0; }

extern "C" int adg3_init_scenario(adg_mesh3* m, const adg_scenario* s, void* stream) {
    if (!m || !s) return fail(ADG_EINVAL, "adg3_init_scenario: NULL argument");
    if (s->kind == ADG_SCEN_COSINE || s->kind == ADG_SCEN_BACKGROUND) {
        if (!m->d.gravity) return fail(ADG_EINVAL, "adg3_init_scenario: bubble scenarios need gravity");
        if (s->kind == ADG_SCEN_COSINE && !(s->a > 0.0)) return fail(ADG_EINVAL, "adg3_init_scenario: radius must be > 0");
    } else if (s->kind != ADG_SCEN_ABC) {
        return fail(ADG_EINVAL, "adg3_init_scenario: cosine bubble, background or ABC field");
    }
    if (int rc = dev3(m)) return rc;
    const long long total = (long long)m->cells * m->n * m->n * m->n;
    adg::k3_init<<<(unsigned)((total + 255) / 256), 256, 0, (cudaStream_t)stream>>>(
        m->u, m->cells, m->n, s->kind, s->A, s->a, s->xc, s->zc, m->t, m->B, m->P);
    ADG_CK(cudaGetLastError(), "adg3_init_scenario launch");
    return ADG_OK;
}

extern "C" int adg3_step(adg_mesh3* m, double dt, int nsteps, void* stream) {
    if (!m) return fail(ADG_EINVAL, "adg3_step: NULL argument");
    if (!(dt > 0.0) || !std::isfinite(dt) || nsteps < 1) return fail(ADG_EINVAL, "adg3_step: dt > 0, nsteps >= 1");
    if (int rc = dev3(m)) return rc;
    cudaStream_t s = (cudaStream_t)stream;
    const adg::Bg3 bg = bg3(m);
    for (int k = 0; k < nsteps; ++k) {
        int e = m->d.precision == ADG_PREC_MIXED
                    ? adg::launch3m_any(m->N, m->u, m->rvol, m->trace, m->cells, (float)dt, m->Bf, m->Pf, m->P,
                                        bg3m(m), s)
                    : adg::launch3_any(m->N, true, m->u, m->rvol, m->trace, m->cells, dt, m->t, m->B, m->P, bg, s,
                                       false, m->Pf);
        if (e) return cuda_fail((cudaError_t)e, "adg3_step predictor");
        e = adg::launch3_any(m->N, false, m->u, m->rvol, m->trace, m->cells, dt, m->t, m->B, m->P, bg, s,
                             m->d.precision == ADG_PREC_MIXED, m->Pf);
        if (e) return cuda_fail((cudaError_t)e, "adg3_step corrector");
        m->t += dt;
    }
    return ADG_OK;
}

extern "C" int adg3_stable_dt(adg_mesh3* m, double cfl, double* dt, void* stream) {
    if (!m || !dt) return fail(ADG_EINVAL, "adg3_stable_dt: NULL argument");
    if (!(cfl > 0.0)) return fail(ADG_EINVAL, "adg3_stable_dt: cfl must be > 0");
    if (int rc = dev3(m)) return rc;
    cudaStream_t s = (cudaStream_t)stream;
    const double h = std::min(m->P.h[0], std::min(m->P.h[1], m->P.h[2]));
    const double eta = (2 * m->N + 1) / (h * std::sqrt(M_PI / 2.0));
    adg::k3_speed<<<m->part_blocks, 256, 0, s>>>(m->u, m->cells, m->n, eta, m->part, m->B, m->P);
    ADG_CK(cudaGetLastError(), "adg3_stable_dt launch");
    std::vector<double> hp(m->part_blocks);
    ADG_CK(cudaMemcpyAsync(hp.data(), m->part, hp.size() * 8, cudaMemcpyDeviceToHost, s), "adg3_stable_dt copy");
    ADG_CK(cudaStreamSynchronize(s), "adg3_stable_dt sync");
    double lam = 0.0;
    for (double v : hp) lam = std::max(lam, v);
    if (!(lam > 0.0) || !std::isfinite(lam)) return fail(ADG_ENONFINITE, "adg3_stable_dt: non-finite or zero wave speed");
    *dt = cfl * h / (3.0 * (2 * m->N + 1) * lam);
    return ADG_OK;
}
