// FP64 predictor body shared by the uniform-mesh and batched kernels
// (adg_fp64.cu) and the adaptive-mesh kernels (adg_amr.cu).  See adg_fp64.cu
// for the method.
#pragma once
#include "adg_fixed.cuh"
#include "adg_internal.h"
#include "adg_physics.cuh"

namespace adg {

// One thread per space-time node (k, j, i) of a cell.  The FP64 pipe binds:
// every derivative and time contraction runs on the integer pipe instead
// (adg_fixed.cuh), and 46 FP64 operations per node and sweep are left, the
// point-wise fluxes.  A thread holds one time node, so a cell's sweep is one
// evaluation deep (a 9 x 9 mesh has a sixteenth of a wave of cells and is
// bound by that depth), and one cell fills 7 warps at degree 5.
template <int N>
struct FxCfg {
    static constexpr int n = N + 1, n2 = n * n, n3 = n2 * n;
    // threads per cell: whole warps, so that a group's largest magnitude is one
    // warp reduction and one shared-memory atomic per warp (degree 1: 8 lanes)
    static constexpr int tpc = n3 <= 8 ? 8 : (n3 + 31) / 32 * 32;
    static constexpr int cpb = N == 1 ? 16 : N == 2 ? 4 : N == 3 ? 2 : 1;
    static constexpr int threads = cpb * tpc;
    // Blocks per SM asked of the register allocator.  The phases of a block
    // alternate between the FP64 and the integer pipe, so blocks in other
    // phases keep both busy: spilling registers for them pays.  Measured (us a
    // step, 81x81 cells): degree 5 1447 / 1376 / 1293 / 1286 / 1309 / 1273 with 2
    // / 3 / 4 / 5 / 6 / 8 blocks, degree 6 2746 / 2552 / 2303 / 2340 with 2 / 3 / 4
    // / 5 (five, for meshes of four to five blocks an SM: 27x27 284 against 345),
    // degree 7 4496 / 4094 / 3965 with 2 / 3 / 4; degree 4 651 / 608 / 613 / 667
    // with 3 / 4 / 5 / 6; within 5% from 3 to 10 below.
    static constexpr int resident = N == 1 ? 5 : N <= 4 ? 4 : N == 5 ? 8 : N == 6 ? 5 : 4;
    // per cell, in 8-byte words: q (4) and the fluxes (5) of every space-time
    // node, the source of the time-dependent form (4), u, D/hx, D/hy, the
    // steady source (3), the face values of q-bar, the group magnitudes
    static constexpr int words(bool tsrc) { return (tsrc ? 13 : 9) * n3 + 9 * n2 + 16 * n + 7; }
    static constexpr size_t smem(bool tsrc) { return ((size_t)cpb * words(tsrc) + n2) * 8; }
};

// D / hx and D / hy of a cell in fixed point, each with its own exponent (a
// common one would cost the longer side of a stretched cell the bits of the
// aspect ratio), in shared memory: in registers the two rows of a node (24 at
// degree 5) leave two resident blocks, and the kernel waits on its own dependent
// chains (1.55 ms on the 81x81 degree-5 mesh).
template <int N>
struct FxRows {
    const Limbs *dx, *dy;  // [n][n]
    int ex, ey;            // exponents of the entries
    int shx, shy;          // |a row times a group| < 2^(57 + sh) in units of the product
    // by all threads tid of the cell; readers wait for a barrier
    __device__ __forceinline__ void make(const Basis& B, Limbs* tab, int tid, double inv_hx, double inv_hy) {
        constexpr int n = N + 1, n2 = n * n;
        ex = fx_exp(fx_mag(B.Dmax * inv_hx));
        ey = fx_exp(fx_mag(B.Dmax * inv_hy));
        shx = fx_row_shift(B.Drow * inv_hx, ex);
        shy = fx_row_shift(B.Drow * inv_hy, ey);
        dx = tab;
        dy = tab + n2;
        for (int a = tid; a < n2; a += FxCfg<N>::tpc) {
            const double d = B.D[a / n][a % n];
            tab[a] = fx_split_centred(fx_from(d * inv_hx, ex));
            tab[n2 + a] = fx_split_centred(fx_from(d * inv_hy, ey));
        }
    }
};

// Place of the FxRows table of group cl in the block's shared memory.
template <int N, bool TSRC>
__device__ __forceinline__ Limbs* fx_tab(double* sm, int cl) {
    using C = FxCfg<N>;
    return reinterpret_cast<Limbs*>(sm + (size_t)cl * C::words(TSRC) + (TSRC ? 13 : 9) * C::n3 + 4 * C::n2);
}

// The limbs of K1^{-1} W, one copy per block.
template <int N>
__device__ __forceinline__ void fx_time_table(Limbs* K, const Basis& B) {
    constexpr int n = N + 1;
    for (int a = threadIdx.x; a < n * n; a += blockDim.x) K[a] = Limbs{B.KwH[a / n][a % n], B.KwL[a / n][a % n]};
}

// Point-wise fluxes (Eqs. 1-5, 7) in 46 FP64 operations (48 with gravity's
// source): the mass fluxes are rho u and rho v themselves; rho u v + sigma_xy
// serves both momentum cross fluxes; with w = d(rho v) - v d(rho),
//   c_v rho grad T = grad E - (E/rho) grad rho - v.w - rho g e_z.
struct FxFlux {
    double f1, xy, f3, g2, g3;  // F[1], F[2] = G[1], F[3], G[2], G[3]
};
__device__ __forceinline__ FxFlux ns_flux5(const double q[4], const double gx[4], const double gy[4], double g, double gz,
                                           double pbar, double gm1, double mu, double mu23, double kR) {
    const double rho = q[0], mx = q[1], my = q[2], E = q[3];
    const double rinv = fx_rcp(rho);
    const double u = mx * rinv, v = my * rinv;
    const double ke2 = fma(my, v, mx * u);
    const double p = gm1 * fma(-0.5, ke2, fma(-gz, rho, E));
    const double eR = E * rinv;
    const double ux = fma(-u, gx[0], gx[1]), uy = fma(-u, gy[0], gy[1]);  // rho times the velocity gradient
    const double vx = fma(-v, gx[0], gx[2]), vy = fma(-v, gy[0], gy[2]);
    const double hx = fma(-v, vx, fma(-u, ux, fma(-eR, gx[0], gx[3])));
    const double hy = fma(-g, rho, fma(-v, vy, fma(-u, uy, fma(-eR, gy[0], gy[3]))));
    const double m23 = mu23 * rinv, kr = kR * rinv;
    const double sxx = m23 * fma(-2.0, ux, vy), syy = m23 * fma(-2.0, vy, ux);
    const double sxy = (-mu * rinv) * (uy + vx);
    const double pp = p - pbar, Ep = E + p;
    FxFlux o;
    o.f1 = fma(mx, u, pp + sxx);
    o.xy = fma(my, u, sxy);
    o.g2 = fma(my, v, pp + syy);
    o.f3 = fma(-kr, hx, fma(u, Ep + sxx, v * sxy));
    o.g3 = fma(-kr, hy, fma(v, Ep + syy, u * sxy));
    return o;
}

// Predictor of one cell by one group of FxCfg<N>::tpc threads (tid: thread of
// the group; all groups of the block run in step, inactive ones on a copy of a
// valid cell without stores).  The cell's geometry arrives as its lower-left
// corner (xorg, yorg) and the cell sizes in P (hx, hy and the penalty eta_x,
// eta_y); pbar, rhobar: background at this thread's node height; gmask: bit f
// set if the corrector needs grad q-bar on face f (a boundary side).  TSRC: the
// time-dependent manufactured source, evaluated at t + xi_k dt.  REC (local
// time stepping, adg_amr.cu): also the face values of every time node k of the
// final iterate, ttrace[cell][k][face][16][n] (q and the normal flux in the
// first eight), from which a finer neighbour forms the trace averaged over its
// own part of this cell's step.
//
// Shared memory of the cell: Q[v][k][node] and F[c][k][node] in limbs; the
// residual takes Q's place once every gradient is formed.  Every component of q
// and of the fluxes has its own exponent (one for the momenta and one for each
// kind of flux would hold a component to the largest of its kind only).
template <int N, bool TSRC = false, bool REC = false>
__device__ __forceinline__ void predictor_fp64_body(const double* __restrict__ u, double* __restrict__ rvol,
                                                    double* __restrict__ trace, int cell, bool active, int tid, double dt,
                                                    const Basis& B, const Phys& P, const FxRows<N>& O, const Limbs* K,
                                                    double xorg, double yorg, double pbar, double rhobar, unsigned gmask,
                                                    double* sm, double t = 0.0, double* __restrict__ ttrace = nullptr) {
    using C = FxCfg<N>;
    constexpr int n = C::n, n2 = C::n2, n3 = C::n3, SL = 4 * n2, NS = TSRC ? 13 : 9;
    const bool on = tid < n3;  // the rest of the last warp repeats the last node without stores
    const int id = on ? tid : n3 - 1;
    const int k = id / n2, node = id - k * n2, j = node / n, i = node - j * n;
    Limbs* Q = reinterpret_cast<Limbs*>(sm);
    Limbs* F = Q + 4 * n3;
    double* US = sm + NS * n3;
    double* SS = US + 6 * n2;
    double* TQ = SS + 3 * n2;
    uint32_t* mx = reinterpret_cast<uint32_t*>(TQ + 16 * n);  // magnitudes: q (4), fluxes (5), sources (z-momentum, 0, 1, 3)
    const double z = yorg + B.xi[j] * P.hy;
    const double g = P.gravity ? P.g : 0.0, gz = g * z;
    const double mu23 = (2.0 / 3.0) * P.mu, kR = P.gm1 * P.kappa * P.invR;

    double q[4], Sm[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int v = 0; v < 4; ++v) q[v] = u[(size_t)cell * SL + v * n2 + node];
    const bool has_src = TSRC || P.source != ADG_SRC_NONE;
    const double x = xorg + B.xi[i] * P.hx;
    if constexpr (TSRC) {
        paper_source(x, z, t + B.xi[k] * dt, P, Sm);
    } else if (has_src && id < n2 && on) {  // once per spatial node: a sine, a cosine and two divisions
        steady_source(x, z, P, Sm);
        SS[node] = Sm[0];
        SS[n2 + node] = Sm[1];  // = Sm[2]
        SS[2 * n2 + node] = Sm[3];
    }

    // largest magnitude of a group over the cell's threads
    auto push = [&](int slot, uint32_t m) {
        if constexpr (C::tpc >= 32) {
            m = __reduce_max_sync(0xffffffffu, m);
            if ((threadIdx.x & 31) == 0) atomicMax(mx + slot, m);
        } else {
#pragma unroll
            for (int o = 1; o < C::tpc; o *= 2) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
            if (tid == 0) mx[slot] = max(mx[slot], m);
        }
    };
    auto push_q = [&]() {
#pragma unroll
        for (int v = 0; v < 4; ++v) push(v, fx_mag(q[v]));
    };
    // Exponents of q (slots 0..3) and the fluxes (4..8), a phase's magnitudes cleared in the phase after the next
    // barrier.  From degree 5 on they are formed again wherever they are used: held through a sweep they would spill
    // (81x81 step, us: degree 5 1281 -> 1272, degree 7 4092 -> 3956; degree 2 with registers to spare 150 -> 148 held).
    int EE[9] = {};
    auto take = [&](int first, int end) {
        if constexpr (N <= 4) {
#pragma unroll
            for (int c = first; c < end; ++c) EE[c] = fx_exp(mx[c]);
        }
    };
    auto E = [&](int slot) { return N <= 4 && slot < 9 ? EE[slot] : fx_exp(mx[slot]); };
    auto store_q = [&](int slice) {
#pragma unroll
        for (int v = 0; v < 4; ++v) Q[(v * n + slice) * n2 + node] = fx_limbs(q[v], E(v));
    };
    for (int a = tid; a < 13; a += C::tpc) mx[a] = 0;
    __syncthreads();
    if (!TSRC && has_src) {
        Sm[0] = SS[node];
        Sm[1] = Sm[2] = SS[n2 + node];
        Sm[3] = SS[2 * n2 + node];
    }
    push_q();
    if (has_src) {
        push(10, fx_mag(Sm[0]));
        push(11, fx_mag(Sm[1]));
        push(12, fx_mag(Sm[3]));
    }
    __syncthreads();
    take(0, 4);
    if (id < n2 && on) {
        store_q(0);
#pragma unroll
        for (int v = 0; v < 4; ++v) US[v * n2 + node] = q[v];
    }
    __syncthreads();

    FxFlux f;
    // sweeps 0..n-1 and the final evaluation r = n; in sweep 0 the iterate is u
    // at every time node: the threads of time node 0 evaluate the fluxes
#pragma unroll 1
    for (int r = 0;; ++r) {
        const int ks = r == 0 ? 0 : k;
        const Limbs* Qk = Q + ks * n2;
        int ER[4];  // exponents of the residual: the largest of its two derivatives' and the source's
        const int dX = O.ex - 1022 + O.shx, dY = O.ey - 1022 + O.shy;
        ER[0] = max(max(E(1) + dX, E(2) + dY), has_src ? E(10) + 1 : 0);
        long long R[4];  // -dF/dx - dG/dy + S; the mass flux is the momentum
        f = FxFlux{0.0, 0.0, 0.0, 0.0, 0.0};
        if (r == 0 && k > 0) {
            FxSum a, b;
#pragma unroll
            for (int p = 0; p < n; ++p) {
                a.add(O.dx[i * n + p], Qk[n3 + j * n + p]);
                b.add(O.dy[j * n + p], Qk[2 * n3 + p * n + i]);
            }
            R[0] = -(a.value() >> fx_down(O.shx, ER[0], E(1) + dX)) - (b.value() >> fx_down(O.shy, ER[0], E(2) + dY));
        } else {
            double gx[4], gy[4];
            {
                FxSum a[4];
#pragma unroll
                for (int p = 0; p < n; ++p) {
                    const Limbs d = O.dx[i * n + p];
#pragma unroll
                    for (int v = 0; v < 4; ++v) a[v].add(d, Qk[v * n3 + j * n + p]);
                }
                R[0] = -(a[1].value() >> fx_down(O.shx, ER[0], E(1) + dX));
#pragma unroll
                for (int v = 0; v < 4; ++v) gx[v] = fx_to(a[v].value(), E(v) + O.ex - 2102);
            }
            {
                FxSum a[4];
#pragma unroll
                for (int p = 0; p < n; ++p) {
                    const Limbs d = O.dy[j * n + p];
#pragma unroll
                    for (int v = 0; v < 4; ++v) a[v].add(d, Qk[v * n3 + p * n + i]);
                }
                R[0] -= a[2].value() >> fx_down(O.shy, ER[0], E(2) + dY);
#pragma unroll
                for (int v = 0; v < 4; ++v) gy[v] = fx_to(a[v].value(), E(v) + O.ey - 2102);
            }
            f = ns_flux5(q, gx, gy, g, gz, pbar, P.gm1, P.mu, mu23, kR);
        }
        if (r == n) break;
        double S2 = Sm[2];
        if (P.gravity) S2 = fma(-g, q[0] - rhobar, S2);
        const double fl[5] = {f.f1, f.xy, f.f3, f.g2, f.g3};
#pragma unroll
        for (int c = 0; c < 5; ++c) push(4 + c, fx_mag(fl[c]));
        if (has_src || P.gravity) push(9, fx_mag(S2));
        __syncthreads();
        take(4, 9);
        if (tid < 4) mx[tid] = 0;
        if (on && (r > 0 || k == 0)) {
#pragma unroll
            for (int c = 0; c < 5; ++c) F[(c * n + k) * n2 + node] = fx_limbs(fl[c], E(4 + c));
        }
        __syncthreads();
        // residual, in Q's place
        {
            // fluxes of residual v: F1 XY F3 along x, XY G2 G3 along y
            auto X = [&](int v) { return E(3 + v) + dX; };
            auto Y = [&](int v) { return E(v == 1 ? 5 : 5 + v) + dY; };
            ER[1] = max(max(X(1), Y(1)), has_src ? E(11) + 1 : 0);
            ER[2] = max(max(X(2), Y(2)), has_src || P.gravity ? E(9) + 1 : 0);
            ER[3] = max(max(X(3), Y(3)), has_src ? E(12) + 1 : 0);
            {
                FxSum a[3];
                const Limbs* Fx = F + ks * n2 + j * n;
#pragma unroll
                for (int p = 0; p < n; ++p) {
                    const Limbs d = O.dx[i * n + p];
#pragma unroll
                    for (int v = 0; v < 3; ++v) a[v].add(d, Fx[v * n3 + p]);
                }
#pragma unroll
                for (int v = 1; v < 4; ++v) R[v] = -(a[v - 1].value() >> fx_down(O.shx, ER[v], X(v)));
            }
            {
                FxSum a[3];
                const Limbs* Gy = F + ks * n2 + i;
#pragma unroll
                for (int p = 0; p < n; ++p) {
                    const Limbs d = O.dy[j * n + p];
                    a[0].add(d, Gy[n3 + p * n]);
                    a[1].add(d, Gy[3 * n3 + p * n]);
                    a[2].add(d, Gy[4 * n3 + p * n]);
                }
#pragma unroll
                for (int v = 1; v < 4; ++v) R[v] -= a[v - 1].value() >> fx_down(O.shy, ER[v], Y(v));
            }
        }
        if (has_src) {
            R[0] += fx_from(Sm[0], ER[0]);
            R[1] += fx_from(Sm[1], ER[1]);
            R[3] += fx_from(Sm[3], ER[3]);
        }
        if (has_src || P.gravity) R[2] += fx_from(S2, ER[2]);
        if (on) {
#pragma unroll
            for (int v = 0; v < 4; ++v) Q[(v * n + k) * n2 + node] = fx_split(R[v]);
        }
        __syncthreads();
        // time contraction: this thread's time node of the next iterate
        {
            FxSum a[4];
#pragma unroll
            for (int kk = 0; kk < n; ++kk) {
                const Limbs d = K[k * n + kk];
#pragma unroll
                for (int v = 0; v < 4; ++v) a[v].add(d, Q[(v * n + kk) * n2 + node]);
            }
#pragma unroll
            for (int v = 0; v < 4; ++v)
                q[v] = fma(dt, fx_to(a[v].value(), ER[v] + B.KwE - 2102), US[v * n2 + node]);
        }
        push_q();
        __syncthreads();
        take(0, 4);
        if (tid < 6) mx[4 + tid] = 0;
        if (on) store_q(k);
        __syncthreads();
    }

    // time averages: slots q (4), F1, XY, F3, G2, G3, then the time-dependent source
    double* A = sm;
    __syncthreads();
    if (on) {
#pragma unroll
        for (int v = 0; v < 4; ++v) A[(v * n + k) * n2 + node] = q[v];
        double* Af = A + (4 * n + k) * n2 + node;
        Af[0] = f.f1;
        Af[n3] = f.xy;
        Af[2 * n3] = f.f3;
        Af[3 * n3] = f.g2;
        Af[4 * n3] = f.g3;
        if constexpr (TSRC) {
#pragma unroll
            for (int v = 0; v < 4; ++v) Af[(5 + v) * n3] = Sm[v];
        }
    }
    __syncthreads();
    // slot of component c of a face record: q, then the normal flux (mass flux = rho v_n)
    auto slot = [](int c, bool xface) {
        return c < 4 ? c : c == 4 ? (xface ? 1 : 2) : xface ? c - 1 : c == 5 ? 5 : c + 1;
    };
    if constexpr (REC) {
        for (int o = tid; o < n * 4 * 8 * n; o += C::tpc) {
            const int m = o % n, c = o / n % 8, fc = o / (8 * n) % 4, kk = o / (32 * n);
            const bool xface = fc < 2;
            const double* phi = (fc == 0 || fc == 2) ? B.phi1 : B.phi0;
            const double* S = A + (slot(c, xface) * n + kk) * n2 + (xface ? m * n : m);
            double s = 0.0;
#pragma unroll
            for (int p = 0; p < n; ++p) s += phi[p] * S[xface ? p : p * n];
            if (active) ttrace[((((size_t)cell * n + kk) * 4 + fc) * 16 + c) * n + m] = s;
        }
        __syncthreads();
    }
    if (on)
        for (int s = k; s < NS; s += n) {
            double a = 0.0;
#pragma unroll
            for (int kk = 0; kk < n; ++kk) a = fma(B.w[kk], A[(s * n + kk) * n2 + node], a);
            A[s * n3 + node] = a;  // time node 0's place, read by this thread alone
        }
    __syncthreads();
    if (on && active) {
        for (int v = k; v < 4; v += n) {
            const double* Ax = A + slot(4 + v, true) * n3 + j * n;
            const double* Ay = A + slot(4 + v, false) * n3 + i;
            double sx = 0.0, sy = 0.0;
#pragma unroll
            for (int p = 0; p < n; ++p) {
                sx = fma(B.Vx[p][i], Ax[p], sx);
                sy = fma(B.Vx[p][j], Ay[p * n], sy);
            }
            double S;
            if constexpr (TSRC) S = A[(9 + v) * n3 + node];
            else S = v == 0 ? Sm[0] : v == 1 ? Sm[1] : v == 2 ? Sm[2] : Sm[3];
            if (P.gravity && v == 2) S = fma(-g, A[node] - rhobar, S);
            rvol[(size_t)cell * SL + v * n2 + node] = fma(sx, P.inv_hx, fma(sy, P.inv_hy, S));
        }
    }
    // boundary-extrapolated traces: faces E, W (x = const), N, S (y = const)
    for (int o = tid; o < 4 * 8 * n; o += C::tpc) {
        const int m = o % n, c = o / n % 8, fc = o / (8 * n);
        const bool xface = fc < 2;
        const double* phi = (fc == 0 || fc == 2) ? B.phi1 : B.phi0;
        const double* S = A + slot(c, xface) * n3 + (xface ? m * n : m);
        double s = 0.0;
#pragma unroll
        for (int p = 0; p < n; ++p) s = fma(phi[p], S[xface ? p : p * n], s);
        if (c < 4) TQ[(fc * 4 + c) * n + m] = s;
        if (active) trace[(((size_t)cell * 4 + fc) * kTraceComps + c) * n + m] = s;
    }
    __syncthreads();
    for (int o = tid; o < 4 * n; o += C::tpc) {
        const int fc = o / n, m = o - fc * n;
        const bool xface = fc < 2;
        double rec[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) rec[v] = TQ[(fc * 4 + v) * n + m];
        const double zf = xface ? yorg + B.xi[m] * P.hy : yorg + (fc == 2 ? P.hy : 0.0);
        if (active) trace[(((size_t)cell * 4 + fc) * kTraceComps + 16) * n + m] = wave_speed(rec, zf, xface, P);
    }
    // grad q-bar on boundary sides: along the normal from the cell's nodes,
    // along the face from the face's own values
    if (gmask && active) {
        for (int o = tid; o < 4 * 8 * n; o += C::tpc) {
            const int m = o % n, c = o / n % 8, fc = o / (8 * n), v = c & 3;
            if (!(gmask >> fc & 1u)) continue;
            const bool xface = fc < 2, normal = xface == (c < 4);
            const double* w = normal ? ((fc == 0 || fc == 2) ? B.dphi1 : B.dphi0) : B.D[m];
            const double* S = normal ? A + v * n3 + (xface ? m * n : m) : TQ + (fc * 4 + v) * n;
            const int st = normal && !xface ? n : 1;
            double s = 0.0;
#pragma unroll
            for (int p = 0; p < n; ++p) s = fma(w[p], S[p * st], s);
            trace[(((size_t)cell * 4 + fc) * kTraceComps + 8 + c) * n + m] = s * (c < 4 ? P.inv_hx : P.inv_hy);
        }
    }
}

}  // namespace adg
