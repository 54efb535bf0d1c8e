// Discrete adjoint of one FP64 ADER-DG step (predictor + corrector).
//
// The forward step is u' = u + dt (rvol(u) - lift(F*(traces(u)))), with the
// predictor (Picard sweeps, Sec. 3) local to each cell and the corrector
// coupling neighbours through the face traces.  Given lam' = dJ/du', the
// adjoint returns lam = dJ/du = lam' + (d(rvol, traces)/du)^T (rvol_bar,
// trace_bar), in two kernels:
//
//  k_corrector_adj_fp64  per cell and face: the adjoint of the face flux F*
//      (lift rows of both cells sharing the face), then of the Rusanov-type
//      flux and, on walls, of the ghost state, giving trace_bar of the cell's
//      own traces (no scatter: each face record belongs to one cell).
//  k_predictor_adj_fp64  per cell: recompute the Picard iterates q^(0..n)
//      into shared memory, then run the predictor backwards: face
//      extrapolation and wave speed, weak volume residual, time averages and
//      final evaluation, and the n sweeps, each through the hand-written
//      reverse of the point-wise flux (ns_flux5_adj).  One thread per
//      space-time node, contractions on the integer pipe, as the forward
//      predictor (adg_fp64_body.cuh, adg_fixed.cuh).
//
// Non-smooth points take one-sided derivatives: max(s_L, s_R) differentiates
// into s_L on ties, |v.n| into sign(v.n) (0 at 0).
#include <cuda_runtime.h>

#include "adg_fp64_body.cuh"
#include "adg_internal.h"
#include "adg_physics.cuh"

namespace adg {

// Predictor adjoint: the thread layout of the forward predictor (FxCfg: one
// thread per space-time node), its contractions on the integer pipe.
template <int N>
struct AdjCfg {
    using F = FxCfg<N>;
    static constexpr int n = F::n, n2 = F::n2, n3 = F::n3;
    static constexpr int cpb = F::cpb, tpc = F::tpc, threads = F::threads;
    static constexpr int resident = 2;  // blocks per SM asked of the register allocator (2 .. 8 within 1%)
    // per cell, in 8-byte words: the limbs of the iterate q^(0) (one time slice);
    // the iterates q^(1..n), limbs while a sweep contracts them and doubles in
    // between (so that the reverse works on the states of the forward, not on
    // their 58-bit images); a work area (fluxes and residual forward; adjoints
    // of q, of the residual and of the gradients backward); u; D/h and -dt D/h;
    // the adjoints of the face records; iterate exponents and group magnitudes
    static constexpr int work = 8 * n3 > 20 * n2 ? 8 * n3 : 20 * n2;
    static constexpr int words = 4 * n2 + 4 * n * n3 + work + 4 * n2 + 4 * n2 + 64 * n + 2 * (n + 1) + 13;
    static constexpr size_t smem = ((size_t)cpb * words + n2 + n) * 8;
};

// ------------------------------------------------------------------ corrector
template <int N, int CPB>
__global__ void __launch_bounds__(CPB*(N + 1) * (N + 1))
k_corrector_adj_fp64(const double* __restrict__ lam, const double* __restrict__ trace,
                     double* __restrict__ trace_bar, int cells, double dt, const Basis B, const Phys P,
                     const Background bg) {
    constexpr int n = N + 1, n2 = n * n, SL = 4 * n2, TR = kTraceComps * n;
    const int cl = threadIdx.x / n2;
    const int node = threadIdx.x - cl * n2;
    const int cell_raw = blockIdx.x * CPB + cl;
    if (cell_raw >= cells) return;  // no barriers in this kernel
    const int cell = cell_raw;
    const int ix = cell % P.nx, iy = cell / P.nx;
    for (int idx = node; idx < 4 * n; idx += n2) {
        const int f = idx / n, m = idx - f * n;
        const bool xface = f < 2;
        const bool wall = xface ? (P.bc_x == ADG_BC_WALL && ((f == 0 && ix == P.nx - 1) || (f == 1 && ix == 0)))
                                : (P.bc_y == ADG_BC_WALL && ((f == 2 && iy == P.ny - 1) || (f == 3 && iy == 0)));
        int nb = -1, nf = -1;
        if (f == 0) { nb = iy * P.nx + (ix + 1 == P.nx ? 0 : ix + 1); nf = 1; }
        else if (f == 1) { nb = iy * P.nx + (ix == 0 ? P.nx - 1 : ix - 1); nf = 0; }
        else if (f == 2) { nb = (iy + 1 == P.ny ? 0 : iy + 1) * P.nx + ix; nf = 3; }
        else { nb = (iy == 0 ? P.ny - 1 : iy - 1) * P.nx + ix; nf = 2; }
        // adjoint of the face value F*: lift rows of the own cell and, on an
        // interior face, of the neighbour that uses the same value
        const double* lo = lam + (size_t)cell * SL;
        double Fb[4];
        auto lift_row = [&](const double* L, int face, double out[4], double sign_acc) {
            // contribution of cell L's use of its face `face` at node m
            const double* w = (face == 0 || face == 2) ? B.lift1 : B.lift0;
            const double sgn = (face == 0 || face == 2) ? -1.0 : 1.0;
            const double h = (face < 2) ? P.inv_hx : P.inv_hy;
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                double s = 0.0;
#pragma unroll
                for (int p = 0; p < n; ++p) s += w[p] * (face < 2 ? L[v * n2 + m * n + p] : L[v * n2 + p * n + m]);
                out[v] += sign_acc * sgn * dt * h * s;
            }
        };
#pragma unroll
        for (int v = 0; v < 4; ++v) Fb[v] = 0.0;
        lift_row(lo, f, Fb, 1.0);
        if (!wall) lift_row(lam + (size_t)nb * SL, nf, Fb, 1.0);

        const double* own = trace + ((size_t)cell * 4 + f) * TR;
        double rec[kTraceComps];
#pragma unroll
        for (int c = 0; c < kTraceComps; ++c) rec[c] = own[c * n + m];
        double qo[4] = {rec[0], rec[1], rec[2], rec[3]};
        double qn[4], fn[4], sn;
        double z = 0.0, pb = 0.0, rb = 0.0;
        if (wall) {
            if (xface) {
                z = P.y0 + (iy + B.xi[m]) * P.hy;
                pb = bg.pbar_node[iy * n + m];
                rb = bg.rhobar_node[iy * n + m];
            } else {
                const int fi = iy + (f == 2 ? 1 : 0);
                z = P.y0 + fi * P.hy;
                pb = bg.pbar_face[fi];
                rb = bg.rhobar_face[fi];
            }
            // ghost (as in the forward wall_ghost)
            const double nx = f == 0 ? 1.0 : f == 1 ? -1.0 : 0.0;
            const double ny = f == 2 ? 1.0 : f == 3 ? -1.0 : 0.0;
            const double mn = rec[1] * nx + rec[2] * ny;
            qn[1] = rec[1] - 2.0 * mn * nx;
            qn[2] = rec[2] - 2.0 * mn * ny;
            qn[0] = P.gravity ? rb : rec[0];
            qn[3] = P.gravity ? pb / P.gm1 + rb * P.g * z : rec[3];
            Flux4 fl;
            ns_flux(qn, rec + 8, rec + 12, z, pb, rb, P, fl, true, 0.0, P.gravity ? -P.g / P.cp : 0.0);
#pragma unroll
            for (int v = 0; v < 4; ++v) fn[v] = xface ? fl.F[v] : fl.G[v];
            sn = wave_speed(qn, z, xface, P);
        } else {
            const double* ot = trace + ((size_t)nb * 4 + nf) * TR;
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                qn[v] = ot[v * n + m];
                fn[v] = ot[(4 + v) * n + m];
            }
            sn = ot[16 * n + m];
        }
        const bool own_left = (f == 0 || f == 2);
        const double sL = own_left ? rec[16] : sn, sR = own_left ? sn : rec[16];
        const double* qL = own_left ? qo : qn;
        const double* qR = own_left ? qn : qo;
        const double s = fmax(sL, sR);
        // Rusanov adjoint
        double s_b = 0.0;
        double q_own_b[4], f_own_b[4], q_oth_b[4], f_oth_b[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            s_b += -0.5 * (qR[v] - qL[v]) * Fb[v];
            f_own_b[v] = 0.5 * Fb[v];
            f_oth_b[v] = 0.5 * Fb[v];
            const double qR_b = -0.5 * s * Fb[v], qL_b = 0.5 * s * Fb[v];
            q_own_b[v] = own_left ? qL_b : qR_b;
            q_oth_b[v] = own_left ? qR_b : qL_b;
        }
        const bool left_wins = sL >= sR;
        double s_own_b = ((left_wins && own_left) || (!left_wins && !own_left)) ? s_b : 0.0;
        const double s_oth_b = s_b - s_own_b;
        double gxb[4] = {0, 0, 0, 0}, gyb[4] = {0, 0, 0, 0};
        if (wall) {
            // ghost flux, ghost speed and ghost state back to the own trace
            double qGb[4] = {0, 0, 0, 0};
            wave_speed_adj(qn, z, xface, P, s_oth_b, qGb);
            const double zero4[4] = {0, 0, 0, 0};
            ns_flux_adj(qn, rec + 8, rec + 12, z, P, xface ? f_oth_b : zero4, xface ? zero4 : f_oth_b, zero4, qGb,
                        gxb, gyb, true);
#pragma unroll
            for (int v = 0; v < 4; ++v) qGb[v] += q_oth_b[v];
            const double nx = f == 0 ? 1.0 : f == 1 ? -1.0 : 0.0;
            const double ny = f == 2 ? 1.0 : f == 3 ? -1.0 : 0.0;
            // qG1 = q1 - 2 (q1 nx + q2 ny) nx, qG2 = q2 - 2 (q1 nx + q2 ny) ny
            const double mnb = -2.0 * (qGb[1] * nx + qGb[2] * ny);
            q_own_b[1] += qGb[1] + mnb * nx;
            q_own_b[2] += qGb[2] + mnb * ny;
            if (!P.gravity) {
                q_own_b[0] += qGb[0];
                q_own_b[3] += qGb[3];
            }
        }
        double* ob = trace_bar + ((size_t)cell * 4 + f) * TR;
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            ob[v * n + m] = q_own_b[v];
            ob[(4 + v) * n + m] = f_own_b[v];
            ob[(8 + v) * n + m] = gxb[v];
            ob[(12 + v) * n + m] = gyb[v];
        }
        ob[16 * n + m] = s_own_b;
    }
}

// ------------------------------------------------------------------ predictor
// Adjoint of ns_flux5: given the adjoints of the fluxes (Fb, Gb; F[2] and G[1]
// are one value) and of the z-momentum source (Sb2), adds the adjoints of the
// state and its gradients.  Written line by line against ns_flux5.
__device__ __forceinline__ void ns_flux5_adj(const double q[4], const double gx[4], const double gy[4], double g, double gz,
                                             double gm1, double mu, double mu23, double kR, const double Fb[4],
                                             const double Gb[4], double Sb2, double qb[4], double gxb[4], double gyb[4]) {
    const double rho = q[0], mx = q[1], my = q[2], E = q[3];
    const double r = fx_rcp(rho);
    const double u = mx * r, v = my * r;
    const double p = gm1 * fma(-0.5, fma(my, v, mx * u), fma(-gz, rho, E));
    const double Ep = E + p, eR = E * r;
    const double ux = fma(-u, gx[0], gx[1]), uy = fma(-u, gy[0], gy[1]);
    const double vx = fma(-v, gx[0], gx[2]), vy = fma(-v, gy[0], gy[2]);
    const double hx = fma(-v, vx, fma(-u, ux, fma(-eR, gx[0], gx[3])));
    const double hy = fma(-g, rho, fma(-v, vy, fma(-u, uy, fma(-eR, gy[0], gy[3]))));
    const double m23 = mu23 * r, kr = kR * r, A = -mu * r;
    const double X = fma(-2.0, ux, vy), Y = fma(-2.0, vy, ux), Z = uy + vx;
    const double sxx = m23 * X, syy = m23 * Y, sxy = A * Z;
    // fluxes
    const double a1 = Fb[1], a3 = Fb[3], b2 = Gb[2], b3 = Gb[3], xb = Fb[2] + Gb[1];
    const double sxxb = fma(a3, u, a1), syyb = fma(b3, v, b2), sxyb = fma(b3, u, fma(a3, v, xb));
    const double Epb = fma(b3, v, a3 * u), pb = gm1 * (Epb + (a1 + b2));
    const double ke = -0.5 * pb;
    double mxb = fma(u, ke, fma(a1, u, Fb[0])), myb = fma(v, ke, fma(b2, v, fma(xb, u, Gb[0])));
    double ub = fma(mx, ke, fma(b3, sxy, fma(a3, Ep + sxx, fma(xb, my, a1 * mx))));
    double vb = fma(my, ke, fma(a3, sxy, fma(b3, Ep + syy, b2 * my)));
    // heat flux, stresses
    const double hxb = -kr * a3, hyb = -kr * b3;
    const double t1 = m23 * sxxb, t2 = m23 * syyb, t3 = A * sxyb;
    const double uxb = fma(-u, hxb, fma(-2.0, t1, t2)), vyb = fma(-v, hyb, fma(-2.0, t2, t1));
    const double uyb = fma(-u, hyb, t3), vxb = fma(-v, hxb, t3);
    ub -= fma(gy[0], uyb, fma(gx[0], uxb, fma(uy, hyb, ux * hxb)));
    vb -= fma(gy[0], vyb, fma(gx[0], vxb, fma(vy, hyb, vx * hxb)));
    const double eRb = -fma(gy[0], hyb, gx[0] * hxb);
    double rb = fma(mu23, fma(syyb, Y, sxxb * X), -mu * (sxyb * Z));
    rb = fma(-kR, fma(hy, b3, hx * a3), rb);
    rb = fma(my, vb, fma(mx, ub, fma(E, eRb, rb)));
    qb[0] += fma(-r, r * rb, fma(-gz, pb, -g * (hyb + Sb2)));
    qb[1] += fma(r, ub, mxb);
    qb[2] += fma(r, vb, myb);
    qb[3] += fma(r, eRb, Epb + pb);
    gxb[0] -= fma(v, vxb, fma(u, uxb, eR * hxb));
    gyb[0] -= fma(v, vyb, fma(u, uyb, eR * hyb));
    gxb[1] += uxb;
    gyb[1] += uyb;
    gxb[2] += vxb;
    gyb[2] += vyb;
    gxb[3] += hxb;
    gyb[3] += hyb;
}

// One cell per group of tpc threads (all groups of the block in step).  The
// iterates of the forward sweeps stay in shared memory as limbs, from which
// the reverse sweeps form the gradients and the node's own state again.
template <int N>
__global__ void __launch_bounds__(AdjCfg<N>::threads, AdjCfg<N>::resident)
k_predictor_adj_fp64(const double* __restrict__ u, const double* __restrict__ lam,
                     const double* __restrict__ trace, const double* __restrict__ trace_bar,
                     double* __restrict__ lam_out, int cells, double dt, const Basis B, const Phys P,
                     const Background bg) {
    using C = AdjCfg<N>;
    constexpr int n = C::n, n2 = C::n2, n3 = C::n3, SL = 4 * n2, TR = kTraceComps * n;
    extern __shared__ double sm[];
    const int cl = threadIdx.x / C::tpc, tid = threadIdx.x - cl * C::tpc;
    const bool on = tid < n3;
    const int id = on ? tid : n3 - 1;
    const int k = id / n2, node = id - k * n2, j = node / n, i = node - j * n;
    double* base = sm + (size_t)cl * C::words;
    Limbs* U0 = reinterpret_cast<Limbs*>(base);  // q^(0) [4][n2]
    Limbs* IT = U0 + 4 * n2;                     // q^(r) at IT + (r - 1) 4 n3, [4][n][n2]
    double* Wd = base + 4 * n2 + 4 * n * n3;
    Limbs* W = reinterpret_cast<Limbs*>(Wd);
    double* US = Wd + C::work;                            // u [4][n2]
    Limbs* DT = reinterpret_cast<Limbs*>(US + 4 * n2);    // D/hx, D/hy [n][n]
    Limbs* DM = DT + 2 * n2;                              // -dt D/hx, -dt D/hy
    double* FR = US + 8 * n2;                             // adjoints of the face records [4][16][n]
    int* EX = reinterpret_cast<int*>(FR + 64 * n);        // exponents of the iterates [n + 1][4]
    // magnitudes; forward: q (4), fluxes (5), sources (z-momentum, 0, 1, 3); reverse, from 13: adjoints of the
    // gradients along x (4) and y (4), of the iterate (4)
    uint32_t* mx = reinterpret_cast<uint32_t*>(EX + 4 * (n + 1));
    Limbs* K = reinterpret_cast<Limbs*>(sm + (size_t)C::cpb * C::words);  // [n][n], then the row sums [n]
    fx_time_table<N>(K, B);
    for (int a = threadIdx.x; a < n; a += blockDim.x) K[n2 + a] = fx_split_centred(fx_from(B.Kw1[a], B.KwE + 3));
    const double dmx = B.Dmax * P.inv_hx, dmy = B.Dmax * P.inv_hy;
    const int ex = fx_exp(fx_mag(dmx)), ey = fx_exp(fx_mag(dmy));
    const int emx = fx_exp(fx_mag(dmx * dt)), emy = fx_exp(fx_mag(dmy * dt));
    const int shx = fx_row_shift(B.Drow * P.inv_hx, ex), shy = fx_row_shift(B.Drow * P.inv_hy, ey);
    for (int a = tid; a < n2; a += C::tpc) {
        const double dx = B.D[a / n][a % n] * P.inv_hx, dy = B.D[a / n][a % n] * P.inv_hy;
        DT[a] = fx_split_centred(fx_from(dx, ex));
        DT[n2 + a] = fx_split_centred(fx_from(dy, ey));
        DM[a] = fx_split_centred(fx_from(-dt * dx, emx));
        DM[n2 + a] = fx_split_centred(fx_from(-dt * dy, emy));
    }
    const int cell_raw = blockIdx.x * C::cpb + cl;
    const bool active = cell_raw < cells;
    const int cell = active ? cell_raw : cells - 1;
    const int ix = cell % P.nx, iy = cell / P.nx;
    const double x = P.x0 + (ix + B.xi[i]) * P.hx, z = P.y0 + (iy + B.xi[j]) * P.hy;
    const double pbar = bg.pbar_node[iy * n + j], rhobar = bg.rhobar_node[iy * n + j];
    const double g = P.gravity ? P.g : 0.0, gz = g * z;
    const double mu23 = (2.0 / 3.0) * P.mu, kR = P.gm1 * P.kappa * P.invR;
    const bool has_src = P.source == ADG_SRC_STEADY;
    double Sm[4] = {0.0, 0.0, 0.0, 0.0};
    if (has_src) steady_source(x, z, P, Sm);

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
    // gradients at this node from the limbs of an iterate's time slice (plane stride ps); mx0, my0: the
    // derivatives of the mass flux as they come
    auto gradients = [&](const Limbs* Qk, int ps, const int* eq, double gx[4], double gy[4], long long& mx0,
                         long long& my0) {
        FxSum a[4], b[4];
#pragma unroll
        for (int p = 0; p < n; ++p) {
            const Limbs d = DT[i * n + p];
#pragma unroll
            for (int v = 0; v < 4; ++v) a[v].add(d, Qk[v * ps + j * n + p]);
        }
        mx0 = a[1].value();
#pragma unroll
        for (int v = 0; v < 4; ++v) gx[v] = fx_to(a[v].value(), eq[v] + ex - 2102);
#pragma unroll
        for (int p = 0; p < n; ++p) {
            const Limbs d = DT[n2 + j * n + p];
#pragma unroll
            for (int v = 0; v < 4; ++v) b[v].add(d, Qk[v * ps + p * n + i]);
        }
        my0 = b[2].value();
#pragma unroll
        for (int v = 0; v < 4; ++v) gy[v] = fx_to(b[v].value(), eq[v] + ey - 2102);
    };

    // ---------------- forward recompute of the iterates (as k_predictor_fp64)
    double q[4];
#pragma unroll
    for (int v = 0; v < 4; ++v) q[v] = u[(size_t)cell * SL + v * n2 + node];
    for (int a = tid; a < 25; a += C::tpc) mx[a] = 0;
    __syncthreads();
    auto push_q = [&]() {
#pragma unroll
        for (int v = 0; v < 4; ++v) push(v, fx_mag(q[v]));
    };
    push_q();
    if (has_src) {
        push(10, fx_mag(Sm[0]));
        push(11, fx_mag(Sm[1]));
        push(12, fx_mag(Sm[3]));
    }
    __syncthreads();
    if (tid < 4) EX[tid] = fx_exp(mx[tid]);
    if (on && k == 0) {
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            U0[v * n2 + node] = fx_limbs(q[v], fx_exp(mx[v]));
            US[v * n2 + node] = q[v];
        }
    }
    __syncthreads();
    if (tid < 4) mx[tid] = 0;
#pragma unroll 1
    for (int r = 0; r < n; ++r) {
        const int ks = r == 0 ? 0 : k, ps = r == 0 ? n2 : n3;
        const Limbs* Qk = r == 0 ? U0 : IT + (r - 1) * 4 * n3 + k * n2;
        int eq[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) eq[v] = EX[4 * r + v];
        double gx[4], gy[4];
        long long R0, R0y;
        gradients(Qk, ps, eq, gx, gy, R0, R0y);
        FxFlux f{0.0, 0.0, 0.0, 0.0, 0.0};
        if (r > 0 || k == 0) f = ns_flux5(q, gx, gy, g, gz, pbar, P.gm1, P.mu, mu23, kR);
        double S2 = Sm[2];
        if (P.gravity) S2 = fma(-g, q[0] - rhobar, S2);
        const double fl[5] = {f.f1, f.xy, f.f3, f.g2, f.g3};
#pragma unroll
        for (int c = 0; c < 5; ++c) push(4 + c, fx_mag(fl[c]));
        if (has_src || P.gravity) push(9, fx_mag(S2));
        __syncthreads();
        int EF[5], ER[4];
#pragma unroll
        for (int c = 0; c < 5; ++c) EF[c] = fx_exp(mx[4 + c]);
        const int ES2 = has_src || P.gravity ? fx_exp(mx[9]) + 1 : 0;
        if (on && (r > 0 || k == 0)) {
#pragma unroll
            for (int c = 0; c < 5; ++c) W[(c * n + k) * n2 + node] = fx_limbs(fl[c], EF[c]);
        }
        if (on && r > 0) {  // every gradient is formed: the iterate itself in place of its limbs
            double* Qd = reinterpret_cast<double*>(IT + (r - 1) * 4 * n3);
#pragma unroll
            for (int v = 0; v < 4; ++v) Qd[(v * n + k) * n2 + node] = q[v];
        }
        __syncthreads();
        if (tid < 6) mx[4 + tid] = 0;
        Limbs* Rn = IT + r * 4 * n3;  // the next iterate's place holds the residual first
        {
            const int dX = ex - 1022 + shx, dY = ey - 1022 + shy;
            const int X[4] = {eq[1] + dX, EF[0] + dX, EF[1] + dX, EF[2] + dX};
            const int Y[4] = {eq[2] + dY, EF[1] + dY, EF[3] + dY, EF[4] + dY};
            const int ES[4] = {has_src ? fx_exp(mx[10]) + 1 : 0, has_src ? fx_exp(mx[11]) + 1 : 0, ES2,
                               has_src ? fx_exp(mx[12]) + 1 : 0};
#pragma unroll
            for (int v = 0; v < 4; ++v) ER[v] = max(max(X[v], Y[v]), ES[v]);
            FxSum a[3], b[3];
            const Limbs* Fx = W + ks * n2 + j * n;
            const Limbs* Gy = W + ks * n2 + i;
#pragma unroll
            for (int p = 0; p < n; ++p) {
                const Limbs d = DT[i * n + p];
#pragma unroll
                for (int v = 0; v < 3; ++v) a[v].add(d, Fx[v * n3 + p]);
            }
#pragma unroll
            for (int p = 0; p < n; ++p) {
                const Limbs d = DT[n2 + j * n + p];
                b[0].add(d, Gy[n3 + p * n]);
                b[1].add(d, Gy[3 * n3 + p * n]);
                b[2].add(d, Gy[4 * n3 + p * n]);
            }
            long long R[4];
            R[0] = -(R0 >> fx_down(shx, ER[0], X[0])) - (R0y >> fx_down(shy, ER[0], Y[0]));
#pragma unroll
            for (int v = 1; v < 4; ++v)
                R[v] = -(a[v - 1].value() >> fx_down(shx, ER[v], X[v])) - (b[v - 1].value() >> fx_down(shy, ER[v], Y[v]));
            if (has_src) {
                R[0] += fx_from(Sm[0], ER[0]);
                R[1] += fx_from(Sm[1], ER[1]);
                R[3] += fx_from(Sm[3], ER[3]);
            }
            if (has_src || P.gravity) R[2] += fx_from(S2, ER[2]);
            if (on) {
#pragma unroll
                for (int v = 0; v < 4; ++v) Rn[(v * n + k) * n2 + node] = fx_split(R[v]);
            }
        }
        __syncthreads();
        {
            FxSum a[4];
#pragma unroll
            for (int kk = 0; kk < n; ++kk) {
                const Limbs d = K[k * n + kk];
#pragma unroll
                for (int v = 0; v < 4; ++v) a[v].add(d, Rn[(v * n + kk) * n2 + node]);
            }
#pragma unroll
            for (int v = 0; v < 4; ++v) q[v] = fma(dt, fx_to(a[v].value(), ER[v] + B.KwE - 2102), US[v * n2 + node]);
        }
        push_q();
        __syncthreads();
        if (tid < 4) EX[4 * (r + 1) + tid] = fx_exp(mx[tid]);
        if (on) {
#pragma unroll
            for (int v = 0; v < 4; ++v) Rn[(v * n + k) * n2 + node] = fx_limbs(q[v], fx_exp(mx[v]));
        }
        __syncthreads();
        if (tid < 4) mx[tid] = 0;
    }

    // ---------------- reverse of the epilogue
    // adjoints of the face records, the wave speed's folded into those of q
    for (int o = tid; o < 4 * n; o += C::tpc) {
        const int f = o / n, m = o - f * n;
        const double* rb = trace_bar + ((size_t)cell * 4 + f) * TR;
        const double* rf = trace + ((size_t)cell * 4 + f) * TR;
        double out[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) out[c] = rb[c * n + m];
        const double sb = rb[16 * n + m];
        if (sb != 0.0) {
            const double qf[4] = {rf[m], rf[n + m], rf[2 * n + m], rf[3 * n + m]};
            const bool xface = f < 2;
            const double zf = xface ? P.y0 + (iy + B.xi[m]) * P.hy : P.y0 + (iy + (f == 2 ? 1 : 0)) * P.hy;
            wave_speed_adj(qf, zf, xface, P, sb, out);
        }
#pragma unroll
        for (int c = 0; c < 16; ++c) FR[(f * 16 + c) * n + m] = c < 4 ? out[c] : rb[c * n + m];
    }
    __syncthreads();
    // adjoints of the time averages at a node: qbar, Fbar, Gbar, qxbar, qybar [5][4][n2], from the faces and
    // the weak volume residual (rvol_bar = dt lam')
    const double* lc = lam + (size_t)cell * SL;
    if (on)
        for (int v = k; v < 4; v += n) {
            auto fr = [&](int f, int c) { return FR[(f * 16 + c + v) * n + (f < 2 ? j : i)]; };
            const double pe = B.phi1[i], pw = B.phi0[i], pn = B.phi1[j], ps = B.phi0[j];
            auto all = [&](int c) { return fma(ps, fr(3, c), fma(pn, fr(2, c), fma(pw, fr(1, c), pe * fr(0, c)))); };
            double sx = 0.0, sy = 0.0;
#pragma unroll
            for (int p = 0; p < n; ++p) {
                sx = fma(B.Vx[i][p], lc[v * n2 + j * n + p], sx);
                sy = fma(B.Vx[j][p], lc[v * n2 + p * n + i], sy);
            }
            Wd[v * n2 + node] = all(0);
            Wd[(4 + v) * n2 + node] = fma(dt * P.inv_hx, sx, fma(pw, fr(1, 4), pe * fr(0, 4)));
            Wd[(8 + v) * n2 + node] = fma(dt * P.inv_hy, sy, fma(ps, fr(3, 4), pn * fr(2, 4)));
            Wd[(12 + v) * n2 + node] = all(8);
            Wd[(16 + v) * n2 + node] = all(12);
        }
    __syncthreads();
    // final evaluation and time averages: q^(n)_k (still in q)
    double qb[4], gxb[4], gyb[4], ub[4] = {0.0, 0.0, 0.0, 0.0};
    {
        const double wk = B.w[k];
        double Fb[4], Gb[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            qb[v] = wk * Wd[v * n2 + node];
            Fb[v] = wk * Wd[(4 + v) * n2 + node];
            Gb[v] = wk * Wd[(8 + v) * n2 + node];
            gxb[v] = wk * Wd[(12 + v) * n2 + node];
            gyb[v] = wk * Wd[(16 + v) * n2 + node];
        }
        double gx[4], gy[4];
        long long R0, R0y;
        gradients(IT + (n - 1) * 4 * n3 + k * n2, n3, EX + 4 * n, gx, gy, R0, R0y);
        ns_flux5_adj(q, gx, gy, g, gz, P.gm1, P.mu, mu23, kR, Fb, Gb, wk * dt * lc[2 * n2 + node], qb, gxb, gyb);
    }
    // fold the gradient adjoints back: q_bar(j,p) += (1/h) sum_i' D[i'][p] qx_bar(j,i'); slices: time nodes that hold data
    auto fold = [&](bool mine) {
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            push(13 + v, mine ? fx_mag(gxb[v]) : 0u);
            push(17 + v, mine ? fx_mag(gyb[v]) : 0u);
        }
        __syncthreads();
        int E[8];
#pragma unroll
        for (int v = 0; v < 8; ++v) E[v] = fx_exp(mx[13 + v]);
        if (on && mine) {
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                W[(v * n + k) * n2 + node] = fx_limbs(gxb[v], E[v]);
                W[((4 + v) * n + k) * n2 + node] = fx_limbs(gyb[v], E[4 + v]);
            }
        }
        __syncthreads();
        if (tid < 8) mx[13 + tid] = 0;
        if (!mine) return;
        FxSum a[4], b[4];
#pragma unroll
        for (int p = 0; p < n; ++p) {
            const Limbs dx = DT[p * n + i], dy = DT[n2 + p * n + j];
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                a[v].add(dx, W[(v * n + k) * n2 + j * n + p]);
                b[v].add(dy, W[((4 + v) * n + k) * n2 + p * n + i]);
            }
        }
#pragma unroll
        for (int v = 0; v < 4; ++v)
            qb[v] += fx_to(a[v].value(), E[v] + ex - 2102) + fx_to(b[v].value(), E[4 + v] + ey - 2102);
    };
    fold(true);

    // ---------------- reverse sweeps r = n .. 1: q^(r)_l = u + dt sum_k Kw[l][k] R_k(q^(r-1));
    // in sweep 1 the residual R(u) is one time slice's, weighted by the row sums of Kw
#pragma unroll 1
    for (int r = n; r >= 1; --r) {
        const bool mine = r > 1 || k == 0;
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            ub[v] += qb[v];
            push(21 + v, fx_mag(qb[v]));
        }
        __syncthreads();  // also: every thread has folded, W is free
        int E[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) E[v] = fx_exp(mx[21 + v]);
        if (on) {
#pragma unroll
            for (int v = 0; v < 4; ++v) W[(v * n + k) * n2 + node] = fx_limbs(qb[v], E[v]);
        }
        // the state of this sweep's evaluation: the iterate, and its limbs in its place for the gradients
        const int* eq = EX + 4 * (r - 1);
        if (r == 1) {
#pragma unroll
            for (int v = 0; v < 4; ++v) q[v] = US[v * n2 + node];
        } else {
            Limbs* Qr = IT + (r - 2) * 4 * n3 + k * n2 + node;
#pragma unroll
            for (int v = 0; v < 4; ++v) q[v] = reinterpret_cast<const double*>(Qr)[v * n3];
            __syncwarp();  // the lanes that repeat the last node have read it
            if (on) {
#pragma unroll
                for (int v = 0; v < 4; ++v) Qr[v * n3] = fx_limbs(q[v], eq[v]);
            }
        }
        __syncthreads();
        if (tid < 4) mx[21 + tid] = 0;
        double R2 = 0.0;
        if (mine) {
            const int eK = r > 1 ? B.KwE : B.KwE + 3;
            FxSum a[4];
#pragma unroll
            for (int l = 0; l < n; ++l) {
                const Limbs d = r > 1 ? K[l * n + k] : K[n2 + l];
#pragma unroll
                for (int v = 0; v < 4; ++v) a[v].add(d, W[(v * n + l) * n2 + node]);
            }
            R2 = fx_to(a[2].value(), E[2] + eK - 2102);
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                E[v] += eK - 2102 + 3 + 1080;  // |sum| < 2^61: below 2^58 after the shift
                if (on) W[((4 + v) * n + k) * n2 + node] = fx_split(a[v].value() >> 3);
            }
        }
        __syncthreads();
#pragma unroll
        for (int v = 0; v < 4; ++v) qb[v] = gxb[v] = gyb[v] = 0.0;
        if (mine) {
            // R_k = -(1/hx) D_x F_k - (1/hy) D_y G_k + S_k: F_bar(j,p) = -(dt/hx) sum_i' D[i'][p] R_bar(j,i')
            double Fb[4], Gb[4];
            {
                FxSum a[4], b[4];
#pragma unroll
                for (int p = 0; p < n; ++p) {
                    const Limbs dx = DM[p * n + i], dy = DM[n2 + p * n + j];
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        a[v].add(dx, W[((4 + v) * n + k) * n2 + j * n + p]);
                        b[v].add(dy, W[((4 + v) * n + k) * n2 + p * n + i]);
                    }
                }
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    Fb[v] = fx_to(a[v].value(), E[v] + emx - 2102);
                    Gb[v] = fx_to(b[v].value(), E[v] + emy - 2102);
                }
            }
            const Limbs* Qk = r == 1 ? U0 : IT + (r - 2) * 4 * n3 + k * n2;
            const int ps = r == 1 ? n2 : n3;
            double gx[4], gy[4];
            long long R0, R0y;
            gradients(Qk, ps, eq, gx, gy, R0, R0y);
            ns_flux5_adj(q, gx, gy, g, gz, P.gm1, P.mu, mu23, kR, Fb, Gb, dt * R2, qb, gxb, gyb);
        }
        fold(mine);
    }
    // sum over the time nodes of the adjoints that reached u
    __syncthreads();
    if (on) {
#pragma unroll
        for (int v = 0; v < 4; ++v) Wd[(v * n + k) * n2 + node] = ub[v] + qb[v];
    }
    __syncthreads();
    if (on && active)
        for (int v = k; v < 4; v += n) {
            double s = lc[v * n2 + node];
#pragma unroll
            for (int l = 0; l < n; ++l) s += Wd[(v * n + l) * n2 + node];
            lam_out[(size_t)cell * SL + v * n2 + node] = s;
        }
}

template <int N>
static int adj_n(const double* u, const double* lam, double* lam_out, const double* trace, double* trace_bar,
                 int cells, double dt, const Basis& B, const Phys& P, const Background& bg, cudaStream_t s) {
    using C = AdjCfg<N>;
    constexpr int cpb = N <= 2 ? 4 : N <= 4 ? 2 : 1;  // cells per block of the corrector's adjoint
    k_corrector_adj_fp64<N, cpb><<<(cells + cpb - 1) / cpb, cpb*(N + 1) * (N + 1), 0, s>>>(lam, trace, trace_bar, cells,
                                                                                      dt, B, P, bg);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return (int)e;
    auto kern = k_predictor_adj_fp64<N>;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::smem);
    if (e != cudaSuccess) return (int)e;
    kern<<<(cells + C::cpb - 1) / C::cpb, C::threads, C::smem, s>>>(u, lam, trace, trace_bar, lam_out, cells, dt, B, P,
                                                               bg);
    return (int)cudaGetLastError();
}

int launch_step_adjoint_fp64(int N, const double* u, const double* lam, double* lam_out, const double* trace,
                             double* trace_bar, int cells, double dt, const Basis& B, const Phys& P,
                             const Background& bg, void* stream) {
    cudaStream_t s = (cudaStream_t)stream;
    switch (N) {
        case 1: return adj_n<1>(u, lam, lam_out, trace, trace_bar, cells, dt, B, P, bg, s);
        case 2: return adj_n<2>(u, lam, lam_out, trace, trace_bar, cells, dt, B, P, bg, s);
        case 3: return adj_n<3>(u, lam, lam_out, trace, trace_bar, cells, dt, B, P, bg, s);
        case 4: return adj_n<4>(u, lam, lam_out, trace, trace_bar, cells, dt, B, P, bg, s);
        case 5: return adj_n<5>(u, lam, lam_out, trace, trace_bar, cells, dt, B, P, bg, s);
    }
    return (int)cudaErrorInvalidValue;
}

}  // namespace adg
