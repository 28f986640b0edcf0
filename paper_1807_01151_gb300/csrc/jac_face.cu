// FP64 face Jacobians (the FP64 block form and the p = 0 Jacobian): dF~/dU_L and dF~/dU_R of the
// Roe flux per face point, on boundary faces the total derivative through the ghost state,
// dF~/dU_L + dF~/dU_ghost dU_ghost/dU_L.  The derivatives are the chain rule written out, in the
// primitive variables W = (rho, v, p) of one side at a time, where most inner derivatives vanish,
// and turned to conservative columns at the end.  Bound by the float64 pipe.  Forward-mode dual
// numbers over the conservative variables took about 2400 float64 operations per point with 255
// registers; this form takes about 800 in 2-D (a flow in the plane: four variables and the
// spanwise column apart) and 1200 in 3-D.  One thread per point and side.  Measured per FP64 V-cycle:
// 128 x 64 p = 4 2.89 -> 1.12 ms, 32 x 16 p = 2 (latency) 0.43 -> 0.22 ms.
#include "dispatch.cuh"
#include "euler.cuh"
#include "fix.cuh"
#include "jacobian.cuh"

namespace emg {

// One side's state: primitives and transport velocities.  NK = 2: no z component (v_z = n_z = 0).
template <int NK>
struct SideV {
    double r, ir, v[NK], p, q, m, E, H;   // q = v.n, m = q - v_r.n, E = rho E, H = (E + p) / rho
};

template <int NK>
__device__ __forceinline__ void side_of(const double U[5], const double n[3], double g, double vrn, SideV<NK>& s) {
    s.r = U[0];
    s.ir = rcp_h3(U[0]);
    double k2 = 0.0;
    s.q = 0.0;
#pragma unroll
    for (int k = 0; k < NK; ++k) {
        s.v[k] = U[1 + k] * s.ir;
        k2 = fma(U[1 + k], s.v[k], k2);
        s.q = fma(s.v[k], n[k], s.q);
    }
    s.m = s.q - vrn;
    s.E = U[4];
    s.p = (g - 1.0) * fma(-0.5, k2, U[4]);
    s.H = (U[4] + s.p) * s.ir;
}

// The Roe flux's intermediates (names as in roe_flux_fast of residual.cu).
template <int NK>
struct RoeV {
    double n[NK], u[NK], dv[NK];
    double rho, c, ic2, hic, rc, rdq, dq, dp, dH, wR, qn, ud, K, H, T;
    double A1, A5, A2, l1, l2, l5, s1, s2, s5, w1, w5, w2, ws, d0, w15, dc;
};

template <int NK>
__device__ __forceinline__ void roe_of(const SideV<NK>& L, const SideV<NK>& R, const double n[3], double g, double vrn,
                                       RoeV<NK>& w) {
    const double s2 = ratio_or_negative(R.r, L.ir, L.r), s = s2 * rsqrt_h3(s2);
    w.wR = s * rcp_h3(1.0 + s);
    w.rho = s * L.r;
    w.K = 0.0;
    w.ud = 0.0;
#pragma unroll
    for (int k = 0; k < NK; ++k) {
        w.n[k] = n[k];
        w.dv[k] = R.v[k] - L.v[k];
        w.u[k] = fma(w.wR, w.dv[k], L.v[k]);
        w.K = fma(0.5 * w.u[k], w.u[k], w.K);
        w.ud = fma(w.u[k], w.dv[k], w.ud);
    }
    w.dH = R.H - L.H;
    w.H = fma(w.wR, w.dH, L.H);
    const double c2 = (g - 1.0) * (w.H - w.K), ic = rsqrt_h3(c2);
    w.c = c2 * ic;
    w.ic2 = ic * ic;
    w.hic = 0.5 * ic;
    w.dq = R.q - L.q;
    w.qn = fma(w.wR, w.dq, L.q);
    w.dp = R.p - L.p;
    w.rc = w.rho * w.c;
    w.rdq = w.rho * w.dq;
    const double rq = w.rc * w.dq, hc = 0.5 * w.ic2, qr = w.qn - vrn;
    w.A1 = (w.dp - rq) * hc;
    w.A5 = (w.dp + rq) * hc;
    w.A2 = fma(-w.dp, w.ic2, R.r - L.r);
    w.s1 = qr - w.c >= 0.0 ? 1.0 : -1.0;   // d|x|/dx = +1 at 0
    w.s2 = qr >= 0.0 ? 1.0 : -1.0;
    w.s5 = qr + w.c >= 0.0 ? 1.0 : -1.0;
    w.l1 = fabs(qr - w.c);
    w.l2 = fabs(qr);
    w.l5 = fabs(qr + w.c);
    w.w1 = w.l1 * w.A1;
    w.w5 = w.l5 * w.A5;
    w.w2 = w.l2 * w.A2;
    w.ws = w.l2 * w.rho;
    w.w15 = w.w1 + w.w5;
    w.d0 = w.w15 + w.w2;
    w.dc = (w.w5 - w.w1) * w.c;
    w.T = fma(-w.qn, w.dq, w.ud);
}

// Column of 2 F~ (mass, momentum, energy: NK + 2 rows) for the primitive DIR of one side: 0 rho,
// 1..NK velocity, NK + 1 p.  sg: -1 for the left side, +1 for the right; W: its Roe weight.
template <int NK, int DIR>
__device__ __forceinline__ void roe_col(const RoeV<NK>& w, const SideV<NK>& o, double g, double sg, double W,
                                        double* out) {
    constexpr bool RHO = DIR == 0, PR = DIR == NK + 1, VEL = !RHO && !PR;
    constexpr int M = VEL ? DIR - 1 : 0;
    const double gr = g / (g - 1.0);
    double kap = 0.0, dqn = 0.0, dH, uu = 0.0, drho = 0.0;
    if (RHO) {
        kap = sg * 0.5 * o.ir * w.wR * (1.0 - w.wR);
        drho = 0.5 * w.rho * o.ir;
        dqn = kap * w.dq;
        uu = kap * w.ud;
        dH = fma(kap, w.dH, -W * gr * o.p * o.ir * o.ir);
    } else if (VEL) {
        dqn = W * w.n[M];
        uu = W * w.u[M];
        dH = W * o.v[M];
    } else {
        dH = W * gr * o.ir;
    }
    const double dc2 = (g - 1.0) * (PR ? dH : dH - uu);
    const double t = w.ic2 * dc2, dcs = w.hic * dc2;
    const double dl1 = w.s1 * (PR ? -dcs : dqn - dcs), dl5 = w.s5 * (PR ? dcs : dqn + dcs), dl2 = w.s2 * dqn;
    double drq = w.rdq * dcs;
    if (RHO) drq = fma(w.c * w.dq, drho, drq);
    if (VEL) drq = fma(w.rc * sg, w.n[M], drq);
    const double hc = 0.5 * w.ic2;
    const double dA1 = fma(-w.A1, t, hc * (PR ? sg - drq : -drq));
    const double dA5 = fma(-w.A5, t, hc * (PR ? sg + drq : drq));
    const double dA2 = RHO ? fma(w.ic2 * w.dp, t, sg) : PR ? w.ic2 * fma(w.dp, t, -sg) : w.ic2 * w.dp * t;
    const double dw1 = fma(dl1, w.A1, w.l1 * dA1), dw5 = fma(dl5, w.A5, w.l5 * dA5);
    const double dw2 = PR ? w.l2 * dA2 : fma(dl2, w.A2, w.l2 * dA2);
    const double dws = RHO ? fma(dl2, w.rho, w.l2 * drho) : PR ? 0.0 : dl2 * w.rho;
    const double dw15 = dw1 + dw5, dd0 = dw15 + dw2;
    const double ddc = fma(dw5 - dw1, w.c, (w.w5 - w.w1) * dcs);
    // mass: rho m on the own side
    out[0] = (RHO ? o.m : VEL ? o.r * w.n[M] : 0.0) - dd0;
    // momentum
    double dpn = PR ? 1.0 - ddc : fma(dws, w.dq, -ddc);
    if (VEL) dpn = fma(w.ws * sg, w.n[M], dpn);
#pragma unroll
    for (int k = 0; k < NK; ++k) {
        double x = fma(dpn, w.n[k], -dd0 * w.u[k]);
        if (!PR) x = fma(-dws, w.dv[k], x);
        if (RHO) x = fma(o.v[k], o.m, fma(-w.d0 * kap, w.dv[k], x));
        if (VEL) x = fma(o.r * o.v[k], w.n[M], x);
        if (VEL && k == M) x += fma(o.r, o.m, fma(-w.d0, W, -w.ws * sg));
        out[1 + k] = x;
    }
    // energy: E m + p q on the own side
    double v2 = 0.0;
    if (RHO) {
#pragma unroll
        for (int k = 0; k < NK; ++k) v2 = fma(o.v[k], o.v[k], v2);
    }
    double x = RHO ? 0.5 * v2 * o.m : VEL ? fma(o.r * o.v[M], o.m, (o.E + o.p) * w.n[M]) : fma(o.m, 1.0 / (g - 1.0), o.q);
    x = fma(-dw15, w.H, fma(-w.w15, dH, fma(-dw2, w.K, fma(-ddc, w.qn, x))));
    if (!PR) x = fma(-w.w2, uu, fma(-w.dc, dqn, fma(-dws, w.T, x)));
    if (RHO) {   // dT = du . dv - dqn dq
        double dd = 0.0;
#pragma unroll
        for (int k = 0; k < NK; ++k) dd = fma(w.dv[k], w.dv[k], dd);
        x = fma(-w.ws * kap, fma(-w.dq, w.dq, dd), x);
    }
    if (VEL) x = fma(-w.ws, fma(W, fma(-w.n[M], w.dq, w.dv[M]), sg * fma(-w.qn, w.n[M], w.u[M])), x);
    out[NK + 1] = x;
}

template <int NK>
__device__ __forceinline__ void roe_cols(const RoeV<NK>& w, const SideV<NK>& o, double g, double sg, double W,
                                         double (*A)[NK + 2]) {
    roe_col<NK, 0>(w, o, g, sg, W, A[0]);
    roe_col<NK, 1>(w, o, g, sg, W, A[1]);
    roe_col<NK, 2>(w, o, g, sg, W, A[2]);
    if constexpr (NK == 3) roe_col<NK, 3>(w, o, g, sg, W, A[3]);
    roe_col<NK, NK + 1>(w, o, g, sg, W, A[NK + 1]);
}

// dU of the spanwise momentum alone where v_z = n_z = 0: only the spanwise flux depends on it.
template <int NK>
__device__ __forceinline__ double roe_span(const RoeV<NK>& w, const SideV<NK>& o, double sg, double W) {
    return fma(o.r, o.m, fma(-w.d0, W, -w.ws * sg));
}

// The primitive columns A of 2 F~ to conservative columns of am F~, row-major 5 x 5.
template <int NK>
__device__ __forceinline__ void cols_out(const double (*A)[NK + 2], double span, const SideV<NK>& o, double g, double am,
                                         double* __restrict__ out) {
    const double ha = 0.5 * am, g1 = g - 1.0;
    double v2 = 0.0;
#pragma unroll
    for (int k = 0; k < NK; ++k) v2 = fma(o.v[k], o.v[k], v2);
#pragma unroll
    for (int a = 0; a < NK + 2; ++a) {
        double* row = out + (a == NK + 1 ? 4 : a) * 5;
        double x = fma(0.5 * g1 * v2, A[NK + 1][a], A[0][a]);
#pragma unroll
        for (int m = 0; m < NK; ++m) {
            const double y = A[1 + m][a] * o.ir;
            x = fma(-o.v[m], y, x);
            row[1 + m] = ha * fma(-g1 * o.v[m], A[NK + 1][a], y);
        }
        row[0] = ha * x;
        row[4] = ha * g1 * A[NK + 1][a];
        if (NK == 2) row[3] = 0.0;
    }
    if (NK == 2) {
        double* row = out + 15;
        row[0] = row[1] = row[2] = row[4] = 0.0;
        row[3] = ha * span * o.ir;
    }
}

// Boundary faces: the ghost in primitives and its derivatives, dG[j][i] = d(ghost i) / d(W_j).  The
// wall (and symmetry plane) mirrors the velocity relative to the frame about nw; the far field is
// farfield_fast of residual.cu on velocities relative to the frame.  Returns the derivative of the
// ghost's spanwise velocity by the inside one (2-D: 0 at an inflow, where it is the free stream's).
template <int NK>
__device__ __forceinline__ double ghost_of(const SideV<NK>& L, int bc, const double n[3], const double* nw,
                                         const double vr[3], const U5& uinf, double g, double UG[5],
                                         double (*dG)[NK + 2]) {
#pragma unroll
    for (int j = 0; j < NK + 2; ++j)
#pragma unroll
        for (int i = 0; i < NK + 2; ++i) dG[j][i] = i == j ? 1.0 : 0.0;
    double r, v[3] = {0.0, 0.0, 0.0}, p, wz = 1.0;
    if (bc == EMG_BC_WALL || bc == EMG_BC_SYMMETRY) {
        double qw = 0.0;
#pragma unroll
        for (int k = 0; k < NK; ++k) qw = fma(L.v[k] - vr[k], nw[k], qw);
#pragma unroll
        for (int k = 0; k < NK; ++k) {
            v[k] = fma(-2.0 * qw, nw[k], L.v[k]);
#pragma unroll
            for (int m = 0; m < NK; ++m) dG[1 + m][1 + k] = (k == m ? 1.0 : 0.0) - 2.0 * nw[m] * nw[k];
        }
        r = L.r;
        p = L.p;
    } else {
        const double ex = 1.0 / (g - 1.0);
        const double ri = uinf.v[0];
        double vi[3], q2 = 0.0, qi = 0.0, vrn = 0.0;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            vi[k] = uinf.v[1 + k] / ri;
            q2 = fma(vi[k], vi[k], q2);
            if (k < NK) {
                qi = fma(vi[k] - vr[k], n[k], qi);
                vrn = fma(vr[k], n[k], vrn);
            }
        }
        const double ci2 = g * (g - 1.0) * (uinf.v[4] / ri - 0.5 * q2), ici = rsqrt_h3(ci2), ci = ci2 * ici;
        const double c2 = g * L.p * L.ir, ic = rsqrt_h3(c2), c = c2 * ic, q = L.q - vrn;
        const double Rp = fma(2.0 * ex, c, q), Rm = fma(-2.0 * ex, ci, qi);
        const double qb = 0.5 * (Rp + Rm), cb = 0.25 * (g - 1.0) * (Rp - Rm);
        const bool in = qb < 0.0;
        const double x = cb * cb * (in ? ici * ici : ic * ic);
        const double pw = fabs(ex - 2.5) < 1e-14 ? x * x * (x * rsqrt_h3(x)) : pow(x, ex);
        r = (in ? ri : L.r) * pw;
        p = r * cb * cb / g;
        if (in) wz = 0.0;
        const double icb = rcp_h3(cb), dq = qb - (in ? qi : q);
#pragma unroll
        for (int k = 0; k < NK; ++k) v[k] = fma(dq, n[k], in ? vi[k] : L.v[k]);
        const double ip = rcp_h3(L.p);
#pragma unroll
        for (int j = 0; j < NK + 2; ++j) {
            const double dc = j == 0 ? -0.5 * c * L.ir : j == NK + 1 ? 0.5 * c * ip : 0.0;
            const double dqj = j > 0 && j <= NK ? n[j > 0 && j <= NK ? j - 1 : 0] : 0.0;
            const double dR = fma(2.0 * ex, dc, dqj), dqb = 0.5 * dR, lcb = 0.25 * (g - 1.0) * dR * icb;
            const double lr = in ? 2.0 * ex * lcb : fma(2.0 * ex, lcb - dc * ic, j == 0 ? L.ir : 0.0);
            dG[j][0] = r * lr;
            dG[j][NK + 1] = p * fma(2.0, lcb, lr);
#pragma unroll
            for (int k = 0; k < NK; ++k)
                dG[j][1 + k] = in ? dqb * n[k] : fma(dqb - dqj, n[k], j == 1 + k ? 1.0 : 0.0);
        }
    }
    double k2 = 0.0;
    UG[0] = r;
    UG[3] = 0.0;
#pragma unroll
    for (int k = 0; k < NK; ++k) {
        UG[1 + k] = r * v[k];
        k2 = fma(v[k], v[k], k2);
    }
    UG[4] = fma(p, 1.0 / (g - 1.0), 0.5 * r * k2);
    return wz;
}

template <int NK>
__device__ __forceinline__ void face_jac_point(const double UL[5], const double UR[5], int side, bool inner, int bc,
                                               const double n[3], const double* nw, const double vr[3], double vrn,
                                               const U5& uinf, double g, double am, double* __restrict__ out) {
    SideV<NK> L, R;
    RoeV<NK> w;
    double A[NK + 2][NK + 2];
    side_of<NK>(UL, n, g, vrn, L);
    if (inner) {
        side_of<NK>(UR, n, g, vrn, R);
        roe_of<NK>(L, R, n, g, vrn, w);
        const double sg = side ? 1.0 : -1.0, W = side ? w.wR : 1.0 - w.wR;
        if (side) L = R;
        roe_cols<NK>(w, L, g, sg, W, A);
        cols_out<NK>(A, roe_span<NK>(w, L, sg, W), L, g, am, out);
        return;
    }
    double UG[5], dG[NK + 2][NK + 2], Ag[NK + 2][NK + 2];
    const double wz = ghost_of<NK>(L, bc, n, nw, vr, uinf, g, UG, dG);
    side_of<NK>(UG, n, g, vrn, R);
    roe_of<NK>(L, R, n, g, vrn, w);
    roe_cols<NK>(w, R, g, 1.0, w.wR, Ag);
    roe_cols<NK>(w, L, g, -1.0, 1.0 - w.wR, A);
#pragma unroll
    for (int j = 0; j < NK + 2; ++j)
#pragma unroll
        for (int a = 0; a < NK + 2; ++a) {
            double x = A[j][a];
#pragma unroll
            for (int i = 0; i < NK + 2; ++i) x = fma(Ag[i][a], dG[j][i], x);
            A[j][a] = x;
        }
    const double span = fma(wz, roe_span<NK>(w, R, 1.0, w.wR), roe_span<NK>(w, L, -1.0, 1.0 - w.wR));
    cols_out<NK>(A, span, L, g, am, out);
}

template <int D, int P, bool ROT>
__global__ void __launch_bounds__(128) k_face_jac64(int F, int F_int, const int* __restrict__ fL,
                                                    const int* __restrict__ fR, const int* __restrict__ fbc,
                                                    const double* __restrict__ fnrm, const double* __restrict__ famag,
                                                    const double* __restrict__ fpsiL, const double* __restrict__ fpsiR,
                                                    const double* __restrict__ fwn, const double* __restrict__ u,
                                                    const double* __restrict__ tr, double g, U5 uinf,
                                                    const double* __restrict__ fvr, double* __restrict__ fjl,
                                                    double* __restrict__ fjr) {
    constexpr int QF = Lv<D, P>::QF;
    // boundary faces, numbered last and with the longest path, start first
    const int64_t idx2 = 2 * (int64_t)F * QF - 1 - ((int64_t)blockIdx.x * blockDim.x + threadIdx.x);
    if (idx2 < 0) return;
    const int64_t idx = idx2 >> 1;
    const int side = (int)(idx2 & 1), f = (int)(idx / QF);
    const bool inner = f < F_int;
    if (!inner && side) return;
    double UL[5], UR[5] = {1.0, 0.0, 0.0, 0.0, 1.0};
    if constexpr (P == 0) {
        const double pl = fpsiL[idx];
        const double* ue = u + (size_t)fL[f] * 5;
#pragma unroll
        for (int a = 0; a < 5; ++a) UL[a] = ue[a] * pl;
        if (inner) {
            const double pr = fpsiR[idx];
            const double* ur = u + (size_t)fR[f] * 5;
#pragma unroll
            for (int a = 0; a < 5; ++a) UR[a] = ur[a] * pr;
        }
    } else {
        const double2* t = reinterpret_cast<const double2*>(tr + idx * 10);
        const double2 t0 = t[0], t1 = t[1], t2 = t[2];
        UL[0] = t0.x, UL[1] = t0.y, UL[2] = t1.x, UL[3] = t1.y, UL[4] = t2.x;
        if (inner) {
            const double2 t3 = t[3], t4 = t[4];
            UR[0] = t2.y, UR[1] = t3.x, UR[2] = t3.y, UR[3] = t4.x, UR[4] = t4.y;
        }
    }
    const double n[3] = {fnrm[idx * 3], fnrm[idx * 3 + 1], fnrm[idx * 3 + 2]};
    double vr[3] = {0.0, 0.0, 0.0}, nw[3] = {0.0, 0.0, 0.0}, vrn = 0.0;
    if constexpr (ROT) {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            vr[k] = fvr[idx * 3 + k];
            vrn = fma(vr[k], n[k], vrn);
        }
    }
    int bc = 0;
    if (!inner) {
        bc = fbc[f];
        const int64_t bi = idx - (int64_t)F_int * QF;
#pragma unroll
        for (int k = 0; k < 3; ++k) nw[k] = fwn[bi * 3 + k];
    }
    double* out = (side ? fjr : fjl) + idx * 25;
    const double am = famag[idx];
    if (D == 2 && UL[3] == 0.0 && UR[3] == 0.0)   // n[2] = 0 in 2-D
        face_jac_point<2>(UL, UR, side, inner, bc, n, nw, vr, vrn, uinf, g, am, out);
    else
        face_jac_point<3>(UL, UR, side, inner, bc, n, nw, vr, vrn, uinf, g, am, out);
}

emg_status launch_face_jacobian(emg_ctx* c, int p, const double* u) {
    LevelDev& L = c->lv[p];
    if (p > 0) {
        const emg_status st = launch_traces(c, p, u, L.trj, PC_FACE_JAC);
        if (st != EMG_OK) return st;
    }
    const int F = (int)c->F, Fi = (int)c->F_int;
    U5 ui;
    for (int a = 0; a < 5; ++a) ui.v[a] = c->uinf[a];
#define EMG_FJ(DD, PP)                                                                                       \
    {                                                                                                        \
        const int64_t nf = 2 * (int64_t)F * Lv<DD, PP>::QF;                                                  \
        ProfScope _ps(c, PC_FACE_JAC);                                                                       \
        (c->rot ? k_face_jac64<DD, PP, true> : k_face_jac64<DD, PP, false>)<<<(unsigned)((nf + 127) / 128), 128, 0, c->stream>>>( \
            F, Fi, c->face_L, c->face_R, c->face_bc, L.fnrm, L.famag, L.fpsiL, L.fpsiR, L.fwn, u, L.trj,       \
            c->prm.gamma, ui, L.fvr, L.fjl, L.fjr);                                                          \
    }
    EMG_DISPATCH_DP(c->dim, p, EMG_FJ)
#undef EMG_FJ
    EMG_CHECK_LAUNCH(c);
    return EMG_OK;
}

}  // namespace emg
