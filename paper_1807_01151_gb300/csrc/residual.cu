// DG residual R_p(U) of Eq. euler3 with the orthonormal basis (mass matrix = I):
//   R_{e,a,i} = sum_q sum_k W_q d_k psi_i(x_q) F_{k,a}(U_h(x_q))
//             - sum_faces sum_t w|n dS| psi_i(x_t) F~_a(U_in, U_out, n)
// Levels p >= 1, three kernels: k_traces evaluates every element's U_h at its own face points;
// k_face_flux forms the Roe flux once per face point (interior faces with both traces, boundary
// faces with the ghost state of Sec. 3.3) and stores w|n dS| F~; k_volume does, per element, the
// volume quadrature and the projection of its faces' fluxes (sign -1 on the L side, +1 on the R
// side: no atomics, deterministic).  The p = 0 level has one mode and no volume term: k_face_flux
// forms its traces itself and k_cell0 sums the faces.
// The contractions with the basis tables (all but the point fluxes) run as fixed-point dot
// products on the integer pipe (fix.cuh); the point fluxes are float64.  With every contraction on
// the float64 pipe (2 multiply-adds per clock and SM) the residual was at that pipe's limit: one
// evaluation alone took 284 us on a 128 x 64 O-grid at p = 4 and 1.82 ms on 3234 hexes at p = 4, now
// 124 us and 0.65 ms one after the other.  What bounds the parts (128 x 64, p = 4, ncu): k_traces 21 us, the latency
// of its staging; k_face_flux 31 us, 80 % of the float64 pipe (Roe fluxes); k_volume 72 us, latency and
// issue at 16 warps per SM (about 6700 instructions per warp of 2 elements, 34 % of the issue slots) and
// 130 MB of tables (a quarter of the DRAM's rate).  3234 hexes, p = 4: 86, 95 (86 % of the float64 pipe) and
// 466 us.  More resident warps with fewer registers (64 to 96 a thread), other block
// sizes and L2 prefetches of the tables measured equal or slower.
// ROT: a frame rotating with angular velocity omega (Eq. euler): the fluxes carry the velocity
// relative to the frame v_r = omega x x (tabulated at the points), F_k - (v_r)_k U, the face
// fluxes move with v_r . n, the ghosts are taken relative to the frame, and the source
// S = (0, -rho omega x v, 0), linear in U, adds -omega x u_{m,i} to the momentum modes (the
// orthonormal basis makes int psi_i S = -omega x (rho v)_i).
#include <cmath>

#include "common.cuh"
#include "dispatch.cuh"
#include "euler.cuh"
#include "fix.cuh"
#include "residual_chain.h"

namespace emg {

// ---- traces ------------------------------------------------------------------------------------
// A block holds ET elements; thread (element, face point) sums the N modes of the five variables.
// The element's side of its faces' basis table goes through shared memory (a thread's row of N
// entries starts N * 8 bytes after its neighbour's, so direct loads would touch one line per lane).
template <int D, int P>
struct TrCfg {
    using L = Lv<D, P>;
    static constexpr int NP = L::NF * L::QF;                               // face points per element
    static constexpr int ET = NP >= 128 ? 1 : 128 / NP;
    static constexpr int THREADS = ((ET * NP + 31) / 32) * 32;
    static constexpr int NS = L::N | 1;                                    // odd row stride (8-byte words)
    static constexpr size_t SMEM = ((size_t)ET * NP * NS + (size_t)ET * L::N * 6) * sizeof(int2);
};

template <int D, int P>
__global__ void __launch_bounds__(TrCfg<D, P>::THREADS) k_traces(int E, const double* __restrict__ u,
                                                                 const int* __restrict__ elem_face,
                                                                 const int2* __restrict__ fpsiL,
                                                                 const int2* __restrict__ fpsiR,
                                                                 const int* __restrict__ texp,
                                                                 double* __restrict__ tr) {
    chain_wait();
    using L = Lv<D, P>;
    using CF = TrCfg<D, P>;
    constexpr int N = L::N, QF = L::QF, B = L::B, NF = L::NF, NP = CF::NP, NS = CF::NS;
    constexpr int ET = CF::ET, T = CF::THREADS;
    extern __shared__ __align__(16) unsigned char smraw[];
    int2* us = reinterpret_cast<int2*>(smraw);      // [ET][N][6]
    int2* ps = us + ET * N * 6;                     // [ET][NP][NS]
    __shared__ int mx[ET * 5], codes[ET * NF];
    const int e0 = blockIdx.x * ET;
    if (threadIdx.x < ET * 5) mx[threadIdx.x] = 0;
    for (int t = threadIdx.x; t < ET * NF; t += T)
        codes[t] = e0 + t / NF < E ? elem_face[(size_t)e0 * NF + t] : 0;
    constexpr int NU = (ET * B + T - 1) / T;
    double x[NU];
#pragma unroll
    for (int k = 0; k < NU; ++k) {
        const int t = threadIdx.x + k * T;
        x[k] = (t < ET * B && e0 + t / B < E) ? u[(size_t)e0 * B + t] : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < NU; ++k) {
        const int t = threadIdx.x + k * T;
        if (t < ET * B) atomicMax(&mx[t / N], fix_key(x[k]));   // t / N = element * 5 + variable
    }
    const int nside = (E - e0 < ET ? E - e0 : ET) * NF, lane = threadIdx.x & 31;
#pragma unroll(D == 2 ? 5 : 1)
    for (int r = threadIdx.x >> 5; r < nside; r += T / 32) {   // a warp per face side
        const int code = codes[r];
        const int2* src = ((code & 1) ? fpsiR : fpsiL) + (size_t)(code >> 1) * QF * N;
        int2* dst = ps + (size_t)r * QF * NS;
        if constexpr (FaceTab<D, P>::paired) {
            constexpr int NQ = QF / 2 * N;   // 16-byte entries (row pair, mode)
#pragma unroll 4
            for (int t = lane; t < NQ; t += 32) {
                const int4 v = reinterpret_cast<const int4*>(src)[t];
                int2* o = dst + (t / N) * 2 * NS + t % N;
                o[0] = make_int2(v.x, v.y);
                o[NS] = make_int2(v.z, v.w);
            }
            if (QF & 1)
                for (int i = lane; i < N; i += 32) dst[(QF - 1) * NS + i] = src[(QF - 1) * N + i];
        } else {
            for (int t = lane; t < QF * N; t += 32) dst[(t / N) * NS + t % N] = src[t];
        }
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < NU; ++k) {
        const int t = threadIdx.x + k * T;
        if (t < ET * B) us[((t / B) * N + t % N) * 6 + (t / N) % 5] = fix_of(x[k], fix_exp(mx[t / N]));
    }
    __syncthreads();
    const int el = threadIdx.x / NP, pt = threadIdx.x % NP, e = e0 + el;
    if (el >= ET || e >= E) return;
    const int code = codes[el * NF + pt / QF];
    const int st = texp[e];
    const int2* pr = ps + (size_t)threadIdx.x * NS;
    const int4* ur = reinterpret_cast<const int4*>(us + el * N * 6);
    long long h[5] = {0, 0, 0, 0, 0}, c[5] = {0, 0, 0, 0, 0};
    const bool w = D == 3 || mx[el * 5 + 3] != 0;   // 2-D flow without a spanwise momentum: 0
#pragma unroll 5
    for (int i = 0; i < N; ++i) {
        const int2 ps_i = pr[i];
        const int4 a = ur[i * 3], b = ur[i * 3 + 1], d = ur[i * 3 + 2];
        fix_mac(h[0], c[0], ps_i, make_int2(a.x, a.y));
        fix_mac(h[1], c[1], ps_i, make_int2(a.z, a.w));
        fix_mac(h[2], c[2], ps_i, make_int2(b.x, b.y));
        if (w) fix_mac(h[3], c[3], ps_i, make_int2(b.z, b.w));
        fix_mac(h[4], c[4], ps_i, make_int2(d.x, d.y));
    }
    double* o = tr + (((size_t)(code >> 1) * QF + pt % QF) * 2 + (code & 1)) * 5;
#pragma unroll
    for (int a = 0; a < 5; ++a) {
        const int key = mx[el * 5 + a];
        o[a] = (a != 3 || w) ? fix_sum(h[a], c[a], fix_scale(FIX_BITS - st - fix_exp(key), key)) : 0.0;
    }
}

// ---- face fluxes ---------------------------------------------------------------------------------
// The Roe flux of euler.cuh's roe_flux in float64, scaled by am, with four special functions
// instead of seven: one reciprocal for both densities, sqrt(rho_R / rho_L) for the averages (weights
// 1 / (1 + s) and s / (1 + s)), and one reciprocal square root for c and 1 / c^2.  The jumps are
// differences of rounded numbers (not fused with the product before them; the pressure's from the
// internal energies, where it rounds least), so that equal states have
// none: the flux along a wall or through a uniform flow is free of dissipation to the last bit.  NK = 2:
// a face in the x-y plane between states without a z momentum (every z term is 0).
template <int NK, bool ROT>
__device__ __forceinline__ void roe_flux_fast(const double UL[5], const double UR[5], const double n[3], double g,
                                              double vrn, double am, double F[5]) {
    const double it = rcp_h3(UL[0] * UR[0]);
    const double irL = it * UR[0], irR = it * UL[0];
    double vL[3], dv[3], u[3];
    double kL = 0.0, kR = 0.0, qL = 0.0, qR = 0.0;
#pragma unroll
    for (int k = 0; k < NK; ++k) {
        vL[k] = UL[1 + k] * irL;
        const double vR = UR[1 + k] * irR;
        kL = fma(UL[1 + k], vL[k], kL);
        kR = fma(UR[1 + k], vR, kR);
        qL = fma(vL[k], n[k], qL);
        qR = fma(vR, n[k], qR);
        dv[k] = __dsub_rn(vR, vL[k]);
    }
    const double iL = fma(-0.5, kL, UL[4]), iR = fma(-0.5, kR, UR[4]);   // p / (g - 1)
    const double pL = (g - 1.0) * iL, pR = (g - 1.0) * iR;
    const double EL = UL[4] + pL, ER = UR[4] + pR;
    const double HL = EL * irL, HR = ER * irR;
    const double s2 = ratio_or_negative(UR[0], irL, UL[0]);
    const double s = s2 * rsqrt_h3(s2);                 // sqrt(rho_R / rho_L)
    const double wR = s * rcp_h3(1.0 + s);              // s_R / (s_L + s_R)
    const double rho = s * UL[0];
    double q2 = 0.0;
#pragma unroll
    for (int k = 0; k < NK; ++k) {
        u[k] = fma(wR, dv[k], vL[k]);
        q2 = fma(u[k], u[k], q2);
    }
    const double H = fma(wR, HR - HL, HL);
    const double c2 = (g - 1.0) * fma(-0.5, q2, H);
    const double ic = rsqrt_h3(c2);
    const double c = c2 * ic, ic2 = ic * ic;
    const double dqn = qR - qL;
    const double qn = fma(wR, dqn, qL);
    const double drho = UR[0] - UL[0], dp = (g - 1.0) * (iR - iL);
    const double rq = rho * c * dqn, hc = 0.5 * ic2;
    const double qr = ROT ? qn - vrn : qn;
    const double l2 = fabs(qr);
    const double w1 = fabs(qr - c) * ((dp - rq) * hc), w5 = fabs(qr + c) * ((dp + rq) * hc);
    const double w2 = l2 * fma(-dp, ic2, drho), ws = l2 * rho;
    const double w15 = w1 + w5, d0 = w15 + w2, dc = (w5 - w1) * c;
    const double mL = ROT ? qL - vrn : qL, mR = ROT ? qR - vrn : qR;   // transport velocities
    const double fL = UL[0] * mL, fR = UR[0] * mR, ha = 0.5 * am;
    F[0] = ha * ((fL + fR) - d0);
    // momentum: F_L + F_R - (d0 u + dc n + ws (dv - dqn n))
    const double pn = (pL + pR) - fma(-ws, dqn, dc);
    double ud = 0.0;
#pragma unroll
    for (int k = 0; k < NK; ++k) {
        const double a = fma(UL[1 + k], mL, UR[1 + k] * mR);
        F[1 + k] = ha * (fma(pn, n[k], a) - fma(d0, u[k], ws * dv[k]));
        ud = fma(u[k], dv[k], ud);
    }
    if (NK == 2) F[3] = 0.0;
    // energy: w15 H + w2 q2/2 + dc qn + ws (u . dv - qn dqn)
    const double d4 = fma(w15, H, fma(w2, 0.5 * q2, fma(dc, qn, ws * fma(-qn, dqn, ud))));
    const double eL = ROT ? fma(UL[4], mL, pL * qL) : EL * qL, eR = ROT ? fma(UR[4], mR, pR * qR) : ER * qR;
    F[4] = ha * ((eL + eR) - d4);
}

// The far field of euler.cuh's farfield_ghost in float64 with the free stream's constants formed on
// the host and one power: with s = p / rho^g of the upwind side, (c_b^2 / (g s))^(1/(g-1)) is
// rho (c_b^2 / c^2)^(1/(g-1)) in that side's rho and c.  For g = 7/5 the power is x^2 sqrt(x).
struct FarField {
    double v[3], rho, c, ic2, ex;   // free stream: velocity, density, c, 1 / c^2; 1 / (g - 1)
    int half5;                      // ex = 5/2 to rounding
};
__device__ __forceinline__ void farfield_fast(const double UL[5], const double n[3], const FarField& ff, double g,
                                              double G[5]) {
    const double ir = rcp_h3(UL[0]);
    double v[3], ke = 0.0, qL = 0.0, qi = 0.0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        v[k] = UL[1 + k] * ir;
        ke = fma(UL[1 + k], v[k], ke);
        qL = fma(v[k], n[k], qL);
        qi = fma(ff.v[k], n[k], qi);
    }
    const double p = (g - 1.0) * fma(-0.5, ke, UL[4]);
    const double c2 = g * p * ir, ic = rsqrt_h3(c2), c = c2 * ic;
    const double Rp = fma(2.0 * ff.ex, c, qL), Rm = fma(-2.0 * ff.ex, ff.c, qi);
    const double qb = 0.5 * (Rp + Rm), cb = 0.25 * (g - 1.0) * (Rp - Rm), cb2 = cb * cb;
    const bool in = qb < 0.0;
    const double x = cb2 * (in ? ff.ic2 : ic * ic);
    const double pw = ff.half5 ? x * x * (x * rsqrt_h3(x)) : pow(x, ff.ex);
    const double rb = (in ? ff.rho : UL[0]) * pw;
    const double dq = qb - (in ? qi : qL);
    double vb[3], kb = 0.0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        vb[k] = fma(dq, n[k], in ? ff.v[k] : v[k]);
        kb = fma(vb[k], vb[k], kb);
        G[1 + k] = rb * vb[k];
    }
    G[0] = rb;
    G[4] = rb * fma(cb2 / g, ff.ex, 0.5 * kb);
}

// One thread per face point, whole faces in a block.  Bound by the float64 pipe (its point flux,
// about 120 operations).  The boundary faces, numbered last and with the longest paths, start
// first.  p >= 1: the fluxes leave as fixed point, one exponent for each face and variable (its
// largest key, in fkey), ready for the projections of both neighbours: rows of 6 pairs, the last
// one unused.  p = 0: float64 rows of 5.
template <int D, int P>
struct FaceCfg {
    static constexpr int QF = Lv<D, P>::QF;
    static constexpr int FB = QF == 36 ? 8 : 128 / QF;               // faces per block (9 warps, or 4)
    static constexpr int THREADS = (FB * QF + 31) / 32 * 32;
};
template <int D, int P, bool ROT>
__global__ void __launch_bounds__(FaceCfg<D, P>::THREADS) k_face_flux(int F, int F_int, const int* __restrict__ fL,
                                                   const int* __restrict__ fR, const int* __restrict__ fbc,
                                                   const double* __restrict__ fnrm,
                                                   const double* __restrict__ famag,
                                                   const double* __restrict__ fpsiL,
                                                   const double* __restrict__ fpsiR,
                                                   const double* __restrict__ fwn,
                                                   const double* __restrict__ u, const double* __restrict__ tr,
                                                   double g, U5 uinf, FarField ff,
                                                   const double* __restrict__ fvr, double* __restrict__ fhat,
                                                   int* __restrict__ fkey) {
    chain_wait();
    using CF = FaceCfg<D, P>;
    constexpr int QF = CF::QF, FB = CF::FB;
    __shared__ int mx[FB * 5];
    const int fb = F - FB * ((int)blockIdx.x + 1);   // the block's first face (negative in the last block)
    const int lf = threadIdx.x / QF, f = fb + lf;
    const bool live = lf < FB && f >= 0;
    if constexpr (P > 0) {
        for (int t = threadIdx.x; t < FB * 5; t += CF::THREADS) mx[t] = 0;
        __syncthreads();
    }
    double Fl[5];
    const int64_t idx = (int64_t)f * QF + threadIdx.x % QF;
    if (live) {
        const double n[3] = {fnrm[idx * 3], fnrm[idx * 3 + 1], fnrm[idx * 3 + 2]};
        const bool inner = f < F_int;
        double UL[5], UR[5];
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
        if (inner) {
        } else if (fbc[f] == EMG_BC_WALL || fbc[f] == EMG_BC_SYMMETRY) {
            // mirror ghost about the reflection normal (body normal on walls, face normal on
            // symmetry planes)
            const int64_t bi = idx - (int64_t)F_int * QF;
            const double nw[3] = {fwn[bi * 3], fwn[bi * 3 + 1], fwn[bi * 3 + 2]};
            if constexpr (ROT) {
                const double vr[3] = {fvr[idx * 3], fvr[idx * 3 + 1], fvr[idx * 3 + 2]};
                wall_ghost_rel(UL, nw, vr, g, UR);
            } else {
                wall_ghost(UL, nw, UR);
            }
        } else {
            if constexpr (ROT) {
                const double vr[3] = {fvr[idx * 3], fvr[idx * 3 + 1], fvr[idx * 3 + 2]};
                farfield_ghost_rel(UL, n, uinf.v, g, vr, UR);
            } else {
                farfield_fast(UL, n, ff, g, UR);
            }
        }
        double vrn = 0.0;
        if constexpr (ROT) vrn = fvr[idx * 3] * n[0] + fvr[idx * 3 + 1] * n[1] + fvr[idx * 3 + 2] * n[2];
        const double am = famag[idx];
        if (D == 2 && UL[3] == 0.0 && UR[3] == 0.0)   // n[2] = 0 in 2-D
            roe_flux_fast<2, ROT>(UL, UR, n, g, vrn, am, Fl);
        else
            roe_flux_fast<3, ROT>(UL, UR, n, g, vrn, am, Fl);
    }
    if constexpr (P == 0) {
        if (live)
#pragma unroll
            for (int a = 0; a < 5; ++a) fhat[idx * 5 + a] = Fl[a];
    } else {
        if (live)
#pragma unroll
            for (int a = 0; a < 5; ++a) atomicMax(&mx[lf * 5 + a], fix_key(Fl[a]));
        __syncthreads();
        for (int t = threadIdx.x; t < FB * 5; t += CF::THREADS)
            if (fb * 5 + t >= 0) fkey[(int64_t)fb * 5 + t] = mx[t];
        if (!live) return;
        int2 v[5];
#pragma unroll
        for (int a = 0; a < 5; ++a) v[a] = fix_of(Fl[a], fix_exp(mx[lf * 5 + a]));
        int4* o = reinterpret_cast<int4*>(fhat) + idx * 3;
        o[0] = make_int4(v[0].x, v[0].y, v[1].x, v[1].y);
        o[1] = make_int4(v[2].x, v[2].y, v[3].x, v[3].y);
        o[2] = make_int4(v[4].x, v[4].y, 0, 0);
    }
}

// ---- volume quadrature and projection -------------------------------------------------------------
// A block holds ET elements.  Points: thread (element, point) reconstructs U_h and its flux;
// projections: thread (element, mode i) accumulates the five variables of R_{e,a,i}.  The fluxes
// are staged in shared memory, first as float64, then in place as fixed point once the largest of
// each (element, direction, variable) is known: QC volume points at a time (all of them in 2-D), then
// the faces', FC faces at a time as k_face_flux left them.  Each direction has accumulators of its
// own, so that its gradients and fluxes keep exponents of their own (fix.cuh).
// S = false: a thread per mode, several elements a block (most work in flight per instruction
// issued).  S = true, for meshes that leave the chip short of warps: four threads per mode, each
// with a quarter of the rows, and fewer elements a block, so that each warp's chain of instructions
// is a quarter as long.
template <int D, int P, bool S>
struct VolCfg {
    using L = Lv<D, P>;
    static constexpr int PARTS = S ? 4 : 1;
    static constexpr int TM = L::N * PARTS;                          // threads of an element's projection
    static constexpr int THREADS = S ? (TM <= 64 ? 64 : (TM + 31) / 32 * 32) : (D == 2 || L::N == 20) ? 64 : 128;
    static constexpr int ET = THREADS / TM;                          // elements per block
    static_assert(S || P == 0 || ET == volume_elems(D, P), "residual_chain.h");
    static constexpr int FS = 6;                                     // padded variable stride
    static constexpr int QMAX = 54;                                  // points of one exact sum (more: no faster)
    static constexpr int QS = THREADS * 288 / (ET * D * FS * 8);     // points that fit the buffer
    static constexpr int QC0 = QS < QMAX ? QS : QMAX;
    static constexpr int QC = QC0 < L::Q ? QC0 & ~1 : L::Q;          // points per chunk (even, or all)
    static constexpr int FC0 = (QC * D) / L::QF;                     // faces that fit the same buffer
    static constexpr int FC1 = FC0 < FIX_TERMS / L::QF ? FC0 : FIX_TERMS / L::QF;
    static constexpr int FC = FC1 < 1 ? 1 : (FC1 > L::NF ? L::NF : FC1);
    // the directions' sums are added with SH bits less: D QC 2^(56 - SH) < 2^63
    static constexpr int SH = D * QC > 120 ? 1 : 0;
    static constexpr int ROWS = QC * D > FC * L::QF ? QC * D : FC * L::QF;
    // 128 registers a thread; the quarter rows of 2-D p = 3, which fit fewer, ten blocks (50 x 25: 41.4 -> 35.8 us)
    static constexpr int MINB = S && D == 2 && P == 3 ? 10 : 512 / THREADS;
    static_assert(QC >= 2 && FC * L::QF <= FIX_TERMS && QC <= FIX_TERMS && D * QC <= 252 && L::N <= FIX_TERMS, "exact sums");
};

// Largest of the keys that the warp's lanes hold for their elements, one atomic per element and key.
template <int K>
__device__ __forceinline__ void row_max(int* mx, int el, const int key[K]) {
    const unsigned grp = __match_any_sync(__activemask(), el);
    const bool lead = (threadIdx.x & 31) == __ffs(grp) - 1;
#pragma unroll
    for (int a = 0; a < K; ++a) {
        const int m = __reduce_max_sync(grp, key[a]);
        if (lead && m > 0) atomicMax(&mx[el * K + a], m);
    }
}

// A row of five float64 in shared memory turned into fixed point in place (ex: their groups' exponents).
template <int D>
__device__ __forceinline__ void row_fix(double* row, const int* ex) {
    double2* r2 = reinterpret_cast<double2*>(row);
    const double2 a = r2[0], b = r2[1];
    const int2 v0 = fix_of(a.x, ex[0]), v1 = fix_of(a.y, ex[1]);
    const int2 v2 = fix_of(b.x, ex[2]), v4 = fix_of(row[4], ex[4]);
    int2 v3 = make_int2(0, 0);
    if (D == 3 || ex[3] != fix_exp(0)) v3 = fix_of(b.y, ex[3]);
    int4* o = reinterpret_cast<int4*>(row);
    o[0] = make_int4(v0.x, v0.y, v1.x, v1.y);
    o[1] = make_int4(v2.x, v2.y, v3.x, v3.y);
    reinterpret_cast<int2*>(row)[4] = v4;
}

// The largest |F_k,a| over an element's points, from above, of a frame at rest: keys of the largest |rho v_1..3|,
// 1 / rho, |p|, |rho E + p|.  A reduction of each of the D x 5 fluxes instead took a tenth of a 3-D residual
// (16 x 16 x 20 hexes a patch, p = 1: 478 us, with five reductions 435); the bound costs no accuracy
// (rms error of the volume sums in emulation, states at 10 % and near stagnation: the same to 2 %).
__device__ __forceinline__ int flux_bound_key(const int* key, int k, int a) {
    auto up = [](int x) { return x == 0 ? 0.0 : __hiloint2double(x + 1, 0); };
    const double m = up(key[k]), v = m * up(key[3]);
    const double b = a == 0 ? m : a == 4 ? up(key[5]) * v : fma(up(key[a - 1]), v, a == 1 + k ? up(key[4]) : 0.0);
    return fix_key(b);
}

__device__ __forceinline__ void row_put(double* row, const double v[5]) {
    reinterpret_cast<double2*>(row)[0] = make_double2(v[0], v[1]);
    reinterpret_cast<double2*>(row)[1] = make_double2(v[2], v[3]);
    row[4] = v[4];
}

// One table entry p times the five variables of a row (W: with the spanwise momentum).
template <bool W>
__device__ __forceinline__ void row_mac(long long* h, long long* c, int2 p, const int4* r) {
    const int4 a = r[0], b = r[1];
    const int2 d = reinterpret_cast<const int2*>(r)[4];
    fix_mac(h[0], c[0], p, make_int2(a.x, a.y));
    fix_mac(h[1], c[1], p, make_int2(a.z, a.w));
    fix_mac(h[2], c[2], p, make_int2(b.x, b.y));
    if (W) fix_mac(h[3], c[3], p, make_int2(b.z, b.w));
    fix_mac(h[4], c[4], p, d);
}

// h, c += sum over a thread's share of `rows` rows of table entry (row, mode) times the row; tab:
// the thread's first entry of the row range (paired: mode i at 2 i); of PARTS threads, thread
// `part` takes every PARTS-th pair.  Row t goes to the sums of direction t % ND (ND = 3: a thread takes
// three pairs, two points, at a time, so that a row's direction is known when compiling).  The G loads
// of a group are issued ahead of its sums, the next group's during them.  R: the number of rows where
// it is known at compile time, else 0.
template <bool W, int ND, int N, bool PAIRED, int PARTS, int R>
__device__ __forceinline__ void rows_mac(long long (&h)[ND * 5], long long (&c)[ND * 5], const int2* __restrict__ tab,
                                         const double* row, int rows, int part) {
    static_assert(ND == 1 || PAIRED, "directions only in paired tables");
    const int4* r = reinterpret_cast<const int4*>(row);
    constexpr int K = R / 2 / PARTS;   // pairs of a thread, when they are the same for all
    constexpr bool EVEN = PAIRED && R > 0 && R % (2 * PARTS) == 0 && ND < 3;
    constexpr int S = ND == 2 ? 5 : 0;   // the second row of a pair
    constexpr int G = !EVEN ? (ND == 2 ? 2 : 4) : K % 4 == 0 ? 4 : K % 5 == 0 ? 5 : K % 3 == 0 ? 3 : K % 2 == 0 ? 2 : 1;
    if constexpr (EVEN) {
        const int4* t4 = reinterpret_cast<const int4*>(tab) + part * N;
        r += part * 6;
        int4 p[G];
#pragma unroll
        for (int g = 0; g < G; ++g) p[g] = t4[g * PARTS * N];
#pragma unroll(K <= 4 * G ? K / G : 1)
        for (int m0 = 0; m0 < K - G; m0 += G) {
            int4 nx[G];
#pragma unroll
            for (int g = 0; g < G; ++g) nx[g] = t4[(m0 + G + g) * PARTS * N];
#pragma unroll
            for (int g = 0; g < G; ++g) {
                row_mac<W>(h, c, make_int2(p[g].x, p[g].y), r + (m0 + g) * PARTS * 6);
                row_mac<W>(h + S, c + S, make_int2(p[g].z, p[g].w), r + (m0 + g) * PARTS * 6 + 3);
                p[g] = nx[g];
            }
        }
#pragma unroll
        for (int g = 0; g < G; ++g) {
            row_mac<W>(h, c, make_int2(p[g].x, p[g].y), r + (K - G + g) * PARTS * 6);
            row_mac<W>(h + S, c + S, make_int2(p[g].z, p[g].w), r + (K - G + g) * PARTS * 6 + 3);
        }
    } else if constexpr (ND == 3) {
        const int pairs = rows >> 1;
        const int4* t4 = reinterpret_cast<const int4*>(tab);
        int4 p[3];
#pragma unroll
        for (int g = 0; g < 3; ++g)
            if (3 * part + g < pairs) p[g] = t4[(3 * part + g) * N];
#pragma unroll 1
        for (int m0 = 3 * part; m0 < pairs; m0 += 3 * PARTS) {
            int4 nx[3];
#pragma unroll
            for (int g = 0; g < 3; ++g)
                if (m0 + 3 * PARTS + g < pairs) nx[g] = t4[(m0 + 3 * PARTS + g) * N];
#pragma unroll
            for (int g = 0; g < 3; ++g) {
                const int m = m0 + g;
                if (m < pairs) {
                    row_mac<W>(h + 2 * g % 3 * 5, c + 2 * g % 3 * 5, make_int2(p[g].x, p[g].y), r + m * 6);
                    row_mac<W>(h + (2 * g + 1) % 3 * 5, c + (2 * g + 1) % 3 * 5, make_int2(p[g].z, p[g].w), r + m * 6 + 3);
                }
                p[g] = nx[g];
            }
        }
    } else if constexpr (PAIRED) {
        const int pairs = rows >> 1;
        const int4* t4 = reinterpret_cast<const int4*>(tab);
        int4 p[G];
#pragma unroll
        for (int g = 0; g < G; ++g)
            if (part + g * PARTS < pairs) p[g] = t4[(part + g * PARTS) * N];
#pragma unroll 1
        for (int m0 = part; m0 < pairs; m0 += G * PARTS) {
            int4 nx[G];
#pragma unroll
            for (int g = 0; g < G; ++g)
                if (m0 + (G + g) * PARTS < pairs) nx[g] = t4[(m0 + (G + g) * PARTS) * N];
#pragma unroll
            for (int g = 0; g < G; ++g) {
                const int m = m0 + g * PARTS;
                if (m < pairs) {
                    row_mac<W>(h, c, make_int2(p[g].x, p[g].y), r + m * 6);
                    row_mac<W>(h + S, c + S, make_int2(p[g].z, p[g].w), r + m * 6 + 3);
                }
                p[g] = nx[g];
            }
        }
    } else {
#pragma unroll 3
        for (int t = part; t < rows; t += PARTS) row_mac<W>(h, c, tab[t * N], r + t * 3);
    }
}

template <int D, int P, bool ROT, bool S>
__global__ void __launch_bounds__(VolCfg<D, P, S>::THREADS, VolCfg<D, P, S>::MINB) k_volume(
    int E, const double* __restrict__ u, const int2* __restrict__ vpsi, const int2* __restrict__ vgw,
    const int* __restrict__ elem_face, const int2* __restrict__ fpsiL, const int2* __restrict__ fpsiR,
    const int* __restrict__ texp, const int* __restrict__ gexp, const int4* __restrict__ fhat,
    const int* __restrict__ fkey, const double* __restrict__ tau, double g,
    const double* __restrict__ vvr, U5 om, double* __restrict__ R) {
    chain_wait();
    using L = Lv<D, P>;
    using CF = VolCfg<D, P, S>;
    using GT = GradTab<D, P>;
    using FT = FaceTab<D, P>;
    constexpr int N = L::N, Q = L::Q, QF = L::QF, B = L::B, NF = L::NF;
    constexpr int ET = CF::ET, QC = CF::QC, FS = CF::FS, T = CF::THREADS, FC = CF::FC, ROWS = CF::ROWS;
    constexpr int PARTS = CF::PARTS;
    constexpr int RV = Q == QC ? Q * D : 0;   // rows of the volume term when it is one chunk
    constexpr int KEYS = ROT ? D * 5 : 6;     // a point's: of every flux, or those of flux_bound_key
    __shared__ __align__(16) int2 us[ET * N * FS];          // [ET][N][6] coefficients
    __shared__ __align__(16) double Fs[ET * ROWS * FS];     // [ET][rows][6] staged fluxes
    __shared__ int mxu[ET * 5], mx[ET * KEYS];            // largest keys, of a chunk
    __shared__ int codes[ET * NF], ex[ET * D * 5];          // ex: exponents of the stage's fluxes
    const int e0 = blockIdx.x * ET;
    for (int t = threadIdx.x; t < ET * KEYS; t += T) {
        if (t < ET * 5) mxu[t] = 0;
        mx[t] = 0;
    }
    for (int t = threadIdx.x; t < ET * NF; t += T)
        codes[t] = e0 + t / NF < E ? elem_face[(size_t)e0 * NF + t] : 0;
    const int ne = E - e0 < ET ? E - e0 : ET;
    constexpr int NU = (ET * B + T - 1) / T;
    double x[NU];
#pragma unroll
    for (int k = 0; k < NU; ++k) {
        const int t = threadIdx.x + k * T;
        x[k] = (t < ET * B && e0 + t / B < E) ? u[(size_t)e0 * B + t] : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < NU; ++k) {
        const int t = threadIdx.x + k * T;
        if (t < ET * B) atomicMax(&mxu[t / N], fix_key(x[k]));   // t / N = element * 5 + variable
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < NU; ++k) {
        const int t = threadIdx.x + k * T;
        if (t < ET * B) us[((t / B) * N + t % N) * FS + (t / N) % 5] = fix_of(x[k], fix_exp(mxu[t / N]));
    }
    // this thread's (element, mode, part of the rows)
    const int el2 = threadIdx.x / CF::TM, i2 = threadIdx.x % CF::TM / PARTS, part = threadIdx.x % PARTS;
    const int e2 = e0 + el2;
    const bool own = el2 < ET && e2 < E;
    double acc[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    // exact sums to acc: the scale is 2^(56 - s_table - s_flux), NaN for a non-finite flux
    auto add_sums = [&](const long long* h, const long long* c, int st, const int* keys, bool w) {
#pragma unroll
        for (int a = 0; a < 5; ++a) {
            if (a == 3 && !w) continue;
            const int key = keys[a];
            acc[a] += fix_sum(h[a], c[a], fix_scale(FIX_BITS - st - fix_exp(key), key));
        }
    };
#pragma unroll 1
    for (int q0 = 0; q0 < Q; q0 += QC) {
        const int nq = (Q - q0) < QC ? (Q - q0) : QC;
        __syncthreads();   // us staged / previous chunk consumed
        // (1) U_h and the Euler flux at the chunk's points
        for (int t = threadIdx.x; t < ET * nq; t += T) {
            const int el = t / nq, qq = t % nq, e = e0 + el;
            if (e >= E) break;
            const int2* pr = vpsi + (size_t)e * Q * N + q0 + qq;
            const int4* ur = reinterpret_cast<const int4*>(us + el * N * FS);
            const bool w = D == 3 || mxu[el * 5 + 3] != 0;   // 2-D flow without a spanwise momentum: 0
            long long h[5] = {0, 0, 0, 0, 0}, c[5] = {0, 0, 0, 0, 0};
            if (w) {
#pragma unroll 5
                for (int i = 0; i < N; ++i) row_mac<true>(h, c, pr[i * Q], ur + i * 3);
            } else {
#pragma unroll 5
                for (int i = 0; i < N; ++i) row_mac<false>(h, c, pr[i * Q], ur + i * 3);
            }
            const int st = texp[e];
            double U[5];
#pragma unroll
            for (int a = 0; a < 5; ++a) {
                const int key = mxu[el * 5 + a];
                U[a] = (a != 3 || w) ? fix_sum(h[a], c[a], fix_scale(FIX_BITS - st - fix_exp(key), key)) : 0.0;
            }
            double vr[3] = {0.0, 0.0, 0.0};
            if constexpr (ROT) {   // F_k - (v_r)_k U
                const double* r = vvr + ((size_t)e * Q + q0 + qq) * 3;
#pragma unroll
                for (int k = 0; k < D; ++k) vr[k] = r[k];
            }
            const double ir = rcp_h3(U[0]);
            const double v0 = U[1] * ir, v1 = U[2] * ir, v2 = U[3] * ir;
            double ke = fma(U[1], v0, U[2] * v1);
            if (w) ke = fma(U[3], v2, ke);
            const double pr_ = (g - 1.0) * fma(-0.5, ke, U[4]);
            const double H = U[4] + pr_;
            const double vv[3] = {v0, v1, v2};
            int key[KEYS];
            if constexpr (!ROT) {
                key[0] = fix_key(U[1]), key[1] = fix_key(U[2]), key[2] = fix_key(U[3]);
                key[3] = fix_key(ir), key[4] = fix_key(pr_), key[5] = fix_key(H);
            }
#pragma unroll
            for (int k = 0; k < D; ++k) {
                double Fk[5];
                Fk[0] = U[1 + k];
                Fk[1] = fma(U[1], vv[k], k == 0 ? pr_ : 0.0);
                Fk[2] = fma(U[2], vv[k], k == 1 ? pr_ : 0.0);
                Fk[3] = w ? fma(U[3], vv[k], k == 2 ? pr_ : 0.0) : 0.0;
                Fk[4] = H * vv[k];
                if constexpr (ROT) {
#pragma unroll
                    for (int a = 0; a < 5; ++a) Fk[a] = fma(-vr[k], U[a], Fk[a]);
                }
                if constexpr (ROT) {
#pragma unroll
                    for (int a = 0; a < 5; ++a) key[k * 5 + a] = fix_key(Fk[a]);
                }
                row_put(Fs + ((size_t)el * nq * D + qq * D + k) * FS, Fk);
            }
            row_max<KEYS>(mx, el, key);
        }
        __syncthreads();
        for (int t = threadIdx.x; t < ET * D * 5; t += T) {
            int key;
            if constexpr (ROT)
                key = mx[t];
            else
                key = flux_bound_key(mx + t / (D * 5) * KEYS, t / 5 % D, t % 5);
            ex[t] = key >= 0x7ff00000 ? FIX_NAN : fix_exp(key);
        }
        __syncthreads();
        for (int t = threadIdx.x; t < ne * D * nq; t += T)
            row_fix<D>(Fs + (size_t)t * FS, ex + (t / (D * nq) * D + t % D) * 5);
        __syncthreads();
        for (int t = threadIdx.x; t < ET * KEYS; t += T) mx[t] = 0;   // for the next chunk
        // (2) projection on the gradients: sum_q sum_k W_q d_k psi_i F_k,a
        if (own) {
            long long h[D * 5], c[D * 5];
#pragma unroll
            for (int a = 0; a < D * 5; ++a) h[a] = c[a] = 0;
            const int2* tab = vgw + (size_t)e2 * D * Q * N + (size_t)q0 * D * N + 2 * i2;
            const double* row = Fs + (size_t)el2 * nq * D * FS;
            const int* e5 = ex + el2 * D * 5;
            int rows = nq * D, ge[D];
#pragma unroll
            for (int k = 0; k < D; ++k) ge[k] = gexp[((size_t)e2 * D + k) * N + i2];
            const bool w = D == 3 || e5[3] != fix_exp(0) || e5[8] != fix_exp(0);
            if (w)
                rows_mac<true, D, N, GT::paired, PARTS, RV>(h, c, tab, row, rows, part);
            else
                rows_mac<false, D, N, GT::paired, PARTS, RV>(h, c, tab, row, rows, part);
            if (D == 3 && (rows & 1) && part == 0) {   // the last row of an odd number: direction 2
                --rows;
                row_mac<true>(h + (D - 1) * 5, c + (D - 1) * 5, (tab - i2)[(size_t)rows * N],
                              reinterpret_cast<const int4*>(row) + rows * 3);
            }
            // the directions' sums at the largest one's exponent, then one conversion a variable (the
            // float64 pipe's): the cut is 2^-56 of (largest gradient) (largest flux) of that direction
#pragma unroll
            for (int a = 0; a < 5; ++a) {
                if (a == 3 && !w) continue;
                int ek[D], lo = 0x7fffffff;
#pragma unroll
                for (int k = 0; k < D; ++k) {
                    ek[k] = ge[k] + e5[k * 5 + a];
                    lo = min(lo, ek[k]);
                }
                long long s = 0;
#pragma unroll
                for (int k = 0; k < D; ++k) s += (h[k * 5 + a] + (c[k * 5 + a] >> FIX_LO)) >> min(ek[k] - lo + CF::SH, 63);
                acc[a] += __ll2double_rn(s) * fix_scale(FIX_BITS + CF::SH - lo);
            }
        }
    }
    // (3) faces: -(L side) / +(R side) sum_t psi_i(x_t) w|n dS| F~_a.  A row is shifted from its
    // face's exponent to the largest of the stage's faces.
#pragma unroll 1
    for (int f0 = 0; f0 < NF; f0 += FC) {
        const int nf = (NF - f0) < FC ? (NF - f0) : FC;
        __syncthreads();
        for (int t = threadIdx.x; t < ne * 5; t += T) {
            int k = 0;
            for (int lf = 0; lf < nf; ++lf) k = max(k, fkey[(size_t)(codes[t / 5 * NF + f0 + lf] >> 1) * 5 + t % 5]);
            mxu[t] = k;   // the coefficients' keys are no longer needed
        }
        __syncthreads();
        for (int t = threadIdx.x; t < ne * nf * QF; t += T) {
            const int el = t / (nf * QF), r = t % (nf * QF);
            const int code = codes[el * NF + f0 + r / QF];
            const int4* src = fhat + ((size_t)(code >> 1) * QF + r % QF) * 3;
            const int* key = fkey + (size_t)(code >> 1) * 5;
            const int4 a = src[0], b = src[1];
            const int2 d = *reinterpret_cast<const int2*>(src + 2);
            const int2 v[5] = {make_int2(a.x, a.y), make_int2(a.z, a.w), make_int2(b.x, b.y), make_int2(b.z, b.w), d};
            int2 o[5];
#pragma unroll
            for (int k = 0; k < 5; ++k) o[k] = fix_shift(v[k], fix_exp(key[k]) - fix_exp(mxu[el * 5 + k]), !(code & 1));
            int4* dst = reinterpret_cast<int4*>(Fs + (size_t)t * FS);
            dst[0] = make_int4(o[0].x, o[0].y, o[1].x, o[1].y);
            dst[1] = make_int4(o[2].x, o[2].y, o[3].x, o[3].y);
            *reinterpret_cast<int2*>(dst + 2) = o[4];
        }
        __syncthreads();
        if (own) {
            long long h[5] = {0, 0, 0, 0, 0}, c[5] = {0, 0, 0, 0, 0};
            const bool w = D == 3 || mxu[el2 * 5 + 3] != 0;
#pragma unroll(D == 2 ? 2 : 1)
            for (int lf = 0; lf < nf; ++lf) {
                const int code = codes[el2 * NF + f0 + lf];
                const int2* side = ((code & 1) ? fpsiR : fpsiL) + (size_t)(code >> 1) * QF * N;
                const int2* tab = side + (FT::paired ? 2 * i2 : i2);
                const double* row = Fs + (size_t)(el2 * nf + lf) * QF * FS;
                if (w)
                    rows_mac<true, 1, N, FT::paired, PARTS, QF>(h, c, tab, row, QF, part);
                else
                    rows_mac<false, 1, N, FT::paired, PARTS, QF>(h, c, tab, row, QF, part);
                if (FT::paired && (QF & 1) && part == 0)
                    row_mac<true>(h, c, side[(QF - 1) * N + i2], reinterpret_cast<const int4*>(row) + (QF - 1) * 3);
            }
            add_sums(h, c, texp[e2], mxu + el2 * 5, w);
        }
    }
    if constexpr (PARTS > 1) {   // the parts' sums of a mode, on neighbouring lanes
        const unsigned live = __ballot_sync(0xffffffffu, own);
        if (own) {
#pragma unroll
            for (int a = 0; a < 5; ++a)
#pragma unroll
                for (int o = 1; o < PARTS; o <<= 1) acc[a] += __shfl_xor_sync(live, acc[a], o);
        }
    }
    if (!own || part != 0) return;
    if constexpr (ROT) {   // source: -omega x (rho v)_i
        const double* ue = u + (size_t)e2 * B + i2;
        const double mx_ = ue[1 * N], my = ue[2 * N], mz = ue[3 * N];
        acc[1] -= om.v[1] * mz - om.v[2] * my;
        acc[2] -= om.v[2] * mx_ - om.v[0] * mz;
        acc[3] -= om.v[0] * my - om.v[1] * mx_;
    }
    double* Re = R + (size_t)e2 * B + i2;
    const double* tu = tau ? tau + (size_t)e2 * B + i2 : nullptr;
#pragma unroll
    for (int a = 0; a < 5; ++a) Re[a * N] = tu ? acc[a] + tu[a * N] : acc[a];
}

// p = 0: thread (element) sums its faces' fluxes.
template <int D, bool ROT>
__global__ void __launch_bounds__(128) k_cell0(int E, const double* __restrict__ u, const int* __restrict__ elem_face,
                                               const double* __restrict__ fpsiL, const double* __restrict__ fpsiR,
                                               const double* __restrict__ fhat, const double* __restrict__ tau, U5 om,
                                               double* __restrict__ R) {
    chain_wait();
    using L = Lv<D, 0>;
    constexpr int QF = L::QF, NF = L::NF;
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= E) return;
    double acc[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int lf = 0; lf < NF; ++lf) {
        const int code = elem_face[(size_t)e * NF + lf];
        const int f = code >> 1;
        const double* ps = ((code & 1) ? fpsiR : fpsiL) + (size_t)f * QF;
        const double* fh = fhat + (size_t)f * QF * 5;
        double s[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
#pragma unroll
        for (int t = 0; t < QF; ++t)
#pragma unroll
            for (int a = 0; a < 5; ++a) s[a] += ps[t] * fh[t * 5 + a];
        const double sg = (code & 1) ? 1.0 : -1.0;
#pragma unroll
        for (int a = 0; a < 5; ++a) acc[a] += sg * s[a];
    }
    if constexpr (ROT) {
        const double* m = u + (size_t)e * 5 + 1;
        acc[1] -= om.v[1] * m[2] - om.v[2] * m[1];
        acc[2] -= om.v[2] * m[0] - om.v[0] * m[2];
        acc[3] -= om.v[0] * m[1] - om.v[1] * m[0];
    }
#pragma unroll
    for (int a = 0; a < 5; ++a) R[(size_t)e * 5 + a] = tau ? acc[a] + tau[(size_t)e * 5 + a] : acc[a];
}

// ---- fixed-point tables (set-up) --------------------------------------------------------------------
// One block per element: the exponents of its basis values (volume and own face points) and of its
// weighted gradients of each direction and mode, then its tables in place as fixed point and in the residual's layouts: vpsi
// from [Q][N] to [N][Q] (k_volume's threads, one per point, read it side by side), vgw from
// [D][Q][N] and the face sides from [QF][N] to row pairs.
template <int D, int P>
__global__ void __launch_bounds__(128) k_fix_tables(double* __restrict__ vpsi, double* __restrict__ vgw,
                                                    const int* __restrict__ elem_face, double* __restrict__ fpsiL,
                                                    double* __restrict__ fpsiR, int* __restrict__ texp,
                                                    int* __restrict__ gexp) {
    using L = Lv<D, P>;
    constexpr int N = L::N, Q = L::Q, QF = L::QF, NF = L::NF;
    extern __shared__ __align__(16) double buf[];   // [D][Q][N] at most
    __shared__ int mx, mxg[D * N];
    const int e = blockIdx.x, tid = threadIdx.x;
    double* vp = vpsi + (size_t)e * Q * N;
    double* vg = vgw + (size_t)e * D * Q * N;
    if (tid == 0) mx = 0;
    for (int t = tid; t < D * N; t += 128) mxg[t] = 0;
    __syncthreads();
    int a = 0;
    for (int t = tid; t < Q * N; t += 128) a = max(a, fix_key(vp[t]));
    for (int t = tid; t < D * Q * N; t += 128) atomicMax(&mxg[t / (Q * N) * N + t % N], fix_key(vg[t]));
    for (int lf = 0; lf < NF; ++lf) {
        const int code = elem_face[(size_t)e * NF + lf];
        const double* fp = ((code & 1) ? fpsiR : fpsiL) + (size_t)(code >> 1) * QF * N;
        for (int t = tid; t < QF * N; t += 128) a = max(a, fix_key(fp[t]));
    }
    atomicMax(&mx, a);
    __syncthreads();
    const int sa = fix_exp(mx);
    if (tid == 0) texp[e] = sa;
    for (int t = tid; t < D * N; t += 128) gexp[(size_t)e * D * N + t] = fix_exp(mxg[t]);
    for (int t = tid; t < Q * N; t += 128) buf[t] = vp[t];
    __syncthreads();
    for (int t = tid; t < Q * N; t += 128) reinterpret_cast<int2*>(vp)[t] = fix_round(buf[(t % Q) * N + t / Q], sa);
    __syncthreads();
    for (int t = tid; t < D * Q * N; t += 128) buf[t] = vg[t];
    __syncthreads();
    for (int t = tid; t < D * Q * N; t += 128) {
        const int r = GradTab<D, P>::row(t), i = GradTab<D, P>::mode(t);
        reinterpret_cast<int2*>(vg)[t] = fix_round(buf[((r % D) * Q + r / D) * N + i], fix_exp(mxg[r % D * N + i]));
    }
    for (int lf = 0; lf < NF; ++lf) {
        const int code = elem_face[(size_t)e * NF + lf];
        double* fp = ((code & 1) ? fpsiR : fpsiL) + (size_t)(code >> 1) * QF * N;
        __syncthreads();
        for (int t = tid; t < QF * N; t += 128) buf[t] = fp[t];
        __syncthreads();
        for (int t = tid; t < QF * N; t += 128)
            reinterpret_cast<int2*>(fp)[t] = fix_round(buf[FaceTab<D, P>::row(t) * N + FaceTab<D, P>::mode(t)], sa);
    }
}

// The level tables of p >= 1 (the p = 0 ones stay float64), after the float32 copies are made.
emg_status fix_tables(emg_ctx* c) {
    for (int p = 1; p <= c->p_max; ++p) {
        LevelDev& L = c->lv[p];
        const size_t sm = (size_t)c->dim * L.Q * L.N * sizeof(double);
#define EMG_FT(DD, PP)                                                                                          \
    if constexpr (PP > 0) {                                                                                     \
        EMG_CUDA_TRY(c, cudaFuncSetAttribute(k_fix_tables<DD, PP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm)); \
        ProfScope _ps(c, PC_SETUP);                                                                             \
        k_fix_tables<DD, PP><<<(unsigned)c->E, 128, sm, c->stream>>>(L.vpsi, L.vgw, c->elem_face, L.fpsiL, L.fpsiR, L.texp, L.gexp); \
    }
        EMG_DISPATCH_DP(c->dim, p, EMG_FT)
#undef EMG_FT
        EMG_CHECK_LAUNCH(c);
    }
    return EMG_OK;
}

// U_h at both sides of every face point of level p >= 1, to tr [F][QF][2][5].
emg_status launch_traces(emg_ctx* c, int p, const double* u, double* tr, int cls) {
    LevelDev& L = c->lv[p];
    const int E = (int)c->E;
#define EMG_TR(DD, PP)                                                                                          \
    if constexpr (PP > 0) {                                                                                     \
        using CF = TrCfg<DD, PP>;                                                                               \
        EMG_CUDA_TRY(c, cudaFuncSetAttribute(k_traces<DD, PP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CF::SMEM)); \
        ProfScope _ps(c, cls);                                                                                  \
        launch_chained(c, k_traces<DD, PP>, (unsigned)((E + CF::ET - 1) / CF::ET), CF::THREADS, CF::SMEM, \
            E, u, c->elem_face, reinterpret_cast<const int2*>(L.fpsiL), reinterpret_cast<const int2*>(L.fpsiR), \
            L.texp, tr);                                                                                        \
    }
    EMG_DISPATCH_DP(c->dim, p, EMG_TR)
#undef EMG_TR
    EMG_CHECK_LAUNCH(c);
    return EMG_OK;
}

// Below this many elements the projections take four threads per mode.  Where the line lies, measured per
// residual (one thread / four threads a mode), us: 2-D p = 1 8192 elements 55.5 / 50.5, 18432 82.2 / 82.9;
// p = 2 4608 45.4 / 45.6, 8192 59.7 / 72.1; p = 3 1152 38.2 / 34.1, 2048 45.3 / 47.9; p = 4 1152 39.2 / 37.1,
// 2048 48.1 / 51.5; 3-D p = 1 4608 103 / 80, 13824 209 / 212; p = 2 2352 130 / 109, 4608 184 / 200; p = 3
// 216 95 / 63, 900 143 / 145; p = 4 216 135 / 111, 900 226 / 272.
constexpr int vol_small_elems(int D, int P) {
    return D == 2 ? (P == 1 ? 16000 : P == 2 ? 4500 : 1500) : P == 1 ? 10000 : P == 2 ? 3500 : P == 3 ? 800 : 450;
}

emg_status launch_residual(emg_ctx* c, int p, const double* u, const double* tau, double* R) {
    LevelDev& L = c->lv[p];
    const int F = (int)c->F, Fi = (int)c->F_int, E = (int)c->E;
    U5 ui;
    for (int a = 0; a < 5; ++a) ui.v[a] = c->uinf[a];
    const double g = c->prm.gamma;
    U5 om{};
    for (int k = 0; k < 3; ++k) om.v[k] = c->prm.omega[k];
    FarField ff;
    ff.rho = ui.v[0];
    double q2 = 0.0;
    for (int k = 0; k < 3; ++k) ff.v[k] = ui.v[1 + k] / ui.v[0], q2 += ff.v[k] * ff.v[k];
    const double c2 = g * (g - 1.0) * (ui.v[4] / ui.v[0] - 0.5 * q2);
    ff.c = std::sqrt(c2), ff.ic2 = 1.0 / c2, ff.ex = 1.0 / (g - 1.0);
    ff.half5 = std::fabs(ff.ex - 2.5) < 1e-14;
    if (p > 0) {
        const emg_status st = launch_traces(c, p, u, L.tr, PC_RES_FACE);
        if (st != EMG_OK) return st;
    }
#define EMG_RES_ROT(DD, PP, RR)                                                                                 \
    {                                                                                                          \
        using FC = FaceCfg<DD, PP>;                                                                            \
        { ProfScope _ps(c, PC_RES_FACE); launch_chained(c, k_face_flux<DD, PP, RR>, (unsigned)((F + FC::FB - 1) / FC::FB), FC::THREADS, 0, \
            F, Fi, c->face_L, c->face_R, c->face_bc, L.fnrm, L.famag, L.fpsiL, L.fpsiR, L.fwn, u, L.tr, g, ui, ff,     \
            L.fvr, L.fhat, L.fkey); }                                                                                         \
        EMG_CHECK_LAUNCH(c);                                                                                   \
        ProfScope _ps(c, PC_RES_VOL);                                                                          \
        if constexpr (PP == 0) {                                                                               \
            launch_chained(c, k_cell0<DD, RR>, (unsigned)((E + 127) / 128), 128, 0, E, u, c->elem_face, L.fpsiL,   \
                L.fpsiR, L.fhat, tau, om, R);                                                                  \
        } else {                                                                                               \
            const bool small = E < vol_small_elems(DD, PP);                                                            \
            const int ET = small ? VolCfg<DD, PP, true>::ET : VolCfg<DD, PP, false>::ET;                       \
            const int T = small ? VolCfg<DD, PP, true>::THREADS : VolCfg<DD, PP, false>::THREADS;              \
            launch_chained(c, (small ? k_volume<DD, PP, RR, true> : k_volume<DD, PP, RR, false>), (unsigned)((E + ET - 1) / ET), T, 0, \
                E, u, reinterpret_cast<const int2*>(L.vpsi), reinterpret_cast<const int2*>(L.vgw),             \
                c->elem_face, reinterpret_cast<const int2*>(L.fpsiL), reinterpret_cast<const int2*>(L.fpsiR),  \
                L.texp, L.gexp, reinterpret_cast<const int4*>(L.fhat), L.fkey, tau, g, L.vvr, om, R);                                                         \
        }                                                                                                      \
    }
#define EMG_RES(DD, PP)                   \
    if (c->rot)                           \
        EMG_RES_ROT(DD, PP, true)         \
    else                                  \
        EMG_RES_ROT(DD, PP, false)
    EMG_DISPATCH_DP(c->dim, p, EMG_RES)
#undef EMG_RES
#undef EMG_RES_ROT
    EMG_CHECK_LAUNCH(c);
    return EMG_OK;
}

}  // namespace emg
