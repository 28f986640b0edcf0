// Exact Jacobian blocks (Sec. 3.3).  The face Jacobians dF~/dU_L, dF~/dU_R (forward-mode AD
// of the Roe flux) are in jac_face.cu, the tensor-core form of the float32 assembly in
// jac_tc.cu; here:
//  * k_diag_blocks: element-diagonal block of Eq. jac1,
//      D[(a,i),(b,j)] = sum_q psi_j(x_q) sum_k W_q d_k psi_i(x_q) A_k[a][b](U_q)
//                       - sum_{L faces} sum_t psi_i psi_j w|n dS| dF~/dU_L[a][b]
//                       + sum_{R faces} sum_t psi_i psi_j w|n dS| dF~/dU_R[a][b]
//    with A_k = dF_k/dU in closed form (Appendix, Eq. dfdu, omega = 0), written either as
//    D or as the PRK operator P = I/dtau - D with dtau of Eq. x3d.
//  * k_bsr0: the p = 0 Jacobian (Eqs. jac1, jac2) as one diagonal and 2d off-diagonal
//    5x5 blocks per element.
#include <algorithm>

#include <cuda_bf16.h>

#include "blocks.cuh"
#include "common.cuh"
#include "dispatch.cuh"
#include "euler.cuh"
#include "fix.cuh"
#include "jacobian.cuh"

namespace emg {

template <int D, int P>
struct DiagCfg {
    static constexpr int QC = D == 2 ? 32 : 16;  // volume points per shared-memory chunk
    static constexpr int THREADS = ((25 * Lv<D, P>::N + 31) / 32) * 32;
};

// Resident blocks asked of the register allocator: about 56 registers per thread for the
// FP32 blocks, 80 for FP64 (its 2N-register accumulator row).
template <int D, int P, class T>
struct DiagMinB {
    static constexpr int R = sizeof(T) == 4 ? 56 : 80;
    static constexpr int T_ = DiagCfg<D, P>::THREADS;
    static constexpr int V = (65536 / (T_ * R)) < 1 ? 1 : 65536 / (T_ * R);
};

// 16-byte vector of T (float4 or double2) for the broadcast reads of the staged basis rows.
template <class T>
struct Vec16;
template <>
struct Vec16<float> {
    using V = float4;
    static constexpr int L = 4;
    __device__ static void get(const float* p, float o[4]) {
        const float4 v = *reinterpret_cast<const float4*>(p);
        o[0] = v.x, o[1] = v.y, o[2] = v.z, o[3] = v.w;
    }
};
template <>
struct Vec16<double> {
    using V = double2;
    static constexpr int L = 2;
    __device__ static void get(const double* p, double o[2]) {
        const double2 v = *reinterpret_cast<const double2*>(p);
        o[0] = v.x, o[1] = v.y;
    }
};

// acc[j] += s * row[j], j < N, with the row read 16 bytes at a time (row padded to NP).
template <int N, int NP, class T>
__device__ __forceinline__ void axpy_row(T (&acc)[N], T s, const T* row) {
    constexpr int VL = Vec16<T>::L;
#pragma unroll
    for (int j0 = 0; j0 < NP; j0 += VL) {
        T v[VL];
        Vec16<T>::get(row + j0, v);
#pragma unroll
        for (int c = 0; c < VL; ++c)
            if (j0 + c < N) acc[j0 + c] += s * v[c];
    }
}

// One CTA per element; thread (a, b, i) accumulates row (a,i), columns (b, 0..N-1).
// T is the block precision: double (FP64 form) or float (FP32 block form, with float
// copies of the basis tables; state and face Jacobians are rounded to float on load).
template <int D, int P, class T>
__global__ void __launch_bounds__(DiagCfg<D, P>::THREADS, (DiagMinB<D, P, T>::V)) k_diag_blocks(
    int E, int nmax, const double* __restrict__ u, const T* __restrict__ vpsi, const T* __restrict__ vgw,
    const int* __restrict__ elem_face, const T* __restrict__ fpsiL, const T* __restrict__ fpsiR,
    const T* __restrict__ fjl, const T* __restrict__ fjr, const double* __restrict__ psic,
    const double* __restrict__ hlen, const double* __restrict__ cfl_dev, double g, int shifted,
    const double* __restrict__ vvr, const int* __restrict__ texp, const int* __restrict__ gexp, T* __restrict__ out) {
    using L = Lv<D, P>;
    constexpr int N = L::N, Q = L::Q, QF = L::QF, B = L::B, NF = L::NF;
    constexpr int QC = DiagCfg<D, P>::QC;
    constexpr bool FX = P > 0 && sizeof(T) == 8;   // the float64 tables of p >= 1 are fixed point
    constexpr int VL = Vec16<T>::L, NP = ((N + VL - 1) / VL) * VL;   // padded basis rows
    // the finished block goes out through shared memory (coalesced) when it fits
    constexpr bool STAGE = (size_t)B * B * sizeof(T) <= 24576;
    __shared__ double ud[B];
    __shared__ T us[B];
    __shared__ T As[QC][D][25];
    __shared__ __align__(16) T ps[QC][NP];
    __shared__ T gs[QC][D][N];
    __shared__ T Us[QC][5];
    __shared__ __align__(16) T fps[QF][NP];
    __shared__ T fjs[QF][25];
    __shared__ __align__(16) T ob[STAGE ? B * B : 1];
    __shared__ double s_dtau;
    const int e = blockIdx.x;
    const int tid = threadIdx.x;
    for (int t = tid; t < B; t += blockDim.x) {
        const double v = u[(size_t)e * B + t];
        ud[t] = v;
        us[t] = (T)v;
    }
    __syncthreads();
    if (tid == 0 && shifted) {
        double Uc[5];
        for (int a = 0; a < 5; ++a) {
            double s = 0.0;
            for (int i = 0; i < N; ++i) s += ud[a * N + i] * psic[(size_t)e * nmax + i];
            Uc[a] = s;
        }
        const double ir = 1.0 / Uc[0];
        const double vx = Uc[1] * ir, vy = Uc[2] * ir, vz = Uc[3] * ir;
        const double q2 = vx * vx + vy * vy + vz * vz;
        const double pr = (g - 1.0) * (Uc[4] - 0.5 * Uc[0] * q2);
        const double cs = sqrt(g * pr * ir);
        s_dtau = cfl_dev[0] * hlen[e] / ((2 * P + 1) * (sqrt(q2) + cs));
    }
    double s_psi = 1.0;
    if constexpr (FX) s_psi = fix_scale(-texp[e], 0);
    const bool active = tid < 25 * N;
    const int ab = tid / N, i = tid % N;
    const int a = ab / 5, b = ab % 5;
    T acc[N];
#pragma unroll
    for (int j = 0; j < N; ++j) acc[j] = (T)0;
    if (P > 0) {
        for (int q0 = 0; q0 < Q; q0 += QC) {
            const int nq = (Q - q0) < QC ? (Q - q0) : QC;
            __syncthreads();
            // stage the chunk's psi and W grad psi, and build U at its points (all threads)
            const T* pg = vpsi + ((size_t)e * Q + q0) * N;
            if constexpr (FX) {   // stored [N][Q]
                const int2* pf = reinterpret_cast<const int2*>(vpsi) + (size_t)e * Q * N + q0;
                for (int t = tid; t < nq * NP; t += blockDim.x) {
                    const int j = t / nq, q = t % nq;
                    ps[q][j] = j < N ? fix_back(pf[j * Q + q]) * s_psi : 0.0;
                }
                __syncthreads();
            } else {
                for (int t = tid; t < nq * NP; t += blockDim.x) {
                    const int q = t / NP, j = t % NP;
                    ps[q][j] = j < N ? pg[q * N + j] : (T)0;
                }
            }
            for (int t = tid; t < D * nq * N; t += blockDim.x) {
                const int k = t / (nq * N), r = t % (nq * N);
                if constexpr (FX)
                    gs[r / N][k][r % N] = fix_back(reinterpret_cast<const int2*>(
                        vgw)[(size_t)e * D * Q * N + GradTab<D, P>::at((q0 + r / N) * D + k, r % N)]) *
                        fix_scale(-gexp[((size_t)e * D + k) * N + r % N], 0);
                else
                    gs[r / N][k][r % N] = vgw[(((size_t)e * D + k) * Q + q0) * N + r];
            }
            for (int t = tid; t < nq * 5; t += blockDim.x) {
                const int q = t / 5, c = t % 5;
                const T* pq = FX ? ps[q] : pg + (size_t)q * N;
                T s = (T)0;
                for (int m = 0; m < N; ++m) s += us[c * N + m] * pq[m];
                Us[q][c] = s;
            }
            __syncthreads();
            for (int t = tid; t < nq * D; t += blockDim.x) {
                flux_jac_k(Us[t / D], (T)g, t % D, As[t / D][t % D]);
                if (vvr) {   // rotating frame: A_k - (v_r)_k I
                    const T vr = (T)vvr[((size_t)e * Q + q0 + t / D) * 3 + t % D];
#pragma unroll
                    for (int a = 0; a < 5; ++a) As[t / D][t % D][a * 6] -= vr;
                }
            }
            __syncthreads();
            if (active) {
                for (int t = 0; t < nq; ++t) {
                    T s = (T)0;
#pragma unroll
                    for (int k = 0; k < D; ++k) s += gs[t][k][i] * As[t][k][ab];
                    axpy_row<N, NP, T>(acc, s, ps[t]);
                }
            }
        }
    }
    // faces, one at a time: stage psi at its points and the face Jacobians of this
    // element's side (sign -1 on the L side, +1 on the R side)
#pragma unroll 1
    for (int lf = 0; lf < NF; ++lf) {
        const int code = elem_face[(size_t)e * NF + lf];
        const T* pt = ((code & 1) ? fpsiR : fpsiL) + ((size_t)(code >> 1) * QF) * N;
        const T* fj = ((code & 1) ? fjr : fjl) + ((size_t)(code >> 1) * QF) * 25;
        __syncthreads();
        for (int t = tid; t < QF * NP; t += blockDim.x) {
            const int q = t / NP, j = t % NP;
            if constexpr (FX)
                fps[q][j] = j < N ? fix_back(reinterpret_cast<const int2*>(pt)[FaceTab<D, P>::at(q, j)]) * s_psi : 0.0;
            else
                fps[q][j] = j < N ? pt[q * N + j] : (T)0;
        }
        for (int t = tid; t < QF * 25; t += blockDim.x) fjs[t / 25][t % 25] = (code & 1) ? fj[t] : -fj[t];
        __syncthreads();
        if (active) {
            for (int t = 0; t < QF; ++t) {
                const T s = fps[t][i] * fjs[t][ab];
                axpy_row<N, NP, T>(acc, s, fps[t]);
            }
        }
    }
    __syncthreads();
    if (active) {
        T* row = STAGE ? ob + (size_t)(a * N + i) * B + b * N : out + (size_t)e * B * B + (size_t)(a * N + i) * B + b * N;
        if (shifted) {
            const T idt = (T)(1.0 / s_dtau);
#pragma unroll
            for (int j = 0; j < N; ++j) row[j] = ((a == b && i == j) ? idt : (T)0) - acc[j];
        } else {
#pragma unroll
            for (int j = 0; j < N; ++j) row[j] = acc[j];
        }
    }
    if (STAGE) {
        __syncthreads();
        T* g = out + (size_t)e * B * B;
        for (int t = tid; t < B * B; t += blockDim.x) g[t] = ob[t];
    }
}

// Register-blocked SIMT form of the float32 assembly (3-D levels, and the 2-D elements that
// k_diag_blocks_pl leaves): thread (a, i, jg) accumulates row (a,i) of the block for all five b and the
// JW columns j of group jg, acc[b][j] += s_b psi_j with s_b = sum_k W d_k psi_i A_k[a][b] formed once
// per point and reused across the JW columns; every staged basis row is read 16 bytes at a time and
// broadcast.  Per entry the terms are summed in the order of k_diag_blocks (points in order,
// then the faces, each product as one FMA), so both forms give bitwise the same blocks.
//
// Bound by the issue of the multiply-adds (50 paired ones a point at N = 20) and, with the 100
// accumulators a thread that make them cheap, by what three blocks an SM can hide: the basis and the flux
// Jacobians of all points are in shared memory before the sums start, and the weighted gradients and the
// faces' data come by asynchronous copies one chunk or face ahead, so that the sums never wait for memory
// (one barrier a chunk in place of four).  A thread's Jacobian entries of a point are four (face: two)
// 16-byte reads.  13824 hexes, p = 3: 9.3 -> 5.6 ms of assembly per mixed V-cycle.
template <int D, int P>
struct DiagRb {
    using L = Lv<D, P>;
    static constexpr int N = L::N, Q = L::Q, QF = L::QF, B = L::B;
    static constexpr int JW = N <= 16 ? ((N + 3) / 4) * 4 : 20;    // columns j per thread
    static constexpr int JG = (N + JW - 1) / JW;                     // column groups
    static constexpr int NPAD = JG * JW;                             // padded basis row
    static constexpr int ROWS = 5 * N;                               // (a, i)
    static constexpr int THREADS = ((ROWS * JG + 31) / 32) * 32;
    static constexpr int QC = 16;                                    // volume points per chunk of gradients
    static constexpr int AK = D == 2 ? 12 : 16;                      // [k][b] entries of a Jacobian row, padded
    static constexpr int OLD = B | 1;                                // row stride of the finished block
    // shared memory (floats); the finished block lies over the tables
    static constexpr int O_PS = 0;                                   // [Q][NPAD]
    static constexpr int O_AS = O_PS + Q * NPAD;                     // [Q][5][AK]
    static constexpr int O_FP = O_AS + Q * 5 * AK;                   // 2 x [QF][NPAD]
    static constexpr int O_FJ = O_FP + 2 * QF * NPAD;                // 2 x [QF][5][8]
    static constexpr int O_GS = O_FJ + 2 * QF * 40;                  // 2 x [QC][D][N]
    static constexpr int O_US = O_GS + 2 * QC * D * N;               // [Q][5]
    static constexpr int PHASE = O_US + Q * 5;
    static constexpr int SM = PHASE > B * OLD ? PHASE : B * OLD;
    static_assert(O_AS % 4 == 0 && O_FP % 4 == 0 && O_FJ % 4 == 0 && O_GS % 4 == 0 && NPAD % 4 == 0, "16-byte reads");
    static constexpr int REGS = 5 * JW > 80 ? 168 : 128;             // register budget per thread
    static constexpr int MINB = (65536 / (THREADS * REGS)) < 1 ? 1 : 65536 / (THREADS * REGS);
    // bytes per asynchronous copy of a basis row: the rows start on its multiples in every table
    static constexpr int CP = N % 4 == 0 ? 16 : N % 2 == 0 ? 8 : 4;
};

template <int BYTES>
__device__ __forceinline__ void cp_async(float* dst, const float* src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    if constexpr (BYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(d), "l"(src), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int LEFT>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(LEFT) : "memory"); }

template <int D, int P>
__device__ __forceinline__ void diag_rb_element(
    int e, int nmax, const double* __restrict__ u, const float* __restrict__ vpsi, const float* __restrict__ vgw,
    const int* __restrict__ elem_face, const float* __restrict__ fpsiL, const float* __restrict__ fpsiR,
    const float* __restrict__ fjl, const float* __restrict__ fjr, const double* __restrict__ psic,
    const double* __restrict__ hlen, const double* __restrict__ cfl_dev, double g, int shifted,
    const double* __restrict__ vvr, float* __restrict__ out) {
    using L = Lv<D, P>;
    using R = DiagRb<D, P>;
    constexpr int N = L::N, Q = L::Q, QF = L::QF, B = L::B, NF = L::NF;
    constexpr int JW = R::JW, JG = R::JG, NPAD = R::NPAD, QC = R::QC, AK = R::AK, T = R::THREADS;
    extern __shared__ __align__(16) float smf[];
    __shared__ double ud[B], Uc[5];
    __shared__ float us[B], s_idt;
    float* ps = smf + R::O_PS;
    float* As = smf + R::O_AS;
    float* Us = smf + R::O_US;
    const int tid = threadIdx.x;
    constexpr int CF = R::CP / 4, NR = N / CF;   // floats per copy, copies per row
    // gradients of the points of chunk c, into buffer c & 1
    auto fetch_gradients = [&](int c) {
        const int q0 = c * QC, nq = Q - q0 < QC ? Q - q0 : QC;
        float* dst = smf + R::O_GS + (c & 1) * QC * D * N;
        for (int t = tid; t < D * nq * NR; t += T) {
            const int row = t / NR, x = t % NR * CF, k = row / nq, q = row % nq;
            cp_async<R::CP>(dst + (q * D + k) * N + x, vgw + (((size_t)e * D + k) * Q + q0 + q) * N + x);
        }
    };
    // basis traces and face Jacobians of face lf, into buffer lf & 1
    auto fetch_face = [&](int lf) {
        const int code = elem_face[(size_t)e * NF + lf];
        const float* pt = ((code & 1) ? fpsiR : fpsiL) + (size_t)(code >> 1) * QF * N;
        const float* fj = ((code & 1) ? fjr : fjl) + (size_t)(code >> 1) * QF * 25;
        float* dp = smf + R::O_FP + (lf & 1) * QF * NPAD;
        float* dj = smf + R::O_FJ + (lf & 1) * QF * 40;
        for (int t = tid; t < QF * NR; t += T) cp_async<R::CP>(dp + t / NR * NPAD + t % NR * CF, pt + t * CF);
        for (int t = tid; t < QF * 25; t += T) cp_async<4>(dj + t / 5 * 8 + t % 5, fj + t);
    };
    const float* pg = vpsi + (size_t)e * Q * N;
    for (int t = tid; t < Q * NR; t += T) cp_async<R::CP>(ps + t / NR * NPAD + t % NR * CF, pg + t * CF);
    cp_async_commit();
    fetch_gradients(0);
    cp_async_commit();
    // padding of the basis rows (the copies never touch it)
    if constexpr (NPAD > N) {
        for (int t = tid; t < Q * (NPAD - N); t += T) ps[t / (NPAD - N) * NPAD + N + t % (NPAD - N)] = 0.0f;
        for (int t = tid; t < 2 * QF * (NPAD - N); t += T)
            smf[R::O_FP + t / (NPAD - N) * NPAD + N + t % (NPAD - N)] = 0.0f;
    }
    for (int t = tid; t < B; t += T) {
        const double v = u[(size_t)e * B + t];
        ud[t] = v;
        us[t] = (float)v;
    }
    cp_async_wait<1>();
    __syncthreads();
    if (shifted && tid < 5) {   // the state at the cell centre
        double s = 0.0;
#pragma unroll 5
        for (int i = 0; i < N; ++i) s += ud[tid * N + i] * psic[(size_t)e * nmax + i];
        Uc[tid] = s;
    }
    for (int t = T - 1 - tid; t < Q * 5; t += T) {
        const int q = t / 5, c = t % 5;
        const float* pq = ps + q * NPAD;
        float s = 0.0f;
#pragma unroll 5
        for (int m = 0; m < N; ++m) s += us[c * N + m] * pq[m];
        Us[t] = s;
    }
    __syncthreads();
    if (tid == 0) {   // dtau of Eq. x3d
        float x = 0.0f;
        if (shifted) {
            const double ir = 1.0 / Uc[0];
            const double vx = Uc[1] * ir, vy = Uc[2] * ir, vz = Uc[3] * ir;
            const double q2 = vx * vx + vy * vy + vz * vz;
            const double pr = (g - 1.0) * (Uc[4] - 0.5 * Uc[0] * q2);
            const double cs = sqrt(g * pr * ir);
            x = (float)(1.0 / (cfl_dev[0] * hlen[e] / ((2 * P + 1) * (sqrt(q2) + cs))));
        }
        s_idt = x;
    }
    for (int t = T - 1 - tid; t < Q * D; t += T) {
        const int q = t / D, k = t % D;
        float A[25];
        flux_jac_k(Us + q * 5, (float)g, k, A);
        if (vvr) {   // rotating frame: A_k - (v_r)_k I
            const float vr = (float)vvr[((size_t)e * Q + q) * 3 + k];
#pragma unroll
            for (int a = 0; a < 5; ++a) A[a * 6] -= vr;
        }
#pragma unroll
        for (int a = 0; a < 5; ++a)
#pragma unroll
            for (int b = 0; b < 5; ++b) As[(q * 5 + a) * AK + k * 5 + b] = A[a * 5 + b];
    }
    // thread (a, i, jg): consecutive threads take consecutive i, so a warp shares a and jg
    const bool active = tid < R::ROWS * JG;
    const int a = active ? tid / (N * JG) : 0, rem = tid % (N * JG);
    const int jg = rem / N, i = rem % N;
    const int j0 = jg * JW;
    float acc[5][JW];
#pragma unroll
    for (int b = 0; b < 5; ++b)
#pragma unroll
        for (int j = 0; j < JW; ++j) acc[b][j] = 0.0f;
    auto add = [&](const float* prow, const float (&s)[5]) {
#pragma unroll
        for (int jj = 0; jj < JW; jj += 4) {
            const float4 v = *reinterpret_cast<const float4*>(prow + j0 + jj);
#pragma unroll
            for (int b = 0; b < 5; ++b) {
                fma2f(s[b], v.x, v.y, acc[b][jj], acc[b][jj + 1]);
                fma2f(s[b], v.z, v.w, acc[b][jj + 2], acc[b][jj + 3]);
            }
        }
    };
    constexpr int NCH = (Q + QC - 1) / QC;
#pragma unroll 1
    for (int c = 0; c < NCH; ++c) {
        cp_async_wait<0>();
        __syncthreads();   // chunk c is in; every thread has finished chunk c - 1, whose buffer is free
        if (c + 1 < NCH)
            fetch_gradients(c + 1);
        else
            fetch_face(0);
        cp_async_commit();
        if (active) {
            const int q0 = c * QC, nq = Q - q0 < QC ? Q - q0 : QC;
            const float* gq = smf + R::O_GS + (c & 1) * QC * D * N + i;
#pragma unroll 1
            for (int t = 0; t < nq; ++t) {
                const float4* Aq = reinterpret_cast<const float4*>(As + ((q0 + t) * 5 + a) * AK);
                float A[AK];
#pragma unroll
                for (int x = 0; x < AK; x += 4) {
                    const float4 v = Aq[x / 4];
                    A[x] = v.x, A[x + 1] = v.y, A[x + 2] = v.z, A[x + 3] = v.w;
                }
                float s[5];
#pragma unroll
                for (int b = 0; b < 5; ++b) s[b] = 0.0f;
#pragma unroll
                for (int k = 0; k < D; ++k) {
                    const float gk = gq[(t * D + k) * N];
#pragma unroll
                    for (int b = 0; b < 5; ++b) s[b] += gk * A[k * 5 + b];
                }
                add(ps + (q0 + t) * NPAD, s);
            }
        }
    }
#pragma unroll 1
    for (int lf = 0; lf < NF; ++lf) {
        cp_async_wait<0>();
        __syncthreads();
        if (lf + 1 < NF) fetch_face(lf + 1);
        cp_async_commit();
        if (active) {
            // the R side enters with the sign +, the L side with -
            const float sg = (elem_face[(size_t)e * NF + lf] & 1) ? 1.0f : -1.0f;
            const float* fp = smf + R::O_FP + (lf & 1) * QF * NPAD;
            const float* fj = smf + R::O_FJ + (lf & 1) * QF * 40 + a * 8;
#pragma unroll 1
            for (int t = 0; t < QF; ++t) {
                const float pi = sg * fp[t * NPAD + i];
                const float4 J = *reinterpret_cast<const float4*>(fj + t * 40);
                const float s[5] = {pi * J.x, pi * J.y, pi * J.z, pi * J.w, pi * fj[t * 40 + 4]};
                add(fp + t * NPAD, s);
            }
        }
    }
    __syncthreads();
    if (active) {
        const float idt = s_idt;
        float* o = smf + (a * N + i) * R::OLD + j0;
#pragma unroll
        for (int b = 0; b < 5; ++b)
#pragma unroll
            for (int j = 0; j < JW; ++j)
                if (j0 + j < N) {
                    const float v = acc[b][j];
                    o[b * N + j] = shifted ? ((a == b && i == j0 + j) ? idt : 0.0f) - v : v;
                }
    }
    __syncthreads();
    float* g_out = out + (size_t)e * B * B;
#pragma unroll 4
    for (int t = tid; t < B * B; t += T) g_out[t] = smf[t / B * R::OLD + t % B];
}

// Every element of the level (list = nullptr, one block each), or those that k_diag_blocks_pl left.
template <int D, int P>
__global__ void __launch_bounds__(DiagRb<D, P>::THREADS, DiagRb<D, P>::MINB) k_diag_blocks_rb(
    int E, int nmax, const double* __restrict__ u, const float* __restrict__ vpsi, const float* __restrict__ vgw,
    const int* __restrict__ elem_face, const float* __restrict__ fpsiL, const float* __restrict__ fpsiR,
    const float* __restrict__ fjl, const float* __restrict__ fjr, const double* __restrict__ psic,
    const double* __restrict__ hlen, const double* __restrict__ cfl_dev, double g, int shifted,
    const double* __restrict__ vvr, float* __restrict__ out, const int* __restrict__ list, int* __restrict__ head) {
    const int n = list ? take_list(head) : E;
#pragma unroll 1
    for (int it = blockIdx.x; it < n; it += gridDim.x) {
        __syncthreads();
        diag_rb_element<D, P>(list ? list[it] : it, nmax, u, vpsi, vgw, elem_face, fpsiL, fpsiR, fjl, fjr, psic, hlen,
                              cfl_dev, g, shifted, vvr, out);
    }
}

// Float copies of the level tables used by the FP32 block path.
__global__ void k_to_float(int64_t n, const double* __restrict__ x, float* __restrict__ y) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = (float)x[i];
}

// p = 0 block-sparse Jacobian: bsr[e][0] = diagonal block, bsr[e][1+lf] = dR_e/du_nb(lf).
__global__ void k_bsr0(int E, int NF, int QF, const int* __restrict__ elem_face, const double* __restrict__ fpsiL,
                       const double* __restrict__ fpsiR, const double* __restrict__ fjl,
                       const double* __restrict__ fjr, int F_int, double* __restrict__ bsr) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (int64_t)E * 25) return;
    const int e = (int)(idx / 25), ab = (int)(idx % 25);
    double diag = 0.0;
    double* row = bsr + (size_t)e * (1 + NF) * 25;
    for (int lf = 0; lf < NF; ++lf) {
        const int code = elem_face[(size_t)e * NF + lf];
        const int f = code >> 1;
        const bool rside = code & 1;
        double sd = 0.0, so = 0.0;
        for (int t = 0; t < QF; ++t) {
            const size_t pidx = (size_t)f * QF + t;
            if (!rside) {
                const double pl = fpsiL[pidx];
                sd -= pl * pl * fjl[pidx * 25 + ab];
                if (f < F_int) so -= pl * fpsiR[pidx] * fjr[pidx * 25 + ab];
            } else {
                const double pr = fpsiR[pidx];
                sd += pr * pr * fjr[pidx * 25 + ab];
                so += pr * fpsiL[pidx] * fjl[pidx * 25 + ab];
            }
        }
        diag += sd;
        row[(1 + lf) * 25 + ab] = so;
    }
    row[ab] = diag;
}

// Jacobian of the rotating frame's source (Eq. euler: S = (0, -omega x (rho v), 0), linear in U):
// dS_m/d(rho v)_n = -eps_{m k n} omega_k, so with the orthonormal basis every element's block
// gains dS/dU on the momentum rows and columns of each mode i (the same i).  The Appendix's
// printed dS/dU (Eq. dsdu) has the opposite sign; the sign here is that of S as written.
// Added to D = dR/du (shifted = 0) or subtracted from P = I/dtau - D (shifted = 1); block rows
// (a, i) of stride ld per element, element stride es.
template <class T>
__global__ void k_add_source(int64_t E, int N, int64_t es, int ld, int shifted, U5 om, T* __restrict__ out) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= E) return;
    const double dS[3][3] = {{0.0, om.v[2], -om.v[1]}, {-om.v[2], 0.0, om.v[0]}, {om.v[1], -om.v[0], 0.0}};
    const double sg = shifted ? -1.0 : 1.0;
    T* b = out + e * es;
    for (int i = 0; i < N; ++i)
        for (int m = 0; m < 3; ++m)
            for (int n = 0; n < 3; ++n)
                if (m != n) b[(size_t)((1 + m) * N + i) * ld + (1 + n) * N + i] += (T)(sg * dS[m][n]);
}

template <class T>
static emg_status add_source_jacobian(emg_ctx* c, int p, int shifted, T* out) {
    if (!c->rot) return EMG_OK;
    const LevelDev& L = c->lv[p];
    U5 om{};
    for (int k = 0; k < 3; ++k) om.v[k] = c->prm.omega[k];
    { ProfScope _ps(c, PC_DIAG); k_add_source<T><<<(unsigned)((c->E + 127) / 128), 128, 0, c->stream>>>(
        c->E, L.N, (int64_t)L.B * L.B, L.B, shifted, om, out); }
    EMG_CHECK_LAUNCH(c);
    return EMG_OK;
}

emg_status launch_diag_blocks(emg_ctx* c, int p, const double* u, const double* cfl_dev, int shifted, double* out) {
    emg_status st = launch_face_jacobian(c, p, u);
    if (st != EMG_OK) return st;
    if (diag_blocks_fx_serves(c->dim, p)) {
        st = launch_diag_blocks_fx(c, p, u, cfl_dev, shifted, out);
        if (st != EMG_OK) return st;
        return add_source_jacobian(c, p, shifted, out);
    }
    LevelDev& L = c->lv[p];
    const int nmax = n_modes(c->dim, c->p_max);
#define EMG_DB(DD, PP)                                                                                      \
    if constexpr (PP == 0 || (DD == 3 && PP == 4)) {                                                        \
        ProfScope _ps(c, PC_DIAG);                                                                          \
        k_diag_blocks<DD, PP, double><<<(unsigned)c->E, DiagCfg<DD, PP>::THREADS, 0, c->stream>>>(          \
            (int)c->E, nmax, u, L.vpsi, L.vgw, c->elem_face, L.fpsiL, L.fpsiR, L.fjl, L.fjr, c->psic, c->h, \
            cfl_dev, c->prm.gamma, shifted, L.vvr, L.texp, L.gexp, out);                                    \
    }
    EMG_DISPATCH_DP(c->dim, p, EMG_DB)
#undef EMG_DB
    EMG_CHECK_LAUNCH(c);
    return add_source_jacobian(c, p, shifted, out);
}

// Block assembly of the float32 block forms (levels p >= 1): on the tensor cores or, where the
// level's choice says so, the SIMT form.
emg_status launch_diag_blocks32(emg_ctx* c, int p, const double* u, const double* cfl_dev, int shifted,
                                float* out) {
    emg_status st = launch_face_jacobian32(c, p, u);
    if (st != EMG_OK) return st;
    LevelDev& L = c->lv[p];
    if (!L.vpsi32) {
        c->err = "FP32 tables not built";
        return EMG_ERR_ARG;
    }
    if (!L.tc_asm) {
        // the SIMT (FMA) form of the same contraction
        const int nmax = n_modes(c->dim, c->p_max);
        const GjWork w = gj_work(L.piv, c->E);
        if (L.asm_plane) {   // then, below, the elements it left (none in plane flow)
            st = launch_diag_blocks_plane(c, p, u, cfl_dev, shifted, out);
            if (st != EMG_OK) return st;
        }
#define EMG_DB32(DD, PP)                                                                                    \
    if constexpr (PP > 0) {                                                                                 \
        EMG_CUDA_TRY(c, cudaFuncSetAttribute(k_diag_blocks_rb<DD, PP>, cudaFuncAttributeMaxDynamicSharedMemorySize, \
                                             DiagRb<DD, PP>::SM * 4));                                      \
        ProfScope _ps(c, PC_DIAG);                                                                          \
        if (c->prm.block_kernels == 3)                                                                      \
            k_diag_blocks<DD, PP, float><<<(unsigned)c->E, DiagCfg<DD, PP>::THREADS, 0, c->stream>>>(       \
                (int)c->E, nmax, u, L.vpsi32, L.vgw32, c->elem_face, L.fpsiL32, L.fpsiR32, L.fjl32, L.fjr32,  \
                c->psic, c->h, cfl_dev, c->prm.gamma, shifted, L.vvr, nullptr, nullptr, out);               \
        else                                                                                                \
            k_diag_blocks_rb<DD, PP><<<L.asm_plane ? list_grid(c->E, DiagRb<DD, PP>::THREADS) : (unsigned)c->E, \
                                       DiagRb<DD, PP>::THREADS, DiagRb<DD, PP>::SM * 4, c->stream>>>(       \
                (int)c->E, nmax, u, L.vpsi32, L.vgw32, c->elem_face, L.fpsiL32, L.fpsiR32, L.fjl32, L.fjr32,  \
                c->psic, c->h, cfl_dev, c->prm.gamma, shifted, L.vvr, out,                                  \
                L.asm_plane ? w.asm_list : nullptr, w.asm_head);                                            \
    }
        EMG_DISPATCH_DP(c->dim, p, EMG_DB32)
#undef EMG_DB32
        EMG_CHECK_LAUNCH(c);
        return add_source_jacobian(c, p, shifted, out);
    }
    st = launch_diag_blocks_tc(c, p, u, cfl_dev, shifted, out);
    if (st != EMG_OK) return st;
    return add_source_jacobian(c, p, shifted, out);
}

emg_status build_float_tables(emg_ctx* c) {
    for (int p = 1; p <= c->p_max; ++p) {
        LevelDev& L = c->lv[p];
        const int64_t n1 = c->E * L.Q * L.N, n2 = c->E * c->dim * L.Q * L.N;
        const int64_t n3 = c->F * L.QF * L.N, n4 = std::max<int64_t>(c->F_int, 1) * L.QF * L.N;
        const double* src[4] = {L.vpsi, L.vgw, L.fpsiL, L.fpsiR};
        float* dst[4] = {L.vpsi32, L.vgw32, L.fpsiL32, L.fpsiR32};
        const int64_t cnt[4] = {n1, n2, n3, n4};
        for (int k = 0; k < 4; ++k) {
            ProfScope _ps(c, PC_SETUP);
            k_to_float<<<(unsigned)((cnt[k] + 255) / 256), 256, 0, c->stream>>>(cnt[k], src[k], dst[k]);
        }
        EMG_CHECK_LAUNCH(c);
    }
    return EMG_OK;
}

emg_status launch_bsr0(emg_ctx* c) {
    LevelDev& L = c->lv[0];
    const int64_t n = c->E * 25;
    { ProfScope _ps(c, PC_BSR0); k_bsr0<<<(unsigned)((n + 127) / 128), 128, 0, c->stream>>>((int)c->E, 2 * c->dim, L.QF, c->elem_face, L.fpsiL,
                                                               L.fpsiR, L.fjl, L.fjr, (int)c->F_int, c->bsr); }
    EMG_CHECK_LAUNCH(c);
    if (c->rot) {   // p = 0: the diagonal 5x5 block (first of each element's row) gains dS/dU
        U5 om{};
        for (int k = 0; k < 3; ++k) om.v[k] = c->prm.omega[k];
        { ProfScope _ps(c, PC_BSR0); k_add_source<double><<<(unsigned)((c->E + 127) / 128), 128, 0, c->stream>>>(
            c->E, 1, (1 + 2 * c->dim) * 25, 5, 0, om, c->bsr); }
        EMG_CHECK_LAUNCH(c);
    }
    return EMG_OK;
}

}  // namespace emg
