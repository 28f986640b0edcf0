// Float32 block assembly (Eq. jac1) of 2-D flow in the plane: a block whose spanwise momentum (variable
// 3) is coupled to nothing has 17 of its 25 variable pairs, a 4 N x 4 N and an N x N system, and leaves
// packed (blocks.cuh, here row-major) for k_gj_split.  The sums are those of k_diag_blocks_rb
// (jacobian.cu), term by term; an element with an entry other than zero at a coupled place goes on a
// list for that kernel, which leaves the whole block.
//
// Bound by the issue of the multiply-adds and their shared-memory reads.  30 / N elements share a
// block of five warps: four of rows of the 4 N system (thread (a, i): four b by all N columns), one of
// spanwise rows, so that no warp mixes the two and 94 % of the lanes have a row at every order.  All
// points' tables are staged at once (one barrier before the sums, none between volume and faces); a
// point's Jacobian row is one 16-byte read.  128 x 64, p = 4: 0.34 -> 0.265 ms a launch, and the packed
// blocks spare the inverse a third of its reads.
#include "blocks.cuh"
#include "common.cuh"
#include "jacobian.cuh"

namespace emg {

template <int P>
struct DiagPl {
    using L = Lv<2, P>;
    static constexpr int N = L::N, Q = L::Q, QF = L::QF, FP = 4 * QF, B4 = 4 * N;
    static constexpr int EC = 30 / N;                     // elements per block
    static constexpr int THREADS = 160;
    // resident blocks: four would leave N = 15 96 registers a thread, 40 too few (340 bytes spilled; the
    // smoothing step of 8192 elements at p = 4 1237 -> 1200 us with three, 18432 elements 2448 -> 2397)
    static constexpr int MINB = N == 15 ? 3 : 4;
    static constexpr int NPAD = (N + 3) / 4 * 4;
    // shared memory (floats), per kind [EC][...]
    static constexpr int O_PS = 0;                        // [Q + FP][NPAD]   basis at the points
    static constexpr int O_A4 = O_PS + EC * (Q + FP) * NPAD;   // [2 Q + FP][4] float4: Jacobian rows
    static constexpr int O_GS = O_A4 + EC * (2 * Q + FP) * 16; // [Q][N] float2: weighted gradients
    static constexpr int O_A3 = O_GS + EC * Q * N * 2;    // [2 Q + FP]       spanwise Jacobian entry
    static constexpr int O_US = O_A3 + EC * (2 * Q + FP); // [Q][5]
    static constexpr int PHASE = O_US + EC * Q * 5;
    static constexpr int PACK = (17 * N * N + 3) / 4 * 4;  // one packed block (over the tables, at the end)
    static constexpr int SM = PHASE > EC * PACK ? PHASE : EC * PACK;
    static_assert(O_A4 % 4 == 0 && O_GS % 2 == 0, "16- and 8-byte reads");
};

template <int P>
__global__ void __launch_bounds__(160, DiagPl<P>::MINB) k_diag_blocks_pl(
    int E, int nmax, const double* __restrict__ u, const float* __restrict__ vpsi, const float* __restrict__ vgw,
    const int* __restrict__ elem_face, const float* __restrict__ fpsiL, const float* __restrict__ fpsiR,
    const float* __restrict__ fjl, const float* __restrict__ fjr, const double* __restrict__ psic,
    const double* __restrict__ hlen, const double* __restrict__ cfl_dev, double g, int shifted,
    float* __restrict__ out, int* __restrict__ flag, int* __restrict__ list, int* __restrict__ head) {
    using C = DiagPl<P>;
    constexpr int N = C::N, Q = C::Q, QF = C::QF, FP = C::FP, EC = C::EC, NPAD = C::NPAD, B = 5 * N, B4 = C::B4;
    constexpr int T = C::THREADS;
    extern __shared__ __align__(16) float smf[];
    float* ps = smf + C::O_PS;                                 // volume points, then face points
    float4* A4 = reinterpret_cast<float4*>(smf + C::O_A4);     // [2 q + k], then face points
    float2* gs = reinterpret_cast<float2*>(smf + C::O_GS);
    float* A3 = smf + C::O_A3;
    float* Us = smf + C::O_US;
    __shared__ double ud[EC * B], Uc[EC][5];
    __shared__ float us[EC * B], idt[EC];
    __shared__ int codes[EC * 4], bad[EC];
    const int tid = threadIdx.x, e0 = blockIdx.x * EC;
    const int ne = E - e0 < EC ? E - e0 : EC;
    for (int t = tid; t < EC * B; t += T) {
        const double v = t < ne * B ? u[(size_t)e0 * B + t] : 1.0;
        ud[t] = v;
        us[t] = (float)v;
    }
    if (tid < EC) bad[tid] = 0;
    if (tid < EC * 4) codes[tid] = tid < ne * 4 ? elem_face[(size_t)e0 * 4 + tid] : 0;
    __syncthreads();
    // tables
    for (int t = tid; t < ne * Q * N; t += T) {
        const int el = t / (Q * N), r = t % (Q * N);
        ps[(el * (Q + FP) + r / N) * NPAD + r % N] = vpsi[(size_t)e0 * Q * N + t];
        gs[t] = make_float2(vgw[((size_t)(e0 + el) * 2) * Q * N + r], vgw[((size_t)(e0 + el) * 2 + 1) * Q * N + r]);
    }
    for (int t = tid; t < ne * FP * N; t += T) {
        const int s = t / (QF * N), r = t % (QF * N), code = codes[s];
        const float* pt = ((code & 1) ? fpsiR : fpsiL) + (size_t)(code >> 1) * QF * N;
        ps[((s >> 2) * (Q + FP) + Q + (s & 3) * QF + r / N) * NPAD + r % N] = pt[r];
    }
    if (NPAD > N)
        for (int t = tid; t < EC * (Q + FP) * (NPAD - N); t += T)
            ps[t / (NPAD - N) * NPAD + N + t % (NPAD - N)] = 0.0f;
    for (int t = tid; t < ne * FP * 25; t += T) {
        const int s = t / (QF * 25), r = t % (QF * 25), code = codes[s], el = s >> 2;
        const float x = (((code & 1) ? fjr : fjl) + (size_t)(code >> 1) * QF * 25)[r];
        const float v = (code & 1) ? x : -x;
        const int a = r % 25 / 5, b = r % 5, pt = el * (2 * Q + FP) + 2 * Q + (s & 3) * QF + r / 25;
        if (a != 3 && b != 3)
            reinterpret_cast<float*>(A4 + pt * 4 + (a == 4 ? 3 : a))[b == 4 ? 3 : b] = v;
        else if (a == b)
            A3[pt] = v;
        else if (!(v == 0.0f))
            bad[el] = 1;
    }
    __syncthreads();
    for (int t = tid; t < EC * Q * 5; t += T) {
        const int el = t / (Q * 5), q = t % (Q * 5) / 5, c = t % 5;
        const float* pq = ps + (el * (Q + FP) + q) * NPAD;
        float s = 0.0f;
        if (el < ne)
            for (int m = 0; m < N; ++m) s += us[el * B + c * N + m] * pq[m];
        Us[t] = s;
    }
    if (shifted && tid >= T - 5 * EC) {   // the state at the cell centres
        const int k = tid - (T - 5 * EC), el = k / 5, a = k % 5;
        double s = 0.0;
        if (el < ne)
            for (int i = 0; i < N; ++i) s += ud[el * B + a * N + i] * psic[(size_t)(e0 + el) * nmax + i];
        Uc[el][a] = s;
    }
    __syncthreads();
    if (tid < ne) {
        float x = 0.0f;
        if (shifted) {   // dtau of Eq. x3d
            const double* U = Uc[tid];
            const double ir = 1.0 / U[0];
            const double vx = U[1] * ir, vy = U[2] * ir, vz = U[3] * ir;
            const double q2 = vx * vx + vy * vy + vz * vz;
            const double pr = (g - 1.0) * (U[4] - 0.5 * U[0] * q2);
            const double cs = sqrt(g * pr * ir);
            x = (float)(1.0 / (cfl_dev[0] * hlen[e0 + tid] / ((2 * P + 1) * (sqrt(q2) + cs))));
        }
        idt[tid] = x;
    }
    for (int t = T - 1 - tid; t < ne * Q * 2; t += T) {
        const int el = t / (Q * 2), qk = t % (Q * 2), pt = el * (2 * Q + FP) + qk;
        float A[25];
        flux_jac_k(Us + (el * Q + qk / 2) * 5, (float)g, qk % 2, A);
        A4[pt * 4 + 0] = make_float4(A[0], A[1], A[2], A[4]);
        A4[pt * 4 + 1] = make_float4(A[5], A[6], A[7], A[9]);
        A4[pt * 4 + 2] = make_float4(A[10], A[11], A[12], A[14]);
        A4[pt * 4 + 3] = make_float4(A[20], A[21], A[22], A[24]);
        A3[pt] = A[18];
        if (!(A[3] == 0.0f && A[8] == 0.0f && A[13] == 0.0f && A[23] == 0.0f && A[15] == 0.0f && A[16] == 0.0f &&
              A[17] == 0.0f && A[19] == 0.0f))
            bad[el] = 1;
    }
    __syncthreads();
    if (__all_sync(0xffffffffu, (tid & 31) >= ne || bad[tid & 31])) {   // nothing to sum: all on the list
        if (tid < ne) {
            flag[e0 + tid] = 0;
            list[atomicAdd(head, 1)] = e0 + tid;
        }
        return;
    }
    const int sw = tid - 128;   // >= 0: spanwise row
    const int el = sw < 0 ? tid / B4 : sw / N;
    const int a4 = sw < 0 ? tid % B4 / N : 0, i = sw < 0 ? tid % N : sw % N;
    const bool act = el < ne;   // thread 120 .. 127, 158, 159: el >= EC
    float acc[4][NPAD];
#pragma unroll
    for (int b = 0; b < 4; ++b)
#pragma unroll
        for (int j = 0; j < NPAD; ++j) acc[b][j] = 0.0f;
    if (act) {
        const float* p = ps + el * (Q + FP) * NPAD;
        if (sw < 0) {
            auto add = [&](const float* prow, const float (&s)[4]) {
#pragma unroll
                for (int j = 0; j < NPAD; j += 4) {
                    const float4 v = *reinterpret_cast<const float4*>(prow + j);
#pragma unroll
                    for (int b = 0; b < 4; ++b) {
                        fma2f(s[b], v.x, v.y, acc[b][j], acc[b][j + 1]);
                        fma2f(s[b], v.z, v.w, acc[b][j + 2], acc[b][j + 3]);
                    }
                }
            };
            const float2* gq = gs + el * Q * N + i;
            const float4* Aq = A4 + el * (2 * Q + FP) * 4 + a4;
#pragma unroll 1
            for (int q = 0; q < Q; ++q) {
                const float2 gk = gq[q * N];
                const float4 A0 = Aq[q * 8], A1 = Aq[q * 8 + 4];
                const float s[4] = {fmaf(gk.y, A1.x, gk.x * A0.x), fmaf(gk.y, A1.y, gk.x * A0.y),
                                    fmaf(gk.y, A1.z, gk.x * A0.z), fmaf(gk.y, A1.w, gk.x * A0.w)};
                add(p + q * NPAD, s);
            }
#pragma unroll 1
            for (int t = 0; t < FP; ++t) {
                const float pi = p[(Q + t) * NPAD + i];
                const float4 J = Aq[(2 * Q + t) * 4];
                const float s[4] = {pi * J.x, pi * J.y, pi * J.z, pi * J.w};
                add(p + (Q + t) * NPAD, s);
            }
        } else {
            auto add = [&](const float* prow, float s) {
#pragma unroll
                for (int j = 0; j < NPAD; j += 4) {
                    const float4 v = *reinterpret_cast<const float4*>(prow + j);
                    fma2f(s, v.x, v.y, acc[0][j], acc[0][j + 1]);
                    fma2f(s, v.z, v.w, acc[0][j + 2], acc[0][j + 3]);
                }
            };
            const float2* gq = gs + el * Q * N + i;
            const float* Aq = A3 + el * (2 * Q + FP);
#pragma unroll 1
            for (int q = 0; q < Q; ++q) {
                const float2 gk = gq[q * N];
                add(p + q * NPAD, fmaf(gk.y, Aq[2 * q + 1], gk.x * Aq[2 * q]));
            }
#pragma unroll 1
            for (int t = 0; t < FP; ++t) add(p + (Q + t) * NPAD, p[(Q + t) * NPAD + i] * Aq[2 * Q + t]);
        }
    }
    __syncthreads();
    // the packed blocks over the tables, then out
    if (act) {
        const float id = idt[el];
        float* o = smf + el * C::PACK + (sw < 0 ? (a4 * N + i) * B4 : B4 * B4 + i * N);
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            if (sw >= 0 && b > 0) break;
            const bool dg = sw >= 0 || b == a4;
#pragma unroll
            for (int j = 0; j < N; ++j) {
                const float v = acc[b][j];
                o[b * N + j] = shifted ? (dg && i == j ? id : 0.0f) - v : v;
            }
        }
    }
    if (tid < ne) {
        flag[e0 + tid] = !bad[tid];
        if (bad[tid]) list[atomicAdd(head, 1)] = e0 + tid;
    }
    __syncthreads();
#pragma unroll 1
    for (int k = 0; k < ne; ++k) {
        if (bad[k]) continue;
        float* o = out + gj_packed_at(e0 + k, B);
        const float* s = smf + k * C::PACK;
        for (int t = tid; t < 17 * N * N / 4; t += T)
            reinterpret_cast<float4*>(o)[t] = reinterpret_cast<const float4*>(s)[t];
        for (int t = 17 * N * N / 4 * 4 + tid; t < 17 * N * N; t += T) o[t] = s[t];
    }
}

template <int P>
static emg_status go(emg_ctx* c, const double* u, const double* cfl_dev, int shifted, float* out) {
    using C = DiagPl<P>;
    LevelDev& L = c->lv[P];
    constexpr int smem = C::SM * (int)sizeof(float);
    EMG_CUDA_TRY(c, cudaFuncSetAttribute(k_diag_blocks_pl<P>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    ProfScope _ps(c, PC_DIAG);
    const GjWork w = gj_work(L.piv, c->E);
    k_diag_blocks_pl<P><<<(unsigned)((c->E + C::EC - 1) / C::EC), C::THREADS, smem, c->stream>>>(
        (int)c->E, n_modes(2, c->p_max), u, L.vpsi32, L.vgw32, c->elem_face, L.fpsiL32, L.fpsiR32, L.fjl32, L.fjr32,
        c->psic, c->h, cfl_dev, c->prm.gamma, shifted, out, w.asm_flag, w.asm_list, w.asm_head);
    EMG_CHECK_LAUNCH(c);
    return EMG_OK;
}

emg_status launch_diag_blocks_plane(emg_ctx* c, int p, const double* u, const double* cfl_dev, int shifted, float* out) {
    switch (p) {
        case 1: return go<1>(c, u, cfl_dev, shifted, out);
        case 2: return go<2>(c, u, cfl_dev, shifted, out);
        case 3: return go<3>(c, u, cfl_dev, shifted, out);
        default: return go<4>(c, u, cfl_dev, shifted, out);
    }
}

}  // namespace emg
