// FP64 block assembly (Eq. jac1) on the integer pipe: the element-diagonal blocks of the FP64 form,
//   D[(a,i),(b,j)] = sum_q psi_j(x_q) s_{ab,i}(q),   s = sum_k W_q d_k psi_i A_k[a][b]  (volume points)
//                                                    s = -/+ psi_i w|n dS| dF~/dU[a][b]  (face points)
// as fixed-point sums (fix.cuh).  Thread (ab, i) of an element's block forms its s of a point from the
// staged tables and adds s psi_j to the N columns of its row.  s has 58 bits and an exponent of its
// own for each (ab, i), from the largest gradients of mode i and Jacobian entries ab; the directions
// are scaled against each other first (A_k by the power of two of the gradients' size along k), so that
// the long side of a stretched cell keeps its bits.  psi_j has the bits that the sums leave room for: 2-D
// 55 (p = 1: 56); 3-D 56, the sums of at most 31 rows going to 96-bit numbers in shared memory.  Error of
// an entry over its own sum of |terms|, worst and rms in units of 2^-53, CPU emulation (float64 / one
// exponent a pair (a, b), s cut to 54 bits / this form): 24 x 12 O-grid, p = 4: 5.7, 0.55 / 44, 2.6 / 5.7,
// 0.39; 128 x 8, p = 3: 4.2, 0.53 / 113, 7.2 / 3.4, 0.30; rectangles of aspect 10^4, p = 4: 5.8, 0.50 /
// 4400, 136 / 7.3, 0.41; sphere shells, p = 2: 16, 0.84 / 1240, 86 / 11, 0.42, p = 3: 12, 0.90 / 304, 30 /
// 6.6, 0.56.  Only the pairs (a, b) with an entry other than zero at
// some point are visited: 17 of 25 in a 2-D flow without a spanwise momentum.  Bound by the integer
// multiply-adds (3 per term): on the float64 pipe the same sums took 16.7 ms of the FP64 V-cycle of
// the 128 x 64 O-grid at p = 4.
#include "dispatch.cuh"
#include "fix.cuh"
#include "jacobian.cuh"

namespace emg {

template <int D, int P>
struct DiagFx {
    using L = Lv<D, P>;
    static constexpr int N = L::N, Q = L::Q, QF = L::QF, NF = L::NF, B = L::B;
    static constexpr int LIVE = D == 2 ? 17 : 25;                      // pairs (a, b) of one pass
    static constexpr int THREADS = (LIVE * N + 31) / 32 * 32;
    static constexpr int NP = (N + 1) & ~1;                            // columns, padded to 16 bytes
    static constexpr int QC = D == 2 || P == 1 ? Q : 24;               // volume points per chunk
    static constexpr int FP = D == 2 ? NF * QF : QF;                   // face points per chunk
    static constexpr int RC = QC > FP ? QC : FP;
    // bits of s and of the staged psi; over the rows of one sum (3-D: RMAX, then to the 96-bit ones)
    //   |h| <= rows 2^(SB - 28) 2^(PB - 28) < 2^63,  |x| <= rows (2^(SB - 28) 2^27 + 2^27 2^(PB - 28)) < 2^63
    static constexpr int SB = 58, PB = D == 2 && P > 1 ? 55 : 56, RMAX = 31;
    static constexpr int SV = D == 2 ? 1 : 2;                          // bits of a sum of D products
    static constexpr bool FOLD = D == 2 && N == 15;                    // x into h after the volume points
    static constexpr int FG = RMAX / QF;                               // 3-D: faces of one sum
    static_assert((D == 3 && P == 4) || (D == 2 ? Q + FP <= (PB == 56 ? 31 : 62) && (FOLD ? QC : Q + FP) <= 56 : QC <= RMAX && FG >= 1), "exact sums");
    // shared memory (8-byte words); the slab that the rows leave through lies over the tables
    static constexpr int O_PS = 0, O_GS = O_PS + RC * NP, O_AS = O_GS + QC * D * N;
    static constexpr int AW = QC * D > FP ? QC * D : FP;               // rows of 25 entries
    static constexpr int TAB = O_AS + AW * 25;
    // 2-D: the face points have places of their own, so that both parts run without a barrier between
    static constexpr int O_FS = TAB, O_FJ = O_FS + FP * NP;
    static constexpr int ALL = D == 2 ? O_FJ + FP * 25 : TAB;
    // resident blocks asked of the register allocator (80 registers a thread for N = 10 and 15 in 2-D, 60 and 67
    // below; 3-D p = 1, 2, 3: 96, 103, 128)
    static constexpr int MINB = D == 2 ? (N == 15 ? 3 : N == 10 ? 4 : 5) : N == 20 ? 1 : N == 10 ? 2 : 4;
    static constexpr int SLAB = N * B;
    static constexpr int O_ACC = ALL > SLAB ? ALL : SLAB;              // 3-D: [3][N][LIVE N] words of the 96-bit sums
    static constexpr size_t SMEM = (size_t)O_ACC * 8 + (D == 3 ? (size_t)3 * N * LIVE * N * 4 : 0);
};

// dF_k/dU (Appendix Eq. dfdu with grad psi -> e_k, omega = 0) less vrk on the diagonal.
__device__ __forceinline__ void flux_jac_fast(const double* U, double g, int k, double vrk, double* A) {
    const double ir = rcp_h3(U[0]), g1 = g - 1.0;
    const double v[3] = {U[1] * ir, U[2] * ir, U[3] * ir};
    const double q2 = fma(v[0], v[0], fma(v[1], v[1], v[2] * v[2]));
    const double a0 = 0.5 * g1 * q2;
    const double p = g1 * fma(-0.5 * U[0], q2, U[4]);
    const double H = (U[4] + p) * ir, vk = k == 0 ? v[0] : k == 1 ? v[1] : v[2];
#pragma unroll
    for (int t = 0; t < 5; ++t) A[t] = t == 1 + k ? 1.0 : 0.0;
    A[0] -= vrk;
#pragma unroll
    for (int m = 0; m < 3; ++m) {
        double* row = A + 5 * (1 + m);
        row[0] = fma(-v[m], vk, m == k ? a0 : 0.0);
#pragma unroll
        for (int l = 0; l < 3; ++l) {
            double x = l == k ? v[m] : 0.0;
            if (m == k) x = fma(-g1, v[l], x);
            if (m == l) x += vk - vrk;
            row[1 + l] = x;
        }
        row[4] = m == k ? g1 : 0.0;
    }
    A[20] = (a0 - H) * vk;
#pragma unroll
    for (int l = 0; l < 3; ++l) A[21 + l] = fma(-g1 * v[l], vk, l == k ? H : 0.0);
    A[24] = fma(g, vk, -vrk);
}

template <int D, int P>
__global__ void __launch_bounds__(DiagFx<D, P>::THREADS, DiagFx<D, P>::MINB) k_diag_blocks_fx(
    int E, int nmax, const double* __restrict__ u, const int2* __restrict__ vpsi, const int2* __restrict__ vgw,
    const int* __restrict__ elem_face, const int2* __restrict__ fpsiL, const int2* __restrict__ fpsiR,
    const int* __restrict__ texp, const int* __restrict__ gexp, const double* __restrict__ fjl, const double* __restrict__ fjr,
    const double* __restrict__ psic, const double* __restrict__ hlen, const double* __restrict__ cfl_dev, double g,
    int shifted, const double* __restrict__ vvr, double* __restrict__ out) {
    using C = DiagFx<D, P>;
    constexpr int N = C::N, Q = C::Q, QF = C::QF, NF = C::NF, B = C::B, NP = C::NP, QC = C::QC, FP = C::FP;
    constexpr int T = C::THREADS;
    extern __shared__ __align__(16) unsigned char smraw[];
    int2* sm = reinterpret_cast<int2*>(smraw);
    int2* ps = sm + C::O_PS;                                    // [points][NP]
    int2* gs = sm + C::O_GS;                                    // [QC][D][N]
    int2* As = sm + C::O_AS;                                    // [QC][D][25], or the face Jacobians [FP][25]
    int2* fs = D == 2 ? sm + C::O_FS : ps;                      // [FP][NP]
    int2* fj = D == 2 ? sm + C::O_FJ : As;                      // [FP][25]
    __shared__ double ud[B], Us[Q][5], s_dtau;
    __shared__ int mxa[25], mxj[25], sa[25], sj[25], live[25], nlive;
    const int e = blockIdx.x, tid = threadIdx.x;
    // the gradients' exponents; dk: along k less the least direction's, ty: of mode i after that scaling
    __shared__ int ge[D * N], dk[D], ty[N], m0;
    for (int t = tid; t < D * N; t += T) ge[t] = gexp[(size_t)e * D * N + t];
    for (int t = tid; t < B; t += T) ud[t] = u[(size_t)e * B + t];
    if (tid < 25) mxa[tid] = mxj[tid] = 0;
    const int tx = texp[e], tp = tx - (FIX_BITS - C::PB);   // exponents of psi, of the staged psi
    __syncthreads();
    if (tid < 32) {
        int mk[D], least = 0x7fffffff;
#pragma unroll
        for (int k = 0; k < D; ++k) {
            mk[k] = 0x7fffffff;
            for (int i = tid; i < N; i += 32) mk[k] = min(mk[k], ge[k * N + i]);
            mk[k] = __reduce_min_sync(0xffffffffu, mk[k]);
            least = min(least, mk[k]);
        }
        for (int i = tid; i < N; i += 32) {
            int m = 0x7fffffff;
#pragma unroll
            for (int k = 0; k < D; ++k) m = min(m, ge[k * N + i] - mk[k]);
            ty[i] = m;
#pragma unroll
            for (int k = 0; k < D; ++k) ge[k * N + i] -= mk[k] + m;   // what is left to shift a staged gradient by
        }
        if (tid == 0) {
            m0 = least;
#pragma unroll
            for (int k = 0; k < D; ++k) dk[k] = mk[k] - least;
        }
    }
    // U at the volume points (float64: 5 N multiply-adds a point), dtau of Eq. x3d
    {
        const double sp = fix_scale(-tx, 0);
        const int2* pv = vpsi + (size_t)e * Q * N;
        for (int t = tid; t < Q * 5; t += T) {
            const int c = t / Q, q = t % Q;
            double s = 0.0;
#pragma unroll 5
            for (int m = 0; m < N; ++m) s = fma(ud[c * N + m], fix_back(pv[m * Q + q]), s);
            Us[q][c] = s * sp;
        }
    }
    if (shifted && tid >= T - 32) {   // the last warp: the state at the cell centre
        const int lane = tid & 31;
        double s = 0.0;
        if (lane < 5)
            for (int i = 0; i < N; ++i) s = fma(ud[lane * N + i], psic[(size_t)e * nmax + i], s);
        double Uc[5];
#pragma unroll
        for (int a = 0; a < 5; ++a) Uc[a] = __shfl_sync(0xffffffffu, s, a);
        if (lane == 0) {
            const double ir = 1.0 / Uc[0];
            const double vx = Uc[1] * ir, vy = Uc[2] * ir, vz = Uc[3] * ir;
            const double q2 = vx * vx + vy * vy + vz * vz;
            const double pr = (g - 1.0) * (Uc[4] - 0.5 * Uc[0] * q2);
            const double cs = sqrt(g * pr * ir);
            s_dtau = cfl_dev[0] * hlen[e] / ((2 * P + 1) * (sqrt(q2) + cs));
        }
    }
    // the face Jacobians' keys: each pair's largest over the element's face points
    for (int t = tid; t < NF * QF * 25; t += T) {
        const int lf = t / (QF * 25), code = elem_face[(size_t)e * NF + lf];
        const int k = fix_key((((code & 1) ? fjr : fjl) + (size_t)(code >> 1) * QF * 25)[t - lf * QF * 25]);
        if (k > 0) atomicMax(&mxj[t % 25], k);
    }
    __syncthreads();
    // the flux Jacobians' keys; where all points fit, the Jacobians stay in shared memory
    double* Ad = reinterpret_cast<double*>(As);
    auto flux_jac_at = [&](int q, int k, double* A) {
        flux_jac_fast(Us[q], g, k, vvr ? vvr[((size_t)e * Q + q) * 3 + k] : 0.0, A);
    };
    for (int t = tid; t < Q * D; t += T) {
        double A[25];
        flux_jac_at(t / D, t % D, A);
#pragma unroll
        for (int x = 0; x < 25; ++x) {
            int k = fix_key(A[x]);
            if (k > 0 && k < 0x7ff00000) k = max(k - (dk[t % D] << 20), 1);
            if (k > mxa[x]) atomicMax(&mxa[x], k);
            if (Q == QC) Ad[t * 25 + x] = A[x];
        }
    }
    __syncthreads();
    if (tid < 32) {   // the live pairs, in order
        const bool on = tid < 25 && (mxa[tid] > 0 || mxj[tid] > 0);
        const unsigned m = __ballot_sync(0xffffffffu, on);
        if (on) live[__popc(m & ((1u << tid) - 1u))] = tid;
        if (tid == 0) nlive = __popc(m);
        if (on) {
            sa[tid] = fix_exp(mxa[tid]);
            sj[tid] = fix_exp(mxj[tid]);
        }
    }
    __syncthreads();
    // tables to shared memory as they are stored; the Jacobians as fixed point
    auto stage_volume = [&](int q0, int nq) {
        const int2* pv = vpsi + (size_t)e * Q * N + q0;
        for (int t = tid; t < nq * NP; t += T) {
            const int j = t / nq, q = t % nq;
            ps[q * NP + j] = j < N ? fix_shift_round(pv[j * Q + q], FIX_BITS - C::PB) : make_int2(0, 0);
        }
        const int2* gv = vgw + (size_t)e * D * Q * N;
        for (int t = tid; t < nq * D * N; t += T) {
            const int r = t / N, i = t % N;
            gs[t] = fix_shift_round(gv[GradTab<D, P>::at(q0 * D + r, i)], ge[r % D * N + i]);
        }
        if (Q == QC) {
            for (int t = tid; t < Q * D * 25; t += T) As[t] = fix_round(Ad[t], sa[t % 25] - dk[t / 25 % D]);
        } else {
            for (int t = tid; t < nq * D; t += T) {
                double A[25];
                flux_jac_at(q0 + t / D, t % D, A);
#pragma unroll
                for (int x = 0; x < 25; ++x) As[t * 25 + x] = fix_round(A[x], sa[x] - dk[t % D]);
            }
        }
    };
    auto stage_faces = [&](int f0, int nf) {
        for (int t = tid; t < nf * QF * NP; t += T) {
            const int r = t / NP, j = t % NP;
            const int code = elem_face[(size_t)e * NF + f0 + r / QF];
            const int2* pf = ((code & 1) ? fpsiR : fpsiL) + (size_t)(code >> 1) * QF * N;
            fs[t] = j < N ? fix_shift_round(pf[FaceTab<D, P>::at(r % QF, j)], FIX_BITS - C::PB) : make_int2(0, 0);
        }
        for (int t = tid; t < nf * QF * 25; t += T) {
            const int lf = t / (QF * 25), code = elem_face[(size_t)e * NF + f0 + lf];
            const double x = (((code & 1) ? fjr : fjl) + (size_t)(code >> 1) * QF * 25)[t - lf * QF * 25];
            fj[t] = fix_round((code & 1) ? x : -x, sj[t % 25]);
        }
    };
    long long h[N], c[N];
    int ab = 0, i = 0, kv = 0, kf = 0, ks = 0;   // shifts to s of the products (below), the exponent of s
    bool act = false;
    auto take_row = [&](int pass) {
        const int l = pass * C::LIVE + tid / N;
        act = tid < C::LIVE * N && l < nlive;
        ab = act ? live[l] : 0;
        i = tid % N;
        // products of the volume (faces) have exponent ev (ef) and, summed over k, 112 + SV (PB + 56) bits;
        // the kind with the smaller values gives up low bits
        const int ev = ty[i] + m0 + sa[ab], ef = tp + sj[ab];
        ks = min(ev - 2 * FIX_BITS - C::SV, ef - FIX_BITS - C::PB) + C::SB;
        kv = min(ev - ks - 53, 63);
        kf = min(ef - ks - 53, 63);
#pragma unroll
        for (int j = 0; j < N; ++j) h[j] = c[j] = 0;
    };
    // s of the exact product h 2^56 + x 2^28, rounded: its upper 60 (+ SV) bits, shifted by k + 1
    auto add_row = [&](long long ph, long long px, int k, const int2* prow) {
        const long long t = (((ph << 4) + (px >> (FIX_LO - 4))) >> k) + 1;   // s = t >> 1
        const int2 sl = make_int2((int)((t + (1ll << FIX_LO)) >> (FIX_LO + 1)), ((int)t << (31 - FIX_LO)) >> (32 - FIX_LO));
        const int4* p4 = reinterpret_cast<const int4*>(prow);
#pragma unroll
        for (int j = 0; j < N; j += 2) {
            const int4 p = p4[j / 2];
            fix_mac(h[j], c[j], sl, make_int2(p.x, p.y));
            if (j + 1 < N) fix_mac(h[j + 1], c[j + 1], sl, make_int2(p.z, p.w));
        }
    };
    auto mac_volume = [&](int nq) {
#pragma unroll 1
        for (int q = 0; q < nq; ++q) {
            long long sh = 0, sx = 0;
#pragma unroll
            for (int k = 0; k < D; ++k) fix_mac(sh, sx, gs[(q * D + k) * N + i], As[(q * D + k) * 25 + ab]);
            add_row(sh, sx, kv, ps + q * NP);
        }
    };
    auto mac_faces = [&](int np) {
#pragma unroll 1
        for (int t = 0; t < np; ++t) {
            long long sh = 0, sx = 0;
            fix_mac(sh, sx, fs[t * NP + i], fj[t * 25 + ab]);
            add_row(sh, sx, kf, fs + t * NP);
        }
    };
    auto fold = [&]() {
#pragma unroll
        for (int j = 0; j < N; ++j) {
            h[j] += (c[j] + (1ll << (FIX_LO - 1))) >> FIX_LO;
            c[j] = 0;
        }
    };
    // 3-D: the sums so far to this thread's 96-bit ones (words [3][N][LIVE N], one thread's apart from another's)
    unsigned* acc = reinterpret_cast<unsigned*>(sm + C::O_ACC) + tid;
    constexpr int AN = C::LIVE * N;
    auto flush = [&](bool first) {
        fold();
#pragma unroll
        for (int j = 0; j < N; ++j) {
            unsigned lo = (unsigned)h[j], mid = (unsigned)(h[j] >> 32), hi = (unsigned)(h[j] >> 63);
            if (!first)
                asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, %5;"
                    : "+r"(lo), "+r"(mid), "+r"(hi)
                    : "r"(acc[j * AN]), "r"(acc[(N + j) * AN]), "r"(acc[(2 * N + j) * AN]));
            acc[j * AN] = lo;
            acc[(N + j) * AN] = mid;
            acc[(2 * N + j) * AN] = hi;
            h[j] = 0;
        }
    };
    double* slab = reinterpret_cast<double*>(smraw);
    double* blk = out + (size_t)e * B * B;
    if constexpr (D == 2) {
        stage_volume(0, Q);
        stage_faces(0, NF);
    }
    __syncthreads();
    const double idt = shifted ? 1.0 / s_dtau : 0.0;
    take_row(0);
    if constexpr (D == 2) {
        if (act) {
            mac_volume(Q);
            if (C::FOLD) fold();
            mac_faces(FP);
        }
    } else {
#pragma unroll 1
        for (int q0 = 0; q0 < Q; q0 += QC) {
            const int nq = Q - q0 < QC ? Q - q0 : QC;
            if (q0 > 0) __syncthreads();
            stage_volume(q0, nq);
            __syncthreads();
            if (act) {
                mac_volume(nq);
                flush(q0 == 0);
            }
        }
#pragma unroll 1
        for (int lf = 0; lf < NF; ++lf) {
            __syncthreads();
            stage_faces(lf, 1);
            __syncthreads();
            if (act) {
                mac_faces(QF);
                if ((lf + 1) % C::FG == 0 || lf + 1 == NF) flush(false);
            }
        }
    }
    // this thread's N entries of its row to `row`: D, or P = I/dtau - D
    auto put_row = [&](double* row) {
        const double scale = fix_scale(FIX_BITS - ks - tp, max(mxa[ab], mxj[ab]));
#pragma unroll
        for (int j = 0; j < N; ++j) {
            double v;
            if constexpr (D == 2) {
                v = fix_sum(h[j], c[j], scale);
            } else {
                const long long up = (long long)(((unsigned long long)acc[(2 * N + j) * AN] << 32) | acc[(N + j) * AN]);
                v = fma(__ll2double_rn(up), 4294967296.0, (double)acc[j * AN]) * scale;
            }
            row[j] = shifted ? ((ab % 6 == 0 && i == j) ? idt : 0.0) - v : v;   // ab % 6 == 0: a == b
        }
    };
    // entry t of row block a where the pair is not live
    auto dead = [&](int a, int t, double* v) {
        const int r = t / B, b = t % B / N, j = t % N;
        *v = (shifted && a == b && r == j) ? idt : 0.0;
        return mxa[a * 5 + b] == 0 && mxj[a * 5 + b] == 0;
    };
    if (D == 2 && nlive > C::LIVE) {   // two passes over the tables: the rows go straight out
        if (act) put_row(blk + (size_t)(ab / 5 * N + i) * B + ab % 5 * N);
        take_row(1);
        if (act) {
            mac_volume(Q);
            if (C::FOLD) fold();
            mac_faces(FP);
            put_row(blk + (size_t)(ab / 5 * N + i) * B + ab % 5 * N);
        }
        for (int a = 0; a < 5; ++a)
            for (int t = tid; t < N * B; t += T) {
                double v;
                if (dead(a, t, &v)) blk[(size_t)a * N * B + t] = v;
            }
        return;
    }
#pragma unroll 1
    for (int a = 0; a < 5; ++a) {   // the N rows of variable a through shared memory
        __syncthreads();
        for (int t = tid; t < N * B; t += T) {
            double v;
            if (dead(a, t, &v)) slab[t] = v;
        }
        if (act && ab / 5 == a) put_row(slab + i * B + ab % 5 * N);
        __syncthreads();
        for (int t = tid; t < N * B; t += T) blk[(size_t)a * N * B + t] = slab[t];
    }
}

// Levels this form serves: p >= 1, but not the 35-mode hexahedra, whose 140 accumulator registers a
// thread leave no room (k_diag_blocks in jacobian.cu).
bool diag_blocks_fx_serves(int dim, int p) { return p >= 1 && !(dim == 3 && p == 4); }

emg_status launch_diag_blocks_fx(emg_ctx* c, int p, const double* u, const double* cfl_dev, int shifted, double* out) {
    LevelDev& L = c->lv[p];
    const int nmax = n_modes(c->dim, c->p_max);
#define EMG_FX(DD, PP)                                                                                             \
    if constexpr (PP >= 1 && !(DD == 3 && PP == 4)) {                                                              \
        using C = DiagFx<DD, PP>;                                                                                  \
        EMG_CUDA_TRY(c, cudaFuncSetAttribute(k_diag_blocks_fx<DD, PP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM)); \
        ProfScope _ps(c, PC_DIAG);                                                                                 \
        k_diag_blocks_fx<DD, PP><<<(unsigned)c->E, C::THREADS, C::SMEM, c->stream>>>(                              \
            (int)c->E, nmax, u, reinterpret_cast<const int2*>(L.vpsi), reinterpret_cast<const int2*>(L.vgw),       \
            c->elem_face, reinterpret_cast<const int2*>(L.fpsiL), reinterpret_cast<const int2*>(L.fpsiR), L.texp, L.gexp, \
            L.fjl, L.fjr, c->psic, c->h, cfl_dev, c->prm.gamma, shifted, L.vvr, out);                              \
    }
    EMG_DISPATCH_DP(c->dim, p, EMG_FX)
#undef EMG_FX
    EMG_CHECK_LAUNCH(c);
    return EMG_OK;
}

}  // namespace emg
