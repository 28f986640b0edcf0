// Batched element-block solves of the PRK smoother (Eq. prk_scalar), FP64 form, and the
// stage GEMV of the float32 forms:
//  * k_lu: LU factorisation with partial pivoting of every P_e = I/dtau_e - D_e, one CTA
//    per element with the block in shared memory; factors stored column-major, the rows in pivot
//    order and the reciprocals of U's diagonal in its place, so that the substitutions read
//    contiguous columns and divide nothing (k_lu_gmem: the same in global memory for blocks larger
//    than shared memory).
//  * k_stage: one warp per element: y = P_e^{-1} r_e (rows gathered in pivot order, unit-lower
//    forward and upper backward substitution), u^(k) = u^n + beta_k y.
//  * k_stage_gemv: the same stage with the explicit inverse of the float32 forms (gj.cu).
// The residual r, u^n and u^(k) are always double.
//
// A block whose spanwise momentum (variable 3) is coupled to no other variable, every entry of its
// rows and columns outside the 3-3 block being exactly 0 (2-D flow in the plane), splits into
// systems of 4 N and N unknowns.  k_lu_split (2-D levels) finds that by looking at the block, factors the
// two apart and marks it (kSplit in the first pivot), or puts it on a list for k_lu; k_stage then
// solves the large one, and the small one only where r has a spanwise part.  The operations left out all
// have a factor 0, so the factors and solutions are those of the whole block.
#include <type_traits>

#include "blocks.cuh"
#include "common.cuh"
#include "fix.cuh"

namespace emg {

constexpr int kSplit = 1 << 20;   // flag on piv[0]: the block is split

// Position c of system `seg` in the block: the whole block (split = false), or variables 0, 1, 2, 4
// (seg 0) and variable 3 (seg 1).
template <int B>
__device__ __forceinline__ int seg_at(bool split, int seg, int c) {
    constexpr int N = B / 5;
    return !split ? c : seg ? 3 * N + c : c < 3 * N ? c : c + N;
}
template <int B>
__device__ __forceinline__ int seg_size(bool split, int seg) {
    return !split ? B : seg ? B / 5 : B / 5 * 4;
}

// Factorisation of an n x n system in shared memory (row stride LD) by 1 + WX WY warps, threads tid = 0
// .. of the block; barriers under id 1, so that other warps of the block may do something else.
// Bound by the float64 pipe (n^3 / 3 multiply-adds) and, per step, two barriers: warp 0 updates the
// next column and finds its pivot while the other warps update the rest.  A warp's update tile is 8
// rows by 4 columns (not 1 by 32), which wastes fewer lanes on the shrinking trailing block, and a
// warp issues only the tiles it has: an operation whose lanes are all off takes the pipe as long (4560
// float64 warp instructions a 60 x 60 block with four tiles always, 2900 needed).
template <int n, int LD, int WX, int WY>
__device__ __forceinline__ void lu_factor(double* a, int* rid, volatile int* s_piv, volatile double* s_inv, int tid) {
    constexpr int T = 32 * (1 + WX * WY), GX = 4 * WX, GY = 8 * WY;
    const int lane = tid & 31, w = (tid >> 5) - 1;
    const int tx = (w % WX) * 4 + (lane & 3), ty = (w / WX) * 8 + (lane >> 2);
    auto barrier = []() { asm volatile("bar.sync 1, %0;" ::"n"(T) : "memory"); };
    // warp 0: the pivot row of step t (the first of the largest |a|), its reciprocal, the row order
    auto find_pivot = [&](int t) {
        long long best = -2;   // every key is >= -1: a NaN row is taken only if no row is a number
        int bi = t;
        for (int r = t + lane; r < n; r += 32) {
            const long long v = piv_key(a[r * LD + t]);
            if (v > best) {
                best = v;
                bi = r;
            }
        }
        for (int o = 16; o > 0; o >>= 1) {
            const long long ob = __shfl_xor_sync(0xffffffffu, best, o);
            const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
            if (ob > best || (ob == best && oi < bi)) {
                best = ob;
                bi = oi;
            }
        }
        const double inv = rcp_h3(a[bi * LD + t]);
        if (lane == 0) {
            *s_piv = bi;
            *s_inv = inv;
            const int r0 = rid[t];
            rid[t] = rid[bi];
            rid[bi] = r0;
        }
    };
    if (w < 0) find_pivot(0);
    barrier();
#pragma unroll 1
    for (int t = 0; t < n; ++t) {
        const int pr = *s_piv;
        const double inv = *s_inv;
        // swap rows t and pr outside column t; column t: the multipliers of the rows below, with the
        // row that was t at pr, and the pivot's reciprocal
        for (int c = tid; c < n; c += T) {
            if (c != t && pr != t) {
                const double t0 = a[t * LD + c];
                a[t * LD + c] = a[pr * LD + c];
                a[pr * LD + c] = t0;
            }
            if (c > t && c != pr) a[c * LD + t] *= inv;
            if (c == t) {
                if (pr != t) a[pr * LD + t] = a[t * LD + t] * inv;
                a[t * LD + t] = inv;
            }
        }
        barrier();
        if (w < 0) {
            // the next column first, then its pivot, while the other warps update the rest
            if (t + 1 < n) {
                const double u = a[t * LD + t + 1];
                for (int r = t + 1 + lane; r < n; r += 32) a[r * LD + t + 1] = fma(-a[r * LD + t], u, a[r * LD + t + 1]);
                __syncwarp();
                find_pivot(t + 1);
            }
        } else {
            // NP of the tiles c0 + p GX at a time, as many as the warp has
            auto tiles = [&](auto np, int c0) {
                constexpr int NP = decltype(np)::value;
                double u[NP];
#pragma unroll
                for (int p = 0; p < NP; ++p) u[p] = c0 + p * GX < n ? a[t * LD + c0 + p * GX] : 0.0;
                for (int r = t + 1 + ty; r < n; r += GY) {
                    double* row = a + r * LD + c0;
                    const double l = a[r * LD + t];
#pragma unroll
                    for (int p = 0; p < NP; ++p)
                        if (c0 + p * GX < n) row[p * GX] = fma(-l, u[p], row[p * GX]);
                }
            };
            for (int c0 = t + 2 + tx, cw = c0 - (lane & 3); cw < n; c0 += 4 * GX, cw += 4 * GX) {
                if (cw + 3 * GX < n)
                    tiles(std::integral_constant<int, 4>{}, c0);
                else if (cw + 2 * GX < n)
                    tiles(std::integral_constant<int, 3>{}, c0);
                else if (cw + GX < n)
                    tiles(std::integral_constant<int, 2>{}, c0);
                else
                    tiles(std::integral_constant<int, 1>{}, c0);
            }
        }
        barrier();
    }
}

template <int B>
struct LuCfg {
    static constexpr int LD = (B + 3) / 8 * 8 + 4;   // row stride: 8 x 4 tiles of a warp hit every bank once
    static constexpr size_t SMEM = (size_t)B * LD * sizeof(double);
    static constexpr int WX = B <= 30 ? 2 : 4;   // update warps across columns (4 each) and rows (8 each)
    static constexpr int WY = B <= 20 ? 1 : 2;
    static constexpr int THREADS = 32 * (1 + WX * WY);   // warp 0: pivots
    static_assert(LD >= B && LD % 8 == 4, "row stride");
};

// Every block of the level (list = nullptr, one CTA each), or those that k_lu_split left.
template <int B>
__global__ void __launch_bounds__(LuCfg<B>::THREADS) k_lu(int E, double* __restrict__ blk, int* __restrict__ piv,
                                                         const int* __restrict__ list, int* __restrict__ head) {
    using C = LuCfg<B>;
    constexpr int LD = C::LD, T = C::THREADS;
    extern __shared__ __align__(16) unsigned char smraw[];
    double* a = reinterpret_cast<double*>(smraw);
    __shared__ int rid[B], s_piv;
    __shared__ double s_inv;
    const int tid = threadIdx.x;
    const int ne = list ? take_list(head) : E;
#pragma unroll 1
    for (int it = blockIdx.x; it < ne; it += gridDim.x) {
        const int e = list ? list[it] : it;
        double* g = blk + (size_t)e * B * B;
        __syncthreads();
        for (int t = tid; t < B * B; t += T) a[(t / B) * LD + t % B] = g[t];
        for (int t = tid; t < B; t += T) rid[t] = t;
        __syncthreads();
        lu_factor<B, LD, C::WX, C::WY>(a, rid, &s_piv, &s_inv, tid);
        __syncthreads();
        for (int t = tid; t < B; t += T) piv[(size_t)e * B + t] = rid[t];
        // column-major out: g[col * B + row]
        for (int t = tid; t < B * B; t += T) g[t] = a[(t % B) * LD + t / B];
    }
}

// 2-D levels: the 4 N x 4 N system by the first warps, the N x N one by the last warp beside them.
// What is left out of shared memory lets six blocks share an SM at N = 15 (four with the whole block).
// FP64 V-cycle of the 128 x 64 O-grid at p = 4: 8.0 -> 4.75 ms in factorisations, 19.5 -> 16.3 ms in all.
template <int N>
struct LuSplit {
    static constexpr int B4 = 4 * N, LD = (B4 + 3) / 8 * 8 + 4, LD3 = N | 1;
    static constexpr int WX = N <= 6 ? 2 : 4, WY = N <= 3 ? 1 : N <= 10 ? 1 : 2;
    static constexpr int MAIN = 32 * (1 + WX * WY), THREADS = MAIN + 32;
    static constexpr size_t SMEM = (size_t)(B4 * LD + N * LD3) * sizeof(double);
    static constexpr int MINB = N == 15 ? 6 : N == 10 ? 10 : 16;
};
template <int N>
__global__ void __launch_bounds__(LuSplit<N>::THREADS, LuSplit<N>::MINB) k_lu_split(int E, double* __restrict__ blk,
                                                                                    int* __restrict__ piv,
                                                                                    int* __restrict__ list,
                                                                                    int* __restrict__ head) {
    using C = LuSplit<N>;
    constexpr int B = 5 * N, B4 = C::B4, LD = C::LD, LD3 = C::LD3, T = C::THREADS;
    extern __shared__ __align__(16) unsigned char smraw[];
    double* a = reinterpret_cast<double*>(smraw);
    double* a3 = a + B4 * LD;
    __shared__ int rid[B4], rid3[N], s_piv;
    __shared__ double s_inv;
    const int e = blockIdx.x, tid = threadIdx.x;
    double* g = blk + (size_t)e * B * B;
    bool coupled = false;
#pragma unroll 4
    for (int t = tid; t < B * B; t += T) {
        const int r = t / B, c = t - r * B, rs = r / N, cs = c / N;
        const double v = g[t];
        if (rs != 3 && cs != 3)
            a[(rs == 4 ? r - N : r) * LD + (cs == 4 ? c - N : c)] = v;
        else if (rs == cs)
            a3[(r - 3 * N) * LD3 + c - 3 * N] = v;
        else
            coupled |= !(v == 0.0);
    }
    for (int t = tid; t < B4; t += T) rid[t] = t;
    if (__syncthreads_or(coupled)) {
        if (tid == 0) list[atomicAdd(head, 1)] = e;
        return;
    }
    if (tid < C::MAIN) {
        lu_factor<B4, LD, C::WX, C::WY>(a, rid, &s_piv, &s_inv, tid);
    } else {   // lane r: row r
        const int lane = tid & 31;
        if (lane < N) rid3[lane] = lane;
        __syncwarp();
#pragma unroll 1
        for (int t = 0; t < N; ++t) {
            long long best = lane >= t && lane < N ? piv_key(a3[lane * LD3 + t]) : -2;
            int p = lane >= t && lane < N ? lane : t;
            for (int o = 16; o > 0; o >>= 1) {
                const long long ob = __shfl_xor_sync(0xffffffffu, best, o);
                const int oi = __shfl_xor_sync(0xffffffffu, p, o);
                if (ob > best || (ob == best && oi < p)) {
                    best = ob;
                    p = oi;
                }
            }
            const double inv = rcp_h3(a3[p * LD3 + t]);
            __syncwarp();
            if (lane < N && p != t) {
                const double t0 = a3[t * LD3 + lane];
                a3[t * LD3 + lane] = a3[p * LD3 + lane];
                a3[p * LD3 + lane] = t0;
            }
            if (lane == 0) {
                const int r0 = rid3[t];
                rid3[t] = rid3[p];
                rid3[p] = r0;
            }
            __syncwarp();
            if (lane > t && lane < N) {
                const double l = a3[lane * LD3 + t] * inv;
                a3[lane * LD3 + t] = l;
                for (int c = t + 1; c < N; ++c) a3[lane * LD3 + c] = fma(-l, a3[t * LD3 + c], a3[lane * LD3 + c]);
            }
            if (lane == t) a3[t * LD3 + t] = inv;
            __syncwarp();
        }
    }
    __syncthreads();
    for (int t = tid; t < B; t += T) {
        const int s = t / N;
        const int r = s == 3 ? 3 * N + rid3[t - 3 * N] : rid[s == 4 ? t - N : t];
        piv[(size_t)e * B + t] = (s != 3 && r >= 3 * N ? r + N : r) | (t == 0 ? kSplit : 0);
    }
    // column-major out: g[col * B + row], the two systems' places only
    for (int t = tid; t < B4 * B4; t += T) {
        const int c = t / B4, r = t % B4;
        g[(size_t)seg_at<B>(true, 0, c) * B + seg_at<B>(true, 0, r)] = a[r * LD + c];
    }
    for (int t = tid; t < N * N; t += T) g[(size_t)(3 * N + t / N) * B + 3 * N + t % N] = a3[t % N * LD3 + t / N];
}

// The same factorisation for blocks that do not fit in shared memory (B = 175 in float64):
// the block is factored in place in global memory (it stays in L2 while its CTA works on it),
// row-major during the elimination, then transposed in place to the column-major layout the
// substitutions read.  Pivot choice and tie rule as in k_lu; never split.
template <int B>
__global__ void __launch_bounds__(256) k_lu_gmem(int E, double* __restrict__ blk, int* __restrict__ piv) {
    __shared__ int rid[B], s_piv;
    const int e = blockIdx.x;
    const int tid = threadIdx.x, nth = blockDim.x;
    double* a = blk + (size_t)e * B * B;
    for (int t = tid; t < B; t += nth) rid[t] = t;
    __syncthreads();
    for (int k = 0; k < B; ++k) {
        if (tid < 32) {
            long long best = -2;
            int bi = k;
            for (int r = k + tid; r < B; r += 32) {
                const long long v = piv_key(a[(size_t)r * B + k]);
                if (v > best) {
                    best = v;
                    bi = r;
                }
            }
            for (int o = 16; o > 0; o >>= 1) {
                const long long ob = __shfl_xor_sync(0xffffffffu, best, o);
                const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
                if (ob > best || (ob == best && oi < bi)) {
                    best = ob;
                    bi = oi;
                }
            }
            if (tid == 0) {
                s_piv = bi;
                const int r0 = rid[k];
                rid[k] = rid[bi];
                rid[bi] = r0;
            }
        }
        __syncthreads();
        const int pr = s_piv;
        if (pr != k)
            for (int cc = tid; cc < B; cc += nth) {
                const double t0 = a[(size_t)k * B + cc];
                a[(size_t)k * B + cc] = a[(size_t)pr * B + cc];
                a[(size_t)pr * B + cc] = t0;
            }
        __syncthreads();
        const double inv = 1.0 / a[(size_t)k * B + k];
        if (k + 1 + tid < B)
            for (int r = k + 1 + tid; r < B; r += nth) a[(size_t)r * B + k] *= inv;
        __syncthreads();
        const int tx = tid & 31, ty = tid >> 5;
        for (int r = k + 1 + ty; r < B; r += 8) {
            const double l = a[(size_t)r * B + k];
            for (int cc = k + 1 + tx; cc < B; cc += 32) a[(size_t)r * B + cc] -= l * a[(size_t)k * B + cc];
        }
        if (tid == 0) a[(size_t)k * B + k] = inv;
        __syncthreads();
    }
    for (int t = tid; t < B; t += nth) piv[(size_t)e * B + t] = rid[t];
    // row-major -> column-major, in place
    for (int t = tid; t < B * B; t += nth) {
        const int r = t / B, cc = t % B;
        if (r < cc) {
            const double t0 = a[(size_t)r * B + cc];
            a[(size_t)r * B + cc] = a[(size_t)cc * B + r];
            a[(size_t)cc * B + r] = t0;
        }
    }
}

// Substitutions of one system by one warp: lane l holds positions l + 32 s (slots s < RS) of y in
// registers; step j broadcasts y_j and every lane takes its entries of column j, which do not depend
// on the steps before: eight columns' loads are issued together.
template <int B, int RS>
__device__ __forceinline__ void substitute(const double* __restrict__ M, bool split, int seg, int n, int lane,
                                           double (&y)[RS]) {
    int row[RS];
#pragma unroll
    for (int s = 0; s < RS; ++s) {
        const int c = lane + 32 * s;
        row[s] = seg_at<B>(split, seg, c < n ? c : n - 1);
    }
    // forward: y_c -= L[c][j] y_j, c > j
#pragma unroll
    for (int sj = 0; sj < RS; ++sj) {
        const int j1 = n < 32 * sj + 32 ? n : 32 * sj + 32;
#pragma unroll 1
        for (int j0 = 32 * sj; j0 < j1; j0 += 8) {
            double m[8][RS];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int j = j0 + q < n ? j0 + q : n - 1;
                const double* col = M + (size_t)seg_at<B>(split, seg, j) * B;
#pragma unroll
                for (int s = sj; s < RS; ++s) m[q][s] = col[row[s]];
            }
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int j = j0 + q;
                if (j < j1) {   // uniform
                    const double yj = __shfl_sync(0xffffffffu, y[sj], j & 31);
                    if (lane + 32 * sj > j) y[sj] = fma(-m[q][sj], yj, y[sj]);
#pragma unroll
                    for (int s = sj + 1; s < RS; ++s) y[s] = fma(-m[q][s], yj, y[s]);
                }
            }
        }
    }
    // backward: x_j = y_j / U[j][j], y_c -= U[c][j] x_j, c < j
    double rd[RS];
#pragma unroll
    for (int s = 0; s < RS; ++s) rd[s] = M[(size_t)row[s] * B + row[s]];
#pragma unroll
    for (int sj = RS - 1; sj >= 0; --sj) {
        const int j1 = n < 32 * sj + 32 ? n : 32 * sj + 32;
#pragma unroll 1
        for (int j0 = j1 - 1; j0 >= 32 * sj; j0 -= 8) {
            double m[8][RS];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int j = j0 - q > 0 ? j0 - q : 0;
                const double* col = M + (size_t)seg_at<B>(split, seg, j) * B;
#pragma unroll
                for (int s = 0; s <= sj; ++s) m[q][s] = col[row[s]];
            }
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int j = j0 - q;
                if (j >= 32 * sj) {   // uniform
                    const double xj = __shfl_sync(0xffffffffu, y[sj] * rd[sj], j & 31);
                    const int c = lane + 32 * sj;
                    y[sj] = c == j ? xj : c < j ? fma(-m[q][sj], xj, y[sj]) : y[sj];
#pragma unroll
                    for (int s = 0; s < sj; ++s) y[s] = fma(-m[q][s], xj, y[s]);
                }
            }
        }
    }
}

// u^(k) = u^n + beta P_e^{-1} r_e with the factors of k_lu.  One launch at 128 x 64, p = 4 reads the
// 369 MB of factors in 143 us (ncu; 370 us with the row swaps one after the other, divisions and the
// columns loaded step by step), the float64 pipe 80 % busy: half of a triangle's lanes are idle.
template <int B>
__global__ void __launch_bounds__(128) k_stage(int E, const double* __restrict__ lu, const int* __restrict__ piv,
                                               const double* __restrict__ r, const double* __restrict__ un,
                                               double beta, double* __restrict__ out) {
    constexpr int N = B / 5;
    const int lane = threadIdx.x & 31;
    const int e = blockIdx.x * 4 + (threadIdx.x >> 5);
    if (e >= E) return;
    const double* M = lu + (size_t)e * B * B;
    const double* re = r + (size_t)e * B;
    const int* pv = piv + (size_t)e * B;
    const bool split = (pv[0] & kSplit) != 0;   // uniform over the warp
    auto solve = [&](auto rs, int seg) {
        constexpr int RS = decltype(rs)::value;
        const int n = seg_size<B>(split, seg);
        double y[RS];
#pragma unroll
        for (int s = 0; s < RS; ++s) {
            const int c = lane + 32 * s;
            y[s] = c < n ? re[pv[seg_at<B>(split, seg, c)] & (kSplit - 1)] : 0.0;
        }
        substitute<B, RS>(M, split, seg, n, lane, y);
#pragma unroll
        for (int s = 0; s < RS; ++s) {
            const int c = lane + 32 * s;
            if (c < n) {
                const size_t o = (size_t)e * B + seg_at<B>(split, seg, c);
                out[o] = un[o] + beta * y[s];
            }
        }
    };
    if (!split) {
        solve(std::integral_constant<int, (B + 31) / 32>{}, 0);
        return;
    }
    solve(std::integral_constant<int, (4 * N + 31) / 32>{}, 0);
    bool any = false;
    for (int i = lane; i < N; i += 32) any |= !(re[3 * N + i] == 0.0);
    if (__any_sync(0xffffffffu, any)) {
        solve(std::integral_constant<int, (N + 31) / 32>{}, 1);
    } else {
        for (int i = lane; i < N; i += 32) out[(size_t)e * B + 3 * N + i] = un[(size_t)e * B + 3 * N + i];
    }
}

// u^(k) = u^n + beta P_e^{-1} r_e with P_e^{-1} column-major: one warp per element, each
// lane owns rows lane, lane+32, ...; every column is a coalesced read.  Bound by the bytes of the
// inverses.  SPLIT (2-D): an element with a packed inverse (blocks.cuh) reads its 16 N^2 floats 16
// bytes at a time, all loads independent: 32 / N groups of N lanes take the columns in turn, lane q of a
// group the rows 4 q .. 4 q + 3, and the groups' sums are added at the end; the N x N spanwise part only
// where r has one.  128 x 64, p = 4: 40 -> 27.5 us a launch (126 MB of inverses).
template <int B, bool SPLIT>
__global__ void __launch_bounds__(128) k_stage_gemv(int E, const float* __restrict__ inv, const int* __restrict__ split,
                                                    const double* __restrict__ r, const double* __restrict__ un,
                                                    double beta, double* __restrict__ out) {
    constexpr int RPL = (B + 31) / 32, N = B / 5, B4 = 4 * N;
    __shared__ __align__(16) float rs[4][(B + 3) / 4 * 4];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int e = blockIdx.x * 4 + warp;
    if (e >= E) return;
    const double* re = r + (size_t)e * B;
    const double* ue = un + (size_t)e * B;
    double* oe = out + (size_t)e * B;
    if (SPLIT && split[e]) {   // uniform over the warp
        constexpr int G = 32 / (N <= 32 ? N : 32), K = (B4 + G - 1) / G;
        const float4* M4 = reinterpret_cast<const float4*>(inv + gj_packed_at(e, B));
        const int q = lane % N, g = lane / N;
        bool any = false;
        for (int t = lane; t < B; t += 32) {   // packed order: variables 0, 1, 2, 4, then 3
            const float v = (float)re[t];
            any |= t / N == 3 && !(re[t] == 0.0);
            rs[warp][t < 3 * N ? t : t < B4 ? t + N : t - N] = v;
        }
        any = __any_sync(0xffffffffu, any);
        __syncwarp();
        float4 acc = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (g < G) {
#pragma unroll 10
            for (int k = 0; k < K; ++k) {
                const int j = k * G + g;
                if (B4 % G == 0 || j < B4) {
                    const float rj = rs[warp][j];
                    const float4 m = __ldg(M4 + j * N + q);
                    acc.x = fmaf(m.x, rj, acc.x);
                    acc.y = fmaf(m.y, rj, acc.y);
                    acc.z = fmaf(m.z, rj, acc.z);
                    acc.w = fmaf(m.w, rj, acc.w);
                }
            }
        }
        float4 sum = acc;
#pragma unroll
        for (int h = 1; h < G; ++h) {
            sum.x += __shfl_sync(0xffffffffu, acc.x, (lane + h * N) & 31);
            sum.y += __shfl_sync(0xffffffffu, acc.y, (lane + h * N) & 31);
            sum.z += __shfl_sync(0xffffffffu, acc.z, (lane + h * N) & 31);
            sum.w += __shfl_sync(0xffffffffu, acc.w, (lane + h * N) & 31);
        }
        float s3 = 0.0f;
        if (any && lane < N) {
            const float* M3 = reinterpret_cast<const float*>(M4) + B4 * B4;
#pragma unroll
            for (int j = 0; j < N; ++j) s3 = fmaf(__ldg(M3 + j * N + lane), rs[warp][B4 + j], s3);
        }
        __syncwarp();
        if (g == 0) *reinterpret_cast<float4*>(&rs[warp][4 * q]) = sum;
        if (lane < N) rs[warp][B4 + lane] = s3;
        __syncwarp();
        for (int t = lane; t < B; t += 32)
            oe[t] = ue[t] + beta * (double)rs[warp][t < 3 * N ? t : t < B4 ? t + N : t - N];
        return;
    }
    for (int t = lane; t < B; t += 32) rs[warp][t] = (float)re[t];
    __syncwarp();
    float acc[RPL];
#pragma unroll
    for (int t = 0; t < RPL; ++t) acc[t] = 0.0f;
    const float* M = inv + (size_t)e * B * B;
#pragma unroll 4
    for (int j = 0; j < B; ++j) {
        const float rj = rs[warp][j];
        const float* col = M + (size_t)j * B;
#pragma unroll
        for (int t = 0; t < RPL; ++t) {
            const int i = lane + 32 * t;
            if (i < B) acc[t] += __ldg(col + i) * rj;
        }
    }
#pragma unroll
    for (int t = 0; t < RPL; ++t) {
        const int i = lane + 32 * t;
        if (i < B) oe[i] = ue[i] + beta * (double)acc[t];
    }
}

template <int N>
static emg_status lu_split(emg_ctx* c, LevelDev& L) {
    using C = LuSplit<N>;
    EMG_CUDA_TRY(c, cudaFuncSetAttribute(k_lu_split<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM));
    EMG_CUDA_TRY(c, cudaFuncSetAttribute(k_lu<5 * N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)LuCfg<5 * N>::SMEM));
    const unsigned E = (unsigned)c->E;
    {
        ProfScope _ps(c, PC_LU);
        k_lu_split<N><<<E, C::THREADS, C::SMEM, c->stream>>>((int)E, L.blk, L.piv, L.lu_list, L.lu_list + E);
    }
    EMG_CHECK_LAUNCH(c);
    ProfScope _ps(c, PC_LU);
    k_lu<5 * N><<<list_grid(c->E, LuCfg<5 * N>::THREADS), LuCfg<5 * N>::THREADS, LuCfg<5 * N>::SMEM, c->stream>>>(
        (int)E, L.blk, L.piv, L.lu_list, L.lu_list + E);
    EMG_CHECK_LAUNCH(c);
    return EMG_OK;
}

template <int B>
static emg_status lu_whole(emg_ctx* c, LevelDev& L) {
    const unsigned E = (unsigned)c->E;
    if constexpr (LuCfg<B>::SMEM > 227 * 1024) {
        ProfScope _ps(c, PC_LU);
        k_lu_gmem<B><<<E, 256, 0, c->stream>>>((int)E, L.blk, L.piv);
    } else {
        const size_t sm = LuCfg<B>::SMEM;
        EMG_CUDA_TRY(c, cudaFuncSetAttribute(k_lu<B>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
        ProfScope _ps(c, PC_LU);
        k_lu<B><<<E, LuCfg<B>::THREADS, sm, c->stream>>>((int)E, L.blk, L.piv, nullptr, nullptr);
    }
    EMG_CHECK_LAUNCH(c);
    return EMG_OK;
}

static emg_status stage_dispatch(emg_ctx* c, int B, const double* lu, const int* piv, const double* r,
                                 const double* un, double beta, double* out) {
    const unsigned E = (unsigned)c->E;
    switch (B) {
#define EMG_ST_CASE(BB)                                                                          \
    case BB: {                                                                                   \
        ProfScope _ps(c, PC_STAGE);                                                              \
        k_stage<BB><<<(E + 3) / 4, 128, 0, c->stream>>>((int)E, lu, piv, r, un, beta, out);      \
    }                                                                                            \
        EMG_CHECK_LAUNCH(c);                                                                     \
        return EMG_OK;
        EMG_BSIZES(EMG_ST_CASE)
#undef EMG_ST_CASE
        default:
            c->err = "unsupported block size";
            return EMG_ERR_ARG;
    }
}

emg_status launch_lu(emg_ctx* c, int p) {
    LevelDev& L = c->lv[p];
    if (c->dim == 2) switch (p) {
            case 1: return lu_split<3>(c, L);
            case 2: return lu_split<6>(c, L);
            case 3: return lu_split<10>(c, L);
            default: return lu_split<15>(c, L);
        }
    switch (p) {
        case 1: return lu_whole<20>(c, L);
        case 2: return lu_whole<50>(c, L);
        case 3: return lu_whole<100>(c, L);
        default: return lu_whole<175>(c, L);
    }
}

emg_status launch_stage(emg_ctx* c, int p, const double* r, const double* un, double beta, double* out) {
    LevelDev& L = c->lv[p];
    return stage_dispatch(c, L.B, L.blk, L.piv, r, un, beta, out);
}

emg_status launch_stage32(emg_ctx* c, int p, const double* r, const double* un, double beta, double* out) {
    LevelDev& L = c->lv[p];
    const unsigned E = (unsigned)c->E;
    switch (L.B) {
#define EMG_GV_CASE(BB)                                                                                  \
    case BB: {                                                                                           \
        ProfScope _ps(c, PC_STAGE);                                                                      \
        if (L.gj_split)                                                                                  \
            k_stage_gemv<BB, (BB <= 75 && BB != 20)><<<(E + 3) / 4, 128, 0, c->stream>>>((int)E, L.blk32, gj_work(L.piv, E).flag, r, un, beta, out); \
        else                                                                                             \
            k_stage_gemv<BB, false><<<(E + 3) / 4, 128, 0, c->stream>>>((int)E, L.blk32, nullptr, r, un, beta, out);                \
    }                                                                                                    \
        EMG_CHECK_LAUNCH(c);                                                                             \
        return EMG_OK;
        EMG_BSIZES(EMG_GV_CASE)
#undef EMG_GV_CASE
        default:
            c->err = "unsupported block size";
            return EMG_ERR_ARG;
    }
}

}  // namespace emg
