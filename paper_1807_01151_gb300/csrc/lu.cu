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
// systems of 4 N and N unknowns.  k_lu finds that by looking at the block, factors the two apart
// and marks it (kSplit in the first pivot); k_stage then solves the large one, and the small one
// only where r has a spanwise part.  The operations left out all have a factor 0, so the factors and
// solutions are those of the whole block.
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

template <int B>
struct LuCfg {
    static constexpr int LD = (B + 3) / 8 * 8 + 4;   // row stride: 8 x 4 tiles of a warp hit every bank once
    static constexpr size_t SMEM = (size_t)B * LD * sizeof(double);
    static constexpr int WX = B <= 30 ? 2 : 4;   // update warps across columns (4 each) and rows (8 each)
    static constexpr int WY = B <= 20 ? 1 : 2;
    static constexpr int THREADS = 32 * (1 + WX * WY);   // warp 0: pivots
    static_assert(LD >= B && LD % 8 == 4, "row stride");
};

// Bound by the float64 pipe (B^3 / 3 multiply-adds) and, per step, two barriers: warp 0 updates the
// next column and finds its pivot while the other warps update the rest.  A warp's update tile is 8
// rows by 4 columns (not 1 by 32), which wastes fewer lanes on the shrinking trailing block.  128 x 64 O-grid, FP64 V-cycle at p = 4: 9.5 ms with search, swap, scaling and a 1-by-32
// update of the whole 75 x 75 block each behind a barrier, 8.0 ms as it is (the float64 pipe 73 %
// busy, the division of a step a correctly rounded one: 8.3).
template <int B>
__global__ void __launch_bounds__(LuCfg<B>::THREADS) k_lu(int E, double* __restrict__ blk, int* __restrict__ piv) {
    using C = LuCfg<B>;
    constexpr int LD = C::LD, T = C::THREADS, N = B / 5, GX = 4 * C::WX, GY = 8 * C::WY;
    extern __shared__ __align__(16) unsigned char smraw[];
    double* a = reinterpret_cast<double*>(smraw);
    __shared__ int rid[B], s_piv;
    __shared__ double s_inv;
    const int e = blockIdx.x, tid = threadIdx.x;
    double* g = blk + (size_t)e * B * B;
    bool coupled = false;
    for (int t = tid; t < B * B; t += T) {
        const int r = t / B, c = t % B;
        const double v = g[t];
        a[r * LD + c] = v;
        coupled |= (r / N == 3) != (c / N == 3) && !(v == 0.0);
    }
    for (int t = tid; t < B; t += T) rid[t] = t;
    const bool split = !__syncthreads_or(coupled);
    const int lane = tid & 31, w = (tid >> 5) - 1;
    const int tx = (w % C::WX) * 4 + (lane & 3), ty = (w / C::WX) * 8 + (lane >> 2);
#pragma unroll 1
    for (int seg = 0; seg < (split ? 2 : 1); ++seg) {
        const int n = seg_size<B>(split, seg);
        // warp 0: the pivot row of step t (the first of the largest |a|), its reciprocal, the row order
        auto find_pivot = [&](int t) {
            const int k = seg_at<B>(split, seg, t);
            long long best = -2;   // every key is >= -1: a NaN row is taken only if no row is a number
            int bi = k;
            for (int c = t + lane; c < n; c += 32) {
                const int r = seg_at<B>(split, seg, c);
                const long long v = piv_key(a[r * LD + k]);
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
            const double inv = rcp_h3(a[bi * LD + k]);
            if (lane == 0) {
                s_piv = bi;
                s_inv = inv;
                const int r0 = rid[k];
                rid[k] = rid[bi];
                rid[bi] = r0;
            }
        };
        if (w < 0) find_pivot(0);
        __syncthreads();
#pragma unroll 1
        for (int t = 0; t < n; ++t) {
            const int k = seg_at<B>(split, seg, t);
            const int pr = s_piv;
            const double inv = s_inv;
            // swap rows k and pr outside column k; column k: the multipliers of the rows below, with the
            // row that was k at pr, and the pivot's reciprocal
            for (int c = tid; c < n; c += T) {
                const int cc = seg_at<B>(split, seg, c);
                if (c != t && pr != k) {
                    const double t0 = a[k * LD + cc];
                    a[k * LD + cc] = a[pr * LD + cc];
                    a[pr * LD + cc] = t0;
                }
                if (c > t && cc != pr) a[cc * LD + k] *= inv;
                if (c == t) {
                    if (pr != k) a[pr * LD + k] = a[k * LD + k] * inv;
                    a[k * LD + k] = inv;
                }
            }
            __syncthreads();
            if (w < 0) {
                // the next column first, then its pivot, while the other warps update the rest
                if (t + 1 < n) {
                    const int kn = seg_at<B>(split, seg, t + 1);
                    const double u = a[k * LD + kn];
                    for (int c = t + 1 + lane; c < n; c += 32) {
                        double* row = a + seg_at<B>(split, seg, c) * LD;
                        row[kn] = fma(-row[k], u, row[kn]);
                    }
                    __syncwarp();
                    find_pivot(t + 1);
                }
            } else {
                for (int c0 = t + 2 + tx; c0 < n; c0 += 4 * GX) {
                    double u[4];
                    int cc[4];
#pragma unroll
                    for (int p = 0; p < 4; ++p) {
                        cc[p] = c0 + p * GX < n ? seg_at<B>(split, seg, c0 + p * GX) : -1;
                        u[p] = cc[p] >= 0 ? a[k * LD + cc[p]] : 0.0;
                    }
                    for (int r = t + 1 + ty; r < n; r += GY) {
                        double* row = a + seg_at<B>(split, seg, r) * LD;
                        const double l = row[k];
#pragma unroll
                        for (int p = 0; p < 4; ++p)
                            if (cc[p] >= 0) row[cc[p]] = fma(-l, u[p], row[cc[p]]);
                    }
                }
            }
            __syncthreads();
        }
    }
    for (int t = tid; t < B; t += T) piv[(size_t)e * B + t] = rid[t] | (split && t == 0 ? kSplit : 0);
    // column-major out: g[col * B + row]
    for (int t = tid; t < B * B; t += T) g[t] = a[(t % B) * LD + t / B];
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

static emg_status lu_dispatch(emg_ctx* c, int B, double* blk, int* piv) {
    const unsigned E = (unsigned)c->E;
    switch (B) {
#define EMG_LU_CASE(BB)                                                                                      \
    case BB: {                                                                                               \
        if constexpr (LuCfg<BB>::SMEM > 227 * 1024) {                                                        \
            ProfScope _ps(c, PC_LU);                                                                         \
            k_lu_gmem<BB><<<E, 256, 0, c->stream>>>((int)E, blk, piv);                                       \
        } else {                                                                                             \
            const size_t sm = LuCfg<BB>::SMEM;                                                               \
            EMG_CUDA_TRY(c, cudaFuncSetAttribute(k_lu<BB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm)); \
            ProfScope _ps(c, PC_LU);                                                                         \
            k_lu<BB><<<E, LuCfg<BB>::THREADS, sm, c->stream>>>((int)E, blk, piv);                            \
        }                                                                                                    \
        EMG_CHECK_LAUNCH(c);                                                                                 \
        return EMG_OK;                                                                                       \
    }
        EMG_BSIZES(EMG_LU_CASE)
#undef EMG_LU_CASE
        default:
            c->err = "unsupported block size";
            return EMG_ERR_ARG;
    }
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

emg_status launch_lu(emg_ctx* c, int p) { return lu_dispatch(c, c->lv[p].B, c->lv[p].blk, c->lv[p].piv); }

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
