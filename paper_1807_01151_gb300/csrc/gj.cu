// Explicit inverses P_e^{-1} of the float32 block forms by Gauss-Jordan elimination with
// partial pivoting (SIMT forms), their variants and the per-device tuner.  The tensor-core
// form is in gj_tc.cu.
#include <algorithm>
#include <cstdio>
#include <map>
#include <mutex>
#include <string>
#include <tuple>

#include "blocks.cuh"
#include "common.cuh"
#include "gj.cuh"

namespace emg {

emg_status launch_gj_tc(emg_ctx* c, int B, float* blk, bool* built);

// Blocked form of the same Gauss-Jordan inversion (right-looking, panels of NB = 8 pivot
// columns), SIMT.  Layout of k_gj_cols: lane tx owns rows tx + 32 i, warp w owns columns
// w + W j; after every panel each thread rotates its column slots by NB / W, so the next
// panel's columns always sit in slots 0 .. NB/W - 1 (no runtime-indexed register access).
// The NB steps of a panel act on every column c outside it as A[:, c] <- T A[:, c],
// T = T_{k0+NB-1} ... T_{k0} (T_k: the elementary Gauss-Jordan transform of step k, identity
// but for column p_k).  T differs from I only in the pivot-row columns P, and the in-place
// rule leaves exactly F = T[:, P] in the panel's columns once the panel is factored, so
//   rows r outside P:  A[r, c] <- A[r, c] + sum_s F[r, s] A[p_s, c]
//   rows r = p_t in P: A[r, c] <-           sum_s F[r, s] A[p_s, c]
// (writing the second case without "A[r, c] +" avoids forming T[p_t, p_t] - 1 in float).
// Per panel: (A) the panel's owners copy its columns to shared memory; (B) warp 0 alone
// factors the panel in registers (the in-place steps of k_gj_rot on B x NB values: pivot
// search by warp reductions, the pivot row by shuffles: no block barrier inside) and
// publishes F and the pivot rows; (C) every warp gathers the pivot rows' entries of its own
// columns in a warp-private buffer (no block barrier) and applies the rank-NB update,
// s = 0 .. NB-1 in order, one FMA per term.  The pivot is the lowest of the unused rows whose |a_rk| is within
// 2^-15 of the largest, a NaN before any number (piv_pack; the unblocked forms in gj_tile.cu and
// gj_cols.cu take the largest itself, a NaN last).  The summation order
// differs from the unblocked forms (results agree to float rounding, not bitwise); the
// variants with different W compute identically.  The inverse is written column-major, as
// by the other forms.
// ---- pieces shared by the blocked forms (k_gj_split, k_gj_blk) ----------------------
// Pivot key of row r: the magnitude bits of |a| without their lowest 8 (pivots within 2^-15
// relative of each other tie), then 255 - r, so that the largest key is a row of (nearly) the
// largest |a| and, among those, the lowest row; a NaN wins (the inverse of such a block is NaN).  One
// logic operation with the row's mask: 0 for a row that has been taken (or is none), so the key of every
// row left is larger.  Rows r < 128.
__device__ __forceinline__ unsigned piv_mask(int r, int B) { return r < B ? 0x7fffff00u | (unsigned)(255 - r) : 0u; }
__device__ __forceinline__ unsigned piv_pack(float x, unsigned mask) { return (__float_as_uint(x) | 0x800000ffu) & mask; }

// The in-place Gauss-Jordan steps of a panel of NB columns held by one warp (lane tx: rows
// tx + 32 i, x[i][c] for panel column c), one warp reduction per pivot: pivot rows are
// recorded in perm[k0 + s] and their steps in invk[p] = k0 + s; mask: the rows' key masks.  Bound by
// the latency of the chain pivot search, broadcast, reciprocal, update: the next column is updated and
// its pivot searched before the other columns' updates are issued, and a key is one operation.  2048
// blocks: B = 100 0.392 -> 0.354 ms, B = 75 split 0.132 -> 0.107 ms, B = 50 0.061 -> 0.053 ms.
template <int B, int RS, int NB>
__device__ __forceinline__ void gj_panel_steps(float (&x)[RS][NB], unsigned (&mask)[RS], int nb, int k0, int tx, int* perm,
                                               int* invk) {
    auto search = [&](int s) {
        unsigned km = piv_pack(x[0][s], mask[0]);
#pragma unroll
        for (int i = 1; i < RS; ++i) km = max(km, piv_pack(x[i][s], mask[i]));
        return __reduce_max_sync(0xffffffffu, km);
    };
    unsigned km = search(0);
#pragma unroll
    for (int s = 0; s < NB; ++s) {
        if (s >= nb) break;   // uniform
        const int p = 255 - (int)(km & 255u);
        const int pl = p & 31, pi = p >> 5;
        float rk[NB];
#pragma unroll
        for (int ii = 0; ii < RS; ++ii)
            if (pi == ii) {   // warp-uniform branch
                rk[s] = __shfl_sync(0xffffffffu, x[ii][s], pl);
#pragma unroll
                for (int c = 0; c < NB; ++c)
                    if (c != s) rk[c] = __shfl_sync(0xffffffffu, x[ii][c], pl);
            }
        const float inv = __frcp_rn(rk[s]);   // correctly rounded, as 1.0f / rk[s]
#pragma unroll
        for (int c = 0; c < NB; ++c) rk[c] = (c == s) ? inv : rk[c] * inv;
        float f[RS];
#pragma unroll
        for (int i = 0; i < RS; ++i) {
            f[i] = -x[i][s];
            x[i][s] = 0.0f;
            if (tx + 32 * i == p) mask[i] = 0u;
        }
        // columns c0, c0 + 1 (or the odd last one) of every row; the pivot row is scaled instead
        auto update = [&](int c0) {
#pragma unroll
            for (int i = 0; i < RS; ++i) {
                if (c0 + 1 < NB)
                    fma2f(f[i], rk[c0], rk[c0 + 1], x[i][c0], x[i][c0 + 1]);
                else
                    x[i][c0] = fmaf(f[i], rk[c0], x[i][c0]);
                if (tx + 32 * i == p) {
                    x[i][c0] = rk[c0];
                    if (c0 + 1 < NB) x[i][c0 + 1] = rk[c0 + 1];
                }
            }
        };
        const int first = s + 1 < NB ? (s + 1) / 2 * 2 : 0;
        update(first);
        if (s + 1 < NB) km = search(s + 1);
#pragma unroll
        for (int c = 0; c < NB; c += 2)
            if (c != first) update(c);
        if (tx == 0) {
            perm[k0 + s] = p;
            invk[p] = k0 + s;
        }
    }
}

// The panel's pivot rows on this warp's non-panel slots j = SPW .. CS-1 into its buffer yw
// (the row of step k0 + s at yw + s YL, 16 bytes at a time), and the factor m[i] that clears
// this lane's pivot rows (they are rebuilt from F alone): 0 for a pivot row, else 1.  Every
// lane writes its own rows at once: invk[r] is the step at which row r was chosen (-1 while
// it has not been; rows >= B never are), so the panel's pivot rows are those with
// k0 <= invk[r] < k0 + nb.
template <int RS, int CS, int SPW, int YL>
__device__ __forceinline__ void gj_gather_pivot_rows(const float (&a)[RS][CS], const int* invk, int k0, int nb,
                                                     int tx, float* yw, float (&m)[RS]) {
#pragma unroll
    for (int i = 0; i < RS; ++i) {
        const int s = invk[tx + 32 * i] - k0;
        const bool piv = (unsigned)s < (unsigned)nb;
        m[i] = piv ? 0.0f : 1.0f;
        if (piv) {
#pragma unroll
            for (int j0 = 0; j0 < CS - SPW; j0 += 4) {
                float4 v;
                v.x = a[i][SPW + j0];
                v.y = (j0 + 1 < CS - SPW) ? a[i][SPW + j0 + 1] : 0.0f;
                v.z = (j0 + 2 < CS - SPW) ? a[i][SPW + j0 + 2] : 0.0f;
                v.w = (j0 + 3 < CS - SPW) ? a[i][SPW + j0 + 3] : 0.0f;
                *reinterpret_cast<float4*>(yw + s * YL + j0) = v;
            }
        }
    }
}

// a[i][j] *= m[i] on the non-panel slots j = SPW .. CS-1, two products per instruction.
template <int RS, int CS, int SPW>
__device__ __forceinline__ void gj_clear_pivot_rows(float (&a)[RS][CS], const float (&m)[RS]) {
#pragma unroll
    for (int i = 0; i < RS; ++i) {
#pragma unroll
        for (int j = SPW; j + 1 < CS; j += 2) {
            const float2 r = __fmul2_rn(make_float2(a[i][j], a[i][j + 1]), make_float2(m[i], m[i]));
            a[i][j] = r.x;
            a[i][j + 1] = r.y;
        }
        if ((CS - SPW) % 2) a[i][CS - 1] *= m[i];
    }
}

// One step of the rank-NB update on the column slots j and j + 1 of a thread,
// a[i][j] += f[i] y0 and a[i][j + 1] += f[i] y1, for the slots in [JLO, CS) only; both slots
// in range take one paired multiply-add per row (bitwise two fmaf).
template <int RS, int CS, int JLO>
__device__ __forceinline__ void gj_update_pair(float (&a)[RS][CS], const float (&f)[RS], int j, float y0, float y1) {
    const bool in0 = j >= JLO && j < CS, in1 = j + 1 >= JLO && j + 1 < CS;
    if (in0 && in1) {
#pragma unroll
        for (int i = 0; i < RS; ++i) fma2f(f[i], y0, y1, a[i][j], a[i][j + 1]);
    } else if (in0) {
#pragma unroll
        for (int i = 0; i < RS; ++i) a[i][j] = fmaf(f[i], y0, a[i][j]);
    } else if (in1) {
#pragma unroll
        for (int i = 0; i < RS; ++i) a[i][j + 1] = fmaf(f[i], y1, a[i][j + 1]);
    }
}

template <int B, int W>
struct GjBlk {
    static constexpr int NB = 8;                        // panel width
    static constexpr int SPW = NB / W;                  // panel columns per warp and panel
    static constexpr int RS = (B + 31) / 32;            // row slots per lane
    static constexpr int R32 = 32 * RS;
    static constexpr int NP = (B + NB - 1) / NB;        // panels
    static constexpr int CS = NP * SPW;                 // column slots per thread
    static constexpr int PLD = NB + 1;                  // row stride of the panel buffers
    static constexpr int YN = CS - SPW;                 // non-panel slots per thread
    static constexpr int YL = YN > 0 ? ((YN + 3) / 4) * 4 : 4;
    static constexpr int LD = (B % 2) ? B + 2 : B + 1;  // row stride of the staging tile
    static constexpr size_t TILE = (size_t)B * LD * sizeof(float);
    static constexpr size_t WORK = (size_t)(2 * R32 * PLD + W * NB * YL) * sizeof(float);
    static constexpr size_t SMEM = ((TILE > WORK ? TILE : WORK) + 15) / 16 * 16;
    static constexpr int MAXV = W == 1 ? 128 : 64;      // values a thread holds
    static constexpr bool VALID = (NB % W == 0) && RS * CS <= MAXV && B <= 128;   // piv_pack: rows < 128
    static constexpr int MINB = RS * CS > 96 ? 10 : RS * CS > 64 ? 12 : 16 / W;
};

// The panels of one block: a[i][j] holds row tx + 32 i, column w + W j, on return the working
// matrix after all B pivots (row r: row invk[r] of the inverse, column c: its column perm[c]).
// invk is all -1 on entry.  `beside` runs once in warp 1 while warp 0 factors the first panel.
template <int B, int W, class Beside>
__device__ __forceinline__ void gj_blk_panels(float (&a)[GjBlk<B, W>::RS][GjBlk<B, W>::CS], float* Pn, float* Fs,
                                              float* yw, int* perm, int* invk, int tx, int w, Beside beside) {
    using G = GjBlk<B, W>;
    constexpr int NB = G::NB, SPW = G::SPW, RS = G::RS, NP = G::NP, CS = G::CS;
    constexpr int PLD = G::PLD, YL = G::YL;
    unsigned used[RS];   // warp 0: key masks of its rows
#pragma unroll
    for (int i = 0; i < RS; ++i) used[i] = piv_mask(tx + 32 * i, B);
#pragma unroll 1
    for (int t = 0; t < NP; ++t) {
        const int k0 = t * NB;
        const int nb = (B - k0) < NB ? (B - k0) : NB;
        __syncthreads();   // the previous panel's F and the staging tile are no longer read
        // (A) the panel's columns k0 + w + W s (slots s < SPW) to the panel buffer
#pragma unroll
        for (int s = 0; s < SPW; ++s)
#pragma unroll
            for (int i = 0; i < RS; ++i) Pn[(tx + 32 * i) * PLD + w + W * s] = a[i][s];
        __syncthreads();
        // (B) warp 0 factors the panel
        if (w == 0) {
            float x[RS][NB];
#pragma unroll
            for (int i = 0; i < RS; ++i)
#pragma unroll
                for (int c = 0; c < NB; ++c) x[i][c] = Pn[(tx + 32 * i) * PLD + c];
            gj_panel_steps<B, RS, NB>(x, used, nb, k0, tx, perm, invk);
#pragma unroll
            for (int i = 0; i < RS; ++i)
#pragma unroll
                for (int c = 0; c < NB; ++c) Fs[(tx + 32 * i) * PLD + c] = x[i][c];
        } else if (w == 1 && t == 0) {
            beside();
        }
        __syncthreads();
        // (C) pivot rows of this warp's non-panel columns into the warp's buffer; the pivot
        // rows' own entries are then cleared (they are rebuilt from F alone)
        __syncwarp();
        float mrow[RS];
        gj_gather_pivot_rows<RS, CS, SPW, YL>(a, invk, k0, nb, tx, yw, mrow);
        __syncwarp();
        gj_clear_pivot_rows<RS, CS, SPW>(a, mrow);
#pragma unroll
        for (int s = 0; s < NB; ++s) {
            if (s >= nb) break;   // uniform
            float f[RS];
#pragma unroll
            for (int i = 0; i < RS; ++i) f[i] = Fs[(tx + 32 * i) * PLD + s];
            const float* yr = yw + s * YL;
#pragma unroll
            for (int j0 = 0; j0 < CS - SPW; j0 += 4) {
                const float4 y4 = *reinterpret_cast<const float4*>(yr + j0);
                const float yv[4] = {y4.x, y4.y, y4.z, y4.w};
#pragma unroll
                for (int q = 0; q < 4; q += 2) gj_update_pair<RS, CS, SPW>(a, f, SPW + j0 + q, yv[q], yv[q + 1]);
            }
        }
        // the panel's own columns become F
#pragma unroll
        for (int s = 0; s < SPW; ++s)
#pragma unroll
            for (int i = 0; i < RS; ++i) a[i][s] = Fs[(tx + 32 * i) * PLD + w + W * s];
        // rotate the column slots by SPW: the next panel's columns move to slots 0 .. SPW-1
#pragma unroll
        for (int i = 0; i < RS; ++i) {
            float t0[SPW];
#pragma unroll
            for (int s = 0; s < SPW; ++s) t0[s] = a[i][s];
#pragma unroll
            for (int j = 0; j < CS - SPW; ++j) a[i][j] = a[i][j + SPW];
#pragma unroll
            for (int s = 0; s < SPW; ++s) a[i][CS - SPW + s] = t0[s];
        }
    }
    // NP rotations by SPW = CS slots: every column is back in its own slot
}

// Every block of the level (list = nullptr, one CTA each), or the blocks that k_gj_split left (list;
// a few CTAs share them).
template <int B, int W>
__global__ void __launch_bounds__(32 * W, GjBlk<B, W>::MINB) k_gj_blk(int E, float* __restrict__ blk, const int* __restrict__ list,
                                                           int* __restrict__ head) {
    using G = GjBlk<B, W>;
    constexpr int RS = G::RS, R32 = G::R32, CS = G::CS, LD = G::LD, T = 32 * W;
    extern __shared__ __align__(16) unsigned char smraw[];
    float* tile = reinterpret_cast<float*>(smraw);      // staging (load and store only)
    float* Pn = tile;                                   // panel columns [R32][PLD]
    float* Fs = tile + R32 * G::PLD;                    // factored panel F [R32][PLD]
    float* Yw = tile + 2 * R32 * G::PLD;                // pivot rows, per warp [W][NB][YL]
    __shared__ int perm[B], invk[R32];
    const int tx = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int n = list ? take_list(head) : E;
#pragma unroll 1
    for (int it = blockIdx.x; it < n; it += gridDim.x) {
        float* g = blk + (size_t)(list ? list[it] : it) * B * B;
        __syncthreads();
        for (int t = threadIdx.x; t < R32; t += T) invk[t] = -1;
        for (int t = threadIdx.x; t < B * B; t += T) tile[(t / B) * LD + (t % B)] = g[t];
        __syncthreads();
        float a[RS][CS];
#pragma unroll
        for (int i = 0; i < RS; ++i)
#pragma unroll
            for (int j = 0; j < CS; ++j) {
                const int r = tx + 32 * i, c = w + W * j;
                a[i][j] = (r < B && c < B) ? tile[r * LD + c] : 0.0f;
            }
        gj_blk_panels<B, W>(a, Pn, Fs, Yw + (size_t)w * G::NB * G::YL, perm, invk, tx, w, []() {});
        __syncthreads();
#pragma unroll
        for (int i = 0; i < RS; ++i)
#pragma unroll
            for (int j = 0; j < CS; ++j) {
                const int r = tx + 32 * i, c = w + W * j;
                if (r < B && c < B) tile[perm[c] * LD + invk[r]] = a[i][j];
            }
        __syncthreads();
        for (int t = threadIdx.x; t < B * B; t += T) g[t] = tile[(t / B) * LD + (t % B)];
    }
}

// 2-D levels: a block whose spanwise momentum (variable 3) is coupled to no other variable (flow in
// the plane) splits into systems of 4 N and N unknowns, whose inverses leave packed (blocks.cuh):
// 0.53 of the multiply-adds and 0.68 of the bytes of the whole block's, and 4 N in place of 5 N
// pivots in the chain that bounds the kernel (warp 1 inverts the N x N system while warp 0 factors the
// first panel).  2048 blocks at N = 15: 0.153 ms whole, 0.107 split.  Blocks come packed from the plane assembly (asm_flag) or whole; one that is coupled is
// left as it is and put on the list for k_gj_blk.
template <int N, int W>
struct GjSplit {
    using G = GjBlk<4 * N, W>;
    static constexpr int B4 = 4 * N, LD = B4 + 1;
    static constexpr size_t TILE = (size_t)(B4 * LD + N * N) * sizeof(float);
    static constexpr size_t WORK = G::WORK + (size_t)N * N * sizeof(float);
    static constexpr size_t SMEM = ((TILE > WORK ? TILE : WORK) + 15) / 16 * 16;
    static constexpr bool VALID = G::VALID;
    static constexpr int MINB = W > 1 && G::RS * G::CS <= 32 ? 28 / W : G::MINB;
};

template <int N, int W>
__global__ void __launch_bounds__(32 * W, GjSplit<N, W>::MINB) k_gj_split(
    int E, float* __restrict__ blk, const int* __restrict__ asm_flag, int* __restrict__ flag, int* __restrict__ list,
    int* __restrict__ head) {
    using S = GjSplit<N, W>;
    using G = typename S::G;
    constexpr int B = 5 * N, B4 = 4 * N, LD = S::LD, RS = G::RS, R32 = G::R32, CS = G::CS, T = 32 * W;
    extern __shared__ __align__(16) unsigned char smraw[];
    float* s3 = reinterpret_cast<float*>(smraw);        // the spanwise block [N][N]
    float* tile = s3 + N * N;                           // the other variables' (load and store only)
    float* Yw = reinterpret_cast<float*>(smraw) + (N * N + 3) / 4 * 4;   // pivot rows, per warp [W][NB][YL]
    float* Pn = Yw + W * G::NB * G::YL;                 // panel columns [R32][PLD]
    float* Fs = Pn + R32 * G::PLD;                      // factored panel F [R32][PLD]
    __shared__ int perm[B4], invk[R32], perm3[N], invk3[32];
    const int tx = threadIdx.x & 31, w = threadIdx.x >> 5, e = blockIdx.x;
    float* g = blk + (size_t)e * B * B;
    for (int t = threadIdx.x; t < R32; t += T) invk[t] = -1;
    if (threadIdx.x < 32) invk3[threadIdx.x] = -1;
    float* out = blk + gj_packed_at(e, B);
    bool coupled = false;
    if (asm_flag && !asm_flag[e]) {   // left whole by the assembly, which found it coupled
        coupled = true;
    } else if (asm_flag) {
#pragma unroll 8
        for (int t = threadIdx.x; t < B4 * B4; t += T) tile[t / B4 * LD + t % B4] = out[t];
        for (int t = threadIdx.x; t < N * N; t += T) s3[t] = out[B4 * B4 + t];
    } else {
#pragma unroll 4
        for (int t = threadIdx.x; t < B * B; t += T) {
            const int r = t / B, c = t - r * B;
            const float v = g[t];
            const int rs = r / N, cs = c / N;
            if (rs != 3 && cs != 3)
                tile[(rs == 4 ? r - N : r) * LD + (cs == 4 ? c - N : c)] = v;
            else if (rs == cs)
                s3[(r - 3 * N) * N + c - 3 * N] = v;
            else
                coupled |= !(v == 0.0f);
        }
    }
    coupled = __syncthreads_or(coupled);
    if (threadIdx.x == 0) {
        flag[e] = !coupled;
        if (coupled) list[atomicAdd(head, 1)] = e;
    }
    if (coupled) return;
    auto spanwise = [&]() {
        float x[1][N];
#pragma unroll
        for (int c = 0; c < N; ++c) x[0][c] = tx < N ? s3[tx * N + c] : 0.0f;
        unsigned used[1] = {piv_mask(tx, N)};
        gj_panel_steps<N, 1, N>(x, used, N, 0, tx, perm3, invk3);
        __syncwarp();
        if (tx < N)
#pragma unroll
            for (int c = 0; c < N; ++c) out[B4 * B4 + perm3[c] * N + invk3[tx]] = x[0][c];
    };
    if (W == 1) spanwise();
    float a[RS][CS];
#pragma unroll
    for (int i = 0; i < RS; ++i)
#pragma unroll
        for (int j = 0; j < CS; ++j) {
            const int r = tx + 32 * i, c = w + W * j;
            a[i][j] = (r < B4 && c < B4) ? tile[r * LD + c] : 0.0f;
        }
    gj_blk_panels<B4, W>(a, Pn, Fs, Yw + (size_t)w * G::NB * G::YL, perm, invk, tx, w, spanwise);
    __syncthreads();
#pragma unroll
    for (int i = 0; i < RS; ++i)
#pragma unroll
        for (int j = 0; j < CS; ++j) {
            const int r = tx + 32 * i, c = w + W * j;
            if (r < B4 && c < B4) tile[perm[c] * LD + invk[r]] = a[i][j];
        }
    __syncthreads();
    for (int t = threadIdx.x; t < B4 * B4; t += T) out[t] = tile[(t / B4) * LD + (t % B4)];
}

// ---- variants of the FP32 Gauss-Jordan kernel and their tuning --------------------------------
// Two families.  Unblocked (variants 0..13): variant v < 4 unrolls the pivot loop kGjUnroll[v]
// times (0 = fully, only for B <= 100); 4..8 are the column-owner form with kGjWarps[v - 4]
// warps per element (valid while a thread's share of the block stays at most 128 values);
// 9..13 the rotating column-owner form with kGjWarps[v - 9] warps.  Blocked (14..17):
// k_gj_blk with kGjBlkWarps[v - 14] warps (valid while a thread holds at most 64 values, 128 with one warp).
// The split form of 2-D levels is a family of its own, timed on whole or on packed blocks.
// Within a family the variants do the same arithmetic in the same order, so the tuner's choice
// never changes a result; the tuner times one family only (the blocked one where it is valid,
// unless emg_params.block_kernels asks for the unblocked forms).
constexpr int kGjUnroll[] = {1, 4, 16, 0};
constexpr int kGjWarps[] = {1, 2, 4, 8, 16};
constexpr int kGjBlkWarps[] = {1, 2, 4, 8};
constexpr int kGjBlkFirst = 14;
constexpr int kGjVariants = 18;

template <int B, int W>
constexpr bool gj_blk_valid() {
    return GjBlk<B, W>::VALID;
}

template <int B>
static bool gj_variant_valid(int v) {
    if (v < 0 || v >= kGjVariants) return false;
    if (v < 4) return kGjUnroll[v] != 0 || B <= 100;
    if (v >= kGjBlkFirst) {
        switch (kGjBlkWarps[v - kGjBlkFirst]) {
            case 1: return gj_blk_valid<B, 1>();
            case 2: return gj_blk_valid<B, 2>();
            case 4: return gj_blk_valid<B, 4>();
            default: return gj_blk_valid<B, 8>();
        }
    }
    const int W = kGjWarps[(v - 4) % 5];
    return ((B + 31) / 32) * ((B + W - 1) / W) <= 128;
}

static std::string gj_variant_name(int v) {
    if (v < 4) return "tile unroll " + std::to_string(kGjUnroll[v]);
    if (v >= kGjBlkFirst) return "blocked " + std::to_string(kGjBlkWarps[v - kGjBlkFirst]) + " warps";
    return std::string(v < 9 ? "cols " : "rotating cols ") + std::to_string(kGjWarps[(v - 4) % 5]) + " warps";
}

template <int B, int W>
static cudaError_t gj_blk_go(unsigned E, float* blk, cudaStream_t st) {
    if constexpr (GjBlk<B, W>::VALID) {
        const size_t sm = GjBlk<B, W>::SMEM;
        cudaError_t e = cudaFuncSetAttribute(k_gj_blk<B, W>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        if (e != cudaSuccess) return e;
        k_gj_blk<B, W><<<E, 32 * W, sm, st>>>((int)E, blk, nullptr, nullptr);
        return cudaGetLastError();
    } else {
        return cudaErrorInvalidValue;   // not reached: gj_dispatch checks the variant first
    }
}

// The split form of a 2-D level: kGjBlkWarps[v] warps per element, then the blocks it left (none in
// plane flow: a few CTAs look at the list's length and end).
template <int N, int W>
static cudaError_t gj_split_go(unsigned E, float* blk, const GjWork& k, bool packed, cudaStream_t st) {
    if constexpr (GjSplit<N, W>::VALID) {
        const size_t sm = GjSplit<N, W>::SMEM;
        cudaError_t e = cudaFuncSetAttribute(k_gj_split<N, W>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        if (e != cudaSuccess) return e;
        k_gj_split<N, W><<<E, 32 * W, sm, st>>>((int)E, blk, packed ? k.asm_flag : nullptr, k.flag, k.list, k.head);
        return cudaGetLastError();
    } else {
        return cudaErrorInvalidValue;   // not reached: gj_split_valid
    }
}
template <int N>
static bool gj_split_valid(int v) {
    return v == 0 ? GjSplit<N, 1>::VALID : v == 1 ? GjSplit<N, 2>::VALID : v == 2 ? GjSplit<N, 4>::VALID : GjSplit<N, 8>::VALID;
}
template <int N>
static cudaError_t gj_split_launch(int v, unsigned E, float* blk, const GjWork& k, bool packed, cudaStream_t st) {
    cudaError_t e = v == 0   ? gj_split_go<N, 1>(E, blk, k, packed, st)
                    : v == 1 ? gj_split_go<N, 2>(E, blk, k, packed, st)
                    : v == 2 ? gj_split_go<N, 4>(E, blk, k, packed, st)
                             : gj_split_go<N, 8>(E, blk, k, packed, st);
    if (e != cudaSuccess) return e;
    using G = GjBlk<5 * N, 4>;
    static_assert(G::VALID, "the blocked form serves every 2-D block");
    e = cudaFuncSetAttribute(k_gj_blk<5 * N, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G::SMEM);
    if (e != cudaSuccess) return e;
    k_gj_blk<5 * N, 4><<<list_grid(E, 128), 128, G::SMEM, st>>>((int)E, blk, k.list, k.head);
    return cudaGetLastError();
}
// packed: the blocks come from the plane assembly.
static cudaError_t gj_split_dispatch(int B, int v, unsigned E, float* blk, int* work, bool packed, cudaStream_t st) {
    const GjWork k = gj_work(work, E);
    switch (B) {
        case 15: return gj_split_launch<3>(v, E, blk, k, packed, st);
        case 30: return gj_split_launch<6>(v, E, blk, k, packed, st);
        case 50: return gj_split_launch<10>(v, E, blk, k, packed, st);
        default: return gj_split_launch<15>(v, E, blk, k, packed, st);
    }
}
static bool gj_split_ok(int B, int v) {
    return B == 15 ? gj_split_valid<3>(v) : B == 30 ? gj_split_valid<6>(v) : B == 50 ? gj_split_valid<10>(v) : gj_split_valid<15>(v);
}

template <int B>
static cudaError_t gj_launch(int v, unsigned E, float* blk, cudaStream_t st) {
    switch (v) {
        case 14: return gj_blk_go<B, 1>(E, blk, st);
        case 15: return gj_blk_go<B, 2>(E, blk, st);
        case 16: return gj_blk_go<B, 4>(E, blk, st);
        case 17: return gj_blk_go<B, 8>(E, blk, st);
        case 9: return gj_rot_go<B, 1>(E, blk, st);
        case 10: return gj_rot_go<B, 2>(E, blk, st);
        case 11: return gj_rot_go<B, 4>(E, blk, st);
        case 12: return gj_rot_go<B, 8>(E, blk, st);
        case 13: return gj_rot_go<B, 16>(E, blk, st);
        case 4: return gj_cols_go<B, 1>(E, blk, st);
        case 5: return gj_cols_go<B, 2>(E, blk, st);
        case 6: return gj_cols_go<B, 4>(E, blk, st);
        case 7: return gj_cols_go<B, 8>(E, blk, st);
        case 8: return gj_cols_go<B, 16>(E, blk, st);
        case 1: return gj_go<B, 4>(E, blk, st);
        case 2: return gj_go<B, 16>(E, blk, st);
        case 3: return gj_go<B, (B <= 100 ? B : 1)>(E, blk, st);
        default: return gj_go<B, 1>(E, blk, st);
    }
}

static cudaError_t gj_dispatch(int B, int v, unsigned E, float* blk, cudaStream_t st, bool* ok) {
    *ok = true;
    switch (B) {
#define EMG_GJ_CASE(BB) \
    case BB:            \
        return gj_variant_valid<BB>(v) ? gj_launch<BB>(v, E, blk, st) : gj_launch<BB>(0, E, blk, st);
        EMG_BSIZES(EMG_GJ_CASE)
#undef EMG_GJ_CASE
        default:
            *ok = false;
            return cudaSuccess;
    }
}

static bool gj_valid(int B, int v) {
    switch (B) {
#define EMG_GJ_CASE(BB) \
    case BB:            \
        return gj_variant_valid<BB>(v);
        EMG_BSIZES(EMG_GJ_CASE)
#undef EMG_GJ_CASE
        default:
            return false;
    }
}

// Deterministic, diagonally dominant stand-in blocks for timing the variants.
// split: the spanwise momentum's rows and columns coupled to nothing, as in plane flow.
__global__ void k_fill_tuning_blocks(int64_t n, int B, bool split, float* __restrict__ blk) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n * B * B) return;
    const int c = (int)(t % B), r = (int)((t / B) % B);
    const uint32_t h = (uint32_t)(t * 2654435761ull) ^ (uint32_t)(t >> 13);
    const bool zero = split && (r / (B / 5) == 3) != (c / (B / 5) == 3);
    blk[t] = zero ? 0.0f : (r == c ? (float)B : 0.0f) + ((float)(h & 0xffffu) / 65536.0f - 0.5f);
}
// The same, packed as the plane assembly leaves them (blocks.cuh).
__global__ void k_fill_tuning_packed(int64_t n, int N, float* __restrict__ blk) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int B4 = 4 * N, len = 17 * N * N;
    if (t >= n * len) return;
    const int o = (int)(t % len), m = o < B4 * B4 ? B4 : N, q = o < B4 * B4 ? o : o - B4 * B4;
    const uint32_t h = (uint32_t)(t * 2654435761ull) ^ (uint32_t)(t >> 13);
    blk[gj_packed_at(t / len, 5 * N) + o] = (q / m == q % m ? 5.0f * N : 0.0f) + ((float)(h & 0xffffu) / 65536.0f - 0.5f);
}

namespace {
std::mutex g_tune_mu;
std::map<std::tuple<int, int, int, int>, int> g_gj_best;   // (device, B, family, log2 of the stand-ins) -> variant
}  // namespace

// Times every valid variant per block size of the FP32 levels on as many stand-in blocks as the level
// has, at most 2048 (32 MB of small ones), packed where the level's own come packed from the assembly, and
// keeps the fastest, once per (device, B, family, power of two of their number) for the process.  Whole
// stand-ins in the place of packed ones chose other variants (128 x 64, p = 4: a smoothing step 1030 us, now
// 946), and so did 512 blocks of B = 15 for 8192 (p = 1: 322 us with 8 warps, 303 with 4).
emg_status tune_gj(emg_ctx* c) {
    if (!blocks_f32(c->prm.prec)) return EMG_OK;
    std::lock_guard<std::mutex> lk(g_tune_mu);
    for (int p = 1; p <= c->p_max; ++p) {
        LevelDev& L = c->lv[p];
        // the split form serves 2-D levels unless the tensor-core or unblocked forms are asked for
        L.gj_split = c->dim == 2 && !L.tc_gj && c->prm.block_kernels != 3;
        L.asm_plane = L.gj_split && !L.tc_asm && !c->rot;
        const bool packed = L.asm_plane;
        const int64_t n = std::min<int64_t>(c->E, std::max(2048, (8 << 20) / (L.B * L.B)));
        int class_n = 0;
        while (n >> (class_n + 1)) ++class_n;
        const auto key = std::make_tuple(c->device, L.B, packed ? 3 : L.gj_split ? 2 : (int)(c->prm.block_kernels == 3), class_n);
        if (L.gj_split)   // the list's length and ticket (piv holds the FP64 form's pivots only)
            EMG_CUDA_TRY(c, cudaMemsetAsync(L.piv, 0, (size_t)c->E * L.B * sizeof(int), c->stream));
        // the family: blocked where a blocked variant is valid (unless the unblocked forms are
        // asked for), else unblocked
        bool blocked = false;
        if (c->prm.block_kernels != 3)
            for (int v = kGjBlkFirst; v < kGjVariants; ++v) blocked = blocked || gj_valid(L.B, v);
        const int v_lo = blocked && !L.gj_split ? kGjBlkFirst : 0;
        const int v_hi = L.gj_split ? 4 : blocked ? kGjVariants : kGjBlkFirst;   // 0..3 / 14..17 / 0..13
        auto valid = [&](int v) { return L.gj_split ? gj_split_ok(L.B, v) : gj_valid(L.B, v); };
        auto name = [&](int v) {
            return L.gj_split ? (packed ? "packed split " : "split ") + std::to_string(kGjBlkWarps[v]) + " warps"
                              : gj_variant_name(v);
        };
        if (!c->prm.autotune) {
            L.gj_variant = 0;
            for (int v = v_lo; v < v_hi; ++v)
                if (valid(v)) {
                    L.gj_variant = v;
                    break;
                }
            continue;
        }
        if (L.tc_gj) {
            c->tuning += "gj B=" + std::to_string(L.B) + ": blocked tensor-core form (not tuned); ";
            continue;
        }
        auto it = g_gj_best.find(key);
        if (it != g_gj_best.end()) {
            L.gj_variant = it->second;
            c->tuning += "gj B=" + std::to_string(L.B) + ": " + name(it->second) +
                         " (tuned earlier in this process); ";
            continue;
        }
        float* scratch = nullptr;
        EMG_CUDA_TRY(c, cudaMallocAsync((void**)&scratch, (size_t)n * L.B * L.B * sizeof(float), c->stream));
        auto fill = [&]() {
            if (packed)
                k_fill_tuning_packed<<<(unsigned)((n * 17 * L.N * L.N + 255) / 256), 256, 0, c->stream>>>(n, L.N, scratch);
            else
                k_fill_tuning_blocks<<<(unsigned)((n * L.B * L.B + 255) / 256), 256, 0, c->stream>>>(n, L.B, L.gj_split, scratch);
        };
        fill();
        if (packed) EMG_CUDA_TRY(c, cudaMemsetAsync(gj_work(L.piv, n).asm_flag, 1, n * sizeof(int), c->stream));
        cudaEvent_t e0, e1;
        EMG_CUDA_TRY(c, cudaEventCreate(&e0));
        EMG_CUDA_TRY(c, cudaEventCreate(&e1));
        int best = v_lo;
        float best_ms = 1e30f;
        std::string note = "gj B=" + std::to_string(L.B) + ":";
        for (int v = v_lo; v < v_hi; ++v) {
            if (!valid(v)) continue;
            bool ok = true;
            float ms = 1e30f;
            for (int rep = 0; rep < 3 && ok; ++rep) {
                if (L.gj_split)   // the inverses left packed are no split blocks
                    fill();
                EMG_CUDA_TRY(c, cudaEventRecord(e0, c->stream));
                if (L.gj_split)
                    EMG_CUDA_TRY(c, gj_split_dispatch(L.B, v, (unsigned)n, scratch, L.piv, packed, c->stream));
                else
                    EMG_CUDA_TRY(c, gj_dispatch(L.B, v, (unsigned)n, scratch, c->stream, &ok));
                EMG_CUDA_TRY(c, cudaEventRecord(e1, c->stream));
                EMG_CUDA_TRY(c, cudaEventSynchronize(e1));
                float t = 0.0f;
                EMG_CUDA_TRY(c, cudaEventElapsedTime(&t, e0, e1));
                if (rep > 0) ms = std::min(ms, t);   // the first run warms up
            }
            char buf[64];
            std::snprintf(buf, sizeof(buf), " %.3f ms, ", ms);
            note += " " + name(v) + buf;
            if (ms < best_ms) {
                best_ms = ms;
                best = v;
            }
        }
        cudaEventDestroy(e0);
        cudaEventDestroy(e1);
        EMG_CUDA_TRY(c, cudaFreeAsync(scratch, c->stream));
        if (L.gj_split) EMG_CUDA_TRY(c, cudaMemsetAsync(L.piv, 0, (size_t)c->E * L.B * sizeof(int), c->stream));
        g_gj_best[key] = best;
        L.gj_variant = best;
        c->tuning += note + "-> " + name(best) + "; ";
    }
    return EMG_OK;
}

emg_status launch_lu32(emg_ctx* c, int p) {
    LevelDev& L = c->lv[p];
    if (L.tc_gj) {
        bool built = false;
        const emg_status st = launch_gj_tc(c, L.B, L.blk32, &built);
        if (built) return st;
    }
    bool ok = true;
    {
        ProfScope _ps(c, PC_LU);
        if (L.gj_split) {
            EMG_CUDA_TRY(c, gj_split_dispatch(L.B, L.gj_variant, (unsigned)c->E, L.blk32, L.piv, L.asm_plane, c->stream));
            ++c->launches;   // two kernels, one counted below
            EMG_CHECK_LAUNCH(c);
            return EMG_OK;
        }
        EMG_CUDA_TRY(c, gj_dispatch(L.B, L.gj_variant, (unsigned)c->E, L.blk32, c->stream, &ok));
    }
    if (!ok) {
        c->err = "unsupported block size";
        return EMG_ERR_ARG;
    }
    return EMG_OK;
}

}  // namespace emg
