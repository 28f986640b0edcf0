// Shared pieces of the block factorisations (LU of the FP64 form, Gauss-Jordan inverses of
// the float32 forms): the pivot key and the list of block sizes B = 5 N the levels use.
#pragma once

#include <cstdint>

namespace emg {

// Pivot magnitude as an ordered integer key: the IEEE bits of |x| order like its value for
// every finite or infinite x; a NaN gets -1, so it never wins against a number.  Comparing
// keys as integers keeps the pivot search deterministic and independent of how the compiler
// treats float comparisons with NaN (where every thread of a warp computes the pivot on its
// own, a disagreement would break the permutation).
__device__ __forceinline__ int piv_key(float x) {
    const unsigned b = __float_as_uint(x) & 0x7fffffffu;
    return b <= 0x7f800000u ? (int)b : -1;
}
__device__ __forceinline__ long long piv_key(double x) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
    return b <= 0x7ff0000000000000ull ? (long long)b : -1ll;
}

// Two fused multiply-adds d_k <- a b_k + d_k (k = 0, 1) issued as one paired float32
// instruction; each component is rounded as by fmaf, so the results are bitwise those of two
// fmaf calls and only the instruction count changes.
__device__ __forceinline__ void fma2f(float a, float b0, float b1, float& d0, float& d1) {
    const float2 r = __ffma2_rn(make_float2(a, a), make_float2(b0, b1), make_float2(d0, d1));
    d0 = r.x;
    d1 = r.y;
}

// Where the packed form of element e starts (floats, 16-byte aligned, within the element's B x B
// place), for blocks that split only (gj.cu): the 4 N x 4 N system over variables 0, 1, 2, 4, then the
// N x N one of variable 3, row-major from the assembly (jac_plane.cu), column-major once inverted.
__host__ __device__ __forceinline__ size_t gj_packed_at(int64_t e, int B) { return ((size_t)e * B * B + 3) & ~(size_t)3; }

// Work space of the split float32 blocks of a 2-D level, in the E x B integers of LevelDev::piv (B >=
// 15): flags of the packed blocks and list of the others, of the assembly and of the inverse.  head: the
// list's length and a ticket.
struct GjWork {
    int *flag, *list, *head, *asm_flag, *asm_list, *asm_head;
};
inline GjWork gj_work(int* w, int64_t E) { return {w, w + E, w + 4 * E, w + 2 * E, w + 3 * E, w + 4 * E + 2}; }

// Length of a list, read by every CTA of a grid; the last one out sets it back to 0 (an empty one is 0).
__device__ __forceinline__ int take_list(int* head) {
    const int n = *reinterpret_cast<volatile int*>(head);
    __syncthreads();   // every thread has read it
    if (n > 0 && threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(head + 1, 1) == (int)gridDim.x - 1) {   // every CTA has
            head[0] = 0;
            head[1] = 0;
        }
    }
    return n;
}
// CTAs that share a list: enough for 32 warps an SM (four CTAs at least, 16 at most), so that a level whose
// blocks are all listed (a 2-D flow with a spanwise momentum) fills the chip.  Smoothing step of 128 x 64,
// float32 blocks, all listed, with 4 CTAs an SM / as here: p = 1 470 / 375 us, p = 2 629 / 530 us; none
// listed 321 / 322 us and 379 / 382 us.
inline unsigned list_grid(int64_t E, int threads) {
    const int64_t per_sm = threads >= 256 ? 4 : threads <= 64 ? 16 : 1024 / threads, n = 152 * per_sm;
    return (unsigned)(E < n ? E : n);
}

// B = 5 N(p): 2-D p = 1..4, then 3-D p = 1..4 (B = 50 serves both dimensions).
#define EMG_BSIZES(X) X(15) X(30) X(50) X(75) X(20) X(100) X(175)

}  // namespace emg
