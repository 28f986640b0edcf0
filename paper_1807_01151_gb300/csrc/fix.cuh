// Float64 dot products on the integer pipe.  GB300 issues 2 float64 multiply-adds per clock and
// SM, but more than 40 32 x 32 -> 64 bit integer ones, so the residual's contractions (traces,
// volume quadrature, projections) take their factors as fixed-point numbers of 56 bits and sign:
//   x = v 2^-s,  v = hi 2^28 + lo,  |v| < 2^56,  -2^27 <= lo < 2^27,
// one exponent s for each group of factors that is summed over, taken from the group's largest
// magnitude: an element's basis values; its weighted gradients of one mode in one direction; its
// coefficients of one variable; its point fluxes of one variable in one direction; a face's fluxes of
// one variable.  Three multiply-adds per term keep the exact sums
//   h = sum hi hi',  x = sum (hi lo' + lo hi')
// and the result is (h 2^56 + x 2^28) 2^(-s-s'); the terms lo lo' (below 2^-58 of the largest
// term) are left out.  With at most FIX_TERMS = 120 terms neither sum can overflow:
// |h|, |x| <= 120 2^56 < 2^63.  A float64 multiply-add chain rounds at 2^-54 of the running sum at
// every term; here a factor is off by 2^-56 of its group's largest (tables, rounded: 2^-57), however
// small it is itself, so a sum is as good as float64's only if its own terms are not small against
// (largest factor) (largest factor) of its two groups.  Hence the groups above: with one exponent for
// all gradients of an element, rows along the long side of a stretched cell kept fewer bits than
// float64 gave them.  Error of a mode's volume sum over its own sum of |terms|, worst and rms over modes
// and elements in units of 2^-53, CPU emulation against 64-bit mantissas (float64 / one exponent an
// element / these groups): rectangles of aspect 100, p = 4: 5.3, 0.98 / 184000, 9300 / 2.1, 0.35; 128 x 8
// O-grid, p = 3: 12, 1.2 / 2400, 62 / 2.1, 0.40; sphere shell of 12 hexes a patch, p = 3: 20, 3.0 /
// 3600, 157 / 2.4, 0.42.  Traces (K <= 35 terms, dominated by the mean) of the 24 x 12 O-grid, p = 4: 7.3,
// 1.4 / 5.8, 1.0.
// A group that holds an infinity or a NaN gets the scale NaN, so every sum over it is NaN.
#pragma once

#include "common.cuh"

namespace emg {

constexpr int FIX_LO = 28;      // bits of the low half
constexpr int FIX_BITS = 56;    // |v| < 2^FIX_BITS
constexpr int FIX_TERMS = 120;  // most terms of one sum

// Magnitude key of x: its high word without the sign (orders like |x| up to the low word).
__device__ __forceinline__ int fix_key(double x) { return __double2hiint(x) & 0x7fffffff; }

// Exponent s of a group whose largest key is `key`: |x| 2^s < 2^56 for every member.  Groups below
// 2^-900 share the exponent of 2^-900 (their members become small integers or 0).
__device__ __forceinline__ int fix_exp(int key) {
    const int f = key >> 20;
    return FIX_BITS + 1022 - (f < 123 ? 123 : f);
}

// 2^e as a double, NaN where the group's key is not that of a finite number.
__device__ __forceinline__ double fix_scale(int e, int key) {
    const int b = 1023 + e;
    const double s = b >= 2047 ? __hiloint2double(0x7ff00000, 0) : b <= 0 ? 0.0 : __hiloint2double(b << 20, 0);
    return key >= 0x7ff00000 ? __hiloint2double(0x7ff80000, 0) : s;
}

// A number v as (hi, lo).
__device__ __forceinline__ int2 fix_pair(long long v) {
    return make_int2((int)((v + (1ll << (FIX_LO - 1))) >> FIX_LO), ((int)v << (32 - FIX_LO)) >> (32 - FIX_LO));
}

// The same with FIX_NAN in the place of an exponent for a group that holds an infinity or a NaN (e is
// then above any number's).
constexpr int FIX_NAN = -100000;
__device__ __forceinline__ double fix_scale(int e) {
    const int b = 1023 + e;
    return b >= 2047 ? __hiloint2double(b > 50000 ? 0x7ff80000 : 0x7ff00000, 0) : b <= 0 ? 0.0 : __hiloint2double(b << 20, 0);
}

// v = x 2^s cut to an integer, as (hi, lo); |x| 2^s < 2^56.
__device__ __forceinline__ int2 fix_of(double x, int s) {
    const int hw = __double2hiint(x);
    const int sh = 1078 - s - ((hw >> 20) & 0x7ff);   // |v| = (mantissa 2^3) >> sh, sh >= 0
    const unsigned long long m =
        (((unsigned long long)((hw & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(x)) << 3;
    const unsigned long long a = sh > 63 ? 0ull : m >> sh;
    return fix_pair(hw < 0 ? -(long long)a : (long long)a);
}

// The same rounded to the nearest integer (2^56 at most): for the tables, at set-up.
__device__ __forceinline__ int2 fix_round(double x, int s) {
    const int hw = __double2hiint(x);
    const int sh = 1078 - s - ((hw >> 20) & 0x7ff);
    const unsigned long long m =
        (((unsigned long long)((hw & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(x)) << 4;
    const unsigned long long a = sh > 63 ? 0ull : ((m >> sh) + 1) >> 1;
    return fix_pair(hw < 0 ? -(long long)a : (long long)a);
}

// (hi, lo) of v 2^-k, k >= 0, negated where neg is set.
__device__ __forceinline__ int2 fix_shift(int2 p, int k, bool neg) {
    long long v = ((long long)p.x << FIX_LO) + (long long)p.y;
    v >>= k > 63 ? 63 : k;
    if (neg) v = -v;
    return fix_pair(v);
}

// (hi, lo) of v 2^-k rounded, k >= 0.
__device__ __forceinline__ int2 fix_shift_round(int2 p, int k) {
    const long long v = ((long long)p.x << FIX_LO) + (long long)p.y;
    return fix_pair(k == 0 ? v : ((v >> min(k - 1, 62)) + 1) >> 1);
}

// v as a double (v 2^-s is the number it stands for).
__device__ __forceinline__ double fix_back(int2 v) {
    return __ll2double_rn(((long long)v.x << FIX_LO) + (long long)v.y);
}

// In PTX: from the C++ form the compiler makes 64 x 64 bit products where a factor was split from a
// 64-bit value in registers (measured: 6 instructions in place of each).
__device__ __forceinline__ void fix_mad(long long& h, int a, int b) {
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(h) : "r"(a), "r"(b));
}
__device__ __forceinline__ void fix_mac(long long& h, long long& x, int2 a, int2 b) {
    fix_mad(h, a.x, b.x);
    fix_mad(x, a.x, b.y);
    fix_mad(x, a.y, b.x);
}

// The sum as a double; scale = 2^(56 - s - s').
__device__ __forceinline__ double fix_sum(long long h, long long x, double scale) {
    return __ll2double_rn(h + ((x + (1ll << (FIX_LO - 1))) >> FIX_LO)) * scale;
}

// Layout of the projections' tables: rows (points) of N modes, two consecutive rows interleaved,
// [R / 2][N][2] (an odd last row follows alone), so that a thread, which owns a mode, takes two rows
// with one 16-byte load.  Face tables whose sides would not start on 16 bytes stay [QF][N].
template <int N, int ROWS, bool PAIRED>
struct RowTab {
    static constexpr bool paired = PAIRED;
    __host__ __device__ static constexpr int at(int r, int i) {
        return !PAIRED || r >= (ROWS & ~1) ? r * N + i : ((r >> 1) * N + i) * 2 + (r & 1);
    }
    __host__ __device__ static constexpr int row(int o) {
        return !PAIRED || o >= (ROWS & ~1) * N ? o / N : o / (2 * N) * 2 + (o & 1);
    }
    __host__ __device__ static constexpr int mode(int o) {
        return !PAIRED || o >= (ROWS & ~1) * N ? o % N : (o % (2 * N)) >> 1;
    }
};
template <int D, int P>
using FaceTab = RowTab<Lv<D, P>::N, Lv<D, P>::QF, (Lv<D, P>::QF * Lv<D, P>::N) % 2 == 0>;
// weighted gradients: row q D + k of element e
template <int D, int P>
using GradTab = RowTab<Lv<D, P>::N, D * Lv<D, P>::Q, (D * Lv<D, P>::Q * Lv<D, P>::N) % 2 == 0>;

// Reciprocal and reciprocal square root of a float64: one third-order step (Householder's method
// for 1/y - a and 1/y^2 - a) on the hardware's approximation, whose error of about 2^-20 becomes
// its cube, below the rounding of the result (within 2 ulp of the exact value).  3 and 5 float64
// operations, where the correctly rounded division and square root take the pipe for 5 and 9.  For
// normal arguments whose result is normal (the reciprocal's of either sign; a negative one's root is
// NaN); 0, denormals and infinities give an infinity or NaN.
__device__ __forceinline__ double rcp_h3(double a) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(a));
    const double e = fma(-a, y, 1.0);
    return fma(y, fma(e, e, e), y);
}
__device__ __forceinline__ double rsqrt_h3(double a) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(a));
    const double e = fma(-a * y, y, 1.0);
    return fma(e * y, fma(0.375, e, 0.5), y);
}

// b / a, negative if either number is: its square root is then NaN as sqrt(a) or sqrt(b) would be, also
// where both are negative (a state without a meaning must not look like one with).
__device__ __forceinline__ double ratio_or_negative(double b, double ia, double a) {
    const double r = b * ia;
    return __hiloint2double(__double2hiint(r) | (__double2hiint(a) & (int)0x80000000), __double2loint(r));
}

}  // namespace emg
