// Whether the kernels of one residual start in each other's tails (common.cuh: launch_chained).  Host C++
// alone, so that the rule can be tested without a GPU.
#pragma once

#include <cstdint>

namespace emg {

// Elements that a block of k_volume takes with one thread per mode (residual.cu asserts that they agree).
constexpr int volume_elems(int dim, int p) {
    return dim == 2 ? (p == 1 ? 21 : p == 2 ? 10 : p == 3 ? 6 : 4) : p == 1 ? 32 : p == 2 ? 12 : 3;
}

// Blocks that wait in the tail of the kernel before them take the places that fall free first, so some
// multiprocessors get many of them and others none: good where the work is short (the launches' latency
// counts) or the grid comes in enough waves to even out, bad between.  Residuals of one solver one after the
// other, us apart / chained: 32 x 16 p = 1 29.9 / 23.2, p = 2 27.9 / 22.7, p = 4 31.0 / 27.6, 45 x 21 p = 4
// 36.7 / 33.7, 216 hexes at p = 1 39.0 / 31.8; 90 x 45 p = 2 47.7 / 55.0, 128 x 64 p = 2 63.7 / 75.5, 110 x
// 50 p = 3 61.7 / 76.8, 256 x 128 p = 0 47.3 / 71.3, 1944 hexes at p = 1 54.5 / 78.6, at p = 3 212 / 233;
// 181 x 80 p = 3 132 / 126, 150 x 70 p = 4 154 / 152 and 128 x 64 p = 4 123 / 125, but with three solvers in
// turn 113 / 109 and 87.2 / 84.5.  3-D gains nothing at any large size with three.
// The lines: 12000 face points (chained 0.77 to 0.96 below; 64 x 32 p = 1, 12384 of them, 1.00, with
// three 1.16), at p = 0 28000 in 2-D (110 x 55, 24420: 0.78; 128 x 64, 33024: 1.06) and 100000 in 3-D (7200 hexes,
// 88800: 0.88); 2-D, 1.6 waves of k_volume's blocks (8 of its 64 threads a multiprocessor).
inline bool residual_chains(int dim, int p, int64_t elems, int64_t face_points) {
    if (face_points <= (p > 0 ? 12000 : dim == 2 ? 28000 : 100000)) return true;
    return dim == 2 && p > 0 && 5 * (elems / volume_elems(dim, p)) >= 8 * (8 * 152);
}

}  // namespace emg
