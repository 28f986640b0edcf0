// Thread blocks of the Arnoldi process (krylov.cu).  Host C++ alone, so that the rule can be tested without a GPU.
#pragma once

#include <algorithm>
#include <cstdint>

namespace emg {

// At most `cap` and what is co-resident (per_sm per SM; two, as the form with rows in registers).  More
// blocks share out the rows' work, fewer make the cross-block reductions shorter, which every block
// repeats.  Measured, us of an EXP1 step (m = 30) with 64, 128, 192 and 256 rows a block: float64, whose
// pipe a block of 256 rows fills, 2560 rows 739 747 801 872, 10240 rows 887 756 806 880, 23040 rows 1111 1132
// 840 905, 40960 rows 1319 (304 blocks) 1322 1352 1384; float32 2560 rows 478 479 495 491, 10240 rows 511 487
// 496 490, 23040 rows 669 585 525 518, 40960 rows 717 720 664 619.  float64 between what 152 blocks of 192
// and of 256 rows hold (304 blocks / 256 rows a block): 30720 rows 1222 / 936, 33280 rows 1209 / 941, 36400 rows
// 1221 / 949.
inline int64_t arnoldi_blocks(int64_t rows, bool f32, int nsm, int per_sm, int64_t cap) {
    auto blocks = [rows](int64_t n) { return (rows + n - 1) / n; };
    const int64_t resident = (int64_t)nsm * std::max(1, std::min(per_sm, 2));
    int64_t nb = resident;
    if (f32)
        nb = blocks(rows <= 10240 ? 128 : 256);
    else
        for (int64_t n : {128, 192, 256})
            if (blocks(n) <= nsm) {
                nb = blocks(n);
                break;
            }
    return std::max<int64_t>(1, std::min({nb, resident, cap}));
}

}  // namespace emg
