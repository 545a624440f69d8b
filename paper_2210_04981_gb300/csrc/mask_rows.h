// Strips of the mask's register sweep (plain C++, no CUDA types).
#pragma once

namespace hdof {

constexpr int SW_OUT = 26;   // output columns per warp
constexpr int SW_ROWS = 32;  // output rows per warp, fewer on small images (sweep_rows)

// warps of the sweep over a W x H image with strips of `rows` output rows
inline long long sweep_warps(int W, int H, int rows) {
    return (long long)((W + SW_OUT - 1) / SW_OUT) * ((H + rows - 1) / rows);
}

// Output rows per warp of one launch's sweep, `warps(rows)` its warps over all
// its images: a warp walks its rows one after another (6 more for the halo),
// so a launch whose few strips leave the machine empty (below 8 warps an SM)
// is cut into shorter ones: the 128x128 mask 35 -> 23 us.  The filtered values
// do not depend on it.  At 1080p (2516 warps) 8 or 16 rows shorten the mask by
// 5% and the frame not at all.  A batch counts all its views: 64 of 256x256
// and 640x480 that each took the line for themselves walked up to 14 rows for
// 8 and took 258 us, with strips of 32 rows 207.
template <class Warps>
int sweep_rows(Warps warps, int sms) {
    int rows = SW_ROWS;
    while (rows > 8 && warps(rows) < 8ll * sms) rows /= 2;
    return rows;
}

}  // namespace hdof
