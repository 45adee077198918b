// The cell grid of the detector's selection (host only, plain C++).
#pragma once

namespace vt {

constexpr int kGfttMaxSide = 65535;  // longest side of a level the detector takes

// Cells of a w x h level: at least min_dist wide, so that corners closer than
// min_dist lie in neighbouring cells, and at most max_cells of them.  A
// min_dist beyond kGfttMaxSide gives the same single cell as that side does
// (and w + cell stays in 32 bits).
inline void gftt_grid(int w, int h, int min_dist, int max_cells, int &cell, int &cx, int &cy) {
    cell = min_dist < kGfttMaxSide ? min_dist : kGfttMaxSide;
    while ((long long)((w + cell - 1) / cell) * ((h + cell - 1) / cell) > max_cells) ++cell;
    cx = (w + cell - 1) / cell;
    cy = (h + cell - 1) / cell;
}

}  // namespace vt
