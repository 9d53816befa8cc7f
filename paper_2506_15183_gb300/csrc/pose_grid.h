// The general pose's scatter grid: plain arithmetic, without CUDA, so that it can be checked on
// the host at the frame sizes that no test can hold.
#pragma once

namespace yoro {

constexpr int kScatterCols = 256;  // columns of a block: one per thread
constexpr int kScatterRows = 4;    // rows of a block

// Blocks of 256 columns x 4 rows over a w x h frame (w, h >= 1, w h < 2^31).  Unsigned
// throughout: w + 255 passes 2^31.  At most 2^29 blocks (one column, 2^31 rows), so one launch
// takes them all, a block each.
struct ScatterGrid {
    unsigned cols, blocks;
};

constexpr ScatterGrid scatter_grid(int w, int h)
{
    const unsigned cols = ((unsigned)w + (kScatterCols - 1u)) / (unsigned)kScatterCols;
    const unsigned rows = ((unsigned)h + (kScatterRows - 1u)) / (unsigned)kScatterRows;
    return {cols, cols * rows};
}

}  // namespace yoro
