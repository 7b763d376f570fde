// imb_host.h -- decisions the host takes before a launch, free of CUDA so that they can be
// compiled and checked without a GPU.
#pragma once

namespace imb {

// Columns of a row to the blocks of the reverse step.  With the inlet and outlet columns transposed in the
// same launch, column 0 must share a block with column 1 and column nx - 1 with column nx - 2.  Where the
// last column would start a block of its own the blocks begin one column further left: the first
// one's first thread is idle then, and the last one holds two columns.
constexpr int ADJ_BLOCK = 256;
struct AdjointGrid {
    int blocks, shift;   // thread t of block b takes column b ADJ_BLOCK + t - shift
};
inline AdjointGrid adjoint_grid(int nx, bool inlet) {
    const int shift = inlet && nx % ADJ_BLOCK == 1 ? 1 : 0;
    return {(nx + shift + ADJ_BLOCK - 1) / ADJ_BLOCK, shift};
}

}  // namespace imb
