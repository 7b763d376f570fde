// imb_host.h -- decisions the host takes before a launch, free of CUDA so that they can be
// compiled and checked without a GPU.
#pragma once
#include <cstddef>
#include <cstdint>

namespace imb {

// Whether [p, p + bytes) is aligned and lies within the one memory range [start, start + size).
inline bool span_covered(uintptr_t p, size_t bytes, size_t align, uintptr_t start, size_t size) {
    return bytes > 0 && p % align == 0 && p >= start && bytes <= size && p - start <= size - bytes;
}

// Whether n arrays of `bytes` each keep out of each other's memory (what one kernel writes to two
// overlapping ones has no order).
inline bool spans_disjoint(const void *const *p, int n, size_t bytes) {
    for (int i = 0; i < n; ++i)
        for (int j = 0; j < i; ++j) {
            const uintptr_t a = (uintptr_t)p[i], b = (uintptr_t)p[j];
            if ((a < b ? b - a : a - b) < bytes) return false;
        }
    return true;
}

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
