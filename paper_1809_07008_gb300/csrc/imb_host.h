// imb_host.h -- decisions the host takes before a launch, in plain C++ so that they can be compiled
// and checked without a GPU.
#pragma once
#include <cmath>
#include <cstddef>
#include <cstdint>
#include <cstring>
#include <mutex>

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

// What was asked once of every device (a kernel's attributes hold for the device they were set on), by
// whichever thread comes first.
template <typename T, int DEVICES = 64>
class PerDevice {
    std::once_flag once[DEVICES];
    T value[DEVICES] = {};

public:
    template <typename F> T get(int device, F ask) {
        if (device < 0 || device >= DEVICES) return ask();
        std::call_once(once[device], [&] { value[device] = ask(); });
        return value[device];
    }
};

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

// Particles of large islands that the DEM's cluster takes: what its blocks hold, and fewer where a cycle has
// few sub-cycles.  Placing the particles (the ranks of the Morton order, the pairs across
// blocks) grows faster than their number, 60 us with 4096, and the sub-cycles must win that back.  Cycles of
// slabs of 1000, 2000 and 4096 disks, cluster / grid: one sub-cycle 128 / 129, 147 / 134 and 217 / 170 us,
// two 133 / 146, 156 / 154 and 232 / 194, five 150 / 207, 189 / 218 and 283 / 249, ten 182 / 310, 235 /
// 322 and 362 / 349, twenty 239 / 515, 333 / 525 and 535 / 556.
constexpr int CLUSTER_PARTICLES = 4096;
inline int cluster_limit(int N_sub) { return N_sub < 12 ? 1000 + 300 * (N_sub - 1) : CLUSTER_PARTICLES; }

// Whether a batch holds its populations in rows padded to whole blocks (`padded` cells of `elem` bytes
// with the padding) or in whole planes without any (`cells`).  `ragged` of its `rows` are no multiple of 16
// cells long.
//
// By speed: a blocked row ends in a part of a 32-byte sector that nothing else completes, and a narrow
// row is mostly padding, so planes win on narrow rows; blocked rows need fewer instructions a cell, so
// they win where that counts: on wider rows and where the populations stay in L2.  ps a cell and step,
// blocked / planes, rows of 160 or 120 cells: 6 M cells FP32, width 3: 108 / 18, 33: 23 / 16, 50: 20 / 16, 65:
// 19 / 16, 160: 14 / 15, 257: 15 / 15; FP16, 24: 23 / 15, 31: 12 / 15, 33: 18 / 15, 50: 13 / 15, 257: 11 /
// 15; 0.3 M cells (22 MB) FP32, width 3: 123 / 38, 11: 32 / 34, 50: 28 / 32, 450: 23 / 31; 1.5 M cells FP16 (54
// MB), 24: 29 / 17, 45: 13 / 17.  (Ragged FP32 rows of 100 to 250 cells in large batches would be up to 10 % faster in
// planes; the line is where blocked rows stop being the slower of the two layouts the sweeps have had, so
// that no width is slower than with row segments of planes: 4 M cells in rows of 90, 70.8 us a step blocked, 68.6
// in segments, 67.8 in planes; in rows of 64 60.5, 60.6 and 64.8.)
//
// By memory: the padding must not cost a call that planes leave room for: two buffers and one domain of
// `most` cells read back as FP64, or three while the launch shapes are timed, with the solid ratios.
inline bool blocked_rows(size_t cells, size_t rows, size_t ragged, size_t padded, size_t most, size_t elem, size_t mem_free) {
    const double state = 9.0 * (double)cells * (double)elem, wide = 9.0 * (double)padded * (double)elem;
    const double ratios = 4.0 * (double)cells, even = 4.0 * (double)padded, read = 72.0 * (double)most;
    const double room = (double)mem_free - 64.0e6;   // contexts, tables, allocation granularity
    if (2.0 * wide + even + read > room && 2.0 * state + ratios + read <= (double)mem_free) return false;
    if (3.0 * wide + even > room && 3.0 * state + ratios <= (double)mem_free) return false;
    const bool small = 2.0 * state < 32.0e6;
    if (cells < (size_t)(small ? 8 : 31) * rows) return false;   // mean width of the rows
    return small || elem == 2 || cells >= 100 * ragged;
}

}  // namespace imb
