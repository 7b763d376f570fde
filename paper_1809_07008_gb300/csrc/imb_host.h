// imb_host.h -- decisions the host takes before a launch, and arithmetic shared with the device,
// in plain C++ so that they can be compiled and checked without a GPU.
#pragma once
#include <cmath>
#include <cstddef>
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define IMB_HD __host__ __device__ __forceinline__
#else
#define IMB_HD inline
#endif

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

// a / b for a constant b > 0 whose correctly rounded reciprocal y = RN(1 / b) is known, rounded
// to nearest: a faithful quotient from the reciprocal, then one step with the exact remainder
// (Markstein 1990: with y correctly rounded and q within an ulp, q + r y rounds to a / b).
// Five FP64 operations, 64 cycles each, instead of the ten of a division.  The argument needs quotient and
// remainder in the normal range: with a and b between 2^-400 and 2^400 the quotient lies between
// 2^-801 and 2^801 and the remainder's last bit above 2^-600.  Everything else (zeros, infinities, NaN
// among it) divides.
IMB_HD unsigned exponent_of(double v) {
#ifdef __CUDA_ARCH__
    return ((unsigned)__double2hiint(v) >> 20) & 0x7ffu;
#else
    uint64_t b;
    std::memcpy(&b, &v, sizeof(b));
    return (unsigned)(b >> 52) & 0x7ffu;
#endif
}
IMB_HD double div_by(const double a, const double b, const double y) {
    if (exponent_of(a) - 623u < 800u && exponent_of(b) - 623u < 800u) {
        double q = a * y;
        q = fma(fma(-b, q, a), y, q);
        return fma(fma(-b, q, a), y, q);
    }
    return a / b;
}

}  // namespace imb
