// imb_sums.h -- sums of FP32 terms that keep the bits of FP64 additions, and the division by a
// constant, in plain C++ so that they can be checked without a GPU.
#pragma once
#include <cmath>
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define IMB_HD __host__ __device__ __forceinline__
#else
#define IMB_HD inline
#endif

namespace imb {

// a + b = s + e exactly, unless s overflows (TwoSum: Knuth, The Art of Computer Programming, Vol. 2, Sec. 4.2.2)
IMB_HD float two_sum(float a, float b, float &e) {
    const float s = a + b, bb = s - a;
    e = (a - (s - bb)) + (b - bb);
    return s;
}

// A sum of FP32 terms in three FP32 parts: what the first part rounds off goes to the second without
// error, what that rounds off to the third: some 70 bits, where FP64 additions keep 53.  An FP64 add
// takes a warp 64 cycles, and the sums of a unit or block are one chain of them; these are FP32
// instructions, with three conversions at the end.  NaN or an infinity, also from a sum beyond
// FP32, ends in a first part that is not finite: the caller then adds the terms in FP64.
struct Sum3 {
    float hi = 0.0f, lo = 0.0f, lo2 = 0.0f;
    IMB_HD void add(float b) {
        float e, e2;
        hi = two_sum(hi, b, e);
        lo = two_sum(lo, e, e2);
        lo2 += e2;
    }
    IMB_HD void add(const Sum3 &o) {
        add(o.hi);
        float e2;
        lo = two_sum(lo, o.lo, e2);
        lo2 += e2 + o.lo2;
    }
    IMB_HD bool finite() const { return hi - hi == 0.0f; }
    IMB_HD double value() const { return (double)hi + ((double)lo + (double)lo2); }
};

// The sum of N terms as FP64 additions in their order give it, or closer.
template <int N> IMB_HD double sum_terms(const float *v) {
    Sum3 s;
    for (int i = 0; i < N; ++i) s.add(v[i]);
    if (s.finite()) return s.value();
    double d = 0.0;
    for (int i = 0; i < N; ++i) d += (double)v[i];
    return d;
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
