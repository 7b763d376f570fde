// imb_batch.cu -- many independent small periodic domains stepped together.
//
// A sweep over resolution, solid fraction, relaxation time and driving force (the paper's
// parameter studies, Sec. 3) is a set of independent lattices.  Each is periodic in x and y,
// driven by a body force (Guo forcing, as in the single-lattice path), and holds fixed disks
// whose summed solid ratio E per cell (exact overlap area, Sec. 2.3) is computed once; its
// relaxation time may carry the Smagorinsky closure of the single-lattice path.  One
// launch advances every domain by one step: each warp takes an equal run of items of 32 or 64 cells
// (finding the domain of its first item by binary search in the domains' first items),
// pulls with the periodic wrap of the domain (Eq. 1), collides with the blend of Eq. 13
// (B from Eq. 14, u_s = 0 for disks at rest) and adds the drag B (j - F) (Eq. 15) of the
// nodes it stepped to the domain's accumulator.  Steps run as a replayed CUDA graph of two launches (A -> B,
// B -> A); the block size and the cells per lane are chosen by timing the candidates on the
// batch itself.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <type_traits>
#include <vector>

#include "../../include/imblbm.h"
#include "imb_device.cuh"
#include "imb_host.h"
#include "imb_kernels.h"

namespace imb {

struct BatchDomain {
    int nx, ny;
    int item0[2];       // first work item of the domain, with one and with two cells per lane
    size_t off;         // element offset of the domain in the population buffers
    size_t row;         // elements from one row to the next
    size_t e_off;       // offset of the domain's solid ratios
    int plane;          // whole planes: elements of one (blocked rows: 0)
    int e_row;          // solid ratios from one row to the next (blocked rows: even)
    float tau, omega0, Fx, Fy;
    float smag_coef;    // 18 sqrt(2) C^2 of the Smagorinsky closure (0: plain BGK)
};

// Layout of the populations: rows of blocks of 128 bytes per plane, the nine planes of a block one
// after another ([y][x / SEGB][slot][x % SEGB]), so that one pointer and compile-time offsets
// reach every plane: with whole planes one after another a node's nine loads and nine stores took
// some 40 of its 330 instructions for addresses.  The planes that a node pulls from the same row
// (c_y = 0, 1, -1) are neighbours: slots 3 g, 3 g + 1, 3 g + 2 hold c_x = 0, 1, -1.
//
// Rows padded to whole blocks take up to 21 times the memory of their cells (three cells of 16
// bits in a block of 64).  A batch of narrow domains, or one that the padding would push out of memory
// (blocked_rows), holds whole planes instead ([slot][y][x], no padding) and is stepped with one cell a
// lane.
template <typename S> __host__ __device__ constexpr int segb() { return 128 / (int)sizeof(S); }
__host__ __device__ constexpr int group_q(int g, int k) { return (g == 0 ? 0x310 : g == 1 ? 0x652 : 0x784) >> (4 * k) & 15; }
__host__ __device__ constexpr int slot_of(int q) {
    for (int i = 0; i < 9; ++i)
        if (group_q(i / 3, i % 3) == q) return i;
    return -1;
}
static_assert(cy_of(2) == 1 && cy_of(5) == 1 && cy_of(6) == 1 && cy_of(4) == -1 && cy_of(8) == -1 && cy_of(7) == -1 &&
                  cx_of(1) == 1 && cx_of(5) == 1 && cx_of(8) == 1 && cx_of(3) == -1 && cx_of(6) == -1 && cx_of(7) == -1,
              "groups of the planes by source row");
// element offset of cell x in a blocked row, slot 0
template <typename S> __host__ __device__ __forceinline__ int col_of(int x) {
    return x / segb<S>() * 9 * segb<S>() + x % segb<S>();
}
// where a cell of a row and a slot of it lie
template <typename S> struct BlockedRows {
    __device__ __forceinline__ explicit BlockedRows(const BatchDomain &) {}
    __device__ __forceinline__ int col(int x) const { return col_of<S>(x); }
    __device__ __forceinline__ int slot(int i) const { return i * segb<S>(); }
};
struct WholePlanes {
    int plane;
    __device__ __forceinline__ explicit WholePlanes(const BatchDomain &D) : plane(D.plane) {}
    __device__ __forceinline__ int col(int x) const { return x; }
    __device__ __forceinline__ int slot(int i) const { return i * plane; }   // 9 nx ny < 2^31 (checked)
};
template <typename S, bool BLOCKED> using Layout = std::conditional_t<BLOCKED, BlockedRows<S>, WholePlanes>;

// The node of a domain whose disks are at rest.  With u_s = 0 the solid operator of Eq. 12
// summed over the covering disks is B (f_{-q} - f^eq_{-q}(u) + f^eq_q(0) - f_q); in the
// shifted variables d_q = f_q - w_q and n_q = d_q - (f^eq_q(u) - w_q) this is
// B (n_{-q} - d_q + w_q drho), and Eq. 13 becomes
//   d*_q = (1 - B) [d_q - omega n_q + (1 - omega / 2) w_q S_q] + B (n_{-q} + w_q drho)
// with S_q / w_q = 3 (c_q - u).F + 9 (c_q.u)(c_q.F) (Guo forcing).  The same algebra as the
// general collision with every solid-velocity moment zero, with fewer operations.
struct Cells1 {           // one cell per lane
    using T = float;
    static __device__ __forceinline__ T all(float a) { return a; }
    static __device__ __forceinline__ T add(T a, T b) { return a + b; }
    static __device__ __forceinline__ T mul(T a, T b) { return a * b; }
    static __device__ __forceinline__ T fma(T a, T b, T c) { return fmaf(a, b, c); }
    template <typename F> static __device__ __forceinline__ T each(T a, F f) { return f(a); }
    static __device__ __forceinline__ bool below(T a, float lim) { return a < lim; }
    static __device__ __forceinline__ float sum(T a) { return a; }
};
struct Cells2 {           // two neighbouring cells per lane, FP32x2 instructions throughout
    using T = float2;
    static __device__ __forceinline__ T all(float a) { return make_float2(a, a); }
    static __device__ __forceinline__ T add(T a, T b) { return __fadd2_rn(a, b); }
    static __device__ __forceinline__ T mul(T a, T b) { return __fmul2_rn(a, b); }
    static __device__ __forceinline__ T fma(T a, T b, T c) { return __ffma2_rn(a, b, c); }
    template <typename F> static __device__ __forceinline__ T each(T a, F f) { return make_float2(f(a.x), f(a.y)); }
    static __device__ __forceinline__ bool below(T a, float lim) { return a.x < lim && a.y < lim; }
    static __device__ __forceinline__ float sum(T a) { return a.x + a.y; }
};
template <int CPL> using CellsOf = std::conditional_t<CPL == 2, Cells2, Cells1>;

// The eight moving directions as four pairs (q, -q), q = 1, 2, 5, 6, whose terms differ only in
// the sign of their odd parts.
__host__ __device__ constexpr int bpair_q(int k) { return k < 2 ? k + 1 : k + 3; }

// d -> post-collision d, in place; the lane's drag (Eq. 15 with u_s = 0) is added to fx, fy.  Returns
// whether |u|^2 lies below the Mach guard (false for NaN).
template <class V>
__device__ __forceinline__ bool rest_node(typename V::T (&d)[9], const typename V::T e, const BatchDomain &D,
                                          typename V::T &fx, typename V::T &fy) {
    using T = typename V::T;
    const T one = V::all(1.0f), neg = V::all(-1.0f);
    auto sub = [&](T a, T b) { return V::fma(b, neg, a); };
    T P[4], M[4];   // d_q + d_-q, d_q - d_-q
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int q = bpair_q(k);
        P[k] = V::add(d[q], d[opp_of(q)]);
        M[k] = sub(d[q], d[opp_of(q)]);
    }
    const T diag = V::add(P[2], P[3]);
    const T drho = V::add(d[0], V::add(V::add(P[0], P[1]), diag));
    const T inv = V::each(V::add(one, drho), [](float r) { return __fdividef(1.0f, r); });
    const T mx = sub(V::add(M[0], M[2]), M[3]), my = V::add(V::add(M[1], M[2]), M[3]);
    const T jx = V::fma(V::all(0.5f), V::all(D.Fx), mx), jy = V::fma(V::all(0.5f), V::all(D.Fy), my);   // Eqs. 3-4
    const T ux = V::mul(jx, inv), uy = V::mul(jy, inv);
    const T jxx = V::mul(jx, ux), juu = V::fma(jy, uy, jxx);
    const T t = V::fma(V::all(-1.5f), juu, drho);   // f^eq_{+-q} - w_q = w_q (t + (3 c.j) (1.5 c.u) +- 3 c.j)
    T omega = V::all(D.omega0), te = V::all(D.tau);
    if (D.smag_coef > 0.0f) {       // Smagorinsky closure; Pi = sum c c f - (drho / 3 + j u) on the diagonal
        const T third = V::fma(V::all(1.0f / 3.0f), drho, jxx), thirdy = V::fma(V::all(1.0f / 3.0f), drho, V::mul(jy, uy));
        const T pxx = sub(V::add(P[0], diag), third), pyy = sub(V::add(P[1], diag), thirdy);
        const T pxy = V::fma(V::mul(jx, neg), uy, sub(P[2], P[3]));
        const T Q = V::fma(pxx, pxx, V::fma(pyy, pyy, V::mul(V::add(pxy, pxy), pxy)));
        const T sq = V::each(Q, [](float v) { return v > 0.0f ? v * rsqrtf(v) : 0.0f; });
        const T disc = V::fma(V::mul(V::all(D.smag_coef), sq), inv, V::all(D.tau * D.tau));
        const T root = V::each(disc, [](float v) { return v * rsqrtf(v); });
        te = V::mul(V::all(0.5f), V::add(V::all(D.tau), root));
        omega = V::each(te, [](float v) { return __fdividef(1.0f, v); });
    }
    const T ec = V::each(e, [](float v) { return fminf(v, 1.0f); });
    const T tm = V::add(te, V::all(-0.5f));
    const T den = V::each(V::add(sub(one, ec), tm), [](float v) { return __fdividef(1.0f, v); });
    const T B = V::mul(V::mul(ec, tm), den);   // Eq. 14 (0 in uncovered cells)
    // d*_q = (1 - B) d_q - (1 - B) omega n_q + B n_{-q} + w_q [(1 - B)(1 - omega / 2) S_q + B drho], summed from
    // the smallest term up to d_q, which alone rounds at its own size;
    //   n_{+-q} = d_{+-q} - w_q (t + 4.5 rho (c.u)^2 +- 3 c.j),  S_{+-q} = 9 (c.u)(c.F) - 3 u.F +- 3 c.F
    const T fl = sub(one, B), flw = V::mul(V::mul(fl, neg), omega);
    const T fls = V::mul(fl, V::fma(V::all(-0.5f), omega, one)), Bd = V::mul(B, drho);
    const T g = V::mul(V::all(-3.0f), V::fma(ux, V::all(D.Fx), V::mul(uy, V::all(D.Fy))));
    const T jx3 = V::mul(V::all(3.0f), jx), jy3 = V::mul(V::all(3.0f), jy);
    const T ux15 = V::mul(V::all(1.5f), ux), uy15 = V::mul(V::all(1.5f), uy);
    const T n0 = V::fma(V::all(-w_of(0)), t, d[0]);
    const T v0 = V::mul(V::all(w_of(0)), V::fma(fls, g, Bd));
    d[0] = V::fma(fl, d[0], V::fma(flw, n0, V::fma(B, n0, v0)));
    const T v4[4] = {ux15, uy15, V::add(ux15, uy15), sub(uy15, ux15)}, j4[4] = {jx3, jy3, V::add(jx3, jy3), sub(jy3, jx3)};
    const float F4[4] = {D.Fx, D.Fy, D.Fx + D.Fy, D.Fy - D.Fx};   // c.F
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int q = bpair_q(k), o = opp_of(q);
        const T w = V::all(-w_of(q)), wp = V::all(w_of(q));
        const T ev = V::fma(j4[k], v4[k], t), se = V::fma(V::all(6.0f * F4[k]), v4[k], g), so = V::all(3.0f * F4[k]);
        const T nq = V::fma(w, V::add(ev, j4[k]), d[q]), no = V::fma(w, sub(ev, j4[k]), d[o]);
        const T vq = V::mul(wp, V::fma(fls, V::add(se, so), Bd)), vo = V::mul(wp, V::fma(fls, sub(se, so), Bd));
        d[q] = V::fma(fl, d[q], V::fma(flw, nq, V::fma(B, no, vq)));
        d[o] = V::fma(fl, d[o], V::fma(flw, no, V::fma(B, nq, vo)));
    }
    fx = V::fma(B, V::add(jx, V::all(-D.Fx)), fx);
    fy = V::fma(B, V::add(jy, V::all(-D.Fy)), fy);
    const T usq = V::mul(juu, inv);
    return V::below(usq, 0.09f);
}

// stored values as loaded (converted to FP32 where they are used), one or two cells
__device__ __forceinline__ float to_f32(float v) { return v; }
__device__ __forceinline__ float to_f32(__half v) { return __half2float(v); }
__device__ __forceinline__ float to_f32(__nv_bfloat16 v) { return __bfloat162float(v); }
template <typename S> struct Pair;
template <> struct Pair<float> {
    using T = float2;
    static __device__ __forceinline__ float2 f32(T v) { return v; }
    static __device__ __forceinline__ T of(float2 v) { return v; }
};
template <> struct Pair<__half> {
    using T = __half2;
    static __device__ __forceinline__ float2 f32(T v) { return __half22float2(v); }
    static __device__ __forceinline__ T of(float2 v) { return __float22half2_rn(v); }
};
template <> struct Pair<__nv_bfloat16> {
    using T = __nv_bfloat162;
    static __device__ __forceinline__ float2 f32(T v) { return __bfloat1622float2(v); }
    static __device__ __forceinline__ T of(float2 v) { return __float22bfloat162_rn(v); }
};

// the pulled values of a lane (Eq. 1, periodic wrap) from the rows y, y - 1 and y + 1 of a domain
template <typename S, int CPL> struct Pulled;
template <typename S> struct Pulled<S, 1> {
    S r[9];
    float e;
    template <class L>
    __device__ __forceinline__ void fetch(const S *const (&R)[3], const float *Er, int x, int nx, const L lay) {
        const int c = lay.col(x), cl = lay.col(x == 0 ? nx - 1 : x - 1), cr = lay.col(x == nx - 1 ? 0 : x + 1);
#pragma unroll
        for (int g = 0; g < 3; ++g) {
            r[3 * g] = __ldg(R[g] + c + lay.slot(3 * g));
            r[3 * g + 1] = __ldg(R[g] + cl + lay.slot(3 * g + 1));
            r[3 * g + 2] = __ldg(R[g] + cr + lay.slot(3 * g + 2));
        }
        e = __ldg(Er + x);
    }
    __device__ __forceinline__ void values(float (&d)[9], bool) const {
#pragma unroll
        for (int i = 0; i < 9; ++i) d[group_q(i / 3, i % 3)] = to_f32(r[i]);
    }
    template <class L> static __device__ __forceinline__ void store(S *p, const float (&d)[9], const L lay) {
#pragma unroll
        for (int q = 0; q < 9; ++q) Store<S>::st(p + lay.slot(slot_of(q)), d[q]);
    }
};
// The cells x (even) and x + 1.  A plane with c_x = 0 is one load of both; the others' sources
// straddle the pairs and are loaded one by one (x - 1 and x, x + 1 and x + 2): no exchange between
// lanes, whose rows may differ.
template <typename S> struct Pulled<S, 2> {
    typename Pair<S>::T c2[3];
    S l0[3], l1[3], r0[3], r1[3];
    float2 e;
    __device__ __forceinline__ void fetch(const S *const (&R)[3], const float *Er, int x, int nx, const BlockedRows<S>) {
        constexpr int G = segb<S>();
        const int in = x % G, c = x / G * 9 * G + in;
        const int cl = x == 0 ? col_of<S>(nx - 1) : (in == 0 ? c - 8 * G - 1 : c - 1);
        const int ca = x + 1 == nx ? 0 : c + 1;
        const int cb = x + 2 >= nx ? 0 : (in == G - 2 ? c + 8 * G + 2 : c + 2);
#pragma unroll
        for (int g = 0; g < 3; ++g) {
            c2[g] = __ldg(reinterpret_cast<const typename Pair<S>::T *>(R[g] + c + 3 * g * G));
            l0[g] = __ldg(R[g] + cl + (3 * g + 1) * G);
            l1[g] = __ldg(R[g] + c + (3 * g + 1) * G);
            r0[g] = __ldg(R[g] + ca + (3 * g + 2) * G);
            r1[g] = __ldg(R[g] + cb + (3 * g + 2) * G);
        }
        e = __ldg(reinterpret_cast<const float2 *>(Er + x));
    }
    // tail: x is the last cell of a row of odd length, and the lane's second cell no cell of the
    // domain.  It takes the first one's values (its solid ratio is 0: no drag).
    __device__ __forceinline__ void values(float2 (&d)[9], bool tail) const {
#pragma unroll
        for (int g = 0; g < 3; ++g) {
            d[group_q(g, 0)] = Pair<S>::f32(c2[g]);
            d[group_q(g, 1)] = make_float2(to_f32(l0[g]), to_f32(l1[g]));
            d[group_q(g, 2)] = make_float2(to_f32(r0[g]), to_f32(r1[g]));
        }
        if (tail) {
#pragma unroll
            for (int q = 0; q < 9; ++q) d[q].y = d[q].x;
        }
    }
    static __device__ __forceinline__ void store(S *p, const float2 (&d)[9], const BlockedRows<S>) {
#pragma unroll
        for (int q = 0; q < 9; ++q)
            *reinterpret_cast<typename Pair<S>::T *>(p + slot_of(q) * segb<S>()) = Pair<S>::of(d[q]);
    }
};

// A work item is 32 CPL cells of a domain, row after row without regard to the rows' ends (with two
// cells per lane, of rows rounded up to even length); only a domain's last item leaves lanes idle.
// Each warp takes an equal run of consecutive items, so the warps finish together whatever the
// domain sizes, and the drag of a domain is summed in registers until the warp leaves it.  The
// loads of the next item of the same domain are issued before the arithmetic of the current one.
//
// What bounds it: with two cells a lane the registers (128, two blocks an SM: 16 warps) and the latency
// of the loads; the schedulers issue on half the cycles and DRAM moves 44 B a cell of the 40 it must
// (16 bits), at 4.3 TB/s.  256 domains, 15.5 M cells, FP16, 100 steps at a time: 195 us a step with whole
// planes one after another, rows cut into segments and one cell a lane, 154 us now (in runs of 5000 steps
// 186 -> 139 us; 155 to 158 us where the variants below were timed); 12 domains of 0.28 M cells together,
// FP32: 11.5 -> 9.4 us.  With the forcing inside the equilibrium that is relaxed to, d_q - omega (d_q - w_q E'_q),
// 150 us, but one more rounding at the size of E' and of d_q: the drag's error against 64 bits was 8.3e-7 (rms over
// 288 FP32 domains), 7.7e-7 with the former sums over direction pairs and 6.1e-7 with these.
// With the collision as a sum of d_q + d_-q and d_q - d_-q (half the operations) 156 us and twice
// the FP32 error; two items ahead 148 us with that form, 176 us (spills) with this one; three
// blocks an SM (80 registers, spills) 187 us; five of 128 threads 151 us.
template <typename S, int CPL, bool BLOCKED>
__global__ void __launch_bounds__(256, CPL == 2 ? 2 : 3)
k_batch_step(const S *__restrict__ fin, S *__restrict__ fout, const BatchDomain *__restrict__ dom,
             int ndom, int nitems, const float *__restrict__ E, double *drag, unsigned *err) {
    using V = CellsOf<CPL>;
    const int lane = threadIdx.x & 31;
    const int gw = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const int nw = (int)((gridDim.x * blockDim.x) >> 5);
    const int per = nitems / nw, rem = nitems % nw;
    const int it0 = gw * per + min(gw, rem);
    int left = per + (gw < rem ? 1 : 0);   // items of the warp
    if (left <= 0) return;   // the whole warp: gw is the same on every lane
    int lo = 0, hi = ndom - 1;   // the domain of the first item
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (dom[mid].item0[CPL - 1] <= it0) lo = mid;
        else hi = mid - 1;
    }
    bool unstable = false;
    for (int dd = lo, first = it0; left > 0; ++dd) {   // domains of the warp
        const BatchDomain D = dom[dd];
        const int nx = D.nx, ny = D.ny, width = (nx + CPL - 1) / CPL;
        first -= dd == lo ? D.item0[CPL - 1] : first;   // item within the domain
        int n = min(left, (int)(((long long)width * ny + 31) / 32) - first);   // items of this domain
        left -= n;
        const int p = first * 32 + lane;
        int y = p / width, x = (p - y * width) * CPL;
        Pulled<S, CPL> r;
        const S *src = fin + D.off;
        S *out = fout + D.off;
        const float *Ed = E + D.e_off;
        const Layout<S, BLOCKED> lay(D);
        auto fetch = [&] {
            if (y >= ny) return;   // past the end of the domain's last item
            const S *R[3] = {src + (size_t)y * D.row, src + (size_t)(y == 0 ? ny - 1 : y - 1) * D.row,
                             src + (size_t)(y == ny - 1 ? 0 : y + 1) * D.row};
            r.fetch(R, Ed + (size_t)y * D.e_row, x, nx, lay);
        };
        fetch();
        typename V::T fx = V::all(0.0f), fy = V::all(0.0f);
        while (n > 0) {
            typename V::T d[9];
            r.values(d, CPL == 2 && x + 1 == nx);
            const auto ec = r.e;
            const bool act = y < ny;
            S *dst = out + (size_t)y * D.row + lay.col(x);
            x += 32 * CPL;
            while (x >= nx) {   // rows of fewer than 32 CPL cells: several at once
                x -= width * CPL;
                ++y;
            }
            if (--n > 0) fetch();   // in flight during this item's arithmetic
            if (act) {
                if (!rest_node<V>(d, ec, D, fx, fy)) unstable = true;   // Mach guard, also catches NaN
                Pulled<S, CPL>::store(dst, d, lay);
            }
        }
        float sx = V::sum(fx), sy = V::sum(fy);   // leaving the domain: add its drag
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            sx += __shfl_xor_sync(0xffffffffu, sx, o);
            sy += __shfl_xor_sync(0xffffffffu, sy, o);
        }
        if (lane == 0 && (sx != 0.0f || sy != 0.0f)) {
            atomicAdd(&drag[2 * dd], (double)sx);
            atomicAdd(&drag[2 * dd + 1], (double)sy);
        }
    }
    if (__any_sync(0xffffffffu, unstable) && lane == 0) set_err(err, ERR_UNSTABLE);
}

// summed solid ratio: one thread per (disk, cell of its bounding box)
__global__ void k_batch_solid(const BatchDomain *__restrict__ dom, const int *__restrict__ disk_dom,
                              const double *__restrict__ xy, const double *__restrict__ r, int ndisk, int span,
                              float *E) {
    const int w = 2 * span + 1;
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (long long)ndisk * w * w) return;
    const int j = (int)(t / (w * w)), cell = (int)(t % (w * w));
    const BatchDomain D = dom[disk_dom[j]];
    const double cx = xy[2 * j], cy = xy[2 * j + 1];
    const int ci = (int)floor(cx), cj = (int)floor(cy);
    const float fx = (float)(cx - ci), fy = (float)(cy - cj), rf = (float)r[j];
    const int di = cell % w - span, dk = cell / w - span;
    const float lox = __fsub_rn((float)di, fx), loy = __fsub_rn((float)dk, fy);
    if (!covers(lox, loy, rf)) return;
    const int i = ((ci + di) % D.nx + D.nx) % D.nx, k = ((cj + dk) % D.ny + D.ny) % D.ny;
    atomicAdd(&E[D.e_off + (size_t)k * D.e_row + i], cell_disk_area(lox, loy, rf));
}

// f(x, t) of one domain (the pull of its post-collision field), as FP64 f = w + (f - w)
template <typename S>
__global__ void k_batch_gather(const S *__restrict__ fin, const BatchDomain *__restrict__ dom, int d,
                               double *out) {
    const BatchDomain D = dom[d];
    const size_t c = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const size_t cells = (size_t)D.nx * D.ny;
    if (c >= cells) return;
    const int x = (int)(c % D.nx), y = (int)(c / D.nx);
#pragma unroll
    for (int q = 0; q < 9; ++q) {
        const int xs = (x - cx_of(q) + D.nx) % D.nx, ys = (y - cy_of(q) + D.ny) % D.ny;
        const size_t at = D.plane ? (size_t)slot_of(q) * D.plane + xs : (size_t)(col_of<S>(xs) + slot_of(q) * segb<S>());
        out[(size_t)q * cells + c] = (double)w_of(q) + (double)Store<S>::ld(fin + D.off + (size_t)ys * D.row + at);
    }
}

}  // namespace imb

using namespace imb;

struct imb_batch {
    int device = 0, storage = 0, elem = 4, ndom = 0, nitems[2] = {0, 0}, ndisk = 0;
    size_t total = 0;          // elements per population buffer
    size_t cells = 0;
    bool blocked = true;       // layout of the populations
    void *buf[2] = {nullptr, nullptr};
    int cur = 0;               // buffer holding the current post-collision field
    BatchDomain *dom = nullptr;
    std::vector<BatchDomain> hdom;
    float *E = nullptr;
    double *drag = nullptr;
    unsigned *err = nullptr;
    long long steps_run = 0;
    cudaStream_t stream = nullptr;
    int block = 256, cpl = 1, grid = 0;
    bool grid_only = false;    // launch_step only sizes the grid
    cudaGraphExec_t graph[2] = {nullptr, nullptr};   // two steps starting from buffer 0 / 1
    std::string last_error;
};

namespace {

int bfail(imb_batch *b, int code, const std::string &msg) {
    if (b) b->last_error = msg;
    return code;
}

#define BCK(call, what)                                                                       \
    do {                                                                                      \
        cudaError_t e_ = (call);                                                              \
        if (e_ != cudaSuccess)                                                                \
            return bfail(b, e_ == cudaErrorMemoryAllocation ? IMB_E_NOMEM : IMB_E_CUDA,       \
                         std::string(what) + ": " + cudaGetErrorString(e_));                   \
    } while (0)

template <typename F>
cudaError_t by_storage_b(int storage, F &&fn) {
    switch (storage) {
    case IMB_STORE_FP32: return fn((float *)nullptr);
    case IMB_STORE_FP16: return fn((__half *)nullptr);
    case IMB_STORE_BF16: return fn((__nv_bfloat16 *)nullptr);
    default: return cudaErrorInvalidValue;
    }
}

template <typename S, int CPL, bool BLOCKED>
cudaError_t launch_step_t(imb_batch *b, int from) {
    auto k = k_batch_step<S, CPL, BLOCKED>;
    if (b->grid == 0) {   // resident blocks of this configuration (set before any capture)
        int per = 0, sms = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k, b->block, 0);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, b->device);
        const long long need = ((long long)b->nitems[CPL - 1] * 32 + b->block - 1) / b->block;
        b->grid = (int)std::max(1LL, std::min(need, (long long)std::max(per, 1) * sms));
        if (b->grid_only) return cudaSuccess;
    }
    if (b->grid_only) return cudaSuccess;
    k<<<b->grid, b->block, 0, b->stream>>>((const S *)b->buf[from], (S *)b->buf[from ^ 1], b->dom, b->ndom,
                                           b->nitems[CPL - 1], b->E, b->drag, b->err);
    return cudaGetLastError();
}

// largest block the kernel of this storage and cells-per-lane can launch (its registers)
int max_block(imb_batch *b) {
    int m = 0;
    by_storage_b(b->storage, [&](auto tag) {
        using S = std::remove_pointer_t<decltype(tag)>;
        cudaFuncAttributes fa{};
        cudaError_t e = !b->blocked   ? cudaFuncGetAttributes(&fa, k_batch_step<S, 1, false>)
                        : b->cpl == 2 ? cudaFuncGetAttributes(&fa, k_batch_step<S, 2, true>)
                                      : cudaFuncGetAttributes(&fa, k_batch_step<S, 1, true>);
        m = e == cudaSuccess ? fa.maxThreadsPerBlock : 0;
        return e;
    });
    return m;
}

cudaError_t launch_step(imb_batch *b, int from) {
    return by_storage_b(b->storage, [&](auto tag) {
        using S = std::remove_pointer_t<decltype(tag)>;
        return !b->blocked   ? launch_step_t<S, 1, false>(b, from)
               : b->cpl == 2 ? launch_step_t<S, 2, true>(b, from)
                             : launch_step_t<S, 1, true>(b, from);
    });
}

void drop_graphs(imb_batch *b) {
    for (auto &g : b->graph)
        if (g) {
            cudaGraphExecDestroy(g);
            g = nullptr;
        }
}

int batch_wait(imb_batch *b) {
    BCK(cudaStreamSynchronize(b->stream), "batch stream");
    unsigned bits = 0;
    BCK(cudaMemcpy(&bits, b->err, sizeof(bits), cudaMemcpyDeviceToHost), "error flags");
    if (bits & ERR_UNSTABLE) {
        cudaMemset(b->err, 0, sizeof(unsigned));
        return bfail(b, IMB_E_UNSTABLE, "NaN or |u| >= 0.3 in a batch domain (Mach guard)");
    }
    return IMB_OK;
}

}  // namespace

extern "C" int imb_batch_create(imb_batch **out, int n_domains, const int *nx, const int *ny, const double *tau,
                                const double *C_smag, const double *Fx, const double *Fy, const int *n_disks,
                                const double *disk_xy, const double *disk_r, int storage) {
    if (!out) return IMB_E_INVALID_ARG;
    *out = nullptr;
    if (n_domains < 1 || !nx || !ny || !tau || !C_smag || !Fx || !Fy || !n_disks || storage < 0 || storage > 2)
        return IMB_E_INVALID_ARG;
    auto *b = new imb_batch();
    b->storage = storage;
    b->elem = storage == IMB_STORE_FP32 ? 4 : 2;
    b->ndom = n_domains;
    double rmax = 0.0;
    size_t cells = 0, rows = 0, ragged = 0, e_cells = 0, most = 0, padded = 0;
    long long items = 0, items2 = 0;   // work items of 32 and of 64 cells
    const size_t G = storage == IMB_STORE_FP32 ? segb<float>() : segb<__half>();
    int ndisk = 0;
    for (int d = 0; d < n_domains; ++d) {
        if (nx[d] < 3 || ny[d] < 3 || 9.0 * nx[d] * ny[d] > 2147483647.0 || !(tau[d] > 0.5) ||
            !(C_smag[d] >= 0.0) || n_disks[d] < 0) {
            delete b;
            return IMB_E_INVALID_ARG;
        }
        BatchDomain D{};
        D.nx = nx[d];
        D.ny = ny[d];
        D.item0[0] = (int)items;
        D.item0[1] = (int)items2;
        D.tau = (float)tau[d];
        D.omega0 = (float)(1.0 / tau[d]);
        D.Fx = (float)Fx[d];
        D.Fy = (float)Fy[d];
        D.smag_coef = (float)(18.0 * std::sqrt(2.0) * C_smag[d] * C_smag[d]);
        b->hdom.push_back(D);
        cells += (size_t)nx[d] * ny[d];
        rows += (size_t)ny[d];
        if (nx[d] % 16) ragged += (size_t)ny[d];
        most = std::max(most, (size_t)nx[d] * ny[d]);
        padded += (nx[d] + G - 1) / G * G * ny[d];
        items += ((long long)ny[d] * nx[d] + 31) / 32;
        items2 += ((long long)ny[d] * ((nx[d] + 1) / 2) + 31) / 32;
        ndisk += n_disks[d];
    }
    if (ndisk > 0 && (!disk_xy || !disk_r)) {
        delete b;
        return IMB_E_INVALID_ARG;
    }
    std::vector<int> ddom(std::max(ndisk, 1));
    for (int d = 0, j = 0; d < n_domains; ++d)
        for (int k = 0; k < n_disks[d]; ++k, ++j) {
            ddom[j] = d;
            const double x = disk_xy[2 * j], y = disk_xy[2 * j + 1], r = disk_r[j];
            if (!(r > 0.0) || !(x >= 0.0 && x < nx[d] && y >= 0.0 && y < ny[d]) || 2.0 * r + 4.0 > std::min(nx[d], ny[d])) {
                delete b;
                return IMB_E_INVALID_ARG;
            }
            rmax = std::max(rmax, r);
        }
    const long long wd = 2LL * ((long long)std::ceil(rmax) + 1) + 1;   // the solid-ratio launch's box
    if (items > 2147483647LL || ((long long)ndisk * wd * wd + 127) / 128 > 2147483647LL) {
        delete b;
        return IMB_E_INVALID_ARG;
    }
    b->nitems[0] = (int)items;
    b->nitems[1] = (int)items2;
    b->ndisk = ndisk;
    b->cells = cells;
    cudaGetDevice(&b->device);
    size_t mem_free = 0, mem_total = 0;
    if (cudaMemGetInfo(&mem_free, &mem_total) != cudaSuccess) cudaGetLastError();
    b->blocked = blocked_rows(cells, rows, ragged, padded, most, (size_t)b->elem, mem_free);
    for (BatchDomain &D : b->hdom) {
        D.off = b->total;
        D.row = b->blocked ? (D.nx + G - 1) / G * 9 * G : (size_t)D.nx;
        D.plane = b->blocked ? 0 : D.nx * D.ny;
        D.e_off = e_cells;
        D.e_row = b->blocked ? (D.nx + 1) / 2 * 2 : D.nx;
        b->total += b->blocked ? D.row * D.ny : 9 * (size_t)D.plane;
        e_cells += (size_t)D.e_row * D.ny;
    }
    cudaError_t e;
    if ((e = cudaStreamCreateWithFlags(&b->stream, cudaStreamNonBlocking)) != cudaSuccess ||
        (e = cudaMalloc(&b->buf[0], b->total * b->elem)) != cudaSuccess ||
        (e = cudaMalloc(&b->buf[1], b->total * b->elem)) != cudaSuccess ||
        (e = cudaMalloc(&b->dom, sizeof(BatchDomain) * n_domains)) != cudaSuccess ||
        (e = cudaMalloc(&b->E, sizeof(float) * e_cells)) != cudaSuccess ||
        (e = cudaMalloc(&b->drag, sizeof(double) * 2 * n_domains)) != cudaSuccess ||
        (e = cudaMalloc(&b->err, sizeof(unsigned))) != cudaSuccess) {
        *out = b;
        return bfail(b, e == cudaErrorMemoryAllocation ? IMB_E_NOMEM : IMB_E_CUDA, "batch buffers");
    }
    *out = b;
    // fluid at rest with rho = 1: f = w, i.e. zero shifted populations
    BCK(cudaMemsetAsync(b->buf[0], 0, b->total * b->elem, b->stream), "clear");
    BCK(cudaMemsetAsync(b->buf[1], 0, b->total * b->elem, b->stream), "clear");
    BCK(cudaMemsetAsync(b->E, 0, sizeof(float) * e_cells, b->stream), "clear");
    BCK(cudaMemsetAsync(b->drag, 0, sizeof(double) * 2 * n_domains, b->stream), "clear");
    BCK(cudaMemsetAsync(b->err, 0, sizeof(unsigned), b->stream), "clear");
    BCK(cudaMemcpyAsync(b->dom, b->hdom.data(), sizeof(BatchDomain) * n_domains, cudaMemcpyHostToDevice, b->stream),
        "domains");
    if (ndisk > 0) {
        struct DiskArrays {   // freed on every return (cudaFree waits for the launch)
            int *dd = nullptr;
            double *xy = nullptr, *r = nullptr;
            ~DiskArrays() {
                if (dd) cudaFree(dd);
                if (xy) cudaFree(xy);
                if (r) cudaFree(r);
            }
        } t;
        BCK(cudaMalloc(&t.dd, sizeof(int) * ndisk), "disks");
        BCK(cudaMalloc(&t.xy, sizeof(double) * 2 * ndisk), "disks");
        BCK(cudaMalloc(&t.r, sizeof(double) * ndisk), "disks");
        BCK(cudaMemcpyAsync(t.dd, ddom.data(), sizeof(int) * ndisk, cudaMemcpyHostToDevice, b->stream), "disks");
        BCK(cudaMemcpyAsync(t.xy, disk_xy, sizeof(double) * 2 * ndisk, cudaMemcpyHostToDevice, b->stream), "disks");
        BCK(cudaMemcpyAsync(t.r, disk_r, sizeof(double) * ndisk, cudaMemcpyHostToDevice, b->stream), "disks");
        const int span = (int)std::ceil(rmax) + 1, w = 2 * span + 1;
        const long long nthreads = (long long)ndisk * w * w;   // grid size checked at validation
        k_batch_solid<<<(unsigned)((nthreads + 127) / 128), 128, 0, b->stream>>>(b->dom, t.dd, t.xy, t.r, ndisk,
                                                                               span, b->E);
        BCK(cudaGetLastError(), "solid ratio");
        BCK(cudaStreamSynchronize(b->stream), "solid ratio");
    }
    return batch_wait(b);
}

extern "C" int imb_batch_run(imb_batch *b, int steps) {
    if (!b) return IMB_E_INVALID_ARG;
    if (steps < 0) return bfail(b, IMB_E_INVALID_ARG, "steps must be >= 0");
    BCK(cudaSetDevice(b->device), "cudaSetDevice");
    for (int s = 0; s + 1 < steps; s += 2) {
        cudaGraphExec_t &g = b->graph[b->cur];
        if (!g) {   // two steps from the current buffer, captured once
            if (b->grid == 0) {
                b->grid_only = true;
                launch_step(b, b->cur);
                b->grid_only = false;
            }
            cudaGraph_t gr;
            BCK(cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal), "capture");
            cudaError_t e1 = launch_step(b, b->cur);
            cudaError_t e2 = launch_step(b, b->cur ^ 1);
            BCK(cudaStreamEndCapture(b->stream, &gr), "capture");
            BCK(e1, "capture launch");
            BCK(e2, "capture launch");
            BCK(cudaGraphInstantiate(&g, gr, 0), "graph");
            cudaGraphDestroy(gr);
        }
        BCK(cudaGraphLaunch(g, b->stream), "graph launch");
    }
    if (steps % 2) {
        BCK(launch_step(b, b->cur), "batch step");
        b->cur ^= 1;
    }
    b->steps_run += steps;
    return batch_wait(b);
}

extern "C" int imb_batch_autotune(imb_batch *b, int steps_per_trial, int *block, int *cells_per_lane,
                                  double *best_ms_per_step) {
    if (!b || steps_per_trial < 1) return IMB_E_INVALID_ARG;
    BCK(cudaSetDevice(b->device), "cudaSetDevice");
    // work on a copy of the state, put it back afterwards
    void *save = nullptr;
    BCK(cudaMalloc(&save, b->total * b->elem), "autotune copy");
    BCK(cudaMemcpyAsync(save, b->buf[b->cur], b->total * b->elem, cudaMemcpyDeviceToDevice, b->stream), "copy");
    double *dsave = nullptr;
    BCK(cudaMalloc(&dsave, sizeof(double) * 2 * b->ndom), "autotune copy");
    BCK(cudaMemcpyAsync(dsave, b->drag, sizeof(double) * 2 * b->ndom, cudaMemcpyDeviceToDevice, b->stream), "copy");
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    const int blocks[3] = {128, 256, 512}, cpls[2] = {1, 2};
    float best = 1e30f;
    int bb = b->block, bc = b->cpl;
    for (int bl : blocks)
        for (int cp : cpls) {
            if (cp == 2 && !b->blocked) continue;   // whole planes: one cell per lane either way
            b->block = bl;
            b->cpl = cp;
            b->grid = 0;
            if (max_block(b) < bl) continue;   // too many registers for this block size
            int from = b->cur;
            BCK(launch_step(b, from), "trial");   // warm-up
            from ^= 1;
            cudaEventRecord(e0, b->stream);
            for (int s = 0; s < steps_per_trial; ++s, from ^= 1) BCK(launch_step(b, from), "trial");
            cudaEventRecord(e1, b->stream);
            BCK(cudaEventSynchronize(e1), "trial");
            float ms = 0.0f;
            cudaEventElapsedTime(&ms, e0, e1);
            if (ms < best) {
                best = ms;
                bb = bl;
                bc = cp;
            }
            BCK(cudaMemcpyAsync(b->buf[b->cur], save, b->total * b->elem, cudaMemcpyDeviceToDevice, b->stream),
                "restore");
        }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    b->block = bb;
    b->cpl = bc;
    b->grid = 0;
    drop_graphs(b);
    BCK(cudaMemcpyAsync(b->drag, dsave, sizeof(double) * 2 * b->ndom, cudaMemcpyDeviceToDevice, b->stream), "copy");
    BCK(cudaStreamSynchronize(b->stream), "autotune");
    cudaFree(save);
    cudaFree(dsave);
    BCK(cudaMemset(b->err, 0, sizeof(unsigned)), "clear");
    if (block) *block = bb;
    if (cells_per_lane) *cells_per_lane = bc;
    if (best_ms_per_step) *best_ms_per_step = best / steps_per_trial;
    return IMB_OK;
}

extern "C" int imb_batch_set_launch(imb_batch *b, int block, int cells_per_lane) {
    if (!b) return IMB_E_INVALID_ARG;
    if ((block != 128 && block != 256 && block != 512) || (cells_per_lane != 1 && cells_per_lane != 2))
        return bfail(b, IMB_E_INVALID_ARG, "block must be 128, 256 or 512 and cells_per_lane 1 or 2");
    BCK(cudaSetDevice(b->device), "cudaSetDevice");
    const int old_block = b->block, old_cpl = b->cpl;
    b->cpl = cells_per_lane;
    if (max_block(b) < block) {
        b->cpl = old_cpl;
        return bfail(b, IMB_E_INVALID_ARG, "the kernel cannot launch blocks of this size");
    }
    if (block != old_block || cells_per_lane != old_cpl) {
        BCK(cudaStreamSynchronize(b->stream), "batch stream");
        b->block = block;
        b->grid = 0;
        drop_graphs(b);
    }
    return IMB_OK;
}

extern "C" int imb_batch_mean_drag(imb_batch *b, double *Fx_mean, double *Fy_mean) {
    if (!b || !Fx_mean || !Fy_mean) return IMB_E_INVALID_ARG;
    int rc = batch_wait(b);
    if (rc) return rc;
    std::vector<double> h(2 * (size_t)b->ndom);
    BCK(cudaMemcpy(h.data(), b->drag, sizeof(double) * h.size(), cudaMemcpyDeviceToHost), "drag");
    const double n = b->steps_run > 0 ? (double)b->steps_run : 1.0;
    for (int d = 0; d < b->ndom; ++d) {
        Fx_mean[d] = h[2 * d] / n;
        Fy_mean[d] = h[2 * d + 1] / n;
    }
    return IMB_OK;
}

extern "C" int imb_batch_get_populations(imb_batch *b, int domain, double *f) {
    if (!b || !f || domain < 0 || domain >= b->ndom) return IMB_E_INVALID_ARG;
    int rc = batch_wait(b);
    if (rc) return rc;
    const size_t cells = (size_t)b->hdom[domain].nx * b->hdom[domain].ny, n = 9 * cells;
    double *t = nullptr;
    BCK(cudaMalloc(&t, sizeof(double) * n), "readback buffer");
    cudaError_t e = by_storage_b(b->storage, [&](auto tag) {
        using S = std::remove_pointer_t<decltype(tag)>;
        k_batch_gather<S><<<(unsigned)((cells + 255) / 256), 256, 0, b->stream>>>(
            (const S *)b->buf[b->cur], b->dom, domain, t);
        return cudaGetLastError();
    });
    if (e == cudaSuccess) e = cudaMemcpyAsync(f, t, sizeof(double) * n, cudaMemcpyDeviceToHost, b->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
    cudaFree(t);
    BCK(e, "populations");
    return IMB_OK;
}

extern "C" long long imb_batch_cells(const imb_batch *b) {
    return b ? (long long)b->cells : 0;
}

extern "C" const char *imb_batch_last_error(const imb_batch *b) {
    return b ? b->last_error.c_str() : "null batch";
}

extern "C" void imb_batch_destroy(imb_batch *b) {
    if (!b) return;
    cudaSetDevice(b->device);
    if (b->stream) cudaStreamSynchronize(b->stream);
    drop_graphs(b);
    cudaFree(b->buf[0]);
    cudaFree(b->buf[1]);
    cudaFree(b->dom);
    cudaFree(b->E);
    cudaFree(b->drag);
    cudaFree(b->err);
    if (b->stream) cudaStreamDestroy(b->stream);
    delete b;
}
