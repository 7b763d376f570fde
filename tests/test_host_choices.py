"""Decisions the host takes before a launch (csrc/imb_host.h) and the sums and the division that keep their
bits (csrc/imb_sums.h), compiled with the host compiler and checked without a GPU."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1809_07008_gb300", "csrc")


def run_cpp(tmp_path, body):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text('#include "imb_host.h"\n#include "imb_sums.h"\n#include <cstdio>\n#include <cstdlib>\nusing namespace imb;\n'
                   '#define CHECK(c) do { if (!(c)) { std::printf("failed: %s\\n", #c); std::exit(1); } } while (0)\n' + body)
    subprocess.run([cxx, "-std=c++17", "-O2", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_adjoint_blocks_hold_the_edge_columns_together(tmp_path):
    # every width a lattice can have (3 rows at least): each column in one block, 0 beside 1, nx - 2 beside
    # nx - 1 (also where every multiple of 32 up to 256 leaves one column: nx = 1 modulo 26880)
    run_cpp(tmp_path, """
int main() {
    for (int nx = 3; nx <= (1 << 27) / 3; ++nx)
        for (int inlet = 0; inlet < 2; ++inlet) {
            const AdjointGrid g = adjoint_grid(nx, inlet);
            auto block = [&](int x) { return (x + g.shift) / ADJ_BLOCK; };
            CHECK(g.shift >= 0 && g.shift < ADJ_BLOCK);
            CHECK(g.blocks > 0 && block(nx - 1) == g.blocks - 1 && block(0) == 0);
            if (inlet) CHECK(block(1) == 0 && block(nx - 2) == g.blocks - 1);
        }
}
""")


def test_pinned_span_decision(tmp_path):
    # an array is written in place only where it is aligned and one memory range holds all of it
    run_cpp(tmp_path, """
int main() {
    const uintptr_t s = 0x10000;                                  // the range [s, s + 4096)
    CHECK(span_covered(s, 4096, 8, s, 4096));
    CHECK(span_covered(s + 4088, 8, 8, s, 4096));
    CHECK(!span_covered(s, 4097, 8, s, 4096));
    CHECK(!span_covered(s + 8, 4096, 8, s, 4096));
    CHECK(!span_covered(s - 8, 16, 8, s, 4096));
    CHECK(!span_covered(s, 8192, 8, s, 4096));                    // ends in a second registration
    CHECK(!span_covered(s + 4, 64, 8, s, 4096));                  // not on a multiple of 8
    CHECK(!span_covered(s + 4100, 0, 4, s, 4096) && !span_covered(s, 0, 8, s, 4096));
    CHECK(!span_covered(s + 8, SIZE_MAX - 7, 8, s, 4096));        // no wrap-around
    CHECK(!span_covered(s, 8, 8, 0, 0));                          // memory the driver doesn't know
    const char *b = (const char *)s;
    const void *apart[] = {b, b + 64, b + 128}, *meet[] = {b, b + 64, b + 120}, *twice[] = {b, b + 64, b + 64};
    CHECK(spans_disjoint(apart, 3, 64) && !spans_disjoint(meet, 3, 64) && !spans_disjoint(twice, 3, 64));
}
""")


def test_div_by_equals_division(tmp_path):
    # random significands at the edges of the windows of both operands, within and beyond them, zeros,
    # infinities, NaN and subnormal values: the quotient of the division, to the bit
    run_cpp(tmp_path, """
#include <random>
static uint64_t bits(double v) { uint64_t b; std::memcpy(&b, &v, 8); return b; }
static bool same(double a, double b) {
    const double q = div_by(a, b, 1.0 / b), d = a / b;
    return bits(q) == bits(d) || (q != q && d != d);
}
int main() {
    std::mt19937_64 g(1);
    auto real = [&](int e) {   // significand with few or many bits, exponent e
        uint64_t m = g() >> 12;
        if (g() & 1) m &= ~0ull << (g() % 52);
        if (g() & 1) m |= 0xfffffffffffffull >> (g() % 52);
        return std::ldexp(1.0 + (double)(m & 0xfffffffffffffull) * 0x1p-52, e);
    };
    const int edge[] = {-1022, -823, -700, -401, -400, -399, -60, -1, 0, 1, 40, 398, 399, 400, 401, 500, 700, 776, 1023};
    for (int ea : edge)
        for (int eb : edge)
            for (int k = 0; k < 4000; ++k) {
                const double a = real(ea), b = real(eb);
                CHECK(same(a, b) && same(-a, b));
            }
    for (int k = 0; k < 20000000; ++k) CHECK(same(real((int)(g() % 60) - 30), real((int)(g() % 40))));
    const double odd[] = {0.0, -0.0, (double)INFINITY, -(double)INFINITY, (double)NAN, 5e-324, 1e-310};
    for (double a : odd)
        for (int eb : edge) CHECK(same(a, real(eb)));
    for (double a : odd)
        for (double b : {(double)INFINITY, 5e-324, 1e-310}) CHECK(same(a, b) && same(1.5, b));
}
""")


def test_batch_layout_leaves_room(tmp_path):
    # whatever batch and free memory: a batch whose unpadded buffers fit (two with the read-back, or three)
    # fits in the layout it is given; rows of at least 100 cells, and of 32 or more where
    # they fill their sectors, are blocked where memory allows, narrow ones not
    run_cpp(tmp_path, """
#include <random>
int main() {
    std::mt19937_64 g(3);
    auto log_uniform = [&](double lo, double hi) { return lo * std::pow(hi / lo, (double)(g() >> 11) * 0x1p-53); };
    for (int k = 0; k < 2000000; ++k) {
        const size_t nx = (size_t)log_uniform(3, 5000), ny = (size_t)log_uniform(3, 5000), n = (size_t)log_uniform(1, 1e5);
        const size_t elem = g() & 1 ? 4 : 2, G = 128 / elem, w = (nx + G - 1) / G * G;
        const size_t cells = n * nx * ny, rows = n * ny, padded = n * w * ny, mem = (size_t)log_uniform(1e8, 3e11);
        const bool b = blocked_rows(cells, rows, nx % 16 ? rows : 0, padded, nx * ny, elem, mem);
        const size_t c = b ? padded : cells;
        const double slack = 1e6;   // what a few tables take
        if (2.0 * 9 * cells * elem + 4.0 * cells + 72.0 * nx * ny <= (double)mem)
            CHECK(2.0 * 9 * c * elem + 4.0 * (b ? n * ny * ((nx + 1) / 2 * 2) : cells) + 72.0 * nx * ny <= (double)mem + slack);
        if (3.0 * 9 * cells * elem + 4.0 * cells <= (double)mem)
            CHECK(3.0 * 9 * c * elem + 4.0 * (b ? n * ny * ((nx + 1) / 2 * 2) : cells) <= (double)mem + slack);
        if ((nx >= 100 || (nx >= 32 && nx % 16 == 0)) && 3.0 * 9 * padded * elem + 4.0 * padded + 72.0 * nx * ny < (double)mem - 1e8) CHECK(b);
        if (nx < 8) CHECK(!b);
    }
}
""")


def test_asked_once_for_every_device(tmp_path):
    # each device gets its own answer, asked once, whichever thread comes first
    run_cpp(tmp_path, """
#include <atomic>
#include <thread>
#include <vector>
int main() {
    static PerDevice<int, 4> v;
    std::atomic<int> asked[6] = {};
    std::vector<std::thread> t;
    for (int k = 0; k < 16; ++k)
        t.emplace_back([&] {
            for (int d = 0; d < 6; ++d) CHECK(v.get(d, [&] { ++asked[d]; return 10 + d; }) == 10 + d);
        });
    for (auto &x : t) x.join();
    for (int d = 0; d < 4; ++d) CHECK(asked[d] == 1);
    CHECK(asked[4] == 16 && asked[5] == 16);   // beyond the table: asked every time
}
""")


def test_sums_in_three_parts(tmp_path):
    # eight FP32 terms of any exponents and signs, cancelling ones among them: no further from the exact sum
    # than one FP64 rounding of it and 2^-68 of the terms; NaN, infinities and sums beyond FP32 as in FP64
    run_cpp(tmp_path, """
#include <random>
#if defined(__x86_64__)
typedef __float128 Quad;
#else
typedef long double Quad;   // 113 bits on Arm
#endif
static bool same(double a, double b) { return a == b || (a != a && b != b); }
int main() {
    std::mt19937_64 g(5);
    auto term = [&](int spread) {
        const float m = 1.0f + (float)(g() >> 41) * 0x1p-23f;
        return std::ldexp(g() & 1 ? m : -m, (int)(g() % (2 * spread + 1)) - spread);
    };
    for (int spread : {0, 2, 8, 24, 40})
        for (int k = 0; k < 1000000; ++k) {
            float v[8];
            for (float &x : v) x = term(spread);
            if (k % 3 == 0) v[7] = -v[0], v[6] = -v[1];
            if (k % 5 == 0) v[2] = 0.0f;
            Quad exact = 0, size = 0;
            Sum3 a, b;
            for (int i = 0; i < 8; ++i) {
                exact += v[i];
                size += std::fabs(v[i]);
                (i < 4 ? a : b).add(v[i]);
            }
            a.add(b);   // as lanes are joined
            for (double got : {sum_terms<8>(v), a.value()}) {
                Quad err = got - exact, bar = exact * 0x1.02p-53 + 0;
                if (err < 0) err = -err;
                if (bar < 0) bar = -bar;
                CHECK(err <= bar + size * 0x1p-68);
            }
        }
    const float inf = INFINITY, big = 3.0e38f;
    const float cases[][8] = {{1, inf, 2, 3, 4, 5, 6, 7}, {1, -inf, 2, 3, 4, 5, 6, 7}, {inf, 0, 0, -inf, 0, 0, 0, 0},
                              {1, NAN, 0, 0, 0, 0, 0, 0}, {big, big, big, 1, 0, 0, 0, 0}, {big, big, -big, -big, 5, 0, 0, 0},
                              {inf, 0, 0, 0, 0, 0, 0, 0}, {0, 0, 0, 0, 0, 0, 0, 0}};
    for (auto &c : cases) {
        double d = 0.0;
        for (float x : c) d += x;
        CHECK(same(sum_terms<8>(c), d));
    }
}
""")


def test_sums_joined_over_a_warp(tmp_path):
    # 32 lanes of two terms each, joined over a butterfly as the reverse step does: every lane ends with the
    # exact sum to one FP64 rounding and 2^-66 of the terms (FP64 additions: 2^-53 a level; a pair of FP32
    # parts is 2^-46 off and fails)
    run_cpp(tmp_path, """
#include <random>
#if defined(__x86_64__)
typedef __float128 Quad;
#else
typedef long double Quad;
#endif
int main() {
    std::mt19937_64 g(7);
    for (int spread : {0, 3, 12, 30})
        for (int k = 0; k < 20000; ++k) {
            Sum3 s[32];
            Quad exact = 0, size = 0;
            for (auto &lane : s)
                for (int i = 0; i < 2; ++i) {
                    const float m = 1.0f + (float)(g() >> 41) * 0x1p-23f;
                    const float x = std::ldexp(g() & 1 ? m : -m, (int)(g() % (2 * spread + 1)) - spread);
                    lane.add(x);
                    exact += x;
                    size += std::fabs(x);
                }
            for (int o = 16; o > 0; o >>= 1) {
                Sum3 n[32];
                for (int l = 0; l < 32; ++l) n[l] = s[l], n[l].add(s[l ^ o]);
                for (int l = 0; l < 32; ++l) s[l] = n[l];
            }
            for (auto &lane : s) {
                Quad err = lane.value() - exact, bar = exact * 0x1.02p-53;
                if (err < 0) err = -err;
                if (bar < 0) bar = -bar;
                CHECK(lane.finite() && err <= bar + size * 0x1p-66);
            }
        }
}
""")


def test_cluster_limit(tmp_path):
    # never beyond what the cluster holds, never less with more sub-cycles, all of it from twelve on
    run_cpp(tmp_path, """
int main() {
    CHECK(cluster_limit(1) == 1000 && cluster_limit(12) == CLUSTER_PARTICLES && cluster_limit(1 << 20) == CLUSTER_PARTICLES);
    for (int n = 1; n < 1000; ++n) CHECK(cluster_limit(n) <= cluster_limit(n + 1) && cluster_limit(n) <= CLUSTER_PARTICLES);
}
""")
