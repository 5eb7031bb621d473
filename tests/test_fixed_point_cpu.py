"""The integer arithmetic of the FP64 path (esdg_fixed.cuh), compiled for the host."""

import os
import shutil
import subprocess

import pytest

from paper_2005_02516_gb300 import _build


def _run(tmp_path, program):
    if not (shutil.which("nvcc") or os.path.exists("/usr/local/cuda/bin/nvcc")):
        pytest.skip("no CUDA compiler")
    src, exe = tmp_path / "t.cu", tmp_path / "t"
    src.write_text('#include "esdg_fixed.cuh"\n#include <cmath>\n#include <cstdio>\n#include <cstdlib>\n#include <random>\n'
                   "using namespace esdg;\n#define CHECK(c) if (!(c)) { printf(\"line %d: %s\\n\", __LINE__, #c); return 1; }\n"
                   + program)
    subprocess.run([_build.nvcc(), "-std=c++17", "-O1", *_build.ARCH, "-I", _build.CSRC, str(src), "-o", str(exe)],
                   check=True)
    p = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert p.returncode == 0, p.stdout


def test_larger_speed_keeps_a_nan_of_either_sign(tmp_path):
    _run(tmp_path, r"""
int main() {
    const double nan = fx_double(0x7ff8000000000000ll), minus_nan = fx_double((long long)0xfff8000000000000ull);
    for (double n : {nan, minus_nan})
        for (double x : {0.0, 1.0, HUGE_VAL, 5e-324}) {
            CHECK(std::isnan(r_max_nonneg(n, x)));
            CHECK(std::isnan(r_max_nonneg(x, n)));
        }
    const double v[] = {0.0, 5e-324, 1e-300, 0.5, 1.0, 1.0 + 0x1p-52, 1e300, HUGE_VAL};
    for (double a : v)
        for (double b : v) CHECK(r_max_nonneg(a, b) == (a > b ? a : b));
    return 0;
}
""")


def test_sums_of_products_stay_within_their_bound(tmp_path):
    """n <= 43 products of values of 58 bits with an operator row of 58 (59) bits: the
    sum against exact integers, within n / 4 + 1 units of 2^56, and the two 64-bit
    sums within 63 bits; with random operands, and with the operands of the largest
    dropped low products and of the fullest cross sum."""
    _run(tmp_path, r"""
static std::mt19937_64 rng(20050251);
static long long below(long long m) { return (long long)(rng() % (uint64_t)(2 * m - 1)) - (m - 1); }
typedef __int128 wide;
static wide size(wide x) { return x < 0 ? -x : x; }

static int check(int n, const long long* v, const long long* q) {
    FxSum s = {0, 0};
    wide exact = 0, hh = 0, mid = 0;
    for (int i = 0; i < n; ++i) {
        const int2 a = fx_limbs(v[i]), b = fx_limbs(q[i]);
        CHECK((long long)a.y * (1ll << FX_LO) + a.x == v[i] && std::abs((long long)a.x) <= 1ll << (FX_LO - 1));
        fx_mac(s, a, b);
        exact += (wide)v[i] * q[i];
        hh += (wide)a.y * b.y;
        mid += (wide)a.x * b.y + (wide)a.y * b.x;
        CHECK(size(hh) < (wide)1 << 63 && size(mid) < (wide)1 << 63);
    }
    CHECK((wide)s.hh == hh && (wide)s.mid == mid);
    const wide off = (wide)fx_value(s) * ((wide)1 << 56) - exact;
    CHECK(size(off) <= ((wide)n << 54) + ((wide)1 << 56));
    return 0;
}

int main() {
    long long v[43], q[43];
    for (int n : {1, 6, 15, 21, 31, 42, 43})
        for (int bits : {FX_ROW, FX_PAIR})
            for (int trial = 0; trial < 3000; ++trial) {
                // a row whose absolute values sum to less than 2^bits, one entry at most half of it
                double w[43], sum = 0;
                for (int i = 0; i < n; ++i) sum += w[i] = std::exp(-8.0 * (trial % 3) * (rng() % 1000) / 1000.0);
                for (int i = 0; i < n; ++i) {
                    const long long most = (long long)(std::fmin(w[i] / sum, 0.5) * std::ldexp(1.0, bits) * 0.999);
                    v[i] = below(1ll << FX_VAL);
                    q[i] = (rng() & 1 ? 1 : -1) * most;
                    if (trial % 2) {  // low limbs of the largest size, of one sign of their product
                        v[i] = (v[i] & ~((1ll << FX_LO) - 1)) + (1ll << (FX_LO - 1)) - 1;
                        q[i] = (q[i] & ~((1ll << FX_LO) - 1)) + (1ll << (FX_LO - 1)) - 1;
                    }
                    if (trial % 5 == 4) {  // the fullest sum of cross products
                        v[i] = ((1ll << (FX_VAL - FX_LO)) - 1) * (1ll << FX_LO) - (1ll << (FX_LO - 1));
                        q[i] = (q[i] & ~((1ll << FX_LO) - 1)) - (1ll << (FX_LO - 1));
                    }
                }
                if (check(n, v, q)) return 1;
            }
    return 0;
}
""")


def test_pair_term_and_conversions_stay_within_their_bounds(tmp_path):
    """T within 3/4 of its unit of the exact integer sum and within its limbs; a
    double through a scale and back to half a unit, over the exponent range."""
    _run(tmp_path, r"""
static std::mt19937_64 rng(20050251);
static long long below(long long m) { return (long long)(rng() % (uint64_t)(2 * m - 1)) - (m - 1); }
typedef __int128 wide;

int main() {
    for (int trial = 0; trial < 200000; ++trial) {
        const int sx = trial % 4 ? 0 : rng() % 40, sy = trial % 4 != 1 ? 0 : rng() % 40;
        const long long qx = below(1ll << 58) >> sx, qy = below(1ll << 58) >> sy;
        const long long h[4] = {below(1ll << FX_MOM), below(1ll << FX_MOM), below(1ll << FX_MOM), below(1ll << FX_MOM)};
        const int2 a = fx_limbs(h[0]), b = fx_limbs(h[1]), c = fx_limbs(h[2]), d = fx_limbs(h[3]);
        const long long t = fx_pair_t(fx_limbs(qx), fx_limbs(qy), make_int2(a.x + b.x, a.y + b.y),
                                      make_int2(c.x + d.x, c.y + d.y));
        const wide exact = (wide)qx * (h[0] + h[1]) + (wide)qy * (h[2] + h[3]);
        wide off = (wide)t * ((wide)1 << 59) - exact;
        if (off < 0) off = -off;
        CHECK(4 * off <= (wide)3 << 59);
        CHECK(std::abs(t) <= (1ll << 58) + 2);
        const int2 l = fx_limbs(t);
        CHECK((long long)l.y * (1ll << FX_LO) + l.x == t);
    }
    for (int x = -1100; x <= 1100; ++x) CHECK(fx_pack_x(fx_pack(x, -x)) == x && fx_pack_y(fx_pack(x, -x)) == -x);
    for (int trial = 0; trial < 400000; ++trial) {
        double x = fx_double((long long)rng());
        if (trial % 3 == 0) x = std::ldexp(x, -1074 - std::ilogb(x) + (int)(rng() % 60));  // about the subnormals
        const int e = fx_exp(x);
        if (e == FX_NONFINITE) continue;
        const int X = fx_scale(e) + (int)(rng() % 60);
        const long long v = fx_from<FX_VAL>(x, X);
        // |v - x 2^(58 - X)| <= 1/2, formed without leaving the range of a double
        const double y = std::ldexp(std::ldexp(x, 600 * (X < 0) - 600 * (X > 0)), FX_VAL - X - 600 * (X < 0) + 600 * (X > 0));
        CHECK(std::fabs((double)v - y) <= 0.5);
        // and back: round(v 2^(X - 58)) to a double, here exact whenever v has 53 bits
        double back;
        fx_to<1>(&v, [&](int) { return X - FX_VAL; }, &back);
        const double want = std::ldexp((double)v, X - FX_VAL);
        CHECK(back == want || std::fabs(back - want) <= std::fabs(want) * 0x1p-52 || std::fabs(back - want) <= 5e-324);
    }
    const long long big = 1ll << 58, zero = 0;
    double x[2];
    fx_to<1>(&big, [](int) { return 1000; }, x);
    CHECK(std::isinf(x[0]));
    fx_to<1>(&zero, [](int) { return -5000; }, x);
    CHECK(x[0] == 0);
    return 0;
}
""")
