"""Fixed-point arithmetic of the double-precision passes (csrc/fx_math.cuh), on
the host: table twiddles, products with them, the butterflies' constant
rotations and the conversions, each against long double.

Bounds, in units of the last place of a result: a product leaves out low x low
terms (below 1/4 each, two of them) and rounds once (1/2), and its factor is off
by up to 4.5 units of 2^-62 (table: 4 from the series, 1/2 from rounding) or
2^-65 (constants) of a value below 2^61.5; a conversion to double is correctly
rounded up to ties, one from double is cut."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2202_12756_gb300", "csrc")

PROGRAM = r"""
#include "fx_math.cuh"
#include <cmath>
#include <cstdio>
#include <random>
using namespace fft3d;
typedef long double LD;
static const LD pi = 3.14159265358979323846264338327950288L;
static std::mt19937_64 rng(7);
// below 2^bits, every fourth at the ends of the range
static int64_t draw(int bits)
{
    const int64_t top = (1LL << bits) - 1, r = (int64_t)(rng() >> (63 - bits)) - (1LL << bits);
    const int k = (int)(rng() & 7);
    return k == 0 ? top : k == 1 ? -top : (r < -top ? -top : r);
}
static LD off(fxc q, fxc z, LD c, LD s)  // against z (c + i s)
{
    return fmaxl(fabsl(q.x - (z.x * c - z.y * s)), fabsl(q.y - (z.x * s + z.y * c)));
}
template <int P> static LD rot()
{
    LD w = 0;
    for (int i = 0; i < 20000; ++i) {
        const fxc z = fx_make(draw(60), draw(60));
        const LD a = -2 * pi * P / 96;
        w = fmaxl(w, off(fx_rot96<P>(z), z, cosl(a), sinl(a)));
    }
    if constexpr (P < 95) return fmaxl(w, rot<P + 1>());
    return w;
}
int main()
{
    LD tw = 0, mul = 0, w8 = 0;
    long long bad = 0;
    for (uint32_t d : {2u, 3u, 8u, 96u, 512u, 768u, 1024u, 1536u, 2048u, 4096u})
        for (uint32_t p = 0; p < d; ++p) {
            int64_t c, s;
            fx_cossin(p, d, &c, &s);
            const LD a = 2 * pi * p / d;
            tw = fmaxl(tw, fmaxl(fabsl(c - ldexpl(cosl(a), 62)), fabsl(s - ldexpl(sinl(a), 62))));
            for (int sh = 2; sh <= 5; ++sh) {
                const fxtw w = fx_twiddle(p, d, sh);
                if (w.xl == INT32_MIN || w.yl == INT32_MIN) ++bad;
                if (fabsl(fx_twiddle_value(w.xh, w.xl, sh) - cosl(a)) > 1.2e-16L) ++bad;
                const fxc z = fx_make(draw(61), draw(61));
                mul = fmaxl(mul, off(cmul(z, w), z, ldexpl(cosl(a), -sh), ldexpl(-sinl(a), -sh)));
                mul = fmaxl(mul, off(cmulc(z, w), z, ldexpl(cosl(a), -sh), ldexpl(sinl(a), -sh)));
            }
        }
    for (int i = 0; i < 100000; ++i) {
        const fxc z = fx_make(draw(60), draw(60));
        const LD r = sqrtl(0.5L);
        w8 = fmaxl(w8, fmaxl(off(w8_1(z), z, r, -r), off(w8_3(z), z, -r, -r)));
    }
    for (int i = 0; i < 400000; ++i) {
        const int64_t X = draw(61) >> (rng() % 62);
        const int e = (int)(rng() % 1900) - 1000;
        const LD t = ldexpl((LD)X, e);
        int32_t big = -1;
        const double a = fx_to(X, e), b = fx_to_big(X, e, big);
        if ((big < 0) != (X >= (1LL << 32) || X < -(1LL << 32))) ++bad;
        // half a unit of the 53-bit result
        if (fabsl(a - t) > fabsl(t) * 0x1.0001p-53L || (big < 0 && fabsl(b - t) > fabsl(t) * 0x1.0001p-53L)) ++bad;
        const int g = 128 + (int)(rng() % 1700);
        const double v = ldexp((double)(draw(53)), g - 1023 - 53 - (int)(rng() % 80));
        if (fx_from(v, g, 61) != (int64_t)truncl(ldexpl((LD)v, 1023 + 61 - g))) ++bad;
        // the scale code's power of two lies above the value and within a factor 4 of it
        const float f = fx_mag(fx_top(v), fx_top(v) & 0x7ff00000);
        const int code = fx_code(fx_top(v), f);
        if (v != 0 && !(fabsl((LD)v) < ldexpl(1, code - 1023) && ldexpl(1, code - 1025) < fabsl((LD)v))) ++bad;
    }
    if (fx_to(0, 5) != 0.0 || fx_from(0.0, 1023, 61) != 0 || fx_from(-0.0, 1023, 61) != 0) ++bad;
    if (fx_code(fx_top(HUGE_VAL), 1.f) != kFxBad || fx_code(fx_top(nan("")), 1.f) != kFxBad || fx_code(0, 64.f) != 0) ++bad;
    printf("%.4Lf %.4Lf %.4Lf %.4Lf %lld\n", tw, mul, rot<0>(), w8, bad);
    return 0;
}
"""


def test_fixed_point_arithmetic_against_long_double(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src, exe = tmp_path / "fx.cu", tmp_path / "fx"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)], check=True,
                   capture_output=True, timeout=300)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=120).stdout.split()
    tw, mul, rot, w8, bad = (float(v) for v in out)
    assert tw <= 4.5          # units of 2^-62
    assert mul <= 0.5 + 2 * 0.25 + 2 * 4.5 / 4 + 0.1  # two table components, their scale 2^-2 at most
    assert rot <= 0.5 + 2 * 0.25 + 0.5
    assert w8 <= 0.5 + 0.25 + 0.5
    assert bad == 0
