"""Scale codes of double lines at the lower end of the exponent range
(csrc/fx_math.cuh), on the host: of the lines whose values lie below 2^-895 only one of
zeros is transformed in fixed point."""
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
using namespace fft3d;
template <int N> static bool fixed(const double2 *v)
{
    const int g = fx_thread_code<N>(v);
    return fx_in_range(g) || !fx_unfit<N>(g, v);
}
template <int N> static int wrong()
{
    int bad = 0;
    double2 v[N];
    for (double2 &z : v) z = make_double2(0.0, -0.0);
    if (fx_thread_code<N>(v) != 0 || !fixed<N>(v)) ++bad;
    for (int k = -1074; k <= -1000; ++k)
        for (int i = 0; i < 2 * N; ++i)
            for (int s = -1; s <= 1; s += 2) {
                for (double2 &z : v) z = make_double2(0.0, -0.0);
                (i < N ? v[i].x : v[i - N].y) = ldexp(s, k);
                if (fixed<N>(v)) ++bad;
            }
    // beside an ordinary value a subnormal one makes no difference
    for (double2 &z : v) z = make_double2(0.0, 0.0);
    v[0].x = 1.0;
    const int g = fx_thread_code<N>(v);
    v[0].y = ldexp(1.0, -1074);
    if (fx_thread_code<N>(v) != g || !fixed<N>(v)) ++bad;
    return bad;
}
int main()
{
    printf("%d\n", wrong<1>() + wrong<8>() + wrong<9>() + wrong<16>() + wrong<24>());
    return 0;
}
"""


def test_subnormal_lines_are_not_lines_of_zeros(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src, exe = tmp_path / "sub.cu", tmp_path / "sub"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)], check=True,
                   capture_output=True, timeout=300)
    assert int(subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=120).stdout) == 0
