"""fast_div and div_by of the library's own header, compiled for the host: the
division by a grid size that cell coordinates, segments and row offsets go through,
at the quotients where a wrong multiplier, shift or truncation shows."""
import os
import subprocess

import pytest

MAIN = r"""
#include <cstdio>
#include <cstdlib>
#include "fsl_internal.cuh"
int main(int argc, char **argv) {
    const int PLANT = atoi(argv[1]);  // added to the multiplier: a planted mistake
    const int top = 2147483647;
    long long wrong = 0, seen = 0;
    auto check = [&](int d, long long n) {
        if (n < 0 || n > top) return;
        fslk::FastDiv f = fslk::fast_div(d);
        f.m += (unsigned)PLANT;
        ++seen;
        wrong += fslk::div_by((int)n, f) != (int)(n / d);
    };
    auto around = [&](int d) {
        for (long long q : {0ll, 1ll, 2ll, 3ll, (long long)top / d - 1, (long long)top / d, (long long)top / (2ll * d), 65535ll, 65536ll})
            for (long long e = -1; e <= 1; ++e) check(d, q * d + e);
        check(d, top);
        for (int k = 0; k < 31; ++k) check(d, (1ll << k) - 1), check(d, 1ll << k);
    };
    for (int d = 1; d <= 70000; ++d) around(d);                   // every ny and nz, nx up to there
    for (int k = 16; k < 31; ++k)
        for (int e = -2; e <= 2; ++e)
            if ((1ll << k) + e <= 16776960) around((1 << k) + e);  // nx up to 65535 * 256
    around(16776960);
    printf("%lld %lld\n", wrong, seen);
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    from paper_1509_07691_gb300 import build as b
    d = tmp_path_factory.mktemp("division")
    (d / "m.cu").write_text(MAIN)
    subprocess.run([b.nvcc(), "-O2", "-std=c++17", "--expt-relaxed-constexpr", *b.ARCH, "-I", b.INCLUDE, "-I", b.CSRC,
                    str(d / "m.cu"), "-o", str(d / "m")], check=True, capture_output=True)
    return os.fspath(d / "m")


def _run(program, plant):
    out = subprocess.run([program, str(plant)], check=True, capture_output=True, text=True).stdout
    wrong, seen = map(int, out.split())
    assert seen > 3_000_000
    return wrong


def test_library_division_is_exact(program):
    assert _run(program, 0) == 0


@pytest.mark.parametrize("plant", [-1, 1])
def test_a_multiplier_off_by_one_shows(program, plant):
    assert _run(program, plant) > 0
