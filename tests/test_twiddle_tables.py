"""The FP64 data path's twiddle factors are the correctly rounded ones, whatever long double the host has."""
import os
import subprocess

import pytest

from tests import fake_runtime as fr

mp = pytest.importorskip("mpmath")

MAIN = r"""
#include <cstdio>
#include <cstdlib>
#include "sfft_internal.h"
int main(int, char** argv) {
    const uint32_t L = (uint32_t)std::atoi(argv[1]);
    std::vector<double2> t;
    sfft::twiddle_tables_exact_host(uint64_t(1) << L, (L + 1) / 2, &t);
    for (const double2& v : t) std::printf("%a %a\n", v.x, v.y);
}
"""


@pytest.mark.parametrize("L", [6, 7, 13, 20, 25])
def test_factors_are_correctly_rounded(tmp_path, L):
    """exp(-2 pi i b / n) - 1 for b < 2^sh, then exp(-2 pi i a 2^sh / n), against 200 bits."""
    fr.load(tmp_path)
    cuda = os.path.dirname(os.path.dirname(fr.build._nvcc())) or "/usr/local/cuda"
    (tmp_path / "main.cpp").write_text(MAIN)
    exe = str(tmp_path / "tables")
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(cuda, "include"), "-I", fr.build.CSRC, "-I",
                    os.path.join(fr.build.ROOT, "include"), str(tmp_path / "main.cpp"), "-o", exe,
                    str(tmp_path / "libsfft_fake.so"), "-Wl,-rpath," + str(tmp_path)], check=True)
    rows = [[float.fromhex(v) for v in line.split()] for line in
            subprocess.run([exe, str(L)], capture_output=True, text=True, check=True).stdout.splitlines()]
    n, sh = 1 << L, (L + 1) // 2
    assert len(rows) == (1 << sh) + (n >> sh)
    with mp.workprec(200):
        for i, got in enumerate(rows):
            m = i if i < 1 << sh else (i - (1 << sh)) << sh
            c, s = mp.cospi(mp.mpf(2 * m) / n), mp.sinpi(mp.mpf(2 * m) / n)
            if i < 1 << sh:
                c = -2 * mp.sinpi(mp.mpf(m) / n) ** 2
            assert got == [float(c), float(-s)], (L, i)
