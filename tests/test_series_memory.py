"""Where a CTA of the series' iterations keeps its CG vectors (csrc/series.h,
vector_fits), on the CPU: sizes whose byte count passes 2^32 do not fit."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MAIN = r"""
#include "%s/paper_2210_06874_gb300/csrc/series.h"
#include <stdio.h>
#include <stdlib.h>
int main(int n, char** v) {
    for (int i = 1; i + 3 < n; i += 4)
        printf("%%d\n", hmc::vector_fits(atoll(v[i]), atoi(v[i + 1]), atoi(v[i + 2]),
                                         atoll(v[i + 3])) ? 1 : 0);
}
"""
# (bytes taken, slices, sites, bytes in all)
CASES = [(0, 1, 2, 16), (1, 1, 2, 16), (0, 1, 2, 15), (24576, 4, 288, 228000),
         (0, 2 ** 28, 2, 228000), (4096, 2 ** 28, 2, 228000), (4096, 2 ** 29 // 2 + 8, 2, 228000),
         (0, 2 ** 29, 2, 228000), (24576, 736439, 1458, 228000), (24576, 368220, 1458, 228000)]


def test_vector_fits(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    (tmp_path / "m.cpp").write_text(MAIN % ROOT)
    subprocess.run([cxx, "-O2", "-o", str(tmp_path / "m"), str(tmp_path / "m.cpp")], check=True)
    args = [str(a) for c in CASES for a in c]
    out = subprocess.run([str(tmp_path / "m")] + args, check=True, capture_output=True,
                         text=True).stdout.split()
    assert [int(o) for o in out] == [int(top + 8 * S * V <= n) for top, S, V, n in CASES]
