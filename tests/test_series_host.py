"""The polynomial of the sparse hopping that stands for E = exp(delta kappa h)
(csrc/series.h), on the CPU: the host code's coefficients, compiled with the
system compiler, against exp over the spectrum [-3, 3] of h.

Tolerance: the series is cut where its tail is below 2e-17 (FP64) and 6e-9
(FP32) of the smallest value e^{-rho}; each coefficient ratio is rounded once,
which moves the polynomial by at most rho roundings of its largest value
e^{rho}."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MAIN = r"""
#include "%s/paper_2210_06874_gb300/csrc/series.h"
#include <stdio.h>
#include <stdlib.h>
int main(int n, char** v) {
    for (int i = 1; i + 2 < n; i += 3) {
        hmc::HopSeries s;
        hmc::hop_series_build(atoi(v[i]), atof(v[i + 1]), atof(v[i + 2]), &s);
        printf("%%d %%d %%d %%.17g %%.9g", s.ok, s.k64, s.k32, s.c0, s.c0f);
        for (int k = 0; k < s.k64; ++k) printf(" %%.17g", s.r64[k]);
        for (int k = 0; k < s.k32; ++k) printf(" %%.9g", s.r32[k]);
        printf("\n");
    }
}
"""
CASES = [(6, 0.0, 1.0), (6, 1e-3, 1.0), (6, 0.125, 1.0), (24, 0.125, 0.9), (3, 0.25, 1.0),
         (1, -0.125, 1.0), (9, 0.5, 1.2), (32, 1.0, 1.0), (5, 4.0 / 3.0, 1.0),
         (5, 1.34, 1.0), (33, 0.125, 1.0)]


@pytest.fixture(scope="module")
def rows(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("series")
    (d / "m.cpp").write_text(MAIN % ROOT)
    subprocess.run([cxx, "-O2", "-o", str(d / "m"), str(d / "m.cpp")], check=True)
    args = [repr(a) for c in CASES for a in c]
    out = subprocess.run([str(d / "m")] + args, check=True, capture_output=True, text=True).stdout
    return [[float(w) for w in line.split()] for line in out.splitlines()]


@pytest.mark.parametrize("i", range(len(CASES)))
def test_series_against_exp(rows, i):
    L, dk, f = CASES[i]
    ok, k64, k32, c0, c0f = rows[i][:5]
    rho = 3 * abs(dk)
    if rho > 4.0 or L > 32:
        assert ok == 0
        return
    assert ok == 1
    k64, k32 = int(k64), int(k32)
    x = np.linspace(-3, 3, 601).astype(np.longdouble)
    want = f * np.exp(np.longdouble(dk) * x)
    for c, r, tail, u in ((c0, rows[i][5:5 + k64], 2e-17, 2.0 ** -53),
                          (c0f, rows[i][5 + k64:], 6e-9, 2.0 ** -24)):
        y = np.ones_like(x)
        for ratio in reversed(r):
            y = 1 + np.longdouble(ratio) * x * y
        bound = f * (tail * np.exp(-rho) + (2 * rho + 2) * u * np.exp(rho))
        assert np.max(np.abs(c * y - want)) <= bound
    assert len(rows[i]) == 5 + k64 + k32
