"""Where the FP64 path takes the polynomial of the sparse hopping and where the
dense E (csrc/series.h, series_pays64), on the CPU: the lattices and degrees that
were measured on both sides; and, on the GPU, both forms against the oracle right
at the line."""
import os
import shutil
import subprocess

import numpy as np
import pytest
import torch

from oracle import lattice, operators as ops
from paper_2210_06874_gb300 import hmc, synth

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MAIN = r"""
#include "%s/paper_2210_06874_gb300/csrc/series.h"
#include <stdio.h>
#include <stdlib.h>
int main(int n, char** v) {
    for (int i = 1; i + 1 < n; i += 2) {
        hmc::HopSeries s;
        const int L = atoi(v[i]);
        hmc::hop_series_build(L, atof(v[i + 1]), 1.0, &s);
        printf("%%d %%d\n", hmc::series_pays64(2 * L * L, s.k64, false) ? 1 : 0,
               hmc::series_pays64(2 * L * L, s.k64, true) ? 1 : 0);
    }
}
"""
# (L, delta kappa, series in an application, series in a solve): the faster side as
# measured
MEASURED = [(2, 0.125, 0, 0), (3, 0.125, 0, 0), (4, 0.25, 0, 0),
            (5, 0.125, 1, 1), (5, 0.25, 1, 0), (5, 0.8, 0, 0), (5, 1.3, 0, 0),
            (6, 0.125, 1, 1), (6, 0.25, 1, 1), (6, 0.5, 1, 1), (6, 0.8, 1, 0), (6, 1.3, 0, 0),
            (7, 0.25, 1, 1), (7, 1.3, 1, 1), (8, 1.0, 1, 1), (12, 0.125, 1, 1),
            (12, 1.3, 1, 1)]


def test_rule_takes_the_measured_side(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    (tmp_path / "m.cpp").write_text(MAIN % ROOT)
    subprocess.run([cxx, "-O2", "-o", str(tmp_path / "m"), str(tmp_path / "m.cpp")], check=True)
    args = [repr(a) for L, dk, *_ in MEASURED for a in (L, dk)]
    out = subprocess.run([str(tmp_path / "m")] + args, check=True, capture_output=True,
                         text=True).stdout.split()
    assert [int(o) for o in out] == [s for m in MEASURED for s in m[2:]]


@pytest.mark.gpu
@pytest.mark.parametrize("L,dk", [(5, 0.25), (5, 0.5), (6, 0.8), (6, 1.0)])
def test_both_sides_of_the_line_against_oracle(L, dk):
    """Tolerance as in test_gpu_series.py: 1e-13 times the condition of E."""
    Nt, U, V = 6, 2.0, 2 * L * L
    c = hmc.Context(hmc.Params(L=L, Nt=Nt, beta=dk * Nt, U=U))
    E = ops.transfer_matrix(lattice.hopping_matrix(L), dk)
    phi = synth.gaussian_field(501, Nt, V, dk * U, scale=0.3)
    psi = synth.complex_gaussian(502, Nt, V)
    tphi, tpsi = torch.from_numpy(phi).cuda(), torch.from_numpy(psi).cuda()
    tol = 1e-13 * max(1.0, np.exp(6 * dk - 0.75))
    for f, want in ((c.apply_M, ops.apply_M), (c.apply_Mdag, ops.apply_Mdag)):
        w = want(E, phi, psi)
        assert np.linalg.norm(f(tphi, tpsi).cpu().numpy() - w) < tol * np.linalg.norm(w)
    if dk > 0.6:
        return
    x, st = c.cg_solve(tphi, tpsi, tol=1e-11)
    r = psi - ops.apply_MMdag(E, phi, x.cpu().numpy())
    assert st.status == 0 and np.linalg.norm(r) < 1e-10 * np.linalg.norm(psi)
