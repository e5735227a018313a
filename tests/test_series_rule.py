"""Where the FP64 path takes the polynomial of the sparse hopping and where the
dense E (csrc/series.h, series_pays64), and where the mixed path takes one cluster
and where a global-memory team (series_on_cluster), on the CPU: the sizes that were
measured on both sides; and, on the GPU, both sides right at the lines."""
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
    if (n == 4) {
        printf("%%d\n", hmc::series_on_cluster(atoi(v[1]), atoi(v[2]), atoi(v[3])) ? 1 : 0);
        return 0;
    }
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


# (L, Nt, CTAs there could be, cluster)
CLUSTER = [(3, 8, 8, 1), (6, 32, 32, 1), (6, 64, 64, 1), (8, 48, 48, 1), (6, 96, 96, 1),
           (6, 128, 128, 1), (6, 150, 150, 1), (9, 24, 24, 1), (8, 36, 36, 1), (3, 200, 152, 1),
           (16, 16, 16, 1), (20, 16, 16, 1), (9, 48, 48, 0), (9, 36, 36, 0), (8, 64, 64, 0),
           (12, 18, 18, 0), (11, 24, 24, 0), (12, 32, 32, 0), (9, 64, 64, 0), (12, 48, 48, 0),
           (16, 32, 32, 0), (7, 96, 96, 0), (7, 128, 128, 0), (12, 64, 64, 0), (24, 96, 96, 0),
           (27, 3, 3, 0), (6, 32, 3, 1), (9, 20, 1, 0)]


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("rule")
    (d / "m.cpp").write_text(MAIN % ROOT)
    subprocess.run([cxx, "-O2", "-o", str(d / "m"), str(d / "m.cpp")], check=True)

    def run(*args):
        return [int(w) for w in subprocess.run([str(d / "m"), *map(repr, args)], check=True,
                                               capture_output=True, text=True).stdout.split()]
    return run


def test_rule_takes_the_measured_side(program):
    out = program(*[a for L, dk, *_ in MEASURED for a in (L, dk)])
    assert out == [s for m in MEASURED for s in m[2:]]


@pytest.mark.parametrize("L,Nt,T,cluster", CLUSTER)
def test_cluster_or_global_team(program, L, Nt, T, cluster):
    assert program(L * L, Nt, T) == [cluster]


@pytest.mark.gpu
@pytest.mark.parametrize("L,Nt", [(8, 48), (9, 48), (6, 128), (8, 64), (9, 33), (24, 17)])
def test_mixed_solves_around_the_cluster_line(L, Nt):
    """Clusters and global teams, even and uneven slices: the FP64 path's residual of
    the mixed solution (1e-10 asked for), and the same bits a second time."""
    V, U, delta = 2 * L * L, 2.0, 0.125
    c = hmc.Context(hmc.Params(L=L, Nt=Nt, beta=delta * Nt, U=U, precision=hmc.PREC_MIXED))
    E = ops.transfer_matrix(lattice.hopping_matrix(L), delta)
    phi = synth.gaussian_field(503, Nt, V, delta * U, scale=0.3)
    chi = synth.complex_gaussian(504, Nt, V)
    tphi, tchi = torch.from_numpy(phi).cuda(), torch.from_numpy(chi).cuda()
    x, st = c.cg_solve(tphi, tchi, tol=1e-10, prec=hmc.PREC_MIXED)
    r = chi - ops.apply_MMdag(E, phi, x.cpu().numpy())
    assert st.status == 0 and np.linalg.norm(r) < 1.2e-10 * np.linalg.norm(chi)
    y, _ = c.cg_solve(tphi, tchi, tol=1e-10, prec=hmc.PREC_MIXED)
    assert torch.equal(x, y)


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
