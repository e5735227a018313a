"""E = exp(delta (kappa h - mu)) by the polynomial of the sparse hopping, on the
GPU, at the edges of its tiles and of the rule that chooses it: one to four
cells per thread, one or several slices per tile, one component at a time,
lattices and delta kappa just inside and just outside (where the dense E takes
over), negative kappa, mu, Nt = 1 and the wrapped bonds of L = 1 and 2.

Tolerance: the FP64 applications' 1e-13 of the other parity tests, times the
condition e^{2 rho} / e^{0.75} of E (rho = 3 |delta kappa|; 0.75 is theirs)."""
import numpy as np
import pytest
import torch

from oracle import hmc as ohmc, lattice, operators as ops
from paper_2210_06874_gb300 import hmc, synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"

# (L, Nt, kappa, delta, mu)
CASES = [(1, 1, 1.0, 0.125, 0.0), (1, 5, -1.0, 0.25, 0.0), (2, 3, 1.0, 0.125, 0.4),
         (5, 7, 0.0, 0.125, 0.0), (15, 2, 1.0, 0.125, 0.0), (16, 3, 1.0, 0.125, 0.0),
         (17, 3, -1.0, 0.125, 0.2), (22, 2, 1.0, 0.125, 0.0), (23, 2, 1.0, 0.125, 0.0),
         (27, 2, 1.0, 0.125, 0.0), (28, 2, 1.0, 0.125, 0.0), (32, 2, 1.0, 0.125, 0.0),
         (33, 2, 1.0, 0.125, 0.0), (3, 200, 1.0, 0.125, 0.0), (6, 4, 1.0, 1.3, 0.0),
         (6, 4, 1.0, 1.4, 0.0)]


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


@pytest.mark.parametrize("L,Nt,kappa,delta,mu", CASES)
def test_fp64_against_oracle(L, Nt, kappa, delta, mu):
    V, U = 2 * L * L, 2.0
    c = hmc.Context(hmc.Params(L=L, Nt=Nt, kappa=kappa, beta=delta * Nt, U=U, mu=mu))
    E = np.exp(-delta * mu) * ops.transfer_matrix(lattice.hopping_matrix(L), delta * kappa)
    phi = synth.gaussian_field(900 + L, Nt, V, delta * U, scale=0.4)
    psi = synth.complex_gaussian(901 + L, Nt, V)
    tol = 1e-13 * max(1.0, np.exp(6 * abs(delta * kappa) - 0.75))
    assert rel(c.apply_M(dev(phi), dev(psi)).cpu().numpy(), ops.apply_M(E, phi, psi)) < tol
    assert rel(c.apply_Mdag(dev(phi), dev(psi)).cpu().numpy(), ops.apply_Mdag(E, phi, psi)) < tol
    F = c.force(dev(phi), dev(psi)).cpu().numpy()
    assert rel(F, ohmc.force_from_solution(E, phi, psi, delta, U)) < 10 * tol
    if delta < 1.0:
        x, st = c.cg_solve(dev(phi), dev(psi), tol=1e-12)
        r = psi - ops.apply_MMdag(E, phi, x.cpu().numpy())
        assert st.status == 0 and np.linalg.norm(r) < 1e-11 * np.linalg.norm(psi)
