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


# mixed path, automatic choice: (L, Nt, team_ctas, kappa, delta, mu) -- one CTA
# with its vectors in registers and in memory, clusters, global-memory teams,
# one and two cells per thread, several and ragged slices per CTA, one slice, and
# the lattices and delta kappa beyond which the tensor-core tiles take over
MIXED = [(1, 1, 0, 1.0, 0.125, 0.0), (1, 3, 1, 1.0, 0.125, 0.0), (2, 1, 0, 1.0, 0.125, 0.0),
         (3, 8, 0, 1.0, 0.25, 0.0), (3, 8, 1, 1.0, 0.25, 0.3), (4, 5, 3, -1.0, 0.125, 0.0),
         (3, 200, 0, 1.0, 0.05, 0.0), (6, 32, 0, 1.0, 0.125, 0.0), (6, 32, 3, 1.0, 0.125, 0.0),
         (5, 7, 0, 0.0, 0.125, 0.0), (9, 20, 0, 1.0, 0.125, 0.0), (9, 37, 0, 1.0, 0.125, 0.0),
         (12, 33, 1, 1.0, 0.125, 0.0), (16, 6, 2, 1.0, 0.125, 0.0), (17, 18, 0, 1.0, 0.125, 0.0),
         (23, 4, 0, 1.0, 0.125, 0.0), (27, 3, 0, 1.0, 0.125, 0.0), (28, 2, 0, 1.0, 0.125, 0.0),
         (4, 6, 0, 1.0, 1.4, 0.0)]


@pytest.mark.parametrize("L,Nt,team,kappa,delta,mu", MIXED)
def test_mixed_against_oracle(L, Nt, team, kappa, delta, mu):
    """Applications to 2e-6 (the bound of every mixed application) and a solve to
    the FP64 residual 1e-10, twice with the same bits."""
    V, U = 2 * L * L, 2.0
    c = hmc.Context(hmc.Params(L=L, Nt=Nt, kappa=kappa, beta=delta * Nt, U=U, mu=mu,
                               team_ctas=team, precision=hmc.PREC_MIXED))
    E = np.exp(-delta * mu) * ops.transfer_matrix(lattice.hopping_matrix(L), delta * kappa)
    phi = synth.gaussian_field(910 + L, Nt, V, delta * U, scale=0.3)
    psi = synth.complex_gaussian(911 + L, Nt, V)
    p32 = dev(psi).to(torch.complex64)
    seen = p32.cpu().numpy().astype(np.complex128)
    tol = 2e-6 * max(1.0, np.exp(6 * abs(delta * kappa) - 1.5))
    assert rel(c.apply_M(dev(phi), p32, prec=hmc.PREC_MIXED).cpu().numpy(),
               ops.apply_M(E, phi, seen)) < tol
    assert rel(c.apply_Mdag(dev(phi), p32, prec=hmc.PREC_MIXED).cpu().numpy(),
               ops.apply_Mdag(E, phi, seen)) < tol
    if delta > 1.0:
        return
    x, st = c.cg_solve(dev(phi), dev(psi), tol=1e-10, prec=hmc.PREC_MIXED)
    r = psi - ops.apply_MMdag(E, phi, x.cpu().numpy())
    assert st.status == 0 and np.linalg.norm(r) < 1.2e-10 * np.linalg.norm(psi)
    x2, st2 = c.cg_solve(dev(phi), dev(psi), tol=1e-10, prec=hmc.PREC_MIXED)
    assert st2.iterations == st.iterations and torch.equal(x, x2)


def test_mixed_trajectory_follows_the_fp64_one():
    """A trajectory on the automatic choice against the plain FP64 path's."""
    L, Nt = 9, 21
    kw = dict(L=L, Nt=Nt, beta=0.125 * Nt, U=3.0, n_md=4, traj_length=0.4)
    phi = dev(synth.gaussian_field(77, Nt, 2 * L * L, 0.375, scale=0.4))
    a, b = phi.clone(), phi.clone()
    oa = hmc.Context(hmc.Params(cg_tol=1e-10, precision=hmc.PREC_MIXED, **kw)).trajectory(a, 3, 1)
    ob = hmc.Context(hmc.Params(cg_tol=1e-12, **kw)).trajectory(b, 3, 1)
    assert oa.status == 0 and oa.accept == ob.accept and abs(oa.dH - ob.dH) < 1e-7
    assert rel(a.cpu().numpy(), b.cpu().numpy()) < 1e-8


def test_batch_puts_large_chains_on_clusters():
    """A batch that leaves the teams to the library runs its chains of over 2048
    sites on clusters of 8 CTAs: against the FP64 path from the same fields."""
    sizes = [(12, 24, 3.0), (3, 8, 2.0), (9, 16, 4.0), (9, 15, 3.5), (24, 4, 3.0)]
    kw = [dict(L=L, Nt=Nt, U=U, beta=0.125 * Nt, n_md=3, traj_length=0.3) for L, Nt, U in sizes]
    b = hmc.Batch([hmc.Params(cg_tol=1e-10, precision=hmc.PREC_MIXED, **k) for k in kw])
    phi = torch.zeros(b.total, dtype=torch.float64, device=DEV)
    starts = [dev(synth.gaussian_field(80 + i, Nt, 2 * L * L, 0.125 * U, scale=0.4))
              for i, (L, Nt, U) in enumerate(sizes)]
    for i, f in enumerate(starts):
        b.view(phi, i).copy_(f)
    outs = b.trajectory(phi, 21, 2)
    for i, k in enumerate(kw):
        want = starts[i].clone()
        o = hmc.Context(hmc.Params(cg_tol=1e-12, **k)).trajectory(want, 21, 2, chain=i)
        assert outs[i].status == 0 and outs[i].max_true_residual <= 1e-10
        assert outs[i].accept == o.accept and abs(outs[i].dH - o.dH) < 1e-7
        assert rel(b.view(phi, i).cpu().numpy(), want.cpu().numpy()) < 1e-8
