"""The bounded waits inside the series' FP32 iterations (csrc/series_cg.cuh), on
the GPU: with a limit of 5 ms and one CTA whose messages carry other numbers than
its peers wait for (host-side injection), the waits run out -- its neighbours' for
its boundary slices, the others' for its norm, its own for theirs -- the launch
ends with HMC_ERR_TIMEOUT, and the context then solves correctly: for
a team that is one cluster (mail in distributed shared memory) and for one
with its mail in global memory, whose sequence numbers carry on from the
failed launch.  (The team padding of test_gpu_waits.py, whose mixed automatic
case is this path too, ends a launch before its first iteration.)"""
import numpy as np
import pytest
import torch

from oracle import hmc as ohmc, lattice, operators as ops
from paper_2210_06874_gb300 import hmc, synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


# 8 CTAs in a cluster; 40 CTAs of one slice each
@pytest.mark.parametrize("L,Nt", [(3, 8), (16, 40)])
@pytest.mark.parametrize("ahead", [64, 1024])
def test_misnumbered_messages_time_out(L, Nt, ahead):
    U, delta = 2.0, 0.125
    V = 2 * L * L
    phi = synth.gaussian_field(401, Nt, V, delta * U, scale=0.3)
    chi = synth.complex_gaussian(402, Nt, V)
    tphi, tchi = torch.from_numpy(phi).to(DEV), torch.from_numpy(chi).to(DEV)
    ctx = hmc.Context(hmc.Params(L=L, Nt=Nt, beta=delta * Nt, U=U, n_md=2, traj_length=0.2,
                                 precision=hmc.PREC_MIXED, cg_tol=1e-10))
    ctx.set_wait_limit(0.005)
    for _ in range(2):                       # the failure repeats, the context survives
        ctx.debug_misnumber(ahead)
        with pytest.raises(hmc.HmcError) as e:
            ctx.cg_solve(tphi, tchi, tol=1e-10, prec=hmc.PREC_MIXED)
        assert e.value.code == hmc.HMC_ERR_TIMEOUT
        with pytest.raises(hmc.HmcError) as e:
            ctx.trajectory(tphi.clone(), 5, 0)
        assert e.value.code == hmc.HMC_ERR_TIMEOUT
        ctx.debug_misnumber(0)
        x, st = ctx.cg_solve(tphi, tchi, tol=1e-10, prec=hmc.PREC_MIXED)
        assert st.status == hmc.HMC_OK and st.true_residual <= 1e-10
    E = ops.transfer_matrix(lattice.hopping_matrix(L), delta)
    xo, _, _ = ohmc.cg_solve(E, phi, chi, tol=1e-13)
    x = x.cpu().numpy()
    assert np.linalg.norm(x - xo) < 1e-8 * np.linalg.norm(xo)


def test_bad_misnumber_arguments():
    ctx = hmc.Context(hmc.Params(L=2, Nt=4))
    for bad in (-1, 1025):
        with pytest.raises(hmc.HmcError) as e:
            ctx.debug_misnumber(bad)
        assert e.value.code == hmc.HMC_ERR_BAD_ARG
