"""Batches on the series (automatic operand mode) whose cluster teams the caller
chose: every team size, uneven slices per CTA, one-CTA chains beside them, two
trajectories in a row; against the FP64 path from the same fields."""
import numpy as np
import pytest
import torch

from paper_2210_06874_gb300 import hmc, synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"

# (L, Nt, U, team): team 1 is replaced by the tested size
CHAINS = [(6, 16, 3.0, 1), (12, 9, 3.5, 1), (9, 17, 4.0, 1), (3, 8, 2.0, 0), (9, 12, 2.5, 0)]


@pytest.mark.parametrize("team", [2, 4, 8])
def test_chosen_teams_follow_the_fp64_path(team):
    kw = [dict(L=L, Nt=Nt, U=U, beta=0.125 * Nt, n_md=3, traj_length=0.3)
          for L, Nt, U, _ in CHAINS]
    b = hmc.Batch([hmc.Params(cg_tol=1e-10, precision=hmc.PREC_MIXED,
                              team_ctas=team if c[3] else 1, **k) for c, k in zip(CHAINS, kw)])
    phi = torch.zeros(b.total, dtype=torch.float64, device=DEV)
    want = []
    for i, (L, Nt, U, _) in enumerate(CHAINS):
        f = torch.from_numpy(synth.gaussian_field(90 + i, Nt, 2 * L * L, 0.125 * U, scale=0.4))
        want.append(f.to(DEV))
        b.view(phi, i).copy_(want[i])
    for traj in (0, 1):
        outs = b.trajectory(phi, 22, traj)
        for i, k in enumerate(kw):
            o = hmc.Context(hmc.Params(cg_tol=1e-12, **k)).trajectory(want[i], 22, traj, chain=i)
            assert outs[i].status == 0 and outs[i].max_true_residual <= 1e-10
            assert outs[i].accept == o.accept and abs(outs[i].dH - o.dH) < 1e-7
            a, w = b.view(phi, i).cpu().numpy(), want[i].cpu().numpy()
            assert np.linalg.norm(a - w) < 1e-8 * np.linalg.norm(w)
            b.view(phi, i).copy_(want[i])      # the next one from the same field
